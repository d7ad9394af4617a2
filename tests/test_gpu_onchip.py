"""The compress kernels that keep x on chip between their two halves: exact parity with the CPU checker at the edges of
their tilings (widths of every alignment, short bands, narrow tiles, shares that do not divide evenly, degenerate and
extreme values that leave the fixed-point quantiser), and their bounded wait."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import division_oracle as orc
from paper_2208_04187_b200 import binding, build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built_library():
    build.build()
    binding.lib()


def check(x_np, block, q, seed, xd="f32", ld="f32", on_chip=1):
    codec = binding.Codec(*x_np.shape, block, q, xd, ld)
    assert codec.plan().on_chip == on_chip
    t = torch.from_numpy(x_np)
    t = (t.view(torch.bfloat16) if xd == "bf16" else t).cuda()
    codec.compress(t, seed=seed)
    ref = orc.compress(x_np, block, q, seed, xd, ld)
    torch.cuda.synchronize()
    assert codec.device_status() == binding.DIV_OK
    np.testing.assert_array_equal(codec.blob.cpu().numpy(), ref.blob())


def make(shape, kind, seed, xd):
    x = synth.activation_map(*shape, kind, seed)
    return synth.to_bf16_bits(x) if xd == "bf16" else x


CLUSTER = [   # n, c, h, w, block, q, x, lfc
    (3, 8, 32, 32, 8, 2, "f32", "f32"), (2, 37, 8, 12, 8, 4, "f32", "bf16"), (5, 4, 7, 7, 8, 2, "f32", "f32"),
    (2, 36, 13, 9, 4, 8, "f32", "f32"), (2, 12, 75, 75, 8, 2, "f32", "bf16"), (3, 8, 61, 47, 16, 2, "bf16", "bf16"),
    (2, 8, 33, 34, 16, 4, "f32", "f32"), (2, 24, 14, 14, 8, 2, "bf16", "f32"), (4, 16, 19, 19, 8, 4, "bf16", "bf16"),
    (1, 4, 5, 5, 4, 2, "f32", "f32"), (2, 16, 30, 10, 12, 2, "f32", "f32"), (2, 8, 21, 6, 6, 8, "f32", "f32"),
    (9, 64, 4, 4, 8, 2, "f32", "f32"), (1, 2048, 7, 7, 8, 2, "f32", "f32"), (2, 3, 100, 100, 8, 4, "f32", "f32"),
]


PLANE_SHARE = [   # n, c, h, w, block, q, x, lfc: odd widths beyond a warp, blocks of 16, quads that straddle planes
    (2, 8, 75, 75, 8, 2, "f32", "f32"), (3, 12, 35, 35, 8, 4, "f32", "bf16"), (2, 5, 40, 40, 16, 4, "f32", "f32"),
    (2, 8, 39, 37, 4, 8, "bf16", "bf16"), (1, 44, 9, 41, 16, 2, "f32", "f32"), (2, 16, 17, 70, 12, 2, "bf16", "f32"),
    (4, 8, 3, 50, 4, 2, "f32", "f32"),
]


@pytest.mark.parametrize("case", CLUSTER + PLANE_SHARE, ids=lambda c: "x".join(map(str, c)))
def test_the_plan_describes_the_launch(case):
    """What runs, not what would run in its place: shares of whole planes that cover the sample, and room for them."""
    n, c, h, w, block, q, xd, ld = case
    plan = (binding.Codec if case in CLUSTER else binding.PlaneGroupCodec)(*case).plan()
    assert plan.on_chip == 1 and plan.grid == n * plan.chunks_per_sample and plan.threads in (256, 384, 512)
    assert plan.chunk_elems % (h * w) == 0 and plan.chunks_per_sample * plan.chunk_elems >= c * h * w
    assert plan.chunk_elems * (4 if xd == "f32" else 2) <= plan.smem_bytes <= 232448
    if case in CLUSTER:
        assert plan.chunks_per_sample in (1, 2, 4, 8, 16) and plan.stages >= 1


@pytest.mark.parametrize("case", CLUSTER, ids=lambda c: "x".join(map(str, c)))
def test_cluster_kernel_matches_the_checker(case):
    n, c, h, w, block, q, xd, ld = case
    check(make((n, c, h, w), "bn" if c % 3 else "relu", 11 + h, xd), block, q, 77, xd, ld)


IN_PLACE = [   # bfloat16, W % 4 == 0, B = 4 or 8: x stays as it is
    (2, 8, 32, 32, 8, 2, "bf16"), (3, 16, 28, 28, 8, 4, "f32"), (2, 40, 20, 12, 4, 8, "bf16"), (2, 24, 5, 36, 8, 2, "f32"),
    (5, 2, 9, 4, 4, 4, "bf16"), (1, 512, 7, 8, 8, 8, "f32"),
]


@pytest.mark.parametrize("case", IN_PLACE, ids=lambda c: "x".join(map(str, c)))
def test_cluster_kernel_with_bfloat16_in_place(case):
    n, c, h, w, block, q, ld = case
    x = make((n, c, h, w), "bn", 21 + h, "bf16")
    check(x, block, q, 78, "bf16", ld)
    x[0] = 0x4050                              # a constant sample leaves the fixed-point route
    check(x, block, q, 79, "bf16", ld)


@pytest.mark.parametrize("case", [(32, 64, 75, 75, 8, "f32"), (64, 1024, 14, 14, 8, "f32"), (24, 512, 28, 28, 8, "f32"),
                                  (30, 64, 90, 90, 16, "bf16")], ids=lambda c: "x".join(map(str, c)))
def test_cluster_kernel_in_wide_blocks(case):
    """Shares of which two fit an SM, more of them than fit at once: the same bytes as the kernel with a pass per half."""
    n, c, h, w, block, xd = case
    x = torch.randn((n, c, h, w), device="cuda", generator=torch.Generator("cuda").manual_seed(4)).to(torch.bfloat16 if xd == "bf16" else torch.float32)
    codec = binding.Codec(n, c, h, w, block, 2, xd, "f32")
    assert codec.plan().on_chip == 1
    blobs = []
    for flags in (0, binding.DIV_FLAG_FORCE_TWO_PASS):
        codec.blob.zero_()
        codec.compress(x, seed=6, flags=flags)
        torch.cuda.synchronize()
        assert codec.device_status() == binding.DIV_OK
        blobs.append(codec.blob.clone())
    assert torch.equal(*blobs)


# A share per SM in a single turn: more threads.
LONELY = [(1, 128, 56, 56, "f32"), (2, 64, 112, 112, "f32"), (1, 512, 28, 28, "f32"), (8, 3, 224, 224, "f32"), (4, 64, 112, 112, "bf16"), (1, 64, 75, 75, "f32")]


@pytest.mark.parametrize("case", LONELY, ids=lambda c: "x".join(map(str, c)))
def test_cluster_kernel_on_small_batches_of_large_samples(case):
    n, c, h, w, xd = case
    x = torch.randn((n, c, h, w), device="cuda", generator=torch.Generator("cuda").manual_seed(4)).to(binding.torch_dtype(xd))
    codec = binding.Codec(n, c, h, w, 8, 2, xd, "f32")
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        plan = codec.plan()
        assert not plan.on_chip or (plan.threads > 256 and plan.stages == 1)
    blobs = []
    for flags in (0, binding.DIV_FLAG_FORCE_TWO_PASS):
        codec.blob.zero_()
        codec.compress(x, seed=6, flags=flags)
        assert codec.device_status() == binding.DIV_OK
        blobs.append(codec.blob.clone())
    assert torch.equal(*blobs)


def test_turns_are_those_of_the_device():
    """148 SMs hold 7 clusters of 16 CTAs with a share per SM each, and 33 clusters of 8 with two: the next sample takes another
    turn.  Where that, or the batch, leaves the device to too few CTAs a kernel that spreads the map runs instead."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the figures are those of 148 SMs")

    def plan(*a):
        return binding.div_plan_query(binding.make_desc(*a))
    assert [plan(n, 64, 112, 112, 8, 2).stages for n in (7, 8)] == [1, 2]
    assert [plan(n, 1024, 14, 14, 8, 2).stages for n in (33, 34)] == [1, 2]
    assert plan(16, 3, 150, 150, 8, 2).chunks_per_sample == 4              # a plane per CTA: no more CTAs than planes
    for spread in ((1, 64, 112, 112, 8, 2, "bf16", "bf16"), (8, 64, 100, 152, 8, 2, "bf16", "bf16"), (64, 64, 112, 112, 8, 2), (64, 1024, 14, 14, 8, 2, "bf16", "bf16")):
        assert plan(*spread).on_chip == 0, spread


@pytest.mark.parametrize("q", [2, 4])
def test_values_outside_the_fixed_point_route(q):
    """Constant, tiny, huge and one-sided samples beside an ordinary one."""
    x = make((6, 16, 14, 14), "bn", 5, "f32")
    x[0] = 3.25
    x[1] *= np.float32(1e-30)
    x[2] *= np.float32(1e30)
    x[3] = 0.0
    x[4, 0, 0, 0] = 1e6
    check(x, 8, q, 9)


def test_cluster_kernel_gives_up_a_wait_that_cannot_end():
    x_np = make((4, 32, 14, 14), "relu", 3, "f32")
    x = torch.from_numpy(x_np).cuda()
    codec = binding.Codec(*x_np.shape, 8, 2)
    assert codec.plan().on_chip == 1
    st = binding.lib().div_debug_compress_starved(
        ctypes.byref(codec.desc), ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(codec.blob.data_ptr()), codec.blob.numel(),
        ctypes.c_void_p(codec.workspace.data_ptr()), codec.workspace.numel(), 0, ctypes.c_void_p(binding.current_stream_handle()),
        0, 2_000_000)
    assert st == binding.DIV_OK
    torch.cuda.synchronize()
    assert codec.device_status() == binding.DIV_ERR_TIMEOUT
    check(x_np, 8, 2, 5)


def debug_call(codec, x, fault, timeout_ns):
    return binding.lib().div_debug_on_chip(codec.desc, x.data_ptr(), codec.blob.data_ptr(), codec.blob.numel(), codec.workspace.data_ptr(),
                                           codec.workspace.numel(), 5, binding.current_stream_handle(), fault, timeout_ns)


def test_a_failure_of_the_same_call_is_not_cleared():
    """The CTA that clears the status word runs in no order with the others, one of which may have failed before it: what
    stands there under the call's own number (1) stays; a failure of another call goes."""
    x_np = make((4, 32, 14, 14), "relu", 3, "f32")
    x = torch.from_numpy(x_np).cuda()
    codec = binding.Codec(*x_np.shape, 8, 2)
    words = codec.workspace.view(torch.int32)
    for status, number, want in ((binding.DIV_ERR_TIMEOUT, 1, binding.DIV_ERR_TIMEOUT), (binding.DIV_ERR_TIMEOUT, 2, binding.DIV_OK),
                                 (-1, -1, binding.DIV_OK), (0, 0, binding.DIV_OK)):
        words[0], words[1] = status, number
        assert debug_call(codec, x, 0, 100_000_000) == binding.DIV_OK
        torch.cuda.synchronize()
        assert codec.device_status() == want
        np.testing.assert_array_equal(codec.blob.cpu().numpy(), orc.compress(x_np, 8, 2, 5).blob())
    assert debug_call(codec, x, 9, 100_000_000) == binding.DIV_ERR_PARAM


@pytest.mark.parametrize("case", [(4, 32, 14, 14, "f32"), (3, 24, 75, 75, "f32"), (4, 32, 32, 32, "bf16"), (40, 64, 75, 75, "f32")],
                         ids=lambda c: "x".join(map(str, c)))
@pytest.mark.parametrize("timeout_ns", [1, 1_000_000])
def test_a_wait_for_x_that_cannot_end(case, timeout_ns):
    """Every warp gives up on its first piece (or, with a limit of 1 ns, some of them on the exchange): the failure is
    recorded, nothing behind the blob is written, and the next call on the same buffers is an ordinary one.  The last
    case takes several turns."""
    n, c, h, w, xd = case
    x = torch.randn((n, c, h, w), device="cuda").to(binding.torch_dtype(xd))
    codec = binding.Codec(n, c, h, w, 8, 2, xd, "f32")
    assert codec.plan().on_chip == 1
    room = torch.full((codec.blob.numel() + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    whole, codec.blob = codec.blob, room[:codec.blob.numel()]
    codec.compress(x, seed=5)
    want = codec.blob.clone()
    assert debug_call(codec, x, 1, timeout_ns) == binding.DIV_OK
    torch.cuda.synchronize()
    assert codec.device_status() == binding.DIV_ERR_TIMEOUT
    assert bool((room[whole.numel():] == 0xA5).all())
    codec.compress(x, seed=5)
    assert codec.device_status() == binding.DIV_OK and torch.equal(codec.blob, want)


@pytest.mark.parametrize("case", PLANE_SHARE, ids=lambda c: "x".join(map(str, c)))
def test_plane_share_kernel_matches_the_checker(case):
    n, c, h, w, block, q, xd, ld = case
    x_np = make((n, c, h, w), "bn", 31 + h, xd)
    if xd == "f32":
        x_np[0, 1] = 0.0                        # a degenerate plane beside ordinary ones
        x_np[-1, 2] *= np.float32(1e-28)        # and one outside the fixed-point route
    codec = binding.PlaneGroupCodec(n, c, h, w, block, q, xd, ld)
    assert codec.plan().on_chip == 1
    t = torch.from_numpy(x_np)
    codec.compress((t.view(torch.bfloat16) if xd == "bf16" else t).cuda(), seed=13)
    np.testing.assert_array_equal(codec.blob.cpu().numpy(), orc.compress_planes(x_np, block, q, 13, xd, ld).blob())


@pytest.mark.parametrize("case", [(3, 12, 35, 35, "f32"), (40, 64, 39, 75, "bf16")], ids=lambda c: "x".join(map(str, c)))
@pytest.mark.parametrize("timeout_ns", [1, 1_000_000])
def test_plane_share_kernel_gives_up_a_wait_that_cannot_end(case, timeout_ns):
    """The planes rebuild as NaN, nothing behind the blob is written, and the next call on the same buffers is an ordinary one."""
    n, c, h, w, xd = case
    x = torch.randn((n, c, h, w), device="cuda").to(binding.torch_dtype(xd))
    codec = binding.PlaneGroupCodec(n, c, h, w, 8, 2, xd, "f32")
    assert codec.plan().on_chip == 1
    size = codec.blob.numel()
    room = torch.full((size + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    codec.blob = room[:size]
    codec.compress(x, seed=5)
    want = codec.blob.clone()
    st = binding.lib().div_debug_on_chip(codec.desc, x.data_ptr(), codec.blob.data_ptr(), size, None, 0, 5, binding.current_stream_handle(), 1, timeout_ns)
    assert st == binding.DIV_OK
    torch.cuda.synchronize()
    assert bool(torch.isnan(codec.decompress()).all())
    assert bool((room[size:] == 0xA5).all())
    codec.compress(x, seed=5)
    assert torch.equal(codec.blob, want)


@pytest.mark.parametrize("case", [(4, 32, 14, 14, 8, "f32"), (3, 16, 39, 39, 8, "bf16"), (2, 8, 32, 32, 8, "f32"), (20, 16, 19, 19, 4, "f32")],
                         ids=lambda c: "x".join(map(str, c)))
def test_a_refused_cluster_launch_leaves_the_map_to_the_next_kernel(case):
    """... over a workspace full of leftovers, which that kernel has to find cleared."""
    n, c, h, w, block, xd = case
    x_np = make((n, c, h, w), "bn", 17, xd)
    t = torch.from_numpy(x_np)
    x = (t.view(torch.bfloat16) if xd == "bf16" else t).cuda()
    codec = binding.Codec(n, c, h, w, block, 2, xd, "f32")
    assert codec.plan().on_chip == 1
    codec.workspace.fill_(0xFF)
    assert debug_call(codec, x, 2, 100_000_000) == binding.DIV_OK
    assert codec.device_status() == binding.DIV_OK
    np.testing.assert_array_equal(codec.blob.cpu().numpy(), orc.compress(x_np, block, 2, 5, xd, "f32").blob())
    assert bool((codec.workspace[64:80] != 0xFF).any())        # the slots were cleared and used: another kernel ran


# Maps that the parking kernel takes before clusters in turns, and before a kernel that reads x twice.
PARKED = [(128, 160, 32, 32, 4, 4, "bf16", "bf16"), (50, 2048, 16, 16, 4, 2, "f32", "f32"), (64, 64, 112, 112, 8, 2, "f32", "f32")]


@pytest.mark.parametrize("case", PARKED, ids=lambda c: "x".join(map(str, c)))
def test_a_refused_parking_launch_leaves_the_map_to_the_kernel_that_the_plan_names(case):
    """... over a workspace full of leftovers.  The cluster kernel leaves the slots as they were cleared, the others use them."""
    n, c, h, w, block, q, xd, ld = case
    x = torch.randn((n, c, h, w), device="cuda", generator=torch.Generator("cuda").manual_seed(4)).to(binding.torch_dtype(xd))
    codec = binding.Codec(*case)
    plan = codec.plan()
    assert plan.parked
    want = codec.compress(x, seed=5).clone()
    codec.workspace.fill_(0xFF)
    codec.blob.zero_()
    assert debug_call(codec, x, 3, 100_000_000) == binding.DIV_OK
    assert codec.device_status() == binding.DIV_OK and torch.equal(codec.blob, want)
    assert bool((codec.workspace[64:] == 0).all()) == bool(plan.on_chip)
    if not plan.on_chip:
        assert debug_call(codec, x, 0, 100_000_000) == binding.DIV_ERR_PARAM
        return
    # the hook's other faults are the clusters', whoever comes before them
    for fault, status in ((0, binding.DIV_OK), (1, binding.DIV_ERR_TIMEOUT), (2, binding.DIV_OK)):
        codec.blob.zero_()
        assert debug_call(codec, x, fault, 1_000_000 if fault == 1 else 100_000_000) == binding.DIV_OK
        assert codec.device_status() == status and (status != binding.DIV_OK or torch.equal(codec.blob, want))


def test_a_refused_plane_share_launch_leaves_the_map_to_the_general_kernel():
    x_np = make((2, 8, 75, 75), "bn", 17, "f32")
    x = torch.from_numpy(x_np).cuda()
    codec = binding.PlaneGroupCodec(2, 8, 75, 75, 8, 2)
    assert codec.plan().on_chip == 1
    st = binding.lib().div_debug_on_chip(codec.desc, x.data_ptr(), codec.blob.data_ptr(), codec.blob.numel(), None, 0, 5, binding.current_stream_handle(),
                                         2, 100_000_000)
    assert st == binding.DIV_OK
    np.testing.assert_array_equal(codec.blob.cpu().numpy(), orc.compress_planes(x_np, 8, 2, 5).blob())
