"""The compress kernel that parks residuals in tensor memory: the same bytes as the kernels with a pass per half, where its tilings end
(last chunks, short bands, narrow tiles, planes larger than a chunk) and where a sample just fits what is parked, or just does not.
(Small maps of every form against the CPU checker: test_gpu_parity, the same flags.)"""
import ctypes

import pytest
import torch

from paper_2208_04187_b200 import binding, build

pytestmark = pytest.mark.gpu

PARKED = binding.DIV_FLAG_NO_STRIP_KERNEL | binding.DIV_FLAG_NO_LAGGED_KERNEL


@pytest.fixture(scope="module", autouse=True)
def built_library():
    build.build()
    binding.lib()


def same_bytes(case, flags):
    n, c, h, w, block, q, xd, ld = case
    gen = torch.Generator("cuda").manual_seed(h * w)
    x = torch.randn((n, c, h, w), device="cuda", generator=gen)
    x[n // 2] *= 1e30                         # one sample off the fixed-point route
    x = x.to(binding.torch_dtype(xd))
    codec = binding.Codec(n, c, h, w, block, q, xd, ld)
    blobs = []
    for f in (flags, binding.DIV_FLAG_FORCE_TWO_PASS, flags):
        codec.blob.zero_()
        codec.compress(x, seed=11, flags=f)
        assert codec.device_status() == binding.DIV_OK
        blobs.append(codec.blob.clone())
    assert torch.equal(blobs[0], blobs[1]) and torch.equal(blobs[0], blobs[2])
    return codec.plan(flags)


PARK = [  # n, c, h, w, block, q, x, lfc
    (5, 64, 112, 112, 8, 2, "f32", "f32"),       # whole units, whole chunks
    (3, 37, 28, 28, 8, 4, "f32", "bf16"),        # short bands, single-strip tiles side by side, a last chunk of few planes
    (2, 19, 36, 36, 8, 8, "bf16", "bf16"),       # strips that do not fill their units
    (300, 8, 4, 4, 4, 2, "f32", "f32"),          # a sample per unit
    (9, 16, 14, 60, 4, 4, "bf16", "f32"),        # two strips a lane, short bands
    (2, 512, 112, 112, 8, 2, "bf16", "f32"),     # a CTA has several chunks of a sample
]


@pytest.mark.parametrize("case", PARK, ids=lambda c: "x".join(map(str, c)))
def test_parking_kernel_matches_the_two_pass_kernels(case):
    plan = same_bytes(case, PARKED)
    assert plan.fused == 6 and plan.parked and plan.threads == 1024 and plan.lag == 0


# More chunks a CTA than it has records for them (from 64 on), twice over for the small samples: stages of 128 to 640 bytes, a
# unit per chunk; then as many units per chunk as there are workers.
MANY_ROUNDS = [(20000, c, 4, 4, 4, 2, "f32", "f32") for c in (2, 4, 6, 8, 10)] + [
    (20000, 2, 8, 8, 8, 2, "f32", "f32"), (20000, 4, 8, 8, 8, 4, "bf16", "bf16"), (1024, 512, 2, 64, 8, 2, "f32", "f32")]


@pytest.mark.parametrize("flags", [0, PARKED], ids=["default", "pinned"])
@pytest.mark.parametrize("case", MANY_ROUNDS, ids=lambda c: "x".join(map(str, c)))
def test_many_rounds(case, flags):
    plan = same_bytes(case, flags)
    if flags and torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert plan.parked and case[0] * plan.chunks_per_sample > 64 * plan.grid


# the last one's planes are more than a chunk
@pytest.mark.parametrize("case", [(64, 64, 112, 112, 8, 2, "f32", "f32"), (128, 160, 32, 32, 4, 4, "bf16", "bf16"), (64, 24, 100, 112, 8, 2, "f32", "f32")], ids=lambda c: "x".join(map(str, c)))
def test_parking_kernel_by_default(case):
    plan = same_bytes(case, 0)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert plan.parked and plan.lag == 0 and plan.threads == 1024 and plan.grid == 148


def test_samples_that_do_not_fit_go_to_the_staged_kernel():
    plan = same_bytes((2, 64, 400, 400, 8, 2, "f32", "f32"), PARKED)          # 41 MB a sample, 38 MB of tensor memory
    assert plan.fused == 6 and plan.lag > 0 and not plan.parked


def test_a_nan_reaches_the_sample_as_it_does_in_the_two_pass_kernels():
    x = torch.randn((5, 64, 112, 112), device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    x[1, 7, 30, 50] = float("nan")
    codec = binding.Codec(5, 64, 112, 112, 8, 2, "f32", "f32")
    rebuilt = []
    for f in (PARKED, binding.DIV_FLAG_FORCE_TWO_PASS):
        codec.compress(x, seed=11, flags=f)
        rebuilt.append(codec.decompress().clone())
    assert codec.plan(PARKED).parked
    torch.testing.assert_close(rebuilt[0], rebuilt[1], rtol=0, atol=0, equal_nan=True)


def test_small_samples_go_where_they_are_faster():
    """Batches of samples of a chunk or two: those that were measured 10 % faster or more on one side run there."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the figures are those of 148 SMs")

    def parked(*a):
        return binding.div_plan_query(binding.make_desc(*a)).parked
    for others in ((3913, 2, 12, 68, 8, 4), (442, 4, 80, 80, 4, 2), (17746, 2, 13, 16, 4, 2), (9814, 12, 8, 8, 8, 2), (2140, 4, 60, 60, 8, 8),
                   (2273, 3, 16, 16, 8, 4, "bf16", "bf16")):
        assert not parked(*others), others
    for here in ((38306, 13, 8, 8, 8, 2, "f32", "bf16"), (18465, 2, 20, 20, 8, 4), (9395, 15, 7, 16, 8, 2), (24230, 2, 102, 8, 4, 2), (1, 818, 84, 84, 4, 2)):
        assert parked(*here), here


def test_the_flag_that_excludes_it_leaves_the_others_in_their_order():
    NO_PARK = binding.DIV_FLAG_NO_PARK_KERNEL
    for case in PARK + MANY_ROUNDS + [(64, 64, 112, 112, 8, 2, "f32", "f32"), (128, 160, 32, 32, 4, 4, "bf16", "bf16"), (8, 64, 1, 768, 8, 4), (3, 5, 7, 9, 4, 1)]:
        desc = binding.make_desc(*case)
        for flags in (0, PARKED, binding.DIV_FLAG_NO_STAGED_KERNEL, binding.DIV_FLAG_FORCE_TWO_PASS):
            with_it, without = binding.div_plan_query(desc, flags), binding.div_plan_query(desc, flags | NO_PARK)
            assert (without.fused, without.on_chip, without.parked) == (with_it.fused, with_it.on_chip, 0), case
            assert with_it.parked or all(getattr(with_it, f) == getattr(without, f) for f, _ in binding.DivPlan._fields_), case
    plan = same_bytes((128, 160, 32, 32, 4, 4, "bf16", "bf16"), NO_PARK)
    assert plan.on_chip == 1 and plan.threads in (256, 384, 512)


RING = binding.DIV_FLAG_NO_LAGGED_KERNEL | binding.DIV_FLAG_NO_STAGED_KERNEL


@pytest.mark.parametrize("flags", [PARKED, PARKED | binding.DIV_FLAG_NO_PARK_KERNEL, RING], ids=["parking", "staged", "strip ring"])
@pytest.mark.parametrize("shape", [(4, 64, 56, 56), (3, 64, 112, 112)], ids=lambda s: "x".join(map(str, s)))
def test_giving_up_at_once_leaves_nothing_behind(flags, shape):
    """A limit of 1 ns runs out while copies may still be on their way: they land before their CTAs leave, nothing behind the blob is
    written, and the calls after it, on the SMs that were left, write what they always do."""
    x = torch.randn(shape, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    codec = binding.Codec(*shape, 8, 2)
    size = codec.blob.numel()
    room = torch.full((size + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    codec.blob = room[:size]
    want = codec.compress(x, seed=5, flags=flags).clone()
    for _ in range(20):
        assert binding.lib().div_debug_compress_starved(
            ctypes.byref(codec.desc), ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(codec.blob.data_ptr()), size, ctypes.c_void_p(codec.workspace.data_ptr()),
            codec.workspace.numel(), 0, ctypes.c_void_p(binding.current_stream_handle()), flags, 1) == binding.DIV_OK
        assert codec.device_status() == binding.DIV_ERR_TIMEOUT
        codec.compress(x, seed=5, flags=flags)
        assert codec.device_status() == binding.DIV_OK and torch.equal(codec.blob, want)
    assert bool((room[size:] == 0xA5).all())
