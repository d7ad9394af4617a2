"""Calls that overlap: kernels start while the one before them on the stream still runs, on several streams and from several
threads at once, and inside a captured graph.  Every result is compared with that of the same call alone on an idle device."""
import threading

import pytest
import torch

from paper_2208_04187_b200 import binding, build

pytestmark = pytest.mark.gpu

LAGGED = binding.DIV_FLAG_NO_STRIP_KERNEL | binding.DIV_FLAG_NO_STAGED_KERNEL
RING = binding.DIV_FLAG_NO_LAGGED_KERNEL | binding.DIV_FLAG_NO_STAGED_KERNEL
PARKED = binding.DIV_FLAG_NO_STRIP_KERNEL | binding.DIV_FLAG_NO_LAGGED_KERNEL
STAGED = PARKED | binding.DIV_FLAG_NO_PARK_KERNEL
NO_STRIPS = STAGED | binding.DIV_FLAG_NO_STAGED_KERNEL
PAIR = binding.DIV_FLAG_TWO_LAUNCH_PLANES


@pytest.fixture(scope="module", autouse=True)
def built_library():
    build.build()
    binding.lib()


class Volume:
    """The 3-D calls with the codec's two methods."""

    def __init__(self, n, c, d, h, w, block, qbits):
        self.desc, self.shape = binding.make_desc_3d(n, c, d, h, w, block, qbits), (n, c, d, h, w)
        layout = binding.div_compressed_bytes_3d(self.desc)
        self.blob = torch.zeros(int(layout.total_bytes), dtype=torch.uint8, device="cuda")
        self.workspace = torch.zeros(int(layout.workspace_bytes), dtype=torch.uint8, device="cuda")
        self.x_dtype = "f32"

    def compress(self, x, seed=0, flags=0):
        binding.div_compress_3d(self.desc, x.data_ptr(), self.blob.data_ptr(), self.blob.numel(), self.workspace.data_ptr(),
                                self.workspace.numel(), seed, binding.current_stream_handle())
        return self.blob

    def decompress(self, out=None):
        out = torch.empty(self.shape, device="cuda") if out is None else out
        binding.div_decompress_3d(self.desc, self.blob.data_ptr(), self.blob.numel(), out.data_ptr(), binding.current_stream_handle())
        return out


# name: maker, flags, what the plan has to say (on_chip, fused) or None
KINDS = {
    "cluster": (lambda: binding.Codec(16, 128, 14, 14, 8, 2), 0, (1, None)),
    "cluster, several turns": (lambda: binding.Codec(40, 64, 75, 75, 8, 2, "f32", "bf16"), 0, (1, None)),
    "cluster, in place": (lambda: binding.Codec(16, 64, 32, 32, 8, 4, "bf16", "bf16"), 0, (1, None)),
    "parking": (lambda: binding.Codec(8, 64, 56, 56, 8, 2), PARKED, (0, 6)),
    "parking, before clusters": (lambda: binding.Codec(128, 160, 32, 32, 4, 4, "bf16", "bf16"), 0, (1, None)),
    "staged": (lambda: binding.Codec(8, 64, 56, 56, 8, 2), STAGED, (0, 6)),
    "lagged": (lambda: binding.Codec(8, 64, 56, 56, 8, 2), LAGGED, (0, 3)),
    "strip ring": (lambda: binding.Codec(8, 64, 56, 56, 8, 2), RING, (0, 2)),
    "planes": (lambda: binding.Codec(8, 64, 14, 14, 8, 2), NO_STRIPS, (0, 7)),
    "planes, two launches": (lambda: binding.Codec(8, 64, 14, 14, 8, 2), PAIR | NO_STRIPS, (0, 4)),
    "lines": (lambda: binding.Codec(8, 64, 1, 768, 8, 4), 0, (0, 8)),
    "lines, two launches": (lambda: binding.Codec(8, 64, 1, 768, 8, 4), PAIR, (0, 5)),
    "general ring": (lambda: binding.Codec(8, 16, 40, 40, 8, 1), 0, (0, 1)),
    "two passes": (lambda: binding.Codec(4, 16, 40, 40, 8, 2), binding.DIV_FLAG_FORCE_TWO_PASS, (0, 0)),
    "per plane, strips": (lambda: binding.PlaneGroupCodec(8, 32, 56, 56, 8, 2), 0, (0, 1)),
    "per plane, small": (lambda: binding.PlaneGroupCodec(8, 64, 14, 14, 8, 2), 0, (0, 2)),
    "per plane, share": (lambda: binding.PlaneGroupCodec(8, 16, 75, 75, 8, 2), 0, (1, 0)),
    "volume": (lambda: Volume(2, 8, 16, 28, 28, 8, 2), 0, None),
    "volume, odd": (lambda: Volume(2, 8, 5, 9, 11, 4, 2), 0, None),
}


def make(kind):
    maker, flags, want = KINDS[kind]
    codec = maker()
    if want is not None:
        plan = codec.plan(flags)
        assert plan.on_chip == want[0] and want[1] in (None, plan.fused), (plan.on_chip, plan.fused)
        assert plan.parked == kind.startswith("parking"), kind
    return codec, flags


def inputs(codec, count, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    return [torch.randn(codec.shape, device="cuda", generator=gen).to(binding.torch_dtype(codec.x_dtype)) for _ in range(count)]


def chain(codec, flags, x, steps=3):
    """compress, rebuild, compress what was rebuilt: every kernel reads what the one before it wrote."""
    kept = []
    for i in range(steps):
        codec.compress(x, seed=i, flags=flags)
        kept.append(codec.blob.clone())
        x = codec.decompress()
    return kept + [x]


def alone(codec, flags, x, steps=3):
    kept = []
    for i in range(steps):
        torch.cuda.synchronize()
        codec.compress(x, seed=i, flags=flags)
        torch.cuda.synchronize()
        kept.append(codec.blob.clone())
        x = codec.decompress()
        torch.cuda.synchronize()
    return kept + [x]


def same(got, want):
    return all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("kind", KINDS)
def test_calls_in_a_row_and_in_a_captured_graph(kind):
    codec, flags = make(kind)
    xs = inputs(codec, 3, 7)
    want = [alone(codec, flags, x) for x in xs]
    for x, w in zip(xs, want):
        assert same(chain(codec, flags, x), w)
    # captured once, replayed with other inputs, back to back
    held = torch.empty_like(xs[0])
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=stream):
        got = chain(codec, flags, held)
    copies = []
    for x in xs:
        held.copy_(x)
        graph.replay()
        copies.append([g.clone() for g in got])
    torch.cuda.synchronize()
    for c, w in zip(copies, want):
        assert same(c, w)


@pytest.mark.parametrize("kinds", [("cluster, several turns", "staged", "lines", "per plane, share"), ("strip ring", "planes", "cluster", "volume"),
                                   ("lagged", "cluster, in place", "general ring", "per plane, small"), ("staged", "staged", "cluster", "cluster"),
                                   ("parking", "parking", "staged", "cluster"), ("parking, before clusters", "parking", "lines", "volume")],
                         ids=lambda k: " + ".join(k))
def test_threads_on_streams_of_their_own(kinds):
    """Kernels whose CTAs wait for one another stay whole beside others of their sort."""
    work = []
    for i, kind in enumerate(kinds):
        codec, flags = make(kind)
        xs = inputs(codec, 2, 20 + i)
        work.append((codec, flags, xs, [alone(codec, flags, x) for x in xs]))
    torch.cuda.synchronize()
    wrong, start = [], threading.Barrier(len(work))

    def run(i):
        codec, flags, xs, want = work[i]
        try:
            stream = torch.cuda.Stream()
            start.wait(30)
            with torch.cuda.stream(stream):
                for _ in range(12):
                    for x, w in zip(xs, want):
                        got = chain(codec, flags, x)
                        stream.synchronize()
                        if not same(got, w):
                            wrong.append((kinds[i], "bytes"))
                if hasattr(codec, "device_status") and codec.device_status() != binding.DIV_OK:
                    wrong.append((kinds[i], "status"))
        except Exception as e:  # noqa: BLE001  (a thread's exception would be lost)
            wrong.append((kinds[i], repr(e)))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    assert not wrong, wrong


def test_one_workspace_for_kernels_in_turn():
    """Whatever an earlier kernel (or nobody) left in the scratch, every kernel's result is the same: the cluster kernel uses its
    status words alone and clears nothing else, the others clear it for themselves."""
    codec = binding.Codec(8, 64, 28, 28, 8, 2)
    x, = inputs(codec, 1, 3)
    order = [0, RING, LAGGED, 0, STAGED, PARKED, NO_STRIPS, 0, PARKED, PAIR | NO_STRIPS, binding.DIV_FLAG_FORCE_TWO_PASS, LAGGED, RING, PARKED, STAGED, 0]
    assert [codec.plan(f).on_chip for f in order] == [int(f == 0) for f in order]
    assert {codec.plan(f).fused for f in order if f} == {2, 3, 6, 7, 4, 0}
    codec.compress(x, seed=2)
    want = codec.blob.clone()
    for fill in (0xFF, 0x00, 0x5A):
        codec.workspace.fill_(fill)
        got = []
        for flags in order:
            codec.blob.fill_(0xEE)
            codec.compress(x, seed=2, flags=flags)
            got.append(codec.blob.clone())
        assert codec.device_status() == binding.DIV_OK
        lo = codec.layout
        for flags, g in zip(order, got):
            for at, size in ((lo.lfc_off, lo.lfc_bytes), (lo.packed_off, lo.packed_bytes), (lo.stats_off, lo.stats_bytes)):
                assert torch.equal(g[at:at + size], want[at:at + size]), flags
