"""Host side of the launches, compiled against a stand-in for the CUDA runtime: no GPU needed."""
import subprocess

import pytest

from paper_2208_04187_b200 import build

SMEM_LIMIT = r"""
#include <cuda_runtime.h>
#include <cstdio>
static int limit = 48 * 1024, sets = 0;
static void (*meanwhile)() = nullptr;            // what another thread does between a call's runtime call and its note of it
static cudaError_t fake_device(int* d) { *d = 0; return cudaSuccess; }
static cudaError_t fake_attribute(int* v, cudaDeviceAttr a, int) { *v = a == cudaDevAttrMultiProcessorCount ? 148 : 232448; return cudaSuccess; }
static cudaError_t fake_attributes(cudaFuncAttributes* a, const void*) { *a = cudaFuncAttributes(); a->sharedSizeBytes = 1000; return cudaSuccess; }
static cudaError_t fake_set(const void*, cudaFuncAttribute, int v) {
    if (v > 232448 - 1000) return cudaErrorInvalidValue;
    limit = v;
    ++sets;
    if (auto f = meanwhile) { meanwhile = nullptr; f(); }
    return cudaSuccess;
}
#define cudaGetDevice fake_device
#define cudaDeviceGetAttribute fake_attribute
#define cudaFuncGetAttributes fake_attributes
#define cudaFuncSetAttribute fake_set
#include "fused.cuh"
static divk::SmemSeen seen[divk::DEVICE_CACHE_SLOTS];
static int kernel;
static bool ask(int bytes) { return divk::ensure_dynamic_smem(&kernel, bytes, seen) && bytes <= limit; }
int main() {
    meanwhile = [] { ask(60 * 1024); };
    const bool first = divk::ensure_dynamic_smem(&kernel, 200 * 1024, seen);
    const bool large = ask(200 * 1024), small = ask(60 * 1024), again = ask(200 * 1024);
    const int before = sets;
    const bool too_large = ask(232448 - 999), most = ask(232448 - 1000);
    printf("%d %d %d %d %d %d %d", first, large, small, again, too_large, most, sets - before);
}
"""


def compiled(source, folder):
    src = folder / "t.cu"
    src.write_text(source)
    exe = str(folder / "t")
    subprocess.run([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I" + build.CSRC, str(src), "-o", exe], check=True,
                   capture_output=True, text=True, timeout=600)
    return exe


def test_threads_with_different_sizes_cannot_lower_a_kernel_s_limit(tmp_path):
    """One thread asks for 200 KB, and while it does another asks for 60 KB: both sizes stay launchable, without setting
    anything again; the device's limit less the kernel's static share is granted, a byte more is refused."""
    got = subprocess.run([compiled(SMEM_LIMIT, tmp_path)], check=True, capture_output=True, text=True, timeout=60).stdout
    assert got.split() == ["1", "1", "1", "1", "0", "1", "0"]


PARK_PLAN = r"""
#include <cuda_runtime.h>
#include <cstdio>
static cudaError_t fake_device(int* d) { *d = 0; return cudaSuccess; }
static cudaError_t fake_attribute(int* v, cudaDeviceAttr a, int) { *v = a == cudaDevAttrMultiProcessorCount ? 148 : 232448; return cudaSuccess; }
#define cudaGetDevice fake_device
#define cudaDeviceGetAttribute fake_attribute
#include "park_plan.cuh"
using namespace divk;
int main() {                                     // descriptors in, ahead, stages, records and rounds out (zeros: not taken)
    int n, c, h, w, block, bf16;
    while (scanf("%d %d %d %d %d %d", &n, &c, &h, &w, &block, &bf16) == 6) {
        div_desc d = {n, c, h, w, block, 2, bf16 ? DIV_BF16 : DIV_F32, DIV_F32};
        Shape s = Shape();
        s.N = n; s.C = c; s.H = h; s.W = w; s.B = s.P2 = block;
        s.Hb = (h + block - 1) / block; s.Wb = (w + block - 1) / block;
        s.HW = h * w; s.CHW = c * s.HW; s.TPP = s.Hb * s.Wb; s.total = (uint64_t)n * s.CHW;
        ParkPlan pl = ParkPlan();
        const bool taken = plan_park(&d, s, &pl);
        printf("%u %u %u %u\n", taken ? pl.ahead : 0u, taken ? pl.stages : 0u, PARK_CHUNKS, taken ? (pl.total_chunks + pl.grid - 1u) / pl.grid : 0u);
    }
}
"""


@pytest.fixture(scope="module")
def park_planner(tmp_path_factory):
    exe = compiled(PARK_PLAN, tmp_path_factory.mktemp("park"))
    return lambda descs: [tuple(map(int, line.split())) for line in subprocess.run(
        [exe], input="\n".join(" ".join(map(str, d)) for d in descs), check=True, capture_output=True, text=True, timeout=60).stdout.splitlines()]


def test_the_producer_of_the_parking_kernel_never_waits_for_a_fill_that_only_it_could_start(park_planner):
    """Its wait for the chunk `ahead` before the next one names a record and a parity: with every copy landed that it has asked
    for, the record has to be past that parity, over many rounds of samples of 32 to 32768 bytes."""
    descs = [(n, c, h, w, block, bf16) for n in (148 * 3, 148 * 70, 148 * 140, 148 * 300) for c in (1, 2, 3, 4, 6, 8, 10, 12, 24, 32) for h, w in
             ((1, 8), (2, 8), (4, 4), (8, 8), (1, 72), (12, 12), (16, 16)) for block in (4, 8) for bf16 in (0, 1) if max(h, w) >= block]
    taken = 0
    for desc, (ahead, stages, records, rounds) in zip(descs, park_planner(descs)):
        if not ahead:
            continue
        taken += 1
        assert 2 <= ahead <= stages, desc
        fills = [0] * records                                   # of each record, all landed
        for it in range(rounds):
            if it >= ahead:
                chunk = it - ahead
                assert (fills[chunk % records] & 1) != ((chunk // records) & 1), (desc, it)
            fills[it % records] += 1
    assert taken > 200
