"""Host side of the launches, compiled against a stand-in for the CUDA runtime: no GPU needed."""
import subprocess

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


def test_threads_with_different_sizes_cannot_lower_a_kernel_s_limit(tmp_path):
    """One thread asks for 200 KB, and while it does another asks for 60 KB: both sizes stay launchable, without setting
    anything again; the device's limit less the kernel's static share is granted, a byte more is refused."""
    src = tmp_path / "t.cu"
    src.write_text(SMEM_LIMIT)
    exe = str(tmp_path / "t")
    subprocess.run([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I" + build.CSRC, str(src), "-o", exe], check=True,
                   capture_output=True, text=True, timeout=600)
    got = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout
    assert got.split() == ["1", "1", "1", "1", "0", "1", "0"]
