// Launch shape of the cluster compress kernel (cluster.cu).
#pragma once

#include "fused.cuh"      // DeviceInfo, gcd_u32

namespace divk {

constexpr uint32_t CL_THREADS = 256;
constexpr uint32_t CL_WARPS = CL_THREADS / 32;
constexpr uint32_t CL_PIECES = 8;          // bulk copies a CTA's share arrives in
constexpr uint32_t CL_MAX = 16;            // CTAs of the largest cluster

struct ClusterPlan {
    uint32_t cs;              // CTAs per cluster (and per sample)
    uint32_t ppc;             // planes per CTA
    uint32_t ppp;             // planes per piece
    uint32_t res_bytes;       // fp32 residuals of a CTA's share (fp32 input lands in the same place)
    uint32_t smem_bytes;
    uint32_t vw;              // columns a lane can read at once: 4, 2 or 1
    uint32_t waves;           // times the device has to be filled
};

// shape of the launch for clusters of cs CTAs; false when a share does not fit
inline bool plan_cluster_cs(const div_desc* d, const Shape& s, uint32_t cs, const DeviceInfo& di, ClusterPlan* out) {
    const uint32_t sx = d->x_dtype == DIV_F32 ? 4u : 2u;
    if (!(d->qbits == 2 || d->qbits == 4 || d->qbits == 8)) return false;
    if (!(s.P2 == 4 || s.P2 == 8 || s.P2 == 16)) return false;
    if (((uint64_t)s.CHW * sx) % 16u != 0 || s.CHW >= (1u << 31)) return false;       // bulk copies: 16-byte boundaries
    if ((uint64_t)s.N * cs >= (1ull << 31)) return false;
    ClusterPlan pl;
    const uint32_t step = (16u / sx) / gcd_u32(16u / sx, s.HW);                       // planes that are whole 16-byte groups
    pl.cs = cs;
    const uint64_t ppc = ((uint64_t)(s.C + cs - 1) / cs + step - 1) / step * step;
    const uint64_t elems = ppc * s.HW;
    if (elems > (1u << 16)) return false;
    pl.ppc = (uint32_t)ppc;
    pl.ppp = (uint32_t)(((ppc + CL_PIECES - 1) / CL_PIECES + step - 1) / step * step);
    pl.res_bytes = (uint32_t)((elems * 4u + 16u + 127u) & ~127ull);                   // + 16: a slot may read up to 3 elements past a row
    pl.smem_bytes = pl.res_bytes + (sx == 2u ? (uint32_t)((elems * 2u + 16u + 127u) & ~127ull) : 0u);
    if (pl.smem_bytes + 1024u > (uint32_t)di.smem_optin) return false;
    pl.vw = (s.W % 4 == 0 && s.B % 4 == 0) ? 4u : (s.W % 2 == 0 && s.B % 2 == 0) ? 2u : 1u;
    // resident CTAs: shared memory, and registers (64 a thread where rows are read 4 columns at a time, else up to 80);
    // clusters of a few CTAs leave 5 % of the places empty
    uint32_t per_sm = (uint32_t)di.smem_optin / (pl.smem_bytes + 2048u);
    const uint32_t by_regs = pl.vw == 4u ? 4u : 3u;
    if (per_sm > by_regs) per_sm = by_regs;
    if (per_sm < 1u) per_sm = 1u;
    const uint64_t places = (uint64_t)per_sm * (uint32_t)di.sms * 95u / 100u;
    pl.waves = (uint32_t)(((uint64_t)s.N * cs + places - 1) / (places ? places : 1u));
    *out = pl;
    return true;
}

// `expect_bytes`: what a CTA waits to receive (0: what its cluster sends; a test may ask for more than ever arrives)
div_status compress_cluster(const div_desc* d, const Shape& s, const div_layout& lo, const ClusterPlan& pl, const void* x, uint8_t* blob,
                            uint32_t* ws, uint64_t seed, cudaStream_t st, uint32_t expect_bytes = 0, uint64_t timeout_ns = 0);

}  // namespace divk
