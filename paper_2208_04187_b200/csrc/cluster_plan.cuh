// Launch shapes of the kernels whose CTAs keep a share of a sample in shared memory (cluster.cu, planeshare.cu).
#pragma once

#include "fused.cuh"      // DeviceInfo, gcd_u32

namespace divk {

constexpr uint32_t SHARE_THREADS = 256;
constexpr uint32_t SHARE_WARPS = SHARE_THREADS / 32;
// threads where at most two CTAs fit an SM and clusters take turns (32 x 64 x 75 x 75 28.6 -> 27.0 us, 64 x 1024 x 14 x 14
// 23.6 -> 23.0 us; where all of x fits at once more threads cost a little, 64 x 2048 x 7 x 7 11.5 -> 12.1 us), and where a CTA has
// an SM to itself (1 x 64 x 112 x 112 10.8 -> 9.7 us, 1 x 128 x 56 x 56 7.4 -> 6.4 us): 64 registers a thread suffice where rows are
// read 4 columns at a time or have 4 rows
__host__ __device__ constexpr uint32_t share_wide_threads(uint32_t p2, uint32_t vw) { return vw == 4 || p2 == 4 ? 512u : 384u; }
// resident CTAs per SM that the registers allow: up to 80 a thread, 64 (48) where they suffice (128 x 64 x 32 x 32: three of
// 78 registers 14.5 us, four of 64 12.8 us)
__host__ __device__ constexpr uint32_t share_by_regs(uint32_t p2, uint32_t vw, uint32_t sx) { return vw == 4 && p2 == 4 && sx == 2 ? 5u : vw == 4 || p2 == 4 ? 4u : 3u; }
// bfloat16 read 4 columns at a time: x stays as it is and half 2 forms the residual again, which would take twice its room
// (128 x 160 x 32 x 32 with B = 4, 42 MB: 126 MB of landing place and residuals 36 us, 47 MB 29.8 us)
__host__ __device__ constexpr bool share_in_place(uint32_t vw, uint32_t sx) { return sx == 2 && vw == 4; }
constexpr uint32_t SHARE_PIECES = 8;       // bulk copies a CTA's share arrives in
constexpr uint32_t CL_MAX = 16;            // CTAs of the largest cluster

// a CTA's share of a sample: a run of whole planes in shared memory
struct SharePlan {
    uint32_t ppc;             // planes per CTA
    uint32_t ppp;             // planes per piece
    uint32_t res_bytes;       // fp32 residuals of a CTA's share (fp32 input lands in the same place), or its tiles' stored values
    uint32_t smem_bytes;
    uint32_t vw;              // columns a lane can read at once: 4, 2 or 1
};
struct ClusterPlan : SharePlan {
    uint32_t cs;              // CTAs per cluster (and per sample)
    uint32_t wide;            // 1: share_wide_threads a CTA, else SHARE_THREADS
    uint32_t turns64;         // 64ths of the times that the device has to be filled: whole times up to two, and where an SM holds one
                              // CTA (the clusters of a turn then end together); beyond that what the clusters make up
    uint32_t per_sm;          // CTAs that fit an SM
    uint32_t load;            // CTAs at once on the busiest SM
};

inline uint32_t cluster_threads(uint32_t p2, const ClusterPlan& pl) { return pl.wide ? share_wide_threads(p2, pl.vw) : SHARE_THREADS; }

// Clusters of 2^log2cs CTAs that the device holds at once where `per_sm` such CTAs fit an SM (a cluster stays within a group of
// SMs, so that some places stay empty: with one CTA per SM 7 clusters of 16, 112 of 148 places; two, 33 of 8, 264 of 296).
// Asked of the driver once per device and form; 0 where it has none.
uint32_t clusters_at_once(const DeviceInfo& di, uint32_t log2cs, uint32_t per_sm);

// planes that are whole groups of 4 elements and 16-byte groups (bulk copies)
inline uint32_t share_step(const div_desc* d, const Shape& s) {
    const uint32_t sx = d->x_dtype == DIV_F32 ? 4u : 2u;
    return (16u / sx) / gcd_u32(16u / sx, s.HW);
}
inline bool share_takes(const div_desc* d, const Shape& s) {
    const uint32_t sx = d->x_dtype == DIV_F32 ? 4u : 2u;
    return (d->qbits == 2 || d->qbits == 4 || d->qbits == 8) && (s.P2 == 4 || s.P2 == 8 || s.P2 == 16) &&
           ((uint64_t)s.CHW * sx) % 16u == 0 && s.CHW < (1u << 31);
}
// a share of `ppc` planes (a multiple of share_step); false when it does not fit
inline bool plan_share(const div_desc* d, const Shape& s, uint64_t ppc, uint32_t extra_smem, bool in_place, const DeviceInfo& di, SharePlan* out) {
    const uint32_t sx = d->x_dtype == DIV_F32 ? 4u : 2u, step = share_step(d, s);
    const uint64_t elems = ppc * s.HW;
    if (elems > (1u << 16)) return false;
    out->ppc = (uint32_t)ppc;
    out->ppp = (uint32_t)(((ppc + SHARE_PIECES - 1) / SHARE_PIECES + step - 1) / step * step);
    out->vw = (s.W % 4 == 0 && s.B % 4 == 0 && s.P2 < 16) ? 4u : (s.W % 2 == 0 && s.B % 2 == 0) ? 2u : 1u;
    // + 16: a slot may read up to 3 elements past a row
    const uint32_t res = (uint32_t)((elems * 4u + 16u + 127u) & ~127ull), land = (uint32_t)((elems * sx + 16u + 127u) & ~127ull);
    out->res_bytes = in_place && share_in_place(out->vw, sx) ? (uint32_t)((ppc * s.TPP * 4u + 127u) & ~127ull) : res;
    out->smem_bytes = out->res_bytes + (sx == 2u ? land : 0u) + extra_smem;
    return out->smem_bytes + 1024u <= (uint32_t)di.smem_optin;
}
// resident CTAs per SM: shared memory, and registers
inline uint32_t share_per_sm(const SharePlan& pl, const DeviceInfo& di, uint32_t by_regs) {
    const uint32_t by_smem = (uint32_t)di.smem_optin / (pl.smem_bytes + 2048u);
    return by_smem < 1u ? 1u : by_smem < by_regs ? by_smem : by_regs;
}

// shape of the launch for clusters of cs CTAs; false when a share does not fit
inline bool plan_cluster_cs(const div_desc* d, const Shape& s, uint32_t log2cs, const DeviceInfo& di, ClusterPlan* out) {
    const uint32_t cs = 1u << log2cs;
    if (!share_takes(d, s) || (uint64_t)s.N * cs >= (1ull << 31)) return false;
    ClusterPlan pl;
    const uint32_t step = share_step(d, s);
    pl.cs = cs;
    if (!plan_share(d, s, ((uint64_t)(s.C + cs - 1) / cs + step - 1) / step * step, 0u, true, di, &pl)) return false;
    const uint32_t per_sm = share_per_sm(pl, di, share_by_regs(s.P2, pl.vw, d->x_dtype == DIV_F32 ? 4u : 2u));
    const uint32_t at_once = clusters_at_once(di, log2cs, per_sm);
    if (at_once == 0u) return false;
    const uint64_t turns64 = per_sm == 1u || s.N <= 2u * at_once ? 64ull * ((s.N + at_once - 1u) / at_once) : 64ull * s.N / at_once;
    if (turns64 >= (1ull << 31)) return false;
    const uint32_t spread = (uint32_t)(((uint64_t)s.N * cs + (uint32_t)di.sms - 1u) / (uint32_t)di.sms);
    pl.turns64 = (uint32_t)turns64;
    pl.per_sm = per_sm;
    pl.load = per_sm < spread ? per_sm : spread;
    pl.wide = per_sm <= 2u && (pl.turns64 > 64u || spread == 1u) ? 1u : 0u;
    *out = pl;
    return true;
}

// What a test may ask of a call beyond the ordinary (zeros: nothing).
struct ShareFault {
    uint32_t expect_bytes;    // what a CTA waits to receive, more than ever arrives, instead of what its cluster sends
    uint32_t no_copies;       // the waits for x never end
    uint32_t more_smem;       // shared memory that the launch asks for beyond what it needs
    uint32_t number;          // the call's number (see share_record)
    uint32_t timeout_ns;      // limit of every wait
    uint32_t no_park;         // more_smem is for the parking kernel's launch, and nothing is asked of the kernels behind it
};
div_status compress_cluster(const div_desc* d, const Shape& s, const div_layout& lo, const ClusterPlan& pl, const void* x, uint8_t* blob,
                            uint32_t* ws, uint64_t seed, cudaStream_t st, const ShareFault& fault = ShareFault());

// per-plane groups (planeshare.cu)
bool plan_plane_share(const div_desc* d, const Shape& s, SharePlan* out);
div_status compress_plane_share(const div_desc* d, const Shape& s, const div_layout& lo, const SharePlan& pl, const void* x, uint8_t* blob,
                                uint64_t seed, cudaStream_t st, const ShareFault& fault = ShareFault());

}  // namespace divk
