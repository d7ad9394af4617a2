// Cluster compress kernel (DIVISION Sec. 4.1; Algorithm 1, forward loop): a thread-block cluster takes one sample,
// which waits in shared memory between the two halves of the work (halves.cuh).
//
// What bounds it: HBM (x is read once and the blob written once) on large maps, instruction issue close behind,
// launch and load latency on small ones.  Why this form:
//   * every CTA of the cluster owns a run of whole planes and brings them into shared memory with a few bulk copies
//     that are all issued at once, so that no warp waits for a global load after its piece has landed;
//   * half 1 works on (tile, columns) slots of any width; it leaves the fp32 RESIDUAL where x was, so that half 2 is
//     a flat pass over groups of 4 consecutive elements: one 16-byte load, Eq. 9, one store, whatever the width of the
//     planes (tables of tile positions cost a third of the instructions of the kernel that re-reads x);
//   * the sample's extremes meet in distributed shared memory: every CTA sends one 8-byte word to each CTA of the
//     cluster, counted by an mbarrier there.  No scratch memory, hence nothing to clear before the launch, and no
//     grid-wide co-residency: clusters that do not fit at once run one after the other.
// Waits are bounded.  A warp whose wait runs out records DIV_ERR_TIMEOUT in the workspace status word; if it waited for x its
// CTA quantises nothing.  The CTA's word is sent all the same (nobody else has to wait for its limit), and no CTA
// leaves before what is on its way to it has come or SHARE_DRAIN_NS have passed.
#include <chrono>

#include "cluster_plan.cuh"
#include "halves.cuh"

namespace divk {

struct ClusterParams : ShareParams {
    float* stats;
    uint32_t log2cs, expect_bytes;
    int32_t qbits;
};
static_assert(sizeof(ClusterParams) <= SHARE_PARAM_BYTES, "dearer launches");

// ------------------------------------------------------------------------------------------------
// cluster and distributed shared memory
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// (relaxed: the only thing it orders is the set-up of the mbarriers, which fence_barrier_init has released; with .release
// every thread waits for its stores of low-frequency values, 20 % of the stalls of the kernel)
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// 8 bytes into CTA `rank`'s copy of *dst, counted on its copy of *bar
__device__ __forceinline__ void st_async_u64(uint64_t* dst, uint64_t v, uint64_t* bar, uint32_t rank) {
    uint32_t d, b;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(smem_u32(dst)), "r"(rank));
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(smem_u32(bar)), "r"(rank));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(d), "l"(v), "r"(b) : "memory");
}

// a word that another CTA of the cluster sent is read behind this wait: acquire for the cluster (the plain form acquires for
// the CTA alone)
struct ClusterScope {
    static __device__ __forceinline__ bool try_wait(uint64_t* bar) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar))
            : "memory");
        return ok != 0;
    }
};

// ------------------------------------------------------------------------------------------------
// half 2: the CTA's residuals, 4 consecutive elements per thread and step
// ------------------------------------------------------------------------------------------------
template <int Q, bool FIXED, uint32_t THREADS>
__device__ __forceinline__ void cl_half2(const float* res, typename PackedUnit<Q>::type* out, uint32_t nq, uint64_t ctr, float delta,
                                         float scale) {
    typedef typename PackedUnit<Q>::type OutT;
    const uint64_t delta2 = pk2(delta, delta);
    const float m = FIXED ? -65536.0f * scale : scale;
    const uint64_t mul2 = pk2(m, m);
    constexpr int U = 4;
    constexpr uint64_t STEP = K_GROUP * (uint64_t)THREADS;
    uint32_t q = threadIdx.x;
    for (; q + (U - 1) * THREADS < nq; q += U * THREADS) {
        ulonglong2 v[U];
#pragma unroll
        for (int k = 0; k < U; ++k) v[k] = reinterpret_cast<const ulonglong2*>(res)[q + k * THREADS];
#pragma unroll
        for (int k = 0; k < U; ++k)
            out[q + k * THREADS] = (OutT)quant4_res<Q, FIXED>(v[k].x, v[k].y, delta2, mul2, rng_mix(ctr + STEP * (uint64_t)k));
        ctr += STEP * U;
    }
    for (; q < nq; q += THREADS) {
        const ulonglong2 v = reinterpret_cast<const ulonglong2*>(res)[q];
        out[q] = (OutT)quant4_res<Q, FIXED>(v.x, v.y, delta2, mul2, rng_mix(ctr));
        ctr += STEP;
    }
}
// The same where x stayed in place (bfloat16, rows read 4 columns at a time): slot by slot as in half 1, the residual formed
// once more from x and the tile's stored low-frequency value.
template <typename XT, int P2, typename G, int Q, bool FIXED, uint32_t THREADS>
__device__ __forceinline__ void cl_half2_slots(const ShareParams& p, const float* stored_of, const XT* land,
                                               typename PackedUnit<Q>::type* out, uint32_t nplanes, uint64_t ctr0, float delta, float scale) {
    typedef typename PackedUnit<Q>::type OutT;
    const uint64_t delta2 = pk2(delta, delta);
    const float m = FIXED ? -65536.0f * scale : scale;
    const uint64_t mul2 = pk2(m, m);
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31, W4 = p.W >> 2;
    const uint32_t nfull = nplanes * p.sppf, first_short = (nfull + 31u) & ~31u, total = first_short + nplanes * p.sppt;
    const uint64_t row_step = K_GROUP * (uint64_t)W4;
    for (uint32_t first = warp * 32u; first < total; first += THREADS) {
        const ShareSlot t = share_slot<P2, G::NC>(p, first, lane, nfull, first_short, total);
        if (t.cols == 0u) continue;
        const float stored = stored_of[t.tile];
        const uint64_t stored2 = pk2(stored, stored);
        const unsigned char* xs = reinterpret_cast<const unsigned char*>(land + t.off);
        const uint32_t row_bytes = p.W * (uint32_t)sizeof(XT);
        OutT* o = out + (t.off >> 2);
        uint64_t ctr = ctr0 + K_GROUP * (uint64_t)(t.off >> 2);
        if (t.rows == (uint32_t)P2) {
            uint64_t xy[P2], zw[P2];
#pragma unroll
            for (int r = 0; r < P2; ++r) StripRow2<XT>::load(xs + r * row_bytes, xy[r], zw[r]);
#pragma unroll
            for (int r = 0; r < P2; ++r) {
                o[r * W4] = (OutT)quant4_res<Q, FIXED>(sub2_rn(xy[r], stored2), sub2_rn(zw[r], stored2), delta2, mul2, rng_mix(ctr));
                ctr += row_step;
            }
        } else {
            for (uint32_t r = 0; r < t.rows; ++r) {
                uint64_t xy, zw;
                StripRow2<XT>::load(xs + r * row_bytes, xy, zw);
                o[r * W4] = (OutT)quant4_res<Q, FIXED>(sub2_rn(xy, stored2), sub2_rn(zw, stored2), delta2, mul2, rng_mix(ctr));
                ctr += row_step;
            }
        }
    }
}
template <typename XT, int P2, typename G, int Q, bool IN_PLACE, uint32_t THREADS>
__device__ __forceinline__ void cl_half2_q(const ClusterParams& p, const float* res, const XT* land, uint32_t n, uint32_t qfirst,
                                           uint32_t nplanes, float rmin, float rmax, bool write_stats) {
    const QParams qp = make_qparams(rmin, rmax, Q);
    if (write_stats) {
        p.stats[2 * (size_t)n + 0] = qp.delta;
        p.stats[2 * (size_t)n + 1] = qp.step;
    }
    typename PackedUnit<Q>::type* out = reinterpret_cast<typename PackedUnit<Q>::type*>(p.packed) + ((uint64_t)n * p.qps + qfirst);
    if constexpr (IN_PLACE) {
        const uint64_t ctr = rng_sample_base(p.seed, n) + K_GROUP * (uint64_t)(qfirst + 1u);
        if (Q <= 4 && fixed_point_ok<Q>(qp, rmax)) cl_half2_slots<XT, P2, G, Q, true, THREADS>(p, res, land, out, nplanes, ctr, qp.delta, qp.scale);
        else cl_half2_slots<XT, P2, G, Q, false, THREADS>(p, res, land, out, nplanes, ctr, qp.delta, qp.scale);
    } else {
        const uint32_t nq = (nplanes * p.HW) >> 2;
        const uint64_t ctr = rng_sample_base(p.seed, n) + K_GROUP * (uint64_t)(qfirst + threadIdx.x + 1u);
        if (Q <= 4 && fixed_point_ok<Q>(qp, rmax)) cl_half2<Q, true, THREADS>(res, out, nq, ctr, qp.delta, qp.scale);
        else cl_half2<Q, false, THREADS>(res, out, nq, ctr, qp.delta, qp.scale);
    }
}

template <typename XT, int P2, typename G, uint32_t THREADS>
__global__ void __launch_bounds__(THREADS, THREADS > SHARE_THREADS ? 2 : share_by_regs(P2, G::VW, sizeof(XT)))
cluster_kernel(const __grid_constant__ ClusterParams p) {
    constexpr bool IN_PLACE = share_in_place(G::VW, sizeof(XT));
    extern __shared__ __align__(128) unsigned char smem[];
    float* res = reinterpret_cast<float*>(smem);
    const XT* land = reinterpret_cast<const XT*>(sizeof(XT) == 4 ? smem : smem + p.res_bytes);
    __shared__ __align__(8) uint64_t full[SHARE_PIECES];
    __shared__ __align__(8) uint64_t xbar;
    __shared__ __align__(8) uint64_t xch[CL_MAX];
    __shared__ uint32_t wkey[2][THREADS / 32];
    __shared__ uint32_t gave_up;              // a warp's wait for a piece ran out
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_ctarank(), n = blockIdx.x >> p.log2cs;
    const uint32_t plane0 = rank * p.ppc;
    const uint32_t nplanes = plane0 < p.C ? min(p.ppc, p.C - plane0) : 0u;
    if (tid == 0) {
#pragma unroll
        for (uint32_t i = 0; i < SHARE_PIECES; ++i) mbar_init(&full[i], p.arrivals);
        mbar_init(&xbar, 1);
        gave_up = 0u;
        fence_barrier_init();
        mbar_arrive_expect_tx(&xbar, p.expect_bytes);
        griddep_wait();
        share_load(p, const_cast<XT*>(land), full, n, plane0, nplanes);
    }
    __syncthreads();
    griddep_wait();
    griddep_launch();
    cluster_arrive();                          // waited for below, before anything is sent to another CTA

    float lo = 3.402823466e+38f, hi = -3.402823466e+38f;
    if (nplanes) share_half1<XT, P2, G, false, IN_PLACE, THREADS>(p, res, land, full, n, plane0, nplanes, nullptr, &gave_up, lo, hi);
    {
        const uint32_t kmin = __reduce_max_sync(0xFFFFFFFFu, ~float_key(lo));
        const uint32_t kmax = __reduce_max_sync(0xFFFFFFFFu, float_key(hi));
        if (lane == 0) {
            wkey[0][warp] = kmin;
            wkey[1][warp] = kmax;
        }
    }
    __syncthreads();                           // also: every residual is in place
    cluster_wait();
    if (warp == 0) {
        const uint32_t kmin = __reduce_max_sync(0xFFFFFFFFu, lane < THREADS / 32 ? wkey[0][lane] : 0u);
        const uint32_t kmax = __reduce_max_sync(0xFFFFFFFFu, lane < THREADS / 32 ? wkey[1][lane] : 0u);
        if (lane < (1u << p.log2cs)) st_async_u64(&xch[rank], ((uint64_t)kmax << 32) | kmin, &xbar, lane);
    }
    // (read here, where the trip to memory passes beside the wait: at the start of the kernel it costs small maps 0.1 to 0.2 us)
    uint64_t status = 0ull;
    if (blockIdx.x == 0 && tid == THREADS - 1) status = ld_relaxed_u64(p.status);
    const bool all_came = __all_sync(0xFFFFFFFFu, share_wait<ClusterScope>(&xbar, p.timeout_ns));
    if (status != 0ull) share_clear_status(p, status);
    if (!all_came || gave_up) {                // gave_up: the same in the whole CTA, written before the barrier above
        if (lane == 0) share_record(p);
        if (!all_came) share_wait<ClusterScope>(&xbar, SHARE_DRAIN_NS);
        if (warp == 0 && gave_up) share_drain(p, full, nplanes);
        return;
    }
    const uint64_t w = lane < (1u << p.log2cs) ? xch[lane] : 0ull;
    const float rmin = key_float(~__reduce_max_sync(0xFFFFFFFFu, (uint32_t)w));
    const float rmax = key_float(__reduce_max_sync(0xFFFFFFFFu, (uint32_t)(w >> 32)));
    if (nplanes == 0) return;
    const uint32_t qfirst = (plane0 * p.HW) >> 2;
    const bool stats = rank == 0 && tid == 0;
    if (p.qbits == 2) cl_half2_q<XT, P2, G, 2, IN_PLACE, THREADS>(p, res, land, n, qfirst, nplanes, rmin, rmax, stats);
    else if (p.qbits == 4) cl_half2_q<XT, P2, G, 4, IN_PLACE, THREADS>(p, res, land, n, qfirst, nplanes, rmin, rmax, stats);
    else cl_half2_q<XT, P2, G, 8, IN_PLACE, THREADS>(p, res, land, n, qfirst, nplanes, rmin, rmax, stats);
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
template <typename XT, int P2, typename G, uint32_t THREADS>
inline div_status launch_cluster_t(const ClusterParams& prm, const ClusterPlan& pl, uint32_t N, cudaStream_t st) {
    auto kern = cluster_kernel<XT, P2, G, THREADS>;
    static SmemSeen smem_set[DEVICE_CACHE_SLOTS], wide_set[DEVICE_CACHE_SLOTS];
    if (!ensure_dynamic_smem((const void*)kern, (int)pl.smem_bytes, smem_set)) return DIV_ERR_CUDA;
    if (pl.cs > 8 && !ensure_wide_cluster((const void*)kern, wide_set)) return DIV_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(N * pl.cs);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = pl.smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = pl.cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    if (cudaLaunchKernelEx(&cfg, kern, prm) != cudaSuccess) {
        cudaGetLastError();
        return DIV_ERR_CUDA;
    }
    return DIV_OK;
}
template <typename XT, int P2, typename G>
inline div_status launch_cluster(const ClusterParams& prm, const ClusterPlan& pl, uint32_t N, cudaStream_t st) {
    // as many threads as the registers allow where only two shares fit an SM
    if (pl.wide) return launch_cluster_t<XT, P2, G, share_wide_threads(P2, G::VW)>(prm, pl, N, st);
    return launch_cluster_t<XT, P2, G, SHARE_THREADS>(prm, pl, N, st);
}
template <typename XT, int P2>
inline div_status launch_cluster_geo(const ClusterParams& prm, const ClusterPlan& pl, uint32_t N, cudaStream_t st) {
    constexpr int NC = P2 == 16 ? 2 : 4;
    if constexpr (NC == 4) {
        if (pl.vw == 4) return launch_cluster<XT, P2, SlotGeo<4, 4>>(prm, pl, N, st);
    }
    return pl.vw >= 2 ? launch_cluster<XT, P2, SlotGeo<NC, 2>>(prm, pl, N, st) : launch_cluster<XT, P2, SlotGeo<NC, 1>>(prm, pl, N, st);
}
template <typename XT>
inline div_status launch_cluster_p2(const ClusterParams& prm, const ClusterPlan& pl, const Shape& s, cudaStream_t st) {
    switch (s.P2) {
        case 4: return launch_cluster_geo<XT, 4>(prm, pl, s.N, st);
        case 8: return launch_cluster_geo<XT, 8>(prm, pl, s.N, st);
        case 16: return launch_cluster_geo<XT, 16>(prm, pl, s.N, st);
    }
    return DIV_ERR_PARAM;
}

static __global__ void place_kernel() {}                       // stands for any kernel in clusters_at_once

uint32_t clusters_at_once(const DeviceInfo& di, uint32_t log2cs, uint32_t per_sm) {
    constexpr uint32_t FORMS = 5, MOST = 8;
    static std::atomic<int> known[DEVICE_CACHE_SLOTS][FORMS][MOST];      // the answer + 1
    if (log2cs >= FORMS || per_sm < 1u || per_sm > MOST) return 0u;
    const bool slot = di.dev >= 0 && di.dev < DEVICE_CACHE_SLOTS;
    if (slot) {
        const int got = known[di.dev][log2cs][per_sm - 1u].load(std::memory_order_relaxed);
        if (got > 0) return (uint32_t)got - 1u;
    }
    static SmemSeen smem_set[DEVICE_CACHE_SLOTS], wide_set[DEVICE_CACHE_SLOTS];
    const int smem = di.smem_optin / (int)per_sm - 2048;                  // per_sm such CTAs fit an SM, one more does not
    if (!ensure_dynamic_smem((const void*)place_kernel, smem, smem_set) || !ensure_wide_cluster((const void*)place_kernel, wide_set)) return 0u;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1u << log2cs);
    cfg.blockDim = dim3(SHARE_THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1u << log2cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, (const void*)place_kernel, &cfg) != cudaSuccess || n < 0) {
        cudaGetLastError();
        return 0u;
    }
    if (slot) known[di.dev][log2cs][per_sm - 1u].store(n + 1, std::memory_order_relaxed);
    return (uint32_t)n;
}

// a number that the failed call before on this workspace is not likely to have had: the low bits of a clock
static inline uint32_t call_number() {
#if defined(__x86_64__)
    return (uint32_t)__builtin_ia32_rdtsc();                   // (no call into the system)
#else
    return (uint32_t)std::chrono::steady_clock::now().time_since_epoch().count();
#endif
}

div_status compress_cluster(const div_desc* d, const Shape& s, const div_layout& lo, const ClusterPlan& plan, const void* x, uint8_t* blob,
                            uint32_t* ws, uint64_t seed, cudaStream_t st, const ShareFault& fault) {
    ClusterPlan pl = plan;
    pl.smem_bytes += fault.more_smem;
    ClusterParams p;
    p.x = x;
    p.lfc = blob + lo.lfc_off;
    p.packed = blob + lo.packed_off;
    p.stats = reinterpret_cast<float*>(blob + lo.stats_off);
    p.status = reinterpret_cast<uint64_t*>(ws);
    p.number = fault.number ? fault.number : call_number();
    p.seed = seed;
    p.arrivals = fault.no_copies ? 2u : 1u;
    p.timeout_ns = fault.timeout_ns ? fault.timeout_ns : 2000000000u;
    fill_share(&p, s, pl, d->lfc_dtype == DIV_BF16);
    p.log2cs = 0;
    while ((1u << p.log2cs) < pl.cs) ++p.log2cs;
    p.expect_bytes = fault.expect_bytes ? fault.expect_bytes : 8u * pl.cs;
    p.qbits = d->qbits;
    return d->x_dtype == DIV_F32 ? launch_cluster_p2<float>(p, pl, s, st) : launch_cluster_p2<__nv_bfloat16>(p, pl, s, st);
}

}  // namespace divk
