// Per-plane groups, any width (see planegroup.cuh for the form): compress with a CTA's planes kept in shared memory between
// the two halves (halves.cuh).  Nothing has to leave the CTA: a plane's extremes meet in shared memory.
//
// What bounds it: HBM, then instruction issue (several CTAs per SM, each loading, reducing or quantising).  It takes the
// shapes that the register-resident strip kernel cannot: odd widths beyond a warp and blocks of 16, where the general kernel
// (a thread per tile, then per packed word) is bound by scalar uncoalesced loads: 50 x 256 x 40 x 40 with B = 16 515 -> 37 us,
// 64 x 96 x 35 x 35 106 -> 21 us, 32 x 64 x 75 x 75 88 -> 29 us.
//
// The only wait is for the CTA's own copies.  It is bounded all the same; there is no status word to record it in, so a CTA that
// gives up stores NaN as the parameters of its planes (which rebuild as NaN), and leaves when the copies have landed or
// SHARE_DRAIN_NS have passed.
#include "halves.cuh"
#include "planegroup.cuh"

namespace divk {

struct PlaneShareParams : ShareParams {
    uint32_t* stats;
    FastDiv by_hw;
};
static_assert(sizeof(PlaneShareParams) <= SHARE_PARAM_BYTES, "dearer launches");

template <typename XT, int P2, typename G, int Q>
__global__ void __launch_bounds__(SHARE_THREADS, 3)
plane_share_kernel(const __grid_constant__ PlaneShareParams p) {
    typedef typename PackedUnit<Q>::type OutT;
    extern __shared__ __align__(128) unsigned char smem[];
    float* res = reinterpret_cast<float*>(smem);
    const uint32_t land_bytes = sizeof(XT) == 4 ? 0u : ((p.ppc * p.HW * 2u + 16u + 127u) & ~127u);
    XT* land = reinterpret_cast<XT*>(sizeof(XT) == 4 ? smem : smem + p.res_bytes);
    float4* par = reinterpret_cast<float4*>(smem + p.res_bytes + land_bytes);      // per plane: delta_b, 1 / Delta_b, -65536 / Delta_b (0: general route)
    uint32_t* keys = reinterpret_cast<uint32_t*>(par + p.ppc);
    __shared__ __align__(8) uint64_t full[SHARE_PIECES];
    __shared__ uint32_t gave_up;              // a warp's wait for a piece ran out
    const uint32_t tid = threadIdx.x;
    const uint32_t n = blockIdx.y, plane0 = blockIdx.x * p.ppc;
    const uint32_t nplanes = min(p.ppc, p.C - plane0);
    if (tid == 0) {
#pragma unroll
        for (uint32_t i = 0; i < SHARE_PIECES; ++i) mbar_init(&full[i], p.arrivals);
        gave_up = 0u;
        fence_barrier_init();
        griddep_wait();
        share_load(p, land, full, n, plane0, nplanes);
    }
    for (uint32_t i = tid; i < 2u * nplanes; i += SHARE_THREADS) keys[i] = 0u;
    __syncthreads();
    griddep_wait();
    griddep_launch();
    float lo, hi;
    share_half1<XT, P2, G, true, false, SHARE_THREADS>(p, res, land, full, n, plane0, nplanes, keys, &gave_up, lo, hi);
    __syncthreads();
    if (gave_up) {                            // the same in the whole CTA
        for (uint32_t i = tid; i < nplanes; i += SHARE_THREADS) p.stats[(uint64_t)n * p.C + plane0 + i] = 0x7FC07FC0u;
        if (tid < 32u) share_drain(p, full, nplanes);
        return;
    }
    for (uint32_t i = tid; i < nplanes; i += SHARE_THREADS) {
        const float rmax = key_float(keys[2u * i + 1u]);
        const PgQ q = pg_params(key_float(~keys[2u * i]), rmax, Q);
        QParams qp;
        qp.delta = q.delta;
        qp.scale = q.scale;
        par[i] = make_float4(q.delta, q.scale, fixed_point_ok<Q>(qp, rmax) ? -65536.0f * q.scale : 0.f, 0.f);
        p.stats[(uint64_t)n * p.C + plane0 + i] = pg_stats_word(q);
    }
    __syncthreads();
    const uint32_t qfirst = (plane0 * p.HW) >> 2, nq = (nplanes * p.HW) >> 2;
    OutT* out = reinterpret_cast<OutT*>(p.packed) + ((uint64_t)n * p.qps + qfirst);
    uint64_t ctr = rng_sample_base(p.seed, n) + K_GROUP * (uint64_t)(qfirst + tid + 1u);
    constexpr uint64_t STEP = K_GROUP * (uint64_t)SHARE_THREADS;
#pragma unroll 4
    for (uint32_t q = tid; q < nq; q += SHARE_THREADS) {
        const ulonglong2 v = reinterpret_cast<const ulonglong2*>(res)[q];
        const uint64_t z = rng_mix(ctr);
        ctr += STEP;
        const uint32_t pl = fdiv(4u * q, p.by_hw);
        const uint32_t rem = 4u * q - pl * p.HW;
        const float4 a = par[pl];
        if (rem + 4u <= p.HW) {
            if (Q <= 4 && a.z < 0.f) out[q] = (OutT)quant4_res<Q, Q <= 4>(v.x, v.y, pk2(a.x, a.x), pk2(a.z, a.z), z);
            else out[q] = (OutT)quant4_general<Q>(v.x, v.y, pk2(a.x, a.x), pk2(a.y, a.y), z);
        } else {
            // the quad runs into the next plane (planes of at least 4 elements: into no other)
            const float4 b = par[pl + 1u];
            const uint32_t own = p.HW - rem;                       // 1, 2 or 3
            const float4 e1 = own > 1u ? a : b, e2 = own > 2u ? a : b;
            uint32_t b0, b1, b2, b3;
            constexpr float qmax = (float)((1 << Q) - 1);
            quant2(v.x, 0ull, pk2(a.x, e1.x), pk2(a.y, e1.y), qmax, (uint32_t)z, b0, b1);
            quant2(v.y, 0ull, pk2(e2.x, b.x), pk2(e2.y, b.y), qmax, (uint32_t)(z >> 32), b2, b3);
            constexpr uint32_t BIAS = QUANT2_BITS * (1u + (1u << Q) + (1u << (2 * Q)) + (1u << (3 * Q)));   // mod 2^32
            out[q] = (OutT)(b0 + (b1 << Q) + (b2 << (2 * Q)) + (b3 << (3 * Q)) - BIAS);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
// Planes per CTA: of the counts up to a third of an SM's shared memory (or the fewest possible) the one whose slots leave
// the fewest lanes of the 8 warps idle.
bool plan_plane_share(const div_desc* d, const Shape& s, SharePlan* out) {
    const DeviceInfo di = device_info();
    if (!di.ok || di.sms < 1 || !share_takes(d, s) || s.HW < 4u || s.N > 65535u) return false;
    const uint32_t step = share_step(d, s), nc = s.P2 == 16 ? 2u : 4u, spb = s.Wb * (s.P2 / nc);
    const bool tail = s.H % s.B != 0;
    const uint64_t full = (uint64_t)(tail ? s.Hb - 1u : s.Hb) * spb, shrt = tail ? spb : 0u;
    double best = 0;
    for (uint64_t ppc = step; ppc <= 2048u; ppc += step) {
        SharePlan pl;
        if (!plan_share(d, s, ppc, (uint32_t)(24u * ppc + 32u), false, di, &pl)) break;
        if (ppc > step && pl.smem_bytes > 72u * 1024u) break;
        const uint64_t units = (ppc * full + 31u) / 32u + (ppc * shrt + 31u) / 32u;
        const double lanes = (double)(ppc * (full + shrt)) / (32.0 * ((units + SHARE_WARPS - 1u) / SHARE_WARPS * SHARE_WARPS));
        const double score = lanes * (double)(pl.smem_bytes < 16u * 1024u ? pl.smem_bytes : 16u * 1024u);      // small shares do not pay for their set-up
        if (score > best * 1.02) {
            best = score;
            *out = pl;
        }
        if (ppc >= s.C) break;
    }
    return best > 0;
}

template <typename XT, int P2, typename G, int Q>
inline div_status launch_plane_share(const PlaneShareParams& prm, const SharePlan& pl, uint32_t N, cudaStream_t st) {
    auto kern = plane_share_kernel<XT, P2, G, Q>;
    static SmemSeen smem_set[DEVICE_CACHE_SLOTS];
    if (!ensure_dynamic_smem((const void*)kern, (int)pl.smem_bytes, smem_set)) return DIV_ERR_CUDA;
    return launch_pdl(kern, dim3((prm.C + pl.ppc - 1u) / pl.ppc, N), SHARE_THREADS, pl.smem_bytes, st, prm);
}
template <typename XT, int P2, typename G>
inline div_status launch_plane_share_q(int qbits, const PlaneShareParams& prm, const SharePlan& pl, uint32_t N, cudaStream_t st) {
    switch (qbits) {
        case 2: return launch_plane_share<XT, P2, G, 2>(prm, pl, N, st);
        case 4: return launch_plane_share<XT, P2, G, 4>(prm, pl, N, st);
        case 8: return launch_plane_share<XT, P2, G, 8>(prm, pl, N, st);
    }
    return DIV_ERR_PARAM;
}
template <typename XT, int P2>
inline div_status launch_plane_share_geo(int qbits, const PlaneShareParams& prm, const SharePlan& pl, uint32_t N, cudaStream_t st) {
    constexpr int NC = P2 == 16 ? 2 : 4;
    if constexpr (NC == 4) {
        if (pl.vw == 4) return launch_plane_share_q<XT, P2, SlotGeo<4, 4>>(qbits, prm, pl, N, st);
    }
    return pl.vw >= 2 ? launch_plane_share_q<XT, P2, SlotGeo<NC, 2>>(qbits, prm, pl, N, st)
                      : launch_plane_share_q<XT, P2, SlotGeo<NC, 1>>(qbits, prm, pl, N, st);
}
template <typename XT>
inline div_status launch_plane_share_p2(uint32_t p2, int qbits, const PlaneShareParams& prm, const SharePlan& pl, uint32_t N, cudaStream_t st) {
    switch (p2) {
        case 4: return launch_plane_share_geo<XT, 4>(qbits, prm, pl, N, st);
        case 8: return launch_plane_share_geo<XT, 8>(qbits, prm, pl, N, st);
        case 16: return launch_plane_share_geo<XT, 16>(qbits, prm, pl, N, st);
    }
    return DIV_ERR_PARAM;
}

div_status compress_plane_share(const div_desc* d, const Shape& s, const div_layout& lo, const SharePlan& plan, const void* x, uint8_t* blob,
                                uint64_t seed, cudaStream_t st, const ShareFault& fault) {
    SharePlan pl = plan;
    pl.smem_bytes += fault.more_smem;
    PlaneShareParams p;
    p.x = x;
    p.lfc = blob + lo.lfc_off;
    p.packed = blob + lo.packed_off;
    p.stats = reinterpret_cast<uint32_t*>(blob + lo.stats_off);
    p.status = nullptr;
    p.number = 0;
    p.arrivals = fault.no_copies ? 2u : 1u;
    p.seed = seed;
    p.timeout_ns = fault.timeout_ns ? fault.timeout_ns : 2000000000u;
    fill_share(&p, s, pl, d->lfc_dtype == DIV_BF16);
    p.by_hw = host_fastdiv(s.HW);
    return d->x_dtype == DIV_F32 ? launch_plane_share_p2<float>(s.P2, d->qbits, p, pl, s.N, st)
                                 : launch_plane_share_p2<__nv_bfloat16>(s.P2, d->qbits, p, pl, s.N, st);
}

}  // namespace divk
