// The two halves of a compress kernel that keeps its share of x on chip, as code shared by such kernels:
//   half 1  one slot = the NC adjacent columns of one tile of one band (tile row) that a lane owns: tile sum in the fixed
//           order, stored low-frequency value, extremes, fp32 residual;
//   half 2  Eq. 9 on groups of 4 consecutive residuals, which needs no notion of tiles.
#pragma once

#include "cluster_plan.cuh" // SharePlan
#include "planes.cuh"       // ColLoad; quant_row, packed pairs

namespace divk {

// ------------------------------------------------------------------------------------------------
// arithmetic
// ------------------------------------------------------------------------------------------------
// sum / cnt, correctly rounded, for a small whole cnt and rcp = RN(1 / cnt): one Newton step on the quotient with an
// exact remainder (Markstein, "Computation of elementary functions on the IBM RISC System/6000", 1990).  Checked
// against IEEE division for every significand of the sum and every count that a tile of up to 16 x 16 can have
// (tests/test_gpu_mean_division.py); scaling by powers of two changes nothing while no intermediate result leaves the
// normal range, hence the guard.
__device__ __forceinline__ float div_by_count(float sum, float cnt, float rcp) {
    const float m = fabsf(sum);
    if (m > 1e-30f && m < 1e30f) {
        const float q = __fmul_rn(sum, rcp);
        return __fmaf_rn(__fmaf_rn(-q, cnt, sum), rcp, q);
    }
    return __fdiv_rn(sum, cnt);
}

// the same codes by the general route (clamped, any parameters)
template <int Q>
__device__ __forceinline__ uint32_t quant4_general(uint64_t xy, uint64_t zw, uint64_t delta2, uint64_t scale2, uint64_t z) {
    return quant_row<Q>(xy, zw, 0ull, delta2, scale2, z);        // r - 0 is r (a zero's sign does not reach the codes)
}
template <int Q, bool FIXED>
__device__ __forceinline__ uint32_t quant4_res(uint64_t xy, uint64_t zw, uint64_t delta2, uint64_t mul2, uint64_t z) {
    if constexpr (FIXED && Q <= 4) return quant4_fixed<Q>(xy, zw, delta2, mul2, z);
    else return quant4_general<Q>(xy, zw, delta2, mul2, z);
}

// ------------------------------------------------------------------------------------------------
// half 1: one slot = NC adjacent columns of one tile of one band
// ------------------------------------------------------------------------------------------------
// How a slot is read: NC columns (4; 2 where 16 rows of 4 would not fit the registers), VW of them at a time (4, 2 or 1:
// what the alignment of the rows allows).  Where a row takes several accesses, lane groups take them in different
// orders: access u reads the columns VW * (u ^ swap) ..., swap from the lane number.  Neighbouring lanes are NC words
// apart, so with one order for all NC / VW lanes would meet in every bank; with these orders none do.  A slot's columns
// then sit in the registers in a lane-dependent order, of which every sum below is independent: swap only exchanges
// the operands of an addition.
template <int NC_, int VW_> struct SlotGeo {
    static constexpr int NC = NC_, VW = VW_, NU = NC_ / VW_, NV = NC_ / 2;
    static __device__ __forceinline__ uint32_t swap(uint32_t lane) { return NU == 4 ? (lane >> 3) & 3u : NU == 2 ? (NC == 4 ? (lane >> 3) & 1u : lane >> 4) : 0u; }
};
template <typename XT, typename G>
__device__ __forceinline__ void slot_row_load(const XT* p, const uint32_t (&col)[G::NU], uint64_t (&v)[G::NV]) {
    if constexpr (G::VW == 4) {
        StripRow2<XT>::load(reinterpret_cast<const unsigned char*>(p), v[0], v[1]);
    } else if constexpr (G::VW == 2) {
#pragma unroll
        for (int u = 0; u < G::NU; ++u) v[u] = ColLoad<XT, 2>::load(p + col[u]);
    } else {
#pragma unroll
        for (int u = 0; u < G::NV; ++u) {
            if constexpr (sizeof(XT) == 4) {
                v[u] = pk2(p[col[2 * u]], p[col[2 * u + 1]]);
            } else {
                const uint16_t* h = reinterpret_cast<const uint16_t*>(p);
                v[u] = pk2u((uint32_t)h[col[2 * u]] << 16, (uint32_t)h[col[2 * u + 1]] << 16);
            }
        }
    }
}

struct SlotSink {
    void* lfc;
    uint64_t lfc_at;          // where the tile's low-frequency value goes
    int32_t lfc_bf16;
    bool writer;              // this lane stores it
    float cnt, rcp;           // count (0: a power of two, multiply), RN(1 / count)
};
// Mean of a slot's tile as it is stored.  Every lane of the warp calls it (lanes of a tile meet by shuffles); columns a
// lane does not own count as zeros.
template <typename XT, int P2, typename G, int ROWS>
__device__ __forceinline__ float slot_mean(const uint64_t (&v)[ROWS][G::NV], const bool (&ok)[G::NU], bool any, const SlotSink& s) {
    constexpr int NV = G::NV;
    constexpr uint32_t LPT = P2 / G::NC;                       // lanes per tile
    // tile sum in the fixed order: balanced tree down the rows of each column (missing rows are zeros), then across the columns
    float part[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        uint64_t t[P2];
#pragma unroll
        for (int r = 0; r < P2; ++r) t[r] = r < ROWS ? v[r < ROWS ? r : 0][k] : 0ull;
#pragma unroll
        for (int w = P2 / 2, left = ROWS; w >= 1; w >>= 1, left = (left + 1) / 2)
#pragma unroll
            for (int i = 0; i < w; ++i)
                if (2 * i < left) t[i] = add2_rn(t[2 * i], 2 * i + 1 < left ? t[2 * i + 1] : 0ull);
        float c0, c1;
        upk2(t[0], c0, c1);
        // what was loaded for a column the lane does not own belongs to somebody else
        if (!ok[G::VW == 1 ? 2 * k : G::VW == 2 ? k : 0]) c0 = 0.f;
        if (!ok[G::VW == 1 ? 2 * k + 1 : G::VW == 2 ? k : 0]) c1 = 0.f;
        part[k] = __fadd_rn(c0, c1);
    }
    float sum = NV == 2 ? __fadd_rn(part[0], part[NV - 1]) : part[0];
#pragma unroll
    for (int m = 1; m < (int)LPT; m <<= 1) sum = __fadd_rn(sum, __shfl_xor_sync(0xFFFFFFFFu, sum, m));
    const float mean = s.cnt == 0.f ? __fmul_rn(sum, s.rcp) : div_by_count(sum, s.cnt, s.rcp);
    if (any && s.writer) {
        if (s.lfc_bf16) Elem<__nv_bfloat16>::store(reinterpret_cast<__nv_bfloat16*>(s.lfc) + s.lfc_at, mean);
        else reinterpret_cast<float*>(s.lfc)[s.lfc_at] = mean;
    }
    return s.lfc_bf16 ? Elem<__nv_bfloat16>::round(mean) : mean;
}

// One slot of half 1 whose residuals go to shared memory.  All slots of a warp have the same number of rows, ROWS; a lane
// owns the first `cols` of its NC columns (0: none; it loads from anywhere in bounds).  xs / rp: first element of the
// slot where x landed / where the residual goes (the same place for fp32).  IN_PLACE (VW = 4): no residuals, rp takes the
// tile's stored low-frequency value.  lo / hi collect the residual's extremes.
template <typename XT, int P2, typename G, bool IN_PLACE, int ROWS>
__device__ __forceinline__ void reduce_slot_rows(const XT* xs, float* rp, uint32_t W, uint32_t cols, const SlotSink& s, float& lo, float& hi) {
    constexpr int NV = G::NV, NU = G::NU;
    const uint32_t sw = G::swap(threadIdx.x & 31u);
    uint32_t col[NU];
    bool ok[NU];
#pragma unroll
    for (int u = 0; u < NU; ++u) {
        col[u] = ((uint32_t)u ^ sw) * G::VW;
        ok[u] = col[u] < cols;
    }
    uint64_t v[ROWS][NV];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) slot_row_load<XT, G>(xs + r * W, col, v[r]);
    const float stored = slot_mean<XT, P2, G, ROWS>(v, ok, cols != 0u, s);
    if (IN_PLACE && cols != 0u && s.writer) *rp = stored;
    if (cols != 0u) {
        // residuals back to shared memory; extremes of x (x -> fl(x - stored) is monotone): of the columns of one access
        // together, or of two rows at a time where every column has to be kept apart
        const uint64_t stored2 = pk2(stored, stored);
        float l[NU], h[NU];
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            l[u] = 3.402823466e+38f;
            h[u] = -3.402823466e+38f;
        }
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            float x[2 * NV], y[2 * NV];
            uint64_t d[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                d[k] = sub2_rn(v[r][k], stored2);
                upk2(v[r][k], x[2 * k], x[2 * k + 1]);
            }
            float* row = rp + r * W;
            if constexpr (G::VW == 4) {
                l[0] = fmin3(fmin3(l[0], x[0], x[1]), x[2], x[3]);
                h[0] = fmax3(fmax3(h[0], x[0], x[1]), x[2], x[3]);
                if constexpr (!IN_PLACE) {
                    ulonglong2 q;
                    q.x = d[0];
                    q.y = d[1];
                    *reinterpret_cast<ulonglong2*>(row) = q;
                }
            } else if constexpr (G::VW == 2) {
#pragma unroll
                for (int u = 0; u < NU; ++u) {
                    l[u] = fmin3(l[u], x[2 * u], x[2 * u + 1]);
                    h[u] = fmax3(h[u], x[2 * u], x[2 * u + 1]);
                    if (ok[u]) *reinterpret_cast<uint64_t*>(row + col[u]) = d[u];
                }
            } else {
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    upk2(v[r % 2 == 1 ? r - 1 : r][k], y[2 * k], y[2 * k + 1]);
                    if (r % 2 == 1 || r + 1 == ROWS) {
#pragma unroll
                        for (int c = 2 * k; c < 2 * k + 2; ++c) {
                            l[c] = fmin3(l[c], x[c], y[c]);
                            h[c] = fmax3(h[c], x[c], y[c]);
                        }
                    }
                    float d0, d1;
                    upk2(d[k], d0, d1);
                    if (ok[2 * k]) row[col[2 * k]] = d0;
                    if (ok[2 * k + 1]) row[col[2 * k + 1]] = d1;
                }
            }
        }
        float lx = 3.402823466e+38f, hx = -3.402823466e+38f;
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            if (NU == 1 || ok[u]) {
                lx = fminf(lx, l[u]);
                hx = fmaxf(hx, h[u]);
            }
        }
        lo = fminf(lo, __fsub_rn(lx, stored));
        hi = fmaxf(hi, __fsub_rn(hx, stored));
    }
}
// the row count is the same in the whole warp: one unrolled body for each
template <typename XT, int P2, typename G, bool IN_PLACE, int ROWS = P2>
__device__ __forceinline__ void reduce_slot(const XT* xs, float* rp, uint32_t W, uint32_t rows, uint32_t cols, const SlotSink& s, float& lo,
                                            float& hi) {
    if (ROWS == 1 || rows == (uint32_t)ROWS) reduce_slot_rows<XT, P2, G, IN_PLACE, ROWS>(xs, rp, W, cols, s, lo, hi);
    else if constexpr (ROWS > 1) reduce_slot<XT, P2, G, IN_PLACE, ROWS - 1>(xs, rp, W, rows, cols, s, lo, hi);
}

// ------------------------------------------------------------------------------------------------
// a CTA's share: a run of whole planes of one sample in shared memory
// ------------------------------------------------------------------------------------------------
struct ShareParams {
    const void* x;
    void* lfc;
    void* packed;
    uint64_t* status;         // where a wait that ran out is recorded (share_record)
    uint64_t seed;
    uint32_t number;          // of the call, recorded with a failure
    uint32_t timeout_ns;
    uint32_t arrivals;        // what a piece's barrier waits for: 1, its copy; in a test 2, the second of which never comes (in the barriers'
                              // set-up, which nothing waits for: as bytes beyond the copy's it cost 5 % on one-plane shares)
    uint32_t C, W, B, Hb, Wb, HW, TPP, qps;
    uint32_t ppc, ppp;        // planes per CTA, planes per piece
    uint32_t res_bytes;       // bf16: where the landing place begins, behind the fp32 residuals
    uint32_t spb;             // slots per band (tile row) of a plane
    uint32_t sppf;            // slots of full-height bands per plane
    uint32_t sppt;            // slots of a short last band per plane (0: H % B == 0)
    uint32_t tail_rows;
    uint32_t partial;         // 1: the last tile of a row is narrower than B
    int32_t lfc_bf16;
    FastDiv by_sppf, by_spb, by_ppp;
    float cnt[4], rcp[4];     // [short band][narrow tile]: count (0: a power of two, the mean is a product), RN(1 / count)
    __host__ __device__ uint64_t failure() const { return (uint64_t)number << 32 | (uint64_t)DIV_ERR_TIMEOUT; }
};
// Launching a kernel with more than 224 bytes of parameters costs the host 0.4 us more: 8 x 64 x 32 x 32, compress and decompress
// 7.0 us with 224 bytes, 7.4 with 232.
constexpr size_t SHARE_PARAM_BYTES = 224;
// The status words, as one 64-bit word: zero, or the failure of a call with the call's number.  One CTA clears what an earlier
// call (or nobody) left there, in no order with the other CTAs of the launch, which may have failed already: it leaves
// alone what carries the number of its own call.  (The replays of a captured call share its number: a failure that one of
// them recorded stays.)
__device__ __forceinline__ void share_record(const ShareParams& p) { atomicExch(reinterpret_cast<unsigned long long*>(p.status), p.failure()); }
__device__ __forceinline__ void share_clear_status(const ShareParams& p, unsigned long long seen) {
    unsigned long long* w = reinterpret_cast<unsigned long long*>(p.status);
    while (seen != 0ull && seen != p.failure()) {            // at most twice: from here on only failure() is written
        const unsigned long long old = atomicCAS(w, seen, 0ull);
        if (old == seen) break;
        seen = old;
    }
}
struct CtaScope {
    static __device__ __forceinline__ bool try_wait(uint64_t* bar) { return mbar_try_wait(bar, 0); }
};
template <typename Scope = CtaScope>
__device__ __forceinline__ bool share_wait(uint64_t* bar, uint64_t timeout_ns) {
    if (Scope::try_wait(bar)) return true;
    uint32_t polls = 0;
    uint64_t t0 = 0;
    while (!Scope::try_wait(bar)) {
        if ((++polls & 15u) == 0) {
            const uint64_t t = now_ns();
            if (t0 == 0) t0 = t;
            if (t - t0 > timeout_ns) return Scope::try_wait(bar);      // the clock may have jumped past the limit
        }
    }
    return true;
}
// what a CTA that gives up still waits for what is on its way into its shared memory, which is somebody else's once it has left
constexpr uint64_t SHARE_DRAIN_NS = 20000000;

// the copies of the share, one thread: piece i completes on full[i]
template <typename XT>
__device__ __forceinline__ void share_load(const ShareParams& p, XT* land, uint64_t* full, uint32_t n, uint32_t plane0, uint32_t nplanes) {
    const XT* src = reinterpret_cast<const XT*>(p.x) + ((uint64_t)n * p.C + plane0) * p.HW;
    for (uint32_t i = 0, a = 0; a < nplanes; ++i, a += p.ppp) {
        const uint32_t bytes = min(p.ppp, nplanes - a) * p.HW * (uint32_t)sizeof(XT);
        mbar_arrive_expect_tx(&full[i], bytes);
        bulk_load(land + (size_t)a * p.HW, src + (size_t)a * p.HW, bytes, &full[i]);
    }
}
// before a CTA leaves with a wait for a piece that ran out: one warp, until every piece has landed or the limit has passed
__device__ __forceinline__ void share_drain(const ShareParams& p, uint64_t* full, uint32_t nplanes) {
    const uint64_t t0 = now_ns();
    for (uint32_t i = 0, a = 0; a < nplanes; ++i, a += p.ppp)
        while (!mbar_try_wait(&full[i], 0))
            if (now_ns() - t0 > SHARE_DRAIN_NS) return;
}

// Slots of the CTA's share are numbered so that every warp holds slots of one height: the full-height bands of all planes
// first, then, from the next multiple of 32, the short last bands.
struct ShareSlot {
    bool valid, short_band, narrow, writer;
    uint32_t plane, tile;     // plane and tile inside the share
    uint32_t off, rows, cols; // first element inside the share; rows; columns this lane owns (0: none)
};
template <int P2, int NC>
__device__ __forceinline__ ShareSlot share_slot(const ShareParams& p, uint32_t first, uint32_t lane, uint32_t nfull, uint32_t first_short,
                                                uint32_t total) {
    constexpr uint32_t LPT = P2 / NC;                          // lanes per tile
    ShareSlot t;
    t.short_band = first >= first_short;                       // the same in the whole warp
    const uint32_t S = first + lane;
    t.valid = t.short_band ? S < total : S < nfull;
    const uint32_t T = t.valid ? (t.short_band ? S - first_short : S) : 0u;
    t.plane = fdiv(T, t.short_band ? p.by_spb : p.by_sppf);
    const uint32_t rem = T - t.plane * (t.short_band ? p.spb : p.sppf);
    const uint32_t bf = fdiv(rem, p.by_spb);
    const uint32_t band = t.short_band ? p.Hb - 1u : bf;
    const uint32_t q = rem - bf * p.spb;                       // slot inside the band (a short band's rem is below spb)
    const uint32_t bw = q / LPT, cw = (q % LPT) * NC;
    t.narrow = p.partial && bw + 1u == p.Wb;
    const uint32_t cols = t.narrow ? p.W - bw * p.B : p.B;
    t.cols = t.valid && cw < cols ? min(cols - cw, (uint32_t)NC) : 0u;
    t.off = t.cols ? t.plane * p.HW + (band * p.B) * p.W + bw * p.B + cw : 0u;
    t.tile = t.plane * p.TPP + band * p.Wb + bw;
    t.writer = cw == 0;
    t.rows = t.short_band ? p.tail_rows : p.B;
    return t;
}

// ------------------------------------------------------------------------------------------------
// half 1 of a CTA's share: planes [plane0, plane0 + nplanes) of sample n, which land in shared memory in SHARE_PIECES pieces
// ------------------------------------------------------------------------------------------------
// IN_PLACE: x stays as it is and res takes the stored low-frequency values of the tiles instead of the residuals.
// keys (PER_PLANE): ~key(min), key(max) of the residuals of each plane; else lo / hi collect the extremes of the thread.
// A wait for a piece that runs out is noted in *gave_up, in shared memory; the warp then works on with whatever is there and waits for
// no further piece (a way out of the loop costs the ordinary case 1 %), and the caller lets nothing of it out.
template <typename XT, int P2, typename G, bool PER_PLANE, bool IN_PLACE, uint32_t THREADS>
__device__ __forceinline__ void share_half1(const ShareParams& p, float* res, const XT* land, uint64_t* full, uint32_t n, uint32_t plane0,
                                         uint32_t nplanes, uint32_t* keys, uint32_t* gave_up, float& lo, float& hi) {
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t nfull = nplanes * p.sppf, first_short = (nfull + 31u) & ~31u, total = first_short + nplanes * p.sppt;
    const uint64_t lfc0 = ((uint64_t)n * p.C + plane0) * p.TPP;
    uint32_t landed = 0;
    for (uint32_t first = warp * 32u; first < total; first += THREADS) {
        const ShareSlot t = share_slot<P2, G::NC>(p, first, lane, nfull, first_short, total);
        // pieces land in order; the unit's last slot needs the latest one
        {
            const uint32_t last = __shfl_sync(0xFFFFFFFFu, t.valid ? t.plane : nplanes - 1u, 31);
            const uint32_t need = fdiv(last, p.by_ppp) + 1u;
            while (landed < need) {
                if (!share_wait(&full[landed], p.timeout_ns)) {
                    *gave_up = 1u;
                    landed = SHARE_PIECES - 1u;
                }
                ++landed;
            }
        }
        const uint32_t which = (t.short_band ? 2u : 0u) + (t.narrow ? 1u : 0u);
        SlotSink sink;
        sink.lfc = p.lfc;
        sink.lfc_at = lfc0 + t.tile;
        sink.lfc_bf16 = p.lfc_bf16;
        sink.writer = t.writer;
        sink.cnt = p.cnt[which];
        sink.rcp = p.rcp[which];
        if constexpr (!PER_PLANE) {
            reduce_slot<XT, P2, G, IN_PLACE>(land + t.off, res + (IN_PLACE ? t.tile : t.off), p.W, t.rows, t.cols, sink, lo, hi);
        } else {
            float l = 3.402823466e+38f, h = -3.402823466e+38f;
            reduce_slot<XT, P2, G, IN_PLACE>(land + t.off, res + (IN_PLACE ? t.tile : t.off), p.W, t.rows, t.cols, sink, l, h);
            // lanes without a slot bring neutral extremes (whose keys are not neutral)
            uint32_t kmin = t.cols ? ~float_key(l) : 0u, kmax = t.cols ? float_key(h) : 0u;
            const uint32_t first_plane = __shfl_sync(0xFFFFFFFFu, t.plane, 0);
            if (__all_sync(0xFFFFFFFFu, t.plane == first_plane || t.cols == 0u)) {
                kmin = __reduce_max_sync(0xFFFFFFFFu, kmin);
                kmax = __reduce_max_sync(0xFFFFFFFFu, kmax);
                if (lane == 0) {
                    atomicMax(&keys[2u * first_plane], kmin);
                    atomicMax(&keys[2u * first_plane + 1u], kmax);
                }
            } else if (t.cols) {
                atomicMax(&keys[2u * t.plane], kmin);
                atomicMax(&keys[2u * t.plane + 1u], kmax);
            }
        }
    }
}

inline void fill_share(ShareParams* p, const Shape& s, const SharePlan& pl, bool lfc_bf16) {
    p->C = s.C; p->W = s.W; p->B = s.B; p->Hb = s.Hb; p->Wb = s.Wb; p->HW = s.HW; p->TPP = s.TPP; p->qps = s.CHW / 4;
    p->ppc = pl.ppc; p->ppp = pl.ppp; p->res_bytes = pl.res_bytes;
    const uint32_t nc = s.P2 == 16 ? 2u : 4u;                  // columns of a slot
    p->spb = s.Wb * (s.P2 / nc);
    const bool tail = s.H % s.B != 0;
    p->sppf = (tail ? s.Hb - 1u : s.Hb) * p->spb;
    p->sppt = tail ? p->spb : 0u;
    p->tail_rows = s.H - (s.Hb - 1u) * s.B;
    p->partial = s.W % s.B != 0 ? 1u : 0u;
    p->lfc_bf16 = lfc_bf16 ? 1 : 0;
    p->by_sppf = host_fastdiv(p->sppf ? p->sppf : 1u);
    p->by_spb = host_fastdiv(p->spb);
    p->by_ppp = host_fastdiv(p->ppp);
    const uint32_t tail_cols = s.W - (s.Wb - 1u) * s.B;
    for (int i = 0; i < 4; ++i) {
        const uint32_t cnt = ((i & 2) ? p->tail_rows : s.B) * ((i & 1) ? tail_cols : s.B);
        p->cnt[i] = (cnt & (cnt - 1u)) == 0 ? 0.f : (float)cnt;
        p->rcp[i] = 1.0f / (float)cnt;
    }
}

}  // namespace divk
