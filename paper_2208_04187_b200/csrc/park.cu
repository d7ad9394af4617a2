// Parking compress kernel (DIVISION Sec. 4.1; Algorithm 1, forward loop) for the common CNN shapes: W % 4 == 0, B in {4, 8},
// Q in {2, 4, 8}, samples that the whole device works on at once.
//
// x is read once, by bulk copies, and its residuals wait in TENSOR MEMORY (256 KB per SM, 38 MB in all) until the sample's extremes are
// known.  The kernel that reads x a second time from L2 (staged.cuh) moves twice the bytes through the L2-to-SM fabric and forms every tile
// mean twice: 64 x 64 x 112 x 112 (205 MB, x alone at the copy rate 31.8 us) 55.6 -> 45.0 us, 64 x 512 x 28 x 28 38.4 -> 31.3 us; the
// cluster kernel, whose samples take turns, bfloat16 128 x 160 x 32 x 32 with B = 4 29.7 -> 22.9 us.
//
//   * a CHUNK is a run of G tile row bands of one sample, contiguous in memory (about 7000 elements).  Chunk j belongs to CTA
//     j mod gridDim.x, so the CTAs sweep the tensor together.  The producer thread brings a CTA's chunks into a ring in shared memory,
//     few at a time (PARK_AHEAD_BYTES).
//   * a STRIP is 4 adjacent columns of one band; a lane owns one strip of 8 rows or two of 4; a UNIT is what the 32 lanes of a warp own,
//     1024 elements.  Worker w of nf * sets takes unit w % nf of the chunks w / nf, w / nf + sets, ...: where its strips lie in a chunk is
//     the same every time and stays in registers.
//   * a worker reduces a unit (tile means in the fixed order, stored low-frequency values, extremes), hands the stage back, parks the residuals
//     in its own columns of tensor memory, and goes on; before it would park more than PARK_DEPTH units it quantises the oldest.
//     Nobody else touches its columns: no barrier stands between the two halves.
//   * a publisher warp folds a chunk's extremes into the sample's slot in global scratch once all its units are reduced, fences, and counts
//     the chunk as arrived; the watcher polls the count of the samples that this CTA needs next (an acquiring load), derives (delta, Delta,
//     scale) and posts them beside the chunk.
//
// What bounds it: the way from a unit's reduction to its sample's parameters, 4 - 5 us of which the fence, the poll and the slowest of a sample's
// CTAs take most, against the 200 KB that an SM can park (without the quantise half 38 us); issue slots next.  Tried: residuals held in
// registers instead (28 warps, 83.6 us), separate reduce and quantise warps over tensor memory (56.8 us), counts without the fence (41 us, but
// nothing then orders the folds before the count).
//
// The launch is cooperative so that all CTAs are resident; no grid-wide barrier is used.  Every wait is bounded: when a limit runs out the
// kernel records DIV_ERR_TIMEOUT in the workspace status word, stops waiting everywhere, lets its own copies land, gives its tensor
// memory back and returns.
//
// Why no wait can last: take the first sample that is not complete and one of its units that has not been reduced, chunk c of CTA Y, worker w.
// w can be stuck on the parameters of a chunk that is at least PARK_DEPTH * sets before c; a CTA has at most that many chunks of one
// sample (plan_park), so that chunk's sample is an earlier one, which is complete.  Or chunk c has not landed because its stage is
// still being read: by a worker that is stuck in the same way, on a chunk even further back.  Or chunk c has not been asked for because
// chunk c - ahead has not landed, which nothing holds up: a record has not been filled again by then (ahead <= stages < PARK_CHUNKS; a
// parity tells a fill from the next and no more).
// Chunk records are reused after PARK_CHUNKS chunks: while chunk a is not quantised its worker does not read chunk a + PARK_DEPTH * sets,
// so that nothing beyond the PARK_MAX_STAGES chunks from there on is on its way.
#include "halves.cuh"
#include "park_plan.cuh"
#include "staged.cuh"

namespace divk {

struct ParkParams {
    Shape s;
    ParkPlan pl;
    FastDiv by_S, by_stages;
    const void* x;
    void* lfc;
    void* packed;
    float* stats;
    uint32_t* ws;
    uint64_t seed;
    uint64_t rng_row_step;         // K_GROUP * (W / 4)
    uint64_t timeout_ns;
    uint32_t expected_chunks;
    uint32_t tail_rows;
    float inv_cnt[4], cnt[4];
};

// ------------------------------------------------------------------------------------------------
// tensor memory: 32 columns (numbers of a lane) of the quarter that the warp may touch
// ------------------------------------------------------------------------------------------------
// (all lanes of the warp together: what is before may have parted them)
__device__ __forceinline__ void tmem_store32(uint32_t at, const uint32_t (&v)[32]) {
    __syncwarp();
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(at),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
        "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
        "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// (the wait names the registers: nothing may touch them between the two)
__device__ __forceinline__ void tmem_load32(uint32_t at, uint32_t (&v)[32]) {
    __syncwarp();
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(at)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;"
        : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
        "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
        "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
        "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
        :
        : "memory");
}
__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ bool p_give_up(const ParkParams& p, ParkCtl* ctl, SWait& w) {
    const long long c = clock64();
    if (w.c0 == 0) {
        w.c0 = c;
        w.t0 = 0;
        return false;
    }
    if (c - w.c0 < S_SLOW_CYCLES) return false;
    w.c0 = c;
    if (lds_volatile(&ctl->failed) || ld_relaxed_u32(p.ws) != 0u) return true;
    const uint64_t t = now_ns();
    if (w.t0 == 0) w.t0 = t;
    return t - w.t0 > p.timeout_ns;
}
__device__ __forceinline__ void p_record(const ParkParams& p, ParkCtl* ctl, uint32_t detail) {
    atomicCAS(p.ws, 0u, (uint32_t)DIV_ERR_TIMEOUT);
    atomicCAS(p.ws + 1, 0u, detail);
    sts_volatile(&ctl->failed, 1u);
}
__device__ __forceinline__ bool p_wait(uint64_t* bar, uint32_t parity, const ParkParams& p, ParkCtl* ctl, uint32_t detail) {
    if (mbar_try_wait(bar, parity)) return true;
    uint32_t polls = 0;
    SWait w = {0, 0};
    while (!mbar_try_wait(bar, parity)) {
        if ((++polls & 7u) == 0 && p_give_up(p, ctl, w)) {
            p_record(p, ctl, detail);
            return false;
        }
    }
    return true;
}
template <int P2> struct ParkStrips { static constexpr int N = 8 / P2; };      // strips of a lane: 32 numbers

template <typename XT, typename LT, int P2, bool FULL>
__device__ __forceinline__ void park_reduce(const ParkParams& p, ParkCtl* ctl, const unsigned char* stage, uint64_t* empty, uint32_t slot,
                                            const uint32_t (&table)[ParkStrips<P2>::N], const float (&inv)[ParkStrips<P2>::N], uint32_t at) {
    constexpr int MS = ParkStrips<P2>::N;
    constexpr uint32_t QSHIFT = sizeof(XT) == 4 ? 4u : 3u;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t row_bytes = p.s.W * (uint32_t)sizeof(XT);
    const ParkDesc& d = ctl->desc[slot];
    const uint32_t ntiles = d.ntiles;
    uint64_t vxy[MS][P2], vzw[MS][P2];
#pragma unroll
    for (int m = 0; m < MS; ++m) {
        const unsigned char* xs = stage + ((size_t)(table[m] & 0x1FFFu) << QSHIFT);
        const uint32_t rows = (table[m] >> 13) & 15u;
#pragma unroll
        for (int r = 0; r < P2; ++r) {
            if (!FULL) {
                vxy[m][r] = 0ull;
                vzw[m][r] = 0ull;
            }
            if (FULL || (uint32_t)r < rows) StripRow2<XT>::load(xs + r * row_bytes, vxy[m][r], vzw[m][r]);
        }
    }
    uint32_t kmin = 0u, kmax = 0u;                              // (keys, so that a NaN that came in stays one)
    uint32_t res[32];
#pragma unroll
    for (int m = 0; m < MS; ++m) {
        const uint32_t rows = (table[m] >> 13) & 15u, which = (table[m] >> 17) & 3u;
        const bool active = rows != 0u && (table[m] >> 21) < ntiles;
        const float mean = s_tile_mean<P2>(vxy[m], vzw[m], active, (table[m] >> 20) & 1u, inv[m], p.cnt[which]);
        if (m == MS - 1) {
            __syncwarp();                                      // every lane has its rows
            if (lane == 0) mbar_arrive(empty);
        }
        const float stored = Elem<LT>::round(mean);
        if (active && (table[m] & (1u << 19))) Elem<LT>::store(reinterpret_cast<LT*>(p.lfc) + d.lfc0 + (table[m] >> 21), mean);
        float blo = 3.402823466e+38f, bhi = -3.402823466e+38f;
        const uint64_t stored2 = pk2(stored, stored);
#pragma unroll
        for (int r = 0; r < P2; ++r) {
            const int i = (m * P2 + r) * 4;
            if (FULL || (uint32_t)r < rows) {
                float a_, b_, c_, d_;
                upk2(vxy[m][r], a_, b_);
                upk2(vzw[m][r], c_, d_);
                blo = fmin3(blo, a_, b_);
                blo = fmin3(blo, c_, d_);
                bhi = fmax3(bhi, a_, b_);
                bhi = fmax3(bhi, c_, d_);
            }
            upk2u(sub2_rn(vxy[m][r], stored2), res[i], res[i + 1]);
            upk2u(sub2_rn(vzw[m][r], stored2), res[i + 2], res[i + 3]);
        }
        if (active) {
            kmin = max(kmin, ~float_key(__fsub_rn(blo, stored)));
            kmax = max(kmax, float_key(__fsub_rn(bhi, stored)));
        }
    }
    tmem_store32(at, res);
    kmin = __reduce_max_sync(0xFFFFFFFFu, kmin);
    kmax = __reduce_max_sync(0xFFFFFFFFu, kmax);
    if (lane == 0) {
        atomicMax(&ctl->kmin[slot], kmin);
        atomicMax(&ctl->kmax[slot], kmax);
        mbar_arrive(&ctl->folded[slot]);
    }
}

template <int P2, int Q, bool FULL>
__device__ __forceinline__ void park_quantise(const ParkParams& p, ParkCtl* ctl, uint32_t slot, const uint32_t (&table)[ParkStrips<P2>::N], uint32_t at) {
    typedef typename PackedUnit<Q>::type OutT;
    uint32_t v[32];
    tmem_load32(at, v);
    const ParkDesc& d = ctl->desc[slot];
    const uint32_t W4 = p.s.W >> 2, ntiles = d.ntiles;
    const float delta = ctl->delta[slot], scale = ctl->scale[slot];
    const uint64_t delta2 = pk2(delta, delta), mul2 = tagged_mul2(scale);
    by_tag<Q>(scale, [&](auto fixed) {
        constexpr bool FIXED = decltype(fixed)::value;
#pragma unroll
        for (int m = 0; m < ParkStrips<P2>::N; ++m) {
            const uint32_t quad = table[m] & 0x1FFFu, rows = (table[m] >> 13) & 15u;
            if (rows != 0u && (table[m] >> 21) < ntiles) {
                uint64_t ctr = d.ctr0 + K_GROUP * (uint64_t)quad;
                OutT* out = reinterpret_cast<OutT*>(p.packed) + d.quad0 + quad;
#pragma unroll
                for (int r = 0; r < P2; ++r) {
                    const int i = (m * P2 + r) * 4;
                    if (FULL || (uint32_t)r < rows)
                        *out = (OutT)quant4_res<Q, FIXED>(pk2u(v[i], v[i + 1]), pk2u(v[i + 2], v[i + 3]), delta2, mul2, rng_mix(ctr));
                    out += W4;
                    ctr += p.rng_row_step;
                }
            }
        }
    });
}

template <typename XT, typename LT, int P2, int Q, bool FULL>
__device__ __forceinline__ void park_work(const ParkParams& p, ParkCtl* ctl, unsigned char* ring, uint32_t n_my, uint32_t it, const uint32_t (&table)[ParkStrips<P2>::N], uint32_t tm) {
    const uint32_t K = p.pl.stages, sets = p.pl.sets;
    float inv[ParkStrips<P2>::N];
#pragma unroll
    for (int m = 0; m < ParkStrips<P2>::N; ++m) inv[m] = p.inv_cnt[(table[m] >> 17) & 3u];
    uint32_t itq = it, bay = 0, filled = 0, st = it;
    while (st >= K) st -= K;
    while (itq < n_my) {
        if (filled == PARK_DEPTH || it >= n_my) {
            const uint32_t slot = itq % PARK_CHUNKS;
            if (!__all_sync(0xFFFFFFFFu, p_wait(&ctl->par[slot], (itq / PARK_CHUNKS) & 1u, p, ctl, 0x10000000u | itq))) return;
            const uint32_t at = bay >= filled ? bay - filled : bay + PARK_DEPTH - filled;          // the oldest one
            park_quantise<P2, Q, FULL>(p, ctl, slot, table, tm + at * 32u);
            itq += sets;
            --filled;
        }
        if (it < n_my) {
            const uint32_t slot = it % PARK_CHUNKS;
            if (!__all_sync(0xFFFFFFFFu, p_wait(&ctl->full[slot], (it / PARK_CHUNKS) & 1u, p, ctl, 0x40000000u | it))) return;
            park_reduce<XT, LT, P2, FULL>(p, ctl, ring + (size_t)st * p.pl.stage_bytes, &ctl->empty[st], slot, table, inv, tm + bay * 32u);
            it += sets;
            st += sets;
            while (st >= K) st -= K;
            bay = bay + 1u == PARK_DEPTH ? 0u : bay + 1u;
            ++filled;
        }
    }
}

template <typename XT, typename LT, int P2, int Q>
__global__ void __launch_bounds__(PARK_THREADS, 1)
park_kernel(const __grid_constant__ ParkParams p) {
    constexpr uint32_t LPT = P2 / 4;
    constexpr int MS = ParkStrips<P2>::N;

    extern __shared__ __align__(128) unsigned char smem[];
    const Shape& s = p.s;
    const uint32_t K = p.pl.stages, nf = p.pl.nf;
    unsigned char* ring = smem;
    uint32_t* table = reinterpret_cast<uint32_t*>(ring + (size_t)K * p.pl.stage_bytes);
    ParkCtl* ctl = reinterpret_cast<ParkCtl*>(reinterpret_cast<unsigned char*>(table) + (size_t)nf * MS * 128u);

    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t S = p.pl.chunks_per_sample, TU = p.pl.total_chunks, grid = gridDim.x;
    const uint32_t n_my = blockIdx.x < TU ? (TU - blockIdx.x + grid - 1u) / grid : 0u;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&ctl->tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // ---- set-up: strip table (its layout and the order of its slots are those of staged.cuh), barriers ----
    {
        const uint32_t spr = s.W >> 2;
        const uint32_t full_bands = p.pl.uniform ? p.pl.G : (p.pl.G / s.Hb) * (s.Hb - 1u);
        for (uint32_t sl = threadIdx.x; sl < nf * MS * 32u; sl += blockDim.x) {
            uint32_t ob, q;
            if (p.pl.paired) {
                const uint32_t pair = sl / (2u * spr), r = sl - pair * 2u * spr;
                const uint32_t two = 2u * (spr - 1u);
                if (r < two) {
                    const uint32_t t = r >> 1, per = (spr - 1u) >> 1;
                    const uint32_t wb = t / per;
                    ob = 2u * pair + wb;
                    q = 2u * (t - wb * per) + (r & 1u);
                } else {
                    ob = 2u * pair + (r - two);
                    q = spr - 1u;
                }
            } else {
                ob = sl / p.pl.spb;
                q = sl - ob * p.pl.spb;
            }
            uint32_t band;
            if (p.pl.uniform) band = ob;
            else if (ob < full_bands) band = ob + ob / (s.Hb - 1u);
            else band = (ob - full_bands) * s.Hb + (s.Hb - 1u);
            const bool ok = sl < p.pl.slots && 4u * q < s.W;
            uint32_t eoff, rows;
            if (p.pl.uniform) {
                eoff = band * s.B * s.W + 4u * q;
                rows = s.B;
            } else {
                const uint32_t pl_ = band / s.Hb, bh = band - pl_ * s.Hb;
                eoff = pl_ * s.HW + bh * s.B * s.W + 4u * q;
                rows = (bh + 1u == s.Hb) ? p.tail_rows : s.B;
            }
            const uint32_t bw = q / LPT;
            const uint32_t which = ((rows != s.B) ? 2u : 0u) + ((bw == s.Wb - 1u && (s.W % s.B) != 0u) ? 1u : 0u);
            const uint32_t writer = (q % LPT) == 0 ? 1u : 0u;
            const uint32_t mate = (LPT == 2u && !(p.pl.paired && q == spr - 1u)) ? 1u : 0u;
            table[sl] = (ok ? (eoff >> 2) : 0u) | ((ok ? rows : 0u) << 13) | (which << 17) | (writer << 19) | (mate << 20) |
                        ((ok ? band * s.Wb + bw : 0u) << 21);
        }
    }
    for (uint32_t i = threadIdx.x; i < PARK_CHUNKS; i += blockDim.x) {
        mbar_init(&ctl->full[i], 1);
        mbar_init(&ctl->folded[i], nf);
        mbar_init(&ctl->par[i], 1);
        if (i < PARK_MAX_STAGES) mbar_init(&ctl->empty[i], nf);
        ctl->kmin[i] = 0u;
        ctl->kmax[i] = 0u;
        if (i == 0) ctl->failed = 0u;
        fence_barrier_init();
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    griddep_wait();
    griddep_launch();

    if (warp == 0) {
        // ---- producer ----
        if (lane == 0) {
            const uint64_t policy = l2_policy_release();
            const uint32_t ahead = p.pl.ahead;
            uint32_t it = 0;
            for (; it < n_my; ++it) {
                const uint32_t turn = fdiv(it, p.by_stages), st = it - turn * K, slot = it % PARK_CHUNKS;
                const uint32_t j = blockIdx.x + it * grid;
                const uint32_t n = fdiv(j, p.by_S), k = j - n * S;
                if ((it >= K && !p_wait(&ctl->empty[st], (turn - 1u) & 1u, p, ctl, 0x80000002u)) ||
                    (it >= ahead && !p_wait(&ctl->full[(it - ahead) % PARK_CHUNKS], ((it - ahead) / PARK_CHUNKS) & 1u, p, ctl, 0x80000005u))) break;
                const uint32_t e0 = k * p.pl.chunk_elems;
                const uint32_t bytes = min(p.pl.chunk_elems, s.CHW - e0) * (uint32_t)sizeof(XT);
                ParkDesc d;
                d.lfc0 = (uint64_t)n * s.C * s.TPP + k * p.pl.G * s.Wb;
                d.quad0 = ((uint64_t)n * s.CHW + e0) >> 2;
                d.ctr0 = rng_sample_base(p.seed, n) + K_GROUP * (uint64_t)((e0 >> 2) + 1u);
                d.ntiles = min(p.pl.G, p.pl.bands_per_sample - k * p.pl.G) * s.Wb;
                d.n = n;
                ctl->desc[slot] = d;
                mbar_arrive_expect_tx(&ctl->full[slot], bytes);
                bulk_load_hint(ring + (size_t)st * p.pl.stage_bytes, reinterpret_cast<const XT*>(p.x) + d.quad0 * 4u, bytes, &ctl->full[slot], policy);
            }
            // the copies on their way land before the CTA may exit, whoever gives up meanwhile (the workers need them all in any case)
            for (uint32_t t = it > K ? it - K : 0u; t < it; ++t) {
                uint32_t polls = 0;
                while (!mbar_try_wait(&ctl->full[t % PARK_CHUNKS], (t / PARK_CHUNKS) & 1u) && ++polls < (1u << 20)) {
                }
            }
        }
    } else if (warp == 1 || warp >= 3 && warp < (uint32_t)PARK_SERVICE_WARPS) {
        // ---- publisher: folds the chunks' extremes into the samples' slots ----
        const uint32_t me = warp == 1 ? 0u : warp - 2u;
        uint32_t next = me, polls = 0;
        SWait w = {0, 0};
        while (next < n_my) {
            const uint32_t it = next + lane * PARK_PUBLISHERS, slot = it % PARK_CHUNKS;
            const bool ready = lane < 4u && it < n_my && mbar_try_wait(&ctl->folded[slot], (it / PARK_CHUNKS) & 1u);
            const uint32_t missing = ~__ballot_sync(0xFFFFFFFFu, ready);
            const uint32_t got = missing ? (uint32_t)__ffs(missing) - 1u : 32u;
            if (got) {
                if (lane < got) {
                    // the folds are ordered before the count, which the watchers read with acquire
                    uint32_t* g = p.ws + WS_HEADER_WORDS + (size_t)ctl->desc[slot].n * WS_SLOT_WORDS;
                    red_max_relaxed(g + 0, ctl->kmin[slot]);
                    red_max_relaxed(g + 1, ctl->kmax[slot]);
                    ctl->kmin[slot] = 0u;
                    ctl->kmax[slot] = 0u;
                    fence_acq_rel_gpu();
                    red_add_relaxed(g + 2, 1u);
                }
                __syncwarp();
                next += got * PARK_PUBLISHERS;
                polls = 0;
                w.c0 = 0;
            } else if ((++polls & 7u) == 0) {
                const bool bad = lane == 0 && p_give_up(p, ctl, w);
                if (__any_sync(0xFFFFFFFFu, bad)) {
                    if (lane == 0) p_record(p, ctl, 0x80000003u);
                    break;
                }
            }
        }
    } else if (warp == 2) {
        // ---- watcher ----
        constexpr uint32_t WIN = 2;
        uint32_t it = lane < WIN ? lane : n_my;
        uint32_t polls = 0;
        SWait w = {0, 0};
        while (true) {
            bool done = false;
            if (it < n_my) {
                const uint32_t j = blockIdx.x + it * grid, n = fdiv(j, p.by_S), slot = it % PARK_CHUNKS;
                const uint32_t* g = p.ws + WS_HEADER_WORDS + (size_t)n * WS_SLOT_WORDS;
                if (ld_acquire_u32(g + 2) == p.expected_chunks) {
                    const uint64_t keys = ld_relaxed_u64(reinterpret_cast<const uint64_t*>(g));
                    const float rmax = key_float((uint32_t)(keys >> 32));
                    const QParams qp = make_qparams(key_float(~(uint32_t)keys), rmax, Q);
                    ctl->delta[slot] = qp.delta;
                    ctl->scale[slot] = tagged_scale<Q>(qp, rmax);
                    mbar_arrive(&ctl->par[slot]);
                    if (j - n * S == 0u) {
                        p.stats[2 * (size_t)n + 0] = qp.delta;
                        p.stats[2 * (size_t)n + 1] = qp.step;
                    }
                    it += WIN;
                    done = true;
                }
            }
            if (!__any_sync(0xFFFFFFFFu, it < n_my)) break;
            if (__any_sync(0xFFFFFFFFu, done)) {
                polls = 0;
                w.c0 = 0;
            } else if ((++polls & 7u) == 0) {
                const bool bad = lane == 0 && p_give_up(p, ctl, w);
                if (__any_sync(0xFFFFFFFFu, bad)) {
                    if (lane == 0) p_record(p, ctl, 0x80000004u);
                    break;
                }
            }
        }
    } else {
        const uint32_t worker = warp - PARK_SERVICE_WARPS, set = worker / nf, k = worker - set * nf;
        if (set < p.pl.sets) {
            uint32_t rec[MS];
            bool whole = true;
#pragma unroll
            for (int m = 0; m < MS; ++m) {
                rec[m] = table[(k * MS + m) * 32u + lane];
                const uint32_t rows = (rec[m] >> 13) & 15u;
                whole = whole && (rows == (uint32_t)P2 || rows == 0u);
            }
            const uint32_t tm = ctl->tmem + ((warp & 3u) << 21) + (worker >> 2) * (32u * PARK_DEPTH);      // lane 32 * quarter; its own columns
            if (__all_sync(0xFFFFFFFFu, whole)) park_work<XT, LT, P2, Q, true>(p, ctl, ring, n_my, set, rec, tm);
            else park_work<XT, LT, P2, Q, false>(p, ctl, ring, n_my, set, rec, tm);
        }
    }
    __syncwarp();
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    __syncwarp();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(ctl->tmem));
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
template <typename XT, typename LT, int P2, int Q>
static div_status launch_park(const ParkParams& prm, cudaStream_t st) {
    auto kern = park_kernel<XT, LT, P2, Q>;
    static SmemSeen smem_set[DEVICE_CACHE_SLOTS];
    if (!ensure_dynamic_smem((const void*)kern, (int)prm.pl.smem_bytes, smem_set)) return DIV_ERR_CUDA;
    void* args[] = {(void*)&prm};
    return launch_coop((const void*)kern, dim3(prm.pl.grid), PARK_THREADS, prm.pl.smem_bytes, st, args) ? DIV_OK : DIV_ERR_CUDA;
}
template <typename XT, typename LT>
static div_status launch_park_q(const ParkParams& prm, int qbits, cudaStream_t st) {
    if (prm.s.P2 == 8) return qbits == 2 ? launch_park<XT, LT, 8, 2>(prm, st) : qbits == 4 ? launch_park<XT, LT, 8, 4>(prm, st) : launch_park<XT, LT, 8, 8>(prm, st);
    return qbits == 2 ? launch_park<XT, LT, 4, 2>(prm, st) : qbits == 4 ? launch_park<XT, LT, 4, 4>(prm, st) : launch_park<XT, LT, 4, 8>(prm, st);
}

div_status compress_park(const div_desc* d, const Shape& s, const div_layout& lo, const ParkPlan& pl, const void* x, uint8_t* blob, uint32_t* ws,
                         uint64_t seed, cudaStream_t st, uint32_t expected_chunks, uint64_t timeout_ns, uint32_t more_smem) {
    ParkParams p;
    p.s = s;
    p.pl = pl;
    p.pl.smem_bytes += more_smem;
    p.by_S = host_fastdiv(pl.chunks_per_sample);
    p.by_stages = host_fastdiv(pl.stages);
    p.x = x;
    p.lfc = blob + lo.lfc_off;
    p.packed = blob + lo.packed_off;
    p.stats = reinterpret_cast<float*>(blob + lo.stats_off);
    p.ws = ws;
    p.seed = seed;
    p.rng_row_step = K_GROUP * (uint64_t)(s.W / 4u);
    p.timeout_ns = timeout_ns ? timeout_ns : 2000000000ull;
    p.expected_chunks = expected_chunks ? expected_chunks : pl.chunks_per_sample;
    p.tail_rows = s.H - (s.Hb - 1u) * s.B;
    const uint32_t tail_cols = s.W - (s.Wb - 1u) * s.B;
    for (int i = 0; i < 4; ++i) {
        const uint32_t cnt = ((i & 2) ? p.tail_rows : s.B) * ((i & 1) ? tail_cols : s.B);
        p.cnt[i] = (float)cnt;
        p.inv_cnt[i] = (cnt & (cnt - 1)) == 0 ? 1.0f / (float)cnt : 0.f;
    }
    typedef __nv_bfloat16 bf16;
    if (d->x_dtype == DIV_F32) return d->lfc_dtype == DIV_F32 ? launch_park_q<float, float>(p, d->qbits, st) : launch_park_q<float, bf16>(p, d->qbits, st);
    return d->lfc_dtype == DIV_F32 ? launch_park_q<bf16, float>(p, d->qbits, st) : launch_park_q<bf16, bf16>(p, d->qbits, st);
}

}  // namespace divk
