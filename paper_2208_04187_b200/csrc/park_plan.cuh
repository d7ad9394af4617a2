// Launch shapes of the parking kernel (park.cu).
#pragma once

#include "fused.cuh"      // DeviceInfo, host_fastdiv

namespace divk {

constexpr uint32_t PARK_PUBLISHERS = 2;                     // (one: 64 x 512 x 28 x 28 32.4 instead of 31.3 us)
constexpr int PARK_SERVICE_WARPS = 2 + (int)PARK_PUBLISHERS;
// Workers in each quarter of tensor memory (a warp reaches the quarter of its number modulo 4), and the units of 32 columns that each
// keeps there.  64 x 64 x 112 x 112, 64 x 512 x 28 x 28, bfloat16 128 x 160 x 32 x 32: 7 workers and 2 units 45.4, 31.1, 25.4 us; 5 and 3 50.2, 36.1, 27.2.
constexpr uint32_t PARK_PER_QUARTER = 7, PARK_DEPTH = 2;
constexpr uint32_t PARK_WORKERS = 4 * PARK_PER_QUARTER;
static_assert(PARK_PER_QUARTER * PARK_DEPTH * 32 <= 512, "columns of tensor memory");
constexpr int PARK_THREADS = 32 * (PARK_SERVICE_WARPS + (int)PARK_WORKERS);
// with 64 registers a thread a CTA fills an SM: whoever else uses tensor memory has left it by then, and nobody ever waits for some
static_assert(PARK_THREADS == 1024, "a CTA takes every register of its SM");
constexpr int PARK_MAX_STAGES = 16;
constexpr uint32_t PARK_CHUNKS = 64;           // chunk records of a CTA: more than can be on their way at once (see park.cu)
static_assert(PARK_MAX_STAGES < PARK_CHUNKS, "a record is not filled again while the chunk in it is on its way");
constexpr uint32_t PARK_MAX_SETS = (PARK_CHUNKS - 1 - PARK_MAX_STAGES) / PARK_DEPTH;
constexpr uint32_t PARK_CHUNK_ELEMS = 7168;    // of a full chunk, about: 7 units (half of it: 64 x 64 x 112 x 112 44 -> 52 us)
constexpr uint32_t PARK_MOST_BYTES = 64 * 1024;// planes up to which chunks may be larger, where a chunk has to be whole planes
// Bytes of copies on their way to an SM at once, in whole chunks, of which at least two are (56 KB for full fp32 chunks, up to 128 KB where a
// chunk is a large plane).  The words by which the CTAs meet come back behind them: 64 x 64 x 112 x 112 with 28, 56, 84, 112 KB and all of
// the ring 57.5, 45.5, 47.4, 49.6, 50.9 us.
constexpr uint32_t PARK_AHEAD_BYTES = 48 * 1024;

struct ParkPlan {
    uint32_t grid, smem_bytes;
    uint32_t stages;               // of the landing ring
    uint32_t G;                    // bands per full chunk
    uint32_t spb;                  // strips per band
    uint32_t paired;               // bands are laid out in pairs (see the table in park.cu)
    uint32_t uniform;              // every band has B rows
    uint32_t slots;                // strip slots per full chunk
    uint32_t nf;                   // units per full chunk
    uint32_t ahead;                // copies on their way at once
    uint32_t sets;                 // chunks that the workers take at once, a worker per unit
    uint32_t per_cta;              // chunks of a sample that one CTA may have
    uint32_t chunk_elems, chunks_per_sample, bands_per_sample, total_chunks, stage_bytes;
};

// Its time in ns, fitted to 550 maps of 4 to 205 MB and 124 of small samples: the units of an SM, how often its workers go round (no oftener than
// the watcher learns of a chunk, two in about 0.9 us), the bytes, and how far a sample is spread.
inline uint64_t park_ns(const ParkPlan& pl) {
    const uint64_t rounds = (pl.total_chunks + pl.grid - 1u) / pl.grid;
    const uint64_t turn = 1930u / pl.sets > 450u ? 1930u / pl.sets : 450u;
    return 7640u + (34u * pl.nf + turn) * rounds + rounds * pl.stage_bytes * 148u / 29700u + 420u * pl.chunks_per_sample / 148u;
}

// what the producer posts for a chunk
struct ParkDesc {
    uint64_t lfc0;                 // its first tile in the tensor
    uint64_t quad0;                // its first group of 4 elements in the tensor
    uint64_t ctr0;                 // counter of the random stream of that group
    uint32_t ntiles;
    uint32_t n;                    // sample
};
struct ParkCtl {
    uint64_t full[PARK_CHUNKS];    // the chunk has landed
    uint64_t folded[PARK_CHUNKS];  // all its units are reduced
    uint64_t par[PARK_CHUNKS];     // its sample's parameters are there
    uint64_t empty[PARK_MAX_STAGES];
    ParkDesc desc[PARK_CHUNKS];
    float delta[PARK_CHUNKS], scale[PARK_CHUNKS];
    uint32_t kmin[PARK_CHUNKS], kmax[PARK_CHUNKS];
    uint32_t failed, tmem;
};

inline bool plan_park(const div_desc* d, const Shape& s, ParkPlan* out) {
    const uint32_t sx = d->x_dtype == DIV_F32 ? 4u : 2u;
    if (s.W % 4 != 0 || !(s.B == 4 || s.B == 8) || s.P2 != s.B || d->qbits == 1) return false;
    // bulk copies start on 16-byte boundaries and move multiples of 16 bytes
    if (((uint64_t)s.CHW * sx) % 16u != 0 || ((uint64_t)s.HW * sx) % 16u != 0 || ((uint64_t)s.B * s.W * sx) % 16u != 0) return false;
    const DeviceInfo di = device_info();
    if (!di.ok || di.sms < 1) return false;
    ParkPlan pl = ParkPlan();
    pl.spb = s.W / 4u;
    pl.paired = (s.P2 == 8u && (pl.spb & 1u)) ? 1u : 0u;
    const uint64_t bands = (uint64_t)s.C * s.Hb;
    if (bands >= (1ull << 31)) return false;
    pl.bands_per_sample = (uint32_t)bands;
    pl.uniform = (s.H % s.B == 0) ? 1u : 0u;
    const uint32_t per_unit = 32u * (8u / s.P2);
    const uint32_t geo1 = pl.uniform ? 1u : s.Hb;
    const uint32_t geo = (pl.paired && (geo1 & 1u)) ? 2u * geo1 : geo1;
    const uint64_t geo_bytes = (pl.uniform ? (uint64_t)s.B * s.W * sx : (uint64_t)s.HW * sx) * (geo / geo1);
    const uint32_t fill = per_unit / gcd_u32(per_unit, pl.spb);
    const uint32_t both = lcm_u32(geo, fill);
    const uint64_t both_bytes = geo_bytes * (both / geo);
    const uint64_t target = (uint64_t)PARK_CHUNK_ELEMS * sx;
    uint32_t G;
    if (both_bytes <= target) G = (uint32_t)(target / both_bytes) * both;
    else if (geo_bytes <= target) G = (uint32_t)(target / geo_bytes) * geo;
    else if (geo_bytes <= PARK_MOST_BYTES) G = geo;
    else return false;
    const uint32_t bands_up = (pl.bands_per_sample + geo - 1u) / geo * geo;
    if (G > bands_up) G = bands_up;
    pl.G = G;
    pl.slots = G * pl.spb;
    if (pl.slots > 4096u || G * s.Wb > 2048u) return false;
    pl.nf = (pl.slots + per_unit - 1u) / per_unit;
    pl.chunk_elems = pl.uniform ? G * s.B * s.W : (G / s.Hb) * s.HW;
    if (pl.chunk_elems >= (1u << 15)) return false;
    pl.chunks_per_sample = (pl.bands_per_sample + G - 1u) / G;
    pl.stage_bytes = (pl.chunk_elems * sx + 127u) & ~127u;
    const uint32_t fixed = pl.nf * per_unit * 4u + (uint32_t)sizeof(ParkCtl) + 128u;
    if ((uint32_t)di.smem_optin < fixed + 2u * pl.stage_bytes) return false;
    pl.stages = ((uint32_t)di.smem_optin - fixed) / pl.stage_bytes;
    if (pl.stages > (uint32_t)PARK_MAX_STAGES) pl.stages = PARK_MAX_STAGES;
    pl.smem_bytes = pl.stages * pl.stage_bytes + fixed;
    pl.ahead = PARK_AHEAD_BYTES / pl.stage_bytes;
    if (pl.ahead < 2u) pl.ahead = 2u;
    if (pl.ahead > pl.stages) pl.ahead = pl.stages;            // (more copies are never on their way)
    const uint64_t total = (uint64_t)pl.chunks_per_sample * s.N;
    if (total >= (1ull << 30)) return false;
    pl.total_chunks = (uint32_t)total;
    pl.grid = total < (uint64_t)di.sms ? (uint32_t)total : (uint32_t)di.sms;
    if (pl.nf > PARK_WORKERS) return false;
    pl.sets = PARK_WORKERS / pl.nf;
    if (pl.sets > PARK_MAX_SETS) pl.sets = PARK_MAX_SETS;
    // a CTA's units of one sample are all parked at once
    const uint32_t per_cta = (pl.chunks_per_sample - 1u) / pl.grid + 1u;
    pl.per_cta = per_cta;
    if (per_cta > PARK_DEPTH * pl.sets) return false;
    *out = pl;
    return true;
}

div_status compress_park(const div_desc* d, const Shape& s, const div_layout& lo, const ParkPlan& pl, const void* x, uint8_t* blob, uint32_t* ws,
                         uint64_t seed, cudaStream_t st, uint32_t expected_chunks = 0, uint64_t timeout_ns = 0, uint32_t more_smem = 0);

}  // namespace divk
