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
constexpr uint32_t PARK_MAX_SETS = (PARK_CHUNKS - 1 - PARK_MAX_STAGES) / PARK_DEPTH;
constexpr uint32_t PARK_CHUNK_ELEMS = 7168;    // of a full chunk, about: 7 units (half of it: 64 x 64 x 112 x 112 44 -> 52 us)
constexpr uint32_t PARK_MOST_BYTES = 64 * 1024;// planes up to which chunks may be larger, where a chunk has to be whole planes
// Bytes of copies on their way to an SM at once.  The words by which the CTAs meet come back behind them: 64 x 64 x 112 x 112 with 28, 56,
// 84, 112 KB and all of the ring 57.5, 45.5, 47.4, 49.6, 50.9 us.
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

// Its time in ns, fitted to 550 maps of 4 to 205 MB (within 10 % for nine in ten): the units of an SM, how often its workers go round, the
// bytes, and how far a sample is spread.
inline uint64_t park_ns(const ParkPlan& pl) {
    const uint64_t rounds = (pl.total_chunks + pl.grid - 1u) / pl.grid;
    return 6640u + 34u * rounds * pl.nf + 1930u * rounds / pl.sets + rounds * pl.stage_bytes * 148u / 29700u + 420u * pl.chunks_per_sample / 148u;
}

bool plan_park(const div_desc* d, const Shape& s, ParkPlan* out);
div_status compress_park(const div_desc* d, const Shape& s, const div_layout& lo, const ParkPlan& pl, const void* x, uint8_t* blob, uint32_t* ws,
                         uint64_t seed, cudaStream_t st, uint32_t expected_chunks = 0, uint64_t timeout_ns = 0);

}  // namespace divk
