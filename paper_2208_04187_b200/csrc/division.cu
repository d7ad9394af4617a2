// Host side of the C ABI declared in include/division.h: argument checks, byte-layout arithmetic,
// kernel selection and launches.  Nothing here allocates device memory; the only device memory the library
// owns is the fixed scratch array of div_compress_static.
#include "../../include/division.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "cluster_plan.cuh"
#include "common.cuh"
#include "decompress.cuh"
#include "fused.cuh"
#include "fused_v.cuh"
#include "lagged.cuh"
#include "lines.cuh"
#include "masks.cuh"
#include "park_plan.cuh"
#include "planegroup.cuh"
#include "planes.cuh"
#include "staged.cuh"
#include "twopass.cuh"
#include "volume.cuh"

namespace {

using namespace divk;
typedef __nv_bfloat16 bf16;

constexpr uint64_t SECTION_ALIGN = 128;
constexpr uint32_t DIV_FLAG_ALL = DIV_FLAG_FORCE_TWO_PASS | DIV_FLAG_NO_STRIP_KERNEL | DIV_FLAG_NO_LAGGED_KERNEL |
                                  DIV_FLAG_NO_PLANE_KERNELS | DIV_FLAG_NO_LINE_KERNELS | DIV_FLAG_NO_STAGED_KERNEL |
                                  DIV_FLAG_TWO_LAUNCH_PLANES | DIV_FLAG_NO_PARK_KERNEL;

inline uint64_t align_up(uint64_t v, uint64_t a) { return (v + a - 1) / a * a; }
inline uint32_t dtype_bytes(int32_t dt) { return dt == DIV_F32 ? 4u : 2u; }

div_status check_desc(const div_desc* d) {
    if (!d) return DIV_ERR_NULL;
    if (d->n < 1 || d->c < 1 || d->h < 1 || d->w < 1) return DIV_ERR_SHAPE;
    if (d->n >= (1ll << 31) || d->c >= (1ll << 32) || d->h >= (1ll << 32) || d->w >= (1ll << 32)) return DIV_ERR_SHAPE;
    // c*h*w < 2^32 (width of the random-number counter), checked without overflow
    const unsigned __int128 chw = (unsigned __int128)d->c * (unsigned __int128)d->h * (unsigned __int128)d->w;
    if (chw >= ((unsigned __int128)1 << 32)) return DIV_ERR_SHAPE;
    if (d->block < 1) return DIV_ERR_PARAM;
    if (!(d->qbits == 1 || d->qbits == 2 || d->qbits == 4 || d->qbits == 8)) return DIV_ERR_PARAM;
    if (!(d->x_dtype == DIV_F32 || d->x_dtype == DIV_BF16)) return DIV_ERR_PARAM;
    if (!(d->lfc_dtype == DIV_F32 || d->lfc_dtype == DIV_BF16)) return DIV_ERR_PARAM;
    return DIV_OK;
}

Shape make_shape(const div_desc* d) {
    Shape s;
    s.N = (uint32_t)d->n;
    s.C = (uint32_t)d->c;
    s.H = (uint32_t)d->h;
    s.W = (uint32_t)d->w;
    // a block larger than both sides behaves like a block equal to the larger side
    const uint32_t big = s.H > s.W ? s.H : s.W;
    s.B = (uint32_t)d->block > big ? big : (uint32_t)d->block;
    s.Hb = (s.H + s.B - 1) / s.B;
    s.Wb = (s.W + s.B - 1) / s.B;
    s.P2 = 1;
    while (s.P2 < s.B) s.P2 <<= 1;
    s.HW = s.H * s.W;
    s.CHW = s.C * s.HW;
    s.TPP = s.Hb * s.Wb;
    s.total = (uint64_t)s.N * s.CHW;
    s.tiles = (uint64_t)s.N * s.C * s.TPP;
    return s;
}

void make_layout(const div_desc* d, const Shape& s, div_layout* out) {
    out->lfc_off = 0;
    out->lfc_bytes = s.tiles * dtype_bytes(d->lfc_dtype);
    out->packed_off = align_up(out->lfc_bytes, SECTION_ALIGN);
    // ceil(total*Q/32) words; total*Q < 2^31 * 2^32 * 8 fits in 64 bits
    out->packed_bytes = ((s.total * (uint64_t)d->qbits + 31) / 32) * 4;
    out->stats_off = align_up(out->packed_off + out->packed_bytes, SECTION_ALIGN);
    out->stats_bytes = 8ull * s.N;
    out->total_bytes = out->stats_off + out->stats_bytes;
    out->closed_form_bytes = out->lfc_bytes + out->packed_bytes + out->stats_bytes;
    out->raw_bytes = s.total * dtype_bytes(d->x_dtype);
    out->workspace_bytes = align_up(4ull * (WS_HEADER_WORDS + (uint64_t)WS_SLOT_WORDS * s.N), 256);
}

// per-plane groups: the same sections, but the stats section holds one bfloat16 pair (4 bytes) per plane and
// no scratch is needed
void make_layout_pg(const div_desc* d, const Shape& s, div_layout* out) {
    make_layout(d, s, out);
    out->stats_bytes = 4ull * s.N * s.C;
    out->total_bytes = out->stats_off + out->stats_bytes;
    out->closed_form_bytes = out->lfc_bytes + out->packed_bytes + out->stats_bytes;
    out->workspace_bytes = 0;
}
inline bool pg_shape_ok(const Shape& s) { return (uint64_t)s.N * s.C < (1ull << 31); }
inline bool pg_decompress_flat_ok(const Shape& s) {
    return (s.total % 4 == 0) && s.HW <= FLAT_MAX_HW && s.TPP <= 65535 && s.total / 4096 < 0x7FFFFFFFull;
}

FastDiv make_fastdiv(uint32_t d) {
    FastDiv f;
    f.d = d;
    uint32_t s = 0;
    while ((1ull << s) < d) ++s;
    f.shift = 31 + s;
    f.mul = (uint32_t)((((1ull << f.shift) - 1) / d) + 1);
    return f;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ------------------------------------------------------------------------------------------
// dispatch helpers: runtime (dtype, dtype, Q) -> template instance
// ------------------------------------------------------------------------------------------
template <typename F>
div_status dispatch_q(int qbits, F&& f) {
    switch (qbits) {
        case 1: return f(std::integral_constant<int, 1>());
        case 2: return f(std::integral_constant<int, 2>());
        case 4: return f(std::integral_constant<int, 4>());
        case 8: return f(std::integral_constant<int, 8>());
    }
    return DIV_ERR_PARAM;
}
template <typename F>
div_status dispatch_types(int x_dtype, int lfc_dtype, F&& f) {
    if (x_dtype == DIV_F32) {
        if (lfc_dtype == DIV_F32) return f((float*)nullptr, (float*)nullptr);
        return f((float*)nullptr, (bf16*)nullptr);
    }
    if (lfc_dtype == DIV_F32) return f((bf16*)nullptr, (float*)nullptr);
    return f((bf16*)nullptr, (bf16*)nullptr);
}

inline div_status launch_status() { return cudaGetLastError() == cudaSuccess ? DIV_OK : DIV_ERR_CUDA; }

// ------------------------------------------------------------------------------------------
// two-pass compress
// ------------------------------------------------------------------------------------------
div_status compress_two_pass(const div_desc* d, const Shape& s, const div_layout& lo, const void* x, uint8_t* blob,
                             uint32_t* ws, uint64_t seed, cudaStream_t st) {
    const uint64_t nwords = lo.packed_bytes / 4;
    const uint64_t g1 = (s.tiles + 255) / 256, g2 = (nwords + 255) / 256;
    if (g1 > 0x7FFFFFFFull || g2 > 0x7FFFFFFFull) return DIV_ERR_SHAPE;
    return dispatch_types(d->x_dtype, d->lfc_dtype, [&](auto* xt, auto* lt) -> div_status {
        typedef std::remove_pointer_t<decltype(xt)> XT;
        typedef std::remove_pointer_t<decltype(lt)> LT;
        lfc_stats_kernel<XT, LT><<<(unsigned)g1, 256, 0, st>>>((const XT*)x, (LT*)(blob + lo.lfc_off), ws, s);
        if (launch_status() != DIV_OK) return DIV_ERR_CUDA;
        return dispatch_q(d->qbits, [&](auto q) -> div_status {
            quant_pack_kernel<XT, LT, decltype(q)::value><<<(unsigned)g2, 256, 0, st>>>(
                (const XT*)x, (const LT*)(blob + lo.lfc_off), ws, (uint32_t*)(blob + lo.packed_off),
                (float*)(blob + lo.stats_off), s, seed, nwords);
            return launch_status();
        });
    });
}

// ------------------------------------------------------------------------------------------
// decompress
// ------------------------------------------------------------------------------------------
constexpr int DEC_QPT = 4;
#ifndef DIVK_FLAT_QPT
#define DIVK_FLAT_QPT 8
#endif
constexpr int FLAT_QPT = DIVK_FLAT_QPT;       // quads per thread of the flat decompress kernel

// Which compress kernels run a descriptor that the cluster kernel (choose_cluster below, asked first) leaves to them, and all
// descriptors where flags exclude it.  Measured on the ResNet / WRN / DenseNet-shaped maps: from about
// 56 MB up with 8 x 8 blocks the staged kernel is fastest (both reads of x staged through shared memory by bulk
// copies), from about 20 MB up the lagged kernel (plain loads, several bands per lane, cheap for small strips),
// below that the strip ring kernel (shorter start-up); the general kernels take what those three cannot.
bool prefer_staged(const div_desc* d, const Shape& s) {
    return s.B == 8 && s.total * dtype_bytes(d->x_dtype) >= (56ull << 20);
}
// Maps whose planes are narrow enough for the fused small-plane kernel (W <= 32 for B = 8): measured faster than the
// strip ring and lagged kernels below 56 MiB (32 x 32 fp32, 34 MB: 19.5 against 25.8 us; 28 x 28, 58 MB: 29.7 against
// 37.0 us; 8 x 8 bf16, 10 MB: 15.2 against 20.4 us), except for bfloat16 maps from 32 MiB up (lagged 36 against 38 - 40 us).
bool prefer_planes(const div_desc* d, const Shape& s) {
    const uint64_t bytes = s.total * dtype_bytes(d->x_dtype);
    return bytes < (56ull << 20) && !(d->x_dtype == DIV_BF16 && bytes >= (32ull << 20));
}
bool prefer_lagged(const div_desc* d, const Shape& s) {
    return s.total * dtype_bytes(d->x_dtype) >= (20ull << 20);
}

struct Choice {
    int code;          // the value div_plan.fused reports
    LineGeom lg;
    SPlan sp;
    LPlan lp;
    VPlan vp;
    PlaneGeom pg;
    PlaneFusedPlan pf;
    LineFused lf;
    FusedPlan fp;
};

void choose_compress(const div_desc* d, const Shape& s, uint32_t flags, Choice* c) {
    const bool two_pass = (flags & DIV_FLAG_FORCE_TWO_PASS) != 0;
    c->code = 0;
    if (two_pass) return;
    if (!(flags & DIV_FLAG_NO_LINE_KERNELS) && plan_lines(d, s, &c->lg)) {
        c->code = (!(flags & DIV_FLAG_TWO_LAUNCH_PLANES) && line_fused_applies(d, s, c->lg, &c->lf)) ? 8 : 5;
        return;
    }
    const bool may_staged = !(flags & DIV_FLAG_NO_STAGED_KERNEL);
    const bool may_lag = !(flags & DIV_FLAG_NO_LAGGED_KERNEL);
    const bool may_strip = !(flags & DIV_FLAG_NO_STRIP_KERNEL);
    // (the preference holds only while no strip kernel is excluded: a flag set that leaves one of them in line gets it)
    if (may_staged && may_lag && may_strip && !(flags & (DIV_FLAG_NO_PLANE_KERNELS | DIV_FLAG_TWO_LAUNCH_PLANES)) &&
        prefer_planes(d, s) && plan_planes(d, s, &c->pg) && plane_fused_applies(d, s, c->pg, &c->pf)) {
        c->code = 7;
        return;
    }
    if (may_staged && prefer_staged(d, s) && plan_staged(d, s, &c->sp) == DIV_OK) {
        c->code = 6;
        return;
    }
    if (may_lag && prefer_lagged(d, s) && plan_lagged(d, s, &c->lp) == DIV_OK) {
        c->code = 3;
        return;
    }
    if (may_strip && plan_v(d, s, &c->vp) == DIV_OK) {
        c->code = 2;
        return;
    }
    if (may_lag && plan_lagged(d, s, &c->lp) == DIV_OK) {
        c->code = 3;
        return;
    }
    if (may_staged && plan_staged(d, s, &c->sp) == DIV_OK) {
        c->code = 6;
        return;
    }
    if (!(flags & DIV_FLAG_NO_PLANE_KERNELS) && plan_planes(d, s, &c->pg)) {
        c->code = (!(flags & DIV_FLAG_TWO_LAUNCH_PLANES) && plane_fused_applies(d, s, c->pg, &c->pf)) ? 7 : 4;
        return;
    }
    if (plan_fused(d, s, &c->fp) == DIV_OK) c->code = 1;
}

// Where the clusters of a map have to take turns, or keep much of the device idle (a single large sample), a kernel that
// spreads the map over the whole device and reads x a second time may be faster.  Both measured on 1217 maps (1 to 192 samples of
// 3 x 224 x 224 to 2048 x 7 x 7, up to 52 M elements, both types):
//   * kernels for planes a warp wide (7, 4) are not within 2 turns (0.45 - 0.97 of their time), nor in any number of them for fp32 blocks
//     up to 8 of which two shares fit an SM (192 x 512 x 19 x 19 0.76).  Else they are: 64 x 1984 x 32 x 8 with B = 16 120 against 71 us in 10;
//     bfloat16, whose residuals take three times the room of x where it is not read 4 columns at a time, 64 x 1024 x 14 x 14 31.3 against
//     26.9 us in 5.  With one share of fp32 per SM blocks of 4 are not (8 x 760 x 31 x 31 23 against 33 us), nor those of 8 in one turn (2 x
//     936 x 32 x 23 11.2 against 14.1 us); in more, and for large shares of blocks of 16, it depends (128 x 1880 x 7 x 7 24 against 27 us in 2,
//     24 x 2048 x 17 x 17 53 against 43 us in 4, 1 x 1064 x 28 x 28 with B = 16 12.8 against 10.4 us): both times are estimated, in ns;
//   * the strip kernels (2, 3, 6) are not within 2 turns of which every SM holds two shares (or one of fp32), but where a share is large and
//     the batch small (1 x 64 x 112 x 112 bfloat16 9.9 against 8.4 us) or the turns are many (64 x 64 x 112 x 112 89 against 60 us).  There
//     both times are estimated; of 453 maps the estimates give 2 to the cluster that it takes 3 - 4 % longer for, and 10 to the others that
//     these take 6 - 23 % longer for;
//   * the general kernels never were (32 x 64 x 75 x 75 27 against 82 us).
uint64_t cluster_ns(const Shape& s, const ClusterPlan& pl) {
    const uint64_t share = (uint64_t)pl.ppc * s.HW, wider = pl.vw == 4u ? 10u : pl.vw == 2u ? 12u : 13u;      // narrow accesses take longer
    return 2400u + pl.turns64 * (1500u + share * (115u * pl.load + 30u) * wider / 10000u) / 64u;
}
uint64_t other_ns(const Shape& s, int code) {
    return code == 7 || code == 4 ? 8000u + s.total * 14u / 10000u : code == 2 ? 7600u + s.total * 15u / 10000u
         : code == 3 ? 15500u + s.total * 105u / 100000u : 14800u + s.total * 87u / 100000u;
}
bool cluster_pays(const div_desc* d, const Shape& s, const ClusterPlan& pl) {
    const uint64_t share = (uint64_t)pl.ppc * s.HW;
    const bool f32 = d->x_dtype == DIV_F32, one_turn = pl.turns64 <= 64u, two_turns = pl.turns64 <= 128u;
    if (one_turn && share < 40000u) return true;
    const uint64_t own = cluster_ns(s, pl);
    Choice ch;
    choose_compress(d, s, 0u, &ch);
    switch (ch.code) {
        case 7:
        case 4:
            if (f32 && pl.per_sm == 1u) return s.P2 <= 4u || (s.P2 <= 8u && one_turn) || own <= other_ns(s, 7);
            return two_turns || (f32 && s.P2 <= 8u);
        case 2:
        case 3:
        case 6: {
            if (!one_turn && two_turns && (f32 || pl.per_sm >= 2u)) return true;
            const uint64_t other = other_ns(s, ch.code);
            return own <= (two_turns ? other : other * 95u / 100u);
        }
    }
    return true;
}

// Does the cluster kernel take a descriptor, and in clusters of how many CTAs?  (Flags pin one of the other kernels.)
bool choose_cluster(const div_desc* d, const Shape& s, uint32_t flags, ClusterPlan* out) {
    if (flags != 0) return false;
    const DeviceInfo di = device_info();
    if (!di.ok || di.sms < 1) return false;
    if (s.H == 1) {
        LineGeom lg;
        if (plan_lines(d, s, &lg)) return false;          // 1-D maps have a kernel of their own
    }
    // Cost in KB of x an SM works through (41 KB take 1 us): its share, and 3 us for every further time the device has
    // to be filled, since the CTAs of one filling load, reduce and quantise in step.  Ties go to the smaller shares, and among
    // equal ones to the smaller clusters (3 planes are 4 CTAs with work and none without: 8 x 3 x 224 x 224 17.9 -> 9.0 us).
    uint64_t best = ~0ull;
    for (uint32_t log2cs = 0; (1u << log2cs) <= CL_MAX; ++log2cs) {
        ClusterPlan pl;
        if (!plan_cluster_cs(d, s, log2cs, di, &pl)) continue;
        const uint64_t share = (uint64_t)pl.ppc * s.HW * 4u / 1024u;
        const uint64_t cost = ((uint64_t)s.N * pl.cs + (uint32_t)di.sms - 1u) / (uint32_t)di.sms * share + 123u * (pl.turns64 - 64u) / 64u;
        if (cost < best || (cost == best && pl.ppc < out->ppc)) {
            best = cost;
            *out = pl;
        }
    }
    return best != ~0ull && cluster_pays(d, s, *out);
}

// Estimated times beside the parking kernel's, in ns.  To the fits above, which are for maps of samples that the device works on together,
// comes what many small samples cost: a sample of the strip and staged kernels (13520 x 5 x 14 x 16 bfloat16 with B = 4 70 us, 38306 x 13 x
// 8 x 8 with B = 8 484 us), a unit of the lagged kernel (57675 x 4 x 4 x 16 110 us), and a turn of the clusters beyond two.  The kernels for planes
// a warp wide are only asked where clusters do not pay, on maps that they take half as long again for (1 x 1282 x 124 x 32 27 us).
uint64_t beside_park_ns(const Shape& s, const ClusterPlan* cl, const Choice& ch) {
    if (cl) return cluster_ns(s, *cl) + (cl->turns64 > 128u ? (cl->turns64 - 128u) * 1000ull / 64u : 0u);
    switch (ch.code) {
        case 2: return 4600u + s.total * 155u / 100000u + 4ull * s.N;
        case 3: return other_ns(s, 3) + ch.lp.total_units * 12u / 10u;
        case 6: return other_ns(s, 6) + s.N * 97ull / 10u;
        case 4:
        case 7: return other_ns(s, 7) * 3u / 2u;
    }
    return 0u;
}
// Does the parking kernel take a descriptor that the rules above give to clusters (cl) or to kernel ch.code?  Measured against both on 800
// random maps (0.1 to 205 MB, both types, all blocks and bit widths that it takes): clusters in one turn are not asked to give way
// (0.8 of its time in the geometric mean); clusters in turns and the kernels that read x twice where the estimated time is shorter:
// 1.3 times faster in the geometric mean there (50 x 2048 x 16 x 16 with B = 4 49.5 -> 27.8 us, 96 x 432 x 15 x 56 with B = 4 74.9 -> 37.2 us).
// Of 600 more, half of them batches of 150 to 60000 small samples, it takes 175: 0.67 of the others' time in the geometric mean, two of them 4 and 10 %
// slower; what it leaves it would mostly need longer for (2169 x 4 x 14 x 16 13.4 against 16.6 us).
// The staged kernel keeps samples of which less than two and a half fit the parked units (8 x 1840 x 56 x 56 58.5 against 68.1 us).
// 1-D maps stay with the line kernels, whose second read of x is from the L1 or L2 and whose units hold whole rows (here a strip has one
// row of four or eight): of 21 random ones up to 8 MB none is faster here and the geometric mean 1.34 times slower (355 x 45 x 64 bfloat16
// 8.3 against 14.5 us, 4 x 936 x 512 with B = 4 10.5 against 13.4 us).  (The general kernels run no map that plan_park accepts.)
bool choose_park(const div_desc* d, const Shape& s, uint32_t flags, const ClusterPlan* cl, const Choice& ch, ParkPlan* out) {
    if (flags != 0u) return ch.code == 6 && plan_park(d, s, out);
    if ((cl && cl->turns64 <= 64u) || !plan_park(d, s, out)) return false;
    if (cl && out->sets < 2u) return false;               // (a chunk at a time: 96 x 16 x 100 x 100 bfloat16 21.8 -> 24.6 us)
    if (!cl && ch.code == 6 && 5u * out->per_cta > 2u * PARK_DEPTH * out->sets) return false;
    return park_ns(*out) <= beside_park_ns(s, cl, ch);
}

// What runs a descriptor: the parking kernel, clusters, or kernel ch.code (which also follows where one of the others is refused).
struct Route {
    bool park, cluster;
    ParkPlan pk;
    ClusterPlan cl;
};
void choose_route(const div_desc* d, const Shape& s, uint32_t flags, Route* r) {
    const uint32_t pins = flags & ~DIV_FLAG_NO_PARK_KERNEL;       // that flag leaves the others' order as it is
    r->cluster = choose_cluster(d, s, pins, &r->cl);
    r->park = false;
    if (pins != flags || (r->cluster && r->cl.turns64 <= 64u)) return;
    Choice ch;
    choose_compress(d, s, flags, &ch);
    r->park = choose_park(d, s, flags, r->cluster ? &r->cl : nullptr, ch, &r->pk);
}

bool decompress_fast_ok(const Shape& s) {
    return (s.W % 4 == 0) && s.B >= 4 && (s.B & (s.B - 1)) == 0 && s.N <= 65535;
}
bool decompress_flat_ok(const Shape& s) {
    return (s.CHW % 4 == 0) && s.HW <= FLAT_MAX_HW && s.TPP <= 65535 && s.N <= 65535 && s.CHW < (1u << 31) &&
           flat_smem_bytes(4u * 256u * FLAT_QPT, s.HW, s.TPP) <= 40000;
}

// bands that a run of `elems` elements can touch, and whether the row kernel takes the map: at most 40 KB of shared memory
uint64_t rows_bands(const Shape& s, uint32_t elems) {
    const uint64_t planes = elems / s.HW + 2u;             // whole or in part
    const uint64_t by_rows = (uint64_t)(elems / s.W + 1u) / s.B + 2u + planes;
    const uint64_t all = planes * s.Hb;
    return by_rows < all ? by_rows : all;
}
// Against the flat kernel the row kernel wins once building the quad table shows (64 x 64 x 90 x 90 54 -> 35 us, 24 x 64 x 61 x 47
// 13.5 -> 8.2 us, 35 x 35 13.3 -> 12.3 us) and loses on small planes, where its bands hold few rows (34 x 34 16.6 against
// 26.7 us, 14 x 14 13.3 against 18.5 us): from 2048 elements per plane on.
bool decompress_rows_ok(const Shape& s) {
    if (decompress_flat_ok(s) && s.HW < 2048u) return false;
    return s.W >= 4 && s.CHW % 4 == 0 && s.N <= 65535 && s.CHW < (1u << 31) &&
           rows_bands(s, 1024u * FLAT_QPT) * s.W * 4u <= 40000u;
}

// the launches of div_compress_ex, whose arguments have been checked
div_status compress_map(const div_desc* desc, const Shape& s, const div_layout& lo, const void* x_dev, uint8_t* blob, uint32_t* ws,
                        uint64_t seed, cudaStream_t stream, uint32_t flags, const ShareFault& fault) {
    // kernels that store bytes or half-words leave the unused top of a partial last word alone: it is zero by contract
    if ((s.total * (uint64_t)desc->qbits) % 32u != 0 &&
        cudaMemsetAsync(blob + lo.packed_off + lo.packed_bytes - 4, 0, 4, stream) != cudaSuccess)
        return DIV_ERR_CUDA;
    Route rt;
    choose_route(desc, s, flags, &rt);
    if (fault.number != 0u) rt.park = rt.park && fault.no_park;      // a test of the clusters, or of what follows a refused parking kernel
    if (rt.park) {
        if (clear_scratch(ws, lo.workspace_bytes, stream) != DIV_OK) return DIV_ERR_CUDA;
        if (compress_park(desc, s, lo, rt.pk, x_dev, blob, ws, seed, stream, 0u, 0u, fault.no_park ? fault.more_smem : 0u) == DIV_OK) return DIV_OK;
    }
    if (rt.cluster && compress_cluster(desc, s, lo, rt.cl, x_dev, blob, ws, seed, stream, fault.no_park ? ShareFault() : fault) == DIV_OK) return DIV_OK;
    if (!rt.park && clear_scratch(ws, lo.workspace_bytes, stream) != DIV_OK) return DIV_ERR_CUDA;
    // The single-launch kernels need all their CTAs resident, so they are launched cooperatively; where the
    // device refuses such a launch (fewer SMs visible to the process than the device reports, for instance) the
    // next kernel in line takes the descriptor: nothing has been enqueued by the refused launch.
    for (uint32_t f = flags;;) {
        Choice ch;
        choose_compress(desc, s, f, &ch);
        div_status r = DIV_OK;
        uint32_t drop = 0;
        switch (ch.code) {
            case 8: return compress_lines(desc, s, lo, ch.lg, x_dev, blob, ws, seed, stream, true);
            case 5: return compress_lines(desc, s, lo, ch.lg, x_dev, blob, ws, seed, stream, false);
            case 6: r = compress_staged(desc, s, lo, ch.sp, x_dev, blob, ws, seed, stream); drop = DIV_FLAG_NO_STAGED_KERNEL; break;
            case 3: r = compress_lagged(desc, s, lo, ch.lp, x_dev, blob, ws, seed, stream); drop = DIV_FLAG_NO_LAGGED_KERNEL; break;
            case 2: r = compress_fused_v(desc, s, lo, ch.vp, x_dev, blob, ws, seed, stream); drop = DIV_FLAG_NO_STRIP_KERNEL; break;
            case 7: return compress_planes(desc, s, lo, ch.pg, x_dev, blob, ws, seed, stream, true);
            case 4: return compress_planes(desc, s, lo, ch.pg, x_dev, blob, ws, seed, stream, false);
            case 1: r = compress_fused(desc, s, lo, ch.fp, x_dev, blob, ws, seed, stream); drop = DIV_FLAG_FORCE_TWO_PASS; break;
            default: return compress_two_pass(desc, s, lo, x_dev, blob, ws, seed, stream);
        }
        if (r != DIV_ERR_CUDA) return r;
        f |= drop;
    }
    return compress_two_pass(desc, s, lo, x_dev, blob, ws, seed, stream);
}

// the same for div_planegroup_compress
div_status compress_planegroup(const div_desc* desc, const Shape& s, const div_layout& lo, const void* x_dev, uint8_t* blob, uint64_t seed,
                               cudaStream_t stream, uint32_t flags, const ShareFault& fault) {
    // kernels that store bytes or half-words leave the unused top of a partial last word alone: it is zero by contract
    if ((s.total * (uint64_t)desc->qbits) % 32u != 0 &&
        cudaMemsetAsync(blob + lo.packed_off + lo.packed_bytes - 4, 0, 4, stream) != cudaSuccess)
        return DIV_ERR_CUDA;
    PgPlan pl;
    if (!(flags & DIV_FLAG_FORCE_TWO_PASS) && plan_pg_strip(desc, s, &pl))
        return compress_pg_strip(desc, s, lo, pl, x_dev, blob, seed, stream);
    if (PgSmall g; !(flags & DIV_FLAG_FORCE_TWO_PASS) && plan_pg_small(desc, s, &g))
        return compress_pg_small(desc, s, lo, g, x_dev, blob, seed, stream);
    // Everything else that fits shared memory.  (Where the two kernels above apply they are faster or as good: 64 x 256 x 56 x 56 53
    // against 70 us, 64 x 2048 x 7 x 7 18.6 against 20.0 us, 64 x 1024 x 14 x 14 30.8 against 28.8 us.)
    // Where the launch is refused the general kernel takes the map.
    if (SharePlan ps; !(flags & DIV_FLAG_FORCE_TWO_PASS) && plan_plane_share(desc, s, &ps) &&
                      compress_plane_share(desc, s, lo, ps, x_dev, blob, seed, stream, fault) == DIV_OK)
        return DIV_OK;
    // general kernel: words shared by two planes (and the zero-padded last word) are merged with atomic ORs
    // into a cleared buffer
    if (((uint64_t)s.HW * (uint64_t)desc->qbits) % 32u != 0 &&
        cudaMemsetAsync(blob + lo.packed_off, 0, lo.packed_bytes, stream) != cudaSuccess)
        return DIV_ERR_CUDA;
    return dispatch_types(desc->x_dtype, desc->lfc_dtype, [&](auto* xt, auto* lt) -> div_status {
        typedef std::remove_pointer_t<decltype(xt)> XT;
        typedef std::remove_pointer_t<decltype(lt)> LT;
        return dispatch_q(desc->qbits, [&](auto q) -> div_status {
            pg_general_kernel<XT, LT, decltype(q)::value><<<s.N * s.C, 256, 0, stream>>>(
                (const XT*)x_dev, (LT*)(blob + lo.lfc_off), (uint32_t*)(blob + lo.packed_off),
                (uint32_t*)(blob + lo.stats_off), s, seed);
            return launch_status();
        });
    });
}

}  // namespace

extern "C" {

const char* div_status_string(div_status s) {
    switch (s) {
        case DIV_OK: return "ok";
        case DIV_ERR_NULL: return "null pointer";
        case DIV_ERR_SHAPE: return "bad shape (need n,c,h,w >= 1, c*h*w < 2^32, n < 2^31)";
        case DIV_ERR_PARAM: return "bad parameter (block >= 1, qbits in {1,2,4,8}, dtype in {f32,bf16})";
        case DIV_ERR_ALIGN: return "device pointer not 16-byte aligned";
        case DIV_ERR_CAPACITY: return "buffer too small";
        case DIV_ERR_CUDA: return "CUDA runtime error";
        case DIV_ERR_TIMEOUT: return "device-side bounded wait expired";
    }
    return "unknown status";
}

div_status div_compressed_bytes(const div_desc* desc, div_layout* out) {
    if (!desc || !out) return DIV_ERR_NULL;
    const div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    make_layout(desc, make_shape(desc), out);
    return DIV_OK;
}

div_status div_plan_query(const div_desc* desc, uint32_t flags, div_plan* out) {
    if (!desc || !out) return DIV_ERR_NULL;
    const div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    if (flags & ~DIV_FLAG_ALL) return DIV_ERR_PARAM;
    const Shape s = make_shape(desc);
    *out = div_plan();
    Choice ch;
    choose_compress(desc, s, flags, &ch);
    out->fused = ch.code;
    if (ch.code == 8) {
        out->grid = (int32_t)(ch.lf.ctas_per_sample * s.N);
        out->threads = 256;
        out->chunk_elems = (int64_t)ch.lf.rpc * s.W;
        out->chunks_per_sample = ch.lf.ctas_per_sample;
    } else if (ch.code == 5) {
        out->grid = (int32_t)((ch.lg.qps + 256 * LINE_QPT - 1) / (256 * LINE_QPT) * s.N);
        out->threads = 256;
        out->chunk_elems = 4 * LINE_QPT * 256;
    } else if (ch.code == 6) {
        out->grid = ch.sp.grid;
        out->threads = ch.sp.threads;
        out->stages = (int32_t)(ch.sp.kr + ch.sp.kq);
        out->lag = (int32_t)ch.sp.lag_steps;
        out->smem_bytes = ch.sp.smem_bytes;
        out->chunk_elems = ch.sp.chunk_elems;
        out->chunks_per_sample = ch.sp.chunks_per_sample;
    } else if (ch.code == 3) {
        out->grid = ch.lp.grid;
        out->threads = ch.lp.threads;
        out->stages = 0;
        out->lag = (int32_t)ch.lp.lag_units;
        out->smem_bytes = 0;
        out->chunk_elems = (int64_t)32 * ch.lp.bands_per_lane * 4 * s.B;       // elements of one full unit
        out->chunks_per_sample = ch.lp.units_per_sample;
    } else if (ch.code == 2) {
        out->grid = ch.vp.grid;
        out->threads = ch.vp.threads;
        out->stages = ch.vp.stages;
        out->lag = ch.vp.lag;
        out->smem_bytes = ch.vp.smem_bytes;
        out->chunk_elems = ch.vp.chunk_elems;
        out->chunks_per_sample = ch.vp.chunks_per_sample;
    } else if (ch.code == 7) {
        out->grid = (int32_t)(ch.pf.ctas_per_sample * s.N);
        out->threads = 256;
        out->smem_bytes = (int32_t)ch.pf.smem;
        out->chunk_elems = (int64_t)ch.pf.ppc * s.HW;
        out->chunks_per_sample = ch.pf.ctas_per_sample;
    } else if (ch.code == 4) {
        out->grid = (int32_t)((ch.pg.qps + 256 * PLANE_QPT - 1) / (256 * PLANE_QPT) * s.N);
        out->threads = 256;
        out->chunk_elems = 4 * PLANE_QPT * 256;
    } else if (ch.code == 1) {
        out->grid = ch.fp.grid;
        out->threads = ch.fp.threads;
        out->stages = ch.fp.stages;
        out->lag = ch.fp.lag;
        out->smem_bytes = ch.fp.smem_bytes;
        out->chunk_elems = ch.fp.chunk_elems;
        out->chunks_per_sample = ch.fp.chunks_per_sample;
    } else {
        out->grid = (int32_t)((s.tiles + 255) / 256);
        out->threads = 256;
    }
    Route rt;
    choose_route(desc, s, flags, &rt);
    out->on_chip = rt.cluster ? 1 : 0;
    out->parked = rt.park ? 1 : 0;
    if (rt.park) {
        out->grid = (int32_t)rt.pk.grid;
        out->threads = PARK_THREADS;
        out->stages = rt.cluster ? (int32_t)((rt.cl.turns64 + 63u) / 64u) : (int32_t)rt.pk.stages;
        out->lag = 0;
        out->smem_bytes = (int32_t)rt.pk.smem_bytes;
        out->chunk_elems = rt.pk.chunk_elems;
        out->chunks_per_sample = rt.pk.chunks_per_sample;
    } else if (rt.cluster) {
        const ClusterPlan& cl = rt.cl;
        out->grid = (int32_t)(s.N * cl.cs);
        out->threads = (int32_t)cluster_threads(s.P2, cl);
        out->stages = (int32_t)((cl.turns64 + 63u) / 64u);
        out->smem_bytes = (int32_t)cl.smem_bytes;
        out->chunk_elems = (int64_t)cl.ppc * s.HW;
        out->chunks_per_sample = cl.cs;
    }
    out->decompress_fast = decompress_fast_ok(s) ? ((s.H == 1 && s.CHW < (1u << 31)) ? 3 : 1) : decompress_rows_ok(s) ? 4 : (decompress_flat_ok(s) ? 2 : 0);
    return DIV_OK;
}

div_status div_compress_ex(const div_desc* desc, const void* x_dev, void* comp_dev, size_t comp_capacity,
                           void* workspace_dev, size_t workspace_bytes, uint64_t seed, void* cuda_stream,
                           uint32_t flags) {
    if (!desc || !x_dev || !comp_dev || !workspace_dev) return DIV_ERR_NULL;
    div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    if (flags & ~DIV_FLAG_ALL) return DIV_ERR_PARAM;
    if (!aligned16(x_dev) || !aligned16(comp_dev) || !aligned16(workspace_dev)) return DIV_ERR_ALIGN;
    const Shape s = make_shape(desc);
    div_layout lo;
    make_layout(desc, s, &lo);
    if (comp_capacity < lo.total_bytes || workspace_bytes < lo.workspace_bytes) return DIV_ERR_CAPACITY;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    uint8_t* blob = (uint8_t*)comp_dev;
    uint32_t* ws = (uint32_t*)workspace_dev;
    return compress_map(desc, s, lo, x_dev, blob, ws, seed, stream, flags, ShareFault());
}

div_status div_debug_compress_starved(const div_desc* desc, const void* x_dev, void* comp_dev, size_t comp_capacity,
                                      void* workspace_dev, size_t workspace_bytes, uint64_t seed, void* cuda_stream,
                                      uint32_t flags, uint64_t timeout_ns) {
    if (!desc || !x_dev || !comp_dev || !workspace_dev) return DIV_ERR_NULL;
    div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    if ((flags & ~DIV_FLAG_ALL) || timeout_ns == 0 || timeout_ns > 100000000ull) return DIV_ERR_PARAM;
    if (!aligned16(x_dev) || !aligned16(comp_dev) || !aligned16(workspace_dev)) return DIV_ERR_ALIGN;
    const Shape s = make_shape(desc);
    div_layout lo;
    make_layout(desc, s, &lo);
    if (comp_capacity < lo.total_bytes || workspace_bytes < lo.workspace_bytes) return DIV_ERR_CAPACITY;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    if (clear_scratch(workspace_dev, lo.workspace_bytes, stream) != DIV_OK) return DIV_ERR_CUDA;
    uint8_t* blob = (uint8_t*)comp_dev;
    uint32_t* ws = (uint32_t*)workspace_dev;
    const uint32_t never = 0xFFFFFFFFu;      // an arrival count no sample reaches
    Route rt;
    choose_route(desc, s, flags, &rt);
    if (rt.park) return compress_park(desc, s, lo, rt.pk, x_dev, blob, ws, seed, stream, never, timeout_ns);
    if (rt.cluster)
        return compress_cluster(desc, s, lo, rt.cl, x_dev, blob, ws, seed, stream, ShareFault{1u << 19, 0u, 0u, 0u, (uint32_t)timeout_ns});
    if (!(flags & DIV_FLAG_NO_STRIP_KERNEL)) {
        VPlan vp;
        if (plan_v(desc, s, &vp) == DIV_OK) return compress_fused_v(desc, s, lo, vp, x_dev, blob, ws, seed, stream, never, timeout_ns);
    }
    if (!(flags & DIV_FLAG_NO_LAGGED_KERNEL)) {
        LPlan lp;
        if (plan_lagged(desc, s, &lp) == DIV_OK) return compress_lagged(desc, s, lo, lp, x_dev, blob, ws, seed, stream, never, timeout_ns);
    }
    if (!(flags & DIV_FLAG_NO_STAGED_KERNEL)) {
        SPlan sp;
        if (plan_staged(desc, s, &sp) == DIV_OK) return compress_staged(desc, s, lo, sp, x_dev, blob, ws, seed, stream, never, timeout_ns);
    }
    if (!(flags & (DIV_FLAG_NO_PLANE_KERNELS | DIV_FLAG_TWO_LAUNCH_PLANES))) {
        PlaneGeom pg;
        if (plan_planes(desc, s, &pg)) return compress_planes(desc, s, lo, pg, x_dev, blob, ws, seed, stream, true, never, timeout_ns);
    }
    return DIV_ERR_PARAM;
}

div_status div_debug_on_chip(const div_desc* desc, const void* x_dev, void* comp_dev, size_t comp_capacity, void* workspace_dev,
                             size_t workspace_bytes, uint64_t seed, void* cuda_stream, int32_t fault, uint64_t timeout_ns) {
    if (!desc || !x_dev || !comp_dev) return DIV_ERR_NULL;
    const div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    if (fault < DIV_FAULT_NONE || fault > DIV_FAULT_PARK_REFUSED || timeout_ns == 0 || timeout_ns > 100000000ull) return DIV_ERR_PARAM;
    if (!aligned16(x_dev) || !aligned16(comp_dev) || !aligned16(workspace_dev)) return DIV_ERR_ALIGN;
    const Shape s = make_shape(desc);
    const bool planes = workspace_dev == nullptr;
    if (planes && !pg_shape_ok(s)) return DIV_ERR_SHAPE;
    div_layout lo;
    if (planes) make_layout_pg(desc, s, &lo);
    else make_layout(desc, s, &lo);
    if (comp_capacity < lo.total_bytes || workspace_bytes < lo.workspace_bytes) return DIV_ERR_CAPACITY;
    ShareFault f = {};
    f.number = 1;
    f.timeout_ns = (uint32_t)timeout_ns;
    f.no_copies = fault == DIV_FAULT_COPIES;
    f.no_park = fault == DIV_FAULT_PARK_REFUSED;
    f.more_smem = fault == DIV_FAULT_REFUSED || f.no_park ? 1u << 20 : 0u;
    const cudaStream_t stream = (cudaStream_t)cuda_stream;
    if (planes) {
        div_plan plan;
        if (div_planegroup_plan_query(desc, 0u, &plan) != DIV_OK || !plan.on_chip || f.no_park) return DIV_ERR_PARAM;
        return compress_planegroup(desc, s, lo, x_dev, (uint8_t*)comp_dev, seed, stream, 0u, f);
    }
    Route rt;
    choose_route(desc, s, 0u, &rt);
    if (!(f.no_park ? rt.park : rt.cluster)) return DIV_ERR_PARAM;
    return compress_map(desc, s, lo, x_dev, (uint8_t*)comp_dev, (uint32_t*)workspace_dev, seed, stream, 0u, f);
}

div_status div_compress(const div_desc* desc, const void* x_dev, void* comp_dev, size_t comp_capacity,
                        void* workspace_dev, size_t workspace_bytes, uint64_t seed, void* cuda_stream) {
    return div_compress_ex(desc, x_dev, comp_dev, comp_capacity, workspace_dev, workspace_bytes, seed, cuda_stream, 0u);
}

div_status div_decompress(const div_desc* desc, const void* comp_dev, size_t comp_bytes, void* xhat_dev,
                          void* cuda_stream) {
    if (!desc || !comp_dev || !xhat_dev) return DIV_ERR_NULL;
    div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    if (!aligned16(comp_dev) || !aligned16(xhat_dev)) return DIV_ERR_ALIGN;
    const Shape s = make_shape(desc);
    div_layout lo;
    make_layout(desc, s, &lo);
    if (comp_bytes < lo.total_bytes) return DIV_ERR_CAPACITY;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const uint8_t* blob = (const uint8_t*)comp_dev;
    const uint64_t nwords = lo.packed_bytes / 4;
    return dispatch_types(desc->x_dtype, desc->lfc_dtype, [&](auto* xt, auto* lt) -> div_status {
        typedef std::remove_pointer_t<decltype(xt)> XT;
        typedef std::remove_pointer_t<decltype(lt)> LT;
        return dispatch_q(desc->qbits, [&](auto q) -> div_status {
            constexpr int Q = decltype(q)::value;
            const LT* lfc = (const LT*)(blob + lo.lfc_off);
            const uint32_t* packed = (const uint32_t*)(blob + lo.packed_off);
            const float* stats = (const float*)(blob + lo.stats_off);
            if (decompress_fast_ok(s) && s.H == 1 && s.CHW < (1u << 31)) {
                DecLine d;
                d.qps = s.CHW / 4;
                d.C = s.C;
                d.Wb = s.Wb;
                d.qpr = s.W / 4;
                d.log2lpt = 0;
                while ((4u << d.log2lpt) < s.B) ++d.log2lpt;
                d.by_qpr = make_fastdiv(d.qpr);
                const uint32_t per_block = 256u * DEC_QPT;
                dim3 grid((d.qps + per_block - 1) / per_block, s.N);
                return launch_pdl(decompress_line_kernel<XT, LT, Q, DEC_QPT>, grid, 256, 0, stream, lfc, packed, stats, (XT*)xhat_dev, d);
            } else if (decompress_fast_ok(s)) {
                DecFast d;
                d.qps = s.CHW / 4;
                d.C = s.C;
                d.TPP = s.TPP;
                d.Wb = s.Wb;
                d.log2B = 0;
                while ((1u << d.log2B) < s.B) ++d.log2B;
                d.H = s.H;
                d.hwq = s.HW / 4;
                d.wq = s.W / 4;
                d.hq_count = (s.H + 3u) / 4u;
                d.ipp = d.hq_count * d.wq;
                d.items = s.C * d.ipp;
                d.by_ipp = make_fastdiv(d.ipp);
                d.by_wq = make_fastdiv(d.wq);
                dim3 grid((d.items + 255u) / 256u, s.N);
                // rows that are not whole 32-byte sectors: the 4 rows of an item spread over the plane (see the kernel)
                if ((s.W * (uint32_t)sizeof(XT)) % 32u != 0 && s.H >= 8u)
                    return launch_pdl(decompress_quad_kernel<XT, LT, Q, DEC_QPT, true, DecFast>, grid, 256, 0, stream, lfc, packed, stats, (XT*)xhat_dev, d);
                else
                    return launch_pdl(decompress_quad_kernel<XT, LT, Q, DEC_QPT, false, DecFast>, grid, 256, 0, stream, lfc, packed, stats, (XT*)xhat_dev, d);
            } else if (decompress_rows_ok(s)) {
                DecRows d;
                d.qps = s.CHW / 4;
                d.tiles = s.C * s.TPP;
                d.H = s.H;
                d.W = s.W;
                d.Hb = s.Hb;
                d.Wb = s.Wb;
                d.bands = (uint32_t)rows_bands(s, 1024u * FLAT_QPT);
                d.step_planes = 1024u / s.W / s.H;
                d.step_rows = 1024u / s.W % s.H;
                d.step_cols = 1024u % s.W;
                d.by_w = make_fastdiv(s.W);
                d.by_h = make_fastdiv(s.H);
                d.by_b = make_fastdiv(s.B);
                dim3 grid((d.qps + 256u * FLAT_QPT - 1) / (256u * FLAT_QPT), s.N);
                return launch_pdl(decompress_rows_kernel<XT, LT, Q, FLAT_QPT, DecRows>, grid, 256, 4u * d.bands * d.W, stream, lfc, packed, stats, (XT*)xhat_dev, d);
            } else if (decompress_flat_ok(s)) {
                DecFlat d;
                d.qps = s.CHW / 4;
                d.C = s.C;
                d.TPP = s.TPP;
                d.Wb = s.Wb;
                d.HW = s.HW;
                d.W = s.W;
                d.B = s.B;
                d.by_hw = make_fastdiv(s.HW);
                d.by_w = make_fastdiv(s.W);
                d.by_b = make_fastdiv(s.B);
                const uint32_t per_block = 256u * FLAT_QPT;
                d.table_words = quad_table_words(s.HW);
                d.period = quad_period(s.HW);
                d.period_planes = quad_period_planes(s.HW);
                d.by_period = make_fastdiv(d.period);
                d.planes_per_cta = flat_planes_per_cta(4u * per_block, s.HW);
                dim3 grid((d.qps + per_block - 1) / per_block, s.N);
                return launch_pdl(decompress_flat_kernel<XT, LT, Q, FLAT_QPT, DecFlat>, grid, 256, flat_smem_bytes(4u * per_block, s.HW, s.TPP), stream,
                                  lfc, packed, stats, (XT*)xhat_dev, d);
            } else {
                const uint64_t g = (nwords + 255) / 256;
                if (g > 0x7FFFFFFFull) return DIV_ERR_SHAPE;
                decompress_general_kernel<XT, LT, Q><<<(unsigned)g, 256, 0, stream>>>(lfc, packed, stats, (XT*)xhat_dev, s, nwords);
            }
            return launch_status();
        });
    });
}

// ------------------------------------------------------------------------------------------------
// div_compress_static: compress with the scratch in a fixed array inside the library
// ------------------------------------------------------------------------------------------------
}  // extern "C"

namespace {

// Scratch of div_compress_static: header + one 128-byte slot per sample, for up to
// DIV_STATIC_MAX_SAMPLES samples.  It lives in every GPU that loads the library until the process ends.
constexpr size_t STATIC_WS_BYTES =
    (4ull * (divk::WS_HEADER_WORDS + (size_t)divk::WS_SLOT_WORDS * DIV_STATIC_MAX_SAMPLES) + 255ull) / 256ull * 256ull;
static __device__ __align__(256) unsigned char g_static_workspace[STATIC_WS_BYTES];

// Device address of g_static_workspace on the current device.  In host code the array's name is only a
// handle for the runtime, not an address a kernel could use, so the address is asked for (a host-side
// query, no allocation); asking on every call keeps the library free of cached pointers that a device reset
// would leave dangling.
div_status static_workspace_ptr(void** out) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_workspace) != cudaSuccess || !ptr) {
        cudaGetLastError();
        return DIV_ERR_CUDA;
    }
    *out = ptr;
    return DIV_OK;
}

}  // namespace

extern "C" {

div_status div_compress_static(const div_desc* desc, const void* x_dev, void* comp_dev, size_t comp_capacity,
                               uint64_t seed, void* cuda_stream) {
    if (!desc) return DIV_ERR_NULL;
    const div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    if (desc->n > DIV_STATIC_MAX_SAMPLES) return DIV_ERR_CAPACITY;      // the fixed scratch has no slot for more samples
    void* ws = nullptr;
    const div_status got = static_workspace_ptr(&ws);
    if (got != DIV_OK) return got;
    // same path as div_compress from here on (it clears the part of the scratch it uses on the stream)
    return div_compress_ex(desc, x_dev, comp_dev, comp_capacity, ws, STATIC_WS_BYTES, seed, cuda_stream, 0u);
}

div_status div_read_static_status(void* cuda_stream, int32_t* out_status) {
    if (!out_status) return DIV_ERR_NULL;
    void* ws = nullptr;
    const div_status got = static_workspace_ptr(&ws);
    if (got != DIV_OK) return got;
    return div_read_device_status(ws, cuda_stream, out_status);
}

// ------------------------------------------------------------------------------------------------
// per-plane quantisation groups
// ------------------------------------------------------------------------------------------------
div_status div_planegroup_bytes(const div_desc* desc, div_layout* out) {
    if (!desc || !out) return DIV_ERR_NULL;
    const div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    const Shape s = make_shape(desc);
    if (!pg_shape_ok(s)) return DIV_ERR_SHAPE;
    make_layout_pg(desc, s, out);
    return DIV_OK;
}

div_status div_planegroup_plan_query(const div_desc* desc, uint32_t flags, div_plan* out) {
    if (!desc || !out) return DIV_ERR_NULL;
    const div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    if (flags & ~DIV_FLAG_FORCE_TWO_PASS) return DIV_ERR_PARAM;
    const Shape s = make_shape(desc);
    if (!pg_shape_ok(s)) return DIV_ERR_SHAPE;
    *out = div_plan();
    PgPlan pl;
    if (!(flags & DIV_FLAG_FORCE_TWO_PASS) && plan_pg_strip(desc, s, &pl)) {
        out->fused = 1;
        out->grid = pl.grid;
        out->threads = (int32_t)pl.threads;
        out->chunk_elems = (int64_t)pl.G * s.HW;
        out->chunks_per_sample = (s.C + pl.G - 1) / pl.G;
    } else if (PgSmall g; !(flags & DIV_FLAG_FORCE_TWO_PASS) && plan_pg_small(desc, s, &g)) {
        out->fused = 2;
        out->grid = (int32_t)((g.planes + g.G - 1) / g.G);
        out->threads = 256;
        out->smem_bytes = (int32_t)pg_small_smem_bytes(g);
        out->chunk_elems = (int64_t)g.G * s.HW;
        out->chunks_per_sample = (s.C + g.G - 1) / g.G;
    } else {
        out->fused = 0;
        out->grid = (int32_t)(s.N * s.C);
        out->threads = 256;
        out->chunk_elems = s.HW;
        out->chunks_per_sample = s.C;
        if (SharePlan ps; !(flags & DIV_FLAG_FORCE_TWO_PASS) && plan_plane_share(desc, s, &ps)) {
            out->on_chip = 1;
            out->chunks_per_sample = (s.C + ps.ppc - 1) / ps.ppc;
            out->grid = (int32_t)(s.N * out->chunks_per_sample);
            out->threads = (int32_t)SHARE_THREADS;
            out->smem_bytes = (int32_t)ps.smem_bytes;
            out->chunk_elems = (int64_t)ps.ppc * s.HW;
        }
    }
    out->decompress_fast = decompress_fast_ok(s) ? 1 : (pg_decompress_flat_ok(s) ? 2 : 0);
    return DIV_OK;
}

div_status div_planegroup_compress(const div_desc* desc, const void* x_dev, void* comp_dev, size_t comp_capacity,
                                   uint64_t seed, void* cuda_stream, uint32_t flags) {
    if (!desc || !x_dev || !comp_dev) return DIV_ERR_NULL;
    div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    if (flags & ~DIV_FLAG_FORCE_TWO_PASS) return DIV_ERR_PARAM;
    if (!aligned16(x_dev) || !aligned16(comp_dev)) return DIV_ERR_ALIGN;
    const Shape s = make_shape(desc);
    if (!pg_shape_ok(s)) return DIV_ERR_SHAPE;
    div_layout lo;
    make_layout_pg(desc, s, &lo);
    if (comp_capacity < lo.total_bytes) return DIV_ERR_CAPACITY;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    uint8_t* blob = (uint8_t*)comp_dev;
    return compress_planegroup(desc, s, lo, x_dev, blob, seed, stream, flags, ShareFault());
}

div_status div_planegroup_decompress(const div_desc* desc, const void* comp_dev, size_t comp_bytes, void* xhat_dev,
                                     void* cuda_stream) {
    if (!desc || !comp_dev || !xhat_dev) return DIV_ERR_NULL;
    div_status st = check_desc(desc);
    if (st != DIV_OK) return st;
    if (!aligned16(comp_dev) || !aligned16(xhat_dev)) return DIV_ERR_ALIGN;
    const Shape s = make_shape(desc);
    if (!pg_shape_ok(s)) return DIV_ERR_SHAPE;
    div_layout lo;
    make_layout_pg(desc, s, &lo);
    if (comp_bytes < lo.total_bytes) return DIV_ERR_CAPACITY;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const uint8_t* blob = (const uint8_t*)comp_dev;
    const uint64_t nwords = lo.packed_bytes / 4;
    return dispatch_types(desc->x_dtype, desc->lfc_dtype, [&](auto* xt, auto* lt) -> div_status {
        typedef std::remove_pointer_t<decltype(xt)> XT;
        typedef std::remove_pointer_t<decltype(lt)> LT;
        return dispatch_q(desc->qbits, [&](auto q) -> div_status {
            constexpr int Q = decltype(q)::value;
            const LT* lfc = (const LT*)(blob + lo.lfc_off);
            const uint32_t* packed = (const uint32_t*)(blob + lo.packed_off);
            const uint32_t* stats = (const uint32_t*)(blob + lo.stats_off);
            if (decompress_fast_ok(s)) {
                DecFast d;
                d.qps = s.CHW / 4;
                d.C = s.C;
                d.TPP = s.TPP;
                d.Wb = s.Wb;
                d.log2B = 0;
                while ((1u << d.log2B) < s.B) ++d.log2B;
                d.H = s.H;
                d.hwq = s.HW / 4;
                d.wq = s.W / 4;
                d.hq_count = (s.H + 3u) / 4u;
                d.ipp = d.hq_count * d.wq;
                d.items = s.C * d.ipp;
                d.by_ipp = make_fastdiv(d.ipp);
                d.by_wq = make_fastdiv(d.wq);
                dim3 grid((d.items + 255u) / 256u, s.N);
                if ((s.W * (uint32_t)sizeof(XT)) % 32u != 0 && s.H >= 8u)
                    return launch_pdl(pg_decompress_quad_kernel<XT, LT, Q, DEC_QPT, true>, grid, 256, 0, stream, lfc, packed, stats, (XT*)xhat_dev, d);
                else
                    return launch_pdl(pg_decompress_quad_kernel<XT, LT, Q, DEC_QPT, false>, grid, 256, 0, stream, lfc, packed, stats, (XT*)xhat_dev, d);
            } else if (pg_decompress_flat_ok(s)) {
                PgDecFlat d;
                d.quads = s.total / 4;
                d.HW = s.HW;
                d.W = s.W;
                d.Wb = s.Wb;
                d.TPP = s.TPP;
                d.table_words = flat_table_words(s.HW);
                d.quads_same_plane = (s.HW % 4u == 0) ? 1u : 0u;
                d.by_hw = make_fastdiv(s.HW);
                d.by_w = make_fastdiv(s.W);
                d.by_b = make_fastdiv(s.B);
                const uint64_t g = (d.quads + 256u * DEC_QPT - 1) / (256u * DEC_QPT);
                pg_decompress_flat_kernel<XT, LT, Q, DEC_QPT><<<(unsigned)g, 256, 4u * d.table_words, stream>>>(
                    lfc, packed, stats, (XT*)xhat_dev, d);
            } else {
                const uint64_t g = (nwords + 255) / 256;
                if (g > 0x7FFFFFFFull) return DIV_ERR_SHAPE;
                pg_decompress_general_kernel<XT, LT, Q><<<(unsigned)g, 256, 0, stream>>>(lfc, packed, stats, (XT*)xhat_dev, s, nwords);
            }
            return launch_status();
        });
    });
}

// ------------------------------------------------------------------------------------------------
// 3-D activation maps
// ------------------------------------------------------------------------------------------------
}  // extern "C"

namespace {

div_status check_desc3(const div_desc3d* d) {
    if (!d) return DIV_ERR_NULL;
    if (d->n < 1 || d->c < 1 || d->d < 1 || d->h < 1 || d->w < 1) return DIV_ERR_SHAPE;
    if (d->n >= (1ll << 31) || d->c >= (1ll << 32) || d->d >= (1ll << 32) || d->h >= (1ll << 32) || d->w >= (1ll << 32))
        return DIV_ERR_SHAPE;
    const unsigned __int128 per = (unsigned __int128)d->c * (unsigned __int128)d->d * (unsigned __int128)d->h * (unsigned __int128)d->w;
    if (per >= ((unsigned __int128)1 << 32)) return DIV_ERR_SHAPE;
    if (d->block < 1) return DIV_ERR_PARAM;
    if (!(d->qbits == 1 || d->qbits == 2 || d->qbits == 4 || d->qbits == 8)) return DIV_ERR_PARAM;
    if (!(d->x_dtype == DIV_F32 || d->x_dtype == DIV_BF16)) return DIV_ERR_PARAM;
    if (!(d->lfc_dtype == DIV_F32 || d->lfc_dtype == DIV_BF16)) return DIV_ERR_PARAM;
    return DIV_OK;
}

Shape3 make_shape3(const div_desc3d* d) {
    Shape3 s;
    s.N = (uint32_t)d->n;
    s.C = (uint32_t)d->c;
    s.D = (uint32_t)d->d;
    s.H = (uint32_t)d->h;
    s.W = (uint32_t)d->w;
    uint32_t big = s.D > s.H ? s.D : s.H;
    if (s.W > big) big = s.W;
    s.B = (uint32_t)d->block > big ? big : (uint32_t)d->block;     // a block larger than every side is the largest side
    s.Db = (s.D + s.B - 1) / s.B;
    s.Hb = (s.H + s.B - 1) / s.B;
    s.Wb = (s.W + s.B - 1) / s.B;
    s.P2 = 1;
    while (s.P2 < s.B) s.P2 <<= 1;
    s.HW = s.H * s.W;
    s.DHW = s.D * s.HW;
    s.CDHW = s.C * s.DHW;
    s.TPV = s.Db * s.Hb * s.Wb;
    s.total = (uint64_t)s.N * s.CDHW;
    s.tiles = (uint64_t)s.N * s.C * s.TPV;
    return s;
}

// quad kernels of the 3-D form: 4 consecutive elements share a block
bool quad3_ok(const Shape3& s) { return s.W % 4 == 0 && s.B % 4 == 0 && s.CDHW < (1u << 31) && s.N <= 65535; }
Quad3 make_quad3(const Shape3& s) {
    Quad3 g;
    g.qps = s.CDHW / 4;
    g.C = s.C;
    g.Db = s.Db;
    g.Hb = s.Hb;
    g.Wb = s.Wb;
    g.B = s.B;
    g.qpr = s.W / 4;
    g.qpp = s.H * g.qpr;
    g.qpv = s.D * g.qpp;
    g.by_qpv = make_fastdiv(g.qpv);
    g.by_qpp = make_fastdiv(g.qpp);
    g.by_qpr = make_fastdiv(g.qpr);
    g.by_b = make_fastdiv(s.B);
    return g;
}

// slices as the row kernels take planes: whether they do, and how
bool rows3(const Shape3& s, DecRows3* d) {
    Shape sl = Shape();
    sl.H = s.H;
    sl.W = s.W;
    sl.B = s.B;
    sl.Hb = s.Hb;
    sl.HW = s.HW;
    const uint64_t bands = rows_bands(sl, 1024u * FLAT_QPT);
    if (s.W < 4u || s.CDHW % 4u != 0 || s.CDHW >= (1u << 31) || s.N > 65535u || bands * s.W * 4u > 40000u) return false;
    d->qps = s.CDHW / 4u;
    d->tiles = s.C * s.TPV;
    d->H = s.H;
    d->W = s.W;
    d->Hb = s.Hb;
    d->Wb = s.Wb;
    d->bands = (uint32_t)bands;
    d->step_planes = 1024u / s.W / s.H;
    d->step_rows = 1024u / s.W % s.H;
    d->step_cols = 1024u % s.W;
    d->by_w = make_fastdiv(s.W);
    d->by_h = make_fastdiv(s.H);
    d->by_b = make_fastdiv(s.B);
    d->D = s.D;
    d->Db = s.Db;
    d->by_hb = make_fastdiv(s.Hb);
    d->by_depth = make_fastdiv(s.D);
    return true;
}

void make_layout3(const div_desc3d* d, const Shape3& s, div_layout* out) {
    out->lfc_off = 0;
    out->lfc_bytes = s.tiles * dtype_bytes(d->lfc_dtype);
    out->packed_off = align_up(out->lfc_bytes, SECTION_ALIGN);
    out->packed_bytes = ((s.total * (uint64_t)d->qbits + 31) / 32) * 4;
    out->stats_off = align_up(out->packed_off + out->packed_bytes, SECTION_ALIGN);
    out->stats_bytes = 8ull * s.N;
    out->total_bytes = out->stats_off + out->stats_bytes;
    out->closed_form_bytes = out->lfc_bytes + out->packed_bytes + out->stats_bytes;
    out->raw_bytes = s.total * dtype_bytes(d->x_dtype);
    out->workspace_bytes = align_up(4ull * (WS_HEADER_WORDS + (uint64_t)WS_SLOT_WORDS * s.N), 256);
}

}  // namespace

extern "C" {

div_status div_compressed_bytes_3d(const div_desc3d* desc, div_layout* out) {
    if (!desc || !out) return DIV_ERR_NULL;
    const div_status st = check_desc3(desc);
    if (st != DIV_OK) return st;
    make_layout3(desc, make_shape3(desc), out);
    return DIV_OK;
}

div_status div_compress_3d(const div_desc3d* desc, const void* x_dev, void* comp_dev, size_t comp_capacity,
                           void* workspace_dev, size_t workspace_bytes, uint64_t seed, void* cuda_stream) {
    if (!desc || !x_dev || !comp_dev || !workspace_dev) return DIV_ERR_NULL;
    div_status st = check_desc3(desc);
    if (st != DIV_OK) return st;
    if (!aligned16(x_dev) || !aligned16(comp_dev) || !aligned16(workspace_dev)) return DIV_ERR_ALIGN;
    const Shape3 s = make_shape3(desc);
    div_layout lo;
    make_layout3(desc, s, &lo);
    if (comp_capacity < lo.total_bytes || workspace_bytes < lo.workspace_bytes) return DIV_ERR_CAPACITY;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    if (clear_scratch(workspace_dev, lo.workspace_bytes, stream) != DIV_OK) return DIV_ERR_CUDA;
    uint8_t* blob = (uint8_t*)comp_dev;
    uint32_t* ws = (uint32_t*)workspace_dev;
    // kernels that store bytes or half-words leave the unused top of a partial last word alone: it is zero by contract
    if ((s.total * (uint64_t)desc->qbits) % 32u != 0 &&
        cudaMemsetAsync(blob + lo.packed_off + lo.packed_bytes - 4, 0, 4, stream) != cudaSuccess)
        return DIV_ERR_CUDA;
    const uint64_t nwords = lo.packed_bytes / 4;
    const uint64_t g1 = (s.tiles + 127) / 128, g2 = (nwords + 255) / 256;
    if (g1 > 0x7FFFFFFFull || g2 > 0x7FFFFFFFull) return DIV_ERR_SHAPE;
    return dispatch_types(desc->x_dtype, desc->lfc_dtype, [&](auto* xt, auto* lt) -> div_status {
        typedef std::remove_pointer_t<decltype(xt)> XT;
        typedef std::remove_pointer_t<decltype(lt)> LT;
        // blocks whose padded side fits a warp: a lane per block column (coalesced); else a thread per block
        const uint32_t bpw = s.P2 <= 32u ? 32u / s.P2 : 0u;
        const uint32_t gpr = bpw ? (s.Wb + bpw - 1u) / bpw : 0u;                       // warp groups per row of blocks
        const uint64_t groups = (uint64_t)s.N * s.C * s.Db * s.Hb * gpr;
        const uint64_t gw = (groups + 7u) / 8u;
        // W % 4 == 0 and B = 4 or 8: a lane per strip of 4 columns (16-byte loads)
        const uint64_t strip_slots = (uint64_t)s.N * s.C * s.Db * s.Hb * s.Wb * (s.B / 4u) * 2u;      // two lanes per strip
        const uint64_t gs = (strip_slots + 127u) / 128u;
        div_status st1 = DIV_OK;
        if (s.W % 4u == 0 && (s.B == 4u || s.B == 8u) && s.P2 == s.B && gs <= 0x7FFFFFFFull) {
            const XT* xs = (const XT*)x_dev;
            LT* lf = (LT*)(blob + lo.lfc_off);
            if (s.B == 8u) st1 = launch_pdl(lfc_stats3d_strip_kernel<XT, LT, 8>, dim3((unsigned)gs), 128, 0, stream, xs, lf, ws, s, strip_slots);
            else st1 = launch_pdl(lfc_stats3d_strip_kernel<XT, LT, 4>, dim3((unsigned)gs), 128, 0, stream, xs, lf, ws, s, strip_slots);
        } else if (bpw && gw <= 0x7FFFFFFFull) {
            const XT* xs = (const XT*)x_dev;
            LT* lf = (LT*)(blob + lo.lfc_off);
            switch (s.P2) {
                case 1: st1 = launch_pdl(lfc_stats3d_warp_kernel<XT, LT, 1>, dim3((unsigned)gw), 256, 0, stream, xs, lf, ws, s, gpr, groups); break;
                case 2: st1 = launch_pdl(lfc_stats3d_warp_kernel<XT, LT, 2>, dim3((unsigned)gw), 256, 0, stream, xs, lf, ws, s, gpr, groups); break;
                case 4: st1 = launch_pdl(lfc_stats3d_warp_kernel<XT, LT, 4>, dim3((unsigned)gw), 256, 0, stream, xs, lf, ws, s, gpr, groups); break;
                case 8: st1 = launch_pdl(lfc_stats3d_warp_kernel<XT, LT, 8>, dim3((unsigned)gw), 256, 0, stream, xs, lf, ws, s, gpr, groups); break;
                case 16: st1 = launch_pdl(lfc_stats3d_warp_kernel<XT, LT, 16>, dim3((unsigned)gw), 256, 0, stream, xs, lf, ws, s, gpr, groups); break;
                default: st1 = launch_pdl(lfc_stats3d_warp_kernel<XT, LT, 32>, dim3((unsigned)gw), 256, 0, stream, xs, lf, ws, s, gpr, groups); break;
            }
        } else {
            lfc_stats3d_kernel<XT, LT><<<(unsigned)g1, 128, 0, stream>>>((const XT*)x_dev, (LT*)(blob + lo.lfc_off), ws, s);
        }
        if (st1 != DIV_OK || launch_status() != DIV_OK) return DIV_ERR_CUDA;
        if (s.W % 4u == 0 && (s.B == 4u || s.B == 8u) && s.P2 == s.B && gs <= 0x7FFFFFFFull && desc->qbits != 1) {
            void* packed = blob + lo.packed_off;
            float* stats = (float*)(blob + lo.stats_off);
            const XT* xs = (const XT*)x_dev;
            const LT* lf = (const LT*)(blob + lo.lfc_off);
#define DIVK_Q3(QQ, PP) return launch_pdl(quant3d_strip_kernel<XT, LT, QQ, PP>, dim3((unsigned)gs), 128, 0, stream, xs, lf, ws, packed, stats, s, seed, strip_slots)
            if (s.B == 8u) {
                if (desc->qbits == 2) DIVK_Q3(2, 8); else if (desc->qbits == 4) DIVK_Q3(4, 8); else DIVK_Q3(8, 8);
            } else {
                if (desc->qbits == 2) DIVK_Q3(2, 4); else if (desc->qbits == 4) DIVK_Q3(4, 4); else DIVK_Q3(8, 4);
            }
#undef DIVK_Q3
            return launch_status();
        }
        if (quad3_ok(s) && desc->qbits != 1) {
            const Quad3 g = make_quad3(s);
            const dim3 grid((g.qps + 256u * DEC_QPT - 1) / (256u * DEC_QPT), s.N);
            void* packed = blob + lo.packed_off;
            float* stats = (float*)(blob + lo.stats_off);
            const XT* xs = (const XT*)x_dev;
            const LT* lf = (const LT*)(blob + lo.lfc_off);
            switch (desc->qbits) {
                case 2: return launch_pdl(quant3d_quad_kernel<XT, LT, 2, DEC_QPT>, grid, 256, 0, stream, xs, lf, ws, packed, stats, g, seed);
                case 4: return launch_pdl(quant3d_quad_kernel<XT, LT, 4, DEC_QPT>, grid, 256, 0, stream, xs, lf, ws, packed, stats, g, seed);
                default: return launch_pdl(quant3d_quad_kernel<XT, LT, 8, DEC_QPT>, grid, 256, 0, stream, xs, lf, ws, packed, stats, g, seed);
            }
            return launch_status();
        }
        // Below a million elements the few CTAs wait for their bands' values (5 x 32 x 13 x 13 x 13, B = 4: 10.4 us a thread per word, 14.8 by rows);
        // above, both compress kernels: 11 x 88 x 8 x 50 x 50 142.4 -> 66.6 us, 13 x 88 x 8 x 13 x 13 21.9 -> 19.8, 28 random ones 1.1 to 2.1 times faster.
        // Where a slice is a single row, with a value in shared memory for every element, from two millions on (rows of 11, B = 3: 1.2 million
        // elements 36.1 a thread per word, 39.9 by rows, 3.4 million 115 -> 106).
        DecRows3 d;
        if (desc->qbits != 1 && s.total >= (s.H == 1u ? 1u << 21 : 1u << 20) && rows3(s, &d)) {
            const dim3 grid((d.qps + 256u * FLAT_QPT - 1) / (256u * FLAT_QPT), s.N);
            void* packed = blob + lo.packed_off;
            float* stats = (float*)(blob + lo.stats_off);
            const XT* xs = (const XT*)x_dev;
            const LT* lf = (const LT*)(blob + lo.lfc_off);
            const size_t smem = 4u * d.bands * d.W;
            switch (desc->qbits) {
                case 2: return launch_pdl(quant3d_rows_kernel<XT, LT, 2, FLAT_QPT>, grid, 256, smem, stream, xs, lf, ws, packed, stats, d, seed);
                case 4: return launch_pdl(quant3d_rows_kernel<XT, LT, 4, FLAT_QPT>, grid, 256, smem, stream, xs, lf, ws, packed, stats, d, seed);
                default: return launch_pdl(quant3d_rows_kernel<XT, LT, 8, FLAT_QPT>, grid, 256, smem, stream, xs, lf, ws, packed, stats, d, seed);
            }
        }
        return dispatch_q(desc->qbits, [&](auto q) -> div_status {
            quant_pack3d_kernel<XT, LT, decltype(q)::value><<<(unsigned)g2, 256, 0, stream>>>(
                (const XT*)x_dev, (const LT*)(blob + lo.lfc_off), ws, (uint32_t*)(blob + lo.packed_off),
                (float*)(blob + lo.stats_off), s, seed, nwords);
            return launch_status();
        });
    });
}

div_status div_decompress_3d(const div_desc3d* desc, const void* comp_dev, size_t comp_bytes, void* xhat_dev,
                             void* cuda_stream) {
    if (!desc || !comp_dev || !xhat_dev) return DIV_ERR_NULL;
    div_status st = check_desc3(desc);
    if (st != DIV_OK) return st;
    if (!aligned16(comp_dev) || !aligned16(xhat_dev)) return DIV_ERR_ALIGN;
    const Shape3 s = make_shape3(desc);
    div_layout lo;
    make_layout3(desc, s, &lo);
    if (comp_bytes < lo.total_bytes) return DIV_ERR_CAPACITY;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const uint8_t* blob = (const uint8_t*)comp_dev;
    const uint64_t nwords = lo.packed_bytes / 4;
    const uint64_t g = (nwords + 255) / 256;
    if (g > 0x7FFFFFFFull) return DIV_ERR_SHAPE;
    return dispatch_types(desc->x_dtype, desc->lfc_dtype, [&](auto* xt, auto* lt) -> div_status {
        typedef std::remove_pointer_t<decltype(xt)> XT;
        typedef std::remove_pointer_t<decltype(lt)> LT;
        // B a power of two: slices as the 2-D kernel takes planes, whole rows side by side.  (A lane per half strip of a block, as compress
        // has it, writes runs of a row's length eight slices apart: 8 x 64 x 16 x 56 x 56 27.1 us.)
        if (s.W % 4u == 0 && s.B >= 4u && (s.B & (s.B - 1u)) == 0u && s.N <= 65535u) {
            DecFast3 d;
            d.qps = s.CDHW / 4u;
            d.C = s.C * s.Db;
            d.TPP = s.Hb * s.Wb;
            d.Wb = s.Wb;
            d.log2B = 0;
            while ((1u << d.log2B) < s.B) ++d.log2B;
            d.H = s.H;
            d.hwq = s.HW / 4u;
            d.wq = s.W / 4u;
            d.hq_count = (s.H + 3u) / 4u;
            d.ipp = d.hq_count * d.wq;
            d.items = s.C * s.D * d.ipp;
            d.by_ipp = make_fastdiv(d.ipp);
            d.by_wq = make_fastdiv(d.wq);
            d.D = s.D;
            d.Db = s.Db;
            d.by_depth = make_fastdiv(s.D);
            const dim3 grid((d.items + 255u) / 256u, s.N);
            const bool spread = (s.W * (uint32_t)sizeof(XT)) % 32u != 0 && s.H >= 8u;
            return dispatch_q(desc->qbits, [&](auto q) -> div_status {
                constexpr int Q = decltype(q)::value;
                const LT* lf = (const LT*)(blob + lo.lfc_off);
                const uint32_t* pk = (const uint32_t*)(blob + lo.packed_off);
                const float* stt = (const float*)(blob + lo.stats_off);
                return spread ? launch_pdl(decompress_quad_kernel<XT, LT, Q, DEC_QPT, true, DecFast3>, grid, 256, 0, stream, lf, pk, stt, (XT*)xhat_dev, d)
                              : launch_pdl(decompress_quad_kernel<XT, LT, Q, DEC_QPT, false, DecFast3>, grid, 256, 0, stream, lf, pk, stt, (XT*)xhat_dev, d);
            });
        }
        if (quad3_ok(s)) {
            const Quad3 g3 = make_quad3(s);
            const dim3 grid((g3.qps + 256u * DEC_QPT - 1) / (256u * DEC_QPT), s.N);
            return dispatch_q(desc->qbits, [&](auto q) -> div_status {
                return launch_pdl(decompress3d_quad_kernel<XT, LT, decltype(q)::value, DEC_QPT>, grid, 256, 0, stream,
                                  (const LT*)(blob + lo.lfc_off), (const uint32_t*)(blob + lo.packed_off),
                                  (const float*)(blob + lo.stats_off), (XT*)xhat_dev, g3);
            });
        }
        // other widths and blocks: volumes as the flat 2-D kernel takes planes, where one's quad table and block values fit (up to 8192
        // elements, about twice what a CTA rebuilds).  16 x 56 x 8 x 21 x 21 bfloat16 23.8 -> 5.6 us, 6 x 64 x 13 x 7 x 7 5.9 -> 2.6.
        if (s.CDHW % 4u == 0 && s.CDHW < (1u << 31) && s.DHW <= FLAT_MAX_HW && s.N <= 65535u &&
            flat_smem_bytes(4u * 256u * FLAT_QPT, s.DHW, s.TPV) <= 40000) {
            DecFlat3 d;
            d.qps = s.CDHW / 4u;
            d.C = s.C;
            d.TPP = s.TPV;
            d.Wb = s.Wb;
            d.HW = s.DHW;
            d.W = s.W;
            d.B = s.B;
            d.by_hw = make_fastdiv(s.DHW);
            d.by_w = make_fastdiv(s.W);
            d.by_b = make_fastdiv(s.B);
            const uint32_t per_block = 256u * FLAT_QPT;
            d.table_words = quad_table_words(s.DHW);
            d.period = quad_period(s.DHW);
            d.period_planes = quad_period_planes(s.DHW);
            d.by_period = make_fastdiv(d.period);
            d.planes_per_cta = flat_planes_per_cta(4u * per_block, s.DHW);
            d.slice = s.HW;
            d.tiles = s.Hb * s.Wb;
            d.by_slice = make_fastdiv(s.HW);
            const dim3 grid((d.qps + per_block - 1) / per_block, s.N);
            return dispatch_q(desc->qbits, [&](auto q) -> div_status {
                return launch_pdl(decompress_flat_kernel<XT, LT, decltype(q)::value, FLAT_QPT, DecFlat3>, grid, 256,
                                  flat_smem_bytes(4u * per_block, s.DHW, s.TPV), stream, (const LT*)(blob + lo.lfc_off),
                                  (const uint32_t*)(blob + lo.packed_off), (const float*)(blob + lo.stats_off), (XT*)xhat_dev, d);
            });
        }
        // larger volumes: slices as the row kernel takes planes (4 x 48 x 32 x 50 x 50 65.6 -> 18.8 us, 16 x 16 x 16 x 64 x 21 bfloat16 32.9 -> 8.5)
        DecRows3 d;
        if (rows3(s, &d)) {
            const dim3 grid((d.qps + 256u * FLAT_QPT - 1) / (256u * FLAT_QPT), s.N);
            return dispatch_q(desc->qbits, [&](auto q) -> div_status {
                return launch_pdl(decompress_rows_kernel<XT, LT, decltype(q)::value, FLAT_QPT, DecRows3>, grid, 256, 4u * d.bands * d.W, stream,
                                  (const LT*)(blob + lo.lfc_off), (const uint32_t*)(blob + lo.packed_off),
                                  (const float*)(blob + lo.stats_off), (XT*)xhat_dev, d);
            });
        }
        return dispatch_q(desc->qbits, [&](auto q) -> div_status {
            decompress3d_kernel<XT, LT, decltype(q)::value><<<(unsigned)g, 256, 0, stream>>>(
                (const LT*)(blob + lo.lfc_off), (const uint32_t*)(blob + lo.packed_off), (const float*)(blob + lo.stats_off),
                (XT*)xhat_dev, s, nwords);
            return launch_status();
        });
    });
}

// ------------------------------------------------------------------------------------------------
// ReLU / dropout operators with a packed 1-bit mask
// ------------------------------------------------------------------------------------------------
}  // extern "C"

namespace {
constexpr uint64_t MASK_MAX_TOTAL = 1ull << 40;
inline uint64_t mask_bytes_of(uint64_t total) { return (total + 31) / 32 * 4; }

div_status mask_forward(const void* x_dev, void* y_dev, void* mask_dev, size_t mask_capacity, uint64_t total,
                        int32_t dtype, bool dropout, uint64_t seed, uint32_t drop_threshold, void* cuda_stream) {
    if (!x_dev || !y_dev || !mask_dev) return DIV_ERR_NULL;
    if (total < 1 || total > MASK_MAX_TOTAL) return DIV_ERR_SHAPE;
    if (!(dtype == DIV_F32 || dtype == DIV_BF16) || drop_threshold > 65536u) return DIV_ERR_PARAM;
    if (!aligned16(x_dev) || !aligned16(y_dev) || !aligned16(mask_dev)) return DIV_ERR_ALIGN;
    if (mask_capacity < mask_bytes_of(total)) return DIV_ERR_CAPACITY;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    uint8_t* mask = (uint8_t*)mask_dev;
    // the kernels store one byte per 8 elements: the rest of a partial last word is zero by contract
    if (total % 32u != 0 && cudaMemsetAsync(mask + mask_bytes_of(total) - 4, 0, 4, stream) != cudaSuccess) return DIV_ERR_CUDA;
    const unsigned grid = (unsigned)((total + 2047) / 2048);
    const uint64_t base = rng_sample_base(seed, 0u);
    if (dtype == DIV_F32) {
        if (dropout) mask_forward_kernel<float, true><<<grid, 256, 0, stream>>>((const float*)x_dev, (float*)y_dev, mask, total, base, drop_threshold);
        else mask_forward_kernel<float, false><<<grid, 256, 0, stream>>>((const float*)x_dev, (float*)y_dev, mask, total, base, 0u);
    } else {
        if (dropout) mask_forward_kernel<bf16, true><<<grid, 256, 0, stream>>>((const bf16*)x_dev, (bf16*)y_dev, mask, total, base, drop_threshold);
        else mask_forward_kernel<bf16, false><<<grid, 256, 0, stream>>>((const bf16*)x_dev, (bf16*)y_dev, mask, total, base, 0u);
    }
    return launch_status();
}
}  // namespace

extern "C" {

div_status div_mask_bytes(uint64_t total, uint64_t* out_bytes) {
    if (!out_bytes) return DIV_ERR_NULL;
    if (total < 1 || total > MASK_MAX_TOTAL) return DIV_ERR_SHAPE;
    *out_bytes = mask_bytes_of(total);
    return DIV_OK;
}

div_status div_relu_forward(const void* x_dev, void* y_dev, void* mask_dev, size_t mask_capacity, uint64_t total,
                            int32_t dtype, void* cuda_stream) {
    return mask_forward(x_dev, y_dev, mask_dev, mask_capacity, total, dtype, false, 0, 0, cuda_stream);
}

div_status div_dropout_forward(const void* x_dev, void* y_dev, void* mask_dev, size_t mask_capacity, uint64_t total,
                               int32_t dtype, uint64_t seed, uint32_t drop_threshold, void* cuda_stream) {
    return mask_forward(x_dev, y_dev, mask_dev, mask_capacity, total, dtype, true, seed, drop_threshold, cuda_stream);
}

div_status div_mask_backward(const void* mask_dev, size_t mask_bytes, const void* grad_out_dev, void* grad_in_dev,
                             uint64_t total, int32_t dtype, void* cuda_stream) {
    if (!mask_dev || !grad_out_dev || !grad_in_dev) return DIV_ERR_NULL;
    if (total < 1 || total > MASK_MAX_TOTAL) return DIV_ERR_SHAPE;
    if (!(dtype == DIV_F32 || dtype == DIV_BF16)) return DIV_ERR_PARAM;
    if (!aligned16(mask_dev) || !aligned16(grad_out_dev) || !aligned16(grad_in_dev)) return DIV_ERR_ALIGN;
    if (mask_bytes < mask_bytes_of(total)) return DIV_ERR_CAPACITY;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const unsigned grid = (unsigned)((total + 2047) / 2048);
    if (dtype == DIV_F32)
        mask_backward_kernel<float><<<grid, 256, 0, stream>>>((const uint8_t*)mask_dev, (const float*)grad_out_dev, (float*)grad_in_dev, total);
    else
        mask_backward_kernel<bf16><<<grid, 256, 0, stream>>>((const uint8_t*)mask_dev, (const bf16*)grad_out_dev, (bf16*)grad_in_dev, total);
    return launch_status();
}

div_status div_read_device_status(const void* workspace_dev, void* cuda_stream, int32_t* out_status) {
    if (!workspace_dev || !out_status) return DIV_ERR_NULL;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    int32_t v = 0;
    if (cudaMemcpyAsync(&v, workspace_dev, sizeof(v), cudaMemcpyDeviceToHost, stream) != cudaSuccess) return DIV_ERR_CUDA;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return DIV_ERR_CUDA;
    *out_status = v;
    return DIV_OK;
}

}  // extern "C"
