// Fused plenoctree render kernel for sm_103a: proxy clip -> octree walk ->
// per-leaf SH emission -> front-to-back emission/absorption compositing
// (paper Sec. 4.1, Eq. 3-5; plenoctree of Sec. 4.2 / Sec. 5).
//
// One thread renders one ray at a time.  The grid is persistent: warps take
// rays from a shared counter (32 at a time; small launches give each warp a
// contiguous chunk) and a lane that finishes its ray takes the next one, so
// a warp does not idle behind its longest ray; each iteration of a warp
// moves every live lane past the cell it is in (advance, then composite),
// then descends every lane towards its next cell, at most 4 levels per
// iteration.  Child slots come from the bits of the point's integer
// coordinates on the finest grid.
//
// What bounds it: the latency of the dependent node loads, then instruction
// issue (64% of the issue slots, depth-9 luminaire, 2M rays), at 15% of the
// DRAM bandwidth.  So the walk is built to need few instructions per cell
// and little shared memory (what is left is L1): fixed-point plane parameters
// (below), no staging of the top nodes (the test for it cost more than the
// L1 hits it saved: 18.7 against 16.5 ms for 9M rays at depth 9), and SH
// emission evaluated for 32 leaves at a time from a per-warp queue (walk_rays).
// Before, with double-float positions, staged top nodes and the emission
// evaluated where a ray meets it (9M rays at depth 9, FP32 leaves / 2M at
// depth 8, BF16 leaves, T < 1e-4 stop): 18.4 / 2.95 ms; now 12.6 / 1.88 ms.
//
// Numerics (no FP64 on the device):
//   * Each axis is mirrored so that the ray goes up it.  The parameter at
//     which a ray crosses a plane of the finest grid is a 64-bit fixed-point
//     number, linear in the plane's index, set up once per ray in
//     double-float arithmetic (pairs of floats, ~2^-46).  Segment lengths are
//     differences of such parameters, so every length has ~1e-7 relative
//     error however far the ray origin is, and the cell sequence matches an
//     FP64 walk except for rays passing within ~1e-13 of a cell edge.
//   * The next cell is found by re-descending from the deepest common
//     ancestor (kept on a per-ray stack) with the tie rule "on a plane, go
//     where the direction points", so progress is guaranteed.
//   * Optical depth is accumulated as a compensated (two-float) sum;
//     T = exp(-OD) or max(0, 1 - OD) is recomputed from it after each leaf.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <string>

#include "plo_internal.h"
#include "sh.cuh"

namespace plo {
namespace {

constexpr int BLOCK = 256;
constexpr int WARPS = BLOCK / 32;
constexpr int64_t RENDER_CLAIM = 32;  // rays a warp claims at a time from the shared cursor (32 measured best of 32-128)
constexpr int DESCEND_LEVELS = 4;  // tree levels a descent goes down per step (measured best of 2, 3, 4, 5, 6)
// Lanes without a ray that wait for each other before they take new ones: ray
// setup is about 900 instructions however few lanes run it (4, 6, 8 lanes,
// 9M rays of the depth-9 luminaire: 12.89, 12.75, 12.67 ms).
constexpr int REFILL = 8;

// One packed tree as the kernels see it.
struct TreeParams {
    const uint2* nodes;   // node table walked by the descent (the brick layout's top tree)
    const int32_t* leaf_ids;
    const uint8_t* sh;
    unsigned int* flags;
    const uint2* bricks;  // brick layout: dense bricks below top_depth (NULL: octree layout)
    int32_t brick_log;    // brick side 2^brick_log finest cells
    int32_t top_depth;    // level of the brick cells (= depth for the octree layout)
    int32_t sh_stride;
    int32_t depth;
    int32_t K, prec;
    int32_t max_steps;
    float bmin[3], inv_ext[3], inv_ext_lo[3];  // 1/extent as a double-float
};

struct KParams {
    TreeParams tree;
    int32_t transmittance, activation;
    float l_max, t_stop, sigma_min;
    int32_t saturate, proxy;
    float sphere[4];  // sphere proxy: centre, radius (world space)
    const float* rays;
    unsigned long long* cursor;  // shared claim counter (NULL: static chunks per warp)
    int64_t claim;               // rays a warp claims from it at a time
    int64_t n;
    int64_t chunk;  // rays per warp
    float* rgb;
    float* T;
    int32_t* status;
    // trace mode
    int32_t trace_max;
    int64_t* tr_leaf;
    float* tr_t;
    int32_t* tr_count;
};

// ---------------------------------------------------------------- double-float
struct DF {
    float hi, lo;
};
__device__ __forceinline__ DF two_sum(float a, float b) {
    float s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
__device__ __forceinline__ DF fast_two_sum(float a, float b) {  // |a| >= |b| or a == 0
    float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
// (a_hi + a_lo) * (r_hi + r_lo) with r = 1/d in double-float.
__device__ __forceinline__ DF df_mul(DF a, float rh, float rl) {
    float p = __fmul_rn(a.hi, rh);
    float e = __fmaf_rn(a.hi, rh, -p);
    e = __fmaf_rn(a.hi, rl, e);
    e = __fmaf_rn(a.lo, rh, e);
    return fast_two_sum(p, e);
}
// double-float reciprocal of d = dh + dl (0 < dh <= 1; infinite or NaN where 1/d overflows)
__device__ __forceinline__ void df_recip(float dh, float dl, float& rh, float& rl) {
    asm("rcp.approx.f32 %0, %1;" : "=f"(rh) : "f"(dh));
    float r = __fmaf_rn(-rh, dh, 1.0f);  // residual of the approximate reciprocal (exact)
    r = __fmaf_rn(-rh, dl, r);
    r = __fmul_rn(r, rh);
    const float h = __fadd_rn(rh, r);
    rl = __fsub_rn(r, __fsub_rn(h, rh));
    rh = h;
}
// p + t * d, all double-float
__device__ __forceinline__ DF df_axpy(DF p, DF t, float dh, float dl) {
    float m = __fmul_rn(t.hi, dh);
    float me = __fmaf_rn(t.hi, dh, -m);
    me = __fmaf_rn(t.lo, dh, me);
    me = __fmaf_rn(t.hi, dl, me);
    DF s = two_sum(p.hi, m);
    float lo = __fadd_rn(__fadd_rn(s.lo, p.lo), me);
    return fast_two_sum(s.hi, lo);
}
__device__ __forceinline__ DF df_sub(DF a, DF b) {
    DF s = two_sum(a.hi, -b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fsub_rn(a.lo, b.lo)));
}
// a * b exactly, as a double-float
__device__ __forceinline__ DF two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ DF df_add(DF a, DF b) {
    DF s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ DF df_mul_df(DF a, DF b) {
    DF p = two_prod(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.lo, p.lo);
    e = __fmaf_rn(a.lo, b.hi, e);
    return fast_two_sum(p.hi, e);
}
__device__ __forceinline__ DF df_neg(DF a) { return {-a.hi, -a.lo}; }
// a / b (b.hi != 0): quotient of the high parts plus one correction step
__device__ __forceinline__ DF df_div(DF a, DF b) {
    const float q1 = __fdiv_rn(a.hi, b.hi);
    const DF r = df_sub(a, df_mul_df(b, DF{q1, 0.0f}));
    return fast_two_sum(q1, __fdiv_rn(r.hi, b.hi));
}
// sqrt(a) for a >= 0: one Newton correction of the FP32 root
__device__ __forceinline__ DF df_sqrt(DF a) {
    const float s = __fsqrt_rn(a.hi);
    if (s == 0.0f) return {0.0f, 0.0f};
    const float e = __fadd_rn(__fmaf_rn(-s, s, a.hi), a.lo);
    return fast_two_sum(s, __fdiv_rn(e, __fmul_rn(2.0f, s)));
}
// (P - p) for an exact float plane P
__device__ __forceinline__ DF df_from_plane(float P, DF p) {
    DF n = two_sum(P, -p.hi);
    return two_sum(n.hi, __fsub_rn(n.lo, p.lo));
}
__device__ __forceinline__ bool df_less(DF a, DF b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
__device__ __forceinline__ bool df_eq(DF a, DF b) { return a.hi == b.hi && a.lo == b.lo; }
__device__ __forceinline__ float pow2i(int e) { return __int_as_float((127 + e) << 23); }  // e in [-126, 127]
// Finest-grid coordinate of p on a mirrored axis (depth D, scale = 2^D):
// floor(p 2^D), clamped to [0, 2^D - 1] (the root box is closed).  A point on
// a grid plane belongs to the cell the ray goes into: the one above it, which
// on a mirrored axis is the one below it in the caller's coordinates (the tie
// rule).  Bit D-1-l of the result is the child bit at level l.
__device__ __forceinline__ uint32_t quantize(DF p, float scale, uint32_t qmax) {
    const float h = p.hi * scale;  // exact: scale is a power of two
    const float f = floorf(h);
    int q = (int)f;
    if (h == f && p.lo < 0.0f) --q;
    q = max(q, 0);
    return min((uint32_t)q, qmax);
}

template <int PREC>
__device__ __forceinline__ float decode_sigma(uint32_t y, int prec) {
    if (PREC == PLO_PREC_FP32 || (PREC < 0 && prec == PLO_PREC_FP32)) return __uint_as_float(y);
    return __uint_as_float((y & 0xFFFFFFu) << 7);  // 24-bit float: exponent + 16 mantissa bits
}

// ---------------------------------------------------------------- SH emission
// sum_k c_{ch,k} Y_k(dir) of the three channels of one record.
template <int K, int PREC>
__device__ __forceinline__ void sh_eval(const uint8_t* rec, const float* dir, float& r, float& g, float& b) {
    float Y[K];
    sh_basis<K>(dir[0], dir[BLOCK], dir[2 * BLOCK], Y);
    float acc[3] = {0.0f, 0.0f, 0.0f};
    if (PREC == PLO_PREC_FP32) {
        constexpr int NV = (3 * K + 3) / 4;
        const float4* v = reinterpret_cast<const float4*>(rec);
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            float4 q = __ldg(v + j);
            float e[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                int gi = 4 * j + u;
                if (gi < 3 * K) acc[gi / K] = __fmaf_rn(e[u], Y[gi % K], acc[gi / K]);
            }
        }
    } else {
        constexpr int NV = (3 * K + 7) / 8;
        const uint4* v = reinterpret_cast<const uint4*>(rec);
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            uint4 q = __ldg(v + j);
            uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                int gi = 8 * j + u;
                if (gi < 3 * K) {
                    uint16_t bits = (uint16_t)(w[u >> 1] >> (16 * (u & 1)));
                    float f = PREC == PLO_PREC_FP16 ? __half2float(__ushort_as_half(bits))
                                                    : __uint_as_float((uint32_t)bits << 16);
                    acc[gi / K] = __fmaf_rn(f, Y[gi % K], acc[gi / K]);
                }
            }
        }
    }
    r = acc[0];
    g = acc[1];
    b = acc[2];
}

// The same with K / PREC given at compile time, or read from the tree when
// K == 0 (the batch kernel mixes trees).
template <int K, int PREC>
__device__ __forceinline__ void sh_record(const TreeParams& tp, uint32_t rec, const float* dir, float& r, float& g,
                                          float& b) {
    const uint8_t* p = tp.sh + (size_t)rec * tp.sh_stride;
    if constexpr (K > 0) {
        sh_eval<K, PREC>(p, dir, r, g, b);
    } else {
#define PLO_SH_CASE(KK, PP) \
    if (tp.K == KK && tp.prec == PP) return sh_eval<KK, PP>(p, dir, r, g, b);
        PLO_SH_CASE(16, PLO_PREC_FP32) PLO_SH_CASE(9, PLO_PREC_FP32) PLO_SH_CASE(16, PLO_PREC_FP16)
        PLO_SH_CASE(9, PLO_PREC_FP16) PLO_SH_CASE(16, PLO_PREC_BF16) PLO_SH_CASE(9, PLO_PREC_BF16)
        PLO_SH_CASE(4, PLO_PREC_FP32) PLO_SH_CASE(4, PLO_PREC_FP16) PLO_SH_CASE(4, PLO_PREC_BF16)
        PLO_SH_CASE(1, PLO_PREC_FP32) PLO_SH_CASE(1, PLO_PREC_FP16) PLO_SH_CASE(1, PLO_PREC_BF16)
        PLO_SH_CASE(25, PLO_PREC_FP32) PLO_SH_CASE(25, PLO_PREC_FP16) PLO_SH_CASE(25, PLO_PREC_BF16)
#undef PLO_SH_CASE
        r = g = b = 0.0f;
    }
}

__device__ __forceinline__ float act_fn(float s, int act, float l_max) {
    return act == PLO_ACT_RELU ? fmaxf(s, 0.0f) : l_max / (1.0f + expf(-s));
}

// ---------------------------------------------------------------- per-ray state
// Lane states: idle (no ray), finished (emission still queued, outputs not
// written; _LIMIT: stopped by the step limit), descending to the cell at its
// current point, or at a leaf cell waiting to composite it.
enum : int { ST_IDLE = 0, ST_DONE = 1, ST_DONE_LIMIT = 2, ST_DESCEND = 3, ST_LEAF = 4 };

// The walk's ray parameter is a 64-bit fixed-point number with T_FRAC
// fractional bits.  It counts from the point where the ray enters the proxy,
// in units that make the largest unit-cube direction component lie in
// [1/2, 1) (a power-of-two scaling of the caller's parameter), so it stays
// below 2.  Every axis is mirrored where the direction is negative, so the
// walk only ever goes up: the exit planes of a cell are its upper faces.
constexpr int T_FRAC = 60;
constexpr long long T_CAP = 5ll << (T_FRAC - 1);  // 2.5: the parameter of a plane the ray never reaches
// Two planes crossed within 2^-44 of each other are crossed together, so that
// a ray through a shared edge or corner goes through it in one step instead
// of leaving a sliver segment behind.
constexpr long long T_TIE = 1ll << (T_FRAC - 44);
constexpr float FLAT = 1.0e30f;  // 1 / direction above which an axis counts as parallel to its planes

struct Ray {
    long long t;              // parameter of the current cell's entry
    uint32_t q[3];            // current point on the mirrored finest (depth-D) grid
    float scale;              // caller's parameter per unit of t (a power of two)
    uint32_t flip;            // bit a: axis a is mirrored (= the child-slot bits to flip)
    float T, r, g, b;
    DF od;
    DF t0;           // caller's parameter at t = 0 (trace only)
    long long tend;  // parameter where the ray leaves the sphere proxy (sphere only)
    uint32_t node;   // node whose child is looked up next (ST_DESCEND); the brick while in one
    uint32_t entry_x, entry_y;
    int level;
    int steps;
    int state;
    int brick;  // the current cell is a finest cell of brick `node`
    int tree;   // index into the batch's tree table (batch kernel only)
};

// What a ray keeps per axis from its start to its end, in shared memory, a
// column per thread: registers for it would cost a resident block per SM or
// spills (depth-9 luminaire, 9M rays: 12.9 ms; 13.9 with the 31-bit values in
// registers, 16.3 with everything in registers and 3 blocks).
//
// Finest-grid plane k of the axis lies at parameter A + min(k, kmax) B (mod
// 2^64): one 64-bit multiply-add, the same value whatever the cell it bounds.
// kmax is the first plane behind the ray's end, which keeps the product in
// range however flat the ray is on that axis.  The position is o31 + t d32
// with 31 fractional bits, rounded down.
struct AxisShared {
    ulonglong2 plane[3 * BLOCK];  // A, B
    uint2 pos[3 * BLOCK];         // o31, d32
    uint32_t kmax[3 * BLOCK];
};
__device__ __forceinline__ AxisShared& axes() {
    __shared__ AxisShared s;
    return s;
}
__device__ __forceinline__ long long plane_at(int a, uint32_t k) {
    const ulonglong2 v = axes().plane[a * BLOCK + threadIdx.x];
    return (long long)(v.x + (unsigned long long)min(k, axes().kmax[a * BLOCK + threadIdx.x]) * v.y);
}

// A double-float in [0, 4) as a walk parameter.
__device__ __forceinline__ long long to_fixed(DF v) {
    const float s = 1152921504606846976.0f;  // 2^T_FRAC
    return __float2ll_rn(v.hi * s) + __float2ll_rn(v.lo * s);
}

// Entry of the finest cell R.q of a brick: index = Morton interleave of the
// brick-local coordinates (mirrored back), x lowest.
__device__ __forceinline__ uint32_t spread3(uint32_t x) { return (x & 1u) | ((x & 2u) << 2) | ((x & 4u) << 4); }
__device__ __forceinline__ void load_brick(const TreeParams& tp, Ray& R) {
    const uint32_t smask = (1u << tp.brick_log) - 1u;
    uint32_t m = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a)
        m |= spread3((R.q[a] ^ ((R.flip >> a) & 1u ? smask : 0u)) & smask) << a;
    const uint2 e = __ldg(tp.bricks + ((size_t)R.node << (3 * tp.brick_log)) + m);
    R.entry_x = e.x;
    R.entry_y = e.y;
}

// Child slot, at the level `sh` bits above the finest one, of the point R.q.
__device__ __forceinline__ uint32_t child_slot(const Ray& R, int sh) {
    return (((R.q[0] >> sh) & 1u) | (((R.q[1] >> sh) & 1u) << 1) | (((R.q[2] >> sh) & 1u) << 2)) ^ R.flip;
}

// Descends from R.node (level R.level) towards the leaf or empty octant that
// holds the point, taking the child bits from the finest-grid coordinates
// R.q, and ends in ST_LEAF (in the brick layout also at a finest cell of the
// brick it reaches).  A step goes down at most DESCEND_LEVELS levels; a
// longer descent goes on in the next step while the other lanes composite.
// A lane needs 2 levels per step on average but the warp ran the longest
// descent among its lanes, 5.7 levels (depth-10 luminaire, 16M room rays):
// 4 levels per step measured 348 -> 365 Mrays/s with FP32 leaves, 390 ->
// 397 with FP16; 2 levels gained nothing and 1 level lost.
template <bool BRICKS>
__device__ __forceinline__ void descend_step(const TreeParams& tp, Ray& R, uint32_t* stack) {
    // the child bits of the levels to come, at the top of a word per axis
    uint32_t x[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
        x[a] = (R.q[a] ^ ((R.flip >> a) & 1u ? 0xFFFFFFFFu : 0u)) << (32 - tp.depth + R.level);
    for (int guard = 0; guard < DESCEND_LEVELS; ++guard) {
        uint32_t slot = x[2] >> 31;
        slot = __funnelshift_l(x[1], slot, 1);
        slot = __funnelshift_l(x[0], slot, 1);
#pragma unroll
        for (int a = 0; a < 3; ++a) x[a] <<= 1;
        uint2 e = __ldg(tp.nodes + (size_t)R.node * 8 + slot);
        ++R.level;
        if ((e.x & LEAF_BIT) || R.level >= tp.top_depth) {  // leaf, empty octant, brick (or a malformed table)
            R.state = ST_LEAF;
            if (BRICKS && tp.bricks && !(e.x & LEAF_BIT) && R.level == tp.top_depth) {
                R.node = e.x;
                R.brick = 1;
                R.level = tp.depth;
                load_brick(tp, R);
                return;
            }
            if (!(e.x & LEAF_BIT)) e = make_uint2(ENTRY_EMPTY, 0u);
            R.entry_x = e.x;
            R.entry_y = e.y;
            return;
        }
        stack[R.level * BLOCK] = e.x;
        R.node = e.x;
    }
}

__device__ __forceinline__ void ray_store(const KParams& kp, int64_t i, const Ray& R, int status = PLO_RAY_OK) {
    kp.rgb[3 * i + 0] = R.r;
    kp.rgb[3 * i + 1] = R.g;
    kp.rgb[3 * i + 2] = R.b;
    kp.T[i] = kp.saturate && R.T < kp.t_stop ? 0.0f : R.T;  // a saturated ray is opaque (Sec. 6.2)
    if (kp.status) kp.status[i] = status;
    if (kp.tr_count) kp.tr_count[i] = R.steps;
}

// Proxy clip.  On a hit the lane enters ST_DESCEND at the root and the
// normalised world direction (for the SH basis) is left in dir; on a miss or
// an invalid ray the outputs are written and the lane stays ST_IDLE.
template <bool TRACE, bool SPHERE>
__device__ void ray_begin(const KParams& kp, const TreeParams& tp, int64_t i, Ray& R, uint32_t* stack, float* dir) {
    const float* q = kp.rays + 6 * i;
    float o[3], dw[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        o[a] = __ldg(q + a);
        dw[a] = __ldg(q + 3 + a);
    }
    R.T = 1.0f;
    R.r = R.g = R.b = 0.0f;
    R.od = {0.0f, 0.0f};
    R.steps = 0;
    R.state = ST_IDLE;
    bool bad = dw[0] == 0.0f && dw[1] == 0.0f && dw[2] == 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) bad |= !isfinite(o[a]) || !isfinite(dw[a]);
    if (bad) {
        R.r = R.g = R.b = R.T = __int_as_float(0x7fc00000);
        ray_store(kp, i, R, PLO_RAY_INVALID);
        return;
    }
    const float inv_n = rsqrtf(__fadd_rn(__fadd_rn(__fmul_rn(dw[0], dw[0]), __fmul_rn(dw[1], dw[1])),
                                         __fmul_rn(dw[2], dw[2])));
    // origin and direction in unit-cube coordinates, (o - bmin) / extent in
    // double-float; the direction then scaled by 2^-e
    DF m[3], du[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (!TRACE) dir[a * BLOCK] = __fmul_rn(dw[a], inv_n);
        m[a] = df_mul(two_sum(o[a], -tp.bmin[a]), tp.inv_ext[a], tp.inv_ext_lo[a]);
        du[a] = df_mul(DF{dw[a], 0.0f}, tp.inv_ext[a], tp.inv_ext_lo[a]);
    }
    const float dmax = fmaxf(fabsf(du[0].hi), fmaxf(fabsf(du[1].hi), fabsf(du[2].hi)));
    const int e = max(-125, min(126, (int)(__float_as_uint(dmax) >> 23) - 126));
    const float up = pow2i(e);
    R.scale = pow2i(-e);
    // slab test in double-float, on mirrored axes (the ray goes up): it enters
    // by the faces at 0 and leaves by those at 1
    R.flip = 0u;
    DF tn = {-INFINITY, 0.0f}, tf = {INFINITY, 0.0f};
    DF near_a[3], rd[3];  // rd: 1 / direction
    bool miss = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (du[a].hi < 0.0f) {
            R.flip |= 1u << a;
            du[a] = df_neg(du[a]);
            m[a] = df_from_plane(1.0f, m[a]);
        }
        du[a].hi *= R.scale;
        du[a].lo *= R.scale;
        near_a[a] = {-INFINITY, 0.0f};
        df_recip(du[a].hi, du[a].lo, rd[a].hi, rd[a].lo);
        if (!(rd[a].hi < FLAT)) {  // (nearly) parallel to the slab: never crosses a plane
            miss |= m[a].hi < 0.0f || m[a].hi > 1.0f || (m[a].hi == 0.0f && m[a].lo < 0.0f) ||
                    (m[a].hi == 1.0f && m[a].lo > 0.0f);
            continue;
        }
        const DF t0 = df_mul(df_neg(m[a]), rd[a].hi, rd[a].lo);
        const DF t1 = df_mul(df_from_plane(1.0f, m[a]), rd[a].hi, rd[a].lo);
        near_a[a] = t0;
        if (df_less(tn, t0)) tn = t0;
        if (df_less(t1, tf)) tf = t1;
    }
    if (miss || !df_less(tn, tf) || !(tf.hi > 0.0f || (tf.hi == 0.0f && tf.lo > 0.0f))) {
        ray_store(kp, i, R);
        return;
    }
    if (SPHERE) {
        // sphere proxy (Sec. 5): keep the part of [tn, tf] inside the ball
        // |o + t d - c| <= r, solved once per ray in world space with
        // double-float arithmetic (about 44 significant bits; no FP64 on the
        // device).  With oc = o - c: a t^2 + 2 b t + q = 0, a = d.d,
        // b = oc.d, q = oc.oc - r^2; the root away from -b comes from
        // m = -(b + sign(b) sqrt(b^2 - a q)) as m / a, the other as q / m, so
        // neither subtracts nearly equal numbers.
        DF a2 = {0.0f, 0.0f}, b = {0.0f, 0.0f}, q = {0.0f, 0.0f};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const DF oc = two_sum(o[a], -kp.sphere[a]);
            const DF dd = {dw[a], 0.0f};
            a2 = df_add(a2, two_prod(dw[a], dw[a]));
            b = df_add(b, df_mul_df(oc, dd));
            q = df_add(q, df_mul_df(oc, oc));
        }
        q = df_sub(q, two_prod(kp.sphere[3], kp.sphere[3]));
        const DF disc = df_sub(df_mul_df(b, b), df_mul_df(a2, q));
        if (!(disc.hi > 0.0f || (disc.hi == 0.0f && disc.lo > 0.0f))) {
            ray_store(kp, i, R);
            return;
        }
        const DF sq = df_sqrt(disc);
        const DF m = df_neg(b.hi >= 0.0f ? df_add(b, sq) : df_sub(b, sq));
        const DF r_far = df_div(m, a2), r_near = df_div(q, m);
        const bool mneg = m.hi < 0.0f;
        DF s0 = mneg ? r_far : r_near, s1 = mneg ? r_near : r_far;
        s0 = {s0.hi * up, s0.lo * up};
        s1 = {s1.hi * up, s1.lo * up};
        if (df_less(tn, s0)) tn = s0;
        if (df_less(s1, tf)) tf = s1;
        if (!df_less(tn, tf) || !(tf.hi > 0.0f || (tf.hi == 0.0f && tf.lo > 0.0f))) {
            ray_store(kp, i, R);
            return;
        }
    }
    const bool outside = tn.hi > 0.0f || (tn.hi == 0.0f && tn.lo > 0.0f);
    if (TRACE) R.t0 = outside ? DF{tn.hi * R.scale, tn.lo * R.scale} : DF{0.0f, 0.0f};
    if (SPHERE) {
        const DF rem = outside ? df_sub(tf, tn) : tf;
        R.tend = rem.hi < 2.5f ? to_fixed(rem) : T_CAP;
    }
    const float grid = pow2i(tp.depth), cell = pow2i(-tp.depth);
    const uint32_t qmax = (1u << tp.depth) - 1u;
    R.t = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        DF p = m[a];
        if (outside) p = df_eq(near_a[a], tn) ? DF{0.0f, 0.0f}  // the face it enters by
                                              : df_axpy(p, tn, du[a].hi, du[a].lo);
        if (p.hi < 0.0f) p = {0.0f, 0.0f};  // rounding guard
        if (p.hi > 1.0f || (p.hi == 1.0f && p.lo > 0.0f)) p = {1.0f, 0.0f};
        const uint32_t qa = quantize(p, grid, qmax);
        const uint32_t k1 = qa + 1u;  // the next finest plane
        R.q[a] = qa;
        // position and direction, rounded down
        const uint32_t o31 = (uint32_t)max(0, (int)__float2uint_rd(p.hi * 2147483648.0f) + __float2int_rd(p.lo * 2147483648.0f));
        unsigned long long B = (unsigned long long)T_CAP, first = (unsigned long long)T_CAP;
        uint32_t n = 1, d32 = 0;
        if (rd[a].hi < FLAT) {
            const uint32_t dh = __float2uint_rd(du[a].hi * 4294967296.0f);
            const int dl = __float2int_rd(du[a].lo * 4294967296.0f);
            d32 = dl < 0 && dh < (uint32_t)-dl ? 0u : dh + (uint32_t)dl;
            const DF v = df_mul(df_from_plane((float)k1 * cell, p), rd[a].hi, rd[a].lo);
            if (v.hi < 2.5f) first = (unsigned long long)max(0ll, to_fixed(v));
            const float b = rd[a].hi * cell;
            if (b < 2.5f) {
                B = (unsigned long long)to_fixed(DF{b, rd[a].lo * cell});
                n = __float2uint_rd(2.25f * grid * du[a].hi) + 1u;
            }
        }
        axes().plane[a * BLOCK + threadIdx.x] = make_ulonglong2(first - (unsigned long long)k1 * B, B);
        axes().pos[a * BLOCK + threadIdx.x] = make_uint2(o31, d32);
        axes().kmax[a * BLOCK + threadIdx.x] = k1 + n;
    }
    stack[0] = 0;
    R.node = 0;
    R.level = 0;
    R.brick = 0;
    R.state = ST_DESCEND;
}

// Composites a segment of length `seg` with density sigma > 0 (Eq. 3-5):
// optical depth as a compensated sum, weight w = T_in (1 - e^{-sigma seg}) or
// the linear model's.
__device__ __forceinline__ float composite(const KParams& kp, Ray& R, float sigma, float seg) {
    const float a = sigma * seg;
    const float Tin = R.T;
    const DF s = two_sum(R.od.hi, a);
    R.od = fast_two_sum(s.hi, __fadd_rn(s.lo, R.od.lo));
    if (kp.transmittance == PLO_TRANS_EXP) {
        R.T = expf(-(R.od.hi + R.od.lo));
        return Tin * (-expm1f(-a));
    }
    R.T = fmaxf(0.0f, __fsub_rn(__fsub_rn(1.0f, R.od.hi), R.od.lo));
    const float dT = fminf(Tin, a);
    return kp.transmittance == PLO_TRANS_LINEAR ? dT : 0.5f * dT * (Tin + R.T);
}

// One cell: exit parameter, advance to the next cell, compositing (w: the
// weight of the cell's emission).  Leaves the lane in ST_DESCEND (next cell),
// in ST_LEAF (the next finest cell of the same brick, whose entry the caller
// loads) or in ST_DONE / ST_DONE_LIMIT.
//
// The cell's three upper faces are finest-grid planes, so their parameters
// are one 64-bit multiply-add each, and the segment is the difference of two
// of them, rounded once to FP32: exact to 2^-60 between planes of one axis, to
// the set-up's double-float error (~2^-46) between two axes.  On the axes the ray does
// not leave by, the next cell comes from the 31-bit position, which is
// rounded down and at most 5 units low.  Where that hides a plane the ray has
// just crossed, the next step finds the plane behind it and moves on with an
// empty segment, so nothing is added to the wrong cell and no step is counted.
template <bool TRACE, bool SPHERE, bool BRICKS>
__device__ __forceinline__ void leaf_step(const KParams& kp, const TreeParams& tp, int64_t i, Ray& R,
                                          const uint32_t* stack, float sigma, float& w) {
    const int down = tp.depth - R.level;
    const uint32_t below = (1u << down) - 1u;
    uint32_t k[3];
    long long tk[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        k[a] = (R.q[a] | below) + 1u;
        tk[a] = plane_at(a, k[a]);
    }
    long long te = min(tk[0], min(tk[1], tk[2]));
    bool last = false;  // the sphere proxy ends inside this cell
    if (SPHERE) {
        last = R.tend <= te;
        te = min(te, R.tend);
    }
    te = max(te, R.t);
    const unsigned long long dt = (unsigned long long)(te - R.t);
    const float seg = __fmaf_rn((float)(uint32_t)(dt >> 32), 3.7252902984619140625e-9f,  // 2^(32 - T_FRAC)
                                (float)(uint32_t)dt * 8.673617379884035472e-19f) *       // 2^-T_FRAC
                      R.scale;
    // the empty segment behind a hidden plane is no cell visited (the trace has none)
    if (TRACE || seg > 0.0f) ++R.steps;
    if (TRACE) {
        auto param = [&](long long t) {  // caller's parameter, rounded once
            const float h = (float)(uint32_t)(t >> 37) * R.scale;  // 24 bits: exact
            const float l = (float)(t & ((1ll << 37) - 1)) * R.scale;
            const DF s = two_sum(R.t0.hi, h * 1.1920928955078125e-7f);  // 2^(37 - T_FRAC)
            return __fadd_rn(s.hi, __fadd_rn(__fadd_rn(s.lo, R.t0.lo), l * 8.673617379884035472e-19f));
        };
        const int c = R.steps - 1;
        if (c < kp.trace_max) {
            const size_t o = (size_t)i * kp.trace_max + c;
            kp.tr_leaf[o] = R.entry_x == ENTRY_EMPTY
                                ? -1
                                : __ldg(tp.leaf_ids + (size_t)stack[(R.level - 1) * BLOCK] * 8 + child_slot(R, down));
            kp.tr_t[2 * o] = param(R.t);
            kp.tr_t[2 * o + 1] = param(te);
        }
    }
    R.t = te;
    const uint32_t t31 = (uint32_t)(te >> (T_FRAC - 31));
    const int qs = 31 - tp.depth;
    uint32_t diff = 0u;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const uint2 v = axes().pos[a * BLOCK + threadIdx.x];
        uint32_t qn = (__umulhi(t31, v.y) + v.x) >> qs;
        qn = min(max(qn, R.q[a]), k[a] - 1u);
        if (TRACE) {  // the exact cell: no empty segments in the trace
            if (qn + 1u < k[a] && plane_at(a, qn + 1u) <= te) ++qn;
        }
        if (tk[a] <= te + T_TIE) qn = k[a];
        diff |= qn ^ R.q[a];
        R.q[a] = qn;
    }
    const int msb = 31 - __clz(diff);  // the coarsest plane crossed

    R.state = ST_DONE;
    if (sigma > 0.0f) {
        w = composite(kp, R, sigma, seg);
        if (R.T < kp.t_stop || R.T <= 0.0f) return;
    }
    if (SPHERE && last) return;
    if (R.steps >= tp.max_steps) {
        atomicOr(tp.flags, 1u);
        R.state = ST_DONE_LIMIT;
        return;
    }
    if (msb >= tp.depth) return;  // left the cube
    if (BRICKS) {
        if (R.brick && msb < tp.brick_log) {
            R.state = ST_LEAF;
            return;
        }
        R.brick = 0;
    }
    // from the deepest common ancestor of this cell and the next
    R.level = tp.depth - 1 - msb;
    R.node = stack[R.level * BLOCK];
    R.state = ST_DESCEND;
}

// Rays to walk, given out to the lanes of a warp.
struct Claim {
    int64_t next, end;  // warp-uniform range being handed out
    bool more;          // the shared counter may have more
};

// Walks rays until none is left: the body of both render kernels.  One
// iteration moves every lane that is at a cell past it, then descends every
// lane towards its next cell.  tps: the tree (K > 0), or the batch's tree
// table, its ray offsets and their number (K == 0).
//
// The emission of a leaf is not evaluated where the ray meets it: about 3 of
// a warp's lanes do in an iteration (depth-9 luminaire), and their SH records
// would be read and summed with the other lanes idle.  The lane puts record,
// weight and itself into the warp's queue instead, and the warp evaluates the
// queue when it holds up to 32 entries, one per lane, or when lanes take new
// rays.  Every ray adds its own entries up in the order in which it met them,
// so its result depends on nothing but itself.  (Pulling 16-bit records into
// L2 when the descent finds them, which helped while they were read one
// iteration later, now costs 3%: 9M rays, depth 9, FP16 12.48 -> 12.10 ms
// without it; FP32 records at the time they are queued: +2%.)
template <int K, int PREC, bool TRACE, bool SPHERE, bool BRICKS>
__device__ __forceinline__ void walk_rays(const KParams& kp, const TreeParams* tps, const long long* offs, int n_trees,
                                          uint32_t* stack, Claim cl) {
    __shared__ float4 s_queue[WARPS * 32];
    __shared__ float s_dir[TRACE ? 1 : 3 * BLOCK];  // direction of each lane's ray, a column per lane
    float* dir = s_dir + threadIdx.x;
    float4* queue = s_queue + (threadIdx.x & ~31);
    const int lane = threadIdx.x & 31;
    const unsigned lanes_below = (1u << lane) - 1u;
    int queued = 0;         // entries of the warp's queue
    unsigned mine = 0u;     // which of them are this lane's
    Ray R;
    R.state = ST_IDLE;
    R.tree = 0;
    int64_t my = 0;
    for (;;) {
        // what the lane's cell emits
        float sigma = 0.0f;
        if (R.state == ST_LEAF && R.entry_x != ENTRY_EMPTY) {
            sigma = decode_sigma<PREC>(R.entry_y, K > 0 ? PREC : tps[R.tree].prec);
            if (!(sigma >= kp.sigma_min)) sigma = 0.0f;
        }
        const uint32_t rec = R.entry_x & ~LEAF_BIT;
        const bool emits = !TRACE && sigma > 0.0f && (rec != NO_SH_RECORD || kp.activation != PLO_ACT_RELU);
        const unsigned em = __ballot_sync(0xffffffffu, emits);
        // lanes take new rays in groups: ray setup runs with at least
        // REFILL of them, or when none is left in flight
        const unsigned free = __ballot_sync(0xffffffffu, R.state <= ST_DONE_LIMIT);
        const bool refill =
            free == 0xffffffffu || (__popc(free) >= REFILL && (cl.more || cl.next < cl.end));
        if (!TRACE && queued > 0 && (refill || queued + __popc(em) > 32)) {
            __syncwarp();
            if (lane < queued) {
                const float4 e = queue[lane];
                const uint32_t w = __float_as_uint(e.z);  // owner lane, scale exponent, tree
                const uint32_t r = __float_as_uint(e.x);
                const TreeParams& tp = K > 0 ? tps[0] : tps[w >> 16];
                float c[3] = {0.0f, 0.0f, 0.0f};
                if (r != NO_SH_RECORD) {
                    sh_record<K, PREC>(tp, r, dir + (int)(w & 31u) - lane, c[0], c[1], c[2]);
                    if (K > 0 ? PREC != PLO_PREC_FP32 : tp.prec != PLO_PREC_FP32) {
                        const float sc = pow2i((int)((w >> 8) & 255u) - 127);
                        c[0] *= sc;
                        c[1] *= sc;
                        c[2] *= sc;
                    }
                }
                queue[lane] = make_float4(act_fn(c[0], kp.activation, kp.l_max), e.y,
                                          act_fn(c[1], kp.activation, kp.l_max), act_fn(c[2], kp.activation, kp.l_max));
            }
            __syncwarp();
            while (mine != 0u) {
                const float4 e = queue[__ffs(mine) - 1];
                mine &= mine - 1u;
                R.r = __fmaf_rn(e.y, e.x, R.r);
                R.g = __fmaf_rn(e.y, e.z, R.g);
                R.b = __fmaf_rn(e.y, e.w, R.b);
            }
            __syncwarp();
            queued = 0;
        }
        if (refill) {
            if (R.state == ST_DONE || R.state == ST_DONE_LIMIT) {
                ray_store(kp, my, R, R.state == ST_DONE ? PLO_RAY_OK : PLO_RAY_STEP_LIMIT);
                R.state = ST_IDLE;
            }
            // rays that miss the proxy finish at once, so repeat while lanes
            // are idle and rays remain
            for (;;) {
                const unsigned idle = __ballot_sync(0xffffffffu, R.state == ST_IDLE);
                if (idle == 0u || (__popc(idle) < REFILL && idle != 0xffffffffu)) break;
                if (cl.next >= cl.end) {
                    if (!cl.more) break;
                    unsigned long long b = 0;
                    if (lane == 0) b = atomicAdd(kp.cursor, (unsigned long long)kp.claim);
                    b = __shfl_sync(0xffffffffu, b, 0);
                    if ((int64_t)b >= kp.n) {
                        cl.more = false;
                        break;
                    }
                    cl.next = (int64_t)b;
                    cl.end = min(cl.next + kp.claim, kp.n);
                }
                const int64_t cand = cl.next + __popc(idle & lanes_below);
                cl.next += __popc(idle);
                if (R.state == ST_IDLE && cand < cl.end) {
                    my = cand;
                    if (K == 0) {
                        int t = 0;
                        while (t + 1 < n_trees && offs[t + 1] <= cand) ++t;
                        R.tree = t;
                    }
                    ray_begin<TRACE, SPHERE>(kp, K > 0 ? tps[0] : tps[R.tree], my, R, stack, dir);
                }
            }
            if (__ballot_sync(0xffffffffu, R.state != ST_IDLE) == 0u) break;
        }
        // every other lane is at a leaf, or part-way down a descent longer
        // than one step allows
        const TreeParams& tp = K > 0 ? tps[0] : tps[R.tree];
        if (R.state == ST_LEAF) {
            const int slot = queued + __popc(em & lanes_below);
            float w = 0.0f;
            leaf_step<TRACE, SPHERE, BRICKS>(kp, tp, my, R, stack, sigma, w);
            if (emits) {
                queue[slot] = make_float4(__uint_as_float(rec), w,
                                          __uint_as_float((uint32_t)lane | (R.entry_y >> 24) << 8 | (uint32_t)R.tree << 16),
                                          0.0f);
                mine |= 1u << slot;
            }
            if (BRICKS && R.state == ST_LEAF) load_brick(tp, R);
        }
        queued += __popc(em);
        if (R.state == ST_DESCEND) descend_step<BRICKS>(tp, R, stack);
    }
}

// Resident blocks per SM: 4 (64 registers) hides the dependent node loads
// best; the trace and sphere-proxy kernels keep more per-ray state and
// degree-4 leaves (K = 25) a larger basis, and take 3 (80 registers).
template <int K, int PREC, bool TRACE, bool SPHERE, bool BRICKS>
__global__ void __launch_bounds__(BLOCK, TRACE || SPHERE || BRICKS || K >= 25 ? 3 : 4)
    k_render(KParams kp) {
    // the node id per level of the current cell's path (top_depth + 1 rows,
    // one column per thread): dynamic shared memory sized by the tree, so
    // that a shallow tree leaves more of the SM's memory to L1
    extern __shared__ uint32_t s_stack[];
    uint32_t* stack = s_stack + threadIdx.x;
    const int64_t warp = (int64_t)blockIdx.x * WARPS + (threadIdx.x >> 5);
    Claim cl = {0, 0, kp.cursor != nullptr};
    if (!kp.cursor) {
        cl.next = warp * kp.chunk;
        if (cl.next >= kp.n) return;  // whole warp exits together
        cl.end = min(cl.next + kp.chunk, kp.n);
    }
    walk_rays<K, PREC, TRACE, SPHERE, BRICKS>(kp, &kp.tree, nullptr, 1, stack, cl);
}

// ---------------------------------------------------------------- batched render
// Several luminaires in one launch: rays of tree t occupy [off[t], off[t+1])
// of one concatenated array.  Persistent warps claim `claim` rays at a time
// from a global cursor (one queue for all trees, so uneven ray counts
// balance themselves); lanes refill from the warp's claim as in k_render.
// Leaf precision and SH degree are read from the tree table per ray.
constexpr int MAX_BATCH = 16;
constexpr int BATCH_TOP_NODES = 73;  // levels 0..2 of a full octree (the configuration's largest top_nodes)

struct BatchParams {
    KParams base;  // render parameters, outputs, cursor (base.tree unused)
    TreeParams trees[MAX_BATCH];
    int64_t off[MAX_BATCH + 1];
    int32_t n_trees;
};

template <bool BRICKS>
__global__ void __launch_bounds__(BLOCK, 3)  // 4 blocks per SM spill: 2.64 against 2.45 ms (6 trees, 2.5M rays)
    k_render_batch(BatchParams bp) {
    extern __shared__ uint32_t s_stack[];  // per-thread node stack, as deep as the deepest tree needs
    __shared__ TreeParams s_tp[MAX_BATCH];
    __shared__ long long s_off[MAX_BATCH + 1];
    if (threadIdx.x < bp.n_trees) s_tp[threadIdx.x] = bp.trees[threadIdx.x];
    if (threadIdx.x <= bp.n_trees) s_off[threadIdx.x] = bp.off[threadIdx.x];
    __syncthreads();
    walk_rays<0, -1, false, false, BRICKS>(bp.base, s_tp, s_off, bp.n_trees, s_stack + threadIdx.x,
                                           Claim{0, 0, true});
}

// Point -> leaf lookup: descent from the root with the same tie rule.
__global__ void k_lookup(const uint2* nodes, const int32_t* leaf_ids, int depth, const float* pts, const float* dirs,
                         int64_t n, int64_t* out_leaf, int32_t* out_level) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float p[3], d[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        p[a] = pts[3 * i + a];
        if (dirs) d[a] = dirs[3 * i + a];
    }
    int64_t res = -2;
    int lev = 0;
    if (p[0] >= 0.0f && p[0] <= 1.0f && p[1] >= 0.0f && p[1] <= 1.0f && p[2] >= 0.0f && p[2] <= 1.0f) {
        uint32_t node = 0, c[3] = {0, 0, 0};
        for (lev = 0; lev < depth;) {
            float sc = pow2i(-(lev + 1));
            int slot = 0;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                float m = (float)(2u * c[a] + 1u) * sc;
                int up = p[a] > m || (p[a] == m && d[a] >= 0.0f);
                c[a] = 2u * c[a] + up;
                slot |= up << a;
            }
            uint2 e = __ldg(nodes + (size_t)node * 8 + slot);
            ++lev;
            if (e.x == ENTRY_EMPTY) {
                res = -1;
                break;
            }
            if (e.x & LEAF_BIT) {
                res = __ldg(leaf_ids + (size_t)node * 8 + slot);
                break;
            }
            node = e.x;
        }
    }
    out_leaf[i] = res;
    if (out_level) out_level[i] = lev;
}

// A small wavefront takes as long as its longest ray, and a warp's iteration
// the longer the more lanes it moves, so its rays are spread over 16 warps
// per SM before a warp takes 32 (1,021 rays of the depth-6 luminaire: 106 ->
// 65 us, 16,384: 111 -> 101 us, of the depth-9 one: 292 -> 196 and 331 -> 279
// us; over all the warps that fit, 16,384 rays take 129 and 352 us: the warps
// then wait for each other's instructions).
constexpr int SPREAD_WARPS = 16;

// Persistent grid: as many blocks as fit on the device at once (occupancy
// API), each warp owning a contiguous chunk of the rays.
template <int K, int PREC, bool TRACE, bool SPHERE, bool BRICKS>
cudaError_t launch_k(KParams kp, int sm_count, size_t smem, cudaStream_t s) {
    auto fn = k_render<K, PREC, TRACE, SPHERE, BRICKS>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, BLOCK, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    const int64_t max_warps = (int64_t)sm_count * per_sm * WARPS, few = (int64_t)sm_count * SPREAD_WARPS;
    kp.chunk = std::max((kp.n + max_warps - 1) / max_warps, std::min<int64_t>((kp.n + few - 1) / few, 32));
    const int64_t warps = std::min(max_warps, (kp.n + kp.chunk - 1) / kp.chunk);
    const int64_t grid = (warps + WARPS - 1) / WARPS;
    fn<<<(unsigned)grid, BLOCK, smem, s>>>(kp);
    return cudaGetLastError();
}

template <bool TRACE, bool SPHERE, bool BRICKS>
cudaError_t dispatch(const plo_tree* t, const KParams& kp, size_t smem, cudaStream_t s) {
#define PLO_CASE(KK, PP)                                                   \
    if (t->K == KK && t->precision == PP) return launch_k<KK, PP, TRACE, SPHERE, BRICKS>(kp, t->sm_count, smem, s);
    PLO_CASE(1, PLO_PREC_FP32) PLO_CASE(4, PLO_PREC_FP32) PLO_CASE(9, PLO_PREC_FP32) PLO_CASE(16, PLO_PREC_FP32)
    PLO_CASE(1, PLO_PREC_FP16) PLO_CASE(4, PLO_PREC_FP16) PLO_CASE(9, PLO_PREC_FP16) PLO_CASE(16, PLO_PREC_FP16)
    PLO_CASE(1, PLO_PREC_BF16) PLO_CASE(4, PLO_PREC_BF16) PLO_CASE(9, PLO_PREC_BF16) PLO_CASE(16, PLO_PREC_BF16)
    PLO_CASE(25, PLO_PREC_FP32) PLO_CASE(25, PLO_PREC_FP16) PLO_CASE(25, PLO_PREC_BF16)
#undef PLO_CASE
    return cudaErrorInvalidValue;
}

// Kernel view of a tree.  `walk_bricks`: the brick layout's top tree and
// bricks (render kernels); otherwise the octree node table (trace, and
// trees packed with the octree layout).
void fill_tree_params(const plo_tree* t, const plo_render_params* p, TreeParams* tp, bool walk_bricks = true) {
    const bool bricks = walk_bricks && t->layout == PLO_LAYOUT_BRICKS;
    tp->nodes = static_cast<const uint2*>(bricks ? t->d_top : t->d_nodes);
    tp->bricks = bricks ? static_cast<const uint2*>(t->d_bricks) : nullptr;
    tp->brick_log = bricks ? t->brick_log : 0;
    tp->top_depth = bricks ? t->brick_level : t->depth;
    tp->leaf_ids = t->d_leaf_ids;
    tp->sh = static_cast<const uint8_t*>(t->d_sh);
    tp->flags = t->d_flags;
    tp->sh_stride = t->sh_stride;
    tp->depth = t->depth;
    tp->K = t->K;
    tp->prec = t->precision;
    tp->max_steps = p->max_steps > 0 ? p->max_steps : 4 * (1 << t->depth) + 64;
    for (int a = 0; a < 3; ++a) {
        tp->bmin[a] = t->bbox_min[a];
        tp->inv_ext[a] = t->inv_ext[a];
        tp->inv_ext_lo[a] = t->inv_ext_lo[a];
    }
}

plo_status check_params(const plo_render_params* p) {
    if (!p) return set_error(PLO_ERR_INVALID_ARG, "params is NULL");
    if (p->transmittance < PLO_TRANS_EXP || p->transmittance > PLO_TRANS_LINEAR_LITERAL)
        return set_error(PLO_ERR_INVALID_ARG, "unknown transmittance model");
    if (p->activation != PLO_ACT_RELU && p->activation != PLO_ACT_SIGMOID)
        return set_error(PLO_ERR_INVALID_ARG, "unknown activation");
    if (!(p->t_stop >= 0.0f && p->t_stop <= 1.0f)) return set_error(PLO_ERR_INVALID_ARG, "t_stop must be in [0, 1]");
    if (!(p->sigma_min >= 0.0f) || !std::isfinite(p->sigma_min))
        return set_error(PLO_ERR_INVALID_ARG, "sigma_min must be finite and >= 0");
    if (p->activation == PLO_ACT_SIGMOID && !std::isfinite(p->l_max))
        return set_error(PLO_ERR_INVALID_ARG, "l_max must be finite");
    if (p->max_steps < 0) return set_error(PLO_ERR_INVALID_ARG, "max_steps must be >= 0");
    if (p->saturate != 0 && p->saturate != 1) return set_error(PLO_ERR_INVALID_ARG, "saturate must be 0 or 1");
    if (p->proxy != PLO_PROXY_BOX && p->proxy != PLO_PROXY_SPHERE)
        return set_error(PLO_ERR_INVALID_ARG, "unknown proxy");
    if (p->proxy == PLO_PROXY_SPHERE) {
        for (int a = 0; a < 4; ++a)
            if (!std::isfinite(p->sphere[a])) return set_error(PLO_ERR_INVALID_ARG, "sphere must be finite");
        if (!(p->sphere[3] > 0.0f)) return set_error(PLO_ERR_INVALID_ARG, "sphere radius must be > 0");
    }
    return PLO_OK;
}


// ---------------------------------------------------------------- ray order
// Large wavefronts are rendered in an order that groups rays entering the
// proxy box near each other: a counting sort by the Morton code of the
// entry point's cell on a 32^3 grid of the box (rays that miss it or are
// invalid are spread over the bins) moves the rays into a scratch copy, the render
// kernel runs on the copy unchanged, and its outputs are moved back.
// Neighbouring rays then walk neighbouring cells, so a warp's lanes share
// node and record loads in L1 and L2 (16M rays of the depth-10 tree with the
// sort: 46.0 -> 40.8 ms with FP32 leaves, 39.6 -> 38.2 with FP16; finer keys
// gained no more).  The sort keeps its
// histograms in shared memory: one block per SM counts its contiguous chunk
// of rays, a scan of the (bin, block) table gives every block its slot in
// every bin, and the block scatters its chunk with shared-memory counters
// (a sort with global atomics cost 2.5 ms per 16M rays, more than it
// saved).  Each ray's result does not depend on the order.
constexpr int ORDER_BITS = 5;                       // cells per axis: 2^5
constexpr int ORDER_BINS = 1 << (3 * ORDER_BITS);  // 32768
constexpr int ORDER_THREADS = 1024;
constexpr size_t ORDER_SMEM = (size_t)ORDER_BINS * 4;  // one counter per bin

__device__ __forceinline__ uint32_t order_spread(uint32_t x) {
    uint32_t r = 0;
#pragma unroll
    for (int b = 0; b < ORDER_BITS; ++b) r |= ((x >> b) & 1u) << (3 * b);
    return r;
}

// Bin of a world-space ray: Morton code of the cell where it enters the
// unit cube of the tree (its origin's cell if it starts inside).  Rays that
// miss it (or are invalid) finish at once wherever they are, so they are
// spread over the bins by their index instead of piling into one shared
// counter (a path tracer's wavefront is mostly misses).
__device__ __forceinline__ uint32_t order_bin(const float* q, int64_t i, float3 bmin, float3 inv_ext) {
    const float bm[3] = {bmin.x, bmin.y, bmin.z}, ie[3] = {inv_ext.x, inv_ext.y, inv_ext.z};
    float u[3], du[3];
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = (__ldg(q + a) - bm[a]) * ie[a];
        du[a] = __ldg(q + 3 + a) * ie[a];
        ok &= isfinite(u[a]) && isfinite(du[a]);
    }
    float tn = 0.0f, tf = INFINITY;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (du[a] == 0.0f) {
            ok &= u[a] >= 0.0f && u[a] <= 1.0f;
            continue;
        }
        const float t0 = -u[a] / du[a], t1 = (1.0f - u[a]) / du[a];
        tn = fmaxf(tn, fminf(t0, t1));
        tf = fminf(tf, fmaxf(t0, t1));
    }
    if (!ok || !(tn <= tf)) return (uint32_t)i & (uint32_t)(ORDER_BINS - 1);
    uint32_t c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float e = fminf(fmaxf(__fmaf_rn(tn, du[a], u[a]), 0.0f), 1.0f) * (float)(1 << ORDER_BITS);
        c[a] = min((uint32_t)e, (1u << ORDER_BITS) - 1u);
    }
    return order_spread(c[0]) | (order_spread(c[1]) << 1) | (order_spread(c[2]) << 2);
}

// Block b counts the bins of rays [b chunk, (b+1) chunk): bins[i], and
// table[bin * gridDim.x + b] = its count of that bin.
__global__ void __launch_bounds__(ORDER_THREADS) k_order_count(const float* rays, int64_t n, int64_t chunk,
                                                               float3 bmin, float3 inv_ext, uint16_t* bins,
                                                               uint32_t* table) {
    extern __shared__ uint32_t s_cnt[];
    for (int j = threadIdx.x; j < ORDER_BINS; j += ORDER_THREADS) s_cnt[j] = 0u;
    __syncthreads();
    const int64_t beg = (int64_t)blockIdx.x * chunk, end = min(beg + chunk, n);
    for (int64_t i = beg + threadIdx.x; i < end; i += ORDER_THREADS) {
        const uint32_t b = order_bin(rays + 6 * i, i, bmin, inv_ext);
        bins[i] = (uint16_t)b;
        atomicAdd(s_cnt + b, 1u);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < ORDER_BINS; j += ORDER_THREADS) table[(size_t)j * gridDim.x + blockIdx.x] = s_cnt[j];
}

// After the exclusive scan of the table: block b gives each ray of its chunk
// the next free position of its bin's slot: order[pos] = i, inv[i] = pos.
__global__ void __launch_bounds__(ORDER_THREADS) k_order_scatter(int64_t n, int64_t chunk, const uint16_t* bins,
                                                                 const uint32_t* table, uint32_t* order,
                                                                 uint32_t* inv) {
    extern __shared__ uint32_t s_pos[];
    for (int j = threadIdx.x; j < ORDER_BINS; j += ORDER_THREADS) s_pos[j] = table[(size_t)j * gridDim.x + blockIdx.x];
    __syncthreads();
    const int64_t beg = (int64_t)blockIdx.x * chunk, end = min(beg + chunk, n);
    for (int64_t i = beg + threadIdx.x; i < end; i += ORDER_THREADS) {
        const uint32_t pos = atomicAdd(s_pos + bins[i], 1u);
        order[pos] = (uint32_t)i;
        inv[i] = pos;
    }
}

// The rays in order: rays_s[pos] = rays[order[pos]] (writes in order, so
// only the reads are scattered).
__global__ void k_order_rays(const float* rays, int64_t n, const uint32_t* order, float* rays_s) {
    const int64_t pos = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (pos >= n) return;
    const float* src = rays + 6 * (int64_t)__ldg(order + pos);  // the caller's rays are only 4-byte aligned
    float* dst = rays_s + 6 * pos;
#pragma unroll
    for (int k = 0; k < 6; ++k) dst[k] = __ldg(src + k);
}

// The outputs back in ray order: ray i's from position inv[i] (writes in
// ray order, reads scattered).
__global__ void k_order_outputs(const uint32_t* inv, int64_t n, const float* rgb_s, const float* T_s,
                                const int32_t* st_s, float* rgb, float* T, int32_t* st) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const int64_t pos = __ldg(inv + i);
    rgb[3 * i] = __ldg(rgb_s + 3 * pos);
    rgb[3 * i + 1] = __ldg(rgb_s + 3 * pos + 1);
    rgb[3 * i + 2] = __ldg(rgb_s + 3 * pos + 2);
    T[i] = __ldg(T_s + pos);
    if (st) st[i] = __ldg(st_s + pos);
}

// ---------------------------------------------------------------- work distribution
// Large wavefronts are handed out dynamically: warps claim RENDER_CLAIM rays
// at a time from a counter allocated for the call, so a warp whose rays are
// long does not hold up the end of the launch (static per-warp chunks are
// kept below DYNAMIC_MIN_RAYS, where they measure as fast and a call must not
// allocate: 300,000, 400,000 and a million rays of the depth-8 luminaire take
// 442, 545 and 1141 us with chunks, 457, 541 and 1082 us with the counter).
constexpr int64_t DYNAMIC_MIN_RAYS = (int64_t)3 << 17;
// Below this many the chunks cost little, so a call that cannot have the
// counter (no memory left) or should not (a captured graph with an allocation
// in it can be instantiated only once) runs without it.
constexpr int64_t DYNAMIC_ALWAYS_RAYS = (int64_t)1 << 20;
// Wavefronts of at least this many rays are also put in entry-cell order
// (above): its fixed cost (a 5M-entry table per call) outweighs the gain on
// smaller ones.  The line is where the two are even: depth-9 luminaire, 3M rays
// 4.63 ms without and 4.70 with the order, 9M rays the same; depth-10, 16M
// rays 46.0 and 40.8.
constexpr int64_t ORDER_MIN_RAYS = (int64_t)1 << 23;

template <bool TRACE>
plo_status render_common(const plo_tree* t, const float* d_rays, int64_t n, const plo_render_params* p,
                         float* d_rgb, float* d_T, int32_t* d_status, int32_t trace_max, int64_t* tr_leaf,
                         float* tr_t, int32_t* tr_count, void* stream) {
    if (!t) return set_error(PLO_ERR_INVALID_ARG, "tree is NULL");
    plo_status st = check_params(p);
    if (st != PLO_OK) return st;
    if (n < 0) return set_error(PLO_ERR_INVALID_ARG, "n must be >= 0");
    if (n == 0) return PLO_OK;
    if (!d_rays || !d_rgb || !d_T) return set_error(PLO_ERR_INVALID_ARG, "rays, rgb or T is NULL");
    if (TRACE && (trace_max <= 0 || !tr_leaf || !tr_t || !tr_count))
        return set_error(PLO_ERR_INVALID_ARG, "trace buffers are NULL or max_cells <= 0");
    if (TRACE && p->proxy != PLO_PROXY_BOX)
        return set_error(PLO_ERR_UNSUPPORTED, "plo_trace_rays follows the box proxy only");
    KParams kp{};
    fill_tree_params(t, p, &kp.tree, !TRACE);
    kp.transmittance = p->transmittance;
    kp.activation = p->activation;
    kp.l_max = p->l_max;
    kp.t_stop = p->t_stop;
    kp.sigma_min = p->sigma_min;
    kp.saturate = p->saturate;
    kp.proxy = p->proxy;
    for (int a = 0; a < 4; ++a) kp.sphere[a] = p->sphere[a];
    kp.rays = d_rays;
    kp.n = n;
    kp.rgb = d_rgb;
    kp.T = d_T;
    kp.status = d_status;
    kp.trace_max = trace_max;
    kp.tr_leaf = tr_leaf;
    kp.tr_t = tr_t;
    kp.tr_count = tr_count;
    const size_t smem = (size_t)(kp.tree.top_depth + 1) * BLOCK * 4;
    cudaError_t e = cudaSuccess;
    cudaStream_t cs = (cudaStream_t)stream;
    unsigned long long* cursor = nullptr;
    uint32_t* inv = nullptr;
    float *rgb_s = nullptr, *T_s = nullptr;
    int32_t* st_s = nullptr;
    const bool ordered = !TRACE && n >= ORDER_MIN_RAYS;
    bool counted = !TRACE && n >= DYNAMIC_MIN_RAYS && !ordered;
    if (counted && n < DYNAMIC_ALWAYS_RAYS) {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(cs, &capture) != cudaSuccess) cudaGetLastError();
        counted = capture == cudaStreamCaptureStatusNone;
    }
    if (counted) {
        e = (cudaError_t)tree_malloc_async(t, (void**)&cursor, sizeof(unsigned long long), cs);
        if (e == cudaErrorMemoryAllocation && n < DYNAMIC_ALWAYS_RAYS) {
            cudaGetLastError();
            cursor = nullptr;
            e = cudaSuccess;
        }
        if (e == cudaSuccess && cursor) e = cudaMemsetAsync(cursor, 0, sizeof(unsigned long long), cs);
        if (e != cudaSuccess) {
            scratch_free_async(cursor, cs);
            return cuda_error(e, "render work counter");
        }
        kp.cursor = cursor;
        kp.claim = cursor ? RENDER_CLAIM : kp.claim;
    }
    if (ordered) {
        // one scratch block: the claim counter, the (bin, block) table, the
        // order and its inverse, the rays and outputs in that order, each
        // ray's bin
        const int nblk = t->sm_count;
        const int64_t chunk = (n + nblk - 1) / nblk;
        auto up = [](size_t b) { return (b + 255) / 256 * 256; };
        const size_t o_table = 256, o_order = o_table + up((size_t)ORDER_BINS * nblk * 4);
        const size_t o_inv = o_order + up((size_t)n * 4);
        const size_t o_rays = o_inv + up((size_t)n * 4), o_rgb = o_rays + up((size_t)n * 24);
        const size_t o_T = o_rgb + up((size_t)n * 12), o_st = o_T + up((size_t)n * 4);
        const size_t o_bins = o_st + (d_status ? up((size_t)n * 4) : 0), total = o_bins + up((size_t)n * 2);
        e = (cudaError_t)tree_malloc_async(t, (void**)&cursor, total, cs);
        if (e == cudaSuccess) e = cudaMemsetAsync(cursor, 0, 256, cs);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_order_count, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)ORDER_SMEM);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_order_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)ORDER_SMEM);
        if (e == cudaSuccess) {
            uint8_t* base = reinterpret_cast<uint8_t*>(cursor);
            uint32_t* table = reinterpret_cast<uint32_t*>(base + o_table);
            uint32_t* order = reinterpret_cast<uint32_t*>(base + o_order);
            inv = reinterpret_cast<uint32_t*>(base + o_inv);
            float* rays_s = reinterpret_cast<float*>(base + o_rays);
            rgb_s = reinterpret_cast<float*>(base + o_rgb);
            T_s = reinterpret_cast<float*>(base + o_T);
            st_s = d_status ? reinterpret_cast<int32_t*>(base + o_st) : nullptr;
            uint16_t* bins = reinterpret_cast<uint16_t*>(base + o_bins);
            const float3 bmin = make_float3(t->bbox_min[0], t->bbox_min[1], t->bbox_min[2]);
            const float3 iext = make_float3(t->inv_ext[0], t->inv_ext[1], t->inv_ext[2]);
            k_order_count<<<nblk, ORDER_THREADS, ORDER_SMEM, cs>>>(d_rays, n, chunk, bmin, iext, bins, table);
            e = cudaGetLastError();
            if (e == cudaSuccess) e = device_exclusive_scan(table, table, (int64_t)ORDER_BINS * nblk, cs, t);
            if (e == cudaSuccess) {
                k_order_scatter<<<nblk, ORDER_THREADS, ORDER_SMEM, cs>>>(n, chunk, bins, table, order, inv);
                k_order_rays<<<(unsigned)((n + 255) / 256), 256, 0, cs>>>(d_rays, n, order, rays_s);
                e = cudaGetLastError();
            }
            kp.rays = rays_s;
            kp.rgb = rgb_s;
            kp.T = T_s;
            kp.status = st_s;
        }
        if (e != cudaSuccess) {
            scratch_free_async(cursor, cs);
            return cuda_error(e, "render work counter and ray order");
        }
        kp.cursor = cursor;
        kp.claim = RENDER_CLAIM;
    }
    const bool bricks = !TRACE && t->layout == PLO_LAYOUT_BRICKS;
    if (TRACE)
        e = dispatch<TRACE, false, false>(t, kp, smem, (cudaStream_t)stream);
    else if (kp.proxy == PLO_PROXY_SPHERE)
        e = bricks ? dispatch<false, true, true>(t, kp, smem, (cudaStream_t)stream)
                   : dispatch<false, true, false>(t, kp, smem, (cudaStream_t)stream);
    else
        e = bricks ? dispatch<false, false, true>(t, kp, smem, (cudaStream_t)stream)
                   : dispatch<false, false, false>(t, kp, smem, (cudaStream_t)stream);
    if (e == cudaSuccess && inv) {
        k_order_outputs<<<(unsigned)((n + 255) / 256), 256, 0, cs>>>(inv, n, rgb_s, T_s, st_s, d_rgb, d_T, d_status);
        e = cudaGetLastError();
    }
    scratch_free_async(cursor, cs);
    if (e != cudaSuccess) return cuda_error(e, "render kernel launch");
    return PLO_OK;
}

}  // namespace
}  // namespace plo

using namespace plo;

extern "C" plo_status plo_render_rays(const plo_tree* tree, const float* d_rays, int64_t n,
                                      const plo_render_params* params, float* d_rgb, float* d_T, int32_t* d_status,
                                      void* stream) {
    return render_common<false>(tree, d_rays, n, params, d_rgb, d_T, d_status, 0, nullptr, nullptr, nullptr,
                                stream);
}

extern "C" plo_status plo_trace_rays(const plo_tree* tree, const float* d_rays, int64_t n,
                                     const plo_render_params* params, int32_t max_cells, int64_t* d_leaf,
                                     float* d_t, int32_t* d_count, void* stream) {
    // The trace runs the render kernel itself (trace instantiation); its
    // radiance goes to a stream-ordered temporary and is discarded.
    if (!tree) return set_error(PLO_ERR_INVALID_ARG, "tree is NULL");
    if (n < 0) return set_error(PLO_ERR_INVALID_ARG, "n must be >= 0");
    if (n == 0) return PLO_OK;
    float* rgbT = nullptr;
    cudaError_t e = (cudaError_t)tree_malloc_async(tree, (void**)&rgbT, (size_t)n * 4 * sizeof(float), (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_error(e, "trace scratch allocation");
    plo_status st = render_common<true>(tree, d_rays, n, params, rgbT, rgbT + 3 * n, nullptr, max_cells, d_leaf,
                                        d_t, d_count, stream);
    scratch_free_async(rgbT, (cudaStream_t)stream);
    return st;
}

extern "C" plo_status plo_lookup_points(const plo_tree* t, const float* d_points, const float* d_dirs, int64_t n,
                                        int64_t* d_leaf, int32_t* d_level, void* stream) {
    if (!t) return set_error(PLO_ERR_INVALID_ARG, "tree is NULL");
    if (n < 0) return set_error(PLO_ERR_INVALID_ARG, "n must be >= 0");
    if (n == 0) return PLO_OK;
    if (!d_points || !d_leaf) return set_error(PLO_ERR_INVALID_ARG, "points or leaf output is NULL");
    int64_t grid = (n + 255) / 256;
    k_lookup<<<(unsigned)grid, 256, 0, (cudaStream_t)stream>>>(static_cast<const uint2*>(t->d_nodes), t->d_leaf_ids,
                                                               t->depth, d_points, d_dirs, n, d_leaf, d_level);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "lookup kernel launch");
    return PLO_OK;
}

// ---------------------------------------------------------------- allocation-free host path
// plo_render_rays_host_noalloc: the host-buffer render for callers that must
// not allocate device memory (see include/plo.h).  Its device staging for
// rays and results is the file-scope array below, so the call itself makes
// no cudaMalloc/cudaFree and no allocating library call.
namespace {

constexpr int64_t kNoAllocMaxRays = 262144;  // 10 floats per ray: 10 MiB in all
// plo_render_rays takes a stream-ordered work counter from DYNAMIC_MIN_RAYS
// rays up; every call of this path stays below that, so it never allocates.
static_assert(kNoAllocMaxRays < DYNAMIC_MIN_RAYS,
              "the allocation-free path must stay below the ray count at which plo_render_rays allocates");
// rays [max][6], then rgb [max][3], then T [max].  Every GPU that loads the
// library holds this array until the process exits.  All calls share it.
__device__ __align__(256) float g_noalloc_stage[kNoAllocMaxRays * 10];

// Device addresses of the staging array, one per CUDA context seen: a new
// primary context (after cudaDeviceReset, say) gets its own lookup instead
// of a stale address.
constexpr int kNoAllocMaxContexts = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_ctx[kNoAllocMaxContexts] = {};
float* g_noalloc_ptr[kNoAllocMaxContexts] = {};
int g_noalloc_used = 0;

using CtxGetCurrentFn = int (*)(void**);  // cuCtxGetCurrent(CUcontext*)

CtxGetCurrentFn ctx_get_current() {
    static CtxGetCurrentFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<CtxGetCurrentFn>(p);
    });
    return fn;
}

// Device address of the staging array in the current context.  In host
// code g_noalloc_stage names a host-side stand-in, never the device memory,
// so only this address may be used.
plo_status noalloc_stage(float** out) {
    CtxGetCurrentFn get = ctx_get_current();
    if (!get) return set_error(PLO_ERR_CUDA, "cuCtxGetCurrent is not available from the driver");
    void* ctx = nullptr;
    if (get(&ctx) != 0 || !ctx) return set_error(PLO_ERR_CUDA, "no current CUDA context");
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    for (int k = 0; k < g_noalloc_used; ++k)
        if (g_noalloc_ctx[k] == ctx) {
            *out = g_noalloc_ptr[k];
            return PLO_OK;
        }
    if (g_noalloc_used == kNoAllocMaxContexts)
        return set_error(PLO_ERR_UNSUPPORTED, "too many CUDA contexts for the allocation-free path's table");
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_stage);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress of the no-allocation staging array");
    g_noalloc_ctx[g_noalloc_used] = ctx;
    g_noalloc_ptr[g_noalloc_used] = static_cast<float*>(p);
    ++g_noalloc_used;
    *out = static_cast<float*>(p);
    return PLO_OK;
}

}  // namespace

extern "C" plo_status plo_render_rays_host_noalloc(const plo_tree* tree, const float* h_rays, int64_t n,
                                                   const plo_render_params* params, float* h_rgb, float* h_T,
                                                   void* stream) {
    if (!tree) return set_error(PLO_ERR_INVALID_ARG, "tree is NULL");
    if (n < 0) return set_error(PLO_ERR_INVALID_ARG, "n must be >= 0");
    if (n > kNoAllocMaxRays)
        return set_error(PLO_ERR_INVALID_ARG, "n = " + std::to_string(n) +
                                                  " exceeds the allocation-free path's maximum of " +
                                                  std::to_string(kNoAllocMaxRays) + " rays per call");
    if (n == 0) return PLO_OK;
    if (!h_rays || !h_rgb || !h_T) return set_error(PLO_ERR_INVALID_ARG, "rays, rgb or T is NULL");
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
    if (dev != tree->device)
        return set_error(PLO_ERR_INVALID_ARG, "the tree lives on another device than the current one");
    float* base = nullptr;
    plo_status st = noalloc_stage(&base);
    if (st != PLO_OK) return st;
    float* d_rays = base;
    float* d_rgb = base + 6 * kNoAllocMaxRays;
    float* d_T = base + 9 * kNoAllocMaxRays;
    cudaStream_t s = (cudaStream_t)stream;
    e = cudaMemcpyAsync(d_rays, h_rays, (size_t)n * 6 * sizeof(float), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_error(e, "host-to-device ray copy");
    st = plo_render_rays(tree, d_rays, n, params, d_rgb, d_T, nullptr, stream);
    if (st != PLO_OK) return st;
    e = cudaMemcpyAsync(h_rgb, d_rgb, (size_t)n * 3 * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h_T, d_T, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_error(e, "plo_render_rays_host_noalloc");
    return PLO_OK;
}

// ---------------------------------------------------------------- batch handle
struct plo_batch {
    BatchParams bp;
    int32_t n_trees;
    int64_t n_rays;
    size_t smem;
    int sm_count;
    int device;
    plo_batch_config cfg;
    bool bricks;                  // some tree uses the brick layout
    unsigned long long* d_cursor;
    cudaGraph_t graph;
    cudaGraphExec_t exec;
};

namespace {

void apply_config(plo_batch* b) {
    int rows = 1;
    for (int t = 0; t < b->n_trees; ++t) rows = std::max(rows, b->bp.trees[t].top_depth + 1);
    b->smem = (size_t)rows * BLOCK * 4;
}

void (*batch_kernel(const plo_batch* b))(BatchParams) {
    return b->bricks ? k_render_batch<true> : k_render_batch<false>;
}

cudaError_t launch_batch(plo_batch* b, cudaStream_t s) {
    auto fn = batch_kernel(b);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b->smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, BLOCK, b->smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    const int bps = b->cfg.blocks_per_sm > 0 && b->cfg.blocks_per_sm < per_sm ? b->cfg.blocks_per_sm : per_sm;
    int64_t warps_needed = (b->n_rays + 31) / 32;
    int64_t grid = std::min<int64_t>((warps_needed + WARPS - 1) / WARPS, (int64_t)b->sm_count * bps);
    if (grid < 1) return cudaSuccess;
    // the configured claim is an upper bound: a warp's claims are at most a
    // sixteenth of its even share, so that the end of the queue is spread over
    // all warps (6 trees, 2.5M rays, claims of 256, 128, 64, 32: 2.77, 2.59,
    // 2.49, 2.45 ms; 3 trees, 300k rays: 1.09, 0.64, 0.53, 0.46 ms)
    const int64_t share = b->n_rays / (grid * WARPS * 16) / 32 * 32;
    b->bp.base.claim = std::max<int64_t>(32, std::min<int64_t>(b->cfg.claim_rays, share));
    e = cudaMemsetAsync(b->d_cursor, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    fn<<<(unsigned)grid, BLOCK, b->smem, s>>>(b->bp);
    return cudaGetLastError();
}

void set_buffers(plo_batch* b, const float* d_rays, float* d_rgb, float* d_T, int32_t* d_status) {
    b->bp.base.rays = d_rays;
    b->bp.base.rgb = d_rgb;
    b->bp.base.T = d_T;
    b->bp.base.status = d_status;
}

void drop_graph(plo_batch* b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
}

}  // namespace

extern "C" plo_status plo_batch_create(const plo_tree* const* trees, int32_t n_trees, const int64_t* ray_offsets,
                                       const plo_render_params* params, plo_batch** out) {
    if (!out) return set_error(PLO_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!trees || !ray_offsets) return set_error(PLO_ERR_INVALID_ARG, "trees or ray_offsets is NULL");
    if (n_trees < 1 || n_trees > MAX_BATCH)
        return set_error(PLO_ERR_INVALID_ARG, "n_trees must be in [1, " + std::to_string(MAX_BATCH) + "]");
    plo_status st = check_params(params);
    if (st != PLO_OK) return st;
    if (params->proxy != PLO_PROXY_BOX)
        return set_error(PLO_ERR_UNSUPPORTED, "the batch render clips to each tree's box (PLO_PROXY_BOX only)");
    if (ray_offsets[0] != 0) return set_error(PLO_ERR_INVALID_ARG, "ray_offsets[0] must be 0");
    for (int t = 0; t < n_trees; ++t) {
        if (!trees[t]) return set_error(PLO_ERR_INVALID_ARG, "a tree is NULL");
        if (ray_offsets[t + 1] < ray_offsets[t]) return set_error(PLO_ERR_INVALID_ARG, "ray_offsets must not decrease");
        if (t > 0 && trees[t]->device != trees[0]->device)
            return set_error(PLO_ERR_INVALID_ARG, "all trees must live on one device");
    }
    plo_batch* b = new (std::nothrow) plo_batch();
    if (!b) return set_error(PLO_ERR_OOM, "host allocation failed");
    b->n_trees = n_trees;
    b->n_rays = ray_offsets[n_trees];
    b->device = trees[0]->device;
    b->sm_count = trees[0]->sm_count;
    KParams& kp = b->bp.base;
    kp.transmittance = params->transmittance;
    kp.activation = params->activation;
    kp.l_max = params->l_max;
    kp.t_stop = params->t_stop;
    kp.sigma_min = params->sigma_min;
    kp.saturate = params->saturate;
    kp.proxy = PLO_PROXY_BOX;
    kp.n = b->n_rays;
    for (int t = 0; t < n_trees; ++t) {
        fill_tree_params(trees[t], params, &b->bp.trees[t]);
        b->bricks |= trees[t]->layout == PLO_LAYOUT_BRICKS;
    }
    for (int t = 0; t <= n_trees; ++t) b->bp.off[t] = ray_offsets[t];
    b->bp.n_trees = n_trees;
    b->cfg = {256, 0, BATCH_TOP_NODES};
    apply_config(b);
    int e = dev_malloc((void**)&b->d_cursor, 256);
    if (e != 0) {
        delete b;
        return cuda_error(e, "batch cursor allocation");
    }
    b->bp.base.cursor = b->d_cursor;
    *out = b;
    return PLO_OK;
}

extern "C" void plo_batch_free(plo_batch* b) {
    if (!b) return;
    cudaDeviceSynchronize();
    drop_graph(b);
    cudaFree(b->d_cursor);
    delete b;
}

extern "C" plo_status plo_batch_set_config(plo_batch* b, const plo_batch_config* cfg) {
    if (!b || !cfg) return set_error(PLO_ERR_INVALID_ARG, "batch or config is NULL");
    if (cfg->claim_rays < 32 || cfg->claim_rays > (1 << 20) || cfg->claim_rays % 32)
        return set_error(PLO_ERR_INVALID_ARG, "claim_rays must be a multiple of 32 in [32, 2^20]");
    if (cfg->blocks_per_sm < 0 || cfg->top_nodes < 0 || cfg->top_nodes > BATCH_TOP_NODES)
        return set_error(PLO_ERR_INVALID_ARG, "blocks_per_sm must be >= 0, top_nodes in [0, 73]");
    b->cfg = *cfg;
    apply_config(b);
    drop_graph(b);
    return PLO_OK;
}

extern "C" plo_status plo_batch_get_config(const plo_batch* b, plo_batch_config* cfg) {
    if (!b || !cfg) return set_error(PLO_ERR_INVALID_ARG, "batch or config is NULL");
    *cfg = b->cfg;
    return PLO_OK;
}

extern "C" plo_status plo_batch_render(plo_batch* b, const float* d_rays, float* d_rgb, float* d_T,
                                       int32_t* d_status, void* stream) {
    if (!b) return set_error(PLO_ERR_INVALID_ARG, "batch is NULL");
    if (b->n_rays == 0) return PLO_OK;
    if (!d_rays || !d_rgb || !d_T) return set_error(PLO_ERR_INVALID_ARG, "rays, rgb or T is NULL");
    set_buffers(b, d_rays, d_rgb, d_T, d_status);
    cudaError_t e = launch_batch(b, (cudaStream_t)stream);
    return e == cudaSuccess ? PLO_OK : cuda_error(e, "batch render launch");
}

extern "C" plo_status plo_batch_capture(plo_batch* b, const float* d_rays, float* d_rgb, float* d_T,
                                        int32_t* d_status, void* stream) {
    if (!b) return set_error(PLO_ERR_INVALID_ARG, "batch is NULL");
    if (!d_rays || !d_rgb || !d_T) return set_error(PLO_ERR_INVALID_ARG, "rays, rgb or T is NULL");
    drop_graph(b);
    set_buffers(b, d_rays, d_rgb, d_T, d_status);
    cudaStream_t cs = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cuda_error(e, "capture stream");
    // the occupancy query and attribute set happen outside the capture
    e = cudaFuncSetAttribute(batch_kernel(b), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b->smem);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        cudaError_t le = launch_batch(b, cs);
        e = cudaStreamEndCapture(cs, &b->graph);
        if (e == cudaSuccess) e = le;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
    cudaStreamDestroy(cs);
    (void)stream;
    if (e != cudaSuccess) {
        drop_graph(b);
        return cuda_error(e, "batch graph capture");
    }
    return PLO_OK;
}

extern "C" plo_status plo_batch_replay(plo_batch* b, void* stream) {
    if (!b) return set_error(PLO_ERR_INVALID_ARG, "batch is NULL");
    if (!b->exec) return set_error(PLO_ERR_INVALID_ARG, "no captured graph: call plo_batch_capture first");
    cudaError_t e = cudaGraphLaunch(b->exec, (cudaStream_t)stream);
    return e == cudaSuccess ? PLO_OK : cuda_error(e, "batch graph launch");
}

extern "C" plo_status plo_batch_autotune(plo_batch* b, const float* d_rays, float* d_rgb, float* d_T, int32_t reps,
                                         void* stream, plo_batch_config* best_out, float* best_ms) {
    if (!b || !best_out) return set_error(PLO_ERR_INVALID_ARG, "batch or output is NULL");
    if (!d_rays || !d_rgb || !d_T) return set_error(PLO_ERR_INVALID_ARG, "rays, rgb or T is NULL");
    if (reps < 1) reps = 1;
    cudaStream_t s = (cudaStream_t)stream;
    set_buffers(b, d_rays, d_rgb, d_T, nullptr);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const plo_batch_config saved = b->cfg;
    plo_batch_config best = saved;
    float best_t = 1e30f;
    const int claims[] = {32, 64, 128, 256, 1024};
    const int bpss[] = {0, 1, 2};
    cudaError_t err = cudaSuccess;
    for (int ci = 0; ci < 5 && err == cudaSuccess; ++ci)
        for (int bi = 0; bi < 3 && err == cudaSuccess; ++bi) {
            b->cfg = {claims[ci], bpss[bi], saved.top_nodes};
            apply_config(b);
            err = launch_batch(b, s);  // warm-up
            if (err != cudaSuccess) break;
            cudaEventRecord(e0, s);
            for (int r = 0; r < reps && err == cudaSuccess; ++r) err = launch_batch(b, s);
            cudaEventRecord(e1, s);
            cudaEventSynchronize(e1);
            float ms = 0.0f;
            cudaEventElapsedTime(&ms, e0, e1);
            ms /= (float)reps;
            if (ms < best_t) {
                best_t = ms;
                best = b->cfg;
            }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->cfg = err == cudaSuccess ? best : saved;
    apply_config(b);
    drop_graph(b);
    if (err != cudaSuccess) return cuda_error(err, "batch autotune");
    *best_out = best;
    if (best_ms) *best_ms = best_t;
    return PLO_OK;
}
