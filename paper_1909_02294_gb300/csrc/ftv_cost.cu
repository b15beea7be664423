// Segment x depth-label matching-cost volume: the persistent cost kernel.
//
// Paper: Eq. 4 (L1 distance of Y, Cb, Cr between a reference point and its transform T[.] into a
// neighbouring view for the considered depth), Eq. 1 (costs of the neighbouring views c' in D are
// combined for every segment of every view), Sec. III-A (segments are the units; depth per segment).
// Here every pixel of a segment is a sample point (window of one pixel), the per-pixel costs of the
// neighbours are combined by min or sum, and the segment's cost is the int32 sum over its pixels.
//
// Work decomposition (GB300 design, not the paper's CPU threading of Sec. IV-A): a work item is one
// tile of kTile consecutive pixels of the listed segments (segments in list order, each segment's
// pixels contiguous) times one block of LB consecutive labels of one (job, reference) unit. Resident
// CTAs take items from a global counter in increasing order, so CTAs that run together work on
// neighbouring tiles and label blocks and share their neighbour-view footprints in L2. Per item:
//   - the N x LB homographies and the neighbour geometry are staged in shared memory; the tile's pixel box then
//     tells which entries sample no pixel, which sample every pixel in view (no tests), and which need the tests;
//   - each label's neighbours are listed by class, so that the pixel loop has no dispatch for the common class;
//   - each thread owns kPPT pixels (position and reference samples in registers), a warp kWarpPix consecutive ones;
//   - for each label, for each listed neighbour: projection, one packed-texel gather, |dY|+|dCb|+|dCr|,
//     running min/sum per pixel in registers;
//   - per label, each run of equal segments among the warp's pixels is summed (in the thread, then one warp
//     reduction and one shared atomic per run), and at the end of the item each segment's row slice is
//     written: plain stores for segments wholly inside the tile, global atomics for segments cut by a tile
//     boundary.
// Positions and segments come from the tile records (tile_kernel), so that an item starts with one dependent load
// instead of a search; a 480x270 8-bit frame's launch went from 86 to 30 us with them and the plan's label blocks.
// The kernel is bound by instruction issue and, where most samples miss the tests, by the L1's data stage (about 80 %
// busy on the 4K rig), so instructions per evaluation decide its time. With one offset per in-view integer-shift entry
// (no tests, no row arithmetic), the listed classes, the sums in the thread and the packed comparisons below, the
// 1920x1080 8-view 250-label rig went from 29.0 to 17.9 ms per launch (24.2 to 16 instructions per evaluation), the
// 3840x2160 15-view 400-label rig from 506 to 435 ms.
// All arithmetic that decides a sample position is explicit round-to-nearest FP32 (no contraction
// freedom is left to the compiler), so the result is bit-identical to any implementation of the same
// sequence; costs are integers, so summation order does not matter.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <climits>
#include <mutex>

#include "ftv_internal.h"
#include "ftv_project.cuh"

namespace ftv {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kSentinel = INT_MAX;
constexpr int kWarpPix = 32 * kPPT;  // consecutive records of one warp
constexpr int kMaxRuns = 48;         // runs of equal segments among a warp's records (more: each pixel on its own)

// Ref: a reference pixel's samples in the form cost() compares. cost(): |dY| + |dCb| + |dCr|, exact integers.
template <int FMT>
struct TexelOps;

// 8-bit samples: one packed absolute difference sums all four bytes (the fourth is zero on both sides).
template <>
struct TexelOps<FMT_U8X4> {
    struct Ref {
        uint32_t t;
    };
    static __device__ __forceinline__ Ref load_ref(const void* base, int64_t i) {
        return {__ldg(static_cast<const uint32_t*>(base) + i)};
    }
    static __device__ __forceinline__ int cost(const void* base, int i, const Ref& r) {
        return (int)__vsadu4(__ldg(static_cast<const uint32_t*>(base) + i), r.t);
    }
};

template <>
struct TexelOps<FMT_P10> {
    struct Ref {
        int a, b, c;
    };
    static __device__ __forceinline__ Ref load_ref(const void* base, int64_t i) {
        const uint32_t t = __ldg(static_cast<const uint32_t*>(base) + i);
        return {(int)(t & 0x3ff), (int)((t >> 10) & 0x3ff), (int)(t >> 20)};
    }
    static __device__ __forceinline__ int cost(const void* base, int i, const Ref& r) {
        const uint32_t t = __ldg(static_cast<const uint32_t*>(base) + i);
        return (int)__sad((int)(t & 0x3ff), r.a, __sad((int)((t >> 10) & 0x3ff), r.b, __sad((int)(t >> 20), r.c, 0u)));
    }
};

// a.lo * lo + a.hi * hi + c with the unsigned 16-bit halves of a (every product and sum fits int).
template <int LO, int HI>
__device__ __forceinline__ int dot_halves(uint32_t a, int c) {
    int d;
    asm("dp2a.lo.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"((LO & 0xff) | ((HI & 0xff) << 8)), "r"(c));
    return d;
}

// 9- to 14-bit samples with their sum S = Y + Cb + Cr in the fourth half-word: |y - r| = y + r - 2 min(y, r), so
// the cost is S + S_r - 2 (the three minima): two packed minima and two dot products (S passes through the
// second minimum against 0xffff; S <= 3 * 16383).
template <>
struct TexelOps<FMT_U16S> {
    struct Ref {
        uint32_t a, b;
        int s;
    };
    static __device__ __forceinline__ Ref load_ref(const void* base, int64_t i) {
        const uint2 t = __ldg(static_cast<const uint2*>(base) + i);
        return {t.x, t.y | 0xffff0000u, (int)(t.y >> 16)};
    }
    static __device__ __forceinline__ int cost(const void* base, int i, const Ref& r) {
        const uint2 t = __ldg(static_cast<const uint2*>(base) + i);
        return dot_halves<-2, 1>(__vminu2(t.y, r.b), dot_halves<-2, -2>(__vminu2(t.x, r.a), r.s));
    }
};

template <>
struct TexelOps<FMT_U16X4> {
    struct Ref {
        int a, b, c;
    };
    static __device__ __forceinline__ Ref load_ref(const void* base, int64_t i) {
        const uint2 t = __ldg(static_cast<const uint2*>(base) + i);
        return {(int)(t.x & 0xffff), (int)(t.x >> 16), (int)t.y};
    }
    static __device__ __forceinline__ int cost(const void* base, int i, const Ref& r) {
        const uint2 t = __ldg(static_cast<const uint2*>(base) + i);
        return (int)__sad((int)(t.x & 0xffff), r.a, __sad((int)(t.x >> 16), r.b, __sad((int)t.y, r.c, 0u)));
    }
};

// Staged per-(neighbour, label) entry: the FP32 homography and the neighbour's geometry, 48 bytes so
// that a thread fetches it with three 128-bit shared loads. `pm` holds the row pitch (low 28 bits)
// and the entry's evaluation mode (high bits):
//   kGeneral  projective homography, evaluated as written in the contract;
//   kAffine   h6 == h7 == 0: Wz = fma(h6, x, fma(h7, y, h8)) is exactly h8 for every pixel, so
//             r = 1/h8 is computed once at staging time and stored in place of h6;
//   kUnit     affine with r == 1: u = X * 1 is exactly X, the multiplications are skipped;
//   kRect     unit with h0 = 1, h1 = 0, h3 = 0, h4 = 1, |h5| < 0.25 (rectified rigs: the row is kept):
//             X = fma(1, x, fma(0, y, h2)) is x + h2 rounded once, and Y = y + h5 rounded once lies
//             within 0.25 + 2^-9 of the integer y < 2^15, so floor(Y + 0.5) is exactly y;
//   kShift    rectified, and the column is x + D for every x < 2^15 with D = floor(h2 + 0.5) (FP64-precision
//             units: see shift_fp64; the FP32 contract: s = x + h2
//             rounded is within 2^-24 (|x| + |h2|) of x + h2; when h2 + 0.5 lies more than twice that
//             from every integer (checked at staging with |x| < 2^15, |h2| < 2^20), s + 0.5 lies more than
//             2^-24 from every integer, where rounding s + 0.5 cannot cross one (below 1 in magnitude its
//             rounding error is at most 2^-24; above, s + 0.5 is exact or only crosses into a binade
//             whose lower end is the integer below it), so floor((s + 0.5) rounded) = x + D. Used when the
//             view's pitch is the reference width and its height at least the reference height: the
//             sample's index is then the pixel's y * W + x plus D, the row needs no test, and the column
//             test is -D <= x < w - D, staged as floats (h[6], h[7]) with D in h[8];
//   kShiftIn  kShift whose every sample of the item's tile is in view (the tile's columns lie within the bounds);
//             h[0] of a kShift entry holds the view's texel offset in the unit's allocation (NbrView::off);
//   kOut      affine with 1/h8 not finite and positive, or no pixel of the item's tile can reach the view
//             (box_class): every sample is out of view;
//   kIn       projective, and at every pixel of the item's tile Wz > 2^-92 and the sample rounds into the
//             view (box_class): r = 1/Wz is a normal reciprocal (no subnormal scaling) and neither the
//             finite-reciprocal test nor a range test can fail, so none is made;
//   kFront    projective, Wz > 2^-92 at every pixel of the tile (box_class): the reciprocal needs no
//             subnormal scaling and is finite and positive; the range tests remain.
// All of them give bit-identical results to the general sequence; they only skip work whose result
// is known exactly.
struct __align__(16) HEntry {
    float h[9];
    uint32_t w, h_, pm;
};
enum : uint32_t { kGeneral = 0, kAffine = 1, kUnit = 2, kOut = 3, kRect = 4, kSlow = 5, kShift = 6, kIn = 7, kFront = 8,
                kShiftIn = 9 };

// FP64-projection entries (kKindPrecise) stage local-frame coefficients in HEntry::h (stage_precise) and
// this alongside: the integer column u0 and row v0 the frame is shifted by, and the tie-test thresholds.
struct __align__(16) PEntry {
    int32_t u0, v0;
    float thr_u, thr_v;
};
constexpr uint32_t kPitchMask = (1u << 28) - 1u;
constexpr float kRound = 0x1.8p23f;  // t + kRound rounds t (|t| < 2^21) to an integer, held in the sum's low bits
constexpr int kRoundBits = 0x4b400000;

__device__ __forceinline__ bool finite_positive(float r) {
    return (unsigned)(__float_as_int(r) - 1) < 0x7f7fffffu;
}

// Position of one sample: reference pixel (x, y) through homography e.h into one neighbour view.
// Returns whether it is in view and its texel index. Equivalent to the contract's float test (Wz > 0,
// 0 <= floor(u + 0.5) <= W - 1, ...): the host guarantees |h| <= 2^100, so X and Y are finite;
// r = 1/Wz is then finite and positive exactly when Wz > 0 and 1/Wz does not overflow (if it does, u
// is +-inf or NaN and the contract says "out"); with finite positive r, u + 0.5 is finite or +-inf,
// and floor-to-int with saturation followed by an unsigned range test decides "in view" exactly as
// the float compares do.
template <bool FAST_RCP>
__device__ __forceinline__ bool pos_general(const float4& a, const float4& b, const float4& c, int pitch, float x,
                                            float y, int& idx) {
    const float X = __fmaf_rn(a.x, x, __fmaf_rn(a.y, y, a.z));
    const float Yh = __fmaf_rn(a.w, x, __fmaf_rn(b.x, y, b.y));
    const float Wz = __fmaf_rn(b.z, x, __fmaf_rn(b.w, y, c.x));
    const float r = contract_rcp<FAST_RCP>(Wz);
    const int ui = __float2int_rd(__fadd_rn(__fmul_rn(X, r), 0.5f));
    const int vi = __float2int_rd(__fadd_rn(__fmul_rn(Yh, r), 0.5f));
    idx = vi * pitch + ui;
    return finite_positive(r) & ((unsigned)ui < __float_as_uint(c.y)) & ((unsigned)vi < __float_as_uint(c.z));
}

// Affine entries: r (finite, positive) was hoisted out of the pixel loop; UNIT means r == 1.
template <bool UNIT>
__device__ __forceinline__ bool pos_affine(const float4& a, const float4& b, const float4& c, float r, int pitch,
                                           float x, float y, int& idx) {
    const float X = __fmaf_rn(a.x, x, __fmaf_rn(a.y, y, a.z));
    const float Yh = __fmaf_rn(a.w, x, __fmaf_rn(b.x, y, b.y));
    const float u = UNIT ? X : __fmul_rn(X, r);
    const float v = UNIT ? Yh : __fmul_rn(Yh, r);
    const int ui = __float2int_rd(__fadd_rn(u, 0.5f));
    const int vi = __float2int_rd(__fadd_rn(v, 0.5f));
    idx = vi * pitch + ui;
    return ((unsigned)ui < __float_as_uint(c.y)) & ((unsigned)vi < __float_as_uint(c.z));
}

// Rectified entries (kRect): u = x + h2, the sample row is the reference row y.
__device__ __forceinline__ bool pos_rect(float h2, uint32_t wv, uint32_t hv, int pitch, float x, int iy, int& idx) {
    const int ui = __float2int_rd(__fadd_rn(__fadd_rn(x, h2), 0.5f));
    idx = iy * pitch + ui;
    return ((unsigned)ui < wv) & ((unsigned)iy < hv);
}

// Folds one sample into the pixel's running combination over views (min or sum). With the kernel's PF
// (min only, the penalty at least the largest possible sample cost) the running minimum starts at the
// penalty, which an out-of-view sample cannot lower; the projective path then lets only in-view
// samples update it (PF here), which pays off where many samples fall outside (wide convergent
// baselines), while the rectified and affine paths keep the select form, measured faster there. Both
// forms give the minimum over in-view costs and penalties of the contract.
//
// Checked builds (FTV_CHECKED): every gather is first tested against the neighbour view's texel count lim;
// an index outside it is recorded in the launch's plan (ST_CHECKED) and the sample is skipped, so a path
// whose in-view claim were wrong shows up as a status instead of an out-of-bounds read. Regular builds drop
// the test (lim and status are unused).
__device__ __forceinline__ bool checked_gather(bool ok, int idx, unsigned lim, uint32_t* status) {
#ifdef FTV_CHECKED
    if (ok && (unsigned)idx >= lim) {
        atomicOr(status, ST_CHECKED);
        return false;
    }
#else
    (void)idx;
    (void)lim;
    (void)status;
#endif
    return ok;
}

template <int FMT, int COMB, bool PF>
__device__ __forceinline__ void accumulate(int& m, bool ok, const void* tex, int idx,
                                           const typename TexelOps<FMT>::Ref& ref, int penalty, unsigned lim,
                                           uint32_t* status) {
    ok = checked_gather(ok, idx, lim, status);
    if (COMB == FTV_COMBINE_MIN && PF) {
        if (ok) m = min(m, TexelOps<FMT>::cost(tex, idx, ref));
    } else {
        int cst = penalty;
        if (ok) cst = TexelOps<FMT>::cost(tex, idx, ref);
        m = COMB == FTV_COMBINE_MIN ? min(m, cst) : m + cst;
    }
}

// The same for a sample known to be in view.
template <int FMT, int COMB>
__device__ __forceinline__ void accumulate_in(int& m, const void* tex, int idx, const typename TexelOps<FMT>::Ref& ref,
                                              int penalty, unsigned lim, uint32_t* status) {
#ifdef FTV_CHECKED
    accumulate<FMT, COMB, false>(m, true, tex, idx, ref, penalty, lim, status);
#else
    (void)penalty;
    (void)lim;
    (void)status;
    const int cst = TexelOps<FMT>::cost(tex, idx, ref);
    m = COMB == FTV_COMBINE_MIN ? min(m, cst) : m + cst;
#endif
}

// Classifies a projective entry for the pixel box [x0, x1] x [y0, y1] (x, y >= 0) under the FP32 contract,
// from the homography evaluated at the box's four corners:
//   kOut     no pixel can sample the wv x hv view. At every corner the point lies left of u = -1 (X + Wz < 0),
//            right of u = wv (X - wv Wz > 0), above v = -1 or below v = hv (the same with Y), or behind the
//            camera (Wz < 0);
//   kIn      at every pixel Wz > 2^-92 and the sample rounds into the view. At every corner Wz is positive
//            (and above 2^-90), X and Y are positive, and (wv - 1) Wz - X and (hv - 1) Wz - Y are positive;
//   kFront   at every pixel Wz > 2^-92 (the corners as for kIn, Wz only);
//   kGeneral otherwise.
// Each corner condition carries a margin of 2^-20 times the magnitude of its terms (sx = |h0| x + |h1| y +
// |h2|, likewise sy, sz). Why the conclusions hold at every pixel: the contract's two fused multiply-adds
// put X, Y and Wz within 2^-23 of those magnitudes of their exact values, at any pixel and at the corners.
// With the margin, each corner condition implies, in exact arithmetic, a condition linear (convex, for
// kOut) in the pixel position with half the margin (for Wz: Wz - 2^-22 sz - 2^-92 > 0), which therefore
// holds at every pixel of the box, and there the FP32 value keeps the sign the conclusion needs:
//   Wz_f32 > 2^-92, so r = 1/Wz is finite, positive and the reciprocal of a normal float;
//   X_f32 >= 0, so u = X r >= 0 and floor(u + 0.5) >= 0;
//   X_f32 <= (wv - 1) Wz_f32, so u <= (wv - 1)(1 + 2^-23) < wv - 1 + 2^-7 (wv <= 2^15), u + 0.5 rounds
//   below wv and floor(u + 0.5) <= wv - 1 (the same for rows);
//   for kOut as before: a point left of u = -1 has u + 0.5 < 0 after rounding, one right of u = wv rounds to
//   a column of at least wv, one behind the camera has Wz <= 0.
// |h| <= 2^100 keeps every term finite; an overflow or a NaN fails the comparisons and gives kGeneral.
__device__ __forceinline__ uint32_t box_class(const float* h, float x0, float x1, float y0, float y1, float wv,
                                              float hv) {
    const float m = 0x1p-20f;
    const float wv1 = wv - 1.0f, hv1 = hv - 1.0f;
    bool left = true, right = true, top = true, bottom = true, behind = true;
    bool front = true, inside = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float x = (k & 1) ? x1 : x0, y = (k & 2) ? y1 : y0;  // x, y >= 0
        const float X = __fmaf_rn(h[0], x, __fmaf_rn(h[1], y, h[2]));
        const float Y = __fmaf_rn(h[3], x, __fmaf_rn(h[4], y, h[5]));
        const float Z = __fmaf_rn(h[6], x, __fmaf_rn(h[7], y, h[8]));
        const float sx = __fmaf_rn(fabsf(h[0]), x, __fmaf_rn(fabsf(h[1]), y, fabsf(h[2])));
        const float sy = __fmaf_rn(fabsf(h[3]), x, __fmaf_rn(fabsf(h[4]), y, fabsf(h[5])));
        const float sz = __fmaf_rn(fabsf(h[6]), x, __fmaf_rn(fabsf(h[7]), y, fabsf(h[8])));
        const float tl = __fadd_rn(X, Z), tr = __fmaf_rn(-wv, Z, X);
        const float tt = __fadd_rn(Y, Z), tb = __fmaf_rn(-hv, Z, Y);
        left = left && tl < -m * (sx + sz + fabsf(tl));
        right = right && tr > m * (sx + wv * sz + fabsf(tr));
        top = top && tt < -m * (sy + sz + fabsf(tt));
        bottom = bottom && tb > m * (sy + hv * sz + fabsf(tb));
        behind = behind && Z < -m * (sz + fabsf(Z));
        front = front && Z > fmaxf(m * (sz + fabsf(Z)), 0x1p-90f);
        const float ir = __fmaf_rn(wv1, Z, -X), ib = __fmaf_rn(hv1, Z, -Y);
        inside = inside && X > m * (sx + fabsf(X)) && Y > m * (sy + fabsf(Y)) &&
                 ir > m * (sx + wv1 * sz + fabsf(ir)) && ib > m * (sy + hv1 * sz + fabsf(ib));
    }
    if (left || right || top || bottom || behind) return kOut;
    if (front) return inside ? kIn : kFront;
    return kGeneral;
}

// Integer-shift entries of the FP64 projection (linear rigs with parallel axes): the unrounded homography
// is exactly [[1, 0, h2], [0, 1, h5], [0, 0, 1]] with |h5| < 0.49 and |h2| < 2^20. The FP64 projection then
// computes X = x + h2 (one rounding; 1 * x and 0 * y are exact), Wz = 1 and X / Wz = X exactly, and
// floor(X + 0.5) rounded once more; likewise the row from y + h5. g = h2 + 0.5 is exact (|h2| < 2^20), and
// with D = floor(g):
//   g an integer: x + h2 = x + D - 0.5 and x + D are exact, so the column is x + D;
//   otherwise the two roundings move x + h2 + 0.5 by less than 2^-31 (|x + h2 + 0.5| < 2^21, unit roundoff
//   2^-53), so when g lies more than 2^-30 from every integer the column is floor(x + g) = x + D.
// The row is y: y + h5 + 0.5 lies in (y + 0.01, y + 0.99) and moves by less than 2^-35.
// Then every pixel's sample is (x + D, y), in view exactly when 0 <= x + D < wv (the view being at least as
// tall as the reference). Returns whether the entry has this form, with D.
__device__ __forceinline__ bool shift_fp64(const double* __restrict__ hg, int& D) {
    const double h0 = __ldg(&hg[0]), h1 = __ldg(&hg[1]), h2 = __ldg(&hg[2]), h3 = __ldg(&hg[3]), h4 = __ldg(&hg[4]),
                 h5 = __ldg(&hg[5]), h6 = __ldg(&hg[6]), h7 = __ldg(&hg[7]), h8 = __ldg(&hg[8]);
    if (!(h0 == 1.0 && h1 == 0.0 && h3 == 0.0 && h4 == 1.0 && h6 == 0.0 && h7 == 0.0 && h8 == 1.0 && fabs(h5) < 0.49 &&
          fabs(h2) < 0x1p20))
        return false;
    const double g = h2 + 0.5, f = floor(g), r = g - f;
    if (!(r == 0.0 || fmin(r, 1.0 - r) > 0x1p-30)) return false;
    D = (int)f;
    return true;
}

// Stages one (neighbour, label) entry of an FP64-precision unit for a tile whose pixels lie in the box
// x0 + [-rx, rx] x y0 + [-ry, ry]. In the local frame x' = x - x0, y' = y - y0 the projection is
//   u = U0 + X'/W, v = V0 + Y'/W,  X' = X - U0 W = a0 x' + a1 y' + a2,  Y' = Y - V0 W = b0 x' + b1 y' + b2,
//   W = c0 x' + c1 y' + c2,
// with (U0, V0) the integer position nearest the box centre's projection. The coefficients are formed in
// FP64 (that is where the cancellation of X - U0 W happens) and rounded to FP32 into h[]; u' = X'/W then
// stays within a few pixels, so the FP32 evaluation is accurate to about 2^-24 of the tile's extent
// instead of 2^-24 of the image coordinates. The bound delta covers, at every pixel of the box:
//   the FP32 rounding of the coefficients and of the two fused multiply-adds (3 * 2^-24 of the magnitude
//   M = |a0| rx + |a1| ry + |a2|), the FP64 rounding of the coefficients (2^-50 of the global magnitudes),
//   the quotient of those errors ((e_X + |u'| e_W) / W), the rounded reciprocal and product (2^-23 |u'|; the
//   remainder from the nearest integer is exact), and the FP64 projection's own error against exact arithmetic
//   (3 * 2^-53 (A_X + |u| A_W) / W + 2 * 2^-53 (|u| + 1)),
// and a sixteenth more. The bounds are formed in FP32: the few roundings of one (at most 2^-18 of it) lie within that
// sixteenth, or are added where a comparison stands without it (up); over random convergent tiles the largest error met
// is 0.51 of the bound. A_X is taken from the local coefficients
// (|H0| <= |a0| + |U0 c0|, |H2| <= |X0| + |H0 x0| + |H1 y0|), W0 from its FP32 rounding; magnitudes that FP32
// cannot hold end in kSlow. FP64 does at most 2 multiply-adds a cycle and SM here, and the bounds were most of its
// work: 975x545, 7 views, 100 labels 2.14 -> 1.98 ms, and 1.90 with the margin above in place of a doubling (near
// evaluations 0.0225 -> 0.011 % of all). Where u' computed in FP32 lies farther than delta from every half-integer, the integer nearest to
// it, plus U0, is the FP64 projection's column floor(u + 0.5) (both see the same side of the same
// half-integer); otherwise the evaluation is redone in FP64. Returns kGeneral (that test applies), kRect (the
// same, rectified: below), kOut (the FP64 projection puts no pixel of the box in view: behind the camera, or wholly
// beyond one image edge by more than the bound) or kSlow (no bound: W may come near zero in the box, or delta is large; every evaluation in FP64).
__device__ uint32_t stage_precise(const double* __restrict__ hg, int x0, int y0, int rx, int ry, int wv, int hv,
                                  float* h, PEntry& P) {
    double H[9];
#pragma unroll
    for (int f = 0; f < 9; ++f) H[f] = __ldg(&hg[f]);
    const double dx0 = (double)x0, dy0 = (double)y0;
    const double X0 = fma(H[0], dx0, fma(H[1], dy0, H[2]));
    const double Y0 = fma(H[3], dx0, fma(H[4], dy0, H[5]));
    const double W0 = fma(H[6], dx0, fma(H[7], dy0, H[8]));
    const float X0f = __double2float_rn(X0), Y0f = __double2float_rn(Y0);
    h[6] = __double2float_rn(H[6]);
    h[7] = __double2float_rn(H[7]);
    h[8] = __double2float_rn(W0);
    const float up = 1.0f + 0x1p-18f;  // above the roundings of any one bound below
    const float frx = (float)rx, fry = (float)ry, ax = fabsf((float)x0) + frx, ay = fabsf((float)y0) + fry;
    const float c0 = fabsf(h[6]), c1 = fabsf(h[7]), c2 = fabsf(h[8]);
    const float AW = up * (2.0f * (c0 * ax + c1 * ay) + c2) + 0x1p-120f;
    const float Rc = c0 * frx + c1 * fry;
    const float gW = up * Rc + 0x1p-48f * AW + 0x1.1p-24f * c2 + 0x1p-120f;
    if (h[8] + gW < 0.0f) return kOut;             // W < 0 at every pixel of the box
    const float Wlo = (h[8] - gW) * (2.0f - up);   // the exact W is at least this at every pixel of the box
    if (!(Wlo > 0x1p-60f && Wlo < 0x1p100f)) return kSlow;
    const float U0 = rintf(fminf(fmaxf(__fdiv_rn(X0f, h[8]), -0x1p24f), 0x1p24f));
    const float V0 = rintf(fminf(fmaxf(__fdiv_rn(Y0f, h[8]), -0x1p24f), 0x1p24f));
    const double dU = (double)U0, dV = (double)V0;
    h[0] = __double2float_rn(fma(-dU, H[6], H[0]));
    h[1] = __double2float_rn(fma(-dU, H[7], H[1]));
    h[2] = __double2float_rn(fma(-dU, W0, X0));
    h[3] = __double2float_rn(fma(-dV, H[6], H[3]));
    h[4] = __double2float_rn(fma(-dV, H[7], H[4]));
    h[5] = __double2float_rn(fma(-dV, W0, Y0));
    const float Ma = up * (fabsf(h[0]) * frx + fabsf(h[1]) * fry + fabsf(h[2])) + 0x1p-120f;
    const float Mb = up * (fabsf(h[3]) * frx + fabsf(h[4]) * fry + fabsf(h[5])) + 0x1p-120f;
    const float Mc = up * (Rc + c2) + 0x1p-120f;
    const float aU = fabsf(U0), aV = fabsf(V0);
    const float AX = up * (2.0f * ((fabsf(h[0]) + aU * c0) * ax + (fabsf(h[1]) + aU * c1) * ay) + fabsf(X0f)) + 0x1p-100f;
    const float AY = up * (2.0f * ((fabsf(h[3]) + aV * c0) * ax + (fabsf(h[4]) + aV * c1) * ay) + fabsf(Y0f)) + 0x1p-100f;
    const float eX = 0x1.82p-23f * Ma + 0x1p-50f * (Ma + AX + aU * AW);
    const float eY = 0x1.82p-23f * Mb + 0x1p-50f * (Mb + AY + aV * AW);
    const float eW = 0x1.82p-23f * Mc + 0x1p-50f * (Mc + AW);
    if (!(Wlo > 2.0f * eW)) return kSlow;
    const float rW = up * __frcp_rn(Wlo - eW);  // 1 / a lower bound of the FP32 W and of the FP64 projection's W
    const float Ub = up * (Ma + 2.0f * eX) * rW, Vb = up * (Mb + 2.0f * eY) * rW;
    const float du = 1.0625f * ((eX + Ub * eW + 0x1.8p-52f * (AX + (aU + Ub) * AW)) * rW + 0x1.01p-23f * Ub +
                             0x1.02p-52f * (aU + Ub + 1.0f)) + 0x1p-30f;
    const float dv = 1.0625f * ((eY + Vb * eW + 0x1.8p-52f * (AY + (aV + Vb) * AW)) * rW + 0x1.01p-23f * Vb +
                             0x1.02p-52f * (aV + Vb + 1.0f)) + 0x1p-30f;
    // every pixel of the box has its column (row) beyond one edge by more than the bound
    const float lu = up * (Ub + du), lv = up * (Vb + dv);
    if (U0 < -0.501f - lu || (float)((int)U0 - wv) > lu - 0.499f || V0 < -0.501f - lv ||
        (float)((int)V0 - hv) > lv - 0.499f)
        return kOut;
    if (!(du < 0.25f && dv < 0.25f && Ub < 0x1p21f && Vb < 0x1p21f)) return kSlow;
    P.u0 = (int)U0 - kRoundBits;  // the kernel adds it to the bits of t + kRound
    P.v0 = (int)V0 - kRoundBits;
    // near a tie when |t - nearest integer| >= thr
    P.thr_u = __fsub_rd(0.5f, __fadd_ru(du, 0x1p-22f));
    P.thr_v = __fsub_rd(0.5f, __fadd_ru(dv, 0x1p-22f));
    // Rectified local frame (linear rigs with parallel axes): with a0 = b1 = c2 = 1 and a1 = b0 = c0 = c1 = 0
    // the general evaluation computes exactly t_u = x' + a2 (rounded) and W = r = 1, so the
    // bound above holds for that shorter sequence; and when |b2| + delta_v < 0.5 every pixel's row decision
    // is floor(y' + b2 + 0.5 +- delta_v) = y', i.e. the row is y' + V0 = y + (V0 - y0) with no test.
    if (h[0] == 1.0f && h[1] == 0.0f && h[3] == 0.0f && h[4] == 1.0f && h[6] == 0.0f && h[7] == 0.0f &&
        h[8] == 1.0f && fabsf(h[5]) + dv < 0.49f) {
        P.v0 = (int)V0 - y0;
        return kRect;
    }
    return kGeneral;
}

// First item of chunk k when n items are split into K nearly equal consecutive chunks (32-bit, no overflow).
__device__ __forceinline__ int chunk_begin(int n, int k, int K) {
    const int q = n / K, r = n - q * K;
    return k * q + min(k, r);
}

__device__ __forceinline__ int find_job(const RefJob* __restrict__ jobs, int n_jobs, int item) {
    int lo = 0, hi = n_jobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&jobs[mid].item_base) <= item) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <int FMT, int COMB, bool FAST_RCP, bool PF, int KIND>
__global__ void __launch_bounds__(kThreads, kMinBlocks) cost_kernel(const RefJob* __restrict__ jobs,
                                                                    Plan* __restrict__ plan, int chunk, int chunks) {
    constexpr bool kProj = KIND == kKindProjective;
    constexpr int kTexel = FMT == FMT_U16X4 || FMT == FMT_U16S ? 8 : 4;
    constexpr bool kShifts = KIND == kKindMixed || KIND == kKindPreciseMixed;  // kinds with integer-shift entries
    using Ref = typename TexelOps<FMT>::Ref;
    __shared__ HEntry sH[kHEntries];
    __shared__ const void* sBase[FTV_MAX_NBRS];
    __shared__ int sAcc[kSegAcc * kMaxLB];
    __shared__ int sWoffs[kSegAcc + 1];  // listed-pixel offsets of the tile's first segments
    __shared__ int s_item, s_culled;
    __shared__ PEntry sP[precise_kind(KIND) ? kHEntries : 1];
    // per label the neighbours to visit, grouped by class (kOut entries are left out): the first group is kIn
    // (projective) or kShiftIn, whose texel offsets are listed in sShift instead
    __shared__ uint8_t sOrd[kHEntries];
    __shared__ int sCnt[kMaxLB];  // sizes of the groups: first | second << 8 | third << 16
    __shared__ int sShift[kShifts ? kHEntries : 1];
    __shared__ uint16_t sKey[kThreads / 32][kMaxRuns];  // per warp: its pixels' segments (relative to k0)
    unsigned n_recomputed = 0;  // FP64-precision evaluations computed in double precision by this thread
    uint32_t* const ck = &plan->checked;  // out-of-view gathers of checked builds

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // this launch's items: [chunk_begin(chunk), chunk_begin(chunk + 1)); only thread 0 needs the first (it
    // recomputes it from the plan when it fetches an item, which keeps it out of every thread's registers)
    const int total = chunk_begin(*reinterpret_cast<volatile int*>(&plan->total_items), chunk + 1, chunks);
    const int n_jobs = *reinterpret_cast<volatile int*>(&plan->n_jobs);
    for (int i = tid; i < kSegAcc * kMaxLB; i += kThreads) sAcc[i] = 0;

    if (tid == 0) s_culled = 0;
    for (;;) {
        __syncthreads();
        if (tid == 0)
            s_item = chunk_begin(*reinterpret_cast<volatile int*>(&plan->total_items), chunk, chunks) +
                     atomicAdd(&plan->counter[chunk], 1);
        __syncthreads();
        const int item = s_item;
        if (item >= total) break;

        const RefJob* Jp = &jobs[find_job(jobs, n_jobs, item)];
        const int q = item - Jp->item_base;
        const int nLB = Jp->nLB, L = Jp->L, N = Jp->N, W = Jp->W, penalty = Jp->penalty;
        const int tile = q / nLB, lb = q - tile * nLB;
        const int d0 = lb * Jp->LB;
        const int LBa = min(Jp->LB, L - d0);
        const int n_rec = Jp->n_rec;
        const int32_t* __restrict__ list = Jp->list;
        const void* ref_tex = Jp->ref_texels;
        const void* all_tex = Jp->all_texels;
        int32_t* __restrict__ cost = Jp->cost;
        const int w0 = tile * kTile;
        const int w1 = min(w0 + kTile, n_rec);
        // the tile's first and last segment (in list order) and its pixel box
        const int4 T = __ldg(&Jp->tiles[tile]);
        const int k0 = T.x, k1 = T.y, X0 = T.z & 0xffff, X1 = T.z >> 16, Y0 = T.w & 0xffff, Y1 = T.w >> 16;
        const int nk = k1 - k0 + 1;

        // This thread's pixels: a warp owns kWarpPix consecutive records, 32 per slot. An empty slot (past the
        // unit's last pixel, its result discarded) takes the box's first corner, so that every slot lies in the
        // box and the unchecked gathers of kIn and kShiftIn entries stay inside the view for it too.
        float px[kPPT], py[kPPT];
        Ref ref[kPPT];
        int run[kPPT], iy[kPPT];  // run[j]: first the pixel's segment, then its index among the warp's runs
        int rowx[kPPT];  // y * W + x (integer-shift entries)
#pragma unroll
        for (int j = 0; j < kPPT; ++j) {
            const int w = w0 + warp * kWarpPix + j * 32 + lane;
            int2 rec = make_int2(X0 | (Y0 << 16), kSentinel);
            if (w < w1) rec = __ldg(&Jp->recs[w]);
            const int x = rec.x & 0xffff, y = (unsigned)rec.x >> 16;
            px[j] = (float)x;
            py[j] = (float)y;
            iy[j] = y;
            rowx[j] = y * W + x;
            ref[j] = TexelOps<FMT>::load_ref(ref_tex, (int64_t)y * W + x);
            run[j] = rec.y;
        }

        // stage homographies and neighbour geometry: entry (n, l) for n < N, l < LBa
        const float* __restrict__ Hg = Jp->H;
        const NbrView* __restrict__ nbrs = Jp->nbrs;
        const int nh = N * LBa;
        for (int e = tid; e < (precise_kind(KIND) ? 0 : nh); e += kThreads) {
            const int n = e / LBa, l = e - n * LBa;
            const float* src = &Hg[((int64_t)n * L + d0 + l) * 9];
            HEntry& E = sH[e];
#pragma unroll
            for (int f = 0; f < 9; ++f) E.h[f] = __ldg(&src[f]);
            uint32_t mode = kGeneral;
            if (E.h[6] == 0.0f && E.h[7] == 0.0f) {
                const float r = __frcp_rn(E.h[8]);
                mode = !finite_positive(r) ? kOut : (r == 1.0f ? kUnit : kAffine);
                if (mode == kUnit && E.h[0] == 1.0f && E.h[1] == 0.0f && E.h[3] == 0.0f && E.h[4] == 1.0f &&
                    fabsf(E.h[5]) < 0.25f)
                    mode = kRect;
                E.h[6] = r;
                E.h[8] = E.h[2];  // Wz is not needed any more; a rectified entry then reads one float4
                if (mode == kRect && nbrs[n].off >= 0 && nbrs[n].pitch == W && nbrs[n].h >= Jp->Href) {
                    const double h2 = (double)E.h[2];
                    const double D = floor(h2 + 0.5), g = h2 + 0.5 - D;
                    if (fabs(h2) < 0x1p20 && fmin(g, 1.0 - g) > 0x1p-23 * (32768.0 + fabs(h2))) {
                        mode = kShift;
                        E.h[0] = __int_as_float(nbrs[n].off);
                        E.h[6] = (float)(-D);
                        E.h[7] = (float)((double)nbrs[n].w - D);
                        E.h[8] = __int_as_float((int)D);
                    }
                }
            }
            // The tile's pixel box decides each entry's class: an entry whose neighbour view no pixel of the tile
            // can reach takes the penalty for every pixel, without sampling: it becomes an all-out entry, which the
            // pixel loop does not visit; entries whose samples all land in view (kIn, kShiftIn) or in front of the
            // camera (kFront) skip the tests they cannot fail. box_class is run for the projective-only
            // instantiation alone: on a rectified rig the column bounds of an integer-shift entry tell the same
            // in two comparisons. FP64-precision units stage their entries below (stage_precise).
            if (kProj && mode == kGeneral) {
                mode = box_class(E.h, (float)X0, (float)X1, (float)Y0, (float)Y1, (float)nbrs[n].w, (float)nbrs[n].h);
                if (mode == kOut) atomicAdd(&s_culled, 1);
            } else if (kShifts && mode == kShift) {
                if ((float)X0 >= E.h[6] && (float)X1 < E.h[7]) mode = kShiftIn;
                else if ((float)X1 < E.h[6] || (float)X0 >= E.h[7]) mode = kOut;
            }
            E.w = (uint32_t)nbrs[n].w;
            E.h_ = (uint32_t)nbrs[n].h;
            E.pm = (uint32_t)nbrs[n].pitch | (mode << 28);
        }
        int fx0 = 0, fy0 = 0;  // local-frame origin (FP64-precision units)
        if constexpr (precise_kind(KIND)) {
            fx0 = (X0 + X1) >> 1;
            fy0 = (Y0 + Y1) >> 1;
            const int rx = max(fx0 - X0, X1 - fx0), ry = max(fy0 - Y0, Y1 - fy0);
            for (int e = tid; e < nh; e += kThreads) {
                const int n = e / LBa, l = e - n * LBa;
                HEntry& E = sH[e];
                const int wv = nbrs[n].w, hv = nbrs[n].h;
                const double* hg = &Jp->H64[((int64_t)n * L + d0 + l) * 9];
                int D = 0;
                uint32_t mode;
                if (kShifts && nbrs[n].off >= 0 && nbrs[n].pitch == W && hv >= Jp->Href && shift_fp64(hg, D)) {
                    // every pixel's FP64 column is x + D and its row y: bounds on the local x' = x - fx0
                    mode = kShift;
                    if (X0 >= -D && X1 < wv - D) mode = kShiftIn;
                    else if (X1 < -D || X0 >= wv - D) mode = kOut;
                    E.h[0] = __int_as_float(nbrs[n].off);
                    E.h[6] = (float)(-D - fx0);
                    E.h[7] = (float)(wv - D - fx0);
                    E.h[8] = __int_as_float(D);
                } else {
                    mode = stage_precise(hg, fx0, fy0, rx, ry, wv, hv, E.h, sP[e]);
                    if (mode == kOut) atomicAdd(&s_culled, 1);
                }
                E.w = (uint32_t)wv;
                E.h_ = (uint32_t)hv;
                E.pm = (uint32_t)nbrs[n].pitch | (mode << 28);
            }
            // into the local frame, so that a slot's local coordinates, row index and FP64 projection arguments
            // name the same reference pixel
#pragma unroll
            for (int j = 0; j < kPPT; ++j) {
                px[j] = (float)((int)px[j] - fx0);
                py[j] = (float)(iy[j] - fy0);
            }
        }
        for (int i = tid; i < N; i += kThreads) sBase[i] = nbrs[i].texels;
        if (tid <= min(nk, kSegAcc)) sWoffs[tid] = Jp->woffs[k0 + tid];
        // The float row: kept in registers except in the mixed kernel, which needs registers for rowx and,
        // on the rigs it serves, rarely takes the general or affine paths that read it (exact conversion).
        auto row_f = [&](int j) { return KIND == kKindMixed ? (float)iy[j] : py[j]; };
        // The runs of equal segments among the warp's pixels (records are in list order). Ballots, not a loop until
        // every pixel is numbered: after a loop whose length depends on the data the compiler keeps the label loop's
        // counters and addresses in vector instead of uniform registers (3840x2160 15-view rig: 473 against 437 ms).
        int n_runs = 0;
        {
            int last = -1;
#pragma unroll
            for (int j = 0; j < kPPT; ++j) {
                const int k = run[j], left = __shfl_up_sync(kFull, k, 1);
                const bool first = k != kSentinel && k != (lane == 0 ? last : left);
                const unsigned starts = __ballot_sync(kFull, first);
                const int r = n_runs + __popc(starts & (kFull >> (31 - lane))) - 1;
                if (first && r < kMaxRuns) sKey[warp][r] = (uint16_t)(k - k0);
                run[j] = k != kSentinel ? r : -1;
                n_runs += __popc(starts);
                last = __shfl_sync(kFull, k, 31);
            }
            if (n_runs > kMaxRuns || nk > 0xffff) n_runs = -1;
        }
        __syncthreads();
        if (tid == 0) {
            if (s_culled > 0) atomicAdd(&plan->culled, (unsigned long long)s_culled * (unsigned)(w1 - w0));
            s_culled = 0;
        }
        // per label, the neighbours to visit grouped by class: one warp per label, N <= 32. The projective kind's
        // groups are kIn, kFront and kGeneral; the others' are kShiftIn and everything else in or partly in view.
        for (int l = warp; l < LBa; l += kThreads / 32) {
            const HEntry* E = &sH[lane * LBa + l];
            const uint32_t mode = lane < N ? (E->pm >> 28) : (uint32_t)kOut;
            const bool g1 = kProj ? mode == kIn : (kShifts && mode == kShiftIn);
            const bool g2 = kProj ? mode == kFront : (!g1 && mode != kOut);
            const bool g3 = kProj && mode == kGeneral;
            const unsigned m1 = __ballot_sync(kFull, g1), m2 = __ballot_sync(kFull, g2), m3 = __ballot_sync(kFull, g3);
            const unsigned lt = (1u << lane) - 1u;
            const int c1 = __popc(m1), c2 = __popc(m2);
            int pos = -1;
            if (g1) pos = __popc(m1 & lt);
            else if (g2) pos = c1 + __popc(m2 & lt);
            else if (g3) pos = c1 + c2 + __popc(m3 & lt);
            if (pos >= 0) sOrd[l * N + pos] = (uint8_t)lane;
            if (kShifts && g1) sShift[l * N + pos] = __float_as_int(E->h[0]) + __float_as_int(E->h[8]);
            if (lane == 0) sCnt[l] = c1 | (c2 << 8) | (__popc(m3) << 16);
        }
        __syncthreads();

        for (int l = 0; l < LBa; ++l) {
            int m[kPPT];
#pragma unroll
            for (int j = 0; j < kPPT; ++j)
                m[j] = (COMB == FTV_COMBINE_MIN && N > 0) ? (PF ? penalty : INT_MAX) : 0;
            const int cnt = sCnt[l];
            const int c1 = cnt & 0xff, c2 = c1 + ((cnt >> 8) & 0xff), c3 = c2 + (cnt >> 16);
            const uint8_t* ord = &sOrd[l * N];
            if constexpr (kProj) {
#pragma unroll 2  // two entries in flight: measured 2 % faster on the 4K rig
                for (int k = 0; k < c1; ++k) {  // every pixel's sample is in view
                    const int n = ord[k];
                    const float4* e4 = reinterpret_cast<const float4*>(&sH[n * LBa + l]);
                    const float4 ha = e4[0], hb = e4[1], hc = e4[2];
                    const void* tex = sBase[n];
                    const int pitch = (int)(__float_as_uint(hc.w) & kPitchMask);
                    const unsigned lim = (unsigned)pitch * __float_as_uint(hc.z);  // texels of the view
#pragma unroll
                    for (int j = 0; j < kPPT; ++j) {
                        const float X = __fmaf_rn(ha.x, px[j], __fmaf_rn(ha.y, py[j], ha.z));
                        const float Yh = __fmaf_rn(ha.w, px[j], __fmaf_rn(hb.x, py[j], hb.y));
                        const float Wz = __fmaf_rn(hb.z, px[j], __fmaf_rn(hb.w, py[j], hc.x));
                        const float r = contract_rcp_normal<FAST_RCP>(Wz);
                        const int ui = __float2int_rd(__fadd_rn(__fmul_rn(X, r), 0.5f));
                        const int vi = __float2int_rd(__fadd_rn(__fmul_rn(Yh, r), 0.5f));
                        accumulate_in<FMT, COMB>(m[j], tex, vi * pitch + ui, ref[j], penalty, lim, ck);
                    }
                }
                for (int k = c1; k < c2; ++k) {  // Wz proven positive and normal: range tests only
                    const int n = ord[k];
                    const float4* e4 = reinterpret_cast<const float4*>(&sH[n * LBa + l]);
                    const float4 ha = e4[0], hb = e4[1], hc = e4[2];
                    const void* tex = sBase[n];
                    const int pitch = (int)(__float_as_uint(hc.w) & kPitchMask);
                    const unsigned lim = (unsigned)pitch * __float_as_uint(hc.z);  // texels of the view
#pragma unroll
                    for (int j = 0; j < kPPT; ++j) {
                        const float X = __fmaf_rn(ha.x, px[j], __fmaf_rn(ha.y, py[j], ha.z));
                        const float Yh = __fmaf_rn(ha.w, px[j], __fmaf_rn(hb.x, py[j], hb.y));
                        const float Wz = __fmaf_rn(hb.z, px[j], __fmaf_rn(hb.w, py[j], hc.x));
                        const float r = contract_rcp_normal<FAST_RCP>(Wz);
                        const int ui = __float2int_rd(__fadd_rn(__fmul_rn(X, r), 0.5f));
                        const int vi = __float2int_rd(__fadd_rn(__fmul_rn(Yh, r), 0.5f));
                        const bool ok = ((unsigned)ui < __float_as_uint(hc.y)) & ((unsigned)vi < __float_as_uint(hc.z));
                        accumulate<FMT, COMB, PF>(m[j], ok, tex, vi * pitch + ui, ref[j], penalty, lim, ck);
                    }
                }
                for (int k = c2; k < c3; ++k) {  // the contract's sequence as written
                    const int n = ord[k];
                    const float4* e4 = reinterpret_cast<const float4*>(&sH[n * LBa + l]);
                    const float4 ha = e4[0], hb = e4[1], hc = e4[2];
                    const void* tex = sBase[n];
                    const int pitch = (int)(__float_as_uint(hc.w) & kPitchMask);
                    const unsigned lim = (unsigned)pitch * __float_as_uint(hc.z);  // texels of the view
#pragma unroll
                    for (int j = 0; j < kPPT; ++j) {
                        int idx;
                        const bool ok = pos_general<FAST_RCP>(ha, hb, hc, pitch, px[j], py[j], idx);
                        accumulate<FMT, COMB, PF>(m[j], ok, tex, idx, ref[j], penalty, lim, ck);
                    }
                }
            }
            if constexpr (kShifts) {  // every sample of the tile in view, at the pixel's own index plus one offset
                const int* sh = &sShift[l * N];
#pragma unroll 2
                for (int k = 0; k < c1; ++k) {
                    const int delta = sh[k];
#ifdef FTV_CHECKED
                    const int n = ord[k];
                    const unsigned lim = (unsigned)W * sH[n * LBa + l].h_;
                    const int own = delta - nbrs[n].off;
#pragma unroll
                    for (int j = 0; j < kPPT; ++j)
                        accumulate_in<FMT, COMB>(m[j], sBase[n], rowx[j] + own, ref[j], penalty, lim, ck);
#else
                    // the offset goes into the base, so that a gather's address is one multiply-add of the pixel's
                    // own index (1920x1080 8-view rig: 18.16 -> 17.88 ms)
                    const void* at = static_cast<const char*>(all_tex) + (int64_t)delta * kTexel;
#pragma unroll
                    for (int j = 0; j < kPPT; ++j)
                        accumulate_in<FMT, COMB>(m[j], at, rowx[j], ref[j], penalty, 0u, ck);
#endif
                }
            }
            for (int k = c1; k < (kProj ? 0 : c2); ++k) {
                const int n = ord[k];
                const float4* e4 = reinterpret_cast<const float4*>(&sH[n * LBa + l]);
                const float4 hc = e4[2];
                const void* tex = sBase[n];
                const uint32_t pm = __float_as_uint(hc.w);
                const uint32_t mode = pm >> 28;
                const int pitch = (int)(pm & kPitchMask);
                const unsigned lim = (unsigned)pitch * __float_as_uint(hc.z);  // texels of the view
                if (precise_kind(KIND)) {
                    const double* h64 = &Jp->H64[((int64_t)n * L + d0 + l) * 9];
                    const int wv = __float_as_int(hc.y), hv = __float_as_int(hc.z);
                    if (mode == kSlow) {
#pragma unroll
                        for (int j = 0; j < kPPT; ++j) {
                            const long long q = project_fp64_packed(h64, (int)px[j] + fx0, iy[j], wv, hv);
                            n_recomputed += run[j] >= 0;
                            const int idx = (int)(q >> 32) * pitch + (int)(unsigned)q;
                            accumulate<FMT, COMB, PF>(m[j], q >= 0, tex, idx, ref[j], penalty, lim, ck);
                        }
                    } else if (kShifts && mode == kShift) {
                        const float4 hb = e4[1];  // (h4, h5, lower and upper bound of x')
                        const int D = __float_as_int(hc.x);
#pragma unroll
                        for (int j = 0; j < kPPT; ++j) {
                            const bool ok = (px[j] >= hb.z) & (px[j] < hb.w);
                            accumulate<FMT, COMB, PF>(m[j], ok, tex, rowx[j] + D, ref[j], penalty, lim, ck);
                        }
                    } else {
                        // The column and row nearest u' = X'/W (as FP32) by the rounding of u' + kRound, whose low
                        // bits hold the integer; t - nearest is exact, and when it lies within the staged threshold
                        // of 0 the FP64 projection rounds the same way. The others (rare) are redone in FP64 below.
                        const float4 pe = reinterpret_cast<const float4*>(sP)[n * LBa + l];
                        const int u0 = __float_as_int(pe.x), v0 = __float_as_int(pe.y);
                        unsigned redo = 0;
                        if (kShifts && mode == kRect) {
                            const float a2 = e4[0].z;
#pragma unroll
                            for (int j = 0; j < kPPT; ++j) {
                                const float tu = __fadd_rn(px[j], a2), ru = __fadd_rn(tu, kRound);
                                const int ui = __float_as_int(ru) + u0, vi = iy[j] + v0;
                                if (fabsf(__fsub_rn(tu, __fsub_rn(ru, kRound))) >= pe.z) {
                                    redo |= 1u << j;
                                } else {
                                    const bool ok = ((unsigned)ui < (unsigned)wv) & ((unsigned)vi < (unsigned)hv);
                                    accumulate<FMT, COMB, PF>(m[j], ok, tex, vi * pitch + ui, ref[j], penalty, lim, ck);
                                }
                            }
                        } else {
                            const float4 ha = e4[0], hb = e4[1];
#pragma unroll
                            for (int j = 0; j < kPPT; ++j) {
                                const float X = __fmaf_rn(ha.x, px[j], __fmaf_rn(ha.y, py[j], ha.z));
                                const float Yh = __fmaf_rn(ha.w, px[j], __fmaf_rn(hb.x, py[j], hb.y));
                                const float Wz = __fmaf_rn(hb.z, px[j], __fmaf_rn(hb.w, py[j], hc.x));
                                const float r = contract_rcp_normal<FAST_RCP>(Wz);
                                const float tu = __fmul_rn(X, r), tv = __fmul_rn(Yh, r);
                                const float ru = __fadd_rn(tu, kRound), rv = __fadd_rn(tv, kRound);
                                const int ui = __float_as_int(ru) + u0, vi = __float_as_int(rv) + v0;
                                if (fabsf(__fsub_rn(tu, __fsub_rn(ru, kRound))) >= pe.z ||
                                    fabsf(__fsub_rn(tv, __fsub_rn(rv, kRound))) >= pe.w) {
                                    redo |= 1u << j;
                                } else {
                                    const bool ok = ((unsigned)ui < (unsigned)wv) & ((unsigned)vi < (unsigned)hv);
                                    accumulate<FMT, COMB, PF>(m[j], ok, tex, vi * pitch + ui, ref[j], penalty, lim, ck);
                                }
                            }
                        }
                        if (redo) {
#pragma unroll
                            for (int j = 0; j < kPPT; ++j)
                                if (redo >> j & 1u) {
                                    const long long q = project_fp64_packed(h64, (int)px[j] + fx0, iy[j], wv, hv);
                                    const int idx = (int)(q >> 32) * pitch + (int)(unsigned)q;
                                    accumulate<FMT, COMB, PF>(m[j], q >= 0, tex, idx, ref[j], penalty, lim, ck);
                                    n_recomputed += run[j] >= 0;
                                }
                        }
                    }
                } else if (mode == kShift) {
                    const float4 hb = e4[1];  // (h4, h5, -D, w - D)
                    const int D = __float_as_int(hc.x);
#pragma unroll
                    for (int j = 0; j < kPPT; ++j) {
                        const bool ok = (px[j] >= hb.z) & (px[j] < hb.w);
                        accumulate<FMT, COMB, false>(m[j], ok, tex, rowx[j] + D, ref[j], penalty, lim, ck);
                    }
                } else if (mode == kRect) {
#pragma unroll
                    for (int j = 0; j < kPPT; ++j) {
                        int idx;
                        const bool ok = pos_rect(hc.x, __float_as_uint(hc.y), __float_as_uint(hc.z), pitch, px[j], iy[j],
                                                 idx);
                        accumulate<FMT, COMB, false>(m[j], ok, tex, idx, ref[j], penalty, lim, ck);
                    }
                } else if (mode == kGeneral) {
                    const float4 ha = e4[0], hb = e4[1];
#pragma unroll
                    for (int j = 0; j < kPPT; ++j) {
                        int idx;
                        const bool ok = pos_general<FAST_RCP>(ha, hb, hc, pitch, px[j], row_f(j), idx);
                        accumulate<FMT, COMB, PF>(m[j], ok, tex, idx, ref[j], penalty, lim, ck);
                    }
                } else if (mode == kUnit) {
                    const float4 ha = e4[0], hb = e4[1];
#pragma unroll
                    for (int j = 0; j < kPPT; ++j) {
                        int idx;
                        const bool ok = pos_affine<true>(ha, hb, hc, 1.0f, pitch, px[j], row_f(j), idx);
                        accumulate<FMT, COMB, false>(m[j], ok, tex, idx, ref[j], penalty, lim, ck);
                    }
                } else {  // kAffine
                    const float4 ha = e4[0], hb = e4[1];
#pragma unroll
                    for (int j = 0; j < kPPT; ++j) {
                        int idx;
                        const bool ok = pos_affine<false>(ha, hb, hc, hb.z, pitch, px[j], row_f(j), idx);
                        accumulate<FMT, COMB, false>(m[j], ok, tex, idx, ref[j], penalty, lim, ck);
                    }
                }
            }
            const int seen = kProj ? c3 : c2;
            if (!(COMB == FTV_COMBINE_MIN && PF) && seen < N) {  // entries out of view: the penalty each
#pragma unroll
                for (int j = 0; j < kPPT; ++j)
                    m[j] = (COMB == FTV_COMBINE_MIN) ? min(m[j], penalty) : m[j] + (N - seen) * penalty;
            }
            // Each run's sum over the warp's pixels: a thread adds its own slots first, so that a label costs one
            // warp reduction per run (128 consecutive pixels meet two or three segments) instead of one per slot.
            if (n_runs >= 0) {
                for (int r = 0; r < n_runs; ++r) {
                    int v = 0;
#pragma unroll
                    for (int j = 0; j < kPPT; ++j) v += run[j] == r ? m[j] : 0;
                    const int sum = __reduce_add_sync(kFull, v);
                    if (lane == 0) {
                        const int k = sKey[warp][r];
                        if (k < kSegAcc) atomicAdd(&sAcc[k * kMaxLB + l], sum);
                        else atomicAdd(&cost[(int64_t)(list ? list[k0 + k] : k0 + k) * L + d0 + l], sum);
                    }
                }
            } else {  // segments of one or two pixels, or a tile spanning 2^16 empty ones: each pixel on its own
#pragma unroll
                for (int j = 0; j < kPPT; ++j)
                    if (run[j] >= 0) {
                        const int k = Jp->recs[w0 + warp * kWarpPix + j * 32 + lane].y - k0;
                        if (k < kSegAcc && nk <= 0xffff) atomicAdd(&sAcc[k * kMaxLB + l], m[j]);
                        else atomicAdd(&cost[(int64_t)(list ? list[k0 + k] : k0 + k) * L + d0 + l], m[j]);
                    }
            }
        }
        __syncthreads();

        if (warp == kThreads / 32 - 1) {  // the entries that no pixel visited (the last warp has the fewest row slices)
            int out = 0;
            for (int l = lane; l < LBa; l += 32) {
                const int cnt = sCnt[l];
                out += N - (cnt & 0xff) - ((cnt >> 8) & 0xff) - (cnt >> 16);
            }
            out = __reduce_add_sync(kFull, out);
            if (lane == 0 && out > 0) atomicAdd(&plan->skipped, (unsigned long long)out * (unsigned)(w1 - w0));
        }
        // write the row slices of this tile's first segments
        const int nacc = nk > 0xffff ? 0 : min(nk, kSegAcc);
        for (int i = tid; i < nacc * LBa; i += kThreads) {
            const int loc = i / LBa, l = i - loc * LBa;
            const int k = k0 + loc;
            const int s = list ? list[k] : k;
            const int v = sAcc[loc * kMaxLB + l];
            sAcc[loc * kMaxLB + l] = 0;
            if ((unsigned)s >= (unsigned)Jp->S) continue;  // an invalid list entry owns no pixels
            const int a = sWoffs[loc], b = sWoffs[loc + 1];
            if (a == b) continue;  // no pixels: the row is clear (an empty segment), or another entry's
            int32_t* dst = &cost[(int64_t)s * L + d0 + l];
            if (a >= w0 && b <= w0 + kTile) *dst = v;
            else atomicAdd(dst, v);
        }
    }
    if constexpr (precise_kind(KIND)) {
        const unsigned n = __reduce_add_sync(kFull, n_recomputed);
        if (lane == 0 && n) atomicAdd(&plan->recomputed, (unsigned long long)n);
    }
}

template <int FMT, int COMB, bool FAST>
int blocks_per_sm_for() {
    int n = 0;
    constexpr int kind = FMT == FMT_U16S ? kKindProjective : kKindMixed;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, cost_kernel<FMT, COMB, FAST, COMB == FTV_COMBINE_MIN, kind>,
                                                      kThreads, 0) != cudaSuccess)
        return 1;
    return n > 0 ? n : 1;
}

// Exhaustive comparison with the IEEE reciprocal over every positive float below 2^126: subnormals go
// through rcp_scaled's scaling, normals through rcp_newton directly.
__global__ void reciprocal_check_kernel(unsigned long long* mismatches) {
    const uint32_t lo = 0x00000001u, hi = 0x7e800000u;
    unsigned long long bad = 0;
    for (uint64_t i = lo + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < hi;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const float w = __uint_as_float((uint32_t)i);
        bad += __float_as_uint(rcp_scaled(w)) != __float_as_uint(__frcp_rn(w));
    }
    bad = __reduce_add_sync(0xffffffffu, (unsigned)bad);
    if ((threadIdx.x & 31) == 0 && bad) atomicAdd(mismatches, bad);
}

std::mutex g_rcp_mutex;
int8_t g_rcp_state[64] = {};  // per device: 0 unknown, 1 exact, -1 not exact

}  // namespace

int64_t reciprocal_mismatches() {
    unsigned long long* d = nullptr;
    if (cudaMalloc(&d, sizeof(unsigned long long)) != cudaSuccess) return -1;
    unsigned long long h = 0;
    int n_sm = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaMemset(d, 0, sizeof(h));
    if (e == cudaSuccess) {
        reciprocal_check_kernel<<<std::max(1, n_sm) * 8, 256>>>(d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? (int64_t)h : -1;
}

bool fast_reciprocal_exact() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lock(g_rcp_mutex);
    if (g_rcp_state[dev] == 0) g_rcp_state[dev] = reciprocal_mismatches() == 0 ? 1 : -1;
    return g_rcp_state[dev] == 1;
}

int cost_blocks_per_sm(int fmt, int combine, bool fast) {
#define FTV_OCC(F, C) (fast ? blocks_per_sm_for<F, C, true>() : blocks_per_sm_for<F, C, false>())
    if (fmt == FMT_U8X4) return combine == FTV_COMBINE_MIN ? FTV_OCC(FMT_U8X4, FTV_COMBINE_MIN)
                                                           : FTV_OCC(FMT_U8X4, FTV_COMBINE_SUM);
    if (fmt == FMT_U16S) return combine == FTV_COMBINE_MIN ? FTV_OCC(FMT_U16S, FTV_COMBINE_MIN)
                                                           : FTV_OCC(FMT_U16S, FTV_COMBINE_SUM);
    if (fmt == FMT_P10) return combine == FTV_COMBINE_MIN ? FTV_OCC(FMT_P10, FTV_COMBINE_MIN)
                                                          : FTV_OCC(FMT_P10, FTV_COMBINE_SUM);
    return combine == FTV_COMBINE_MIN ? FTV_OCC(FMT_U16X4, FTV_COMBINE_MIN) : FTV_OCC(FMT_U16X4, FTV_COMBINE_SUM);
#undef FTV_OCC
}

namespace {

// Shared-memory carveout hint: the smallest split that still holds kMinBlocks CTAs of this kernel, so
// that the rest of the SM's L1 caches the neighbour-view gathers. Once per instantiation and process.
template <typename Kernel>
bool prefer_l1(Kernel kernel) {
    cudaFuncAttributes a{};
    int dev = 0, smem_sm = 0;
    if (cudaFuncGetAttributes(&a, kernel) == cudaSuccess && cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) == cudaSuccess &&
        smem_sm > 0) {
        const size_t need = (size_t)kMinBlocks * (a.sharedSizeBytes + 1024);
        const int pct = (int)std::min<size_t>(100, (need * 100 + smem_sm - 1) / smem_sm);
        cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
    }
    cudaGetLastError();  // a hint only
    return true;
}

template <int FMT, int COMB, bool FAST, bool PF, int KIND>
void launch_one(const RefJob* jobs, Plan* p, int ck, int nck, int grid, cudaStream_t s) {
    static const bool hinted = prefer_l1(cost_kernel<FMT, COMB, FAST, PF, KIND>);
    (void)hinted;
    cost_kernel<FMT, COMB, FAST, PF, KIND><<<grid, kThreads, 0, s>>>(jobs, p, ck, nck);
}

// Kinds an instantiation exists for: FMT_U16S units are all projective; FMT_P10 ones have affine entries, or share
// a batch with units that do (cost_format()).
constexpr bool kind_of_format(int fmt, int kind) {
    return fmt == FMT_U16S ? kind == kKindProjective || kind == kKindPrecise
                           : fmt != FMT_P10 || kind == kKindMixed || kind == kKindPreciseMixed;
}

template <int FMT, int COMB, bool FAST, bool PF, int KIND>
cudaError_t launch_if(const RefJob* jobs, Plan* p, int ck, int nck, int grid, cudaStream_t s) {
    if constexpr (kind_of_format(FMT, KIND)) {
        launch_one<FMT, COMB, FAST, PF, KIND>(jobs, p, ck, nck, grid, s);
        return cudaSuccess;
    } else {
        return cudaErrorInvalidValue;
    }
}

template <int FMT, int COMB, bool FAST, bool PF>
cudaError_t launch_kind(const RefJob* jobs, Plan* p, int kind, int ck, int nck, int grid, cudaStream_t s) {
    if (kind == kKindPrecise) return launch_if<FMT, COMB, FAST, PF, kKindPrecise>(jobs, p, ck, nck, grid, s);
    if (kind == kKindPreciseMixed) return launch_if<FMT, COMB, FAST, PF, kKindPreciseMixed>(jobs, p, ck, nck, grid, s);
    if (kind == kKindProjective) return launch_if<FMT, COMB, FAST, PF, kKindProjective>(jobs, p, ck, nck, grid, s);
    return launch_if<FMT, COMB, FAST, PF, kKindMixed>(jobs, p, ck, nck, grid, s);
}

template <int FMT, int COMB>
cudaError_t launch_fast_pf(const RefJob* jobs, Plan* p, bool fast, bool pf, int kind, int ck, int nck, int grid,
                    cudaStream_t s) {
    const bool use_pf = COMB == FTV_COMBINE_MIN && pf;
    if (fast) {
        if (use_pf) return launch_kind<FMT, COMB, true, true>(jobs, p, kind, ck, nck, grid, s);
        return launch_kind<FMT, COMB, true, false>(jobs, p, kind, ck, nck, grid, s);
    }
    if (use_pf) return launch_kind<FMT, COMB, false, true>(jobs, p, kind, ck, nck, grid, s);
    return launch_kind<FMT, COMB, false, false>(jobs, p, kind, ck, nck, grid, s);
}

template <int FMT>
cudaError_t launch_comb(const RefJob* jobs, Plan* p, int combine, bool fast, bool pf, int kind, int ck, int nck, int grid,
                 cudaStream_t s) {
    if (combine == FTV_COMBINE_MIN) return launch_fast_pf<FMT, FTV_COMBINE_MIN>(jobs, p, fast, pf, kind, ck, nck, grid, s);
    return launch_fast_pf<FMT, FTV_COMBINE_SUM>(jobs, p, fast, pf, kind, ck, nck, grid, s);
}

}  // namespace

cudaError_t launch_cost(const RefJob* jobs, const Plan* plan, int fmt, int combine, bool fast, bool pf, int kind,
                        int chunk, int chunks, int grid, cudaStream_t s) {
    if (chunks < 1 || chunks > kMaxChunks || chunk < 0 || chunk >= chunks) return cudaErrorInvalidValue;
    Plan* p = const_cast<Plan*>(plan);
    cudaError_t e;
    if (fmt == FMT_U8X4) e = launch_comb<FMT_U8X4>(jobs, p, combine, fast, pf, kind, chunk, chunks, grid, s);
    else if (fmt == FMT_U16S) e = launch_comb<FMT_U16S>(jobs, p, combine, fast, pf, kind, chunk, chunks, grid, s);
    else if (fmt == FMT_P10) e = launch_comb<FMT_P10>(jobs, p, combine, fast, pf, kind, chunk, chunks, grid, s);
    else e = launch_comb<FMT_U16X4>(jobs, p, combine, fast, pf, kind, chunk, chunks, grid, s);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace ftv
