// Device-side building blocks shared by the UPSLAM kernels (sm_103a).
//
// The FP32 functions here implement the binning rule stated in upslam.h with
// explicit round-to-nearest intrinsics, so no multiply-add is ever contracted
// into an FMA: the pixel a point falls in, and therefore every z-buffer winner
// and every projective correspondence, is a bit-exact function of the inputs.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <float.h>
#include <math.h>
#include <stdint.h>

#include <atomic>

#include "../../include/upslam.h"

namespace upslam {

constexpr float kPiF = 3.14159265358979323846f;
constexpr float kHalfPiF = 1.57079632679489661923f;
constexpr unsigned long long kEmptyKey = 0xffffffffffffffffull;
constexpr int kNumSums = 29;  // 21 (J^T J) + 6 (J^T r) + sse + inliers

// ----------------------------------------------------------------------------- FP32 decisions

// atan2 reduced by octant symmetry to atan(t), t in [0, 1], with the odd
// polynomial of Abramowitz & Stegun 4.4.49 (|error| <= 2e-8 before rounding).
__device__ __forceinline__ float atan2p(float y, float x) {
    const float ax = fabsf(x), ay = fabsf(y);
    const float mx = ax > ay ? ax : ay;
    const float mn = ax > ay ? ay : ax;
    if (mx == 0.0f) return 0.0f;
    const float t = __fdiv_rn(mn, mx);
    const float s = __fmul_rn(t, t);
    float p = 0.0028662257f;
    p = __fadd_rn(__fmul_rn(p, s), -0.0161657367f);
    p = __fadd_rn(__fmul_rn(p, s), 0.0429096138f);
    p = __fadd_rn(__fmul_rn(p, s), -0.0752896400f);
    p = __fadd_rn(__fmul_rn(p, s), 0.1065626393f);
    p = __fadd_rn(__fmul_rn(p, s), -0.1420889944f);
    p = __fadd_rn(__fmul_rn(p, s), 0.1999355085f);
    p = __fadd_rn(__fmul_rn(p, s), -0.3333314528f);
    p = __fadd_rn(__fmul_rn(p, s), 1.0f);
    float a = __fmul_rn(t, p);
    if (ay > ax) a = __fsub_rn(kHalfPiF, a);
    if (x < 0.0f) a = __fsub_rn(kPiF, a);
    if (y < 0.0f) a = -a;
    return a;
}

// Pixel (row, col) and range of an FP32 point; false when outside the panorama.
__device__ __forceinline__ bool bin_point(float x, float y, float z, const upslam_pano &pp, int &row, int &col,
                                          float &r) {
    const float xy2 = __fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y));
    r = __fsqrt_rn(__fadd_rn(xy2, __fmul_rn(z, z)));
    if (!(r >= pp.r_min && r <= pp.r_max)) return false;
    const float rho = __fsqrt_rn(xy2);
    const float az = atan2p(y, x);
    const float el = atan2p(z, rho);
    const float fc = __fmul_rn(__fsub_rn(kPiF, az), pp.s_az);
    const float fr = __fmul_rn(__fsub_rn(pp.el_top, el), pp.s_el);
    if (!(fr >= 0.0f) || !(fr < (float)pp.rows)) return false;
    row = (int)floorf(fr);
    col = (int)floorf(fc);
    if (row >= pp.rows) return false;
    if (col >= pp.cols) col -= pp.cols;
    if (col < 0) col += pp.cols;
    return true;
}

// A panorama's binning rule with what the fast form below needs, made on the host (make_bin_rule).
struct BinRule {
    upslam_pano pp;
    float r2_min, r2_max;  // sqrt_rn(r2) lies in [r_min, r_max] exactly when r2 lies in [r2_min, r2_max]
    float el0;             // el_top s_el - 1/2, in pixels
    float az[5];           // k pi/2 s_az - 1/2, k = 0..4
    float lim_r, lim_c;    // 1/2 minus the guard, row and column; negative: the fast form is off
};

__device__ __forceinline__ float rcp_approx(float x) {  // relative error below 2^-23
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_approx(float x) {  // relative error below 2^-22.9
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Two FP32 values operated on by one instruction, each rounded as the scalar operation rounds it.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 twice(float v) { return pack2(v, v); }

// The polynomial of atan2p, fused: P(s) with atan(t) = t P(t^2), |t| <= 1.
__device__ __forceinline__ f32x2 atan_poly2(f32x2 s) {
    f32x2 p = fma2(twice(0.0028662257f), s, twice(-0.0161657367f));
    p = fma2(p, s, twice(0.0429096138f));
    p = fma2(p, s, twice(-0.0752896400f));
    p = fma2(p, s, twice(0.1065626393f));
    p = fma2(p, s, twice(-0.1420889944f));
    p = fma2(p, s, twice(0.1999355085f));
    p = fma2(p, s, twice(-0.3333314528f));
    return fma2(p, s, twice(1.0f));
}

// The pixel of an FP32 point, the same as bin_point's bit for bit, usually without its roundings: the two angles
// are formed with approximate reciprocals and fused multiply-adds, in pixels, and the point's cell is the rule's
// whenever both coordinates keep a guard away from a cell's edge, the guard being more than the two forms can
// differ by (make_bin_rule derives it; about 3e-4 of a pixel at 1024 columns, so fewer than one point in a
// thousand is binned again by the rule itself).  The range test needs no root: it compares the rounded squared
// range with the squares' exact limits.  A point more than 45 degrees up or down takes its row from the inverse ratio
// in bin_rest_cell, and whatever makes a NaN here (a point on the axis) goes to the rule.  The rule spends two
// divisions, two square roots and thirty-two unfused polynomial operations, about 200 instructions a point; this form
// about 70, both polynomials in one packed evaluation.  It serves the kernels that bin many samples a thread (the registration's steps, the batched form,
// the grid search).  A kernel that bins once or twice a thread (projection, averaging, hole fill, consistency)
// keeps the rule: it waits for its slowest warp, and some warp always has a point near an edge and would do both
// (a keyframe update measured 11.0 against 10.0 us, a consistency check 22.7 against 20.7).  Two points to an
// instruction throughout (packed transforms and angles) was no faster in any of the three: 89.5 against 85.0 us in
// the grid search, and the assembler contracts packed products and sums, which the rule forbids.
//
// bin_fast: cell = row * cols + col, or -1 outside the panorama; false when bin_rest_cell has to decide, for a point
// within the range limits.  No branch, so that a caller's other work fills its dependent chain.
__device__ __forceinline__ bool bin_fast(float x, float y, float z, const BinRule &b, int &cell) {
    const float xy2 = __fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y));
    const float z2 = __fmul_rn(z, z);
    const float r2 = __fadd_rn(xy2, z2);
    const bool in_range = (r2 >= b.r2_min) & (r2 <= b.r2_max);
    const float te = z * rsqrt_approx(xy2);
    const bool swap = fabsf(y) > fabsf(x), back = y < 0.0f;
    const float ta = (swap ? -x : y) * rcp_approx(swap ? y : x);
    const float b_swap = back ? b.az[3] : b.az[1], b_neg = back ? b.az[4] : b.az[0];
    float pr, pc;
    unpack2(atan_poly2(pack2(te * te, ta * ta)), pr, pc);
    const float fr = fmaf(te * -b.pp.s_el, pr, b.el0);
    const float fc = fmaf(ta * -b.pp.s_az, pc, swap ? b_swap : (x < 0.0f ? b_neg : b.az[2]));
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
    const float mr = __fadd_rn(fr, kMagic), mc = __fadd_rn(fc, kMagic);
    const float dr = __fsub_rn(fr, __fsub_rn(mr, kMagic)), dc = __fsub_rn(fc, __fsub_rn(mc, kMagic));
    const int row = __float_as_int(mr) - __float_as_int(kMagic), col = __float_as_int(mc) - __float_as_int(kMagic);
    const bool in = in_range & ((unsigned)row < (unsigned)b.pp.rows);
    cell = in ? row * b.pp.cols + col : -1;
    // (NaN distances fail these tests, so they go to the rule)
    const bool row_sure = (z2 <= xy2) & (fabsf(dr) <= b.lim_r);
    const bool col_sure = (fabsf(dc) <= b.lim_c) & ((unsigned)col < (unsigned)b.pp.cols);
    return !in_range | (row_sure & (!in | col_sure));
}

// P(s) of atan_poly2, one value.
__device__ __forceinline__ float atan_poly(float s) {
    float p = fmaf(0.0028662257f, s, -0.0161657367f);
    p = fmaf(p, s, 0.0429096138f);
    p = fmaf(p, s, -0.0752896400f);
    p = fmaf(p, s, 0.1065626393f);
    p = fmaf(p, s, -0.1420889944f);
    p = fmaf(p, s, 0.1999355085f);
    p = fmaf(p, s, -0.3333314528f);
    return fmaf(p, s, 1.0f);
}

// The pixel a coordinate rounds to; false within `guard` of a pixel's edge.
__device__ __forceinline__ bool sure_pixel(float f, float guard, int &i) {
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
    const float m = __fadd_rn(f, kMagic);
    i = __float_as_int(m) - __float_as_int(kMagic);
    return fabsf(__fsub_rn(f, __fsub_rn(m, kMagic))) <= 0.5f - guard;
}

// The guards of a steep point's row and column in radians (make_bin_rule).
__device__ __forceinline__ float bin_steep_row_guard(float el_top) {
    return 1.1f / 16777216.0f * (10.7f + 5.0f * (fabsf(el_top) + 1.58f));
}
constexpr float kSteepColGuard = 1.1f * 37.0f / 16777216.0f;

// What bin_fast leaves: the cell of a point steeper than 45 degrees, el = +-pi/2 - atan(rho / z), with guards of its own,
// and the rule for the rest; row * cols + col, or -1 outside the panorama.  Out of line: the kernels bin at many
// places, and the rule's divisions and roots at each of them made the ICP kernel's instructions a fifth longer.
// With the rule alone here, a panorama that looks up (89 to 46 degrees, every sample steep) paid for both: 305 us for
// 729 candidates of the grid search, where the rule at every point takes 289; now 257 (a batch 6.77 ms, 6.91, 5.81).
// The ordinary points' time hangs on the registers that this call takes from its callers: handed bin_fast's column
// instead of forming it again, 122.0 against 119.8 us for 14 steps on a 64x1024 sweep; with both polynomials in one
// packed evaluation, 1 us more for 8 steps into a 1024x4096 keyframe; in this form within 0.2 us of the rule alone.
static __device__ __noinline__ int bin_rest_cell(float x, float y, float z, upslam_pano pp) {
    const float xy2 = __fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y));
    int row, col;
    if (__fmul_rn(z, z) > xy2) {
        // (a guard of half a pixel or more, as for coordinates too large for the magic sums, leaves no point here)
        const float te = xy2 * rsqrt_approx(xy2) * rcp_approx(z);
        const float fr = fmaf(te * pp.s_el, atan_poly(te * te),
                              fmaf(z > 0.0f ? -kHalfPiF : kHalfPiF, pp.s_el, fmaf(pp.el_top, pp.s_el, -0.5f)));
        if (sure_pixel(fr, bin_steep_row_guard(pp.el_top) * pp.s_el, row)) {
            if ((unsigned)row >= (unsigned)pp.rows) return -1;
            const bool swap = fabsf(y) > fabsf(x);
            const float ta = (swap ? -x : y) * rcp_approx(swap ? y : x);
            const float quarters = swap ? (y < 0.0f ? 3.0f : 1.0f) : (x < 0.0f ? (y < 0.0f ? 4.0f : 0.0f) : 2.0f);
            const float fc = fmaf(ta * -pp.s_az, atan_poly(ta * ta), fmaf(quarters * kHalfPiF, pp.s_az, -0.5f));
            if (sure_pixel(fc, kSteepColGuard * pp.s_az, col) && (unsigned)col < (unsigned)pp.cols)
                return row * pp.cols + col;
        }
    }
    float r;
    return bin_point(x, y, z, pp, row, col, r) ? row * pp.cols + col : -1;
}

// The cell.
__device__ __forceinline__ int bin_pixel(float x, float y, float z, const BinRule &b) {
    int cell;
    if (__builtin_expect(!bin_fast(x, y, z, b, cell), 0)) cell = bin_rest_cell(x, y, z, b.pp);
    return cell;
}

// Pose rounded to FP32, row-major [R | t].
struct PoseF {
    float r[12];
};

__device__ __forceinline__ PoseF pose_to_f32(const double *T) {
    PoseF p;
#pragma unroll
    for (int i = 0; i < 12; ++i) p.r[i] = (float)T[i];
    return p;
}

// The CTA's pose in FP32, converted once: threads 0..11 convert one entry each
// into shared memory and every thread reads the FP32 copy.  (An FP64 -> FP32
// conversion issues on GB300's FP64 pipe; converting per thread would cost
// every warp twelve slow instructions.)  Must be reached by the whole CTA.
__device__ __forceinline__ PoseF cta_pose_f32(const double *T, bool through_l2 = false) {
    __shared__ float ps[12];
    __syncthreads();
    if (threadIdx.x < 12) ps[threadIdx.x] = (float)(through_l2 ? __ldcg(T + threadIdx.x) : T[threadIdx.x]);
    __syncthreads();
    PoseF p;
#pragma unroll
    for (int i = 0; i < 12; ++i) p.r[i] = ps[i];
    return p;
}

// Pose read through L2 only (never a stale L1 line): for poses other CTAs rewrite.
__device__ __forceinline__ PoseF pose_to_f32_cg(const double *T) {
    PoseF p;
#pragma unroll
    for (int i = 0; i < 12; ++i) p.r[i] = (float)__ldcg(T + i);
    return p;
}

// p = R q + t, fixed order ((r0 x + r1 y) + r2 z) + t0, no contraction.
__device__ __forceinline__ float3 xform(const PoseF &T, float qx, float qy, float qz) {
    const float *r = T.r;
    float3 p;
    p.x = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(r[0], qx), __fmul_rn(r[1], qy)), __fmul_rn(r[2], qz)), r[3]);
    p.y = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(r[4], qx), __fmul_rn(r[5], qy)), __fmul_rn(r[6], qz)), r[7]);
    p.z = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(r[8], qx), __fmul_rn(r[9], qy)), __fmul_rn(r[10], qz)), r[11]);
    return p;
}

// q = R^T (s - t), fixed order.
__device__ __forceinline__ float3 xform_inv(const PoseF &T, float sx, float sy, float sz) {
    const float *r = T.r;
    const float dx = __fsub_rn(sx, r[3]), dy = __fsub_rn(sy, r[7]), dz = __fsub_rn(sz, r[11]);
    float3 q;
    q.x = __fadd_rn(__fadd_rn(__fmul_rn(r[0], dx), __fmul_rn(r[4], dy)), __fmul_rn(r[8], dz));
    q.y = __fadd_rn(__fadd_rn(__fmul_rn(r[1], dx), __fmul_rn(r[5], dy)), __fmul_rn(r[9], dz));
    q.z = __fadd_rn(__fadd_rn(__fmul_rn(r[2], dx), __fmul_rn(r[6], dy)), __fmul_rn(r[10], dz));
    return q;
}

// Rotation only (values, FMA allowed).
__device__ __forceinline__ float3 rotate(const PoseF &T, float x, float y, float z) {
    const float *r = T.r;
    return make_float3(r[0] * x + r[1] * y + r[2] * z, r[4] * x + r[5] * y + r[6] * z,
                       r[8] * x + r[9] * y + r[10] * z);
}

// FP32 point of pixel (v, u) at depth d from the direction table: d * (ce*ca, ce*sa, se).
__device__ __forceinline__ float3 pixel_point(const float *dirs, int rows, int v, int u, float d) {
    const float2 e = __ldg(reinterpret_cast<const float2 *>(dirs) + v);
    const float2 a = __ldg(reinterpret_cast<const float2 *>(dirs + 2 * rows) + u);
    return make_float3(__fmul_rn(d, __fmul_rn(e.x, a.x)), __fmul_rn(d, __fmul_rn(e.x, a.y)), __fmul_rn(d, e.y));
}

// ----------------------------------------------------------------------------- storage helpers

__device__ __forceinline__ float4 unpack_nw(uint2 raw) {
    const __half2 a = *reinterpret_cast<const __half2 *>(&raw.x);
    const __half2 b = *reinterpret_cast<const __half2 *>(&raw.y);
    const float2 fa = __half22float2(a), fb = __half22float2(b);
    return make_float4(fa.x, fa.y, fb.x, fb.y);
}

__device__ __forceinline__ float4 load_nw(const void *base, int64_t k, int precision) {
    if (precision == UPSLAM_F32) return __ldg(reinterpret_cast<const float4 *>(base) + k);
    return unpack_nw(__ldg(reinterpret_cast<const uint2 *>(base) + k));
}

// Same load, an ordinary one through L1 (for data that the launch before may still write when this kernel's CTAs are
// placed).
__device__ __forceinline__ float4 load_nw_l1(const void *base, int64_t k, int precision) {
    if (precision == UPSLAM_F32) return reinterpret_cast<const float4 *>(base)[k];
    return unpack_nw(reinterpret_cast<const uint2 *>(base)[k]);
}

// Same load, through L2 only (for data rewritten during the kernel's lifetime by other CTAs).
__device__ __forceinline__ float4 load_nw_cg(const void *base, int64_t k, int precision) {
    if (precision == UPSLAM_F32) return __ldcg(reinterpret_cast<const float4 *>(base) + k);
    const uint2 raw = __ldcg(reinterpret_cast<const uint2 *>(base) + k);
    const __half2 a = *reinterpret_cast<const __half2 *>(&raw.x);
    const __half2 b = *reinterpret_cast<const __half2 *>(&raw.y);
    const float2 fa = __half22float2(a), fb = __half22float2(b);
    return make_float4(fa.x, fa.y, fb.x, fb.y);
}

__device__ __forceinline__ void store_nw(void *base, int64_t k, int precision, float4 v) {
    if (precision == UPSLAM_F32) {
        reinterpret_cast<float4 *>(base)[k] = v;
        return;
    }
    const __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
    uint2 raw;
    raw.x = *reinterpret_cast<const unsigned int *>(&a);
    raw.y = *reinterpret_cast<const unsigned int *>(&b);
    reinterpret_cast<uint2 *>(base)[k] = raw;
}

// ----------------------------------------------------------------------------- reductions

// Warp reduce-scatter: lane L ends with the sum over the warp's lanes of v[L]
// (32 values per lane, 31 shuffles in all; v is overwritten).
__device__ __forceinline__ float warp_reduce_scatter(float v[32]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float send = upper ? v[i] : v[i + o];
            const float keep = upper ? v[i + o] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return v[0];
}

// ----------------------------------------------------------------------------- FP64 solve
//
// GB300 runs FP64 at a small fraction of its FP32 rate, and a dependent FP64
// FMA costs tens of cycles (a division an order of magnitude more), so the
// solve is written for a short dependency chain: fully unrolled (every value
// in a register), no FP64 division or square root on the critical path.

// FP64 helpers that stay off the FP64 pipe.  Comparisons, maxima, sign flips
// and format changes work on the bit patterns with integer instructions: for
// doubles that are not NaN, the signed 64-bit order of the bit patterns of
// non-negative values is their numeric order.
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ bool dfinite(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff; }
__device__ __forceinline__ double dneg(double x) {
    return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ull);
}

// Exact FP32 -> FP64 widening: the exponent is rebiased (+896) and the
// mantissa shifted into place with integer instructions.  Zero, subnormal,
// infinite and NaN inputs take the conversion instruction.
__device__ __forceinline__ double f2d(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned e = (b >> 23) & 0xffu;
    if (e == 0u || e == 0xffu) return (double)f;
    const unsigned m = b & 0x7fffffu;
    return __hiloint2double((int)((b & 0x80000000u) | ((e + 896u) << 20) | (m >> 3)), (int)(m << 29));
}

// 1/d for a positive d.  The FP32 seed is d's exponent and top 23 mantissa bits
// (truncation: relative error below 2^-23), formed and widened back with integer
// instructions; one FP64 Newton step then leaves a relative error below 2^-44,
// far below the FP32 accumulation error of the normal equations.  d outside
// [2^-126, 2^126) takes an FP64 division.
__device__ __forceinline__ double rcp64(double d) {
    const int hi = __double2hiint(d), lo = __double2loint(d);
    const int e = ((hi >> 20) & 0x7ff) - (1023 - 127);
    if (hi < 0 || e < 1 || e > 252) return 1.0 / d;
    const float f = __int_as_float((e << 23) | ((hi & 0xfffff) << 3) | (int)((unsigned)lo >> 29));
    const int rb = __float_as_int(__frcp_rn(f));  // normal: f in [2^-126, 2^126)
    const int m = rb & 0x7fffff;
    const double x = __hiloint2double((((rb >> 23) & 0xff) + (1023 - 127)) << 20 | (m >> 3), m << 29);
    return fma(x, fma(-d, x, 1.0), x);
}

// 1/d for a positive normal d whose reciprocal is normal, as rcp64 without its range: the seed comes from d's
// mantissa, rounded to FP32 (relative error below 2^-22.4 with the approximate reciprocal, 2^-44 after the step),
// and d's exponent is taken off the result.
__device__ __forceinline__ double rcp64_scaled(double d) {
    const int hi = __double2hiint(d), lo = __double2loint(d);
    const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, lo);  // in [1, 2)
    const float f = __int_as_float(0x3f800000 + (((hi & 0xfffff) << 3) | (int)((unsigned)lo >> 29)) +
                                   (int)(((unsigned)lo >> 28) & 1u));
    const int rb = __float_as_int(rcp_approx(f));  // about [1/2, 1]
    const int rm = rb & 0x7fffff;
    const double x = __hiloint2double((((rb >> 23) & 0xff) + (1023 - 127)) << 20 | (rm >> 3), rm << 29);
    const double y = fma(x, fma(-m, x, 1.0), x);
    return __hiloint2double(__double2hiint(y) - (((hi >> 20) & 0x7ff) - 1023) * (1 << 20), __double2loint(y));
}

// sin(t)/t, (1 - cos t)/t^2, (t - sin t)/t^3 from t^2: Taylor series (truncation
// below 1e-18 for t <= 0.25), sincos otherwise.
__device__ __forceinline__ void se3_coeffs(double th2, double &A, double &B, double &C) {
    if (th2 <= 0.0625) {
        A = fma(th2, fma(th2, fma(th2, fma(th2, fma(th2, fma(th2, 1.0 / 6227020800.0, -1.0 / 39916800.0),
                                                    1.0 / 362880.0), -1.0 / 5040.0), 1.0 / 120.0), -1.0 / 6.0), 1.0);
        B = fma(th2, fma(th2, fma(th2, fma(th2, fma(th2, fma(th2, 1.0 / 87178291200.0, -1.0 / 479001600.0),
                                                    1.0 / 3628800.0), -1.0 / 40320.0), 1.0 / 720.0), -1.0 / 24.0), 0.5);
        C = fma(th2, fma(th2, fma(th2, fma(th2, fma(th2, fma(th2, 1.0 / 1307674368000.0, -1.0 / 6227020800.0),
                                                    1.0 / 39916800.0), -1.0 / 362880.0), 1.0 / 5040.0), -1.0 / 120.0),
                1.0 / 6.0);
    } else {
        const double th = sqrt(th2);
        double sn, cs;
        sincos(th, &sn, &cs);
        A = sn / th;
        B = (1.0 - cs) / th2;
        C = (th - sn) / (th2 * th);
    }
}

// T <- exp(xi^) T (left update), xi = (omega, v): Rodrigues rotation
// R = I + A W + B W^2 and translation V v with V = I + B W + C W^2, where
// W = [omega]_x and W^2 = omega omega^T - |omega|^2 I.
__device__ __forceinline__ void se3_exp_left(const double xi[6], double T[12]) {
    const double w0 = xi[0], w1 = xi[1], w2 = xi[2];
    const double th2 = fma(w0, w0, fma(w1, w1, w2 * w2));
    double A, B, C;
    se3_coeffs(th2, A, B, C);
    const double W[9] = {0.0, -w2, w1, w2, 0.0, -w0, -w1, w0, 0.0};
    const double om[3] = {w0, w1, w2};
    double R[9], V[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double W2 = fma(om[i], om[j], i == j ? -th2 : 0.0);
            const double I = i == j ? 1.0 : 0.0;
            R[3 * i + j] = fma(A, W[3 * i + j], fma(B, W2, I));
            V[3 * i + j] = fma(B, W[3 * i + j], fma(C, W2, I));
        }
    double Tn[12];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = 0; j < 3; ++j)
            Tn[4 * i + j] = fma(R[3 * i], T[j], fma(R[3 * i + 1], T[4 + j], R[3 * i + 2] * T[8 + j]));
        const double te = fma(V[3 * i], xi[3], fma(V[3 * i + 1], xi[4], V[3 * i + 2] * xi[5]));
        Tn[4 * i + 3] = fma(R[3 * i], T[3], fma(R[3 * i + 1], T[7], fma(R[3 * i + 2], T[11], te)));
    }
#pragma unroll
    for (int i = 0; i < 12; ++i) T[i] = Tn[i];
}

// Solve M x = rhs for the symmetric positive-definite 6x6 M given by its
// row-major upper triangle, by the square-root-free Cholesky factorisation
// M = L D L^T (elimination on the upper triangle, then back substitution).
// Returns false when a pivot D_j <= pivot_eps * max diagonal (the same
// quantity a square-root Cholesky compares before its square root).
__device__ __forceinline__ bool solve6(const double *Aup, const double *rhs, double pivot_eps, double *x) {
    double U[6][6];
    double y[6], r[6];
    {
        int p = 0;
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
            for (int j = i; j < 6; ++j) U[i][j] = Aup[p++];
    }
    double dmax = U[0][0];
#pragma unroll
    for (int i = 1; i < 6; ++i) dmax = fmax(dmax, U[i][i]);
    if (!(dmax > 0.0)) return false;
    const double lim = pivot_eps * dmax;
#pragma unroll
    for (int i = 0; i < 6; ++i) y[i] = rhs[i];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const double d = U[j][j];
        if (!(d > lim) || !(d > 1e-300)) return false;
        r[j] = rcp64(d);
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            const double l = U[j][i] * r[j];  // M symmetric: row j, column i of the reduced matrix
#pragma unroll
            for (int k = i; k < 6; ++k) U[i][k] = fma(-l, U[j][k], U[i][k]);
            y[i] = fma(-l, y[j], y[i]);
        }
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        double s = y[i];
#pragma unroll
        for (int k = i + 1; k < 6; ++k) s = fma(-U[i][k], x[k], s);
        x[i] = s * r[i];
    }
    return true;
}

// 1/sqrt(x) for a positive normal x: FP32 seed, two FP64 Newton steps.
__device__ __forceinline__ double rsqrt64(double x) {
    double y = (double)rsqrtf((float)x);
    const double hx = 0.5 * x;
    y = y * fma(-hx * y, y, 1.5);
    y = y * fma(-hx * y, y, 1.5);
    return y;
}

// Gram-Schmidt on the rows of the rotation of a 3x4 pose (FP64, one thread).
__device__ __forceinline__ void orthonormalise_rows(double *T) {
    double *r0 = T, *r1 = T + 4, *r2 = T + 8;
    double n = rsqrt64(fma(r0[0], r0[0], fma(r0[1], r0[1], r0[2] * r0[2])));
    r0[0] *= n;
    r0[1] *= n;
    r0[2] *= n;
    const double d = fma(r0[0], r1[0], fma(r0[1], r1[1], r0[2] * r1[2]));
    r1[0] = fma(-d, r0[0], r1[0]);
    r1[1] = fma(-d, r0[1], r1[1]);
    r1[2] = fma(-d, r0[2], r1[2]);
    n = rsqrt64(fma(r1[0], r1[0], fma(r1[1], r1[1], r1[2] * r1[2])));
    r1[0] *= n;
    r1[1] *= n;
    r1[2] *= n;
    r2[0] = r0[1] * r1[2] - r0[2] * r1[1];
    r2[1] = r0[2] * r1[0] - r0[0] * r1[2];
    r2[2] = r0[0] * r1[1] - r0[1] * r1[0];
}

// C = A B for 3x4 poses on one warp: lane e < 12 computes entry e.  C may alias an input: every
// lane reads its operands before any lane writes.
__device__ __forceinline__ void warp_pose_mul(const double *A, const double *B, double *C) {
    const int lane = threadIdx.x & 31;
    const int i = lane < 12 ? lane / 4 : 0, j = lane < 12 ? lane % 4 : 0;
    const double v =
        fma(A[4 * i], B[j], fma(A[4 * i + 1], B[4 + j], fma(A[4 * i + 2], B[8 + j], j == 3 ? A[4 * i + 3] : 0.0)));
    __syncwarp();
    if (lane < 12) C[lane] = v;
    __syncwarp();
}

// C = A^-1 = [R^T | -R^T t] on one warp.
__device__ __forceinline__ void warp_pose_inv(const double *A, double *C) {
    const int lane = threadIdx.x & 31;
    const int i = lane < 12 ? lane / 4 : 0, j = lane < 12 ? lane % 4 : 0;
    const double v = j < 3 ? A[4 * j + i] : -fma(A[i], A[3], fma(A[4 + i], A[7], A[8 + i] * A[11]));
    __syncwarp();
    if (lane < 12) C[lane] = v;
    __syncwarp();
}

// Neumaier-compensated FP32 accumulation: (s, c) holds s + c.
__device__ __forceinline__ void kadd(float &s, float &c, float v) {
    const float t = s + v;
    c += fabsf(s) >= fabsf(v) ? (s - t) + v : (v - t) + s;
    s = t;
}

// Lane of the upper-triangle element (i, k), i <= k, in row-major order (0..20).
__device__ __forceinline__ int uidx(int i, int k) { return i * 6 - (i * (i - 1)) / 2 + (k - i); }

// d's mantissa as a double in [1, 2) (its exponent field set to the bias) and its unbiased exponent.
__device__ __forceinline__ double dmant(double d) {
    return __longlong_as_double((__double_as_longlong(d) & ~(0x7ffLL << 52)) | (1023LL << 52));
}
__device__ __forceinline__ int dexpo(double d) { return ((__double2hiint(d) >> 20) & 0x7ff) - 1023; }

// x * 2^-e by exponent arithmetic (exact for normal results); zero stays zero, results below the
// normal range become signed zero and above it signed infinity.
__device__ __forceinline__ double dscale2(double x, int e) {
    const long long b = __double_as_longlong(x);
    const int ef = (int)((b >> 52) & 0x7ff);
    if (ef == 0) return x;
    const int en = ef - e;
    const long long sign = b & (long long)0x8000000000000000ull;
    if (en <= 0) return __longlong_as_double(sign);
    if (en >= 0x7ff) return __longlong_as_double(sign | (0x7ffLL << 52));
    return __longlong_as_double((b & ~(0x7ffLL << 52)) | ((long long)en << 52));
}

// FP64 solve of A xi = -b for the symmetric 6x6 A by elimination (the square-root-free Cholesky
// factorisation A = L D L^T, i.e. symmetric Gaussian elimination), spread over the
// lanes of one warp: lanes 0..20 hold the upper triangle of A (lane uidx(i, k)),
// lanes 21..26 the right-hand side.  GB300 issues an FP64 warp instruction every
// 64 cycles whatever its active lanes, so independent work goes across lanes and
// the elimination is division-free: step j replaces every later row by
//     row <- mant(D_j) row - (L_jrow 2^-exp(D_j)) row_j,
// i.e. the Schur complement scaled by D_j / 2^exp(D_j) in [1, 2), with the power
// of two taken off by exponent arithmetic: one multiply and one multiply-add per
// step and no reciprocal on the chain.  Row j then holds F_j times the standard
// pivot row (F_j = prod_{m<j} mant(D_m) < 2^j), so the pivot test uses
// D_j / F_j, and the back substitution, which the common factor of a row does
// not change, scales every row by its reciprocal pivot in one instruction and
// then takes one multiply-add per unknown.  Comparisons, maxima and sign flips
// are integer instructions on the bit patterns.
// False when a standard pivot D_j / F_j <= max(pivot_eps * max diagonal, 1e-300),
// a pivot is not finite, or the solution is not finite.
// (Out of line: it solves only what warp_solve6 below leaves to it.  Returns xi[k] in lane k < 6 as *x.)
static __device__ __noinline__ bool warp_solve6_pivots(const double *tot, double pivot_eps, double *x) {
    double xi[6];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool is_u = lane < 21, is_y = lane >= 21 && lane < 27;
    int li = -1, lk = -1;
    if (is_u) {
        int i = 0, rem = lane;
        while (rem >= 6 - i) {
            rem -= 6 - i;
            ++i;
        }
        li = i;
        lk = i + rem;
    } else if (is_y) {
        li = lane - 21;
        lk = 6;
    }
    const double t = (is_u || is_y) ? tot[lane] : 0.0;
    double u = is_y ? dneg(t) : t;
    long long dm = dbits(tot[0]);
#pragma unroll
    for (int i = 1; i < 6; ++i) dm = max(dm, dbits(tot[uidx(i, i)]));
    if (!(dm > 0) || !dfinite(__longlong_as_double(dm))) return false;
    const double lim = __longlong_as_double(max(dbits(pivot_eps * __longlong_as_double(dm)), dbits(1e-300)));
    double piv[6], mnt[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const double d = __shfl_sync(full, u, uidx(j, j));
        const bool act = li > j;
        const int src_l = act ? uidx(j, li) : lane;
        const int src_k = act ? (is_u ? uidx(j, lk) : 21 + j) : lane;
        const double ujl = __shfl_sync(full, u, src_l);
        const double ujk = __shfl_sync(full, u, src_k);
        piv[j] = d;
        mnt[j] = dmant(d);
        if (act) u = fma(-dscale2(ujl, dexpo(d)), ujk, mnt[j] * u);
    }
    // pivot test on the standard pivots D_j / F_j: lane j < 6 forms F_j = prod_{m<j} mant(D_m)
    double F = 1.0;
#pragma unroll
    for (int m = 0; m < 5; ++m) F = m < lane ? F * mnt[m] : F;
    const int jl = lane < 6 ? lane : 0;
    double pj = piv[0];
#pragma unroll
    for (int j = 1; j < 6; ++j) pj = jl == j ? piv[j] : pj;
    const bool bad = lane < 6 && (!dfinite(pj) || !(dbits(pj) > dbits(lim * F)));
    if (__any_sync(full, bad)) return false;
    // back substitution: lane (i, k) -> S_ik / D_i, lane 21 + i -> y_i / D_i
    double di = piv[0];
#pragma unroll
    for (int j = 1; j < 6; ++j) di = li == j ? piv[j] : di;
    double v = li >= 0 ? u * rcp64(di) : 0.0;
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        const double x = __shfl_sync(full, v, 21 + i);
        xi[i] = x;
        if (i > 0) {
            const bool act = is_y && li < i;
            const double lmi = __shfl_sync(full, v, act ? uidx(li, i) : lane);
            if (act) v = fma(-lmi, x, v);
        }
    }
    bool fin = true;
    double r = xi[0];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        fin = fin && dfinite(xi[i]);
        r = lane == i ? xi[i] : r;
    }
    *x = r;
    return fin;
}

// Field `lane` (5 bits each, lanes 0..11) of a packed table of lane numbers.
__device__ __forceinline__ int lane_tab(unsigned long long tab, int lane) { return (int)(tab >> (5 * lane)) & 31; }
constexpr unsigned long long lane_tab6(int a, int b, int c, int d, int e, int f) {
    return (unsigned long long)a | (unsigned long long)b << 5 | (unsigned long long)c << 10 |
           (unsigned long long)d << 15 | (unsigned long long)e << 20 | (unsigned long long)f << 25;
}

// FP64 solve of A xi = -b on one warp, by 3 x 3 blocks.  With A = [P Q; Q^T S], C = adj P and d = det P,
//     W = C Q, v = C b_1, S'' = d S - Q^T W, z = d b_2 - Q^T v, C'' = adj S'', d'' = det S'',
//     x_2 = C'' z / d'', x_1 = (v - W x_2) / d, xi = -x,
// every line a set of sums of two to four products, one sum to a lane: 21 dependent FP64 instructions and seven
// exchanges between lanes, where the pivoting elimination above takes 30 and nineteen.  An FP64 instruction takes
// 64 cycles of its warp whatever its active lanes, so the number on the chain is the time: 3851 cycles
// (1.86 us) for the elimination, 2177 (1.05 us) for this form.
//
// Which systems it solves: a difference of products is good to 2^-53 of the products, not of itself, so this form
// loses what d is below the product of P's diagonal and what det S is below that of S's.  Both losses are read off
// the exponents and may come to kBlockLoss bits; neither depends on the units of A's rows.  Beyond, where a pivot is
// not certain to be above 2^-24 of the largest diagonal element, whenever pivot_eps asks for more, and when a value
// is not finite, the elimination solves the system and decides whether it is degenerate (then both are paid for).
// The 3062 systems of streams, registrations and batches of hypotheses on sweeps of 16x512 to 128x2048 lose one bit
// at most; largest relative error of xi there against 113-bit solutions 7e-15 (elimination: 1.0e-14).  Of random
// spectra in random bases, with and without rows of unlike scale, and of corridors, round tunnels, ground planes and
// frames far from their points, the accepted ones: 4.8e-14 (5.5e-14); at five bits or more some lose more digits
// here than there.
// *x: lane k < 6 holds xi[k].
constexpr int kBlockLoss = 3;
__device__ __forceinline__ bool warp_solve6(const double *tot, double pivot_eps, double *x) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    // symmetric 3 x 3 matrices: elements (0,0) (0,1) (0,2) (1,1) (1,2) (2,2) in lanes 0..5; cofactor p is
    // m[a] m[b] - m[c] m[d]
    constexpr unsigned long long kCa = lane_tab6(3, 2, 1, 0, 1, 0), kCb = lane_tab6(5, 4, 4, 5, 2, 3),
                                 kCc = lane_tab6(4, 1, 2, 2, 0, 1), kCd = lane_tab6(4, 5, 3, 2, 4, 1);
    const int l6 = lane < 6 ? lane : 0;
    const int ca = lane_tab(kCa, l6), cb = lane_tab(kCb, l6), cc = lane_tab(kCc, l6), cd = lane_tab(kCd, l6);
    // element e of P in the upper triangle: 0 1 2 6 7 11
    constexpr unsigned long long kP = lane_tab6(0, 1, 2, 6, 7, 11);
    const double c1 = fma(tot[lane_tab(kP, ca)], tot[lane_tab(kP, cb)],
                          dneg(tot[lane_tab(kP, cc)] * tot[lane_tab(kP, cd)]));
    // W (lanes 0..8), v (9..11), d (12): rows of C times columns of Q, b_1, the first row of P
    const int wi = lane < 9 ? lane / 3 : (lane < 12 ? lane - 9 : 0), wj = lane - 3 * (lane / 3);
    const int x0 = lane < 9 ? 3 + wj : (lane < 12 ? 21 : 0), x1i = lane < 9 ? 8 + wj : (lane < 12 ? 22 : 1),
              x2i = lane < 9 ? 12 + wj : (lane < 12 ? 23 : 2);
    const int r0 = wi, r1 = wi == 0 ? 1 : wi + 2, r2 = wi == 0 ? 2 : wi + 3;  // row wi of a symmetric matrix
    const double wv = fma(__shfl_sync(full, c1, r0), tot[x0],
                          fma(__shfl_sync(full, c1, r1), tot[x1i], __shfl_sync(full, c1, r2) * tot[x2i]));
    const double det = __shfl_sync(full, wv, 12);
    // S'' (lanes 0..5), z (6..8)
    const int si = lane < 6 ? lane_tab(lane_tab6(0, 0, 0, 1, 1, 2), lane) : (lane < 9 ? lane - 6 : 0);
    const int sj = lane_tab(lane_tab6(0, 1, 2, 1, 2, 2), l6);
    const int w0 = lane < 6 ? sj : 9, w1 = lane < 6 ? 3 + sj : 10, w2 = lane < 6 ? 6 + sj : 11;
    const double top = tot[lane < 6 ? 15 + lane : (lane < 9 ? 18 + lane : 15)];
    const double sz = fma(dneg(tot[3 + si]), __shfl_sync(full, wv, w0),
                          fma(dneg(tot[8 + si]), __shfl_sync(full, wv, w1),
                              fma(dneg(tot[12 + si]), __shfl_sync(full, wv, w2), det * top)));
    const double c2 = fma(__shfl_sync(full, sz, ca), __shfl_sync(full, sz, cb),
                          dneg(__shfl_sync(full, sz, cc) * __shfl_sync(full, sz, cd)));
    // C'' z (lanes 0..2), d'' (lane 3)
    const int ui = lane < 3 ? lane : 0, ub = lane < 3 ? 6 : 0;
    const int u1 = ui == 0 ? 1 : ui + 2, u2 = ui == 0 ? 2 : ui + 3;
    const double ud = fma(__shfl_sync(full, c2, ui), __shfl_sync(full, sz, ub),
                          fma(__shfl_sync(full, c2, u1), __shfl_sync(full, sz, ub + 1),
                              __shfl_sync(full, c2, u2) * __shfl_sync(full, sz, ub + 2)));
    const double det2 = __shfl_sync(full, ud, 3);
    // 1 / d'' in lanes 0..2, 1 / d elsewhere
    const double rc = rcp64_scaled(lane < 3 ? det2 : det);
    const double xb = ud * rc;  // x_2 in lanes 0..2
    const double rd = __shfl_sync(full, rc, 3);
    const int l3 = lane < 3 ? lane : 0;
    const double q0 = __shfl_sync(full, wv, 3 * l3), q1 = __shfl_sync(full, wv, 3 * l3 + 1),
                 q2 = __shfl_sync(full, wv, 3 * l3 + 2), vi = __shfl_sync(full, wv, 9 + l3);
    const double xa = fma(dneg(q0), __shfl_sync(full, xb, 0),
                          fma(dneg(q1), __shfl_sync(full, xb, 1), fma(dneg(q2), __shfl_sync(full, xb, 2), vi))) * rd;
    const double xb3 = __shfl_sync(full, xb, lane >= 3 && lane < 6 ? lane - 3 : 0);
    *x = dneg(lane < 3 ? xa : xb3);
    // every pivot certainly above 2^-24 of the largest diagonal element (in [2^em, 2^(em+1)))?  The pivots are
    // P_00, minor / P_00, d / minor, S''_00 / d, minor'' / (S''_00 d), d'' / (minor'' d)
    const int d0 = __double2hiint(tot[0]), d1 = __double2hiint(tot[6]), d2 = __double2hiint(tot[11]),
              d3 = __double2hiint(tot[15]), d4 = __double2hiint(tot[18]), d5 = __double2hiint(tot[20]);
    const int hm = max(max(max(d0, d1), max(d2, d3)), max(d4, d5));
    const int h1 = __shfl_sync(full, __double2hiint(c1), 5), h2 = __double2hiint(det);
    const int h3 = __shfl_sync(full, __double2hiint(sz), 0), h4 = __shfl_sync(full, __double2hiint(c2), 5),
              h5 = __double2hiint(det2);
    const int em = (hm >> 20) - 1023, e0 = (d0 >> 20) - 1023, e1 = (h1 >> 20) - 1023, e2 = (h2 >> 20) - 1023,
              e3 = (h3 >> 20) - 1023, e4 = (h4 >> 20) - 1023, e5 = (h5 >> 20) - 1023;
    const int low = em - 23 + 1;
    // bits that d is below P_00 P_11 P_22, and d'' = d^3 det S below d^3 S_00 S_11 S_22
    const int loss1 = (d0 >> 20) + (d1 >> 20) + (d2 >> 20) - 3 * 1023 - e2;
    const int loss2 = (d3 >> 20) + (d4 >> 20) + (d5 >> 20) - 3 * 1023 + 3 * e2 - e5;
    // (d'' is a product of twelve elements, between 2^(12 em - 288) and 2^(12 em + 12) with such pivots: em keeps it
    // and its reciprocal normal numbers.  Below, d'' underflows to zero, whose exponent field is no exponent.)
    const bool good = (d0 | h1 | h2 | h3 | h4 | h5) >= 0 && e0 >= low && e1 - e0 > low && e2 - e1 > low &&
                      e3 - e2 > low && e4 - e3 - e2 - 1 > low && e5 - e4 - e2 - 1 > low && loss1 <= kBlockLoss &&
                      loss1 + loss2 <= kBlockLoss && em > -59 && em < 83 &&
                      dbits(pivot_eps) <= dbits(2.9802322387695312e-08);  // 2^-25
    if (good && __all_sync(full, dfinite(*x))) return true;
    return warp_solve6_pivots(tot, pivot_eps, x);
}

// (-1)^n / (2n + 1 + c)!: the n-th Taylor coefficient in t^2 of sin(t)/t (c = 0),
// (1 - cos t)/t^2 (c = 1) and (t - sin t)/t^3 (c = 2).
__device__ __forceinline__ double se3_taylor_coef(int n, int c) {
    constexpr double k[6][3] = {
        {1.0, 1.0 / 2.0, 1.0 / 6.0},
        {-1.0 / 6.0, -1.0 / 24.0, -1.0 / 120.0},
        {1.0 / 120.0, 1.0 / 720.0, 1.0 / 5040.0},
        {-1.0 / 5040.0, -1.0 / 40320.0, -1.0 / 362880.0},
        {1.0 / 362880.0, 1.0 / 3628800.0, 1.0 / 39916800.0},
        {-1.0 / 39916800.0, -1.0 / 479001600.0, -1.0 / 6227020800.0},
    };
    return c == 0 ? k[n][0] : (c == 1 ? k[n][1] : k[n][2]);
}

// The same coefficients for any t, by sincos (out of line: a step is rarely above a quarter of a radian).
static __device__ __noinline__ double se3_coef_large(double th2, int c) {
    double A, B, C;
    se3_coeffs(th2, A, B, C);
    return c == 0 ? A : (c == 1 ? B : C);
}

// T <- exp(xi^) T on one warp, xi[k] in lane k < 6; returns whether |omega|^2 < er2 and |v|^2 < et2.
// R = I + A W + B W^2 (lanes 0..8, one entry each) and V = I + B W + C W^2 (lanes 9..17), W^2 entry by entry as
// omega_i omega_j or -(omega_j^2 + omega_k^2); the same three instructions give |omega|^2 (lane 18) and |v|^2
// (lane 19).  Lanes 0..2 evaluate the coefficients A, B, C by their series, cut where the remainder (below the
// first omitted term) is under 5e-17 relative: degree 1 in t^2 for t^2 <= 2^-24, 2 for 2^-14, 3 for 2^-9, 4 for
// 2^-6, 5 for 2^-4, sincos beyond.  Then lanes 0..11 each compose one entry of R T and lanes 12..14 one entry of
// V v, which the translation lanes add.  T lives in shared memory (12 doubles) and is updated in place; Tf, when
// given, receives the new pose in FP32.  0.67 us a call: 10 to 12 FP64 instructions on the chain, where an
// update and a separate convergence test took 16 and 1.02 us.
__device__ __forceinline__ bool warp_se3_update(double x, double *T, float *Tf, double er2, double et2) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int e = lane < 9 ? lane : (lane < 18 ? lane - 9 : 0);
    const int ei = e / 3, ek = e - 3 * (e / 3);
    const bool norm = lane == 18 || lane == 19;  // lane 18: omega, lane 19: v
    const int nb = lane == 19 ? 3 : 0;
    const bool diag = ei == ek;
    const int o1 = ei == 2 ? 0 : ei + 1, o2 = ei == 0 ? 2 : ei - 1;  // the two other axes of a diagonal entry
    // p = a b + c^2 + f^2: omega_i omega_k; omega_j^2 + omega_k^2; the squared norms
    const double pa = __shfl_sync(full, x, norm ? nb + 2 : (diag ? o1 : ei));
    const double pb = __shfl_sync(full, x, norm ? nb + 2 : (diag ? o1 : ek));
    const double pc0 = __shfl_sync(full, x, norm ? nb + 1 : o2), pf0 = __shfl_sync(full, x, nb);
    const int wl = diag ? 0 : 3 - ei - ek;
    const double wx = __shfl_sync(full, x, wl);  // the component of an off-diagonal entry of W
    const double pc = norm || diag ? pc0 : 0.0, pf = norm ? pf0 : 0.0;
    const double pp = fma(pf, pf, fma(pc, pc, pa * pb));
    const double th2 = __shfl_sync(full, pp, 18);
    const bool below = dbits(pp) < dbits(lane == 18 ? er2 : et2);
    const bool conv = ((__ballot_sync(full, below) >> 18) & 3u) == 3u;
    const double W2 = diag ? dneg(pp) : pp;
    const long long tb = dbits(th2);
    const int c = lane < 3 ? lane : 0;
    double coef;
    if (tb <= dbits(5.9604644775390625e-08)) {  // 2^-24
        coef = fma(th2, se3_taylor_coef(1, c), se3_taylor_coef(0, c));
    } else if (tb <= dbits(6.103515625e-05)) {  // 2^-14
        coef = fma(th2, fma(th2, se3_taylor_coef(2, c), se3_taylor_coef(1, c)), se3_taylor_coef(0, c));
    } else if (tb <= dbits(0.0625)) {
        const int deg = tb <= dbits(0.001953125) ? 3 : (tb <= dbits(0.015625) ? 4 : 5);
        coef = deg == 5 ? se3_taylor_coef(5, c) : 0.0;
        coef = deg >= 4 ? fma(th2, coef, se3_taylor_coef(4, c)) : 0.0;
#pragma unroll
        for (int n = 3; n >= 0; --n) coef = fma(th2, coef, se3_taylor_coef(n, c));
    } else {
        coef = se3_coef_large(th2, c);
    }
    const double c1 = __shfl_sync(full, coef, lane < 9 ? 0 : 1), c2 = __shfl_sync(full, coef, lane < 9 ? 1 : 2);
    // W = [omega]_x: W[i][k] = -eps_ikl omega_l
    const bool neg = ek - ei == 1 || ek - ei == -2;
    const double Wik = diag ? 0.0 : (neg ? dneg(wx) : wx);
    const double ent = fma(c1, Wik, fma(c2, W2, diag ? 1.0 : 0.0));
    // lanes 0..11: (R T)(i, j), i = lane / 4, j = lane % 4; lanes 12..14: (V v)(lane - 12)
    const bool comp = lane < 12, tv = lane >= 12 && lane < 15;
    const int oi = comp ? lane / 4 : (tv ? lane - 12 : 0), oj = comp ? lane % 4 : 0;
    const int src = tv ? 9 + 3 * oi : 3 * oi;
    const double v0 = __shfl_sync(full, x, 3), v1 = __shfl_sync(full, x, 4), v2 = __shfl_sync(full, x, 5);
    const double X0 = tv ? v0 : T[oj], X1 = tv ? v1 : T[4 + oj], X2 = tv ? v2 : T[8 + oj];
    const double M0 = __shfl_sync(full, ent, src), M1 = __shfl_sync(full, ent, src + 1),
                 M2 = __shfl_sync(full, ent, src + 2);
    const double o = fma(M0, X0, fma(M1, X1, M2 * X2));
    const double te = __shfl_sync(full, o, 12 + oi);
    const double out = oj == 3 ? o + te : o;
    __syncwarp();
    if (lane < 12) {
        T[lane] = out;
        if (Tf) Tf[lane] = (float)out;
    }
    __syncwarp();
    return conv;
}

// ----------------------------------------------------------------------------- exact order-free sums
//
// A float v is held as the integer X = v * 2^48 (truncated toward zero below 2^-48, saturated at |v| = 2^47).
// Within a CTA X is split into 24-bit chunks, which 32-bit integer reductions add exactly; between CTAs into
// words X = w0 + w1 2^32 + w2 2^64 that add into 64-bit integers with no carry between them.  A sum of floats
// formed this way is exact and does not depend on the order of the additions (integer atomics from any number
// of CTAs give every reader the same bits).

// X = v * 2^48 as four 24-bit chunks (the upper one of a pair signed): X = c[0] + c[1] 2^24 + c[2] 2^48 + c[3] 2^72.
__device__ __forceinline__ void fx_chunks24(float v, int c[4]) {
    const unsigned b = __float_as_uint(v);
    const int e = (int)((b >> 23) & 0xffu);
    // (an infinity or NaN counts as the largest value)
    int m = (int)((e == 0xff ? 0u : b & 0x7fffffu) | (e ? 0x800000u : 0u));
    int sh = min((e ? e : 1) - 150 + 48, 71);  // X = m * 2^sh, |X| < 2^95
    m >>= min(max(-sh, 0), 24);
    sh = max(sh, 0);
    m = (int)b < 0 ? -m : m;
    const int q = sh >= 48 ? 2 : (sh >= 24 ? 1 : 0);
    const int r = sh - 24 * q;
    const int lo = (int)(((unsigned)m << r) & 0xffffffu), hi = m >> (24 - r);  // m 2^r = hi 2^24 + lo
    c[0] = q == 0 ? lo : 0;
    c[1] = q == 1 ? lo : (q == 0 ? hi : 0);
    c[2] = q == 2 ? lo : (q == 1 ? hi : 0);
    c[3] = q == 2 ? hi : 0;
}

// The sum of up to 16 numbers' 24-bit chunks as three words s0 + s1 2^32 + s2 2^64, each below 2^36 in magnitude.
__device__ __forceinline__ void fx_words(int r0, int r1, int r2, int r3, long long w[3]) {
    const long long a = (long long)r0 + ((long long)r1 << 24), b = (long long)r2 + ((long long)r3 << 24);
    w[0] = a & 0xffffffffll;
    w[1] = (a >> 32) + ((b & 0xffffll) << 16);  // b 2^48 = (b mod 2^16) 2^48 + (b >> 16) 2^64
    w[2] = b >> 16;
}

// (s0 + s1 2^32 + s2 2^64) * 2^-48 as the nearest double (ties to even), integer instructions only: the sum as
// 128 bits, its magnitude shifted to the top, rounded at bit 11 of the upper half.
__device__ __forceinline__ double fx_value(long long s0, long long s1, long long s2) {
    const long long t1 = s1 + (s0 >> 32);
    long long hs = s2 + (t1 >> 32);
    unsigned long long l = ((unsigned long long)t1 << 32) | (unsigned)s0;
    const bool neg = hs < 0;
    unsigned long long h = (unsigned long long)hs;
    if (neg) {
        l = 0ull - l;
        h = ~h + (l == 0ull ? 1ull : 0ull);
    }
    if ((h | l) == 0ull) return 0.0;
    int n = 0;  // leading zeros of the 128 bits
    if (h == 0ull) {
        h = l;
        l = 0ull;
        n = 64;
    }
    const int z = __clzll((long long)h);
    n += z;
    const unsigned long long top = (h << z) | ((l >> 1) >> (63 - z)), rest = l << z;
    unsigned long long m = top >> 11;
    const bool up = (top >> 10) & 1ull, sticky = (top & 0x3ffull) != 0ull || rest != 0ull;
    if (up && (sticky || (m & 1ull))) ++m;
    // the value is (m 2^-52) 2^(127 - n - 48), m in [2^52, 2^53]; m's leading one is added into the exponent
    const unsigned long long bits =
        ((neg ? 0x800ull : 0ull) << 52) + ((unsigned long long)(127 - n - 48 + 1023 - 1) << 52) + m;
    return __longlong_as_double((long long)bits);
}

// ----------------------------------------------------------------------------- sweep front end (Sec. III-A)
//
// The per-point and per-pixel bodies of projection, resolve and normals, shared by
// the standalone kernels and the fused register launch so both give the same bits.
// kCg selects L2-only loads for z-buffer words that the same launch wrote earlier.

// Pass 1 of the z-buffer: the point's key (bits(range) << 32 | index) into its pixel.
__device__ __forceinline__ void project_point(const float4 *pts, int i, const upslam_pano &pp,
                                              unsigned long long *zbuf) {
    const float4 p = __ldg(pts + i);
    if (p.w == 0.0f) return;
    int v, u;
    float r;
    if (!bin_point(p.x, p.y, p.z, pp, v, u, r)) return;
    const unsigned long long key = ((unsigned long long)__float_as_uint(r) << 32) | (unsigned int)i;
    atomicMin(zbuf + (size_t)v * pp.cols + u, key);
}

// Pass 2: decode the pixel's word into depth / index / point and (kReset) reset the word.
template <bool kCg, bool kReset = true>
__device__ __forceinline__ void resolve_pixel(const float4 *pts, int k, unsigned long long *zbuf, float *depth,
                                              int *idx, float4 *pix) {
    const unsigned long long key = kCg ? __ldcg(zbuf + k) : zbuf[k];
    if (key == kEmptyKey) {
        depth[k] = 0.0f;
        idx[k] = -1;
        if (pix) pix[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
        if (kReset) zbuf[k] = kEmptyKey;
        const int i = (int)(key & 0xffffffffull);
        depth[k] = __uint_as_float((unsigned int)(key >> 32));
        idx[k] = i;
        if (pix) {
            const float4 p = __ldg(pts + i);
            pix[k] = make_float4(p.x, p.y, p.z, 1.0f);
        }
    }
}

// Pixel data for the normals, read from the resolved arrays (point with validity in .w, range) by ordinary loads: the
// launch before may still be writing them when the kernel's CTAs are placed.
struct PixArrays {
    const float4 *pix;
    const float *depth;
    __device__ __forceinline__ float4 point(int k) const { return pix[k]; }
    __device__ __forceinline__ float range(int k) const { return depth[k]; }
};

// The same data decoded straight from the z-buffer words (winner index and range in the key),
// before any resolve pass has run: a pixel's normal can then be formed in the pass that resolves it.
struct PixZbuf {
    const float4 *pts;
    const unsigned long long *zbuf;
    __device__ __forceinline__ float4 point(int k) const {
        const unsigned long long key = __ldcg(zbuf + k);
        if (key == kEmptyKey) return make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 p = __ldg(pts + (int)(key & 0xffffffffull));
        return make_float4(p.x, p.y, p.z, 1.0f);
    }
    __device__ __forceinline__ float range(int k) const {
        const unsigned long long key = __ldcg(zbuf + k);
        return key == kEmptyKey ? 0.0f : __uint_as_float((unsigned int)(key >> 32));
    }
};

// Normal of pixel k: a toward column + 1 (wrapping), b toward row + 1, each replaced by the
// opposite neighbour with the sign flipped when unusable; n = a x b, normalised, toward the
// sensor; (0, 0, 0, 0) when there is none.  A neighbour is usable when it holds a point and its
// range is within jump_rel * d + jump_abs of the pixel's (FP32, round to nearest).
template <typename Acc>
__device__ __forceinline__ float4 normal_pixel(const Acc &px, const upslam_pano &pp, const upslam_normal_params &np,
                                               int k) {
    const int H = pp.rows, W = pp.cols;
    const int v = k / W, u = k - v * W;
    const int kr = v * W + (u + 1 == W ? 0 : u + 1);
    const int kl = v * W + (u == 0 ? W - 1 : u - 1);
    const int kd = v + 1 < H ? k + W : k, ku = v >= 1 ? k - W : k;  // (past the edge: k, unused)
    // every pixel the normal may use, read before any test, so the reads overlap
    const float4 c = px.point(k), qr = px.point(kr), ql = px.point(kl), qd = px.point(kd), qu = px.point(ku);
    const float d = px.range(k), dr = px.range(kr), dl = px.range(kl), dd = px.range(kd), du = px.range(ku);
    float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c.w == 0.0f) return out;
    const float lim = __fadd_rn(__fmul_rn(np.jump_rel, d), np.jump_abs);
    auto usable = [&](const float4 &q, float dn) { return q.w != 0.0f && !(fabsf(__fsub_rn(dn, d)) > lim); };
    float3 a, b;
    if (usable(qr, dr)) {
        a = make_float3(qr.x - c.x, qr.y - c.y, qr.z - c.z);
    } else if (usable(ql, dl)) {
        a = make_float3(c.x - ql.x, c.y - ql.y, c.z - ql.z);
    } else {
        return out;
    }
    if (v + 1 < H && usable(qd, dd)) {
        b = make_float3(qd.x - c.x, qd.y - c.y, qd.z - c.z);
    } else if (v >= 1 && usable(qu, du)) {
        b = make_float3(c.x - qu.x, c.y - qu.y, c.z - qu.z);
    } else {
        return out;
    }
    const float3 n = make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
    const float nn = sqrtf(n.x * n.x + n.y * n.y + n.z * n.z);
    const float na = sqrtf(a.x * a.x + a.y * a.y + a.z * a.z);
    const float nb = sqrtf(b.x * b.x + b.y * b.y + b.z * b.z);
    if (nn >= np.min_cross * na * nb && nn > 0.0f) {
        float s = 1.0f / nn;
        if (n.x * c.x + n.y * c.y + n.z * c.z > 0.0f) s = -s;
        out = make_float4(n.x * s, n.y * s, n.z * s, 1.0f);
    }
    return out;
}

// ----------------------------------------------------------------------------- keyframe update pieces

// Everything one keyframe update reads and writes.
struct FuseView {
    upslam_pano kp;
    float *kdepth;
    void *knw;
    int kprec;
    const float *kdirs;
    upslam_pano sp;
    const float4 *spix;
    const void *snrm;
    int sprec;
    float d_max2, cos_min, w_max, accept;
    unsigned long long *zbuf;
};

// Average the sweep sample that keyframe pixel k (point s, normal + count nk,
// depth d, nk.w > 0) projects onto into the pixel, if the similarity gate keeps
// the pair (Sec. III-C).  Shared by upslam_fuse and the fused register+update.
__device__ __forceinline__ void fuse_average(const FuseView &f, const PoseF &T, int k, float3 s, float4 nk, float d) {
    const float w = nk.w;
    const float3 q = xform_inv(T, s.x, s.y, s.z);
    int jv, ju;
    float rr;
    if (!bin_point(q.x, q.y, q.z, f.sp, jv, ju, rr)) return;
    const int j = jv * f.sp.cols + ju;
    const float4 P = __ldcg(f.spix + j);
    const float4 m = load_nw_cg(f.snrm, j, f.sprec);
    if (P.w == 0.0f || m.w == 0.0f) return;
    const float *r = T.r;
    const float px = fmaf(r[0], P.x, fmaf(r[1], P.y, fmaf(r[2], P.z, r[3])));
    const float py = fmaf(r[4], P.x, fmaf(r[5], P.y, fmaf(r[6], P.z, r[7])));
    const float pz = fmaf(r[8], P.x, fmaf(r[9], P.y, fmaf(r[10], P.z, r[11])));
    const float ex = px - s.x, ey = py - s.y, ez = pz - s.z;
    if (!(fmaf(ex, ex, fmaf(ey, ey, ez * ez)) <= f.d_max2)) return;
    const float3 Rm = rotate(T, m.x, m.y, m.z);
    if (!(fmaf(Rm.x, nk.x, fmaf(Rm.y, nk.y, Rm.z * nk.z)) >= f.cos_min)) return;
    const float dm = sqrtf(fmaf(px, px, fmaf(py, py, pz * pz)));
    const float inv = 1.0f / (w + 1.0f);
    f.kdepth[k] = fmaf(w, d, dm) * inv;
    const float nx = fmaf(w, nk.x, Rm.x), ny = fmaf(w, nk.y, Rm.y), nz = fmaf(w, nk.z, Rm.z);
    const float l = rsqrtf(fmaf(nx, nx, fmaf(ny, ny, nz * nz)));
    const float wn = w + 1.0f < f.w_max ? w + 1.0f : f.w_max;
    store_nw(f.knw, k, f.kprec, make_float4(nx * l, ny * l, nz * l, wn));
}

// Hole fill, first pass for sweep pixel j: its z-buffer key into the empty
// keyframe pixel it lands on.  Returns false when it lands on no empty pixel.
__device__ __forceinline__ bool holefill_key(const FuseView &f, const PoseF &T, int j, int &k,
                                             unsigned long long &key, float &range, float4 &m) {
    const float4 P = __ldcg(f.spix + j);
    m = load_nw_cg(f.snrm, j, f.sprec);  // read with the point (unused when the point is empty)
    if (P.w == 0.0f) return false;
    if (m.w == 0.0f) return false;
    const float3 p = xform(T, P.x, P.y, P.z);
    int v, u;
    if (!bin_point(p.x, p.y, p.z, f.kp, v, u, range)) return false;
    k = v * f.kp.cols + u;
    key = ((unsigned long long)__float_as_uint(range) << 32) | (unsigned int)j;
    return true;
}

// Hole fill, second pass: the winning sweep pixel writes the keyframe pixel
// (d = range, n = unit(R m), w = 1) and resets its z-buffer word.
__device__ __forceinline__ void holefill_write(const FuseView &f, const PoseF &T, int k, float range, float4 m) {
    f.zbuf[k] = 0xffffffffffffffffull;
    const float3 Rm = rotate(T, m.x, m.y, m.z);
    const float l = rsqrtf(fmaf(Rm.x, Rm.x, fmaf(Rm.y, Rm.y, Rm.z * Rm.z)));
    f.kdepth[k] = range;
    store_nw(f.knw, k, f.kprec, make_float4(Rm.x * l, Rm.y * l, Rm.z * l, 1.0f));
}

// ----------------------------------------------------------------------------- programmatic dependent launch
//
// Where one entry point runs several kernels in a row, the later ones are launched with
// launch_dependent: their CTAs may be placed while the kernel before them drains, and each runs
// pdl_wait() before it reads anything that this kernel or one before it writes (the wait returns once the
// previous grid has finished and its writes are visible).  A kernel lets its successor start early with
// pdl_release(); without it the successor starts at its end, as an ordinary launch would.  A dependent
// kernel waits before it ends, and releases after its wait; one that releases without a wait is launched
// as an ordinary one.  So the previous grid's end is also the end of all before it.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace upslam

// ----------------------------------------------------------------------------- host helpers

#define UPSLAM_CHECK_LAUNCH()                                     \
    do {                                                          \
        if (cudaPeekAtLastError() != cudaSuccess) {               \
            (void)cudaGetLastError();                             \
            return UPSLAM_ERR_CUDA;                               \
        }                                                         \
    } while (0)

// A launch that may overlap the previous kernel on the stream (the kernel must call pdl_wait()
// before it reads that kernel's results).  False when the launch fails.
template <typename... KArgs, typename... Args>
static inline bool launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                    Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kernel, args...) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return true;
}

static inline bool upslam_pano_ok(const upslam_pano *pp) {
    return pp && pp->rows > 0 && pp->cols > 0 && (int64_t)pp->rows * pp->cols < (int64_t(1) << 31) &&
           pp->s_az > 0.0f && pp->s_el > 0.0f && pp->r_max >= pp->r_min;
}

// The binning rule of a panorama for bin_pixel.
//
// Guard: the largest amount by which the rule's column or row coordinate and bin_pixel's can differ, in radians,
// with u = 2^-24 (one rounding, relative to the value; a ratio t in [0, 1] enters atan by at most half its relative
// error):
//   atan, the rule: the division u/2 (for a row also the root: u), the square 0.15 u, the unfused polynomial's
//     partial sums 1.92 u, its product with t u/2: 3.1 u (row 3.6 u);
//   atan, bin_pixel: the approximate reciprocal (2^-23, or 2^-22.9 for a reciprocal root) and its product 1.7 u, the
//     square 0.15 u, the fused polynomial 1.35 u, the product with t s 0.8 u: 4.0 u;
//   column: the rule rounds pi/2 - a (u), pi - a (2 u), pi - az (4 u) and the product with s_az (2 pi u);
//     bin_pixel rounds az[k] and the sum (2 pi u each): 25.9 u;
//   row: the rule rounds el_top - el and the product with s_el, bin_pixel el0 and the sum: 4 u of at most
//     |el_top| + pi/4;
//   row of a steep point: the rule rounds pi/2 - atan too (u); the ratio rho / z is a reciprocal root, a reciprocal
//     and two products (6.2 u, half of it in the angle: with the rest as above 5.4 u); the base with pi/2 is one
//     rounding more, 5 u of at most |el_top| + pi/2; and where the rule takes the other ratio (the two tests of 45
//     degrees may differ by a rounding) the polynomial's own error counts twice, 0.7 u;
//   column of a steep point: 3 pi/2 rounded (4 u) more than a column's.
// Together below 33 u = 2.0e-6 for a column, (7.6 + 4 (|el_top| + 0.79)) u for a row, and 37 u and (10.7 + 5 (|el_top| +
// 1.58)) u for a steep point's; a tenth more is taken.
// A panorama whose coordinates reach 2^20 pixels or whose guard passes a quarter of a pixel, and an unlimited
// range, take the rule for every point.
static inline upslam::BinRule make_bin_rule(const upslam_pano &pp) {
    upslam::BinRule b;
    b.pp = pp;
    // (sqrtf rounds to nearest, as the device's root does, and is monotonic: the limits are found by stepping)
    float lo = 0.0f;
    if (pp.r_min > 0.0f) {
        lo = pp.r_min * pp.r_min;
        if (lo > FLT_MAX) lo = FLT_MAX;
        while (lo > 0.0f && sqrtf(lo) >= pp.r_min) lo = nextafterf(lo, 0.0f);
        while (sqrtf(lo) < pp.r_min) lo = nextafterf(lo, INFINITY);
    }
    float hi = -1.0f;
    if (pp.r_max >= 0.0f) {
        hi = pp.r_max * pp.r_max;
        if (hi > FLT_MAX && pp.r_max <= FLT_MAX) hi = FLT_MAX;
        while (hi <= FLT_MAX && sqrtf(hi) <= pp.r_max) hi = nextafterf(hi, INFINITY);
        while (sqrtf(hi) > pp.r_max) hi = nextafterf(hi, 0.0f);
    }
    b.r2_min = lo;
    b.r2_max = hi;
    const double s_az = pp.s_az, s_el = pp.s_el, top = pp.el_top;
    b.el0 = (float)(top * s_el - 0.5);
    for (int k = 0; k < 5; ++k) b.az[k] = (float)(k * (double)upslam::kHalfPiF * s_az - 0.5);
    const double u = 1.0 / 16777216.0;
    const double g_c = 1.1 * 33.0 * u * s_az, g_r = 1.1 * (7.6 + 4.0 * (fabs(top) + 0.79)) * u * s_el;
    const double most = 1048576.0;
    const bool on = pp.rows < most && pp.cols < most && 6.4 * s_az < most && (fabs(top) + 1.6) * s_el < most &&
                    g_c < 0.25 && g_r < 0.25 && hi <= FLT_MAX;
    b.lim_c = on ? (float)(0.5 - g_c) : -1.0f;
    b.lim_r = on ? (float)(0.5 - g_r) : -1.0f;
    return b;
}

static inline bool upslam_aligned(const void *p, size_t a) { return ((uintptr_t)p % a) == 0; }

static inline bool upslam_icp_params_ok(const upslam_icp_params *ip) {
    return ip && ip->d_max > 0.0f && ip->max_iters >= 0 && ip->min_inliers >= 0 &&
           (ip->loss == UPSLAM_LOSS_L2 || (ip->loss == UPSLAM_LOSS_L1 && ip->loss_delta > 0.0f)) &&
           ip->coarse_iters >= 0 && (ip->coarse_iters == 0 || ip->d_max_fine > 0.0f);
}

// Multiprocessor count of the current device, cached per device ordinal.  Any host thread may call
// the library, so the cache is atomic (every writer stores the same value).
static inline int upslam_sm_count() {
    static std::atomic<int> cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
    int sms = cache[dev].load(std::memory_order_relaxed);
    if (sms == 0) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 152;
        cache[dev].store(sms, std::memory_order_relaxed);
    }
    return sms;
}

// Grid for a grid-stride loop over `work` items: enough CTAs to fill every SM
// several times over, never more than the work needs.
static inline int upslam_grid(int64_t work, int threads, int per_sm = 8) {
    const int64_t want = (work + threads - 1) / threads;
    const int64_t cap = (int64_t)upslam_sm_count() * per_sm;
    return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}
