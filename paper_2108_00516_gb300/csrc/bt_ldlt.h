// bt_ldlt.h -- solve of a symmetric positive-definite FP64 system H x = y by
// one CTA of 256 threads: by an FP32 inverse and corrections from the
// double-float residual, or, where the inverse declines (pivots too small or
// corrections that do not settle), in FP64 by the square-root-free Cholesky
// factorisation H = L D L^T with a one-column look-ahead (forward substitution
// L z = y carried along), D w = z, and a blocked back substitution L^T x = w.
// Used by the Gauss-Newton step of Sec. IV-D (bt_solve.cu) and by the learned
// warm start's relative-pose averaging (bt_warmstart.cu).
//
// On GB300 a dependent FP64 operation costs ~64 cycles or more and a warp-wide
// FP64 instruction holds its sub-partition's DP unit for ~64 cycles whatever
// the number of active lanes.  The inverse therefore runs on the FP32 pipes,
// and so do its corrections: there the system, the right-hand side and the
// solution are pairs of FP32 numbers h + l (double-float, 48 bits), the system
// scaled by powers of two to a diagonal in [1, 4) (exact, and it keeps every
// value inside the FP32 exponent range).  The factorisation is arranged for
// short dependency chains and for many lanes behind each FP64 instruction.
//
// Measured in the solve kernel (chains of correspondence sets, the diagonal
// scaled away; cycles of one solve, inverse against factorisation): n = 6:
// 7.6 k against 9.1 k, n = 18: 12.2 k against 16.1 k, n = 54: 25 k against 56 k,
// n = 114: 80 k against 233 k, n = 138: 138 k against 366 k.  Trying the inverse
// in vain costs 4.5 k, 22 k and about 90 k cycles at n = 6, 54 and 114.  One
// pivot a step of the inverse instead of six: 33 k at n = 54, 138 k at n = 114.
// Error of the solution against an 80-bit one, relative to its largest entry
// (worst of the systems of 6 .. 138 unknowns with condition numbers in the
// given range): where the inverse is taken, up to 1e3: 9e-13 (factorisation
// 2e-11), 1e3 .. 1e4: 1e-11 (4e-10), 1e4 .. 1e5: 1e-11 (4e-10); where it
// declines, 1e5 .. 9e5: 2e-8.  A factorisation in double-float numbers took
// half the cycles of the FP64 one, but left errors of up to 9e-6 there.
#pragma once

#include "bt_internal.h"

#include <cmath>
#include <cstring>

namespace bt {

// Double-float numbers (x: leading part, y: trailing part).  Every operation
// is written out: no contraction, no reassociation.
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float ff_add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float ff_sub_(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float ff_mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float ff_fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
inline float ff_add_(float a, float b) { return a + b; }
inline float ff_sub_(float a, float b) { return a - b; }
inline float ff_mul_(float a, float b) { return a * b; }
inline float ff_fma_(float a, float b, float c) { return std::fmaf(a, b, c); }
#endif

// h + l with |l| at most half a unit in the last place of h (|h| >= |l| given).
__host__ __device__ __forceinline__ float2 ff_norm(float h, float l)
{
    const float s = ff_add_(h, l);
    return make_float2(s, ff_sub_(l, ff_sub_(s, h)));
}

// c - a b, the trailing part not renormalised: the product's leading part is
// exact (multiply and fused remainder), the difference of the leading parts
// exact by Knuth's two-sum, the small terms in single precision.  12
// instructions.
__host__ __device__ __forceinline__ float2 ff_msub_acc(float2 c, float2 a, float2 b)
{
    const float p = ff_mul_(a.x, b.x);
    float e = ff_fma_(a.x, b.x, -p);
    e = ff_fma_(a.x, b.y, e);
    e = ff_fma_(a.y, b.x, e);
    const float s = ff_sub_(c.x, p);
    const float v = ff_sub_(s, c.x);
    const float w = ff_sub_(ff_sub_(c.x, ff_sub_(s, v)), ff_add_(p, v));
    return make_float2(s, ff_add_(w, ff_sub_(c.y, e)));
}

__host__ __device__ __forceinline__ float2 ff_add(float2 a, float2 b)
{
    const float s = ff_add_(a.x, b.x);
    const float v = ff_sub_(s, a.x);
    const float w = ff_add_(ff_sub_(a.x, ff_sub_(s, v)), ff_sub_(b.x, v));
    return ff_norm(s, ff_add_(w, ff_add_(a.y, b.y)));
}

// Exponent field of an FP64 number (0 for zero and subnormal numbers).
__host__ __device__ __forceinline__ int f64_exponent(double x)
{
#ifdef __CUDA_ARCH__
    return (__double2hiint(x) >> 20) & 0x7ff;
#else
    long long b;
    std::memcpy(&b, &x, 8);
    return (int)(b >> 52) & 0x7ff;
#endif
}

// x 2^k as a double-float, with integer and FP32 operations only (an FP64
// conversion would hold the DP unit): the top 24 bits of the significand,
// then the other 29 rounded to 24.  Results outside the FP32 range become 0
// or infinity.
__host__ __device__ __forceinline__ float2 ff_from_f64(double x, int k)
{
#ifdef __CUDA_ARCH__
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
#else
    unsigned long long b;
    std::memcpy(&b, &x, 8);
#endif
    const int f = (int)(b >> 52) & 0x7ff;
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    const int E = f - 1023 + k;
    unsigned hb = sign, lb = sign;
    if (f == 0x7ff || E > 127) {
        hb |= f == 0x7ff ? 0x7fc00000u : 0x7f800000u;
        lb = 0u;
    } else if (f == 0 || E < -126) {
        lb = 0u;
    } else {
        hb |= (unsigned)(E + 127) << 23 | ((unsigned)(b >> 29) & 0x7fffffu);
        lb = E < -74 ? 0u : lb | (unsigned)(E - 52 + 127) << 23;
    }
    float h, q;
#ifdef __CUDA_ARCH__
    h = __uint_as_float(hb);
    q = __uint_as_float(lb);
#else
    std::memcpy(&h, &hb, 4);
    std::memcpy(&q, &lb, 4);
#endif
    return ff_norm(h, ff_mul_((float)((unsigned)b & 0x1fffffffu), q));
}

// (h + l) 2^k in FP64 (exact unless the result is subnormal).
__host__ __device__ __forceinline__ double ff_to_f64(float2 v, int k)
{
    const double x = (double)v.x + (double)v.y;
#ifdef __CUDA_ARCH__
    if (k > -1000 && k < 1000) return x * __hiloint2double((k + 1023) << 20, 0);
#endif
    return ldexp(x, k);
}

// Largest system: 6 unknowns per free node.  The back substitution splits
// the rows above a block of 32 unknowns into min(4, 256 / r0) column chunks
// (256 threads), which needs r0 < n <= 256.
constexpr int kLdltMaxN = 6 * (kMaxNodes - 1);
static_assert(kLdltMaxN <= 256, "ldlt_solve: at most 256 unknowns for one 256-thread CTA");
// Unknowns eliminated between two barriers of the inverse: one node's.
constexpr int kPan = 6;

// Row groups of the inverse by size of the system: entries of a column in a
// thread's registers (a multiple of six) and groups, one warp a group and
// block of 32 columns.
struct InvShape {
    int rows, groups;
};
__host__ __device__ constexpr InvShape inv_shape(int n)
{
    return n <= 12 ? InvShape{6, 2} : n <= 30 ? InvShape{6, 5} : n <= 60 ? InvShape{18, 4} : n <= 96 ? InvShape{48, 2}
         : n <= 120 ? InvShape{60, 2} : InvShape{138, 1};
}
static_assert(kLdltMaxN <= 138, "the inverse holds the largest system");
__host__ __device__ constexpr int inv_stride(int kR) { return (kR + 3) & ~3; }      // of a row group, in floats
// Two panels of six columns and six rows, the solution, the right-hand side.
__host__ __device__ constexpr size_t inv_floats(int n)
{
    return 2 * kPan * (size_t)(inv_stride(inv_shape(n).rows) * inv_shape(n).groups + n) + 4 * (size_t)n;
}

// Shared-memory scratch of ldlt_solve for an n x n system.
struct LdltScratch {
    double* work;   // [ldlt_work_doubles(n)], 16-byte aligned: the inverse's panels and vectors; the factorisation's
                    // scaled look-ahead column, double-buffered [2][n], and (row, column) table of the trailing triangle
    double* rD;     // [n]      1 / D_k
    double* part;   // [256]    partial dot products
    int* shift;     // [n + 1]  power-of-two scaling of each row and of y
};
__host__ __device__ constexpr size_t ldlt_work_doubles(int n)
{
    const size_t inv = (inv_floats(n) + 1) / 2, fac = 2 * (size_t)n + ((size_t)n * (n + 1) / 2 + 1) / 2;
    return inv > fac ? inv : fac;
}
__host__ __device__ constexpr size_t ldlt_shift_doubles(size_t n) { return (n + 2) / 2; }

// H: n x n (n a multiple of 6, at most kLdltMaxN) in shared memory, row-major
// with leading dimension ld = n + 1, lower triangle filled; the rest of it is
// overwritten.  y: [n] right-hand side in shared memory, overwritten with x.
// *fail (shared memory, zero on entry) is set when a pivot is not positive; x
// is then meaningless, and the caller reads *fail after the call (the call
// ends with a barrier).  inverse: whether to try the inverse first (a system
// whose predecessor was declined will most often be declined too).  t_mid:
// every thread's clock after the inverse's solve, or after the factorisation
// and D w = z.  idle(warp): called once by each of warps 1-7 while warp 0
// alone runs the first block of the back substitution (work the caller has for
// otherwise idle warps; it must not touch H, y or the scratch, and is not
// called when a pivot failed).  Returns whether the system was factorised, and
// idle called for (false: solved by the inverse, without a time when warps are
// idle).  All threads of the CTA (blockDim.x == 256) must call it.
struct LdltNoIdle {
    __device__ void operator()(int) const {}
};

#ifdef __CUDACC__
// 1/d for a positive FP64 pivot: the hardware approximation (rcp.approx.f64,
// relative error below 1e-6 on GB300) refined by one Newton step
// r <- r + r (1 - d r), which leaves a relative error below 1e-12 (measured
// on 1M pivots spanning 1e-6 .. 1e6) -- ample for a factorisation whose
// results are compared at 1e-5, and two dependent FP64 operations shorter
// than the correctly rounded reciprocal on the column chain.
__device__ __forceinline__ double rcp_fp64(double d)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    const double e = fma(-d, r, 1.0);
    return fma(r, e, r);
}

// Trailing rows from which warp 4 joins the bulk update (see ldlt_solve).
#ifndef BT_LDLT_WIDE_ROWS
#define BT_LDLT_WIDE_ROWS 30
#endif
constexpr int kWideBulkRows = BT_LDLT_WIDE_ROWS;

// H x = b by the FP32 inverse W of the scaled system and corrections of x from
// its double-float residual, x += W (b - H x), until they settle (at most
// eight).  The normal equations of dense graphs in the object's frame have
// scaled condition numbers of 20 .. 60 (six graphs of 18 .. 138 unknowns;
// chains of correspondence sets reach 1e3): there W is good to about 1e-6 and
// two corrections reach the accuracy of the double-float residual, without the
// n dependent pivots of the factorisation below.  W is formed by Gauss-Jordan
// elimination in steps of six unknowns, one barrier a step: lane = column,
// warps = column blocks x kG row groups, kR entries of a column in a thread's
// registers (kR a multiple of six, so that a panel's rows lie in one group);
// the panel (six columns, six rows) of the next step goes through shared
// memory, and every thread factorises the 6 x 6 pivot block for itself.
// Returns false when a pivot is below 2^-10 (the diagonal is in [1, 4)), so
// that the system may not be positive definite, or when the corrections do not
// shrink by at least four each; the caller then factorises.
// F: upper triangle of the scaled system, leading dimension ld; buf: panels,
// 12 (inv_stride(kR) kG + n) floats (16-byte aligned); part: kG n; x: n.
template <int kR, int kG>
__device__ __forceinline__ bool inverse_solve(const float2* __restrict__ F, int ld, int n, const float2* __restrict__ b,
                                              float* __restrict__ buf, float2* __restrict__ part,
                                              float2* __restrict__ x)
{
    static_assert(kR % kPan == 0, "a panel's rows in one group");
    constexpr int kS = inv_stride(kR), kRows = kS * kG, kCol = kPan * kRows;      // floats of a column, of a column panel
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = (n + 31) >> 5, cb = warp % nb, g = warp / nb;
    const bool active = g < kG;
    const int j = cb * 32 + lane, jc = min(j, n - 1), i0 = g * kR;
    float* rows = buf + 2 * kCol;                            // [2][6][n]
    float w[kS];
    // publishes the panel of columns and rows c0 .. c0 + 5
    auto publish = [&](int c0, int par) {
        const int jp = j - c0;
        if ((unsigned)jp < (unsigned)kPan) {
            float4* c = reinterpret_cast<float4*>(buf + par * kCol + jp * kRows + g * kS);
#pragma unroll
            for (int r = 0; r < kS / 4; ++r) c[r] = make_float4(w[4 * r], w[4 * r + 1], w[4 * r + 2], w[4 * r + 3]);
        }
        float* to = rows + par * kPan * n + jc;
#pragma unroll
        for (int q = 0; q < kR / kPan; ++q)
            if (i0 + kPan * q == c0) {
#pragma unroll
                for (int e = 0; e < kPan; ++e)
                    if (j < n) to[e * n] = w[kPan * q + e];
            }
    };
    if (active) {
#pragma unroll
        for (int r = 0; r < kS; ++r) {
            const int i = i0 + r;
            w[r] = r < kR && i < n ? F[min(i, jc) * ld + max(i, jc)].x : 0.f;
        }
        publish(0, 0);
    }
    __syncthreads();
    bool ok = true;
    int par = 0;
    for (int c0 = 0; c0 < n; c0 += kPan, par ^= 1) {
        if (active) {
            const float* C = buf + par * kCol;
            const float* R = rows + par * kPan * n + jc;
            const float* Cd = C + c0 / kR * kS + c0 % kR;      // the panel's own rows
            float D[kPan][kPan], z[kPan], rinv[kPan];
#pragma unroll
            for (int q = 0; q < kPan; ++q)
#pragma unroll
                for (int p = q; p < kPan; ++p) D[p][q] = Cd[q * kRows + p];
            const int jp = j - c0;
            const bool in_panel = (unsigned)jp < (unsigned)kPan;
#pragma unroll
            for (int q = 0; q < kPan; ++q) {
                const float a = R[q * n];
                z[q] = in_panel ? (q == jp ? 1.f : 0.f) : a;
            }
            // D = L D' L^T in place (L below the diagonal), then D^-1 z
#pragma unroll
            for (int p = 0; p < kPan; ++p) {
                ok = ok && D[p][p] > 0.0009765625f;
                asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rinv[p]) : "f"(D[p][p]));
#pragma unroll
                for (int r = p + 1; r < kPan; ++r) {
                    const float l = D[r][p] * rinv[p];
#pragma unroll
                    for (int c = p + 1; c <= r; ++c) D[r][c] = fmaf(-l, D[c][p], D[r][c]);
                    z[r] = fmaf(-l, z[p], z[r]);
                }
            }
#pragma unroll
            for (int p = kPan - 1; p >= 0; --p) {
#pragma unroll
                for (int r = kPan - 1; r > p; --r) z[p] = fmaf(-D[r][p], z[r], z[p]);
                z[p] *= rinv[p];
            }
            // the panel's own columns become those of the inverse
            if (in_panel) {
#pragma unroll
                for (int r = 0; r < kS; ++r) w[r] = 0.f;
            }
#pragma unroll
            for (int q = 0; q < kPan; ++q) {
                const float2 zq = make_float2(-z[q], -z[q]);
                const float4* c = reinterpret_cast<const float4*>(C + q * kRows + g * kS);
#pragma unroll
                for (int r = 0; r < kS / 4; ++r) {
                    const float4 c4 = c[r];
                    const float2 lo = __ffma2_rn(make_float2(c4.x, c4.y), zq, make_float2(w[4 * r], w[4 * r + 1]));
                    const float2 hi = __ffma2_rn(make_float2(c4.z, c4.w), zq, make_float2(w[4 * r + 2], w[4 * r + 3]));
                    w[4 * r] = lo.x;
                    w[4 * r + 1] = lo.y;
                    w[4 * r + 2] = hi.x;
                    w[4 * r + 3] = hi.y;
                }
            }
            // and its own rows D^-1 times what they were
#pragma unroll
            for (int q = 0; q < kR / kPan; ++q)
                if (i0 + kPan * q == c0) {
#pragma unroll
                    for (int e = 0; e < kPan; ++e) w[kPan * q + e] = z[e];
                }
            if (c0 + kPan < n) publish(c0 + kPan, par ^ 1);
        }
        __syncthreads();
    }
    if (__syncthreads_or(!ok)) return false;
    float* v = buf;                      // FP32 right-hand side of a correction, zeros in the padding
    float* top = buf + kRows;            // [8] per-warp maxima of |x|, then [8] of |dx|
    float* pf = reinterpret_cast<float*>(part);
    const int vi = tid / kR * kS + tid % kR;      // place of entry tid among the row groups
    if (tid < kRows) v[tid] = 0.f;
    __syncthreads();
    if (tid < n) {
        v[vi] = b[tid].x;
        x[tid] = make_float2(0.f, 0.f);
    }
    __syncthreads();
    float before = INFINITY;
    for (int it = 0; it < 8; ++it) {
        if (active) {
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int r = 0; r < kS / 4; ++r) {
                const float4 v4 = *reinterpret_cast<const float4*>(v + g * kS + 4 * r);
                s0 = fmaf(w[4 * r], v4.x, s0);
                s1 = fmaf(w[4 * r + 1], v4.y, s1);
                s0 = fmaf(w[4 * r + 2], v4.z, s0);
                s1 = fmaf(w[4 * r + 3], v4.w, s1);
            }
            if (j < n) pf[g * n + j] = s0 + s1;
        }
        __syncthreads();
        float dx = 0.f, ax = 0.f;
        if (tid < n) {
#pragma unroll
            for (int q = 0; q < kG; ++q) dx += pf[q * n + tid];
            const float2 xn = ff_add(x[tid], make_float2(dx, 0.f));
            x[tid] = xn;
            ax = fabsf(xn.x);
            dx = fabsf(dx);
        }
        // maxima of the bit patterns: a NaN counts as large
        const unsigned mx = __reduce_max_sync(0xffffffffu, __float_as_uint(ax)),
                       md = __reduce_max_sync(0xffffffffu, __float_as_uint(dx));
        if (lane == 0) {
            top[warp] = __uint_as_float(mx);
            top[8 + warp] = __uint_as_float(md);
        }
        __syncthreads();
        unsigned ux = 0, ud = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            ux = max(ux, __float_as_uint(top[q]));
            ud = max(ud, __float_as_uint(top[8 + q]));
        }
        const float X = __uint_as_float(ux), step = __uint_as_float(ud);
        if (!(X < INFINITY) || !(step <= 0.25f * before)) return false;
        // the next correction would be about step^2 / before: below 2^-45 of x?
        if (step == 0.f || (it > 0 && step * (step / before) <= 2.8e-14f * X)) return true;
        before = step;
        if (active) {
            float2 s0 = g == 0 ? b[jc] : make_float2(0.f, 0.f), s1 = make_float2(0.f, 0.f);
            const int k1 = min(i0 + kR, n);
            // H_jk: row k of the upper triangle up to column j, row j after it
            int k = i0;
            for (; k + 1 < k1; k += 2) {
                s0 = ff_msub_acc(s0, F[min(k, jc) * ld + max(k, jc)], x[k]);
                s1 = ff_msub_acc(s1, F[min(k + 1, jc) * ld + max(k + 1, jc)], x[k + 1]);
            }
            if (k < k1) s0 = ff_msub_acc(s0, F[min(k, jc) * ld + max(k, jc)], x[k]);
            if (j < n) part[g * n + j] = ff_add(s0, s1);
        }
        __syncthreads();
        if (tid < n) {
            float2 s = part[tid];
#pragma unroll
            for (int q = 1; q < kG; ++q) s = ff_add(s, part[q * n + tid]);
            v[vi] = s.x + s.y;
        }
        __syncthreads();
    }
    return false;
}

template <typename Idle = LdltNoIdle>
__device__ __forceinline__ bool ldlt_solve(double* __restrict__ H, int ld, int n, double* __restrict__ y,
                                           const LdltScratch& sc, bool inverse, int* fail, unsigned long long& t_mid,
                                           const Idle& idle = Idle())
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x;
    if (inverse) {
        // the scaled system beside H: entry (i, j), i >= j, at F[j ld + i], the
        // places right of H's diagonal (H and y stay as they are for the
        // factorisation)
        float2* F = reinterpret_cast<float2*>(H) + 1;
        float* buf = reinterpret_cast<float*>(sc.work);
        float2* x = reinterpret_cast<float2*>(buf + inv_floats(n)) - 2 * n;
        float2* b = x + n;
        float2* p = reinterpret_cast<float2*>(sc.part);
        int* shift = sc.shift;
        // row i by 2^shift[i], so that the diagonal lies in [1, 4), and the
        // right-hand side so that its largest entry lies in [1, 2)
        bool bad = false;
        for (int i = tid; i < n; i += nt) {
            const double d = H[i * ld + i];
            const int f = f64_exponent(d);
            bad = bad || f == 0 || f == 0x7ff || __double2hiint(d) < 0;     // not positive, or not finite
            shift[i] = -((f - 1023) >> 1);
        }
        if (!__syncthreads_or(bad)) {
            for (int i = warp; i < n; i += nt >> 5) {
                // a row's parts together: the compiler keeps loads behind the stores
                // to the same memory
                constexpr int kParts = (kLdltMaxN + 31) / 32;
                double h[kParts];
                int e[kParts];
#pragma unroll
                for (int q = 0; q < kParts; ++q) {
                    const int j = min(lane + 32 * q, i);
                    h[q] = H[i * ld + j];
                    e[q] = shift[j];
                }
                const int si = shift[i];
#pragma unroll
                for (int q = 0; q < kParts; ++q) {
                    const int j = lane + 32 * q;
                    if (32 * q > i) break;
                    const float2 f = ff_from_f64(h[q], si + e[q]);
                    if (j <= i) F[j * ld + i] = f;
                }
            }
            if (warp == 7) {
                int e = -100000;
                for (int i = lane; i < n; i += 32) {
                    const int f = f64_exponent(y[i]);
                    if (f != 0 && f != 0x7ff) e = max(e, f - 1023 + shift[i]);
                }
#pragma unroll
                for (int off = 16; off >= 1; off >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
                e = e > -100000 ? -e : 0;
                if (lane == 0) shift[n] = e;
                for (int i = lane; i < n; i += 32) b[i] = ff_from_f64(y[i], shift[i] + e);
            }
            __syncthreads();
            const bool done = n <= 12    ? inverse_solve<6, 2>(F, ld, n, b, buf, p, x)
                              : n <= 30  ? inverse_solve<6, 5>(F, ld, n, b, buf, p, x)
                              : n <= 60  ? inverse_solve<18, 4>(F, ld, n, b, buf, p, x)
                              : n <= 96  ? inverse_solve<48, 2>(F, ld, n, b, buf, p, x)
                              : n <= 120 ? inverse_solve<60, 2>(F, ld, n, b, buf, p, x)
                                         : inverse_solve<138, 1>(F, ld, n, b, buf, p, x);
            if (done) {
                t_mid = clock64();
                for (int i = tid; i < n; i += nt) y[i] = ff_to_f64(x[i], shift[i] - shift[n]);
                __syncthreads();
                return false;
            }
        }
        __syncthreads();
    }
    double* rD = sc.rD;
    double* colb = sc.work;
    int* tab = reinterpret_cast<int*>(sc.work + 2 * n);
    // LDL^T with a one-column look-ahead, one barrier per column.  At step k
    // warp 0 prepares column k+1 -- its update by column k, the pivot
    // D_{k+1} and reciprocal, and the scaled l_{i,k+1} -- while warps
    // {1,2,3,5,6,7} (no FP64 pipe shared with warp 0) apply column k to the
    // trailing triangle of rows and columns >= k+2 and carry the forward
    // substitution.  The scaled column is double-buffered; L is stored
    // transposed in the upper triangle, L_ik at (k, i).  A failed pivot
    // (not positive) sets *fail and a zero reciprocal; the loop still runs
    // to the end (same bounds, finite or discarded values), which keeps a
    // shared-memory read and a branch off every column of the chain.
    for (int ip = tid; ip < n; ip += nt)
        for (int jp = 0; jp <= ip; ++jp) tab[ip * (ip + 1) / 2 + jp] = (ip << 16) | jp;
    if (warp == 0) {
        double r = 0.0;
        if (lane == 0) {
            const double d = H[0];
            if (!(d > 0.0)) *fail = 1; else r = rcp_fp64(d);
            rD[0] = r;
        }
        r = __shfl_sync(0xffffffffu, r, 0);
        for (int i = 1 + lane; i < n; i += 32) {
            const double l = H[i * ld] * r;
            colb[i] = l;
            H[i] = l;
        }
    }
    __syncthreads();
    // bulk warps: {1,2,3,5,6,7}, and also warp 4 while the trailing triangle
    // is large (the early columns, where the bulk update and not warp 0's
    // chain sets the pace; warp 4 shares warp 0's FP64 unit, which has slack
    // there)
    const int bt6 = (warp != 0 && warp != 4 && warp < 8) ? (warp < 4 ? warp - 1 : warp - 2) * 32 + lane : -1;
    const int bt7 = (warp != 0 && warp < 8) ? (warp - 1) * 32 + lane : -1;
    for (int k = 0; k < n - 1; ++k) {
        const double* ck = colb + (k & 1) * n;        // l_{i,k}
        double* cn = colb + ((k + 1) & 1) * n;        // l_{i,k+1}, written now
        const bool wide = n - k - 2 >= kWideBulkRows;
        const int nbulk = wide ? 7 * 32 : 6 * 32;
        const int bt = wide ? bt7 : bt6;
        const bool bulk = bt >= 0;
        if (warp == 0) {
            // column p = k + 1, rows i = p .. n-1 in slots of 32: u_i = H_ip -
            // l_ik H_pk (the pivot is u_p), then every lane forms 1 / u_p
            // itself (no divergent branch, no second broadcast) and scales
            const int p = k + 1;
            const double hpk = H[p * ld + k];         // unscaled H_{k+1,k}
            const int nq = (n - p + 31) >> 5;         // active slots (warp-uniform)
            constexpr int kRows = (kLdltMaxN + 31) / 32;
            double hv[kRows], cv[kRows], u[kRows];
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                if (q >= nq) break;
                const int i = p + lane + 32 * q;
                hv[q] = i < n ? H[i * ld + p] : 0.0;
                cv[q] = i < n ? ck[i] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                if (q >= nq) break;
                u[q] = hv[q] - cv[q] * hpk;
            }
            const double h = __shfl_sync(0xffffffffu, u[0], 0);
            // h > 0 as an integer test on the bits (positive, not NaN): no
            // FP64 compare on the chain
            const long long hb = __double_as_longlong(h);
            const bool ok = hb > 0ll && hb <= 0x7ff0000000000000ll;
            const double rp = ok ? rcp_fp64(h) : 0.0;
            if (lane == 0) {
                if (!ok) *fail = 1;
                H[p * ld + p] = h;
                rD[p] = rp;
            }
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                if (q >= nq) break;
                const int i = p + lane + 32 * q;
                if (i > p && i < n) {
                    const double l = u[q] * rp;
                    H[i * ld + p] = u[q];
                    cn[i] = l;
                    H[p * ld + i] = l;
                }
            }
        } else if (bulk) {
            const int m1 = n - k - 2, tri = m1 * (m1 + 1) / 2;
            const double zk = y[k];
            for (int i = k + 1 + bt; i < n; i += nbulk) y[i] -= ck[i] * zk;
            int t = bt;
            for (; t + nbulk < tri; t += 2 * nbulk) {
                const int e0 = tab[t], e1 = tab[t + nbulk];
                const int i0 = k + 2 + (e0 >> 16), j0 = k + 2 + (e0 & 0xffff);
                const int i1 = k + 2 + (e1 >> 16), j1 = k + 2 + (e1 & 0xffff);
                const double a0 = H[i0 * ld + j0], a1 = H[i1 * ld + j1];
                const double l0 = ck[i0], l1 = ck[i1];
                const double b0 = H[j0 * ld + k], b1 = H[j1 * ld + k];
                H[i0 * ld + j0] = a0 - l0 * b0;
                H[i1 * ld + j1] = a1 - l1 * b1;
            }
            for (; t < tri; t += nbulk) {
                const int e = tab[t];
                const int i = k + 2 + (e >> 16), j = k + 2 + (e & 0xffff);
                H[i * ld + j] -= ck[i] * H[j * ld + k];
            }
        }
        __syncthreads();
    }
    for (int i = tid; i < n; i += nt) y[i] *= rD[i];   // D w = z
    __syncthreads();
    t_mid = clock64();
    const bool failed = *fail != 0;
    // L^T x = w, unit diagonal (L_ki is stored at (i, k)), in blocks of 32
    // unknowns from the last block up.  Warp 0 runs the chain of one block
    // with the block's values in registers, lane l holding row r0 + l: x_k
    // is broadcast from its lane with a shuffle, and the FP64 instructions
    // issued do not grow with the size of the system.  The rows above the
    // block then take the
    // block's unknowns as dot products, split into column chunks over
    // several warps (partial sums in shared memory, added per row).
    double* part = sc.part;
    for (int r0 = ((n - 1) >> 5) << 5; r0 >= 0; r0 -= 32) {
        const int r1 = min(n, r0 + 32);
        if (warp == 0) {
            const int i = r0 + lane;
            double wv = i < r1 ? y[i] : 0.0;
            int k = r1 - 1;
            // two unknowns a step: x_k is final; every lane forms
            // x_{k-1} = w_{k-1} - L_{k,k-1} x_k itself from the broadcast
            // values (the same FMA its owner would apply), so the chain is
            // one shuffle and two FMAs deep per two unknowns; each row takes
            // x_k, then x_{k-1}, exactly as in the one-at-a-time order
            for (; k > r0 + 1; k -= 2) {
                const double hk = i < k ? H[i * ld + k] : 0.0;
                const double hk1 = i < k - 1 ? H[i * ld + k - 1] : 0.0;
                const double lk = H[(k - 1) * ld + k];        // L_{k,k-1}
                const double xk = __shfl_sync(0xffffffffu, wv, k - r0);
                const double wk1 = __shfl_sync(0xffffffffu, wv, k - 1 - r0);
                const double xk1 = fma(-lk, xk, wk1);
                if (i < k) wv = fma(-hk, xk, wv);
                if (i < k - 1) wv = fma(-hk1, xk1, wv);
            }
            if (k == r0 + 1) {
                const double hk = i < k ? H[i * ld + k] : 0.0;
                const double xk = __shfl_sync(0xffffffffu, wv, k - r0);
                if (i < k) wv = fma(-hk, xk, wv);
            }
            if (i < r1) y[i] = wv;
        } else if (r0 + 32 >= n && !failed) {
            idle(warp);
        }
        __syncthreads();
        if (r0 == 0) break;
        const int chunks = min(4, 256 / r0);      // r0 <= 128: at least 2
        if (tid < chunks * r0) {
            const int i = tid % r0, c = tid / r0;
            double s0 = 0.0, s1 = 0.0;
            int k = r0 + c;
            for (; k + chunks < r1; k += 2 * chunks) {
                s0 = fma(H[i * ld + k], y[k], s0);
                s1 = fma(H[i * ld + k + chunks], y[k + chunks], s1);
            }
            if (k < r1) s0 = fma(H[i * ld + k], y[k], s0);
            part[c * r0 + i] = s0 + s1;
        }
        __syncthreads();
        for (int i = tid; i < r0; i += nt) {
            double s = part[i];
            for (int c = 1; c < chunks; ++c) s += part[c * r0 + i];
            y[i] -= s;
        }
        __syncthreads();
    }
    return true;
}
#endif

}  // namespace bt
