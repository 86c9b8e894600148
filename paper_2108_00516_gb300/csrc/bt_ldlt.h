// bt_ldlt.h -- solve of a symmetric positive-definite FP64 system H x = y by
// one CTA of 256 threads: by an FP32 inverse and corrections from the
// double-float residual (up to 120 unknowns), or, for larger ones and where
// the corrections do not settle, by the square-root-free Cholesky
// factorisation H = L D L^T with a one-panel look-ahead (forward substitution
// L z = y carried along), D w = z, and a blocked back substitution L^T x = w.
// Used by the Gauss-Newton step of Sec. IV-D (bt_solve.cu) and by the learned
// warm start's relative-pose averaging (bt_warmstart.cu).
//
// Arithmetic: the system, the right-hand side and the solution are pairs of
// FP32 numbers h + l (double-float, 48 bits), on the FP32 pipes.  On GB300 a
// dependent FP64 operation costs ~64 cycles or more and a warp-wide FP64
// instruction holds its sub-partition's DP unit for ~64 cycles whatever the
// number of active lanes; a double-float multiply-subtract is 12 FP32
// instructions with a dependent chain of ~30 cycles.  The system is first
// scaled by powers of two to a diagonal in [1, 4) (exact, and it keeps every
// value inside the FP32 exponent range).
// Error of the solution against an 80-bit one, relative to its largest entry
// (60 Gauss-Newton systems, worst of each size): inverse and corrections
// 3e-14 .. 1.5e-13 for 18 .. 120 unknowns, factorisation up to 3.6e-13 there
// and 6e-13 at 138; an FP64 factorisation with pivots' reciprocals good to
// 1e-12: 7e-13 .. 2.5e-12.
// Measured in the solve kernel (cycles of one solve, inverse against
// factorisation with back substitution): n = 6: 8.0 k against 10.7 k, n = 18:
// 11.0 k against 16.5 k, n = 54: 24.4 k against 36.1 k, n = 114: 106 k against
// 136 k.  One pivot a step instead of six, without the redundant 6 x 6
// factorisations: 33 k at n = 54, 138 k at n = 114.
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

// a b, not renormalised.
__host__ __device__ __forceinline__ float2 ff_mul_acc(float2 a, float2 b)
{
    const float p = ff_mul_(a.x, b.x);
    float e = ff_fma_(a.x, b.x, -p);
    e = ff_fma_(a.x, b.y, e);
    return make_float2(p, ff_fma_(a.y, b.x, e));
}

__host__ __device__ __forceinline__ float2 ff_add(float2 a, float2 b)
{
    const float s = ff_add_(a.x, b.x);
    const float v = ff_sub_(s, a.x);
    const float w = ff_add_(ff_sub_(a.x, ff_sub_(s, v)), ff_sub_(b.x, v));
    return ff_norm(s, ff_add_(w, ff_add_(a.y, b.y)));
}

// 1 / d, not renormalised: the hardware approximation r0 (relative error
// below 2^-22) and its remainder e = 1 - d r0, as r0 (1 + e + e^2); relative
// error below 2^-44.  The leading part is ready as soon as r0 is.
__host__ __device__ __forceinline__ float2 ff_rcp(float2 d)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d.x));
#else
    const float r = 1.0f / d.x;
#endif
    float e = ff_fma_(-d.x, r, 1.0f);
    e = ff_fma_(-d.y, r, e);
    return make_float2(r, ff_mul_(r, ff_fma_(e, e, e)));
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
// Columns factorised between two barriers: one node's unknowns.
constexpr int kPan = 6;
// Rows below the panel's own six that one warp takes through a panel.
constexpr int kPanRows = 32 - kPan;
static_assert((kLdltMaxN + 1 - kPan + kPanRows - 1) / kPanRows <= 8, "a panel's rows fit the CTA's eight warps");

// Shared-memory scratch of ldlt_solve for an n x n system.
struct LdltScratch {
    double* pan;    // [ldlt_pan_doubles(n)]: columns u and l = u / D of a panel by row, double-buffered (16-byte aligned)
    int* shift;     // [2 ldlt_shift_doubles(n)]: power-of-two scaling of each row and of y, two work counters
    double* part;   // [256]    partial dot products of the back substitution
};
__host__ __device__ constexpr size_t ldlt_pan_doubles(size_t n) { return 4 * kPan * (n + 1); }
__host__ __device__ constexpr size_t ldlt_shift_doubles(size_t n) { return (n + 4) / 2; }

// H: n x n (n a multiple of 6, at most kLdltMaxN) FP64 in shared memory,
// row-major with leading dimension ld = n + 1, lower triangle filled;
// overwritten (H and the scratch hold double-floats during the call).  y =
// H + n ld: right-hand side, overwritten with x (FP64).  *fail (shared
// memory, zero on entry) is set when a pivot is not positive; x is then
// meaningless, and the caller reads *fail after the call (the call ends with
// a barrier).  t_mid: every thread's clock after the factorisation.
// idle(warp): called once by each of warps 1-7 while warp 0 alone runs the
// first block of the back substitution (work the caller has for otherwise
// idle warps; it must not touch H, y or the scratch, and is not called when
// a pivot failed).  Returns whether idle was called for (false: the system
// was solved by its FP32 inverse, without a time when warps are idle).  All
// threads of the CTA (blockDim.x == 256) must call it.
struct LdltNoIdle {
    __device__ void operator()(int) const {}
};

// Systems that are solved by their FP32 inverse: its entries stay in the
// threads' registers, and its panels have to fit the factorisation's.
constexpr int kInvMaxN = 120;

#ifdef __CUDACC__
// H x = b by the FP32 inverse W of the scaled system and corrections of x from
// its double-float residual, x += W (b - H x).  The scaled normal equations of
// a pose graph in the object's frame have condition numbers of 20 .. 60, so W
// is good to about 1e-6 and two corrections reach the accuracy of the
// double-float residual, without the n dependent double-float pivots of the
// factorisation below.  W is formed by Gauss-Jordan elimination in steps of
// six unknowns, one barrier a step: lane = column, warps = column blocks x kG
// row groups, kR entries of a column in a thread's registers (kR a multiple of
// six, so that a panel's rows lie in one group); the panel (six columns, six
// rows) of the next step goes through shared memory, and every thread
// factorises the 6 x 6 pivot block for itself.
// Returns false, F and b untouched, when a pivot is below 2^-10 (the diagonal
// is in [1, 4)), so that the system may not be positive definite, or when the
// corrections do not shrink by at least four each; the caller then factorises.
// F: lower triangle, leading dimension ld; buf: 12 (inv_stride(kR) kG + n)
// floats (16-byte aligned); part: kG n; x: n.
__host__ __device__ constexpr int inv_stride(int kR) { return (kR + 3) & ~3; }                 // of a row group, in floats
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
            w[r] = r < kR && i < n ? F[max(i, jc) * ld + min(i, jc)].x : 0.f;
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
            // H_jk: row j of the triangle up to the diagonal, column j below it
            int k = i0;
            for (; k + 1 < k1; k += 2) {
                s0 = ff_msub_acc(s0, F[max(k, jc) * ld + min(k, jc)], x[k]);
                s1 = ff_msub_acc(s1, F[max(k + 1, jc) * ld + min(k + 1, jc)], x[k + 1]);
            }
            if (k < k1) s0 = ff_msub_acc(s0, F[max(k, jc) * ld + min(k, jc)], x[k]);
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

// The six values of row i of a panel buffer.
__device__ __forceinline__ void pan_load(const float2* pan, int i, float2 (&v)[kPan])
{
    const float4* p = reinterpret_cast<const float4*>(pan + i * kPan);
#pragma unroll
    for (int q = 0; q < kPan / 2; ++q) {
        const float4 x = p[q];
        v[2 * q] = make_float2(x.x, x.y);
        v[2 * q + 1] = make_float2(x.z, x.w);
    }
}

__device__ __forceinline__ void pan_store(float2* pan, int i, const float2 (&v)[kPan])
{
    float4* p = reinterpret_cast<float4*>(pan + i * kPan);
#pragma unroll
    for (int q = 0; q < kPan / 2; ++q) p[q] = make_float4(v[2 * q].x, v[2 * q].y, v[2 * q + 1].x, v[2 * q + 1].y);
}

// Warp w's share of the panel of columns c0 .. c0 + 5: lanes 0-5 hold the
// panel's own rows (the same in every warp: the six pivots are formed by
// each warp for itself, which saves a barrier and a shared-memory round trip
// inside the panel), lanes 6-31 the rows c0 + 6 + 26 w onwards (row n is the
// right-hand side).  First the previous panel (pu, pl; NULL for the first) is
// applied to these six columns, then per column the pivot and the panel's
// other entries of its row come by shuffle and every lane forms 1 / D
// itself.  On the chain from pivot to pivot lie one shuffle, the reciprocal
// and two products; everything that renormalises runs beside it.  Written:
// u and l by row, L transposed into the upper triangle, w = z / D (the l of
// row n) over the finished entries of y.
__device__ __forceinline__ void ldlt_panel(float2* F, int ld, int n, int c0, int w, const float2* pu, const float2* pl,
                                           float2* wu, float2* wl, int* fail)
{
    const int lane = threadIdx.x & 31;
    const bool diag = lane < kPan;
    const int i = c0 + lane + (diag ? 0 : kPanRows * w);
    const int ic = min(i, n);
    float2 a[kPan], l[kPan];
#pragma unroll
    for (int c = 0; c < kPan; ++c) a[c] = lane >= c ? F[ic * ld + c0 + c] : make_float2(0.f, 0.f);
    if (pu) {
        pan_load(pl, ic, l);
#pragma unroll
        for (int c = 0; c < kPan; ++c) {
            float2 u[kPan];
            pan_load(pu, c0 + c, u);
#pragma unroll
            for (int q = 0; q < kPan; ++q) a[c] = ff_msub_acc(a[c], l[q], u[q]);
        }
    }
    bool ok = true;
#pragma unroll
    for (int p = 0; p < kPan; ++p) {
        float2 u[kPan];
#pragma unroll
        for (int c = p; c < kPan; ++c)
            u[c] = make_float2(__shfl_sync(0xffffffffu, a[p].x, c), __shfl_sync(0xffffffffu, a[p].y, c));
        a[p] = ff_norm(a[p].x, a[p].y);
        ok = ok && u[p].x > 0.f && u[p].x < INFINITY;
        const float2 r = ff_rcp(u[p]);
        l[p] = ff_mul_acc(a[p], r);
#pragma unroll
        for (int c = p + 1; c < kPan; ++c) a[c] = ff_msub_acc(a[c], l[p], ff_norm(u[c].x, u[c].y));
    }
    if (!ok && lane == 0) *fail = 1;
#pragma unroll
    for (int c = 0; c < kPan; ++c) l[c] = ff_norm(l[c].x, l[c].y);
    if (!diag && i <= n) {
        pan_store(wu, i, a);
        pan_store(wl, i, l);
    }
    if (i == n) {
#pragma unroll
        for (int c = 0; c < kPan; ++c) F[n * ld + c0 + c] = l[c];
    } else if (i < n && (!diag || w == 0)) {
#pragma unroll
        for (int c = 0; c < kPan; ++c)
            if (i > c0 + c) F[(c0 + c) * ld + i] = l[c];
    }
}

// Applies a panel (pu, pl) to the trailing columns c1 .. n - 1, rows down to
// n: tiles of 2 x 2 entries, 32 tiles a warp at a time from the counter, so
// that warps join when their part of the next panel is done.  12
// instructions a product leave the FP32 pipes the limit; a tile reads 16
// 16-byte words of shared memory for its 24 products (one entry a thread: 14
// for six, more than the shared memory delivers at that rate).
__device__ __forceinline__ void ldlt_trailing(float2* F, int ld, int n, int c1, const float2* pu, const float2* pl,
                                              int* counter)
{
    const int lane = threadIdx.x & 31;
    const int h = (n - c1) >> 1, tiles = h * (h + 3) / 2;      // column pairs; row pairs h + 1, the last with row n alone
    for (;;) {
        int t0 = 0;
        if (lane == 0) t0 = atomicAdd(counter, 32);
        t0 = __shfl_sync(0xffffffffu, t0, 0);
        if (t0 >= tiles) return;
        const int t = t0 + lane;
        if (t >= tiles) continue;
        // tiles numbered from the last column pair back: t = r (r + 3) / 2 + c
        // for column pair h - 1 - r and row pair h - c; r from the square
        // root, corrected by one step either way (t < 2^12)
        int r = (int)((sqrtf(8.0f * (float)t + 9.0f) - 3.0f) * 0.5f);
        if (r * (r + 3) / 2 > t) --r;
        if ((r + 1) * (r + 4) / 2 <= t) ++r;
        const int j = c1 + 2 * (h - 1 - r), i = c1 + 2 * (h - (t - r * (r + 3) / 2));
        const int i1 = min(i + 1, n);
        float2* f0 = F + i * ld + j;
        float2* f1 = F + i1 * ld + j;
        float2 v00 = f0[0], v01 = f0[1], v10 = f1[0], v11 = f1[1];
        const float4* u0 = reinterpret_cast<const float4*>(pu + j * kPan);
        const float4* l0 = reinterpret_cast<const float4*>(pl + i * kPan);
        const float4* l1 = reinterpret_cast<const float4*>(pl + i1 * kPan);
#pragma unroll
        for (int q = 0; q < kPan / 2; ++q) {
            const float4 ua = u0[q], ub = u0[q + kPan / 2], la = l0[q], lb = l1[q];
            v00 = ff_msub_acc(v00, make_float2(la.x, la.y), make_float2(ua.x, ua.y));
            v01 = ff_msub_acc(v01, make_float2(la.x, la.y), make_float2(ub.x, ub.y));
            v10 = ff_msub_acc(v10, make_float2(lb.x, lb.y), make_float2(ua.x, ua.y));
            v11 = ff_msub_acc(v11, make_float2(lb.x, lb.y), make_float2(ub.x, ub.y));
            v00 = ff_msub_acc(v00, make_float2(la.z, la.w), make_float2(ua.z, ua.w));
            v01 = ff_msub_acc(v01, make_float2(la.z, la.w), make_float2(ub.z, ub.w));
            v10 = ff_msub_acc(v10, make_float2(lb.z, lb.w), make_float2(ua.z, ua.w));
            v11 = ff_msub_acc(v11, make_float2(lb.z, lb.w), make_float2(ub.z, ub.w));
        }
        f0[0] = v00;
        if (i > j) f0[1] = v01;
        if (i < n) {
            f1[0] = v10;
            f1[1] = v11;
        }
    }
}

template <typename Idle = LdltNoIdle>
__device__ __forceinline__ bool ldlt_solve(double* __restrict__ H, int ld, int n, double* __restrict__ y,
                                           const LdltScratch& sc, int* fail, unsigned long long& t_mid,
                                           const Idle& idle = Idle())
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x;
    float2* F = reinterpret_cast<float2*>(H);
    float2* yf = reinterpret_cast<float2*>(y);     // row n of F
    float2* pan = reinterpret_cast<float2*>(sc.pan);
    const int pan_len = kPan * (n + 1);            // buffer b: u at pan + 2 b pan_len, l after it
    int* shift = sc.shift;
    // scaling: row i by 2^shift[i], so that the diagonal lies in [1, 4), and
    // the right-hand side so that its largest entry lies in [1, 2)
    for (int i = tid; i < n; i += nt) {
        const double d = H[i * ld + i];
        const int f = f64_exponent(d);
        if (f == 0 || f == 0x7ff || __double2hiint(d) < 0) *fail = 1;     // not positive (or not finite)
        shift[i] = -((f - 1023) >> 1);
    }
    __syncthreads();
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
            if (j <= i) F[i * ld + j] = f;
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
        for (int i = lane; i < n; i += 32) yf[i] = ff_from_f64(y[i], shift[i] + e);
    }
    __syncthreads();
    if (n <= kInvMaxN && *fail == 0) {
        float* buf = reinterpret_cast<float*>(pan);
        float2* p = reinterpret_cast<float2*>(sc.part);
        // rows (with padding) of the row groups, by size
        const int rows = n <= 12 ? inv_stride(6) * 2 : n <= 30 ? inv_stride(6) * 5 : n <= 60 ? inv_stride(18) * 4 : n <= 96 ? 48 * 2 : 60 * 2;
        float2* x = reinterpret_cast<float2*>(buf + 2 * kPan * (rows + n));
        const bool done = n <= 12   ? inverse_solve<6, 2>(F, ld, n, yf, buf, p, x)
                          : n <= 30 ? inverse_solve<6, 5>(F, ld, n, yf, buf, p, x)
                          : n <= 60 ? inverse_solve<18, 4>(F, ld, n, yf, buf, p, x)
                          : n <= 96 ? inverse_solve<48, 2>(F, ld, n, yf, buf, p, x)
                                    : inverse_solve<60, 2>(F, ld, n, yf, buf, p, x);
        if (done) {
            t_mid = clock64();
            for (int i = tid; i < n; i += nt) y[i] = ff_to_f64(x[i], shift[i] - shift[n]);
            __syncthreads();
            return false;
        }
        __syncthreads();
    }
    // LDL^T in panels of six columns (one node), the right-hand side carried
    // along as row n, one barrier a panel: the warps that hold the panel's
    // rows bring it up to date and factorise it -- the serial chain of the
    // solve -- while the others apply the panel before it to the rest of the
    // trailing triangle, where the first ones then join.  L is stored
    // transposed in the upper triangle, L_ik at (k, i).  A failed pivot sets
    // *fail; the loop still runs to the end (same bounds, discarded values).
    for (int c0 = 0; c0 < n; c0 += kPan) {
        const int b = (c0 / kPan) & 1;
        float2* wu = pan + 2 * b * pan_len;
        const float2* pu = pan + 2 * (b ^ 1) * pan_len;      // the panel before this one
        if (kPanRows * warp < n + 1 - kPan - c0)
            ldlt_panel(F, ld, n, c0, warp, c0 > 0 ? pu : nullptr, pu + pan_len, wu, wu + pan_len, fail);
        if (c0 > 0) ldlt_trailing(F, ld, n, c0 + kPan, pu, pu + pan_len, shift + n + 1 + b);
        if (tid == 0) shift[n + 1 + (b ^ 1)] = 0;            // the next panel's counter
        __syncthreads();
    }
    t_mid = clock64();
    const bool failed = *fail != 0;
    // L^T x = w, unit diagonal (L_ki is stored at (i, k)), in blocks of 32
    // unknowns from the last block up.  Warp 0 runs the chain of one block
    // with the block's values in registers, lane l holding row r0 + l: x_k
    // is broadcast from its lane with a shuffle.  The rows above the block
    // then take the block's unknowns as dot products, split into column
    // chunks over several warps (partial sums in shared memory, added per
    // row).
    float2* part = reinterpret_cast<float2*>(sc.part);
    for (int r0 = ((n - 1) >> 5) << 5; r0 >= 0; r0 -= 32) {
        const int r1 = min(n, r0 + 32);
        if (warp == 0) {
            const int i = r0 + lane;
            const float2 zero = make_float2(0.f, 0.f);
            float2 wv = i < r1 ? yf[i] : zero;
            // two unknowns a step: x_k is final; every lane forms
            // x_{k-1} = w_{k-1} - L_{k,k-1} x_k itself from the broadcast
            // values (the same operation its owner would apply), so the
            // chain is one shuffle and two multiply-subtracts deep per two
            // unknowns; the next step's values of L are read ahead.  (An odd
            // number of unknowns in the block starts one row past it, where
            // L and w are taken as zero.)
            const float2* row = F + min(i, n - 1) * ld + r0;
            int k = (r1 - r0 - 1) | 1;
            auto at = [&](int q) { return lane < q && r0 + q < r1 ? row[q] : zero; };
            float2 hk = at(k), hk1 = at(k - 1);
            for (; k > 0; k -= 2) {
                const float2 nk = at(k - 2), nk1 = at(k - 3);
                const float2 lk = make_float2(__shfl_sync(0xffffffffu, hk.x, k - 1), __shfl_sync(0xffffffffu, hk.y, k - 1));
                const float2 xk = make_float2(__shfl_sync(0xffffffffu, wv.x, k), __shfl_sync(0xffffffffu, wv.y, k));
                const float2 wk1 = make_float2(__shfl_sync(0xffffffffu, wv.x, k - 1),
                                               __shfl_sync(0xffffffffu, wv.y, k - 1));
                const float2 xk1 = ff_msub_acc(wk1, lk, xk);
                wv = ff_msub_acc(wv, hk, xk);
                wv = ff_msub_acc(wv, hk1, xk1);
                hk = nk;
                hk1 = nk1;
            }
            if (i < r1) yf[i] = ff_norm(wv.x, wv.y);
        } else if (r0 + 32 >= n && !failed) {
            idle(warp);
        }
        __syncthreads();
        if (r0 == 0) break;
        const int chunks = min(4, 256 / r0);      // r0 <= 128: at least 2
        if (tid < chunks * r0) {
            const int i = tid % r0, c = tid / r0;
            float2 s0 = make_float2(0.f, 0.f), s1 = s0;
            int k = r0 + c;
            for (; k + chunks < r1; k += 2 * chunks) {
                s0 = ff_msub_acc(s0, F[i * ld + k], yf[k]);
                s1 = ff_msub_acc(s1, F[i * ld + k + chunks], yf[k + chunks]);
            }
            if (k < r1) s0 = ff_msub_acc(s0, F[i * ld + k], yf[k]);
            part[c * r0 + i] = ff_add(s0, s1);
        }
        __syncthreads();
        for (int i = tid; i < r0; i += nt) {
            float2 s = part[i];
            for (int c = 1; c < chunks; ++c) s = ff_add(s, part[c * r0 + i]);
            yf[i] = ff_add(yf[i], s);
        }
        __syncthreads();
    }
    for (int i = tid; i < n; i += nt) {
        const float2 x = yf[i];
        y[i] = ff_to_f64(x, shift[i] - shift[n]);
    }
    __syncthreads();
    return true;
}
#endif

}  // namespace bt
