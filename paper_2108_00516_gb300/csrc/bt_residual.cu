// bt_residual.cu -- sm_103a kernels of the pose-graph hot path (BundleTrack,
// Sec. IV-D, Eq. 1-3): frame preparation and the residual pass.
//
//   prep_*          frame preparation: per-pixel target map (z, n) and the
//                   compacted list of valid masked source pixels (pi_D^-1).
//   residual_kernel one launch per Gauss-Newton iteration: CTAs [0, E) take
//                   one correspondence set each (Eq. 2), CTAs [E, E+T) stage
//                   one tile of source pixels in shared memory and loop over
//                   every target node (Eq. 3): association, gates,
//                   point-to-plane residual, Jacobian, Huber weight, and a
//                   deterministic reduction of the 21 + 6 unique J^T W J /
//                   J^T W r terms per (tile, target).
//
// The reduction into FP64 blocks, the solve and the update are in bt_solve.cu.
//
// Perturbations.  The library solves for right perturbations,
// T_i <- T_i exp(d_i) with d = (v, w).  This is a linear change of tangent
// coordinates (d_left = Ad_{T_i} d_right) of the left-perturbation system,
// so every Gauss-Newton iterate is the same pose as with left perturbations;
// it lets a dense pair (i -> j) contribute one block K' to (i,i), (j,j) and
// -K' to (i,j), (j,i).
//
// Association decision.  Keep / drop and the looked-up pixel are integers
// decided in single precision by the device functions of bt_assoc.cuh (fused
// multiply-adds, the hardware reciprocal, packed FP32x2 arithmetic).  Another
// single-precision evaluation -- or the exact one -- can differ from it only
// for pixels within rounding of a half-pixel edge, the image edge or a gate;
// bt_debug_associate exports the decisions so that they can be checked pixel
// by pixel.  Residual values, Jacobians and weights are FP32 as well.
#include "bt_internal.h"
#include "bt_assoc.cuh"

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

namespace bt {

// ---------------------------------------------------------------------------
// K0: frame preparation
// ---------------------------------------------------------------------------

// A warp takes kPixPerThread groups of 32 consecutive pixels, one pixel a
// lane, so that every load and store of a group is contiguous and a pixel's
// rank among the valid ones follows from ballots.
struct Pixel {
    float z;
    float3 n;
    bool ok;
};

// The pixel's mask, depth and normal, all loads issued together (gating the
// normal on the mask and the depth would make them a chain of three).
__device__ __forceinline__ Pixel load_pixel(const float* depth, const float* normals, const uint8_t* mask, int pix,
                                            int HW)
{
    Pixel x{0.f, make_float3(0.f, 0.f, 0.f), false};
    if (pix < HW) {
        const uint8_t m = __ldg(mask + pix);
        x.z = __ldg(depth + pix);
        const float* n = normals + 3 * (size_t)pix;
        x.n = make_float3(__ldg(n), __ldg(n + 1), __ldg(n + 2));
        x.ok = m != 0 && x.z > 0.f && isfinite(x.z) && isfinite(x.n.x) && isfinite(x.n.y) && isfinite(x.n.z);
    }
    return x;
}

// 16-bit storage helpers (BF16 / FP16 as raw bits)
template <int P>
__device__ __forceinline__ unsigned short to16(float x)
{
    if constexpr (P == 1) return __bfloat16_as_ushort(__float2bfloat16_rn(x));
    else return __half_as_ushort(__float2half_rn(x));
}
template <int P>
__device__ __forceinline__ float from16(unsigned short b)
{
    if constexpr (P == 1) return __bfloat162float(__ushort_as_bfloat16(b));
    else return __half2float(__ushort_as_half(b));
}
template <int P>
__device__ __forceinline__ unsigned short nan16()
{
    return P == 1 ? (unsigned short)0x7FC0 : (unsigned short)0x7E00;
}

size_t prep_scratch_bytes(int HW)
{
    const size_t nblk = (HW + kPrepPix - 1) / kPrepPix;
    return (nblk + 1) * (sizeof(int) + sizeof(double)) + 16;
}

// Count of valid pixels of each block of kPrepPix pixels and, for the 16-bit
// encodings (kSum), the sum of their depths.
template <bool kSum>
__global__ void __launch_bounds__(kThreads) prep_count_kernel(
    const float* __restrict__ depth, const float* __restrict__ normals,
    const uint8_t* __restrict__ mask, int HW, int* __restrict__ blockcnt, double* __restrict__ blocksum)
{
    __shared__ int sc[kThreads / 32];
    __shared__ double sz[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int base = blockIdx.x * kPrepPix + warp * (32 * kPixPerThread) + lane;
    Pixel px[kPixPerThread];
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k) px[k] = load_pixel(depth, normals, mask, base + 32 * k, HW);
    int c = 0;
    double dz = 0.0;
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k) {
        c += __popc(__ballot_sync(0xffffffffu, px[k].ok));
        if constexpr (kSum) {      // four neighbours in FP32, then FP64
            const float z = px[k].ok ? px[k].z : 0.f;
            float q = z + __shfl_down_sync(0xffffffffu, z, 1);
            q += __shfl_down_sync(0xffffffffu, z, 2);
            q += __shfl_down_sync(0xffffffffu, z, 3);
            if ((lane & 3) == 0) dz += (double)q;
        }
    }
    if constexpr (kSum) {
#pragma unroll
        for (int o = 16; o >= 4; o >>= 1) dz += __shfl_xor_sync(0xffffffffu, dz, o);
    }
    if (lane == 0) {
        sc[warp] = c;
        sz[warp] = dz;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int total = 0;
        double t = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) {
            total += sc[w];
            t += sz[w];
        }
        blockcnt[blockIdx.x] = total;
        if constexpr (kSum) blocksum[blockIdx.x] = t;
    }
}

// Target map of every pixel and the compacted source list of the valid ones.
// A CTA takes a run of consecutive blocks.  It adds up the counts of all
// blocks before its own for itself (a scan kernel between the two would be
// one more launch; the serial one this replaced took 28 us of a VGA frame's
// 42); the last CTA writes the valid count M, and every CTA of a 16-bit
// encoding forms the reference depth, the mean valid depth.
template <int P>
__global__ void __launch_bounds__(kThreads) prep_write_kernel(
    const float* __restrict__ depth, const float* __restrict__ normals,
    const uint8_t* __restrict__ mask, int W, int HW, float cx, float cy, float ifx, float ify,
    const int* __restrict__ blockcnt, const double* __restrict__ blocksum, int nblk, int* __restrict__ out2,
    int* __restrict__ host_out2, void* __restrict__ tgt_v, void* __restrict__ src_p_v, void* __restrict__ src_n_v)
{
    constexpr int kWarps = kThreads / 32;
    __shared__ int sc[2][kWarps], sw[kWarps];
    __shared__ double sz[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b0 = (int)((long long)blockIdx.x * nblk / gridDim.x), b1 = (int)((long long)(blockIdx.x + 1) * nblk / gridDim.x);
    int before = 0, all = 0;
    double z = 0.0;
    for (int b = tid; b < nblk; b += kThreads) {
        const int c = __ldg(blockcnt + b);
        all += c;
        before += b < b0 ? c : 0;
        if constexpr (P != 0) z += __ldg(blocksum + b);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        before += __shfl_xor_sync(0xffffffffu, before, o);
        all += __shfl_xor_sync(0xffffffffu, all, o);
        if constexpr (P != 0) z += __shfl_xor_sync(0xffffffffu, z, o);
    }
    if (lane == 0) {
        sc[0][warp] = before;
        sc[1][warp] = all;
        sz[warp] = z;
    }
    __syncthreads();
    int off = 0, M = 0;
    z = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        off += sc[0][w];
        M += sc[1][w];
        if constexpr (P != 0) z += sz[w];
    }
    const float zref = P == 0 || M == 0 ? 0.f : (float)(z / M);
    if (blockIdx.x == gridDim.x - 1 && tid == 0) {
        out2[0] = M;
        out2[1] = __float_as_int(zref);
        if (host_out2) {      // the host's read-back slot (mapped pinned memory)
            host_out2[0] = M;
            host_out2[1] = __float_as_int(zref);
        }
    }
    for (int b = b0; b < b1; ++b) {
        const int base = b * kPrepPix + warp * (32 * kPixPerThread) + lane;
        Pixel px[kPixPerThread];
#pragma unroll
        for (int k = 0; k < kPixPerThread; ++k) px[k] = load_pixel(depth, normals, mask, base + 32 * k, HW);
        unsigned bits[kPixPerThread];
        int c = 0;
#pragma unroll
        for (int k = 0; k < kPixPerThread; ++k) {
            bits[k] = __ballot_sync(0xffffffffu, px[k].ok);
            c += __popc(bits[k]);
        }
        if (lane == 0) sw[warp] = c;
        __syncthreads();
        int at = off;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const int cw = sw[w];
            at += w < warp ? cw : 0;
            off += cw;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kPixPerThread; ++k) {
            const int pix = base + 32 * k;
            const bool ok = px[k].ok;
            const float zz = px[k].z;
            const float3 nn = px[k].n;
            if (pix < HW) {
                // NaN depth where the pixel cannot be a target: no distance gate accepts it
                if constexpr (P == 0) {
                    reinterpret_cast<float4*>(tgt_v)[pix] =
                        ok ? make_float4(zz, nn.x, nn.y, nn.z) : make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
                } else {
                    // nor can one much nearer than the mean depth whose offset
                    // comes back (decode_target) as a depth that is not positive
                    ushort4 t;
                    const unsigned short dz = to16<P>(zz - zref);
                    t.x = ok && zref + from16<P>(dz) > 0.f ? dz : nan16<P>();
                    t.y = ok ? to16<P>(nn.x) : (unsigned short)0;
                    t.z = ok ? to16<P>(nn.y) : (unsigned short)0;
                    t.w = ok ? to16<P>(nn.z) : (unsigned short)0;
                    reinterpret_cast<ushort4*>(tgt_v)[pix] = t;
                }
            }
            if (ok) {
                const int o = at + __popc(bits[k] & ((1u << lane) - 1u));
                const int u = pix % W, v = pix / W;
                // pi_D^-1(x): (u - cx) z / fx, (v - cy) z / fy, z
                const float px_ = ((float)u - cx) * zz * ifx;
                const float py_ = ((float)v - cy) * zz * ify;
                if constexpr (P == 0) {
                    reinterpret_cast<float4*>(src_p_v)[o] = make_float4(px_, py_, zz, 0.f);
                    reinterpret_cast<float4*>(src_n_v)[o] = make_float4(nn.x, nn.y, nn.z, 0.f);
                } else {
                    reinterpret_cast<ushort4*>(src_p_v)[o] =
                        make_ushort4(to16<P>(px_), to16<P>(py_), to16<P>(zz - zref), 0);
                    reinterpret_cast<ushort4*>(src_n_v)[o] =
                        make_ushort4(to16<P>(nn.x), to16<P>(nn.y), to16<P>(nn.z), 0);
                }
            }
            at += __popc(bits[k]);
        }
    }
}

template <int P>
static void launch_prep_p(const float* depth, const float* normals, const uint8_t* mask, int W, int HW, float cx, float cy,
                          float ifx, float ify, void* tgt, void* src_p, void* src_n, int* blockcnt, double* blocksum,
                          int nblk, int* out2, int* host_out2, cudaStream_t s)
{
    // at most eight CTAs an SM: each reads every block's count once
    constexpr int kMaxCtas = 8 * 152;
    prep_count_kernel<P != 0><<<nblk, kThreads, 0, s>>>(depth, normals, mask, HW, blockcnt, blocksum);
    prep_write_kernel<P><<<std::min(nblk, kMaxCtas), kThreads, 0, s>>>(depth, normals, mask, W, HW, cx, cy, ifx, ify,
                                                                       blockcnt, blocksum, nblk, out2, host_out2, tgt,
                                                                       src_p, src_n);
}

cudaError_t launch_prep(const float* depth, const float* normals, const uint8_t* mask, int W, int H, float cx,
                        float cy, float ifx, float ify, int precision, void* tgt, void* src_p, void* src_n,
                        void* block_scratch, int* out2, int* host_out2, cudaStream_t s)
{
    const int HW = W * H;
    const int nblk = (HW + kPrepPix - 1) / kPrepPix;
    int* blockcnt = static_cast<int*>(block_scratch);
    double* blocksum = reinterpret_cast<double*>(
        (reinterpret_cast<uintptr_t>(blockcnt + nblk + 1) + 15) & ~static_cast<uintptr_t>(15));
    auto run = precision == 1 ? launch_prep_p<1> : precision == 2 ? launch_prep_p<2> : launch_prep_p<0>;
    run(depth, normals, mask, W, HW, cx, cy, ifx, ify, tgt, src_p, src_n, blockcnt, blocksum, nblk, out2, host_out2, s);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Residual pass
// ---------------------------------------------------------------------------

// Per-target constants of a tile, staged in shared memory by the CTA.
struct PairConst {
    PairK k;
    const void* tgt;
    float zref;                          // target frame's reference depth (16-bit maps)
};

__device__ __forceinline__ void fill_pair_const(const SolveArgs& a, int i, int j, const NodeDev& Nj, PairConst& c)
{
    float m[12];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float4 v = *(reinterpret_cast<const float4*>(a.xf + (size_t)(i * a.N + j) * 12) + q);
        m[4 * q] = v.x;
        m[4 * q + 1] = v.y;
        m[4 * q + 2] = v.z;
        m[4 * q + 3] = v.w;
    }
    c.k = make_pair_k(m, Nj.fx, Nj.fy, Nj.cx, Nj.cy, Nj.ifx, Nj.ify, Nj.W, Nj.H);
    c.tgt = Nj.tgt;
    c.zref = Nj.zref;
}

// One entry of a target map as it is stored (z, nx, ny, nz), and its decoding
// to FP32.  The gather is predicated: where `ok` is false the depth is NaN,
// which no distance gate accepts, and the other values are whatever they were.
template <int P>
struct Texel {
    float4 v;
};
template <>
struct Texel<1> {
    uint2 v;
};
template <>
struct Texel<2> {
    uint2 v;
};

template <int P>
__device__ __forceinline__ void gather_target(Texel<P>& t, const void* tgt, int idx, bool ok)
{
    if constexpr (P == 0) {
        t.v.x = __int_as_float(0x7fc00000);
        if (ok) t.v = __ldg(reinterpret_cast<const float4*>(tgt) + idx);
    } else {
        t.v.x = nan16<P>();
        if (ok) t.v = __ldg(reinterpret_cast<const uint2*>(tgt) + idx);
    }
}

template <int P>
__device__ __forceinline__ float4 decode_target(const Texel<P>& t, float zref)
{
    if constexpr (P == 0) {
        return t.v;
    } else {
        return make_float4(zref + from16<P>((unsigned short)(t.v.x & 0xffffu)), from16<P>((unsigned short)(t.v.x >> 16)),
                           from16<P>((unsigned short)(t.v.y & 0xffffu)), from16<P>((unsigned short)(t.v.y >> 16)));
    }
}

template <int P>
__device__ __forceinline__ void load_source(const NodeDev& Ni, int idx, float4& p, float4& n)
{
    if constexpr (P == 0) {
        p = __ldg(reinterpret_cast<const float4*>(Ni.src_p) + idx);
        n = __ldg(reinterpret_cast<const float4*>(Ni.src_n) + idx);
    } else {
        const ushort4 a = __ldg(reinterpret_cast<const ushort4*>(Ni.src_p) + idx);
        const ushort4 b = __ldg(reinterpret_cast<const ushort4*>(Ni.src_n) + idx);
        p = make_float4(from16<P>(a.x), from16<P>(a.y), Ni.zref + from16<P>(a.z), 0.f);
        n = make_float4(from16<P>(b.x), from16<P>(b.y), from16<P>(b.z), 0.f);
    }
}

// Warp reduce-scatter of 32 values: afterwards lane l holds the warp total of
// value l (recursive halving, 31 shuffles instead of 5 x 32).
__device__ __forceinline__ float warp_transpose_reduce(float (&v)[kDenseVals], int lane)
{
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
        const bool upper = (lane & step) != 0;
#pragma unroll
        for (int k = 0; k < step; ++k) {
            const float send = upper ? v[k] : v[k + step];
            const float keep = upper ? v[k + step] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, step);
        }
    }
    return v[0];
}

size_t residual_smem_bytes(int N, int shape)
{
    const int nt = N > 1 ? N - 1 : 1;
    return 2 * sizeof(float4) * shape_tile(shape) + sizeof(PairConst) * kMaxNodes +
           sizeof(float) * (size_t)nt * (kShapeThreads[shape] / 32) * kDenseVals;
}

// The 21 + 6 + 2 sums of a lane as register pairs: entries of J J^T that a
// packed FP32x2 instruction forms from pairs of J and their swapped copies,
// (J0, J1) (J2, J3) (J4, J5), without a broadcast per entry.
struct Sums {
    float2 p[13];               // (00,11) (02,13) (03,12) (04,15) (05,14) (22,33) (24,35) (25,34) (44,55) g01 g23 g45 (rho, 1)
    float s01, s23, s45;
};

__device__ __forceinline__ void accumulate_pair(Sums& a, float2 J01, float2 J23, float2 J45, float w, float r, float rho)
{
    const float2 ww = make_float2(w, w), rr = make_float2(r, r);
    const float2 J32 = make_float2(J23.y, J23.x), J54 = make_float2(J45.y, J45.x);
    const float2 w01 = __fmul2_rn(J01, ww), w23 = __fmul2_rn(J23, ww), w45 = __fmul2_rn(J45, ww);
    a.p[0] = __ffma2_rn(w01, J01, a.p[0]);
    a.p[1] = __ffma2_rn(w01, J23, a.p[1]);
    a.p[2] = __ffma2_rn(w01, J32, a.p[2]);
    a.p[3] = __ffma2_rn(w01, J45, a.p[3]);
    a.p[4] = __ffma2_rn(w01, J54, a.p[4]);
    a.p[5] = __ffma2_rn(w23, J23, a.p[5]);
    a.p[6] = __ffma2_rn(w23, J45, a.p[6]);
    a.p[7] = __ffma2_rn(w23, J54, a.p[7]);
    a.p[8] = __ffma2_rn(w45, J45, a.p[8]);
    a.p[9] = __ffma2_rn(w01, rr, a.p[9]);
    a.p[10] = __ffma2_rn(w23, rr, a.p[10]);
    a.p[11] = __ffma2_rn(w45, rr, a.p[11]);
    a.p[12] = __fadd2_rn(a.p[12], make_float2(rho, 1.f));
    a.s01 = fmaf(w01.x, J01.y, a.s01);
    a.s23 = fmaf(w23.x, J23.y, a.s23);
    a.s45 = fmaf(w45.x, J45.y, a.s45);
}

// The sums in the order of dpart: the upper triangle row-major ((0,b) = b,
// (1,b) = 5 + b, (2,b) = 9 + b, (3,b) = 12 + b, (4,b) = 14 + b, (5,5) = 20),
// [21..26] gradient, [27] cost, [28] count.
__device__ __forceinline__ void ordered_sums(const Sums& a, float (&v)[kDenseVals])
{
    v[0] = a.p[0].x;   v[6] = a.p[0].y;
    v[2] = a.p[1].x;   v[8] = a.p[1].y;
    v[3] = a.p[2].x;   v[7] = a.p[2].y;
    v[4] = a.p[3].x;   v[10] = a.p[3].y;
    v[5] = a.p[4].x;   v[9] = a.p[4].y;
    v[11] = a.p[5].x;  v[15] = a.p[5].y;
    v[13] = a.p[6].x;  v[17] = a.p[6].y;
    v[14] = a.p[7].x;  v[16] = a.p[7].y;
    v[18] = a.p[8].x;  v[20] = a.p[8].y;
    v[21] = a.p[9].x;  v[22] = a.p[9].y;
    v[23] = a.p[10].x; v[24] = a.p[10].y;
    v[25] = a.p[11].x; v[26] = a.p[11].y;
    v[27] = a.p[12].x; v[28] = a.p[12].y;
    v[1] = a.s01;
    v[12] = a.s23;
    v[19] = a.s45;
    v[29] = v[30] = v[31] = 0.f;
}

// Pixels per lane and step, and resident threads per SM the residual kernels
// are compiled for.  The full pass keeps two steps in flight and 29 sums a
// lane (128 registers, 16 warps a SM); the cost-only pass keeps two sums, so
// it hides its gathers with four pixels a step and 24 warps instead.
// Measured on 20 VGA views (44.4 M pixel pairs; full / cost pass, cold): one
// step at a time, a branch per gate and 24 warps 273 / 176 us; this form
// 216 / 161 us, 108 instead of 141 instructions a pixel pair.  Two steps in
// flight at 20 and 24 warps (96 and 80 registers: spills) gain nothing
// (217 us) or lose (300 us); nor does a tile divided over two CTAs (245 us:
// its sources are staged twice).
constexpr int step_pix(bool full) { return full ? 2 : 4; }
constexpr bool residual_pipelined(bool full) { return full; }
constexpr int residual_threads_per_sm(bool full) { return full ? 512 : 768; }

// One step of a warp in flight: its lanes' pixels after projection, with
// their target gathers issued.
template <int P, int kN>
struct Step {
    Texel<P> t[kN];
    float2 qxy[kN], uv[kN];
    float qz[kN];
};

// One tile of kT x kB source pixels of node i against every other node j.
// The work of the tile is (N-1) x kW units -- unit (jj, c) = target jj, chunk
// c of 32 x kB consecutive tile pixels -- in target-major order, and warp w
// takes the N-1 consecutive units [w (N-1), (w+1) (N-1)), of which it runs
// those whose chunk holds valid pixels.  A warp keeps its 21 + 6 + 2 sums in
// registers while its units stay on one target and reduces them across its
// lanes (a 31-shuffle reduce-scatter) only when the target changes: about
// (N-1)/kW + 1 reductions per warp instead of N-1.  A unit is taken in steps
// of kN pixels a lane, software-pipelined: the next step's pixels are
// projected and their target gathers issued (also across a change of target)
// before the current step's gathers are used, so that a gather's latency
// passes behind the gates, Jacobians and sums of a step.  The warp totals are
// parked in shared memory; one barrier at the end, then the (N-1) x 32 block
// sums of the tile are written to dpart[tile][jj] (each the sum, in warp
// order, of the warps that covered that target).
template <bool kFull, int kT, int kB, int P>
__device__ void dense_tile(const SolveArgs& a, int tile, unsigned char* dsm)
{
    constexpr int kW = kT / 32;
    constexpr int kTile = kT * kB;
    constexpr int kUnit = 32 * kB;
    constexpr int kMaxN = residual_pipelined(kFull) ? kB / 2 : kB;      // pipelined: at least two steps a unit
    constexpr int kN = kMaxN < step_pix(kFull) ? kMaxN : step_pix(kFull);
    constexpr int kSteps = kB / kN;
    static_assert(kSteps * kN == kB, "a unit is a whole number of steps");
    const int N = a.N, M1 = N - 1;
    const int i = a.tile_node[tile];
    const NodeDev& Ni = a.nodes[i];
    const int base = (tile - Ni.tile0) * kTile;
    const int nvalid = min(kTile, Ni.M - base);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float4* sp = reinterpret_cast<float4*>(dsm);
    float4* sn = sp + kTile;
    PairConst* pc = reinterpret_cast<PairConst*>(sn + kTile);      // by jj
    float* red = reinterpret_cast<float*>(pc + kMaxNodes);         // [N-1][kW][32]
    const float nan = __int_as_float(0x7fc00000);
    for (int s = threadIdx.x; s < kTile; s += kT) {
        // past the last valid pixel: NaN, which projects into no image
        float4 pp = make_float4(nan, nan, nan, 0.f), nn = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s < nvalid) load_source<P>(Ni, base + s, pp, nn);
        sp[s] = pp;
        sn[s] = nn;
    }
    const int my_j = (int)threadIdx.x < i ? threadIdx.x : threadIdx.x + 1;
    NodeDev Nj;
    if ((int)threadIdx.x < M1) Nj = a.nodes[my_j];
    // the source tile and the nodes are data of before the solve; the
    // transforms below were written by the predecessor (the previous update),
    // so the wait goes here
    pdl_wait_and_release();
    if ((int)threadIdx.x < M1) fill_pair_const(a, i, my_j, Nj, pc[threadIdx.x]);
    __syncthreads();
    const float dmax2 = a.dmax2, cmin = a.cmin, hub = a.huber_dense;
    const int nC = (nvalid + kUnit - 1) / kUnit;      // chunks with valid pixels
    const int u_end = (warp + 1) * M1;
    static_assert((kW & (kW - 1)) == 0, "warps of a CTA: a power of two");
    // the next unit of the warp's range whose chunk holds valid pixels
    auto valid_from = [&](int u) { return (u & (kW - 1)) < nC ? u : (u | (kW - 1)) + 1; };
    Sums acc;
    auto clear = [&]() {
#pragma unroll
        for (int k = 0; k < 13; ++k) acc.p[k] = make_float2(0.f, 0.f);
        acc.s01 = acc.s23 = acc.s45 = 0.f;
    };
    clear();
    // step `sub` of unit u: projection of its pixels, gathers issued
    auto issue = [&](Step<P, kN>& x, int u, int sub) {
        const PairConst& C = pc[u / kW];
        const PairK& K = C.k;
        const int s0 = (u & (kW - 1)) * kUnit + sub * (32 * kN) + lane;
#pragma unroll
        for (int k = 0; k < kN; ++k) {
            const int s = s0 + k * 32;
            const float4 p = sp[BT_CHECK_IDX(s < kTile, kChkSourceTile, a.ctrl) ? s : 0];
            int iu, iv;
            bool ok = assoc_project(K, p.x, p.y, p.z, x.qxy[k], x.qz[k], x.uv[k], iu, iv);
            ok = ok && BT_CHECK_IDX((unsigned)iu < (unsigned)K.W && (unsigned)iv < (unsigned)K.H, kChkGather, a.ctrl);
            gather_target<P>(x.t[k], C.tgt, iv * K.W + iu, ok);
        }
    };
    // the gates, residuals, Jacobians and sums of that step
    auto use = [&](const Step<P, kN>& x, int u, int sub) {
        const PairConst& C = pc[u / kW];
        const PairK& K = C.k;
        const float zref = P == 0 ? 0.f : C.zref;
        const float4* nn = sn + (u & (kW - 1)) * kUnit + sub * (32 * kN) + lane;
        // the gates of all the step's pixels side by side, without branches:
        // they are one dependent chain a pixel
        bool in[kN];
        float2 txy[kN], nxy[kN];
        float tz[kN], nz[kN], r[kN];
#pragma unroll
        for (int k = 0; k < kN; ++k) {
            const float4 t = decode_target<P>(x.t[k], zref);
            const float4 n = nn[k * 32];
            float2 dxy;
            float dz;
            tz[k] = t.x;
            in[k] = assoc_distance(K, x.uv[k], t.x, x.qxy[k], x.qz[k], dmax2, txy[k], dxy, dz) &
                    assoc_normal(K, n.x, n.y, n.z, t.y, t.z, t.w, cmin, nxy[k], nz[k]);
            // r = n' . (t - q), the point-to-plane distance of Eq. 3 expressed in camera j
            r[k] = assoc_residual(nxy[k], nz[k], dxy, dz);
        }
#pragma unroll
        for (int k = 0; k < kN; ++k) {
            if (!in[k]) continue;
            const float ar = fabsf(r[k]);
            const float m = fminf(ar, hub);
            const float rho = m * fmaf(-0.5f, m, ar);
            if constexpr (kFull) {
                const float w = ar <= hub ? 1.f : hub * rcp_approx(ar);
                const float2 J23 = make_float2(nz[k], fmaf(txy[k].y, nz[k], -tz[k] * nxy[k].y));
                const float2 J45 =
                    make_float2(fmaf(tz[k], nxy[k].x, -txy[k].x * nz[k]), fmaf(txy[k].x, nxy[k].y, -txy[k].y * nxy[k].x));
                accumulate_pair(acc, nxy[k], J23, J45, w, r[k], rho);
            } else {
                acc.p[12] = __fadd2_rn(acc.p[12], make_float2(rho, 1.f));
            }
        }
    };
    auto flush = [&](int jj) {
        float* slot = red + ((size_t)(BT_CHECK_IDX(jj < M1 && warp < kW, kChkRedSlot, a.ctrl) ? jj : 0) * kW + warp) *
                                kDenseVals;
        if constexpr (kFull) {
            float v[kDenseVals];
            ordered_sums(acc, v);
            slot[lane] = warp_transpose_reduce(v, lane);
        } else {
            float c0 = acc.p[12].x, c1 = acc.p[12].y;
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                c0 += __shfl_xor_sync(0xffffffffu, c0, o);
                c1 += __shfl_xor_sync(0xffffffffu, c1, o);
            }
            if (lane == 0) {
                slot[27] = c0;
                slot[28] = c1;
            }
        }
        clear();
    };
    int u = nC > 0 ? valid_from(warp * M1) : u_end;
    if constexpr (residual_pipelined(kFull)) {
        static_assert(kSteps % 2 == 0, "two steps in flight");
        Step<P, kN> x0, x1;
        if (u < u_end) issue(x0, u, 0);
        while (u < u_end) {
            const int un = valid_from(u + 1);
#pragma unroll
            for (int sub = 0; sub < kSteps; sub += 2) {
                issue(x1, u, sub + 1);
                use(x0, u, sub);
                if (sub + 2 < kSteps) issue(x0, u, sub + 2);
                else if (un < u_end) issue(x0, un, 0);
                use(x1, u, sub + 1);
            }
            if (un / kW != u / kW || un >= u_end) flush(u / kW);      // the warp's last unit of this target
            u = un;
        }
    } else {
        while (u < u_end) {
            const int un = valid_from(u + 1);
#pragma unroll
            for (int sub = 0; sub < kSteps; ++sub) {
                Step<P, kN> x;
                issue(x, u, sub);
                use(x, u, sub);
            }
            if (un / kW != u / kW || un >= u_end) flush(u / kW);
            u = un;
        }
    }
    __syncthreads();
    const int nout = M1 * kDenseVals;
    for (int o = threadIdx.x; o < nout; o += kT) {
        const int jj = o / kDenseVals, v = o % kDenseVals;
        if (!kFull && v != 27 && v != 28) continue;
        // warps that covered target jj: units [jj kW, (jj+1) kW), warp = unit / (N-1)
        const int w0 = (jj * kW) / M1, w1 = ((jj + 1) * kW - 1) / M1;
        float s = 0.f, cmp = 0.f;
        for (int w = w0; w <= w1; ++w) {
            if (w * M1 - jj * kW >= nC) break;      // this warp's chunks of the target, and all later ones, are empty
            const float x = red[((size_t)jj * kW + w) * kDenseVals + v];
            if constexpr (P == 0) {
                s += x;
            } else {               // compensated (Kahan) sum of the warps' block sums
                const float y = x - cmp;
                const float t2 = s + y;
                cmp = (t2 - s) - y;
                s = t2;
            }
        }
        if (BT_CHECK_IDX(tile < a.n_tiles && jj < M1, kChkOutput, a.ctrl))
            a.dpart[((size_t)tile * M1 + jj) * kDenseVals + v] = s;
    }
}

// Sparse term of one correspondence set (Eq. 2): e = T_i^-1 p_m - T_j^-1 p_n
// in the object frame, Huber weight from ||e||, and the 39 moments from which
// the right-perturbation blocks are rebuilt in FP64:
//   [0] sum w  [1..3] sum w a  [4..6] sum w b  [7..12] sum w a a^T (xx xy xz yy yz zz)
//   [13..18] sum w b b^T  [19..27] sum w b a^T (row-major)  [28..30] sum w e
//   [31..33] sum w a x e  [34..36] sum w b x e  [37] sum rho  [38] count
template <bool kFull>
__device__ void sparse_edge(const SolveArgs& a, int e)
{
    __shared__ float sred[kThreads / 32][kSparseVals];
    const EdgeDev E = a.edges[e];
    float Ti[12], Tj[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        Ti[k] = a.xinv[E.i * 12 + k];
        Tj[k] = a.xinv[E.j * 12 + k];
    }
    const float hub = a.huber_sparse;
    float acc[kSparseVals];
#pragma unroll
    for (int k = 0; k < kSparseVals; ++k) acc[k] = 0.f;
    for (int k = threadIdx.x; k < E.count; k += blockDim.x) {
        const float pmx = __ldg(E.pa + 3 * k), pmy = __ldg(E.pa + 3 * k + 1), pmz = __ldg(E.pa + 3 * k + 2);
        const float pnx = __ldg(E.pb + 3 * k), pny = __ldg(E.pb + 3 * k + 1), pnz = __ldg(E.pb + 3 * k + 2);
        const float ax = fmaf(Ti[0], pmx, fmaf(Ti[1], pmy, fmaf(Ti[2], pmz, Ti[3])));
        const float ay = fmaf(Ti[4], pmx, fmaf(Ti[5], pmy, fmaf(Ti[6], pmz, Ti[7])));
        const float az = fmaf(Ti[8], pmx, fmaf(Ti[9], pmy, fmaf(Ti[10], pmz, Ti[11])));
        const float bx = fmaf(Tj[0], pnx, fmaf(Tj[1], pny, fmaf(Tj[2], pnz, Tj[3])));
        const float by = fmaf(Tj[4], pnx, fmaf(Tj[5], pny, fmaf(Tj[6], pnz, Tj[7])));
        const float bz = fmaf(Tj[8], pnx, fmaf(Tj[9], pny, fmaf(Tj[10], pnz, Tj[11])));
        const float ex = ax - bx, ey = ay - by, ez = az - bz;
        const float ne = sqrtf(fmaf(ex, ex, fmaf(ey, ey, ez * ez)));
        const bool inl = ne <= hub;
        acc[37] += inl ? 0.5f * ne * ne : hub * (ne - 0.5f * hub);
        acc[38] += 1.f;
        if constexpr (kFull) {
            const float w = inl ? 1.f : hub / ne;
            const float wax = w * ax, way = w * ay, waz = w * az;
            const float wbx = w * bx, wby = w * by, wbz = w * bz;
            acc[0] += w;
            acc[1] += wax; acc[2] += way; acc[3] += waz;
            acc[4] += wbx; acc[5] += wby; acc[6] += wbz;
            acc[7] = fmaf(wax, ax, acc[7]);  acc[8] = fmaf(wax, ay, acc[8]);  acc[9] = fmaf(wax, az, acc[9]);
            acc[10] = fmaf(way, ay, acc[10]); acc[11] = fmaf(way, az, acc[11]); acc[12] = fmaf(waz, az, acc[12]);
            acc[13] = fmaf(wbx, bx, acc[13]); acc[14] = fmaf(wbx, by, acc[14]); acc[15] = fmaf(wbx, bz, acc[15]);
            acc[16] = fmaf(wby, by, acc[16]); acc[17] = fmaf(wby, bz, acc[17]); acc[18] = fmaf(wbz, bz, acc[18]);
            acc[19] = fmaf(wbx, ax, acc[19]); acc[20] = fmaf(wbx, ay, acc[20]); acc[21] = fmaf(wbx, az, acc[21]);
            acc[22] = fmaf(wby, ax, acc[22]); acc[23] = fmaf(wby, ay, acc[23]); acc[24] = fmaf(wby, az, acc[24]);
            acc[25] = fmaf(wbz, ax, acc[25]); acc[26] = fmaf(wbz, ay, acc[26]); acc[27] = fmaf(wbz, az, acc[27]);
            const float wex = w * ex, wey = w * ey, wez = w * ez;
            acc[28] += wex; acc[29] += wey; acc[30] += wez;
            acc[31] = fmaf(ay, wez, fmaf(-az, wey, acc[31]));
            acc[32] = fmaf(az, wex, fmaf(-ax, wez, acc[32]));
            acc[33] = fmaf(ax, wey, fmaf(-ay, wex, acc[33]));
            acc[34] = fmaf(by, wez, fmaf(-bz, wey, acc[34]));
            acc[35] = fmaf(bz, wex, fmaf(-bx, wez, acc[35]));
            acc[36] = fmaf(bx, wey, fmaf(-by, wex, acc[36]));
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < kSparseVals; ++k) {
        if (!kFull && k < 37) continue;
        float v = acc[k];
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) sred[warp][k] = v;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kSparseVals; k += blockDim.x) {   // blocks of 32 threads too
        if (!kFull && k < 37) continue;
        if (!BT_CHECK_IDX(e < a.n_edges, kChkOutput, a.ctrl)) continue;
        float s = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sred[w][k];
        a.spart[(size_t)e * kSparseVals + k] = s;
    }
}


template <bool kFull, int kT, int kB, int P>
__global__ void __launch_bounds__(kT, residual_threads_per_sm(kFull) / kT) residual_kernel(SolveArgs a)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    if ((int)blockIdx.x < a.n_edges) {
        pdl_wait_and_release();
        sparse_edge<kFull>(a, blockIdx.x);
    } else {
        dense_tile<kFull, kT, kB, P>(a, blockIdx.x - a.n_edges, dsm);   // waits after staging its tile
    }
}

// Batched residual pass: CTA b takes work item work[b] = (graph, item).
template <bool kFull, int kT, int kB, int P>
__global__ void __launch_bounds__(kT, residual_threads_per_sm(kFull) / kT) batch_residual_kernel(const SolveArgs* __restrict__ args,
                                                                       const int2* __restrict__ work)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ SolveArgs sa;
    const int2 w = work[blockIdx.x];     // the work list and arguments: written before the solve
    if (threadIdx.x == 0) sa = args[w.x];
    __syncthreads();
    if (w.y < sa.n_edges) {
        pdl_wait_and_release();
        sparse_edge<kFull>(sa, w.y);
    } else
        dense_tile<kFull, kT, kB, P>(sa, w.y - sa.n_edges, dsm);
}

// Diagnostic export of the association of the ordered pair (i -> j): one
// thread per source entry, the same decision functions and the same target
// gather as dense_tile, out[s] = target pixel or -1.
template <int P>
__global__ void __launch_bounds__(kThreads) assoc_debug_kernel(SolveArgs a, int i, int j, int* __restrict__ out)
{
    pdl_wait_and_release();
    __shared__ PairConst pc;
    if (threadIdx.x == 0) fill_pair_const(a, i, j, a.nodes[j], pc);
    __syncthreads();
    const NodeDev Ni = a.nodes[i];
    const PairK& K = pc.k;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < Ni.M; s += gridDim.x * blockDim.x) {
        float4 p, n;
        load_source<P>(Ni, s, p, n);
        float2 qxy, uv;
        float qz;
        int iu, iv;
        int res = -1;
        if (assoc_project(K, p.x, p.y, p.z, qxy, qz, uv, iu, iv)) {
            Texel<P> x = {};
            gather_target<P>(x, pc.tgt, iv * K.W + iu, true);
            const float4 t = decode_target<P>(x, pc.zref);
            float2 txy, dxy, nxy;
            float dz, nz;
            if (assoc_distance(K, uv, t.x, qxy, qz, a.dmax2, txy, dxy, dz) &&
                assoc_normal(K, n.x, n.y, n.z, t.y, t.z, t.w, a.cmin, nxy, nz))
                res = iv * K.W + iu;
        }
        out[s] = res;
    }
}

cudaError_t launch_assoc_debug(const SolveArgs& a, int i, int j, int M, int* out, cudaStream_t s)
{
    const int grid = std::max(1, std::min((M + kThreads - 1) / kThreads, 4096));
    if (a.precision == 1) return launch_chained(assoc_debug_kernel<1>, dim3(grid), dim3(kThreads), 0, s, a, i, j, out);
    if (a.precision == 2) return launch_chained(assoc_debug_kernel<2>, dim3(grid), dim3(kThreads), 0, s, a, i, j, out);
    return launch_chained(assoc_debug_kernel<0>, dim3(grid), dim3(kThreads), 0, s, a, i, j, out);
}

template <int S, int P>
static void set_residual_attrs_p()
{
    constexpr int kT = kShapeThreads[S], kB = kShapePix[S];
    const int mx = (int)residual_smem_bytes(kMaxNodes, S);
    cudaFuncSetAttribute(residual_kernel<true, kT, kB, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    cudaFuncSetAttribute(residual_kernel<false, kT, kB, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    cudaFuncSetAttribute(batch_residual_kernel<true, kT, kB, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    cudaFuncSetAttribute(batch_residual_kernel<false, kT, kB, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
}

template <int S>
static void set_residual_attrs()
{
    set_residual_attrs_p<S, 0>();
    set_residual_attrs_p<S, 1>();
    set_residual_attrs_p<S, 2>();
}

// Once per process (a function-local static: thread-safe initialisation).
static void ensure_residual_attrs()
{
    static const bool done = [] {
        set_residual_attrs<0>();
        set_residual_attrs<1>();
        set_residual_attrs<2>();
        set_residual_attrs<3>();
        set_residual_attrs<4>();
        set_residual_attrs<5>();
        return true;
    }();
    (void)done;
}

template <int S, int P>
static cudaError_t launch_residual_shape(const SolveArgs& a, bool full, int grid, size_t smem, cudaStream_t s)
{
    constexpr int kT = kShapeThreads[S], kB = kShapePix[S];
    if (full) return launch_chained(residual_kernel<true, kT, kB, P>, dim3(grid), dim3(kT), smem, s, a);
    return launch_chained(residual_kernel<false, kT, kB, P>, dim3(grid), dim3(kT), smem, s, a);
}

template <int S>
static cudaError_t launch_residual_s(const SolveArgs& a, bool full, int grid, size_t smem, cudaStream_t s)
{
    if (a.precision == 1) return launch_residual_shape<S, 1>(a, full, grid, smem, s);
    if (a.precision == 2) return launch_residual_shape<S, 2>(a, full, grid, smem, s);
    return launch_residual_shape<S, 0>(a, full, grid, smem, s);
}

cudaError_t launch_residual(const SolveArgs& a, bool full, cudaStream_t s, int shape)
{
    ensure_residual_attrs();
    const int grid = a.n_edges + a.n_tiles;
    if (grid == 0) return cudaSuccess;
    const size_t smem = residual_smem_bytes(a.N, shape);
    switch (shape) {
    case 1: return launch_residual_s<1>(a, full, grid, smem, s);
    case 2: return launch_residual_s<2>(a, full, grid, smem, s);
    case 3: return launch_residual_s<3>(a, full, grid, smem, s);
    case 4: return launch_residual_s<4>(a, full, grid, smem, s);
    case 5: return launch_residual_s<5>(a, full, grid, smem, s);
    default: return launch_residual_s<0>(a, full, grid, smem, s);
    }
}

template <int S, int P>
static cudaError_t launch_batch_residual_shape(const SolveArgs* args, const int2* work, int n, size_t smem,
                                               bool full, cudaStream_t s)
{
    constexpr int kT = kShapeThreads[S], kB = kShapePix[S];
    if (full) return launch_chained(batch_residual_kernel<true, kT, kB, P>, dim3(n), dim3(kT), smem, s, args, work);
    return launch_chained(batch_residual_kernel<false, kT, kB, P>, dim3(n), dim3(kT), smem, s, args, work);
}

template <int S>
static cudaError_t launch_batch_residual_s(const SolveArgs* args, const int2* work, int n, size_t smem, bool full,
                                           int precision, cudaStream_t s)
{
    if (precision == 1) return launch_batch_residual_shape<S, 1>(args, work, n, smem, full, s);
    if (precision == 2) return launch_batch_residual_shape<S, 2>(args, work, n, smem, full, s);
    return launch_batch_residual_shape<S, 0>(args, work, n, smem, full, s);
}

cudaError_t launch_batch_residual(const SolveArgs* args_dev, const int2* work_res, int n_work, int max_N, bool full,
                                  int shape, int precision, cudaStream_t s)
{
    ensure_residual_attrs();
    if (n_work == 0) return cudaSuccess;
    const size_t smem = residual_smem_bytes(max_N, shape);
    switch (shape) {
    case 1: return launch_batch_residual_s<1>(args_dev, work_res, n_work, smem, full, precision, s);
    case 2: return launch_batch_residual_s<2>(args_dev, work_res, n_work, smem, full, precision, s);
    case 3: return launch_batch_residual_s<3>(args_dev, work_res, n_work, smem, full, precision, s);
    case 4: return launch_batch_residual_s<4>(args_dev, work_res, n_work, smem, full, precision, s);
    case 5: return launch_batch_residual_s<5>(args_dev, work_res, n_work, smem, full, precision, s);
    default: return launch_batch_residual_s<0>(args_dev, work_res, n_work, smem, full, precision, s);
    }
}

void prepare_residual_attributes() { ensure_residual_attrs(); }

}  // namespace bt
