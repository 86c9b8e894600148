// bt_warmstart.cu -- kernels of the learned warm start (see bt_ws.h): sample
// preparation, the set network's forward and backward passes, the gradient
// reduction, Adam, and the FP64 relative-pose averaging solve that turns the
// predicted edge increments into node poses for Gauss-Newton (Sec. IV-D).
//
// Forward pass: a persistent CTA per SM keeps the BF16 W2 (in the tensor
// cores' core-matrix layout) in shared memory and walks an equal share of the
// chunks of 128 points of all sets.  Its warps form two groups that work on
// different chunks at the same time: eight run layer 1 (K = 6) on the FP32
// pipes, rounded to BF16 into one of two shared-memory tiles, from which one
// thread issues the 128 x 256 x 128 contraction of layer 2 to the
// fifth-generation tensor cores (tcgen05.mma, BF16 in, FP32 accumulators in
// tensor memory, completion signalled on an mbarrier); the other eight read
// the accumulators of earlier chunks back (tcgen05.ld) into running
// per-channel maxima and form the features of later ones.  The maxima are
// combined over the CTAs of a set with 64-bit atomic maxima (value, then
// first row).  The 256 -> 128 -> 6 head of all sets is a launch of its own.
// Every wait on the tensor cores is bounded (globaltimer); a wait that runs
// out sets the network's fault word, drains the contractions in flight, frees
// the tensor memory and ends the kernel, and the host reports BT_ERR_TIMEOUT.
// Backward pass: only the rows that hold a channel's maximum receive
// gradient, so layer 1 and layer 2 gradients are outer products over at most
// 256 rows, recomputed from the inputs with the forward pass's arithmetic.
#include "bt_ldlt.h"
#include "bt_ws.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>

namespace bt {
namespace ws {

namespace {

constexpr int kFwdThreads = 512;          // forward kernel: two groups of eight warps
constexpr int kGroupThreads = 256;        // one of them; also the head kernel
constexpr int kChunk = 128;     // points per layer-2 tile: the M of one tensor-core contraction
constexpr int kLd3 = 258;       // padded row length (BF16) of the layer-3 weights (odd word stride)

__device__ __forceinline__ float bf2f(__nv_bfloat16 b) { return __bfloat162float(b); }

// Features of one point pair (p in camera i, q in camera j: v = px py pz qx
// qy qz), FP32 with a fixed operation order (the backward pass recomputes
// them bit for bit).
__device__ __forceinline__ void features_from(const float v[6], const float* m, const float* c, float x[6])
{
    const float px = v[0], py = v[1], pz = v[2];
    const float qx = v[3], qy = v[4], qz = v[5];
    const float ux = __fmaf_rn(m[0], px, __fmaf_rn(m[1], py, __fmaf_rn(m[2], pz, m[3])));
    const float uy = __fmaf_rn(m[4], px, __fmaf_rn(m[5], py, __fmaf_rn(m[6], pz, m[7])));
    const float uz = __fmaf_rn(m[8], px, __fmaf_rn(m[9], py, __fmaf_rn(m[10], pz, m[11])));
    x[0] = __fmul_rn(__fsub_rn(ux, c[0]), kInvSP);
    x[1] = __fmul_rn(__fsub_rn(uy, c[1]), kInvSP);
    x[2] = __fmul_rn(__fsub_rn(uz, c[2]), kInvSP);
    x[3] = __fmul_rn(__fsub_rn(qx, ux), kInvSR);
    x[4] = __fmul_rn(__fsub_rn(qy, uy), kInvSR);
    x[5] = __fmul_rn(__fsub_rn(qz, uz), kInvSR);
}

// Features of point k of a set.
__device__ __forceinline__ void point_features(const float* __restrict__ p, const float* __restrict__ q,
                                               const float* m, const float* c, int k, float x[6])
{
    const float v[6] = {p[3 * k], p[3 * k + 1], p[3 * k + 2], q[3 * k], q[3 * k + 1], q[3 * k + 2]};
    features_from(v, m, c, x);
}

// Layer-1 pre-activation of one unit (weights w[6], bias b), fixed order.
__device__ __forceinline__ float z1_unit(const float* w, float b, const float x[6])
{
    float a = b;
#pragma unroll
    for (int k = 0; k < 6; ++k) a = __fmaf_rn(w[k], x[k], a);
    return a;
}

// ---------------------------------------------------------------------------
// Fifth-generation tensor cores (PTX ISA: tcgen05 instructions, shared-memory
// matrix descriptors, instruction descriptor of kind::f16)
// ---------------------------------------------------------------------------

// Both operands of the layer-2 contraction are K-major BF16 with K = 128,
// stored without swizzling as core matrices of 8 rows x 16 bytes (8 values of
// K): element (row, k) at core_off(row, k).  In the matrix descriptor the
// leading-dimension offset is the distance between core matrices that follow
// each other along K, the stride-dimension offset the distance between
// neighbouring groups of 8 rows.
constexpr uint32_t kCoreK = 128;                    // bytes from one core matrix to the next along K
constexpr uint32_t kCoreRows = (kH1 / 8) * kCoreK;  // 2048: bytes from one group of 8 rows to the next
constexpr uint32_t kH1TileBytes = kChunk * kH1 * 2; // one BF16 [128][128] tile of layer-1 outputs
__host__ __device__ constexpr uint32_t core_off(int row, int k)
{
    return (uint32_t)(row >> 3) * kCoreRows + (uint32_t)(k >> 3) * kCoreK + (uint32_t)(row & 7) * 16u +
           (uint32_t)(k & 7) * 2u;
}

// Matrix descriptor: start address >> 4 (bits 0-13), leading-dimension byte
// offset >> 4 (16-29), stride-dimension byte offset >> 4 (32-45), the fixed
// value 1 in bits 46-48, base offset 0, no swizzling.
__device__ __forceinline__ uint64_t mat_desc(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kCoreK >> 4) << 16) |
           ((uint64_t)(kCoreRows >> 4) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor: FP32 accumulator (bits 4-5 = 1), A and B BF16
// (bits 7-9 = 1, 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 in bits
// 17-22, M >> 4 in bits 24-28.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kH2 >> 3) << 17) |
                            ((uint32_t)(kChunk >> 4) << 24);
static_assert(kChunk == 128 && kH2 % 16 == 0 && kH2 <= 256, "shape of one kind::f16 contraction (M = 128)");

constexpr int kTmemCols = 2 * kH2;                 // two FP32 [128][256] accumulators
constexpr long long kTensorWaitNs = 1000000000LL;  // default bound of a wait on the tensor cores (1 s)

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// D[128][256] (tensor memory at d_tmem) = A[128][128] . B[256][128]^T, A and B
// K-major in shared memory: eight K = 16 steps, the first overwriting D; the
// completion of all eight arrives on the mbarrier at `bar`.  One thread.
__device__ __forceinline__ void issue_layer2(uint32_t d_tmem, uint32_t a_saddr, uint32_t b_saddr, uint32_t bar)
{
#pragma unroll
    for (int k = 0; k < kH1 / 16; ++k) {
        const uint64_t ad = mat_desc(a_saddr + 2 * kCoreK * k), bd = mat_desc(b_saddr + 2 * kCoreK * k);
        asm volatile(
            "{\n\t.reg .pred acc;\n\tsetp.ne.b32 acc, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, acc;\n\t}"
            ::"r"(d_tmem), "l"(ad), "l"(bd), "r"(kIdesc), "r"((uint32_t)(k > 0))
            : "memory");
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// Waits until phase `parity` of the mbarrier at `bar` has completed, for at
// most limit_ns of the global timer (read only once the first try, which
// suspends the thread for a while, has come back without it); limit_ns <= 0
// gives up without polling.
__device__ __forceinline__ bool wait_tensor(uint32_t bar, uint32_t parity, long long limit_ns)
{
    if (limit_ns <= 0) return false;
    unsigned long long t0 = 0;
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        const unsigned long long t = global_ns();
        if (t0 == 0) t0 = t;
        if ((long long)(t - t0) > limit_ns) return false;
    }
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Barrier of the kGroupThreads threads of the layer-1 group; true in all of
// them when any passes `fail`.
__device__ __forceinline__ bool group_sync_or(bool fail)
{
    uint32_t any;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(any)
        : "r"((uint32_t)fail), "n"(kGroupThreads)
        : "memory");
    return any != 0;
}

// Eight 16-lane x 256-bit blocks of tensor memory from taddr on (columns
// taddr + 8j .. + 8j + 7 for block j), waited for: lane l of the warp gets
// v[4j], v[4j+1] = row (l / 4), columns 8j + 2 (l % 4) + {0, 1}, and
// v[4j+2], v[4j+3] = row (l / 4) + 8, the same columns.
__device__ __forceinline__ void tmem_load_16x256b_x8(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}

// Row stride (floats) of the features of a chunk in shared memory: the 16-byte
// loads of eight neighbouring rows fall into different banks.
constexpr int kLdX = 12;

// Layer 1 of a chunk, this thread's share: rows lane + 32 r (r = 0..3), units
// 16 w .. 16 w + 15 of warp w; ReLU, rounded to BF16, into the core-matrix
// layout of the tile.  Two units a packed FP32x2 instruction (each half rounds
// as the scalar one: the backward pass forms the same bits with z1_unit); a
// pair's weights are one warp-uniform read for four rows.  sW: per unit pair
// (w0 w0' w1 w1' .. w5 w5' b b'), 16 floats.
__device__ __forceinline__ void layer1_rows(unsigned char* tile, const float* sW, const float* sX, int warp, int lane)
{
    float2 x[4][6];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float* xr = sX + (lane + 32 * r) * kLdX;
        const float4 a = *reinterpret_cast<const float4*>(xr);
        const float2 b = *reinterpret_cast<const float2*>(xr + 4);
        x[r][0] = make_float2(a.x, a.x);
        x[r][1] = make_float2(a.y, a.y);
        x[r][2] = make_float2(a.z, a.z);
        x[r][3] = make_float2(a.w, a.w);
        x[r][4] = make_float2(b.x, b.x);
        x[r][5] = make_float2(b.y, b.y);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {      // eight units: one 16-byte core-matrix row of each of the four rows
        uint32_t o[4][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float4* w4 = reinterpret_cast<const float4*>(sW + (8 * warp + 4 * h + e) * 16);
            const float4 w01 = w4[0], w23 = w4[1], w45 = w4[2], bb = w4[3];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                float2 z = __ffma2_rn(make_float2(w01.x, w01.y), x[r][0], make_float2(bb.x, bb.y));
                z = __ffma2_rn(make_float2(w01.z, w01.w), x[r][1], z);
                z = __ffma2_rn(make_float2(w23.x, w23.y), x[r][2], z);
                z = __ffma2_rn(make_float2(w23.z, w23.w), x[r][3], z);
                z = __ffma2_rn(make_float2(w45.x, w45.y), x[r][4], z);
                z = __ffma2_rn(make_float2(w45.z, w45.w), x[r][5], z);
                __nv_bfloat162 b = __floats2bfloat162_rn(fmaxf(z.x, 0.f), fmaxf(z.y, 0.f));
                o[r][e] = *reinterpret_cast<uint32_t*>(&b);
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
            *reinterpret_cast<uint4*>(tile + core_off(lane + 32 * r, 16 * warp + 8 * h)) =
                make_uint4(o[r][0], o[r][1], o[r][2], o[r][3]);
    }
}

__device__ __forceinline__ int set_chunks(int n) { return n > kChunk ? (n + kChunk - 1) / kChunk : 1; }

// Shared-memory layout of the forward kernel (byte offsets).
struct Fwd {
    static constexpr size_t W2 = 0;                                          // bf16 [256][128], core_off layout
    static constexpr size_t H1 = W2 + 2 * (size_t)kH2 * kH1;                 // 2 x bf16 [128][128], core_off layout
    static constexpr size_t W1 = H1 + 2 * (size_t)kH1TileBytes;              // float [64][16]: unit pairs (layer1_rows)
    static constexpr size_t B2 = W1 + 4 * (size_t)kH1 * 8;                   // float [256]
    static constexpr size_t X = B2 + 4 * (size_t)kH2;                        // 2 x float [128][kLdX]
    static constexpr size_t SCAN = X + 8 * (size_t)kChunk * kLdX;            // int [16 + 2], fault word
    static constexpr size_t BAR = SCAN + 80;                                 // six mbarriers (u64)
    static constexpr size_t TM = BAR + 48;                                   // tensor-memory base address
    static constexpr size_t Total = TM + 16;
};
static_assert(Fwd::H1 % 16 == 0 && Fwd::W1 % 16 == 0 && Fwd::X % 16 == 0 && Fwd::BAR % 8 == 0, "alignment");
static_assert(Fwd::Total <= 227 * 1024, "shared memory of one CTA");
static_assert(Fwd::Total > 114 * 1024, "one CTA per SM: the two accumulators take all of its tensor memory");
static_assert(kFwdThreads == 2 * kGroupThreads && kGroupThreads == kH2 && kGroupThreads == 2 * kChunk, "thread mappings");

// The forward pass up to the max-pool.  pool[s][256]: running maximum of each
// channel, (float bits of relu(max z + b2)) << 32 | ~row (row 0xffffffff where
// it is not kept), zero on entry.  The chunks of all sets, in order, are
// divided evenly over the CTAs, wherever the sets begin and end.  What bounds it
// is the layer-1 group: ~3.2 k cycles a chunk, of which the tensor cores work
// ~1.0 k (2048 sets of 450 points: 91 us; one CTA an SM that walked whole sets,
// 233 us; two CTAs an SM over even shares, 108 us).
template <bool kTrain>
__global__ void __launch_bounds__(kFwdThreads, 1)
    forward_kernel(Net net, const Sample* __restrict__ smp, const int* __restrict__ ids, int n_sets,
                   unsigned long long* __restrict__ pool)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    float* sW1 = reinterpret_cast<float*>(sm + Fwd::W1);
    float* sB2 = reinterpret_cast<float*>(sm + Fwd::B2);
    float* sX = reinterpret_cast<float*>(sm + Fwd::X);
    int* sScan = reinterpret_cast<int*>(sm + Fwd::SCAN);
    volatile int* sFault = sScan + 18;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // this CTA's share of the chunks: each thread adds up a run of sets, the
    // thread whose run holds the first chunk finds its set
    auto id_of = [&](int s) { return ids ? __ldg(ids + s) : s; };
    auto points_of = [&](int s) { return __ldg(&smp[id_of(s)].n); };
    const int r0 = (int)((long long)tid * n_sets / kFwdThreads), r1 = (int)((long long)(tid + 1) * n_sets / kFwdThreads);
    int mine = 0;
#pragma unroll 4
    for (int s = r0; s < r1; ++s) mine += set_chunks(points_of(s));
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) sScan[warp] = incl;
    __syncthreads();
    int total = 0, before = 0;
#pragma unroll
    for (int w = 0; w < kFwdThreads / 32; ++w) {
        before += w < warp ? sScan[w] : 0;
        total += sScan[w];
    }
    before += incl - mine;
    const int x0 = (int)((long long)blockIdx.x * total / gridDim.x);
    const int count = (int)((long long)(blockIdx.x + 1) * total / gridDim.x) - x0;
    if (count <= 0) return;
    if (before <= x0 && x0 < before + mine) {
        int s = r0, at = before;
        for (;; ++s) {
            const int k = set_chunks(points_of(s));
            if (x0 < at + k) break;
            at += k;
        }
        sScan[16] = s;
        sScan[17] = x0 - at;
    }

    // stage the weights once per CTA; W2 as 16-byte core-matrix rows
#pragma unroll 8
    for (int k = tid; k < kH2 * kH1 / 8; k += kFwdThreads) {
        const int row = k >> 4, k8 = (k & 15) * 8;
        *reinterpret_cast<uint4*>(sm + Fwd::W2 + core_off(row, k8)) =
            *reinterpret_cast<const uint4*>(net.wb + bW2 + row * kH1 + k8);
    }
    for (int k = tid; k < kH1 * 8; k += kFwdThreads) {
        const int u = 2 * (k >> 4) + (k & 1), e = (k & 15) >> 1;
        sW1[k] = e < kIn ? bf2f(net.wb[bW1 + u * kIn + e]) : (e == kIn ? net.master[ob1 + u] : 0.f);
    }
    if (tid < kH2) sB2[tid] = net.master[ob2 + tid];

    // mbarriers of the two buffers: contraction done (the accumulator is full,
    // the tile free), accumulator free again (one arrival a read-out warp),
    // features ready (one a feature warp)
    const uint32_t bar = smem_u32(sm + Fwd::BAR);
    const uint32_t bar_done = bar, bar_free = bar + 16, bar_x = bar + 32;
    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_done + 8 * b, 1);
            mbar_init(bar_free + 8 * b, kGroupThreads / 32);
            mbar_init(bar_x + 8 * b, kChunk / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *sFault = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(sm + Fwd::TM)),
                     "r"((uint32_t)kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the tensor cores read W2 and the layer-1 tiles through the async proxy
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(sm + Fwd::TM);
    const uint32_t w2_s = smem_u32(sm + Fwd::W2), h1_s = smem_u32(sm + Fwd::H1);
    int issued = 0;                          // contractions issued (thread 0)

    if (warp < kGroupThreads / 32) {
        // layer 1 of chunk i into tile i % 2, once its features are there and
        // the contraction of chunk i - 2 has read the tile; then the
        // contraction, once the accumulator of chunk i - 2 has been read
        for (int i = 0; i < count; ++i) {
            const uint32_t b = i & 1, ph = (i >> 1) & 1;
            bool ok = wait_tensor(bar_x + 8 * b, ph, net.wait_ns);
            if (i >= 2) ok = ok && wait_tensor(bar_done + 8 * b, ph ^ 1, net.wait_ns);
            layer1_rows(sm + Fwd::H1 + b * kH1TileBytes, sW1, sX + b * kChunk * kLdX, warp, lane);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            if (group_sync_or(!ok || *sFault != 0)) {
                *sFault = 1;
                break;
            }
            tc_fence_after();
            if (tid == 0) {
                if (i < 2 || wait_tensor(bar_free + 8 * b, ph ^ 1, net.wait_ns)) {
                    tc_fence_after();
                    issue_layer2(tmem + b * kH2, h1_s + b * kH1TileBytes, w2_s, bar_done + 8 * b);
                    issued = i + 1;
                } else {
                    *sFault = 1;             // seen by the group at its next barrier
                }
            }
        }
    } else {
        const int gw = warp - kGroupThreads / 32, gt = tid - kGroupThreads;
        int s = sScan[16], c = sScan[17];    // the set and the chunk of it to be read out
        // features (the first kChunk threads of the group, one row each) are
        // formed two chunks ahead of the read-out, and their points loaded one
        // chunk before that; (fs, fc) is the chunk whose points are in pq, and
        // the description of its set and of the next is kept in registers so
        // that a change of set waits for no chain of loads
        int fs = s, fc = c;
        struct Set {
            const Sample* S;
            const float* p;
            const float* q;
            int n;
        };
        auto describe = [&](int set) {
            Set d;
            d.S = smp + id_of(min(set, n_sets - 1));
            d.n = __ldg(&d.S->n);
            d.p = reinterpret_cast<const float*>(__ldg(reinterpret_cast<const unsigned long long*>(&d.S->p)));
            d.q = reinterpret_cast<const float*>(__ldg(reinterpret_cast<const unsigned long long*>(&d.S->q)));
            return d;
        };
        Set cur, nxt;
        float pq[6];
        auto load_points = [&]() {
            const int k = fc * kChunk + gt;
            const bool in = k < cur.n;
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                pq[e] = in ? __ldg(cur.p + 3 * (size_t)k + e) : 0.f;
                pq[3 + e] = in ? __ldg(cur.q + 3 * (size_t)k + e) : 0.f;
            }
        };
        // features of (fs, fc) into buffer b, then the points of the chunk after it
        auto features = [&](uint32_t b, bool more) {
            float x[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            float m[12], cc[3];
#pragma unroll
            for (int e = 0; e < 12; ++e) m[e] = __ldg(cur.S->m + e);
#pragma unroll
            for (int e = 0; e < 3; ++e) cc[e] = __ldg(cur.S->c + e);
            if (fc * kChunk + gt < cur.n) features_from(pq, m, cc, x);
            float* xr = sX + b * kChunk * kLdX + gt * kLdX;
            *reinterpret_cast<float4*>(xr) = make_float4(x[0], x[1], x[2], x[3]);
            *reinterpret_cast<float2*>(xr + 4) = make_float2(x[4], x[5]);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_x + 8 * b);
            if (!more) return;
            if (fc + 1 < set_chunks(cur.n)) {
                ++fc;
            } else {
                ++fs;
                fc = 0;
                cur = nxt;
                nxt = describe(fs + 1);
            }
            load_points();
        };
        if (gt < kChunk) {
            cur = describe(fs);
            nxt = describe(fs + 1);
            load_points();
            features(0, count > 1);
            if (count > 1) features(1, count > 2);
        }
        // read-out: warp gw takes the tensor-memory lanes (rows of a chunk)
        // 32 (gw % 4) .. + 31 and the columns 128 (gw / 4) .. + 127; a lane holds
        // 32 of those columns (idx: column 128 cw + 8 (idx / 2) + 2 (lane % 4) + idx % 2)
        const int qr = gw & 3, cw = gw >> 2;
        // running maxima of the thread's 32 columns; training keeps relu(z + b)
        // and the row that holds it (first row on ties), inference the largest z:
        // adding the bias and the ReLU are monotonic, so they follow the maximum
        float best[32];
        int bestr[kTrain ? 32 : 1];
        auto reset = [&]() {
#pragma unroll
            for (int k = 0; k < 32; ++k) {
                best[k] = kTrain ? -1.f : -INFINITY;
                if constexpr (kTrain) bestr[k] = 0;
            }
        };
        reset();
        int n = points_of(s), n_next = points_of(min(s + 1, n_sets - 1));
        for (int i = 0; i < count; ++i) {
            const uint32_t b = i & 1, ph = (i >> 1) & 1;
            if (__any_sync(0xffffffffu, !wait_tensor(bar_done + 8 * b, ph, net.wait_ns))) {
                if (lane == 0) *sFault = 1;
                break;
            }
            tc_fence_after();
            // the contraction has read the tile, so layer 1 is done with the features of chunk i
            if (gt < kChunk && i + 2 < count) features(b, i + 3 < count);
            // the running maximum over the rows of the chunk, in increasing order
            const uint32_t tacc = tmem + b * kH2 + 128 * cw;
#pragma unroll
            for (int lh = 0; lh < 2; ++lh) {
                const int rb = c * kChunk + 32 * qr + 16 * lh;
                if (rb >= n) break;   // the same for the whole warp
                const int ra = rb + (lane >> 2), rc = ra + 8;
                const bool va = ra < n, vc = rc < n;
#pragma unroll
                for (int cq = 0; cq < 2; ++cq) {
                    uint32_t v[32];
                    tmem_load_16x256b_x8(tacc + ((uint32_t)(32 * qr + 16 * lh) << 16) + 64 * cq, v);
#pragma unroll
                    for (int g = 0; g < 8; ++g)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int k = 2 * (8 * cq + g) + e;
                            if constexpr (kTrain) {
                                const float b2 = sB2[128 * cw + 8 * (k >> 1) + 2 * (lane & 3) + (k & 1)];
                                const float za = fmaxf(__uint_as_float(v[4 * g + e]) + b2, 0.f);
                                if (va && za > best[k]) {
                                    best[k] = za;
                                    bestr[k] = ra;
                                }
                                const float zc = fmaxf(__uint_as_float(v[4 * g + 2 + e]) + b2, 0.f);
                                if (vc && zc > best[k]) {
                                    best[k] = zc;
                                    bestr[k] = rc;
                                }
                            } else {
                                if (va) best[k] = fmaxf(best[k], __uint_as_float(v[4 * g + e]));
                                if (vc) best[k] = fmaxf(best[k], __uint_as_float(v[4 * g + 2 + e]));
                            }
                        }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_free + 8 * b);
            const bool last = c + 1 == set_chunks(n);      // the last chunk of its set
            if (last || i + 1 == count) {
                // combine the 8 lanes of each column by recursive halving: lane l
                // ends with the columns idx0 .. idx0 + 3, idx0 = its bits 4, 3, 2
                int idx0 = 0;
#pragma unroll
                for (int st = 0; st < 3; ++st) {
                    const int half = 16 >> st;
                    const bool upper = (lane & half) != 0;
#pragma unroll
                    for (int k = 0; k < half; ++k) {
                        const float send = upper ? best[k] : best[k + half];
                        float keep = upper ? best[k + half] : best[k];
                        const float got = __shfl_xor_sync(0xffffffffu, send, half);
                        if constexpr (kTrain) {
                            const int rsend = upper ? bestr[k] : bestr[k + half];
                            int rkeep = upper ? bestr[k + half] : bestr[k];
                            const int rgot = __shfl_xor_sync(0xffffffffu, rsend, half);
                            if (got > keep || (got == keep && rgot < rkeep)) {
                                keep = got;
                                rkeep = rgot;
                            }
                            bestr[k] = rkeep;
                        } else {
                            keep = fmaxf(keep, got);
                        }
                        best[k] = keep;
                    }
                    idx0 += upper ? half : 0;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int idx = idx0 + k;
                    const int col = 128 * cw + 8 * (idx >> 1) + 2 * (lane & 3) + (idx & 1);
                    const float g = kTrain ? best[k] : fmaxf(best[k] + sB2[col], 0.f);
                    const unsigned row = kTrain ? ~(unsigned)bestr[k] : 0u;
                    if (g > 0.f || (kTrain && g == 0.f))
                        atomicMax(pool + (size_t)s * kH2 + col, ((unsigned long long)__float_as_uint(g) << 32) | row);
                }
                reset();
            }
            if (last) {
                ++s;
                c = 0;
                n = n_next;
                n_next = points_of(min(s + 1, n_sets - 1));
            } else {
                ++c;
            }
        }
    }
    __syncthreads();
    if (*sFault != 0 && tid == 0) {
        // give the contractions in flight time to finish before the tensor
        // memory is freed
        for (int i = max(0, issued - 2); i < issued; ++i) wait_tensor(bar_done + 8 * (i & 1), (i >> 1) & 1, kTensorWaitNs);
        *reinterpret_cast<volatile int*>(net.fault) = 1;
        __threadfence_system();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)kTmemCols)
                     : "memory");
    }
}

// The 256 -> 128 -> 6 head of kHeadSets sets a CTA: W3 is staged once (rows
// padded to an odd word stride) and each of its values read once for all of
// them (2048 sets: 12 us, the latency of staging and of the sums).
constexpr int kHeadSets = 8;
struct Head {
    static constexpr size_t W3 = 0;                                                   // bf16 [128][kLd3]
    static constexpr size_t G = W3 + ((2 * (size_t)kH3 * kLd3 + 15) / 16) * 16;       // float [256][kHeadSets]
    static constexpr size_t P = G + 4 * (size_t)kH2 * kHeadSets;                      // float [2][kHeadSets][128]
    static constexpr size_t Total = P + 8 * (size_t)kHeadSets * kH3;
};

template <bool kTrain>
__global__ void __launch_bounds__(kGroupThreads)
    head_kernel(Net net, const Sample* __restrict__ smp, const int* __restrict__ ids, int n_sets,
                const unsigned long long* __restrict__ pool, float* __restrict__ y_out, Cache* __restrict__ cache)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    __nv_bfloat16* sW3 = reinterpret_cast<__nv_bfloat16*>(sm + Head::W3);
    float* sG = reinterpret_cast<float*>(sm + Head::G);
    float* sP = reinterpret_cast<float*>(sm + Head::P);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s0 = blockIdx.x * kHeadSets, m = min(kHeadSets, n_sets - s0);
    constexpr int kPer = kH3 * kH2 / 8 / kGroupThreads;
    uint4 w16[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k)
        w16[k] = __ldg(reinterpret_cast<const uint4*>(net.wb + bW3) + tid + k * kGroupThreads);
    float w4[kOut][kH3 / 32], b4[kOut];
#pragma unroll
    for (int k = 0; k < kOut; ++k) {
#pragma unroll
        for (int i = 0; i < kH3 / 32; ++i) w4[k][i] = bf2f(net.wb[bW4 + k * kH3 + lane + 32 * i]);
        b4[k] = net.master[ob4 + k];
    }
    const float b3 = net.master[ob3 + (tid & (kH3 - 1))];
    // everything above is parameters; the maxima come from the predecessor
    pdl_wait_and_release();
#pragma unroll
    for (int k = 0; k < kPer; ++k) {   // eight values, rows padded to kLd3
        const int at = (tid + k * kGroupThreads) * 8;
        uint32_t* to = reinterpret_cast<uint32_t*>(sW3 + (at / kH2) * kLd3 + at % kH2);
        to[0] = w16[k].x;
        to[1] = w16[k].y;
        to[2] = w16[k].z;
        to[3] = w16[k].w;
    }
#pragma unroll
    for (int q = 0; q < kHeadSets; ++q) {
        const unsigned long long v = q < m ? __ldcg(pool + (size_t)(s0 + q) * kH2 + tid) : 0ull;
        const float g = __uint_as_float((unsigned)(v >> 32));
        sG[tid * kHeadSets + q] = g;
        if (kTrain && q < m) {
            cache[s0 + q].g[tid] = g;
            cache[s0 + q].r[tid] = (int)~(unsigned)v;
        }
    }
    __syncthreads();
    {   // layer 3: unit tid % 128, input half tid / 128; the odd row stride
        // kLd3 / 2 words puts the 32 units of a warp in 32 banks
        const int o = tid & (kH3 - 1), half = tid >> 7;
        const __nv_bfloat16* w = sW3 + o * kLd3 + half * 128;
        float a[kHeadSets];
#pragma unroll
        for (int q = 0; q < kHeadSets; ++q) a[q] = 0.f;
#pragma unroll 4
        for (int k = 0; k < 128; k += 2) {
            const __nv_bfloat162 w2 = *reinterpret_cast<const __nv_bfloat162*>(w + k);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float wk = e == 0 ? __low2float(w2) : __high2float(w2);
                const float4* g = reinterpret_cast<const float4*>(sG + (half * 128 + k + e) * kHeadSets);
#pragma unroll
                for (int q = 0; q < kHeadSets / 4; ++q) {
                    const float4 g4 = g[q];
                    a[4 * q] = __fmaf_rn(wk, g4.x, a[4 * q]);
                    a[4 * q + 1] = __fmaf_rn(wk, g4.y, a[4 * q + 1]);
                    a[4 * q + 2] = __fmaf_rn(wk, g4.z, a[4 * q + 2]);
                    a[4 * q + 3] = __fmaf_rn(wk, g4.w, a[4 * q + 3]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kHeadSets; ++q) sP[(half * kHeadSets + q) * kH3 + o] = a[q];
    }
    __syncthreads();
    if (tid < kH3) {
#pragma unroll
        for (int q = 0; q < kHeadSets; ++q) {
            const float z = b3 + (sP[q * kH3 + tid] + sP[(kHeadSets + q) * kH3 + tid]);
            if (kTrain && q < m) cache[s0 + q].z3[tid] = z;
            sP[q * kH3 + tid] = fmaxf(z, 0.f);
        }
    }
    __syncthreads();
    // layer 4: one warp per set, then its outputs in turn
    static_assert(kGroupThreads / 32 == kHeadSets, "one warp per set");
    if (warp < m) {
        const int s = s0 + warp;
        const bool empty = __ldg(&smp[ids ? __ldg(ids + s) : s].n) <= 0;       // no prediction
#pragma unroll
        for (int k = 0; k < kOut; ++k) {
            float a = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                a = __fmaf_rn(w4[k][i], sP[warp * kH3 + lane + 32 * i], a);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
            const float y = empty ? 0.f : b4[k] + a;
            if (lane == 0) {
                y_out[(size_t)s * kOut + k] = y;
                if (kTrain) cache[s].y[k] = y;
            }
        }
    }
}

template <bool kTrain>
struct ForwardAttr {
    static void set()
    {
        static const bool done = [] {      // once per process, thread-safe
            cudaFuncSetAttribute(forward_kernel<kTrain>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)Fwd::Total);
            cudaFuncSetAttribute(head_kernel<kTrain>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Head::Total);
            return true;
        }();
        (void)done;
    }
};

int num_sms()
{
    static const int n = [] {             // once per process, thread-safe
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 1;
    }();
    return n;
}

// ---------------------------------------------------------------------------
// Backward pass: one CTA per set of the minibatch leaves what the set
// contributes to the gradient in factored form (a BwdRec of 12.5 KiB), and
// one launch over the parameters sums the contributions of all sets.  The
// gradients of layers 2, 3 and 4 are sums of outer products over the sets, so
// writing them out per set first (264 KiB a set, read back by the sum) cost
// 71 + 37 us for a minibatch of 256 sets.
// ---------------------------------------------------------------------------

// 1024 threads: a set's chain of loads and sums is what takes the time, and
// splitting its sums over 256 outputs eight and four ways shortens it (256
// threads: 32 us for 256 sets).
constexpr int kBwdThreads = 1024;

__global__ void __launch_bounds__(kBwdThreads)
    backward_kernel(Net net, const Sample* __restrict__ smp, const int* __restrict__ ids, int n_sets,
                    Cache* __restrict__ cache, float inv_n, BwdRec* __restrict__ rec)
{
    constexpr int kPartsO = kBwdThreads / kH2, kO = kH3 / kPartsO;      // layer 3: units of a part
    constexpr int kPartsC = kBwdThreads / kH1, kC = kH2 / kPartsC;      // layer 1: channels of a part
    __shared__ float sdz2[kH2], sdz3[kH3], sMC[16], sg[kPartsO][kH2];
    __shared__ float sxr[kH2 * 8];           // features of channel c's row at 8 c
    __shared__ float spart[kPartsC][kH1][7];
    const int s = blockIdx.x, tid = threadIdx.x;
    const int sid = ids ? ids[s] : s;
    const Sample* S = smp + sid;
    BwdRec& R = rec[s];
    const int n = S->n;
    const int c = tid & (kH2 - 1), part = tid >> 8, j = tid & (kH1 - 1), seg = tid >> 7;
    // parameters and the set's own data first: the cache comes from the predecessor
    float w3[kO], w1[6], w2[kC];
#pragma unroll
    for (int o = 0; o < kO; ++o) w3[o] = bf2f(net.wb[bW3 + (part * kO + o) * kH2 + c]);
#pragma unroll
    for (int k = 0; k < 6; ++k) w1[k] = bf2f(net.wb[bW1 + j * kIn + k]);
    const float b1 = net.master[ob1 + j];
    if (tid < 12) sMC[tid] = S->m[tid];
    else if (tid < 15) sMC[tid] = S->c[tid - 12];
    pdl_wait_and_release();
    if (n <= 0) {      // no forward pass: contributes nothing
        if (tid < kH2) cache[s].g[tid] = 0.f;
        float* f = reinterpret_cast<float*>(&R);
        for (int k = tid; k < (int)(sizeof(BwdRec) / sizeof(float)); k += kBwdThreads) f[k] = 0.f;
        return;
    }
    const Cache* C = cache + s;
    float dy[kOut];
#pragma unroll
    for (int m = 0; m < kOut; ++m) dy[m] = __ldcg(&C->y[m]) - __ldg(&S->ystar[m]);
    const float g = __ldcg(&C->g[c]);
    const int row = min(max(__ldcg(&C->r[c]), 0), n - 1);
    __syncthreads();      // sMC
    if (tid == 0) {
        float l = 0.f;
#pragma unroll
        for (int m = 0; m < kOut; ++m) l = __fmaf_rn(dy[m], dy[m], l);
        R.loss = 0.5f * l * inv_n;
#pragma unroll
        for (int m = 0; m < kOut; ++m) R.dy[m] = dy[m] * inv_n;
    }
    // layer 4
    if (tid < kH3) {
        const float z3 = __ldcg(&C->z3[tid]);
        float a = 0.f;
#pragma unroll
        for (int m = 0; m < kOut; ++m) a = __fmaf_rn(bf2f(net.wb[bW4 + m * kH3 + tid]), dy[m] * inv_n, a);
        const float d = z3 > 0.f ? a : 0.f;
        sdz3[tid] = d;
        R.dz3[tid] = d;
        R.h3[tid] = fmaxf(z3, 0.f);
    } else if (part == 1) {
        float x[6];
        point_features(S->p, S->q, sMC, sMC + 12, row, x);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            sxr[c * 8 + k] = x[k];
            R.x[c][k] = x[k];
        }
    }
    __syncthreads();
    // layer 3: dg = W3^T dz3, and ReLU' at the row holding the maximum
    {
        float a = 0.f;
#pragma unroll
        for (int o = 0; o < kO; ++o) a = __fmaf_rn(w3[o], sdz3[part * kO + o], a);
        sg[part][c] = a;
    }
#pragma unroll
    for (int q = 0; q < kC; ++q) w2[q] = bf2f(net.wb[bW2 + (seg * kC + q) * kH1 + j]);
    __syncthreads();
    if (part == 0) {
        float a = sg[0][c];
#pragma unroll
        for (int q = 1; q < kPartsO; ++q) a += sg[q][c];
        const float d = g > 0.f ? a : 0.f;
        sdz2[c] = d;
        R.x[c][6] = d;
    }
    __syncthreads();
    // layer 1: dW1[j][k] = sum_c dz2[c] W2[c][j] [z1(r_c, j) > 0] x(r_c)[k]
    float a[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < kC; ++q) {
        const int ch = seg * kC + q;
        const float4 xa = *reinterpret_cast<const float4*>(sxr + ch * 8);
        const float2 xb = *reinterpret_cast<const float2*>(sxr + ch * 8 + 4);
        const float xc[6] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y};
        // added only where the unit is active: the row's features need not be
        // finite where it is not (a NaN point's layer-1 outputs are all zero)
        const float d = sdz2[ch], w = d * w2[q];
        const bool on = z1_unit(w1, b1, xc) > 0.f && d != 0.f;
#pragma unroll
        for (int k = 0; k < 6; ++k) a[k] = on ? __fmaf_rn(w, xc[k], a[k]) : a[k];
        a[6] = on ? a[6] + w : a[6];
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) spart[seg][j][k] = a[k];
    __syncthreads();
    if (tid < kH1 * 7) {
        const int jj = tid / 7, k = tid % 7;
        float v = spart[0][jj][k];
#pragma unroll
        for (int q = 1; q < kPartsC; ++q) v += spart[q][jj][k];
        R.dw1[k < 6 ? jj * kIn + k : kH1 * kIn + jj] = v;
    }
}

// grad = the sum over sets of each parameter's contributions, in a fixed
// order: four groups of sets side by side in a CTA, then the groups.  CTAs
// [0, 128): two rows of dW2 each, dW2[c][j] = sum_s dz2[c] bf16(relu(z1(row
// r_c, unit j))) with the layer-1 output formed again from the row's features;
// [128, 160): four rows of dW3 = sum_s dz3 g^T each (one row a CTA would read
// the pooled features 128 times); the others 256 of the remaining parameters
// each.
constexpr int kSumThreads = 1024, kSumGroups = 4, kSumSets = 128;
constexpr int kSumRows = 4, kSumW2 = kH2 / 2, kSumW3 = kH3 / kSumRows;
constexpr int kSumRest = kH1 * kIn + kH1 + kH2 + kH3 + kOut * kH3 + kOut;
constexpr int kSumBlocks = kSumW2 + kSumW3 + (kSumRest + 255) / 256;

__global__ void __launch_bounds__(kSumThreads, 1)
    gradient_kernel(Net net, const BwdRec* __restrict__ rec, const Cache* __restrict__ cache, int n,
                    float* __restrict__ grad, double* __restrict__ loss)
{
    __shared__ float4 sx[kSumSets][2][2];        // features and dz2 of two channels' rows
    __shared__ float part[kSumGroups][256];
    pdl_wait_and_release();
    const int tid = threadIdx.x, col = tid & 255, grp = tid >> 8, b = blockIdx.x;
    float a = 0.f;
    int p = -1;                                  // the parameter this thread's column sums
    if (b < kSumW2) {
        const int j = col & 127, cl = col >> 7;
        p = oW2 + (2 * b + cl) * kH1 + j;
        float w1[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) w1[k] = bf2f(net.wb[bW1 + j * kIn + k]);
        const float b1 = net.master[ob1 + j];
        for (int s0 = 0; s0 < n; s0 += kSumSets) {
            const int m = min(kSumSets, n - s0);
            __syncthreads();
            if (tid < 4 * m)
                sx[tid >> 2][(tid >> 1) & 1][tid & 1] =
                    __ldcg(reinterpret_cast<const float4*>(rec[s0 + (tid >> 2)].x[2 * b + ((tid >> 1) & 1)]) + (tid & 1));
            __syncthreads();
#pragma unroll 4
            for (int s = grp; s < m; s += kSumGroups) {
                const float4 xa = sx[s][cl][0], xb = sx[s][cl][1];
                const float x[6] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y};
                const float h = __bfloat162float(__float2bfloat16_rn(fmaxf(z1_unit(w1, b1, x), 0.f)));
                a = __fmaf_rn(xb.z, h, a);
            }
        }
    } else if (b < kSumW2 + kSumW3) {
        const int o = (b - kSumW2) * kSumRows;
        float r[kSumRows] = {0.f, 0.f, 0.f, 0.f};
        // eight sets' loads in flight (left to the compiler they follow one another)
        for (int s0 = grp; s0 < n; s0 += 8 * kSumGroups) {
            float4 d[8];
            float g[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int s = s0 + u * kSumGroups;
                d[u] = s < n ? __ldcg(reinterpret_cast<const float4*>(&rec[s].dz3[o])) : make_float4(0.f, 0.f, 0.f, 0.f);
                g[u] = s < n ? __ldcg(&cache[s].g[col]) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                r[0] = __fmaf_rn(d[u].x, g[u], r[0]);
                r[1] = __fmaf_rn(d[u].y, g[u], r[1]);
                r[2] = __fmaf_rn(d[u].z, g[u], r[2]);
                r[3] = __fmaf_rn(d[u].w, g[u], r[3]);
            }
        }
#pragma unroll
        for (int q = 0; q < kSumRows; ++q) {
            __syncthreads();
            part[grp][col] = r[q];
            __syncthreads();
            if (grp == 0) grad[oW3 + (o + q) * kH2 + col] = (part[0][col] + part[1][col]) + (part[2][col] + part[3][col]);
        }
        return;
    } else {
        const int q = (b - kSumW2 - kSumW3) * 256 + col;
        constexpr int e1 = kH1 * kIn, e2 = e1 + kH1, e3 = e2 + kH2, e4 = e3 + kH3, e5 = e4 + kOut * kH3;
        if (q < kSumRest) {
            p = q < e1 ? oW1 + q : q < e2 ? ob1 + q - e1 : q < e3 ? ob2 + q - e2 : q < e4 ? ob3 + q - e3
                : q < e5 ? oW4 + q - e4 : ob4 + q - e5;
            // where in a set's record the parameter's terms are (a product of two for W4)
            const int at = q < e2   ? (int)(offsetof(BwdRec, dw1) / 4) + q      // dW1, then db1
                           : q < e3 ? 8 * (q - e2) + 6
                           : q < e4 ? (int)(offsetof(BwdRec, dz3) / 4) + q - e3
                           : q < e5 ? (int)(offsetof(BwdRec, h3) / 4) + (q - e4) % kH3
                                    : (int)(offsetof(BwdRec, dy) / 4) + q - e5;
            const int fac = q >= e4 && q < e5 ? (int)(offsetof(BwdRec, dy) / 4) + (q - e4) / kH3 : -1;
            for (int s0 = grp; s0 < n; s0 += 8 * kSumGroups) {
                float v[8], f[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int s = s0 + u * kSumGroups;
                    const float* R = reinterpret_cast<const float*>(rec + min(s, n - 1));
                    v[u] = s < n ? __ldcg(R + at) : 0.f;
                    f[u] = s >= n ? 0.f : fac >= 0 ? __ldcg(R + fac) : 1.f;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) a = __fmaf_rn(v[u], f[u], a);
            }
        }
        if (b == kSumBlocks - 1 && tid >= kSumThreads - 32) {
            double l = 0.0;
            for (int s = tid & 31; s < n; s += 32) l += (double)__ldcg(&rec[s].loss);
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
            if ((tid & 31) == 0) *loss = l;
        }
    }
    part[grp][col] = a;
    __syncthreads();
    if (grp == 0 && p >= 0) grad[p] = (part[0][col] + part[1][col]) + (part[2][col] + part[3][col]);
}

__device__ __forceinline__ int bf16_index(int p)
{
    if (p < ob1) return bW1 + (p - oW1);
    if (p >= oW2 && p < ob2) return bW2 + (p - oW2);
    if (p >= oW3 && p < ob3) return bW3 + (p - oW3);
    if (p >= oW4 && p < ob4) return bW4 + (p - oW4);
    return -1;
}

__global__ void adam_kernel(Net net, const float* __restrict__ grad, float lr, float beta1, float beta2,
                            float eps, float c1, float c2)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= kNumParams) return;
    const float g = grad[p];
    const float m = beta1 * net.m[p] + (1.f - beta1) * g;
    const float v = beta2 * net.v[p] + (1.f - beta2) * g * g;
    net.m[p] = m;
    net.v[p] = v;
    const float w = net.master[p] - lr * (m * c1) / (sqrtf(v * c2) + eps);
    net.master[p] = w;
    const int b = bf16_index(p);
    if (b >= 0) net.wb[b] = __float2bfloat16_rn(w);
}

__global__ void to_bf16_kernel(Net net)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= kNumParams) return;
    const int b = bf16_index(p);
    if (b >= 0) net.wb[b] = __float2bfloat16_rn(net.master[p]);
}

// ---------------------------------------------------------------------------
// FP64 rigid-motion helpers (3x4 row-major [R | t]); twists ordered (v, omega)
// ---------------------------------------------------------------------------

__device__ void pose_mul(const double* A, const double* B, double* C)
{
    for (int r = 0; r < 3; ++r) {
        for (int c = 0; c < 4; ++c) {
            double s = A[r * 4 + 0] * B[0 * 4 + c] + A[r * 4 + 1] * B[1 * 4 + c] + A[r * 4 + 2] * B[2 * 4 + c];
            if (c == 3) s += A[r * 4 + 3];
            C[r * 4 + c] = s;
        }
    }
}

__device__ void pose_inv(const double* A, double* C)
{
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) C[r * 4 + c] = A[c * 4 + r];
    for (int r = 0; r < 3; ++r)
        C[r * 4 + 3] = -(A[0 * 4 + r] * A[3] + A[1 * 4 + r] * A[7] + A[2 * 4 + r] * A[11]);
}

// Rodrigues coefficients: A = sin t / t, B = (1 - cos t) / t^2, C = (1 - A) / t^2.
__device__ void rodrigues_coeffs(double th, double& A, double& B, double& C)
{
    const double t2 = th * th;
    if (th < 1e-4) {
        A = 1.0 - t2 / 6.0;
        B = 0.5 - t2 / 24.0;
        C = 1.0 / 6.0 - t2 / 120.0;
    } else {
        const double s = sin(th), c = cos(th);
        A = s / th;
        B = (1.0 - c) / t2;
        C = (1.0 - A) / t2;
    }
}

// T = exp(xi) for xi = (v, w): R = I + A [w]x + B [w]x^2, t = (I + B [w]x + C [w]x^2) v.
__device__ void se3_exp(const double* xi, double* T)
{
    const double* v = xi;
    const double* w = xi + 3;
    const double th = sqrt(w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
    double A, B, C;
    rodrigues_coeffs(th, A, B, C);
    const double W[9] = {0.0, -w[2], w[1], w[2], 0.0, -w[0], -w[1], w[0], 0.0};
    double W2[9];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c)
            W2[r * 3 + c] = W[r * 3 + 0] * W[0 * 3 + c] + W[r * 3 + 1] * W[1 * 3 + c] + W[r * 3 + 2] * W[2 * 3 + c];
    for (int r = 0; r < 3; ++r) {
        double t = 0.0;
        for (int c = 0; c < 3; ++c) {
            const double id = r == c ? 1.0 : 0.0;
            T[r * 4 + c] = id + A * W[r * 3 + c] + B * W2[r * 3 + c];
            t += (id + B * W[r * 3 + c] + C * W2[r * 3 + c]) * v[c];
        }
        T[r * 4 + 3] = t;
    }
}

// w = log(R) of the rotation block of a 3x4 pose.
__device__ void so3_log(const double* T, double* w, double& th)
{
    double c = 0.5 * (T[0] + T[5] + T[10] - 1.0);
    c = c > 1.0 ? 1.0 : (c < -1.0 ? -1.0 : c);
    th = acos(c);
    const double k = th < 1e-4 ? 0.5 + th * th / 12.0 : 0.5 * th / sin(th);
    w[0] = k * (T[9] - T[6]);
    w[1] = k * (T[2] - T[8]);
    w[2] = k * (T[4] - T[1]);
}

// xi = log(T): w = log(R), v = V^-1 t with V^-1 = I - [w]x / 2 + D [w]x^2,
// D = (1 - A / (2 B)) / t^2.
__device__ void se3_log(const double* T, double* xi)
{
    double w[3], th;
    so3_log(T, w, th);
    double A, B, C;
    rodrigues_coeffs(th, A, B, C);
    const double D = th < 1e-4 ? 1.0 / 12.0 + th * th / 720.0 : (1.0 - A / (2.0 * B)) / (th * th);
    const double W[9] = {0.0, -w[2], w[1], w[2], 0.0, -w[0], -w[1], w[0], 0.0};
    for (int r = 0; r < 3; ++r) {
        double v = 0.0;
        for (int c = 0; c < 3; ++c) {
            double w2 = W[r * 3 + 0] * W[0 * 3 + c] + W[r * 3 + 1] * W[1 * 3 + c] + W[r * 3 + 2] * W[2 * 3 + c];
            v += ((r == c ? 1.0 : 0.0) - 0.5 * W[r * 3 + c] + D * w2) * T[c * 4 + 3];
        }
        xi[r] = v;
        xi[3 + r] = w[r];
    }
}

// The increment D of an edge from its output y and centre c:
// D(x) = R (x - c) + c + u, R = exp(omega).
__device__ void increment_from_output(const float* y, const float* c, double* D)
{
    double xi[6] = {0.0, 0.0, 0.0, y[0] * kSW, y[1] * kSW, y[2] * kSW};
    se3_exp(xi, D);
    for (int r = 0; r < 3; ++r) {
        const double Rc = D[r * 4 + 0] * c[0] + D[r * 4 + 1] * c[1] + D[r * 4 + 2] * c[2];
        D[r * 4 + 3] = (double)c[r] + y[3 + r] * kSU - Rc;
    }
}

// ---------------------------------------------------------------------------
// Sample preparation: centre, M0 (float) and label, one warp per item
// ---------------------------------------------------------------------------

__global__ void prep_kernel(Sample* __restrict__ smp, const PrepItem* __restrict__ items, int n_items)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= n_items) return;
    const PrepItem it = items[w];
    Sample* S = smp + it.sample;
    const int n = S->n;
    const float* q = S->q;
    // the centre: compensated FP32 sums per lane, combined in FP64 (a warp's
    // FP64 instruction, a conversion included, holds its DP unit as long as
    // a full one whatever the active lanes, so the per-point work stays off it)
    float s3[3] = {0.f, 0.f, 0.f}, k3[3] = {0.f, 0.f, 0.f};
    for (int k = lane; k < n; k += 32)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float y = q[3 * k + d] - k3[d];
            const float t = s3[d] + y;
            k3[d] = (t - s3[d]) - y;
            s3[d] = t;
        }
    double sx = (double)s3[0] - (double)k3[0], sy = (double)s3[1] - (double)k3[1],
           sz = (double)s3[2] - (double)k3[2];
    for (int off = 16; off > 0; off >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, off);
        sy += __shfl_xor_sync(0xffffffffu, sy, off);
        sz += __shfl_xor_sync(0xffffffffu, sz, off);
    }
    // M0 = T_j T_i^-1 one entry a lane (lanes 0-11, the operations of
    // pose_inv and pose_mul), the centre on lanes 12-14
    if (lane < 12) {
        const int r = lane >> 2, cc = lane & 3;
        const double* Ti = it.Ti0;
        const double* Tj = it.Tj0;
        double v;
        if (cc < 3) {
            v = Tj[r * 4 + 0] * Ti[cc * 4 + 0] + Tj[r * 4 + 1] * Ti[cc * 4 + 1] + Tj[r * 4 + 2] * Ti[cc * 4 + 2];
        } else {
            double iv[3];
            for (int k = 0; k < 3; ++k) iv[k] = -(Ti[0 * 4 + k] * Ti[3] + Ti[1 * 4 + k] * Ti[7] + Ti[2 * 4 + k] * Ti[11]);
            v = Tj[r * 4 + 0] * iv[0] + Tj[r * 4 + 1] * iv[1] + Tj[r * 4 + 2] * iv[2];
            v += Tj[r * 4 + 3];
        }
        S->m[lane] = (float)v;
    } else if (lane < 15) {
        const double sd = lane == 12 ? sx : lane == 13 ? sy : sz;
        S->c[lane - 12] = (float)(n > 0 ? sd / n : 0.0);
    } else if (lane == 15) {
        S->c[3] = 0.f;
    } else if (lane < 22 && !it.Ti1) {
        S->ystar[lane - 16] = 0.f;
    }
    if (lane != 0 || !it.Ti1) return;
    // training label (one lane): the increment from M0 to the converged M
    const double c[3] = {n > 0 ? sx / n : 0.0, n > 0 ? sy / n : 0.0, n > 0 ? sz / n : 0.0};
    double inv[12], M0[12];
    pose_inv(it.Ti0, inv);
    pose_mul(it.Tj0, inv, M0);
    {
        double M[12], M0inv[12], D[12], w[3], th;
        pose_inv(it.Ti1, inv);
        pose_mul(it.Tj1, inv, M);
        pose_inv(M0, M0inv);
        pose_mul(M, M0inv, D);
        so3_log(D, w, th);
        for (int r = 0; r < 3; ++r) {
            const double Rc = D[r * 4 + 0] * c[0] + D[r * 4 + 1] * c[1] + D[r * 4 + 2] * c[2];
            S->ystar[r] = (float)(w[r] / kSW);
            S->ystar[3 + r] = (float)((D[r * 4 + 3] + Rc - c[r]) / kSU);
        }
    }
}

__global__ void rebase_kernel(Sample* __restrict__ smp, int n, const float* old_p, const float* new_p,
                              const float* old_q, const float* new_q)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    smp[k].p = new_p + (smp[k].p - old_p);
    smp[k].q = new_q + (smp[k].q - old_q);
}

// ---------------------------------------------------------------------------
// Relative-pose averaging, one CTA per graph (FP64)
// ---------------------------------------------------------------------------

constexpr int kAvgThreads = 256;
constexpr int kScr = kAvgScratch;   // scratch doubles per edge (bt_ws.h)
constexpr int kScrP = 54;           // P = A^T W A, lower triangle (21)
constexpr int kScrG = 75;           // A^T W e (6)
static_assert(kScrG + 6 <= kScr, "averaging scratch per edge");

// Row and column of entry q (0..20) of a 6x6 lower triangle, row by row.
__device__ __forceinline__ void tri_rc(int q, int& r, int& c)
{
    r = 0;
    while ((r + 1) * (r + 2) / 2 <= q) ++r;
    c = q - r * (r + 1) / 2;
}

__global__ void __launch_bounds__(kAvgThreads) average_kernel(const AvgGraph* __restrict__ graphs)
{
    extern __shared__ __align__(16) double asm_[];
    __shared__ int s_sing;
    const AvgGraph G = graphs[blockIdx.x];
    const int N = G.N, E = G.n_edges, nf = G.n_free, n = 6 * nf, ld = n + 1;
    const int tid = threadIdx.x;
    double* sT0 = asm_;                      // [N][12]
    double* sT = sT0 + 12 * N;               // [N][12]
    double* H = sT + 12 * N;                 // [n][ld]
    double* b = H + (size_t)n * ld;          // [n]
    LdltScratch sc;                          // the solve's scratch (bt_ldlt.h)
    sc.work = b + n;                         // 16-byte aligned: n is even
    sc.part = sc.work + ldlt_work_doubles(n);  // [256]
    sc.rD = sc.part + 256;                   // [n]
    int* eof = reinterpret_cast<int*>(sc.rD + n);       // [N][N]
    int* freenode = eof + N * N;             // [nf]
    sc.shift = freenode + nf;
    const double Wd[6] = {1.0 / (kSU * kSU), 1.0 / (kSU * kSU), 1.0 / (kSU * kSU),
                          1.0 / (kSW * kSW), 1.0 / (kSW * kSW), 1.0 / (kSW * kSW)};
    if (tid == 0) s_sing = 0;
    for (int k = tid; k < 12 * N; k += kAvgThreads) sT0[k] = sT[k] = G.pose[k];
    for (int k = tid; k < N * N; k += kAvgThreads) eof[k] = -1;
    for (int k = tid; k < N; k += kAvgThreads)
        if (G.nodes[k].free_idx >= 0) freenode[G.nodes[k].free_idx] = k;
    __syncthreads();
    for (int e = tid; e < E; e += kAvgThreads) {
        const EdgeDev ed = G.edges[e];
        if (G.smp[e].n > 0) {
            eof[ed.i * N + ed.j] = e;
            eof[ed.j * N + ed.i] = e;
            increment_from_output(G.y + (size_t)e * kOut, G.smp[e].c, G.scratch + (size_t)e * kScr);
        }
    }
    __syncthreads();
    // 1. anchor every free node on its edge to the lowest fixed node
    for (int j = tid; j < N; j += kAvgThreads) {
        if (G.nodes[j].free_idx < 0) continue;
        for (int f = 0; f < N; ++f) {
            if (G.nodes[f].free_idx >= 0) continue;
            const int e = eof[f * N + j];
            if (e < 0) continue;
            const double* D = G.scratch + (size_t)e * kScr;
            double out[12];
            if (G.edges[e].i == f) {                       // D predicts T_j T_f^-1
                pose_mul(D, sT0 + 12 * j, out);
            } else {                                       // D predicts T_f T_j^-1
                double a[12], bq[12], Dinv[12], fi[12];
                pose_inv(sT0 + 12 * f, fi);
                pose_mul(sT0 + 12 * j, fi, a);
                pose_inv(D, Dinv);
                pose_mul(a, Dinv, bq);
                pose_mul(bq, sT0 + 12 * f, out);
            }
            for (int k = 0; k < 12; ++k) sT[12 * j + k] = out[k];
            break;
        }
    }
    __syncthreads();
    // 2. per edge: e = log(D M0 M^-1) and A = Ad(M) at the anchored poses
    for (int e = tid; e < E; e += kAvgThreads) {
        if (G.smp[e].n <= 0) continue;
        const int i = G.edges[e].i, j = G.edges[e].j;
        double* scr = G.scratch + (size_t)e * kScr;
        double inv[12], M0[12], M[12], Minv[12], t1[12], t2[12];
        pose_inv(sT0 + 12 * i, inv);
        pose_mul(sT0 + 12 * j, inv, M0);
        pose_inv(sT + 12 * i, inv);
        pose_mul(sT + 12 * j, inv, M);
        pose_inv(M, Minv);
        pose_mul(scr, M0, t1);
        pose_mul(t1, Minv, t2);
        se3_log(t2, scr + 12);
        double* A = scr + 18;
        const double tx[9] = {0.0, -M[11], M[7], M[11], 0.0, -M[3], -M[7], M[3], 0.0};
        for (int r = 0; r < 6; ++r)
            for (int c = 0; c < 6; ++c) A[r * 6 + c] = 0.0;
        for (int r = 0; r < 3; ++r)
            for (int c = 0; c < 3; ++c) {
                A[r * 6 + c] = M[r * 4 + c];
                A[(r + 3) * 6 + (c + 3)] = M[r * 4 + c];
                A[r * 6 + (c + 3)] = tx[r * 3 + 0] * M[0 * 4 + c] + tx[r * 3 + 1] * M[1 * 4 + c] +
                                     tx[r * 3 + 2] * M[2 * 4 + c];
            }
    }
    __syncthreads();
    // 3. normal equations over the free nodes (lower triangle) and right-hand
    // side.  The edge (i, j) has Jacobians J_i = -A, J_j = I on its
    // residual e (weights W): its i-side diagonal block A^T W A and its
    // gradient term A^T W e are formed once per edge, with the lanes packed
    // over (edge, entry) -- a warp's FP64 instruction takes its DP unit as
    // long whether 6 or 32 lanes are active -- then summed per node.
    for (int idx = tid; idx < E * 27; idx += kAvgThreads) {
        const int e = idx / 27, q = idx % 27;
        if (G.smp[e].n <= 0) continue;
        double* scr = G.scratch + (size_t)e * kScr;
        const double* A = scr + 18;
        double v = 0.0;
        if (q < 21) {
            int al, be;
            tri_rc(q, al, be);
            for (int g = 0; g < 6; ++g) v += A[g * 6 + al] * Wd[g] * A[g * 6 + be];
            scr[kScrP + q] = v;
        } else {
            const int al = q - 21;
            for (int g = 0; g < 6; ++g) v += A[g * 6 + al] * Wd[g] * scr[12 + g];
            scr[kScrG + al] = v;
        }
    }
    __syncthreads();
    // diagonal blocks: free node a's edges, A^T W A where a is the i side, W
    // where it is the j side
    for (int idx = tid; idx < nf * 21; idx += kAvgThreads) {
        const int f = idx / 21;
        int al, be;
        tri_rc(idx % 21, al, be);
        const int a = freenode[f];
        double v = 0.0;
        for (int m = 0; m < N; ++m) {
            const int e = m == a ? -1 : eof[a * N + m];
            if (e < 0) continue;
            if (G.edges[e].j == a) v += al == be ? Wd[al] : 0.0;
            else v += G.scratch[(size_t)e * kScr + kScrP + idx % 21];
        }
        H[(6 * f + al) * ld + 6 * f + be] = v;
    }
    // off-diagonal blocks: -A^T W (a = i) or -W A (a = j) of the edge between
    for (int idx = tid; idx < n * n; idx += kAvgThreads) {
        const int r = idx / n, c = idx % n;
        if (c > r || r / 6 == c / 6) continue;
        const int a = freenode[r / 6], al = r % 6, bn = freenode[c / 6], be = c % 6;
        double v = 0.0;
        const int e = eof[a * N + bn];
        if (e >= 0) {
            const double* A = G.scratch + (size_t)e * kScr + 18;
            if (G.edges[e].i == a) v = -A[be * 6 + al] * Wd[be];      // J_a = -A, J_b = I
            else v = -Wd[al] * A[al * 6 + be];                        // J_a = I, J_b = -A
        }
        H[r * ld + c] = v;
    }
    for (int r = tid; r < n; r += kAvgThreads) {
        const int a = freenode[r / 6], al = r % 6;
        double v = 0.0;
        for (int m = 0; m < N; ++m) {
            const int e = m == a ? -1 : eof[a * N + m];
            if (e < 0) continue;
            const double* scr = G.scratch + (size_t)e * kScr;
            if (G.edges[e].j == a) v += Wd[al] * scr[12 + al];
            else v -= scr[kScrG + al];
        }
        b[r] = v;
    }
    __syncthreads();
    // 4-5. H d = b by the FP32 inverse with double-float corrections, or
    // FP64 LDL^T where it declines (bt_ldlt.h); a pivot that is not positive,
    // or a solution that is not finite, leaves the poses as they were
    if (n > 0) {
        unsigned long long t_unused;
        ldlt_solve(H, ld, n, b, sc, true, &s_sing, t_unused);
        for (int i = tid; i < n; i += kAvgThreads)
            if (!isfinite(b[i])) s_sing = 1;
        __syncthreads();
    }
    if (s_sing) {
        if (tid == 0) *G.status = 1;
        return;
    }
    // 6. T_j <- exp(d_j) T_j for the free nodes
    for (int j = tid; j < N; j += kAvgThreads) {
        const int f = G.nodes[j].free_idx;
        if (f < 0) continue;
        double E6[12], out[12];
        se3_exp(b + 6 * f, E6);
        pose_mul(E6, sT + 12 * j, out);
        for (int k = 0; k < 12; ++k) G.pose[12 * j + k] = out[k];
    }
    if (tid == 0) *G.status = 0;
}

}  // namespace

cudaError_t launch_prep(Sample* smp, const PrepItem* items, int n, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    prep_kernel<<<(n + 7) / 8, 256, 0, s>>>(smp, items, n);
    return cudaGetLastError();
}

cudaError_t launch_to_bf16(Net net, cudaStream_t s)
{
    to_bf16_kernel<<<(kNumParams + 255) / 256, 256, 0, s>>>(net);
    return cudaGetLastError();
}

template <bool kTrain>
static cudaError_t launch_forward_t(Net net, const Sample* smp, const int* ids, int n, unsigned long long* pool,
                                    float* y_out, Cache* cache, cudaStream_t s)
{
    ForwardAttr<kTrain>::set();
    const cudaError_t e = cudaMemsetAsync(pool, 0, pool_bytes(n), s);
    if (e != cudaSuccess) return e;
    forward_kernel<kTrain><<<num_sms(), kFwdThreads, Fwd::Total, s>>>(net, smp, ids, n, pool);
    const cudaError_t f = cudaGetLastError();
    if (f != cudaSuccess) return f;
    return launch_chained(head_kernel<kTrain>, dim3((n + kHeadSets - 1) / kHeadSets), dim3(kGroupThreads), Head::Total, s,
                          net, smp, ids, n, pool, y_out, cache);
}

cudaError_t launch_forward(Net net, const Sample* smp, const int* ids, int n, unsigned long long* pool, float* y_out,
                           Cache* cache, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    return cache ? launch_forward_t<true>(net, smp, ids, n, pool, y_out, cache, s)
                 : launch_forward_t<false>(net, smp, ids, n, pool, y_out, nullptr, s);
}

cudaError_t launch_backward(Net net, const Sample* smp, const int* ids, int n, Cache* cache, BwdRec* rec,
                            float* grad, double* loss, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const cudaError_t e = launch_chained(backward_kernel, dim3(n), dim3(kBwdThreads), 0, s, net, smp, ids, n, cache,
                                         1.0f / (float)n, rec);
    if (e != cudaSuccess) return e;
    return launch_chained(gradient_kernel, dim3(kSumBlocks), dim3(kSumThreads), 0, s, net, rec, cache, n, grad, loss);
}

cudaError_t launch_adam(Net net, const float* grad, float lr, float beta1, float beta2, float eps, float c1,
                        float c2, cudaStream_t s)
{
    adam_kernel<<<(kNumParams + 255) / 256, 256, 0, s>>>(net, grad, lr, beta1, beta2, eps, c1, c2);
    return cudaGetLastError();
}

size_t average_smem_bytes(int max_free, int max_N)
{
    const size_t n = 6 * (size_t)max_free;
    return sizeof(double) * (24 * (size_t)max_N + n * (n + 1) + 2 * n + ldlt_work_doubles((int)n) + 256 + ldlt_shift_doubles(n)) +
           sizeof(int) * ((size_t)max_N * max_N + max_free) + 16;
}

cudaError_t launch_average(const AvgGraph* graphs, int n_graphs, int max_free, cudaStream_t s)
{
    if (n_graphs <= 0) return cudaSuccess;
    const size_t smem = average_smem_bytes(max_free, kMaxNodes);
    static const bool attr = [] {         // once per process, thread-safe
        cudaFuncSetAttribute(average_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)average_smem_bytes(kMaxNodes - 1, kMaxNodes));
        return true;
    }();
    (void)attr;
    average_kernel<<<n_graphs, kAvgThreads, smem, s>>>(graphs);
    return cudaGetLastError();
}

cudaError_t launch_rebase(Sample* smp, int n, const float* old_p, const float* new_p, const float* old_q,
                          const float* new_q, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    rebase_kernel<<<(n + 255) / 256, 256, 0, s>>>(smp, n, old_p, new_p, old_q, new_q);
    return cudaGetLastError();
}

}  // namespace ws
}  // namespace bt
