// Learned pivot proposal: a per-correspondence inlier-scoring MLP.
//
//   features f_i (8): (x_i - mean x) / rms_x (3), (y_i - mean y) / rms_y (3),
//                     degree_i / N, SC^2 row score_i / max_j row score_j
//   MLP 8 -> 64 -> 128 -> 64 -> 1, ReLU between layers, p_i = sigmoid(z4)
//   weights and activations in BF16, FP32 accumulation
//
// Parameter vector (FP32 master copy, 17217 values, row-major [out][in]):
//   W1[64][8] b1[64] W2[128][64] b2[128] W3[64][128] b3[64] W4[64] b4[1]
//
// Forward (inference): one CTA of 128 threads per 128 rows.
// Layer 1 (K = 8) and layer 4 (N = 1) run on CUDA cores; layers 2 and 3 run
// on the tensor cores (tcgen05.mma kind::f16, BF16 operands, FP32 TMEM
// accumulators) with operands written to shared memory in the 128-byte
// swizzled K-major layout by the threads themselves.
// Training: forward and backward of a 128-sample tile in one kernel, the
// activations in shared memory only; the activation gradients of layers 3 and
// 2 and the weight gradients of layers 2 and 3 on the tensor cores (BF16
// operands, FP32 accumulation, the weight gradients accumulated in tensor
// memory over a CTA's tiles); layers 1 and 4 and the biases on CUDA cores.
// Adam on CUDA cores.
#include <cuda_bf16.h>

#include "tr_common.cuh"
#include "tr_problem.h"
#include "tr_mlp.h"

namespace tr {

namespace {

constexpr int kRows = 128;
// shared-memory layout of the forward kernel (offsets from a 1024-aligned base)
constexpr int kOffH1 = 0;                       // A of layer 2: 128 rows x 64 bf16
constexpr int kOffW2 = kOffH1 + 128 * 128;      // B of layer 2: 128 rows (out) x 64 bf16 (in)
constexpr int kOffH2 = kOffW2 + 128 * 128;      // A of layer 3: 2 K-blocks x 128 rows x 64 bf16
constexpr int kOffW3 = kOffH2 + 2 * 128 * 128;  // B of layer 3: 2 K-blocks x 64 rows x 64 bf16
constexpr int kOffSmall = kOffW3 + 2 * 64 * 128;
constexpr int kSmallFloats = 512 + 64 + 128 + 64 + 64 + 1;   // W1 b1 b2 b3 W4 b4
constexpr int kOffBar = kOffSmall + ((kSmallFloats * 4 + 127) / 128) * 128;
constexpr int kFwdSmem = kOffBar + 128 + 1024;
constexpr uint32_t kIdescL2 = idesc_f32acc(1u, 1u, 128, 128);   // BF16 x BF16 -> F32, M 128, N 128
constexpr uint32_t kIdescL3 = idesc_f32acc(1u, 1u, 128, 64);    // M 128, N 64

// byte offset of 16-byte chunk c of row r in a K-major 128-byte-swizzled tile
__device__ __forceinline__ int sw128(int r, int c) { return (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ float bf16r(float a) { return __bfloat162float(__float2bfloat16_rn(a)); }

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Set-up of a forward CTA: the weights into shared memory (B operands in the
// swizzled layout), the mbarrier and 256 tensor-memory columns; returns the
// tensor-memory address.  All threads of the CTA call it.
__device__ uint32_t mlp_setup_cta(const float* __restrict__ wbf, uint8_t* smem)
{
    uint8_t* sW2 = smem + kOffW2;
    uint8_t* sW3 = smem + kOffW3;
    float* sW1 = reinterpret_cast<float*>(smem + kOffSmall);
    float* sb1 = sW1 + 512;
    float* sb2 = sb1 + 64;
    float* sb3 = sb2 + 128;
    float* sW4 = sb3 + 64;
    float* sb4 = sW4 + 64;
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + kOffBar);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + kOffBar + 16);
    const int t = threadIdx.x, warp = t >> 5;

    // weights (already BF16-rounded values stored as FP32) -> shared memory
    for (int q = t; q < 512; q += kRows) sW1[q] = wbf[kW1 + q];
    for (int q = t; q < 64; q += kRows) { sb1[q] = wbf[kB1 + q]; sb3[q] = wbf[kB3 + q]; sW4[q] = wbf[kW4 + q]; }
    for (int q = t; q < 128; q += kRows) sb2[q] = wbf[kB2 + q];
    if (t == 0) sb4[0] = wbf[kB4];
    {   // W2 row t (64 inputs) as B operand row t of layer 2
        const float* w = wbf + kW2 + t * 64;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            *reinterpret_cast<uint4*>(sW2 + sw128(t, c)) =
                make_uint4(pack_bf16(w[8 * c + 0], w[8 * c + 1]), pack_bf16(w[8 * c + 2], w[8 * c + 3]),
                           pack_bf16(w[8 * c + 4], w[8 * c + 5]), pack_bf16(w[8 * c + 6], w[8 * c + 7]));
    }
    if (t < 64) {   // W3 row t (128 inputs) as B operand row t of layer 3 (two K-blocks)
        const float* w = wbf + kW3 + t * 128;
#pragma unroll
        for (int c = 0; c < 16; ++c)
            *reinterpret_cast<uint4*>(sW3 + (c >> 3) * 8192 + sw128(t, c & 7)) =
                make_uint4(pack_bf16(w[8 * c + 0], w[8 * c + 1]), pack_bf16(w[8 * c + 2], w[8 * c + 3]),
                           pack_bf16(w[8 * c + 4], w[8 * c + 5]), pack_bf16(w[8 * c + 6], w[8 * c + 7]));
    }
    if (t == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc(tslot, 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    return *tslot;
}

// One tile of 128 rows (row0 ..) after mlp_setup_cta: completes two phases of
// the CTA's mbarrier (parities 0 then 1), so tiles can follow one another.
// Returns this thread's probability (0 for rows past m).
__device__ float mlp_tile(const float* __restrict__ feat, int m, int row0, float* prob, uint8_t* smem, uint32_t tmem,
                          uint32_t* err)
{
    uint8_t* sH1 = smem + kOffH1;
    uint8_t* sW2 = smem + kOffW2;
    uint8_t* sH2 = smem + kOffH2;
    uint8_t* sW3 = smem + kOffW3;
    float* sW1 = reinterpret_cast<float*>(smem + kOffSmall);
    float* sb1 = sW1 + 512;
    float* sb2 = sb1 + 64;
    float* sb3 = sb2 + 128;
    float* sW4 = sb3 + 64;
    float* sb4 = sW4 + 64;
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + kOffBar);
    const int t = threadIdx.x, warp = t >> 5;

    // layer 1 on CUDA cores: row = t
    const int row = row0 + t;
    float f[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) f[k] = row < m ? bf16r(feat[(size_t)row * 8 + k]) : 0.f;
#pragma unroll 1
    for (int c = 0; c < 8; ++c) {   // 8 outputs of layer 1 per 16-byte chunk of the A operand
        float h8[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int o = 8 * c + q;
            float z = sb1[o];
#pragma unroll
            for (int k = 0; k < 8; ++k) z = fmaf(sW1[o * 8 + k], f[k], z);
            h8[q] = fmaxf(z, 0.f);
        }
        *reinterpret_cast<uint4*>(sH1 + sw128(t, c)) =
            make_uint4(pack_bf16(h8[0], h8[1]), pack_bf16(h8[2], h8[3]), pack_bf16(h8[4], h8[5]),
                       pack_bf16(h8[6], h8[7]));
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    // layer 2 on the tensor cores: D[128 x 128] = H1[128 x 64] * W2^T
    if (t == 0) {
        tc_fence_after();
        const uint32_t a0 = smem_u32(sH1), b0 = smem_u32(sW2);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)   // K = 16 BF16 (32 bytes) per MMA
            mma_f16(tmem, sdesc_k_sw128(a0 + ks * 32), sdesc_k_sw128(b0 + ks * 32), kIdescL2, ks > 0 ? 1u : 0u);
        mma_commit(bar);
    }
    __syncwarp();
    if (!mbar_wait(bar, 0)) atomicOr(err, TR_ERR_TIMEOUT);
    tc_fence_after();
    // bias + ReLU, BF16, into the A operand of layer 3 (two K-blocks of 64)
    const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
#pragma unroll 1
    for (int cb = 0; cb < 4; ++cb) {
        uint32_t acc[32];
        tmem_ld32(tmem + lane_base + cb * 32, acc);
        tmem_ld_wait32(acc);
        float hv[32];
#pragma unroll
        for (int q = 0; q < 32; ++q) hv[q] = bf16r(fmaxf(__uint_as_float(acc[q]) + sb2[cb * 32 + q], 0.f));
#pragma unroll
        for (int c4 = 0; c4 < 4; ++c4) {
            const int k8 = cb * 4 + c4;   // 16-byte chunk index over the 128 inputs of layer 3
            *reinterpret_cast<uint4*>(sH2 + (k8 >> 3) * 16384 + sw128(t, k8 & 7)) =
                make_uint4(pack_bf16(hv[8 * c4 + 0], hv[8 * c4 + 1]), pack_bf16(hv[8 * c4 + 2], hv[8 * c4 + 3]),
                           pack_bf16(hv[8 * c4 + 4], hv[8 * c4 + 5]), pack_bf16(hv[8 * c4 + 6], hv[8 * c4 + 7]));
        }
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    // layer 3 on the tensor cores: D[128 x 64] = H2[128 x 128] * W3^T, TMEM columns 128..191
    if (t == 0) {
        tc_fence_after();
        const uint32_t a0 = smem_u32(sH2), b0 = smem_u32(sW3);
#pragma unroll
        for (int kb = 0; kb < 2; ++kb)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma_f16(tmem + 128, sdesc_k_sw128(a0 + kb * 16384 + ks * 32), sdesc_k_sw128(b0 + kb * 8192 + ks * 32),
                        kIdescL3, (kb | ks) != 0 ? 1u : 0u);
        mma_commit(bar);
    }
    __syncwarp();
    if (!mbar_wait(bar, 1)) atomicOr(err, TR_ERR_TIMEOUT);
    tc_fence_after();
    float z4 = sb4[0];
#pragma unroll 1
    for (int cb = 0; cb < 2; ++cb) {
        uint32_t acc[32];
        tmem_ld32(tmem + lane_base + 128 + cb * 32, acc);
        tmem_ld_wait32(acc);
        float hv[32];
#pragma unroll
        for (int q = 0; q < 32; ++q) {
            hv[q] = bf16r(fmaxf(__uint_as_float(acc[q]) + sb3[cb * 32 + q], 0.f));
            z4 = fmaf(sW4[cb * 32 + q], hv[q], z4);
        }
    }
    float pr = 0.f;
    if (row < m) {
        pr = 1.f / (1.f + __expf(-z4));
        prob[row] = pr;
    }
    // the tile's tensor-memory reads are complete before the next tile's MMAs
    tc_fence_before();
    __syncthreads();
    return pr;
}

__device__ void mlp_teardown_cta(uint32_t tmem)
{
    if ((threadIdx.x >> 5) == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 256);
    }
}

__device__ __forceinline__ uint8_t* aligned_smem(uint8_t* raw)
{
    return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
}

// Standalone forward over an arbitrary feature array.
__global__ void __launch_bounds__(kRows, 1) mlp_fwd_kernel(const float* feat, int m, const float* wbf, float* prob,
                                                           uint32_t* err)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = aligned_smem(smem_raw);
    const uint32_t tmem = mlp_setup_cta(wbf, smem);
    mlp_tile(feat, m, blockIdx.x * kRows, prob, smem, tmem, err);
    mlp_teardown_cta(tmem);
}

// Registration path: persistent CTAs (weights, mbarrier and tensor memory set
// up once, before the wait for the features) take the 128-row tiles of all
// problems in turn: rows of a problem's feature buffer -> its prob buffer,
// and the problem's largest probability into its control block (bounds of
// the learned pivot weights for the selection passes).
__global__ void __launch_bounds__(kRows, 2) mlp_proposal_kernel(Batch bt, int total, const float* wbf)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = aligned_smem(smem_raw);
    const uint32_t tmem = mlp_setup_cta(wbf, smem);
    pdl_wait();
    pdl_release();
    for (int tile = blockIdx.x; tile < total; tile += gridDim.x) {
        int lb;
        const ProbView v = bt.views[locate(bt, ST_MLP, tile, lb)];
        float pm = mlp_tile(v.feat, v.n, lb * kRows, v.prob, smem, tmem, &v.ctl->err);
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) pm = fmaxf(pm, __shfl_xor_sync(0xffffffffu, pm, off));
        if ((threadIdx.x & 31) == 0 && pm > 0.f) atomicMax(&v.ctl->pmax_bits, __float_as_uint(pm));
    }
    mlp_teardown_cta(tmem);
}

// Features of one problem (one block of 1024 threads per problem).
__global__ void __launch_bounds__(1024) features_kernel(ManyViews vs)
{
    pdl_wait();
    pdl_release();
    __shared__ float red[32][8];
    __shared__ float tot[8];
    int lb;
    const ProbView v = vs.get(ST_FEAT, blockIdx.x, lb);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // pass 1: sums of x, y and the largest row score
    float s[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int k = threadIdx.x; k < v.n; k += blockDim.x) {
        const float4* r = reinterpret_cast<const float4*>(v.pts8 + (size_t)k * 8);
        const float4 a = r[0], b = r[1];
        s[0] += a.x; s[1] += a.y; s[2] += a.z; s[3] += a.w; s[4] += b.x; s[5] += b.y;
        s[6] = fmaxf(s[6], static_cast<float>(v.rowscore[k]));
    }
    for (int q = 0; q < 7; ++q)
        for (int off = 16; off >= 1; off >>= 1) {
            const float o = __shfl_xor_sync(0xffffffffu, s[q], off);
            s[q] = q == 6 ? fmaxf(s[q], o) : s[q] + o;
        }
    if (lane == 0)
        for (int q = 0; q < 7; ++q) red[warp][q] = s[q];
    __syncthreads();
    if (threadIdx.x < 7) {
        float a = threadIdx.x == 6 ? 0.f : 0.f;
        for (int w = 0; w < 32; ++w) a = threadIdx.x == 6 ? fmaxf(a, red[w][6]) : a + red[w][threadIdx.x];
        tot[threadIdx.x] = threadIdx.x == 6 ? a : a / static_cast<float>(v.n);
    }
    __syncthreads();
    // pass 2: mean squared distances to the centroids
    float d[2] = {0.f, 0.f};
    for (int k = threadIdx.x; k < v.n; k += blockDim.x) {
        const float4* r = reinterpret_cast<const float4*>(v.pts8 + (size_t)k * 8);
        const float4 a = r[0], b = r[1];
        const float ex = a.x - tot[0], ey = a.y - tot[1], ez = a.z - tot[2];
        const float fx = a.w - tot[3], fy = b.x - tot[4], fz = b.y - tot[5];
        d[0] += ex * ex + ey * ey + ez * ez;
        d[1] += fx * fx + fy * fy + fz * fz;
    }
    for (int q = 0; q < 2; ++q)
        for (int off = 16; off >= 1; off >>= 1) d[q] += __shfl_xor_sync(0xffffffffu, d[q], off);
    __syncthreads();
    if (lane == 0) { red[warp][0] = d[0]; red[warp][1] = d[1]; }
    __syncthreads();
    __shared__ float inv[2];
    if (threadIdx.x < 2) {
        float a = 0.f;
        for (int w = 0; w < 32; ++w) a += red[w][threadIdx.x];
        const float rms = sqrtf(a / static_cast<float>(v.n));
        inv[threadIdx.x] = rms > 0.f ? 1.f / rms : 0.f;
    }
    __syncthreads();
    const float invn = 1.f / static_cast<float>(v.n);
    const float invr = tot[6] > 0.f ? 1.f / tot[6] : 0.f;
    for (int k = threadIdx.x; k < v.n; k += blockDim.x) {
        const float4* r = reinterpret_cast<const float4*>(v.pts8 + (size_t)k * 8);
        const float4 a = r[0], b = r[1];
        float4* o = reinterpret_cast<float4*>(v.feat + (size_t)k * 8);
        o[0] = make_float4((a.x - tot[0]) * inv[0], (a.y - tot[1]) * inv[0], (a.z - tot[2]) * inv[0],
                           (a.w - tot[3]) * inv[1]);
        o[1] = make_float4((b.x - tot[4]) * inv[1], (b.y - tot[5]) * inv[1], static_cast<float>(v.deg[k]) * invn,
                           static_cast<float>(v.rowscore[k]) * invr);
    }
}

// ---------------- training: forward and backward in one kernel ----------------
//
// Persistent CTAs of 512 threads take 128-sample tiles; thread t works for
// sample t % 128 on a quarter of the columns (t / 128), which is also its
// tensor-memory lane and column part.  Per tile:
//   h1 = relu(W1 x + b1)                         (CUDA cores)
//   h2 = relu(W2 h1 + b2), h3 = relu(W3 h2 + b3)  forward MMAs
//   z4 = W4 h3 + b4,  dz4 = (sigmoid(z4) - y) / m   (mean binary cross-entropy)
//   dz3 = W4 dz4 * [h3 > 0]                      (CUDA cores)
//   dz2 = (dz3 W3) * [h2 > 0]                    MMA1: D1[128 x 128] = DZ3[128 x 64] W3
//   dz1 = (dz2 W2) * [h1 > 0]                    MMA2: D2[128 x 64] = DZ2[128 x 128] W2
// and the weight gradients, summed over the samples and kept in tensor memory
// over all tiles of the CTA:
//   dW3^T[128 in x 64 out] += H2^T[128 x 128 s] DZ3[128 s x 64]     MMA3 (G3)
//   dW2[128 out x 64 in]    += DZ2^T[128 x 128 s] H1[128 s x 64]     MMA4 (G2)
// dW1 = dz1^T x, dW4 = h3^T dz4 and the biases (sums of dz over the samples)
// on CUDA cores in FP32, in registers over the tiles.  The MMAs take BF16
// operands (dz rounded to BF16; weights and activations are the forward's BF16
// values) and accumulate in FP32.
// Every operand is stored once, in the forward's swizzled K-major layout; where
// an MMA contracts over the samples or over a weight's outputs it reads the
// same buffer as an MN-major operand, so nothing is transposed or stored twice.
// Bound by the chain of its seven barriers and four MMA phases per tile (about
// 6 us) and by shared-memory reads (half of the path's rate).  Separate forward
// and backward kernels of 128 threads, with the activations through global
// memory and transposed operands written element by element, took 113 + 146 us
// at m = 131 072 and 22 + 54 us at m = 16 384; this one takes 54 to 57
// and 18 us.
constexpr int kTrainThreads = 512;
constexpr int kTOffH1 = 0;                       // [128 s][64]
constexpr int kTOffW2 = kTOffH1 + 16384;         // [128 out][64 in]
constexpr int kTOffH2 = kTOffW2 + 16384;         // 2 blocks of [128 s][64]
constexpr int kTOffW3 = kTOffH2 + 32768;         // 2 blocks of [64 out][64 in]
constexpr int kTOffDz3 = kTOffW3 + 16384;        // [128 s][64]
constexpr int kTOffDz2 = kTOffDz3 + 16384;       // 2 blocks of [128 s][64]
constexpr int kTOffH3 = kTOffDz2 + 32768;        // [128 s][64], read on CUDA cores only
constexpr int kTDz1Ld = 68;                      // FP32 dz1 [128 s][68]: rows 16 bytes apart in the banks
constexpr int kTOffDz1 = kTOffH3 + 16384;
constexpr int kTOffX = kTOffDz1 + 128 * kTDz1Ld * 4;   // FP32 2 x [2 halves][128 s][4] features (alternating tiles)
constexpr int kTOffW1 = kTOffX + 2 * 128 * 8 * 4;      // FP32 [32 output pairs][8 inputs][2]
constexpr int kTOffSmall = kTOffW1 + 512 * 4;          // FP32 b1[64] b2[128] b3[64] W4[64] b4
constexpr int kTOffZ = kTOffSmall + 336 * 4;           // FP32 [4][128] partial sums of z4
constexpr int kTOffG4 = kTOffZ + 512 * 4;              // FP32 [128] dz4
constexpr int kTOffBar = kTOffG4 + 128 * 4;
constexpr int kTrainSmem = kTOffBar + 128 + 1024;
static_assert(kTrainSmem <= 232448 && kTOffW1 % 16 == 0 && kTOffSmall % 16 == 0, "shared-memory plan");
// the final sums over the CTA's threads reuse dz2, h3 and dz1: dW1 + b1 [16][576], W4 + b3 [16][128], b2 [8][128]
static_assert((16 * 576 + 16 * 128 + 8 * 128) * 4 <= kTOffX - kTOffDz2, "scratch of the final sums");
constexpr uint32_t kTrainTmemCols = 512;   // layer 2 and D1 0..127, layer 3 and D2 128..191, G3 192..255, G2 256..319
constexpr uint32_t kMnA = 1u << 15, kMnB = 1u << 16;   // instruction descriptor: A / B MN-major

// Clears the gradient, the loss and the error bits.  It releases the training
// kernel at once: that one's set-up (weights into shared memory, tensor memory)
// and first tiles run meanwhile, and it waits before it writes any of them (a wait
// that gave up is kept in a register until then).  With a
// memset in front of it a step at m = 131 072 took 88 us and a gradient at
// m = 16 384 42 us per call, so 87 and 38.
__global__ void __launch_bounds__(256) mlp_clear_kernel(float* g, int count)
{
    pdl_release();
    const int k = blockIdx.x * 256 + threadIdx.x;
    if (k < count) g[k] = 0.f;
}

__global__ void __launch_bounds__(kTrainThreads, 1)
    mlp_train_kernel(const float* __restrict__ feat, const float* __restrict__ label, int m,
                     const float* __restrict__ wbf, float* grad, float* loss, uint32_t* err, uint32_t dbg)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = aligned_smem(smem_raw);
    uint8_t *sH1 = smem + kTOffH1, *sW2 = smem + kTOffW2, *sH2 = smem + kTOffH2, *sW3 = smem + kTOffW3;
    uint8_t *sDz3 = smem + kTOffDz3, *sDz2 = smem + kTOffDz2, *sH3 = smem + kTOffH3;
    float* sDz1 = reinterpret_cast<float*>(smem + kTOffDz1);
    float* sX = reinterpret_cast<float*>(smem + kTOffX);
    float* sW1 = reinterpret_cast<float*>(smem + kTOffW1);
    float* sb1 = reinterpret_cast<float*>(smem + kTOffSmall);
    float *sb2 = sb1 + 64, *sb3 = sb2 + 128, *sW4 = sb3 + 64, *sb4 = sW4 + 64;
    float* sZ = reinterpret_cast<float*>(smem + kTOffZ);
    float* sG4 = reinterpret_cast<float*>(smem + kTOffG4);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + kTOffBar);
    uint64_t* bar4 = bar + 1;   // MMA4 of the tile complete (its operands may be overwritten)
    uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + kTOffBar + 16);
    uint64_t* never = bar + 3;  // failure injection (tests only): nothing arrives here
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int sl = t & 127, part = t >> 7;   // sample of the tile, column part
    const int ntiles = (m + kRows - 1) / kRows;

    // weights -> shared memory, 8 inputs (16 bytes) per step
    static_assert(kW2 % 4 == 0 && kW3 % 4 == 0, "16-byte loads of the weight rows");
    for (int q = t; q < 1024; q += kTrainThreads) {
        const float4* w = reinterpret_cast<const float4*>(wbf + kW2) + 2 * q;   // row q / 8 (64 inputs), chunk q % 8
        const float4* u = reinterpret_cast<const float4*>(wbf + kW3) + 2 * q;   // row q / 16 (128 inputs), chunk q % 16
        const float4 w0 = w[0], w1 = w[1], u0 = u[0], u1 = u[1];
        *reinterpret_cast<uint4*>(sW2 + sw128(q >> 3, q & 7)) =
            make_uint4(pack_bf16(w0.x, w0.y), pack_bf16(w0.z, w0.w), pack_bf16(w1.x, w1.y), pack_bf16(w1.z, w1.w));
        *reinterpret_cast<uint4*>(sW3 + ((q >> 3) & 1) * 8192 + sw128(q >> 4, q & 7)) =
            make_uint4(pack_bf16(u0.x, u0.y), pack_bf16(u0.z, u0.w), pack_bf16(u1.x, u1.y), pack_bf16(u1.z, u1.w));
    }
    sW1[(t >> 4) * 16 + (t & 7) * 2 + ((t >> 3) & 1)] = wbf[kW1 + t];   // output t / 8, input t % 8
    if (t < 64) {
        sb1[t] = wbf[kB1 + t];
        sb3[t] = wbf[kB3 + t];
        sW4[t] = wbf[kW4 + t];
    } else if (t < 192) {
        sb2[t - 64] = wbf[kB2 + t - 64];
    } else if (t == 192) {
        sb4[0] = wbf[kB4];
        mbar_init(bar, 1);
        mbar_init(bar4, 1);
        mbar_init(never, 1);
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc(tslot, kTrainTmemCols);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const uint32_t tl = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);   // this warp's lanes
    const float inv_m = 1.f / static_cast<float>(m);
    bool expired = false;
    auto wait_on = [&](uint64_t* b, uint32_t parity) {
        if (!mbar_wait(b, parity)) expired = true;
        tc_fence_after();
    };
    if (dbg & TR_DBG_STALL_TRAIN) expired = !mbar_wait(never, 0u, kStallWaitNs);
    auto wait = [&](uint32_t parity) { wait_on(bar, parity); };

    // sums over the tiles.  dW1 and b1, W4 and b3: columns 2 lane, 2 lane + 1,
    // samples 8 warp ..; b2: columns 2 (t % 64), + 1, samples 16 (t / 64) ..
    const int o1 = t & 63, s1 = 16 * (t >> 6);
    float gW1[2][8] = {};
    float gb1[2] = {0.f, 0.f}, gb2[2] = {0.f, 0.f}, gb3[2] = {0.f, 0.f}, gW4[2] = {0.f, 0.f}, gb4 = 0.f, lsum = 0.f;
    // this thread's two of the next tile's 1024 features, and its sample's label
    float xf[2], yl;
    auto fetch = [&](int tile) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const size_t x = static_cast<size_t>(tile) * (kRows * 8) + t + q * kTrainThreads;
            xf[q] = tile < ntiles && x < static_cast<size_t>(m) * 8 ? feat[x] : 0.f;
        }
        const int s = tile * kRows + sl;
        yl = tile < ntiles && s < m ? label[s] : 0.f;
    };
    fetch(blockIdx.x);
    uint32_t first = 0u;   // accumulate flag of the weight gradients' first MMA
    uint32_t par4 = 0u;    // parity of this tile's phase of bar4
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        float* x = sX;
        sX += (sX == reinterpret_cast<float*>(smem + kTOffX)) ? 1024 : -1024;
        // inputs 0..3 of the samples, then inputs 4..7: a warp's 16-byte reads are conflict-free
        x[((t >> 2) & 1) * 512 + (t >> 3) * 4 + (t & 3)] = bf16r(xf[0]);
        x[((t >> 2) & 1) * 512 + (64 + (t >> 3)) * 4 + (t & 3)] = bf16r(xf[1]);
        const float y = yl;
        const bool valid = tile * kRows + sl < m;
        const float4 *xa = reinterpret_cast<const float4*>(x), *xb = xa + 128;
        fetch(tile + gridDim.x);
        if (first) wait_on(bar4, par4 ^ 1u);   // the previous tile's MMA4 has read H1 and DZ2
        __syncthreads();
        // ---- layer 1: outputs 4 warp .. + 3 of samples lane + 32 i ----
        // (a thread's 16 outputs in a 4 x 4 block: 16 shared-memory reads of 16
        // bytes; a row of 16 outputs of one sample took 34, and every such read
        // occupies the read path for four cycles, broadcast or not)
        {
            f2 w[2][8], bz[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const ulonglong2* wq = reinterpret_cast<const ulonglong2*>(sW1 + (2 * warp + q) * 16);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const ulonglong2 wk = wq[k];
                    w[q][2 * k] = f2{wk.x};
                    w[q][2 * k + 1] = f2{wk.y};
                }
                bz[q] = f2{reinterpret_cast<const unsigned long long*>(sb1)[2 * warp + q]};
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int s = lane + 32 * i;
                const float4 fa = xa[s], fb = xb[s];
                const float f[8] = {fa.x, fa.y, fa.z, fa.w, fb.x, fb.y, fb.z, fb.w};
                const bool vs = tile * kRows + s < m;
                uint32_t h[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    f2 z = bz[q];
#pragma unroll
                    for (int k = 0; k < 8; ++k) z = fma2(w[q][k], pk(f[k], f[k]), z);
                    float a, b;
                    upk(z, a, b);
                    h[q] = vs ? pack_bf16(fmaxf(a, 0.f), fmaxf(b, 0.f)) : 0u;
                }
                *reinterpret_cast<uint2*>(sH1 + sw128(s, warp >> 1) + (warp & 1) * 8) = make_uint2(h[0], h[1]);
            }
        }
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        if (t == 0) {   // layer 2: D[128 s x 128] = H1 W2^T
            tc_fence_after();
            const uint32_t a0 = smem_u32(sH1), b0 = smem_u32(sW2);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)   // K = 16 BF16 per MMA
                mma_f16(tmem, sdesc_k_sw128(a0 + ks * 32), sdesc_k_sw128(b0 + ks * 32), kIdescL2, ks > 0 ? 1u : 0u);
            mma_commit(bar);
        }
        __syncwarp();
        wait(0u);
        uint32_t mask2 = 0u;   // h2 > 0 of columns 32 part .. + 31
        {
            uint32_t acc[32];
            tmem_ld32(tl + part * 32, acc);
            tmem_ld_wait32(acc);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t h[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int e = 8 * c + 2 * q;
                    const float2 b = reinterpret_cast<const float2*>(sb2)[part * 16 + (e >> 1)];
                    h[q] = pack_bf16(fmaxf(__uint_as_float(acc[e]) + b.x, 0.f), fmaxf(__uint_as_float(acc[e + 1]) + b.y, 0.f));
                    if (!valid) h[q] = 0u;
                    mask2 |= (__uint_as_float(h[q] << 16) > 0.f ? 1u : 0u) << e;
                    mask2 |= (__uint_as_float(h[q] & 0xFFFF0000u) > 0.f ? 1u : 0u) << (e + 1);
                }
                const int k8 = part * 4 + c;
                *reinterpret_cast<uint4*>(sH2 + (k8 >> 3) * 16384 + sw128(sl, k8 & 7)) = make_uint4(h[0], h[1], h[2], h[3]);
            }
        }
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        if (t == 0) {   // layer 3: D[128 s x 64] = H2 W3^T
            tc_fence_after();
            const uint32_t a0 = smem_u32(sH2), b0 = smem_u32(sW3);
#pragma unroll
            for (int kb = 0; kb < 2; ++kb)
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    mma_f16(tmem + 128, sdesc_k_sw128(a0 + kb * 16384 + ks * 32), sdesc_k_sw128(b0 + kb * 8192 + ks * 32),
                            kIdescL3, (kb | ks) != 0 ? 1u : 0u);
            mma_commit(bar);
        }
        __syncwarp();
        wait(1u);
        uint32_t h3[8];   // columns 16 part .. + 15, BF16 pairs
        {
            uint32_t acc[16];
            tmem_ld16(tl + 128 + part * 16, acc);
            tmem_ld_wait16(acc);
            float z = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float2 b = reinterpret_cast<const float2*>(sb3)[part * 8 + q];
                const float2 w = reinterpret_cast<const float2*>(sW4)[part * 8 + q];
                h3[q] = pack_bf16(fmaxf(__uint_as_float(acc[2 * q]) + b.x, 0.f), fmaxf(__uint_as_float(acc[2 * q + 1]) + b.y, 0.f));
                if (!valid) h3[q] = 0u;
                z = fmaf(w.x, __uint_as_float(h3[q] << 16), z);
                z = fmaf(w.y, __uint_as_float(h3[q] & 0xFFFF0000u), z);
            }
            sZ[t] = z;
#pragma unroll
            for (int c = 0; c < 2; ++c)
                *reinterpret_cast<uint4*>(sH3 + sw128(sl, part * 2 + c)) =
                    make_uint4(h3[4 * c], h3[4 * c + 1], h3[4 * c + 2], h3[4 * c + 3]);
        }
        __syncthreads();
        // ---- dz4 (every thread of the sample), dz3 ----
        {
            float g4 = 0.f;
            if (valid) {
                const float z = sb4[0] + ((sZ[sl] + sZ[128 + sl]) + (sZ[256 + sl] + sZ[384 + sl]));
                const float p = 1.f / (1.f + __expf(-z));
                g4 = (p - y) * inv_m;
                if (part == 0) {
                    lsum += log1pf(__expf(-fabsf(z))) + fmaxf(z, 0.f) - y * z;
                    gb4 += g4;
                }
            }
            if (part == 0) sG4[sl] = g4;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t d[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float2 w = reinterpret_cast<const float2*>(sW4)[part * 8 + 4 * c + q];
                    d[q] = pack_bf16(__uint_as_float(h3[4 * c + q] << 16) > 0.f ? w.x * g4 : 0.f,
                                     __uint_as_float(h3[4 * c + q] & 0xFFFF0000u) > 0.f ? w.y * g4 : 0.f);
                }
                *reinterpret_cast<uint4*>(sDz3 + sw128(sl, part * 2 + c)) = make_uint4(d[0], d[1], d[2], d[3]);
            }
        }
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        if (t == 0) {   // MMA1 (D1 = DZ3 W3) and MMA3 (G3 += H2^T DZ3)
            tc_fence_after();
            const uint32_t dz3 = smem_u32(sDz3), w3 = smem_u32(sW3), h2 = smem_u32(sH2);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma_f16(tmem, sdesc_k_sw128(dz3 + ks * 32), sdesc_mn_sw128(w3 + ks * 2048, 8192), kIdescL2 | kMnB,
                        ks > 0 ? 1u : 0u);
            mma_commit(bar);   // MMA3 is complete at the commit behind MMA2
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                mma_f16(tmem + 192, sdesc_mn_sw128(h2 + ks * 2048, 16384), sdesc_mn_sw128(dz3 + ks * 2048, 16384),
                        kIdescL3 | kMnA | kMnB, ks > 0 ? 1u : first);
        }
        __syncwarp();
        // meanwhile: W4 and b3 (columns 2 lane, + 1 over 8 samples)
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int s = 8 * warp + q, off = sw128(s, lane >> 2) + (lane & 3) * 4;
            const uint32_t hv = *reinterpret_cast<const uint32_t*>(sH3 + off);
            const uint32_t dv = *reinterpret_cast<const uint32_t*>(sDz3 + off);
            const float g4 = sG4[s];
            gW4[0] = fmaf(g4, __uint_as_float(hv << 16), gW4[0]);
            gW4[1] = fmaf(g4, __uint_as_float(hv & 0xFFFF0000u), gW4[1]);
            gb3[0] += __uint_as_float(dv << 16);
            gb3[1] += __uint_as_float(dv & 0xFFFF0000u);
        }
        wait(0u);
        // ---- dz2 = D1 * [h2 > 0] ----
        {
            uint32_t acc[32];
            tmem_ld32(tl + part * 32, acc);
            tmem_ld_wait32(acc);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t d[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int e = 8 * c + 2 * q;
                    d[q] = pack_bf16((mask2 >> e) & 1u ? __uint_as_float(acc[e]) : 0.f,
                                     (mask2 >> (e + 1)) & 1u ? __uint_as_float(acc[e + 1]) : 0.f);
                }
                const int k8 = part * 4 + c;
                *reinterpret_cast<uint4*>(sDz2 + (k8 >> 3) * 16384 + sw128(sl, k8 & 7)) = make_uint4(d[0], d[1], d[2], d[3]);
            }
        }
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        if (t == 0) {   // MMA2 (D2 = DZ2 W2) and MMA4 (G2 += DZ2^T H1)
            tc_fence_after();
            const uint32_t dz2 = smem_u32(sDz2), w2 = smem_u32(sW2), h1 = smem_u32(sH1);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                mma_f16(tmem + 128, sdesc_k_sw128(dz2 + (ks >> 2) * 16384 + (ks & 3) * 32),
                        sdesc_mn_sw128(w2 + ks * 2048, 16384), kIdescL3 | kMnB, ks > 0 ? 1u : 0u);
            mma_commit(bar);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                mma_f16(tmem + 256, sdesc_mn_sw128(dz2 + ks * 2048, 16384), sdesc_mn_sw128(h1 + ks * 2048, 16384),
                        kIdescL3 | kMnA | kMnB, ks > 0 ? 1u : first);
            mma_commit(bar4);
        }
        __syncwarp();
        // meanwhile: b2 (columns 2 o1, + 1 over 16 samples)
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const uint32_t dv = *reinterpret_cast<const uint32_t*>(sDz2 + (o1 >> 5) * 16384 + sw128(s1 + q, (o1 & 31) >> 2) +
                                                                   (o1 & 3) * 4);
            gb2[0] += __uint_as_float(dv << 16);
            gb2[1] += __uint_as_float(dv & 0xFFFF0000u);
        }
        wait(1u);
        // ---- dz1 = D2 * [h1 > 0] (FP32) -> dW1, b1 ----
        {
            uint32_t acc[16];
            tmem_ld16(tl + 128 + part * 16, acc);
            uint32_t h[8];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const uint4 q = *reinterpret_cast<const uint4*>(sH1 + sw128(sl, part * 2 + c));
                h[4 * c] = q.x; h[4 * c + 1] = q.y; h[4 * c + 2] = q.z; h[4 * c + 3] = q.w;
            }
            tmem_ld_wait16(acc);
            float4* d = reinterpret_cast<float4*>(sDz1 + sl * kTDz1Ld + part * 16);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t hv = h[2 * c + (q >> 1)];
                    v[q] = __uint_as_float(q & 1 ? hv & 0xFFFF0000u : hv << 16) > 0.f ? __uint_as_float(acc[4 * c + q]) : 0.f;
                }
                d[c] = make_float4(v[0], v[1], v[2], v[3]);
            }
        }
        tc_fence_before();
        __syncthreads();
        // (two outputs per thread: each sample's 32 bytes of inputs, read by all
        // lanes, serve 16 products)
#pragma unroll 2
        for (int q = 0; q < 8; ++q) {
            const int s = 8 * warp + q;
            const float2 a = *reinterpret_cast<const float2*>(sDz1 + s * kTDz1Ld + 2 * lane);
            const float4 fa = xa[s], fb = xb[s];
            const float f[8] = {fa.x, fa.y, fa.z, fa.w, fb.x, fb.y, fb.z, fb.w};
            gb1[0] += a.x;
            gb1[1] += a.y;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                gW1[0][k] = fmaf(a.x, f[k], gW1[0][k]);
                gW1[1][k] = fmaf(a.y, f[k], gW1[1][k]);
            }
        }
        par4 ^= 1u;
        first = 1u;
    }
    // ---- the CTA's sums into the global gradient ----
    if (first) wait_on(bar4, par4 ^ 1u);
    pdl_wait();   // the gradient, the loss and the error bits are cleared
    if (expired) atomicOr(err, TR_ERR_TIMEOUT);
    {
        uint32_t g3[16], g2[16];
        tmem_ld16(tl + 192 + part * 16, g3);   // dW3[out = column][in = lane]
        tmem_ld16(tl + 256 + part * 16, g2);   // dW2[out = lane][in = column]
        tmem_ld_wait16(g3);
        tmem_ld_wait16(g2);
#pragma unroll
        for (int q = 0; q < 16; ++q) atomicAdd(&grad[kW3 + (part * 16 + q) * 128 + sl], __uint_as_float(g3[q]));
        static_assert(kW2 % 4 == 0, "16-byte additions to dW2");
#pragma unroll
        for (int q = 0; q < 4; ++q)
            atomicAdd(reinterpret_cast<float4*>(grad + kW2 + sl * 64 + part * 16 + 4 * q),
                      make_float4(__uint_as_float(g2[4 * q]), __uint_as_float(g2[4 * q + 1]),
                                  __uint_as_float(g2[4 * q + 2]), __uint_as_float(g2[4 * q + 3])));
    }
    __syncthreads();   // the last tile's buffers are consumed
    float* r1 = reinterpret_cast<float*>(sDz2);   // [16][576]: dW1 [64][8], b1 [64]
    float* r4 = r1 + 16 * 576;        // [16][128]: W4 [64], b3 [64]
    float* r2 = r4 + 16 * 128;        // [8][128]: b2
#pragma unroll
    for (int k = 0; k < 2; ++k) {
#pragma unroll
        for (int q = 0; q < 8; ++q) r1[warp * 576 + (2 * lane + k) * 8 + q] = gW1[k][q];
        r1[warp * 576 + 512 + 2 * lane + k] = gb1[k];
        r4[warp * 128 + 2 * lane + k] = gW4[k];
        r4[warp * 128 + 64 + 2 * lane + k] = gb3[k];
        r2[(t >> 6) * 128 + 2 * o1 + k] = gb2[k];
    }
    for (int off = 16; off >= 1; off >>= 1) {
        lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
        gb4 += __shfl_xor_sync(0xffffffffu, gb4, off);
    }
    if (warp < 4 && lane == 0) {   // the part-0 threads
        atomicAdd(loss, lsum * inv_m);
        atomicAdd(&grad[kB4], gb4);
    }
    __syncthreads();
    for (int q = t; q < 576 + 256; q += kTrainThreads) {
        float a = 0.f;
        int dst;
        if (q < 576) {
            for (int r = 0; r < 16; ++r) a += r1[r * 576 + q];
            dst = q < 512 ? kW1 + q : kB1 + q - 512;
        } else if (q < 704) {
            for (int r = 0; r < 16; ++r) a += r4[r * 128 + q - 576];
            dst = q < 640 ? kW4 + q - 576 : kB3 + q - 640;
        } else {
            for (int r = 0; r < 8; ++r) a += r2[r * 128 + q - 704];
            dst = kB2 + q - 704;
        }
        atomicAdd(&grad[dst], a);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, kTrainTmemCols);
    }
}

// ---------------- training: Adam (CUDA cores) ----------------

// Adam (bias-corrected), FP32 master weights; the forward's BF16-rounded copy
// is refreshed from them.  loss_out (page-locked host memory, or null) receives
// the step's loss.  A gradient whose kernel gave up on a wait (err) is left out:
// nothing is updated, and skipped (page-locked host memory) counts the step.
__global__ void __launch_bounds__(256) mlp_adam_kernel(float* w, float* mom, float* vel, const float* g, float* wbf,
                                                       int step, float lr, float b1, float b2, float eps,
                                                       const float* loss, float* loss_out, const uint32_t* err,
                                                       uint32_t* skipped)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (k == 0 && loss_out != nullptr) *loss_out = *loss;
    const uint32_t bad = *err;   // in flight with the loads below
    if (k >= kMlpParams) return;
    const float gk = g[k], m0 = mom[k], v0 = vel[k], w0 = w[k];
    if (bad != 0u) {
        if (k == 0) *skipped += 1u;
        return;
    }
    const float m1 = b1 * m0 + (1.f - b1) * gk;
    const float v1 = b2 * v0 + (1.f - b2) * gk * gk;
    mom[k] = m1;
    vel[k] = v1;
    const float mh = m1 / (1.f - powf(b1, static_cast<float>(step)));
    const float vh = v1 / (1.f - powf(b2, static_cast<float>(step)));
    const float nw = w0 - lr * mh / (sqrtf(vh) + eps);
    w[k] = nw;
    wbf[k] = bf16r(nw);
}

__global__ void __launch_bounds__(256) mlp_round_kernel(const float* w, float* wbf)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kMlpParams) wbf[k] = bf16r(w[k]);
}

}  // namespace

cudaError_t mlp_setup()
{
    cudaError_t e = cudaFuncSetAttribute(mlp_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(mlp_proposal_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTrainSmem);
    return e;
}

void launch_mlp_round(const float* w, float* wbf, cudaStream_t s)
{
    mlp_round_kernel<<<(kMlpParams + 255) / 256, 256, 0, s>>>(w, wbf);
}

void launch_features(const Batch& b, cudaStream_t s) { launch_pdl(features_kernel, b.num, 1024, 0, s, ManyViews{b}); }

void launch_mlp_proposal(const Batch& b, int total, const float* wbf, cudaStream_t s)
{
    const int sms = device_sms();
    const int grid = total < 2 * sms ? total : 2 * sms;
    launch_pdl(mlp_proposal_kernel, grid, kRows, kFwdSmem, s, b, total, wbf);
}

void launch_mlp_forward(const float* feat, int m, const float* wbf, float* prob, uint32_t* err, cudaStream_t s)
{
    mlp_fwd_kernel<<<(m + kRows - 1) / kRows, kRows, kFwdSmem, s>>>(feat, m, wbf, prob, err);
}

int mlp_train_blocks(int m)
{
    const int ntiles = (m + kRows - 1) / kRows, sms = device_sms();
    return ntiles < sms ? ntiles : sms;   // one CTA per SM (shared memory and tensor memory)
}

void launch_mlp_train(const float* feat, const float* label, int m, const float* wbf, float* grad, float* loss,
                      uint32_t* err, uint32_t dbg, cudaStream_t s)
{
    const int grid = mlp_train_blocks(m);
    mlp_clear_kernel<<<(kMlpParams + 2 + 255) / 256, 256, 0, s>>>(grad, kMlpParams + 2);
    launch_pdl(mlp_train_kernel, grid, kTrainThreads, kTrainSmem, s, feat, label, m, wbf, grad, loss, err,
               dbg);
}

void launch_mlp_adam(float* w, float* mom, float* vel, const float* g, float* wbf, int step, float lr,
                     const float* loss, float* loss_out, const uint32_t* err, uint32_t* skipped, cudaStream_t s)
{
    launch_pdl(mlp_adam_kernel, (kMlpParams + 255) / 256, 256, 0, s, w, mom, vel, g, wbf, step, lr, 0.9f, 0.999f, 1e-8f,
               loss, loss_out, err, skipped);
}

}  // namespace tr
