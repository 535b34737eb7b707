// BF16 tensor-core (tcgen05) kernels of the learned relaxation surrogate.
//
// gemm_kernel: D (M x N, FP32) = A (M x K, BF16, row-major) * B (N x K, BF16, row-major)^T, one
// CTA (one warpgroup) per 128-row tile of A: the tile and B are staged in shared memory in the
// core-matrix layout, thread 0 issues the K / 16 MMAs into TMEM, the mbarrier of the commit
// releases the warpgroup, and each thread reads its row of D from its TMEM lane.
#include <cuda_runtime.h>

#include <algorithm>

#include "lpdf_device.cuh"
#include "lpdf_internal.h"
#include "lpdf_tc.cuh"

namespace lpdf {

namespace {

constexpr int kTile = 128;              // rows per CTA (TMEM lanes)
constexpr int kMaxK = 128;
constexpr int kMaxN = 256;

struct GemmSmem {
    alignas(1024) unsigned char a[kTile * kMaxK * 2];
    alignas(1024) unsigned char b[kMaxN * kMaxK * 2];
    unsigned long long bar;
    uint32_t tmem;
};

__host__ __device__ inline uint32_t tmem_cols(int n)
{
    uint32_t c = 32;
    while ((int)c < n) c <<= 1;
    return c;
}

__global__ void __launch_bounds__(kTile, 1) gemm_kernel(const __nv_bfloat16* __restrict__ A,
                                                        const __nv_bfloat16* __restrict__ B, float* __restrict__ D,
                                                        int M, int N, int K, unsigned* __restrict__ error)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    GemmSmem& sm = *reinterpret_cast<GemmSmem*>(smem_raw);
    const int tid = threadIdx.x, wid = tid >> 5;
    const int r0 = blockIdx.x * kTile;
    // stage the operands (BF16, core-matrix layout)
    for (int i = tid; i < kTile * K; i += kTile) {
        const int r = i / K, k = i - (i / K) * K;
        const __nv_bfloat16 v = r0 + r < M ? A[(size_t)(r0 + r) * K + k] : __float2bfloat16(0.0f);
        *reinterpret_cast<__nv_bfloat16*>(sm.a + tc::core_offset(r, k, K)) = v;
    }
    for (int i = tid; i < N * K; i += kTile) {
        const int r = i / K, k = i - (i / K) * K;
        *reinterpret_cast<__nv_bfloat16*>(sm.b + tc::core_offset(r, k, K)) = B[(size_t)r * K + k];
    }
    const uint32_t ncols = tmem_cols(N);
    if (wid == 0) {
        tc::tmem_alloc(&sm.tmem, ncols);
        tc::tmem_relinquish();
    }
    if (tid == 0) tc::mbar_init1(&sm.bar);
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = sm.tmem;
    if (tid == 0) tc::gemm_issue(tmem, sm.a, sm.b, N, K, &sm.bar);
    bool ok = tc::mbar_wait(&sm.bar, 0);
    if (!ok) {
        atomicOr(error, 1u);
        ok = tc::mbar_wait(&sm.bar, 0);   // the MMAs in flight once more, then stop
    }
    tc::fence_after_sync();
    if (ok) {
        const int row = r0 + tid;
        for (int c0 = 0; c0 < N; c0 += 16) {
            float v[16];
            tc::tmem_ld16(tmem + ((uint32_t)(32 * (wid & 3)) << 16) + (uint32_t)c0, v);
            tc::wait_ld();
            if (row < M)
#pragma unroll
                for (int j = 0; j < 16; ++j) D[(size_t)row * N + c0 + j] = v[j];
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (wid == 0) tc::tmem_dealloc(tmem, ncols);
}

}  // namespace

cudaError_t launch_tc_gemm(const void* A, const void* B, float* D, int M, int N, int K, unsigned* error,
                           cudaStream_t st)
{
    if (M <= 0 || N < 16 || N > kMaxN || N % 16 || K < 16 || K > kMaxK || K % 16) return cudaErrorInvalidValue;
    static bool configured = false;
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(GemmSmem));
        if (e != cudaSuccess) return e;
        configured = true;
    }
    gemm_kernel<<<(unsigned)((M + kTile - 1) / kTile), kTile, sizeof(GemmSmem), st>>>(
        static_cast<const __nv_bfloat16*>(A), static_cast<const __nv_bfloat16*>(B), D, M, N, K, error);
    return cudaGetLastError();
}

}  // namespace lpdf

// ==========================================================================================
// The surrogate network: 8 -> 128 -> 128 -> 128 -> 7, tanh, on 128-row tiles (layouts in
// lpdf_internal.h, namespace mlp).
// ==========================================================================================
namespace lpdf {

namespace {

using namespace mlp;

// 8 consecutive values of row r from column k (a multiple of 8): one 16-byte piece of the core layout
__device__ __forceinline__ void put8(unsigned char* dst, int r, int k, int K, const float* v)
{
    uint4 q;
    uint32_t* w = reinterpret_cast<uint32_t*>(&q);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
        w[j] = *reinterpret_cast<const uint32_t*>(&b);
    }
    *reinterpret_cast<uint4*>(dst + tc::core_offset(r, k, K)) = q;
}
__device__ __forceinline__ void get8(const unsigned char* src, int r, int k, int K, float* v)
{
    const uint4 q = *reinterpret_cast<const uint4*>(src + tc::core_offset(r, k, K));
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v[2 * j] = __uint_as_float(w[j] << 16);
        v[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
    }
}

// A training step's two kernels follow one another closely (follow_grid): 50 steps of 1024 rows
// 1.53 -> 1.29 ms
template <class... P, class... A>
cudaError_t launch_following(void (*kernel)(P...), unsigned grid, int threads, uint32_t smem, bool follow, cudaStream_t st,
                             A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = follow ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

constexpr int kNetThreads = 512, kLossThreads = 128;   // kTrain: the loss has threads of its own
constexpr uint32_t kPackBytes = 2 * kPack, kXBytes = 2 * kH * kInP, kHBytes = 2 * kH * kH;

// dynamic shared memory: the weight pack, then per group the inputs and the activations (one buffer
// that every layer overwrites, or with kTrain the three layers'), then dZ4 with kTrain
template <int kGroups, bool kTrain>
constexpr uint32_t net_smem()
{
    return kPackBytes + kGroups * (kXBytes + (kTrain ? 3 : 1) * kHBytes) + (kTrain ? kXBytes : 0);
}

// thread order of the columns after the halving reduction below: lane l holds column l
// (the sums of 32 columns of a warp's rows; the same additions as 32 butterflies)
__device__ __forceinline__ float column_sums32(float* v, int lane)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int j = 0; j < o; ++j) {
            const float keep = up ? v[j + o] : v[j], give = up ? v[j] : v[j + o];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    return v[0];
}

// The network on 128-row tiles, one tile per group of 512 / kGroups threads at a time, the grid's groups
// striding over the tiles. feat (B x 8, FP32) is standardised with norm's feature means and deviations;
// out (may be NULL: B x 16, the 7 standardised outputs, then zeros), out_user (may be NULL: B x 7, in
// target units). With kTrain (a tile per CTA) the backward pass follows in the same launch: the gradient
// of the mean squared error over the 7 standardised outputs (weights norm[nW]) with respect to every
// parameter as this tile's partial sums, and the tile's loss.
//
// What bounds it: the chain of GEMM, TMEM read, tanh, shared-memory store, barrier through the layers of
// a tile, at a few tiles; the tanh instructions of the whole grid (2 x 10^7 per 50,000 rows) at many. So
// the epilogue of a tile is spread over 512 threads (a warp takes 32 rows x 32 columns), or over 256 with
// two tiles in flight per SM, one computing while the other waits (kGroups = 2, when there are more
// tiles than SMs). The weights arrive as one bulk copy of the pack, already in the operand layout, once
// per CTA. The backward needs no transposed copies: the transposed operands are the same buffers read
// MN-major, dZ overwrites the activations it came from, and the weight gradient and the next error
// signal are issued together into the two halves of TMEM.
template <int kGroups, bool kTrain>
__global__ void __launch_bounds__(kNetThreads + (kTrain ? kLossThreads : 0), 1)
                                                  mlp_kernel(const float* __restrict__ feat, const float* __restrict__ tgt,
                                                             int64_t B, const float* __restrict__ P,
                                                             const __nv_bfloat16* __restrict__ pack,
                                                             const float* __restrict__ norm, float* __restrict__ out,
                                                             float* __restrict__ out_user, float* __restrict__ part,
                                                             double* __restrict__ lpart, unsigned* __restrict__ error)
{
    static_assert(!kTrain || kGroups == 1, "a tile per CTA");
    constexpr int GT = kNetThreads / kGroups, kCols = kH / (GT / 128);   // columns per thread of an epilogue
    constexpr uint32_t kTmem = kTrain ? 256 : (kGroups == 1 ? 128 : 256);
    extern __shared__ __align__(1024) unsigned char dyn[];
    __shared__ float sb[3 * kH + kOutP], snorm[kNorm], wpart[4][kH];
    __shared__ float sout[kTrain ? 2 : 1][kTrain ? kOut : 1][kTrain ? kH : 1];   // a tile's outputs, for the loss
    __shared__ unsigned long long wbar, gbar[kGroups];
    __shared__ uint32_t tmem_slot;
    const int g = threadIdx.x / GT, t = threadIdx.x - g * GT, warp = t >> 5, lane = t & 31;
    const int quad = warp & 3, cb = warp >> 2, r = 32 * quad + lane;     // the thread's row and column block
    unsigned char* const w1 = dyn;
    unsigned char* const w2 = w1 + 2 * (pW2 - pW1);
    unsigned char* const w3 = w2 + kHBytes;
    unsigned char* const w4 = w3 + kHBytes;
    unsigned char* const x = dyn + kPackBytes + g * (kXBytes + (kTrain ? 3 : 1) * kHBytes);
    unsigned char* const h[3] = {x + kXBytes, x + kXBytes + (kTrain ? kHBytes : 0), x + kXBytes + (kTrain ? 2 * kHBytes : 0)};
    auto sync = [&]() {
        if (kGroups == 1 && !kTrain) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(GT) : "memory");
    };
    if (threadIdx.x == 0) {
        tc::mbar_init1(&wbar);
        for (int q = 0; q < kGroups; ++q) tc::mbar_init1(&gbar[q]);
    }
    if (threadIdx.x < 32) {
        tc::tmem_alloc(&tmem_slot, kTmem);
        tc::tmem_relinquish();
    }
    if (kTrain) follow_grid();   // the reduction that wrote P and pack, and read part and lpart
    if (threadIdx.x == 0) {
        asm volatile("fence.proxy.async.global;" ::: "memory");   // the pack was written by ordinary stores
        mbar_expect_tx(&wbar, kPackBytes);
        bulk_load(dyn, pack, kPackBytes, &wbar);
    }
    for (int i = threadIdx.x; i < 3 * kH + kOutP; i += blockDim.x)
        sb[i] = load_after(P + (i < kH ? ob1 + i : (i < 2 * kH ? ob2 - kH + i : (i < 3 * kH ? ob3 - 2 * kH + i : ob4 - 3 * kH + i))));
    for (int i = threadIdx.x; i < kNorm; i += blockDim.x) snorm[i] = norm[i];
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot + (kGroups == 1 ? 0u : 128u * g);
    const uint32_t lanes = (uint32_t)(32 * quad) << 16;
    unsigned long long* const bar = &gbar[g];
    uint32_t phase = 0;
    bool first = true;
    // after everyone's shared-memory stores: thread 0 of the group issues the GEMMs; all wait for them
    auto gemms = [&](auto issue) {
        tc::fence_async_smem();
        tc::fence_before_sync();
        sync();
        tc::fence_after_sync();
        if (t == 0) {
            if (first && !tc::mbar_wait(&wbar, 0)) atomicOr(error, 1u);
            issue();
            tc::mma_commit(bar);
        }
        first = false;
        if (!tc::mbar_wait(bar, phase)) {
            atomicOr(error, 1u);
            tc::mbar_wait(bar, phase);
        }
        phase ^= 1u;
        tc::fence_after_sync();
    };
    const int64_t ntiles = (B + kH - 1) / kH;
    // the hand-over of a tile's outputs to the loss's threads; the two buffers used in turn
    auto hand_over = [&]() { asm volatile("bar.sync 15, %0;" ::"n"(kNetThreads + kLossThreads) : "memory"); };
    int turn = 0;
    if (kTrain && threadIdx.x >= kNetThreads) {
        // the loss of a row in FP64, beside the backward pass: 7 divisions of 600 cycles each held the
        // network's warps up; 50 steps of 1024 rows 1.68 -> 1.53 ms (with the targets loaded ahead)
        for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, turn ^= 1) {
            const int64_t row = tile * kH + t;
            double s = 0.0;
            hand_over();
#pragma unroll
            for (int j = 0; j < kOut; ++j)
                if (row < B) {
                    const double y = ((double)tgt[row * kOut + j] - snorm[nTM + j]) / snorm[nTS + j];
                    const double d = (double)sout[turn][j][t] - y;
                    s += snorm[nW + j] * d * d;
                }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) lpart[tile * kLossParts + warp] = s;
        }
    }
    for (int64_t tile = kTrain && threadIdx.x >= kNetThreads ? ntiles : (int64_t)blockIdx.x * kGroups + g;
         tile < ntiles; tile += (int64_t)gridDim.x * kGroups) {
        const int64_t row0 = tile * kH, row = row0 + r;
        const bool live = row < B;
        // the inputs: a thread standardises 2 (4) columns of a row; columns 8..15 are zero
        {
            constexpr int kPer = kIn * kH / GT;
            const int rr = t / (kIn / kPer), k0 = kPer * (t % (kIn / kPer));
            float v[kPer];
#pragma unroll
            for (int k = 0; k < kPer; ++k)
                v[k] = row0 + rr < B ? (feat[(row0 + rr) * kIn + k0 + k] - snorm[nFM + k0 + k]) / snorm[nFS + k0 + k] : 0.0f;
#pragma unroll
            for (int k = 0; k < kPer; k += 2)
                *reinterpret_cast<__nv_bfloat162*>(x + tc::core_offset(rr, k0 + k, kInP)) = __floats2bfloat162_rn(v[k], v[k + 1]);
            if (t < kH) *reinterpret_cast<uint4*>(x + tc::core_offset(t, kIn, kInP)) = make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            gemms([&]() {
                if (l == 0) tc::gemm_issue_op(tmem, tc::k_major(x, kInP), tc::k_major(w1, kInP), kH, 1, false, false);
                else tc::gemm_issue_op(tmem, tc::k_major(h[l - 1], kH), tc::k_major(l == 1 ? w2 : w3, kH), kH, 8, false, false);
            });
#pragma unroll 1
            for (int c0 = cb * kCols; c0 < (cb + 1) * kCols; c0 += 32) {
                float v[32];
                tc::tmem_ld32(tmem + lanes + c0, v);
                tc::wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = tanhf(v[j] + sb[l * kH + c0 + j]);
#pragma unroll
                for (int j = 0; j < 32; j += 8) put8(h[l], r, c0 + j, kH, v + j);
            }
        }
        float target[kOut];   // kTrain: loaded while the last GEMM runs
        if (kTrain && cb == 0) {
#pragma unroll
            for (int j = 0; j < kOut; ++j) target[j] = live ? tgt[row * kOut + j] : 0.0f;
        }
        gemms([&]() { tc::gemm_issue_op(tmem, tc::k_major(h[2], kH), tc::k_major(w4, kH), kOutP, 8, false, false); });
        unsigned char* const z4 = x + kXBytes + 3 * kHBytes;   // kTrain
        if (cb == 0) {
            float v[16];
            tc::tmem_ld16(tmem + lanes, v);
            tc::wait_ld();
#pragma unroll
            for (int j = 0; j < kOutP; ++j) v[j] = j < kOut ? v[j] + sb[3 * kH + j] : 0.0f;
            if (!kTrain) {
                if (live && out)
#pragma unroll
                    for (int j = 0; j < kOutP; j += 4)
                        *reinterpret_cast<float4*>(out + row * kOutP + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                if (live && out_user)
#pragma unroll
                    for (int j = 0; j < kOut; ++j) out_user[row * kOut + j] = v[j] * snorm[nTS + j] + snorm[nTM + j];
            } else {
#pragma unroll
                for (int j = 0; j < kOut; ++j) sout[turn][j][r] = v[j];
                // dZ4 = d loss / d out: 2 (out - target) w_j / (7 B)
                float s[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) s[j] = 0.0f;
#pragma unroll
                for (int j = 0; j < kOut; ++j)
                    if (live) {
                        const float y = (target[j] - snorm[nTM + j]) / snorm[nTS + j];
                        s[j] = 2.0f * (v[j] - y) * snorm[nW + j] / (float)(kOut * B);
                    }
                put8(z4, r, 0, kOutP, s);
                put8(z4, r, 8, kOutP, s + 8);
                const float cs = column_sums32(s, lane);
                if (lane < kOutP) wpart[quad][lane] = cs;
            }
        }
        if constexpr (kTrain) {
            hand_over();
            turn ^= 1;
            float* const pp = part + (size_t)tile * kPart;
            // a layer: dW^T of the layer above (its input as the rows, its dZ as the columns) into the
            // upper half of TMEM and dH = dZ W into the lower; then dZ = dH (1 - h^2) over h, the bias
            // gradient (column sums of dZ) and dW^T to the partials
#pragma unroll
            for (int l = 2; l >= 0; --l) {
                gemms([&]() {
                    if (l == 2) {
                        tc::gemm_issue_op(tmem, tc::k_major(z4, kOutP), tc::mn_major(w4, kH), kH, 1, false, true);
                        tc::gemm_issue_op(tmem + 128, tc::mn_major(h[2], kH), tc::mn_major(z4, kOutP), kOutP, 8, true, true);
                    } else {
                        tc::gemm_issue_op(tmem, tc::k_major(h[l + 1], kH), tc::mn_major(l == 1 ? w3 : w2, kH), kH, 8, false, true);
                        tc::gemm_issue_op(tmem + 128, tc::mn_major(h[l], kH), tc::mn_major(h[l + 1], kH), kH, 8, true, true);
                    }
                });
                if (t < (l == 2 ? kOutP : kH))
                    pp[(l == 2 ? gb4 : (l == 1 ? gb3 : gb2)) + t] = wpart[0][t] + wpart[1][t] + wpart[2][t] + wpart[3][t];
                const int c0 = 32 * cb;
                float v[32];
                tc::tmem_ld32(tmem + lanes + c0, v);
                tc::wait_ld();
                sync();   // wpart is read
#pragma unroll
                for (int j = 0; j < 32; j += 8) {
                    float a[8];
                    get8(h[l], r, c0 + j, kH, a);
#pragma unroll
                    for (int q = 0; q < 8; ++q) v[j + q] = live ? v[j + q] * (1.0f - a[q] * a[q]) : 0.0f;
                    put8(h[l], r, c0 + j, kH, v + j);
                }
                wpart[quad][c0 + lane] = column_sums32(v, lane);
                if (l == 2) {
                    if (cb == 0) {
                        tc::tmem_ld16(tmem + 128 + lanes, v);
                        tc::wait_ld();
#pragma unroll
                        for (int j = 0; j < kOutP; j += 4)
                            *reinterpret_cast<float4*>(pp + gW4 + r * kOutP + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                    }
                } else {
                    tc::tmem_ld32(tmem + 128 + lanes + c0, v);
                    tc::wait_ld();
#pragma unroll
                    for (int j = 0; j < 32; j += 4)
                        *reinterpret_cast<float4*>(pp + (l == 1 ? gW3 : gW2) + r * kH + c0 + j) =
                            make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                }
            }
            // dW1 = dZ1^T X: a row per output
            gemms([&]() { tc::gemm_issue_op(tmem, tc::mn_major(h[0], kH), tc::mn_major(x, kInP), kInP, 8, true, true); });
            if (t < kH) pp[gb1 + t] = wpart[0][t] + wpart[1][t] + wpart[2][t] + wpart[3][t];
            if (cb == 1) {
                float v[16];
                tc::tmem_ld16(tmem + lanes, v);
                tc::wait_ld();
#pragma unroll
                for (int j = 0; j < kInP; j += 4)
                    *reinterpret_cast<float4*>(pp + gW1 + r * kInP + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (threadIdx.x < 32) tc::tmem_dealloc(tmem_slot, kTmem);
}

// parameters that exist (the padding stays zero)
__device__ __forceinline__ bool is_param(int i)
{
    if (i < ob1) return i % kInP < kIn;
    if (i >= oW4 && i < ob4) return (i - oW4) / kH < kOut;
    if (i >= ob4) return i - ob4 < kOut;
    return true;
}

// parameter i in the BF16 pack (biases are not packed)
__device__ __forceinline__ void pack_param(__nv_bfloat16* __restrict__ pack, int i, float p)
{
    int at = -1;
    if (i < ob1) at = pW1 + (int)tc::core_offset(i / kInP, i % kInP, kInP) / 2;
    else if (i >= oW2 && i < ob2) at = pW2 + (int)tc::core_offset((i - oW2) / kH, (i - oW2) % kH, kH) / 2;
    else if (i >= oW3 && i < ob3) at = pW3 + (int)tc::core_offset((i - oW3) / kH, (i - oW3) % kH, kH) / 2;
    else if (i >= oW4 && i < ob4) at = pW4 + (int)tc::core_offset((i - oW4) / kH, (i - oW4) % kH, kH) / 2;
    if (at >= 0) pack[at] = __float2bfloat16(p);
}

__global__ void mlp_pack_kernel(float* __restrict__ P, __nv_bfloat16* __restrict__ pack)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kParams) return;
    if (!is_param(i)) P[i] = 0.0f;
    pack_param(pack, i, P[i]);
}

// The tiles' partials summed in tile order in FP64, per parameter; with grad they go there, else Adam
// step `step` (from 1) follows with the new pack. The last block sums the losses.
__global__ void mlp_reduce_kernel(const float* __restrict__ part, const double* __restrict__ lpart, int nparts, int64_t B,
                                  float* __restrict__ grad, float* __restrict__ P, float* __restrict__ m,
                                  float* __restrict__ v, float lr, float b1, float b2, float eps, int step,
                                  __nv_bfloat16* __restrict__ pack, double* __restrict__ loss)
{
    __shared__ float corr[2];
    if (threadIdx.x < 2 && !grad) corr[threadIdx.x] = 1.0f - powf(threadIdx.x ? b2 : b1, (float)step);
    follow_grid();   // the kernel that wrote part and lpart
    if (blockIdx.x == gridDim.x - 1) {
        if (threadIdx.x >= 32) return;
        double s = 0.0;
        for (int q = threadIdx.x; q < nparts * kLossParts; q += 32) s += load_after(lpart + q);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) loss[0] = s / (double)(kOut * B);
        return;
    }
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kParams) return;
    int src;   // the partial that holds parameter i
    if (i < ob1) src = gW1 + i;
    else if (i < oW2) src = gb1 + (i - ob1);
    else if (i < ob2) { const int j = i - oW2, o = j / kH, k = j % kH; src = gW2 + k * kH + o; }
    else if (i < oW3) src = gb2 + (i - ob2);
    else if (i < ob3) { const int j = i - oW3, o = j / kH, k = j % kH; src = gW3 + k * kH + o; }
    else if (i < oW4) src = gb3 + (i - ob3);
    else if (i < ob4) { const int j = i - oW4, o = j / kH, k = j % kH; src = gW4 + k * kOutP + o; }
    else src = gb4 + (i - ob4);
    double s = 0.0;
#pragma unroll 8
    for (int c = 0; c < nparts; ++c) s += load_after(part + (size_t)c * kPart + src);
    const float gi = (float)s;
    if (grad) {
        grad[i] = gi;
        return;
    }
    if (!is_param(i)) return;
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / corr[0], vh = vi / corr[1];
    const float p = P[i] - lr * mh / (sqrtf(vh) + eps);
    P[i] = p;
    pack_param(pack, i, p);
}

// column c of the data set (features 0..7, then targets 8..14): mean and deviation (one block each;
// a deviation below 1e-6 max(1, |mean|) is taken as 1, so a constant column stays finite)
__global__ void mlp_fit_norm_kernel(const float* __restrict__ feat, const float* __restrict__ tgt, int64_t B,
                                    float* __restrict__ norm)
{
    __shared__ double sh[2][256];
    const int c = blockIdx.x;
    const float* src = c < kIn ? feat + c : tgt + (c - kIn);
    const int ld = c < kIn ? kIn : kOut;
    double s = 0.0, q = 0.0;
    for (int64_t r = threadIdx.x; r < B; r += blockDim.x) {
        const double v = src[r * ld];
        s += v;
        q += v * v;
    }
    sh[0][threadIdx.x] = s;
    sh[1][threadIdx.x] = q;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + o];
            sh[1][threadIdx.x] += sh[1][threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double mean = sh[0][0] / (double)B;
        const double var = fmax(sh[1][0] / (double)B - mean * mean, 0.0);
        double sd = sqrt(var);
        if (!(sd >= 1e-6 * fmax(1.0, fabs(mean)))) sd = 1.0;
        if (c < kIn) {
            norm[nFM + c] = (float)mean;
            norm[nFS + c] = (float)sd;
        } else {
            norm[nTM + c - kIn] = (float)mean;
            norm[nTS + c - kIn] = (float)sd;
        }
    }
}

}  // namespace

cudaError_t mlp_configure()
{
    cudaError_t e = cudaFuncSetAttribute(mlp_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)net_smem<1, false>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(mlp_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)net_smem<2, false>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(mlp_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)net_smem<1, true>());
    return e;
}

cudaError_t launch_mlp_forward(const float* feat, int64_t B, const float* P, const void* pack, const float* norm,
                               float* out, float* out_user, unsigned* error, cudaStream_t st)
{
    if (B <= 0) return cudaSuccess;
    const int64_t tiles = (B + kH - 1) / kH;
    const __nv_bfloat16* pk = static_cast<const __nv_bfloat16*>(pack);
    const int sms = sm_count();
    // a tile per SM is soonest done by all its threads; more tiles than SMs go two at a time
    if (tiles <= sms)
        mlp_kernel<1, false><<<(unsigned)tiles, kNetThreads, net_smem<1, false>(), st>>>(feat, nullptr, B, P, pk, norm, out,
                                                                                         out_user, nullptr, nullptr, error);
    else
        mlp_kernel<2, false><<<(unsigned)std::min<int64_t>((tiles + 1) / 2, sms), kNetThreads, net_smem<2, false>(), st>>>(
            feat, nullptr, B, P, pk, norm, out, out_user, nullptr, nullptr, error);
    return cudaGetLastError();
}

cudaError_t launch_mlp_gradient(const float* feat, const float* tgt, int64_t B, const float* P, const void* pack,
                                const float* norm, float* part, double* lpart, unsigned* error, bool follow, cudaStream_t st)
{
    if (B <= 0) return cudaSuccess;
    const int64_t tiles = (B + kH - 1) / kH;
    return launch_following(mlp_kernel<1, true>, (unsigned)std::min<int64_t>(tiles, sm_count()), kNetThreads + kLossThreads,
                            net_smem<1, true>(), follow, st, feat, tgt, B, P, static_cast<const __nv_bfloat16*>(pack), norm,
                            nullptr, nullptr, part, lpart, error);
}

cudaError_t launch_mlp_reduce(const float* part, const double* lpart, int64_t B, float* grad, float* P, float* m,
                              float* v, float lr, int step, void* pack, double* loss, cudaStream_t st)
{
    return launch_following(mlp_reduce_kernel, (unsigned)((kParams + 127) / 128 + 1), 128, 0, true, st, part, lpart,
                            (int)((B + kH - 1) / kH), B, grad, P, m, v, lr, 0.9f, 0.999f, 1e-8f, step,
                            static_cast<__nv_bfloat16*>(pack), loss);
}

cudaError_t launch_mlp_pack(float* P, void* pack, cudaStream_t st)
{
    mlp_pack_kernel<<<(kParams + 255) / 256, 256, 0, st>>>(P, static_cast<__nv_bfloat16*>(pack));
    return cudaGetLastError();
}

cudaError_t launch_mlp_fit_norm(const float* feat, const float* tgt, int64_t B, float* norm, cudaStream_t st)
{
    if (B <= 0) return cudaSuccess;
    mlp_fit_norm_kernel<<<kIn + kOut, 256, 0, st>>>(feat, tgt, B, norm);
    return cudaGetLastError();
}

}  // namespace lpdf
