// Learned coarse level: a 16 -> 128 -> 128 -> 1 ReLU network in BF16 with FP32
// accumulation, trained by mean squared error on (low-degree moments ->
// degree-n quadratic form) pairs the method itself produces.  It is a project
// addition; its nearest relative in the paper is the regression control
// variate of Section 5.4.  The multilevel estimator stays unbiased for any
// network, because the network's level is corrected by an exact level above it.
//
// One CTA handles a tile of 128 samples, forward and backward, with 512 threads:
// warps 4g .. 4g+3 hold the tile's samples (TMEM lanes) for columns 32g .. 32g+31,
// so each epilogue's work is split four ways.  The GEMMs themselves are idle
// time to the tensor cores (14 MFLOP a tile); the tile is bound by the serial
// chain weights -> shared memory, MMA, TMEM load, shared-memory stores, MMA, ...
// With 128 threads, two-byte weight copies and 80 shuffles per 16 column sums a
// training launch of 16 tiles took 54 us; with 512 threads, 16-byte copies
// and row stores and 16 shuffles it takes 21 us (forward only 30 -> 11), every
// sum in the same order.
// The GEMM-shaped steps run on the 5th-generation tensor cores: operands are
// staged in shared memory in the canonical no-swizzle K-major layout (core
// matrices of 8 rows x 16 bytes; 128 bytes to the next 8 columns, K/8 * 128
// bytes to the next 8 rows), one elected thread issues tcgen05.mma with an
// FP32 accumulator in tensor memory, tcgen05.commit arrives on an mbarrier,
// and each thread reads its accumulator row back with tcgen05.ld:
//   layer 1   D1 = X  W1^T     (M 128 samples, N 128, K 16)
//   layer 2   D2 = H1 W2^T     (M 128, N 128, K 128)
//   backward  D3 = dH2 W2      (M 128, N 128, K 128)
//             D4 = dH2^T H1    (M 128 outputs, N 128 inputs, K 128 samples)  -> dW2
//             D5 = dH1^T X     (M 128, N 16, K 128 samples)                  -> dW1
// Every mbarrier wait is bounded; a wait that runs out sets the error flag and
// the CTA stops issuing work.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "mlt_internal.h"

namespace mlt {

namespace {

constexpr int kIn = MLP_IN;
constexpr int kHid = MLP_HID;
constexpr int kTile = 128;
constexpr int kThreadsMlp = 512;
constexpr int kColsWarp = 32;                      // columns of an epilogue one warp handles
constexpr uint32_t kTmemCols = 512;

// shared-memory tiles (bytes); 1024-byte aligned offsets
constexpr uint32_t kW1s = 0;                       // 128 x 16  (W1, rows = outputs)
constexpr uint32_t kW2s = kW1s + 128 * 16 * 2;     // 128 x 128 (W2, rows = outputs)
constexpr uint32_t kW2Ts = kW2s + 128 * 128 * 2;   // 128 x 128 (W2^T, rows = inputs)
constexpr uint32_t kXs = kW2Ts + 128 * 128 * 2;    // 128 x 16  (X, rows = samples)
constexpr uint32_t kXTs = kXs + 128 * 16 * 2;      // 16 x 128  (X^T, rows = features)
constexpr uint32_t kH1s = kXTs + 16 * 128 * 2;     // 128 x 128 (H1, rows = samples)
constexpr uint32_t kH1Ts = kH1s + 128 * 128 * 2;   // 128 x 128 (H1^T, rows = units)
constexpr uint32_t kG2s = kH1Ts + 128 * 128 * 2;   // 128 x 128 (dH2, later dH1^T)
constexpr uint32_t kG2Ts = kG2s + 128 * 128 * 2;   // 128 x 128 (dH2^T, rows = units)
constexpr uint32_t kRed = kG2Ts + 128 * 128 * 2;   // 4 warps x 3 x 128 floats of column sums
constexpr uint32_t kBias = kRed + 4 * 3 * 128 * 4; // b1, b2, w3 (3 x 128 floats), then y (128 floats)
constexpr uint32_t kSmemBytes = kBias + 4 * 128 * 4;
// A tile's partial gradients: the parameters, then the loss, padded to 16 bytes.
constexpr int kPartStride = (MLP_NPARAMS + 1 + 3) & ~3;

// byte offset of element (r, k) in a canonical K-major tile with K columns
__device__ __forceinline__ uint32_t cofs(int r, int k, int K)
{
    return (uint32_t)((((r >> 3) * (K >> 3)) + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor: start, leading-dimension byte offset (next
// 8 columns), stride byte offset (next 8 rows), descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t mdesc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo & 0x3FFFFu) >> 4) << 16;
    d |= (uint64_t)((sbo & 0x3FFFFu) >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint64_t* mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(mbar))
                 : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_smem_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ bool mbar_try_wait(uint64_t* mbar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(mbar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the mbarrier phase with an iteration limit; false if it ran out.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* mbar, uint32_t parity)
{
    for (uint32_t it = 0; it < (1u << 20); ++it)
        if (mbar_try_wait(mbar, parity)) return true;
    return false;
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void st_bf16(uint8_t* base, uint32_t off, float v)
{
    *reinterpret_cast<__nv_bfloat16*>(base + off) = __float2bfloat16_rn(v);
}

// Eight values of one row, columns k .. k+7 (k a multiple of 8), which are 16
// consecutive bytes of the canonical layout.
__device__ __forceinline__ void st_row8(uint8_t* base, uint32_t off, const float* v)
{
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        memcpy(&w[i], &h, 4);
    }
    *reinterpret_cast<uint4*>(base + off) = make_uint4(w[0], w[1], w[2], w[3]);
}

// Sum of v over the warp's 32 lanes (samples) for each of 16 columns c0 .. c0+15,
// to red_w[c0 + j].  The pairs that are added are those of a butterfly over
// distances 16, 8, 4, 2, 1; at each distance a lane keeps half of its columns
// and sends the other half, 16 shuffles instead of 80.
__device__ __forceinline__ void column_sums16(const float (&v)[16], float* red_w, int c0)
{
    const int lane = threadIdx.x & 31;
    float x[8];
    const bool u16 = lane & 16, u8 = lane & 8, u4 = lane & 4, u2 = lane & 2;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        x[j] = (u16 ? v[8 + j] : v[j]) + __shfl_xor_sync(0xFFFFFFFFu, u16 ? v[j] : v[8 + j], 16);
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = (u8 ? x[4 + j] : x[j]) + __shfl_xor_sync(0xFFFFFFFFu, u8 ? x[j] : x[4 + j], 8);
#pragma unroll
    for (int j = 0; j < 2; ++j) x[j] = (u4 ? x[2 + j] : x[j]) + __shfl_xor_sync(0xFFFFFFFFu, u4 ? x[j] : x[2 + j], 4);
    x[0] = (u2 ? x[1] : x[0]) + __shfl_xor_sync(0xFFFFFFFFu, u2 ? x[0] : x[1], 2);
    x[0] += __shfl_xor_sync(0xFFFFFFFFu, x[0], 1);
    if (!(lane & 1)) red_w[c0 + (u16 ? 8 : 0) + (u8 ? 4 : 0) + (u4 ? 2 : 0) + (u2 ? 1 : 0)] = x[0];
}

struct MlpArgs {
    const float* X;        // n x 16 features
    const float* T;        // n targets (training)
    int64_t n;
    float inv_n;           // 1 / (number of samples in the loss mean)
    const __nv_bfloat16* W1b;   // 128 x 16
    const __nv_bfloat16* W2b;   // 128 x 128
    const __nv_bfloat16* W2Tb;  // 128 x 128 (transpose)
    const float* P;        // fp32 parameters (biases and w3 are read from here)
    int train;             // 0: predict y; else loss and gradient partials
    float* y;              // predictions (predict mode)
    float* part;           // per-CTA partials [gridDim.x][kPartStride]: gradient, then loss
    int* err;
};

__global__ void __launch_bounds__(kThreadsMlp, 1) mlp_tile_kernel(MlpArgs a)
{
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int failed;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int t = tid & (kTile - 1);                // sample of the tile (TMEM lane)
    const int cg = tid >> 7, cw = cg * kColsWarp;   // column group, its first column
    const int64_t row = (int64_t)blockIdx.x * kTile + t;
    const bool valid = row < a.n;
    float* red = reinterpret_cast<float*>(sm + kRed);
    float* b1 = reinterpret_cast<float*>(sm + kBias);
    float* b2 = b1 + kHid;
    float* w3 = b2 + kHid;
    float* ys = w3 + kHid;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        failed = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&mbar)), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // features into the canonical layouts; what lies before the wait reads no
    // result of an earlier kernel of a training run (X and T are its inputs)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    {
        float x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = valid ? a.X[row * kIn + 4 * cg + k] : 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            st_bf16(sm, kXs + cofs(t, 4 * cg + k, kIn), x[k]);
            if (a.train) st_bf16(sm, kXTs + cofs(4 * cg + k, t, kTile), x[k]);
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // weights, a 16-byte row of a core matrix at a time; consecutive threads fill
    // consecutive rows (no bank conflicts)
    {
        const uint4* w1 = reinterpret_cast<const uint4*>(a.W1b);
        const uint4* w2 = reinterpret_cast<const uint4*>(a.W2b);
        const uint4* w2t = reinterpret_cast<const uint4*>(a.W2Tb);
        uint4 x2[4], x2t[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = i * kThreadsMlp + tid, r = (e >> 7) * 8 + (e & 7), k8 = (e >> 3) & 15;
            x2[i] = w2[r * 16 + k8];
            if (a.train) x2t[i] = w2t[r * 16 + k8];
        }
        if (tid < 256) {
            const int r = (tid >> 4) * 8 + (tid & 7), k8 = (tid >> 3) & 1;
            *reinterpret_cast<uint4*>(sm + kW1s + cofs(r, 8 * k8, kIn)) = w1[r * 2 + k8];
        }
        if (tid < 3 * kHid) b1[tid] = a.P[(tid < kHid ? MLP_OFF_B1 : (tid < 2 * kHid ? MLP_OFF_B2 : MLP_OFF_W3)) + t];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = i * kThreadsMlp + tid, r = (e >> 7) * 8 + (e & 7), k8 = (e >> 3) & 15;
            *reinterpret_cast<uint4*>(sm + kW2s + cofs(r, 8 * k8, kHid)) = x2[i];
            if (a.train) *reinterpret_cast<uint4*>(sm + kW2Ts + cofs(r, 8 * k8, kHid)) = x2t[i];
        }
    }
    fence_smem_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tm = tmem_base;
    const uint32_t tl = tm + ((uint32_t)((warp & 3) * 32) << 16);   // this warp's 32 TMEM lanes
    const uint32_t sbase = smem_u32(sm);
    uint32_t phase = 0;

    auto issue_wait = [&](auto&& issue) -> bool {
        if (tid == 0) {
            issue();
            mma_commit(&mbar);
        }
        const bool ok = mbar_wait_bounded(&mbar, phase);
        phase ^= 1u;
        if (!ok) {
            atomicOr(a.err, 1);
            failed = 1;
        }
        fence_after();
        return ok;
    };

    // ---- layer 1: D1[b][o] = sum_k X[b][k] W1[o][k]
    bool ok = issue_wait([&] {
        mma_bf16(tm + 0, mdesc(sbase + kXs, 128, 256), mdesc(sbase + kW1s, 128, 256), idesc_bf16(128, 128), 0);
    });
    uint32_t live = 0;   // bit j: H1 (as stored, BF16) of column cw + j is positive
    if (ok) {
#pragma unroll
        for (int i = 0; i < kColsWarp / 16; ++i) {
            const int c0 = cw + 16 * i;
            float v[16];
            tmem_ld16(tl + c0, v);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                v[j] = fmaxf(v[j] + b1[c0 + j], 0.0f);
                if (a.train) {
                    const __nv_bfloat16 h = __float2bfloat16_rn(v[j]);
                    *reinterpret_cast<__nv_bfloat16*>(sm + kH1Ts + cofs(c0 + j, t, kTile)) = h;
                    if (__bfloat162float(h) > 0.0f) live |= 1u << (16 * i + j);
                }
            }
            st_row8(sm, kH1s + cofs(t, c0, kHid), v);
            st_row8(sm, kH1s + cofs(t, c0 + 8, kHid), v + 8);
        }
    }
    fence_smem_async();
    fence_before();
    __syncthreads();
    fence_after();
    // ---- layer 2: D2[b][o] = sum_k H1[b][k] W2[o][k]
    if (!failed)
        ok = issue_wait([&] {
            for (int s = 0; s < kHid / 16; ++s)
                mma_bf16(tm + 128, mdesc(sbase + kH1s + 256 * s, 128, 2048), mdesc(sbase + kW2s + 256 * s, 128, 2048),
                         idesc_bf16(128, 128), s > 0);
        });
    // the output, one chain over the 128 columns per sample (column group 0)
    if (cg == 0) {
        float y = a.P[MLP_OFF_B3];
        if (!failed) {
#pragma unroll 2
            for (int c0 = 0; c0 < kHid; c0 += 16) {
                float v[16];
                tmem_ld16(tl + 128 + c0, v);
#pragma unroll
                for (int j = 0; j < 16; ++j) y = fmaf(w3[c0 + j], fmaxf(v[j] + b2[c0 + j], 0.0f), y);
            }
        }
        ys[t] = y;
    }
    __syncthreads();
    const float y = ys[t];
    float* part = a.part + (size_t)blockIdx.x * kPartStride;
    if (!a.train) {
        if (cg == 0 && valid && !failed) a.y[row] = y;
    } else {
        const float r = valid ? (y - a.T[row]) : 0.0f;
        const float dy = 2.0f * r * a.inv_n;
        // dH2 = dy w3 (.) [pre2 > 0]; column sums dw3 = sum dy h2, db2 = sum dH2
        if (!failed) {
#pragma unroll
            for (int i = 0; i < kColsWarp / 16; ++i) {
                const int c0 = cw + 16 * i;
                float v[16], g[16];
                tmem_ld16(tl + 128 + c0, v);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float pre = v[j] + b2[c0 + j];
                    g[j] = pre > 0.0f ? dy * w3[c0 + j] : 0.0f;
                    v[j] = dy * fmaxf(pre, 0.0f);
                    st_bf16(sm, kG2Ts + cofs(c0 + j, t, kTile), g[j]);
                }
                st_row8(sm, kG2s + cofs(t, c0, kHid), g);
                st_row8(sm, kG2s + cofs(t, c0 + 8, kHid), g + 8);
                column_sums16(g, red + (warp & 3) * 384, c0);          // db2 -> red[w][0..127]
                column_sums16(v, red + (warp & 3) * 384 + 128, c0);    // dw3 -> red[w][128..255]
            }
        }
        fence_smem_async();
        fence_before();
        __syncthreads();
        fence_after();
        for (int c = tid; c < kHid; c += kThreadsMlp) {
            float s2 = 0.0f, s3 = 0.0f;
            for (int w = 0; w < 4; ++w) {
                s2 += red[w * 384 + c];
                s3 += red[w * 384 + 128 + c];
            }
            part[MLP_OFF_B2 + c] = s2;
            part[MLP_OFF_W3 + c] = s3;
        }
        // ---- D3 = dH2 W2 (dH1 before the ReLU mask) and D4 = dH2^T H1 (dW2)
        if (!failed)
            ok = issue_wait([&] {
                for (int s = 0; s < kHid / 16; ++s)
                    mma_bf16(tm + 0, mdesc(sbase + kG2s + 256 * s, 128, 2048),
                             mdesc(sbase + kW2Ts + 256 * s, 128, 2048), idesc_bf16(128, 128), s > 0);
                for (int s = 0; s < kTile / 16; ++s)
                    mma_bf16(tm + 256, mdesc(sbase + kG2Ts + 256 * s, 128, 2048),
                             mdesc(sbase + kH1Ts + 256 * s, 128, 2048), idesc_bf16(128, 128), s > 0);
            });
        __syncthreads();   // every thread has read red before it is reused
        if (!failed) {
#pragma unroll
            for (int i = 0; i < kColsWarp / 16; ++i) {
                const int c0 = cw + 16 * i;
                float v[16];
                tmem_ld16(tl + c0, v);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    v[j] = (live >> (16 * i + j)) & 1u ? v[j] : 0.0f;
                    st_bf16(sm, kG2s + cofs(c0 + j, t, kTile), v[j]);   // dH1^T over the old dH2 tile
                }
                column_sums16(v, red + (warp & 3) * 384, c0);           // db1 -> red[w][0..127]
            }
            // dW2 row t of this tile's partial
#pragma unroll
            for (int i = 0; i < kColsWarp / 16; ++i) {
                const int c0 = cw + 16 * i;
                float v[16];
                tmem_ld16(tl + 256 + c0, v);
                float4* out = reinterpret_cast<float4*>(part + MLP_OFF_W2 + t * kHid + c0);
#pragma unroll
                for (int j = 0; j < 4; ++j) out[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            }
        }
        fence_smem_async();
        fence_before();
        __syncthreads();
        fence_after();
        for (int c = tid; c < kHid; c += kThreadsMlp) {
            float s1 = 0.0f;
            for (int w = 0; w < 4; ++w) s1 += red[w * 384 + c];
            part[MLP_OFF_B1 + c] = s1;
        }
        // ---- D5 = dH1^T X (dW1), N = 16
        if (!failed)
            ok = issue_wait([&] {
                for (int s = 0; s < kTile / 16; ++s)
                    mma_bf16(tm + 384, mdesc(sbase + kG2s + 256 * s, 128, 2048),
                             mdesc(sbase + kXTs + 256 * s, 128, 2048), idesc_bf16(128, 16), s > 0);
            });
        if (!failed && cg == 0) {
            float v[16];
            tmem_ld16(tl + 384, v);
            float4* out = reinterpret_cast<float4*>(part + MLP_OFF_W1 + t * kIn);
#pragma unroll
            for (int j = 0; j < 4; ++j) out[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        }
        // loss and db3 (= sum dy): warp butterflies, then warps in order
        __syncthreads();
        if (cg == 0) {
            float l = r * r, g3 = dy;
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                l += __shfl_xor_sync(0xFFFFFFFFu, l, o);
                g3 += __shfl_xor_sync(0xFFFFFFFFu, g3, o);
            }
            if ((t & 31) == 0) {
                red[warp * 2] = l;
                red[warp * 2 + 1] = g3;
            }
        }
        __syncthreads();
        if (tid == 0) {
            float l = 0.0f, g3 = 0.0f;
            for (int w = 0; w < 4; ++w) {
                l += red[w * 2];
                g3 += red[w * 2 + 1];
            }
            part[MLP_OFF_B3] = g3;
            part[MLP_NPARAMS] = l;
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(kTmemCols));
}

constexpr int kThreadsRed = 128;

// Parameter p's partials added in tile order; eight loads in flight.
__device__ __forceinline__ double sum_tiles(const float* part, int nblk, int p)
{
    double s = 0.0;
    int b = 0;
    for (; b + 8 <= nblk; b += 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = part[(size_t)(b + u) * kPartStride + p];
#pragma unroll
        for (int u = 0; u < 8; ++u) s += v[u];
    }
    for (; b < nblk; ++b) s += part[(size_t)b * kPartStride + p];
    return s;
}

// grads[p] = sum over CTAs (in CTA order) of the partials; also the loss sum.
__global__ void __launch_bounds__(kThreadsRed) mlp_reduce_kernel(const float* part, int nblk, float* grads, double* loss)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > MLP_NPARAMS) return;
    const double s = sum_tiles(part, nblk, p);
    if (p < MLP_NPARAMS) grads[p] = (float)s;
    else *loss = s;
}

struct AdamArgs {
    float *P, *m, *v;
    float lr, b1, b2, eps, c1, c2;
    __nv_bfloat16 *W1b, *W2b, *W2Tb;
};

// The new weight p of an Adam step with gradient gp.
__device__ __forceinline__ float adam_update(const AdamArgs& a, int p, float gp)
{
    const float mp = a.b1 * a.m[p] + (1.0f - a.b1) * gp;
    const float vp = a.b2 * a.v[p] + (1.0f - a.b2) * gp * gp;
    a.m[p] = mp;
    a.v[p] = vp;
    const float w = a.P[p] - a.lr * (mp / a.c1) / (sqrtf(vp / a.c2) + a.eps);
    a.P[p] = w;
    return w;
}

// The BF16 copies the tiles read.
__device__ __forceinline__ void store_bf16(const AdamArgs& a, int p, float w)
{
    if (p >= MLP_OFF_W1 && p < MLP_OFF_W1 + kHid * kIn) {
        a.W1b[p - MLP_OFF_W1] = __float2bfloat16_rn(w);
    } else if (p >= MLP_OFF_W2 && p < MLP_OFF_W2 + kHid * kHid) {
        const int e = p - MLP_OFF_W2;
        const __nv_bfloat16 wb = __float2bfloat16_rn(w);
        a.W2b[e] = wb;
        a.W2Tb[(e & 127) * kHid + (e >> 7)] = wb;
    }
}

// A training step's end in one launch: the partials summed as above, the Adam
// step on the FP32 master parameters, and the BF16 copies (8 us for 16 tiles,
// where a sum launch and an Adam launch took 8.5 + 6).
__global__ void __launch_bounds__(kThreadsRed) mlp_reduce_adam_kernel(const float* part, int nblk, double* loss, AdamArgs a)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > MLP_NPARAMS) return;
    const double s = sum_tiles(part, nblk, p);
    if (p == MLP_NPARAMS) {
        *loss = s;
        return;
    }
    store_bf16(a, p, adam_update(a, p, (float)s));
}

// The BF16 copies of the parameters as they are.
__global__ void __launch_bounds__(kThreadsRed) mlp_copy_kernel(AdamArgs a)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < MLP_NPARAMS) store_bf16(a, p, a.P[p]);
}

}  // namespace

// A launch that may begin while the kernel before it on the stream ends
// (programmatic dependent launch): the kernels wait for it to complete before
// they read its results or write anything but their shared and tensor memory.
template <typename... P, typename... A>
static cudaError_t launch_chained(bool chained, void (*kernel)(P...), int blocks, int threads, size_t smem,
                                  cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

size_t mlp_smem_bytes() { return kSmemBytes; }
int mlp_part_stride() { return kPartStride; }

int mlp_launch_tiles(const MlpDev& D, const float* X, const float* T, int64_t n, float inv_n, int train,
                     float* y, int* err, cudaStream_t s)
{
    if (n <= 0) return MLT_OK;
    static bool attr_set = false;
    if (!attr_set) {
        MLT_CUDA_TRY(cudaFuncSetAttribute(mlp_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)kSmemBytes));
        attr_set = true;
    }
    MlpArgs a;
    a.X = X;
    a.T = T;
    a.n = n;
    a.inv_n = inv_n;
    a.W1b = D.W1b;
    a.W2b = D.W2b;
    a.W2Tb = D.W2Tb;
    a.P = D.P;
    a.train = train;
    a.y = y;
    a.part = D.part;
    a.err = err;
    const int nblk = (int)((n + kTile - 1) / kTile);
    {
        ProfScope ps(train ? "mlp_fwd_bwd" : "mlp_forward", s);
        // within a training run each kernel starts while the one before ends (its
        // first, 2, may follow the kernel that writes X and is launched plainly)
        MLT_CUDA_TRY(launch_chained(train == 3, mlp_tile_kernel, nblk, kThreadsMlp, kSmemBytes, s, a));
    }
    if (train == 1) {
        ProfScope ps("mlp_reduce", s);
        mlp_reduce_kernel<<<(MLP_NPARAMS + kThreadsRed) / kThreadsRed, kThreadsRed, 0, s>>>(D.part, nblk, D.G, D.loss);
        MLT_CUDA_TRY(cudaGetLastError());
    }
    return MLT_OK;
}

static AdamArgs adam_args(const MlpDev& D)
{
    AdamArgs a{};
    a.P = D.P;
    a.m = D.M;
    a.v = D.V;
    a.W1b = D.W1b;
    a.W2b = D.W2b;
    a.W2Tb = D.W2Tb;
    return a;
}

int mlp_reduce_adam(const MlpDev& D, int64_t n, float lr, int64_t step, cudaStream_t s)
{
    AdamArgs a = adam_args(D);
    a.lr = lr;
    a.b1 = 0.9f;
    a.b2 = 0.999f;
    a.eps = 1e-8f;
    a.c1 = 1.0f - powf(a.b1, (float)step);
    a.c2 = 1.0f - powf(a.b2, (float)step);
    ProfScope ps("mlp_reduce_adam", s);
    return cuda_fail(launch_chained(true, mlp_reduce_adam_kernel, (MLP_NPARAMS + kThreadsRed) / kThreadsRed, kThreadsRed,
                                    0, s, (const float*)D.part, (int)((n + kTile - 1) / kTile), D.loss, a),
                     "mlp_reduce_adam_kernel");
}

int mlp_refresh(const MlpDev& D, cudaStream_t s)
{
    mlp_copy_kernel<<<(MLP_NPARAMS + kThreadsRed - 1) / kThreadsRed, kThreadsRed, 0, s>>>(adam_args(D));
    return cuda_fail(cudaGetLastError(), "mlp_copy_kernel");
}

}  // namespace mlt
