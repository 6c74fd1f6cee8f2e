// Learned lambda-interpolant of the member statistics: a 4-layer MLP
// (width 256, SiLU) that models the per-lambda densities p(Q, R | lambda),
// p(log eps | lambda) and p(log omega^2 | lambda) as a softmax over the
// histogram bins, trained on the members' own histograms in BF16 with FP32
// accumulation, so that the lambda mixture (Sec. II, Eq. ensemble_hypothesis;
// Sec. IV, Eq. gaussian_lambda_pdf) can be evaluated on a fine lambda
// quadrature between the simulated lambda values.  The paper has no such
// component; the member-quadrature mixture (ens_mixture) stays the reference
// against which the surrogate's error is measured (Hellinger distance).
//
// All contractions run on the 5th-generation tensor cores (tcgen05.mma,
// kind::f16, BF16 operands from shared memory, FP32 accumulator in tensor
// memory).  Inference and the forward pass of training run one fused kernel
// (k_mlp_infer_pair); the backward pass and the weight gradients are in
// ens_train.cuh.  A plain GEMM kernel per layer (k_gemm_tc) remains as the
// layer-by-layer forward pass that checks the fused one.
#include "../../include/ens.h"
#include "ens_internal.h"
#include "ens_tc.cuh"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <type_traits>
#include <vector>

namespace ens {

constexpr int kHid = 256;     // hidden width
constexpr int kIn = 64;       // input features (padded)
constexpr int kFeat = 31;     // used input features

// ---------------------------------------------------------------------------
// GEMM: C[M][N] (FP32) = A[M][K] * B[N][K]^T, BF16 K-major operands.
// CTA tile 128 x BN, K in blocks of 64; blockIdx.z splits K (partials at
// C + z * c_split).  M % 128 == 0, N % BN == 0, K per split % 64 == 0.
// ---------------------------------------------------------------------------
template <int BN>
__global__ void __launch_bounds__(128, 1)
k_gemm_tc(const __nv_bfloat16 *__restrict__ A, int lda, const __nv_bfloat16 *__restrict__ B, int ldb,
          float *__restrict__ C, int ldc, long long c_split, int k_per_split, int *err)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = sm;                  // 128 x 64 BF16
    unsigned char *sB = sm + 128 * 128;      // BN x 64 BF16
    uint64_t *bar = reinterpret_cast<uint64_t *>(sB + BN * 128);
    uint32_t *holder = reinterpret_cast<uint32_t *>(bar + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long m0 = (long long)blockIdx.x * 128, n0 = (long long)blockIdx.y * BN;
    const long long k0 = (long long)blockIdx.z * k_per_split;
    if (warp == 0) tmem_alloc(holder, BN);
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = *holder;
    constexpr uint32_t idesc = idesc_bf16(128, BN);
    bool ok = true;
    const int nkb = k_per_split / 64;
    int kb = 0;
    for (; kb < nkb; ++kb) {
        for (int idx = tid; idx < 128 * 8; idx += 128) {
            const int r = idx >> 3, ch = idx & 7;
            const uint4 v = *reinterpret_cast<const uint4 *>(A + (m0 + r) * lda + k0 + kb * 64 + ch * 8);
            *reinterpret_cast<uint4 *>(sA + r * 128 + ((ch ^ (r & 7)) << 4)) = v;
        }
        for (int idx = tid; idx < BN * 8; idx += 128) {
            const int r = idx >> 3, ch = idx & 7;
            const uint4 v = *reinterpret_cast<const uint4 *>(B + (n0 + r) * ldb + k0 + kb * 64 + ch * 8);
            *reinterpret_cast<uint4 *>(sB + r * 128 + ((ch ^ (r & 7)) << 4)) = v;
        }
        fence_proxy_async_smem();   // generic shared stores -> tensor-core (async proxy) reads
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
            const uint64_t da = desc_sw128(sA), db = desc_sw128(sB);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                tc_mma_bf16(taddr, da + 2 * k, db + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
            tc_commit(bar);
        }
        ok = mbar_wait_warp(bar, (uint32_t)(kb & 1));
        tc_fence_after();
        if (!__syncthreads_and(ok)) {
            ok = false;
            break;
        }
    }
    if (ok) {
        const long long row = m0 + warp * 32 + lane;
        float *crow = C + blockIdx.z * c_split + row * ldc + n0;
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
            float v[32];
            tc_ld_32cols(taddr + ((uint32_t)(warp * 32) << 16) + (uint32_t)c, v);
#pragma unroll
            for (int i = 0; i < 32; i += 4)
                *reinterpret_cast<float4 *>(crow + c + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        }
    } else {
        if (tid == 0) atomicExch(err, 1);
        // the MMAs of the stuck k-block may still be running: wait (bounded) before freeing
        mbar_wait_warp(bar, (uint32_t)(kb & 1));
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(taddr, BN);
}

// dynamic shared memory: alignment slack, the two operand tiles, barrier and
// TMEM holder, plus 48 KB of unused headroom past the tiles
template <int BN>
constexpr size_t gemm_smem() { return 1024 + 128 * 128 + BN * 128 + 64 + 48 * 1024; }

static cudaError_t gemm_prepare()
{
    cudaError_t e = cudaFuncSetAttribute(k_gemm_tc<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem<256>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_gemm_tc<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem<128>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_gemm_tc<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem<64>());
    return e;
}

// C = A B^T with optional split of K; returns false on an unsupported shape
static bool gemm(const __nv_bfloat16 *A, int lda, const __nv_bfloat16 *B, int ldb, float *C, int ldc, int M, int N,
                 int K, int ksplit, int *err, cudaStream_t s)
{
    if (M % 128 || K % (64 * ksplit) || ksplit < 1) return false;
    const int kps = K / ksplit;
    const long long cs = (long long)M * ldc;
    if (N % 256 == 0) {
        dim3 grid(M / 128, N / 256, ksplit);
        k_gemm_tc<256><<<grid, 128, gemm_smem<256>(), s>>>(A, lda, B, ldb, C, ldc, cs, kps, err);
    } else if (N % 128 == 0) {
        dim3 grid(M / 128, N / 128, ksplit);
        k_gemm_tc<128><<<grid, 128, gemm_smem<128>(), s>>>(A, lda, B, ldb, C, ldc, cs, kps, err);
    } else if (N % 64 == 0) {
        dim3 grid(M / 128, N / 64, ksplit);
        k_gemm_tc<64><<<grid, 128, gemm_smem<64>(), s>>>(A, lda, B, ldb, C, ldc, cs, kps, err);
    } else {
        return false;
    }
    return true;
}

// ---------------------------------------------------------------------------
// MLP pieces (CUDA cores)
// ---------------------------------------------------------------------------
struct RowSpec {
    int nq, nt;          // bins of the Q-R histogram per axis and of each tail histogram
    int per_member;      // nq*nq + 2*nt rows per lambda value
};

// input features of (lambda, bin): scaled bin coordinates, lambda / 5, the
// PDF kind, and sin/cos(pi k s) of the bin coordinates for k = 1..4
__device__ void row_features(const RowSpec &rs, double lam, int bin, float *f)
{
    for (int i = 0; i < kIn; ++i) f[i] = 0.f;
    float q = 0.f, r = 0.f, x = 0.f;
    int kind;
    if (bin < rs.nq * rs.nq) {
        kind = 0;
        q = (float)(((bin / rs.nq) + 0.5) / rs.nq * 2.0 - 1.0);
        r = (float)(((bin % rs.nq) + 0.5) / rs.nq * 2.0 - 1.0);
    } else {
        const int b = bin - rs.nq * rs.nq;
        kind = b < rs.nt ? 1 : 2;
        x = (float)(((b % rs.nt) + 0.5) / rs.nt * 2.0 - 1.0);
    }
    f[0] = q;
    f[1] = r;
    f[2] = (float)(lam / 5.0);
    f[3] = x;
    f[4] = kind == 0 ? 1.f : 0.f;   // one-hot kind, compile-time slots (keeps f in registers)
    f[5] = kind == 1 ? 1.f : 0.f;
    f[6] = kind == 2 ? 1.f : 0.f;
    const float s3[3] = {q, r, x};
    int o = 7;
    for (int c = 0; c < 3; ++c) {
        // sin, cos (pi k s), k = 1..4: one evaluation, then the angle-addition
        // recurrence sin((k+1) a) = sin(k a) cos a + cos(k a) sin a (and the
        // cosine likewise); far below the BF16 rounding of the features
        float s1, c1;
        sincospif(s3[c], &s1, &c1);
        float sk = s1, ck = c1;
#pragma unroll
        for (int k = 1; k <= 4; ++k) {
            f[o++] = sk;
            f[o++] = ck;
            const float sn = fmaf(sk, c1, ck * s1), cn = fmaf(ck, c1, -sk * s1);
            sk = sn;
            ck = cn;
        }
    }
}

__global__ void k_features(RowSpec rs, const double *lams, int nlam, long long rows_pad, __nv_bfloat16 *X)
{
    const long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= rows_pad) return;
    float f[kIn];
    const long long real = (long long)nlam * rs.per_member;
    if (row < real) {
        row_features(rs, lams[row / rs.per_member], (int)(row % rs.per_member), f);
    } else {
        for (int i = 0; i < kIn; ++i) f[i] = 0.f;
    }
    for (int i = 0; i < kIn; ++i) X[row * kIn + i] = __float2bfloat16(f[i]);
}

// sigmoid(z) = (1 + tanh(z/2)) / 2 from the hardware tanh approximation: one
// special-function-unit operation per element (the epilogues are bound by
// that unit), relative error far below the BF16 rounding of the activations
__device__ __forceinline__ float tanh_approx(float x)
{
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// SiLU z sigmoid(z) written with h = z / 2 as h + h tanh(h): two FMAs and one
// tanh (the fused inference forms h = v / 2 + b / 2 in one FMA with halved
// biases, bit for bit the same h as (v + b) / 2)
__device__ __forceinline__ float silu_h(float h) { return fmaf(h, tanh_approx(h), h); }
__device__ __forceinline__ float silu(float z) { return silu_h(0.5f * z); }
// BF16 rounding (round to nearest, ties to even) on the integer pipe: the
// upper 16 bits of the result are the BF16 of f, bit for bit the conversion
// instruction's result for every non-NaN f (a NaN stays a NaN).
__device__ __forceinline__ uint32_t bf16_rne_bits(float f)
{
    const uint32_t u = __float_as_uint(f);
    return u + 0x7FFFu + ((u >> 16) & 1u);
}
// two BF16 values in one word: lo in bits 0..15, hi in bits 16..31
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    return __byte_perm(bf16_rne_bits(lo), bf16_rne_bits(hi), 0x7632);
}
// the same with the conversion instruction (round to nearest even, one
// instruction for the pair): the fused inference's epilogues, where it
// measured faster than the integer-pipe form
__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// a * b + c on both halves with one packed FP32x2 instruction (each half
// rounded as the scalar FMA)
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(r)
        : "l"(*reinterpret_cast<const unsigned long long *>(&a)), "l"(*reinterpret_cast<const unsigned long long *>(&b)),
          "l"(*reinterpret_cast<const unsigned long long *>(&c)));
    return *reinterpret_cast<const float2 *>(&r);
}
// SiLU of two pre-activations in the halved form h = (z + b) / 2 (see
// silu_h): the FMAs packed, one hardware tanh per element
__device__ __forceinline__ float2 silu_pair(float2 v, float2 bh)
{
    const float2 h = fma2(make_float2(0.5f, 0.5f), v, bh);
    return fma2(h, make_float2(tanh_approx(h.x), tanh_approx(h.y)), h);
}

// H = SiLU(Z + bias) as BF16 (layer-by-layer forward pass)
__global__ void k_bias_silu(const float *Z, const float *bias, long long rows, __nv_bfloat16 *H)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * kHid) return;
    H[i] = __float2bfloat16(silu(Z[i] + bias[i % kHid]));
}

// logit = H3 . w4 + b4, one warp per row
__global__ void k_head(const __nv_bfloat16 *H, const float *w4, const float *b4, long long rows, float *logit)
{
    const long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= rows) return;
    float s = 0.f;
    for (int c = lane; c < kHid; c += 32) s += __bfloat162float(H[row * kHid + c]) * w4[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) logit[row] = s + b4[0];
}

// Per group (one lambda value and one PDF kind): log-softmax over its bins,
// densities q, cross-entropy against the target probabilities p (optional),
// dlogit = (q - p) * weight.  One block per group.
__global__ void k_softmax_ce(const float *logit, const float *target, int nq, int nt, double weight, float *q,
                             float *dlogit, double *loss_partial)
{
    const int g = blockIdx.x;
    const int member = g / 3, kind = g % 3;
    const int per = nq * nq + 2 * nt;
    const long long off = (long long)member * per + (kind == 0 ? 0 : nq * nq + (kind - 1) * nt);
    const int len = kind == 0 ? nq * nq : nt;
    __shared__ float red[32];
    __shared__ float bval;
    // up to kKeep logits per thread stay in registers between the three sweeps: every
    // group of up to 8192 bins in training (1024 threads), of up to 2048 in inference
    // (256 threads), where a longer group is read three times
    constexpr int kKeep = 8;
    const bool held = len <= kKeep * (int)blockDim.x;
    float keep[kKeep];
    float mx = -INFINITY;
    if (held) {
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
            const int i = threadIdx.x + k * blockDim.x;
            keep[k] = i < len ? logit[off + i] : -INFINITY;
            mx = fmaxf(mx, keep[k]);
        }
    } else {
        for (int i = threadIdx.x; i < len; i += blockDim.x) mx = fmaxf(mx, logit[off + i]);
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = red[0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, red[w]);
        bval = m;
    }
    __syncthreads();
    mx = bval;
    float se = 0.f;
    if (held) {
#pragma unroll
        for (int k = 0; k < kKeep; ++k)
            if (threadIdx.x + k * blockDim.x < len) se += __expf(keep[k] - mx);
    } else {
        for (int i = threadIdx.x; i < len; i += blockDim.x) se += __expf(logit[off + i] - mx);
    }
    for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = se;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
        bval = s;
    }
    __syncthreads();
    const float lse = mx + __logf(bval);
    float l = 0.f;
    const float w_hi = (float)weight, w_lo = (float)(weight - (double)w_hi);
    auto out = [&](int i, float z) {
        const float lq = z - lse;
        const float qi = __expf(lq);
        if (q) q[off + i] = qi;
        if (target) {
            const float p = target[off + i];
            if (p > 0.f) l -= p * lq;
            if (dlogit) {
                // (qi - p) weight with the FP64 weight as two FP32 parts: FP64 runs on
                // two lanes per SM and clock here
                const float d = qi - p;
                dlogit[off + i] = fmaf(d, w_hi, d * w_lo);
            }
        }
    };
    if (held) {
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
            const int i = threadIdx.x + k * blockDim.x;
            if (i < len) out(i, keep[k]);
        }
    } else {
        for (int i = threadIdx.x; i < len; i += blockDim.x) out(i, logit[off + i]);
    }
    if (loss_partial) {
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = l;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
            loss_partial[g] = s * weight;
        }
    }
}

// sum of split-K partials (fixed order)
__global__ void k_sum_splits(const float *part, int splits, long long n, float *out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float s = 0.f;
    for (int z = 0; z < splits; ++z) s += part[(long long)z * n + i];
    out[i] = s;
}

// Adam on the FP32 master parameters; refresh the BF16 operand copies
struct ParamLayout {
    long long W1, b1, W2, b2, W3, b3, w4, b4, total;
};

__host__ __device__ inline ParamLayout param_layout()
{
    ParamLayout L{};
    long long o = 0;
    L.W1 = o; o += (long long)kHid * kIn;
    L.b1 = o; o += kHid;
    L.W2 = o; o += (long long)kHid * kHid;
    L.b2 = o; o += kHid;
    L.W3 = o; o += (long long)kHid * kHid;
    L.b3 = o; o += kHid;
    L.w4 = o; o += kHid;
    L.b4 = o; o += 1;
    L.total = o;
    return L;
}

__global__ void k_adam(float *p, const float *g, float *m1, float *m2, long long n, float lr, float b1, float b2,
                       float eps, float bc1, float bc2)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float a = b1 * m1[i] + (1.f - b1) * gi;
    const float b = b2 * m2[i] + (1.f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = b;
    p[i] -= lr * (a / bc1) / (sqrtf(b / bc2) + eps);
}

// byte offset of W[o][k] in the shared-memory image of a [256 out][K in]
// weight: K-blocks of 64 (32 KB each: 256 rows x 128 bytes, 128-byte swizzle)
__device__ __forceinline__ uint32_t wimg_offset(int o, int k)
{
    return (uint32_t)((k >> 6) * 32768) + sw128_offset(o, k & 63);
}

// biases and head weights of the fused kernels: read by value from the
// constant bank (inference: warp-uniform addresses, broadcasts) or from
// memory (training, where they change every step without a host round trip)
struct MlpBias {
    float b1[kHid], b2[kHid], b3[kHid];   // halved: the epilogues form (z + b) / 2 in one FMA (exact in FP32)
    float w4[kHid];
    float b4;
};

// Operands of the fused kernels from the FP32 parameters: the swizzled BF16
// shared-memory images of W1, W2, W3 (bulk copies) and the biases and head
__global__ void k_pack_weights_img(const float *p, unsigned char *img1, unsigned char *img2, unsigned char *img3,
                                   MlpBias *bias)
{
    const ParamLayout L = param_layout();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < (long long)kHid * kIn) {
        const int o = (int)(i / kIn), k = (int)(i % kIn);
        *reinterpret_cast<__nv_bfloat16 *>(img1 + wimg_offset(o, k)) = __float2bfloat16(p[L.W1 + i]);
    }
    if (i < (long long)kHid * kHid) {
        const int o = (int)(i / kHid), k = (int)(i % kHid);
        *reinterpret_cast<__nv_bfloat16 *>(img2 + wimg_offset(o, k)) = __float2bfloat16(p[L.W2 + i]);
        *reinterpret_cast<__nv_bfloat16 *>(img3 + wimg_offset(o, k)) = __float2bfloat16(p[L.W3 + i]);
    }
    if (i < kHid) {
        bias->b1[i] = 0.5f * p[L.b1 + i];
        bias->b2[i] = 0.5f * p[L.b2 + i];
        bias->b3[i] = 0.5f * p[L.b3 + i];
        bias->w4[i] = p[L.w4 + i];
    }
    if (i == 0) bias->b4 = p[L.b4];
}

// BF16 weights W1 [256][64], W2, W3 [256][256] of the layer-by-layer forward pass
__global__ void k_pack_weights(const float *p, __nv_bfloat16 *W1b, __nv_bfloat16 *W2b, __nv_bfloat16 *W3b)
{
    const ParamLayout L = param_layout();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < (long long)kHid * kIn) W1b[i] = __float2bfloat16(p[L.W1 + i]);
    if (i < (long long)kHid * kHid) {
        W2b[i] = __float2bfloat16(p[L.W2 + i]);
        W3b[i] = __float2bfloat16(p[L.W3 + i]);
    }
}

// mixture of the surrogate densities over a lambda quadrature: pdf(b) =
// sum_j w_j q(b | lambda_j) / width(b); pdf[per] = *err (one copy to the host
// brings both).  32 bins per block, the quadrature points over 8 threads per
// bin: 110 us with a thread per bin (18 blocks), FP64 and load latency.
__global__ void __launch_bounds__(256)
k_quad_mix(const float *__restrict__ q, const double *__restrict__ w, int nlam, int per, int nq, double dq, double dr,
           double dt, double *pdf, const int *err)
{
    __shared__ double part[256];
    const int b = blockIdx.x * 32 + (threadIdx.x & 31), slice = threadIdx.x >> 5;
    double s = 0.0;
    if (b < per) {
#pragma unroll 8
        for (int j = slice; j < nlam; j += 8) s += w[j] * (double)q[(long long)j * per + b];
    }
    part[threadIdx.x] = s;
    __syncthreads();
    if (slice == 0 && b < per) {
        for (int k = 1; k < 8; ++k) s += part[32 * k + threadIdx.x];
        pdf[b] = s / (b < nq * nq ? dq * dr : dt);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) pdf[per] = (double)*err;
}

__global__ void k_quad_weights(double lo, double hi, int n, int kind, double c, double Z, double mu, double sigma,
                               double *lam, double *w)
{
    // midpoint rule over [lo, hi]; cell masses of the lambda distribution
    // (one block of whole warps; the masses added up by a tree: one thread
    // adding them took 40 us for 512 points)
    __shared__ double scratch[32];
    double sum = 0.0;
    const double d = (hi - lo) / n;
    const double m = kind == 0 ? -4.5 * c * Z : mu;
    const double s = kind == 0 ? sqrt(9.0 * c * Z) : sigma;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const double a = lo + j * d, b = a + d;
        lam[j] = a + 0.5 * d;
        const double za = (a - m) / s, zb = (b - m) / s;
        w[j] = za >= 0.0 ? 0.5 * (erfc(za * 0.70710678118654752440) - erfc(zb * 0.70710678118654752440))
                         : 0.5 * (erfc(-zb * 0.70710678118654752440) - erfc(-za * 0.70710678118654752440));
        sum += w[j];
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = sum;
    __syncthreads();
    double tot = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) tot += scratch[k];
    for (int j = threadIdx.x; j < n; j += blockDim.x) w[j] = tot > 0.0 ? w[j] / tot : 0.0;
}

__global__ void k_init_params(float *p, long long n, unsigned long long seed)
{
    // He-style uniform init from a counter hash; biases zero
    const ParamLayout L = param_layout();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned long long z = seed + (unsigned long long)(i + 1) * 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    z ^= z >> 31;
    const float u = (float)((z >> 40) * (1.0 / 16777216.0)) * 2.f - 1.f;
    float scale = 0.f;
    if (i >= L.W1 && i < L.b1) scale = sqrtf(6.f / kFeat);
    else if ((i >= L.W2 && i < L.b2) || (i >= L.W3 && i < L.b3)) scale = sqrtf(6.f / kHid);
    else if (i >= L.w4 && i < L.b4) scale = sqrtf(3.f / kHid);
    p[i] = u * scale;
}

// Feature rows of the fused inference: every bin's row with lambda = 0, as
// packed BF16 pairs (the row does not depend on lambda except for input 2),
// and per lambda value the BF16 of lambda / 5, which the kernel puts in
// place of input 2 (the low half of word 1): the same bits as computing the
// row for that lambda.
__global__ void k_feature_table(RowSpec rs, const double *lams, int nlam, uint4 *ftab, uint32_t *lam5)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nlam) lam5[i] = bf16_rne_bits((float)(lams[i] / 5.0)) >> 16;
    if (i >= rs.per_member) return;
    float f[kIn];
    row_features(rs, 0.0, i, f);
    uint32_t w[kIn / 2];
#pragma unroll
    for (int j = 0; j < kIn / 2; ++j) w[j] = pack_bf16x2(f[2 * j], f[2 * j + 1]);
#pragma unroll
    for (int j = 0; j < kIn / 8; ++j) ftab[(long long)i * (kIn / 8) + j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
}

// 16 per-column parameters of an epilogue chunk as pairs, from memory by four
// 16-byte loads placed where they are written: hoisted by the compiler, or
// fetched a chunk ahead, they spill (96 registers per thread; the backward
// kernel took 344 us against 296)
struct Cols16 {
    float2 v[8];
    __device__ __forceinline__ explicit Cols16(const float *q)
    {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(v[2 * k].x), "=f"(v[2 * k].y), "=f"(v[2 * k + 1].x), "=f"(v[2 * k + 1].y)
                         : "l"(q + 4 * k));
    }
    __device__ __forceinline__ float2 operator[](int k) const { return v[k]; }
};
// the same from the constant bank or shared memory, in place
struct Cols16Ref {
    const float2 *p;
    __device__ __forceinline__ explicit Cols16Ref(const float *q) : p(reinterpret_cast<const float2 *>(q)) {}
    __device__ __forceinline__ float2 operator[](int k) const { return p[k]; }
};

// The training kernels keep the halved biases of the first two layers behind
// their barriers in shared memory (all that is left of it); the third layer's
// and the head's come from memory.  The operand tiles need 1024-byte alignment and leave no slack to align
// by hand: the kernels check it.
constexpr size_t kTrainSmem = 2 * 65536 + 3 * 32768 + 256 + 2 * kHid * sizeof(float);

// Images of the training operands (activations and their gradients): per 64-row half tile its 64-column
// blocks one after another, 64 rows x 128 bytes each, swizzled as in shared
// memory, so a half tile is one bulk copy.  `blocks`: 4 (256 columns) or 1.
__device__ __forceinline__ unsigned char *image_row(unsigned char *img, long long tile, int row, int block, int blocks)
{
    return img + (((tile * 2 + (row >> 6)) * blocks + block) << 13) + (row & 63) * 128;
}
constexpr long long kHalfTile = 4 * 8192;   // bytes of a 64-row half tile of 256 columns

// 32 bytes (16 BF16 columns from column 16 part of a 64-column block) of row r
// into the swizzled 128-byte row at `dst`: two 16-byte words that the swizzle
// keeps inside one 32-byte sector, in one 32-byte store
__device__ __forceinline__ void store_row32(unsigned char *dst, int r, int part, const uint32_t (&w)[8])
{
    const bool sw = r & 1;
    unsigned char *p = dst + ((part ^ ((r >> 1) & 3)) << 5);
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(sw ? w[4] : w[0]),
                 "r"(sw ? w[5] : w[1]), "r"(sw ? w[6] : w[2]), "r"(sw ? w[7] : w[3]), "r"(sw ? w[0] : w[4]),
                 "r"(sw ? w[1] : w[5]), "r"(sw ? w[2] : w[6]), "r"(sw ? w[3] : w[7])
                 : "memory");
}

// ---------------------------------------------------------------------------
// Fused inference: features -> 3 x (tcgen05 GEMM + bias + SiLU) -> head, per
// 128-row tile; activations never leave the SM.  Persistent CTAs, two tiles
// in flight per CTA (tiles A and B of a tile pair), so that the tensor cores
// work on one tile while the epilogue warps work on the other.  Per CTA:
//   TMEM          one 256-column FP32 accumulator per tile (512 columns)
//   shared memory H_A, H_B: 4 K-blocks of 128 rows x 64 BF16 each (64 KB
//                 each; K-block 0 also holds the tile's features, K-block 1
//                 the head's partial sums); a ring of three 32 KB slots for
//                 the weight K-blocks, streamed in the order they are used
//                 (W1, W2 blocks 0-3, W3 blocks 0-3 per tile pair)
//   warps 0-15    epilogues, in the order E1(A) E1(B) E2(A) E2(B) head(A)
//                 head(B): TMEM -> bias + SiLU -> BF16 K-blocks of the next
//                 layer's A operand (one arrival per warp and chunk), the
//                 head's dot product with w4; the next pair's features
//   warp 16       MMA issue: per hidden layer A0 A1 A2 B0 B1 B2 A3 B3
//                 (K-block c of tile X once its chunk c is written and the
//                 block has landed); a weight slot is released by a commit
//                 after the B tile's MMAs on it
//   warp 17       bulk copies of the weight K-blocks into free slots
// An accumulator is reused by the next layer of its tile: every epilogue
// warp loads all four chunks of it before its first chunk arrival, so the
// next layer's first MMA (which overwrites it) waits on that arrival.
// Epilogue warp w reads TMEM lanes 32 (w mod 4) .. +31 (its rows) and, in
// chunk c, columns 64 c + 16 (w / 4) .. +15; SiLU(z + b) = h + h tanh(h)
// with h = z / 2 + b / 2 (halved biases), the activations rounded to BF16,
// the head's partial sums over each warp's columns added in a fixed order.
// Every wait is bounded; a role whose wait gives up leaves its loop, sets
// *err, and the CTA drains its copies and MMAs before freeing the TMEM.
// ---------------------------------------------------------------------------
constexpr int kPairWarps = 16;                           // epilogue warps
constexpr int kPairThreads = 32 * (kPairWarps + 2);      // + MMA warp + copy warp
constexpr int kPairSlots = 3;                            // weight K-block slots
constexpr size_t kPairSmem = 1024 + 2 * 65536 + (size_t)kPairSlots * 32768 + 256;

// TRAIN (the forward pass of training): biases and head from memory (*mem),
// where they change every step without a host round trip, instead of the
// kernel parameters, and H1, H2 of every tile also written to the images that
// the backward pass and the weight gradients read.
template <bool TRAIN>
__global__ void __launch_bounds__(kPairThreads, 1)
k_mlp_infer_pair(RowSpec rs, const uint4 *__restrict__ ftab, const uint32_t *__restrict__ lam5, long long real,
                 long long ntiles, const unsigned char *__restrict__ img1, const unsigned char *__restrict__ img2,
                 const unsigned char *__restrict__ img3, const __grid_constant__ MlpBias val,
                 const MlpBias *__restrict__ mem, unsigned char *__restrict__ imgH1,
                 unsigned char *__restrict__ imgH2, float *__restrict__ logit, int *err)
{
    const MlpBias &bias = TRAIN ? *mem : val;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *sm = smem_raw;
    if constexpr (TRAIN) {
        if (smem_u32(sm) & 1023u) {
            if (threadIdx.x == 0) atomicExch(err, 1);
            return;
        }
    } else {
        sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    }
    unsigned char *const sH0 = sm, *const sH1 = sm + 65536;   // H of tile A, B
    unsigned char *const sW = sm + 2 * 65536;                  // weight slots
    uint64_t *bars = reinterpret_cast<uint64_t *>(sW + kPairSlots * 32768);
    uint64_t *full = bars;                       // [3] slot holds its K-block
    uint64_t *empty = bars + 3;                  // [3] slot's MMAs done (both tiles)
    uint64_t *accr = bars + 6;                   // [2] a layer's MMAs of tile X done
    uint64_t *chunk = bars + 8;                  // [2][4] chunk c of tile X written
    uint64_t *feat = bars + 16;                  // [2] features written, accumulator read
    uint64_t *drain = bars + 18;                 // every issued MMA done
    uint64_t *partd = bars + 19;                 // [2] head partial sums of tile X written
    uint32_t *holder = reinterpret_cast<uint32_t *>(bars + 21);
    float *sB = reinterpret_cast<float *>(bars + 32);   // TRAIN: b1, b2
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) tmem_alloc(holder, 512);
    if (tid == 0) {
        for (int s = 0; s < kPairSlots; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int x = 0; x < 2; ++x) {
            mbar_init(&accr[x], 1);
            mbar_init(&feat[x], kPairWarps);
            mbar_init(&partd[x], kPairWarps);
        }
        for (int i = 0; i < 8; ++i) mbar_init(&chunk[i], kPairWarps);
        mbar_init(drain, 1);
        fence_mbar_init();
    }
    if constexpr (TRAIN) {
        for (int i = tid; i < kHid; i += kPairThreads) {
            sB[i] = bias.b1[i];
            sB[kHid + i] = bias.b2[i];
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = *holder;
    const float *const hb1 = TRAIN ? sB : bias.b1, *const hb2 = TRAIN ? sB + kHid : bias.b2;
    const long long npairs = (ntiles + 1) / 2;
    auto slot = [&](long long q) { return sW + (int)(q % kPairSlots) * 32768; };
    bool ok = true;
    if (warp == kPairWarps + 1) {
        // ---- copy warp: K-block q of the sequence into slot q mod 3 once the
        // block that held it (q - 3) is released ----
        long long q = 0;
        long long lastq[kPairSlots] = {-1, -1, -1};
        for (long long p = blockIdx.x; ok && p < npairs; p += gridDim.x) {
            for (int j = 0; j < 9; ++j, ++q) {
                const int s = (int)(q % kPairSlots);
                if (q >= kPairSlots) ok = mbar_wait_warp(&empty[s], (uint32_t)(((q / kPairSlots) & 1) ^ 1));
                if (!ok) break;
                if (lane == 0) {
                    const unsigned char *src = j == 0 ? img1 : (j < 5 ? img2 + (j - 1) * 32768 : img3 + (j - 5) * 32768);
                    mbar_arrive_expect_tx(&full[s], 32768);
                    bulk_g2s(sW + s * 32768, src, 32768, &full[s]);
                }
                lastq[s] = q;
            }
        }
        if (!ok) {
            // the copies this warp issued complete before the CTA ends (bounded)
            for (int s = 0; s < kPairSlots; ++s)
                if (lastq[s] >= 0) mbar_wait_warp(&full[s], (uint32_t)((lastq[s] / kPairSlots) & 1));
        }
    } else if (warp == kPairWarps) {
        // ---- MMA warp ----
        constexpr uint32_t idesc = idesc_bf16(128, kHid);
        uint32_t nfeat[2] = {0, 0}, nchunk[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        long long q = 0;
        auto wfull = [&](long long qq) {
            return mbar_wait_warp(&full[qq % kPairSlots], (uint32_t)((qq / kPairSlots) & 1));
        };
        auto wchunk = [&](int x, int c) {
            const bool r = mbar_wait_warp(&chunk[4 * x + c], nchunk[4 * x + c] & 1);
            if (r) ++nchunk[4 * x + c];
            return r;
        };
        // the four K = 16 MMAs of one K-block of tile x (a: its A operand block)
        auto mma_kb = [&](int x, const unsigned char *a, const unsigned char *b, bool first) {
            if (lane == 0) {
                tc_fence_after();
                const uint64_t da = desc_sw128(a), db = desc_sw128(b);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    tc_mma_bf16(taddr + 256u * x, da + 2 * k, db + 2 * k, idesc, (!first || k > 0) ? 1u : 0u);
            }
            __syncwarp();
        };
        for (long long p = blockIdx.x; ok && p < npairs; p += gridDim.x) {
            // layer 1 (K = 64: one block, the features)
            ok = wfull(q) && mbar_wait_warp(&feat[0], nfeat[0] & 1);
            if (!ok) break;
            ++nfeat[0];
            mma_kb(0, sH0, slot(q), true);
            if (lane == 0) tc_commit(&accr[0]);
            ok = mbar_wait_warp(&feat[1], nfeat[1] & 1);
            if (!ok) break;
            ++nfeat[1];
            mma_kb(1, sH1, slot(q), true);
            if (lane == 0) {
                tc_commit(&accr[1]);
                tc_commit(&empty[q % kPairSlots]);
            }
            ++q;
            // layers 2 and 3: A0 A1 A2 B0 B1 B2 A3 B3
            for (int l = 0; l < 2 && ok; ++l, q += 4) {
                for (int c = 0; c < 3 && ok; ++c) {
                    ok = wfull(q + c) && wchunk(0, c);
                    if (ok) mma_kb(0, sH0 + c * 16384, slot(q + c), c == 0);
                }
                for (int c = 0; c < 3 && ok; ++c) {
                    ok = wchunk(1, c);
                    if (ok) {
                        mma_kb(1, sH1 + c * 16384, slot(q + c), c == 0);
                        if (lane == 0) tc_commit(&empty[(q + c) % kPairSlots]);
                    }
                }
                if (ok) ok = wfull(q + 3) && wchunk(0, 3);
                if (ok) {
                    mma_kb(0, sH0 + 3 * 16384, slot(q + 3), false);
                    if (lane == 0) tc_commit(&accr[0]);
                    ok = wchunk(1, 3);
                }
                if (ok) {
                    mma_kb(1, sH1 + 3 * 16384, slot(q + 3), false);
                    if (lane == 0) {
                        tc_commit(&accr[1]);
                        tc_commit(&empty[(q + 3) % kPairSlots]);
                    }
                }
            }
        }
        // every MMA this warp issued completes before the TMEM is freed (bounded)
        if (lane == 0) tc_commit(drain);
        __syncwarp();
        mbar_wait_warp(drain, 0);
    } else {
        // ---- epilogue warps ----
        const int quarter = warp & 3, cpart = warp >> 2;
        const int row = quarter * 32 + lane;                  // this thread's TMEM lane = tile row
        const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
        uint32_t nacc[2] = {0, 0}, npart[2] = {0, 0};
        // the features of tile t into K-block 0 of H, spread over every
        // epilogue thread: row tid / 4, 16-byte words 2 (tid mod 4) and the
        // next one; the bin's row of the table with lambda / 5 in place of
        // input 2 (the low half of word 1)
        auto features = [&](long long t, unsigned char *H) {
            const int r = tid >> 2, j0 = (tid & 3) * 2;
            const long long rr = t * 128 + r;
            uint4 v0 = make_uint4(0u, 0u, 0u, 0u), v1 = v0;
            if (rr < real) {
                const int li = (int)(rr / rs.per_member);
                const long long bin = rr - (long long)li * rs.per_member;
                v0 = ftab[bin * (kIn / 8) + j0];
                v1 = ftab[bin * (kIn / 8) + j0 + 1];
                if (j0 == 0) v0.y = (v0.y & 0xFFFF0000u) | lam5[li];
            }
            *reinterpret_cast<uint4 *>(H + sw128_offset(r, 8 * j0)) = v0;
            *reinterpret_cast<uint4 *>(H + sw128_offset(r, 8 * j0 + 8)) = v1;
        };
        // the first pair's features
        features(2 * (long long)blockIdx.x, sH0);
        features(2 * (long long)blockIdx.x + 1, sH1);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
            mbar_arrive(&feat[0]);
            mbar_arrive(&feat[1]);
        }
        // epilogue of a hidden layer of tile x (bias bv): H_x chunk c, arrival c
        // (every chunk's load is waited for before the first arrival: the
        // next layer's first MMA overwrites the whole accumulator)
        auto epilogue = [&](int x, const float *bv, unsigned char *img, long long t) {
            if (!(ok && mbar_wait_warp(&accr[x], nacc[x] & 1))) return false;
            ++nacc[x];
            tc_fence_after();
            unsigned char *H = x ? sH1 : sH0;
            const uint32_t acc = taddr + 256u * x + lanes + (uint32_t)(16 * cpart);
            uint32_t r[4][16];
#pragma unroll
            for (int c = 0; c < 4; ++c) tc_ld_16cols_issue(acc + 64u * c, r[c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) tc_ld_wait16(r[c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t *rc = r[c];
                const Cols16Ref b(bv + 64 * c + 16 * cpart);
                uint32_t w[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float2 y = silu_pair(make_float2(__uint_as_float(rc[2 * k]), __uint_as_float(rc[2 * k + 1])), b[k]);
                    w[k] = cvt_bf16x2(y.x, y.y);
                }
                unsigned char *blk = H + c * 16384;
                *reinterpret_cast<uint4 *>(blk + sw128_offset(row, 16 * cpart)) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4 *>(blk + sw128_offset(row, 16 * cpart + 8)) =
                    make_uint4(w[4], w[5], w[6], w[7]);
                fence_proxy_async_smem();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&chunk[4 * x + c]);
                if constexpr (TRAIN) {
                    if (t < ntiles) store_row32(image_row(img, t, row, c, 4), row, cpart, w);
                }
            }
            return true;
        };
        // head of tile x (tile index t): logit = sum_c BF16(SiLU(z3 + b3)) w4 + b4.
        // Every warp writes its partial sums and arrives on partd[x]; warps
        // 0-3 (one row each, threads 0..127) wait for them and write the
        // logits; every warp then puts its share of the next pair's features
        // of this slot (tile tn) into K-block 0.  The feature arrival comes
        // last: the next layer-1 MMAs (which overwrite the accumulator) and
        // the epilogues after them (which overwrite K-block 1, the partial
        // sums) wait for it.
        auto head = [&](int x, long long t, bool next, long long tn) {
            if (!(ok && mbar_wait_warp(&accr[x], nacc[x] & 1))) return false;
            ++nacc[x];
            tc_fence_after();
            unsigned char *H = x ? sH1 : sH0;
            float *part = reinterpret_cast<float *>(H + 16384);   // [4][128] in K-block 1
            const uint32_t acc = taddr + 256u * x + lanes + (uint32_t)(16 * cpart);
            uint32_t r[4][16];
#pragma unroll
            for (int c = 0; c < 4; ++c) tc_ld_16cols_issue(acc + 64u * c, r[c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) tc_ld_wait16(r[c]);
            float2 sum = make_float2(0.f, 0.f);   // even and odd columns
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t *rc = r[c];
                using Cols = std::conditional_t<TRAIN, Cols16, Cols16Ref>;
                const Cols b3(bias.b3 + 64 * c + 16 * cpart), w4(bias.w4 + 64 * c + 16 * cpart);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float2 y = silu_pair(make_float2(__uint_as_float(rc[2 * k]), __uint_as_float(rc[2 * k + 1])), b3[k]);
                    const uint32_t hb = cvt_bf16x2(y.x, y.y);   // the activations rounded to BF16
                    sum = fma2(make_float2(__uint_as_float(hb << 16), __uint_as_float(hb & 0xFFFF0000u)), w4[k], sum);
                }
            }
            part[cpart * 128 + row] = sum.x + sum.y;
            __syncwarp();
            if (lane == 0) mbar_arrive(&partd[x]);
            bool good = true;
            if (warp < 4) {
                good = mbar_wait_warp(&partd[x], npart[x] & 1);
                if (good && t * 128 + tid < real)
                    logit[t * 128 + tid] = ((part[tid] + part[128 + tid]) + (part[256 + tid] + part[384 + tid])) + bias.b4;
            }
            ++npart[x];
            if (good && next) features(tn, H);
            fence_proxy_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0 && good) mbar_arrive(&feat[x]);
            return good;
        };
        for (long long p = blockIdx.x; p < npairs; p += gridDim.x) {
            const long long pn = p + gridDim.x;
            const bool next = pn < npairs;
            ok = epilogue(0, hb1, imgH1, 2 * p);
            ok = epilogue(1, hb1, imgH1, 2 * p + 1);
            ok = epilogue(0, hb2, imgH2, 2 * p);
            ok = epilogue(1, hb2, imgH2, 2 * p + 1);
            ok = head(0, 2 * p, next, 2 * pn);
            ok = head(1, 2 * p + 1, next, 2 * pn + 1);
            if (!ok) break;   // (each warp on its own: no CTA-wide barrier in the loop)
        }
    }
    if (!ok && lane == 0) atomicExch(err, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(taddr, 512);
}

}  // namespace ens

#include "ens_train.cuh"

using namespace ens;

// ---------------------------------------------------------------------------
// surrogate object
// ---------------------------------------------------------------------------
// device memory that grows on demand and is kept for later calls
struct Buf {
    void *p = nullptr;
    size_t cap = 0;
    bool need(size_t bytes)
    {
        if (bytes <= cap) return true;
        if (p) cudaFree(p);
        p = nullptr;
        cap = 0;
        if (cudaMalloc(&p, bytes) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        cap = bytes;
        return true;
    }
    template <class T>
    T *as() const { return static_cast<T *>(p); }
    ~Buf() { if (p) cudaFree(p); }
};

struct ens_surrogate {
    cudaStream_t s = nullptr;
    ParamLayout L{};
    float *p = nullptr, *g = nullptr, *m1 = nullptr, *m2 = nullptr;
    int *err = nullptr;
    long long steps = 0;
    double *lam = nullptr, *wq = nullptr, *pdf = nullptr;
    uint32_t *lam5 = nullptr;       // BF16 of lambda / 5 per lambda value
    unsigned char *img = nullptr;   // swizzled W1 | W2 | W3 images of the fused kernels
    MlpBias *bias = nullptr;        // biases and head in device memory (with img)
    MlpBias hbias{};                // the same on the host, valid while hbias_ok
    bool hbias_ok = false;
    int sms = 0;
    Buf logit, q, ftab, loss;                                  // every path
    Buf counts, target, dlogit, images, part, head_part;       // training
    Buf X, H, Z, Wb;                                           // layer-by-layer forward pass
};

namespace {

constexpr int kMaxSplit = 32;

cudaError_t train_prepare()
{
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_mlp_infer_pair<false>, attr, (int)kPairSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_infer_pair<true>, attr, (int)kTrainSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_back, attr, (int)kTrainSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_wgrad, attr, (int)kWgSmem);
    return e;
}

int blocks(long long n, int t) { return (int)((n + t - 1) / t); }
long long pad128(long long r) { return (r + 127) / 128 * 128; }

// rows' logits and densities, the feature table and the group losses
bool alloc_rows(ens_surrogate *S, const RowSpec &rs, long long rows, int groups)
{
    return S->logit.need(sizeof(float) * rows) && S->q.need(sizeof(float) * rows) &&
           S->ftab.need(sizeof(uint4) * (kIn / 8) * rs.per_member) && S->loss.need(sizeof(double) * (groups + 1));
}

// CTAs per layer of the weight-gradient kernel: one wave over the SMs, in
// proportion to the bytes of a half tile (64 + 64 KB, 64 + 64 KB, 64 + 16 KB)
WgradSplits wgrad_splits(const ens_surrogate *S, long long halves)
{
    const int sms = std::max(S->sms, 3);
    WgradSplits sp;
    sp.n[2] = sp.n[1] = std::max(1, sms * 8 / 21);
    sp.n[0] = std::max(1, sms - 2 * sp.n[1]);
    for (int &n : sp.n) n = (int)std::min<long long>(n, halves);
    return sp;
}

TrainImages train_images(const ens_surrogate *S, long long rows)
{
    const size_t b = sizeof(__nv_bfloat16) * rows * kHid;
    unsigned char *p = S->images.as<unsigned char>();
    return TrainImages{p + 5 * b, p, p + b, p + 2 * b, p + 3 * b, p + 4 * b};
}

bool alloc_train(ens_surrogate *S, long long rows)
{
    const WgradSplits sp = wgrad_splits(S, rows / 64);
    return S->target.need(sizeof(float) * rows) && S->dlogit.need(sizeof(float) * rows) &&
           S->images.need(sizeof(__nv_bfloat16) * rows * (5 * kHid + kIn)) &&
           S->part.need(sizeof(float) * kPartStride * (sp.n[0] + sp.n[1] + sp.n[2])) &&
           S->head_part.need(sizeof(float) * kHeadPart * std::max(S->sms, 1));
}

// the fused kernels' operands after a change of the parameters
void pack_params(ens_surrogate *S)
{
    k_pack_weights_img<<<blocks((long long)kHid * kHid, 256), 256, 0, S->s>>>(S->p, S->img, S->img + 32768,
                                                                              S->img + 32768 + 131072, S->bias);
    S->hbias_ok = false;
}

// buffers of the layer-by-layer forward pass
bool alloc_layers(ens_surrogate *S, long long rows)
{
    return S->X.need(sizeof(__nv_bfloat16) * rows * kIn) && S->H.need(sizeof(__nv_bfloat16) * rows * kHid) &&
           S->Z.need(sizeof(float) * rows * kHid) && S->Wb.need(sizeof(__nv_bfloat16) * (kHid * kIn + 2 * kHid * kHid));
}

// layer-by-layer forward pass (one GEMM launch per layer) for `rows` padded
// rows of the lambda values in S->lam: the check of the fused kernels
bool forward_layers(ens_surrogate *S, const RowSpec &rs, int nlam, long long rows)
{
    cudaStream_t s = S->s;
    const ParamLayout &L = S->L;
    __nv_bfloat16 *X = S->X.as<__nv_bfloat16>(), *H = S->H.as<__nv_bfloat16>();
    __nv_bfloat16 *W1 = S->Wb.as<__nv_bfloat16>(), *W2 = W1 + kHid * kIn, *W3 = W2 + kHid * kHid;
    float *Z = S->Z.as<float>();
    k_features<<<blocks(rows, 256), 256, 0, s>>>(rs, S->lam, nlam, rows, X);
    k_pack_weights<<<blocks((long long)kHid * kHid, 256), 256, 0, s>>>(S->p, W1, W2, W3);
    if (!gemm(X, kIn, W1, kIn, Z, kHid, (int)rows, kHid, kIn, 1, S->err, s)) return false;
    k_bias_silu<<<blocks(rows * kHid, 256), 256, 0, s>>>(Z, S->p + L.b1, rows, H);
    if (!gemm(H, kHid, W2, kHid, Z, kHid, (int)rows, kHid, kHid, 1, S->err, s)) return false;
    k_bias_silu<<<blocks(rows * kHid, 256), 256, 0, s>>>(Z, S->p + L.b2, rows, H);
    if (!gemm(H, kHid, W3, kHid, Z, kHid, (int)rows, kHid, kHid, 1, S->err, s)) return false;
    k_bias_silu<<<blocks(rows * kHid, 256), 256, 0, s>>>(Z, S->p + L.b3, rows, H);
    k_head<<<blocks(rows * 32, 256), 256, 0, s>>>(H, S->p + L.w4, S->p + L.b4, rows, S->logit.as<float>());
    return true;
}

// feature table and lambda words of the lambda values in S->lam
void feature_table(ens_surrogate *S, const RowSpec &rs, int nlam)
{
    k_feature_table<<<blocks(std::max(rs.per_member, nlam), 256), 256, 0, S->s>>>(rs, S->lam, nlam,
                                                                                  S->ftab.as<uint4>(), S->lam5);
}

// the fused forward kernel over `real` rows (one CTA per tile pair, at most
// one per SM) into S->logit; with images: the forward pass of training
void launch_infer(ens_surrogate *S, const RowSpec &rs, long long real, const TrainImages *im)
{
    const long long ntiles = (real + 127) / 128;
    const int grid = (int)std::min<long long>((ntiles + 1) / 2, S->sms > 0 ? S->sms : 1);
    unsigned char *i1 = S->img, *i2 = S->img + 32768, *i3 = S->img + 32768 + 131072;
    const uint4 *ftab = S->ftab.as<uint4>();
    if (im)
        k_mlp_infer_pair<true><<<grid, kPairThreads, kTrainSmem, S->s>>>(rs, ftab, S->lam5, real, ntiles, i1, i2, i3,
                                                                        S->hbias, S->bias, im->H1, im->H2,
                                                                        S->logit.as<float>(), S->err);
    else
        k_mlp_infer_pair<false><<<grid, kPairThreads, kPairSmem, S->s>>>(rs, ftab, S->lam5, real, ntiles, i1, i2, i3,
                                                                         S->hbias, S->bias, nullptr, nullptr,
                                                                         S->logit.as<float>(), S->err);
}

// biases and head on the host (kernel parameters of the inference kernel)
bool host_bias(ens_surrogate *S)
{
    if (S->hbias_ok) return true;
    S->hbias_ok = cudaMemcpyAsync(&S->hbias, S->bias, sizeof(MlpBias), cudaMemcpyDeviceToHost, S->s) == cudaSuccess &&
                  cudaStreamSynchronize(S->s) == cudaSuccess;
    return S->hbias_ok;
}

// fused inference of `real` rows (lambda values in S->lam) into S->logit
bool forward_fused(ens_surrogate *S, const RowSpec &rs, long long real)
{
    if (!host_bias(S)) return false;
    feature_table(S, rs, (int)(real / rs.per_member));
    launch_infer(S, rs, real, nullptr);
    return cudaGetLastError() == cudaSuccess;
}

// loss (loss null: not wanted) and gradient of the batch in S->lam, S->target
void loss_grad_kernels(ens_surrogate *S, const RowSpec &rs, int n, long long rows, long long real, bool want_loss)
{
    cudaStream_t s = S->s;
    const double wgt = 1.0 / (3.0 * n);
    const TrainImages im = train_images(S, rows);
    launch_infer(S, rs, real, &im);
    // one wave of large groups: 1024 threads each
    k_softmax_ce<<<3 * n, 1024, 0, s>>>(S->logit.as<float>(), S->target.as<float>(), rs.nq, rs.nt, wgt, nullptr,
                                       S->dlogit.as<float>(), want_loss ? S->loss.as<double>() : nullptr);
    const long long ntiles = rows / 128;
    const int grid = (int)std::min<long long>(ntiles, S->sms > 0 ? S->sms : 1);
    k_mlp_back<<<grid, kPairThreads, kTrainSmem, s>>>(rs, S->ftab.as<uint4>(), S->lam5, real, ntiles, S->img,
                                                     S->img + 32768, S->img + 32768 + 131072, S->bias,
                                                     S->dlogit.as<float>(), im, S->head_part.as<float>(), S->err);
    const WgradSplits sp = wgrad_splits(S, rows / 64);
    k_mlp_wgrad<<<sp.n[0] + sp.n[1] + sp.n[2], kWgThreads, kWgSmem, s>>>(im, rows / 64, sp, S->part.as<float>(), S->err);
    k_grad_sum<<<blocks(S->L.total, 256), 256, 0, s>>>(S->part.as<float>(), sp, S->head_part.as<float>(), grid, S->g,
                                                       S->err, S->loss.as<double>() + 3 * n);
}

}  // namespace

extern "C" {

ens_status ens_surrogate_create(uint64_t seed, void *stream, ens_surrogate **out)
{
    if (!out) return ENS_EINVAL;
    *out = nullptr;
    ens_surrogate *S = new ens_surrogate();
    S->s = (cudaStream_t)stream;
    S->L = param_layout();
    const long long n = S->L.total;
    bool ok = gemm_prepare() == cudaSuccess;
    ok = ok && cudaMalloc(&S->p, sizeof(float) * n) == cudaSuccess && cudaMalloc(&S->g, sizeof(float) * n) == cudaSuccess &&
         cudaMalloc(&S->m1, sizeof(float) * n) == cudaSuccess && cudaMalloc(&S->m2, sizeof(float) * n) == cudaSuccess &&
         cudaMalloc(&S->lam, sizeof(double) * 4096) == cudaSuccess &&
         cudaMalloc(&S->lam5, sizeof(uint32_t) * 4096) == cudaSuccess &&
         cudaMalloc(&S->bias, sizeof(MlpBias)) == cudaSuccess &&
         cudaMalloc(&S->err, sizeof(int)) == cudaSuccess && cudaMalloc(&S->wq, sizeof(double) * 4096) == cudaSuccess &&
         cudaMalloc(&S->pdf, sizeof(double) * ((1 << 20) + 1)) == cudaSuccess &&
         cudaMalloc(&S->img, 32768 + 2 * 131072) == cudaSuccess &&
         train_prepare() == cudaSuccess;
    int dev = 0;
    ok = ok && cudaGetDevice(&dev) == cudaSuccess &&
         cudaDeviceGetAttribute(&S->sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
    if (!ok) {
        ens_surrogate_destroy(S);
        return ENS_ENOMEM;
    }
    cudaMemsetAsync(S->err, 0, sizeof(int), S->s);
    cudaMemsetAsync(S->m1, 0, sizeof(float) * n, S->s);
    cudaMemsetAsync(S->m2, 0, sizeof(float) * n, S->s);
    k_init_params<<<blocks(n, 256), 256, 0, S->s>>>(S->p, n, seed);
    pack_params(S);
    if (cudaStreamSynchronize(S->s) != cudaSuccess) {
        ens_surrogate_destroy(S);
        return ENS_ECUDA;
    }
    *out = S;
    return ENS_OK;
}

ens_status ens_surrogate_destroy(ens_surrogate *S)
{
    if (!S) return ENS_EINVAL;
    cudaStreamSynchronize(S->s);
    for (void *p : {(void *)S->p, (void *)S->g, (void *)S->m1, (void *)S->m2, (void *)S->err, (void *)S->wq,
                    (void *)S->pdf, (void *)S->img, (void *)S->bias, (void *)S->lam, (void *)S->lam5})
        if (p) cudaFree(p);
    delete S;
    return ENS_OK;
}

size_t ens_surrogate_param_count(void) { return (size_t)param_layout().total; }

ens_status ens_surrogate_get_params(ens_surrogate *S, float *host)
{
    if (!S || !host) return ENS_EINVAL;
    if (cudaMemcpyAsync(host, S->p, sizeof(float) * S->L.total, cudaMemcpyDeviceToHost, S->s) != cudaSuccess ||
        cudaStreamSynchronize(S->s) != cudaSuccess)
        return ENS_ECUDA;
    return ENS_OK;
}

ens_status ens_surrogate_set_params(ens_surrogate *S, const float *host)
{
    if (!S || !host) return ENS_EINVAL;
    if (cudaMemcpyAsync(S->p, host, sizeof(float) * S->L.total, cudaMemcpyHostToDevice, S->s) != cudaSuccess)
        return ENS_ECUDA;
    pack_params(S);
    if (cudaStreamSynchronize(S->s) != cudaSuccess) return ENS_ECUDA;
    return ENS_OK;
}

// rows and lambda values of a call; with counts, the training targets too
static ens_status load_batch(ens_surrogate *S, int n, const double *lambdas, const uint64_t *counts,
                             const ens_hist_spec *h, long long *rows_pad, long long *real, RowSpec *rs)
{
    if (!S || n <= 0 || n > 4096 || !lambdas || !h || h->qr_bins < 1 || h->tail_bins < 1) return ENS_EINVAL;
    rs->nq = h->qr_bins;
    rs->nt = h->tail_bins;
    rs->per_member = h->qr_bins * h->qr_bins + 2 * h->tail_bins;
    *real = (long long)n * rs->per_member;
    *rows_pad = pad128(*real);
    if (!alloc_rows(S, *rs, *rows_pad, 3 * n)) return ENS_ENOMEM;
    if (cudaMemcpyAsync(S->lam, lambdas, sizeof(double) * n, cudaMemcpyHostToDevice, S->s) != cudaSuccess)
        return ENS_ECUDA;
    if (counts) {
        const long long L = counts_len_of(h->qr_bins, h->tail_bins, h->grad_bins);
        if (!alloc_train(S, *rows_pad) || !S->counts.need(sizeof(uint64_t) * n * L)) return ENS_ENOMEM;
        if (cudaMemcpyAsync(S->counts.p, counts, sizeof(uint64_t) * n * L, cudaMemcpyHostToDevice, S->s) != cudaSuccess)
            return ENS_ECUDA;
        k_targets<<<dim3(target_parts(rs->nq, rs->nt), n), 256, 0, S->s>>>(S->counts.as<unsigned long long>(), L, rs->nq, rs->nt, S->target.as<float>());
        feature_table(S, *rs, n);
    }
    return ENS_OK;
}

static ens_status check_err(ens_surrogate *S)
{
    int e = 0;
    if (cudaMemcpyAsync(&e, S->err, sizeof(int), cudaMemcpyDeviceToHost, S->s) != cudaSuccess ||
        cudaStreamSynchronize(S->s) != cudaSuccess)
        return ENS_ECUDA;
    return e ? ENS_ETIMEOUT : ENS_OK;
}

ens_status ens_surrogate_loss_grad(ens_surrogate *S, int n, const double *lambdas, const uint64_t *counts,
                                   const ens_hist_spec *h, double *loss, float *grad_host)
{
    long long rows, real;
    RowSpec rs;
    if (!counts) return ENS_EINVAL;
    ens_status st = load_batch(S, n, lambdas, counts, h, &rows, &real, &rs);
    if (st != ENS_OK) return st;
    loss_grad_kernels(S, rs, n, rows, real, true);
    if (cudaGetLastError() != cudaSuccess) return ENS_ECUDA;
    std::vector<double> lp(3 * n + 1);   // group losses and the kernels' status
    if (cudaMemcpyAsync(lp.data(), S->loss.p, sizeof(double) * lp.size(), cudaMemcpyDeviceToHost, S->s) != cudaSuccess)
        return ENS_ECUDA;
    if (grad_host &&
        cudaMemcpyAsync(grad_host, S->g, sizeof(float) * S->L.total, cudaMemcpyDeviceToHost, S->s) != cudaSuccess)
        return ENS_ECUDA;
    if (cudaStreamSynchronize(S->s) != cudaSuccess) return ENS_ECUDA;
    if (lp[3 * n] != 0.0) return ENS_ETIMEOUT;
    if (loss) {
        double t = 0.0;
        for (int i = 0; i < 3 * n; ++i) t += lp[i];
        *loss = t;
    }
    return ENS_OK;
}

ens_status ens_surrogate_train(ens_surrogate *S, int n, const double *lambdas, const uint64_t *counts,
                               const ens_hist_spec *h, int steps, double lr, double *final_loss)
{
    long long rows, real;
    RowSpec rs;
    if (!counts || steps < 0 || !(lr > 0.0)) return ENS_EINVAL;
    ens_status st = load_batch(S, n, lambdas, counts, h, &rows, &real, &rs);
    if (st != ENS_OK) return st;
    const long long np = S->L.total;
    for (int it = 0; it < steps; ++it) {
        loss_grad_kernels(S, rs, n, rows, real, it == steps - 1);
        S->steps += 1;
        const float b1 = 0.9f, b2 = 0.999f;
        const float bc1 = 1.f - powf(b1, (float)S->steps), bc2 = 1.f - powf(b2, (float)S->steps);
        // cosine decay over the call's steps, from lr to lr / 20
        const double lr_t = lr * (0.05 + 0.95 * 0.5 * (1.0 + std::cos(3.14159265358979323846 * it / steps)));
        k_adam<<<blocks(np, 256), 256, 0, S->s>>>(S->p, S->g, S->m1, S->m2, np, (float)lr_t, b1, b2, 1e-8f, bc1, bc2);
        pack_params(S);
    }
    if (cudaGetLastError() != cudaSuccess) return ENS_ECUDA;
    st = check_err(S);
    if (st != ENS_OK) return st;
    if (final_loss && steps > 0) {
        std::vector<double> lp(3 * n);
        if (cudaMemcpyAsync(lp.data(), S->loss.p, sizeof(double) * 3 * n, cudaMemcpyDeviceToHost, S->s) != cudaSuccess ||
            cudaStreamSynchronize(S->s) != cudaSuccess)
            return ENS_ECUDA;
        double t = 0.0;
        for (double v : lp) t += v;
        *final_loss = t;
    }
    return ENS_OK;
}

ens_status ens_surrogate_density(ens_surrogate *S, int n, const double *lambdas, const ens_hist_spec *h,
                                 double *probs)
{
    long long rows, real;
    RowSpec rs;
    ens_status st = load_batch(S, n, lambdas, nullptr, h, &rows, &real, &rs);
    if (st != ENS_OK) return st;
    if (!forward_fused(S, rs, real)) return ENS_ECUDA;
    k_softmax_ce<<<3 * n, 256, 0, S->s>>>(S->logit.as<float>(), nullptr, rs.nq, rs.nt, 1.0, S->q.as<float>(), nullptr,
                                         nullptr);
    if (cudaGetLastError() != cudaSuccess) return ENS_ECUDA;
    std::vector<float> q((size_t)real);
    if (cudaMemcpyAsync(q.data(), S->q.p, sizeof(float) * real, cudaMemcpyDeviceToHost, S->s) != cudaSuccess)
        return ENS_ECUDA;
    st = check_err(S);
    if (st != ENS_OK) return st;
    for (long long i = 0; i < real; ++i) probs[i] = q[i];
    return ENS_OK;
}

ens_status ens_surrogate_mixture(ens_surrogate *S, const ens_hist_spec *h, const ens_weight_spec *w, double lam_lo,
                                 double lam_hi, int nquad, ens_mixture_out *out)
{
    if (!S || !h || !w || !out || nquad < 1 || nquad > 4096 || !(lam_hi > lam_lo)) return ENS_EINVAL;
    if (w->kind != ENS_W_GAUSS_PAPER && w->kind != ENS_W_GAUSS) return ENS_EINVAL;
    RowSpec rs{h->qr_bins, h->tail_bins, h->qr_bins * h->qr_bins + 2 * h->tail_bins};
    const long long real = (long long)nquad * rs.per_member, rows = pad128(real);
    if (rs.per_member > (1 << 20)) return ENS_EINVAL;
    if (!alloc_rows(S, rs, rows, 3 * nquad)) return ENS_ENOMEM;
    k_quad_weights<<<1, 512, 0, S->s>>>(lam_lo, lam_hi, nquad, w->kind, w->c, w->Z, w->mu, w->sigma, S->lam, S->wq);
    if (!forward_fused(S, rs, real)) return ENS_ECUDA;
    k_softmax_ce<<<3 * nquad, 256, 0, S->s>>>(S->logit.as<float>(), nullptr, rs.nq, rs.nt, 1.0, S->q.as<float>(),
                                             nullptr, nullptr);
    const double dq = 2.0 * h->q_lim / h->qr_bins, dr = 2.0 * h->r_lim / h->qr_bins;
    const double dt = (h->tail_hi - h->tail_lo) / h->tail_bins;
    k_quad_mix<<<blocks(rs.per_member, 32), 256, 0, S->s>>>(S->q.as<float>(), S->wq, nquad, rs.per_member, rs.nq, dq,
                                                            dr, dt, S->pdf, S->err);
    if (cudaGetLastError() != cudaSuccess) return ENS_ECUDA;
    std::vector<double> pdf(rs.per_member + 1);
    if (cudaMemcpyAsync(pdf.data(), S->pdf, sizeof(double) * pdf.size(), cudaMemcpyDeviceToHost, S->s) != cudaSuccess ||
        cudaStreamSynchronize(S->s) != cudaSuccess)
        return ENS_ECUDA;
    if (pdf[rs.per_member] != 0.0) return ENS_ETIMEOUT;
    const int nq2 = rs.nq * rs.nq;
    if (out->pdf_qr) std::memcpy(out->pdf_qr, pdf.data(), sizeof(double) * nq2);
    if (out->pdf_eps) std::memcpy(out->pdf_eps, pdf.data() + nq2, sizeof(double) * rs.nt);
    if (out->pdf_ens) std::memcpy(out->pdf_ens, pdf.data() + nq2 + rs.nt, sizeof(double) * rs.nt);
    out->covered = 1.0;
    return ENS_OK;
}

// average time of the hidden-layer GEMM (rows x 256 x 256) on the object's
// buffers, CUDA events on its stream (profiling)
ens_status ens_surrogate_time_gemm(ens_surrogate *S, long long rows, int iters, double *ms)
{
    if (!S || rows <= 0 || iters < 1 || !ms) return ENS_EINVAL;
    rows = pad128(rows);
    if (!alloc_layers(S, rows)) return ENS_ENOMEM;
    cudaMemsetAsync(S->H.p, 0, sizeof(__nv_bfloat16) * rows * kHid, S->s);
    cudaMemsetAsync(S->Wb.p, 0, sizeof(__nv_bfloat16) * (kHid * kIn + 2 * kHid * kHid), S->s);
    const __nv_bfloat16 *H = S->H.as<__nv_bfloat16>(), *W = S->Wb.as<__nv_bfloat16>() + kHid * kIn;
    auto launch = [&]() { gemm(H, kHid, W, kHid, S->Z.as<float>(), kHid, (int)rows, kHid, kHid, 1, S->err, S->s); };
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    launch();   // warm-up
    cudaEventRecord(a, S->s);
    for (int i = 0; i < iters; ++i) launch();
    cudaEventRecord(b, S->s);
    float t = 0.f;
    const cudaError_t e = cudaEventSynchronize(b);
    if (e == cudaSuccess) cudaEventElapsedTime(&t, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (e != cudaSuccess) return ENS_ECUDA;
    *ms = t / iters;
    return check_err(S);
}

// logits of the network at n lambda values, by the fused inference kernel
// (fused != 0) or by the layer-by-layer forward pass (tests)
ens_status ens_surrogate_logits(ens_surrogate *S, int n, const double *lambdas, const ens_hist_spec *h, int fused,
                                float *logits)
{
    long long rows, real;
    RowSpec rs;
    if (!logits) return ENS_EINVAL;
    ens_status st = load_batch(S, n, lambdas, nullptr, h, &rows, &real, &rs);
    if (st != ENS_OK) return st;
    if (!fused && !alloc_layers(S, rows)) return ENS_ENOMEM;
    if (fused ? !forward_fused(S, rs, real) : !forward_layers(S, rs, n, rows)) return ENS_ECUDA;
    if (cudaMemcpyAsync(logits, S->logit.p, sizeof(float) * real, cudaMemcpyDeviceToHost, S->s) != cudaSuccess)
        return ENS_ECUDA;
    return check_err(S);
}

// average time of the fused inference kernel over nquad lambda values of a
// histogram layout, CUDA events on the object's stream (profiling)
ens_status ens_surrogate_time_infer(ens_surrogate *S, const ens_hist_spec *h, int nquad, int iters, double *ms)
{
    if (!S || !h || nquad < 1 || nquad > 4096 || iters < 1 || !ms) return ENS_EINVAL;
    RowSpec rs{h->qr_bins, h->tail_bins, h->qr_bins * h->qr_bins + 2 * h->tail_bins};
    const long long real = (long long)nquad * rs.per_member, rows = pad128(real);
    if (!alloc_rows(S, rs, rows, 3 * nquad)) return ENS_ENOMEM;
    k_quad_weights<<<1, 512, 0, S->s>>>(-5.0, 5.0, nquad, 1, 0.0, 0.0, 0.0, 1.0, S->lam, S->wq);
    if (!host_bias(S)) return ENS_ECUDA;
    feature_table(S, rs, nquad);
    auto launch = [&]() { launch_infer(S, rs, real, nullptr); };
    launch();   // warm-up
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    cudaEventRecord(a, S->s);
    for (int i = 0; i < iters; ++i) launch();
    cudaEventRecord(b, S->s);
    float t = 0.f;
    const cudaError_t e = cudaEventSynchronize(b);
    if (e == cudaSuccess) cudaEventElapsedTime(&t, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (e != cudaSuccess || cudaGetLastError() != cudaSuccess) return ENS_ECUDA;
    *ms = t / iters;
    return check_err(S);
}

// tensor-core GEMM check: C = A B^T for host BF16 bit patterns (tests)
ens_status ens_tc_gemm_check(const uint16_t *A, const uint16_t *B, float *C, int M, int N, int K, int ksplit)
{
    if (!A || !B || !C || M <= 0 || N <= 0 || K <= 0 || ksplit < 1 || ksplit > kMaxSplit) return ENS_EINVAL;
    if (M % 128 || K % (64 * ksplit) || N % 64) return ENS_EINVAL;
    if (gemm_prepare() != cudaSuccess) return ENS_ECUDA;
    void *dA = nullptr, *dB = nullptr, *dC = nullptr, *dE = nullptr;
    ens_status st = ENS_OK;
    if (cudaMalloc(&dA, sizeof(uint16_t) * M * K) != cudaSuccess || cudaMalloc(&dB, sizeof(uint16_t) * N * K) != cudaSuccess ||
        cudaMalloc(&dC, sizeof(float) * M * N * ksplit) != cudaSuccess || cudaMalloc(&dE, sizeof(int)) != cudaSuccess)
        st = ENS_ENOMEM;
    if (st == ENS_OK) {
        cudaMemcpy(dA, A, sizeof(uint16_t) * M * K, cudaMemcpyHostToDevice);
        cudaMemcpy(dB, B, sizeof(uint16_t) * N * K, cudaMemcpyHostToDevice);
        cudaMemset(dE, 0, sizeof(int));
        gemm((const __nv_bfloat16 *)dA, K, (const __nv_bfloat16 *)dB, K, (float *)dC, N, M, N, K, ksplit, (int *)dE, 0);
        if (ksplit > 1) {
            k_sum_splits<<<blocks((long long)M * N, 256), 256>>>((const float *)dC, ksplit, (long long)M * N,
                                                                (float *)dC + (long long)M * N * (ksplit - 1));
        }
        int e = 0;
        if (cudaDeviceSynchronize() != cudaSuccess) st = ENS_ECUDA;
        cudaMemcpy(&e, dE, sizeof(int), cudaMemcpyDeviceToHost);
        if (e) st = ENS_ETIMEOUT;
        if (st == ENS_OK)
            cudaMemcpy(C, (float *)dC + (ksplit > 1 ? (long long)M * N * (ksplit - 1) : 0), sizeof(float) * M * N,
                       cudaMemcpyDeviceToHost);
    }
    for (void *p : {dA, dB, dC, dE})
        if (p) cudaFree(p);
    return st;
}

}  // extern "C"
