// Training step of the learned lambda interpolant on the tensor cores.
//
//   forward   k_mlp_infer_pair<true> (the fused inference kernel): logits, and
//             the BF16 activations H1, H2 as tile images
//   softmax   k_softmax_ce: cross-entropy and dlogit per (lambda, kind) group
//   backward  k_mlp_back: per 128-row tile the pre-activations again from the
//             images, then the chain dZ3 -> dZ2 -> dZ1 back through the layers;
//             dZ3, dZ2, dZ1 and the features become tile images too
//   gradients k_mlp_wgrad: dW_l = dZ_l^T H_{l-1} from the images, split over
//             the rows, and the bias gradients (column sums of dZ_l)
//   sums      k_grad_sum: the splits' partials added in a fixed order
//
// Why the pre-activations are formed twice: one layer's FP32 Z of 295 k rows is
// 302 MB, and the backward pass needs three of them.  Writing and reading them
// costs 1.8 GB of HBM traffic (0.27 ms at 6.8 TB/s); forming them again from the
// BF16 activations costs 87 GFLOP of products that run behind the epilogues,
// and no pre-activation ever leaves the tensor memory.
//
// One operand layout serves every product.  A tile of 128 rows x 64 columns
// of BF16 in the 128-byte swizzle is, read one way, the K-major A operand of a
// layer (M = rows, K = columns) and, read the other way, an MN-major operand
// of a weight gradient (K = rows, M or N = columns): the descriptors differ,
// the bytes do not, so nothing is transposed in memory.  The same holds for
// the weights: the K-major image W_l [out][in] of the forward product, taken
// by 64 rows of `out`, is the MN-major B operand of dH_{l-1} = dZ_l W_l.
//
// Measured (GB300, 64 members x 4608 bins, one loss and gradient through the
// library call): 8.69 ms with one GEMM launch per product, separate bias,
// SiLU, transpose and column-sum kernels and FP32 pre-activations in memory;
// 0.68 ms in this form (forward 0.136, backward 0.256, weight gradients 0.123,
// targets, softmax and sums 0.05 ms, the rest copies and launches).
#pragma once

namespace ens {

// shared-memory descriptor of an MN-major operand in the 128-byte swizzle:
// 64 columns (128 bytes) per row, 8-row groups of K 1024 bytes apart, the next
// 64 columns `lbo` bytes further
__device__ __forceinline__ uint64_t desc_mn128(const void *tile, uint32_t lbo)
{
    const uint64_t addr = smem_u32(tile);
    uint64_t d = (addr >> 4) & 0x3FFFull;
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;   // leading byte offset: next 64 columns
    d |= (uint64_t)(1024 >> 4) << 32;              // stride byte offset: next 8 rows of K
    d |= 1ull << 46;
    d |= 2ull << 61;
    return d;
}
constexpr uint32_t kMajorA = 1u << 15, kMajorB = 1u << 16;   // instruction descriptor: operand is MN-major

// SiLU'(z) from h = z / 2 and t = tanh(h)
__device__ __forceinline__ float dsilu_ht(float h, float t)
{
    const float s = fmaf(0.5f, t, 0.5f);
    return s * fmaf(2.f * h, 1.f - s, 1.f);
}

// sums over the 32 lanes of each of 16 values: lane l returns the sum of
// value l / 2 (halving butterfly: 16 shuffles instead of 5 per value)
__device__ __forceinline__ float lane_sums16(float (&v)[16], int lane)
{
#pragma unroll
    for (int o = 16; o >= 2; o >>= 1) {
        const bool up = lane & o;
        const int half = o >> 1;   // values kept after this round
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float give = up ? v[i] : v[i + half], keep = up ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

struct TrainImages {
    unsigned char *X, *H1, *H2, *dZ1, *dZ2, *dZ3;
};

// ---------------------------------------------------------------------------
// Backward pass of 128-row tiles, one tile in flight per persistent CTA (18
// warps).  TMEM: two 256-column accumulators A, B.  Shared memory: two
// four-block operand buffers P, Q (64 KB each) and three 32 KB weight slots.
//
//   (copies)  H2 -> P, H1 -> Q          from the forward pass's images
//   M3  H2(P) W3^T      -> A
//   M2  H1(Q) W2^T      -> B            (behind E3)
//   E3  dZ3 = dlogit w4 SiLU'(A)  -> Q  (image dZ3; head gradient sums)
//   M4  dZ3(Q) W3       -> A
//   E4  dZ2 = A SiLU'(B)          -> P  (image dZ2)
//   M5  dZ2(P) W2       -> A            (Z2 in B is used up; features into Q0)
//   M6  X(Q0) W1^T      -> B
//   E5  dZ1 = A SiLU'(B)                (image dZ1; the next tile's copies run)
//
// The FP32 pre-activations are formed again from the BF16 activations (M3,
// M2, M6) and never leave the tensor memory.  An epilogue loads its whole
// accumulator A before its first chunk arrival, so the next product may start
// on chunk 0 while the later chunks are still being formed; B is rewritten
// only after every warp has read it (`feat` arrivals for M6).  The next tile's
// products, M3 included, wait for the `fin` arrivals behind E5; only its copies
// run beside E5.  Weight K-blocks stream through the three slots in
// the order of use, 17 per tile; M4 and M5 take 64 rows of the weight image
// (four 8 KB pieces) as MN-major operands.  Every wait is bounded; a role
// whose wait gives up sets *err and the CTA drains.
//
// Bound by the three epilogues of a tile and the products between them, one
// after another: a tile fills the tensor memory, so no second tile runs
// beside it.  0.256 ms for 295 k rows (2304 tiles, 16 rounds of 152 CTAs; 0.356
// ms with H1, H2 formed again from the features, five epilogues per tile, 0.296
// ms with every bias read from global memory).
// ---------------------------------------------------------------------------
constexpr int kHeadPart = kHid + 4;   // floats of a CTA's head partial: dlogit H3 [256], dlogit [1], padding

__global__ void __launch_bounds__(kPairThreads, 1)
k_mlp_back(RowSpec rs, const uint4 *__restrict__ ftab, const uint32_t *__restrict__ lam5, long long real,
           long long ntiles, const unsigned char *__restrict__ img1, const unsigned char *__restrict__ img2,
           const unsigned char *__restrict__ img3, const MlpBias *__restrict__ bias, const float *__restrict__ dlogit,
           TrainImages im, float *__restrict__ head_part, int *err)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *sm = smem_raw;
    if (smem_u32(sm) & 1023u) {
        if (threadIdx.x == 0) atomicExch(err, 1);
        return;
    }
    unsigned char *const sP = sm, *const sQ = sm + 65536;
    unsigned char *const sW = sm + 2 * 65536;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sW + kPairSlots * 32768);
    uint64_t *full = bars;          // [3] slot holds its block
    uint64_t *empty = bars + 3;     // [3] slot's MMAs done
    uint64_t *accr = bars + 6;      // [2] accumulator A (M3, M4), B (M2; M6 with M5) complete
    uint64_t *chunk = bars + 8;     // [4] operand chunk c written
    uint64_t *opnd = bars + 12;     // [2] H2 in P, H1 in Q
    uint64_t *feat = bars + 14;     // features in Q0, B read
    uint64_t *fin = bars + 15;      // tile's accumulators read by every warp (after E5)
    uint64_t *freed = bars + 16;    // P and Q read by the tile's last products
    uint64_t *drain = bars + 17;
    uint32_t *holder = reinterpret_cast<uint32_t *>(bars + 18);
    float *sB = reinterpret_cast<float *>(bars + 32);   // b1, b2
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) tmem_alloc(holder, 512);
    if (tid == 0) {
        for (int s = 0; s < kPairSlots; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int x = 0; x < 2; ++x) {
            mbar_init(&accr[x], 1);
            mbar_init(&opnd[x], 1);
        }
        for (int c = 0; c < 4; ++c) mbar_init(&chunk[c], kPairWarps);
        mbar_init(feat, kPairWarps);
        mbar_init(fin, kPairWarps);
        mbar_init(freed, 1);
        mbar_init(drain, 1);
        fence_mbar_init();
    }
    for (int i = tid; i < kHid; i += kPairThreads) {
        sB[i] = bias->b1[i];
        sB[kHid + i] = bias->b2[i];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = *holder;
    bool ok = true;
    float hsum[5] = {0.f, 0.f, 0.f, 0.f, 0.f};   // epilogue warps: head gradient sums at the end
    if (warp == kPairWarps + 1) {
        // ---- copy warp ----
        long long q = 0, it = 0;
        long long lastq[kPairSlots] = {-1, -1, -1};
        for (long long t = blockIdx.x; ok && t < ntiles; t += gridDim.x, ++it) {
            for (int j = 0; j < 17; ++j, ++q) {
                if (j == 3) {   // the slots are full: the operands, once the previous tile is through with P and Q
                    if (it > 0) ok = mbar_wait_warp(freed, (uint32_t)((it - 1) & 1));
                    if (!ok) break;
                    if (lane == 0) {
                        for (int x = 0; x < 2; ++x) {   // image order: half tiles, then blocks
                            const unsigned char *src = (x == 0 ? im.H2 : im.H1) + t * 2 * kHalfTile;
                            unsigned char *dst = x == 0 ? sP : sQ;
                            mbar_arrive_expect_tx(&opnd[x], 65536);
                            for (int b = 0; b < 8; ++b)
                                bulk_g2s(dst + (b & 3) * 16384 + (b >> 2) * 8192, src + b * 8192, 8192, &opnd[x]);
                        }
                    }
                    __syncwarp();
                }
                const int s = (int)(q % kPairSlots);
                if (q >= kPairSlots) ok = mbar_wait_warp(&empty[s], (uint32_t)(((q / kPairSlots) & 1) ^ 1));
                if (!ok) break;
                if (lane == 0) {
                    unsigned char *dst = sW + s * 32768;
                    mbar_arrive_expect_tx(&full[s], 32768);
                    if (j < 8 || j == 16) {
                        const unsigned char *src = j == 16 ? img1 : (j < 4 ? img3 + j * 32768 : img2 + (j - 4) * 32768);
                        bulk_g2s(dst, src, 32768, &full[s]);
                    } else {
                        const unsigned char *src = j < 12 ? img3 + (j - 8) * 8192 : img2 + (j - 12) * 8192;
                        for (int b = 0; b < 4; ++b) bulk_g2s(dst + b * 8192, src + b * 32768, 8192, &full[s]);
                    }
                }
                lastq[s] = q;
            }
        }
        if (!ok) {   // copies in flight complete before the CTA ends (bounded)
            for (int s = 0; s < kPairSlots; ++s)
                if (lastq[s] >= 0) mbar_wait_warp(&full[s], (uint32_t)((lastq[s] / kPairSlots) & 1));
            for (int x = 0; x < 2; ++x) mbar_wait_warp(&opnd[x], (uint32_t)(it & 1));
        }
    } else if (warp == kPairWarps) {
        // ---- MMA warp ----
        constexpr uint32_t idesc = idesc_bf16(128, kHid), idesc_t = idesc | kMajorB;
        uint32_t tile = 0, nchunk = 0;
        long long q = 0;
        // one K-block (64): A operand block a, weight slot of block q
        auto mma_kb = [&](uint32_t acc, const unsigned char *a, bool transposed, bool first) {
            const unsigned char *b = sW + (int)(q % kPairSlots) * 32768;
            if (lane == 0) {
                tc_fence_after();
                const uint64_t da = desc_sw128(a), db = transposed ? desc_mn128(b, 8192) : desc_sw128(b);
                const uint32_t step = transposed ? 128 : 2;   // 16 rows of K, or 32 bytes
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    tc_mma_bf16(taddr + acc, da + 2 * k, db + step * k, transposed ? idesc_t : idesc,
                                (!first || k > 0) ? 1u : 0u);
                tc_commit(&empty[q % kPairSlots]);
            }
            __syncwarp();
            ++q;
        };
        auto wfull = [&]() { return mbar_wait_warp(&full[q % kPairSlots], (uint32_t)((q / kPairSlots) & 1)); };
        // the product over a whole operand buffer; chunks: as they are written
        auto layer = [&](uint32_t acc, const unsigned char *a, bool transposed, bool chunks) {
            for (int c = 0; c < 4; ++c) {
                if (!wfull() || (chunks && !mbar_wait_warp(&chunk[c], nchunk & 1))) return false;
                mma_kb(acc, a + c * 16384, transposed, c == 0);
            }
            if (chunks) ++nchunk;
            return true;
        };
        for (long long t = blockIdx.x; ok && t < ntiles; t += gridDim.x, ++tile) {
            if (tile > 0) ok = mbar_wait_warp(fin, (tile - 1) & 1);
            ok = ok && mbar_wait_warp(&opnd[0], tile & 1) && layer(0, sP, false, false);     // M3
            if (!ok) break;
            if (lane == 0) tc_commit(&accr[0]);
            ok = mbar_wait_warp(&opnd[1], tile & 1) && layer(256, sQ, false, false);         // M2
            if (!ok) break;
            if (lane == 0) tc_commit(&accr[1]);
            ok = layer(0, sQ, true, true);                                                   // M4
            if (!ok) break;
            if (lane == 0) tc_commit(&accr[0]);
            ok = layer(0, sP, true, true);                                                   // M5
            if (!ok) break;
            ok = wfull() && mbar_wait_warp(feat, tile & 1);
            if (!ok) break;
            mma_kb(256, sQ, false, true);                                                    // M6
            if (lane == 0) {
                tc_commit(&accr[1]);
                tc_commit(freed);
            }
        }
        if (lane == 0) tc_commit(drain);
        __syncwarp();
        mbar_wait_warp(drain, 0);
    } else {
        // ---- epilogue warps: TMEM lanes 32 (warp mod 4) .. +31, in chunk c
        // columns 64 c + 16 (warp / 4) .. +15 ----
        const int quarter = warp & 3, cpart = warp >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
        const uint32_t accA = taddr + lanes + (uint32_t)(16 * cpart), accB = accA + 256;
        uint32_t nacc[2] = {0, 0};
        float gw[4] = {0.f, 0.f, 0.f, 0.f}, gb = 0.f;   // head gradient: column 64 c + 16 cpart + lane / 2, and sum of dlogit
        auto features = [&](long long t, unsigned char *H, unsigned char *img) {
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
            if (img) {
                const uint32_t w[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
                store_row32(image_row(img, t, r, 0, 1), r, tid & 3, w);
            }
        };
        auto arrive = [&](uint64_t *bar) {
            fence_proxy_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar);
        };
        auto wait_acc = [&](int x) {
            const bool r = mbar_wait_warp(&accr[x], nacc[x] & 1);
            if (r) {
                ++nacc[x];
                tc_fence_after();
            }
            return r;
        };
        // chunk c of an operand into shared memory, for the next product
        auto put = [&](unsigned char *buf, int c, const uint32_t (&w)[8]) {
            unsigned char *blk = buf + c * 16384;
            *reinterpret_cast<uint4 *>(blk + sw128_offset(row, 16 * cpart)) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4 *>(blk + sw128_offset(row, 16 * cpart + 8)) = make_uint4(w[4], w[5], w[6], w[7]);
            arrive(&chunk[c]);
        };
        // dZ = dH(acc A) SiLU'(Z (acc B) + b) into the image and, unless null,
        // the operand buffer
        auto back = [&](int x, const float *bv, unsigned char *buf, unsigned char *img, long long t) {
            if (!wait_acc(x)) return false;
            uint32_t r[4][16], z[16];
#pragma unroll
            for (int c = 0; c < 4; ++c) tc_ld_16cols_issue(accA + 64u * c, r[c]);
            tc_ld_16cols_issue(accB, z);
#pragma unroll
            for (int c = 0; c < 4; ++c) tc_ld_wait16(r[c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const Cols16Ref b(bv + 64 * c + 16 * cpart);
                tc_ld_wait16(z);
                uint32_t w[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float2 h = fma2(make_float2(0.5f, 0.5f),
                                          make_float2(__uint_as_float(z[2 * k]), __uint_as_float(z[2 * k + 1])), b[k]);
                    w[k] = cvt_bf16x2(__uint_as_float(r[c][2 * k]) * dsilu_ht(h.x, tanh_approx(h.x)),
                                      __uint_as_float(r[c][2 * k + 1]) * dsilu_ht(h.y, tanh_approx(h.y)));
                }
                if (c < 3) tc_ld_16cols_issue(accB + 64u * (c + 1), z);
                if (buf) put(buf, c, w);
                store_row32(image_row(img, t, row, c, 4), row, cpart, w);
            }
            return true;
        };
        for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
            // E3: dZ3 = dlogit w4 SiLU'(Z3), head gradient sums dlogit H3
            const long long rr = t * 128 + row;
            const float dl = rr < real ? dlogit[rr] : 0.f;
            ok = wait_acc(0);
            if (!ok) break;
            {
                uint32_t r[4][16];
#pragma unroll
                for (int c = 0; c < 4; ++c) tc_ld_16cols_issue(accA + 64u * c, r[c]);
#pragma unroll
                for (int c = 0; c < 4; ++c) tc_ld_wait16(r[c]);
                gb += dl;
                // dZ3 replaces H1 in Q: M2 has read it
                ok = wait_acc(1);
                if (!ok) break;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const Cols16 b(bias->b3 + 64 * c + 16 * cpart), wh(bias->w4 + 64 * c + 16 * cpart);
                    uint32_t w[8];
                    float hg[16];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float2 h = fma2(make_float2(0.5f, 0.5f),
                                              make_float2(__uint_as_float(r[c][2 * k]), __uint_as_float(r[c][2 * k + 1])),
                                              b[k]);
                        const float2 w4 = wh[k];
                        const float tx = tanh_approx(h.x), ty = tanh_approx(h.y);
                        const uint32_t hb = cvt_bf16x2(fmaf(h.x, tx, h.x), fmaf(h.y, ty, h.y));   // H3
                        hg[2 * k] = dl * __uint_as_float(hb << 16);
                        hg[2 * k + 1] = dl * __uint_as_float(hb & 0xFFFF0000u);
                        w[k] = cvt_bf16x2(dl * w4.x * dsilu_ht(h.x, tx), dl * w4.y * dsilu_ht(h.y, ty));
                    }
                    put(sQ, c, w);
                    store_row32(image_row(im.dZ3, t, row, c, 4), row, cpart, w);
                    gw[c] += lane_sums16(hg, lane);
                }
            }
            ok = back(0, sB + kHid, sP, im.dZ2, t);        // E4 (M3 has read P: E3 waited for it)
            if (!ok) break;
            features(t, sQ, im.X);                        // M4 has read Q: E4 waited for it
            arrive(feat);
            ok = back(1, sB, nullptr, im.dZ1, t);   // E5
            if (!ok) break;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(fin);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) hsum[c] = gw[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) gb += __shfl_xor_sync(0xffffffffu, gb, o);
        hsum[4] = gb;
    }
    if (!ok && lane == 0) atomicExch(err, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(taddr, 512);
    // head partials of the CTA: [4 quarters][256 columns], then the sums of dlogit [4]
    float *red = reinterpret_cast<float *>(sW);
    if (warp < kPairWarps) {
        const int quarter = warp & 3, cpart = warp >> 2;
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (!(lane & 1)) red[quarter * kHid + 64 * c + 16 * cpart + (lane >> 1)] = hsum[c];
        if (cpart == 0 && lane == 0) red[4 * kHid + quarter] = hsum[4];
    }
    __syncthreads();
    float *hp = head_part + (long long)blockIdx.x * kHeadPart;
    if (tid < kHid) hp[tid] = (red[tid] + red[kHid + tid]) + (red[2 * kHid + tid] + red[3 * kHid + tid]);
    if (tid == kHid) hp[kHid] = (red[4 * kHid] + red[4 * kHid + 1]) + (red[4 * kHid + 2] + red[4 * kHid + 3]);
}

// ---------------------------------------------------------------------------
// Weight and bias gradients: dW_l [256 out][in] = sum over rows of dZ_l^T
// H_{l-1}, rows split over the CTAs of a layer (split s takes the half tiles
// s, s + splits, ...).  Both operands are MN-major images; the accumulator is
// the layer's whole gradient (M = 2 x 128 rows of `out`, N = in: all 512 TMEM
// columns at in = 256).  Half tiles (64 rows, 2 x 32 KB) stream through three
// stages by bulk copies; 8 worker warps add the columns of dZ for the bias
// gradient from the same stage.  Bound by HBM: every image is read once (793
// MB at 295 k rows in 0.123 ms, 6.4 TB/s, 95% of the copy rate; the split-K GEMM
// launches and column sums before took 2.8 ms).
// ---------------------------------------------------------------------------
constexpr int kWgStages = 3;
constexpr int kWgWorkers = 8;
constexpr int kWgThreads = 32 * (kWgWorkers + 2);
constexpr size_t kWgSmem = 1024 + (size_t)kWgStages * 2 * kHalfTile + 128 + 2 * 128 * sizeof(float2);
constexpr long long kPartW = (long long)kHid * kHid;             // floats of a layer's partial gradient
constexpr long long kPartStride = kPartW + kHid;                 // with its bias partial

struct WgradSplits {
    int n[3];   // CTAs of layer 1, 2, 3
};

__global__ void __launch_bounds__(kWgThreads, 1)
k_mlp_wgrad(TrainImages im, long long halves, WgradSplits sp, float *__restrict__ part, int *err)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *full = reinterpret_cast<uint64_t *>(sm + kWgStages * 2 * kHalfTile);
    uint64_t *empty = full + kWgStages, *done = empty + kWgStages;
    uint32_t *holder = reinterpret_cast<uint32_t *>(done + 1);
    float2 *csum = reinterpret_cast<float2 *>(sm + kWgStages * 2 * kHalfTile + 128);   // [2][128] column pairs
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int split = blockIdx.x, layer = 2;   // layer 3 first (index 2), then 2, then 1
    while (layer > 0 && split >= sp.n[layer]) split -= sp.n[layer--];
    const int nsplit = sp.n[layer];
    const unsigned char *gA = layer == 2 ? im.dZ3 : layer == 1 ? im.dZ2 : im.dZ1;
    const unsigned char *gB = layer == 2 ? im.H2 : layer == 1 ? im.H1 : im.X;
    const uint32_t bytesB = layer == 0 ? 8192u : (uint32_t)kHalfTile;
    if (warp == 0) tmem_alloc(holder, 512);
    if (tid == 0) {
        for (int s = 0; s < kWgStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1 + kWgWorkers);
        }
        mbar_init(done, 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = *holder;
    bool ok = true;
    if (warp == kWgWorkers + 1) {
        long long it = 0;
        for (long long h = split; h < halves; h += nsplit, ++it) {
            const int s = (int)(it % kWgStages);
            if (it >= kWgStages) ok = mbar_wait_warp(&empty[s], (uint32_t)(((it / kWgStages) & 1) ^ 1));
            if (!ok) break;
            if (lane == 0) {
                unsigned char *st = sm + s * 2 * kHalfTile;
                mbar_arrive_expect_tx(&full[s], (uint32_t)kHalfTile + bytesB);
                bulk_g2s(st, gA + h * kHalfTile, (uint32_t)kHalfTile, &full[s]);
                bulk_g2s(st + kHalfTile, gB + h * bytesB, bytesB, &full[s]);
            }
        }
        if (!ok) {   // copies of the stages still in flight (bounded)
            for (long long j = it > kWgStages ? it - kWgStages : 0; j < it; ++j)
                mbar_wait_warp(&full[j % kWgStages], (uint32_t)((j / kWgStages) & 1));
        }
    } else if (warp == kWgWorkers) {
        const uint32_t idesc = idesc_bf16(128, layer == 0 ? kIn : kHid) | kMajorA | kMajorB;
        long long it = 0;
        for (long long h = split; h < halves; h += nsplit, ++it) {
            const int s = (int)(it % kWgStages);
            ok = mbar_wait_warp(&full[s], (uint32_t)((it / kWgStages) & 1));
            if (!ok) break;
            if (lane == 0) {
                tc_fence_after();
                const unsigned char *st = sm + s * 2 * kHalfTile;
                const uint64_t db = desc_mn128(st + kHalfTile, 8192);
#pragma unroll
                for (int mh = 0; mh < 2; ++mh) {
                    const uint64_t da = desc_mn128(st + mh * 16384, 8192);
#pragma unroll
                    for (int k = 0; k < 4; ++k)   // 16 rows = 2048 bytes per step
                        tc_mma_bf16(taddr + 256u * mh, da + 128 * k, db + 128 * k, idesc, (it > 0 || k > 0) ? 1u : 0u);
                }
                tc_commit(&empty[s]);
            }
            __syncwarp();
        }
        if (lane == 0) tc_commit(done);
        __syncwarp();
        mbar_wait_warp(done, 0);   // every MMA completes before the TMEM is read or freed (bounded)
    } else {
        // bias gradient: thread <-> column pair tid mod 128, rows 32 (tid / 128) .. +31
        const int pair = tid & 127, blk = pair >> 5, pp = pair & 31, r0 = (tid >> 7) * 32;
        float2 acc = make_float2(0.f, 0.f);
        long long it = 0;
        for (long long h = split; h < halves; h += nsplit, ++it) {
            const int s = (int)(it % kWgStages);
            ok = mbar_wait_warp(&full[s], (uint32_t)((it / kWgStages) & 1));
            if (!ok) break;
            const unsigned char *b = sm + s * 2 * kHalfTile + blk * 8192;
            float2 sum = make_float2(0.f, 0.f);
#pragma unroll
            for (int r = 0; r < 32; ++r) {
                const uint32_t v = *reinterpret_cast<const uint32_t *>(
                    b + (r0 + r) * 128 + (((pp >> 2) ^ (r & 7)) << 4) + (pp & 3) * 4);
                sum.x += __uint_as_float(v << 16);
                sum.y += __uint_as_float(v & 0xFFFF0000u);
            }
            acc.x += sum.x;
            acc.y += sum.y;
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s]);
        }
        csum[(tid >> 7) * 128 + pair] = acc;
        ok = ok && mbar_wait_warp(done, 0);
    }
    if (!ok && lane == 0) atomicExch(err, 1);
    const bool all = __syncthreads_and(ok);
    tc_fence_after();
    if (all && warp < kWgWorkers) {
        float *out = part + (long long)blockIdx.x * kPartStride;
        const int mh = warp >> 2, quarter = warp & 3;
        const int in = layer == 0 ? kIn : kHid;
        float *row = out + (long long)(mh * 128 + quarter * 32 + lane) * in;
#pragma unroll 1
        for (int c = 0; c < in; c += 32) {
            float v[32];
            tc_ld_32cols(taddr + 256u * mh + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c, v);
#pragma unroll
            for (int i = 0; i < 32; i += 4)
                *reinterpret_cast<float4 *>(row + c + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        }
        if (tid < 128) {
            const float2 a = csum[tid], b = csum[128 + tid];
            *reinterpret_cast<float2 *>(out + kPartW + 2 * tid) = make_float2(a.x + b.x, a.y + b.y);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(taddr, 512);
}

// Gradient vector from the partials: weights and biases over the layer's
// splits, head over the backward CTAs (fixed order, eight running sums; 19 us,
// 47 with sixteen).  *status = *err, beside the group losses,
// so that one copy brings both to the host.
__global__ void k_grad_sum(const float *__restrict__ part, WgradSplits sp, const float *__restrict__ head_part,
                           int back_ctas, float *__restrict__ g, const int *err, double *status)
{
    const ParamLayout L = param_layout();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *status = (double)*err;
    if (i >= L.total) return;
    const float *src;
    long long stride;
    int n;
    if (i < L.w4) {
        const int layer = i < L.W2 ? 0 : i < L.W3 ? 1 : 2;
        const long long W = layer == 0 ? L.W1 : layer == 1 ? L.W2 : L.W3;
        const long long b = layer == 0 ? L.b1 : layer == 1 ? L.b2 : L.b3;
        const int first = layer == 2 ? 0 : layer == 1 ? sp.n[2] : sp.n[2] + sp.n[1];
        src = part + (long long)first * kPartStride + (i < b ? i - W : kPartW + (i - b));
        stride = kPartStride;
        n = sp.n[layer];
    } else {
        src = head_part + (i - L.w4);
        stride = kHeadPart;
        n = back_ctas;
    }
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int k = 0; k < n; k += 8) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (k + j < n) s[j] += src[(long long)(k + j) * stride];
    }
    g[i] = ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
}

// Targets of the cross-entropy: each (member, kind) histogram normalised to
// unit sum, (float)((double)c / s).  Grid (parts of kTargetPart bins, members):
// every block adds up its whole histogram (whole numbers, exact) and divides
// its own part.  FP64 division runs on two lanes per SM and clock here, so it
// is taken only where a count or sum is not an FP32 number: up to 2^24 the
// FP32 quotient of the exact operands is the same value (a quotient rounded
// to 53 bits and then to 24 equals the one rounded once, 53 >= 2 x 24 + 2).
// 64 members x 4608 bins: 49 us with FP64 division, one block per histogram.
constexpr int kTargetPart = 512;

__host__ __device__ inline int target_parts(int nq, int nt)
{
    return (nq * nq + kTargetPart - 1) / kTargetPart + 2 * ((nt + kTargetPart - 1) / kTargetPart);
}

__global__ void k_targets(const unsigned long long *__restrict__ counts, long long counts_len, int nq, int nt,
                          float *__restrict__ target)
{
    const int pq = (nq * nq + kTargetPart - 1) / kTargetPart, pt = (nt + kTargetPart - 1) / kTargetPart;
    int part = blockIdx.x, kind = 0;
    if (part >= pq) {
        kind = 1 + (part - pq) / pt;
        part = (part - pq) % pt;
    }
    const int member = blockIdx.y;
    const int off = kind == 0 ? 0 : nq * nq + (kind - 1) * nt;
    const int len = kind == 0 ? nq * nq : nt;
    const unsigned long long *c = counts + member * counts_len + off;
    float *t = target + (long long)member * (nq * nq + 2 * nt) + off;
    __shared__ unsigned long long red[32];
    unsigned long long s = 0;
    for (int i = threadIdx.x; i < len; i += blockDim.x) s += c[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    s = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    const int end = min(len, (part + 1) * kTargetPart);
    for (int i = part * kTargetPart + threadIdx.x; i < end; i += blockDim.x) {
        const unsigned long long v = c[i];
        float q = 0.f;
        if (v && s <= (1ull << 24)) q = __fdiv_rn((float)v, (float)s);
        else if (v) q = (float)((double)v / (double)s);
        t[i] = q;
    }
}

}  // namespace ens
