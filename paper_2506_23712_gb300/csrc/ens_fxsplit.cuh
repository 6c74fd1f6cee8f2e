// The last pass of an RK stage split in two launches (an autotuner variant
// of the fused k_fwd_x MODE 0):
//
//   k_fwd_x_fft : forward transform along x of the three n fields of buffer
//                 A, the kept kx rows written unscaled into the compact
//                 spectral layout [3][kx NK][ky NK][kz NZp] (in buffer A,
//                 from field 3 on, free at this point of the stage)
//   k_update    : per kept mode, 1/N^3, Leray projection, constant-power band
//                 forcing, integrating-factor RK stage and the FP64 partial
//                 sums of E, dissipation and band energy (Sec. IV)
//
// The split moves 2 x 3 compact fields more through HBM than the fused pass,
// but each launch is light (no staged tile, more resident warps); the
// arithmetic per mode is the fused pass's, in the same order.
#pragma once

#include "ens_kernels.cuh"

namespace ens {

template <int N>
__device__ __forceinline__ float2 *nhat_of(const Geo &g, int m)
{
    return g.A + ((long long)m * kFields + 3) * Dims<N>::SA;
}

// grid (NK*NZp/T, 3, members), block T*P
template <int N, int T>
__global__ void __launch_bounds__(ColCfg<N, T>::threads)
k_fwd_x_fft(Geo g)
{
    constexpr int V = PlanInfo<N>::V;
    extern __shared__ __align__(16) float2 sm[];
    using CS = ColSlots<N, 0>;
    float2 *tw = sm, *buf = sm + N;
    load_col_twiddles<N, 0>(tw, g.tw);
    const int c = threadIdx.x % T, p = threadIdx.x / T;
    const int q = blockIdx.y, m = blockIdx.z;
    const int col = blockIdx.x * T + c;                  // (ky, kz) flat
    const int iy = col / Dims<N>::NZP, kz = col % Dims<N>::NZP;
    const bool valid = kz < Dims<N>::NZ;
    const float2 *src = g.A + ((long long)m * kFields + q) * Dims<N>::SA + ((long long)iy * N + p) * Dims<N>::NZP + kz;
    constexpr unsigned rowU = Dims<N>::NK * Dims<N>::NZP;
    float2 *dst = nhat_of<N>(g, m) + q * Dims<N>::SU;
    const unsigned off = p * rowU + col;
    float2 v[V];
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = valid ? src[CS::in(i) * Dims<N>::NZP] : make_float2(0.f, 0.f);
    fft_line<N, true, 0, false, true>(v, p, tw, [&](int pos) { return &buf[pos * T + c]; });
    store_kept<N, 0>(v, p, kz < Dims<N>::NZS,
                     [&](auto s, float2 w) { at32(dst, off + (unsigned)CS::row(s.value) * rowU) = w; });
}

constexpr int kUpdThreads = 256;
constexpr int kUpdPairs = kUpdChunk / (2 * kUpdThreads);   // mode pairs per thread

template <int N>
constexpr int update_blocks()
{
    return (int)((Dims<N>::SU + kUpdChunk - 1) / kUpdChunk);
}

// grid (update_blocks<N>(), members), block kUpdThreads.  Thread t takes
// the mode pairs (2j, 2j + 1), j = first + t + u * kUpdThreads: 16-byte
// loads and stores, and every load of a pair issued before its arithmetic.
// A pair never straddles a kz row (NZp is even); modes past the kept kz are
// written as zero up to the end of their 64 bytes.
template <int N>
__global__ void __launch_bounds__(kUpdThreads, 4)
k_update(Geo g, MemberDev *md, int stage, int last_stage)
{
    using D = Dims<N>;
    static_assert(D::NZP % 2 == 0 && D::SU % 2 == 0, "mode pairs must not straddle a row");
    __shared__ double scratch[(kUpdThreads / 32) * 3];
    const int m = blockIdx.y;
    const UpdCoef c = upd_coef<N>(md[g.first + m], stage);
    const float4 *nh = reinterpret_cast<const float4 *>(nhat_of<N>(g, m));
    const float4 *U = reinterpret_cast<const float4 *>(g.U + (long long)m * 3 * D::SU);
    const float4 *S = reinterpret_cast<const float4 *>(g.S + (long long)m * 3 * D::SU);
    float4 *dst = reinterpret_cast<float4 *>((last_stage ? g.U : g.S) + (long long)m * 3 * D::SU);
    constexpr long long rowU = (long long)D::NK * D::NZP;
    constexpr long long SU2 = D::SU / 2;   // pairs per component
    float se = 0.f, sd = 0.f, sb = 0.f;
    const long long first = (long long)blockIdx.x * (kUpdChunk / 2) + threadIdx.x;
#pragma unroll
    for (int u = 0; u < kUpdPairs; ++u) {
        const long long j = first + (long long)u * kUpdThreads;
        const long long mi = 2 * j;
        const int ix = (int)(mi / rowU);
        const int rem = (int)(mi % rowU);
        const int iy = rem / D::NZP, kz = rem % D::NZP;
        const bool any = j < SU2 && kz < D::NZS;
        float4 n4[3], u4[3], s4[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
            const bool ld = any && kz < D::NZ;
            n4[q] = ld ? nh[q * SU2 + j] : z4;
            u4[q] = ld ? U[q * SU2 + j] : z4;
            s4[q] = (ld && stage != 0) ? S[q * SU2 + j] : u4[q];
        }
        if (!any) continue;
        const int kx = ix <= D::KC ? ix : ix - D::NK;
        const int ky = iy <= D::KC ? iy : iy - D::NK;
        float4 o4[3];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float2 n[3], un[3], us[3], o[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                n[q] = h ? make_float2(n4[q].z, n4[q].w) : make_float2(n4[q].x, n4[q].y);
                un[q] = h ? make_float2(u4[q].z, u4[q].w) : make_float2(u4[q].x, u4[q].y);
                us[q] = h ? make_float2(s4[q].z, s4[q].w) : make_float2(s4[q].x, s4[q].y);
            }
            bool band;
            float k2;
            const float a2 = update_mode(c, kx, ky, kz + h, n, un, us, o, band, k2);
            const bool keep = kz + h < D::NZ;
            const float wgt = (kz + h) == 0 ? 1.f : 2.f;   // Hermitian multiplicity in the full spectrum
            if (keep) {
                se += 0.5f * wgt * a2;
                sd += c.nu * k2 * wgt * a2;
                if (band) sb += 0.5f * wgt * a2;
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float2 v = keep ? o[q] : make_float2(0.f, 0.f);
                if (h == 0) { o4[q].x = v.x; o4[q].y = v.y; } else { o4[q].z = v.x; o4[q].w = v.y; }
            }
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) dst[q * SU2 + j] = o4[q];
    }
    double vals[3] = {(double)se, (double)sd, (double)sb};
    double *out = g.partial + ((long long)(g.first + m) * g.partial_blocks + blockIdx.x) * 4;
    block_sum_to<3>(out, vals, scratch);
}

}  // namespace ens
