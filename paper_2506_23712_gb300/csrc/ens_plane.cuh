// The middle of an RK stage in one kernel for small grids (N <= 64): inverse y,
// z pass and forward y of one x plane of one member.
//
// After the x transform the planes of constant x are independent until the
// forward x transform.  A plane's six half spectra fit one SM's shared memory
// up to 64^3 (6 x 64 x 26 complex, 80 KB), so buffer B is never written: the
// plane is read from buffer A, transformed along y into shared memory, taken
// through the z pass row by row in place (inverse z, n = u x omega, max|u|,
// forward z), and transformed back along y into buffer A.
//
// What bounds these sizes is not bandwidth (16 x 64^3 fits the L2 but for buffer
// B) but launches, tails and the latency of each pass's first loads; two of
// every five launches of a stage go, and the traffic of buffer B with them
// (27 of 57 MB per stage and 16 members).  The transforms are those of the
// separate passes, value for value; only the n_z rows that share a complex
// line are paired differently.
//
// Warp-local lines throughout: in the y passes a warp takes CW neighbouring kz
// columns (32 bytes or more per row of A: whole sectors), P threads per
// column, so the three phases need two block barriers between them and none
// inside.  8 warps, two CTAs per SM.
//
// Measured (step, RK3 but for 32^3 x 1 with RK2): 16 x 64^3 346 -> 290 us (269 with
// the split last pass), 4 x 64^3 125 -> 103, 64 x 64^3 1270 -> 1030, 1 x 32^3 64 -> 54,
// 16 x 32^3 97 -> 80, 64 x 16^3 82 -> 66.
#pragma once

#include "ens_znl.cuh"

namespace ens {

__host__ __device__ constexpr bool has_plane(int N) { return N <= 64; }

struct WarpSync {
    __device__ __forceinline__ void operator()() const { __syncwarp(); }
};

template <int N>
struct PlaneCfg {
    using D = Dims<N>;
    using CP = PlanInfo<N, 0>;                               // column plan
    using ZP = WPlanInfo<N, 0>;                              // row plan
    static constexpr int WPB = 8;                            // warps per CTA
    static constexpr int CW = 32 / CP::P;                    // columns per warp
    static constexpr int KG = (D::NZ + CW - 1) / CW;         // column groups
    static constexpr int LPW = 32 / ZP::P;                   // rows per warp
    static constexpr int GR = N / LPW;                       // row groups
    static constexpr int max2(int a, int b) { return a > b ? a : b; }
    // row pitch: the columns the y pass writes, the z pass's zero tail, the columns it writes
    static constexpr int PITCH = (max2(max2(stage_pitch<N, 0>(), KG * CW), D::NZS) + 1) / 2 * 2;
    static constexpr int FS = N * PITCH;                     // field stride
    // exchange slot of a column line: CW columns side by side, one pad per R0
    // positions (the threads of a line store R0 positions apart)
    static __device__ __forceinline__ int slot(int pos) { return (pos + pos / CP::R0) * CW; }
    static constexpr int COLBUF = (N + N / CP::R0) * CW;
    static constexpr int BUF = max2(COLBUF, LPW * WPadV<N, 0>::SROW);   // per warp
    static constexpr size_t smem() { return sizeof(float2) * (size_t)(N + 6 * FS + WPB * BUF); }
    static_assert(CP::NP == 2 && WPadV<N, 0>::on && GR >= 1, "plans of the small sizes");
};

// grid (N, members), block 32 * WPB
template <int N>
__global__ void __launch_bounds__(32 * PlaneCfg<N>::WPB, 2)
k_plane(Geo g, MemberDev *md, int stage_idx)
{
    using C = PlaneCfg<N>;
    using D = Dims<N>;
    using CS = ColSlots<N, 0>;
    using ZP = typename C::ZP;
    constexpr int V = CS::V, ZV = ZP::V, P = ZP::P, LPW = C::LPW, WPB = C::WPB, PITCH = C::PITCH, FS = C::FS;
    extern __shared__ __align__(16) float2 sm[];
    float2 *tw = sm, *plane = sm + N, *bufs = plane + 6 * FS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int x = blockIdx.x, m = blockIdx.y;
    float2 *buf = bufs + warp * C::BUF;
    ColTw<N, 0>::load(tw, g.tw, threadIdx.x, blockDim.x);
    constexpr int TAIL = PITCH - C::KG * C::CW;   // columns the y pass does not write
    if constexpr (TAIL > 0) {
        for (int e = threadIdx.x; e < 6 * N * TAIL; e += blockDim.x)
            plane[(e / TAIL) * PITCH + C::KG * C::CW + e % TAIL] = make_float2(0.f, 0.f);
    }

    // ---- inverse y: columns of buffer A into the plane ----
    constexpr unsigned row = N * D::NZP;
    float2 *A = g.A + (long long)m * kFields * D::SA + (long long)x * D::NZP;
    const int c = lane % C::CW, p = lane / C::CW;
    auto at = [&](int pos) { return &buf[C::slot(pos) + c]; };
    auto load = [&](float2 *v, int item) {
        const int kz = item % C::KG * C::CW + c;
        const float2 *src = A + (long long)(item / C::KG) * D::SA;
        const unsigned off = p * row + kz;
        load_kept<N, 0>(v, p, kz < D::NZ, [&](auto s) { return at32(src, off + (unsigned)CS::row(s.value) * row); });
    };
    {
        constexpr int ITEMS = 6 * C::KG;
        float2 v[V], nxt[V];
        if (warp < ITEMS) load(v, warp);
        __syncthreads();   // twiddle table
        for (int item = warp; item < ITEMS; item += WPB) {
            if (item + WPB < ITEMS) load(nxt, item + WPB);   // in flight during this transform
            fft_line<N, false, 0, true, true>(v, p, tw, at, WarpSync());
            float2 *dst = plane + (item / C::KG) * FS + p * PITCH + item % C::KG * C::CW + c;
#pragma unroll
            for (int i = 0; i < V; ++i) {
                dst[CS::out(i) * PITCH] = v[i];
                v[i] = nxt[i];
            }
        }
    }
    __syncthreads();

    // ---- z pass on the plane's rows, in place ----
    {
        const int line = lane / P, q = lane % P;
        WarpTw<N, 0> TW;
        TW.init(q, g.tw);
        float2 *myrow = buf + line * WPadV<N, 0>::SROW;
        float umax = 0.f, nzp[ZV];
        float2 *pend = nullptr;   // row whose n_z waits in nzp
        for (int gr = warp; gr < C::GR; gr += WPB) {
            float2 *X = plane + (gr * LPW + line) * PITCH;
            float2 a[ZV], b[ZV], e[ZV];
            PairSlots<N, 0, 0>::load(a, X, X + FS, q);
            PairSlots<N, 0, 0>::load(b, X + 2 * FS, X + 3 * FS, q);
            PairSlots<N, 0, 0>::load(e, X + 4 * FS, X + 5 * FS, q);
            fft_line_warp_pad<N, false, 0, true>(a, q, TW, myrow);
            fft_line_warp_pad<N, false, 0, true>(b, q, TW, myrow);
            fft_line_warp_pad<N, false, 0, true>(e, q, TW, myrow);
            // a = ux + i uy, b = uz + i wx, e = wy + i wz; max|u| of the first stage only (CFL step)
            if (stage_idx == 0) {
#pragma unroll
                for (int i = 0; i < ZV; ++i) umax = fmaxf(umax, fmaxf(fabsf(a[i].x), fmaxf(fabsf(a[i].y), fabsf(b[i].x))));
            }
            float nz[ZV];
#pragma unroll
            for (int i = 0; i < ZV; ++i) {
                const float ux = a[i].x, uy = a[i].y, uz = b[i].x;
                const float wx = b[i].y, wy = e[i].x, wz = e[i].y;
                a[i] = make_float2(uy * wz - uz * wy, uz * wx - ux * wz);
                nz[i] = ux * wy - uy * wx;
            }
            forward_pair_store_shfl<N, 0>(a, q, line, TW, myrow, X, X + FS);
            if (pend) {
#pragma unroll
                for (int i = 0; i < ZV; ++i) a[i] = make_float2(nzp[i], nz[i]);
                forward_pair_store_shfl<N, 0>(a, q, line, TW, myrow, pend, X + 2 * FS);
                pend = nullptr;
            } else {
#pragma unroll
                for (int i = 0; i < ZV; ++i) nzp[i] = nz[i];
                pend = X + 2 * FS;
            }
        }
        if (pend) {
            float2 w[ZV];
#pragma unroll
            for (int i = 0; i < ZV; ++i) w[i] = make_float2(nzp[i], 0.f);
            forward_pair_store_shfl<N, 0>(w, q, line, TW, myrow, pend, nullptr);
        }
        if (stage_idx == 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) umax = fmaxf(umax, __shfl_xor_sync(0xffffffffu, umax, o));
            if (lane == 0 && warp < C::GR) atomicMax(&md[g.first + m].umax_bits[0], __float_as_uint(umax));
        }
    }
    __syncthreads();

    // ---- forward y: the plane's columns back into buffer A (kept ky only) ----
    for (int item = warp; item < 3 * C::KG; item += WPB) {
        const int kz = item % C::KG * C::CW + c;
        const float2 *src = plane + (item / C::KG) * FS + p * PITCH + kz;
        float2 *dst = A + (long long)(item / C::KG) * D::SA;
        const unsigned off = p * row + kz;
        float2 v[V];
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] = src[CS::in(i) * PITCH];   // zero past the kept kz
        fft_line<N, true, 0, false, true>(v, p, tw, at, WarpSync());
        store_kept<N, 0>(v, p, kz < D::NZS,
                         [&](auto s, float2 w) { at32(dst, off + (unsigned)CS::row(s.value) * row) = w; });
    }
}

}  // namespace ens
