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
// Measured (us per step, mean of 200 graph replays between two events, fixed step,
// RK3 but for 1 x 32^3 with RK2; separate passes with 8-column y tiles -> this
// kernel, both with the split last pass): 1 x 32^3 49 -> 41, 16 x 32^3 105 -> 85,
// 64 x 16^3 101 -> 71, 1 x 64^3 84 -> 74, 4 x 64^3 123 -> 100, 16 x 64^3 338 -> 260,
// 64 x 64^3 1208 -> 969.
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

// grid (N + fin, members), block 32 * WPB.  fin: the block past the planes ends the
// previous stage of its member (k_finish's work, which this pass does not need
// and the next update does; a launch less)
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
    if (blockIdx.x == N) {
        // the partial sums of the k_chain launch before: one per column tile
        finish_block(md, g.partial, g.partial_blocks, g.NK * g.NZp / kTile, stage_idx - 1, 0, 0, g.first + blockIdx.y,
                     reinterpret_cast<double *>(sm));
        return;
    }
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

// Last pass of a stage and first pass of the next in one launch, for the small
// grids (N <= 64): forward x transform of the three components, RK update, and
// the inverse x transforms of the next stage's u and omega, all on the same
// columns, so the new state goes from the update into the transforms in
// registers.  Thread (c, p) holds the positions p, p + P, p + 2 P, ... of its
// column after the forward transform and needs the same ones before the
// inverse (both passes of a two-pass plan deal positions out modulo P), and it
// has all three components of each, which is what projection, forcing and
// omega = i k x u need.  Registers bound the use: three lines of V values and
// two in work (V = 8 up to 64^3).
// One launch per stage less, the state's second read and the staged tile gone;
// the stage's end moves into the next PLANE launch.  Step (measured as for k_plane;
// fused last pass on 8-column tiles -> chained): 1 x 32^3 37 -> 31 us, 16 x 32^3 78 -> 64,
// 64 x 16^3 63 -> 53, 1 x 64^3 74 -> 57, 4 x 64^3 102 -> 84.  With more members of 64^3
// the split last pass catches up: chained against split 148 / 154 us at 8, 211 / 216
// at 12, 275 / 260 at 16, 985 / 969 at 64.
template <int N>
struct ChainCfg {
    static constexpr int T = kTile;
    using CS = ColSlots<N, 0>;
    static constexpr int V = CS::V, P = CS::P, TH = T * P;
    // output slot that holds the position of input slot i
    static __host__ __device__ constexpr int out_of(int i)
    {
        for (int o = 0; o < V; ++o)
            if (CS::out(o) == CS::in(i)) return o;
        return -1;
    }
    static constexpr size_t smem() { return smem_cols<N, T>(); }
};

// kept mode I of the three lines: the stage update of (n0, n1, n2) into u, and to dst
template <int N, int I = 0>
struct ChainUpdate {
    using CS = ColSlots<N, 0>;
    using D = Dims<N>;
    static constexpr unsigned rowU = D::NK * D::NZP, SU = (unsigned)D::SU;
    template <class Ld>
    static __device__ __forceinline__ void run(const UpdCoef &c, int p, int ky, int kz, bool valid, bool stored,
                                               unsigned off, const Ld &ld, float2 *dst, float2 *u0, float2 *u1,
                                               float2 *u2, float &se, float &sd, float &sb)
    {
        if constexpr (I < CS::V) {
            constexpr int C = CS::out(I);
            constexpr auto kind = CS::kind(C);
            if constexpr (kind == CS::kZero) {
                u0[I] = u1[I] = u2[I] = make_float2(0.f, 0.f);
            } else {
                bool keep = true;
                if constexpr (kind == CS::kLowMixed) keep = p <= CS::KC - C;
                if constexpr (kind == CS::kNegMixed) keep = p >= N - CS::KC - C;
                const unsigned o = off + (unsigned)CS::row(C) * rowU;
                float2 un[3], us[3], n[3] = {u0[I], u1[I], u2[I]}, out[3];
                ld(o, keep && valid, un, us);
                bool band;
                float k2;
                const float a2 = update_mode(c, p + CS::wave(C), ky, kz, n, un, us, out, band, k2);
                const bool real = keep && valid;
                const float s = real ? (kz == 0 ? 1.f : 2.f) * a2 : 0.f;   // Hermitian multiplicity
                se += 0.5f * s;
                sd += c.nu * k2 * s;
                if (band) sb += 0.5f * s;
                u0[I] = real ? out[0] : make_float2(0.f, 0.f);
                u1[I] = real ? out[1] : make_float2(0.f, 0.f);
                u2[I] = real ? out[2] : make_float2(0.f, 0.f);
                if (keep && stored) {
                    at32(dst, o) = u0[I];
                    at32(dst, o + SU) = u1[I];
                    at32(dst, o + 2 * SU) = u2[I];
                }
            }
            ChainUpdate<N, I + 1>::run(c, p, ky, kz, valid, stored, off, ld, dst, u0, u1, u2, se, sd, sb);
        }
    }
};

// first-pass inputs of an inverse transform from a line of modes u (output
// slots): u, or (DX) i kx u
template <int N, bool DX, int I = 0>
__device__ __forceinline__ void chain_input(float2 *v, const float2 *u, int p)
{
    using CS = ColSlots<N, 0>;
    if constexpr (I < CS::V) {
        constexpr int C = CS::in(I), O = ChainCfg<N>::out_of(I);
        if constexpr (CS::kind(C) == CS::kZero) v[I] = make_float2(0.f, 0.f);
        else if constexpr (DX) v[I] = mul_i(cscale(u[O], (float)(p + CS::wave(C))));
        else v[I] = u[O];
        chain_input<N, DX, I + 1>(v, u, p);
    }
}

// grid (NK NZp / 16, members), block 16 P
template <int N>
__global__ void __launch_bounds__(ChainCfg<N>::TH, 512 / ChainCfg<N>::TH)
k_chain(Geo g, MemberDev *md, int stage)
{
    using C = ChainCfg<N>;
    using CS = ColSlots<N, 0>;
    using D = Dims<N>;
    constexpr int V = C::V, T = C::T;
    extern __shared__ __align__(16) float2 sm[];
    float2 *tw = sm, *buf = sm + N;
    load_col_twiddles<N, 0>(tw, g.tw);
    const int c = threadIdx.x % T, p = threadIdx.x / T, m = blockIdx.y;
    const unsigned col = blockIdx.x * T + c;                          // (ky, kz) flat
    const int iy = col / D::NZP, kz = col % D::NZP;
    const bool valid = kz < D::NZ, stored = kz < D::NZS;
    float2 *A = g.A + (long long)m * kFields * D::SA;
    const unsigned a0 = ((unsigned)iy * N + p) * D::NZP + kz;
    auto at = [&](int pos) { return &buf[pos * T + c]; };
    float2 u0[V], u1[V], u2[V];
    auto load = [&](float2 *v, int q) {
#pragma unroll
        for (int i = 0; i < V; ++i)
            v[i] = valid ? at32(A + q * D::SA, a0 + (unsigned)CS::in(i) * D::NZP) : make_float2(0.f, 0.f);
    };
    load(u0, 0);
    load(u1, 1);
    load(u2, 2);
    fft_line<N, true, 0>(u0, p, tw, at);
    fft_line<N, true, 0>(u1, p, tw, at);
    fft_line<N, true, 0>(u2, p, tw, at);
    // stage update: the new state to S (this is not the last stage) and in registers
    const UpdCoef uc = upd_coef<N>(md[g.first + m], stage);
    const int kyi = iy <= D::KC ? iy : iy - D::NK;
    const long long base = (long long)m * 3 * D::SU;
    const float2 *U = g.U + base, *S = g.S + base;
    const unsigned SU = (unsigned)D::SU;
    float se = 0.f, sd = 0.f, sb = 0.f;
    auto ld = [&](unsigned o, bool ok, float2 (&un)[3], float2 (&us)[3]) {
#pragma unroll
        for (int q = 0; q < 3; ++q) un[q] = ok ? at32(U, o + q * SU) : make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 3; ++q) us[q] = ok && stage != 0 ? at32(S, o + q * SU) : un[q];
    };
    ChainUpdate<N>::run(uc, p, kyi, kz, valid, stored, p * (unsigned)(D::NK * D::NZP) + col, ld, g.S + base, u0, u1, u2,
                        se, sd, sb);
    // next stage: u and omega = i k x u, transformed along x (as inv_x_body)
    const float ky = (float)kyi, kzf = (float)kz;
    auto store = [&](const float2 *v, int f) {
        if (stored) {
            float2 *dst = A + f * D::SA;
#pragma unroll
            for (int i = 0; i < V; ++i) at32(dst, a0 + (unsigned)CS::out(i) * D::NZP) = v[i];
        }
    };
    float2 Ua[V], Ub[V];
    chain_input<N, false>(Ua, u1, p);
    fft_line<N, false, 0, true>(Ua, p, tw, at);                       // uy
    store(Ua, 1);
    chain_input<N, false>(Ub, u2, p);
    fft_line<N, false, 0, true>(Ub, p, tw, at);                       // uz
    store(Ub, 2);
#pragma unroll
    for (int i = 0; i < V; ++i)
        Ua[i] = mul_i(make_float2(ky * Ub[i].x - kzf * Ua[i].x, ky * Ub[i].y - kzf * Ua[i].y));
    store(Ua, 3);                                                     // omega_x
    chain_input<N, false>(Ua, u0, p);
    fft_line<N, false, 0, true>(Ua, p, tw, at);                       // ux
    store(Ua, 0);
    chain_input<N, true>(Ub, u2, p);
    fft_line<N, false, 0, true>(Ub, p, tw, at);                       // i kx uz
#pragma unroll
    for (int i = 0; i < V; ++i)
        Ub[i] = make_float2(-kzf * Ua[i].y - Ub[i].x, kzf * Ua[i].x - Ub[i].y);
    store(Ub, 4);                                                     // omega_y
    chain_input<N, true>(Ub, u1, p);
    fft_line<N, false, 0, true>(Ub, p, tw, at);                       // i kx uy
#pragma unroll
    for (int i = 0; i < V; ++i) Ub[i] = make_float2(Ub[i].x + ky * Ua[i].y, Ub[i].y - ky * Ua[i].x);
    store(Ub, 5);                                                     // omega_z
    __syncthreads();   // buf is reused as reduction scratch
    double vals[3] = {(double)se, (double)sd, (double)sb};
    double *out = g.partial + ((long long)(g.first + m) * g.partial_blocks + blockIdx.x) * 4;
    block_sum_to<3>(out, vals, reinterpret_cast<double *>(buf));
}

}  // namespace ens
