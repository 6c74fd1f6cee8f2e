// Non-templated kernels (reductions, initial field, twiddles, edges, mixture)
// and the table of per-N pass launchers (each grid size compiles in its own
// translation unit, ens_sized.cu).
#include "ens_launch.h"
#include "ens_plane.cuh"
#include "ens_stats.cuh"
#include "ens_znl.cuh"

#include <climits>
#include <cmath>

namespace ens {

// ---------------------------------------------------------------------------
// spectral sums of U (init / after upload), same partial layout as FXU: block b
// of a member adds the modes [b chunk, (b + 1) chunk).  Bound by HBM (the state
// read once): a thread per (ky, kz) column looping over kx, 129 blocks per
// 256^3 member, read it at 1.5 TB/s (45 us per member; chunks: 14 us).
// ---------------------------------------------------------------------------
constexpr int kSumThreads = 256;
__global__ void __launch_bounds__(kSumThreads)
k_state_sums(Geo g, const MemberDev *md, int chunk)
{
    const int m = blockIdx.y;
    const MemberDev &d = md[g.first + m];
    const float nu = (float)d.nu;
    const int lo2 = d.band_lo2, hi2 = d.band_hi2;
    const unsigned rowU = g.NK * g.NZp, end = (unsigned)min((long long)(blockIdx.x + 1) * chunk, g.sU);
    const float2 *U = g.U + (long long)m * 3 * g.sU;
    float se = 0.f, sd = 0.f, sb = 0.f;
#pragma unroll 4
    for (unsigned i = blockIdx.x * chunk + threadIdx.x; i < end; i += kSumThreads) {
        const int ix = i / rowU, rem = i % rowU;
        const int iy = rem / g.NZp, kz = rem % g.NZp;
        if (kz >= g.NZ) continue;
        float a2 = 0.f;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float2 v = U[q * g.sU + i];
            a2 += v.x * v.x + v.y * v.y;
        }
        const int kx = ix <= g.kc ? ix : ix - g.NK, ky = iy <= g.kc ? iy : iy - g.NK;
        const int k2i = kx * kx + ky * ky + kz * kz;
        const float w = (kz == 0 ? 1.f : 2.f) * a2;
        se += 0.5f * w;
        sd += nu * (float)k2i * w;
        if (k2i >= lo2 && k2i <= hi2) sb += 0.5f * w;
    }
    __shared__ double scratch[(kSumThreads / 32) * 3];
    double vals[3] = {(double)se, (double)sd, (double)sb};
    double *out = g.partial + ((long long)(g.first + m) * g.partial_blocks + blockIdx.x) * 4;
    block_sum_to<3>(out, vals, scratch);
}

// End of a stage, a block per member of a group, from the nblk partial sums per
// member that the launch before wrote (9993 for a 512^3 member).  Steps with 256
// threads against one warp: 512^3 8.80 / 9.25 ms, 384^3 4.00 / 4.17, 128^3 0.164 / 0.170.
// Up to 64^3, with few partials, one warp is the shorter chain: 64 x 16^3 53.4 against
// 54.7 us, 16 x 32^3 63.5 / 65.5, 16 x 64^3 260 / 263, 1 x 32^3 and one 64^3 the same.  (The
// update pass's last CTA doing it, which saves the launch, measured 1% better at
// 512^3 but 4% worse at 16 x 64^3: a fence, a counter and this sum at the end of
// a short kernel.)
constexpr int kFinishThreads = 256;
__global__ void __launch_bounds__(kFinishThreads)
k_finish(MemberDev *md, const double *__restrict__ partial, int partial_blocks, int nblk, int first, int stage,
         int last_stage, int mode)
{
    __shared__ double scratch[3 * kFinishThreads / 32];
    finish_block(md, partial, partial_blocks, nblk, stage, last_stage, mode, first + blockIdx.x, scratch);
}

// ---------------------------------------------------------------------------
// initial field: shell targets E0(s) ~ s^4 exp(-s^2/2), total init_energy
// ---------------------------------------------------------------------------
__global__ void k_ic_factors(MemberDev *md, Geo g)
{
    const int m = blockIdx.x;
    double *shell = g.shell + (long long)m * g.shells;
    __shared__ double total;
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int s = 1; s < g.shells; ++s)
            if (shell[s] > 0.0) t += pow((double)s, 4.0) * exp(-0.5 * s * s);
        total = t;
    }
    __syncthreads();
    const double E0 = md[g.first + m].init_energy;
    for (int s = threadIdx.x; s < g.shells; s += blockDim.x) {
        double f = 0.0;
        if (s > 0 && shell[s] > 0.0 && total > 0.0)
            f = sqrt(E0 * pow((double)s, 4.0) * exp(-0.5 * s * s) / (total * shell[s]));
        shell[s] = f;   // shell sums are replaced by the rescaling factors
    }
}

__global__ void k_ic_scale(Geo g)
{
    const int m = blockIdx.y;
    const long long ncols = (long long)g.NK * g.NZp;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;   // (kx, ky, kz) flat
    if (idx >= (long long)g.NK * ncols) return;
    const int ix = (int)(idx / ncols);
    const int col = (int)(idx % ncols);
    const int iy = col / g.NZp, kz = col % g.NZp;
    float2 *U = g.U + (long long)m * 3 * g.sU + idx;
    if (kz >= g.NZ) {
        for (int q = 0; q < 3; ++q) U[q * g.sU] = make_float2(0.f, 0.f);
        return;
    }
    const int kx = ix <= g.kc ? ix : ix - g.NK, ky = iy <= g.kc ? iy : iy - g.NK;
    const int s = (int)lrint(sqrt((double)(kx * kx + ky * ky + kz * kz)));
    const float f = (float)g.shell[(long long)m * g.shells + s];
    for (int q = 0; q < 3; ++q) U[q * g.sU] = cscale(U[q * g.sU], f);
}

__global__ void k_twiddles(float2 *tw, int N)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        double s, c;
        sincospi(-2.0 * (double)i / (double)N, &s, &c);
        tw[i] = make_float2((float)c, (float)s);
    }
}

__global__ void k_edges(float *eq, float *er, float *et, float *eg, int nq, int nt, int ng, double q_lim,
                        double r_lim, double t_lo, double t_hi, double g_lim)
{
    for (int b = threadIdx.x; b <= ng; b += blockDim.x) eg[b] = (float)(-g_lim + 2.0 * g_lim * (double)b / (double)ng);
    for (int b = threadIdx.x; b <= nq; b += blockDim.x) {
        eq[b] = (float)(-q_lim + 2.0 * q_lim * (double)b / (double)nq);
        er[b] = (float)(-r_lim + 2.0 * r_lim * (double)b / (double)nq);
    }
    for (int b = threadIdx.x; b <= nt; b += blockDim.x)
        et[b] = (float)pow(10.0, t_lo + (t_hi - t_lo) * (double)b / (double)nt);
}

// one block of kNMom x 8 threads per member: the partial moments of its blocks
constexpr int kFinishSlices = 8;
__global__ void __launch_bounds__(kNMom * kFinishSlices)
k_finish_stats(const double *__restrict__ mom_partial, int stride, int blocks, double *moments, int first,
               int accumulate)
{
    const int gm = first + blockIdx.x, q = threadIdx.x % kNMom, slice = threadIdx.x / kNMom;
    __shared__ double part[kNMom * kFinishSlices];
    double s = 0.0;
    const double *pp = mom_partial + (long long)gm * stride * kNMom;
    for (int b = slice; b < blocks; b += kFinishSlices) s += pp[(long long)b * kNMom + q];
    part[threadIdx.x] = s;
    __syncthreads();
    if (slice != 0) return;
    for (int k = 1; k < kFinishSlices; ++k) s += part[k * kNMom + q];
    moments[gm * kNMom + q] = accumulate ? moments[gm * kNMom + q] + s : s;
}

// ---------------------------------------------------------------------------
// mixture (Sec. II, Eqs. ensemble_hypothesis / pdf_superposition; Sec. IV,
// Eq. gaussian_lambda_pdf and the lambda-bin weights; Appendix,
// Eq. truncated_gaussian), FP64
// ---------------------------------------------------------------------------
__device__ double norm_cdf(double x) { return 0.5 * erfc(-x * 0.70710678118654752440); }
__device__ double norm_sf(double x) { return 0.5 * erfc(x * 0.70710678118654752440); }

__device__ double interval_mass(double a, double b, double mu, double sigma)
{
    const double za = (a - mu) / sigma, zb = (b - mu) / sigma;
    if (za >= 0.0) return norm_sf(za) - norm_sf(zb);
    return norm_cdf(zb) - norm_cdf(za);
}

// mu of the truncated Gaussian so that int P e^lambda = 1 (bisection in logs)
__device__ double trunc_mu(double c, double Z)
{
    const double sigma = sqrt(9.0 * c * Z);
    double lo = -4.5 * c * Z - 10.0 * sigma - 1.0, hi = 10.0;
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        const double f = mid + 0.5 * sigma * sigma + log(norm_cdf((Z - mid - sigma * sigma) / sigma)) -
                         log(norm_cdf((Z - mid) / sigma));
        if (f < 0.0) lo = mid;
        else hi = mid;
    }
    return 0.5 * (lo + hi);
}

// sum of one value per thread over the block (at most 1024 threads, whole
// warps), for every thread
__device__ double block_total(double v, double *scratch)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v += scratch[k];
    return v;
}

// doubles as integers in the same order (-0 and +0 the same), and back; a NaN
// above everything, where it is nobody's neighbour
__device__ long long order_key(double x)
{
    if (x != x) return LLONG_MAX;
    const long long b = __double_as_longlong(x + 0.0);
    return b >= 0 ? b : LLONG_MIN - b;
}
__device__ double from_key(long long k) { return __longlong_as_double(k >= 0 ? k : LLONG_MIN - k); }

// one block, a thread per member (whole warps)
__global__ void k_mix_weights(const double *lam, int n, MixWeightArgs wa, double *w, double *covered)
{
    const int i = threadIdx.x;
    __shared__ double scratch[32];
    __shared__ long long key[1024];   // lambdas as integers of the same order (FP64 compares run on two lanes per SM)
    if (i < n) key[i] = order_key(lam[i]);
    __syncthreads();
    double v = 0.0;
    if (i < n) {
        const double li = lam[i];
        const long long ki = key[i];
        long long kprev = LLONG_MIN, knext = LLONG_MAX;
        int mult = 0;
        for (int j = 0; j < n && li == li; ++j) {
            const long long kj = key[j];
            if (kj == ki) ++mult;
            else if (kj < ki && kj > kprev) kprev = kj;
            else if (kj > ki && kj < knext) knext = kj;
        }
        const double prev = kprev == LLONG_MIN ? -INFINITY : from_key(kprev);
        const double next = knext == LLONG_MAX ? INFINITY : from_key(knext);
        double lo, hi;
        if (prev == -INFINITY && next == INFINITY) {
            lo = -INFINITY;
            hi = INFINITY;
        } else {
            lo = prev == -INFINITY ? li - 0.5 * (next - li) : 0.5 * (prev + li);
            hi = next == INFINITY ? li + 0.5 * (li - prev) : 0.5 * (li + next);
        }
        if (wa.kind == 2) {
            v = wa.user[i];
        } else if (wa.kind == 0 && wa.Z == 0.0) {
            v = (lo <= 0.0 && 0.0 < hi) ? 1.0 / mult : 0.0;
        } else if (wa.kind == 0 || wa.kind == 1) {
            const double mu = wa.kind == 0 ? -4.5 * wa.c * wa.Z : wa.mu;
            const double sg = wa.kind == 0 ? sqrt(9.0 * wa.c * wa.Z) : wa.sigma;
            v = interval_mass(lo, hi, mu, sg) / mult;
        } else if (wa.kind == 3) {
            const double mu = trunc_mu(wa.c, wa.Z), sg = sqrt(9.0 * wa.c * wa.Z);
            const double b = fmin(hi, wa.Z);
            v = b > lo ? interval_mass(lo, b, mu, sg) / norm_cdf((wa.Z - mu) / sg) / mult : 0.0;
        }
    }
    const double tot = block_total(v, scratch);
    if (i == 0) *covered = tot;
    if (i < n) w[i] = (wa.renormalize && tot > 0.0) ? v / tot : v;
}

// skewness / flatness / hyper-flatness of gradient components from mixed
// moments (Sec. VII, Eq. def_skewness_flatness and the skewness prediction),
// isotropy-averaged over the 3 longitudinal and 6 transverse components
__device__ void mix_ratios(const double *mom_mix, double *ratios)
{
    const int lon[3] = {0, 4, 8}, tra[6] = {1, 2, 3, 5, 6, 7};
    double L[4] = {0, 0, 0, 0}, T[4] = {0, 0, 0, 0};
    for (int q = 0; q < 4; ++q) {
        for (int c = 0; c < 3; ++c) L[q] += mom_mix[4 * lon[c] + q] / 3.0;
        for (int c = 0; c < 6; ++c) T[q] += mom_mix[4 * tra[c] + q] / 6.0;
    }
    ratios[0] = L[1] / (L[0] * sqrt(L[0]));
    ratios[1] = L[2] / (L[0] * L[0]);
    ratios[2] = T[2] / (T[0] * T[0]);
    ratios[3] = L[3] / (L[0] * L[0] * L[0]);
    ratios[4] = T[3] / (T[0] * T[0] * T[0]);
}

// Mixed PDF, moments and moment ratios.  Block b < last: kMixBins bins, the
// members shared out over kMixSlices threads per bin (coalesced over the
// bins); the last block: the moments and the ratios.  Bound by the latency of
// the counts' loads and by FP64, two lanes per SM and clock here, hence the
// spread over all SMs and one division per member (weight / points) instead of
// one per member and bin: 64 members x 4608 bins 184 us with a thread per bin
// looping over the members, 18 blocks.
constexpr int kMixBins = 32, kMixSlices = 8;

__global__ void __launch_bounds__(kMixBins * kMixSlices)
k_mix_pdf(const unsigned long long *__restrict__ counts, const double *__restrict__ moments,
          const double *__restrict__ w, int n, MixPdfArgs a, double *pdf, double *mom_mix, double *ratios)
{
    constexpr int TH = kMixBins * kMixSlices;
    const int L = a.counts_len;
    const int off_c = a.nq * a.nq + 2 * a.nt;
    __shared__ double wn[1024], part[TH], mom[kNMom];
    __shared__ bool points[1024];
    for (int i = threadIdx.x; i < n; i += TH) {
        const double npts = (double)counts[(long long)i * L + off_c + 6];
        wn[i] = npts > 0.0 ? w[i] / npts : 0.0;
        points[i] = npts > 0.0;
    }
    __syncthreads();
    if (blockIdx.x + 1 < gridDim.x) {
        const int b = blockIdx.x * kMixBins + threadIdx.x % kMixBins, slice = threadIdx.x / kMixBins;
        const bool in = b < mix_pdf_len(a);
        // gradient bins follow the 8 counters; 3 longitudinal and 6
        // transverse samples per grid point
        const bool grad = b >= off_c;
        double s = 0.0;
        if (in) {
            const unsigned long long *c = counts + (grad ? b + 8 : b);
#pragma unroll 4
            for (int i = slice; i < n; i += kMixSlices) s += wn[i] * (double)c[(long long)i * L];
        }
        part[threadIdx.x] = s;
        __syncthreads();
        if (slice == 0 && in) {
            for (int k = 1; k < kMixSlices; ++k) s += part[k * kMixBins + threadIdx.x];
            double width = b < a.nq * a.nq ? a.dq * a.dr : a.dt;
            if (grad) width = a.dg * (b < off_c + a.ng ? 3.0 : 6.0);
            pdf[b] = s / width;
        }
        return;
    }
    constexpr int MS = TH / kNMom;   // member slices of the moments
    const int q = threadIdx.x % kNMom, slice = threadIdx.x / kNMom;
    double s = 0.0;
    if (slice < MS)
        for (int i = slice; i < n; i += MS) {
            const double mi = moments[(long long)i * kNMom + q];
            // a member without points stays out, whatever its sums hold (0 x NaN is no zero)
            if (points[i]) s += wn[i] * mi;
        }
    part[threadIdx.x] = s;
    __syncthreads();
    if (slice == 0) {
        for (int k = 1; k < MS; ++k) s += part[k * kNMom + q];
        mom[q] = s;
        mom_mix[q] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) mix_ratios(mom, ratios);
}

// ---------------------------------------------------------------------------
// launch dispatch
// ---------------------------------------------------------------------------
#define ENS_SUPPORTED_N(X) X(16) X(32) X(64) X(128) X(256) X(384) X(512)

bool supported_n(int N)
{
#define X(n) if (N == n) return true;
    ENS_SUPPORTED_N(X)
#undef X
    return false;
}

// The stage's middle in one launch where a plane fits (N <= 64) and the tuning
// asks for the plain variants; the failure test needs the z pass's bulk copies.
bool plane_fused(const Geo &g)
{
    return has_plane(g.N) && g.z_mode == 0 && g.tile_y == kTile && g.z_skip_member < 0;
}

// and its last pass does the next stage's inverse x transforms (k_chain)
bool chain_fused(const Geo &g) { return plane_fused(g) && g.fx_split == 0 && g.tile_x == kTile && g.plan_x == 0; }

int plan_threads(int N)
{
#define X(n) if (N == n) return PlanInfo<n>::P;
    ENS_SUPPORTED_N(X)
#undef X
    return 0;
}

size_t stats_smem(int N, int nq, int nt, int ng)
{
#define X(n) if (N == n) return smem_stats<n>(nq, nt, ng);
    ENS_SUPPORTED_N(X)
#undef X
    return 0;
}

int stats_blocks(int N)
{
#define X(n) if (N == n) return stats_ctas<n>() * stats_most_sub<n>();
    ENS_SUPPORTED_N(X)
#undef X
    return 0;
}

const SizedOps *sized_ops(int N)
{
#define X(n) if (N == n) return sized_ops_for<n>();
    ENS_SUPPORTED_N(X)
#undef X
    return nullptr;
}

cudaError_t prepare_kernels(int N, int smem_optin)
{
    const SizedOps *o = sized_ops(N);
    return o ? o->prepare(smem_optin) : cudaErrorInvalidValue;
}

bool plan_variant_available(int N) { return has_plan_variant(N); }

int znl_ctas_per_sm(int N, int var)
{
    const SizedOps *o = sized_ops(N);
    return o ? o->znl_ctas_per_sm(var) : 0;
}

bool zplan_variant_available(int N) { return has_zplan_variant(N); }

bool fx_ws_available(int N)
{
    const SizedOps *o = sized_ops(N);
    return o && o->fx_ws();
}

void launch_pass(Pass pass, int mode, const Geo &g, MemberDev *md, const HistDev *h, int stage, int last, int arg,
                 cudaStream_t s)
{
    if (const SizedOps *o = sized_ops(g.N)) o->launch(pass, mode, g, md, h, stage, last, arg, s);
}

// Partial sums per member that FX mode 0 (or CHAIN) writes with g's variants:
// one per column tile of the fused pass, one per kUpdChunk modes of the split one.
static int update_partials(const Geo &g)
{
    if (g.fx_split == 1) return (int)((g.sU + kUpdChunk - 1) / kUpdChunk);
    return g.NK * g.NZp / (g.fx_split == 2 ? kTile : g.tile_x);
}

static void launch_finish(const Geo &g, MemberDev *md, int nblk, int stage, int last, int mode, cudaStream_t s)
{
    k_finish<<<g.members, g.N <= 64 ? 32 : kFinishThreads, 0, s>>>(md, g.partial, g.partial_blocks, nblk, g.first, stage,
                                                                   last, mode);
}

void launch_stage_end(const Geo &g, MemberDev *md, int stage, int last, cudaStream_t s)
{
    launch_finish(g, md, update_partials(g), stage, last, 0, s);
}

void launch_state_sums(const Geo &g, MemberDev *md, cudaStream_t s)
{
    const int blocks = (int)((g.sU + kUpdChunk - 1) / kUpdChunk);
    k_state_sums<<<dim3(blocks, g.members), kSumThreads, 0, s>>>(g, md, (int)((g.sU + blocks - 1) / blocks));
    launch_finish(g, md, blocks, 0, 0, 1, s);
}

void launch_ic(const Geo &g, MemberDev *md, cudaStream_t s)
{
    // white noise -> forward along z, y, x with projection and shell sums
    cudaMemsetAsync(g.shell, 0, sizeof(double) * g.shells * g.members, s);
    launch_pass(Pass::Z, 1, g, md, nullptr, 0, 0, 0, s);
    launch_pass(Pass::FY, 0, g, md, nullptr, 0, 0, 0, s);
    launch_pass(Pass::FX, 2, g, md, nullptr, 0, 0, 0, s);
    k_ic_factors<<<g.members, 128, 0, s>>>(md, g);
    const long long modes = (long long)g.NK * g.NK * g.NZp;
    dim3 grid((unsigned)((modes + 255) / 256), g.members);
    k_ic_scale<<<grid, 256, 0, s>>>(g);
}

void launch_twiddles(float2 *tw, int N, cudaStream_t s) { k_twiddles<<<(N + 255) / 256, 256, 0, s>>>(tw, N); }

void launch_edges(float *eq, float *er, float *et, float *eg, int nq, int nt, int ng, double q_lim, double r_lim,
                  double t_lo, double t_hi, double g_lim, cudaStream_t s)
{
    k_edges<<<1, 256, 0, s>>>(eq, er, et, eg, nq, nt, ng, q_lim, r_lim, t_lo, t_hi, g_lim);
}

// the statistics pass's bin rule alone, on values already in an axis's
// units (0 Q, 1 R, 2 log10 tail, 3 gradient component), edges in global
// memory: the device functions k_z_stats calls per point
__global__ void k_bin_check(HistDev h, int axis, const float *__restrict__ x, int n, int *__restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float v = x[i];
    int b;
    if (axis == 0) b = bin_lin(v, lin_map(h.q_lo, h.q_inv_w), h.edges_q, h.nq);
    else if (axis == 1) b = bin_lin(v, lin_map(h.r_lo, h.r_inv_w), h.edges_r, h.nq);
    else if (axis == 2) b = bin_log(v, log_map(h.t_lo, h.t_inv_w), h.edges_t, h.nt);
    else b = bin_lin(v, lin_map(h.g_lo, h.g_inv_w), h.edges_g, h.ng);
    out[i] = b;
}

void launch_bin_check(const HistDev &h, int axis, const float *x, int n, int *out, cudaStream_t s)
{
    if (n > 0) k_bin_check<<<(n + 255) / 256, 256, 0, s>>>(h, axis, x, n, out);
}

void launch_finish_stats(const Geo &g, double *moments, int accumulate, cudaStream_t s)
{
    const SizedOps *o = sized_ops(g.N);
    if (!o) return;
    k_finish_stats<<<g.members, kNMom * kFinishSlices, 0, s>>>(g.mom_partial, g.mom_blocks,
                                                               o->stats_used(g.members, g.sms), moments, g.first,
                                                               accumulate);
}

void launch_mixture(const double *lam, int n, const MixWeightArgs &wa, const unsigned long long *counts,
                    const double *moments, const MixPdfArgs &pa, double *w, double *covered, double *pdf,
                    double *mom_mix, double *ratios, cudaStream_t s)
{
    k_mix_weights<<<1, (n + 31) / 32 * 32, 0, s>>>(lam, n, wa, w, covered);
    const int nb = mix_pdf_len(pa);
    k_mix_pdf<<<(nb + kMixBins - 1) / kMixBins + 1, kMixBins * kMixSlices, 0, s>>>(counts, moments, w, n, pa, pdf,
                                                                                   mom_mix, ratios);
}

}  // namespace ens
