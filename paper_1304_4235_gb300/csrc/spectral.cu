// Shielded photoionisation rate (Eq. gamma_shld) and ionisation equilibrium
// (App. C3, Eqs. dxdt / xroots / xphys).
//
// Gamma: for one origin with columns tau_k (threshold optical depth) and a
// binned spectrum (s_j = sigma_j / sigma_th, w_j with sum w_j = Gamma_thin),
//   Gamma / Gamma_thin = (1/R) sum_k sum_j w^_j exp(-s_j tau_k),  w^ = w / Gamma_thin.
// Each ray's inner sum is factored as exp(-s_min tau_k) S_k with
//   S_k = sum_j w^_j exp(-(s_j - s_min) tau_k)  in [w^_jmin, 1],
// so ln(Gamma_k / Gamma_thin) = -s_min tau_k + ln S_k never underflows; the
// rays are then combined with a log-sum-exp in double, which keeps tau_eff
// finite where Gamma itself underflows.
#include <algorithm>
#include <cmath>

#include "spectral_device.cuh"

namespace urchin {

namespace {

constexpr int kGammaThreads = 256;

// Threads (local, k) fold ray k of row `local` (fold_ray: the exponent of
// every bin formed without rounding error); the per-row log-sum-exp runs with
// one thread per row packed into the first lanes.
template <typename Real>
__global__ void __launch_bounds__(kGammaThreads) k_gamma(GammaJob J)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool kF32 = sizeof(Real) == 4;
    double* lk = reinterpret_cast<double*>(smem_raw);
    Real* e2 = reinterpret_cast<Real*>(lk + kGammaThreads);
    Real* wn = e2 + J.F;
    Real* e2t = kF32 ? wn + J.F : nullptr;
    __shared__ double sh[2];
    fold_prepare<Real>(J.s, J.w, J.F, e2, e2t, wn, nullptr, sh);
    const int rows_per_block = kGammaThreads / J.R;
    const int local = threadIdx.x / J.R;
    const int k = threadIdx.x % J.R;
    const double gthin = sh[0];
    const double smin = sh[1];
    for (int64_t row0 = (int64_t)blockIdx.x * rows_per_block; row0 < J.n_rows;
         row0 += (int64_t)gridDim.x * rows_per_block) {
        const int64_t row = row0 + local;
        if (local < rows_per_block && row < J.n_rows) {
            const Real tau = static_cast<const Real*>(J.tau)[row * J.row_stride + (int64_t)k * J.k_stride];
            Real S, S2;
            fold_ray<false>(tau, e2, e2t, wn, nullptr, J.F, S, S2);
            lk[local * J.R + k] = ray_lnrate(smin, tau, S);
        }
        __syncthreads();
        const int p = threadIdx.x;
        const int64_t prow = row0 + p;
        if (p < rows_per_block && prow < J.n_rows) {
            RayMean<Real> lse;
            for (int r = 0; r < J.R; ++r) lse.add(lk[p * J.R + r]);
            const double lmean = lse.mean(J.R);     // ln(Gamma / Gamma_thin)
            J.gamma_out[prow] = gthin * exp(lmean);
            if (J.tau_eff_out) J.tau_eff_out[prow] = (float)(-lmean);
        }
        __syncthreads();
    }
}

// The same with fewer threads than rays (fold_rows): the same bits.
template <typename Real>
__global__ void __launch_bounds__(kFoldThreads) k_gamma_rows(GammaJob J, FoldSplit sp)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FoldTable<Real> T(smem_raw, J.F);
    double* lk = reinterpret_cast<double*>(smem_raw + FoldTable<Real>::kBytes * (size_t)((J.F + 1) & ~1));
    __shared__ double sh[2];
    T.prepare(J.s, J.w, J.F, sh);
    const double gthin = sh[0];
    const Real* tau = static_cast<const Real*>(J.tau);
    fold_rows<Real>(
        sp, J.n_rows, J.R, J.F, T, gthin, sh[1], lk,
        [&](int64_t row, int k) { return tau[row * J.row_stride + (int64_t)k * J.k_stride]; },
        [&](int64_t row, double lmean) {
            J.gamma_out[row] = gthin * exp(lmean);
            if (J.tau_eff_out) J.tau_eff_out[row] = (float)(-lmean);
        });
}

// FP32: a thread for several rays where the rays still give 850 threads per SM
// two each (at 768 the last wave is nearly empty: 240000 rays, 1400 bins 0.231
// against 0.244 ms), and the spectrum's table (24 B per bin) leaves an SM its
// blocks.  An odd number of rays leaves one that is folded alone, which only many
// rows make up for (3 rays, 400000, 1000 bins 0.252 against 0.270, but 1200000,
// 100 bins faster by 7 %); with one or two rays there is nothing to gain.
// 12 rays, ms with a thread per ray / per several: 60000 rows, 50 / 400 / 1000
// bins 0.050 / 0.179 / 0.403 against 0.043 / 0.169 / 0.386, 400003 rows 0.243 /
// 1.03 / 2.40 against 0.167 / 0.96 / 2.33; 192 rays, 8000 rows, 50 / 400 bins
// 0.438 / 0.567 against 0.122 / 0.354.  Fewer rays: 2000 rows of 12 rays, 400 /
// 1000 bins 0.0252 / 0.0426 against 0.0363 / 0.0705 with two rays per thread;
// more bins: 2000 rows of 192 rays, 2000 bins 0.507 against 0.578.  FP64, whose
// pipe leaves nothing to fold together: only where a row's log-sum-exp outweighs
// its bins and the rows are many (192 rays, 8000 rows, 20 bins 3.19 against
// 1.90 ms; 48 rays, 10000 rows, 200 bins 4.38 against 4.90).
constexpr int kRowsMaxBins = 1400;

template <typename Real>
int launch_gamma_t(const GammaJob& J, cudaStream_t s)
{
    int dev = 0, sms = 0;
    URCHIN_TRY_CUDA(cudaGetDevice(&dev));
    URCHIN_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    constexpr bool kF32 = sizeof(Real) == 4;
    const int64_t rays = J.n_rows * J.R;
    const bool odd = (J.R & 1) && J.R < 16;
    const bool several = kF32 ? J.R > 2 && rays >= (odd ? 6000 : 1700) * (int64_t)sms && J.F <= kRowsMaxBins
                              : rays >= 6000 * (int64_t)sms && J.F < J.R;
    const FoldSplit sp = several ? fold_split(J.n_rows, J.R, 1536 * (int64_t)sms, kF32 ? 2 : 1) : FoldSplit{};
    const void* fn = several ? (const void*)k_gamma_rows<Real> : (const void*)k_gamma<Real>;
    auto bytes = [several](int F, size_t logs) {     // the table and the rays' log rates
        if (several) return FoldTable<Real>::kBytes * (size_t)((F + 1) & ~1) + logs;
        return sizeof(double) * kGammaThreads + (kF32 ? 3 : 2) * (size_t)F * sizeof(Real);
    };
    const size_t smem = bytes(J.F, sp.lk_bytes);
    URCHIN_TRY(allow_shared(fn, smem, bytes(URCHIN_MAX_BINS, kFoldLogs)));
    const int rows = several ? sp.rows : kGammaThreads / J.R;
    const int64_t need = (J.n_rows + rows - 1) / rows;
    int grid = 0;
    URCHIN_TRY(grid_for(fn, kGammaThreads, smem, &grid));
    if (need < grid) grid = (int)std::max<int64_t>(need, 1);
    if (several) k_gamma_rows<Real><<<grid, kFoldThreads, smem, s>>>(J, sp);
    else k_gamma<Real><<<grid, kGammaThreads, smem, s>>>(J);
    URCHIN_TRY(launched());
    return URCHIN_OK;
}

__global__ void k_equilibrium(const double* __restrict__ gamma, const float* __restrict__ tau_eff,
                              const double* __restrict__ nH, const double* __restrict__ T, int64_t n,
                              int case_rule, double y, double* x_out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const bool caseB = case_rule == URCHIN_CASE_B ||
                           (case_rule == URCHIN_CASE_AUTO && tau_eff[i] >= 1.0f);
        const Rates r = hg97_case(T[i], caseB);
        x_out[i] = x_equilibrium(gamma[i], nH[i], r.alphaA, r.gamma_c, y);
    }
}

// the double loop for one ray; ws(b) = w_b s_b, smin the smallest s_b
template <typename Ws>
__device__ __forceinline__ double rate_bar(double c, double t, const double* ss, Ws ws, int F, double smin)
{
    double S = 0.0;
    for (int b = 0; b < F; ++b) S += ws(b) * exp(-(ss[b] - smin) * t);
    return c != 0.0 && S > 0.0 ? -copysign(exp(log(fabs(c)) - smin * t + log(S)), c) : 0.0;
}

// Reverse mode of Eq. gamma_shld, in double.  With c_o = gamma_bar_o / R:
//   tau_bar_ok = -c_o sum_b w_b s_b exp(-s_b tau_ok)
//              = -sign(c_o) exp(ln|c_o| - s_min tau_ok + ln sum_b w_b s_b exp(-(s_b - s_min) tau_ok)),
// written so that a large |c_o| (deeply shielded origins) does not overflow
// where exp(-s_min tau) underflows.
__global__ void k_gamma_vjp_tau(const double* __restrict__ tau, int64_t n_rays, int R, const double* __restrict__ sv,
                                const double* __restrict__ wv, int F, const double* __restrict__ gbar, double* tau_bar)
{
    extern __shared__ double sm[];
    double* ss = sm;
    double* ws = sm + F;
    __shared__ double smin_s;
    for (int b = threadIdx.x; b < F; b += blockDim.x) {
        ss[b] = sv[b];
        ws[b] = wv[b] * sv[b];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = ss[0];
        for (int b = 1; b < F; ++b) m = fmin(m, ss[b]);
        smin_s = m;
    }
    __syncthreads();
    const double smin = smin_s;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n_rays; r += (int64_t)gridDim.x * blockDim.x) {
        const double c = gbar[r / R] / (double)R;
        tau_bar[r] = rate_bar(c, tau[r], ss, [&](int b) { return ws[b]; }, F, smin);
    }
}

// The same for FP32 columns without the double exponential per ray and bin
// (FP64 runs at 1/64 of the FP32 rate here).  With x = (s_b - s_min) log2(e) tau
// held as a float pair p + err (as in the fold), p = k / 64 + r exactly, and
//   2^-x = 2^-(k / 64) (1 + q),  q = 2^-(r + err) - 1,  |q| < 0.006,
// 2^-(k mod 64 / 64) from a table of float pairs (a table-driven exponential
// after Tang, 1989) and q from its series to third order; the weights and the
// products are float pairs and the sum is compensated, so that S is good to
// about 1e-9 and the FP32 result is the rounded one, as with double sums
// (measured against 64 bits over 786432 rays: 2.5e-8 either way).  s_min is
// taken over the bins with a weight.  65536 rows of 12 rays, 200 bins: 5.4 ->
// 0.23 ms.
// The pairs have the range of float, so the double loop stays for spectra whose
// w_b s_b span more than 2^80 (a thermal spectrum's hard bins, which carry all
// of a deeply shielded ray's rate; within 2^80 of the largest, S and every term
// that counts in it are far above the smallest float, and the terms dropped
// beyond 2^-140 are below 2^-60 of S) or lie at the ends of double, and for
// columns outside [0, 1e30).
constexpr int kExpTab = 64;
constexpr double kPairSpan = 0x1p80;

__global__ void __launch_bounds__(256) k_gamma_vjp_tau32(const float* __restrict__ tau, int64_t n_rays, int R,
                                                         const double* __restrict__ sv, const double* __restrict__ wv,
                                                         int F, const double* __restrict__ gbar, float* tau_bar)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4* cf = reinterpret_cast<float4*>(smem_raw);            // [F] exponent coefficient and weight, each a float pair
    double* ss = reinterpret_cast<double*>(smem_raw);            // the double loop: [F] s_b and [F] w_b s_b
    double* ws = ss + F;
    __shared__ float2 tab[kExpTab];
    __shared__ double red[8][4], par[4];
    {
        // smallest s_b, of all bins and of those with a weight; largest and smallest weight
        double ma = INFINITY, m = INFINITY, big = 0.0, lo = INFINITY;
        for (int b = threadIdx.x; b < F; b += blockDim.x) {
            const double q = wv[b] * sv[b];
            ma = fmin(ma, sv[b]);
            big = fmax(big, fabs(q));
            if (q != 0.0) {
                m = fmin(m, sv[b]);
                lo = fmin(lo, fabs(q));
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            ma = fmin(ma, __shfl_xor_sync(0xffffffffu, ma, o));
            m = fmin(m, __shfl_xor_sync(0xffffffffu, m, o));
            big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
            lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        }
        double* r = red[threadIdx.x >> 5];
        if ((threadIdx.x & 31) == 0) {
            r[0] = ma;
            r[1] = m;
            r[2] = big;
            r[3] = lo;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int i = 1; i < 8; ++i) {
                ma = fmin(ma, red[i][0]);
                m = fmin(m, red[i][1]);
                big = fmax(big, red[i][2]);
                lo = fmin(lo, red[i][3]);
            }
            par[0] = ma;
            par[1] = m < INFINITY ? m : 0.0;
            par[2] = big;
            par[3] = lo;
        }
        __syncthreads();
    }
    const double sall = par[0], smin = par[1], scale = par[2];
    if (scale > 0.0 && !(scale < 1e290 && scale > 1e-290 && par[3] * kPairSpan >= scale)) {
        for (int b = threadIdx.x; b < F; b += blockDim.x) {
            ss[b] = sv[b];
            ws[b] = wv[b] * sv[b];
        }
        __syncthreads();
        for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n_rays; r += (int64_t)gridDim.x * blockDim.x)
            tau_bar[r] = (float)rate_bar(gbar[r / R] / (double)R, (double)tau[r], ss, [&](int b) { return ws[b]; }, F, sall);
        return;
    }
    const double iscale = scale > 0.0 ? 1.0 / scale : 0.0;
    for (int b = threadIdx.x; b < F; b += blockDim.x) {
        const double ws = wv[b] * sv[b] * iscale, c = ws != 0.0 ? (sv[b] - smin) * 1.4426950408889634 : 0.0;
        cf[b] = make_float4((float)c, (float)(c - (double)(float)c), (float)ws, (float)(ws - (double)(float)ws));
    }
    for (int i = threadIdx.x; i < kExpTab; i += blockDim.x) {
        const double v = exp2(-(double)i / kExpTab);
        tab[i] = make_float2((float)v, (float)(v - (double)(float)v));
    }
    __syncthreads();
    const double e0 = smin * 1.4426950408889634;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n_rays; r += (int64_t)gridDim.x * blockDim.x) {
        const double c = gbar[r / R] / (double)R;
        const float t = tau[r];
        float out = 0.f;
        if (t >= 0.f && t < 1e30f) {
            float S = 0.f, C = 0.f;
            for (int b = 0; b < F; ++b) {
                const float4 q = cf[b];
                const float p = q.x * t;
                float err = fmaf(q.y, t, fmaf(q.x, t, -p));
                const bool far = p > 140.f;                       // 2^-140 against terms of order one
                const float pc = far ? 0.f : p;
                err = far ? 0.f : err;
                const float kf = fmaf(pc, (float)kExpTab, 12582912.f);   // 1.5 2^23: the sum's low bits are rint(64 p)
                const unsigned k = __float_as_uint(kf) - 0x4b400000u;
                const float z = -0.6931471805599453f * (fmaf(kf - 12582912.f, -1.f / kExpTab, pc) + err);
                const float e = z * fmaf(z, fmaf(z, 0.16666667f, 0.5f), 1.f);
                const float2 T = tab[k & (kExpTab - 1)];
                const float lo = fmaf(T.x, e, T.y);
                const float P = q.z * T.x;
                const float pl = fmaf(q.z, lo, fmaf(q.w, T.x, fmaf(q.z, T.x, -P)));
                // 2^-(k / 64): two halves, so that 2^-140 stays representable in the product
                const unsigned n = far ? 252u : k / kExpTab;
                const float sc = __uint_as_float((127u - n / 2u) << 23) * __uint_as_float((127u - (n - n / 2u)) << 23);
                const float v = P * sc;
                const float u = S + v;
                const float bb = u - S;
                C += (S - (u - bb)) + (v - bb) + pl * sc;
                S = u;
            }
            const double Sd = (double)S + (double)C;
            if (c != 0.0 && Sd > 0.0) {
                // -c exp(-s_min tau) S without leaving the range of double: 2^-(s_min tau log2 e) in two factors
                const double x = e0 * (double)t, n = rint(x), cs = c * scale;
                if (fabs(cs) < 1e290 && fabs(cs) > 1e-290) out = (float)-(n < 4000.0 ? scalbn(cs * Sd * exp2(n - x), -(int)n) : 0.0);
                else out = (float)-copysign(exp(log(fabs(c)) + log(scale) - smin * (double)t + log(Sd)), c);
            }
        } else {
            out = (float)rate_bar(c, (double)t, sv, [&](int b) { return wv[b] * sv[b]; }, F, sall);
        }
        tau_bar[r] = out;
    }
}

// w_bar_b partial sums over rays r with a coefficient c_r = sg_r exp(lc_r):
// partial[block * F + b] = sum over the block's rays of sg_r exp(lc_r - s_b tau_r).
// Rays are staged in tiles; each thread owns a set of bins, so no two
// threads add to the same sum.
constexpr int kWTile = 128;
template <typename Real>
__global__ void k_wbar_tiles(const Real* __restrict__ tau, int64_t n_rays, const double* __restrict__ lc_in,
                             const double* __restrict__ sg_in, const double* __restrict__ sv, int F, double* partial)
{
    extern __shared__ double sm[];
    double* ss = sm;
    double* acc = sm + F;
    double* tt = acc + F;
    double* lc = tt + kWTile;
    double* sg = lc + kWTile;
    for (int b = threadIdx.x; b < F; b += blockDim.x) {
        ss[b] = sv[b];
        acc[b] = 0.0;
    }
    const int64_t tiles = (n_rays + kWTile - 1) / kWTile;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        __syncthreads();
        for (int i = threadIdx.x; i < kWTile; i += blockDim.x) {
            const int64_t r = tile * kWTile + i;
            const bool in = r < n_rays;
            tt[i] = in ? (double)tau[r] : 0.0;
            lc[i] = in ? lc_in[r] : -INFINITY;
            sg[i] = in ? sg_in[r] : 0.0;
        }
        __syncthreads();
        for (int b = threadIdx.x; b < F; b += blockDim.x) {
            const double sb = ss[b];
            double a = acc[b];
            for (int i = 0; i < kWTile; ++i) a += sg[i] * exp(lc[i] - sb * tt[i]);
            acc[b] = a;
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < F; b += blockDim.x) partial[(int64_t)blockIdx.x * F + b] = acc[b];
}

// The FP32 form of k_wbar_tiles: with l_r = lc_r - s_min tau_r and m the
// largest l_r of the tile, every term is sg_r exp(l_r - m) (a float in
// [-1, 1], from one double exp per ray) times exp(-(s_b - s_min) tau_r)
// (the fold's float exponent with its rounding error carried, see
// fold_ray), summed over the tile in float with compensation and added to
// the bin's double sum times exp(m): one double operation per tile and bin
// instead of a double exp per ray and bin.
__global__ void k_wbar_tiles_f32(const float* __restrict__ tau, int64_t n_rays, const double* __restrict__ lc_in,
                                 const double* __restrict__ sg_in, const double* __restrict__ sv, int F,
                                 double* partial)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* acc = reinterpret_cast<double*>(smem_raw);           // [F]
    double* ld = acc + F;                                         // [kWTile]
    float* e2 = reinterpret_cast<float*>(ld + kWTile);            // [F]
    float* e2t = e2 + F;                                          // [F]
    float* tt = e2t + F;                                          // [kWTile]
    float* fr = tt + kWTile;                                      // [kWTile]
    __shared__ double sh_smin, sh_m;
    if (threadIdx.x == 0) {
        double m = sv[0];
        for (int b = 1; b < F; ++b) m = fmin(m, sv[b]);
        sh_smin = m;
    }
    __syncthreads();
    const double smin = sh_smin;
    for (int b = threadIdx.x; b < F; b += blockDim.x) {
        const double c = (sv[b] - smin) * 1.4426950408889634;
        e2[b] = (float)c;
        e2t[b] = (float)(c - (double)(float)c);
        acc[b] = 0.0;
    }
    const int64_t tiles = (n_rays + kWTile - 1) / kWTile;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        __syncthreads();
        for (int i = threadIdx.x; i < kWTile; i += blockDim.x) {
            const int64_t r = tile * kWTile + i;
            const bool in = r < n_rays;
            const float t = in ? tau[r] : 0.f;
            tt[i] = t < 1e30f ? t : (t == t ? 1e30f : t);
            ld[i] = in ? fma(-smin, (double)t, lc_in[r]) : -INFINITY;
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            double m = -INFINITY;
            for (int i = threadIdx.x; i < kWTile; i += 32) m = fmax(m, ld[i]);
            for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (threadIdx.x == 0) sh_m = m;
        }
        __syncthreads();
        const double m = sh_m;
        if (!(m > -INFINITY)) continue;                            // no coefficient in this tile
        for (int i = threadIdx.x; i < kWTile; i += blockDim.x) {
            const int64_t r = tile * kWTile + i;
            fr[i] = (r < n_rays && ld[i] > -INFINITY) ? (float)(sg_in[r] * exp(ld[i] - m)) : 0.f;
        }
        __syncthreads();
        const double em = exp(m);
        for (int b = threadIdx.x; b < F; b += blockDim.x) {
            const float eb = e2[b], ebt = e2t[b];
            float S = 0.f, c = 0.f;
            for (int i = 0; i < kWTile; ++i) {
                const float t = tt[i];
                const float p = eb * t;
                const float err = fmaf(ebt, t, fmaf(eb, t, -p));
                const float v0 = fr[i] * exp2f(-p);
                const float v = fmaf(-v0, err * 0.6931471805599453f, v0);
                const float yy = v - c;
                const float u = S + yy;
                c = (u - S) - yy;
                S = u;
            }
            acc[b] = fma((double)S, em, acc[b]);
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < F; b += blockDim.x) partial[(int64_t)blockIdx.x * F + b] = acc[b];
}

// coefficient of Eq. gamma_shld's reverse mode, the same for the rays of a
// row: c = gamma_bar_o / R.  A block takes `rows` rows (at most its threads) at
// a time: a thread per row for the logarithms, then all of them write (a thread
// that wrote its row's rays took 500 rows of 192 rays from 0.091 to 0.129 ms).
__global__ void __launch_bounds__(256) k_gamma_coef(int64_t n_rows, int R, int rows, const double* __restrict__ gbar,
                                                    double* lc, double* sg)
{
    __shared__ double l[256], g[256];
    for (int64_t o0 = (int64_t)blockIdx.x * rows; o0 < n_rows; o0 += (int64_t)gridDim.x * rows) {
        const int m = (int)(n_rows - o0 < rows ? n_rows - o0 : rows);
        if ((int)threadIdx.x < m) {
            const double c = gbar[o0 + threadIdx.x] / (double)R;
            l[threadIdx.x] = c != 0.0 ? log(fabs(c)) : -INFINITY;
            g[threadIdx.x] = c < 0.0 ? -1.0 : 1.0;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < m * R; i += blockDim.x) {
            const int q = i / R;
            lc[o0 * R + i] = l[q];
            sg[o0 * R + i] = g[q];
        }
        __syncthreads();
    }
}

// out[b] += sum over blocks of partial[block * F + b] (fixed order: 32 strided
// sums, one per lane, added pairwise), a warp per bin
__global__ void k_sum_partials(const double* __restrict__ partial, int nb, int F, double* out)
{
    const int lane = threadIdx.x & 31;
    for (int b = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); b < F; b += (int)((gridDim.x * blockDim.x) >> 5)) {
        double t = 0.0;
        for (int q = lane; q < nb; q += 32) t += partial[(int64_t)q * F + b];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) out[b] += t;
    }
}

// gamma_bar_i = x_bar_i dx_i/dGamma_i (App. C3 root, case as in k_equilibrium)
__global__ void k_equilibrium_vjp(const double* __restrict__ gamma, const float* __restrict__ tau_eff,
                                  const double* __restrict__ nH, const double* __restrict__ T, int64_t n,
                                  int case_rule, double y, const double* __restrict__ x_bar, double* gamma_bar)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const bool caseB = case_rule == URCHIN_CASE_B ||
                           (case_rule == URCHIN_CASE_AUTO && tau_eff[i] >= 1.0f);
        const Rates r = hg97_case(T[i], caseB);
        const double alpha = r.alphaA;
        const double x = x_equilibrium(gamma[i], nH[i], alpha, r.gamma_c, y);
        gamma_bar[i] = x_bar[i] * dx_dgamma(x, nH[i], alpha, r.gamma_c, gamma[i], y);
    }
}

// Near/far rate per origin (Eqs. gammafar, gammashldk, gammashld), in double:
// ln(Gamma_far,k / Gamma_thin) by the factored fold and the slab solution, one
// thread per ray, then a log-sum-exp over the rays: the row's largest by one
// thread, the exponentials by the rays' threads, their sum in order by one
// thread.  Bound by the FP64 pipe (numerical slab in FP32: by its evaluations).
// (One thread per origin for all of it left most of the GPU idle, and one for the
// log-sum-exp, an exponential after the other, made 48 rays slower than that:
// numerical slab, ms, 50021 rows, 12 rays x 100 bins 0.79 -> 0.59, 48 x 20 2.09
// -> 2.57 with it, 1.88 without.)  Up to 4 rays, blocks of 64 threads, so that
// few origins reach more SMs (700 rows of one ray, analytic slab 0.27 -> 0.15 ms;
// one thread per origin 0.16); beyond, blocks of 64 leave more threads without a
// ray (300000 rows, 12 rays 3.39 against 2.55 ms with 256).
constexpr int kNearFarThreads = 256;
constexpr int kNearFarFew = 64;
template <typename Real>
__global__ void __launch_bounds__(kNearFarThreads)
k_gamma_nearfar(const Real* __restrict__ tf, const Real* __restrict__ tn, int64_t n_orig, int R,
                const double* __restrict__ sv, const double* __restrict__ wv, int F, const double* __restrict__ nH,
                const double* __restrict__ T, const uint8_t* __restrict__ caseB, SpecTable poly, double* gamma_out,
                float* tau_eff_out)
{
    extern __shared__ double sm[];
    double* ss = sm;
    double* ws = sm + F;
    __shared__ double sh[2];
    __shared__ double lk[kNearFarThreads], al[kNearFarThreads], gc[kNearFarThreads];
    if (threadIdx.x == 0) {
        double g = 0.0, m = sv[0];
        for (int b = 0; b < F; ++b) {
            g += wv[b];
            m = fmin(m, sv[b]);
        }
        sh[0] = g;
        sh[1] = m;
    }
    __syncthreads();
    const double gthin = sh[0], smin = sh[1];
    for (int b = threadIdx.x; b < F; b += blockDim.x) {
        ss[b] = sv[b] - smin;
        ws[b] = wv[b] / gthin;
    }
    __syncthreads();
    const int rows = (int)blockDim.x / R, local = threadIdx.x / R, k = threadIdx.x - local * R;
    // the ray's share (1/R) of the radiation lights its slab; rates add over rays
    const double lnR = log((double)R);
    for (int64_t row0 = (int64_t)blockIdx.x * rows; row0 < n_orig; row0 += (int64_t)gridDim.x * rows) {
        const int64_t mine = row0 + threadIdx.x;
        if (threadIdx.x < rows && mine < n_orig) {
            const Rates r = hg97_case(T[mine], caseB && caseB[mine]);
            al[threadIdx.x] = r.alphaA;
            gc[threadIdx.x] = r.gamma_c;
        }
        __syncthreads();
        const int64_t o = row0 + local;
        if (local < rows && o < n_orig) {
            const double t = (double)tf[o * R + k], near = (double)tn[o * R + k], n_ = nH[o];
            double l;
            if (poly.tab) {
                // FP32 columns: the slab's table and x_eq in FP32 (see slab_poly_lnratio32)
                l = (sizeof(Real) == 4 ? slab_poly_lnratio32(poly, gthin, t, near, n_, al[local], gc[local], -lnR)
                                       : slab_poly_lnratio(poly, gthin, t, near, n_, al[local], gc[local], -lnR)) +
                    lnR;
            } else {
                double S = 0.0;
                for (int b = 0; b < F; ++b) S += ws[b] * exp(-ss[b] * t);
                l = slab_lnratio(-smin * t + log(S) - lnR, gthin, near, n_, al[local], gc[local]) + lnR;
            }
            lk[local * R + k] = l;
        }
        __syncthreads();
        // (al holds the row's largest from here on)
        if (threadIdx.x < rows && mine < n_orig) {
            double m = -INFINITY;
            for (int q = 0; q < R; ++q) {
                const double l = lk[threadIdx.x * R + q];
                if (l > m) m = l;
            }
            al[threadIdx.x] = m;
        }
        __syncthreads();
        if (local < rows && o < n_orig) {
            const double l = lk[local * R + k];
            lk[local * R + k] = l > -INFINITY ? exp(l - al[local]) : 0.0;
        }
        __syncthreads();
        if (threadIdx.x < rows && mine < n_orig) {
            double acc = 0.0;
            for (int q = 0; q < R; ++q) acc += lk[threadIdx.x * R + q];
            const double lr = al[threadIdx.x] + log(acc / (double)R);
            gamma_out[mine] = gthin * exp(lr);
            if (tau_eff_out) tau_eff_out[mine] = (float)(-lr);
        }
        __syncthreads();
    }
}

// tab[i] = (ln sum_b w_b e^{-s_b tau_i}, d/du), tau_i = e^{u_i} - 1, u_i = i umax / nt,
// in double with the factored sum; smin_out[0] = min_b s_b
__global__ void k_spec_table(const double* __restrict__ sv, const double* __restrict__ wv, int F, int nt,
                             double umax, double2* tab, float2* tab32, double* smin_out)
{
    double smin = sv[0], gthin = 0.0;
    for (int b = 1; b < F; ++b) smin = fmin(smin, sv[b]);
    for (int b = 0; b < F; ++b) gthin += wv[b];
    const double lnthin = log(gthin);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        smin_out[0] = smin;
        smin_out[1] = lnthin;
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= nt; i += gridDim.x * blockDim.x) {
        const double u = umax * (double)i / (double)nt;
        const double tau = expm1(u);
        double S = 0.0, S1 = 0.0;
        for (int b = 0; b < F; ++b) {
            const double e = wv[b] * exp(-(sv[b] - smin) * tau);
            S += e;
            S1 += sv[b] * e;
        }
        // d/du = (d/dtau)(1 + tau), d ln Gamma / d tau = -S1 / S
        tab[i] = make_double2(-smin * tau + log(S), -(S1 / S) * (1.0 + tau));
        tab32[i] = make_float2((float)(-smin * tau + log(S) - lnthin), (float)(-(S1 / S) * (1.0 + tau)));
    }
}

// Rate behind H I, He I and He II columns, one thread per origin in double:
// per ray E_j = s_j tau + s1_j tau1 + s2_j tau2, ln sum_j w^_j exp(-E_j) with
// the smallest E_j factored out, then a log-sum-exp over the rays.
template <typename Real>
__global__ void k_gamma_he(const Real* __restrict__ t0, const Real* __restrict__ t1, const Real* __restrict__ t2,
                           int64_t n_orig, int R, const double* __restrict__ sv, const double* __restrict__ s1v,
                           const double* __restrict__ s2v, const double* __restrict__ wv, int F, double* gamma_out,
                           float* tau_eff_out)
{
    extern __shared__ double sm[];
    double* ss = sm;
    double* s1 = sm + F;
    double* s2 = sm + 2 * F;
    double* ws = sm + 3 * F;
    __shared__ double gsh;
    if (threadIdx.x == 0) {
        double g = 0.0;
        for (int b = 0; b < F; ++b) g += wv[b];
        gsh = g;
    }
    __syncthreads();
    const double gthin = gsh;
    for (int b = threadIdx.x; b < F; b += blockDim.x) {
        ss[b] = sv[b];
        s1[b] = s1v[b];
        s2[b] = s2v[b];
        ws[b] = wv[b] / gthin;
    }
    __syncthreads();
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < n_orig; o += (int64_t)gridDim.x * blockDim.x) {
        double m = -INFINITY, acc = 0.0;
        for (int k = 0; k < R; ++k) {
            const double a = (double)t0[o * R + k], b1 = (double)t1[o * R + k], b2 = (double)t2[o * R + k];
            double emin = INFINITY;
            for (int b = 0; b < F; ++b) emin = fmin(emin, ss[b] * a + s1[b] * b1 + s2[b] * b2);
            double S = 0.0;
            for (int b = 0; b < F; ++b) S += ws[b] * exp(-(ss[b] * a + s1[b] * b1 + s2[b] * b2 - emin));
            const double l = -emin + log(S);
            if (!(l > -INFINITY)) continue;
            if (l > m) {
                acc = acc * exp(m - l) + 1.0;
                m = l;
            } else {
                acc += exp(l - m);
            }
        }
        const double lr = m + log(acc / (double)R);
        gamma_out[o] = gthin * exp(lr);
        if (tau_eff_out) tau_eff_out[o] = (float)(-lr);
    }
}


template <typename Real>
int gamma_vjp_t(const Real* tau, int64_t n_orig, int R, const urchin_spectrum* sp, const double* gbar,
                Real* tau_bar, double* w_bar, cudaStream_t s)
{
    const int64_t n_rays = n_orig * (int64_t)R;
    const int F = sp->F;
    if (tau_bar) {
        constexpr bool kF32 = sizeof(Real) == 4;
        const size_t smem = 16 * (size_t)F;          // two doubles or a float4 per bin
        void (*fn)(const Real*, int64_t, int, const double*, const double*, int, const double*, Real*);
        if constexpr (kF32) fn = k_gamma_vjp_tau32;
        else fn = k_gamma_vjp_tau;
        URCHIN_TRY(allow_shared((const void*)fn, smem, 16 * (size_t)URCHIN_MAX_BINS));
        int grid = 0;
        URCHIN_TRY(grid_for((const void*)fn, 256, smem, &grid));
        grid = (int)std::max<int64_t>(1, std::min<int64_t>(grid, (n_rays + 255) / 256));
        fn<<<grid, 256, smem, s>>>(tau, n_rays, R, sp->s, sp->w, F, gbar, tau_bar);
        URCHIN_TRY(launched());
    }
    if (w_bar) {
        Scratch cf;
        URCHIN_TRY(cf.alloc(2 * sizeof(double) * (size_t)n_rays + 256, s));
        double* lc = cf.at<double>(0);
        double* sg = lc + n_rays;
        // blocks for every SM while the rows last
        const int rows = (int)std::max<int64_t>(1, std::min<int64_t>(256, n_orig / 1024));
        const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n_orig + rows - 1) / rows, 4096));
        k_gamma_coef<<<g, 256, 0, s>>>(n_orig, R, rows, gbar, lc, sg);
        URCHIN_TRY(launched());
        URCHIN_TRY(launch_wbar(tau, sizeof(Real) == 8 ? URCHIN_F64 : URCHIN_F32, n_rays, lc, sg, sp->s, F, w_bar, s));
        cf.release();
    }
    return URCHIN_OK;
}

}  // namespace

size_t spec_table_bytes() { return sizeof(double2) * (kSpecTab + 1) + 64 + sizeof(float2) * (kSpecTab + 1); }

int build_spec_table(const double* s, const double* w, int F, void* buf, SpecTable* out, cudaStream_t st)
{
    double2* tab = static_cast<double2*>(buf);
    double* sc = reinterpret_cast<double*>(tab + kSpecTab + 1);          // smin, ln Gamma_thin
    float2* tab32 = reinterpret_cast<float2*>(reinterpret_cast<char*>(sc) + 64);
    // one warp per block: the nodes spread over the SMs' FP64 pipes
    k_spec_table<<<(kSpecTab + 32) / 32, 32, 0, st>>>(s, w, F, kSpecTab, log1p(kSpecTauMax), tab, tab32, sc);
    URCHIN_TRY(launched());
    double h[2] = {0.0, 0.0};
    URCHIN_TRY_CUDA(cudaMemcpyAsync(h, sc, sizeof(h), cudaMemcpyDeviceToHost, st));
    URCHIN_TRY_CUDA(cudaStreamSynchronize(st));
    *out = SpecTable{tab, kSpecTab, log1p(kSpecTauMax), h[0], tab32, h[1]};
    return URCHIN_OK;
}

int launch_wbar(const void* tau, int precision, int64_t n_rays, const double* lc, const double* sg, const double* sv,
                int F, double* w_bar, cudaStream_t s)
{
    if (n_rays <= 0) return URCHIN_OK;
    const bool f64 = precision == URCHIN_F64;
    auto bytes = [f64](size_t bins) {
        return f64 ? sizeof(double) * (2 * bins + 3 * kWTile)
                   : sizeof(double) * (bins + kWTile) + sizeof(float) * (2 * bins + 2 * kWTile);
    };
    const size_t smem = bytes((size_t)F);
    const void* fn = f64 ? (const void*)k_wbar_tiles<double> : (const void*)k_wbar_tiles_f32;
    URCHIN_TRY(allow_shared(fn, smem, bytes(URCHIN_MAX_BINS)));
    const int64_t tiles = (n_rays + kWTile - 1) / kWTile;
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, 608));
    Scratch part;
    URCHIN_TRY(part.alloc(sizeof(double) * (size_t)nb * F, s));
    if (precision == URCHIN_F64)
        k_wbar_tiles<double><<<nb, 256, smem, s>>>(static_cast<const double*>(tau), n_rays, lc, sg, sv, F,
                                                   part.at<double>(0));
    else
        k_wbar_tiles_f32<<<nb, 256, smem, s>>>(static_cast<const float*>(tau), n_rays, lc, sg, sv, F,
                                               part.at<double>(0));
    URCHIN_TRY(launched());
    k_sum_partials<<<(F + 7) / 8, 256, 0, s>>>(part.at<double>(0), nb, F, w_bar);
    URCHIN_TRY(launched());
    part.release();
    return URCHIN_OK;
}

int launch_gamma(const GammaJob& J, cudaStream_t s)
{
    if (J.n_rows <= 0) return URCHIN_OK;
    if (J.precision == URCHIN_F64) return launch_gamma_t<double>(J, s);
    return launch_gamma_t<float>(J, s);
}

int launch_equilibrium(const double* gamma, const float* tau_eff, const double* nH, const double* T,
                       int64_t n, int case_rule, double y, double* x_out, cudaStream_t s)
{
    if (n <= 0) return URCHIN_OK;
    unsigned grid = (unsigned)std::min<int64_t>((n + 255) / 256, 4096);
    k_equilibrium<<<grid, 256, 0, s>>>(gamma, tau_eff, nH, T, n, case_rule, y, x_out);
    URCHIN_TRY(launched());
    return URCHIN_OK;
}

}  // namespace urchin

extern "C" int urchin_gamma(const void* tau, int precision, int64_t n_orig, int R, const urchin_spectrum* sp,
                            double* gamma_out, float* tau_eff_out, urchin_stream_t stream)
{
    using namespace urchin;
    clear_error();
    if (precision != URCHIN_F32 && precision != URCHIN_F64)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma: unknown precision %d", precision);
    if (R < 1 || R > URCHIN_MAX_RAYS) return set_error(URCHIN_ERR_ARG, "urchin_gamma: R = %d out of range", R);
    if (n_orig < 0) return set_error(URCHIN_ERR_ARG, "urchin_gamma: n_orig < 0");
    if (!sp || !sp->s || !sp->w) return set_error(URCHIN_ERR_ARG, "urchin_gamma: NULL spectrum");
    if (sp->F < 1 || sp->F > URCHIN_MAX_BINS)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma: F = %d out of range [1, %d]", sp->F, URCHIN_MAX_BINS);
    if (spectrum_has_he(sp)) return set_error(URCHIN_ERR_ARG, "urchin_gamma: helium spectrum (use urchin_gamma_he)");
    if (n_orig == 0) return URCHIN_OK;
    if (!tau || !gamma_out) return set_error(URCHIN_ERR_ARG, "urchin_gamma: NULL tau or gamma_out");
    GammaJob J{};
    J.tau = tau;
    J.precision = precision;
    J.n_rows = n_orig;
    J.R = R;
    J.row_stride = R;
    J.k_stride = 1;
    J.s = sp->s;
    J.w = sp->w;
    J.F = sp->F;
    J.gamma_out = gamma_out;
    J.tau_eff_out = tau_eff_out;
    return launch_gamma(J, (cudaStream_t)stream);
}

extern "C" int urchin_equilibrium(const double* gamma, const float* tau_eff, const double* nH, const double* T,
                                  int64_t n, int case_rule, double y, double* x_out, urchin_stream_t stream)
{
    using namespace urchin;
    clear_error();
    if (n < 0) return set_error(URCHIN_ERR_ARG, "urchin_equilibrium: n < 0");
    if (case_rule != URCHIN_CASE_A && case_rule != URCHIN_CASE_B && case_rule != URCHIN_CASE_AUTO)
        return set_error(URCHIN_ERR_ARG, "urchin_equilibrium: unknown case_rule %d", case_rule);
    if (!(y >= 0.0) || !std::isfinite(y)) return set_error(URCHIN_ERR_ARG, "urchin_equilibrium: y must be >= 0");
    if (n == 0) return URCHIN_OK;
    if (!gamma || !nH || !T || !x_out) return set_error(URCHIN_ERR_ARG, "urchin_equilibrium: NULL array");
    if (case_rule == URCHIN_CASE_AUTO && !tau_eff)
        return set_error(URCHIN_ERR_ARG, "urchin_equilibrium: CASE_AUTO needs tau_eff");
    return launch_equilibrium(gamma, tau_eff, nH, T, n, case_rule, y, x_out, (cudaStream_t)stream);
}

extern "C" int urchin_gamma_vjp(const void* tau, int precision, int64_t n_orig, int R, const urchin_spectrum* sp,
                                const double* gamma_bar, void* tau_bar_out, double* w_bar, urchin_stream_t stream)
{
    using namespace urchin;
    clear_error();
    if (precision != URCHIN_F32 && precision != URCHIN_F64)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma_vjp: unknown precision %d", precision);
    if (R < 1 || R > URCHIN_MAX_RAYS) return set_error(URCHIN_ERR_ARG, "urchin_gamma_vjp: R = %d out of range", R);
    if (n_orig < 0) return set_error(URCHIN_ERR_ARG, "urchin_gamma_vjp: n_orig < 0");
    if (!sp || !sp->s || !sp->w) return set_error(URCHIN_ERR_ARG, "urchin_gamma_vjp: NULL spectrum");
    if (sp->F < 1 || sp->F > URCHIN_MAX_BINS)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma_vjp: F = %d out of range [1, %d]", sp->F, URCHIN_MAX_BINS);
    if (spectrum_has_he(sp)) return set_error(URCHIN_ERR_ARG, "urchin_gamma_vjp: no helium columns in reverse mode");
    if (n_orig == 0) return URCHIN_OK;
    if (!tau || !gamma_bar) return set_error(URCHIN_ERR_ARG, "urchin_gamma_vjp: NULL tau or gamma_bar");
    if (!tau_bar_out && !w_bar) return set_error(URCHIN_ERR_ARG, "urchin_gamma_vjp: no output requested");
    cudaStream_t s = (cudaStream_t)stream;
    if (precision == URCHIN_F64)
        return gamma_vjp_t<double>(static_cast<const double*>(tau), n_orig, R, sp, gamma_bar,
                                   static_cast<double*>(tau_bar_out), w_bar, s);
    return gamma_vjp_t<float>(static_cast<const float*>(tau), n_orig, R, sp, gamma_bar,
                              static_cast<float*>(tau_bar_out), w_bar, s);
}

extern "C" int urchin_equilibrium_vjp(const double* gamma, const float* tau_eff, const double* nH, const double* T,
                                      int64_t n, int case_rule, double y, const double* x_bar, double* gamma_bar_out,
                                      urchin_stream_t stream)
{
    using namespace urchin;
    clear_error();
    if (n < 0) return set_error(URCHIN_ERR_ARG, "urchin_equilibrium_vjp: n < 0");
    if (case_rule != URCHIN_CASE_A && case_rule != URCHIN_CASE_B && case_rule != URCHIN_CASE_AUTO)
        return set_error(URCHIN_ERR_ARG, "urchin_equilibrium_vjp: unknown case_rule %d", case_rule);
    if (!(y >= 0.0) || !std::isfinite(y)) return set_error(URCHIN_ERR_ARG, "urchin_equilibrium_vjp: y must be >= 0");
    if (n == 0) return URCHIN_OK;
    if (!gamma || !nH || !T || !x_bar || !gamma_bar_out)
        return set_error(URCHIN_ERR_ARG, "urchin_equilibrium_vjp: NULL array");
    if (case_rule == URCHIN_CASE_AUTO && !tau_eff)
        return set_error(URCHIN_ERR_ARG, "urchin_equilibrium_vjp: CASE_AUTO needs tau_eff");
    cudaStream_t s = (cudaStream_t)stream;
    unsigned grid = (unsigned)std::min<int64_t>((n + 255) / 256, 4096);
    k_equilibrium_vjp<<<grid, 256, 0, s>>>(gamma, tau_eff, nH, T, n, case_rule, y, x_bar, gamma_bar_out);
    return launched();
}

extern "C" int urchin_gamma_nearfar(const void* tau_far, const void* tau_near, int precision, int64_t n_orig, int R,
                                    const urchin_spectrum* sp, const double* nH, const double* T,
                                    const unsigned char* caseB, int slab, double* gamma_out, float* tau_eff_out,
                                    urchin_stream_t stream)
{
    using namespace urchin;
    clear_error();
    if (precision != URCHIN_F32 && precision != URCHIN_F64)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma_nearfar: unknown precision %d", precision);
    if (R < 1 || R > URCHIN_MAX_RAYS) return set_error(URCHIN_ERR_ARG, "urchin_gamma_nearfar: R = %d out of range", R);
    if (n_orig < 0) return set_error(URCHIN_ERR_ARG, "urchin_gamma_nearfar: n_orig < 0");
    if (!sp || !sp->s || !sp->w) return set_error(URCHIN_ERR_ARG, "urchin_gamma_nearfar: NULL spectrum");
    if (sp->F < 1 || sp->F > URCHIN_MAX_BINS)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma_nearfar: F = %d out of range [1, %d]", sp->F, URCHIN_MAX_BINS);
    if (n_orig == 0) return URCHIN_OK;
    if (slab != URCHIN_SLAB_THRESHOLD && slab != URCHIN_SLAB_SPECTRUM)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma_nearfar: unknown slab model %d", slab);
    if (spectrum_has_he(sp)) return set_error(URCHIN_ERR_ARG, "urchin_gamma_nearfar: the slab is hydrogen only");
    if (!tau_far || !tau_near || !nH || !T || !gamma_out)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma_nearfar: NULL tau_far, tau_near, nH, T or gamma_out");
    cudaStream_t s = (cudaStream_t)stream;
    Scratch tb;
    SpecTable poly{nullptr, kSpecTab, log1p(kSpecTauMax), 0.0, nullptr, 0.0};
    if (slab == URCHIN_SLAB_SPECTRUM) {
        URCHIN_TRY(tb.alloc(spec_table_bytes(), s));
        URCHIN_TRY(build_spec_table(sp->s, sp->w, sp->F, tb.at<void>(0), &poly, s));
    }
    const size_t smem = sizeof(double) * 2 * (size_t)sp->F;
    const bool f64 = precision == URCHIN_F64;
    const void* fn = f64 ? (const void*)k_gamma_nearfar<double> : (const void*)k_gamma_nearfar<float>;
    URCHIN_TRY(allow_shared(fn, smem, sizeof(double) * 2 * URCHIN_MAX_BINS));
    const int threads = R <= 4 ? kNearFarFew : kNearFarThreads, rows = threads / R;
    int grid = 0;
    URCHIN_TRY(grid_for(fn, threads, smem, &grid));
    grid = (int)std::max<int64_t>(1, std::min<int64_t>(grid, (n_orig + rows - 1) / rows));
    if (f64)
        k_gamma_nearfar<double><<<grid, threads, smem, s>>>(
            static_cast<const double*>(tau_far), static_cast<const double*>(tau_near), n_orig, R, sp->s, sp->w, sp->F, nH,
            T, caseB, poly, gamma_out, tau_eff_out);
    else
        k_gamma_nearfar<float><<<grid, threads, smem, s>>>(
            static_cast<const float*>(tau_far), static_cast<const float*>(tau_near), n_orig, R, sp->s, sp->w, sp->F, nH, T,
            caseB, poly, gamma_out, tau_eff_out);
    URCHIN_TRY(launched());
    tb.release();
    return URCHIN_OK;
}

extern "C" int urchin_gamma_he(const void* tau, const void* tau_he1, const void* tau_he2, int precision,
                               int64_t n_orig, int R, const urchin_spectrum* sp, double* gamma_out,
                               float* tau_eff_out, urchin_stream_t stream)
{
    using namespace urchin;
    clear_error();
    if (precision != URCHIN_F32 && precision != URCHIN_F64)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma_he: unknown precision %d", precision);
    if (R < 1 || R > URCHIN_MAX_RAYS) return set_error(URCHIN_ERR_ARG, "urchin_gamma_he: R = %d out of range", R);
    if (n_orig < 0) return set_error(URCHIN_ERR_ARG, "urchin_gamma_he: n_orig < 0");
    if (!sp || !sp->s || !sp->w || !sp->s_he1 || !sp->s_he2)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma_he: the spectrum needs s, w, s_he1 and s_he2");
    if (sp->F < 1 || sp->F > URCHIN_MAX_BINS)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma_he: F = %d out of range [1, %d]", sp->F, URCHIN_MAX_BINS);
    if (n_orig == 0) return URCHIN_OK;
    if (!tau || !tau_he1 || !tau_he2 || !gamma_out)
        return set_error(URCHIN_ERR_ARG, "urchin_gamma_he: NULL column or gamma_out");
    cudaStream_t s = (cudaStream_t)stream;
    const size_t smem = sizeof(double) * 4 * (size_t)sp->F;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n_orig + 127) / 128, 4096));
    URCHIN_TRY(allow_shared(precision == URCHIN_F64 ? (const void*)k_gamma_he<double> : (const void*)k_gamma_he<float>,
                            smem, sizeof(double) * 4 * URCHIN_MAX_BINS));
    if (precision == URCHIN_F64) {
        k_gamma_he<double><<<grid, 128, smem, s>>>(static_cast<const double*>(tau), static_cast<const double*>(tau_he1),
                                                   static_cast<const double*>(tau_he2), n_orig, R, sp->s, sp->s_he1,
                                                   sp->s_he2, sp->w, sp->F, gamma_out, tau_eff_out);
    } else {
        k_gamma_he<float><<<grid, 128, smem, s>>>(static_cast<const float*>(tau), static_cast<const float*>(tau_he1),
                                                  static_cast<const float*>(tau_he2), n_orig, R, sp->s, sp->s_he1,
                                                  sp->s_he2, sp->w, sp->F, gamma_out, tau_eff_out);
    }
    return launched();
}

