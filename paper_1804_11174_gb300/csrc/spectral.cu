// spectral.cu -- exact Fourier-space evaluation of the leave-one-out CV
// (Sec. II.B, Eq. cv_def) for a uniform width.
//
// The von Mises kernel is K(t) = (1/2pi) sum_m A_m e^{imt}, A_m = I_m/I_0.
// With the structure factor S_m = sum_j e^{i m theta_j}:
//   sum_{i,j} K(theta_i - theta_j) = (1/2pi) (n^2 + 2 sum_{m>=1} A_m |S_m|^2)
//   int fhat^2                     = (1/(2pi n^2)) (n^2 + 2 sum_{m>=1} A_m^2 |S_m|^2)
//   n K(0)                         = n norm(kappa)
//   sum_j K(theta_i - theta_j)     = (1/2pi) (n + 2 sum_{m>=1} A_m Re(e^{i m theta_i} conj(S_m)))
// These are identities; modes are cut where A_m < 1e-17.  The cost is
// O(N M) for S_m (M ~ sqrt(78 kappa_max)) instead of O(N^2) pairs per
// candidate, and all candidates share one S_m; large samples are sorted into
// intervals, whose Chebyshev moments give all S_m at once (spec_moments).
//
// Particle by particle, phases are exact: m theta_j = 2 pi (m u_j mod 2^32) / 2^32 in integer
// arithmetic, then one FP32 sincospi for the first of every SP_Q consecutive
// modes and a rotation by e^{i theta_j} for the next ones (an ulp or two each).
// Sub-chunk sums run in FP32 and are
// combined in FP64 in a fixed order; the CV combination and the leave-one-out
// sums are FP64.  Particles may come in any order (no sort).
#include "common.cuh"
#include "fp64.cuh"
#include "proxy.cuh"

#define SP_THREADS 256
#define SP_SUB 256
#define SP_MAXCHUNK 16384
#define SP_Q 8         // consecutive modes a thread in the structure factor
#define SP_SF_THREADS 128  // threads of a structure-factor block (SP_Q SP_SF_THREADS modes)

// A_m(kappa), m = 0..M, into A[0..M]; r scratch of M + tail + 1 doubles.
// Backward recurrence r_m = 1 / (2m/kappa + r_{m+1}) for r_m = I_m / I_{m-1},
// started at index M + 64 + 2 sqrt(kappa) from the estimate
// kappa / (m + 1/2 + sqrt((m + 1/2)^2 + kappa^2)), then A_m = r_1 ... r_m.
__device__ void spec_ratios(double kappa, int M, double *A)
{
    const int start = M + 64 + (int)(2.0 * sqrt(kappa));
    double r = kappa / (start + 0.5 + sqrt((start + 0.5) * (start + 0.5) + kappa * kappa));
    for (int m = start; m > M; --m) r = 1.0 / (2.0 * m / kappa + r);
    // now r = r_{M+1}; store r_m for m = M..1 in A[m]
    for (int m = M; m >= 1; --m) {
        r = 1.0 / (2.0 * m / kappa + r);
        A[m] = r;
    }
    A[0] = 1.0;
    for (int m = 1; m <= M; ++m) A[m] *= A[m - 1];
}

// structure factor partials: block (chunk, mode block); thread = SP_Q consecutive
// modes m0 .. m0 + SP_Q - 1: one exact-phase sincospi for m0, then each further mode by
// a rotation with e^{i theta_j} (tabulated per particle in shared memory), which costs
// four FP32 operations instead of a sincospi and adds at most an ulp or two per step.
// The partials are laid out with stride M; modes above *mlim (when given) are skipped.
__global__ void __launch_bounds__(SP_SF_THREADS)
    spec_sf_kernel(const uint32_t *__restrict__ u, int64_t N, int64_t chunk, int M, const int *mlim, double2 *part)
{
    extern __shared__ __align__(8) uint32_t us[];
    float2 *e1 = (float2 *)(us + ((chunk + 1) & ~1LL));  // (cos, sin) of theta_j
    const int Me = mlim ? min(M, *mlim) : M;
    const int mb = 1 + (int)blockIdx.y * SP_SF_THREADS * SP_Q;
    if (mb > Me) return;  // the whole mode block is above the limit
    const int64_t j0 = (int64_t)blockIdx.x * chunk;
    const int n = (int)(N - j0 < chunk ? N - j0 : chunk);
    for (int k = threadIdx.x; k < n; k += SP_SF_THREADS) {
        const uint32_t uk = u[j0 + k];
        us[k] = uk;
        float s1, c1;
        sincospif((float)(int32_t)uk * (1.0f / 2147483648.0f), &s1, &c1);
        e1[k] = make_float2(c1, s1);
    }
    __syncthreads();
    const int m0 = mb + threadIdx.x * SP_Q;
    if (m0 > Me) return;
    double cr[SP_Q], ci[SP_Q];
#pragma unroll
    for (int q = 0; q < SP_Q; ++q) cr[q] = ci[q] = 0.0;
    for (int k0 = 0; k0 < n; k0 += SP_SUB) {
        const int k1 = k0 + SP_SUB < n ? k0 + SP_SUB : n;
        float fr[SP_Q], fi[SP_Q];
#pragma unroll
        for (int q = 0; q < SP_Q; ++q) fr[q] = fi[q] = 0.f;
#pragma unroll 2
        for (int k = k0; k < k1; ++k) {
            const uint32_t ph = (uint32_t)m0 * us[k];  // m0 theta / (2 pi) in 2^-32 turns
            float s, c;
            sincospif((float)(int32_t)ph * (1.0f / 2147483648.0f), &s, &c);
            const float2 e = e1[k];
            fr[0] += c;
            fi[0] += s;
#pragma unroll
            for (int q = 1; q < SP_Q; ++q) {
                const float cn = fmaf(c, e.x, -s * e.y), sn = fmaf(s, e.x, c * e.y);
                c = cn;
                s = sn;
                fr[q] += c;
                fi[q] += s;
            }
        }
#pragma unroll
        for (int q = 0; q < SP_Q; ++q) {
            cr[q] += (double)fr[q];
            ci[q] += (double)fi[q];
        }
    }
#pragma unroll
    for (int q = 0; q < SP_Q; ++q)
        if (m0 + q <= Me) part[(size_t)blockIdx.x * M + (m0 + q - 1)] = make_double2(cr[q], ci[q]);
}

// S_m = sum over the chunks (modes up to *mlim when given) in a fixed order, in two
// stages: block (32 modes, chunk group g) -- warp w adds chunks c0 + w, c0 + w + 8, ...
// of the group in order, then the eight warp sums in warp order -- and then the
// SPR_G group sums in group order
#define SPR_G 8
__global__ void __launch_bounds__(256) spec_reduce_kernel(const double2 *part, int nchunks, int M, const int *mlim,
                                                          double2 *gpart)
{
    __shared__ double2 ws[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int Me = mlim ? min(M, *mlim) : M;
    const int m = (int)blockIdx.x * 32 + lane;
    const int c0 = (int)((int64_t)nchunks * blockIdx.y / SPR_G), c1 = (int)((int64_t)nchunks * (blockIdx.y + 1) / SPR_G);
    double sr = 0.0, si = 0.0;
    if (m < Me) {
#pragma unroll 4
        for (int c = c0 + warp; c < c1; c += 8) {
            const double2 p = part[(size_t)c * M + m];
            sr += p.x;
            si += p.y;
        }
    }
    ws[warp][lane] = make_double2(sr, si);
    __syncthreads();
    if (warp == 0 && m < Me) {
        double2 t = ws[0][lane];
#pragma unroll
        for (int w = 1; w < 8; ++w) {
            t.x += ws[w][lane].x;
            t.y += ws[w][lane].y;
        }
        gpart[(size_t)blockIdx.y * M + m] = t;
    }
}

__global__ void spec_reduce2_kernel(const double2 *gpart, int M, const int *mlim, double2 *S)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= (mlim ? min(M, *mlim) : M)) return;
    double2 t = gpart[m];
#pragma unroll
    for (int g = 1; g < SPR_G; ++g) {
        const double2 p = gpart[(size_t)g * M + m];
        t.x += p.x;
        t.y += p.y;
    }
    S[m] = t;
}

// one CTA per candidate (caller's order): Bessel ratios (sequential recurrence,
// one thread; skipped when Atab already holds this candidate list's ratios), then the
// three mode sums over the block and CV (x units)
__global__ void __launch_bounds__(SP_THREADS)
    spec_cv_kernel(const double2 *S, CandList cl, int64_t N, double L, int Astride, double *Atab, int ratios_ready,
                   double *cv_out)
{
    __shared__ double r0[SP_THREADS], r1[SP_THREADS], r2[SP_THREADS];
    const int c = blockIdx.x;
    const double n = (double)N;
    const double kappa = cl.k[c];
    const int M = kde_spec_modes(kappa);
    double *A = Atab + (size_t)c * Astride;
    if (threadIdx.x == 0 && !ratios_ready) spec_ratios(kappa, M, A);
    __syncthreads();
    double sA = 0.0, sAS = 0.0, sA2S = 0.0;
    for (int m = 1 + threadIdx.x; m <= M; m += SP_THREADS) {
        const double2 s = S[m - 1];
        const double p = s.x * s.x + s.y * s.y;
        const double a = A[m];
        sA += a;
        sAS += a * p;
        sA2S += a * a * p;
    }
    r0[threadIdx.x] = sA;
    r1[threadIdx.x] = sAS;
    r2[threadIdx.x] = sA2S;
    __syncthreads();
    for (int o = SP_THREADS / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            r0[threadIdx.x] += r0[threadIdx.x + o];
            r1[threadIdx.x] += r1[threadIdx.x + o];
            r2[threadIdx.x] += r2[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double f2 = (n * n + 2.0 * r2[0]) / (KDE_TWO_PI * n * n);
        const double pairs = (n * n + 2.0 * r1[0] - n - 2.0 * n * r0[0]) / KDE_TWO_PI;
        cv_out[c] = (KDE_TWO_PI / L) * (f2 - 2.0 * pairs / (n * (n - 1.0)));
    }
}

// the density table of the leave-one-out densities (below)
#define LT_P 7
#define LT_IV 4        // intervals of a block, LT_P lanes each
#define LT_GROUPS 8    // warps that share the modes of its points
#define LT_CH 512      // modes staged at a time

__host__ __device__ inline int lt_intervals(double kappa)
{
    const int C = (int)ceil(KDE_PI / 0.2646 * sqrt(kappa + 1.5));
    return C < 4 ? 4 : C;
}

// the selected width kappa* = cand[*argmin]: its mode count, Bessel ratios A[0..M]
// and normalisation 1 / (2 pi I0e(kappa*)), for the leave-one-out pass
struct SpecSel {
    int M;
    int C;         // intervals of the density table (lt_intervals)
    double kappa;  // the width (for particle-wise widths the factor on them)
    double norm;
    const double *A;  // the ratios A[0..M]: a row of the candidates' table, or the kernel's own output
};
// argmin (smallest index on ties) over the first n of cv, by a warp; every lane has it
__device__ __forceinline__ int spec_argmin(const double *cv, int n, int lane)
{
    double v = 1.0e300;
    int at = 0x7fffffff;
    for (int q = lane; q < n; q += 32) {
        const double x = cv[q];
        if (at == 0x7fffffff || x < v) {
            v = x;
            at = q;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double w = __shfl_xor_sync(0xffffffffu, v, o);
        const int k = __shfl_xor_sync(0xffffffffu, at, o);
        if (k != 0x7fffffff && (at == 0x7fffffff || w < v || (w == v && k < at))) {
            v = w;
            at = k;
        }
    }
    return at;
}

// the selected candidate: its index and width, and (sel given) what the leave-one-out pass
// needs of it.  cv: the curve, or nullptr when *argmin is known.  Atab: the candidates' ratio
// table (row stride Astride) when the caller has it, else the ratios are worked out into A
__global__ void __launch_bounds__(32) spec_select_kernel(const double *cv, CandList cl, int *argmin, double *kstar,
                                                         SpecSel *sel, double *A, const double *Atab, int Astride)
{
    const int best = cv ? spec_argmin(cv, cl.n, threadIdx.x) : *argmin;
    if (threadIdx.x != 0) return;
    if (cv) *argmin = best;
    const double kappa = cl.k[best];
    if (kstar) *kstar = kappa;
    if (!sel) return;
    const int M = kde_spec_modes(kappa);
    if (Atab) {
        sel->A = Atab + (size_t)best * Astride;
    } else {
        spec_ratios(kappa, M, A);
        sel->A = A;
    }
    sel->M = M;
    sel->C = lt_intervals(kappa);
    sel->kappa = kappa;
    sel->norm = f64_norm(kappa);
}

// A_m S_m in FP32 for the leave-one-out sums
__global__ void spec_as_kernel(const double2 *S, const SpecSel *sel, float2 *AS)
{
    const int m = 1 + blockIdx.x * blockDim.x + threadIdx.x;
    if (m > sel->M) return;
    const double *A = sel->A;
    const double2 s = S[m - 1];
    AS[m - 1] = make_float2((float)(A[m] * s.x), (float)(A[m] * s.y));
}

// ---------------------------------------------------------------------------
// Leave-one-out densities from a density series sum_j K(theta - theta_j) = (1/2pi)(n + 2 f(theta)),
// f(theta) = sum_{m=1}^{M} Re(e^{i m theta} conj(c_m)).  f is smooth on the scale of the narrowest
// kernel, so it is tabulated: C equal intervals, chosen on the device from the largest width in
// force, with seven Chebyshev points each (proxy.cuh, y <= 0.2646), and every particle reads its
// interval's seven coefficients, the first in FP64 (the density is nearly constant over an
// interval, so the others need FP32 only).  M sines a point instead of M a particle: 2^18
// particles at kappa* = 450 83 -> 12 us.
// ---------------------------------------------------------------------------
// row of an interval's coefficients of f / n
struct __align__(32) LtRow {
    double c0;
    float c[6];
};

// lanes are points, warps take blocks of eight modes in turn: exact integer phases (a sincospi a
// mode: rotations would triple the error of the densities), compensated sums
__global__ void __launch_bounds__(32 * LT_GROUPS)
    spec_table_kernel(const float2 *__restrict__ AS, const SpecSel *__restrict__ sel, const float *__restrict__ cp,
                      double inv_n, LtRow *tab)
{
    __shared__ float2 sAS[LT_CH];
    __shared__ double val[LT_GROUPS][32];
    const int M = sel->M, C = sel->C;
    if (blockIdx.x * LT_IV >= C) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int iv = lane / LT_P, a = lane - iv * LT_P, i = blockIdx.x * LT_IV + iv;
    // the point: interval middle and Chebyshev point, to a code (2^-33 of the circle)
    const float x = cp[LT_P + a] * (0.5f * (float)LT_P);
    const double pos = ((double)i + 0.5 + 0.5 * (double)x) * (4294967296.0 / (double)C);
    const uint32_t code = (uint32_t)(unsigned long long)__double2ll_rn(pos);
    float acc = 0.f, comp = 0.f;
    for (int m0 = 1; m0 <= M; m0 += LT_CH) {
        const int cnt = min(LT_CH, M - m0 + 1);
        __syncthreads();
        for (int k = threadIdx.x; k < LT_CH; k += 32 * LT_GROUPS)
            sAS[k] = k < cnt ? AS[m0 - 1 + k] : make_float2(0.f, 0.f);
        __syncthreads();
        for (int k = warp * 8; k < cnt; k += LT_GROUPS * 8) {
#pragma unroll
            for (int h = 0; h < 8; ++h) {
                const uint32_t ph = (uint32_t)(m0 + k + h) * code;
                float s, c;
                sincospif((float)(int32_t)ph * (1.0f / 2147483648.0f), &s, &c);
                const float2 q = sAS[k + h];
                // Re(e^{i m theta} conj(c_m)) = cos * Re + sin * Im
                const float y = fmaf(c, q.x, s * q.y) - comp;
                const float t = acc + y;
                comp = (t - acc) - y;
                acc = t;
            }
        }
    }
    val[warp][lane] = (double)acc - (double)comp;
    __syncthreads();
    if (warp == 0) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < LT_GROUPS; ++w) v += val[w][lane];
        val[0][lane] = v * inv_n;
        __syncwarp();
        if (iv < LT_IV && i < C) {
            const double *f = &val[0][iv * LT_P];
            if (a == 0) {
                double t = 0.0;
                for (int q = 0; q < LT_P; ++q) t += f[q];
                tab[i].c0 = t * (1.0 / LT_P);
            } else {
                // the points' differences from the first: the sum of a row of the matrix is 0
                float t = 0.f;
                for (int q = 1; q < LT_P; ++q) t = fmaf(cp[a * LT_P + q], (float)(f[q] - f[0]), t);
                tab[i].c[a - 1] = t;
            }
        }
    }
}

// loo_i = (2 pi / L) (sum_j K - own kernel) / (n - 1) from the table; own kernel: sel->norm, or
// norm(sel->kappa kr_i) for particle-wise widths
// (fa = xs n / (2 pi (n - 1)), fb = xs / (n - 1))
__global__ void __launch_bounds__(SP_THREADS)
    spec_loo_kernel(const uint32_t *__restrict__ u, const float *__restrict__ kr, int64_t N,
                    const LtRow *__restrict__ tab, const SpecSel *__restrict__ sel, double fa, double fb,
                    const float2 *__restrict__ ntab, float *loo)
{
    const int C = sel->C;
    const double base = kr ? fa : fma(-fb, sel->norm, fa), fa2 = 2.0 * fa;
    const float kap = (float)sel->kappa;
    for (int64_t i = (int64_t)blockIdx.x * SP_THREADS + threadIdx.x; i < N; i += (int64_t)gridDim.x * SP_THREADS) {
        const uint32_t ui = u[i];
        const float x = (float)(int32_t)((ui * (uint32_t)C) ^ 0x80000000u) * (1.f / 2147483648.f);
        const uint4 *r = (const uint4 *)(tab + __umulhi(ui, (uint32_t)C));
        const uint4 a = __ldg(r), b = __ldg(r + 1);
        const float x2 = x + x;
        float b1 = __uint_as_float(b.w), b2 = 0.f, t;
#define LT_STEP(w) t = fmaf(x2, b1, __uint_as_float(w) - b2); b2 = b1; b1 = t
        LT_STEP(b.z);
        LT_STEP(b.y);
        LT_STEP(b.x);
        LT_STEP(a.w);
        LT_STEP(a.z);
#undef LT_STEP
        const double g = __hiloint2double((int)a.y, (int)a.x) + (double)fmaf(x, b1, -b2);
        double v = fma(fa2, g, base);
        if (kr) v = fma(-fb, (double)kde_norm_tab(ntab, kap * kr[i]), v);
        loo[i] = (float)v;
    }
}

// table and densities from the series coefficients AS (modes 1..sel->M) of a sample whose
// widths are at most kappa_max
static kde_status spec_loo_table(kde_ctx *ctx, const uint32_t *u, const float *kr, int64_t N, double L,
                                 const float2 *AS, const SpecSel *sel, double kappa_max, float *loo)
{
    const int C = lt_intervals(kappa_max);
    LtRow *tab = (LtRow *)kde_ws(ctx, WS_LTAB, (size_t)C * sizeof(LtRow));
    if (!tab) return KDE_ENOMEM;
    KdeProfScope _ps(ctx, PROF_CV_LOO);
    spec_table_kernel<<<(C + LT_IV - 1) / LT_IV, 32 * LT_GROUPS, 0, ctx->stream>>>(
        AS, sel, ctx->pxy_tab + pxy_tab_off(LT_P), 1.0 / (double)N, tab);
    KDE_LAUNCHED(ctx, "spec_table_kernel");
    const int64_t want = (N + SP_THREADS - 1) / SP_THREADS, cap = 8LL * (ctx->sm_count > 0 ? ctx->sm_count : 1);
    spec_loo_kernel<<<(unsigned)(want < cap ? want : cap), SP_THREADS, 0, ctx->stream>>>(
        u, kr, N, tab, sel, (double)N / (L * (double)(N - 1)), KDE_TWO_PI / (L * (double)(N - 1)), ctx->norm_tab, loo);
    KDE_LAUNCHED(ctx, "spec_loo_kernel");
    return KDE_OK;
}

// the selected candidate's row of F in FP32, and its limits, for particle-wise widths
__global__ void __launch_bounds__(256) spec_as_scale_kernel(const double2 *F, int Mst, CandList cl, const int *argmin,
                                                            double kr_max, float2 *AS, SpecSel *sel)
{
    const int c = *argmin, m = blockIdx.x * 256 + threadIdx.x;
    if (m < Mst) {
        const double2 f = F[(size_t)c * Mst + m];
        AS[m] = make_float2((float)f.x, (float)f.y);
    }
    if (m == 0) {
        const double k = cl.k[c] * kr_max;
        sel->M = min(Mst, kde_spec_modes(k));
        sel->C = lt_intervals(k);
        sel->kappa = cl.k[c];
        sel->norm = 0.0;
    }
}

kde_status kde_loo_series(kde_ctx *ctx, const uint32_t *u, const float *kr, int64_t N, double L, const double2 *F,
                          int Mst, const CandList &cl, const int *argmin_dev, double kappa_max, float *loo)
{
    double smax = 0.0;
    for (int c = 0; c < cl.n; ++c) smax = cl.k[c] > smax ? cl.k[c] : smax;
    float2 *AS = (float2 *)kde_ws(ctx, WS_SP_AS, (size_t)Mst * sizeof(float2) + 64);
    SpecSel *sel = (SpecSel *)kde_ws(ctx, WS_SP_SEL, sizeof(SpecSel));
    if (!AS || !sel) return KDE_ENOMEM;
    spec_as_scale_kernel<<<(Mst + 255) / 256, 256, 0, ctx->stream>>>(F, Mst, cl, argmin_dev, kappa_max / smax, AS, sel);
    KDE_LAUNCHED(ctx, "spec_as_scale_kernel");
    return spec_loo_table(ctx, u, kr, N, L, AS, sel, kappa_max, loo);
}

// leave-one-out densities at cand[*argmin] from the structure factor S (modes 1..M(kappa*)
// present); with cv_dev the argmin (and *kstar_dev) of that curve is found on the way
static kde_status spec_loo_from_S(kde_ctx *ctx, const uint32_t *u, int64_t N, double L, const double2 *S,
                                  const CandList &cl, int Mmax, int *argmin_dev, float *loo,
                                  const double *cv_dev = nullptr, double *kstar_dev = nullptr,
                                  const double *Atab = nullptr, int Astride = 0)
{
    double *Asel = (double *)kde_ws(ctx, WS_SP_ASEL, (size_t)(Mmax + 1) * 8 + 64);
    float2 *AS = (float2 *)kde_ws(ctx, WS_SP_AS, (size_t)Mmax * sizeof(float2) + 64);
    SpecSel *sel = (SpecSel *)kde_ws(ctx, WS_SP_SEL, sizeof(SpecSel));
    if (!Asel || !AS || !sel) return KDE_ENOMEM;
    spec_select_kernel<<<1, 32, 0, ctx->stream>>>(cv_dev, cl, argmin_dev, kstar_dev, sel, Asel, Atab, Astride);
    KDE_LAUNCHED(ctx, "spec_select_kernel");
    spec_as_kernel<<<(Mmax + 255) / 256, 256, 0, ctx->stream>>>(S, sel, AS);
    KDE_LAUNCHED(ctx, "spec_as_kernel");
    double kmax = 0.0;
    for (int c = 0; c < cl.n; ++c) kmax = cl.k[c] > kmax ? cl.k[c] : kmax;
    return spec_loo_table(ctx, u, nullptr, N, L, AS, sel, kmax, loo);
}

// ---------------------------------------------------------------------------
// Structure factor of a large sample from moments.  Over an interval of half-width a = pi / C the
// phase e^{i m theta} is its Chebyshev interpolant with SM_P points to 2 (m a / 2)^P / P!, below
// 1e-10 for m a <= 3.08.  So the particles, sorted into C intervals, leave SM_P Chebyshev moments
// an interval; SM_P discrete Fourier transforms over the intervals take those to every mode at
// once, and a mode is the sum of its SM_P values with the interpolant's coefficients:
//   S_m = e^{i m a} sum_k c_k(m) sum_b M_{b,k} e^{2 pi i m b / C}.
// Bound by launches and the sort.  2^20 particles and 893 modes took 348 us particle by particle,
// 2^18 took 91: a CV call over 64 candidates and 2^18 particles went from 182 to 130 us, a 50-step
// PIC period with one at 2^20 from 2292 to 2018 us.  Moments are summed as integers (FP32 values of at most 2^13 with steps
// of 2^-30, so the sum is exact and in no order), and from there on all is FP64: the intervals'
// phases and coefficients are few, and their rounding would not average out.
// ---------------------------------------------------------------------------
#define SM_P 16
#define SM_THREADS 128
#define SM_MAXRANGE 8192
#define SM_LGC_MAX 13
#define SM_LGC_MIN 8
#define SM_SPLIT 8  // blocks a transform: the modes m = r mod SM_SPLIT

// blocks below R: moments of `range` sorted particles, interval by interval; the rest: the table
// E[j] = e^{i pi j / C}, j < 2 C
__global__ void __launch_bounds__(SM_THREADS)
    spec_moments_kernel(const uint32_t *__restrict__ us, int64_t N, int range, int R, int lgC, unsigned long long *mom,
                        double2 *E)
{
    extern __shared__ uint32_t u[];
    __shared__ float part[SM_THREADS / 32][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, shift = 32 - lgC;
    if ((int)blockIdx.x >= R) {
        const int j = ((int)blockIdx.x - R) * SM_THREADS + tid;
        if (j < 2 << lgC) {
            double sn, cs;
            sincospi(ldexp((double)j, -lgC), &sn, &cs);
            E[j] = make_double2(cs, sn);
        }
        return;
    }
    const int64_t i0 = (int64_t)blockIdx.x * range;
    const int n = (int)(N - i0 < range ? N - i0 : range);
    for (int k = tid; k < n; k += SM_THREADS) u[k] = us[i0 + k];
    __syncthreads();
    for (int s = 0; s < n;) {
        const uint32_t bin = u[s] >> shift;
        int lo = s, hi = n;  // the interval's end: first particle of a later one
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (u[mid] >> shift == bin) lo = mid;
            else hi = mid;
        }
        float v[32];
#pragma unroll
        for (int p = 0; p < 32; ++p) v[p] = 0.f;
        for (int k = s + tid; k < hi; k += SM_THREADS) {
            const float x = (float)(int32_t)((u[k] << lgC) ^ 0x80000000u) * (1.f / 2147483648.f), x2 = x + x;
            float t0 = 1.f, t1 = x;
#pragma unroll
            for (int p = 0; p < SM_P; ++p) {
                v[p] += t0;
                const float t2 = fmaf(x2, t1, -t0);
                t0 = t1;
                t1 = t2;
            }
        }
        part[warp][lane] = warp_transpose_sum32(v, lane);
        __syncthreads();
        if (tid < SM_P) {
            float m = 0.f;
#pragma unroll
            for (int w = 0; w < SM_THREADS / 32; ++w) m += part[w][tid];
            atomicAdd(mom + ((size_t)tid << lgC) + bin, (unsigned long long)__double2ll_rn((double)m * 1073741824.0));
        }
        __syncthreads();
        s = hi;
    }
}

// modes m = r mod SM_SPLIT of the transform of moment k (k = blockIdx.y, r = blockIdx.x): one
// step of decimation in frequency takes the C intervals to L = C / SM_SPLIT, then radix 2
__global__ void __launch_bounds__(SM_THREADS)
    spec_fft_kernel(const long long *__restrict__ mom, const double2 *__restrict__ E, int lgC, double2 *F)
{
    extern __shared__ double2 buf[];  // two of L
    const int C = 1 << lgC, L = C / SM_SPLIT, mask = 2 * C - 1, r = blockIdx.x, tid = threadIdx.x;
    const long long *x = mom + ((size_t)blockIdx.y << lgC);
    double2 w[SM_SPLIT];  // e^{2 pi i r j / SM_SPLIT}
#pragma unroll
    for (int j = 0; j < SM_SPLIT; ++j) w[j] = E[(r * j * (2 * C / SM_SPLIT)) & mask];
    for (int n = tid; n < L; n += SM_THREADS) {
        double yr = 0.0, yi = 0.0;
#pragma unroll
        for (int j = 0; j < SM_SPLIT; ++j) {
            const double v = (double)x[n + j * L];
            yr = fma(v, w[j].x, yr);
            yi = fma(v, w[j].y, yi);
        }
        const double2 e = E[(2 * r * n) & mask];
        buf[n] = make_double2((yr * e.x - yi * e.y) * 0x1p-30, (yr * e.y + yi * e.x) * 0x1p-30);
    }
    __syncthreads();
    double2 *a = buf, *b = buf + L;
    for (int h = L / 2, s = 1, ls = 0; h >= 1; h >>= 1, s <<= 1, ++ls) {
        for (int t = tid; t < L / 2; t += SM_THREADS) {
            const int q = t & (s - 1), p = t >> ls;
            const double2 c = a[q + s * p], d = a[q + s * (p + h)], e = E[(p * SM_SPLIT * 2) << ls];
            const double2 g = make_double2(c.x - d.x, c.y - d.y);
            b[q + s * 2 * p] = make_double2(c.x + d.x, c.y + d.y);
            b[q + s * (2 * p + 1)] = make_double2(g.x * e.x - g.y * e.y, g.x * e.y + g.y * e.x);
        }
        __syncthreads();
        double2 *o = a;
        a = b;
        b = o;
    }
    for (int q = tid; q < L; q += SM_THREADS) F[((size_t)blockIdx.y << lgC) + SM_SPLIT * q + r] = a[q];
}

// a mode from its SM_P values, eight lanes a mode: lane p has the points +-x_p, which share the
// cosine (even moments) and the sine (odd ones); modes above *mlim (when given) are skipped
__global__ void __launch_bounds__(SM_THREADS)
    spec_modes_kernel(const double2 *__restrict__ F, const double2 *__restrict__ E, int lgC, int M, const int *mlim, double2 *S)
{
    __shared__ double ct[4 * SM_P];  // cos(pi j / (2 SM_P))
    if (threadIdx.x < 4 * SM_P) ct[threadIdx.x] = cospi((double)threadIdx.x / (2 * SM_P));
    __syncthreads();
    const int Me = mlim ? min(M, *mlim) : M;
    const int m = 1 + (int)(blockIdx.x * SM_THREADS + threadIdx.x) / (SM_P / 2), p = threadIdx.x & (SM_P / 2 - 1);
    const int mc = m <= Me ? m : 0;
    double er = 0.5 * F[mc].x, ei = 0.5 * F[mc].y, odr = 0.0, odi = 0.0;
#pragma unroll
    for (int k = 1; k < SM_P; ++k) {
        const double t = ct[(k * (2 * p + 1)) & (4 * SM_P - 1)];
        const double2 f = F[((size_t)k << lgC) + mc];
        if (k & 1) {
            odr = fma(t, f.x, odr);
            odi = fma(t, f.y, odi);
        } else {
            er = fma(t, f.x, er);
            ei = fma(t, f.y, ei);
        }
    }
    double sn, cs;
    sincospi(ldexp((double)mc * ct[2 * p + 1], -lgC), &sn, &cs);
    double gr = fma(cs, er, -sn * odi), gi = fma(cs, ei, sn * odr);
#pragma unroll
    for (int o = SM_P / 4; o; o >>= 1) {
        gr += __shfl_xor_sync(0xffffffffu, gr, o);
        gi += __shfl_xor_sync(0xffffffffu, gi, o);
    }
    if (p == 0 && m <= Me) {
        const double2 e = E[m];
        const double f = 4.0 / SM_P;  // both points of a pair, and the 2 of the coefficients
        S[m - 1] = make_double2(f * (gr * e.x - gi * e.y), f * (gr * e.y + gi * e.x));
    }
}

// the structure factor so, where it pays; *taken is false where the particles go one by one
static kde_status spec_moments(kde_ctx *ctx, const uint32_t *u, int64_t N, int M, const int *mlim, double2 *S, bool *taken)
{
    *taken = false;
    int lgC = SM_LGC_MIN;
    while (lgC < SM_LGC_MAX && (double)(1 << lgC) * 3.08 < KDE_PI * (double)M) ++lgC;
    const int C = 1 << lgC;
    if ((double)C * 3.08 < KDE_PI * (double)M) return KDE_OK;
    int64_t range = (N + 511) / 512;
    range = range < 512 ? 512 : (range > SM_MAXRANGE ? SM_MAXRANGE : range);
    const int64_t R = (N + range - 1) / range;
    // The sort, the transforms and the tables grow with the intervals, the particles one by one
    // with N M.  CV calls of 16 candidates, so against one by one: 2^20 particles and 62 modes
    // 112 against 184 us, 400,003 and 153 94 against 122, 150,000 and 279 90 against 97, 65,536
    // and 883 100 against 99, 32,768 and 1530 128 against 97.
    if ((double)N * M < 1e7 + 6e4 * C || N < 16 * (int64_t)C || R > 1 << 20) return KDE_OK;
    uint32_t *us = (uint32_t *)kde_ws(ctx, WS_SORT_U, (size_t)N * 4);
    const size_t momb = (size_t)SM_P * 8 << SM_LGC_MAX, tabb = (size_t)sizeof(double2) * 2 << SM_LGC_MAX;
    char *ws = (char *)kde_ws(ctx, WS_SP_PX, 3 * momb + tabb);
    if (!us || !ws) return KDE_OK;  // no room for them: one by one
    unsigned long long *mom = (unsigned long long *)ws;
    double2 *F = (double2 *)(ws + momb), *E = (double2 *)(ws + 3 * momb);
    KDE_TRY(kde_sort_by_bin(ctx, u, N, C, us, nullptr, 0, nullptr));
    KDE_CUDA(ctx, cudaMemsetAsync(mom, 0, (size_t)SM_P * C * 8, ctx->stream), "moments memset");
    KdeProfScope _ps(ctx, PROF_SPECTRAL);
    spec_moments_kernel<<<(unsigned)(R + 2 * C / SM_THREADS), SM_THREADS, (size_t)range * 4, ctx->stream>>>(
        us, N, (int)range, (int)R, lgC, mom, E);
    KDE_LAUNCHED(ctx, "spec_moments_kernel");
    spec_fft_kernel<<<dim3(SM_SPLIT, SM_P), SM_THREADS, (size_t)2 * (C / SM_SPLIT) * sizeof(double2), ctx->stream>>>(
        (const long long *)mom, E, lgC, F);
    KDE_LAUNCHED(ctx, "spec_fft_kernel");
    spec_modes_kernel<<<(unsigned)((M * (SM_P / 2) + SM_THREADS - 1) / SM_THREADS), SM_THREADS, 0, ctx->stream>>>(
        F, E, lgC, M, mlim, S);
    KDE_LAUNCHED(ctx, "spec_modes_kernel");
    *taken = true;
    return KDE_OK;
}

// structure factor for modes 1..M (or up to *mlim) into S
static kde_status spec_structure(kde_ctx *ctx, const uint32_t *u, int64_t N, int M, const int *mlim, double2 **S_out)
{
    // about a thousand chunks keep every SM busy (2^18 particles and 893 modes: 124 us in 256
    // chunks of 1024, 91 in 1024 of 256; 50,021 and 1724 modes: 101 and 45 us); the partials stay
    // under 2^22 entries (64 MB)
    int64_t chunk = 256;
    while (((N + chunk - 1) / chunk > 1024 || (N + chunk - 1) / chunk * M > (1 << 22)) && chunk < SP_MAXCHUNK)
        chunk *= 2;
    double2 *S = (double2 *)kde_ws(ctx, WS_SP_S, (size_t)M * sizeof(double2));
    if (!S) return KDE_ENOMEM;
    *S_out = S;
    bool taken = false;
    KDE_TRY(spec_moments(ctx, u, N, M, mlim, S, &taken));
    if (taken) return KDE_OK;
    const int nchunks = (int)((N + chunk - 1) / chunk);
    double2 *part = (double2 *)kde_ws(ctx, WS_SP_PART, (size_t)(nchunks + SPR_G) * M * sizeof(double2));
    double2 *gpart = part + (size_t)nchunks * M;  // the chunk groups' sums
    if (!part) return KDE_ENOMEM;
    static bool attr = false;
    if (!attr) {
        KDE_CUDA(ctx, cudaFuncSetAttribute(spec_sf_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           SP_MAXCHUNK * 12 + 8),
                 "spec_sf_kernel attribute");
        attr = true;
    }
    {
        KdeProfScope _ps(ctx, PROF_SPECTRAL);
        dim3 grid((unsigned)nchunks, (unsigned)((M + SP_SF_THREADS * SP_Q - 1) / (SP_SF_THREADS * SP_Q)));
        spec_sf_kernel<<<grid, SP_SF_THREADS, (size_t)((chunk + 1) & ~1LL) * 4 + (size_t)chunk * 8, ctx->stream>>>(
            u, N, chunk, M, mlim, part);
    }
    KDE_LAUNCHED(ctx, "spec_sf_kernel");
    spec_reduce_kernel<<<dim3((unsigned)((M + 31) / 32), SPR_G), 256, 0, ctx->stream>>>(part, nchunks, M, mlim, gpart);
    KDE_LAUNCHED(ctx, "spec_reduce_kernel");
    spec_reduce2_kernel<<<(M + 255) / 256, 256, 0, ctx->stream>>>(gpart, M, mlim, S);
    KDE_LAUNCHED(ctx, "spec_reduce2_kernel");
    return KDE_OK;
}

kde_status kde_spec_structure(kde_ctx *ctx, const uint32_t *u, int64_t N, int M, double2 **S_out)
{
    return spec_structure(ctx, u, N, M, nullptr, S_out);
}

// selected width's mode count, for the structure factor of the leave-one-out pass
__global__ void spec_mlim_kernel(CandList cl, const int *argmin, int *mlim) { *mlim = kde_spec_modes(cl.k[*argmin]); }

kde_status kde_loo_spectral_device(kde_ctx *ctx, const uint32_t *u, int64_t N, double L, const double *cand_host,
                                   int n_cand, const int *argmin_dev, float *loo)
{
    CandList cl{};
    cl.n = n_cand;
    double kmax = 0.0;
    for (int c = 0; c < n_cand; ++c) {
        cl.k[c] = cand_host[c];
        kmax = cand_host[c] > kmax ? cand_host[c] : kmax;
    }
    const int Mmax = kde_spec_modes(kmax);
    int *mlim = (int *)kde_ws(ctx, WS_SP_MLIM, 64);
    if (!mlim) return KDE_ENOMEM;
    spec_mlim_kernel<<<1, 1, 0, ctx->stream>>>(cl, argmin_dev, mlim);
    KDE_LAUNCHED(ctx, "spec_mlim_kernel");
    double2 *S = nullptr;
    KDE_TRY(spec_structure(ctx, u, N, Mmax, mlim, &S));
    return spec_loo_from_S(ctx, u, N, L, S, cl, Mmax, const_cast<int *>(argmin_dev), loo);
}

kde_status kde_cv_spectral_device(kde_ctx *ctx, const uint32_t *u, int64_t N, double L, const double *cand_host,
                                  int n_cand, double *cv_dev, int *argmin_dev, float *loo, double *kstar_dev)
{
    CandList cl{};
    cl.n = n_cand;
    cl.scale_mode = 0;
    double kmax = 0.0;
    for (int c = 0; c < n_cand; ++c) {
        cl.k[c] = cand_host[c];
        kmax = cand_host[c] > kmax ? cand_host[c] : kmax;
    }
    const int M = kde_spec_modes(kmax);
    const int Astride = M + 1;
    double *Atab = (double *)kde_ws(ctx, WS_SP_A, (size_t)n_cand * Astride * 8 + 64 * 1024 * 8);
    if (!Atab) return KDE_ENOMEM;
    double2 *S = nullptr;
    KDE_TRY(spec_structure(ctx, u, N, M, nullptr, &S));
    // the Bessel ratios depend on the candidates only: a width schedule that repeats its
    // candidate list reuses the table the previous call left in the workspace
    std::vector<double> key(cand_host, cand_host + n_cand);
    const bool ready = ctx->sp_atab == (void *)Atab && ctx->sp_atab_cands == key;
    spec_cv_kernel<<<n_cand, SP_THREADS, 0, ctx->stream>>>(S, cl, N, L, Astride, Atab, ready ? 1 : 0, cv_dev);
    ctx->sp_atab = (void *)Atab;
    ctx->sp_atab_cands = key;
    KDE_LAUNCHED(ctx, "spec_cv_kernel");
    if (loo) return spec_loo_from_S(ctx, u, N, L, S, cl, M, argmin_dev, loo, cv_dev, kstar_dev, Atab, Astride);
    spec_select_kernel<<<1, 32, 0, ctx->stream>>>(cv_dev, cl, argmin_dev, kstar_dev, nullptr, nullptr, nullptr, 0);
    KDE_LAUNCHED(ctx, "spec_select_kernel");
    return KDE_OK;
}
