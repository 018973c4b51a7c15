// scalecv.cu -- Fourier form of the leave-one-out CV for particle-wise widths (Sec. II.B with
// the widths cand[c] kappa_j of the source particles; kde_cv with KDE_CV_SCALE).
//
// With K_kappa(t) = (1/2pi) sum_m A_m(kappa) e^{imt}, S_m = sum_i e^{im theta_i} and
// F_cm = sum_j A_m(cand_c kappa_j) e^{im theta_j}:
//   sum_{i,j} K_{kappa_jc}(theta_i - theta_j) = (1/2pi) (n^2 + 2 sum_{m>=1} Re(conj(S_m) F_cm))
//   int fhat_c^2                              = (1/(2pi n^2)) (n^2 + 2 sum_{m>=1} |F_cm|^2)
//   sum_j K_{kappa_jc}(theta_i - theta_j)     = (1/2pi) (n + 2 sum_{m>=1} Re(e^{im theta_i} conj(F_cm)))
// and the pairs i = j are sum_j norm(cand_c kappa_j).  F needs every particle's own A_m; as a
// function of ln kappa A_m(cand_c kappa) is smooth, so the particles are sorted into bands of
// ln kappa (SC_L wide, SC_Q Chebyshev points, interpolation error below 1e-9) and
//   F_cm = sum_bands sum_q A_m(cand_c kappa_bq) H_bqm,   H_bqm = sum_{j in b} l_q(kappa_j) e^{im theta_j}:
// one pass over the particles for all candidates, 2 SC_Q multiply-adds a (particle, mode),
// with modes only up to the band's own limit (narrow kernels alone have high modes).
//
// What bounds it: FP32 multiply-adds of the band factors and sines of the structure factor,
// N M(kappa) in all, against N^2 exponentials a candidate of the pair sums.  Measured: 50,021
// particles with widths in [5, 5e3], 16 candidates and the leave-one-out densities 8332 us by
// pairs, 353 us here; error of the CV curve 2.2e-7 by pairs, 3e-8 here.
//
// Phases are exact integers and one FP32 sincospi for the first of four consecutive modes;
// sums run in FP32 over 512 particles, then in FP64.
#include "common.cuh"
#include "proxy.cuh"

#define SC_Q 12
#define SC_L 1.2
#define SC_MAXB 16
#define SC_SUB 512        // particles summed in FP32
#define SC_MODES 4        // consecutive modes a thread
#define SC_THREADS 128
#define SC_MAXCHUNKS 256
#define SC_MAXM 8192

struct ScBands {
    int nb, Mst;             // bands; mode stride (largest mode count)
    float l0, inv_l;         // ln of the smallest width; 1 / band length
    float lc[SC_MAXB], inv_lh;  // middle of a band in ln kappa; 1 / its half-length
    int M[SC_MAXB];          // modes a band's kernels have
    int chunk;               // particles of a chunk (a multiple of SC_SUB)
};

// partial extremes of the widths, then one block's reduction to out = (smallest, largest)
__global__ void __launch_bounds__(256) sc_range_kernel(const float *kr, int64_t N, unsigned int *range, unsigned int *status)
{
    float lo = 3.0e38f, hi = 0.f;
    for (int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x; j < N; j += (int64_t)gridDim.x * 256) {
        float k = kr[j];
        if (!(k > 0.f && k <= (float)KDE_KAPPA_MAX)) {
            kde_flag(status, KDE_DEV_KAPPA_RANGE, (unsigned)j);
            k = (float)KDE_KAPPA_MAX;
        }
        lo = fminf(lo, k);
        hi = fmaxf(hi, k);
    }
    kde_krange_add(range, lo, hi);
}

__global__ void __launch_bounds__(256) sc_key_kernel(const float *kr, int64_t N, ScBands B, uint32_t *key)
{
    const int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (j >= N) return;
    const int b = max(0, min(B.nb - 1, (int)((logf(kr[j]) - B.l0) * B.inv_l)));
    key[j] = (uint32_t)b << 28;
}

// first particle of every band in the sorted order (N < 2^32)
__global__ void __launch_bounds__(256) sc_starts_kernel(const uint32_t *key, int64_t N, uint32_t *starts)
{
    const int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (j >= N) return;
    const int b = (int)(key[j] >> 28), a = j ? (int)(key[j - 1] >> 28) : -1;
    for (int k = a + 1; k <= b; ++k) starts[k] = (uint32_t)j;
    if (j == N - 1)
        for (int k = b + 1; k <= SC_MAXB; ++k) starts[k] = (uint32_t)N;
}

// chunks of a band
__device__ __forceinline__ int sc_chunks(const ScBands &B, const uint32_t *starts, int b)
{
    const uint32_t n = starts[b + 1] - starts[b], c = (uint32_t)B.chunk;
    return (int)(n / c + (n % c ? 1u : 0u));
}
// the chunk x of the bands' chunk lists: its band, first particle and number, or false past the end
__device__ __forceinline__ bool sc_chunk(const ScBands &B, const uint32_t *starts, int x, int &b, uint32_t &j0, int &nj)
{
    for (b = 0; b < B.nb; ++b) {
        const int nc = sc_chunks(B, starts, b);
        if (x < nc) {
            j0 = starts[b] + (uint32_t)x * (uint32_t)B.chunk;
            nj = (int)min(starts[b + 1] - j0, (uint32_t)B.chunk);
            return true;
        }
        x -= nc;
    }
    return false;
}

// partial sums of T_q(s_j) e^{im theta_j} over a chunk, q < SC_Q, four consecutive modes a thread
__global__ void __launch_bounds__(SC_THREADS)
    sc_factor_kernel(const uint32_t *__restrict__ u, const float *__restrict__ kr, ScBands B, const uint32_t *starts,
                     double2 *part)
{
    __shared__ uint32_t us[SC_SUB];
    __shared__ __align__(16) float tq[SC_SUB][SC_Q];
    __shared__ float2 e1[SC_SUB];
    int b, nj;
    uint32_t j0;
    if (!sc_chunk(B, starts, blockIdx.x, b, j0, nj)) return;
    u += j0;
    kr += j0;
    const int mb = 1 + blockIdx.y * SC_THREADS * SC_MODES;
    if (mb > B.M[b]) return;
    const int m0 = mb + threadIdx.x * SC_MODES;
    double2 *out = part + (size_t)blockIdx.x * SC_Q * B.Mst + (m0 - 1);
    for (int s0 = 0; s0 < nj; s0 += SC_SUB) {
        const int n = min(SC_SUB, nj - s0);
        __syncthreads();
        for (int k = threadIdx.x; k < n; k += SC_THREADS) {
            const uint32_t uk = u[s0 + k];
            us[k] = uk;
            float sn, cs;
            sincospif((float)(int32_t)uk * (1.0f / 2147483648.0f), &sn, &cs);
            e1[k] = make_float2(cs, sn);
            const float s = (logf(kr[s0 + k]) - B.lc[b]) * B.inv_lh;
            float t0 = 1.f, t1 = s;
#pragma unroll
            for (int q = 0; q < SC_Q; ++q) {
                tq[k][q] = t0;
                const float t2 = fmaf(s + s, t1, -t0);
                t0 = t1;
                t1 = t2;
            }
        }
        __syncthreads();
        if (m0 > B.M[b]) continue;
        float ar[SC_MODES][SC_Q], ai[SC_MODES][SC_Q];
#pragma unroll
        for (int h = 0; h < SC_MODES; ++h)
#pragma unroll
            for (int q = 0; q < SC_Q; ++q) ar[h][q] = ai[h][q] = 0.f;
#pragma unroll 1
        for (int k = 0; k < n; ++k) {
            const uint32_t ph = (uint32_t)m0 * us[k];
            float s, c;
            sincospif((float)(int32_t)ph * (1.0f / 2147483648.0f), &s, &c);
            const float2 e = e1[k];
            float t[SC_Q];
#pragma unroll
            for (int q = 0; q < SC_Q; q += 4) *(float4 *)(t + q) = *(const float4 *)&tq[k][q];
#pragma unroll
            for (int h = 0; h < SC_MODES; ++h) {
#pragma unroll
                for (int q = 0; q < SC_Q; ++q) {
                    ar[h][q] = fmaf(t[q], c, ar[h][q]);
                    ai[h][q] = fmaf(t[q], s, ai[h][q]);
                }
                const float cn = fmaf(c, e.x, -s * e.y), sn = fmaf(s, e.x, c * e.y);
                c = cn;
                s = sn;
            }
        }
#pragma unroll
        for (int h = 0; h < SC_MODES; ++h) {
            if (m0 + h > B.M[b]) break;
#pragma unroll
            for (int q = 0; q < SC_Q; ++q) {
                double2 *o = out + (size_t)q * B.Mst + h;
                double2 v = make_double2((double)ar[h][q], (double)ai[h][q]);
                if (s0 > 0) {
                    const double2 w = *o;
                    v.x += w.x;
                    v.y += w.y;
                }
                *o = v;
            }
        }
    }
}

// G summed over a band's chunks in order, then H_q' = sum_q c_q[q'] G_q (proxy.cuh's matrix in
// FP64); block (32 modes, band), warp w the sums of q = w, w + 8
__global__ void __launch_bounds__(256) sc_reduce_kernel(const double2 *part, ScBands B, const uint32_t *starts, double2 *H)
{
    __shared__ double2 G[SC_Q][32];
    __shared__ double cm[4 * SC_Q];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.y;
    const int m = blockIdx.x * 32 + lane;  // mode m + 1
    if ((int)(blockIdx.x * 32) >= B.M[b]) return;
    if (threadIdx.x < 4 * SC_Q) cm[threadIdx.x] = cospi((double)threadIdx.x / (2.0 * SC_Q));
    int x0 = 0;
    for (int k = 0; k < b; ++k) x0 += sc_chunks(B, starts, k);
    const int nc = sc_chunks(B, starts, b);
    for (int q = warp; q < SC_Q; q += 8) {
        double2 s = make_double2(0.0, 0.0);
        if (m < B.M[b])
            for (int x = 0; x < nc; ++x) {
                const double2 p = part[((size_t)(x0 + x) * SC_Q + q) * B.Mst + m];
                s.x += p.x;
                s.y += p.y;
            }
        G[q][lane] = s;
    }
    __syncthreads();
    for (int a = warp; a < SC_Q; a += 8) {
        double2 s = make_double2(0.0, 0.0);
        for (int q = 0; q < SC_Q; ++q) {
            const double c = (q ? 2.0 : 1.0) / SC_Q * cm[(q * (2 * a + 1)) % (4 * SC_Q)];
            s.x += c * G[q][lane].x;
            s.y += c * G[q][lane].y;
        }
        if (m < B.M[b]) H[((size_t)b * SC_Q + a) * B.Mst + m] = s;
    }
}

// A_m(cand_c kappa_ba) for m = 1 .. M_b by Miller's backward recurrence
// I_{m-1} = (2m / kappa) I_m + I_{m+1}, one multiply-add a step, unnormalised; inv = 1 / I_0.
// One thread a (band, point, candidate); row m of a band: SC_Q n_cand values.
__global__ void __launch_bounds__(32) sc_bessel_kernel(ScBands B, CandList cl, const size_t *aoff, double *A, double *inv)
{
    const int ns = SC_Q * cl.n, i = blockIdx.x * 32 + threadIdx.x, b = blockIdx.y;
    if (i >= ns) return;
    const int a = i / cl.n, c = i - a * cl.n;
    const double kappa = cl.k[c] * exp((double)B.lc[b] + cospi((2.0 * a + 1.0) / (2.0 * SC_Q)) / (double)B.inv_lh);
    // modes beyond the width's own count are below 1e-17: zero
    const int M = min(B.M[b], kappa < 1e-6 ? 3 : kde_spec_modes(kappa));
    const double two_ik = 2.0 / kappa;
    double *row = A + aoff[b] + i;
    for (int m = B.M[b]; m > M; --m) row[(size_t)(m - 1) * ns] = 0.0;
    // small widths converge at once, and their I_0 / I_m would leave the range further up
    int m = M + (kappa < 1.0 ? 2 : 24 + (int)(0.25 * sqrt(kappa)));
    double hi = 0.0, lo = 1e-200;  // I_{m+1}, I_m
    double f = two_ik * (double)m;
    for (; m >= 1; --m) {
        if (m <= M) row[(size_t)(m - 1) * ns] = lo;
        const double t = fma(f, lo, hi);
        f = two_ik * (double)(m - 1);
        hi = lo;
        lo = t;
    }
    inv[(size_t)b * ns + i] = 1.0 / lo;
}

// F_cm over the bands (block: 64 modes of a candidate), and the block's share of
// sum Re(conj(S) F) and sum |F|^2
__global__ void __launch_bounds__(64) sc_combine_kernel(ScBands B, int nc, const size_t *aoff, const double *A,
                                                        const double *inv, const double2 *H, const double2 *S,
                                                        double2 *F, double2 *psum)
{
    __shared__ double2 red[64];
    const int c = blockIdx.y, m = blockIdx.x * 64 + threadIdx.x, ns = SC_Q * nc;
    double2 f = make_double2(0.0, 0.0), s = f;
    if (m < B.Mst) {
        for (int b = 0; b < B.nb; ++b) {
            if (m >= B.M[b]) continue;
            const double *row = A + aoff[b] + (size_t)m * ns + c, *iv = inv + (size_t)b * ns + c;
            const double2 *h = H + (size_t)b * SC_Q * B.Mst + m;
#pragma unroll
            for (int q = 0; q < SC_Q; ++q) {
                const double w = row[q * nc] * iv[q * nc];
                const double2 g = h[(size_t)q * B.Mst];
                f.x = fma(w, g.x, f.x);
                f.y = fma(w, g.y, f.y);
            }
        }
        F[(size_t)c * B.Mst + m] = f;
        const double2 t = S[m];
        s.x = t.x * f.x + t.y * f.y;
        s.y = f.x * f.x + f.y * f.y;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 32; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            red[threadIdx.x].x += red[threadIdx.x + o].x;
            red[threadIdx.x].y += red[threadIdx.x + o].y;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) psum[(size_t)c * gridDim.x + blockIdx.x] = red[0];
}

// sum_j norm(cand_c kappa_j) per block of particles (FP32 tabulated norms, FP64 sums)
__global__ void __launch_bounds__(256) sc_self_kernel(const float *kr, int64_t N, CandList cl, const float2 *ntab, double *pself)
{
    __shared__ double red[8];
    const int c = blockIdx.y;
    double s = 0.0;
    for (int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x; j < N; j += (int64_t)gridDim.x * 256)
        s += (double)kde_norm_tab(ntab, (float)(cl.k[c] * (double)kr[j]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) s += red[w];
        pself[(size_t)c * gridDim.x + blockIdx.x] = s;
    }
}

// CV of every candidate (one thread each) and the argmin, smallest index on ties
__global__ void __launch_bounds__(256) sc_cv_kernel(CandList cl, int64_t N, double L, const double2 *psum, int np,
                                                    const double *pself, int nself, double *cv, int *argmin)
{
    const int c = threadIdx.x;
    const double n = (double)N;
    if (c < cl.n) {
        double sf = 0.0, ff = 0.0, self = 0.0;
        for (int k = 0; k < np; ++k) {
            sf += psum[(size_t)c * np + k].x;
            ff += psum[(size_t)c * np + k].y;
        }
        for (int k = 0; k < nself; ++k) self += pself[(size_t)c * nself + k];
        const double f2 = (n * n + 2.0 * ff) / (KDE_TWO_PI * n * n);
        const double pairs = (n * n + 2.0 * sf) / KDE_TWO_PI - self;
        cv[c] = (KDE_TWO_PI / L) * (f2 - 2.0 * pairs / (n * (n - 1.0)));
    }
    __syncthreads();
    if (c == 0) {
        int best = 0;
        for (int k = 1; k < cl.n; ++k)
            if (cv[k] < cv[best]) best = k;
        *argmin = best;
    }
}

// makes the context's stream wait for its second one, at the latest when it goes out of scope:
// no return, not one on an error, leaves work behind that later calls on the context's stream
// (which reuse the workspace) do not wait for
struct ScJoin {
    kde_ctx *ctx;
    bool done = false;
    void now()
    {
        if (!done) cudaStreamWaitEvent(ctx->stream, ctx->aux_ev[1], 0);
        done = true;
    }
    ~ScJoin() { now(); }
};

kde_status kde_cv_scale_fourier(kde_ctx *ctx, const uint32_t *u, const float *kr, int64_t N, double L,
                                const double *cand_host, int n_cand, double *cv_dev, int *argmin_dev, float *loo,
                                bool *taken)
{
    *taken = false;
    // samples whose pair sums take at most 0.3 ms even with the widest kernels never pay (see
    // below), and spare the host the wait for the range (some 30 us: a server's batch of eight
    // requests of 4000 to 8000 particles took 1.27 ms with it, 1.18 without)
    if (N < 4096 || (double)N * N * n_cand < 1.07e9) return KDE_OK;
    unsigned int *range = (unsigned int *)kde_ws(ctx, WS_WMAX, 64);
    if (!range) return KDE_ENOMEM;
    KDE_CUDA(ctx, kde_krange_reset(range, ctx->stream), "width range memset");
    const int sms = ctx->sm_count > 0 ? ctx->sm_count : 1;
    const int nblk = (int)std::min<int64_t>((N + 255) / 256, 4LL * sms);
    sc_range_kernel<<<nblk, 256, 0, ctx->stream>>>(kr, N, range, ctx->d_status);
    KDE_LAUNCHED(ctx, "sc_range_kernel");
    unsigned int rb[2];
    KDE_CUDA(ctx, cudaMemcpyAsync(rb, range, 8, cudaMemcpyDeviceToHost, ctx->stream), "width range copy");
    KDE_CUDA(ctx, cudaStreamSynchronize(ctx->stream), "width range wait");
    float kmaxf, kminf;
    memcpy(&kmaxf, &rb[0], 4);
    memcpy(&kminf, &rb[1], 4);
    CandList cl{};
    cl.n = n_cand;
    cl.scale_mode = 1;
    double smax = 0.0;
    for (int c = 0; c < n_cand; ++c) {
        cl.k[c] = cand_host[c];
        smax = std::max(smax, cand_host[c]);
    }
    // widths beyond the library's range of one particle's keep the pair sums
    if (!(kminf > 0.f && kmaxf >= kminf) || (double)kmaxf * smax > KDE_KAPPA_MAX) return KDE_OK;
    ScBands B{};
    const double l0 = log((double)kminf), l1 = log((double)kmaxf);
    B.nb = std::max(1, (int)ceil((l1 - l0) / SC_L));
    if (B.nb > SC_MAXB) return KDE_OK;
    const double len = std::max((l1 - l0) / B.nb, 1e-3);
    B.l0 = (float)l0;
    B.inv_l = (float)(1.0 / len);
    B.inv_lh = (float)(2.0 / len);
    double sM = 0.0;
    size_t aoff_h[SC_MAXB], atot = 0;
    for (int b = 0; b < B.nb; ++b) {
        B.lc[b] = (float)(l0 + (b + 0.5) * len);
        // a point of the band may sit a rounding above the largest width
        B.M[b] = kde_spec_modes(exp(l0 + (b + 1) * len + 1e-5) * smax);
        sM += B.M[b];
        aoff_h[b] = atot;
        atot += (size_t)B.M[b] * SC_Q * n_cand;
    }
    B.Mst = B.M[B.nb - 1];
    if (B.Mst > SC_MAXM) return KDE_OK;
    // cost rule, from whole calls: the pair sums take 0.2 ms and 3.5e12 exponentials a second
    // over the smallest width's reach, N^2 a candidate (8192 particles, widths in [5, 5e3], 16
    // candidates 450 us, 16,384 1140 us); here 0.3 ms, 1.4 ps a (particle, mode) and 94 ns a
    // mode for the Bessel rows before they ran beside the rest (470 and 508 us)
    double sfrac = 0.0;
    for (int c = 0; c < n_cand; ++c) {
        const double s2 = KDE_XCUT * KDE_LN2 / (2.0 * cand_host[c] * (double)kminf);
        sfrac += s2 >= 1.0 ? 1.0 : 2.0 * asin(sqrt(s2)) / KDE_PI;
    }
    const double t_pairs = 2e-4 + (double)N * (double)N * sfrac / 3.5e12;
    const double t_four = 3e-4 + (double)N * B.Mst * 1.4e-12 + 5e-8 * B.Mst;
    if (t_four > t_pairs) return KDE_OK;
    // the leave-one-out densities are differences of the whole density and the particle's own
    // kernel: kept to samples where that kernel is below a fifth of the mean density
    if (loo && kde_norm((double)kmaxf * smax) > 0.03 * (double)N) return KDE_OK;

    const int64_t maxc = SC_MAXCHUNKS - B.nb;
    B.chunk = SC_SUB;
    while ((N + B.chunk - 1) / B.chunk > maxc) B.chunk += SC_SUB;
    const int nchunks = (int)((N + B.chunk - 1) / B.chunk) + B.nb;
    const int ns = SC_Q * n_cand, np = (B.Mst + 63) / 64, nself = std::min(nblk, 64);
    // the workspace beyond the pair sums' (a server's share of its budget may be less); slots
    // grow by a quarter more than they are asked for
    const size_t part_b = (size_t)nchunks * SC_Q * B.Mst * sizeof(double2);
    if ((double)(part_b + atot * 8) * 1.25 + 32e6 > (double)ctx->cv_fourier_bytes) return KDE_OK;
    uint32_t *key = (uint32_t *)kde_ws(ctx, WS_CV_KR, (size_t)N * 4);
    uint32_t *keys = (uint32_t *)kde_ws(ctx, WS_SORT_U, (size_t)N * 4);
    uint32_t *us = (uint32_t *)kde_ws(ctx, WS_SORT_P0, (size_t)N * 4);
    float *krs = (float *)kde_ws(ctx, WS_SORT_P1, (size_t)N * 4);
    double2 *part = (double2 *)kde_ws(ctx, WS_CV_PART, part_b);
    double *A = (double *)kde_ws(ctx, WS_CV_LNORM, atot * 8);
    // H, F, the partial sums, the inverse I_0 and the small index tables
    const size_t nH = (size_t)B.nb * SC_Q * B.Mst, nF = (size_t)n_cand * B.Mst, nP = (size_t)n_cand * np;
    unsigned char *w = (unsigned char *)kde_ws(
        ctx, WS_CV_ACC, (nH + nF + nP) * 16 + ((size_t)B.nb * ns + (size_t)n_cand * nself) * 8 + 512);
    if (!key || !keys || !us || !krs || !part || !A || !w) return KDE_ENOMEM;
    double2 *H = (double2 *)w, *F = H + nH, *psum = F + nF;
    double *inv = (double *)(psum + nP), *pself = inv + (size_t)B.nb * ns;
    size_t *aoff = (size_t *)(pself + (size_t)n_cand * nself);
    uint32_t *starts = (uint32_t *)(aoff + SC_MAXB);
    KDE_CUDA(ctx, cudaMemcpyAsync(aoff, aoff_h, sizeof(size_t) * B.nb, cudaMemcpyHostToDevice, ctx->stream), "offsets copy");

    KdeProfScope _ps(ctx, PROF_SPECTRAL);
    // the Bessel rows depend on the widths' range alone and are one long chain of dependent
    // operations on few threads (190 us at 1724 modes): beside the passes over the particles
    KDE_TRY(kde_aux_stream(ctx));
    KDE_CUDA(ctx, cudaEventRecord(ctx->aux_ev[0], ctx->stream), "fork");
    KDE_CUDA(ctx, cudaStreamWaitEvent(ctx->aux, ctx->aux_ev[0], 0), "fork wait");
    sc_bessel_kernel<<<dim3((ns + 31) / 32, B.nb), 32, 0, ctx->aux>>>(B, cl, aoff, A, inv);
    ++ctx->launches;
    const cudaError_t be = cudaGetLastError();
    KDE_CUDA(ctx, cudaEventRecord(ctx->aux_ev[1], ctx->aux), "join");
    ScJoin join{ctx};
    KDE_CUDA(ctx, be, "sc_bessel_kernel");
    const unsigned gN = (unsigned)((N + 255) / 256);
    sc_key_kernel<<<gN, 256, 0, ctx->stream>>>(kr, N, B, key);
    KDE_LAUNCHED(ctx, "sc_key_kernel");
    SortPayload pl[2] = {SortPayload{u, us, 4}, SortPayload{kr, krs, 4}};
    KDE_TRY(kde_sort_by_bin(ctx, key, N, SC_MAXB, keys, pl, 2, nullptr));
    sc_starts_kernel<<<gN, 256, 0, ctx->stream>>>(keys, N, starts);
    KDE_LAUNCHED(ctx, "sc_starts_kernel");
    sc_factor_kernel<<<dim3(nchunks, (B.Mst + SC_THREADS * SC_MODES - 1) / (SC_THREADS * SC_MODES)), SC_THREADS, 0,
                       ctx->stream>>>(us, krs, B, starts, part);
    KDE_LAUNCHED(ctx, "sc_factor_kernel");
    sc_reduce_kernel<<<dim3((B.Mst + 31) / 32, B.nb), 256, 0, ctx->stream>>>(part, B, starts, H);
    KDE_LAUNCHED(ctx, "sc_reduce_kernel");
    sc_self_kernel<<<dim3(nself, n_cand), 256, 0, ctx->stream>>>(kr, N, cl, ctx->norm_tab, pself);
    KDE_LAUNCHED(ctx, "sc_self_kernel");
    double2 *S = nullptr;
    KDE_TRY(kde_spec_structure(ctx, u, N, B.Mst, &S));
    join.now();
    sc_combine_kernel<<<dim3(np, n_cand), 64, 0, ctx->stream>>>(B, n_cand, aoff, A, inv, H, S, F, psum);
    KDE_LAUNCHED(ctx, "sc_combine_kernel");
    sc_cv_kernel<<<1, 256, 0, ctx->stream>>>(cl, N, L, psum, np, pself, nself, cv_dev, argmin_dev);
    KDE_LAUNCHED(ctx, "sc_cv_kernel");
    if (loo) KDE_TRY(kde_loo_series(ctx, u, kr, N, L, F, B.Mst, cl, argmin_dev, (double)kmaxf * smax, loo));
    *taken = true;
    return KDE_OK;
}
