// gtable.cu -- FP32 gather of particles in any order from tables of the smoothed field.
//
// For one width the gathered field E(theta) = sum_g (2 pi / Ng) K_kappa(theta_g - theta) E_g is
// a smooth function of the position, so it is tabulated: the circle is cut into C equal
// intervals, each with the coefficients of its Chebyshev interpolant (proxy.cuh: the field at
// the interval's Chebyshev points, from the nodes).  For particle-wise widths E(theta, kappa)
// is tabulated in both: bands of half an octave of kappa (the widths below 1/2 are one band,
// mapped linearly), each with its own C, so that narrow kernels get short intervals.  A
// particle reads its interval's coefficients and evaluates the polynomial: no sort, no
// permutation, and a cost that does not depend on its window.
//
// What bounds it: the particles' pass reads 4 to 8 bytes, writes 4, and fetches 32 (one width)
// or 128 bytes of coefficients from the L1 / L2 caches; the table costs about 40 Ng (node,
// interval) pairs a band.  Only the bands that hold widths are built (a pass over the widths
// finds their range).  Measured, whole calls: 1,000,003 particles, 1024 nodes, widths in
// [5, 5e3] 215 -> 61 us (sorted sweep before: 50 us of it the sort, 174 the sweep; now range 5,
// bands 26, particles 30); 5000 particles, 256 nodes, one width 21.5 -> 11.8 us.
#include "common.cuh"
#include "proxy.cuh"

#define GT_THREADS 256
#define GT_WARPS 8
#define GT_BANDS 35       // half-octave bands from 1/2 up to GT_KMAX, and the linear one below
#define GT_KMAX 65536.f   // wider kappas sweep their window (at most 30 nodes of a 4096-node grid)
#define GT_P1 8           // one width: degree in position (y <= 0.388)
#define GT_P 7            // bands: coefficients p + q < 7 (28, padded to 32)
#define GT_NC 32
#define GT_KR_BLOCKS 304

struct GtBands {
    int C[GT_BANDS];           // intervals
    int off[GT_BANDS];         // first interval of the band in the table
    uint32_t step[GT_BANDS];   // floor(2^32 / 2C)
    int W[GT_BANDS];           // nodes on either side of a cell that the band's kernels reach
};

struct GtArgs {
    const uint32_t *u;
    const float *kappa;
    float kappa_u, norm_u, coef;
    int64_t N;
    const float *field;
    PxyGrid grid;
    const float *pxt;
    const float2 *ntab;
    float *tab;
    const float2 *kr;  // partial ranges of the widths (smallest, largest)
    int nkr;
    float *out;
    unsigned int *status;
};

// widths of band b at s in [-1, 1]
__device__ __forceinline__ float gt_band_kappa(int b, float s)
{
    if (b == 0) return 0.25f + 0.25f * s;
    return 0.5f * exp2f(0.5f * ((float)(b - 1) + 0.5f * (1.f + s)));
}
// band and s of a width
__device__ __forceinline__ int gt_band(float k, float &s)
{
    if (k <= 0.5f) {
        s = fmaf(4.f, k, -1.f);
        return 0;
    }
    const float t = fmaf(2.f, log2f(k), 2.f);  // half octaves above 1/2
    // the last band ends at GT_KMAX, where t (rounded, from 65535.94 on) is a whole number already
    const float f = fminf(floorf(t), (float)(GT_BANDS - 2));
    s = fmaf(2.f, t - f, -1.f);
    return 1 + (int)f;
}
__device__ __forceinline__ float gt_checked(const GtArgs &A, float k, int64_t j)
{
    if (!(k > 0.f && k <= (float)KDE_KAPPA_MAX)) {
        kde_flag(A.status, KDE_DEV_KAPPA_RANGE, (unsigned)j);
        k = (float)KDE_KAPPA_MAX;
    }
    return k;
}
__device__ __forceinline__ int gt_window(float kappa, int Ng)
{
    const float s2 = (float)(KDE_XCUT * KDE_LN2 / 2.0) / kappa;
    if (s2 >= 1.0f) return Ng;
    const float r = 2.0f * asinf(sqrtf(s2));
    const int w = (int)ceilf(r * (float)Ng * (float)(1.0 / KDE_TWO_PI)) + 1;
    return w >= Ng ? Ng : w;
}

// smallest and largest width of every block's share of the particles
__global__ void __launch_bounds__(GT_THREADS) gt_range_kernel(GtArgs A, float2 *kr)
{
    __shared__ float2 red[GT_WARPS];
    float lo = 3.0e38f, hi = 0.f;
    const int64_t step = (int64_t)gridDim.x * GT_THREADS;
    for (int64_t j0 = (int64_t)blockIdx.x * GT_THREADS + threadIdx.x; j0 < A.N; j0 += 4 * step) {
        float k[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) k[q] = j0 + q * step < A.N ? A.kappa[j0 + q * step] : -1.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (j0 + q * step >= A.N) continue;
            const float c = gt_checked(A, k[q], j0 + q * step);
            lo = fminf(lo, c);
            hi = fmaxf(hi, c);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float2(lo, hi);
    __syncthreads();
    kde_pdl_trigger();
    if (threadIdx.x == 0) {
        for (int w = 1; w < GT_WARPS; ++w) {
            lo = fminf(lo, red[w].x);
            hi = fmaxf(hi, red[w].y);
        }
        kr[blockIdx.x] = make_float2(lo, hi);
    }
}

// coefficients of one interval from the field at its proxies, f[a QM + b], by a warp
template <int PM, int QM>
__device__ __forceinline__ void gt_coefs(float *f, const float *nk, const float *cp, const float *cq, float *row)
{
    constexpr int PQ = PM * QM;
    const int lane = threadIdx.x & 31;
    constexpr int PL = (PQ + 31) / 32;
    // U[p][b] = sum_a c_p[a] f[a][b], in place
    float U[PL];
#pragma unroll
    for (int h = 0; h < PL; ++h) {
        const int m = h * 32 + lane, p = m / QM, b = m - p * QM;
        U[h] = 0.f;
        if (m < PQ) {
#pragma unroll
            for (int a = 0; a < PM; ++a) U[h] = fmaf(cp[p * PM + a], f[a * QM + b], U[h]);
            U[h] *= nk[b];
        }
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < PL; ++h)
        if (h * 32 + lane < PQ) f[h * 32 + lane] = U[h];
    __syncwarp();
    constexpr int NC = QM == 1 ? PM : GT_NC;
    if (lane < NC) {
        float t = 0.f;
        if (QM == 1) {
            t = f[lane];
        } else {
            int p = 0, q = lane;  // coefficient `lane` of the triangle p + q < PM
            while (p < PM && q >= PM - p) q -= PM - p++;
            if (p < PM) {
#pragma unroll
                for (int b = 0; b < QM; ++b) t = fmaf(cq[q * QM + b], f[p * QM + b], t);
            }
        }
        row[lane] = t;
    }
    __syncwarp();
}

// nodes of interval i: the first of R
__device__ __forceinline__ int gt_nodes(int Ng, int C, int i, int W, int &R)
{
    const int c0 = (int)((uint32_t)i * (uint32_t)Ng / (uint32_t)C);
    const int c1 = (int)(((uint32_t)(i + 1) * (uint32_t)Ng - 1u) / (uint32_t)C);
    R = c1 + W - (c0 - W) + 1;
    if (R < Ng) return c0 - W;
    R = Ng;
    return 0;
}

// coefficients of one interval i < C by a group of wpi warps (warp w of the group): the
// field at the PM x QM proxies, every lane a node with all the proxies' values in registers
// (PM sines and PM QM exponentials that do not depend on one another), summed over the lanes
// by butterflies, then the interpolation matrices.  Every warp of the CTA calls it together,
// those without an interval with on = false.  scd: sine and cosine of half the proxies' angles
// from the interval's middle, (pi / 2) x_a / C; part: PM QM floats a warp
template <int PM, int QM>
__device__ __forceinline__ void gt_interval(const GtArgs &A, bool on, int C, uint32_t step, int i, int w, int wpi, int W,
                                            const float *k2, const float *nk, const float *cp, const float *cq,
                                            const float2 *scd, float *part, float *tab)
{
    constexpr int PQ = PM * QM, NR = (PQ + 31) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, Ng = A.grid.Ng;
    if (on) {
        // the interval's middle as a code and a fraction (node 2i + 1 of a grid of 2C)
        PxyGrid G2;
        G2.Ng = 2 * C;
        G2.step = step;
        G2.rem = 0u - step * (uint32_t)(2 * C);  // 2^32 - step 2C
        uint32_t mid;
        float mfrac;
        pxy_node(G2, 2 * i + 1, mid, mfrac);
        int R;
        const int g_lo = gt_nodes(Ng, C, i, W, R);
        float acc[NR * 32], kk[QM];
#pragma unroll
        for (int m = 0; m < NR * 32; ++m) acc[m] = 0.f;
#pragma unroll
        for (int b = 0; b < QM; ++b) kk[b] = k2[b];
#pragma unroll 1
        for (int r = w * 32 + lane; r < R; r += 32 * wpi) {
            int g = g_lo + r;
            g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
            const float e = A.field[g];
            uint32_t nc;
            float nf, sn, cn;
            pxy_node(A.grid, g, nc, nf);
            pxy_sincos(nc, nf, mid, mfrac, sn, cn);
#pragma unroll
            for (int a = 0; a < PM; ++a) {
                // half the angle to the proxy from that to the middle: with y <= 0.39 the proxies
                // are a small part of the kernel's width from it, so the difference keeps 1e-8 of
                // that width
                const float2 d = scd[a];
                const float sa = fmaf(sn, d.y, -cn * d.x), s2 = sa * sa;
#pragma unroll
                for (int b = 0; b < QM; ++b) acc[a * QM + b] = fmaf(kde_ex2(s2 * kk[b]), e, acc[a * QM + b]);
            }
        }
#pragma unroll
        for (int h = 0; h < NR; ++h) {
            float v[32];
#pragma unroll
            for (int m = 0; m < 32; ++m) v[m] = acc[h * 32 + m];
            const float t = warp_transpose_sum32(v, lane);
            if (h * 32 + lane < PQ) part[warp * PQ + h * 32 + lane] = t;
        }
    }
    if (wpi > 1) {
        // the group's warps' sums, by its first warp
        __syncthreads();
        if (on && w == 0)
            for (int m = lane; m < PQ; m += 32) {
                float t = part[warp * PQ + m];
                for (int q = 1; q < wpi; ++q) t += part[(warp + q) * PQ + m];
                part[warp * PQ + m] = t;
            }
    }
    __syncwarp();
    if (on && w == 0) gt_coefs<PM, QM>(part + warp * PQ, nk, cp, cq, tab + (size_t)i * (QM == 1 ? PM : GT_NC));
    if (wpi > 1) __syncthreads();
}

// the same for a window of at most 32 nodes, a warp an interval: a lane holds a node, the proxies'
// values are the lanes' own sums over the nodes.  200,003 particles on 256 nodes, whole calls, before
// with the window's nodes over the lanes and butterflies over 49 values: widths of 2000 to 20,000
// (13,000 intervals) 42 -> 35 us, of 5 to 5000 45 -> 39
#define GT_SHORT 32
template <int PM, int QM>
__device__ __forceinline__ void gt_interval_short(const GtArgs &A, int C, uint32_t step, int i, int W, const float *k2,
                                                  const float *nk, const float *cp, const float *cq, const float2 *scd,
                                                  float *part, float *tab)
{
    constexpr int PQ = PM * QM, H = (PQ + 31) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, Ng = A.grid.Ng;
    PxyGrid G2;
    G2.Ng = 2 * C;
    G2.step = step;
    G2.rem = 0u - step * (uint32_t)(2 * C);
    uint32_t mid, nc;
    float mfrac, nf, sn, cn;
    pxy_node(G2, 2 * i + 1, mid, mfrac);
    int R;
    int g = gt_nodes(Ng, C, i, W, R) + (lane < GT_SHORT ? lane : 0);
    g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
    g = lane < R ? g : 0;
    const float e = lane < R ? A.field[g] : 0.f;
    pxy_node(A.grid, g, nc, nf);
    pxy_sincos(nc, nf, mid, mfrac, sn, cn);
    float2 d[H];
    float kk[H], f[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int m = min(h * 32 + lane, PQ - 1);
        d[h] = scd[m / QM];
        kk[h] = k2[m % QM];
        f[h] = 0.f;
    }
#pragma unroll 4
    for (int r = 0; r < R; ++r) {
        const float s = __shfl_sync(0xffffffffu, sn, r), c = __shfl_sync(0xffffffffu, cn, r);
        const float er = __shfl_sync(0xffffffffu, e, r);
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const float sa = fmaf(s, d[h].y, -c * d[h].x);
            f[h] = fmaf(kde_ex2(sa * sa * kk[h]), er, f[h]);
        }
    }
#pragma unroll
    for (int h = 0; h < H; ++h)
        if (h * 32 + lane < PQ) part[warp * PQ + h * 32 + lane] = f[h];
    __syncwarp();
    gt_coefs<PM, QM>(part + warp * PQ, nk, cp, cq, tab + (size_t)i * (QM == 1 ? PM : GT_NC));
}

// warps that share an interval's window: about eight nodes a lane and more
__device__ __forceinline__ int gt_wpi(int W, int Ng, int C)
{
    const int R = min(Ng, 2 * W + Ng / C + 2);
    return R <= 256 ? 1 : (R <= 512 ? 2 : (R <= 1024 ? 4 : 8));
}

__global__ void __launch_bounds__(GT_THREADS) gt_table_one_kernel(GtArgs A, int C, uint32_t step)
{
    __shared__ float part[GT_WARPS * GT_P1], cp[GT_P1 * GT_P1], k2[1], nk[1], one[1];
    __shared__ float2 scd[GT_P1];
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid < GT_P1 * GT_P1) cp[tid] = A.pxt[pxy_tab_off(GT_P1) + tid];
    if (tid < GT_P1) {
        const float x = A.pxt[pxy_tab_off(GT_P1) + GT_P1 + tid] * (0.5f * (float)GT_P1);
        sincospif(x * (0.5f / (float)C), &scd[tid].x, &scd[tid].y);
    }
    if (tid == 0) {
        k2[0] = (float)(-2.0 * KDE_LOG2E) * A.kappa_u;
        nk[0] = A.coef * A.norm_u;
        one[0] = 1.f;
    }
    const int W = gt_window(A.kappa_u, A.grid.Ng), wpi = gt_wpi(W, A.grid.Ng, C), ipc = GT_WARPS / wpi;
    __syncthreads();
    kde_pdl_trigger();
    for (int i0 = blockIdx.x * ipc; i0 < C; i0 += gridDim.x * ipc) {
        const int i = i0 + warp / wpi;
        gt_interval<GT_P1, 1>(A, i < C, C, step, i, warp % wpi, wpi, W, k2, nk, cp, one, scd, part, A.tab);
    }
}

__global__ void __launch_bounds__(GT_THREADS, 2) gt_table_bands_kernel(GtArgs A, GtBands T)
{
    constexpr int PM = GT_P;
    __shared__ float part[GT_WARPS * PM * PM], cp[PM * PM], xc[PM], k2s[GT_WARPS][PM], nks[GT_WARPS][PM];
    __shared__ float2 scds[GT_WARPS][PM];
    __shared__ float2 red[GT_WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < PM * PM) cp[tid] = A.pxt[pxy_tab_off(PM) + tid];
    if (tid < PM) xc[tid] = A.pxt[pxy_tab_off(PM) + PM + tid] * (0.5f * (float)PM);
    kde_pdl_wait();
    kde_pdl_trigger();
    float lo = 3.0e38f, hi = 0.f;
    for (int i = tid; i < A.nkr; i += GT_THREADS) {
        const float2 k = A.kr[i];
        lo = fminf(lo, k.x);
        hi = fmaxf(hi, k.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) red[warp] = make_float2(lo, hi);
    __syncthreads();
#pragma unroll
    for (int w = 0; w < GT_WARPS; ++w) {
        lo = fminf(lo, red[w].x);
        hi = fmaxf(hi, red[w].y);
    }
    float s;
    const int b0 = gt_band(lo, s), b1 = gt_band(fminf(hi, GT_KMAX), s);
    float *k2 = k2s[warp], *nk = nks[warp];
    float2 *scd = scds[warp];
    int turn = (int)blockIdx.x;  // items of all bands are dealt to the CTAs in turn
    for (int b = b0; b <= b1; ++b) {
        const int C = T.C[b];
        const int W = T.W[b], wpi = gt_wpi(W, A.grid.Ng, C);
        const int ipc = GT_WARPS / wpi, items = (C + ipc - 1) / ipc;
        if (turn < items) {
            __syncwarp();
            if (lane < PM) {  // every warp its own copy
                const float k = gt_band_kappa(b, xc[lane]);
                k2[lane] = (float)(-2.0 * KDE_LOG2E) * k;
                nk[lane] = A.coef * kde_norm_tab(A.ntab, k);
                sincospif(xc[lane] * (0.5f / (float)C), &scd[lane].x, &scd[lane].y);
            }
            __syncwarp();
            const bool narrow = 2 * W + A.grid.Ng / C + 2 <= GT_SHORT;  // wpi is 1 then
            for (; turn < items; turn += (int)gridDim.x) {
                const int i = turn * ipc + warp / wpi;
                if (narrow) {
                    if (i < C)
                        gt_interval_short<PM, PM>(A, C, T.step[b], i, W, k2, nk, cp, cp, scd, part,
                                                  A.tab + (size_t)T.off[b] * GT_NC);
                    continue;
                }
                gt_interval<PM, PM>(A, i < C, C, T.step[b], i, warp % wpi, wpi, W, k2, nk, cp, cp, scd, part,
                                    A.tab + (size_t)T.off[b] * GT_NC);
            }
        }
        turn -= items;
    }
}

// interval and place in it: u C / 2^32 = i + (x + 1) / 2
__device__ __forceinline__ int gt_place(uint32_t u, int C, float &x)
{
    x = (float)(int32_t)((u * (uint32_t)C) ^ 0x80000000u) * (1.f / 2147483648.f);
    return (int)__umulhi(u, (uint32_t)C);
}

__global__ void __launch_bounds__(GT_THREADS) gt_eval_one_kernel(GtArgs A, int C)
{
    constexpr int NP = 4;
    const int64_t j0 = (int64_t)blockIdx.x * GT_THREADS * NP + threadIdx.x;
    uint32_t u[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) u[h] = j0 + h * GT_THREADS < A.N ? A.u[j0 + h * GT_THREADS] : 0u;
    kde_pdl_wait();  // the table
    kde_pdl_trigger();
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        float x;
        const float4 *c = (const float4 *)A.tab + 2 * gt_place(u[h], C, x);
        const float4 a = __ldg(c), b = __ldg(c + 1);
        // Clenshaw's recurrence
        const float x2 = x + x;
        float b1 = b.w, b2 = 0.f, t;
#define GT_STEP(cf) t = fmaf(x2, b1, (cf) - b2); b2 = b1; b1 = t
        GT_STEP(b.z);
        GT_STEP(b.y);
        GT_STEP(b.x);
        GT_STEP(a.w);
        GT_STEP(a.z);
        GT_STEP(a.y);
#undef GT_STEP
        const int64_t j = j0 + h * GT_THREADS;
        if (j < A.N) A.out[j] = fmaf(x, b1, a.x - b2);
    }
}

__global__ void __launch_bounds__(GT_THREADS) gt_eval_bands_kernel(GtArgs A, GtBands T)
{
    constexpr int NP = 2;
    __shared__ int2 sb[GT_BANDS];
    if (threadIdx.x < GT_BANDS) sb[threadIdx.x] = make_int2(T.C[threadIdx.x], T.off[threadIdx.x]);
    const int64_t j0 = (int64_t)blockIdx.x * GT_THREADS * NP + threadIdx.x;
    uint32_t u[NP];
    float k[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        const int64_t j = j0 + h * GT_THREADS;
        u[h] = j < A.N ? A.u[j] : 0u;
        k[h] = j < A.N ? A.kappa[j] : 0.f;
    }
    __syncthreads();
    kde_pdl_wait();  // the table
    kde_pdl_trigger();
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        const int64_t j = j0 + h * GT_THREADS;
        if (j >= A.N) break;
        // widths outside the range were reported by the range pass
        const float kap = (k[h] > 0.f && k[h] <= (float)KDE_KAPPA_MAX) ? k[h] : (float)KDE_KAPPA_MAX;
        float e = 0.f;
        if (kap <= GT_KMAX) {
            float s, x;
            const int b = gt_band(kap, s);
            const int i = gt_place(u[h], sb[b].x, x);
            const float4 *c4 = (const float4 *)A.tab + (size_t)(sb[b].y + i) * (GT_NC / 4);
            float c[28];
#pragma unroll
            for (int m = 0; m < 7; ++m) {
                const float4 v = __ldg(c4 + m);
                c[4 * m] = v.x;
                c[4 * m + 1] = v.y;
                c[4 * m + 2] = v.z;
                c[4 * m + 3] = v.w;
            }
            float tq[GT_P];
            tq[0] = 1.f;
            tq[1] = s;
#pragma unroll
            for (int q = 2; q < GT_P; ++q) tq[q] = fmaf(s + s, tq[q - 1], -tq[q - 2]);
            float t0 = 1.f, t1 = x;
            int m = 0;
#pragma unroll
            for (int p = 0; p < GT_P; ++p) {
                float row = c[m++];
#pragma unroll
                for (int q = 1; q < GT_P - p; ++q) row = fmaf(c[m++], tq[q], row);
                if (p == 0) {
                    e = row;
                } else {
                    e = fmaf(row, t1, e);
                    const float t2 = fmaf(x + x, t1, -t0);
                    t0 = t1;
                    t1 = t2;
                }
            }
        } else {
            // a kernel far narrower than any band: its own few nodes
            const int Ng = A.grid.Ng, W = gt_window(kap, Ng), c0 = kde_cell(u[h], Ng);
            const int len = min(Ng, 2 * W + 1);
            const float k2 = (float)(-2.0 * KDE_LOG2E) * kap;
            int g = c0 - W;
            g = len == Ng ? 0 : (g < 0 ? g + Ng : g);
            for (int r = 0; r < len; ++r) {
                uint32_t nc;
                float nf;
                pxy_node(A.grid, g, nc, nf);
                e = fmaf(kde_ex2(k2 * pxy_sin2(nc, nf, u[h], 0.f)), A.field[g], e);
                g = g + 1 == Ng ? 0 : g + 1;
            }
            e *= A.coef * kde_norm_tab(A.ntab, kap);
        }
        A.out[j] = e;
    }
}

// small calls: GT_FLAT lanes a particle sweep the particle's own window, node by node.  A warp takes
// NB rounds of four particles, and what a particle needs first (norm, window, place) is worked
// out by 32 / (4 NB) lanes, not by all of its eight: more rounds where that leaves the SMs their warps
// (200,003 particles, widths of 5 to 5000, 64 nodes 30 -> 25 us)
#define GT_FLAT 8
template <int NB> __global__ void __launch_bounds__(GT_THREADS) gt_flat_kernel(GtArgs A)
{
    constexpr int PW = 32 / GT_FLAT * NB;  // particles a warp
    const int lane = threadIdx.x & 31, sub = lane & (GT_FLAT - 1), Ng = A.grid.Ng;
    const int64_t j0 = ((int64_t)blockIdx.x * GT_WARPS + (threadIdx.x >> 5)) * PW;
    if (j0 >= A.N) return;  // the whole warp
    const int64_t j = j0 + (lane & (PW - 1)), jj = j < A.N ? j : A.N - 1;
    const uint32_t u = A.u[jj];
    float k = A.kappa_u, nm = A.norm_u;
    if (A.kappa) {
        k = gt_checked(A, A.kappa[jj], jj);
        nm = kde_norm_tab(A.ntab, k);
    }
    const int W = gt_window(k, Ng), len = min(Ng, 2 * W + 1);
    const float k2 = (float)(-2.0 * KDE_LOG2E) * k;
    const int g0 = len == Ng ? 0 : kde_cell(u, Ng) - W;
    // the node's code and fraction move on by GT_FLAT nodes at a time (round the circle the
    // codes wrap by themselves)
    const uint32_t dn = GT_FLAT * A.grid.step + GT_FLAT * A.grid.rem / (uint32_t)Ng;
    const float df = (float)(GT_FLAT * A.grid.rem % (uint32_t)Ng) / (float)Ng;
    float mine = 0.f;
#pragma unroll 1
    for (int b = 0; b < NB; ++b) {
        const int p = b * (32 / GT_FLAT) + lane / GT_FLAT;  // the lane's particle of this round
        const uint32_t pu = __shfl_sync(0xffffffffu, u, p);
        const float pk = __shfl_sync(0xffffffffu, k2, p);
        const int pl = __shfl_sync(0xffffffffu, len, p);
        int g = __shfl_sync(0xffffffffu, g0, p) + sub;
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        uint32_t nc;
        float nf, e = 0.f;
        pxy_node(A.grid, g < Ng ? g : 0, nc, nf);
#pragma unroll 2
        for (int r = sub; r < pl; r += GT_FLAT) {
            e = fmaf(kde_ex2(pk * pxy_sin2(nc, nf, pu, 0.f)), A.field[g], e);
            g += GT_FLAT;
            while (g >= Ng) g -= Ng;
            nc += dn;
            nf += df;
            if (nf >= 1.f) {
                nf -= 1.f;
                ++nc;
            }
        }
#pragma unroll
        for (int o = GT_FLAT / 2; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
        const float v = __shfl_sync(0xffffffffu, e, (lane & (32 / GT_FLAT - 1)) * GT_FLAT);
        if ((lane & (PW - 1)) / (32 / GT_FLAT) == b) mine = v;
    }
    if (lane < PW && j < A.N) A.out[j] = mine * nm * A.coef;
}

// intervals of a width's (or a band's largest width's) table: half-width a = pi / C with
// a sqrt(kappa + 1.5) at most ymax
static int gt_intervals_of(double kappa, double ymax)
{
    const int C = (int)ceil(KDE_PI / ymax * sqrt(kappa + 1.5));
    return C < 4 ? 4 : C;
}

static uint32_t gt_step(int C) { return (uint32_t)((1ull << 32) / (uint64_t)(2 * C)); }

struct GtLayout {
    GtBands T;
    int total;
};
static const GtLayout &gt_layout()
{
    static const GtLayout lay = [] {
        GtLayout l;
        l.total = 0;
        for (int b = 0; b < GT_BANDS; ++b) {
            // the triangle of degree 6 keeps 5e-8 of the peak (2e-8 in L2) up to y = 0.16
            l.T.C[b] = gt_intervals_of(0.5 * exp2(0.5 * b), 0.16);
            l.T.off[b] = l.total;
            l.T.step[b] = gt_step(l.T.C[b]);
            l.total += l.T.C[b];
        }
        return l;
    }();
    return lay;
}

// table and partial ranges, always of the bands' size (4.2 MB; one width needs at most 260 KB),
// so that a context that has gathered once gathers anything under capture
static float *gt_workspace(kde_ctx *ctx)
{
    return (float *)kde_ws(ctx, WS_GTAB, (size_t)gt_layout().total * GT_NC * 4 + GT_KR_BLOCKS * sizeof(float2));
}

kde_status kde_gather_table_reserve(kde_ctx *ctx) { return gt_workspace(ctx) ? KDE_OK : KDE_ENOMEM; }

kde_status kde_gather_table(kde_ctx *ctx, const uint32_t *u, const float *kappa, double kappa_u, int64_t N,
                            const float *field, int Ng, float *out)
{
    GtArgs A{};
    A.u = u;
    A.kappa = kappa;
    A.kappa_u = (float)kappa_u;
    A.norm_u = kappa ? 0.f : (float)kde_norm(kappa_u);
    A.coef = (float)(KDE_TWO_PI / Ng);
    A.N = N;
    A.field = field;
    A.grid = pxy_grid(Ng);
    A.pxt = ctx->pxy_tab;
    A.ntab = ctx->norm_tab;
    A.out = out;
    A.status = ctx->d_status;
    A.tab = gt_workspace(ctx);
    if (!A.tab) return KDE_ENOMEM;
    const int sms = ctx->sm_count > 0 ? ctx->sm_count : 1;
    KdeProfScope _ps(ctx, PROF_GATHER);
    // few (particle, node) pairs: one launch that sweeps them, for about 0.086 / NB ns a particle and
    // 1e-3 a pair over 4 us, where the two launches of one width's table take 8 us and the bands' three
    // 20 (narrow ranges of widths) to 42 (5 to 5000): swept and from tables, 65,536 particles and 512
    // nodes 31 and 20, 37 and 41; 200,003 and 64 25 and 18, 25 and 41
    const int64_t full = 64LL * sms * (32 / GT_FLAT);  // particles of a full machine at one round
    const int nb = N >= 8 * full ? 8 : (N >= 4 * full ? 4 : (N >= 2 * full ? 2 : 1));
    if (kappa ? (double)N * (0.086 / nb + 1e-3 * Ng) <= 4.0e4 : (double)N * Ng <= 4194304.0) {
        const int64_t per = (int64_t)GT_WARPS * (32 / GT_FLAT) * nb;
        const unsigned gf = (unsigned)((N + per - 1) / per);
        switch (nb) {
        case 8: gt_flat_kernel<8><<<gf, GT_THREADS, 0, ctx->stream>>>(A); break;
        case 4: gt_flat_kernel<4><<<gf, GT_THREADS, 0, ctx->stream>>>(A); break;
        case 2: gt_flat_kernel<2><<<gf, GT_THREADS, 0, ctx->stream>>>(A); break;
        default: gt_flat_kernel<1><<<gf, GT_THREADS, 0, ctx->stream>>>(A);
        }
        KDE_LAUNCHED(ctx, "gt_flat_kernel");
        return KDE_OK;
    }
    if (!kappa) {
        const int C = gt_intervals_of(kappa_u, 0.388);
        const int grid = C < 4 * sms ? C : 4 * sms;
        gt_table_one_kernel<<<grid, GT_THREADS, 0, ctx->stream>>>(A, C, gt_step(C));
        KDE_LAUNCHED(ctx, "gt_table_one_kernel");
        const unsigned ge = (unsigned)((N + 4 * GT_THREADS - 1) / (4 * GT_THREADS));
        KDE_CUDA(ctx, kde_launch(ctx, true, gt_eval_one_kernel, dim3(ge), dim3(GT_THREADS), 0, A, C), "gt_eval_one_kernel");
        KDE_LAUNCHED(ctx, "gt_eval_one_kernel");
        return KDE_OK;
    }
    GtBands T = gt_layout().T;
    for (int b = 0; b < GT_BANDS; ++b) T.W[b] = b ? std::min(Ng, kde_window_nodes(0.5 * exp2(0.5 * (b - 1)), Ng) + 1) : Ng;
    const int64_t want = (N + 4 * GT_THREADS - 1) / (4 * GT_THREADS);
    A.nkr = (int)(want < GT_KR_BLOCKS ? want : GT_KR_BLOCKS);
    float2 *kr = (float2 *)(A.tab + (size_t)gt_layout().total * GT_NC);
    A.kr = kr;
    gt_range_kernel<<<A.nkr, GT_THREADS, 0, ctx->stream>>>(A, kr);
    KDE_LAUNCHED(ctx, "gt_range_kernel");
    KDE_CUDA(ctx, kde_launch(ctx, true, gt_table_bands_kernel, dim3(2 * sms), dim3(GT_THREADS), 0, A, T),
             "gt_table_bands_kernel");
    KDE_LAUNCHED(ctx, "gt_table_bands_kernel");
    const unsigned ge = (unsigned)((N + 2 * GT_THREADS - 1) / (2 * GT_THREADS));
    KDE_CUDA(ctx, kde_launch(ctx, true, gt_eval_bands_kernel, dim3(ge), dim3(GT_THREADS), 0, A, T), "gt_eval_bands_kernel");
    KDE_LAUNCHED(ctx, "gt_eval_bands_kernel");
    return KDE_OK;
}
