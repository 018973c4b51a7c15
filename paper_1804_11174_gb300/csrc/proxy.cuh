// proxy.cuh -- compression of many particles into few proxy particles.
//
// A kernel value f(theta_g; theta, kappa) = exp(-2 kappa sin^2((theta_g - theta)/2)), and
// norm(kappa) f as well, is a smooth function of the particle's position and width, so over
// an interval of positions of half-width a and widths in [kmin, kmax] it equals its
// Chebyshev interpolant
//     f(theta_g; theta, kappa) = sum_{a<P, b<Q} l_a(x) l_b(s) f(theta_g; theta_a, kappa_b),
// x in [-1, 1] the position in the interval and s that of the width in its range, theta_a
// and kappa_b the Chebyshev points (first kind).  A deposit sums its particles' weights into
// P Q moments, turns these into P Q proxy particles (theta_a, kappa_b) with signed weights
// and sweeps the nodes with the proxies alone; a gather evaluates the field at the proxies
// and interpolates it at the particles.
//
// Degrees.  With y = a sqrt(kmax + 1.5) the interpolation error in position is below
// 2 (y/2)^P / sqrt(P!) of the kernel's peak (derivatives of a Gaussian of variance 1/kappa;
// the 1.5 covers small widths, where the cosine and not kappa sets the scale).  In the width
// it depends on the range alone and holds for every distance: a linear map of kappa for
// narrow ranges (by r = (kmax - kmin) / (kmax + kmin)), a linear map of ln kappa for wide
// ones (by ln(kmax / kmin)).  P and Q are the smallest that keep each error below 2e-8 of
// the peak: below one FP32 rounding, and below the 2^-24 at which kernels are truncated.
#pragma once

#include "common.cuh"

#define PXY_MAXP 16
#define PXY_MAXQ 40

// interpolation matrices of degree D, c[p][a] = (2 - [p = 0]) / D cos(pi p (2a + 1) / (2D)),
// D = 1 .. PXY_MAXQ one after another (built in FP64 when the context is created)
__host__ __device__ constexpr int pxy_tab_off(int D) { return (D - 1) * D * (2 * D - 1) / 6; }
#define PXY_TAB_N pxy_tab_off(PXY_MAXQ + 1)

// smallest P with 2 (y/2)^P / sqrt(P!) <= 2e-8; PXY_MAXP + 1 when there is none up to PXY_MAXP
__device__ __forceinline__ int pxy_degree_pos(float y)
{
    return 3 + (y > 0.0058f) + (y > 0.0298f) + (y > 0.0811f) + (y > 0.1606f) + (y > 0.2646f) + (y > 0.3880f) +
           (y > 0.5260f) + (y > 0.6746f) + (y > 0.8304f) + (y > 0.9909f) + (y > 1.1544f) + (y > 1.3193f) +
           (y > 1.4845f) + (y > 1.6493f);
}
// the linear map of kappa reaches 2e-8 with six points up to this r
#define PXY_LIN_R 0.12f
// smallest Q whose interpolant of e^{-s e^t} in t has an error of at most 2e-8 for every
// s >= 0 over a range of length l = ln(kmax / kmin) (measured; 4.5 + 4.86 l bounds it above
// l = 0.379); above PXY_MAXQ when the range is too wide
__device__ __forceinline__ int pxy_degree_log(float l)
{
    if (l <= 0.379f) return 3 + (l > 0.0208f) + (l > 0.0861f) + (l > 0.2077f);
    return (int)fminf(ceilf(fmaf(4.86f, l, 4.5f)), 1000.f);
}

// an Ng-node grid in position codes: node g is at code g step + (g rem) / Ng, with
// 2^32 = step Ng + rem (g rem < 2^24)
struct PxyGrid {
    int Ng;
    uint32_t step, rem;
};
inline PxyGrid pxy_grid(int Ng)
{
    PxyGrid g;
    g.Ng = Ng;
    g.step = (uint32_t)((1ull << 32) / (uint64_t)Ng);  // Ng = 1: 2^32 wraps to 0, and the only node is 0
    g.rem = (uint32_t)((1ull << 32) % (uint64_t)Ng);
    return g;
}
__device__ __forceinline__ void pxy_node(const PxyGrid &G, int g, uint32_t &code, float &frac)
{
    code = (uint32_t)g * G.step;
    frac = 0.f;
    if (G.rem) {
        const uint32_t m = (uint32_t)g * G.rem, q = m / (uint32_t)G.Ng;
        code += q;
        frac = (float)(m - q * (uint32_t)G.Ng) / (float)G.Ng;
    }
}

// interval of positions and range of widths
struct PxyBox {
    uint32_t mid;  // middle position (code)
    float hw;      // half-width in codes
    float inv_hw;
    float kc, kh, inv_kh;  // middle and half-length of the range of kappa (linear) or ln kappa
    int P, Q;              // degrees (Q = 1: one width)
    bool lin;
};

// positions of the whole cells [c_first, c_last], 0 <= c_first <= c_last < Ng
__device__ __forceinline__ void pxy_box_pos(PxyBox &B, const PxyGrid &G, int c_first, int c_last, float kmax)
{
    uint32_t lo, hi;
    float f;
    pxy_node(G, c_first, lo, f);
    pxy_node(G, c_last + 1, hi, f);  // the end of the grid, 2^32, wraps to 0
    if (c_last + 1 == G.Ng) hi = 0u;
    const uint32_t len = hi - lo;  // 0: the whole circle
    const uint32_t half = len ? (len >> 1) + (len & 1u) : 0x80000000u;
    B.mid = lo + half;
    B.hw = (float)half;
    B.inv_hw = 1.f / B.hw;
    B.P = pxy_degree_pos(B.hw * (float)(KDE_TWO_PI / 4294967296.0) * sqrtf(kmax + 1.5f));
}
// a range of widths narrow enough for the linear map
__device__ __forceinline__ bool pxy_narrow(float kmin, float kmax) { return kmax - kmin <= PXY_LIN_R * (kmax + kmin); }
// middle and half-length of a narrow range of widths.  The middle is rounded, so over a range of
// a few roundings the ends would lie outside [-1, 1] (at 2 for two neighbouring floats, where the
// highest polynomials reach 1e3 and their rounding 1e-5 of the result): at least 1e-5 of the
// middle, and 1e-30 for the widths next to zero, whose kernels are all the constant one
__device__ __forceinline__ void pxy_lin_range(float kmin, float kmax, float &kc, float &kh)
{
    kc = 0.5f * (kmin + kmax);
    kh = fmaxf(0.5f * (kmax - kmin), fmaxf(1e-5f * kc, 1e-30f));
}
__device__ __forceinline__ void pxy_box_width(PxyBox &B, float kmin, float kmax)
{
    B.lin = pxy_narrow(kmin, kmax);
    if (kmin == kmax) {
        B.Q = 1;
        B.kc = kmin;
        B.kh = B.inv_kh = 0.f;
    } else if (B.lin) {
        B.Q = 6;
        pxy_lin_range(kmin, kmax, B.kc, B.kh);
        B.inv_kh = 1.f / B.kh;
    } else {
        const float l0 = logf(kmin), l1 = logf(kmax);
        B.Q = pxy_degree_log(l1 - l0);
        B.kc = 0.5f * (l0 + l1);
        B.kh = 0.5f * (l1 - l0);
        B.inv_kh = 1.f / B.kh;
    }
}

// norms of the proxy widths of a narrow range, behind the range's two words: PXY_NORM7 + b for
// Q = 7, PXY_NORM6 + b for Q = 6, in FP64 and rounded (kde_krange_block).  The proxies' norms
// are a factor on the whole density, so the table's 5e-7 would be the field's.
#define PXY_NORM7 4
#define PXY_NORM6 12
// width of proxy b (of Q) of a narrow range, c = c[1][b] of the matrix of degree Q
__device__ __forceinline__ float pxy_lin_kappa(float kc, float kh, float c, int Q)
{
    return fmaf(kh, c * (0.5f * (float)Q), kc);
}

// 1 / k!^2 and the coefficients of Hankel's series, prod_{j <= k} (2j - 1)^2 / (8j)
struct PxySeries {
    double inv_fact_sq[64], hankel[32];
    constexpr PxySeries() : inv_fact_sq(), hankel()
    {
        inv_fact_sq[0] = hankel[0] = 1.0;
        for (int k = 1; k < 64; ++k) inv_fact_sq[k] = inv_fact_sq[k - 1] / ((double)k * k);
        for (int k = 1; k < 32; ++k) hankel[k] = hankel[k - 1] * ((2.0 * k - 1.0) * (2.0 * k - 1.0) / (8.0 * k));
    }
};
static __device__ const PxySeries pxy_series{};

// 1 / (2 pi I0e(x)) in FP64 of two values by a warp, lane 0 the first's and lane 1 the second's: the
// series of kde_i0e with a term or two a lane, below 30 sum (x^2 / 4)^k / k!^2 (64 terms), above sum
// hankel_k / x^k (32 terms, still falling there).  A dependent FP64 operation takes some 40 clocks
// here: term by term, on a lane a value, the series took 5 us
__device__ __forceinline__ double pxy_norm_warp(const double (&x)[2], int lane)
{
    double z[2], p[2] = {1.0, 1.0}, t[2];
#pragma unroll
    for (int v = 0; v < 2; ++v) z[v] = x[v] < 30.0 ? 0.25 * x[v] * x[v] : 1.0 / x[v];
#pragma unroll
    for (int b = 0; b < 5; ++b)  // p = z^lane, z = z^32 at the end
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            if (lane >> b & 1) p[v] *= z[v];
            z[v] *= z[v];
        }
#pragma unroll
    for (int v = 0; v < 2; ++v)
        t[v] = x[v] < 30.0 ? p[v] * fma(z[v], pxy_series.inv_fact_sq[lane + 32], pxy_series.inv_fact_sq[lane])
                           : p[v] * pxy_series.hankel[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int v = 0; v < 2; ++v) t[v] += __shfl_xor_sync(0xffffffffu, t[v], o);
    const double y = lane ? x[1] : x[0], s = KDE_TWO_PI * (lane ? t[1] : t[0]);
    return (y < 30.0 ? exp(y) : sqrt(KDE_TWO_PI * y)) / s;
}

// the range of the widths that a kernel writes (KDE_KRANGE_ACC): called once by all 256 threads of every
// block with the extremes of the thread's own (lo = 3e38, hi = 0 without any).  One pair of atomics a
// block (the first blocks all find the range unset, and a pair a warp queued up on the one
// address); the last block moves the range to its place, adds the norms of the proxy widths of a
// narrow one and leaves the gathering words reset: a kernel of its own for that, and memsets before
// every pass, took 8 us of a call
__device__ __forceinline__ void kde_krange_block(unsigned int *krange, const float *pxt, float lo, float hi)
{
    __shared__ unsigned int rl[8], rh[8], last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned int *acc = krange + KDE_KRANGE_ACC;
    const unsigned int h = __reduce_max_sync(0xffffffffu, __float_as_uint(hi));
    const unsigned int l = __reduce_min_sync(0xffffffffu, __float_as_uint(lo));
    if (lane == 0) {
        rh[warp] = h;
        rl[warp] = l;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int a = rh[0], b = rl[0];
#pragma unroll
        for (int w = 1; w < 8; ++w) {
            a = max(a, rh[w]);
            b = min(b, rl[w]);
        }
        if (a > __ldcg(&acc[0])) atomicMax(&acc[0], a);
        if (b < __ldcg(&acc[1])) atomicMin(&acc[1], b);
        __threadfence();
        last = atomicAdd(&acc[2], 1u) == gridDim.x - 1 ? 1u : 0u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const unsigned int bh = __ldcg(&acc[0]), bl = __ldcg(&acc[1]);
    const float kmax = __uint_as_float(bh), kmin = __uint_as_float(bl);
    __syncthreads();  // read by all before the reset
    if (threadIdx.x == 0) {
        krange[0] = bh;
        krange[1] = bl;
        acc[0] = 0u;
        acc[1] = 0x7f7f7f7fu;
        acc[2] = 0u;
    }
    if (!pxy_narrow(kmin, kmax)) return;
    float kc, kh;
    pxy_lin_range(kmin, kmax, kc, kh);
    // values 0 .. 6 are those of Q = 7, 7 .. 12 those of Q = 6
    const int i0 = min(2 * warp, 12), i1 = min(2 * warp + 1, 12);
    auto width = [&](int i) {
        const int Q = i < 7 ? 7 : 6;
        return (double)pxy_lin_kappa(kc, kh, pxt[pxy_tab_off(Q) + Q + (i < 7 ? i : i - 7)], Q);
    };
    const double x[2] = {width(i0), width(i1)};
    const double n = pxy_norm_warp(x, lane);
    const int i = lane ? i1 : i0;
    if (lane < 2) krange[i < 7 ? PXY_NORM7 + i : PXY_NORM6 + i - 7] = __float_as_uint((float)n);
}

// position in the box, [-1, 1]: the code difference is exact
__device__ __forceinline__ float pxy_x(const PxyBox &B, uint32_t u) { return (float)(int32_t)(u - B.mid) * B.inv_hw; }
__device__ __forceinline__ float pxy_s(const PxyBox &B, float kappa)
{
    return ((B.lin ? kappa : logf(kappa)) - B.kc) * B.inv_kh;
}
// proxy a of P at Chebyshev point x: code and fraction of a code (the rounding of the
// product is carried exactly)
__device__ __forceinline__ void pxy_pos(const PxyBox &B, float x, uint32_t &code, float &frac)
{
    const float p = B.hw * x, e = fmaf(B.hw, x, -p), r = rintf(p);
    code = B.mid + (uint32_t)__float2int_rn(r);
    frac = (p - r) + e;
}
// proxy width at Chebyshev point s
__device__ __forceinline__ float pxy_kappa(const PxyBox &B, float s)
{
    const float k = fmaf(B.kh, s, B.kc);
    return B.lin ? k : expf(k);
}

// sine and cosine of half the angle between two positions: sin(pi f), cos(pi f), f in
// [-1/2, 1/2] the difference in turns, by their Taylor series (the first terms left out are
// below 7e-10 relative to the sine and 6e-9 of the cosine's unit)
__device__ __forceinline__ void pxy_sincos(uint32_t na, float fa, uint32_t nb, float fb, float &s, float &c)
{
    const float f = ((float)(int32_t)(na - nb) + (fa - fb)) * (1.f / 4294967296.f), t = f * f;
    s = (float)(0.00046630280576761256);  // pi^13 / 13!
    s = fmaf(s, t, (float)(-0.0073704309457143504));
    s = fmaf(s, t, (float)(0.082145886611128228));
    s = fmaf(s, t, (float)(-0.59926452932079208));
    s = fmaf(s, t, (float)(2.5501640398773454));
    s = fmaf(s, t, (float)(-5.1677127800499701));
    s = fmaf(s, t, (float)(3.1415926535897932));
    s *= f;
    c = (float)(0.0019295743094039231);  // pi^12 / 12!
    c = fmaf(c, t, (float)(-0.025806891390014061));
    c = fmaf(c, t, (float)(0.23533063035889321));
    c = fmaf(c, t, (float)(-1.3352627688545895));
    c = fmaf(c, t, (float)(4.0587121264167682));
    c = fmaf(c, t, (float)(-4.9348022005446793));
    c = fmaf(c, t, 1.f);
}

// sin^2 of half the angle between two positions given as codes and fractions.  The code
// difference is exact, so near pairs keep full relative accuracy; sin(pi f) for
// f in [-1/2, 1/2] by its Taylor series (the first term left out is below 7e-10 relative)
__device__ __forceinline__ float pxy_sin2(uint32_t na, float fa, uint32_t nb, float fb)
{
    const float f = ((float)(int32_t)(na - nb) + (fa - fb)) * (1.f / 4294967296.f), t = f * f;
    float s = (float)(0.00046630280576761256);  // pi^13 / 13!
    s = fmaf(s, t, (float)(-0.0073704309457143504));
    s = fmaf(s, t, (float)(0.082145886611128228));
    s = fmaf(s, t, (float)(-0.59926452932079208));
    s = fmaf(s, t, (float)(2.5501640398773454));
    s = fmaf(s, t, (float)(-5.1677127800499701));
    s = fmaf(s, t, (float)(3.1415926535897932));
    s *= f;
    return s * s;
}
