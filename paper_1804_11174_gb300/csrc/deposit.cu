// deposit.cu -- KDE deposit (Eq. kde evaluated at the grid nodes).
//
//   rho_g = sum_i w_i (2 pi / L) norm(kappa_i) exp(-2 kappa_i sin^2((theta_g - theta_i)/2))
//
// Layout: particles are counting-sorted by cell (small plain calls keep their
// order).  One CTA takes a range of consecutive particles and finds the node
// range their truncated kernels can reach.  FP32 ranges whose positions and
// widths span a small box are compressed into interpolation points with signed
// weights (proxy.cuh); the others stage (beta sin, beta cos, w*norm) of each
// particle in shared memory.  Lanes own nodes (node-owner formulation): a warp
// sweeps 32 consecutive nodes over a slice of the points, so every point is a
// shared-memory broadcast and each lane accumulates in a register without
// atomics.  Slices are combined in a fixed order in shared memory.  A CTA's
// sums are converted to int64 fixed point (an exact power-of-two scale below
// the largest possible node value) and added with integer atomics, so the grid
// sum is exact and independent of the order in which CTAs finish: results are
// bitwise reproducible.
#include "common.cuh"
#include "fp64.cuh"
#include "proxy.cuh"

#define DEP_THREADS 256
#define DEP_WARPS (DEP_THREADS / 32)
#define DEP_CHUNK 1024
#define CV_MAXM 8192

template <typename T> struct V2;
template <> struct V2<float> { typedef float2 t; };
template <> struct V2<double> { typedef double2 t; };

template <typename T> struct DepRec {
    T bs, bc, wn;
};

template <typename T> struct DepSrc {
    const uint32_t *u;
    int64_t N;
    const T *kappa;      // per-particle widths, or nullptr
    T kappa_u;           // uniform width
    T kscale;            // CV: widths are kscale * kappa[j] in scale mode, else 1
    const T *norm;       // FP64: per-particle norm, or nullptr (computed from the width when kappa != nullptr)
    const float *lnorm;  // log2 of per-particle norm (CV scale mode), or nullptr
    T norm_u;            // uniform norm
    const T *w;          // per-particle weights, or nullptr
    T w_u;               // uniform weight
    T coef;              // 2 pi / L (x units) or 1 (theta units)
    int Ng;
    const typename V2<T>::t *nodes;  // (sin, cos) of half node angles; nullptr: Ng is a power of two
    long long *acc;
    double bound;                    // largest possible node value
    const unsigned int *wmax_bits;   // if not null: bound = N * coef * norm_bound * w_max (float bits)
    double norm_bound;
    unsigned int *status;
    int scale_exp;  // KDE_ES_FROM_BOUND, or the exponent es of the fixed-point scale 2^es
    const float2 *ntab;  // FP32 norm table (kde_norm_tab) for per-particle widths
    float xcut = (float)KDE_XCUT;  // FP32 packed kernels: truncation cut exponent (kde_fp32_cut)
    int nbins = 0;                   // sort bins of the particles: 0 the cells, -1 not sorted at all
    PxyGrid grid;                    // the nodes as position codes
    const float *pxt;                // interpolation matrices (proxy.cuh)
    const unsigned int *krange;      // float bits of the largest and smallest width, or null
};

#define KDE_ES_FROM_BOUND (-100000)

// exponent es of the fixed-point scale kde_acc_scale(bound) = 2^es
__device__ __forceinline__ int acc_scale_exp(double bound)
{
    int e;
    frexp(bound > 0 ? bound : 1.0, &e);
    return 62 - e;
}

// x 2^es rounded to the nearest integer, ties to even, in integer arithmetic: for
// -100 <= es <= 100 the same value as __double2ll_rn((double)x * 2^es) (the product
// is exact in FP64), without touching the FP64 pipe, which is slow on this part.
// |x| 2^es must stay below 2^62 (the scale's bound guarantees it).
__device__ __forceinline__ long long fix_pow2(float x, int es)
{
    const uint32_t b = __float_as_uint(x);
    const int be = (int)((b >> 23) & 0xffu);
    if (be == 0) return 0;  // zero or subnormal: |x| 2^es < 2^-126 2^100 < 1/2
    const int ex = be - 150 + es;  // |x| 2^es = m 2^ex with the 24-bit significand m
    const uint32_t m = (b & 0x7fffffu) | 0x800000u;
    long long q;
    if (ex >= 0) {
        q = (long long)m << (ex < 39 ? ex : 39);
    } else if (ex < -24) {
        q = 0;  // below 1/2
    } else {
        const int sh = -ex;  // 1 .. 24
        const uint32_t qq = m >> sh, rem = m & ((1u << sh) - 1u), half = 1u << (sh - 1);
        q = (long long)(qq + ((rem > half || (rem == half && (qq & 1u))) ? 1u : 0u));
    }
    return (b >> 31) ? -q : q;
}

__device__ __forceinline__ int window_nodes_f(float kappa, int Ng, float xcut)
{
    float s2 = xcut * (float)(KDE_LN2 / 2.0) / kappa;
    if (s2 >= 1.0f) return Ng;
    float r = 2.0f * asinf(sqrtf(s2));
    int w = (int)ceilf(r * (float)Ng * (float)(1.0 / KDE_TWO_PI)) + 1;
    return w >= Ng ? Ng : w;
}

template <typename T>
__device__ __forceinline__ void node_sc(const DepSrc<T> &S, int g, T &s, T &c)
{
    if (S.nodes) {
        typename V2<T>::t v = S.nodes[g];
        s = v.x;
        c = v.y;
    } else {
        // power-of-two grid: g / Ng is exact
        float sf, cf;
        sincospif((float)g / (float)S.Ng, &sf, &cf);
        s = sf;
        c = cf;
    }
}

// a chunk of particles in any order (kde_deposit_noalloc)
template <typename T>
__device__ void deposit_chunk_body(const DepSrc<T> &S, int64_t chunk, DepRec<T> *rec, T *part, int *red, int *cmm)
{
    const int64_t i0 = chunk * DEP_CHUNK;
    if (i0 >= S.N) return;
    const int n = (int)(S.N - i0 < DEP_CHUNK ? S.N - i0 : DEP_CHUNK);
    const int Ng = S.Ng;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    int wloc = 0;
    int cmin = 0x7fffffff, cmax = -1;
    for (int t = tid; t < n; t += DEP_THREADS) {
        int64_t j = i0 + t;
        uint32_t uu = S.u[j];
        int cc = kde_cell(uu, S.Ng);
        cmin = cc < cmin ? cc : cmin;
        cmax = cc > cmax ? cc : cmax;
        T k = S.kappa ? S.kappa[j] : S.kappa_u;
        if (!(k > (T)0 && k <= (T)KDE_KAPPA_MAX)) {
            kde_flag(S.status, KDE_DEV_KAPPA_RANGE, (unsigned)j);
            k = (T)KDE_KAPPA_MAX;
        }
        const T nm = S.kappa ? (T)kde_norm((double)k) : S.norm_u;
        T wj = S.w ? S.w[j] : S.w_u;
        T sh, ch;
        kde_half_sincos(uu, sh, ch);
        T beta = sqrt((T)(2.0 * KDE_LOG2E) * k);
        rec[t].bs = beta * sh;
        rec[t].bc = beta * ch;
        rec[t].wn = wj * S.coef * nm;
        int wn_ = window_nodes_f((float)k, Ng, (float)KdeCut<T>::x);
        wloc = wn_ > wloc ? wn_ : wloc;
    }
    // block maximum of the window
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        int v = __shfl_xor_sync(0xffffffffu, wloc, o);
        wloc = v > wloc ? v : wloc;
    }
    if (lane == 0) red[warp] = wloc;
    __syncthreads();
    int W = 0;
#pragma unroll
    for (int k = 0; k < DEP_WARPS; ++k) W = red[k] > W ? red[k] : W;
    // the chunk's linear cell range (a range that wraps around the grid falls back to the whole
    // grid below)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cmin = min(cmin, __shfl_xor_sync(0xffffffffu, cmin, o));
        cmax = max(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
    }
    if (lane == 0) {
        cmm[warp] = cmin;
        cmm[DEP_WARPS + warp] = cmax;
    }
    __syncthreads();
    int c_first = cmm[0], c_last = cmm[DEP_WARPS];
#pragma unroll
    for (int k = 1; k < DEP_WARPS; ++k) {
        c_first = min(c_first, cmm[k]);
        c_last = max(c_last, cmm[DEP_WARPS + k]);
    }
    int g_lo = c_first - W;
    int R = c_last + W - g_lo + 1;
    if (R >= Ng || c_last < c_first) {
        g_lo = 0;
        R = Ng;
    }
    const int ngroups = (R + 31) >> 5;

    double bound = S.bound;
    if (S.wmax_bits) bound = (double)S.N * (double)S.coef * S.norm_bound * (double)__uint_as_float(*S.wmax_bits);
    const double scale = kde_acc_scale(bound);

    if (ngroups >= DEP_WARPS) {
        for (int gi = warp; gi < ngroups; gi += DEP_WARPS) {
            int r = gi * 32 + lane;
            int g = g_lo + r;
            g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
            T Sg, Cg;
            node_sc(S, r < R ? g : 0, Sg, Cg);
            T acc = 0;
#pragma unroll 4
            for (int p = 0; p < n; ++p) {
                DepRec<T> q = rec[p];
                T s = Sg * q.bc - Cg * q.bs;
                acc += kde_ex2(-s * s) * q.wn;
            }
            if (r < R) {
                long long v = __double2ll_rn((double)acc * scale);
                if (v) atomicAdd((unsigned long long *)&S.acc[g], (unsigned long long)v);
            }
        }
        return;
    }
    const int slices = DEP_WARPS / ngroups;
    const int gi = warp % ngroups, sl = warp / ngroups;
    if (sl < slices) {
        int p0 = (int)((int64_t)n * sl / slices), p1 = (int)((int64_t)n * (sl + 1) / slices);
        int r = gi * 32 + lane;
        int g = g_lo + r;
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        T Sg, Cg;
        node_sc(S, r < R ? g : 0, Sg, Cg);
        T acc = 0;
#pragma unroll 4
        for (int p = p0; p < p1; ++p) {
            DepRec<T> q = rec[p];
            T s = Sg * q.bc - Cg * q.bs;
            acc += kde_ex2(-s * s) * q.wn;
        }
        part[sl * (DEP_WARPS * 32) + r] = acc;
    }
    __syncthreads();
    for (int r = tid; r < ngroups * 32; r += DEP_THREADS) {
        if (r >= R) continue;
        T acc = 0;
        for (int k = 0; k < slices; ++k) acc += part[k * (DEP_WARPS * 32) + r];
        int g = g_lo + r;
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        long long v = __double2ll_rn((double)acc * scale);
        if (v) atomicAdd((unsigned long long *)&S.acc[g], (unsigned long long)v);
    }
}

// ---------------------------------------------------------------------------
// FP32 chunk body of the CV's integral term, with packed pair arithmetic: each lane owns two
// nodes (a warp pass covers 64 consecutive nodes) and every particle record is staged
// pre-duplicated, so that one 128-bit and one 64-bit broadcast load feed the f32x2 multiply-adds
// of both nodes.  Same node range, slicing and fixed-order combination as the scalar body.  The
// kernel value is 2^-(S_g beta c_j - C_g beta s_j)^2 with (s, c) the sine and cosine of half the
// angle, records (beta s, beta s, beta c, beta c) and (w n, w n): four multiply-adds per pair.
// ---------------------------------------------------------------------------
#define DEP2_PART 512
#define DEP2_UNROLL_P1 4
#define DEP2_UNROLL_P2 8

// node phase of the packed deposit: each lane owns P pairs of nodes, so a warp pass
// covers 64 P consecutive nodes of the chunk's range [g_lo, g_lo + R); with fewer
// groups than warps the warps split the particles into slices whose partial sums
// are combined in a fixed order
template <int P>
__device__ __forceinline__ void dep2_nodes(const DepSrc<float> &S, int n, int g_lo, int R, int es,
                                           const float4 *rsc, const float2 *rwn, float *part)
{
    constexpr int GW = 64 * P;
    constexpr int U = P == 2 ? DEP2_UNROLL_P2 : DEP2_UNROLL_P1;  // particle loop unrolling
    const int Ng = S.Ng;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ngroups = (R + GW - 1) / GW;
    const bool fix_int = es >= -100 && es <= 100;
    // the FP64 conversion, for extreme bounds only; 2^es built from its bits
    const double scale = __longlong_as_double((long long)(1023 + (es < -1000 ? -1000 : (es > 1000 ? 1000 : es))) << 52);

    int gn[2 * P];
    bool ok[2 * P];
    kde_f2 SS[P], CC[P], acc[P];
    auto nodes_of = [&](int gi) {
#pragma unroll
        for (int m = 0; m < 2 * P; ++m) {
            const int r = gi * GW + m * 32 + lane;
            ok[m] = r < R;
            int g = g_lo + r;
            g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
            gn[m] = g;
        }
#pragma unroll
        for (int q = 0; q < P; ++q) {
            float sa, ca, sb, cb;
            node_sc(S, ok[2 * q] ? gn[2 * q] : 0, sa, ca);
            node_sc(S, ok[2 * q + 1] ? gn[2 * q + 1] : 0, sb, cb);
            SS[q] = kde_pk(sa, sb);
            CC[q] = kde_pk(-ca, -cb);
        }
    };
    auto sweep = [&](int p0, int p1) {
#pragma unroll
        for (int q = 0; q < P; ++q) acc[q] = kde_pk(0.f, 0.f);
#pragma unroll U
        for (int p = p0; p < p1; ++p) {
            const float4 r4 = rsc[p];
            const float2 w2 = rwn[p];
            const kde_f2 qs = kde_pk(r4.z, r4.w), qc = kde_pk(r4.x, r4.y), w = kde_pk(w2.x, w2.y);
            // s = S_g (beta cos_j) - C_g (beta sin_j)
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const kde_f2 sv = kde_fma2(SS[q], qs, kde_mul2(CC[q], qc));
                acc[q] = kde_fma2(kde_ex2neg2(kde_mul2(sv, sv)), w, acc[q]);
            }
        }
    };
    auto fix = [&](float a) -> long long { return fix_int ? fix_pow2(a, es) : __double2ll_rn((double)a * scale); };

    if (ngroups >= DEP_WARPS) {
        for (int gi = warp; gi < ngroups; gi += DEP_WARPS) {
            nodes_of(gi);
            sweep(0, n);
#pragma unroll
            for (int q = 0; q < P; ++q) {
                float a0, a1;
                kde_upk(acc[q], a0, a1);
                long long v;
                if (ok[2 * q] && (v = fix(a0)) != 0) atomicAdd((unsigned long long *)&S.acc[gn[2 * q]], (unsigned long long)v);
                if (ok[2 * q + 1] && (v = fix(a1)) != 0)
                    atomicAdd((unsigned long long *)&S.acc[gn[2 * q + 1]], (unsigned long long)v);
            }
        }
        return;
    }
    // every warp works: warp w takes node group w mod ngroups and one of that group's
    // particle slices (the groups' slice counts differ by at most one); ngroups GW <= DEP2_PART
    const int gi = warp % ngroups, sl = warp / ngroups;
    const int slices = (DEP_WARPS - gi + ngroups - 1) / ngroups;
    {
        const int p0 = (int)((int64_t)n * sl / slices), p1 = (int)((int64_t)n * (sl + 1) / slices);
        nodes_of(gi);
        sweep(p0, p1);
#pragma unroll
        for (int q = 0; q < P; ++q) {
            float a0, a1;
            kde_upk(acc[q], a0, a1);
            part[sl * DEP2_PART + gi * GW + 64 * q + lane] = a0;
            part[sl * DEP2_PART + gi * GW + 64 * q + 32 + lane] = a1;
        }
    }
    __syncthreads();
    for (int r = tid; r < ngroups * GW; r += DEP_THREADS) {
        if (r >= R) continue;
        const int gr = r / GW, sr = (DEP_WARPS - gr + ngroups - 1) / ngroups;
        float a = 0.f;
        for (int k = 0; k < sr; ++k) a += part[k * DEP2_PART + r];
        int g = g_lo + r;
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        const long long v = fix(a);
        if (v) atomicAdd((unsigned long long *)&S.acc[g], (unsigned long long)v);
    }
}

__device__ void deposit_chunk_body_x2(const DepSrc<float> &S, int64_t chunk, float4 *rsc, float2 *rwn, float *part,
                                      int *red)
{
    const int64_t i0 = chunk * DEP_CHUNK;
    if (i0 >= S.N) return;
    const int n = (int)(S.N - i0 < DEP_CHUNK ? S.N - i0 : DEP_CHUNK);
    const int Ng = S.Ng;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // every input of the thread's particles loaded at once (one global-load latency per
    // chunk); the smallest width sets the window
    constexpr int PER = DEP_CHUNK / DEP_THREADS;
    uint32_t ru[PER];
    float rk[PER], rn[PER];
    float kmin = (float)KDE_KAPPA_MAX;
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int t = tid + p * DEP_THREADS;
        const bool ok = t < n;
        const int64_t j = i0 + (ok ? t : 0);
        ru[p] = S.u[j];
        float k = S.kappa ? S.kscale * S.kappa[j] : S.kappa_u;
        rn[p] = S.lnorm ? S.lnorm[j] : 0.f;
        if (ok && !(k > 0.f && k <= (float)KDE_KAPPA_MAX)) {
            kde_flag(S.status, KDE_DEV_KAPPA_RANGE, (unsigned)j);
            k = (float)KDE_KAPPA_MAX;
        }
        rk[p] = k;
        if (ok) kmin = fminf(kmin, k);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kmin = fminf(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
    if (lane == 0) red[warp] = __float_as_int(kmin);
    __syncthreads();
    const int es = S.scale_exp;
#pragma unroll
    for (int k = 0; k < DEP_WARPS; ++k) kmin = fminf(kmin, __int_as_float(red[k]));
    // the window shrinks as the width grows: the smallest width's window covers all
    const int W = window_nodes_f(kmin, Ng, S.xcut);
    // the particle records
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int t = tid + p * DEP_THREADS;
        if (t >= n) break;
        const uint32_t uu = ru[p];
        const float k = rk[p];
        const float nm = S.lnorm ? exp2f(rn[p]) : S.norm_u;
        const float wn = S.w_u * S.coef * nm;
        float sh, ch;
        kde_half_sincos(uu, sh, ch);
        const float beta = sqrtf((float)(2.0 * KDE_LOG2E) * k);
        rsc[t] = make_float4(beta * sh, beta * sh, beta * ch, beta * ch);
        rwn[t] = make_float2(wn, wn);
    }
    __syncthreads();
    const int c_first = kde_cell(S.u[i0], Ng), c_last = kde_cell(S.u[i0 + n - 1], Ng);
    int g_lo = c_first - W;
    int R = c_last + W - g_lo + 1;
    if (R >= Ng || R < 1 || c_last < c_first) {
        g_lo = 0;
        R = Ng;
    }
    // two node pairs a lane halve the particle loads per pair: taken where the wider
    // groups compute no extra nodes and their partial sums fit the buffer
    const int n64 = (R + 63) >> 6, n128 = (R + 127) >> 7;
    if (2 * n128 == n64 && (n128 >= DEP_WARPS || n128 * 128 <= DEP2_PART))
        dep2_nodes<2>(S, n, g_lo, R, es, rsc, rwn, part);
    else
        dep2_nodes<1>(S, n, g_lo, R, es, rsc, rwn, part);
}

// ---------------------------------------------------------------------------
// FP64 deposit of cell-sorted particles.  Bound by the FP64 pipe (two lanes a clock and SM):
// eleven operations a (particle, node) pair, against about 23 with exp2, and chunks short
// enough to reach every SM.  A CTA stages its chunk (beta sin, beta cos, w norm) and hands
// out (node, slice of the particles) tasks to its threads; the slices of a node are added in
// order, then the node's sum goes to the int64 accumulators as in the FP32 chunk kernels.
// Measured: 4096 particles on 64 nodes 363 -> 13 us, 65,537 particles with particle-wise
// widths on 100 nodes 958 -> 200 us.
// ---------------------------------------------------------------------------
#define DEP64_MAXCHUNK 256
#define DEP64_TASKS 1024

__global__ void __launch_bounds__(DEP_THREADS) deposit64_kernel(DepSrc<double> S, int chunk, const double *__restrict__ tab2)
{
    __shared__ __align__(16) double tab[F64_TAB];
    __shared__ double bs[DEP64_MAXCHUNK], bc[DEP64_MAXCHUNK], wn[DEP64_MAXCHUNK], part[DEP64_TASKS];
    __shared__ int red[DEP_WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, Ng = S.Ng;
    const int64_t i0 = (int64_t)blockIdx.x * chunk;
    const int n = (int)(S.N - i0 < chunk ? S.N - i0 : chunk);
    f64_tab_load(tab, tab2, tid, DEP_THREADS);
    int W = 0;
    for (int t = tid; t < n; t += DEP_THREADS) {
        const int64_t j = i0 + t;
        double k = S.kappa ? S.kappa[j] : S.kappa_u;
        if (!(k > 0.0 && k <= KDE_KAPPA_MAX)) {
            kde_flag(S.status, KDE_DEV_KAPPA_RANGE, (unsigned)j);
            k = KDE_KAPPA_MAX;
        }
        const double nm = S.norm ? S.norm[j] : (S.kappa ? f64_norm(k) : S.norm_u);
        double sh, ch;
        kde_half_sincos(S.u[j], sh, ch);
        const double beta = sqrt(2.0 * KDE_LOG2E * k);
        bs[t] = beta * sh;
        bc[t] = beta * ch;
        wn[t] = (S.w ? S.w[j] : S.w_u) * S.coef * nm;
        W = max(W, window_nodes_f((float)k, Ng, (float)KDE_XCUT64));
    }
    W = __reduce_max_sync(0xffffffffu, W);
    if (lane == 0) red[warp] = W;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < DEP_WARPS; ++w) W = max(W, red[w]);
    const int c_first = kde_cell(S.u[i0], Ng), c_last = kde_cell(S.u[i0 + n - 1], Ng);
    int g_lo = c_first - W, R = c_last + W - g_lo + 1;
    if (R >= Ng || R < 1 || c_last < c_first) {
        g_lo = 0;
        R = Ng;
    }
    const double bound = S.wmax_bits
                             ? (double)S.N * S.coef * S.norm_bound * (double)__uint_as_float(*S.wmax_bits)
                             : S.bound;
    const double scale = kde_acc_scale(bound);
    auto add = [&](int r, double a) {
        int g = g_lo + r;
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        // the quantum is far below a node's value but not below its rounding, and there are many
        // chunks: the remainder goes to a second word, in units of 2^-24 of the quantum
        const double x = a * scale;
        const long long v = __double2ll_rn(x), l = __double2ll_rn((x - (double)v) * 16777216.0);
        if (v) atomicAdd((unsigned long long *)&S.acc[g], (unsigned long long)v);
        if (l) atomicAdd((unsigned long long *)&S.acc[Ng + g], (unsigned long long)l);
    };
    auto sum = [&](int r, int p0, int dp) -> double {
        int g = g_lo + r;
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        const double2 sc = S.nodes[g];
        double acc = 0.0;
#pragma unroll 4
        for (int p = p0; p < n; p += dp) {
            const double s = fma(sc.x, bc[p], -(sc.y * bs[p]));
            double T, q;
            f64_exp2neg(tab, s, T, q);
            const double tw = T * wn[p];
            acc = fma(tw, q, acc) + tw;
        }
        return acc;
    };
    const int SL = min(n, DEP64_TASKS / R);
    if (SL <= 1) {
        for (int r = tid; r < R; r += DEP_THREADS) add(r, sum(r, 0, 1));
        return;
    }
    for (int t = tid; t < R * SL; t += DEP_THREADS) {
        const int sl = t / R;
        part[t] = sum(t - sl * R, sl, SL);
    }
    __syncthreads();
    for (int r = tid; r < R; r += DEP_THREADS) {
        double a = 0.0;
        for (int k = 0; k < SL; ++k) a += part[k * R + r];
        add(r, a);
    }
}

// ---------------------------------------------------------------------------
// FP32 deposit of cell-sorted particles over a balanced persistent grid.
//
// G = min(3 x SMs, ceil(N / 256)) CTAs (one wave); CTA c owns the contiguous
// particles [c N / G, (c + 1) N / G), so every CTA carries the same number of
// particles and, since a particle's cost is its window, nearly the same work.
// The CTA's node window is fixed up front: its first and last cell widened by the
// window of its smallest width.  Its particles are taken in sub-chunks of
// DEPP_SUB records (one float4 each: the two angle terms and the weighted norm;
// a Landau-size run of 2^20 particles has one sub-chunk a CTA), the inputs of a
// sub-chunk loaded in batches of register loads, and swept by node-owner lanes as
// in the chunk kernel (f32x2 pairs of nodes, fixed-order combination of particle
// slices).  After every sub-chunk the FP32 node sums become int64 fixed point and are
// added to the grid's sums by integer reductions in the L2, at most Ng a CTA (456 x 256
// at Landau size, about 1 us), exact and independent of any order.  Rows per CTA and a
// second pass over them took 8 us a step of the field kernel.
// ---------------------------------------------------------------------------
#define DEPP_THREADS 256
#define DEPP_WARPS 8
#define DEPP_MINB 3  // CTAs an SM (80 registers a thread): 7% faster than 4 at 64 registers
#define DEPP_SUB 2304  // records a sub-chunk: a 2^20-particle run has one sub-chunk a CTA
#define DEPP_PART 512

struct DepPlan {
    int G;            // CTAs
    long long *acc;   // [Ng] node sums, zero before
    float inv_share;  // 1 / CTAs an SM, at most DEPP_MINB of them (depp_compress_pays)
};
// node pairs of the persistent deposit: each lane owns P pairs of nodes (64 P
// consecutive nodes a warp pass) of the window [g_lo, g_lo + R); the n records of
// the sub-chunk are split into slices when there are fewer node groups than warps.
// flush(r, a) receives the FP32 sum of window node r over the sub-chunk, once per node.
template <int P, typename F>
__device__ __forceinline__ void depp_sweep(const DepSrc<float> &S, int n, int g_lo, int R, bool cosf,
                                           const float4 *rec, float *part, F &&flush)
{
    constexpr int GW = 64 * P;
    constexpr int U = 4;
    const int Ng = S.Ng;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ngroups = (R + GW - 1) / GW;
    kde_f2 SS[P], CC[P], acc[P];
    auto nodes_of = [&](int gi) {
#pragma unroll
        for (int q = 0; q < P; ++q) {
            float sa, ca, sb, cb;
            const int ra = gi * GW + 64 * q + lane, rb = ra + 32;
            int ga = g_lo + ra, gb = g_lo + rb;
            ga = ga < 0 ? ga + Ng : (ga >= Ng ? ga - Ng : ga);
            gb = gb < 0 ? gb + Ng : (gb >= Ng ? gb - Ng : gb);
            node_sc(S, ra < R ? ga : 0, sa, ca);
            node_sc(S, rb < R ? gb : 0, sb, cb);
            if (cosf) {
                SS[q] = kde_pk(2.f * sa * ca, 2.f * sb * cb);
                CC[q] = kde_pk((ca - sa) * (ca + sa), (cb - sb) * (cb + sb));
            } else {
                SS[q] = kde_pk(sa, sb);
                CC[q] = kde_pk(-ca, -cb);
            }
        }
    };
    // record (a, b, w): cosine form a = K cos x_j, b = K sin x_j, exponent
    // S_g b + C_g a = K cos(x_j - x_g); half-angle form a = beta sin, b = beta cos of
    // half the angle, s = S_g b - C_g a and the exponent -s^2
    auto sweep = [&](int p0, int p1) {
#pragma unroll
        for (int q = 0; q < P; ++q) acc[q] = kde_pk(0.f, 0.f);
        if (cosf) {
#pragma unroll U
            for (int p = p0; p < p1; ++p) {
                const float4 r4 = rec[p];
                const kde_f2 qa = kde_pk(r4.x, r4.x), qb = kde_pk(r4.y, r4.y), w = kde_pk(r4.z, r4.z);
#pragma unroll
                for (int q = 0; q < P; ++q)
                    acc[q] = kde_fma2(kde_ex22(kde_fma2(SS[q], qb, kde_mul2(CC[q], qa))), w, acc[q]);
            }
        } else {
#pragma unroll U
            for (int p = p0; p < p1; ++p) {
                const float4 r4 = rec[p];
                const kde_f2 qa = kde_pk(r4.x, r4.x), qb = kde_pk(r4.y, r4.y), w = kde_pk(r4.z, r4.z);
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const kde_f2 sv = kde_fma2(SS[q], qb, kde_mul2(CC[q], qa));
                    acc[q] = kde_fma2(kde_ex2neg2(kde_mul2(sv, sv)), w, acc[q]);
                }
            }
        }
    };
    if (ngroups >= DEPP_WARPS) {
        for (int gi = warp; gi < ngroups; gi += DEPP_WARPS) {
            nodes_of(gi);
            sweep(0, n);
#pragma unroll
            for (int q = 0; q < P; ++q) {
                float a0, a1;
                kde_upk(acc[q], a0, a1);
                const int ra = gi * GW + 64 * q + lane;
                if (ra < R) flush(ra, a0);
                if (ra + 32 < R) flush(ra + 32, a1);
            }
        }
        return;
    }
    // every warp works: warp w takes node group w mod ngroups and one of that group's
    // particle slices (slice counts differ by at most one); ngroups GW <= DEPP_PART
    const int gi = warp % ngroups, sl = warp / ngroups;
    const int slices = (DEPP_WARPS - gi + ngroups - 1) / ngroups;
    {
        const int p0 = (int)((int64_t)n * sl / slices), p1 = (int)((int64_t)n * (sl + 1) / slices);
        nodes_of(gi);
        sweep(p0, p1);
#pragma unroll
        for (int q = 0; q < P; ++q) {
            float a0, a1;
            kde_upk(acc[q], a0, a1);
            part[sl * DEPP_PART + gi * GW + 64 * q + lane] = a0;
            part[sl * DEPP_PART + gi * GW + 64 * q + 32 + lane] = a1;
        }
    }
    __syncthreads();
    for (int r = tid; r < ngroups * GW; r += DEPP_THREADS) {
        if (r >= R) continue;
        const int gr = r / GW, sr = (DEPP_WARPS - gr + ngroups - 1) / ngroups;
        float a = 0.f;
        for (int k = 0; k < sr; ++k) a += part[k * DEPP_PART + r];
        flush(r, a);
    }
}

// narrow windows (R <= 32 NPL nodes): the records are kept in particle pairs, recAB[k] =
// (a_2k, a_2k+1, b_2k, b_2k+1) and recW[k] = (w_2k, w_2k+1), so that one packed operation
// serves two particles of the same node.  A lane owns NPL nodes (j, j + LG, ...) of its
// group of LG lanes; the 32 / LG groups of a warp (slices) and the eight warps take
// interleaved particle pairs.  Slice sums are combined by a fixed butterfly over the lane
// bits above LG, warp sums in warp order; flush(r, a) receives each node's sum once.
template <int LG, int NPL, typename F>
__device__ __forceinline__ void depp_sweep_pairs(const DepSrc<float> &S, int n, int g_lo, int R, bool cosf,
                                                 const float4 *recAB, const float2 *recW, float *part, F &&flush)
{
    constexpr int SL = 32 / LG;
    constexpr int U = 4;
    const int Ng = S.Ng;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j = lane & (LG - 1), sl = lane / LG;
    kde_f2 SS[NPL], CC[NPL], acc[NPL];
#pragma unroll
    for (int t = 0; t < NPL; ++t) {
        const int r = j + LG * t;
        int g = g_lo + r;
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        float sg, cg;
        node_sc(S, r < R ? g : 0, sg, cg);
        if (cosf) {
            const float sf = 2.f * sg * cg, cf = (cg - sg) * (cg + sg);
            SS[t] = kde_pk(sf, sf);
            CC[t] = kde_pk(cf, cf);
        } else {
            SS[t] = kde_pk(sg, sg);
            CC[t] = kde_pk(-cg, -cg);
        }
        acc[t] = kde_pk(0.f, 0.f);
    }
    const int np = (n + 1) >> 1;
    const int k0 = (int)((int64_t)np * warp / DEPP_WARPS), k1 = (int)((int64_t)np * (warp + 1) / DEPP_WARPS);
    if (cosf) {
#pragma unroll U
        for (int k = k0 + sl; k < k1; k += SL) {
            const float4 ab = recAB[k];
            const float2 w = recW[k];
            const kde_f2 A = kde_pk(ab.x, ab.y), B = kde_pk(ab.z, ab.w), W2 = kde_pk(w.x, w.y);
#pragma unroll
            for (int t = 0; t < NPL; ++t) acc[t] = kde_fma2(kde_ex22(kde_fma2(SS[t], B, kde_mul2(CC[t], A))), W2, acc[t]);
        }
    } else {
#pragma unroll U
        for (int k = k0 + sl; k < k1; k += SL) {
            const float4 ab = recAB[k];
            const float2 w = recW[k];
            const kde_f2 A = kde_pk(ab.x, ab.y), B = kde_pk(ab.z, ab.w), W2 = kde_pk(w.x, w.y);
#pragma unroll
            for (int t = 0; t < NPL; ++t) {
                const kde_f2 sv = kde_fma2(SS[t], B, kde_mul2(CC[t], A));
                acc[t] = kde_fma2(kde_ex2neg2(kde_mul2(sv, sv)), W2, acc[t]);
            }
        }
    }
#pragma unroll
    for (int t = 0; t < NPL; ++t) {
        float a0, a1;
        kde_upk(acc[t], a0, a1);
        float a = a0 + a1;
#pragma unroll
        for (int o = LG; o < 32; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (sl == 0) part[warp * DEPP_PART + j + LG * t] = a;
    }
    __syncthreads();
    for (int r = tid; r < R; r += DEPP_THREADS) {
        float a = 0.f;
#pragma unroll
        for (int w = 0; w < DEPP_WARPS; ++w) a += part[w * DEPP_PART + r];
        flush(r, a);
    }
}

// ---------------------------------------------------------------------------
// Compressed form of a CTA's deposit (proxy.cuh): its particles, an interval of whole
// cells with widths in [kmin, kmax], become P Q proxy particles, and only the proxies sweep
// the node window.  Moments M_pq = sum_i w_i T_p(x_i) T_q(s_i), three ways:
//  * one width (Q = 1): P sums a thread in registers;
//  * a narrow range of widths and P <= 8: a thread's products in registers too (the
//    normalisation is interpolated with the kernel, so no norm is read);
//  * otherwise a small matrix product: a warp stages the T_p (times weight and norm) of 16
//    particles and their T_q, and its lanes own 4 x 4 tiles of the P x Q sums.
// Warp and CTA sums follow in a fixed order.
//
// What bounds it: the direct sweep spends one exp2 and three or four multiply-adds on every
// (particle, node) pair, 256 a particle for whole-grid windows; here a particle costs the
// Chebyshev values and 28 to 48 multiply-adds (a few hundred in the matrix form) whatever the
// window, and is bound by instruction fetch and issue and load latency.  Measured (by events around
// the launch): 2^20 particles, 256 nodes, widths near 14 45.0 -> 15.0 us; 4,000,037 particles, 4096
// nodes, widths log-uniform in [5, 5e3] 2389 -> 315 us.
// ---------------------------------------------------------------------------
#define PXY_STAGE 16  // particles a warp stages at a time

__device__ __forceinline__ float depp_kappa(const DepSrc<float> &S, float k, int64_t j)
{
    if (!(k > 0.f && k <= (float)KDE_KAPPA_MAX)) {
        kde_flag(S.status, KDE_DEV_KAPPA_RANGE, (unsigned)j);
        k = (float)KDE_KAPPA_MAX;
    }
    return k;
}

// the moments kept by the register form: all of PM x QM, or with TRI those with
// p / PM + q / QM < 1 (the coefficients of the joint interpolant fall off in p and q together)
template <int PM, int QM, bool TRI>
__host__ __device__ constexpr bool depp_kept(int p, int q)
{
    return !TRI || p * QM + q * PM < PM * QM;
}
template <int PM, int QM, bool TRI> __host__ __device__ constexpr int depp_count(int upto)
{
    int n = 0;
    for (int i = 0; i < upto; ++i) n += depp_kept<PM, QM, TRI>(i / QM, i % QM) ? 1 : 0;
    return n;
}

// FP32 sums of particles run over PXY_SEG particles of the CTA at most, 16 a thread; beyond, sums
// are pairs of floats (FP64, slow on this part, took 4 us a launch for the same).  One weight for
// all makes the zeroth moment add the same number every time, so that its rounding is a bias
// which all threads and CTAs share: over a thread's whole share it was 2.7e-7 (rms) of the
// density at 2^22 particles, 4e-6 at 2^26 and growing with N.  Four particles are added up first,
// so the segment's chain of equal terms is four long, which loses nothing.
#define PXY_SEG 4096

// (s.x + s.y) + v with s.x the rounded sum and s.y what it lost (Knuth's two-sum)
__device__ __forceinline__ float2 depp_add2(float2 s, float v)
{
    const float t = s.x + v, b = t - s.x;
    return make_float2(t, s.y + ((s.x - (t - b)) + (v - b)));
}

template <int PM, int QM, bool TRI>
__device__ __forceinline__ void depp_moments_reg(const DepSrc<float> &S, int64_t i0, int n, const PxyBox &B,
                                                 float *part, float *M)
{
    constexpr int NM = depp_count<PM, QM, TRI>(PM * QM), QB = 4;
    constexpr int NR = (NM + 31) / 32;
    static_assert(PXY_SEG % (QB * DEPP_THREADS) == 0, "whole rounds a segment");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t *u = S.u + i0;
    const float *kap = S.kappa ? S.kappa + i0 : nullptr, *w = S.w ? S.w + i0 : nullptr;
    float2 *tot = (float2 *)part + warp * 64;  // the warp's sums, moments lane and lane + 32 a lane's own
#pragma unroll
    for (int h = 0; h < NR; ++h) tot[h * 32 + lane] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int s0 = 0; s0 < n; s0 += PXY_SEG) {
        const int s1 = min(n, s0 + PXY_SEG);
        float acc[NM];
#pragma unroll
        for (int i = 0; i < NM; ++i) acc[i] = 0.f;
#pragma unroll 1
        for (int b0 = s0 + tid; b0 < s1; b0 += QB * DEPP_THREADS) {
            uint32_t ru[QB];
            float rk[QB], rw[QB], sum[PM];
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                const int t = b0 + q * DEPP_THREADS;
                const int j = t < s1 ? t : 0;
                ru[q] = u[j];
                rk[q] = QM > 1 ? kap[j] : 0.f;
                rw[q] = t < s1 ? (w ? w[j] : S.w_u) : 0.f;
            }
#pragma unroll
            for (int p = 0; p < PM; ++p) sum[p] = 0.f;
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                if (b0 - tid + q * DEPP_THREADS >= s1) break;  // the CTA has no particle left
                const float x = pxy_x(B, ru[q]), x2 = x + x;
                float tp[PM];
                tp[0] = rw[q];
                tp[1] = tp[0] * x;
#pragma unroll
                for (int p = 2; p < PM; ++p) tp[p] = fmaf(x2, tp[p - 1], -tp[p - 2]);
#pragma unroll
                for (int p = 0; p < PM; ++p) sum[p] += tp[p];
                if constexpr (QM > 1) {
                    float k = rk[q];
                    if (!(k > 0.f && k <= (float)KDE_KAPPA_MAX)) k = depp_kappa(S, k, i0 + b0 + q * DEPP_THREADS);
                    const float sv = (k - B.kc) * B.inv_kh, s2 = sv + sv;
                    // t0 = T_{r-1}(s), t1 = T_r(s)
                    float t0 = 1.f, t1 = sv;
#pragma unroll
                    for (int r = 1; r < QM; ++r) {
#pragma unroll
                        for (int p = 0; p < PM; ++p)
                            if (depp_kept<PM, QM, TRI>(p, r)) {
                                const int m = depp_count<PM, QM, TRI>(p * QM + r);
                                acc[m] = fmaf(tp[p], t1, acc[m]);
                            }
                        const float t2 = fmaf(s2, t1, -t0);
                        t0 = t1;
                        t1 = t2;
                    }
                }
            }
#pragma unroll
            for (int p = 0; p < PM; ++p) acc[depp_count<PM, QM, TRI>(p * QM)] += sum[p];
        }
        // lane l has the warp's sums of moments l, l + 32
        if (NM <= 8) {
            float mine = 0.f;
#pragma unroll
            for (int i = 0; i < NM; ++i) {
                float v = acc[i];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == i) mine = v;
            }
            tot[lane] = depp_add2(tot[lane], mine);
        } else {
#pragma unroll
            for (int h = 0; h < NR; ++h) {
                float v[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = h * 32 + i < NM ? acc[h * 32 + i < NM ? h * 32 + i : 0] : 0.f;
                tot[h * 32 + lane] = depp_add2(tot[h * 32 + lane], warp_transpose_sum32(v, lane));
            }
        }
    }
    const float2 *wsum = (const float2 *)part;
    __syncthreads();
    for (int i = tid; i < PM * QM; i += DEPP_THREADS) {
        float2 a = make_float2(0.f, 0.f);
        int m = i;  // position of moment (p, q) among the kept ones
        bool kept = true;
        if (TRI) {
            kept = depp_kept<PM, QM, TRI>(i / QM, i % QM);
            m = 0;
            for (int p = 0; p < i / QM; ++p) m += (QM * (PM - p) + PM - 1) / PM;
            m += i % QM;
        }
        if (kept) {
#pragma unroll
            for (int k = 0; k < DEPP_WARPS; ++k) {
                const float2 v = wsum[k * 64 + m];
                a = depp_add2(a, v.x);
                a.y += v.y;
            }
        }
        M[i] = (a.x + a.y) * S.coef;
    }
}

// moments of any degrees (P <= 16, Q <= 40) as a matrix product; mem: the CTA's DEPP_SUB float4.
// A lane's chain in registers is 64 / KS particles long (half that at KS <= 2), then part adds up
// those of a segment of PXY_MMSEG particles, and the segments are added up in pairs of floats (the
// request-size deposit below 472 -> 491 us for the whole call)
#define PXY_MMSEG 4096
#define PXY_ROWS (PXY_STAGE * 60)  // floats of a warp's staged rows, RS <= 60 each

__device__ __forceinline__ void depp_moments_mm(const DepSrc<float> &S, int64_t i0, int n, const PxyBox &B,
                                                float *mem, float *part, float *M)
{
    static_assert(DEPP_WARPS * PXY_ROWS + 2 * PXY_MAXP * PXY_MAXQ <= 4 * DEPP_SUB, "rows and sums fit");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t *u = S.u + i0;
    const float *kap = S.kappa + i0, *w = S.w ? S.w + i0 : nullptr;
    float *stage = mem + warp * PXY_ROWS;
    float2 *tot = (float2 *)(mem + DEPP_WARPS * PXY_ROWS);  // the moments of the segments so far
    float4 *pw = (float4 *)part + warp * 128 + lane;          // part[warp][row of the tile][lane][4]
    const int LP = (B.P + 3) >> 2, LQ = (B.Q + 3) >> 2;
    const int RS = 4 * ((LP + LQ) | 1);  // an odd number of 16-byte words
    const int tiles = LP * LQ;
    int KS = 1;  // particles taken at once (power of two, KS tiles <= 32)
    while (2 * KS * tiles <= 32 && 2 * KS <= PXY_STAGE) KS *= 2;
    const int ks = lane / tiles, tile = lane - ks * tiles, lp = tile / LQ, lq = tile - lp * LQ;
    const bool on = ks < KS;
    const int row = lane & (PXY_STAGE - 1);  // the particle this lane stages
    const bool roleB = lane >= PXY_STAGE;    // lanes 0..15 the T_p, lanes 16..31 the T_q
    constexpr int QB = 4;
    constexpr int step = DEPP_WARPS * PXY_STAGE;
    for (int i = tid; i < B.P * B.Q; i += DEPP_THREADS) tot[i] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int s0 = 0; s0 < n; s0 += PXY_MMSEG) {
        const int s1 = min(n, s0 + PXY_MMSEG);
        float acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            pw[a * 32] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
        }
        auto fold = [&]() {
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float4 v = pw[a * 32];
                pw[a * 32] = make_float4(v.x + acc[a][0], v.y + acc[a][1], v.z + acc[a][2], v.w + acc[a][3]);
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
            }
        };
#pragma unroll 1
        for (int g0 = s0 + warp * PXY_STAGE; g0 < s1; g0 += QB * step) {
            uint32_t ru[QB];
            float rk[QB], rw[QB];
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                const int t = g0 + q * step + row;
                const int j = t < s1 ? t : 0;
                ru[q] = u[j];
                rk[q] = kap[j];
                rw[q] = w ? w[j] : S.w_u;
            }
#pragma unroll 1
            for (int q = 0; q < QB; ++q) {
                const int t0 = g0 + q * step;
                if (t0 >= s1) break;
                const bool ok = t0 + row < s1;
                // the first of the recurrence: the weight or 1; rows past the end have no weight and sit
                // in the middle of the box (values far outside it would overflow, and 0 inf is no 0)
                float z = 0.f, y0 = roleB ? 1.f : 0.f;
                if (ok) {
                    const float k = depp_kappa(S, rk[0], i0 + t0 + row);
                    z = roleB ? pxy_s(B, k) : pxy_x(B, ru[0]);
                    if (!roleB) y0 = rw[0] * S.coef * kde_norm_tab(S.ntab, k);
                }
#pragma unroll
                for (int i = 0; i + 1 < QB; ++i) {
                    ru[i] = ru[i + 1];
                    rk[i] = rk[i + 1];
                    rw[i] = rw[i + 1];
                }
                float y1 = y0 * z;
                const float z2 = z + z;
                float4 *dst = (float4 *)(stage + row * RS) + (roleB ? LP : 0);
                const int n4 = roleB ? LQ : LP;
                for (int i = 0; i < n4; ++i) {
                    const float y2 = fmaf(z2, y1, -y0), y3 = fmaf(z2, y2, -y1);
                    dst[i] = make_float4(y0, y1, y2, y3);
                    y0 = fmaf(z2, y3, -y2);
                    y1 = fmaf(z2, y0, -y3);
                }
                __syncwarp();
                if (on) {
#pragma unroll 4
                    for (int r = ks; r < PXY_STAGE; r += KS) {
                        const float4 A = *(const float4 *)(stage + r * RS + 4 * lp);
                        const float4 Q4 = *(const float4 *)(stage + r * RS + 4 * (LP + lq));
                        const float av[4] = {A.x, A.y, A.z, A.w}, bv[4] = {Q4.x, Q4.y, Q4.z, Q4.w};
#pragma unroll
                        for (int a = 0; a < 4; ++a)
#pragma unroll
                            for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(av[a], bv[b], acc[a][b]);
                    }
                }
                if (KS <= 2 && q == 1) fold();
                __syncwarp();
            }
            fold();
        }
        // moment (p, q) over the warps and their particle groups
        __syncthreads();
        for (int i = tid; i < B.P * B.Q; i += DEPP_THREADS) {
            const int p = i / B.Q, q = i - p * B.Q;
            const int off = ((p & 3) * 32 + (p >> 2) * LQ + (q >> 2)) * 4 + (q & 3);
            float2 m = tot[i];
            for (int v = 0; v < DEPP_WARPS; ++v) {
                float a = 0.f;
                for (int g = 0; g < KS; ++g) a += part[v * 512 + g * tiles * 4 + off];
                m = depp_add2(m, a);
            }
            tot[i] = m;
            M[i] = m.x + m.y;
        }
        __syncthreads();
    }
}

// moments -> proxies -> node window: flush(r, a) receives the sum at window node r.
// mem: at least 2 P Q + 2 P + Q floats; part: DEPP_WARPS DEPP_PART floats
template <typename F>
__device__ __forceinline__ void depp_proxies(const DepSrc<float> &S, const PxyBox &B, int g_lo, int R,
                                             const float *M, float *mem, float *part, F &&flush)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int P = B.P, Q = B.Q, PQ = P * Q, Ng = S.Ng;
    const float *cp = S.pxt + pxy_tab_off(P), *cq = S.pxt + pxy_tab_off(Q);
    float *U = mem, *W = U + PQ, *sd = W + PQ, *cd = sd + P, *k2 = cd + P;
    // sine and cosine of half the proxies' angles from the box's middle, and exponent factors -2 kappa_b log2 e (the Chebyshev points are
    // the matrices' second rows times D / 2)
    if (tid < P)
        sincospif(cp[P + tid] * (0.5f * (float)P) * (B.hw * (1.f / 4294967296.f)), &sd[tid], &cd[tid]);
    if (tid >= 64 && tid < 64 + Q) {
        const int b = tid - 64;
        k2[b] = (float)(-2.0 * KDE_LOG2E) * pxy_kappa(B, cq[Q + b] * (0.5f * (float)Q));
    }
    __syncthreads();  // also: the moments are written
    for (int i = tid; i < PQ; i += DEPP_THREADS) {
        const int a = i / Q, q = i - a * Q;
        float s = 0.f;
        for (int p = 0; p < P; ++p) s = fmaf(cp[p * P + a], M[p * Q + q], s);
        U[i] = s;
    }
    __syncthreads();
    for (int i = tid; i < PQ; i += DEPP_THREADS) {
        const int a = i / Q, b = i - a * Q;
        float s = 0.f;
        for (int q = 0; q < Q; ++q) s = fmaf(cq[q * Q + b], U[a * Q + q], s);
        W[i] = s;
    }
    __syncthreads();
    // a thread takes a node and every SL-th proxy position; the widest kernels (last b)
    // come first, and a kernel below 2^-32 of its peak ends the row
    const int ng = (R + 31) >> 5;  // node groups of a warp
    const int SL = ng >= DEPP_WARPS ? 1 : DEPP_WARPS / ng;
    auto node = [&](int r, int a0, int da) -> float {
        int g = g_lo + r;
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        uint32_t nc;
        float nf;
        pxy_node(S.grid, g, nc, nf);
        float acc = 0.f, sn, cn;
        pxy_sincos(nc, nf, B.mid, 0.f, sn, cn);
#pragma unroll 1
        for (int a = a0; a < P; a += da) {
            // the box is at most 1.65 standard deviations of its narrowest kernel wide on either
            // side, so the angle difference keeps 1e-7 of that width
            const float sa = fmaf(sn, cd[a], -cn * sd[a]), s2 = sa * sa;
            const float *w = W + a * Q;
            int b = Q - 1;
            for (; b >= 3; b -= 4) {  // four at a time: the first has the largest value
                const float e = s2 * k2[b];
                if (e < -32.f) break;
                const float e0 = kde_ex2(e) * w[b], e1 = kde_ex2(s2 * k2[b - 1]) * w[b - 1];
                const float e2 = kde_ex2(s2 * k2[b - 2]) * w[b - 2], e3 = kde_ex2(s2 * k2[b - 3]) * w[b - 3];
                acc += (e0 + e1) + (e2 + e3);
            }
            if (b < 3)
                for (; b >= 0; --b) acc = fmaf(kde_ex2(s2 * k2[b]), w[b], acc);
        }
        return acc;
    };
    if (SL == 1) {
#pragma unroll 1
        for (int r = tid; r < R; r += DEPP_THREADS) flush(r, node(r, 0, 1));
        return;
    }
    const int gi = warp % ng, sl = warp / ng, r = gi * 32 + lane;
    if (sl < SL) part[sl * DEPP_PART + r] = r < R ? node(r, sl, SL) : 0.f;
    __syncthreads();
    for (int q = tid; q < R; q += DEPP_THREADS) {
        float a = 0.f;
        for (int k = 0; k < SL; ++k) a += part[k * DEPP_PART + q];
        flush(q, a);
    }
}

// the same for the degrees of the register forms, unrolled (the proxies carry the widths'
// norms); mem: 2 PM QM + 2 PM + QM + PM PM + QM QM floats
template <int PM, int QM, typename F>
__device__ __forceinline__ void depp_proxies_reg(const DepSrc<float> &S, const PxyBox &B, int g_lo, int R, const float *M,
                                                 const float *tabs, bool shared_range, float *mem, float *part, F &&flush)
{
    constexpr int PQ = PM * QM;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, Ng = S.Ng;
    const float *cp = tabs, *cq = tabs + PM * PM;
    float *U = mem, *W = U + PQ + (PQ & 1), *k2 = W + PQ, *nk = k2 + QM;
    float2 *sc = (float2 *)(nk + QM + (PQ & 1));  // an even number of floats from mem
    static_assert((PQ + (PQ & 1) + PQ + 2 * QM + (PQ & 1)) % 2 == 0, "float2 alignment");
    if (tid < PM) {
        const float x = cp[PM + tid] * (0.5f * (float)PM);
        float sn, cs;
        sincospif(x * (B.hw * (1.f / 4294967296.f)), &sn, &cs);
        sc[tid] = make_float2(sn, cs);
    }
    if (tid >= 32 && tid < 32 + QM) {
        const int b = tid - 32;
        const float k = QM > 1 ? pxy_lin_kappa(B.kc, B.kh, cq[QM + b], QM) : B.kc;
        k2[b] = (float)(-2.0 * KDE_LOG2E) * k;
        if (!S.kappa) nk[b] = S.norm_u;
        else if (QM > 1 && shared_range) nk[b] = __uint_as_float(S.krange[(QM == 7 ? PXY_NORM7 : PXY_NORM6) + b]);
        else nk[b] = kde_norm_tab(S.ntab, k);
    }
    __syncthreads();  // also: the moments are written
    if (tid < PQ) {
        const int a = tid / QM, q = tid % QM;
        float s = 0.f;
#pragma unroll
        for (int p = 0; p < PM; ++p) s = fmaf(cp[p * PM + a], M[p * QM + q], s);
        U[tid] = s;
    }
    __syncthreads();
    if (tid < PQ) {
        const int a = tid / QM, b = tid % QM;
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < QM; ++q) s = fmaf(cq[q * QM + b], U[a * QM + q], s);
        W[tid] = s * nk[b];
    }
    __syncthreads();
    float kk[QM];
#pragma unroll
    for (int b = 0; b < QM; ++b) kk[b] = k2[b];
    // a thread takes a node and every SL-th proxy position
    const int ng = (R + 31) >> 5;
    const int SL = ng >= DEPP_WARPS ? 1 : DEPP_WARPS / ng;
    auto node = [&](int r, int a0) -> float {
        int g = g_lo + r;
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        uint32_t nc;
        float nf, sn, cn, acc = 0.f;
        pxy_node(S.grid, g, nc, nf);
        pxy_sincos(nc, nf, B.mid, 0.f, sn, cn);
#pragma unroll 1
        for (int a = a0; a < PM; a += SL) {
            const float2 p = sc[a];
            const float sa = fmaf(sn, p.y, -cn * p.x), s2 = sa * sa;
            const float *w = W + a * QM;
#pragma unroll
            for (int b = 0; b < QM; ++b) acc = fmaf(kde_ex2(s2 * kk[b]), w[b], acc);
        }
        return acc;
    };
    if (SL == 1) {
#pragma unroll 1
        for (int r = tid; r < R; r += DEPP_THREADS) flush(r, node(r, 0));
        return;
    }
    const int gi = warp % ng, sl = warp / ng, r = gi * 32 + lane;
    if (sl < SL) part[sl * DEPP_PART + r] = r < R ? node(r, sl) : 0.f;
    __syncthreads();
    for (int q = tid; q < R; q += DEPP_THREADS) {
        float a = 0.f;
        for (int k = 0; k < SL; ++k) a += part[k * DEPP_PART + q];
        flush(q, a);
    }
}

// the register forms: 1, 2 one width with P <= 8 or 16, 3, 4 a narrow range of widths with P <= 6 or 8;
// 5 the matrix product, 0 degrees beyond it (its moment tiles have to fit a warp)
__device__ __forceinline__ int depp_form(const PxyBox &B)
{
    if (B.P > PXY_MAXP || B.Q > PXY_MAXQ || ((B.P + 3) >> 2) * ((B.Q + 3) >> 2) > 32) return 0;
    if (B.Q == 1) return B.P <= 8 ? 1 : 2;
    return B.lin && B.P <= 8 ? (B.P <= 6 ? 3 : 4) : 5;
}

// Costs of the forms in ns of an SM, per CTA, fitted to 867 launches with either form forced (40,000 to
// 4,000,037 particles, 64 to 4096 nodes, uniform widths and ranges from 0.5 to 20,000; 5 to 9% off).
// What a launch waits for once (barriers, table loads, the chain of small steps), /share of it a
// CTA, is beyond the sweep's.  Deposits of a PIC step, swept and compressed: widths of 7 to 20 on 256
// nodes, 65,536 particles 12.9 and 18.3 us, 2^20 48.7 and 44.7, on 1024 nodes 20.5 and 24.2, 152 and
// 51 (form 5); widths near 315, 1024 nodes, 131,072 particles 12.2 and 12.5, 4,000,037 121 and 35
// (form 4); width 5000 on 256 nodes, 2^20 particles 14.2 and 16.3 (form 2); width 14 on 512 nodes,
// 524,288 particles 37.9 and 11.2 (form 1)
__host__ __device__ inline float depp_sweep_ns(float n, float R, bool cosf, float inv_share)
{
    return n * fmaf(cosf ? 0.0196f : 0.0229f, R, 0.82f) + 4.5f * R * inv_share;
}
// cost c.x n + c.y R + (c.z + c.w R) / share of the register forms
__host__ __device__ inline float4 depp_reg_cost(int form)
{
    return form == 1 ? make_float4(0.47f, 0.7f, 180.f, 0.8f)
                     : (form == 2 ? make_float4(0.53f, 2.0f, 500.f, 0.f)
                                  : (form == 3 ? make_float4(0.61f, 1.03f, 1450.f, 1.45f) : make_float4(0.89f, 2.1f, 2300.f, 0.f)));
}
__device__ __forceinline__ bool depp_compress_pays(const PxyBox &B, int form, int n, int R, bool cosf, float inv_share)
{
    // nodes as the sweep's warps take them
    const int Rs = R > 128 ? (R + 63) & ~63 : (R > 64 ? 128 : (R > 32 ? 64 : (R > 16 ? 32 : (R > 8 ? 16 : 8))));
    const float direct = depp_sweep_ns((float)n, (float)Rs, cosf, inv_share);
    float4 c = depp_reg_cost(form);
    if (form == 5) {
        const float P = (float)B.P, Q = (float)B.Q;
        const int LP = (B.P + 3) >> 2, LQ = (B.Q + 3) >> 2, tiles = LP * LQ;
        const float iKS = tiles > 16 ? 1.f : (tiles > 8 ? 0.5f : (tiles > 4 ? 0.25f : 0.125f));  // 1 / particles taken at once
        c = make_float4(2.9f + 4.4f * iKS + 0.04f * (float)max(LP, LQ), P * (0.615f + 0.0022f * Q),
                        4150.f + 0.53f * P * Q * (P + Q), 0.f);
    }
    return form && (float)n * c.x + (float)R * c.y + fmaf(c.w, (float)R, c.z) * inv_share < direct;
}

// COMP: with the compressed form, chosen per CTA; without it where no CTA would take it
template <bool COMP>
__global__ void __launch_bounds__(DEPP_THREADS, DEPP_MINB) deposit_persist_kernel(DepSrc<float> S, DepPlan Pl)
{
    __shared__ float4 rec[DEPP_SUB];
    __shared__ __align__(16) float part[DEPP_WARPS * DEPP_PART];  // also read as float2 and float4
    __shared__ float sred[2 * DEPP_WARPS];
    __shared__ int s_es;
    constexpr int PER = DEPP_SUB / DEPP_THREADS;  // particles of a sub-chunk per thread
    const int Ng = S.Ng;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = blockIdx.x;
    const int64_t i0 = S.N * c / Pl.G, i1 = S.N * (c + 1) / Pl.G;  // non-empty: G <= N
    kde_pdl_wait();  // everything read below comes from the sort before
    kde_pdl_trigger();

    // smallest and largest width of the CTA's particles (the window and the form): the range of all
    // where it is known and narrow, else a pass over the CTA's widths, PER loads in flight per
    // thread -- a few wide kernels among narrow ones, or widths that follow the density, would
    // otherwise give every CTA the widest one's window (one width in 1e5 5 and the others 2000, a run
    // of 10 steps: 2^18 particles on 256 nodes 445 us with the range of all, 397 with the CTAs',
    // 2^20 on 1024 nodes 1587 and 1297)
    float kmin = (float)KDE_KAPPA_MAX, kmax = 0.f;
    bool shared_range = false;
    if (S.krange) {
        const float hi = __uint_as_float(S.krange[0]), lo = __uint_as_float(S.krange[1]);
        shared_range = pxy_narrow(lo, hi);
        if (shared_range) {
            kmax = hi;
            kmin = lo;
        }
    }
    if (!S.kappa) {
        kmin = kmax = S.kappa_u;
    } else if (!shared_range) {
        for (int64_t j0 = i0; j0 < i1; j0 += (int64_t)PER * DEPP_THREADS) {
            float kk[PER];
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                const int64_t j = j0 + tid + p * DEPP_THREADS;
                kk[p] = S.kappa[j < i1 ? j : i0];
            }
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                const float k = (kk[p] > 0.f && kk[p] <= (float)KDE_KAPPA_MAX) ? kk[p] : (float)KDE_KAPPA_MAX;
                kmin = fminf(kmin, k);
                kmax = fmaxf(kmax, k);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        kmin = fminf(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
        kmax = fmaxf(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
    }
    if (lane == 0) {
        sred[warp] = kmin;
        sred[DEPP_WARPS + warp] = kmax;
    }
    if (tid == 0) {
        int es = S.scale_exp;
        if (es == KDE_ES_FROM_BOUND) {
            double bound = S.bound;
            if (S.wmax_bits)
                bound = (double)S.N * (double)S.coef * S.norm_bound * (double)__uint_as_float(*S.wmax_bits);
            es = acc_scale_exp(bound);
        }
        s_es = es;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < DEPP_WARPS; ++k) {
        kmin = fminf(kmin, sred[k]);
        kmax = fmaxf(kmax, sred[DEPP_WARPS + k]);
    }
    const int es = s_es;
    const bool cosf = kmax <= KDE_COSFORM_KMAX;
    const int W = window_nodes_f(kmin, Ng, S.xcut);
    // the CTA's cells: those of its first and last sort bin (unsorted particles: all)
    int c_first = 0, c_last = Ng - 1;
    if (S.nbins == 0) {
        c_first = kde_cell(S.u[i0], Ng);
        c_last = kde_cell(S.u[i1 - 1], Ng);
    } else if (S.nbins > 0) {
        c_first = kde_cell(S.u[i0], S.nbins) * Ng / S.nbins;
        c_last = ((kde_cell(S.u[i1 - 1], S.nbins) + 1) * Ng - 1) / S.nbins;
    }
    int g_lo = c_first - W;
    int R = c_last + W - g_lo + 1;
    if (R >= Ng || R < 1 || c_last < c_first) {
        g_lo = 0;
        R = Ng;
    }
    // windows of up to 128 nodes: records in particle pairs (depp_sweep_pairs); wider ones:
    // 4, 2 or 1 node pairs a lane, the widest that computes no extra nodes and whose slice
    // sums fit the buffer
    const bool pairs = R <= 128;
    float4 *recAB = rec;
    float2 *recW = (float2 *)(rec + DEPP_SUB / 2);
    const int n64 = (R + 63) >> 6, n128 = (R + 127) >> 7, n256 = (R + 255) >> 8;
    const int P = (4 * n256 == n64 && (n256 >= DEPP_WARPS || n256 * 256 <= DEPP_PART))   ? 4
                  : (2 * n128 == n64 && (n128 >= DEPP_WARPS || n128 * 128 <= DEPP_PART)) ? 2
                                                                                          : 1;
    // node sums of a sub-chunk into the grid's int64 sums: reductions without a return value,
    // exact, so the result does not depend on their order
    auto flush = [&](int r, float a) {
        int g = g_lo + r;
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        // x 2^es in integer arithmetic; the FP64 product only for extreme bounds
        const long long v = (es >= -100 && es <= 100) ? fix_pow2(a, es) : __double2ll_rn(ldexp((double)a, es));
        if (v) atomicAdd((unsigned long long *)&Pl.acc[g], (unsigned long long)v);
    };
    if constexpr (COMP) {
    if (c_last >= c_first) {
        // the default cut: compressed where that is less work (a cut the caller has set keeps
        // the sweep over the particles that it is defined for)
        PxyBox B;
        pxy_box_pos(B, S.grid, c_first, c_last, kmax);
        pxy_box_width(B, kmin, kmax);
        const int n = (int)(i1 - i0);
        const int form = depp_form(B);
        if (depp_compress_pays(B, form, n, R, cosf, Pl.inv_share)) {
            __shared__ float M[PXY_MAXP * PXY_MAXQ];
            // the register forms' interpolation matrices, beside the records' space
            float *tabs = (float *)rec, *mem = tabs + PXY_MAXP * PXY_MAXP + 64;
            auto load_tabs = [&](int P, int Q) {
                const float *cp = S.pxt + pxy_tab_off(P), *cq = S.pxt + pxy_tab_off(Q);
                for (int i = tid; i < P * P; i += DEPP_THREADS) tabs[i] = cp[i];
                if (tid < Q * Q) tabs[P * P + tid] = cq[tid];
            };
            if (form == 1) {
                load_tabs(8, 1);
                depp_moments_reg<8, 1, false>(S, i0, n, B, part, M);
                depp_proxies_reg<8, 1>(S, B, g_lo, R, M, tabs, shared_range, mem, part, flush);
            } else if (form == 2) {
                load_tabs(16, 1);
                depp_moments_reg<16, 1, false>(S, i0, n, B, part, M);
                depp_proxies_reg<16, 1>(S, B, g_lo, R, M, tabs, shared_range, mem, part, flush);
            } else if (form == 3) {
                load_tabs(7, 7);
                depp_moments_reg<7, 7, true>(S, i0, n, B, part, M);
                depp_proxies_reg<7, 7>(S, B, g_lo, R, M, tabs, shared_range, mem, part, flush);
            } else if (form == 4) {
                load_tabs(8, 6);
                depp_moments_reg<8, 6, false>(S, i0, n, B, part, M);
                depp_proxies_reg<8, 6>(S, B, g_lo, R, M, tabs, shared_range, mem, part, flush);
            } else {
                depp_moments_mm(S, i0, n, B, (float *)rec, part, M);
                depp_proxies(S, B, g_lo, R, M, (float *)rec, part, flush);
            }
            return;
        }
    }
    }

    for (int64_t b0 = i0; b0 < i1; b0 += DEPP_SUB) {
        const int n = (int)(i1 - b0 < DEPP_SUB ? i1 - b0 : DEPP_SUB);
        const bool first = b0 == i0;
        if (!first) __syncthreads();  // the previous sub-chunk's readers of rec and part are done
        // the particle records (a, b, w n) of the form in use, in groups of four particles a
        // thread whose inputs are loaded together (one global-load latency per group)
        constexpr int QB = 4;
#pragma unroll 1
        for (int p0 = 0; p0 < PER; p0 += QB) {
            uint32_t ru[QB];
            float rk[QB], rw[QB];
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                const int t = tid + (p0 + q) * DEPP_THREADS;
                const int64_t j = b0 + (t < n ? t : 0);
                ru[q] = S.u[j];
                rk[q] = S.kappa ? S.kappa[j] : S.kappa_u;
                rw[q] = S.w ? S.w[j] : S.w_u;
            }
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                const int t = tid + (p0 + q) * DEPP_THREADS;
                if (t >= n) break;
                float k = rk[q];
                if (!(k > 0.f && k <= (float)KDE_KAPPA_MAX)) {
                    kde_flag(S.status, KDE_DEV_KAPPA_RANGE, (unsigned)(b0 + t));
                    k = (float)KDE_KAPPA_MAX;
                }
                const float nm = S.kappa ? kde_norm_tab(S.ntab, k) : S.norm_u;
                const float wn = rw[q] * S.coef * nm;
                float sh, ch;
                kde_half_sincos(ru[q], sh, ch);
                float ra, rb, rw2;
                if (cosf) {
                    const float K = (float)KDE_LOG2E * k;
                    ra = K * ((ch - sh) * (ch + sh));
                    rb = K * (2.f * sh * ch);
                    rw2 = wn * kde_ex2(-K);
                } else {
                    const float beta = sqrtf((float)(2.0 * KDE_LOG2E) * k);
                    ra = beta * sh;
                    rb = beta * ch;
                    rw2 = wn;
                }
                if (pairs) {
                    float *ab = (float *)recAB + (t >> 1) * 4 + (t & 1);
                    ab[0] = ra;
                    ab[2] = rb;
                    ((float *)recW)[t] = rw2;
                } else {
                    rec[t] = make_float4(ra, rb, rw2, 0.f);
                }
            }
        }
        if (pairs && (n & 1) && tid == 0) {
            // the odd particle's partner: no weight (a finite exponent times zero)
            float *ab = (float *)recAB + (n >> 1) * 4 + 1;
            ab[0] = 0.f;
            ab[2] = 0.f;
            ((float *)recW)[n] = 0.f;
        }
        __syncthreads();
        if (pairs) {
            if (R <= 8) depp_sweep_pairs<8, 1>(S, n, g_lo, R, cosf, recAB, recW, part, flush);
            else if (R <= 16) depp_sweep_pairs<16, 1>(S, n, g_lo, R, cosf, recAB, recW, part, flush);
            else if (R <= 32) depp_sweep_pairs<32, 1>(S, n, g_lo, R, cosf, recAB, recW, part, flush);
            else if (R <= 64) depp_sweep_pairs<32, 2>(S, n, g_lo, R, cosf, recAB, recW, part, flush);
            else depp_sweep_pairs<32, 4>(S, n, g_lo, R, cosf, recAB, recW, part, flush);
        } else if (P == 4) depp_sweep<4>(S, n, g_lo, R, cosf, rec, part, flush);
        else if (P == 2) depp_sweep<2>(S, n, g_lo, R, cosf, rec, part, flush);
        else depp_sweep<1>(S, n, g_lo, R, cosf, rec, part, flush);
    }
}

// acc -> real values
template <typename T>
__global__ void acc_to_real_kernel(const long long *acc, int Ng, double bound, const unsigned int *wmax_bits,
                                   double wscale, T *out, const long long *lo)
{
    int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= Ng) return;
    double b = wmax_bits ? wscale * (double)__uint_as_float(*wmax_bits) : bound;
    const double a = lo ? (double)acc[g] + (double)lo[g] * (1.0 / 16777216.0) : (double)acc[g];
    out[g] = (T)(a / kde_acc_scale(b));
}

// largest weight (non-negative floats order like their bit patterns)
template <typename T>
__global__ void wmax_kernel(const T *w, int64_t N, unsigned int *wmax_bits, unsigned int *status)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float m = 0.f;
    for (; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        float v = (float)w[i];
        if (!(v >= 0.f) || isinf(v)) kde_flag(status, KDE_DEV_BAD_ARG, (unsigned)i);
        else m = fmaxf(m, v);
    }
    __shared__ unsigned int red[8];
    const unsigned int h = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = h;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int b = red[0];
        for (int w = 1; w < 8; ++w) b = b > red[w] ? b : red[w];
        // the maximum rounded up by one ulp so that the float bound of a double weight still
        // bounds it; most blocks find a larger one already
        if (b > 0u && b + 1u > *(volatile unsigned int *)wmax_bits) atomicMax(wmax_bits, b + 1u);
    }
}

// ---------------------------------------------------------------------------
kde_status kde_krange_begin(kde_ctx *ctx, unsigned int *krange)
{
    // reset by the pass before, unless that failed half-way; a captured pass, whose replays may come
    // after such a one, resets them itself
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(ctx->stream, &cap);
    if (!ctx->range_reset || cap != cudaStreamCaptureStatusNone) {
        KDE_CUDA(ctx, kde_krange_reset(krange + KDE_KRANGE_ACC, ctx->stream), "width range memset");
        KDE_CUDA(ctx, cudaMemsetAsync(krange + KDE_KRANGE_ACC + 2, 0, 4, ctx->stream), "width range memset");
    }
    ctx->range_reset = false;
    return KDE_OK;
}

void kde_krange_end(kde_ctx *ctx)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(ctx->stream, &cap);
    ctx->range_reset = cap == cudaStreamCaptureStatusNone;
}

// grids of int64 node sums: two for the PIC step's deposits (see DepSums), and one for
// kde_deposit, which every call leaves zero
static long long *depp_sums(kde_ctx *ctx)
{
    if (ctx->ws_bytes[WS_DEP_SUMS] == 0) {
        ctx->sums_zero = false;
        ctx->sums_ng = 0;
    }
    return (long long *)kde_ws(ctx, WS_DEP_SUMS, (size_t)3 * KDE_MAX_NG * 8);
}

// out = sums 2^-es, and the sums back to zero
__global__ void __launch_bounds__(256) sums_to_real_kernel(long long *acc, int Ng, double bound, const unsigned int *wmax_bits,
                                                           double wscale, float *out)
{
    const int g = blockIdx.x * 256 + threadIdx.x;
    kde_pdl_wait();
    kde_pdl_trigger();
    if (g >= Ng) return;
    const double b = wmax_bits ? wscale * (double)__uint_as_float(*wmax_bits) : bound;
    const long long a = __ldcg(&acc[g]);
    acc[g] = 0;
    out[g] = (float)((double)a / kde_acc_scale(b));
}

kde_status kde_deposit_reserve(kde_ctx *ctx) { return depp_sums(ctx) ? KDE_OK : KDE_ENOMEM; }

kde_status kde_deposit_sums_reset(kde_ctx *ctx, int Ng)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(ctx->stream, &cap);
    if (cap != cudaStreamCaptureStatusNone) ctx->sums_captured = true;
    long long *s = depp_sums(ctx);
    if (!s) return KDE_ENOMEM;
    // the grid whose turn it is was zeroed by the last field kernel, if that had as many nodes and
    // every deposit its field kernel.  Replays of a captured call use the grids in the turn they had
    // then: a context with one zeroes them always
    if (ctx->sums_ng == Ng && !ctx->sums_captured) return KDE_OK;
    ctx->sums_ng = 0;
    ctx->sums_flip = false;
    KDE_CUDA(ctx, cudaMemsetAsync(s, 0, (size_t)2 * KDE_MAX_NG * 8, ctx->stream), "node sums memset");
    return KDE_OK;
}

template <typename T>
static kde_status deposit_sorted_impl(kde_ctx *ctx, const uint32_t *u, const T *kappa, T kappa_u, const T *norm,
                                      T norm_u, const T *w, T w_u, int64_t N, int Ng, double coef, long long *acc,
                                      double bound, const unsigned int *wmax_bits, double norm_bound,
                                      float xcut = 0.f, const unsigned int *krange = nullptr, int nbins = 0, bool sweep = false)
{
    // (the FP32 callers zero their sums)
    if (sizeof(T) == 8)
        KDE_CUDA(ctx, cudaMemsetAsync(acc, 0, (size_t)2 * Ng * sizeof(long long), ctx->stream), "acc memset");
    if (N == 0) return KDE_OK;
    const void *nodes = kde_node_table(ctx, Ng, sizeof(T) == 8);
    if (!nodes) return KDE_ENOMEM;
    DepSrc<T> S{};
    S.u = u;
    S.N = N;
    S.kappa = kappa;
    S.kappa_u = kappa_u;
    S.kscale = (T)1;
    S.norm = norm;
    S.lnorm = nullptr;
    S.norm_u = norm_u;
    S.w = w;
    S.w_u = w_u;
    S.coef = (T)coef;
    S.Ng = Ng;
    S.nodes = (const typename V2<T>::t *)nodes;
    S.acc = acc;
    S.bound = bound;
    S.wmax_bits = wmax_bits;
    S.norm_bound = norm_bound;
    S.status = ctx->d_status;
    S.scale_exp = KDE_ES_FROM_BOUND;
    if (!wmax_bits) {
        // the scale exponent from the host-known bound, as acc_scale_exp computes it
        int e;
        frexp(bound > 0 ? bound : 1.0, &e);
        S.scale_exp = 62 - e;
    }
    S.ntab = ctx->norm_tab;
    S.xcut = xcut > 0.f ? xcut : kde_fp32_cut(ctx);
    S.grid = pxy_grid(Ng);
    S.pxt = ctx->pxy_tab;
    S.krange = krange;
    S.nbins = nbins;
    if constexpr (sizeof(T) == 4) {
        DepPlan Pl{};
        // unsorted particles sweep the whole grid: shorter shares, so that small calls reach more SMs
        const int64_t gmax = (int64_t)DEPP_MINB * ctx->sm_count;
        const int64_t gn = nbins < 0 ? (N + 63) / 64 : (N + 255) / 256;
        Pl.G = (int)(gn < gmax ? gn : gmax);
        Pl.acc = acc;
        const float share = std::max(1.f, std::min((float)DEPP_MINB, (float)Pl.G / (float)(ctx->sm_count > 0 ? ctx->sm_count : 1)));
        Pl.inv_share = 1.f / share;
        {
            KdeProfScope _ps(ctx, PROF_DEPOSIT);
            // the compressed form is for the default cut (one the caller has set keeps the sweep
            // over the particles that it is defined for), and where the best that can be expected of
            // it spares 0.3 us (the kernel that chooses takes up to 2 us longer when it then sweeps:
            // particle-wise widths, 2^20 particles on 64 nodes 26.7 against 24.8 us).  One width has a form
            // by the positions of an average CTA; particle-wise widths form 3 at best, with P <= 6 on
            // fewer than 80 nodes only for widths below 15.
            const float n = (float)((double)N / Pl.G);
            int form = Ng < 80 ? 0 : 3;
            double Rw = Ng;
            if (!kappa) {
                const double cells = std::min((double)Ng, (double)Ng / Pl.G + 1.0);
                const double y = KDE_PI * cells / Ng * sqrt((double)kappa_u + 1.5);
                form = y <= 0.388 ? 1 : (y <= 1.65 ? 2 : 0);
                Rw = std::min(Rw, 2.0 * kde_window_nodes((double)kappa_u, Ng) + cells);
            }
            const float4 c = depp_reg_cost(form);
            const float gain = depp_sweep_ns(n, (float)Rw, true, Pl.inv_share) - n * c.x - (float)Rw * c.y -
                               (c.z + c.w * (float)Rw) * Pl.inv_share;
            const bool comp = nbins >= 0 && !sweep && S.xcut == (float)KDE_XCUT && form && gain * share > 300.f;
            KDE_CUDA(ctx,
                     kde_launch(ctx, true, comp ? deposit_persist_kernel<true> : deposit_persist_kernel<false>,
                                dim3(Pl.G), dim3(DEPP_THREADS), 0, S, Pl),
                     "deposit_persist_kernel");
        }
        KDE_LAUNCHED(ctx, "deposit_persist_kernel");
    } else {
        // four chunks an SM where that leaves them 16 particles or more, 256 at most
        const int64_t per = N / (4LL * (ctx->sm_count > 0 ? ctx->sm_count : 1)) + 1;
        const int chunk = (int)(per < 16 ? 16 : (per > DEP64_MAXCHUNK ? DEP64_MAXCHUNK : per));
        {
            KdeProfScope _ps(ctx, PROF_DEPOSIT);
            deposit64_kernel<<<(unsigned)((N + chunk - 1) / chunk), DEP_THREADS, 0, ctx->stream>>>(S, chunk, ctx->f64_tab);
        }
        KDE_LAUNCHED(ctx, "deposit64_kernel");
    }
    return KDE_OK;
}

kde_status kde_deposit_sorted_f64(kde_ctx *ctx, const uint32_t *u, const double *kappa, double kappa_u,
                                  const double *norm, double norm_u, const double *w, double w_u, int64_t N, int Ng,
                                  double coef, long long *acc, double bound, const unsigned int *wmax_bits,
                                  double norm_bound)
{
    return deposit_sorted_impl<double>(ctx, u, kappa, kappa_u, norm, norm_u, w, w_u, N, Ng, coef, acc, bound, wmax_bits,
                                       norm_bound);
}

kde_status kde_deposit_sums_f32(kde_ctx *ctx, const uint32_t *u, const float *kappa, float kappa_u, float norm_u,
                                int64_t N, int Ng, double coef, float w_u, double bound, DepSums *out,
                                float xcut, const unsigned int *krange)
{
    if (N < 1) return kde_fail(ctx, KDE_EINVAL, "deposit sums: need N >= 1");
    long long *s = depp_sums(ctx);
    if (!s) return KDE_ENOMEM;
    out->acc = s + (ctx->sums_flip ? KDE_MAX_NG : 0);
    out->next = s + (ctx->sums_flip ? 0 : KDE_MAX_NG);
    ctx->sums_flip = !ctx->sums_flip;
    ctx->sums_ng = 0;  // known again after the field kernel
    return deposit_sorted_impl<float>(ctx, u, kappa, kappa_u, nullptr, norm_u, nullptr, w_u, N, Ng, coef, out->acc, bound,
                                      nullptr, 0.0, xcut, krange, 0, kappa && !krange);
}

template <typename T>
kde_status kde_acc_to_real(kde_ctx *ctx, const long long *acc, int Ng, double bound, const unsigned int *wmax_bits,
                           double wscale, T *out)
{
    acc_to_real_kernel<T><<<(Ng + 255) / 256, 256, 0, ctx->stream>>>(acc, Ng, bound, wmax_bits, wscale, out,
                                                                     sizeof(T) == 8 ? acc + Ng : nullptr);
    KDE_LAUNCHED(ctx, "acc_to_real_kernel");
    return KDE_OK;
}

template kde_status kde_acc_to_real<float>(kde_ctx *, const long long *, int, double, const unsigned int *, double,
                                           float *);
template kde_status kde_acc_to_real<double>(kde_ctx *, const long long *, int, double, const unsigned int *, double,
                                            double *);

// ---------------------------------------------------------------------------
// CV integral term: the deposit of every candidate on its own power-of-two
// grid of M_c points (theta units, w = 1/N), one grid per blockIdx.y.
// ---------------------------------------------------------------------------
__host__ __device__ inline int cv_grid_points(double kappa_max)
{
    // the trapezoid rule on M points integrates fhat^2 exactly up to aliased
    // modes near M/2, whose weight A_{M/2}^2 ~ exp(-(M/2)^2 / kappa) is below
    // 1e-17 once M >= 12.5 sqrt(kappa)
    double need = 12.5 * sqrt(kappa_max) + 1.0;
    int M = 64;
    while (M < need && M < CV_MAXM) M <<= 1;
    return M;
}

// per-candidate parameters of the grid deposit
struct GridPar {
    float k;       // the candidate: uniform width, or the scale of the relative widths
    float norm_u;  // uniform norm (uniform widths)
    int M;         // grid points
    int es;        // fixed-point scale 2^es of the grid sums
    float w_u;     // the weight 1/N
};

// one thread per candidate: the FP64 Bessel norm of the largest width, the grid size and
// the fixed-point scale, worked out once instead of in every thread of the deposit
__global__ void cv_grid_par_kernel(CandList cl, const unsigned int *krmax_bits, int64_t N, GridPar *par)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cl.n) return;
    const double kmax = cl.scale_mode ? cl.k[c] * (double)__uint_as_float(*krmax_bits) : cl.k[c];
    const double nb = kde_norm(kmax);  // bound of a node value: N * (1/N) * the largest norm
    GridPar p;
    p.k = (float)cl.k[c];
    p.norm_u = (float)nb;
    p.M = cv_grid_points(kmax);
    p.es = acc_scale_exp(nb);
    p.w_u = (float)(1.0 / (double)N);
    par[c] = p;
}

// four CTAs an SM (62 registers): left to itself the compiler goes for five at 48 registers, with fewer
// records in flight (20,000 particles, 3 factors on widths of 1e-5 to 1e5: 291 us, 234 with four)
__global__ void __launch_bounds__(DEP_THREADS, 4)
    cv_grid_deposit_kernel(const uint32_t *u, int64_t N, const float *kappa_rel, const float *lnorm, int scale_mode,
                           const GridPar *par, long long *acc, unsigned int *status)
{
    __shared__ float4 rsc[DEP_CHUNK];
    __shared__ float2 rwn[DEP_CHUNK];
    __shared__ float part[DEP_WARPS * DEP2_PART];
    __shared__ int red[2 * DEP_WARPS];
    const int c = blockIdx.y;
    const GridPar p = par[c];
    DepSrc<float> S{};
    S.u = u;
    S.N = N;
    S.coef = 1.0f;
    S.w = nullptr;
    S.w_u = p.w_u;
    S.nodes = nullptr;
    S.acc = acc + (size_t)c * CV_MAXM;
    S.status = status;
    S.wmax_bits = nullptr;
    S.norm = nullptr;
    if (scale_mode) {
        S.kappa = kappa_rel;
        S.kscale = p.k;
        S.lnorm = lnorm + (size_t)c * N;
    } else {
        S.kappa = nullptr;
        S.kappa_u = p.k;
        S.kscale = 1.0f;
        S.lnorm = nullptr;
        S.norm_u = p.norm_u;
    }
    S.scale_exp = p.es;
    S.Ng = p.M;
    // the CV integral term keeps the half-angle form: its sums carry the CV's accuracy
    deposit_chunk_body_x2(S, blockIdx.x, rsc, rwn, part, red);
}

// FP64 trapezoid sum of fhat^2 on each candidate's grid: f2[c] = (2 pi / M) sum_g fhat_g^2
__global__ void cv_grid_square_kernel(const long long *acc, const GridPar *par, double *f2)
{
    const int c = blockIdx.x;
    const int M = par[c].M;
    const double inv = __longlong_as_double((long long)(1023 - par[c].es) << 52);  // 2^-es
    __shared__ double red[256];
    double s = 0.0;
    for (int g = threadIdx.x; g < M; g += blockDim.x) {
        double f = (double)acc[(size_t)c * CV_MAXM + g] * inv;
        s += f * f;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) f2[c] = KDE_TWO_PI / M * red[0];
}

kde_status kde_cv_integral_term(kde_ctx *ctx, const uint32_t *u_sorted, int64_t N, const float *kappa_rel,
                                const float *lnorm, const unsigned int *krmax_bits, const CandList &cl,
                                double *f2_out)
{
    long long *acc = (long long *)kde_ws(ctx, WS_CV_ACC, (size_t)cl.n * CV_MAXM * sizeof(long long));
    if (!acc) return KDE_ENOMEM;
    KDE_CUDA(ctx, cudaMemsetAsync(acc, 0, (size_t)cl.n * CV_MAXM * sizeof(long long), ctx->stream), "cv acc memset");
    GridPar *par = (GridPar *)kde_ws(ctx, WS_CV_GPAR, (size_t)cl.n * sizeof(GridPar));
    if (!par) return KDE_ENOMEM;
    cv_grid_par_kernel<<<(cl.n + 63) / 64, 64, 0, ctx->stream>>>(cl, krmax_bits, N, par);
    KDE_LAUNCHED(ctx, "cv_grid_par_kernel");
    dim3 grid((unsigned)((N + DEP_CHUNK - 1) / DEP_CHUNK), (unsigned)cl.n);
    {
        KdeProfScope _ps(ctx, PROF_CV_GRID);
        cv_grid_deposit_kernel<<<grid, DEP_THREADS, 0, ctx->stream>>>(u_sorted, N, kappa_rel, lnorm, cl.scale_mode,
                                                                        par, acc, ctx->d_status);
    }
    KDE_LAUNCHED(ctx, "cv_grid_deposit_kernel");
    cv_grid_square_kernel<<<cl.n, 256, 0, ctx->stream>>>(acc, par, f2_out);
    KDE_LAUNCHED(ctx, "cv_grid_square_kernel");
    return KDE_OK;
}

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
// largest weight into the workspace's word (float bits), or nullptr without weights
template <typename T>
static kde_status deposit_wmax(kde_ctx *ctx, const T *weight, int64_t N, unsigned int **out)
{
    *out = nullptr;
    if (!weight) return KDE_OK;
    unsigned int *wmax = (unsigned int *)kde_ws(ctx, WS_WMAX, 64);
    if (!wmax) return KDE_ENOMEM;
    KDE_CUDA(ctx, cudaMemsetAsync(wmax, 0, 4, ctx->stream), "wmax memset");
    int blocks = (int)((N + 255) / 256);
    blocks = blocks > ctx->sm_count * 4 ? ctx->sm_count * 4 : blocks;
    wmax_kernel<T><<<blocks, 256, 0, ctx->stream>>>(weight, N, wmax, ctx->d_status);
    KDE_LAUNCHED(ctx, "wmax_kernel");
    *out = wmax;
    return KDE_OK;
}

static kde_status deposit_api_f64(kde_ctx *ctx, const uint32_t *u, const double *kappa, double kappa_u,
                                  const double *weight, int64_t N, int Ng, double L, double *rho_out)
{
    cudaSetDevice(ctx->device);
    long long *acc = (long long *)kde_ws(ctx, WS_ACC, (size_t)2 * Ng * sizeof(long long));
    if (!acc) return KDE_ENOMEM;
    if (N == 0) {
        KDE_CUDA(ctx, cudaMemsetAsync(rho_out, 0, (size_t)Ng * 8, ctx->stream), "rho memset");
        return KDE_OK;
    }
    uint32_t *us = (uint32_t *)kde_ws(ctx, WS_SORT_U, (size_t)N * 4);
    double *ks = kappa ? (double *)kde_ws(ctx, WS_SORT_P0, (size_t)N * 8) : nullptr;
    double *ws = weight ? (double *)kde_ws(ctx, WS_SORT_P1, (size_t)N * 8) : nullptr;
    if (!us || (kappa && !ks) || (weight && !ws)) return KDE_ENOMEM;
    SortPayload pl[2];
    int npl = 0;
    if (kappa) pl[npl++] = SortPayload{kappa, ks, 8};
    if (weight) pl[npl++] = SortPayload{weight, ws, 8};
    KDE_TRY(kde_sort_by_bin(ctx, u, N, Ng, us, pl, npl, nullptr));
    const double coef = KDE_TWO_PI / L;
    const double norm_u = kappa ? 0.0 : kde_norm(kappa_u);
    const double norm_bound = kappa ? kde_norm(KDE_KAPPA_MAX) : norm_u;
    const double w_u = L / (double)N;
    const double bound = (double)N * w_u * coef * norm_bound;
    unsigned int *wmax = nullptr;
    KDE_TRY(deposit_wmax<double>(ctx, weight, N, &wmax));
    KDE_TRY(kde_deposit_sorted_f64(ctx, us, ks, kappa_u, nullptr, norm_u, ws, w_u, N, Ng, coef, acc, bound, wmax, norm_bound));
    return kde_acc_to_real<double>(ctx, acc, Ng, bound, wmax, (double)N * coef * norm_bound, rho_out);
}

static kde_status deposit_api_f32(kde_ctx *ctx, const uint32_t *u, const float *kappa, double kappa_u,
                                  const float *weight, int64_t N, int Ng, double L, float *rho_out)
{
    cudaSetDevice(ctx->device);
    if (N == 0) {
        KDE_CUDA(ctx, cudaMemsetAsync(rho_out, 0, (size_t)Ng * 4, ctx->stream), "rho memset");
        return KDE_OK;
    }
    // few (particle, node) pairs: the particles as they are over the whole grid, at the default
    // truncation (a cut the caller has set keeps its windows).  2^25 pairs take about 8 us, the
    // sort they spare 16 to 20
    const bool flat = (double)N * Ng <= 33554432.0 && kde_fp32_cut(ctx) == (float)KDE_XCUT;
    // the sort groups the particles for the CTAs' windows, which have at most a few hundred
    // CTAs' worth of resolution: 1024 bins at most.  4,000,037 particles with widths of 5 to 5000
    // on 4096 nodes: 470 us; 528 with 2048 bins and 540 sorted by cells (the count table and the
    // scatter's short runs), 1712 with 512 (a bin is then too wide for proxies at the largest widths)
    const int nbins = flat ? -1 : (Ng > 1024 ? 1024 : Ng);
    const uint32_t *us = u;
    const float *ks = kappa, *ws = weight;
    if (!flat) {
        uint32_t *uo = (uint32_t *)kde_ws(ctx, WS_SORT_U, (size_t)N * 4);
        float *ko = kappa ? (float *)kde_ws(ctx, WS_SORT_P0, (size_t)N * 4) : nullptr;
        float *wo = weight ? (float *)kde_ws(ctx, WS_SORT_P1, (size_t)N * 4) : nullptr;
        if (!uo || (kappa && !ko) || (weight && !wo)) return KDE_ENOMEM;
        SortPayload pl[2];
        int npl = 0;
        if (kappa) pl[npl++] = SortPayload{kappa, ko, 4};
        if (weight) pl[npl++] = SortPayload{weight, wo, 4};
        KDE_TRY(kde_sort_by_bin(ctx, u, N, nbins, uo, pl, npl, nullptr));
        us = uo;
        ks = ko;
        ws = wo;
    }
    const double coef = KDE_TWO_PI / L;
    const double norm_u = kappa ? 0.0 : kde_norm(kappa_u);
    const double norm_bound = kappa ? kde_norm(KDE_KAPPA_MAX) : norm_u;
    const double w_u = L / (double)N;
    const double bound = (double)N * w_u * coef * norm_bound;
    unsigned int *wmax = nullptr;
    KDE_TRY(deposit_wmax<float>(ctx, weight, N, &wmax));
    // the sums are zero from the call before, unless it failed half-way; a captured call, whose
    // replays may come after such a one, zeroes them itself
    long long *acc = depp_sums(ctx);
    if (!acc) return KDE_ENOMEM;
    acc += 2 * KDE_MAX_NG;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(ctx->stream, &cap);
    if (!ctx->sums_zero || cap != cudaStreamCaptureStatusNone)
        KDE_CUDA(ctx, cudaMemsetAsync(acc, 0, (size_t)KDE_MAX_NG * 8, ctx->stream), "node sums memset");
    ctx->sums_zero = false;
    KDE_TRY(deposit_sorted_impl<float>(ctx, us, ks, (float)kappa_u, nullptr, (float)norm_u, ws, (float)w_u, N, Ng, coef,
                                       acc, bound, wmax, norm_bound, 0.f, nullptr, nbins == Ng ? 0 : nbins));
    KDE_CUDA(ctx,
             kde_launch(ctx, true, sums_to_real_kernel, dim3((Ng + 255) / 256), dim3(256), 0, acc, Ng, bound,
                        (const unsigned int *)wmax, (double)N * coef * norm_bound, rho_out),
             "sums_to_real_kernel");
    KDE_LAUNCHED(ctx, "sums_to_real_kernel");
    ctx->sums_zero = cap == cudaStreamCaptureStatusNone;
    return KDE_OK;
}

extern "C" kde_status kde_deposit(kde_ctx *ctx, const uint32_t *u, const void *kappa, double kappa_uniform,
                                  const void *weight, int64_t N, int32_t Ng, double L, void *rho_out, uint32_t flags)
{
    if (!ctx) return KDE_EINVAL;
    if (N < 0 || Ng < 1 || Ng > KDE_MAX_NG || !(L > 0) || !rho_out || (N > 0 && !u))
        return kde_fail(ctx, KDE_EINVAL, "kde_deposit: need N >= 0, 1 <= Ng <= %d, L > 0, non-null u and rho_out",
                        KDE_MAX_NG);
    if (!kappa && !(kappa_uniform > 0 && kappa_uniform <= KDE_KAPPA_MAX))
        return kde_fail(ctx, KDE_EINVAL, "kde_deposit: kappa_uniform must be in (0, 1e6]");
    if (N > 0xFFFFFFFFll) return kde_fail(ctx, KDE_EINVAL, "kde_deposit: N must be below 2^32");
    if (flags & ~KDE_F64) return kde_fail(ctx, KDE_ENOTSUP, "kde_deposit: unsupported flags 0x%x", flags);
    if (flags & KDE_F64)
        return deposit_api_f64(ctx, u, (const double *)kappa, kappa_uniform, (const double *)weight, N, Ng, L,
                               (double *)rho_out);
    return deposit_api_f32(ctx, u, (const float *)kappa, kappa_uniform, (const float *)weight, N, Ng, L, (float *)rho_out);
}

// ---------------------------------------------------------------------------
// Allocation-free deposit.
//
// Some callers cannot call cudaMalloc once they are running: code that records
// its work into a CUDA graph or runs under a host allocator policy that
// forbids device allocations after start-up, plugins that must not touch the
// host process's memory pools, and real-time loops that may not block on the
// driver's allocator.  kde_deposit_noalloc serves them: it needs no context and
// no workspace.  Particles may come in any order (nothing is sorted); every
// scratch byte it uses -- the int64 grid accumulators, the node table and the
// largest-weight word -- lives in the file-scope array below, which every GPU
// that loads this library holds (KDE_NOALLOC_SCRATCH_BYTES) until the process
// exits.  Every call shares that one array: calls that overlap on the GPU
// (concurrent streams, or several host threads) race on it.
// ---------------------------------------------------------------------------
#define NOALLOC_ACC_OFF 0
#define NOALLOC_NODE_OFF (KDE_MAX_NG * 8)
#define NOALLOC_WMAX_OFF (NOALLOC_NODE_OFF + KDE_MAX_NG * 16)
static_assert(KDE_NOALLOC_SCRATCH_BYTES >= NOALLOC_WMAX_OFF + 256, "scratch layout exceeds the declared size");

static __device__ __align__(256) unsigned char kde_noalloc_scratch[KDE_NOALLOC_SCRATCH_BYTES];

template <typename T>
__global__ void __launch_bounds__(DEP_THREADS) deposit_chunk_unsorted_kernel(DepSrc<T> S)
{
    __shared__ DepRec<T> rec[DEP_CHUNK];
    __shared__ T part[DEP_WARPS * 32 * DEP_WARPS];
    __shared__ int red[DEP_WARPS];
    __shared__ int cmm[2 * DEP_WARPS];
    deposit_chunk_body<T>(S, blockIdx.x, rec, part, red, cmm);
}

template <typename T2>
__global__ void noalloc_node_kernel(T2 *tab, int Ng)
{
    int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= Ng) return;
    double s, c;
    sincospi((double)g / (double)Ng, &s, &c);
    tab[g].x = s;
    tab[g].y = c;
}

// device address of the scratch array on the current device.  Looked up on every
// call (a host-side table lookup once the module is loaded): a cached address
// would go stale if the device's context were reset and the module reloaded.
static unsigned char *noalloc_scratch_address()
{
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, kde_noalloc_scratch) != cudaSuccess || !p) return nullptr;
    return (unsigned char *)p;
}

// every launch goes through cudaLaunchKernel, whose return value is that launch's
// own status (a trailing cudaGetLastError would also report, and clear, errors of
// unrelated earlier launches on this thread)
template <typename T>
static kde_status deposit_noalloc_impl(cudaStream_t stream, unsigned char *scr, const uint32_t *u, const T *kappa,
                                       double kappa_u, const T *weight, int64_t N, int Ng, double L, T *rho_out)
{
    typedef typename V2<T>::t T2;
    long long *acc = (long long *)(scr + NOALLOC_ACC_OFF);
    T2 *nodes = (T2 *)(scr + NOALLOC_NODE_OFF);
    unsigned int *wmax = (unsigned int *)(scr + NOALLOC_WMAX_OFF);
    if (cudaMemsetAsync(acc, 0, (size_t)Ng * sizeof(long long), stream) != cudaSuccess) return KDE_ECUDA;
    if (N == 0) return cudaMemsetAsync(rho_out, 0, (size_t)Ng * sizeof(T), stream) == cudaSuccess ? KDE_OK : KDE_ECUDA;
    {
        void *args[] = {&nodes, &Ng};
        if (cudaLaunchKernel((const void *)noalloc_node_kernel<T2>, dim3((Ng + 255) / 256), dim3(256), args, 0,
                             stream) != cudaSuccess)
            return KDE_ECUDA;
    }
    const double coef = KDE_TWO_PI / L;
    const double norm_u = kappa ? 0.0 : kde_norm(kappa_u);
    const double norm_bound = kappa ? kde_norm(KDE_KAPPA_MAX) : norm_u;
    const double w_u = L / (double)N;
    double bound = (double)N * w_u * coef * norm_bound;
    if (weight) {
        if (cudaMemsetAsync(wmax, 0, 4, stream) != cudaSuccess) return KDE_ECUDA;
        int blocks = (int)((N + 255) / 256);
        blocks = blocks > 1024 ? 1024 : blocks;
        unsigned int *no_status = nullptr;
        void *args[] = {(void *)&weight, &N, &wmax, &no_status};
        if (cudaLaunchKernel((const void *)wmax_kernel<T>, dim3(blocks), dim3(256), args, 0, stream) != cudaSuccess)
            return KDE_ECUDA;
    }
    DepSrc<T> S{};
    S.u = u;
    S.N = N;
    S.kappa = kappa;
    S.kappa_u = (T)kappa_u;
    S.kscale = (T)1;
    S.norm_u = (T)norm_u;
    S.w = weight;
    S.w_u = (T)w_u;
    S.coef = (T)coef;
    S.Ng = Ng;
    S.nodes = nodes;
    S.acc = acc;
    S.bound = bound;
    S.wmax_bits = weight ? wmax : nullptr;
    S.norm_bound = norm_bound;
    S.status = nullptr;
    {
        void *args[] = {&S};
        if (cudaLaunchKernel((const void *)deposit_chunk_unsorted_kernel<T>,
                             dim3((unsigned)((N + DEP_CHUNK - 1) / DEP_CHUNK)), dim3(DEP_THREADS), args, 0,
                             stream) != cudaSuccess)
            return KDE_ECUDA;
    }
    {
        const unsigned int *wb = weight ? wmax : nullptr;
        double wscale = (double)N * coef * norm_bound;
        const long long *lo = nullptr;
        void *args[] = {&acc, &Ng, &bound, (void *)&wb, &wscale, &rho_out, (void *)&lo};
        if (cudaLaunchKernel((const void *)acc_to_real_kernel<T>, dim3((Ng + 255) / 256), dim3(256), args, 0,
                             stream) != cudaSuccess)
            return KDE_ECUDA;
    }
    return KDE_OK;
}

extern "C" kde_status kde_deposit_noalloc(void *stream, const uint32_t *u, const void *kappa, double kappa_uniform,
                                          const void *weight, int64_t N, int32_t Ng, double L, void *rho_out,
                                          uint32_t flags)
{
    if (N < 0 || N > 0xFFFFFFFFll || Ng < 1 || Ng > KDE_NOALLOC_MAX_NG || !(L > 0) || !rho_out || (N > 0 && !u))
        return KDE_EINVAL;
    if (!kappa && !(kappa_uniform > 0 && kappa_uniform <= KDE_KAPPA_MAX)) return KDE_EINVAL;
    if (flags & ~KDE_F64) return KDE_ENOTSUP;
    unsigned char *scr = noalloc_scratch_address();
    if (!scr) return KDE_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;
    if (flags & KDE_F64)
        return deposit_noalloc_impl<double>(s, scr, u, (const double *)kappa, kappa_uniform, (const double *)weight, N,
                                            Ng, L, (double *)rho_out);
    return deposit_noalloc_impl<float>(s, scr, u, (const float *)kappa, kappa_uniform, (const float *)weight, N, Ng, L,
                                       (float *)rho_out);
}
