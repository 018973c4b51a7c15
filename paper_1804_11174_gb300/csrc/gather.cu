// gather.cu -- field interpolation through the deposit's kernels, fused with
// the leap-frog push of the PIC cycle (Sec. III.A).
//
//   E_i = (2 pi / Ng) norm(kappa_i) sum_g E_g exp(-2 kappa_i sin^2((theta_g - theta_i)/2))
//
// Forms.  gather_tile_kernel (FP32, default cut, sorted particles of a PIC
// step): a CTA smooths the field at the interpolation points of its tile and
// the particles take the interpolant.  gather2_kernel (FP32 otherwise): the
// whole grid (half-angle sine, cosine, field) in shared memory, threads own
// particles (a sorted warp's share a few cells), each warp sweeps one node
// window covering all of its lanes' truncated supports, so every node read is
// a broadcast.  gather64_kernel: the FP64 form.  The push, the write-back of
// the particle state and the field energy ride in the same kernel.  Plain
// FP32 calls at the default cut go through the tables of gtable.cu.
#include "common.cuh"
#include "fp64.cuh"
#include "proxy.cuh"

#define GAT_THREADS 256

template <typename T> struct V2g;
template <> struct V2g<float> { typedef float2 t; };
template <> struct V2g<double> { typedef double2 t; };

template <typename T> struct GatherArgs {
    const uint32_t *u;
    const T *kappa;
    T kappa_u;
    const T *norm;  // FP64: norms of the particles, or null
    T norm_u;
    int64_t N;
    const T *field;
    int Ng;
    const typename V2g<T>::t *nodes;
    T coef;  // 2 pi / Ng
    T *out;
    const uint32_t *perm;
    // push (active when u_out != nullptr)
    const T *v_in;
    uint32_t *u_out;
    T *v_out;
    T *kappa_out;
    const T *norm_in;  // FP64
    T *norm_out;
    const uint32_t *id_in;
    uint32_t *id_out;
    T kick_qm_dt;
    T dt_scale;
    double *energy;
    const double *kstar_in;
    double *kstar_out;
    double dx;
    unsigned int *status;
    const float2 *ntab;  // FP32 norm table (kde_norm_tab) for per-particle widths
    // push only: count table of the next step's cell sort, or null (counts of the new
    // positions are added with one atomic per warp and distinct cell)
    unsigned int *counts;
    int cnt_nblk, cnt_shift;
    float xcut = (float)KDE_XCUT;  // FP32 packed gather: truncation cut exponent
    PxyGrid grid;                    // the nodes as position codes
    const float *pxt;                // interpolation matrices (proxy.cuh)
    const unsigned int *krange;      // float bits of the largest and smallest width, or null
    int tile;                        // particles of a CTA of gather_tile_kernel
};

__device__ __forceinline__ int window_nodes_g(float kappa, int Ng, float xcut)
{
    float s2 = xcut * (float)(KDE_LN2 / 2.0) / kappa;
    if (s2 >= 1.0f) return Ng;
    float r = 2.0f * asinf(sqrtf(s2));
    int w = (int)ceilf(r * (float)Ng * (float)(1.0 / KDE_TWO_PI)) + 1;
    return w >= Ng ? Ng : w;
}

__device__ __forceinline__ uint32_t advance_position(uint32_t u, float d)
{
    // d = displacement in units of 2^-32 L
    if (fabsf(d) < 2147483520.0f) return u + (uint32_t)__float2int_rn(d);
    d = fmodf(d, 4294967296.0f);
    return u + (uint32_t)(long long)__float2ll_rn(d);
}
__device__ __forceinline__ uint32_t advance_position(uint32_t u, double d)
{
    d = fmod(d, 4294967296.0);
    return u + (uint32_t)(long long)__double2ll_rn(d);
}

// ---------------------------------------------------------------------------
// FP64 gather and push.  Bound by the FP64 pipe like the deposit: eleven operations a
// (particle, node) pair.  A CTA takes PB particles (few for a small run, so that it reaches
// every SM); one thread a particle forms its terms, then GAT_THREADS / PB lanes a particle
// sweep the particle's own window, and the particle's thread pushes it.  Measured: 4096
// particles on 64 nodes 41 -> 12 us.
// ---------------------------------------------------------------------------
template <int PB>
__global__ void __launch_bounds__(GAT_THREADS) gather64_kernel(GatherArgs<double> A, const double *__restrict__ tab2)
{
    constexpr int LP = GAT_THREADS / PB;
    __shared__ __align__(16) double tab[F64_TAB];
    __shared__ double bs[PB], bc[PB], ei[PB];
    __shared__ int g0[PB], gl[PB];
    const int tid = threadIdx.x, Ng = A.Ng;
    f64_tab_load(tab, tab2, tid, GAT_THREADS);
    if (blockIdx.x == 0 && A.energy) {
        __shared__ double red[GAT_THREADS];
        double s = 0.0;
        for (int g = tid; g < Ng; g += GAT_THREADS) s += A.field[g] * A.field[g];
        red[tid] = s;
        __syncthreads();
        for (int o = GAT_THREADS / 2; o > 0; o >>= 1) {
            if (tid < o) red[tid] += red[tid + o];
            __syncthreads();
        }
        if (tid == 0) {
            A.energy[0] = 0.5 * red[0] * A.dx;
            if (A.kstar_out) A.kstar_out[0] = A.kstar_in ? A.kstar_in[0] : A.kappa_u;
        }
    }
    const int64_t j = (int64_t)blockIdx.x * PB + tid;
    const bool mine = tid < PB && j < A.N;
    uint32_t uu = 0u;
    double k = A.kappa_u, nm = A.norm_u;
    if (mine) {
        uu = A.u[j];
        if (A.kappa) k = A.kappa[j];
        if (!(k > 0.0 && k <= KDE_KAPPA_MAX)) {
            kde_flag(A.status, KDE_DEV_KAPPA_RANGE, (unsigned)j);
            k = KDE_KAPPA_MAX;
        }
        if (A.norm) nm = A.norm[j];
        else if (A.kappa) nm = f64_norm(k);
        double sh, ch;
        kde_half_sincos(uu, sh, ch);
        const double beta = sqrt(2.0 * KDE_LOG2E * k);
        bs[tid] = beta * sh;
        bc[tid] = beta * ch;
        const int W = window_nodes_g((float)k, Ng, (float)KDE_XCUT64), len = min(Ng, 2 * W + 1);
        int g = len == Ng ? 0 : kde_cell(uu, Ng) - W;
        g0[tid] = g < 0 ? g + Ng : g;
        gl[tid] = len;
    } else if (tid < PB) {
        gl[tid] = 0;
    }
    __syncthreads();
    {
        const int p = tid / LP, l = tid % LP, len = gl[p];
        double acc = 0.0;
        if (len > 0) {
            const double ps = bs[p], pc = bc[p];
            int g = g0[p] + l;
            g = g >= Ng ? g - Ng : g;
#pragma unroll 4
            for (int r = l; r < len; r += LP) {
                const double2 sc = A.nodes[g];
                const double s = fma(sc.x, pc, -(sc.y * ps));
                double T, q;
                f64_exp2neg(tab, s, T, q);
                const double te = T * A.field[g];
                acc = fma(te, q, acc) + te;
                g += LP;
                g = g >= Ng ? g - Ng : g;
            }
        }
#pragma unroll
        for (int o = LP / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (l == 0) ei[p] = acc;
    }
    __syncthreads();
    if (!mine) return;
    const double Ei = ei[tid] * nm * A.coef;
    if (A.u_out) {
        const double v = A.v_in[j] + A.kick_qm_dt * Ei;
        A.v_out[j] = v;
        A.u_out[j] = advance_position(uu, v * A.dt_scale);
        if (A.kappa_out) A.kappa_out[j] = k;
        if (A.norm_out) A.norm_out[j] = A.norm_in[j];
        if (A.id_out) A.id_out[j] = A.id_in[j];
    } else {
        A.out[A.perm ? A.perm[j] : j] = Ei;
    }
}

// ---------------------------------------------------------------------------
// FP32 gather with packed pair arithmetic: each lane carries GAT2_NP = 4
// particles (a warp covers 128 consecutive sorted particles) as two f32x2
// pairs, and every node record is kept pre-duplicated in shared memory, so one
// 128-bit and one 64-bit broadcast load feed four particles' multiply-adds.  The
// node loop runs as two contiguous segments (before and after the wrap point), so
// it carries no per-node index arithmetic.  The form of the kernel value is chosen
// per block by its largest width, as in the packed deposit:
//  * half-angle: nodes (sin, sin, -cos, -cos) of half the node angle, particles
//    (beta sin, beta cos) of half theirs, 2^-(S_g beta c_j - C_g beta s_j)^2;
//  * cosine (largest width <= KDE_COSFORM_KMAX): nodes (sin, sin, cos, cos) of the
//    full angle, particles (K cos, K sin), 2^(K cos(x_j - x_g)), and 2^-K folded into
//    the particle's norm; three multiply-adds per pair instead of four.
// ---------------------------------------------------------------------------
// Tile shapes (template parameters of gather2_kernel, chosen per call by the variant
// table below): NP particles a lane (even), node-loop unrolling UD for windows of
// GAT2_DEEP_LEN nodes or more and US below, and a launch bound of MINB resident
// blocks per SM.  Variants with the same NP compute the same sums in the same order
// (NP sets each warp's node window), so their results are bitwise identical and only
// the speed differs.
#define GAT2_WARPS 4
#define GAT2_DEEP_LEN 128

// the node loop of the packed gather over the window's two contiguous segments
// [g0, e1) and [0, e2): NPP particle pairs a lane, U nodes unrolled
template <int U, bool COS, int NPP>
__device__ __forceinline__ void gat2_nodes(const float4 *SC, const float2 *FF, int g0, int e1, int e2,
                                           const kde_f2 (&psP)[NPP], const kde_f2 (&pcP)[NPP], kde_f2 (&acc)[NPP])
{
    auto node = [&](int g) {
        const float4 r4 = SC[g];
        const float2 f = FF[g];
        const kde_f2 S2 = kde_pk(r4.x, r4.y), C2 = kde_pk(r4.z, r4.w), F2 = kde_pk(f.x, f.y);
#pragma unroll
        for (int q = 0; q < NPP; ++q) {
            const kde_f2 ev = kde_fma2(S2, psP[q], kde_mul2(C2, pcP[q]));
            if (COS) acc[q] = kde_fma2(kde_ex22(ev), F2, acc[q]);  // 2^(K cos(x_j - x_g))
            else acc[q] = kde_fma2(kde_ex2neg2(kde_mul2(ev, ev)), F2, acc[q]);  // 2^-(beta sin((x_j - x_g)/2))^2
        }
    };
#pragma unroll U
    for (int g = g0; g < e1; ++g) node(g);
#pragma unroll U
    for (int g = 0; g < e2; ++g) node(g);
}

// the end of a warp's gather of NP particles a lane (particle base + 32 h + lane) with codes
// uu and fields ea: the push and the write-back of the state, or the plain output.  VIN: the
// velocities are in vin already
template <bool VIN, int NP>
__device__ __forceinline__ void gat_finish(const GatherArgs<float> &A, int64_t base, int lane, const uint32_t (&uu)[NP],
                                           const float (&ea)[NP], const float *vpre)
{
    const int Ng = A.Ng;
    if (A.u_out) {
        // the push's inputs of four particles at a time first (one load latency per group;
        // the stores below alias nothing the loads read, but the compiler cannot know
        // that), then the stores
        constexpr int HB = NP % 4 == 0 ? 4 : (NP % 3 == 0 ? 3 : 2);
#pragma unroll
        for (int h0 = 0; h0 < NP; h0 += HB) {
            float vin[HB], kin[HB];
            uint32_t idin[HB];
#pragma unroll
            for (int hh = 0; hh < HB; ++hh) {
                const int64_t j = base + (h0 + hh) * 32 + lane;
                const bool ok = j < A.N;
                vin[hh] = VIN ? vpre[h0 + hh] : (ok ? A.v_in[j] : 0.f);
                kin[hh] = (ok && A.kappa_out) ? (A.kappa ? A.kappa[j] : A.kappa_u) : 0.f;
                idin[hh] = (ok && A.id_out) ? A.id_in[j] : 0u;
            }
#pragma unroll
            for (int hh = 0; hh < HB; ++hh) {
                const int h = h0 + hh;
                const int64_t j = base + h * 32 + lane;
                int key = -1;
                if (j < A.N) {
                    const float v = fmaf(A.kick_qm_dt, ea[h], vin[hh]);
                    A.v_out[j] = v;
                    const uint32_t nu = advance_position(uu[h], v * A.dt_scale);
                    A.u_out[j] = nu;
                    if (A.kappa_out) {
                        const float k = (kin[hh] > 0.f && kin[hh] <= (float)KDE_KAPPA_MAX) ? kin[hh] : (float)KDE_KAPPA_MAX;
                        A.kappa_out[j] = k;
                        if (A.norm_out) A.norm_out[j] = kde_norm_tab(A.ntab, k);
                    }
                    if (A.id_out) A.id_out[j] = idin[hh];
                    key = kde_cell(nu, Ng);
                }
                if (A.counts) {  // warp-uniform; the 32 particles of a round share one sort tile
                    const unsigned int peers = __match_any_sync(0xffffffffu, key);
                    if (key >= 0 && lane == __ffs(peers) - 1)
                        atomicAdd(&A.counts[(size_t)key * A.cnt_nblk + (size_t)(j >> A.cnt_shift)],
                                  (unsigned int)__popc(peers));
                }
            }
        }
    } else {
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            const int64_t j = base + h * 32 + lane;
            if (j < A.N) A.out[A.perm ? A.perm[j] : j] = ea[h];
        }
    }
}

template <int NP, int UD, int US, int MINB>
__global__ void __launch_bounds__(GAT2_WARPS * 32, MINB) gather2_kernel(GatherArgs<float> A)
{
    constexpr int GAT2_NP = NP, GAT2_ITEM = 32 * NP;
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ float kred[GAT2_WARPS];
    const int Ng = A.Ng;
    float4 *SC = (float4 *)sm;         // node angle records
    float2 *FF = (float2 *)(SC + Ng);  // (E, E)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = ((int64_t)blockIdx.x * GAT2_WARPS + warp) * GAT2_ITEM;
    // held across the node loop: positions and norms; widths until the particle terms
    // are formed; the push's other inputs are loaded after the loop (registers are the
    // limit with eight particles a lane, and other warps cover the load latency)
    float nm[GAT2_NP], kap[GAT2_NP];
    uint32_t uu[GAT2_NP];
    int lo = 0x3fffffff, hi = -0x3fffffff;  // the warp's first and last cell, then its window
    float kmax = 0.f, kmin = (float)KDE_KAPPA_MAX;
#pragma unroll
    for (int h = 0; h < GAT2_NP; ++h) {
        const int64_t j = base + h * 32 + lane;
        const bool valid = j < A.N;
        uu[h] = valid ? A.u[j] : 0u;
        float k = A.kappa ? (valid ? A.kappa[j] : 1.0f) : A.kappa_u;
        if (valid && !(k > 0.f && k <= (float)KDE_KAPPA_MAX)) {
            kde_flag(A.status, KDE_DEV_KAPPA_RANGE, (unsigned)j);
            k = (float)KDE_KAPPA_MAX;
        }
        kap[h] = k;
        nm[h] = A.kappa ? kde_norm_tab(A.ntab, k) : A.norm_u;
        if (valid) {
            kmax = fmaxf(kmax, k);
            kmin = fminf(kmin, k);
            const int cell = kde_cell(uu[h], Ng);
            lo = min(lo, cell);
            hi = max(hi, cell);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        kmax = fmaxf(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
        kmin = fminf(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
    }
    // one window for the warp: the widest kernel's reach around its cell range (it holds
    // every particle's own window, since the widest kernel has the smallest kappa)
    if (lo <= hi) {
        const int W = window_nodes_g(kmin, Ng, A.xcut);
        lo -= W;
        hi += W;
    }
    if (lane == 0) kred[warp] = kmax;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < GAT2_WARPS; ++w) kmax = fmaxf(kmax, kred[w]);
    const bool cosf = kmax <= KDE_COSFORM_KMAX;
    for (int g = threadIdx.x; g < Ng; g += GAT2_WARPS * 32) {
        const float2 sc = A.nodes[g];
        if (cosf) {
            const float sf = 2.f * sc.x * sc.y, cf = (sc.y - sc.x) * (sc.y + sc.x);
            SC[g] = make_float4(sf, sf, cf, cf);
        } else {
            SC[g] = make_float4(sc.x, sc.x, -sc.y, -sc.y);
        }
    }
    // the field is the previous kernel's output; so far only the sorted particles (two or
    // more kernels back) and the node table have been read
    kde_pdl_wait();
    kde_pdl_trigger();
    for (int g = threadIdx.x; g < Ng; g += GAT2_WARPS * 32) {
        const float f = A.field[g];
        FF[g] = make_float2(f, f);
    }
    if (blockIdx.x == 0 && A.energy) {
        __shared__ double red[GAT2_WARPS * 32];
        double sum = 0.0;
        for (int g = threadIdx.x; g < Ng; g += GAT2_WARPS * 32) sum += (double)A.field[g] * (double)A.field[g];
        red[threadIdx.x] = sum;
        __syncthreads();
        for (int o = GAT2_WARPS * 16; o > 0; o >>= 1) {
            if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            A.energy[0] = 0.5 * red[0] * A.dx;
            if (A.kstar_out) A.kstar_out[0] = A.kstar_in ? A.kstar_in[0] : (double)A.kappa_u;
        }
    }
    __syncthreads();

    int len = hi - lo + 1;
    if (len >= Ng) {
        lo = 0;
        len = Ng;
    }
    if (len <= 0) return;  // whole warp past the end
    // (ps, pc) pair with the node's (sin, sin) and (c, c) columns: half-angle (beta cos,
    // beta sin) of half the particle angle, cosine form (K sin, K cos) of the full one
    float ps[GAT2_NP], pc[GAT2_NP];
#pragma unroll
    for (int h = 0; h < GAT2_NP; ++h) {
        float sh, ch;
        kde_half_sincos(uu[h], sh, ch);
        if (cosf) {
            const float K = (float)KDE_LOG2E * kap[h];
            ps[h] = K * (2.f * sh * ch);
            pc[h] = K * ((ch - sh) * (ch + sh));
            nm[h] *= kde_ex2(-K);
        } else {
            const float beta = sqrtf((float)(2.0 * KDE_LOG2E) * kap[h]);
            ps[h] = beta * ch;
            pc[h] = beta * sh;
        }
    }
    int g0 = lo % Ng;
    if (g0 < 0) g0 += Ng;
    constexpr int NPP = GAT2_NP / 2;  // packed particle pairs a lane
    kde_f2 psP[NPP], pcP[NPP], acc[NPP];
#pragma unroll
    for (int q = 0; q < NPP; ++q) {
        psP[q] = kde_pk(ps[2 * q], ps[2 * q + 1]);
        pcP[q] = kde_pk(pc[2 * q], pc[2 * q + 1]);
        acc[q] = kde_pk(0.f, 0.f);
    }
    const int e1 = g0 + len < Ng ? g0 + len : Ng;  // first segment [g0, e1), then [0, len - (e1 - g0))
    const int e2 = len - (e1 - g0);
    // long windows take the deeper unrolling (more exp2 in flight), short ones the
    // shallower (less remainder work)
    const bool deep = len >= GAT2_DEEP_LEN;
    if (cosf) {
        if (deep) gat2_nodes<UD, true, NPP>(SC, FF, g0, e1, e2, psP, pcP, acc);
        else gat2_nodes<US, true, NPP>(SC, FF, g0, e1, e2, psP, pcP, acc);
    } else {
        if (deep) gat2_nodes<UD, false, NPP>(SC, FF, g0, e1, e2, psP, pcP, acc);
        else gat2_nodes<US, false, NPP>(SC, FF, g0, e1, e2, psP, pcP, acc);
    }
    float ea[GAT2_NP];
#pragma unroll
    for (int q = 0; q < NPP; ++q) kde_upk(acc[q], ea[2 * q], ea[2 * q + 1]);
#pragma unroll
    for (int h = 0; h < GAT2_NP; ++h) ea[h] *= nm[h] * A.coef;
    gat_finish<false>(A, base, lane, uu, ea, nullptr);
}

// ---------------------------------------------------------------------------
// Gather + push of cell-sorted particles through proxies (proxy.cuh): a CTA takes
// A.tile consecutive particles -- an interval of whole cells, widths in [kmin, kmax] --
// evaluates the field at P Q proxy particles from the nodes, turns these values into the
// coefficients of the joint Chebyshev interpolant and evaluates that at its particles.  A
// particle then costs its Chebyshev values and P (one width) or 28 to 48 multiply-adds
// (packed for two particles) whatever the window, and no norm is read: the normalisation is
// interpolated with the kernel.  Tiles whose range of widths is too wide, or whose windows are short
// beside P Q, sweep the nodes particle by particle as gather2_kernel does (GATT_WARPS
// warps, 128 particles each at a time).
// Everything before kde_pdl_wait() -- the box, the proxies -- overlaps the field kernel.
// Bound by instruction issue and fetch (a tile runs straight through its code) and latency.
// Measured: 2^20 particles on 256 nodes, widths near 14, 38.6 us swept, 22.8 in tiles and 14.5
// with gatt_run's loop without bounds checks.
// ---------------------------------------------------------------------------
#define GATT_THREADS 256
#define GATT_WARPS 8
#define GATT_UNIT 1024  // particles the CTA's warps take in a round, 4 a lane

// sums over the warp of v[0..7] (lane l ends with the sum of v[(l >> 2) & 7])
__device__ __forceinline__ float warp_sum8(float (&v)[8], int lane)
{
#pragma unroll
    for (int o = 4; o >= 1; o >>= 1) {
        const bool up = (lane & (o * 4)) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float send = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o * 4);
        }
    }
    float r = v[0];
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    return r;
}

// field at the PM x QM proxies of the box from the window nodes, then coefficients
// C[p QM + q] (the normalisation and coef included), each stored twice for the packed
// evaluation.  s2: sin^2 of the thread's first node (r = tid) and every proxy position, known
// before the field; tabs: the interpolation matrices of PM and QM in shared memory;
// part: GATT_WARPS x PM x QM floats; F: 2 PM QM floats
template <int PM, int QM>
__device__ __forceinline__ void gatt_coefs(const GatherArgs<float> &A, int g_lo, int R, const float *s2a,
                                           const uint32_t *cd, const float *fr, const float *k2, const float *nk,
                                           const float *tabs, float *part, float *F, float2 *C)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, Ng = A.Ng;
    constexpr int PQ = PM * QM;
    auto wrap = [&](int r) {
        const int g = g_lo + r;
        return g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
    };
    const float e0 = tid < R ? A.field[wrap(tid)] : 0.f;
    float kk[QM];
#pragma unroll
    for (int b = 0; b < QM; ++b) kk[b] = k2[b];
#pragma unroll(QM == 1 ? PM : 1)
    for (int a = 0; a < PM; ++a) {
        float v[8];
        const float s2 = s2a[a * GATT_THREADS + tid];
#pragma unroll
        for (int b = 0; b < 8; ++b) v[b] = b < QM ? kde_ex2(s2 * kk[b < QM ? b : 0]) * e0 : 0.f;
        if (R > GATT_THREADS) {
            const uint32_t ca = cd[a];
            const float fa = fr[a];
#pragma unroll 1
            for (int r = tid + GATT_THREADS; r < R; r += GATT_THREADS) {
                const int g = wrap(r);
                uint32_t nc;
                float nf;
                pxy_node(A.grid, g, nc, nf);
                const float s2r = pxy_sin2(nc, nf, ca, fa), e = A.field[g];
#pragma unroll
                for (int b = 0; b < QM; ++b) v[b] = fmaf(kde_ex2(s2r * kk[b]), e, v[b]);
            }
        }
        if (QM == 1) {
            float w = v[0];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            if (lane == 0) part[warp * PM + a] = w;
        } else {
            const float w = warp_sum8(v, lane);
            if ((lane & 3) == 0 && (lane >> 2) < QM) part[(warp * PM + a) * QM + (lane >> 2)] = w;
        }
    }
    __syncthreads();
    const float *cp = tabs, *cq = tabs + PM * PM;
    for (int i = tid; i < PQ; i += GATT_THREADS) {
        float f = 0.f;
#pragma unroll
        for (int w = 0; w < GATT_WARPS; ++w) f += part[w * PQ + i];
        F[i] = f * nk[i % QM];
    }
    __syncthreads();
    float *U = F + PQ;
    for (int i = tid; i < PQ; i += GATT_THREADS) {
        const int p = i / QM, b = i % QM;
        float f = 0.f;
#pragma unroll
        for (int a = 0; a < PM; ++a) f = fmaf(cp[p * PM + a], F[a * QM + b], f);
        U[i] = f;
    }
    if (QM > 1) __syncthreads();
    for (int i = tid; i < PQ; i += GATT_THREADS) {
        const int p = i / QM, q = i % QM;
        float f = 0.f;
#pragma unroll
        for (int b = 0; b < QM; ++b) f = fmaf(cq[q * QM + b], U[p * QM + b], f);
        C[i] = make_float2(f, f);
    }
    __syncthreads();
}

// the interpolant at four particles a lane (two packed pairs); TRI: the coefficients with
// p / PM + q / QM < 1 alone
template <int PM, int QM, bool TRI>
__device__ __forceinline__ void gatt_eval(const float2 *C, const float (&xs)[4], const float (&ss)[4], float (&ea)[4])
{
    const kde_f2 one = kde_pk(1.f, 1.f), neg = kde_pk(-1.f, -1.f);
    kde_f2 x[2], x2[2], s[2], t0[2], t1[2], acc[2], tq[QM][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        x[h] = kde_pk(xs[2 * h], xs[2 * h + 1]);
        x2[h] = kde_pk(2.f * xs[2 * h], 2.f * xs[2 * h + 1]);
        s[h] = kde_pk(ss[2 * h], ss[2 * h + 1]);
        tq[0][h] = one;
        if (QM > 1) tq[1 % QM][h] = s[h];
#pragma unroll
        for (int q = 2; q < QM; ++q) {
            const kde_f2 sq = kde_fma2(s[h], tq[q - 1][h], kde_pk(0.f, 0.f));
            tq[q][h] = kde_fma2(kde_pk(2.f, 2.f), sq, kde_mul2(neg, tq[q - 2][h]));
        }
        t0[h] = one;
        t1[h] = x[h];
    }
#pragma unroll
    for (int p = 0; p < PM; ++p) {
        kde_f2 row[2];
#pragma unroll
        for (int q = 0; q < QM; ++q) {
            if (TRI && p * QM + q * PM >= PM * QM) continue;
            const float2 c2 = C[p * QM + q];
            const kde_f2 c = kde_pk(c2.x, c2.y);
#pragma unroll
            for (int h = 0; h < 2; ++h) row[h] = q == 0 ? c : kde_fma2(c, tq[q][h], row[h]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (p == 0) {
                acc[h] = row[h];
            } else {
                acc[h] = kde_fma2(row[h], t1[h], acc[h]);
                const kde_f2 t2 = kde_fma2(x2[h], t1[h], kde_mul2(neg, t0[h]));
                t0[h] = t1[h];
                t1[h] = t2;
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) kde_upk(acc[h], ea[2 * h], ea[2 * h + 1]);
}

// the places xs, ss of four particles a lane (base + 32 h + lane) in the box
template <int QM>
__device__ __forceinline__ void gatt_place(const GatherArgs<float> &A, const PxyBox &B, int64_t base, int lane,
                                           const uint32_t (&uu)[4], const float (&kap)[4], float (&xs)[4], float (&ss)[4])
{
    bool ok = true;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        xs[h] = pxy_x(B, uu[h]);
        ss[h] = QM > 1 ? (kap[h] - B.kc) * B.inv_kh : 0.f;
        ok = ok && kap[h] > 0.f && kap[h] <= (float)KDE_KAPPA_MAX;
    }
    if (QM > 1 && !ok) {
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            if (kap[h] > 0.f && kap[h] <= (float)KDE_KAPPA_MAX) continue;
            const int64_t j = base + h * 32 + lane;
            if (j < A.N) kde_flag(A.status, KDE_DEV_KAPPA_RANGE, (unsigned)j);
            ss[h] = ((float)KDE_KAPPA_MAX - B.kc) * B.inv_kh;
        }
    }
}

// the steps of a run but the last of a call (positions and velocities written, counts added,
// nothing else), for whole groups of 128 particles: pointers once a group, no bounds checks;
// returns the first group left.  Half the instructions of the general loop.
template <int PM, int QM, bool TRI>
__device__ __forceinline__ int64_t gatt_run(const GatherArgs<float> &A, const PxyBox &B, const float2 *C, int64_t base,
                                            int64_t t1, int lane, uint32_t (&uu)[4], float (&kap)[4], float (&vin)[4])
{
#pragma unroll 1
    while (base + 128 <= t1) {
        const int64_t next = base + GATT_UNIT;
        uint32_t nu[4];
        float nk[4], nv[4];
        if (next + 128 <= t1) {  // the next group's loads
            const uint32_t *pu = A.u + next + lane;
            const float *pk = A.kappa + next + lane, *pv = A.v_in + next + lane;
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                nu[h] = pu[32 * h];
                nk[h] = QM > 1 ? pk[32 * h] : 0.f;
                nv[h] = pv[32 * h];
            }
        } else {
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                nu[h] = 0u;
                nk[h] = nv[h] = 0.f;
            }
        }
        float xs[4], ss[4], ea[4];
        gatt_place<QM>(A, B, base, lane, uu, kap, xs, ss);
        gatt_eval<PM, QM, TRI>(C, xs, ss, ea);
        float *vo = A.v_out + base + lane;
        uint32_t *uo = A.u_out + base + lane;
        unsigned int *pc = A.counts + (base >> A.cnt_shift);  // the group lies in one sort tile
        float d[4];
        bool small = true;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const float v = fmaf(A.kick_qm_dt, ea[h], vin[h]);
            vo[32 * h] = v;
            d[h] = v * A.dt_scale;
            small = small && fabsf(d[h]) < 2147483520.0f;
        }
        uint32_t un[4];
        if (small) {
#pragma unroll
            for (int h = 0; h < 4; ++h) un[h] = uu[h] + (uint32_t)__float2int_rn(d[h]);
        } else {
#pragma unroll
            for (int h = 0; h < 4; ++h) un[h] = advance_position(uu[h], d[h]);
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            uo[32 * h] = un[h];
            const unsigned int key = __umulhi(un[h], (unsigned int)A.Ng);
            const unsigned int peers = __match_any_sync(0xffffffffu, key);
            if (lane == 31 - __clz(peers)) atomicAdd(&pc[key * (unsigned int)A.cnt_nblk], (unsigned int)__popc(peers));
            uu[h] = nu[h];
            kap[h] = nk[h];
            vin[h] = nv[h];
        }
        base = next;
    }
    return base;
}

// the direct sweep of one warp's 128 particles: node tables SC and FF of the whole grid in
// shared memory, in the form cosf
__device__ __forceinline__ void gatt_direct(const GatherArgs<float> &A, const float4 *SC, const float2 *FF, bool cosf,
                                            int64_t base, int lane, const uint32_t (&uu)[4], const float (&kap)[4],
                                            float (&ea)[4])
{
    const int Ng = A.Ng;
    float ps[4], pc[4], nm[4];
    int lo = 0x3fffffff, hi = -0x3fffffff;
    float kmin = (float)KDE_KAPPA_MAX;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int64_t j = base + h * 32 + lane;
        const bool valid = j < A.N;
        float k = kap[h];
        if (!(k > 0.f && k <= (float)KDE_KAPPA_MAX)) {
            if (valid) kde_flag(A.status, KDE_DEV_KAPPA_RANGE, (unsigned)j);
            k = (float)KDE_KAPPA_MAX;
        }
        nm[h] = A.kappa ? kde_norm_tab(A.ntab, k) : A.norm_u;
        if (valid) {
            kmin = fminf(kmin, k);
            const int cell = kde_cell(uu[h], Ng);
            lo = min(lo, cell);
            hi = max(hi, cell);
        }
        float sh, ch;
        kde_half_sincos(uu[h], sh, ch);
        if (cosf) {
            const float K = (float)KDE_LOG2E * k;
            ps[h] = K * (2.f * sh * ch);
            pc[h] = K * ((ch - sh) * (ch + sh));
            nm[h] *= kde_ex2(-K);
        } else {
            const float beta = sqrtf((float)(2.0 * KDE_LOG2E) * k);
            ps[h] = beta * ch;
            pc[h] = beta * sh;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        kmin = fminf(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
    }
    if (lo <= hi) {
        const int W = window_nodes_g(kmin, Ng, A.xcut);
        lo -= W;
        hi += W;
    }
    int len = hi - lo + 1;
    if (len >= Ng) {
        lo = 0;
        len = Ng;
    }
    kde_f2 psP[2], pcP[2], acc[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        psP[q] = kde_pk(ps[2 * q], ps[2 * q + 1]);
        pcP[q] = kde_pk(pc[2 * q], pc[2 * q + 1]);
        acc[q] = kde_pk(0.f, 0.f);
    }
    if (len > 0) {
        int g0 = lo % Ng;
        if (g0 < 0) g0 += Ng;
        const int e1 = g0 + len < Ng ? g0 + len : Ng, e2 = len - (e1 - g0);
        const bool deep = len >= GAT2_DEEP_LEN;
        if (cosf) {
            if (deep) gat2_nodes<8, true, 2>(SC, FF, g0, e1, e2, psP, pcP, acc);
            else gat2_nodes<4, true, 2>(SC, FF, g0, e1, e2, psP, pcP, acc);
        } else {
            if (deep) gat2_nodes<8, false, 2>(SC, FF, g0, e1, e2, psP, pcP, acc);
            else gat2_nodes<4, false, 2>(SC, FF, g0, e1, e2, psP, pcP, acc);
        }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) kde_upk(acc[q], ea[2 * q], ea[2 * q + 1]);
#pragma unroll
    for (int h = 0; h < 4; ++h) ea[h] *= nm[h] * A.coef;
}

// C of the compressed forms: degrees (P, Q) as evaluated
#define GATT_FORM_P(f) ((f) == 1 ? 8 : ((f) == 2 ? 16 : ((f) == 3 ? 7 : 8)))
#define GATT_FORM_Q(f) ((f) <= 2 ? 1 : ((f) == 3 ? 7 : 6))

__global__ void __launch_bounds__(GATT_THREADS, 3) gather_tile_kernel(GatherArgs<float> A)
{
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ uint32_t cd[PXY_MAXP];
    __shared__ float fr[PXY_MAXP], k2[8], nk[8];
    __shared__ float tabs[PXY_MAXP * PXY_MAXP + 8], part[GATT_WARPS * 49], F[2 * 49];
    __shared__ __align__(16) float s2a[PXY_MAXP * GATT_THREADS];  // also the energy sum's doubles
    __shared__ __align__(16) float2 C[50];
    __shared__ float kred[2 * GATT_WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, Ng = A.Ng;
    if (A.energy && blockIdx.x == gridDim.x - 1) {
        // the last CTA of the grid has the field energy alone
        double *red = (double *)s2a;
        kde_pdl_wait();
        kde_pdl_trigger();
        double sum = 0.0;
        for (int g = tid; g < Ng; g += GATT_THREADS) sum += (double)A.field[g] * (double)A.field[g];
        red[tid] = sum;
        __syncthreads();
        for (int o = GATT_THREADS / 2; o > 0; o >>= 1) {
            if (tid < o) red[tid] += red[tid + o];
            __syncthreads();
        }
        if (tid == 0) {
            A.energy[0] = 0.5 * red[0] * A.dx;
            if (A.kstar_out) A.kstar_out[0] = A.kstar_in ? A.kstar_in[0] : (double)A.kappa_u;
        }
        return;
    }
    const int64_t t0 = (int64_t)blockIdx.x * A.tile;
    const int64_t t1 = t0 + A.tile < A.N ? t0 + A.tile : A.N;  // not empty
    // the warp's first particles, in flight over everything up to the field
    uint32_t uu[4];
    float kap[4], vin[4];
    auto load = [&](int64_t base, uint32_t (&lu)[4], float (&lk)[4], float (&lv)[4]) {
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int64_t j = base + h * 32 + lane;
            const int64_t jj = j < A.N ? j : A.N - 1;
            lu[h] = A.u[jj];
            lk[h] = A.kappa ? A.kappa[jj] : A.kappa_u;
            lv[h] = A.u_out ? ((const float *)A.v_in)[jj] : 0.f;
        }
    };
    load(t0 + warp * 128, uu, kap, vin);
    float kmin, kmax;
    if (!A.kappa) {
        kmin = kmax = A.kappa_u;
    } else if (A.krange) {
        kmax = __uint_as_float(A.krange[0]);
        kmin = __uint_as_float(A.krange[1]);
    } else {
        kmin = (float)KDE_KAPPA_MAX;
        kmax = 0.f;
        for (int64_t j = t0 + tid; j < t1; j += GATT_THREADS) {
            float k = A.kappa[j];
            if (!(k > 0.f && k <= (float)KDE_KAPPA_MAX)) k = (float)KDE_KAPPA_MAX;
            kmin = fminf(kmin, k);
            kmax = fmaxf(kmax, k);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            kmin = fminf(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
            kmax = fmaxf(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
        }
        if (lane == 0) {
            kred[warp] = kmin;
            kred[GATT_WARPS + warp] = kmax;
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < GATT_WARPS; ++w) {
            kmin = fminf(kmin, kred[w]);
            kmax = fmaxf(kmax, kred[GATT_WARPS + w]);
        }
    }
    const int c_first = kde_cell(A.u[t0], Ng), c_last = kde_cell(A.u[t1 - 1], Ng);
    const int W = window_nodes_g(kmin, Ng, A.xcut);
    int g_lo = c_first - W, R = c_last + W - g_lo + 1;
    if (R >= Ng || R < 1 || c_last < c_first) {
        g_lo = 0;
        R = Ng;
    }
    PxyBox B;
    pxy_box_pos(B, A.grid, c_first, max(c_first, c_last), kmax);
    pxy_box_width(B, kmin, kmax);
    // the form of the tile: one width, P <= 8 or 16; a narrow range of widths, P <= 6 or 8;
    // else direct.  In instructions of a lane: compressed about 20 a particle and 0.8 a
    // coefficient, 5 a (node, proxy) and the tile's fixed steps; direct 2.6 a (particle, node)
    int form = 0;
    if (c_last >= c_first && A.xcut == (float)KDE_XCUT) {
        if (B.Q == 1) form = B.P <= 8 ? 1 : (B.P <= 16 ? 2 : 0);
        else if (B.lin) form = B.P <= 6 ? 3 : (B.P <= 8 ? 4 : 0);
        if (form) {
            const float n = (float)(t1 - t0), PQ = form == 1 ? 8.f : (form == 2 ? 16.f : (form == 3 ? 28.f : 48.f));
            const float comp = n * (20.f + 0.8f * PQ) + (float)R * PQ * 5.f + 60000.f;
            if (comp >= n * 2.6f * (float)R) form = 0;
        }
    }
    // what does not depend on the field, while the kernel before may still run
    float4 *SC = (float4 *)sm;
    float2 *FF = (float2 *)(SC + Ng);
    bool cosf = false;
    if (form) {
        const int P = GATT_FORM_P(form), Q = GATT_FORM_Q(form);
        const float *cp = A.pxt + pxy_tab_off(P), *cq = A.pxt + pxy_tab_off(Q);
        for (int i = tid; i < P * P; i += GATT_THREADS) tabs[i] = cp[i];
        if (tid < Q * Q) tabs[P * P + tid] = cq[tid];
        if (tid < P) pxy_pos(B, cp[P + tid] * (0.5f * (float)P), cd[tid], fr[tid]);
        if (tid >= 32 && tid < 32 + Q) {
            const int b = tid - 32;
            const float k = Q > 1 ? pxy_lin_kappa(B.kc, B.kh, cq[Q + b], Q) : kmin;
            k2[b] = (float)(-2.0 * KDE_LOG2E) * k;
            float nm = A.norm_u;
            if (A.kappa)
                nm = Q > 1 && A.krange ? __uint_as_float(A.krange[(Q == 7 ? PXY_NORM7 : PXY_NORM6) + b])
                                       : kde_norm_tab(A.ntab, k);
            nk[b] = A.coef * nm;
        }
        __syncthreads();
        int g = g_lo + (tid < R ? tid : 0);
        g = g < 0 ? g + Ng : (g >= Ng ? g - Ng : g);
        uint32_t nc;
        float nf;
        pxy_node(A.grid, g, nc, nf);
        for (int a = 0; a < P; ++a) s2a[a * GATT_THREADS + tid] = pxy_sin2(nc, nf, cd[a], fr[a]);
    } else {
        cosf = kmax <= KDE_COSFORM_KMAX;
        for (int g = tid; g < Ng; g += GATT_THREADS) {
            const float2 sc = A.nodes[g];
            if (cosf) {
                const float sf = 2.f * sc.x * sc.y, cf = (sc.y - sc.x) * (sc.y + sc.x);
                SC[g] = make_float4(sf, sf, cf, cf);
            } else {
                SC[g] = make_float4(sc.x, sc.x, -sc.y, -sc.y);
            }
        }
    }
    kde_pdl_wait();  // the field from here on
    kde_pdl_trigger();
    switch (form) {
    case 1: gatt_coefs<8, 1>(A, g_lo, R, s2a, cd, fr, k2, nk, tabs, part, F, C); break;
    case 2: gatt_coefs<16, 1>(A, g_lo, R, s2a, cd, fr, k2, nk, tabs, part, F, C); break;
    case 3: gatt_coefs<7, 7>(A, g_lo, R, s2a, cd, fr, k2, nk, tabs, part, F, C); break;
    case 4: gatt_coefs<8, 6>(A, g_lo, R, s2a, cd, fr, k2, nk, tabs, part, F, C); break;
    default:
        for (int g = tid; g < Ng; g += GATT_THREADS) {
            const float f = A.field[g];
            FF[g] = make_float2(f, f);
        }
        __syncthreads();
    }
    int64_t base = t0 + warp * 128;
    if (A.u_out && !A.kappa_out && !A.id_out && A.counts) {
        switch (form) {
        case 1: base = gatt_run<8, 1, false>(A, B, C, base, t1, lane, uu, kap, vin); break;
        case 2: base = gatt_run<16, 1, false>(A, B, C, base, t1, lane, uu, kap, vin); break;
        case 3: base = gatt_run<7, 7, true>(A, B, C, base, t1, lane, uu, kap, vin); break;
        case 4: base = gatt_run<8, 6, false>(A, B, C, base, t1, lane, uu, kap, vin); break;
        default: break;
        }
    }
    // the rest: a call's last step, plain gathers, the last particles, the direct sweep
#pragma unroll 1
    for (; base < t1; base += GATT_UNIT) {
        load(base, uu, kap, vin);
        float xs[4], ss[4], ea[4];
        if (form >= 3) gatt_place<2>(A, B, base, lane, uu, kap, xs, ss);
        else if (form) gatt_place<1>(A, B, base, lane, uu, kap, xs, ss);
        switch (form) {
        case 1: gatt_eval<8, 1, false>(C, xs, ss, ea); break;
        case 2: gatt_eval<16, 1, false>(C, xs, ss, ea); break;
        case 3: gatt_eval<7, 7, true>(C, xs, ss, ea); break;
        case 4: gatt_eval<8, 6, false>(C, xs, ss, ea); break;
        default: gatt_direct(A, SC, FF, cosf, base, lane, uu, kap, ea);
        }
        gat_finish<true>(A, base, lane, uu, ea, vin);
    }
}

// the tile-shape variants of the packed gather: (particles a lane, deep and short
// unrolling, launch bound)
#define GAT2_NVARIANTS 3

template <int NP, int UD, int US, int MINB>
static kde_status gat2_launch(kde_ctx *ctx, const GatherArgs<float> &A)
{
    auto kern = gather2_kernel<NP, UD, US, MINB>;
    static bool attr = false;
    if (!attr) {
        KDE_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           KDE_MAX_NG * (int)(sizeof(float4) + sizeof(float2))),
                 "gather2 attribute");
        attr = true;
    }
    const size_t smem = (size_t)A.Ng * (sizeof(float4) + sizeof(float2));
    unsigned grid = (unsigned)((A.N + GAT2_WARPS * 32 * NP - 1) / (GAT2_WARPS * 32 * NP));
    if (grid == 0) grid = 1;
    // with the push (the PIC step) the kernel before is the field kernel, which writes
    // none of the sorted particle arrays the prologue reads before its wait; a plain
    // gather may follow the sort that wrote them, so it starts after it as usual
    KDE_CUDA(ctx, kde_launch(ctx, A.u_out != nullptr, kern, dim3(grid), dim3(GAT2_WARPS * 32), smem, A),
             "gather2_kernel");
    KDE_LAUNCHED(ctx, "gather2_kernel");
    return KDE_OK;
}

static kde_status gat2_variant(kde_ctx *ctx, const GatherArgs<float> &A, int v)
{
    // all with four particles a lane: the warps' particle sets, and so their node windows
    // and kernel forms, are the same in every variant.  Launch bounds of 6, 7 and 8 blocks
    // an SM; the default 7 (71 registers) puts a Landau-size run (2048 blocks) in two
    // nearly full waves and measured best or within 1% of best from whole-grid to
    // five-node windows.  (Eight particles a lane, which makes a Landau-size run one
    // wave, measured 10% slower: the 64-register bound leaves the node loop less room.)
    switch (v) {
    case 1: return gat2_launch<4, 4, 4, 8>(ctx, A);
    case 2: return gat2_launch<4, 8, 4, 6>(ctx, A);
    default: return gat2_launch<4, 8, 4, 7>(ctx, A);
    }
}

// the gather through proxies: at the default truncation, in the PIC step (and its truncation
// tuner).  The rest -- particle-wise widths outside a schedule and cuts the caller has set -- sweeps
// the nodes (gather2_kernel)
// For one width the host knows the outcome: where the tiles would sweep the nodes anyway,
// gather2_kernel does it.
static int gatt_tile(kde_ctx *ctx, const GatherArgs<float> &A)
{
    // one wave of three CTAs an SM, whole rounds of 1024 particles, which spread the tile's
    // fixed steps (a warp's 128 particles stay in one tile of the sort).  Particle-wise widths,
    // whose tiles may sweep their nodes: shares of whole warps above 1024 particles, since whole rounds left
    // a quarter of the slots empty at 2^20 (50 steps with widths over a factor of three: 256 nodes 4.37
    // -> 4.18 ms, 1024 nodes 6.66 -> 6.08; one width on 512 nodes, which interpolates, 0.36 -> 0.38)
    const int64_t slots = 3LL * (ctx->sm_count > 0 ? ctx->sm_count : 1);
    const int64_t step = A.kappa && A.N > slots * GATT_UNIT ? 128 : GATT_UNIT;
    const int64_t units = (A.N + step - 1) / step;
    return (int)((units + slots - 1) / slots * step);
}
static bool gatt_applies(kde_ctx *ctx, GatherArgs<float> &A)
{
    if (A.xcut != (float)KDE_XCUT || !(A.kappa ? A.krange != nullptr : A.u_out != nullptr)) return false;
    A.tile = gatt_tile(ctx, A);
    // particle-wise widths: a range is given for those of a width schedule (Silverman's rule
    // around one width, a narrow range unless the density varies much).  Below 65,536 particles a wide
    // range's sweep by four times as many blocks would miss more than a narrow range's tiles spare: 50
    // steps on 256 nodes, tiles and gather2_kernel, narrow 49,152 1194 and 1376 us, 65,536 1224 and
    // 1466, 262,144 1346 and 1642; over a factor of three 1619 and 1461, 1701 and 1539, 1897 and 1776
    if (A.kappa) return A.N >= 64 * GATT_UNIT;
    const double n = (double)(A.N < A.tile ? A.N : A.tile), share = n / (double)A.N;
    const double a = KDE_PI * std::min(1.0, share + 2.0 / A.Ng), y = a * sqrt((double)A.kappa_u + 1.5);
    const double R = std::min((double)A.Ng, 2.0 * kde_window_nodes(A.kappa_u, A.Ng) + share * A.Ng + 2.0);
    return y < 1.6 && n * (y < 0.38 ? 26.0 : 33.0) + R * (y < 0.38 ? 40.0 : 80.0) + 60000.0 < n * 2.6 * R;
}

// Whether the step's gather is gather2_kernel with few blocks for the chip: launched while the field
// kernel's CTAs hold some SMs, its blocks crowd on the others, and where the windows are long that
// kernel should let it start only at its end: where the smallest width is at most the value returned (0:
// never).  Steps with widths over three decades (windows of the whole grid), started at once and at
// the end: 65,536 particles, 4096 nodes 215 and 181 us; 131,072, 1024 nodes 97 and 74; 262,144, 1024
// nodes 139 and 121; 131,072, 512 nodes 52.6 and 47.9, 256 nodes 36.5 and 35.2.  With blocks for less than half or for most
// of the chip, or shorter windows, it costs the 1 to 3 us of overlap: 16,384, 1024 nodes 50.0 and 52.0,
// 131,072, 4096 nodes 246 and 247, 262,144, 256 nodes 45.2 and 46.5; 60,000, 512 nodes 41 and 43;
// widths near 315 (windows of 55 nodes), 60,000, 512 nodes 26.3 and 29.2.
float kde_gather_crowds(kde_ctx *ctx, int64_t N, int Ng, bool per_particle, const unsigned int *krange, float xcut)
{
    if (!per_particle) return 0.f;  // one width: short windows, the others take tiles
    if (krange && xcut == (float)KDE_XCUT && N >= 64 * GATT_UNIT) return 0.f;
    const int64_t sms = ctx->sm_count > 0 ? ctx->sm_count : 1, blocks = (N + 511) / 512;
    const int64_t fit = std::min<int64_t>(7, 227 * 1024 / ((int64_t)Ng * (sizeof(float4) + sizeof(float2)) + 2064));
    if (2 * blocks <= sms || 2 * blocks > fit * sms) return 0.f;
    const int nodes = blocks < sms ? 768 : (blocks <= 2 * sms ? 256 : 384);  // the shortest window it is for
    if (Ng < nodes) return 0.f;
    const double s = sin(KDE_PI * nodes / (2.0 * Ng));
    return (float)((double)xcut * KDE_LN2 / (2.0 * s * s));
}

static kde_status gatt_launch(kde_ctx *ctx, GatherArgs<float> &A)
{
    static bool attr = false;
    if (!attr) {
        KDE_CUDA(ctx, cudaFuncSetAttribute(gather_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           KDE_MAX_NG * (int)(sizeof(float4) + sizeof(float2))),
                 "gather_tile attribute");
        attr = true;
    }
    const unsigned grid = (unsigned)((A.N + A.tile - 1) / A.tile) + (A.energy ? 1u : 0u);
    const size_t smem = (size_t)A.Ng * (sizeof(float4) + sizeof(float2));
    KDE_CUDA(ctx, kde_launch(ctx, A.u_out != nullptr, gather_tile_kernel, dim3(grid), dim3(GATT_THREADS), smem, A),
             "gather_tile_kernel");
    KDE_LAUNCHED(ctx, "gather_tile_kernel");
    return KDE_OK;
}

static uint64_t gat2_key(const GatherArgs<float> &A)
{
    return kde_width_key(A.N, A.Ng, A.kappa != nullptr, (double)A.kappa_u);
}

// the variant for this call: the tuned one for its key; with autotuning on and no stream
// capture, a key seen for the first time is tuned on this call's own data (every variant
// runs twice, timed by events on the stream, the fastest second run wins), provided that
// repeating the call cannot change its result (no output aliases an input)
static kde_status launch_gather2(kde_ctx *ctx, GatherArgs<float> &A)
{
    const void *nodes = kde_node_table(ctx, A.Ng, false);
    if (!nodes) return KDE_ENOMEM;
    A.nodes = (const float2 *)nodes;
    A.status = ctx->d_status;
    A.ntab = ctx->norm_tab;
    A.grid = pxy_grid(A.Ng);
    A.pxt = ctx->pxy_tab;
    const uint64_t key = gat2_key(A);
    if (gatt_applies(ctx, A)) {
        // one shape: nothing to tune, and the key counts as tuned with the default
        if (ctx->autotune) ctx->gat2_tuned.insert({key, 0});
        KdeProfScope _ps(ctx, PROF_GATHER);
        return gatt_launch(ctx, A);
    }
    auto it = ctx->gat2_tuned.find(key);
    int v = it != ctx->gat2_tuned.end() ? it->second : 0;
    bool tune = false;
    if (it == ctx->gat2_tuned.end() && ctx->autotune) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        cudaStreamIsCapturing(ctx->stream, &cap);
        auto apart = [](const void *out, const void *in) { return !out || out != in; };
        const bool idem = !A.u_out || (apart(A.u_out, A.u) && apart(A.v_out, A.v_in) && apart(A.kappa_out, A.kappa) &&
                                       apart(A.id_out, A.id_in));
        tune = cap == cudaStreamCaptureStatusNone && idem;
    }
    if (!tune) {
        KdeProfScope _ps(ctx, PROF_GATHER);
        return gat2_variant(ctx, A, v);
    }
    cudaEvent_t ev[2 * GAT2_NVARIANTS + 1];
    for (auto &e : ev) KDE_CUDA(ctx, cudaEventCreate(&e), "autotune event");
    KDE_CUDA(ctx, cudaEventRecord(ev[0], ctx->stream), "autotune event");
    // the timed runs add no sort counts (they repeat the gather); the chosen shape runs
    // once more below with the caller's arguments
    GatherArgs<float> T = A;
    T.counts = nullptr;
    for (int r = 0; r < 2; ++r)
        for (int k = 0; k < GAT2_NVARIANTS; ++k) {
            KDE_TRY(gat2_variant(ctx, T, k));
            KDE_CUDA(ctx, cudaEventRecord(ev[1 + r * GAT2_NVARIANTS + k], ctx->stream), "autotune event");
        }
    KDE_CUDA(ctx, cudaEventSynchronize(ev[2 * GAT2_NVARIANTS]), "autotune wait");
    float best = 3.0e38f;
    for (int k = 0; k < GAT2_NVARIANTS; ++k) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev[GAT2_NVARIANTS + k], ev[GAT2_NVARIANTS + k + 1]);
        if (ms < best) {
            best = ms;
            v = k;
        }
    }
    for (auto &e : ev) cudaEventDestroy(e);
    ctx->gat2_tuned[key] = v;
    if (A.counts) {
        KdeProfScope _ps(ctx, PROF_GATHER);
        return gat2_variant(ctx, A, v);
    }
    return KDE_OK;
}

static kde_status launch_gather64(kde_ctx *ctx, GatherArgs<double> &A)
{
    const void *nodes = kde_node_table(ctx, A.Ng, true);
    if (!nodes) return KDE_ENOMEM;
    A.nodes = (const double2 *)nodes;
    A.status = ctx->d_status;
    // particles a CTA: 32 until four CTAs an SM have 64, 128 when they have that many
    const int64_t per = A.N / (4LL * (ctx->sm_count > 0 ? ctx->sm_count : 1));
    KdeProfScope _ps(ctx, PROF_GATHER);
    if (per < 64) gather64_kernel<32><<<(unsigned)((A.N + 31) / 32), GAT_THREADS, 0, ctx->stream>>>(A, ctx->f64_tab);
    else if (per < 128) gather64_kernel<64><<<(unsigned)((A.N + 63) / 64), GAT_THREADS, 0, ctx->stream>>>(A, ctx->f64_tab);
    else gather64_kernel<128><<<(unsigned)((A.N + 127) / 128), GAT_THREADS, 0, ctx->stream>>>(A, ctx->f64_tab);
    KDE_LAUNCHED(ctx, "gather64_kernel");
    return KDE_OK;
}

template <typename T>
kde_status kde_gather_sorted(kde_ctx *ctx, const uint32_t *u, const T *kappa, T kappa_u, const T *norm, T norm_u,
                             int64_t N, const T *field, int Ng, double coef, T *out, const uint32_t *perm,
                             const PushArgs *push, float xcut, const unsigned int *krange)
{
    GatherArgs<T> A{};
    A.u = u;
    A.kappa = kappa;
    A.kappa_u = kappa_u;
    A.norm = norm;
    A.norm_u = norm_u;
    A.N = N;
    A.field = field;
    A.Ng = Ng;
    A.coef = (T)coef;
    A.out = out;
    A.perm = perm;
    A.xcut = xcut > 0.f ? xcut : (push && push->xcut > 0.f ? push->xcut : kde_fp32_cut(ctx));
    A.krange = push ? push->krange : krange;
    if (push) {
        A.v_in = (const T *)push->v_in;
        A.u_out = push->u_out;
        A.v_out = (T *)push->v_out;
        A.kappa_out = (T *)push->kappa_out;
        A.norm_in = (const T *)push->norm_in;
        A.norm_out = (T *)push->norm_out;
        A.id_in = push->id_in;
        A.id_out = push->id_out;
        A.kick_qm_dt = (T)(push->kick * push->qm_dt);
        A.dt_scale = (T)push->dt_scale;
        A.energy = push->energy;
        A.kstar_in = push->kstar_in;
        A.kstar_out = push->kstar_out;
        A.dx = push->dx;
        A.counts = push->counts;
        A.cnt_nblk = push->cnt_nblk;
        A.cnt_shift = push->cnt_shift;
    }
    if constexpr (sizeof(T) == 4) return launch_gather2(ctx, A);
    else return launch_gather64(ctx, A);
}

template kde_status kde_gather_sorted<float>(kde_ctx *, const uint32_t *, const float *, float, const float *, float,
                                             int64_t, const float *, int, double, float *, const uint32_t *,
                                             const PushArgs *, float, const unsigned int *);
template kde_status kde_gather_sorted<double>(kde_ctx *, const uint32_t *, const double *, double, const double *,
                                              double, int64_t, const double *, int, double, double *,
                                              const uint32_t *, const PushArgs *, float, const unsigned int *);

// ---------------------------------------------------------------------------
template <typename T>
static kde_status gather_api(kde_ctx *ctx, const uint32_t *u, const T *kappa, double kappa_u, int64_t N,
                             const T *field, int Ng, double L, T *out)
{
    cudaSetDevice(ctx->device);
    if constexpr (sizeof(T) == 4) {
        // at the default truncation from tables of the smoothed field, without a sort; a cut
        // the caller has set keeps the sweep over the nodes that it is defined for
        if (kde_fp32_cut(ctx) == (float)KDE_XCUT) {
            // no tile shapes to tune: the key counts as tuned with the default
            if (ctx->autotune) ctx->gat2_tuned.insert({kde_width_key(N, Ng, kappa != nullptr, kappa_u), 0});
            return kde_gather_table(ctx, u, kappa, kappa_u, N, field, Ng, out);
        }
    }
    uint32_t *us = (uint32_t *)kde_ws(ctx, WS_SORT_U, (size_t)N * 4);
    uint32_t *perm = (uint32_t *)kde_ws(ctx, WS_SORT_PERM, (size_t)N * 4);
    T *ks = kappa ? (T *)kde_ws(ctx, WS_SORT_P0, (size_t)N * sizeof(T)) : nullptr;
    if (!us || !perm || (kappa && !ks)) return KDE_ENOMEM;
    SortPayload pl[1];
    int npl = 0;
    if (kappa) pl[npl++] = SortPayload{kappa, ks, (int)sizeof(T)};
    KDE_TRY(kde_sort_by_bin(ctx, u, N, Ng, us, pl, npl, perm));
    double norm_u = kappa ? 0.0 : kde_norm(kappa_u);
    return kde_gather_sorted<T>(ctx, us, ks, (T)kappa_u, nullptr, (T)norm_u, N, field, Ng, KDE_TWO_PI / Ng, out, perm,
                                nullptr);
}

extern "C" kde_status kde_gather(kde_ctx *ctx, const uint32_t *u, const void *kappa, double kappa_uniform, int64_t N,
                                 const void *field, int32_t Ng, double L, void *out, uint32_t flags)
{
    if (!ctx) return KDE_EINVAL;
    if (N < 0 || Ng < 1 || Ng > KDE_MAX_NG || !(L > 0) || !field || (N > 0 && (!u || !out)))
        return kde_fail(ctx, KDE_EINVAL, "kde_gather: need N >= 0, 1 <= Ng <= %d, L > 0, non-null arrays",
                        KDE_MAX_NG);
    if (!kappa && !(kappa_uniform > 0 && kappa_uniform <= KDE_KAPPA_MAX))
        return kde_fail(ctx, KDE_EINVAL, "kde_gather: kappa_uniform must be in (0, 1e6]");
    if (N > 0xFFFFFFFFll) return kde_fail(ctx, KDE_EINVAL, "kde_gather: N must be below 2^32");
    if (flags & ~KDE_F64) return kde_fail(ctx, KDE_ENOTSUP, "kde_gather: unsupported flags 0x%x", flags);
    if (N == 0) return KDE_OK;
    if (flags & KDE_F64)
        return gather_api<double>(ctx, u, (const double *)kappa, kappa_uniform, N, (const double *)field, Ng, L,
                                  (double *)out);
    return gather_api<float>(ctx, u, (const float *)kappa, kappa_uniform, N, (const float *)field, Ng, L,
                             (float *)out);
}
