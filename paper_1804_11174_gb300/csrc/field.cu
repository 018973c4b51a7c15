// field.cu -- periodic Poisson solve and field energy.
//
// The solve is the circular convolution E_j = sum_l G[(j - l) mod Ng] rho'_l
// with the Green's function of ctx.cu (spectral symbol 1/(i k_m), or the
// finite-difference symbol of Sec. III.A); rho' is the total charge density
// with its mean removed in FP64 (G annihilates constants, and removing the
// mean first keeps the FP32 sum free of cancellation).  Ng <= 4096, so the
// whole grid lives in shared memory; each warp owns one output node, its lanes
// take every 32nd term and a shuffle tree adds them (Ng / 8 blocks of 8 warps).
#include "common.cuh"

#define POI_THREADS 256

template <typename T>
__global__ void __launch_bounds__(POI_THREADS)
    poisson_kernel(const T *rho, const long long *acc, double acc_inv, int Ng, double charge, double background,
                   const T *G, T *E)
{
    extern __shared__ __align__(16) unsigned char sm[];
    T *rt = (T *)sm;
    T *Gs = rt + Ng;
    __shared__ double red[POI_THREADS];
    auto value = [&](int l) -> double {
        if (!acc) return (double)rho[l];
        if (sizeof(T) == 8) return ((double)acc[l] + (double)acc[Ng + l] * (1.0 / 16777216.0)) * acc_inv;
        return (double)acc[l] * acc_inv;
    };
    double local = 0.0;
    for (int l = threadIdx.x; l < Ng; l += POI_THREADS) {
        double r = value(l);
        local += background + charge * r;
    }
    red[threadIdx.x] = local;
    __syncthreads();
    for (int o = POI_THREADS / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    const double mean = red[0] / Ng;
    for (int l = threadIdx.x; l < Ng; l += POI_THREADS) {
        double r = value(l);
        rt[l] = (T)(background + charge * r - mean);
        Gs[l] = G[l];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int j = blockIdx.x * (POI_THREADS / 32) + (threadIdx.x >> 5);
    if (j >= Ng) return;
    T s = 0;
    for (int l = lane; l < Ng; l += 32) {
        const int d = j - l;
        s += Gs[d < 0 ? d + Ng : d] * rt[l];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) E[j] = s;
}

// ---------------------------------------------------------------------------
// Field of the PIC step from the FP32 deposit's int64 node sums.  Every CTA loads all Ng sums,
// finds the grid total exactly (as sums of the upper and lower 32 bits, which cannot overflow),
// forms rho'_g = charge acc_inv (n_g - M) with M the mean to FP32 precision (the background is
// a constant and drops out; so does the tiny remainder of the mean, which the zero-sum Green's
// function annihilates) and convolves for its own nodes, a node a warp at a time.  No FP64,
// which is slow on this part, and no exchange between CTAs.  CTA 0 zeroes the other grid of
// sums for the next deposit.  Bound by latency: one round of loads, one block sum, Ng / 32
// products a lane; 8.7 us when it summed 456 rows in a cluster of eight CTAs, 3.9 us at 256
// nodes now.
// ---------------------------------------------------------------------------
#define FIELD_THREADS 256
#define FIELD_WARPS 8

__global__ void __launch_bounds__(FIELD_THREADS)
    field_sums_kernel(const long long *__restrict__ acc, long long *__restrict__ next, int Ng, int per, float scale62,
                      float inv_ng, const float *__restrict__ Gf, float *E, float late,
                      const unsigned int *krange)
{
    __shared__ float rt[KDE_MAX_NG];
    __shared__ float gs[KDE_MAX_NG];
    __shared__ long long red[2 * FIELD_WARPS];
    constexpr int PT = KDE_MAX_NG / FIELD_THREADS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool at_end = late > 0.f && __uint_as_float(krange[1]) <= late;  // written before the sort
    // the sums come from the deposit before, and on a grid's first use the Green's function from
    // a kernel launched between the two
    kde_pdl_wait();
    if (!at_end) kde_pdl_trigger();  // else the CTA's end triggers
    long long n[PT];
    float gv[PT];
    long long hi = 0, lo = 0;
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int g = tid + i * FIELD_THREADS;
        if (i * FIELD_THREADS >= Ng) break;
        n[i] = g < Ng ? __ldcg(&acc[g]) : 0;
        gv[i] = g < Ng ? __ldcg(&Gf[g]) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        if (i * FIELD_THREADS >= Ng) break;
        hi += n[i] >> 32;
        lo += n[i] & 0xffffffffll;
        const int g = tid + i * FIELD_THREADS;
        if (g < Ng) gs[g] = gv[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        hi += __shfl_xor_sync(0xffffffffu, hi, o);
        lo += __shfl_xor_sync(0xffffffffu, lo, o);
    }
    if (lane == 0) {
        red[warp] = hi;
        red[FIELD_WARPS + warp] = lo;
    }
    if (blockIdx.x == 0)
        for (int g = tid; g < Ng; g += FIELD_THREADS) next[g] = 0;
    __syncthreads();
    hi = lo = 0;
#pragma unroll
    for (int w = 0; w < FIELD_WARPS; ++w) {
        hi += red[w];
        lo += red[FIELD_WARPS + w];
    }
    const long long mean = __float2ll_rn(fmaf(__ll2float_rn(hi), 4294967296.f, __ll2float_rn(lo)) * inv_ng);
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int g = tid + i * FIELD_THREADS;
        if (i * FIELD_THREADS >= Ng) break;
        // (n_g - M) charge acc_inv as (n_g - M) 2^-62 (exact) times charge acc_inv 2^62
        if (g < Ng) rt[g] = __ll2float_rn(n[i] - mean) * 0x1p-62f * scale62;
    }
    __syncthreads();
    // E_j = sum_l G[(j - l) mod Ng] rho'_l
    const int j1 = min(Ng, (int)(blockIdx.x + 1) * per);
    for (int j = blockIdx.x * per + warp; j < j1; j += FIELD_WARPS) {
        float s = 0.f;
#pragma unroll 4
        for (int l = lane; l < Ng; l += 32) {
            const int d = j - l;
            s = fmaf(gs[d < 0 ? d + Ng : d], rt[l], s);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) E[j] = s;
    }
}

kde_status kde_field_from_sums(kde_ctx *ctx, const DepSums &ds, int Ng, double L, double acc_inv, double charge, bool fd,
                               float *E_out, float late, const unsigned int *krange)
{
    const float *Gf = (const float *)kde_green_table(ctx, Ng, L, fd, false);
    if (!Gf) return KDE_ENOMEM;
    // a node a warp up to one CTA an SM, more beyond (every CTA loads the whole grid)
    const int sms = ctx->sm_count > 0 ? ctx->sm_count : 1;
    int per = FIELD_WARPS;
    while ((Ng + per - 1) / per > sms) per += FIELD_WARPS;
    {
        KdeProfScope _ps(ctx, PROF_POISSON);
        KDE_CUDA(ctx, kde_launch(ctx, true, field_sums_kernel, dim3((Ng + per - 1) / per), dim3(FIELD_THREADS), 0,
                                 (const long long *)ds.acc, ds.next, Ng, per, (float)(charge * acc_inv * 0x1p62),
                                 1.f / (float)Ng, Gf, E_out, krange ? late : 0.f, krange),
                 "field_sums_kernel");
    }
    KDE_LAUNCHED(ctx, "field_sums_kernel");
    ctx->sums_ng = Ng;
    return KDE_OK;
}

template <typename T>
__global__ void energy_kernel(const T *E, int Ng, double dx, double *out)
{
    __shared__ double red[256];
    double s = 0.0;
    for (int g = threadIdx.x; g < Ng; g += 256) s += (double)E[g] * (double)E[g];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = 0.5 * red[0] * dx;
}

template <typename T>
kde_status kde_poisson_impl(kde_ctx *ctx, const T *rho, const long long *acc, double acc_inv, int Ng, double L,
                            double charge, double background, bool fd, T *E_out)
{
    const T *G = (const T *)kde_green_table(ctx, Ng, L, fd, sizeof(T) == 8);
    if (!G) return KDE_ENOMEM;
    size_t smem = (size_t)2 * Ng * sizeof(T);
    static bool attr[2] = {false, false};
    if (!attr[sizeof(T) == 8]) {
        cudaFuncSetAttribute(poisson_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             2 * KDE_MAX_NG * (int)sizeof(T));
        attr[sizeof(T) == 8] = true;
    }
    {
        KdeProfScope _ps(ctx, PROF_POISSON);
    poisson_kernel<T><<<(Ng + POI_THREADS / 32 - 1) / (POI_THREADS / 32), POI_THREADS, smem, ctx->stream>>>(
        rho, acc, acc_inv, Ng, charge, background, G, E_out);
    }
    KDE_LAUNCHED(ctx, "poisson_kernel");
    return KDE_OK;
}

template <typename T>
kde_status kde_energy_impl(kde_ctx *ctx, const T *E, int Ng, double L, double *energy_out)
{
    energy_kernel<T><<<1, 256, 0, ctx->stream>>>(E, Ng, L / Ng, energy_out);
    KDE_LAUNCHED(ctx, "energy_kernel");
    return KDE_OK;
}

template kde_status kde_poisson_impl<float>(kde_ctx *, const float *, const long long *, double, int, double, double,
                                            double, bool, float *);
template kde_status kde_poisson_impl<double>(kde_ctx *, const double *, const long long *, double, int, double,
                                             double, double, bool, double *);
template kde_status kde_energy_impl<float>(kde_ctx *, const float *, int, double, double *);
template kde_status kde_energy_impl<double>(kde_ctx *, const double *, int, double, double *);

extern "C" kde_status kde_poisson(kde_ctx *ctx, const void *rho, int32_t Ng, double L, double charge,
                                  double background, void *E_out, double *energy_out, uint32_t flags)
{
    if (!ctx) return KDE_EINVAL;
    if (Ng < 1 || Ng > KDE_MAX_NG || !(L > 0) || !rho || !E_out || rho == E_out)
        return kde_fail(ctx, KDE_EINVAL, "kde_poisson: need 1 <= Ng <= %d, L > 0, distinct non-null arrays",
                        KDE_MAX_NG);
    if (flags & ~(KDE_F64 | KDE_POISSON_FD))
        return kde_fail(ctx, KDE_ENOTSUP, "kde_poisson: unsupported flags 0x%x", flags);
    cudaSetDevice(ctx->device);
    bool fd = (flags & KDE_POISSON_FD) != 0;
    if (flags & KDE_F64) {
        KDE_TRY(kde_poisson_impl<double>(ctx, (const double *)rho, nullptr, 0.0, Ng, L, charge, background, fd,
                                         (double *)E_out));
        if (energy_out) KDE_TRY(kde_energy_impl<double>(ctx, (const double *)E_out, Ng, L, energy_out));
    } else {
        KDE_TRY(kde_poisson_impl<float>(ctx, (const float *)rho, nullptr, 0.0, Ng, L, charge, background, fd,
                                        (float *)E_out));
        if (energy_out) KDE_TRY(kde_energy_impl<float>(ctx, (const float *)E_out, Ng, L, energy_out));
    }
    return KDE_OK;
}
