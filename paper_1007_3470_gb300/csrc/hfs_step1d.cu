// hfs_step1d.cu -- the generic instantiations of the fused 1D step kernel
// (FP32 and FP64, perturbation kind and box symmetry read per instance), the
// launch dispatcher over the specialised FP32 variants, the norm / energy
// diagnostics and the twiddle tables.
#include "hfs_step1d.cuh"

namespace hfs {

HFS_STEP1D_VARIANT(, float, -1, false)
HFS_STEP1D_VARIANT(, double, -1, false)
HFS_STEP1D_VARIANT(extern, float, HFS_VI_NONE, false)
HFS_STEP1D_VARIANT(extern, float, HFS_VI_X4, false)
HFS_STEP1D_VARIANT(extern, float, HFS_VI_COS, false)
HFS_STEP1D_VARIANT(extern, float, -1, true)
HFS_STEP1D_VARIANT(extern, float, HFS_VI_NONE, true)
HFS_STEP1D_VARIANT(extern, float, HFS_VI_X4, true)
HFS_STEP1D_VARIANT(extern, float, HFS_VI_COS, true)

// ---------------------------------------------------------------------------
// diagnostics: norm and energy (FP64 accumulation)
// ---------------------------------------------------------------------------
template <typename R, int N, int E, bool ALT>
__device__ __forceinline__ void diag_item(const Diag1DArgs &a, const WorkItem &it, cpx<R> *smem)
{
    constexpr int T = N / E;
    const int g = threadIdx.x / T;
    const int t = threadIdx.x - g * T;
    const bool active = g < it.count;
    const int idx = a.order[it.first + (active ? g : 0)];
    const DevInst &ip = a.inst[idx];
    const cpx<R> *psi = reinterpret_cast<const cpx<R> *>(a.psi) + ip.off;
    cpx<R> *sm = smem + g * smem_elems(N);
    const auto *tw = reinterpret_cast<const typename TwOf<R>::type *>(a.tw);
    const double w2 = law_omega2(ip, *a.t_dev);
    cpx<R> v[E];
    double nrm = 0.0, pot = 0.0, inter = 0.0, kin = 0.0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        v[e] = active ? psi[t + T * e] : cpx<R>{R(0), R(0)};
        const double x = ip.xc[0] + (double)(t + T * e - N / 2) * ip.dx[0];
        const double d = (double)v[e].x * v[e].x + (double)v[e].y * v[e].y;
        nrm += d;
        pot += (0.5 * ip.mu * w2 * x * x + ip.eps * vi_eval(ip.vi_kind, x, ip.vi_k)) * d;
        inter += 0.5 * ip.sigma * d * d;
    }
    FftPlan<N, E, ALT>::template run<false, R>(v, sm, t, tw);
    const double kunit = 2.0 * 3.14159265358979323846 / ip.len[0];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int k = t + T * e;
        const double kk = kunit * (double)((k < N / 2) ? k : k - N);
        kin += kk * kk * ((double)v[e].x * v[e].x + (double)v[e].y * v[e].y);
    }
    const double energy = kin / N / (2.0 * ip.mu) + pot + inter;
    __syncthreads();
    double *red = reinterpret_cast<double *>(smem);
    red[2 * threadIdx.x] = nrm;
    red[2 * threadIdx.x + 1] = energy;
    __syncthreads();
    if (active && t == 0) {
        double sn = 0.0, se = 0.0;
        for (int u = 0; u < T; ++u) {
            sn += red[2 * (threadIdx.x + u)];
            se += red[2 * (threadIdx.x + u) + 1];
        }
        a.out[2 * idx] = sn * ip.dx[0];
        a.out[2 * idx + 1] = se * ip.dx[0];
    }
    __syncthreads();
}

template <typename R> __global__ void __launch_bounds__(kCtaThreads) diag1d_kernel(const Diag1DArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<R> *smem = reinterpret_cast<cpx<R> *>(smem_raw);
    __shared__ int s_item;
    for (;;) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(a.ticket, 1u);
        __syncthreads();
        const int w = s_item;
        if (w >= a.nwork) break;
        const WorkItem it = a.work[w];
        switch (it.plan) {
#define HFS_CASE(NN, EE, AA)                                                                                      \
    case plan_id(NN, EE, AA):                                                                                     \
        diag_item<R, NN, EE, AA>(a, it, smem);                                                                    \
        break;
            HFS_FOR_EACH_PLAN(HFS_CASE)
            HFS_FOR_EACH_WIDE_PLAN(HFS_CASE)
#undef HFS_CASE
        default:
            break;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// twiddle tables (layout: tw_pass_offset), computed in FP64: entry
// (r - 1) NS + j of region (L, R) is exp(-2 pi i j r / L)
__global__ void twiddle_kernel(float4 *tf, double2 *td)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= kTwiddleTotal) return;
    int L = 4;
    while (i >= tw_pass_offset(2 * L, 2)) L <<= 1;
    int R = 2;
    while (R < 16 && i >= tw_pass_offset(L, 2 * R)) R <<= 1;
    const int64_t s = i - tw_pass_offset(L, R);
    const int NS = L / R;
    const int64_t r = s / NS + 1, j = s % NS;
    double sn, cs;
    sincospi(2.0 * (double)(j * r) / (double)L, &sn, &cs);
    td[i] = make_double2(cs, -sn);
    const float ch = (float)cs, sh = (float)-sn;
    tf[i] = make_float4(ch, sh, (float)(cs - (double)ch), (float)(-sn - (double)sh));
}

__global__ void twiddle_plain_kernel(float2 *tp)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= kTwiddleTotal) return;
    int L = 4;
    while (i >= tw_pass_offset(2 * L, 2)) L <<= 1;
    int R = 2;
    while (R < 16 && i >= tw_pass_offset(L, 2 * R)) R <<= 1;
    const int64_t s = i - tw_pass_offset(L, R);
    const int NS = L / R;
    const int64_t r = s / NS + 1, j = s % NS;
    double sn, cs;
    sincospi(2.0 * (double)(j * r) / (double)L, &sn, &cs);
    tp[i] = make_float2((float)cs, (float)-sn);
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
size_t step1d_smem_bytes(bool fp64)
{
    const size_t r = fp64 ? sizeof(double) : sizeof(float);
    return ((size_t)2 * step1d_exchange_elems + step1d_vtable_elems) * r + step1d_slot_floats * sizeof(float);
}

static cudaError_t prepare_diag(bool fp64)
{
    static bool done[2] = {false, false};
    if (done[fp64]) return cudaSuccess;
    const int bytes = (int)step1d_smem_bytes(fp64);
    const cudaError_t e =
        fp64 ? cudaFuncSetAttribute(diag1d_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)
             : cudaFuncSetAttribute(diag1d_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done[fp64] = true;
    return e;
}

template <bool WIDE> static int ctas_per_sm_f(int variant)
{
    switch (variant) {
    case HFS_VI_NONE: return step1d_ctas_per_sm_t<float, HFS_VI_NONE, WIDE>();
    case HFS_VI_X4: return step1d_ctas_per_sm_t<float, HFS_VI_X4, WIDE>();
    case HFS_VI_COS: return step1d_ctas_per_sm_t<float, HFS_VI_COS, WIDE>();
    default: return step1d_ctas_per_sm_t<float, -1, WIDE>();
    }
}

int step1d_ctas_per_sm(bool fp64, int variant, bool wide)
{
    if (fp64) return step1d_ctas_per_sm_t<double, -1, false>();
    return wide ? ctas_per_sm_f<true>(variant) : ctas_per_sm_f<false>(variant);
}

template <bool WIDE>
static cudaError_t launch_f(int variant, const Step1DArgs &a, int grid, cudaStream_t st, int prio)
{
    switch (variant) {
    case HFS_VI_NONE: return step1d_launch_t<float, HFS_VI_NONE, WIDE>(a, grid, st, prio);
    case HFS_VI_X4: return step1d_launch_t<float, HFS_VI_X4, WIDE>(a, grid, st, prio);
    case HFS_VI_COS: return step1d_launch_t<float, HFS_VI_COS, WIDE>(a, grid, st, prio);
    default: return step1d_launch_t<float, -1, WIDE>(a, grid, st, prio);
    }
}

cudaError_t launch_step1d(bool fp64, int variant, const Step1DArgs &a, int grid, cudaStream_t st, bool wide,
                          int priority)
{
    if (fp64) return wide ? cudaErrorInvalidValue : step1d_launch_t<double, -1, false>(a, grid, st, priority);
    return wide ? launch_f<true>(variant, a, grid, st, priority) : launch_f<false>(variant, a, grid, st, priority);
}

int step1d_variant(const hfs_instance *inst, int64_t count)
{
    // the perturbation kind each instance's team uses (none where eps = 0)
    auto kind = [](const hfs_instance &p) { return p.eps != 0.0 ? p.vi_kind : HFS_VI_NONE; };
    if (count < 1) return -1;
    const int k = kind(inst[0]);
    if (k != HFS_VI_NONE && k != HFS_VI_X4 && k != HFS_VI_COS) return -1;
    for (int64_t i = 0; i < count; ++i) {
        // same box centre expression as the device instance record
        if (0.5 * (inst[i].lo[0] + inst[i].hi[0]) != 0.0 || kind(inst[i]) != k) return -1;
    }
    return k;
}

cudaError_t launch_diag1d(bool fp64, const Diag1DArgs &a, int grid, cudaStream_t st)
{
    cudaError_t e = prepare_diag(fp64);
    if (e != cudaSuccess) return e;
    const size_t bytes = step1d_smem_bytes(fp64);
    if (fp64) diag1d_kernel<double><<<grid, kCtaThreads, bytes, st>>>(a);
    else diag1d_kernel<float><<<grid, kCtaThreads, bytes, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_twiddles_plain(void *tw_p, cudaStream_t st)
{
    twiddle_plain_kernel<<<(unsigned)((kTwiddleTotal + 255) / 256), 256, 0, st>>>((float2 *)tw_p);
    return cudaGetLastError();
}

cudaError_t launch_twiddles(void *tw_f, void *tw_d, cudaStream_t st)
{
    twiddle_kernel<<<(unsigned)((kTwiddleTotal + 255) / 256), 256, 0, st>>>((float4 *)tw_f, (double2 *)tw_d);
    return cudaGetLastError();
}

}  // namespace hfs
