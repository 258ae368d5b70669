// hfs_step1d.cu -- the generic instantiations of the fused 1D step kernel
// (FP32 and FP64, perturbation kind and box symmetry read per instance), the
// launch dispatcher over the specialised FP32 variants, the norm / energy
// diagnostics and the twiddle tables.
#include <algorithm>

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
// the sum over a team's threads (teams of T threads are aligned): in shuffles,
// then the team's warps through slots
template <int T> __device__ __forceinline__ double team_sum(double s, double *slots)
{
    constexpr int W = T < 32 ? T : 32;
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if constexpr (T > 32) {
        const int bar = 1 + threadIdx.x / T, w0 = (threadIdx.x / T) * (T / 32);
        exchange_sync<T, true>(bar);
        if ((threadIdx.x & 31) == 0) slots[threadIdx.x >> 5] = s;
        exchange_sync<T, true>(bar);
        s = 0.0;
#pragma unroll
        for (int w = 0; w < T / 32; ++w) s += slots[w0 + w];
    }
    return s;
}

// Norm alone: one pass over the state, bound by the FP64 pipe (two FMAs and two
// conversions a point at 2 lanes a cycle) a little above the memory time.
template <typename R, int T, int E>
__device__ __forceinline__ void norm_item(const Diag1DArgs &a, const WorkItem &it, double *slots)
{
    const int g = threadIdx.x / T, t = threadIdx.x - g * T;
    const bool active = g < it.count;
    const int idx = a.order[it.first + (active ? g : 0)];
    const DevInst &ip = a.inst[idx];
    const cpx<R> *psi = reinterpret_cast<const cpx<R> *>(a.psi) + ip.off;
    double s = 0.0;
    if (active) {
        cpx<R> v[E];
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = psi[t + T * e];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const double x = v[e].x, y = v[e].y;
            s = fma(x, x, fma(y, y, s));
        }
    }
    s = team_sum<T>(s, slots);
    if (active && t == 0) a.out[2 * idx] = s * ip.dx[0];
}

// FP32 pairs hi + lo: sum += m2 |v|^2, every product and the sum exact to 2^-48
struct Sum2 {
    float hi = 0.0f, lo = 0.0f;
};
__device__ __forceinline__ void add_m2_abs2(Sum2 &s, float m2, cpx<float> v)
{
    const float p = v.x * v.x, q = v.y * v.y;
    const float pq = p + q, bb = pq - p;
    const float lo = (p - (pq - bb)) + (q - bb) + fmaf(v.x, v.x, -p) + fmaf(v.y, v.y, -q);
    const float t = m2 * pq;
    const float tl = fmaf(m2, lo, fmaf(m2, pq, -t));
    const float h = s.hi + t, hb = h - s.hi;
    s.lo += (s.hi - (h - hb)) + (t - hb) + tl;
    s.hi = h;
}

// Energy.  Bound by the FP64 pipe: the potential's sum takes eight FP64
// instructions a point (cos k x by c_{e+1} = 2 cos(k T dx) c_e - c_{e-1} over the
// thread's points instead of cos; its error of some E^2 roundings is far below
// the transform's), the kinetic sum of an FP32 state is formed in FP32 pairs.
// 4096 mixed-size FP32 instances: norm and energy took 1.19 ms together (0.32 ms
// now, copies included) as two runs of one kernel with cos and all sums in FP64.
template <typename R, int N, int E, bool ALT>
__device__ __forceinline__ void energy_item(const Diag1DArgs &a, const WorkItem &it, cpx<R> *smem, double *slots)
{
    constexpr int T = N / E;
    const int g = threadIdx.x / T;
    const int t = threadIdx.x - g * T;
    const bool active = g < it.count;
    if ((threadIdx.x & ~31) / T >= it.count) return;  // no instance in this warp
    const int idx = a.order[it.first + (active ? g : 0)];
    const DevInst &ip = a.inst[idx];
    const cpx<R> *psi = reinterpret_cast<const cpx<R> *>(a.psi) + ip.off;
    cpx<R> *sm = smem + g * smem_elems(N);
    const auto *tw = reinterpret_cast<const typename TwOf<R>::type *>(a.tw);
    cpx<R> v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = active ? psi[t + T * e] : cpx<R>{R(0), R(0)};
    double pot = 0.0;
    if (active) {
        const StageFGE pre = a.pre[idx];
        const double c2 = pre.f, hs = 0.5 * ip.sigma, step = T * ip.dx[0];
        const int kind = ip.eps != 0.0 ? ip.vi_kind : HFS_VI_NONE;
        double x = ip.xc[0] + (double)(t - N / 2) * ip.dx[0];
        double c = 0.0, cn = 0.0, f = 0.0;
        if (kind == HFS_VI_COS) {
            double sn, cs;
            sincos(ip.vi_k * x, &sn, &cs);
            f = 2.0 * pre.g;
            c = ip.eps * cs;
            cn = ip.eps * (cs * pre.g - sn * pre.e);
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const double vx = v[e].x, vy = v[e].y;
            const double d = fma(vx, vx, vy * vy), xx = x * x;
            double w = fma(hs, d, c2 * xx);
            if (kind == HFS_VI_COS) {
                w += c;
                const double next = fma(f, cn, -c);
                c = cn;
                cn = next;
            } else if (kind == HFS_VI_X4) {
                w = fma(ip.eps * xx, xx, w);
            }
            pot = fma(w, d, pot);
            x += step;
        }
    }
    FftPlan<N, E, ALT>::template run<false, R, 1, true>(v, sm, t, tw, 1 + g);
    const double ku = 2.0 * 3.14159265358979323846 / ip.len[0], ck = ku * ku / N / (2.0 * ip.mu);
    bool pairs = sizeof(R) == 4;
    double s = 0.0;
    if constexpr (sizeof(R) == 4) {
        Sum2 kin;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const float m = (float)(t + T * e - (2 * e < E ? 0 : N));
            add_m2_abs2(kin, m * m, v[e]);
        }
        s = team_sum<T>((double)kin.hi + (double)kin.lo, slots);
        // pairs hold 48 bits while squares stay clear of FP32's range; a state of
        // another size (or not finite) is summed in FP64
        pairs = !active || (s > 1e-18 && s < 1e30);
        if constexpr (T < 32) pairs = __all_sync(0xffffffffu, pairs);
    }
    if (!pairs) {
        double kin = 0.0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int m = t + T * e - (2 * e < E ? 0 : N);
            const double vx = v[e].x, vy = v[e].y;
            kin = fma(square64(m), fma(vx, vx, vy * vy), kin);
        }
        s = team_sum<T>(kin, slots);
    }
    s = fma(s, ck, team_sum<T>(pot, slots));
    if (active && t == 0) a.out[2 * idx + 1] = s * ip.dx[0];
}

// What every thread of an instance needs, once per instance: mu omega^2 / 2 and
// cos, sin of k T dx (with the law's sine and this sincos in every thread the two
// calls took 0.34 ms)
__global__ void energy_pre_kernel(const Diag1DArgs a)
{
    const int w = blockIdx.x, i = threadIdx.x;
    const WorkItem it = a.work[w];
    if (i >= it.count) return;
    const int idx = a.order[it.first + i];
    const DevInst &ip = a.inst[idx];
    StageFGE r{};
    r.f = 0.5 * ip.mu * law_omega2(ip, *a.t_dev);
    sincos(ip.vi_k * (ip.dx[0] * (ip.n[0] / plan_ept(it.diag))), &r.e, &r.g);
    a.pre[idx] = r;
}

// items of a batch hold about the same number of points each, so CTAs take them
// in turn
template <typename R, bool ENERGY> __global__ void __launch_bounds__(kCtaThreads) diag1d_kernel(const Diag1DArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<R> *smem = reinterpret_cast<cpx<R> *>(smem_raw);
    __shared__ double slots[kCtaThreads / 32];
    for (int w = blockIdx.x; w < a.nwork; w += gridDim.x) {
        const WorkItem it = a.work[w];
        switch (it.diag) {
#define HFS_CASE(NN, EE, AA)                                                                                      \
    case plan_id(NN, EE, AA):                                                                                     \
        if constexpr (ENERGY) energy_item<R, NN, EE, AA>(a, it, smem, slots);                                      \
        else norm_item<R, NN / EE, EE>(a, it, slots);                                                             \
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

template <typename R, bool ENERGY> static cudaError_t diag_t(const Diag1DArgs &a, int sms, cudaStream_t st)
{
    // the exchange buffers of the step kernels without the table behind them
    const int bytes = ENERGY ? (int)(step1d_exchange_elems * sizeof(cpx<R>)) : 0;
    static int per_sm = 0;
    if (!per_sm) {
        cudaError_t e = cudaFuncSetAttribute(diag1d_kernel<R, ENERGY>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        int n = 0;
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, diag1d_kernel<R, ENERGY>, kCtaThreads, bytes);
        if (e != cudaSuccess) return e;
        per_sm = std::max(1, n);
    }
    if (ENERGY) energy_pre_kernel<<<a.nwork, 64, 0, st>>>(a);  // at most 64 instances an item
    diag1d_kernel<R, ENERGY><<<std::max(1, std::min(a.nwork, sms * per_sm)), kCtaThreads, bytes, st>>>(a);
    return cudaGetLastError();
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

cudaError_t launch_diag1d(bool fp64, bool energy, const Diag1DArgs &a, int sms, cudaStream_t st)
{
    if (fp64) return energy ? diag_t<double, true>(a, sms, st) : diag_t<double, false>(a, sms, st);
    return energy ? diag_t<float, true>(a, sms, st) : diag_t<float, false>(a, sms, st);
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
