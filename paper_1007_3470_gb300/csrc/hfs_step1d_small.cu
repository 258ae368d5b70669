// hfs_step1d_small.cu -- the 1D step of few complex64 instances, where a call
// waits on latencies: the chain of exchanges and phases of one instance, the
// fetch of code that a call of one step runs through once, and the launches of
// the schedule before it.
//
// One CTA takes one instance, up to 1024 points with four values a thread: the
// transforms and phases of the plans with sixteen values a thread, on four times the threads and with the
// same bits (lane_fft; the norm projection alone sums in another order and reads
// the compensated twiddles).  The twiddles stay in registers over all steps and
// the next sub-stage's record is loaded a sub-stage ahead.  A short call's
// records are computed by the CTA itself and the last CTA advances the device
// time: one launch in place of six.  One instance: a call of one step of 1024
// points 36.2 -> 13.9 us, 1000 steps of 256 points 2.69 -> 0.86 ms (1.93 ms in the
// batch kernel without idle warps); 1200 instances of 128 points, 100 steps: 316
// -> 152 us.  (Plain radix-4 transforms on the same threads: 0.77 ms, but other
// roundings, which strongly nonlinear runs amplify beyond 1e-4.)
#include "hfs_schedule.cuh"
#include "hfs_step1d.cuh"

namespace hfs {

namespace {

constexpr int kSmallMaxN = 1024, kBigMaxN = 4096;

template <bool BIG> constexpr size_t small_smem()
{
    constexpr int n = BIG ? kBigMaxN : kSmallMaxN;
    return (size_t)smem_elems(n) * sizeof(cpx<float>) + (size_t)n * sizeof(float);
}

// records of sub-stages 0 .. nstage of one instance
template <int FLOW> __device__ void small_flows(const DevInst &p, const SchedConst &sc, double t0, int nstage, StageFGE *out,
                                                unsigned *status)
{
    for (int s = threadIdx.x; s < nstage; s += 32) {
        const int n = s / sc.m, st = s - n * sc.m;
        const double tau = t0 + (double)n * sc.h + sc.h * sc.cuma[st];
        const double w = sc.a[st] * sc.h;
        StageFGE r{};
        stage_fge<FLOW>(p, 1, 0, stage_nodes<FLOW, -1>(p, tau, w), w, r.f, r.g, r.e);
        if (!isfinite(r.f) || !isfinite(r.g) || !isfinite(r.e)) atomicOr(status, (unsigned)ST_NONFINITE);
        out[s] = r;
    }
}
__device__ __noinline__ void small_records(const DevInst &p, const SchedConst &sc, double t0, int nstage, StageFGE *fge,
                                           RecF *rec, unsigned *status)
{
    if (threadIdx.x >= 32) return;
    if (sc.split == HFS_SPLIT_HO) {
        if (sc.flow == HFS_FLOW_CF4) small_flows<HFS_FLOW_CF4>(p, sc, t0, nstage, fge, status);
        else if (sc.flow == HFS_FLOW_LEMMA2) small_flows<HFS_FLOW_LEMMA2>(p, sc, t0, nstage, fge, status);
        else small_flows<HFS_FLOW_M6>(p, sc, t0, nstage, fge, status);
        __syncwarp();
    }
    const RecScale c = rec_scale(p, sc);
    for (int j = threadIdx.x; j <= nstage; j += 32) {
        if (sc.split == HFS_SPLIT_HO) record1d<RecF, HFS_SPLIT_HO>(p, sc, c, t0, j, nstage, fge, rec + j, status);
        else record1d<RecF, HFS_SPLIT_FOURIER>(p, sc, c, t0, j, nstage, fge, rec + j, status);
    }
}

template <int N, bool PROJ>
__device__ __forceinline__ void small_item(const Step1DArgs &a, int idx, const RecF *rec, cpx<float> *sm, float *vtab,
                                           float *slots)
{
    constexpr int T = N / 4, T16 = N / 16, E = 4;
    if (threadIdx.x >= T) return;
    const int q = threadIdx.x & 3, b = threadIdx.x >> 2, t = b + T16 * q;  // see lane_fft
    const DevInst &ip = a.inst[idx];
    const TeamParams<float> tp = team_params<float>(ip);
    cpx<float> *psi = reinterpret_cast<cpx<float> *>(a.psi) + ip.off;
    const float4 *tw = reinterpret_cast<const float4 *>(a.tw);
    cpx<float> v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = ld_state(psi + t + T * e, a.streaming);
    // eps V_I as the plans with sixteen values a thread form it
    if (threadIdx.x < T16) vi_table<N, 16, -1>(vtab, threadIdx.x, tp);
    exchange_sync<T, true, true>(1);
    float target = 0.0f;
    if constexpr (PROJ) {
        if (a.proj == PROJ_USE) target = a.norm_target[idx];
    }
    RecF rc = rec[a.j0];
    for (int64_t j = a.j0; j < a.j1; ++j) {
        const RecF next = rec[j + 1];
        float dsum = 0.0f;
        xphase<N, E, -1>(v, t, rc, tp, vtab, dsum);
        if constexpr (PROJ) dsum = team_sum_begin<T>(dsum, slots);
        lane_fft<N, false>(v, sm, b, q, tw);
        float C = 1.0f;
        if constexpr (PROJ) {
            const float s = team_sum_end<T>(dsum, slots, 0);
            if (j == a.j0 && a.proj == PROJ_SET) {
                target = s;
                if (t == 0) a.norm_target[idx] = s;
            } else if (target > 0.0f && s > 0.0f && isfinite(s)) {
                C = sqrtf(target / s);
            }
        }
        kphase<N, E, PROJ>(v, t, rc, C);
        lane_fft<N, true>(v, sm, b, q, tw);
        rc = next;
    }
    if (a.final_x) {
        float dsum = 0.0f;
        xphase<N, E, -1>(v, t, rc, tp, vtab, dsum);
    }
    bool bad = false;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        st_state(psi + t + T * e, v[e], a.streaming);
        bad |= !(isfinite(v[e].x) && isfinite(v[e].y));
    }
    if (bad) atomicOr(a.status, (unsigned)ST_NONFINITE);
}

// 2048 points: eight values a thread or, under the projection, sixteen; 4096:
// sixteen, as default_ept for the batch kernel (with four, 512 and 1024 threads of 64
// registers, 4096 points took 11.8 us a step; 4.5 here)
template <int N, int E, bool PROJ, int VI>
__device__ __forceinline__ void big_item(const Step1DArgs &a, int idx, const RecF *rec, cpx<float> *sm, float *vtab,
                                         float *slots)
{
    constexpr int T = N / E;
    static_assert(T <= kCtaThreads, "one CTA is the team");
    if (threadIdx.x >= T) return;
    const DevInst &ip = a.inst[idx];
    const TeamParams<float> tp = team_params<float>(ip);
    cpx<float> *psi = reinterpret_cast<cpx<float> *>(a.psi) + ip.off;
    const float4 *tw = reinterpret_cast<const float4 *>(a.tw);
    const int t = threadIdx.x;
    cpx<float> v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = ld_state(psi + t + T * e, a.streaming);
    vi_table<N, E, VI>(vtab, t, tp);
    step_loop<float, VI, N, E, false, PROJ>(a, v, t, 0, true, idx, rec, tp, sm, tw, vtab, slots);
    bool bad = false;
    if (a.final_x) {
        float dsum = 0.0f;
        xphase<N, E, VI>(v, t, rec[a.j1], tp, vtab, dsum);
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
        st_state(psi + t + T * e, v[e], a.streaming);
        bad |= !(isfinite(v[e].x) && isfinite(v[e].y));
    }
    if (bad) atomicOr(a.status, (unsigned)ST_NONFINITE);
}

// VI: as step1d_kernel (the larger sizes alone gain from the fixed kind: 5 %)
template <bool PROJ, bool BIG, int VI>
__global__ void __launch_bounds__(kCtaThreads, 1) small1d_kernel(const Small1DArgs s)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<float> *sm = reinterpret_cast<cpx<float> *>(smem_raw);
    float *vtab = reinterpret_cast<float *>(sm + smem_elems(BIG ? kBigMaxN : kSmallMaxN));
    __shared__ float slots[kCtaThreads / 32];
    __shared__ RecF s_rec[kSmallSchedStages + 1];
    __shared__ StageFGE s_fge[kSmallSchedStages];
    const Step1DArgs &a = s.a;
    const int idx = a.order[blockIdx.x];
    const RecF *rec = reinterpret_cast<const RecF *>(a.rec) + (int64_t)idx * a.nrec;
    if (s.sched_steps > 0) {
        const double t0 = *s.t_dev;
        small_records(a.inst[idx], s.sc, t0, s.sched_steps * s.sc.m, s_fge, s_rec, a.status);
        __syncthreads();
        if (threadIdx.x == 0) {
            // every CTA has read the time before it counts itself
            __threadfence();
            if (atomicAdd(s.done, 1u) + 1 == gridDim.x) {
                *s.done = 0;
                *s.t_dev = t0 + (double)s.sched_steps * s.sc.h;
            }
        }
        rec = s_rec;
    }
    switch (a.inst[idx].n[0]) {
    case 128: small_item<128, PROJ>(a, idx, rec, sm, vtab, slots); break;
    case 256: small_item<256, PROJ>(a, idx, rec, sm, vtab, slots); break;
    case 512: small_item<512, PROJ>(a, idx, rec, sm, vtab, slots); break;
    case 1024: small_item<1024, PROJ>(a, idx, rec, sm, vtab, slots); break;
    default:
        if constexpr (BIG) {
            if (a.inst[idx].n[0] == 2048) big_item<2048, PROJ ? 16 : 8, PROJ, VI>(a, idx, rec, sm, vtab, slots);
            else big_item<4096, 16, PROJ, VI>(a, idx, rec, sm, vtab, slots);
        }
    }
}

template <bool PROJ, bool BIG, int VI>
cudaError_t launch_t(const Small1DArgs &s, int threads, cudaStream_t st, int priority)
{
    auto kernel = small1d_kernel<PROJ, BIG, VI>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)small_smem<BIG>());
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)s.count);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = small_smem<BIG>();
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributePriority;
    at[0].val.priority = priority;
    cfg.attrs = at;
    cfg.numAttrs = priority != 0 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, s);
}

}  // namespace

// As long as every instance has an SM for itself, or, up to 1024 points, as
// long as the batch's threads (a quarter of its points) make 256 an SM: beyond
// that the transforms with more values per thread do less work for each point.
bool small1d_ok(const DevInst *inst, int64_t count, int64_t points, int sms)
{
    int nmax = 0;
    for (int64_t i = 0; i < count; ++i) nmax = nmax > inst[i].n[0] ? nmax : inst[i].n[0];
    return nmax <= kSmallMaxN ? points / 4 <= (int64_t)sms * 256 : count <= sms;
}

cudaError_t launch_small1d(const Small1DArgs &s, int nmax, int variant, cudaStream_t st, int priority)
{
    const bool proj = s.a.proj != PROJ_OFF;
    if (nmax <= kSmallMaxN)
        return proj ? launch_t<true, false, -1>(s, nmax / 4, st, priority)
                    : launch_t<false, false, -1>(s, nmax / 4, st, priority);
    if (variant == HFS_VI_COS)
        return proj ? launch_t<true, true, HFS_VI_COS>(s, kCtaThreads, st, priority)
                    : launch_t<false, true, HFS_VI_COS>(s, kCtaThreads, st, priority);
    return proj ? launch_t<true, true, -1>(s, kCtaThreads, st, priority)
                : launch_t<false, true, -1>(s, kCtaThreads, st, priority);
}

}  // namespace hfs
