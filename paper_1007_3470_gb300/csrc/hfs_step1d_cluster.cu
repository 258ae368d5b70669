// hfs_step1d_cluster.cu -- the 1D step of few complex128 instances of one grid
// size: an instance on a cluster of G CTAs.
//
// The FP64 pipe of one SM (2 lanes a cycle) bounds an instance that one CTA holds:
// 1024 points take 35 us a sub-stage there whatever the number of threads.  Here
// the transform is split as N = N1 N2 (n = n1 N2 + n2, k = k1 + N1 k2): CTA c
// holds N2/G columns n2 for the transforms over n1 and N1/G rows k1 for those
// over n2, each within the CTA, four values a thread; between them stand the
// twiddles W_N^{n2 k1} and one exchange of the whole instance through
// distributed shared memory with one cluster barrier.  The kinetic phase is
// applied in row order, so a sub-stage takes two such exchanges, into two
// buffers: a buffer is written again only after the barrier of the other, which
// every CTA reaches after reading the first.  One instance of 1024 points: 35 ->
// 18 us a sub-stage (201 us with idle teams and cos in the sub-stage), 19 of 4096
// points 150 -> 43 us; the rest is latency, with a warp or four in each CTA.
// Rounding: radix 4 multiplies by a twiddle factor more often than radix 16 (1024
// points: five times a transform against two), so 25 steps of NI5(8,4) end 2e-14
// to 5e-14 off (256 to 1024 points; 9e-14 at 2048, 2.5e-13 at 4096) where the
// plans of 16 values end 1e-14 to 2e-14 off (4e-14, 2.1e-13) and those of 8
// values 1e-14 to 2e-14.  A set plan keeps its own kernel.
#include "hfs_step1d.cuh"

namespace hfs {

namespace {

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// element i of the buffer at shared address `base` of CTA `cta`
__device__ __forceinline__ void put(uint32_t base, int i, uint32_t cta, cpx<double> v)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(base + (uint32_t)i * 16u), "r"(cta));
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}

template <int N> struct ClusterGeo {
    static constexpr int G = N >= 1024 ? 8 : N / 128;  // a warp or more in every CTA
    static constexpr int N1 = N == 256 ? 16 : N <= 1024 ? 32 : 64, N2 = N / N1;
    static constexpr int W2 = N2 / G, W1 = N1 / G;  // columns, rows of a CTA
    static constexpr int P = N / G, E = 4, THREADS = P / E;
    static constexpr size_t SMEM = (size_t)3 * P * sizeof(cpx<double>);
};

template <int N>
__global__ void __launch_bounds__(ClusterGeo<N>::THREADS, 1) cluster1d_kernel(const Step1DArgs a)
{
    using GEO = ClusterGeo<N>;
    constexpr int N1 = GEO::N1, N2 = GEO::N2, W1 = GEO::W1, W2 = GEO::W2, E = GEO::E, T1 = N1 / E, T2 = N2 / E;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<double> *loc = reinterpret_cast<cpx<double> *>(smem_raw);  // exchanges within the CTA
    cpx<double> *bufk = loc + GEO::P, *bufx = bufk + GEO::P;       // to row and to column order
    const uint32_t ka = (uint32_t)__cvta_generic_to_shared(bufk), xa = (uint32_t)__cvta_generic_to_shared(bufx);
    const int rank = (int)cluster_rank();
    const int idx = a.order[blockIdx.x / GEO::G];
    const DevInst &ip = a.inst[idx];
    const TeamParams<double> tp = team_params<double>(ip);
    cpx<double> *psi = reinterpret_cast<cpx<double> *>(a.psi) + ip.off;
    const double2 *tw = reinterpret_cast<const double2 *>(a.tw);
    const RecD *rec = reinterpret_cast<const RecD *>(a.rec) + (int64_t)idx * a.nrec;
    // column order: column n2, points n1 = t1 + T1 e; row order: row k1, k2 (or n2) = t2 + T2 e
    const int l1 = threadIdx.x % W2, t1 = threadIdx.x / W2, n2 = rank * W2 + l1;
    const int l2 = threadIdx.x % W1, t2 = threadIdx.x / W1, k1 = rank * W1 + l2;
    cpx<double> v[E];
    double vt[E], wc[E], ws[E], xc[E], xs[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int n = (t1 + T1 * e) * N2 + n2;
        v[e] = ld_state(psi + n, a.streaming);
        vt[e] = tp.eps * vi_eval(tp.vikind, fma((double)(n - N / 2), tp.dx, tp.xc), tp.vik);
        // W_N^m, m = n2 k1 in column and in row order, from the radix-2 region of the table
        const int m1 = (n2 * (t1 + T1 * e)) & (N - 1), m2 = (k1 * (t2 + T2 * e)) & (N - 1);
        const double2 w1 = tw[tw_pass_offset(N, 2) + (m1 & (N / 2 - 1))], w2 = tw[tw_pass_offset(N, 2) + (m2 & (N / 2 - 1))];
        wc[e] = m1 >= N / 2 ? -w1.x : w1.x;
        ws[e] = m1 >= N / 2 ? -w1.y : w1.y;
        xc[e] = m2 >= N / 2 ? -w2.x : w2.x;
        xs[e] = m2 >= N / 2 ? -w2.y : w2.y;
    }
    auto xphase_c = [&](const RecD &rc) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int m = (t1 + T1 * e) * N2 + n2 - N / 2;
            const double dens = fma(v[e].x, v[e].x, v[e].y * v[e].y);
            double turns = rc.sb2pi * fma(tp.sigma, dens, vt[e]);
            if (tp.asym) turns += fma(rc.k1, (double)m, rc.k0);
            v[e] = apply_turns(v[e], fma(rc.k2, square64(m), turns), 1.0);
        }
    };
    cluster_sync();  // every CTA of the cluster runs before the first remote store
    RecD rc = rec[a.j0];
    for (int64_t j = a.j0; j < a.j1; ++j) {
        const RecD next = rec[j + 1];
        xphase_c(rc);
        FftPlan<N1, E>::template run<false, double, W2>(v, loc + l1, t1, tw);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int k = t1 + T1 * e;
            put(ka, n2 * W1 + k % W1, (uint32_t)(k / W1), mulw(v[e], wc[e], ws[e]));
        }
        cluster_sync();
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = bufk[(t2 + T2 * e) * W1 + l2];
        FftPlan<N2, E>::template run<false, double, W1>(v, loc + l2, t2, tw);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int k = k1 + N1 * (t2 + T2 * e);
            v[e] = apply_turns(v[e], rc.g * square64(k < N / 2 ? k : k - N), 1.0 / N);
        }
        FftPlan<N2, E>::template run<true, double, W1>(v, loc + l2, t2, tw);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int n = t2 + T2 * e;
            put(xa, k1 * W2 + n % W2, (uint32_t)(n / W2), mulw(v[e], xc[e], -xs[e]));
        }
        cluster_sync();
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = bufx[(t1 + T1 * e) * W2 + l1];
        FftPlan<N1, E>::template run<true, double, W2>(v, loc + l1, t1, tw);
        rc = next;
    }
    if (a.final_x) xphase_c(rc);
    bool bad = false;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        st_state(psi + (t1 + T1 * e) * N2 + n2, v[e], a.streaming);
        bad |= !(isfinite(v[e].x) && isfinite(v[e].y));
    }
    if (bad) atomicOr(a.status, (unsigned)ST_NONFINITE);
}

template <int N> cudaError_t launch_t(const Step1DArgs &a, int count, cudaStream_t st, int priority)
{
    using GEO = ClusterGeo<N>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(count * GEO::G));
    cfg.blockDim = dim3((unsigned)GEO::THREADS);
    cfg.dynamicSmemBytes = GEO::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = GEO::G;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributePriority;
    at[1].val.priority = priority;
    cfg.attrs = at;
    cfg.numAttrs = priority != 0 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, cluster1d_kernel<N>, a);
}

}  // namespace

// From 256 points (at 128 a CTA is one warp already), while every CTA of the
// clusters has an SM: beyond that the SMs' FP64 pipes are busy either way.
bool cluster1d_ok(const DevInst *inst, int64_t count, int sms)
{
    const int n = inst[0].n[0];
    for (int64_t i = 1; i < count; ++i)
        if (inst[i].n[0] != n) return false;
    const int g = n >= 1024 ? 8 : n / 128;
    return n >= 256 && count * g <= sms;
}

cudaError_t launch_cluster1d(const Step1DArgs &a, int n, int count, cudaStream_t st, int priority)
{
    switch (n) {
    case 256: return launch_t<256>(a, count, st, priority);
    case 512: return launch_t<512>(a, count, st, priority);
    case 1024: return launch_t<1024>(a, count, st, priority);
    case 2048: return launch_t<2048>(a, count, st, priority);
    case 4096: return launch_t<4096>(a, count, st, priority);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace hfs
