// hfs_step1d_cluster.cu -- the 1D step of few complex128 instances of one grid
// size: an instance on a cluster of G CTAs.
//
// The FP64 pipe of one SM (2 lanes a cycle) bounds an instance that one CTA holds:
// 1024 points take 35 us a sub-stage there whatever the number of threads.  Here
// the transform of the plans with sixteen values a thread (radix 16 first) is
// spread over the cluster: CTA c holds the positions n with n mod 16 in [c W,
// (c + 1) W), W = 16 / G, of the state and of its transform alike.  The inputs b +
// (N/16) r of a radix-16 butterfly of the first pass lie in one CTA; its outputs 16
// b + k go to the CTA of k, through distributed shared memory and one cluster
// barrier; the later passes keep a position's residue mod 16 and stay within the
// CTA.  Four threads hold a butterfly (lane_dft16), four values each.  A sub-stage
// takes two such exchanges, into two buffers: a buffer is written again only after
// the barrier of the other, which every CTA reaches after reading the first.  One
// instance of 1024 points: 35 -> 19 us a sub-stage (201 us with idle teams and cos in
// the sub-stage), 19 of 4096 points 150 -> 41 us.  Bound by the FP64 pipe of the one
// to four SM quarters that a CTA's warps occupy (64 cycles a warp instruction each).
// Rounding: the radices and with them the twiddle products of the 16-value plans, so
// that 25 steps of NI5(8,4) end as far from 64 bits as theirs (1024 points: 1.37e-14
// / 1.28e-14, 8 seeds; 4096: 1.49e-13 both).  Radix 4 within N = N1 N2 and a factor
// between them multiplied by five twiddles where this takes two: 3.7e-14 and 1.8e-13.
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
    static constexpr int W = 16 / G;                   // residues mod 16 of a CTA
    static constexpr int P = N / G, E = 4, THREADS = P / E;
    static constexpr size_t SMEM = (size_t)3 * P * sizeof(cpx<double>);
};

// input of a radix-RAD butterfly that value e of lane q is
template <int RAD> __device__ __forceinline__ int input_of(int e, int q)
{
    return RAD == 2 ? e >> 1 : RAD == 4 ? e : RAD == 8 ? 2 * e + (q >> 1) : 4 * e + q;
}

// what a thread keeps over all sub-stages: its butterfly b (bh, bl: b / 16, b mod
// W), its lane q, the slot rd of its first value and the twiddles of the second and
// third pass.  Position p of the CTA is in slot p / 16 W + p mod W of a buffer.
template <int N> struct ClusterLane {
    int b, bh, bl, q, rd;
    double2 w2[4], w3[4];
};

template <int N, bool INV>
__device__ __forceinline__ void cluster_fft(cpx<double> (&v)[4], const ClusterLane<N> &l, const cpx<double> *far,
                                            cpx<double> *loc)
{
    using GEO = ClusterGeo<N>;
    constexpr int W = GEO::W, RAD = N / 256, STEP = N / 64 * W;
    auto twiddle = [](cpx<double> a, double2 w) { return mulw(a, w.x, INV ? -w.y : w.y); };
    lane_dft16<INV>(v, l.q);
    const uint32_t at = (uint32_t)__cvta_generic_to_shared(far);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int out = l.q + 4 * k;
        put(at, l.b * W + (out & (W - 1)), (uint32_t)(out / W), v[k]);
    }
    cluster_sync();
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = twiddle(far[l.rd + e * STEP], l.w2[e]);
    lane_dft16<INV>(v, l.q);
    if constexpr (RAD > 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k) loc[(l.bh * 16 + l.q + 4 * k) * W + l.bl] = v[k];
        if constexpr (GEO::THREADS == 32) __syncwarp();
        else __syncthreads();
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = twiddle(loc[l.rd + e * STEP], l.w3[e]);
        if constexpr (RAD == 16) lane_dft16<INV>(v, l.q);
        else if constexpr (RAD == 8) lane_dft8<INV>(v, l.q);
        else if constexpr (RAD == 4) dft4<INV>(v[0], v[1], v[2], v[3]);
        else {
            dft2<INV>(v[0], v[2]);
            dft2<INV>(v[1], v[3]);
        }
    }
}

template <int N>
__global__ void __launch_bounds__(ClusterGeo<N>::THREADS, 1) cluster1d_kernel(const Step1DArgs a)
{
    using GEO = ClusterGeo<N>;
    constexpr int E = GEO::E, W = GEO::W, RAD = N / 256;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<double> *loc = reinterpret_cast<cpx<double> *>(smem_raw);  // exchanges within the CTA
    cpx<double> *fwd = loc + GEO::P, *inv = fwd + GEO::P;          // and between the CTAs, by direction
    const int rank = (int)cluster_rank();
    const int idx = a.order[blockIdx.x / GEO::G];
    const DevInst &ip = a.inst[idx];
    const TeamParams<double> tp = team_params<double>(ip);
    cpx<double> *psi = reinterpret_cast<cpx<double> *>(a.psi) + ip.off;
    const double2 *tw = reinterpret_cast<const double2 *>(a.tw);
    const RecD *rec = reinterpret_cast<const RecD *>(a.rec) + (int64_t)idx * a.nrec;
    ClusterLane<N> l;
    l.q = threadIdx.x & 3;
    l.bl = (threadIdx.x >> 2) & (W - 1);
    l.bh = (threadIdx.x >> 2) / W;
    l.b = l.bh * 16 + rank * W + l.bl;
    l.rd = (l.bh + N / 256 * l.q) * W + l.bl;
    const int t = l.b + N / 16 * l.q;  // positions t + (N/4) e
    cpx<double> v[E];
    double vt[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int n = t + N / 4 * e, r2 = input_of<16>(e, l.q);
        v[e] = ld_state(psi + n, a.streaming);
        vt[e] = tp.eps * vi_eval(tp.vikind, fma((double)(n - N / 2), tp.dx, tp.xc), tp.vik);
        l.w2[e] = l.w3[e] = make_double2(1.0, 0.0);
        if (r2 > 0) l.w2[e] = tw[tw_pass_offset(256, 16) + (r2 - 1) * 16 + (l.b & 15)];
        if constexpr (RAD > 1) {
            const int r3 = input_of<RAD>(e, l.q);
            if (r3 > 0) l.w3[e] = tw[tw_pass_offset(N, RAD) + (r3 - 1) * 256 + (n & 255)];
        }
    }
    auto xphase_c = [&](const RecD &rc) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int m = t + N / 4 * e - N / 2;
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
        cluster_fft<N, false>(v, l, fwd, loc);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int m = t + N / 4 * e - (2 * e < E ? 0 : N);
            v[e] = apply_turns(v[e], rc.g * square64(m), 1.0 / N);
        }
        cluster_fft<N, true>(v, l, inv, loc);
        rc = next;
    }
    if (a.final_x) xphase_c(rc);
    bool bad = false;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        st_state(psi + t + N / 4 * e, v[e], a.streaming);
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
