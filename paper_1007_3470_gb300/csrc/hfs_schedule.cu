// hfs_schedule.cu -- device-side FP64 schedule of the Magnus and
// decomposition coefficients.
//
// Kernel 1 (stage_flow_kernel): for every instance, stage and axis, the
// harmonic flow of one A stage over [tau, tau + a_i h] as kick(f) .
// drift(g) . kick(e), e applied first:
//   * exact flow for constant omega (Lemma 2 with mu, omega):
//       g = sin(omega s)/(mu omega), f = e = mu omega tan(omega s/2);
//   * commutator-free Magnus-4 (Eq. CommutatorFree): two half steps with
//       omega_L^2 = al w1 + be w2, omega_R^2 = be w1 + al w2 (R first),
//       w_k = omega^2(tau + c_k s), c = 1/2 -+ sqrt(3)/6, al = 1/2 - 1/sqrt3,
//     decomposed by Theorem 2;
//   * sixth-order Magnus (Sec. 4.2), omega^2 read at the three Gauss nodes,
//     decomposed by Theorem 1.
// The trigonometric quantities are written in the forms C(w,t)=cos(sqrt(w)t)
// and S(w,t)=sin(sqrt(w)t)/sqrt(w), continued to w <= 0, with
// 1 - cos = 2 sin^2(half angle), so that no difference of nearly equal
// numbers is formed for small steps.
//
// Kernel 2 (records kernels): merges adjacent chirps and B flows as in
// Eq. prod-genHarmOsc -- the kick between drifts i and i+1 is f_i + e_{i+1}
// and the B flows at a step boundary add (b_{m+1} + b_1) h (FSAL) -- and
// converts every coefficient into phase "turns" per unit integer index:
//   kick   kappa x^2/2 / (2 pi),   x = xc + m dx
//          -> K2 = kappa dx^2/(4 pi), K1 = kappa xc dx/(2 pi), K0 = kappa xc^2/(4 pi) mod 1
//   drift  g k^2/2 / (2 pi),       k = 2 pi m_k / L  ->  G = g pi / L^2
//   B      s (eps V_I + sigma |u|^2) / (2 pi)       ->  sb2pi = s / (2 pi)
// For the F split (Eq. FourierSplit) the drift is g = a_i h / mu and the
// trap mu omega^2(tau) x^2/2 of every B flow joins the kick at its frozen
// time.
#include <math.h>

#include <algorithm>
#include <cstdint>

#include "hfs_internal.cuh"
#include "hfs_law.cuh"
#include "hfs_sched.h"
#include "hfs_schedule.cuh"

namespace hfs {

// the shape factors of every stage of the chunk, once for a batch whose
// instances share the law and its parameters (read from instance 0)
template <int FLOW, int LAW>
__global__ void law_nodes_kernel(const DevInst *__restrict__ inst, SchedConst sc, const double *__restrict__ t_dev,
                                 double t_off, int nstage, NodeS *__restrict__ nodes)
{
    const int sg = blockIdx.x * blockDim.x + threadIdx.x;
    if (sg >= nstage) return;
    const int n = sg / sc.m, st = sg - n * sc.m;
    const double tau = *t_dev + t_off + (double)n * sc.h + sc.h * sc.cuma[st];
    nodes[sg] = stage_nodes<FLOW, LAW>(inst[0], tau, sc.a[st] * sc.h);
}

// Work of a thread of the schedule kernels: (instance, entry of its chunk).  A
// block takes one instance (x) and strides over its entries (y), or, where a
// chunk has fewer than kFlatBelow entries an instance, threads take instances
// and entries in one line (with an integer division each; one block of 128 for
// every instance left 127 threads idle on calls of one step: 65 + 45 us for
// 16384 instances).
constexpr int kFlatBelow = 16;
struct ItemAt {
    int64_t i;
    int n, stride;  // stride 0: none of this thread's
};
template <bool FLAT> __device__ __forceinline__ ItemAt item_at(int64_t count, int per)
{
    if constexpr (FLAT) {
        const int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
        if (u >= count * per) return {0, 0, 0};
        const int64_t i = u < ((int64_t)1 << 32) ? (int64_t)((unsigned)u / (unsigned)per) : u / per;
        return {i, (int)(u - i * per), per};
    } else {
        return {(int64_t)blockIdx.x, (int)(blockIdx.y * blockDim.x + threadIdx.x), (int)(gridDim.y * blockDim.x)};
    }
}
static dim3 item_grid(int64_t count, int64_t per, bool flat)
{
    if (flat) return dim3((unsigned)((count * per + 127) / 128));
    return dim3((unsigned)count, (unsigned)std::min<int64_t>((per + 127) / 128, 65535));
}

// one thread per (instance, time step of the chunk), all m stages of the
// step.  SHARED: the shape factors come from law_nodes_kernel instead of being
// evaluated per instance.
template <int FLOW, int LAW, bool SHARED, bool FLAT>
__global__ void stage_flow_kernel(const DevInst *__restrict__ inst, int64_t count, int dim, SchedConst sc,
                                  const double *__restrict__ t_dev, double t_off, int nsteps,
                                  const NodeS *__restrict__ nodes, StageFGE *__restrict__ out, unsigned *status)
{
    const ItemAt at = item_at<FLAT>(count, nsteps);
    if (FLAT && at.stride == 0) return;
    const int64_t i = at.i;
    const DevInst &p = inst[i];
    const double t0 = *t_dev + t_off;
    const int64_t nstage = (int64_t)nsteps * sc.m;
    for (int n = at.n; n < nsteps; n += at.stride) {
        for (int st = 0; st < sc.m; ++st) {
            const double tau = t0 + (double)n * sc.h + sc.h * sc.cuma[st];
            const double s = sc.a[st] * sc.h;
            const int64_t sg = (int64_t)n * sc.m + st;
            NodeS ns;
            if constexpr (SHARED) ns = nodes[sg];
            else ns = stage_nodes<FLOW, LAW>(p, tau, s);
            for (int d = 0; d < dim; ++d) {
                double f, g, e;
                stage_fge<FLOW>(p, dim, d, ns, s, f, g, e);
                if (!isfinite(f) || !isfinite(g) || !isfinite(e)) atomicOr(status, (unsigned)ST_NONFINITE);
                StageFGE r;
                r.f = f;
                r.g = g;
                r.e = e;
                r.tau = tau;
                out[(i * nstage + sg) * dim + d] = r;
            }
        }
    }
}

// one thread per (instance, sub-stage j in [0, nstage]) -- 1D records
template <typename RecT, int SPLIT, bool FLAT>
__global__ void records1d_kernel(const DevInst *__restrict__ inst, int64_t count, SchedConst sc,
                                 const double *__restrict__ t_dev, double t_off, int nstage,
                                 const StageFGE *__restrict__ fge, RecT *__restrict__ rec, unsigned *status)
{
    const int64_t nrec = (int64_t)nstage + 1;
    const ItemAt at = item_at<FLAT>(count, (int)nrec);
    if (FLAT && at.stride == 0) return;
    const int64_t i = at.i;
    const DevInst &p = inst[i];
    const double t0 = *t_dev + t_off;
    RecScale c;
    if constexpr (FLAT) {
        c = rec_scale(p, sc);
    } else {
        // the block's instance factors, computed once (one FP64 division per block, not per record)
        __shared__ RecScale s_c;
        if (threadIdx.x == 0) s_c = rec_scale(p, sc);
        __syncthreads();
        c = s_c;
    }
    for (int j = at.n; j <= nstage; j += at.stride)
        record1d<RecT, SPLIT>(p, sc, c, t0, j, nstage, fge + i * (int64_t)nstage, rec + i * nrec + j, status);
}

// 3D records (symmetric boxes): one per sub-stage, all three axes
template <typename RecT, int SPLIT>
__global__ void records3d_kernel(const DevInst *__restrict__ inst, SchedConst sc, const double *__restrict__ t_dev,
                                 double t_off, int nstage, const StageFGE *__restrict__ fge,
                                 RecT *__restrict__ rec, unsigned *status)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j > nstage) return;
    const DevInst p = inst[0];
    const double t0 = *t_dev + t_off;
    RecT r;
    double SB = 0.0;
    for (int d = 0; d < 3; ++d) {
        double kappa, bs, g;
        merged_coeffs<SPLIT>(p, 3, d, sc, t0, j, nstage, fge, kappa, bs, g);
        const double K2 = kappa * p.dx[d] * p.dx[d] / (4.0 * kPi);
        const double G = g * kPi / (p.len[d] * p.len[d]);
        SB = bs * sc.h / (2.0 * kPi);
        if (!isfinite(K2) || !isfinite(G)) atomicOr(status, (unsigned)ST_NONFINITE);
        if constexpr (sizeof(r.k2[0]) == sizeof(float)) {
            split_hi_lo(K2, r.k2[d], r.k2lo[d]);
            split_hi_lo(G, r.g[d], r.glo[d]);
        } else {
            r.k2[d] = K2;
            r.g[d] = G;
            r.k2lo[d] = 0.0;
            r.glo[d] = 0.0;
        }
    }
    r.sb2pi = SB;
    rec[j] = r;
}

__global__ void set_time_kernel(double *t_dev, double t) { *t_dev = t; }
__global__ void advance_time_kernel(double *t_dev, double dt) { *t_dev += dt; }

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static inline unsigned blocks_for(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

int uniform_law(const hfs_instance *inst, int64_t count)
{
    if (count < 1) return -1;
    for (int64_t i = 1; i < count; ++i)
        if (inst[i].omega_law != inst[0].omega_law) return -1;
    return inst[0].omega_law;
}

bool law_shared(const hfs_instance *inst, int64_t count)
{
    if (uniform_law(inst, count) < 0) return false;
    for (int64_t i = 1; i < count; ++i)
        for (int k = 0; k < 3; ++k)
            if (inst[i].law[k] != inst[0].law[k]) return false;
    return true;
}

size_t law_nodes_bytes(int64_t nstage) { return sizeof(NodeS) * (size_t)nstage; }

template <int FLOW, int LAW>
static void launch_stage_flow_fl(bool shared, const DevInst *inst, int64_t count, int dim, const SchedConst &sc,
                                 const double *t_dev, double t_off, int nsteps, void *nodes, StageFGE *out,
                                 unsigned *status, cudaStream_t st)
{
    NodeS *nd = static_cast<NodeS *>(nodes);
    const bool flat = nsteps < kFlatBelow;
    const dim3 grid = item_grid(count, nsteps, flat);
    if constexpr (LAW >= 0) {
        if (shared && nd) {
            const int nstage = nsteps * sc.m;
            law_nodes_kernel<FLOW, LAW><<<blocks_for(nstage, 128), 128, 0, st>>>(inst, sc, t_dev, t_off, nstage, nd);
            if (flat)
                stage_flow_kernel<FLOW, LAW, true, true>
                    <<<grid, 128, 0, st>>>(inst, count, dim, sc, t_dev, t_off, nsteps, nd, out, status);
            else
                stage_flow_kernel<FLOW, LAW, true, false>
                    <<<grid, 128, 0, st>>>(inst, count, dim, sc, t_dev, t_off, nsteps, nd, out, status);
            return;
        }
    }
    if (flat)
        stage_flow_kernel<FLOW, LAW, false, true>
            <<<grid, 128, 0, st>>>(inst, count, dim, sc, t_dev, t_off, nsteps, nullptr, out, status);
    else
        stage_flow_kernel<FLOW, LAW, false, false>
            <<<grid, 128, 0, st>>>(inst, count, dim, sc, t_dev, t_off, nsteps, nullptr, out, status);
}

template <int FLOW>
static void launch_stage_flow_law(int law, bool shared, const DevInst *inst, int64_t count, int dim,
                                  const SchedConst &sc, const double *t_dev, double t_off, int nsteps, void *nodes,
                                  StageFGE *out, unsigned *status, cudaStream_t st)
{
#define HFS_SF(L) launch_stage_flow_fl<FLOW, L>(shared, inst, count, dim, sc, t_dev, t_off, nsteps, nodes, out, status, st)
    switch (law) {
    case HFS_OMEGA_CONST: HFS_SF(HFS_OMEGA_CONST); break;
    case HFS_OMEGA_SIN: HFS_SF(HFS_OMEGA_SIN); break;
    case HFS_OMEGA_COS_SQ: HFS_SF(HFS_OMEGA_COS_SQ); break;
    case HFS_OMEGA_PULSE: HFS_SF(HFS_OMEGA_PULSE); break;
    default: HFS_SF(-1); break;
    }
#undef HFS_SF
}

cudaError_t launch_stage_flow(const DevInst *inst, int64_t count, int dim, const SchedConst &sc, const double *t_dev,
                              double t_off, int64_t nstage, int uniform_law, bool shared, void *nodes,
                              StageFGE *out, unsigned *status, cudaStream_t st)
{
    if (count == 0 || nstage == 0) return cudaSuccess;
    if (nstage >= INT32_MAX || nstage % sc.m != 0 || count > INT32_MAX) return cudaErrorInvalidValue;
    const int nsteps = (int)(nstage / sc.m);
    switch (sc.flow) {
    case HFS_FLOW_LEMMA2:
        launch_stage_flow_law<HFS_FLOW_LEMMA2>(uniform_law, shared, inst, count, dim, sc, t_dev, t_off, nsteps,
                                               nodes, out, status, st);
        break;
    case HFS_FLOW_CF4:
        launch_stage_flow_law<HFS_FLOW_CF4>(uniform_law, shared, inst, count, dim, sc, t_dev, t_off, nsteps,
                                               nodes, out, status, st);
        break;
    default:
        launch_stage_flow_law<HFS_FLOW_M6>(uniform_law, shared, inst, count, dim, sc, t_dev, t_off, nsteps,
                                               nodes, out, status, st);
        break;
    }
    return cudaGetLastError();
}

cudaError_t launch_records1d(bool fp64, const DevInst *inst, int64_t count, const SchedConst &sc, const double *t_dev,
                             double t_off, int64_t nstage, const StageFGE *fge, void *rec, unsigned *status,
                             cudaStream_t st)
{
    if (count == 0) return cudaSuccess;
    if (nstage >= INT32_MAX || count > INT32_MAX) return cudaErrorInvalidValue;
    const bool ho = sc.split == HFS_SPLIT_HO, flat = nstage + 1 < kFlatBelow;
    const dim3 grid = item_grid(count, nstage + 1, flat);
    auto launch = [&](auto kernel, auto *r) {
        kernel<<<grid, 128, 0, st>>>(inst, count, sc, t_dev, t_off, (int)nstage, fge, r, status);
    };
    if (fp64) {
        RecD *r = (RecD *)rec;
        if (ho) flat ? launch(records1d_kernel<RecD, HFS_SPLIT_HO, true>, r) : launch(records1d_kernel<RecD, HFS_SPLIT_HO, false>, r);
        else flat ? launch(records1d_kernel<RecD, HFS_SPLIT_FOURIER, true>, r) : launch(records1d_kernel<RecD, HFS_SPLIT_FOURIER, false>, r);
    } else {
        RecF *r = (RecF *)rec;
        if (ho) flat ? launch(records1d_kernel<RecF, HFS_SPLIT_HO, true>, r) : launch(records1d_kernel<RecF, HFS_SPLIT_HO, false>, r);
        else flat ? launch(records1d_kernel<RecF, HFS_SPLIT_FOURIER, true>, r) : launch(records1d_kernel<RecF, HFS_SPLIT_FOURIER, false>, r);
    }
    return cudaGetLastError();
}

cudaError_t launch_records3d(bool fp64, const DevInst *inst, const SchedConst &sc, const double *t_dev, double t_off,
                             int64_t nstage, const StageFGE *fge, void *rec, unsigned *status, cudaStream_t st)
{
    const int64_t n = nstage + 1;
    if (nstage >= INT32_MAX) return cudaErrorInvalidValue;
    const unsigned b = blocks_for(n, 128);
    const bool ho = sc.split == HFS_SPLIT_HO;
    if (fp64 && ho)
        records3d_kernel<Rec3D, HFS_SPLIT_HO><<<b, 128, 0, st>>>(inst, sc, t_dev, t_off, (int)nstage, fge, (Rec3D *)rec, status);
    else if (fp64)
        records3d_kernel<Rec3D, HFS_SPLIT_FOURIER><<<b, 128, 0, st>>>(inst, sc, t_dev, t_off, (int)nstage, fge, (Rec3D *)rec, status);
    else if (ho)
        records3d_kernel<Rec3F, HFS_SPLIT_HO><<<b, 128, 0, st>>>(inst, sc, t_dev, t_off, (int)nstage, fge, (Rec3F *)rec, status);
    else
        records3d_kernel<Rec3F, HFS_SPLIT_FOURIER><<<b, 128, 0, st>>>(inst, sc, t_dev, t_off, (int)nstage, fge, (Rec3F *)rec, status);
    return cudaGetLastError();
}

cudaError_t launch_set_time(double *t_dev, double t, cudaStream_t st)
{
    set_time_kernel<<<1, 1, 0, st>>>(t_dev, t);
    return cudaGetLastError();
}

cudaError_t launch_advance_time(double *t_dev, double dt, cudaStream_t st)
{
    advance_time_kernel<<<1, 1, 0, st>>>(t_dev, dt);
    return cudaGetLastError();
}

}  // namespace hfs
