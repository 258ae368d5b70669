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
template <int T> __device__ __forceinline__ double team_warps(double s, double *slots)
{
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
template <int T> __device__ __forceinline__ double team_sum(double s, double *slots)
{
    constexpr int W = T < 32 ? T : 32;
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return team_warps<T>(s, slots);
}

// Unevaluated FP32 sums hi + lo.  The FP64 pipe takes 16 cycles a warp
// instruction, an FP32 instruction a quarter of one (an SM), so sums over an FP32
// state are formed in two or three floats with exact products and additions
// (Dekker, Knuth), and only a thread's total enters FP64.
struct Pair {
    float hi, lo;
};
__device__ __forceinline__ Pair two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ Pair quick_sum(float a, float b)  // |a| >= |b|
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ Pair two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ Pair add(Pair a, Pair b)
{
    const Pair s = two_sum(a.hi, b.hi);
    return quick_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ Pair mul(Pair a, Pair b)
{
    const Pair p = two_prod(a.hi, b.hi);
    return quick_sum(p.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo)));
}
__device__ __forceinline__ Pair abs2(cpx<float> v)
{
    const Pair x = two_prod(v.x, v.x), y = two_prod(v.y, v.y), s = two_sum(x.hi, y.hi);
    return quick_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}
__device__ __forceinline__ Pair to_pair(double a)
{
    const float h = (float)a;
    return {h, (float)(a - (double)h)};
}
template <int T> __device__ __forceinline__ double team_sum(Pair s, double *slots)
{
    constexpr int W = T < 32 ? T : 32;
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1)
        s = add(s, Pair{__shfl_xor_sync(0xffffffffu, s.hi, o), __shfl_xor_sync(0xffffffffu, s.lo, o)});
    return team_warps<T>((double)s.hi + (double)s.lo, slots);
}

// Norm alone: one pass over the state.  With two FMAs and two conversions a point
// the FP64 pipe bounds it (a complex128 state's still); an FP32 state's squares
// are summed exactly in three floats (to 2^-72), 44 FP32 instructions a point.
// Squares outside FP32's range, or not finite, are summed again in FP64.
// One copy of the loop for all plans: unrolled in each, a warp waited for
// instructions 8 cycles of the 24 it took per issue (37 us for 4096 instances; 30
// us now).
__device__ __noinline__ double norm_floats(const cpx<float> *psi, int T, int E)
{
    float hi = 0.0f, mid = 0.0f, lo = 0.0f;
#pragma unroll 1
    for (int e0 = 0; e0 < E; e0 += 4) {
        cpx<float> v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = psi[T * (e0 + e)];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const Pair x = two_prod(v[e].x, v[e].x), y = two_prod(v[e].y, v[e].y);
            const Pair d = two_sum(x.hi, y.hi), r = two_sum(x.lo, y.lo);
            const Pair h = two_sum(hi, d.hi);
            const Pair m0 = two_sum(mid, h.lo), m1 = two_sum(m0.hi, d.lo), m2 = two_sum(m1.hi, r.hi);
            hi = h.hi;
            mid = m2.hi;
            lo += (m0.lo + m1.lo) + (m2.lo + r.lo);
        }
    }
    return (double)hi + ((double)mid + (double)lo);
}
template <typename R, int T, int E>
__device__ __forceinline__ void norm_item(const Diag1DArgs &a, const WorkItem &it, double *slots)
{
    const int g = threadIdx.x / T, t = threadIdx.x - g * T;
    const bool active = g < it.count;
    const int idx = a.order[it.first + (active ? g : 0)];
    const DevInst &ip = a.inst[idx];
    const cpx<R> *psi = reinterpret_cast<const cpx<R> *>(a.psi) + ip.off;
    double s = 0.0;
    bool done = false;
    if constexpr (sizeof(R) == 4) {
        s = team_sum<T>(active ? norm_floats(psi + t, T, E) : 0.0, slots);
        done = !active || (s > 1e-18 && s < 1e30);
        if constexpr (T < 32) done = __all_sync(0xffffffffu, done);
    }
    if (!done) {
        s = 0.0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const cpx<R> u = active ? psi[t + T * e] : cpx<R>{R(0), R(0)};
            const double x = u.x, y = u.y;
            s = fma(x, x, fma(y, y, s));
        }
        s = team_sum<T>(s, slots);
    }
    if (active && t == 0) a.out[2 * idx] = s * ip.dx[0];
}

// an integer as a double: behind the exponent of 2^52, one FP64 addition
__device__ __forceinline__ double int64_of(int m)
{
    return __hiloint2double(0x43300000, (int)((unsigned)m ^ 0x80000000u)) - 4503601774854144.0;  // 2^52 + 2^31
}

// The potential's sum over a thread's points in FP64, nine FP64 instructions a point.
// cos k x of point t + T e is that of the sum of k x_t and k T e dx.  The lanes of a
// warp form the second ones' cosines and sines once, one e each, and pass them round:
// two roundings a point whatever its e, where the recurrence c_{e+1} = 2 cos(k T dx)
// c_e - c_{e-1} reached 1.7e-14 at e = 15 and a cosine for every point takes 45
// instructions.  The points are read from memory, and once more for the transform: over
// its registers the loop spilled.  c2 = mu omega^2 / 2.  Every lane of a warp calls this.
template <int N, int E>
__device__ __forceinline__ double potential_fp64(const DevInst &ip, const cpx<double> *psi, bool active, int t, double c2)
{
    constexpr int T = N / E, GW = T < E ? T : E;  // lanes that share the E cosines: of one team
    const double hs = 0.5 * ip.sigma, dx = ip.dx[0], xc = ip.xc[0];
    const int kind = ip.eps != 0.0 ? ip.vi_kind : HFS_VI_NONE, lane = threadIdx.x & 31;
    bool cosine = kind == HFS_VI_COS;
    if constexpr (T < 32) cosine = __any_sync(0xffffffffu, cosine);
    double ac = 0.0, as = 0.0, bc[E / GW], bs[E / GW];
    if (cosine) {
        // a neighbour's lanes in a warp of several teams add zero
        const double eps = kind == HFS_VI_COS ? ip.eps : 0.0, k = kind == HFS_VI_COS ? ip.vi_k : 0.0;
        sincos(k * fma(int64_of(t - N / 2), dx, xc), &as, &ac);
        ac *= eps;
        as *= -eps;
#pragma unroll
        for (int j = 0; j < E / GW; ++j) sincos(k * (int64_of(T * ((lane & (GW - 1)) + GW * j)) * dx), &bs[j], &bc[j]);
    }
    double pot = 0.0;
#pragma unroll 4
    for (int e = 0; e < E; ++e) {
        const cpx<double> v = active ? psi[t + T * e] : cpx<double>{0.0, 0.0};
        const double vx = v.x, vy = v.y, x = fma(int64_of(t + T * e - N / 2), dx, xc);
        const double d = fma(vx, vx, vy * vy), xx = x * x;
        double w = fma(hs, d, c2 * xx);
        if (cosine) {
            const int from = (lane & ~(GW - 1)) | (e & (GW - 1));
            const bool second = e >= GW;
            const double c = __shfl_sync(0xffffffffu, bc[second ? E / GW - 1 : 0], from);
            const double sn = __shfl_sync(0xffffffffu, bs[second ? E / GW - 1 : 0], from);
            w = fma(as, sn, fma(ac, c, w));
        }
        if (kind == HFS_VI_X4) w = fma(ip.eps * xx, xx, w);
        pot = fma(w, d, pot);
    }
    return pot;
}

// What the FP32 energy needs of an instance, in units of the mesh: x = (m + r) dx,
// the trap as a m^2, eps V_I as b m^4 or cos, sin of k T dx.  a.hi is NaN where a
// parameter is outside the range of the pairs (the instance is summed in FP64).
struct alignas(16) EnergyPre {
    Pair r, a, b, e;
};
static_assert(sizeof(EnergyPre) == sizeof(StageFGE), "one record per instance");

// The same sum of an FP32 state in pairs (products and sums to 2^-46, against
// 1e-8 of the transform), about 100 FP32 instructions a point and FP64 only for
// the first cosines.  One copy of the code for all plans, reading the points from
// memory: unrolled over registers it spilled, and its fetch cost more than its
// issue.
__device__ __noinline__ Pair potential_pairs(const DevInst &ip, const EnergyPre &pre, Pair hs, const cpx<float> *psi, int t,
                                             int T, int E)
{
    const int kind = ip.vi_kind_eff, n = T * E;
    Pair c{}, cn{};
    if (kind == HFS_VI_COS) {
        const double g = (double)pre.b.hi + (double)pre.b.lo, sg = (double)pre.e.hi + (double)pre.e.lo;
        double sn, cs;
        sincos(ip.vi_k * (ip.xc[0] + (double)(t - n / 2) * ip.dx[0]), &sn, &cs);
        c = to_pair(ip.eps * cs);
        cn = to_pair(ip.eps * (cs * g - sn * sg));
    }
    const Pair r = pre.r, a = pre.a, b = pre.b, f{2.0f * b.hi, 2.0f * b.lo};
    Pair pot{};
    float den = 0.0f;
#pragma unroll 1
    for (int e0 = 0; e0 < E; e0 += 4) {
        cpx<float> v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = psi[t + T * (e0 + e)];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const Pair m = two_sum((float)(t - n / 2 + T * (e0 + e)), r.hi), x = quick_sum(m.hi, m.lo + r.lo);
            const Pair xx = mul(x, x), d = abs2(v[e]);
            Pair w = add(mul(a, xx), mul(hs, d));
            if (kind == HFS_VI_COS) {
                w = add(w, c);
                const Pair p = mul(f, cn), next = add(p, Pair{-c.hi, -c.lo});
                c = cn;
                cn = next;
            } else if (kind == HFS_VI_X4) {
                w = add(w, mul(b, mul(xx, xx)));
            }
            pot = add(pot, mul(w, d));
            den += d.hi;
        }
    }
    if (!(den < 1e6f)) pot.hi = __int_as_float(0x7fffffff);
    return pot;
}
// and in FP64 for a state that the pairs do not hold
__device__ __noinline__ double potential_wide(const DevInst &ip, double now, const cpx<float> *psi, int t, int T, int E)
{
    const double c2 = 0.5 * ip.mu * law_omega2(ip, now);
    double pot = 0.0;
#pragma unroll 1
    for (int e = 0; e < E; ++e) {
        const int j = t + T * e;
        const double x = ip.xc[0] + (double)(j - T * E / 2) * ip.dx[0], vx = psi[j].x, vy = psi[j].y;
        const double d = fma(vx, vx, vy * vy), xx = x * x;
        double w = fma(0.5 * ip.sigma, d, c2 * xx);
        if (ip.vi_kind_eff == HFS_VI_COS) w = fma(ip.eps, cos(ip.vi_k * x), w);
        if (ip.vi_kind_eff == HFS_VI_X4) w = fma(ip.eps * xx, xx, w);
        pot = fma(w, d, pot);
    }
    return pot;
}

// Energy.  4096 mixed-size FP32 instances: norm and energy took 1.19 ms together
// (copies included) as two runs of one kernel with cos and all sums in FP64,
// 0.32 ms with cos by recurrence and the kinetic sum in pairs, which left the FP64
// pipe 62 % (energy) and 80 % (norm) busy; 0.17 ms with every sum of an FP32 state
// in floats and two CTAs an SM (128 registers; FP64 sums over registers took 255).
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
    if constexpr (sizeof(R) == 4) {
        const EnergyPre pre = reinterpret_cast<const EnergyPre *>(a.pre)[idx];
        Pair pot{};
        if (active) pot = potential_pairs(ip, pre, reinterpret_cast<const Pair *>(a.out)[2 * idx], psi, t, T, E);
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = active ? psi[t + T * e] : cpx<R>{R(0), R(0)};
        FftPlan<N, E, ALT>::template run<false, R, 1, true>(v, sm, t, tw, 1 + g);
        Pair kin{};
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const float m = (float)(t + T * e - (2 * e < E ? 0 : N));  // m^2 is exact
            const Pair d = abs2(v[e]);
            kin = add(kin, mul(Pair{m * m, 0.0f}, d));
        }
        const double s = team_sum<T>(kin, slots), p = team_sum<T>(pot, slots);
        // pairs hold 46 bits while squares stay clear of FP32's range: sum |v|^2 >=
        // 4 s / N^3; a state of another size (or not finite) is summed in FP64
        bool pairs = !active || (s > 1e-12 * N * N * N && s < 1e30 && p > -1e30 && p < 1e30);
        if constexpr (T < 32) pairs = __all_sync(0xffffffffu, pairs);
        if (pairs) {
            if (active && t == 0) a.out[2 * idx + 1] = fma(s, a.out[2 * idx + 1], p) * ip.dx[0];
            return;
        }
    }
    double pot = 0.0, kin = 0.0;
    if constexpr (sizeof(R) == 4) {
        if (active) pot = potential_wide(ip, *a.t_dev, psi, t, T, E);
        // in a loop through the exchange buffer: its last readers are behind team_sum
#pragma unroll
        for (int e = 0; e < E; ++e) sm[t + T * e] = v[e];
#pragma unroll 1
        for (int e = 0; e < E; ++e) {
            const double m = t + T * e - (2 * e < E ? 0 : N), vx = sm[t + T * e].x, vy = sm[t + T * e].y;
            kin = fma(m * m, fma(vx, vx, vy * vy), kin);
        }
    } else {
        const double c2 = a.pre[idx].f;
        pot = potential_fp64<N, E>(ip, psi, active, t, c2);
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = active ? psi[t + T * e] : cpx<R>{R(0), R(0)};
        FftPlan<N, E, ALT>::template run<false, R, 1, true>(v, sm, t, tw, 1 + g);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int m = t + T * e - (2 * e < E ? 0 : N);
            kin = fma(square64(m), fma(v[e].x, v[e].x, v[e].y * v[e].y), kin);
        }
    }
    kin = team_sum<T>(kin, slots);
    pot = team_sum<T>(pot, slots);
    if (active && t == 0) a.out[2 * idx + 1] = fma(kin, a.out[2 * idx + 1], pot) * ip.dx[0];
}

// What every thread of an instance needs, once per instance: mu omega^2 / 2 and the
// kinetic factor, for an FP32 state cos, sin of k T dx as well, all in pairs (with the
// law's sine and this sincos in every thread the two calls took 0.34 ms).  One
// thread per instance: a CTA per work item left most lanes idle (16 us for 4096
// instances, 11 us now, the latency of one thread).  The energy's slots of out
// hold the kinetic factor and, for an FP32 state, sigma / 2 until it is written.
template <typename R> __global__ void energy_pre_kernel(const Diag1DArgs a)
{
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= a.count) return;
    const DevInst &ip = a.inst[idx];
    const int n = ip.n[0];
    const double ku = 2.0 * 3.14159265358979323846 / ip.len[0];
    a.out[2 * idx + 1] = ku * ku / n / (2.0 * ip.mu);
    const double c2 = 0.5 * ip.mu * law_omega2(ip, *a.t_dev);
    if constexpr (sizeof(R) == 8) {
        StageFGE r{};
        r.f = c2;
        a.pre[idx] = r;
    } else {
        double sn, cs;
        sincos(ip.vi_k * (ip.dx[0] * (n / a.ept[size_class(n)])), &sn, &cs);
        const double dx = ip.dx[0], d2 = dx * dx, ca = c2 * d2, cb = ip.eps * d2 * d2, r = ip.xc[0] / dx;
        const bool cosine = ip.vi_kind_eff == HFS_VI_COS;
        // zero, or within 1e-12 .. 1e8: with |m + r| <= 1e5 and |psi|^2 <= 1e6 no
        // product leaves FP32's range and no error term that counts underflows
        auto fits = [](double c) { return c == 0.0 || (fabs(c) >= 1e-12 && fabs(c) <= 1e8); };
        const bool ok = fabs(r) <= 9e4 && fits(ca) && fits(0.5 * ip.sigma) && fits(cosine ? ip.eps : cb);
        EnergyPre p;
        p.r = to_pair(r);
        p.a = ok ? to_pair(ca) : Pair{__int_as_float(0x7fffffff), 0.0f};
        p.b = to_pair(cosine ? cs : cb);
        p.e = to_pair(sn);
        reinterpret_cast<EnergyPre *>(a.pre)[idx] = p;
        reinterpret_cast<Pair *>(a.out)[2 * idx] = to_pair(0.5 * ip.sigma);
    }
}

// items of a batch hold about the same number of points each, so CTAs take them
// in turn
template <typename R, bool ENERGY>
__global__ void __launch_bounds__(kCtaThreads, sizeof(R) == 8 ? 1 : ENERGY ? 2 : 4) diag1d_kernel(const Diag1DArgs a)
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
    if (ENERGY) energy_pre_kernel<R><<<(unsigned)((a.count + 63) / 64), 64, 0, st>>>(a);
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
