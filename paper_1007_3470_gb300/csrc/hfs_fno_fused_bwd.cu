// hfs_fno_fused_bwd.cu -- the surrogate's backward pass and optimizer step in
// 2 layers + 4 kernels, the mirror image of hfs_fno_fused.cu: a CTA takes a
// sample from one mixing product back to the one before it,
//   head:   dO of the loss, dQ, dH of the projection and its gradients (rows of
//           all samples in tiles of 128);
//   layer:  dH = dZ_up W_up^T + F2^T dS_up, dZ = dH GELU'(Z), dY = G^T dZ, and
//           H^T dZ summed over the CTA's samples;
//   mix:    dS_k = dY_k R_k^T (64 samples a CTA) and the gradient of R_k (16
//           rows a CTA, all samples).
// GEMM by GEMM this took 80 launches that wrote and re-read dQ, dZ, dH in FP32
// and BF16: a training step of 256 samples (256 x 64, 32 modes, 4 layers) took
// 1.24 ms, with the fused kernels 0.30 ms.  Operands round to BF16 where the GEMM form rounds them, sums and
// gradients are FP32.
#include <algorithm>

#include "hfs_fno_frag.cuh"
#include "hfs_fno_fused.h"

namespace hfs {
namespace fno {

namespace {

constexpr int kThreads = 512, kWarps = 16;
constexpr int kHeadRows = 128;

__host__ __device__ inline int modes_pad(int M) { return M < 16 ? 16 : M; }

// two adjacent gradient entries; their vector form needs an 8-byte boundary
__device__ __forceinline__ void grad_add2(float *p, float a, float b)
{
    if (((uintptr_t)p & 7) == 0) {
        asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b) : "memory");
    } else {
        atomicAdd(p, a);
        atomicAdd(p + 1, b);
    }
}
// an accumulator's 8 NT columns at (m0, n0) of a row-major gradient
template <int NT>
__device__ __forceinline__ void grad_add(float *g, int ld, int m0, int n0, const float (&c)[NT][4], int lane)
{
    const int r = m0 + (lane >> 2), q = n0 + (lane & 3) * 2;
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        grad_add2(g + (int64_t)r * ld + q + 8 * j, c[j][0], c[j][1]);
        grad_add2(g + (int64_t)(r + 8) * ld + q + 8 * j, c[j][2], c[j][3]);
    }
}

__device__ __forceinline__ float cta_sum(const float *p, int n, int stride)
{
    float v = 0.0f;
    for (int i = 0; i < n; ++i) v += p[i * stride];
    return v;
}

// ---------------------------------------------------------------------------
// projection
// ---------------------------------------------------------------------------
template <int C> __host__ __device__ constexpr int head_units() { return C >= 32 ? C / 32 : 1; }

size_t head_smem(int C, int P)
{
    return (size_t)kHeadRows * P * 2 + (size_t)kHeadRows * C * 2 + (size_t)C * P * 2 + (size_t)kHeadRows * 8 * 4;
}

// Bound by erff and expf on the FP32 and MUFU pipes (2 x 128 values a row) and
// by Qpre's 4 P bytes a row.  A thread keeps one pair of columns of Q, so the
// column sums of c1 and P2 stay in its registers over all rows.  65536 rows with
// P = 128: 49 us, 78 us before the rows' loads were grouped and the sums added
// once per CTA.
template <int C, int OCM>
__global__ void __launch_bounds__(kThreads) head_bwd_kernel(const HeadBwdArgs a)
{
    constexpr int LGC = ilog2(C / 8), U = head_units<C>();
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const int P = a.d.P, L = a.d.L, oc = a.d.out_ch, lgP = 31 - __clz(P >> 3), lgL = 31 - __clz(L);
    bf16 *Qs = reinterpret_cast<bf16 *>(smem_raw);        // [128][P]
    bf16 *P1s = Qs + kHeadRows * P;                       // [C][P]
    bf16 *Hs = P1s + C * P;                               // [128][C]
    float *dOs = reinterpret_cast<float *>(Hs + kHeadRows * C);  // [128][8], rounded to BF16
    const uint32_t Qa = smem_u32(Qs), Pa = smem_u32(P1s), Ha = smem_u32(Hs);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const LaneAt lc = lane_at(lane, LGC), lp = lane_at(lane, lgP);
    const int64_t rows = (int64_t)a.B * L;
    tile_load(P1s, lgP, 0, C, lgP, a.P1b, P, tid, kThreads);
    const int pairs = P >> 1, groups = kThreads / pairs, col = (tid & (pairs - 1)) * 2, rg = tid / pairs;
    float p2[2][OCM], gp2[2][OCM], gc1[2] = {0.0f, 0.0f}, gc2[OCM];
#pragma unroll
    for (int o = 0; o < OCM; ++o) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            p2[i][o] = o < oc ? __bfloat162float(a.P2b[(col + i) * oc + o]) : 0.0f;
            gp2[i][o] = 0.0f;
        }
        gc2[o] = 0.0f;
    }
    float gp1[U][2][4], gb[U][4];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        zero_acc(gp1[u]);
#pragma unroll
        for (int q = 0; q < 4; ++q) gb[u][q] = 0.0f;
    }
    pdl_wait();
    pdl_trigger();
    for (int64_t r0 = (int64_t)blockIdx.x * kHeadRows; r0 < rows; r0 += (int64_t)gridDim.x * kHeadRows) {
        const int valid = (int)(rows - r0 < kHeadRows ? rows - r0 : kHeadRows);
        tile_load(Hs, LGC, 0, kHeadRows, LGC, a.H + r0 * C, C, tid, kThreads, valid);
        if (tid < kHeadRows) {
            const int64_t b = (r0 + tid) >> lgL;
            float nd = 0.0f;
            if (tid < valid) nd = sqrtf(a.sums[2 * b] * a.sums[2 * b + 1]);
#pragma unroll
            for (int o = 0; o < OCM; ++o) {
                float v = 0.0f;
                if (tid < valid && o < oc && nd > 0.0f) {
                    const int64_t i = (r0 + tid) * oc + o;
                    v = (a.O[i] - a.y[i]) / (nd * (float)a.B);
                }
                gc2[o] += v;
                dOs[tid * 8 + o] = __bfloat162float(__float2bfloat16(v));
            }
        }
        __syncthreads();
        for (int r8 = rg; r8 < kHeadRows; r8 += 8 * groups) {
            float2 zs[8];  // the loads of eight rows in flight
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int r = r8 + i * groups;
                zs[i] = r < valid ? *reinterpret_cast<const float2 *>(a.Qpre + (r0 + r) * P + col) : make_float2(0.0f, 0.0f);
            }
#pragma unroll 1
            for (int i = 0; i < 8; i += 2) {  // two rows' chains of erff and expf side by side
                if (r8 + i * groups >= kHeadRows) break;
                float e[4], v[2], q[4];
                const float z[4] = {zs[0].x, zs[0].y, zs[1].x, zs[1].y};
#pragma unroll
                for (int k = 0; k < 6; ++k) zs[k] = zs[k + 2];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    e[k] = 1.0f + erff(z[k] * 0.70710678118654752f);
                    q[k] = __bfloat162float(__float2bfloat16(0.5f * z[k] * e[k]));
                    e[k] = 0.5f * e[k] + z[k] * expf(-0.5f * z[k] * z[k]) * 0.39894228040143268f;
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = r8 + (i + h) * groups;
                    if (r >= kHeadRows) break;
                    // dO is zero in rows past the end, and with it their dQ and sums
                    v[0] = v[1] = 0.0f;
#pragma unroll
                    for (int o = 0; o < OCM; ++o) {
                        const float d = dOs[r * 8 + o];
                        v[0] = fmaf(d, p2[0][o], v[0]);
                        v[1] = fmaf(d, p2[1][o], v[1]);
                        gp2[0][o] = fmaf(q[2 * h], d, gp2[0][o]);
                        gp2[1][o] = fmaf(q[2 * h + 1], d, gp2[1][o]);
                    }
                    v[0] *= e[2 * h];
                    v[1] *= e[2 * h + 1];
                    gc1[0] += v[0];
                    gc1[1] += v[1];
                    *reinterpret_cast<unsigned *>(Qs + tile_at(r, col >> 3, lgP) + (col & 7)) = pack2(v[0], v[1]);
                }
            }
        }
        cp_wait_all();
        __syncthreads();
#pragma unroll
        for (int u = 0; u < U; ++u) {
            // gradient of P1: 16 channels x 16 columns of Q a unit, all 128 rows
            const int w = warp + kWarps * u, m0 = (w % (C / 16)) * 16, n0 = (w / (C / 16)) * 16;
            if (n0 < P) {
#pragma unroll
                for (int k0 = 0; k0 < kHeadRows; k0 += 16) {
                    unsigned af[4], bf[4];
                    frag_a_t(af, Ha, lc, LGC, m0, k0);
                    frag_b(bf, Qa, lp, lgP, k0, n0);
                    mma16(gp1[u][0], gp1[u][1], af, bf);
                }
            }
            // dH = dQ P1^T: 16 rows x 16 channels a unit
            const int mr = (w % 8) * 16, nc = (w / 8) * 16;
            if (nc < C) {
                float h[2][4];
                zero_acc(h);
#pragma unroll 4
                for (int k0 = 0; k0 < P; k0 += 16) {
                    unsigned af[4], bf[4];
                    frag_a(af, Qa, lp, lgP, mr, k0);
                    frag_b_nk(bf, Pa, lp, lgP, k0, nc);
                    mma16(h[0], h[1], af, bf);
                }
                const int r = mr + (lane >> 2), c = nc + (lane & 3) * 2;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    gb[u][2 * j] += h[j][0] + h[j][2];
                    gb[u][2 * j + 1] += h[j][1] + h[j][3];
                    if (r < valid) *reinterpret_cast<unsigned *>(a.dZ + (r0 + r) * C + c + 8 * j) = pack2(h[j][0], h[j][1]);
                    if (r + 8 < valid)
                        *reinterpret_cast<unsigned *>(a.dZ + (r0 + r + 8) * C + c + 8 * j) = pack2(h[j][2], h[j][3]);
                }
            }
        }
        __syncthreads();
    }
    // sums over the CTA's rows, each entry added once per CTA (added by every
    // warp, hundreds of additions to the same few addresses were the longest
    // part of the kernel's end)
    float *red = reinterpret_cast<float *>(smem_raw);
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int w = warp + kWarps * u, m0 = (w % (C / 16)) * 16, n0 = (w / (C / 16)) * 16;
        if (n0 < P) grad_add<2>(a.gP1, P, m0, n0, gp1[u], lane);
        const int nc = (w / 8) * 16;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int s = 4; s < 32; s <<= 1) gb[u][q] += __shfl_xor_sync(0xffffffffu, gb[u][q], s);
        // channels nc .. nc + 15 from the eight warps of their rows
        if (nc < C && lane < 4) {
#pragma unroll
            for (int q = 0; q < 4; ++q) red[(w % 8) * C + nc + (q >> 1) * 8 + lane * 2 + (q & 1)] = gb[u][q];
        }
    }
    __syncthreads();
    if (tid < C) atomicAdd(a.gb + tid, cta_sum(red + tid, 8, C));
    // columns of Q from the groups of rows
    __syncthreads();
    red[2 * tid] = gc1[0];
    red[2 * tid + 1] = gc1[1];
    __syncthreads();
    if (tid < P) atomicAdd(a.gc1 + tid, cta_sum(red + tid, groups, P));
#pragma unroll
    for (int o = 0; o < OCM; ++o) {
        if (o >= oc) break;
        __syncthreads();
        red[2 * tid] = gp2[0][o];
        red[2 * tid + 1] = gp2[1][o];
        __syncthreads();
        if (tid < P) atomicAdd(a.gP2 + tid * oc + o, cta_sum(red + tid, groups, P));
        float v = gc2[o];
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
        if (lane == 0 && tid < kHeadRows) atomicAdd(a.gc2 + o, v);
    }
}

// ---------------------------------------------------------------------------
// layer
// ---------------------------------------------------------------------------
struct LayerSmem {
    int Z, H, G, F2, W, dS, X, total;
};
__host__ __device__ inline LayerSmem layer_smem(int L, int C, int M, LayerBwd mode)
{
    LayerSmem s{};
    const int Mp = modes_pad(M);
    int o = 0;
    auto take = [&](int bytes) {
        const int at = o;
        o += bytes;
        return at;
    };
    s.Z = take(L * C * 2);
    if (mode != LayerBwd::kLift) {
        s.H = take(L * C * 2);
        s.G = take(L * 2 * Mp * 2);
    }
    if (mode != LayerBwd::kTop) {
        s.F2 = take(2 * M * L * 2);
        s.W = take(C * C * 2);
        s.dS = take(2 * M * C * 2);
    }
    if (mode == LayerBwd::kLift) s.X = take((L + 1) * 16);
    s.total = o > 16384 ? o : 16384;  // the warps' sums at the end: at most [16][8][32] floats
    return s;
}

// Bound by the tensor pipe and latency at one CTA of 16 warps an SM (the
// sample's tiles and the two transforms' matrices take 144 KB at 256 x 64 with
// 32 modes).  Warps own 16 rows of L for dZ; then one part of them takes blocks
// of dY, the other keeps a block of the gradient of W over all samples.  256
// samples: 24 us a layer (34 us with every warp adding its own column sums to
// the gradient), 12 us for the last and the lift.
template <int C, LayerBwd MODE>
__global__ void __launch_bounds__(kThreads) layer_bwd_kernel(const LayerBwdArgs a)
{
    constexpr int NT = C / 8, LGC = ilog2(C / 8);
    constexpr int SN = C >= 32 ? 4 : 2, NG = C / (8 * SN);  // n-tiles of a block, blocks across C
    constexpr int WU = (C / 16) * NG;                       // blocks of the gradient of W
    static_assert(WU < kWarps, "a warp for each block of W and one for dY");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const int L = a.d.L, M = a.d.M, Mp = modes_pad(M);
    const int lgL = 31 - __clz(L >> 3), lgG = 31 - __clz(Mp >> 2);
    const LayerSmem so = layer_smem(L, C, M, MODE);
    bf16 *Zs = reinterpret_cast<bf16 *>(smem_raw + so.Z), *Hs = reinterpret_cast<bf16 *>(smem_raw + so.H);
    bf16 *Gs = reinterpret_cast<bf16 *>(smem_raw + so.G), *Fs = reinterpret_cast<bf16 *>(smem_raw + so.F2);
    bf16 *Ws = reinterpret_cast<bf16 *>(smem_raw + so.W), *Ds = reinterpret_cast<bf16 *>(smem_raw + so.dS);
    bf16 *Xs = reinterpret_cast<bf16 *>(smem_raw + so.X);
    const uint32_t Za = smem_u32(Zs), Ha = smem_u32(Hs), Ga = smem_u32(Gs), Fa = smem_u32(Fs), Wa = smem_u32(Ws),
                   Da = smem_u32(Ds), Xa = smem_u32(Xs);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, t2 = (lane & 3) * 2;
    const LaneAt lc = lane_at(lane, LGC), lg = lane_at(lane, lgG), ll = lane_at(lane, lgL);
    if constexpr (MODE != LayerBwd::kLift) {
        const int lgm = 31 - __clz(M >> 3);
        for (int part = 0; part < 2; ++part) {
            const bf16 *src = part ? a.Gim : a.Gre;
            for (int u = tid; u < (L << lgm); u += kThreads) {
                const int r = u >> lgm, c = u & ((1 << lgm) - 1);
                cp16(Gs + tile_at(r, part * (Mp >> 3) + c, lgG), src + (int64_t)r * M + c * 8, true);
            }
        }
        if (M < Mp)
            for (int u = tid; u < 2 * L; u += kThreads)
                *reinterpret_cast<uint4 *>(Gs + tile_at(u >> 1, (u & 1) * (Mp >> 3) + 1, lgG)) = make_uint4(0, 0, 0, 0);
    }
    if constexpr (MODE != LayerBwd::kTop) {
        tile_load(Fs, lgL, 0, 2 * M, lgL, a.F2, L, tid, kThreads);
        tile_load(Ws, LGC, 0, C, LGC, a.Wup, C, tid, kThreads);
    }
    if (MODE == LayerBwd::kLift && tid < 8) Xs[L * 8 + tid] = __float2bfloat16(0.0f);
    float gb[NT][2], gw[SN][4];
    zero_acc(gw);
#pragma unroll
    for (int j = 0; j < NT; ++j) gb[j][0] = gb[j][1] = 0.0f;
    pdl_wait();
    pdl_trigger();
    for (int b = blockIdx.x; b < a.B; b += gridDim.x) {
        const int64_t base = (int64_t)b * L * C;
        tile_load(Zs, LGC, 0, L, LGC, a.dZ + base, C, tid, kThreads);
        if constexpr (MODE != LayerBwd::kTop) {
            for (int u = tid; u < ((2 * M) << LGC); u += kThreads) {
                const int r = u >> LGC, c = u & (NT - 1);
                cp16(Ds + tile_at(r, c, LGC), a.dSup + ((int64_t)r * a.d.Bm + b) * C + c * 8, true);
            }
        }
        if constexpr (MODE != LayerBwd::kLift) tile_load(Hs, LGC, 0, L, LGC, a.Hin + base, C, tid, kThreads);
        if constexpr (MODE == LayerBwd::kLift) {
            for (int u = tid; u < L * 8; u += kThreads)
                Xs[u] = __float2bfloat16((u & 7) < a.d.in_ch ? a.x[((int64_t)b * L + (u >> 3)) * a.d.in_ch + (u & 7)]
                                                             : 0.0f);
        }
        cp_wait_all();
        __syncthreads();
        const int m0 = warp * 16;
        if (MODE != LayerBwd::kTop && m0 < L) {
            float h[NT][4], s[NT][4];
            zero_acc(h);
            zero_acc(s);
#pragma unroll
            for (int k0 = 0; k0 < C; k0 += 16) {
                unsigned af[4];
                frag_a(af, Za, lc, LGC, m0, k0);
#pragma unroll
                for (int j = 0; j < NT; j += 2) {
                    unsigned bf[4];
                    frag_b_nk(bf, Wa, lc, LGC, k0, 8 * j);
                    mma16(h[j], h[j + 1], af, bf);
                }
            }
            for (int k0 = 0; k0 < 2 * M; k0 += 16) {
                unsigned af[4];
                frag_a_t(af, Fa, ll, lgL, m0, k0);
#pragma unroll
                for (int j = 0; j < NT; j += 2) {
                    unsigned bf[4];
                    frag_b(bf, Da, lc, LGC, k0, 8 * j);
                    mma16(s[j], s[j + 1], af, bf);
                }
            }
            const int64_t at = base + (int64_t)(m0 + (lane >> 2)) * C + t2;
#pragma unroll
            for (int j = 0; j < NT; ++j) {
#pragma unroll
                for (int q = 0; q < 4; ++q) h[j][q] = s[j][q] + h[j][q];
                if constexpr (MODE == LayerBwd::kMid) {
                    const float2 z0 = *reinterpret_cast<const float2 *>(a.pre + at + 8 * j);
                    const float2 z1 = *reinterpret_cast<const float2 *>(a.pre + at + 8 * C + 8 * j);
                    h[j][0] *= gelu_grad_f(z0.x);
                    h[j][1] *= gelu_grad_f(z0.y);
                    h[j][2] *= gelu_grad_f(z1.x);
                    h[j][3] *= gelu_grad_f(z1.y);
                }
                gb[j][0] += h[j][0] + h[j][2];
                gb[j][1] += h[j][1] + h[j][3];
            }
            __syncwarp();  // every lane has read the warp's rows of Z
            acc_to_tile(Za, LGC, m0, 0, h, lane);
            if constexpr (MODE == LayerBwd::kMid) {
                __syncwarp();
                for (int u = lane; u < (16 << LGC); u += 32)
                    *reinterpret_cast<uint4 *>(a.dZ + base + (int64_t)(m0 + (u >> LGC)) * C + (u & (NT - 1)) * 8) =
                        *reinterpret_cast<const uint4 *>(Zs + tile_at(m0 + (u >> LGC), u & (NT - 1), LGC));
            }
        }
        __syncthreads();
        if constexpr (MODE == LayerBwd::kLift) {
            // gradient of P_in: 8 inputs x 8 SN channels, rows of L split over the warps
            const int n0 = (warp % NG) * 8 * SN;
            for (int k0 = (warp / NG) * 16; k0 < L; k0 += (kWarps / NG) * 16) {
                unsigned af[4];
                const int r = (lane & 8) ? L : k0 + (lane & 7) + ((lane >> 4) & 1) * 8;
                lds_frag_t(af, Xa + r * 16);
#pragma unroll
                for (int j = 0; j < SN; j += 2) {
                    unsigned bf[4];
                    frag_b(bf, Za, lc, LGC, k0, n0 + 8 * j);
                    mma16(gw[j], gw[j + 1], af, bf);
                }
            }
        } else if (warp >= kWarps - WU) {
            const int u = warp - (kWarps - WU), c0 = (u / NG) * 16, n0 = (u % NG) * 8 * SN;
#pragma unroll 4
            for (int k0 = 0; k0 < L; k0 += 16) {
                unsigned af[4];
                frag_a_t(af, Ha, lc, LGC, c0, k0);
#pragma unroll
                for (int j = 0; j < SN; j += 2) {
                    unsigned bf[4];
                    frag_b(bf, Za, lc, LGC, k0, n0 + 8 * j);
                    mma16(gw[j], gw[j + 1], af, bf);
                }
            }
        } else {
            for (int u = warp; u < (Mp >> 3) * NG; u += kWarps - WU) {
                const int k = (u / NG) * 16, n0 = (u % NG) * 8 * SN;
                float y[SN][4];
                zero_acc(y);
#pragma unroll 4
                for (int k0 = 0; k0 < L; k0 += 16) {
                    unsigned af[4];
                    frag_a_t(af, Ga, lg, lgG, k, k0);
#pragma unroll
                    for (int j = 0; j < SN; j += 2) {
                        unsigned bf[4];
                        frag_b(bf, Za, lc, LGC, k0, n0 + 8 * j);
                        mma16(y[j], y[j + 1], af, bf);
                    }
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int r = k + (lane >> 2) + 8 * q, part = r >= Mp, mode = r - part * Mp;
                    if (mode >= M) continue;
                    bf16 *dst = a.dY + ((int64_t)mode * a.d.Bm + b) * 2 * C + part * C + n0 + t2;
#pragma unroll
                    for (int j = 0; j < SN; ++j)
                        *reinterpret_cast<unsigned *>(dst + 8 * j) = pack2(y[j][2 * q], y[j][2 * q + 1]);
                }
            }
        }
        __syncthreads();
    }
    float *red = reinterpret_cast<float *>(smem_raw);
    if constexpr (MODE != LayerBwd::kTop) {
#pragma unroll
        for (int j = 0; j < NT; ++j) {
#pragma unroll
            for (int s = 4; s < 32; s <<= 1) {
                gb[j][0] += __shfl_xor_sync(0xffffffffu, gb[j][0], s);
                gb[j][1] += __shfl_xor_sync(0xffffffffu, gb[j][1], s);
            }
            if (lane < 4) *reinterpret_cast<float2 *>(red + warp * C + 8 * j + t2) = make_float2(gb[j][0], gb[j][1]);
        }
        __syncthreads();
        if (tid < C) atomicAdd(a.gb + tid, cta_sum(red + tid, kWarps, C));
    }
    if constexpr (MODE == LayerBwd::kLift) {
        // rows 0..7 of the warps' blocks: [warp / NG][8][C]
        __syncthreads();
        float *w = red + ((warp / NG) * 8 + (lane >> 2)) * C + (warp % NG) * 8 * SN + t2;
#pragma unroll
        for (int j = 0; j < SN; ++j) *reinterpret_cast<float2 *>(w + 8 * j) = make_float2(gw[j][0], gw[j][1]);
        __syncthreads();
        for (int i = tid; i < a.d.in_ch * C; i += kThreads) atomicAdd(a.gW + i, cta_sum(red + i, kWarps / NG, 8 * C));
    } else if (warp >= kWarps - WU) {
        const int u = warp - (kWarps - WU);
        grad_add<SN>(a.gW, C, (u / NG) * 16, (u % NG) * 8 * SN, gw, lane);
    }
}

// ---------------------------------------------------------------------------
// mixing product
// ---------------------------------------------------------------------------
constexpr int kMixRows = 64;
template <int C> constexpr size_t mix_bwd_smem()
{
    const size_t ds = (size_t)(kMixRows * 2 * C + 2 * C * 2 * C) * 2;
    const size_t dr = (size_t)2 * (2 * kMixRows * 16 + kMixRows * 2 * C) * 2;
    return ds > dr ? ds : dr;
}

template <int C>
__global__ void __launch_bounds__(256) mix_bwd_kernel(const FusedDims d, int B, const bf16 *__restrict__ S,
                                                      const bf16 *__restrict__ dY, const bf16 *__restrict__ R1,
                                                      const bf16 *__restrict__ R2, bf16 *__restrict__ dS,
                                                      float *__restrict__ gRre, float *__restrict__ gRim)
{
    constexpr int NT = C / 8, LGC = ilog2(C / 8), LG2 = LGC + 1;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, k = blockIdx.y;
    const int tiles = (B + kMixRows - 1) / kMixRows;
    const LaneAt l2 = lane_at(lane, LG2);
    if ((int)blockIdx.x < tiles) {
        // dS of 64 samples: rows of 16, the two parts in alternate warps
        bf16 *Rs = reinterpret_cast<bf16 *>(smem_raw), *Ys = Rs + 4 * C * C;
        const uint32_t Ra = smem_u32(Rs), Ya = smem_u32(Ys);
        const int b0 = blockIdx.x * kMixRows, m0 = (warp >> 1) * 16, part = warp & 1;
        tile_load(Rs, LG2, 0, C, LG2, R1 + (int64_t)k * C * 2 * C, 2 * C, tid, 256);
        tile_load(Rs, LG2, C, C, LG2, R2 + (int64_t)k * C * 2 * C, 2 * C, tid, 256);
        pdl_wait();
        pdl_trigger();
        tile_load(Ys, LG2, 0, kMixRows, LG2, dY + ((int64_t)k * d.Bm + b0) * 2 * C, 2 * C, tid, 256, B - b0);
        cp_wait_all();
        __syncthreads();
        float s[NT][4];
        zero_acc(s);
#pragma unroll
        for (int k0 = 0; k0 < 2 * C; k0 += 16) {
            unsigned af[4];
            frag_a(af, Ya, l2, LG2, m0, k0);
#pragma unroll
            for (int j = 0; j < NT; j += 2) {
                unsigned bf[4];
                frag_b_nk(bf, Ra, l2, LG2, k0, part * C + 8 * j);
                mma16(s[j], s[j + 1], af, bf);
            }
        }
        __syncthreads();
        acc_to_tile(Ya, LGC, part * kMixRows + m0, 0, s, lane);
        __syncwarp();
        for (int i = lane; i < 16 * NT; i += 32) {
            const int r = m0 + i / NT, c = i % NT;
            if (b0 + r < B)
                *reinterpret_cast<uint4 *>(dS + ((int64_t)(part * d.M + k) * d.Bm + b0 + r) * C + c * 8) =
                    *reinterpret_cast<const uint4 *>(Ys + tile_at(part * kMixRows + r, c, LGC));
        }
    } else {
        // gradient of 16 rows of R_re and R_im over all samples: the four
        // products S_re dY_re, S_im dY_im, S_re dY_im, S_im dY_re in pairs of warps
        constexpr int NH = C / 2 > 16 ? C / 2 : 16;  // columns a warp
        bf16 *Ss = reinterpret_cast<bf16 *>(smem_raw);  // two of [2][64][16]
        bf16 *Ys = Ss + 2 * 2 * kMixRows * 16;          // two of [64][2C]
        const int c0 = ((int)blockIdx.x - tiles) * 16;
        const int prod = warp >> 1, half = warp & 1, sp = prod & 1, yp = prod == 1 || prod == 2;
        const bool busy = half * NH < C;
        const LaneAt l1 = lane_at(lane, 1);
        pdl_wait();
        pdl_trigger();
        auto load = [&](int tile, int buf) {
            if (tile < tiles) {
                const int b0 = tile * kMixRows;
                for (int part = 0; part < 2; ++part)
                    tile_load(Ss + buf * 2 * kMixRows * 16, 1, part * kMixRows, kMixRows, 1,
                              S + ((int64_t)(part * d.M + k) * d.Bm + b0) * C + c0, C, tid, 256, B - b0);
                tile_load(Ys + buf * kMixRows * 2 * C, LG2, 0, kMixRows, LG2, dY + ((int64_t)k * d.Bm + b0) * 2 * C,
                          2 * C, tid, 256, B - b0);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        float r[NH / 8][4];
        zero_acc(r);
        load(0, 0);
        for (int tile = 0; tile < tiles; ++tile) {
            load(tile + 1, (tile + 1) & 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncthreads();
            const uint32_t Sa = smem_u32(Ss + (tile & 1) * 2 * kMixRows * 16) + sp * kMixRows * 32;
            const uint32_t Ya = smem_u32(Ys + (tile & 1) * kMixRows * 2 * C);
            if (busy) {
#pragma unroll
                for (int k0 = 0; k0 < kMixRows; k0 += 16) {
                    unsigned af[4];
                    frag_a_t(af, Sa, l1, 1, 0, k0);
#pragma unroll
                    for (int j = 0; j < NH / 8; j += 2) {
                        unsigned bf[4];
                        frag_b(bf, Ya, l2, LG2, k0, yp * C + half * NH + 8 * j);
                        mma16(r[j], r[j + 1], af, bf);
                    }
                }
            }
            __syncthreads();
        }
        float *f = reinterpret_cast<float *>(smem_raw);  // [4][16][C]
        if (busy) {
#pragma unroll
            for (int j = 0; j < NH / 8; ++j) {
                float *w = f + (prod * 16 + (lane >> 2)) * C + half * NH + 8 * j + (lane & 3) * 2;
                *reinterpret_cast<float2 *>(w) = make_float2(r[j][0], r[j][1]);
                *reinterpret_cast<float2 *>(w + 8 * C) = make_float2(r[j][2], r[j][3]);
            }
        }
        __syncthreads();
        for (int i = tid; i < 16 * C; i += 256) {
            const int64_t at = ((int64_t)k * C + c0) * C + i;
            gRre[at] = f[i] + f[16 * C + i];
            gRim[at] = f[2 * 16 * C + i] - f[3 * 16 * C + i];
        }
    }
}

// ---------------------------------------------------------------------------
// optimizer and BF16 weights: 28 bytes a parameter and its copies, one launch
// in place of one for each weight matrix
// ---------------------------------------------------------------------------
template <bool ADAM> __global__ void refresh_kernel(const RefreshArgs r, const AdamArgs a)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= r.n) return;
    float p = r.p[i];
    if constexpr (ADAM) {
        const float gi = a.g[i];
        const float mi = a.b1 * a.m[i] + (1.0f - a.b1) * gi;
        const float vi = a.b2 * a.v[i] + (1.0f - a.b2) * gi * gi;
        a.m[i] = mi;
        a.v[i] = vi;
        p -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
        r.p[i] = p;
    }
    const int C = r.C;
    if (i < r.bin) {
        r.Pinb[i] = __float2bfloat16(p);
    } else if (i >= r.layer0 && i < r.P1) {
        const int64_t o = i - r.layer0, l = o / r.layer_stride, j = o - l * r.layer_stride;
        const int64_t mcc = (int64_t)r.M * C * C;
        if (j < 2 * mcc) {
            const bool im = j >= mcc;
            const int64_t e = im ? j - mcc : j, row = e / C, c = e - row * C;  // row: mode and input channel
            bf16 *R1 = r.R1 + l * 2 * mcc + row * 2 * C + c, *R2 = r.R2 + l * 2 * mcc + row * 2 * C + c;
            R1[im ? C : 0] = __float2bfloat16(p);
            R2[im ? 0 : C] = __float2bfloat16(im ? -p : p);
        } else if (j < 2 * mcc + (int64_t)C * C) {
            r.Wb[l * C * C + (j - 2 * mcc)] = __float2bfloat16(p);
        }
    } else if (i >= r.P1 && i < r.c1) {
        r.P1b[i - r.P1] = __float2bfloat16(p);
    } else if (i >= r.P2 && i < r.c2) {
        r.P2b[i - r.P2] = __float2bfloat16(p);
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
template <int C, int OCM> cudaError_t head_t(const HeadBwdArgs &a, cudaStream_t st)
{
    static ResidentSlot slot;
    const size_t smem = head_smem(C, a.d.P);
    int ctas = 0;
    const cudaError_t e = resident_ctas(slot, head_bwd_kernel<C, OCM>, kThreads, smem, &ctas);
    if (e != cudaSuccess) return e;
    const int64_t tiles = ((int64_t)a.B * a.d.L + kHeadRows - 1) / kHeadRows;
    return launch_k(head_bwd_kernel<C, OCM>, dim3((unsigned)std::min<int64_t>(tiles, ctas)), kThreads, smem, st, true,
                    a);
}

template <int C, LayerBwd MODE> cudaError_t layer_t(const LayerBwdArgs &a, cudaStream_t st)
{
    static ResidentSlot slot;
    const size_t smem = (size_t)layer_smem(a.d.L, C, a.d.M, MODE).total;
    int ctas = 0;
    const cudaError_t e = resident_ctas(slot, layer_bwd_kernel<C, MODE>, kThreads, smem, &ctas);
    if (e != cudaSuccess) return e;
    return launch_k(layer_bwd_kernel<C, MODE>, dim3((unsigned)std::min(a.B, ctas)), kThreads, smem, st, true, a);
}

template <int C> cudaError_t layer_c(const LayerBwdArgs &a, LayerBwd mode, cudaStream_t st)
{
    switch (mode) {
    case LayerBwd::kTop: return layer_t<C, LayerBwd::kTop>(a, st);
    case LayerBwd::kMid: return layer_t<C, LayerBwd::kMid>(a, st);
    default: return layer_t<C, LayerBwd::kLift>(a, st);
    }
}

template <int C>
cudaError_t mix_bwd_t(const FusedDims &d, int B, const bf16 *S, const bf16 *dY, const bf16 *R1, const bf16 *R2,
                      bf16 *dS, float *gRre, float *gRim, cudaStream_t st)
{
    static ResidentSlot slot;
    const size_t smem = mix_bwd_smem<C>();
    int ctas = 0;
    const cudaError_t e = resident_ctas(slot, mix_bwd_kernel<C>, 256, smem, &ctas);
    if (e != cudaSuccess) return e;
    const int tiles = (B + kMixRows - 1) / kMixRows;
    return launch_k(mix_bwd_kernel<C>, dim3((unsigned)(tiles + C / 16), (unsigned)d.M), 256, smem, st, true, d, B, S, dY,
                    R1, R2, dS, gRre, gRim);
}

}  // namespace

bool fused_train_ok(const FusedDims &d)
{
    return fused_ok(d) && d.P <= 128 && layer_smem(d.L, d.C, d.M, LayerBwd::kMid).total <= 227 * 1024;
}

cudaError_t launch_head_bwd(const HeadBwdArgs &a, cudaStream_t st)
{
    const bool two = a.d.out_ch <= 2;
    switch (a.d.C) {
    case 16: return two ? head_t<16, 2>(a, st) : head_t<16, 8>(a, st);
    case 32: return two ? head_t<32, 2>(a, st) : head_t<32, 8>(a, st);
    case 64: return two ? head_t<64, 2>(a, st) : head_t<64, 8>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_layer_bwd(const LayerBwdArgs &a, LayerBwd mode, cudaStream_t st)
{
    switch (a.d.C) {
    case 16: return layer_c<16>(a, mode, st);
    case 32: return layer_c<32>(a, mode, st);
    case 64: return layer_c<64>(a, mode, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_mix_bwd(const FusedDims &d, int B, const bf16 *S, const bf16 *dY, const bf16 *R1, const bf16 *R2,
                           bf16 *dS, float *gRre, float *gRim, cudaStream_t st)
{
    switch (d.C) {
    case 16: return mix_bwd_t<16>(d, B, S, dY, R1, R2, dS, gRre, gRim, st);
    case 32: return mix_bwd_t<32>(d, B, S, dY, R1, R2, dS, gRre, gRim, st);
    case 64: return mix_bwd_t<64>(d, B, S, dY, R1, R2, dS, gRre, gRim, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_refresh(const RefreshArgs &r, const AdamArgs *adam, cudaStream_t st)
{
    const unsigned blocks = (unsigned)((r.n + 255) / 256);
    if (adam) refresh_kernel<true><<<blocks, 256, 0, st>>>(r, *adam);
    else refresh_kernel<false><<<blocks, 256, 0, st>>>(r, AdamArgs{});
    return cudaGetLastError();
}

}  // namespace fno
}  // namespace hfs
