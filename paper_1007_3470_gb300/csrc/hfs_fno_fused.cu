// hfs_fno_fused.cu -- the surrogate's forward pass in 2 layers + 1 kernels.
//
// A sample's activations (L points x C channels, 32 KB in BF16 at 256 x 64)
// fit in shared memory, so one CTA takes a sample through everything between
// two mixing products, which are the only step that needs many samples at
// once (a C x 2C weight matrix of its own for every mode):
//   stage:  U = G Y (inverse truncated DFT), Z = H W + b + U, H' = GELU(Z),
//           then S' = F2 H' (truncated DFT of the next layer), or after the
//           last layer Q = GELU(H P1 + c1), O = Q P2 + c2;
//   mix:    Y_k = S_re,k R1_k + S_im,k R2_k, one mode and 64 samples a CTA.
// The GEMM-by-GEMM form wrote and re-read every intermediate (U, Z, an FP32
// and a BF16 copy of H, Q) in device memory, 39 launches.  Here a layer reads
// H and Y once and writes H' and S' once.  The products keep the GEMM kernels'
// operand roundings, mma.sync shape and order of accumulation, so results are
// bit-identical to theirs.
#include <algorithm>

#include "hfs_fno_frag.cuh"
#include "hfs_fno_fused.h"

namespace hfs {
namespace fno {

// Sizes: powers of two, so that tiles need no ragged edge and chunk positions
// are shifts and masks; C up to 64 (a warp's 16 x C accumulators stay in
// registers).  Everything else takes the GEMM-by-GEMM path.
static bool pow2(int v) { return v > 0 && (v & (v - 1)) == 0; }
static int modes_pad(int M) { return M < 16 ? 16 : M; }

struct StageSmem {
    int H, Y, G, W, F2, P1, P2, red, bias, total;  // byte offsets
};
static __host__ __device__ StageSmem stage_smem(int L, int C, int Mp, int P, bool mix, bool head)
{
    StageSmem s{};
    int o = 0;
    s.H = o;
    o += L * C * 2;
    s.Y = o;
    if (mix || !head) o += 2 * Mp * C * 2;  // also the staging of S
    if (mix) {
        s.G = o;
        o += L * 2 * Mp * 2;
        s.W = o;
        o += C * C * 2;
    }
    if (!head) {
        s.F2 = o;
        o += 2 * Mp * L * 2;
    } else {
        s.P1 = o;
        o += C * P * 2;
        s.P2 = o;
        o += P * 16;
        s.red = o;
        o += 128;
    }
    s.bias = o;
    o += C * 4;
    s.total = o;
    return s;
}

bool fused_ok(const FusedDims &d)
{
    if (d.C != 16 && d.C != 32 && d.C != 64) return false;
    if (!pow2(d.L) || d.L < 32 || d.L > 256) return false;
    if (!pow2(d.M) || d.M < 8 || d.M > 64 || 2 * d.M > d.L) return false;
    if (!pow2(d.P) || d.P < 16 || d.P > 256) return false;
    if (d.out_ch > 8 || d.in_ch > 8) return false;
    return stage_smem(d.L, d.C, modes_pad(d.M), d.P, true, false).total <= 227 * 1024 &&
           stage_smem(d.L, d.C, modes_pad(d.M), d.P, true, true).total <= 227 * 1024;
}

// Bound by issue and the tensor pipe together (52 % and 26 % busy).  Two CTAs of
// sixteen warps an SM, so that one's loads and barriers lie under the other's
// products.  Each warp owns rows of L for the pointwise part (H' overwrites H
// row by row), and 16 x 16 blocks of S.  4096 samples of 256 x 64, 32 modes:
// 170-190 us a launch; the 9 launches of a forward pass take 0.89 ms where the
// 39 of the GEMM-by-GEMM path took 3.52 ms (one sample: 75 us, 251 us).
template <int C, bool LIFT, bool MIX, bool HEAD>
__global__ void __launch_bounds__(512, 2) stage_kernel(const StageArgs a)
{
    constexpr int NT = C / 8, LGC = ilog2(C / 8);
    constexpr int HT = C >= 32 ? 4 : 2;  // n-tiles of H' at a time
    constexpr int SN = 2;                // n-tiles of a block of S
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const int L = a.d.L, M = a.d.M, Mp = M < 16 ? 16 : M, P = a.d.P;
    const int lgL = 31 - __clz(L >> 3), lgG = 31 - __clz(Mp >> 2), lgP = 31 - __clz(P >> 3);
    const StageSmem so = stage_smem(L, C, Mp, P, MIX, HEAD);
    bf16 *Hs = reinterpret_cast<bf16 *>(smem_raw + so.H), *Ys = reinterpret_cast<bf16 *>(smem_raw + so.Y);
    bf16 *Gs = reinterpret_cast<bf16 *>(smem_raw + so.G), *Ws = reinterpret_cast<bf16 *>(smem_raw + so.W);
    bf16 *Fs = reinterpret_cast<bf16 *>(smem_raw + so.F2);
    bf16 *P1s = reinterpret_cast<bf16 *>(smem_raw + so.P1), *P2s = reinterpret_cast<bf16 *>(smem_raw + so.P2);
    float(*s_red)[16] = reinterpret_cast<float(*)[16]>(smem_raw + so.red);
    float *bs = reinterpret_cast<float *>(smem_raw + so.bias);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x, nwarps = nthr >> 5;
    const int g = lane >> 2, t2 = (lane & 3) * 2;
    const bf16 zero = __float2bfloat16(0.0f);
    const uint32_t Ha = smem_u32(Hs), Ya = smem_u32(Ys), Ga = smem_u32(Gs), Wa = smem_u32(Ws), Fa = smem_u32(Fs),
                   Pa = smem_u32(P1s), P2a = smem_u32(P2s);
    const LaneAt lc = lane_at(lane, LGC), lg_ = lane_at(lane, lgG), ll = lane_at(lane, lgL), lp = lane_at(lane, lgP);

    // constants of the launch
    if constexpr (MIX) {
        const int lgm = 31 - __clz(M >> 3);
        for (int part = 0; part < 2; ++part) {
            const bf16 *src = part ? a.Gim : a.Gre;
            for (int u = tid; u < (L << lgm); u += nthr) {
                const int r = u >> lgm, c = u & ((1 << lgm) - 1);
                cp16(Gs + tile_at(r, part * (Mp >> 3) + c, lgG), src + (int64_t)r * M + c * 8, true);
            }
        }
        if (M < Mp) {  // pad columns of G and pad rows of Y
            for (int u = tid; u < 2 * L; u += nthr)
                *reinterpret_cast<uint4 *>(Gs + tile_at(u >> 1, (u & 1) * (Mp >> 3) + 1, lgG)) = make_uint4(0, 0, 0, 0);
            for (int u = tid; u < 16 * NT; u += nthr) {
                const int r = u / NT;
                *reinterpret_cast<uint4 *>(Ys + tile_at((r >> 3) * Mp + 8 + (r & 7), u % NT, LGC)) =
                    make_uint4(0, 0, 0, 0);
            }
        }
        tile_load(Ws, LGC, 0, C, LGC, a.W, C, tid, nthr);
    }
    if constexpr (!HEAD) tile_load(Fs, lgL, 0, 2 * M, lgL, a.F2, L, tid, nthr);
    if constexpr (HEAD) {
        tile_load(P1s, lgP, 0, C, lgP, a.P1b, P, tid, nthr);
        for (int u = tid; u < P * 8; u += nthr)
            P2s[u] = (u & 7) < a.d.out_ch ? a.P2b[(u >> 3) * a.d.out_ch + (u & 7)] : zero;
    }
    unsigned pin[LIFT ? NT : 1];
    if constexpr (LIFT) {
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            __nv_bfloat162 v;
            v.x = a.Pinb[t2 * C + 8 * j + g];
            v.y = a.Pinb[(t2 + 1) * C + 8 * j + g];
            pin[j] = *reinterpret_cast<const unsigned *>(&v);
        }
    }
    if (tid < C) bs[tid] = MIX ? a.bias[tid] : a.bin[tid];
    pdl_wait();
    pdl_trigger();

    for (int b = blockIdx.x; b < a.B; b += gridDim.x) {
        // H of the sample, each warp its own rows
        for (int m0 = warp * 16; m0 < L; m0 += nwarps * 16) {
            if constexpr (LIFT) {
                const float *x0 = a.x + ((int64_t)b * L + m0 + g) * a.d.in_ch, *x8 = x0 + 8 * a.d.in_ch;
                const bool v0 = t2 < a.d.in_ch, v1 = t2 + 1 < a.d.in_ch;
                const unsigned af[4] = {pack2(v0 ? x0[t2] : 0.0f, v1 ? x0[t2 + 1] : 0.0f),
                                        pack2(v0 ? x8[t2] : 0.0f, v1 ? x8[t2 + 1] : 0.0f), 0u, 0u};
                unsigned hp[NT][2];
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const unsigned bf[2] = {pin[j], 0u};
                    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    mma_bf16(acc, af, bf);
                    const float2 bb = __ldg(reinterpret_cast<const float2 *>(a.bin + 8 * j + t2));
                    hp[j][0] = pack2(acc[0] + bb.x, acc[1] + bb.y);
                    hp[j][1] = pack2(acc[2] + bb.x, acc[3] + bb.y);
                }
                packed_to_tile(Ha, LGC, m0, 0, hp, lane);
            } else {
                tile_load(Hs, LGC, m0, 16, LGC, a.Hin + ((int64_t)b * L + m0) * C, C, lane, 32);
            }
        }
        if constexpr (MIX) {
            for (int u = tid; u < ((2 * M) << LGC); u += nthr) {
                const int r = u >> LGC, c = u & (NT - 1), part = r >= M, k = r - part * M;
                cp16(Ys + tile_at(part * Mp + k, c, LGC), a.Y + ((int64_t)k * a.d.Bm + b) * 2 * C + part * C + c * 8,
                     true);
            }
        }
        cp_wait_all();
        __syncthreads();
        float num = 0.0f, den = 0.0f;
        for (int m0 = warp * 16; m0 < L; m0 += nwarps * 16) {
            const int64_t row = (int64_t)b * L + m0 + g;
            if constexpr (MIX) {
                // HT n-tiles at a time (64 registers: 32 warps an SM); H' stays
                // packed in registers until the warp's rows of H are read
                unsigned hp[NT][2];
#pragma unroll
                for (int h = 0; h < NT / HT; ++h) {
                    float u[HT][4], z[HT][4];
                    zero_acc(u);
                    zero_acc(z);
#pragma unroll 2
                    for (int k0 = 0; k0 < Mp; k0 += 16) {
                        unsigned a0[4], a1[4];
                        frag_a(a0, Ga, lg_, lgG, m0, k0);
                        frag_a(a1, Ga, lg_, lgG, m0, Mp + k0);
#pragma unroll
                        for (int j = 0; j < HT; j += 2) {
                            unsigned bf[4];
                            frag_b(bf, Ya, lc, LGC, k0, 8 * (h * HT + j));
                            mma16(u[j], u[j + 1], a0, bf);
                            frag_b(bf, Ya, lc, LGC, Mp + k0, 8 * (h * HT + j));
                            mma16(z[j], z[j + 1], a1, bf);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < HT; ++j)
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            u[j][q] = z[j][q] + u[j][q];
                            z[j][q] = 0.0f;
                        }
#pragma unroll
                    for (int k0 = 0; k0 < C; k0 += 16) {
                        unsigned af[4];
                        frag_a(af, Ha, lc, LGC, m0, k0);
#pragma unroll
                        for (int j = 0; j < HT; j += 2) {
                            unsigned bf[4];
                            frag_b(bf, Wa, lc, LGC, k0, 8 * (h * HT + j));
                            mma16(z[j], z[j + 1], af, bf);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < HT; ++j) {
                        const int n = 8 * (h * HT + j) + t2;
                        const float2 bb = *reinterpret_cast<const float2 *>(bs + n);
                        z[j][0] = (z[j][0] + bb.x) + u[j][0];
                        z[j][1] = (z[j][1] + bb.y) + u[j][1];
                        z[j][2] = (z[j][2] + bb.x) + u[j][2];
                        z[j][3] = (z[j][3] + bb.y) + u[j][3];
                        if (a.pre) {
                            *reinterpret_cast<float2 *>(a.pre + row * C + n) = make_float2(z[j][0], z[j][1]);
                            *reinterpret_cast<float2 *>(a.pre + (row + 8) * C + n) = make_float2(z[j][2], z[j][3]);
                        }
                        const uint2 v = HEAD ? make_uint2(pack2(z[j][0], z[j][1]), pack2(z[j][2], z[j][3]))
                                             : gelu4(z[j][0], z[j][1], z[j][2], z[j][3]);
                        hp[h * HT + j][0] = v.x;
                        hp[h * HT + j][1] = v.y;
                    }
                }
                __syncwarp();  // every lane has read the warp's rows of H
                packed_to_tile(Ha, LGC, m0, 0, hp, lane);
            }
            __syncwarp();
            if (a.Hout) {
                for (int u = lane; u < (16 << LGC); u += 32)
                    *reinterpret_cast<uint4 *>(a.Hout + ((int64_t)b * L + m0 + (u >> LGC)) * C + (u & (NT - 1)) * 8) =
                        *reinterpret_cast<const uint4 *>(Hs + tile_at(m0 + (u >> LGC), u & (NT - 1), LGC));
            }
            if constexpr (HEAD) {
                unsigned hf[C / 16][4];
#pragma unroll
                for (int k = 0; k < C / 16; ++k) frag_a(hf[k], Ha, lc, LGC, m0, 16 * k);
                float o[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                for (int p0 = 0; p0 < P; p0 += 16) {
                    float q0[4] = {0.0f, 0.0f, 0.0f, 0.0f}, q1[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                    for (int k = 0; k < C / 16; ++k) {
                        unsigned bf[4];
                        frag_b(bf, Pa, lp, lgP, 16 * k, p0);
                        mma16(q0, q1, hf[k], bf);
                    }
                    const float2 ca = *reinterpret_cast<const float2 *>(a.c1 + p0 + t2);
                    const float2 cb = *reinterpret_cast<const float2 *>(a.c1 + p0 + 8 + t2);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        q0[q] += (q & 1) ? ca.y : ca.x;
                        q1[q] += (q & 1) ? cb.y : cb.x;
                    }
                    if (a.Qpre) {
                        float *w = a.Qpre + row * P + p0 + t2;
                        *reinterpret_cast<float2 *>(w) = make_float2(q0[0], q0[1]);
                        *reinterpret_cast<float2 *>(w + 8) = make_float2(q1[0], q1[1]);
                        *reinterpret_cast<float2 *>(w + 8 * P) = make_float2(q0[2], q0[3]);
                        *reinterpret_cast<float2 *>(w + 8 * P + 8) = make_float2(q1[2], q1[3]);
                    }
                    const uint2 g0 = gelu4(q0[0], q0[1], q0[2], q0[3]), g1 = gelu4(q1[0], q1[1], q1[2], q1[3]);
                    const unsigned af[4] = {g0.x, g0.y, g1.x, g1.y};
                    unsigned bf[2];
                    lds_frag2_t(bf, P2a + (p0 + (lane & 15)) * 16);
                    mma_bf16(o, af, bf);
                }
                const int oc = a.d.out_ch;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int n = t2 + (q & 1);
                    if (n >= oc) continue;
                    const int64_t at = (row + (q >> 1) * 8) * oc + n;
                    const float v = o[q] + a.c2[n];
                    a.O[at] = v;
                    if (a.y) {
                        const float y = a.y[at], d = v - y;
                        num += d * d;
                        den += y * y;
                    }
                }
            }
        }
        if constexpr (HEAD) {
            if (a.y) {
#pragma unroll
                for (int s = 16; s > 0; s >>= 1) {
                    num += __shfl_xor_sync(0xffffffffu, num, s);
                    den += __shfl_xor_sync(0xffffffffu, den, s);
                }
                if (lane == 0) {
                    s_red[0][warp] = num;
                    s_red[1][warp] = den;
                }
            }
        }
        __syncthreads();
        if constexpr (HEAD) {
            if (a.y && tid < 2) {
                float v = 0.0f;
                for (int w = 0; w < nwarps; ++w) v += s_red[tid][w];
                a.sums[2 * b + tid] = v;
            }
        } else {
            // S = F2 H', blocks of 16 modes x 8 SN channels
            constexpr int NG = C / (8 * SN);
            for (int u = warp; u < (M >> 3) * NG; u += nwarps) {
                const int m0 = (u / NG) * 16, n0 = (u % NG) * 8 * SN;
                float s[SN][4];
                zero_acc(s);
#pragma unroll 4
                for (int k0 = 0; k0 < L; k0 += 16) {
                    unsigned af[4];
                    frag_a(af, Fa, ll, lgL, m0, k0);
#pragma unroll
                    for (int j = 0; j < SN; j += 2) {
                        unsigned bf[4];
                        frag_b(bf, Ha, lc, LGC, k0, n0 + 8 * j);
                        mma16(s[j], s[j + 1], af, bf);
                    }
                }
                acc_to_tile(Ya, LGC, m0, n0, s, lane);
                __syncwarp();
                for (int i = lane; i < 16 * SN; i += 32) {
                    const int r = m0 + i / SN, c = (n0 >> 3) + i % SN;
                    *reinterpret_cast<uint4 *>(a.S + ((int64_t)r * a.d.Bm + b) * C + c * 8) =
                        *reinterpret_cast<const uint4 *>(Ys + tile_at(r, c, LGC));
                }
            }
            if constexpr (MIX) {
                if (M < Mp) {  // the staging of S ran over the pad rows of Y
                    __syncthreads();
                    for (int u = tid; u < 16 * NT; u += nthr) {
                        const int r = u / NT;
                        *reinterpret_cast<uint4 *>(Ys + tile_at((r >> 3) * Mp + 8 + (r & 7), u % NT, LGC)) =
                            make_uint4(0, 0, 0, 0);
                    }
                }
            }
            __syncthreads();
        }
    }
}

// Bound by memory: per mode and 64 samples 16 KB of S in and 16 KB of Y out.
// A warp keeps the weights of its 16 columns of Y in registers (32 of them at
// C = 64) for the whole launch and takes tiles of 64 samples in turn, the next
// tile's copies under the products of the current one; with the weights read
// from shared memory for each 16 rows, shared-memory bandwidth was the bound
// (21.5 us a launch at 4096 samples x 32 modes, 23.5 us before).
constexpr int MIX_ROWS = 64;
template <int C>
__global__ void __launch_bounds__(256, 2) mix_kernel(const FusedDims d, int B, const bf16 *__restrict__ S,
                                                     const bf16 *__restrict__ R1, const bf16 *__restrict__ R2,
                                                     bf16 *__restrict__ Y)
{
    constexpr int LGC = ilog2(C / 8), LG2 = LGC + 1, KS = C / 16;
    constexpr int CS = 2 * C / 16, RG = 8 / CS;  // column slices, row groups of warps
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    bf16 *As = reinterpret_cast<bf16 *>(smem_raw);  // two of [2][64][C], each then Y as [64][2C]
    bf16 *Rs = As + 4 * MIX_ROWS * C;               // [2][C][2C]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, k = blockIdx.y;
    const int tiles = (B + MIX_ROWS - 1) / MIX_ROWS;
    const uint32_t Ra = smem_u32(Rs);
    const LaneAt lc = lane_at(lane, LGC), l2 = lane_at(lane, LG2);
    const int n0 = (warp % CS) * 16, rg = warp / CS;
    tile_load(Rs, LG2, 0, C, LG2, R1 + (int64_t)k * C * 2 * C, 2 * C, tid, 256);
    tile_load(Rs, LG2, C, C, LG2, R2 + (int64_t)k * C * 2 * C, 2 * C, tid, 256);
    cp_wait_all();
    __syncthreads();
    unsigned w[2][KS][4];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) frag_b(w[p][ks], Ra, l2, LG2, p * C + 16 * ks, n0);
    pdl_wait();
    pdl_trigger();
    auto load = [&](int tile, int buf) {
        if (tile < tiles) {
            const int b0 = tile * MIX_ROWS;
#pragma unroll
            for (int part = 0; part < 2; ++part)
                tile_load(As + buf * 2 * MIX_ROWS * C, LGC, part * MIX_ROWS, MIX_ROWS, LGC,
                          S + ((int64_t)(part * d.M + k) * d.Bm + b0) * C, C, tid, 256, B - b0);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    load(blockIdx.x, 0);
    int buf = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, buf ^= 1) {
        load(tile + gridDim.x, buf ^ 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        bf16 *At = As + buf * 2 * MIX_ROWS * C;
        const uint32_t Aa = smem_u32(At);
        float y[4 / RG][2][4];
#pragma unroll
        for (int i = 0; i < 4 / RG; ++i) {
            const int m0 = (i * RG + rg) * 16;
            float y1[2][4];
            zero_acc(y[i]);
            zero_acc(y1);
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                unsigned a0[4], a1[4];
                frag_a(a0, Aa, lc, LGC, m0, 16 * ks);
                frag_a(a1, Aa, lc, LGC, MIX_ROWS + m0, 16 * ks);
                mma16(y[i][0], y[i][1], a0, w[0][ks]);
                mma16(y1[0], y1[1], a1, w[1][ks]);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) y[i][j][q] = y1[j][q] + y[i][j][q];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4 / RG; ++i) acc_to_tile(Aa, LG2, (i * RG + rg) * 16, n0, y[i], lane);
        __syncthreads();
        const int b0 = tile * MIX_ROWS;
        for (int i = tid; i < (MIX_ROWS << LG2); i += 256) {
            const int r = i >> LG2, c = i & ((1 << LG2) - 1);
            if (b0 + r < B)
                *reinterpret_cast<uint4 *>(Y + ((int64_t)k * d.Bm + b0 + r) * 2 * C + c * 8) =
                    *reinterpret_cast<const uint4 *>(At + tile_at(r, c, LG2));
        }
        __syncthreads();  // the tile after next is copied into this buffer
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
template <int C, bool LIFT, bool MIX, bool HEAD>
static cudaError_t stage_t(const StageArgs &a, bool pdl, cudaStream_t st)
{
    static ResidentSlot slot;
    const int threads = 32 * std::min(16, a.d.L / 16);
    const size_t smem = (size_t)stage_smem(a.d.L, C, modes_pad(a.d.M), a.d.P, MIX, HEAD).total;
    int ctas = 0;
    const cudaError_t e = resident_ctas(slot, stage_kernel<C, LIFT, MIX, HEAD>, threads, smem, &ctas);
    if (e != cudaSuccess) return e;
    return launch_k(stage_kernel<C, LIFT, MIX, HEAD>, dim3((unsigned)std::min(a.B, ctas)), threads, smem, st, pdl, a);
}

template <int C>
static cudaError_t stage_c(const StageArgs &a, bool lift, bool mix, bool head, bool pdl, cudaStream_t st)
{
    if (!mix) return stage_t<C, true, false, false>(a, pdl, st);
    if (lift) return head ? stage_t<C, true, true, true>(a, pdl, st) : stage_t<C, true, true, false>(a, pdl, st);
    return head ? stage_t<C, false, true, true>(a, pdl, st) : stage_t<C, false, true, false>(a, pdl, st);
}

cudaError_t launch_stage(const StageArgs &a, bool lift, bool mix, bool head, bool pdl, cudaStream_t st)
{
    switch (a.d.C) {
    case 16: return stage_c<16>(a, lift, mix, head, pdl, st);
    case 32: return stage_c<32>(a, lift, mix, head, pdl, st);
    case 64: return stage_c<64>(a, lift, mix, head, pdl, st);
    default: return cudaErrorInvalidValue;
    }
}

template <int C>
static cudaError_t mix_t(const FusedDims &d, int B, const bf16 *S, const bf16 *R1, const bf16 *R2, bf16 *Y,
                         cudaStream_t st)
{
    static ResidentSlot slot;
    const size_t smem = (size_t)(4 * MIX_ROWS * C + 4 * C * C) * sizeof(bf16);
    int ctas = 0;
    const cudaError_t e = resident_ctas(slot, mix_kernel<C>, 256, smem, &ctas);
    if (e != cudaSuccess) return e;
    const int tiles = (B + MIX_ROWS - 1) / MIX_ROWS;
    return launch_k(mix_kernel<C>, dim3((unsigned)std::min(tiles, std::max(1, ctas / d.M)), (unsigned)d.M), 256, smem, st,
                    true, d, B, S, R1, R2, Y);
}

cudaError_t launch_mix(const FusedDims &d, int B, const bf16 *S, const bf16 *R1, const bf16 *R2, bf16 *Y,
                       cudaStream_t st)
{
    switch (d.C) {
    case 16: return mix_t<16>(d, B, S, R1, R2, Y, st);
    case 32: return mix_t<32>(d, B, S, R1, R2, Y, st);
    case 64: return mix_t<64>(d, B, S, R1, R2, Y, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fno
}  // namespace hfs
