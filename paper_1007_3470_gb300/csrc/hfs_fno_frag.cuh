// hfs_fno_frag.cuh -- the warp-level primitives of the surrogate's kernels, and
// the shared-memory tiles and tensor-core fragments of the fused ones
// (hfs_fno_fused.cu).
//
// Tiles are rows of BF16 in 16-byte chunks, 2^LG chunks a row, stored without
// padding: chunk c of row r sits at c ^ s(r), where s runs through the chunk
// positions of a 128-byte line as r does, so that the eight rows of a matrix
// that ldmatrix reads, or an accumulator's eight rows, lie in distinct banks.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "hfs_resident.h"

namespace hfs {
namespace fno {

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z)
{
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

__device__ __forceinline__ void ldsm_x4(unsigned (&r)[4], const bf16 *p)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}
__device__ __forceinline__ void ldsm_x2(unsigned (&r)[2], const bf16 *p)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], const unsigned (&b)[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void ldsm_x4_t(unsigned (&r)[4], const bf16 *p)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}
__device__ __forceinline__ void ldsm_x2_t(unsigned (&r)[2], const bf16 *p)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}
// 16-byte asynchronous copy; an invalid chunk is zero-filled (source size 0)
__device__ __forceinline__ void cp16(bf16 *dst, const bf16 *src, bool valid)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}


// element offset of chunk `chunk` of row `row`
__device__ __forceinline__ int tile_at(int row, int chunk, int lg)
{
    const int s = lg >= 3 ? (row & 7) : ((row >> (3 - lg)) & ((1 << lg) - 1));
    return ((row << lg) + (chunk ^ s)) * 8;
}

// Shared-memory addresses of the fragments.  Fragments start at rows and
// columns that are multiples of 16, so the lane's share of an address, its row
// and its position in the row, does not change from one to the next: chunk
// c0 | b of row r0 + r is at (tile + r0 rows + lane part) ^ 16 c0, one
// operation or an immediate offset where the general form takes eight.  Tiles
// start at multiples of their row's bytes.
struct LaneAt {
    uint32_t n, t;  // lane parts: rows lane & 15 (n), rows in the order of a transposed operand (t)
};
__device__ __forceinline__ LaneAt lane_at(int lane, int lg)
{
    const int rt = (lane & 7) + ((lane >> 4) & 1) * 8;
    return {(uint32_t)tile_at(lane & 15, lane >> 4, lg) * 2u, (uint32_t)tile_at(rt, (lane >> 3) & 1, lg) * 2u};
}
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void lds_frag(unsigned (&r)[4], uint32_t a)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void lds_frag_t(unsigned (&r)[4], uint32_t a)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void lds_frag2_t(unsigned (&r)[2], uint32_t a)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(a)
                 : "memory");
}
// A fragment (16 x 16 at row m0, column k0): stored [m][k], or [k][m] (trans)
__device__ __forceinline__ void frag_a(unsigned (&r)[4], uint32_t t, LaneAt l, int lg, int m0, int k0)
{
    lds_frag(r, (t + l.n + ((uint32_t)m0 << (lg + 4))) ^ (uint32_t)(k0 * 2));
}
__device__ __forceinline__ void frag_a_t(unsigned (&r)[4], uint32_t t, LaneAt l, int lg, int m0, int k0)
{
    lds_frag_t(r, ((t + l.t) ^ (uint32_t)(m0 * 2)) + ((uint32_t)k0 << (lg + 4)));
}
// B fragments of columns n0..n0+7 (r[0], r[1]) and n0+8..n0+15 (r[2], r[3]),
// rows k0..k0+15: stored [k][n], or [n][k] (the transposed product)
__device__ __forceinline__ void frag_b(unsigned (&r)[4], uint32_t t, LaneAt l, int lg, int k0, int n0)
{
    lds_frag_t(r, ((t + l.n) ^ (uint32_t)(n0 * 2)) + ((uint32_t)k0 << (lg + 4)));
}
__device__ __forceinline__ void frag_b_nk(unsigned (&r)[4], uint32_t t, LaneAt l, int lg, int k0, int n0)
{
    lds_frag(r, (t + l.t + ((uint32_t)n0 << (lg + 4))) ^ (uint32_t)(k0 * 2));
}
// one A fragment against 16 columns
__device__ __forceinline__ void mma16(float (&c0)[4], float (&c1)[4], const unsigned (&a)[4], const unsigned (&b)[4])
{
    const unsigned b0[2] = {b[0], b[1]}, b1[2] = {b[2], b[3]};
    mma_bf16(c0, a, b0);
    mma_bf16(c1, a, b1);
}

template <int NT> __device__ __forceinline__ void zero_acc(float (&c)[NT][4])
{
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) c[j][q] = 0.0f;
}

__device__ __forceinline__ unsigned pack2(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned *>(&v);
}

// GELU rounded to BF16, four values at a time: bf16(gelu_f(z)) bit for bit at
// less than half of erff's instructions.  1 - Phi comes from the rational
// approximation of Abramowitz and Stegun 7.1.26 (error of erf below 1.5e-7),
// so the value v differs from gelu_f(z), whose own error is below 1.5e-7 |z|,
// by less than d = 6e-7 |z|.  Where v - d and v + d round to the same BF16
// number, so does gelu_f(z); in the other cases (1 in 1000 values to 7000,
// and every z below -5) the accurate function decides.  Over all 2^32 values of z
// the result is equal but for z = -0, where this gives +0 (test_gelu_over_all_inputs).
// The time depends on the values: a group with one below -5 takes both paths; 4096
// samples whose every pre-activation is near -8 take 1.18 ms, 0.89 with the usual ones
// (3.52 ms GEMM by GEMM, either way).
static __device__ __noinline__ uint2 gelu4_accurate(float a, float b, float c, float d)
{
    return make_uint2(pack2(gelu_f(a), gelu_f(b)), pack2(gelu_f(c), gelu_f(d)));
}
__device__ __forceinline__ unsigned gelu2_bounds(float z0, float z1, unsigned &other)
{
    const float2 az = make_float2(fminf(fabsf(z0), 16.0f), fminf(fabsf(z1), 16.0f));
    const auto bc = [](float c) { return make_float2(c, c); };
    const float2 den = __ffma2_rn(az, bc(0.3275911f * 0.70710678f), bc(1.0f));
    float2 t, e;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t.x) : "f"(den.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t.y) : "f"(den.y));
    const float2 zz = __fmul2_rn(az, __fmul2_rn(az, bc(-0.5f * 1.44269504f)));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(zz.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(zz.y));
    float2 p = __ffma2_rn(t, bc(0.5f * 1.061405429f), bc(0.5f * -1.453152027f));
    p = __ffma2_rn(t, p, bc(0.5f * 1.421413741f));
    p = __ffma2_rn(t, p, bc(0.5f * -0.284496736f));
    p = __ffma2_rn(t, p, bc(0.5f * 0.254829592f));
    p = __fmul2_rn(__fmul2_rn(t, p), e);  // 1 - Phi(|z|)
    const float2 na = make_float2(-az.x, -az.y);
    const float2 v = __ffma2_rn(na, p, make_float2(fmaxf(z0, 0.0f), fmaxf(z1, 0.0f)));
    const float2 lo = __ffma2_rn(az, bc(-6e-7f), v), hi = __ffma2_rn(az, bc(6e-7f), v);
    other = pack2(hi.x, hi.y);
    return pack2(lo.x, lo.y);
}
__device__ __forceinline__ uint2 gelu4(float a, float b, float c, float d)
{
    unsigned h0, h1;
    uint2 r = make_uint2(gelu2_bounds(a, b, h0), gelu2_bounds(c, d, h1));
    if (r.x != h0 || r.y != h1) r = gelu4_accurate(a, b, c, d);
    return r;
}

// accumulator rows g, g + 8 of 8 NT columns at (m0, n0) into a tile
template <int NT>
__device__ __forceinline__ void packed_to_tile(uint32_t t, int lg, int m0, int n0, const unsigned (&c)[NT][2], int lane)
{
    const uint32_t w = t + (uint32_t)tile_at(lane >> 2, 0, lg) * 2u + (lane & 3) * 4u + ((uint32_t)m0 << (lg + 4));
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const uint32_t at = w ^ (uint32_t)(n0 * 2 + 16 * j);
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(at), "r"(c[j][0]) : "memory");
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(at + (8u << (lg + 4))), "r"(c[j][1]) : "memory");
    }
}
template <int NT>
__device__ __forceinline__ void acc_to_tile(uint32_t t, int lg, int m0, int n0, const float (&c)[NT][4], int lane)
{
    unsigned v[NT][2];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        v[j][0] = pack2(c[j][0], c[j][1]);
        v[j][1] = pack2(c[j][2], c[j][3]);
    }
    packed_to_tile(t, lg, m0, n0, v, lane);
}

// rows [r0, r0 + rows) x chunks [c0, c0 + nc) of a tile from / to global rows
// of `ld` elements, by `n` threads of index i (asynchronous copies on the way in)
__device__ __forceinline__ void tile_load(bf16 *t, int lg, int r0, int rows, int lgc, const bf16 *g, int64_t ld, int i,
                                          int n, int valid = 1 << 30)
{
    for (int u = i; u < (rows << lgc); u += n) {
        const int r = u >> lgc, c = u & ((1 << lgc) - 1);
        const bool ok = r < valid;
        cp16(t + tile_at(r0 + r, c, lg), ok ? g + (int64_t)r * ld + c * 8 : g, ok);
    }
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// programmatic dependent launch: nothing before pdl_wait() reads what the
// kernel before wrote; the kernel after may read, before its own wait, only
// what was written before this kernel's predecessor ended
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P>
inline cudaError_t launch_k(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, bool pdl, P... a)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, a...);
}

// CTAs of a persistent grid: as many as fit (remembered, see ResidentSlot).  Every
// kernel is allowed the most shared memory that a CTA may have (none has static
// arrays), whatever its launch takes, so that models of different sizes do not undo
// each other's setting.
constexpr int kMaxSmem = 227 * 1024;
template <typename K>
inline cudaError_t resident_ctas(ResidentSlot &slot, K kernel, int threads, size_t smem, int *ctas)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return (cudaError_t)slot.get(dev, threads, smem, [&](int *n) -> int {
        int sms = 0, per = 0;
        cudaError_t q = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (q == cudaSuccess) q = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (q == cudaSuccess) q = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem);
        if (q == cudaSuccess && per < 1) q = cudaErrorInvalidConfiguration;
        *n = sms * per;
        return (int)q;
    }, ctas);
}

__host__ __device__ constexpr int ilog2(int v) { return v <= 1 ? 0 : 1 + ilog2(v >> 1); }

}  // namespace fno
}  // namespace hfs
