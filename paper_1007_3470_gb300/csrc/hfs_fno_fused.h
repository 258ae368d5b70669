// hfs_fno_fused.h -- launchers of the surrogate's fused forward kernels
// (hfs_fno_fused.cu) and backward kernels (hfs_fno_fused_bwd.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace hfs {
namespace fno {

typedef __nv_bfloat16 bf16;

// the sizes that the fused kernels are built for (fused_ok)
struct FusedDims {
    int L, C, M, P, in_ch, out_ch, layers;
    int Bm;  // samples that the buffers are laid out for
};

bool fused_ok(const FusedDims &d);

// One pass over the samples (see stage_kernel).  Null outputs are not written.
struct StageArgs {
    FusedDims d;
    int B;
    const float *x;      // [B][L][in_ch]
    const bf16 *Pinb;    // [8][C], rows in_ch..7 zero
    const float *bin;
    const bf16 *Hin;     // [B][L][C]
    const bf16 *Y;       // [M][Bm][2C]
    const bf16 *W;       // [C][C]
    const float *bias;
    float *pre;          // [B][L][C]
    bf16 *Hout;          // [B][L][C]
    const bf16 *F2;      // [2M][L]
    const bf16 *Gre, *Gim;  // [L][M]
    bf16 *S;             // [2M][Bm][C]
    const bf16 *P1b;     // [C][P]
    const float *c1;
    const bf16 *P2b;     // [P][out_ch]
    const float *c2;
    float *Qpre;         // [B][L][P]
    float *O;            // [B][L][out_ch]
    const float *y;      // targets: with them the sums of the loss
    float *sums;         // [B][2]
};

// lift: H from x; mix: the spectral layer; head: the projection (else S)
cudaError_t launch_stage(const StageArgs &a, bool lift, bool mix, bool head, bool pdl, cudaStream_t st);

// Y_k = S_re,k R1_k + S_im,k R2_k of every mode
cudaError_t launch_mix(const FusedDims &d, int B, const bf16 *S, const bf16 *R1, const bf16 *R2, bf16 *Y,
                       cudaStream_t st);

// ---- backward ----
bool fused_train_ok(const FusedDims &d);

// The projection and the loss's gradient; dZ of the last layer (BF16) and the
// gradients of P1, c1, P2, c2 and of the last layer's bias.
struct HeadBwdArgs {
    FusedDims d;
    int B;
    const float *O, *y, *sums;  // outputs, targets, per-sample sums of the loss
    const float *Qpre;          // [B][L][P]
    const bf16 *H;              // [B][L][C], the last layer's output
    const bf16 *P1b, *P2b;
    bf16 *dZ;                   // [B][L][C]
    float *gP1, *gc1, *gP2, *gc2, *gb;
};
cudaError_t launch_head_bwd(const HeadBwdArgs &a, cudaStream_t st);

// One layer: dZ (given for the last layer, otherwise from the layer above:
// dZ_up W_up^T + F2^T dS_up times GELU'), dY = G^T dZ, the gradients of W and b;
// lift: the gradients of P_in and b_in instead.
struct LayerBwdArgs {
    FusedDims d;
    int B;
    bf16 *dZ;                   // [B][L][C]: the layer above's on entry, this layer's on return
    const bf16 *Wup;            // [C][C]
    const bf16 *dSup;           // [2M][Bm][C]
    const bf16 *F2, *Gre, *Gim;
    const float *pre;           // [B][L][C]
    const bf16 *Hin;            // [B][L][C]
    bf16 *dY;                   // [M][Bm][2C]
    const float *x;             // lift: [B][L][in_ch]
    float *gW, *gb;             // lift: P_in, b_in
};
enum class LayerBwd { kTop, kMid, kLift };
cudaError_t launch_layer_bwd(const LayerBwdArgs &a, LayerBwd mode, cudaStream_t st);

// dS_re,k = dY_k R1_k^T, dS_im,k = dY_k R2_k^T and the gradients of R_re, R_im
cudaError_t launch_mix_bwd(const FusedDims &d, int B, const bf16 *S, const bf16 *dY, const bf16 *R1, const bf16 *R2,
                           bf16 *dS, float *gRre, float *gRim, cudaStream_t st);

// One Adam step on every parameter (adam null: none) and the BF16 copies of
// the weights
struct AdamArgs {
    const float *g;
    float *m, *v;
    float lr, b1, b2, eps, c1, c2;
};
struct RefreshArgs {
    int64_t n, bin, layer0, layer_stride, P1, c1, P2, c2;  // offsets in the parameter vector
    int in_ch, C, M, P, out_ch;
    float *p;
    bf16 *Pinb, *Wb, *R1, *R2, *P1b, *P2b;
};
cudaError_t launch_refresh(const RefreshArgs &r, const AdamArgs *adam, cudaStream_t st);

}  // namespace fno
}  // namespace hfs
