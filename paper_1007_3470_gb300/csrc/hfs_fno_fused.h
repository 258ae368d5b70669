// hfs_fno_fused.h -- launchers of the surrogate's fused forward kernels
// (hfs_fno_fused.cu).
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

}  // namespace fno
}  // namespace hfs
