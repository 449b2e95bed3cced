// Internal interface of the batch of layer calls (batch.cu): groups of layers that go through one launch together.
#pragma once
#include "layer.cuh"

namespace dp {

constexpr int kGroupLayers = 64;      // layers per grouped launch (their table travels as a kernel parameter)

// ---- normalisation-affine layers (affine_batch.cu)
struct AffineSeg {
    const void *X, *dY;
    float *dgamma, *dbeta;            // [B][C]: the caller's G_w / G_b, or scratch
    float *factor;                    // [B][2] scratch (fused clip)
    float *sqnorm, *clip_out, *acc_w, *acc_b;
    long long sq_stride;
    long long part_off;               // first float of the layer's pixel-chunk partials [B][chunks][2][C]
    int B, HW, C;
    int tcv, pix, chunks;             // channel vectors and pixels per block, pixel chunks per example
    int clip, separate;
};
struct AffineGroup {
    int n;
    float C_l;
    float *partial;
    int start1[kGroupLayers], start2[kGroupLayers], start3[kGroupLayers];   // first block of every layer in the three launches
    AffineSeg seg[kGroupLayers];
};
bool affine_batch_eligible(int dtype, int C);
// beside: shaped for the form that runs beside tensor-core launches (any form takes it)
void affine_batch_shape(int dtype, int B, int HW, int C, bool beside, AffineSeg &s);
// tickets: two cleared words for the form that runs beside tensor-core launches, which are in later launches; null: the GPU is free
// begun (with tickets): recorded when every block of that form runs
dp_status launch_affine_batch(int dtype, AffineGroup &grp, int *tickets, cudaEvent_t begun, cudaStream_t st);

}  // namespace dp
