// One layer call of dp_per_example_wgrad, after its arguments have been checked: shared by the single-call entry point
// and by the batch of calls.
#pragma once
#include "wgrad_simple.cuh"

namespace dp {

bool valid_desc(const dp_layer_desc *d);
ConvGeom geom_of(const dp_layer_desc *d);
// Element type of X and dY in memory: DP_TF32 only changes the arithmetic of the tensor-core kernel.
inline int storage_type(const dp_layer_desc *d) { return d->dtype == DP_TF32 ? DP_F32 : d->dtype; }
inline bool has_bias_tensor(const dp_layer_desc *d) { return d->kind == DP_LAYER_NORM_AFFINE || d->has_bias != 0; }
inline int groups_of(const dp_layer_desc *d) { return (d->bias_separate && has_bias_tensor(d)) ? 2 : 1; }

// Implementation chosen for the layer and where its scratch lies: the header (status word, tickets) comes first.
struct WgradPlan {
    bool use_tc, use_thin;
    int slots, w_slots;
    size_t status_off, partial_off, factor_off, db_off, chunk_off, dg_off, tc_off, total;
};
void make_layer_plan(const dp_layer_desc *d, int epi, WgradPlan &pl);

// The buffers of one call, as dp_per_example_wgrad takes them.
struct LayerBuffers {
    const void *X, *dY;
    float *G_w, *G_b, *sqnorm;
    long long sqnorm_stride;
    float *acc_w, *acc_b, *clip_out;
};
dp_status check_layer(const dp_layer_desc *d, int epi, const LayerBuffers &io, float C_l);
// `header`: an initialised workspace header; `scratch`: where offset kWsHeaderBytes of the plan lies.
dp_status run_layer(const dp_layer_desc *d, int epi, const LayerBuffers &io, float C_l, const WgradPlan &pl, char *header,
                    char *scratch, cudaStream_t st);

}  // namespace dp
