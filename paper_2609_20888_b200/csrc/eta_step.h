// What eta_decode hands to the one-kernel step (eta_step.cu)
#pragma once

#include "eta_common.cuh"

namespace eta {

constexpr int STEP_MAX_BLOCKS = 512;     // of a row: their bounds and the list of survivors stay in shared memory
constexpr int STEP_MAX_TILES = 4096;     // of 64 (or 32) tokens, of all rows
constexpr int STEP_MAX_CLUSTER = MAX_CLUSTER;     // CTAs of a row

struct StepArgs {
    const __nv_bfloat16* q;
    const __half* musig;
    const float* mnorm;
    const int32_t* seq_lens;
    const float* tau;
    const float* head_const;
    float z, a, scale, beta;
    int lwb, rescue_window;
    uint32_t flags;
    int Hq, b_shift, t_cap, nb_cap;
    int shared;                          // set by launch_step: the bounds of a row are shared out over its CTAs
    const int32_t* block_table;          // paged cache (null: contiguous)
    int table_stride;
    FastDiv div_hkv;
    float* out;
    uint8_t* sel_mask;
    int32_t* stats;
    uint32_t* status;
};
// CTAs that a row gets in the one-kernel step; 0: the problem is not one for it, or the GPU does not hold such clusters
int step_cluster_rule(int rows, int nb_cap, int b, const int* fit);
int step_cluster(int rows, int nb_cap, int b, int D, int TS, int G, bool packed);
int launch_step(StepArgs a, const CUtensorMap& tmK, const CUtensorMap& tmV, int rows, int D, int TS, int G, int n_ranks, cudaStream_t s);

}  // namespace eta
