// wq4_stage_host.h -- internal interface between the chain planner and the
// batched decode stages (wq4_stage.cu).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "wq4.h"

namespace wq4 {

enum StStageType { kStQKV = 0, kStO = 1, kStGU = 2, kStDOWN = 3, kStLM = 4 };

// Workspace buffers of the batched path (device pointers).
struct StageBuffers {
    const uint16_t* x_stage;   // [B][H] token input
    uint16_t* pV;              // [L+1][B][H]
    uint16_t* pQKV;            // [L][B][Nqkv]
    uint16_t* pO;              // [L][B][H]
    uint16_t* pX1;             // [L][B][H]
    uint16_t* pGU;             // [L][B][2F]
    uint16_t* pM;              // [L][B][F]
    uint16_t* pD;              // [L][B][H]
    uint16_t* pX2;             // [L][B][H]
    uint16_t* logits;          // [B][V]
    uint16_t* qA;              // [B][H] the query block, O's input
    float* sq;                 // 3 x [B][stage_sq_ld(H)] sums of squares (u, a, x1)
};

// Row tiles of a stage hold at least 16 rows.
inline int stage_sq_ld(int H) { return H / 16; }

struct StageModel {
    const wq4_layer_table* table;
    int H, F, Nqkv, V, B;
    StageBuffers buf;
    int sms;
    size_t smem_max;
    uint32_t* err;
};

// Records the decode step's attention of layer `layer` on `cs`, between its
// QKV and O stages: it sets *o_in to the O stage's [B][H] input and leaves the
// sums of squares of its 128-element tiles in sq.
struct StageAttnHook {
    int (*record)(void* ctx, int layer, cudaStream_t cs, const uint16_t** o_in, float* sq);
    void* ctx;
};

// Records one token (the squares of its input and every stage kernel) on
// `cs`; with `att`, the attention of every layer between its QKV and O stages.
int stage_record_token(const StageModel& m, cudaStream_t cs, const StageAttnHook* att = nullptr);

// Records the sums of squares of the 128-element tiles of a [B][H] input.
int stage_launch_squares(const uint16_t* x, int H, int B, float* sq, cudaStream_t cs);

}  // namespace wq4
