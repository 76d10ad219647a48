// Whole decoding steps of the CUDA-core path in one launch (library-private interface).
#pragma once
#include "kernels.h"

namespace llma {

// Projection of a pass: 4 l + {0 QKV, 1 output, 2 gate/up, 3 down} of layer l, then the LM head
struct SimtOp {
    const void *w0, *w1, *w2;
    const float* gain;   // RMSNorm of the input rows, or nullptr
};
struct SimtGeo {         // shape of a class of projections (QKV, output, gate/up, down, LM head)
    int32_t n_units;     // groups of four pairs of output features
    int32_t k_in;
    int32_t n_pieces;    // pieces of eight 16-byte loads that a weight row consists of
    int32_t split_lg;    // log2 of the warps that share a unit
    int32_t sweep_rows, sweep_cols;  // 2 * threads activations, as rows and columns of this width
};
struct SimtStep {
    ModelDims dims;
    TailArgs tail;       // n, k
    SimtGeo geo[5];
    const SimtOp* ops;   // [4 n_layers + 1], device
    const void* emb;
    RowDesc* rows;
    // activations on their way from CTA to CTA: [row_cap][width] words of a value and the number of the projection that wrote it
    unsigned long long *ll_x, *ll_qkv, *ll_attn, *ll_h;
    unsigned long long* ll_part;         // [CTAs][row_cap][2]: LM-head maximum and its index
    unsigned long long* ll_rows;         // two steps in turn: [2 + 4 row_cap]: rows in use, 0; token, position, sequence, its first row
    uint32_t epoch;                      // first number of this launch
    float *x, *qkv, *attn, *h, *logits;  // plain copies (inspection); logits may be nullptr
    void *kcache, *vcache;
    const float *rope_cos, *rope_sin;
    uint32_t* barrier;
    int32_t* dev_err;
    int32_t pass_rows;   // rows that one pass over the weights takes
    int32_t passes;      // most passes of a step
    int32_t ring_offset, gain_offset, ops_offset;  // bytes of dynamic shared memory before the weight ring, a norm's gains, the ops
    int32_t max_steps;   // steps of this launch; it ends early once no sequence has anything left to do
    int32_t patience;    // polls before a wait gives up
};
// numbers that a step takes: at least one per projection, and an odd number (ll_rows has a half for odd and one for even steps)
__host__ __device__ inline uint32_t simt_epochs(const ModelDims& d) { return 4u * d.n_layers + 3u; }
inline size_t simt_rows_words(int row_cap) { return 2 * (2 + 4 * (size_t)row_cap); }

// Whether the shape can run this way; fills geo, pass_rows, the offsets and the launch's shared memory.
bool step_simt_shape(const ModelDims& d, bool bf16, int y_cap, int num_sms, SimtStep* s, size_t* smem);
cudaError_t init_step_simt(bool bf16, int head_dim, size_t smem, bool* fits);
// What a step gives does not depend on the number of CTAs (two at least).
cudaError_t launch_step_simt(cudaStream_t st, bool bf16, const SimtStep& s, size_t smem, int ctas);

}  // namespace llma
