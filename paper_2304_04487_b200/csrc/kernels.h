// Launch wrappers of the engine's kernels (library-private).
#pragma once
#include "common.cuh"

namespace llma {

// ---- integer side (kernels_int.cu) ----------------------------------------------------
// Arguments of step_tail_kernel: acceptance + K/V commit of the forward pass that has just finished
// (do_accept) and trigger search + copy + row packing for the one that follows (do_plan).
struct TailArgs {
    ModelDims dims;
    SeqState* st;
    RowDesc* rows;
    const int32_t* ref;        // [max_batch][3][max_ref]: reference tokens, start and end of each one's document
    int32_t* y;
    int32_t y_cap;
    int32_t n, k;
    int32_t do_accept, do_plan;
    // accept
    const float* part_max;     // [n_tiles][row_cap] per-tile maxima of the LM head
    const int32_t* part_idx;
    int32_t n_tiles;
    int32_t* out_tok;          // [row_cap]
    int32_t n_rows;            // row slots of a decoding step (decode_rows)
    // replay
    const int32_t* trace;      // [max_batch][trace_cap][2] = (rows, emitted) of every step, or nullptr
    const int32_t* target;     // [max_batch][y_cap] the text to reproduce
    int32_t trace_cap;
    int32_t* dev_err;
};


void launch_step_tail(cudaStream_t st, const TailArgs& a);
// embedding gather over the first n_rows row slots (rows not in use are zero-filled)
void launch_embed(cudaStream_t st, const ModelDims& dims, bool bf16, int n_rows, const RowDesc* rows, const void* emb,
                  float* x, int32_t* dev_err);
// bf16 embedding gather with the first RMSNorm folded in: x, xs = split(x * gain), ss[tile][row]
void launch_embed_norm(cudaStream_t st, const ModelDims& dims, int n_rows, const RowDesc* rows, const void* emb,
                       const float* gain, float* x, void* xs, float* ss, int32_t* dev_err);

// the same for a prompt pass: row r is token toks[r]; rc = row capacity of xs
void launch_embed_prompt(cudaStream_t st, const ModelDims& dims, int n_rows, int rc, const int32_t* toks, const void* emb,
                         const float* gain, float* x, void* xs, float* ss);

// ---- CUDA-core projections, fp32 or bf16 weights (kernels_simt.cu) ----------------------
enum RowMode : int32_t {
    kRowQKV = 0,     // w0, w1, w2 = wq, wk, wv; rotary embedding; q, k, v -> out [rows][3 HD] (q rotated), k and v -> cache
    kRowResid = 1,   // out[r, n] += sum
    kRowSwiGLU = 2,  // w0, w1 = gate, up; out[r, f] = silu(gate) * up
    kRowHead = 3,    // logits to out unless it is nullptr; per-CTA (max, argmax) of every row
};
struct RowGemm {
    int32_t mode;
    const RowDesc* rows;
    const void *w0, *w1, *w2;
    const float* act;       // [rows][k_in]
    const float* gain;      // RMSNorm of the input rows (every mode but kRowResid)
    float eps;
    int32_t n_units;        // pairs of output features
    int32_t n_out, k_in;
    float* out;
    int32_t ld;
    ModelDims dims;
    int32_t layer;
    const float *rope_cos, *rope_sin;
    void *kcache, *vcache;
    float* part_max;        // kRowHead: [grid][row_cap]
    int32_t* part_idx;
    int32_t split_lg;       // set by launch_rowgemm: log2 of the warps that share a unit
    int32_t pass_rows;      // ... and the rows that one pass over the weights takes
};
cudaError_t init_rowgemm(bool bf16);
// row_bound: most rows of a step (more than a pass takes: further passes over the weights inside the launch)
void launch_rowgemm(cudaStream_t st, bool bf16, RowGemm g, int row_bound, int num_sms);
// passes over a matrix with inputs of this width
int rowgemm_passes(int rows, int k_in);
// CTAs of a launch (the number of partial maxima of kRowHead)
int rowgemm_grid(int n_units, int k_in, int row_bound, int num_sms);
// causal attention of every used row over its sequence's cache rows [0, pos]; n_rows = the row slots of the pass
void launch_attention_simt(cudaStream_t st, bool bf16, const ModelDims& dims, int layer, int n_rows,
                           const RowDesc* rows, const float* qkv, const void* kcache, const void* vcache,
                           float* attn_out);

}  // namespace llma
