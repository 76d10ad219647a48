// Engine object behind the C ABI (library-private).
#pragma once
#include <map>
#include <utility>
#include <vector>

#include "../../include/llma.h"
#include "attention_mma.cuh"
#include "device_gate.h"
#include "gemm_tcgen05.cuh"
#include "kernels.h"
#include "step_simt.cuh"

struct llma_engine {
    llma_config cfg;
    llma::ModelDims dims;
    bool bf16 = false;
    int gemm_impl = LLMA_GEMM_SIMT;
    cudaStream_t stream = nullptr;
    int device = 0;

    // borrowed weights (host copies of the per-layer pointer arrays)
    const void *tok_emb = nullptr, *lm_head = nullptr;
    const float* final_norm = nullptr;
    std::vector<const float*> attn_norm, ffn_norm;
    std::vector<const void*> wq, wk, wv, wo, w_gate, w_up, w_down;

    // device state
    llma::SeqState* seq_state = nullptr;
    llma::RowDesc* rows = nullptr;
    int32_t *ref = nullptr, *y = nullptr, *out_tok = nullptr;  // ref: [max_batch][3][max_ref] = tokens, document starts, ends
    int32_t* dev_err = nullptr;                                // the word behind seq_state (one copy brings both)
    int32_t y_cap = 0;
    float *x = nullptr, *qkv = nullptr, *logits = nullptr;
    void *x_hat = nullptr, *attn = nullptr, *h = nullptr;
    float *rope_cos = nullptr, *rope_sin = nullptr;
    void *kcache = nullptr, *vcache = nullptr;

    // row capacities: the activation buffers of decoding steps (and of the CUDA-core path's prompt passes) hold row_cap
    // rows; a decoding step uses at most decode_rows = max_batch * (max_k + 1) of them, rounded up to 16
    int row_cap = 0, decode_rows = 0, prefill_rows = 0;  // prefill_rows: CUDA-core path

    // tensor-core GEMM path (bf16): TMA descriptors of weights and activation buffers, work buffers
    struct LayerMaps { CUtensorMap wq, wk, wv, wo, w_gate, w_up, w_down; };
    std::vector<LayerMaps> maps;    // 2-D views (gemm_wide_kernel; gate/up of both kernels)
    std::vector<LayerMaps> maps2;   // chunk-pair views (gemm_ws_kernel; gate/up entries are the 2-D ones)
    CUtensorMap map_lm_head, map_lm_head2;
    struct PairMap { CUtensorMap map; int gate_second; };   // gate and up matrices of a layer in one view (gemm_ws_kernel)
    std::vector<PairMap> gate_up_map;
    // activation operands of gemm_wide_kernel: boxes of min(32, nr), min(64, nr), min(128, nr) and nr rows (the kernel
    // takes the smallest that holds the step's rows)
    struct ActMaps { CUtensorMap x_hat[4], attn[4], h[4]; };
    ActMaps act_decode;
    bool decode_wide = false;       // decoding steps of more than 32 rows use gemm_wide_kernel
    int decode_nr = 32;             // rows the decoding GEMMs are shaped for (16 / 32 narrow, decode_rows wide)
    int cur_rows = 32;              // row slots of the launches being enqueued (decoding step or CUDA-core prompt pass)
    int num_sms = 0;
    unsigned long long* stamps = nullptr;  // timeline blocks (allocated in measurement builds only)
    int launch_seq = 0;                    // projections enqueued since the step began
    float* gemm_ws = nullptr;       // partial tiles of gemm_ws_kernel [num_sms][8][128] float4
    float* gemm_ws_wide = nullptr;  // partial tiles of gemm_wide_kernel [num_sms][2][wide_nr / 4][128] float4
    uint32_t* gemm_flags = nullptr; // gemm_wide_kernel's hand-over flags [num_sms][2]
    size_t gemm_ws_bytes = 0;
    float* norm_ss = nullptr;       // per-tile sums of squares of the residual rows [d/128][row_cap]
    float* part_max = nullptr;      // LM-head per-tile maxima [tiles][row_cap]
    int32_t* part_idx = nullptr;

    // Prompt passes of the tensor-core path: up to prompt_rc positions of one sequence at a time, with buffers of their own
    int prompt_rc = 0;
    int prompt_pairs = 0;           // CTA pairs of gemm_prompt_kernel that run at once
    int32_t* p_tok = nullptr;       // [max_seq] the prompt
    float *p_x = nullptr, *p_q = nullptr, *p_ss = nullptr;
    void *p_x_hat = nullptr, *p_attn = nullptr, *p_h = nullptr;
    CUtensorMap map_kcache_64, map_vcache_64;  // boxes of kPromptKV rows

    // tensor-core attention: TMA descriptors of the K/V cache, chunk partials
    CUtensorMap map_kcache, map_vcache;
    int attn_chunks = 0;
    int attn_tiles = 1;             // 128-position tiles per attention CTA in decoding steps (a function of the capacity only)
    float *attn_ws_o = nullptr, *attn_ws_ml = nullptr;

    // whole steps in one launch (step_simt.cu): CUDA-core path, and narrow decoders of the tensor-core path
    bool step_simt = false;
    bool plain_acts = false;        // attn and h hold fp32 rows (of a whole step), whatever the path
    llma::SimtStep simt{};          // everything that does not change from launch to launch
    size_t simt_smem = 0;
    unsigned long long* ll_words = nullptr;   // activations on their way from CTA to CTA; behind them the barrier's word and the ops
    size_t ll_count = 0;
    uint32_t* grid_barrier = nullptr;
    uint32_t ll_epoch = 1;                    // first number of the next launch

    llma::GateMember gate;                    // turns with the other engines of the device

    // replay of a given step sequence (llma_generate_forced)
    int32_t *trace = nullptr, *target = nullptr;
    int32_t trace_cap = 0;

    // Page-locked host memory, one block.  h_state mirrors seq_state between calls (nothing runs then): calls that only change a
    // sequence's bookkeeping change the mirror, and the next call that launches kernels uploads it in one copy.
    char* h_block = nullptr;
    llma::SeqState* h_state = nullptr;
    int32_t* h_err = nullptr;               // the word behind h_state
    bool state_dirty = false;               // the mirror is ahead of seq_state
    bool state_stale = false;               // a call failed on the way: seq_state has to be read again
    llma::RowDesc* h_rows = nullptr;
    int32_t* h_y = nullptr;                 // [max_batch][y_cap]: emitted tokens on their way to the caller
    int32_t* h_ref[2] = {nullptr, nullptr}; // [3][max_ref] each: references on their way to the device, used in turn
    cudaEvent_t ref_ev[2] = {nullptr, nullptr};
    int ref_turn = 0;
    float* h_logits = nullptr;              // kLogitStage floats (llma_debug_logits)

    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    // captured steps by (n, k): of llma_generate, and of llma_step (there null until use kCaptureAt); at most kStepGraphs each
    struct StepGraph { cudaGraphExec_t exec; uint64_t used; int uses; };
    typedef std::map<std::pair<int, int>, StepGraph> StepGraphs;
    StepGraphs step_graphs, lone_graphs;
    uint64_t graph_clock = 0;
    bool can_capture = true;     // false on the legacy default stream, which CUDA does not capture: steps are launched directly
    int64_t launches_per_step = 0;
    int64_t launch_counter = 0;  // kernels enqueued since it was last cleared
    bool last_step_valid = false;
    bool prof_on = false;               // llma_profile_steps: record an event after every launch
    std::vector<cudaEvent_t> prof_ev;
    std::vector<int> prof_cls;
    size_t prof_n = 0;
    std::vector<int32_t> prompt_last;  // last prompt token of every sequence (the first pending input)
};

namespace llma {
constexpr int kPromptPassRows = 2048;    // most positions of a prompt pass (110 KB of buffers per position at the 7B widths)
constexpr int kPromptPassRowsMin = 128;  // ... and the fewest where memory is short
constexpr size_t kStepGraphs = 64;     // n is any positive number: the pair used longest ago makes room
// llma_step launches kernel by kernel until an (n, k) has been used this often: capturing a step costs what a graph saves in 12 to
// 23 of them (two layers of width 1024 115 against 10 us, three of width 512 170 against 8, the 7B shape 1400 against 60).
constexpr int kCaptureAt = 16;
// Steps of one launch of a whole-step kernel, which ends by itself once there is nothing left to do: enough that launching costs
// nothing (5 us against 32 steps of 20 us and more), few enough that other streams get the GPU every millisecond or so.
constexpr int kStepsPerLaunch = 32;
// Steps that an engine launches at a time where engines of the other kind wait for their turns (device_gate.h).  Decodes per second of two
// engines side by side, as launches that overlapped -> turns of 8 steps (turns of 32 whole steps): two fp32 layers of width 256 beside two
// 7B-shaped layers 143 and 150 -> 233 and 129 (397 and 89), beside two bf16 layers of width 1024 320 and 379 -> 411 and 229 (567
// and 127).  The first engine alone: 721 a second, 684 with a look at its state every 8 steps.
constexpr int kStepsPerTurn = 8;
constexpr size_t kLogitStage = 1u << 17;  // floats
int sync_state(llma_engine* e);  // h_state up to date
void gemm_count_engine(int dev, int by);  // the last engine of a device takes the scratch that llma_gemm_rows32_bf16 keeps with it
void note_cuda_error(cudaError_t err);  // remembers the code for llma_last_cuda_error, clears the sticky flag
}

#define CU_TRY(expr)                          \
    do {                                      \
        cudaError_t _e = (expr);              \
        if (_e != cudaSuccess) {              \
            llma::note_cuda_error(_e);        \
            return LLMA_ERR_CUDA;             \
        }                                     \
    } while (0)
