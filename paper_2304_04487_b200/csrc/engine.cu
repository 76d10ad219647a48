// C ABI of the LLMA engine: object lifetime, prompt prefill, reference upload, the decoding
// step (Algorithm 1's loop body) and the whole decoding loop.  See include/llma.h.
#include "engine.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

using namespace llma;

static thread_local int g_last_cuda_error = 0;
void llma::note_cuda_error(cudaError_t err) {
    g_last_cuda_error = (int)err;
    (void)cudaGetLastError();
}

static size_t esize(const llma_engine* e) { return e->bf16 ? 2 : 4; }

template <typename T>
static cudaError_t dalloc(T** p, size_t count, bool zero = true) {
    cudaError_t r = cudaMalloc((void**)p, count * sizeof(T));
    if (r != cudaSuccess) return r;
    if (zero) r = cudaMemset(*p, 0, count * sizeof(T));
    return r;
}

extern "C" int llma_last_cuda_error(void) { return g_last_cuda_error; }

extern "C" const char* llma_strerror(int s) {
    switch (s) {
        case LLMA_OK: return "ok";
        case LLMA_ERR_NULL: return "required pointer is NULL";
        case LLMA_ERR_CONFIG: return "unsupported or inconsistent configuration";
        case LLMA_ERR_TOKEN_RANGE: return "token id outside [0, vocab)";
        case LLMA_ERR_CAPACITY: return "sequence capacity (max_seq / max_batch) exceeded";
        case LLMA_ERR_REF_TOO_LONG: return "reference too long or malformed document offsets";
        case LLMA_ERR_STATE: return "call not valid in the current state";
        case LLMA_ERR_CUDA: return "CUDA call failed";
        case LLMA_ERR_DEVICE_TIMEOUT: return "bounded device-side wait ran out";
        case LLMA_ERR_ARG: return "argument out of range";
        default: return "unknown status";
    }
}

static void free_prompt_buffers(llma_engine* e) {
    for (void* b : {(void*)e->p_x, (void*)e->p_q, (void*)e->p_ss, e->p_x_hat, e->p_attn, e->p_h}) cudaFree(b);
    e->p_x = e->p_q = e->p_ss = nullptr;
    e->p_x_hat = e->p_attn = e->p_h = nullptr;
}

static void free_engine(llma_engine* e) {
    if (!e) return;
    gate_quit(&e->gate);
    for (auto* graphs : {&e->step_graphs, &e->lone_graphs})
        for (auto& kv : *graphs) if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
    cudaFree(e->seq_state); cudaFree(e->rows); cudaFree(e->ref);
    cudaFree(e->y); cudaFree(e->out_tok); cudaFree(e->x); cudaFree(e->qkv);
    cudaFree(e->logits); cudaFree(e->x_hat); cudaFree(e->attn); cudaFree(e->h);
    cudaFree(e->rope_cos); cudaFree(e->rope_sin); cudaFree(e->kcache); cudaFree(e->vcache);
    cudaFree(e->attn_ws_o); cudaFree(e->attn_ws_ml); cudaFree(e->trace); cudaFree(e->target);
    cudaFree(e->gemm_ws); cudaFree(e->stamps); cudaFree(e->gemm_ws_wide); cudaFree(e->gemm_flags); cudaFree(e->part_max); cudaFree(e->part_idx); cudaFree(e->norm_ss);
    cudaFree(e->p_tok); cudaFree(e->ll_words);
    free_prompt_buffers(e);
    if (e->h_block) cudaFreeHost(e->h_block);
    for (int i = 0; i < 2; ++i)
        if (e->ref_ev[i]) cudaEventDestroy(e->ref_ev[i]);
    for (cudaEvent_t ev : e->prof_ev) cudaEventDestroy(ev);
    if (e->ev0) cudaEventDestroy(e->ev0);
    if (e->ev1) cudaEventDestroy(e->ev1);
    delete e;
}

// The buffers of a prompt pass of prompt_rc positions, all of them or none
static cudaError_t alloc_prompt_buffers(llma_engine* e) {
    const ModelDims& d = e->dims;
    const size_t rows = (size_t)e->prompt_rc;
    cudaError_t r = dalloc(&e->p_x, rows * d.d_model, false);
    if (r == cudaSuccess) r = dalloc(&e->p_q, rows * d.hd_total, false);
    if (r == cudaSuccess) r = dalloc(&e->p_ss, rows * (d.d_model / 128), false);
    // rows past a pass are multiplied too (their results go nowhere): zeroed, so that they stay finite
    if (r == cudaSuccess) r = dalloc((char**)&e->p_x_hat, rows * d.d_model * 4);
    if (r == cudaSuccess) r = dalloc((char**)&e->p_attn, rows * d.hd_total * 4);
    if (r == cudaSuccess) r = dalloc((char**)&e->p_h, rows * d.d_ffn * 4);
    if (r != cudaSuccess) free_prompt_buffers(e);
    return r;
}

// Where whole steps on the CUDA cores pay.  They save the ends of launches, some 10 us a layer, and lose where a step has many rows: a matrix
// is read once per pass, the rows of a pass are bounded by the widest input, and their products cost more here.  Decodes alternate
// between steps of one row a sequence and steps of all rows; the lines were drawn with references that agree with 60 and 95 % of
// the text (a tenth to a fifth and a third to a half of the steps are copies).  Times launches / whole steps, 60 and 95 %:
//
// Against launches on the CUDA cores (fp32; bf16 the same), width / FFN width, rows of one or four sequences: 256 / 1024 4 x 19 1.70, 1.39;
// 512 / 1408 4 x 19 1.35, 1.17; 1024 / 2816 16 rows in two passes 1.55, 1.16, 4 x 9 in four for three 1.14, 0.92, 4 x 19 in eight for five 1.15, 0.92;
// 1536 / 4096 9 rows in two passes for one 1.31, 1.03, 16 in three for one 1.54, 1.08; 2048 / 5632 5 in two for one 1.19, 0.93, 9 in three for
// one 1.26, 0.95, and where only two rows fit a pass: 2048 / 8192 5 rows 1.07, 0.77, 1024 / 8192 9 rows 1.08, 0.74, 512 / 8192 5 rows 1.20, 0.86.
// So at least four rows have to fit, and matrices may be read twice more than by the launches at most.
//
// Against tensor cores, width, FFN width, vocabulary, rows, positions: 256, 1024, 4096, 16, 650 1.62, 1.42; 512, 1408, 5000, 16, 300 1.47, 1.20, at 650
// 1.29, 1.08; vocabulary 32000, 9, 300 1.24, 1.04, 16, 650 1.16, 0.97; 128000, 5, 300 1.19, 1.05, 16, 300 1.17, 0.90; six layers 512, 2048, 32000, 16, 300 1.25,
// 1.03, at 650 1.10, 0.92; more than a pass: 512, 4096, 5000, 9, 60 1.18, 0.89, 512, 8192, 5000, 9, 300 0.73, 0.47.  Width 1024, two layers, 13 rows,
// 2000 positions lost a third (a row and head is one CTA's work here, 0.6 us per 64 positions).  So one pass, and the products of a layer
// and of a part of the LM head bounded by a line that falls with the positions.
static bool whole_steps_pay(const llma_engine* e, const SimtStep& s) {
    const ModelDims& d = e->dims;
    const int rows = d.max_batch * d.kp1;
    if (e->gemm_impl != LLMA_GEMM_TCGEN05) {
        if (s.passes > 1 && s.pass_rows < 4) return false;
        for (int k_in : {d.d_model, d.hd_total, d.d_ffn})
            if (s.passes > rowgemm_passes(rows, k_in) + 2) return false;
        return true;
    }
    const int64_t layer = 4ll * d.d_model * d.hd_total + 3ll * d.d_model * d.d_ffn, head = (int64_t)d.d_model * d.vocab / (4 * d.n_layers);
    return s.passes == 1 && d.d_model <= 512 && d.d_model * d.max_batch <= 1024 && d.max_seq <= 768 &&
           rows * (layer + head) <= 190000ll * (1100 - d.max_seq);
}

// A stream of a green context has some of the SMs only, where a launch that needs them all would never get its CTAs together.
static bool has_every_sm(const llma_engine* e) {
    auto entry = [](const char* name) -> void* {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        return cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &q) == cudaSuccess ? p : nullptr;
    };
    auto of_stream = reinterpret_cast<CUresult (*)(CUstream, CUgreenCtx*)>(entry("cuStreamGetGreenCtx"));
    auto resource = reinterpret_cast<CUresult (*)(CUgreenCtx, CUdevResource*, CUdevResourceType)>(entry("cuGreenCtxGetDevResource"));
    CUgreenCtx green = nullptr;
    CUdevResource sms;
    if (!of_stream || !resource || of_stream(e->stream, &green) != CUDA_SUCCESS || !green) return true;
    return resource(green, &sms, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS && (int)sms.sm.smCount >= e->num_sms;
}

// Whole decoding steps in one launch, where they are possible and pay
static cudaError_t init_whole_steps(llma_engine* e) {
    const ModelDims& d = e->dims;
    SimtStep& s = e->simt;
    bool fits = false;
    if (!step_simt_shape(d, e->bf16, e->y_cap, e->num_sms, &s, &e->simt_smem) || !whole_steps_pay(e, s) || !has_every_sm(e)) return cudaSuccess;
    cudaError_t r = init_step_simt(e->bf16, d.head_dim, e->simt_smem, &fits);
    if (r != cudaSuccess || !fits) return r;
    std::vector<SimtOp> ops;
    for (int l = 0; l < d.n_layers; ++l) {
        ops.push_back({e->wq[l], e->wk[l], e->wv[l], e->attn_norm[l]});
        ops.push_back({e->wo[l], nullptr, nullptr, nullptr});
        ops.push_back({e->w_gate[l], e->w_up[l], nullptr, e->ffn_norm[l]});
        ops.push_back({e->w_down[l], nullptr, nullptr, nullptr});
    }
    ops.push_back({e->lm_head, nullptr, nullptr, e->final_norm});
    const size_t rc = (size_t)e->row_cap, parts = 2 * (size_t)e->num_sms * rc;
    e->ll_count = rc * (d.d_model + 4 * (size_t)d.hd_total + d.d_ffn) + parts + simt_rows_words(e->row_cap);
    // one block: the words, the barrier's, the ops
    const size_t words = e->ll_count + 1 + (ops.size() * sizeof(SimtOp) + 7) / 8;
    r = dalloc(&e->ll_words, words);
    if (r == cudaErrorMemoryAllocation) {  // no room for them: steps are launched kernel by kernel, which needs none
        cudaGetLastError();
        e->ll_words = nullptr;
        return cudaSuccess;
    }
    if (r != cudaSuccess) return r;
    e->grid_barrier = reinterpret_cast<uint32_t*>(e->ll_words + e->ll_count);
    SimtOp* step_ops = reinterpret_cast<SimtOp*>(e->ll_words + e->ll_count + 1);
    if ((r = cudaMemcpy(step_ops, ops.data(), ops.size() * sizeof(SimtOp), cudaMemcpyHostToDevice)) != cudaSuccess) return r;
    s.ll_x = e->ll_words; s.ll_qkv = s.ll_x + rc * d.d_model; s.ll_attn = s.ll_qkv + rc * 3 * d.hd_total;
    s.ll_h = s.ll_attn + rc * d.hd_total; s.ll_part = s.ll_h + rc * d.d_ffn; s.ll_rows = s.ll_part + parts;
    s.dims = d; s.ops = step_ops; s.emb = e->tok_emb; s.rows = e->rows;
    s.x = e->x; s.qkv = e->qkv; s.attn = (float*)e->attn; s.h = (float*)e->h; s.logits = e->cfg.keep_logits ? e->logits : nullptr;
    s.kcache = e->kcache; s.vcache = e->vcache; s.rope_cos = e->rope_cos; s.rope_sin = e->rope_sin;
    s.barrier = e->grid_barrier; s.dev_err = e->dev_err;
    e->step_simt = true;
    return cudaSuccess;
}

extern "C" int llma_create(const llma_config* cfg, const llma_weights* w, void* cuda_stream, llma_engine** out) {
    if (!cfg || !w || !out) return LLMA_ERR_NULL;
    *out = nullptr;
    const int L = cfg->n_layers;
    if (L < 1 || cfg->d_model < 64 || cfg->n_heads < 1 || cfg->d_ffn < 64 || cfg->vocab < 2) return LLMA_ERR_CONFIG;
    if (cfg->head_dim != 64 && cfg->head_dim != 128) return LLMA_ERR_CONFIG;
    const int HD = cfg->n_heads * cfg->head_dim;
    if (cfg->d_model % 64 || HD % 64 || cfg->d_ffn % 64) return LLMA_ERR_CONFIG;
    if (cfg->dtype != LLMA_DTYPE_F32 && cfg->dtype != LLMA_DTYPE_BF16) return LLMA_ERR_CONFIG;
    if (cfg->max_batch < 1 || cfg->max_batch > kSeqCap || cfg->max_k < 0 ||
        (int64_t)cfg->max_batch * (cfg->max_k + 1) > kRowCap)
        return LLMA_ERR_CONFIG;
    if (cfg->max_seq < 2 || cfg->max_ref < 0 || !(cfg->rms_eps >= 0.f) || !(cfg->rope_theta > 0.f)) return LLMA_ERR_CONFIG;
    if (cfg->gemm_impl < LLMA_GEMM_AUTO || cfg->gemm_impl > LLMA_GEMM_TCGEN05) return LLMA_ERR_CONFIG;
    if (!w->tok_emb || !w->lm_head || !w->final_norm || !w->attn_norm || !w->wq || !w->wk || !w->wv || !w->wo ||
        !w->ffn_norm || !w->w_gate || !w->w_up || !w->w_down)
        return LLMA_ERR_NULL;
    for (int l = 0; l < L; ++l)
        if (!w->attn_norm[l] || !w->wq[l] || !w->wk[l] || !w->wv[l] || !w->wo[l] || !w->ffn_norm[l] ||
            !w->w_gate[l] || !w->w_up[l] || !w->w_down[l])
            return LLMA_ERR_NULL;

    // the kernels read weight rows in 16-byte pieces, gains and embeddings value by value
    auto off = [](const void* p, size_t grid) { return reinterpret_cast<uintptr_t>(p) % grid != 0; };
    const size_t value = cfg->dtype == LLMA_DTYPE_BF16 ? 2 : 4;
    bool misaligned = off(w->tok_emb, value) || off(w->lm_head, 16) || off(w->final_norm, 4);
    for (int l = 0; l < L; ++l) {
        misaligned = misaligned || off(w->attn_norm[l], 4) || off(w->ffn_norm[l], 4);
        for (const void* m : {w->wq[l], w->wk[l], w->wv[l], w->wo[l], w->w_gate[l], w->w_up[l], w->w_down[l]}) misaligned = misaligned || off(m, 16);
    }
    if (misaligned) return LLMA_ERR_CONFIG;

    int dev = 0;
    CU_TRY(cudaGetDevice(&dev));
    llma_engine* e = new (std::nothrow) llma_engine();
    if (!e) return LLMA_ERR_CUDA;
    e->cfg = *cfg;
    e->device = dev;
    e->stream = (cudaStream_t)cuda_stream;
    e->can_capture = e->stream != nullptr && e->stream != cudaStreamLegacy;
    e->bf16 = cfg->dtype == LLMA_DTYPE_BF16;
    const bool tc_ok = cfg->dtype == LLMA_DTYPE_BF16 && HD % 128 == 0 && cfg->d_model % 128 == 0;
    if (cfg->gemm_impl == LLMA_GEMM_TCGEN05 && !tc_ok) { delete e; return LLMA_ERR_CONFIG; }
    e->gemm_impl = cfg->gemm_impl == LLMA_GEMM_AUTO ? (tc_ok ? LLMA_GEMM_TCGEN05 : LLMA_GEMM_SIMT) : cfg->gemm_impl;
    ModelDims& d = e->dims;
    d.n_layers = L; d.d_model = cfg->d_model; d.n_heads = cfg->n_heads; d.head_dim = cfg->head_dim;
    d.d_ffn = cfg->d_ffn; d.vocab = cfg->vocab; d.hd_total = HD; d.max_batch = cfg->max_batch;
    d.max_seq = cfg->max_seq; d.max_ref = cfg->max_ref > 0 ? cfg->max_ref : 1; d.kp1 = cfg->max_k + 1;
    d.rms_eps = cfg->rms_eps; d.eos_id = cfg->eos_id;
    // Row capacities (the tensor-core path has buffers of their own for prompt passes, the CUDA-core path pushes up to
    // prefill_rows consecutive positions of one sequence through the decoding kernels)
    e->decode_rows = (d.max_batch * d.kp1 + 15) / 16 * 16;
    e->prefill_rows = std::max(e->decode_rows, 32);
    e->row_cap = std::max(e->decode_rows, 32);
    d.row_cap = e->row_cap;
    e->tok_emb = w->tok_emb; e->lm_head = w->lm_head; e->final_norm = w->final_norm;
    for (int l = 0; l < L; ++l) {
        e->attn_norm.push_back(w->attn_norm[l]); e->ffn_norm.push_back(w->ffn_norm[l]);
        e->wq.push_back(w->wq[l]); e->wk.push_back(w->wk[l]); e->wv.push_back(w->wv[l]); e->wo.push_back(w->wo[l]);
        e->w_gate.push_back(w->w_gate[l]); e->w_up.push_back(w->w_up[l]); e->w_down.push_back(w->w_down[l]);
    }
    e->y_cap = d.max_seq;
    e->prompt_last.assign((size_t)d.max_batch, 0);

#define CREATE_TRY(expr)                              \
    do {                                              \
        cudaError_t _e = (expr);                      \
        if (_e != cudaSuccess) {                      \
            llma::note_cuda_error(_e);                \
            free_engine(e);                           \
            return LLMA_ERR_CUDA;                     \
        }                                             \
    } while (0)

    const size_t B = d.max_batch, es = esize(e);
    CREATE_TRY(dalloc((char**)&e->seq_state, B * sizeof(SeqState) + sizeof(int32_t)));
    e->dev_err = reinterpret_cast<int32_t*>(e->seq_state + B);
    CREATE_TRY(dalloc(&e->rows, 1));
    CREATE_TRY(dalloc(&e->ref, B * 3 * d.max_ref));
    CREATE_TRY(dalloc(&e->y, B * e->y_cap));
    const size_t RC = (size_t)e->row_cap;
    CREATE_TRY(dalloc(&e->out_tok, RC));
    e->trace_cap = e->y_cap;
    CREATE_TRY(dalloc(&e->trace, B * e->trace_cap * 2));
    CREATE_TRY(dalloc(&e->target, B * e->y_cap));
    CREATE_TRY(dalloc(&e->x, RC * d.d_model));
    CREATE_TRY(dalloc(&e->qkv, RC * 3 * HD));
    if (cfg->keep_logits) CREATE_TRY(dalloc(&e->logits, RC * d.vocab));
    // activation operands: fp32 [rc][K] (CUDA cores, which need no x_hat) or split bf16 [2 rc][K] (tensor cores): 4 bytes per element
    if (e->gemm_impl == LLMA_GEMM_TCGEN05) CREATE_TRY(dalloc((char**)&e->x_hat, RC * d.d_model * 4));
    CREATE_TRY(dalloc((char**)&e->attn, RC * HD * 4));
    CREATE_TRY(dalloc((char**)&e->h, RC * d.d_ffn * 4));
    const size_t kv_elems = (size_t)L * B * d.n_heads * d.max_seq * d.head_dim;
    CREATE_TRY(dalloc((char**)&e->kcache, kv_elems * es));
    CREATE_TRY(dalloc((char**)&e->vcache, kv_elems * es));

    // rotary table: angle(pos, i) = pos * theta^(-2i/hd), evaluated in double on the host
    {
        const int half = d.head_dim / 2;
        std::vector<float> c((size_t)d.max_seq * half), s((size_t)d.max_seq * half);
        for (int i = 0; i < half; ++i) {
            const double inv = std::pow((double)cfg->rope_theta, -2.0 * (double)i / (double)d.head_dim);
            for (int p = 0; p < d.max_seq; ++p) {
                const double a = (double)p * inv;
                c[(size_t)p * half + i] = (float)std::cos(a);
                s[(size_t)p * half + i] = (float)std::sin(a);
            }
        }
        CREATE_TRY(dalloc(&e->rope_cos, c.size(), false));
        CREATE_TRY(dalloc(&e->rope_sin, s.size(), false));
        CREATE_TRY(cudaMemcpy(e->rope_cos, c.data(), c.size() * 4, cudaMemcpyHostToDevice));
        CREATE_TRY(cudaMemcpy(e->rope_sin, s.data(), s.size() * 4, cudaMemcpyHostToDevice));
    }
    CREATE_TRY(cudaDeviceGetAttribute(&e->num_sms, cudaDevAttrMultiProcessorCount, dev));
    const int vt = (d.vocab + 127) / 128;  // LM-head tiles; the CUDA-core kernel has at most two CTAs per SM
    const size_t parts_max = std::max<size_t>(vt, (size_t)2 * e->num_sms);
    CREATE_TRY(dalloc(&e->part_max, parts_max * RC));
    CREATE_TRY(dalloc(&e->part_idx, parts_max * RC));
    if (e->gemm_impl != LLMA_GEMM_TCGEN05) {
        CREATE_TRY(init_rowgemm(e->bf16));
        CREATE_TRY(init_whole_steps(e));
    }
    if (e->gemm_impl == LLMA_GEMM_TCGEN05) {
        int major = 0;
        CREATE_TRY(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
        if (major != 10) { free_engine(e); return LLMA_ERR_CONFIG; }  // tcgen05 needs sm_100
        // hand-over slots start out empty: every word the all-ones pattern (see gemm_ws_kernel)
        e->gemm_ws_bytes = gemm_ws_bytes(e->num_sms);
        CREATE_TRY(dalloc((char**)&e->gemm_ws, e->gemm_ws_bytes, false));
        CREATE_TRY(cudaMemset(e->gemm_ws, 0xFF, e->gemm_ws_bytes));
        CREATE_TRY(dalloc(&e->norm_ss, (size_t)((d.d_model + 127) / 128) * RC));
#ifdef LLMA_STAMPS
        CREATE_TRY(dalloc(&e->stamps, (size_t)kStampLaunches * kStampSlots * 8));
#endif
        e->maps.resize(L);
        e->maps2.resize(L);
        e->gate_up_map.resize(L);
        bool pair_ok = true;
        int bad = 0;
        for (int l = 0; l < L; ++l) {
            llma_engine::LayerMaps& m = e->maps[l];
            bad |= make_tensor_map_bf16(&m.wq, e->wq[l], HD, d.d_model, 128);
            bad |= make_tensor_map_bf16(&m.wk, e->wk[l], HD, d.d_model, 128);
            bad |= make_tensor_map_bf16(&m.wv, e->wv[l], HD, d.d_model, 128);
            bad |= make_tensor_map_bf16(&m.wo, e->wo[l], d.d_model, HD, 128);
            bad |= make_tensor_map_bf16(&m.w_gate, e->w_gate[l], d.d_ffn, d.d_model, 64);
            bad |= make_tensor_map_bf16(&m.w_up, e->w_up[l], d.d_ffn, d.d_model, 64);
            bad |= make_tensor_map_bf16(&m.w_down, e->w_down[l], d.d_model, d.d_ffn, 128);
            llma_engine::LayerMaps& m2 = e->maps2[l];
            bad |= make_tensor_map_bf16_chunks(&m2.wq, e->wq[l], HD, d.d_model, 128);
            bad |= make_tensor_map_bf16_chunks(&m2.wk, e->wk[l], HD, d.d_model, 128);
            bad |= make_tensor_map_bf16_chunks(&m2.wv, e->wv[l], HD, d.d_model, 128);
            bad |= make_tensor_map_bf16_chunks(&m2.wo, e->wo[l], d.d_model, HD, 128);
            bad |= make_tensor_map_bf16_chunks(&m2.w_down, e->w_down[l], d.d_model, d.d_ffn, 128);
            m2.w_gate = m.w_gate; m2.w_up = m.w_up;
            // one view over both matrices; if they lie too far apart for one, every pass uses the wide kernel
            if (make_tensor_map_bf16_pair(&e->gate_up_map[l].map, e->w_gate[l], e->w_up[l], d.d_ffn, d.d_model,
                                          &e->gate_up_map[l].gate_second) != 0)
                pair_ok = false;
        }
        bad |= make_tensor_map_bf16(&e->map_lm_head, e->lm_head, d.vocab, d.d_model, 128);
        bad |= make_tensor_map_bf16_chunks(&e->map_lm_head2, e->lm_head, d.vocab, d.d_model, 128);
        // the MMA shape of decoding steps is fixed per engine (by its row capacity), never per step
        e->decode_wide = e->decode_rows > 32 || !pair_ok;
        e->decode_nr = e->decode_wide ? std::max(e->decode_rows, 32) : (e->decode_rows <= 16 ? 16 : 32);
        // activation operands of the wide kernel: one box of nr rows per (buffer, use)
        auto act_maps = [&](llma_engine::ActMaps& m, int nr) {
            int bad2 = 0;
            for (int i = 0; i < 4; ++i) {
                const int box = wide_box_rows(nr, i);
                bad2 |= make_tensor_map_bf16_terms(&m.x_hat[i], e->x_hat, RC, d.d_model, box);
                bad2 |= make_tensor_map_bf16_terms(&m.attn[i], e->attn, RC, HD, box);
                bad2 |= make_tensor_map_bf16_terms(&m.h[i], e->h, RC, d.d_ffn, box);
            }
            return bad2;
        };
        if (e->decode_wide) {
            bad |= act_maps(e->act_decode, e->decode_nr);
            CREATE_TRY(dalloc(&e->gemm_ws_wide, (size_t)e->num_sms * 2 * 128 * RC, false));
            CREATE_TRY(dalloc(&e->gemm_flags, (size_t)e->num_sms * 2));
        }
        if (bad) { free_engine(e); return LLMA_ERR_CONFIG; }  // misaligned weight pointer or bad shape
        CREATE_TRY(init_gemm_tcgen05());
        CREATE_TRY(init_gemm_wide());
        e->attn_chunks = (d.max_seq + kAttnChunk - 1) / kAttnChunk;
        // With far more (sequence, head, 128-position tile) triples than CTAs fit on the GPU, a CTA takes several tiles in
        // a row: fewer chunk partials, and the next tile's copies overlap the arithmetic.  A function of the engine's
        // capacity only, so a row's result does not depend on the step.  Thresholds from the one-layer grid (batch x
        // cached length): from four CTAs per resident slot on two tiles pay, from eight on four; at about one CTA per
        // slot (one sequence, 2 k positions) two tiles cost 5 % of the step.
        {
            const long long triples = (long long)d.max_batch * d.n_heads * e->attn_chunks, slots = 3LL * e->num_sms;
            e->attn_tiles = (d.kp1 <= 16 && triples >= 8 * slots) ? 4 : ((d.kp1 <= 16 && triples >= 4 * slots) ? 2 : 1);
        }
        const size_t parts = (size_t)d.n_heads * e->attn_chunks * RC;
        CREATE_TRY(dalloc(&e->attn_ws_o, parts * d.head_dim));
        CREATE_TRY(dalloc(&e->attn_ws_ml, parts * 2));
        const uint64_t kv_rows = (uint64_t)L * B * d.n_heads * d.max_seq;
        if (make_tensor_map_bf16(&e->map_kcache, e->kcache, kv_rows, d.head_dim, kAttnChunk) ||
            make_tensor_map_bf16(&e->map_vcache, e->vcache, kv_rows, d.head_dim, kAttnChunk)) {
            free_engine(e);
            return LLMA_ERR_CONFIG;
        }
        CREATE_TRY(init_attention_mma());
        {
            CREATE_TRY(dalloc(&e->p_tok, (size_t)d.max_seq));
            // as many positions as a pass pays for, or fewer where memory is short (results do not depend on it)
            e->prompt_rc = std::min(kPromptPassRows, (d.max_seq - 1 + 31) / 32 * 32);
            cudaError_t pe = alloc_prompt_buffers(e);
            while (pe == cudaErrorMemoryAllocation && e->prompt_rc > kPromptPassRowsMin) {
                cudaGetLastError();
                e->prompt_rc = std::max(kPromptPassRowsMin, e->prompt_rc / 64 * 32);
                pe = alloc_prompt_buffers(e);
            }
            CREATE_TRY(pe);
            if (make_tensor_map_bf16(&e->map_kcache_64, e->kcache, kv_rows, d.head_dim, kPromptKV) ||
                make_tensor_map_bf16(&e->map_vcache_64, e->vcache, kv_rows, d.head_dim, kPromptKV)) {
                free_engine(e);
                return LLMA_ERR_CONFIG;
            }
            CREATE_TRY(init_gemm_prompt(&e->prompt_pairs));
            CREATE_TRY(init_attention_prompt());
            if (e->prompt_pairs < 1) { free_engine(e); return LLMA_ERR_CONFIG; }
        }
    }
    // (an engine asked for the tensor cores keeps to them)
    if (e->gemm_impl == LLMA_GEMM_TCGEN05 && cfg->gemm_impl == LLMA_GEMM_AUTO) CREATE_TRY(init_whole_steps(e));
    {
        // page-locked memory in one piece: every such allocation costs about a millisecond
        size_t total = 0;
        auto place = [&](size_t bytes) { const size_t at = total; total += (bytes + 255) / 256 * 256; return at; };
        const size_t at_state = place(B * sizeof(SeqState) + sizeof(int32_t)), at_rows = place(sizeof(RowDesc)),
                     at_y = place(B * e->y_cap * sizeof(int32_t)), ref_bytes = (size_t)3 * d.max_ref * sizeof(int32_t),
                     at_r0 = place(ref_bytes), at_r1 = place(ref_bytes),
                     at_logits = place(cfg->keep_logits ? kLogitStage * sizeof(float) : 0);
        CREATE_TRY(cudaMallocHost((void**)&e->h_block, total));
        std::memset(e->h_block, 0, at_rows);
        e->h_state = reinterpret_cast<SeqState*>(e->h_block + at_state);
        e->h_err = reinterpret_cast<int32_t*>(e->h_state + B);
        e->h_rows = reinterpret_cast<RowDesc*>(e->h_block + at_rows);
        e->h_y = reinterpret_cast<int32_t*>(e->h_block + at_y);
        e->h_ref[0] = reinterpret_cast<int32_t*>(e->h_block + at_r0);
        e->h_ref[1] = reinterpret_cast<int32_t*>(e->h_block + at_r1);
        e->h_logits = reinterpret_cast<float*>(e->h_block + at_logits);
    }
    for (int i = 0; i < 2; ++i) CREATE_TRY(cudaEventCreateWithFlags(&e->ref_ev[i], cudaEventDisableTiming));
    CREATE_TRY(cudaEventCreate(&e->ev0));
    CREATE_TRY(cudaEventCreate(&e->ev1));
    CREATE_TRY(gate_join(&e->gate, dev, e->stream, e->step_simt));
    CREATE_TRY(cudaDeviceSynchronize());
#undef CREATE_TRY
    llma::gemm_count_engine(dev, 1);
    *out = e;
    return LLMA_OK;
}

extern "C" int llma_destroy(llma_engine* e) {
    if (!e) return LLMA_OK;
    cudaStreamSynchronize(e->stream);
    const int dev = e->device;
    free_engine(e);
    llma::gemm_count_engine(dev, -1);
    return LLMA_OK;
}
