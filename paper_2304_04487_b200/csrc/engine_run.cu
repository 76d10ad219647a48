// Decoding entry points of the C ABI: prefill, reference upload, step, generate.
#include <algorithm>
#include <chrono>
#include <climits>
#include <cstring>
#include <vector>

#include "engine.h"

using namespace llma;

// ---- one decoder forward over the rows described by e->rows ---------------------------------
// Every kernel reads the row descriptors from device memory, so the same launch sequence
// serves any mix of rows (greedy, copy steps, prompt chunks) and can be replayed as a graph.
// When profiling is on, an event after every launch lets llma_profile_steps attribute the
// stream time between consecutive events to the kernel class just launched.
static inline void mark(llma_engine* e, int cls) {
    if (!e->prof_on) return;
    if (e->prof_n >= e->prof_ev.size()) {
        cudaEvent_t ev = nullptr;
        if (cudaEventCreate(&ev) != cudaSuccess) { e->prof_on = false; return; }
        e->prof_ev.push_back(ev);
        e->prof_cls.push_back(cls);
    }
    e->prof_cls[e->prof_n] = cls;
    cudaEventRecord(e->prof_ev[e->prof_n++], e->stream);
}

static GemmArgs gemm_args(llma_engine* e, int mode, int n_out, int n_tiles, int k_in, int tiles_per_map) {
    GemmArgs a;
    std::memset(&a, 0, sizeof(a));
    a.mode = mode; a.n_out = n_out; a.n_tiles = n_tiles; a.chunks = k_in / 64; a.tiles_per_map = tiles_per_map;
    a.rows = e->rows; a.dev_err = e->dev_err;
    a.rc = e->row_cap; a.nr = e->decode_nr;
    a.flags = e->gemm_flags; a.launch_seq = e->launch_seq++;
    a.stamps = e->stamps; a.launch_id = a.launch_seq % kStampLaunches;
    a.ws = e->decode_wide ? e->gemm_ws_wide : e->gemm_ws;
    a.dims = e->dims;
    return a;
}

static void run_gemm(llma_engine* e, GemmArgs& a, const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& a2,
                     const void* act, const CUtensorMap* act_map) {
    a.act = act;
    const int grid = gemm_grid_for((int64_t)a.n_tiles * a.chunks, e->num_sms);
    if (e->decode_wide) launch_gemm_wide(e->stream, grid, true, a, a0, a1, a2, act_map);
    else launch_gemm_tcgen05(e->stream, grid, true, a, a0, a1, a2);
}

// Tensor-core path (bf16): 5 kernels per layer.  Every projection is fused with what follows
// it, and the RMSNorms are folded into the projections around them: the producer of the
// residual stream emits split(x * gain) and per-tile sums of squares, the consumer scales its
// accumulators by rsqrt(mean square + eps).
static void with_norm(llma_engine* e, GemmArgs& a) {
    a.ss_in = e->norm_ss; a.ss_tiles = (e->dims.d_model + 127) / 128;
    a.norm_inv = 1.f / (float)e->dims.d_model; a.norm_eps = e->dims.rms_eps;
}

static void enqueue_forward_tc(llma_engine* e) {
    const ModelDims& d = e->dims;
    cudaStream_t st = e->stream;
    const int HD = d.hd_total, F = d.d_ffn, D = d.d_model;
    const llma_engine::ActMaps* am = e->decode_wide ? &e->act_decode : nullptr;
    for (int l = 0; l < d.n_layers; ++l) {
        const llma_engine::LayerMaps& m = e->decode_wide ? e->maps[l] : e->maps2[l];
        GemmArgs q = gemm_args(e, kGemmQKV, HD, 3 * HD / 128, D, HD / 128);
        with_norm(e, q);
        q.out_f32 = e->qkv; q.ld = 3 * HD; q.layer = l; q.rope_cos = e->rope_cos; q.rope_sin = e->rope_sin;
        q.kcache = (__nv_bfloat16*)e->kcache; q.vcache = (__nv_bfloat16*)e->vcache;
        run_gemm(e, q, m.wq, m.wk, m.wv, e->x_hat, am ? am->x_hat : nullptr);
        mark(e, LLMA_K_GEMM_QKV);
        AttnArgs at;
        at.dims = d; at.layer = l; at.rows = e->rows; at.qkv = e->qkv;
        at.tiles = e->attn_tiles;
        at.chunk_pos = kAttnChunk * at.tiles;
        at.n_chunks = (d.max_seq + at.chunk_pos - 1) / at.chunk_pos;
        at.n_rows = e->cur_rows;
        at.attn_out = e->attn; at.ws_o = e->attn_ws_o; at.ws_ml = e->attn_ws_ml;
        at.dev_err = e->dev_err;
        at.stamps = e->stamps;
        at.seq_state = e->seq_state;
        launch_attention_mma(st, at, e->map_kcache, e->map_vcache);
        mark(e, LLMA_K_ATTN);
        GemmArgs o = gemm_args(e, kGemmResid, D, (D + 127) / 128, HD, (D + 127) / 128);
        o.out_f32 = e->x; o.ld = D; o.gain_next = e->ffn_norm[l]; o.xs_out = e->x_hat; o.ss_out = e->norm_ss;
        run_gemm(e, o, m.wo, m.wo, m.wo, e->attn, am ? am->attn : nullptr);
        mark(e, LLMA_K_GEMM_O);
        GemmArgs gu = gemm_args(e, kGemmSwiGLU, F, (F + 63) / 64, D, (F + 63) / 64);
        with_norm(e, gu);
        gu.out_act = e->h;
        if (e->decode_wide) {
            run_gemm(e, gu, m.w_gate, m.w_up, m.w_up, e->x_hat, am->x_hat);
        } else {  // one view over both matrices; whichever lies lower in memory fills the tile's first 64 rows
            gu.gate_second = e->gate_up_map[l].gate_second;
            run_gemm(e, gu, e->gate_up_map[l].map, e->gate_up_map[l].map, e->gate_up_map[l].map, e->x_hat, nullptr);
        }
        mark(e, LLMA_K_GEMM_GATEUP);
        GemmArgs dn = gemm_args(e, kGemmResid, D, (D + 127) / 128, F, (D + 127) / 128);
        dn.out_f32 = e->x; dn.ld = D; dn.xs_out = e->x_hat; dn.ss_out = e->norm_ss;
        dn.gain_next = l + 1 < d.n_layers ? e->attn_norm[l + 1] : e->final_norm;
        run_gemm(e, dn, m.w_down, m.w_down, m.w_down, e->h, am ? am->h : nullptr);
        mark(e, LLMA_K_GEMM_DOWN);
        e->launch_counter += 6;
    }
    const int vt = (d.vocab + 127) / 128;
    GemmArgs lm = gemm_args(e, kGemmLmHead, d.vocab, vt, D, vt);
    with_norm(e, lm);
    lm.out_f32 = e->cfg.keep_logits ? e->logits : nullptr; lm.ld = d.vocab;
    lm.part_max = e->part_max; lm.part_idx = e->part_idx;
    const CUtensorMap& lmm = e->decode_wide ? e->map_lm_head : e->map_lm_head2;
    run_gemm(e, lm, lmm, lmm, lmm, e->x_hat, am ? am->x_hat : nullptr);
    mark(e, LLMA_K_GEMM_LMHEAD);
    e->launch_counter += 1;
}

// most rows that a CUDA-core projection can meet in a decoding step or a prompt pass
static int row_bound(const llma_engine* e, bool decode) { return decode ? e->dims.max_batch * e->dims.kp1 : e->prefill_rows; }

static void enqueue_forward(llma_engine* e, bool lm_head) {
    if (e->gemm_impl == LLMA_GEMM_TCGEN05) { enqueue_forward_tc(e); return; }  // decoding steps only

    // CUDA-core path: 5 kernels per layer, norms folded into the projections that read the residual stream
    const ModelDims& d = e->dims;
    cudaStream_t st = e->stream;
    const bool b = e->bf16;
    const int HD = d.hd_total, F = d.d_ffn, D = d.d_model;
    const int bound = row_bound(e, lm_head);
    auto args = [&](int mode, const void* w0, const void* w1, const void* w2, const float* act, const float* gain, int n_units,
                    int n_out, int k_in, float* out, int ld) {
        RowGemm g;
        std::memset(&g, 0, sizeof(g));
        g.mode = mode; g.rows = e->rows; g.w0 = w0; g.w1 = w1; g.w2 = w2; g.act = act; g.gain = gain; g.eps = d.rms_eps;
        g.n_units = n_units; g.n_out = n_out; g.k_in = k_in; g.out = out; g.ld = ld; g.dims = d;
        return g;
    };
    float *attn = (float*)e->attn, *h = (float*)e->h;
    for (int l = 0; l < d.n_layers; ++l) {
        RowGemm q = args(kRowQKV, e->wq[l], e->wk[l], e->wv[l], e->x, e->attn_norm[l], 3 * HD / 2, 3 * HD, D, e->qkv, 3 * HD);
        q.layer = l; q.rope_cos = e->rope_cos; q.rope_sin = e->rope_sin; q.kcache = e->kcache; q.vcache = e->vcache;
        launch_rowgemm(st, b, q, bound, e->num_sms);
        mark(e, LLMA_K_GEMM_QKV);
        if (!lm_head && l == d.n_layers - 1) break;  // a prompt pass leaves nothing but its K/V rows
        launch_attention_simt(st, b, d, l, lm_head ? d.max_batch * d.kp1 : e->cur_rows, e->rows, e->qkv, e->kcache, e->vcache, attn);
        mark(e, LLMA_K_ATTN);
        launch_rowgemm(st, b, args(kRowResid, e->wo[l], nullptr, nullptr, attn, nullptr, (D + 1) / 2, D, HD, e->x, D), bound, e->num_sms);
        mark(e, LLMA_K_GEMM_O);
        launch_rowgemm(st, b, args(kRowSwiGLU, e->w_gate[l], e->w_up[l], nullptr, e->x, e->ffn_norm[l], F, F, D, h, F), bound, e->num_sms);
        mark(e, LLMA_K_GEMM_GATEUP);
        launch_rowgemm(st, b, args(kRowResid, e->w_down[l], nullptr, nullptr, h, nullptr, (D + 1) / 2, D, F, e->x, D), bound, e->num_sms);
        mark(e, LLMA_K_GEMM_DOWN);
        e->launch_counter += 5;
    }
    if (lm_head) {
        RowGemm g = args(kRowHead, e->lm_head, nullptr, nullptr, e->x, e->final_norm, (d.vocab + 1) / 2, d.vocab, D,
                         e->cfg.keep_logits ? e->logits : nullptr, d.vocab);
        g.part_max = e->part_max; g.part_idx = e->part_idx;
        launch_rowgemm(st, b, g, bound, e->num_sms);
        mark(e, LLMA_K_GEMM_LMHEAD);
        e->launch_counter += 1;
    }
}

static void enqueue_embed(llma_engine* e) {
    if (e->gemm_impl == LLMA_GEMM_TCGEN05)
        launch_embed_norm(e->stream, e->dims, e->cur_rows, e->rows, e->tok_emb, e->attn_norm[0], e->x, e->x_hat,
                          e->norm_ss, e->dev_err);
    else
        launch_embed(e->stream, e->dims, e->bf16, e->cur_rows, e->rows, e->tok_emb, e->x, e->dev_err);
}

// the integer kernel between forward passes: acceptance + K/V commit of the pass that has finished,
// trigger search + copy + row packing for the one that follows
static TailArgs tail_args(const llma_engine* e, int n, int k) {
    TailArgs t;
    std::memset(&t, 0, sizeof(t));
    t.dims = e->dims; t.st = e->seq_state; t.rows = e->rows; t.ref = e->ref; t.y = e->y; t.y_cap = e->y_cap; t.n = n; t.k = k;
    t.part_max = e->part_max; t.part_idx = e->part_idx;
    t.n_tiles = e->gemm_impl == LLMA_GEMM_TCGEN05 ? (e->dims.vocab + 127) / 128
                                                  : rowgemm_grid((e->dims.vocab + 1) / 2, e->dims.d_model, row_bound(e, true), e->num_sms);
    t.out_tok = e->out_tok; t.n_rows = e->decode_rows;
    t.trace = e->trace; t.target = e->target; t.trace_cap = e->trace_cap;
    t.dev_err = e->dev_err;
    return t;
}

static void enqueue_tail(llma_engine* e, int n, int k, bool accept, bool plan) {
    TailArgs t = tail_args(e, n, k);
    t.do_accept = accept ? 1 : 0; t.do_plan = plan ? 1 : 0;
    launch_step_tail(e->stream, t);
    mark(e, accept ? LLMA_K_ACCEPT : LLMA_K_PLAN);
    e->launch_counter += 1;
}

// One decoding step after its plan: embedding gather -> forward -> accept + K/V commit, and (inside
// llma_generate's graph) the plan of the next step in the same launch.
static void enqueue_step_body(llma_engine* e, int n, int k, bool plan_next) {
    e->cur_rows = e->decode_rows;
    e->plain_acts = false;
    e->launch_seq = 0;
    enqueue_embed(e);
    mark(e, LLMA_K_EMBED);
    e->launch_counter += 1;
    enqueue_forward(e, true);
    enqueue_tail(e, n, k, true, plan_next);
}

// Up to `steps` decoding steps as launches of the whole-step kernel on `ctas` SMs (fewer if no sequence has anything left to do), each with
// its plan
static int enqueue_whole_steps(llma_engine* e, int n, int k, int steps, int ctas) {
    SimtStep s = e->simt;
    e->plain_acts = true;
    s.tail = tail_args(e, n, k);
    s.patience = (int)std::min<int64_t>(1 << 22, (int64_t)s.patience * e->num_sms / ctas);
    const uint32_t per_step = simt_epochs(e->dims);
    for (; steps > 0; steps -= kStepsPerLaunch) {
        s.max_steps = std::min(steps, kStepsPerLaunch);
        if (e->ll_epoch > 0xFFFFFFFFu - per_step * (kStepsPerLaunch + 2)) {  // the numbers begin again
            CU_TRY(cudaMemsetAsync(e->ll_words, 0, e->ll_count * sizeof(unsigned long long), e->stream));
            e->ll_epoch = 1;
        }
        s.epoch = e->ll_epoch;
        e->ll_epoch += per_step * (uint32_t)s.max_steps;
        CU_TRY(launch_step_simt(e->stream, e->bf16, s, e->simt_smem, ctas));
        e->launch_counter += 1;
    }
    return LLMA_OK;
}

// The state on its way to and from the device.  Every call that launches kernels brings the mirror up to date, uploads
// it if it has changed, and reads it back (with the error word behind it) before it returns.
int llma::sync_state(llma_engine* e) {
    if (!e->state_stale) return LLMA_OK;
    CU_TRY(cudaMemcpyAsync(e->h_state, e->seq_state, e->dims.max_batch * sizeof(SeqState), cudaMemcpyDeviceToHost, e->stream));
    CU_TRY(cudaStreamSynchronize(e->stream));
    e->state_stale = false;
    e->state_dirty = false;
    return LLMA_OK;
}

static int push_state(llma_engine* e) {  // the caller waits for the stream before it changes the mirror again
    if (e->state_dirty)
        CU_TRY(cudaMemcpyAsync(e->seq_state, e->h_state, e->dims.max_batch * sizeof(SeqState), cudaMemcpyHostToDevice, e->stream));
    e->state_dirty = false;
    e->state_stale = true;  // until pull_state has seen what the kernels made of it
    return LLMA_OK;
}

static int pull_state(llma_engine* e) {
    CU_TRY(cudaMemcpyAsync(e->h_state, e->seq_state, e->dims.max_batch * sizeof(SeqState) + sizeof(int32_t),
                           cudaMemcpyDeviceToHost, e->stream));
    CU_TRY(cudaStreamSynchronize(e->stream));
    e->state_stale = false;
    return LLMA_OK;
}

// Tokens y0 .. y1 - 1 of every sequence, on their way to h_y (same columns)
static int copy_tokens(llma_engine* e, int y0, int y1) {
    if (y1 <= y0) return LLMA_OK;
    const size_t pitch = (size_t)e->y_cap * sizeof(int32_t);
    CU_TRY(cudaMemcpy2DAsync(e->h_y + y0, pitch, e->y + y0, pitch, (size_t)(y1 - y0) * sizeof(int32_t), (size_t)e->dims.max_batch,
                             cudaMemcpyDeviceToHost, e->stream));
    return LLMA_OK;
}

// Reports the error word that pull_state brought, and clears it on the device.
static int check_device_error(llma_engine* e) {
    const int32_t code = *e->h_err;
    if (code == kDevErrNone) return LLMA_OK;
    CU_TRY(cudaMemsetAsync(e->dev_err, 0, sizeof(int32_t), e->stream));
    // a kernel that gave up may have left partial tiles in the hand-over slots: empty them again, so that
    // a caller who carries on after the error does not sum stale partials into later projections
    if (code == kDevErrTimeout && e->gemm_ws) CU_TRY(cudaMemsetAsync(e->gemm_ws, 0xFF, e->gemm_ws_bytes, e->stream));
    if (e->grid_barrier) CU_TRY(cudaMemsetAsync(e->grid_barrier, 0, sizeof(uint32_t), e->stream));
    CU_TRY(cudaStreamSynchronize(e->stream));
    *e->h_err = kDevErrNone;
    if (code == kDevErrTimeout || code == kDevErrSteps) return LLMA_ERR_DEVICE_TIMEOUT;
    if (code == kDevErrCapacity) return LLMA_ERR_CAPACITY;
    return LLMA_ERR_TOKEN_RANGE;
}

// After pull_state: whether launches of whole steps have given up and are to be repeated.  They do when something else keeps SMs from
// their CTAs for long; the state is then that after the last step that was whole, and the words and rows of the unfinished one
// are written again.  For half a minute at most, after which the error is reported.
static int whole_steps_again(llma_engine* e, std::chrono::steady_clock::time_point* since, bool* again) {
    *again = false;
    if (*e->h_err != kDevErrSteps) return LLMA_OK;
    const auto now = std::chrono::steady_clock::now();
    if (since->time_since_epoch().count() == 0) *since = now;
    if (now - *since > std::chrono::seconds(30)) return LLMA_OK;
    CU_TRY(cudaMemsetAsync(e->dev_err, 0, sizeof(int32_t), e->stream));
    CU_TRY(cudaMemsetAsync(e->grid_barrier, 0, sizeof(uint32_t), e->stream));
    *e->h_err = kDevErrNone;
    *again = true;
    return LLMA_OK;
}

// Positions p0 .. p0 + n - 1 of a prompt (tokens in e->p_tok) through the decoder, into the K/V cache.  Nothing but the cache
// outlives the pass, so the last layer ends with its K/V rows.
static int enqueue_prompt_pass(llma_engine* e, int seq, int p0, int n) {
    const ModelDims& d = e->dims;
    cudaStream_t st = e->stream;
    const int HD = d.hd_total, F = d.d_ffn, D = d.d_model;
    auto args = [&](int mode, int n_out, int n_tiles, int k_in, int tiles_per_map, const void* act) {
        GemmArgs a;
        std::memset(&a, 0, sizeof(a));
        a.mode = mode; a.n_out = n_out; a.n_tiles = n_tiles; a.chunks = k_in / 64; a.tiles_per_map = tiles_per_map;
        a.act = act; a.rc = e->prompt_rc; a.dev_err = e->dev_err; a.dims = d; a.pos0 = p0; a.seq0 = seq;
        return a;
    };
    auto norm_in = [&](GemmArgs& a) { a.ss_in = e->p_ss; a.ss_tiles = D / 128; a.norm_inv = 1.f / (float)D; a.norm_eps = d.rms_eps; };
    launch_embed_prompt(st, d, n, e->prompt_rc, e->p_tok + p0, e->tok_emb, e->attn_norm[0], e->p_x, e->p_x_hat, e->p_ss);
    int bad = 0;
    for (int l = 0; l < d.n_layers && !bad; ++l) {
        const llma_engine::LayerMaps& m = e->maps[l];
        GemmArgs q = args(kGemmQKV, HD, 3 * HD / 128, D, HD / 128, e->p_x_hat);
        norm_in(q);
        q.out_f32 = e->p_q; q.ld = HD; q.layer = l; q.rope_cos = e->rope_cos; q.rope_sin = e->rope_sin;
        q.kcache = (__nv_bfloat16*)e->kcache; q.vcache = (__nv_bfloat16*)e->vcache;
        bad |= launch_gemm_prompt(st, q, n, e->prompt_pairs, m.wq, m.wk, m.wv);
        if (l == d.n_layers - 1) break;
        PromptAttnArgs at;
        at.dims = d; at.layer = l; at.seq = seq; at.pos0 = p0; at.n_rows = n; at.q = e->p_q; at.attn_out = e->p_attn;
        at.rc = e->prompt_rc; at.dev_err = e->dev_err;
        launch_attention_prompt(st, at, e->map_kcache_64, e->map_vcache_64);
        GemmArgs o = args(kGemmResid, D, D / 128, HD, D / 128, e->p_attn);
        o.out_f32 = e->p_x; o.ld = D; o.gain_next = e->ffn_norm[l]; o.xs_out = e->p_x_hat; o.ss_out = e->p_ss;
        bad |= launch_gemm_prompt(st, o, n, e->prompt_pairs, m.wo, m.wo, m.wo);
        GemmArgs gu = args(kGemmSwiGLU, F, F / 64, D, F / 64, e->p_x_hat);
        norm_in(gu);
        gu.out_act = e->p_h;
        bad |= launch_gemm_prompt(st, gu, n, e->prompt_pairs, m.w_gate, m.w_up, m.w_up);
        GemmArgs dn = args(kGemmResid, D, D / 128, F, D / 128, e->p_h);
        dn.out_f32 = e->p_x; dn.ld = D; dn.gain_next = e->attn_norm[l + 1]; dn.xs_out = e->p_x_hat; dn.ss_out = e->p_ss;
        bad |= launch_gemm_prompt(st, dn, n, e->prompt_pairs, m.w_down, m.w_down, m.w_down);
    }
    return bad ? LLMA_ERR_CONFIG : LLMA_OK;
}

// Tokens 0 .. n_cache - 1 of a prompt on their way through the decoder, into the K/V cache
static int enqueue_prompt(llma_engine* e, int seq, const int32_t* prompt, int n_cache) {
    if (e->gemm_impl == LLMA_GEMM_TCGEN05) {
        if (n_cache == 0) return LLMA_OK;
        // passes of equal length
        std::memcpy(e->h_y, prompt, (size_t)n_cache * sizeof(int32_t));
        CU_TRY(cudaMemcpyAsync(e->p_tok, e->h_y, (size_t)n_cache * sizeof(int32_t), cudaMemcpyHostToDevice, e->stream));
        const int passes = (n_cache + e->prompt_rc - 1) / e->prompt_rc;
        const int each = std::min(e->prompt_rc, ((n_cache + passes - 1) / passes + 31) / 32 * 32);
        for (int p0 = 0; p0 < n_cache; p0 += each) {
            const int rc = enqueue_prompt_pass(e, seq, p0, std::min(each, n_cache - p0));
            if (rc) return rc;
        }
        CU_TRY(cudaGetLastError());
        return LLMA_OK;
    }
    e->cur_rows = e->prefill_rows;
    for (int p0 = 0; p0 < n_cache; p0 += e->prefill_rows) {
        const int cnt = std::min(e->prefill_rows, n_cache - p0);
        RowDesc* R = e->h_rows;
        for (int r = 0; r < kRowCap; ++r) {
            R->tok[r] = r < cnt ? prompt[p0 + r] : 0;
            R->pos[r] = r < cnt ? p0 + r : -1;
            R->seq[r] = seq;
        }
        for (int s2 = 0; s2 < kSeqCap; ++s2) { R->seq_first[s2] = 0; R->seq_cnt[s2] = 0; R->seq_maxpos[s2] = -1; }
        R->seq_first[seq] = 0; R->seq_cnt[seq] = cnt; R->seq_maxpos[seq] = p0 + cnt - 1;
        R->rows_used = cnt;
        R->max_pos = p0 + cnt - 1;
        CU_TRY(cudaMemcpyAsync(e->rows, R, sizeof(RowDesc), cudaMemcpyHostToDevice, e->stream));
        enqueue_embed(e);
        enqueue_forward(e, false);
        CU_TRY(cudaGetLastError());
        CU_TRY(cudaStreamSynchronize(e->stream));  // h_rows is reused by the next chunk
    }
    return LLMA_OK;
}

extern "C" int llma_prefill(llma_engine* e, int32_t seq, const int32_t* prompt, int32_t n_prompt) {
    if (!e || !prompt) return LLMA_ERR_NULL;
    const ModelDims& d = e->dims;
    if (seq < 0 || seq >= d.max_batch) return LLMA_ERR_CAPACITY;
    if (n_prompt < 1) return LLMA_ERR_ARG;
    if (n_prompt > d.max_seq) return LLMA_ERR_CAPACITY;
    for (int i = 0; i < n_prompt; ++i)
        if (prompt[i] < 0 || prompt[i] >= d.vocab) return LLMA_ERR_TOKEN_RANGE;
    int rc = sync_state(e);
    if (rc) return rc;
    // push prompt[0 .. P-2] through the decoder
    rc = enqueue_prompt(e, seq, prompt, n_prompt - 1);
    if (rc) {
        cudaStreamSynchronize(e->stream);  // copies out of the staging memory may be under way: the next call writes to it
        return rc;
    }
    SeqState& S = e->h_state[seq];
    const int32_t keep_ref = S.ref_len;
    std::memset(&S, 0, sizeof(S));
    S.active = 1; S.kv_len = n_prompt - 1; S.pending = prompt[n_prompt - 1]; S.ref_len = keep_ref;
    S.prompt_len = n_prompt; S.pos = -1; S.last_pos = -1; S.target_len = 0; S.done = 1;
    e->state_dirty = true;
    e->prompt_last[seq] = prompt[n_prompt - 1];
    e->last_step_valid = false;
    CU_TRY(cudaMemcpyAsync(e->h_err, e->dev_err, sizeof(int32_t), cudaMemcpyDeviceToHost, e->stream));
    CU_TRY(cudaStreamSynchronize(e->stream));
    return check_device_error(e);
}

extern "C" int llma_set_reference(llma_engine* e, int32_t seq, const int32_t* tokens, int32_t n_tokens,
                                  const int32_t* doc_offsets, int32_t n_docs) {
    if (!e) return LLMA_ERR_NULL;
    const ModelDims& d = e->dims;
    if (seq < 0 || seq >= d.max_batch) return LLMA_ERR_CAPACITY;
    if (n_tokens < 0) return LLMA_ERR_ARG;
    if (n_tokens > 0 && !tokens) return LLMA_ERR_NULL;
    if (n_tokens > e->cfg.max_ref) return LLMA_ERR_REF_TOO_LONG;
    if (doc_offsets) {
        if (n_docs < 1 || doc_offsets[0] != 0 || doc_offsets[n_docs] != n_tokens) return LLMA_ERR_REF_TOO_LONG;
        for (int j = 0; j < n_docs; ++j)
            if (doc_offsets[j + 1] < doc_offsets[j]) return LLMA_ERR_REF_TOO_LONG;
    }
    for (int i = 0; i < n_tokens; ++i)
        if (tokens[i] < 0 || tokens[i] >= d.vocab) return LLMA_ERR_TOKEN_RANGE;
    const int rc = sync_state(e);
    if (rc) return rc;
    if (n_tokens > 0) {
        // tokens, document starts and document ends leave in one copy from page-locked memory; two buffers in turn,
        // so that a call waits for the copy before the last one at most
        const int t = e->ref_turn;
        e->ref_turn ^= 1;
        CU_TRY(cudaEventSynchronize(e->ref_ev[t]));
        int32_t *st = e->h_ref[t], *ds = st + n_tokens, *de = ds + n_tokens;
        std::memcpy(st, tokens, (size_t)n_tokens * sizeof(int32_t));
        if (doc_offsets) {
            for (int j = 0; j < n_docs; ++j)
                for (int i = doc_offsets[j]; i < doc_offsets[j + 1]; ++i) { ds[i] = doc_offsets[j]; de[i] = doc_offsets[j + 1]; }
        } else {
            for (int i = 0; i < n_tokens; ++i) { ds[i] = 0; de[i] = n_tokens; }
        }
        const size_t nb = (size_t)n_tokens * sizeof(int32_t);
        CU_TRY(cudaMemcpy2DAsync(e->ref + (size_t)seq * 3 * d.max_ref, (size_t)d.max_ref * sizeof(int32_t), st, nb, nb, 3,
                                 cudaMemcpyHostToDevice, e->stream));
        CU_TRY(cudaEventRecord(e->ref_ev[t], e->stream));
    }
    e->h_state[seq].ref_len = n_tokens;
    e->state_dirty = true;
    return LLMA_OK;
}

static int check_nk(const llma_engine* e, int n, int k) {
    if (n < 1 || k < 0 || k > e->cfg.max_k) return LLMA_ERR_ARG;
    return LLMA_OK;
}

// The entry of (n, k), made (with no graph yet) if there is none
static llma_engine::StepGraph& graph_entry(llma_engine* e, llma_engine::StepGraphs& graphs, int n, int k) {
    auto it = graphs.find({n, k});
    if (it == graphs.end()) {
        if (graphs.size() >= kStepGraphs) {  // nothing runs between calls: a graph can go at once
            auto old = graphs.begin();
            for (auto g = graphs.begin(); g != graphs.end(); ++g)
                if (g->second.used < old->second.used) old = g;
            if (old->second.exec) cudaGraphExecDestroy(old->second.exec);
            graphs.erase(old);
        }
        it = graphs.insert({{n, k}, {nullptr, 0, 0}}).first;
    }
    it->second.used = ++e->graph_clock;
    return it->second;
}

template <typename Enqueue>
static int capture(llma_engine* e, cudaGraphExec_t* out, Enqueue enqueue) {
    cudaGraph_t g = nullptr;
    const int64_t before = e->launch_counter;
    CU_TRY(cudaStreamBeginCapture(e->stream, cudaStreamCaptureModeThreadLocal));
    enqueue();
    cudaError_t ce = cudaStreamEndCapture(e->stream, &g);
    e->launch_counter = before;
    CU_TRY(ce);
    ce = cudaGraphInstantiate(out, g, 0);
    cudaGraphDestroy(g);
    if (ce != cudaSuccess) *out = nullptr;
    CU_TRY(ce);
    return LLMA_OK;
}

// How this engine's decoding steps wait inside a launch (device_gate.h)
static int turn_kind(const llma_engine* e, bool whole) {
    return whole ? kTurnSteps : (e->gemm_impl == LLMA_GEMM_TCGEN05 ? kTurnTiles : kTurnNone);
}

static int enqueue_lone_step(llma_engine* e, int n, int k, int ctas) {  // plan, forward pass, acceptance
    if (e->step_simt) return enqueue_whole_steps(e, n, k, 1, ctas);
    auto enqueue = [&] { enqueue_tail(e, n, k, false, true); enqueue_step_body(e, n, k, false); };
    llma_engine::StepGraph& g = graph_entry(e, e->lone_graphs, n, k);
    if (!e->can_capture || g.uses + 1 < kCaptureAt) {
        ++g.uses;
        enqueue();
        CU_TRY(cudaGetLastError());
        return LLMA_OK;
    }
    if (!g.exec) {
        const int rc = capture(e, &g.exec, enqueue);
        if (rc) return rc;
    }
    CU_TRY(cudaGraphLaunch(g.exec, e->stream));
    return LLMA_OK;
}

extern "C" int llma_step(llma_engine* e, int32_t n, int32_t k, int32_t* out_tokens, int32_t* n_out) {
    if (!e || !out_tokens || !n_out) return LLMA_ERR_NULL;
    int rc = check_nk(e, n, k);
    if (rc) return rc;
    const ModelDims& d = e->dims;
    rc = sync_state(e);
    if (rc) return rc;
    bool any = false;
    std::vector<int32_t> y0((size_t)d.max_batch, 0);
    int y_lo = INT_MAX, y_hi = 0;
    for (int s = 0; s < d.max_batch; ++s) {
        SeqState& S = e->h_state[s];
        y0[s] = S.y_len;
        if (!S.active) continue;
        if (S.kv_len + 1 > d.max_seq || S.y_len + 1 > e->y_cap) return LLMA_ERR_CAPACITY;
        any = true;
        y_lo = std::min(y_lo, S.y_len);
        y_hi = std::max(y_hi, std::min(e->y_cap, S.y_len + k + 1));
    }
    if (!any) return LLMA_ERR_STATE;
    for (int s = 0; s < d.max_batch; ++s) {
        SeqState& S = e->h_state[s];
        if (!S.active) continue;
        // a lone step has no output budget of its own: only the capacities bound the copy
        const int32_t target = std::min(e->y_cap, S.y_len + (d.max_seq - S.kv_len));
        if (S.target_len != target || S.done) { S.target_len = target; S.done = 0; e->state_dirty = true; }
    }
    GateCall call(e->gate);
    rc = push_state(e);
    if (rc) return rc;
    std::chrono::steady_clock::time_point gave_up{};
    for (bool again = true; again;) {
        GateTurn turn(e->gate, turn_kind(e, e->step_simt), e->num_sms);
        CU_TRY(turn.error());
        rc = enqueue_lone_step(e, n, k, turn.ctas());
        if (rc) return rc;
        CU_TRY(turn.end());
        // the tokens a step can have emitted come back with the state
        rc = copy_tokens(e, y_lo, y_hi);
        if (rc) return rc;
        rc = pull_state(e);
        if (rc) return rc;
        again = false;
        if (e->step_simt) {
            rc = whole_steps_again(e, &gave_up, &again);
            if (rc) return rc;
            for (int s = 0; s < d.max_batch; ++s) again = again && e->h_state[s].y_len == y0[s];  // (the step itself may have been whole)
        }
    }
    rc = check_device_error(e);
    if (rc) return rc;
    for (int s = 0; s < d.max_batch; ++s) {
        const SeqState& S = e->h_state[s];
        const int m = S.active ? S.y_len - y0[s] : 0;
        n_out[s] = m;
        if (m > 0) std::memcpy(out_tokens + (size_t)s * d.kp1, e->h_y + (size_t)s * e->y_cap + y0[s], (size_t)m * sizeof(int32_t));
    }
    e->last_step_valid = true;
    return LLMA_OK;
}

// A step of llma_generate as a graph, or no graph where the stream cannot be captured
static int get_step_graph(llma_engine* e, int n, int k, cudaGraphExec_t* out) {
    *out = nullptr;
    if (!e->can_capture) return LLMA_OK;
    llma_engine::StepGraph& g = graph_entry(e, e->step_graphs, n, k);
    if (!g.exec) {
        const int rc = capture(e, &g.exec, [&] {
            const int64_t before = e->launch_counter;
            enqueue_step_body(e, n, k, true);
            e->launches_per_step = e->launch_counter - before;
        });
        if (rc) return rc;
    }
    *out = g.exec;
    return LLMA_OK;
}

static int launch_steps(llma_engine* e, cudaGraphExec_t graph, int n, int k, int steps) {
    for (int i = 0; i < steps; ++i) {
        if (graph) {
            CU_TRY(cudaGraphLaunch(graph, e->stream));
        } else {
            const int64_t before = e->launch_counter;
            enqueue_step_body(e, n, k, true);
            e->launches_per_step = e->launch_counter - before;
            e->launch_counter = before;
            CU_TRY(cudaGetLastError());
        }
    }
    return LLMA_OK;
}

extern "C" int llma_generate(llma_engine* e, int32_t max_new, int32_t n, int32_t k, int32_t* out_tokens,
                             int32_t* n_out, llma_stats* stats) {
    if (!e || !out_tokens || !n_out) return LLMA_ERR_NULL;
    int rc = check_nk(e, n, k);
    if (rc) return rc;
    if (max_new < 0) return LLMA_ERR_ARG;
    const ModelDims& d = e->dims;
    rc = sync_state(e);
    if (rc) return rc;
    bool any = false;
    int y_lo = INT_MAX, y_hi = 0;
    std::vector<SeqState> s0(e->h_state, e->h_state + d.max_batch);
    for (int s = 0; s < d.max_batch; ++s) {
        const SeqState& S = s0[s];
        if (!S.active) continue;
        if (S.kv_len + max_new > d.max_seq || S.y_len + max_new > e->y_cap) return LLMA_ERR_CAPACITY;
        any = true;
        y_lo = std::min(y_lo, S.y_len);
        y_hi = std::max(y_hi, S.y_len + max_new);
    }
    if (!any) return LLMA_ERR_STATE;
    for (int s = 0; s < d.max_batch; ++s) {
        SeqState& S = e->h_state[s];
        if (!S.active) continue;
        S.target_len = S.y_len + max_new;
        S.done = max_new == 0;
        e->state_dirty = true;
    }
    const bool whole = e->step_simt;
    GateCall call(e->gate);
    const int kind = turn_kind(e, whole);
    const bool shared = kind != kTurnNone && gate_shared(e->gate);  // few steps at a time: other engines' turns come between
    cudaGraphExec_t graph = nullptr;
    if (!whole) {
        rc = get_step_graph(e, n, k, &graph);
        if (rc) return rc;
    }

    rc = push_state(e);
    if (rc) return rc;

    // Each step emits between 1 and k+1 tokens per sequence, so ceil(left / (k+1)) more steps
    // can never be too many.  Launch that many back to back, look at the counters once, repeat.
    // (A launch of the whole-step kernel ends by itself when there is nothing left to do: twice that many may be asked for.)
    int64_t launches = 0;
    bool have_tokens = false, stepped = false;
    std::chrono::steady_clock::time_point gave_up{};
    CU_TRY(cudaEventRecord(e->ev0, e->stream));
    // the first step's plan; every graph launch then ends with the plan of the step after it
    if (!whole || max_new == 0) {
        const int64_t before = e->launch_counter;
        enqueue_tail(e, n, k, false, true);
        launches += e->launch_counter - before;
        e->launch_counter = before;
    }
    for (;;) {
        int left = 0;
        for (int s = 0; s < d.max_batch; ++s) {
            const SeqState& S = e->h_state[s];
            if (S.active && !S.done) left = std::max(left, S.target_len - S.y_len);
        }
        if (left <= 0) break;
        int batch = (left + k) / (k + 1);
        GateTurn turn(e->gate, kind, e->num_sms);
        CU_TRY(turn.error());
        if (whole) {
            const int64_t before = e->launch_counter;
            const int most = shared ? kStepsPerTurn : std::max(kStepsPerLaunch, 2 * batch);
            rc = enqueue_whole_steps(e, n, k, std::min(left, most), turn.ctas());
            launches += e->launch_counter - before;
            e->launch_counter = before;
        } else {
            if (shared) batch = std::min(batch, kStepsPerTurn);
            rc = launch_steps(e, graph, n, k, batch);
            launches += (int64_t)batch * e->launches_per_step;
        }
        if (rc) return rc;
        CU_TRY(turn.end());
        stepped = true;
        // the last look at the state brings the tokens too (a few kilobytes at most: it may be any look)
        const bool with_tokens = (size_t)(y_hi - y_lo) * d.max_batch <= 16384;
        if (with_tokens) { rc = copy_tokens(e, y_lo, y_hi); if (rc) return rc; }
        CU_TRY(cudaEventRecord(e->ev1, e->stream));
        rc = pull_state(e);
        if (rc) return rc;
        have_tokens = with_tokens;
        if (whole) {
            bool again;
            rc = whole_steps_again(e, &gave_up, &again);
            if (rc) return rc;
        }
        if (*e->h_err != kDevErrNone) break;
    }
    if (!stepped) {  // no step was taken
        CU_TRY(cudaEventRecord(e->ev1, e->stream));
        rc = pull_state(e);
        if (rc) return rc;
    }
    rc = check_device_error(e);
    if (rc) return rc;
    if (!have_tokens) {
        rc = copy_tokens(e, y_lo, y_hi);
        if (rc) return rc;
        CU_TRY(cudaStreamSynchronize(e->stream));
    }

    llma_stats st;
    std::memset(&st, 0, sizeof(st));
    for (int s = 0; s < d.max_batch; ++s) {
        const SeqState& S = e->h_state[s];
        const int m = S.active ? S.y_len - s0[s].y_len : 0;
        n_out[s] = m;
        if (m > 0)
            std::memcpy(out_tokens + (size_t)s * max_new, e->h_y + (size_t)s * e->y_cap + s0[s].y_len, (size_t)m * sizeof(int32_t));
        if (S.active) {
            st.steps += S.steps - s0[s].steps;
            st.trigger_steps += S.trigger_steps - s0[s].trigger_steps;
            st.copied_accepted += S.copied_accepted - s0[s].copied_accepted;
            st.tokens += m;
        }
    }
    st.launches = launches;
    CU_TRY(cudaEventElapsedTime(&st.device_ms, e->ev0, e->ev1));
    if (stats) *stats = st;
    e->last_step_valid = launches > 0;
    return LLMA_OK;
}

// Replay of a given sequence of step shapes (the paper's target-guided measurement, Section 3.2 and
// Algorithm 2): the forward passes are the real ones, the trigger and acceptance decisions come from the trace.
extern "C" int llma_generate_forced(llma_engine* e, int32_t seq, const int32_t* trace, int32_t n_steps,
                                    const int32_t* target, int32_t n_target, llma_stats* stats) {
    if (!e || !trace || !target) return LLMA_ERR_NULL;
    const ModelDims& d = e->dims;
    if (seq < -1 || seq >= d.max_batch) return LLMA_ERR_CAPACITY;
    if (n_steps < 1 || n_target < 1 || n_steps > e->trace_cap) return LLMA_ERR_ARG;
    int64_t total = 0;
    for (int i = 0; i < n_steps; ++i) {
        const int r = trace[2 * i], m = trace[2 * i + 1];
        if (r < 1 || r > d.kp1 || m < 1 || m > r) return LLMA_ERR_ARG;
        total += m;
    }
    if (total != n_target) return LLMA_ERR_ARG;
    for (int i = 0; i < n_target; ++i)
        if (target[i] < 0 || target[i] >= d.vocab) return LLMA_ERR_TOKEN_RANGE;
    int rc = sync_state(e);
    if (rc) return rc;
    // the sequences that replay: the given one, or (seq = -1) every prefilled one; all others must be at rest
    std::vector<int> who;
    for (int s = 0; s < d.max_batch; ++s) {
        const SeqState& S = e->h_state[s];
        if (s == seq || (seq < 0 && S.active)) who.push_back(s);
        else if (S.active && !S.done) return LLMA_ERR_STATE;
    }
    if (who.empty()) return LLMA_ERR_STATE;
    std::vector<SeqState> s0(e->h_state, e->h_state + d.max_batch);
    for (int s : who) {
        if (!s0[s].active) return LLMA_ERR_STATE;
        if (s0[s].kv_len + n_target > d.max_seq || s0[s].y_len + n_target > e->y_cap) return LLMA_ERR_CAPACITY;
    }
    for (int s : who) {
        CU_TRY(cudaMemcpyAsync(e->trace + (size_t)s * e->trace_cap * 2, trace, (size_t)n_steps * 2 * sizeof(int32_t),
                               cudaMemcpyHostToDevice, e->stream));
        CU_TRY(cudaMemcpyAsync(e->target + (size_t)s * e->y_cap + s0[s].y_len, target, (size_t)n_target * sizeof(int32_t),
                               cudaMemcpyHostToDevice, e->stream));
        SeqState& S = e->h_state[s];
        S.target_len = S.y_len + n_target; S.done = 0; S.forced_rows = 1; S.forced_emit = 1; S.trace_step = 0;
        e->state_dirty = true;
    }
    rc = push_state(e);
    if (rc) return rc;
    CU_TRY(cudaStreamSynchronize(e->stream));  // the host arrays may go after this
    const bool whole = e->step_simt;
    GateCall call(e->gate);
    cudaGraphExec_t graph = nullptr;
    if (!whole) {
        rc = get_step_graph(e, 1, 0, &graph);
        if (rc) return rc;
    }
    CU_TRY(cudaEventRecord(e->ev0, e->stream));
    const int64_t before = e->launch_counter;
    const int kind = turn_kind(e, whole);
    const bool shared = kind != kTurnNone && gate_shared(e->gate);
    if (!whole) enqueue_tail(e, 1, 0, false, true);
    int64_t launches = e->launch_counter - before;
    std::chrono::steady_clock::time_point gave_up{};
    for (bool again = true; again;) {
        for (int at = 0; at < n_steps;) {
            const int now = std::min(n_steps - at, shared ? kStepsPerTurn : n_steps);
            if (at > 0) CU_TRY(cudaStreamSynchronize(e->stream));
            GateTurn turn(e->gate, kind, e->num_sms);
            CU_TRY(turn.error());
            e->launch_counter = before;
            if (whole) rc = enqueue_whole_steps(e, 1, 0, now, turn.ctas());
            else rc = launch_steps(e, graph, 1, 0, now);
            if (rc) return rc;
            launches += whole ? e->launch_counter - before : (int64_t)now * e->launches_per_step;
            CU_TRY(turn.end());
            at += now;
        }
        e->launch_counter = before;
        CU_TRY(cudaEventRecord(e->ev1, e->stream));
        rc = pull_state(e);
        if (rc) return rc;
        again = false;
        if (whole) rc = whole_steps_again(e, &gave_up, &again);  // (launches beyond the trace's end find nothing to do)
        if (rc) return rc;
    }
    rc = check_device_error(e);
    if (rc) return rc;
    llma_stats st;
    std::memset(&st, 0, sizeof(st));
    bool complete = true;
    for (int s : who) {
        SeqState& T = e->h_state[s];
        st.steps += T.steps - s0[s].steps; st.trigger_steps += T.trigger_steps - s0[s].trigger_steps;
        st.copied_accepted += T.copied_accepted - s0[s].copied_accepted; st.tokens += T.y_len - s0[s].y_len;
        complete = complete && T.y_len - s0[s].y_len == n_target;
        T.forced_rows = 0; T.forced_emit = 0; T.trace_step = 0;
        e->state_dirty = true;
    }
    st.launches = launches;
    CU_TRY(cudaEventElapsedTime(&st.device_ms, e->ev0, e->ev1));
    if (stats) *stats = st;
    e->last_step_valid = false;
    return complete ? LLMA_OK : LLMA_ERR_STATE;
}

extern "C" int llma_debug_set_device_error(llma_engine* e, int32_t code) {
    if (!e) return LLMA_ERR_NULL;
    if (code < kDevErrNone || code > kDevErrSteps) return LLMA_ERR_ARG;
    CU_TRY(cudaMemcpyAsync(e->dev_err, &code, sizeof(int32_t), cudaMemcpyHostToDevice, e->stream));
    CU_TRY(cudaStreamSynchronize(e->stream));
    return LLMA_OK;
}

extern "C" int llma_profile_steps(llma_engine* e, int32_t n, int32_t k, int32_t steps, llma_profile* out) {
    if (!e || !out) return LLMA_ERR_NULL;
    int rc = check_nk(e, n, k);
    if (rc) return rc;
    if (steps < 1) return LLMA_ERR_ARG;
    std::memset(out, 0, sizeof(*out));
    GateCall call(e->gate);
    for (int i = 0; i < steps; ++i) {
        // same state handling as llma_step, but the launches are bracketed by events
        rc = sync_state(e);
        if (rc) return rc;
        bool any = false;
        for (int s = 0; s < e->dims.max_batch; ++s) {
            SeqState& S = e->h_state[s];
            if (!S.active) continue;
            if (S.kv_len + 1 > e->dims.max_seq) return LLMA_ERR_CAPACITY;
            S.target_len = std::min(e->y_cap, S.y_len + (e->dims.max_seq - S.kv_len));
            S.done = 0;
            e->state_dirty = true;
            any = true;
        }
        if (!any) return LLMA_ERR_STATE;
        rc = push_state(e);
        if (rc) return rc;
        e->prof_on = true;
        e->prof_n = 0;
        GateTurn turn(e->gate, turn_kind(e, false), e->num_sms);
        CU_TRY(turn.error());
        mark(e, -1);
        enqueue_tail(e, n, k, false, true);
        enqueue_step_body(e, n, k, false);
        e->prof_on = false;
        CU_TRY(cudaGetLastError());
        CU_TRY(turn.end());
        rc = pull_state(e);
        if (rc) return rc;
        rc = check_device_error(e);
        if (rc) return rc;
        for (size_t j = 1; j < e->prof_n; ++j) {
            float ms = 0.f;
            CU_TRY(cudaEventElapsedTime(&ms, e->prof_ev[j - 1], e->prof_ev[j]));
            const int c = e->prof_cls[j];
            if (c >= 0 && c < LLMA_K_COUNT) { out->ms[c] += ms; out->launches[c] += 1; }
            out->total_ms += ms;
        }
        out->steps += 1;
    }
    e->last_step_valid = true;
    return LLMA_OK;
}
