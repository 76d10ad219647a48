// The integer work between two forward passes of an LLMA decoding step, as a device function of one CTA: trigger search + copy
// (Section 2.2 of the paper, Algorithm 1's match and copy steps) and acceptance + K/V commit (Algorithm 1's acceptance
// loop).  step_tail_kernel (kernels_int.cu) is this function alone, the whole-step kernels run it in one of their CTAs.
// All results here are exact integer work.
#pragma once
#include "kernels.h"

namespace llma {

// --------------------------------------------------------------------------------------
// step_tail: ONE CTA does the integer work between two forward passes, for all sequences:
//
//   accept (Algorithm 1's acceptance loop, when a forward pass has just finished)
//     final argmax of every row over the LM head's per-tile partials;
//     o_0 is always kept, o_{i+1} is kept while o_i equals the copied token d_{pos+i};
//     the kept outputs are appended to y, kv_len advances past the rows whose inputs were
//     valid (later rows stay in the cache as garbage and are overwritten by later steps),
//     the last kept output becomes the pending input, statistics are updated.
//   plan (Section 2.2: trigger and copy, when a forward pass follows)
//     among reference positions `pos` (inside one document, with at
//     least one token after it) whose preceding n tokens equal the last n generated tokens,
//     pick the one whose agreement with the generated text extends furthest backwards; ties go
//     to the smallest position.  k_eff = min(k, tokens left in the document, tokens still to
//     emit - 1, K/V rows left - 1).  Rows of the step: [pending, ref[pos], ..., ref[pos+k_eff-1]]
//     at positions kv_len .. kv_len+k_eff; the rows of all sequences are packed back to back.
//
// A sequence in replay mode (forced_rows > 0 in its state) skips both decisions: the shapes come
// from a trace and the tokens from a target text (Algorithm 2's use in Section 3.2).
// --------------------------------------------------------------------------------------
constexpr int kStateWords = sizeof(SeqState) / sizeof(int32_t);

struct TailShared {
    SeqState st[kSeqCap];
    int first[kSeqCap + 1];
    int tok[kRowCap];
    unsigned long long best[kSeqCap];
};
// What the work reads and writes.  A CTA that does it step after step has all of it in its shared memory.
struct TailLocal {
    SeqState* st;             // [B]
    int* first;               // [B + 1]: first row of every sequence, rows in use
    int* tok;                 // [rows]: final token of every row
    unsigned long long* best; // [B]
    int* ref;                 // [B][3][max_ref]
    int* y;                   // [B][y_cap]
};

// The work on what `v` points to.  kLocal: all of it in shared memory, kept from step to step, with the rows' final tokens in v.tok
// already (the caller's threads have met at a barrier since); otherwise states and first rows are on their way to
// shared memory and v.ref and v.y lie in global memory.
// emit(row, token, position, sequence, first row of the sequence) hands a row of the next step over, emit_count their number.
// All kTailThreads threads of the CTA call it; it begins and ends without a barrier.
template <int kTailThreads, bool kLocal, typename Emit, typename EmitCount>
__device__ __forceinline__ void step_tail_on(const TailArgs& a, const TailLocal& v, Emit emit, EmitCount emit_count) {
    const ModelDims& dims = a.dims;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int n_warps = kTailThreads / 32;
    const int B = dims.max_batch;
    SeqState* const s_st = v.st;
    int* const s_first = v.first;
    int* const s_tok = v.tok;
    unsigned long long* const s_best = v.best;
    auto ld_ref = [](const int* p) { return kLocal ? *p : __ldg(p); };  // references do not change
    auto ld_y = [](const int* p) { return kLocal ? *p : __ldcg(p); };
#pragma unroll 1
    for (int s = threadIdx.x; s < B; s += kTailThreads) s_best[s] = 0ull;
    if (a.do_accept) {
        // ---- final token of every row slot a decoding step can use (lowest index on ties) --------------------
        const int n_slots = kLocal ? 0 : a.n_rows;
#pragma unroll 1
        for (int r = warp; r < n_slots; r += n_warps) {
            float bv = -INFINITY; int bi = 0x7fffffff;
#pragma unroll 1
            for (int t0 = 0; t0 < a.n_tiles; t0 += 32 * 8) {  // eight loads of each array in flight per lane
                float v[8]; int ix[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int t = t0 + u * 32 + lane;
                    v[u] = t < a.n_tiles ? __ldcg(&a.part_max[(int64_t)t * dims.row_cap + r]) : -INFINITY;
                    ix[u] = t < a.n_tiles ? __ldcg(&a.part_idx[(int64_t)t * dims.row_cap + r]) : 0x7fffffff;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (v[u] > bv || (v[u] == bv && ix[u] < bi)) { bv = v[u]; bi = ix[u]; }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
            }
            if (lane == 0) { s_tok[r] = bi; a.out_tok[r] = bi; }
        }
        __syncthreads();
        // ---- acceptance + commit, one warp per sequence -------------------------------------------------------
#pragma unroll 1
        for (int s = warp; s < B; s += n_warps) {
            SeqState& S = s_st[s];
            const int nrows = S.nrows;
            if (nrows <= 0) {
                if (lane == 0) { S.last_pos = -1; S.last_k_eff = 0; S.last_accepted = 0; S.last_emitted = 0; }
                continue;
            }
            const int* rs = v.ref + (int64_t)s * 3 * dims.max_ref;
            const int* o = s_tok + s_first[s];
            int* ys = v.y + (int64_t)s * a.y_cap;
            int* yg = a.y + (int64_t)s * a.y_cap;
            const int k_eff = S.k_eff, pos = S.pos, ylen = S.y_len;
            int m, done = 0, pending;
            if (S.forced_rows > 0) {
                // replay: the trace says how many tokens the step emits, the target text which ones
                m = S.forced_emit;
                const int* tg = a.target + (int64_t)s * a.y_cap;
#pragma unroll 1
                for (int j = lane; j < m; j += 32) {
                    ys[ylen + j] = tg[ylen + j];
                    if (kLocal) yg[ylen + j] = tg[ylen + j];
                }
                pending = tg[ylen + m - 1];
            } else {
                // first copied token the model disagrees with (32 comparisons per round), then the first EOS
                int acc = k_eff;
#pragma unroll 1
                for (int j0 = 0; j0 < k_eff; j0 += 32) {
                    const int j = j0 + lane;
                    const bool differs = j < k_eff && o[j] != ld_ref(&rs[pos + j]);
                    const unsigned mask = __ballot_sync(0xffffffffu, differs);
                    if (mask) { acc = j0 + __ffs(mask) - 1; break; }
                }
                m = acc + 1;
                if (dims.eos_id >= 0) {
#pragma unroll 1
                    for (int j0 = 0; j0 < m; j0 += 32) {
                        const int j = j0 + lane;
                        const unsigned mask = __ballot_sync(0xffffffffu, j < m && o[j] == dims.eos_id);
                        if (mask) { m = j0 + __ffs(mask); done = 1; break; }
                    }
                }
#pragma unroll 1
                for (int j = lane; j < m; j += 32) {
                    ys[ylen + j] = o[j];
                    if (kLocal) yg[ylen + j] = o[j];
                }
                pending = o[m - 1];
                // adaptive copy length: twice as many tokens after a copy the model agreed with in full, half as
                // many (rounded up) after one it cut short; within [k_min, the engine's largest k]
                if (lane == 0 && S.k_cur > 0 && k_eff > 0)
                    S.k_cur = acc == k_eff ? min(2 * S.k_cur, dims.kp1 - 1) : max(S.k_min, (S.k_cur + 1) >> 1);
            }
            __syncwarp();
            if (lane == 0) {
                S.pending = pending;
                S.y_len = ylen + m;
                S.kv_len += m;
                S.steps += 1;
                S.trigger_steps += (k_eff > 0);
                S.copied_accepted += m - 1;
                S.last_pos = pos; S.last_k_eff = k_eff; S.last_accepted = m - 1; S.last_emitted = m;
                if (ylen + m >= S.target_len) done = 1;
                S.done = done;
                S.nrows = 0;
            }
        }
    }
    __syncthreads();
    if (a.do_plan) {
        // ---- trigger search: every thread takes reference positions of every live sequence ---------------------
        // key = (ext << 32) | (0x7fffffff - pos): the maximum is the longest agreement, then the earliest position
        if (a.k > 0 && a.n >= 1) {
            // the 32 warps are dealt over the sequences (all of them on one sequence at batch 1, two per sequence at
            // batch 16, one warp for several sequences beyond 32), so that every sequence's loads are in flight at once
            int lg = 0;
            while ((B << (lg + 1)) <= n_warps) ++lg;
            const int per_seq = 1 << lg;                             // warps that share a sequence
            const int groups = n_warps >> lg;                        // sequences scanned at a time
            const int sub = warp & (per_seq - 1);
#pragma unroll 1
            for (int s = warp >> lg; s < B; s += groups) {
                const SeqState& S = s_st[s];
                const int ylen = S.y_len, ref_len = S.ref_len;
                const bool live = S.active && !S.done && ylen < S.target_len;
                if (!live || S.forced_rows != 0 || ylen < a.n || ref_len <= 0) continue;   // uniform over the warp
                const int* ys = v.y + (int64_t)s * a.y_cap;
                const int* rs = v.ref + (int64_t)s * 3 * dims.max_ref;
                const int* ds = rs + dims.max_ref;
                const int* de = ds + dims.max_ref;
                const int last = S.pending;  // the newest generated token (ylen >= 1 here)
                const int stride = 32 * per_seq;
#pragma unroll 1
                for (int p0 = 1 + sub * 32 + lane; p0 < ref_len; p0 += 2 * stride) {
                    // two candidates per round, their loads in flight together
                    int tokv[2], endv[2], begv[2];
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int p = p0 + u * stride;
                        const bool in = p < ref_len;
                        tokv[u] = in ? ld_ref(&rs[p - 1]) : -1;
                        endv[u] = in ? ld_ref(&de[p - 1]) : 0;
                        begv[u] = in ? ld_ref(&ds[p - 1]) : 0;
                    }
#pragma unroll 1
                    for (int u = 0; u < 2; ++u) {
                        const int p = p0 + u * stride;
                        // candidate: ref[p-1] is the last matched token; p must stay inside its document
                        if (p >= ref_len || (u ? tokv[1] : tokv[0]) != last || p >= (u ? endv[1] : endv[0])) continue;
                        // how far the agreement extends backwards: four tokens of each side per round trip
                        int t = 1;
                        const int lim = min(ylen, p - (u ? begv[1] : begv[0]));  // most tokens that can agree
                        for (bool go = true; go && t < lim;) {
                            int av[4], bv[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const int k = min(t + i, lim - 1);
                                av[i] = ld_ref(&rs[p - k - 1]);
                                bv[i] = ld_y(&ys[ylen - k - 1]);
                            }
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                go = go && t < lim && av[i] == bv[i];
                                if (go) ++t;
                            }
                        }
                        if (t >= a.n) atomicMax(&s_best[s], ((unsigned long long)(unsigned)t << 32) | (unsigned)(0x7fffffff - p));
                    }
                }
            }
        }
        __syncthreads();
        // ---- copy length, one thread per sequence ---------------------------------------------------------------
#pragma unroll 1
        for (int s = threadIdx.x; s < B; s += kTailThreads) {
            SeqState& S = s_st[s];
            const bool live = S.active && !S.done && S.y_len < S.target_len;
            const int ylen = S.y_len;
            int pos = -1, k_eff = 0, nrows = 0;
            if (live && a.trace && S.forced_rows != 0) {
                // replay: shape of the next step from the trace
                const int step = S.trace_step;
                int fr = 1, fe = 1;
                if (step < a.trace_cap) {
                    fr = a.trace[((int64_t)s * a.trace_cap + step) * 2];
                    fe = a.trace[((int64_t)s * a.trace_cap + step) * 2 + 1];
                }
                fr = max(1, min(fr, min(dims.kp1, dims.max_seq - S.kv_len)));
                fe = max(1, min(fe, min(fr, S.target_len - ylen)));
                nrows = fr; k_eff = fr - 1;
                S.forced_rows = fr; S.forced_emit = fe; S.trace_step = step + 1;
            } else if (live) {
                const unsigned long long best = s_best[s];
                if (best != 0ull) {
                    const int* de = v.ref + ((int64_t)s * 3 + 2) * dims.max_ref;
                    pos = 0x7fffffff - (int)(unsigned)(best & 0xffffffffull);
                    const int room_doc = ld_ref(&de[pos - 1]) - pos;
                    const int room_out = S.target_len - ylen - 1;
                    const int room_kv = dims.max_seq - S.kv_len - 1;
                    const int k_want = S.k_cur > 0 ? min(S.k_cur, a.k) : a.k;
                    k_eff = min(min(k_want, room_doc), min(room_out, room_kv));
                    if (k_eff <= 0) { k_eff = 0; pos = -1; }
                }
                nrows = k_eff + 1;
                if (S.kv_len + nrows > dims.max_seq) {  // no room even for the pending token
                    atomicExch(a.dev_err, kDevErrCapacity);
                    nrows = 0; pos = -1; k_eff = 0;
                }
            }
            S.pos = pos; S.k_eff = k_eff; S.nrows = nrows;
        }
        __syncthreads();
        // ---- pack the rows: sequence s owns rows first[s] .. first[s] + nrows - 1 -------------------------------
        if (threadIdx.x == 0) {
            int used = 0, mp = -1;
#pragma unroll 1
            for (int s = 0; s < B; ++s) {
                const int nr = s_st[s].nrows;
                s_first[s] = used;
                if (nr > 0) mp = max(mp, s_st[s].kv_len + nr - 1);
                used += nr;
            }
            if (used > a.n_rows) { atomicExch(a.dev_err, kDevErrCapacity); used = 0; }
            s_first[B] = used;
            a.rows->rows_used = used;
            emit_count(used);
            a.rows->max_pos = mp;
            atomicAdd(&a.rows->step_no, 1);
        }
        __syncthreads();
        const int used = s_first[B];
#pragma unroll 1
        for (int s = threadIdx.x; s < B; s += kTailThreads) {
            const int nr = used > 0 ? s_st[s].nrows : 0;
            a.rows->seq_first[s] = s_first[s];
            a.rows->seq_cnt[s] = nr;
            a.rows->seq_maxpos[s] = nr > 0 ? s_st[s].kv_len + nr - 1 : -1;
        }
#pragma unroll 1
        for (int s = warp; s < B; s += n_warps) {
            const SeqState& S = s_st[s];
            if (used == 0) break;  // the capacity error above voided the step
            const int* rs = v.ref + (int64_t)s * 3 * dims.max_ref;
            const int* tg = a.target ? a.target + (int64_t)s * a.y_cap : nullptr;
            const int first = s_first[s];
#pragma unroll 1
            for (int j = lane; j < S.nrows; j += 32) {
                int tok;
                if (j == 0) tok = S.pending;
                else if (S.forced_rows > 0) tok = tg[min(S.y_len + j - 1, a.y_cap - 1)];  // replay: the target's next tokens
                else tok = ld_ref(&rs[S.pos + j - 1]);
                a.rows->tok[first + j] = tok;
                a.rows->pos[first + j] = S.kv_len + j;
                a.rows->seq[first + j] = s;
                emit(first + j, tok, S.kv_len + j, s, first);
            }
        }
#pragma unroll 1
        for (int r = used + threadIdx.x; r < dims.row_cap; r += kTailThreads) {
            a.rows->tok[r] = 0; a.rows->pos[r] = -1; a.rows->seq[r] = 0;
            emit(r, 0, -1, 0, r);
        }
    }
}

// The work is a chain of small dependent steps, so what it costs is the number of global-memory round
// trips on that chain: the sequences' state is staged in shared memory once and written back at the end,
// the rows' final tokens stay in shared memory, and loads that do not depend on one another are issued together.
template <int kTailThreads>
__device__ __forceinline__ void step_tail(const TailArgs& a, TailShared& sh) {
    const TailLocal v = {sh.st, sh.first, sh.tok, sh.best, const_cast<int*>(a.ref), a.y};
    const int B = a.dims.max_batch;
    {
        const int32_t* src = reinterpret_cast<const int32_t*>(a.st);
        int32_t* dst = reinterpret_cast<int32_t*>(sh.st);
#pragma unroll 1
        for (int i = threadIdx.x; i < B * kStateWords; i += kTailThreads) dst[i] = __ldcg(src + i);
#pragma unroll 1
        for (int s = threadIdx.x; s < B; s += kTailThreads) sh.first[s] = __ldcg(&a.rows->seq_first[s]);
    }
    step_tail_on<kTailThreads, false>(a, v, [](int, int, int, int, int) {}, [](int) {});
    __syncthreads();
    {
        const int32_t* src = reinterpret_cast<const int32_t*>(sh.st);
        int32_t* dst = reinterpret_cast<int32_t*>(a.st);
#pragma unroll 1
        for (int i = threadIdx.x; i < B * kStateWords; i += kTailThreads) dst[i] = src[i];
    }
}

}  // namespace llma
