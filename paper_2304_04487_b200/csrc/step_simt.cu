// Whole decoding steps on the CUDA cores (decoders of the CUDA-core path and narrow bf16 decoders, where that pays: the rule and what it
// measured are in engine.cu) in one launch: embedding gather, layers, LM head, acceptance and the next plan, step after step.
//
// At the widths this path serves a step is a chain of short phases and costs their latency.  As launches of their own
// (kernels_simt.cu, attention_simt.cu) a phase is released about 1 us after its predecessor has ended, fetches its rows, and runs
// code that the SM has to fetch first.  A grid barrier instead costs as much: 0.6 us until a CTA's stores have reached L2, 0.4 us for
// the word that says so, 0.6 us to fetch the rows.  So activations travel as 8-byte words of a value and the number of the projection
// that wrote it, and a reader polls the words themselves: one trip to L2 each way.  A word is written again only by a CTA that has
// seen a result of every reader of its old value (a projection's results depend on all of its rows' values), so there is nothing to
// clear and nothing to wait for.  One grid barrier per step makes the step's cache rows visible to the next one (the step itself takes
// its own K/V rows from the words); it is passed while the next step's first projection runs, and the last one stands before the state is
// written back.
//
// CTA 0 does acceptance and plan, with states, references and emitted tokens in its shared memory.  The others, one per SM (of all, or of
// a share of them: device_gate.h), sixteen warps each, do everything else.  A warp takes four pairs of output features (of a rotary pair, of gate and up, of neighbours):
// eight lanes per pair, each with its own columns of the two weight rows, all rows' sums in registers, the rows themselves in
// shared memory, where a warp's access is one 128-byte line; 2 to 16 warps share the columns of a unit.  Units are dealt over the SMs
// first, so that every SM pulls weights whatever the width.  Weights come through a ring of four pieces per warp: four more warps
// request the first pieces of every unit, projections and steps ahead (no kernel writes weights), and a warp the rest of a long unit.
//
// What bounds it: per phase a trip of the words (0.85 to 1 us from a store to the last poll, measured alone with 148 CTAs) and the
// chain of instructions of a warp that has its scheduler almost to itself.  So waits fetch all that is missing together (one by one:
// 42 -> 34 us per step of width 256 for this alone), one and two rows have code of their own, and nothing is spilled: local memory does not
// fit what 226 KB of shared memory leave of L1, and a reload comes from L2 or further (2 us at the end of the attention phase of
// width 1024).  Feeders give up registers for the warps that multiply for that reason.
// us per decode, as launches -> here: two fp32 layers of width 256, 64 tokens, up to five rows 2483 -> 1443; of width 1024, up to nine
// rows 2709 -> 1863 (its weights, 135 MB a step, take 450); up to 76 rows, in five passes over the weights, 3435 -> 3430.
//
// Every sum is a fixed sequence of operations that depends on its own row's data and on the shapes only, never on how many rows the
// step has.
#include <type_traits>

#include "grid_barrier.cuh"
#include "simt_common.cuh"
#include "step_simt.cuh"
#include "step_tail.cuh"

namespace llma {

using namespace ptx;

constexpr int kSW = 16;                        // warps per CTA
constexpr int kST = kSW * 32;
constexpr int kFeeders = 4;                    // warps that request weights, for a quarter of the others each
constexpr int kThreads = kST + 32 * kFeeders;
constexpr int kSR = 16;                        // most activation rows per pass over the weights
constexpr int kRing = 4;                       // pieces of weights (1 KB) under way per warp (a power of two)
constexpr int kSweep = 2 * kST;                // activations that the CTA fetches at a time
constexpr size_t kStepSmem = 205 * 1024;       // most dynamic shared memory
constexpr size_t kRingBytes = (size_t)kSW * kRing * 1024;

enum : int { kOpQKV = 0, kOpO = 1, kOpGateUp = 2, kOpDown = 3, kOpHead = 4 };

// ---- words of a value and its number -------------------------------------------------------------------------------
typedef unsigned long long LLWord;
__device__ __forceinline__ LLWord ll_word(float v, uint32_t epoch) { return ((LLWord)epoch << 32) | __float_as_uint(v); }
__device__ __forceinline__ void ll_store(LLWord* p, float v, uint32_t epoch) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(ll_word(v, epoch)) : "memory");
}
__device__ __forceinline__ void ll_store2(LLWord* p, float v0, float v1, uint32_t epoch) {  // two neighbouring words, 16-byte aligned
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(ll_word(v0, epoch)), "l"(ll_word(v1, epoch)) : "memory");
}
struct LL2 { LLWord a, b; };
__device__ __forceinline__ LL2 ll_load2(const LLWord* p) {
    LL2 w;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.a), "=l"(w.b) : "l"(p) : "memory");
    return w;
}
__device__ __forceinline__ bool ll_ready(const LL2& w, uint32_t epoch) { return (uint32_t)(w.a >> 32) == epoch && (uint32_t)(w.b >> 32) == epoch; }
__device__ __forceinline__ float2 ll_values(const LL2& w) { return make_float2(__uint_as_float((uint32_t)w.a), __uint_as_float((uint32_t)w.b)); }
// A wait runs out when the launch's CTAs are not on the GPU together, because something else holds SMs for long.  Such a launch is as
// good as not made: a CTA that has given up (its flag is up) passes no further barrier, CTA 0 writes no state back unless every CTA has
// passed the barrier that ends the last step, what else has been written belongs to positions that the state does not reach, and
// the host launches the steps again.  (Keeping what has not arrived from being published instead, by barriers that tell all threads of a
// CTA, cost 0.4 to 1.5 us a step; a mark in global memory ahead of it 0.3 to 1.4.)
struct Waits {
    volatile int* failed;  // of the CTA
    int patience;          // polls
};
// Polls until every pair of words carries the number: at(u) is where pair u lies, nullptr if there is none.  The pairs that are missing are
// fetched together, so that the wait ends a trip to L2 after the last of them has landed.  Bounded: the CTA gives up when the wait runs
// out, and no wait of the CTA lasts once it has.
template <int U, typename At>
__device__ __forceinline__ void ll_fetch(LL2 (&w)[U], uint32_t epoch, const Waits& up, At at) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
        w[u].a = w[u].b = (LLWord)epoch << 32;
        if (const LLWord* p = at(u)) w[u] = ll_load2(p);
    }
    int left = up.patience;
#pragma unroll 1
    for (;;) {
        bool all = true;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!ll_ready(w[u], epoch)) {
                all = false;
                w[u] = ll_load2(at(u));
            }
        }
        if (all) break;
        if (--left == 0) *up.failed = 1;
        if (*up.failed) break;
    }
}
__device__ __forceinline__ void ll_wait2(LL2& w, const LLWord* p, uint32_t epoch, const Waits& up) {  // w has been fetched once
    int left = up.patience;
#pragma unroll 1
    while (!ll_ready(w, epoch)) {
        w = ll_load2(p);
        if (--left == 0) *up.failed = 1;
        if (*up.failed) break;
    }
}

// whether the phase is over, without waiting
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void l2_prefetch(const void* p, int bytes) {  // both multiples of 16
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ void workers_sync() { named_bar_sync(1, kST); }
// the barrier counts this thread's arrival once all of its cp.async copies so far have landed
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

// Where the rows of the step belong
struct StepRows {
    int tok[kRowCap], pos[kRowCap], seq[kRowCap];
    int first[kRowCap];  // first row of the same sequence
    int used;
};
__device__ __forceinline__ LLWord* ll_rows_of(const SimtStep& a, uint32_t epoch) { return a.ll_rows + (epoch & 1) * (2 + 4 * (size_t)a.dims.row_cap); }

// N consecutive cache values of a lane, from the cache (past L1) or from shared memory
template <int N> __device__ __forceinline__ void load_few(bool cached, const float* p, const float* fresh, float (&v)[N]) {
    if constexpr (N == 4) {
        const float4 x = cached ? __ldcg(reinterpret_cast<const float4*>(p)) : *reinterpret_cast<const float4*>(fresh);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
        const float2 x = cached ? __ldcg(reinterpret_cast<const float2*>(p)) : *reinterpret_cast<const float2*>(fresh);
        v[0] = x.x; v[1] = x.y;
    }
}
template <int N> __device__ __forceinline__ void load_few(bool cached, const __nv_bfloat16* p, const __nv_bfloat16* fresh, float (&v)[N]) {
    uint32_t w[2];
    if constexpr (N == 4) {
        const uint2 x = cached ? __ldcg(reinterpret_cast<const uint2*>(p)) : *reinterpret_cast<const uint2*>(fresh);
        w[0] = x.x; w[1] = x.y;
    } else {
        w[0] = cached ? __ldcg(reinterpret_cast<const uint32_t*>(p)) : *reinterpret_cast<const uint32_t*>(fresh);
    }
#pragma unroll
    for (int i = 0; i < N / 2; ++i) { v[2 * i] = __uint_as_float(w[i] << 16); v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
}

// Causal attention of row r and one head over positions 0 .. pos.  A warp takes four positions in every 64 (eight lanes score one) with a
// running maximum, sum and output; the sixteen warps are combined at the end.  Positions below the sequence's first row of the
// step are read from the cache, the others come with the words (rounded as the cache has them).
// sm: q, the sequence's own K and V rows of the step, then the warps' partial results.
template <typename T, int HD>
__device__ __forceinline__ void attend(const SimtStep& a, const StepRows& R, int layer, int head, int r, uint32_t epoch, float* sm,
                                       const Waits& up) {
    constexpr int NJ = HD / 32;   // float4 of k per lane of an eight-lane group
    constexpr int NF = HD / 32;   // output values per lane
    const ModelDims& dims = a.dims;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, e = lane & 7, g = lane >> 3;
    const int pos = R.pos[r], r_first = R.first[r], pos0 = R.pos[r_first], fresh = r - r_first + 1;
    const int HT = dims.hd_total;
    float* s_q = sm;
    T* s_k = reinterpret_cast<T*>(s_q + HD);
    T* s_v = s_k + dims.kp1 * HD;
    float* s_o = reinterpret_cast<float*>(s_v + dims.kp1 * HD);
    float *s_m = s_o + kSW * HD, *s_l = s_m + kSW;
    // k and v of the step's rows up to this one (q with the last of them): 3 HD / 2 pairs a row, from the newest row back
    {
        constexpr int P = HD / 2;
        const LLWord* words = a.ll_qkv + head * HD;
#pragma unroll 1
        for (int i = threadIdx.x; i < P + 2 * P * fresh; i += kST) {
            const int s = i / P, c = 2 * (i % P);  // 0 q; then k and v of a row in turn
            const int row = r - (s > 0 ? (s - 1) >> 1 : 0), part = s == 0 ? 0 : 2 - (s & 1);
            LL2 w[1];
            ll_fetch(w, epoch, up, [&](int) { return words + (3 * row + part) * HT + c; });
            const float2 v = ll_values(w[0]);
            if (s == 0) {
                *reinterpret_cast<float2*>(s_q + c) = v;
            } else {
                T* dst = (part == 1 ? s_k : s_v) + (row - r_first) * HD + c;
                dst[0] = from_f32<T>(v.x); dst[1] = from_f32<T>(v.y);
            }
        }
    }
    workers_sync();
    const int64_t base = kv_row_index(dims, layer, R.seq[r], head, 0) * HD;
    const T* K = reinterpret_cast<const T*>(a.kcache) + base + e * 4;
    const T* V = reinterpret_cast<const T*>(a.vcache) + base + lane * NF;
    const T *fk = s_k - pos0 * HD + e * 4, *fv = s_v - pos0 * HD + lane * NF;
    float4 q[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) q[j] = *reinterpret_cast<const float4*>(s_q + (j * 8 + e) * 4);
    float o[NF] = {};
    float M = -INFINITY, l = 0.f;
    const float scale = rsqrtf((float)HD);
    float k[NJ][4], v[4][NF];
    auto load = [&](int b) {
        const int p = min(b + g, pos) * HD;
#pragma unroll
        for (int j = 0; j < NJ; ++j) load_few(p < pos0 * HD, K + p + j * 32, fk + p + j * 32, k[j]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int pv = min(b + u, pos) * HD;
            load_few(pv < pos0 * HD, V + pv, fv + pv, v[u]);
        }
    };
    int b = 4 * warp;
    load(b);
#pragma unroll 1
    while (b <= pos) {
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            s = fmaf(q[j].x, k[j][0], s); s = fmaf(q[j].y, k[j][1], s);
            s = fmaf(q[j].z, k[j][2], s); s = fmaf(q[j].w, k[j][3], s);
        }
        float x[4][NF];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int c = 0; c < NF; ++c) x[u][c] = v[u][c];
        const bool on = b + g <= pos;
        b += 4 * kSW;
        load(b);  // the next sweep's rows, on their way meanwhile (past the end: the last ones again)
#pragma unroll
        for (int i = 1; i <= 4; i <<= 1) s += __shfl_xor_sync(0xffffffffu, s, i);
        s = on ? s * scale : -INFINITY;
        float m = fmaxf(M, s);
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 8));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
        const float ref = m == -INFINITY ? 0.f : m;         // (scores that have overflowed, and nothing else so far)
        const float f = expf(M - ref);                      // 0 at first
        M = m;
        s = expf(s - ref);  // 0 past pos
        l = fmaf(l, f, s);
#pragma unroll
        for (int c = 0; c < NF; ++c) o[c] *= f;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float w = __shfl_sync(0xffffffffu, s, 8 * u);
#pragma unroll
            for (int c = 0; c < NF; ++c) o[c] = fmaf(w, x[u][c], o[c]);
        }
    }
    l += __shfl_xor_sync(0xffffffffu, l, 8);
    l += __shfl_xor_sync(0xffffffffu, l, 16);
    if (lane == 0) { s_m[warp] = M; s_l[warp] = l; }
#pragma unroll
    for (int c = 0; c < NF; ++c) s_o[warp * HD + lane * NF + c] = o[c];
    workers_sync();
    if (warp < HD / 32) {
        const float mw = s_m[lane & (kSW - 1)];
        float mx = mw;
#pragma unroll 1
        for (int i = kSW / 2; i > 0; i >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, i));
        const float f = expf(mw - mx);  // 0 for warps without a position
        float den = f * s_l[lane & (kSW - 1)];
#pragma unroll 1
        for (int i = kSW / 2; i > 0; i >>= 1) den += __shfl_xor_sync(0xffffffffu, den, i);
        float num = 0.f;
#pragma unroll 4
        for (int w = 0; w < kSW; ++w) num = fmaf(__shfl_sync(0xffffffffu, f, w), s_o[w * HD + threadIdx.x], num);
        const int at = r * HT + head * HD + threadIdx.x;
        const float val = num / den;
        ll_store(a.ll_attn + at, val, epoch);
        a.attn[at] = val;
    }
    workers_sync();
}

// The launch before has given up: this one would meet the barrier half passed, and its steps are launched again anyway.  (A CTA that only
// gets an SM when others of its own launch have given up may see it too.)
__device__ __forceinline__ bool given_up(const SimtStep& a) { return threadIdx.x == 0 && __ldcg(a.dev_err) == kDevErrSteps; }

// Acceptance and plan, step after step (CTA 0)
__device__ __forceinline__ void tail_cta(const SimtStep& a, uint8_t* sm, const Waits& up) {
    const ModelDims& d = a.dims;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, B = d.max_batch;
    const int n_parts = min((int)gridDim.x - 1, a.geo[kOpHead].n_units);
    TailLocal v;
    v.best = reinterpret_cast<unsigned long long*>(sm);
    v.st = reinterpret_cast<SeqState*>(v.best + B);
    v.first = reinterpret_cast<int*>(v.st + B);
    v.tok = v.first + B + 1;
    v.ref = v.tok + d.row_cap;
    v.y = v.ref + B * 3 * d.max_ref;
    for (int i = tid; i < B * kStateWords; i += kThreads) reinterpret_cast<int*>(v.st)[i] = __ldcg(reinterpret_cast<const int*>(a.tail.st) + i);
    __syncthreads();
#pragma unroll 1
    for (int s = 0; s < B; ++s) {
#pragma unroll 1
        for (int i = tid; i < v.st[s].ref_len; i += kThreads) {
#pragma unroll
            for (int j = 0; j < 3; ++j) v.ref[(s * 3 + j) * d.max_ref + i] = __ldcg(a.tail.ref + ((int64_t)s * 3 + j) * d.max_ref + i);
        }
#pragma unroll 1
        for (int i = tid; i < v.st[s].y_len; i += kThreads) v.y[s * a.tail.y_cap + i] = __ldcg(a.tail.y + (int64_t)s * a.tail.y_cap + i);
    }
    if (__syncthreads_or(given_up(a))) return;
    GridBarrier bar(a.barrier);
    uint32_t epoch = a.epoch;
    auto publish = [&](int r, int tok, int pos, int seq, int first) {
        LLWord* w = ll_rows_of(a, epoch) + 2 + 4 * r;
        ll_store2(w, __int_as_float(tok), __int_as_float(pos), epoch);
        ll_store2(w + 2, __int_as_float(seq), __int_as_float(first), epoch);
    };
    auto publish_count = [&](int used) { ll_store2(ll_rows_of(a, epoch), __int_as_float(used), 0.f, epoch); };
    __syncthreads();
    bool begun = false;  // thread 0: a barrier is under way
    // step -1: the plan of the first step
#pragma unroll 1
    for (int step = -1; step < a.max_steps; ++step) {
        TailArgs t = a.tail;
        t.do_accept = 0; t.do_plan = 1;
        if (step >= 0) {
            const bool last = step + 1 == a.max_steps;
            const int rows_used = v.first[B];
            if (rows_used == 0) break;
            if (tid == 0) {  // rows are published into the other half of ll_rows: every CTA has read what was there
                if (step > 0 && !bar.wait(600ull * a.patience)) *up.failed = 1;
                bar.arrive();
                begun = true;
            }
#pragma unroll 1
            for (int r = warp; r < rows_used; r += kThreads / 32) {  // final token: lowest index on ties
                float m = -INFINITY;
                int i = 0x7fffffff;
#pragma unroll 1
                for (int p = lane; p < n_parts; p += 160) {
                    LL2 w[5];
                    ll_fetch(w, epoch + 4 * d.n_layers, up,
                             [&](int u) { return p + 32 * u < n_parts ? a.ll_part + 2 * ((int64_t)(p + 32 * u) * d.row_cap + r) : nullptr; });
#pragma unroll
                    for (int u = 0; u < 5; ++u) {
                        const float2 x = ll_values(w[u]);
                        const int xi = __float_as_int(x.y);
                        if (p + 32 * u < n_parts && (x.x > m || (x.x == m && xi < i))) { m = x.x; i = xi; }
                    }
                }
#pragma unroll 1
                for (int w = 16; w > 0; w >>= 1) {
                    const float om = __shfl_xor_sync(0xffffffffu, m, w);
                    const int oi = __shfl_xor_sync(0xffffffffu, i, w);
                    if (om > m || (om == m && oi < i)) { m = om; i = oi; }
                }
                if (lane == 0) { v.tok[r] = i; a.tail.out_tok[r] = i; }
            }
            if (__syncthreads_or(*up.failed)) break;
            epoch += simt_epochs(d);
            t.do_accept = 1; t.do_plan = !last;
        }
        step_tail_on<kThreads, true>(t, v, publish, publish_count);
        __syncthreads();
    }
    if (begun && !bar.wait(600ull * a.patience)) *up.failed = 1;
    if (__syncthreads_or(*up.failed)) {
        if (tid == 0) atomicExch(a.dev_err, kDevErrSteps);
        return;
    }
    for (int i = tid; i < B * kStateWords; i += kThreads) reinterpret_cast<int*>(a.tail.st)[i] = reinterpret_cast<const int*>(v.st)[i];
}

template <typename T, int HD>
__global__ void __launch_bounds__(kThreads, 1) step_simt_kernel(const __grid_constant__ SimtStep a) {
    constexpr int VN = Vec16<T>::N;              // values per 16 bytes
    extern __shared__ __align__(16) float sA[];  // rows of a pass; scratch of the attention phase.  Then the weight ring, then the ops
    __shared__ StepRows R;
    __shared__ float s_rs[kSR];                  // RMSNorm scale of a row
    __shared__ int s_fail, s_stop;               // a wait ran out; the feeders may go
    __shared__ int s_steps, s_passes[2];         // steps begun, passes over the weights in the last two of them
    __shared__ uint64_t s_bar[2][kSW][kRing];    // a place of a warp's weight ring is full, is empty
    __shared__ float2 s_part[2][kSW][4][kSR];    // a warp's sums of the two features of its four pairs, rounds in turn
    if (threadIdx.x == 0) { s_fail = 0; s_stop = 0; s_steps = 0; }
    if (threadIdx.x < kSW * kRing) {
        mbar_init(smem_u32(&s_bar[0][0][0]) + 8 * threadIdx.x, 32);
        mbar_init(smem_u32(&s_bar[1][0][0]) + 8 * threadIdx.x, 1);
    }
    fence_mbar_init();
    __syncthreads();
    const Waits up = {&s_fail, a.patience};
    if (blockIdx.x == 0) {
        tail_cta(a, reinterpret_cast<uint8_t*>(sA), up);
        return;
    }
    const ModelDims& d = a.dims;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, cta = blockIdx.x - 1, G = gridDim.x - 1;
    const int n_ops = 4 * d.n_layers + 1, pass = a.pass_rows;
    // Rows in shared memory: four columns of every row side by side, [column / 4][row][4], an odd number of 16-byte places apart: the
    // eight lanes of a pair fall into different banks, and a row is a constant offset.
    const int pitch = 4 * (pass | 1);
    constexpr int half = HD >> 1;
    const int HT = d.hd_total;
    const int pq = lane >> 3, kq = lane & 7;         // pair of the unit, place among its eight lanes
    const T* emb = reinterpret_cast<const T*>(a.emb);
    SimtOp* s_ops = reinterpret_cast<SimtOp*>(reinterpret_cast<char*>(sA) + a.ops_offset);
    {
        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(a.ops);
        for (int i = tid; i < n_ops * (int)(sizeof(SimtOp) / 8); i += kThreads) reinterpret_cast<unsigned long long*>(s_ops)[i] = __ldg(src + i);
    }
    if (__syncthreads_or(given_up(a))) return;
    GridBarrier bar(a.barrier);
    float* s_gain = sA + a.gain_offset / 4;  // the norm's gains

    auto qkv_pair = [&](int p, int& mat, int& head, int& i) {
        mat = (p >= (HT >> 1) ? 1 : 0) + (p >= HT ? 1 : 0);
        const int v = p - mat * (HT >> 1);
        head = v / half;
        i = v % half;
    };

    // A unit's weights: the first pair's two rows, the bytes between pairs' rows, and the last row of the matrix seen from the first
    struct UnitRows { const char *p0, *p1; int stride, last; };
    auto unit_rows = [&](int op, int m, int unit) {
        const SimtOp& o = s_ops[op];
        const int p = 4 * unit;
        const void *b0 = o.w0, *b1 = o.w0;
        int r0 = 2 * p, r1 = r0 + 1, n = 2;
        if (m == kOpQKV) {
            int mat, head, i;
            qkv_pair(p, mat, head, i);
            if (mat > 0) b0 = b1 = mat == 1 ? o.w1 : o.w2;
            r0 = head * HD + i; r1 = r0 + half; n = 1;
        } else if (m == kOpGateUp) {
            r0 = r1 = p; n = 1;
            b1 = o.w1;
        }
        const int row_bytes = a.geo[m].n_pieces * 128;
        return UnitRows{reinterpret_cast<const char*>(b0) + (int64_t)r0 * row_bytes, reinterpret_cast<const char*>(b1) + (int64_t)r1 * row_bytes,
                        n * row_bytes, m == kOpHead ? d.vocab - 1 - r0 : 1 << 20};
    };
    auto lane_rows = [&](UnitRows u, const char*& q0, const char*& q1) {  // this lane's 16 bytes of the unit's first piece
        if (u.last < 8) {  // the vocabulary ends within the unit: its last row again
            q0 = u.p0 + (int64_t)min(2 * pq, u.last) * (u.stride >> 1) + kq * 16;
            q1 = u.p1 + (int64_t)min(2 * pq + 1, u.last) * (u.stride >> 1) + kq * 16 - (u.stride >> 1);
        } else {
            q0 = u.p0 + pq * u.stride + kq * 16;
            q1 = u.p1 + pq * u.stride + kq * 16;
        }
    };
    const uint32_t full0 = smem_u32(&s_bar[0][0][0]), empty0 = smem_u32(&s_bar[1][0][0]);
    const uint32_t ring0 = smem_u32(sA) + a.ring_offset + lane * 16;
    if (warp >= kSW) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");  // 4 x 32 x (96 - 64) registers = 16 x 32 x (104 - 96)
        // ---- feeders: lane i holds what warp first + i multiplies next, the whole warp requests it ------------------------------
        // The pieces of a warp come in the order in which it multiplies them: steps, projections, passes, units, pieces part, part + split, ...
        // The feeder requests the first kRing of a unit as places come free, before the unit has begun and beyond the end of the projection;
        // the rest the warp requests itself, each into the place that it has just read.
        constexpr int kEach = kSW / kFeeders;
        const int mine = (warp - kSW) * kEach + (lane & (kEach - 1));  // (lanes from kEach on repeat the first ones and request nothing)
        int op = -1, m = 0, lg = 0, unit = 0, units = 0, piece = 0, pieces = 0, pass_no = kRowCap, step = 0, slot = 0;
        uint32_t phases = (1u << kRing) - 1u;  // of the places' empty barriers
        UnitRows u = {nullptr, nullptr, 0, 0};
        bool find = true, any = true;  // the unit's rows have to be found; the warp has something to multiply at all
        volatile int *stop = &s_stop, *steps = &s_steps, *passes = s_passes;
        // (what the lanes read one by one may change between them: such a decision is the warp's, or they would part for good)
        while (!__any_sync(0xffffffffu, *stop)) {
            bool ready = any;
            if (any && unit >= units) {  // done with a pass over a projection, or not begun
                // (how many passes a step has is known once it has begun, and is read of the step that is being fed: the next one may
                // have begun meanwhile, the one after it not before this warp's part of the next one has been fed)
                if (op < 0 || a.passes == 1 || *steps > step) {
                    find = true;
                    unit = (mine >> lg) * G + cta;
                    if (op < 0 || ++pass_no >= (a.passes == 1 ? 1 : passes[step & 1])) {  // the next projection that has pieces for the warp
                        int left = n_ops + 1;
                        do {
                            if (++op == n_ops) { op = 0; ++step; }
                            m = op == n_ops - 1 ? kOpHead : op & 3;
                            lg = a.geo[m].split_lg; units = a.geo[m].n_units; pieces = a.geo[m].n_pieces;
                            unit = (mine >> lg) * G + cta; piece = mine & ((1 << lg) - 1);
                        } while ((unit >= units || piece >= pieces) && --left > 0);
                        pass_no = 0;
                        any = left > 0;
                    }
                }
                ready = any && unit < units;
            }
            if (ready && find) {
                find = false;
                u = unit_rows(op, m, unit);
            }
            bool idle = true;
            for (unsigned todo = __ballot_sync(0xffffffffu, ready && lane < kEach); todo; todo &= todo - 1) {
                const int i = __ffs(todo) - 1;
                UnitRows v;
                v.p0 = reinterpret_cast<const char*>(__shfl_sync(0xffffffffu, (unsigned long long)u.p0, i));
                v.p1 = reinterpret_cast<const char*>(__shfl_sync(0xffffffffu, (unsigned long long)u.p1, i));
                v.stride = __shfl_sync(0xffffffffu, u.stride, i); v.last = __shfl_sync(0xffffffffu, u.last, i);
                const int qlg = __shfl_sync(0xffffffffu, lg, i), end = min(__shfl_sync(0xffffffffu, pieces, i), kRing << qlg);
                int pc = __shfl_sync(0xffffffffu, piece, i), sl = __shfl_sync(0xffffffffu, slot, i);
                uint32_t ph = __shfl_sync(0xffffffffu, phases, i);
                const char *q0, *q1;
                lane_rows(v, q0, q1);
                const int place0 = ((warp - kSW) * kEach + i) * kRing;
                while (pc < end && __all_sync(0xffffffffu, mbar_test(empty0 + 8 * (place0 + sl), (ph >> sl) & 1u))) {
                    const uint32_t dst = ring0 + (place0 + sl) * 1024;
                    cp_async_16(dst, q0 + pc * 128);
                    cp_async_16(dst + 512, q1 + pc * 128);
                    cp_async_arrive(full0 + 8 * (place0 + sl));
                    ph ^= 1u << sl;
                    sl = (sl + 1) & (kRing - 1);
                    pc += 1 << qlg;
                    idle = false;
                }
                if (lane == i) { piece = pc; slot = sl; phases = ph; }
            }
            if (ready && piece >= min(pieces, kRing << lg)) {
                const int part = mine & ((1 << lg) - 1), all = (pieces - part + (1 << lg) - 1) >> lg;  // the unit's pieces
                slot = (slot + max(all - kRing, 0)) & (kRing - 1);
                piece = part;
                unit += (kSW >> lg) * G;
                find = true;
            }
            __syncwarp();
            if (idle) __nanosleep(40);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
    }
    const uint32_t ring = ring0 + warp * (kRing * 1024), full = full0 + 8 * warp * kRing, empty = empty0 + 8 * warp * kRing;

    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    int c_slot = 0;  // the piece multiplied next
    uint32_t c_phase = 0;
    int rows_used = 0;

    // ---- one projection of the step: rows into shared memory, products, what follows them -------------------------------------
    // Up to two and up to eight rows in code of their own, since a phase costs its instructions: what a chain of dependent instructions
    // costs a warp that is alone on its scheduler
    auto project = [&](auto rows_tag, int m, int op, uint32_t epoch) {
        constexpr int NR = decltype(rows_tag)::value;  // rows whose sums are held
        constexpr bool kFew = NR == 2;
        const bool norm = m == kOpQKV || m == kOpGateUp || m == kOpHead;
        const int K = a.geo[m].k_in, lg = a.geo[m].split_lg, n_units = a.geo[m].n_units, n_pieces = a.geo[m].n_pieces;
        const int step_units = (kSW >> lg) * G;
        // end of a unit: a thread per (unit slot, pair, row)
        const int e_row = kFew ? tid & 1 : tid & 15, e_pair = (kFew ? tid >> 1 : tid >> 4) & 3, e_slot = kFew ? tid >> 3 : tid >> 6;
        float best = -INFINITY;
        int best_i = 0x7fffffff;
#pragma unroll 1
        for (int r0 = 0; r0 < rows_used; r0 += pass) {
            const int nr = NR < kSR ? rows_used : min(pass, rows_used - r0);
            const int row = r0 + e_row;  // of this thread at the end of a unit
            const bool e_on = e_row < nr && e_slot < (kSW >> lg);
            if (r0 > 0) workers_sync();
            // what the end of a unit needs besides its sums (residual values, rotary factors) and where its results go
            float e0 = 0.f, e1 = 0.f;
            LL2 ex = {0, 0};
            int64_t e_at = 0, e_cache = 0;
            int e_mat = 0;
            auto fetch_end = [&](int e_unit) {
                if (!e_on || e_unit >= n_units) return;
                const int p = 4 * e_unit + e_pair;
                if (m == kOpQKV) {
                    int head, i;
                    qkv_pair(p, e_mat, head, i);
                    const int pos = R.pos[row];
                    if (e_mat < 2) {
                        e0 = __ldg(&a.rope_cos[(int64_t)pos * half + i]);
                        e1 = __ldg(&a.rope_sin[(int64_t)pos * half + i]);
                    }
                    e_at = ((int64_t)row * 3 + e_mat) * HT + head * HD + i;
                    e_cache = kv_row_index(d, op >> 2, R.seq[row], head, pos) * HD + i;
                } else if (m == kOpGateUp) {
                    e_at = (int64_t)row * d.d_ffn + p;
                } else if (m == kOpHead) {
                    e_at = (int64_t)row * d.vocab + 2 * p;
                } else {
                    e_at = (int64_t)row * d.d_model + 2 * p;
                    if (m == kOpO && op == kOpO) {  // first layer: the residual stream is still the embedding
                        const T* er = emb + (int64_t)R.tok[row] * d.d_model + 2 * p;
                        e0 = to_f32<T>(er[0]); e1 = to_f32<T>(er[1]);
                    } else {
                        ex = ll_load2(a.ll_x + e_at);
                    }
                }
            };
            fetch_end(e_slot * G + cta);
            // ---- rows (and the gains of their norm) into shared memory ------------------------------------------------------
            if (norm) {
                const float* gain = s_ops[op].gain;
                for (int k = tid; k < K; k += kST) s_gain[k] = __ldg(gain + k);
            }
            {
                const int total = nr * K, sweep_cols = a.geo[m].sweep_cols, sweep_rows = a.geo[m].sweep_rows;
                int rr = 0, k = 2 * tid;  // row and column of this thread's next two values
                while (k >= K) { k -= K; ++rr; }
                auto put = [&](float2 v) {
                    *reinterpret_cast<float2*>(sA + (k >> 2) * pitch + rr * 4 + (k & 3)) = v;
                    k += sweep_cols; rr += sweep_rows;
                    if (k >= K) { k -= K; ++rr; }
                };
                if (op == 0) {
#pragma unroll 2
                    for (int i = 2 * tid; i < total; i += kSweep) {
                        const T* er = emb + (int64_t)R.tok[r0 + rr] * K + k;
                        put(make_float2(to_f32<T>(er[0]), to_f32<T>(er[1])));
                    }
                } else {
                    constexpr int U = kFew ? 3 : 4;
                    const LLWord* src = (norm ? a.ll_x : (m == kOpO ? a.ll_attn : a.ll_h)) + (int64_t)r0 * K;
                    const uint32_t want = epoch - 1;  // the projection before this one (attention: with the number of its QKV projection)
#pragma unroll 1
                    for (int i0 = 2 * tid; i0 < total; i0 += U * kSweep) {
                        LL2 w[U];
                        ll_fetch(w, want, up, [&](int u) { return i0 + u * kSweep < total ? src + i0 + u * kSweep : nullptr; });
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (i0 + u * kSweep < total) put(ll_values(w[u]));
                    }
                }
            }
            workers_sync();
#pragma unroll 1
            for (int round = 0, unit = (warp >> lg) * G + cta, e_unit = e_slot * G + cta; round * step_units + cta < n_units;
                 ++round, unit += step_units, e_unit += step_units) {
                float2 (*parts)[4][kSR] = s_part[round & 1];
                if (unit < n_units) {
                    float acc[2][NR];  // [side][row]
#pragma unroll
                    for (int i = 0; i < NR; ++i) acc[0][i] = acc[1][i] = 0.f;
                    const char *q0 = nullptr, *q1 = nullptr;
                    if (n_pieces > kRing << lg) lane_rows(unit_rows(op, m, unit), q0, q1);
#pragma unroll 1
                    for (int c = warp & ((1 << lg) - 1); c < n_pieces; c += 1 << lg) {
                        if (!mbar_wait(full + 8 * c_slot, c_phase)) *up.failed = 1;
                        uint4 w0, w1;
                        {
                            const uint32_t src = ring + c_slot * 1024;
                            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w0.x), "=r"(w0.y), "=r"(w0.z), "=r"(w0.w) : "r"(src) : "memory");
                            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w1.x), "=r"(w1.y), "=r"(w1.z), "=r"(w1.w) : "r"(src + 512) : "memory");
                        }
                        float wa[VN], wb[VN];
                        Vec16<T>::widen(w0, wa);
                        Vec16<T>::widen(w1, wb);
                        if (norm) {
                            const float* gp = s_gain + (c * 8 + kq) * VN;
#pragma unroll
                            for (int v4 = 0; v4 < VN; v4 += 4) {
                                const float4 gn = *reinterpret_cast<const float4*>(gp + v4);
                                wa[v4] *= gn.x; wa[v4 + 1] *= gn.y; wa[v4 + 2] *= gn.z; wa[v4 + 3] *= gn.w;
                                wb[v4] *= gn.x; wb[v4 + 1] *= gn.y; wb[v4 + 2] *= gn.z; wb[v4 + 3] *= gn.w;
                            }
                        }
                        const float* ap = sA + (c * 8 + kq) * (VN / 4) * pitch;
#pragma unroll
                        for (int q = 0; q < NR; q += 2) {
                            if (q >= nr) break;
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
#pragma unroll
                                for (int v4 = 0; v4 < VN; v4 += 4) {
                                    const float4 b = *reinterpret_cast<const float4*>(ap + (v4 >> 2) * pitch + (q + u) * 4);
                                    acc[0][q + u] = fmaf(wa[v4], b.x, acc[0][q + u]); acc[1][q + u] = fmaf(wb[v4], b.x, acc[1][q + u]);
                                    acc[0][q + u] = fmaf(wa[v4 + 1], b.y, acc[0][q + u]); acc[1][q + u] = fmaf(wb[v4 + 1], b.y, acc[1][q + u]);
                                    acc[0][q + u] = fmaf(wa[v4 + 2], b.z, acc[0][q + u]); acc[1][q + u] = fmaf(wb[v4 + 2], b.z, acc[1][q + u]);
                                    acc[0][q + u] = fmaf(wa[v4 + 3], b.w, acc[0][q + u]); acc[1][q + u] = fmaf(wb[v4 + 3], b.w, acc[1][q + u]);
                                }
                            }
                        }
                        const int more = c + (kRing << lg);
                        if (more < n_pieces) {  // (a lane reads what it has requested itself)
                            cp_async_16(ring + c_slot * 1024, q0 + more * 128);
                            cp_async_16(ring + c_slot * 1024 + 512, q1 + more * 128);
                            cp_async_arrive(full + 8 * c_slot);
                        } else {
                            __syncwarp();
                            if (lane == 0) mbar_arrive(empty + 8 * c_slot);  // every lane has its weights
                        }
                        if (++c_slot == kRing) { c_slot = 0; c_phase ^= 1u; }
                    }
                    // Sums over the pair's eight lanes: the halves of the values are exchanged, over the same tree of lanes (4, 2, 1)
                    // whatever their number; lane kq ends with side kq >> 2 of some of the rows.
                    float* dst = reinterpret_cast<float*>(&parts[warp][pq][0]) + (kq >> 2);  // row r's sum at 2 r
                    auto halve = [&](float x0, float x1, int w) {  // x0 kept by the lower lane, x1 by the upper one
                        const bool up = kq & w;
                        const float send = up ? x0 : x1, keep = up ? x1 : x0;
                        return keep + __shfl_xor_sync(0xffffffffu, send, w);
                    };
                    if constexpr (kFew) {
                        const float s0 = halve(acc[0][0], acc[1][0], 4), s1 = halve(acc[0][1], acc[1][1], 4);
                        float t = halve(s0, s1, 2);
                        t += __shfl_xor_sync(0xffffffffu, t, 1);
                        dst[kq & 2] = t;  // (two lanes with the same value)
                    } else if constexpr (NR == 8) {
                        float s[8], t[4];
#pragma unroll
                        for (int i = 0; i < 8; ++i) s[i] = halve(acc[0][i], acc[1][i], 4);
#pragma unroll
                        for (int i = 0; i < 4; ++i) t[i] = halve(s[i], s[4 + i], 2);
#pragma unroll
                        for (int i = 0; i < 2; ++i) dst[2 * (2 * (kq & 3) + i)] = halve(t[i], t[2 + i], 1);
                    } else {
                        float s[16], t[8];
#pragma unroll
                        for (int i = 0; i < 16; ++i) s[i] = halve(acc[0][i], acc[1][i], 4);
#pragma unroll
                        for (int i = 0; i < 8; ++i) t[i] = halve(s[i], s[8 + i], 2);
#pragma unroll
                        for (int i = 0; i < 4; ++i) dst[2 * (4 * (kq & 3) + i)] = halve(t[i], t[4 + i], 1);
                    }
                }
                if (norm && round == 0 && kSW - 1 - warp < nr) {  // the rows' norm scales, by the warps that have the fewest units
                    const float* xr = sA + (kSW - 1 - warp) * 4;
                    float sq = 0.f;
#pragma unroll 4
                    for (int k = lane; k < K >> 2; k += 32) {
                        const float4 v = *reinterpret_cast<const float4*>(xr + k * pitch);
                        sq = __fmaf_rn(v.x, v.x, sq); sq = __fmaf_rn(v.y, v.y, sq); sq = __fmaf_rn(v.z, v.z, sq); sq = __fmaf_rn(v.w, v.w, sq);
                    }
#pragma unroll
                    for (int x = 16; x > 0; x >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, x);
                    if (lane == 0) s_rs[kSW - 1 - warp] = rsqrtf(sq / (float)K + d.rms_eps);
                }
                workers_sync();
                // ---- end of the units -----------------------------------------------------------------------------------------
                if (e_on && e_unit < n_units) {
                    float v0 = 0.f, v1 = 0.f;
                    const float2* part = &parts[e_slot << lg][e_pair][e_row];
#pragma unroll 1
                    for (int i0 = 0; i0 < 1 << lg; i0 += 8) {  // the unit's warps in column order
                        float2 x[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) x[i] = i0 + i < 1 << lg ? part[(i0 + i) * 4 * kSR] : make_float2(0.f, 0.f);
#pragma unroll
                        for (int i = 0; i < 8; ++i) { v0 += x[i].x; v1 += x[i].y; }
                    }
                    if (norm) { v0 *= s_rs[e_row]; v1 *= s_rs[e_row]; }
                    if (m == kOpQKV) {
                        float a0 = v0, a1 = v1;
                        if (e_mat < 2) { a0 = v0 * e0 - v1 * e1; a1 = v0 * e1 + v1 * e0; }
                        if (e_mat == 0) { v0 = a0; v1 = a1; }
                        const T c0 = from_f32<T>(a0), c1 = from_f32<T>(a1);
                        if (e_mat > 0) { a0 = to_f32<T>(c0); a1 = to_f32<T>(c1); }
                        ll_store(a.ll_qkv + e_at, a0, epoch); ll_store(a.ll_qkv + e_at + half, a1, epoch);
                        if (e_mat > 0) {
                            T* cache = reinterpret_cast<T*>(e_mat == 1 ? a.kcache : a.vcache) + e_cache;
                            cache[0] = c0; cache[half] = c1;
                        }
                        a.qkv[e_at] = v0; a.qkv[e_at + half] = v1;
                    } else if (m == kOpGateUp) {
                        const float v = v0 / (1.f + expf(-v0)) * v1;
                        ll_store(a.ll_h + e_at, v, epoch);
                        a.h[e_at] = v;
                    } else if (m != kOpHead) {
                        if (!(m == kOpO && op == kOpO)) {
                            ll_wait2(ex, a.ll_x + e_at, epoch - 2, up);  // the residual projection before this one
                            e0 = ll_values(ex).x; e1 = ll_values(ex).y;
                        }
                        ll_store2(a.ll_x + e_at, e0 + v0, e1 + v1, epoch);
                        *reinterpret_cast<float2*>(a.x + e_at) = make_float2(e0 + v0, e1 + v1);
                    } else {
                        const int p = 4 * e_unit + e_pair;
#pragma unroll
                        for (int s = 0; s < 2; ++s) {
                            const int n = 2 * p + s;
                            const float v = s ? v1 : v0;
                            if (n < d.vocab) {
                                if (a.logits) a.logits[e_at + s] = v;
                                if (v > best || (v == best && n < best_i)) { best = v; best_i = n; }
                            }
                        }
                    }
                }
                if (e_unit + step_units < n_units) fetch_end(e_unit + step_units);
            }
            if (m == kOpHead) {  // the CTA's (maximum, lowest index) of every row
                constexpr int kE = kFew ? kSW * 4 / 2 : 32;  // threads that hold one row's candidates
                static_assert(kE == 32 && kSW >= kSR && kST / 64 * 4 == 32, "a lane per (slot, pair), a warp per row");
                workers_sync();
                float* bv = reinterpret_cast<float*>(&s_part[0][0][0][0]);  // [32][rows]
                int* bi = reinterpret_cast<int*>(&s_part[1][0][0][0]);
                bv[tid] = best; bi[tid] = best_i;
                best = -INFINITY; best_i = 0x7fffffff;
                workers_sync();
                if (warp < nr) {
                    float v = bv[lane * (kFew ? 2 : 16) + warp];
                    int i = bi[lane * (kFew ? 2 : 16) + warp];
#pragma unroll
                    for (int w = 16; w > 0; w >>= 1) {
                        const float ov = __shfl_xor_sync(0xffffffffu, v, w);
                        const int oi = __shfl_xor_sync(0xffffffffu, i, w);
                        if (ov > v || (ov == v && oi < i)) { v = ov; i = oi; }
                    }
                    if (lane == 0) ll_store2(a.ll_part + 2 * ((int64_t)cta * d.row_cap + r0 + warp), v, __int_as_float(i), epoch);
                }
            }
            if (NR < kSR) break;
        }
    };

    uint32_t epoch0 = a.epoch;
#pragma unroll 1
    for (int step = 0; step < a.max_steps; ++step, epoch0 += simt_epochs(d)) {
        {
            const LLWord* w = ll_rows_of(a, epoch0);
#pragma unroll 1
            for (int r = tid; r < a.tail.n_rows; r += kST) {
                LL2 v[3];
                ll_fetch(v, epoch0, up, [&](int u) { return u == 2 ? w : w + 2 + 4 * r + 2 * u; });
                const LL2 &x = v[0], &y = v[1], &z = v[2];
                int tok = (int)(uint32_t)x.a;
                if (tok < 0 || tok >= d.vocab) {
                    if (cta == 0) atomicCAS(a.dev_err, kDevErrNone, kDevErrToken);  // (not over the mark of a CTA that has given up)
                    tok = 0;
                }
                R.tok[r] = tok; R.pos[r] = (int)(uint32_t)x.b; R.seq[r] = (int)(uint32_t)y.a; R.first[r] = (int)(uint32_t)y.b;
                if (r == 0) R.used = (int)(uint32_t)z.a;
            }
        }
        workers_sync();
        rows_used = R.used;

        if (rows_used == 0 || *up.failed) break;  // nothing left to do, or a wait ran out
        if (tid == 0 && a.passes > 1) {
            int n = 1;
            for (int r = pass; r < rows_used; r += pass) ++n;
            *(volatile int*)&s_passes[step & 1] = n;
            __threadfence_block();
            *(volatile int*)&s_steps = step + 1;
        }
#pragma unroll 1
        for (int op = 0; op < n_ops; ++op) {
            const int m = op == n_ops - 1 ? kOpHead : op & 3;
            const uint32_t epoch = epoch0 + op;  // what this projection writes
            if (m == kOpQKV && warp == 0) {  // cache rows of this CTA's part of the attention, on their way to L2
#pragma unroll 1
                for (int it = cta + lane * G; it < rows_used * d.n_heads; it += 32 * G) {
                    const int r = it / d.n_heads, n = R.pos[R.first[r]] * HD * (int)sizeof(T);
                    const int64_t at = kv_row_index(d, op >> 2, R.seq[r], it - r * d.n_heads, 0) * HD;
                    if (n > 0) {
                        l2_prefetch(reinterpret_cast<const T*>(a.kcache) + at, n);
                        l2_prefetch(reinterpret_cast<const T*>(a.vcache) + at, n);
                    }
                }
            }
            if (cta < a.geo[m].n_units) {
                if (rows_used <= 2) project(std::integral_constant<int, 2>{}, m, op, epoch);
                else if (rows_used <= min(8, pass)) project(std::integral_constant<int, 8>{}, m, op, epoch);
                else project(std::integral_constant<int, kSR>{}, m, op, epoch);
            }
            if (m == kOpQKV) {
                if (op == 0 && step > 0 && tid == 0 && !bar.wait(600ull * a.patience)) *up.failed = 1;  // the cache rows of the step before
                workers_sync();
#pragma unroll 1
                for (int it = cta; it < rows_used * d.n_heads; it += G) {
                    const int r = it / d.n_heads;
                    attend<T, HD>(a, R, op >> 2, it - r * d.n_heads, r, epoch, sA, up);
                }
            }
        }
        workers_sync();
        if (tid == 0 && !*up.failed) bar.arrive();
    }
    *(volatile int*)&s_stop = 1;
    if (tid == 0 && *up.failed) atomicExch(a.dev_err, kDevErrSteps);
}

// ---- host side -----------------------------------------------------------------------------------------------------
bool step_simt_shape(const ModelDims& d, bool bf16, int y_cap, int num_sms, SimtStep* s, size_t* smem) {
    const int k_max = d.d_model > d.d_ffn ? (d.d_model > d.hd_total ? d.d_model : d.hd_total)
                                          : (d.d_ffn > d.hd_total ? d.d_ffn : d.hd_total);
    if (num_sms < 2) return false;
    const size_t gains = (size_t)d.d_model * 4, ops = sizeof(SimtOp) * (4 * (size_t)d.n_layers + 1);
    const size_t es = bf16 ? 2 : 4, attend = d.head_dim * 4 + 2 * es * d.kp1 * d.head_dim + (size_t)kSW * (d.head_dim + 2) * 4;
    // as many rows per pass as there are and fit (they are multiplied in twos), passes of equal length
    const int bound = d.max_batch * d.kp1;
    int rows = bound < kSR ? (bound + 1) / 2 * 2 : kSR;
    while (rows > 0 && (size_t)(rows | 1) * k_max * 4 + kRingBytes + gains + ops > kStepSmem) rows -= 2;
    if (rows < 2) return false;
    const int passes = (bound + rows - 1) / rows;
    s->passes = passes;
    s->pass_rows = rows = ((bound + passes - 1) / passes + 1) / 2 * 2;
    size_t at = (size_t)(rows | 1) * k_max * 4;
    if (at < attend) at = attend;
    at = (at + 127) / 128 * 128;
    s->ring_offset = (int)at;
    s->gain_offset = (int)(at + kRingBytes);
    s->ops_offset = (int)(at + kRingBytes + gains);
    *smem = at + kRingBytes + gains + ops;
    // Polls take 0.6 us and more: 20 ms, and 2.5 ms per projection and pass, some thirty times what the slowest take.  A CTA may have
    // nothing to do for a whole step, so that is what the bound is made for.
    const long long polls = 32768 + 4096ll * (4 * d.n_layers + 1) * passes;
    s->patience = (int)(polls < 1 << 22 ? polls : 1 << 22);
    const size_t B = d.max_batch, tail = B * (8 + sizeof(SeqState) + 4) + 4 + ((size_t)d.row_cap + B * (3 * (size_t)d.max_ref + y_cap)) * 4;
    if (*smem < tail) *smem = (tail + 15) / 16 * 16;
    if (*smem > kStepSmem) return false;
    const int pairs[5] = {3 * d.hd_total / 2, d.d_model / 2, d.d_ffn, d.d_model / 2, (d.vocab + 1) / 2};
    const int ks[5] = {d.d_model, d.hd_total, d.d_model, d.d_ffn, d.d_model};
    for (int m = 0; m < 5; ++m) {
        SimtGeo& g = s->geo[m];
        g.n_units = (pairs[m] + 3) / 4; g.k_in = ks[m];
        g.n_pieces = ks[m] / (bf16 ? 64 : 32);
        g.sweep_rows = kSweep / ks[m]; g.sweep_cols = kSweep % ks[m];
        // Warps per unit: the fewest pieces in a row, counting a round of units as two pieces more
        const int here = (g.n_units + num_sms - 2) / (num_sms - 1);
        int best = 1 << 30;
        for (int lg = 1; lg <= 4; ++lg) {
            const int rounds = (here + (kSW >> lg) - 1) / (kSW >> lg), cost = rounds * (((g.n_pieces + (1 << lg) - 1) >> lg) + 2);
            if (cost < best) { best = cost; g.split_lg = lg; }
        }
    }
    return true;
}

template <typename T, int HD>
static cudaError_t init_typed(size_t smem, bool* fits) {
    cudaError_t e = cudaFuncSetAttribute(step_simt_kernel<T, HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStepSmem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, step_simt_kernel<T, HD>, kThreads, smem);
    *fits = per_sm >= 1;
    return e;
}
cudaError_t init_step_simt(bool bf16, int head_dim, size_t smem, bool* fits) {
    if (bf16) return head_dim == 128 ? init_typed<__nv_bfloat16, 128>(smem, fits) : init_typed<__nv_bfloat16, 64>(smem, fits);
    return head_dim == 128 ? init_typed<float, 128>(smem, fits) : init_typed<float, 64>(smem, fits);
}

template <typename T, int HD>
static cudaError_t launch_typed(cudaStream_t st, const SimtStep& s, size_t smem, int ctas) {
    void* args[] = {const_cast<SimtStep*>(&s)};
    // (Not a cooperative launch: while one waits for all of its SMs to come free at once, no other stream's CTAs start, and a kernel whose
    // CTAs wait for one another then waits for good.  A launch of these CTAs one by one that does not get them together gives up.)
    return cudaLaunchKernel(reinterpret_cast<const void*>(step_simt_kernel<T, HD>), dim3(ctas), dim3(kThreads), args, smem, st);
}
cudaError_t launch_step_simt(cudaStream_t st, bool bf16, const SimtStep& s, size_t smem, int ctas) {
    if (bf16) return s.dims.head_dim == 128 ? launch_typed<__nv_bfloat16, 128>(st, s, smem, ctas) : launch_typed<__nv_bfloat16, 64>(st, s, smem, ctas);
    return s.dims.head_dim == 128 ? launch_typed<float, 128>(st, s, smem, ctas) : launch_typed<float, 64>(st, s, smem, ctas);
}

}  // namespace llma
