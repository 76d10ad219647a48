// Split-KV causal attention for the k+1 query rows of a step (bf16 K/V cache).
//
// Grid (chunk, head, sequence).  A CTA owns 128 consecutive cache positions of one head:
// its K and V tiles arrive by TMA (128-byte swizzle) and are read ONCE for all the rows of
// the step, which is what makes verification of k+1 positions cost the K/V traffic of one.
// Each of the 4 warps takes 32 of the positions: S = Q K^T and O = P V on the tensor cores
// (mma.sync m16n8k16, bf16 in, fp32 accumulate), softmax statistics by warp shuffles.
// Q and P enter the MMAs as hi + lo bf16 pairs, so they keep 16 mantissa bits; Q is loaded
// from global memory directly into operand registers with all loads in flight at once, which
// keeps a CTA at 73 KB of shared memory: three CTAs per SM, one wave up to about 1.8 k cached
// positions at 32 heads.
#include <cuda.h>

#include "attention_frag.cuh"
#include "attention_mma.cuh"
#include "ptx_sm100.cuh"

namespace llma {

using namespace ptx;

template <int HD>
struct AttnSmem {
    static constexpr int kBoxes = HD / 64;                    // 64-column TMA boxes per K (or V) tile
    static constexpr uint32_t kBoxBytes = kAttnChunk * 128;   // 128 rows x 128 bytes
    static constexpr uint32_t kTileBytes = kBoxes * kBoxBytes;
    static constexpr uint32_t offK = 0, offV = kTileBytes;
    static constexpr uint32_t offO = 2 * kTileBytes;                     // fp32 [16][HD] merged tile
    static constexpr uint32_t offStat = offO + 16 * HD * 4;              // m_w[4][16], l_w[4][16], misc
    static constexpr uint32_t kBytes = offStat + 2 * 4 * 16 * 4 + 64;  // + barriers
};

template <int HD>
__global__ void __launch_bounds__(128, 3) attention_mma_kernel(const AttnArgs a, const __grid_constant__ CUtensorMap map_k,
                                                            const __grid_constant__ CUtensorMap map_v) {
    using L = AttnSmem<HD>;
    pdl_trigger();
    const int chunk = blockIdx.x, head = blockIdx.y, seq = blockIdx.z;
    // timeline (min, max over the CTAs): 0/1 CTA start, 2/3 dependency released, 4/5 K tile landed, 6/7 CTA end
    [[maybe_unused]] unsigned long long* stp = LLMA_STAMP_PTR(a.stamps, 300 + a.layer, 0);
    if (threadIdx.x == 0) LLMA_STAMP_MINMAX(stp, 0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const ModelDims& d = a.dims;
    const int c0 = chunk * kAttnChunk;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
    float* sO = reinterpret_cast<float*>(gbase + L::offO);
    float* s_m = reinterpret_cast<float*>(gbase + L::offStat);   // [4][16]
    float* s_l = s_m + 64;                                        // [4][16]
    uint64_t* bar = reinterpret_cast<uint64_t*>(s_l + 64);
    volatile uint32_t* flag = reinterpret_cast<volatile uint32_t*>(bar + 2);
    const uint32_t bar_u = smem_u32(bar), bar_v = bar_u + 8;  // K tile, V tile

    auto fetch_kv = [&]() {  // one thread
        const int32_t row0 = (int32_t)kv_row_index(d, a.layer, seq, head, c0);
        // K first, on a barrier of its own: S = Q K^T and the softmax run while V is still arriving
        mbar_arrive_expect_tx(bar_u, L::kTileBytes);
        for (int b = 0; b < L::kBoxes; ++b) tma_load_2d(base + L::offK + b * L::kBoxBytes, &map_k, bar_u, b * 64, row0);
        mbar_arrive_expect_tx(bar_v, L::kTileBytes);
        for (int b = 0; b < L::kBoxes; ++b) tma_load_2d(base + L::offV + b * L::kBoxBytes, &map_v, bar_v, b * 64, row0);
    };
    // A chunk that lies wholly below the length committed before this step cannot change during the step
    // (new K/V rows go to positions at or above that length), so its tiles are requested before waiting
    // for the QKV projection: the loads overlap that kernel's tail.
    // (kv_len as read here may be that of an earlier step: it only grows.)
    const int kv_len = __ldcg(&a.seq_state[seq].kv_len);
    const bool early = c0 + kAttnChunk <= kv_len;
    if (threadIdx.x == 0) {
        mbar_init(bar_u, 1); mbar_init(bar_v, 1); fence_mbar_init(); flag[0] = 0;
        if (early) fetch_kv();
    }
    pdl_wait();  // row descriptors, q and the K/V rows of this step come from the kernels before
    if (threadIdx.x == 0) LLMA_STAMP_MINMAX(stp, 2);
    // the chunk that holds position kv_len is needed by any row of the sequence: requested before the rows are known
    const bool fetched = early || c0 <= kv_len;
    if (!early && fetched && threadIdx.x == 0) fetch_kv();

    // rows of this sequence in the step: packed back to back, at consecutive positions up to maxpos
    const int first = __ldcg(&a.rows->seq_first[seq]), cnt = __ldcg(&a.rows->seq_cnt[seq]);
    const int maxpos = __ldcg(&a.rows->seq_maxpos[seq]);
    if (cnt == 0 || c0 > maxpos) {  // uniform over the CTA; tiles already requested must land before the CTA goes
        if (fetched && threadIdx.x == 0) { (void)mbar_wait(bar_u, 0); (void)mbar_wait(bar_v, 0); }
        return;
    }
    const int pos0 = maxpos - cnt + 1;  // position of the sequence's first row
    if (!fetched && threadIdx.x == 0) fetch_kv();
    // Q (this head, 16 of this sequence's rows) goes straight from global memory into the MMA's
    // A-operand registers as hi / lo bf16 pairs: lane (g, t) holds rows g and g + 8, columns
    // 16 ks + 2t, +1, +8, +9.  All loads are issued before any is used; rows past cnt are zero.
    const int g8 = lane >> 2, t4 = lane & 3;
    uint32_t qh[HD / 16][4], ql[HD / 16][4];
    auto load_q = [&](int mt) {
        const int r0 = mt * 16 + g8, r1 = r0 + 8;
        const int64_t ldq = 3 * (int64_t)d.hd_total;
        const float* q0 = a.qkv + (first + r0) * ldq + head * HD + 2 * t4;
        const float* q1 = q0 + 8 * ldq;
        float2 x[HD / 16][4];
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
            const float2 z = make_float2(0.f, 0.f);
            x[ks][0] = r0 < cnt ? __ldcg(reinterpret_cast<const float2*>(q0 + ks * 16)) : z;
            x[ks][1] = r1 < cnt ? __ldcg(reinterpret_cast<const float2*>(q1 + ks * 16)) : z;
            x[ks][2] = r0 < cnt ? __ldcg(reinterpret_cast<const float2*>(q0 + ks * 16 + 8)) : z;
            x[ks][3] = r1 < cnt ? __ldcg(reinterpret_cast<const float2*>(q1 + ks * 16 + 8)) : z;
        }
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
#pragma unroll
            for (int i = 0; i < 4; ++i) split_pack(x[ks][i].x, x[ks][i].y, qh[ks][i], ql[ks][i]);
        }
    };
    // The first tile's rows go through shared memory: the CTA fetches them as whole 16-byte accesses (a few per thread
    // instead of 32 eight-byte loads per lane, which filled the load/store queues once a sequence had more than a
    // row or two) into the buffer that later holds the merged tile, columns XOR-ed by (row & 3) * 8 so that the fragment
    // reads of a half-warp (four rows) fall into different banks.  With one or two rows the direct loads are few and
    // spare the barrier.
    if (cnt <= 2) {
        load_q(0);
    } else {
        float* sQ = sO;
        const int64_t ldq = 3 * (int64_t)d.hd_total;
        for (int idx = threadIdx.x; idx < 16 * (HD / 4); idx += blockDim.x) {
            const int r = idx / (HD / 4), c4 = idx - r * (HD / 4);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r < cnt) v = __ldcg(reinterpret_cast<const float4*>(a.qkv + (first + r) * ldq + head * HD) + c4);
            *reinterpret_cast<float4*>(sQ + r * HD + ((c4 * 4) ^ ((r & 3) << 3))) = v;
        }
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int row = (i & 1) ? g8 + 8 : g8;
                const int col = ks * 16 + 2 * t4 + ((i >> 1) ? 8 : 0);
                const float2 x = *reinterpret_cast<const float2*>(sQ + row * HD + (col ^ ((row & 3) << 3)));
                split_pack(x.x, x.y, qh[ks][i], ql[ks][i]);
            }
        }
    }
    if (threadIdx.x == 0) {
        const bool ok = mbar_wait(bar_u, 0);
        if (!ok) { atomicExch(a.dev_err, kDevErrTimeout); flag[0] = 1; }
    }
    __syncthreads();
    if (flag[0]) return;  // the copy never landed: give up (error word is set)
    if (threadIdx.x == 0) LLMA_STAMP_MINMAX(stp, 4);

    const float scale = rsqrtf((float)HD);
    const int n_mt = (cnt + 15) >> 4;
    const int wpos0 = warp * 32;  // this warp's positions inside the chunk
    // chunk partials are indexed by the row's slot in the step: [head][chunk][row][HD]
    const int64_t part_base = ((int64_t)head * a.n_chunks + chunk) * d.row_cap + first;

    for (int mt = 0; mt < n_mt; ++mt) {
        if (mt > 0) load_q(mt);
        // ---------------- S = Q K^T over this warp's 32 positions ----------------------------
        float s[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { s[i][0] = s[i][1] = s[i][2] = s[i][3] = 0.f; }
        const int mi = lane >> 3, t8 = lane & 7;
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
            const uint32_t (&ah)[4] = qh[ks];
            const uint32_t (&al)[4] = ql[ks];
#pragma unroll
            for (int np = 0; np < 2; ++np) {
                const int row = wpos0 + np * 16 + (mi >> 1) * 8 + t8;
                const int col = ks * 16 + (mi & 1) * 8;
                const uint32_t kaddr = base + L::offK + (uint32_t)(col >> 6) * L::kBoxBytes + (uint32_t)row * 128 +
                                       ((((uint32_t)(col & 63) >> 3) ^ ((uint32_t)row & 7u)) << 4);
                uint32_t b[4];
                ldsm_x4(kaddr, b);
                mma_bf16(s[2 * np], ah, b[0], b[1]);
                mma_bf16(s[2 * np], al, b[0], b[1]);
                mma_bf16(s[2 * np + 1], ah, b[2], b[3]);
                mma_bf16(s[2 * np + 1], al, b[2], b[3]);
            }
        }
        // ---------------- causal mask, softmax statistics of the warp's span --------------------
        const int r_lo = mt * 16 + (lane >> 2), r_hi = r_lo + 8;
        const int lim_lo = r_lo < cnt ? pos0 + r_lo : -1;
        const int lim_hi = r_hi < cnt ? pos0 + r_hi : -1;
        float m_lo = -INFINITY, m_hi = -INFINITY;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int p = c0 + wpos0 + nt * 8 + 2 * (lane & 3) + (e & 1);
                const int lim = e < 2 ? lim_lo : lim_hi;
                const float v = p <= lim ? s[nt][e] * scale : -INFINITY;
                s[nt][e] = v;
                if (e < 2) m_lo = fmaxf(m_lo, v); else m_hi = fmaxf(m_hi, v);
            }
        }
        m_lo = fmaxf(m_lo, __shfl_xor_sync(0xffffffffu, m_lo, 1)); m_lo = fmaxf(m_lo, __shfl_xor_sync(0xffffffffu, m_lo, 2));
        m_hi = fmaxf(m_hi, __shfl_xor_sync(0xffffffffu, m_hi, 1)); m_hi = fmaxf(m_hi, __shfl_xor_sync(0xffffffffu, m_hi, 2));
        const float ref_lo = m_lo == -INFINITY ? 0.f : m_lo, ref_hi = m_hi == -INFINITY ? 0.f : m_hi;
        float l_lo = 0.f, l_hi = 0.f;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float pe = expf(s[nt][e] - (e < 2 ? ref_lo : ref_hi));  // exp(-inf) = 0 for masked positions
                s[nt][e] = pe;
                if (e < 2) l_lo += pe; else l_hi += pe;
            }
        }
        l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1); l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
        l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1); l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);

        // ---------------- O = P V ----------------------------------------------------------------
        if (mt == 0) {
            if (threadIdx.x == 0 && !mbar_wait(bar_v, 0)) { atomicExch(a.dev_err, kDevErrTimeout); flag[0] = 1; }
            __syncthreads();
            if (flag[0]) return;  // uniform: the copy never landed (error word is set)
        }
        float o[HD / 8][4];
#pragma unroll
        for (int i = 0; i < HD / 8; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
#pragma unroll
        for (int kp = 0; kp < 2; ++kp) {
            uint32_t ph[4], pl[4];
            split_pack(s[2 * kp][0], s[2 * kp][1], ph[0], pl[0]);
            split_pack(s[2 * kp][2], s[2 * kp][3], ph[1], pl[1]);
            split_pack(s[2 * kp + 1][0], s[2 * kp + 1][1], ph[2], pl[2]);
            split_pack(s[2 * kp + 1][2], s[2 * kp + 1][3], ph[3], pl[3]);
#pragma unroll
            for (int nn = 0; nn < HD / 16; ++nn) {
                const int row = wpos0 + kp * 16 + (mi & 1) * 8 + t8;
                const int col = nn * 16 + (mi >> 1) * 8;
                const uint32_t vaddr = base + L::offV + (uint32_t)(col >> 6) * L::kBoxBytes + (uint32_t)row * 128 +
                                       ((((uint32_t)(col & 63) >> 3) ^ ((uint32_t)row & 7u)) << 4);
                uint32_t b[4];
                ldsm_x4_trans(vaddr, b);
                mma_bf16(o[2 * nn], ph, b[0], b[1]);
                mma_bf16(o[2 * nn], pl, b[0], b[1]);
                mma_bf16(o[2 * nn + 1], ph, b[2], b[3]);
                mma_bf16(o[2 * nn + 1], pl, b[2], b[3]);
            }
        }
        // ---------------- merge the 4 warps in warp order, chunk partial -> workspace -----------------
        if ((lane & 3) == 0) {
            s_m[warp * 16 + (lane >> 2)] = m_lo; s_m[warp * 16 + (lane >> 2) + 8] = m_hi;
            s_l[warp * 16 + (lane >> 2)] = l_lo; s_l[warp * 16 + (lane >> 2) + 8] = l_hi;
        }
        const int rows_here = min(16, cnt - mt * 16);
        if (n_mt == 1) {
            // The K tile is dead (every warp passed the barrier after its scores): each warp parks its
            // unscaled partial there, [warp][16 rows][HD] with the column XOR-ed by (row & 3) * 8 so that
            // neither the stores nor the float4 reads below conflict; then all threads combine the four
            // partials of their elements in warp order and write the chunk's partial straight to global memory.
            float* buf = reinterpret_cast<float*>(gbase + L::offK) + warp * 16 * HD;
#pragma unroll
            for (int nt = 0; nt < HD / 8; ++nt) {
                const int col = nt * 8 + 2 * t4;
                *reinterpret_cast<float2*>(buf + g8 * HD + (col ^ ((g8 & 3) << 3))) = make_float2(o[nt][0], o[nt][1]);
                *reinterpret_cast<float2*>(buf + (g8 + 8) * HD + (col ^ ((g8 & 3) << 3))) = make_float2(o[nt][2], o[nt][3]);
            }
            __syncthreads();
            const float* all = reinterpret_cast<const float*>(gbase + L::offK);
            for (int e = threadIdx.x; e < rows_here * (HD / 4); e += blockDim.x) {
                const int r = e / (HD / 4), c4 = e - r * (HD / 4);
                float M = -INFINITY;
#pragma unroll
                for (int w = 0; w < 4; ++w) M = fmaxf(M, s_m[w * 16 + r]);
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const float mw = s_m[w * 16 + r];
                    const float f = mw == -INFINITY ? 0.f : expf(mw - M);
                    const float4 v = *reinterpret_cast<const float4*>(all + (w * 16 + r) * HD + ((c4 * 4) ^ ((r & 3) << 3)));
                    if (w == 0) {
                        acc = make_float4(__fmul_rn(f, v.x), __fmul_rn(f, v.y), __fmul_rn(f, v.z), __fmul_rn(f, v.w));
                    } else {
                        acc.x = __fmaf_rn(f, v.x, acc.x); acc.y = __fmaf_rn(f, v.y, acc.y);
                        acc.z = __fmaf_rn(f, v.z, acc.z); acc.w = __fmaf_rn(f, v.w, acc.w);
                    }
                }
                *reinterpret_cast<float4*>(a.ws_o + (part_base + r) * HD + c4 * 4) = acc;
            }
        } else {
            // several 16-row tiles share the K and V tiles: accumulate in a buffer of its own, warp by warp
            // (the same products and fused multiply-adds as above, so a row's bits do not depend on the path)
            __syncthreads();
            float M_lo = -INFINITY, M_hi = -INFINITY;
#pragma unroll
            for (int w = 0; w < 4; ++w) { M_lo = fmaxf(M_lo, s_m[w * 16 + (lane >> 2)]); M_hi = fmaxf(M_hi, s_m[w * 16 + (lane >> 2) + 8]); }
            const float f_lo = m_lo == -INFINITY ? 0.f : expf(m_lo - M_lo);
            const float f_hi = m_hi == -INFINITY ? 0.f : expf(m_hi - M_hi);
            for (int w = 0; w < 4; ++w) {
                if (warp == w) {
#pragma unroll
                    for (int nt = 0; nt < HD / 8; ++nt) {
                        float* p_lo = sO + (lane >> 2) * HD + nt * 8 + 2 * (lane & 3);
                        float* p_hi = p_lo + 8 * HD;
                        if (w == 0) {
                            p_lo[0] = __fmul_rn(f_lo, o[nt][0]); p_lo[1] = __fmul_rn(f_lo, o[nt][1]);
                            p_hi[0] = __fmul_rn(f_hi, o[nt][2]); p_hi[1] = __fmul_rn(f_hi, o[nt][3]);
                        } else {
                            p_lo[0] = __fmaf_rn(f_lo, o[nt][0], p_lo[0]); p_lo[1] = __fmaf_rn(f_lo, o[nt][1], p_lo[1]);
                            p_hi[0] = __fmaf_rn(f_hi, o[nt][2], p_hi[0]); p_hi[1] = __fmaf_rn(f_hi, o[nt][3], p_hi[1]);
                        }
                    }
                }
                __syncthreads();
            }
            for (int idx = threadIdx.x; idx < rows_here * HD; idx += blockDim.x) {
                const int r = idx / HD, i = idx - r * HD;
                a.ws_o[(part_base + mt * 16 + r) * HD + i] = sO[r * HD + i];
            }
        }
        if (threadIdx.x < rows_here) {
            const int r = threadIdx.x;
            float M = -INFINITY;
            for (int w = 0; w < 4; ++w) M = fmaxf(M, s_m[w * 16 + r]);
            float lsum = 0.f;
            for (int w = 0; w < 4; ++w) {
                const float mw = s_m[w * 16 + r];
                lsum += mw == -INFINITY ? 0.f : expf(mw - M) * s_l[w * 16 + r];
            }
            a.ws_ml[(part_base + mt * 16 + r) * 2] = M;
            a.ws_ml[(part_base + mt * 16 + r) * 2 + 1] = lsum;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) LLMA_STAMP_MINMAX(stp, 6);
}

// Long contexts, many sequences: a CTA takes kT consecutive 128-position tiles of one (sequence, head) instead of one,
// so that the chunk partials (and the merge pass over them) shrink by kT and the next tile's K and V are already on
// their way while the current one is being multiplied.  Each warp keeps its 32-position slice's running maximum, sum
// and output across the tiles; the four warps are combined once, at the end, exactly as in attention_mma_kernel.
// For steps of at most 16 rows per sequence; which kT an engine uses depends on its capacity only (never on the step).
template <int HD, int kT>
__global__ void __launch_bounds__(128, 3) attention_long_kernel(const AttnArgs a, const __grid_constant__ CUtensorMap map_k,
                                                             const __grid_constant__ CUtensorMap map_v) {
    using L = AttnSmem<HD>;
    pdl_trigger();
    const int chunk = blockIdx.x, head = blockIdx.y, seq = blockIdx.z;
    [[maybe_unused]] unsigned long long* stp = LLMA_STAMP_PTR(a.stamps, 300 + a.layer, 0);
    if (threadIdx.x == 0) LLMA_STAMP_MINMAX(stp, 0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const ModelDims& d = a.dims;
    const int c0 = chunk * kAttnChunk * kT;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
    float* sO = reinterpret_cast<float*>(gbase + L::offO);
    float* s_m = reinterpret_cast<float*>(gbase + L::offStat);   // [4][16]
    float* s_l = s_m + 64;                                        // [4][16]
    uint64_t* bar = reinterpret_cast<uint64_t*>(s_l + 64);
    volatile uint32_t* flag = reinterpret_cast<volatile uint32_t*>(bar + 2);
    const uint32_t bar_u = smem_u32(bar), bar_v = bar_u + 8;  // K tile, V tile

    // (rows that come through once per step, 67 MB and more a layer: see l2_evict_first; sixteen 7B-shaped sequences of 4096 positions 33.6 -> 32.0 ms,
    // where one sequence's rows in attention_mma_kernel are better left alone, 64.2 against 64.7)
    auto fetch_k = [&](int t) {  // one thread
        const int32_t row0 = (int32_t)kv_row_index(d, a.layer, seq, head, c0 + t * kAttnChunk);
        mbar_arrive_expect_tx(bar_u, L::kTileBytes);
        for (int b = 0; b < L::kBoxes; ++b) tma_load_2d(base + L::offK + b * L::kBoxBytes, &map_k, bar_u, b * 64, row0, l2_evict_first());
    };
    auto fetch_v = [&](int t) {
        const int32_t row0 = (int32_t)kv_row_index(d, a.layer, seq, head, c0 + t * kAttnChunk);
        mbar_arrive_expect_tx(bar_v, L::kTileBytes);
        for (int b = 0; b < L::kBoxes; ++b) tma_load_2d(base + L::offV + b * L::kBoxBytes, &map_v, bar_v, b * 64, row0, l2_evict_first());
    };
    // the first tile may be requested before the QKV projection has finished if it lies wholly below the committed length
    const int kv_len = __ldcg(&a.seq_state[seq].kv_len);
    const bool early = c0 + kAttnChunk <= kv_len;
    if (threadIdx.x == 0) {
        mbar_init(bar_u, 1); mbar_init(bar_v, 1); fence_mbar_init(); flag[0] = 0;
        if (early) { fetch_k(0); fetch_v(0); }
    }
    pdl_wait();
    if (threadIdx.x == 0) LLMA_STAMP_MINMAX(stp, 2);
    const bool fetched = early || c0 <= kv_len;
    if (!early && fetched && threadIdx.x == 0) { fetch_k(0); fetch_v(0); }

    const int first = __ldcg(&a.rows->seq_first[seq]), cnt = __ldcg(&a.rows->seq_cnt[seq]);
    const int maxpos = __ldcg(&a.rows->seq_maxpos[seq]);
    if (cnt == 0 || c0 > maxpos) {
        if (fetched && threadIdx.x == 0) { (void)mbar_wait(bar_u, 0); (void)mbar_wait(bar_v, 0); }
        return;
    }
    if (cnt > 16) {  // not this kernel's case: the host never launches it for such steps
        if (threadIdx.x == 0) {
            atomicExch(a.dev_err, kDevErrCapacity);
            if (fetched) { (void)mbar_wait(bar_u, 0); (void)mbar_wait(bar_v, 0); }
        }
        return;
    }
    const int pos0 = maxpos - cnt + 1;
    if (!fetched && threadIdx.x == 0) { fetch_k(0); fetch_v(0); }
    const int n_tiles = min(kT, (maxpos - c0) / kAttnChunk + 1);  // tiles that hold a position some row attends to

    const int g8 = lane >> 2, t4 = lane & 3;
    uint32_t qh[HD / 16][4], ql[HD / 16][4];
    {   // the step's rows of q for this head through shared memory (see attention_mma_kernel)
        float* sQ = sO;
        const int64_t ldq = 3 * (int64_t)d.hd_total;
        for (int idx = threadIdx.x; idx < 16 * (HD / 4); idx += blockDim.x) {
            const int r = idx / (HD / 4), c4 = idx - r * (HD / 4);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r < cnt) v = __ldcg(reinterpret_cast<const float4*>(a.qkv + (first + r) * ldq + head * HD) + c4);
            *reinterpret_cast<float4*>(sQ + r * HD + ((c4 * 4) ^ ((r & 3) << 3))) = v;
        }
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int row = (i & 1) ? g8 + 8 : g8;
                const int col = ks * 16 + 2 * t4 + ((i >> 1) ? 8 : 0);
                const float2 x = *reinterpret_cast<const float2*>(sQ + row * HD + (col ^ ((row & 3) << 3)));
                split_pack(x.x, x.y, qh[ks][i], ql[ks][i]);
            }
        }
    }
    const float scale = rsqrtf((float)HD);
    const int wpos0 = warp * 32;
    const int mi = lane >> 3, t8 = lane & 7;
    const int r_lo = g8, r_hi = g8 + 8;
    const int lim_lo = r_lo < cnt ? pos0 + r_lo : -1;
    const int lim_hi = r_hi < cnt ? pos0 + r_hi : -1;
    float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;
    float o[HD / 8][4];
#pragma unroll
    for (int i = 0; i < HD / 8; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }

#pragma unroll 1
    for (int t = 0; t < n_tiles; ++t) {
        const uint32_t par = (uint32_t)(t & 1);
        if (threadIdx.x == 0 && !mbar_wait(bar_u, par)) { atomicExch(a.dev_err, kDevErrTimeout); flag[0] = 1; }
        __syncthreads();
        if (flag[0]) break;  // uniform; what is still in flight is awaited below
        if (t == 0 && threadIdx.x == 0) LLMA_STAMP_MINMAX(stp, 4);
        float sc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { sc[i][0] = sc[i][1] = sc[i][2] = sc[i][3] = 0.f; }
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
            const uint32_t (&ah)[4] = qh[ks];
            const uint32_t (&al)[4] = ql[ks];
#pragma unroll
            for (int np = 0; np < 2; ++np) {
                const int row = wpos0 + np * 16 + (mi >> 1) * 8 + t8;
                const int col = ks * 16 + (mi & 1) * 8;
                const uint32_t kaddr = base + L::offK + (uint32_t)(col >> 6) * L::kBoxBytes + (uint32_t)row * 128 +
                                       ((((uint32_t)(col & 63) >> 3) ^ ((uint32_t)row & 7u)) << 4);
                uint32_t b[4];
                ldsm_x4(kaddr, b);
                mma_bf16(sc[2 * np], ah, b[0], b[1]);
                mma_bf16(sc[2 * np], al, b[0], b[1]);
                mma_bf16(sc[2 * np + 1], ah, b[2], b[3]);
                mma_bf16(sc[2 * np + 1], al, b[2], b[3]);
            }
        }
        __syncthreads();  // every warp has read the K tile: the next one may land in it
        if (threadIdx.x == 0 && t + 1 < n_tiles) fetch_k(t + 1);
        const int p0 = c0 + t * kAttnChunk + wpos0;
        float bm_lo = -INFINITY, bm_hi = -INFINITY;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int p = p0 + nt * 8 + 2 * (lane & 3) + (e & 1);
                const int lim = e < 2 ? lim_lo : lim_hi;
                const float v = p <= lim ? sc[nt][e] * scale : -INFINITY;
                sc[nt][e] = v;
                if (e < 2) bm_lo = fmaxf(bm_lo, v); else bm_hi = fmaxf(bm_hi, v);
            }
        }
        bm_lo = fmaxf(bm_lo, __shfl_xor_sync(0xffffffffu, bm_lo, 1)); bm_lo = fmaxf(bm_lo, __shfl_xor_sync(0xffffffffu, bm_lo, 2));
        bm_hi = fmaxf(bm_hi, __shfl_xor_sync(0xffffffffu, bm_hi, 1)); bm_hi = fmaxf(bm_hi, __shfl_xor_sync(0xffffffffu, bm_hi, 2));
        const float n_lo = fmaxf(m_lo, bm_lo), n_hi = fmaxf(m_hi, bm_hi);
        const float ref_lo = n_lo == -INFINITY ? 0.f : n_lo, ref_hi = n_hi == -INFINITY ? 0.f : n_hi;
        const float f_lo = m_lo == -INFINITY ? 0.f : expf(m_lo - ref_lo);
        const float f_hi = m_hi == -INFINITY ? 0.f : expf(m_hi - ref_hi);
        float bl_lo = 0.f, bl_hi = 0.f;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float pe = expf(sc[nt][e] - (e < 2 ? ref_lo : ref_hi));
                sc[nt][e] = pe;
                if (e < 2) bl_lo += pe; else bl_hi += pe;
            }
        }
        bl_lo += __shfl_xor_sync(0xffffffffu, bl_lo, 1); bl_lo += __shfl_xor_sync(0xffffffffu, bl_lo, 2);
        bl_hi += __shfl_xor_sync(0xffffffffu, bl_hi, 1); bl_hi += __shfl_xor_sync(0xffffffffu, bl_hi, 2);
        l_lo = __fmaf_rn(l_lo, f_lo, bl_lo); l_hi = __fmaf_rn(l_hi, f_hi, bl_hi);
        m_lo = n_lo; m_hi = n_hi;
#pragma unroll
        for (int i = 0; i < HD / 8; ++i) { o[i][0] *= f_lo; o[i][1] *= f_lo; o[i][2] *= f_hi; o[i][3] *= f_hi; }
        if (threadIdx.x == 0 && !mbar_wait(bar_v, par)) { atomicExch(a.dev_err, kDevErrTimeout); flag[0] = 1; }
        __syncthreads();
        if (flag[0]) break;
#pragma unroll
        for (int kp = 0; kp < 2; ++kp) {
            uint32_t ph[4], pl[4];
            split_pack(sc[2 * kp][0], sc[2 * kp][1], ph[0], pl[0]);
            split_pack(sc[2 * kp][2], sc[2 * kp][3], ph[1], pl[1]);
            split_pack(sc[2 * kp + 1][0], sc[2 * kp + 1][1], ph[2], pl[2]);
            split_pack(sc[2 * kp + 1][2], sc[2 * kp + 1][3], ph[3], pl[3]);
#pragma unroll
            for (int nn = 0; nn < HD / 16; ++nn) {
                const int row = wpos0 + kp * 16 + (mi & 1) * 8 + t8;
                const int col = nn * 16 + (mi >> 1) * 8;
                const uint32_t vaddr = base + L::offV + (uint32_t)(col >> 6) * L::kBoxBytes + (uint32_t)row * 128 +
                                       ((((uint32_t)(col & 63) >> 3) ^ ((uint32_t)row & 7u)) << 4);
                uint32_t b[4];
                ldsm_x4_trans(vaddr, b);
                mma_bf16(o[2 * nn], ph, b[0], b[1]);
                mma_bf16(o[2 * nn], pl, b[0], b[1]);
                mma_bf16(o[2 * nn + 1], ph, b[2], b[3]);
                mma_bf16(o[2 * nn + 1], pl, b[2], b[3]);
            }
        }
        __syncthreads();  // every warp has read the V tile
        if (threadIdx.x == 0 && t + 1 < n_tiles) fetch_v(t + 1);
    }
    if (flag[0]) {
        // a copy never landed (error word is set): the K copy of the next tile may still be in flight
        if (threadIdx.x == 0) {
            (void)mbar_wait(bar_u, 0, 100000000ull); (void)mbar_wait(bar_u, 1, 100000000ull);
            (void)mbar_wait(bar_v, 0, 100000000ull); (void)mbar_wait(bar_v, 1, 100000000ull);
        }
        return;
    }
    // ---------------- the four warps' (max, sum, output) combined in warp order -> the chunk's partial ----------------
    const int64_t part_base = ((int64_t)head * a.n_chunks + chunk) * d.row_cap + first;
    if ((lane & 3) == 0) {
        s_m[warp * 16 + g8] = m_lo; s_m[warp * 16 + g8 + 8] = m_hi;
        s_l[warp * 16 + g8] = l_lo; s_l[warp * 16 + g8 + 8] = l_hi;
    }
    {
        float* buf = reinterpret_cast<float*>(gbase + L::offK) + warp * 16 * HD;  // the K tile is dead
#pragma unroll
        for (int nt = 0; nt < HD / 8; ++nt) {
            const int col = nt * 8 + 2 * t4;
            *reinterpret_cast<float2*>(buf + g8 * HD + (col ^ ((g8 & 3) << 3))) = make_float2(o[nt][0], o[nt][1]);
            *reinterpret_cast<float2*>(buf + (g8 + 8) * HD + (col ^ ((g8 & 3) << 3))) = make_float2(o[nt][2], o[nt][3]);
        }
        __syncthreads();
        const float* all = reinterpret_cast<const float*>(gbase + L::offK);
        for (int e = threadIdx.x; e < cnt * (HD / 4); e += blockDim.x) {
            const int r = e / (HD / 4), c4 = e - r * (HD / 4);
            float M = -INFINITY;
#pragma unroll
            for (int w = 0; w < 4; ++w) M = fmaxf(M, s_m[w * 16 + r]);
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const float mw = s_m[w * 16 + r];
                const float f = mw == -INFINITY ? 0.f : expf(mw - M);
                const float4 v = *reinterpret_cast<const float4*>(all + (w * 16 + r) * HD + ((c4 * 4) ^ ((r & 3) << 3)));
                if (w == 0) {
                    acc = make_float4(__fmul_rn(f, v.x), __fmul_rn(f, v.y), __fmul_rn(f, v.z), __fmul_rn(f, v.w));
                } else {
                    acc.x = __fmaf_rn(f, v.x, acc.x); acc.y = __fmaf_rn(f, v.y, acc.y);
                    acc.z = __fmaf_rn(f, v.z, acc.z); acc.w = __fmaf_rn(f, v.w, acc.w);
                }
            }
            *reinterpret_cast<float4*>(a.ws_o + (part_base + r) * HD + c4 * 4) = acc;
        }
    }
    if (threadIdx.x < cnt) {
        const int r = threadIdx.x;
        float M = -INFINITY;
        for (int w = 0; w < 4; ++w) M = fmaxf(M, s_m[w * 16 + r]);
        float lsum = 0.f;
        for (int w = 0; w < 4; ++w) {
            const float mw = s_m[w * 16 + r];
            lsum += mw == -INFINITY ? 0.f : expf(mw - M) * s_l[w * 16 + r];
        }
        a.ws_ml[(part_base + r) * 2] = M;
        a.ws_ml[(part_base + r) * 2 + 1] = lsum;
    }
    if (threadIdx.x == 0) LLMA_STAMP_MINMAX(stp, 6);
}

// Second pass: one warp per (head, row) combines the row's chunk partials in ascending chunk
// order.  A kernel of its own, so that every head is merged at once instead of by whichever CTA of the
// head happened to finish last; a row's result still depends on its own position only.
template <int HD>
__global__ void __launch_bounds__(128) attention_merge_kernel(const AttnArgs a) {
    pdl_trigger();
    // timeline (min, max over the warps): 2/3 dependency released, 6/7 warp end
    [[maybe_unused]] unsigned long long* stp = LLMA_STAMP_PTR(a.stamps, 400 + a.layer, 0);
    extern __shared__ float s_w[];  // [4 warps][n_chunks] weights, then [4][n_chunks] weighted sums
    const int head = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const ModelDims& d = a.dims;
    const int r = blockIdx.y * 4 + warp;  // row slot of the step (below the pass's row slots: they come in fours)
    const int64_t head_base = (int64_t)head * a.n_chunks * d.row_cap;
    float* w_c = s_w + warp * a.n_chunks;
    float* wl_c = s_w + (4 + warp) * a.n_chunks;
    // The first CTAs take a turn that loads and stores nothing before they wait: a warp runs this code once, and fetching its
    // instructions would otherwise stand on the path between the attention kernel and the output projection (three layers
    // of width 512 at up to six rows: 116.5 -> 114.9 us per pass; two of width 1024, sixteen sequences: 173.7 -> 171.0; four
    // of the 7B widths, sixteen sequences: 1360 -> 1343; one 7B sequence, whose attention CTAs fill the SMs until they end: no
    // difference).  CTAs past the first wave start when there is nothing left to wait for.
    constexpr int kFirstWave = 512;
    int turn;
    asm volatile("mov.s32 %0, %1;" : "=r"(turn) : "r"((int)(blockIdx.y * gridDim.x + blockIdx.x) < kFirstWave ? 0 : 1));  // (opaque: one copy of the code)
#pragma unroll 1
    for (; turn < 2; ++turn) {
        const bool live = turn == 1;
        if (live) {
            pdl_wait();
            if (lane == 0) LLMA_STAMP_MINMAX(stp, 2);
        }
        constexpr int kB = 8;  // partials requested together
        // The kernel is a chain of dependent loads, so everything whose address is known is requested at once:
        // the row's position, the (max, sum) pairs of every chunk slot and the first sixteen chunk partials.
        // Slots past the row's last chunk hold older (finite) values; they are read but never used.
        const int rows_used = live ? __ldcg(&a.rows->rows_used) : r + 1;
        const int pos = live ? __ldcg(&a.rows->pos[r]) : (min(a.n_chunks, 2 * kB) - 1) * a.chunk_pos;
        // a step shaped for many rows (batched decoding) usually uses a fraction of its row slots: there a warp first
        // learns whether its slot is in use, at the price of one more round trip for those that are
        if (a.n_rows > 32 && (r >= rows_used || pos < 0)) return;
        const float4* src = reinterpret_cast<const float4*>(a.ws_o + (head_base + r) * HD) + (lane < HD / 4 ? lane : 0);
        float2 ml[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int c = lane + 32 * u;
            ml[u] = live && c < a.n_chunks ? __ldcg(reinterpret_cast<const float2*>(a.ws_ml) + head_base + (int64_t)c * d.row_cap + r)
                                           : make_float2(0.f, 0.f);
        }
        float4 p[2][kB];
#pragma unroll
        for (int u = 0; u < 2 * kB; ++u)
            p[u / kB][u % kB] = live ? __ldcg(src + (int64_t)min(u, a.n_chunks - 1) * d.row_cap * (HD / 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (r >= rows_used || pos < 0) return;
        const int nc = pos / a.chunk_pos + 1;
        float M = -INFINITY;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int c = lane + 32 * u;
            if (c < nc) { w_c[c] = ml[u].x; wl_c[c] = ml[u].y; M = fmaxf(M, ml[u].x); }
        }
#pragma unroll 1
        for (int c = lane + 64; c < nc; c += 32) {  // contexts beyond 64 chunks
            const float2 m2 = __ldcg(reinterpret_cast<const float2*>(a.ws_ml) + head_base + (int64_t)c * d.row_cap + r);
            w_c[c] = m2.x; wl_c[c] = m2.y;
            M = fmaxf(M, m2.x);
        }
        for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        __syncwarp();
#pragma unroll 1
        for (int c = lane; c < nc; c += 32) {
            const float mc = w_c[c];
            const float f = mc == -INFINITY ? 0.f : expf(mc - M);
            w_c[c] = f; wl_c[c] = f * wl_c[c];
        }
        __syncwarp();
        float den = 0.f;
#pragma unroll 4
        for (int c = 0; c < nc; ++c) den += wl_c[c];  // ascending order, the same in every lane
        if (lane < HD / 4) {
            float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
            for (int c0 = 0; c0 < nc; c0 += 2 * kB) {  // two batches in registers: the next ones are requested as these are used
#pragma unroll
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int u = 0; u < kB; ++u) {
                        const int c = c0 + h * kB + u;
                        if (c < nc) {
                            const float f = w_c[c];
                            num.x += f * p[h][u].x; num.y += f * p[h][u].y; num.z += f * p[h][u].z; num.w += f * p[h][u].w;
                        }
                        if (c + 2 * kB < nc) p[h][u] = __ldcg(src + (int64_t)(c + 2 * kB) * d.row_cap * (HD / 4));
                    }
                }
            }
            const int64_t col = (int64_t)head * HD + lane * 4;
            const float inv = 1.f / den;
            uint32_t h0, l0, h1, l1;
            split_pack(num.x * inv, num.y * inv, h0, l0);
            split_pack(num.z * inv, num.w * inv, h1, l1);
            __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(a.attn_out) + (int64_t)r * d.hd_total + col;
            if (live) {
                *reinterpret_cast<uint2*>(dst) = make_uint2(h0, h1);
                *reinterpret_cast<uint2*>(dst + (int64_t)d.row_cap * d.hd_total) = make_uint2(l0, l1);
            }
        }
    }
    if (lane == 0) LLMA_STAMP_MINMAX(stp, 6);
}

cudaError_t init_attention_mma() {
    cudaError_t e = cudaFuncSetAttribute(attention_mma_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(AttnSmem<128>::kBytes + 1024));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(attention_mma_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(AttnSmem<64>::kBytes + 1024));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(attention_long_kernel<128, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(AttnSmem<128>::kBytes + 1024));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(attention_long_kernel<128, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(AttnSmem<128>::kBytes + 1024));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(attention_long_kernel<64, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(AttnSmem<64>::kBytes + 1024));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(attention_long_kernel<64, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(AttnSmem<64>::kBytes + 1024));
}

void launch_attention_mma(cudaStream_t st, const AttnArgs& a, const CUtensorMap& map_k, const CUtensorMap& map_v) {
    dim3 grid(a.n_chunks, a.dims.n_heads, a.dims.max_batch);
    dim3 mgrid(a.dims.n_heads, (a.n_rows + 3) / 4);
    const size_t msmem = (size_t)8 * a.n_chunks * sizeof(float);
    if (a.tiles > 1) {  // long contexts, many sequences: several tiles per CTA
        if (a.dims.head_dim == 128) {
            if (a.tiles == 4) launch_pdl(st, true, grid, dim3(128), AttnSmem<128>::kBytes + 1024, attention_long_kernel<128, 4>, a, map_k, map_v);
            else launch_pdl(st, true, grid, dim3(128), AttnSmem<128>::kBytes + 1024, attention_long_kernel<128, 2>, a, map_k, map_v);
            launch_pdl(st, true, mgrid, dim3(128), msmem, attention_merge_kernel<128>, a);
        } else {
            if (a.tiles == 4) launch_pdl(st, true, grid, dim3(128), AttnSmem<64>::kBytes + 1024, attention_long_kernel<64, 4>, a, map_k, map_v);
            else launch_pdl(st, true, grid, dim3(128), AttnSmem<64>::kBytes + 1024, attention_long_kernel<64, 2>, a, map_k, map_v);
            launch_pdl(st, true, mgrid, dim3(128), msmem, attention_merge_kernel<64>, a);
        }
        return;
    }
    if (a.dims.head_dim == 128) {
        launch_pdl(st, true, grid, dim3(128), AttnSmem<128>::kBytes + 1024, attention_mma_kernel<128>, a, map_k, map_v);
        launch_pdl(st, true, mgrid, dim3(128), msmem, attention_merge_kernel<128>, a);
    } else {
        launch_pdl(st, true, grid, dim3(128), AttnSmem<64>::kBytes + 1024, attention_mma_kernel<64>, a, map_k, map_v);
        launch_pdl(st, true, mgrid, dim3(128), msmem, attention_merge_kernel<64>, a);
    }
}

}  // namespace llma
