// Causal attention of a prompt pass: up to two thousand query rows of one sequence against its cached positions.
//
// One CTA of four warps per (64 query rows, head); a warp holds 16 rows' queries (hi + lo bf16 fragments) and running
// maximum, sum and output in registers and walks over the positions in tiles of 64, whose K and V arrive by TMA in two
// stages.  Nothing is combined across warps and nothing goes through global memory, where a pass of 128 rows in
// attention_mma_kernel writes chunk partials for a merge kernel and reads every K/V tile once per 128 rows.
// Bound by mma.sync: Q and P enter as hi + lo pairs, so a 16 x 64 tile costs 256 m16n8k16 MMAs at head_dim 128
// against 64 ldmatrix.  The row tiles with the most positions start first.  A tile's P V has accumulators of its own and is added to
// the running output rounded to nearest: mma.sync rounds its additions towards zero, and with the running output as accumulator
// the cached codes of the next layer differ 6 % more often at 2299 positions (0.655 against 0.616 %).  Four 7B layers, 1535
// positions: 3.04 -> 3.06 ms.
#include <cuda.h>

#include "attention_frag.cuh"
#include "attention_mma.cuh"
#include "ptx_sm100.cuh"

namespace llma {

using namespace ptx;

template <int HD>
struct PromptSmem {
    static constexpr int kBoxes = HD / 64;
    static constexpr uint32_t kBoxBytes = kPromptKV * 128;
    static constexpr uint32_t kTile = kBoxes * kBoxBytes;   // K (or V) of a tile
    static constexpr uint32_t offBar = 4 * kTile;           // [stage][K, V] tiles, then the barriers
    static constexpr uint32_t kBytes = offBar + 64 + 1024;  // + alignment
};

template <int HD>
__global__ void __launch_bounds__(128, 2)
attention_prompt_kernel(const PromptAttnArgs a, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v) {
    using L = PromptSmem<HD>;
    pdl_trigger();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const ModelDims& d = a.dims;
    const int head = blockIdx.x;
    const int q0 = ((int)gridDim.y - 1 - (int)blockIdx.y) * 64;  // first query row of the CTA
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t bar0 = base + L::offBar;
    auto bar_k = [&](int st) { return bar0 + 16u * st; };
    auto bar_v = [&](int st) { return bar0 + 16u * st + 8u; };
    auto tile_k = [&](int st) { return base + (uint32_t)(2 * st) * L::kTile; };
    auto tile_v = [&](int st) { return base + (uint32_t)(2 * st + 1) * L::kTile; };
    const int n_tiles = (a.pos0 + min(q0 + 64, a.n_rows) - 1) / kPromptKV + 1;  // tiles up to the last row's own position

    auto fetch = [&](int t) {  // one thread
        const int st = t & 1;
        const int32_t row0 = (int32_t)kv_row_index(d, a.layer, a.seq, head, t * kPromptKV);
        mbar_arrive_expect_tx(bar_k(st), L::kTile);
        for (int b = 0; b < L::kBoxes; ++b) tma_load_2d(tile_k(st) + b * L::kBoxBytes, &map_k, bar_k(st), b * 64, row0);
        mbar_arrive_expect_tx(bar_v(st), L::kTile);
        for (int b = 0; b < L::kBoxes; ++b) tma_load_2d(tile_v(st) + b * L::kBoxBytes, &map_v, bar_v(st), b * 64, row0);
    };
    if (threadIdx.x == 0) {
        for (int st = 0; st < 2; ++st) { mbar_init(bar_k(st), 1); mbar_init(bar_v(st), 1); }
        fence_mbar_init();
    }
    pdl_wait();  // q and the K/V rows of this pass come from the projection before
    __syncthreads();
    if (threadIdx.x == 0) {
        fetch(0);
        if (n_tiles > 1) fetch(1);
    }
    // Q fragments: lane (g, t) holds rows g and g + 8, columns 16 ks + 2t, +1, +8, +9
    const int g8 = lane >> 2, t4 = lane & 3, mi = lane >> 3, t8 = lane & 7;
    const int r_lo = q0 + warp * 16 + g8, r_hi = r_lo + 8;
    const bool on_lo = r_lo < a.n_rows, on_hi = r_hi < a.n_rows;
    const int lim_lo = on_lo ? a.pos0 + r_lo : -1, lim_hi = on_hi ? a.pos0 + r_hi : -1;
    const int first_row = q0 + warp * 16, last_row = min(first_row + 15, a.n_rows - 1);
    uint32_t qh[HD / 16][4], ql[HD / 16][4];
    {
        const float* p_lo = a.q + (int64_t)r_lo * d.hd_total + head * HD + 2 * t4;
        const float* p_hi = p_lo + 8 * (int64_t)d.hd_total;
        const float2 z = make_float2(0.f, 0.f);
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
            const float2 x0 = on_lo ? __ldcg(reinterpret_cast<const float2*>(p_lo + ks * 16)) : z;
            const float2 x1 = on_hi ? __ldcg(reinterpret_cast<const float2*>(p_hi + ks * 16)) : z;
            const float2 x2 = on_lo ? __ldcg(reinterpret_cast<const float2*>(p_lo + ks * 16 + 8)) : z;
            const float2 x3 = on_hi ? __ldcg(reinterpret_cast<const float2*>(p_hi + ks * 16 + 8)) : z;
            split_pack(x0.x, x0.y, qh[ks][0], ql[ks][0]);
            split_pack(x1.x, x1.y, qh[ks][1], ql[ks][1]);
            split_pack(x2.x, x2.y, qh[ks][2], ql[ks][2]);
            split_pack(x3.x, x3.y, qh[ks][3], ql[ks][3]);
        }
    }
    const float scale = rsqrtf((float)HD);
    float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;  // l: this lane's columns only, until the end
    float o[HD / 8][4];
#pragma unroll
    for (int i = 0; i < HD / 8; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
    bool landed = true;

#pragma unroll 1
    for (int t = 0; t < n_tiles; ++t) {
        const int st = t & 1;
        const uint32_t par = (uint32_t)((t >> 1) & 1);
        const int p0 = t * kPromptKV;
        // rows past the pass and tiles beyond the warp's last row have nothing to do; the warp still meets the barrier below
        if (landed && first_row < a.n_rows && p0 <= a.pos0 + last_row) {
            landed = mbar_wait(bar_k(st), par);
            float sc[8][4];
#pragma unroll
            for (int i = 0; i < 8; ++i) { sc[i][0] = sc[i][1] = sc[i][2] = sc[i][3] = 0.f; }
#pragma unroll
            for (int ks = 0; ks < HD / 16; ++ks) {
#pragma unroll
                for (int np = 0; np < 4; ++np) {
                    const int row = np * 16 + (mi >> 1) * 8 + t8;
                    const int col = ks * 16 + (mi & 1) * 8;
                    const uint32_t kaddr = tile_k(st) + (uint32_t)(col >> 6) * L::kBoxBytes + (uint32_t)row * 128 +
                                           ((((uint32_t)(col & 63) >> 3) ^ ((uint32_t)row & 7u)) << 4);
                    uint32_t b[4];
                    ldsm_x4(kaddr, b);
                    mma_bf16(sc[2 * np], qh[ks], b[0], b[1]);
                    mma_bf16(sc[2 * np + 1], qh[ks], b[2], b[3]);
                    mma_bf16(sc[2 * np], ql[ks], b[0], b[1]);
                    mma_bf16(sc[2 * np + 1], ql[ks], b[2], b[3]);
                }
            }
            const bool diagonal = p0 + kPromptKV - 1 > a.pos0 + first_row;  // uniform: some position lies beyond some row
            float bm_lo = -INFINITY, bm_hi = -INFINITY;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float v = sc[nt][e] * scale;
                    if (diagonal) v = p0 + nt * 8 + 2 * t4 + (e & 1) <= (e < 2 ? lim_lo : lim_hi) ? v : -INFINITY;
                    sc[nt][e] = v;
                    if (e < 2) bm_lo = fmaxf(bm_lo, v); else bm_hi = fmaxf(bm_hi, v);
                }
            }
            bm_lo = fmaxf(bm_lo, __shfl_xor_sync(0xffffffffu, bm_lo, 1)); bm_lo = fmaxf(bm_lo, __shfl_xor_sync(0xffffffffu, bm_lo, 2));
            bm_hi = fmaxf(bm_hi, __shfl_xor_sync(0xffffffffu, bm_hi, 1)); bm_hi = fmaxf(bm_hi, __shfl_xor_sync(0xffffffffu, bm_hi, 2));
            const float n_lo = fmaxf(m_lo, bm_lo), n_hi = fmaxf(m_hi, bm_hi);
            const float ref_lo = n_lo == -INFINITY ? 0.f : n_lo, ref_hi = n_hi == -INFINITY ? 0.f : n_hi;
            const float f_lo = expf(m_lo - ref_lo), f_hi = expf(m_hi - ref_hi);  // 0 in the first tile
            float bl_lo = 0.f, bl_hi = 0.f;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float pe = expf(sc[nt][e] - (e < 2 ? ref_lo : ref_hi));
                    sc[nt][e] = pe;
                    if (e < 2) bl_lo += pe; else bl_hi += pe;
                }
            }
            l_lo = __fmaf_rn(l_lo, f_lo, bl_lo); l_hi = __fmaf_rn(l_hi, f_hi, bl_hi);
            m_lo = n_lo; m_hi = n_hi;
            landed = mbar_wait(bar_v(st), par) && landed;
            uint32_t ph[4][4], pl[4][4];
#pragma unroll
            for (int kp = 0; kp < 4; ++kp) {
                split_pack(sc[2 * kp][0], sc[2 * kp][1], ph[kp][0], pl[kp][0]);
                split_pack(sc[2 * kp][2], sc[2 * kp][3], ph[kp][1], pl[kp][1]);
                split_pack(sc[2 * kp + 1][0], sc[2 * kp + 1][1], ph[kp][2], pl[kp][2]);
                split_pack(sc[2 * kp + 1][2], sc[2 * kp + 1][3], ph[kp][3], pl[kp][3]);
            }
#pragma unroll
            for (int n0 = 0; n0 < HD / 16; n0 += 2) {  // 32 columns of V: four accumulators for the tile, added to the running output
                float pv[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i) { pv[i][0] = pv[i][1] = pv[i][2] = pv[i][3] = 0.f; }
#pragma unroll
                for (int kp = 0; kp < 4; ++kp) {
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int row = kp * 16 + (mi & 1) * 8 + t8;
                        const int col = (n0 + u) * 16 + (mi >> 1) * 8;
                        const uint32_t vaddr = tile_v(st) + (uint32_t)(col >> 6) * L::kBoxBytes + (uint32_t)row * 128 +
                                               ((((uint32_t)(col & 63) >> 3) ^ ((uint32_t)row & 7u)) << 4);
                        uint32_t b[4];
                        ldsm_x4_trans(vaddr, b);
                        mma_bf16(pv[2 * u], ph[kp], b[0], b[1]);
                        mma_bf16(pv[2 * u + 1], ph[kp], b[2], b[3]);
                        mma_bf16(pv[2 * u], pl[kp], b[0], b[1]);
                        mma_bf16(pv[2 * u + 1], pl[kp], b[2], b[3]);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float (&a4)[4] = o[2 * n0 + i];
                    a4[0] = __fmaf_rn(a4[0], f_lo, pv[i][0]); a4[1] = __fmaf_rn(a4[1], f_lo, pv[i][1]);
                    a4[2] = __fmaf_rn(a4[2], f_hi, pv[i][2]); a4[3] = __fmaf_rn(a4[3], f_hi, pv[i][3]);
                }
            }
            landed = __all_sync(0xffffffffu, landed);
        }
        __syncthreads();  // every warp has read the tile: its stage may be filled again
        if (threadIdx.x == 0 && t + 2 < n_tiles) fetch(t + 2);
    }
    if (!landed && lane == 0) atomicExch(a.dev_err, kDevErrTimeout);
    // copies that no warp waited for must land before the CTA goes
    if (threadIdx.x == 0) {
        for (int t = max(0, n_tiles - 2); t < n_tiles; ++t) {
            (void)mbar_wait(bar_k(t & 1), (uint32_t)((t >> 1) & 1)); (void)mbar_wait(bar_v(t & 1), (uint32_t)((t >> 1) & 1));
        }
    }
    l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1); l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
    l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1); l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
    const float i_lo = 1.f / l_lo, i_hi = 1.f / l_hi;
    __nv_bfloat16* out_lo = reinterpret_cast<__nv_bfloat16*>(a.attn_out) + (int64_t)r_lo * d.hd_total + head * HD + 2 * t4;
    __nv_bfloat16* out_hi = out_lo + 8 * (int64_t)d.hd_total;
    const int64_t lo_term = (int64_t)a.rc * d.hd_total;
#pragma unroll
    for (int nt = 0; nt < HD / 8; ++nt) {
        uint32_t h, l;
        if (on_lo) {
            split_pack(o[nt][0] * i_lo, o[nt][1] * i_lo, h, l);
            *reinterpret_cast<uint32_t*>(out_lo + nt * 8) = h;
            *reinterpret_cast<uint32_t*>(out_lo + lo_term + nt * 8) = l;
        }
        if (on_hi) {
            split_pack(o[nt][2] * i_hi, o[nt][3] * i_hi, h, l);
            *reinterpret_cast<uint32_t*>(out_hi + nt * 8) = h;
            *reinterpret_cast<uint32_t*>(out_hi + lo_term + nt * 8) = l;
        }
    }
}

cudaError_t init_attention_prompt() {
    cudaError_t e = cudaFuncSetAttribute(attention_prompt_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PromptSmem<128>::kBytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(attention_prompt_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PromptSmem<64>::kBytes);
}

void launch_attention_prompt(cudaStream_t st, const PromptAttnArgs& a, const CUtensorMap& map_k, const CUtensorMap& map_v) {
    const dim3 grid(a.dims.n_heads, (a.n_rows + 63) / 64);
    if (a.dims.head_dim == 128) launch_pdl(st, true, grid, dim3(128), PromptSmem<128>::kBytes, attention_prompt_kernel<128>, a, map_k, map_v);
    else launch_pdl(st, true, grid, dim3(128), PromptSmem<64>::kBytes, attention_prompt_kernel<64>, a, map_k, map_v);
}

}  // namespace llma
