// Epilogues of the weight-streaming GEMM: what happens to a finished 128 x 32 fp32 block.
// Called by the 128 epilogue threads after the block has been staged in shared memory:
// stage[f][j] is the result for output feature f of the tile (thread `row` staged its own
// feature) and activation row j < nj <= 32 (gemm_ws_kernel: one block per tile).
// red_f / red_i are [4][32] scratch for per-warp reductions.  With live = false nothing is stored to global memory
// (the turn that only brings the code in).
//
// The loops over activation rows are deliberately NOT unrolled over all 32 rows: this code
// runs once per tile, so its cost is dominated by instruction fetch, and compact loops
// with a few independent loads in flight beat long straight-line code.
#pragma once
#include "gemm_tcgen05.cuh"
#include "ptx_sm100.cuh"

namespace llma {

constexpr int kXPre = 13;  // residual epilogue: x rows 0..11 of the column, then the next norm's gain, requested early

constexpr uint32_t kEpiBar = 1;  // named barrier of the 128 epilogue threads

__device__ __forceinline__ void epi_sync() { ptx::named_bar_sync(kEpiBar, 128); }

__device__ __forceinline__ float warp_sum(float v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// x[r, n] += acc  (output projection and FFN down projection, residual stream in fp32).
// When the next RMSNorm is folded in (g.xs_out): also xs = split(x * gain) and this tile's
// per-row sums of squares, reduced over the 128 columns in an order fixed by the column index.
// xpre holds x[0..11, col] and the gain, read earlier by the caller.
__device__ __forceinline__ void epilogue_resid(const GemmArgs& g, int tile, int row, int nj, float (*stage)[33],
                                               const float (&xpre)[kXPre], bool live) {
    const int col = tile * 128 + row;
    const bool valid = col < g.n_out;
    const bool fold = g.xs_out != nullptr;
    const float gain = xpre[kXPre - 1];
    const unsigned group = 0xffu << (row & 24);  // the eight lanes that share an activation row below
    // x is added into the staged tile with a few loads in flight; the per-row work is a rolled loop
#pragma unroll
    for (int u = 0; u < kXPre - 1; ++u)
        if (u < nj) stage[row][u] += xpre[u];
    for (int j0 = kXPre - 1; j0 < nj; j0 += 8) {
        float xv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            xv[u] = (valid && j0 + u < nj) ? __ldcg(&g.out_f32[(int64_t)(j0 + u) * g.ld + col]) : 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (j0 + u < nj) stage[row][j0 + u] += xv[u];
    }
    if (!valid) {
        for (int j = 0; j < nj; ++j) stage[row][j] = 0.f;  // columns past the matrix add nothing to the sums of squares
    } else {
#pragma unroll 1
        for (int j = 0; j < nj; ++j) {
            const float xn = stage[row][j];
            if (live) g.out_f32[(int64_t)j * g.ld + col] = xn;
            if (fold && live) store_split(g.xs_out, g.rc, j, col, g.n_out, xn * gain);
        }
    }
    if (!fold) return;
    // Sums of squares: eight threads per activation row, each over sixteen consecutive features in
    // ascending order, then a three-step shuffle tree: the order depends on the feature index only.
    epi_sync();
    for (int j = row >> 3; j < nj; j += 16) {  // nj is uniform over the eight threads of a row
        const int f0 = (row & 7) * 16;
        float sq = 0.f;
#pragma unroll
        for (int u = 0; u < 16; ++u) { const float v = stage[f0 + u][j]; sq = __fmaf_rn(v, v, sq); }
        sq += __shfl_xor_sync(group, sq, 1);
        sq += __shfl_xor_sync(group, sq, 2);
        sq += __shfl_xor_sync(group, sq, 4);
        if ((row & 7) == 0 && live) g.ss_out[(int64_t)tile * g.rc + j] = sq;
    }
    epi_sync();
}

// out[r, n] = acc
__device__ __forceinline__ void epilogue_store(const GemmArgs& g, int tile, int row, int nj, float (*stage)[33]) {
    const int col = tile * 128 + row;
    if (col >= g.n_out) return;
#pragma unroll 1
    for (int j = 0; j < nj; ++j) g.out_f32[(int64_t)j * g.ld + col] = stage[row][j];
}

// QKV: rotary embedding on q and k (pair (i, i + hd/2)), q to the fp32 qkv buffer, k and v
// rows into the bf16 cache at (sequence, position) of every used row.
//   row_pos[r] / row_seq[r]: position (-1: unused) and sequence slot of activation row r;
//   rope_s: (cos, sin) of every row's position, staged in shared memory, [j][hd/2].
__device__ __forceinline__ void epilogue_qkv(const GemmArgs& g, int tile, int row, int nj, float (*stage)[33], const int* row_pos,
                                             const int* row_seq, const float2* rope_s, bool live) {
    const ModelDims& d = g.dims;
    const int mat = (tile >= g.tiles_per_map ? 1 : 0) + (tile >= 2 * g.tiles_per_map ? 1 : 0);
    const int col = (tile - mat * g.tiles_per_map) * 128 + row;
    const int hd = d.head_dim, half = hd >> 1;  // head_dim 128 or 64
    const int head = hd == 128 ? col >> 7 : col >> 6, idx = col & (hd - 1);
    const bool lower = idx < half;
    const int prow = lower ? row + half : row - half;
    const int fi = idx & (half - 1);
    if (col < g.n_out) {
#pragma unroll 1
        for (int j = 0; j < nj; ++j) {
            const int pos = live ? row_pos[j] : 0;
            if (pos < 0) continue;
            float val = stage[row][j];
            if (mat < 2) {
                const float2 cs = rope_s[j * half + fi];
                const float other = stage[prow][j];
                val = lower ? (val * cs.x - other * cs.y) : (other * cs.y + val * cs.x);
            }
            if (!live) continue;
            if (mat == 0) {
                g.out_f32[(int64_t)j * g.ld + col] = val;
            } else {
                __nv_bfloat16* cache = mat == 1 ? g.kcache : g.vcache;
                cache[kv_row_index(d, g.layer, row_seq[j], head, pos) * hd + idx] = __float2bfloat16_rn(val);
            }
        }
    }
    epi_sync();
}

// SwiGLU: tile rows 0..63 are gate features, 64..127 the matching up features.
__device__ __forceinline__ void epilogue_swiglu(const GemmArgs& g, int tile, int row, int nj, float (*stage)[33], bool live) {
    const int fi = row & 63, f = tile * 64 + fi;
    if (f < g.n_out) {
#pragma unroll 1
        for (int j = row >> 6; j < nj; j += 2) {
            const float gate = stage[g.gate_second ? 64 + fi : fi][j], up = stage[g.gate_second ? fi : 64 + fi][j];
            const float v = gate / (1.f + expf(-gate)) * up;
            if (live) store_split(g.out_act, g.rc, j, f, g.n_out, v);
        }
    }
    epi_sync();
}

// LM head: optional logits store, then the tile's (max, lowest argmax) for every used row.  Row-major like the
// epilogues above: thread t takes activation row j = t & 31 and 32 consecutive features, so a row costs no shuffles
// (five steps of two per row before: 25 us per 144-row tile, 3 us at nine rows).
__device__ __forceinline__ void epilogue_lmhead(const GemmArgs& g, int tile, int t, int nj, float (*stage)[33], float* red_f, int* red_i,
                                                bool live) {
    const int j = t & 31, w = t >> 5, f0 = 32 * w;
    const int v0 = tile * 128 + f0, nv = min(32, g.n_out - v0);  // nv <= 0: past the vocabulary
    if (j < nj) {
        float bv = -INFINITY;
        int bi = 0x7fffffff;
        if (nv == 32) {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const float a = stage[f0 + i][j];
                if (a > bv) { bv = a; bi = v0 + i; }
            }
        } else {
            for (int i = 0; i < nv; ++i) {
                const float a = stage[f0 + i][j];
                if (a > bv) { bv = a; bi = v0 + i; }
            }
        }
        red_f[w * 32 + j] = bv;
        red_i[w * 32 + j] = bi;
        if (g.out_f32 && live) {
            float* o = g.out_f32 + (int64_t)j * g.ld + v0;
            if (nv == 32 && (g.ld & 3) == 0) {
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    reinterpret_cast<float4*>(o)[u] = make_float4(stage[f0 + 4 * u][j], stage[f0 + 4 * u + 1][j], stage[f0 + 4 * u + 2][j],
                                                                  stage[f0 + 4 * u + 3][j]);
            } else {
                for (int i = 0; i < nv; ++i) o[i] = stage[f0 + i][j];
            }
        }
    }
    epi_sync();
    if (w == 0 && j < nj) {
        float bv = red_f[j];
        int bi = red_i[j];
#pragma unroll
        for (int u = 1; u < 4; ++u)  // ascending features: the lowest index on ties
            if (red_f[u * 32 + j] > bv) { bv = red_f[u * 32 + j]; bi = red_i[u * 32 + j]; }
        if (live) {
            g.part_max[(int64_t)tile * g.rc + j] = bv;
            g.part_idx[(int64_t)tile * g.rc + j] = bi;
        }
    }
    epi_sync();
}

// ---- blocks of 32 rows (gemm_wide_kernel, gemm_prompt_kernel) --------------------------------------------------------
// The block is staged row by row, st[j][f] (thread f wrote feature f of every row), and a warp takes whole rows: four
// consecutive features per lane, so that the residual stream, rotary factors, split operands, cache rows and logits move as
// full 128-byte lines.  (One row per lane with 16 or 32 features each -- the layout before -- touched 32 lines per
// access: 3 us per block of the output projection against 1.2.)  The loads a block needs are requested before its
// barrier.  Every function begins with the block staged but not yet synchronised and ends synchronised.
constexpr int kBlockLd = 132;  // row length of the staged block: 16-byte rows, conflict-free either way

__device__ __forceinline__ uint32_t pack_bf16x2(float x, float y) {
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x)) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(y)) << 16);
}
// hi = bf16(v), lo = bf16(v - hi) of four values, stored at dst and dst + lo_term
__device__ __forceinline__ void store_split4(__nv_bfloat16* dst, int64_t lo_term, const float4& v) {
    const __nv_bfloat16 a = __float2bfloat16_rn(v.x), b = __float2bfloat16_rn(v.y), c = __float2bfloat16_rn(v.z), d = __float2bfloat16_rn(v.w);
    *reinterpret_cast<uint2*>(dst) = make_uint2((uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16),
                                                (uint32_t)__bfloat16_as_ushort(c) | ((uint32_t)__bfloat16_as_ushort(d) << 16));
    *reinterpret_cast<uint2*>(dst + lo_term) = make_uint2(pack_bf16x2(v.x - __bfloat162float(a), v.y - __bfloat162float(b)),
                                                          pack_bf16x2(v.z - __bfloat162float(c), v.w - __bfloat162float(d)));
}

// Stage a block: thread f = `feature` holds acc[j] of rows jb + j, scaled by the rows' norm scales where there are any
// (scale: 16-byte aligned, 32 entries).
__device__ __forceinline__ void stage_block(float (*st)[kBlockLd], int feature, const float (&acc)[32], const float* scale) {
    if (scale) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 c = reinterpret_cast<const float4*>(scale)[q];
            st[4 * q][feature] = acc[4 * q] * c.x; st[4 * q + 1][feature] = acc[4 * q + 1] * c.y;
            st[4 * q + 2][feature] = acc[4 * q + 2] * c.z; st[4 * q + 3][feature] = acc[4 * q + 3] * c.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) st[j][feature] = acc[j];
    }
}

// A warp's rows (warp, warp + 4, ...) are worked on side by side, four or, in a block of more than 16 rows, eight: there is
// one warp per scheduler, so a chain of dependent instructions costs its full latency.  Rows past nj are computed
// (their staged values are whatever the accumulator held) and not stored.
template <typename F>
__device__ __forceinline__ void each_row(bool two, F f) {  // f(u): row warp + 4 u of the block; u a constant after unrolling
#pragma unroll
    for (int u = 0; u < 4; ++u) f(u);
    if (two) {
#pragma unroll
        for (int u = 4; u < 8; ++u) f(u);
    }
}

// x[r, n] += acc, the next norm's split operand and the tile's sums of squares; n_out % 128 == 0
template <typename Sync>
__device__ __forceinline__ void block_resid(const GemmArgs& g, int tile, int warp, int lane, int jb, int nj, float (*st)[kBlockLd],
                                            Sync sync) {
    const int col = tile * 128 + 4 * lane;
    float* x = g.out_f32 + (int64_t)jb * g.ld + col;
    const bool two = nj > 16;
    float4 v[8];
    each_row(two, [&](int u) { v[u] = __ldcg(reinterpret_cast<const float4*>(x + (int64_t)min(warp + 4 * u, nj - 1) * g.ld)); });
    const float4 gn = load4_each(g.gain_next + col);
    sync();
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(g.xs_out) + (int64_t)jb * g.n_out + col;
    const int64_t lo_term = (int64_t)g.rc * g.n_out;
    float sq[8] = {};
    each_row(two, [&](int u) {
        const float4 a = *reinterpret_cast<const float4*>(&st[warp + 4 * u][4 * lane]);
        v[u].x += a.x; v[u].y += a.y; v[u].z += a.z; v[u].w += a.w;
        sq[u] = __fmaf_rn(v[u].w, v[u].w, __fmaf_rn(v[u].z, v[u].z, __fmaf_rn(v[u].y, v[u].y, v[u].x * v[u].x)));
    });
    each_row(two, [&](int u) {
        const int j = warp + 4 * u;
        if (j < nj) {
            *reinterpret_cast<float4*>(x + (int64_t)j * g.ld) = v[u];
            store_split4(xs + (int64_t)j * g.n_out, lo_term, make_float4(v[u].x * gn.x, v[u].y * gn.y, v[u].z * gn.z, v[u].w * gn.w));
        }
    });
    // eight sums over 32 lanes: halves are exchanged until a lane holds one row's, then added over the last four lanes
#pragma unroll
    for (int w = 16, n = 4; n >= 1; w >>= 1, n >>= 1) {
        const bool up = lane & w;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float send = up ? sq[i] : sq[i + n], keep = up ? sq[i + n] : sq[i];
            sq[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
        }
    }
    sq[0] += __shfl_xor_sync(0xffffffffu, sq[0], 2);
    sq[0] += __shfl_xor_sync(0xffffffffu, sq[0], 1);
    const int j = warp + 4 * (((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1));
    if ((lane & 3) == 0 && j < nj) g.ss_out[(int64_t)tile * g.rc + jb + j] = sq[0];
    sync();
}

// rotary embedding of q and k; q to the fp32 buffer, k and v to the cache.  pos_of(j), seq_of(j): position and sequence slot
// of row jb + j.  head_dim 64 or 128: a tile of 128 features holds whole heads.
template <typename PosOf, typename SeqOf, typename Sync>
__device__ __forceinline__ void block_qkv(const GemmArgs& g, int tile, int warp, int lane, int jb, int nj, float (*st)[kBlockLd],
                                          PosOf pos_of, SeqOf seq_of, Sync sync) {
    const ModelDims& d = g.dims;
    const int mat = (tile >= g.tiles_per_map ? 1 : 0) + (tile >= 2 * g.tiles_per_map ? 1 : 0);
    const int f = 4 * lane, col = (tile - mat * g.tiles_per_map) * 128 + f;
    const int hd = d.head_dim, half = hd >> 1;
    const int head = hd == 128 ? col >> 7 : col >> 6, idx = col & (hd - 1), fi = idx & (half - 1);
    const bool lower = idx < half;
    const int partner = lower ? f + half : f - half;
    const bool two = nj > 16;
    if (mat == 2) {
        sync();
        each_row(two, [&](int u) {
            const int j = warp + 4 * u;
            const float4 v = *reinterpret_cast<const float4*>(&st[j][f]);
            if (j < nj)
                *reinterpret_cast<uint2*>(g.vcache + kv_row_index(d, g.layer, seq_of(j), head, pos_of(j)) * hd + idx) =
                    make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
        });
    } else {
        float4 c[8], sn[8];
        each_row(two, [&](int u) {
            const int64_t at = (int64_t)pos_of(min(warp + 4 * u, nj - 1)) * half + fi;
            c[u] = __ldg(reinterpret_cast<const float4*>(g.rope_cos + at));
            sn[u] = __ldg(reinterpret_cast<const float4*>(g.rope_sin + at));
            if (lower) { sn[u].x = -sn[u].x; sn[u].y = -sn[u].y; sn[u].z = -sn[u].z; sn[u].w = -sn[u].w; }
        });
        sync();
        each_row(two, [&](int u) {
            const int j = warp + 4 * u;
            const float4 a = *reinterpret_cast<const float4*>(&st[j][f]), b = *reinterpret_cast<const float4*>(&st[j][partner]);
            // lower half: a cos - b sin, upper half: a cos + b sin
            const float4 v = make_float4(__fmaf_rn(b.x, sn[u].x, a.x * c[u].x), __fmaf_rn(b.y, sn[u].y, a.y * c[u].y),
                                         __fmaf_rn(b.z, sn[u].z, a.z * c[u].z), __fmaf_rn(b.w, sn[u].w, a.w * c[u].w));
            if (j < nj) {
                if (mat == 0)
                    *reinterpret_cast<float4*>(g.out_f32 + (int64_t)(jb + j) * g.ld + col) = v;
                else
                    *reinterpret_cast<uint2*>(g.kcache + kv_row_index(d, g.layer, seq_of(j), head, pos_of(j)) * hd + idx) =
                        make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
            }
        });
    }
    sync();
}

// h = silu(gate) * up, the tile's features 0..63 and 64..127: half a warp per row; n_out % 64 == 0
template <typename Sync>
__device__ __forceinline__ void block_swiglu(const GemmArgs& g, int tile, int warp, int lane, int jb, int nj, float (*st)[kBlockLd],
                                             Sync sync) {
    const int f = 4 * (lane & 15);
    __nv_bfloat16* h = reinterpret_cast<__nv_bfloat16*>(g.out_act) + (int64_t)jb * g.n_out + tile * 64 + f;
    const int64_t lo_term = (int64_t)g.rc * g.n_out;
    sync();
    auto row = [&](int u) {
        const int j = 2 * (warp + 4 * u) + (lane >> 4);
        const float4 a = *reinterpret_cast<const float4*>(&st[j][f]);
        const float4 b = *reinterpret_cast<const float4*>(&st[j][64 + f]);
        const float4 v = make_float4(a.x / (1.f + expf(-a.x)) * b.x, a.y / (1.f + expf(-a.y)) * b.y, a.z / (1.f + expf(-a.z)) * b.z,
                                     a.w / (1.f + expf(-a.w)) * b.w);
        if (j < nj) store_split4(h + (int64_t)j * g.n_out, lo_term, v);
    };
    row(0);
    row(1);
    if (nj > 16) { row(2); row(3); }
    sync();
}

// optional logits, and the tile's (max, lowest argmax) of every row
template <typename Sync>
__device__ __forceinline__ void block_lmhead(const GemmArgs& g, int tile, int warp, int lane, int jb, int nj, float (*st)[kBlockLd],
                                             Sync sync) {
    const int v0 = tile * 128 + 4 * lane;
    const int nv = min(4, g.n_out - v0);  // <= 0: past the vocabulary
    sync();
    const bool two = nj > 16;
    float4 a[8];
    unsigned key[8];  // the bits of the lane's maximum, in an order that unsigned comparison follows
    each_row(two, [&](int u) {
        a[u] = *reinterpret_cast<const float4*>(&st[warp + 4 * u][4 * lane]);
        float m = nv > 0 ? a[u].x : -INFINITY;
        if (nv > 1) m = fmaxf(m, a[u].y);
        if (nv > 2) m = fmaxf(m, a[u].z);
        if (nv > 3) m = fmaxf(m, a[u].w);
        const unsigned b = __float_as_uint(m + 0.f);  // -0 becomes +0: equal values, equal keys
        key[u] = b & 0x80000000u ? ~b : b | 0x80000000u;
    });
    unsigned top[8];
    each_row(two, [&](int u) { top[u] = __reduce_max_sync(0xffffffffu, key[u]); });
    each_row(two, [&](int u) {
        const int j = warp + 4 * u;
        const float m = __uint_as_float(top[u] & 0x80000000u ? top[u] & 0x7fffffffu : ~top[u]);
        int i = 0x7fffffff;  // lowest index of the lane that holds the maximum
        if (nv > 3 && a[u].w == m) i = v0 + 3;
        if (nv > 2 && a[u].z == m) i = v0 + 2;
        if (nv > 1 && a[u].y == m) i = v0 + 1;
        if (nv > 0 && a[u].x == m) i = v0;
        const int first = __reduce_min_sync(0xffffffffu, i);
        if (j < nj) {
            if (g.out_f32) {
                float* o = g.out_f32 + (int64_t)(jb + j) * g.ld + v0;
                if (nv == 4 && (g.ld & 3) == 0) {
                    *reinterpret_cast<float4*>(o) = a[u];
                } else {
                    if (nv > 0) o[0] = a[u].x;
                    if (nv > 1) o[1] = a[u].y;
                    if (nv > 2) o[2] = a[u].z;
                    if (nv > 3) o[3] = a[u].w;
                }
            }
            if (lane == 0) {
                g.part_max[(int64_t)tile * g.rc + jb + j] = m;
                g.part_idx[(int64_t)tile * g.rc + jb + j] = first;
            }
        }
    });
    sync();
}

// Partial tiles in the workspace: [cta][q][feature] float4, q = group of four activation rows (qn groups per
// slot).  The 32 features of a warp are 512 consecutive bytes, so one store or polling load of a warp touches four lines.
__device__ __forceinline__ float4* ws_slot(float* ws, int qn, int slot, int feature) {
    return reinterpret_cast<float4*>(ws) + (int64_t)slot * ((int64_t)qn * 128) + feature;
}

}  // namespace llma
