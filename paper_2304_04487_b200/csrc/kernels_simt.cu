// CUDA-core projections of the decoder forward: fp32 models (where tensor cores would break the 1e-4 logit tolerance)
// and the plain cross-check of the tensor-core path for bf16 models.
//
// out[r, n] = sum_k W[n, k] * a[r, k] for the rows of a step, with what surrounds the product folded in: the RMSNorm of
// its input (the gains multiply the rows as they are staged, the row's scale multiplies its sums), rotary embedding and
// K/V append (QKV), the residual sum (output and down projections), SiLU gating (gate/up), the per-row maximum (LM
// head).  A layer is then five launches where separate norm, rotary, gating, q, k, v, gate and up kernels made twelve.
//
// At these sizes a step is a chain of short kernels, so a kernel costs its latency: the activation rows are fetched once
// per CTA with every load in flight and stay in shared memory for all its warps; a warp takes two output features (the
// two of a rotary pair, gate and up of one feature, two neighbours), holds all rows' sums in registers, and has
// the weights of its next 512 columns on the way while it multiplies the current ones -- the first of them
// requested before the kernel before has finished, since no kernel writes weights.  Two features and sixteen rows make 32
// sums, which one 31-shuffle exchange turns into one sum per lane.
// Measured with attention_simt.cu against the kernels that the two replaced: a pass of a 2-layer fp32 decoder of width
// 256 at up to five rows 124 -> 68 us, of width 1024 at up to nine rows 443 -> 126 us (its weights: 20 us of HBM time).  5 of
// these 68 us went with the integer divisions that found a unit's place (a launch waits for the code it runs).
//
// Every sum is a fixed sequence of operations that depends on its own row's data and on the matrix shape only -- never on
// how many rows the step has.  That is what makes a (k+1)-row verification step bit-identical to k+1 one-row steps.
#include <type_traits>

#include "simt_common.cuh"

namespace llma {

constexpr int kWarps = 8;        // warps per CTA
constexpr int kRB = 16;          // most activation rows per pass over the weights
constexpr int kKC = 512;         // columns whose weights a warp holds at a time
constexpr size_t kResidentBytes = 200 * 1024;  // activation rows that fit stay in shared memory whole

// The sums of 32 (feature, row) pairs, one per lane: value f * 16 + r of every lane is added over the lanes and
// ends in lane f * 16 + r.  The same tree for every value.
__device__ __forceinline__ float exchange32(float (&v)[32], int lane) {
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
        const bool up = lane & w;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const float send = up ? v[i] : v[i + w];
            const float keep = up ? v[i + w] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
        }
    }
    return v[0];
}

// How the rows of a pass lie in shared memory; a kernel each, so that each carries one staging loop only (its code is fetched anew
// by nearly every launch, and a pass length read from the arguments costs fp32 and bf16 widths of 192 to 512 another 1 to 2 %).
enum Rows : int {
    kChunked,  // a 512-wide chunk at a time, 16 rows a pass: not even four rows fit whole
    kWhole,    // whole, 16 rows a pass
    kFewer,    // whole, g.pass_rows (4, 8 or 12) a pass
};
template <typename T, int MODE, int ROWS>
__global__ void __launch_bounds__(kWarps * 32, 2) rowgemm_kernel(const RowGemm g) {
    constexpr bool kNorm = MODE != kRowResid;  // the projections that read the residual stream
    constexpr int VN = Vec16<T>::N;
    constexpr int NV = kKC / (32 * VN);  // 16-byte pieces of a weight row per lane and chunk
    pdl_trigger();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr bool RES = ROWS != kChunked;
    const int K = g.k_in, KS = RES ? K : kKC;
    const int pass = ROWS == kFewer ? g.pass_rows : kRB;
    extern __shared__ __align__(16) float sA[];  // [rows of a pass][KS]
    __shared__ float s_ss[kRB][kWarps];
    __shared__ float s_part[kWarps][32];
    __shared__ float s_bv[kWarps][kRB];
    __shared__ int s_bi[kWarps][kRB];
    const int n_chunks = (K + kKC - 1) / kKC, n_turns = (n_chunks + (1 << g.split_lg) - 1) >> g.split_lg;
    // split = 1 << g.split_lg warps share a unit, taking its chunks in turn
    const int split = 1 << g.split_lg, per_cta = kWarps >> g.split_lg, part = warp & (split - 1), slot = warp >> g.split_lg;
    const int per_round = gridDim.x * per_cta;
    int rounds = 0;  // the same for the whole CTA
    for (int u = (int)blockIdx.x * per_cta; u < g.n_units; u += per_round) ++rounds;
    const int half = g.dims.head_dim >> 1, hd = g.dims.head_dim, HD = g.dims.hd_total;  // head_dim 128 or 64
    // unit of the QKV projection -> matrix, head, rotary pair (counted and shifted: a division is 25 instructions)
    auto qkv_unit = [&](int unit, int& mat, int& head, int& i) {
        mat = (unit >= (HD >> 1) ? 1 : 0) + (unit >= HD ? 1 : 0);
        const int v = unit - mat * (HD >> 1);
        head = hd == 128 ? v >> 6 : v >> 5;
        i = v & (half - 1);
    };

    // the two weight rows of a unit
    auto weight_rows = [&](int unit, const T*& p0, const T*& p1) {
        if (MODE == kRowQKV) {
            int mat, head, i;
            qkv_unit(unit, mat, head, i);
            const T* W = reinterpret_cast<const T*>(mat == 0 ? g.w0 : (mat == 1 ? g.w1 : g.w2));
            p0 = W + (int64_t)(head * hd + i) * K;
            p1 = p0 + (int64_t)half * K;
        } else if (MODE == kRowSwiGLU) {
            p0 = reinterpret_cast<const T*>(g.w0) + (int64_t)unit * K;
            p1 = reinterpret_cast<const T*>(g.w1) + (int64_t)unit * K;
        } else {
            p0 = reinterpret_cast<const T*>(g.w0) + (int64_t)(2 * unit) * K;
            p1 = 2 * unit + 1 < g.n_out ? p0 + K : p0;
        }
    };
    auto load_weights = [&](int round, int chunk, uint4 (&w)[2][NV]) {
        const int unit = min(round * per_round + (int)blockIdx.x * per_cta + slot, g.n_units - 1);
        const T *p0, *p1;
        weight_rows(unit, p0, p1);
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int k = chunk * kKC + (i * 32 + lane) * VN;
            const uint4 z = make_uint4(0u, 0u, 0u, 0u);
            w[0][i] = k < K ? __ldg(reinterpret_cast<const uint4*>(p0 + k)) : z;
            w[1][i] = k < K ? __ldg(reinterpret_cast<const uint4*>(p1 + k)) : z;
        }
    };
    uint4 w_next[2][NV];
    load_weights(0, part, w_next);
    pdl_wait();
    const int rows_used = __ldcg(&g.rows->rows_used);

#pragma unroll 1
    for (int r0 = 0; r0 < rows_used; r0 += pass) {
        const int nr = min(pass, rows_used - r0);
        if (r0 > 0) __syncthreads();
        // Rows r0 .. r0 + nr - 1, columns [k0, k1), into shared memory.  With kSquares every thread also adds up the squares of
        // its columns (the same columns of every row, so a row's sum has the same order whatever the number of rows).
        auto stage = [&](auto squares_tag, auto store_tag, int k0, int k1) {
            constexpr bool kSquares = decltype(squares_tag)::value, kStore = decltype(store_tag)::value;
            float sq[kSquares ? kRB : 1];
#pragma unroll
            for (int r = 0; r < (kSquares ? kRB : 1); ++r) sq[r] = 0.f;
#pragma unroll 1
            for (int k = k0 + 4 * tid; k < k1; k += 4 * kWarps * 32) {
                float4 gn = make_float4(1.f, 1.f, 1.f, 1.f);
                if (kNorm && kStore) gn = load4_each(g.gain + k);
#pragma unroll
                for (int q = 0; q < kRB; q += 4) {  // four rows' loads in flight
                    if (q < nr) {
                        float4 v[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            v[u] = q + u < nr ? __ldcg(reinterpret_cast<const float4*>(g.act + (int64_t)(r0 + q + u) * K + k))
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            if (kSquares) {
                                float s = sq[kSquares ? q + u : 0];
                                s = __fmaf_rn(v[u].x, v[u].x, s); s = __fmaf_rn(v[u].y, v[u].y, s);
                                s = __fmaf_rn(v[u].z, v[u].z, s); s = __fmaf_rn(v[u].w, v[u].w, s);
                                sq[kSquares ? q + u : 0] = s;
                            }
                            if (kStore)
                                *reinterpret_cast<float4*>(sA + (q + u) * KS + (k - k0)) =
                                    kNorm ? make_float4(v[u].x * gn.x, v[u].y * gn.y, v[u].z * gn.z, v[u].w * gn.w) : v[u];
                        }
                    }
                }
            }
            if constexpr (kSquares) {  // sixteen rows' sums over the lanes: as in exchange32, lanes 2 r and 2 r + 1 end with row r
#pragma unroll
                for (int w = 16, n = 8; n >= 1; w >>= 1, n >>= 1) {
                    const bool up = lane & w;
#pragma unroll
                    for (int r = 0; r < n; ++r) {
                        const float send = up ? sq[r] : sq[r + n], keep = up ? sq[r + n] : sq[r];
                        sq[r] = keep + __shfl_xor_sync(0xffffffffu, send, w);
                    }
                }
                sq[0] += __shfl_xor_sync(0xffffffffu, sq[0], 1);
                if ((lane & 1) == 0) s_ss[lane >> 1][warp] = sq[0];
            }
        };
        using Yes = std::true_type;
        using No = std::false_type;
        if constexpr (RES) {
            stage(std::integral_constant<bool, kNorm>{}, Yes{}, 0, K);
            __syncthreads();
        } else if constexpr (kNorm) {
            stage(Yes{}, No{}, 0, K);
        }
        const int my_row = lane & 15, side = lane >> 4;  // after the exchange a lane holds one row's sum of one feature
        const bool row_on = my_row < nr;
        const int pos = MODE == kRowQKV && row_on ? __ldcg(&g.rows->pos[r0 + my_row]) : -1;
        const int seq = MODE == kRowQKV && row_on ? __ldcg(&g.rows->seq[r0 + my_row]) : 0;
        float best = -INFINITY;
        int best_i = 0x7fffffff;

#pragma unroll 1
        for (int round = 0; round < rounds; ++round) {
            const int unit = round * per_round + (int)blockIdx.x * per_cta + slot;
            const bool unit_on = unit < g.n_units && part == 0;
            float x_old = 0.f;
            if (MODE == kRowResid && row_on && unit_on && 2 * unit + side < g.n_out)
                x_old = __ldcg(&g.out[(int64_t)(r0 + my_row) * g.ld + 2 * unit + side]);
            float acc[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = 0.f;
#pragma unroll 1
            for (int cc = 0; cc < n_turns; ++cc) {  // the same number of turns for every warp; a turn past the end multiplies zeros
                const int c = (cc << g.split_lg) + part;
                if constexpr (!RES) {
                    __syncthreads();
                    stage(No{}, Yes{}, c * kKC, min(K, (c + 1) * kKC));  // (split is 1 here: one chunk for all warps)
                    __syncthreads();
                }
                uint4 w[2][NV];
#pragma unroll
                for (int i = 0; i < NV; ++i) { w[0][i] = w_next[0][i]; w[1][i] = w_next[1][i]; }
                // the next turn's weights: of this unit, of the next one, or of the first one again for the next pass
                const bool more = cc + 1 < n_turns, last = round + 1 == rounds;
                if (more || !last || r0 + pass < rows_used) load_weights(more ? round : (last ? 0 : round + 1), more ? c + split : part, w_next);
                const int c0 = RES ? c * kKC : 0;
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    const int kl = (i * 32 + lane) * VN;
                    if (c * kKC + i * 32 * VN < K) {  // uniform: a chunk may end early
                        const bool in = c * kKC + kl < K;
                        float wa[VN], wb[VN];
                        Vec16<T>::widen(w[0][i], wa);
                        Vec16<T>::widen(w[1][i], wb);
                        const float* ap = sA + c0 + (in ? kl : 0);
#pragma unroll
                        for (int q = 0; q < kRB; q += 4) {
                            if (q < nr) {
#pragma unroll
                                for (int u = 0; u < 4; ++u) {
#pragma unroll
                                    for (int v4 = 0; v4 < VN; v4 += 4) {
                                        const float4 a = *reinterpret_cast<const float4*>(ap + (q + u) * KS + v4);
                                        acc[q + u] = fmaf(wa[v4], a.x, acc[q + u]); acc[16 + q + u] = fmaf(wb[v4], a.x, acc[16 + q + u]);
                                        acc[q + u] = fmaf(wa[v4 + 1], a.y, acc[q + u]); acc[16 + q + u] = fmaf(wb[v4 + 1], a.y, acc[16 + q + u]);
                                        acc[q + u] = fmaf(wa[v4 + 2], a.z, acc[q + u]); acc[16 + q + u] = fmaf(wb[v4 + 2], a.z, acc[16 + q + u]);
                                        acc[q + u] = fmaf(wa[v4 + 3], a.w, acc[q + u]); acc[16 + q + u] = fmaf(wb[v4 + 3], a.w, acc[16 + q + u]);
                                    }
                                }
                            }
                        }
                    }
                }
            }
            float val = exchange32(acc, lane);
            if (split > 1) {  // the unit's warps in chunk order
                s_part[warp][lane] = val;
                __syncthreads();
                if (part == 0)
#pragma unroll 1
                    for (int i = 1; i < split; ++i) val += s_part[warp + i][lane];
                __syncthreads();
            }
            if (kNorm) {
                float tot = 0.f;
#pragma unroll
                for (int w = 0; w < kWarps; ++w) tot += s_ss[my_row][w];  // fixed order
                val *= rsqrtf(tot / (float)K + g.eps);
            }
            const float other = __shfl_xor_sync(0xffffffffu, val, 16);  // the unit's other feature, same row
            if (!unit_on || !row_on) continue;
            if constexpr (MODE == kRowQKV) {
                if (pos < 0) continue;
                int mat, head, i;
                qkv_unit(unit, mat, head, i);
                const int idx = i + side * half;
                float rot = val;
                if (mat < 2) {
                    const float cs = __ldg(&g.rope_cos[(int64_t)pos * half + i]), sn = __ldg(&g.rope_sin[(int64_t)pos * half + i]);
                    rot = side == 0 ? val * cs - other * sn : other * sn + val * cs;
                }
                g.out[(int64_t)(r0 + my_row) * g.ld + mat * HD + head * hd + idx] = mat == 0 ? rot : val;
                if (mat > 0) {
                    T* cache = reinterpret_cast<T*>(mat == 1 ? g.kcache : g.vcache);
                    cache[kv_row_index(g.dims, g.layer, seq, head, pos) * hd + idx] = from_f32<T>(rot);
                }
            } else if constexpr (MODE == kRowSwiGLU) {
                if (side == 0) g.out[(int64_t)(r0 + my_row) * g.ld + unit] = val / (1.f + expf(-val)) * other;
            } else {
                const int n = 2 * unit + side;
                if (n >= g.n_out) continue;
                if constexpr (MODE == kRowResid) {
                    g.out[(int64_t)(r0 + my_row) * g.ld + n] = x_old + val;
                } else {
                    if (g.out) g.out[(int64_t)(r0 + my_row) * g.ld + n] = val;
                    if (val > best || (val == best && n < best_i)) { best = val; best_i = n; }
                }
            }
        }
        if constexpr (MODE == kRowHead) {  // the CTA's (maximum, lowest index) of every row
            const float ov = __shfl_xor_sync(0xffffffffu, best, 16);
            const int oi = __shfl_xor_sync(0xffffffffu, best_i, 16);
            if (ov > best || (ov == best && oi < best_i)) { best = ov; best_i = oi; }
            if (side == 0) { s_bv[warp][my_row] = best; s_bi[warp][my_row] = best_i; }
            __syncthreads();
            if (tid < nr) {
                float bv = s_bv[0][tid];
                int bi = s_bi[0][tid];
                for (int w = 1; w < kWarps; ++w)
                    if (s_bv[w][tid] > bv || (s_bv[w][tid] == bv && s_bi[w][tid] < bi)) { bv = s_bv[w][tid]; bi = s_bi[w][tid]; }
                g.part_max[(int64_t)blockIdx.x * g.dims.row_cap + r0 + tid] = bv;
                g.part_idx[(int64_t)blockIdx.x * g.dims.row_cap + r0 + tid] = bi;
            }
        }
    }
}

// ---- launchers -------------------------------------------------------------------------------
template <typename T, int MODE, int ROWS>
static cudaError_t opt_in() {
    return cudaFuncSetAttribute(rowgemm_kernel<T, MODE, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResidentBytes);
}
template <typename T, int ROWS>
static cudaError_t opt_in_modes() {
    cudaError_t e;
    if ((e = opt_in<T, kRowQKV, ROWS>()) != cudaSuccess) return e;
    if ((e = opt_in<T, kRowResid, ROWS>()) != cudaSuccess) return e;
    if ((e = opt_in<T, kRowSwiGLU, ROWS>()) != cudaSuccess) return e;
    return opt_in<T, kRowHead, ROWS>();
}
// (First mentioned in this order: instances lie in the library in the reverse order of their first mention, and what a launch costs
// depends on where its code lies, fetched anew as it is.  64 tokens of a fp32 decoder of width 256 take 2514 us with the kWhole
// instances ahead of the kFewer ones, 2524 behind them and 2540 with those of every mode side by side; 2497 without any kFewer.)
cudaError_t init_rowgemm(bool bf16) {  // the chunked instances stay within the default shared memory
    const cudaError_t e = bf16 ? opt_in_modes<__nv_bfloat16, kFewer>() : opt_in_modes<float, kFewer>();
    if (e != cudaSuccess) return e;
    return bf16 ? opt_in_modes<__nv_bfloat16, kWhole>() : opt_in_modes<float, kWhole>();
}

// Rows per pass over the weights (a multiple of 4): 16, or fewer where 16 rows do not fit shared memory whole and fewer do; the
// passes then share a step's rows evenly.  Fetching rows chunk by chunk, for every turn of the units and between two barriers, costs more
// than reading the weights once more.  us per step, chunk by chunk -> whole in more passes (one warp per output before): two bf16
// layers of width 4160, 16 rows 2831 -> 1283 (2157), 144 rows 24400 -> 10650 (17660); width 5184, 9 rows 3308 -> 1810 (2401); one of
// width 8256, 5 rows 1767 -> 869 (964); two fp32 layers of width 4096, 16 rows 2562 -> 1420 (3314).
static int pass_rows_of(int row_bound, int k_in) {
    const int rows = (row_bound + 3) / 4 * 4;
    const int most = (int)(kResidentBytes / (4 * sizeof(float) * k_in)) * 4;
    if (most < 4 || most >= kRB) return rows < kRB ? rows : kRB;
    const int passes = (rows + most - 1) / most;
    return ((rows + passes - 1) / passes + 3) / 4 * 4;
}
int rowgemm_passes(int rows, int k_in) {
    const int each = pass_rows_of(rows, k_in);
    return (rows + each - 1) / each;
}
static bool is_resident(int pass_rows, int k_in) { return (size_t)pass_rows * k_in * sizeof(float) <= kResidentBytes; }
static int cta_cap(int k_in, int pass_rows, int num_sms) {  // CTAs that the GPU holds at once
    return num_sms * (is_resident(2 * pass_rows, k_in) ? 2 : 1);
}
// Warps per unit: more than one where the units leave SMs without work and the columns make several chunks (output and down
// projections of narrow decoders: 512 units of width 1024 are 64 CTAs).
static int rowgemm_split(int n_units, int k_in, int pass_rows, int num_sms) {
    if (!is_resident(pass_rows, k_in)) return 1;
    const int cap = cta_cap(k_in, pass_rows, num_sms), chunks = (k_in + kKC - 1) / kKC;
    int split = 1;
    while (split < 4 && 2 * split <= chunks && (n_units * 2 * split + kWarps - 1) / kWarps <= cap) split *= 2;
    return split;
}
// Beyond what the GPU holds at once the units are dealt in equal rounds.
int rowgemm_grid(int n_units, int k_in, int row_bound, int num_sms) {
    const int rows = pass_rows_of(row_bound, k_in);
    const int per_cta = kWarps / rowgemm_split(n_units, k_in, rows, num_sms), cap = cta_cap(k_in, rows, num_sms);
    const int ctas = (n_units + per_cta - 1) / per_cta;
    const int rounds = (ctas + cap - 1) / cap;
    return (ctas + rounds - 1) / rounds;
}

template <typename T, int ROWS>
static void launch_typed(cudaStream_t st, int grid, size_t smem, const RowGemm& g) {
    switch (g.mode) {
        case kRowQKV: launch_pdl(st, true, dim3(grid), dim3(kWarps * 32), smem, rowgemm_kernel<T, kRowQKV, ROWS>, g); break;
        case kRowResid: launch_pdl(st, true, dim3(grid), dim3(kWarps * 32), smem, rowgemm_kernel<T, kRowResid, ROWS>, g); break;
        case kRowSwiGLU: launch_pdl(st, true, dim3(grid), dim3(kWarps * 32), smem, rowgemm_kernel<T, kRowSwiGLU, ROWS>, g); break;
        default: launch_pdl(st, true, dim3(grid), dim3(kWarps * 32), smem, rowgemm_kernel<T, kRowHead, ROWS>, g); break;
    }
}
template <typename T>
static void launch_rows(cudaStream_t st, int grid, size_t smem, Rows rows, const RowGemm& g) {
    if (rows == kWhole) launch_typed<T, kWhole>(st, grid, smem, g);
    else if (rows == kFewer) launch_typed<T, kFewer>(st, grid, smem, g);
    else launch_typed<T, kChunked>(st, grid, smem, g);
}

void launch_rowgemm(cudaStream_t st, bool bf16, RowGemm g, int row_bound, int num_sms) {
    g.pass_rows = pass_rows_of(row_bound, g.k_in);
    const bool resident = is_resident(g.pass_rows, g.k_in);
    const size_t smem = (size_t)g.pass_rows * (resident ? g.k_in : kKC) * sizeof(float);
    const int split = rowgemm_split(g.n_units, g.k_in, g.pass_rows, num_sms);
    g.split_lg = split == 4 ? 2 : split - 1;
    const int grid = rowgemm_grid(g.n_units, g.k_in, row_bound, num_sms);
    // (a step of no more rows than a pass takes has one pass whatever its length)
    const Rows rows = !resident ? kChunked : (g.pass_rows < kRB && row_bound > g.pass_rows ? kFewer : kWhole);
    if (bf16) launch_rows<__nv_bfloat16>(st, grid, smem, rows, g);
    else launch_rows<float>(st, grid, smem, rows, g);
}

}  // namespace llma
