// Weight-streaming GEMM for up to 256 activation rows (batched decoding steps).
// Same contract, work split and fused epilogues as gemm_ws_kernel (see gemm_tcgen05.cuh); what differs:
//   * the activation tiles are large enough for TMA to pay: a ring stage holds the weight tile of one 64-wide
//     k-chunk and, behind it, the chunk's activation tile (the nr hi rows, then the nr lo rows, fetched by one
//     copy through a 3-D view of the split buffer); two producer warps fill the two halves of a stage, because
//     only the activations have to wait for the kernel before;
//   * an accumulator has 2 nr columns [hi | lo], summed by the epilogue: up to 128 rows one MMA of N = 2 nr per
//     k-slice and two accumulators in turn; beyond, two MMAs per k-slice (N = the rows in use rounded up to 16,
//     a run-time field of the instruction descriptor) and a single accumulator.  An MMA of this shape (M 128, K 16)
//     takes 21.7 ns at N = 32, 35 at 128 and 69 at 256 (N / 256 of the full rate from 128 on), so a 16 KB weight tile
//     costs 0.09 to 0.28 us of tensor time against 0.37 us of HBM time;
//   * the rows a copy brings (nr: 32, 64, 128 or the launch's capacity) are chosen per step from the rows in use;
//   * the epilogue walks a finished 128 x nr accumulator in blocks of 32 rows; tiles cut by a range boundary
//     are summed and finished block by block by all the CTAs that share them.
//
// Roles inside one CTA of 224 threads:
//   warps 0-3  epilogue: TMEM -> registers -> workspace (cut tiles) or fused epilogue, block by block; then the
//              blocks of cut tiles dealt to this CTA
//   warp  4    one thread issues the TMA loads of the weight tiles (they depend on no earlier kernel)
//   warp  5    MMA: allocates TMEM; one thread issues tcgen05.mma and the commits
//   warp  6    one thread issues the TMA loads of the activation tiles (after the dependency wait)
//
// The start and the end of a launch run code for the first time, and integer divisions by run-time values were 5 KB of it: with
// the ranges, tiles, stages and the dealing of blocks counted up instead, a pass of two layers of width 1024 with sixteen
// sequences takes 163 us (171 before), of four layers of the 7B widths with four sequences 542 us (559).
//
// Every wait is bounded: when one runs out the kernel raises the device error word, stops
// issuing work, lets its outstanding copies land, frees TMEM and returns.
#include <cuda.h>

#include <type_traits>

#include "gemm_epilogue.cuh"
#include "gemm_tcgen05.cuh"
#include "ptx_sm100.cuh"

namespace llma {

using namespace ptx;

constexpr size_t kWideStageBytes = 32 * kBlockLd * 4;
constexpr size_t kWideTailBytes = 5120;  // barriers, flags, per-row scales, reduction scratch, row positions and slots

template <int MODE>
__global__ void __launch_bounds__(kGemmWideThreads, 1)
gemm_wide_kernel(const __grid_constant__ GemmArgs g, const __grid_constant__ CUtensorMap map_a0, const __grid_constant__ CUtensorMap map_a1,
                 const __grid_constant__ CUtensorMap map_a2, const __grid_constant__ CUtensorMap map_b0,
                 const __grid_constant__ CUtensorMap map_b1, const __grid_constant__ CUtensorMap map_b2,
                 const __grid_constant__ CUtensorMap map_b3, const int S, const uint32_t tmem_cols) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));
    // g.nr is the row capacity the launch was shaped for; the rows a copy brings (nr below) are chosen per step from
    // the rows in use, by every role that needs them, once the planning kernel's count may be read
    const uint32_t stage_bytes = kGemmABytes + (uint32_t)g.nr * 256u;  // weight tile, then the largest activation tile
    auto box_index = [&](int rows_used) {
        int i = 0;
        while (i < 3 && wide_box_rows(g.nr, i) < rows_used) ++i;
        return i;
    };
    const uint32_t sA = base, sB = base + kGemmABytes;   // stage s: sA + s * stage_bytes, sB + s * stage_bytes
    uint8_t* after = gen_base + (size_t)S * stage_bytes;
    float (*stage)[kBlockLd] = reinterpret_cast<float (*)[kBlockLd]>(after);
    uint8_t* tail = after + kWideStageBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(tail);  // full[8], empty[8], acc_full[2], acc_empty[2]
    volatile uint32_t* sh = reinterpret_cast<volatile uint32_t*>(tail + 20 * 8);  // [0] TMEM base, [1] abort, [2] broadcast
    float* rscale = reinterpret_cast<float*>(tail + 20 * 8 + 16);                 // [256] per-row norm scales
    int* s_pos = reinterpret_cast<int*>(rscale + kRowCap);                                                     // [256] (QKV mode)
    int* s_seq = s_pos + kRowCap;                                                 // [256]
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };  // both halves of a stage: two arrivals with their byte counts
    auto empty_bar = [&](int s) { return bar0 + 8u * (8 + s); };
    auto accf_bar = [&](int i) { return bar0 + 8u * (16 + i); };
    auto acce_bar = [&](int i) { return bar0 + 8u * (18 + i); };

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int G = gridDim.x, b = blockIdx.x;
    const int C = g.chunks;
    const int work = g.n_tiles * C;
    // equal ranges, the first `extra` CTAs one item longer
    const int share = work / G, extra = work - share * G;
    auto begin_of = [&](int cta) { return cta * share + min(cta, extra); };
    const int w_beg = begin_of(b), w_end = begin_of(b + 1);
    const int tile0 = w_beg / C, c_beg = w_beg - tile0 * C;  // the first item: tile and chunk within it
    const int n_items = w_end - w_beg;

    grid_launch_dependents();  // the next kernel may begin its own prologue now
    [[maybe_unused]] unsigned long long* stp = LLMA_STAMP_PTR(g.stamps, g.launch_id, blockIdx.x);
    if (threadIdx.x == 0) LLMA_STAMP(stp, 0);
    if (threadIdx.x == 0) {
        for (int s = 0; s < 8; ++s) {
            mbar_init(full_bar(s), 2); mbar_init(empty_bar(s), 1);
        }
        for (int i = 0; i < 2; ++i) { mbar_init(accf_bar(i), 1); mbar_init(acce_bar(i), 4); }
        sh[1] = 0; sh[2] = 0;
        fence_mbar_init();
    }
    if (warp == 5) {
        tmem_alloc(smem_u32((const void*)&sh[0]), tmem_cols);
        tmem_relinquish();
    }
    if (warp == 4 && lane == 0) {
        tma_prefetch_desc(&map_a0);
        if (MODE == kGemmQKV) { tma_prefetch_desc(&map_a1); tma_prefetch_desc(&map_a2); }
        if (MODE == kGemmSwiGLU) tma_prefetch_desc(&map_a1);
    }
    if (warp == 6 && lane == 0) { tma_prefetch_desc(&map_b0); tma_prefetch_desc(&map_b1); tma_prefetch_desc(&map_b2); tma_prefetch_desc(&map_b3); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh[0];

    // Stage, parity, tile and chunk of the next item are kept as running counters: divisions by run-time values would
    // cost the issuing threads as much as the copies.
    if (warp == 4) {
        // ------------------------------- weight producer ------------------------------------------
        if (elect_one()) {
            const uint64_t policy = l2_evict_first();
            int it = 0;
            int tile = tile0, c = c_beg;
            int m = 0, rt = tile;  // matrix and tile inside it
            if (MODE == kGemmQKV)
                for (; rt >= g.tiles_per_map; ++m) rt -= g.tiles_per_map;
            int s = 0;
            uint32_t ph = 0;
#pragma unroll 1
            for (; it < n_items && !sh[1]; ++it) {
                if (it >= S && !mbar_wait(empty_bar(s), ph ^ 1u)) { atomicExch(g.dev_err, kDevErrTimeout); sh[1] = 1; break; }
                mbar_arrive_expect_tx(full_bar(s), kGemmABytes);
                const uint32_t dstA = sA + (uint32_t)s * stage_bytes;
                if (MODE == kGemmSwiGLU) {
                    tma_load_2d(dstA, &map_a0, full_bar(s), c * 64, tile * 64, policy);
                    tma_load_2d(dstA + kGemmABytes / 2, &map_a1, full_bar(s), c * 64, tile * 64, policy);
                } else {
                    const CUtensorMap* mp = m == 0 ? &map_a0 : (m == 1 ? &map_a1 : &map_a2);
                    tma_load_2d(dstA, mp, full_bar(s), c * 64, rt * 128, policy);
                }
                if (++c == C) { c = 0; ++tile; if (++rt == g.tiles_per_map) { rt = 0; ++m; } }
                if (++s == S) { s = 0; ph ^= 1u; }
            }
            if (sh[1]) {  // give up: let the copies already issued land before the CTA's memory goes away
#pragma unroll 1
                for (int j = it - 1; j >= 0 && j >= it - S; --j)
                    (void)mbar_wait(full_bar(j % S), (uint32_t)((j / S) & 1), 100000000ull);
            }
        }
    } else if (warp == 6) {
        // ------------------------------- activation producer --------------------------------------
        if (elect_one()) {
            grid_dependency_wait();  // activations are written by the kernel before this one
            const int bi = box_index(g.rows ? min(__ldcg(&g.rows->rows_used), g.nr) : g.nr);
            const CUtensorMap* map_b = bi == 0 ? &map_b0 : (bi == 1 ? &map_b1 : (bi == 2 ? &map_b2 : &map_b3));
            const uint32_t b_slot = (uint32_t)wide_box_rows(g.nr, bi) * 256u;  // hi rows, then lo rows, of one k-chunk
            int q = 0;
            int c = c_beg;
            int s = 0;
            uint32_t ph = 0;
#pragma unroll 1
            for (; q < n_items && !sh[1]; ++q) {
                if (q >= S && !mbar_wait(empty_bar(s), ph ^ 1u)) { atomicExch(g.dev_err, kDevErrTimeout); sh[1] = 1; break; }
                mbar_arrive_expect_tx(full_bar(s), b_slot);
                tma_load_3d(sB + (uint32_t)s * stage_bytes, map_b, full_bar(s), c * 64, 0, 0);
                if (++c == C) c = 0;
                if (++s == S) { s = 0; ph ^= 1u; }
            }
            if (sh[1]) {
#pragma unroll 1
                for (int j = q - 1; j >= 0 && j >= q - S; --j)
                    (void)mbar_wait(full_bar(j % S), (uint32_t)((j / S) & 1), 100000000ull);
            }
        }
    } else if (warp == 5) {
        // ------------------------------- MMA issuer ---------------------------------------------
        if (elect_one()) {
            grid_dependency_wait();  // the count of rows in use comes from the planning kernel
            int rows_used = g.rows ? __ldcg(&g.rows->rows_used) : g.nr;
            rows_used = max(1, min(rows_used, g.nr));
            const int nr = wide_box_rows(g.nr, box_index(rows_used));  // hi rows at 0, lo rows nr further on
            // An accumulator has 2 nr columns [hi | lo]; two accumulators take turns while they fit the 512 TMEM
            // columns, else there is one.
            const int acc_cols = 2 * nr;
            const int n_acc = 2 * acc_cols <= 512 ? 2 : 1;
            // Up to 128 rows: one MMA per k-slice over the hi and the lo rows together (N = 2 nr, columns [hi | lo]).
            // Beyond (N = 2 nr would pass the instruction's 256): two MMAs per k-slice, the hi rows into the first
            // nr columns and the lo rows into the next nr, N = the rows in use rounded up to 16.  Either way a
            // column is summed over k in the same order, so a row's result does not depend on which applies.
            const bool one_mma = 2 * nr <= 256;
            const uint32_t idesc = idesc_bf16_m128(one_mma ? (uint32_t)(2 * nr) : (uint32_t)((rows_used + 15) & ~15));
            int ia = 0;
            int s = 0;            // ring stage of item ia and the parity of its use: kept by hand, a division by the
            uint32_t s_ph = 0;    // run-time ring depth would cost this thread more than a commit
            int seg = 0;
#ifdef LLMA_STAMPS
            // measurement build: time this thread spends waiting for ring stages (word 6), in ns
            unsigned long long wait_a = 0, tw;
#define LLMA_WAIT_BEGIN() (tw = globaltimer_ns())
#define LLMA_WAIT_END(acc) (acc += globaltimer_ns() - tw)
#else
#define LLMA_WAIT_BEGIN() ((void)0)
#define LLMA_WAIT_END(acc) ((void)0)
#endif
#pragma unroll 1
            for (int w = w_beg, c0 = c_beg; w < w_end && !sh[1]; ++seg, c0 = 0) {
                const int c1 = min(C, c0 + (w_end - w));
                const int buf = n_acc == 2 ? (seg & 1) : 0;
                const uint32_t use = (uint32_t)(n_acc == 2 ? seg >> 1 : seg);
                if (!mbar_wait(acce_bar(buf), (use & 1u) ^ 1u)) { atomicExch(g.dev_err, kDevErrTimeout); sh[1] = 1; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)buf * (uint32_t)acc_cols;
#pragma unroll 1
                for (int c = c0; c < c1 && !sh[1]; ++c, ++ia) {
                    LLMA_WAIT_BEGIN();
                    if (!mbar_wait(full_bar(s), s_ph)) { atomicExch(g.dev_err, kDevErrTimeout); sh[1] = 1; break; }
                    LLMA_WAIT_END(wait_a);
                    if (ia == 0) LLMA_STAMP(stp, 2);
                    tc_fence_after();
                    const uint64_t da = smem_desc_sw128(sA + (uint32_t)s * stage_bytes);
                    const uint64_t db = smem_desc_sw128(sB + (uint32_t)s * stage_bytes);
                    const uint64_t db_lo = smem_desc_sw128(sB + (uint32_t)s * stage_bytes + (uint32_t)nr * 128u);
                    const uint32_t acc_on = c > c0 ? 1u : 0u;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {  // 4 x K=16 slices of the 64-wide chunk: +32 bytes each
                        umma_bf16(d_tmem, da + 2 * kk, db + 2 * kk, idesc, (acc_on || kk > 0) ? 1u : 0u);
                        if (!one_mma) umma_bf16(d_tmem + (uint32_t)nr, da + 2 * kk, db_lo + 2 * kk, idesc, (acc_on || kk > 0) ? 1u : 0u);
                    }
                    umma_commit(empty_bar(s));  // the stage is free once these MMAs have read it
                    if (++s == S) { s = 0; s_ph ^= 1u; }
                }
                if (sh[1]) break;
                umma_commit(accf_bar(buf));  // accumulator complete
                LLMA_STAMP(stp, 3);
                w += c1 - c0;
            }
#ifdef LLMA_STAMPS
            if (stp) stp[6] = wait_a;
#endif
        }
    } else {
        // ------------------------------- epilogue warps ------------------------------------------
        grid_dependency_wait();  // everything below reads or writes what earlier kernels produced
        if (threadIdx.x == 0) LLMA_STAMP(stp, 1);
        const int rows_used = g.rows ? min(g.rows->rows_used, g.nr) : g.nr;
        const int nr = wide_box_rows(g.nr, box_index(max(rows_used, 1)));  // as the MMA warp sees it
        const int acc_cols = 2 * nr;
        const int n_acc = 2 * acc_cols <= 512 ? 2 : 1;
        const int nblk = (rows_used + 31) >> 5;
        const int row = threadIdx.x;  // 0..127 = TMEM lane = output feature inside the tile
        if (g.ss_in) {  // folded RMSNorm: one scale per activation row, tiles summed in ascending order
#pragma unroll 1
            for (int r = row; r < rows_used; r += 128) {
                float ssum = 0.f;
                int t = 0;
#pragma unroll 1
                for (; t + 8 <= g.ss_tiles; t += 8) {  // eight loads in flight
                    float v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u] = __ldcg(&g.ss_in[(int64_t)(t + u) * g.rc + r]);
#pragma unroll
                    for (int u = 0; u < 8; ++u) ssum += v[u];
                }
#pragma unroll 1
                for (; t < g.ss_tiles; ++t) ssum += __ldcg(&g.ss_in[(int64_t)t * g.rc + r]);
                rscale[r] = rsqrtf(ssum * g.norm_inv + g.norm_eps);
            }
        }
        if (MODE == kGemmQKV) {  // the rows' positions and sequence slots, read once per CTA
#pragma unroll 1
            for (int r = row; r < rows_used; r += 128) {
                s_pos[r] = __ldcg(&g.rows->pos[r]);
                s_seq[r] = __ldcg(&g.rows->seq[r]);
            }
        }
        epi_sync();
        // Tiles cut by a range boundary are summed block by block: every CTA of such a tile writes its whole partial into its own
        // workspace slot -- slot 0 for the tile its range begins in, slot 1 for any other -- and raises the slot's flag to
        // this launch's number.  The tile's rows are dealt over its CTAs in blocks of 32 (of 16 where the tile has at
        // least as many CTAs as 16-row blocks): after its last segment a CTA waits for the flags of all the tile's CTAs, adds
        // up the partials of its blocks in ascending k order, two CTAs' loads in flight, and runs the blocks' epilogues.
        // Launch numbers differ from step to step (the planning kernel counts the steps), so nothing is reset.  (Words that
        // read as "empty" until handed over, polled one CTA at a time and reset, had cost 12 us at the end of a launch at
        // 36 rows and 25 at 144.)
        // slots are laid out for the engine's row capacity
        const int qn = g.rc >> 2;
        const int tile_first = tile0;
        const uint32_t epoch = (g.rows ? (uint32_t)__ldcg(&g.rows->step_no) : 0u) * 65536u + (uint32_t)g.launch_seq + 1u;
        int tile_last = tile0;
        while ((tile_last + 1) * C < w_end) ++tile_last;
        // One loop over everything this CTA stages and finishes -- first the blocks of its accumulators (those of cut tiles go
        // to the workspace instead), then the blocks of cut tiles dealt to it -- with one copy of the epilogue: the end of a
        // launch runs its code for the first time, so what it costs is also the code it has to fetch.
        int w = w_beg, seg = 0, rb = 0, tile = 0, buf = 0;  // accumulators: next item, segment, block, tile, TMEM buffer
        bool in_seg = false, shared_tile = false, collecting = w_beg >= w_end;
        int which = 0, u = 0, n_units = 0, unit = 32;       // cut tiles: first and last tile of the range, unit of rows
        int b_first = 0, b_last = 0, P = 1, odd = -1, dealt = 0, carry = 0;
        bool waited = false;
        unsigned long long give_up = 0;
#pragma unroll 1
        for (;;) {
            float acc[32];
            int r_lo, r_hi;
            if (!collecting) {
                if (!in_seg) {
                    if (w >= w_end) { collecting = true; give_up = globaltimer_ns() + 2000000000ull; continue; }
                    tile = tile0 + seg;
                    w = min(w_end, (tile + 1) * C);
                    buf = n_acc == 2 ? (seg & 1) : 0;
                    const uint32_t use = (uint32_t)(n_acc == 2 ? seg >> 1 : seg);
                    if (threadIdx.x == 0) {
                        bool ok = !sh[1] && mbar_wait(accf_bar(buf), use & 1u);
                        if (!ok) { atomicExch(g.dev_err, kDevErrTimeout); sh[1] = 1; }
                        sh[2] = ok ? 1u : 0u;
                    }
                    epi_sync();
                    const bool ok = sh[2] != 0;
                    epi_sync();
                    if (!ok) break;
                    if (threadIdx.x == 0) LLMA_STAMP(stp, 4);
                    tc_fence_after();
                    shared_tile = w_beg > tile * C || w_end < (tile + 1) * C;
                    in_seg = true;
                    rb = 0;
                }
                if (rb == nblk) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acce_bar(buf));  // MMA may overwrite this accumulator
                    if (shared_tile) {
                        epi_sync();
                        if (threadIdx.x == 0) { __threadfence(); st_release(g.flags + 2 * b + (tile == tile_first ? 0 : 1), epoch); }
                    }
                    in_seg = false;
                    ++seg;
                    continue;
                }
                const uint32_t t0 = tmem_base + ((uint32_t)(warp * 32) << 16) + (uint32_t)buf * (uint32_t)acc_cols + (uint32_t)rb * 32u;
                tmem_ld_32cols(t0, acc);
                {
                    float lo[32];
                    tmem_ld_32cols(t0 + (uint32_t)nr, lo);
#pragma unroll
                    for (int j = 0; j < 32; ++j) acc[j] += lo[j];  // W * hi + W * lo
                }
                r_lo = rb * 32;
                r_hi = min(rows_used, r_lo + 32);
                ++rb;
                if (shared_tile) {
                    float4* dst = ws_slot(g.ws, qn, 2 * b + (tile == tile_first ? 0 : 1), row) + (r_lo >> 2) * 128;
#pragma unroll
                    for (int q = 0; q < 8; ++q)  // only the columns of rows in use travel
                        if (r_lo + 4 * q < r_hi) dst[q * 128] = make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
                    continue;
                }
            } else {
                if (u == n_units) {
                    if (which == 2 || w_beg >= w_end) break;
                    tile = which == 0 ? tile_first : tile_last;
                    const int t_lo = tile * C, t_hi = t_lo + C;
                    u = n_units = 0;
                    if (++which == 2 && tile_last == tile_first) break;
                    if (!(w_beg > t_lo || w_end < t_hi)) continue;  // the whole tile was this CTA's: finished above
                    // the tile's CTAs: those whose ranges hold its first and its last chunk, and everyone between
                    b_first = b;
                    while (begin_of(b_first) > t_lo) --b_first;
                    b_last = b;
                    while (begin_of(b_last + 1) < t_hi) ++b_last;
                    P = b_last - b_first + 1;
                    odd = begin_of(b_first) < t_lo ? b_first : -1;  // the one CTA that may have it in slot 1
                    waited = false;
                    // units of 32 rows, or of 16 where that gives more of the tile's CTAs something to finish without
                    // giving any of them two units
                    unit = nblk < P && ((rows_used + 15) >> 4) <= P ? 16 : 32;
                    n_units = unit == 16 ? (rows_used + 15) >> 4 : nblk;
                    dealt = carry = 0;
                    continue;
                }
                const int mine = u++, to = dealt;  // unit i goes to the tile's CTA i P / n_units, rounded down
                for (carry += P; carry >= n_units; carry -= n_units) ++dealt;
                if (to != b - b_first) continue;
                if (!waited) {
#pragma unroll 1
                    for (int i = row; i < P; i += 128) {
                        const uint32_t* f = g.flags + 2 * (b_first + i) + (b_first + i == odd ? 1 : 0);
                        while (ld_acquire(f) != epoch) {
                            if (sh[1] || globaltimer_ns() > give_up) { atomicExch(g.dev_err, kDevErrTimeout); sh[1] = 1; break; }
                        }
                    }
                    epi_sync();
                    waited = true;
                }
                r_lo = mine * unit;
                r_hi = min(rows_used, r_lo + unit);
#pragma unroll
                for (int j = 0; j < 32; ++j) acc[j] = 0.f;
                constexpr int U = 2;  // CTAs whose partials are requested together
#pragma unroll 1
                for (int bb = b_first; bb <= b_last; bb += U) {  // ascending k: a fixed summation order
                    float4 p[U][8];
#pragma unroll
                    for (int v = 0; v < U; ++v) {
                        const int cta = min(bb + v, b_last);
                        const float4* src = ws_slot(g.ws, qn, 2 * cta + (cta == odd ? 1 : 0), row) + (r_lo >> 2) * 128;
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            if (r_lo + 4 * q < r_hi) p[v][q] = __ldcg(src + q * 128);
                    }
#pragma unroll
                    for (int v = 0; v < U; ++v) {
                        if (bb + v <= b_last) {
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                if (r_lo + 4 * q < r_hi) {
                                    acc[4 * q] += p[v][q].x; acc[4 * q + 1] += p[v][q].y;
                                    acc[4 * q + 2] += p[v][q].z; acc[4 * q + 3] += p[v][q].w;
                                }
                            }
                        }
                    }
                }
            }
            // rows r_lo .. r_hi - 1 are in acc: staged (scaled by the folded RMSNorm), then the fused epilogue
            stage_block(stage, row, acc, g.ss_in ? rscale + r_lo : nullptr);
            const int nj = r_hi - r_lo;
            auto sync = [] { epi_sync(); };
            if constexpr (MODE == kGemmQKV)
                block_qkv(g, tile, warp, lane, r_lo, nj, stage, [&](int j) { return s_pos[r_lo + j]; }, [&](int j) { return s_seq[r_lo + j]; }, sync);
            else if constexpr (MODE == kGemmResid) block_resid(g, tile, warp, lane, r_lo, nj, stage, sync);
            else if constexpr (MODE == kGemmSwiGLU) block_swiglu(g, tile, warp, lane, r_lo, nj, stage, sync);
            else block_lmhead(g, tile, warp, lane, r_lo, nj, stage, sync);
        }
    }
    if (threadIdx.x == 0) LLMA_STAMP(stp, 5);
    tc_fence_before();
    __syncthreads();
    if (warp == 5) {
        tc_fence_after();
        tmem_dealloc(tmem_base, tmem_cols);
    }
}

// ---- host side ------------------------------------------------------------------------------------
GemmWideCfg gemm_wide_cfg(int nr) {
    GemmWideCfg c;
    const size_t budget = (size_t)227 * 1024 - 1024 - kWideStageBytes - kWideTailBytes;
    const size_t stage_bytes = kGemmABytes + (size_t)nr * 256;
    int S = (int)(budget / stage_bytes);  // as many stages as fit, at most 8
    if (S > 8) S = 8;
    c.stages = S;
    uint32_t cols = 32;
    for (int i = 0; i < 4; ++i) {  // the largest need over the row counts a step may choose (as in the kernel)
        const uint32_t acc_cols = 2u * (uint32_t)wide_box_rows(nr, i);
        while (cols < (2u * acc_cols <= 512u ? 2u : 1u) * acc_cols) cols <<= 1;
    }
    c.tmem_cols = cols;
    c.smem_bytes = 1024 + (size_t)S * stage_bytes + kWideStageBytes + kWideTailBytes;
    if (c.smem_bytes < 120 * 1024) c.smem_bytes = 120 * 1024;  // one CTA per SM, as for the narrow kernel
    return c;
}

template <int MODE>
static cudaError_t wide_opt_in() {
    return cudaFuncSetAttribute(gemm_wide_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

cudaError_t init_gemm_wide() {
    cudaError_t e;
    if ((e = wide_opt_in<kGemmQKV>()) != cudaSuccess) return e;
    if ((e = wide_opt_in<kGemmResid>()) != cudaSuccess) return e;
    if ((e = wide_opt_in<kGemmSwiGLU>()) != cudaSuccess) return e;
    return wide_opt_in<kGemmLmHead>();
}

void launch_gemm_wide(cudaStream_t st, int grid, bool pdl, const GemmArgs& args, const CUtensorMap& a0,
                      const CUtensorMap& a1, const CUtensorMap& a2, const CUtensorMap* map_b) {
    const GemmWideCfg c = gemm_wide_cfg(args.nr);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kGemmWideThreads);
    cfg.dynamicSmemBytes = c.smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    const int stages = c.stages;
    const uint32_t cols = c.tmem_cols;
    switch (args.mode) {
        case kGemmQKV: cudaLaunchKernelEx(&cfg, gemm_wide_kernel<kGemmQKV>, args, a0, a1, a2, map_b[0], map_b[1], map_b[2], map_b[3], stages, cols); break;
        case kGemmResid: cudaLaunchKernelEx(&cfg, gemm_wide_kernel<kGemmResid>, args, a0, a1, a2, map_b[0], map_b[1], map_b[2], map_b[3], stages, cols); break;
        case kGemmSwiGLU: cudaLaunchKernelEx(&cfg, gemm_wide_kernel<kGemmSwiGLU>, args, a0, a1, a2, map_b[0], map_b[1], map_b[2], map_b[3], stages, cols); break;
        default: cudaLaunchKernelEx(&cfg, gemm_wide_kernel<kGemmLmHead>, args, a0, a1, a2, map_b[0], map_b[1], map_b[2], map_b[3], stages, cols); break;
    }
}

}  // namespace llma
