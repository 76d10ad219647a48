// Integer side of an LLMA decoding step as kernels of their own: step_tail (trigger search, copy, acceptance, K/V commit)
// and the embedding gather.
#include "step_tail.cuh"

namespace llma {

// step_tail (step_tail.cuh) as a kernel of one CTA
constexpr int kTailThreads = 1024;
__global__ void __launch_bounds__(kTailThreads) step_tail_kernel(const TailArgs a) {
    __shared__ TailShared sh;
    pdl_trigger();
    pdl_wait();
    step_tail<kTailThreads>(a, sh);
}

// --------------------------------------------------------------------------------------
// embedding gather: x[r, :] = tok_emb[tok[r], :] as fp32 (zero for unused rows)
// --------------------------------------------------------------------------------------
template <typename T>
__global__ void embed_kernel(ModelDims dims, const RowDesc* __restrict__ rows, const T* __restrict__ emb,
                             float* __restrict__ x, int32_t* __restrict__ dev_err) {
    pdl_trigger();
    pdl_wait();
    const int r = blockIdx.x;
    const int d = dims.d_model;
    float* xr = x + (int64_t)r * d;
    const int tok = rows->tok[r];
    const bool used = rows->pos[r] >= 0;
    const bool ok = used && tok >= 0 && tok < dims.vocab;
    if (used && !ok && threadIdx.x == 0) atomicExch(dev_err, kDevErrToken);
    const T* er = emb + (int64_t)(ok ? tok : 0) * d;
    for (int i = threadIdx.x; i < d; i += blockDim.x) xr[i] = ok ? to_f32<T>(er[i]) : 0.f;
}

// Embedding gather for the tensor-core path, with the first RMSNorm folded in: besides x it
// writes xs = split(x * gain) and, per 128-column tile, each row's sum of squares (the
// projections multiply by rsqrt(mean square + eps) afterwards).  One CTA of 128 threads per (row, 128-column tile).
__global__ void __launch_bounds__(128) embed_norm_kernel(ModelDims dims, const RowDesc* __restrict__ rows,
                                                         const __nv_bfloat16* __restrict__ emb,
                                                         const float* __restrict__ gain, float* __restrict__ x,
                                                         void* __restrict__ xs, float* __restrict__ ss,
                                                         int32_t* __restrict__ dev_err) {
    pdl_trigger();
    pdl_wait();
    const int r = blockIdx.x, t = blockIdx.y, d = dims.d_model;
    const int tok = rows->tok[r];
    const bool used = rows->pos[r] >= 0;
    const bool ok = used && tok >= 0 && tok < dims.vocab;
    if (used && !ok && t == 0 && threadIdx.x == 0) atomicExch(dev_err, kDevErrToken);
    const __nv_bfloat16* er = emb + (int64_t)(ok ? tok : 0) * d;
    __shared__ float red[4];
    const int col = t * 128 + threadIdx.x;
    float v = 0.f;
    if (col < d) {
        v = ok ? __bfloat162float(er[col]) : 0.f;
        x[(int64_t)r * d + col] = v;
        store_split(xs, dims.row_cap, r, col, d, v * gain[col]);
    }
    float sq = v * v;
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sq;
    __syncthreads();
    if (threadIdx.x == 0) ss[(int64_t)t * dims.row_cap + r] = ((red[0] + red[1]) + red[2]) + red[3];
}

// The same for the rows of a prompt pass (their tokens were checked on the host): one CTA of 128 threads per row.
__global__ void __launch_bounds__(128) embed_prompt_kernel(int d, int rc, const int32_t* __restrict__ toks,
                                                           const __nv_bfloat16* __restrict__ emb, const float* __restrict__ gain,
                                                           float* __restrict__ x, void* __restrict__ xs, float* __restrict__ ss) {
    pdl_trigger();
    pdl_wait();
    const int r = blockIdx.x;
    const __nv_bfloat16* er = emb + (int64_t)__ldg(&toks[r]) * d;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int t = warp; t < d / 128; t += 4) {  // d is a multiple of 128 on the tensor-core path
        const int col = t * 128 + lane * 4;
        const float4 v = load4_each(er + col), gn = load4_each(gain + col);
        *reinterpret_cast<float4*>(x + (int64_t)r * d + col) = v;
        store_split(xs, rc, r, col, d, v.x * gn.x);
        store_split(xs, rc, r, col + 1, d, v.y * gn.y);
        store_split(xs, rc, r, col + 2, d, v.z * gn.z);
        store_split(xs, rc, r, col + 3, d, v.w * gn.w);
        float sq = (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (lane == 0) ss[(int64_t)t * rc + r] = sq;
    }
}

// ---- launchers -----------------------------------------------------------------------
void launch_step_tail(cudaStream_t st, const TailArgs& a) {
    launch_pdl(st, true, dim3(1), dim3(kTailThreads), 0, step_tail_kernel, a);
}

void launch_embed(cudaStream_t st, const ModelDims& dims, bool bf16, int n_rows, const RowDesc* rows, const void* emb,
                  float* x, int32_t* dev_err) {
    if (bf16)
        launch_pdl(st, true, dim3(n_rows), dim3(256), 0, embed_kernel<__nv_bfloat16>, dims, rows, (const __nv_bfloat16*)emb, x, dev_err);
    else
        launch_pdl(st, true, dim3(n_rows), dim3(256), 0, embed_kernel<float>, dims, rows, (const float*)emb, x, dev_err);
}

void launch_embed_norm(cudaStream_t st, const ModelDims& dims, int n_rows, const RowDesc* rows, const void* emb,
                       const float* gain, float* x, void* xs, float* ss, int32_t* dev_err) {
    launch_pdl(st, true, dim3(n_rows, (dims.d_model + 127) / 128), dim3(128), 0, embed_norm_kernel, dims, rows,
               (const __nv_bfloat16*)emb, gain, x, xs, ss, dev_err);
}

void launch_embed_prompt(cudaStream_t st, const ModelDims& dims, int n_rows, int rc, const int32_t* toks, const void* emb,
                         const float* gain, float* x, void* xs, float* ss) {
    launch_pdl(st, true, dim3(n_rows), dim3(128), 0, embed_prompt_kernel, dims.d_model, rc, toks, (const __nv_bfloat16*)emb, gain,
               x, xs, ss);
}

}  // namespace llma
