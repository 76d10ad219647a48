// Stand-alone entry points for the weight-streaming GEMM.
//
// The product itself takes 5 to 40 us, so what surrounds it decides what a call costs: device properties and kernel
// attributes are looked up once per device, the kernel reads the caller's bf16 rows in place (one term, no split
// copy), and the scratch of llma_gemm_rows32_bf16 is borrowed from a small pool whose blocks keep the state that the
// kernel leaves them in (hand-over slots empty).  With cudaMalloc, cudaFree and five memory operations per call
// 4096 x 4096 took 4.9 ms alone and 15 ms in a row of calls.
#include <cstring>
#include <mutex>
#include <vector>

#include "engine.h"

using namespace llma;

namespace {

constexpr int kMaxDevices = 64;
// Blocks of 2.3 MB that a device keeps between calls.  One is in use per concurrent call, and a call without one pays a cudaMalloc
// and a cudaFree (milliseconds, and the device stops for them), so there are as many as callers a program may reasonably have
// at once; 39 MB is the most that this can hold.
constexpr size_t kMaxIdle = 16;

// One call's scratch.  Between calls: every hand-over word all-ones, *err zero.
struct Block {
    float* ws = nullptr;     // device: gemm_ws_bytes(sms)
    int32_t* err = nullptr;  // page-locked host word that the kernel writes when a wait runs out
};

struct Device {
    std::mutex mu;
    bool ready = false;
    int sms = 0;
    std::vector<Block> idle;
    int engines = 0;  // alive on this device
};
Device g_dev[kMaxDevices];

void free_block(const Block& b) {
    cudaFree(b.ws);
    if (b.err) cudaFreeHost(b.err);
}

cudaError_t new_block(int sms, Block* b) {
    cudaError_t e = cudaMalloc((void**)&b->ws, gemm_ws_bytes(sms));
    if (e == cudaSuccess) e = cudaHostAlloc((void**)&b->err, sizeof(int32_t), cudaHostAllocMapped | cudaHostAllocPortable);
    if (e == cudaSuccess) { *b->err = 0; e = cudaMemset(b->ws, 0xFF, gemm_ws_bytes(sms)); }
    if (e == cudaSuccess) e = cudaStreamSynchronize(0);  // the caller's stream need not wait for the default stream
    if (e != cudaSuccess) { free_block(*b); *b = Block(); }
    return e;
}

}  // namespace

namespace llma {

// Device facts and kernel attributes, looked up once per device.
int gemm_device(int* dev_out, int* sms) {
    int dev = 0;
    CU_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return LLMA_ERR_CONFIG;
    Device& d = g_dev[dev];
    std::lock_guard<std::mutex> lock(d.mu);
    if (!d.ready) {
        int major = 0, count = 0;
        CU_TRY(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
        CU_TRY(cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev));
        if (major != 10) return LLMA_ERR_CONFIG;
        CU_TRY(init_gemm_tcgen05());
        d.sms = count;
        d.ready = true;
    }
    *dev_out = dev;
    *sms = d.sms;
    return LLMA_OK;
}

// TMA descriptor and one launch; `a` is the caller's [32][k_in].  A W off the 16-byte grid has no descriptor.
int gemm_rows32_launch(const void* W, const void* a, float* out, int32_t n_out, int32_t k_in, float* ws,
                       int32_t* dev_err, int grid, cudaStream_t st) {
    CUtensorMap ma;
    if (reinterpret_cast<uintptr_t>(a) % sizeof(__nv_bfloat16) || reinterpret_cast<uintptr_t>(out) % sizeof(float)) return LLMA_ERR_ARG;
    if (make_tensor_map_bf16_chunks(&ma, W, (uint64_t)n_out, (uint64_t)k_in, 128) != 0) return LLMA_ERR_ARG;
    GemmArgs g;
    std::memset(&g, 0, sizeof(g));
    g.mode = kGemmStore; g.n_out = n_out; g.n_tiles = (n_out + 127) / 128; g.chunks = k_in / 64;
    g.tiles_per_map = g.n_tiles; g.rows = nullptr; g.ws = ws; g.dev_err = dev_err;
    g.out_f32 = out; g.ld = n_out; g.act = a;
    g.rc = 32; g.nr = 32;
    launch_gemm_tcgen05(st, grid, false, g, ma, ma, ma);
    CU_TRY(cudaGetLastError());
    return LLMA_OK;
}

// An engine has come (+1) or gone (-1).  With a device's last engine its idle scratch goes too (a later call allocates again).
void gemm_count_engine(int dev, int by) {
    if (dev < 0 || dev >= kMaxDevices) return;
    std::vector<Block> idle;
    {
        std::lock_guard<std::mutex> lock(g_dev[dev].mu);
        g_dev[dev].engines += by;
        if (by < 0 && g_dev[dev].engines == 0) idle.swap(g_dev[dev].idle);
    }
    if (idle.empty()) return;
    int current = 0;
    cudaGetDevice(&current);
    cudaSetDevice(dev);
    for (const Block& b : idle) free_block(b);
    cudaSetDevice(current);
}

}  // namespace llma

extern "C" int llma_gemm_rows32_bf16(const void* W, const void* a, float* out, int32_t n_out, int32_t k_in,
                                     void* cuda_stream) {
    if (!W || !a || !out) return LLMA_ERR_NULL;
    if (n_out < 1 || k_in < 64 || k_in % 64) return LLMA_ERR_ARG;
    int dev = 0, sms = 0;
    int rc = gemm_device(&dev, &sms);
    if (rc) return rc;
    Device& d = g_dev[dev];
    Block b;
    {
        std::lock_guard<std::mutex> lock(d.mu);
        if (!d.idle.empty()) { b = d.idle.back(); d.idle.pop_back(); }
    }
    if (!b.ws) CU_TRY(new_block(sms, &b));
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int grid = gemm_grid_for((int64_t)((n_out + 127) / 128) * (k_in / 64), sms);
    // the kernel reaches the page-locked word through its device address
    int32_t* err_dev = nullptr;
    GateTurn turn(dev, st);  // until the wait below is over
    cudaError_t ce = turn.error();
    if (ce == cudaSuccess) ce = cudaHostGetDevicePointer((void**)&err_dev, b.err, 0);
    if (ce == cudaSuccess) rc = gemm_rows32_launch(W, a, out, n_out, k_in, b.ws, err_dev, grid, st);
    if (ce == cudaSuccess && rc == LLMA_OK) ce = cudaStreamSynchronize(st);  // synchronous: the block is free again after this
    const bool clean = ce == cudaSuccess && (rc == LLMA_OK || rc == LLMA_ERR_ARG) && *(volatile int32_t*)b.err == kDevErrNone;
    if (ce == cudaSuccess && rc == LLMA_OK && !clean) rc = LLMA_ERR_DEVICE_TIMEOUT;
    turn.end();
    {
        std::lock_guard<std::mutex> lock(d.mu);
        if (clean && d.idle.size() < kMaxIdle) { d.idle.push_back(b); b = Block(); }
    }
    if (b.ws) free_block(b);  // one too many, or left in an unknown state
    if (ce != cudaSuccess) { llma::note_cuda_error(ce); return LLMA_ERR_CUDA; }
    return rc;
}
