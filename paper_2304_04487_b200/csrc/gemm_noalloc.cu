// llma_gemm_rows32_bf16_noalloc: the stand-alone projection GEMM for callers that must not
// allocate.  Its partial tiles (handed between CTAs) live in one file-scope __device__ array instead of cudaMalloc'ed memory.
#include <mutex>

#include "engine.h"

using namespace llma;

namespace llma {
int gemm_device(int* dev_out, int* sms);
int gemm_rows32_launch(const void* W, const void* a, float* out, int32_t n_out, int32_t k_in, float* ws,
                       int32_t* dev_err, int grid, cudaStream_t st);
}

namespace {

constexpr int kMaxGrid = 160;        // CTAs whose partial tiles fit (a B200 has 148 SMs)
constexpr int kMaxTiles = 2048;      // n_out <= 262144
constexpr int kMaxK = 16384;
constexpr size_t kWsBytes = gemm_ws_bytes(kMaxGrid);  // 2,621,440

// Every GPU that loads this library holds this array until the process exits.  In host code the name below is only a
// handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kWsBytes];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
struct Scratch {
    float* ws = nullptr;   // device address of the array
    bool clean = false;    // every hand-over word is empty: the calls before have ended well, one at a time
    int calls = 0;         // under way now
    bool mixed = false;    // ... more than one at some time: what they leave is anyone's guess
};
Scratch g_scratch[kMaxDevices];
// Error words, one per device, that the kernel writes when a wait runs out: host memory of the library's own, pinned by the first
// call, so that a call reads them without a copy.  A page to themselves, since pages are what is pinned.
alignas(4096) int32_t g_err[4096 / sizeof(int32_t)];
int32_t* g_err_dev = nullptr;  // ... as the devices see them

}  // namespace

extern "C" int llma_gemm_rows32_bf16_noalloc(const void* W, const void* a, float* out, int32_t n_out, int32_t k_in,
                                             void* cuda_stream) {
    if (!W || !a || !out) return LLMA_ERR_NULL;
    if (n_out < 1 || k_in < 64 || k_in % 64) return LLMA_ERR_ARG;
    const int n_tiles = (n_out + 127) / 128;
    if (n_tiles > kMaxTiles || k_in > kMaxK) return LLMA_ERR_CAPACITY;
    int dev = 0, sms = 0;
    int rc = gemm_device(&dev, &sms);
    if (rc) return rc;
    Scratch& sc = g_scratch[dev];
    float* ws = nullptr;
    int32_t* err_dev = nullptr;
    bool clean = false;
    {
        // set-up, with the device current: the array's address and the pinned words
        std::lock_guard<std::mutex> lock(g_mu);
        if (!sc.ws) {
            void* p = nullptr;
            CU_TRY(cudaGetSymbolAddress(&p, g_noalloc_scratch));
            if (!g_err_dev) {
                void* q = nullptr;
                CU_TRY(cudaHostRegister(g_err, sizeof(g_err), cudaHostRegisterPortable | cudaHostRegisterMapped));
                CU_TRY(cudaHostGetDevicePointer(&q, g_err, 0));
                g_err_dev = static_cast<int32_t*>(q);
            }
            sc.ws = static_cast<float*>(p);
        }
        ws = sc.ws;
        err_dev = g_err_dev + dev;
        clean = sc.clean && sc.calls == 0;
        sc.mixed = sc.mixed || sc.calls > 0;
        sc.calls += 1;
        sc.clean = false;
    }
    struct Leave {  // the call is over, by whichever return
        Scratch& sc;
        bool well = false;
        ~Leave() {
            std::lock_guard<std::mutex> lock(g_mu);
            if (--sc.calls > 0) return;
            sc.clean = well && !sc.mixed;
            sc.mixed = false;
        }
    } leave{sc};
    cudaStream_t st = (cudaStream_t)cuda_stream;
    GateTurn turn(dev, st);  // until the call returns
    CU_TRY(turn.error());
    int grid = gemm_grid_for((int64_t)n_tiles * (k_in / 64), sms);
    if (grid > kMaxGrid) grid = kMaxGrid;
    // A call leaves the hand-over slots empty (all-ones words), as it needs them.  After one that did not end well, and for the first, all of them
    // are emptied: 2.6 MB, which with the error word copied back was a quarter of a call (22016 x 4096: 61.5 -> 49.0 us).
    volatile int32_t* err = g_err + dev;
    if (!clean) CU_TRY(cudaMemsetAsync(ws, 0xFF, kWsBytes, st));
    *err = kDevErrNone;
    rc = gemm_rows32_launch(W, a, out, n_out, k_in, ws, err_dev, grid, st);
    if (rc && rc != LLMA_ERR_ARG) return rc;
    CU_TRY(cudaStreamSynchronize(st));
    if (rc == LLMA_OK && *err != kDevErrNone) return LLMA_ERR_DEVICE_TIMEOUT;
    leave.well = true;
    return rc;
}
