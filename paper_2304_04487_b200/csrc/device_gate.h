// Turns of kernels whose CTAs wait for one another (library-private).
//
// A whole-step launch (step_simt.cu) and a projection that adds up partial tiles (gemm_tcgen05.cu, gemm_wide.cu) need all of their CTAs on
// the GPU before any of them can finish.  Side by side on two streams, one of each kind can stop the other, with some of the SMs
// each, until its waits run out: a whole-step engine beside a tensor-core engine did, within milliseconds of starting both.  So
// launches of the two kinds from different streams take turns: whoever launches has its stream wait for what calls under way on other streams
// have launched of the other kind.  (Projections of several streams go on side by side, as do kernels without such waits.)  Only
// engines of one device concern each other, and only where one takes whole steps.
//
// Whole-step launches of several streams share the SMs: each takes as many CTAs as there are SMs for every call under way that takes
// whole steps, down to a quarter (what a step gives does not depend on the number of CTAs), and waits for the oldest launches that hold
// more than that leaves.  Decodes per second of 1, 2, 4 and 8 decoders with a thread each, launches one by one -> all SMs in turns -> shares:
// fp32 width 256 425, 655, 1338, 1874 -> 721, 757, 757, 756 -> 719, 1267, 1948, 1510; bf16 width 512 453, 846, 1568, 2340 -> 573, 587, 586,
// 586 -> 575, 890, 1421, 1493; fp32 width 1024 332, 505, 721, 762 -> 441, 449, 449, 448 -> 444, 591, 736, 749.  Shares of an eighth:
// 1850 at four and 765 at eight of the first.
#pragma once
#include <cuda_runtime.h>

#include <mutex>

namespace llma {

enum : int { kTurnNone = -1, kTurnTiles = 0, kTurnSteps = 1 };  // what is launched: nothing that waits, one kind, the other

struct GateMember {  // an engine
    int device = -1;
    cudaStream_t stream = nullptr;
    bool steps = false;                            // takes whole steps
    cudaEvent_t ev[2] = {nullptr, nullptr};        // behind its last launches of each kind
    bool in_call = false, launched[2] = {false, false};  // a call is under way, and has launched kernels of the kind
    unsigned calls = 0;                                  // begun so far
    int ctas = 0;                                        // of its last whole-step launches, and their number among all
    unsigned long long turn = 0;
};

// (An engine that takes whole steps waits for the calls under way: they may have launched without taking turns.)
cudaError_t gate_join(GateMember* m, int device, cudaStream_t stream, bool steps);
void gate_quit(GateMember* m);
bool gate_shared(const GateMember& m);  // engines of the other kind may want turns: launch few steps at a time

// A call under way.  Calls wait for what they have launched before they return, so nobody waits for a member without one.
class GateCall {
public:
    explicit GateCall(GateMember& m);
    ~GateCall();
private:
    GateMember& m_;
};

// Held while kernels of a kind are launched; error() after construction and end().
class GateTurn {
public:
    GateTurn(GateMember& m, int kind, int num_sms);
    // a call that is no engine's (kTurnTiles): the turn lasts until its destruction, which the caller's wait for the stream precedes
    GateTurn(int device, cudaStream_t stream);
    cudaError_t error() const { return err_; }
    int ctas() const { return ctas_; }  // of a whole-step launch
    cudaError_t end();  // everything has been launched
private:
    void wait_for_others(const GateMember* self, cudaStream_t stream, int kind);
    void share_sms(int num_sms);
    std::unique_lock<std::mutex> lock_;
    GateMember* m_ = nullptr;
    int device_, kind_, ctas_ = 0;
    cudaError_t err_ = cudaSuccess;
};

}  // namespace llma
