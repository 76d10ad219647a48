// Turns of kernels whose CTAs wait for one another: see device_gate.h.
#include "device_gate.h"

#include <algorithm>
#include <condition_variable>
#include <utility>
#include <vector>

namespace llma {

namespace {
constexpr int kMaxDevices = 64;
constexpr int kMostShares = 4;  // launches of whole steps side by side
struct Gate {
    std::mutex mu;
    std::vector<GateMember*> members;
    std::condition_variable over;  // a call is
    int steppers = 0;              // members that take whole steps
    unsigned long long turns = 0;  // of whole-step launches so far
};
Gate g_gates[kMaxDevices];
bool known(int device) { return device >= 0 && device < kMaxDevices; }
}  // namespace

cudaError_t gate_join(GateMember* m, int device, cudaStream_t stream, bool steps) {
    if (!known(device)) return cudaErrorInvalidDevice;
    for (cudaEvent_t& ev : m->ev) {
        const cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (e != cudaSuccess) return e;
    }
    m->device = device; m->stream = stream; m->steps = steps;
    Gate& g = g_gates[device];
    std::unique_lock<std::mutex> lock(g.mu);
    std::vector<std::pair<GateMember*, unsigned>> before;
    for (GateMember* o : g.members)
        if (o->in_call) before.push_back({o, o->calls});
    g.members.push_back(m);
    if (!steps) return cudaSuccess;
    ++g.steppers;
    g.over.wait(lock, [&] {
        return std::none_of(before.begin(), before.end(), [&](const std::pair<GateMember*, unsigned>& b) {
            return std::find(g.members.begin(), g.members.end(), b.first) != g.members.end() && b.first->in_call && b.first->calls == b.second;
        });
    });
    return cudaSuccess;
}

void gate_quit(GateMember* m) {
    if (known(m->device)) {
        Gate& g = g_gates[m->device];
        std::lock_guard<std::mutex> lock(g.mu);
        g.members.erase(std::remove(g.members.begin(), g.members.end(), m), g.members.end());
        g.steppers -= m->steps ? 1 : 0;
    }
    m->device = -1;
    for (cudaEvent_t& ev : m->ev) {
        if (ev) cudaEventDestroy(ev);
        ev = nullptr;
    }
}

bool gate_shared(const GateMember& m) {
    Gate& g = g_gates[m.device];
    std::lock_guard<std::mutex> lock(g.mu);
    return m.steps ? (int)g.members.size() > g.steppers : g.steppers > 0;
}

GateCall::GateCall(GateMember& m) : m_(m) {
    std::lock_guard<std::mutex> lock(g_gates[m_.device].mu);
    m_.in_call = true;
    ++m_.calls;
    m_.launched[0] = m_.launched[1] = false;
}
GateCall::~GateCall() {
    std::lock_guard<std::mutex> lock(g_gates[m_.device].mu);
    m_.in_call = false;
    g_gates[m_.device].over.notify_all();
}

void GateTurn::wait_for_others(const GateMember* self, cudaStream_t stream, int kind) {
    for (const GateMember* o : g_gates[device_].members) {
        if (err_ != cudaSuccess) return;
        if (o != self && o->stream != stream && o->in_call && o->launched[1 - kind]) err_ = cudaStreamWaitEvent(stream, o->ev[1 - kind], 0);
    }
}

// The launches of other calls, newest first: those that this one does not fit beside have to be over before it begins.
void GateTurn::share_sms(int num_sms) {
    std::vector<const GateMember*> others;
    int callers = 1;
    for (const GateMember* o : g_gates[device_].members) {
        if (o == m_ || o->stream == m_->stream || !o->in_call || !o->steps) continue;
        ++callers;
        if (o->launched[kTurnSteps]) others.push_back(o);
    }
    std::sort(others.begin(), others.end(), [](const GateMember* x, const GateMember* y) { return x->turn > y->turn; });
    ctas_ = std::max(num_sms / callers, num_sms / kMostShares);
    int room = num_sms - ctas_;
    for (const GateMember* o : others) {
        room -= o->ctas;
        if (room < 0 && err_ == cudaSuccess) err_ = cudaStreamWaitEvent(m_->stream, o->ev[kTurnSteps], 0);
    }
}

GateTurn::GateTurn(GateMember& m, int kind, int num_sms) : m_(&m), device_(m.device), kind_(kind), ctas_(num_sms) {
    if (kind == kTurnNone) return;
    std::unique_lock<std::mutex> lock(g_gates[device_].mu);
    if (g_gates[device_].steppers == 0) return;  // (an engine that changes this waits for the call to end)
    lock_ = std::move(lock);
    wait_for_others(m_, m.stream, kind);
    if (kind == kTurnSteps) share_sms(num_sms);
}
GateTurn::GateTurn(int device, cudaStream_t stream) : device_(device), kind_(kTurnTiles) {
    if (!known(device)) return;
    std::unique_lock<std::mutex> lock(g_gates[device].mu);
    if (g_gates[device].steppers == 0) return;
    lock_ = std::move(lock);
    wait_for_others(nullptr, stream, kTurnTiles);
}

cudaError_t GateTurn::end() {
    if (!lock_.owns_lock()) return err_;
    if (m_) {
        if (g_gates[device_].members.size() > 1) {
            const cudaError_t e = cudaEventRecord(m_->ev[kind_], m_->stream);
            if (err_ == cudaSuccess) err_ = e;
        }
        m_->launched[kind_] = true;
        if (kind_ == kTurnSteps) {
            m_->ctas = ctas_;
            m_->turn = ++g_gates[device_].turns;
        }
    }
    lock_.unlock();
    return err_;
}

}  // namespace llma
