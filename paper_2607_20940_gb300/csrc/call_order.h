// One call after the other on a workspace that several streams or threads use.
#pragma once

#include <cuda_runtime.h>

#include <mutex>

namespace msf {

// The last call that wrote scratch of a plan's workspace. fp32 attention and its
// gradient keep their operands' planes there, and a caller may have several such
// calls of one plan in flight on different streams (each with tensors of its
// own): every call waits on the device for the one before it. An event is
// recorded after each call, since the stream of an earlier call may be gone by
// the time a later one wants to wait for it; calls of one stream need no wait.
// Under capture the same holds among the calls of one capture; a graph's replay
// is ordered with other work by the caller.
struct CallOrder {
    std::mutex mu;
    cudaEvent_t done = nullptr;  // after the last call
    int device = -1;             // of `done`
    bool recorded = false;
    unsigned long long stream = 0;  // id of the last call's stream
    cudaEvent_t captured = nullptr;  // after the last call of capture `capture`
    unsigned long long capture = 0;
    cudaStream_t captured_stream = nullptr;  // (an id cannot be asked for under capture)
};

// The order's mutex, and the wait; the destructor records.
class CallTurn {
public:
    CallTurn(CallOrder& order, cudaStream_t st);
    ~CallTurn();
    cudaError_t error() const { return error_; }
    // After the call's launches (the destructor does it otherwise).
    cudaError_t end();

private:
    CallOrder& o_;
    std::lock_guard<std::mutex> lock_;
    cudaStream_t st_;
    bool capturing_ = false, open_ = true;
    unsigned long long id_ = 0, capture_ = 0;
    cudaError_t error_ = cudaSuccess;
};

CallOrder* call_order_new();
void call_order_free(CallOrder* o);

}  // namespace msf
