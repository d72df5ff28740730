#include "call_order.h"

#include <new>

namespace msf {

CallTurn::CallTurn(CallOrder& order, cudaStream_t st) : o_(order), lock_(order.mu), st_(st) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    error_ = cudaStreamGetCaptureInfo(st, &cs, &capture_);
    if (error_ != cudaSuccess) return;
    capturing_ = cs == cudaStreamCaptureStatusActive;
    if (capturing_) {
        if (o_.captured && o_.capture == capture_ && o_.captured_stream != st)
            error_ = cudaStreamWaitEvent(st, o_.captured, 0);
        return;
    }
    error_ = cudaStreamGetId(st, &id_);
    if (error_ == cudaSuccess && o_.recorded && o_.stream != id_) error_ = cudaStreamWaitEvent(st, o_.done, 0);
}

cudaError_t CallTurn::end() {
    if (!open_) return cudaSuccess;
    open_ = false;
    cudaError_t e = cudaSuccess;
    if (capturing_) {
        if (!o_.captured) e = cudaEventCreateWithFlags(&o_.captured, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventRecord(o_.captured, st_);
        o_.capture = e == cudaSuccess ? capture_ : 0;
        o_.captured_stream = st_;
        return e;
    }
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess && (!o_.done || o_.device != dev)) {
        if (o_.done) cudaEventDestroy(o_.done);
        o_.done = nullptr;
        o_.recorded = false;
        e = cudaEventCreateWithFlags(&o_.done, cudaEventDisableTiming);
        o_.device = dev;
    }
    if (e == cudaSuccess) e = cudaEventRecord(o_.done, st_);
    o_.recorded = e == cudaSuccess;
    o_.stream = id_;
    return e;
}

CallTurn::~CallTurn() {
    if (error_ == cudaSuccess) end();
}

CallOrder* call_order_new() { return new (std::nothrow) CallOrder; }

void call_order_free(CallOrder* o) {
    if (!o) return;
    if (o->done) cudaEventDestroy(o->done);
    if (o->captured) cudaEventDestroy(o->captured);
    delete o;
}

}  // namespace msf
