// dirotq_linear_host: the layer on host buffers, row chunks pipelined over two copy streams.
#include "common.h"
#include "host_chunks.h"

#include <mutex>

namespace dirotq {
namespace {

// Copy streams and events, created when first needed and kept for the device (no device memory involved).
struct HostPipe {
    std::mutex mutex;  // held while a call is enqueued: its calls share the events
    bool ready = false;
    unsigned long long user = 0;  // id of the caller's stream of the last call
    cudaStream_t h2d = nullptr, d2h = nullptr;
    cudaEvent_t start = nullptr, done = nullptr, copied[kMaxHostChunks] = {}, computed[kMaxHostChunks] = {};
};
// Two pipes per device.  Long calls share one, in the order they are made: their copies fill the link in either direction, and more
// copy streams would have to share the device's eight queues with the callers' own (the four FLUX layers on four streams: 5.5 ms
// with one pipe, 5.5 to 6.4 with four).  Short calls wait for nobody: one takes the other pipe if no call of another stream is
// under way on it, and otherwise stays on its own stream, in one piece.
constexpr int kLongCallRows = 2048;
struct DevicePipes {
    HostPipe long_calls, short_calls;
} g_device[64];

// Looking at an event and making streams and events must not disturb a capture that some other thread has under way.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

bool create(HostPipe& p) {
    auto event = [](cudaEvent_t& e) { return e != nullptr || cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess; };
    auto streams = [](cudaStream_t& s) { return s != nullptr || cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess; };
    bool ok = streams(p.h2d) && streams(p.d2h) && event(p.start) && event(p.done);
    for (int i = 0; i < kMaxHostChunks && ok; ++i) ok = event(p.copied[i]) && event(p.computed[i]);
    return p.ready = ok;  // (what a failed attempt has made is there for the next one)
}

// Locks the pipe that a call of M rows on `stream` runs on; an empty lock: the call stays in one piece on its own stream.
HostPipe* take_pipe(int device, int M, cudaStream_t stream, std::unique_lock<std::mutex>& lock) {
    if (M < kMinPipelinedRows || device < 0 || device >= 64) return nullptr;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    // (a call that is being captured: the copy streams would be part of the capture until it ends)
    if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone || cudaStreamGetId(stream, &id) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    RelaxedCapture relaxed;
    const bool shares = M >= kLongCallRows;
    HostPipe& p = shares ? g_device[device].long_calls : g_device[device].short_calls;
    lock = shares ? std::unique_lock<std::mutex>(p.mutex) : std::unique_lock<std::mutex>(p.mutex, std::try_to_lock);
    bool ok = lock.owns_lock() && (p.ready || create(p));
    if (ok && !shares && p.user != id) ok = cudaEventQuery(p.done) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();  // neither a call still under way nor a missing pipe is an error of this call
        if (lock.owns_lock()) lock.unlock();
        return nullptr;
    }
    p.user = id;
    return &p;
}

// The steps of run_host_chunks on a pipe.  The chunks' kernels run one after another on `stream`, so they share the workspace.
struct PipeOps {
    HostPipe& p;
    cudaStream_t stream;
    const dirotq_layer_t* layer;
    const char* x_host;
    char *y_host, *x_dev, *y_dev;
    size_t xrow, yrow;
    void* workspace;
    size_t workspace_bytes;
    dirotq_status_t st = DIROTQ_OK;

    bool cuda(cudaError_t e) {
        if (e == cudaSuccess) return true;
        set_error("host pipeline", e);
        st = DIROTQ_ERR_CUDA;
        return false;
    }
    bool fork() {  // the staging buffers may still be in use by earlier work on `stream`
        return cuda(cudaEventRecord(p.start, stream)) && cuda(cudaStreamWaitEvent(p.h2d, p.start, 0)) && cuda(cudaStreamWaitEvent(p.d2h, p.start, 0));
    }
    bool copy_in(int c, int m0, int rows) {
        return cuda(cudaMemcpyAsync(x_dev + xrow * m0, x_host + xrow * m0, xrow * rows, cudaMemcpyHostToDevice, p.h2d)) &&
               cuda(cudaEventRecord(p.copied[c], p.h2d)) && cuda(cudaStreamWaitEvent(stream, p.copied[c], 0));
    }
    bool compute(int c, int m0, int rows) {
        st = dirotq_linear(x_dev + xrow * m0, rows, layer, y_dev + yrow * m0, workspace, workspace_bytes, stream);
        return st == DIROTQ_OK && cuda(cudaEventRecord(p.computed[c], stream)) && cuda(cudaStreamWaitEvent(p.d2h, p.computed[c], 0));
    }
    bool copy_out(int, int m0, int rows) {
        return cuda(cudaMemcpyAsync(y_host + yrow * m0, y_dev + yrow * m0, yrow * rows, cudaMemcpyDeviceToHost, p.d2h));
    }
    // later work on `stream` (and its synchronisation) comes after every copy: out of y_dev, and, where a step failed, into x_dev too
    bool join(bool ok) {
        if (ok) return cuda(cudaEventRecord(p.done, p.d2h)) && cuda(cudaStreamWaitEvent(stream, p.done, 0));
        for (const cudaStream_t copies : {p.h2d, p.d2h})
            if (cudaEventRecord(p.done, copies) != cudaSuccess || cudaStreamWaitEvent(stream, p.done, 0) != cudaSuccess) cudaStreamSynchronize(copies);
        return true;  // (the first failure is the one reported)
    }
};

}  // namespace
}  // namespace dirotq

using namespace dirotq;

extern "C" dirotq_status_t dirotq_linear_host(const void* x_host, int M, const dirotq_layer_t* layer, void* y_host, void* x_dev,
                                              void* y_dev, void* workspace, size_t workspace_bytes, dirotq_stream_t stream) {
    dirotq_status_t st = check_call(layer, M, workspace, workspace_bytes);
    if (st != DIROTQ_OK) return st;
    if (!x_host || !y_host || !x_dev || !y_dev) return DIROTQ_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t xrow = static_cast<size_t>(layer->geo.K) * 2, yrow = static_cast<size_t>(layer->geo.N) * 2;
    // Token rows are independent: the call is cut into row chunks whose host-to-device copy, computation and
    // device-to-host copy overlap (copy engines in both directions + SMs).
    std::unique_lock<std::mutex> lock;
    HostPipe* p = take_pipe(layer->device, M, s, lock);
    if (!p) {
        cudaError_t e = cudaMemcpyAsync(x_dev, x_host, xrow * M, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) { set_error("cudaMemcpyAsync(H2D)", e); return DIROTQ_ERR_CUDA; }
        st = dirotq_linear(x_dev, M, layer, y_dev, workspace, workspace_bytes, stream);
        if (st != DIROTQ_OK) return st;
        e = cudaMemcpyAsync(y_host, y_dev, yrow * M, cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) { set_error("cudaMemcpyAsync(D2H)", e); return DIROTQ_ERR_CUDA; }
        return DIROTQ_OK;
    }
    int rows[kMaxHostChunks];
    const int n = plan_host_chunks(M, xrow, yrow, rows);
    PipeOps ops = {*p, s, layer, static_cast<const char*>(x_host), static_cast<char*>(y_host), static_cast<char*>(x_dev), static_cast<char*>(y_dev),
                   xrow, yrow, workspace, workspace_bytes};
    return run_host_chunks(rows, n, ops) ? DIROTQ_OK : ops.st;
}
