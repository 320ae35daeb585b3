// dirotq_linear_host: the layer on host buffers, row chunks pipelined over two copy streams.
#include "common.h"
#include "host_chunks.h"

#include <mutex>

namespace dirotq {
namespace {

// Copy streams and events of dirotq_linear_host, created once per device (no device memory involved).
struct HostPipe {
    bool ready = false;
    cudaStream_t h2d = nullptr, d2h = nullptr;
    cudaEvent_t start = nullptr, done = nullptr, copied[kMaxHostChunks] = {}, computed[kMaxHostChunks] = {};
};
std::mutex g_pipe_mutex;
HostPipe g_pipe[64];

// Caller holds g_pipe_mutex (also while it enqueues on the pipe: its events are shared by all calls on the device).
dirotq_status_t host_pipe(int dev, HostPipe** out) {
    if (dev < 0 || dev >= 64) return DIROTQ_ERR_INVALID_ARG;
    HostPipe& p = g_pipe[dev];
    if (!p.ready) {
        cudaError_t e = cudaStreamCreateWithFlags(&p.h2d, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p.d2h, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p.start, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p.done, cudaEventDisableTiming);
        for (int i = 0; i < kMaxHostChunks && e == cudaSuccess; ++i) {
            e = cudaEventCreateWithFlags(&p.copied[i], cudaEventDisableTiming);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p.computed[i], cudaEventDisableTiming);
        }
        if (e != cudaSuccess) { set_error("host pipeline set-up", e); return DIROTQ_ERR_CUDA; }
        p.ready = true;
    }
    *out = &p;
    return DIROTQ_OK;
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
    if (M < kMinPipelinedRows) {
        cudaError_t e = cudaMemcpyAsync(x_dev, x_host, xrow * M, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) { set_error("cudaMemcpyAsync(H2D)", e); return DIROTQ_ERR_CUDA; }
        st = dirotq_linear(x_dev, M, layer, y_dev, workspace, workspace_bytes, stream);
        if (st != DIROTQ_OK) return st;
        e = cudaMemcpyAsync(y_host, y_dev, yrow * M, cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) { set_error("cudaMemcpyAsync(D2H)", e); return DIROTQ_ERR_CUDA; }
        return DIROTQ_OK;
    }
    std::lock_guard<std::mutex> lock(g_pipe_mutex);
    HostPipe* p = nullptr;
    st = host_pipe(layer->device, &p);
    if (st != DIROTQ_OK) return st;
    int rows[kMaxHostChunks];
    const int n = plan_host_chunks(M, xrow, yrow, rows);
    PipeOps ops = {*p, s, layer, static_cast<const char*>(x_host), static_cast<char*>(y_host), static_cast<char*>(x_dev), static_cast<char*>(y_dev),
                   xrow, yrow, workspace, workspace_bytes};
    return run_host_chunks(rows, n, ops) ? DIROTQ_OK : ops.st;
}
