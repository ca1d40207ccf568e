// Capture of a step's launches as a CUDA graph.
#pragma once
#include <cuda_runtime_api.h>

namespace orbc {

// What body() launches on `stream` as an executable graph.  Nullptr when there
// is none (the stream cannot be captured, a call of the body ended the
// capture, no room for the graph): nothing has run, the error is cleared and
// the caller makes the launches themselves.  Capturing runs no kernel, so
// undo() takes back what body advanced on the host, whether or not there is a
// graph; an exception of body closes the capture and passes on.
template <typename Body, typename Undo>
cudaGraphExec_t capture_graph(cudaStream_t stream, Body&& body, Undo&& undo) {
    if (cudaStreamBeginCapture(stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    cudaGraph_t g = nullptr;
    try {
        body();
    } catch (...) {
        cudaStreamEndCapture(stream, &g);
        if (g) cudaGraphDestroy(g);
        cudaGetLastError();
        undo();
        throw;
    }
    cudaGraphExec_t exec = nullptr;
    const bool ok = cudaStreamEndCapture(stream, &g) == cudaSuccess && g && cudaGraphInstantiate(&exec, g, 0) == cudaSuccess;
    if (g) cudaGraphDestroy(g);
    undo();
    if (ok) return exec;
    cudaGetLastError();
    return nullptr;
}

}  // namespace orbc
