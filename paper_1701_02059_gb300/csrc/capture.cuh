// Capture of a step's launches as a CUDA graph.
#pragma once
#include <cuda_runtime_api.h>

namespace orbc {

// What body(stream) launches as an executable graph.  The stream is one of the
// capture's own, on which nothing runs: a stream that a caller shares between
// handles or threads would take the others' work into the graph, and a
// blocking one would fail on any use of the legacy stream meanwhile.
// Nullptr when there is no graph (no stream, a call of the body ended the
// capture, no room): nothing has run, the error is cleared and the caller
// makes the launches themselves.  Capturing runs no kernel, so undo() takes
// back what body advanced on the host, whether or not there is a graph; an
// exception of body closes the capture and passes on.
template <typename Body, typename Undo>
cudaGraphExec_t capture_graph(Body&& body, Undo&& undo) {
    cudaStream_t s = nullptr;
    if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        cudaStreamDestroy(s);
        cudaGetLastError();
        return nullptr;
    }
    cudaGraph_t g = nullptr;
    cudaGraphExec_t exec = nullptr;
    auto close = [&](bool instantiate) {
        bool ok = cudaStreamEndCapture(s, &g) == cudaSuccess && g;
        if (ok && instantiate) ok = cudaGraphInstantiate(&exec, g, 0) == cudaSuccess;
        if (g) cudaGraphDestroy(g);
        cudaStreamDestroy(s);
        if (!ok) {
            cudaGetLastError();
            exec = nullptr;
        }
        undo();
    };
    try {
        body(s);
    } catch (...) {
        close(false);
        throw;
    }
    close(true);
    return exec;
}

}  // namespace orbc
