// capture_graph (capture.cuh) against a fake of the CUDA calls it makes:
// argv[1] is the call that fails ("none", "stream", "begin", "end",
// "end_null", "instantiate"; "throw": the body).  Prints whether a graph came back, what
// the host's note holds afterwards (1 while the body has advanced it), the
// body's runs, the captures left open, the graphs and streams left, a pending
// error, and whether each capture was of a non-blocking stream made for it,
// which the body got.
#include "capture.cuh"

#include <cstdio>
#include <cstring>
#include <stdexcept>

static const char* fail = "none";
static int open_captures = 0, graphs = 0, streams = 0, error = 0, own = 1;
static cudaStream_t const made = (cudaStream_t)&streams;
static int hit(const char* what, cudaError_t e) { return std::strcmp(fail, what) ? 0 : (error = e); }

extern "C" {
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned flags) {
    if (hit("stream", cudaErrorMemoryAllocation)) return (cudaError_t)error;
    own &= flags == cudaStreamNonBlocking;
    streams++;
    *s = made;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    own &= s == made;
    streams--;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    own &= s == made;
    if (hit("begin", cudaErrorStreamCaptureUnsupported)) return (cudaError_t)error;
    open_captures++;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    open_captures--;
    *g = nullptr;
    if (hit("end", cudaErrorStreamCaptureInvalidated)) return (cudaError_t)error;
    if (!std::strcmp(fail, "end_null")) return cudaSuccess;
    graphs++;
    *g = (cudaGraph_t)&graphs;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
    if (hit("instantiate", cudaErrorMemoryAllocation)) return (cudaError_t)error;
    *x = (cudaGraphExec_t)&graphs;
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { graphs--; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { const int e = error; error = 0; return (cudaError_t)e; }
}

int main(int argc, char** argv) {
    if (argc > 1) fail = argv[1];
    int note = 0, runs = 0, thrown = 0;
    cudaGraphExec_t exec = nullptr;
    try {
        exec = orbc::capture_graph(
            [&](cudaStream_t s) {
                own &= s == made;
                runs++;
                note = 1;
                if (!std::strcmp(fail, "throw")) throw std::runtime_error("body");
            },
            [&] { note = 0; });
    } catch (const std::runtime_error&) {
        thrown = 1;
    }
    std::printf("graph %d note %d runs %d thrown %d open %d graphs %d streams %d error %d own %d\n", exec != nullptr, note, runs, thrown,
                open_captures, graphs, streams, error, own);
}
