// lbm_step_graphs.h -- steps replayed from graphs: when a graph is
// made, which steps of a call replay it, and what follows a failure.  Host code
// of the CUDA runtime only.
#pragma once

#include <cuda_runtime_api.h>

#include <cstring>

namespace lbm {

// Steps of one graph (even, so that a replay leaves buf[cur] current).
// On this GPU a kernel that follows another in a stream starts 2.4 us later
// than the same kernel as the next node of a graph (chains of small dependent
// kernels: 4.1 us each in a stream, 1.8 us in a graph; at 1 M nodes 24.7 and
// 22.3 us), so steps are replayed 16 at a time and the rest of a call 4 at a time.
// More steps per graph gain nothing (the stream's gap between two graphs is
// 0.15 us a step at 16) and make the graph, paid once per context and launch
// shape, longer to build.
constexpr long STEP_GRAPH[2] = {16, 4};
// A graph is made once the steps it could have replayed, those of the present
// call among them, reach these counts: making it costs what it
// saves over about as many steps (16 steps of one launch: 60 us against 2.3 us a
// step; Shan-Chen, two launches: 90 against 4.4; a batch, with up to 32 KB of
// parameters a launch: 185 against 5.8).  A context that is stepped little then
// pays for plain launches alone.  Made at once, the first 16 steps of a fresh
// context took 109 us instead of 88 (256^2 fluid), 169 instead of 153 (32^3
// Shan-Chen), 321 instead of 258 (four 32^3 Shan-Chen domains), and calls of 31
// steps of that batch 470 instead of 440.
constexpr long STEP_GRAPH_AFTER[2] = {32, 16};

struct StepGraphs {
    cudaGraphExec_t exec[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};  // [STEP_GRAPH size][buf current]
    long missed[2][2] = {{0, 0}, {0, 0}};  // steps that the graph could have replayed
    int shape[6] = {-1, -1, -1, -1, -1, -1};  // launch shape of the graphs
    bool failed = false;  // of this shape's graphs one could not be made or launched: steps are launched one by one

    bool any() const { return exec[0][0] || exec[0][1] || exec[1][0] || exec[1][1]; }

    // `wait`: the stream whose replays may still be running, or null if idle.
    void drop(const cudaStream_t* wait) {
        if (any() && wait) cudaStreamSynchronize(*wait);
        for (int size = 0; size < 2; ++size)
            for (int k = 0; k < 2; ++k) {
                if (exec[size][k]) cudaGraphExecDestroy(exec[size][k]);
                exec[size][k] = nullptr;
                missed[size][k] = 0;
            }
        failed = false;
    }
};

// A graph being made of the kernels that launch_step would launch, a chain.  It
// is built node by node and not by capturing a stream: while any stream of the
// context is captured CUDA refuses device-wide synchronisations, those of the
// program's other threads too.
struct GraphRecord {
    cudaGraph_t graph = nullptr;
    cudaGraphNode_t last = nullptr;
};

// The graph of what `launch()` launches through launch_step while `record`
// points to it; nullptr if it cannot be made.
template <class Launch>
cudaGraphExec_t record_graph(GraphRecord*& record, Launch launch) {
    // relaxed: not disturbed by a capture on another thread
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    cudaGraphExec_t exec = nullptr;
    GraphRecord r;
    cudaError_t e = cudaGraphCreate(&r.graph, 0);
    if (e == cudaSuccess) {
        record = &r;
        e = launch();
        record = nullptr;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, r.graph, 0);
    if (r.graph) cudaGraphDestroy(r.graph);
    if (e != cudaSuccess) {
        cudaGetLastError();
        exec = nullptr;
    }
    cudaThreadExchangeStreamCaptureMode(&mode);
    return exec;
}

// n steps on `stream`: whole graphs, then single launches.  `launch(n)` enqueues
// n steps on `stream`, or adds them to the graph at `record`, and flips `cur` once
// per step.  While the caller is capturing the stream every step is a plain
// launch, which the capture records.
template <class Launch>
cudaError_t run_steps(StepGraphs& g, const int (&shape)[6], cudaStream_t stream, GraphRecord*& record, int& cur,
                      long n, Launch launch) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    bool replay = n >= STEP_GRAPH[1];
    if (replay && (cudaStreamIsCapturing(stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone)) {
        cudaGetLastError();
        replay = false;
    }
    if (replay && std::memcmp(shape, g.shape, sizeof(shape)) != 0) {
        g.drop(&stream);
        std::memcpy(g.shape, shape, sizeof(shape));
    }
    for (int size = 0; size < 2 && replay && !g.failed; ++size) {
        const int k = cur;
        const long steps = (size == 0 ? n : n % STEP_GRAPH[0]) / STEP_GRAPH[size] * STEP_GRAPH[size];
        cudaGraphExec_t& exec = g.exec[size][k];
        if (!exec && steps > 0) {
            g.missed[size][k] += steps;
            if (g.missed[size][k] < STEP_GRAPH_AFTER[size]) continue;
            exec = record_graph(record, [&] { return launch(STEP_GRAPH[size]); });
            cur = k;
            g.failed = !exec;
        }
        for (long s = 0; s < steps && !g.failed; s += STEP_GRAPH[size]) {
            // a refused replay (no device memory left for the graph) has run nothing
            g.failed = cudaGraphLaunch(exec, stream) != cudaSuccess;
            if (g.failed)
                cudaGetLastError();
            else
                n -= STEP_GRAPH[size];
        }
    }
    return n > 0 ? launch(n) : cudaSuccess;
}

}  // namespace lbm
