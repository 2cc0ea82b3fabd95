"""When steps are replayed from graphs, and what follows a graph that cannot be made, instantiated or replayed: the host
code of lbm_step_graphs.h against a fake of the CUDA runtime that records its calls and fails the wanted one."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HARNESS = r"""
#include "lbm_step_graphs.h"
#include <cstdio>
#include <cstdlib>
#include <map>
#include <string>
static std::map<std::string, int> fail;  // call -> which use of it fails (-1: every one)
static std::map<std::string, int> used;
static cudaError_t call(const char* what) {
    const int k = ++used[what];
    auto f = fail.find(what);
    return f != fail.end() && (f->second < 0 || f->second == k) ? cudaErrorMemoryAllocation : cudaSuccess;
}
static bool user_capture = false;
static long recorded = 0, ran_plain = 0, ran_graph = 0;
static cudaStream_t U = (cudaStream_t)16;
extern "C" {
cudaError_t cudaStreamSynchronize(cudaStream_t) { return call("sync"); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return call("destroy"); }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) {
    recorded = 0;
    *g = (cudaGraph_t)8;
    return call("create");
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
    const cudaError_t e = call("instantiate");
    if (e == cudaSuccess) *x = (cudaGraphExec_t)recorded;  // an executable graph "is" its number of steps
    return e;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) {
    if (s != U || !x) abort();
    const cudaError_t e = call("replay");
    if (e == cudaSuccess) ran_graph += (long)x;
    return e;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
    *c = user_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
}
// arguments: n = a call of n steps; shape:k = another launch shape; fail:what:k, ok:what; user:0/1 = caller's capture
int main(int argc, char** argv) {
    lbm::StepGraphs g;
    int shape[6] = {0, 0, 0, 0, 0, 0}, cur = 0;
    lbm::GraphRecord* record = nullptr;
    for (int i = 1; i < argc; ++i) {
        const std::string a = argv[i];
        if (a.rfind("shape:", 0) == 0) { shape[1] = atoi(a.c_str() + 6); continue; }
        if (a.rfind("user:", 0) == 0) { user_capture = a[5] == '1'; continue; }
        if (a.rfind("ok:", 0) == 0) { fail.erase(a.substr(3)); continue; }
        if (a.rfind("fail:", 0) == 0) {
            const size_t c = a.rfind(':');
            fail[a.substr(5, c - 5)] = atoi(a.c_str() + c + 1);
            continue;
        }
        const long n = atol(argv[i]);
        ran_plain = ran_graph = 0;
        used["create"] = used["instantiate"] = used["replay"] = 0;
        const int start = cur;
        const cudaError_t e = lbm::run_steps(g, shape, U, record, cur, n, [&](long k) {
            (record ? recorded : ran_plain) += k;
            cur ^= k & 1;
            return record ? call("node") : cudaSuccess;
        });
        if (e != cudaSuccess || record || ran_plain + ran_graph != n || cur != (start ^ (int)(n & 1))) {
            printf("wrong\n");
            return 1;
        }
        printf("%ld/%ld/%d%s ", ran_graph, ran_plain, used["create"], g.failed ? "F" : "");
    }
    g.drop(nullptr);
    printf("\n");
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    from paper_2010_01628_gb300 import build
    d = tmp_path_factory.mktemp("step_graphs")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    r = subprocess.run([shutil.which("g++") or "c++", "-std=c++17", "-Wall", "-I", build.CSRC, "-I", cuda, str(src),
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(*args):
        p = subprocess.run([str(exe), *[str(a) for a in args]], capture_output=True, text=True, timeout=60)
        assert p.returncode == 0, (args, p.stdout, p.stderr)
        return p.stdout.split()  # per call: steps replayed / launched singly / graphs begun, F once failed

    return run


def test_long_calls_replay_at_once(harness):
    assert harness(32) == ["32/0/1"]
    assert harness(100, 100, 100, 100) == ["96/4/1", "96/4/0", "96/4/0", "100/0/1"]
    assert harness(47, 47) == ["32/15/1", "32/15/1"]  # the other buffer is current in the second call


def test_short_calls_replay_four_steps_at_a_time(harness):
    assert harness(*[3] * 20) == ["0/3/0"] * 20
    assert harness(*[4] * 5) == ["0/4/0"] * 3 + ["4/0/1", "4/0/0"]
    assert harness(*[10] * 4) == ["0/10/0", "8/2/1", "8/2/0", "8/2/0"]
    assert harness(*[15] * 6) == ["0/15/0"] * 2 + ["12/3/1"] * 2 + ["12/3/0"] * 2  # the buffers in turn


def test_first_short_calls_of_a_context_make_no_graph(harness):
    assert harness(16) == ["0/16/0"]
    assert harness(16, 16, 16) == ["0/16/0", "16/0/1", "16/0/0"]
    # 31 = 16 + 12 + 3, the buffers in turn
    assert harness(*[31] * 6) == ["0/31/0", "0/31/0", "28/3/2", "28/3/2", "28/3/0", "28/3/0"]


@pytest.mark.parametrize("call", ["create", "node", "instantiate"])
def test_a_graph_that_cannot_be_made_is_not_tried_again(harness, call):
    out = harness(f"fail:{call}:-1", 64, f"ok:{call}", 64, 64)
    assert out == ["0/64/1F", "0/64/0F", "0/64/0F"]
    # the graph of 4 steps fails after that of 16 was made
    assert harness(44, f"fail:{call}:-1", 44, f"ok:{call}", 44) == ["32/12/1", "32/12/1F", "0/44/0F"]


def test_a_refused_replay_falls_back_to_launches(harness):
    assert harness("fail:replay:2", 64, 64) == ["16/48/1F", "0/64/0F"]


def test_a_new_launch_shape_starts_over(harness):
    assert harness("fail:instantiate:-1", 64, "ok:instantiate", "shape:2", 64, 64) == ["0/64/1F", "64/0/1", "64/0/0"]
    assert harness(64, "shape:2", 16, 64) == ["64/0/1", "0/16/0", "64/0/1"]


def test_a_callers_capture_records_plain_launches(harness):
    assert harness("user:1", 64, "shape:2", 64, "user:0", 64) == ["0/64/0", "0/64/0", "64/0/1"]
