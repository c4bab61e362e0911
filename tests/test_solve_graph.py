"""A solve's graph and the tables it points to (`csrc/solve_graph.h`).

On the CPU, against a stand-in for the CUDA runtime: a graph captured for one
plan's tables keeps them alive and does not match a plan built again with the
same CTA count, in whatever order the two are freed; and a capture that loses
a launch (the runtime's error, or the launcher's refusal) gives an error and no
graph, since the loop would lack the kernel that ends it, and destroys no body
twice.

On the GPU: a request that does not fit between two equal single-precision
solves (the plan, and with it its tables, is built again) leaves the iterates
as a fresh handle's, bit for bit."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2310_09410_gb300", "csrc")

RUNTIME = r"""
#pragma once
typedef void *cudaGraphExec_t;
typedef void *cudaGraph_t;
typedef void *cudaGraphNode_t;
typedef void *cudaStream_t;
typedef unsigned long long cudaGraphConditionalHandle;
enum cudaError_t { cudaSuccess, cudaErrorInvalidValue, cudaErrorInvalidConfiguration };
enum { cudaGraphCondAssignDefault, cudaGraphNodeTypeConditional, cudaGraphCondTypeWhile, cudaStreamCaptureModeRelaxed };
struct cudaGraphNodeParams {
    int type;
    struct { cudaGraphConditionalHandle handle; int type; unsigned size; cudaGraph_t *phGraph_out; } conditional;
};
inline int destroyed = 0, alive = 0, instantiated = 0, capturing = 0, broken = 0, ended_twice = 0, mark;
inline cudaError_t last = cudaSuccess;
inline cudaGraph_t loop_body = &mark;
inline int cudaGraphExecDestroy(cudaGraphExec_t) { ++destroyed; --alive; return 0; }
inline int cudaGraphDestroy(cudaGraph_t) { ++destroyed; --alive; ended_twice += broken; return 0; }
inline cudaError_t cudaGraphCreate(cudaGraph_t *g, unsigned) { *g = &mark; ++alive; broken = 0; return cudaSuccess; }
inline cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle *h, cudaGraph_t, unsigned, unsigned) {
    *h = 7; return cudaSuccess;
}
inline cudaError_t cudaGraphAddNode(cudaGraphNode_t *, cudaGraph_t, const cudaGraphNode_t *, const void *, unsigned,
                                    cudaGraphNodeParams *p) { p->conditional.phGraph_out = &loop_body; return cudaSuccess; }
// a launch that fails under capture invalidates it, and its end destroys the body graph
inline void launch_fails(cudaError_t e) { last = e; broken = 1; }
inline cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
inline cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t *, const void *, unsigned,
                                                 int) { ++capturing; return cudaSuccess; }
inline cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) {
    --capturing; return broken ? cudaErrorInvalidValue : cudaSuccess;
}
inline cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned) {
    *x = &mark; ++alive; ++instantiated; return cudaSuccess;
}
inline const char *cudaGetErrorString(cudaError_t) { return "error"; }
"""

DRIVER = r"""
#include "solve_graph.h"
#include <cstdio>
struct Tables { int *freed; ~Tables() { ++*freed; } };
static int line = 0;
#define CHECK(x) do { if (!(x)) { std::printf("FAIL %d: %s\n", line, #x); return 1; } ++line; } while (0)
int main() {
    int freed = 0, one = 1;
    GraphCache g;
    auto plan = std::make_shared<Tables>(Tables{&freed});     // the plan's tables
    freed = 0;                                                // (the temporary's end)
    g.exec = g.graph = &one;
    g.kind = 4; g.rho = 100.0; g.k = 50; g.R = 1000; g.P = 10304; g.tables = plan;
    CHECK(g.matches(4, 100.0, 50, 1000, false, 10304, plan));
    plan.reset();                                             // a request that does not fit replaces them
    CHECK(freed == 0);                                        // the graph still points to them
    plan = std::make_shared<Tables>(Tables{&freed});          // built again for the same CTA count
    freed = 0;
    CHECK(plan != g.tables && !g.matches(4, 100.0, 50, 1000, false, 10304, plan));
    CHECK(!g.matches(4, 100.0, 50, 1000, false, 10304, nullptr));
    g.reset();
    CHECK(freed == 1 && destroyed == 2 && !g.tables);         // freed with the graph, not before
    CHECK(!g.matches(4, 100.0, 50, 1000, false, 10304, plan));
    // captures: whole; a launch that fails; a launcher that refuses; whole after an older error
    alive = 0;
    std::string why;
    auto capture = [&](cudaError_t launch, int refused) {
        return capture_while(&g, nullptr, [&](cudaGraphConditionalHandle c) {
            if (launch != cudaSuccess) launch_fails(launch);
            return c == 7 ? refused : 1;
        }, &why);
    };
    CHECK(capture(cudaSuccess, 0) == cudaSuccess && g.exec && alive == 2 && instantiated == 1);
    g.kind = 4;
    CHECK(capture(cudaErrorInvalidValue, 0) == cudaErrorInvalidValue && !why.empty());
    // (the parent, whose body is gone, is left alone)
    CHECK(!g.exec && !g.graph && alive == 1 && ended_twice == 0 && instantiated == 1 && capturing == 0 && g.kind == -1);
    alive = 0;
    CHECK(capture(cudaSuccess, 1) != cudaSuccess && !g.exec && alive == 0 && instantiated == 1 && capturing == 0);
    last = cudaErrorInvalidValue;
    CHECK(capture(cudaSuccess, 0) == cudaSuccess && g.exec && alive == 2 && instantiated == 2);
    g.reset();
    std::printf("ok\n");
    return 0;
}
"""


def test_graph_holds_its_tables_and_needs_its_launches(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "driver.cpp").write_text(DRIVER)
    exe = tmp_path / "driver"
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-Wall", "-I", str(tmp_path), "-I", CSRC,
                           str(tmp_path / "driver.cpp"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.rstrip().endswith("ok"), out.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "mixed"])
def test_request_that_does_not_fit_between_equal_solves(precision):
    from paper_2310_09410_gb300 import opf, synth

    feeder = synth.make_feeder(1000, 690, 83, depth_max=60, p_single=0.7, seed=11)
    prec = opf.PREC_FP32 if precision == "fp32" else opf.PREC_MIXED

    def solved(s, **how):
        s.reset()
        s.solve(eps_rel=0.0, max_iter=1100, check_every=50, precision=prec, **how)
        return s.locals() + s.solution()

    got = []
    with opf.Solver.from_feeder(feeder) as s:
        s.precompute()
        for how in ({}, {"engine": opf.ENGINE_PERSISTENT}):
            got.append(solved(s, **how))
            for ctas in (2, 1):                  # thousands of slots per CTA
                with pytest.raises(opf.OPFError) as e:
                    solved(s, engine=opf.ENGINE_PERSISTENT, cluster=ctas)
                assert e.value.code == opf.OPF_E_CAPACITY
                got.append(solved(s, **how))
    with opf.Solver.from_feeder(feeder) as fresh:
        fresh.precompute()
        want = solved(fresh)
    for g in got:
        for a, b in zip(g, want):
            assert np.array_equal(a, b)
