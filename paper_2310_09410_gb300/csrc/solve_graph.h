// A solve's WHILE graph: the captured loop body, what it was captured for, and
// the device tables that its launches point to.
#pragma once

#include <cuda_runtime.h>

#include <cstring>
#include <memory>
#include <string>

struct GraphCache {
    cudaGraphExec_t exec = nullptr;
    cudaGraph_t graph = nullptr;
    bool host_loop = false;
    double rho = 0;
    int k = 0, R = 0, kind = -1, P = 0;
    // A captured launch holds raw pointers.  Tables that belong to a plan and
    // are freed when the plan is built again are kept here as long as the graph,
    // so neither the memory nor the address can be another plan's while the
    // graph exists: the same object means the same contents.
    std::shared_ptr<const void> tables;

    bool matches(int kind_, double rho_, int k_, int R_, bool host_loop_, int P_,
                 const std::shared_ptr<const void> &tables_) const {
        return kind == kind_ && rho == rho_ && k == k_ && R == R_ && host_loop == host_loop_ && P == P_ &&
               tables == tables_;
    }
    void reset() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        exec = nullptr;
        graph = nullptr;
        kind = -1;
        tables.reset();
    }
};

// Captures "while (condition) body" into *gc: body(cond) enqueues one pass on
// `s`, its kernels set the condition; it returns nonzero when a launch was
// refused.  A graph that lacks one of its launches is dropped: the loop might
// run without the kernel that ends it, for ever.
// cudaSuccess, or the error with *err telling where (gc is empty then).  A
// launch that fails under capture invalidates the capture, and ending that one
// destroys the graph it went into: the body, which its parent would destroy a
// second time (the process ends there, seen with a launch of too much shared
// memory).  So the parent of an invalidated body is left alone.
template <typename Body>
cudaError_t capture_while(GraphCache *gc, cudaStream_t s, Body body, std::string *err) {
    gc->reset();
    gc->host_loop = false;
    auto failed = [&](const char *where, cudaError_t e) {
        *err = std::string(where) + ": " + cudaGetErrorString(e);
        gc->reset();
        return e;
    };
    cudaError_t e = cudaGraphCreate(&gc->graph, 0);
    if (e != cudaSuccess) return failed("cudaGraphCreate", e);
    cudaGraphConditionalHandle cond;
    e = cudaGraphConditionalHandleCreate(&cond, gc->graph, 1, cudaGraphCondAssignDefault);
    if (e != cudaSuccess) return failed("cudaGraphConditionalHandleCreate", e);
    // the parameter union has no default constructor in C++: zeroed storage
    alignas(cudaGraphNodeParams) unsigned char raw[sizeof(cudaGraphNodeParams)];
    memset(raw, 0, sizeof(raw));
    cudaGraphNodeParams *cp = reinterpret_cast<cudaGraphNodeParams *>(raw);
    cp->type = cudaGraphNodeTypeConditional;
    cp->conditional.handle = cond;
    cp->conditional.type = cudaGraphCondTypeWhile;
    cp->conditional.size = 1;
    cudaGraphNode_t node;
    e = cudaGraphAddNode(&node, gc->graph, nullptr, nullptr, 0, cp);
    if (e != cudaSuccess) return failed("cudaGraphAddNode", e);
    cudaGetLastError();                  // an older error is not this capture's
    e = cudaStreamBeginCaptureToGraph(s, cp->conditional.phGraph_out[0], nullptr, nullptr, 0,
                                      cudaStreamCaptureModeRelaxed);
    if (e != cudaSuccess) return failed("cudaStreamBeginCaptureToGraph", e);
    const int refused = body(cond);
    cudaError_t launch = cudaGetLastError();
    if (launch == cudaSuccess && refused) launch = cudaErrorInvalidConfiguration;
    cudaGraph_t captured = nullptr;
    e = cudaStreamEndCapture(s, &captured);
    if (e != cudaSuccess) gc->graph = nullptr;
    if (launch != cudaSuccess) return failed("launch under stream capture", launch);
    if (e != cudaSuccess) return failed("stream capture", e);
    e = cudaGraphInstantiate(&gc->exec, gc->graph, 0);
    if (e != cudaSuccess) return failed("cudaGraphInstantiate", e);
    return cudaSuccess;
}
