// A solve's WHILE graph: the captured loop body, what it was captured for, and
// the device tables that its launches point to.
#pragma once

#include <cuda_runtime.h>

#include <memory>

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
