// scalar.cuh -- interfaces of the decoupled scheme's scalar solves: the WHILE
// loop capture shared by the graph-form solves, and the elliptic solve on its
// one field (amg_scalar.cu).
#pragma once

#include <functional>

#include "amg_internal.cuh"

namespace bd {

// A device-controlled WHILE loop in a graph being captured on s: the handle first
// (the kernel that opens the loop needs it), then the body captured on s2.
struct WhileNode {
    cudaGraphConditionalHandle cond = 0;
    cudaGraphNode_t node = nullptr;
};
int while_handle(cudaStream_t s, WhileNode *w);
int while_begin(cudaStream_t s, cudaStream_t s2, WhileNode *w);
int while_end(cudaStream_t s, cudaStream_t s2, WhileNode *w);
void drop_capture(cudaStream_t s);  // end a failed capture quietly
bool solve_graph_off();             // BD_SOLVE_GRAPH=0

// report of a graph-form solve from its scalar block; returns the status
int info_from_scal(const double *scal, float ms, solve_info *info);

// x = C r with the projected coarsest inverse, n unknowns
int coarse_solve(int n, const double *C, const double *r, double *x, cudaStream_t s);
int coarse_solve(int n, const double *C, const float *r, float *x, cudaStream_t s);

// amg_options.autotune for an operator in block-CSR form: *lanes, the rule's choice,
// gives way to the candidate run(T) is fastest with (operators of few blocks keep it)
int tune_csr_lanes(const BSR &M, const std::function<int(int)> &run, cudaStream_t s, int *lanes);

// Elliptic hierarchies (bd_elliptic_setup): the scalar form of the V-cycle.
int scalar_build(amg_hierarchy *h, const bd_system *sys, cudaStream_t s);
// whether the scalar solve runs (not with live timing, strict mode, graphs off or
// a degree-1 smoother: the block solve serves those)
bool scalar_ready(amg_hierarchy *h, const solve_options *o);
// amg_set_level_lanes' form T for a one-field operator: as many lanes a row (a
// sliced form stands for its lanes, with the same bits), and for the form setup chose
// for the block operator the one it chose here
void scalar_set_lanes(amg_hierarchy *h, int level, int op, int T);
// (Ai + Ae) x = f from the x given; f, x: N doubles on the device
int scalar_solve(amg_hierarchy *h, const double *f, double *x, const solve_options *o, cudaStream_t s, solve_info *info);

}  // namespace bd
