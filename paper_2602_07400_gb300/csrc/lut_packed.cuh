// Interface of lut_packed.cu inside the library.
#pragma once

#include "common.cuh"

namespace bitlogic {

// Where a node's output gradient dY[j][.] comes from.
//   rows:  dY + (j / group) * B   (group = 1: one row per node; group = g:
//          the head's per-class gradient, shared by the g nodes of a class)
//   terms: sum over e in [off[j], off[j+1]) of terms[edge[e]][.] in
//          increasing e -- the next layer's input gradient, reduced on the
//          fly from its per-edge terms instead of being materialised.  With
//          edge == nullptr the term rows are stored in CSR order (row e).
struct GradSource {
    const float* dY;
    int group;
    const float* terms;
    const int* off;
    const int* edge;
    int n_edges;
};

// Layer backward with per-edge input-gradient terms, k = 3..6, any B and
// alignment: dtheta, and P[row(e)][s] for edge e = j*k + i, row(e) = epos[e]
// when epos is given.  Returns a bitlogic status code.
int launch_backward_packed(int k, const float* X, int w_in, long long B, const int* conn, const float* theta, int w,
                           int node, const GradSource& gs, float* dtheta, float* P, const int* epos, float* dY_out,
                           cudaStream_t st);

}  // namespace bitlogic
