// Core numbers and removal rounds of the static graph (core.cu).
#pragma once
#include "internal.cuh"

namespace folty {

// Control words of the kernel that the preprocessing reads back.
enum { CORE_ERR = 2, CORE_ROUNDS = 3, CORE_ALPHA = 4 };

// Writes g->core and rnd (removal round of every vertex: u leaves before v when rnd[u] <
// rnd[v], or they are equal and u < v) from the CSR rows of the n vertices (adj_src: the row of every entry) with degrees
// g->deg; returns the control words (device): error (1: a grid barrier wait ran out, 2: a
// vertex list overflowed), rounds in all, highest level. One block per SM on `blocks` SMs.
const int* enqueue_core_numbers(folty_graph* g, const int32_t* rowptr, const int32_t* adj, const int32_t* adj_src,
                                int32_t* rnd, int blocks, Scratch& sc, cudaStream_t s);

}  // namespace folty
