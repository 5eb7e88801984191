// Shared by the two forms of the coefficient gradients (dq_grad.cu, dq_grad_panel.cu).
#pragma once

#include <cstddef>

#include <cuda_runtime.h>

#include "dq_internal.h"

namespace dq {

// The sector's gradient workspace, grown to `need` bytes (kept with the sector). 0 or a cudaError_t.
int grad_workspace(const dq_sector* s, size_t need, char** ws);

// All terms in one pass over panels. *taken is false, and nothing was done, when the sector or the term
// list does not fit; else queues the kernels on `st`. 0 or a cudaError_t.
int launch_grad_panel(const dq_sector* s, const dq_term* terms, int n_terms, const void* x, const void* dy, int dtype,
                      int cols, double* d_grads, cudaStream_t st, bool* taken);

}  // namespace dq
