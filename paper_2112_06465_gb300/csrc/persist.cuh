// persist.cuh -- the persistent single-kernel solvers (persist.cu)
#pragma once

#include "krylov.cuh"

namespace hz {

enum PsKind { PS_BICG = 0, PS_MIXED = 1, PS_TFQMR = 2 };

// whether a solve on this handle runs as one persistent kernel: a binary64
// handle in the row-per-lane layout, the Krylov vectors of its rows within
// the shared memory of the GPU's SMs
bool ps_fits(const hz_mat *A, PsKind k);
// (taken: false where the device has no room for the launch; nothing ran)
hz_status ps_solve(hz_mat *A, PsKind kind, const Ctl &c, Info *out, int *restarts, cudaStream_t s, bool *taken);
void ps_solver_free(void *p);

// a sweep of binary64 BiCGStab solves as one launch, each system on CTAs of
// its own: the CTAs of each (0 for an empty system), or false where the
// handles, their number or their sizes do not fit
bool ps_batch_plan(hz_mat *const *A, int ns, std::vector<int> *ncta);
hz_status ps_solve_batched(hz_mat *const *A, int ns, const std::vector<int> &ncta, const double2 *const *b,
                           double2 *const *x, double tol, int maxit, Info *out, cudaStream_t s, bool *taken);
void ps_batch_free(void *p);

}  // namespace hz
