// Solver entry points shared between solver.cu (even-odd BiCGStab with FP64
// defect correction) and precond.cu (flexible GCR with the learned preconditioner).
#pragma once
#include "dirac.cuh"

namespace laph {

// Solves K x = b for right-hand sides [first, first+nr) of the ABI arrays with the even-odd
// BiCGStab path of prm.mode (PLAIN_FP64 or MIXED_FP32); writes sol and rep[first..].
void solve_block(laph_ctx *ctx, const DiracOp &op, const c64 *rhs, c64 *sol, int first, int nr,
                 const laph_solver_params &prm, laph_solve_report *rep, cudaStream_t s);

// The FP32 inner BiCGStab in one kernel, a cluster per right-hand side (bicg_small.cu): whether the
// lattice and block are small enough that it is the faster form, and the solve (x = 0 start, device
// iters / status per right-hand side: 0 budget spent, 1 converged, 2 breakdown).
bool bicg_small_fits(const DiracOp &op, int nr);
void bicg_small(const DiracOp &op, int nr, const c32 *b, c32 *x, double rel_tol, int maxiter, int *iters, int *status,
                cudaStream_t s);

// Same contract with FP64 defect correction around FP32 flexible GCR preconditioned by the
// network of weights (device pointer, layout of laph_precond_train).
void solve_block_learned(laph_ctx *ctx, const DiracOp &op, const float *weights, const c64 *rhs, c64 *sol, int first,
                         int nr, const laph_solver_params &prm, laph_solve_report *rep, cudaStream_t s);

}  // namespace laph
