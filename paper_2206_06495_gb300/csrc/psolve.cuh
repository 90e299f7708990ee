// The preconditioned pressure solve as one resident kernel (psolve.cu), and
// the direct solve of small systems (dsolve.cu).
#pragma once

#include "amg.cuh"
#include "common.cuh"

namespace rbffd {

struct PSolve;

// polls of a grid barrier's wait in the kernels that `ctx` launches
long long barrier_polls(const rbffd_ctx* ctx);

// Up to this many rows the resident kernel is the faster form.  Milliseconds of
// a step for each of its pressure iterations, resident against launched, of two
// flows: rows of 28 entries, FP64, 0.69 and 0.63 against 0.71 and 0.66 at 1.10M
// rows, 0.71 and 0.81 against 0.66 and 0.74 at 1.21M, 0.90 and 0.89 against
// 0.83 and 0.83 at 1.32M, 1.24 against 1.11 at 2.0M (1.69M alone is even);
// MIXED 0.53 against 0.53 and 0.54 at 1.10M, 0.58 and 0.57 against 0.56 and
// 0.55 at 1.21M, 0.87 against 0.83 at 2.0M.  Rows of another width, whose
// products are loops, FP64 at 2.0M: 1.51 against 1.54 (21 entries) and 1.66
// against 1.95 (composed); larger systems have not been measured.
constexpr int64_t kResidentMax28 = 1150000, kResidentMax = 1 << 21;

struct PSolveResult {
  int iters = 0;
  int status = 0;  // as KScal::status of step.cu
  double relres = 0.0;
  bool converged = false;
};

// A solve's result and, behind it, its barrier's words: one copy to the host.
constexpr int kBarrierWords = 3;
struct SolveStatus {
  PSolveResult res;
  unsigned int bar[kBarrierWords];
};

// Build the solve's copies for one plan: the scaled pressure operator (idx, w
// [k][ld], rank-one column es, row sums a1; M rows) in the hierarchy's level-0
// order, in FP64, or in FP32 when `mix` is set, and its work vectors.  *out
// stays null when the memory or the SMs do not suffice (the caller then solves
// as separate launches), as in the builders below.
int psolve_build(rbffd_ctx* ctx, int64_t M, int64_t ld, int k, const int32_t* idx,
                 const double* w, const double* es, const double* a1, const Amg* amg, bool mix,
                 PSolve** out, cudaStream_t st);
void psolve_free(PSolve* p);

// Right-preconditioned BiCGSTAB on the scaled pressure system, x (in: the
// initial iterate, not read when x_zero; out: the solution) and b in P-node
// order; T = float or double as the plan was built.  Synchronises `st`.
// `launches` is increased by the kernels launched.
template <typename T>
int psolve_run(rbffd_ctx* ctx, PSolve* p, T* x, const T* b, double tol, int maxit, uint32_t seed,
               bool x_zero, PSolveResult* res, int64_t* launches, cudaStream_t st);

// Small systems (M <= kDenseMax) are solved directly: the dense FP64 inverse
// of the scaled pressure operator, built once per plan, applied with iterative
// refinement.
//
// Where the line lies: a solve is one or two products with the inverse and
// their residuals, 50 us with cold caches at 1,600 rows, against 40 to 55 us for
// EACH of the 40 to 500 Krylov iterations that these sizes take.  At 4,096 the
// inverse (134 MB) no longer fits L2; beyond it the inversion (n^3 FP64 FMAs)
// would cost a first pass more than the hierarchy it replaces.
constexpr int kDenseMax = 4096;
struct DSolve;

// *out stays null when the operator is numerically singular, too (the caller
// then takes the Krylov solve).  Synchronises `st`.
int dsolve_build(rbffd_ctx* ctx, int64_t M, int64_t ld, int k, const int32_t* idx,
                 const double* w, const double* es, DSolve** out, cudaStream_t st);
void dsolve_free(DSolve* d);
// x (in: the initial iterate, out: the solution) and b in P-node order.
// Refines until the relative residual is at most tol; res->iters counts the
// products with the inverse.  status 5: the refinement stalled above tol.
int dsolve_run(rbffd_ctx* ctx, DSolve* d, double* x, const double* b, double tol,
               PSolveResult* res, int64_t* launches, cudaStream_t st);

// The viscous systems of a small flow, both components in one resident kernel:
// BiCGSTAB on x + w x = b with the component's weights wu or wv (the same
// pointer in a closed flow) on shared indices.
struct VSolve;
int vsolve_build(rbffd_ctx* ctx, int64_t N, int64_t ld, int k, const int32_t* idx,
                 const double* wu, const double* wv, VSolve** out, cudaStream_t st);
void vsolve_free(VSolve* v);

// The two solves of a small flow's step, enqueued without waiting for their
// results, so that the host can run steps ahead of the GPU.  `fail` (device)
// is 0 or what ended an earlier step: then nothing is done.  A solve that
// misses its tolerance sets it to (step << 4) | kFail*.  *res (device) gets
// the result.  small_reset before a run of steps.
constexpr int kFailViscous = 1, kFailPressure = 2, kFailWait = 3;
struct SmallStep {
  PSolveResult visc, pres;
};
cudaError_t small_reset(VSolve* v, DSolve* d, int* fail, cudaStream_t st);
// accept: a relative residual up to which a viscous solve short of tol passes
cudaError_t vsolve_enqueue(VSolve* v, double* const* x, const double* const* b, double tol,
                           double accept, int maxit, PSolveResult* res, int* fail, int step,
                           long long polls, cudaStream_t st);
cudaError_t dsolve_enqueue(DSolve* d, double* x, const double* b, double tol, PSolveResult* res,
                           int* fail, int step, long long polls, cudaStream_t st);

}  // namespace rbffd
