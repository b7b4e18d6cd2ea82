// The step rule of the device-resident CG (solver.cu).  Plain C++, so that it can be checked on a
// machine without a GPU.
#pragma once

#ifdef __CUDACC__
#define KQR_HD __host__ __device__ __forceinline__
#else
#define KQR_HD inline
#endif

namespace kqr {

// CG status (S_CGST): running, met tol, stopped at a non-positive curvature, non-finite, maxit.
enum CgState { CG_RUN = 0, CG_MET = 1, CG_TRUNC = 2, CG_NONFINITE = 3, CG_MAXIT = 4 };

struct CgStep {
  double a;      // step length
  int state;     // CG_RUN, or why CG stops with this step
};

// The operator is positive definite; a curvature at or below the product's rounding level (floor) is
// rounding in directions whose eigenvalues lie below its accuracy (a numerically low-rank K), and
// dividing by it would blow the step up.  Truncate: keep x, or, with unit_first, take the
// preconditioned residual itself at the first step (a Newton step with the preconditioner as the
// Hessian model).  A solve that is not a Newton step (the adjoint systems of the held-out gradient)
// keeps x, zero at its first step: the preconditioned residual is no solution of its equations.
KQR_HD CgStep cg_step_rule(double pAp, double floor, double rz, bool first, bool unit_first) {
  if (!(pAp - pAp == 0.0)) return {0.0, CG_NONFINITE};
  if (!(pAp > floor)) return {first && unit_first ? 1.0 : 0.0, CG_TRUNC};
  return {rz / pAp, CG_RUN};
}

}  // namespace kqr
