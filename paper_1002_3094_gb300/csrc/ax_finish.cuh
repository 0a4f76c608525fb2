// Scalar steps of the iterations, performed by the last CTA of a right-hand
// side to finish a kernel.  One iteration needs three sums over the grid; as
// separate one-warp launches each costs about 1.2 us of a captured graph's time
// plus its own latency (2.9-4.3 us in a serialised trace), the larger half of an
// iteration of one right-hand side; here it costs one atomic per CTA.
#pragma once
#include "ax_common.cuh"

namespace ax {

// The rule of `f` for right-hand side m with the summed partials v (one
// thread).  bb: ||phi||^2 (kFinStart only).
__device__ inline void finish_rule(const Finish &f, int m, double v, double bb) {
  RhsState s = f.st[m];
  switch (f.kind) {
    case kFinAlpha:
      if (!(v > 0.0) || !isfinite(v) || !isfinite(s.rho)) {
        s.state = kFailed;
        s.status = AX_ERR_BREAKDOWN;
      } else {
        s.alpha = s.rho / v;
      }
      break;
    case kFinUpdate:
      // After the x, r update: count the iteration and test the recursive
      // residual.  on_converge == kDue: a right-hand side that passes its
      // threshold goes on to the end of the iteration and is marked due for the
      // replacement step there (mixed PCG).
      if (s.state != kActive) return;  // kRedo: x and r were not changed
      s.rr = v;
      s.iters += 1;
      if (!isfinite(v)) {
        s.state = kFailed;
        s.status = AX_ERR_BREAKDOWN;
      } else if (v <= s.thresh2) {
        if (f.on_converge == kDue) s.due = 1;
        else s.state = f.on_converge;
      } else if (s.iters >= s.max_iter) {
        s.state = (f.on_converge == kDone) ? kDone : kFailed;
        if (f.on_converge != kDone) s.status = AX_ERR_NO_CONVERGENCE;
      }
      break;
    case kFinBeta: {
      // use_prev: the right-hand side already took this iteration's direction
      // update from its recursive residual; the new beta refers to the rho
      // before that update (mixed PCG residual replacement)
      const bool prev = s.state == kRedo && s.use_prev != 0;
      const double rho = prev ? s.rho_prev : s.rho;
      if (!isfinite(v) || rho == 0.0) {
        s.state = kFailed;
        s.status = AX_ERR_BREAKDOWN;
      } else {
        if (!prev) s.rho_prev = rho;
        s.beta = v / rho;
        s.rho = v;
        s.state = kActive;
      }
      break;
    }
    case kFinGateRes:
      s.gate_res = v;
      [[fallthrough]];
    case kFinRho:
      s.rho = v;
      s.beta = 0.0;
      if (f.kind == kFinRho && !isfinite(v)) {
        s.state = kFailed;
        s.status = AX_ERR_BREAKDOWN;
      }
      break;
    case kFinGatePhi: s.gate_phi = v; break;
    case kFinTrueCheck:  // the true residual of a right-hand side in kCheck
      s.rr = v;
      if (v <= s.thresh2) {
        s.state = kDone;
      } else if (s.iters >= s.max_iter) {
        s.state = kFailed;
        s.status = AX_ERR_NO_CONVERGENCE;
      } else {
        s.state = kRedo;
        s.alpha = 0.0;
        s.use_prev = 0;
      }
      break;
    case kFinReplace: {
      // Residual replacement: v = ||phi - A x||^2 just computed.  The
      // iteration's z and rho came from the recursive residual: when the true
      // one differs noticeably (||r||^2 by more than 1%: typically once the
      // recursion has run below the FP32 accuracy of x), z = B^-1 r and beta are
      // recomputed from the new r (kRedo).
      const double tol2 = f.par[0], delta2 = f.par[1];
      const bool consistent = fabs(v - s.rr) <= 1e-2 * v;
      s.rr = v;
      s.due = 0;
      s.tmp += 1.0;  // replacements
      s.xbase = s.iters + f.xoff;
      if (!isfinite(v)) {
        s.state = kFailed;
        s.status = AX_ERR_BREAKDOWN;
      } else if (v <= tol2 * s.bb) {
        s.state = kDone;
      } else if (s.iters >= s.max_iter) {
        s.state = kFailed;
        s.status = AX_ERR_NO_CONVERGENCE;
      } else {
        s.thresh2 = fmax(delta2 * v, 0.25 * tol2 * s.bb);
        if (!consistent) {
          s.state = kRedo;
          s.alpha = 0.0;
          s.use_prev = 1;
          atomicAdd(f.chk, 1);
        }
      }
      break;
    }
    case kFinStart: {
      // Mixed PCG with residual replacement: start.  v = ||phi - A x||^2; the
      // FP32 iteration runs until its recursive residual falls below
      // thresh2 = max(delta^2 rr_true, (tol/2)^2 bb), then the true residual
      // replaces it.
      const double tol2 = f.par[0], delta2 = f.par[1];
      s = RhsState{};
      s.rr = v;
      s.bb = bb;
      s.max_iter = f.max_iter;
      s.status = AX_OK;
      s.xbase = f.xoff;
      if (!isfinite(v) || !isfinite(bb)) {
        s.state = kFailed;
        s.status = AX_ERR_BREAKDOWN;
      } else if (v <= tol2 * bb || bb == 0.0) {
        s.state = kDone;
      } else {
        s.state = kActive;
        s.thresh2 = fmax(delta2 * v, 0.25 * tol2 * bb);
      }
      break;
    }
    case kFinCheb: {
      // Chebyshev: v = ||A y - phi||^2 of the current iterate; stop or continue
      // and advance alpha_{k+1} = 4 / (4 - rho0^2 alpha_k) (alpha for the first
      // step is 1).  check = 0: a step without the residual norm.
      const double rho0sq = f.chp[2 * m + 1];
      const double rr = f.check ? v : s.rr;
      s.rr = rr;
      if (!isfinite(rr)) {
        s.state = kFailed;
        s.status = AX_ERR_BREAKDOWN;
      } else if (f.check && rr <= s.thresh2) {
        s.state = f.on_converge;
      } else if (s.iters >= s.max_iter) {
        s.state = (f.on_converge == kDone) ? kDone : kFailed;
        if (f.on_converge != kDone) s.status = AX_ERR_NO_CONVERGENCE;
      } else {
        if (s.iters == 0) {
          s.cheb_a = 1.0;  // y_1 = y_0 - tau B^-1 (A y_0 - phi) (the y_{-1} term drops out)
        } else {
          const double prev = (s.iters == 1) ? 2.0 : s.cheb_a;
          s.cheb_a = 4.0 / (4.0 - rho0sq * prev);
        }
        s.iters += 1;
      }
      break;
    }
    default: return;
  }
  f.st[m] = s;
}

// Arrival of a CTA at right-hand side m (one thread, after it has written the
// CTA's partial; the CTA's other use of the state is behind a barrier): true for
// the last of `total`, which also returns the count to zero for the next launch.
__device__ __forceinline__ bool finish_arrive(const Finish &f, int m, unsigned total) {
  __threadfence();
  const bool last = atomicAdd(f.count + m, 1u) == total - 1;
  if (last) {
    f.count[m] = 0;
    __threadfence();
  }
  return last;
}

// The last CTA (every thread): sums the nb partials (each thread a stride of
// them, then block_sum: an order fixed by nb and the block size) and applies the
// rule.
__device__ __forceinline__ void finish_last(const Finish &f, int m, const double *part, int nb, double *red) {
  double v = 0.0, bb = 0.0;
  if (part != nullptr) {
#pragma unroll 4
    for (int i = threadIdx.x; i < nb; i += blockDim.x) v += __ldcg(part + i);
  }
  v = block_sum(v, red);
  if (f.kind == kFinStart) {
    if (f.bb != nullptr) {
      for (int i = threadIdx.x; i < f.nbb; i += blockDim.x) bb += __ldcg(f.bb + (size_t)m * kPartialStride + i);
      bb = block_sum(bb, red);
    } else {
      bb = v;
    }
  }
  if (threadIdx.x == 0) finish_rule(f, m, v, bb);
}

// Called by every thread of every CTA of right-hand side m after thread 0 has
// written the CTA's partial; `total` = CTAs of this right-hand side, part its
// nb partials, red as in block_sum.
__device__ __forceinline__ void finish_rhs(const Finish &f, int m, unsigned total, const double *part, int nb,
                                           double *red) {
  if (f.kind == kFinNone) return;
  __shared__ int s_last;
  if (threadIdx.x == 0) s_last = finish_arrive(f, m, total);
  __syncthreads();
  if (s_last) finish_last(f, m, part, nb, red);
}

}  // namespace ax
