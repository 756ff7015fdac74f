// ig_mixed.cuh -- the finish steps of the mixed-precision solve (see ig_pcg_mixed.cu), shared by its
// multi-CTA and resident kernels.
#pragma once

#include "ig_device.cuh"

namespace ig {
namespace {

// ------------------------------------------------------------------------------- bookkeeping
__device__ __noinline__ void finish_init_mixed(SolveScal* s, int k, const double* acc, double tol, double inner_tol,
                                               int max_iter, int max_refine) {
  int nact = 0, bad = 0;
  for (int c = 0; c < kMaxK; ++c) {
    const double bb = c < k ? acc[c] : 0.0;
    if (c < k && !is_finite(bb)) bad = 1;
    const int act = (c < k && positive_finite(bb)) ? 1 : 0;
    s->rhs2[c] = bb;
    s->bnorm2[c] = 0.0;
    s->active64[c] = act;
    s->active[c] = 0;
    s->relres2[c] = act ? 1.0 : 0.0;
    s->scale[c] = act ? sqrt(bb) : 1.0;
    s->rz[c] = 0.0;
    s->alpha[c] = 0.0;
    s->beta[c] = 0.0;
    s->trueres[c] = -1.0;
    nact += act;
  }
  s->k = k;
  s->cnt[0] = 0u;
  s->cnt[1] = 0u;
  s->iter = 0;
  s->refine = 0;
  s->inner_iter = 0;
  s->inner_cap = max_iter < 4000 ? max_iter : 4000;
  s->phase = kPhaseRestart;
  s->members = 0;
  s->off_chip = 0;
  s->tol2 = tol * tol;
  s->inner_tol2 = inner_tol * inner_tol;
  s->max_iter = max_iter;
  s->max_refine = max_refine;
  s->status = bad ? IG_ERR_NONFINITE : IG_OK;
  s->done = (bad || nact == 0) ? 1 : 0;
}

// The finish steps below run on the 32 lanes of warp 0 of the CTA that completes a mesh: lane c
// handles column c, lane 0 the mesh's own fields (written after the warp's votes). They read the
// scalars from cur, a shared-memory copy, and write them to s.

// After r64 = rhs - A64 x64: FP64 convergence test per column, the scale of the next inner
// right-hand side, and the refinement cap.
__device__ __noinline__ void finish_residual(SolveScal* s, const SolveScal& cur, int k, const double* res2) {
  const int c = threadIdx.x & 31;
  const int refine = cur.refine + 1;
  int act = 0, bad = 0;
  if (c < k && cur.active64[c] != 0) {
    if (!is_finite(res2[c])) {
      bad = 1;
    } else {
      const double rel2 = quotient(res2[c], cur.rhs2[c]);  // squares, as in finish_update
      s->relres2[c] = rel2;
      if (not_above(rel2, cur.tol2) || !positive_finite(res2[c])) {
        s->active64[c] = 0;
      } else {
        s->scale[c] = sqrt(res2[c]);
        act = 1;
      }
    }
  }
  const int nact = __popc(__ballot_sync(0xffffffffu, act));
  const int anybad = __any_sync(0xffffffffu, bad);
  if (c == 0) {
    s->refine = refine;
    if (anybad) {
      s->status = IG_ERR_NONFINITE;
      s->done = 1;
    } else if (nact == 0) {
      s->done = 1;
    } else if (refine >= cur.max_refine || cur.iter >= cur.max_iter) {
      s->status = IG_ERR_NOT_CONVERGED;
      s->done = 1;
    } else {
      s->phase = kPhaseRestart;
    }
  }
}

// After forming r32 = r64 / scale: start a new inner solve. Returns (on lane 0) the new phase.
__device__ __forceinline__ int finish_restart_step(SolveScal* s, const SolveScal& cur, int k, const double* acc) {
  const int c = threadIdx.x & 31;
  int act = 0;
  if (c < k) {
    act = (cur.active64[c] && positive_finite(acc[k + c])) ? 1 : 0;
    s->active[c] = act;
    s->rz[c] = acc[c];
    s->bnorm2[c] = acc[k + c];
    s->alpha[c] = 0.0;
    s->beta[c] = 0.0;
  }
  const int nact = __popc(__ballot_sync(0xffffffffu, act));
  const int phase = nact ? kPhaseInner : kPhaseApply;
  if (c == 0) {
    s->inner_iter = 0;
    s->phase = phase;
  }
  return phase;
}
__device__ __noinline__ int finish_restart(SolveScal* s, const SolveScal& cur, int k, const double* acc) {
  return finish_restart_step(s, cur, k, acc);
}

// Inner FP32 iteration: inner convergence test, beta, switch to Apply when the inner solve is done.
// Returns (on lane 0) the phase after it, or -1 when the mesh is done (a non-finite sum).
__device__ __forceinline__ int finish_update_mixed_step(SolveScal* s, const SolveScal& cur, int k, const double* acc) {
  const int c = threadIdx.x & 31, col = c & 7;
  int act = 0, bad = 0;
  const double* den = c < 8 ? cur.rz : cur.bnorm2;  // the divisions side by side, the test on squares (finish_update)
  const double* num = c < 8 ? acc : acc + k;
  double quot = 0.0;
  if (col < k && c < 16) quot = quotient(num[col], den[col]);
  const double rel2 = __shfl_down_sync(0xffffffffu, quot, 8);
  if (c < k && cur.active[c] != 0) {
    const double rzn = acc[c], rr = acc[k + c];
    if (!is_finite(rzn) || !is_finite(rr)) {
      bad = 1;
    } else {
      const double bta = quot;
      if (not_above(rel2, cur.inner_tol2) || !positive_finite(rzn)) {
        s->active[c] = 0;
        s->beta[c] = 0.0;
      } else {
        s->beta[c] = bta;
        s->rz[c] = rzn;
        act = 1;
      }
    }
  }
  const int nact = __popc(__ballot_sync(0xffffffffu, act));
  const int anybad = __any_sync(0xffffffffu, bad);
  int phase = kPhaseInner;
  if (c == 0) {
    const int it = cur.iter + 1, inner = cur.inner_iter + 1;
    s->iter = it;
    s->inner_iter = inner;
    if (anybad) {
      s->status = IG_ERR_NONFINITE;
      s->done = 1;
      phase = -1;
    } else if (nact == 0 || inner >= cur.inner_cap || it >= cur.max_iter) {
      s->phase = kPhaseApply;
      phase = kPhaseApply;
    }
  }
  return phase;
}
__device__ __noinline__ int finish_update_mixed(SolveScal* s, const SolveScal& cur, int k, const double* acc) {
  return finish_update_mixed_step(s, cur, k, acc);
}

}  // namespace
}  // namespace ig
