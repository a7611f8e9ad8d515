// Device parts of the PCG loop shared by the kernels that end an iteration or record vectors.
#pragma once
#include <cuda_runtime.h>

#include "loop.h"
#include "vecops.h"

namespace dd {

// the history slot of the current iteration, or null
__device__ __forceinline__ double* record_slot(const RecDst& r, int64_t n) {
  if (!r.dst) return nullptr;
  const int its = r.ctl->its;
  if (r.inclusive ? its > r.limit : its >= r.limit) return nullptr;
  return r.dst + (int64_t)its * n;
}

// end of one iteration (one thread): counts it, records alpha and applies the stopping test
__device__ __forceinline__ void loop_check(LoopCtl* ctl, const double* sc, double* alphas,
                                           cudaGraphConditionalHandle h, int in_graph) {
  const int its = ctl->its + 1;
  ctl->its = its;
  if (its - 1 < ctl->maxit) alphas[its - 1] = sc[SC_ALPHA];
  ctl->nalpha = its;
  int go = 1;
  if (sc[SC_FLAG] != 0.0) {
    ctl->status = LOOP_BREAKDOWN;
    go = 0;
  } else {
    const double rel = sqrt(sc[SC_RR]) / ctl->ref;
    ctl->rel = rel;
    if (!isfinite(rel)) {
      ctl->status = LOOP_BREAKDOWN;
      go = 0;
    } else if (rel < ctl->rtol) {
      go = 0;
    } else if (its >= ctl->maxit) {
      ctl->status = LOOP_NOT_CONVERGED;
      go = 0;
    }
  }
  ctl->go = go;
  if (in_graph) cudaGraphSetConditional(h, (unsigned)go);
}

}  // namespace dd
