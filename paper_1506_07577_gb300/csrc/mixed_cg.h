// Mixed-precision PCG solve in one launch (mixed_cg.cu), for one mesh or a batch.
#pragma once

#include <vector>

#include "ebb_internal.h"

namespace ebb {

// Result of one mesh's solve.
struct MixedResult {
  double rr, bb;
  int iter, status;
};

// Vectors of the solve, set up by the caller: r = b, p = z = r / diag(A), y = 0
// (FP64 planes), pe = p and acc = 0 (FP32 4-value elements).  q and p2 are scratch.
struct MixedVectors {
  const float* u;          // displacement, 4-value elements
  const void* pin;
  int pin_bytes;           // 1 or 4
  const double *mass, *dinv;
  double *r, *p, *p2, *y, *q;
  float *pe, *acc;
};

// Can this relation's FP32 solves run so?  `vstart`: first vertex of each mesh and
// the vertex count (nmesh + 1 entries).  Builds the plan (kept in *plan, freed with
// free_mixed_plan) on first use; false when the kernel cannot be resident, memory is
// short or the batch has too many meshes for it.
struct MixedPlan;
bool mixed_cg_ready(ebb_ctx_s* ctx, ebb_rel_s* rel, const std::vector<int>& vstart, MixedPlan** plan);
void free_mixed_plan(MixedPlan* plan);

// Solve, ordered after the work on `st` and before later work there (asynchronous).
// The meshes' results are left on the device, one per mesh.
cudaError_t launch_mixed_cg(ebb_rel_s* rel, MixedPlan* plan, int model, float mu0, float lam0, const MixedVectors& v,
                            double dt, double rtol, int max_iters, cudaStream_t st);
const MixedResult* mixed_results(const MixedPlan* plan);

}  // namespace ebb
