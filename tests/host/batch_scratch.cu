// Host driver: batched.cu's prepare_batch with host memory that runs out at the
// k-th allocation, k = 1, 2, ..., and a second call that has memory.  On
// fake_cuda.h.  Prints per k "<failed> <whole>": did the first call fail, and
// does the second leave every table in place.
#include <cstdio>
#include <cstdlib>
#include <new>

#include "../../paper_1506_07577_gb300/csrc/batched.cu"

FakeCuda fake_cuda;

static long allocs_left = -1;   // -1: no limit
#ifndef __CUDA_ARCH__
void* operator new(size_t n) {
  if (allocs_left == 0) throw std::bad_alloc();
  if (allocs_left > 0) --allocs_left;
  void* p = malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }
#endif

namespace ebb {
ebb_status_t set_error(ebb_ctx_s*, ebb_status_t code, const std::string&) { return code; }
ebb_status_t cuda_check(ebb_ctx_s*, cudaError_t e, const char*) { return e == cudaSuccess ? EBB_OK : EBB_ERR_CUDA; }
template <typename T>
cudaError_t launch_tet_map(ebb_rel_s*, int, int, ebb_reduce_t, T, T, const MapIO<T>&, const int*, cudaStream_t) {
  return cudaSuccess;
}
template cudaError_t launch_tet_map<float>(ebb_rel_s*, int, int, ebb_reduce_t, float, float, const MapIO<float>&,
                                           const int*, cudaStream_t);
template cudaError_t launch_tet_map<double>(ebb_rel_s*, int, int, ebb_reduce_t, double, double, const MapIO<double>&,
                                            const int*, cudaStream_t);
bool mixed_cg_ready(ebb_ctx_s*, ebb_rel_s*, const std::vector<int>&, MixedPlan**) { return false; }
void free_mixed_plan(MixedPlan*) {}
cudaError_t launch_mixed_cg(ebb_rel_s*, MixedPlan*, int, float, float, const MixedVectors&, double, double, int,
                            cudaStream_t) {
  return cudaSuccess;
}
const MixedResult* mixed_results(const MixedPlan*) { return nullptr; }
}  // namespace ebb

int main() {
  int n = 0;
#undef cudaGetLastError
  if (cudaGetDeviceCount(&n) == cudaSuccess && n > 0) return 77;   // host pointers must not reach a device
  const int ids[6] = {0, 0, 1, 1, 1, 2};
  for (long k = 0; k < 100; ++k) {
    ebb_ctx_s ctx;
    ebb_rel_s verts, tets;
    verts.size = 6;
    tets.verts = &verts;
    bool failed = false;
    allocs_left = k;
    try {
      failed = ebb::prepare_batch(&ctx, &tets, ids, 1, 3) != EBB_OK;
    } catch (const std::bad_alloc&) {
      failed = true;
    }
    allocs_left = -1;
    bool whole = ebb::prepare_batch(&ctx, &tets, ids, 1, 3) == EBB_OK;
    const ebb::BatchScratch* s = tets.batch;
    whole = whole && s && s->tb.nblocks == 3 && s->tb.blk_mesh && s->tb.mesh_nblk && s->h_sc.size() == 3 &&
            s->vstart.size() == 4;
    if (whole)
      for (int m = 0; m < 3; ++m) whole = whole && s->tb.blk_mesh[m] == m && s->tb.mesh_nblk[m] == 1;
    printf("%d %d\n", failed ? 1 : 0, whole ? 1 : 0);
    ebb::free_batch_scratch(&tets);
    if (!failed) break;
  }
  return 0;
}
