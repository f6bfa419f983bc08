// Host driver: which storage launch_assemble puts K in when allocations fail or
// the stream is being captured.  Linked with edges.cu and row_matrix.cu on
// fake_cuda.h.  Prints one line per step: "<status> <on rows> <in blocks>".
#include <cstdio>

#include "../../paper_1506_07577_gb300/csrc/row_matrix.cuh"

FakeCuda fake_cuda;

namespace ebb {
ebb_status_t set_error(ebb_ctx_s*, ebb_status_t code, const std::string&) { return code; }
ebb_status_t cuda_check(ebb_ctx_s*, cudaError_t e, const char*) { return e == cudaSuccess ? EBB_OK : EBB_ERR_CUDA; }
}  // namespace ebb

int main() {
  int n = 0;
#undef cudaGetLastError
  if (cudaGetDeviceCount(&n) == cudaSuccess && n > 0) return 77;   // host pointers must not reach a device
  cudaGetLastError();
  ebb_ctx_s ctx;
  ebb_rel_s verts, tets;
  verts.ctx = tets.ctx = &ctx;
  verts.size = 40;
  tets.size = 100;
  tets.verts = &verts;
  int dummy[64] = {};
  tets.vindex.off = tets.vindex.ent = tets.vindex.order = dummy;
  tets.edges.row_off = tets.edges.col = dummy;
  tets.edges.nnzb = 60;
  auto show = [&](int p, cudaError_t e) {
    printf("%d %d %d\n", e == cudaSuccess ? 0 : 1, tets.rows && tets.rows->val[p] ? 1 : 0,
           tets.edges.blocks[p] ? 1 : 0);
  };
  auto assemble32 = [&] {
    show(0, ebb::launch_assemble<float>(&tets, EBB_STVK, 1.f, 1.f, ebb::MapIO<float>(), nullptr));
  };
  auto assemble64 = [&] {
    show(1, ebb::launch_assemble<double>(&tets, EBB_STVK, 1.0, 1.0, ebb::MapIO<double>(), nullptr));
  };
  // FP32: no room for the rows' records (28,800 bytes), then room
  fake_cuda.max_alloc = 20000;
  assemble32();
  fake_cuda.max_alloc = ~(size_t)0;
  assemble32();
  fake_cuda.capturing = true;
  assemble32();
  // FP64: first use inside a capture, then outside, then inside again
  assemble64();
  fake_cuda.capturing = false;
  assemble64();
  fake_cuda.capturing = true;
  assemble64();
  return 0;
}
