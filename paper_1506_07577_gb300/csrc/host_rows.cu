// The fused map on packed host rows that the GPU reaches itself
// (EBB_MAP_HOST_XYZ with page-locked buffers).
//
// Kernels read the (x, y, z) rows from host memory straight into the 4-float
// fields and write the results straight back: over the host link they are as fast
// as copies (202 GB/s in, 187 out, 155 each at once, measured), need no staging
// pass, and take any set of rows per launch.  So each chunk of tiles gets exactly
// the row blocks it is the first to touch, and hands back those it is the last to
// touch, whatever the vertex order; with copies of row ranges, a chunk waited for
// every row up to its highest, and most rows came back after the last chunk.  A
// chunk is three launches and two events; each further call of the copying form
// was 1.5 us of host time, 110 us in all, more than small maps take.
#include <algorithm>
#include <vector>

#include "async_copy.cuh"
#include "ebb_internal.h"

namespace ebb {

// Row blocks in the order of the chunks that first (in) and last (out) touch them.
struct HostRows {
  unsigned gen = ~0u;
  int K = 0, nblocks = 0;
  std::vector<int> tile_off, in_off, out_off;   // K + 1 each
  int* list = nullptr;                          // in: nblocks, out: nblocks
  cudaStream_t s_in = nullptr, s_out = nullptr;
  cudaEvent_t ev_start = nullptr, ev_end = nullptr;
  cudaEvent_t ev_in[HostPlan::kChunks] = {}, ev_map[HostPlan::kChunks] = {};
};

namespace {

constexpr int kRowBlock = 256;   // rows
// Few threads and registers: a block fits beside the map's CTAs on every SM, one for
// each direction.
constexpr int kRowThreads = 64;

// Chunks a map of so many tiles is cut into.  Measured per call, us, 1 / 2 / 6 chunks:
// 68 tiles 34 / 43 / 71, 4,320 tiles 80 / 72 / 97, 14,580 tiles 182 / 150 / 152, 34,560
// tiles 375 / 288 / 270.  The copying form: 105, 132, 211 and 361.
int host_rows_chunks(int ntiles) { return ntiles < 5000 ? 1 : (ntiles < 20000 ? 2 : HostPlan::kChunks); }

// First and last chunk that touches each row block; tet t is of chunk c when
// bound[c] <= t < bound[c + 1].
struct ChunkBounds {
  int K, bound[HostPlan::kChunks + 1];
};
__global__ void block_chunks_kernel(int nt, const int4* __restrict__ keys, ChunkBounds b, int* first, int* last) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nt) return;
  int c = 0;
  while (c + 1 < b.K && t >= b.bound[c + 1]) ++c;
  const int4 k = keys[t];
  const int v[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int r = v[a] / kRowBlock;
    if (first[r] > c) atomicMin(first + r, c);
    if (last[r] < c) atomicMax(last + r, c);
  }
}

// Packed host rows of the listed blocks into 4-float elements, one or two fields.
// The rows travel by asynchronous copies into shared memory, a block ahead: the
// link needs about 1 MB in flight, which so few threads' registers cannot hold
// (with loads, both directions at once ran at 100 GB/s each).  A16: all host rows
// start on 16-byte bounds (blocks are 3,072 bytes), else copies of 4 bytes.
template <bool A16>
__device__ __forceinline__ void fetch_rows(float* dst, const float* __restrict__ src, int n) {
  if constexpr (A16) {
    int i = 4 * threadIdx.x;
    for (; i + 4 <= n; i += 4 * kRowThreads) cp_async_16(dst + i, src + i);
    for (i = (n & ~3) + threadIdx.x; i < n; i += kRowThreads) cp_async_elem(dst + i, src + i);
  } else {
    for (int i = threadIdx.x; i < n; i += kRowThreads) cp_async_elem(dst + i, src + i);
  }
}

template <bool A16>
__global__ void __launch_bounds__(kRowThreads, 32)
rows_in_kernel(const int* __restrict__ list, int n, int nv, const float* __restrict__ ha, const float* __restrict__ hb,
               float4* __restrict__ da, float4* __restrict__ db) {
  __shared__ __align__(16) float s[2][2][3 * kRowBlock];
  auto fetch = [&](int b, int stage) {
    if (b < n) {
      const int r0 = list[b] * kRowBlock, m = 3 * min(kRowBlock, nv - r0);
      fetch_rows<A16>(s[stage][0], ha + 3 * (size_t)r0, m);
      if (hb != nullptr) fetch_rows<A16>(s[stage][1], hb + 3 * (size_t)r0, m);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(blockIdx.x, 0);
  int stage = 0;
  for (int b = blockIdx.x; b < n; b += gridDim.x, stage ^= 1) {
    fetch(b + gridDim.x, stage ^ 1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const int r0 = list[b] * kRowBlock, rows = min(kRowBlock, nv - r0);
    for (int f = 0; f < (hb != nullptr ? 2 : 1); ++f) {
      const float* x = s[stage][f];
      float4* dst = (f ? db : da) + r0;
      for (int r = threadIdx.x; r < rows; r += kRowThreads)
        dst[r] = make_float4(x[3 * r], x[3 * r + 1], x[3 * r + 2], 0.f);
    }
    __syncthreads();
  }
}

// And back.
template <bool A16>
__global__ void __launch_bounds__(kRowThreads, 32)
rows_out_kernel(const int* __restrict__ list, int n, int nv, const float4* __restrict__ da,
                const float4* __restrict__ db, float* __restrict__ ha, float* __restrict__ hb) {
  __shared__ __align__(16) float s[3 * kRowBlock];
  for (int b = blockIdx.x; b < n; b += gridDim.x) {
    const int r0 = list[b] * kRowBlock, rows = min(kRowBlock, nv - r0);
    for (int f = 0; f < 2; ++f) {
      const float4* src = (f ? db : da) + r0;
      float* dst = (f ? hb : ha) + 3 * (size_t)r0;
#pragma unroll
      for (int k = 0; k < kRowBlock / kRowThreads; ++k) {
        const int r = threadIdx.x + kRowThreads * k;
        const float4 q = r < rows ? src[r] : make_float4(0.f, 0.f, 0.f, 0.f);
        s[3 * r] = q.x;
        s[3 * r + 1] = q.y;
        s[3 * r + 2] = q.z;
      }
      __syncthreads();
      const int m = 3 * rows;
      if constexpr (A16) {
        for (int i = 4 * threadIdx.x; i + 4 <= m; i += 4 * kRowThreads)
          *reinterpret_cast<float4*>(dst + i) = *reinterpret_cast<const float4*>(s + i);
        for (int i = (m & ~3) + threadIdx.x; i < m; i += kRowThreads) dst[i] = s[i];
      } else {
        for (int i = threadIdx.x; i < m; i += kRowThreads) dst[i] = s[i];
      }
      __syncthreads();
    }
  }
}

int row_grid(int n) { return std::min(n, 152); }

ebb_status_t host_rows_plan(ebb_ctx_s* ctx, ebb_rel_s* tets, HostRows** out) {
  HostRows* p = tets->hrows;
  if (p && p->gen == tets->layout_gen) {
    *out = p;
    return EBB_OK;
  }
  cudaError_t e = cudaSuccess;
  if (!p) {
    p = new HostRows();
    tets->hrows = p;
    // the map's split of L1 and shared memory, or an SM that runs maps takes no block
    // of these kernels
    const void* kernels[4] = {(const void*)rows_in_kernel<true>, (const void*)rows_in_kernel<false>,
                              (const void*)rows_out_kernel<true>, (const void*)rows_out_kernel<false>};
    for (const void* k : kernels)
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p->s_in, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p->s_out, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->ev_start, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->ev_end, cudaEventDisableTiming);
    for (int c = 0; c < HostPlan::kChunks && e == cudaSuccess; ++c) {
      e = cudaEventCreateWithFlags(&p->ev_in[c], cudaEventDisableTiming);
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->ev_map[c], cudaEventDisableTiming);
    }
    if (e != cudaSuccess) {
      free_host_rows(tets);
      return cuda_check(ctx, e, "host-map streams");
    }
  }
  p->gen = ~0u;
  cudaFree(p->list);
  p->list = nullptr;
  const Tiles& tl = tets->tiles;
  const int nt = (int)tets->size, nv = (int)tets->verts->size;
  const int nb = (nv + kRowBlock - 1) / kRowBlock;
  p->nblocks = nb;
  p->K = std::min(host_rows_chunks(tl.ntiles), tl.ntiles);
  p->tile_off.assign(p->K + 1, 0);
  ChunkBounds b;
  b.K = p->K;
  b.bound[0] = 0;
  cudaStream_t st = ctx->stream;
  for (int c = 1; c <= p->K && e == cudaSuccess; ++c) {
    p->tile_off[c] = chunk_first_tile(c, tl.ntiles, p->K);
    b.bound[c] = nt;
    if (c < p->K) {
      int4 h;
      e = cudaMemcpyAsync(&h, tl.blob32 + (size_t)p->tile_off[c] * tl.L32.bytes, sizeof h, cudaMemcpyDeviceToHost, st);
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      if (e == cudaSuccess) b.bound[c] = h.z;
    }
  }
  std::vector<int> fl((size_t)2 * nb);
  // blocks nothing touches go in first and out last
  if (e == cudaSuccess) e = cudaMalloc(&p->list, (size_t)2 * nb * sizeof(int));
  if (e == cudaErrorMemoryAllocation) {
    p->list = nullptr;
    cudaGetLastError();
    return set_error(ctx, EBB_ERR_NOMEM, "device allocation for the host-map row lists failed");
  }
  std::fill(fl.begin(), fl.begin() + nb, p->K);
  std::fill(fl.begin() + nb, fl.end(), -1);
  if (e == cudaSuccess) e = cudaMemcpyAsync(p->list, fl.data(), fl.size() * sizeof(int), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    block_chunks_kernel<<<(nt + 255) / 256, 256, 0, st>>>(nt, tets->keys, b, p->list, p->list + nb);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(fl.data(), p->list, fl.size() * sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) {
    std::vector<int> list;
    list.reserve((size_t)2 * nb);
    p->in_off.assign(p->K + 1, 0);
    p->out_off.assign(p->K + 1, 0);
    for (int c = 0; c < p->K; ++c) {
      for (int r = 0; r < nb; ++r)
        if (fl[r] == c || (c == 0 && fl[r] == p->K)) list.push_back(r);
      p->in_off[c + 1] = (int)list.size();
    }
    for (int c = 0; c < p->K; ++c) {
      for (int r = 0; r < nb; ++r)
        if (fl[nb + r] == c || (c == p->K - 1 && fl[nb + r] < 0)) list.push_back(r);
      p->out_off[c + 1] = (int)list.size() - nb;
    }
    e = cudaMemcpyAsync(p->list, list.data(), list.size() * sizeof(int), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  if (e != cudaSuccess) return cuda_check(ctx, e, "host-map row lists");
  p->gen = tets->layout_gen;
  *out = p;
  return EBB_OK;
}

// The device's address of `bytes` of host memory that it reaches throughout; null if
// it does not.
float* device_address(const void* h, size_t bytes) {
  cudaPointerAttributes a, z;
  if (cudaPointerGetAttributes(&a, h) != cudaSuccess ||
      cudaPointerGetAttributes(&z, static_cast<const char*>(h) + bytes - 1) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  if (a.type != cudaMemoryTypeHost || z.type != cudaMemoryTypeHost || a.devicePointer == nullptr ||
      static_cast<char*>(z.devicePointer) - static_cast<char*>(a.devicePointer) != (ptrdiff_t)(bytes - 1) ||
      (reinterpret_cast<uintptr_t>(a.devicePointer) & 3u) != 0)
    return nullptr;
  return static_cast<float*>(a.devicePointer);
}

}  // namespace

void free_host_rows(ebb_rel_s* tets) {
  HostRows* p = tets->hrows;
  if (!p) return;
  cudaFree(p->list);
  for (int c = 0; c < HostPlan::kChunks; ++c) {
    if (p->ev_in[c]) cudaEventDestroy(p->ev_in[c]);
    if (p->ev_map[c]) cudaEventDestroy(p->ev_map[c]);
  }
  if (p->ev_start) cudaEventDestroy(p->ev_start);
  if (p->ev_end) cudaEventDestroy(p->ev_end);
  if (p->s_in) cudaStreamDestroy(p->s_in);
  if (p->s_out) cudaStreamDestroy(p->s_out);
  delete p;
  tets->hrows = nullptr;
}

ebb_status_t host_map_rows(ebb_ctx_s* ctx, ebb_rel_s* tets, void* const* dev, bool same_input, const void* u_host,
                           const void* w_host, void* f_host, void* Kw_host, const ebb_map_opts_t* opts, bool* done) {
  *done = false;
  // On large meshes in the library's own vertex order, copies of row ranges overlap
  // the map fully and run at the copy engines' rate (128^3 mesh 515 us, 543 here; 96^3
  // 305 and 270).
  if (tets->vown >= 0 && tets->tiles.ntiles >= 50000) return EBB_OK;
  const int nv = (int)tets->verts->size;
  const size_t bytes = 12 * (size_t)nv;
  const float* hu = device_address(u_host, bytes);
  const float* hw = hu ? device_address(w_host, bytes) : nullptr;
  float* hf = hw ? device_address(f_host, bytes) : nullptr;
  float* hk = hf ? device_address(Kw_host, bytes) : nullptr;
  if (!hk) return EBB_OK;
  HostRows* P = nullptr;
  const ebb_status_t s = host_rows_plan(ctx, tets, &P);
  if (s) return s;
  *done = true;
  const bool a16 = ((reinterpret_cast<uintptr_t>(hu) | reinterpret_cast<uintptr_t>(hw) |
                     reinterpret_cast<uintptr_t>(hf) | reinterpret_cast<uintptr_t>(hk)) & 15u) == 0;
  cudaStream_t st = ctx->stream;
  const bool cut = P->K > 1;   // one chunk: everything in order on the map's stream
  cudaStream_t s_in = cut ? P->s_in : st, s_out = cut ? P->s_out : st;
  cudaError_t e = cudaSuccess;
  if (cut) {
    e = cudaEventRecord(P->ev_start, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s_in, P->ev_start, 0);
  }
  MapIO<float> io;
  io.u = (const float*)dev[0];
  io.w = (const float*)dev[1];
  io.f = (float*)dev[2];
  io.Kw = (float*)dev[3];
  io.aos = true;
  for (int c = 0; c < P->K && e == cudaSuccess; ++c) {
    const int i0 = P->in_off[c], ni = P->in_off[c + 1] - i0, o0 = P->out_off[c], no = P->out_off[c + 1] - o0;
    if (ni > 0) {
      auto* k = a16 ? rows_in_kernel<true> : rows_in_kernel<false>;
      k<<<row_grid(ni), kRowThreads, 0, s_in>>>(P->list + i0, ni, nv, hu, same_input ? nullptr : hw, (float4*)dev[0],
                                                (float4*)dev[1]);
      e = cudaGetLastError();
    }
    if (c == 0 && e == cudaSuccess && (opts->flags & EBB_MAP_ZERO_OUT))
      e = zero_fields(dev + 2, 2, 16 * (size_t)nv, st);
    if (cut) {
      if (e == cudaSuccess) e = cudaEventRecord(P->ev_in[c], s_in);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(st, P->ev_in[c], 0);
    }
    io.tile_begin = P->tile_off[c];
    io.tile_end = P->tile_off[c + 1];
    if (e == cudaSuccess)
      e = launch_tet_map<float>(tets, opts->model, OP_FORCE | OP_KV, EBB_REDUCE_TILED, (float)opts->mu,
                                (float)opts->lambda, io, nullptr, st);
    if (cut) {
      if (e == cudaSuccess) e = cudaEventRecord(P->ev_map[c], st);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(s_out, P->ev_map[c], 0);
    }
    if (no > 0 && e == cudaSuccess) {
      auto* k = a16 ? rows_out_kernel<true> : rows_out_kernel<false>;
      k<<<row_grid(no), kRowThreads, 0, s_out>>>(P->list + P->nblocks + o0, no, nv, (const float4*)dev[2],
                                                 (const float4*)dev[3], hf, hk);
      e = cudaGetLastError();
    }
  }
  if (cut) {
    if (e == cudaSuccess) e = cudaEventRecord(P->ev_end, s_out);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, P->ev_end, 0);
  }
  return cuda_check(ctx, e, "host-buffer map");
}

}  // namespace ebb
