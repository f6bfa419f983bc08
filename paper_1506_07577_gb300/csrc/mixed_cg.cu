// PCG of the mixed-precision implicit step in one cooperative launch: FP32
// matrix-free K p by the tiled map, FP64 vectors (Sections 7.2 and 7.3), for one
// mesh or for many independent ones.
//
// The solve as one map launch and one to three vector launches per iteration
// spent as long on the vectors as on the map, and each waited for the other
// although they use different units: the map issues FP32 and shared-memory
// instructions, the vectors are bound by GB300's FP64 pipe (one instruction per 19
// cycles and SM).  Here an SM runs one block of five tile walkers (the map's CTAs,
// side by side) and kAuxWarps more warps; per iteration
//   map      acc += K p by the walkers; beside it the other warps finish the
//            previous iteration's y += alpha p, which nothing waits for  | (a)
//   A        q = M p + dt^2 acc, p.q                                      | alpha
//   B        r -= alpha q, z = r / diag A, r.z, r.r                       | beta
//   C        p' = z + beta p, its FP32 copy, acc = 0                      | (b)
// with a grid barrier at each |, four to an iteration; p and p' alternate between two
// arrays, so that y can be late.  The arithmetic is the separate kernels'.
//
// A batch is solved as two groups of meshes by two such kernels at once, each with
// two walkers per SM: nothing ties them together, so that one group's vectors and
// the other's maps share the SM.
//
// A block owns consecutive vertices, cut where a mesh ends into segments; a mesh's
// dot products are the sums over its segments in order, formed alike in every
// block that has one of them, so no scalars are exchanged.
//
// Measured, whole steps against one map and one to three vector launches per
// iteration: 64^3 mesh (1.31 M tets) 2775 -> 2453 us; batch of 256 meshes (3.4 M
// tets) 2677 -> 2539 us as one group, 2164 us as two.  Four walkers instead of
// five: 2652 us on the 64^3 mesh.  An iteration there is 61,000 to 66,000 cycles
// of map and 35,000 of FP64 vectors; a barrier takes 3,000.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "fp64_lean.cuh"
#include "grid_barrier.cuh"
#include "mixed_cg.h"
#include "tile_map.cuh"

namespace ebb {

struct MixedSeg {
  int mesh, v0, v1;
  int part0, npart;    // the mesh's segments
  int lead;            // the mesh's first segment: counts it and reports its result
};

// A segment's scalars, kept by its block.
struct MixedCg {
  double rz, alpha, beta, tol, rr, bb;
  int active, late;    // iterating; y += alpha p still to come
  int iter, status;
};

// The part of a plan that one kernel solves.
struct MixedGroup {
  int v0 = 0, v1 = 0, tile0 = 0, tile1 = 0;
  int nseg = 0;
  MixedSeg* seg = nullptr;
  int* first = nullptr;       // grid + 1: first segment of each block
  MixedCg* cg = nullptr;
  double* part = nullptr;     // 2 values x nseg, and 1 x nseg
  unsigned* ctl = nullptr;    // [0] barrier counter, [1] meshes that iterate
};

struct MixedPlan {
  int ngroup = 0, grid = 0;
  unsigned layout_gen = 0;    // the tiles the groups were cut from
  MixedGroup group[2];
  MixedResult* res = nullptr;
  void* slab = nullptr;
  cudaStream_t side = nullptr;   // the second group's stream
  cudaEvent_t fork = nullptr, join = nullptr;
};

namespace {

// A block's shape: walkers, further warps, and how many threads run the vector
// passes (a value's partials fit a walker's output rows).
template <int WALKERS, int AUX, int VEC>
struct Shape {
  static constexpr int walkers = WALKERS, aux = AUX, vec = VEC;
  static constexpr int map_threads = WALKERS * kTileThreads, threads = map_threads + 32 * AUX;
};
using One = Shape<5, 3, 768>;    // one block per SM
using Half = Shape<2, 4, 448>;   // two blocks per SM, one of each group
constexpr int kSegBatch = 6;    // segments whose sums are formed together
constexpr int kCached = 4;      // segments of a block kept in shared memory
using Tile = TileSmem<float, OP_KV>;
static_assert(Tile::OB * Tile::out_elems * sizeof(float) >= One::vec * sizeof(double), "room for a value's partials");

struct MixedArgs {
  int nv, ntiles, v_lo;
  unsigned v_span;
  const unsigned char* blobs;
  BlobLayout L;
  const int* perm;
  float mu0, lam0;
  int* err;
  MixedVectors v;
  const MixedSeg* seg;
  const int* first;
  int nseg;
  MixedCg* cg;
  double* part;
  MixedResult* res;
  unsigned* ctl;
  double dt, rtol;
  int max_iters;
  size_t walker_smem;
};

template <typename PT>
__device__ __forceinline__ bool pin_at(const PT* pin, int v) {
  return pin != nullptr && pin[v] != 0;
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

struct MixedShared {
  double* v[2];   // a value per vector thread each: the first two walkers' output rows, idle between maps
  double w[2][4];
  double tot[kSegBatch][2];
  MixedCg cg[kCached];
  MixedSeg seg[kCached];
  int ok, bad;
};

// Partial sums of NV values of segment `s` (block-uniform) from every thread.
template <int VEC, int NV>
__device__ __forceinline__ void segment_partial(MixedShared& sh, const double (&x)[NV], double* part, int nseg, int s) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < VEC) {
#pragma unroll
    for (int j = 0; j < NV; ++j) sh.v[j][tid] = x[j];
  }
  __syncthreads();
  if (warp < 4 * NV) {
    const int j = warp >> 2, g = warp & 3, at = g * 32 + lane;
    double t = sh.v[j][at];
#pragma unroll
    for (int i = 1; i < (VEC + 127) / 128; ++i)
      if (VEC % 128 == 0 || at + 128 * i < VEC) t += sh.v[j][at + 128 * i];
    t = warp_sum(t);
    if (lane == 0) sh.w[j][g] = t;
  }
  __syncthreads();
  if (tid < NV) part[(size_t)tid * nseg + s] = (sh.w[tid][0] + sh.w[tid][1]) + (sh.w[tid][2] + sh.w[tid][3]);
}

// Barrier: every thread of the block gets past it when the whole grid has arrived.
__device__ __forceinline__ bool grid_join(MixedShared& sh, const unsigned* bar, unsigned round) {
  if (threadIdx.x == 0) sh.ok = wait_acquire(bar, round * gridDim.x);
  __syncthreads();
  return sh.ok != 0;
}

// Sums over the meshes of this block's n_seg segments: for each, `fin(cg, seg,
// totals)` runs in one thread.
template <int NV, typename Fin>
__device__ __forceinline__ void segment_totals(MixedShared& sh, const double* part, int nseg, const MixedSeg* seg,
                                               MixedCg* cg, int n_seg, Fin fin) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int b = 0; b < n_seg; b += kSegBatch) {
    const int s = b + warp / 2, j = warp % 2;
    const bool mine = warp < 2 * kSegBatch && s < n_seg;
    if (mine && j < NV) {
      const int p0 = seg[s].part0, n = seg[s].npart;
      const double* x = part + (size_t)j * nseg + p0;
      double t = 0.0;
      for (int i = lane; i < n; i += 256) {
        double y[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) y[k] = i + 32 * k < n ? __ldcg(x + i + 32 * k) : 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (i - lane + 32 * k < n) t += y[k];
      }
      t = warp_sum(t);
      if (lane == 0) sh.tot[s - b][j] = t;
    }
    __syncthreads();
    if (mine && threadIdx.x == 64 * (s - b)) fin(cg[s], seg[s], sh.tot[s - b]);
    __syncthreads();
  }
}

template <typename SH, int MODEL, typename PT>
__global__ void __launch_bounds__(SH::threads, SH::threads > 512 ? 1 : 2) mixed_cg_kernel(MixedArgs a) {
  constexpr int kWalkers = SH::walkers, kVecThreads = SH::vec, kMixThreads = SH::threads;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ MixedShared sh;
  const int tid = threadIdx.x;
  const int g = tid / kTileThreads;   // walker, or kWalkers for the other warps
  const bool maps = g < kWalkers;
  const int nwalk = (int)gridDim.x * kWalkers, walker = (int)blockIdx.x * kWalkers + (maps ? g : 0);
  const int n_my = maps && walker < a.ntiles ? (a.ntiles - walker + nwalk - 1) / nwalk : 0;
  const TileView<float, OP_KV> V = tile_view<float, OP_KV>(smem + (maps ? g : 0) * a.walker_smem, a.L,
                                                           tid - g * kTileThreads, walker, nwalk, 1 + g);
  if (maps) tile_init(V);
  if (tid == 0) sh.bad = 0;
  if (tid < 2) sh.v[tid] = reinterpret_cast<double*>(smem + tid * a.walker_smem + Tile::out_off(a.L));
  const PT* pin = static_cast<const PT*>(a.v.pin);
  // this block's segments and their scalars: in shared memory when they are few
  const int nv = a.nv, s0 = a.first[blockIdx.x], n_seg = a.first[blockIdx.x + 1] - s0;
  const bool cached = n_seg <= kCached;
  if (cached && tid < n_seg) sh.seg[tid] = a.seg[s0 + tid];
  const MixedSeg* const seg = cached ? sh.seg : a.seg + s0;
  MixedCg* const cg = cached ? sh.cg : a.cg + s0;
  double *const part2 = a.part, *const part1 = a.part + 2 * (size_t)a.nseg;
  const int vt = tid < kVecThreads ? tid : 0x40000000;   // the other warps run no vector passes
  const double dt2 = a.dt * a.dt;
  const float dt2f = (float)dt2;
  unsigned* bar = a.ctl;
  unsigned round = 0;
  MapIO<float> io;
  io.u = a.v.u;
  io.w = a.v.pe;
  io.Kw = a.v.acc;
  io.aos = true;
  io.v_lo = a.v_lo;
  io.v_span = a.v_span;
  __syncthreads();

  // r.z and r.r of the start
  for (int s = 0; s < n_seg; ++s) {
    double x[2] = {0.0, 0.0};
    const int v1 = seg[s].v1;
    for (int v = seg[s].v0 + vt; v < v1; v += kVecThreads)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double r = a.v.r[(size_t)k * nv + v];
        x[0] = fma(r, a.v.p[(size_t)k * nv + v], x[0]);
        x[1] = fma(r, r, x[1]);
      }
    segment_partial<kVecThreads, 2>(sh, x, part2, a.nseg, s0 + s);
  }
  grid_arrive(bar, round);
  bool ok = grid_join(sh, bar, round);
  if (ok) {
    segment_totals<2>(sh, part2, a.nseg, seg, cg, n_seg, [&](MixedCg& cg, const MixedSeg& seg, const double* t) {
      cg.rz = t[0];
      cg.rr = cg.bb = t[1];
      cg.alpha = cg.beta = 0.0;
      cg.tol = a.rtol * sqrt(t[1]);
      cg.active = a.max_iters > 0 && sqrt(t[1]) > cg.tol;
      cg.late = cg.iter = 0;
      cg.status = EBB_OK;
      if (cg.active && seg.lead) atomicAdd(a.ctl + 1, 1u);
    });
    grid_arrive(bar, round);
    ok = grid_join(sh, bar, round);
  }
  // y += alpha p of the segments' last iteration, p in `ps`; threads `me` of `n`
  auto finish_y = [&](const double* ps, int me, int n) {
    for (int s = 0; s < n_seg; ++s) {
      if (!cg[s].late) continue;
      const double alpha = cg[s].alpha;
      const int v1 = seg[s].v1;
      // (few threads: several vertices' loads in flight)
      constexpr int U = 3;
      for (int v = seg[s].v0 + me; v < v1; v += U * n) {
        double x[U][3], y[U][3];
        bool on[U];
#pragma unroll
        for (int h = 0; h < U; ++h) {
          const int w = v + h * n;
          on[h] = w < v1 && !pin_at(pin, w);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const size_t i = (size_t)k * nv + (w < v1 ? w : v);
            x[h][k] = ps[i];
            y[h][k] = a.v.y[i];
          }
        }
#pragma unroll
        for (int h = 0; h < U; ++h)
          if (on[h]) {
#pragma unroll
            for (int k = 0; k < 3; ++k) a.v.y[(size_t)k * nv + v + h * n] = fma(alpha, x[h][k], y[h][k]);
          }
      }
    }
  };

  double *p = a.v.p, *pn = a.v.p2;   // this iteration's direction, the next one's
  int it = 0;
  while (ok) {
    // everyone sees the same count: it changes only between (beta) and (b)
    if (__ldcg(a.ctl + 1) == 0u) break;
    if (maps) {
      if (n_my > 0 && !tile_map_pass<float, MODEL, OP_KV, true, false>(V, n_my, it * n_my, nv, a.blobs, a.L, a.perm,
                                                                       a.mu0, a.lam0, io, a.err, -1, kWaitCycles))
        sh.bad = 1;
    } else if (it > 0) {
      finish_y(pn, tid - SH::map_threads, 32 * SH::aux);
    }
    grid_arrive(bar, round);
    ok = grid_join(sh, bar, round) && sh.bad == 0;
    if (!ok) break;
    // A
    for (int s = 0; s < n_seg; ++s) {
      if (!cg[s].active) continue;
      double x[1] = {0.0};
      const int v1 = seg[s].v1;
#pragma unroll 2
      for (int v = seg[s].v0 + vt; v < v1; v += kVecThreads) {
        if (pin_at(pin, v)) continue;
        const double m = a.v.mass[v];
        const float4 k4 = __ldcg(reinterpret_cast<const float4*>(a.v.acc) + v);
        const float kv[3] = {k4.x, k4.y, k4.z};
        double pv[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) pv[k] = p[(size_t)k * nv + v];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const double q = fma(m, pv[k], widen(dt2f * kv[k]));
          a.v.q[(size_t)k * nv + v] = q;
          x[0] = fma(pv[k], q, x[0]);
        }
      }
      segment_partial<kVecThreads, 1>(sh, x, part1, a.nseg, s0 + s);
    }
    grid_arrive(bar, round);
    ok = grid_join(sh, bar, round);
    if (!ok) break;
    segment_totals<1>(sh, part1, a.nseg, seg, cg, n_seg, [&](MixedCg& cg, const MixedSeg& seg, const double* t) {
      cg.late = 0;
      if (!cg.active) return;
      if (t[0] > 0.0) {
        cg.alpha = cg.rz / t[0];
        cg.late = 1;
      } else {
        cg.alpha = 0.0;
        cg.status = EBB_ERR_CG_BREAKDOWN;
        cg.active = 0;
        if (seg.lead) atomicSub(a.ctl + 1, 1u);
      }
    });
    // B
    for (int s = 0; s < n_seg; ++s) {
      if (!cg[s].active) continue;
      const double alpha = cg[s].alpha;
      double x[2] = {0.0, 0.0};
      const int v1 = seg[s].v1;
#pragma unroll 2
      for (int v = seg[s].v0 + vt; v < v1; v += kVecThreads) {
        if (pin_at(pin, v)) continue;
        double qv[3], rv[3], dv[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const size_t i = (size_t)k * nv + v;
          qv[k] = a.v.q[i];
          rv[k] = a.v.r[i];
          dv[k] = a.v.dinv[i];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const size_t i = (size_t)k * nv + v;
          const double ri = fma(-alpha, qv[k], rv[k]);
          const double zi = ri * dv[k];
          a.v.r[i] = ri;
          a.v.q[i] = zi;
          x[0] = fma(ri, zi, x[0]);
          x[1] = fma(ri, ri, x[1]);
        }
      }
      segment_partial<kVecThreads, 2>(sh, x, part2, a.nseg, s0 + s);
    }
    grid_arrive(bar, round);
    ok = grid_join(sh, bar, round);
    if (!ok) break;
    segment_totals<2>(sh, part2, a.nseg, seg, cg, n_seg, [&](MixedCg& cg, const MixedSeg& seg, const double* t) {
      if (!cg.active) return;
      cg.beta = t[0] / cg.rz;
      cg.rz = t[0];
      cg.rr = t[1];
      ++cg.iter;
      cg.active = cg.iter < a.max_iters && sqrt(t[1]) > cg.tol;
      if (!cg.active && seg.lead) atomicSub(a.ctl + 1, 1u);
    });
    // C
    for (int s = 0; s < n_seg; ++s) {
      const bool go = cg[s].active != 0;
      const double beta = cg[s].beta;
      const int v1 = seg[s].v1;
#pragma unroll 2
      for (int v = seg[s].v0 + vt; v < v1; v += kVecThreads) {
        reinterpret_cast<float4*>(a.v.acc)[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!go) continue;
        const bool fixed = pin_at(pin, v);
        double x[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const size_t i = (size_t)k * nv + v;
          x[k] = fixed ? 0.0 : fma(beta, p[i], a.v.q[i]);
          pn[i] = x[k];
        }
        reinterpret_cast<float4*>(a.v.pe)[v] = make_float4(narrow(x[0]), narrow(x[1]), narrow(x[2]), 0.f);
      }
    }
    double* const t = p;
    p = pn;
    pn = t;
    ++it;
    grid_arrive(bar, round);
    ok = grid_join(sh, bar, round);
  }
  if (ok && it > 0) finish_y(pn, tid, kMixThreads);
  // results, by each mesh's first segment
  for (int s = tid; s < n_seg; s += kMixThreads)
    if (seg[s].lead) {
      MixedResult h;
      h.rr = cg[s].rr;
      h.bb = cg[s].bb;
      h.iter = cg[s].iter;
      h.status = ok ? cg[s].status : EBB_ERR_TIMEOUT;
      a.res[seg[s].mesh] = h;
    }
}

template <typename SH, int MODEL, typename PT>
cudaError_t launch(const MixedArgs& a, int grid, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(SH::threads);
  cfg.dynamicSmemBytes = SH::walkers * a.walker_smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, mixed_cg_kernel<SH, MODEL, PT>, a);
}

size_t walker_bytes(const BlobLayout& L) { return (Tile::bytes(L) + 127) / 128 * 128; }

// Do `want` blocks fit an SM?
template <typename SH, int MODEL, typename PT>
bool resident(size_t walker, int want) {
  int n = 0;
  const size_t smem = SH::walkers * walker;
  auto* k = mixed_cg_kernel<SH, MODEL, PT>;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return false;
  if (cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100) != cudaSuccess) return false;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, SH::threads, smem) == cudaSuccess && n >= want;
}

// Where the tiles of the vertices < v and those of the vertices >= v part: the last
// tile with a tet of the former, the first with a tet of the latter, and whether a tet
// joins both.  Every tet is looked at: the tets lie mesh by mesh only when the same ids
// were the "batch" field of finalize, and a step takes any field.
struct Border {
  int last, first, joined;
};

__global__ void __launch_bounds__(kTileTets)
border_kernel(const int4* __restrict__ keys, const unsigned char* __restrict__ blobs, int blob_bytes, int ntiles, int v,
              Border* out) {
  int last = -1, first = ntiles;
  bool joined = false;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int4 h = *reinterpret_cast<const int4*>(blobs + (size_t)tile * blob_bytes);   // tets, slots, first tet
    if ((int)threadIdx.x >= h.x) continue;
    const int4 k = keys[h.z + threadIdx.x];
    const bool below = min(min(k.x, k.y), min(k.z, k.w)) < v, above = max(max(k.x, k.y), max(k.z, k.w)) >= v;
    if (below) last = tile;
    if (above) first = min(first, tile);
    joined |= below && above;
  }
  last = __reduce_max_sync(0xffffffffu, last);
  first = __reduce_min_sync(0xffffffffu, first);
  joined = __any_sync(0xffffffffu, joined);
  if ((threadIdx.x & 31) != 0) return;
  if (last >= 0) atomicMax(&out->last, last);
  if (first < ntiles) atomicMin(&out->first, first);
  if (joined) out->joined = 1;
}

// That on the host; false when a call fails.
bool find_border(ebb_rel_s* rel, int v, Border* b, cudaStream_t st) {
  const int ntiles = rel->tiles.ntiles;
  *b = Border{-1, ntiles, 0};
  Border* d = nullptr;
  cudaError_t e = cudaMalloc(&d, sizeof(Border));
  if (e == cudaSuccess) e = cudaMemcpyAsync(d, b, sizeof(Border), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    border_kernel<<<std::min(ntiles, 2432), kTileTets, 0, st>>>(rel->keys, rel->tiles.blob32, rel->tiles.L32.bytes,
                                                                ntiles, v, d);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(b, d, sizeof(Border), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(d);
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess;
}

// Segments of the vertices [v0, v1) over `grid` blocks; meshes numbered as in vstart.
void cut_segments(const std::vector<int>& vstart, int v0, int v1, int grid, std::vector<MixedSeg>& seg,
                  std::vector<int>& first) {
  const int n = v1 - v0;
  first.assign(grid + 1, 0);
  std::vector<int> part0;   // first segment of each mesh met, in order
  std::vector<int> meshes;
  int mesh = (int)(std::upper_bound(vstart.begin(), vstart.end(), v0) - vstart.begin()) - 1;
  for (int b = 0; b < grid; ++b) {
    first[b] = (int)seg.size();
    int v = v0 + (int)((long long)b * n / grid);
    const int end = v0 + (int)((long long)(b + 1) * n / grid);
    while (v < end) {
      while (vstart[mesh + 1] <= v) ++mesh;
      const int e = std::min(end, vstart[mesh + 1]);
      MixedSeg s;
      s.mesh = mesh;
      s.v0 = v;
      s.v1 = e;
      s.lead = v == vstart[mesh] ? 1 : 0;
      s.part0 = s.npart = 0;
      if (s.lead) {
        part0.push_back((int)seg.size());
        meshes.push_back(mesh);
      }
      seg.push_back(s);
      v = e;
    }
  }
  first[grid] = (int)seg.size();
  part0.push_back((int)seg.size());
  for (MixedSeg& s : seg) {
    const int k = s.mesh - meshes[0];
    s.part0 = part0[k];
    s.npart = part0[k + 1] - part0[k];
  }
}

}  // namespace

void free_mixed_plan(MixedPlan* plan) {
  if (!plan) return;
  cudaFree(plan->slab);
  if (plan->fork) cudaEventDestroy(plan->fork);
  if (plan->join) cudaEventDestroy(plan->join);
  if (plan->side) cudaStreamDestroy(plan->side);
  delete plan;
}

const MixedResult* mixed_results(const MixedPlan* plan) { return plan->res; }

bool mixed_cg_ready(ebb_ctx_s* ctx, ebb_rel_s* rel, const std::vector<int>& vstart, MixedPlan** out) {
  if (*out && (*out)->layout_gen != rel->layout_gen) {   // tiles cut again
    free_mixed_plan(*out);
    *out = nullptr;
  }
  if (*out) return (*out)->grid > 0;
  MixedPlan* m = new MixedPlan();
  *out = m;   // grid 0: does not apply
  m->layout_gen = rel->layout_gen;
  const int nv = vstart.back(), nmesh = (int)vstart.size() - 1;
  int nsm = 0;
  if (rel->tiles.ntiles == 0 || nv == 0 ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess || nsm < 1) {
    cudaGetLastError();
    return false;
  }
  // A block per SM and group: small meshes too, for whose few vertices and tiles
  // more SMs mean shorter passes.
  const int grid = nsm;
  // Segments are summed one after the other: a batch of very many small meshes is
  // better off with a block per mesh.  Whole steps, one launch and separate ones, of
  // 300, 450, 600 and 1000 meshes of 27 vertices: 222 and 248, 261 and 259, 290 and
  // 278, 462 and 394 us; of 600 and 1000 meshes of 125 vertices: 327 and 344, 520 and
  // 488 us; of 729 vertices: 772 and 879, 1299 and 1372 us.
  if (nmesh > 16 * grid || (nmesh > 3 * grid && nv / nmesh < 512)) return false;
  const size_t walker = walker_bytes(rel->tiles.L32);
  if (!resident<One, EBB_STVK, unsigned char>(walker, 1) || !resident<One, EBB_NEOHOOKEAN, unsigned char>(walker, 1) ||
      !resident<One, EBB_STVK, int>(walker, 1) || !resident<One, EBB_NEOHOOKEAN, int>(walker, 1)) {
    cudaGetLastError();
    return false;
  }
  m->ngroup = 1;
  m->group[0].v1 = nv;
  m->group[0].tile1 = rel->tiles.ntiles;
  // Two groups, cut between meshes nearest the middle vertex.
  if (nmesh > 1 && resident<Half, EBB_STVK, unsigned char>(walker, 2) &&
      resident<Half, EBB_NEOHOOKEAN, unsigned char>(walker, 2)) {
    int cut = 1;
    for (int k = 2; k < nmesh; ++k)
      if (std::abs(2LL * vstart[k] - nv) < std::abs(2LL * vstart[cut] - nv)) cut = k;
    // Each group maps the tiles that hold its tets.  In one order over all meshes (ids
    // bound after finalize) both groups would map nearly every tile, so the tiles may
    // overlap by the one at the border only; and groups that share a tet would read each
    // other's vectors.  Otherwise one group solves them all.
    Border border;
    if (find_border(rel, vstart[cut], &border, ctx->stream) && !border.joined && border.last <= border.first &&
        cudaStreamCreateWithFlags(&m->side, cudaStreamNonBlocking) == cudaSuccess &&
        cudaEventCreateWithFlags(&m->fork, cudaEventDisableTiming) == cudaSuccess &&
        cudaEventCreateWithFlags(&m->join, cudaEventDisableTiming) == cudaSuccess) {
      m->ngroup = 2;
      m->group[0].v1 = m->group[1].v0 = vstart[cut];
      m->group[1].v1 = nv;
      m->group[0].tile1 = border.last + 1;
      m->group[1].tile0 = border.first;
      m->group[1].tile1 = rel->tiles.ntiles;
    }
  }
  cudaGetLastError();
  auto up = [](size_t n) { return (n + 127) / 128 * 128; };
  std::vector<MixedSeg> seg[2];
  std::vector<int> first[2];
  size_t total = up(nmesh * sizeof(MixedResult));
  for (int g = 0; g < m->ngroup; ++g) {
    cut_segments(vstart, m->group[g].v0, m->group[g].v1, grid, seg[g], first[g]);
    const size_t n = seg[g].size();
    m->group[g].nseg = (int)n;
    total += up(n * sizeof(MixedCg)) + up(3 * n * sizeof(double)) + up(n * sizeof(MixedSeg)) +
             up((grid + 1) * sizeof(int)) + 128;
  }
  if (cudaMalloc(&m->slab, total) != cudaSuccess) {
    m->slab = nullptr;
    cudaGetLastError();
    return false;
  }
  char* d = static_cast<char*>(m->slab);
  auto take = [&](size_t n) {
    char* at = d;
    d += up(n);
    return at;
  };
  m->res = reinterpret_cast<MixedResult*>(take(nmesh * sizeof(MixedResult)));
  for (int g = 0; g < m->ngroup; ++g) {
    MixedGroup& q = m->group[g];
    const size_t n = q.nseg;
    q.cg = reinterpret_cast<MixedCg*>(take(n * sizeof(MixedCg)));
    q.part = reinterpret_cast<double*>(take(3 * n * sizeof(double)));
    q.seg = reinterpret_cast<MixedSeg*>(take(n * sizeof(MixedSeg)));
    q.first = reinterpret_cast<int*>(take((grid + 1) * sizeof(int)));
    q.ctl = reinterpret_cast<unsigned*>(take(128));
    // On the context's stream, which the solve's streams follow: a copy from pageable
    // memory may return before it has landed, and none of them waits for the legacy
    // default stream.
    cudaStream_t up_st = ctx->stream;
    cudaError_t e = cudaMemcpyAsync(q.seg, seg[g].data(), n * sizeof(MixedSeg), cudaMemcpyHostToDevice, up_st);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(q.first, first[g].data(), (grid + 1) * sizeof(int), cudaMemcpyHostToDevice, up_st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(up_st);
    if (e != cudaSuccess) {
      cudaGetLastError();
      cudaFree(m->slab);
      m->slab = nullptr;
      return false;
    }
  }
  m->grid = grid;
  return true;
}

cudaError_t launch_mixed_cg(ebb_rel_s* rel, MixedPlan* m, int model, float mu0, float lam0, const MixedVectors& v,
                            double dt, double rtol, int max_iters, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  if (m->ngroup == 2) {
    e = cudaEventRecord(m->fork, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(m->side, m->fork, 0);
  }
  for (int g = 0; g < m->ngroup && e == cudaSuccess; ++g) {
    const MixedGroup& q = m->group[g];
    cudaStream_t gs = g == 0 ? st : m->side;
    e = cudaMemsetAsync(q.ctl, 0, 2 * sizeof(unsigned), gs);
    if (e != cudaSuccess) break;
    MixedArgs a;
    a.nv = (int)rel->verts->size;
    a.ntiles = q.tile1 - q.tile0;
    a.v_lo = q.v0;
    a.v_span = (unsigned)(q.v1 - q.v0);
    a.L = rel->tiles.L32;
    a.blobs = rel->tiles.blob32 + (size_t)q.tile0 * a.L.bytes;
    a.perm = rel->tet_perm;
    a.mu0 = mu0;
    a.lam0 = lam0;
    a.err = rel->ctx->d_err;
    a.v = v;
    a.seg = q.seg;
    a.first = q.first;
    a.nseg = q.nseg;
    a.cg = q.cg;
    a.part = q.part;
    a.res = m->res;
    a.ctl = q.ctl;
    a.dt = dt;
    a.rtol = rtol;
    a.max_iters = max_iters;
    a.walker_smem = walker_bytes(a.L);
    if (m->ngroup == 2)   // batches pin by bytes
      e = model == EBB_STVK ? launch<Half, EBB_STVK, unsigned char>(a, m->grid, gs)
                            : launch<Half, EBB_NEOHOOKEAN, unsigned char>(a, m->grid, gs);
    else if (v.pin_bytes == 4)
      e = model == EBB_STVK ? launch<One, EBB_STVK, int>(a, m->grid, gs)
                            : launch<One, EBB_NEOHOOKEAN, int>(a, m->grid, gs);
    else
      e = model == EBB_STVK ? launch<One, EBB_STVK, unsigned char>(a, m->grid, gs)
                            : launch<One, EBB_NEOHOOKEAN, unsigned char>(a, m->grid, gs);
  }
  if (m->ngroup == 2 && e == cudaSuccess) {
    e = cudaEventRecord(m->join, m->side);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, m->join, 0);
  }
  return e;
}

}  // namespace ebb
