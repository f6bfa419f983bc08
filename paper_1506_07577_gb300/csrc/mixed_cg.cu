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
// with a grid barrier at each |; p and p' alternate between two arrays, so that y
// can be late.  At (b) the walkers' first tile copies are already on their way:
// the producers wait there themselves.  The arithmetic is the separate kernels'.
//
// A block owns consecutive vertices, cut where a mesh ends into segments; a mesh's
// dot products are the sums over its segments in order, formed alike in every
// block that has one of them, so no scalars are exchanged.
#include <algorithm>
#include <cmath>

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

struct MixedPlan {
  int nmesh = 0, nseg = 0, grid = 0;
  std::vector<int> vstart;
  void* slab = nullptr;
  MixedSeg* seg = nullptr;
  int* first = nullptr;       // grid + 1: first segment of each block
  MixedCg* cg = nullptr;
  double* part = nullptr;     // 2 values x nseg, and 1 x nseg
  MixedResult* res = nullptr;
  unsigned* ctl = nullptr;    // [0] barrier counter, [1] meshes that iterate
};

namespace {

constexpr int kWalkers = 5;
constexpr int kAuxWarps = 3;
constexpr int kMapThreadsAll = kWalkers * kTileThreads;
constexpr int kMixThreads = kMapThreadsAll + 32 * kAuxWarps;
constexpr int kVecThreads = 768;                       // run the vector passes
static_assert(kVecThreads <= kMapThreadsAll, "the vector passes' threads are walkers'");
constexpr int kSegBatch = 8;    // segments whose sums are formed together
constexpr int kCached = 4;      // segments of a block kept in shared memory
using Tile = TileSmem<float, OP_KV>;
static_assert(Tile::OB * Tile::out_elems * sizeof(float) >= kVecThreads * sizeof(double), "room for a value's partials");

struct MixedArgs {
  int nv, ntiles;
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

// An FP32 value in FP64, exactly, by integer instructions: a conversion costs as
// much of the FP64 pipe as a multiplication.  Zero and normal values; the others
// take the conversion.
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
  if (m == 0u) return __hiloint2double((int)u, 0);
  return (double)x;
}

// The FP32 value of x (round to nearest even), likewise: a conversion costs the
// FP64 pipe as much.  Results in FP32's normal range and zero; the others
// take the conversion.
__device__ __forceinline__ float narrow(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned m = hi & 0x7fffffffu;
  if (m - 0x38100000u < 0x0fd00000u) {   // 2^-126 <= |x| < 2^127
    const unsigned t = ((m - 0x38000000u) << 3) | (lo >> 29), rest = lo << 3;   // kept bits, dropped bits
    const unsigned up = rest > 0x80000000u || (rest == 0x80000000u && (t & 1u)) ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | (t + up));
  }
  if ((m | lo) == 0u) return __uint_as_float(hi);
  return (float)x;
}

struct MixedShared {
  double* v[2];   // kVecThreads values each: the first two walkers' output rows, idle between maps
  double w[2][4];
  double tot[kSegBatch][2];
  MixedCg cg[kCached];
  MixedSeg seg[kCached];
  int ok, bad;
};

// Partial sums of NV values of segment `s` (block-uniform) from every thread.
template <int NV>
__device__ __forceinline__ void segment_partial(MixedShared& sh, const double (&x)[NV], double* part, int nseg, int s) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < kVecThreads) {
#pragma unroll
    for (int j = 0; j < NV; ++j) sh.v[j][tid] = x[j];
  }
  __syncthreads();
  if (warp < 4 * NV) {
    const int j = warp >> 2, g = warp & 3, at = g * 32 + lane;
    double t = sh.v[j][at];
#pragma unroll
    for (int i = 1; i < kVecThreads / 128; ++i) t += sh.v[j][at + 128 * i];
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

// The producers' gate at the end of an iteration (b).
struct IterationGate {
  const unsigned* bar;
  unsigned target;
  __device__ __forceinline__ bool operator()() const { return wait_acquire(bar, target); }
};

template <int MODEL, typename PT>
__global__ void __launch_bounds__(kMixThreads, 1) mixed_cg_kernel(MixedArgs a) {
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
    segment_partial<2>(sh, x, part2, a.nseg, s0 + s);
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
      const IterationGate gate{bar, round * gridDim.x};
      if (n_my > 0 && !tile_map_pass<float, MODEL, OP_KV, true, false, IterationGate>(
                          V, n_my, it * n_my, nv, a.blobs, a.L, a.perm, a.mu0, a.lam0, io, a.err, -1, kWaitCycles, gate))
        sh.bad = 1;
    } else if (it > 0) {
      finish_y(pn, tid - kMapThreadsAll, 32 * kAuxWarps);
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
      segment_partial<1>(sh, x, part1, a.nseg, s0 + s);
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
      segment_partial<2>(sh, x, part2, a.nseg, s0 + s);
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
    // The producers wait for (b) themselves; the rest may not read the count
    // before it.
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

template <int MODEL, typename PT>
cudaError_t launch(const MixedArgs& a, int grid, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kMixThreads);
  cfg.dynamicSmemBytes = kWalkers * a.walker_smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, mixed_cg_kernel<MODEL, PT>, a);
}

size_t walker_bytes(const BlobLayout& L) { return (Tile::bytes(L) + 127) / 128 * 128; }

template <int MODEL, typename PT>
bool resident(size_t smem) {
  int n = 0;
  if (cudaFuncSetAttribute(mixed_cg_kernel<MODEL, PT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return false;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, mixed_cg_kernel<MODEL, PT>, kMixThreads, smem) ==
             cudaSuccess &&
         n >= 1;
}

}  // namespace

void free_mixed_plan(MixedPlan* plan) {
  if (!plan) return;
  cudaFree(plan->slab);
  delete plan;
}

const MixedResult* mixed_results(const MixedPlan* plan) { return plan->res; }

bool mixed_cg_ready(ebb_ctx_s* ctx, ebb_rel_s* rel, const std::vector<int>& vstart, MixedPlan** out) {
  if (*out) return (*out)->grid > 0;
  MixedPlan* m = new MixedPlan();
  *out = m;   // grid 0: does not apply
  const int nv = vstart.back(), nmesh = (int)vstart.size() - 1;
  int nsm = 0;
  if (rel->tiles.ntiles == 0 || nv == 0 ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess || nsm < 1) {
    cudaGetLastError();
    return false;
  }
  // A block per SM: small meshes too, for whose few vertices and tiles more SMs
  // mean shorter passes.
  const int grid = nsm;
  // Segments are summed one after the other: a batch of very many meshes is better
  // off with a block per mesh.
  if (nmesh > 16 * grid) return false;
  const size_t smem = kWalkers * walker_bytes(rel->tiles.L32);
  if (!resident<EBB_STVK, unsigned char>(smem) || !resident<EBB_NEOHOOKEAN, unsigned char>(smem) ||
      !resident<EBB_STVK, int>(smem) || !resident<EBB_NEOHOOKEAN, int>(smem)) {
    cudaGetLastError();
    return false;
  }
  std::vector<MixedSeg> seg;
  std::vector<int> first(grid + 1, 0), part0(nmesh + 1, 0);
  int mesh = 0;
  for (int b = 0; b < grid; ++b) {
    first[b] = (int)seg.size();
    int v = (int)((long long)b * nv / grid);
    const int end = (int)((long long)(b + 1) * nv / grid);
    while (v < end) {
      while (vstart[mesh + 1] <= v) ++mesh;
      const int e = std::min(end, vstart[mesh + 1]);
      MixedSeg s;
      s.mesh = mesh;
      s.v0 = v;
      s.v1 = e;
      s.lead = v == vstart[mesh] ? 1 : 0;
      s.part0 = s.npart = 0;
      if (s.lead) part0[mesh] = (int)seg.size();
      seg.push_back(s);
      v = e;
    }
  }
  first[grid] = (int)seg.size();
  const int nseg = (int)seg.size();
  part0[nmesh] = nseg;
  for (MixedSeg& s : seg) {
    s.part0 = part0[s.mesh];
    s.npart = part0[s.mesh + 1] - part0[s.mesh];
  }
  auto up = [](size_t n) { return (n + 127) / 128 * 128; };
  const size_t b_cg = up(nseg * sizeof(MixedCg)), b_part = up(3 * (size_t)nseg * sizeof(double)),
               b_res = up(nmesh * sizeof(MixedResult)), b_seg = up(nseg * sizeof(MixedSeg)),
               b_first = up((grid + 1) * sizeof(int));
  char* d = nullptr;
  if (cudaMalloc(&m->slab, b_cg + b_part + b_res + b_seg + b_first + 128) != cudaSuccess) {
    m->slab = nullptr;
    cudaGetLastError();
    return false;
  }
  d = static_cast<char*>(m->slab);
  m->cg = reinterpret_cast<MixedCg*>(d);
  m->part = reinterpret_cast<double*>(d += b_cg);
  m->res = reinterpret_cast<MixedResult*>(d += b_part);
  m->seg = reinterpret_cast<MixedSeg*>(d += b_res);
  m->first = reinterpret_cast<int*>(d += b_seg);
  m->ctl = reinterpret_cast<unsigned*>(d += b_first);
  if (cudaMemcpy(m->seg, seg.data(), nseg * sizeof(MixedSeg), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(m->first, first.data(), (grid + 1) * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(m->slab);
    m->slab = nullptr;
    return false;
  }
  m->nmesh = nmesh;
  m->nseg = nseg;
  m->grid = grid;
  return true;
}

cudaError_t launch_mixed_cg(ebb_rel_s* rel, MixedPlan* m, int model, float mu0, float lam0, const MixedVectors& v,
                            double dt, double rtol, int max_iters, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(m->ctl, 0, 2 * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  MixedArgs a;
  a.nv = (int)rel->verts->size;
  a.ntiles = rel->tiles.ntiles;
  a.blobs = rel->tiles.blob32;
  a.L = rel->tiles.L32;
  a.perm = rel->tet_perm;
  a.mu0 = mu0;
  a.lam0 = lam0;
  a.err = rel->ctx->d_err;
  a.v = v;
  a.seg = m->seg;
  a.first = m->first;
  a.nseg = m->nseg;
  a.cg = m->cg;
  a.part = m->part;
  a.res = m->res;
  a.ctl = m->ctl;
  a.dt = dt;
  a.rtol = rtol;
  a.max_iters = max_iters;
  a.walker_smem = walker_bytes(a.L);
  if (v.pin_bytes == 4)
    return model == EBB_STVK ? launch<EBB_STVK, int>(a, m->grid, st) : launch<EBB_NEOHOOKEAN, int>(a, m->grid, st);
  return model == EBB_STVK ? launch<EBB_STVK, unsigned char>(a, m->grid, st)
                           : launch<EBB_NEOHOOKEAN, unsigned char>(a, m->grid, st);
}

}  // namespace ebb
