// FP64 implicit step on the assembled row matrix.
//
// The same step as cg.cu (Sections 7.2 and 7.3: A = M + dt^2 K, b = dt (f + M g
// - dt K v), Jacobi PCG from dv = 0, v += dv, u += dt v), for FP64 element
// arithmetic.  GB300 issues one FP64 instruction per 19 cycles and SM
// (measured; 64 cycles when a single warp issues), and the matrix-free K p
// costs about 300 of them per tet and iteration.  An assembled row costs 9 per
// block, about 30 per tet, so K(u) is assembled once per step (row_matrix.cuh)
// and the CG iterations run on the rows:
//   element_block_kernel  element blocks and forces, one thread per tet
//   row_block_kernel      the rows' off-diagonal blocks of dt^2 K
//   row_cg_kernel         in one cooperative launch the diagonal blocks, b and
//                         1/diag(A), the whole PCG solve and the update of u, v
// No atomics on floating-point data: results repeat bit for bit, whatever
// reduction the caller names.
// Measured, against the matrix-free step with two launches per iteration: 8^3
// StVK step (2,560 tets) 504 -> 137 us; 20-step rollout and gradient on the
// 32^3 mesh (163,840 tets) 213 -> 46.7 ms.  The small step's solve in one cluster
// of 16 blocks, sums through distributed shared memory: 185 us, 16 SMs' FP64
// pipes being too few.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>

#include "grid_barrier.cuh"
#include "row_matrix.cuh"

namespace ebb {

// Result of a solve, written to page-locked host memory by the last kernel.
struct RowResult {
  double rr, bb;
  int iter, status;
  int err_code, err_index;   // the context's device status word
};

struct RowStep {
  int nv = 0;
  void* slab = nullptr;      // everything below but the host result
  double *elem = nullptr, *val = nullptr;
  double *r = nullptr, *z = nullptr, *p = nullptr, *y = nullptr, *s = nullptr, *w = nullptr, *dinv = nullptr;
  double* mass = nullptr;
  double* part = nullptr;
  unsigned* bar = nullptr;
  RowResult* host = nullptr;
  RowResult* host_dev = nullptr;
  double rho = -1.0;
  double* vjp = nullptr;     // w, lam, K lam, x.q: planes of nv each (adjoint only)
  double* state = nullptr;   // u, v in the internal vertex order (reordered relations)
  unsigned char* pin = nullptr;
};

namespace {

constexpr int kPlainThreads = 768;   // row_cg_kernel, one CTA per SM
constexpr int kSplitThreads = 128;   // its form for few slices
constexpr int kMaxGrid = kRowMaxGrid;   // partial sums per set

// Streaming load of a matrix value (read once per product: not kept in L1,
// which the gathered vector entries use). Not through the read-only path: the
// kernel itself writes the diagonal blocks at its start.
__device__ __forceinline__ double ld_stream(const double* p) {
  double x;
  asm volatile("ld.global.L1::no_allocate.f64 %0, [%1];" : "=d"(x) : "l"(p));
  return x;
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

template <typename PT>
__device__ __forceinline__ bool pinned_at(const PT* pin, int v) {
  return pin != nullptr && pin[v] != 0;
}

__global__ void row_mass_kernel(int nv, const int* __restrict__ off, const int* __restrict__ ent,
                                const double* __restrict__ V, double rho, double* m) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nv) return;
  double s = 0.0;
  for (int e = off[v]; e < off[v + 1]; ++e) s += V[ent[e] >> 2];
  m[v] = 0.25 * rho * s;
}

// ---- the solve --------------------------------------------------------------
enum RowFinish { FIN_STEP = 0, FIN_VELOCITY = 1, FIN_ADJOINT = 2 };

struct RowCgArgs {
  RowView m;
  int nv;
  double* val;
  double* dinv;
  double *r, *z, *p, *y, *s, *w;   // CG vectors, [3 v + c]
  double* part;                 // 2 sets of kSums x kMaxGrid
  unsigned* bar;
  const int* err;               // the context's device status word
  RowResult* res;
  int max_iters;
  double rtol, dt;
  int finish;
  bool fresh;                   // the diagonal blocks are still to be formed
  const int* __restrict__ voff;
  const int* __restrict__ vent;
  const double* __restrict__ elem;
  const double* __restrict__ mass;
  double g[3];
  double *u, *v;                // FIN_STEP: the state, planes, updated in place
  double* out;                  // FIN_VELOCITY: v + dv; FIN_ADJOINT: the solution (planes)
  const double *gu, *gv;        // FIN_ADJOINT: the right-hand side is gv + dt gu
};

constexpr int kSums = 3;        // r.z, w.z, r.r

template <int NP>
struct RowCgShared {
  double v[kSums][NP];
  double w[kSums][2];
  double tot[kSums];
  double alpha, beta, pq;       // of this iteration; pq = p.Ap
  double inv[2];                // 1 / r.z, by iteration parity
  int active, ok;
};

template <int NP>
__device__ __forceinline__ bool grid_join(RowCgShared<NP>& sh, const unsigned* bar, unsigned round) {
  if (threadIdx.x == 0) sh.ok = wait_acquire(bar, round * gridDim.x);
  __syncthreads();
  return sh.ok != 0;
}

// Grid-wide sums of kSums values per participating thread (the first NP), and
// a grid barrier: every block writes its partials, waits until all have, and
// adds the partials in block order, one value per warp, so that every block
// obtains the same sums (in sh.tot).  A block writes its partials again only after
// the barrier at the end of an iteration, which every block reaches with the sums
// read; the count of rounds rises by two between sums, so they stay in one of the
// two sets.
template <int NP>
__device__ __forceinline__ bool grid_sum(RowCgShared<NP>& sh, const double (&x)[kSums], double* part, unsigned* bar,
                                         unsigned& round) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double* set = part + (size_t)(round & 1u) * kSums * kMaxGrid;
  ++round;
  if (tid < NP) {
#pragma unroll
    for (int j = 0; j < kSums; ++j) sh.v[j][tid] = x[j];
  }
  if (tid == 0) sh.ok = 1;
  __syncthreads();
  // two warps per value (one where a warp's lanes are all there is): FP64 adds
  // are issue-bound, so few of them, spread over the SM's sub-partitions
  constexpr int W = NP > 32 ? 2 : 1;
  if (warp < W * kSums) {
    const int j = warp / W, h = warp % W;
    double s = sh.v[j][h * 32 + lane];
#pragma unroll
    for (int i = 1; i < NP / (32 * W); ++i) s += sh.v[j][h * 32 + lane + 32 * W * i];
    s = warp_sum(s);
    if (lane == 0) sh.w[j][h] = s;
  }
  __syncthreads();
  if (warp < kSums) {
    if (tid == 0) {
#pragma unroll
      for (int j = 0; j < kSums; ++j) set[j * kMaxGrid + blockIdx.x] = W == 2 ? sh.w[j][0] + sh.w[j][1] : sh.w[j][0];
      arrive_release(bar);
    }
    const bool ok = wait_acquire(bar, round * gridDim.x);
    double t[kMaxGrid / 32];
#pragma unroll
    for (int i = 0; i < kMaxGrid / 32; ++i) {
      const int b = lane + 32 * i;
      t[i] = b < (int)gridDim.x ? __ldcg(set + warp * kMaxGrid + b) : 0.0;
    }
    double s = t[0];
#pragma unroll
    for (int i = 1; i < kMaxGrid / 32; ++i)
      if (32 * i < (int)gridDim.x) s += t[i];
    s = warp_sum(s);
    if (lane == 0) {
      sh.tot[warp] = s;
      if (!ok) sh.ok = 0;
    }
  }
  __syncthreads();
  return sh.ok != 0;
}

// The PCG solve, every block resident (cooperative launch), in the form whose
// two scalars come from one reduction (Chronopoulos and Gear, "s-step
// iterative methods for symmetric linear systems", 1989): per iteration
//   w = A z;  r.z, w.z, r.r
//   | beta = r.z / (r.z)', alpha = r.z / (w.z - beta r.z / alpha');  p = z + beta p;
//     s = w + beta s (= A p);  y += alpha p;  r -= alpha s;  z = r / diag A  |
// with two grid barriers (|) where the usual form has three.  Measured on the
// 32^3 mesh, in SM cycles of an iteration: product 20,000 (17,500 at the FP64
// issue rate), reduction 8,500 (5,000 when no block is late), scalars 1,800,
// vectors 1,300, barrier 3,000; in the usual form with vectors in memory and
// slices of unequal length the iteration took 50,000.
// A warp owns whole slices, a lane one component of one row, in every pass,
// so all vectors but z stay with their thread: in registers for the warp's
// first slice (all of them on meshes of up to 36,000 vertices), in memory for
// the others.  SPLIT: four warps share a slice's slots and the first adds
// their sums; for meshes with at most two slices per SM, where one warp's chain
// of FP64 operations (64 cycles each) would be the iteration.  Whole steps, split
// and not: 12^3 mesh (1.4 slices per SM) 142 and 164 us, 13^3 (1.8) 142 and 162,
// 14^3 (2.2) 186 and 175, 16^3 (3.2) 230 and 184.
template <int NT, bool SPLIT, typename PT>
__global__ void __launch_bounds__(NT, 1) row_cg_kernel(RowCgArgs a, const PT* __restrict__ pin) {
  constexpr int NP = SPLIT ? 32 : NT;
  __shared__ RowCgShared<NP> sh;
  __shared__ double s_acc[SPLIT ? 4 : 1][5][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool lane_on = lane < 3 * kSliceRows;
  const int i = lane_on ? lane / 3 : 0, c = lane_on ? lane - 3 * i : 0;
  const int first = first_slice(blockIdx.x, gridDim.x, a.m.nslice) + (SPLIT ? 0 : warp);
  const int last = first_slice(blockIdx.x + 1, gridDim.x, a.m.nslice);
  constexpr int sstep = SPLIT ? 1 : NT / 32;
  const int k0 = SPLIT ? warp : 0;
  constexpr int kstep = SPLIT ? 4 : 1;
  const bool vec = !SPLIT || warp == 0;   // this warp runs the vector passes
  unsigned round = 0;
  auto row = [&](int s) { return lane_on ? a.m.row_of[s * kSliceRows + i] : -1; };
  // sum of x over the four warps of a split slice, in warp 0 (slot f of s_acc)
  auto join = [&](double x, int f) {
    if constexpr (SPLIT) {
      s_acc[warp][f][lane] = x;
      __syncthreads();
      x = (s_acc[0][f][lane] + s_acc[1][f][lane]) + (s_acc[2][f][lane] + s_acc[3][f][lane]);
      __syncthreads();
    }
    return x;
  };
  // this lane's entry of A z
  auto product = [&](int q0, int nk) {
    double acc = 0.0;
    const int* col = a.m.col + (size_t)q0 * kSliceRows + i;
    const double* val = a.val + (size_t)q0 * 96 + lane;
    // groups of U slots; the next group's columns are loaded a group ahead
    constexpr int U = SPLIT ? 5 : 3;
    int j[U];
#pragma unroll
    for (int g = 0; g < U; ++g) j[g] = k0 + g * kstep < nk ? col[(k0 + g * kstep) * kSliceRows] : 0;
    for (int k = k0; k < nk; k += U * kstep) {
      double x[U][3], w[U][3];
#pragma unroll
      for (int g = 0; g < U; ++g) {
        const bool in = k + g * kstep < nk;
        const double* xv = a.z + 3 * (size_t)j[g];
        const double* wv = val + (size_t)(in ? k + g * kstep : 0) * 96;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          x[g][d] = xv[d];
          w[g][d] = ld_stream(wv + 32 * d);
        }
      }
#pragma unroll
      for (int g = 0; g < U; ++g) {
        const int kn = k + (U + g) * kstep;
        j[g] = kn < nk ? col[kn * kSliceRows] : 0;
      }
#pragma unroll
      for (int g = 0; g < U; ++g)
        if (k + g * kstep < nk) {
#pragma unroll
          for (int d = 0; d < 3; ++d) acc = fma(w[g][d], x[g][d], acc);
        }
    }
    return join(acc, 0);
  };
  // the first slice's rows, and this lane's vector entries of it
  const int fq0 = first < last ? a.m.slice_off[first] : 0;
  const int fnk = first < last ? a.m.slice_off[first + 1] - fq0 : 0;
  const int fv = vec && fnk > 0 ? row(first) : -1;
  const size_t fo = fv >= 0 ? 3 * (size_t)fv + c : 0;
  double fr = 0.0, fz = 0.0, fp = 0.0, fs = 0.0, fy = 0.0, fd = 0.0, fw = 0.0;

  // Diagonal blocks (minus the sum of the row's others, plus the mass), the
  // right-hand side, and z = r / diag(A).
  const bool rhs = a.finish != FIN_ADJOINT;
  for (int s = first; s < last; s += sstep) {
    const int q0 = a.m.slice_off[s], nk = a.m.slice_off[s + 1] - q0;
    if (nk == 0) continue;
    const int v = row(s);
    const bool on = v >= 0 && !pinned_at(pin, v);
    double* val = a.val + (size_t)q0 * 96 + lane;
    double b = 0.0, dcc = 1.0;
    if (a.fresh) {
      double dg[3] = {0.0, 0.0, 0.0}, kv = 0.0, f = 0.0;
      const int* col = a.m.col + (size_t)q0 * kSliceRows + i;
#pragma unroll 2
      for (int k = k0; k < nk; k += kstep) {
        if (k == 0) continue;
        const int j = col[k * kSliceRows];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const double x = val[k * 96 + 32 * d];
          dg[d] -= x;
          if (rhs) kv = fma(x, a.v[(size_t)d * a.nv + j], kv);
        }
      }
      if (rhs && on) {
        const int e1 = a.voff[v + 1];
#pragma unroll 2
        for (int e = a.voff[v] + k0; e < e1; e += kstep) {
          const int code = a.vent[e], corner = code & 3;
          const double* rec = a.elem + (size_t)(code >> 2) * kElemLen + 4 * c + 3;
          if (corner == 0)
            f -= rec[0] + rec[12] + rec[24];
          else
            f += rec[12 * (corner - 1)];
        }
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) dg[d] = join(dg[d], d);
      if (rhs) {
        kv = join(kv, 3);
        f = join(f, 4);
      }
      if (vec) {
        const double m = on ? a.mass[v] : 0.0;
        if (rhs && on) {
#pragma unroll
          for (int d = 0; d < 3; ++d) kv = fma(dg[d], a.v[(size_t)d * a.nv + v], kv);
          b = a.dt * (f + m * a.g[c]) - kv;
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          if (d == c) dg[d] += m;
          val[32 * d] = dg[d];
          if (d == c && on) dcc = dg[d];
        }
      }
    }
    if (vec && v >= 0) {
      const size_t o = 3 * (size_t)v + c;
      const double di = a.fresh ? 1.0 / dcc : a.dinv[o];
      if (!rhs && on) {
        const size_t pl = (size_t)c * a.nv + v;
        b = a.gv[pl] + a.dt * a.gu[pl];
      }
      if (a.fresh) a.dinv[o] = di;
      const double z = b * di;
      a.z[o] = z;
      if (s == first) {
        fr = b;
        fz = z;
        fd = di;
      } else {
        a.r[o] = b;
        a.p[o] = 0.0;
        a.s[o] = 0.0;
        a.y[o] = 0.0;
      }
    }
  }
  int status = EBB_OK, it = 0;
  double bb = 0.0, rr = 0.0, tol = 0.0;
  grid_arrive(a.bar, round);
  bool ok = grid_join(sh, a.bar, round);
  while (ok) {
    double sums[kSums] = {0.0, 0.0, 0.0};
    if (SPLIT ? first < last : fnk > 0) {
      fw = product(fq0, fnk);
      if (fv >= 0) {
        sums[0] = fr * fz;
        sums[1] = fw * fz;
        sums[2] = fr * fr;
      }
    }
    for (int s = first + sstep; s < last; s += sstep) {
      const int q0 = a.m.slice_off[s], nk = a.m.slice_off[s + 1] - q0;
      if (nk == 0) continue;
      const double acc = product(q0, nk);
      const int v = vec ? row(s) : -1;
      if (v >= 0) {
        const size_t o = 3 * (size_t)v + c;
        const double ri = a.r[o], zi = a.z[o];
        a.w[o] = acc;
        sums[0] = fma(ri, zi, sums[0]);
        sums[1] = fma(acc, zi, sums[1]);
        sums[2] = fma(ri, ri, sums[2]);
      }
    }
    ok = grid_sum(sh, sums, a.part, a.bar, round);
    if (!ok) break;
    rr = sh.tot[2];
    if (it == 0) bb = rr;
    // The scalars, by one thread each: alpha and beta, the convergence test,
    // and 1 / r.z for the next iteration (the divisions are FP64 chains).
    const double rz = sh.tot[0];
    if (threadIdx.x == 0) {
      double beta = 0.0, pq = sh.tot[1];
      if (it > 0) {
        beta = rz * sh.inv[~it & 1];
        pq -= beta * (rz * (sh.pq * sh.inv[~it & 1]));   // 1 / alpha' = (p.Ap)' / (r.z)'
      }
      sh.pq = pq;
      sh.alpha = rz / pq;
      sh.beta = beta;
    } else if (threadIdx.x == 32) {
      if (it == 0) tol = a.rtol * sqrt(bb);
      sh.active = it < a.max_iters && sqrt(rr) > tol;
    } else if (threadIdx.x == 64) {
      sh.inv[it & 1] = 1.0 / rz;
    }
    __syncthreads();
    if (!sh.active) break;
    if (!(sh.pq > 0.0)) {
      status = EBB_ERR_CG_BREAKDOWN;
      break;
    }
    const double alpha = sh.alpha, beta = sh.beta;
    const double zold = fz;
    if (fv >= 0) {
      fs = fma(beta, fs, fw);
      fr = fma(-alpha, fs, fr);
      fz = fr * fd;
      a.z[fo] = fz;
    }
    if (vec)
      for (int s = first + sstep; s < last; s += sstep) {
        const int v = row(s);
        if (v < 0) continue;
        const size_t o = 3 * (size_t)v + c;
        const double pi = fma(beta, a.p[o], a.z[o]), si = fma(beta, a.s[o], a.w[o]);
        const double ri = fma(-alpha, si, a.r[o]);
        a.p[o] = pi;
        a.s[o] = si;
        a.y[o] = fma(alpha, pi, a.y[o]);
        a.r[o] = ri;
        a.z[o] = ri * a.dinv[o];
      }
    ++it;
    grid_arrive(a.bar, round);
    fp = fma(beta, fp, zold);
    fy = fma(alpha, fp, fy);
    ok = grid_join(sh, a.bar, round);
  }
  if (!ok) status = EBB_ERR_TIMEOUT;
  if (vec && ok)
    for (int s = first; s < last; s += sstep) {
      const int v = row(s);
      if (v < 0) continue;
      const double dv = s == first ? fy : a.y[3 * (size_t)v + c];
      const size_t pl = (size_t)c * a.nv + v;
      if (a.finish == FIN_STEP) {
        const double vi = a.v[pl] + dv;
        a.v[pl] = vi;
        a.u[pl] += a.dt * vi;
      } else {
        a.out[pl] = a.finish == FIN_VELOCITY ? a.v[pl] + dv : dv;
      }
    }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    RowResult h;
    h.rr = rr;
    h.bb = bb;
    h.iter = it;
    h.status = status;
    h.err_code = a.err[ERRW_CODE];
    h.err_index = a.err[ERRW_INDEX];
    *a.res = h;
    __threadfence_system();
  }
}

// K lam and x.q accumulators cleared; w = v' (given, or already there).
__global__ void row_vjp_prep_kernel(int n, const double* __restrict__ v_next, double* w, double* acc_kl,
                                    double* acc_xq) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (v_next != nullptr) w[i] = v_next[i];
    acc_kl[i] = 0.0;
    acc_xq[i] = 0.0;
  }
}

// dL/du = gu - dt K lam - dt^2 d/dx[lam^T K v'];  dL/dv = gv + dt gu - dt^2 K lam.
__global__ void row_vjp_finish_kernel(int n, double dt, const double* __restrict__ acc_kl,
                                      const double* __restrict__ acc_xq, double* gu, double* gv) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double g = gu[i], kl = acc_kl[i];
    gu[i] = g - dt * kl - dt * dt * acc_xq[i];
    gv[i] = gv[i] + dt * g - dt * dt * kl;
  }
}

template <int NT, bool SPLIT, typename PT>
cudaError_t launch_cg(const RowCgArgs& a, const PT* pin, int grid, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(NT);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, row_cg_kernel<NT, SPLIT, PT>, a, pin);
}

template <typename PT>
cudaError_t solve(const RowCgArgs& a, const PT* pin, int grid, cudaStream_t st) {
  const int slices = (a.nv + kSliceRows - 1) / kSliceRows;   // that hold rows
  if (slices <= 2 * grid) return launch_cg<kSplitThreads, true, PT>(a, pin, grid, st);
  return launch_cg<kPlainThreads, false, PT>(a, pin, grid, st);
}

// The step's buffers, in one allocation.  *fits is false when the device has
// no room for them (the caller falls back to the matrix-free step).
ebb_status_t ensure_row_step(ebb_ctx_s* ctx, ebb_rel_s* tets, bool* fits) {
  *fits = true;
  if (tets->row_step) return EBB_OK;
  RowStep* s = new RowStep();
  const RowMatrix& m = *tets->rows;
  const int nv = (int)tets->verts->size;
  s->nv = nv;
  const size_t n3 = (size_t)3 * nv;
  const size_t elem = (size_t)tets->size * kElemLen, val = (size_t)m.nslots * 96;
  const size_t total = elem + val + 7 * n3 + nv + 2 * kSums * kMaxGrid + 2;
  cudaError_t e = cudaMalloc(&s->slab, total * sizeof(double));
  if (e == cudaSuccess) e = cudaHostAlloc(&s->host, sizeof(RowResult), cudaHostAllocMapped);
  if (e == cudaSuccess) e = cudaHostGetDevicePointer(&s->host_dev, s->host, 0);
  if (e != cudaSuccess) {
    cudaFree(s->slab);
    if (s->host) cudaFreeHost(s->host);
    delete s;
    cudaGetLastError();
    *fits = false;
    return e == cudaErrorMemoryAllocation ? EBB_OK : cuda_check(ctx, e, "implicit-step scratch");
  }
  double* d = static_cast<double*>(s->slab);
  auto take = [&](size_t k) {
    double* at = d;
    d += k;
    return at;
  };
  s->elem = take(elem);
  s->val = take(val);
  s->r = take(n3);
  s->z = take(n3);
  s->p = take(n3);
  s->y = take(n3);
  s->s = take(n3);
  s->w = take(n3);
  s->dinv = take(n3);
  s->mass = take(nv);
  s->part = take(2 * kSums * kMaxGrid);
  s->bar = reinterpret_cast<unsigned*>(take(2));
  e = cudaMemsetAsync(s->val, 0, val * sizeof(double), ctx->stream);   // unused entries stay zero
  if (e != cudaSuccess) {
    cudaFree(s->slab);
    cudaFreeHost(s->host);
    delete s;
    return cuda_check(ctx, e, "implicit-step scratch");
  }
  tets->row_step = s;
  return EBB_OK;
}

// A solve that goes on past rounding (rtol 0) ends when r.r or r.z underflows: 1 / r.z
// then overflows and p.Ap, which the kernel has from differences, is no number to
// trust.  Such a solve is done, not broken down.  1e-290: diag(A) up to 1e18 lies
// between the two; the residual has to be past rounding too.
ebb_status_t solve_status(const RowResult& h) {
  const bool underflow = h.iter > 0 && h.rr < 1e-290 && h.rr <= 1e-32 * h.bb;
  return h.status == EBB_ERR_CG_BREAKDOWN && underflow ? EBB_OK : h.status;
}

struct RowVjp {
  double *gu, *gv, *gmu, *glam;
  const double* v_next;
};

template <typename PT>
ebb_status_t row_step_impl(ebb_ctx_s* ctx, ebb_rel_s* tets, double* u, double* v, const PT* pin,
                           const ebb_step_params_t* prm, ebb_cg_report_t* rep, const RowVjp* vjp) {
  RowStep* s = tets->row_step;
  const RowMatrix& m = *tets->rows;
  const int nv = s->nv, n = 3 * nv;
  cudaStream_t st = ctx->stream;
  cudaError_t e = cudaSuccess;
  if (s->rho != prm->rho) {
    row_mass_kernel<<<(nv + 255) / 256, 256, 0, st>>>(nv, tets->vindex.off, tets->vindex.ent, tets->s64.V, prm->rho,
                                                       s->mass);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_check(ctx, e, "lumped mass");
    s->rho = prm->rho;
  }
  const bool forward = vjp == nullptr || vjp->v_next == nullptr;
  e = launch_element_blocks<double>(tets, prm->model, prm->mu, prm->lambda, u, false, forward, s->elem, st);
  if (e != cudaSuccess) return cuda_check(ctx, e, "element blocks");
  RowCgArgs ca;
  memset(&ca, 0, sizeof ca);
  ca.m = RowView{m.nslice, m.slice_off, m.row_of, m.col};
  e = cudaMemsetAsync(s->bar, 0, sizeof(unsigned), st);
  if (e == cudaSuccess)
    e = launch_row_blocks<double>(m, s->elem, pin, (int)sizeof(PT), prm->dt * prm->dt, s->val, st);
  if (e != cudaSuccess) return cuda_check(ctx, e, "rows of the step matrix");
  ca.nv = nv;
  ca.val = s->val;
  ca.dinv = s->dinv;
  ca.r = s->r;
  ca.z = s->z;
  ca.p = s->p;
  ca.y = s->y;
  ca.s = s->s;
  ca.w = s->w;
  ca.part = s->part;
  ca.bar = s->bar;
  ca.fresh = true;
  ca.voff = tets->vindex.off;
  ca.vent = tets->vindex.ent;
  ca.elem = s->elem;
  ca.mass = s->mass;
  for (int k = 0; k < 3; ++k) ca.g[k] = prm->gravity[k];
  ca.err = ctx->d_err;
  ca.res = s->host_dev;
  ca.max_iters = prm->max_iters;
  ca.rtol = prm->rtol;
  ca.dt = prm->dt;
  ca.finish = vjp ? FIN_VELOCITY : FIN_STEP;
  ca.u = u;
  ca.v = v;
  double *w = nullptr, *lam = nullptr, *kl = nullptr, *xq = nullptr;
  if (vjp) {
    w = s->vjp;
    lam = w + n;
    kl = lam + n;
    xq = kl + n;
    ca.out = w;
  }
  ebb_status_t status = EBB_OK;
  if (forward) {
    e = solve<PT>(ca, pin, m.grid, st);
    if (e == cudaSuccess && vjp) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_check(ctx, e, "CG solve");
    if (vjp && solve_status(*s->host) != EBB_OK)
      return set_error(ctx, s->host->status, "forward solve failed inside the step VJP");
    ca.fresh = false;   // the adjoint solve takes the same matrix
  }
  if (vjp) {
    row_vjp_prep_kernel<<<4 * 152, 256, 0, st>>>(n, vjp->v_next, w, kl, xq);
    e = cudaGetLastError();
    if (e == cudaSuccess && forward) e = cudaMemsetAsync(s->bar, 0, sizeof(unsigned), st);
    ca.finish = FIN_ADJOINT;
    ca.out = lam;
    ca.gu = vjp->gu;
    ca.gv = vjp->gv;
    if (e == cudaSuccess) e = solve<PT>(ca, pin, m.grid, st);
    if (e == cudaSuccess)
      e = launch_adjoint_map(tets, prm->mu, prm->lambda, u, lam, w, kl, xq, vjp->gmu, vjp->glam, prm->dt, st);
    if (e == cudaSuccess) {
      row_vjp_finish_kernel<<<4 * 152, 256, 0, st>>>(n, prm->dt, kl, xq, vjp->gu, vjp->gv);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_check(ctx, e, "adjoint solve");
  }
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_check(ctx, e, "step finish");
  const RowResult h = *s->host;
  status = solve_status(h);
  const double rel = h.bb > 0.0 ? std::sqrt(h.rr / h.bb) : 0.0;
  if (rep) {
    rep->iters = h.iter;
    rep->rel_residual = rel;
  }
  char buf[128];
  if (h.err_code != 0) {
    // Device-raised errors (inverted elements) take precedence.
    cudaMemsetAsync(ctx->d_err, 0, ERRW_WORDS * sizeof(int), st);
    cudaStreamSynchronize(st);
    snprintf(buf, sizeof buf, "device error %d (inverted element?) at tet row %d", h.err_code, h.err_index);
    status = set_error(ctx, h.err_code, buf);
  } else if (status == EBB_ERR_CG_BREAKDOWN) {
    snprintf(buf, sizeof buf, "PCG breakdown (p^T A p <= 0) at iteration %d", h.iter);
    set_error(ctx, status, buf);
  } else if (status == EBB_ERR_TIMEOUT) {
    set_error(ctx, status, "a bounded device wait of the CG solve gave up");
  } else if (prm->fail_on_max_iters && h.iter >= prm->max_iters && rel > prm->rtol) {
    snprintf(buf, sizeof buf, "PCG not converged after %d iterations (rel residual %.3e)", h.iter, rel);
    status = set_error(ctx, EBB_ERR_NOT_CONVERGED, buf);
  }
  if (rep) rep->status = status;
  return status;
}

template <typename PT>
ebb_status_t run_rows(ebb_ctx_s* ctx, ebb_rel_s* tets, double* u, double* v, const void* pin,
                      const ebb_step_params_t* p, ebb_cg_report_t* rep, const RowVjp* vjp) {
  return row_step_impl<PT>(ctx, tets, u, v, static_cast<const PT*>(pin), p, rep, vjp);
}

}  // namespace

void free_row_step(ebb_rel_s* tets) {
  RowStep* s = tets->row_step;
  if (!s) return;
  cudaFree(s->slab);
  cudaFree(s->vjp);
  cudaFree(s->state);
  cudaFree(s->pin);
  cudaFreeHost(s->host);
  delete s;
  tets->row_step = nullptr;
}

// Does the row form take this relation's FP64 steps?  Builds the pattern and
// the buffers on first use.
ebb_status_t row_step_ready(ebb_ctx_s* ctx, ebb_rel_s* tets, bool* yes) {
  *yes = false;
  ebb_status_t s = ensure_row_pattern(ctx, tets, ctx->stream);
  if (s) return s;
  if (tets->rows->state != 1 || tets->rows->no_step) return EBB_OK;
  bool fits = false;
  s = ensure_row_step(ctx, tets, &fits);
  if (s) return s;
  if (!fits) {
    tets->rows->no_step = true;   // no room: the matrix-free step from now on
    return EBB_OK;
  }
  *yes = true;
  return EBB_OK;
}

ebb_status_t run_row_step(ebb_ctx_s* ctx, ebb_rel_s* tets, double* u, double* v, const void* pinned,
                          ebb_dtype_t pinned_dtype, const ebb_step_params_t* p, ebb_cg_report_t* rep) {
  RowStep* s = tets->row_step;
  const int nv = s->nv;
  if (!tets->vperm)
    return pinned_dtype == EBB_I32 ? run_rows<int>(ctx, tets, u, v, pinned, p, rep, nullptr)
                                   : run_rows<unsigned char>(ctx, tets, u, v, pinned, p, rep, nullptr);
  // Reordered vertices: the step runs on the state in the internal order.
  cudaError_t e = cudaSuccess;
  if (!s->state) e = cudaMalloc(&s->state, (size_t)6 * nv * sizeof(double));
  if (e == cudaSuccess && !s->pin) e = cudaMalloc(&s->pin, (size_t)nv);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return set_error(ctx, EBB_ERR_NOMEM, "device allocation for the reordered state failed");
  }
  double *ui = s->state, *vi = s->state + (size_t)3 * nv;
  e = gather_vertex_field<double>(nv, tets->vperm, u, ui, ctx->stream);
  if (e == cudaSuccess) e = gather_vertex_field<double>(nv, tets->vperm, v, vi, ctx->stream);
  if (e == cudaSuccess)
    e = pinned_dtype == EBB_I32
            ? gather_pinned<int>(nv, tets->vperm, (const int*)pinned, s->pin, ctx->stream)
            : gather_pinned<unsigned char>(nv, tets->vperm, (const unsigned char*)pinned, s->pin, ctx->stream);
  if (e != cudaSuccess) return cuda_check(ctx, e, "reordering the state");
  const ebb_status_t r = run_rows<unsigned char>(ctx, tets, ui, vi, s->pin, p, rep, nullptr);
  e = scatter_vertex_field(nv, tets->vperm, ui, u, ctx->stream);
  if (e == cudaSuccess) e = scatter_vertex_field(nv, tets->vperm, vi, v, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) return cuda_check(ctx, e, "restoring the state order");
  return r;
}

ebb_status_t run_row_vjp(ebb_ctx_s* ctx, ebb_rel_s* tets, const double* u, const double* v, const double* v_next,
                         const void* pinned, ebb_dtype_t pinned_dtype, double* gu, double* gv, double* gmu,
                         double* glam, const ebb_step_params_t* p, ebb_cg_report_t* rep) {
  RowStep* s = tets->row_step;
  if (!s->vjp) {
    cudaError_t e = cudaMalloc(&s->vjp, (size_t)12 * s->nv * sizeof(double));
    if (e != cudaSuccess) {
      s->vjp = nullptr;
      cudaGetLastError();
      return set_error(ctx, EBB_ERR_NOMEM, "device allocation for the step VJP failed");
    }
  }
  // u and v are read only: the adjoint replaces the step's update.
  RowVjp a{gu, gv, gmu, glam, v_next};
  double *mu = const_cast<double*>(u), *mv = const_cast<double*>(v);
  return pinned_dtype == EBB_I32 ? run_rows<int>(ctx, tets, mu, mv, pinned, p, rep, &a)
                                 : run_rows<unsigned char>(ctx, tets, mu, mv, pinned, p, rep, &a);
}

}  // namespace ebb
