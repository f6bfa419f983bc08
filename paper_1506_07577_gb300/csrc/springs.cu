// Spring-mass system on the edge relation: the paper's introductory example
// (Section 4.1, Figure 1) as a second workload on the same runtime.
//
// The springs are the mesh's edges (the edge relation of EBB_FINALIZE_EDGES,
// each vertex's row listing its neighbours).  Per step, one kernel walks
// every vertex's row -- computeInternalForces, a per-vertex loop over the
// directed edges leaving it, one thread per vertex summing its springs in row
// order (no atomics; bitwise reproducible; measured faster than 2, 4 or 8
// lanes per vertex with a shuffle tree) -- and then applies the force to that
// vertex (applyForces):
//   f_v = sum_h K (L_vh dir - dq),  dq = q_v - q_h,  dir = dq / |dq|
//   qdd = f_v / m_v,  q_v += qd_v dt + qdd dt^2 / 2,  qd_v += qdd dt
// (the restoring reading of the figure's force; a zero-length dq gives no
// direction and a vertex with m <= 0 does not move).  Positions are read from
// one buffer and written to another (the two kernels of the figure, whose
// phases keep force accumulation and position update apart, fused by double
// buffering), velocities in place.  measureTotalEnergy is a two-pass sum of
// m |qd|^2 / 2 in FP64 in a fixed order.
#include <algorithm>

#include "async_copy.cuh"
#include "ebb_internal.h"
#include "row_matrix.cuh"

namespace ebb {

namespace {

constexpr int kSpringThreads = 256;
constexpr int kEnergyBlocks = 304;

// 1 / |dq| from |dq|^2 (CUDA's reciprocal square roots: within 2 ulp in
// FP32 and 1 ulp in FP64, one call where a square root and a division
// would be two; FP64 division and square root are long sequences on GB300's
// FP64 pipe).
template <typename T>
__device__ __forceinline__ T inv_len(T n2);
template <>
__device__ __forceinline__ float inv_len<float>(float n2) { return rsqrtf(n2); }
template <>
__device__ __forceinline__ double inv_len<double>(double n2) { return rsqrt(n2); }

// ---- spring slots -----------------------------------------------------------
// The springs of a vertex, self-loop left out, in slices of 32 rows: slot k of
// slice s holds the k-th spring of each of its rows, lane by lane, so that a
// warp reads other ends and rest lengths as lines of consecutive words (read
// from the edge relation's rows, each thread walks a run of its own).  Rows are
// taken in order of first use by the tets and sorted by length in windows of
// kSpringWindow rows, so that a slice's rows have nearly equal lengths; the
// order within a row stays that of the edge relation.  During a run positions,
// velocities and masses are held in row order too (loaded before the first step,
// stored after the last): a vertex's own data are then consecutive across a
// warp, and its neighbours' positions near each other.
constexpr int kSpringWindow = 1024;

__global__ void __launch_bounds__(kSpringWindow)
spring_window_kernel(int nv, const int* __restrict__ order, const int* __restrict__ row_off, int* row_of, int* place,
                     int* slots) {
  __shared__ int s_len[kSpringWindow];
  const int i = threadIdx.x;
  const int x = blockIdx.x * kSpringWindow + i;
  const int v = x < nv ? order[x] : -1;
  const int l = v >= 0 ? row_off[v + 1] - row_off[v] - 1 : 0;   // without the self-loop
  s_len[i] = l;
  __syncthreads();
  int rank = 0;
  for (int j = 0; j < kSpringWindow; ++j) rank += s_len[j] > l || (s_len[j] == l && j < i);
  row_of[blockIdx.x * kSpringWindow + rank] = v;
  if (v >= 0) place[v] = blockIdx.x * kSpringWindow + rank;
  if (rank % 32 == 0) slots[blockIdx.x * (kSpringWindow / 32) + rank / 32] = l;
}

// Other ends as rows (the row itself where it has no k-th spring)
// and rest lengths, in the positions' precision and the other one.
template <typename T, typename U>
__global__ void __launch_bounds__(kSpringThreads)
spring_fill_kernel(int nv, int nslice, const int* __restrict__ row_off, const int* __restrict__ col,
                   const int* __restrict__ row_of, const int* __restrict__ place, const int* __restrict__ slice_off,
                   const T* __restrict__ X, int* __restrict__ end, T* __restrict__ rest, U* __restrict__ rest_other) {
  const int r = blockIdx.x * kSpringThreads + threadIdx.x;
  const int s = r >> 5, lane = r & 31;
  if (s >= nslice) return;
  const int v = row_of[r];
  const int q0 = slice_off[s], nk = slice_off[s + 1] - q0;
  int e = v >= 0 ? row_off[v] : 0;
  const int e1 = v >= 0 ? row_off[v + 1] : 0;
  for (int k = 0; k < nk; ++k) {
    if (e < e1 && col[e] == v) ++e;
    const size_t at = (size_t)(q0 + k) * 32 + lane;
    const int h = e < e1 ? col[e] : 0;
    T len = T(0);
    const bool spring = e < e1;
    if (spring) {
      T n2 = T(0);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const T d = X[(size_t)c * nv + h] - X[(size_t)c * nv + v];
        n2 += d * d;
      }
      len = sqrt(n2);
      ++e;
    }
    end[at] = spring ? place[h] : r;
    rest[at] = len;
    rest_other[at] = (U)len;
  }
}

// Four-value vertex elements: one (FP32) or two (FP64) 16-byte accesses.
template <typename T>
struct alignas(16) Quad {
  T x, y, z, w;
};

// Positions, and velocities with 1 / m (0 for m <= 0), into row order.
template <typename T>
__global__ void __launch_bounds__(kSpringThreads)
spring_load_kernel(int nv, int nrows, const int* __restrict__ row_of, const T* __restrict__ q,
                   const T* __restrict__ qd, const T* __restrict__ mass, Quad<T>* __restrict__ pos,
                   Quad<T>* __restrict__ vel) {
  const int r = blockIdx.x * kSpringThreads + threadIdx.x;
  if (r >= nrows) return;
  const int v = row_of[r];
  if (v < 0) return;
  const size_t n = nv;
  const T m = mass[v];
  pos[r] = Quad<T>{q[v], q[n + v], q[2 * n + v], T(0)};
  vel[r] = Quad<T>{qd[v], qd[n + v], qd[2 * n + v], m > T(0) ? T(1) / m : T(0)};
}

// One step, a thread per row.  FP32: bound by the lines of the scattered
// position loads; FP64: by the FP64 pipe.  The last step writes positions and
// velocities to the caller's planes.  Steps are launched to overlap: a step's
// blocks take the places of the last step's as these end, read what no step
// writes, and wait for the last step's positions then.  Positions and velocities
// are therefore plain pointers: another launch may still be writing them when this
// one starts, so they are not constant during the kernel, as __restrict__ on a
// read-only pointer would promise (and allow loads that skip coherence).  Measured per FP32 step on
// the 64^3 mesh (274,625 vertices, 3.2 M directed springs): 9.3 us; groups of 4
// or 9 springs, or more blocks with fewer registers, 10 to 15 us; a thread walking
// its row of the edge relation, 17.1 us.
constexpr int kStepThreads = 128, kStepGroup = 6;

template <typename T>
__global__ void __launch_bounds__(kStepThreads, sizeof(T) == 4 ? 8 : 4)
spring_step_kernel(int nv, int nslice, const int* __restrict__ row_of, const int* __restrict__ slice_off,
                   const int* __restrict__ end, const T* __restrict__ rest, T k, T dt, const Quad<T>* qin,
                   Quad<T>* qout, Quad<T>* vel, T* q_planes, T* qd_planes) {
  release_next_kernel();
  const int r = blockIdx.x * kStepThreads + threadIdx.x;
  const int s = r >> 5, lane = r & 31;
  const int v = s < nslice ? row_of[r] : -1;
  const int q0 = s < nslice ? slice_off[s] : 0, nk = s < nslice ? slice_off[s + 1] - q0 : 0;
  const int* ep = end + (size_t)q0 * 32 + lane;
  const T* rp = rest + (size_t)q0 * 32 + lane;
  // groups of kStepGroup springs; the next group's ends are loaded a group ahead
  int h[kStepGroup];
#pragma unroll
  for (int g = 0; g < kStepGroup; ++g) h[g] = g < nk ? ep[g * 32] : r;
  wait_prior_kernel();
  if (v < 0) return;
  const Quad<T> own = qin[r];
  const Quad<T> vi = vel[r];
  const T qr[3] = {own.x, own.y, own.z}, vr[3] = {vi.x, vi.y, vi.z};
  T f[3] = {T(0), T(0), T(0)};
  for (int e = 0; e < nk; e += kStepGroup) {
    T oq[kStepGroup][3], len[kStepGroup];
    bool on[kStepGroup];
#pragma unroll
    for (int g = 0; g < kStepGroup; ++g) {
      const Quad<T> o = qin[h[g]];
      oq[g][0] = o.x;
      oq[g][1] = o.y;
      oq[g][2] = o.z;
      on[g] = h[g] != r;   // unused slots name the row itself
      len[g] = e + g < nk ? rp[(e + g) * 32] : T(0);
    }
#pragma unroll
    for (int g = 0; g < kStepGroup; ++g) h[g] = e + kStepGroup + g < nk ? ep[(e + kStepGroup + g) * 32] : r;
#pragma unroll
    for (int g = 0; g < kStepGroup; ++g) {
      T dq[3], n2 = T(0);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dq[c] = qr[c] - oq[g][c];
        n2 += dq[c] * dq[c];
      }
      const T w = n2 > T(0) ? len[g] * inv_len(n2) : T(0);
      if (on[g]) {
#pragma unroll
        for (int c = 0; c < 3; ++c) f[c] += k * (w * dq[c] - dq[c]);
      }
    }
  }
  T qn[3], vn[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const T a = f[c] * vi.w;
    qn[c] = qr[c] + vr[c] * dt + T(0.5) * a * dt * dt;
    vn[c] = vr[c] + a * dt;
  }
  if (q_planes != nullptr) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      q_planes[(size_t)c * nv + v] = qn[c];
      qd_planes[(size_t)c * nv + v] = vn[c];
    }
  } else {
    qout[r] = Quad<T>{qn[0], qn[1], qn[2], T(0)};
    vel[r] = Quad<T>{vn[0], vn[1], vn[2], vi.w};
  }
}

// Per-block partial sums of m |qd|^2 / 2 (FP64), block order fixed.
template <typename T>
__global__ void __launch_bounds__(kSpringThreads)
energy_partial_kernel(int nv, const T* __restrict__ qd, const T* __restrict__ mass, double* part) {
  __shared__ double s[kSpringThreads];
  double e = 0.0;
  for (int v = blockIdx.x * kSpringThreads + threadIdx.x; v < nv; v += gridDim.x * kSpringThreads) {
    double q2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double x = (double)qd[(size_t)c * nv + v];
      q2 += x * x;
    }
    e += 0.5 * (double)mass[v] * q2;
  }
  s[threadIdx.x] = e;
  __syncthreads();
  for (int w = kSpringThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

__global__ void energy_final_kernel(const double* part, int n, double* out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double e = 0.0;
  for (int i = 0; i < n; ++i) e += part[i];
  *out = e;
}

template <typename T>
cudaError_t springs_run_t(ebb_rel_s* tets, T* q, T* qd, const T* mass, double k, double dt, int steps, double* energy,
                          cudaStream_t st) {
  EdgeIndex& E = tets->edges;
  const int p = sizeof(T) == 4 ? 0 : 1;
  const int nv = (int)tets->verts->size;
  // positions, double-buffered, and velocities in row order
  const int nrows = E.spring_slices * 32;
  if (steps > 0 && nv > 0 && E.qbuf[p] == nullptr) {
    cudaError_t e = cudaMalloc(&E.qbuf[p], (size_t)12 * nrows * sizeof(T));
    if (e != cudaSuccess) {
      E.qbuf[p] = nullptr;
      return e;
    }
  }
  Quad<T>* buf = static_cast<Quad<T>*>(E.qbuf[p]);
  const T* rest = static_cast<const T*>(E.rest[p]);
  if (steps > 0 && nv > 0) {
    Quad<T>* vel = buf + (size_t)2 * nrows;
    const int grid = (nrows + kSpringThreads - 1) / kSpringThreads;
    spring_load_kernel<T><<<grid, kSpringThreads, 0, st>>>(nv, nrows, E.spring_row, q, qd, mass, buf, vel);
    for (int s = 0; s < steps; ++s) {
      const bool last = s + 1 == steps;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((nrows + kStepThreads - 1) / kStepThreads);
      cfg.blockDim = dim3(kStepThreads);
      cfg.stream = st;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      at[0].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = at;
      cfg.numAttrs = s > 0 ? 1 : 0;   // the first step follows whatever ran before
      const Quad<T>* qin = buf + (size_t)(s & 1) * nrows;
      cudaError_t e = cudaLaunchKernelEx(&cfg, spring_step_kernel<T>, nv, E.spring_slices,
                                         (const int*)E.spring_row, (const int*)E.spring_off, (const int*)E.spring_end,
                                         rest, (T)k, (T)dt, qin, buf + (size_t)((s + 1) & 1) * nrows, vel,
                                         last ? q : nullptr, last ? qd : nullptr);
      if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (energy != nullptr) {
    double* dpart = E.epart;
    energy_partial_kernel<T><<<kEnergyBlocks, kSpringThreads, 0, st>>>(nv, qd, mass, dpart);
    energy_final_kernel<<<1, 32, 0, st>>>(dpart, kEnergyBlocks, dpart + kEnergyBlocks);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(energy, dpart + kEnergyBlocks, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t springs_init(ebb_rel_s* tets, const void* X, bool f64, cudaStream_t st) {
  EdgeIndex& E = tets->edges;
  const int nv = (int)tets->verts->size;
  if (E.epart == nullptr) {
    cudaError_t e = cudaMalloc(&E.epart, (kEnergyBlocks + 1) * sizeof(double));
    if (e != cudaSuccess) {
      E.epart = nullptr;
      return e;
    }
  }
  if (nv == 0) {
    E.springs_ready = true;
    return cudaSuccess;
  }
  const int nwin = (nv + kSpringWindow - 1) / kSpringWindow, nslice = nwin * (kSpringWindow / 32);
  cudaError_t e = cudaSuccess;
  if (E.spring_end == nullptr) {
    // The slots, once per relation (synchronous).
    int* slots = nullptr;
    int total = 0;
    e = cudaMalloc(&slots, nslice * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&E.spring_place, (size_t)nv * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&E.spring_off, ((size_t)nslice + 1) * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&E.spring_row, (size_t)nwin * kSpringWindow * sizeof(int));
    if (e == cudaSuccess) {
      spring_window_kernel<<<nwin, kSpringWindow, 0, st>>>(nv, tets->vindex.order, E.row_off, E.spring_row,
                                                         E.spring_place, slots);
      e = exclusive_scan(nslice, slots, E.spring_off, st);
    }
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(&total, E.spring_off + nslice, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    const size_t n = std::max<size_t>(1, (size_t)total * 32);
    if (e == cudaSuccess) e = cudaMalloc(&E.rest[0], n * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&E.rest[1], n * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&E.spring_end, n * sizeof(int));
    cudaFree(slots);
    if (e != cudaSuccess) {
      cudaFree(E.spring_off);
      cudaFree(E.spring_row);
      cudaFree(E.spring_place);
      cudaFree(E.rest[0]);
      cudaFree(E.rest[1]);
      E.spring_off = E.spring_row = E.spring_place = E.spring_end = nullptr;
      E.rest[0] = E.rest[1] = nullptr;
      return e;
    }
    E.spring_slices = nslice;
  }
  const int grid = (nslice * 32 + kSpringThreads - 1) / kSpringThreads;
  if (f64)
    spring_fill_kernel<double, float><<<grid, kSpringThreads, 0, st>>>(
        nv, nslice, E.row_off, E.col, E.spring_row, E.spring_place, E.spring_off, static_cast<const double*>(X), E.spring_end,
        static_cast<double*>(E.rest[1]), static_cast<float*>(E.rest[0]));
  else
    spring_fill_kernel<float, double><<<grid, kSpringThreads, 0, st>>>(
        nv, nslice, E.row_off, E.col, E.spring_row, E.spring_place, E.spring_off, static_cast<const float*>(X), E.spring_end,
        static_cast<float*>(E.rest[0]), static_cast<double*>(E.rest[1]));
  e = cudaGetLastError();
  if (e == cudaSuccess) E.springs_ready = true;
  return e;
}

cudaError_t springs_run(ebb_rel_s* tets, void* q, void* qd, const void* mass, bool f64, double k, double dt, int steps,
                        double* energy, cudaStream_t st) {
  return f64 ? springs_run_t<double>(tets, (double*)q, (double*)qd, (const double*)mass, k, dt, steps, energy, st)
             : springs_run_t<float>(tets, (float*)q, (float*)qd, (const float*)mass, k, dt, steps, energy, st);
}

}  // namespace ebb
