// Row matrix: pattern (built on the device from the vertex index) and the
// element blocks its rows are summed from (see row_matrix.cuh).
//
// Assembly runs in two passes without atomics.  The element pass, one thread
// per tet, writes the blocks of the tet's six corner pairs to a record; the
// row pass (its user's kernel) sums, for every block of a row, the records
// the block's contribution list names, in increasing tet order: bitwise
// reproducible.  The diagonal block is minus the sum of its row's other
// blocks (K annihilates translations), so 6 of the 16 corner pairs are
// formed per tet, each once.
#include <algorithm>

#include "row_matrix.cuh"
#include "tet_io.cuh"
#include "tet_math.cuh"

namespace ebb {

namespace {

constexpr int kSortWarps = 4;
constexpr int kSortLen = 512;            // >= 3 * kRowMaxTets, a power of two
static_assert(kSortLen >= 3 * kRowMaxTets, "sort buffer");
constexpr int kScanThreads = 1024;

// The other corners of the tets around vertex v, sorted by (vertex, entry):
// buf[0 .. n) = vertex << 12 | 4 * (entry - off[v]) + corner; returns n.  One
// warp; n <= 3 * kRowMaxTets (larger rows return -1).
__device__ __forceinline__ int sort_row(int v, const int* __restrict__ off, const int* __restrict__ ent,
                                        const int4* __restrict__ keys, unsigned long long* buf) {
  const int lane = threadIdx.x & 31;
  const int e0 = off[v], ne = off[v + 1] - e0;
  if (ne > kRowMaxTets) return -1;
  const int n = 3 * ne;
  int P = 32;
  while (P < n) P <<= 1;
  for (int x = lane; x < P; x += 32) {
    unsigned long long key = ~0ull;
    if (x < n) {
      const int le = x / 3, r = x - 3 * le;
      const int code = ent[e0 + le];
      const int a = code & 3;
      const int b = r + (r >= a ? 1 : 0);
      const int4 k = keys[code >> 2];
      const int j = b == 0 ? k.x : (b == 1 ? k.y : (b == 2 ? k.z : k.w));
      key = ((unsigned long long)(unsigned)j << 12) | (unsigned)(4 * le + b);
    }
    buf[x] = key;
  }
  __syncwarp();
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = lane; i < P / 2; i += 32) {
        const int lo = ((i & ~(j - 1)) << 1) | (i & (j - 1));
        const int hi = lo | j;
        const unsigned long long x = buf[lo], y = buf[hi];
        if ((x > y) == ((lo & k) == 0)) {
          buf[lo] = y;
          buf[hi] = x;
        }
      }
      __syncwarp();
    }
  return n;
}

// Row lengths in blocks, the diagonal one included; *too_long is set when a
// vertex has more than kRowMaxTets tets.
__global__ void __launch_bounds__(32 * kSortWarps)
row_length_kernel(int nv, const int* __restrict__ off, const int* __restrict__ ent, const int4* __restrict__ keys,
                  int* len, int* too_long) {
  __shared__ unsigned long long s[kSortWarps][kSortLen];
  const int v = blockIdx.x * kSortWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (v >= nv) return;
  unsigned long long* buf = s[threadIdx.x >> 5];
  const int n = sort_row(v, off, ent, keys, buf);
  int heads = 0;
  for (int x = lane; x < n; x += 32) heads += x == 0 || (buf[x] >> 12) != (buf[x - 1] >> 12);
  heads = __reduce_add_sync(0xffffffffu, heads);
  if (lane == 0) {
    len[v] = 1 + heads;
    if (n < 0) *too_long = 1;
  }
}

// One block per window: rows sorted by decreasing length (ties in order of
// first use), the slices they make up in alternating quads, where each vertex
// went, and the slices' slot counts.
__global__ void __launch_bounds__(kWindowRows)
window_kernel(int nv, const int* __restrict__ order, const int* __restrict__ len, int* row_of, int* place,
              int* slots) {
  __shared__ int s_len[kWindowRows];
  const int i = threadIdx.x;
  const int x = blockIdx.x * kWindowRows + i;
  const int v = x < nv ? order[x] : -1;
  const int l = v >= 0 ? len[v] : 0;
  s_len[i] = l;
  __syncthreads();
  int rank = 0;
  for (int j = 0; j < kWindowRows; ++j) rank += s_len[j] > l || (s_len[j] == l && j < i);
  // slices by decreasing length; quads of them alternate from both ends
  const int sl = rank / kSliceRows, quad = sl / 4;
  const int pos = 4 * (quad < kWindowSlices / 8 ? 2 * quad : 2 * (kWindowSlices / 4 - 1 - quad) + 1) + sl % 4;
  const int at = (blockIdx.x * kWindowSlices + pos) * kSliceRows + rank % kSliceRows;
  row_of[at] = v;
  if (v >= 0) place[v] = at;
  if (rank % kSliceRows == 0) slots[blockIdx.x * kWindowSlices + pos] = l;
}

// Exclusive sums of n counts into out[0 .. n], by one block.
__global__ void __launch_bounds__(kScanThreads)
scan_kernel(int n, const int* __restrict__ in, int* out) {
  __shared__ int s_warp[kScanThreads / 32];
  __shared__ int s_run;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_run = 0;
  __syncthreads();
  for (int b = 0; b < n; b += kScanThreads) {
    const int i = b + threadIdx.x;
    const int x = i < n ? in[i] : 0;
    int inc = x;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) s_warp[w] = inc;
    __syncthreads();
    if (w == 0) {
      int t = s_warp[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += y;
      }
      s_warp[lane] = t;
    }
    __syncthreads();
    const int base = s_run + (w > 0 ? s_warp[w - 1] : 0);
    if (i < n) out[i] = base + inc - x;
    __syncthreads();
    if (threadIdx.x == kScanThreads - 1) s_run = base + inc;
    __syncthreads();
  }
  if (threadIdx.x == 0) out[n] = s_run;
}

// Columns and contribution lists.  Warp per row: the row's 3 x tets entries in
// sorted order are the contributions of its blocks, consecutive per block.
__global__ void __launch_bounds__(32 * kSortWarps)
row_fill_kernel(int nv, const int* __restrict__ off, const int* __restrict__ ent, const int4* __restrict__ keys,
                const int* __restrict__ place, const int* __restrict__ slice_off, int* col, int2* crange,
                int* slot_slice, int* contrib) {
  __shared__ unsigned long long s[kSortWarps][kSortLen];
  const int v = blockIdx.x * kSortWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (v >= nv) return;
  unsigned long long* buf = s[threadIdx.x >> 5];
  const int n = sort_row(v, off, ent, keys, buf);
  const int c0 = 3 * off[v];
  const int sl = place[v] / kSliceRows, i = place[v] - sl * kSliceRows;
  const int q0 = slice_off[sl], nk = slice_off[sl + 1] - q0;
  if (lane == 0) col[(size_t)q0 * kSliceRows + i] = v;
  if (i == 0)   // the slice's longest row
    for (int r = lane; r < nk; r += 32) slot_slice[q0 + r] = sl;
  int k = 1;
  for (int b = 0; b < n; b += 32) {
    const int x = b + lane;
    bool head = false;
    int j = 0;
    if (x < n) {
      const unsigned long long key = buf[x];
      j = (int)(key >> 12);
      head = x == 0 || (buf[x - 1] >> 12) != (key >> 12);
      const int le = (int)(key & 0xfffu) >> 2, cb = (int)(key & 3u);
      const int code = ent[off[v] + le];
      const int ca = code & 3, lo = min(ca, cb), hi = max(ca, cb);
      const int pair = lo == 0 ? hi - 1 : lo + hi;   // 01 02 03 12 13 23
      contrib[(size_t)c0 + x] = 16 * (code >> 2) + 2 * pair + (ca > cb ? 1 : 0);
    }
    const unsigned m = __ballot_sync(0xffffffffu, head);
    if (head) {
      const size_t at = (size_t)(q0 + k + __popc(m & ((1u << lane) - 1u))) * kSliceRows + i;
      int end = x + 1;
      while (end < n && (int)(buf[end] >> 12) == j) ++end;
      col[at] = j;
      crange[at] = make_int2(c0 + x, c0 + end);
    }
    k += __popc(m);
  }
  for (int r = k + lane; r < nk; r += 32) col[(size_t)(q0 + r) * kSliceRows + i] = v;
}

// ---- element pass ---------------------------------------------------------
// K_ab[c][d] of corners a < b (b_a = row a-1 of Dm^-1, b_0 = minus their sum):
//   StVK: V (delta_cd b_a.S b_b + mu (F F^T)_cd b_a.b_b + mu r_b,c r_a,d
//            + lam r_b,d r_a,c),   r_a = F b_a
//   NH:   V (mu delta_cd b_a.b_b + (mu - lam ln J) h_b,c h_a,d + lam h_b,d h_a,c),
//         h_a = F^-T b_a.
// FP64: bound by the FP64 pipe (about 400 FP64 instructions per tet at 530
// G/s); the 512 B stored per tet ride along.
constexpr int kElemThreads = 64;

template <typename T, int MODEL, bool AOS, bool FORCE>
__global__ void __launch_bounds__(kElemThreads)
element_block_kernel(int nt, int nv, const int4* __restrict__ keys, const int* __restrict__ perm, TetStreams<T> s,
                     T mu0, T lam0, const T* __restrict__ u, T* __restrict__ elem, int* err) {
  const int t = blockIdx.x * kElemThreads + threadIdx.x;
  if (t >= nt) return;
  const int4 k4 = keys[t];
  const int kk[4] = {k4.x, k4.y, k4.z, k4.w};
  T B[9], V, mu, lam;
  load_tet(s, nt, t, mu0, lam0, B, V, mu, lam);
  T Du[9], Dw[9];
  MapIO<T> io;
  io.u = u;
  load_edges<T, OP_FORCE, AOS>(io, nv, kk, Du, Dw);
  T G[9];
  mm(Du, B, G);
  T* rec = elem + (size_t)t * kElemLen;
  // The volume goes into the Lame parameters once, so that every product below
  // carries it.  vec[a]: r_a or h_a; bab: V mu b_a.b_b and bSb: V b_a.S b_b in
  // the pair order.
  const T vmu = V * mu, vlam = V * lam;
  T vec[4][3], bab[6], bSb[6], FFt[6], f[9];
  T c1, c2 = vlam;
  // b_a . b_b of corners 1..3: M = B B^T
  T M[9];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j)
      M[i * 3 + j] = M[j * 3 + i] = B[i * 3] * B[j * 3] + B[i * 3 + 1] * B[j * 3 + 1] + B[i * 3 + 2] * B[j * 3 + 2];
  if (MODEL == EBB_STVK) {
    // V S = 2 V mu E + V lam tr(E) I, 2 E = G + G^T + G^T G
    T S[6];   // 00 01 02 11 12 22
    T e2[6];
    {
      int q = 0;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j)
          e2[q++] = G[i] * G[j] + (G[3 + i] * G[3 + j] + (G[6 + i] * G[6 + j] + (G[i * 3 + j] + G[j * 3 + i])));
    }
    const T ltr = T(0.5) * vlam * (e2[0] + e2[3] + e2[5]);
#pragma unroll
    for (int q = 0; q < 6; ++q) S[q] = (q == 0 || q == 3 || q == 5) ? vmu * e2[q] + ltr : vmu * e2[q];
    T F[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) F[i] = G[i] + ((i % 4 == 0) ? T(1) : T(0));
    {
      int q = 0;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j)
          FFt[q++] = F[i * 3] * F[j * 3] + F[i * 3 + 1] * F[j * 3 + 1] + F[i * 3 + 2] * F[j * 3 + 2];
    }
    T N[9];   // V b_a . S b_b of corners 1..3
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const T b0 = B[a * 3], b1 = B[a * 3 + 1], b2 = B[a * 3 + 2];
      const T Sb[3] = {S[0] * b0 + S[1] * b1 + S[2] * b2, S[1] * b0 + S[3] * b1 + S[4] * b2,
                       S[2] * b0 + S[4] * b1 + S[5] * b2};
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        vec[a + 1][i] = F[i * 3] * b0 + F[i * 3 + 1] * b1 + F[i * 3 + 2] * b2;
        // f_a = -V P b_a = -F (V S b_a); F = I + G as in S + G S
        if (FORCE) f[3 * a + i] = -(Sb[i] + (G[i * 3] * Sb[0] + G[i * 3 + 1] * Sb[1] + G[i * 3 + 2] * Sb[2]));
      }
#pragma unroll
      for (int b = a; b < 3; ++b)
        N[a * 3 + b] = N[b * 3 + a] = Sb[0] * B[b * 3] + Sb[1] * B[b * 3 + 1] + Sb[2] * B[b * 3 + 2];
    }
    c1 = vmu;
#pragma unroll
    for (int b = 0; b < 3; ++b) bSb[b] = -(N[b] + N[3 + b] + N[6 + b]);
    bSb[3] = N[1];
    bSb[4] = N[2];
    bSb[5] = N[5];
  } else {
    NhState<T> sn;
    if (!nh_state(G, sn)) {
      raise_error(err, EBB_ERR_INVERTED, perm[t]);
#pragma unroll
      for (int i = 0; i < kElemLen; ++i) rec[i] = T(0);
      return;
    }
    if (FORCE) {
      T P[9];
      nh_P(sn, vmu, vlam, P);
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c)
          f[3 * a + c] = -(P[c * 3] * B[a * 3] + P[c * 3 + 1] * B[a * 3 + 1] + P[c * 3 + 2] * B[a * 3 + 2]);
    }
    c1 = vmu - vlam * sn.lnJ;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int i = 0; i < 3; ++i)
        vec[a + 1][i] = sn.FiT[i * 3] * B[a * 3] + sn.FiT[i * 3 + 1] * B[a * 3 + 1] + sn.FiT[i * 3 + 2] * B[a * 3 + 2];
  }
  if (FORCE) {
#pragma unroll
    for (int i = 0; i < 9; ++i) rec[kElemForce + i] = f[i];
  }
#pragma unroll
  for (int b = 0; b < 3; ++b) bab[b] = -vmu * (M[b] + M[3 + b] + M[6 + b]);
  bab[3] = vmu * M[1];
  bab[4] = vmu * M[2];
  bab[5] = vmu * M[5];
#pragma unroll
  for (int i = 0; i < 3; ++i) vec[0][i] = -(vec[1][i] + vec[2][i] + vec[3][i]);
#pragma unroll
  for (int b = 1; b < 4; ++b) {
    T v1[3], v2[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      v1[i] = c1 * vec[b][i];
      v2[i] = c2 * vec[b][i];
    }
#pragma unroll
    for (int a = 0; a < b; ++a) {
      const int p = a == 0 ? b - 1 : a + b;
      T x[6];   // the part that is symmetric in (c, d)
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        const bool dg = q == 0 || q == 3 || q == 5;
        if (MODEL == EBB_STVK)
          x[q] = dg ? bab[p] * FFt[q] + bSb[p] : bab[p] * FFt[q];
        else
          x[q] = dg ? bab[p] : T(0);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const int lo = c < d ? c : d, hi = c < d ? d : c;
          const int q = lo == 0 ? hi : (lo == 1 ? 2 + hi : 5);   // 00 01 02 11 12 22
          rec[9 * p + 3 * c + d] = v1[c] * vec[a][d] + (v2[d] * vec[a][c] + x[q]);
        }
    }
  }
}

template <typename T>
const TetStreams<T>& elem_streams(const ebb_rel_s* rel);
template <>
const TetStreams<float>& elem_streams<float>(const ebb_rel_s* rel) { return rel->s32; }
template <>
const TetStreams<double>& elem_streams<double>(const ebb_rel_s* rel) { return rel->s64; }

template <typename T, int MODEL, bool AOS>
void launch_elem(ebb_rel_s* rel, T mu0, T lam0, const T* u, bool force, T* elem, cudaStream_t st) {
  const int nt = (int)rel->size, nv = (int)rel->verts->size;
  const int grid = (nt + kElemThreads - 1) / kElemThreads;
  if (force)
    element_block_kernel<T, MODEL, AOS, true><<<grid, kElemThreads, 0, st>>>(
        nt, nv, rel->keys, rel->tet_perm, elem_streams<T>(rel), mu0, lam0, u, elem, rel->ctx->d_err);
  else
    element_block_kernel<T, MODEL, AOS, false><<<grid, kElemThreads, 0, st>>>(
        nt, nv, rel->keys, rel->tet_perm, elem_streams<T>(rel), mu0, lam0, u, elem, rel->ctx->d_err);
}

}  // namespace

template <typename T>
cudaError_t launch_element_blocks(ebb_rel_s* rel, int model, T mu0, T lam0, const T* u, bool aos, bool force, T* elem,
                                  cudaStream_t st) {
  if (rel->size == 0) return cudaSuccess;
  if constexpr (sizeof(T) == 4) {
    if (aos) {
      if (model == EBB_STVK)
        launch_elem<T, EBB_STVK, true>(rel, mu0, lam0, u, force, elem, st);
      else
        launch_elem<T, EBB_NEOHOOKEAN, true>(rel, mu0, lam0, u, force, elem, st);
      return cudaGetLastError();
    }
  }
  if (aos) return cudaErrorInvalidValue;
  if (model == EBB_STVK)
    launch_elem<T, EBB_STVK, false>(rel, mu0, lam0, u, force, elem, st);
  else
    launch_elem<T, EBB_NEOHOOKEAN, false>(rel, mu0, lam0, u, force, elem, st);
  return cudaGetLastError();
}
template cudaError_t launch_element_blocks<double>(ebb_rel_s*, int, double, double, const double*, bool, bool, double*,
                                                   cudaStream_t);

void free_row_matrix(ebb_rel_s* tets) {
  RowMatrix* m = tets->rows;
  if (!m) return;
  cudaFree(m->slice_off);
  cudaFree(m->row_of);
  cudaFree(m->col);
  cudaFree(m->crange);
  cudaFree(m->slot_slice);
  cudaFree(m->contrib);
  delete m;
  tets->rows = nullptr;
}

ebb_status_t ensure_row_pattern(ebb_ctx_s* ctx, ebb_rel_s* tets, cudaStream_t st) {
  if (tets->rows) return EBB_OK;
  RowMatrix* m = new RowMatrix();
  tets->rows = m;
  m->state = -1;
  const int nv = (int)tets->verts->size;
  const int64_t nt = tets->size;
  // contribution codes are 16 t + ..., their offsets 12 t + ...
  if (tets->vindex.off == nullptr || nv == 0 || nt > (int64_t)0x7fffffff / 16) return EBB_OK;
  const int nwin = (nv + kWindowRows - 1) / kWindowRows;
  m->nslice = nwin * kWindowSlices;
  // scratch: row lengths, places, slot counts, the too-long flag
  int* tmp = nullptr;
  const size_t ntmp = 2 * (size_t)nv + m->nslice + 1;
  cudaError_t e = cudaMalloc(&tmp, ntmp * sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&m->slice_off, ((size_t)m->nslice + 1) * sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&m->row_of, (size_t)nwin * kWindowRows * sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&m->contrib, std::max<size_t>(1, (size_t)nt * 12) * sizeof(int));
  int nsm = 0;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device);
  m->grid = std::min({std::max(nsm, 1), kRowMaxGrid, m->nslice});
  int host[2] = {0, 0};   // total slots, too-long flag
  int *len = tmp, *place = tmp + nv, *slots = tmp + 2 * (size_t)nv, *flag = slots + m->nslice;
  const int sort_grid = (nv + kSortWarps - 1) / kSortWarps;
  if (e == cudaSuccess) {
    const VertexIndex& x = tets->vindex;
    e = cudaMemsetAsync(flag, 0, sizeof(int), st);
    row_length_kernel<<<sort_grid, 32 * kSortWarps, 0, st>>>(nv, x.off, x.ent, tets->keys, len, flag);
    window_kernel<<<nwin, kWindowRows, 0, st>>>(nv, x.order, len, m->row_of, place, slots);
    scan_kernel<<<1, kScanThreads, 0, st>>>(m->nslice, slots, m->slice_off);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(&host[0], m->slice_off + m->nslice, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&host[1], flag, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  bool apply = e == cudaSuccess && host[1] == 0;
  if (apply) {
    m->nslots = host[0];
    const size_t n = std::max<size_t>(1, (size_t)m->nslots * kSliceRows);
    e = cudaMalloc(&m->col, n * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&m->crange, n * sizeof(int2));
    if (e == cudaSuccess) e = cudaMalloc(&m->slot_slice, std::max<size_t>(1, (size_t)m->nslots) * sizeof(int));
    // rows that hold no vertex: a valid column, no contributions
    if (e == cudaSuccess) e = cudaMemsetAsync(m->col, 0, n * sizeof(int), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->crange, 0, n * sizeof(int2), st);
    if (e == cudaSuccess) {
      const VertexIndex& x = tets->vindex;
      row_fill_kernel<<<sort_grid, 32 * kSortWarps, 0, st>>>(nv, x.off, x.ent, tets->keys, place, m->slice_off, m->col,
                                                             m->crange, m->slot_slice, m->contrib);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    apply = e == cudaSuccess;
  }
  cudaFree(tmp);
  if (!apply) {
    cudaFree(m->slice_off);
    cudaFree(m->row_of);
    cudaFree(m->col);
    cudaFree(m->crange);
    cudaFree(m->slot_slice);
    cudaFree(m->contrib);
      *m = RowMatrix();
    m->state = -1;
    if (e == cudaSuccess || e == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      return EBB_OK;
    }
    return cuda_check(ctx, e, "building the row pattern");
  }
  m->state = 1;
  return EBB_OK;
}

}  // namespace ebb
