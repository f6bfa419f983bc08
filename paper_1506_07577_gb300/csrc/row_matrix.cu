// Row matrix: pattern (built on the device from the vertex index) and the
// element blocks its rows are summed from (see row_matrix.cuh).
//
// Assembly runs in two passes without atomics.  The element pass, one thread
// per tet, writes the blocks of the tet's six corner pairs to a record; the
// row pass (its user's kernel) sums, for every block of a row, the records
// the block's contribution list names, in increasing tet order: bitwise
// reproducible.  The diagonal block is minus the sum of its row's other
// blocks (K annihilates translations), so 6 of the 16 corner pairs are
// formed per tet, each once.  Measured on the 64^3 mesh (1.31 M tets, FP32):
// records 80 us, rows 143 us, product 45 us; one atomic per block entry and
// tet took 716 us.
#include <algorithm>

#include "row_matrix.cuh"
#include "tet_io.cuh"
#include "tet_math.cuh"

namespace ebb {

namespace {

constexpr int kSortWarps = 4;
constexpr int kShortTets = 40;           // rows of up to so many tets take the small tables
constexpr int kScanThreads = 1024;

// Columns and contribution lists of a row, one warp per vertex.  The other
// corners of the vertex's tets go into a small hash table in shared memory;
// the distinct vertices, ranked by number, are the row's columns, and a
// corner's place in its column's list is the count of equal corners before
// it, so that the lists keep the order of the vertex index (increasing tets).
// Row v owns [3 off[v], 3 off[v + 1]) of contrib, colv and colb: its
// contributions column by column, its columns, and where each column's list
// begins.  len[v]: blocks of the row, the diagonal one included.  A vertex of
// more than kRowMaxTets tets sets *too_long.  Launched for rows of up to
// kShortTets tets (LONG false), then for the longer ones, whose tables leave
// room for few warps.
template <int MAXT, int HASH, bool LONG>
__global__ void __launch_bounds__(32 * kSortWarps)
row_columns_kernel(int nv, const int* __restrict__ off, const int* __restrict__ ent, const int4* __restrict__ keys,
                   int* __restrict__ contrib, int* __restrict__ colv, int* __restrict__ colb, int* __restrict__ len,
                   int* too_long) {
  static_assert(HASH >= 6 * MAXT && (HASH & (HASH - 1)) == 0, "hash load");
  constexpr int G = (3 * MAXT + 31) / 32;
  __shared__ int s_key[kSortWarps][HASH];
  __shared__ short s_cnt[kSortWarps][HASH], s_uniq[kSortWarps][3 * MAXT], s_at[kSortWarps][3 * MAXT];
  __shared__ short s_slot[kSortWarps][3 * MAXT];
  const int v = blockIdx.x * kSortWarps + (threadIdx.x >> 5);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (v >= nv) return;
  int* key = s_key[w];
  short *cnt = s_cnt[w], *uniq = s_uniq[w], *at = s_at[w], *slot_of = s_slot[w];
  const int e0 = off[v], ne = off[v + 1] - e0;
  if (LONG ? ne <= kShortTets : ne > MAXT) return;
  if (LONG && ne > MAXT) {
    if (lane == 0) {
      len[v] = 1;
      *too_long = 1;
    }
    return;
  }
  const int n = 3 * ne;
  int size = 64;
  while (size < 2 * n) size <<= 1;
  for (int x = lane; x < size; x += 32) {
    key[x] = -1;
    cnt[x] = 0;
  }
  __syncwarp();
  // insert; slot_of[x] and at[x] (entries of the same vertex before x)
  for (int b = 0; b < n; b += 32) {
    const int x = b + lane;
    const unsigned on = __ballot_sync(0xffffffffu, x < n);
    if (x < n) {
      const int le = x / 3, r = x - 3 * le;
      const int code = ent[e0 + le];
      const int c = r + (r >= (code & 3) ? 1 : 0);
      const int4 k = keys[code >> 2];
      const int j = c == 0 ? k.x : (c == 1 ? k.y : (c == 2 ? k.z : k.w));
      unsigned h = ((unsigned)j * 2654435761u) >> 16 & (unsigned)(size - 1);
      while (true) {
        const int old = atomicCAS(&key[h], -1, j);
        if (old == -1 || old == j) break;
        h = (h + 1) & (unsigned)(size - 1);
      }
      slot_of[x] = (short)h;
      const unsigned same = __match_any_sync(on, j);
      const int before = cnt[h];
      __syncwarp(on);
      at[x] = (short)(before + __popc(same & ((1u << lane) - 1u)));
      if (lane == __ffs(same) - 1) cnt[h] = (short)(before + __popc(same));
    }
    __syncwarp();
  }
  // the distinct vertices' slots
  int m = 0;
  for (int b = 0; b < size; b += 32) {
    const bool used = key[b + lane] >= 0;
    const unsigned u = __ballot_sync(0xffffffffu, used);
    if (used) uniq[m + __popc(u & ((1u << lane) - 1u))] = (short)(b + lane);
    m += __popc(u);
  }
  __syncwarp();
  // rank by vertex number and start of each list; cnt becomes the start
  const int c0 = 3 * e0;
  int starts[G];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int x = 32 * g + lane;
    starts[g] = 0;
    if (x < m) {
      const int j = key[uniq[x]];
      int rank = 0;
      for (int y = 0; y < m; ++y) {
        const int o = uniq[y];
        if (key[o] < j) {
          ++rank;
          starts[g] += cnt[o];
        }
      }
      colv[(size_t)c0 + rank] = j;
      colb[(size_t)c0 + rank] = c0 + starts[g];
    }
  }
  __syncwarp();
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int x = 32 * g + lane;
    if (x < m) cnt[uniq[x]] = (short)starts[g];
  }
  __syncwarp();
  for (int x = lane; x < n; x += 32) {
    const int le = x / 3, r = x - 3 * le;
    const int code = ent[e0 + le], ca = code & 3;
    const int cb = r + (r >= ca ? 1 : 0);
    const int lo = min(ca, cb), hi = max(ca, cb);
    const int pair = lo == 0 ? hi - 1 : lo + hi;   // 01 02 03 12 13 23
    contrib[(size_t)c0 + cnt[slot_of[x]] + at[x]] = 16 * (code >> 2) + 2 * pair + (ca > cb ? 1 : 0);
  }
  if (lane == 0) len[v] = 1 + m;
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

// The rows' columns in slot order; eight lanes per row.
__global__ void __launch_bounds__(256)
row_fill_kernel(int nv, const int* __restrict__ off, const int* __restrict__ len, const int* __restrict__ colv,
                const int* __restrict__ place, const int* __restrict__ slice_off, int* col) {
  const int v = (blockIdx.x * 256 + threadIdx.x) >> 3, lane = threadIdx.x & 7;
  if (v >= nv) return;
  const int c0 = 3 * off[v], m = len[v] - 1;
  const int sl = place[v] / kSliceRows, i = place[v] - sl * kSliceRows;
  const int q0 = slice_off[sl], nk = slice_off[sl + 1] - q0;
  for (int k = lane; k < nk; k += 8)
    col[(size_t)(q0 + k) * kSliceRows + i] = k > 0 && k <= m ? colv[c0 + k - 1] : v;
}

// Place of the first of n increasing columns that is >= v.
__device__ __forceinline__ int lower_bound(const int* __restrict__ col, int n, int v) {
  int lo = 0;
  while (lo < n) {
    const int mid = (lo + n) >> 1;
    if (col[mid] < v)
      lo = mid + 1;
    else
      n = mid;
  }
  return lo;
}

// Block pairs (RowMatrix::pairs) of the rows of each slice, one warp per slice:
// first their number (FILL false), then the pairs.
template <bool FILL>
__global__ void __launch_bounds__(256)
row_pair_kernel(int nslice, const int* __restrict__ row_of, const int* __restrict__ off, const int* __restrict__ len,
                const int* __restrict__ colv, const int* __restrict__ colb, const int* __restrict__ place,
                const int* __restrict__ slice_off, int* count, const int* __restrict__ pair_off, int4* pairs) {
  const int s = (blockIdx.x * 256 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (s >= nslice) return;
  const int v = lane < kSliceRows ? row_of[s * kSliceRows + lane] : -1;
  int c0 = 0, m = 0, lo = 0;
  if (v >= 0) {
    c0 = 3 * off[v];
    m = len[v] - 1;
    lo = lower_bound(colv + c0, m, v);
  }
  const int n = m - lo;
  int inc = n;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if constexpr (!FILL) {
    if (lane == 31) count[s] = inc;
  } else {
    const int base = pair_off[s] + inc - n;
    for (int i = 0; i < kSliceRows; ++i) {
      const int vi = __shfl_sync(0xffffffffu, v, i), ci = __shfl_sync(0xffffffffu, c0, i);
      const int mi = __shfl_sync(0xffffffffu, m, i), li = __shfl_sync(0xffffffffu, lo, i);
      const int bi = __shfl_sync(0xffffffffu, base, i);
      for (int k = li + lane; k < mi; k += 32) {
        const int w = colv[ci + k];
        int mate = -1;
        if (w != vi) {
          const int pw = place[w], sw = pw / kSliceRows;
          const int kw = lower_bound(colv + 3 * off[w], len[w] - 1, vi);
          mate = (slice_off[sw] + 1 + kw) * kSliceRows + pw - sw * kSliceRows;
        }
        pairs[bi + k - li] = make_int4((slice_off[s] + 1 + k) * kSliceRows + i, mate, colb[ci + k],
                                       k + 1 < mi ? colb[ci + k + 1] : 3 * off[vi + 1]);
      }
    }
  }
}

// ---- element pass ---------------------------------------------------------
// K_ab[c][d] of corners a < b (b_a = row a-1 of Dm^-1, b_0 = minus their sum):
//   StVK: V (delta_cd b_a.S b_b + mu (F F^T)_cd b_a.b_b + mu r_b,c r_a,d
//            + lam r_b,d r_a,c),   r_a = F b_a
//   NH:   V (mu delta_cd b_a.b_b + (mu - lam ln J) h_b,c h_a,d + lam h_b,d h_a,c),
//         h_a = F^-T b_a.
// FP64: bound by the FP64 pipe (about 400 FP64 instructions per tet at 530
// G/s); the 512 B stored per tet ride along.
// FP32: bound by the records' writes, which go through shared memory a warp
// at a time, so that each store is a line of consecutive words (written
// straight from the threads, a store touches 32 lines).
constexpr int kElemThreads = 64;

template <typename T, int MODEL, bool AOS, bool FORCE>
__device__ __forceinline__ void element_record(int t, int nt, int nv, const int4* __restrict__ keys,
                                               const int* __restrict__ perm, const TetStreams<T>& s, T mu0, T lam0,
                                               const T* __restrict__ u, T* rec, int* err) {
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
      for (int c = 0; c < 3; ++c) {
        T k[4];
        k[3] = FORCE && 3 * p + c < 9 ? f[3 * p + c < 9 ? 3 * p + c : 0] : T(0);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const int lo = c < d ? c : d, hi = c < d ? d : c;
          const int q = lo == 0 ? hi : (lo == 1 ? 2 + hi : 5);   // 00 01 02 11 12 22
          k[d] = v1[c] * vec[a][d] + (v2[d] * vec[a][c] + x[q]);
        }
        if constexpr (sizeof(T) == 8) {
          double2* out = reinterpret_cast<double2*>(rec + 4 * (3 * p + c));
          out[0] = make_double2(k[0], k[1]);
          out[1] = make_double2(k[2], k[3]);
        } else {
#pragma unroll
          for (int d = 0; d < 4; ++d) rec[4 * (3 * p + c) + d] = k[d];
        }
      }
    }
  }
}

template <typename T, int MODEL, bool AOS, bool FORCE>
__global__ void __launch_bounds__(kElemThreads)
element_block_kernel(int nt, int nv, const int4* __restrict__ keys, const int* __restrict__ perm, TetStreams<T> s,
                     T mu0, T lam0, const T* __restrict__ u, T* __restrict__ elem, int* err) {
  constexpr bool STAGE = sizeof(T) == 4;
  constexpr int L = kElemLen;
  __shared__ T s_rec[STAGE ? kElemThreads : 1][STAGE ? L + 1 : 1];
  const int t = blockIdx.x * kElemThreads + threadIdx.x;
  if (!STAGE && t >= nt) return;
  const int tt = t < nt ? t : nt - 1;
  T* rec = STAGE ? &s_rec[STAGE ? threadIdx.x : 0][0] : elem + (size_t)t * L;
  element_record<T, MODEL, AOS, FORCE>(tt, nt, nv, keys, perm, s, mu0, lam0, u, rec, err);
  if constexpr (STAGE) {
    __syncwarp();
    const int w0 = (int)threadIdx.x & ~31, lane = threadIdx.x & 31;
    const int t0 = (int)blockIdx.x * kElemThreads + w0;
    const int n = warp_tets(t0, nt) * L;   // words of the warp's records
    T* dst = elem + (size_t)t0 * L;
    for (int x = lane; x < n; x += 32) dst[x] = s_rec[w0 + x / L][x % L];
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
  if (sizeof(T) == 8 && force)
    element_block_kernel<T, MODEL, AOS, sizeof(T) == 8><<<grid, kElemThreads, 0, st>>>(
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

// ---- assembled K for ebb_assemble_tet_K / ebb_spmv_tet_K --------------------
namespace {

constexpr int kAsmThreads = 256;

// Column c of a 3x3 block whose row c this lane holds, rows in lanes row0 + c.
template <typename T>
__device__ __forceinline__ void transpose3(const T (&x)[3], int c, int row0, T (&y)[3]) {
  // lane c gets entry c of lanes c + 1 and c + 2 (mod 3)
  const int n1 = c == 2 ? 0 : c + 1, n2 = c == 0 ? 2 : c - 1;
  const T give1 = c == 0 ? x[2] : (c == 1 ? x[0] : x[1]);
  const T give2 = c == 0 ? x[1] : (c == 1 ? x[2] : x[0]);
  const T own = c == 0 ? x[0] : (c == 1 ? x[1] : x[2]);
  const T got1 = __shfl_sync(0xffffffffu, give1, row0 + n1);
  const T got2 = __shfl_sync(0xffffffffu, give2, row0 + n2);
  y[0] = c == 0 ? own : (c == 1 ? got2 : got1);
  y[1] = c == 1 ? own : (c == 2 ? got2 : got1);
  y[2] = c == 2 ? own : (c == 0 ? got2 : got1);
}

// Off-diagonal blocks of scale * K, ten block pairs per warp, a lane per row of
// the first block: the sum of the pair's contributions in increasing tet order,
// stored as it is and, transposed, at its mate's place.  K is symmetric, and both
// orders would add the same values in the same order.  Blocks of a record are
// stored for a < b; the other way round they are transposed.  FP32: a lane loads
// its row of the stored block, one 16-byte load per contribution (the loads'
// lines bound the kernel: with one load per entry or nine lanes per block it took
// 3 times as long), adds stored and transposed contributions apart and swaps the
// transposed sums between its row's lanes at the end.  FP64: the adds bound it,
// so transposed entries are loaded as such.  Measured against each block summed
// by itself: 64^3 mesh, FP32 182 -> 143 us (160 with the mates stored entry by
// entry, 30 sectors a store instead of 10); 32^3 mesh, FP64 73 -> 38 us.
template <typename T, typename PT>
__global__ void __launch_bounds__(kAsmThreads)
row_block_kernel(int npair, const int4* __restrict__ pairs, const int* __restrict__ col,
                 const int* __restrict__ contrib, const T* __restrict__ elem, const PT* __restrict__ pin, T scale,
                 T* __restrict__ val) {
  const int64_t warp = ((int64_t)blockIdx.x * kAsmThreads + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int i = lane / 3, c = lane - 3 * i;
  const int64_t n = warp * kSliceRows + i;
  const bool own = lane < 3 * kSliceRows && n < npair;
  int4 p = own ? pairs[n] : make_int4(0, -1, 0, 0);
  bool zero = false, zero_mate = false;   // rows of pinned vertices
  if (pin != nullptr && own) {
    zero_mate = pin[col[p.x]] != 0;
    zero = p.y >= 0 ? pin[col[p.y]] != 0 : zero_mate;
    if (zero && zero_mate) p.w = p.z;
  }
  T x[3] = {T(0), T(0), T(0)};
  if constexpr (sizeof(T) == 4) {
    T xt[3] = {T(0), T(0), T(0)};
#pragma unroll 4
    for (int e = p.z; e < p.w; ++e) {
      const int code = contrib[e];
      const float4 k = __ldg(reinterpret_cast<const float4*>(elem + (size_t)(code >> 4) * kElemLen +
                                                             12 * ((code >> 1) & 7) + 4 * c));
      if (code & 1) {
        xt[0] += k.x;
        xt[1] += k.y;
        xt[2] += k.z;
      } else {
        x[0] += k.x;
        x[1] += k.y;
        x[2] += k.z;
      }
    }
    T y[3];
    transpose3(xt, c, lane - c, y);
#pragma unroll
    for (int d = 0; d < 3; ++d) x[d] += y[d];
  } else if (p.z < p.w) {
    auto rec_of = [&](int code, int& st) {
      const bool tr = (code & 1) != 0;
      st = tr ? 4 : 1;
      return elem + (size_t)(code >> 4) * kElemLen + 12 * ((code >> 1) & 7) + (tr ? c : 4 * c);
    };
    int st;
    const T* rec = rec_of(contrib[p.z], st);
#pragma unroll
    for (int d = 0; d < 3; ++d) x[d] = rec[d * st];
#pragma unroll 4
    for (int e = p.z + 1; e < p.w; ++e) {
      rec = rec_of(contrib[e], st);
#pragma unroll
      for (int d = 0; d < 3; ++d) x[d] += rec[d * st];
    }
  }
  T y[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) x[d] *= scale;
  transpose3(x, c, lane - c, y);
  if (!own) return;
  const int q = p.x / kSliceRows;
  T* at = val + (size_t)q * 96 + 3 * (p.x - q * kSliceRows) + c;
#pragma unroll
  for (int d = 0; d < 3; ++d) at[32 * d] = zero ? T(0) : x[d];
  if (p.y < 0) return;
  const int qm = p.y / kSliceRows;
  at = val + (size_t)qm * 96 + 3 * (p.y - qm * kSliceRows) + c;
#pragma unroll
  for (int d = 0; d < 3; ++d) at[32 * d] = zero_mate ? T(0) : y[d];
}

__device__ __forceinline__ float ld_once(const float* p) {
  float x;
  asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(x) : "l"(p));
  return x;
}
__device__ __forceinline__ double ld_once(const double* p) {
  double x;
  asm volatile("ld.global.nc.L1::no_allocate.f64 %0, [%1];" : "=d"(x) : "l"(p));
  return x;
}

// y_r += sum_j K_rj (w_j - w_r): the diagonal block, minus the sum of the row's
// others, is in the difference.  Warp per slice, lane per row and component,
// fixed order.  FP32: bound by the blocks' one pass through memory.
template <typename T, bool AOS>
__global__ void __launch_bounds__(kAsmThreads)
row_product_kernel(RowView m, int nv, const T* __restrict__ val, const T* __restrict__ w, T* y, const int* active) {
  if (active != nullptr && *active == 0) return;
  const int s = (blockIdx.x * kAsmThreads + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (s >= m.nslice || lane >= 3 * kSliceRows) return;
  const int i = lane / 3, c = lane - 3 * i;
  const int v = m.row_of[s * kSliceRows + i];
  if (v < 0) return;
  const int q0 = m.slice_off[s], nk = m.slice_off[s + 1] - q0;
  auto load = [&](int j, T (&x)[3]) {
    if constexpr (AOS) {
      const float4 f = reinterpret_cast<const float4*>(w)[j];
      x[0] = f.x;
      x[1] = f.y;
      x[2] = f.z;
    } else {
#pragma unroll
      for (int d = 0; d < 3; ++d) x[d] = w[(size_t)d * nv + j];
    }
  };
  // groups of U slots; the next group's columns are loaded a group ahead
  constexpr int U = 4;
  const int* col = m.col + (size_t)q0 * kSliceRows + i;
  const T* bv = val + (size_t)q0 * 96 + lane;
  int j[U];
#pragma unroll
  for (int g = 0; g < U; ++g) j[g] = 1 + g < nk ? col[(1 + g) * kSliceRows] : v;
  T wr[3];
  load(v, wr);
  T acc = T(0);
  for (int k = 1; k < nk; k += U) {
    T x[U][3], b[U][3];
#pragma unroll
    for (int g = 0; g < U; ++g) {
      const T* at = bv + (size_t)(k + g < nk ? k + g : 0) * 96;
#pragma unroll
      for (int d = 0; d < 3; ++d) b[g][d] = ld_once(at + 32 * d);
      load(j[g], x[g]);
    }
#pragma unroll
    for (int g = 0; g < U; ++g) j[g] = k + U + g < nk ? col[(k + U + g) * kSliceRows] : v;
#pragma unroll
    for (int g = 0; g < U; ++g)
      if (k + g < nk) {
#pragma unroll
        for (int d = 0; d < 3; ++d) acc += b[g][d] * (x[g][d] - wr[d]);
      }
  }
  y[AOS ? 4 * (size_t)v + c : (size_t)c * nv + v] += acc;
}

}  // namespace

template <typename T>
cudaError_t launch_row_blocks(const RowMatrix& m, const T* elem, const void* pin, int pin_bytes, T scale, T* val,
                              cudaStream_t st) {
  if (m.npair == 0) return cudaSuccess;
  const int64_t warps = ((int64_t)m.npair + kSliceRows - 1) / kSliceRows;
  const unsigned grid = (unsigned)((warps * 32 + kAsmThreads - 1) / kAsmThreads);
  if (pin_bytes == 4)
    row_block_kernel<T, int><<<grid, kAsmThreads, 0, st>>>(m.npair, m.pairs, m.col, m.contrib, elem,
                                                           static_cast<const int*>(pin), scale, val);
  else
    row_block_kernel<T, unsigned char><<<grid, kAsmThreads, 0, st>>>(
        m.npair, m.pairs, m.col, m.contrib, elem, static_cast<const unsigned char*>(pin), scale, val);
  return cudaGetLastError();
}
template cudaError_t launch_row_blocks<double>(const RowMatrix&, const double*, const void*, int, double, double*,
                                               cudaStream_t);

template <typename T>
cudaError_t launch_row_assemble(ebb_rel_s* rel, int model, T mu0, T lam0, const MapIO<T>& io, cudaStream_t st,
                                bool* done) {
  *done = false;
  const int p = sizeof(T) == 4 ? 0 : 1;
  RowMatrix* m = rel->rows;
  if (m == nullptr || m->val[p] == nullptr) {
    // first use: pattern and memory, never inside a stream capture
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &cs);
    if (e != cudaSuccess) return e;
    if (cs != cudaStreamCaptureStatusNone) return m != nullptr && m->state != 1 ? cudaSuccess
                                                                                : cudaErrorStreamCaptureUnsupported;
    if (ensure_row_pattern(rel->ctx, rel, st) != EBB_OK) return cudaErrorUnknown;
    m = rel->rows;
    if (m->state != 1) return cudaSuccess;
    e = cudaMalloc(&m->val[p], std::max<size_t>(1, (size_t)m->nslots * 96) * sizeof(T));
    if (e == cudaSuccess) e = cudaMalloc(&m->elem[p], std::max<size_t>(1, (size_t)rel->size * kElemLen) * sizeof(T));
    if (e == cudaSuccess) e = cudaMemsetAsync(m->val[p], 0, (size_t)m->nslots * 96 * sizeof(T), st);   // unused entries
    if (e != cudaSuccess) {
      cudaFree(m->val[p]);
      cudaFree(m->elem[p]);
      m->val[p] = m->elem[p] = nullptr;
      cudaGetLastError();
      return e == cudaErrorMemoryAllocation ? cudaSuccess : e;
    }
  }
  if (m->state != 1) return cudaSuccess;
  T* elem = static_cast<T*>(m->elem[p]);
  cudaError_t e = launch_element_blocks<T>(rel, model, mu0, lam0, io.u, io.aos, false, elem, st);
  if (e != cudaSuccess) return e;
  e = launch_row_blocks<T>(*m, elem, nullptr, 1, T(1), static_cast<T*>(m->val[p]), st);
  if (e != cudaSuccess) return e;
  *done = true;
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_row_product(ebb_rel_s* rel, const T* w, T* y, bool aos, const int* active, cudaStream_t st,
                               bool* done) {
  *done = false;
  const int p = sizeof(T) == 4 ? 0 : 1;
  const RowMatrix* m = rel->rows;
  if (m == nullptr || m->val[p] == nullptr) return cudaSuccess;
  const int nv = (int)rel->verts->size;
  const RowView view{m->nslice, m->slice_off, m->row_of, m->col};
  const int grid = (m->nslice * 32 + kAsmThreads - 1) / kAsmThreads;
  const T* val = static_cast<const T*>(m->val[p]);
  *done = true;
  if (aos) {
    if constexpr (sizeof(T) == 4) {
      row_product_kernel<T, true><<<grid, kAsmThreads, 0, st>>>(view, nv, val, w, y, active);
      return cudaGetLastError();
    }
    return cudaErrorInvalidValue;
  }
  row_product_kernel<T, false><<<grid, kAsmThreads, 0, st>>>(view, nv, val, w, y, active);
  return cudaGetLastError();
}

template cudaError_t launch_row_assemble<float>(ebb_rel_s*, int, float, float, const MapIO<float>&, cudaStream_t,
                                                bool*);
template cudaError_t launch_row_assemble<double>(ebb_rel_s*, int, double, double, const MapIO<double>&, cudaStream_t,
                                                 bool*);
template cudaError_t launch_row_product<float>(ebb_rel_s*, const float*, float*, bool, const int*, cudaStream_t,
                                               bool*);
template cudaError_t launch_row_product<double>(ebb_rel_s*, const double*, double*, bool, const int*, cudaStream_t,
                                                bool*);
template cudaError_t launch_element_blocks<double>(ebb_rel_s*, int, double, double, const double*, bool, bool, double*,
                                                   cudaStream_t);

cudaError_t exclusive_scan(int n, const int* in, int* out, cudaStream_t st) {
  scan_kernel<<<1, kScanThreads, 0, st>>>(n, in, out);
  return cudaGetLastError();
}

void free_row_matrix(ebb_rel_s* tets) {
  RowMatrix* m = tets->rows;
  if (!m) return;
  cudaFree(m->slice_off);
  cudaFree(m->row_of);
  cudaFree(m->col);
  cudaFree(m->pairs);
  cudaFree(m->contrib);
  for (int p = 0; p < 2; ++p) {
    cudaFree(m->val[p]);
    cudaFree(m->elem[p]);
  }
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
  // scratch: row lengths, places, slot counts, the too-long flag, columns
  int* tmp = nullptr;
  const size_t ntmp = 2 * (size_t)nv + 2 * (size_t)m->nslice + 2 + (size_t)nt * 24;
  cudaError_t e = cudaMalloc(&tmp, ntmp * sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&m->slice_off, ((size_t)m->nslice + 1) * sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&m->row_of, (size_t)nwin * kWindowRows * sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&m->contrib, std::max<size_t>(1, (size_t)nt * 12) * sizeof(int));
  int nsm = 0;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device);
  m->grid = std::min({std::max(nsm, 1), kRowMaxGrid, m->nslice});
  int host[2] = {0, 0};   // total slots, too-long flag
  int *len = tmp, *place = tmp + nv, *slots = tmp + 2 * (size_t)nv, *flag = slots + m->nslice;
  int *pair_off = flag + 1, *colv = pair_off + m->nslice + 1, *colb = colv + (size_t)nt * 12;
  if (e == cudaSuccess) {
    const VertexIndex& x = tets->vindex;
    e = cudaMemsetAsync(flag, 0, sizeof(int), st);
    const int cg = (nv + kSortWarps - 1) / kSortWarps;
    row_columns_kernel<kShortTets, 256, false><<<cg, 32 * kSortWarps, 0, st>>>(nv, x.off, x.ent, tets->keys,
                                                                               m->contrib, colv, colb, len, flag);
    row_columns_kernel<kRowMaxTets, 1024, true><<<cg, 32 * kSortWarps, 0, st>>>(nv, x.off, x.ent, tets->keys,
                                                                                m->contrib, colv, colb, len, flag);
    window_kernel<<<nwin, kWindowRows, 0, st>>>(nv, x.order, len, m->row_of, place, slots);
    scan_kernel<<<1, kScanThreads, 0, st>>>(m->nslice, slots, m->slice_off);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(&host[0], m->slice_off + m->nslice, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&host[1], flag, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  // places of entries are 32-bit
  bool apply = e == cudaSuccess && host[1] == 0 && host[0] <= 0x7fffffff / kSliceRows;
  if (apply) {
    m->nslots = host[0];
    const size_t n = std::max<size_t>(1, (size_t)m->nslots * kSliceRows);
    const int sg = (m->nslice * 32 + 255) / 256;
    e = cudaMalloc(&m->col, n * sizeof(int));
    // rows that hold no vertex: a valid column
    if (e == cudaSuccess) e = cudaMemsetAsync(m->col, 0, n * sizeof(int), st);
    if (e == cudaSuccess) {
      row_fill_kernel<<<(nv + 31) / 32, 256, 0, st>>>(nv, tets->vindex.off, len, colv, place, m->slice_off, m->col);
      row_pair_kernel<false><<<sg, 256, 0, st>>>(m->nslice, m->row_of, tets->vindex.off, len, colv, colb, place,
                                                 m->slice_off, slots, nullptr, nullptr);
      scan_kernel<<<1, kScanThreads, 0, st>>>(m->nslice, slots, pair_off);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(&m->npair, pair_off + m->nslice, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = cudaMalloc(&m->pairs, std::max<size_t>(1, (size_t)m->npair) * sizeof(int4));
    if (e == cudaSuccess) {
      row_pair_kernel<true><<<sg, 256, 0, st>>>(m->nslice, m->row_of, tets->vindex.off, len, colv, colb, place,
                                                m->slice_off, slots, pair_off, m->pairs);
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
    cudaFree(m->pairs);
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
