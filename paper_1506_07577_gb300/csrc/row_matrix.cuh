// Row matrix of a tets relation: the assembled stiffness with three lanes per
// vertex row (device layout, shared by the assembly, the product and the CG
// solve on it).
//
// A vertex's row holds one 3x3 block per vertex that shares a tet with it,
// itself first (slot 0), the others by increasing vertex number.  Rows are
// gathered into slices of kSliceRows rows; lane 3 i + c of a warp owns
// component c of the slice's row i (30 of 32 lanes).  A slice has as many
// slots as its longest row.  Slot k of slice s is slot number
// slice_off[s] + k =: q, and holds
//   col[q * kSliceRows + i]        vertex of row i's k-th block
//   val[(q * 3 + d) * 32 + lane]   the block's entry (c, d)
// so that every load of a warp is one line of consecutive words, and a
// lane's product is a plain sum over its own entries, with no reduction
// between lanes: on GB300 an FP64 add costs a warp 64 cycles, so adds that
// only combine lanes are what the layout avoids.  Unused entries are zero and
// unused columns name the row's own vertex.
//
// Rows enter the slices in windows of kWindowRows vertices (taken in order of
// first use by the tets, so that neighbours stay close), sorted by length
// within the window: a slice's rows then have nearly equal lengths, whatever
// the vertex numbering.
#pragma once

#include <cstdint>

#include "ebb_internal.h"

namespace ebb {

constexpr int kSliceRows = 10;                       // rows per slice (30 lanes)
constexpr int kWindowSlices = 32;
constexpr int kWindowRows = kSliceRows * kWindowSlices;
constexpr int kRowMaxTets = 128;                     // tets around one vertex
constexpr int kRowMaxGrid = 256;                     // thread blocks of a kernel over all slices
// Element record, in values: for each of the six corner pairs (a < b, order 01
// 02 03 12 13 23) the three rows of its block, four values each, so that a
// row is one or two 16-byte accesses.  The fourth values of rows 0 .. 8 hold the
// corner forces of corners 1..3 (FP64 steps; corner 0 is minus their sum).
constexpr int kElemLen = 72;

struct RowMatrix {
  int state = 0;              // 0 not built, 1 built, -1 does not apply to this relation
  int nslice = 0;
  int64_t nslots = 0;
  int* slice_off = nullptr;   // nslice + 1
  int* row_of = nullptr;      // nslice * kSliceRows: vertex of each row, -1 for none
  int* col = nullptr;         // nslots * kSliceRows
  // Blocks (v, w), w >= v, slice by slice: x the place of (v, w) as in col, y that
  // of (w, v) (-1 when w is v), [z, w) its contributions.
  int npair = 0;
  int4* pairs = nullptr;
  int* contrib = nullptr;     // 12 per tet, row by row: 16 t + 2 pair + transposed
  bool no_step = false;       // the FP64 step's buffers did not fit (row_step.cu)
  int grid = 0;               // thread blocks of a kernel over all slices (at most one per SM)
  // Assembled K of ebb_assemble_tet_K ([0] FP32, [1] FP64): off-diagonal
  // blocks only (the product takes w_j - w_r), and the element records.
  void* val[2] = {nullptr, nullptr};
  void* elem[2] = {nullptr, nullptr};
};

// The vertex order and index arrays of the matrix, as the kernels take them.
struct RowView {
  int nslice;
  const int* __restrict__ slice_off;
  const int* __restrict__ row_of;
  const int* __restrict__ col;
};

// Tets of a warp that starts at tet t0 (signed: a block's second warp may start
// past the last tet).
__host__ __device__ inline int warp_tets(int t0, int nt) {
  const int n = nt - t0;
  return n < 0 ? 0 : (n < 32 ? n : 32);
}

// First slice of block b of `grid`, which take consecutive slices.
__host__ __device__ inline int first_slice(int b, int grid, int nslice) {
  return (int)((long long)b * nslice / grid);
}

// Build the pattern on first use (device work on `stream`, synchronous).
// EBB_OK with rm.state == -1: a vertex has more than kRowMaxTets tets, or the
// memory does not suffice; the caller then keeps to the matrix-free maps.
ebb_status_t ensure_row_pattern(ebb_ctx_s* ctx, ebb_rel_s* tets, cudaStream_t stream);
// Exclusive sums of n counts: out[0 .. n] (device arrays).
cudaError_t exclusive_scan(int n, const int* in, int* out, cudaStream_t st);

// Element records of K(u) and, with `force` (FP64 only), the element forces:
// u in planes (stride nv) or interleaved 4-float elements (aos).
template <typename T>
cudaError_t launch_element_blocks(ebb_rel_s* rel, int model, T mu0, T lam0, const T* u, bool aos, bool force, T* elem,
                                  cudaStream_t st);

// Off-diagonal blocks of scale * K, zero on the rows of pinned vertices (pin may
// be null; pin_bytes 1 or 4), from the element records.  Unused entries of val are
// left as they are: its owner zeroes them once.
template <typename T>
cudaError_t launch_row_blocks(const RowMatrix& m, const T* elem, const void* pin, int pin_bytes, T scale, T* val,
                              cudaStream_t st);

// Assembled K(u) on the rows and y += K w; *done is false when the rows do not
// apply to the relation (or, for the product, hold no K in this precision).
template <typename T>
cudaError_t launch_row_assemble(ebb_rel_s* rel, int model, T mu0, T lam0, const MapIO<T>& io, cudaStream_t st,
                                bool* done);
template <typename T>
cudaError_t launch_row_product(ebb_rel_s* rel, const T* w, T* y, bool aos, const int* active, cudaStream_t st,
                               bool* done);

}  // namespace ebb
