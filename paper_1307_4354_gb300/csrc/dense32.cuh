// FP32 level passes on brick-dense vectors (dense32.cu): the extension by
// units, the stencil by brick rows and the linear transfers.
//
// A brick-dense vector holds 4^d values per occupied brick of the level
// (slot = brick * 4^d + node of the brick, x fastest), whether or not the node
// is a band or ghost node, and one more brick that stands for absent ones.
// Every brick row of four nodes is one aligned 16-byte word, so boxes and
// stencils are read with vector loads, a neighbour inside the brick needs no
// index, and one across a face needs only the neighbouring brick's number.
// About two thirds of the slots are points; values at the others are never
// used.
#pragma once

#include "ops.cuh"

namespace cpm {

// Extension units of a set of points (see ExtUnits).
struct UnitsView {
  const uint32_t* tiles;
  const float4* pts[2];
  const uint32_t* cidx[2];
  int32_t ntiles;
};

// Brick rows of a set of nodes (row = brick * 4^(d-1) + row of the brick):
// a list, or all n rows of the level.
struct RowsView {
  const uint32_t* list;
  uint32_t n;
};

// Plain-pointer view of a level's brick-dense structures.
struct DenseView {
  const uint64_t* bmask;   // band occupancy per brick
  const int32_t* bstart;   // first band index of the brick
  const int4* bface;       // 2 per brick: {-x, +x, -y, +y}, {-z, +z, -, -}; nbricks if absent
  const int32_t* bfwd;     // 8 per brick: brick at (+i, +j, +k), index i + 2 j + 4 k
  const uint32_t* slot;    // band order -> slot, B then G
  int32_t nbricks;
  int32_t nB;
  int64_t nplus;
  int dim;
  float inv_h2, gamma;
  UnitsView all;           // the extension over B+
  int variant;             // launch shape of the extension (0, 1, 2)
  const float* dA;         // brick-dense omega / diag(A)
  const float* c;          // brick-dense c, or null (constant)
};

// Units of the extension (dense32.cu) over a set of points.
struct ExtUnits {
  int32_t ntiles = 0;
  uint32_t* tiles = nullptr;               // header words of the tiles that hold points of the set
  float4* pts[2] = {nullptr, nullptr};     // a unit's first and second point: slot (bits) and cp fractions
  uint32_t* cidx[2] = {nullptr, nullptr};  // their band indices (Dense32::all only)
  DBuf<float4> data;                       // holds them all
};
// The nodes of a level that a pass inside a cycle has to visit: rows of the
// stencil, and the points whose w = E u they take (dense32.cu).
struct NeedSet {
  ExtUnits units;
  uint32_t* rows = nullptr;
  int32_t nrows = 0;
  // the same for FP64 passes in band order (PointSet)
  int32_t *list = nullptr, *tstart = nullptr;
  uint32_t* epos = nullptr;
  int32_t nlist = 0;
  DBuf<uint32_t> data;  // holds them all
};
// Brick-dense structures of one level.
struct Dense32 {
  Part<int4> bface;
  Part<int32_t> bfwd;
  Part<uint32_t> slot;
  DBuf<unsigned char> tables;  // holds these three
  ExtUnits all;          // every point of B+
  DBuf<float> dA, c;     // brick-dense omega / diag(A) and c
  // levels of a V-cycle
  NeedSet resid;         // residual that is restricted (every level but the coarsest)
  NeedSet sweep;         // sweeps (levels between the finest and the coarsest)
};
// Targets of a linear transfer: base nodes of their cells in the source grid
// (packed), fractions (SoA, d x n).
struct TransferCells {
  const uint64_t* base = nullptr;
  const float* fr = nullptr;
  int32_t n = 0;
};
// Linear transfer from a brick-dense source: per target the slot (bits) of the
// cell's first node and the fractions, and where the result goes.
struct DenseTransfer {
  float4* rec = nullptr;
  uint32_t* dst = nullptr;
  int32_t n = 0;
  DBuf<float4> data;  // holds both
};
UnitsView units_view(const ExtUnits& U);
inline PointSet point_set(const NeedSet& S) { return {S.list, S.nlist, S.tstart, S.epos}; }
inline RowsView rows_view(const NeedSet& S) { return {S.rows, (uint32_t)S.nrows}; }
inline RowsView all_rows(const DenseView& L) { return {nullptr, (uint32_t)L.nbricks << (2 * (L.dim - 1))}; }
// A transfer to the points of B of a level, from the cells of all of them:
// written brick-dense or in band order, only to the level's sweep set if pruned.
struct TransferIn {
  TransferCells cells;
  const Level* source = nullptr;
  bool dense_dst = false, pruned = false;
  DenseTransfer* out = nullptr;  // null: none
};
// What a level's part in a cycle follows from: the cells of the restriction to
// the next level (none: the coarsest level), those of the finer level's points
// in this one (none: the finest level), and the transfers into this level.
struct CycleCells {
  TransferCells restrict_from, prolong_from;
  TransferIn in[2];
};
// Scratch of build_dense32, kept from level to level.
struct DenseScratch {
  DBuf<int64_t> counts;
  DBuf<uint64_t> mask;
  DBuf<uint8_t> keep;
};
inline size_t dense_size(const Level& L) { return (size_t)(L.nbricks + 1) << (2 * L.dim); }
// Everything of D but dA and c; with cyc also the needed sets (D.resid where there
// is a restriction, D.sweep where the level is prolonged from too) and the
// transfers into the level.  The scratch is in use until st has caught up.
void build_dense32(const Level& L, Dense32& D, const CycleCells* cyc, DenseScratch& sc, cudaStream_t st);
// D.dA (and D.c) from the band-order vectors.
void dense_static(const Level& L, Dense32& D, const float* dA, const float* c, cudaStream_t st);
DenseView dense_view(const Level& L, const Dense32& D);

// Layout of a vector handed to a pass.
template <typename T>
struct Vec32 {
  T* dense;    // brick-dense, or
  T* compact;  // band order (used when dense is null)
};

// w (brick-dense) = E u over the set S.  u brick-dense or in band order.
void launch_extend32(const DenseView& L, const UnitsView& S, Vec32<const float> u, float* w, cudaStream_t st);
// w (band order, the first npts points of B+) = E u, u in band order.
void launch_extend32_compact(const DenseView& L, const float* u, float* w, int32_t npts, cudaStream_t st);
// Stencil pass of `mode` (APPLY, RESID, JACOBI, JAC_RED, JAC_BLACK) from w = E u (brick-dense):
// out = M u, out = f - c u + M u, or out = u + (f - c u + M u) dA (out may be u).  f has u's layout;
// where that is band order and fd is given, f is also written there brick-dense.
void launch_lap32(const DenseView& L, LapMode mode, Vec32<const float> u, const float* w, const float* f,
                  float cval, Vec32<float> out, float* fd, const RowsView& rows, cudaStream_t st);
// u = f dA, the first Jacobi sweep from u = 0 (all brick-dense).
void launch_jacobi_zero32(const DenseView& L, const float* f, float* u, const RowsView& rows, cudaStream_t st);
// out[dst] (+)= linear interpolation of the brick-dense src (a vector of level `source`).
void launch_transfer32(const DenseTransfer& T, const DenseView& source, const float* src, float* out, bool add,
                       cudaStream_t st);
// out[slot[j]] += linear interpolation of src in band order (tv.idx set).
void launch_prolong_coarsest32(const TransferView<float>& tv, const uint32_t* slot, const float* src, float* out,
                               cudaStream_t st);
// Layout changes of vectors on B.
void launch_scatter32(const DenseView& L, const float* x, float* d, cudaStream_t st);
void launch_gather32(const DenseView& L, const float* d, float* x, cudaStream_t st);
void launch_scale_dense(const DenseView& L, const double* r, const double* norms, float* fd, cudaStream_t st);
void launch_axpy_dense(const DenseView& L, double* u, const float* d, const double* norms, cudaStream_t st);
// The fastest of the extension's launch shapes on a level (over B+, one warm-up
// and three timed launches each, events on st); ms[v] gets each shape's time.
// u, w: brick-dense scratch.
int tune_extend32(const DenseView& L, const float* u, float* w, cudaStream_t st, float ms[3]);

}  // namespace cpm
