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
  // units of the extension over B+ (ExtUnits)
  const uint32_t* tiles;
  const float4* pts[2];
  const uint32_t* cidx[2];
  int32_t ntiles;
  int variant;             // launch shape of the extension (0, 1, 2)
  const float* dA;         // brick-dense omega / diag(A)
  const float* c;          // brick-dense c, or null (constant)
};

// Units of the extension (dense32.cu) over a set of points.
struct ExtUnits {
  int32_t ntiles = 0;
  DBuf<uint32_t> tiles;  // header words of the tiles that hold points of the set
  DBuf<float4> pts[2];   // a unit's first and second point: slot (bits) and cp fractions
  DBuf<uint32_t> cidx[2];  // their band indices
};
// Brick-dense structures of one level.
struct Dense32 {
  DBuf<int4> bface;
  DBuf<int32_t> bfwd;
  DBuf<uint32_t> slot;
  ExtUnits all;          // every point of B+
  DBuf<float> dA, c;     // brick-dense omega / diag(A) and c
};
inline size_t dense_size(const Level& L) { return (size_t)(L.nbricks + 1) << (2 * L.dim); }
void build_dense32(const Level& L, Dense32& D, cudaStream_t st);
// D.dA (and D.c) from the band-order vectors.
void dense_static(const Level& L, Dense32& D, const float* dA, const float* c, cudaStream_t st);
DenseView dense_view(const Level& L, const Dense32& D);

// Layout of a vector handed to a pass.
template <typename T>
struct Vec32 {
  T* dense;    // brick-dense, or
  T* compact;  // band order (used when dense is null)
};

// w (brick-dense) = E u over B+.  u brick-dense or in band order.
void launch_extend32(const DenseView& L, Vec32<const float> u, float* w, cudaStream_t st);
// w (band order, the first npts points of B+) = E u, u in band order.
void launch_extend32_compact(const DenseView& L, const float* u, float* w, int32_t npts, cudaStream_t st);
// Stencil pass of `mode` (APPLY, RESID, JACOBI, JAC_RED, JAC_BLACK) from w = E u (brick-dense):
// out = M u, out = f - c u + M u, or out = u + (f - c u + M u) dA (out may be u).  f has u's layout;
// where that is band order and fd is given, f is also written there brick-dense.
void launch_lap32(const DenseView& L, LapMode mode, Vec32<const float> u, const float* w, const float* f,
                  float cval, Vec32<float> out, float* fd, cudaStream_t st);
// Time the extension's launch shapes (as tune_extension).
int tune_extend32(const DenseView& L, const float* u, float* w, cudaStream_t st, float ms[3]);

}  // namespace cpm
