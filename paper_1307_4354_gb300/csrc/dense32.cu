// FP32 level passes on brick-dense vectors (see dense32.cuh): the closest-point
// extension w = E u (Sec. 3.1, Eq. 3.1), the stencil of M = diag(L) +
// (L - diag L) E (Sec. 2.3 Eq. 2.10) with its residual and Jacobi update
// (Eq. 4.1), and the build of the structures they read.
//
// Extension units.  The points of B+ whose cubic stencil base lies in one 4^d
// brick (an extension tile, ext.cu) read one 7^d box of u, and about 6.6 of
// them share each base on a smooth surface.  A unit is up to two points with
// one base: a thread that evaluates both needs each of the base's 4^(d-1) rows
// once, half the shared-memory loads that bound the pass.
#include <vector>

#include "dense32.cuh"
#include "pdl.cuh"

namespace cpm {

static unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Strides (floats) of the staged box: a row is four 16-byte windows and one of
// padding, a plane seven rows and one more window, so that eight rows (four in
// y, two in z) written together start in eight different bank groups.
constexpr int kRowStride = 20, kPlaneStride = 144;
// Threads per SM that the extension is compiled for.
#ifndef CPM_EXT_THREADS_SM
#define CPM_EXT_THREADS_SM 896
#endif
constexpr int kExtThreadsSM = CPM_EXT_THREADS_SM;

// A tile's header words: 0..7 brick numbers of the box (index i + 2 j + 4 k,
// the number of bricks if absent), 8 the range of base positions (2 bits lo,
// 2 bits hi per axis), 9 and 10 the first unit and the one after the last.
constexpr int kTileWords = 12;
constexpr int kTileBox = 8, kTileBeg = 9, kTileEnd = 10;
// A unit is an entry of pts[0] and one of pts[1]: slot and cp fractions of each
// point, the slot's top three bits holding half of the base position (low half
// in pts[0]); a unit of one point repeats it.
constexpr int kSlotBits = 29;
constexpr uint32_t kSlotMask = (1u << kSlotBits) - 1u;

// ----------------------------------------------------------------- build
__global__ void k_dense_bricks(BrickView v, const uint32_t* bcoord, int dim, int4* bface, int32_t* bfwd) {
  const int32_t b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= v.nbricks) return;
  const int bx = bcoord[b] & 1023, by = (bcoord[b] >> 10) & 1023, bz = (bcoord[b] >> 20) & 1023;
  auto at = [&](int x, int y, int z) -> int32_t {
    if (x < 0 || y < 0 || z < 0 || x >= v.nbx || y >= v.nby || z >= v.nbz) return v.nbricks;
    const int32_t q = v.map[((size_t)z * v.nby + y) * v.nbx + x];
    return q < 0 ? v.nbricks : q;
  };
  bface[2 * (int64_t)b] = make_int4(at(bx - 1, by, bz), at(bx + 1, by, bz), at(bx, by - 1, bz), at(bx, by + 1, bz));
  bface[2 * (int64_t)b + 1] = dim == 3 ? make_int4(at(bx, by, bz - 1), at(bx, by, bz + 1), 0, 0)
                                       : make_int4(v.nbricks, v.nbricks, 0, 0);
  for (int q = 0; q < 8; ++q)
    bfwd[8 * (int64_t)b + q] = dim == 2 && q >= 4 ? v.nbricks : at(bx + (q & 1), by + ((q >> 1) & 1), bz + (q >> 2));
}

__global__ void k_dense_slots(BrickView v, const uint64_t* key, int64_t nplus, int dim, uint32_t* slot) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nplus) return;
  const uint64_t k = key[i];
  const int x = key_x(k), y = key_y(k), z = dim == 3 ? key_z(k) : 0;
  const int32_t b = v.map[((size_t)(z >> 2) * v.nby + (y >> 2)) * v.nbx + (x >> 2)];
  slot[i] = ((uint32_t)b << (2 * dim)) | (uint32_t)((x & 3) | ((y & 3) << 2) | ((z & 3) << 4));
}

// Points per base of a tile (kept points only).  One warp per tile; lane l
// returns the counts of bases l and l + 32.
__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ int2 tile_bases(const uint32_t* erec, const uint8_t* keep, int32_t beg, int32_t end,
                                           int* hist) {
  const int lane = threadIdx.x;
  hist[lane] = hist[lane + 32] = 0;
  __syncwarp();
  for (int32_t k = beg + lane; k < end; k += 32)
    if (!keep || keep[erec[k] >> 6]) atomicAdd(hist + (erec[k] & 63u), 1);
  __syncwarp();
  return make_int2(hist[lane], hist[lane + 32]);
}

__global__ void __launch_bounds__(32) k_units_count(const int32_t* tile_start, const uint32_t* erec,
                                                    const uint8_t* keep, int64_t* nunits, int64_t* used) {
  __shared__ int hist[64];
  const int32_t tile = blockIdx.x;
  const int2 n = tile_bases(erec, keep, tile_start[tile], tile_start[tile + 1], hist);
  const int u = warp_sum((n.x + 1) / 2 + (n.y + 1) / 2);
  if (threadIdx.x == 0) {
    nunits[tile] = u;
    used[tile] = u > 0;
  }
}

__global__ void __launch_bounds__(32) k_units_emit(BrickView v, const uint32_t* tile_brick,
                                                   const uint32_t* tile_box, const int32_t* tile_start,
                                                   const uint32_t* erec, const float* efr, int64_t nplus,
                                                   int dim, const uint8_t* keep, const uint32_t* slot,
                                                   const int64_t* unit0, int64_t ubase, const int64_t* tile0,
                                                   int64_t tbase, const int32_t* bfwd, uint32_t* tiles,
                                                   float4* pts0, float4* pts1, uint32_t* cidx0,
                                                   uint32_t* cidx1) {
  __shared__ int hist[64], key[64], start[64];
  const int lane = threadIdx.x;
  const int32_t tile = blockIdx.x;
  const int32_t beg = tile_start[tile], end = tile_start[tile + 1];
  const int2 n = tile_bases(erec, keep, beg, end, hist);
  const int units = warp_sum((n.x + 1) / 2 + (n.y + 1) / 2);
  if (units == 0) return;
  // order of the bases: the window of base (x, y, z) starts in 16-byte bank
  // group (x + 5 y + 36 z) mod 8, so bases of different groups are dealt in
  // turn; units of one base stay together (their loads coincide)
  auto group = [](int b) { return ((b & 3) + 5 * ((b >> 2) & 3) + 4 * (b >> 4)) & 7; };
  for (int h = 0; h < 2; ++h) {
    const int b = lane + 32 * h;
    int rr = 0;
    for (int q = 0; q < b; ++q) rr += hist[q] > 0 && group(q) == group(b);
    key[b] = hist[b] > 0 ? 8 * rr + group(b) : 1 << 20;
  }
  __syncwarp();
  for (int h = 0; h < 2; ++h) {
    const int b = lane + 32 * h;
    int s = 0;
    for (int q = 0; q < 64; ++q) s += key[q] < key[b] ? (hist[q] + 1) / 2 : 0;
    start[b] = s;
  }
  __syncwarp();
  const uint32_t tb = tile_brick[tile];
  const int bx = tb & 1023, by = (tb >> 10) & 1023, bz = (tb >> 20) & 1023;
  const int32_t home = v.map[((size_t)bz * v.nby + by) * v.nbx + bx];
  uint32_t* hdr = tiles + (tile0[tile] - tbase) * kTileWords;
  const int64_t u0 = unit0[tile] - ubase;
  if (lane < kTileWords) {
    uint32_t word = 0;
    if (lane < 8) word = (uint32_t)bfwd[8 * (int64_t)home + lane];
    if (lane == kTileBox) word = tile_box[tile];
    if (lane == kTileBeg) word = (uint32_t)u0;
    if (lane == kTileEnd) word = (uint32_t)(u0 + units);
    hdr[lane] = word;
  }
  for (int32_t k = beg + lane; k < end; k += 32) {
    const uint32_t rec = erec[k];
    const uint32_t idx = rec >> 6;
    if (keep && !keep[idx]) continue;
    const uint32_t b = rec & 63u;
    int r = 0;  // rank among the kept points of the base
    for (int32_t q = beg; q < k; ++q) r += (erec[q] & 63u) == b && (!keep || keep[erec[q] >> 6]);
    const int64_t p = u0 + start[b] + (r >> 1);
    const uint32_t s = slot[idx];
    const float fx = efr[k], fy = efr[nplus + k], fz = dim == 3 ? efr[2 * nplus + k] : 0.f;
    if (!(r & 1)) {
      pts0[p] = make_float4(__uint_as_float(s | ((b & 7u) << kSlotBits)), fx, fy, fz);
      if (cidx0) cidx0[p] = idx;
    }
    if ((r & 1) || r == hist[b] - 1) {  // (an odd count's last unit repeats its point)
      pts1[p] = make_float4(__uint_as_float(s | ((b >> 3) << kSlotBits)), fx, fy, fz);
      if (cidx1) cidx1[p] = idx;
    }
  }
}

UnitsView units_view(const ExtUnits& U) {
  UnitsView v;
  v.tiles = U.tiles;
  v.ntiles = U.ntiles;
  for (int h = 0; h < 2; ++h) {
    v.pts[h] = U.pts[h];
    v.cidx[h] = U.cidx[h];
  }
  return v;
}

DenseView dense_view(const Level& L, const Dense32& D) {
  DenseView v;
  v.bmask = L.bmask.get();
  v.bstart = L.bstart.get();
  v.bface = D.bface.get();
  v.bfwd = D.bfwd.get();
  v.slot = D.slot.get();
  v.nbricks = L.nbricks;
  v.nB = L.nB;
  v.nplus = L.nplus();
  v.dim = L.dim;
  v.inv_h2 = (float)(1.0 / (L.dx * L.dx));
  v.gamma = (float)(2.0 * L.dim / (L.dx * L.dx));
  v.all = units_view(D.all);
  v.variant = L.ext_variant;
  v.dA = D.dA.get();
  v.c = D.c.get();
  return v;
}

// ----------------------------------------------------------------- extension
// Cubic weights at two fractions at once, packed.  With t1 = 1 - s, t2 = 2 - s
// the closed forms of the proof of Theorem 3.3 are w_-1 = -s t1 t2 / 6,
// w_0 = (1 + s) t1 t2 / 2, w_1 = (1 + s) s t2 / 2, w_2 = -s t1 (1 + s) / 6.
__device__ __forceinline__ void cubic32x2(float2 s, float2 w[4]) {
  const float2 one = make_float2(1.f, 1.f), two = make_float2(2.f, 2.f), neg = make_float2(-1.f, -1.f);
  const float2 t1 = __ffma2_rn(s, neg, one), t2 = __ffma2_rn(s, neg, two), sp1 = __fadd2_rn(s, one);
  const float2 p = __fmul2_rn(__fmul2_rn(s, t1), make_float2(-1.f / 6.f, -1.f / 6.f));
  const float2 q = __fmul2_rn(__fmul2_rn(sp1, t2), make_float2(0.5f, 0.5f));
  w[0] = __fmul2_rn(p, t2);
  w[1] = __fmul2_rn(q, t1);
  w[2] = __fmul2_rn(q, s);
  w[3] = __fmul2_rn(p, sp1);
}

// A brick row of four values of a band-order vector (the row's points are
// consecutive).
template <int DIM>
__device__ __forceinline__ float4 load_row_ordered(const DenseView& L, const float* __restrict__ u, int32_t brick,
                                                   int row) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (brick >= L.nbricks) return v;
  const uint64_t m = __ldg(L.bmask + brick);
  const uint32_t nib = (uint32_t)(m >> (4 * row)) & 15u;
  const float* p = u + __ldg(L.bstart + brick) + __popcll(m & ((1ull << (4 * row)) - 1ull));
  if (nib & 1u) v.x = ld_prior(p);
  if (nib & 2u) v.y = ld_prior(p + (nib & 1u));
  if (nib & 4u) v.z = ld_prior(p + __popc(nib & 3u));
  if (nib & 8u) v.w = ld_prior(p + __popc(nib & 7u));
  return v;
}

// One warp per tile and one lane per unit.  The lanes stage the box's rows (two
// aligned 16-byte loads each, eight lanes on one 128-byte line) as the windows
// of four values that a base can start at; the records of the lane's first unit
// are loaded meanwhile.  A
// unit's two points are evaluated together from one 16-byte shared-memory load
// per row: y and z by packed FMAs on two x positions, then x.
//
// Bound by the L1 data pipe (73 % of its peak: the 16 row loads of a unit, the
// window stores, the staging) with issue slots at 52 %.  Unit sphere,
// dx = 1/256, 8.16 M points: 73 us, against 108 us for one thread per point on
// boxes gathered value by value from band order (16 row loads per point).
// Chunks of up to six points whose 64 values stay in registers halve the row
// loads again but leave 13 warps on an SM: 111 us.
template <int DIM, bool CIN, bool COUT, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, kExtThreadsSM / (32 * WARPS))
    k_extend_units(DenseView L, UnitsView S, const float* __restrict__ u, float* __restrict__ w, int32_t npts) {
  constexpr int NC = DIM == 3 ? 4 : 1, RS = kRowStride, NH = DIM == 3 ? 2 : 1;
  __shared__ __align__(16) float box[WARPS][DIM == 3 ? 7 * kPlaneStride : 8 * RS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* win = box[warp];
  const int32_t tile = blockIdx.x * WARPS + warp;
  release_next();
  if (tile >= S.ntiles) return;
  const uint32_t hdr = __ldg(S.tiles + (size_t)tile * kTileWords + min(lane, kTileWords - 1));
  const uint32_t tbox = __shfl_sync(0xffffffffu, hdr, kTileBox);
  const int32_t beg = (int32_t)__shfl_sync(0xffffffffu, hdr, kTileBeg);
  const int32_t end = (int32_t)__shfl_sync(0xffffffffu, hdr, kTileEnd);
  int32_t k = beg + lane;
  float4 ra, rb;
  if (k < end) {
    ra = __ldg(S.pts[0] + k);
    rb = __ldg(S.pts[1] + k);
  }
  wait_prior();
  // row r = lane + 32 h of the 2^(d-1) columns of bricks along x: column r / 4^(d-1),
  // row r mod 4^(d-1) of its bricks
  const int xhi = (tbox >> 2) & 3;
  const uint32_t ylo = (tbox >> 4) & 3, ny = ((tbox >> 6) & 3) + 3 - ylo;
  const uint32_t zlo = (tbox >> 8) & 3, nz = ((tbox >> 10) & 3) + 3 - zlo;
  float4 lo[NH], hi[NH];
  bool in[NH];
#pragma unroll
  for (int h = 0; h < NH; ++h) {
    const int q = DIM == 3 ? 2 * h + (lane >> 4) : (lane >> 2) & 1;
    const int row = DIM == 3 ? lane & 15 : lane & 3;
    const int32_t blo = (int32_t)__shfl_sync(0xffffffffu, hdr, 2 * q);
    const int32_t bhi = (int32_t)__shfl_sync(0xffffffffu, hdr, 2 * q + 1);
    const uint32_t y = 4 * (q & 1) + (row & 3), z = 4 * (q >> 1) + (row >> 2);
    in[h] = y - ylo <= ny && (DIM == 3 ? z - zlo <= nz : lane < 8);
    hi[h] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!in[h]) continue;
    if constexpr (CIN) {
      lo[h] = load_row_ordered<DIM>(L, u, blo, row);
      if (xhi > 0) hi[h] = load_row_ordered<DIM>(L, u, bhi, row);
    } else {
      lo[h] = ld_prior(reinterpret_cast<const float4*>(u + ((size_t)blo << (2 * DIM))) + row);
      if (xhi > 0) hi[h] = ld_prior(reinterpret_cast<const float4*>(u + ((size_t)bhi << (2 * DIM))) + row);
    }
  }
#pragma unroll
  for (int h = 0; h < NH; ++h)
    if (in[h]) {
      const int q = DIM == 3 ? 2 * h + (lane >> 4) : (lane >> 2) & 1;
      const int row = DIM == 3 ? lane & 15 : lane & 3;
      float4* o = reinterpret_cast<float4*>(win + (4 * (q & 1) + (row & 3)) * RS +
                                            (4 * (q >> 1) + (row >> 2)) * kPlaneStride);
      o[0] = lo[h];
      if (xhi > 0) o[1] = make_float4(lo[h].y, lo[h].z, lo[h].w, hi[h].x);
      if (xhi > 1) o[2] = make_float4(lo[h].z, lo[h].w, hi[h].x, hi[h].y);
      if (xhi > 2) o[3] = make_float4(lo[h].w, hi[h].x, hi[h].y, hi[h].z);
    }
  __syncwarp();
#pragma unroll 1
  for (; k < end; k += 32) {
    const uint32_t sa = __float_as_uint(ra.x), sb = __float_as_uint(rb.x);
    const int px = (sa >> kSlotBits) & 3, py = ((sa >> 31) & 1) | ((sb >> (kSlotBits - 1)) & 2), pz = sb >> 30;
    float2 wa[4], wb[4], wz[4];  // (x, y) weights of either point, z weights of both
    cubic32x2(make_float2(ra.y, ra.z), wa);
    cubic32x2(make_float2(rb.y, rb.z), wb);
    if (DIM == 3) cubic32x2(make_float2(ra.w, rb.w), wz);
    const float* base = win + pz * kPlaneStride + py * RS + px * 4;
    float2 qa01, qa23, qb01, qb23;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      float2 pa01, pa23, pb01, pb23;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const float4 x = *reinterpret_cast<const float4*>(base + c * kPlaneStride + b * RS);
        const float2 x01 = make_float2(x.x, x.y), x23 = make_float2(x.z, x.w);
        const float2 ya = make_float2(wa[b].y, wa[b].y), yb = make_float2(wb[b].y, wb[b].y);
        if (b == 0) {
          pa01 = __fmul2_rn(ya, x01);
          pa23 = __fmul2_rn(ya, x23);
          pb01 = __fmul2_rn(yb, x01);
          pb23 = __fmul2_rn(yb, x23);
        } else {
          pa01 = __ffma2_rn(ya, x01, pa01);
          pa23 = __ffma2_rn(ya, x23, pa23);
          pb01 = __ffma2_rn(yb, x01, pb01);
          pb23 = __ffma2_rn(yb, x23, pb23);
        }
      }
      const float2 za = make_float2(wz[c].x, wz[c].x), zb = make_float2(wz[c].y, wz[c].y);
      if (DIM == 2) {
        qa01 = pa01;
        qa23 = pa23;
        qb01 = pb01;
        qb23 = pb23;
      } else if (c == 0) {
        qa01 = __fmul2_rn(za, pa01);
        qa23 = __fmul2_rn(za, pa23);
        qb01 = __fmul2_rn(zb, pb01);
        qb23 = __fmul2_rn(zb, pb23);
      } else {
        qa01 = __ffma2_rn(za, pa01, qa01);
        qa23 = __ffma2_rn(za, pa23, qa23);
        qb01 = __ffma2_rn(zb, pb01, qb01);
        qb23 = __ffma2_rn(zb, pb23, qb23);
      }
    }
    const float va = (wa[0].x * qa01.x + wa[2].x * qa23.x) + (wa[1].x * qa01.y + wa[3].x * qa23.y);
    const float vb = (wb[0].x * qb01.x + wb[2].x * qb23.x) + (wb[1].x * qb01.y + wb[3].x * qb23.y);
    if (COUT) {
      const int32_t ia = (int32_t)__ldg(S.cidx[0] + k), ib = (int32_t)__ldg(S.cidx[1] + k);
      if (ia < npts) w[ia] = va;
      if (ib < npts) w[ib] = vb;
    } else {
      w[sa & kSlotMask] = va;
      w[sb & kSlotMask] = vb;
    }
    if (k + 32 < end) {
      ra = __ldg(S.pts[0] + k + 32);
      rb = __ldg(S.pts[1] + k + 32);
    }
  }
}

// Launch shapes (variant 0, 1, 2): one, two or four tiles (warps) per CTA.
template <int DIM, bool CIN, bool COUT>
static void extend_units(const DenseView& L, const UnitsView& S, int variant, const float* u, float* w,
                         int32_t npts, cudaStream_t st) {
  if (S.ntiles <= 0) return;
  if (variant == 2)
    launch_pdl(k_extend_units<DIM, CIN, COUT, 4>, nblk(S.ntiles, 4), 128, st, L, S, u, w, npts);
  else if (variant == 1)
    launch_pdl(k_extend_units<DIM, CIN, COUT, 2>, nblk(S.ntiles, 2), 64, st, L, S, u, w, npts);
  else
    launch_pdl(k_extend_units<DIM, CIN, COUT, 1>, S.ntiles, 32, st, L, S, u, w, npts);
}

static void extend32(const DenseView& L, const UnitsView& S, int variant, Vec32<const float> u, float* w,
                     cudaStream_t st) {
  if (L.dim == 3) {
    if (u.dense) extend_units<3, false, false>(L, S, variant, u.dense, w, 0, st);
    else extend_units<3, true, false>(L, S, variant, u.compact, w, 0, st);
  } else {
    if (u.dense) extend_units<2, false, false>(L, S, variant, u.dense, w, 0, st);
    else extend_units<2, true, false>(L, S, variant, u.compact, w, 0, st);
  }
}

void launch_extend32(const DenseView& L, const UnitsView& S, Vec32<const float> u, float* w, cudaStream_t st) {
  extend32(L, S, L.variant, u, w, st);
  count_launch();
}

void launch_extend32_compact(const DenseView& L, const float* u, float* w, int32_t npts, cudaStream_t st) {
  if (L.dim == 3) extend_units<3, true, true>(L, L.all, L.variant, u, w, npts, st);
  else extend_units<2, true, true>(L, L.all, L.variant, u, w, npts, st);
  count_launch();
}

int tune_extend32(const DenseView& L, const float* u, float* w, cudaStream_t st, float ms[3]) {
  int best = 0;
  for (int v = 0; v < 3; ++v) ms[v] = 0.f;
  if (L.all.ntiles <= 0) return best;
  struct Events {
    cudaEvent_t e[6] = {};
    ~Events() {
      for (cudaEvent_t q : e)
        if (q) cudaEventDestroy(q);
    }
  } ev;
  for (cudaEvent_t& q : ev.e) CPM_CUDA_TRY(cudaEventCreate(&q));
  constexpr int kReps = 3;
  const Vec32<const float> uv{u, nullptr};
  for (int v = 0; v < 3; ++v) {  // one wait for all three
    extend32(L, L.all, v, uv, w, st);  // warm-up
    CPM_CUDA_TRY(cudaEventRecord(ev.e[2 * v], st));
    for (int r = 0; r < kReps; ++r) extend32(L, L.all, v, uv, w, st);
    CPM_CUDA_TRY(cudaEventRecord(ev.e[2 * v + 1], st));
  }
  CPM_CUDA_TRY(cudaEventSynchronize(ev.e[5]));
  for (int v = 0; v < 3; ++v) {
    CPM_CUDA_TRY(cudaEventElapsedTime(&ms[v], ev.e[2 * v], ev.e[2 * v + 1]));
    ms[v] /= kReps;
    if (ms[v] < ms[best]) best = v;
  }
  return best;
}

// ----------------------------------------------------------------- stencil
// One thread per brick row of four nodes.  Brick-dense vectors make the pass a
// stream of aligned 16-byte loads at addresses known from the thread number:
// w of the row and of its -y, +y, -z, +z rows (inside the brick or from the
// face neighbour), u, f and omega/diag of the row; only the rows across faces
// wait for the brick's neighbour numbers, and the two x neighbours across faces
// are single values.  CIN: u and f come in band order (the first sweep on a
// caller's vectors); f is then also left brick-dense in fd.
//
// Bound by HBM and by the latency of its one round of loads: 31 bytes per point
// at two thirds of the slots used, against 44 with a table of six neighbour
// indices.  Unit sphere, dx = 1/256, 6.8 M points: 45 us a Jacobi sweep (53 us
// with the table).
template <int DIM, int MODE, bool CIN>
__global__ void __launch_bounds__(256) k_lap_rows(DenseView L, const float* u, const float* __restrict__ w,
                                                  const float* __restrict__ f, float cval, Vec32<float> out,
                                                  float* __restrict__ fd, RowsView rows) {
  constexpr int ROWS = DIM == 3 ? 16 : 4, SH = 2 * DIM;
  uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  release_next();
  if (t >= rows.n) return;
  if (rows.list) t = __ldg(rows.list + t);
  const int32_t b = (int32_t)(t / ROWS);
  const int row = (int)(t % ROWS);
  const int y = row & 3, z = row >> 2;
  const size_t s0 = ((size_t)b << SH) + 4 * row;
  auto load4 = [](const float* p) { return ld_prior(reinterpret_cast<const float4*>(p)); };
  const int4 fa = __ldg(L.bface + 2 * (int64_t)b);
  const int4 fb = DIM == 3 ? __ldg(L.bface + 2 * (int64_t)b + 1) : make_int4(0, 0, 0, 0);
  const bool ordered = CIN || !out.dense;  // band-order data on either side
  const uint64_t m = ordered ? __ldg(L.bmask + b) : 0ull;
  const int32_t start = ordered ? __ldg(L.bstart + b) : 0;
  float4 uu, ff = make_float4(0.f, 0.f, 0.f, 0.f), dd = ff, cc = make_float4(cval, cval, cval, cval);
  if (MODE != LAP_APPLY && MODE != LAP_RESID) dd = __ldg(reinterpret_cast<const float4*>(L.dA + s0));
  if (MODE != LAP_APPLY && L.c) cc = __ldg(reinterpret_cast<const float4*>(L.c + s0));
  wait_prior();
  const float4 w0 = load4(w + s0);
  if (!CIN) {
    uu = load4(u + s0);
    if (MODE != LAP_APPLY) ff = load4(f + s0);
  }
  auto row4 = [&](int32_t bb, int rr) { return load4(w + ((size_t)bb << SH) + 4 * rr); };
  const float4 ym = row4(y > 0 ? b : fa.z, y > 0 ? row - 1 : row + 3);
  const float4 yp = row4(y < 3 ? b : fa.w, y < 3 ? row + 1 : row - 3);
  float4 zm = make_float4(0.f, 0.f, 0.f, 0.f), zp = zm;
  if (DIM == 3) {
    zm = row4(z > 0 ? b : fb.x, z > 0 ? row - 4 : row + 12);
    zp = row4(z < 3 ? b : fb.y, z < 3 ? row + 4 : row - 12);
  }
  const float xm = ld_prior(w + ((size_t)fa.x << SH) + 4 * row + 3);
  const float xp = ld_prior(w + ((size_t)fa.y << SH) + 4 * row);
  const uint32_t nib = (uint32_t)(m >> (4 * row)) & 15u;
  const int32_t i0 = start + __popcll(m & ((1ull << (4 * row)) - 1ull));
  const int32_t off[4] = {0, (int)(nib & 1u), __popc(nib & 3u), __popc(nib & 7u)};
  if (CIN) {
    float a4[4] = {0.f, 0.f, 0.f, 0.f}, b4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < 4; ++a)
      if ((nib >> a) & 1u) {
        a4[a] = ld_prior(u + i0 + off[a]);
        if (MODE != LAP_APPLY) b4[a] = ld_prior(f + i0 + off[a]);
      }
    uu = make_float4(a4[0], a4[1], a4[2], a4[3]);
    ff = make_float4(b4[0], b4[1], b4[2], b4[3]);
    if (fd) *reinterpret_cast<float4*>(fd + s0) = ff;
  }
  const float wc[6] = {xm, w0.x, w0.y, w0.z, w0.w, xp};
  const float wym[4] = {ym.x, ym.y, ym.z, ym.w}, wyp[4] = {yp.x, yp.y, yp.z, yp.w};
  const float wzm[4] = {zm.x, zm.y, zm.z, zm.w}, wzp[4] = {zp.x, zp.y, zp.z, zp.w};
  const float u4[4] = {uu.x, uu.y, uu.z, uu.w}, f4[4] = {ff.x, ff.y, ff.z, ff.w};
  const float d4[4] = {dd.x, dd.y, dd.z, dd.w}, c4[4] = {cc.x, cc.y, cc.z, cc.w};
  float rr[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const float wi = wc[a + 1], ui = u4[a];
    float s = wc[a] - wi;
    s += wc[a + 2] - wi;
    s += wym[a] - wi;
    s += wyp[a] - wi;
    if (DIM == 3) {
      s += wzm[a] - wi;
      s += wzp[a] - wi;
    }
    const float Mu = s * L.inv_h2 + L.gamma * (wi - ui);
    const float r = f4[a] - c4[a] * ui + Mu;
    rr[a] = MODE == LAP_APPLY ? Mu : MODE == LAP_RESID ? r : ui + r * d4[a];
    if ((MODE == LAP_JAC_RED || MODE == LAP_JAC_BLACK) && ((a + y + z) & 1) != (MODE == LAP_JAC_BLACK ? 1 : 0))
      rr[a] = ui;
  }
  if (out.dense) {
    *reinterpret_cast<float4*>(out.dense + s0) = make_float4(rr[0], rr[1], rr[2], rr[3]);
  } else {
#pragma unroll
    for (int a = 0; a < 4; ++a)
      if ((nib >> a) & 1u) out.compact[i0 + off[a]] = rr[a];
  }
}

template <int MODE>
static void lap32(const DenseView& L, Vec32<const float> u, const float* w, const float* f, float cval,
                  Vec32<float> out, float* fd, RowsView rows, cudaStream_t st) {
  if (rows.n == 0) return;
  const unsigned g = nblk(rows.n, 256);
  if (L.dim == 3) {
    if (u.dense) launch_pdl(k_lap_rows<3, MODE, false>, g, 256, st, L, u.dense, w, f, cval, out, (float*)nullptr, rows);
    else launch_pdl(k_lap_rows<3, MODE, true>, g, 256, st, L, u.compact, w, f, cval, out, fd, rows);
  } else {
    if (u.dense) launch_pdl(k_lap_rows<2, MODE, false>, g, 256, st, L, u.dense, w, f, cval, out, (float*)nullptr, rows);
    else launch_pdl(k_lap_rows<2, MODE, true>, g, 256, st, L, u.compact, w, f, cval, out, fd, rows);
  }
  count_launch();
}

void launch_lap32(const DenseView& L, LapMode mode, Vec32<const float> u, const float* w, const float* f,
                  float cval, Vec32<float> out, float* fd, const RowsView& rows, cudaStream_t st) {
  if (mode == LAP_APPLY) lap32<LAP_APPLY>(L, u, w, f, cval, out, fd, rows, st);
  if (mode == LAP_RESID) lap32<LAP_RESID>(L, u, w, f, cval, out, fd, rows, st);
  if (mode == LAP_JACOBI) lap32<LAP_JACOBI>(L, u, w, f, cval, out, fd, rows, st);
  if (mode == LAP_JAC_RED) lap32<LAP_JAC_RED>(L, u, w, f, cval, out, fd, rows, st);
  if (mode == LAP_JAC_BLACK) lap32<LAP_JAC_BLACK>(L, u, w, f, cval, out, fd, rows, st);
}

// The first Jacobi sweep from u = 0: E u and M u vanish, u = f dA.
__global__ void __launch_bounds__(256) k_jacobi_zero(const float* __restrict__ f, const float* __restrict__ dA,
                                                     float* __restrict__ u, RowsView rows) {
  uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  release_next();
  if (t >= rows.n) return;
  if (rows.list) t = __ldg(rows.list + t);
  const float4 d = __ldg(reinterpret_cast<const float4*>(dA) + t);
  wait_prior();
  const float4 a = ld_prior(reinterpret_cast<const float4*>(f) + t);
  reinterpret_cast<float4*>(u)[t] = make_float4(a.x * d.x, a.y * d.y, a.z * d.z, a.w * d.w);
}
void launch_jacobi_zero32(const DenseView& L, const float* f, float* u, const RowsView& rows, cudaStream_t st) {
  if (rows.n == 0) return;
  launch_pdl(k_jacobi_zero, nblk(rows.n, 256), 256, st, f, L.dA, u, rows);
  count_launch();
}

// ----------------------------------------------------------------- transfers
// Linear closest-point interpolation (Sec. 4.3) at a list of targets from a
// brick-dense source: a record holds the slot of the cell's first node and the
// fractions, the other nodes follow from the slot (and, across a face, from
// the brick's forward neighbours), so a target reads 20 bytes instead of 44
// with a table of the eight node indices.
template <int DIM, bool ADD>
__global__ void __launch_bounds__(256) k_transfer_dense(const float4* __restrict__ rec,
                                                        const uint32_t* __restrict__ dst, int32_t n,
                                                        const int32_t* __restrict__ bfwd,
                                                        const float* __restrict__ src, float* __restrict__ out) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  release_next();
  if (j >= n) return;
  const float4 r = __ldg(rec + j);
  const uint32_t d = __ldg(dst + j);
  wait_prior();
  const float old = ADD ? ld_prior(out + d) : 0.f;
  const uint32_t s = __float_as_uint(r.x);
  const int32_t b = (int32_t)(s >> (2 * DIM));
  const int x = s & 3, y = (s >> 2) & 3, z = DIM == 3 ? (s >> 4) & 3 : 0;
  const float wx[2] = {1.f - r.y, r.y}, wy[2] = {1.f - r.z, r.z}, wz[2] = {1.f - r.w, r.w};
  float acc = 0.f;
#pragma unroll
  for (int c = 0; c < (DIM == 3 ? 2 : 1); ++c) {
    float accy = 0.f;
#pragma unroll
    for (int bb = 0; bb < 2; ++bb) {
      const int q = (((y + bb) >> 2) << 1) | (((z + c) >> 2) << 2);
      const int row = ((y + bb) & 3) * 4 + (DIM == 3 ? ((z + c) & 3) * 16 : 0);
      const int32_t b0 = q ? __ldg(bfwd + 8 * (int64_t)b + q) : b;
      const int32_t b1 = x == 3 ? __ldg(bfwd + 8 * (int64_t)b + q + 1) : b0;
      const float v0 = ld_prior(src + ((size_t)b0 << (2 * DIM)) + row + x);
      const float v1 = ld_prior(src + ((size_t)b1 << (2 * DIM)) + row + ((x + 1) & 3));
      accy += wy[bb] * (wx[0] * v0 + wx[1] * v1);
    }
    acc += (DIM == 3 ? wz[c] : 1.f) * accy;
  }
  out[d] = ADD ? old + acc : acc;
}
void launch_transfer32(const DenseTransfer& T, const DenseView& source, const float* src, float* out, bool add,
                       cudaStream_t st) {
  if (T.n <= 0) return;
  const unsigned g = nblk(T.n, 256);
  const float4* r = T.rec;
  const uint32_t* d = T.dst;
  if (source.dim == 3) {
    if (add) launch_pdl(k_transfer_dense<3, true>, g, 256, st, r, d, T.n, source.bfwd, src, out);
    else launch_pdl(k_transfer_dense<3, false>, g, 256, st, r, d, T.n, source.bfwd, src, out);
  } else {
    if (add) launch_pdl(k_transfer_dense<2, true>, g, 256, st, r, d, T.n, source.bfwd, src, out);
    else launch_pdl(k_transfer_dense<2, false>, g, 256, st, r, d, T.n, source.bfwd, src, out);
  }
  count_launch();
}

// Prolongation from the coarsest level, whose solution is in band order.
template <int DIM>
__global__ void __launch_bounds__(256) k_prolong_coarsest(TransferView<float> tv, const uint32_t* __restrict__ slot,
                                                          const float* __restrict__ src, float* __restrict__ out) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  release_next();
  if (j >= tv.n) return;
  const float sx = __ldg(tv.fr + j), sy = __ldg(tv.fr + tv.n + j);
  const float sz = DIM == 3 ? __ldg(tv.fr + 2 * (int64_t)tv.n + j) : 0.f;
  const float wx[2] = {1.f - sx, sx}, wy[2] = {1.f - sy, sy}, wz[2] = {1.f - sz, sz};
  const uint32_t d = __ldg(slot + j);
  wait_prior();
  float acc = 0.f;
#pragma unroll
  for (int c = 0; c < (DIM == 3 ? 2 : 1); ++c) {
    float accy = 0.f;
#pragma unroll
    for (int bb = 0; bb < 2; ++bb) {
      const int q = 4 * c + 2 * bb;
      const float v0 = ld_prior(src + __ldg(tv.idx + (int64_t)q * tv.n + j));
      const float v1 = ld_prior(src + __ldg(tv.idx + (int64_t)(q + 1) * tv.n + j));
      accy += wy[bb] * (wx[0] * v0 + wx[1] * v1);
    }
    acc += (DIM == 3 ? wz[c] : 1.f) * accy;
  }
  out[d] = ld_prior(out + d) + acc;
}
void launch_prolong_coarsest32(const TransferView<float>& tv, const uint32_t* slot, const float* src, float* out,
                               cudaStream_t st) {
  if (tv.n <= 0) return;
  if (tv.dim == 3) launch_pdl(k_prolong_coarsest<3>, nblk(tv.n, 256), 256, st, tv, slot, src, out);
  else launch_pdl(k_prolong_coarsest<2>, nblk(tv.n, 256), 256, st, tv, slot, src, out);
  count_launch();
}

// ----------------------------------------------------------------- needed points
// Inside a cycle a coarse level's u is read only at the nodes of the stencils
// (interpolation at its own closest points and at the finer level's), its
// residual only at the nodes that the restriction reads.  A sweep there has to
// update the former, which takes w = E u at them and their Laplacian
// neighbours; the residual of any level takes w at the latter and their
// neighbours.  On a sphere these are 0.73 and 0.36 of B, with w at 0.77 and
// 0.47 of B+ (the band keeps a margin on both sides of the stencils).

// bit of grid node (x, y, z) in per-brick masks
__device__ __forceinline__ bool mask_bit(const BrickView& v, const uint64_t* mask, int x, int y, int z) {
  if ((unsigned)x >= (unsigned)v.n || (unsigned)y >= (unsigned)v.n || (unsigned)z >= (unsigned)v.n) return false;
  const int32_t b = v.map[((size_t)(z >> 2) * v.nby + (y >> 2)) * v.nbx + (x >> 2)];
  return b >= 0 && ((mask[b] >> ((x & 3) | ((y & 3) << 2) | ((z & 3) << 4))) & 1ull);
}
__device__ __forceinline__ void set_mask_bit(const BrickView& v, uint64_t* mask, int x, int y, int z) {
  const int32_t b = v.map[((size_t)(z >> 2) * v.nby + (y >> 2)) * v.nbx + (x >> 2)];
  if (b < 0) return;
  const unsigned long long bit = 1ull << ((x & 3) | ((y & 3) << 2) | ((z & 3) << 4));
  if (!(mask[b] & bit)) atomicOr(reinterpret_cast<unsigned long long*>(mask + b), bit);
}
// the 2^d nodes of each target's cell
__global__ void k_mark_cells(const uint64_t* base, int32_t n, int dim, BrickView src, uint64_t* mask) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const uint64_t k = base[j];
  const int x = (int)(k & 0xffffu), y = (int)((k >> 16) & 0xffffu), z = (int)((k >> 32) & 0xffffu);
  for (int q = 0; q < (dim == 3 ? 8 : 4); ++q)
    set_mask_bit(src, mask, x + (q & 1), y + ((q >> 1) & 1), z + (q >> 2));
}
// the 4^d nodes of every stencil, one warp per tile
__global__ void __launch_bounds__(32) k_mark_stencils(BrickView v, const uint32_t* tile_brick,
                                                      const int32_t* tile_start, const uint32_t* erec, int dim,
                                                      const int32_t* bfwd, uint64_t* mask) {
  __shared__ uint32_t has[2], box[8][2];
  const int lane = threadIdx.x;
  const int32_t tile = blockIdx.x;
  if (lane < 2) has[lane] = 0u;
  if (lane < 8) box[lane][0] = box[lane][1] = 0u;
  __syncwarp();
  for (int32_t k = tile_start[tile] + lane; k < tile_start[tile + 1]; k += 32)
    atomicOr(has + ((erec[k] >> 5) & 1u), 1u << (erec[k] & 31u));
  __syncwarp();
  for (int b = lane; b < 64; b += 32) {
    if (!((has[b >> 5] >> (b & 31)) & 1u)) continue;
    const int lx = b & 3, ly = (b >> 2) & 3, lz = b >> 4;
    const uint32_t lo = (0xFu << lx) & 0xFu, hi = 0xFu >> (4 - lx);
    for (int c = 0; c < (dim == 3 ? 4 : 1); ++c)
      for (int a = 0; a < 4; ++a) {
        const int y = ly + a, z = lz + c, q = ((y >> 2) << 1) | ((z >> 2) << 2);
        const int sh = 4 * (y & 3) + 16 * (z & 3);
        atomicOr(&box[q][sh >> 5], lo << (sh & 31));
        if (hi) atomicOr(&box[q + 1][sh >> 5], hi << (sh & 31));
      }
  }
  __syncwarp();
  const uint32_t tb = tile_brick[tile];
  const int32_t home = v.map[((size_t)((tb >> 20) & 1023) * v.nby + ((tb >> 10) & 1023)) * v.nbx + (tb & 1023)];
  if (lane < 8) {
    const int32_t b = bfwd[8 * (int64_t)home + lane];
    const unsigned long long m = box[lane][0] | ((unsigned long long)box[lane][1] << 32);
    if (b < v.nbricks && (mask[b] & m) != m) atomicOr(reinterpret_cast<unsigned long long*>(mask + b), m);
  }
}
// keep[i]: point i of B+ is a marked node or a Laplacian neighbour of one
__global__ void k_keep_near(BrickView v, const uint64_t* key, int64_t nplus, int dim, const uint64_t* mask,
                            uint8_t* keep) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nplus) return;
  const uint64_t k = key[i];
  const int x = key_x(k), y = key_y(k), z = dim == 3 ? key_z(k) : 0;
  bool in = mask_bit(v, mask, x, y, z) || mask_bit(v, mask, x - 1, y, z) || mask_bit(v, mask, x + 1, y, z) ||
            mask_bit(v, mask, x, y - 1, z) || mask_bit(v, mask, x, y + 1, z);
  if (dim == 3) in = in || mask_bit(v, mask, x, y, z - 1) || mask_bit(v, mask, x, y, z + 1);
  keep[i] = in;
}
__global__ void k_or_masks(uint64_t* a, const uint64_t* b, int32_t n) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] |= b[i];
}
__global__ void k_row_flags(const uint64_t* mask, int64_t nrows, int per, int64_t* flag) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < nrows) flag[t] = ((mask[t / per] >> (4 * (t % per))) & 15ull) != 0;
}
__global__ void k_row_emit(const uint64_t* mask, int64_t nrows, int per, const int64_t* pos, int64_t base,
                           uint32_t* rows) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < nrows && ((mask[t / per] >> (4 * (t % per))) & 15ull)) rows[pos[t] - base] = (uint32_t)t;
}

// FP64 lists: flags of the marked points of B, flags of the kept E-order
// positions, and their scatter.
__global__ void k_list_flags(const uint32_t* slot, int32_t n, int dim, const uint64_t* mask, int64_t* flag) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t s = slot[i];
  flag[i] = (mask[s >> (2 * dim)] >> (s & ((1u << (2 * dim)) - 1u))) & 1ull;
}
__global__ void k_list_emit(const uint32_t* slot, int32_t n, int dim, const uint64_t* mask, const int64_t* pos,
                            int64_t base, int32_t* list) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t s = slot[i];
  if ((mask[s >> (2 * dim)] >> (s & ((1u << (2 * dim)) - 1u))) & 1ull) list[pos[i] - base] = i;
}
__global__ void k_epos_flags(const uint32_t* erec, int64_t n, const uint8_t* keep, int64_t* flag) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) flag[k] = keep[erec[k] >> 6];
}
__global__ void k_epos_emit(const uint32_t* erec, int64_t n, const uint8_t* keep, const int64_t* pos, int64_t base,
                            uint32_t* epos) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n && keep[erec[k] >> 6]) epos[pos[k] - base] = (uint32_t)k;
}
__global__ void k_epos_starts(const int32_t* tile_start, int32_t ntiles, int64_t n, const int64_t* pos, int64_t base,
                              int32_t total, int32_t* tstart) {
  const int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t > ntiles) return;
  const int32_t k = t < ntiles ? tile_start[t] : (int32_t)n;
  tstart[t] = k < n ? (int32_t)(pos[k] - base) : total;
}

// flag[j]: target j (a point of B of the target level) is wanted
__global__ void k_target_flags(const uint32_t* slot, int32_t n, int dim, const uint64_t* mask, int64_t* flag) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const uint32_t s = slot[j];
  flag[j] = !mask || ((mask[s >> (2 * dim)] >> (s & ((1u << (2 * dim)) - 1u))) & 1ull);
}
__global__ void k_transfer_emit(const uint64_t* base, const float* fr, int32_t n, int dim, BrickView src,
                                const uint32_t* slot, bool dense_dst, const uint64_t* mask, const int64_t* pos,
                                int64_t base0, float4* rec, uint32_t* dst) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const uint32_t sj = slot[j];
  if (mask && !((mask[sj >> (2 * dim)] >> (sj & ((1u << (2 * dim)) - 1u))) & 1ull)) return;
  const uint64_t k = base[j];
  const int x = (int)(k & 0xffffu), y = (int)((k >> 16) & 0xffffu), z = (int)((k >> 32) & 0xffffu);
  const int32_t b = src.map[((size_t)(z >> 2) * src.nby + (y >> 2)) * src.nbx + (x >> 2)];
  const uint32_t s = ((uint32_t)max(b, 0) << (2 * dim)) | (uint32_t)((x & 3) | ((y & 3) << 2) | ((z & 3) << 4));
  const int64_t p = pos[j] - base0;
  rec[p] = make_float4(__uint_as_float(s), fr[j], fr[n + j], dim == 3 ? fr[2 * (int64_t)n + j] : 0.f);
  dst[p] = dense_dst ? sj : (uint32_t)j;
}

// ----------------------------------------------------------------- build
// out[q] = d[at[q]]
struct ScanMarks {
  static constexpr int kMax = 16;
  int64_t at[kMax];
};
__global__ void k_pick(const int64_t* d, ScanMarks m, int n, int64_t* out) {
  if ((int)threadIdx.x < n) out[threadIdx.x] = d[m.at[threadIdx.x]];
}

// At least n elements of scratch (what was there is lost).
template <typename T>
static void grow(DBuf<T>& d, size_t n, cudaStream_t st) {
  if (d.n >= n) return;
  CPM_CUDA_TRY(cudaStreamSynchronize(st));  // the old block may be in use
  d.alloc(n);
}

// The counts of all of a level's sets are scanned in one go, so that a level
// costs one wait of the host.  With a scan, its scratch and a wait per set and
// list, hierarchies without a dense inverse took 14.0 ms to build (sphere at
// dx = 1/96), 9.3 (circle at 1/640), 5.1 (sphere at 1/32), so 10.4, 6.3 and 4.1 ms
// (7.9, 5.5 and 3.3 since workspaces and tables share blocks of memory).
class CountScan {
 public:
  CountScan(DBuf<int64_t>& d, cudaStream_t st) : d_(d), st_(st) {}
  // A segment of n > 0 counts; data(q) once all segments are known.
  int segment(int64_t n) {
    CPM_CHECK(n > 0 && begin_.size() + 1 < ScanMarks::kMax, CPM_ERR_ARG, "bad scan segment");
    begin_.push_back(total_);
    total_ += n;
    return (int)begin_.size() - 1;
  }
  void allocate() {  // the counts, the entry that receives their sum, the picked values, the scan's scratch
    grow(d_, (size_t)(total_ + 1 + ScanMarks::kMax) + scan_scratch(total_ + 1), st_);
  }
  int64_t* data(int q) { return d_.get() + begin_[q]; }
  // Exclusive scan over all segments; synchronous.
  void run() {
    const int n = (int)begin_.size();
    int64_t* picked = d_.get() + total_ + 1;
    CPM_CUDA_TRY(cudaMemsetAsync(d_.get() + total_, 0, sizeof(int64_t), st_));
    scan_exclusive_async(d_.get(), total_ + 1, picked + ScanMarks::kMax, st_);
    ScanMarks m{};
    for (int q = 0; q < n; ++q) m.at[q] = begin_[q];
    m.at[n] = total_;
    k_pick<<<1, 32, 0, st_>>>(d_.get(), m, n + 1, picked);
    CPM_CUDA_TRY(cudaGetLastError());
    base_.resize(n + 1);
    CPM_CUDA_TRY(cudaMemcpyAsync(base_.data(), picked, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToHost, st_));
    CPM_CUDA_TRY(cudaStreamSynchronize(st_));
  }
  int64_t base(int q) const { return base_[q]; }                  // scanned value where segment q starts
  int64_t count(int q) const { return base_[q + 1] - base_[q]; }  // sum of segment q

 private:
  DBuf<int64_t>& d_;
  cudaStream_t st_;
  int64_t total_ = 0;
  std::vector<int64_t> begin_, base_;
};

// One set of a level: segments of its counts, and where its lists go.
namespace {
struct SetBuild {
  const uint64_t* mask = nullptr;  // null: every point of B+
  uint8_t* keep = nullptr;
  ExtUnits* units = nullptr;
  NeedSet* need = nullptr;
  int units_seg = 0, tiles_seg = 0, rows_seg = 0, list_seg = 0, epos_seg = 0;
};
}  // namespace

static void alloc_units(ExtUnits& U, int64_t ntiles, int64_t nunits, bool with_band) {
  U.ntiles = (int32_t)ntiles;
  // records of both points, band indices (two words each per unit), headers
  const size_t words = (size_t)(with_band ? 2 * nunits : 0) + (size_t)ntiles * kTileWords;
  U.data.alloc((size_t)(2 * nunits) + (words + 3) / 4);
  U.pts[0] = U.data.get();
  U.pts[1] = U.pts[0] + nunits;
  uint32_t* w = reinterpret_cast<uint32_t*>(U.pts[1] + nunits);
  for (int h = 0; h < 2; ++h) U.cidx[h] = with_band ? w + h * nunits : nullptr;
  U.tiles = w + (with_band ? 2 * nunits : 0);
}

static void alloc_need(NeedSet& S, int64_t nrows, int64_t nlist, int64_t ne, int64_t ntiles) {
  S.nrows = (int32_t)nrows;
  S.nlist = (int32_t)nlist;
  S.data.alloc((size_t)(nrows + nlist + ne + ntiles + 1));
  S.rows = S.data.get();
  S.list = reinterpret_cast<int32_t*>(S.rows + nrows);
  S.epos = S.rows + nrows + nlist;
  S.tstart = reinterpret_cast<int32_t*>(S.epos + ne);
}

void build_dense32(const Level& L, Dense32& D, const CycleCells* cyc, DenseScratch& sc, cudaStream_t st) {
  CPM_CHECK((int64_t)dense_size(L) <= (int64_t)kSlotMask, CPM_ERR_ARG, "too many bricks on one level");
  const int64_t nt = L.ntiles, np = L.nplus(), nB = L.nB;
  const int per = L.dim == 3 ? 16 : 4;
  const int64_t nrows = (int64_t)L.nbricks * per;
  auto carve = [&](Carver take) {
    take(D.bface, (size_t)2 * L.nbricks);
    take(D.bfwd, (size_t)8 * L.nbricks);
    take(D.slot, (size_t)np);
    return take.used;
  };
  D.tables.alloc(carve(Carver{}));
  carve(Carver{D.tables.get()});
  k_dense_bricks<<<nblk(L.nbricks, 256), 256, 0, st>>>(L.view(), L.bcoord.get(), L.dim, D.bface.get(),
                                                       D.bfwd.get());
  k_dense_slots<<<nblk(np, 256), 256, 0, st>>>(L.view(), L.key.get(), np, L.dim, D.slot.get());
  CPM_CUDA_TRY(cudaGetLastError());
  if (nt <= 0) return;

  // masks of the needed nodes, and the points of B+ whose w they take
  SetBuild set[3];
  int nset = 1;
  set[0].units = &D.all;
  const uint64_t* sweep_mask = nullptr;
  if (cyc && cyc->restrict_from.n > 0) {
    grow(sc.mask, (size_t)2 * L.nbricks, st);
    grow(sc.keep, (size_t)(2 * np), st);
    uint64_t *mr = sc.mask.get(), *mu = mr + L.nbricks;
    CPM_CUDA_TRY(cudaMemsetAsync(mr, 0, sizeof(uint64_t) * 2 * L.nbricks, st));
    const TransferCells &r = cyc->restrict_from, &p = cyc->prolong_from;
    k_mark_cells<<<nblk(r.n, 256), 256, 0, st>>>(r.base, r.n, L.dim, L.view(), mr);
    set[nset].mask = mr;
    set[nset].units = &D.resid.units;
    set[nset++].need = &D.resid;
    if (p.n > 0) {  // a coarse level: its sweeps can be restricted too
      k_mark_cells<<<nblk(p.n, 256), 256, 0, st>>>(p.base, p.n, L.dim, L.view(), mu);
      k_mark_stencils<<<(unsigned)nt, 32, 0, st>>>(L.view(), L.tile_brick.get(), L.tile_start.get(), L.erec.get(),
                                                   L.dim, D.bfwd.get(), mu);
      k_or_masks<<<nblk(L.nbricks, 256), 256, 0, st>>>(mu, mr, L.nbricks);
      sweep_mask = mu;
      set[nset].mask = mu;
      set[nset].units = &D.sweep.units;
      set[nset++].need = &D.sweep;
    }
    for (int q = 1; q < nset; ++q) {
      set[q].keep = sc.keep.get() + (q - 1) * np;
      k_keep_near<<<nblk(np, 256), 256, 0, st>>>(L.view(), L.key.get(), np, L.dim, set[q].mask, set[q].keep);
    }
    CPM_CUDA_TRY(cudaGetLastError());
  }

  // counts of everything, one scan
  CountScan scan(sc.counts, st);
  for (int q = 0; q < nset; ++q) {
    set[q].units_seg = scan.segment(nt);
    set[q].tiles_seg = scan.segment(nt);
    if (!set[q].need) continue;
    set[q].rows_seg = scan.segment(nrows);
    set[q].list_seg = scan.segment(nB);
    set[q].epos_seg = scan.segment(np);
  }
  const TransferIn* in[2] = {nullptr, nullptr};
  int in_seg[2] = {0, 0};
  for (int q = 0; cyc && q < 2; ++q)
    if (cyc->in[q].out && cyc->in[q].cells.n > 0) {
      in[q] = &cyc->in[q];
      in_seg[q] = scan.segment(in[q]->cells.n);
    }
  scan.allocate();
  for (int q = 0; q < nset; ++q) {
    const SetBuild& s = set[q];
    k_units_count<<<(unsigned)nt, 32, 0, st>>>(L.tile_start.get(), L.erec.get(), s.keep, scan.data(s.units_seg),
                                               scan.data(s.tiles_seg));
    if (!s.need) continue;
    k_row_flags<<<nblk(nrows, 256), 256, 0, st>>>(s.mask, nrows, per, scan.data(s.rows_seg));
    k_list_flags<<<nblk(nB, 256), 256, 0, st>>>(D.slot.get(), L.nB, L.dim, s.mask, scan.data(s.list_seg));
    k_epos_flags<<<nblk(np, 256), 256, 0, st>>>(L.erec.get(), np, s.keep, scan.data(s.epos_seg));
  }
  for (int q = 0; q < 2; ++q)
    if (in[q])
      k_target_flags<<<nblk(in[q]->cells.n, 256), 256, 0, st>>>(
          D.slot.get(), in[q]->cells.n, L.dim, in[q]->pruned ? sweep_mask : nullptr, scan.data(in_seg[q]));
  CPM_CUDA_TRY(cudaGetLastError());
  scan.run();

  for (int q = 0; q < nset; ++q) {
    const SetBuild& s = set[q];
    alloc_units(*s.units, scan.count(s.tiles_seg), scan.count(s.units_seg), s.need == nullptr);
    k_units_emit<<<(unsigned)nt, 32, 0, st>>>(
        L.view(), L.tile_brick.get(), L.tile_box.get(), L.tile_start.get(), L.erec.get(), L.efr32.get(), np, L.dim,
        s.keep, D.slot.get(), scan.data(s.units_seg), scan.base(s.units_seg), scan.data(s.tiles_seg),
        scan.base(s.tiles_seg), D.bfwd.get(), s.units->tiles, s.units->pts[0], s.units->pts[1], s.units->cidx[0],
        s.units->cidx[1]);
    if (!s.need) continue;
    const int64_t ne = scan.count(s.epos_seg);
    alloc_need(*s.need, scan.count(s.rows_seg), scan.count(s.list_seg), ne, nt);
    k_row_emit<<<nblk(nrows, 256), 256, 0, st>>>(s.mask, nrows, per, scan.data(s.rows_seg), scan.base(s.rows_seg),
                                                 s.need->rows);
    k_list_emit<<<nblk(nB, 256), 256, 0, st>>>(D.slot.get(), L.nB, L.dim, s.mask, scan.data(s.list_seg),
                                               scan.base(s.list_seg), s.need->list);
    k_epos_emit<<<nblk(np, 256), 256, 0, st>>>(L.erec.get(), np, s.keep, scan.data(s.epos_seg),
                                               scan.base(s.epos_seg), s.need->epos);
    k_epos_starts<<<nblk(nt + 1, 256), 256, 0, st>>>(L.tile_start.get(), L.ntiles, np, scan.data(s.epos_seg),
                                                     scan.base(s.epos_seg), (int32_t)ne, s.need->tstart);
  }
  for (int q = 0; q < 2; ++q) {
    if (!in[q]) continue;
    const TransferCells& c = in[q]->cells;
    DenseTransfer& T = *in[q]->out;
    T.n = (int32_t)scan.count(in_seg[q]);
    T.data.alloc((size_t)T.n + (T.n + 3) / 4);
    T.rec = T.data.get();
    T.dst = reinterpret_cast<uint32_t*>(T.rec + T.n);
    k_transfer_emit<<<nblk(c.n, 256), 256, 0, st>>>(c.base, c.fr, c.n, L.dim, in[q]->source->view(), D.slot.get(),
                                                    in[q]->dense_dst, in[q]->pruned ? sweep_mask : nullptr,
                                                    scan.data(in_seg[q]), scan.base(in_seg[q]), T.rec, T.dst);
  }
  CPM_CUDA_TRY(cudaGetLastError());
}

// ----------------------------------------------------------------- layout changes
__global__ void k_scatter32(const float* __restrict__ x, const uint32_t* __restrict__ slot, int32_t n, float* d) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[slot[i]] = x[i];
}
void launch_scatter32(const DenseView& L, const float* x, float* d, cudaStream_t st) {
  if (L.nB <= 0) return;
  k_scatter32<<<nblk(L.nB, 256), 256, 0, st>>>(x, L.slot, L.nB, d);
  count_launch();
}
__global__ void k_gather32(const float* __restrict__ d, const uint32_t* __restrict__ slot, int32_t n, float* x) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] = d[slot[i]];
}
void launch_gather32(const DenseView& L, const float* d, float* x, cudaStream_t st) {
  if (L.nB <= 0) return;
  k_gather32<<<nblk(L.nB, 256), 256, 0, st>>>(d, L.slot, L.nB, x);
  count_launch();
}
// fd = r / max|r|, brick-dense.
__global__ void k_scale_dense(const double* __restrict__ r, const double* __restrict__ norms,
                              const uint32_t* __restrict__ slot, int32_t n, float* __restrict__ fd) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) fd[slot[i]] = (float)(r[i] * norms[2]);
}
void launch_scale_dense(const DenseView& L, const double* r, const double* norms, float* fd, cudaStream_t st) {
  k_scale_dense<<<nblk(L.nB, 256), 256, 0, st>>>(r, norms, L.slot, L.nB, fd);
  count_launch();
}
// u += max|r| d
__global__ void k_axpy_dense(double* __restrict__ u, const float* __restrict__ d, const uint32_t* __restrict__ slot,
                             const double* __restrict__ norms, int32_t n) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) u[i] += norms[0] * (double)d[slot[i]];
}
void launch_axpy_dense(const DenseView& L, double* u, const float* d, const double* norms, cudaStream_t st) {
  k_axpy_dense<<<nblk(L.nB, 256), 256, 0, st>>>(u, d, L.slot, norms, L.nB);
  count_launch();
}

void dense_static(const Level& L, Dense32& D, const float* dA, const float* c, cudaStream_t st) {
  const size_t n = dense_size(L);
  auto put = [&](DBuf<float>& d, const float* x) {
    d.alloc(n);
    CPM_CUDA_TRY(cudaMemsetAsync(d.get(), 0, n * sizeof(float), st));
    k_scatter32<<<nblk(L.nB, 256), 256, 0, st>>>(x, D.slot.get(), L.nB, d.get());
    CPM_CUDA_TRY(cudaGetLastError());
  };
  put(D.dA, dA);
  if (c) put(D.c, c);
}

}  // namespace cpm
