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
#include <algorithm>

#include "dense32.cuh"

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
#ifndef CPM_EXT_WARPS
#define CPM_EXT_WARPS 2
#endif

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
                                                   const int64_t* unit0, const int64_t* tile0,
                                                   const int32_t* bfwd, uint32_t* tiles, float4* pts0,
                                                   float4* pts1, uint32_t* cidx0, uint32_t* cidx1) {
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
  uint32_t* hdr = tiles + tile0[tile] * kTileWords;
  const int64_t u0 = unit0[tile];
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
      cidx0[p] = idx;
    }
    if ((r & 1) || r == hist[b] - 1) {  // (an odd count's last unit repeats its point)
      pts1[p] = make_float4(__uint_as_float(s | ((b >> 3) << kSlotBits)), fx, fy, fz);
      cidx1[p] = idx;
    }
  }
}

static void build_units(const Level& L, const Dense32& D, const uint8_t* keep, ExtUnits& out, cudaStream_t st) {
  const int64_t nt = L.ntiles;
  out.ntiles = 0;
  if (nt <= 0) return;
  DBuf<int64_t> nu(nt), used(nt);
  k_units_count<<<(unsigned)nt, 32, 0, st>>>(L.tile_start.get(), L.erec.get(), keep, nu.get(), used.get());
  CPM_CUDA_TRY(cudaGetLastError());
  const int64_t nunits = scan_exclusive_i64(nu.get(), nt, st);
  out.ntiles = (int32_t)scan_exclusive_i64(used.get(), nt, st);
  out.tiles.alloc((size_t)out.ntiles * kTileWords);
  for (int h = 0; h < 2; ++h) {
    out.pts[h].alloc((size_t)nunits);
    out.cidx[h].alloc((size_t)nunits);
  }
  k_units_emit<<<(unsigned)nt, 32, 0, st>>>(L.view(), L.tile_brick.get(), L.tile_box.get(), L.tile_start.get(),
                                            L.erec.get(), L.efr32.get(), L.nplus(), L.dim, keep, D.slot.get(),
                                            nu.get(), used.get(), D.bfwd.get(), out.tiles.get(), out.pts[0].get(),
                                            out.pts[1].get(), out.cidx[0].get(), out.cidx[1].get());
  CPM_CUDA_TRY(cudaGetLastError());
}

void build_dense32(const Level& L, Dense32& D, cudaStream_t st) {
  CPM_CHECK((int64_t)dense_size(L) <= (int64_t)kSlotMask, CPM_ERR_ARG, "too many bricks on one level");
  D.bface.alloc((size_t)2 * L.nbricks);
  D.bfwd.alloc((size_t)8 * L.nbricks);
  D.slot.alloc((size_t)L.nplus());
  k_dense_bricks<<<nblk(L.nbricks, 256), 256, 0, st>>>(L.view(), L.bcoord.get(), L.dim, D.bface.get(),
                                                       D.bfwd.get());
  k_dense_slots<<<nblk(L.nplus(), 256), 256, 0, st>>>(L.view(), L.key.get(), L.nplus(), L.dim, D.slot.get());
  CPM_CUDA_TRY(cudaGetLastError());
  build_units(L, D, nullptr, D.all, st);
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
  v.tiles = D.all.tiles.get();
  for (int h = 0; h < 2; ++h) {
    v.pts[h] = D.all.pts[h].get();
    v.cidx[h] = D.all.cidx[h].get();
  }
  v.ntiles = D.all.ntiles;
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
  if (nib & 1u) v.x = __ldg(p);
  if (nib & 2u) v.y = __ldg(p + (nib & 1u));
  if (nib & 4u) v.z = __ldg(p + __popc(nib & 3u));
  if (nib & 8u) v.w = __ldg(p + __popc(nib & 7u));
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
// dx = 1/256, 8.16 M points: 74 us, against 108 us for one thread per point on
// boxes gathered value by value from band order (16 row loads per point).
// Chunks of up to six points whose 64 values stay in registers halve the row
// loads again but leave 13 warps on an SM: 111 us.
template <int DIM, bool CIN, bool COUT, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, kExtThreadsSM / (32 * WARPS))
    k_extend_units(DenseView L, const float* __restrict__ u, float* __restrict__ w, int32_t npts) {
  constexpr int NC = DIM == 3 ? 4 : 1, RS = kRowStride, NH = DIM == 3 ? 2 : 1;
  __shared__ __align__(16) float box[WARPS][DIM == 3 ? 7 * kPlaneStride : 8 * RS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* win = box[warp];
  const int32_t tile = blockIdx.x * WARPS + warp;
  if (tile >= L.ntiles) return;
  const uint32_t hdr = __ldg(L.tiles + (size_t)tile * kTileWords + min(lane, kTileWords - 1));
    const uint32_t tbox = __shfl_sync(0xffffffffu, hdr, kTileBox);
    const int32_t beg = (int32_t)__shfl_sync(0xffffffffu, hdr, kTileBeg);
    const int32_t end = (int32_t)__shfl_sync(0xffffffffu, hdr, kTileEnd);
    int32_t k = beg + lane;
    float4 ra, rb;
    if (k < end) {
      ra = __ldg(L.pts[0] + k);
      rb = __ldg(L.pts[1] + k);
    }
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
        lo[h] = __ldg(reinterpret_cast<const float4*>(u + ((size_t)blo << (2 * DIM))) + row);
        if (xhi > 0) hi[h] = __ldg(reinterpret_cast<const float4*>(u + ((size_t)bhi << (2 * DIM))) + row);
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
      const int32_t ia = (int32_t)__ldg(L.cidx[0] + k), ib = (int32_t)__ldg(L.cidx[1] + k);
      if (ia < npts) w[ia] = va;
      if (ib < npts) w[ib] = vb;
    } else {
      w[sa & kSlotMask] = va;
      w[sb & kSlotMask] = vb;
    }
    if (k + 32 < end) {
      ra = __ldg(L.pts[0] + k + 32);
      rb = __ldg(L.pts[1] + k + 32);
    }
    }
}

// Launch shapes (variant 0, 1, 2): one, two or four tiles (warps) per CTA.
template <int DIM, bool CIN, bool COUT>
static void extend_units(const DenseView& L, int variant, const float* u, float* w, int32_t npts,
                         cudaStream_t st) {
  if (L.ntiles <= 0) return;
  if (variant == 2)
    k_extend_units<DIM, CIN, COUT, 4><<<nblk(L.ntiles, 4), 128, 0, st>>>(L, u, w, npts);
  else if (variant == 1)
    k_extend_units<DIM, CIN, COUT, 2><<<nblk(L.ntiles, 2), 64, 0, st>>>(L, u, w, npts);
  else
    k_extend_units<DIM, CIN, COUT, 1><<<L.ntiles, 32, 0, st>>>(L, u, w, npts);
}

static void extend32(const DenseView& L, int variant, Vec32<const float> u, float* w, cudaStream_t st) {
  if (L.dim == 3) {
    if (u.dense) extend_units<3, false, false>(L, variant, u.dense, w, 0, st);
    else extend_units<3, true, false>(L, variant, u.compact, w, 0, st);
  } else {
    if (u.dense) extend_units<2, false, false>(L, variant, u.dense, w, 0, st);
    else extend_units<2, true, false>(L, variant, u.compact, w, 0, st);
  }
}

void launch_extend32(const DenseView& L, Vec32<const float> u, float* w, cudaStream_t st) {
  extend32(L, L.variant, u, w, st);
  count_launch();
}

void launch_extend32_compact(const DenseView& L, const float* u, float* w, int32_t npts, cudaStream_t st) {
  if (L.dim == 3) extend_units<3, true, true>(L, L.variant, u, w, npts, st);
  else extend_units<2, true, true>(L, L.variant, u, w, npts, st);
  count_launch();
}

int tune_extend32(const DenseView& L, const float* u, float* w, cudaStream_t st, float ms[3]) {
  int best = 0;
  for (int v = 0; v < 3; ++v) ms[v] = 0.f;
  if (L.ntiles <= 0) return best;
  cudaEvent_t e0, e1;
  CPM_CUDA_TRY(cudaEventCreate(&e0));
  CPM_CUDA_TRY(cudaEventCreate(&e1));
  constexpr int kReps = 3;
  const Vec32<const float> uv{u, nullptr};
  for (int v = 0; v < 3; ++v) {
    extend32(L, v, uv, w, st);  // warm-up
    CPM_CUDA_TRY(cudaEventRecord(e0, st));
    for (int r = 0; r < kReps; ++r) extend32(L, v, uv, w, st);
    CPM_CUDA_TRY(cudaEventRecord(e1, st));
    CPM_CUDA_TRY(cudaEventSynchronize(e1));
    CPM_CUDA_TRY(cudaEventElapsedTime(&ms[v], e0, e1));
    ms[v] /= kReps;
    if (ms[v] < ms[best]) best = v;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  CPM_CUDA_TRY(cudaGetLastError());
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
// indices.  Unit sphere, dx = 1/256, 6.8 M points: 47 us a Jacobi sweep (53 us
// with the table).
template <int DIM, int MODE, bool CIN>
__global__ void __launch_bounds__(256) k_lap_rows(DenseView L, const float* u, const float* __restrict__ w,
                                                  const float* __restrict__ f, float cval, Vec32<float> out,
                                                  float* __restrict__ fd) {
  constexpr int ROWS = DIM == 3 ? 16 : 4, SH = 2 * DIM;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int32_t b = (int32_t)(t / ROWS);
  const int row = (int)(t % ROWS);
  if (b >= L.nbricks) return;
  const int y = row & 3, z = row >> 2;
  const size_t s0 = ((size_t)b << SH) + 4 * row;
  auto load4 = [](const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); };
  const int4 fa = __ldg(L.bface + 2 * (int64_t)b);
  const int4 fb = DIM == 3 ? __ldg(L.bface + 2 * (int64_t)b + 1) : make_int4(0, 0, 0, 0);
  const bool ordered = CIN || !out.dense;  // band-order data on either side
  const uint64_t m = ordered ? __ldg(L.bmask + b) : 0ull;
  const int32_t start = ordered ? __ldg(L.bstart + b) : 0;
  const float4 w0 = load4(w + s0);
  float4 uu, ff = make_float4(0.f, 0.f, 0.f, 0.f), dd = ff, cc = make_float4(cval, cval, cval, cval);
  if (!CIN) {
    uu = *reinterpret_cast<const float4*>(u + s0);
    if (MODE != LAP_APPLY) ff = load4(f + s0);
  }
  if (MODE != LAP_APPLY && MODE != LAP_RESID) dd = load4(L.dA + s0);
  if (MODE != LAP_APPLY && L.c) cc = load4(L.c + s0);
  auto row4 = [&](int32_t bb, int rr) { return load4(w + ((size_t)bb << SH) + 4 * rr); };
  const float4 ym = row4(y > 0 ? b : fa.z, y > 0 ? row - 1 : row + 3);
  const float4 yp = row4(y < 3 ? b : fa.w, y < 3 ? row + 1 : row - 3);
  float4 zm = make_float4(0.f, 0.f, 0.f, 0.f), zp = zm;
  if (DIM == 3) {
    zm = row4(z > 0 ? b : fb.x, z > 0 ? row - 4 : row + 12);
    zp = row4(z < 3 ? b : fb.y, z < 3 ? row + 4 : row - 12);
  }
  const float xm = __ldg(w + ((size_t)fa.x << SH) + 4 * row + 3);
  const float xp = __ldg(w + ((size_t)fa.y << SH) + 4 * row);
  const uint32_t nib = (uint32_t)(m >> (4 * row)) & 15u;
  const int32_t i0 = start + __popcll(m & ((1ull << (4 * row)) - 1ull));
  const int32_t off[4] = {0, (int)(nib & 1u), __popc(nib & 3u), __popc(nib & 7u)};
  if (CIN) {
    float a4[4] = {0.f, 0.f, 0.f, 0.f}, b4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < 4; ++a)
      if ((nib >> a) & 1u) {
        a4[a] = u[i0 + off[a]];
        if (MODE != LAP_APPLY) b4[a] = __ldg(f + i0 + off[a]);
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
                  Vec32<float> out, float* fd, cudaStream_t st) {
  if (L.nbricks <= 0) return;
  const unsigned g = nblk((int64_t)L.nbricks * (L.dim == 3 ? 16 : 4), 256);
  if (L.dim == 3) {
    if (u.dense) k_lap_rows<3, MODE, false><<<g, 256, 0, st>>>(L, u.dense, w, f, cval, out, nullptr);
    else k_lap_rows<3, MODE, true><<<g, 256, 0, st>>>(L, u.compact, w, f, cval, out, fd);
  } else {
    if (u.dense) k_lap_rows<2, MODE, false><<<g, 256, 0, st>>>(L, u.dense, w, f, cval, out, nullptr);
    else k_lap_rows<2, MODE, true><<<g, 256, 0, st>>>(L, u.compact, w, f, cval, out, fd);
  }
  count_launch();
}

void launch_lap32(const DenseView& L, LapMode mode, Vec32<const float> u, const float* w, const float* f,
                  float cval, Vec32<float> out, float* fd, cudaStream_t st) {
  if (mode == LAP_APPLY) lap32<LAP_APPLY>(L, u, w, f, cval, out, fd, st);
  if (mode == LAP_RESID) lap32<LAP_RESID>(L, u, w, f, cval, out, fd, st);
  if (mode == LAP_JACOBI) lap32<LAP_JACOBI>(L, u, w, f, cval, out, fd, st);
  if (mode == LAP_JAC_RED) lap32<LAP_JAC_RED>(L, u, w, f, cval, out, fd, st);
  if (mode == LAP_JAC_BLACK) lap32<LAP_JAC_BLACK>(L, u, w, f, cval, out, fd, st);
}

__global__ void k_scatter32(const float* __restrict__ x, const uint32_t* __restrict__ slot, int32_t n, float* d) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[slot[i]] = x[i];
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
