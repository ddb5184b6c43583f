// Explicit FP64 inverse of the coarsest-level matrix (Algorithm 4.1 step 2, at
// setup): in-place Gauss-Jordan with partial pivoting, in blocks of kBlk
// columns.
//
// Eliminating a set of columns K with pivot rows r_j turns A into T A, where
// T e_i = e_i for the rows that are not pivots; the columns K are replaced by
// the columns T e_{r_j} (the multipliers), and every other column a becomes
//   a_i (0 for pivot rows) + sum_j (T e_{r_j})_i a_{r_j}.
// So a block is: the multipliers Q (n x kBlk) by elimination inside the block's
// own columns, in panels of kPan; then one rank-kBlk product Q U over all other
// columns, U the pivot rows as they were.  Rows are never exchanged: after the
// last block A holds the inverse with rows and columns permuted by the pivots.
//
// The product has 2 n^3 flops, 0.62 s at this chip's FP64 rate for 7190 rows.
// It is evaluated exactly enough on the tensor cores instead (the error-free
// slicing of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012): every
// row of Q and every column of U is scaled by a power of two and cut into
// kSlices balanced base-256 digits, integers of at most 128 in magnitude and
// so exact in BF16.  A product of two slices over kBlk = 128 terms is an
// integer below 2^21, and the at most seven products of one weight sum below
// 2^24, exact in FP32 accumulators.  The weights are combined in 64-bit
// integers and added to A with one FP64 operation per entry.  56 bits of every
// operand enter, below the rounding of an FP64 product relative to the largest
// entry of the row and the column: direct solves on 16 levels (circles 312 ..
// 4536 points, spheres 4358 .. 7190, an ellipsoid; constant coefficients) are
// 0.66 to 1.41 times as far from the solution as with FP64 elimination, 0.97 in
// the mean.
//
// An entry far below its row's and its column's largest keeps few of those 56
// bits, so the slices serve matrices whose rows have one scale (kMaxSpread).
// Others (a diffusion coefficient or a c over decades) and matrices with an Inf
// or a NaN, which no integer carries on, take the products in FP64.
//
// 7190 rows: 0.15 s (product 86 ms, panels 33 ms, panel updates 18 ms), against
// 1.36 s for 7190 rank-one steps over the matrix in HBM.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "ops.cuh"

namespace cg = cooperative_groups;

namespace cpm {

static unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr int kBlk = 128;   // columns per block (the K of the product)
constexpr int kPan = 16;    // columns eliminated by one panel kernel
constexpr int kSlices = 7;
// Largest ratio of the rows' scales (largest magnitude off the diagonal) and of
// the diagonal's magnitudes for the sliced products.  Row-wise backward error of
// direct solves in units of 2^-53, circles of 360 to 712 points, slices against
// FP64 products.  Ratio off the diagonal (a over decades) 13 to 17: 1116, 605 at
// worst; 27: 870, 246; 140: 2200, 240; 1.5e4: 9819, 26; 1.9e6: 498425, 90.  On
// the diagonal (c over decades) 8: 61, 41; 22: 125, 31; 2e3: 500, 21.  Levels
// with constant coefficients have ratios of 1.3 to 8.8.
constexpr double kMaxSpread = 16.0;

// ----------------------------------------------------------------- panels
// One cluster eliminates `steps` <= kPan columns c0 .. of Q (n rows of kBlk
// doubles).  The thread blocks share the rows; at each step every block offers
// its largest unused entry of the column with the row that holds it to all the
// others through distributed shared memory, and after one cluster barrier each
// picks the same winner and updates its rows.  With a row per thread (ONE) the
// rows stay in registers.  Latency-bound: a cluster barrier, two block
// reductions and 16 FP64 operations per row and step; magnitudes are compared
// as integers, since the FP64 pipe would need longer for the comparisons than
// for the update.
constexpr int kPanThreads = 512;
constexpr int kPanMaxCtas = 16;

// An entry on offer: the bits of its magnitude (ordered as an integer), its row.
struct Offer {
  unsigned long long key;
  int32_t row;
};
// The larger magnitude, then the smaller row (-1: none).
__device__ __forceinline__ bool better(const Offer& a, const Offer& b) {
  return a.key > b.key || (a.key == b.key && (unsigned)a.row < (unsigned)b.row);
}
template <int LANES>
__device__ __forceinline__ void best_offer(Offer& o, int& tag) {
#pragma unroll
  for (int d = LANES / 2; d > 0; d >>= 1) {
    const Offer q{__shfl_xor_sync(0xffffffffu, o.key, d), __shfl_xor_sync(0xffffffffu, o.row, d)};
    const int t = __shfl_xor_sync(0xffffffffu, tag, d);
    if (better(q, o)) {
      o = q;
      tag = t;
    }
  }
}
__device__ __forceinline__ Offer make_offer(double v, int32_t row) {
  // a NaN is no pivot, but an unused row stays on offer
  const double m = v == v ? fabs(v) : 0.0;
  return {(unsigned long long)__double_as_longlong(m), row};
}

struct PanelRow {
  double x[kPan];
  __device__ __forceinline__ void load(const double* q) {
#pragma unroll
    for (int c = 0; c < kPan / 2; ++c) {
      const double2 t = reinterpret_cast<const double2*>(q)[c];
      x[2 * c] = t.x;
      x[2 * c + 1] = t.y;
    }
  }
  __device__ __forceinline__ void store(double* q) const {
#pragma unroll
    for (int c = 0; c < kPan / 2; ++c) reinterpret_cast<double2*>(q)[c] = make_double2(x[2 * c], x[2 * c + 1]);
  }
  __device__ __forceinline__ double at(int j) const {
    double v = x[0];
#pragma unroll
    for (int c = 1; c < kPan; ++c) v = c == j ? x[c] : v;
    return v;
  }
  // step j with the scaled pivot row s
  __device__ __forceinline__ void step(int j, const double* s, bool pivot) {
    const double m = pivot ? -1.0 : at(j);
#pragma unroll
    for (int c = 0; c < kPan; ++c) {
      const double old = pivot || c == j ? 0.0 : x[c];
      x[c] = old - m * s[c];
    }
  }
};

template <bool ONE>
__global__ void __launch_bounds__(kPanThreads) k_gj_panel(double* Q, int32_t n, int c0, int steps, int32_t first,
                                                          int32_t* rows, int32_t* owner, double* U, int32_t* err) {
  __shared__ Offer offers[2][kPanMaxCtas];
  __shared__ double orow[2][kPanMaxCtas][kPan];
  __shared__ Offer woffer[kPanThreads / 32];
  __shared__ double crow[kPan], srow[kPan];
  cg::cluster_group cluster = cg::this_cluster();
  const int nc = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int32_t i0 = rank * kPanThreads + tid, stride = nc * kPanThreads;
  const Offer none{0ull, -1};
  Offer best = none;
  PanelRow own;
  bool own_used = true;
  if (ONE) {
    if (i0 < n) {
      own.load(Q + (size_t)i0 * kBlk + c0);
      own_used = owner[i0] >= 0;
      if (!own_used) best = make_offer(own.x[0], i0);
    }
  } else {
    for (int32_t i = i0; i < n; i += stride)
      if (owner[i] < 0) {
        const Offer o = make_offer(Q[(size_t)i * kBlk + c0], i);
        if (better(o, best)) best = o;
      }
  }
  for (int j = 0; j < steps; ++j) {
    const int par = j & 1;
    // the block's candidate and its row
    int tag = 0;
    best_offer<32>(best, tag);
    if (lane == 0) woffer[warp] = best;
    __syncthreads();
    best = woffer[lane % (kPanThreads / 32)];
    best_offer<kPanThreads / 32>(best, tag);
    if (ONE) {
      if (i0 == best.row) {
#pragma unroll
        for (int c = 0; c < kPan; ++c) crow[c] = own.x[c];
      }
      __syncthreads();
    }
    // to every block (the buffers alternate: a block is at most one step ahead)
    if (tid < nc * kPan) {
      const int d = tid / kPan, e = tid % kPan;
      const double v = best.row < 0 ? 0.0 : ONE ? crow[e] : Q[(size_t)best.row * kBlk + c0 + e];
      *cluster.map_shared_rank(&orow[par][rank][e], d) = v;
      if (e == 0) *cluster.map_shared_rank(&offers[par][rank], d) = best;
    }
    cluster.sync();
    int win = lane % kPanMaxCtas;
    Offer o = win < nc ? offers[par][win] : none;
    best_offer<kPanMaxCtas>(o, win);
    const int32_t p = o.row;
    if (tid < kPan) {
      const double a = orow[par][win][j];
      const double inv = a != 0.0 ? 1.0 / a : 0.0;
      srow[tid] = tid == j ? inv : orow[par][win][tid] * inv;
    }
    if (rank == 0 && tid == 0) {
      rows[c0 + j] = p;
      if (!(__longlong_as_double((long long)o.key) > 1e-300)) atomicOr(err, 1);
    }
    __syncthreads();
    best = none;
    if (ONE) {
      if (i0 < n) {
        own.step(j, srow, i0 == p);
        if (i0 == p) {
          owner[i0] = first + j;
          own_used = true;
        }
        if (!own_used) best = make_offer(own.at(j + 1 < kPan ? j + 1 : j), i0);
      }
    } else {
      for (int32_t i = i0; i < n; i += stride) {
        double* q = Q + (size_t)i * kBlk + c0;
        PanelRow r;
        r.load(q);
        r.step(j, srow, i == p);
        r.store(q);
        if (i == p) owner[i] = first + j;
        else if (owner[i] < 0) {
          const Offer f = make_offer(r.at(j + 1 < kPan ? j + 1 : j), i);
          if (better(f, best)) best = f;
        }
      }
    }
  }
  if (ONE && i0 < n) own.store(Q + (size_t)i0 * kBlk + c0);
  cluster.sync();
  // the pivot rows of the block's other columns, as they were
  if (rank == 0)
    for (int e = tid; e < steps * kBlk; e += kPanThreads)
      U[e] = Q[(size_t)rows[c0 + e / kBlk] * kBlk + e % kBlk];
}

// The panel's transformation on the block's other columns.
constexpr int kInnerRows = 64;
__global__ void __launch_bounds__(256) k_gj_inner(double* Q, int32_t n, int c0, int steps, int32_t first,
                                                  const int32_t* owner, const double* U) {
  __shared__ double P[kInnerRows][kPan];
  const int tid = threadIdx.x, c = tid & (kBlk - 1), half = tid >> 7;
  const int32_t r0 = blockIdx.x * kInnerRows;
  for (int e = tid; e < kInnerRows * kPan; e += 256) {
    const int32_t i = r0 + e / kPan;
    P[e / kPan][e % kPan] = i < n && e % kPan < steps ? Q[(size_t)i * kBlk + c0 + e % kPan] : 0.0;
  }
  double u[kPan];
#pragma unroll
  for (int j = 0; j < kPan; ++j) u[j] = j < steps ? U[j * kBlk + c] : 0.0;
  __syncthreads();
  if (c >= c0 && c < c0 + steps) return;
  for (int r = half; r < kInnerRows && r0 + r < n; r += 2) {
    const int32_t i = r0 + r, o = owner[i];
    double s = o >= first && o < first + steps ? 0.0 : Q[(size_t)i * kBlk + c];
#pragma unroll
    for (int j = 0; j < kPan; ++j) s += P[r][j] * u[j];
    Q[(size_t)i * kBlk + c] = s;
  }
}

// Q = columns k0 .. k0 + b - 1 of A (zero beyond b).
__global__ void k_gj_gather(const double* A, int32_t n, int32_t k0, int b, double* Q) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)n * kBlk) return;
  const int c = (int)(e % kBlk);
  Q[e] = c < b ? A[(e / kBlk) * n + k0 + c] : 0.0;
}
__global__ void k_gj_put(double* A, int32_t n, int32_t k0, int b, const double* Q) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)n * kBlk) return;
  const int c = (int)(e % kBlk);
  if (c < b) A[(e / kBlk) * n + k0 + c] = Q[e];
}

// ----------------------------------------------------------------- row scales
// out[0], out[1]: the smallest and the largest row scale (largest magnitude off
// the diagonal, as bits; zeros are left out), out[2], out[3]: the same of the
// diagonal, out[4]: whether any entry is not finite.  One warp per row.
__global__ void __launch_bounds__(256) k_row_scales(const double* __restrict__ A, int32_t n,
                                                    unsigned long long* out) {
  const int32_t i = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  double m = 0.0;
  bool bad = false;
  for (int32_t j = lane; j < n; j += 32) {
    const double x = fabs(A[(size_t)i * n + j]);
    bad |= !isfinite(x);
    if (j != i) m = fmax(m, x);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  bad = __any_sync(0xffffffffu, bad);
  if (lane > 1) return;
  const double x = lane == 0 ? m : fabs(A[(size_t)i * n + i]);
  if (x > 0.0) {
    atomicMin(out + 2 * lane, (unsigned long long)__double_as_longlong(x));
    atomicMax(out + 2 * lane + 1, (unsigned long long)__double_as_longlong(x));
  }
  if (bad) atomicOr(out + 4, 1ull);
}
// Whether the products of an inverse of A may be sliced.  Synchronous.
static bool sliced_products(const double* A, int32_t n, cudaStream_t st) {
  DBuf<unsigned long long> d(5);
  unsigned long long h[5] = {~0ull, 0ull, ~0ull, 0ull, 0ull};
  CPM_CUDA_TRY(cudaMemcpyAsync(d.get(), h, sizeof(h), cudaMemcpyHostToDevice, st));
  k_row_scales<<<nblk(n, 8), 256, 0, st>>>(A, n, d.get());
  CPM_CUDA_TRY(cudaGetLastError());
  CPM_CUDA_TRY(cudaMemcpyAsync(h, d.get(), sizeof(h), cudaMemcpyDeviceToHost, st));
  CPM_CUDA_TRY(cudaStreamSynchronize(st));
  auto one_scale = [&](int k) {
    double lo, hi;
    std::memcpy(&lo, &h[k], sizeof(lo));
    std::memcpy(&hi, &h[k + 1], sizeof(hi));
    return h[k + 1] == 0 || hi <= kMaxSpread * lo;
  };
  return h[4] == 0 && one_scale(0) && one_scale(2);
}

// ----------------------------------------------------------------- slices
// The power of two 2^e above twice the largest magnitude m (so that the scaled
// values are at most 1/2), and the digits of x: x = 2^e sum_s d_s 256^-(s+1).
__device__ __forceinline__ int scale_exp(double m) { return m > 0.0 ? ilogb(m) + 2 : 0; }
__device__ __forceinline__ void digits(double x, int e, __nv_bfloat16 (&d)[kSlices]) {
  double t = scalbn(x, 8 - e);
#pragma unroll
  for (int s = 0; s < kSlices; ++s) {
    const double r = rint(t);
    d[s] = __float2bfloat16_rn((float)r);
    t = (t - r) * 256.0;
  }
}

// Rows of Q: one warp per row, four columns per lane.
__global__ void __launch_bounds__(256) k_slice_rows(const double* Q, int32_t n, __nv_bfloat16* S, int32_t* ex) {
  const int32_t i = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  double x[4], m = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    x[q] = Q[(size_t)i * kBlk + 4 * lane + q];
    m = fmax(m, fabs(x[q]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int e = scale_exp(m);
  if (lane == 0) ex[i] = e;
  __nv_bfloat16 d[4][kSlices];
#pragma unroll
  for (int q = 0; q < 4; ++q) digits(x[q], e, d[q]);
#pragma unroll
  for (int s = 0; s < kSlices; ++s) {
    __nv_bfloat162 v[2] = {__nv_bfloat162(d[0][s], d[1][s]), __nv_bfloat162(d[2][s], d[3][s])};
    *reinterpret_cast<uint2*>(S + ((size_t)s * n + i) * kBlk + 4 * lane) = *reinterpret_cast<uint2*>(v);
  }
}

// Columns of U = the pivot rows of A, transposed: S[s][c][j] from A[rows[j]][c].
constexpr int kSliceCols = 32;
__global__ void __launch_bounds__(256) k_slice_cols(const double* A, int32_t n, const int32_t* rows, int b,
                                                    __nv_bfloat16* S, int32_t* ex) {
  __shared__ double tile[kBlk][kSliceCols + 1];
  const int32_t c0 = blockIdx.x * kSliceCols;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int j = warp; j < kBlk; j += 8)
    tile[j][lane] = j < b && c0 + lane < n ? A[(size_t)rows[j] * n + c0 + lane] : 0.0;
  __syncthreads();
  for (int c = warp; c < kSliceCols && c0 + c < n; c += 8) {
    double x[4], m = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      x[q] = tile[4 * lane + q][c];
      m = fmax(m, fabs(x[q]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    const int e = scale_exp(m);
    if (lane == 0) ex[c0 + c] = e;
    __nv_bfloat16 d[4][kSlices];
#pragma unroll
    for (int q = 0; q < 4; ++q) digits(x[q], e, d[q]);
#pragma unroll
    for (int s = 0; s < kSlices; ++s) {
      __nv_bfloat162 v[2] = {__nv_bfloat162(d[0][s], d[1][s]), __nv_bfloat162(d[2][s], d[3][s])};
      *reinterpret_cast<uint2*>(S + ((size_t)s * n + c0 + c) * kBlk + 4 * lane) = *reinterpret_cast<uint2*>(v);
    }
  }
}

// ----------------------------------------------------------------- product
// A = (A without the pivot rows) + Q U on the columns outside the block.  A CTA
// takes consecutive tiles of kTM x kTN entries along a strip of rows: the
// strip's slices of Q stay in shared memory (115 KB), the slices of U of the
// next tile (57 KB) are copied while the current one is multiplied.  Each of
// the 16 warps holds the seven weights' accumulators of 16 x 8 entries and runs
// the 28 slice products of weight below kSlices.
constexpr int kTM = 64, kTN = 32, kProdThreads = 512;
struct GjShared {
  __nv_bfloat16 a[kSlices][kTM * kBlk];
  __nv_bfloat16 b[2][kSlices][kTN * kBlk];
};
static_assert(sizeof(GjShared) <= 227 * 1024, "shared memory of one block");

// 16-byte word w of row r of a slice tile (rows of 256 bytes, words swizzled so
// that eight rows' equal words lie in different banks).
__device__ __forceinline__ int swz(int r, int w) { return r * kBlk + ((w ^ (r & 7)) << 3); }
__device__ __forceinline__ void cp16(void* smem, const void* gmem, bool ok) {
  const uint32_t bytes = ok ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t (&d)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
               : "r"(addr));
}
__device__ __forceinline__ void mma16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// v = sum over the slice products of weight d = s + q < kSlices of the warp's
// 16 x 8 entries, in units of 256^-7 (the last weight rounded).  Weight s is
// complete after the products of slice s of Q and moves into v; the
// accumulators shift down, so that the loop over s stays rolled (unrolled, it
// spilled 200 registers).
__device__ __forceinline__ void slice_products(uint32_t As, uint32_t Bs, int wm, int wn, long long (&v)[4]) {
  constexpr uint32_t kSliceA = kTM * kBlk * 2, kSliceB = kTN * kBlk * 2;  // bytes of a slice's tile
  const int lane = threadIdx.x & 31;
  const int ra = wm + (lane & 15), wa = lane >> 4, rb = wn + (lane & 7), wb = lane >> 3;
  uint32_t ao[8], bo[4];
#pragma unroll
  for (int kc = 0; kc < 8; ++kc) ao[kc] = As + 2 * swz(ra, 2 * kc + wa);
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2) bo[k2] = Bs + 2 * swz(rb, 4 * k2 + wb);
  float acc[kSlices][4];
#pragma unroll
  for (int d = 0; d < kSlices; ++d)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[d][e] = 0.f;
#pragma unroll 1
  for (int s = 0; s < kSlices; ++s) {
    uint32_t a[8][4];
#pragma unroll
    for (int kc = 0; kc < 8; ++kc) ldsm4(a[kc], ao[kc] + s * kSliceA);
#pragma unroll
    for (int q = 0; q < kSlices; ++q) {
      if (q >= kSlices - s) break;
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) {
        uint32_t bb[4];
        ldsm4(bb, bo[k2] + q * kSliceB);
        mma16(acc[q], a[2 * k2], bb[0], bb[1]);
        mma16(acc[q], a[2 * k2 + 1], bb[2], bb[3]);
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int x = __float2int_rn(acc[0][e]);
      v[e] += s < kSlices - 1 ? (long long)x << (40 - 8 * s) : (long long)((x + 128) >> 8);
#pragma unroll
      for (int d = 0; d + 1 < kSlices; ++d) acc[d][e] = acc[d + 1][e];
      acc[kSlices - 1][e] = 0.f;
    }
  }
}

__global__ void __launch_bounds__(kProdThreads, 1) k_gj_product(double* A, int32_t n, int32_t k0, int b,
                                                    const __nv_bfloat16* QS, const int32_t* qe,
                                                    const __nv_bfloat16* US, const int32_t* ue,
                                                    const int32_t* owner, int32_t ntm, int32_t ntn) {
  extern __shared__ __align__(16) unsigned char raw[];
  GjShared& S = *reinterpret_cast<GjShared*>(raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = 16 * (warp & 3), wn = 8 * (warp >> 2);
  const int64_t tiles = (int64_t)ntm * ntn;
  const int64_t t0 = tiles * blockIdx.x / gridDim.x, t1 = tiles * (blockIdx.x + 1) / gridDim.x;
  auto fetch_b = [&](int64_t t, int buf) {
    const int32_t c0 = (int32_t)(t % ntn) * kTN;
#pragma unroll 1
    for (int e = tid; e < kSlices * kTN * 16; e += kProdThreads) {
      const int s = e / (kTN * 16), r = (e / 16) % kTN, w = e % 16;
      const bool ok = c0 + r < n;
      cp16(&S.b[buf][s][swz(r, w)], US + ((size_t)s * n + (ok ? c0 + r : 0)) * kBlk + 8 * w, ok);
    }
  };
  auto fetch_a = [&](int64_t t) {
    const int32_t r0 = (int32_t)(t / ntn) * kTM;
#pragma unroll 1
    for (int e = tid; e < kSlices * kTM * 16; e += kProdThreads) {
      const int s = e / (kTM * 16), r = (e / 16) % kTM, w = e % 16;
      const bool ok = r0 + r < n;
      cp16(&S.a[s][swz(r, w)], QS + ((size_t)s * n + (ok ? r0 + r : 0)) * kBlk + 8 * w, ok);
    }
  };
  if (t0 >= t1) return;
  fetch_a(t0);
  fetch_b(t0, 0);
  int buf = 0;
  for (int64_t t = t0; t < t1; ++t, buf ^= 1) {
    if (t > t0 && t % ntn == 0) {  // a new strip of rows
      __syncthreads();
      fetch_a(t);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (t + 1 < t1) fetch_b(t + 1, buf ^ 1);
    // the thread's four entries of A, in flight during the product
    const int32_t r0 = (int32_t)(t / ntn) * kTM, c0 = (int32_t)(t % ntn) * kTN;
    double old[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int32_t i = r0 + wm + (lane >> 2) + 8 * (e >> 1), c = c0 + wn + 2 * (lane & 3) + (e & 1);
      old[e] = i < n && c < n ? A[(size_t)i * n + c] : 0.0;
    }
    long long v[4] = {0, 0, 0, 0};
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(&S.a[0][0]);
    const uint32_t sb = (uint32_t)__cvta_generic_to_shared(&S.b[buf][0][0]);
    slice_products(sa, sb, wm, wn, v);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int32_t i = r0 + wm + (lane >> 2) + 8 * (e >> 1), c = c0 + wn + 2 * (lane & 3) + (e & 1);
      if (i >= n || c >= n || (c >= k0 && c < k0 + b)) continue;
      const int32_t o = owner[i];
      const int ex = qe[i] + ue[c] - 56;
      double x = (double)v[e];
      x = ex > -1000 && ex < 1000 ? x * __hiloint2double((ex + 1023) << 20, 0) : scalbn(x, ex);
      A[(size_t)i * n + c] = (o >= k0 && o < k0 + b ? 0.0 : old[e]) + x;
    }
  }
}

// The same in FP64: R the pivot rows as they were (kBlk rows of n doubles, zero
// beyond b).  64 x 64 entries per block, 4 x 4 per thread.  Bound by the FP64
// pipe (2 n^3 flops in all: 7190 rows 0.61 s; a build with them 0.68 s, with the
// slices 0.15 s, with rank-one steps 1.35 s).
constexpr int kP64 = 64, kP64K = 16;
__global__ void k_gj_rows(const double* A, int32_t n, const int32_t* rows, int b, double* R) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)n * kBlk) return;
  const int j = (int)(e / n);
  R[e] = j < b ? A[(size_t)rows[j] * n + e % n] : 0.0;
}
__global__ void __launch_bounds__(256) k_gj_product64(double* A, int32_t n, int32_t k0, int b,
                                                      const double* __restrict__ Q, const double* __restrict__ R,
                                                      const int32_t* __restrict__ owner) {
  __shared__ double qs[kP64K][kP64 + 1], rs[kP64K][kP64];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int32_t i0 = blockIdx.y * kP64, c0 = blockIdx.x * kP64;
  double acc[4][4] = {};
  for (int j0 = 0; j0 < kBlk; j0 += kP64K) {
    for (int e = tid; e < kP64 * kP64K; e += 256) {
      const int32_t i = i0 + e / kP64K, c = c0 + e % kP64;
      qs[e % kP64K][e / kP64K] = i < n ? Q[(size_t)i * kBlk + j0 + e % kP64K] : 0.0;
      rs[e / kP64][e % kP64] = c < n ? R[(size_t)(j0 + e / kP64) * n + c] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kP64K; ++j) {
      double q[4], r[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        q[k] = qs[j][ty + 16 * k];
        r[k] = rs[j][tx + 16 * k];
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] += q[a] * r[c];
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int32_t i = i0 + ty + 16 * a, c = c0 + tx + 16 * k;
      if (i >= n || c >= n || (c >= k0 && c < k0 + b)) continue;
      const int32_t o = owner[i];
      double* x = A + (size_t)i * n + c;
      *x = (o >= k0 && o < k0 + b ? 0.0 : *x) + acc[a][k];
    }
}

// The inverse is A[rows[k]][j] at row k and column rows[j].  In place, with a
// buffer of b columns (rows moved) and then of b rows (columns moved) at a time: a
// second matrix would double the memory of the build.  owner is the inverse
// permutation of rows.  7190 rows: a build takes 150.7 ms, with a second matrix
// 150.4; with b = 128 151.7.
__global__ void k_gj_copy_columns(const double* A, int32_t n, int32_t k0, int b, double* buf) {
  const int c = blockIdx.y * blockDim.x + threadIdx.x;
  if (c < b) buf[(size_t)blockIdx.x * b + c] = A[(size_t)blockIdx.x * n + k0 + c];
}
__global__ void k_gj_move_rows(double* A, int32_t n, int32_t k0, int b, const double* buf, const int32_t* rows) {
  const int c = blockIdx.y * blockDim.x + threadIdx.x;
  if (c < b) A[(size_t)blockIdx.x * n + k0 + c] = buf[(size_t)rows[blockIdx.x] * b + c];
}
__global__ void k_gj_move_columns(double* A, int32_t n, int32_t i0, const double* buf, const int32_t* owner) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) A[(size_t)(i0 + blockIdx.y) * n + j] = buf[(size_t)blockIdx.y * n + owner[j]];
}

void invert_dense(double* A, int32_t n, cudaStream_t st, int32_t* err) {
  if (n <= 0) return;
  DBuf<double> Q((size_t)n * kBlk), U(kPan * kBlk), R;
  DBuf<__nv_bfloat16> S;  // slices of Q, then of U
  DBuf<int32_t> qe(n), ue(n), owner(n), rows(n);
  const bool sliced = n > kBlk && sliced_products(A, n, st);
  if (sliced) {
    S.alloc((size_t)2 * kSlices * n * kBlk);
  } else if (n > kBlk) {  // (one block has no product)
    R.alloc((size_t)n * kBlk);
  }
  CPM_CUDA_TRY(cudaMemsetAsync(owner.get(), 0xff, sizeof(int32_t) * n, st));
  CPM_CUDA_TRY(cudaFuncSetAttribute(k_gj_product, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sizeof(GjShared)));
  // the panel's cluster: 16 blocks where the device takes that size, else 8
  auto panel = n <= 8 * kPanThreads ? k_gj_panel<true> : k_gj_panel<false>;
  CPM_CUDA_TRY(cudaFuncSetAttribute(k_gj_panel<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  CPM_CUDA_TRY(cudaFuncSetAttribute(k_gj_panel<false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  cudaLaunchConfig_t cfg{};
  cfg.blockDim = dim3(kPanThreads);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  for (unsigned nc = kPanMaxCtas;; nc = 8) {
    at.val.clusterDim.x = nc;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(nc);
    int active = 0;
    if (nc == 8) break;
    if (cudaOccupancyMaxActiveClusters(&active, k_gj_panel<true>, &cfg) == cudaSuccess && active > 0 &&
        cudaOccupancyMaxActiveClusters(&active, k_gj_panel<false>, &cfg) == cudaSuccess && active > 0) {
      if (n <= (int32_t)nc * kPanThreads) panel = k_gj_panel<true>;
      break;
    }
    cudaGetLastError();
  }
  const int64_t nq = (int64_t)n * kBlk;
  __nv_bfloat16 *QS = S.get(), *US = sliced ? QS + (size_t)kSlices * n * kBlk : nullptr;
  const int32_t ntm = (n + kTM - 1) / kTM, ntn = (n + kTN - 1) / kTN;
  const unsigned grid = (unsigned)std::min<int64_t>((int64_t)ntm * ntn, 152);
  for (int32_t k0 = 0; k0 < n; k0 += kBlk) {
    const int b = std::min(kBlk, n - k0);
    k_gj_gather<<<nblk(nq, 256), 256, 0, st>>>(A, n, k0, b, Q.get());
    for (int c0 = 0; c0 < b; c0 += kPan) {
      const int steps = std::min(kPan, b - c0);
      CPM_CUDA_TRY(cudaLaunchKernelEx(&cfg, panel, Q.get(), n, c0, steps, k0 + c0, rows.get() + k0,
                                      owner.get(), U.get(), err));
      k_gj_inner<<<nblk(n, kInnerRows), 256, 0, st>>>(Q.get(), n, c0, steps, k0 + c0, owner.get(), U.get());
    }
    if (sliced) {
      k_slice_rows<<<nblk(n, 8), 256, 0, st>>>(Q.get(), n, QS, qe.get());
      k_slice_cols<<<nblk(n, kSliceCols), 256, 0, st>>>(A, n, rows.get() + k0, b, US, ue.get());
      k_gj_product<<<grid, kProdThreads, sizeof(GjShared), st>>>(A, n, k0, b, QS, qe.get(), US, ue.get(),
                                                        owner.get(), ntm, ntn);
    } else if (n > kBlk) {
      const dim3 g64(nblk(n, kP64), nblk(n, kP64));
      k_gj_rows<<<nblk(nq, 256), 256, 0, st>>>(A, n, rows.get() + k0, b, R.get());
      k_gj_product64<<<g64, 256, 0, st>>>(A, n, k0, b, Q.get(), R.get(), owner.get());
    }
    k_gj_put<<<nblk(nq, 256), 256, 0, st>>>(A, n, k0, b, Q.get());
    CPM_CUDA_TRY(cudaGetLastError());
  }
  // (the slices' space holds 448 columns of doubles)
  double* buf = sliced ? reinterpret_cast<double*>(S.get()) : Q.get();
  const int wide = sliced ? 2 * kSlices * kBlk / 4 : kBlk;
  for (int32_t k0 = 0; k0 < n; k0 += wide) {
    const int b = std::min(wide, n - k0);
    const dim3 g(n, nblk(b, 256));
    k_gj_copy_columns<<<g, 256, 0, st>>>(A, n, k0, b, buf);
    k_gj_move_rows<<<g, 256, 0, st>>>(A, n, k0, b, buf, rows.get());
  }
  for (int32_t i0 = 0; i0 < n; i0 += wide) {
    const int b = std::min(wide, n - i0);
    CPM_CUDA_TRY(cudaMemcpyAsync(buf, A + (size_t)i0 * n, sizeof(double) * b * n, cudaMemcpyDeviceToDevice, st));
    k_gj_move_columns<<<dim3(nblk(n, 256), b), 256, 0, st>>>(A, n, i0, buf, owner.get());
  }
  CPM_CUDA_TRY(cudaGetLastError());
  CPM_CUDA_TRY(cudaStreamSynchronize(st));
}

}  // namespace cpm
