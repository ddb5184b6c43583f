// Device operators of one level: the closest-point extension E (Sec. 3.1,
// Eq. 3.1), the operator M = diag(L) + (L - diag L) E (Sec. 2.3 Eq. 2.10,
// Remark 3.2), Jacobi smoothing (Eq. 4.1, Eq. 4.2), residuals, closest-point
// restriction and prolongation (Sec. 4.3), norms, and the setup kernels for
// diag(M) and the coarsest-level matrix.
#include <cmath>
#include <cstring>

#include "ops.cuh"
#include "gemv.cuh"
#include "pair.cuh"
#include "pdl.cuh"

#include <atomic>

namespace cpm {

static unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

static std::atomic<int64_t> g_launches{0};
static thread_local bool g_capturing = false;
void count_launch(int64_t n) {
  if (!g_capturing) g_launches.fetch_add(n, std::memory_order_relaxed);
}
void set_capturing(bool on) { g_capturing = on; }
int64_t launches_total() { return g_launches.load(std::memory_order_relaxed); }

// ----------------------------------------------------------------- weights
// 1-D cubic Lagrange weights at fraction s for nodes -1, 0, 1, 2
// (the closed forms of the proof of Theorem 3.3, a = s dx):
//   l_-1 = -s(s-1)(s-2)/6, l_0 = (s+1)(s-1)(s-2)/2,
//   l_1  = -(s+1)s(s-2)/2, l_2 = (s+1)s(s-1)/6.
template <typename T>
__device__ __forceinline__ void cubic_w(T s, T w[4]) {
  const T sm1 = s - T(1), sm2 = s - T(2), sp1 = s + T(1);
  const T a = s * sm1, b = sp1 * sm2;
  w[0] = -(a * sm2) * T(1.0 / 6.0);
  w[1] = (b * sm1) * T(0.5);
  w[2] = -(b * s) * T(0.5);
  w[3] = (a * sp1) * T(1.0 / 6.0);
}

// ----------------------------------------------------------------- block reduce
__device__ inline void block_max_sum(double m, double s, double* part) {
  __shared__ double sm[32], ss[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) { sm[wid] = m; ss[wid] = s; }
  __syncthreads();
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    m = lane < nw ? sm[lane] : 0.0;
    s = lane < nw ? ss[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
      s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    if (lane == 0) {
      part[2 * blockIdx.x] = m;
      part[2 * blockIdx.x + 1] = s;
    }
  }
}

// ----------------------------------------------------------------- M stencil
template <typename T>
static unsigned lap_grid(const LevelView<T>& L) {
  return nblk(L.nB, 256);
}
int lap_blocks_f64(const LevelView<double>& L) { return (int)lap_grid(L); }

// MODE (LapMode, plus the Ruuth-Merriman pieces):
//   APPLY : out = M u
//   RESID : out = f - c u + M u, block partials of max|out|, sum out^2
//   JACOBI: u += (f - c u + M u) * dA (in place)
//   RESID_REL: RESID from the relative extension (w = delta, refv)
//   RM_JAC / RM_RES: band-restricted Laplacian L_B on u (ghost neighbours
//           dropped): out = u + omega (f - (cI - L_B) u) / (c + gamma), or
//           out = f - (cI - L_B) u
constexpr int LAP_RM_JAC = 8, LAP_RM_RES = 9, LAP_BAND = 10, LAP_VARD = 11;

// Stencil passes on B, one thread per band point, its 2d neighbours read
// from the per-point index table (B+ indices, the node itself where a
// neighbour is missing).  Ruuth-Merriman modes drop ghost neighbours.
template <typename T, int DIM, int MODE>
__global__ void __launch_bounds__(256) k_lap_idx(LevelView<T> L, const T* u, const T* __restrict__ w,
                                                 const T* __restrict__ f, const T* __restrict__ cvec,
                                                 T cval, const T* __restrict__ dA, T omega, T* out,
                                                 T* u_inout, double* part, const T* __restrict__ refv,
                                                 const int32_t* __restrict__ list, int32_t nlist) {
  constexpr bool RM = MODE == LAP_RM_JAC || MODE == LAP_RM_RES || MODE == LAP_BAND || MODE == LAP_VARD;
  int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  release_next();
  double rm = 0.0, rs = 0.0;
  bool active = i < (list ? nlist : L.nB);
  if (list && active) i = __ldg(list + i);
  if (active && (MODE == LAP_JAC_RED || MODE == LAP_JAC_BLACK)) {
    const uint64_t kk = __ldg(L.key + i);
    active = ((key_x(kk) + key_y(kk) + (DIM == 3 ? key_z(kk) : 0)) & 1) == (MODE == LAP_JAC_BLACK ? 1 : 0);
  }
  if (active) {
    int32_t k[6];
#pragma unroll
    for (int q = 0; q < 2 * DIM; ++q) k[q] = __ldg(L.nbr + (int64_t)q * L.nB + i);
    wait_prior();
    const T ui = ld_prior(u + i);
    if (MODE == LAP_VARD) {  // out = L~ u, refv = the diffusion coefficient a
      const T ai = ld_prior(refv + i);
      T s = T(0);
#pragma unroll
      for (int q = 0; q < 2 * DIM; ++q)
        if (k[q] < L.nB && k[q] != i) s += (T(0.5) * (ai + ld_prior(refv + k[q]))) * (ld_prior(u + k[q]) - ui);
      out[i] = s * L.inv_h2;
    } else if (RM) {
      T s = T(0);
#pragma unroll
      for (int q = 0; q < 2 * DIM; ++q)
        if (k[q] < L.nB && k[q] != i) s += ld_prior(u + k[q]);
      if (MODE == LAP_BAND) {
        out[i] = s * L.inv_h2 - L.gamma * ui;
      } else {
        const T c = cvec ? __ldg(cvec + i) : cval;
        const T diag = c + L.gamma;
        const T r = ld_prior(f + i) - diag * ui + s * L.inv_h2;
        out[i] = MODE == LAP_RM_JAC ? ui + omega * r / diag : r;
      }
    } else {
      const T wi = ld_prior(w + i);
      T s = T(0), Mu;
      if (MODE == LAP_RESID_REL || MODE == LAP_JAC_REL) {
        const T ri = ld_prior(refv + i);
#pragma unroll
        for (int q = 0; q < 2 * DIM; ++q) s += (ld_prior(refv + k[q]) - ri) + (ld_prior(w + k[q]) - wi);
        Mu = s * L.inv_h2 + L.gamma * ((ri - ui) + wi);
      } else {
#pragma unroll
        for (int q = 0; q < 2 * DIM; ++q) s += ld_prior(w + k[q]) - wi;
        Mu = s * L.inv_h2 + L.gamma * (wi - ui);
      }
      if (MODE == LAP_APPLY) {
        out[i] = Mu;
      } else {
        const T c = cvec ? __ldg(cvec + i) : cval;
        const T r = ld_prior(f + i) - c * ui + Mu;
        if (MODE == LAP_RESID || MODE == LAP_RESID_REL) {
          out[i] = r;
          rm = fabs((double)r);
          rs = (double)r * (double)r;
        } else {
          u_inout[i] = ui + r * __ldg(dA + i);
        }
      }
    }
  }
  if ((MODE == LAP_RESID || MODE == LAP_RESID_REL) && part) block_max_sum(rm, rs, part);
}

template <int DIM, int MODE, typename T>
static void lap_dispatch(const LevelView<T>& L, const T* u, const T* w, const T* f, const T* cvec,
                         T cval, const T* dA, T omega, T* out, T* u_inout, double* part,
                         const T* refv, cudaStream_t st) {
  launch_pdl(k_lap_idx<T, DIM, MODE>, lap_grid(L), 256, st, L, u, w, f, cvec, cval, dA, omega, out, u_inout, part,
             refv, (const int32_t*)nullptr, 0);
  count_launch();
}

template <int MODE, typename T>
static void lap_dim(const LevelView<T>& L, const T* u, const T* w, const T* f, const T* cvec, T cval,
                    const T* dA, T omega, T* out, T* u_inout, double* part, const T* refv,
                    cudaStream_t st) {
  if (L.nB <= 0) return;
  if (L.dim == 3)
    lap_dispatch<3, MODE>(L, u, w, f, cvec, cval, dA, omega, out, u_inout, part, refv, st);
  else
    lap_dispatch<2, MODE>(L, u, w, f, cvec, cval, dA, omega, out, u_inout, part, refv, st);
}

void launch_lap(const LevelView<double>& L, LapMode mode, const double* u, const double* w,
                const double* f, const double* cvec, double cval, const double* dA, double omega,
                double* out, double* u_inout, double* part, int nblocks_part, cudaStream_t st) {
  using T = double;
  (void)nblocks_part;
  if (mode == LAP_APPLY) lap_dim<LAP_APPLY>(L, u, w, f, cvec, cval, dA, omega, out, u_inout, part, (const T*)nullptr, st);
  if (mode == LAP_RESID) lap_dim<LAP_RESID>(L, u, w, f, cvec, cval, dA, omega, out, u_inout, part, (const T*)nullptr, st);
  if (mode == LAP_JACOBI) lap_dim<LAP_JACOBI>(L, u, w, f, cvec, cval, dA, omega, out, u_inout, part, (const T*)nullptr, st);
  if (mode == LAP_JAC_RED) lap_dim<LAP_JAC_RED>(L, u, w, f, cvec, cval, dA, omega, out, u_inout, part, (const T*)nullptr, st);
  if (mode == LAP_JAC_BLACK) lap_dim<LAP_JAC_BLACK>(L, u, w, f, cvec, cval, dA, omega, out, u_inout, part, (const T*)nullptr, st);
}

template <int MODE>
static void lap_set(const LevelView<double>& L, const PointSet& S, const double* u, const double* w,
                    const double* f, const double* cvec, double cval, const double* dA, double* out,
                    double* u_inout, cudaStream_t st) {
  if (S.n <= 0) return;
  auto kernel = L.dim == 3 ? k_lap_idx<double, 3, MODE> : k_lap_idx<double, 2, MODE>;
  launch_pdl(kernel, nblk(S.n, 256), 256, st, L, u, w, f, cvec, cval, dA, 0.0, out, u_inout, (double*)nullptr,
             (const double*)nullptr, S.list, S.n);
  count_launch();
}
void launch_lap_set(const LevelView<double>& L, LapMode mode, const PointSet& S, const double* u, const double* w,
                    const double* f, const double* cvec, double cval, const double* dA, double* out,
                    double* u_inout, cudaStream_t st) {
  if (mode == LAP_RESID) lap_set<LAP_RESID>(L, S, u, w, f, cvec, cval, dA, out, u_inout, st);
  else lap_set<LAP_JACOBI>(L, S, u, w, f, cvec, cval, dA, out, u_inout, st);
}

__global__ void __launch_bounds__(256) k_jacobi_zero64(const double* __restrict__ f, const double* __restrict__ dA,
                                                       const int32_t* __restrict__ list, int32_t n, double* u) {
  int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  release_next();
  if (i >= n) return;
  if (list) i = __ldg(list + i);
  const double d = __ldg(dA + i);
  wait_prior();
  u[i] = ld_prior(f + i) * d;
}
void launch_jacobi_zero(const LevelView<double>& L, const PointSet* S, const double* f, const double* dA, double* u,
                        cudaStream_t st) {
  const int32_t n = S ? S->n : L.nB;
  if (n <= 0) return;
  launch_pdl(k_jacobi_zero64, nblk(n, 256), 256, st, f, dA, S ? S->list : (const int32_t*)nullptr, n, u);
  count_launch();
}

template <typename T>
void launch_lap_rel(const LevelView<T>& L, LapMode mode, const T* u, const T* delta, const T* refv,
                    const T* f, const T* cvec, T cval, const T* dA, T* out, T* u_inout, double* part,
                    cudaStream_t st) {
  if (mode == LAP_RESID_REL)
    lap_dim<LAP_RESID_REL>(L, u, delta, f, cvec, cval, dA, T(0), out, u_inout, part, refv, st);
  else
    lap_dim<LAP_JAC_REL>(L, u, delta, f, cvec, cval, dA, T(0), out, u_inout, part, refv, st);
}

void launch_resid_rel(const LevelView<double>& L, const double* u, const double* delta,
                      const double* refv, const double* f, const double* cvec, double cval,
                      double* r, double* part, cudaStream_t st) {
  lap_dim<LAP_RESID_REL>(L, u, delta, f, cvec, cval, (const double*)nullptr, 0.0, r, (double*)nullptr,
                         part, refv, st);
}

// ---------------------------------------------------- outer residual, FP32 pairs
// r = f - c u + M u on B from the pair extension (delta_j pairs, ref_j floats):
// M u_i = S / dx^2 + gamma ((ref_i - u_i) + delta_i) with
// S = sum over the 2d neighbours k of (ref_k - ref_i) + (delta_k - delta_i),
// summed in pairs (the reference differences are exact TwoSums of floats),
// scaled by 1/dx^2 and gamma as pairs.  FP64 work per point: ref_i - u_i,
// f - c u_i and the sum with M u_i, and r^2 for the norm (the maximum is taken
// on the bit patterns of |r|).  Each thread takes kPairPts points (strided by
// the block), so the block's norm reduction is shared by several points.
constexpr int kPairPts = 2;
// Fewer points than fill the chip that way take one point per thread (circle,
// 2912 points: 7.7 us with four in a row, 140 us at 8.5 M points with two, 147 with four).
constexpr int64_t kPairSmall = 152 * 1024;

// Largest |x| and sum of x^2 over the block into part[2 b], part[2 b + 1];
// m holds the bit pattern of a non-negative double (ordered as an integer).
__device__ inline void block_maxbits_sum(unsigned long long m, double s, double* part) {
  __shared__ unsigned long long sm[32];
  __shared__ double ss[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) { sm[wid] = m; ss[wid] = s; }
  __syncthreads();
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    m = lane < nw ? sm[lane] : 0ull;
    s = lane < nw ? ss[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    if (lane == 0) {
      part[2 * blockIdx.x] = __longlong_as_double((long long)m);
      part[2 * blockIdx.x + 1] = s;
    }
  }
}

template <int DIM, int PTS>
__global__ void __launch_bounds__(256) k_resid_pair(LevelView<double> L, const double* __restrict__ u,
                                                    const float2* __restrict__ dp,
                                                    const float* __restrict__ rp,
                                                    const double* __restrict__ f,
                                                    const double* __restrict__ cvec, double cval,
                                                    float2 ih2, float2 gam, double* __restrict__ r,
                                                    double* part) {
  unsigned long long rm = 0ull;
  double rs = 0.0;
  release_next();
  wait_prior();
#pragma unroll
  for (int j = 0; j < PTS; ++j) {
    const int32_t i = (blockIdx.x * PTS + j) * blockDim.x + threadIdx.x;
    if (i >= L.nB) continue;  // (not break: the points' loads can then overlap)
    int32_t k[2 * DIM];
#pragma unroll
    for (int q = 0; q < 2 * DIM; ++q) k[q] = __ldg(L.nbr + (int64_t)q * L.nB + i);
    const float ri = ld_prior(rp + i);
    const float2 di = ld_prior(dp + i);
    const double ui = ld_prior(u + i), fi = ld_prior(f + i);
    float rn[2 * DIM];
    float2 dn[2 * DIM];
#pragma unroll
    for (int q = 0; q < 2 * DIM; ++q) {
      rn[q] = ld_prior(rp + k[q]);
      dn[q] = ld_prior(dp + k[q]);
    }
    float sh = 0.f, sl = 0.f;
#pragma unroll
    for (int q = 0; q < 2 * DIM; ++q) {
      const float rk = rn[q];
      const float2 dk = dn[q];
      float ah, al, bh, bl, ch, cl, t;
      two_sum(rk, -ri, ah, al);
      two_sum(dk.x, -di.x, bh, bl);
      two_sum(ah, bh, ch, cl);
      two_sum(sh, ch, sh, t);
      sl = __fadd_rn(sl, __fadd_rn(__fadd_rn(al, bl), __fadd_rn(cl, t)));
      sl = __fadd_rn(sl, __fsub_rn(dk.y, di.y));
    }
    float Sh, Sl, lh, ll;
    fast_two_sum(sh, sl, Sh, Sl);
    pair_mul(Sh, Sl, ih2.x, ih2.y, lh, ll);             // S / dx^2
    const float2 e = pair_split(pair_f2d(ri) - ui);      // ref_i - u_i
    float th, tl, gh, gl, mh, ml;
    pair_add(e.x, e.y, di.x, di.y, th, tl);
    pair_mul(th, tl, gam.x, gam.y, gh, gl);             // gamma ((ref_i - u_i) + delta_i)
    pair_add(lh, ll, gh, gl, mh, ml);                   // M u_i
    const double c = cvec ? __ldg(cvec + i) : cval;
    const double res = (fi - c * ui) + pair_to_f64(mh, ml);
    r[i] = res;
    rm = max(rm, (unsigned long long)__double_as_longlong(res) & 0x7FFFFFFFFFFFFFFFull);  // |res|
    if (part) rs += res * res;
  }
  if (part) block_maxbits_sum(rm, rs, part);
}

int resid_pair_blocks(const LevelView<double>& L) {
  const int pts = L.nB < kPairSmall ? 1 : kPairPts;
  return (int)((L.nB + 256 * pts - 1) / (256 * pts));
}

void launch_resid_pair(const LevelView<double>& L, const double* u, const float2* delta,
                       const float* refv, const double* f, const double* cvec, double cval, double* r,
                       double* part, cudaStream_t st) {
  if (L.nB <= 0) return;
  const unsigned nb = (unsigned)resid_pair_blocks(L);
  const double ih2 = (double)L.inv_h2, gam = (double)L.gamma;
  const float ih2h = (float)ih2, gamh = (float)gam;
  const float2 ih2p = make_float2(ih2h, (float)(ih2 - (double)ih2h));
  const float2 gamp = make_float2(gamh, (float)(gam - (double)gamh));
  const bool small = L.nB < kPairSmall;
  auto kernel = L.dim == 3 ? (small ? k_resid_pair<3, 1> : k_resid_pair<3, kPairPts>)
                           : (small ? k_resid_pair<2, 1> : k_resid_pair<2, kPairPts>);
  launch_pdl(kernel, nb, 256, st, L, u, delta, refv, f, cvec, cval, ih2p, gamp, r, part);
  count_launch();
}

// ------------------------------------------------- pointwise FP64 residual check
// After an outer residual in FP32 pairs that meets the tolerance only within
// its error estimate, only the band points whose |r_i| exceeds thr = (tol -
// estimate) max|f| can violate the tolerance.  k_check_select lists them (at
// most cap; *count may exceed cap, the list is then incomplete) and
// k_check_points evaluates r_i there in FP64, in the relative form with the
// point's own value as the common reference: delta_j = sum_m E_jm (u_m - u_i)
// for j = i and its 2d neighbours (cubic weights from the fractions, stencil
// nodes through the brick tables), M u_i = sum_q (delta_kq - delta_i) / dx^2 +
// gamma delta_i, r_i = f_i - c_i u_i + M u_i; the maximum |r_i| goes to *maxbits
// (bit pattern of a non-negative double).  The stencil rows of one point are
// summed with shared-memory atomics, so the last bits of r_i may vary from
// run to run.
__global__ void k_check_select(const double* __restrict__ r, int32_t nB, unsigned long long thr_bits,
                               int32_t* __restrict__ list, int32_t cap, int32_t* count) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nB) return;
  const unsigned long long a = (unsigned long long)__double_as_longlong(r[i]) & 0x7FFFFFFFFFFFFFFFull;
  if (a > thr_bits) {
    const int32_t p = atomicAdd(count, 1);
    if (p < cap) list[p] = i;
  }
}

// One warp per candidate point i: the 2d + 1 extension values it needs (at i
// and at its Laplacian neighbours) are split into 4-node rows of their cubic
// stencils, spread over the lanes, and summed per value in shared memory.
constexpr int kCheckWarps = 4;

template <int DIM>
__global__ void __launch_bounds__(kCheckWarps * 32) k_check_points(
    LevelView<double> L, const double* __restrict__ u, const double* __restrict__ f,
    const double* __restrict__ cvec, double cval, const int32_t* __restrict__ list,
    const int32_t* count, int32_t cap, unsigned long long* maxbits) {
  constexpr int R = DIM == 3 ? 16 : 4;  // stencil rows of 4 nodes per value
  constexpr int NJ = 2 * DIM + 1;       // values: the point, then its neighbours
  __shared__ double part[kCheckWarps][NJ];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t n = min(*count, cap);
  for (int32_t t = blockIdx.x * kCheckWarps + warp; t < n; t += gridDim.x * kCheckWarps) {
    const int32_t i = list[t];
    const double ui = u[i];
    if (lane < NJ) part[warp][lane] = 0.0;
    __syncwarp();
    for (int e = lane; e < NJ * R; e += 32) {
      const int jj = e / R, row = e % R;
      const int32_t j = jj == 0 ? i : __ldg(L.nbr + (int64_t)(jj - 1) * L.nB + i);
      const uint64_t kk = __ldg(L.key + j);
      const int bx = key_x(kk) + key_ox(kk), by = key_y(kk) + key_oy(kk);
      const int bz = DIM == 3 ? key_z(kk) + key_oz(kk) : 0;
      const int b = row & 3, c = row >> 2;
      double w[3][4];  // cubic Lagrange weights at nodes -1, 0, 1, 2 per axis
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        const double sf = __ldg(L.fr + a * L.nplus + j);
        const double sm1 = sf - 1.0, sm2 = sf - 2.0, sp1 = sf + 1.0;
        const double p = sf * sm1, q = sp1 * sm2;
        w[a][0] = -(p * sm2) * (1.0 / 6.0);
        w[a][1] = (q * sm1) * 0.5;
        w[a][2] = -(q * sf) * 0.5;
        w[a][3] = (p * sp1) * (1.0 / 6.0);
      }
      double acc = 0.0;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const int32_t m = band_index(L.bv, bx + a, by + b, bz + c);
        acc += w[0][a] * ((m >= 0 ? __ldg(u + m) : ui) - ui);
      }
      atomicAdd(&part[warp][jj], w[1][b] * (DIM == 3 ? w[2][c] : 1.0) * acc);
    }
    __syncwarp();
    if (lane == 0) {
      const double di = part[warp][0];
      double s = 0.0;
      for (int q = 1; q < NJ; ++q) s += part[warp][q] - di;
      const double c = cvec ? cvec[i] : cval;
      const double r = f[i] - c * ui + (s * L.inv_h2 + L.gamma * di);
      atomicMax(maxbits, (unsigned long long)__double_as_longlong(r) & 0x7FFFFFFFFFFFFFFFull);
    }
    __syncwarp();
  }
}

void launch_pointwise_check(const LevelView<double>& L, const double* u, const double* f,
                            const double* cvec, double cval, const double* r, double thr,
                            int32_t* list, int32_t cap, int32_t* count, unsigned long long* maxbits,
                            cudaStream_t st) {
  CPM_CUDA_TRY(cudaMemsetAsync(count, 0, sizeof(int32_t), st));
  CPM_CUDA_TRY(cudaMemsetAsync(maxbits, 0, sizeof(unsigned long long), st));
  if (L.nB <= 0) return;
  unsigned long long thr_bits = 0ull;
  if (thr > 0.0) std::memcpy(&thr_bits, &thr, sizeof(thr));
  k_check_select<<<nblk(L.nB, 256), 256, 0, st>>>(r, L.nB, thr_bits, list, cap, count);
  const unsigned grid = 2 * 152;  // warps loop over the candidates
  if (L.dim == 3)
    k_check_points<3><<<grid, kCheckWarps * 32, 0, st>>>(L, u, f, cvec, cval, list, count, cap, maxbits);
  else
    k_check_points<2><<<grid, kCheckWarps * 32, 0, st>>>(L, u, f, cvec, cval, list, count, cap, maxbits);
  count_launch(2);
}

// ----------------------------------------------------------------- Ruuth-Merriman
template <typename T>
void launch_rm_jacobi(const LevelView<T>& L, const T* u, const T* f, const T* cvec, T cval, T omega,
                      T* out, cudaStream_t st) {
  lap_dim<LAP_RM_JAC>(L, u, (const T*)nullptr, f, cvec, cval, (const T*)nullptr, omega, out,
                      (T*)nullptr, nullptr, (const T*)nullptr, st);
}
template <typename T>
void launch_rm_resid(const LevelView<T>& L, const T* u, const T* f, const T* cvec, T cval, T* out,
                     cudaStream_t st) {
  lap_dim<LAP_RM_RES>(L, u, (const T*)nullptr, f, cvec, cval, (const T*)nullptr, T(0), out,
                      (T*)nullptr, nullptr, (const T*)nullptr, st);
}

// ----------------------------------------------------------------- paper form
// The paper's own scheme (Sec. 3.1, Eq. 3.3): M u = E_1 (L_B u) - gamma (u - E_3 u)
// on B, with L_B the band-restricted 2d+1-point Laplacian, E_1 linear and
// E_3 cubic interpolation at cp.  Given v = L_B u (launch_lap_band) and
// w = E_3 u on B (launch_extend over B), one thread per band point gathers v
// at the 2^d linear-stencil nodes of cp(x_i) (the middle nodes of its cubic
// stencil, same fractions) through the brick tables.
template <typename T>
void launch_lap_band(const LevelView<T>& L, const T* u, T* v, cudaStream_t st) {
  lap_dim<LAP_BAND>(L, u, (const T*)nullptr, (const T*)nullptr, (const T*)nullptr, T(0),
                    (const T*)nullptr, T(0), v, (T*)nullptr, nullptr, (const T*)nullptr, st);
}

template <typename T>
void launch_lap_vard(const LevelView<T>& L, const T* u, const T* a, T* v, cudaStream_t st) {
  lap_dim<LAP_VARD>(L, u, (const T*)nullptr, (const T*)nullptr, (const T*)nullptr, T(0),
                    (const T*)nullptr, T(0), v, (T*)nullptr, nullptr, a, st);
}

template <typename T, int DIM, int MODE>
__global__ void __launch_bounds__(256) k_paper(LevelView<T> L, const T* u, const T* __restrict__ v,
                                               const T* __restrict__ w, const T* __restrict__ f,
                                               const T* __restrict__ cvec, T cval,
                                               const T* __restrict__ dA, T* out, T* u_inout,
                                               double* part, const T* __restrict__ avec) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  double rm = 0.0, rs = 0.0;
  const uint64_t k = i < L.nB ? __ldg(L.key + i) : 0ull;
  const bool skip = (MODE == LAP_JAC_RED || MODE == LAP_JAC_BLACK) &&
                    ((key_x(k) + key_y(k) + (DIM == 3 ? key_z(k) : 0)) & 1) != (MODE == LAP_JAC_BLACK ? 1 : 0);
  if (i < L.nB && !skip) {
    const int bx = key_x(k) + key_ox(k) + 1, by = key_y(k) + key_oy(k) + 1;
    const int bz = DIM == 3 ? key_z(k) + key_oz(k) + 1 : 0;
    const T sx = __ldg(L.fr + i), sy = __ldg(L.fr + L.nplus + i);
    const T sz = DIM == 3 ? __ldg(L.fr + 2 * L.nplus + i) : T(0);
    const T wx[2] = {T(1) - sx, sx}, wy[2] = {T(1) - sy, sy}, wz[2] = {T(1) - sz, sz};
    T e1v = T(0);
#pragma unroll
    for (int c = 0; c < (DIM == 3 ? 2 : 1); ++c) {
      T accy = T(0);
#pragma unroll
      for (int bb = 0; bb < 2; ++bb) {
        const int32_t j0 = band_index(L.bv, bx, by + bb, bz + c);
        const int32_t j1 = band_index(L.bv, bx + 1, by + bb, bz + c);
        accy += wy[bb] * (wx[0] * v[j0 < 0 ? i : j0] + wx[1] * v[j1 < 0 ? i : j1]);
      }
      e1v += (DIM == 3 ? wz[c] : T(1)) * accy;
    }
    const T ui = u[i];
    const T g = avec ? L.gamma * avec[i] : L.gamma;  // side-condition weight gamma a_i
    const T Mu = e1v - g * (ui - w[i]);
    if (MODE == LAP_APPLY) {
      out[i] = Mu;
    } else {
      const T cc = cvec ? cvec[i] : cval;
      const T r = f[i] - cc * ui + Mu;
      if (MODE == LAP_RESID) {
        out[i] = r;
        rm = fabs((double)r);
        rs = (double)r * (double)r;
      } else {
        u_inout[i] = ui + r * dA[i];
      }
    }
  }
  if (MODE == LAP_RESID && part) block_max_sum(rm, rs, part);
}

// The same operator in one pass over the extension tiles: E_1 L_B u at cp(x_i)
// needs L_B u at the 2^d middle nodes of the cubic stencil, whose Laplacian
// neighbours all lie in the stencil and so in B.  With linear weights l over
// the middle nodes and their second differences e (weights l_0, l_1 - 2 l_0,
// l_0 - 2 l_1, l_1 over the four nodes of an axis), E_1 L_B u is the sum over
// the axes of the products with e on that axis and l on the others, so each
// stencil row is contracted with the cubic weights, with l and with e.  In 3-D
// the sums are ordered for their rounding: the cubic part axis by axis, the
// small terms of the outer planes and rows before the large ones.  FP32 M u on
// spheres and tori has 0.94 to 0.98 of the rms error of the three passes (1.12
// to 1.14 with one sum over the products of two weights).  Taken for FP32, and
// in 2-D: in 3-D FP64 the extra products cost more FP64 time than the two passes
// they save.  u and out must not overlap.  M u on a circle of 29 thousand
// points, FP64: one launch of 8.7 us against three of 10.5 us (a call 16.6
// against 23.6 us); on the unit sphere at dx = 1/256, FP32: 197 us against
// 268 us.
template <typename T, int DIM, int MODE>
__global__ void __launch_bounds__(64) k_paper_tiles(LevelView<T> L, const T* __restrict__ u,
                                                    const T* __restrict__ f, const T* __restrict__ cvec, T cval,
                                                    const T* __restrict__ dA, T* __restrict__ out) {
  constexpr int NZ = DIM == 3 ? 7 : 1, RS = 9;
  __shared__ T box[NZ * 7 * RS];
  const int32_t tile = blockIdx.x;
  release_next();
  const int32_t beg = __ldg(L.tile_start + tile), end = __ldg(L.tile_mid + tile);
  if (beg == end) return;  // ghost points only
  // this thread's first point: its records are in flight while the box is staged
  uint32_t rec = 0;
  T s[3] = {T(0), T(0), T(0)}, w3[3][4];
  auto load = [&](int32_t k) {
    rec = __ldg(L.erec + k);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      if constexpr (sizeof(T) == 8) {
#pragma unroll
        for (int j = 0; j < 4; ++j) w3[a][j] = __ldg(L.ew64 + (int64_t)(4 * a + j) * L.nplus + k);
        s[a] = __ldg(L.fr + (int64_t)a * L.nplus + (rec >> 6));
      } else {
        s[a] = __ldg(L.efr + (int64_t)a * L.nplus + k);
        cubic_w(s[a], w3[a]);
      }
    }
  };
  int32_t k = beg + threadIdx.x;
  if (k < end) load(k);
  wait_prior();
  for (int q = threadIdx.x; q < NZ * 49; q += 64) {
    const int x = q % 7, y = (q / 7) % 7, z = q / 49;
    const int j = (x >> 2) | ((y >> 2) << 1) | ((z >> 2) << 2);
    const uint64_t bit = 1ull << ((x & 3) | ((y & 3) << 2) | ((z & 3) << 4));
    const uint64_t m = __ldg(L.tile_mask + 8 * (int64_t)tile + j);
    T v = T(0);
    if (m & bit) v = ld_prior(u + __ldg(L.tile_bstart + 8 * (int64_t)tile + j) + __popcll(m & (bit - 1ull)));
    box[(z * 7 + y) * RS + x] = v;
  }
  __syncthreads();
  for (; k < end; k += 64) {
    const int32_t i = (int32_t)(rec >> 6);
    const int bx = rec & 3, by = (rec >> 2) & 3, bz = (rec >> 4) & 3;
    T l[3][4], e[3][4];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      const T l0 = T(1) - s[a], l1 = s[a];
      l[a][0] = T(0);
      l[a][1] = l0;
      l[a][2] = l1;
      l[a][3] = T(0);
      e[a][0] = l0;
      e[a][1] = l1 - T(2) * l0;
      e[a][2] = l0 - T(2) * l1;
      e[a][3] = l1;
    }
    T e3 = T(0), e1l = T(0);
    if constexpr (DIM == 2) {
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const T* row = box + (by + b) * RS + bx;
        T v[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) v[a] = row[a];
        const T x3 = w3[0][0] * v[0] + w3[0][1] * v[1] + w3[0][2] * v[2] + w3[0][3] * v[3];
        e3 += w3[1][b] * x3;
        const T xl = l[0][1] * v[1] + l[0][2] * v[2];
        e1l += e[1][b] * xl;
        if (b == 1 || b == 2) {
          const T xe = e[0][0] * v[0] + e[0][1] * v[1] + e[0][2] * v[2] + e[0][3] * v[3];
          e1l += l[1][b] * xe;
        }
      }
    } else {  // FP32
      float2 q01, q23;  // contracted in y and z, by x
      float mid[2];     // the middle planes' sums over x and y
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        const int c = cc == 0 ? 0 : cc == 1 ? 3 : cc - 1;  // the outer planes first
        const bool mz = c == 1 || c == 2;
        float2 p01, p23;
        float xl[4], xe[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const float* row = box + ((bz + c) * 7 + by + b) * RS + bx;
          float v[4];
#pragma unroll
          for (int a = 0; a < 4; ++a) v[a] = row[a];
          const float2 wy = make_float2(w3[1][b], w3[1][b]), v01 = make_float2(v[0], v[1]), v23 = make_float2(v[2], v[3]);
          p01 = b == 0 ? __fmul2_rn(wy, v01) : __ffma2_rn(wy, v01, p01);
          p23 = b == 0 ? __fmul2_rn(wy, v23) : __ffma2_rn(wy, v23, p23);
          const bool my = b == 1 || b == 2;
          if (my || mz) xl[b] = l[0][1] * v[1] + l[0][2] * v[2];
          if (my && mz) xe[b] = e[0][0] * v[0] + e[0][1] * v[1] + e[0][2] * v[2] + e[0][3] * v[3];
        }
        const float2 wz = make_float2(w3[2][c], w3[2][c]);
        q01 = cc == 0 ? __fmul2_rn(wz, p01) : __ffma2_rn(wz, p01, q01);
        q23 = cc == 0 ? __fmul2_rn(wz, p23) : __ffma2_rn(wz, p23, q23);
        e1l += e[2][c] * (l[1][1] * xl[1] + l[1][2] * xl[2]);
        if (mz) {
          float m = e[1][0] * xl[0] + e[1][3] * xl[3];
          m += e[1][1] * xl[1];
          m += e[1][2] * xl[2];
          m += l[1][1] * xe[1];
          m += l[1][2] * xe[2];
          mid[c - 1] = m;
        }
      }
      e1l += l[2][1] * mid[0];
      e1l += l[2][2] * mid[1];
      e3 = (w3[0][0] * q01.x + w3[0][2] * q23.x) + (w3[0][1] * q01.y + w3[0][3] * q23.y);
    }
    const T ui = ld_prior(u + i);
    const T Mu = e1l * L.inv_h2 - L.gamma * (ui - e3);
    if (MODE == LAP_APPLY) {
      out[i] = Mu;
    } else {
      const T cc = cvec ? __ldg(cvec + i) : cval;
      const T r = ld_prior(f + i) - cc * ui + Mu;
      out[i] = MODE == LAP_RESID ? r : ui + r * __ldg(dA + i);
    }
    if (k + 64 < end) load(k + 64);
  }
}

template <typename T>
bool paper_fused(const LevelView<T>& L) {
  return sizeof(T) == 4 || L.dim == 2;
}
template <typename T>
void launch_paper_fused(const LevelView<T>& L, LapMode mode, const T* u, const T* f, const T* cvec, T cval,
                        const T* dA, T* out, cudaStream_t st) {
  if (L.ntiles <= 0) return;
  if (L.dim == 3) {
    if constexpr (sizeof(T) == 4) {
      auto k = mode == LAP_APPLY ? k_paper_tiles<T, 3, LAP_APPLY>
               : mode == LAP_RESID ? k_paper_tiles<T, 3, LAP_RESID> : k_paper_tiles<T, 3, LAP_JACOBI>;
      launch_pdl(k, L.ntiles, 64, st, L, u, f, cvec, cval, dA, out);
    }
  } else {
    auto k = mode == LAP_APPLY ? k_paper_tiles<T, 2, LAP_APPLY>
             : mode == LAP_RESID ? k_paper_tiles<T, 2, LAP_RESID> : k_paper_tiles<T, 2, LAP_JACOBI>;
    launch_pdl(k, L.ntiles, 64, st, L, u, f, cvec, cval, dA, out);
  }
  count_launch();
}

int paper_blocks(const LevelView<double>& L) { return (int)nblk(L.nB, 256); }

template <typename T>
void launch_paper(const LevelView<T>& L, LapMode mode, const T* u, const T* v, const T* w, const T* f,
                  const T* cvec, T cval, const T* dA, T* out, T* u_inout, double* part,
                  const T* avec, cudaStream_t st) {
  if (L.nB <= 0) return;
  const unsigned g = nblk(L.nB, 256);
#define CPM_PAPER(DIM, MODE) \
  k_paper<T, DIM, MODE><<<g, 256, 0, st>>>(L, u, v, w, f, cvec, cval, dA, out, u_inout, part, avec)
  if (L.dim == 3) {
    if (mode == LAP_APPLY) CPM_PAPER(3, LAP_APPLY);
    else if (mode == LAP_RESID) CPM_PAPER(3, LAP_RESID);
    else if (mode == LAP_JAC_RED) CPM_PAPER(3, LAP_JAC_RED);
    else if (mode == LAP_JAC_BLACK) CPM_PAPER(3, LAP_JAC_BLACK);
    else CPM_PAPER(3, LAP_JACOBI);
  } else {
    if (mode == LAP_APPLY) CPM_PAPER(2, LAP_APPLY);
    else if (mode == LAP_RESID) CPM_PAPER(2, LAP_RESID);
    else if (mode == LAP_JAC_RED) CPM_PAPER(2, LAP_JAC_RED);
    else if (mode == LAP_JAC_BLACK) CPM_PAPER(2, LAP_JAC_BLACK);
    else CPM_PAPER(2, LAP_JACOBI);
  }
#undef CPM_PAPER
  count_launch();
}

// ----------------------------------------------------------------- transfers
// Closest-point restriction / prolongation (Sec. 4.3): linear interpolation
// at each target's cp from the 2^d source nodes around it.  The nodes are
// found from the packed base node through the source brick map and masks
// (cached loads shared by neighbouring targets), not from a per-target index
// table.
template <typename T, int DIM>
__global__ void __launch_bounds__(256) k_transfer(TransferView<T> tv, const T* __restrict__ src,
                                                  T* __restrict__ dst, bool add) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  release_next();
  if (j >= tv.n) return;
  const T sx = __ldg(tv.fr + j), sy = __ldg(tv.fr + tv.n + j);
  const T sz = DIM == 3 ? __ldg(tv.fr + 2 * tv.n + j) : T(0);
  const T wx[2] = {T(1) - sx, sx}, wy[2] = {T(1) - sy, sy}, wz[2] = {T(1) - sz, sz};
  int x = 0, y = 0, z = 0;
  if (!tv.idx) {
    const uint64_t kb = __ldg(tv.base + j);
    x = (int)(kb & 0xffffu);
    y = (int)((kb >> 16) & 0xffffu);
    z = (int)((kb >> 32) & 0xffffu);
  }
  wait_prior();
  T acc = T(0);
#pragma unroll
  for (int c = 0; c < (DIM == 3 ? 2 : 1); ++c) {
    T accy = T(0);
#pragma unroll
    for (int bb = 0; bb < 2; ++bb) {
      const int q = 4 * c + 2 * bb;
      const int32_t i0 = tv.idx ? __ldg(tv.idx + (int64_t)q * tv.n + j) : band_index(tv.src, x, y + bb, z + c);
      const int32_t i1 = tv.idx ? __ldg(tv.idx + (int64_t)(q + 1) * tv.n + j)
                                : band_index(tv.src, x + 1, y + bb, z + c);
      const T v0 = ld_prior(src + (i0 < 0 ? 0 : i0));
      const T v1 = ld_prior(src + (i1 < 0 ? 0 : i1));
      accy += wy[bb] * (wx[0] * v0 + wx[1] * v1);
    }
    acc += (DIM == 3 ? wz[c] : T(1)) * accy;
  }
  dst[j] = add ? ld_prior(dst + j) + acc : acc;
}

// Cubic restriction / prolongation: degree-3 interpolation at the target's cp
// from the 4^d source nodes around it (base = floor - 1), tensor-product
// Lagrange weights, contracted x, then y, then z.
template <typename T, int DIM>
__global__ void __launch_bounds__(256) k_transfer3(TransferView<T> tv, const T* __restrict__ src,
                                                   T* __restrict__ dst, bool add) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= tv.n) return;
  const uint64_t kb = __ldg(tv.base + j);
  const int x = (int)(kb & 0xffffu), y = (int)((kb >> 16) & 0xffffu), z = (int)((kb >> 32) & 0xffffu);
  T wx[4], wy[4], wz[4] = {T(1), T(0), T(0), T(0)};
  cubic_w(__ldg(tv.fr + j), wx);
  cubic_w(__ldg(tv.fr + tv.n + j), wy);
  if (DIM == 3) cubic_w(__ldg(tv.fr + 2 * tv.n + j), wz);
  T acc = T(0);
#pragma unroll
  for (int c = 0; c < (DIM == 3 ? 4 : 1); ++c) {
    T accy = T(0);
#pragma unroll
    for (int bb = 0; bb < 4; ++bb) {
      T accx = T(0);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const int32_t i = band_index(tv.src, x + a, y + bb, z + c);
        accx += wx[a] * __ldg(src + (i < 0 ? 0 : i));
      }
      accy += wy[bb] * accx;
    }
    acc += wz[c] * accy;
  }
  dst[j] = add ? dst[j] + acc : acc;
}

template <typename T>
void launch_transfer(const TransferView<T>& tv, const T* src, T* dst, bool add, cudaStream_t st) {
  if (tv.n <= 0) return;
  if (tv.deg == 3) {
    if (tv.dim == 3) k_transfer3<T, 3><<<nblk(tv.n, 256), 256, 0, st>>>(tv, src, dst, add);
    else k_transfer3<T, 2><<<nblk(tv.n, 256), 256, 0, st>>>(tv, src, dst, add);
  } else {
    if (tv.dim == 3) launch_pdl(k_transfer<T, 3>, nblk(tv.n, 256), 256, st, tv, src, dst, add);
    else launch_pdl(k_transfer<T, 2>, nblk(tv.n, 256), 256, st, tv, src, dst, add);
  }
  count_launch();
}

// ----------------------------------------------------------------- norms
template <typename T>
__global__ void k_norm_partials(const T* __restrict__ x, int64_t n, double* part) {
  double m = 0.0, s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double v = (double)x[i];
    m = fmax(m, fabs(v));
    s += v * v;
  }
  block_max_sum(m, s, part);
}

template <typename T>
void launch_norm_partials(const T* x, int64_t n, double* part, cudaStream_t st) {
  k_norm_partials<T><<<kNormBlocks, 256, 0, st>>>(x, n, part);
  count_launch();
}

// out[0] = max|x|, out[1] = sum x^2, out[2] = 1 / max|x| (0 if max is 0);
// out[3] = the largest of the kPairSlots float slots of dmax (non-negative,
// compared as integers), which are reset to 0, or 0 without dmax.
__global__ void __launch_bounds__(1024) k_norm_final(const double* part, int nblocks, double* out, uint32_t* dmax) {
  __shared__ double sm[32], ss[32];
  __shared__ uint32_t sd[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  release_next();
  wait_prior();
  uint32_t dm = 0u;
  if (dmax)
    for (int i = threadIdx.x; i < kPairSlots; i += blockDim.x) {
      dm = max(dm, dmax[i]);
      dmax[i] = 0u;
    }
  double m = 0.0, s = 0.0;
  for (int i = threadIdx.x; i < nblocks; i += blockDim.x) {
    m = fmax(m, ld_prior(part + 2 * i));
    s += ld_prior(part + 2 * i + 1);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  dm = __reduce_max_sync(0xffffffffu, dm);
  if (lane == 0) {
    sm[wid] = m;
    ss[wid] = s;
    sd[wid] = dm;
  }
  __syncthreads();
  if (wid == 0) {
    const bool on = lane < (int)(blockDim.x >> 5);
    m = on ? sm[lane] : 0.0;
    s = on ? ss[lane] : 0.0;
    dm = __reduce_max_sync(0xffffffffu, on ? sd[lane] : 0u);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
      s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    if (lane == 0) {
      out[0] = m;
      out[1] = s;
      out[2] = m > 0.0 ? 1.0 / m : 0.0;
      out[3] = (double)__uint_as_float(dm);
    }
  }
}

void launch_norm_final(const double* part, int nblocks, double* out, cudaStream_t st, uint32_t* dmax) {
  launch_pdl(k_norm_final, 1, 1024, st, part, nblocks, out, dmax);
  count_launch();
}

// ----------------------------------------------------------------- mixed precision
__global__ void k_scale_to_f32(const double* __restrict__ r, const double* __restrict__ norms,
                               float* __restrict__ r32, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r32[i] = (float)(r[i] * norms[2]);
}
void launch_scale_to_f32(const double* r, const double* norms, float* r32, int64_t n, cudaStream_t st) {
  k_scale_to_f32<<<nblk(n, 256), 256, 0, st>>>(r, norms, r32, n);
  count_launch();
}

__global__ void k_axpy_scaled(double* __restrict__ u, const float* __restrict__ d,
                              const double* __restrict__ norms, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) u[i] += norms[0] * (double)d[i];
}
void launch_axpy_scaled(double* u, const float* d, const double* norms, int64_t n, cudaStream_t st) {
  k_axpy_scaled<<<nblk(n, 256), 256, 0, st>>>(u, d, norms, n);
  count_launch();
}

__global__ void k_axpy64(double* __restrict__ u, const double* __restrict__ d, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  release_next();
  wait_prior();
  if (i < n) u[i] = ld_prior(u + i) + ld_prior(d + i);
}
void launch_axpy64(double* u, const double* d, int64_t n, cudaStream_t st) {
  launch_pdl(k_axpy64, nblk(n, 256), 256, st, u, d, n);
  count_launch();
}

template <typename T>
__global__ void k_cast_to_f64(const T* x, double* y, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = (double)x[i];
}
template <typename T>
__global__ void k_cast_from_f64(const double* x, T* y, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = (T)x[i];
}
template <typename T>
void launch_cast_to_f64(const T* x, double* y, int64_t n, cudaStream_t st) {
  k_cast_to_f64<T><<<nblk(n, 256), 256, 0, st>>>(x, y, n);
}
template <typename T>
void launch_cast_from_f64(const double* x, T* y, int64_t n, cudaStream_t st) {
  k_cast_from_f64<T><<<nblk(n, 256), 256, 0, st>>>(x, y, n);
}

// ----------------------------------------------------------------- coarse solve
// x_g = Ainv b_g with the FP64 inverse (chunked dense product, FP64 accumulation).
template <typename T>
void launch_coarse_gemv(const double* Ainv, const T* const* b, T* const* x, int G, int32_t n,
                        cudaStream_t st) {
  launch_dense_gemv<double, T, false>(Ainv, b, x, G, n, st);
  count_launch((G + kGemvMaxVectors - 1) / kGemvMaxVectors);
}

// ----------------------------------------------------------------- setup: diag(M)
// M_ii = -gamma + (1/dx^2) sum_{k in N(i)} E_{k,i}: the weight of node i in
// the cubic stencil of cp(x_k) for each Laplacian neighbour k of i.
template <int DIM>
__global__ void k_diag_M(LevelView<double> L, double* __restrict__ diagM) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= L.nB) return;
  const uint64_t ki = L.key[i];
  const int own[3] = {key_x(ki), key_y(ki), key_z(ki)};
  const int d[6][3] = {{-1, 0, 0}, {1, 0, 0}, {0, -1, 0}, {0, 1, 0}, {0, 0, -1}, {0, 0, 1}};
  double s = 0.0;
  for (int q = 0; q < 2 * DIM; ++q) {
    const int32_t kk = node_index(L.bv, own[0] + d[q][0], own[1] + d[q][1], own[2] + d[q][2]);
    if (kk < 0) continue;
    const uint64_t key = L.key[kk];
    const int base[3] = {key_x(key) + key_ox(key), key_y(key) + key_oy(key), key_z(key) + key_oz(key)};
    double wprod = 1.0;
    bool inside = true;
    for (int a = 0; a < DIM; ++a) {
      const int off = own[a] - base[a];
      if (off < 0 || off > 3) { inside = false; break; }
      double w[4];
      cubic_w(L.fr[a * L.nplus + kk], w);
      wprod *= w[off];
    }
    if (inside) s += wprod;
  }
  diagM[i] = -L.gamma + s * L.inv_h2;
}

void launch_diag_M(const LevelView<double>& L, double* diagM, cudaStream_t st) {
  if (L.dim == 3) k_diag_M<3><<<nblk(L.nB, 256), 256, 0, st>>>(L, diagM);
  else k_diag_M<2><<<nblk(L.nB, 256), 256, 0, st>>>(L, diagM);
}

// ----------------------------------------------------------------- setup: paper form
// diag(M_p)_ii = sum_j (E_1)_ij (L_B)_ji - gamma (1 - (E_3)_ii): over the 2^d
// linear-stencil nodes j of cp(x_i), (L_B)_ji is -2d/dx^2 for j = i and
// 1/dx^2 for a Laplacian neighbour j of i; (E_3)_ii is the cubic weight of
// node i in its own stencil (0 if it lies outside).
// Variable diffusion (a != null): (L~)_ji = (a_j + a_i) / (2 dx^2) for a
// Laplacian neighbour j of i in B, (L~)_ii = -sum over the neighbours k of i
// in B of (a_i + a_k) / (2 dx^2), and the side condition is weighted by
// gamma a_i.
__device__ __forceinline__ double vard_ii(const LevelView<double>& L, const double* a, int x, int y,
                                          int z, int dim, int32_t i) {
  const int d[6][3] = {{-1, 0, 0}, {1, 0, 0}, {0, -1, 0}, {0, 1, 0}, {0, 0, -1}, {0, 0, 1}};
  double s = 0.0;
  for (int q = 0; q < 2 * dim; ++q) {
    const int32_t k = band_index(L.bv, x + d[q][0], y + d[q][1], z + d[q][2]);
    if (k >= 0) s -= 0.5 * (a[i] + a[k]) * L.inv_h2;
  }
  return s;
}

template <int DIM>
__global__ void k_diag_Mp(LevelView<double> L, double* __restrict__ diagM, const double* __restrict__ acoef) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= L.nB) return;
  const uint64_t k = L.key[i];
  const int own[3] = {key_x(k), key_y(k), key_z(k)};
  const int b3[3] = {key_x(k) + key_ox(k), key_y(k) + key_oy(k), key_z(k) + key_oz(k)};
  double s[3], w3[3][4];
  for (int a = 0; a < DIM; ++a) {
    s[a] = L.fr[a * L.nplus + i];
    cubic_w(s[a], w3[a]);
  }
  double e1l = 0.0;
  for (int c = 0; c < (DIM == 3 ? 2 : 1); ++c)
    for (int b = 0; b < 2; ++b)
      for (int a = 0; a < 2; ++a) {
        const int j[3] = {b3[0] + 1 + a, b3[1] + 1 + b, DIM == 3 ? b3[2] + 1 + c : 0};
        const double w1 = (a ? s[0] : 1.0 - s[0]) * (b ? s[1] : 1.0 - s[1]) *
                          (DIM == 3 ? (c ? s[2] : 1.0 - s[2]) : 1.0);
        int dist = 0;
        for (int q = 0; q < DIM; ++q) dist += abs(j[q] - own[q]);
        if (!acoef) {
          if (dist == 0) e1l += w1 * (-L.gamma);
          else if (dist == 1) e1l += w1 * L.inv_h2;
        } else if (dist == 0) {
          e1l += w1 * vard_ii(L, acoef, own[0], own[1], own[2], DIM, i);
        } else if (dist == 1) {
          const int32_t jj = band_index(L.bv, j[0], j[1], j[2]);
          if (jj >= 0) e1l += w1 * 0.5 * (acoef[jj] + acoef[i]) * L.inv_h2;
        }
      }
  double e3 = 1.0;
  for (int q = 0; q < DIM; ++q) {
    const int off = own[q] - b3[q];
    e3 = (off < 0 || off > 3) ? 0.0 : e3 * w3[q][off];
  }
  diagM[i] = e1l - (acoef ? L.gamma * acoef[i] : L.gamma) * (1.0 - e3);
}

void launch_diag_Mp(const LevelView<double>& L, double* diagM, const double* a, cudaStream_t st) {
  if (L.dim == 3) k_diag_Mp<3><<<nblk(L.nB, 256), 256, 0, st>>>(L, diagM, a);
  else k_diag_Mp<2><<<nblk(L.nB, 256), 256, 0, st>>>(L, diagM, a);
}

// Row i of A_p = cI - M_p = (c + gamma) I - E_1 L_B - gamma E_3.  One thread per row.
template <int DIM, typename M>
__global__ void k_assemble_Ap(LevelView<double> L, const double* cvec, double cval, M* A,
                              const double* acoef) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const int32_t n = L.nB;
  if (i >= n) return;
  M* row = A + (size_t)i * n;
  const double gi = acoef ? L.gamma * acoef[i] : L.gamma;
  row[i] += (M)((cvec ? cvec[i] : cval) + gi);
  const uint64_t k = L.key[i];
  const int b3[3] = {key_x(k) + key_ox(k), key_y(k) + key_oy(k), key_z(k) + key_oz(k)};
  double s[3] = {0.0, 0.0, 0.0}, w3[3][4] = {{1.0, 0.0, 0.0, 0.0}, {1.0, 0.0, 0.0, 0.0}, {1.0, 0.0, 0.0, 0.0}};
  for (int a = 0; a < DIM; ++a) {
    s[a] = L.fr[a * L.nplus + i];
    cubic_w(s[a], w3[a]);
  }
  for (int c = 0; c < (DIM == 3 ? 4 : 1); ++c)
    for (int b = 0; b < 4; ++b)
      for (int a = 0; a < 4; ++a) {
        const int32_t j = band_index(L.bv, b3[0] + a, b3[1] + b, DIM == 3 ? b3[2] + c : 0);
        if (j >= 0) row[j] -= (M)(gi * w3[0][a] * w3[1][b] * w3[2][c]);
      }
  const int d[6][3] = {{-1, 0, 0}, {1, 0, 0}, {0, -1, 0}, {0, 1, 0}, {0, 0, -1}, {0, 0, 1}};
  for (int c = 0; c < (DIM == 3 ? 2 : 1); ++c)
    for (int b = 0; b < 2; ++b)
      for (int a = 0; a < 2; ++a) {
        const int jx = b3[0] + 1 + a, jy = b3[1] + 1 + b, jz = DIM == 3 ? b3[2] + 1 + c : 0;
        const double w1 = (a ? s[0] : 1.0 - s[0]) * (b ? s[1] : 1.0 - s[1]) *
                          (DIM == 3 ? (c ? s[2] : 1.0 - s[2]) : 1.0);
        const int32_t jj = band_index(L.bv, jx, jy, jz);
        if (!acoef) {
          if (jj >= 0) row[jj] -= (M)(w1 * -L.gamma);
          for (int q = 0; q < 2 * DIM; ++q) {
            const int32_t kk = band_index(L.bv, jx + d[q][0], jy + d[q][1], jz + d[q][2]);
            if (kk >= 0) row[kk] -= (M)(w1 * L.inv_h2);
          }
        } else if (jj >= 0) {  // row jj of L~ (its own band-restricted neighbours)
          for (int q = 0; q < 2 * DIM; ++q) {
            const int32_t kk = band_index(L.bv, jx + d[q][0], jy + d[q][1], jz + d[q][2]);
            if (kk < 0) continue;
            const double face = 0.5 * (acoef[jj] + acoef[kk]) * L.inv_h2;
            row[kk] -= (M)(w1 * face);
            row[jj] += (M)(w1 * face);
          }
        }
      }
}

template <typename M>
void launch_assemble_Ap(const LevelView<double>& L, const double* cvec, double cval, M* A,
                        const double* a, cudaStream_t st) {
  if (L.dim == 3) k_assemble_Ap<3, M><<<nblk(L.nB, 128), 128, 0, st>>>(L, cvec, cval, A, a);
  else k_assemble_Ap<2, M><<<nblk(L.nB, 128), 128, 0, st>>>(L, cvec, cval, A, a);
}
template void launch_assemble_Ap<double>(const LevelView<double>&, const double*, double, double*,
                                         const double*, cudaStream_t);
template void launch_assemble_Ap<float>(const LevelView<double>&, const double*, double, float*,
                                        const double*, cudaStream_t);

// ----------------------------------------------------------------- setup: dense A
// Row i of A = diag(c) - M: A_ii += c_i + gamma, A_ij -= E_{k,j}/dx^2 for each
// neighbour k of i and stencil node j of cp(x_k).  One thread per row.
template <int DIM, typename M>
__global__ void k_assemble_A(LevelView<double> L, const double* cvec, double cval, M* A) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const int32_t n = L.nB;
  if (i >= n) return;
  M* row = A + (size_t)i * n;
  row[i] += (M)((cvec ? cvec[i] : cval) + L.gamma);
  const uint64_t ki = L.key[i];
  const int own[3] = {key_x(ki), key_y(ki), key_z(ki)};
  const int d[6][3] = {{-1, 0, 0}, {1, 0, 0}, {0, -1, 0}, {0, 1, 0}, {0, 0, -1}, {0, 0, 1}};
  for (int q = 0; q < 2 * DIM; ++q) {
    const int32_t kk = node_index(L.bv, own[0] + d[q][0], own[1] + d[q][1], own[2] + d[q][2]);
    if (kk < 0) continue;
    const uint64_t key = L.key[kk];
    const int bx = key_x(key) + key_ox(key), by = key_y(key) + key_oy(key),
              bz = key_z(key) + key_oz(key);
    double wx[4], wy[4], wz[4] = {1.0, 0.0, 0.0, 0.0};
    cubic_w(L.fr[kk], wx);
    cubic_w(L.fr[L.nplus + kk], wy);
    if (DIM == 3) cubic_w(L.fr[2 * L.nplus + kk], wz);
    for (int c = 0; c < (DIM == 3 ? 4 : 1); ++c)
      for (int b = 0; b < 4; ++b)
        for (int a = 0; a < 4; ++a) {
          const int32_t j = band_index(L.bv, bx + a, by + b, DIM == 3 ? bz + c : 0);
          if (j >= 0) row[j] -= (M)(wx[a] * wy[b] * wz[c] * L.inv_h2);
        }
  }
}

template <typename M>
void launch_assemble_A(const LevelView<double>& L, const double* cvec, double cval, M* A,
                       cudaStream_t st) {
  if (L.dim == 3) k_assemble_A<3, M><<<nblk(L.nB, 128), 128, 0, st>>>(L, cvec, cval, A);
  else k_assemble_A<2, M><<<nblk(L.nB, 128), 128, 0, st>>>(L, cvec, cval, A);
}
template void launch_assemble_A<double>(const LevelView<double>&, const double*, double, double*,
                                        cudaStream_t);
template void launch_assemble_A<float>(const LevelView<double>&, const double*, double, float*,
                                       cudaStream_t);

// ----------------------------------------------------------------- instantiations
#define CPM_INST(T)                                                                              \
  template void launch_rm_jacobi<T>(const LevelView<T>&, const T*, const T*, const T*, T, T, T*, \
                                    cudaStream_t);                                               \
  template void launch_rm_resid<T>(const LevelView<T>&, const T*, const T*, const T*, T, T*,     \
                                   cudaStream_t);                                                \
  template void launch_transfer<T>(const TransferView<T>&, const T*, T*, bool, cudaStream_t);    \
  template void launch_lap_band<T>(const LevelView<T>&, const T*, T*, cudaStream_t);            \
  template void launch_lap_rel<T>(const LevelView<T>&, LapMode, const T*, const T*, const T*,   \
                                  const T*, const T*, T, const T*, T*, T*, double*, cudaStream_t); \
  template void launch_paper<T>(const LevelView<T>&, LapMode, const T*, const T*, const T*,     \
                                const T*, const T*, T, const T*, T*, T*, double*, const T*,      \
                                cudaStream_t);                                                   \
  template bool paper_fused<T>(const LevelView<T>&);                                            \
  template void launch_paper_fused<T>(const LevelView<T>&, LapMode, const T*, const T*, const T*, T, const T*, \
                                      T*, cudaStream_t);                                        \
  template void launch_lap_vard<T>(const LevelView<T>&, const T*, const T*, T*, cudaStream_t);  \
  template void launch_norm_partials<T>(const T*, int64_t, double*, cudaStream_t);               \
  template void launch_cast_to_f64<T>(const T*, double*, int64_t, cudaStream_t);                 \
  template void launch_cast_from_f64<T>(const double*, T*, int64_t, cudaStream_t);               \
  template void launch_coarse_gemv<T>(const double*, const T* const*, T* const*, int, int32_t, \
                                      cudaStream_t);
CPM_INST(double)
CPM_INST(float)

}  // namespace cpm
