// Learned smoother: a per-band-point network (31 -> 64 -> 64 -> 1) that
// replaces the first pre-smoothing Jacobi sweep (Eq. 4.1) of the finest
// level, with plain weighted Jacobi as its fallback and judge.  The paper has
// no learned component.
//
// Features of band point i: the residual at the 3x3x3 grid neighbourhood of
// x_i (0 off the band) divided by s_i = max |r| over it, (x_i - cp(x_i))/dx,
// and dx^2 M_ii.  Correction du_i = s_i dx^2 y_i, y = w3 . relu(W2^T
// relu(W1^T x + b1) + b2) + b3.
//
// Forward: BF16 weights and features, FP32 accumulation on the tensor cores
// (warp-level mma.sync m16n8k16, one warp per 32 points).  Training: the loss
// of a residual field r is ||r - A du||^2 / ||r||^2; its gradient with
// respect to du is -2 A^T (r - A du) / ||r||^2 (A^T through a transposed
// neighbour gather and a transposed extension scatter over the extension
// tiles), back-propagated through the network on the tensor cores (the three
// contractions as BF16 mma.sync with FP32 accumulation, bias gradients in
// FP32), reduced per CTA and summed in a fixed order; Adam on FP32 master
// weights.
#include <cuda_bf16.h>

#include <cmath>
#include <vector>

#include "mlp.cuh"

namespace cpm {

static unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// ----------------------------------------------------------------- static data
// nbr27[q * nB + i]: band index of x_i + (a, b, c) dx, q = (a+1) + 3(b+1) + 9(c+1),
// or -1; stat[a * nB + i]: (x_i - cp_i)/dx for a < 3, dx^2 M_ii for a = 3.
__global__ void k_mlp_static(BrickView v, const uint64_t* key, const double* cp, int64_t nplus,
                             int32_t nB, double lo, double dx, const double* diagM, int32_t* nbr27,
                             float* stat) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nB) return;
  const uint64_t k = key[i];
  const int x = key_x(k), y = key_y(k), z = key_z(k);
  int q = 0;
  for (int c = -1; c <= 1; ++c)
    for (int b = -1; b <= 1; ++b)
      for (int a = -1; a <= 1; ++a, ++q) nbr27[(int64_t)q * nB + i] = band_index(v, x + a, y + b, z + c);
  const int own[3] = {x, y, z};
  for (int a = 0; a < 3; ++a) {
    const double xa = lo + own[a] * dx;
    stat[(int64_t)a * nB + i] = (float)((xa - cp[a * nplus + i]) / dx);
  }
  stat[(int64_t)3 * nB + i] = (float)(dx * dx * diagM[i]);
}

// ----------------------------------------------------------------- forward
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <bool TRANS>
__device__ __forceinline__ void ldmatrix4(uint32_t (&d)[4], const __nv_bfloat16* p) {
  if (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)));
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)));
}

constexpr int kFwdWarps = 8;
constexpr int kW1S = 40;  // padded row (k) stride of the transposed W1 in shared memory (bf16)
constexpr int kW2S = 72;  // same for W2
constexpr int kXS = 40;   // padded row stride of the per-warp feature tile

struct MlpFwdArgs {
  const float* params;   // FP32 master parameters (layout in mlp.cuh)
  const float* r;        // residual on B (FP32)
  const int32_t* nbr27;
  const float* stat;
  int32_t nB;
  float dx2;
  float* du;             // out: correction ...
  float* u;              // ... or u += correction
  const uint32_t* uslot; // u's slots (brick-dense u), or null (band order)
  // training outputs
  __nv_bfloat16* Xs;     // nB x 32
  __nv_bfloat16* H1;     // nB x 64
  __nv_bfloat16* H2;     // nB x 64
  float* S;              // nB
};

// MODE: 0 du = correction, 1 u += correction, 2 du and the training outputs.
// Bound by the feature gather (27 indices, then 27 values, all in flight per
// lane) and the L1 data pipe, which also carries the weights: a warp reads each
// weight fragment once (ldmatrix) for its 32 points.  1.63 M points: 106 us with
// a point per lane and three CTAs on an SM; 113 us with the weights read once per
// 16 points, 170 us with a point per lane of a half warp.
template <int MODE>
__global__ void __launch_bounds__(kFwdWarps * 32, MODE == 2 ? 2 : 3) k_mlp_forward(MlpFwdArgs A) {
  __shared__ __align__(16) __nv_bfloat16 w1t[64 * kW1S];  // w1t[n][k] = W1[k][n]
  __shared__ __align__(16) __nv_bfloat16 w2t[64 * kW2S];
  __shared__ __align__(8) float bias1[64], bias2[64], w3s[64];
  __shared__ __align__(16) __nv_bfloat16 xs[kFwdWarps][32 * kXS];
  __shared__ float ss[kFwdWarps][32];
  for (int q = threadIdx.x; q < 64 * 32; q += blockDim.x) {
    const int n = q & 63, k = q >> 6;
    w1t[n * kW1S + k] = __float2bfloat16_rn(A.params[kOffW1 + k * 64 + n]);
  }
  for (int q = threadIdx.x; q < 64 * 64; q += blockDim.x) {
    const int n = q & 63, k = q >> 6;
    w2t[n * kW2S + k] = __float2bfloat16_rn(A.params[kOffW2 + k * 64 + n]);
  }
  for (int q = threadIdx.x; q < 64; q += blockDim.x) {
    bias1[q] = A.params[kOffB1 + q];
    bias2[q] = A.params[kOffB2 + q];
    w3s[q] = A.params[kOffW3 + q];
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int32_t nsteps = (A.nB + 31) / 32;
  for (int32_t step = (int32_t)blockIdx.x * kFwdWarps + warp; step < nsteps; step += (int32_t)gridDim.x * kFwdWarps) {
    // features: one point per lane
    {
      const int32_t p = step * 32 + lane;
      __nv_bfloat16* xw = xs[warp];
      float f[32];
      float smax = 0.f;
      if (p < A.nB) {
        int32_t j[27];
#pragma unroll
        for (int q = 0; q < 27; ++q) j[q] = __ldg(A.nbr27 + (int64_t)q * A.nB + p);
#pragma unroll
        for (int q = 0; q < 4; ++q) f[27 + q] = __ldg(A.stat + (int64_t)q * A.nB + p);
#pragma unroll
        for (int q = 0; q < 27; ++q) f[q] = j[q] >= 0 ? __ldg(A.r + j[q]) : 0.f;
#pragma unroll
        for (int q = 0; q < 27; ++q) smax = fmaxf(smax, fabsf(f[q]));
        const float inv = smax > 0.f ? 1.f / smax : 0.f;
#pragma unroll
        for (int q = 0; q < 27; ++q) f[q] *= inv;
      } else {
#pragma unroll
        for (int q = 0; q < 31; ++q) f[q] = 0.f;
      }
      f[31] = 0.f;
#pragma unroll
      for (int q = 0; q < 32; q += 8) {
        uint4 v;
        v.x = pack_bf16(f[q], f[q + 1]);
        v.y = pack_bf16(f[q + 2], f[q + 3]);
        v.z = pack_bf16(f[q + 4], f[q + 5]);
        v.w = pack_bf16(f[q + 6], f[q + 7]);
        *reinterpret_cast<uint4*>(&xw[lane * kXS + q]) = v;
        if (MODE == 2 && A.Xs && p < A.nB) reinterpret_cast<uint4*>(A.Xs + (int64_t)p * 32)[q / 8] = v;
      }
      ss[warp][lane] = smax;
    }
    __syncwarp();
    const int32_t p0 = step * 32 + g;  // this lane's rows: p0 + 8 q, q = 0 .. 3
    // layer 1: [32 x 32] x [32 x 64]
    uint32_t a[2][2][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int kc = 0; kc < 2; ++kc)
        ldmatrix4<false>(a[m][kc], &xs[warp][(16 * m + (lane & 15)) * kXS + kc * 16 + (lane >> 4) * 8]);
    // relu(h1) as the A operand of layer 2 (C tiles 2j, 2j+1 form k-chunk j)
    uint32_t a2[2][4][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      uint32_t wb[4];
      ldmatrix4<false>(wb, &w1t[(nt * 8 + (lane & 7)) * kW1S + (lane >> 3) * 8]);
      const float2 bb = *reinterpret_cast<const float2*>(&bias1[nt * 8 + 2 * t]);
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        float h[4] = {bb.x, bb.y, bb.x, bb.y};
#pragma unroll
        for (int kc = 0; kc < 2; ++kc) mma_bf16(h, a[m][kc], wb[2 * kc], wb[2 * kc + 1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) h[e] = fmaxf(h[e], 0.f);
        a2[m][nt / 2][2 * (nt & 1)] = pack_bf16(h[0], h[1]);
        a2[m][nt / 2][2 * (nt & 1) + 1] = pack_bf16(h[2], h[3]);
      }
    }
    if (MODE == 2 && A.H1) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int32_t r = p0 + 8 * q;
        if (r < A.nB)
#pragma unroll
          for (int nt = 0; nt < 8; ++nt)
            *reinterpret_cast<uint32_t*>(A.H1 + (int64_t)r * 64 + nt * 8 + 2 * t) = a2[q / 2][nt / 2][2 * (nt & 1) + (q & 1)];
      }
    }
    // layer 2: [32 x 64] x [64 x 64], then relu and the dot with w3
    float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
    for (int nt = 0; nt < 8; ++nt) {
      const int n = nt * 8 + 2 * t;
      uint32_t wb[2][4];
#pragma unroll
      for (int k2 = 0; k2 < 2; ++k2)
        ldmatrix4<false>(wb[k2], &w2t[(nt * 8 + (lane & 7)) * kW2S + 32 * k2 + (lane >> 3) * 8]);
      const float2 bb = *reinterpret_cast<const float2*>(&bias2[n]), w3 = *reinterpret_cast<const float2*>(&w3s[n]);
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        float c[4] = {bb.x, bb.y, bb.x, bb.y};
#pragma unroll
        for (int kc = 0; kc < 4; ++kc) mma_bf16(c, a2[m][kc], wb[kc / 2][2 * (kc & 1)], wb[kc / 2][2 * (kc & 1) + 1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) c[e] = fmaxf(c[e], 0.f);
        if (MODE == 2 && A.H2) {
          const int32_t r0 = p0 + 16 * m, r1 = r0 + 8;
          if (r0 < A.nB) *reinterpret_cast<uint32_t*>(A.H2 + (int64_t)r0 * 64 + n) = pack_bf16(c[0], c[1]);
          if (r1 < A.nB) *reinterpret_cast<uint32_t*>(A.H2 + (int64_t)r1 * 64 + n) = pack_bf16(c[2], c[3]);
        }
        y[2 * m] += c[0] * w3.x + c[1] * w3.y;
        y[2 * m + 1] += c[2] * w3.x + c[3] * w3.y;
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      y[q] += __shfl_xor_sync(0xffffffffu, y[q], 1);
      y[q] += __shfl_xor_sync(0xffffffffu, y[q], 2);
    }
    // lane t of a row's four writes row p0 + 8 t
    {
      const int32_t r = p0 + 8 * t;
      const float yt = t == 0 ? y[0] : t == 1 ? y[1] : t == 2 ? y[2] : y[3];
      if (r < A.nB) {
        const float sc = ss[warp][8 * t + g];
        const float d = sc * A.dx2 * (yt + __ldg(A.params + kOffB3));
        if (MODE == 1) A.u[A.uslot ? A.uslot[r] : r] += d; else A.du[r] = d;
        if (MODE == 2 && A.S) A.S[r] = sc;
      }
    }
    __syncwarp();
  }
}

// ----------------------------------------------------------------- backward
// The backward pass runs on a fixed grid of kBwdCtas CTAs, each writing one
// partial gradient (kBwdCtas x 25 KB whatever the band size).
constexpr int kBwdCtas = 2 * 152;

// Tensor-core backward.  A CTA of 8 warps loops over groups of kBwdPts points,
// copied to shared memory (two CTAs on an SM: one waits for its copies while the
// other contracts); BF16 mma.sync.m16n8k16, FP32 accumulation:
//   dz1 = (dz2 W2^T) [h1 > 0]    M = points, N = 64, K = 64       (warp w: points 16 w .. 16 w + 15)
//   dW2 += H1^T dz2              M = 64, N = 64, K = points       (warp w: rows 16 (w / 2), columns 32 (w % 2))
//   dW1 += X^T dz1               M = 32, N = 64, K = points       (warp w: rows 16 (w / 4), columns 16 (w % 4))
// with dz2 = dy w3 [h2 > 0].  All operands lie in shared memory point by point;
// the contractions over points read them with transposing matrix loads.  The
// dW accumulators and the FP32 bias sums stay in registers over all the CTA's
// groups; each CTA writes one partial gradient, summed by k_grad_reduce.
// Bound by the reads of the stored activations (324 bytes per point) and three
// barriers per group: 342 thousand points 56 us, against 528 us with 16 points
// per step copied value by value.
constexpr int kBwdWarps = 8;
constexpr int kBwdPts = 16 * kBwdWarps;
constexpr int kRowX = 40;  // row strides (bf16) in shared memory
constexpr int kRowH = 72;

struct BwdStage {
  __nv_bfloat16 x[kBwdPts * kRowX];
  __nv_bfloat16 h1[kBwdPts * kRowH];
  __nv_bfloat16 h2[kBwdPts * kRowH];
  float dy[kBwdPts];
};
struct BwdShared {
  BwdStage st;
  __nv_bfloat16 dz1[kBwdPts * kRowH];
  __nv_bfloat16 w2[64 * kRowH];  // w2[k][j] = W2[k][j]
  float w3[64];
  float red[3][kBwdWarps][64];
};

__device__ __forceinline__ void copy16_or_zero(void* smem, const void* gmem, bool ok) {
  const uint32_t n = ok ? 16 : 0;  // bytes read; the rest is zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem), "r"(n)
               : "memory");
}
// Copies of one group (zero rows past the last point).
__device__ __forceinline__ void bwd_fetch(BwdStage& s, const float* dy, const __nv_bfloat16* Xs,
                                          const __nv_bfloat16* H1, const __nv_bfloat16* H2, int64_t p0,
                                          int32_t nB) {
  for (int q = threadIdx.x; q < kBwdPts * 20; q += blockDim.x) {  // 16-byte words: 4 of x, 8 of h1, 8 of h2
    const int p = q / 20, c = q - 20 * p;
    const bool ok = p0 + p < nB;
    const int64_t gp = ok ? p0 + p : 0;
    if (c < 4) copy16_or_zero(s.x + p * kRowX + 8 * c, Xs + gp * 32 + 8 * c, ok);
    else if (c < 12) copy16_or_zero(s.h1 + p * kRowH + 8 * (c - 4), H1 + gp * 64 + 8 * (c - 4), ok);
    else copy16_or_zero(s.h2 + p * kRowH + 8 * (c - 12), H2 + gp * 64 + 8 * (c - 12), ok);
  }
  for (int p = threadIdx.x; p < kBwdPts; p += blockDim.x) s.dy[p] = p0 + p < nB ? __ldg(dy + p0 + p) : 0.f;
  asm volatile("cp.async.commit_group;" ::: "memory");
}

__global__ void __launch_bounds__(kBwdWarps * 32, 2) k_mlp_backward_tc(const float* params, const float* dy,
                                                                    const __nv_bfloat16* Xs,
                                                                    const __nv_bfloat16* H1,
                                                                    const __nv_bfloat16* H2, int32_t nB,
                                                                    float* part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BwdShared& S = *reinterpret_cast<BwdShared*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  const int64_t ngroups = ((int64_t)nB + kBwdPts - 1) / kBwdPts;
  if (blockIdx.x < ngroups) bwd_fetch(S.st, dy, Xs, H1, H2, (int64_t)blockIdx.x * kBwdPts, nB);
  for (int q = tid; q < 64 * 64; q += blockDim.x)
    S.w2[(q >> 6) * kRowH + (q & 63)] = __float2bfloat16_rn(params[kOffW2 + q]);
  if (tid < 64) S.w3[tid] = params[kOffW3 + tid];
  __syncthreads();
  const int j2 = 2 * lane;  // column pair of the elementwise step
  const float w3a = S.w3[j2], w3b = S.w3[j2 + 1];
  float acc2[4][4], acc1[2][4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
#pragma unroll
    for (int a = 0; a < 4; ++a) acc2[a][e] = 0.f;
#pragma unroll
    for (int a = 0; a < 2; ++a) acc1[a][e] = 0.f;
  }
  float sb2[2] = {0.f, 0.f}, sw3[2] = {0.f, 0.f}, sb3 = 0.f, sb1[8][2];
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) sb1[nt][0] = sb1[nt][1] = 0.f;
  BwdStage& s = S.st;
  for (int64_t grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
    __nv_bfloat16* dz2 = s.h2;  // takes h2's place, element by element
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // this group has arrived
    // dz2 and the column sums: warp w the points 16 w .. 16 w + 15, a column pair per lane
#pragma unroll 4
    for (int i = 0; i < 16; ++i) {
      const int p = 16 * warp + i;
      const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(s.h2 + p * kRowH + j2);
      const float ha = __low2float(h), hb = __high2float(h), d = s.dy[p];
      const float da = ha > 0.f ? d * w3a : 0.f, db = hb > 0.f ? d * w3b : 0.f;
      sb2[0] += da;
      sb2[1] += db;
      sw3[0] += d * ha;
      sw3[1] += d * hb;
      sb3 += d;
      *reinterpret_cast<uint32_t*>(dz2 + p * kRowH + j2) = pack_bf16(da, db);
    }
    __syncwarp();
    // dz1 of the warp's 16 points
    {
      uint32_t a[4][4];
#pragma unroll
      for (int kc = 0; kc < 4; ++kc)
        ldmatrix4<false>(a[kc], dz2 + (16 * warp + (lane & 15)) * kRowH + 16 * kc + 8 * (lane >> 4));
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k2 = 0; k2 < 2; ++k2) {
          uint32_t b[4];
          ldmatrix4<false>(b, S.w2 + (8 * nt + (lane & 7)) * kRowH + 32 * k2 + 8 * (lane >> 3));
          mma_bf16(c, a[2 * k2], b[0], b[1]);
          mma_bf16(c, a[2 * k2 + 1], b[2], b[3]);
        }
        const int k0 = 8 * nt + 2 * t;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int p = 16 * warp + g + 8 * r;
          const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(s.h1 + p * kRowH + k0);
          const float va = __low2float(h) > 0.f ? c[2 * r] : 0.f, vb = __high2float(h) > 0.f ? c[2 * r + 1] : 0.f;
          sb1[nt][0] += va;
          sb1[nt][1] += vb;
          *reinterpret_cast<uint32_t*>(S.dz1 + p * kRowH + k0) = pack_bf16(va, vb);
        }
      }
    }
    __syncthreads();
    // dW2 and dW1 over the group's points
    const int m2 = 16 * (warp >> 1), n2 = 32 * (warp & 1), m1 = 16 * (warp >> 2), n1 = 16 * (warp & 3);
#pragma unroll 2
    for (int kc = 0; kc < kBwdPts / 16; ++kc) {
      // transposed 8 x 8 blocks: rows are points, so a lane's address is a point's row
      const int ra = 16 * kc + (lane & 7) + 8 * (lane >> 4), ca = 8 * ((lane >> 3) & 1);
      const int rb = 16 * kc + (lane & 15), cb = 8 * (lane >> 4);
      uint32_t a[4], b[4];
      ldmatrix4<true>(a, s.h1 + ra * kRowH + m2 + ca);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        ldmatrix4<true>(b, dz2 + rb * kRowH + n2 + 16 * h + cb);
        mma_bf16(acc2[2 * h], a, b[0], b[1]);
        mma_bf16(acc2[2 * h + 1], a, b[2], b[3]);
      }
      ldmatrix4<true>(a, s.x + ra * kRowX + m1 + ca);
      ldmatrix4<true>(b, S.dz1 + rb * kRowH + n1 + cb);
      mma_bf16(acc1[0], a, b[0], b[1]);
      mma_bf16(acc1[1], a, b[2], b[3]);
    }
    __syncthreads();  // every warp has left the group
    if (grp + gridDim.x < ngroups) bwd_fetch(s, dy, Xs, H1, H2, (grp + gridDim.x) * kBwdPts, nB);
  }
  float* out = part + (int64_t)blockIdx.x * kNParams;
#pragma unroll
  for (int nt = 0; nt < 4; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int k = 16 * (warp >> 1) + g + (e >> 1) * 8, j = 32 * (warp & 1) + 8 * nt + 2 * t + (e & 1);
      out[kOffW2 + k * 64 + j] = acc2[nt][e];
    }
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int f = 16 * (warp >> 2) + g + (e >> 1) * 8, k = 16 * (warp & 3) + 8 * nt + 2 * t + (e & 1);
      out[kOffW1 + f * 64 + k] = acc1[nt][e];
    }
  // bias sums: over the lanes of a column, then over the warps in order
#pragma unroll
  for (int nt = 0; nt < 8; ++nt)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float v = sb1[nt][e];
      v += __shfl_xor_sync(0xffffffffu, v, 4);
      v += __shfl_xor_sync(0xffffffffu, v, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 16);
      if (g == 0) S.red[0][warp][8 * nt + 2 * t + e] = v;
    }
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    S.red[1][warp][j2 + e] = sb2[e];
    S.red[2][warp][j2 + e] = sw3[e];
  }
  __syncthreads();
  if (tid < 192) {
    const int which = tid >> 6, q = tid & 63;
    float v = 0.f;
    for (int w = 0; w < kBwdWarps; ++w) v += S.red[which][w][q];
    out[(which == 0 ? kOffB1 : which == 1 ? kOffB2 : kOffW3) + q] = v;
  }
  __syncthreads();
  if (lane == 0) S.red[0][warp][0] = sb3;
  __syncthreads();
  if (tid == 0) {
    float v = 0.f;
    for (int w = 0; w < kBwdWarps; ++w) v += S.red[0][w][0];
    out[kOffB3] = v;
  }
}

// grad[q] = sum over CTAs of part[c][q] (fixed order).
// A block takes 32 parameters, its 8 warps every eighth partial.
__global__ void __launch_bounds__(256) k_grad_reduce(const float* part, int nparts, float* grad) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int q = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (q < kNParams)
    for (int c = warp; c < nparts; c += 8) s += part[(int64_t)c * kNParams + q];
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && q < kNParams) {
    for (int w = 1; w < 8; ++w) s += red[w][lane];
    grad[q] = s;
  }
}

// Adam (Kingma & Ba) on the FP32 master parameters.
__global__ void k_adam(float* params, const float* grad, float* m, float* v, float lr, float b1,
                       float b2, float eps, float bc1, float bc2) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= kNParams) return;
  if (q >= kOffW1 + 31 * 64 && q < kOffW1 + 32 * 64) return;  // zero-feature row stays 0
  const float g = grad[q];
  const float mq = b1 * m[q] + (1.f - b1) * g;
  const float vq = b2 * v[q] + (1.f - b2) * g * g;
  m[q] = mq;
  v[q] = vq;
  params[q] -= lr * (mq / bc1) / (sqrtf(vq / bc2) + eps);
}

// ----------------------------------------------------------------- A^T
// t[k] = sum of z_i over the grid neighbours i of k (k in B+) that are in B.
__global__ void k_nbr_transpose(BrickView v, const uint64_t* key, int64_t nplus, int dim,
                                const float* z, float* t) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nplus) return;
  const uint64_t kk = key[k];
  const int x = key_x(kk), y = key_y(kk), zc = key_z(kk);
  const int d[6][3] = {{-1, 0, 0}, {1, 0, 0}, {0, -1, 0}, {0, 1, 0}, {0, 0, -1}, {0, 0, 1}};
  float s = 0.f;
  for (int q = 0; q < 2 * dim; ++q) {
    const int32_t i = band_index(v, x + d[q][0], y + d[q][1], zc + d[q][2]);
    if (i >= 0) s += z[i];
  }
  t[k] = s;
}

// out[j] += sum_k E_{kj} t[k], one warp per extension tile.  Each lane takes a
// base and sums its points' 4^3 weighted values in registers (6.6 points share
// a base on a smooth surface), then adds them to the tile's box in shared
// memory; the box is added to out.  342 thousand points: 36 us, against 148 us
// with one shared-memory addition per point and node.
constexpr int kExtTWarps = 2;
__global__ void __launch_bounds__(32 * kExtTWarps) k_extend_transpose(LevelView<float> L, const float* t,
                                                                      float* out) {
  __shared__ float boxes[kExtTWarps][344];
  __shared__ int32_t runs[kExtTWarps][64][4];  // per base: its points of B and of G, begin and end
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t tile = blockIdx.x * kExtTWarps + warp;
  if (tile >= L.ntiles) return;
  float* box = boxes[warp];
  for (int q = lane; q < 343; q += 32) box[q] = 0.f;
  for (int q = lane; q < 256; q += 32) runs[warp][q >> 2][q & 3] = 0;
  __syncwarp();
  const int32_t beg = L.tile_start[tile], mid = L.tile_mid[tile], end = L.tile_start[tile + 1];
  for (int32_t k = beg + lane; k < end; k += 32) {
    const uint32_t pos = L.erec[k] & 63u;
    const int part = k < mid ? 0 : 2;
    if (k == beg || k == mid || (L.erec[k - 1] & 63u) != pos) runs[warp][pos][part] = k;
    if (k + 1 == end || k + 1 == mid || (L.erec[k + 1] & 63u) != pos) runs[warp][pos][part + 1] = k + 1;
  }
  __syncwarp();
  const int64_t np = L.nplus;
  // the bases that have points, dealt to the lanes in turn
  uint32_t has0 = __ballot_sync(0xffffffffu, runs[warp][lane][1] + runs[warp][lane][3] > 0);
  uint32_t has1 = __ballot_sync(0xffffffffu, runs[warp][lane + 32][1] + runs[warp][lane + 32][3] > 0);
  const int n0 = __popc(has0), nbase = n0 + __popc(has1);
  for (int q = lane; q < nbase; q += 32) {
    const int pos = q < n0 ? (int)__fns(has0, 0, q + 1) : 32 + (int)__fns(has1, 0, q - n0 + 1);
    float acc[64];
#pragma unroll
    for (int e = 0; e < 64; ++e) acc[e] = 0.f;
#pragma unroll 1
    for (int part = 0; part < 4; part += 2) {
      const int32_t k1 = runs[warp][pos][part + 1];
#pragma unroll 1
      for (int32_t k = runs[warp][pos][part]; k < k1; ++k) {
        const float tv = t[L.erec[k] >> 6];
        const float s3[3] = {L.efr[k], L.efr[np + k], L.efr[2 * np + k]};
        float w[3][4];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const float s = s3[a], sm1 = s - 1.f, sm2 = s - 2.f, sp1 = s + 1.f;
          const float p = s * sm1, qq = sp1 * sm2;
          w[a][0] = (p * sm2) * (-1.f / 6.f);
          w[a][1] = (qq * sm1) * 0.5f;
          w[a][2] = (qq * s) * -0.5f;
          w[a][3] = (p * sp1) * (1.f / 6.f);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const float v = w[2][c] * w[1][b] * tv;
#pragma unroll
            for (int a = 0; a < 4; ++a) acc[(c * 4 + b) * 4 + a] += w[0][a] * v;
          }
      }
    }
    const int lx = pos & 3, ly = (pos >> 2) & 3, lz = pos >> 4;
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a)
          atomicAdd(&box[((lz + c) * 7 + ly + b) * 7 + lx + a], acc[(c * 4 + b) * 4 + a]);
  }
  __syncwarp();
  for (int q = lane; q < 343; q += 32) {
    const float val = box[q];
    if (val == 0.f) continue;
    const int x = q % 7, y = (q / 7) % 7, z = q / 49;
    const int j = (x >> 2) | ((y >> 2) << 1) | ((z >> 2) << 2);
    const uint64_t bit = 1ull << ((x & 3) | ((y & 3) << 2) | ((z & 3) << 4));
    const uint64_t m = __ldg(L.tile_mask + 8 * (int64_t)tile + j);
    if (m & bit) atomicAdd(out + __ldg(L.tile_bstart + 8 * (int64_t)tile + j) + __popcll(m & (bit - 1)), val);
  }
}

// dy = -2 (A^T z) s dx^2 / ||r||^2 with A^T z = (c + gamma) z - ext^T / dx^2.
__global__ void k_mlp_dy(const float* z, const float* et, const float* cvec, float cval, float gamma,
                         float inv_h2, const float* S, float dx2, const double* nr2, int32_t nB,
                         float* dy) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nB) return;
  const float c = cvec ? cvec[i] : cval;
  const float atz = (c + gamma) * z[i] - et[i] * inv_h2;
  dy[i] = (float)(-2.0 / nr2[0]) * atz * S[i] * dx2;
}

// z = r - (c du - M du) given Mdu; partial sums of z^2 and r^2 per block.
__global__ void k_mlp_resid(const float* r, const float* du, const float* Mdu, const float* cvec,
                            float cval, int32_t nB, float* z, double* part) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  double zz = 0.0, rr = 0.0;
  if (i < nB) {
    const float c = cvec ? cvec[i] : cval;
    const float zi = r[i] - (c * du[i] - Mdu[i]);
    z[i] = zi;
    zz = (double)zi * zi;
    rr = (double)r[i] * r[i];
  }
  __shared__ double s1[8], s2[8];
  for (int o = 16; o > 0; o >>= 1) {
    zz += __shfl_xor_sync(0xffffffffu, zz, o);
    rr += __shfl_xor_sync(0xffffffffu, rr, o);
  }
  if ((threadIdx.x & 31) == 0) { s1[threadIdx.x >> 5] = zz; s2[threadIdx.x >> 5] = rr; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, b = 0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) { a += s1[q]; b += s2[q]; }
    part[2 * blockIdx.x] = a;
    part[2 * blockIdx.x + 1] = b;
  }
}

// out[0] = ||z||^2, out[1] = ||r||^2 (fixed order).
__global__ void __launch_bounds__(1024) k_mlp_loss_final(const double* part, int nblocks, double* out) {
  double a = 0.0, b = 0.0;
  for (int q = threadIdx.x; q < nblocks; q += blockDim.x) {
    a += part[2 * q];
    b += part[2 * q + 1];
  }
  __shared__ double sa[32], sb[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) {
    sa[threadIdx.x >> 5] = a;
    sb[threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = b = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += sa[w];
      b += sb[w];
    }
    out[0] = a;
    out[1] = b;
  }
}

// ----------------------------------------------------------------- host side
void MlpLevelData::build(const Level& lev, const double* diagM, cudaStream_t st) {
  nB = lev.nB;
  nbr27.alloc((size_t)27 * nB);
  stat.alloc((size_t)4 * nB);
  k_mlp_static<<<nblk(nB, 256), 256, 0, st>>>(lev.view(), lev.key.get(), lev.cp.get(), lev.nplus(), nB,
                                              lev.lo, lev.dx, diagM, nbr27.get(), stat.get());
  CPM_CUDA_TRY(cudaGetLastError());
}

void mlp_forward(const float* params, const MlpLevelData& D, const float* r, float dx2, float* du,
                 float* u_add, const uint32_t* uslot, const MlpTrainBuffers* tb, cudaStream_t st) {
  MlpFwdArgs a{};
  a.params = params;
  a.r = r;
  a.nbr27 = D.nbr27.get();
  a.stat = D.stat.get();
  a.nB = D.nB;
  a.dx2 = dx2;
  a.du = du;
  a.u = u_add;
  a.uslot = uslot;
  if (tb) {
    a.Xs = tb->Xs.get();
    a.H1 = tb->H1.get();
    a.H2 = tb->H2.get();
    a.S = tb->S.get();
  }
  const int64_t steps = ((int64_t)D.nB + 31) / 32;
  const unsigned grid = (unsigned)std::min<int64_t>((steps + kFwdWarps - 1) / kFwdWarps, 152 * 6);
  if (u_add)
    k_mlp_forward<1><<<grid, kFwdWarps * 32, 0, st>>>(a);
  else if (tb)
    k_mlp_forward<2><<<grid, kFwdWarps * 32, 0, st>>>(a);
  else
    k_mlp_forward<0><<<grid, kFwdWarps * 32, 0, st>>>(a);
  count_launch();
}

void MlpTrainBuffers::ensure(int32_t nB, int64_t nplus, int64_t slots) {
  nparts = kBwdCtas;
  if (nB <= n && nplus <= np && slots <= ns) return;  // capacity suffices
  n = nB = std::max(n, nB);
  np = nplus = std::max(np, nplus);
  ns = slots = std::max(ns, slots);
  Xs.alloc((size_t)nB * 32);
  H1.alloc((size_t)nB * 64);
  H2.alloc((size_t)nB * 64);
  S.alloc(nB);
  du.alloc(nB);
  Mdu.alloc(nB);
  z.alloc(nB);
  w.alloc(slots);
  t.alloc(nplus);
  et.alloc(nB);
  dy.alloc(nB);
  nparts = kBwdCtas;
  part.alloc((size_t)nparts * kNParams);
  lpart.alloc(2 * (size_t)((nB + 255) / 256));
  loss.alloc(2);
  grad.alloc(kNParams);
}

// Loss and gradient of one residual field (FP32 on level 0 of the view L).
void mlp_loss_grad(const float* params, const MlpLevelData& D, const LevelView<float>& L,
                   const DenseView& DL, const float* cvec, float cval, const float* r, MlpTrainBuffers& tb,
                   cudaStream_t st) {
  const int32_t nB = L.nB;
  const float dx2 = 1.f / L.inv_h2;
  // (per call: the attribute belongs to the device that is current)
  CPM_CUDA_TRY(cudaFuncSetAttribute(k_mlp_backward_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sizeof(BwdShared)));
  tb.ensure(nB, L.nplus, ((int64_t)DL.nbricks + 1) << (2 * DL.dim));
  mlp_forward(params, D, r, dx2, tb.du.get(), nullptr, nullptr, &tb, st);
  // M du (extension over B+ then the stencil)
  const Vec32<const float> du{nullptr, tb.du.get()};
  launch_extend32(DL, DL.all, du, tb.w.get(), st);
  launch_lap32(DL, LAP_APPLY, du, tb.w.get(), nullptr, 0.f, Vec32<float>{nullptr, tb.Mdu.get()}, nullptr,
               all_rows(DL), st);
  const int nb256 = (int)((nB + 255) / 256);
  k_mlp_resid<<<nb256, 256, 0, st>>>(r, tb.du.get(), tb.Mdu.get(), cvec, cval, nB, tb.z.get(),
                                      tb.lpart.get());
  k_mlp_loss_final<<<1, 1024, 0, st>>>(tb.lpart.get(), nb256, tb.loss.get());
  // A^T z = (c + gamma) z - E^T (N^T z) / dx^2
  k_nbr_transpose<<<nblk(L.nplus, 256), 256, 0, st>>>(L.bv, L.key, L.nplus, L.dim, tb.z.get(),
                                                       tb.t.get());
  CPM_CUDA_TRY(cudaMemsetAsync(tb.et.get(), 0, sizeof(float) * nB, st));
  k_extend_transpose<<<nblk(L.ntiles, kExtTWarps), 32 * kExtTWarps, 0, st>>>(L, tb.t.get(), tb.et.get());
  k_mlp_dy<<<nb256, 256, 0, st>>>(tb.z.get(), tb.et.get(), cvec, cval, L.gamma, L.inv_h2, tb.S.get(),
                                   dx2, tb.loss.get() + 1, nB, tb.dy.get());
  k_mlp_backward_tc<<<tb.nparts, kBwdWarps * 32, sizeof(BwdShared), st>>>(params, tb.dy.get(), tb.Xs.get(), tb.H1.get(),
                                                         tb.H2.get(), nB, tb.part.get());
  k_grad_reduce<<<nblk(kNParams, 32), 256, 0, st>>>(tb.part.get(), tb.nparts, tb.grad.get());
  count_launch(9);
  CPM_CUDA_TRY(cudaGetLastError());
}

void mlp_adam(float* params, const float* grad, float* m, float* v, int64_t step, float lr,
              cudaStream_t st) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float bc1 = 1.f - std::pow(b1, (float)step), bc2 = 1.f - std::pow(b2, (float)step);
  k_adam<<<nblk(kNParams, 256), 256, 0, st>>>(params, grad, m, v, lr, b1, b2, 1e-8f, bc1, bc2);
  count_launch();
}

}  // namespace cpm
