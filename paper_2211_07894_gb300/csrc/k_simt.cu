// CUDA-core (FP64 / FP32) forms of the two contractions.  These serve the
// FP64 and FP32 precisions (k-point systems through the stacked real operand);
// the tensor-core forms live in k_tc.cu.
//
// GEMM1: X_k = Psi^T diag(a_k) Psi   (H-breve' = Psi~^T H~' Psi~, §II.C),
//        upper-triangular tiles over ranges of the grid rows, both triangles
//        written.
// GEMM2: drho_k(r) = g sum_j sum_{i<=j} Psi_ri X''_k,ij Psi_rj with X'' the
//        Loewner-scaled matrix with doubled strict upper triangle (the
//        diagonal of Psi X' Psi^T, Eq. densityResponse, using X' = X'^T);
//        Psi X'' is held in registers, never written to memory.
//
// FP32: bound by the FMA pipe, 128 fma a clock and SM.  Tiles of 128 x 128 (or
// 64 x 64 for small subspaces), 8 x 8 outputs a thread as packed pairs
// (fma.rn.f32x2: one issue slot for two fma, so that the operand loads and
// the packing fit beside them), warp tiles of 32 x 64; a warp whose columns
// lie below the diagonal skips its work.  The former 64 x 64 tiles with 4 x 4
// outputs spent half their issue slots on shared loads (26 % and 30 % of the
// FMA peak).  One GB300, 48^3 / 512, K = 8: GEMM1 11.2 -> 5.4 ms (64 % of the FMA
// pipe), GEMM2 9.7 -> 5.0 ms (68 %); 72^3 / 2048, K = 2: 120 -> 59 and 158 -> 57 ms.
//
// FP64: bound by the FP64 pipe, two fma a clock and SM, so what counts is the
// number of fma executed and an even spread over the SMs.  Tiles of 32 states
// (a 64-wide tile computes 4 times what 32 states need), only the upper half
// of a diagonal tile, and row ranges chosen to fill the SMs.  GEMM1, GEMM2 on one
// GB300, before -> now: 16^3 / 32, K = 4: 269 -> 24 us, 79 -> 24 us; 20 x 18 x 16 /
// 120, K = 3: 566 -> 303, 403 -> 246 us; 48^3 / 512, K = 2: 62.9 -> 49.4, 53.0 ->
// 47.5 ms.
#include "lrdm_internal.h"

namespace lrdm {
namespace {

__device__ __forceinline__ void tri_index(int p, int& I, int& J) {
  int j = (int)((sqrtf(8.0f * p + 1.0f) - 1.0f) * 0.5f);
  while (j * (j + 1) / 2 > p) --j;
  while ((j + 1) * (j + 2) / 2 <= p) ++j;
  J = j;
  I = p - j * (j + 1) / 2;
}

// ---------------------------------------------------------------------------
// FP32
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t p, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p));
}
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// T x T tile of T * T / 64 threads; BK deep stages, two of them.
template <int T>
struct F32Cfg {
  static constexpr int THREADS = T * T / 64;
  static constexpr int BK = T / 8;
  static constexpr int QUADS = BK * T / 4 / THREADS;      // float4 per operand, thread and stage
  static constexpr int BLOCKS = T == 128 ? 2 : 6;         // resident per SM
  static constexpr int LDP = T + 4;                       // row of the transposed Psi tile
  static_assert(QUADS * THREADS * 4 == BK * T, "stage loads");
};

// Warp tile 32 x 64: rows wr + (lane / 8) * 4 + {0..3, 16..19}, columns
// wc + (lane % 8) * 4 + {0..3, 32..35}: every shared load is 16 bytes a lane
// from 64 or 128 consecutive bytes.  acc[m][p]: columns 2 p, 2 p + 1 of row m.
__device__ __forceinline__ int f32_row(int lane, int m) { return (lane >> 3) * 4 + (m & 3) + (m >> 2) * 16; }
__device__ __forceinline__ int f32_col(int lane, int n) { return (lane & 7) * 4 + (n & 3) + (n >> 2) * 32; }

__device__ __forceinline__ void f32_step(const float* __restrict__ A, const float* __restrict__ B,
                                         int lane, uint64_t (&acc)[8][4]) {
  float a[8];
  *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(A + f32_row(lane, 0));
  *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(A + f32_row(lane, 4));
  ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(B + f32_col(lane, 0));
  ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(B + f32_col(lane, 4));
  const uint64_t b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const uint64_t aa = pack2(a[m], a[m]);
#pragma unroll
    for (int p = 0; p < 4; ++p) fma2(acc[m][p], aa, b[p]);
  }
}

// Four consecutive elements p[0..3] of a row, of which n are in range.
__device__ __forceinline__ float4 f32_quad(const float* __restrict__ p, int n, bool vec) {
  if (n <= 0) return make_float4(0.f, 0.f, 0.f, 0.f);
  if (vec) return __ldg(reinterpret_cast<const float4*>(p));      // ns a multiple of 4: all in range
  return make_float4(__ldg(p), n > 1 ? __ldg(p + 1) : 0.f, n > 2 ? __ldg(p + 2) : 0.f,
                     n > 3 ? __ldg(p + 3) : 0.f);
}

template <int T>
__global__ void __launch_bounds__(F32Cfg<T>::THREADS, F32Cfg<T>::BLOCKS)
    k_gemm1_f32(const float* __restrict__ psi, int ns, long long Ng, const float* __restrict__ a,
                long long a_stride, int nq, float* __restrict__ Xpart, long long rows_per, int vec) {
  using C = F32Cfg<T>;
  constexpr int BK = C::BK;
  __shared__ __align__(16) float As[2][BK][T];
  __shared__ __align__(16) float Bs[2][BK][T];
  int I, J;
  tri_index(blockIdx.x, I, J);
  const int q = blockIdx.y, split = blockIdx.z;
  const int i0 = I * T, j0 = J * T;
  const float* aq = a + (long long)q * a_stride;
  const long long rb = (long long)split * rows_per;
  const long long re = min(Ng, rb + rows_per);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wr = (warp % (T / 32)) * 32, wc = (warp / (T / 32)) * 64;
  const bool mine = i0 + wr <= j0 + wc + 63;             // some i <= j in this warp's tile
  uint64_t acc[8][4];
#pragma unroll
  for (int m = 0; m < 8; ++m)
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[m][p] = 0;
  // the next stage's values, weighted only when they are stored (a product
  // here would wait for the loads before the current stage is multiplied)
  float4 pa[C::QUADS], pb[C::QUADS];
  float pw[C::QUADS];
  auto fetch = [&](long long r0) {
#pragma unroll
    for (int u = 0; u < C::QUADS; ++u) {
      const int e = threadIdx.x + u * C::THREADS;
      const long long r = r0 + e / (T / 4);
      const int c = 4 * (e % (T / 4));
      const bool in = r < re;
      pw[u] = in ? __ldg(aq + r) : 0.f;
      pa[u] = f32_quad(psi + r * ns + i0 + c, in ? ns - i0 - c : 0, vec);
      pb[u] = f32_quad(psi + r * ns + j0 + c, in ? ns - j0 - c : 0, vec);
    }
  };
  auto stash = [&](int b) {
#pragma unroll
    for (int u = 0; u < C::QUADS; ++u) {
      const int e = threadIdx.x + u * C::THREADS;
      const int rr = e / (T / 4), c = 4 * (e % (T / 4));
      const float w = pw[u];
      *reinterpret_cast<float4*>(&As[b][rr][c]) = make_float4(pa[u].x * w, pa[u].y * w, pa[u].z * w, pa[u].w * w);
      *reinterpret_cast<float4*>(&Bs[b][rr][c]) = pb[u];
    }
  };
  if (rb < re) {
    fetch(rb);
    stash(0);
  }
  __syncthreads();
  int buf = 0;
  for (long long r0 = rb; r0 < re; r0 += BK) {
    const bool more = r0 + BK < re;
    if (more) fetch(r0 + BK);
    if (mine) {
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) f32_step(&As[buf][kk][wr], &Bs[buf][kk][wc], lane, acc);
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  if (!mine) return;
  float* Xq = Xpart + ((long long)split * nq + q) * (long long)ns * ns;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int i = i0 + wr + f32_row(lane, m);
    float v[8];
#pragma unroll
    for (int p = 0; p < 4; ++p) unpack2(acc[m][p], v[2 * p], v[2 * p + 1]);
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      const int j = j0 + wc + f32_col(lane, n);
      if (i <= j && j < ns) {
        Xq[(long long)i * ns + j] = v[n];
        if (i < j) Xq[(long long)j * ns + i] = v[n];
      }
    }
  }
}

// out = factor * sum (- v): io dtype with v, the compute type, or added to an
// FP64 accumulator
__device__ __forceinline__ void simt_store(const SimtOut& o, int q, long long r, double sum) {
  const double d = o.factor * sum;
  const long long at = q * o.stride + r;
  if (o.mode == SIMT_OUT_ADD) {
    static_cast<double*>(o.out)[at] += d;
  } else if (o.mode == SIMT_OUT_F) {
    const long long vt = q * o.v_stride + r;
    if (o.f64) static_cast<double*>(o.out)[at] = d - static_cast<const double*>(o.v)[vt];
    else static_cast<float*>(o.out)[at] = (float)(d - (double)static_cast<const float*>(o.v)[vt]);
  } else {
    if (o.f64) static_cast<double*>(o.out)[at] = d;
    else static_cast<float*>(o.out)[at] = (float)d;
  }
}

template <int T>
__global__ void __launch_bounds__(F32Cfg<T>::THREADS, F32Cfg<T>::BLOCKS)
    k_gemm2_f32(const float* __restrict__ psi, int ns, long long Ng, const float* __restrict__ Xpp,
                SimtOut o, int vec) {
  using C = F32Cfg<T>;
  constexpr int BK = C::BK;
  __shared__ __align__(16) float Ps[2][BK][C::LDP];      // transposed: [state][row]
  __shared__ __align__(16) float Xs[2][BK][T];
  __shared__ double red[T];
  const int q = blockIdx.y;
  const long long r0 = (long long)blockIdx.x * T;
  const float* Xq = Xpp + (long long)q * ns * ns;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wr = (warp % (T / 32)) * 32, wc = (warp / (T / 32)) * 64;
  // row sums over the j-tiles as FP32 pairs: accurate as FP64 sums of these
  // FP32 terms, without the FP64 pipe
  Pair32 ps[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) ps[m] = Pair32{0.f, 0.f};
  float4 pa[C::QUADS], px[C::QUADS];
  auto fetch = [&](int i0, int iend, int j0) {
#pragma unroll
    for (int u = 0; u < C::QUADS; ++u) {
      const int e = threadIdx.x + u * C::THREADS;
      const long long r = r0 + e / (BK / 4);
      const int i = i0 + 4 * (e % (BK / 4));
      pa[u] = r < Ng ? f32_quad(psi + r * ns + i, iend - i, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
      const int k = i0 + e / (T / 4), j = j0 + 4 * (e % (T / 4));
      px[u] = k < iend ? f32_quad(Xq + (long long)k * ns + j, ns - j, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto stash = [&](int b) {
#pragma unroll
    for (int u = 0; u < C::QUADS; ++u) {
      const int e = threadIdx.x + u * C::THREADS;
      const int rr = e / (BK / 4), k = 4 * (e % (BK / 4));
      Ps[b][k][rr] = pa[u].x;
      Ps[b][k + 1][rr] = pa[u].y;
      Ps[b][k + 2][rr] = pa[u].z;
      Ps[b][k + 3][rr] = pa[u].w;
      *reinterpret_cast<float4*>(&Xs[b][e / (T / 4)][4 * (e % (T / 4))]) = px[u];
    }
  };
  for (int j0 = 0; j0 < ns; j0 += T) {
    const int iend = min(ns, j0 + T);
    uint64_t acc[8][4];
#pragma unroll
    for (int m = 0; m < 8; ++m)
#pragma unroll
      for (int p = 0; p < 4; ++p) acc[m][p] = 0;
    fetch(0, iend, j0);
    stash(0);
    __syncthreads();
    int buf = 0;
    for (int i0 = 0; i0 < iend; i0 += BK) {
      const bool more = i0 + BK < iend;
      if (more) fetch(i0 + BK, iend, j0);
      if (i0 <= j0 + wc + 63) {                          // X'' is zero below its diagonal
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) f32_step(&Ps[buf][kk][wr], &Xs[buf][kk][wc], lane, acc);
      }
      if (more) stash(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
    // row-dot against the Psi(rows, J) tile
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const long long r = r0 + wr + f32_row(lane, m);
      if (r < Ng) {
        float v[8];
#pragma unroll
        for (int p = 0; p < 4; ++p) unpack2(acc[m][p], v[2 * p], v[2 * p + 1]);
        float s = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int j = j0 + wc + f32_col(lane, 4 * h);
          const float4 x = f32_quad(psi + r * ns + j, ns - j, vec);
          s += v[4 * h] * x.x + v[4 * h + 1] * x.y + v[4 * h + 2] * x.z + v[4 * h + 3] * x.w;
        }
        pair_add(ps[m], Pair32{s, 0.f});
      }
    }
  }
  // lanes of a row, then the column halves (warps wc = 0 and 64)
  double tot[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    double p = pair_value(ps[m]);
    for (int s = 4; s > 0; s >>= 1) p += __shfl_xor_sync(0xffffffffu, p, s);
    tot[m] = p;
    if (wc == 64 && (lane & 7) == 0) red[wr + f32_row(lane, m)] = p;
  }
  if (T == 128) __syncthreads();
  if (wc == 0 && (lane & 7) == 0) {
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int row = wr + f32_row(lane, m);
      if (r0 + row < Ng) simt_store(o, q, r0 + row, tot[m] + (T == 128 ? red[row] : 0.0));
    }
  }
}

// ---------------------------------------------------------------------------
// FP64
// ---------------------------------------------------------------------------

constexpr int D1 = 32;                  // GEMM1 tile (states)
constexpr int D2R = 64, D2C = 32;       // GEMM2: rows, columns of a j-tile
constexpr int DK = 16;

// 32 x 32 tile, 2 x 2 outputs a thread; a diagonal tile's threads take the 136
// micro-tiles on and above the diagonal (five warps of eight).
__global__ void __launch_bounds__(256) k_gemm1_f64(const double* __restrict__ psi, int ns, long long Ng,
                                                   const double* __restrict__ a, long long a_stride,
                                                   int nq, double* __restrict__ Xpart,
                                                   long long rows_per) {
  __shared__ __align__(16) double As[2][DK][D1];
  __shared__ __align__(16) double Bs[2][DK][D1];
  int I, J;
  tri_index(blockIdx.x, I, J);
  const int q = blockIdx.y, split = blockIdx.z;
  const int i0 = I * D1, j0 = J * D1;
  const double* aq = a + (long long)q * a_stride;
  const long long rb = (long long)split * rows_per;
  const long long re = min(Ng, rb + rows_per);
  int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  bool mine = true;
  if (I == J) {
    mine = threadIdx.x < 136;
    if (mine) tri_index(threadIdx.x, ty, tx);
  }
  // a micro-tile past the last state has nothing to do either
  if (i0 + 2 * ty >= ns || j0 + 2 * tx >= ns) mine = false;
  const int cc = threadIdx.x & 31, rr = threadIdx.x >> 5;          // rows rr, rr + 8 of a stage
  double pa[2], pb[2], pw[2];
  auto fetch = [&](long long r0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const long long r = r0 + rr + 8 * u;
      const bool in = r < re;
      pw[u] = in ? aq[r] : 0.0;
      pa[u] = in && i0 + cc < ns ? psi[r * ns + i0 + cc] : 0.0;
      pb[u] = in && j0 + cc < ns ? psi[r * ns + j0 + cc] : 0.0;
    }
  };
  auto stash = [&](int b) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      As[b][rr + 8 * u][cc] = pa[u] * pw[u];
      Bs[b][rr + 8 * u][cc] = pb[u];
    }
  };
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  if (rb < re) {
    fetch(rb);
    stash(0);
  }
  __syncthreads();
  int buf = 0;
  for (long long r0 = rb; r0 < re; r0 += DK) {
    const bool more = r0 + DK < re;
    if (more) fetch(r0 + DK);
    if (mine) {
#pragma unroll
      for (int kk = 0; kk < DK; ++kk) {
        const double2 x = *reinterpret_cast<const double2*>(&As[buf][kk][2 * ty]);
        const double2 y = *reinterpret_cast<const double2*>(&Bs[buf][kk][2 * tx]);
        acc[0][0] += x.x * y.x;
        acc[0][1] += x.x * y.y;
        acc[1][0] += x.y * y.x;
        acc[1][1] += x.y * y.y;
      }
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  if (!mine) return;
  double* Xq = Xpart + ((long long)split * nq + q) * (long long)ns * ns;
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const int i = i0 + 2 * ty + m, j = j0 + 2 * tx + n;
      if (i <= j && j < ns) {
        Xq[(long long)i * ns + j] = acc[m][n];
        if (i < j) Xq[(long long)j * ns + i] = acc[m][n];
      }
    }
}

// 64 rows x 32 columns: warp w takes columns 4 w .. 4 w + 3, its lanes the
// rows lane and lane + 32; a warp stops at its last column's state (X'' is
// zero below its diagonal).
__global__ void __launch_bounds__(256) k_gemm2_f64(const double* __restrict__ psi, int ns, long long Ng,
                                                   const double* __restrict__ Xpp, SimtOut o) {
  __shared__ __align__(16) double Ps[2][DK][D2R + 1];    // transposed: [state][row]
  __shared__ __align__(16) double Xs[2][DK][D2C];
  __shared__ double red[8][D2R];
  const int q = blockIdx.y;
  const long long r0 = (long long)blockIdx.x * D2R;
  const double* Xq = Xpp + (long long)q * ns * ns;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double part[2] = {0.0, 0.0};
  double pa[4], px[2];
  auto fetch = [&](int i0, int iend, int j0) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {                        // 16 states x 64 rows, states fastest
      const int e = threadIdx.x + 256 * u;
      const long long r = r0 + e / DK;
      const int i = i0 + e % DK;
      pa[u] = r < Ng && i < iend ? psi[r * ns + i] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = threadIdx.x + 256 * u;
      const int i = i0 + e / D2C, j = j0 + e % D2C;
      px[u] = i < iend && j < ns ? Xq[(long long)i * ns + j] : 0.0;
    }
  };
  auto stash = [&](int b) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = threadIdx.x + 256 * u;
      Ps[b][e % DK][e / DK] = pa[u];
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = threadIdx.x + 256 * u;
      Xs[b][e / D2C][e % D2C] = px[u];
    }
  };
  for (int j0 = 0; j0 < ns; j0 += D2C) {
    const int iend = min(ns, j0 + D2C);
    const int jw = j0 + 4 * warp;                        // first column of this warp
    const int last = jw < ns ? jw + 4 : 0;               // states this warp multiplies
    double acc[2][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int n = 0; n < 4; ++n) acc[m][n] = 0.0;
    fetch(0, iend, j0);
    stash(0);
    __syncthreads();
    int buf = 0;
    for (int i0 = 0; i0 < iend; i0 += DK) {
      const bool more = i0 + DK < iend;
      if (more) fetch(i0 + DK, iend, j0);
      const int n = min(DK, last - i0);
#pragma unroll 4
      for (int kk = 0; kk < n; ++kk) {
        const double x0 = Ps[buf][kk][lane], x1 = Ps[buf][kk][lane + 32];
        const double2 y0 = *reinterpret_cast<const double2*>(&Xs[buf][kk][4 * warp]);
        const double2 y1 = *reinterpret_cast<const double2*>(&Xs[buf][kk][4 * warp + 2]);
        acc[0][0] += x0 * y0.x;
        acc[0][1] += x0 * y0.y;
        acc[0][2] += x0 * y1.x;
        acc[0][3] += x0 * y1.y;
        acc[1][0] += x1 * y0.x;
        acc[1][1] += x1 * y0.y;
        acc[1][2] += x1 * y1.x;
        acc[1][3] += x1 * y1.y;
      }
      if (more) stash(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const long long r = r0 + lane + 32 * m;
      if (r < Ng)
#pragma unroll
        for (int n = 0; n < 4; ++n)
          if (jw + n < ns) part[m] += acc[m][n] * psi[r * ns + jw + n];
    }
  }
  red[warp][lane] = part[0];
  red[warp][lane + 32] = part[1];
  __syncthreads();
  if (threadIdx.x < D2R && r0 + threadIdx.x < Ng) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += red[w][threadIdx.x];
    simt_store(o, q, r0 + threadIdx.x, s);
  }
}

// Tile edge of the FP32 kernels: 128 unless 64-wide tiles compute clearly less
// (per fma the 64-wide form runs at about 0.85 of the 128-wide one's rate).
int f32_tile(int ns) {
  auto tri = [&](int t) {
    const double n = (ns + t - 1) / t;
    // executed states^2 of the upper tiles; a diagonal 128-tile skips a quarter
    return t == 128 ? 0.5 * n * (n - 1) * t * t + 0.75 * n * t * t : 0.5 * n * (n + 1) * t * t;
  };
  return tri(64) < 0.85 * tri(128) ? 64 : 128;
}

}  // namespace

// Grid-row ranges of GEMM1 for K directions, at most `slots` / K and 64.
// FP32: the count whose blocks fill the resident waves best (the smallest
// within 3 % of the best), ranges of at least 128 rows.  FP64: an SM's pipe is
// busy with one block, so the time is the SM with the most work: the blocks'
// mean load (a diagonal tile counts 0.625) plus half a block where they are
// dealt dynamically, or the largest block where every SM gets one at most,
// with a block's start and end taken as 6 rows; ranges of at least 32 rows.
int simt_split(int fp64, int ns, long long Ng, int K, int slots) {
  const int T = fp64 ? D1 : f32_tile(ns);
  const long long nt = (ns + T - 1) / T, tri = nt * (nt + 1) / 2;
  const long long k = K > 0 ? K : 1, sms = 152;
  long long most = Ng / (fp64 ? 32 : 128);
  if (most > slots / k) most = slots / k;
  if (most > 64) most = 64;
  if (most < 1) most = 1;
  int best = 1;
  if (fp64) {
    const double off = nt > 1 ? 1.0 : 0.625, mean = (double)(tri - nt) + 0.625 * (double)nt;
    double low = 1e300;
    for (long long sp = 1; sp <= most; ++sp) {
      const double rows = (double)((Ng + sp - 1) / sp + 6);
      const double cost = tri * k * sp <= sms ? off * rows : rows * (mean * k * sp / sms + 0.5 * off);
      if (cost < 0.97 * low) {            // the consumers add the partials
        low = cost;
        best = (int)sp;
      }
    }
    return best;
  }
  const long long units = sms * (T == 128 ? F32Cfg<128>::BLOCKS : F32Cfg<64>::BLOCKS);
  auto fill = [&](long long sp) {
    const long long b = tri * k * sp;
    return (double)b / (double)((b + units - 1) / units * units);
  };
  double top = 0.0;
  for (long long sp = 1; sp <= most; ++sp) top = fill(sp) > top ? fill(sp) : top;
  for (long long sp = 1; sp <= most; ++sp)
    if (fill(sp) >= 0.97 * top) return (int)sp;
  return best;
}

cudaError_t launch_gemm1_simt(int fp64, const void* psi, int ns, long long Ng, const void* a,
                              long long a_stride, int nq, void* Xpart, int nsplit,
                              cudaStream_t st) {
  if (nq == 0) return cudaSuccess;
  const int T = fp64 ? D1 : f32_tile(ns);
  const int nt = (ns + T - 1) / T;
  const long long rows_per = (Ng + nsplit - 1) / nsplit;
  const dim3 grid(nt * (nt + 1) / 2, nq, nsplit);
  if (fp64) {
    k_gemm1_f64<<<grid, 256, 0, st>>>(static_cast<const double*>(psi), ns, Ng, static_cast<const double*>(a),
                                      a_stride, nq, static_cast<double*>(Xpart), rows_per);
  } else {
    const int vec = ns % 4 == 0;                          // psi is a context's own allocation
    auto k = T == 128 ? k_gemm1_f32<128> : k_gemm1_f32<64>;
    k<<<grid, T * T / 64, 0, st>>>(static_cast<const float*>(psi), ns, Ng, static_cast<const float*>(a),
                                   a_stride, nq, static_cast<float*>(Xpart), rows_per, vec);
  }
  return cudaGetLastError();
}

cudaError_t launch_gemm2_simt(int fp64, const void* psi, int ns, long long Ng, const void* Xpp,
                              int nq, const SimtOut& o, cudaStream_t st) {
  if (nq == 0) return cudaSuccess;
  const int T = fp64 ? D2R : f32_tile(ns);
  const dim3 grid((unsigned)((Ng + T - 1) / T), nq);
  if (fp64) {
    k_gemm2_f64<<<grid, 256, 0, st>>>(static_cast<const double*>(psi), ns, Ng,
                                      static_cast<const double*>(Xpp), o);
  } else {
    const int vec = ns % 4 == 0;
    auto k = T == 128 ? k_gemm2_f32<128> : k_gemm2_f32<64>;
    k<<<grid, T * T / 64, 0, st>>>(static_cast<const float*>(psi), ns, Ng, static_cast<const float*>(Xpp), o,
                                   vec);
  }
  return cudaGetLastError();
}

}  // namespace lrdm
