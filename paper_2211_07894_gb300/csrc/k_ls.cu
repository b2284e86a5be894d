// The low-rank least-squares step (Eqs. plowrank, relativeError, quasinewton):
//   S_kl = <f_k, f_l>, c_k = <f_k, R>, ||R||^2   (partial sums in a fixed order)
//   a = S^+ c: by elimination (S = L D L^T) when S is certified to have no
//   eigenvalue below the cutoff, else S = Q diag(lambda) Q^T by parallel cyclic
//   Jacobi rotations (lambda < rcond lambda_max dropped -> SINGULAR flag); FP64
//   Delta = sum_k a_k v_k, rho <- rho - alpha Delta, s_rel = ||F a - R|| / ||R||
//
// GB300 executes two FP64 operations per clock and SM against 128 in FP32, so
// the grid-length sums of FP32 data run as compensated FP32 sums: products and
// sums are split into value and rounding error (x y = p + e with
// e = fma(x, y, -p); Knuth's two-sum), the errors summed in a second word
// (the Dot2 algorithm of Ogita, Rump and Oishi, 2005), at eleven FP32 operations a
// product in place of one FP64 fma at 64 times the cost.  A product and an
// addition are good to about 2^-48.  The second word is itself an FP32 sum: left
// to grow beside the first, its rounding grows with the square of the number of
// terms, so it is folded back (dot4, UPD_NORM), and sums go to FP64 at GR_SEG.
#include "lrdm_internal.h"

#include <math.h>
#include <string.h>

#include <atomic>

namespace lrdm {
namespace {

// values per block: K(K+1)/2 Gram entries (upper, row-major), K RHS, 1 ||R||^2
// (FP64-rate bound: FP64 data, and short FP32 data, see LS_N32)
template <typename T>
__global__ void __launch_bounds__(256) k_gram(const T* __restrict__ F, const T* __restrict__ R, int K,
                                              long long n, double* __restrict__ partial) {
  __shared__ double Fs[KMAX_LIMIT][LS_CHUNK];
  __shared__ double Rs[LS_CHUNK];
  const int npair = K * (K + 1) / 2;
  const int nval = npair + K + 1;
  double acc[9];
#pragma unroll
  for (int t = 0; t < 9; ++t) acc[t] = 0.0;
  for (long long base = (long long)blockIdx.x * LS_CHUNK; base < n;
       base += (long long)gridDim.x * LS_CHUNK) {
    for (int e = threadIdx.x; e < (K + 1) * LS_CHUNK; e += blockDim.x) {
      int k = e / LS_CHUNK, c = e % LS_CHUNK;
      long long r = base + c;
      double x = 0.0;
      if (r < n) x = (double)(k < K ? F[(long long)k * n + r] : R[r]);
      if (k < K) Fs[k][c] = x;
      else Rs[c] = x;
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      int idx = threadIdx.x + t * blockDim.x;
      if (idx < nval) {
        const double* x;
        const double* y;
        if (idx < npair) {
          // row-major upper triangle enumeration: idx -> (k, l), k <= l
          int k = 0, rem = idx;
          while (rem >= K - k) { rem -= K - k; ++k; }
          x = Fs[k];
          y = Fs[k + rem];
        } else if (idx < npair + K) {
          x = Fs[idx - npair];
          y = Rs;
        } else {
          x = Rs;
          y = Rs;
        }
        double s = 0.0;
        for (int c = 0; c < LS_CHUNK; ++c) s += x[c] * y[c];
        acc[t] += s;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int t = 0; t < 9; ++t) {
    int idx = threadIdx.x + t * blockDim.x;
    if (idx < nval) partial[(long long)blockIdx.x * nval + idx] = acc[t];
  }
}

// FP32 data of fewer points is summed in FP64: an FP32 pair's rounding
// (2^-48) averages out over the lanes' sums only when there are many.  Relative
// error of the coefficients against extended precision, pairs / FP64: n =
// 4,097, K = 1: 8e-16 / 2e-16; 32,768, K = 1 with data falling off by e^-40:
// 1.9e-15 / 5e-16; 70,000, K = 16: 4e-16 / 4e-16; 884,736, K = 16: 3e-16 / 3e-16
// (all with the elimination; 2e-15 with the Jacobi rotations).
constexpr long long LS_N32 = 65536;

// a += x . y over four points.  The four products are summed first and the
// rounding errors of products and of sums kept apart until the end: a square's
// error word ends in fixed bits (x^2 = 1 mod 8), and dropping them one product
// at a time against the growing sum biased <f, f> by 6e-15 (now 3e-16; FP64
// sums: 1e-16 to 7e-16).  The pair leaves renormalised: over 128 steps of constant
// data the error of a lane's sum was 2e-12 without (above the default cutoff of
// the pseudo-inverse), 7e-14 with it.
__device__ __forceinline__ void dot4(Pair32& a, const float (&x)[4], const float (&y)[4]) {
  float p[4], e[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    p[u] = __fmul_rn(x[u], y[u]);
    e[u] = __fmaf_rn(x[u], y[u], -p[u]);
  }
  float s01, r01, s23, r23, s, r, t;
  two_sum(p[0], p[1], s01, r01);
  two_sum(p[2], p[3], s23, r23);
  two_sum(s01, s23, s, r);
  float S;
  two_sum(a.s, s, S, t);
  const float es = __fadd_rn(__fadd_rn(e[0], e[1]), __fadd_rn(e[2], e[3]));
  const float rs = __fadd_rn(__fadd_rn(r01, r23), __fadd_rn(r, t));
  const float lo = __fadd_rn(a.c, __fadd_rn(es, rs));
  a.s = __fadd_rn(S, lo);
  a.c = __fsub_rn(lo, __fsub_rn(a.s, S));
}

// Gram sums of FP32 data.  The K + 1 vectors (f_0 .. f_{K-1}, R) are taken in
// groups of four; a task is one pair of groups.  A warp runs the tasks of its
// bin one after the other, each over its share of the grid points with up to
// 16 compensated sums per lane in registers, 128 points a step read straight
// from global memory (the block's other warps find them in L1).  The host
// deals the tasks over 1, 2, 4 or 8 bins by their products (gram_plan); the
// block's eight warps are that many bins times slices of the points.  Bound by
// FP32 issue (eleven operations a product).  At 96^3, K = 16: 89 us (54 us of
// issue; 85 us without the renormalisation), against 378 us with one FP64 fma a
// product.  Two blocks an SM at 128 registers, 28 bytes of them spilled.
//
// FP32 range: the sums stay finite while the values of a warp's range stay below
// 2^56 (256 products a lane, 32 lanes: below 2^125), and a product's error word
// is exact while their largest is not below 2^-48 (its products' last bits then
// stay above 2^-149; smaller values in the range lose less than 2^-53 of the
// sum).  A warp whose range breaks this (or holds an infinity) repeats its range
// in FP64.
constexpr int GR_WARPS = 8;
constexpr int GR_RED = 160;                             // sums of 16 a block holds in shared memory
constexpr int GR_TASKS = 153;                           // K = 64: 17 groups
// Steps a lane sums in FP32 pairs (256 points) before its sums go to FP64.  Relative
// error of a lane's sum of positive products over 64 steps, largest of 400 draws:
// random data 3e-14, data constant over the grid 5e-14 (6e-14 where lanes differ);
// a warp's sums of random data are good to 1e-14 and average out over the warps
// (884,736 points: 3e-16).  Sending them to FP64 costs four steps.
constexpr int GR_SEG = 64;
constexpr float GR_MAX = 7.2057594037927936e16f;        // 2^56
constexpr float GR_MIN = 3.552713678800501e-15f;        // 2^-48

struct GramPlan {
  int bins;                                             // 1, 2, 4 or 8
  int tasks;
  short off[GR_WARPS + 1];                              // tasks off[b] .. off[b + 1] of bin b
  unsigned char A[GR_TASKS], B[GR_TASKS];
};

// index of entry (k, l), k <= l <= K, in a block's values: Gram upper triangle
// row-major, then the right-hand sides, then <R, R>
__device__ __forceinline__ int gr_index(int k, int l, int K) {
  if (k == K) return K * (K + 1) / 2 + K;
  if (l == K) return K * (K + 1) / 2 + k;
  return k * K - k * (k - 1) / 2 + (l - k);
}

// Points of one lane in the step at `base`: four consecutive (vector loads) or
// every 32nd; zero past the end.
__device__ __forceinline__ void gr_load(const float* __restrict__ p, long long base, long long n,
                                        int lane, bool vec, float (&x)[4]) {
  if (vec) {
    const long long r = base + 4 * lane;
    if (r < n) {                        // n is a multiple of 4
      const float4 t = __ldg(reinterpret_cast<const float4*>(p + r));
      x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
    } else {
      x[0] = x[1] = x[2] = x[3] = 0.f;
    }
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long r = base + lane + 32 * u;
      x[u] = r < n ? __ldg(p + r) : 0.f;
    }
  }
}

__device__ __forceinline__ float max4(float m, const float (&x)[4]) {
  return fmaxf(fmaxf(m, fmaxf(fabsf(x[0]), fabsf(x[1]))), fmaxf(fabsf(x[2]), fabsf(x[3])));
}

// One task: group A (NA vectors) against group B (NB); DIAG: A = B, upper part.
// out[4 i + j] = the sum for (A_i, B_j) over the warp's points, by lane 0.
template <int NA, int NB, bool DIAG>
__device__ __forceinline__ void gr_task(const float* __restrict__ F, const float* __restrict__ R,
                                        int A, int B, int K, long long n, long long first,
                                        long long step, int lane, bool vec, double* out) {
  auto vecp = [&](int v) { return v < K ? F + (long long)v * n : R; };
  bool fresh = true;
  long long seg = first, lim;
  do {
    lim = min(n, seg + step * GR_SEG);
    Pair32 acc[NA][NB];
    float ma[NA], mb[NB];
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      ma[i] = 0.f;
#pragma unroll
      for (int j = 0; j < NB; ++j) acc[i][j] = Pair32{0.f, 0.f};
    }
#pragma unroll
    for (int j = 0; j < NB; ++j) mb[j] = 0.f;
    for (long long base = seg; base < lim; base += step) {
      float x[NA][4];
#pragma unroll
      for (int i = 0; i < NA; ++i) gr_load(vecp(4 * A + i), base, n, lane, vec, x[i]);
#pragma unroll
      for (int i = 0; i < NA; ++i) ma[i] = max4(ma[i], x[i]);
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        if (DIAG) {
#pragma unroll
          for (int i = 0; i <= j; ++i) dot4(acc[i][j], x[i], x[j]);
        } else {
          float y[4];
          gr_load(vecp(4 * B + j), base, n, lane, vec, y);
          mb[j] = max4(mb[j], y);
#pragma unroll
          for (int i = 0; i < NA; ++i) dot4(acc[i][j], x[i], y);
        }
      }
    }
    // range of the data this warp has summed (NaN: the sums are NaN already)
    bool wide = false;
    auto range = [&](float m) {
      const float r = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
      wide = wide || r > GR_MAX || (r != 0.f && r < GR_MIN);
    };
#pragma unroll
    for (int i = 0; i < NA; ++i) range(ma[i]);
    if (!DIAG) {
#pragma unroll
      for (int j = 0; j < NB; ++j) range(mb[j]);
    }
    if (!wide) {
#pragma unroll
      for (int i = 0; i < NA; ++i)
#pragma unroll
        for (int j = DIAG ? i : 0; j < NB; ++j) {
          const Pair32 a = pair_warp_sum(acc[i][j]);
          if (lane == 0) out[4 * i + j] = (fresh ? 0.0 : out[4 * i + j]) + ((double)a.s + (double)a.c);
        }
    } else {
#pragma unroll 1
      for (int i = 0; i < NA; ++i)
#pragma unroll 1
        for (int j = DIAG ? i : 0; j < NB; ++j) {
          double t = 0.0;
          for (long long base = seg; base < lim; base += step) {
            float x[4], y[4];
            gr_load(vecp(4 * A + i), base, n, lane, vec, x);
            gr_load(vecp(4 * B + j), base, n, lane, vec, y);
#pragma unroll
            for (int u = 0; u < 4; ++u) t += (double)x[u] * (double)y[u];
          }
          for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
          if (lane == 0) out[4 * i + j] = (fresh ? 0.0 : out[4 * i + j]) + t;
        }
    }
    fresh = false;
    seg += step * GR_SEG;
  } while (seg < n);
}

__global__ void __launch_bounds__(32 * GR_WARPS, 2)
    k_gram32(const __grid_constant__ GramPlan P, const float* __restrict__ F,
             const float* __restrict__ R, int K, long long n, int vec, double* __restrict__ partial) {
  __shared__ double red[GR_RED][16];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bin = warp % P.bins, slice = warp / P.bins, slices = GR_WARPS / P.bins;
  const long long first = 128LL * ((long long)blockIdx.x * slices + slice);
  const long long step = 128LL * gridDim.x * slices;
  for (int t = P.off[bin]; t < P.off[bin + 1]; ++t) {
    const int A = P.A[t], B = P.B[t];
    const int nb = min(4, K + 1 - 4 * B);
    double* out = red[slice * P.tasks + t];
    if (A == B) {
      if (nb == 4) gr_task<4, 4, true>(F, R, A, B, K, n, first, step, lane, vec, out);
      else if (nb == 3) gr_task<3, 3, true>(F, R, A, B, K, n, first, step, lane, vec, out);
      else if (nb == 2) gr_task<2, 2, true>(F, R, A, B, K, n, first, step, lane, vec, out);
      else gr_task<1, 1, true>(F, R, A, B, K, n, first, step, lane, vec, out);
    } else {
      if (nb == 4) gr_task<4, 4, false>(F, R, A, B, K, n, first, step, lane, vec, out);
      else if (nb == 3) gr_task<4, 3, false>(F, R, A, B, K, n, first, step, lane, vec, out);
      else if (nb == 2) gr_task<4, 2, false>(F, R, A, B, K, n, first, step, lane, vec, out);
      else gr_task<4, 1, false>(F, R, A, B, K, n, first, step, lane, vec, out);
    }
  }
  __syncthreads();
  // the slices of each task in order
  const int nval = K * (K + 1) / 2 + K + 1;
  for (int e = threadIdx.x; e < 16 * P.tasks; e += blockDim.x) {
    const int t = e >> 4, q = e & 15;
    const int k = 4 * P.A[t] + (q >> 2), l = 4 * P.B[t] + (q & 3);
    if (k <= l && l <= K) {
      double s = red[t][q];
      for (int u = 1; u < slices; ++u) s += red[u * P.tasks + t][q];
      partial[(long long)blockIdx.x * nval + gr_index(k, l, K)] = s;
    }
  }
}

// One warp per value: the sum of its per-block partials times w, in a fixed
// order.  (One block adding them inside the solve is bound by its SM's FP64
// rate: 46,512 additions at K = 16, 12 us.)
__global__ void __launch_bounds__(128) k_ls_sum(const double* __restrict__ partial, int nblk, int nval,
                                                double w, double* __restrict__ sums) {
  const int v = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (v >= nval) return;
  double s = 0.0;
#pragma unroll 4
  for (int b = lane; b < nblk; b += 32) s += partial[(long long)b * nval + v];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) sums[v] = w * s;
}

// One block of LS_SOLVE_THREADS threads: a = S^+ c.
//
// First by elimination on [S | I | c] without pivoting: S = L D L^T, the rows
// of the identity become L^-1, so tr S^-1 = sum_ik (L^-1)_ik^2 / d_i comes with
// the solution.  lambda_min >= 1 / tr S^-1 and lambda_max <= tr S, so
// tr S tr S^-1 < 1 / rcond certifies that no eigenvalue falls below the
// cutoff and a = S^-1 c = L^-T D^-1 L^-1 c is the answer; LS_CERT keeps the
// certificate itself (relative error about 1e-16 tr S tr S^-1) and the
// elimination's accuracy clear of FP64's limits.  Everything else (a
// non-positive pivot, a matrix near the cutoff) goes to the Jacobi rotations.
// A serial chain of K - 1 divisions: K = 16 17 us, against 308 us (Jacobi), and
// ten times closer to extended precision.
constexpr double LS_CERT = 1e10;
constexpr int LS_SOLVE_THREADS = 256;

__global__ void __launch_bounds__(LS_SOLVE_THREADS, 1) k_ls_solve(const double* __restrict__ sums,
                                                         int K, double rcond,
                                                         double* __restrict__ coef,
                                                         double* __restrict__ coeff_out,
                                                         double* __restrict__ scal,
                                                         int* __restrict__ status) {
  // dynamic shared memory: A(K, K+1), Q(K, K+1) (FP64)
  extern __shared__ double dyn[];
  const int ldk = K + 1;
  double* Abuf = dyn;
  double* Qbuf = dyn + (size_t)K * ldk;
#define A(i, j) Abuf[(i) * ldk + (j)]
#define Q(i, j) Qbuf[(i) * ldk + (j)]
  __shared__ double c[KMAX_LIMIT];
  __shared__ double lam[KMAX_LIMIT];
  __shared__ int bad, easy;
  const int npair = K * (K + 1) / 2;
  const int t = threadIdx.x;
  if (t == 0) { bad = 0; easy = 1; }
  __syncthreads();
  auto load = [&] {                      // S and c; Q = I
    for (int e = t; e < K * K; e += blockDim.x) {
      const int i = e / K, j = e - i * K;
      const int k = min(i, j), l = max(i, j);
      const double x = sums[k * K - k * (k - 1) / 2 + (l - k)];
      A(i, j) = x;
      Q(i, j) = i == j ? 1.0 : 0.0;
      if (!isfinite(x)) bad = 1;
    }
    for (int i = t; i < K; i += blockDim.x) {
      const double x = sums[npair + i];
      c[i] = x;
      if (!isfinite(x)) bad = 1;
    }
  };
  load();
  const double r2s = sums[npair + K];
  __syncthreads();
  if (bad) {
    if (t == 0) atomicOr(status, STATUS_NONFINITE);
    if (t < K) { coef[t] = 0.0; if (coeff_out) coeff_out[t] = 0.0; }
    if (t == 0) { scal[0] = r2s; }
    return;
  }
  {
    // row i after step j: A(i, k) (k > j) the trailing matrix, Q(i, k) (k <= j)
    // the rows of L^-1, lam[j] = 1 / d_j (0 for a pivot that is not positive)
    __shared__ double y0[KMAX_LIMIT];
    __shared__ double red_s[LS_SOLVE_THREADS / 32], red_i[LS_SOLVE_THREADS / 32];
    double tr = 0.0;                     // tr S, by warp 0
    if (t < 32) {
      for (int i = t; i < K; i += 32) tr += A(i, i);
      for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
      if (t == 0) lam[0] = A(0, 0) > 0.0 ? 1.0 / A(0, 0) : 0.0;
    }
    for (int i = t; i < K; i += blockDim.x) y0[i] = c[i];
    __syncthreads();
    for (int j = 0; j < K - 1; ++j) {
      const double inv = lam[j];
      // a warp takes whole rows i > j: lane q the columns k > j of A, k <= j of
      // L^-1 and y; warp 0 row j + 1 alone, whose pivot's division the next
      // step waits for
      const int w = t >> 5, nw = LS_SOLVE_THREADS / 32;
      for (int i = j + 1 + w; i < K; i += w == 0 ? K : nw - 1) {
        const double m = A(i, j) * inv;
        for (int q = t & 31; q <= K; q += 32) {
          const int k = j + 1 + q;       // A(j, k) = A(k, j): the strict upper part is kept too
          if (k < K) {
            const double x = A(i, k) - m * A(j, k);
            A(i, k) = x;
            if (i == j + 1 && k == j + 1) lam[i] = x > 0.0 ? 1.0 / x : 0.0;
          } else if (q < K) {
            Q(i, k - K) -= m * Q(j, k - K);            // 0 .. j
          } else {
            y0[i] -= m * y0[j];
          }
        }
      }
      __syncthreads();
    }
    // tr S^-1 and a = L^-T (D^-1 y)
    double ti = 0.0;
    for (int e = t; e < K * K; e += blockDim.x) {
      const int i = e / K, k = e - i * K;
      if (k <= i) ti += Q(i, k) * Q(i, k) * lam[i];
    }
    for (int o = 16; o > 0; o >>= 1) ti += __shfl_xor_sync(0xffffffffu, ti, o);
    if ((t & 31) == 0) red_i[t >> 5] = ti;
    if (t < K && !(lam[t] > 0.0)) easy = 0;
    if (t == 0) red_s[0] = tr;
    __syncthreads();
    double tinv = 0.0;
    for (int i = 0; i < LS_SOLVE_THREADS / 32; ++i) tinv += red_i[i];
    const double cond = red_s[0] * tinv;
    if (easy && cond < LS_CERT && cond * rcond < 0.5) {
      if (t < K) {
        double x = 0.0;
        for (int i = t; i < K; ++i) x += Q(i, t) * (lam[i] * y0[i]);
        coef[t] = x;
        if (coeff_out) coeff_out[t] = x;
      }
      if (t == 0) scal[0] = r2s;
      return;
    }
    __syncthreads();
    load();
    __syncthreads();
  }
  // Parallel cyclic Jacobi sweeps (round-robin ordering): a sweep is n - 1
  // rounds (n = K rounded up to even; index K is a dummy when K is odd); a
  // round rotates the n / 2 disjoint pairs (p, q) at once, A <- J^T A J and
  // Q <- Q J, so every pair is rotated once per sweep.
  __shared__ double rc[KMAX_LIMIT / 2], rs[KMAX_LIMIT / 2], rt[KMAX_LIMIT / 2];
  __shared__ double rpq[KMAX_LIMIT / 2], rpp[KMAX_LIMIT / 2], rqq[KMAX_LIMIT / 2];
  __shared__ int rp[KMAX_LIMIT / 2], rq[KMAX_LIMIT / 2];
  __shared__ double red_o[LS_SOLVE_THREADS / 32], red_d[LS_SOLVE_THREADS / 32];
  const int n_rr = K + (K & 1);
  const int nrot = n_rr / 2;
  for (int sweep = 0; sweep < 40; ++sweep) {
    // off-diagonal and diagonal Frobenius sums, fixed reduction order
    double o = 0.0, d = 0.0;
    if (t < K)
      for (int j = 0; j < K; ++j) {
        const double x = A(t, j);
        if (j == t) d += x * x;
        else o += x * x;
      }
    for (int s = 16; s > 0; s >>= 1) {
      o += __shfl_xor_sync(0xffffffffu, o, s);
      d += __shfl_xor_sync(0xffffffffu, d, s);
    }
    if ((t & 31) == 0) { red_o[t >> 5] = o; red_d[t >> 5] = d; }
    __syncthreads();
    o = 0.0;
    d = 0.0;
    for (int wi = 0; wi < (int)(blockDim.x >> 5); ++wi) { o += red_o[wi]; d += red_d[wi]; }
    if (!(o > 1e-30 * d) || o == 0.0) break;
    for (int r = 0; r < n_rr - 1; ++r) {
      // the rotation of pair m (thread m)
      if (t < nrot) {
        int p, q;
        if (t == 0) { p = r; q = n_rr - 1; }
        else { p = (r + t) % (n_rr - 1); q = (r - t + n_rr - 1) % (n_rr - 1); }
        if (p > q) { const int x = p; p = q; q = x; }
        double cs = 1.0, sn = 0.0, tt = 0.0, apq = 0.0, app = 0.0, aqq = 0.0;
        if (q < K) {
          apq = A(p, q);
          app = A(p, p);
          aqq = A(q, q);
          if (apq != 0.0 && fabs(apq) >= 1e-300) {
            const double tau = (aqq - app) / (2.0 * apq);
            tt = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
            cs = 1.0 / sqrt(1.0 + tt * tt);
            sn = tt * cs;
          }
        }
        rp[t] = p; rq[t] = q; rc[t] = cs; rs[t] = sn; rt[t] = tt;
        rpq[t] = apq; rpp[t] = app; rqq[t] = aqq;
      }
      __syncthreads();
      // columns: B = A J, Q <- Q J, one (row, pair) task per thread (each
      // task owns the entries (i, p) and (i, q): no two tasks share one)
      for (int task = t; task < K * nrot; task += blockDim.x) {
        const int i = task % K, m = task / K;
        const int p = rp[m], q = rq[m];
        if (q >= K || rt[m] == 0.0) continue;
        const double c = rc[m], s = rs[m];
        const double ap = A(i, p), aq = A(i, q);
        A(i, p) = c * ap - s * aq;
        A(i, q) = s * ap + c * aq;
        const double qp = Q(i, p), qq = Q(i, q);
        Q(i, p) = c * qp - s * qq;
        Q(i, q) = s * qp + c * qq;
      }
      __syncthreads();
      // rows: A <- J^T B, one (column, pair) task per thread
      for (int task = t; task < K * nrot; task += blockDim.x) {
        const int j = task % K, m = task / K;
        const int p = rp[m], q = rq[m];
        if (q >= K || rt[m] == 0.0) continue;
        const double c = rc[m], s = rs[m];
        const double bp = A(p, j), bq = A(q, j);
        A(p, j) = c * bp - s * bq;
        A(q, j) = s * bp + c * bq;
      }
      __syncthreads();
      // exact symmetry (the lower triangle mirrors the upper) and the closed
      // form of each rotated 2 x 2 block
      if (t < K)
        for (int j = t + 1; j < K; ++j) A(j, t) = A(t, j);
      __syncthreads();
      if (t < nrot && rq[t] < K && rt[t] != 0.0) {
        const int p = rp[t], q = rq[t];
        A(p, p) = rpp[t] - rt[t] * rpq[t];
        A(q, q) = rqq[t] + rt[t] * rpq[t];
        A(p, q) = 0.0;
        A(q, p) = 0.0;
      }
      __syncthreads();
    }
  }
  if (t < K) lam[t] = A(t, t);
  __syncthreads();
  __shared__ double lmax;
  __shared__ int dropped;
  if (t == 0) {
    double m = 0.0;
    for (int i = 0; i < K; ++i) m = fmax(m, lam[i]);
    lmax = m;
    dropped = 0;
  }
  __syncthreads();
  // y = diag(lambda^+) Q^T c
  __shared__ double y[KMAX_LIMIT];
  if (t < K) {
    double s = 0.0;
    for (int i = 0; i < K; ++i) s += Q(i, t) * c[i];
    if (lmax > 0.0 && lam[t] > rcond * lmax) {
      y[t] = s / lam[t];
    } else {
      y[t] = 0.0;
      atomicOr(&dropped, 1);
    }
  }
  __syncthreads();
  if (t < K) {
    double s = 0.0;
    for (int i = 0; i < K; ++i) s += Q(t, i) * y[i];
    coef[t] = s;
    if (coeff_out) coeff_out[t] = s;
  }
  if (t == 0) {
    scal[0] = r2s;
    if (dropped) atomicOr(status, STATUS_SINGULAR);
  }
#undef A
#undef Q
}

// Delta = sum_k a_k v_k; rho <- rho - alpha Delta (alpha != 0) or Delta;
// partial sums of (sum_k a_k f_k - R)^2.  FP64 arithmetic.
template <typename T>
__global__ void __launch_bounds__(256) k_update64(const T* __restrict__ v, const T* __restrict__ f,
                                                  const T* __restrict__ R, int K, long long n,
                                                  double alpha, const double* __restrict__ coef,
                                                  T* __restrict__ rho,
                                                  double* __restrict__ upd_partial) {
  __shared__ double a[KMAX_LIMIT];
  if (threadIdx.x < K) a[threadIdx.x] = coef[threadIdx.x];
  __syncthreads();
  double acc = 0.0;
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < n;
       r += (long long)gridDim.x * blockDim.x) {
    double d = 0.0, fa = 0.0;
    for (int k = 0; k < K; ++k) {
      d += a[k] * (double)v[(long long)k * n + r];
      fa += a[k] * (double)f[(long long)k * n + r];
    }
    const double res = fa - (double)R[r];
    acc += res * res;
    if (rho) rho[r] = (T)(alpha != 0.0 ? (double)rho[r] - alpha * d : d);
  }
  __shared__ double sw[32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += sw[i];
    upd_partial[blockIdx.x] = s;
  }
}

// a += (h + l) x with h + l one coefficient's leading and trailing FP32 words
__device__ __forceinline__ void axpy2(Pair32& a, float h, float l, float x) {
  const float p = __fmul_rn(h, x);
  const float e = __fmaf_rn(l, x, __fmaf_rn(h, x, -p));
  float r;
  two_sum(a.s, p, a.s, r);
  a.c = __fadd_rn(a.c, __fadd_rn(e, r));
}
// The same for FP32 data, in compensated FP32 (2 K fma a point in FP64 bound
// it to the FP64 rate).  Two points a thread, the K loop unrolled for loads in
// flight; what is the same for all threads is made once a block (a division
// and an exponent in FP64 by every thread took 5 us).  The residual is scaled
// by a power of two to the size of ||R|| before it is squared, so the squares
// stay in range; a point whose compensated sums leave the FP32 range (not
// finite) is repeated in FP64.  At 96^3, K = 16 (124 MB to move: 19 us): 25 us,
// against 127 us in FP64 (44 us with the loads in the K loop itself).
constexpr int UPD_COEF = -96;                           // below 2^-96 a factor's second word is not normal
constexpr double UPD_RMS2 = 6.842277657836020854e-49;   // 2^-160: an error word's 2^-149 is 2^-69 of rms(R)
constexpr float UPD_OUT = 1.262177448353618888658765e-29f;                  // 2^-96

// 0 < |x| < 2^e, in integer operations
__host__ __device__ __forceinline__ bool below(double x, int e) {
  uint64_t b;
  memcpy(&b, &x, sizeof(b));
  b <<= 1;
  return b != 0 && b < (uint64_t)(1023 + e) << 53;
}

template <bool RHO>
__global__ void __launch_bounds__(256) k_update32(const float* __restrict__ v,
                                                  const float* __restrict__ f,
                                                  const float* __restrict__ R, int K, long long n,
                                                  double wn, int vec, double alpha, int wide0,
                                                  const double* __restrict__ coef,
                                                  const double* __restrict__ scal,
                                                  float* __restrict__ rho,
                                                  double* __restrict__ upd_partial) {
  constexpr int UB = 4, UPD_NORM = 16;                  // directions a batch, and between renormalisations
  __shared__ float2 a[KMAX_LIMIT + UB];                 // zero past K
  __shared__ int se;
  __shared__ double sw[8];
  bool tiny = wide0 != 0;
  if (threadIdx.x < KMAX_LIMIT + UB) {
    const double c = threadIdx.x < K ? coef[threadIdx.x] : 0.0;
    const Pair32 p = pair_split(c);
    a[threadIdx.x] = make_float2(p.s, p.c);
    tiny = tiny || below(c, UPD_COEF);
  }
  if (threadIdx.x == 128) {
    // 2^e near 1 / rms(R); e = 0 for R = 0 or not finite
    const double ms = scal[0] / wn;
    se = ms > 0.0 && isfinite(ms) ? max(-120, min(120, -ilogb(ms) / 2)) : 0;
    tiny = tiny || (ms > 0.0 && ms < UPD_RMS2);
  }
  const bool wide = __syncthreads_or(tiny);
  const Pair32 al = pair_split(alpha);
  const int e = se;
  const float sc = __int_as_float((127 + e) << 23);
  double acc = 0.0;
  Pair32 sq{0.f, 0.f};
  const long long items = (n + 1) / 2;
  for (long long it = blockIdx.x * (long long)blockDim.x + threadIdx.x; it < items;
       it += (long long)gridDim.x * blockDim.x) {
    const long long r0 = 2 * it;
    const bool two = r0 + 1 < n;
    Pair32 d[2] = {{0.f, 0.f}, {0.f, 0.f}}, fa[2] = {{0.f, 0.f}, {0.f, 0.f}};
    auto norm = [&] {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        pair_norm(fa[u]);
        if (RHO) pair_norm(d[u]);
      }
    };
    if (vec) {
      // batches of UB directions, the next batch's loads in flight during a
      // batch's arithmetic (past K: coefficient 0, the last row again)
      float2 fx[UB], vx[UB];
      auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          const long long o = (long long)min(k0 + u, K - 1) * n + r0;
          fx[u] = __ldg(reinterpret_cast<const float2*>(f + o));
          if (RHO) vx[u] = __ldg(reinterpret_cast<const float2*>(v + o));
        }
      };
      fetch(0);
      for (int k0 = 0; k0 < K; k0 += UB) {
        float2 gx[UB], wx[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          gx[u] = fx[u];
          if (RHO) wx[u] = vx[u];
        }
        if (k0 + UB < K) fetch(k0 + UB);
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          const float2 c = a[k0 + u];
          axpy2(fa[0], c.x, c.y, gx[u].x);
          axpy2(fa[1], c.x, c.y, gx[u].y);
          if (RHO) {
            axpy2(d[0], c.x, c.y, wx[u].x);
            axpy2(d[1], c.x, c.y, wx[u].y);
          }
        }
        if (k0 % UPD_NORM == UPD_NORM - UB) norm();
      }
    } else {
#pragma unroll 4
      for (int k = 0; k < K; ++k) {
        const float2 c = a[k];
        const long long o = (long long)k * n + r0;
        axpy2(fa[0], c.x, c.y, __ldg(f + o));
        axpy2(fa[1], c.x, c.y, two ? __ldg(f + o + 1) : 0.f);
        if (RHO) {
          axpy2(d[0], c.x, c.y, __ldg(v + o));
          axpy2(d[1], c.x, c.y, two ? __ldg(v + o + 1) : 0.f);
        }
        if (k % UPD_NORM == UPD_NORM - 1) norm();
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (u == 1 && !two) break;
      const long long r = r0 + u;
      const float Rr = R[r];
      // res = fa - R as a pair, scaled
      float t, lo;
      two_sum(fa[u].s, -Rr, t, lo);
      lo = __fadd_rn(lo, fa[u].c);
      const float hs = __fadd_rn(t, lo);
      const float hi = __fmul_rn(hs, sc);
      const float rl = __fmul_rn(__fsub_rn(lo, __fsub_rn(hs, t)), sc);
      const float p = __fmul_rn(hi, hi);
      float out = 0.f, old = 0.f;
      if (RHO) {
        old = rho[r];
        if (alpha != 0.0) {
          const float q = __fmul_rn(al.s, d[u].s);
          const float qe = __fmaf_rn(al.c, d[u].s, __fmaf_rn(al.s, d[u].c, __fmaf_rn(al.s, d[u].s, -q)));
          float o, oe;
          two_sum(old, -q, o, oe);
          out = __fadd_rn(o, __fsub_rn(oe, qe));
        } else {
          out = __fadd_rn(d[u].s, d[u].c);
        }
      }
      const bool low = RHO && fabsf(out) < UPD_OUT && d[u].s != 0.f;
      if (!wide && !low && isfinite(p) && isfinite(out)) {
        const float pe = __fmaf_rn(__fadd_rn(hi, hi), rl, __fmaf_rn(hi, hi, -p));
        pair_add(sq, Pair32{p, pe});
        pair_norm(sq);
      } else {
        double dd = 0.0, ff = 0.0;
        for (int k = 0; k < K; ++k) {
          ff += coef[k] * (double)f[(long long)k * n + r];
          if (RHO) dd += coef[k] * (double)v[(long long)k * n + r];
        }
        const double res = ff - (double)Rr;
        acc += res * res;
        out = (float)(alpha != 0.0 ? (double)old - alpha * dd : dd);
      }
      if (RHO) rho[r] = out;
    }
  }
  sq = pair_warp_sum(sq);
  if (__any_sync(0xffffffffu, acc != 0.0))
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = acc + ldexp((double)sq.s + (double)sq.c, -2 * e);
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < 8; ++i) s += sw[i];
    upd_partial[blockIdx.x] = s;
  }
}

__global__ void k_srel(const double* __restrict__ upd_partial, int nblk, double w,
                       const double* __restrict__ scal, double* __restrict__ s_rel_out) {
  __shared__ double sw[32];
  double s = 0.0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += upd_partial[b];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tot += sw[i];
    double r2 = scal[0];
    double val = r2 > 0.0 ? sqrt(w * tot / r2) : 0.0;
    if (s_rel_out) s_rel_out[0] = val;
    // scal layout: [0] = <R, R>, [1] = s_rel
    const_cast<double*>(scal)[1] = val;
  }
}

}  // namespace

namespace {

bool ls_aligned(const void* p, uintptr_t bytes) { return (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0; }

// The tasks of K directions dealt over 1, 2, 4 or 8 bins, largest first to the
// least loaded bin.  More bins leave each warp a longer range of points for
// one reduction over its lanes, fewer balance better: the cheaper of the four
// in FP32 operations of the busiest warp (40 a product and step of 128 points,
// 60 a value for the reduction) is taken.
void gram_plan(int K, long long n, GramPlan& best) {
  const int G = (K + 1 + 3) / 4, T = G * (G + 1) / 2;
  unsigned char A[GR_TASKS], B[GR_TASKS], w[GR_TASKS];
  int t = 0;
  for (int want = 16; want > 0; --want)              // by decreasing number of products
    for (int a = 0; a < G; ++a)
      for (int b = a; b < G; ++b) {
        const int nb = min(4, K + 1 - 4 * b);
        const int x = a == b ? nb * (nb + 1) / 2 : 4 * nb;
        if (x != want) continue;
        A[t] = (unsigned char)a;
        B[t] = (unsigned char)b;
        w[t++] = (unsigned char)x;
      }
  double cost = 1e300;
  for (int bins = 1; bins <= GR_WARPS; bins *= 2) {
    const int slices = GR_WARPS / bins;
    if (slices * T > GR_RED) continue;
    int load[GR_WARPS] = {}, owner[GR_TASKS];
    for (int i = 0; i < T; ++i) {
      int at = 0;
      for (int b = 1; b < bins; ++b)
        if (load[b] < load[at]) at = b;
      owner[i] = at;
      load[at] += w[i];
    }
    int top = 0;
    for (int b = 0; b < bins; ++b) top = max(top, load[b]);
    const long long per = 128LL * LS_BLOCKS * slices;
    const double c = top * (40.0 * (double)((n + per - 1) / per) + 60.0);
    if (c >= cost) continue;
    cost = c;
    best.bins = bins;
    best.tasks = T;
    int m = 0;
    for (int b = 0; b < bins; ++b) {
      best.off[b] = (short)m;
      for (int i = 0; i < T; ++i)
        if (owner[i] == b) {
          best.A[m] = A[i];
          best.B[m++] = B[i];
        }
    }
    best.off[bins] = (short)m;
  }
}

// Per-block Gram sums, LS_BLOCKS blocks of K (K + 1) / 2 + K + 1 values.
cudaError_t gram_launch(const void* f, const void* R, int io_dtype, int K, long long n,
                        double* partial, cudaStream_t st) {
  if (io_dtype == LRDM_DTYPE_F32 && n < LS_N32) {
    k_gram<float><<<LS_BLOCKS, 256, 0, st>>>(static_cast<const float*>(f), static_cast<const float*>(R),
                                             K, n, partial);
  } else if (io_dtype == LRDM_DTYPE_F32) {
    GramPlan P;
    gram_plan(K, n, P);
    const int vec = n % 4 == 0 && ls_aligned(f, 16) && ls_aligned(R, 16);
    k_gram32<<<LS_BLOCKS, 32 * GR_WARPS, 0, st>>>(P, static_cast<const float*>(f),
                                                  static_cast<const float*>(R), K, n, vec, partial);
  } else {
    k_gram<double><<<LS_BLOCKS, 256, 0, st>>>(static_cast<const double*>(f),
                                              static_cast<const double*>(R), K, n, partial);
  }
  return cudaGetLastError();
}

cudaError_t update_launch(const void* v, const void* f, const void* R, int io_dtype, int K,
                          long long n, double w, double alpha, const double* coef,
                          const double* scal, void* rho, double* upd_partial, cudaStream_t st) {
  if (io_dtype == LRDM_DTYPE_F32 && n < LS_N32) {
    k_update64<float><<<UPD_BLOCKS, 256, 0, st>>>(static_cast<const float*>(v), static_cast<const float*>(f),
                                                  static_cast<const float*>(R), K, n, alpha, coef,
                                                  static_cast<float*>(rho), upd_partial);
  } else if (io_dtype == LRDM_DTYPE_F32) {
    const int vec = n % 2 == 0 && ls_aligned(v, 8) && ls_aligned(f, 8);
    auto kern = rho ? k_update32<true> : k_update32<false>;
    kern<<<UPD_BLOCKS, 256, 0, st>>>(static_cast<const float*>(v), static_cast<const float*>(f),
                                     static_cast<const float*>(R), K, n, w * (double)n, vec, alpha,
                                     (int)below(alpha, UPD_COEF), coef, scal, static_cast<float*>(rho), upd_partial);
  } else {
    k_update64<double><<<UPD_BLOCKS, 256, 0, st>>>(static_cast<const double*>(v),
                                                   static_cast<const double*>(f),
                                                   static_cast<const double*>(R), K, n, alpha, coef,
                                                   static_cast<double*>(rho), upd_partial);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_ls(const void* R, const void* v, const void* f, int io_dtype, int K,
                      long long n, double w, double alpha, double rcond, void* rho_inout,
                      double* coef, double* coeff_out, double* s_rel_out, double* partial,
                      double* sums, double* scal, double* upd_partial, int* status, cudaStream_t st,
                      const AllReduce* ar, int* ar_failed) {
  cudaError_t e = gram_launch(f, R, io_dtype, K, n, partial, st);
  if (e != cudaSuccess) return e;
  const int nval = K * (K + 1) / 2 + K + 1;
  // grid-row sharding: each rank's per-block sums, summed over the ranks
  // block by block, so that every rank reduces the same values in the same order
  if (ar && ar->fn && ar->fn(ar->user, partial, (long long)LS_BLOCKS * nval, LRDM_DTYPE_F64, st) != 0) {
    if (ar_failed) *ar_failed = 1;
    return cudaSuccess;
  }
  k_ls_sum<<<(nval + 3) / 4, 128, 0, st>>>(partial, LS_BLOCKS, nval, w, sums);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t smem = 2 * (size_t)K * (K + 1) * sizeof(double);
  // the shared-memory limit is a per-device function attribute: one bit per
  // device ordinal records that it was raised (a racing first call from
  // another host thread sets the same value again)
  static std::atomic<unsigned long long> attr_set{0};
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (!bit || !(attr_set.load(std::memory_order_acquire) & bit)) {
    e = cudaFuncSetAttribute(k_ls_solve, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             2 * KMAX_LIMIT * (KMAX_LIMIT + 1) * (int)sizeof(double));
    if (e != cudaSuccess) return e;
    attr_set.fetch_or(bit, std::memory_order_acq_rel);
  }
  k_ls_solve<<<1, LS_SOLVE_THREADS, smem, st>>>(sums, K, rcond, coef, coeff_out, scal, status);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = update_launch(v, f, R, io_dtype, K, n, w, alpha, coef, scal, rho_inout, upd_partial, st);
  if (e != cudaSuccess) return e;
  if (ar && ar->fn && ar->fn(ar->user, upd_partial, (long long)UPD_BLOCKS, LRDM_DTYPE_F64, st) != 0) {
    if (ar_failed) *ar_failed = 1;
    return cudaSuccess;
  }
  k_srel<<<1, 256, 0, st>>>(upd_partial, UPD_BLOCKS, w, scal, s_rel_out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Allocation-free form of the least-squares step (lrdm_apply_static).
//
// Its scratch -- the per-block partial sums, the coefficients, <R, R> and
// s_rel, the per-block residual sums and the status word -- lives in one
// file-scope device array instead of a context's workspaces, so a call needs
// no lrdm_create and allocates nothing.  The array is sized for at most
// STATIC_K_MAX directions (about 370 KB) and is held by every GPU that loads
// this library until the process exits.  All calls share it: the partial sums
// are fully rewritten by every call and the status word is cleared at its
// start, but two calls that overlap on the GPU (different streams, or several
// host threads) race on it.
// ---------------------------------------------------------------------------

namespace {

constexpr int STATIC_K_MAX = 16;
constexpr int STATIC_NVAL = STATIC_K_MAX * (STATIC_K_MAX + 1) / 2 + STATIC_K_MAX + 1;
constexpr int SC_PARTIAL = 0;                                   // [LS_BLOCKS][STATIC_NVAL]
constexpr int SC_SUMS = SC_PARTIAL + LS_BLOCKS * STATIC_NVAL;   // [STATIC_NVAL]
constexpr int SC_COEF = SC_SUMS + STATIC_NVAL;                  // [STATIC_K_MAX]
constexpr int SC_SCAL = SC_COEF + STATIC_K_MAX;                 // [4]
constexpr int SC_UPD = SC_SCAL + 4;                             // [UPD_BLOCKS]
constexpr int SC_STATUS = SC_UPD + UPD_BLOCKS;                  // one double slot for the int status
constexpr int SC_TOTAL = SC_STATUS + 1;

static __device__ __align__(256) double g_ls_scratch[SC_TOTAL];

constexpr int MAX_DEVICES = 64;
// Device address of g_ls_scratch per device ordinal.  Host threads that race
// on a device's first call each look the address up and store the same value;
// the atomics make that race well defined.  The address belongs to the
// device's primary context: after cudaDeviceReset the process must reload
// the library before calling lrdm_apply_static again.
std::atomic<double*> g_scratch_addr[MAX_DEVICES];

// Device address of g_ls_scratch on the current device (looked up once per
// device with that device current; the host-side symbol is not a device
// address).
cudaError_t static_scratch(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  double* a = g_scratch_addr[dev].load(std::memory_order_acquire);
  if (!a) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_ls_scratch);
    if (e != cudaSuccess) return e;
    a = static_cast<double*>(p);
    g_scratch_addr[dev].store(a, std::memory_order_release);
  }
  *out = a;
  return cudaSuccess;
}

}  // namespace

int static_k_max() { return STATIC_K_MAX; }

cudaError_t launch_ls_static(const void* R, const void* v, const void* f, int io_dtype, int K,
                             long long n, double w, double alpha, double rcond, void* rho_inout,
                             double* coeff_out, double* s_rel_out, int* status_out,
                             cudaStream_t st) {
  double* sc = nullptr;
  cudaError_t e = static_scratch(&sc);
  if (e != cudaSuccess) return e;
  int* status = reinterpret_cast<int*>(sc + SC_STATUS);
  e = cudaMemsetAsync(status, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  double* partial = sc + SC_PARTIAL;
  double* coef = sc + SC_COEF;
  double* scal = sc + SC_SCAL;
  double* upd = sc + SC_UPD;
  if ((e = gram_launch(f, R, io_dtype, K, n, partial, st)) != cudaSuccess) return e;
  const int nval = K * (K + 1) / 2 + K + 1;
  k_ls_sum<<<(nval + 3) / 4, 128, 0, st>>>(partial, LS_BLOCKS, nval, w, sc + SC_SUMS);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t smem = 2 * (size_t)K * (K + 1) * sizeof(double);   // <= 4352 bytes for K <= 16
  k_ls_solve<<<1, LS_SOLVE_THREADS, smem, st>>>(sc + SC_SUMS, K, rcond, coef, coeff_out, scal, status);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = update_launch(v, f, R, io_dtype, K, n, w, alpha, coef, scal, rho_inout, upd, st);
  if (e != cudaSuccess) return e;
  k_srel<<<1, 256, 0, st>>>(upd, UPD_BLOCKS, w, scal, s_rel_out);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (status_out)
    e = cudaMemcpyAsync(status_out, status, sizeof(int), cudaMemcpyDeviceToDevice, st);
  return e;
}

}  // namespace lrdm
