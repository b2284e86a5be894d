// Kernels of the Brillouin-zone-sampled response (§II.C, closing paragraphs;
// Eq. tracelessCondition) around the two contractions.  Every precision runs
// the real contractions on the stacked operand C = [A B] (N_g x 2 N_s) of
// psi = A + i B: P = C^T diag(a) C holds Re X = P11 + P22 and Im X = P12 - P21
// of X = Psi^H diag(a) Psi, and the density diag(Psi Gamma Psi^H) equals
// diag(C M C^T) with the symmetric M = [[Re G, Im G], [-Im G, Re G]],
// G = Gamma = L o (X - mu' I).  The upper triangle of a 2 N_s-wide real product
// costs what the Hermitian half of the complex one does (4 N_g N_s^2 flops).
//   mu'_k = sum_kappa w_kappa sum_i L_ii Re X_ii / sum_kappa w_kappa sum_i L_ii;
//   drho_k(r) = g sum_kappa w_kappa diag(C M C^T), accumulated over k-points in
//   FP64.
#include <cuda_bf16.h>

#include "lrdm_internal.h"

namespace lrdm {
namespace {

// mu'_k over all k-points: one block per direction over all (point, state)
// pairs, FP64 sums by as many threads as in trace_sums (k_elem.cu; 48^3, 4
// points of 512: 12 us, 256 or 1024 threads 13 and 15), the states one after the
// other.
template <typename T>
constexpr int KP_DMU_THREADS = sizeof(T) == 8 ? 256 : 512;
template <typename T>
__global__ void __launch_bounds__(KP_DMU_THREADS<T>)
    k_kp_dmu(const __grid_constant__ KpDmuArgs A, double* __restrict__ dmu, double* __restrict__ dmu_out) {
  constexpr int W = KP_DMU_THREADS<T> / 32;
  __shared__ double sn[W], sd[W];
  const int k = blockIdx.x;
  const long long mat = (long long)A.ld * A.ld;
  double num = 0.0, den = 0.0;
#pragma unroll 1
  for (int e = threadIdx.x; e < A.nk * A.ns; e += blockDim.x) {
    const int kp = e / A.ns, i = e - kp * A.ns;
    const double l = A.kw[kp] * A.L[kp][(long long)i * A.ns + i];
    const T* P = static_cast<const T*>(A.P[kp]) + k * mat + (long long)i * A.ld + i;
    num += l * (sum_strided(P, A.nsplit, A.K * mat) +
                sum_strided(P + (long long)A.ns * A.ld + A.ns, A.nsplit, A.K * mat));
    den += l;
  }
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, o);
    den += __shfl_xor_sync(0xffffffffu, den, o);
  }
  if ((threadIdx.x & 31) == 0) {
    sn[threadIdx.x >> 5] = num;
    sd[threadIdx.x >> 5] = den;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    num = den = 0.0;
    for (int w = 0; w < W; ++w) {
      num += sn[w];
      den += sd[w];
    }
    const double v = den != 0.0 ? num / den : 0.0;
    dmu[k] = v;
    if (dmu_out) dmu_out[k] = v;
  }
}

// M'' at [k][i][j] for i <= j < 2 ns: c_ij M_ij with c = 2 off the diagonal (below
// it the buffer keeps the zeros it was created with), summed over the row ranges.  P and L
// are symmetric, so every read takes the entry whose column follows j.
template <typename Tc>
__global__ void k_kp_scale(const Tc* __restrict__ P, int nsplit, int K, int k0, int ns,
                           const double* __restrict__ L, const double* __restrict__ dmu,
                           Tc* __restrict__ Y) {
  const int n2 = 2 * ns;
  const int j = blockIdx.y * blockDim.x + threadIdx.x;
  const int i = blockIdx.x, k = blockIdx.z;            // rows in x: a grid's y ends at 65,535
  if (j >= n2 || i > j) return;
  const long long mat = (long long)n2 * n2, tot = (long long)K * mat;
  const Tc* Pk = P + (long long)(k0 + k) * mat;
  auto at = [&](int r, int c) { return sum_strided(Pk + (long long)r * n2 + c, nsplit, tot); };
  const int a = i < ns ? i : i - ns, b = j < ns ? j : j - ns;
  const double l = L[(long long)a * ns + b];
  double m;
  if ((i < ns) == (j < ns)) m = l * (at(a, b) + at(ns + a, ns + b) - (a == b ? dmu[k0 + k] : 0.0));
  else m = l * (at(a, ns + b) - at(ns + a, b));          // Im X_ab = P12 - P21
  Y[(long long)k * mat + (long long)i * n2 + j] = (Tc)(i < j ? 2.0 * m : m);
}

// f = drho - v in the io dtype
__global__ void k_kp_finish(const double* __restrict__ drho, const void* __restrict__ v, int io,
                            long long n, void* __restrict__ f) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    if (io == LRDM_DTYPE_F64)
      static_cast<double*>(f)[e] = drho[e] - static_cast<const double*>(v)[e];
    else
      static_cast<float*>(f)[e] = (float)(drho[e] - (double)static_cast<const float*>(v)[e]);
  }
}

// rho = (first ? floor : rho) + g w sum_i f_i (A_i^2 + B_i^2), one warp per grid
// point; A, B rows of leading dimension ld
template <typename Tc>
__global__ void k_kp_density(const Tc* __restrict__ pr, const Tc* __restrict__ pi, int ns, int ld,
                             long long Ng, const double* __restrict__ occ, double gw, int first,
                             double floor, double* __restrict__ rho) {
  const int lane = threadIdx.x & 31;
  const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long r = warp; r < Ng; r += nwarps) {
    double acc = 0.0;
    for (int i = lane; i < ns; i += 32) {
      const double a = pr[r * ld + i], b = pi[r * ld + i];
      acc += occ[i] * (a * a + b * b);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) rho[r] = (first ? floor : rho[r]) + gw * acc;
  }
}

// one plane of the caller's Psi (io dtype, leading dimension ld) into the
// compute type, [N_g][N_s]
template <typename Tc>
__global__ void k_kp_copy(const void* __restrict__ src, int io, int ld, long long Ng, int ns,
                          Tc* __restrict__ dst, int ldd, int col0) {
  const long long tot = Ng * ns;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
       e += (long long)gridDim.x * blockDim.x) {
    const long long r = e / ns;
    const int i = (int)(e - r * ns);
    const double x = io == LRDM_DTYPE_F64 ? static_cast<const double*>(src)[r * ld + i]
                                          : (double)static_cast<const float*>(src)[r * ld + i];
    dst[r * ldd + col0 + i] = (Tc)x;
  }
}

// M'' at [k][j][i] (i fastest) for i <= j < 2 ns: c_ij M_ij with c = 2 off the
// diagonal; zero elsewhere (padding included).  One thread per four columns of
// a row, looping over the directions so that L is read and split into an FP32
// pair once; P (both triangles written by GEMM1) and L are symmetric, so every
// read takes the entry whose column follows i.  Sums and products as FP32
// pairs (about 2^-47; the stored operand keeps 16 bits): in FP64, five
// operations an entry, the kernel was bound by the FP64 pipe: 48^3, 512
// complex states, K = 8: 187 us a point, now 62 (59 MB to move).
__global__ void __launch_bounds__(128) k_kp_scale_tc(const float* __restrict__ P, int nsplit, int K, int ns,
                                                     int ld, const double* __restrict__ L,
                                                     const double* __restrict__ dmu, int layout,
                                                     void* __restrict__ out, __nv_bfloat16* __restrict__ out_lo) {
  const int c0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  const int j = blockIdx.y;
  if (c0 >= ld) return;
  const long long mat = (long long)ld * ld, tot = (long long)K * mat;
  const int n2 = 2 * ns;
  const int b = j < ns ? j : j - ns;
  // per column: the two entries of P that make it (r1 + sg r2), L as a pair
  // (0 where the entry is zero), the diagonal's FP64 L
  Pair32 l[4];
  long long o1[4], o2[4];
  float sg[4];
  double ld64 = 0.0;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int i = c0 + e;
    const int a = i < ns ? i : i - ns;
    l[e] = Pair32{0.f, 0.f};
    o1[e] = o2[e] = 0;
    sg[e] = 1.f;
    if (i > j || j >= n2) continue;
    const double x = L[(long long)b * ns + a];
    const double c = i < j ? 2.0 * x : x;
    l[e].s = (float)c;
    l[e].c = (float)(c - (double)l[e].s);
    if (i == j) ld64 = x;
    if ((i < ns) == (j < ns)) {              // diagonal blocks: Re Gamma_ab = L_ab (P11 + P22 - mu')
      o1[e] = (long long)b * ld + a;
      o2[e] = (long long)(ns + b) * ld + ns + a;
    } else {                                 // i in block 0, j in block 1: Im Gamma_ab = L_ab (P12 - P21)
      o1[e] = (long long)(ns + b) * ld + a;
      o2[e] = (long long)b * ld + ns + a;
      sg[e] = -1.f;
    }
  }
  const bool any = c0 <= j && j < n2;
  // all four columns on or above the diagonal, in one block of columns:
  // 16-byte loads of both entries (ld is a multiple of 4)
  const bool quad = c0 + 3 <= j && j < n2 && ns % 4 == 0;
#pragma unroll 2
  for (int k = 0; k < K; ++k) {
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (any) {
      const float* Pk = P + (long long)k * mat;
      Pair32 xs[4];
      for (int p = 0; p < nsplit; ++p) {
        float y1[4], y2[4];
        if (quad) {
          *reinterpret_cast<float4*>(y1) = *reinterpret_cast<const float4*>(Pk + p * tot + o1[0]);
          *reinterpret_cast<float4*>(y2) = *reinterpret_cast<const float4*>(Pk + p * tot + o2[0]);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            y1[e] = Pk[p * tot + o1[e]];
            y2[e] = Pk[p * tot + o2[e]];
          }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (p == 0) xs[e] = Pair32{y1[e], 0.f};
          else pair_add(xs[e], Pair32{y1[e], 0.f});
          pair_add(xs[e], Pair32{sg[e] * y2[e], 0.f});
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (c0 + e > j) continue;
        const Pair32 x = xs[e];
        if (c0 + e == j) {
          v[e] = (float)(ld64 * (pair_value(x) - (j < n2 ? dmu[k] : 0.0)));
        } else {
          const float q = __fmul_rn(l[e].s, x.s);
          const float qe = __fmaf_rn(l[e].c, x.s, __fmaf_rn(l[e].s, x.c, __fmaf_rn(l[e].s, x.s, -q)));
          v[e] = pair_round(Pair32{q, qe});
        }
      }
    }
    const long long o = ((long long)k * ld + j) * ld + c0;
    if (layout == 1) {
      float4 t;
      t.x = tf32_rna(v[0]);
      t.y = tf32_rna(v[1]);
      t.z = tf32_rna(v[2]);
      t.w = tf32_rna(v[3]);
      *reinterpret_cast<float4*>(static_cast<float*>(out) + o) = t;
    } else {
      const __nv_bfloat162 h01 = __floats2bfloat162_rn(v[0], v[1]);
      const __nv_bfloat162 h23 = __floats2bfloat162_rn(v[2], v[3]);
      const float2 f01 = __bfloat1622float2(h01), f23 = __bfloat1622float2(h23);
      const __nv_bfloat162 l01 = __floats2bfloat162_rn(v[0] - f01.x, v[1] - f01.y);
      const __nv_bfloat162 l23 = __floats2bfloat162_rn(v[2] - f23.x, v[3] - f23.y);
      uint2 hw, lw;
      hw.x = *reinterpret_cast<const uint32_t*>(&h01);
      hw.y = *reinterpret_cast<const uint32_t*>(&h23);
      lw.x = *reinterpret_cast<const uint32_t*>(&l01);
      lw.y = *reinterpret_cast<const uint32_t*>(&l23);
      *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(out) + o) = hw;
      *reinterpret_cast<uint2*>(out_lo + o) = lw;
    }
  }
}

// The points' FP32 contributions at o, added as an FP32 pair (in FP64 the
// conversions and additions bound the kernel: 24 us at 48^3, 4 points, K = 8).
__device__ __forceinline__ Pair32 kp_parts(const KpSumArgs& A, long long o) {
  Pair32 d{A.part[0][o], 0.f};
  for (int q = 1; q < A.nk; ++q) pair_add(d, Pair32{A.part[q][o], 0.f});
  return d;
}
// The same in FP64, where the pair's sum has left the FP32 range.
__device__ __noinline__ double kp_parts64(const KpSumArgs& A, long long o) {
  double x = 0.0;
  for (int q = 0; q < A.nk; ++q) x += (double)A.part[q][o];
  return x;
}

// f = sum_kappa part_kappa - v
__global__ void k_kp_sum(const __grid_constant__ KpSumArgs A, const void* __restrict__ v, int io, long long n,
                         void* __restrict__ f) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    Pair32 d = kp_parts(A, e);
    if (io == LRDM_DTYPE_F64) {
      const double x = isfinite(d.s) ? pair_value(d) : kp_parts64(A, e);
      static_cast<double*>(f)[e] = x - static_cast<const double*>(v)[e];
    } else {
      const float ve = static_cast<const float*>(v)[e];
      const bool in = isfinite(d.s);
      pair_add(d, Pair32{-ve, 0.f});
      static_cast<float*>(f)[e] = in ? pair_round(d) : (float)(kp_parts64(A, e) - (double)ve);
    }
  }
}

// out[k][r] (compute type, row stride ld; k = blockIdx.y) = sum_kappa
// part_kappa[k][r] (use_parts: FP32 contributions) or drho[k][r] (FP64
// accumulator); zero for N_g <= r < ld.
__global__ void k_kp_collect(const __grid_constant__ KpSumArgs A, int use_parts,
                             const double* __restrict__ drho, long long Ng, long long ld,
                             void* __restrict__ out, int fp64) {
  const long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x, k = blockIdx.y;
  if (r >= ld) return;
  Pair32 d{0.f, 0.f};
  double d64 = 0.0;
  bool pair = use_parts;
  if (r < Ng) {
    if (use_parts) d = kp_parts(A, k * Ng + r);
    else d64 = drho[k * Ng + r];
    if (use_parts && !isfinite(d.s)) {
      d64 = kp_parts64(A, k * Ng + r);
      pair = false;
    }
  }
  if (fp64) static_cast<double*>(out)[k * ld + r] = pair ? pair_value(d) : d64;
  else static_cast<float*>(out)[k * ld + r] = pair ? pair_round(d) : (float)d64;
}

inline unsigned kp_grid(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  if (b > 152LL * 32) b = 152LL * 32;
  return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace

cudaError_t launch_kp_dmu(const KpDmuArgs& A, double* dmu, double* dmu_out, cudaStream_t st) {
  if (A.K == 0) return cudaSuccess;
  auto kern = A.fp64 ? k_kp_dmu<double> : k_kp_dmu<float>;
  kern<<<A.K, A.fp64 ? KP_DMU_THREADS<double> : KP_DMU_THREADS<float>, 0, st>>>(A, dmu, dmu_out);
  return cudaGetLastError();
}

cudaError_t launch_kp_scale(int fp64, const void* P, int nsplit, int K, int k0, int kn, int ns,
                            const double* L, const double* dmu, void* Y, cudaStream_t st) {
  if (kn == 0) return cudaSuccess;
  const dim3 grid((unsigned)(2 * ns), (unsigned)((2 * ns + 127) / 128), (unsigned)kn);
  if (fp64)
    k_kp_scale<double><<<grid, 128, 0, st>>>(static_cast<const double*>(P), nsplit, K, k0, ns, L, dmu,
                                             static_cast<double*>(Y));
  else
    k_kp_scale<float><<<grid, 128, 0, st>>>(static_cast<const float*>(P), nsplit, K, k0, ns, L, dmu,
                                            static_cast<float*>(Y));
  return cudaGetLastError();
}

cudaError_t launch_kp_finish(const double* drho, const void* v, int io, long long n, void* f,
                             cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_kp_finish<<<kp_grid(n, 256), 256, 0, st>>>(drho, v, io, n, f);
  return cudaGetLastError();
}

cudaError_t launch_kp_density(int fp64, const void* pr, const void* pi, int ns, int ld, long long Ng,
                              const double* occ, double gw, int first, double floor, double* rho,
                              cudaStream_t st) {
  const unsigned g = kp_grid(Ng * 32, 256);
  if (fp64)
    k_kp_density<double><<<g, 256, 0, st>>>(static_cast<const double*>(pr), static_cast<const double*>(pi),
                                            ns, ld, Ng, occ, gw, first, floor, rho);
  else
    k_kp_density<float><<<g, 256, 0, st>>>(static_cast<const float*>(pr), static_cast<const float*>(pi),
                                           ns, ld, Ng, occ, gw, first, floor, rho);
  return cudaGetLastError();
}

cudaError_t launch_kp_copy(int fp64, const void* src, int io, int ld, long long Ng, int ns, void* dst,
                           int ldd, int col0, cudaStream_t st) {
  const unsigned g = kp_grid(Ng * ns, 256);
  if (fp64) k_kp_copy<double><<<g, 256, 0, st>>>(src, io, ld, Ng, ns, static_cast<double*>(dst), ldd, col0);
  else k_kp_copy<float><<<g, 256, 0, st>>>(src, io, ld, Ng, ns, static_cast<float*>(dst), ldd, col0);
  return cudaGetLastError();
}

cudaError_t launch_kp_scale_tc(const float* P, int nsplit, int K, int ns, int ld, const double* L,
                               const double* dmu, int layout, void* out, void* out_lo, cudaStream_t st) {
  if (K == 0) return cudaSuccess;
  dim3 grid((unsigned)((ld / 4 + 127) / 128), (unsigned)ld);
  k_kp_scale_tc<<<grid, 128, 0, st>>>(P, nsplit, K, ns, ld, L, dmu, layout, out,
                                      static_cast<__nv_bfloat16*>(out_lo));
  return cudaGetLastError();
}

cudaError_t launch_kp_collect(const KpSumArgs* A, const double* drho, int K, long long Ng, long long ld,
                              void* out, int fp64, cudaStream_t st) {
  if (K == 0) return cudaSuccess;
  KpSumArgs a{};
  if (A) a = *A;
  const dim3 grid((unsigned)((ld + 255) / 256), (unsigned)K);
  k_kp_collect<<<grid, 256, 0, st>>>(a, A ? 1 : 0, drho, Ng, ld, out, fp64);
  return cudaGetLastError();
}

cudaError_t launch_kp_sum(const KpSumArgs& A, const void* v, int io, long long n, void* f,
                          cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_kp_sum<<<kp_grid(n, 256), 256, 0, st>>>(A, v, io, n, f);
  return cudaGetLastError();
}

}  // namespace lrdm
