// Set-up kernels run once by lrdm_create: operand copies of Psi, the density
// and the LDA exchange kernel, and the Loewner matrix of the Fermi function.
#include "lrdm_internal.h"

#include <math.h>

namespace lrdm {
namespace {

// round-to-nearest into the TF32 format (the tensor cores read 10 mantissa bits)
__device__ __forceinline__ float to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

__device__ __forceinline__ double load_io(const void* p, int io_dtype, long long i) {
  return io_dtype == LRDM_DTYPE_F64 ? static_cast<const double*>(p)[i]
                                    : (double)static_cast<const float*>(p)[i];
}

// Row-major copies: psi64 / psi32 [Ng][ns]
__global__ void k_copy_rowmajor(const void* __restrict__ src, int io_dtype, int ld, long long Ng,
                                int ns, double* __restrict__ d64, float* __restrict__ d32) {
  long long total = Ng * ns;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    long long r = e / ns;
    int i = (int)(e - r * ns);
    double x = load_io(src, io_dtype, r * ld + i);
    if (d64) d64[e] = x;
    if (d32) d32[e] = (float)x;
  }
}

__device__ __forceinline__ uint32_t pack_bf2(__nv_bfloat16 a, __nv_bfloat16 b) {
  const __nv_bfloat162 v = __halves2bfloat162(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// x = hi + lo: four values as 8 bytes of hi and of lo
__device__ __forceinline__ void split4(const float (&x)[4], uint2& hi, uint2& lo) {
  __nv_bfloat16 h[4], l[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    h[c] = __float2bfloat16_rn(x[c]);
    l[c] = __float2bfloat16_rn(x[c] - __bfloat162float(h[c]));
  }
  hi = make_uint2(pack_bf2(h[0], h[1]), pack_bf2(h[2], h[3]));
  lo = make_uint2(pack_bf2(l[0], l[1]), pack_bf2(l[2], l[3]));
}

// Padded row-major [Ng_pad][ns_pad] and transposed tile-major copies for the
// tensor-core paths; split into bf16 hi/lo (x = hi + lo, lo = bf16(x - hi)) or
// rounded to TF32.  The transposed copies are [i / 128][r / RB][i % 128][r % RB]
// with RB = 64 bytes of the operand type (16 TF32, 32 bf16; the exact FP32 copy
// of the split mode shares the bf16 RB = 32), so that one (128 states x RB rows)
// tensor-core operand tile is a contiguous block.
//
// A block converts 32 rows x 128 states through shared memory: one such tile of
// the split mode (8 or 16 KB written in a piece), two of TF32.  Bound by HBM
// (20 bytes a value split, 12 TF32); four values a thread, 16-byte loads (vec:
// FP32 rows on 16-byte boundaries) and 8- or 16-byte stores.  48^3, N_s = 512:
// 239 -> 133 us (32 x 32 tiles with 2-byte stores before; 135 us at the copy
// rate).
__global__ void __launch_bounds__(256)
    k_copy_tc(const void* __restrict__ src, int io_dtype, int ld, long long Ng, int ns, long long Ng_pad,
              int ns_pad, int vec, float* __restrict__ R32, float* __restrict__ T32,
              __nv_bfloat16* __restrict__ Rhi, __nv_bfloat16* __restrict__ Rlo,
              __nv_bfloat16* __restrict__ Thi, __nv_bfloat16* __restrict__ Tlo, float* __restrict__ Tf) {
  __shared__ float tile[128][33];                  // [state][row]
  const long long r0 = (long long)blockIdx.x * 32;
  const int i0 = blockIdx.y * 128;
  for (int e = threadIdx.x; e < 32 * 32; e += 256) {
    const int rr = e >> 5, ii = 4 * (e & 31), i = i0 + ii;
    const long long r = r0 + rr;
    float x[4] = {0.f, 0.f, 0.f, 0.f};
    if (r < Ng) {
      if (vec && i + 3 < ns) {
        const float4 v = *reinterpret_cast<const float4*>(static_cast<const float*>(src) + r * ld + i);
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (i + c < ns) x[c] = (float)load_io(src, io_dtype, r * ld + i + c);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) tile[ii + c][rr] = x[c];
    const long long o = r * ns_pad + i;            // (Ng_pad and ns_pad are multiples of 128)
    if (R32) *reinterpret_cast<float4*>(R32 + o) =
        make_float4(to_tf32(x[0]), to_tf32(x[1]), to_tf32(x[2]), to_tf32(x[3]));
    if (Rhi) {
      uint2 hi, lo;
      split4(x, hi, lo);
      *reinterpret_cast<uint2*>(Rhi + o) = hi;
      *reinterpret_cast<uint2*>(Rlo + o) = lo;
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 128 * 8; e += 256) {
    const int ii = e >> 3, rr = 4 * (e & 7);
    const float x[4] = {tile[ii][rr], tile[ii][rr + 1], tile[ii][rr + 2], tile[ii][rr + 3]};
    if (T32) {
      const long long o = (((long long)blockIdx.y * (Ng_pad / 16) + (r0 + rr) / 16) * 128 + ii) * 16 + rr % 16;
      *reinterpret_cast<float4*>(T32 + o) = make_float4(to_tf32(x[0]), to_tf32(x[1]), to_tf32(x[2]), to_tf32(x[3]));
    } else {
      const long long o = (((long long)blockIdx.y * (Ng_pad / 32) + blockIdx.x) * 128 + ii) * 32 + rr;
      if (Thi) {
        uint2 hi, lo;
        split4(x, hi, lo);
        *reinterpret_cast<uint2*>(Thi + o) = hi;
        *reinterpret_cast<uint2*>(Tlo + o) = lo;
      }
      if (Tf) *reinterpret_cast<float4*>(Tf + o) = make_float4(x[0], x[1], x[2], x[3]);
    }
  }
}

// rho(r) = g sum_i f_i psi_i(r)^2 + floor, one warp per grid point (Eq. densityChFSI)
__global__ void k_density(const void* __restrict__ psi, int io_dtype, int ld, long long Ng, int ns,
                          const double* __restrict__ occ, double g, double floor,
                          double* __restrict__ rho) {
  int lane = threadIdx.x & 31;
  long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long r = warp; r < Ng; r += nwarps) {
    double acc = 0.0;
    for (int i = lane; i < ns; i += 32) {
      double p = load_io(psi, io_dtype, r * ld + i);
      acc += occ[i] * p * p;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) rho[r] = g * acc + floor;
  }
}

__global__ void k_copy_rho(const void* __restrict__ src, int io_dtype, long long Ng,
                           double* __restrict__ rho) {
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < Ng;
       r += (long long)gridDim.x * blockDim.x)
    rho[r] = load_io(src, io_dtype, r);
}

// LDA exchange kernel dV_x/drho = -(1/3) c rho^(-2/3), c = (3/pi)^(1/3)
// (restricted) or (6/pi)^(1/3) (one spin channel); density floored at 1e-12.
__global__ void k_fx(const double* __restrict__ rho, long long Ng, int spin_polarized,
                     double* __restrict__ fx) {
  const double c = spin_polarized ? 1.2407009817988002 /* (6/pi)^(1/3) */
                                  : 0.98474502184269654 /* (3/pi)^(1/3) */;
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < Ng;
       r += (long long)gridDim.x * blockDim.x) {
    double x = fmax(rho[r], 1e-12);
    double t = rcbrt(x);
    fx[r] = -(c / 3.0) * t * t;
  }
}

__device__ __forceinline__ double log_cosh(double y) {
  double a = fabs(y);
  return a + log1p(exp(-2.0 * a)) - 0.69314718055994531;
}

// log(sinh(u)/u), even in u
__device__ __forceinline__ double log_sinhc(double u) {
  double a = fabs(u);
  if (a == 0.0) return 0.0;
  if (a < 0.5) return log1p(sinh(a) / a - 1.0);
  return a + log1p(-exp(-2.0 * a)) - 0.69314718055994531 - log(a);
}

// Loewner matrix of the Fermi function at eps:
//   L_ij = -sinhc((x_i - x_j)/2) / (4 kT cosh(x_i/2) cosh(x_j/2)), x = (eps - mu)/kT,
// equal to (f_i - f_j)/(eps_i - eps_j) and to -f(1-f)/kT on the diagonal, with no
// cancellation for near-degenerate pairs.  Log domain where a factor could overflow.
// occ_mode: divided differences of the given occupations, midpoint derivative
// for |eps_i - eps_j| <= degen_tol kT.
__global__ void k_loewner_f32(const double* __restrict__ L, int ns, int ns_pad,
                              float* __restrict__ Lf) {
  const long long total = (long long)ns_pad * ns_pad;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e / ns_pad), j = (int)(e - (long long)i * ns_pad);
    Lf[e] = (i < ns && j < ns) ? (float)L[(long long)i * ns + j] : 0.f;
  }
}

// artanh(w) / w, even in w, |w| < 1
__device__ __forceinline__ double artanhc(double w) {
  const double a = fabs(w);
  if (a < 1e-4) return 1.0 + a * a / 3.0;
  return atanh(a) / a;
}

// Loewner matrix of f_T(e) = 1 / (1 + exp(g(e))), g = c artanh(u), c = 2^(T+1),
// u = (e - mu) / (c kT), |u| < 1: with
//   f_i - f_j = -sinh((g_i - g_j)/2) / (2 cosh(g_i/2) cosh(g_j/2)) and
//   g_i - g_j = c artanh(w), w = (u_i - u_j) / (1 - u_i u_j),  u_i - u_j = (e_i - e_j)/(c kT),
//   L_ij = -sinhc((g_i - g_j)/2) artanhc(w) / (4 kT (1 - u_i u_j) cosh(g_i/2) cosh(g_j/2)),
// free of cancellation for close e_i, e_j; in the log domain where a factor
// would overflow.  The diagonal (w = 0) is f_T'.
__device__ double loewner_T(double ei, double ej, double mu, double kT, int T) {
  const double c = ldexp(1.0, T + 1);
  const double ui = (ei - mu) / (c * kT), uj = (ej - mu) / (c * kT);
  const double gi = c * atanh(ui), gj = c * atanh(uj);
  const double den = 1.0 - ui * uj;
  const double w = (ui - uj) / den;
  const double hd = 0.5 * (gi - gj);
  if (fabs(gi) < 1400.0 && fabs(gj) < 1400.0 && fabs(hd) < 700.0) {
    const double sc = hd == 0.0 ? 1.0 : sinh(hd) / hd;
    return -sc * artanhc(w) / (4.0 * kT * den * cosh(0.5 * gi) * cosh(0.5 * gj));
  }
  const double lm = log_sinhc(hd) + log(artanhc(w)) - log(4.0 * kT * den) - log_cosh(0.5 * gi) -
                    log_cosh(0.5 * gj);
  return -exp(lm);
}

// A block takes the 32 x 32 entries (I, J), I <= J, and writes them to (J, I) as
// well: L is symmetric.  cosh(x / 2) of its 64 states once, a sinh and two
// divisions an entry remain; FP64-bound.  N_s = 512: 64 -> 22 us.
__global__ void __launch_bounds__(256)
    k_loewner(const double* __restrict__ eps, const double* __restrict__ occ, int ns, double mu, double kT,
              int occ_mode, double degen_tol, int fermi_T, double* __restrict__ L) {
  __shared__ double xs[64], ch[64];                // x = (eps - mu) / kT and cosh(x / 2) of rows, columns
  int I = 0, t = blockIdx.x;                       // block t: column J = I + t of row I of the triangle
  for (int len = (ns + 31) / 32; t >= len; --len, ++I) t -= len;
  const int i0 = 32 * I, j0 = 32 * (I + t);
  if (threadIdx.x < 64) {
    const int q = threadIdx.x < 32 ? i0 + threadIdx.x : j0 + threadIdx.x - 32;
    const double x = q < ns ? (eps[q] - mu) / kT : 0.0;
    xs[threadIdx.x] = x;
    ch[threadIdx.x] = cosh(0.5 * x);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 1024; e += 256) {
    const int li = e >> 5, lj = e & 31, i = i0 + li, j = j0 + lj;
    if (j < i || j >= ns) continue;
    double val;
    if (fermi_T > 0) {
      val = loewner_T(eps[i], eps[j], mu, kT, fermi_T);
    } else if (occ_mode) {
      double de = eps[i] - eps[j];
      if (fabs(de) <= degen_tol * kT) {
        double fb = 0.5 * (occ[i] + occ[j]);
        val = -fb * (1.0 - fb) / kT;
      } else {
        val = (occ[i] - occ[j]) / de;
      }
    } else {
      double xi = xs[li], xj = xs[32 + lj];
      double u = 0.5 * (xi - xj);
      if (fabs(xi) < 700.0 && fabs(xj) < 700.0 && fabs(u) < 700.0) {
        double sc = (u == 0.0) ? 1.0 : sinh(u) / u;
        val = -sc / (4.0 * kT * ch[li] * ch[32 + lj]);
      } else {
        double lm = log_sinhc(u) - log(4.0 * kT) - log_cosh(0.5 * xi) - log_cosh(0.5 * xj);
        val = -exp(lm);
      }
    }
    L[(long long)i * ns + j] = val;
    L[(long long)j * ns + i] = val;
  }
}

__global__ void k_to_io(const double* __restrict__ src, long long n, void* __restrict__ dst,
                        int io_dtype) {
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < n;
       r += (long long)gridDim.x * blockDim.x) {
    if (io_dtype == LRDM_DTYPE_F64) static_cast<double*>(dst)[r] = src[r];
    else static_cast<float*>(dst)[r] = (float)src[r];
  }
}

inline int grid_for(long long n, int block) {
  long long b = (n + block - 1) / block;
  if (b > 152LL * 64) b = 152LL * 64;
  if (b < 1) b = 1;
  return (int)b;
}

}  // namespace

cudaError_t launch_convert_psi(const void* src, int io_dtype, int ld, long long Ng, int ns,
                               Channel& c, int prec, long long Ng_pad, cudaStream_t st) {
  if (prec == LRDM_FP64 || prec == LRDM_FP32) {
    k_copy_rowmajor<<<grid_for(Ng * ns, 256), 256, 0, st>>>(src, io_dtype, ld, Ng, ns, c.psi64,
                                                             c.psi32);
    return cudaGetLastError();
  }
  static_assert(TC_PAD_GRID % 32 == 0 && TC_PAD_STATES == 128, "tiles of k_copy_tc");
  const int vec = io_dtype == LRDM_DTYPE_F32 && ld % 4 == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
  k_copy_tc<<<dim3((unsigned)(Ng_pad / 32), (unsigned)(c.ns_pad / 128)), 256, 0, st>>>(
      src, io_dtype, ld, Ng, ns, Ng_pad, c.ns_pad, vec, c.psiR32, c.psiT32, c.psiR_hi, c.psiR_lo, c.psiT_hi,
      c.psiT_lo, c.psiTf);
  return cudaGetLastError();
}

cudaError_t launch_density(const void* psi_src, int io_dtype, int ld, long long Ng, int ns,
                           const double* occ, double g, double floor, double* rho,
                           cudaStream_t st) {
  k_density<<<grid_for(Ng * 32, 256), 256, 0, st>>>(psi_src, io_dtype, ld, Ng, ns, occ, g, floor,
                                                     rho);
  return cudaGetLastError();
}

cudaError_t launch_copy_rho(const void* src, int io_dtype, long long Ng, double* rho,
                            cudaStream_t st) {
  k_copy_rho<<<grid_for(Ng, 256), 256, 0, st>>>(src, io_dtype, Ng, rho);
  return cudaGetLastError();
}

cudaError_t launch_fx(const double* rho, long long Ng, int spin_polarized, double* fx,
                      cudaStream_t st) {
  k_fx<<<grid_for(Ng, 256), 256, 0, st>>>(rho, Ng, spin_polarized, fx);
  return cudaGetLastError();
}

cudaError_t launch_loewner(const double* eps, const double* occ, int ns, double mu, double kT,
                           int occ_mode, double degen_tol, int fermi_T, double* L,
                           cudaStream_t st) {
  const long long nt = (ns + 31) / 32;
  k_loewner<<<(unsigned)(nt * (nt + 1) / 2), 256, 0, st>>>(eps, occ, ns, mu, kT, occ_mode, degen_tol, fermi_T, L);
  return cudaGetLastError();
}

cudaError_t launch_loewner_f32(const double* L, int ns, int ns_pad, float* Lf, cudaStream_t st) {
  k_loewner_f32<<<grid_for((long long)ns_pad * ns_pad, 256), 256, 0, st>>>(L, ns, ns_pad, Lf);
  return cudaGetLastError();
}

cudaError_t launch_to_io(const double* src, long long n, void* dst, int io_dtype,
                         cudaStream_t st) {
  k_to_io<<<grid_for(n, 256), 256, 0, st>>>(src, n, dst, io_dtype);
  return cudaGetLastError();
}

}  // namespace lrdm
