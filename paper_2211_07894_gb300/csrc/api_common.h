// Helpers shared by the host-side files of the C ABI (lrdm_api.cu: contexts,
// forward, least squares, adjoint; lrdm_lrdma.cu: the accumulated LRDM
// driver; lrdm_kpoint_api.cu: Brillouin-zone-sampled systems).  Not part of
// the public interface.
#pragma once

#include <vector>

#include "lrdm_internal.h"

namespace lrdm {
namespace api {

// CUDA / cuFFT result -> lrdm_status (LRDM_DEBUG=1 prints the CUDA error)
lrdm_status from_cuda(cudaError_t e);
lrdm_status from_cufft(cufftResult r);

#define LRDM_CK(expr)                          \
  do {                                         \
    lrdm_status _s = (expr);                   \
    if (_s != LRDM_OK) return _s;              \
  } while (0)
#define LRDM_CU(expr) LRDM_CK(from_cuda(expr))
#define LRDM_FFT(expr) LRDM_CK(from_cufft(expr))

// Destroys the plans kept from closed contexts; whether there were any.
bool release_idle();
// cudaMalloc, again without those plans where memory is short; a refusal leaves
// no pending CUDA error behind (the create calls try again with less).
lrdm_status device_alloc(void** q, size_t bytes);

// Device allocation owned by the context (freed by lrdm_destroy), zeroed
// unless zero == false.  The zeroing is ordered on the stream of the set-up
// (ctx->setup_st), which the create calls wait for before they return: on the
// legacy stream it could run after the first kernels of a stream that does not
// wait for that one, over what they had written.  A context has some 25 small buffers (up to 2 MB at
// N_s = 512) beside the operand copies, each with its cudaMalloc, cudaMemset and
// cudaFree: up to ARENA_MAX bytes they are cut from blocks of ARENA_BLOCK, which
// are zeroed once (48^3, N_s = 512: create 1.75 -> 1.65 ms, destroy 1.06 -> 0.91
// ms; the rest of both is the large buffers, 0.5 us a MB to free).  A context
// made where memory is short (ctx->lean) has no blocks.
constexpr size_t ARENA_BLOCK = 8u << 20, ARENA_MAX = 2u << 20, ARENA_ALIGN = 512;

template <typename T>
lrdm_status dalloc(lrdm_ctx* ctx, T** p, size_t count, bool zero = true) {
  *p = nullptr;
  if (count == 0) count = 1;
  const size_t bytes = count * sizeof(T);
  if (bytes <= ARENA_MAX && !ctx->lean) {
    const size_t need = (bytes + ARENA_ALIGN - 1) / ARENA_ALIGN * ARENA_ALIGN;
    if (need > ctx->arena_left) {
      void* q = nullptr;
      if (cudaMalloc(&q, ARENA_BLOCK) == cudaSuccess) {
        ctx->allocs.push_back(q);
        LRDM_CU(cudaMemsetAsync(q, 0, ARENA_BLOCK, ctx->setup_st));
        ctx->arena = static_cast<char*>(q);
        ctx->arena_left = ARENA_BLOCK;
      } else {
        (void)cudaGetLastError();       // no room for a block: an allocation of its own below
      }
    }
    if (need <= ctx->arena_left) {
      *p = reinterpret_cast<T*>(ctx->arena);
      ctx->arena += need;
      ctx->arena_left -= need;
      return LRDM_OK;
    }
  }
  void* q = nullptr;
  LRDM_CK(device_alloc(&q, bytes));
  ctx->allocs.push_back(q);
  if (zero) LRDM_CU(cudaMemsetAsync(q, 0, bytes, ctx->setup_st));
  *p = static_cast<T*>(q);
  return LRDM_OK;
}

inline bool is_tc(int prec) { return prec == LRDM_TF32 || prec == LRDM_BF16X3; }
size_t io_size(int io);
// numerically stable Fermi function f = 1/(1 + exp(x))
double fermi_host(double x);

// profiling records (lrdm_profile_enable): event pairs and launch counts
int prof_begin(lrdm_ctx* ctx, int kind, cudaStream_t st);
void prof_end(lrdm_ctx* ctx, int i, cudaStream_t st);
void count(lrdm_ctx* ctx, int n);

// Poisson transforms, symbol table and buffers of system S; V_H in place in
// S.fft_real for all k_max slots
lrdm_status setup_poisson(lrdm_ctx* ctx, SysState& S, cudaStream_t st);
lrdm_status hartree(lrdm_ctx* ctx, SysState& S, int K, cudaStream_t st);
// grouped tensor-core launch of ctx->tc_entries (gemm 1: projection, 2: response)
lrdm_status tc_group(lrdm_ctx* ctx, int gemm, int out_is_io, cudaStream_t st);
int tc_split(long long items, long long units, int nch, int smax);
// launch-shape tuner of the tensor-core contractions (options.autotune)
lrdm_status autotune(lrdm_ctx* ctx, cudaStream_t st);
void free_ctx(lrdm_ctx* ctx);

// the forward of every system of a context; one forward call of the direction
// drivers (system sys only; k-point contexts run kp_forward)
lrdm_status forward_all(lrdm_ctx* ctx, const void* const* v, const int* K, void* const* f,
                        double* dmu_out, cudaStream_t st);
lrdm_status forward_one(lrdm_ctx* ctx, int sys, const void* const* v, const int* K, void* const* f,
                        cudaStream_t st);
// Brillouin-zone-sampled contexts (lrdm_kpoint_api.cu)
lrdm_status kp_forward(lrdm_ctx* ctx, const void* v, int K, void* f_out, double* dmu_out, cudaStream_t st);
lrdm_status kp_backward(lrdm_ctx* ctx, const void* const* f_bar, void* const* v_bar,
                        double* const* eps_bar, double* const* occ_bar, cudaStream_t st);

// CUDA graph of a forward call: captured on the first call with a given key
// (buffers, K's, stream), replayed afterwards.  Not used on the legacy
// default stream or while profiling.
bool use_graph(const lrdm_ctx* ctx, cudaStream_t st);
template <typename Body>
lrdm_status graph_call(lrdm_ctx* ctx, const std::vector<const void*>& key, cudaStream_t st, Body body) {
  if (ctx->graph_exec && key == ctx->graph_key) return from_cuda(cudaGraphLaunch(ctx->graph_exec, st));
  if (ctx->graph_exec) {
    cudaGraphExecDestroy(ctx->graph_exec);
    ctx->graph_exec = nullptr;
  }
  LRDM_CU(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
  lrdm_status rc = body();
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamEndCapture(st, &g);
  if (rc != LRDM_OK) {
    if (g) cudaGraphDestroy(g);
    return rc;
  }
  LRDM_CU(e);
  e = cudaGraphInstantiate(&ctx->graph_exec, g, 0);
  cudaGraphDestroy(g);
  LRDM_CU(e);
  ctx->graph_key = key;
  return from_cuda(cudaGraphLaunch(ctx->graph_exec, st));
}

}  // namespace api
}  // namespace lrdm
