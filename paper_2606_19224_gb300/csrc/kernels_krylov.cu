// Host side of the preconditioned solve in Krylov coordinates (krylov.cuh): which configurations
// take it, its launch plan and its launch.
#include <algorithm>

#include "krylov.cuh"

namespace enkf {

template <int NT>
__global__ void __launch_bounds__(kKT, 1) krylov_kernel(KrylovParams p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_slot;
  KCta cta;
  krylov_begin(cta, smem, &mbar, &tmem_slot, p.status);
  GridBarrier bar{p.bar, reinterpret_cast<int*>(p.bar + 1), p.status, gridDim.x, 0u};
  krylov_body<NT>(p, (int)gridDim.x, (int)blockIdx.x, bar, cta);
  krylov_end(cta);
}

// R, 1/R and 1/sqrt(R) in double-float, once per handle
__global__ void krylov_rows_kernel(const double* __restrict__ r, int64_t m, df32* __restrict__ rdf,
                                   df32* __restrict__ rinv, df32* __restrict__ rsq) {
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < m; i += (int64_t)gridDim.x * kThreads) {
    const double v = r[i];
    rdf[i] = df32(v);
    rinv[i] = df32(1.0 / v);
    rsq[i] = df32(1.0 / sqrt(v));
  }
}

// CG preconditioned by R in the FP32 and (split) tensor-core modes. Plain CG is not confined to
// R^{-1} span(HA); a step count fixed by the caller, a cap on the steps between refreshes and
// single-part operands are about the recurrences on m-vectors and keep them.
bool krylov_config(const enkf_config& c) {
  return c.variant == ENKF_CGD && c.precision != ENKF_FP64 && c.precondition == 1 && c.fixed_iters == 0 &&
         (c.precision == ENKF_FP32 || (c.lowprec_terms != 1 && c.refresh_every <= 0));
}

static void* krylov_fn(int NT) {
  return NT == 32 ? (void*)krylov_kernel<32> : NT == 64 ? (void*)krylov_kernel<64> : (void*)krylov_kernel<128>;
}
static size_t krylov_smem(int NT) {
  return NT == 32 ? KLayout<32>::bytes : NT == 64 ? KLayout<64>::bytes : KLayout<128>::bytes;
}

size_t krylov_part_bytes(const enkf_handle_s* h) {
  return sizeof(df32) * (size_t)krylov_part(h->cfg.N) * std::max(h->launch.G, 2);
}

cudaError_t plan_krylov(enkf_handle_s* h) {
  const int N = h->cfg.N;
  const int NT = N <= 32 ? 32 : (N <= 64 ? 64 : 128);
  void* fn = krylov_fn(NT);
  const size_t smem = krylov_smem(NT);
  cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  int occ = 0;
  err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kKT, smem);
  if (err != cudaSuccess) return err;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  // one CTA per SM (it holds the SM's tensor memory), and no more than have a tile of rows (times
  // the column groups) or a column of the recurrences to work on
  const int64_t tiles = (h->cfg.m + kKR - 1) / kKR * (NT == 128 ? 2 : 1);
  int G = (int)std::min<int64_t>(h->sms, std::max<int64_t>(tiles, N));
  if (h->cfg.grid_blocks > 0) G = std::min(h->cfg.grid_blocks, h->sms);
  h->launch.G = G;
  h->launch.NT = NT;
  h->launch.smem = smem;
  return cudaSuccess;
}

cudaError_t launch_krylov_rows(const double* r, int64_t m, df32* rdf, df32* rinv, df32* rsq, cudaStream_t s) {
  const int blocks = (int)std::min<int64_t>((m + kThreads - 1) / kThreads, 4096);
  krylov_rows_kernel<<<blocks, kThreads, 0, s>>>(r, m, rdf, rinv, rsq);
  return cudaGetLastError();
}
cudaError_t launch_krylov_rows(enkf_handle_s* h) {
  auto& ws = h->ws;
  return launch_krylov_rows(ws.r, h->cfg.m, static_cast<df32*>(ws.rdf), static_cast<df32*>(ws.rinv),
                            static_cast<df32*>(ws.rsq), h->stream);
}

cudaError_t launch_krylov(enkf_handle_s* h, int phase, const float* w0, const double* wnorm) {
  const auto& c = h->cfg;
  auto& ws = h->ws;
  KrylovParams p{};
  p.m = c.m;
  p.N = c.N;
  p.HAdf = static_cast<const df32*>(ws.HAdf);
  p.Ddf = static_cast<const df32*>(ws.Ddf);
  p.Zdf = static_cast<df32*>(ws.Zdf);
  p.B = static_cast<float*>(ws.B);
  p.rdf = static_cast<const df32*>(ws.rdf);
  p.rinv = static_cast<const df32*>(ws.rinv);
  p.rsq = static_cast<const df32*>(ws.rsq);
  p.hs = ws.hs;
  p.umax = ws.hamax;
  df32* q = static_cast<df32*>(ws.kpart);
  p.part = q;
  q = static_cast<df32*>(ws.ksmall);   // four N x N matrices and three N-vectors
  const int NN = c.N * c.N;
  p.Kred = q;
  p.Fred = q + NN;
  p.wred = q + 2 * NN;
  p.Tred = q + 3 * NN;
  p.sums = q + 4 * NN;
  p.hold = reinterpret_cast<int*>(q + 4 * NN + 2 * c.N);
  p.rrpart = ws.rrpart;
  p.W = ws.W;
  p.tol = c.tol;
  p.max_iter = c.max_iter;
  // max_refine bounds the FP32 mode's refreshes; the tensor-core modes end on a stalled column
  p.max_refine = c.precision == ENKF_FP32 ? c.max_refine : 1 << 30;
  p.col_iters = ws.col_iters;
  p.col_relres = ws.col_relres;
  p.col_true = ws.col_true;
  p.status = ws.status;
  p.bar = ws.bar;
  p.prof = h->prof_enabled ? ws.prof : nullptr;
  p.phase = phase;
  p.w0 = w0;
  p.wnorm = wnorm;
  p.warm_accept = c.warm_accept;
  p.col_warm = ws.col_warm;
  cudaError_t err = cudaMemsetAsync(ws.bar, 0, 4 * sizeof(unsigned), h->stream);
  if (err == cudaSuccess && phase != 2) err = cudaMemsetAsync(ws.status, 0, 4 * sizeof(int32_t), h->stream);
  if (err != cudaSuccess) return err;
  void* args[] = {&p};
  return cudaLaunchCooperativeKernel(krylov_fn(h->launch.NT), dim3(h->launch.G), dim3(kKT), args,
                                     h->launch.smem, h->stream);
}

}  // namespace enkf
