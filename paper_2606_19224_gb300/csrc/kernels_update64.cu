// The ensemble update of FP64 ensembles on the tensor cores: X_a = X_f + A W with A = X_f - xbar 1^T
// (Fig. 2, Algorithm 1), or X_a = X_f V (Algorithm 2), as a product of FP64 operands (slices64.cuh).
//
// A tile is up to 80 rows of X_f: its rows (their anomalies for A W), scaled by the power of two above each row's
// largest entry, are operand A (K-major, 64 or 128 members deep), 64 columns of W, scaled per column, operand
// B, 64 members at a time. X_a leaves through shared memory, so that the stores are whole rows (X_a may be host
// memory). X_a may be X_f itself: a tile's rows are read before any of them is written.
// What bounds it are the digits and the sums of an entry (integer operations). The product on the FP64
// unit (n N^2 / 2 clocks of one SM) took 325 us at n = 10,000, N = 100; this takes 36.
#include <algorithm>

#include "common.cuh"
#include "slices64.cuh"

namespace enkf {

template <bool WIDE> struct Upd64 {
  static constexpr int KW = WIDE ? 128 : 64;          // depth of operand A
  static constexpr int AP = kDR * KW * 2, BP = 64 * 64 * 2, LDO = 65;
  static constexpr int off_b = kDg * AP;
  static constexpr int off_o = WIDE ? off_b : off_b + kDg * BP;   // X_a's 64 columns (WIDE: over B, dead by then)
  static constexpr int end0 = off_b + kDg * BP, end1 = off_o + kDR * LDO * 8;
  static constexpr int off_row = (end0 > end1 ? end0 : end1) + 64;   // exponents of rows and columns
  static constexpr int off_col = off_row + kDR * 4;
  static constexpr int off_part = off_col + 128 * 4;                 // [4][80] partial sums (FP64) or maxima
  static constexpr int need = off_part + 4 * kDR * 8;
  static constexpr int bytes = need < 120 * 1024 ? 120 * 1024 : need;   // one CTA per SM: each holds all of its tensor memory
  // operand A of M = 128 reads on past its 80 rows (lanes that no result uses)
  static_assert((kDg - 1) * AP + 128 * KW * 2 <= bytes && bytes <= 226 * 1024, "shared memory");
};

template <bool WIDE, bool ANOM>
__global__ void __launch_bounds__(kDT, 1) update64_kernel(const double* Xf, double* Xa, const double* __restrict__ W, int64_t n,
                                                          int N, int64_t rows_per, int* status) {
  using L = Upd64<WIDE>;
  constexpr int NB = WIDE ? 2 : 1;   // blocks of 64 members
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_slot;
  KCta cta;
  krylov_begin(cta, smem, &mbar, &tmem_slot, status);
  if (dynamic_smem_bytes() < (unsigned)L::bytes) {
    if (threadIdx.x == 0) atomicOr(status, DS_SMEM);
    krylov_end(cta);
    return;
  }
  const int t = threadIdx.x, lane = t & 31;
  const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  int* s_row = reinterpret_cast<int*>(smem + L::off_row);
  int* s_col = reinterpret_cast<int*>(smem + L::off_col);
  double* s_sum = reinterpret_cast<double*>(smem + L::off_part);
  int* s_max = reinterpret_cast<int*>(smem + L::off_part);
  double* s_out = reinterpret_cast<double*>(smem + L::off_o);
  const uint32_t base = smem_addr(smem), lead = warp == 0 ? elect_lane() : 0u;
  const double inv_n = 1.0 / (double)N;
  // exponents of W's columns
  for (int j = t; j < 128; j += kDT) s_col[j] = 0;
  __syncthreads();
  for (int e = t; e < N * N; e += kDT) atomicMax(&s_col[e % N], dg_abs_hi(W[e]));
  __syncthreads();
  for (int j = t; j < 128; j += kDT) s_col[j] = dg_exp(s_col[j]);
  __syncthreads();
  // W[64 kb .., 64 jb ..] into operand B: row j, 64 members deep
  auto stage_w = [&](int kb, int jb) {
    if (warp < 16) {
      const int r = warp / 2 * 8 + (lane & 7), kc = warp % 2 * 32 + (lane >> 3) * 8, j = 64 * jb + r;
      double x[8];
      int E[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int k = 64 * kb + kc + e;
        x[e] = (k < N && j < N) ? W[k * N + j] : 0.0;
        E[e] = s_col[j];
      }
      Digits8 dg;
      dg.make(x, E);
      dg.store(smem + L::off_b + (r >> 3) * 1024 + (kc >> 3) * 128 + (r & 7) * 16, L::BP);
    }
  };
  // this thread's item of a tile: row r and members [kc, kc + 8) of each block of 64
  const int r = warp / 2 * 8 + (lane & 7), kc = warp % 2 * 32 + (lane >> 3) * 8;
  const int64_t row0 = imin64(n, blockIdx.x * rows_per), row1 = imin64(n, row0 + rows_per);
  const int tiles = (int)((row1 - row0 + kDR - 1) / kDR), per = tiles > 0 ? (int)((row1 - row0 + tiles - 1) / tiles) : 0;
  if (!WIDE && tiles > 0) stage_w(0, 0);
  for (int tile = 0; tile < tiles && cta.ok; ++tile) {
    const int64_t c0 = imin64(row1, row0 + (int64_t)tile * per);
    const int rows = (int)(imin64(row1, c0 + per) - c0);
    double x[NB][8];
    double sum = 0.0;
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int k = 64 * b + kc + e;
        x[b][e] = (r < rows && k < N) ? Xf[(c0 + r) * N + k] : 0.0;
        if (ANOM) sum += x[b][e];
      }
    if (ANOM) {
      sum += __shfl_xor_sync(0xffffffffu, sum, 8);
      sum += __shfl_xor_sync(0xffffffffu, sum, 16);
      if (lane < 8) s_sum[warp % 2 * kDR + r] = sum;
      __syncthreads();
      const double mean = (s_sum[r] + s_sum[kDR + r]) * inv_n;
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (r < rows && 64 * b + kc + e < N) x[b][e] -= mean;
      __syncthreads();   // s_max lies over the sums
    }
    int mx = 0;
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int e = 0; e < 8; ++e) mx = max(mx, dg_abs_hi(x[b][e]));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
    if (lane < 8) s_max[warp % 2 * kDR + r] = mx;
    __syncthreads();
    const int er = dg_exp(max(s_max[r], s_max[kDR + r]));
    if (warp % 2 == 0 && lane < 8) s_row[r] = er;
    const int E[8] = {er, er, er, er, er, er, er, er};
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      Digits8 dg;
      dg.make(x[b], E);
      dg.store(smem + (r >> 3) * (L::KW / 8 * 128) + (8 * b + (kc >> 3)) * 128 + (r & 7) * 16, L::AP);
    }
#pragma unroll 1
    for (int jb = 0; jb < NB && 64 * jb < N; ++jb) {
#pragma unroll 1
      for (int kb = 0; kb < NB && 64 * kb < N; ++kb) {
        if (WIDE) stage_w(kb, jb);
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        if (warp == 0) {
          tc_fence_after();
          dg_issue<false, false, L::AP, 256, L::BP, 256>(cta.tmem, umma_desc(base + kb * 1024, 128, L::KW / 8 * 128),
                                                         umma_desc(base + L::off_b, 128, 1024), (min(64, N - 64 * kb) + 15) / 16,
                                                         kb > 0, cta.mbar, lead);
        }
        k_wait(cta);
      }
      const int qd = warp & 3, ln = 32 * qd + lane;
      if (32 * qd < rows) {   // uniform in the warp
        const int ea = s_row[min(ln, kDR - 1)];
#pragma unroll 1
        for (int q0 = (warp >> 2) * 4; q0 < min(64, N - 64 * jb); q0 += 4 * (kDT / 128)) {
          float lv[kDl][4];
          tmem_ld_levels<kDl, 4>(cta.tmem + ((uint32_t)(32 * qd) << 16) + q0, 64, lv);
          if (ln < rows)
#pragma unroll
            for (int q = 0; q < 4; ++q) s_out[ln * L::LDO + q0 + q] = dg_value(dg_join(lv, q), ea, s_col[64 * jb + q0 + q]);
        }
      }
      tc_fence_before();
      __syncthreads();
      const int cols = min(64, N - 64 * jb);
      for (int e = t; e < rows * 64; e += kDT) {
        const int i = e / 64, c = e % 64;
        if (c < cols) {
          const int64_t at = (c0 + i) * N + 64 * jb + c;
          const double v = s_out[i * L::LDO + c];
          Xa[at] = ANOM ? Xf[at] + v : v;
        }
      }
      __syncthreads();   // s_out (over operand B if WIDE), s_row and the sums are rewritten
    }
  }
  krylov_end(cta);
}

template <bool WIDE, bool ANOM>
static cudaError_t launch_one64(const double* Xf, double* Xa, const double* W, int64_t n, int N, int* status, int sms, cudaStream_t s) {
  using L = Upd64<WIDE>;
  cudaError_t e = cudaFuncSetAttribute(update64_kernel<WIDE, ANOM>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::bytes);
  if (e != cudaSuccess) return e;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n + 31) / 32, sms));
  update64_kernel<WIDE, ANOM><<<grid, kDT, L::bytes, s>>>(Xf, Xa, W, n, N, (n + grid - 1) / grid, status);
  return cudaGetLastError();
}

cudaError_t launch_update64(enkf_handle_s* h, const void* Xf, void* Xa, bool product) {
  const auto& c = h->cfg;
  const double* x = static_cast<const double*>(Xf);
  double* xa = static_cast<double*>(Xa);
  int* st = h->ws.status;
  if (c.N > 64)
    return product ? launch_one64<true, false>(x, xa, h->ws.W, c.n, c.N, st, h->sms, h->stream)
                   : launch_one64<true, true>(x, xa, h->ws.W, c.n, c.N, st, h->sms, h->stream);
  return product ? launch_one64<false, false>(x, xa, h->ws.W, c.n, c.N, st, h->sms, h->stream)
                 : launch_one64<false, true>(x, xa, h->ws.W, c.n, c.N, st, h->sms, h->stream);
}

}  // namespace enkf
