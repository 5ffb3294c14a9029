// CGD-EnKF-Reduced (Sec. 5.2): Algorithm 2 with (I + P^T P)^{-1} applied by CG.
//
//   P = L^{-1} HA with L L^T = R_N = (N-1) R (L diagonal here), so
//   G = I + P^T P          = I + HA^T R^{-1} HA / (N-1)                  (N x N)
//   M = I + P^T L^{-1} Y~  = I + HA^T R^{-1} Y~ / (N-1),  Y~ = (y - zbar) 1^T + E
//   V = G^{-1} M by N independent CG recurrences (one per column of M), X_a = X_f V.
//
//   gram64_kernel,         one pass over the observation rows: gathers the rows of X_f that
//   gram_tc_kernel         H touches, forms HA and D for a tile of rows in a buffer that stays in L2,
//   (FP64, FP32 ensembles) and accumulates this CTA's partial HA^T R^{-1} [HA | Y~] (the paper's
//                          "dominant cost ... formation of an N x N matrix", Sec. 6.2.2) on the tensor
//                          cores from exact integer slices
//   reduced_sum_kernel     fixed-order sum of the CTA partials -> G, M (FP64)
//   reduced_cg_kernel      one CTA per column of M; G staged in shared memory; FP64 CG
//   update (kernels_fp.cu) X_a = X_f V (plain product mode)
//
// The same pass serves the paper's sEnKF comparator (Algorithm 3, the diagonal-inverse
// approximation): with the weights 1/s_i, s_i = |HA_i|^2 + (N-1) r_i (the diagonal of
// HA HA^T + R_N) instead of 1/r_i, and the innovation row D_i = Y~_i - HA_i as the only right
// factor (an N x N product per row instead of N x 2N), it forms
// W = sum_i HA_i^T D_i / s_i = HA^T diag(HA HA^T + R_N)^{-1} D, and X_a = X_f + A W (the
// CGD-EnKF update) with no solve at all.
#include "common.cuh"
#include "innov_device.cuh"
#include "gram_stages.cuh"
#include "krylov.cuh"
#include "slices64.cuh"

#include <algorithm>

namespace enkf {

// ------------------------------------------------------------------ FP64 ensembles
// K = U^T U and F = U^T V with U = w HA, w_i = 1/sqrt(r_i) (sEnKF: 1/sqrt(s_i)) and V = w Y~ (sEnKF: w D), as
// products of FP64 operands on the tensor cores (slices64.cuh). A CTA forms HA and D of a tile of up to 80
// rows in a buffer of its own (it stays in L2), then cuts 64 columns at a time into digits, each column
// scaled by the power of two above its largest entry in the tile: N <= 64, [U | V]^T U (M = 128: rows of
// K, then of F^T); N > 64, [U_0 | U_1]^T times U_0, U_1, V_0 and V_1 in turn. At m = 10,000, N = 100 it takes
// 171 us, most of them the FP64 logarithms and sines of the drawn perturbations; with the products on the FP64
// unit it took 1.0 ms.
struct Gram64 {
  const double* Xf;
  const int32_t* rowptr;
  const int32_t* col;
  const double* w;
  const double* y;
  const double* r;
  const double* E;
  int emode;
  uint64_t seed, counter;
  int64_t m, rows_per;
  int N;
  bool senkf;
  double* part;      // [grid][2][N][N]: K and F (sEnKF: F in the first)
  double* scratch;   // [grid][2][kDR][N]: HA and D of a tile
  int* status;
};
struct Gram64Smem {
  static constexpr int AP = kDR * 128 * 2, BR = kDg * 64 * 16;   // bytes per digit of A; per row group of B
  static constexpr int off_b = kDg * AP, off_max = off_b + kDR / 8 * BR;
  static constexpr int off_exp = off_max + kDR / 8 * 64 * 4, off_w = off_exp + 3 * 64 * 4, bytes = off_w + kDR * 8;
  static_assert(bytes <= 226 * 1024, "shared memory");
};

__global__ void __launch_bounds__(kDT, 1) gram64_kernel(Gram64 g) {
  using L = Gram64Smem;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_slot;
  KCta cta;
  krylov_begin(cta, smem, &mbar, &tmem_slot, g.status);
  const int N = g.N, t = threadIdx.x, lane = t & 31;
  const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  if (dynamic_smem_bytes() < (unsigned)L::bytes) {
    if (t == 0) atomicOr(g.status, DS_SMEM);
    krylov_end(cta);
    return;
  }
  int* s_max = reinterpret_cast<int*>(smem + L::off_max);      // [10][64] largest |x| (high words)
  int* s_exp = reinterpret_cast<int*>(smem + L::off_exp);      // exponents of A's two column blocks and B's
  double* s_w = reinterpret_cast<double*>(smem + L::off_w);
  const bool wide = N > 64;
  const int64_t row0 = imin64(g.m, blockIdx.x * g.rows_per), row1 = imin64(g.m, row0 + g.rows_per);
  const int tiles = max(1, (int)((row1 - row0 + kDR - 1) / kDR)), per = (int)((row1 - row0 + tiles - 1) / tiles);
  double* HA = g.scratch + (int64_t)blockIdx.x * 2 * kDR * N;
  double* D = HA + kDR * N;
  double* out = g.part + (int64_t)blockIdx.x * 2 * N * N;
  const uint32_t base = smem_addr(smem), lead = warp == 0 ? elect_lane() : 0u;
  // this thread's item: row r and columns [cc, cc + 8) of a block of 64
  const int r = warp / 2 * 8 + (lane & 7), cc = warp % 2 * 32 + (lane >> 3) * 8;
  for (int tile = 0; tile < tiles && cta.ok; ++tile) {   // at least one: a CTA without rows writes zeros
    const int64_t c0 = imin64(row1, row0 + (int64_t)tile * per);
    const int rows = (int)(imin64(row1, c0 + per) - c0), ks = (rows + 15) / 16;
    innov_rows_f64<double>(g.Xf, g.rowptr, g.col, g.w, g.y, g.r, g.E, g.emode, g.seed, g.counter, N, HA, D, c0,
                           c0 + rows, warp, kDT / 32, c0);
    __syncthreads();
    if (g.senkf) {
      for (int i = warp; i < rows; i += kDT / 32) {
        double q = 0.0;
        for (int k = lane; k < N; k += 32) q = fma(HA[i * N + k], HA[i * N + k], q);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        if (lane == 0) s_w[i] = 1.0 / sqrt(q + (double)(N - 1) * g.r[c0 + i]);
      }
    } else if (t < rows) {
      s_w[t] = 1.0 / sqrt(g.r[c0 + t]);
    }
    __syncthreads();
    // columns [64 c, 64 c + 64) of U (v = false) or V into operand A's block `to_a` (if >= 0) and operand B
    auto block = [&](bool v, int c, int to_a, bool to_b) {
      double x[8];
      int E[8];
      const double wr = r < rows ? s_w[r] : 0.0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int k = 64 * c + cc + e;
        const bool in = r < rows && k < N;
        double q = 0.0;
        if (in) {
          const double* at = HA + r * N + k;
          q = !v ? at[0] : g.senkf ? at[kDR * N] : at[kDR * N] + at[0];
        }
        x[e] = q * wr;
        E[e] = dg_abs_hi(x[e]);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) E[e] = max(E[e], __shfl_xor_sync(0xffffffffu, E[e], o));
      }
      if ((lane & 7) == 0)
#pragma unroll
        for (int e = 0; e < 8; ++e) s_max[warp / 2 * 64 + cc + e] = E[e];
      tc_fence_before();
      __syncthreads();   // (and the reads of the last product's sums and scales are done)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        int mx = 0;
#pragma unroll
        for (int b = 0; b < kDR / 8; ++b) mx = max(mx, s_max[b * 64 + cc + e]);
        E[e] = dg_exp(mx);
        if (r == 0) {
          if (to_a >= 0) s_exp[to_a * 64 + cc + e] = E[e];
          if (to_b) s_exp[128 + cc + e] = E[e];
        }
      }
      Digits8 dg;
      dg.make(x, E);
      if (to_a >= 0) dg.store(smem + ((r >> 3) * 16 + to_a * 8 + (cc >> 3)) * 128 + (r & 7) * 16, L::AP);
      if (to_b) dg.store(smem + L::off_b + (r >> 3) * L::BR + (cc >> 3) * 128 + (r & 7) * 16, 64 * 16);
      fence_async_smem();
      __syncthreads();
    };
    // A^T B, then put(lane row, column, value)
    auto product = [&](auto put) {
      if (warp == 0) {
        tc_fence_after();
        dg_issue<true, true, L::AP, 2 * 2048, 64 * 16, 2 * L::BR>(cta.tmem, umma_desc(base, 2048, 128),
                                                                 umma_desc(base + L::off_b, L::BR, 128), max(ks, 1), false, cta.mbar, lead);
      }
      k_wait(cta);
      if (warp < 16) {
        const int qd = warp & 3, ln = 32 * qd + lane, ea = s_exp[ln];
#pragma unroll 1
        for (int q0 = (warp >> 2) * 16; q0 < (warp >> 2) * 16 + 16; q0 += 4) {
          float lv[kDl][4];
          tmem_ld_levels<kDl, 4>(cta.tmem + ((uint32_t)(32 * qd) << 16) + q0, 64, lv);
#pragma unroll
          for (int q = 0; q < 4; ++q) put(ln, q0 + q, dg_value(dg_join(lv, q), ea, s_exp[128 + q0 + q]));
        }
      }
    };
    auto add = [&](int64_t e, double v) { out[e] = tile > 0 ? out[e] + v : v; };
    const int64_t fo = g.senkf ? 0 : (int64_t)N * N;
    if (!wide) {
      block(false, 0, 0, true);
      block(true, 0, 1, false);
      product([&](int ln, int c, double v) {
        if (c >= N) return;
        if (ln < 64) {
          if (ln < N && !g.senkf) add(c * N + ln, v);   // K is symmetric
        } else if (ln - 64 < N) {
          add(fo + c * N + (ln - 64), v);               // F[c][ln - 64]
        }
      });
    } else {
      block(false, 0, 0, !g.senkf);
      block(false, 1, 1, false);
      for (int q = g.senkf ? 2 : 0; q < 4; ++q) {
        if (q > 0) block(q >= 2, q & 1, -1, true);
        product([&](int ln, int c, double v) {
          const int j = 64 * (q & 1) + c;
          if (ln >= N || j >= N) return;
          if (q < 2) add(j * N + ln, v);
          else add(fo + ln * N + j, v);
        });
      }
    }
    __syncthreads();   // s_w and the buffer are rewritten
  }
  krylov_end(cta);
}

// ------------------------------------------------------------------ FP32 ensembles: products on tensor cores
// The same products from pass G of krylov.cuh (U^T U and U^T V with U = w HA, V = w D, w_i = 1/sqrt(r_i), or
// 1/sqrt(s_i) for the sEnKF, whose W is U^T V; Reduced: Y~ = D + HA, so HA^T R^{-1} Y~ = F + K). A CTA forms HA
// and D of up to kChunk of its rows with the innovations' double-float rows into a buffer of its own (it
// stays in L2), then runs pass G over them. At m = 65,536, N = 64 the stage takes 0.16 ms, half of it the
// innovations' rows; the products in double-float on the CUDA cores took 0.47 ms (Reduced) and 0.37 ms
// (sEnKF), FP32-issue-bound at 12 operations per term.
constexpr int kChunk = 512;

struct GramTc {
  const float* Xf;
  const int32_t* rowptr;
  const int32_t* col;
  const double* w;
  const double* y;
  const double* r;
  const double* E;
  int emode;
  uint64_t seed, counter;
  int64_t m, rows_per;
  int N;
  bool senkf;
  const df32* rsq;
  df32* part;      // [grid][column groups][krylov_part(N)]
  df32* scratch;   // [grid][2 chunk N + chunk]: HA, D and (sEnKF) the weights of a chunk (chunk % 8 == 0)
  int64_t chunk;
  int* status;
};

template <int NT>
__global__ void __launch_bounds__(kKT, 1) gram_tc_kernel(GramTc g) {
  using L = KLayout<NT>;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_slot;
  __shared__ unsigned umax;
  KCta cta;
  krylov_begin(cta, smem, &mbar, &tmem_slot, g.status);
  const int N = g.N, t = threadIdx.x;
  if (dynamic_smem_bytes() < (unsigned)L::bytes) {
    if (t == 0) atomicOr(g.status, DS_SMEM);
  } else {
    const int ngr = (N + L::JC - 1) / L::JC;
    const int64_t row0 = imin64(g.m, blockIdx.x * g.rows_per), row1 = imin64(g.m, row0 + g.rows_per);
    df32* HA = g.scratch + (int64_t)blockIdx.x * (2 * g.chunk * N + g.chunk);
    df32* D = HA + g.chunk * N;
    df32* wsq = D + g.chunk * N;
    KrylovParams p{};
    p.N = N;
    p.HAdf = HA;
    p.Ddf = D;
    p.umax = &umax;
    int64_t c0 = row0;
    do {   // at least once: a CTA without rows writes zeros
      const int64_t c1 = imin64(row1, c0 + g.chunk);
      if (t == 0) umax = 0u;
      __syncthreads();
      innov_rows_df<float, (NT <= 64)>(g.Xf, g.rowptr, g.col, g.w, g.y, g.r, g.E, g.emode, g.seed, g.counter, N, nullptr, nullptr,
                                       nullptr, HA, D, c0, c1, t >> 5, kKT / 32, nullptr,
                                       InnovRows{nullptr, g.rsq, &umax, c0, g.senkf, wsq});
      __syncthreads();
      p.rsq = g.senkf ? wsq : g.rsq + c0;
      for (int c = 0; c < ngr; ++c)
        pass_gram<NT>(p, false, c, 0, c1 - c0, cta, g.part + ((int64_t)blockIdx.x * ngr + c) * krylov_part(N), c0 > row0);
      c0 = c1;
    } while (c0 < row1 && cta.ok);
  }
  krylov_end(cta);
}

// Fixed-order totals of the CTAs' partials, 32 consecutive entries (k, j) per CTA: G = I + K/(N-1) and
// M = I + (F + K)/(N-1), or W = F.
__global__ void __launch_bounds__(kThreads) gram_tc_sum_kernel(const df32* __restrict__ part, int grid, int N,
                                                               double* __restrict__ Gm, double* __restrict__ Mm,
                                                               double* __restrict__ W) {
  constexpr int NW = kThreads / 32;
  __shared__ double sk[NW][32], sf[NW][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
  const int NJ = min(64, N), ngr = (N + 63) / 64, k = e / N, j = e % N, c = j / 64, jl = j % 64;
  const int64_t PS = krylov_part(N);
  df32 a, f;
  if (e < N * N)
#pragma unroll 4
    for (int b = warp; b < grid; b += NW) {
      const df32* src = part + ((int64_t)b * ngr + c) * PS + k * NJ + jl;
      a = a + src[0];
      f = f + src[(int64_t)N * NJ];
    }
  sk[warp][lane] = (double)a;
  sf[warp][lane] = (double)f;
  __syncthreads();
  if (warp == 0 && e < N * N) {
    double K = 0.0, F = 0.0;
    for (int q = 0; q < NW; ++q) {
      K += sk[q][lane];
      F += sf[q][lane];
    }
    const double inv = 1.0 / (double)(N - 1), eye = k == j ? 1.0 : 0.0;
    if (W) W[e] = F;
    else {
      Gm[e] = fma(K, inv, eye);
      Mm[e] = fma(F + K, inv, eye);
    }
  }
}

// Fixed-order sum over b < nparts of part[b * pstride + e], e < count: a CTA takes 32
// consecutive e (one per lane), warp w adds b = w, w + 8, ... in order, and warp 0 adds the
// eight warp sums in warp order before handing (e, total) to store.
template <typename Store>
__device__ __forceinline__ void sum_partials(const double* __restrict__ part, int nparts,
                                             int64_t pstride, int count, Store&& store) {
  constexpr int W = kThreads / 32;
  __shared__ double wsum[W][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (e < count)
    for (int b = warp; b < nparts; b += W) s += part[(int64_t)b * pstride + e];
  wsum[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && e < count) {
    double tot = wsum[0][lane];
#pragma unroll
    for (int q = 1; q < W; ++q) tot += wsum[q][lane];
    store(e, tot);
  }
}

// G = I + sum_b part_b[0] / (N-1), M = I + sum_b part_b[1] / (N-1).
__global__ void __launch_bounds__(kThreads) reduced_sum_kernel(const double* __restrict__ part, int nparts, int N,
                                                               double* __restrict__ Gm, double* __restrict__ Mm) {
  const int NN = N * N;
  const double inv = 1.0 / (double)(N - 1);
  sum_partials(part, nparts, 2 * (int64_t)NN, 2 * NN, [&](int e, double s) {
    const int half = e / NN, ee = e % NN;
    (half == 0 ? Gm : Mm)[ee] = s * inv + ((ee / N) == (ee % N) ? 1.0 : 0.0);
  });
}

// sEnKF: W = sum_b part_b[0] (= HA^T diag^{-1} D).
__global__ void __launch_bounds__(kThreads) senkf_sum_kernel(const double* __restrict__ part, int nparts, int N,
                                                             double* __restrict__ W) {
  sum_partials(part, nparts, 2 * (int64_t)N * N, N * N, [&](int e, double s) { W[e] = s; });
}

// One CTA per column j of M: CG for G v_j = m_j (FP64), G staged in shared memory; V is [N][N] row-major
// (V[k][j]). The step has one product and one round of sums: with g = G r, (p, G p) =
// (r, g) - beta^2 (p, G p)_old and G p = g + beta (G p)_old. What bounds it is the FP64 unit (2 per clock
// per SM; a warp's instruction holds its scheduler's unit for about 64 cycles): N^2 DFMAs are 2,048
// cycles at N = 64, so the scalars run on one warp, the reciprocal for beta beside the product, and the sums of a
// step share one shuffle tree per warp. 28 steps at N = 64 take 105 us; the two-reduction form, with every
// warp folding every sum and dividing, took 128.
__global__ void __launch_bounds__(kThreads) reduced_cg_kernel(
    const double* __restrict__ Gm, const double* __restrict__ Mm, int N, double tol, int max_iter,
    int fixed_iters, double* __restrict__ V, int* __restrict__ col_iters,
    double* __restrict__ col_relres, double* __restrict__ col_true, int* __restrict__ status) {
  extern __shared__ __align__(16) double sm[];
  // G with row stride N + 1: lanes on consecutive rows k then read distinct banks
  const int ld = N + 1;
  double* sG = sm;                 // N x (N + 1)
  double* su = sG + N * ld;        // N: the product's operand
  double* spart = su + N;          // [kThreads] partial row sums of the product
  __shared__ double red[2][4], sc[5];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int j = blockIdx.x;
  // the product: thread t forms the partial sum of row k = t % NP over columns l = g, g + P, ...
  // (g = t / NP, P = kThreads / NP groups); thread k adds the P partials of row k in order
  const int NP = N <= 64 ? 64 : 128, P = kThreads / NP, NW = NP / 32;
  for (int e = t; e < N * N; e += kThreads) sG[(e / N) * ld + e % N] = Gm[e];
  const bool own = t < N;          // thread k keeps row k of the vectors
  const double b = own ? Mm[t * N + j] : 0.0;
  double x = 0.0, r = b, p = 0.0, h = 0.0;
  if (own) su[t] = b;
  __syncthreads();
  auto product = [&]() -> double {
    const int k = t % NP, g = t / NP;
    double a0 = 0.0, a1 = 0.0;
    if (k < N) {
      int l = g;
      for (; l + P < N; l += 2 * P) {
        a0 = fma(sG[k * ld + l], su[l], a0);
        a1 = fma(sG[k * ld + l + P], su[l + P], a1);
      }
      if (l < N) a0 = fma(sG[k * ld + l], su[l], a0);
    }
    spart[t] = a0 + a1;
    __syncthreads();
    double s = 0.0;
    if (own) {
      s = spart[t];
      for (int g2 = 1; g2 < P; ++g2) s += spart[g2 * NP + t];
    }
    return s;
  };
  // totals of two values over the CTA's owners, into red (warp w's part in red[.][w])
  auto fold = [&](double u, double v) {
    if (warp < NW) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        u += __shfl_xor_sync(0xffffffffu, u, o);
        v += __shfl_xor_sync(0xffffffffu, v, o);
      }
      if (lane == 0) {
        red[0][warp] = u;
        red[1][warp] = v;
      }
    }
    __syncthreads();
  };
  auto folded = [&](int q) {
    double s = red[q][0];
    for (int w = 1; w < NW; ++w) s += red[q][w];
    return s;
  };
  const bool fixed = fixed_iters > 0;
  const int limit = fixed ? fixed_iters : max_iter;
  double bn2 = 0.0, rr = 0.0, pq = 0.0, stop2 = 0.0;   // warp 0's
  int it = 0;
  for (;;) {
    // one thread divides for the next beta beside the product
    if (it > 0 && t == kThreads - 1) sc[3] = 1.0 / sc[4];
    const double g = product();
    fold(r * r, r * g);
    if (warp == 0) {
      const double r2 = folded(0), rg = folded(1);
      if (it == 0) {
        // |r| <= tol |b| compared in squares, with tol shrunk by 4 ulps so that a stop always gives
        // sqrt(rr / bn2) <= tol for the residual reported below
        const double tol_s = tol * (1.0 - 4.0 * 2.220446049250313e-16);
        bn2 = r2;
        stop2 = tol_s * tol_s * bn2;
      }
      bool go = it < limit && (it == 0 || fixed ? r2 > 0.0 : r2 > stop2);
      // (a NaN in G or m_j fails the comparisons at step 0; an infinity makes q below non-finite)
      if (!go && !isfinite(r2) && lane == 0) atomicOr(status, DS_NONFINITE);
      const double be = go && it > 0 ? r2 * sc[3] : 0.0;
      double al = 0.0;
      if (go) {
        const double q = fma(-be * be, pq, rg);
        if (!(q > 0.0) || !isfinite(q)) {
          if (lane == 0) atomicOr(status, isfinite(q) ? DS_BREAKDOWN : DS_NONFINITE);
          go = false;
        } else {
          pq = q;
          al = r2 / q;
        }
      }
      rr = r2;
      if (lane == 0) {
        sc[0] = al;
        sc[1] = be;
        sc[2] = go ? 1.0 : 0.0;
        sc[4] = r2;
      }
    }
    __syncthreads();
    if (sc[2] == 0.0) break;
    const double al = sc[0], be = sc[1];
    if (own) {
      p = fma(be, p, r);
      h = fma(be, h, g);
      x = fma(al, p, x);
      r = fma(-al, h, r);
      su[t] = r;
    }
    ++it;
    __syncthreads();
  }
  // true residual m_j - G v_j (FP64)
  if (own) su[t] = x;
  __syncthreads();
  const double d = b - product();
  fold(own ? d * d : 0.0, 0.0);
  if (own) V[t * N + j] = x;
  if (t == 0) {
    const double tr2 = folded(0);
    col_iters[j] = it;
    const bool fin = isfinite(bn2) && isfinite(rr);
    const double rel = !fin ? (double)NAN : bn2 > 0.0 ? sqrt(rr / bn2) : 0.0;
    col_relres[j] = rel;
    col_true[j] = !fin ? (double)NAN : bn2 > 0.0 ? sqrt(tr2 / bn2) : 0.0;
    if (!fixed && !(rel <= tol)) atomicOr(status, DS_NOT_CONVERGED);
  }
}

// ------------------------------------------------------------------ launchers
int reduced_grid(const enkf_handle_s* h) {
  const bool f64 = h->cfg.precision == ENKF_FP64;
  const int64_t rows = f64 ? 32 : kKR;   // a tile
  return (int)std::max<int64_t>(1, std::min<int64_t>((h->cfg.m + rows - 1) / rows, h->sms));
}
static int64_t gram_rows_per(const enkf_handle_s* h) { return (h->cfg.m + reduced_grid(h) - 1) / reduced_grid(h); }
// (a multiple of 8: every CTA's buffers then begin on a 16-byte boundary, as the rows' stores need)
static int64_t gram_chunk(const enkf_handle_s* h) { return std::min<int64_t>(kChunk, (gram_rows_per(h) + 7) / 8 * 8); }
size_t gram64_scratch_bytes(const enkf_handle_s* h) { return sizeof(double) * (size_t)reduced_grid(h) * 2 * kDR * h->cfg.N; }
size_t gram_tc_part_bytes(const enkf_handle_s* h) {
  return sizeof(df32) * (size_t)krylov_part(h->cfg.N) * ((h->cfg.N + 63) / 64) * reduced_grid(h);
}
size_t gram_tc_scratch_bytes(const enkf_handle_s* h) {
  return sizeof(df32) * (size_t)reduced_grid(h) * gram_chunk(h) * (2 * h->cfg.N + 1);
}

template <int NT>
static cudaError_t gram_tc_launch(const GramTc& g, int grid, cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(gram_tc_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, KLayout<NT>::bytes);
  if (e != cudaSuccess) return e;
  gram_tc_kernel<NT><<<grid, kKT, KLayout<NT>::bytes, s>>>(g);
  return cudaGetLastError();
}
static cudaError_t launch_gram_tc(enkf_handle_s* h, const void* Xf, const double* y, const double* E, int emode,
                                  uint64_t seed, uint64_t counter) {
  const auto& c = h->cfg;
  auto& ws = h->ws;
  const GramTc g{static_cast<const float*>(Xf), ws.rowptr, ws.col, ws.w, y, ws.r, E, emode, seed, counter, c.m,
                 gram_rows_per(h), c.N, c.variant == ENKF_SENKF, static_cast<const df32*>(ws.rsq),
                 static_cast<df32*>(ws.kpart), static_cast<df32*>(ws.HAdf), gram_chunk(h), ws.status};
  if (c.N <= 32) return gram_tc_launch<32>(g, reduced_grid(h), h->stream);
  if (c.N <= 64) return gram_tc_launch<64>(g, reduced_grid(h), h->stream);
  return gram_tc_launch<128>(g, reduced_grid(h), h->stream);
}

static cudaError_t launch_gram64(enkf_handle_s* h, const void* Xf, const double* y, const double* E, int emode,
                                 uint64_t seed, uint64_t counter) {
  const auto& c = h->cfg;
  auto& ws = h->ws;
  const Gram64 g{static_cast<const double*>(Xf), ws.rowptr, ws.col, ws.w, y, ws.r, E, emode, seed, counter, c.m,
                 gram_rows_per(h), c.N, c.variant == ENKF_SENKF, ws.Tpart, static_cast<double*>(ws.HAdf), ws.status};
  const cudaError_t e = cudaFuncSetAttribute(gram64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Gram64Smem::bytes);
  if (e != cudaSuccess) return e;
  gram64_kernel<<<reduced_grid(h), kDT, Gram64Smem::bytes, h->stream>>>(g);
  return cudaGetLastError();
}

cudaError_t launch_gram_stage(enkf_handle_s* h, const void* Xf, const double* y, const double* E,
                              int emode, uint64_t seed, uint64_t counter) {
  const auto& c = h->cfg;
  auto& ws = h->ws;
  const bool senkf = c.variant == ENKF_SENKF;
  cudaError_t e = cudaMemsetAsync(ws.status, 0, 4 * sizeof(int32_t), h->stream);
  if (senkf) {   // no solve: the per-column statistics read back as 0 iterations, residual 0
    if (e == cudaSuccess) e = cudaMemsetAsync(ws.col_iters, 0, sizeof(int32_t) * c.N, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws.col_relres, 0, sizeof(double) * c.N, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws.col_true, 0, sizeof(double) * c.N, h->stream);
  }
  if (e != cudaSuccess) return e;
  return c.precision == ENKF_FP64 ? launch_gram64(h, Xf, y, E, emode, seed, counter)
                                  : launch_gram_tc(h, Xf, y, E, emode, seed, counter);
}

cudaError_t launch_nxn_stage(enkf_handle_s* h) {
  const auto& c = h->cfg;
  auto& ws = h->ws;
  const int grid = reduced_grid(h);
  const bool f64 = c.precision == ENKF_FP64;
  if (!f64) {
    const bool senkf = c.variant == ENKF_SENKF;
    gram_tc_sum_kernel<<<(c.N * c.N + 31) / 32, kThreads, 0, h->stream>>>(
        static_cast<const df32*>(ws.kpart), grid, c.N, ws.Tred, ws.Wacc, senkf ? ws.W : nullptr);
    if (senkf) return cudaGetLastError();
  } else if (c.variant == ENKF_SENKF) {
    const int NN = c.N * c.N;
    senkf_sum_kernel<<<(NN + 31) / 32, kThreads, 0, h->stream>>>(ws.Tpart, grid, c.N, ws.W);
    return cudaGetLastError();
  }
  double* Gm = ws.Tred;            // N x N
  double* Mm = ws.Wacc;            // N x N
  const int NN2 = 2 * c.N * c.N;
  if (f64) reduced_sum_kernel<<<(NN2 + 31) / 32, kThreads, 0, h->stream>>>(ws.Tpart, grid, c.N, Gm, Mm);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // (the limit belongs to the kernel: set for the largest N, also between another thread's limit and launch)
  auto bytes = [](size_t N) { return sizeof(double) * (N * (N + 1) + N + kThreads); };
  const size_t smem = bytes(c.N);
  e = cudaFuncSetAttribute(reduced_cg_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(128));
  if (e != cudaSuccess) return e;
  reduced_cg_kernel<<<c.N, kThreads, smem, h->stream>>>(Gm, Mm, c.N, c.tol, c.max_iter, c.fixed_iters,
                                                       ws.W, ws.col_iters, ws.col_relres, ws.col_true,
                                                       ws.status);
  return cudaGetLastError();
}

cudaError_t launch_reduced(enkf_handle_s* h, const void* Xf, const double* y, const double* E,
                           int emode, uint64_t seed, uint64_t counter) {
  cudaError_t e = launch_gram_stage(h, Xf, y, E, emode, seed, counter);
  return e != cudaSuccess ? e : launch_nxn_stage(h);
}

}  // namespace enkf
