// CG on S Z = D for FP64 ensembles of up to 64 members, its products on the tensor cores.
//
// The recurrences are those of solve_body.cuh (one reduction per step: T = HA^T p carried as
// T_{k+1} = HA^T z_{k+1} + beta_k T_k, (p, S p) = ||T||^2/(N-1) + sum r_i p_i^2), in FP64. Its two products per step,
// u = HA T and HA^T z, took 0.87 of the chip's FP64 rate at m = 16,384, N = 64: 267 us per step. Here they are
// products of FP64 operands in exact digits (slices64.cuh), and what is left for the FP64 unit are the
// step's nine operations per entry.
//
// Persistent cooperative kernel, one CTA per SM. A CTA walks its rows in tiles of up to 64:
//   HA tile    digits per row (scaled by the row's largest entry), used twice: K-major over the members as the
//              operand of u, MN-major as the operand of HA^T z
//   u = HA T   arrives as D[j][i]: a thread owns one column j and eight rows. T is operand A in two copies, so
//              that all 128 lanes carry work (the upper lanes take the rows 32 to 63 of a tile)
//   z          each thread's eight rows of its column, times the rows' scales, scaled by the column's
//              largest entry in the tile; in halves of 32 rows (shared memory)
// and every step ends in the sum of the CTAs' partials and two grid barriers, as before.
#include <algorithm>

#include "common.cuh"
#include "slices64.cuh"

namespace enkf {

constexpr int kQT = 512, kQR = 64;

struct Solve64Params {
  int64_t m;
  int N;
  const double* HA;    // [m][N]
  const double* D;
  const double* r;
  double* X;           // [m][N]: solution, residual, direction
  double* Res;
  double* P;
  double* part;        // [G][N N + 4 N]: HA^T z (column by column) and the column sums of the CTAs
  double* Tred;        // [N N + 4 N]
  double* Told[2];     // [N N] each: T of the steps, alternating (W and another array, both free during the steps)
  double* W;
  double tol;
  int max_iter, fixed_iters, true_residual;
  int* col_iters;
  double* col_relres;
  double* col_true;
  int* status;
  unsigned* bar;
  unsigned long long* prof;
};

struct Solve64Smem {
  static constexpr int TP = 128 * 64 * 2, HP = kQR * 64 * 2, ZP = 64 * 32 * 2;   // bytes per digit
  static constexpr int off_h = kDg * TP, off_z = off_h + kDg * HP, off_max = off_z + kDg * ZP;
  static constexpr int off_row = off_max + 8 * 64 * 4;   // exponents: rows of HA, columns of T and of z
  static constexpr int off_colt = off_row + 64 * 4, off_colz = off_colt + 64 * 4;
  static constexpr int off_int = off_colz + 64 * 4;      // go, iterations, ended
  static constexpr int off_r = off_int + 3 * 64 * 4;     // r and 1/r of a tile
  static constexpr int off_col = off_r + 2 * 64 * 8;     // al, be, gamma, den, |b|^2, |r|^2
  static constexpr int off_sum = off_col + 6 * 64 * 8;   // [2][64]
  static constexpr int bytes = off_sum + 2 * 64 * 8;
  static_assert(bytes <= 226 * 1024, "shared memory");
  static_assert(4 * 8 * 64 * 8 <= off_h && kQT * 8 <= off_h, "column sums and reduction lie over the T operand");
};

// x 2^(E - 1022)
__device__ __forceinline__ double dg_times(double x, int E) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 2047, e = ex + E - 1022;
  if (ex == 0 || e <= 0) return 0.0;
  if (E == 2047 || ex == 2047) return __longlong_as_double(0x7FF8000000000000ll);
  if (e >= 2047) return __hiloint2double((hi & 0x80000000) | 0x7FF00000, 0);
  return __hiloint2double(hi + ((E - 1022) << 20), __double2loint(x));
}

enum : int { S64_INIT, S64_STEP, S64_SUM, S64_RESID };

template <bool PC>
__global__ void __launch_bounds__(kQT, 1) solve64_kernel(Solve64Params p) {
  using L = Solve64Smem;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_slot;
  KCta cta;
  krylov_begin(cta, smem, &mbar, &tmem_slot, p.status);
  if (dynamic_smem_bytes() < (unsigned)L::bytes) {
    if (threadIdx.x == 0) atomicOr(p.status, DS_SMEM);
    krylov_end(cta);
    return;
  }
  GridBarrier bar{p.bar, reinterpret_cast<int*>(p.bar + 1), p.status, gridDim.x, 0u};
  const int N = p.N, G = gridDim.x, b = blockIdx.x, t = threadIdx.x, lane = t & 31;
  const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  const int NN = N * N, NE = NN + 4 * N;
  int* s_max = reinterpret_cast<int*>(smem + L::off_max);
  int* s_row = reinterpret_cast<int*>(smem + L::off_row);
  int* s_colt = reinterpret_cast<int*>(smem + L::off_colt);
  int* s_colz = reinterpret_cast<int*>(smem + L::off_colz);
  int* s_go = reinterpret_cast<int*>(smem + L::off_int);
  int* s_it = s_go + 64;
  int* s_end = s_it + 64;
  double* s_r = reinterpret_cast<double*>(smem + L::off_r);   // r, then 1/r
  double* s_al = reinterpret_cast<double*>(smem + L::off_col);
  double* s_be = s_al + 64;
  double* s_gam = s_be + 64;
  double* s_den = s_gam + 64;
  double* s_bn2 = s_den + 64;
  double* s_gm = s_bn2 + 64;
  double* s_sum = reinterpret_cast<double*>(smem + L::off_sum);
  double* scratch = reinterpret_cast<double*>(smem);          // over the T operand, between steps
  const uint32_t base = smem_addr(smem), aH = base + L::off_h, aZ = base + L::off_z, lead = warp == 0 ? elect_lane() : 0u;
  const double inv = 1.0 / (double)(N - 1);
  const bool fixed = p.fixed_iters > 0;
  const int64_t rows_per = (p.m + G - 1) / G, row0 = imin64(p.m, b * rows_per), row1 = imin64(p.m, row0 + rows_per);
  const int nrows = (int)(row1 - row0), tiles = (nrows + kQR - 1) / kQR;
  const int per = tiles > 0 ? ((nrows + tiles - 1) / tiles + 7) / 8 * 8 : 0;
  double* part = p.part + (int64_t)b * NE;
  int par = 0;   // p.Told[par] takes this step's T
  const bool prof = p.prof != nullptr && b == 0 && t == 0;
  unsigned long long ph[PH_COUNT] = {0, 0, 0, 0, 0, 0, 0, 0}, tp = prof ? global_ns() : 0ull;
  auto tick = [&](int slot) {
    if (prof) {
      const unsigned long long now = global_ns();
      ph[slot] += now - tp;
      tp = now;
    }
  };
  // items of a 64 x 64 operand: row ir, columns [ic, ic + 8)
  const int ir = warp / 2 * 8 + (lane & 7), ic = warp % 2 * 32 + (lane >> 3) * 8;
  // entries: column j, rows [r0, r0 + 8) of a tile
  const int qd = warp & 3, sub = warp >> 2, ln = 32 * qd + lane, copy = qd >> 1, j = ln & 63, grp = copy * 4 + sub, r0 = 8 * grp;
  const bool live = j < N;
  if (t < 64) {
    s_it[t] = 0;
    s_end[t] = t >= N;
    s_go[t] = 0;
  }
  __syncthreads();

  // One pass over the CTA's rows. first: no step has been taken (residual D, no solution or direction yet).
  auto pass = [&](int mode, bool first) {
    const bool has_u = mode == S64_STEP || mode == S64_RESID, has_z = mode != S64_RESID;
    double q0 = 0.0, q1 = 0.0, q2 = 0.0, q3 = 0.0;   // the thread's share of the column sums
    for (int tile = 0; tile < tiles && cta.ok; ++tile) {
      const int64_t c0 = row0 + (int64_t)tile * per;
      const int rows = (int)imin64(per, row1 - c0);   // (may be <= 0 for a last tile: zeros)
      // the HA tile
      {
        double x[8];
        int mx = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          x[e] = (ir < rows && ic + e < N) ? p.HA[(c0 + ir) * N + ic + e] : 0.0;
          mx = max(mx, dg_abs_hi(x[e]));
        }
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
        if (lane < 8) s_max[warp % 2 * 64 + ir] = mx;
        if (t < kQR) {
          const double ri = t < rows ? p.r[c0 + t] : 1.0;
          s_r[t] = ri;
          s_r[64 + t] = PC ? 1.0 / ri : 1.0;
        }
        tc_fence_before();
        __syncthreads();
        const int er = dg_exp(max(s_max[ir], s_max[64 + ir]));
        if (warp % 2 == 0 && lane < 8) s_row[ir] = er;
        const int E[8] = {er, er, er, er, er, er, er, er};
        Digits8 dg;
        dg.make(x, E);
        dg.store(smem + L::off_h + (ir >> 3) * 1024 + (ic >> 3) * 128 + (ir & 7) * 16, L::HP);
      }
      fence_async_smem();
      __syncthreads();
      if (has_u && warp == 0) {
        tc_fence_after();
        dg_issue<false, false, L::TP, 256, L::HP, 256>(cta.tmem, umma_desc(base, 128, 1024), umma_desc(aH, 128, 1024), (N + 15) / 16,
                                                       false, cta.mbar, lead);
      }
      // this thread's entries, in flight behind the product
      const int64_t e0 = (c0 + r0) * N + j;
      const int nr = live ? max(0, min(8, rows - r0)) : 0;
      double z[8], pv[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const bool in = q < nr;
        const int64_t at = e0 + (int64_t)q * N;
        if (mode == S64_SUM) z[q] = in && !first ? p.X[at] : 0.0;
        else if (mode == S64_STEP && !first) z[q] = in ? p.Res[at] : 0.0;   // the residual, until the product is there
        else z[q] = in ? p.D[at] : 0.0;
        pv[q] = 0.0;
        if (mode == S64_STEP && !first) pv[q] = in ? p.P[at] : 0.0;
        if (mode == S64_RESID) pv[q] = in ? p.X[at] : 0.0;
      }
      if (has_u) k_wait(cta);
      const int ea = s_colt[j];
      if (mode == S64_STEP) {
        const double al = s_al[j], be = s_be[j];
        const bool go = s_go[j] != 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float lv[kDl][4];
          tmem_ld_levels<kDl, 4>(cta.tmem + ((uint32_t)(32 * qd) << 16) + r0 + 4 * h, 64, lv);
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) {
            const int q = 4 * h + q4;
            if (q >= nr) continue;
            const int64_t at = e0 + (int64_t)q * N;
            if (!go) {   // the column has ended
              if (first) {
                p.X[at] = 0.0;
                p.Res[at] = z[q];
              }
              z[q] = 0.0;
              continue;
            }
            const double ri = s_r[r0 + q], u = dg_value(dg_join(lv, q4), ea, s_row[r0 + q]);
            const double zo = PC ? z[q] * s_r[64 + r0 + q] : z[q];
            const double pn = first ? zo : fma(be, pv[q], zo);
            const double sv = fma(u, inv, ri * pn);
            const double rn = fma(-al, sv, z[q]);
            const double zn = PC ? rn * s_r[64 + r0 + q] : rn, rz = ri * zn;
            p.X[at] = first ? al * pn : fma(al, pn, p.X[at]);
            p.Res[at] = rn;
            p.P[at] = pn;
            if (PC) q0 = fma(rn, zn, q0);
            q1 = fma(rn, rn, q1);
            q2 = fma(rz, zn, q2);
            q3 = fma(rz, pn, q3);
            z[q] = zn;
          }
        }
      } else if (mode == S64_RESID) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float lv[kDl][4];
          tmem_ld_levels<kDl, 4>(cta.tmem + ((uint32_t)(32 * qd) << 16) + r0 + 4 * h, 64, lv);
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) {
            const int q = 4 * h + q4;
            if (q >= nr) continue;
            const double u = dg_value(dg_join(lv, q4), ea, s_row[r0 + q]);
            const double rt = z[q] - fma(u, inv, s_r[r0 + q] * pv[q]);
            q0 = fma(rt, rt, q0);
          }
        }
      } else if (mode == S64_INIT) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (q >= nr) continue;
          const double d = z[q], zn = PC ? d * s_r[64 + r0 + q] : d;
          if (PC) q0 = fma(d, zn, q0);
          q1 = fma(d, d, q1);
          q2 = fma(s_r[r0 + q] * zn, zn, q2);
          z[q] = zn;
        }
      } else if (first) {   // S64_SUM before any step: the solution is zero
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q < nr) p.X[e0 + (int64_t)q * N] = 0.0;
      }
      if (!has_z) {
        tc_fence_before();
        __syncthreads();   // the tile's operands are rewritten
        continue;
      }
      // HA^T z: the rows' scales go to z
      int mx = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        z[q] = q < nr ? dg_times(z[q], s_row[r0 + q]) : 0.0;
        mx = max(mx, dg_abs_hi(z[q]));
      }
      s_max[grp * 64 + j] = mx;
      tc_fence_before();
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 8; ++q) mx = max(mx, s_max[q * 64 + j]);
      const int ez = dg_exp(mx);
      if (grp == 0) s_colz[j] = ez;
      const int E[8] = {ez, ez, ez, ez, ez, ez, ez, ez};
      Digits8 dg;
      dg.make(z, E);
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        if (half == 1 && rows <= 32) break;
        if (copy == half) dg.store(smem + L::off_z + (j >> 3) * 512 + sub * 128 + (j & 7) * 16, L::ZP);
        fence_async_smem();
        __syncthreads();
        if (warp == 0) {
          tc_fence_after();
          dg_issue<true, false, L::HP, 2 * 1024, L::ZP, 256>(cta.tmem, umma_desc(aH + half * 4096, 1024, 128), umma_desc(aZ, 128, 512),
                                                             max(1, (min(32, rows - 32 * half) + 15) / 16), half > 0, cta.mbar, lead);
        }
        k_wait(cta);
      }
      if (qd < 2) {   // lanes k < 64
#pragma unroll 1
        for (int c = sub * 16; c < min(N, sub * 16 + 16); c += 4) {
          float lv[kDl][4];
          tmem_ld_levels<kDl, 4>(cta.tmem + ((uint32_t)(32 * qd) << 16) + c, 64, lv);
          if (ln < N)
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (c + q < N) {
                const double v = dg_value(dg_join(lv, q), 1022, s_colz[c + q]);
                double* at = part + (c + q) * N + ln;
                *at = tile > 0 ? *at + v : v;
              }
        }
      }
    }
    if (tiles == 0 && has_z)
      for (int e = t; e < NN; e += kQT) part[e] = 0.0;
    // column sums over the eight row groups
    __syncthreads();
    scratch[(0 * 8 + grp) * 64 + j] = PC || mode == S64_RESID ? q0 : q1;
    scratch[(1 * 8 + grp) * 64 + j] = q1;
    scratch[(2 * 8 + grp) * 64 + j] = q2;
    scratch[(3 * 8 + grp) * 64 + j] = q3;
    __syncthreads();
    if (t < 256 && (t & 63) < N) {
      double s = 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q) s += scratch[((t >> 6) * 8 + q) * 64 + (t & 63)];
      part[NN + (t >> 6) * N + (t & 63)] = s;
    }
  };
  // sums of the CTAs' partials in a fixed order, each CTA a slice of them, between two barriers
  auto reduce = [&]() -> bool {
    if (!bar.sync()) return false;
    tick(PH_BAR1);
    const int chunk = (NE + G - 1) / G, e0 = min(NE, b * chunk), n = min(NE, e0 + chunk) - e0;
    if (n > 0) {
      const int parts = max(1, kQT / n);
      for (int e = e0 + t % n; t / n < parts && e < e0 + n; e += kQT) {   // (one turn when n <= kQT)
        const int w = n <= kQT ? t / n : 0;
        double s = 0.0;
        const int q1 = (int)((int64_t)(w + 1) * G / parts);
#pragma unroll 4
        for (int q = (int)((int64_t)w * G / parts); q < q1; ++q) s += __ldcg(p.part + (int64_t)q * NE + e);
        if (n <= kQT) scratch[t] = s;
        else p.Tred[e] = s;
      }
      __syncthreads();
      if (n <= kQT && t < n) {
        double s = scratch[t];
        for (int w = 1; w < parts; ++w) s += scratch[w * n + t];
        p.Tred[e0 + t] = s;
      }
    }
    tick(PH_RED);
    const bool ok = bar.sync();
    tick(PH_BAR2);
    return ok;
  };
  // T (+)= beta T_old as operand A, its column norms into s_sum (column ir of T is row ir)
  auto stage_t = [&](bool carry, bool keep) {
    double x[8], n2 = 0.0;
    int mx = 0;
    const double be = carry && ir < N ? s_be[ir] : 0.0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const bool in = ir < N && ic + e < N;
      const int at = ir * N + ic + e;
      x[e] = in ? __ldcg(p.Tred + at) : 0.0;
      if (carry && in) x[e] = fma(be, __ldcg(p.Told[par ^ 1] + at), x[e]);
      if (keep && in && t % G == b) p.Told[par][at] = x[e];   // (every CTA forms all of T and stores its share)
      n2 = fma(x[e], x[e], n2);
      mx = max(mx, dg_abs_hi(x[e]));
    }
#pragma unroll
    for (int o = 8; o <= 16; o <<= 1) {
      n2 += __shfl_xor_sync(0xffffffffu, n2, o);
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane < 8) {
      s_sum[warp % 2 * 64 + ir] = n2;
      s_max[warp % 2 * 64 + ir] = mx;
    }
    __syncthreads();
    const int er = dg_exp(max(s_max[ir], s_max[64 + ir]));
    if (warp % 2 == 0 && lane < 8) s_colt[ir] = er;
    const int E[8] = {er, er, er, er, er, er, er, er};
    Digits8 dg;
    dg.make(x, E);
    unsigned char* at = smem + (ir >> 3) * 1024 + (ic >> 3) * 128 + (ir & 7) * 16;
    dg.store(at, L::TP);
    dg.store(at + 8192, L::TP);
  };
  // every CTA alike: the column sums of the step before -> beta, T, (p, S p), alpha and who goes on
  bool ok = true;
  int steps = 0;
  tick(PH_SETUP);
  pass(S64_INIT, true);
  tick(PH_PASS);
  ok = reduce();
  while (ok) {
    if (t < N) {
      const double g1 = __ldcg(p.Tred + NN + t), gm = __ldcg(p.Tred + NN + N + t), g3 = __ldcg(p.Tred + NN + 2 * N + t);
      if (steps == 0) {
        s_bn2[t] = gm;
        s_den[t] = g3;
        s_gam[t] = g1;
        s_gm[t] = gm;
        s_be[t] = 0.0;
      } else if (!s_end[t]) {
        const double be = g1 / s_gam[t];
        s_den[t] = fma(be, fma(be, s_den[t], 2.0 * __ldcg(p.Tred + NN + 3 * N + t)), g3);
        s_gam[t] = g1;
        s_gm[t] = gm;
        s_be[t] = be;
      }
    }
    __syncthreads();
    stage_t(steps > 0, true);
    par ^= 1;
    int go = 0;
    if (t < N) {
      if (!s_end[t]) {
        const double gm = s_gm[t], itm = p.tol * (1.0 - 4.0 * 2.220446049250313e-16);
        int bad = 0;
        go = s_it[t] < (fixed ? p.fixed_iters : p.max_iter) && (steps > 0 || gm > 0.0);
        if (go && !isfinite(gm)) { bad = DS_NONFINITE; go = 0; }
        else if (go && steps > 0 && (fixed ? gm == 0.0 : gm <= itm * itm * s_bn2[t])) go = 0;
        if (go) {
          const double pq = fma(s_sum[t] + s_sum[64 + t], inv, s_den[t]);
          if (!isfinite(pq)) { bad = DS_NONFINITE; go = 0; }
          else if (pq <= 0.0) { bad = DS_BREAKDOWN; go = 0; }
          else s_al[t] = s_gam[t] / pq;
        }
        if (bad && b == 0) atomicOr(p.status, bad);
        if (go) ++s_it[t];
        else s_end[t] = 1;
      }
      s_go[t] = go;
    }
    fence_async_smem();
    const int any = __syncthreads_or(go);
    tick(PH_SCAL);
    if (!any) break;
    pass(S64_STEP, steps == 0);
    ++steps;
    tick(PH_PASS);
    ok = reduce() && cta.ok;
  }
  // ---- W = HA^T Z/(N-1) and the true residual D - S Z
  if (ok) {
    pass(S64_SUM, steps == 0);
    ok = reduce() && cta.ok;
  }
  double rel_true = -1.0;
  if (ok) {
    for (int e = b * kQT + t; e < NN; e += G * kQT) p.W[(int64_t)(e % N) * N + e / N] = __ldcg(p.Tred + e) * inv;
    if (p.true_residual) {
      stage_t(false, false);
      fence_async_smem();
      __syncthreads();
      pass(S64_RESID, false);
      ok = bar.sync() && cta.ok;
      if (ok && b == 0) {
        const int c = t & 63, w = t >> 6;
        double s = 0.0;
        if (c < N)
          for (int q = w; q < G; q += 8) s += __ldcg(p.part + (int64_t)q * NE + NN + c);
        scratch[t] = s;
        __syncthreads();
        if (t < N) {
          for (int q = 1; q < 8; ++q) s += scratch[q * 64 + t];
          const bool fin = isfinite(s_bn2[t]) && isfinite(s);
          if (!fin) atomicOr(p.status, DS_NONFINITE);
          rel_true = !fin ? (double)NAN : (s_bn2[t] > 0.0 ? sqrt(s / s_bn2[t]) : 0.0);
        }
      }
    }
  }
  tick(PH_REFRESH);
  if (b == 0) {
    if (t < N) {
      const double dn2 = s_bn2[t], gm = s_gm[t];
      p.col_iters[t] = s_it[t];
      p.col_relres[t] = dn2 > 0.0 ? sqrt(gm / dn2) : 0.0;
      p.col_true[t] = rel_true;
      if (!fixed && ok && !(dn2 == 0.0 || sqrt(gm) <= p.tol * sqrt(dn2))) atomicOr(p.status, DS_NOT_CONVERGED);
    }
    if (t == 0) p.status[1] = p.true_residual ? 1 : 0;
    if (prof)
      for (int q = 0; q < PH_COUNT; ++q) p.prof[q] = ph[q];
  }
  krylov_end(cta);
}

// Whether FP64 CG ends before rounding decides where it goes. Preconditioned by R, or with R a multiple of the
// identity, it sees at most N + 1 distinct eigenvalues and takes some 25 steps to 1e-8 (m = 16,384, N = 64): two
// evaluation orders then agree to 1e-13. (With few rows per member it takes more, 38 at m = 438, N = 66, and
// half a unit in HA's last place moves the analysis by up to 1e-8 here too, at the same distance from the exact
// one: results of this route and of the persistent solve agree to tol there, 4e-9.) Without, a varying R spreads the spectrum: 90 steps, the recurrences
// lose their orthogonality, and inputs that differ in the last bit give analyses that differ by as much as
// the tolerance leaves, 2.5e-8. Such an analysis keeps the persistent solve of solve_body.cuh and with it its results.
bool steady_fp64(const enkf_handle_s* h) { return h->cfg.precondition != 0 || h->r_const; }

// FP64, up to 64 members
bool solve64_config(const enkf_handle_s* h) {
  const enkf_config& c = h->cfg;
  return c.variant == ENKF_CGD && c.precision == ENKF_FP64 && c.N <= 64 && steady_fp64(h);
}

static void* solve64_fn(bool pc) { return pc ? (void*)solve64_kernel<true> : (void*)solve64_kernel<false>; }

cudaError_t plan_solve64(enkf_handle_s* h) {
  const cudaError_t e = cudaFuncSetAttribute(solve64_fn(h->cfg.precondition != 0), cudaFuncAttributeMaxDynamicSharedMemorySize, Solve64Smem::bytes);
  if (e != cudaSuccess) return e;
  // one CTA per SM (it holds the SM's tensor memory), 32 rows or more each
  int G = (int)std::min<int64_t>(h->sms, std::max<int64_t>(1, (h->cfg.m + 31) / 32));
  if (h->cfg.grid_blocks > 0) G = std::min(h->cfg.grid_blocks, h->sms);
  h->launch.G = G;
  h->launch.NT = h->cfg.N <= 32 ? 32 : 64;
  h->launch.smem = Solve64Smem::bytes;
  return cudaSuccess;
}

cudaError_t launch_solve64(enkf_handle_s* h) {
  const auto& c = h->cfg;
  auto& ws = h->ws;
  Solve64Params p{};
  p.m = c.m;
  p.N = c.N;
  p.HA = ws.HA64;
  p.D = ws.D;
  p.r = ws.r;
  p.X = ws.Z;
  p.Res = static_cast<double*>(ws.Res);
  p.P = static_cast<double*>(ws.P);
  p.part = ws.Tpart;
  p.Tred = ws.Tred;
  p.Told[0] = ws.W;
  p.Told[1] = ws.Wacc;
  p.W = ws.W;
  p.tol = c.tol;
  p.max_iter = c.max_iter;
  p.fixed_iters = c.fixed_iters;
  p.true_residual = c.true_residual;
  p.col_iters = ws.col_iters;
  p.col_relres = ws.col_relres;
  p.col_true = ws.col_true;
  p.status = ws.status;
  p.bar = ws.bar;
  p.prof = h->prof_enabled ? ws.prof : nullptr;
  cudaError_t e = cudaMemsetAsync(ws.bar, 0, 4 * sizeof(unsigned), h->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(ws.status, 0, 4 * sizeof(int32_t), h->stream);
  if (e != cudaSuccess) return e;
  void* args[] = {&p};
  return cudaLaunchCooperativeKernel(solve64_fn(c.precondition != 0), dim3(h->launch.G), dim3(kQT), args, h->launch.smem, h->stream);
}

}  // namespace enkf
