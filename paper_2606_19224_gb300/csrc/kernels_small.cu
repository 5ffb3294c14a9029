// CG on S Z = D for problems whose HA fits the shared memory of a few SMs: one thread-block cluster per
// column. The N recurrences are independent (Sec. 3.1-3.3 of the paper); the persistent solve of
// solve_body.cuh shares each pass over HA among the columns and pays for it with a reduction over the
// whole grid and two grid barriers per step, which is most of a step when HA is small (17 us per
// step at m = 3,001, N = 37 in FP32; 26 us at m = N = 20 in FP64, where one CTA also computes a padded
// 64 x 32 tile at the FP64 rate). Here the C CTAs of cluster j hold all of HA, a block of its rows each, and
// run column j alone: a step exchanges N + 4 partial sums through distributed shared memory behind one
// cluster barrier (none for C = 1), and clusters never wait for each other.
//
// The step is the one-reduction Hestenes-Stiefel form (see passH in cg_device.cuh): T = HA^T p carried as
// T_{k+1} = HA^T z_{k+1} + beta_k T_k and (p, S p) = ||T||^2/(N-1) + sum r_i p_i^2 from the sums
// [(r, z) | (r, r) | sum r_i z^2 | sum r_i z p]; scalars in FP64. FP64 mode: X is the solution, with a true
// residual after the solve. FP32 mode: inner solves from zero refined by the double-float residual
// (HA's low parts read from global memory), as in the persistent solve.
#include <cooperative_groups.h>

#include <algorithm>

#include "solve_body.cuh"

namespace cg = cooperative_groups;

namespace enkf {

constexpr int kST = 256;

struct SmallParams {
  int64_t m;
  int N, C, rp;          // rp: rows per CTA
  const void* HA;        // [m][N] in VT
  const double* D;
  const double* r;
  const df32* HAdf;      // FP32 mode
  const df32* Ddf;
  df32* Zdf;
  double* Z;             // FP64 mode
  double* W;
  double tol, inner_tol;
  int max_iter, fixed_iters, max_refine, true_residual;
  int* col_iters;
  double* col_relres;
  double* col_true;
  int* status;
  unsigned long long* prof;
};

template <typename VT> struct SmallLayout {
  int NP, RG, LD, rp, C;
  __host__ __device__ SmallLayout(int N, int rp_, int C_)
      : NP(N <= 32 ? 32 : (N <= 64 ? 64 : 128)), RG(kST / (N <= 32 ? 32 : (N <= 64 ? 64 : 128))), LD(N | 1), rp(rp_), C(C_) {}
  __host__ __device__ size_t xch() const { return 0; }                                   // [2][C][NP + 8] FP64
  __host__ __device__ size_t part() const { return xch() + 2 * (size_t)C * (NP + 8) * 8; }   // [RG][NP] FP64
  __host__ __device__ size_t T() const { return part() + (size_t)kST * 8; }              // [NP] FP64
  __host__ __device__ size_t scal() const { return T() + (size_t)NP * 8; }                // [16] FP64
  __host__ __device__ size_t Tv() const { return scal() + 16 * 8; }                       // [NP] T in VT
  __host__ __device__ size_t vec() const { return Tv() + (size_t)NP * 8; }                // z (df32), then x, res, p, b, r
  __host__ __device__ size_t H() const {
    return vec() + (size_t)((rp + 1) & ~1) * (sizeof(VT) == 4 ? 8 + 5 * 4 : 5 * 8);
  }
  __host__ __device__ size_t bytes() const { return H() + (size_t)rp * LD * sizeof(VT); }
};

template <typename VT, bool PC>
__global__ void __launch_bounds__(kST) small_cg_kernel(SmallParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  const SmallLayout<VT> L(p.N, p.rp, p.C);
  cg::cluster_group cluster = cg::this_cluster();
  const int N = p.N, C = p.C, NP = L.NP, RG = L.RG, LD = L.LD;
  const int rank = C > 1 ? (int)cluster.block_rank() : 0, j = (int)blockIdx.x / C;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t row0 = (int64_t)rank * p.rp;
  const int nr = (int)max((int64_t)0, min((int64_t)p.rp, p.m - row0));   // this CTA's rows
  double* xch = reinterpret_cast<double*>(smem + L.xch());
  double* spart = reinterpret_cast<double*>(smem + L.part());
  double* sT = reinterpret_cast<double*>(smem + L.T());
  double* sc = reinterpret_cast<double*>(smem + L.scal());
  VT* sTv = reinterpret_cast<VT*>(smem + L.Tv());   // T as the products read it
  const int rpe = (p.rp + 1) & ~1;
  df32* sz = reinterpret_cast<df32*>(smem + L.vec());                    // FP32 mode: the solution
  VT* sx = reinterpret_cast<VT*>(smem + L.vec() + (sizeof(VT) == 4 ? (size_t)rpe * 8 : 0));
  VT* sres = sx + rpe;
  VT* sp = sres + rpe;
  VT* sb = sp + rpe;    // z = M^{-1} r of the step
  VT* sr = sb + rpe;
  VT* sH = reinterpret_cast<VT*>(smem + L.H());
  const VT* HA = static_cast<const VT*>(p.HA);
  const double inv = 1.0 / (double)(N - 1);
  const bool refine = sizeof(VT) == 4, fixed = p.fixed_iters > 0;
  // lanes per row of u = HA T, so that a CTA with few rows keeps its warps busy
  int SUB = 1;
  while (SUB < 16 && nr * SUB * 2 <= kST) SUB *= 2;
  const bool prof = p.prof != nullptr && blockIdx.x == 0 && t == 0;
  unsigned long long ph[PH_COUNT] = {0, 0, 0, 0, 0, 0, 0, 0}, tp = prof ? global_ns() : 0ull;
  auto tick = [&](int slot) {
    if (prof) {
      const unsigned long long now = global_ns();
      ph[slot] += now - tp;
      tp = now;
    }
  };
  for (int e = t; e < nr * N; e += kST) sH[(e / N) * LD + e % N] = HA[row0 * N + e];
  for (int i = t; i < nr; i += kST) {
    sr[i] = (VT)p.r[row0 + i];
    if (refine) sz[i] = df32(0.f, 0.f);
  }
  int buf = 0;
  // totals over the cluster of the CTA's spart-combined vector v(k), k < NP, and of nq scalars in sc[8..]:
  // every CTA stores its part into all of the cluster's exchange buffers and adds them in rank order
  auto exchange = [&](bool vec, int nq) {
    // (spart and sc[8..] are complete: the caller has synchronised)
    double v = 0.0;
    if (vec && t < N)
      for (int g = 0; g < RG; ++g) v += spart[g * NP + t];
    double* mine = xch + (size_t)buf * C * (NP + 8) + (size_t)rank * (NP + 8);
    const bool q = t >= NP && t < NP + nq;   // (NP = 128, nq = 4: t < 132)
    const double s = q ? sc[8 + t - NP] : 0.0;
    if ((vec && t < N) || q) {
      if (C == 1) mine[t] = q ? s : v;
      else
        for (int c = 0; c < C; ++c) *cluster.map_shared_rank(mine + t, c) = q ? s : v;
    }
    if (C == 1) __syncthreads();
    else cluster.sync();
    const double* all = xch + (size_t)buf * C * (NP + 8);
    buf ^= 1;   // the other buffer is free: every CTA read it before the barrier just passed
    return all;
  };
  auto total = [&](const double* all, int e) {
    double v = 0.0;
    for (int c = 0; c < C; ++c) v += all[(size_t)c * (NP + 8) + e];
    return v;
  };
  auto wsum = [](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  // per-thread partials of HA^T v over the rows (thread (k, g)); a VT accumulator, FP64 across threads
  auto gram = [&](const VT* v) {
    const int k = t % NP, g = t / NP;
    VT a = VT(0);
    if (k < N)
      for (int i = g; i < nr; i += RG) a = fma(sH[i * LD + k], v[i], a);
    spart[g * NP + k] = (double)a;
  };
  // warp w < nq: sc[8 + w] = sum over the rows of f(w, i)
  auto sums = [&](int nq, auto f) {
    if (warp < nq) {
      double a = 0.0;
      if constexpr (sizeof(VT) == 8) {
        for (int i = lane; i < nr; i += 32) a += f(warp, i);
      } else {
        float b = 0.f;
        for (int i = lane; i < nr; i += 32) b += f(warp, i);
        a = (double)b;
      }
      a = wsum(a);
      if (lane == 0) sc[8 + warp] = a;
    }
  };
  __syncthreads();
  // ||d_j||^2
  if (warp == 0) {
    double a = 0.0;
    for (int i = lane; i < nr; i += 32) {
      const double d = p.D[(row0 + i) * N + j];
      a = fma(d, d, a);
    }
    a = wsum(a);
    if (lane == 0) sc[8] = a;
  }
  __syncthreads();
  const double dn2 = total(exchange(false, 1), NP);
  int iters = 0, refinements = 0;
  double rel_true = dn2 == 0.0 ? 0.0 : -1.0, rel_rec = 0.0, itol = refine ? p.inner_tol : p.tol;
  bool done = dn2 == 0.0, conv_rec = dn2 == 0.0;
  // right-hand side of the first solve
  for (int i = t; i < nr; i += kST) {
    sres[i] = (VT)p.D[(row0 + i) * N + j];
    sx[i] = VT(0);
  }
  __syncthreads();
  tick(PH_SETUP);
  for (int outer = 0;; ++outer) {
    // ---- the inner solve of S x = res from x = 0
    for (int i = t; i < nr; i += kST) {
      sb[i] = PC ? sres[i] * (VT(1) / sr[i]) : sres[i];
      sp[i] = VT(0);
      sx[i] = VT(0);
    }
    if (t < NP) sT[t] = 0.0;
    __syncthreads();
    gram(sb);
    sums(4, [&](int q, int i) -> VT {
      const VT z = sb[i], rr = sres[i];
      return q == 0 ? rr * z : q == 1 ? rr * rr : q == 2 ? (sr[i] * z) * z : VT(0);
    });
    __syncthreads();
    const double* all = exchange(true, 4);
    double gamma = total(all, NP), gm = total(all, NP + 1), den = total(all, NP + 2);
    const double bn2 = gm;
    double beta = 0.0;
    const int limit = fixed ? p.fixed_iters : p.max_iter - iters;
    tick(PH_SETUP);
    for (int it = 0;; ++it) {
      // T = HA^T z + beta T, ||T||^2, then the step's scalars (the same in every CTA of the cluster)
      double t2 = 0.0;
      if (t < NP) {
        const double v = t < N ? total(all, t) + (it > 0 ? beta * sT[t] : 0.0) : 0.0;
        // the FP32 mode applies T in FP32, and its norm is that of the rounded T
        const double vr = sizeof(VT) == 4 ? (double)(float)v : v;
        sT[t] = vr;
        sTv[t] = (VT)v;
        t2 = wsum(vr * vr);
        if (lane == 0) sc[warp] = t2;
      }
      __syncthreads();
      if (warp == 0) {
        double tn2 = sc[0];
        for (int w = 1; w < NP / 32; ++w) tn2 += sc[w];
        int go = !done && it < limit && (it > 0 || gm > 0.0);
        int bad = 0;
        if (go && it > 0) {
          const double itm = itol * (1.0 - 4.0 * 2.220446049250313e-16);
          if (!isfinite(gm)) { bad = DS_NONFINITE; go = 0; }
          else if (fixed ? gm == 0.0 : gm <= itm * itm * bn2) go = 0;
        }
        double al = 0.0;
        if (go) {
          const double pq = fma(tn2, inv, den);
          if (!isfinite(pq)) { bad = DS_NONFINITE; go = 0; }
          else if (pq <= 0.0) { bad = DS_BREAKDOWN; go = 0; }
          else al = gamma / pq;
        }
        if (lane == 0) {
          sc[4] = al;
          sc[5] = (double)go;
          if (bad && rank == 0) atomicOr(p.status, bad);
        }
      }
      __syncthreads();
      if (sc[5] == 0.0) break;
      const VT al = (VT)sc[4], be = (VT)beta, vinv = (VT)inv;
      // u = HA T, SUB lanes per row, and the step on the row
      for (int i0 = 0; i0 < nr; i0 += kST / SUB) {
        const int i = i0 + t / SUB, s = t % SUB;
        VT u = VT(0);
        if (i < nr)
          for (int k = s; k < N; k += SUB) u = fma(sH[i * LD + k], sTv[k], u);
        for (int o = SUB / 2; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
        if (i < nr && s == 0) {
          const VT z = sb[i], ri = sr[i];
          const VT pn = it == 0 ? z : fma(be, sp[i], z);
          const VT q = fma(u, vinv, ri * pn);
          const VT rn = fma(-al, q, sres[i]);
          sp[i] = pn;
          sx[i] = fma(al, pn, sx[i]);
          sres[i] = rn;
          sb[i] = PC ? rn * (VT(1) / ri) : rn;
        }
      }
      __syncthreads();
      gram(sb);
      sums(4, [&](int q, int i) -> VT {
        const VT z = sb[i], rr = sres[i];
        return q == 0 ? rr * z : q == 1 ? rr * rr : (sr[i] * z) * (q == 2 ? z : sp[i]);
      });
      __syncthreads();
      all = exchange(true, 4);
      const double g1 = total(all, NP);
      beta = g1 / gamma;
      den = total(all, NP + 2) + 2.0 * beta * total(all, NP + 3) + beta * beta * den;
      gamma = g1;
      gm = total(all, NP + 1);
      ++iters;
    }
    tick(PH_PASS);
    rel_rec = dn2 > 0.0 ? sqrt(gm / dn2) : 0.0;
    conv_rec = dn2 == 0.0 || sqrt(gm) <= p.tol * sqrt(dn2);
    // ---- W = HA^T Z/(N-1) and the true residual D - S Z
    __syncthreads();
    if constexpr (sizeof(VT) == 8) {
      gram(sx);
      __syncthreads();
      all = exchange(true, 0);
      if (t < NP) {
        const double v = t < N ? total(all, t) : 0.0;
        sTv[t] = (VT)v;
        if (rank == 0 && t < N) p.W[(int64_t)t * N + j] = v * inv;
      }
      for (int i = t; i < nr; i += kST) p.Z[(row0 + i) * N + j] = sx[i];
      if (!p.true_residual) break;
      __syncthreads();
      for (int i0 = 0; i0 < nr; i0 += kST / SUB) {
        const int i = i0 + t / SUB, s = t % SUB;
        VT u = VT(0);
        if (i < nr)
          for (int k = s; k < N; k += SUB) u = fma(sH[i * LD + k], sTv[k], u);
        for (int o = SUB / 2; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
        if (i < nr && s == 0) sres[i] = (VT)p.D[(row0 + i) * N + j] - fma(u, (VT)inv, sr[i] * sx[i]);
      }
    } else {
      // double-float: Z += X, T = HA^T Z by thread (k, g), then the rows
      for (int i = t; i < nr; i += kST) {
        sz[i] = sz[i] + df32((float)sx[i], 0.f);
        p.Zdf[(row0 + i) * N + j] = sz[i];
      }
      __syncthreads();
      {
        const int k = t % NP, g = t / NP;
        DFAcc a;
        if (k < N) {
          int n = 0;
#pragma unroll 4
          for (int i = g; i < nr; i += RG) {
            a.add(p.HAdf[(row0 + i) * N + k], sz[i]);
            if ((++n & 3) == 0) a.renorm();
          }
        }
        spart[g * NP + k] = (double)a.value();
      }
      __syncthreads();
      all = exchange(true, 0);
      if (t < NP) sT[t] = t < N ? total(all, t) : 0.0;
      if (rank == 0 && t < N) p.W[(int64_t)t * N + j] = sT[t] * inv;
      __syncthreads();
      df32* sTd = reinterpret_cast<df32*>(spart);   // T/(N-1) in double-float
      if (t < NP) sTd[t] = df32(sT[t] * inv);
      __syncthreads();
      for (int i0 = 0; i0 < nr; i0 += kST / SUB) {
        const int i = i0 + t / SUB, s = t % SUB;
        DFAcc a;
        if (i < nr) {
          int n = 0;
#pragma unroll 4
          for (int k = s; k < N; k += SUB) {
            a.add(p.HAdf[(row0 + i) * N + k], sTd[k]);
            if ((++n & 3) == 0) a.renorm();
          }
        }
        df32 u = a.value();
        for (int o = SUB / 2; o > 0; o >>= 1)
          u = u + df32(__shfl_xor_sync(0xffffffffu, u.hi, o), __shfl_xor_sync(0xffffffffu, u.lo, o));
        if (i < nr && s == 0) {
          const df32 q = fma(df32(p.r[row0 + i]), sz[i], u);
          sres[i] = (VT)(p.Ddf[(row0 + i) * N + j] - q).hi;
        }
      }
    }
    __syncthreads();
    sums(1, [&](int, int i) -> VT { return sres[i] * sres[i]; });
    __syncthreads();
    const double rr = total(exchange(false, 1), NP);
    ++refinements;
    const bool fin = isfinite(dn2) && isfinite(rr);
    if (!fin && rank == 0 && t == 0) atomicOr(p.status, DS_NONFINITE);
    rel_true = !fin ? (double)NAN : (dn2 > 0.0 ? sqrt(rr / dn2) : 0.0);
    tick(PH_REFRESH);
    if (!refine) break;
    if (!fin || rel_true <= p.tol) done = true;
    if (fixed || done || outer >= p.max_refine || iters >= p.max_iter) break;
    itol = fmin(0.5, fmax(p.inner_tol, rel_true > 0.0 ? 0.1 * p.tol / rel_true : p.inner_tol));
  }
  if (rank == 0 && t == 0) {
    p.col_iters[j] = iters;
    p.col_relres[j] = refine ? rel_true : rel_rec;
    p.col_true[j] = rel_true;
    const bool conv = fixed ? true : refine ? (rel_true >= 0.0 && rel_true <= p.tol) : conv_rec;
    if (!conv) atomicOr(p.status, DS_NOT_CONVERGED);
    atomicMax(p.status + 1, refinements);
    if (prof)
      for (int q = 0; q < PH_COUNT; ++q) p.prof[q] = ph[q];
  }
  if (C > 1) cluster.sync();   // no CTA leaves while a peer may still store into its exchange buffer
}

// ------------------------------------------------------------------ host side
static void* small_fn(bool fp64, bool pc) {
  if (fp64) return pc ? (void*)small_cg_kernel<double, true> : (void*)small_cg_kernel<double, false>;
  return pc ? (void*)small_cg_kernel<float, true> : (void*)small_cg_kernel<float, false>;
}
static size_t small_smem(bool fp64, int N, int rp, int C) {
  return fp64 ? SmallLayout<double>(N, rp, C).bytes() : SmallLayout<float>(N, rp, C).bytes();
}

// A cluster size C in {1, 2, 4, 8} for which all clusters are resident at once (N C SMs) and the row block
// fits in shared memory, or 0. Among those the largest that leaves 128 rows per CTA: more CTAs shorten
// the two products, and below that the cluster barrier costs more than they do.
int small_cluster(const enkf_config& c, int sms) {
  if (c.variant != ENKF_CGD || c.precision > ENKF_FP32 || c.warm_start || c.grid_blocks > 0) return 0;
  int best = 0;
  for (int C = 1; C <= 8; C *= 2) {
    const int64_t rp = (c.m + C - 1) / C;
    if ((int64_t)c.N * C > sms || rp > 65536) continue;
    if (small_smem(c.precision == ENKF_FP64, c.N, (int)rp, C) > 224 * 1024) continue;
    if (best == 0 || rp >= 128) best = C;
  }
  return best;
}

cudaError_t plan_small(enkf_handle_s* h) {
  const auto& c = h->cfg;
  const int C = h->small_c, rp = (int)((c.m + C - 1) / C);
  const bool fp64 = c.precision == ENKF_FP64;
  return cudaFuncSetAttribute(small_fn(fp64, c.precondition != 0), cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)small_smem(fp64, c.N, rp, C));
}

cudaError_t launch_small(enkf_handle_s* h) {
  const auto& c = h->cfg;
  auto& ws = h->ws;
  const bool fp64 = c.precision == ENKF_FP64;
  SmallParams p{};
  p.m = c.m;
  p.N = c.N;
  p.C = h->small_c;
  p.rp = (int)((c.m + p.C - 1) / p.C);
  p.HA = fp64 ? (const void*)ws.HA64 : (const void*)ws.HA32;
  p.D = ws.D;
  p.r = ws.r;
  p.HAdf = static_cast<const df32*>(ws.HAdf);
  p.Ddf = static_cast<const df32*>(ws.Ddf);
  p.Zdf = static_cast<df32*>(ws.Zdf);
  p.Z = ws.Z;
  p.W = ws.W;
  p.tol = c.tol;
  p.inner_tol = c.inner_tol;
  p.max_iter = c.max_iter;
  p.fixed_iters = c.fixed_iters;
  p.max_refine = c.max_refine;
  p.true_residual = c.true_residual;
  p.col_iters = ws.col_iters;
  p.col_relres = ws.col_relres;
  p.col_true = ws.col_true;
  p.status = ws.status;
  p.prof = h->prof_enabled ? ws.prof : nullptr;
  cudaError_t err = cudaMemsetAsync(ws.status, 0, 4 * sizeof(int32_t), h->stream);
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(c.N * p.C));
  cfg.blockDim = dim3(kST);
  cfg.dynamicSmemBytes = small_smem(fp64, c.N, p.rp, p.C);
  cfg.stream = h->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = p.C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  void* args[] = {&p};
  return cudaLaunchKernelExC(&cfg, small_fn(fp64, c.precondition != 0), args);
}

}  // namespace enkf
