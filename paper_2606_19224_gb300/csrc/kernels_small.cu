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
// [(r, z) | (r, r) | sum r_i z^2 | sum r_i z p]. FP64 mode: scalars in FP64, X is the solution, with a true
// residual after the solve. FP32 mode: scalars and sums in double-float, inner solves from zero refined by the
// double-float residual (HA's low parts read from global memory), as in the persistent solve.
// Measured (analysis, persistent solve before): m = N = 20 in FP64 685 -> 116 us, m = 3,001, N = 37 in
// FP32 without preconditioning 2,550 -> 672 us.
#include <cooperative_groups.h>

#include <algorithm>

#include "krylov.cuh"
#include "solve_body.cuh"

namespace cg = cooperative_groups;

namespace enkf {

constexpr int kST = 512;    // threads per CTA, FP32 (the products wait on shared-memory reads)
constexpr int kST64 = 256;  // FP64 (the FP64 units are the limit; more warps add barrier time only)

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

// Shared memory, by byte offset; every part begins on a 16-byte boundary.
struct Small64Layout {
  int NP, RG, LD, rp, C;
  __host__ __device__ Small64Layout(int N, int rp_, int C_)
      : NP(N <= 32 ? 32 : (N <= 64 ? 64 : 128)), RG(kST64 / (N <= 32 ? 32 : (N <= 64 ? 64 : 128))), LD(N | 1), rp(rp_), C(C_) {}
  __host__ __device__ size_t xch() const { return 0; }                                        // [2][C][NP + 8]
  __host__ __device__ size_t part() const { return xch() + 2 * (size_t)C * (NP + 8) * 8; }    // [RG][NP]
  __host__ __device__ size_t scal() const { return part() + (size_t)kST64 * 8; }              // [16]
  __host__ __device__ size_t Tv() const { return scal() + 16 * 8; }                           // [NP]: T
  __host__ __device__ size_t vec() const { return Tv() + (size_t)NP * 8; }                    // x, res, p, z, r
  __host__ __device__ size_t H() const { return vec() + (size_t)((rp + 1) & ~1) * 5 * 8; }
  __host__ __device__ size_t bytes() const { return H() + (size_t)rp * LD * 8; }
};
struct Small32Layout {
  int NP, LD, rp, C;   // LD: N rounded up to an odd number of 16-byte quads (conflict-free 16-byte reads)
  __host__ __device__ Small32Layout(int N, int rp_, int C_)
      : NP(N <= 32 ? 32 : (N <= 64 ? 64 : 128)), LD(4 * (((N + 3) / 4) | 1)), rp(rp_), C(C_) {}
  __host__ __device__ int rpe() const { return (rp + 3) & ~3; }
  __host__ __device__ size_t xch() const { return 0; }                                        // [2][C][NP + 8] (8 bytes)
  __host__ __device__ size_t part() const { return xch() + 2 * (size_t)C * (NP + 8) * 8; }    // [16][NP + 8] FP32, or [kST] FP64
  __host__ __device__ size_t sums() const {                                                   // [16][4]
    return part() + ((size_t)kST / 32 * (NP + 8) * 4 > (size_t)kST * 8 ? (size_t)kST / 32 * (NP + 8) * 4 : (size_t)kST * 8);
  }
  __host__ __device__ size_t T() const { return sums() + 16 * 4 * 8; }                        // [NP]
  __host__ __device__ size_t scal() const { return T() + (size_t)NP * 4; }                    // [16]
  __host__ __device__ size_t vec() const { return scal() + 16 * 4; }                          // z (df32), x, res, p, b, r
  __host__ __device__ size_t H() const { return vec() + (size_t)rpe() * (8 + 5 * 4); }
  __host__ __device__ size_t bytes() const { return H() + (size_t)rp * LD * 4; }
};

// FP64. What bounds a step is the FP64 unit, two operations per clock per SM: scalars run on one warp
// while the threads of T add up HA^T z.
template <bool PC>
__global__ void __launch_bounds__(kST64) small_cg_f64_kernel(SmallParams p) {
  constexpr int kST = kST64;
  extern __shared__ __align__(1024) unsigned char smem[];
  const Small64Layout L(p.N, p.rp, p.C);
  cg::cluster_group cluster = cg::this_cluster();
  const int N = p.N, C = p.C, NP = L.NP, RG = L.RG, LD = L.LD;
  const int rank = C > 1 ? (int)cluster.block_rank() : 0, j = (int)blockIdx.x / C;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t row0 = (int64_t)rank * p.rp;
  const int nr = (int)max((int64_t)0, min((int64_t)p.rp, p.m - row0));   // this CTA's rows
  double* xch = reinterpret_cast<double*>(smem + L.xch());
  double* spart = reinterpret_cast<double*>(smem + L.part());
  double* sc = reinterpret_cast<double*>(smem + L.scal());
  double* sTv = reinterpret_cast<double*>(smem + L.Tv());
  const int rpe = (p.rp + 1) & ~1;
  double* sx = reinterpret_cast<double*>(smem + L.vec());
  double* sres = sx + rpe;
  double* sp = sres + rpe;
  double* sb = sp + rpe;    // z = M^{-1} r of the step
  double* sr = sb + rpe;
  double* sH = reinterpret_cast<double*>(smem + L.H());
  const double* HA = static_cast<const double*>(p.HA);
  const double inv = 1.0 / (double)(N - 1);
  const bool fixed = p.fixed_iters > 0;
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
  for (int i = t; i < nr; i += kST) sr[i] = p.r[row0 + i];
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
  // per-thread partials of HA^T v over the rows (thread (k, g))
  auto gram = [&](const double* v) {
    const int k = t % NP, g = t / NP;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    if (k < N) {
      int i = g;
      for (; i + 3 * RG < nr; i += 4 * RG)
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = fma(sH[(i + q * RG) * LD + k], v[i + q * RG], a[q]);
      for (; i < nr; i += RG) a[0] = fma(sH[i * LD + k], v[i], a[0]);
    }
    spart[g * NP + k] = nr > 3 * RG ? (a[0] + a[1]) + (a[2] + a[3]) : a[0];
  };
  // (HA T)_i over the SUB lanes s of row i (every lane of the warp calls it)
  auto row_dot = [&](int i, int s) {
    double a = 0.0, b = 0.0;
    if (i < nr) {
      const double* h = sH + i * LD;
      int k = s;
#pragma unroll 4
      for (; k + SUB < N; k += 2 * SUB) {
        a = fma(h[k], sTv[k], a);
        b = fma(h[k + SUB], sTv[k + SUB], b);
      }
      if (k < N) a = fma(h[k], sTv[k], a);
    }
    double u = a + b;
    for (int o = SUB / 2; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
    return u;
  };
  // warp w < nq: sc[8 + w] = sum over the rows of f(w, i)
  auto sums = [&](int nq, auto f) {
    if (warp < nq) {
      double a = 0.0;
      for (int i = lane; i < nr; i += 32) a += f(warp, i);
      a = wsum(a);
      if (lane == 0) sc[8 + warp] = a;
    }
  };
  // every CTA of the cluster has started (a peer's shared memory may not be stored into before) and HA is staged
  if (C > 1) cluster.sync();
  else __syncthreads();
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
  const bool zero = dn2 == 0.0;
  int iters = 0;
  for (int i = t; i < nr; i += kST) {
    const double d = p.D[(row0 + i) * N + j];
    sres[i] = d;
    sb[i] = PC ? d * (1.0 / sr[i]) : d;
    sp[i] = 0.0;
    sx[i] = 0.0;
  }
  __syncthreads();
  gram(sb);
  sums(4, [&](int q, int i) -> double {
    const double z = sb[i], rr = sres[i];
    return q == 0 ? rr * z : q == 1 ? rr * rr : q == 2 ? (sr[i] * z) * z : 0.0;
  });
  __syncthreads();
  const double* all = exchange(true, 4);
  double gamma = 0.0, den = 0.0, bn2 = 0.0, gm = 0.0;   // warp 0's
  const int limit = fixed ? p.fixed_iters : p.max_iter;
  tick(PH_SETUP);
  for (int it = 0;; ++it) {
    // warp 0: the column sums (lane e < 4 sum e) and beta, while the threads of T add up HA^T z
    if (warp == 0) {
      const double v = lane < 4 ? total(all, NP + lane) : 0.0;
      const double g1 = __shfl_sync(0xffffffffu, v, 0), g3 = __shfl_sync(0xffffffffu, v, 2);
      gm = __shfl_sync(0xffffffffu, v, 1);
      double be = 0.0;
      if (it == 0) {
        bn2 = gm;
        den = g3;
      } else {
        be = g1 * sc[13];
        den = fma(be, fma(be, den, 2.0 * __shfl_sync(0xffffffffu, v, 3)), g3);
      }
      gamma = g1;
      if (lane == 0) sc[6] = be;
    }
    const int k = t - 64;   // T's threads: [64, 64 + NP), beside warp 0
    const double tz = k >= 0 && k < N ? total(all, k) : 0.0;
    __syncthreads();
    // T = HA^T z + beta T
    if (k >= 0 && k < NP) {
      const double v = it > 0 && k < N ? fma(sc[6], sTv[k], tz) : tz;
      sTv[k] = v;
      const double t2 = wsum(v * v);
      if (lane == 0) sc[warp - 2] = t2;
    }
    __syncthreads();
    if (warp == 0) {
      double tn2 = sc[0];
      for (int w = 1; w < NP / 32; ++w) tn2 += sc[w];
      int go = !zero && it < limit && (it > 0 || gm > 0.0);
      int bad = 0;
      if (go && it > 0) {
        const double itm = p.tol * (1.0 - 4.0 * 2.220446049250313e-16);
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
        sc[7] = gm;
        sc[12] = gamma;
        if (bad && rank == 0) atomicOr(p.status, bad);
      }
    }
    __syncthreads();
    if (sc[5] == 0.0) break;
    const double al = sc[4], be = sc[6];
    if (t == kST - 1) sc[13] = 1.0 / sc[12];   // for the next beta, beside the products
    // u = HA T, SUB lanes per row, and the step on the row
    for (int i0 = 0; i0 < nr; i0 += kST / SUB) {
      const int i = i0 + t / SUB, s = t % SUB;
      double u = row_dot(i, s);
      if (i < nr && s == 0) {
        const double z = sb[i], ri = sr[i];
        const double pn = it == 0 ? z : fma(be, sp[i], z);
        const double q = fma(u, inv, ri * pn);
        const double rn = fma(-al, q, sres[i]);
        sp[i] = pn;
        sx[i] = fma(al, pn, sx[i]);
        sres[i] = rn;
        sb[i] = PC ? rn * (1.0 / ri) : rn;
      }
    }
    __syncthreads();
    gram(sb);
    sums(4, [&](int q, int i) -> double {
      const double z = sb[i], rr = sres[i];
      return q == 0 ? rr * z : q == 1 ? rr * rr : (sr[i] * z) * (q == 2 ? z : sp[i]);
    });
    __syncthreads();
    all = exchange(true, 4);
    ++iters;
  }
  tick(PH_PASS);
  gm = sc[7];
  // ---- W = HA^T Z/(N-1) and the true residual D - S Z
  __syncthreads();
  gram(sx);
  __syncthreads();
  all = exchange(true, 0);
  if (t < NP) {
    const double v = t < N ? total(all, t) : 0.0;
    sTv[t] = v;
    if (rank == 0 && t < N) p.W[(int64_t)t * N + j] = v * inv;
  }
  for (int i = t; i < nr; i += kST) p.Z[(row0 + i) * N + j] = sx[i];
  double rel_true = zero ? 0.0 : -1.0;
  int refinements = 0;
  if (p.true_residual) {
    __syncthreads();
    for (int i0 = 0; i0 < nr; i0 += kST / SUB) {
      const int i = i0 + t / SUB, s = t % SUB;
      const double u = row_dot(i, s);
      if (i < nr && s == 0) sres[i] = p.D[(row0 + i) * N + j] - fma(u, inv, sr[i] * sx[i]);
    }
    __syncthreads();
    sums(1, [&](int, int i) -> double { return sres[i] * sres[i]; });
    __syncthreads();
    const double rr = total(exchange(false, 1), NP);
    refinements = 1;
    const bool fin = isfinite(dn2) && isfinite(rr);
    if (!fin && rank == 0 && t == 0) atomicOr(p.status, DS_NONFINITE);
    rel_true = !fin ? (double)NAN : (dn2 > 0.0 ? sqrt(rr / dn2) : 0.0);
    tick(PH_REFRESH);
  }
  if (rank == 0 && t == 0) {
    p.col_iters[j] = iters;
    p.col_relres[j] = dn2 > 0.0 ? sqrt(gm / dn2) : 0.0;
    p.col_true[j] = rel_true;
    if (!fixed && !zero && !(sqrt(gm) <= p.tol * sqrt(dn2))) atomicOr(p.status, DS_NOT_CONVERGED);
    atomicMax(p.status + 1, refinements);
    if (prof)
      for (int q = 0; q < PH_COUNT; ++q) p.prof[q] = ph[q];
  }
  if (C > 1) cluster.sync();   // no CTA leaves while a peer may still store into its exchange buffer
}

// a / b; divisors outside the range in which FP32 reciprocals and error terms are exact go through FP64
__device__ __forceinline__ df32 small_div(const df32& a, const df32& b) {
  const float m = fabsf(b.hi);
  return m > 1e-24f && m < 1e24f && fabsf(a.hi) < 1e24f ? df_div(a, b) : df32((double)a / (double)b);
}

// FP32: inner solves from zero refined by the double-float residual. What bounds a step is the reads of HA
// from shared memory (once along its rows, once along its columns, 16 bytes at a time: m N / 16 wavefronts
// in all) and the chain of four barriers and the scalars; everything that leaves a thread is double-float
// (FP64 sums, conversions and divisions took half of a step of 7.8 us at 751 rows per CTA, N = 37).
template <bool PC>
__global__ void __launch_bounds__(kST) small_cg_f32_kernel(SmallParams p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const Small32Layout L(p.N, p.rp, p.C);
  cg::cluster_group cluster = cg::this_cluster();
  const int N = p.N, C = p.C, NP = L.NP, LD = L.LD, SP = NP + 8, Q4 = (N + 3) / 4;
  const int rank = C > 1 ? (int)cluster.block_rank() : 0, j = (int)blockIdx.x / C;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t row0 = (int64_t)rank * p.rp;
  const int nr = (int)max((int64_t)0, min((int64_t)p.rp, p.m - row0));   // this CTA's rows
  const int rpe = L.rpe();
  df32* xch = reinterpret_cast<df32*>(smem + L.xch());
  float* spart = reinterpret_cast<float*>(smem + L.part());
  double* sdpart = reinterpret_cast<double*>(smem + L.part());   // the refresh's partials
  df32* ssum = reinterpret_cast<df32*>(smem + L.sums());
  float* sT = reinterpret_cast<float*>(smem + L.T());
  float* sc = reinterpret_cast<float*>(smem + L.scal());
  df32* sz = reinterpret_cast<df32*>(smem + L.vec());            // the solution
  float* sx = reinterpret_cast<float*>(sz + rpe);
  float* sres = sx + rpe;
  float* sp = sres + rpe;
  float* sb = sp + rpe;    // z = M^{-1} r of the step
  float* sr = sb + rpe;
  float* sH = reinterpret_cast<float*>(smem + L.H());
  const float* HA = static_cast<const float*>(p.HA);
  const double inv = 1.0 / (double)(N - 1);
  const bool fixed = p.fixed_iters > 0;
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
  for (int i = warp; i < nr; i += kST / 32)
    for (int k = lane; k < LD; k += 32) sH[i * LD + k] = k < N ? HA[(row0 + i) * N + k] : 0.f;
  for (int i = t; i < nr; i += kST) {
    sr[i] = (float)p.r[row0 + i];
    sz[i] = df32(0.f, 0.f);
  }
  int buf = 0;
  // entry e of this CTA's sums goes to every CTA of the cluster; all entries are readable behind sync()
  auto mine = [&]() { return xch + ((size_t)buf * C + rank) * SP; };
  auto send = [&](int e, const df32& v, int c) {
    if (C == 1) mine()[e] = v;
    else *cluster.map_shared_rank(mine() + e, c) = v;
  };
  auto sync = [&]() {
    if (C == 1) __syncthreads();
    else cluster.sync();
    const df32* all = xch + (size_t)buf * C * SP;
    buf ^= 1;   // the other buffer is free: every CTA read it before the barrier just passed
    return all;
  };
  auto total = [&](const df32* all, int e) {   // in rank order
    df32 v = all[e];
    for (int c = 1; c < C; ++c) v = v + all[c * SP + e];
    return v;
  };
  auto send64 = [&](int e, double v) {
    df32 d;
    *reinterpret_cast<double*>(&d) = v;
    for (int c = 0; c < C; ++c) send(e, d, c);
  };
  auto total64 = [&](const df32* all, int e) {
    double v = 0.0;
    for (int c = 0; c < C; ++c) v += *reinterpret_cast<const double*>(all + c * SP + e);
    return v;
  };
  auto wsum = [](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  // HA^T z over the warp's rows, 16 bytes of a row per lane (NP/4 lanes per row), into spart[warp][.]
  const int QL = NP / 4, RW = 32 / QL;
  auto gram = [&]() {
    const int q = lane % QL, sub = lane / QL;
    float4 a = {0.f, 0.f, 0.f, 0.f}, b = a;
    if (q < Q4) {
      const float* h = sH + 4 * q;
      constexpr int W = kST / 32;
      int i = warp * RW + sub;
#pragma unroll 2
      for (; i + W * RW < nr; i += 2 * W * RW) {
        const float4 x = *reinterpret_cast<const float4*>(h + i * LD), y = *reinterpret_cast<const float4*>(h + (i + W * RW) * LD);
        const float u = sb[i], v = sb[i + W * RW];
        a.x = fmaf(x.x, u, a.x); a.y = fmaf(x.y, u, a.y); a.z = fmaf(x.z, u, a.z); a.w = fmaf(x.w, u, a.w);
        b.x = fmaf(y.x, v, b.x); b.y = fmaf(y.y, v, b.y); b.z = fmaf(y.z, v, b.z); b.w = fmaf(y.w, v, b.w);
      }
      if (i < nr) {
        const float4 x = *reinterpret_cast<const float4*>(h + i * LD);
        const float u = sb[i];
        a.x = fmaf(x.x, u, a.x); a.y = fmaf(x.y, u, a.y); a.z = fmaf(x.z, u, a.z); a.w = fmaf(x.w, u, a.w);
      }
    }
    a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
    for (int o = QL; o < 32; o <<= 1) {
      a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
      a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
      a.z += __shfl_xor_sync(0xffffffffu, a.z, o);
      a.w += __shfl_xor_sync(0xffffffffu, a.w, o);
    }
    if (sub == 0) *reinterpret_cast<float4*>(spart + warp * SP + 4 * q) = a;
  };
  // the warp's sums of four values per thread into ssum[warp][0..3]: two exchanges leave value
  // lane / 8 % 4 with each lane, three more add up the eight lanes that hold it
  auto warp_sums = [&](float v0, float v1, float v2, float v3) {
    const bool h1 = lane & 16, h0 = lane & 8;
    df32 a(h1 ? v2 : v0, 0.f), b(h1 ? v3 : v1, 0.f);
    a = a + df32(__shfl_xor_sync(0xffffffffu, h1 ? v0 : v2, 16), 0.f);
    b = b + df32(__shfl_xor_sync(0xffffffffu, h1 ? v1 : v3, 16), 0.f);
    const df32 o = df_shfl_xor(h0 ? a : b, 8);
    a = (h0 ? b : a) + o;
    a = a + df_shfl_xor(a, 4);
    a = a + df_shfl_xor(a, 2);
    a = a + df_shfl_xor(a, 1);
    if ((lane & 7) == 0) ssum[warp * 4 + (lane >> 4) * 2 + (h0 ? 1 : 0)] = a;
  };
  // the CTA's totals to the cluster: entries [0, N) HA^T z (four threads per column), NP + q and
  // NP + 4 + q the halves of sum q
  auto exchange = [&]() {
    constexpr int W = kST / 32;
    if (t < 4 * NP) {
      const int k = t >> 2, part = t & 3;
      df32 v(spart[part * SP + k], 0.f);
#pragma unroll
      for (int w = 1; w < W / 4; ++w) v = v + df32(spart[(4 * w + part) * SP + k], 0.f);
      v = v + df_shfl_xor(v, 1);
      v = v + df_shfl_xor(v, 2);
      if (k < N)
        for (int c = part; c < C; c += 4) send(k, v, c);
    }
    if (warp >= W - 2) {
      const int e = t - (kST - 64);   // (warp, sum) pairs
      df32 v = ssum[e];
      v = v + df_shfl_xor(v, 4);
      v = v + df_shfl_xor(v, 8);
      v = v + df_shfl_xor(v, 16);
      const int c = lane >> 2;
      if (c < C) send(NP + (e >> 5) * 4 + (lane & 3), v, c);
    }
    return sync();
  };
  // (HA T)_i and (HA T)_k over the SUB lanes s of the rows i and k (every lane of the warp calls it): two rows
  // share the reads of T
  auto row_dots = [&](int i, int k, int s, float& u, float& v) {
    float4 a = {0.f, 0.f, 0.f, 0.f}, b = a;
    const float* h = sH + min(i, nr - 1) * LD;   // (nr > 0 where rows are walked)
    const float* g = sH + min(k, nr - 1) * LD;
#pragma unroll 4
    for (int q = s; q < Q4; q += SUB) {
      const float4 y = *reinterpret_cast<const float4*>(sT + 4 * q);
      const float4 x = *reinterpret_cast<const float4*>(h + 4 * q), w = *reinterpret_cast<const float4*>(g + 4 * q);
      a.x = fmaf(x.x, y.x, a.x); a.y = fmaf(x.y, y.y, a.y); a.z = fmaf(x.z, y.z, a.z); a.w = fmaf(x.w, y.w, a.w);
      b.x = fmaf(w.x, y.x, b.x); b.y = fmaf(w.y, y.y, b.y); b.z = fmaf(w.z, y.z, b.z); b.w = fmaf(w.w, y.w, b.w);
    }
    u = (a.x + a.y) + (a.z + a.w);
    v = (b.x + b.y) + (b.z + b.w);
    for (int o = SUB / 2; o > 0; o >>= 1) {
      u += __shfl_xor_sync(0xffffffffu, u, o);
      v += __shfl_xor_sync(0xffffffffu, v, o);
    }
  };
  // sum over the cluster's rows of f(i), in FP64
  auto sum64 = [&](auto f) {
    double a = 0.0;
    for (int i = t; i < nr; i += kST) a += f(i);
    a = wsum(a);
    if (lane == 0) sdpart[warp] = a;
    __syncthreads();
    if (t == 0) {
      for (int w = 1; w < kST / 32; ++w) a += sdpart[w];
      send64(NP, a);
    }
    return total64(sync(), NP);
  };
  if (C > 1) cluster.sync();   // every CTA has started: a peer's shared memory may not be stored into before
  const double dn2 = sum64([&](int i) {
    const double d = p.D[(row0 + i) * N + j];
    return d * d;
  });
  int iters = 0, refinements = 0;
  double rel_true = dn2 == 0.0 ? 0.0 : -1.0, itol = p.inner_tol;
  bool done = dn2 == 0.0;
  for (int i = t; i < nr; i += kST) sres[i] = (float)p.D[(row0 + i) * N + j];   // of the first solve
  __syncthreads();
  for (int outer = 0;; ++outer) {
    // ---- the inner solve of S x = res from x = 0
    {
      float v0 = 0.f, v1 = 0.f, v2 = 0.f;
      for (int i = t; i < nr; i += kST) {
        const float rr = sres[i], ri = sr[i], z = PC ? rr * (1.f / ri) : rr;
        sb[i] = z;
        sp[i] = 0.f;
        sx[i] = 0.f;
        v0 = fmaf(rr, z, v0);
        v1 = fmaf(rr, rr, v1);
        v2 = fmaf(ri * z, z, v2);
      }
      warp_sums(v0, v1, v2, 0.f);
    }
    __syncthreads();
    gram();
    __syncthreads();
    const df32* all = exchange();
    // warp 0's scalars: (r, z), (p, S p) - |T|^2/(N-1), and the stopping value of |r|^2
    df32 gamma, den, stop, vinv(inv);
    const int limit = fixed ? p.fixed_iters : p.max_iter - iters;
    tick(PH_SETUP);
    for (int it = 0;; ++it) {
      if (warp == 0) {
        df32 v = lane < 8 ? total(all, NP + lane) : df32(0.f, 0.f);
        v = v + df_shfl_xor(v, 4);
        auto pick = [&](int q) { return df32(__shfl_sync(0xffffffffu, v.hi, q), __shfl_sync(0xffffffffu, v.lo, q)); };
        const df32 g1 = pick(0), gm = pick(1), g3 = pick(2), g4 = pick(3);
        df32 be;
        if (it == 0) {
          // |r| <= tol |b| compared in squares, tol shrunk by a few ulps of FP64
          const double itm = itol * (1.0 - 4.0 * 2.220446049250313e-16);
          stop = df32(itm * itm) * gm;
          den = g3;
        } else {
          be = small_div(g1, gamma);
          den = fma(be, fma(be, den, g4 + g4), g3);
        }
        gamma = g1;
        // T = HA^T z + beta T, applied in FP32; its norm is that of the rounded T
        SqAcc n2;
        for (int k = lane; k < NP; k += 32) {
          float tv = k < N ? total(all, k).hi : 0.f;
          if (it > 0) tv = fmaf(be.hi, sT[k], tv);
          sT[k] = tv;
          n2.add(tv);
        }
        df32 tn2 = df_fast2sum(n2.s, n2.c);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tn2 = tn2 + df_shfl_xor(tn2, o);
        int go = !done && it < limit && (it > 0 || gm.hi > 0.f), bad = 0;
        if (go && it > 0) {
          if (!isfinite(gm.hi)) { bad = DS_NONFINITE; go = 0; }
          else if (fixed ? gm.hi == 0.f : (gm - stop).hi <= 0.f) go = 0;
        }
        float al = 0.f;
        if (go) {
          const df32 pq = fma(tn2, vinv, den);
          if (!isfinite(pq.hi)) { bad = DS_NONFINITE; go = 0; }
          else if (pq.hi <= 0.f) { bad = DS_BREAKDOWN; go = 0; }
          else al = small_div(gamma, pq).hi;
        }
        if (lane == 0) {
          sc[0] = al;
          sc[1] = be.hi;
          sc[2] = (float)go;
          if (bad && rank == 0) atomicOr(p.status, bad);
        }
      }
      __syncthreads();
      if (sc[2] == 0.f) break;
      const float al = sc[0], be = sc[1], finv = (float)inv;
      // u = HA T, SUB lanes per row, the step on the row, and the sums of the next one
      float v0 = 0.f, v1 = 0.f, v2 = 0.f, v3 = 0.f;
      auto step = [&](int i, float u) {
        const float z = sb[i], ri = sr[i];
        const float pn = it == 0 ? z : fmaf(be, sp[i], z);
        const float q = fmaf(u, finv, ri * pn);
        const float rn = fmaf(-al, q, sres[i]);
        const float zn = PC ? rn * (1.f / ri) : rn, rz = ri * zn;
        sp[i] = pn;
        sx[i] = fmaf(al, pn, sx[i]);
        sres[i] = rn;
        sb[i] = zn;
        v0 = fmaf(rn, zn, v0);
        v1 = fmaf(rn, rn, v1);
        v2 = fmaf(rz, zn, v2);
        v3 = fmaf(rz, pn, v3);
      };
      for (int i0 = 0; i0 < nr; i0 += 2 * kST / SUB) {
        const int i = i0 + t / SUB, k = i + kST / SUB, s = t % SUB;
        float u, v;
        row_dots(i, k, s, u, v);
        if (i < nr && s == 0) step(i, u);
        if (k < nr && s == 0) step(k, v);
      }
      warp_sums(v0, v1, v2, v3);
      __syncthreads();
      gram();
      __syncthreads();
      all = exchange();
      ++iters;
    }
    tick(PH_PASS);
    // ---- Z += X, W = HA^T Z/(N-1) and the true residual D - S Z in double-float
    for (int i = t; i < nr; i += kST) {
      sz[i] = sz[i] + df32(sx[i], 0.f);
      p.Zdf[(row0 + i) * N + j] = sz[i];
    }
    __syncthreads();
    const int RG = kST / NP;
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
      sdpart[t] = (double)a.value();
    }
    __syncthreads();
    if (t < N) {
      double v = 0.0;
      for (int g = 0; g < RG; ++g) v += sdpart[g * NP + t];
      send64(t, v);
    }
    all = sync();
    df32* sTd = reinterpret_cast<df32*>(sdpart);   // T/(N-1) in double-float
    double wk = 0.0;
    if (t < N) {
      wk = total64(all, t) * inv;
      if (rank == 0) p.W[(int64_t)t * N + j] = wk;
    }
    if (t < NP) sTd[t] = df32(wk);   // (the partials were read before the barrier)
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
      for (int o = SUB / 2; o > 0; o >>= 1) u = u + df_shfl_xor(u, o);
      if (i < nr && s == 0) {
        const df32 q = fma(df32(p.r[row0 + i]), sz[i], u);
        sres[i] = (p.Ddf[(row0 + i) * N + j] - q).hi;
      }
    }
    __syncthreads();
    const double rr = sum64([&](int i) { return (double)sres[i] * (double)sres[i]; });
    ++refinements;
    const bool fin = isfinite(dn2) && isfinite(rr);
    if (!fin && rank == 0 && t == 0) atomicOr(p.status, DS_NONFINITE);
    rel_true = !fin ? (double)NAN : (dn2 > 0.0 ? sqrt(rr / dn2) : 0.0);
    tick(PH_REFRESH);
    if (!fin || rel_true <= p.tol) done = true;
    if (fixed || done || outer >= p.max_refine || iters >= p.max_iter) break;
    itol = fmin(0.5, fmax(p.inner_tol, rel_true > 0.0 ? 0.1 * p.tol / rel_true : p.inner_tol));
  }
  if (rank == 0 && t == 0) {
    p.col_iters[j] = iters;
    p.col_relres[j] = rel_true;
    p.col_true[j] = rel_true;
    if (!fixed && !(rel_true >= 0.0 && rel_true <= p.tol)) atomicOr(p.status, DS_NOT_CONVERGED);
    atomicMax(p.status + 1, refinements);
    if (prof)
      for (int q = 0; q < PH_COUNT; ++q) p.prof[q] = ph[q];
  }
  if (C > 1) cluster.sync();   // no CTA leaves while a peer may still store into its exchange buffer
}

// ------------------------------------------------------------------ host side
static void* small_fn(bool fp64, bool pc) {
  if (fp64) return pc ? (void*)small_cg_f64_kernel<true> : (void*)small_cg_f64_kernel<false>;
  return pc ? (void*)small_cg_f32_kernel<true> : (void*)small_cg_f32_kernel<false>;
}
static size_t small_smem(bool fp64, int N, int rp, int C) {
  return fp64 ? Small64Layout(N, rp, C).bytes() : Small32Layout(N, rp, C).bytes();
}

static void small_launch_config(const enkf_config& c, int C, cudaStream_t stream, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at) {
  const bool fp64 = c.precision == ENKF_FP64;
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)(c.N * C));
  cfg.blockDim = dim3(fp64 ? kST64 : kST);
  cfg.dynamicSmemBytes = small_smem(fp64, c.N, (int)((c.m + C - 1) / C), C);
  cfg.stream = stream;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
}

// A cluster size C <= 8 for which all N clusters are resident at once and the row block fits in shared
// memory, or 0. Among those the largest that leaves 128 rows per CTA: more CTAs shorten the two
// products, and below that the cluster barrier costs more than they do. (N C SMs need not suffice: a cluster
// lies in one part of the chip. 37 clusters of 4 ran as two waves, 1.92 ms against 0.98.)
// (The limit on dynamic shared memory belongs to the kernel, not to the handle, so it is never set lower.)
constexpr int kSmallSmem = 224 * 1024;
int small_cluster(const enkf_handle_s* h) {
  const enkf_config& c = h->cfg;
  if (c.variant != ENKF_CGD || c.precision > ENKF_FP32 || c.warm_start || c.grid_blocks > 0) return 0;
  const bool fp64 = c.precision == ENKF_FP64;
  if (fp64 && !steady_fp64(h)) return 0;
  void* fn = small_fn(fp64, c.precondition != 0);
  auto fits = [&](int C) { return (c.m + C - 1) / C <= 65536 && small_smem(fp64, c.N, (int)((c.m + C - 1) / C), C) <= kSmallSmem; };
  // from the largest down (a query of the driver only for a size that would be taken)
  for (int C = std::min(8, h->sms / c.N); C >= 1 && fits(C); --C) {
    if (C > 1 && (c.m + C - 1) / C < 128 && fits(C - 1)) continue;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    small_launch_config(c, C, nullptr, cfg, at);
    int resident = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&resident, fn, &cfg) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (resident >= c.N) return C;
  }
  return 0;
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
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  small_launch_config(c, p.C, h->stream, cfg, at);
  void* args[] = {&p};
  return cudaLaunchKernelExC(&cfg, small_fn(fp64, c.precondition != 0), args);
}

}  // namespace enkf
