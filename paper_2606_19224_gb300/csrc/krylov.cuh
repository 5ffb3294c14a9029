// CG preconditioned by R on S Z = D, carried in the coordinates of its Krylov space.
//
// With the preconditioner M = R, z0 = R^{-1} b has the residual b - S z0 = -HA (HA^T R^{-1} b)/(N-1),
// and every later iterate, direction and residual of the CG recurrences is R^{-1} or S times a
// combination of the columns of HA: z_k = R^{-1} (b - HA w_k) with an N-vector w_k per column.
// In these coordinates, with K = HA^T R^{-1} HA / (N-1) and g = HA^T R^{-1} b / (N-1), the residual
// is r_k = -HA rho_k, rho_k = g - (I + K) w_k, its preconditioned norm is (r_k, R^{-1} r_k) =
// (N-1) rho_k^T K rho_k, and a direction p = R^{-1} HA f has (p, S p) = (N-1) (K f)^T (f + K f): the
// same alpha, beta and iterates as the recurrences on m-vectors (Sec. 3.1-3.3 of the paper, Eq.
// matvec_decomp for S p), with one N x N product per step in place of two passes over HA.
// What remains of a solve is three passes over the observation rows:
//
//   pass G   K and F = HA^T R^{-1} b                           (two products m N^2)
//   CG       N independent recurrences, one CTA per column, vectors of length N
//   pass Z   Z += R^{-1} (b - HA w), T = HA^T Z                 (two products)
//   pass R   the true residual D - R Z - HA T/(N-1)            (one product)
//
// and a column whose true residual misses the tolerance gets another cycle with that residual
// as b (iterative refinement). Z is formed entry by entry and certified by its own true
// residual, as before; nothing in the certificate uses K or F.
//
// The products need more than FP32 (the residual's terms cancel to 1e-8 and below), and double-
// float products on the CUDA cores cost 12 FP32 operations per term: 0.16 ms per product pair at
// m = 65,536, N = 64, measured 0.33 ms per refresh, with the tensor cores idle. Here every operand
// is a fixed-point number of five signed slices (9 bits, then four times 10: 48 bits below a power
// of two at least the largest entry of its row or column), each slice an integer of at most 256
// (the first) or 512 in FP16. Sums of integer products below 2^24 accumulate in FP32 in tensor
// memory without rounding (measured with constant, alternating and random operands), and a tile of
// 64 terms stays there: the products of slices i and j with i + j = g belong to one power of two
// and share a sum, at most 2^22 for g = 0 and 2^24 for g = 1. (For g = 2 the bound is 2^25: only
// operands whose low slices all sit at their limits with one sign can round there, by 2^-42.) The
// sums of an entry are then combined into a double-float number with error-free additions. The
// products over the rows (K, F and T = HA^T Z, whose error S amplifies) take the slice products
// with i + j <= 5, those over the members (u = HA T) i + j <= 4. An emulation against 64 bits of
// the residual of a double-float Z with an ensemble whose condition is 10^7 (one member 300 times
// the others) gives 5e-9 of ||d|| with i + j <= 4 and a tenth of that with i + j <= 5, next to
// 1e-10 from rounding Z itself; five equal 9-bit slices gave 5e-8 and missed a tolerance of 1e-8.
#pragma once

#include "tc_mixed.cuh"

namespace enkf {

constexpr int kSl = 5;       // slices per operand
constexpr int kKR = 64;      // observation rows per tile
constexpr int kKT = 512;     // threads per CTA: four warps per scheduler hide the latency of the slicing
                             // and joining chains (256 threads spent 5 of 8 cycles waiting)

struct KrylovParams {
  int64_t m;
  int N;
  const df32* HAdf;     // [m][N]
  const df32* Ddf;      // [m][N]
  df32* Zdf;            // [m][N]
  float* B;             // [m][N] residual of the current Z, the next cycle's right-hand side
  const df32* rdf;      // [m] R, 1/R and 1/sqrt(R) in double-float
  const df32* rinv;
  const df32* rsq;
  const float* hs;      // [m] a power of two above the largest |HA| of each row
  const unsigned* umax; // largest |HA_ik| / sqrt(r_i) (float bits)
  df32* part;           // [G][krylov_part(N)] partial products and column sums of the CTAs
  df32* Kred;           // [N][N]
  df32* Fred;           // [N][N] F^T: row j is column j of F
  df32* wred;           // [N][N] row j holds w_j
  df32* Tred;           // [N][N] T^T
  df32* sums;           // [2][N] ||d_j||^2 and (b_j, R^{-1} b_j)
  int* hold;            // [N] columns whose recurrences of this cycle gained nothing
  double* rrpart;       // [2][G][NT]
  double* W;            // [N][N]
  double tol;
  int max_iter, max_refine;
  int* col_iters;
  double* col_relres;
  double* col_true;
  int* status;
  unsigned* bar;
  unsigned long long* prof;
  int phase;               // 0: the whole solve; 1: pass G only; 2: what follows pass G
  // learned start (phase 2): w0 [N][N] (column j starts at w = w0_j), ||d_j - S z0_j||^2 per column
  const float* w0;
  const double* wnorm;
  int warm_accept;
  double* col_warm;
};

// kernels_krylov.cu: R, 1/R and 1/sqrt(R) in double-float from R in FP64
cudaError_t launch_krylov_rows(const double* r, int64_t m, df32* rdf, df32* rinv, df32* rsq, cudaStream_t s);

// entries of one CTA's partial: K and F columns of its column group, then two column sums
__host__ __device__ constexpr int krylov_part(int N) { return 2 * N * (N < 64 ? N : 64) + 2 * 64; }

template <int NT> struct KLayout {
  static constexpr int JC = NT < 64 ? NT : 64;       // columns j of one CTA
  static constexpr int BR = kSl * JC * 16;            // pass G, operand B: bytes per row group (all slices)
  static constexpr int TROWS = NT == 128 ? 64 : 128;  // rows of the T operand (copies of its JC columns for NT <= 64)
  static constexpr int NB = NT == 128 ? 1 : 2;        // HA images: the next tile is sliced behind the products
  static constexpr int HP = kKR * NT * 2;             // bytes per slice of the HA tile
  static constexpr int CP = kKR * 128 * 2;            // ... of the pass G operand A
  static constexpr int TP = TROWS * NT * 2;           // ... of the T operand
  static constexpr int VP = JC * kKR * 2;             // ... of the Z tile (rows j, K-major over i)
  static constexpr int off_t = 0;
  static constexpr int off_h = kSl * TP;
  static constexpr int off_v = off_h + NB * kSl * HP;
  // (an M = 128 operand of fewer rows or columns reads on into the next region: rows that no
  // result uses)
  static constexpr int end_z = off_v + kSl * VP;
  static constexpr int off_gu = kSl * CP;             // pass G operands B: slices of U, then (NT = 128) of V
  static constexpr int off_gv = off_gu + 8 * BR;
  static constexpr int SQ = 24;                       // column sums of squares, floats per thread
  static constexpr int off_sq = off_gv + (NT == 128 ? 8 * BR : 0);
  static constexpr int end_g = off_sq + SQ * 4 * kKT;
  static constexpr int end_cg = 16 * NT * 8 + 16 * kKT * 8 + 64;   // the recurrences of 16 columns
  static constexpr int uni0 = end_z > end_g ? end_z : end_g;
  static constexpr int uni = uni0 > end_cg ? uni0 : end_cg;
  // scalars: six FP64 and two int arrays of NT; per tile buffer the rows' scales and r (or 1/r); the
  // T operand's column scales; column maxima and scales of a tile; scratch
  static constexpr int off_scal = uni;
  static constexpr int off_row = off_scal + NT * (6 * 8 + 2 * 4);
  static constexpr int off_col = off_row + 2 * 12 * kKR;
  static constexpr int off_max = off_col + 4 * 128;
  static constexpr int off_scr = off_max + 4 * (8 * 64 + 64);
  static constexpr int need = off_scr + kKT * 8;
  // one CTA per SM whatever NT: each holds all of its SM's tensor memory
  static constexpr int bytes = need < 120 * 1024 ? 120 * 1024 : need;
  static_assert(bytes <= 226 * 1024, "shared memory");
};

// The power of two above |mx| (inv) and its inverse (scale). Entries below 2^-86 count as that size,
// which keeps scale 2^28 finite (a row or column of zeros has scale 2^86).
__device__ __forceinline__ void pow2_of(float mx, float& scale, float& inv) {
  int E = (int)((__float_as_uint(mx) >> 23) & 0xFFu);
  E = max(40, min(252, E));
  scale = __uint_as_float((uint32_t)(253 - E) << 23);
  inv = __uint_as_float((uint32_t)(E + 1) << 23);
}

// the five slices of (h + l) scale, |h scale| <= 1: integers in FP32, weights 2^-8, 2^-18, ... 2^-48
__device__ __forceinline__ void slice5(float h, float l, float scale, float (&v)[kSl]) {
  constexpr float M = 12582912.f;   // adding and subtracting it rounds to an integer (|x| < 2^22)
  const float x = __fmul_rn(h, scale * 256.f);
  v[0] = __fsub_rn(__fadd_rn(x, M), M);
  const float d0 = __fsub_rn(x, v[0]);
  v[1] = __fsub_rn(__fmaf_rn(d0, 1024.f, M), M);
  const float d1 = __fmaf_rn(d0, 1024.f, -v[1]);
  float s, e;
  df_two_sum(__fmul_rn(d1, 1024.f), __fmul_rn(l, scale * 0x1p28f), s, e);   // l in units of the third slice
  v[2] = __fsub_rn(__fadd_rn(s, M), M);
  const float d2 = __fadd_rn(__fsub_rn(s, v[2]), e);
  v[3] = __fsub_rn(__fmaf_rn(d2, 1024.f, M), M);
  const float d3 = __fmaf_rn(d2, 1024.f, -v[3]);
  v[4] = __fsub_rn(__fmaf_rn(d3, 1024.f, M), M);
}
__device__ __forceinline__ uint32_t pack_half2(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// eight consecutive elements along the 16-byte direction of a core row, each slice one store
struct Slices8 {
  uint4 w[kSl];
  __device__ __forceinline__ void make(const df32 (&x)[8], const float (&scale)[8]) {
    uint32_t u[kSl][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float a[kSl], b[kSl];
      slice5(x[2 * q].hi, x[2 * q].lo, scale[2 * q], a);
      slice5(x[2 * q + 1].hi, x[2 * q + 1].lo, scale[2 * q + 1], b);
#pragma unroll
      for (int s = 0; s < kSl; ++s) u[s][q] = pack_half2(a[s], b[s]);
    }
#pragma unroll
    for (int s = 0; s < kSl; ++s) w[s] = make_uint4(u[s][0], u[s][1], u[s][2], u[s][3]);
  }
  __device__ __forceinline__ void make(const df32 (&x)[8], float scale) {
    const float sc[8] = {scale, scale, scale, scale, scale, scale, scale, scale};
    make(x, sc);
  }
  __device__ __forceinline__ void store(unsigned char* at, int slice_bytes) const {
#pragma unroll
    for (int s = 0; s < kSl; ++s) *reinterpret_cast<uint4*>(at + s * slice_bytes) = w[s];
  }
};

__device__ __forceinline__ df32 ld_df(const df32* p) {   // through L2: other CTAs of this launch wrote it
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return df32(v.x, v.y);
}

// tcgen05.ld of LC columns of the six sums of an entry (`stride` columns apart; LV of them in use)
constexpr int kLv = 6;
template <int LV, int LC>   // LC: 8 or 4 columns
__device__ __forceinline__ void tmem_ld_levels(uint32_t taddr, uint32_t stride, float (&a)[LV][LC]) {
  uint32_t r[LV][LC];
#pragma unroll
  for (int g = 0; g < LV; ++g) {
    if constexpr (LC == 8)
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                   : "=r"(r[g][0]), "=r"(r[g][1]), "=r"(r[g][2]), "=r"(r[g][3]), "=r"(r[g][4]), "=r"(r[g][5]),
                     "=r"(r[g][6]), "=r"(r[g][7])
                   : "r"(taddr + g * stride));
    else
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                   : "=r"(r[g][0]), "=r"(r[g][1]), "=r"(r[g][2]), "=r"(r[g][3]) : "r"(taddr + g * stride));
  }
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int g = 0; g < LV; ++g)
#pragma unroll
    for (int q = 0; q < LC; ++q) {
      // keep every use of the loaded registers behind the wait
      asm volatile("" : "+r"(r[g][q]));
      a[g][q] = __uint_as_float(r[g][q]);
    }
}
// The value of an entry from its sums as an unevaluated pair (s, l): the levels down to 2^-20 enter
// exactly, the rest are 2^-30 of the first's unit and below.
// Row products: a[g] = level g = 0..5.
template <int LC>
__device__ __forceinline__ void join_rows(const float (&a)[kLv][LC], int q, float& s, float& l) {
  float t, e, e2;
  df_two_sum(a[0][q], __fmul_rn(a[1][q], 0x1p-10f), t, e);
  df_two_sum(t, __fmul_rn(a[2][q], 0x1p-20f), s, e2);
  const float low = __fmaf_rn(a[5][q], 0x1p-50f, __fmaf_rn(a[4][q], 0x1p-40f, __fmul_rn(a[3][q], 0x1p-30f)));
  l = __fadd_rn(__fadd_rn(e, e2), low);
}
// Member products: levels 0..4; SPLIT: level 1 as two sums in a[1] and a[5].
template <bool SPLIT, int LV, int LC>
__device__ __forceinline__ void join_members(const float (&a)[LV][LC], int q, float& s, float& l) {
  float t, e, e2, e3 = 0.f;
  df_two_sum(a[0][q], __fmul_rn(a[1][q], 0x1p-10f), t, e);
  if constexpr (SPLIT) {
    float t2;
    df_two_sum(t, __fmul_rn(a[5][q], 0x1p-10f), t2, e3);
    t = t2;
  }
  df_two_sum(t, __fmul_rn(a[2][q], 0x1p-20f), s, e2);
  const float low = __fmaf_rn(a[4][q], 0x1p-40f, __fmul_rn(a[3][q], 0x1p-30f));
  l = __fadd_rn(__fadd_rn(__fadd_rn(e, e3), e2), low);
}

__device__ __forceinline__ void umma_lead(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc,
                                          uint32_t lead) {
  asm volatile("{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
               " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
               ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(lead));
}
// kind::f16 descriptor of FP16 operands with M = 128 and each operand K-major or MN-major
__host__ __device__ constexpr uint32_t sl_idesc(int N, bool a_mn, bool b_mn) {
  return umma_idesc(0, N, b_mn) | ((a_mn ? 1u : 0u) << 15);
}
// The slice products of D = A B, level g = i + j <= GMAX in the JC columns at d + g JC, over KS blocks of
// 16 along K. The slices of B lie one behind the other along N (B_SL bytes apart), so that
// A_i [B_j0 .. B_j1] is one MMA into the consecutive levels i + j0 .. i + j1: with M = 128 an MMA takes
// 64 cycles for any N <= 64, 75 for 128 and 135 for 256 (the reads of A bound the narrow ones), and
// the 19 products of 64 columns 2,700 cycles per 64 terms instead of 4,900. SPLIT: the product (1, 0)
// goes to level column 5 (K = 128 would let level 1 reach 2^25). Called by one whole warp with `lead`
// on one lane, so that addresses stay warp-uniform.
template <int KS, int GMAX, bool SPLIT, int JC, bool AMN, bool BMN, int A_PART, int A_STEP, int B_SL, int B_STEP>
__device__ __forceinline__ void issue_levels(uint32_t d, uint64_t a, uint64_t b, uint64_t* mbar, uint32_t lead) {
  // recomputed here for each tile: hoisted out of the tile loop the descriptors would be spilled
  asm volatile("" : "+l"(a), "+l"(b), "+r"(d));
  constexpr int NMAX = 256 / JC < kSl ? 256 / JC : kSl;   // slices of B per MMA at most
  auto mma = [&](int i, int j0, int nj, int kb, int col, bool acc) {
    umma_lead(d + (uint32_t)(col * JC), a + (uint64_t)((i * A_PART + kb * A_STEP) >> 4),
              b + (uint64_t)((j0 * B_SL + kb * B_STEP) >> 4), sl_idesc(nj * JC, AMN, BMN), acc ? 1u : 0u, lead);
  };
#pragma unroll
  for (int kb = 0; kb < KS; ++kb)
#pragma unroll
    for (int i = 0; i < kSl; ++i) {
      const int nj = GMAX - i + 1 < kSl ? GMAX - i + 1 : kSl;   // j = 0 .. nj - 1
      int j = 0;
      if (SPLIT && i == 1) {
        mma(1, 0, 1, kb, 5, kb > 0);
        j = 1;
      }
      // the level GMAX of GMAX = kSl begins at (1, kSl - 1): on its own in the first block along K
      const int end = (GMAX == kSl && i == 1 && kb == 0) ? nj - 1 : nj;
#pragma unroll
      for (int q = 0; q < kSl; ++q)   // in pieces of even size, at most NMAX slices each
        if (j < end) {
          const int left = end - j, pieces = (left + NMAX - 1) / NMAX, n = (left + pieces - 1) / pieces;
          mma(i, j, n, kb, i + j, i > 0 || kb > 0);
          j += n;
        }
      if (end < nj) mma(i, end, 1, kb, i + end, false);
    }
  if (lead) umma_commit(mbar);
}
__device__ __forceinline__ uint32_t elect_lane() {
  uint32_t v;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(v));
  return v;
}
// what the passes of one CTA share
struct KCta {
  unsigned char* smem;
  uint32_t tmem;
  uint64_t* mbar;
  uint32_t phase;
  int* status;
  bool ok;
};
__device__ __forceinline__ void k_wait(KCta& c) {
  // a few hardware waits before the bounded one, which reads the global timer
  uint32_t done = 0;
#pragma unroll 1
  for (int q = 0; q < 4 && !done; ++q)
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done) : "r"(smem_addr(c.mbar)), "r"(c.phase) : "memory");
  if (!done && !mbar_wait(c.mbar, c.phase, c.status)) c.ok = false;
  c.phase ^= 1u;
  tc_fence_after();
}

// Eight consecutive df32 of a row of N, zeros past N or when !ok. N % 8 == 0: unconditional 16-byte
// loads (from row 0 of the array when !ok), so that several rows' loads are in flight together.
__device__ __forceinline__ void load_row8(df32 (&x)[8], const df32* base, int64_t i, int c0, int N, bool ok) {
  if ((N & 7) == 0) {
    const bool in = ok && c0 < N;
    const df32* row = base + (in ? i * N + c0 : 0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(row + 2 * q);
      x[2 * q] = in ? df32(v.x, v.y) : df32(0.f, 0.f);
      x[2 * q + 1] = in ? df32(v.z, v.w) : df32(0.f, 0.f);
    }
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const bool in = ok && c0 + q < N;
      const float2 v = *reinterpret_cast<const float2*>(base + (in ? i * N + c0 + q : 0));
      x[q] = in ? df32(v.x, v.y) : df32(0.f, 0.f);
    }
  }
}

// Who slices what: an item is eight columns of one row, a warp takes eight rows (lane & 7: their
// 16-byte pieces of a core matrix are one 128-byte line, so the stores are free of bank conflicts)
// of four column groups (lane >> 3). W columns: 2 W / 8 warp items per tile of 64 rows.
template <int W> struct KItems {
  static constexpr int G4 = W / 32;                       // warp items per eight rows
  static constexpr int N = (8 * G4 + 15) / 16;            // items per thread (W = 32: half the warps)
  __device__ static bool live(int warp, int it) { return warp + 16 * it < 8 * G4; }
  __device__ static int row(int warp, int lane, int it) { return (warp + 16 * it) / G4 * 8 + (lane & 7); }
  __device__ static int col(int warp, int lane, int it) { return (warp + 16 * it) % G4 * 32 + (lane >> 3) * 8; }
};

// The T operand of u = HA T: JC columns of a reduced N x N matrix (row j of `src` is column j; other
// CTAs wrote it) as ROWS rows of W, row q holding column q % JC, each scaled by a power of two above
// its largest entry (s_inv: the scale's inverse).
template <int W, int ROWS, int JC>
__device__ __forceinline__ void stage_columns(const df32* __restrict__ src, int j0, int N, unsigned char* img,
                                              float* s_inv) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int q = 8 * warp + (lane & 7), j = j0 + q % JC;
  if (8 * warp >= ROWS) return;   // uniform in the warp
  df32 x[W / 32][8];
  float mx = 0.f;
#pragma unroll
  for (int g = 0; g < W / 32; ++g)
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int k = 32 * g + (lane >> 3) * 8 + e;
      x[g][e] = (j < N && k < N) ? ld_df(src + (int64_t)j * N + k) : df32(0.f, 0.f);
      mx = fmaxf(mx, fabsf(x[g][e].hi));
    }
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
  float sc, inv;
  pow2_of(mx, sc, inv);
#pragma unroll
  for (int g = 0; g < W / 32; ++g) {
    Slices8 sl;
    sl.make(x[g], sc);
    sl.store(img + core_idx(q, 32 * g + (lane >> 3) * 8, W) * 2, ROWS * W * 2);
  }
  if (lane < 8) s_inv[q] = inv;
}

// ------------------------------------------------------------------ pass G
// The CTA's rows of U = R^{-1/2} HA and V = R^{-1/2} b (b = D, or the FP32 residual B), sliced per tile
// (add: onto what `out` holds):
// U scaled by the power of two above its largest entry in the problem (the innovations record it),
// each column of V by that of its largest entry in the tile; K = U^T U and F = U^T V accumulate over
// the tiles in double-float registers. Column group c takes the columns [64 c, 64 c + JC) of K and F.
// NT <= 64: one product [U | V]^T U (M = 128: rows k of K, then rows j of F^T); NT = 128: U^T U_c, then
// U^T V. Operand A holds [U | V] (U) slice by slice, operand B the slices of U_c (and V) side by side;
// the loads of the next tile are in flight behind the products.
template <int NT>
__device__ __noinline__ void pass_gram(const KrylovParams& p, bool from_b, int c, int64_t row0, int64_t row1,
                                       KCta& cta, df32* __restrict__ out, bool add = false) {
  using L = KLayout<NT>;
  using UI = KItems<NT>;
  using VI = KItems<L::JC>;
  constexpr int JC = L::JC;
  constexpr bool PRE = NT <= 64;     // the next tile's U is held in registers behind the products
  constexpr int LC = PRE ? 8 : 4;
  float* s_max = reinterpret_cast<float*>(cta.smem + L::off_max);     // [8 row blocks][64]
  float* s_sc = reinterpret_cast<float*>(cta.smem + L::off_col);      // [64] inverse scales of V
  const int N = p.N, t = threadIdx.x, lane = t & 31, qd = (t >> 5) & 3, sub = t >> 7;
  const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);               // warp-uniform
  const int ln = 32 * qd + lane;
  constexpr int NC = JC / 4;         // columns of a product per thread
  DFAcc acc[NC], accF[NT == 128 ? NC : 1];
  // ||b_j||^2 over the thread's rows as compensated pairs and (b_j, R^{-1} b_j): in shared memory,
  // [24][threads] (in registers they spilled the accumulators)
  float* s_sq = reinterpret_cast<float*>(cta.smem + L::off_sq) + t;
#pragma unroll
  for (int e = 0; e < L::SQ; ++e) s_sq[e * kKT] = 0.f;
  float su, uinv;
  pow2_of(__uint_as_float(*(volatile const unsigned*)p.umax), su, uinv);
  const uint32_t base = smem_addr(cta.smem), lead = warp == 0 ? elect_lane() : 0u;
  const bool vlive = VI::live(warp, 0);
  const int vr = VI::row(warp, lane, 0), vc = VI::col(warp, lane, 0), cv0 = c * 64 + vc;
  df32 u[PRE ? UI::N : 1][8], v[8], uq[PRE ? UI::N : 1], vq;
  auto load_u = [&](int64_t i0, int it, int slot) {
    const int64_t i = i0 + UI::row(warp, lane, it);
    const bool in = UI::live(warp, it) && i < row1;
    load_row8(u[slot], p.HAdf, i, UI::col(warp, lane, it), N, in);
    uq[slot] = p.rsq[in ? i : 0];
  };
  auto load = [&](int64_t i0) {
    if (PRE)
#pragma unroll
      for (int it = 0; it < UI::N; ++it) load_u(i0, it, it);
    const int64_t i = i0 + vr;
    const bool in = vlive && i < row1;
    if (from_b) {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = df32((in && cv0 + e < N) ? p.B[i * N + cv0 + e] : 0.f, 0.f);
    } else {
      load_row8(v, p.Ddf, i, cv0, N, in);
    }
    vq = p.rsq[in ? i : 0];
  };
  // address of core row (r, column cc of slice 0) of an operand B
  auto b_at = [&](int off, int r, int cc) {
    return cta.smem + off + (r >> 3) * L::BR + (cc >> 3) * 128 + (r & 7) * 16;
  };
  // the tile from i0 on into the operands: U at once, V after its column maxima
  auto slice = [&](int64_t i0) {
#pragma unroll(PRE ? UI::N : 1)
    for (int it = 0; it < UI::N; ++it) {
      const int q = PRE ? it : 0;
      if (!PRE) load_u(i0, it, 0);
#pragma unroll
      for (int e = 0; e < 8; ++e) u[q][e] = u[q][e] * uq[q];
      if (UI::live(warp, it)) {
        const int r = UI::row(warp, lane, it), cc = UI::col(warp, lane, it);
        Slices8 sl;
        sl.make(u[q], su);
        sl.store(cta.smem + core_idx(r, cc, 128) * 2, L::CP);
        if (NT < 128 || (cc >> 6) == c) sl.store(b_at(L::off_gu, r, cc & (JC - 1)), JC * 16);
      }
    }
    float mx[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      SqAcc sq;
      sq.s = s_sq[e * kKT];
      sq.c = s_sq[(8 + e) * kKT];
      sq.add(v[e].hi);
      s_sq[e * kKT] = sq.s;
      s_sq[(8 + e) * kKT] = sq.c;
      v[e] = v[e] * vq;
      s_sq[(16 + e) * kKT] = fmaf(v[e].hi, v[e].hi, s_sq[(16 + e) * kKT]);
      mx[e] = fabsf(v[e].hi);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], o));
    }
    if (vlive && (lane & 7) == 0) {
      *reinterpret_cast<float4*>(s_max + (vr >> 3) * 64 + vc) = make_float4(mx[0], mx[1], mx[2], mx[3]);
      *reinterpret_cast<float4*>(s_max + (vr >> 3) * 64 + vc + 4) = make_float4(mx[4], mx[5], mx[6], mx[7]);
    }
    __syncthreads();
    if (vlive) {
      float sv[8];
#pragma unroll
      for (int w = 0; w < 8; ++w)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 m4 = *reinterpret_cast<const float4*>(s_max + w * 64 + vc + 4 * h);
          mx[4 * h] = fmaxf(mx[4 * h], m4.x);
          mx[4 * h + 1] = fmaxf(mx[4 * h + 1], m4.y);
          mx[4 * h + 2] = fmaxf(mx[4 * h + 2], m4.z);
          mx[4 * h + 3] = fmaxf(mx[4 * h + 3], m4.w);
        }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float inv;
        pow2_of(mx[e], sv[e], inv);
        if (vr == 0) s_sc[vc + e] = inv;
      }
      Slices8 sl;
      sl.make(v, sv);
      if (NT == 128) sl.store(b_at(L::off_gv, vr, vc), JC * 16);
      else sl.store(cta.smem + core_idx(vr, NT + vc, 128) * 2, L::CP);
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
  };
  auto flush = [&](DFAcc* a, float rs, const float* cs) {   // cs: column scales or nullptr (U's)
#pragma unroll
    for (int q0 = 0; q0 < NC; q0 += LC) {
      float lv[kLv][LC];
      tmem_ld_levels<kLv, LC>(cta.tmem + ((uint32_t)(32 * qd) << 16) + sub * NC + q0, JC, lv);
#pragma unroll
      for (int q = 0; q < LC; ++q) {
        float s, l, tt, e;
        join_rows(lv, q, s, l);
        const float f = rs * (cs ? cs[sub * NC + q0 + q] : uinv);
        df_two_sum(a[q0 + q].s, s * f, tt, e);
        a[q0 + q].s = tt;
        a[q0 + q].c = __fadd_rn(a[q0 + q].c, __fmaf_rn(l, f, e));
        a[q0 + q].renorm();
      }
    }
  };
  // K = rows of the tile, both operands MN-major (columns contiguous)
  auto issue = [&](int boff) {
    if (warp == 0) {
      tc_fence_after();
      issue_levels<kKR / 16, 5, false, JC, true, true, L::CP, 2 * 2048, JC * 16, 2 * L::BR>(
          cta.tmem, umma_desc(base, 2048, 128), umma_desc(base + boff, L::BR, 128), cta.mbar, lead);
    }
  };
  if (row0 < row1) {
    load(row0);
    slice(row0);
    issue(L::off_gu);
  }
  for (int64_t i0 = row0; i0 < row1 && cta.ok; i0 += kKR) {
    const bool more = i0 + kKR < row1;
    if (more) load(i0 + kKR);
    k_wait(cta);
    if constexpr (NT == 128) {
      flush(acc, uinv * 0x1p-16f, nullptr);
      tc_fence_before();
      __syncthreads();
      issue(L::off_gv);
      k_wait(cta);
      flush(accF, uinv * 0x1p-16f, s_sc);
    } else {
      // lanes [NT, 2 NT) hold F^T: row scale of V's column
      flush(acc, (ln < NT ? uinv : s_sc[ln & (NT - 1)]) * 0x1p-16f, nullptr);
    }
    if (more) {
      __syncthreads();   // s_sc is rewritten with the operands
      slice(i0 + kKR);
      issue(L::off_gu);
    }
  }
  // the CTA's partial: K[k][jl] at k NJ + jl, F[k][jl] behind it, then the column sums
  const int NJ = min(JC, N);
  auto put = [&](int e, const df32& v) { out[e] = add ? out[e] + v : v; };
  if constexpr (NT == 128) {
    if (ln < N)
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        const int jl = sub * NC + q;
        put(ln * NJ + jl, acc[q].value());
        put(N * NJ + ln * NJ + jl, accF[q].value());
      }
  } else {
    // lanes [0, NT): K[k = lane][col]; lanes [NT, 2 NT): F^T[j = lane - NT][k = col]
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const int col = sub * NC + q;
      if (col < N) {
        if (ln < N) put(ln * NJ + col, acc[q].value());
        else if (ln >= NT && ln - NT < N) put(N * NJ + col * NJ + (ln - NT), acc[q].value());
      }
    }
  }
  // column sums over the threads of each column, fixed order
  double* red = reinterpret_cast<double*>(cta.smem);   // [2][64 rows][JC]
  __syncthreads();
  if (vlive)
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      red[vr * JC + vc + e] = (double)s_sq[e * kKT] + (double)s_sq[(8 + e) * kKT];
      red[(64 + vr) * JC + vc + e] = (double)s_sq[(16 + e) * kKT];
    }
  __syncthreads();
  if (t < 2 * JC) {
    const int which = t / JC, j = t % JC;
    double s = 0.0;
    for (int q = 0; q < 64; ++q) s += red[(which * 64 + q) * JC + j];
    put(2 * N * NJ + which * 64 + j, df32(s));
  }
  __syncthreads();
}

// Entries [0, ngr cnt) of the partials (entry e of column group c: part[c cstride + q stride + e],
// q < RB), summed over q in a fixed order: this CTA (b of G) takes a contiguous chunk, several
// threads per entry where the chunk is shorter than the CTA, and hands (c, e, total) to store.
template <class Store>
__device__ __forceinline__ void reduce_parts(const df32* __restrict__ part, int64_t cstride, int64_t stride, int RB,
                                             int ngr, int cnt, int G, int b, df32* scratch, Store&& store) {
  const int t = threadIdx.x, total = ngr * cnt;
  const int chunk = (total + G - 1) / G;
  const int e0 = min(total, b * chunk), n = min(total, e0 + chunk) - e0;
  auto add_range = [&](int e, int q0, int q1) {
    const df32* src = part + (int64_t)(e / cnt) * cstride + e % cnt;
    DFAcc a;
#pragma unroll 8
    for (int q = q0; q < q1; ++q) {
      const float2 v = __ldcg(reinterpret_cast<const float2*>(src + q * stride));
      float s, r;
      df_two_sum(a.s, v.x, s, r);
      a.s = s;
      a.c = __fadd_rn(a.c, __fadd_rn(r, v.y));
    }
    return a.value();
  };
  if (n <= 0) return;
  if (n >= kKT) {
    for (int e = e0 + t; e < e0 + n; e += kKT) store(e / cnt, e % cnt, add_range(e, 0, RB));
    return;
  }
  const int parts = kKT / n, el = t % n, w = t / n;
  scratch[t] = w < parts ? add_range(e0 + el, (int)((int64_t)w * RB / parts), (int)((int64_t)(w + 1) * RB / parts))
                         : df32(0.f, 0.f);
  __syncthreads();
  if (t < n) {
    df32 v = scratch[t];
    for (int q = 1; q < parts; ++q) v = v + scratch[q * n + t];
    const int e = e0 + t;
    store(e / cnt, e % cnt, v);
  }
  __syncthreads();
}

// Every CTA sums the G CTAs' column sums part[q NT + j] in the same fixed order.
template <int NT>
__device__ __forceinline__ void total_columns(const double* __restrict__ part, int G, int N, double* out,
                                              double* scratch) {
  constexpr int Q = kKT / NT;
  const int t = threadIdx.x, j = t % NT, q = t / NT;
  double s = 0.0;
  if (j < N) {
    const int b0 = (int)((int64_t)q * G / Q), b1 = (int)((int64_t)(q + 1) * G / Q);
#pragma unroll 8
    for (int b = b0; b < b1; ++b) s += __ldcg(part + (int64_t)b * NT + j);
  }
  scratch[t] = s;
  __syncthreads();
  if (t < NT) {
    double v = 0.0;
    for (int qq = 0; qq < Q; ++qq) v += scratch[qq * NT + t];
    out[t] = v;
  }
  __syncthreads();
}

// ------------------------------------------------------------------ CG in the coordinates
__device__ __forceinline__ df32 df_div(const df32& a, const df32& b) {   // two corrections: about 46 bits
  const float r = __frcp_rn(b.hi);
  const float q0 = __fmul_rn(a.hi, r);
  df32 e = a - b * df32(q0, 0.f);
  const float q1 = __fmul_rn(e.hi, r);
  e = e - b * df32(q1, 0.f);
  const df32 q = df_fast2sum(q0, q1);
  return q + df32(__fmul_rn(e.hi, r), 0.f);
}
__device__ __forceinline__ df32 df_shfl_xor(const df32& v, int o) {
  return df32(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}
// Columns j0, j0 + step, ... (nc <= 16, one per warp) of this cycle: (I + K) w = g from w = 0 (or the
// learned start) by the recurrences at the head of this file until (r, R^{-1} r) <= itol^2
// (b, R^{-1} b) or the column's step limit; w into row j of wred, the steps taken added to
// col_iters[j]. Everything is double-float: on this part an FP64 instruction holds a scheduler's
// FP64 unit for about 64 cycles, and the first form of this loop, with the vectors and scalars of
// a step in FP64 (some 60 such instructions in one warp's serial chain), took 2.9 us per step at
// N = 64 and 5.3 at N = 128. A step is one product (each thread keeps its block of K in
// registers, shared by the CTA's columns) and one round of sums: with kr = K rho and h = K f of the step
// before, (p, S p) is (rho + kr, kr) + 2 beta (rho + kr, h) + beta^2 (p, S p)_old. (The middle sum is
// -beta (p, S p)_old while directions are conjugate. Without it a member 10^4 times the others, one eigenvalue
// of K far above the rest, took 796 steps of the first cycle to a residual of 9.1 ||d||; it takes 146 to 0.083
// and the second cycle ends at 1.8e-6. At m = 65,536, N = 64 a solve takes 29 steps either way.)
// These sums go from |K g|^2 down to the tolerance, more than FP32's exponents hold once the variances of
// R lie some 10^8 below those of HA; the vectors of a column are therefore carried times a power of two
// that puts |K rho|^2 of the start just below the top of the range. The recurrences start from
// R^{-1} b, whose residual is larger than b by up to the largest eigenvalue of K, and where they end early (the
// step limit, or rounding at such an R) it may still be: a column whose (r, R^{-1} r) is not below
// (b, R^{-1} b) is held for this cycle (w = 0, Z as it was).
template <int NT>
struct KMat {
  static constexpr int TPR = kKT / NT, KPT = NT / TPR;   // threads per row, entries per thread
  df32 k[KPT];
};
struct KColumns {
  const df32* K;         // [N][N]
  const df32* F;         // [N][N]
  df32* w;               // [N][N]
  const double* bb;      // shared: (b_j, R^{-1} b_j), tolerance, done and rejected starts per column
  const double* itol;
  const int* done;
  const int* bad;
  const float* w0;       // learned start or nullptr
  int* iters;            // [N] steps so far (global)
  int* hold;             // [N] (global)
  bool first;            // first cycle: iters is not read
  int max_iter;
  int* status;
};
template <int NT>
__device__ __forceinline__ void krylov_cg(const KMat<NT>& M, int N, const df32 inv_nm1, int j0, int step, int nc,
                                          const KColumns& C, unsigned char* sm) {
  constexpr int TPR = KMat<NT>::TPR, KPT = KMat<NT>::KPT, EPL = NT / 32;
  df32* s_rho = reinterpret_cast<df32*>(sm);                  // [16][NT]
  df32* s_part = s_rho + 16 * NT;                             // [16][TPR][NT]
  int* s_act = reinterpret_cast<int*>(s_part + 16 * kKT); // [16]
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, r = t % NT, g = t / NT;
  const bool mine = warp < nc;
  const int j = j0 + warp * step;
  df32 rho[EPL], f[EPL], h[EPL], w[EPL], rr, pq;
  float stop = 0.f, top = 0.f, last = 0.f;   // (r, R^{-1} r)/(N-1): tolerance, of b, of the last step
  float kmax = 0.f, unscale = 1.f;
  int it = 0, limit = 0, used = 0, act = 0;
  bool start = false;
  if (mine) {
    used = C.first ? 0 : *(volatile int*)&C.iters[j];
    limit = C.done[j] ? 0 : max(0, C.max_iter - used);
    start = C.w0 && !C.bad[j] && !C.done[j];
    act = 1;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const int k = lane + 32 * e;
      rho[e] = k < N ? ld_df(C.F + (int64_t)j * N + k) * inv_nm1 : df32(0.f, 0.f);
      if (k < N) kmax = fmaxf(kmax, fabsf(ld_df(C.K + k * N + k).hi));   // (K is positive semidefinite)
      if (start && k < N) w[e] = df32(C.w0[(int64_t)k * N + j], 0.f);
      if (C.w0) s_rho[warp * NT + k] = w[e];
    }
  }
  if (t < 16) s_act[t] = t < nc;
  // K times the vectors in s_rho of the active columns: thread (g, r) its entries of row r
  auto product = [&]() {
#pragma unroll 1
    for (int c = 0; c < nc; ++c) {
      if (!s_act[c]) continue;
      const df32* v = s_rho + c * NT + g * KPT;
      DFAcc a0, a1;
#pragma unroll
      for (int q = 0; q < KPT; q += 2) {   // KPT = 2, 8 or 32
        const float4 x = *reinterpret_cast<const float4*>(v + q);
        a0.add(M.k[q], df32(x.x, x.y));
        a1.add(M.k[q + 1], df32(x.z, x.w));
        if ((q & 7) == 6) { a0.renorm(); a1.renorm(); }
      }
      s_part[c * kKT + g * NT + r] = a0.value() + a1.value();
    }
    __syncthreads();
  };
  auto row = [&](int k) {
    df32 s[TPR];
#pragma unroll
    for (int q = 0; q < TPR; ++q) s[q] = s_part[warp * kKT + q * NT + k];
#pragma unroll
    for (int o = TPR / 2; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < o; ++q) s[q] = s[q] + s[q + o];
    return s[0];
  };
  if (C.w0) {   // rho = g - (I + K) w0 (the same for every column; without a start w = 0)
    __syncthreads();
    product();
    if (start)
#pragma unroll
      for (int e = 0; e < EPL; ++e) rho[e] = rho[e] - (w[e] + row(lane + 32 * e));
  }
  if (mine) {
    // rho and w times 2^-ex: N^2 max|K| max|rho| to about 2^60
    float rmax = 0.f;
#pragma unroll
    for (int e = 0; e < EPL; ++e) rmax = fmaxf(rmax, fmaxf(fabsf(rho[e].hi), fabsf(w[e].hi)));
    const unsigned kb = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(kmax, 1.f)));
    const unsigned rb = __reduce_max_sync(0xffffffffu, __float_as_uint(rmax));
    const int ex = max(-100, min(100, (int)(kb >> 23) - 127 + (int)(rb >> 23) - 127 + 2 * (31 - __clz(N)) + 2 - 60));
    const float sc = __uint_as_float((uint32_t)(127 - ex) << 23);
    unscale = __uint_as_float((uint32_t)(127 + ex) << 23);
    const double t2 = C.bb[j] * (double)inv_nm1.hi * __hiloint2double((1023 - 2 * ex) << 20, 0);
    top = (float)t2;
    stop = (float)(C.itol[j] * C.itol[j] * t2);
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      rho[e] = df32(rho[e].hi * sc, rho[e].lo * sc);
      w[e] = df32(w[e].hi * sc, w[e].lo * sc);
      s_rho[warp * NT + lane + 32 * e] = rho[e];
    }
  }
  while (__syncthreads_or(act)) {
    product();
    if (act) {
      df32 kr[EPL], d1, d2, d3;   // (rho, kr), (kr, kr), (rho + kr, h)
#pragma unroll
      for (int e = 0; e < EPL; ++e) {
        kr[e] = row(lane + 32 * e);
        d1 = fma(rho[e], kr[e], d1);
        d2 = fma(kr[e], kr[e], d2);
        d3 = fma(rho[e] + kr[e], h[e], d3);   // (h = 0 before the first step)
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        d1 = d1 + df_shfl_xor(d1, o);
        d2 = d2 + df_shfl_xor(d2, o);
        d3 = d3 + df_shfl_xor(d3, o);
      }
      // a non-finite value ends the column (the true residual reports it); so does a (p, S p) that
      // is not positive: rounding has used up this cycle
      last = d1.hi;
      if (!isfinite(d1.hi)) {
        if (lane == 0) atomicOr(C.status, DS_NONFINITE);
        act = 0;
      } else if (d1.hi <= stop || it >= limit) {
        act = 0;
      } else {
        df32 beta;
        if (it > 0) beta = df_div(d1, rr);
        pq = fma(beta, fma(beta, pq, d3 + d3), d1 + d2);
        rr = d1;
        if (!(pq.hi > 0.f) || !isfinite(pq.hi)) {
          act = 0;
        } else {
          const df32 alpha = df_div(rr, pq);
#pragma unroll
          for (int e = 0; e < EPL; ++e) {
            f[e] = it > 0 ? fma(beta, f[e], rho[e]) : rho[e];
            h[e] = it > 0 ? fma(beta, h[e], kr[e]) : kr[e];
            w[e] = fma(alpha, f[e], w[e]);
            rho[e] = rho[e] - alpha * (f[e] + h[e]);
            s_rho[warp * NT + lane + 32 * e] = rho[e];
          }
          ++it;
        }
      }
      if (!act && lane == 0) s_act[warp] = 0;
    }
  }
  if (mine) {
    const bool gain = last <= top;   // (false for NaN)
#pragma unroll
    for (int e = 0; e < EPL; ++e)
      if (lane + 32 * e < N)
        C.w[(int64_t)j * N + lane + 32 * e] = gain ? df32(w[e].hi * unscale, w[e].lo * unscale) : df32(0.f, 0.f);
    if (lane == 0) {
      C.iters[j] = used + it;
      C.hold[j] = gain ? 0 : 1;
    }
  }
  __syncthreads();
}

// ------------------------------------------------------------------ passes Z and R
// Both passes: u = HA T for a tile arrives as D[j][i] (lane j, tensor-memory column i), so that a
// thread owns one column j and RPT consecutive rows, its accesses to D and Z are contiguous
// across the warp, and column sums and maxima stay in the thread. For NT <= 64 the T operand holds
// 128 / NT copies of its columns, so that all 128 lanes carry work (copy d takes the rows
// [64 d / copies, ...) of a tile); at NT = 128 two such copies do not fit and half of the lanes idle.
// RESID = false: Z (+)= R^{-1} (b - u), then T += HA^T Z (out: T[k][jl]).
// RESID = true: B = D - R Z - u/(N-1) and rr[j] = ||B_j||^2 over the CTA's rows.
// NT <= 64: the next tile is loaded and sliced behind the products of the current one.
template <int NT, bool RESID>
__device__ __noinline__ void pass_rows(const KrylovParams& p, bool from_b, int c, int64_t row0, int64_t row1,
                                       KCta& cta, const int* s_hold, df32* __restrict__ out, double* rr_out) {
  using L = KLayout<NT>;
  using HI = KItems<NT>;
  constexpr int JC = L::JC, NB = L::NB;
  constexpr bool PRE = NT <= 64;                  // the next tile's loads are held in registers
  constexpr int LC = PRE ? 8 : 4;
  constexpr int CP = NT == 128 ? 1 : 128 / NT;    // copies
  constexpr int NSUB = NT == 32 ? 2 : 4;          // warps per copy and 32 lanes
  constexpr int GRP = CP * NSUB;                  // row groups of a tile: 8, 8, 4
  constexpr int RPT = kKR / GRP;                  // rows per thread: 8, 8, 16
  constexpr bool SPL = NT == 128;                 // level 1 of u in two sums
  unsigned char* sV = cta.smem + L::off_v;
  float* s_row = reinterpret_cast<float*>(cta.smem + L::off_row);         // [2][64] row scales of HA
  df32* s_r = reinterpret_cast<df32*>(cta.smem + L::off_row + 2 * 4 * kKR);   // [2][64] 1/r or r
  const float* s_col = reinterpret_cast<const float*>(cta.smem + L::off_col);   // [128] scales of T
  float* s_max = reinterpret_cast<float*>(cta.smem + L::off_max);         // [GRP][64], then [64] scales of V
  const int N = p.N, t = threadIdx.x, lane = t & 31, qd = (t >> 5) & 3, sub = t >> 7;
  const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  const int ln = 32 * qd + lane, jl = ln % JC, j = 64 * c + jl;
  const int copy = ln / JC;                       // NT = 128: lanes 64.. hold no column
  const bool mine = copy < CP && sub < NSUB, live = mine && j < N;
  // a column that is done or held keeps its Z: its right-hand side and w are zero
  const bool frozen = !RESID && live && s_hold[j];
  const int rg = mine ? copy * NSUB + sub : 0, r0 = rg * RPT;   // this thread's rows of the tile
  const uint32_t lead = warp == 0 ? elect_lane() : 0u;
  const uint32_t aT = smem_addr(cta.smem + L::off_t), aH = smem_addr(cta.smem + L::off_h), aV = smem_addr(sV);
  constexpr uint32_t hst = (NT / 8) * 128;
  const float tsc = s_col[min(ln, L::TROWS - 1)] * 0x1p-16f;
  const df32 inv_nm1(1.0 / (double)(N - 1));
  constexpr int NC = JC / 4;
  DFAcc acc[RESID ? 1 : NC];
  float rr = 0.f;
  double rr64 = 0.0;
  df32 x[PRE ? HI::N : 1][8];
  float xs[PRE ? HI::N : 1];
  auto load_x = [&](int64_t i0, int it, int slot) {
    const int64_t i = i0 + HI::row(warp, lane, it);
    const bool in = HI::live(warp, it) && i < row1;
    load_row8(x[slot], p.HAdf, i, HI::col(warp, lane, it), N, in);
    xs[slot] = p.hs[in ? i : 0];
  };
  auto load = [&](int64_t i0) {
    if (PRE)
#pragma unroll
      for (int it = 0; it < HI::N; ++it) load_x(i0, it, it);
  };
  auto slice = [&](int b, int64_t i0, int rb) {   // image b, row data rb (two of them at every NT)
#pragma unroll(PRE ? HI::N : 1)
    for (int it = 0; it < HI::N; ++it) {
      const int q = PRE ? it : 0;
      if (!PRE) load_x(i0, it, 0);
      // 1/xs: xs is a power of two (2^e -> 2^-e by the exponent field)
      const float sc = __uint_as_float((254u << 23) - __float_as_uint(xs[q]));
      if (HI::live(warp, it)) {
        Slices8 sl;
        sl.make(x[q], sc);
        sl.store(cta.smem + L::off_h + b * (kSl * L::HP) + core_idx(HI::row(warp, lane, it), HI::col(warp, lane, it), NT) * 2,
                 L::HP);
      }
    }
    if (t < kKR) {
      const int64_t i = i0 + t;
      s_row[rb * kKR + t] = i < row1 ? p.hs[i] : 1.f;
      s_r[rb * kKR + t] = i < row1 ? (RESID ? p.rdf[i] : p.rinv[i]) : df32(0.f, 0.f);
    }
    fence_async_smem();
  };
  auto issue_u = [&](int b) {
    if (warp == 0) {
      tc_fence_after();
      issue_levels<NT / 16, 4, SPL, kKR, false, false, L::TP, 256, L::HP, 256>(
          cta.tmem, umma_desc(aT, 128, hst), umma_desc(aH + b * (kSl * L::HP), 128, hst), cta.mbar, lead);
    }
  };
  int b = 0, rb = 0;
  if (row0 < row1) {
    load(row0);
    slice(0, row0, 0);
    tc_fence_before();
    __syncthreads();
    issue_u(0);
  }
  for (int64_t i0 = row0; i0 < row1 && cta.ok; i0 += kKR, b ^= NB - 1, rb ^= 1) {
    const bool more = i0 + kKR < row1;
    // this thread's entries, in flight behind the products (NT = 128: four rows at a time)
    constexpr int DE = PRE ? RPT : LC;
    df32 d[DE], z[RESID ? DE : RPT];
    auto entries = [&](int q0) {
#pragma unroll
      for (int q = 0; q < DE; ++q) {
        const int64_t i = i0 + r0 + q0 + q;
        const bool in = live && i < row1;
        const int64_t e = in ? i * N + j : 0;
        df32 dv(0.f, 0.f), zv(0.f, 0.f);
        if (!RESID && from_b) dv.hi = p.B[e];
        else dv = p.Ddf[e];
        if (RESID || from_b) zv = p.Zdf[e];
        d[q] = in && !frozen ? dv : df32(0.f, 0.f);
        z[(RESID ? 0 : q0) + q] = in ? zv : df32(0.f, 0.f);
      }
    };
    entries(0);
    if (RESID && NB == 2 && more) {
      load(i0 + kKR);
      slice(b ^ 1, i0 + kKR, rb ^ 1);
    }
    k_wait(cta);
    float mx = 0.f;
    if (mine || 32 * qd < JC * CP) {   // (the second condition is uniform in the warp)
#pragma unroll
      for (int q0 = 0; q0 < RPT; q0 += LC) {
        if (!PRE && q0 > 0) entries(q0);
        float lv[SPL ? 6 : 5][LC];
        tmem_ld_levels<(SPL ? 6 : 5), LC>(cta.tmem + ((uint32_t)(32 * qd) << 16) + r0 + q0, kKR, lv);
#pragma unroll
        for (int q = 0; q < LC; ++q) {
          const int rq = r0 + q0 + q;
          const int64_t i = i0 + rq;
          if (!(live && i < row1)) continue;
          float s, l;
          join_members<SPL>(lv, q, s, l);
          const float sr = s_row[rb * kKR + rq], f = tsc * sr;
          const df32 u = df_fast2sum(s * f, l * f);
          const df32 ri = s_r[rb * kKR + rq];
          const int qd0 = PRE ? q0 + q : q;
          if (RESID) {
            const df32 res = d[qd0] - fma(ri, z[RESID ? qd0 : 0], u * inv_nm1);
            rr = __fmaf_rn(res.hi, res.hi, rr);
            p.B[i * N + j] = res.hi;
          } else {
            const df32 zn = z[q0 + q] + (d[qd0] - u) * ri;
            p.Zdf[i * N + j] = zn;
            // times the HA row's scale: HA_ik z_ij = (HA_ik / s_i) (z_ij s_i)
            z[q0 + q] = df32(zn.hi * sr, zn.lo * sr);
            mx = fmaxf(mx, fabsf(z[q0 + q].hi));
          }
        }
      }
    }
    if constexpr (RESID) {
      rr64 += (double)rr;
      rr = 0.f;
      if (NB == 1 && more) slice(0, i0 + kKR, rb ^ 1);
    } else {
      if (mine) s_max[rg * 64 + jl] = mx;
      __syncthreads();
      if (mine) {
        float m2 = mx;
#pragma unroll
        for (int q = 0; q < GRP; ++q) m2 = fmaxf(m2, s_max[q * 64 + jl]);
        float sc, inv;
        pow2_of(m2, sc, inv);
#pragma unroll
        for (int q0 = 0; q0 < RPT; q0 += 8) {
          const df32 y[8] = {z[q0], z[q0 + 1], z[q0 + 2], z[q0 + 3], z[q0 + 4], z[q0 + 5], z[q0 + 6], z[q0 + 7]};
          Slices8 sl;
          sl.make(y, sc);
          sl.store(sV + core_idx(jl, r0 + q0, kKR) * 2, L::VP);
        }
        if (rg == 0) s_max[GRP * 64 + jl] = inv;
      }
      fence_async_smem();
      tc_fence_before();
      __syncthreads();
      if (warp == 0) {
        tc_fence_after();
        // T[k][jl]: A = the HA tile MN-major (M = k), B = the Z tile K-major
        issue_levels<kKR / 16, 5, false, JC, true, false, L::HP, 2 * hst, L::VP, 256>(
            cta.tmem, umma_desc(aH + b * (kSl * L::HP), hst, 128), umma_desc(aV, 128, 1024), cta.mbar, lead);
      }
      if (NB == 2 && more) {
        load(i0 + kKR);
        slice(b ^ 1, i0 + kKR, rb ^ 1);
      }
      k_wait(cta);
      if (32 * qd < N) {   // uniform in the warp
#pragma unroll
        for (int q0 = 0; q0 < NC; q0 += LC) {
          float lv[kLv][LC];
          tmem_ld_levels<kLv, LC>(cta.tmem + ((uint32_t)(32 * qd) << 16) + sub * NC + q0, JC, lv);
#pragma unroll
          for (int q = 0; q < LC; ++q) {
            float s, l, tt, e;
            join_rows(lv, q, s, l);
            const float f = s_max[GRP * 64 + sub * NC + q0 + q] * 0x1p-16f;
            df_two_sum(acc[q0 + q].s, s * f, tt, e);
            acc[q0 + q].s = tt;
            acc[q0 + q].c = __fadd_rn(acc[q0 + q].c, __fmaf_rn(l, f, e));
            acc[q0 + q].renorm();
          }
        }
      }
      if (NB == 1 && more) slice(0, i0 + kKR, rb ^ 1);
    }
    tc_fence_before();
    __syncthreads();
    if (more) issue_u(NB == 2 ? b ^ 1 : 0);
  }
  if constexpr (RESID) {
    double* red = reinterpret_cast<double*>(cta.smem + L::off_h);   // [GRP][64]
    __syncthreads();
    if (mine) red[rg * 64 + jl] = rr64;
    __syncthreads();
    if (t < JC) {
      double s = 0.0;
      for (int q = 0; q < GRP; ++q) s += red[q * 64 + t];
      rr_out[64 * c + t] = s;
    }
    __syncthreads();
  } else {
    const int NJ = min(JC, N);
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const int col = sub * NC + q;
      if (ln < N && col < NJ) out[ln * NJ + col] = acc[q].value();
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ the solve
// CTA b of the G co-resident CTAs of one problem (the grid, or a team of a batched launch). The
// rows are split over G / CG row blocks; at NT = 128 two CTAs share a row block, one per column
// group (a single CTA takes both groups in turn). Partial sums are reduced in a fixed order.
template <int NT>
__device__ void krylov_body(const KrylovParams& p, const int G, const int b, GridBarrier& bar, KCta& cta) {
  using L = KLayout<NT>;
  constexpr int JC = L::JC;
  double* s_dn2 = reinterpret_cast<double*>(cta.smem + L::off_scal);
  double* s_true = s_dn2 + NT;
  double* s_prev = s_true + NT;
  double* s_itol = s_prev + NT;
  double* s_tmp = s_itol + NT;
  double* s_bb = s_tmp + NT;
  int* s_done = reinterpret_cast<int*>(s_bb + NT);
  int* s_bad = s_done + NT;     // rejected learned starts, then the columns held in this cycle
  double* scratch = reinterpret_cast<double*>(cta.smem + L::off_scr);
  const int N = p.N, t = threadIdx.x, NJ = min(JC, N);
  if (dynamic_smem_bytes() < (unsigned)L::bytes) {
    if (t == 0) atomicOr(p.status, DS_SMEM);
    return;
  }
  const int ngr = (N + JC - 1) / JC;              // column groups in use
  const int RB = max(1, G / ngr);                 // row blocks
  const int rb = G >= ngr ? b / ngr : 0;
  const int c0 = G >= ngr ? b % ngr : 0, c1 = G >= ngr ? c0 + 1 : ngr;
  const bool has_rows = rb < RB;
  const int64_t rows_per = (p.m + RB - 1) / RB;
  const int64_t row0 = has_rows ? imin64(p.m, (int64_t)rb * rows_per) : p.m;
  const int64_t row1 = imin64(p.m, row0 + rows_per);
  const int64_t PS = krylov_part(N);
  auto part_of = [&](int q, int c) { return p.part + ((int64_t)q * ngr + c) * PS; };
  const double inv_nm1 = 1.0 / (double)(N - 1);
  const bool prof = p.prof != nullptr && b == 0 && t == 0;
  unsigned long long ph[PH_COUNT] = {0, 0, 0, 0, 0, 0, 0, 0};
  unsigned long long tp = prof ? global_ns() : 0ull;
  auto tick = [&](int slot) {
    if (prof) {
      const unsigned long long now = global_ns();
      ph[slot] += now - tp;
      tp = now;
    }
  };
  int par = 0;
  bool ok = true;
  if (t < NT) {
    s_done[t] = t >= N;
    s_true[t] = -1.0;
    s_prev[t] = 0.0;
    s_dn2[t] = 0.0;
    s_itol[t] = fmin(0.5, fmax(0.02 * p.tol, 1e-14));
  }
  __syncthreads();
  // a reduction over the G CTAs' per-column sums (s_tmp in, s_tmp out)
  auto column_totals = [&]() -> bool {
    if (t < NT) p.rrpart[((int64_t)par * G + b) * NT + t] = s_tmp[t];
    if (!bar.sync()) return false;
    total_columns<NT>(p.rrpart + (int64_t)par * G * NT, G, N, s_tmp, scratch);
    par ^= 1;
    return true;
  };
  tick(PH_SETUP);

  int cycles = 0;
  for (;;) {
    const bool from_b = cycles > 0;
    if (from_b || p.phase != 2) {
    // ---- pass G and its reduction
    for (int c = c0; c < c1; ++c)
      if (has_rows) pass_gram<NT>(p, from_b, c, row0, row1, cta, part_of(rb, c));
    tick(PH_SETUP);
    if (!(ok = bar.sync() && cta.ok)) break;
    tick(PH_BAR1);
    reduce_parts(p.part, PS, ngr * PS, RB, ngr, 2 * N * NJ + 128, G, b,
                 reinterpret_cast<df32*>(scratch), [&](int c, int e, df32 v) {
      const int nj = min(JC, N - 64 * c);
      if (e < N * NJ) {
        const int k = e / NJ, jl = e % NJ;
        if (jl < nj) p.Kred[k * N + 64 * c + jl] = df32((double)v * inv_nm1);
      } else if (e < 2 * N * NJ) {
        const int k = (e - N * NJ) / NJ, jl = (e - N * NJ) % NJ;
        if (jl < nj) p.Fred[(int64_t)(64 * c + jl) * N + k] = v;
      } else {
        const int which = (e - 2 * N * NJ) / 64, jl = (e - 2 * N * NJ) % 64;
        if (jl < nj) p.sums[which * N + 64 * c + jl] = v;
      }
    });
    tick(PH_RED);
    if (!from_b && p.phase == 1) return;
    if (!(ok = bar.sync())) break;
    tick(PH_BAR2);
    }
    if (t < N) {
      const float2 a = __ldcg(reinterpret_cast<const float2*>(p.sums + t));
      const float2 q = __ldcg(reinterpret_cast<const float2*>(p.sums + N + t));
      if (!from_b) {
        s_dn2[t] = (double)a.x + (double)a.y;
        if (s_dn2[t] == 0.0) { s_done[t] = 1; s_true[t] = 0.0; }
      }
      s_bb[t] = (double)q.x + (double)q.y;
    }
    __syncthreads();
    if (!from_b && p.w0) {
      // the learned start's true residual judges it: a column whose start is non-finite or (unless
      // warm_accept) whose residual is larger than the zero start's (d_j) starts from w = 0
      if (t < NT) {
        const double v = t < N ? p.wnorm[t] : 0.0;
        const bool zero = t >= N || s_dn2[t] == 0.0;
        s_bad[t] = !zero && (p.warm_accept ? !isfinite(v) : !(v <= s_dn2[t])) ? 1 : 0;
        if (b == 0 && t < N) p.col_warm[t] = zero ? 0.0 : sqrt(v / s_dn2[t]);
      }
      const int nbad = __syncthreads_count(t < NT && s_bad[t]);
      if (b == 0 && t == 0) p.status[2] = nbad;
    }
    // ---- the recurrences, column j on CTA j mod G
    if (b < N) {
      KMat<NT> M;
      const int r = t % NT, g = t / NT;
#pragma unroll
      for (int q = 0; q < KMat<NT>::KPT; ++q) {
        const int k = g * KMat<NT>::KPT + q;
        M.k[q] = df32(0.f, 0.f);
        if (k < N && r < N) {
          M.k[q] = ld_df(p.Kred + k * N + r);
        }
      }
      const KColumns C{p.Kred, p.Fred, p.wred, s_bb, s_itol, s_done, s_bad, from_b ? nullptr : p.w0,
                       p.col_iters, p.hold, !from_b, p.max_iter, p.status};
      for (int j = b; j < N; j += 16 * G)
        krylov_cg<NT>(M, N, df32(inv_nm1), j, G, min(16, (N - j + G - 1) / G), C, cta.smem);
    }
    tick(PH_PASS);
    if (!(ok = bar.sync())) break;
    tick(PH_BAR1);
    if (t < NT) s_bad[t] = t < N && (__ldcg(p.hold + t) || (from_b && s_done[t])) ? 1 : 0;
    __syncthreads();
    // ---- pass Z and the reduction of T (W = T/(N-1))
    for (int c = c0; c < c1; ++c)
      if (has_rows) {
        stage_columns<NT, L::TROWS, JC>(p.wred, 64 * c, N, cta.smem + L::off_t, reinterpret_cast<float*>(cta.smem + L::off_col));
        __syncthreads();
        pass_rows<NT, false>(p, from_b, c, row0, row1, cta, s_bad, part_of(rb, c), nullptr);
      }
    tick(PH_REFRESH);
    if (!(ok = bar.sync() && cta.ok)) break;
    tick(PH_BAR1);
    reduce_parts(p.part, PS, ngr * PS, RB, ngr, N * NJ, G, b, reinterpret_cast<df32*>(scratch),
                 [&](int c, int e, df32 v) {
      const int k = e / NJ, jl = e % NJ;
      if (jl < min(JC, N - 64 * c)) {
        p.Tred[(int64_t)(64 * c + jl) * N + k] = v;
        p.W[k * N + 64 * c + jl] = (double)v * inv_nm1;
      }
    });
    tick(PH_RED);
    if (!(ok = bar.sync())) break;
    tick(PH_BAR2);
    // ---- pass R: the true residual
    if (t < NT) s_tmp[t] = 0.0;
    __syncthreads();
    for (int c = c0; c < c1; ++c)
      if (has_rows) {
        stage_columns<NT, L::TROWS, JC>(p.Tred, 64 * c, N, cta.smem + L::off_t, reinterpret_cast<float*>(cta.smem + L::off_col));
        __syncthreads();
        pass_rows<NT, true>(p, from_b, c, row0, row1, cta, s_bad, nullptr, s_tmp);
      }
    if (!(ok = column_totals() && cta.ok)) break;
    ++cycles;
    if (t < N) {
      // a non-finite residual or ||d_j|| (NaN or Inf in the inputs) ends the column with the
      // non-finite status
      const bool fin = isfinite(s_dn2[t]) && isfinite(s_tmp[t]);
      if (!fin) atomicOr(p.status, DS_NONFINITE);
      const double tr = !fin ? (double)NAN : (s_dn2[t] > 0.0 ? sqrt(s_tmp[t] / s_dn2[t]) : 0.0);
      s_true[t] = tr;
      const int used = *(volatile int*)&p.col_iters[t];
      // done: converged, non-finite, held, stalled (no halving over a cycle) or out of steps
      if (!fin || tr <= p.tol || s_bad[t] || (cycles >= 2 && tr > 0.5 * s_prev[t]) || used >= p.max_iter) s_done[t] = 1;
      s_prev[t] = tr;
      s_itol[t] = fmin(0.5, fmax(tr > 0.0 ? 0.02 * p.tol / tr : 0.5, 1e-14));
    }
    const int all_done = __syncthreads_and(t >= N || s_done[t]);
    tick(PH_REFRESH);
    if (all_done || cycles > p.max_refine) break;
  }
  if (b == 0) {
    if (t < N) {
      p.col_relres[t] = s_true[t];
      p.col_true[t] = s_true[t];
      if (ok && !(s_true[t] >= 0.0 && s_true[t] <= p.tol)) atomicOr(p.status, DS_NOT_CONVERGED);
    }
    if (t == 0) p.status[1] = cycles;
    if (prof)
      for (int q = 0; q < PH_COUNT; ++q) p.prof[q] = ph[q];
  }
}

// tensor memory and the completion barrier of a CTA (all 512 columns: one CTA per SM)
__device__ __forceinline__ void krylov_begin(KCta& cta, unsigned char* smem, uint64_t* mbar, uint32_t* tmem_slot,
                                             int* status) {
  if (threadIdx.x == 0) mbar_init(mbar);
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cta = KCta{smem, *tmem_slot, mbar, 0u, status, true};
}
__device__ __forceinline__ void krylov_end(const KCta& cta) {
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(cta.tmem), "r"(512));
}

}  // namespace enkf
