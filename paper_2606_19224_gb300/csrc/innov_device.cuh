// The row-range form of the innovation step (Algorithm 1: Zobs = H X_f, HA = Zobs - zbar 1^T,
// D = y 1^T + E - Zobs) with the observation perturbations E drawn from Philox4x32-10 and
// Box-Muller: shared by the single-analysis innovations kernel (kernels_fp.cu) and the batched
// kernel (kernels_batch.cu).
#pragma once

#include "cg_device.cuh"

namespace enkf {

// ------------------------------------------------------------------ K1: innovations
// Standard normals of members (j, j + 1), j even, from one Philox block and one Box-Muller
// pair (the definition of perturbation_normal for both members, computed once).
__device__ __forceinline__ void perturbation_pair(int64_t i, int j, uint64_t seed, uint64_t counter,
                                                  double& n_even, double& n_odd) {
  uint32_t c0 = (uint32_t)i, c1 = (uint32_t)(j >> 1), c2 = (uint32_t)counter, c3 = (uint32_t)(counter >> 32);
  philox4x32_10(c0, c1, c2, c3, (uint32_t)seed, (uint32_t)(seed >> 32));
  const uint64_t x1 = ((uint64_t)c0 << 21) | (c1 >> 11);
  const uint64_t x2 = ((uint64_t)c2 << 21) | (c3 >> 11);
  const double u1 = ((double)x1 + 0.5) * 0x1p-53;
  const double u2 = (double)x2 * 0x1p-53;
  const double rho = sqrt(-2.0 * log(u1));
  double sn, cs;
  sincos(6.283185307179586 * u2, &sn, &cs);
  n_even = rho * cs;
  n_odd = rho * sn;
}

// The same pair in single precision, for the modes that compute in FP32 (FP32 and the
// tensor-core modes): the same Philox block and the same 53-bit uniforms u1 = (x1 + 1/2)
// 2^-53 and u2 = x2 2^-53, rounded to float, with float log (log1p of -(1 - u1) when
// u1 >= 1/2, where 1 - u1 is formed exactly from the integer), square root and sin/cos of
// pi 2 u2. Each normal is within about 1e-7 (relative to its size) of the FP64 form, and the
// FP64 log and sincos, which dominate the innovations on a GPU whose FP64 rate is a small
// fraction of its FP32 rate, are avoided.
// Conversions that stay off the FP64 pipe (two operations per clock per SM on this part; the
// 64-bit conversion instructions run there too).
// The float nearest to the 53-bit integer a 2^21 + b (a < 2^32, b < 2^21), as a 64-bit to
// float conversion rounds it, from 32-bit conversions: for a >= 2^25 the rounding drops at
// least two bits of a, so ORing "b != 0" into its lowest bit supplies the sticky bit without
// touching the round bit; otherwise a >> 1 and ((a & 1) << 21) | b are exact floats and one
// FP32 fused multiply-add rounds their exact sum once.
__device__ __forceinline__ float u53_to_float(uint32_t a, uint32_t b) {
  if (a >= (1u << 25)) return __uint2float_rn(a | (b != 0u ? 1u : 0u)) * 0x1p21f;
  return fmaf(__uint2float_rn(a >> 1), 0x1p22f, __uint2float_rn(((a & 1u) << 21) | b));
}
// (double)x by exponent rebias and mantissa shift for normal x and zero; subnormals,
// infinities and NaN take the conversion instruction.
__device__ __forceinline__ double f2d_bits(float x) {
  const uint32_t u = __float_as_uint(x);
  const uint32_t e = (u >> 23) & 0xFFu;
  if ((u & 0x7FFFFFFFu) == 0u) return __longlong_as_double((long long)((uint64_t)u << 32));
  if (e == 0u || e == 0xFFu) return (double)x;
  return __longlong_as_double((long long)(((uint64_t)(u >> 31) << 63) | ((uint64_t)(e + 896u) << 52) |
                                          ((uint64_t)(u & 0x7FFFFFu) << 29)));
}
// hi + lo rounded to FP64, as (double)hi + (double)lo: one FP64 addition
__device__ __forceinline__ double df_to_double(const df32& v) { return f2d_bits(v.hi) + f2d_bits(v.lo); }
// df32(x) for a double x: hi = x rounded to float, lo = (x - hi) rounded to float, with the
// widening of hi done by f2d_bits (three FP64-pipe operations instead of four)
__device__ __forceinline__ df32 df_from_double(double x) {
  const float hi = __double2float_rn(x);
  return df32(hi, __double2float_rn(x - f2d_bits(hi)));
}

__device__ __forceinline__ void perturbation_pair_f32(int64_t i, int j, uint64_t seed, uint64_t counter,
                                                      float& n_even, float& n_odd) {
  uint32_t c0 = (uint32_t)i, c1 = (uint32_t)(j >> 1), c2 = (uint32_t)counter, c3 = (uint32_t)(counter >> 32);
  philox4x32_10(c0, c1, c2, c3, (uint32_t)seed, (uint32_t)(seed >> 32));
  const uint64_t x1 = ((uint64_t)c0 << 21) | (c1 >> 11);
  float lg;
  if (x1 < (1ull << 52)) {
    lg = logf(fmaf(u53_to_float(c0, c1 >> 11), 0x1p-53f, 0x1p-54f));
  } else {
    const uint64_t y1 = (1ull << 53) - x1;   // 1 - u1 = (y1 - 1/2) 2^-53, y1 <= 2^52
    const float w = fmaf(u53_to_float((uint32_t)(y1 >> 21), (uint32_t)(y1 & 0x1FFFFFu)), 0x1p-53f, -0x1p-54f);
    lg = log1pf(-w);
  }
  const float rho = sqrtf(-2.f * lg);
  float sn, cs;
  sincospif(u53_to_float(c2, c3 >> 11) * 0x1p-52f, &sn, &cs);
  n_even = rho * cs;
  n_odd = rho * sn;
}
__device__ __forceinline__ void perturbation_pair_f32(int64_t i, int j, uint64_t seed, uint64_t counter,
                                                      double& n_even, double& n_odd) {
  float a, b;
  perturbation_pair_f32(i, j, seed, counter, a, b);
  n_even = (double)a;
  n_odd = (double)b;
}

// Rows [i_begin, i_end) of the observation operator, one warp per row: `warp` is this warp's
// index among `nwarps` warps sharing the range. Lane l owns members 2l, 2l + 1, 2l + 64,
// 2l + 65, so each perturbation pair is drawn once.
template <typename VT>
__device__ __forceinline__ void innov_rows_f64(
    const VT* __restrict__ Xf, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
    const double* __restrict__ w, const double* __restrict__ y, const double* __restrict__ r,
    const double* __restrict__ E, int emode, uint64_t seed, uint64_t counter, int N,
    double* __restrict__ HA64, double* __restrict__ D, int64_t i_begin, int64_t i_end, int64_t warp, int64_t nwarps,
    int64_t out0 = 0 /* outputs are written from row out0 on */) {
  // FP64 instructions are scarce on this part (2 per clock per SM): 1/N is applied as a
  // product and members 64..127 are skipped when N <= 64
  const int lane = threadIdx.x & 31;
  const double inv_n = 1.0 / (double)N;
  const bool wide = N > 64;   // members 64..127 present (warp-uniform)
  for (int64_t i = i_begin + warp; i < i_end; i += nwarps) {
    double z[4] = {0.0, 0.0, 0.0, 0.0};
    const int k0 = rowptr[i], k1 = rowptr[i + 1];
    for (int k = k0; k < k1; ++k) {
      const double wk = w[k];
      const VT* xr = Xf + (int64_t)col[k] * N;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = 2 * lane + (q & 1) + 64 * (q >> 1);
        if (j < N) z[q] = fma(wk, (double)xr[j], z[q]);
      }
    }
    double s = z[0] + z[1];
    if (wide) s += z[2] + z[3];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double zbar = s * inv_n;
    const double yi = y[i], ri = r[i];
    const double sr = emode == 2 ? sqrt(ri) : 0.0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int jp = 2 * lane + 64 * h;   // even member of the pair
      if (jp >= N) continue;
      double nrm[2] = {0.0, 0.0};
      if (emode == 2) perturbation_pair(i, jp, seed, counter, nrm[0], nrm[1]);
      const int64_t ein = i * N + jp, e0 = ein - out0 * N;   // of the inputs, of the outputs
      double hv[2], dv[2];
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        double pert = 0.0;
        if (jp + b < N) {
          if (emode == 1) pert = E[ein + b];
          else if (emode == 2) pert = sr * nrm[b];
        }
        hv[b] = z[2 * h + b] - zbar;
        dv[b] = (yi - z[2 * h + b]) + pert;
      }
      if ((N & 1) == 0) {
        // both members present and e0 even: one 8- or 16-byte store per array per lane, so a
        // warp writes contiguous row segments
        *reinterpret_cast<double2*>(HA64 + e0) = make_double2(hv[0], hv[1]);
        *reinterpret_cast<double2*>(D + e0) = make_double2(dv[0], dv[1]);
      } else {
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          if (jp + b >= N) continue;
          const int64_t e = e0 + b;
          HA64[e] = hv[b];
          D[e] = dv[b];
        }
      }
    }
  }
}

// What the products on the tensor cores (krylov.cuh) take from the innovations besides HA and D (FP32
// ensembles): a power of two above the largest |HA| of each row, and the largest |HA_ik| times the row's
// weight 1/sqrt(r_i) (atomic maximum of the float bits). senkf: the weight is 1/sqrt(s_i) instead,
// s_i = |HA_i|^2 + (N-1) r_i, and goes to wsq. Outputs are written from row row0 on.
struct InnovRows {
  float* scale = nullptr;
  const df32* rsq = nullptr;
  unsigned* umax = nullptr;
  int64_t row0 = 0;
  bool senkf = false;
  df32* wsq = nullptr;
};
// 1/sqrt(s) in double-float: the FP32 value y and two terms of its correction, e = 1 - s y^2 about 2^-22
__device__ __forceinline__ df32 df_rsqrt(const df32& s) {
  const float y = rsqrtf(s.hi);
  const df32 y2 = df32(y, 0.f) * df32(y, 0.f);
  const df32 e = df32(1.f, 0.f) - s * y2;
  return df32(y, 0.f) + df32(y, 0.f) * (e * df32(fmaf(0.375f, e.hi, 0.5f), 0.f));
}

// The same rows for FP32 ensembles (the FP32 and tensor-core modes), in double-float (FP32
// pair) arithmetic: this part issues FP32 at 64x its FP64 rate, and the FP64 version spends
// its time in FP64 adds and FP32<->FP64 conversions. z = sum w_k x_k accumulates exact
// products of the double-float weight and the FP32 member value, z-bar is a double-float warp
// sum (each lane adds the same operands in the same order: the double-float sum is
// commutative), HA = z - z-bar and D = (y - z) + E are double-float (about 48 significant
// bits, the precision of the HAdf and Ddf arrays they fill), E = sqrt(r_i) times the FP32
// normal as an exact double-float product; HA32 and B32 are the high parts, and only the
// FP64 copy of D is widened per element.
//
// A row takes the lanes of half a warp for N <= 64 (HALF) and of a whole one otherwise, four members each
// (2 l, 2 l + 1 and the same 32 or 64 further on, so that each perturbation pair is drawn once). What bounds it is
// latency: a row was a chain of four dependent loads, and the tree of its mean took as many
// instructions for two members per lane as for four. The offsets, first columns and row values of 32 rows are read
// ahead, lane q for row q of the warp, and each row's first gather is in flight behind the row before.
template <typename VT, bool HALF>
__device__ __forceinline__ void innov_rows_df(
    const VT* __restrict__ Xf, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
    const double* __restrict__ w, const double* __restrict__ y, const double* __restrict__ r,
    const double* __restrict__ E, int emode, uint64_t seed, uint64_t counter, int N,
    double* __restrict__ D, float* __restrict__ HA32, float* __restrict__ B32, df32* __restrict__ HAdf,
    df32* __restrict__ Ddf, int64_t i_begin, int64_t i_end, int64_t warp, int64_t nwarps, unsigned* hamax,
    const InnovRows kr) {
  static_assert(sizeof(VT) == 4, "double-float innovations take an FP32 ensemble");
  constexpr int GL = HALF ? 16 : 32, RW = 32 / GL;   // lanes per row, rows per warp
  const int lane = threadIdx.x & 31, gl = lane % GL, sub = lane / GL;
  const unsigned group = HALF ? 0xFFFFu << (16 * sub) : 0xffffffffu;
  float hmax = 0.f;   // largest |HA| of the warp's rows (hamax: atomic maximum of the float bits)
  float umax = 0.f;   // largest |HA| / sqrt(r) of the warp's rows
  const df32 inv_n(1.0 / (double)N);
  const bool even = (N & 1) == 0, vec = even && (reinterpret_cast<uintptr_t>(Xf) & 7) == 0;
  bool in[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) in[q] = 2 * gl + (q & 1) + 2 * GL * (q >> 1) < N;
  // the row's members of this lane
  auto gather = [&](int c, float (&x)[4]) {
    const VT* xr = Xf + (int64_t)c * N + 2 * gl;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (vec) {   // both members of a pair, at an 8-byte boundary
        const float2 v = in[2 * h] ? *reinterpret_cast<const float2*>(xr + 2 * GL * h) : make_float2(0.f, 0.f);
        x[2 * h] = v.x;
        x[2 * h + 1] = v.y;
      } else {
        x[2 * h] = in[2 * h] ? (float)xr[2 * GL * h] : 0.f;
        x[2 * h + 1] = in[2 * h + 1] ? (float)xr[2 * GL * h + 1] : 0.f;
      }
    }
  };
  // The warp's rows are i0 + q nwarps, q = 0, 1, ...; the per-row values that come from FP64
  // inputs (y_i, sqrt(r_i) and the weight of the row's first operator entry as double-float
  // pairs) are formed for 32 rows at a time, lane q for row i0 + q nwarps, and handed to the
  // other lanes by shuffles: one FP64 evaluation per row instead of one per lane.
  for (int64_t i0 = i_begin + warp; i0 < i_end; i0 += 32 * nwarps) {
    const int64_t il = i0 + (int64_t)lane * nwarps;
    df32 y_l, s_l, w_l, r_l;
    int k_l = 0, n_l = 0, c_l = 0;   // first entry, entries after it (-1: none), its column
    float q_l = 0.f;
    if (il < i_end) {
      k_l = rowptr[il];
      n_l = rowptr[il + 1] - k_l - 1;
      if (kr.umax && !kr.senkf) q_l = kr.rsq[il].hi;
      if (kr.senkf) r_l = df_from_double(r[il]);
      y_l = df_from_double(y[il]);
      if (emode == 2) s_l = df_from_double(sqrt(r[il]));
      if (n_l >= 0) {
        c_l = col[k_l];
        w_l = df_from_double(w[k_l]);
      }
    }
    float xn[4];
    gather(__shfl_sync(0xffffffffu, c_l, sub), xn);   // (column 0 where there is no entry: weight 0)
#pragma unroll 1
    for (int q32 = 0; q32 < 32; q32 += RW) {
      const int64_t i = i0 + (int64_t)(q32 + sub) * nwarps;
      if (i0 + (int64_t)q32 * nwarps >= i_end) break;   // warp-uniform
      const bool row = i < i_end;
      const int src = q32 + sub;
      const df32 yd(__shfl_sync(0xffffffffu, y_l.hi, src), __shfl_sync(0xffffffffu, y_l.lo, src));
      const df32 sr(__shfl_sync(0xffffffffu, s_l.hi, src), __shfl_sync(0xffffffffu, s_l.lo, src));
      const df32 w0(__shfl_sync(0xffffffffu, w_l.hi, src), __shfl_sync(0xffffffffu, w_l.lo, src));
      const int more = __shfl_sync(0xffffffffu, n_l, src), k0 = __shfl_sync(0xffffffffu, k_l, src);
      const float wq = __shfl_sync(0xffffffffu, q_l, src);
      df32 z[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (more >= 0) z[q] = w0 * df32(xn[q], 0.f);
      gather(__shfl_sync(0xffffffffu, c_l, min(src + RW, 31)), xn);
      for (int k = 1; k <= more; ++k) {
        const df32 wk = df_from_double(w[k0 + k]);
        float x[4];
        gather(col[k0 + k], x);
#pragma unroll
        for (int q = 0; q < 4; ++q) z[q] = fma(wk, df32(x[q], 0.f), z[q]);
      }
      __syncwarp();
      df32 s = (z[0] + z[1]) + (z[2] + z[3]);   // (zeros past N)
#pragma unroll
      for (int o = GL / 2; o > 0; o >>= 1)
        s = s + df32(__shfl_xor_sync(0xffffffffu, s.hi, o), __shfl_xor_sync(0xffffffffu, s.lo, o));
      const df32 zbar = s * inv_n;
      df32 hv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        hv[q] = z[q] - zbar;
        if (in[q] && row) hmax = fmaxf(hmax, fabsf(hv[q].hi));
      }
      if (kr.umax) {
        float rm = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (in[q]) rm = fmaxf(rm, fabsf(hv[q].hi));
        rm = __uint_as_float(__reduce_max_sync(group, __float_as_uint(rm)));
        float wt = wq;
        if (kr.senkf) {
          df32 q2;
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (in[q]) q2 = fma(hv[q], hv[q], q2);
#pragma unroll
          for (int o = GL / 2; o > 0; o >>= 1)
            q2 = q2 + df32(__shfl_xor_sync(0xffffffffu, q2.hi, o), __shfl_xor_sync(0xffffffffu, q2.lo, o));
          const df32 rs = df_rsqrt(q2 + df32((float)(N - 1), 0.f) *
                                            df32(__shfl_sync(0xffffffffu, r_l.hi, src), __shfl_sync(0xffffffffu, r_l.lo, src)));
          if (row && gl == 0) kr.wsq[i - kr.row0] = rs;
          wt = rs.hi;
        }
        if (row) {
          umax = fmaxf(umax, rm * wt);
          // the exponent field of the power of two above rm (bounded away from both ends of the range)
          const int Ex = max(40, min(252, (int)(__float_as_uint(rm) >> 23)));
          if (kr.scale && gl == 0) kr.scale[i - kr.row0] = __uint_as_float((uint32_t)(Ex + 1) << 23);
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int jp = 2 * gl + 2 * GL * h;   // even member of the pair
        if (!in[2 * h] || !row) continue;
        float nrm[2] = {0.f, 0.f};
        if (emode == 2) perturbation_pair_f32(i, jp, seed, counter, nrm[0], nrm[1]);
        const int64_t ein = i * N + jp, e0 = ein - kr.row0 * N;   // of the inputs, of the outputs
        df32 dv[2];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          df32 pert;
          if (in[2 * h + b]) {
            if (emode == 1) pert = df_from_double(E[ein + b]);
            else if (emode == 2) pert = sr * df32(nrm[b], 0.f);
          }
          dv[b] = (yd - z[2 * h + b]) + pert;
        }
        const df32* ha = hv + 2 * h;
        if (even) {
          // both members present and e0 even: one 8- or 16-byte store per array per lane
          if (D) *reinterpret_cast<double2*>(D + e0) = make_double2(df_to_double(dv[0]), df_to_double(dv[1]));
          if (HA32) *reinterpret_cast<float2*>(HA32 + e0) = make_float2(ha[0].hi, ha[1].hi);
          if (B32) *reinterpret_cast<float2*>(B32 + e0) = make_float2(dv[0].hi, dv[1].hi);
          if (HAdf) *reinterpret_cast<float4*>(HAdf + e0) = make_float4(ha[0].hi, ha[0].lo, ha[1].hi, ha[1].lo);
          if (Ddf) *reinterpret_cast<float4*>(Ddf + e0) = make_float4(dv[0].hi, dv[0].lo, dv[1].hi, dv[1].lo);
        } else {
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            if (!in[2 * h + b]) continue;
            const int64_t e = e0 + b;
            if (D) D[e] = df_to_double(dv[b]);
            if (HA32) HA32[e] = ha[b].hi;
            if (B32) B32[e] = dv[b].hi;
            if (HAdf) HAdf[e] = ha[b];
            if (Ddf) Ddf[e] = dv[b];
          }
        }
      }
    }
  }
  if (kr.umax && gl == 0 && umax > 0.f) atomicMax(kr.umax, __float_as_uint(umax));
  if (hamax) {
    // non-negative floats order as their bit patterns
    const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(hmax));
    if (lane == 0 && mb > 0u) atomicMax(hamax, mb);
  }
}

}  // namespace enkf
