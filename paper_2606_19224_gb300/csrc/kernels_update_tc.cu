// The ensemble update X_a = X_f + A W (Fig. 2, Algorithm 1: A = X_f - xbar 1^T, W = HA^T Z/(N-1))
// on the 5th-generation tensor cores, for FP32 ensembles.
//
// Per 128-row tile of X_f: the rows are staged in shared memory (the next tile's are in flight in
// registers meanwhile; two CTAs per SM for N <= 64, so that one converts while the other's stores drain),
// each row's mean and largest anomaly are formed, and the anomalies scaled by an exact power of two per
// row (so FP16 neither overflows nor flushes) are split into hi + lo FP16 parts in the canonical K-major core-matrix layout,
// the lo part stored times 2^11 so that it stays in FP16's normal range. W is staged once per
// CTA the same way (rows j, K-major over k, a power-of-two scale per column). D = A W runs as
// three M = 128 x N = NT x K = NT MMAs per K block with FP32 accumulation in TMEM: hi*hi into
// one accumulator, hi*lo' + lo'*hi into a second, so D = D1 + 2^-11 D2 carries about 22
// significant bits per product; the epilogue reads both row by row, undoes the scales, forms
// X_a = X_f + D in place of the staged tile and then writes the tile out with coalesced
// 16-byte stores (a row per thread would scatter every store over 32 rows). X_a may be
// X_f itself: a tile is read into shared memory before any of its rows is written, and no CTA
// reads another CTA's tiles.
#include <algorithm>
#include <cmath>

#include "tc_mixed.cuh"

namespace enkf {

constexpr int kUT = 512;   // threads: four per row of a tile (with two per row and 256 threads the conversion of a
                          // tile took three times as long as its bytes: 65 us at n = 262,144, N = 64 and 471 us at
                          // n = 1,048,576, N = 128)

template <int NT> struct UpdLayout {
  static constexpr int LDX = NT + 4;                       // staged X_f row stride (floats)
  static constexpr int XT = kTR * LDX * 4;                 // bytes per staged tile
  static constexpr int AIMG = 2 * kTR * NT * 2;            // A image: hi and lo parts
  static constexpr int BIMG = 2 * NT * NT * 2;             // W image: hi and lo parts
  static constexpr int off_x = 0;
  static constexpr int off_a = ((XT + 1023) / 1024) * 1024;
  static constexpr int off_b = off_a + AIMG;
  static constexpr int off_rs = off_b + BIMG;              // per-row 2^-e scale [128]
  static constexpr int off_ws = off_rs + 4 * kTR;          // per-column 1/scale of W [NT]
  static constexpr int bytes = off_ws + 4 * NT;
  static_assert(off_a % 1024 == 0 && off_b % 1024 == 0, "operand alignment");
};
template <int NT> __host__ __device__ constexpr int update_tc_smem_bytes() { return UpdLayout<NT>::bytes; }

// 2^-e with 2^e >= max|v| > 2^(e-1) (1 for v = 0): scales v into (1/2, 1] exactly
__device__ __forceinline__ float pow2_scale(float vmax) {
  if (!(vmax > 0.f) || !isfinite(vmax)) return 1.f;
  int e;
  frexpf(vmax, &e);
  return ldexpf(1.f, -e);
}

template <int NT>
__global__ void __launch_bounds__(kUT, NT <= 64 ? 2 : 1) update_tc_kernel(
    const float* Xf, float* Xa, const double* __restrict__ W, int64_t n, int N, int* status) {
  using L = UpdLayout<NT>;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_base;
  constexpr int TMC = 2 * NT;   // D1 (hi*hi) at column 0, D2 (the cross terms) at column NT
  constexpr uint32_t idesc = umma_idesc(H16<__half>::fmt, NT);
  constexpr uint32_t sbo = (NT / 8) * 128;
  constexpr int C4 = NT / 4;
  constexpr int EP = NT < 64 ? 2 : 4, CH = NT / EP / 16;   // epilogue: column parts, 16-column chunks of each
  constexpr int PRE = kTR * C4 / kUT;                      // 16-byte pieces of a tile per thread
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, qd = warp & 3, part = warp >> 2;
  float* sX = reinterpret_cast<float*>(smem + L::off_x);
  __half* sA = reinterpret_cast<__half*>(smem + L::off_a);
  __half* sB = reinterpret_cast<__half*>(smem + L::off_b);
  float* s_rs = reinterpret_cast<float*>(smem + L::off_rs);
  float* s_ws = reinterpret_cast<float*>(smem + L::off_ws);
  if (dynamic_smem_bytes() < (unsigned)L::bytes) {
    if (t == 0) atomicOr(status, DS_SMEM);
    return;
  }
  if (t == 0) mbar_init(&mbar);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base)), "r"(TMC));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  // W: per-column power-of-two scale, then the hi/lo image (rows j, K-major over k)
  {
    constexpr int WP = kUT / NT, WK = NT / WP;   // threads per column, entries of each
    const int j = t % NT, w = t / NT;
    float v[WK], mx = 0.f;
#pragma unroll
    for (int q = 0; q < WK; ++q) {
      const int k = w + q * WP;
      v[q] = (j < N && k < N) ? (float)__ldcg(W + k * N + j) : 0.f;
      mx = fmaxf(mx, fabsf(v[q]));
    }
    sX[w * NT + j] = mx;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < WP; ++q) mx = fmaxf(mx, sX[q * NT + j]);
    const float sc = pow2_scale(mx);
    if (w == 0) s_ws[j] = 1.f / sc;                       // exact (a power of two)
#pragma unroll
    for (int q = 0; q < WK; ++q) {
      const float x = v[q] * sc;
      const __half hi = __float2half_rn(x);
      sB[core_idx(j, w + q * WP, NT)] = hi;
      sB[NT * NT + core_idx(j, w + q * WP, NT)] = __float2half_rn((x - __half2float(hi)) * 2048.f);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const bool vec = rows_vec(Xf, Xa, N);
  const int64_t ntiles = (n + kTR - 1) / kTR;
  uint32_t ph = 0;
  bool ok = true;
  // the next tile waits in registers
  float4 pre[PRE];
  auto fetch = [&](int64_t tile) {
#pragma unroll
    for (int q = 0; q < PRE; ++q) {
      const int c = t + q * kUT, r = c / C4, c0 = (c % C4) * 4;
      const int64_t i = tile * kTR + r;
      float a[4] = {0.f, 0.f, 0.f, 0.f};
      if (i < n && c0 < N) ld4<float>(a, Xf + i * N, c0, N, vec);
      pre[q] = make_float4(a[0], a[1], a[2], a[3]);
    }
  };
  if (blockIdx.x < ntiles) fetch(blockIdx.x);
  for (int64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
#pragma unroll
    for (int q = 0; q < PRE; ++q) {
      const int c = t + q * kUT;
      *reinterpret_cast<float4*>(sX + c / C4 * L::LDX + (c % C4) * 4) = pre[q];
    }
    if (tile + gridDim.x < ntiles) fetch(tile + gridDim.x);
    __syncthreads();
    // row means and the largest anomaly of each row: four threads per row, each with every fourth group of
    // eight members in registers
    {
      constexpr int KC = NT / 32;
      const int r = t >> 2, hf = t & 3;
      float x[KC][8], sum = 0.f;
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        const float* src = sX + r * L::LDX + (4 * c + hf) * 8;
        const float4 a = *reinterpret_cast<const float4*>(src), b = *reinterpret_cast<const float4*>(src + 4);
        x[c][0] = a.x; x[c][1] = a.y; x[c][2] = a.z; x[c][3] = a.w;
        x[c][4] = b.x; x[c][5] = b.y; x[c][6] = b.z; x[c][7] = b.w;
        sum += ((a.x + a.y) + (a.z + a.w)) + ((b.x + b.y) + (b.z + b.w));   // (zeros past N)
      }
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      const float mean = sum / (float)N;
      float mx = 0.f;
#pragma unroll
      for (int c = 0; c < KC; ++c)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          x[c][e] = (4 * c + hf) * 8 + e < N ? x[c][e] - mean : 0.f;
          mx = fmaxf(mx, fabsf(x[c][e]));
        }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float sc = pow2_scale(mx);
      if (hf == 0) s_rs[r] = sc;
      // the scaled anomalies as hi + lo FP16, one 16-byte core row at a time
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        __align__(16) __half hv[8], lv[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float a = x[c][e] * sc;
          hv[e] = __float2half_rn(a);
          lv[e] = __float2half_rn((a - __half2float(hv[e])) * 2048.f);
        }
        const int kc = (4 * c + hf) * 8;
        *reinterpret_cast<uint4*>(sA + core_idx(r, kc, NT)) = *reinterpret_cast<const uint4*>(hv);
        *reinterpret_cast<uint4*>(sA + kTR * NT + core_idx(r, kc, NT)) = *reinterpret_cast<const uint4*>(lv);
      }
    }
    fence_async_smem();
    __syncthreads();
    if (t == 0) {
      tc_fence_after();
      const uint32_t au = smem_addr(sA), bu = smem_addr(sB);
#pragma unroll
      for (int kb = 0; kb < NT / 16; ++kb) {
        umma_f16(tmem, umma_desc(au + kb * 256, 128, sbo), umma_desc(bu + kb * 256, 128, sbo), idesc, kb > 0 ? 1u : 0u);
        umma_f16(tmem + NT, umma_desc(au + kb * 256, 128, sbo), umma_desc(bu + 2 * NT * NT + kb * 256, 128, sbo), idesc,
                 kb > 0 ? 1u : 0u);
        umma_f16(tmem + NT, umma_desc(au + 2 * kTR * NT + kb * 256, 128, sbo), umma_desc(bu + kb * 256, 128, sbo), idesc, 1u);
      }
      umma_commit(&mbar);
    }
    if (!mbar_wait(&mbar, ph, status)) ok = false;
    ph ^= 1u;
    tc_fence_after();
    // X_a = X_f + D / (row scale * column scale), one row per thread (TMEM lane = row)
    const int rt = 32 * qd + lane;
    const int64_t i = tile * kTR + rt;
    const float irs = 1.f / s_rs[rt];
    if (part < EP)
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const int j0 = (part * CH + c) * 16;
      float d[16], d2[16];
      tmem_ld16(tmem + ((uint32_t)(32 * qd) << 16) + j0, d);
      tmem_ld16(tmem + ((uint32_t)(32 * qd) << 16) + NT + j0, d2);
#pragma unroll
      for (int y = 0; y < 16; ++y) d[y] = fmaf(d2[y], 0x1p-11f, d[y]);
      if (i < n) {
#pragma unroll
        for (int y4 = 0; y4 < 4; ++y4) {
          const int jj = j0 + 4 * y4;
          if (jj < N) {
            float* xr = sX + rt * L::LDX + jj;
            const float4 xf = *reinterpret_cast<const float4*>(xr);
            *reinterpret_cast<float4*>(xr) = make_float4(fmaf(d[4 * y4] * irs, s_ws[jj], xf.x),
                                                         fmaf(d[4 * y4 + 1] * irs, s_ws[jj + 1], xf.y),
                                                         fmaf(d[4 * y4 + 2] * irs, s_ws[jj + 2], xf.z),
                                                         fmaf(d[4 * y4 + 3] * irs, s_ws[jj + 3], xf.w));
          }
        }
      }
    }
    tc_fence_before();
    __syncthreads();
    // the finished tile out: consecutive threads on consecutive 16-byte pieces of a row
    for (int c = t; c < kTR * C4; c += kUT) {
      const int r = c / C4, c0 = (c % C4) * 4;
      const int64_t ig = tile * kTR + r;
      if (ig < n && c0 < N) {
        const float4 v = *reinterpret_cast<const float4*>(sX + r * L::LDX + c0);
        const float o[4] = {v.x, v.y, v.z, v.w};
        st4<float>(Xa + ig * N, c0, N, vec, o);
      }
    }
    __syncthreads();   // the staged tile, the A image and TMEM are rewritten by the next tile
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMC));
}

template <int NT>
static cudaError_t launch_one(const float* Xf, float* Xa, const double* W, int64_t n, int N, int* status,
                              int sms, cudaStream_t s) {
  constexpr int smem = update_tc_smem_bytes<NT>();
  cudaError_t e = cudaFuncSetAttribute(update_tc_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (n + kTR - 1) / kTR;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)sms * (NT <= 64 ? 2 : 1)));
  update_tc_kernel<NT><<<grid, kUT, smem, s>>>(Xf, Xa, W, n, N, status);
  return cudaGetLastError();
}

// X_a = X_f + (X_f - xbar 1^T) W for FP32 ensembles on the tensor cores.
cudaError_t launch_update_tc(enkf_handle_s* h, const void* Xf, void* Xa) {
  const auto& c = h->cfg;
  const float* x = static_cast<const float*>(Xf);
  float* xa = static_cast<float*>(Xa);
  const int NT = c.N <= 32 ? 32 : (c.N <= 64 ? 64 : 128);
  if (NT == 32) return launch_one<32>(x, xa, h->ws.W, c.n, c.N, h->ws.status, h->sms, h->stream);
  if (NT == 64) return launch_one<64>(x, xa, h->ws.W, c.n, c.N, h->ws.status, h->sms, h->stream);
  return launch_one<128>(x, xa, h->ws.W, c.n, c.N, h->ws.status, h->sms, h->stream);
}

}  // namespace enkf
