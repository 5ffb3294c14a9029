// Learned CG warm start: the MLP's forward, backward and Adam kernels, and the three
// warm-start maps of an analysis (features, prediction, decoder).
//
// The paper's CG starts from zero (Sec. 3.3). Every solution column of S Z = D satisfies
// R z_j = d_j - HA c_j with c_j = W e_j, W = HA^T Z/(N-1) (rearranging S Z = D with
// Eq. matvec_decomp), so the model predicts the N-vector c_j and the decoder forms
// z0_j = R^{-1}(d_j - HA c_j), whose residual lies in span(HA).
//
// Model (per column j): features f_j = [d_j(sketch)/s_j, g_j/s_j] with a sketch of K rows
// i_k = floor(k m / K), s_j the RMS of d_j over the sketch (1 if 0), g_j = HA^T R^-1 d_j/(N-1);
// standardised per feature; L hidden layers of width H with GELU (x Phi(x), Hendrycks &
// Gimpel 2016); linear output = standardised c_j/s_j. Loss: mean squared error in
// standardised units; optimiser: Adam (Kingma & Ba 2015, Algorithm 1).
//
// Parameter layout (FP32): per layer W [out][in] then b [out]; then mu_in [in], sd_in [in],
// mu_out [out], sd_out [out].
//
// The dense layers are FP32 tiles on the CUDA cores, split along K over thread-block clusters
// (mlp_gemm_kernel).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "solve_body.cuh"

namespace enkf {

struct MlpLayout {
  int in, hidden, layers, out;
  int64_t w_off[8], b_off[8];   // per layer (layers + 1 <= 8)
  int64_t mu_in, sd_in, mu_out, sd_out, total, trained;
};

static bool mlp_layout(const enkf_mlp_shape* s, MlpLayout& L) {
  if (!s || s->in_dim < 1 || s->hidden < 1 || s->layers < 1 || s->layers > 7 || s->out_dim < 1) return false;
  L.in = s->in_dim;
  L.hidden = s->hidden;
  L.layers = s->layers;
  L.out = s->out_dim;
  int64_t off = 0;
  for (int l = 0; l <= L.layers; ++l) {
    const int64_t fi = l == 0 ? L.in : L.hidden, fo = l == L.layers ? L.out : L.hidden;
    L.w_off[l] = off;
    off += fi * fo;
    L.b_off[l] = off;
    off += fo;
  }
  L.trained = off;
  L.mu_in = off;
  off += L.in;
  L.sd_in = off;
  off += L.in;
  L.mu_out = off;
  off += L.out;
  L.sd_out = off;
  off += L.out;
  L.total = off;
  return true;
}

__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// ------------------------------------------------------------------ tiled FP32 GEMM
// C[M][N] = sum_k A(m, k) B(k, n) with A(m, k) = A[m * sam + k * sak] and
// B(k, n) = B[k * sbk + n * sbn], and a fused epilogue. One of sam, sak and one of sbk, sbn is 1.
// 64 x 64 outputs per CTA of 256 threads, 4 x 4 per thread, operands staged 32 deep as [row][k] and read
// four k at a time (12 shared-memory wavefronts against 16 FMA cycles per warp and four k); K is split over
// a cluster of up to 8 CTAs, whose partial tiles are added in rank order through distributed shared memory:
// the network's products have 8 to 136 tiles, which alone leave most SMs idle. Loads run along the
// contiguous index of each operand. (32 x 32 tiles with 2 x 2 outputs per thread and loads along the
// strided index took 15 to 30 us per product at batch 256, 1088 -> 512^3 -> 64; loss and gradient 345 us, now
// 158.)
constexpr int GT = 64, GBK = 32, GLD = GBK + 4;

enum : int { EPI_HIDDEN = 0, EPI_OUT = 1, EPI_BWD = 2, EPI_STORE = 3 };

struct GemmArgs {
  const float* A;
  int64_t sam, sak;
  const float* B;
  int64_t sbk, sbn;
  int M, N, K;
  const float* bias;     // EPI_HIDDEN / EPI_OUT
  const float* zprev;    // EPI_BWD: pre-activations whose GELU' scales the product
  float* C;              // main output [M][N]
  float* C2;             // EPI_HIDDEN: GELU(C); EPI_OUT: raw output mu_out + sd_out * C
  const float* mu_out;
  const float* sd_out;
  float* rowsum;         // EPI_STORE: sum_k A(m, k) (the bias gradient) or nullptr
  int split;             // CTAs per cluster along K
};

// rows [r0, r0 + 64) and k in [k0, k0 + 32) of an operand X(r, k) = X[r sr + k sk] as [row][k]
struct GemmTile {
  float v[8];
  __device__ __forceinline__ void fetch(const float* X, int64_t sr, int64_t sk, int r0, int rows, int k0, int k1) {
    const int t = threadIdx.x;
    if (sk == 1) {   // along k: eight threads per row, four k each, rows t / 8 and t / 8 + 32
      const bool vec = (sr & 3) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = r0 + t / 8 + 32 * h, k = k0 + (t % 8) * 4;
        const float* src = X + (int64_t)r * sr + k;
        if (vec && r < rows && k + 4 <= k1) {
          const float4 q = *reinterpret_cast<const float4*>(src);
          v[4 * h] = q.x; v[4 * h + 1] = q.y; v[4 * h + 2] = q.z; v[4 * h + 3] = q.w;
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) v[4 * h + e] = (r < rows && k + e < k1) ? src[e] : 0.f;
        }
      }
    } else {         // along the rows: 64 consecutive threads per k, k t / 64 + 4 e
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int r = r0 + t % 64, k = k0 + t / 64 + 4 * e;
        v[e] = (r < rows && k < k1) ? X[(int64_t)r * sr + (int64_t)k * sk] : 0.f;
      }
    }
  }
  __device__ __forceinline__ void put(float* s, int64_t sk) const {
    const int t = threadIdx.x;
    if (sk == 1) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
        *reinterpret_cast<float4*>(s + (t / 8 + 32 * h) * GLD + (t % 8) * 4) =
            make_float4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) s[(t % 64) * GLD + t / 64 + 4 * e] = v[e];
    }
  }
};

template <int EPI>
__global__ void __launch_bounds__(256) mlp_gemm_kernel(const GemmArgs g) {
  __shared__ __align__(16) float As[2][GT * GLD];
  __shared__ __align__(16) float Bs[2][GT * GLD];
  // this CTA's partial, column 64 the row sums of A: over the operands once they are used up
  static_assert(sizeof(float) * GT * (GT + 1) <= sizeof(As), "the partial tile lies over As");
  float (*tile)[GT + 1] = reinterpret_cast<float(*)[GT + 1]>(&As[0][0]);
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int S = g.split, rank = S > 1 ? (int)cluster.block_rank() : 0;
  const int t = threadIdx.x, tx = t % 16, ty = t / 16;
  const int m0 = blockIdx.y * GT, n0 = (blockIdx.x / S) * GT;
  const int steps = (g.K + GBK - 1) / GBK, per = (steps + S - 1) / S;
  const int kb = min(g.K, rank * per * GBK), ke = min(g.K, kb + per * GBK);
  float acc[4][4] = {}, rs[4] = {};
  const bool rows = EPI == EPI_STORE && g.rowsum != nullptr && n0 == 0 && tx == 0;
  GemmTile ta, tb;
  if (kb < ke) {
    ta.fetch(g.A, g.sam, g.sak, m0, g.M, kb, ke);
    tb.fetch(g.B, g.sbn, g.sbk, n0, g.N, kb, ke);
  }
  int buf = 0;
  for (int k0 = kb; k0 < ke; k0 += GBK, buf ^= 1) {
    ta.put(As[buf], g.sak);
    tb.put(Bs[buf], g.sbk);
    __syncthreads();   // (the other buffer's readers passed the barrier of the step before)
    if (k0 + GBK < ke) {
      ta.fetch(g.A, g.sam, g.sak, m0, g.M, k0 + GBK, ke);
      tb.fetch(g.B, g.sbn, g.sbk, n0, g.N, k0 + GBK, ke);
    }
    // thread (ty, tx): rows ty + 16 x of A, columns tx + 16 y of B
#pragma unroll
    for (int kk = 0; kk < GBK; kk += 4) {
      float4 a[4], b[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) a[x] = *reinterpret_cast<const float4*>(&As[buf][(ty + 16 * x) * GLD + kk]);
#pragma unroll
      for (int y = 0; y < 4; ++y) b[y] = *reinterpret_cast<const float4*>(&Bs[buf][(tx + 16 * y) * GLD + kk]);
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          acc[x][y] = fmaf(a[x].x, b[y].x, acc[x][y]);
          acc[x][y] = fmaf(a[x].y, b[y].y, acc[x][y]);
          acc[x][y] = fmaf(a[x].z, b[y].z, acc[x][y]);
          acc[x][y] = fmaf(a[x].w, b[y].w, acc[x][y]);
        }
      if (rows)
#pragma unroll
        for (int x = 0; x < 4; ++x) rs[x] += (a[x].x + a[x].y) + (a[x].z + a[x].w);
    }
  }
  __syncthreads();
#pragma unroll
  for (int x = 0; x < 4; ++x) {
#pragma unroll
    for (int y = 0; y < 4; ++y) tile[ty + 16 * x][tx + 16 * y] = acc[x][y];
    if (tx == 0) tile[ty + 16 * x][GT] = rs[x];
  }
  if (S > 1) cluster.sync();
  else __syncthreads();
  // rank r finishes the rows [r 64/S, ...) of the tile
  const int nrow = GT / S;
  for (int e = t; e < nrow * GT; e += 256) {
    const int r = rank * nrow + e / GT, c = e % GT, m = m0 + r, n = n0 + c;
    float v = 0.f;
    for (int q = 0; q < S; ++q) v += S > 1 ? *cluster.map_shared_rank(&tile[r][c], q) : tile[r][c];
    if (m >= g.M || n >= g.N) continue;
    const int64_t o = (int64_t)m * g.N + n;
    if (EPI == EPI_HIDDEN) {
      v += g.bias[n];
      g.C[o] = v;
      g.C2[o] = gelu_f(v);
    } else if (EPI == EPI_OUT) {
      v += g.bias[n];
      g.C[o] = v;
      if (g.C2) g.C2[o] = g.mu_out[n] + g.sd_out[n] * v;
    } else if (EPI == EPI_BWD) {
      g.C[o] = v * gelu_grad_f(g.zprev[o]);
    } else {
      g.C[o] = v;
    }
  }
  if (EPI == EPI_STORE && g.rowsum != nullptr && n0 == 0 && t < nrow) {
    const int r = rank * nrow + t;
    float v = 0.f;
    for (int q = 0; q < S; ++q) v += S > 1 ? *cluster.map_shared_rank(&tile[r][GT], q) : tile[r][GT];
    if (m0 + r < g.M) g.rowsum[m0 + r] = v;
  }
  if (S > 1) cluster.sync();   // the tiles stay until every rank has read them
}

template <int EPI>
static cudaError_t gemm(GemmArgs a, cudaStream_t s) {
  const int tn = (a.N + GT - 1) / GT, tm = (a.M + GT - 1) / GT, steps = (a.K + GBK - 1) / GBK;
  // up to two CTAs per SM, and a step along K per CTA at least
  a.split = 1;
  while (a.split < 8 && (int64_t)tn * tm * a.split * 2 <= 304 && steps >= 2 * a.split) a.split *= 2;
  if (a.split == 1) {
    mlp_gemm_kernel<EPI><<<dim3(tn, tm), 256, 0, s>>>(a);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(tn * a.split, tm);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = a.split;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  void* args[] = {&a};
  return cudaLaunchKernelExC(&cfg, (const void*)mlp_gemm_kernel<EPI>, args);
}

// Loss and output gradient: diff = y_std - (t - mu_out)/sd_out over B x out entries (rows of
// T optionally gathered); G = 2 diff/(B out); loss = sum diff^2/(B out). One cluster of 8 CTAs, fixed
// order (a single CTA took 30 us for a batch of 256, 8 x 256 threads 15: the entries' loads are latency).
constexpr int kMT = 1024;
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(kMT) mse_kernel(const float* __restrict__ Y, const float* __restrict__ T,
                                                  const int32_t* __restrict__ rows, int B, int out,
                                                  const float* __restrict__ mu_out,
                                                  const float* __restrict__ sd_out, float* __restrict__ G,
                                                  float* __restrict__ loss) {
  __shared__ double red[kMT / 32], part;
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int t = threadIdx.x;
  const double inv = 1.0 / ((double)B * out);
  const float g2 = (float)(2.0 * inv);
  double s = 0.0;
  const int64_t total = (int64_t)B * out;
  const bool small = total < (1ll << 31);   // 32-bit divisions
  for (int64_t e = (int64_t)blockIdx.x * kMT + t; e < total; e += 8 * kMT) {
    const int b = small ? (int)e / out : (int)(e / out), o = (int)(e - (int64_t)b * out);
    const int64_t row = rows ? (int64_t)rows[b] : (int64_t)b;
    const float tt = (T[row * out + o] - mu_out[o]) / sd_out[o];
    const float d = Y[e] - tt;
    G[e] = g2 * d;
    s += (double)d * d;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((t & 31) == 0) red[t / 32] = s;
  __syncthreads();
  if (t == 0) {
    double v = 0.0;
    for (int w = 0; w < kMT / 32; ++w) v += red[w];
    part = v;
  }
  cluster.sync();
  if (blockIdx.x == 0 && t == 0 && loss) {
    double v = 0.0;
    for (int q = 0; q < 8; ++q) v += *cluster.map_shared_rank(&part, q);
    *loss = (float)(v * inv);
  }
  cluster.sync();
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int64_t count, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// Per-column mean and standard deviation over `rows` rows (population form; 1 where 0).
__global__ void colstats_kernel(const float* __restrict__ X, int64_t rows, int cols, float* __restrict__ mu,
                                float* __restrict__ sd) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  double s = 0.0;
  for (int64_t r = 0; r < rows; ++r) s += X[r * cols + c];
  const double mean = s / (double)rows;
  double q = 0.0;
  for (int64_t r = 0; r < rows; ++r) {
    const double d = X[r * cols + c] - mean;
    q += d * d;
  }
  const double sdv = sqrt(q / (double)rows);
  mu[c] = (float)mean;
  sd[c] = sdv > 0.0 ? (float)sdv : 1.f;
}

// Gather rows of X [*][in] through `rows` (identity if NULL) and standardise per feature.
__global__ void standardize_rows_kernel(const float* __restrict__ X, const int32_t* __restrict__ rows, int B,
                                        int in, const float* __restrict__ mu, const float* __restrict__ sd,
                                        float* __restrict__ Xs) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)B * in;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int b = (int)(e / in), k = (int)(e % in);
    const int64_t row = rows ? (int64_t)rows[b] : (int64_t)b;
    Xs[e] = (X[row * in + k] - mu[k]) / sd[k];
  }
}

// ------------------------------------------------------------------ MLP, host side
struct MlpWork {
  float* Xs;     // standardised (gathered) input [B][in]
  float* Z[8];   // pre-activations per hidden layer [B][H]
  float* A[8];   // activations per hidden layer [B][H]
  float* Y;      // standardised output [B][out]
  float* G0;     // gradient buffers [B][max(H, out)]
  float* G1;
};

static size_t mlp_work_floats(const MlpLayout& L, int B) {
  const size_t w = (size_t)std::max(L.hidden, L.out);
  return (size_t)B * L.in + (size_t)2 * L.layers * B * L.hidden + (size_t)B * L.out + 2 * (size_t)B * w;
}

static MlpWork carve(const MlpLayout& L, int B, float* base) {
  MlpWork W{};
  float* q = base;
  W.Xs = q; q += (size_t)B * L.in;
  for (int l = 0; l < L.layers; ++l) {
    W.Z[l] = q; q += (size_t)B * L.hidden;
    W.A[l] = q; q += (size_t)B * L.hidden;
  }
  W.Y = q; q += (size_t)B * L.out;
  const size_t w = (size_t)std::max(L.hidden, L.out);
  W.G0 = q; q += (size_t)B * w;
  W.G1 = q;
  return W;
}

static int ew_grid(int64_t count) { return (int)std::min<int64_t>(4096, std::max<int64_t>(1, (count + 255) / 256)); }

static cudaError_t mlp_forward_impl(const MlpLayout& L, const float* P, const float* X, const int32_t* rows,
                                    int B, const MlpWork& W, float* Yraw, cudaStream_t s) {
  standardize_rows_kernel<<<ew_grid((int64_t)B * L.in), 256, 0, s>>>(X, rows, B, L.in, P + L.mu_in, P + L.sd_in, W.Xs);
  cudaError_t e = cudaGetLastError();
  for (int l = 0; l <= L.layers && e == cudaSuccess; ++l) {
    const int fi = l == 0 ? L.in : L.hidden, fo = l == L.layers ? L.out : L.hidden;
    GemmArgs a{};
    a.A = l == 0 ? W.Xs : W.A[l - 1];
    a.sam = fi;
    a.sak = 1;
    a.B = P + L.w_off[l];   // B(k, n) = W_l[n][k]
    a.sbk = 1;
    a.sbn = fi;
    a.M = B;
    a.N = fo;
    a.K = fi;
    a.bias = P + L.b_off[l];
    if (l < L.layers) {
      a.C = W.Z[l];
      a.C2 = W.A[l];
      e = gemm<EPI_HIDDEN>(a, s);
    } else {
      a.C = W.Y;
      a.C2 = Yraw;
      a.mu_out = P + L.mu_out;
      a.sd_out = P + L.sd_out;
      e = gemm<EPI_OUT>(a, s);
    }
  }
  return e;
}

static cudaError_t mlp_loss_grad_impl(const MlpLayout& L, const float* P, const float* X, const float* T,
                                      const int32_t* rows, int B, float* grad, float* loss, const MlpWork& W,
                                      cudaStream_t s) {
  cudaError_t e = mlp_forward_impl(L, P, X, rows, B, W, nullptr, s);
  if (e != cudaSuccess) return e;
  mse_kernel<<<8, kMT, 0, s>>>(W.Y, T, rows, B, L.out, P + L.mu_out, P + L.sd_out, W.G0, loss);
  e = cudaGetLastError();
  float* g = W.G0;    // dL/dz of layer l, [B][fo]
  float* gn = W.G1;
  for (int l = L.layers; l >= 0 && e == cudaSuccess; --l) {
    const int fi = l == 0 ? L.in : L.hidden, fo = l == L.layers ? L.out : L.hidden;
    // dW_l[o][i] = sum_b g[b][o] a_{l-1}[b][i]
    GemmArgs a{};
    a.A = g;
    a.sam = 1;
    a.sak = fo;
    a.B = l == 0 ? W.Xs : W.A[l - 1];
    a.sbk = fi;
    a.sbn = 1;
    a.M = fo;
    a.N = fi;
    a.K = B;
    a.C = grad + L.w_off[l];
    a.rowsum = grad + L.b_off[l];   // db_l[o] = sum_b g[b][o]
    e = gemm<EPI_STORE>(a, s);
    if (l > 0 && e == cudaSuccess) {
      // g_{l-1}[b][i] = (sum_o g[b][o] W_l[o][i]) GELU'(z_{l-1}[b][i])
      GemmArgs d{};
      d.A = g;
      d.sam = fo;
      d.sak = 1;
      d.B = P + L.w_off[l];
      d.sbk = fi;
      d.sbn = 1;
      d.M = B;
      d.N = fi;
      d.K = fo;
      d.zprev = W.Z[l - 1];
      d.C = gn;
      e = gemm<EPI_BWD>(d, s);
      std::swap(g, gn);
    }
  }
  return e;
}

// ------------------------------------------------------------------ warm-start maps
// Partial N x N products over row blocks: part[b][0][k][j] = sum_{i in block b} HA[i][k] D[i][j] / r_i
// and part[b][1][k][j] = sum_{i in block b} HA[i][k] HA[i][j] / r_i (FP32 products of the FP32
// copies, FP32 within a block); the reduce kernel sums the blocks in a fixed order in FP64.
// AM x AM outputs of each product per thread (AM = NT / 16).
constexpr int kWarmRows = 32;

template <int AM>
__global__ void __launch_bounds__(kThreads) warm_gram_kernel(const df32* __restrict__ HA,
                                                             const df32* __restrict__ D,
                                                             const float* __restrict__ r32, int64_t m, int N,
                                                             int64_t rows_per, double* __restrict__ part) {
  constexpr int NT = 16 * AM, LD = NT + 4, RW = AM == 8 ? kWarmRows / 2 : kWarmRows;   // static smem < 48 KB
  __shared__ __align__(16) float sH[RW][LD];
  __shared__ __align__(16) float sD[RW][LD];
  __shared__ __align__(16) float sHr[RW][LD];
  __shared__ float sRi[RW];
  const int t = threadIdx.x;
  const int64_t i0 = (int64_t)blockIdx.x * rows_per, i1 = imin64(m, i0 + rows_per);
  // thread (tk, tj) owns the AM x AM block k in [AM tk, AM tk + AM), j in [AM tj, AM tj + AM)
  const int tk = t / 16, tj = t % 16, k0 = AM * tk, c0 = AM * tj;
  float acc[AM][AM] = {}, accG[AM][AM] = {};
  for (int64_t ib = i0; ib < i1; ib += RW) {
    __syncthreads();
    if (t < RW) {
      const int64_t i = ib + t;
      sRi[t] = i < i1 ? 1.f / r32[i] : 0.f;
    }
    __syncthreads();
    for (int e = t; e < RW * NT; e += kThreads) {
      const int ii = e / NT, k = e % NT;
      const int64_t i = ib + ii;
      const bool in = i < i1 && k < N;
      const float rinv = sRi[ii];
      const float h = in ? HA[i * N + k].hi : 0.f;
      sH[ii][k] = h;
      sHr[ii][k] = h * rinv;
      sD[ii][k] = in ? D[i * N + k].hi * rinv : 0.f;
    }
    __syncthreads();
#pragma unroll 4
    for (int ii = 0; ii < RW; ++ii) {
      float h[AM], d[AM], hr[AM];
#pragma unroll
      for (int a = 0; a < AM; a += 2) {
        const float2 v = *reinterpret_cast<const float2*>(&sH[ii][k0 + a]);
        h[a] = v.x;
        h[a + 1] = v.y;
        const float2 w = *reinterpret_cast<const float2*>(&sD[ii][c0 + a]);
        d[a] = w.x;
        d[a + 1] = w.y;
        const float2 q = *reinterpret_cast<const float2*>(&sHr[ii][c0 + a]);
        hr[a] = q.x;
        hr[a + 1] = q.y;
      }
#pragma unroll
      for (int a = 0; a < AM; ++a)
#pragma unroll
        for (int c = 0; c < AM; ++c) {
          acc[a][c] = fmaf(h[a], d[c], acc[a][c]);
          accG[a][c] = fmaf(h[a], hr[c], accG[a][c]);
        }
    }
  }
  double* out = part + (int64_t)blockIdx.x * 2 * N * N;
#pragma unroll
  for (int a = 0; a < AM; ++a)
#pragma unroll
    for (int c = 0; c < AM; ++c) {
      const int k = k0 + a, j = c0 + c;
      if (k < N && j < N) {
        out[k * N + j] = acc[a][c];
        out[N * N + k * N + j] = accG[a][c];
      }
    }
}

// g[k][j] = sum over the row-block partials in block order (one thread per entry).
__global__ void warm_reduce_kernel(const double* __restrict__ part, int nparts, int NN, double* __restrict__ g) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= NN) return;
  double s = 0.0;
#pragma unroll 8
  for (int b = 0; b < nparts; ++b) s += part[(int64_t)b * NN + e];
  g[e] = s;
}

// The same sums from the products of a solve in Krylov coordinates: K = HA^T R^-1 HA/(N-1) and
// F^T = (HA^T R^-1 D)^T in double-float.
__global__ void warm_sums_kernel(const df32* __restrict__ K, const df32* __restrict__ F, int N, double* __restrict__ g) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N * N) return;
  const int k = e / N, j = e % N;
  g[e] = (double)F[(int64_t)j * N + k];
  g[N * N + e] = (double)K[e] * (double)(N - 1);
}

// Features of column j (one CTA per column): sketch values, their RMS s_j, and g_j/s_j.
__global__ void __launch_bounds__(kThreads) warm_features_kernel(const df32* __restrict__ D, int64_t m, int N,
                                                                 int K, const double* __restrict__ gsum,
                                                                 float* __restrict__ F,
                                                                 float* __restrict__ s_out) {
  __shared__ double red[kThreads];
  const int j = blockIdx.x, t = threadIdx.x;
  const double inv_nm1 = 1.0 / (double)(N - 1);
  double q = 0.0;
  for (int k = t; k < K; k += kThreads) {
    const int64_t i = ((int64_t)k * m) / K;
    const double v = (double)D[i * N + j];
    q += v * v;
  }
  red[t] = q;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (t < w) red[t] += red[t + w];
    __syncthreads();
  }
  const double rms = sqrt(red[0] / (double)K);
  const double sj = rms > 0.0 ? rms : 1.0;
  const int in = K + N;
  for (int k = t; k < K; k += kThreads) {
    const int64_t i = ((int64_t)k * m) / K;
    F[(int64_t)j * in + k] = (float)((double)D[i * N + j] / sj);
  }
  for (int k = t; k < N; k += kThreads) F[(int64_t)j * in + K + k] = (float)(gsum[k * N + j] * inv_nm1 / sj);
  if (t == 0) s_out[j] = (float)sj;
}

// Targets of the training pairs: T[j][k] = W[k][j] / s_j.
__global__ void warm_targets_kernel(const double* __restrict__ W, const float* __restrict__ s, int N,
                                    float* __restrict__ T) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N * N) return;
  const int j = e / N, k = e % N;
  T[e] = (float)(W[k * N + j] / (double)s[j]);
}

// Coefficients of column j (one CTA per column): c_j = Y[j] s_j (the prediction in raw units)
// and e_j = c_j + (Gw c_j - g~_j)/(N-1) with Gw = HA^T R^-1 HA, g~_j = HA^T R^-1 d_j, so that the
// start z0_j = R^-1 (d_j - HA c_j) has residual d_j - S z0_j = HA e_j (from S = HA HA^T/(N-1) + R).
__global__ void __launch_bounds__(128) warm_coef_kernel(const float* __restrict__ Y, const float* __restrict__ s,
                                                        const double* __restrict__ gsum, int N,
                                                        float* __restrict__ C, float* __restrict__ Ecoef) {
  __shared__ double sc[128];
  const int j = blockIdx.x, t = threadIdx.x;
  const double sj = s[j];
  for (int k = t; k < N; k += 128) sc[k] = (double)Y[j * N + k] * sj;
  __syncthreads();
  const double* g = gsum;                 // [k][j] = HA^T R^-1 D
  const double* Gw = gsum + N * N;        // [k][l] = HA^T R^-1 HA
  const double inv = 1.0 / (double)(N - 1);
  for (int k = t; k < N; k += 128) {
    double acc = 0.0;
    for (int l = 0; l < N; ++l) acc = fma(Gw[k * N + l], sc[l], acc);
    C[k * N + j] = (float)sc[k];
    Ecoef[k * N + j] = (float)(sc[k] + (acc - g[k * N + j]) * inv);
  }
}

// Decoder: z0[i][j] = (d_ij - sum_k HA[i][k] C[k][j]) / r_i as the double-float starting solution
// of the FP32 solve, and its residual B[i][j] = sum_k HA[i][k] E[k][j] as the first inner
// right-hand side (FP32; the refreshes recompute the true residual in double-float).
template <int RB>
__global__ void __launch_bounds__(kThreads) warm_decode_kernel(const df32* __restrict__ HA,
                                                               const df32* __restrict__ D,
                                                               const float* __restrict__ r32, int64_t m, int N,
                                                               const float* __restrict__ C,
                                                               const float* __restrict__ Ecoef,
                                                               df32* __restrict__ Z0, float* __restrict__ B) {
  extern __shared__ float wsm[];   // C [N][N + 1], E [N][N + 1], a 16-row tile of HA [16][N + 1]
  const int LD = N + 1;
  float* sC = wsm;
  float* sE = wsm + N * LD;
  float* sHt = wsm + 2 * N * LD;
  const int t = threadIdx.x;
  for (int e = t; e < N * N; e += kThreads) {
    const int k = e / N, j = e % N;
    sC[k * LD + j] = C[e];
    sE[k * LD + j] = Ecoef[e];
  }
  // thread (column j, group g of RB consecutive rows of the 16-row block): the C and E entries
  // of column j are loaded once per k for RB rows (RB = 2, 4, 8 for N <= 32, 64, 128)
  for (int64_t ib = (int64_t)blockIdx.x * 16; ib < m; ib += (int64_t)gridDim.x * 16) {
    __syncthreads();
    for (int e = t; e < 16 * N; e += kThreads) {
      const int ii = e / N, k = e % N;
      const int64_t i = ib + ii;
      sHt[ii * LD + k] = i < m ? HA[i * N + k].hi : 0.f;
    }
    __syncthreads();
    constexpr int NGR = 16 / RB;   // row groups covering the 16 rows
    for (int e = t; e < N * NGR; e += kThreads) {
      const int j = e % N, g = e / N;
      float a1[RB], a2[RB];
#pragma unroll
      for (int x = 0; x < RB; ++x) { a1[x] = 0.f; a2[x] = 0.f; }
#pragma unroll 4
      for (int k = 0; k < N; ++k) {
        const float c = sC[k * LD + j], ev = sE[k * LD + j];
#pragma unroll
        for (int x = 0; x < RB; ++x) {
          const float h = sHt[(g * RB + x) * LD + k];
          a1[x] = fmaf(h, c, a1[x]);
          a2[x] = fmaf(h, ev, a2[x]);
        }
      }
#pragma unroll
      for (int x = 0; x < RB; ++x) {
        const int64_t i = ib + g * RB + x;
        if (i < m) {
          const float z = (D[i * N + j].hi - a1[x]) / r32[i];
          Z0[i * N + j] = df32(z, 0.f);
          B[i * N + j] = a2[x];
        }
      }
    }
  }
}

// ||B_j||^2 of the start's residual B = HA E alone (a solve in Krylov coordinates starts from C
// itself): 16-row tiles as in the decoder, column sums in FP64 per CTA, then over the CTAs in order.
template <int RB>
__global__ void __launch_bounds__(kThreads) warm_resid_kernel(const df32* __restrict__ HA, int64_t m, int N,
                                                              const float* __restrict__ Ecoef,
                                                              double* __restrict__ part) {
  extern __shared__ float wsm[];   // E [N][N + 1], a 16-row tile of HA [16][N + 1], then column sums
  const int LD = N + 1;
  float* sE = wsm;
  float* sHt = wsm + N * LD;
  const int t = threadIdx.x;
  constexpr int NGR = 16 / RB;
  for (int e = t; e < N * N; e += kThreads) sE[(e / N) * LD + e % N] = Ecoef[e];
  double sum = 0.0;   // N NGR <= kThreads: one (column, row group) per thread
  for (int64_t ib = (int64_t)blockIdx.x * 16; ib < m; ib += (int64_t)gridDim.x * 16) {
    __syncthreads();
    for (int e = t; e < 16 * N; e += kThreads) {
      const int ii = e / N, k = e % N;
      sHt[ii * LD + k] = ib + ii < m ? HA[(ib + ii) * N + k].hi : 0.f;
    }
    __syncthreads();
    if (t < N * NGR) {
      const int j = t % N, g = t / N;
      float a[RB];
#pragma unroll
      for (int x = 0; x < RB; ++x) a[x] = 0.f;
#pragma unroll 4
      for (int k = 0; k < N; ++k) {
        const float ev = sE[k * LD + j];
#pragma unroll
        for (int x = 0; x < RB; ++x) a[x] = fmaf(sHt[(g * RB + x) * LD + k], ev, a[x]);
      }
      float q = 0.f;
#pragma unroll
      for (int x = 0; x < RB; ++x) q = fmaf(a[x], a[x], q);
      sum += (double)q;
    }
  }
  __syncthreads();
  double* red = reinterpret_cast<double*>(wsm);
  if (t < N * NGR) red[t] = sum;
  __syncthreads();
  if (t < N) {
    double s = 0.0;
    for (int g = 0; g < NGR; ++g) s += red[g * N + t];
    part[(int64_t)blockIdx.x * N + t] = s;
  }
}

}  // namespace enkf

// ------------------------------------------------------------------ host side
namespace enkf {

struct WarmState {
  MlpLayout L{};
  const float* params = nullptr;   // caller-owned model (enkf_set_warm_model)
  int K = 0;                       // sketch size of the model (in_dim - N)
  int nparts = 0;
  double* part = nullptr;          // [nparts][2][N][N]
  double* gsum = nullptr;          // [2][N][N]: HA^T R^-1 D, HA^T R^-1 HA
  float* C = nullptr;              // [N][N] predicted coefficients (column j = c_j)
  float* E = nullptr;              // [N][N] residual coefficients of the start
  float* F = nullptr;              // [N][K + N] features of the current analysis
  float* s = nullptr;              // [N] column scales
  float* Y = nullptr;              // [N][N] raw predictions
  float* work = nullptr;           // MLP activations for a batch of N rows
  double* rpart = nullptr;         // [2 SMs + 1][N] residual norms of the start per CTA, then their sum
  int K_alloc = 0;
};

static cudaError_t warm_alloc(enkf_handle_s* h, int K) {
  if (!h->warm) h->warm = new WarmState();
  WarmState& w = *h->warm;
  const int N = h->cfg.N;
  cudaError_t e = cudaSuccess;
  if (!w.part) {
    w.nparts = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)h->sms, (h->cfg.m + 255) / 256));
    e = cudaMalloc((void**)&w.part, sizeof(double) * (size_t)w.nparts * 2 * N * N);
    if (e == cudaSuccess) e = cudaMalloc((void**)&w.gsum, sizeof(double) * 2 * N * N);
    if (e == cudaSuccess) e = cudaMalloc((void**)&w.C, sizeof(float) * N * N);
    if (e == cudaSuccess) e = cudaMalloc((void**)&w.E, sizeof(float) * N * N);
    if (e == cudaSuccess) e = cudaMalloc((void**)&w.s, sizeof(float) * N);
    if (e == cudaSuccess) e = cudaMalloc((void**)&w.Y, sizeof(float) * N * N);
    if (e == cudaSuccess) e = cudaMalloc((void**)&w.rpart, sizeof(double) * (2 * (size_t)h->sms + 1) * N);
  }
  if (e == cudaSuccess && K > w.K_alloc) {
    if (w.F) cudaFree(w.F);
    w.F = nullptr;
    e = cudaMalloc((void**)&w.F, sizeof(float) * (size_t)N * (K + N));
    if (e == cudaSuccess) w.K_alloc = K;
  }
  return e;
}

// HA^T R^-1 D and HA^T R^-1 HA of the last analysis's innovations into w.gsum
static cudaError_t warm_sums(enkf_handle_s* h) {
  WarmState& w = *h->warm;
  const auto& c = h->cfg;
  const int64_t rows_per = (c.m + w.nparts - 1) / w.nparts;
  const df32* HAdf = static_cast<const df32*>(h->ws.HAdf);
  const df32* Ddf = static_cast<const df32*>(h->ws.Ddf);
  if (c.N <= 32)
    warm_gram_kernel<2><<<w.nparts, kThreads, 0, h->stream>>>(HAdf, Ddf, h->ws.r32, c.m, c.N, rows_per, w.part);
  else if (c.N <= 64)
    warm_gram_kernel<4><<<w.nparts, kThreads, 0, h->stream>>>(HAdf, Ddf, h->ws.r32, c.m, c.N, rows_per, w.part);
  else
    warm_gram_kernel<8><<<w.nparts, kThreads, 0, h->stream>>>(HAdf, Ddf, h->ws.r32, c.m, c.N, rows_per, w.part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  warm_reduce_kernel<<<(2 * c.N * c.N + 255) / 256, 256, 0, h->stream>>>(w.part, w.nparts, 2 * c.N * c.N, w.gsum);
  return cudaGetLastError();
}
static cudaError_t warm_features_into(enkf_handle_s* h, int K, float* F) {
  WarmState& w = *h->warm;
  const auto& c = h->cfg;
  warm_features_kernel<<<c.N, kThreads, 0, h->stream>>>(static_cast<const df32*>(h->ws.Ddf), c.m, c.N, K, w.gsum, F, w.s);
  return cudaGetLastError();
}

cudaError_t warm_features(enkf_handle_s* h, int K, float* F, float* T) {
  cudaError_t e = warm_alloc(h, 0);
  if (e == cudaSuccess) e = warm_sums(h);
  if (e == cudaSuccess) e = warm_features_into(h, K, F);
  if (e == cudaSuccess && T) {
    warm_targets_kernel<<<(h->cfg.N * h->cfg.N + 255) / 256, 256, 0, h->stream>>>(h->ws.W, h->warm->s, h->cfg.N, T);
    e = cudaGetLastError();
  }
  return e;
}

cudaError_t warm_set_model(enkf_handle_s* h, const enkf_mlp_shape* shape, const float* params, std::string& err) {
  MlpLayout L;
  if (!mlp_layout(shape, L)) { err = "bad MLP shape"; return cudaErrorInvalidValue; }
  const int N = h->cfg.N;
  if (L.out != N || L.in <= N) { err = "the model must map K + N features to N outputs (K >= 1)"; return cudaErrorInvalidValue; }
  cudaError_t e = warm_alloc(h, L.in - N);
  if (e != cudaSuccess) { err = "allocation"; return e; }
  WarmState& w = *h->warm;
  if (w.work) cudaFree(w.work);
  w.work = nullptr;
  e = cudaMalloc((void**)&w.work, sizeof(float) * mlp_work_floats(L, N));
  if (e != cudaSuccess) { err = "allocation"; return e; }
  // limits for the largest N: they belong to the kernels, and a handle of fewer members must not lower them
  constexpr int smem = (int)(sizeof(float) * (2 * 128 + 16) * (128 + 1)), rsm = (int)(sizeof(float) * (128 + 16) * (128 + 1));
  e = cudaFuncSetAttribute(warm_decode_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(warm_decode_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(warm_decode_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(warm_resid_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, rsm);
  if (e != cudaSuccess) { err = "decoder shared memory"; return e; }
  w.L = L;
  w.params = params;
  w.K = L.in - N;
  return cudaSuccess;
}

bool warm_ready(const enkf_handle_s* h) { return h->warm && h->warm->params; }

// Learned start of one analysis: features -> MLP -> decoder into the solve's Zdf.
cudaError_t warm_prepare(enkf_handle_s* h) {
  WarmState& w = *h->warm;
  const auto& c = h->cfg;
  cudaError_t e = cudaSuccess;
  if (h->krylov) {   // the solve's own products, formed ahead of it
    e = launch_krylov(h, 1);
    if (e != cudaSuccess) return e;
    const df32* small = static_cast<const df32*>(h->ws.ksmall);
    warm_sums_kernel<<<(c.N * c.N + 255) / 256, 256, 0, h->stream>>>(small, small + c.N * c.N, c.N, w.gsum);
    e = cudaGetLastError();
  } else {
    e = warm_sums(h);
  }
  if (e == cudaSuccess) e = warm_features_into(h, w.K, w.F);
  if (e != cudaSuccess) return e;
  const MlpWork W = carve(w.L, c.N, w.work);
  e = mlp_forward_impl(w.L, w.params, w.F, nullptr, c.N, W, w.Y, h->stream);
  if (e != cudaSuccess) return e;
  warm_coef_kernel<<<c.N, 128, 0, h->stream>>>(w.Y, w.s, w.gsum, c.N, w.C, w.E);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int grid = (int)std::min<int64_t>(2 * (int64_t)h->sms, (c.m + 15) / 16);
  if (h->krylov) {
    const size_t rsm = std::max(sizeof(float) * (size_t)(c.N + 16) * (c.N + 1), sizeof(double) * (size_t)kThreads);
    const df32* HAk = static_cast<const df32*>(h->ws.HAdf);
    if (c.N <= 32)
      warm_resid_kernel<2><<<grid, kThreads, rsm, h->stream>>>(HAk, c.m, c.N, w.E, w.rpart);
    else if (c.N <= 64)
      warm_resid_kernel<4><<<grid, kThreads, rsm, h->stream>>>(HAk, c.m, c.N, w.E, w.rpart);
    else
      warm_resid_kernel<8><<<grid, kThreads, rsm, h->stream>>>(HAk, c.m, c.N, w.E, w.rpart);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    warm_reduce_kernel<<<(c.N + 255) / 256, 256, 0, h->stream>>>(w.rpart, grid, c.N, w.rpart + (size_t)2 * h->sms * c.N);
    return cudaGetLastError();
  }
  const size_t smem = sizeof(float) * (size_t)(2 * c.N + 16) * (c.N + 1);
  const df32* HAdf = static_cast<const df32*>(h->ws.HAdf);
  const df32* Ddf = static_cast<const df32*>(h->ws.Ddf);
  df32* Z0 = static_cast<df32*>(h->ws.Zdf);
  float* B0 = static_cast<float*>(h->ws.B);
  if (c.N <= 32)
    warm_decode_kernel<2><<<grid, kThreads, smem, h->stream>>>(HAdf, Ddf, h->ws.r32, c.m, c.N, w.C, w.E, Z0, B0);
  else if (c.N <= 64)
    warm_decode_kernel<4><<<grid, kThreads, smem, h->stream>>>(HAdf, Ddf, h->ws.r32, c.m, c.N, w.C, w.E, Z0, B0);
  else
    warm_decode_kernel<8><<<grid, kThreads, smem, h->stream>>>(HAdf, Ddf, h->ws.r32, c.m, c.N, w.C, w.E, Z0, B0);
  return cudaGetLastError();
}

cudaError_t warm_solve(enkf_handle_s* h) {
  const WarmState& w = *h->warm;
  return launch_krylov(h, 2, w.C, w.rpart + (size_t)2 * h->sms * h->cfg.N);
}

void warm_free(enkf_handle_s* h) {
  WarmState* w = h->warm;
  if (!w) return;
  void* ptrs[] = {w->part, w->gsum, w->C, w->E, w->F, w->s, w->Y, w->work, w->rpart};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete w;
  h->warm = nullptr;
}

int64_t mlp_param_count(const enkf_mlp_shape* s) {
  MlpLayout L;
  return mlp_layout(s, L) ? L.total : -1;
}

int64_t mlp_work_bytes(const enkf_mlp_shape* s, int B) {
  MlpLayout L;
  return (mlp_layout(s, L) && B > 0) ? (int64_t)(sizeof(float) * mlp_work_floats(L, B)) : -1;
}

cudaError_t mlp_forward(const enkf_mlp_shape* s, const float* P, const float* X, const int32_t* rows, int B,
                        float* Y, void* work, cudaStream_t st) {
  MlpLayout L;
  if (!mlp_layout(s, L) || B < 1) return cudaErrorInvalidValue;
  return mlp_forward_impl(L, P, X, rows, B, carve(L, B, static_cast<float*>(work)), Y, st);
}

cudaError_t mlp_loss_grad(const enkf_mlp_shape* s, const float* P, const float* X, const float* T,
                          const int32_t* rows, int B, float* grad, float* loss, void* work, cudaStream_t st) {
  MlpLayout L;
  if (!mlp_layout(s, L) || B < 1) return cudaErrorInvalidValue;
  return mlp_loss_grad_impl(L, P, X, T, rows, B, grad, loss, carve(L, B, static_cast<float*>(work)), st);
}

cudaError_t mlp_adam(int64_t count, float* P, const float* g, float* m, float* v, int step, float lr, float b1,
                     float b2, float eps, cudaStream_t st) {
  const float c1 = (float)(1.0 - std::pow((double)b1, step)), c2 = (float)(1.0 - std::pow((double)b2, step));
  adam_kernel<<<ew_grid(count), 256, 0, st>>>(P, g, m, v, count, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

cudaError_t mlp_train_epoch(const enkf_mlp_shape* s, float* P, float* m, float* v, const float* X, const float* T,
                            const int32_t* perm, int64_t rows, int B, int step0, float lr, float* losses,
                            void* work, float* grad, cudaStream_t st) {
  MlpLayout L;
  if (!mlp_layout(s, L) || B < 1 || rows < B) return cudaErrorInvalidValue;
  const MlpWork W = carve(L, B, static_cast<float*>(work));
  cudaError_t e = cudaSuccess;
  const int64_t nb = rows / B;
  for (int64_t q = 0; q < nb && e == cudaSuccess; ++q) {
    e = mlp_loss_grad_impl(L, P, X, T, perm + q * B, B, grad, losses ? losses + q : nullptr, W, st);
    if (e == cudaSuccess) e = mlp_adam(L.trained, P, grad, m, v, step0 + (int)q + 1, lr, 0.9f, 0.999f, 1e-8f, st);
  }
  return e;
}

cudaError_t mlp_standardize(const enkf_mlp_shape* s, float* P, const float* X, const float* T, int64_t rows,
                            cudaStream_t st) {
  MlpLayout L;
  if (!mlp_layout(s, L) || rows < 1) return cudaErrorInvalidValue;
  colstats_kernel<<<(L.in + 127) / 128, 128, 0, st>>>(X, rows, L.in, P + L.mu_in, P + L.sd_in);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) colstats_kernel<<<(L.out + 127) / 128, 128, 0, st>>>(T, rows, L.out, P + L.mu_out, P + L.sd_out);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace enkf
