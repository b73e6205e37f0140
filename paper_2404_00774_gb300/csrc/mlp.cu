// Learned probe count (not part of the paper): per-query features, labels,
// and a small MLP with its own forward, backward and Adam kernels.
//
// Features z(q) = [q || its top-64 centroid scores <q, C_i>, descending].
// Label t*(q) = the smallest probe count whose recall@k reaches the target:
// a true neighbour v is found at probe count t exactly when one of v's
// partitions sits at probe position <= t, so t* is the ceil(target k)-th
// smallest of those positions (position = 1 + #centroids ranked before p,
// ties to the lower id).
// Network: y = w3 . relu(W2 relu(W1 z + b1) + b2) + b3, trained by mean
// squared error against log t*; t(q) = clamp(ceil(alpha exp(y)), 1, c).
//
// Parameters live in one fp32 buffer: W1 [H][D] | b1 [H] | W2 [H][H] | b2 [H]
// | W3 [H] | b3 [1].  In bf16 mode the weights and inputs of every product
// are rounded to bf16 (round to nearest even) and products accumulate in fp32;
// the fp32 master weights take the Adam updates.
#include <algorithm>
#include <cmath>

#include "internal.cuh"

namespace soar {

namespace {

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// 64 x 64 tile of C = A B on the CUDA cores, shared by the network's products.
// The sum of every output runs over k in ascending order with one fp32 FMA a
// term, so the activations do not depend on the tiling: in bf16 mode the next
// product rounds them, where another order would now and then round the other
// way (the tensor cores' accumulation order is therefore not used here).
// Bound: the FMA pipe.  128 threads hold 8 x 4 outputs each (3 16-byte shared
// loads feed 32 FMAs; the 4 x 4 outputs of 256 threads took 2 for 16); 64-row
// tiles keep 256 blocks busy on a 4 096-row batch of a 256-unit layer, where
// 128-row tiles would leave SMs idle.  The next 16 k are loaded into registers
// while the current ones are multiplied.
constexpr int kTile = 64, kStep = 16, kPad = kTile + 4, kGemmThreads = 128;
using GemmTile = float[kStep][kPad];

// How an operand lies in memory: kAlongK: element (i, k) at p[i * ld + k];
// kAcross: at p[k * ld + i].
enum class Order { kAlongK, kAcross };

template <Order O>
struct Operand {
  const float* __restrict__ p;
  int64_t ld;
  int count;              // valid i
  static constexpr int kPer = kTile * kStep / kGemmThreads;
  __device__ static int row(int u) { return O == Order::kAlongK ? threadIdx.x / kStep + u * (kGemmThreads / kStep) : threadIdx.x % kTile; }
  __device__ static int col(int u) { return O == Order::kAlongK ? threadIdx.x % kStep : threadIdx.x / kTile + u * (kGemmThreads / kTile); }
  __device__ void load(float (&v)[kPer], int i0, int64_t k0, int64_t kend) const {
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int i = i0 + row(u);
      const int64_t k = k0 + col(u);
      v[u] = (i < count && k < kend) ? (O == Order::kAlongK ? p[i * ld + k] : p[k * ld + i]) : 0.f;
    }
  }
  __device__ static void store(const float (&v)[kPer], bool round, GemmTile& t) {
#pragma unroll
    for (int u = 0; u < kPer; ++u) t[col(u)][row(u)] = round ? bf16r(v[u]) : v[u];
  }
};

// acc[i][j] (row 8 * (tid / 16) + i, column 4 * (tid % 16) + j of the tile at
// (m0, n0)) = sum over k in [k0, kend).  With `sums`, sums[0] collects this
// thread's share of the unrounded A column sums (kAcross: column tid % 64,
// every second k).
template <Order OA, Order OB>
__device__ void gemm_tile(const Operand<OA>& A, const Operand<OB>& B, int m0, int n0, int64_t k0, int64_t kend,
                          bool round, float (&acc)[8][4], float* sums) {
  __shared__ __align__(16) GemmTile As, Bs;
  constexpr int kPer = Operand<OA>::kPer;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  float va[kPer], vb[kPer];
  A.load(va, m0, k0, kend);
  B.load(vb, n0, k0, kend);
  for (; k0 < kend; k0 += kStep) {
    __syncthreads();
    Operand<OA>::store(va, round, As);
    Operand<OB>::store(vb, round, Bs);
    if (sums) {
#pragma unroll
      for (int u = 0; u < kPer; ++u) *sums += va[u];
    }
    __syncthreads();
    if (k0 + kStep < kend) {
      A.load(va, m0, k0 + kStep, kend);
      B.load(vb, n0, k0 + kStep, kend);
    }
#pragma unroll
    for (int kk = 0; kk < kStep; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[kk][8 * ty]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[kk][8 * ty + 4]);
      const float4 b = *reinterpret_cast<const float4*>(&Bs[kk][4 * tx]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
  }
}

// H [M][N] = relu(X W^T + bias), X [M][K], W [N][K].
__global__ void __launch_bounds__(kGemmThreads) layer_forward(const float* __restrict__ X, const float* __restrict__ W,
                                                              const float* __restrict__ bias, int M, int N, int K,
                                                              int round, float* __restrict__ H) {
  const int m0 = blockIdx.x * kTile, n0 = blockIdx.y * kTile;
  float acc[8][4];
  gemm_tile<Order::kAlongK, Order::kAlongK>({X, K, M}, {W, K, N}, m0, n0, 0, K, round != 0, acc, nullptr);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + 8 * ty + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 4 * tx + j;
      if (n < N) H[(int64_t)m * N + n] = fmaxf(acc[i][j] + bias[n], 0.f);
    }
  }
}

// gA1 [M][N] = (gA2 W2) where H1 > 0 (0 elsewhere), gA2 [M][N], W2 [N][N].
__global__ void __launch_bounds__(kGemmThreads) layer_backward(const float* __restrict__ gA2,
                                                               const float* __restrict__ W2,
                                                               const float* __restrict__ H1, int M, int N, int round,
                                                               float* __restrict__ gA1) {
  const int m0 = blockIdx.x * kTile, n0 = blockIdx.y * kTile;
  float acc[8][4];
  gemm_tile<Order::kAlongK, Order::kAcross>({gA2, N, M}, {W2, N, N}, m0, n0, 0, N, round != 0, acc, nullptr);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + 8 * ty + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 4 * tx + j;
      if (n < N) gA1[(int64_t)m * N + n] = H1[(int64_t)m * N + n] > 0.f ? acc[i][j] : 0.f;
    }
  }
}

// y [M] = H2 w3 + b3, each row's sum over h in ascending order: 32 rows a
// block, staged 256 columns at a time (whole lines, 64 loads in flight a
// thread), one lane of warp 0 adding up a row.  Optionally gy = 2 (y - target)
// / M and the probe count clamp(ceil(alpha exp(y)), 1, c).
constexpr int kHeadRows = 32, kHeadCols = 256;
__global__ void __launch_bounds__(128) head_forward(const float* __restrict__ H2, const float* __restrict__ w3,
                                                    const float* __restrict__ b3, int M, int N, int round,
                                                    float* __restrict__ y, const float* __restrict__ target,
                                                    float* __restrict__ gy, float alpha, int c,
                                                    int32_t* __restrict__ t) {
  __shared__ float hs[kHeadRows][kHeadCols + 1], ws[kHeadCols];
  const int64_t m0 = (int64_t)blockIdx.x * kHeadRows;
  float acc = 0.f;
  for (int n0 = 0; n0 < N; n0 += kHeadCols) {
    __syncthreads();
#pragma unroll 16
    for (int i = threadIdx.x; i < kHeadRows * kHeadCols; i += 128) {
      const int r = i / kHeadCols, n = n0 + i % kHeadCols;
      const float v = (m0 + r < M && n < N) ? H2[(m0 + r) * N + n] : 0.f;
      hs[r][i % kHeadCols] = round ? bf16r(v) : v;
    }
    for (int i = threadIdx.x; i < kHeadCols; i += 128) {
      const float v = n0 + i < N ? w3[n0 + i] : 0.f;
      ws[i] = round ? bf16r(v) : v;
    }
    __syncthreads();
    if (threadIdx.x < kHeadRows) {
#pragma unroll 16
      for (int n = 0; n < kHeadCols; ++n) acc = fmaf(hs[threadIdx.x][n], ws[n], acc);
    }
  }
  const int64_t m = m0 + threadIdx.x;
  if (threadIdx.x >= kHeadRows || m >= M) return;
  const float v = acc + *b3;
  if (y) y[m] = v;
  if (gy) gy[m] = 2.f * (v - target[m]) / (float)M;
  if (t) t[m] = (int32_t)fminf(fmaxf(ceilf(alpha * expf(v)), 1.f), (float)c);
}

// Rows [r0, r1) of split blockIdx.x: gA2 = gy w3^T where H2 > 0, and the
// split's partial sums of the head's gradients (gW3, gb2, gb3) and of the
// squared error, written at their places in `part` (a copy of the parameter
// layout, then the loss).  32 columns a block, its warps taking every eighth
// row: a thread per column and whole split left most SMs idle (49 us on a
// 4 096 x 256 batch).
constexpr int kHbWarps = 8;
__global__ void __launch_bounds__(32 * kHbWarps) head_backward(
    const float* __restrict__ H2, const float* __restrict__ w3, const float* __restrict__ y,
    const float* __restrict__ target, const float* __restrict__ gy, int M, int N, int rows, int round, int64_t at_w3,
    int64_t at_b2, int64_t at_b3, int64_t plen, float* __restrict__ gA2, float* __restrict__ part) {
  __shared__ float sw[kHbWarps][32], sb[kHbWarps][32];
  const int r0 = blockIdx.x * rows, r1 = min(M, r0 + rows);
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, n = blockIdx.y * 32 + lane;
  float* mine = part + (int64_t)blockIdx.x * plen;
  float gw = 0.f, gb = 0.f;
  if (n < N) {
    const float w = round ? bf16r(w3[n]) : w3[n];
#pragma unroll 8
    for (int r = r0 + warp; r < r1; r += kHbWarps) {
      const float h = H2[(int64_t)r * N + n], g0 = __ldg(gy + r), g = round ? bf16r(g0) : g0;
      const float ga = h > 0.f ? fmaf(g, w, 0.f) : 0.f;
      gA2[(int64_t)r * N + n] = ga;
      gw = fmaf(g, round ? bf16r(h) : h, gw);
      gb += ga;
    }
  }
  sw[warp][lane] = gw;
  sb[warp][lane] = gb;
  __syncthreads();
  if (warp == 0 && n < N) {
    for (int u = 1; u < kHbWarps; ++u) {
      gw += sw[u][lane];
      gb += sb[u][lane];
    }
    mine[at_w3 + n] = gw;
    mine[at_b2 + n] = gb;
  }
  if (blockIdx.y == 0 && warp == 1) {
    float sg = 0.f, se = 0.f;
    for (int r = r0 + lane; r < r1; r += 32) {
      const float e = y[r] - target[r];
      sg += gy[r];
      se = fmaf(e, e, se);
    }
    sg = warp_sum(sg);
    se = warp_sum(se);
    if (lane == 0) {
      mine[at_b3] = sg;
      mine[plen - 1] = se;
    }
  }
}

// Weight gradients of both hidden layers over the rows of split blockIdx.z:
// gW2 = gA2^T H1 (blockIdx.y < t2: column tiles of H), gW1 = gA1^T Z (the
// other column tiles, of D) and, beside gW1's first column tile, gb1 = the
// column sums of gA1.  A batch has thousands of rows and the gradients only
// H x (H + D) entries, so the rows are split: one block a tile would leave 28
// of 152 SMs busy with a 4 096-long sum.
__global__ void __launch_bounds__(kGemmThreads) weight_grads(const float* __restrict__ gA2,
                                                             const float* __restrict__ H1,
                                                             const float* __restrict__ gA1,
                                                             const float* __restrict__ Z, int M, int H, int D,
                                                             int rows, int t2, int round, int64_t at_w1,
                                                             int64_t at_b1, int64_t at_w2, int64_t plen,
                                                             float* __restrict__ part) {
  const int64_t r0 = (int64_t)blockIdx.z * rows, r1 = min((int64_t)M, r0 + rows);
  float* mine = part + (int64_t)blockIdx.z * plen;
  const bool second = (int)blockIdx.y < t2;
  const int m0 = blockIdx.x * kTile, n0 = (second ? blockIdx.y : blockIdx.y - t2) * kTile;
  const int N = second ? H : D;
  const bool bias = !second && n0 == 0;
  float acc[8][4], sum = 0.f;
  gemm_tile<Order::kAcross, Order::kAcross>({second ? gA2 : gA1, H, H}, {second ? H1 : Z, N, N}, m0, n0, r0, r1,
                                            round != 0, acc, bias ? &sum : nullptr);
  float* out = mine + (second ? at_w2 : at_w1);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + 8 * ty + i;
    if (m >= H) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 4 * tx + j;
      if (n < N) out[(int64_t)m * N + n] = acc[i][j];
    }
  }
  if (bias) {                       // uniform in the block
    __shared__ float half[kTile];
    if (threadIdx.x >= kTile) half[threadIdx.x - kTile] = sum;
    __syncthreads();
    if (threadIdx.x < kTile && m0 + (int)threadIdx.x < H) mine[at_b1 + m0 + threadIdx.x] = sum + half[threadIdx.x];
  }
}

// G[i] = the splits' partial gradients added in split order; the entry behind
// them is the squared error, written to loss as a mean.
__global__ void sum_splits(const float* __restrict__ part, int splits, int64_t plen, int M, float* __restrict__ G,
                           float* __restrict__ loss) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= plen) return;
  float s = 0.f;
#pragma unroll 8
  for (int k = 0; k < splits; ++k) s += part[(int64_t)k * plen + i];
  if (i < plen - 1) G[i] = s;
  else if (loss) *loss = s / (float)M;
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                            float* __restrict__ m2, int64_t n, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float a = b1 * m1[i] + (1.f - b1) * gi;
  const float b = b2 * m2[i] + (1.f - b2) * gi * gi;
  m1[i] = a;
  m2[i] = b;
  p[i] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
}

// Features: [q || top-`top` centroid scores, descending] (top list from top-t).
template <typename QT>
__global__ void build_features(const QT* __restrict__ Q, int64_t nq, int d, const float* __restrict__ top_s, int top,
                               float* __restrict__ Z) {
  const int64_t q = blockIdx.x;
  const int D = d + top;
  for (int i = threadIdx.x; i < D; i += blockDim.x)
    Z[q * D + i] = i < d ? load_elem(Q, q * d + i) : top_s[q * top + (i - d)];
}

// Label kernel: block per query.  Position of partition p in the query's
// probe order = 1 + #{i : s_i > s_p or (s_i == s_p and i < p)}.
__global__ void label_kernel(const float* __restrict__ S, int c, const int64_t* __restrict__ truth, int k,
                             const int32_t* __restrict__ assign, int a, int64_t n, int need,
                             int32_t* __restrict__ labels) {
  extern __shared__ int32_t posv[];   // [k]
  const int64_t q = blockIdx.x;
  const float* row = S + q * c;
  __shared__ int32_t red[32];
  for (int v = 0; v < k; ++v) {
    const int64_t id = truth[q * k + v];
    int best = 0x7fffffff;           // an id outside [0, n) is never found
    if (id >= 0 && id < n) {
      for (int j = 0; j < a; ++j) {
        const int p = assign[id * a + j];
        const float sp = row[p];
        int cnt = 0;
        for (int i = threadIdx.x; i < c; i += blockDim.x) {
          const float si = row[i];
          cnt += (si > sp) || (si == sp && i < p);
        }
        cnt = warp_sum(cnt);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = cnt;
        __syncthreads();
        if (threadIdx.x == 0) {
          int tot = 0;
          for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
          best = min(best, tot + 1);
        }
        __syncthreads();
      }
    }
    if (threadIdx.x == 0) posv[v] = best;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // need-th smallest position (insertion sort of k values)
    for (int i = 1; i < k; ++i) {
      const int x = posv[i];
      int j = i - 1;
      while (j >= 0 && posv[j] > x) { posv[j + 1] = posv[j]; --j; }
      posv[j + 1] = x;
    }
    labels[q] = posv[need - 1];
  }
}

struct Layout {
  int64_t W1, b1, W2, b2, W3, b3, total;
  Layout(int D, int H) {
    W1 = 0;
    b1 = W1 + (int64_t)H * D;
    W2 = b1 + H;
    b2 = W2 + (int64_t)H * H;
    W3 = b2 + H;
    b3 = W3 + H;
    total = b3 + 1;
  }
};

}  // namespace

int64_t mlp_param_count(int D, int H) { return Layout(D, H).total; }

// The hidden layers into caller-provided activations (H1, H2 of [B][H]).
static void hidden_forward(const float* P, const Layout& L, int D, int H, const float* Z, int B, bool bf16, float* H1,
                           float* H2, cudaStream_t s) {
  const dim3 grid(ceil_div(B, kTile), ceil_div(H, kTile));
  layer_forward<<<grid, kGemmThreads, 0, s>>>(Z, P + L.W1, P + L.b1, B, H, D, bf16, H1);
  SOAR_LAUNCHED();
  layer_forward<<<grid, kGemmThreads, 0, s>>>(H1, P + L.W2, P + L.b2, B, H, H, bf16, H2);
  SOAR_LAUNCHED();
}

// Splits of a batch's rows for the weight gradients: 128 rows each where that
// gives at most 32, and never more than 256 MB of partial sums.
static int grad_splits(int B, int64_t plen) {
  const int64_t most = std::max<int64_t>(1, ((int64_t)64 << 20) / plen);
  return (int)std::min<int64_t>({(B + 127) / 128, (int64_t)32, most});
}

// Measured (batch 4 096, 164 -> 256 -> 256 -> 1, bf16, with the Adam step):
// before, every layer was computed twice (with and without the relu), the
// weight gradients ran as one 4 096-long sum per output on 16 blocks and the
// bias gradients on one thread per column: 1 841 us; now 117.
void mlp_backward(const float* P, int D, int H, const float* Z, const float* target, int B, bool bf16, float* G,
                  float* loss, cudaStream_t s, Scratch& scr) {
  const Layout L(D, H);
  const int64_t plen = L.total + 1;
  const int want = grad_splits(B, plen);
  const int rows = (B + want - 1) / want, splits = (B + rows - 1) / rows;
  const int64_t bh = (int64_t)B * H;
  float* act = scr.get<float>((size_t)4 * bh + 2 * (size_t)B);
  float *H1 = act, *H2 = act + bh, *gA2 = act + 2 * bh, *gA1 = act + 3 * bh, *y = act + 4 * bh, *gy = y + B;
  float* part = scr.get<float>((size_t)splits * plen);
  hidden_forward(P, L, D, H, Z, B, bf16, H1, H2, s);
  head_forward<<<ceil_div(B, kHeadRows), 128, 0, s>>>(H2, P + L.W3, P + L.b3, B, H, bf16, y, target, gy, 0.f, 1, nullptr);
  SOAR_LAUNCHED();
  head_backward<<<dim3(splits, ceil_div(H, 32)), 32 * kHbWarps, 0, s>>>(H2, P + L.W3, y, target, gy, B, H, rows, bf16,
                                                                       L.W3, L.b2, L.b3, plen, gA2, part);
  SOAR_LAUNCHED();
  layer_backward<<<dim3(ceil_div(B, kTile), ceil_div(H, kTile)), kGemmThreads, 0, s>>>(gA2, P + L.W2, H1, B, H, bf16,
                                                                                      gA1);
  SOAR_LAUNCHED();
  const unsigned t2 = ceil_div(H, kTile);
  weight_grads<<<dim3(ceil_div(H, kTile), t2 + ceil_div(D, kTile), splits), kGemmThreads, 0, s>>>(
      gA2, H1, gA1, Z, B, H, D, rows, (int)t2, bf16, L.W1, L.b1, L.W2, plen, part);
  SOAR_LAUNCHED();
  sum_splits<<<ceil_div(plen, 128), 128, 0, s>>>(part, splits, plen, B, G, loss);
  SOAR_LAUNCHED();
}

void mlp_adam(float* P, const float* G, float* m1, float* m2, int64_t n, int step, float lr, float b1, float b2,
              float eps, cudaStream_t s) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  adam_kernel<<<ceil_div(n, 256), 256, 0, s>>>(P, G, m1, m2, n, lr, b1, b2, eps, c1, c2);
  SOAR_LAUNCHED();
}

void mlp_predict(const float* P, int D, int H, const float* Z, int B, bool bf16, float alpha, int c, float* y_out,
                 int32_t* t_out, cudaStream_t s, Scratch& scr) {
  const Layout L(D, H);
  float* H1 = scr.get<float>((size_t)2 * B * H);
  float* H2 = H1 + (size_t)B * H;
  hidden_forward(P, L, D, H, Z, B, bf16, H1, H2, s);
  head_forward<<<ceil_div(B, kHeadRows), 128, 0, s>>>(H2, P + L.W3, P + L.b3, B, H, bf16, y_out, nullptr, nullptr, alpha, c,
                                               t_out);
  SOAR_LAUNCHED();
}

void probe_features(const IndexData& ix, const void* Q, soar_dtype dt, int64_t nq, int top, float* Z,
                    cudaStream_t s, Scratch& scr) {
  int32_t* t_ids = scr.get<int32_t>((size_t)nq * top);
  float* t_s = scr.get<float>((size_t)nq * top);
  select_partitions(ix, Q, dt, nq, top, t_ids, t_s, s, scr);
  if (dt == SOAR_F32)
    build_features<float><<<(unsigned)nq, 128, 0, s>>>(static_cast<const float*>(Q), nq, ix.d, t_s, top, Z);
  else
    build_features<__nv_bfloat16><<<(unsigned)nq, 128, 0, s>>>(static_cast<const __nv_bfloat16*>(Q), nq, ix.d, t_s,
                                                               top, Z);
  SOAR_LAUNCHED();
}

void features_from_scores(const void* Q, soar_dtype dt, int64_t nq, int d, const float* top_s, int top, float* Z,
                          cudaStream_t s) {
  if (dt == SOAR_F32)
    build_features<float><<<(unsigned)nq, 128, 0, s>>>(static_cast<const float*>(Q), nq, d, top_s, top, Z);
  else
    build_features<__nv_bfloat16><<<(unsigned)nq, 128, 0, s>>>(static_cast<const __nv_bfloat16*>(Q), nq, d, top_s,
                                                               top, Z);
  SOAR_LAUNCHED();
}

void probe_labels(const IndexData& ix, const void* Q, soar_dtype dt, int64_t nq, const int64_t* truth, int k,
                  float target, int32_t* labels, cudaStream_t s, Scratch& scr) {
  // every centroid score of every query, computed exactly as the search ranks them
  float* S = scr.get<float>((size_t)nq * ix.c);
  centroid_scores(ix, Q, dt, nq, S, s, scr);
  const int need = std::max(1, (int)ceilf(target * (float)k - 1e-6f));
  label_kernel<<<(unsigned)nq, 256, sizeof(int32_t) * k, s>>>(S, ix.c, truth, k, ix.assign, 1 + ix.spills, ix.n,
                                                             std::min(need, k), labels);
  SOAR_LAUNCHED();
}

}  // namespace soar
