// mlp.cu -- training and inference kernels of the learned slicing proposer:
// a 3-layer MLP (features -> H -> H -> 1, ReLU, FP32) trained with a mean
// squared error on log2 contraction costs. Parameters are one flat array:
// W1 (H x F), b1 (H), W2 (H x H), b2 (H), W3 (H), b3 (1), weights row-major
// (output x input). Every reduction runs in a fixed order (no atomics), so
// a training step is deterministic.
//
// A backward pass is six launches: two layers forward, the head (prediction,
// its derivative and the loss's partial sums), the hidden layer backward, and
// every parameter's gradient over chunks of rows, added up in chunk order.
// What bounds it: at a training batch of 1024 rows the launches (each matrix
// has 8 to 64 tiles); at 10^5 rows the FP32 pipe, through the shared-memory
// loads of a 4 x 4 register tile.
// GB300, before (one thread per column for every sum over rows) and now: an
// epoch of 8256 rows in batches of 1024, 3.0 -> 1.1 ms; the gradient over
// 162805 rows (1.7e10 flops) 42.5 -> 1.14 ms, 15 TFLOP/s.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "../../include/tnq.h"

namespace tnq {
void set_error(const std::string& msg);

namespace {
constexpr int MT = 128;  // threads of a matrix tile
constexpr int MK = 16;   // summed values per shared-memory step
constexpr int TM = 4;    // a thread's tile: TM x TM results
constexpr int BM = 16 * TM, BN = 8 * TM;  // a block's

// acc += A B over k in [k0, k1), in increasing order, for the tile of BM x BN
// results at (m0, p0); la(m, k) and lb(p, k) are the operands inside M x P.
// LA / LB::kfast: consecutive k (else consecutive m / p) are consecutive memory.
// 4 x 4 results a thread: 64 such tiles of a 128-wide layer at 1024 rows keep
// four times as many SMs busy as 8 x 8 would (epoch 1.1 against 2.4 ms), and at
// 10^5 rows more blocks an SM hide the fetches better (1.14 against 1.33 ms).
template <class LA, class LB>
__device__ __forceinline__ void tile_product(const LA& la, const LB& lb, int m0, int p0, int M, int P, int k0, int k1,
                                             float (&acc)[TM][TM], float* sh) {
  constexpr int NA = BM * MK / MT, NB = BN * MK / MT;
  float(*sa)[BM + 4] = reinterpret_cast<float(*)[BM + 4]>(sh);
  float(*sb)[BN + 4] = reinterpret_cast<float(*)[BN + 4]>(sh + MK * (BM + 4));
  const int t = threadIdx.x, tx = t & 7, ty = t >> 3;
  float ra[NA], rb[NB];
  auto place = [&](bool kfast, int e, int B, int* row, int* k) {
    *k = kfast ? e % MK : e / B;
    *row = kfast ? e / MK : e % B;
  };
  auto fetch = [&](int kb) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      int r, k;
      place(LA::kfast, t + i * MT, BM, &r, &k);
      ra[i] = m0 + r < M && kb + k < k1 ? la(m0 + r, kb + k) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      int r, k;
      place(LB::kfast, t + i * MT, BN, &r, &k);
      rb[i] = p0 + r < P && kb + k < k1 ? lb(p0 + r, kb + k) : 0.f;
    }
  };
  fetch(k0);
  for (int kb = k0; kb < k1; kb += MK) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      int r, k;
      place(LA::kfast, t + i * MT, BM, &r, &k);
      sa[k][r] = ra[i];
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      int r, k;
      place(LB::kfast, t + i * MT, BN, &r, &k);
      sb[k][r] = rb[i];
    }
    __syncthreads();
    if (kb + MK < k1) fetch(kb + MK);  // in flight while this step is computed
#pragma unroll
    for (int k = 0; k < MK; ++k) {
      const float4 va = *reinterpret_cast<const float4*>(&sa[k][4 * ty]);
      const float4 vb = *reinterpret_cast<const float4*>(&sb[k][4 * tx]);
      const float a[TM] = {va.x, va.y, va.z, va.w}, b[TM] = {vb.x, vb.y, vb.z, vb.w};
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
  }
}
constexpr int TILE_FLOATS = MK * (BM + 4 + BN + 4);
// Row / column of acc[i][j] within the tile.
__device__ __forceinline__ int tile_row(int i) { return 4 * (threadIdx.x >> 3) + i; }
__device__ __forceinline__ int tile_col(int j) { return 4 * (threadIdx.x & 7) + j; }

struct RowMajor {  // X[row][k]
  static constexpr bool kfast = true;
  const float* p;
  int ld;
  __device__ float operator()(int r, int k) const { return p[(size_t)r * ld + k]; }
};
struct ColMajor {  // X[k][row]
  static constexpr bool kfast = false;
  const float* p;
  int ld;
  __device__ float operator()(int r, int k) const { return p[(size_t)k * ld + r]; }
};
// dZ2[i][j] = dP[i] W3[j] where H2[i][j] > 0, read by rows (kfast) or by columns
template <bool K>
struct HeadGrad {
  static constexpr bool kfast = K;
  const float *dP, *W3, *H2;
  int H;
  __device__ float at(int i, int j) const { return H2[(size_t)i * H + j] > 0.f ? dP[i] * W3[j] : 0.f; }
  __device__ float operator()(int r, int k) const { return K ? at(r, k) : at(k, r); }
};

// C = relu(A W^T + b): A (M x K), W (P x K)
__global__ void __launch_bounds__(MT) k_layer(const float* __restrict__ A, const float* __restrict__ W,
                                              const float* __restrict__ bias, float* __restrict__ C, int M, int K,
                                              int P) {
  __shared__ __align__(16) float sh[TILE_FLOATS];
  const int m0 = blockIdx.x * BM, p0 = blockIdx.y * BN;
  float acc[TM][TM] = {};
  tile_product(RowMajor{A, K}, RowMajor{W, K}, m0, p0, M, P, 0, K, acc, sh);
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) {
      const int r = m0 + tile_row(i), c = p0 + tile_col(j);
      if (r < M && c < P) {
        const float v = acc[i][j] + bias[c];
        C[(size_t)r * P + c] = v > 0.f ? v : 0.f;
      }
    }
}

// dZ1 = (dZ2 W2) where H1 > 0
__global__ void __launch_bounds__(MT) k_hidden_back(HeadGrad<true> dZ2, const float* __restrict__ W2,
                                                    const float* __restrict__ H1, float* __restrict__ dZ1, int M,
                                                    int H) {
  __shared__ __align__(16) float sh[TILE_FLOATS];
  const int m0 = blockIdx.x * BM, p0 = blockIdx.y * BN;
  float acc[TM][TM] = {};
  tile_product(dZ2, ColMajor{W2, H}, m0, p0, M, H, 0, H, acc, sh);
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) {
      const int r = m0 + tile_row(i), c = p0 + tile_col(j);
      if (r < M && c < H) dZ1[(size_t)r * H + c] = H1[(size_t)r * H + c] > 0.f ? acc[i][j] : 0.f;
    }
}

constexpr int HEAD_ROWS = 8;  // rows per block of k_head: one per warp

// pred[i] = H2[i] . W3 + b3; with y: dP[i] = (pred[i] - y[i]) / n and the
// block's partial sum of (pred - y)^2, else out[i] = pred[i].
__global__ void __launch_bounds__(32 * HEAD_ROWS) k_head(const float* __restrict__ H2, const float* __restrict__ W3,
                                                         const float* __restrict__ b3, const float* __restrict__ y,
                                                         float* __restrict__ out, float* __restrict__ part, int n,
                                                         int H) {
  __shared__ float s_sq[HEAD_ROWS];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, i = blockIdx.x * HEAD_ROWS + w;
  float a = 0.f;
  if (i < n)
    for (int k = lane; k < H; k += 32) a = fmaf(H2[(size_t)i * H + k], W3[k], a);
  for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
  a += *b3;
  if (!y) {
    if (i < n && lane == 0) out[i] = a;
    return;
  }
  const float e = i < n ? a - y[i] : 0.f;
  if (i < n && lane == 0) out[i] = e / (float)n;
  if (lane == 0) s_sq[w] = e * e;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int q = 0; q < HEAD_ROWS; ++q) s += s_sq[q];
    part[blockIdx.x] = s;
  }
}

struct GradArgs {
  const float *x, *H1, *H2, *W3, *dP, *dZ1;
  float* part;         // chunk c's sums at part + c * stride, laid out like the parameters
  size_t stride;
  int n, F, H, rows;   // rows per chunk
  int t2, t1;          // tiles of W2 and W1
};

// One chunk's part of every gradient (blockIdx.y): blocks 0..t2-1 tiles of dW2
// = dZ2^T H1, then t1 tiles of dW1 = dZ1^T x, then blocks of MT columns of the
// biases' and W3's sums.
__global__ void __launch_bounds__(MT) k_grads(const GradArgs g) {
  __shared__ __align__(16) float sh[TILE_FLOATS];
  const int r0 = blockIdx.y * g.rows, r1 = min(g.n, r0 + g.rows);
  float* W1 = g.part + blockIdx.y * g.stride;
  float* b1 = W1 + (size_t)g.H * g.F;
  float* W2 = b1 + g.H;
  float* b2 = W2 + (size_t)g.H * g.H;
  float* W3 = b2 + g.H;
  int b = blockIdx.x;
  const HeadGrad<false> dZ2{g.dP, g.W3, g.H2, g.H};
  if (b < g.t2 + g.t1) {
    const bool second = b < g.t2;
    if (!second) b -= g.t2;
    const int P = second ? g.H : g.F, cols = (P + BN - 1) / BN;
    const int m0 = b / cols * BM, p0 = b % cols * BN;
    float acc[TM][TM] = {};
    if (second) tile_product(dZ2, ColMajor{g.H1, g.H}, m0, p0, g.H, P, r0, r1, acc, sh);
    else tile_product(ColMajor{g.dZ1, g.H}, ColMajor{g.x, g.F}, m0, p0, g.H, P, r0, r1, acc, sh);
    float* dst = second ? W2 : W1;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TM; ++j) {
        const int r = m0 + tile_row(i), c = p0 + tile_col(j);
        if (r < g.H && c < P) dst[(size_t)r * P + c] = acc[i][j];
      }
    return;
  }
  b -= g.t2 + g.t1;
  const int c = b * MT + threadIdx.x;
  if (c < g.H) {
    float s1 = 0.f, s2 = 0.f, s3 = 0.f;
    const float w3 = g.W3[c];
#pragma unroll 4
    for (int r = r0; r < r1; ++r) {
      const float h2 = g.H2[(size_t)r * g.H + c], d = g.dP[r];
      s1 += g.dZ1[(size_t)r * g.H + c];
      s2 += h2 > 0.f ? d * w3 : 0.f;
      s3 = fmaf(d, h2, s3);
    }
    b1[c] = s1;
    b2[c] = s2;
    W3[c] = s3;
  }
  if (b == 0 && threadIdx.x < 32) {  // db3: lanes in turn, then over the lanes
    float s = 0.f;
    for (int r = r0 + (int)threadIdx.x; r < r1; r += 32) s += g.dP[r];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (threadIdx.x == 0) W3[g.H] = s;
  }
}

// grads = the chunks' sums in chunk order (part == grads: they are there
// already); the last block adds the loss's partial sums, in a fixed order.
__global__ void __launch_bounds__(256) k_add_up(const float* part, size_t stride, int chunks, float* grads, size_t count,
                                                const float* __restrict__ sq, int n_sq, float* loss, float scale) {
  if (blockIdx.x + 1 == gridDim.x) {
    __shared__ float s[256];
    float a = 0.f;
    for (int i = threadIdx.x; i < n_sq; i += 256) a += sq[i];
    s[threadIdx.x] = a;
    __syncthreads();
    for (int off = 128; off > 0; off >>= 1) {
      if ((int)threadIdx.x < off) s[threadIdx.x] += s[threadIdx.x + off];
      __syncthreads();
    }
    if (threadIdx.x == 0 && loss) *loss = s[0] * scale;
    return;
  }
  const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (part == grads || i >= count) return;
  float a = 0.f;
#pragma unroll 8
  for (int c = 0; c < chunks; ++c) a += part[c * stride + i];
  grads[i] = a;
}

// SGD with momentum: v = mu v + g ; w -= lr v.
__global__ void k_sgd(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ v, size_t n, float lr,
                      float mu) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float vi = mu * v[i] + g[i];
    v[i] = vi;
    w[i] -= lr * vi;
  }
}

struct Views {
  const float *W1, *b1, *W2, *b2, *W3, *b3;
};
Views views(const float* p, int F, int H) {
  Views v;
  v.W1 = p;
  v.b1 = v.W1 + (size_t)H * F;
  v.W2 = v.b1 + H;
  v.b2 = v.W2 + (size_t)H * H;
  v.W3 = v.b2 + H;
  v.b3 = v.W3 + H;
  return v;
}

int up(int a, int b) { return (a + b - 1) / b; }

void layer(const float* A, const float* W, const float* bias, float* C, int M, int K, int P, cudaStream_t s) {
  k_layer<<<dim3(up(M, BM), up(P, BN)), MT, 0, s>>>(A, W, bias, C, M, K, P);
}
}  // namespace
}  // namespace tnq

using namespace tnq;

extern "C" {

int32_t tnq_learned_features(void);
size_t tnq_learned_param_count(int32_t hidden);

size_t tnq_mlp_workspace_floats(int32_t hidden, size_t n) { return n * (5 * (size_t)hidden + 4) + 16; }

// Forward pass for n rows of features x (device, n x F) -> out (device, n).
tnq_status tnq_mlp_forward(const float* params, int32_t hidden, const float* x, size_t n, float* out, float* work,
                           void* stream) {
  if (!params || !x || !out || !work || hidden <= 0) { set_error("NULL argument"); return TNQ_EINVAL; }
  const int F = tnq_learned_features(), H = hidden, N = (int)n;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  Views v = views(params, F, H);
  float* H1 = work;
  float* H2 = H1 + (size_t)N * H;
  layer(x, v.W1, v.b1, H1, N, F, H, s);
  layer(H1, v.W2, v.b2, H2, N, H, H, s);
  k_head<<<up(N, HEAD_ROWS), 32 * HEAD_ROWS, 0, s>>>(H2, v.W3, v.b3, nullptr, out, nullptr, N, H);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(cudaGetErrorString(e)); return TNQ_ECUDA; }
  return TNQ_OK;
}

// Gradient of the mean squared error (1/2n) sum (f(x) - y)^2 with respect to
// every parameter, into grads (device, same layout as params); *loss (device).
tnq_status tnq_mlp_backward(const float* params, int32_t hidden, const float* x, const float* y, size_t n,
                            float* grads, float* loss, float* work, void* stream) {
  if (!params || !x || !y || !grads || !work || hidden <= 0 || n == 0) { set_error("bad argument"); return TNQ_EINVAL; }
  const int F = tnq_learned_features(), H = hidden, N = (int)n;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  Views v = views(params, F, H);
  const size_t nh = (size_t)N * H, count = (size_t)H * F + H + (size_t)H * H + 2 * (size_t)H + 1;
  float* H1 = work;         // N x H
  float* H2 = H1 + nh;      // N x H
  float* dZ1 = H2 + nh;     // N x H
  float* dP = dZ1 + nh;     // N
  float* sq = dP + N;       // N: the loss's partial sums
  float* part = sq + N;     // the rest of the workspace, 2 N H + 2 N + 16 floats: the chunks' gradients
  layer(x, v.W1, v.b1, H1, N, F, H, s);
  layer(H1, v.W2, v.b2, H2, N, H, H, s);
  const int n_sq = up(N, HEAD_ROWS);
  k_head<<<n_sq, 32 * HEAD_ROWS, 0, s>>>(H2, v.W3, v.b3, y, dP, sq, N, H);
  const HeadGrad<true> dZ2{dP, v.W3, H2, H};
  k_hidden_back<<<dim3(up(N, BM), up(H, BN)), MT, 0, s>>>(dZ2, v.W2, H1, dZ1, N, H);
  // chunks of at least 64 rows, as many as the workspace holds; one writes grads itself
  const size_t room = (2 * nh + 2 * (size_t)N + 16) / count;
  const int most = up(N, 64);
  int chunks = (int)std::min<size_t>(room, (size_t)std::min(most, 512));
  GradArgs g;
  g.rows = up(N, std::max(chunks, 1));
  chunks = up(N, g.rows);
  g.x = x, g.H1 = H1, g.H2 = H2, g.W3 = v.W3, g.dP = dP, g.dZ1 = dZ1;
  g.part = chunks > 1 ? part : grads;
  g.stride = count;
  g.n = N, g.F = F, g.H = H;
  g.t2 = up(H, BM) * up(H, BN);
  g.t1 = up(H, BM) * up(F, BN);
  const dim3 grid(g.t2 + g.t1 + up(H, MT), chunks);
  k_grads<<<grid, MT, 0, s>>>(g);
  k_add_up<<<(unsigned)((count + 255) / 256) + 1, 256, 0, s>>>(g.part, count, chunks, grads, count, sq, n_sq, loss,
                                                                1.f / (2.f * (float)N));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(cudaGetErrorString(e)); return TNQ_ECUDA; }
  return TNQ_OK;
}

tnq_status tnq_mlp_sgd(float* params, const float* grads, float* momentum, size_t count, float lr, float mu,
                       void* stream) {
  if (!params || !grads || !momentum) { set_error("NULL argument"); return TNQ_EINVAL; }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int blocks = (int)((count + 255) / 256 < 1024 ? (count + 255) / 256 : 1024);
  k_sgd<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(params, grads, momentum, count, lr, mu);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(cudaGetErrorString(e)); return TNQ_ECUDA; }
  return TNQ_OK;
}

}  // extern "C"
