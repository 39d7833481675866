// Mass-preconditioner network: a multilayer perceptron (ReLU hidden layers,
// linear output) trained by mean squared error with Adam, all on the device.
// The matrix products run on the tensor cores as BF16 operands with FP32
// accumulation (mma.sync m16n8k16); parameters, Adam moments and every other
// quantity stay FP32.  The paper's HMC uses the diagonal Fourier mass of Eq.
// Mass_matrix; the mass affects efficiency only (Sec. 4.1.2), and the network
// predicts per-bin log multipliers of it from binned features of the problem.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "bps_internal.h"

namespace bps {
namespace {

constexpr int MLP_MAX_LAYERS = 4;
constexpr int MLP_MAX_WIDTH = 512;
constexpr float MASSNET_ZMAX = 4.0f;   // clamp of the standardised network-mass features

// ------------------------------------------------------------------ GEMM
// C[M x N] = op(A)[M x K] op(B)[K x N] (+ bias[N]) (ReLU if act), FP32 in and
// out, BF16 operands.  TA: A is stored K x M (element (m,k) at A[k*lda + m]);
// TB: B is stored N x K (element (k,n) at B[n*ldb + k]).  One warp computes one
// 16 x 8 tile of C; operands are converted to BF16 as they are loaded.
// With `mask` (same layout as C) the result is multiplied by (mask > 0): the
// ReLU derivative of a backward pass.
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

template <bool TA, bool TB>
__global__ void __launch_bounds__(128) k_gemm(int M, int N, int K, const float* __restrict__ A, int lda,
                                              const float* __restrict__ B, int ldb, float* __restrict__ C, int ldc,
                                              const float* __restrict__ bias, int act,
                                              const float* __restrict__ mask) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int tiles_n = (N + 7) / 8;
  const int tm = warp / tiles_n, tn = warp % tiles_n;
  if (tm * 16 >= M) return;
  const int g = lane >> 2, q = lane & 3;
  auto a_at = [&](int m, int k) -> float {
    if (m >= M || k >= K) return 0.f;
    return TA ? A[(long long)k * lda + m] : A[(long long)m * lda + k];
  };
  auto b_at = [&](int k, int n) -> float {
    if (k >= K || n >= N) return 0.f;
    return TB ? B[(long long)n * ldb + k] : B[(long long)k * ldb + n];
  };
  const int m0 = tm * 16, n0 = tn * 8;
  float c[4] = {0.f, 0.f, 0.f, 0.f};
  for (int k0 = 0; k0 < K; k0 += 16) {
    uint32_t a[4], b[2];
    a[0] = pack_bf16(a_at(m0 + g, k0 + 2 * q), a_at(m0 + g, k0 + 2 * q + 1));
    a[1] = pack_bf16(a_at(m0 + g + 8, k0 + 2 * q), a_at(m0 + g + 8, k0 + 2 * q + 1));
    a[2] = pack_bf16(a_at(m0 + g, k0 + 2 * q + 8), a_at(m0 + g, k0 + 2 * q + 9));
    a[3] = pack_bf16(a_at(m0 + g + 8, k0 + 2 * q + 8), a_at(m0 + g + 8, k0 + 2 * q + 9));
    b[0] = pack_bf16(b_at(k0 + 2 * q, n0 + g), b_at(k0 + 2 * q + 1, n0 + g));
    b[1] = pack_bf16(b_at(k0 + 2 * q + 8, n0 + g), b_at(k0 + 2 * q + 9, n0 + g));
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + g + (i >= 2 ? 8 : 0);
    const int n = n0 + 2 * q + (i & 1);
    if (m < M && n < N) {
      float v = c[i];
      if (bias) v += bias[n];
      if (act) v = fmaxf(v, 0.f);
      if (mask && !(mask[(long long)m * ldc + n] > 0.f)) v = 0.f;
      C[(long long)m * ldc + n] = v;
    }
  }
}

// column sums of G [M x N] into out[N] (bias gradients)
__global__ void k_colsum(int M, int N, const float* __restrict__ G, float* __restrict__ out) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  float s = 0.f;
  for (int m = 0; m < M; ++m) s += G[(long long)m * N + n];
  out[n] = s;
}

// d loss / d y = 2 (y - t) / (M N) and the loss sum (per-block FP64 partials)
__global__ void k_mse(int total, float scale, const float* __restrict__ y, const float* __restrict__ t,
                      float* __restrict__ g, double* __restrict__ part) {
  __shared__ double sh[8];
  double acc = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const float r = y[i] - t[i];
    g[i] = 2.f * r * scale;
    acc += (double)r * r;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w];
    part[blockIdx.x] = s * scale;
  }
}

// Adam with bias correction, in place on one FP32 parameter
constexpr float ADAM_B1 = 0.9f, ADAM_B2 = 0.999f, ADAM_EPS = 1e-8f;
__device__ __forceinline__ void adam_update(float* p, float g, float* m, float* v, float lr, float c1, float c2) {
  const float mi = ADAM_B1 * *m + (1.f - ADAM_B1) * g;
  const float vi = ADAM_B2 * *v + (1.f - ADAM_B2) * g * g;
  *m = mi;
  *v = vi;
  *p -= lr * (mi / c1) / (sqrtf(vi / c2) + ADAM_EPS);
}
__global__ void k_adam(int n, float* __restrict__ p, const float* __restrict__ grad, float* __restrict__ m,
                       float* __restrict__ v, float lr, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) adam_update(p + i, grad[i], m + i, v + i, lr, c1, c2);
}

// rows idx[0..B) of X [n x d] into out [B x d]; idx drawn from Philox
__global__ void k_gather(int B, int d, int n, uint64_t seed, uint64_t step, const float* __restrict__ X,
                         const float* __restrict__ T, int dt, float* __restrict__ xo, float* __restrict__ to) {
  const int r = blockIdx.x;
  if (r >= B) return;
  __shared__ int src;
  if (threadIdx.x == 0) {
    P4 w = philox((uint64_t)r, step, 100, 0, seed);
    src = (int)(w.w[0] % (uint64_t)n);
  }
  __syncthreads();
  for (int j = threadIdx.x; j < d; j += blockDim.x) xo[(long long)r * d + j] = X[(long long)src * d + j];
  for (int j = threadIdx.x; j < dt; j += blockDim.x) to[(long long)r * dt + j] = T[(long long)src * dt + j];
}

// ------------------------------------------------------------------ training steps in one kernel
// A minibatch step of a small network is sixteen launches of a few microseconds
// each, with one warp per output tile and little to do per launch (75 us per step
// at 32 -> 128 -> 128 -> 64 and 64 rows; 19.5 us here, bound by the instruction
// streams and L2 latencies of six stages).  Here one thread-block cluster runs many
// steps: the stages of a step are separated by cluster barriers, every warp takes
// output tiles of the stage's products, and parameters, moments and activations
// stay in L2 (they are read past L1: the barrier's acquire orders them).  Stage by
// stage the arithmetic is that of the launch-per-stage kernels (the same tiles,
// the same order of products and sums), so the parameters are the same bits.
// Stages of a step with L layers: L forward products (the last also forms the
// loss gradient), then for l = L-1 .. 0 the weight and bias gradients of layer l,
// the gradient of its input, and Adam on layer l + 1, whose weights nothing reads
// any more; layer 0 applies Adam where its gradients are formed.  2 L barriers.
constexpr int TRAIN_THREADS = 512, TRAIN_CHUNK = 256, TRAIN_MAX_BATCH = 1024;
constexpr long long TRAIN_MAX_TILES = 3000;   // of a step, all stages (train_in_cluster)

struct TrainArgs {
  int L, B, n, steps;
  int sizes[MLP_MAX_LAYERS + 1];
  long long off_w[MLP_MAX_LAYERS], off_b[MLP_MAX_LAYERS];
  float *p, *g, *m, *v;
  float *act[MLP_MAX_LAYERS + 1], *grad[MLP_MAX_LAYERS + 1];
  const float *X, *T;
  uint64_t seed;
  unsigned long long step0;
  float lr;
  double* loss;   // NULL, or where the last step's loss goes
};
struct TrainCorr {
  float c1[TRAIN_CHUNK], c2[TRAIN_CHUNK];   // Adam's bias corrections of every step
};

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The elements k and k + 1 of one row of A or column of B, read past L1, for an
// operand stored along k (`pair`: rows 8-byte aligned) ...
struct AlongK {
  const float* p;
  bool pair;
  __device__ __forceinline__ float2 full(int k) const {
    if (pair) return __ldcg(reinterpret_cast<const float2*>(p + k));
    return make_float2(__ldcg(p + k), __ldcg(p + k + 1));
  }
  __device__ __forceinline__ float at(int k) const { return __ldcg(p + k); }
};
// ... across k (elements ld apart), and for columns of minibatch rows of X
struct AcrossK {
  const float* p;
  int ld;
  __device__ __forceinline__ float2 full(int k) const { return make_float2(__ldcg(p + k * ld), __ldcg(p + (k + 1) * ld)); }
  __device__ __forceinline__ float at(int k) const { return __ldcg(p + k * ld); }
};
struct AcrossRows {
  const float* p;
  const int* src;
  int ld;
  __device__ __forceinline__ float at(int k) const { return __ldcg(p + (long long)src[k] * ld); }
  __device__ __forceinline__ float2 full(int k) const { return make_float2(at(k), at(k + 1)); }
};

// One 16 x 8 tile of C = A B (K terms) by one warp, BF16 operands, FP32 sums.  a0,
// a1: rows m0 + lane / 4 and 8 below; b: column n0 + lane / 4; rows and columns
// beyond the matrix are any others (their results are not used).  With two warps
// per scheduler a stage is bound by the length of a warp's instruction stream, so
// bounds are checked in the last K step only.
template <class A, class B>
__device__ __forceinline__ void mma_tile(int K, const A& a0, const A& a1, const B& b, float (&c)[4]) {
  const int k2 = 2 * (threadIdx.x & 3);
  c[0] = c[1] = c[2] = c[3] = 0.f;
  auto step = [&](float2 x0, float2 x1, float2 x2, float2 x3, float2 y0, float2 y1) {
    const uint32_t ra[4] = {pack_bf16(x0.x, x0.y), pack_bf16(x1.x, x1.y), pack_bf16(x2.x, x2.y), pack_bf16(x3.x, x3.y)};
    const uint32_t rb[2] = {pack_bf16(y0.x, y0.y), pack_bf16(y1.x, y1.y)};
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(ra[0]), "r"(ra[1]), "r"(ra[2]), "r"(ra[3]), "r"(rb[0]), "r"(rb[1]));
  };
  constexpr int U = 4;
  int k = k2;
  const int full = K / 16;
  int i = 0;
  for (; i + U <= full; i += U) {
    float2 x[U][4], y[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u, k += 16) {
      x[u][0] = a0.full(k);
      x[u][1] = a1.full(k);
      x[u][2] = a0.full(k + 8);
      x[u][3] = a1.full(k + 8);
      y[u][0] = b.full(k);
      y[u][1] = b.full(k + 8);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) step(x[u][0], x[u][1], x[u][2], x[u][3], y[u][0], y[u][1]);
  }
#pragma unroll 1
  for (; i < full; ++i, k += 16) step(a0.full(k), a1.full(k), a0.full(k + 8), a1.full(k + 8), b.full(k), b.full(k + 8));
  if (K % 16) {
    auto tail = [&](const auto& r, int j) { return make_float2(j < K ? r.at(j) : 0.f, j + 1 < K ? r.at(j + 1) : 0.f); };
    step(tail(a0, k), tail(a1, k), tail(a0, k + 8), tail(a1, k + 8), tail(b, k), tail(b, k + 8));
  }
}

__device__ __forceinline__ bool pairs_ok(const float* p, int ld) {
  return ld % 2 == 0 && (reinterpret_cast<uintptr_t>(p) & 7) == 0;
}

__global__ void __launch_bounds__(TRAIN_THREADS, 1)
    k_train(const __grid_constant__ TrainArgs a, const __grid_constant__ TrainCorr corr) {
  __shared__ int s_src[2][TRAIN_MAX_BATCH];   // the minibatch's rows, this step's and the next one's
  __shared__ double s_red[TRAIN_THREADS / 32];
  const int t = threadIdx.x, lane = t & 31, g = lane >> 2, q2 = 2 * (lane & 3);
  // consecutive tiles to different blocks, so that few tiles use every block
  const int warp = (t >> 5) * (int)gridDim.x + (int)blockIdx.x, warps = TRAIN_THREADS / 32 * (int)gridDim.x;
  const int L = a.L, B = a.B, bt = (B + 15) / 16;
  const int no = a.sizes[L], total = B * no;
  const float scale = 1.f / (float)total;
  auto draw_rows = [&](int s) {
    for (int r = t; r < B; r += TRAIN_THREADS) {
      const P4 w = philox((uint64_t)r, a.step0 + s, 100, 0, a.seed);
      s_src[s & 1][r] = (int)(w.w[0] % (uint64_t)a.n);
    }
  };
  draw_rows(0);
  __syncthreads();
  for (int s = 0; s < a.steps; ++s) {
    const int* src = s_src[s & 1];
    const float c1 = corr.c1[s], c2 = corr.c2[s];
    // ---- forward
    for (int l = 0; l < L; ++l) {
      const int ni = a.sizes[l], nl = a.sizes[l + 1], nt = (nl + 7) / 8;
      const float* W = a.p + a.off_w[l];
      const float* bias = a.p + a.off_b[l];
      const float* h = a.act[l];
      const bool last = l == L - 1, pa = pairs_ok(l == 0 ? a.X : h, ni);
      for (int q = warp; q < bt * nt; q += warps) {
        const int m = q / nt * 16 + g, n = q % nt * 8;
        const int ma = min(m, B - 1), mb = min(m + 8, B - 1);
        const float* r0 = l == 0 ? a.X + (long long)src[ma] * ni : h + ma * ni;
        const float* r1 = l == 0 ? a.X + (long long)src[mb] * ni : h + mb * ni;
        // the epilogue's bias and target, in flight with the operands
        float be[2], te[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int mi = i < 2 ? ma : mb, ne = min(n + q2 + (i & 1), nl - 1);
          if (i < 2) be[i] = __ldcg(bias + ne);
          te[i] = last ? __ldg(a.T + (long long)src[mi] * nl + ne) : 0.f;
        }
        float c[4];
        mma_tile(ni, AlongK{r0, pa}, AlongK{r1, pa}, AcrossK{W + min(n + g, nl - 1), nl}, c);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int me = m + (i >= 2 ? 8 : 0), ne = n + q2 + (i & 1);
          if (me >= B || ne >= nl) continue;
          float y = c[i] + be[i & 1];
          if (!last) y = fmaxf(y, 0.f);
          a.act[l + 1][me * nl + ne] = y;
          if (last) {               // d loss / d y = 2 (y - t) / (B n)
            const float r = y - te[i];
            a.grad[L][me * nl + ne] = 2.f * r * scale;
          }
        }
      }
      cluster_barrier();
    }
    if (a.loss && s == a.steps - 1 && blockIdx.x == 0) {
      double acc = 0.0;
      for (int i = t; i < total; i += TRAIN_THREADS) {
        const float r = __ldcg(a.act[L] + i) - __ldg(a.T + (long long)src[i / no] * no + i % no);
        acc += (double)r * r;
      }
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
      if (lane == 0) s_red[t >> 5] = acc;
      __syncthreads();
      if (t == 0) {
        double sum = 0.0;
        for (int w = 0; w < TRAIN_THREADS / 32; ++w) sum += s_red[w];
        *a.loss = sum * scale;
      }
    }
    draw_rows(s + 1);   // the barriers below order it before the next step
    // ---- backward
    for (int l = L - 1; l >= 0; --l) {
      const int ni = a.sizes[l], nl = a.sizes[l + 1];
      const float* G = a.grad[l + 1];
      const float* W = a.p + a.off_w[l];
      const float* h = a.act[l];
      float* gw = a.g + a.off_w[l];
      float* gb = a.g + a.off_b[l];
      const bool pg = pairs_ok(G, nl), pw = pairs_ok(W, nl);
      const int it = (ni + 7) / 8, mt = (ni + 15) / 16, nt = (nl + 7) / 8;
      const int n_in = l > 0 ? bt * it : 0, n_w = mt * nt, n_b = (nl + 31) / 32;
      const long long first = l < L - 1 ? a.off_w[l + 1] : 0;   // layer l + 1: weights, then biases
      const int n_par = l < L - 1 ? a.sizes[l + 1] * a.sizes[l + 2] + a.sizes[l + 2] : 0;
      const int n_adam = (n_par + 127) / 128;
      for (int q = warp; q < n_in + n_w + n_b + n_adam; q += warps) {
        if (q < n_in) {             // G_l = (G_{l+1} W_l^T) relu'(z_l)
          const int m = q / it * 16 + g, n = q % it * 8;
          const int ma = min(m, B - 1), mb = min(m + 8, B - 1);
          float z[4], c[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) z[i] = __ldcg(h + (i < 2 ? ma : mb) * ni + min(n + q2 + (i & 1), ni - 1));
          mma_tile(nl, AlongK{G + ma * nl, pg}, AlongK{G + mb * nl, pg}, AlongK{W + min(n + g, ni - 1) * nl, pw}, c);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int me = m + (i >= 2 ? 8 : 0), ne = n + q2 + (i & 1);
            if (me < B && ne < ni) a.grad[l][me * ni + ne] = z[i] > 0.f ? c[i] : 0.f;
          }
        } else if (q < n_in + n_w) {   // dW_l = h_l^T G_{l+1}; layer 0: and Adam on it
          const int i0 = q - n_in, m = i0 / nt * 16 + g, n = i0 % nt * 8;
          const int ma = min(m, ni - 1), mb = min(m + 8, ni - 1);
          const AcrossK cols{G + min(n + g, nl - 1), nl};
          float c[4];
          if (l == 0) mma_tile(B, AcrossRows{a.X + ma, src, ni}, AcrossRows{a.X + mb, src, ni}, cols, c);
          else mma_tile(B, AcrossK{h + ma, ni}, AcrossK{h + mb, ni}, cols, c);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int me = m + (i >= 2 ? 8 : 0), ne = n + q2 + (i & 1);
            if (me >= ni || ne >= nl) continue;
            const int e = me * nl + ne;
            gw[e] = c[i];
            if (l == 0) adam_update(a.p + a.off_w[0] + e, c[i], a.m + a.off_w[0] + e, a.v + a.off_w[0] + e, a.lr, c1, c2);
          }
        } else if (q < n_in + n_w + n_b) {   // bias gradients: column sums in row order
          const int n = (q - n_in - n_w) * 32 + lane;
          if (n < nl) {
            float sum = 0.f;
#pragma unroll 16
            for (int m = 0; m < B; ++m) sum += __ldcg(G + m * nl + n);
            gb[n] = sum;
            if (l == 0) adam_update(a.p + a.off_b[0] + n, sum, a.m + a.off_b[0] + n, a.v + a.off_b[0] + n, a.lr, c1, c2);
          }
        } else {                        // Adam on layer l + 1
          const int i0 = (q - n_in - n_w - n_b) * 128 + lane;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + 32 * u;
            if (i < n_par) {
              const long long e = first + i;
              adam_update(a.p + e, __ldcg(a.g + e), a.m + e, a.v + e, a.lr, c1, c2);
            }
          }
        }
      }
      cluster_barrier();
    }
  }
}

__global__ void k_sum(const double* part, int n, double* out) {
  double s = 0.0;
  for (int i = 0; i < n; ++i) s += part[i];
  *out = s;
}

__global__ void k_to_bf16(long long n, const float* __restrict__ src, __nv_bfloat16* __restrict__ dst) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = __float2bfloat16_rn(src[i]);
}

__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

}  // namespace

// ------------------------------------------------------------------ in-graph inference
// One device allocation: this header, then per layer the BF16 weights and the
// FP32 biases at the byte offsets below (16-byte aligned).
struct MassNet {
  int n_layers;
  int sizes[MLP_MAX_LAYERS + 1];
  long long off_w[MLP_MAX_LAYERS], off_b[MLP_MAX_LAYERS];
  float mean[MLP_MAX_WIDTH], sd[MLP_MAX_WIDTH];
  float log_clamp;
};

namespace {

// One block per chain: the features [ln P_m, ln W_m] of the chain's current
// state, standardised and clamped to +-MASSNET_ZMAX (a state far outside the
// training range, e.g. a bin whose P drifts, must not drive the network to
// arbitrary outputs), through the network with the numerics of the training
// kernels (operands rounded to BF16, FP32 accumulation, FP32 bias and ReLU),
// then s_j = exp(clamp(y_j)) into the chain's mass scales.  A matrix-vector
// product per layer (at most 512 x 512): FP32 FMAs over coalesced weight rows.
__global__ void __launch_bounds__(256) k_mass_net(ScalarArgs a, const MassNet* __restrict__ m) {
  await_previous();
  DevState* ds = a.ds + blockIdx.y;
  __shared__ float h[2][MLP_MAX_WIDTH];
  const int t = threadIdx.x, nb = a.n_bins;
  const char* base = reinterpret_cast<const char*>(m);
  const int n0 = m->sizes[0];
  for (int i = t; i < n0; i += blockDim.x) {
    const float f = i < nb ? (float)log(ds->P[i]) : ds->wfeat[i - nb];
    const float z = (f - m->mean[i]) / m->sd[i];
    h[0][i] = bf16_round(fminf(fmaxf(z, -MASSNET_ZMAX), MASSNET_ZMAX));
  }
  __syncthreads();
  int cur = 0;
  const int L = m->n_layers;
  for (int l = 0; l < L; ++l) {
    const int ni = m->sizes[l], no = m->sizes[l + 1];
    const __nv_bfloat16* W = reinterpret_cast<const __nv_bfloat16*>(base + m->off_w[l]);
    const float* b = reinterpret_cast<const float*>(base + m->off_b[l]);
    for (int j = t; j < no; j += blockDim.x) {
      float acc = 0.f;
      for (int i = 0; i < ni; ++i) acc = fmaf(h[cur][i], __bfloat162float(W[(long long)i * no + j]), acc);
      float v = acc + b[j];
      if (l < L - 1) v = bf16_round(fmaxf(v, 0.f));
      h[cur ^ 1][j] = v;
    }
    __syncthreads();
    cur ^= 1;
  }
  const float c = m->log_clamp;
  for (int j = t; j < m->sizes[L]; j += blockDim.x) ds->mass_scale[j] = exp((double)fminf(fmaxf(h[cur][j], -c), c));
}

}  // namespace

int massnet_width(const bps_mlp* net, int output);
bps_status massnet_create(const bps_mlp* net, const float* mean, const float* sd, double log_clamp, MassNet** out);
void massnet_destroy(MassNet* m) { cudaFree(m); }

void launch_mass_net(const ScalarArgs& a, const MassNet* m, int nch, cudaStream_t s) {
  launch_dep(k_mass_net, dim3(1, nch), dim3(256), 0, s, a, m);
}

}  // namespace bps

using namespace bps;

struct bps_mlp {
  int L = 0;                       // number of layers
  int sizes[MLP_MAX_LAYERS + 1] = {0};
  size_t n_params = 0;
  size_t off_w[MLP_MAX_LAYERS] = {0}, off_b[MLP_MAX_LAYERS] = {0};
  cudaStream_t stream = nullptr;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  // activations for a batch of up to cap rows
  int cap = 0;
  float* act[MLP_MAX_LAYERS + 1] = {nullptr};   // act[0] = input copy, act[l] = layer output
  float* grad_act[MLP_MAX_LAYERS + 1] = {nullptr};
  float *xb = nullptr, *tb = nullptr;           // minibatch buffers of the trainer
  double* part = nullptr;
  double* loss_dev = nullptr;
  long long adam_t = 0;
  std::string err;
};

namespace {

bps_status mfail(bps_mlp* n, bps_status s, const char* msg) {
  if (n) n->err = msg;
  set_last_error(msg);
  return s;
}

void gemm(bps_mlp* net, bool ta, bool tb, int M, int N, int K, const float* A, int lda, const float* B, int ldb,
          float* C, int ldc, const float* bias, int act, const float* mask) {
  const int warps = ((M + 15) / 16) * ((N + 7) / 8);
  const int blocks = (warps * 32 + 127) / 128;
  if (!ta && !tb) k_gemm<false, false><<<blocks, 128, 0, net->stream>>>(M, N, K, A, lda, B, ldb, C, ldc, bias, act, mask);
  else if (ta && !tb) k_gemm<true, false><<<blocks, 128, 0, net->stream>>>(M, N, K, A, lda, B, ldb, C, ldc, bias, act, mask);
  else if (!ta && tb) k_gemm<false, true><<<blocks, 128, 0, net->stream>>>(M, N, K, A, lda, B, ldb, C, ldc, bias, act, mask);
  else k_gemm<true, true><<<blocks, 128, 0, net->stream>>>(M, N, K, A, lda, B, ldb, C, ldc, bias, act, mask);
}

bps_status ensure_cap(bps_mlp* net, int B) {
  if (B <= net->cap) return BPS_OK;
  for (int l = 0; l <= net->L; ++l) {
    cudaFree(net->act[l]);
    cudaFree(net->grad_act[l]);
    net->act[l] = net->grad_act[l] = nullptr;
  }
  cudaFree(net->xb);
  cudaFree(net->tb);
  cudaFree(net->part);
  bool ok = true;
  for (int l = 0; l <= net->L && ok; ++l) {
    ok = cudaMalloc((void**)&net->act[l], (size_t)B * net->sizes[l] * sizeof(float)) == cudaSuccess &&
         cudaMalloc((void**)&net->grad_act[l], (size_t)B * net->sizes[l] * sizeof(float)) == cudaSuccess;
  }
  ok = ok && cudaMalloc((void**)&net->xb, (size_t)B * net->sizes[0] * sizeof(float)) == cudaSuccess &&
       cudaMalloc((void**)&net->tb, (size_t)B * net->sizes[net->L] * sizeof(float)) == cudaSuccess &&
       cudaMalloc((void**)&net->part, 256 * sizeof(double)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    net->cap = 0;
    return mfail(net, BPS_ENOMEM, "network buffers do not fit");
  }
  net->cap = B;
  return BPS_OK;
}

// forward pass of B rows from x (device, B x n0); outputs in act[L]
void forward(bps_mlp* net, int B, const float* x) {
  const float* h = x;
  for (int l = 0; l < net->L; ++l) {
    const int ni = net->sizes[l], no = net->sizes[l + 1];
    gemm(net, false, false, B, no, ni, h, ni, net->p + net->off_w[l], no, net->act[l + 1], no,
         net->p + net->off_b[l], l < net->L - 1 ? 1 : 0, nullptr);
    h = net->act[l + 1];
  }
}

// loss and gradients for B rows (x, t device); gradients into net->g
void backward(bps_mlp* net, int B, const float* x, const float* t) {
  const int L = net->L, no = net->sizes[L];
  const int total = B * no;
  k_mse<<<64, 256, 0, net->stream>>>(total, 1.f / (float)total, net->act[L], t, net->grad_act[L], net->part);
  k_sum<<<1, 1, 0, net->stream>>>(net->part, 64, net->loss_dev);
  for (int l = L - 1; l >= 0; --l) {
    const int ni = net->sizes[l], nl = net->sizes[l + 1];
    const float* hin = l == 0 ? x : net->act[l];
    // dW_l = h_l^T G_{l+1}  (K = B)
    gemm(net, true, false, ni, nl, B, hin, ni, net->grad_act[l + 1], nl, net->g + net->off_w[l], nl, nullptr, 0,
         nullptr);
    k_colsum<<<(nl + 127) / 128, 128, 0, net->stream>>>(B, nl, net->grad_act[l + 1], net->g + net->off_b[l]);
    if (l > 0) {
      // G_l = (G_{l+1} W_l^T) * relu'(z_l)
      gemm(net, false, true, B, ni, nl, net->grad_act[l + 1], nl, net->p + net->off_w[l], nl, net->grad_act[l], ni,
           nullptr, 0, net->act[l]);
    }
  }
}

// the next step's bias corrections
void adam_advance(bps_mlp* net, float* c1, float* c2) {
  net->adam_t += 1;
  *c1 = 1.f - powf(ADAM_B1, (float)net->adam_t);
  *c2 = 1.f - powf(ADAM_B2, (float)net->adam_t);
}

void adam(bps_mlp* net, float lr) {
  float c1, c2;
  adam_advance(net, &c1, &c2);
  const int n = (int)net->n_params;
  k_adam<<<(n + 255) / 256, 256, 0, net->stream>>>(n, net->p, net->g, net->m, net->v, lr, c1, c2);
}

// Blocks of the training cluster: 16 where the GPU can place such a cluster (an
// opt-in size), else 8; 0 if it places neither.
int train_cluster_ctas() {
  static thread_local int known_dev = -1, ctas = 0;   // the attribute and the answer are per device
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (dev == known_dev) return ctas;
  known_dev = dev;
  ctas = 0;
  cudaFuncSetAttribute(k_train, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  for (int n : {16, 8}) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(n);
    lc.blockDim = dim3(TRAIN_THREADS);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)n;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, k_train, &lc) == cudaSuccess && fit > 0) {
      ctas = n;
      break;
    }
    cudaGetLastError();
  }
  return ctas;
}

// Whether the training steps of a minibatch of B rows run in one cluster (k_train)
// or as launches over the whole GPU: the cluster's 256 warps win while a stage
// gives each of them few tiles.  Measured, launches and cluster, in us per step:
// 32-128-128-64 with 64 rows (512 tiles) 75.0 and 19.5, 64-300-64 with 300 rows
// (2546) 82 and 49, 32-256-256-64 with 256 rows (2880) 115 and 91, 128-512-512-64
// with 64 rows (3872) 117 and 108, with 256 rows (7040) 144 and 294.
bool train_in_cluster(const bps_mlp* net, int B) {
  if (B > TRAIN_MAX_BATCH) return false;
  long long tiles = 0;
  for (int l = 0; l < net->L; ++l) {
    const long long bt = (B + 15) / 16, ni = net->sizes[l], nl = net->sizes[l + 1];
    tiles += bt * ((nl + 7) / 8) + ((ni + 15) / 16) * ((nl + 7) / 8) + (l > 0 ? bt * ((ni + 7) / 8) : 0);
  }
  return tiles <= TRAIN_MAX_TILES;
}

}  // namespace

extern "C" {

bps_status bps_mlp_create(int n_layers, const int* sizes, void* cuda_stream, bps_mlp** out) {
  if (!out || !sizes) return mfail(nullptr, BPS_EINVAL, "null argument");
  *out = nullptr;
  if (n_layers < 1 || n_layers > MLP_MAX_LAYERS) return mfail(nullptr, BPS_EINVAL, "1..4 layers");
  for (int l = 0; l <= n_layers; ++l)
    if (sizes[l] < 1 || sizes[l] > MLP_MAX_WIDTH) return mfail(nullptr, BPS_EINVAL, "layer widths must be in 1..512");
  bps_mlp* net = new bps_mlp();
  net->L = n_layers;
  net->stream = (cudaStream_t)cuda_stream;
  size_t off = 0;
  for (int l = 0; l <= n_layers; ++l) net->sizes[l] = sizes[l];
  for (int l = 0; l < n_layers; ++l) {
    net->off_w[l] = off;
    off += (size_t)sizes[l] * sizes[l + 1];
    net->off_b[l] = off;
    off += sizes[l + 1];
  }
  net->n_params = off;
  bool ok = cudaMalloc((void**)&net->p, off * sizeof(float)) == cudaSuccess &&
            cudaMalloc((void**)&net->g, off * sizeof(float)) == cudaSuccess &&
            cudaMalloc((void**)&net->m, off * sizeof(float)) == cudaSuccess &&
            cudaMalloc((void**)&net->v, off * sizeof(float)) == cudaSuccess &&
            cudaMalloc((void**)&net->loss_dev, sizeof(double)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    delete net;
    return mfail(nullptr, BPS_ENOMEM, "network allocation failed");
  }
  cudaMemsetAsync(net->p, 0, off * sizeof(float), net->stream);
  cudaMemsetAsync(net->m, 0, off * sizeof(float), net->stream);
  cudaMemsetAsync(net->v, 0, off * sizeof(float), net->stream);
  *out = net;
  return BPS_OK;
}

void bps_mlp_destroy(bps_mlp* net) {
  if (!net) return;
  cudaStreamSynchronize(net->stream);
  for (int l = 0; l <= net->L; ++l) {
    cudaFree(net->act[l]);
    cudaFree(net->grad_act[l]);
  }
  cudaFree(net->xb);
  cudaFree(net->tb);
  cudaFree(net->part);
  cudaFree(net->p);
  cudaFree(net->g);
  cudaFree(net->m);
  cudaFree(net->v);
  cudaFree(net->loss_dev);
  delete net;
}

size_t bps_mlp_num_params(const bps_mlp* net) { return net ? net->n_params : 0; }

bps_status bps_mlp_set_params(bps_mlp* net, const float* params) {
  if (!net || !params) return mfail(net, BPS_EINVAL, "null argument");
  if (cudaMemcpy(net->p, params, net->n_params * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(net->m, 0, net->n_params * sizeof(float)) != cudaSuccess ||
      cudaMemset(net->v, 0, net->n_params * sizeof(float)) != cudaSuccess)
    return mfail(net, BPS_ECUDA, "parameter upload failed");
  net->adam_t = 0;
  return BPS_OK;
}

bps_status bps_mlp_get_params(bps_mlp* net, float* params) {
  if (!net || !params) return mfail(net, BPS_EINVAL, "null argument");
  cudaStreamSynchronize(net->stream);
  if (cudaMemcpy(params, net->p, net->n_params * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
    return mfail(net, BPS_ECUDA, "parameter download failed");
  return BPS_OK;
}

bps_status bps_mlp_forward(bps_mlp* net, int batch, const float* x_dev, float* y_dev) {
  if (!net || !x_dev || !y_dev || batch < 1) return mfail(net, BPS_EINVAL, "bad argument");
  bps_status st = ensure_cap(net, batch);
  if (st != BPS_OK) return st;
  forward(net, batch, x_dev);
  const int no = net->sizes[net->L];
  cudaMemcpyAsync(y_dev, net->act[net->L], (size_t)batch * no * sizeof(float), cudaMemcpyDeviceToDevice,
                  net->stream);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(net->stream) != cudaSuccess)
    return mfail(net, BPS_ECUDA, "forward pass failed");
  return BPS_OK;
}

bps_status bps_mlp_loss_grad(bps_mlp* net, int batch, const float* x_dev, const float* t_dev, double* loss,
                             float* grads) {
  if (!net || !x_dev || !t_dev || batch < 1) return mfail(net, BPS_EINVAL, "bad argument");
  bps_status st = ensure_cap(net, batch);
  if (st != BPS_OK) return st;
  forward(net, batch, x_dev);
  backward(net, batch, x_dev, t_dev);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(net->stream) != cudaSuccess)
    return mfail(net, BPS_ECUDA, "backward pass failed");
  if (loss) cudaMemcpy(loss, net->loss_dev, sizeof(double), cudaMemcpyDeviceToHost);
  if (grads) cudaMemcpy(grads, net->g, net->n_params * sizeof(float), cudaMemcpyDeviceToHost);
  return BPS_OK;
}

bps_status bps_mlp_adam_step(bps_mlp* net, float lr) {
  if (!net) return mfail(nullptr, BPS_EINVAL, "null argument");
  adam(net, lr);
  if (cudaGetLastError() != cudaSuccess) return mfail(net, BPS_ECUDA, "Adam step failed");
  return BPS_OK;
}

bps_status bps_mlp_export(bps_mlp* net, const float* feat_mean, const float* feat_std, double log_clamp, void* blob,
                          size_t* bytes) {
  if (!net || !bytes) return mfail(net, BPS_EINVAL, "null argument");
  const size_t need = 12 + 4 * (size_t)(net->L + 1) + 8 + 2 * 4 * (size_t)net->sizes[0] + 4 * net->n_params;
  if (!blob) {
    *bytes = need;
    return BPS_OK;
  }
  if (*bytes < need) return mfail(net, BPS_EINVAL, "buffer too small for the preconditioner");
  if (!feat_mean || !feat_std) return mfail(net, BPS_EINVAL, "null argument");
  unsigned char* b = static_cast<unsigned char*>(blob);
  size_t off = 0;
  auto put = [&](const void* src, size_t n) {
    std::memcpy(b + off, src, n);
    off += n;
  };
  const uint32_t version = 1, L = (uint32_t)net->L;
  put("BPSM", 4);
  put(&version, 4);
  put(&L, 4);
  for (int l = 0; l <= net->L; ++l) {
    const uint32_t w = (uint32_t)net->sizes[l];
    put(&w, 4);
  }
  put(&log_clamp, 8);
  put(feat_mean, 4 * (size_t)net->sizes[0]);
  put(feat_std, 4 * (size_t)net->sizes[0]);
  std::vector<float> p(net->n_params);
  bps_status st = bps_mlp_get_params(net, p.data());
  if (st != BPS_OK) return st;
  put(p.data(), 4 * net->n_params);
  *bytes = need;
  return BPS_OK;
}

bps_status bps_mlp_train(bps_mlp* net, int n_examples, const float* x_dev, const float* t_dev, int batch, int steps,
                         float lr, uint64_t seed, double* last_loss) {
  if (!net || !x_dev || !t_dev || n_examples < 1 || batch < 1 || steps < 0)
    return mfail(net, BPS_EINVAL, "bad argument");
  bps_status st = ensure_cap(net, batch);
  if (st != BPS_OK) return st;
  const int d = net->sizes[0], dt = net->sizes[net->L];
  int done = 0;
  const int ctas = steps > 0 && train_in_cluster(net, batch) ? train_cluster_ctas() : 0;
  if (ctas > 0) {
    TrainArgs a{};
    a.L = net->L;
    a.B = batch;
    a.n = n_examples;
    for (int l = 0; l <= net->L; ++l) {
      a.sizes[l] = net->sizes[l];
      a.act[l] = net->act[l];
      a.grad[l] = net->grad_act[l];
    }
    for (int l = 0; l < net->L; ++l) {
      a.off_w[l] = (long long)net->off_w[l];
      a.off_b[l] = (long long)net->off_b[l];
    }
    a.p = net->p;
    a.g = net->g;
    a.m = net->m;
    a.v = net->v;
    a.X = x_dev;
    a.T = t_dev;
    a.seed = seed;
    a.lr = lr;
    while (done < steps) {
      TrainCorr corr;
      a.step0 = (unsigned long long)net->adam_t;
      a.steps = std::min(TRAIN_CHUNK, steps - done);
      for (int i = 0; i < a.steps; ++i) adam_advance(net, &corr.c1[i], &corr.c2[i]);
      done += a.steps;
      a.loss = done == steps ? net->loss_dev : nullptr;
      cudaLaunchConfig_t lc = {};
      lc.gridDim = dim3(ctas);
      lc.blockDim = dim3(TRAIN_THREADS);
      lc.stream = net->stream;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)ctas;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      lc.attrs = at;
      lc.numAttrs = 1;
      if (cudaLaunchKernelEx(&lc, k_train, a, corr) != cudaSuccess) return mfail(net, BPS_ECUDA, "training failed");
    }
  }
  for (int s = done; s < steps; ++s) {
    k_gather<<<batch, 64, 0, net->stream>>>(batch, d, n_examples, seed, (uint64_t)net->adam_t, x_dev, t_dev, dt,
                                            net->xb, net->tb);
    forward(net, batch, net->xb);
    backward(net, batch, net->xb, net->tb);
    adam(net, lr);
  }
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(net->stream) != cudaSuccess)
    return mfail(net, BPS_ECUDA, "training failed");
  if (last_loss) cudaMemcpy(last_loss, net->loss_dev, sizeof(double), cudaMemcpyDeviceToHost);
  return BPS_OK;
}

}  // extern "C"

namespace bps {

int massnet_width(const bps_mlp* net, int output) { return output ? net->sizes[net->L] : net->sizes[0]; }

bps_status massnet_create(const bps_mlp* net, const float* mean, const float* sd, double log_clamp, MassNet** out) {
  *out = nullptr;
  MassNet h{};
  h.n_layers = net->L;
  auto up16 = [](long long x) { return (x + 15) & ~15LL; };
  long long off = up16((long long)sizeof(MassNet));
  for (int l = 0; l <= net->L; ++l) h.sizes[l] = net->sizes[l];
  for (int l = 0; l < net->L; ++l) {
    h.off_w[l] = off;
    off = up16(off + 2LL * net->sizes[l] * net->sizes[l + 1]);
    h.off_b[l] = off;
    off = up16(off + 4LL * net->sizes[l + 1]);
  }
  for (int i = 0; i < net->sizes[0]; ++i) {
    h.mean[i] = mean[i];
    h.sd[i] = sd[i];
  }
  h.log_clamp = (float)log_clamp;
  char* blob = nullptr;
  if (cudaMalloc((void**)&blob, (size_t)off) != cudaSuccess) {
    cudaGetLastError();
    return mfail(nullptr, BPS_ENOMEM, "network copy allocation failed");
  }
  cudaStream_t s = net->stream;
  bool ok = cudaMemcpyAsync(blob, &h, sizeof(MassNet), cudaMemcpyHostToDevice, s) == cudaSuccess;
  for (int l = 0; l < net->L && ok; ++l) {
    const long long nw = (long long)net->sizes[l] * net->sizes[l + 1];
    k_to_bf16<<<(unsigned)((nw + 255) / 256), 256, 0, s>>>(nw, net->p + net->off_w[l],
                                                          reinterpret_cast<__nv_bfloat16*>(blob + h.off_w[l]));
    ok = cudaMemcpyAsync(blob + h.off_b[l], net->p + net->off_b[l], 4 * (size_t)net->sizes[l + 1],
                         cudaMemcpyDeviceToDevice, s) == cudaSuccess;
  }
  ok = ok && cudaGetLastError() == cudaSuccess && cudaStreamSynchronize(s) == cudaSuccess;
  if (!ok) {
    cudaFree(blob);
    return mfail(nullptr, BPS_ECUDA, "network copy failed");
  }
  *out = reinterpret_cast<MassNet*>(blob);
  return BPS_OK;
}

}  // namespace bps
