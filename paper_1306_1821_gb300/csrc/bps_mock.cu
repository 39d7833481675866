// Artificial surveys on the device (Sec. 5 of the paper; App. D; Eq. rel_bias):
// the true density field, the galaxy counts of every subsample (Poisson, or
// the paper's Gaussian noise), the survey response of a spherical cap times a
// tabulated radial selection, and on the host the Schechter selection tables,
// the mean numbers per magnitude bin and the luminosity-dependent bias.
//
// Every FP64 step that decides an integer (a count, whether a voxel is
// inside the survey) is written with round-to-nearest intrinsics in a fixed
// order, without contraction into fused multiply-adds, so the results are the
// ones any IEEE 754 implementation of the same definition gives from the same
// inputs.  The ABI is declared and documented in include/bps.h.
#include <cmath>
#include <cstdint>
#include <algorithm>
#include <cstring>
#include <vector>

#include "bps_internal.h"
#include "bps_passes.cuh"

namespace bps {
namespace {

constexpr uint64_t ST_MOCK_FIELD = 8, ST_MOCK_COUNTS = 9;
constexpr double CHUNK_MEAN = 32.0;    // largest mean of one inversion chunk
constexpr double LAMBDA_MAX = 4096.0;  // larger means give the out-of-range count 65536
constexpr int MAX_STEPS = 200;         // bound of one chunk's inversion search

// amplitudes A = sqrt(P / V_cell) of every |n|^2 (0 for k = 0): FP64, rounded to FP32
__global__ void k_mock_amp(const double* __restrict__ P, int n, double vc, float* __restrict__ amp) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) amp[i] = i == 0 ? 0.f : __double2float_rn(__dsqrt_rn(__ddiv_rn(P[i], vc)));
}

struct Coef {
  double c[11];   // 1/j!, j = 0..10
};
constexpr Coef make_coef() {
  Coef k{};
  double fact = 1.0;
  for (int j = 0; j <= 10; ++j) {
    if (j > 0) fact *= j;
    k.c[j] = 1.0 / fact;
  }
  return k;
}
__constant__ Coef c_coef = make_coef();

// e^-mu for 0 <= mu <= 32: mu 2^-10 (exact), Taylor series of e^-x to degree
// 10 by Horner's rule, then ten squarings (IEEE-exact operations only)
__device__ __forceinline__ double exp_neg(double mu) {
  const double y = -__dmul_rn(mu, 0x1p-10);
  double s = c_coef.c[10];
#pragma unroll
  for (int j = 9; j >= 0; --j) s = __dadd_rn(__dmul_rn(s, y), c_coef.c[j]);
#pragma unroll
  for (int q = 0; q < 10; ++q) s = __dmul_rn(s, s);
  return s;
}

// b and Nbar of every subsample, and their splits into two FP32 parts
struct MockSub {
  double b[MAXS], nbar[MAXS];
  float2 b2[MAXS], nbar2[MAXS];
};

// FP32 pairs (x + y, |y| <= half an ulp of x): about 46 significant bits from
// FP32 arithmetic.  FP64 instructions, conversions included, issue at 1/64 of
// the FP32 rate here, so the mock kernels decide in pairs and keep FP64 for
// what the pairs cannot decide.
__device__ __forceinline__ float2 pair_quick(float a, float b) {   // |a| >= |b| or a = 0
  const float s = __fadd_rn(a, b);
  return make_float2(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ float2 pair_sum(float a, float b) {
  const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
  return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z)));
}
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  return pair_quick(p, __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, __fmaf_rn(a.x, b.x, -p))));
}
__device__ __forceinline__ float2 pair_add(float2 a, float2 b) {
  const float2 s = pair_sum(a.x, b.x);
  return pair_quick(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}

// Inversion of the Poisson distribution function of mean mu (0 < mu <= 32) at u:
// the smallest k with u <= F_k, in the FP64 operations that define the counts.
__device__ __noinline__ int poisson_invert(double mu, double u) {
  double p = exp_neg(mu), F = p;
  int k = 0;
  while (u > F && k < MAX_STEPS) {
    ++k;
    p = __ddiv_rn(__dmul_rn(p, mu), (double)k);
    F = __dadd_rn(F, p);
  }
  return k;
}

// 1 / k and the width of the undecided band around F_k, in units of F_k
struct ScreenTable {
  float inv[MAX_STEPS + 8], tol[MAX_STEPS + 8];
};
constexpr ScreenTable make_screen_table() {
  ScreenTable t{};
  for (int k = 0; k < MAX_STEPS + 8; ++k) {
    t.inv[k] = k == 0 ? 0.f : (float)(1.0 / (double)k);
    t.tol[k] = (float)((k + 2) * 4e-7);
  }
  return t;
}
__constant__ ScreenTable c_screen = make_screen_table();

// The same search in FP32 for the mean mu (an FP32 pair, off by less than 1e-10),
// with a bound on how far its F_k can be from the FP64 one; -1 where u lies
// within the bound of some F_k it meets, for the caller to decide in FP64.
// Bound, in units of 2^-24: e^-mu is off by 5 (expf 4, the pair's second part
// 1), each step of p by 4 (mu, 1 / k and two products) and each addition by 1,
// so F_k is off by at most (5 + 5 k) 2^-24 < (k + 1) 3e-7 of itself; u is rounded
// to FP32 (2^-24 of itself, and F is as large where it matters) from its upper
// 32 bits (2.4e-10).  Taken as (k + 2) 4e-7 F + 1e-9, it leaves about 1e-6 (k + 2)
// of the draws undecided.  The lanes of a warp walk through the same k together,
// four steps between tests: the chain of a step is one product and one sum.
__device__ __forceinline__ int poisson_screen(float2 mu, uint64_t w) {
  float p = expf(-mu.x);
  p = fmaf(-p, mu.y, p);
  const float u = __fmul_rn(__uint2float_rn((uint32_t)(w >> 32)), 0x1p-32f);
  float F = p;
  int n = 0;
  bool unsure = false;
  for (int k = 0; k < MAX_STEPS; k += 4) {
    float d = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      d = u - F;
      unsure |= fabsf(d) <= fmaf(F, c_screen.tol[k + j], 1e-9f);
      n += d > 0.f;
      p *= mu.x * c_screen.inv[k + j + 1];
      F += p;
    }
    if (d < 0.f || unsure) return unsure ? -1 : n;
  }
  return -1;
}

// The Poisson count of voxel i and subsample l with response r and field d by
// definition: lambda = (r Nbar) max(0, 1 + b d), in ceil(lambda / 32) chunks of equal mean.
__device__ __noinline__ int poisson_exact(float r, float d, double b, double nbar, long long i, int l, uint64_t seed) {
  const double rn = __dmul_rn((double)r, nbar);
  const double t = fmax(0.0, __dadd_rn(1.0, __dmul_rn(b, (double)d)));
  const double lam = __dmul_rn(rn, t);
  if (!(lam <= LAMBDA_MAX)) return 65536;
  const double K = ceil(__ddiv_rn(lam, CHUNK_MEAN));
  const double mu = K > 0.0 ? __ddiv_rn(lam, K) : 0.0;
  const int nk = (int)K;
  const float m = (float)mu;
  const float2 m2 = make_float2(m, (float)(mu - (double)m));
  int total = 0;
  P4 w{};
  for (int j = 0; j < nk; ++j) {
    if ((j & 3) == 0) w = philox((uint64_t)i, (uint64_t)(j >> 2), ST_MOCK_COUNTS, (uint64_t)l, seed);
    const uint64_t wj = (j & 3) == 0 ? w.w[0] : (j & 3) == 1 ? w.w[1] : (j & 3) == 2 ? w.w[2] : w.w[3];
    int k = poisson_screen(m2, wj);
    if (k < 0) k = poisson_invert(mu, u52(wj));
    total += k;
  }
  return total;
}

// The same count without FP64 where FP32 pairs decide it: one chunk (lambda
// safely below 32) of ordinary factors.  The pair for 1 + b d is off by less
// than 2^-43 (1 + |b d|), that for lambda by less than 2^-42 r Nbar (1 + |b d|),
// which is below 1e-10 for the factors let through.  |b d| < 1e12 keeps what r Nbar
// loses below FP32's smallest value (2^-149) as small; b and Nbar have ordinary
// splits (mock_counts).
__device__ __noinline__ int poisson_count(float r, float d, float2 b, float2 nb, double b64, double nbar64, long long i,
                                          int l, uint64_t seed) {
  const float q = __fmul_rn(b.x, d);
  const float2 bd = pair_quick(q, __fmaf_rn(b.y, d, __fmaf_rn(b.x, d, -q)));
  const float2 t = pair_add(make_float2(1.f, 0.f), bd);
  const float2 rn = pair_mul(make_float2(r, 0.f), nb);
  if (r > 0.f && fmaxf(rn.x, 4e-10f) * (1.f + fabsf(q)) < 400.f) {   // false for NaN
    if (t.x <= -1e-6f * (1.f + fabsf(q))) return 0;   // lambda = 0
    float2 lam = pair_mul(rn, t);
    if (lam.x < 0.f) lam = make_float2(0.f, 0.f);     // 1 + b d = 0 to within the pair's error
    if (lam.x < 31.9f) {
      const int k = poisson_screen(lam, philox((uint64_t)i, 0, ST_MOCK_COUNTS, (uint64_t)l, seed).w[0]);
      if (k >= 0) return k;
    }
  }
  return poisson_exact(r, d, b64, nbar64, i, l, seed);
}

// The paper's Gaussian noise: round((r Nbar)(1 + b d) + sqrt(r Nbar) z) clipped at 0.
__device__ __forceinline__ int gauss_count(float r, float d, double b, double nbar, long long i, int l,
                                           uint64_t seed) {
  const double rn = __dmul_rn((double)r, nbar);
  if (!(rn > 0.0)) return 0;
  const double m = __dmul_rn(rn, __dadd_rn(1.0, __dmul_rn(b, (double)d)));
  const P4 w = philox((uint64_t)i, 0, ST_MOCK_COUNTS, (uint64_t)l, seed);
  const double u1 = u52(w.w[0]), u2 = u52(w.w[1]);
  const double z = sqrt(-2.0 * log(u1)) * cos(__dmul_rn(2.0 * 3.141592653589793, u2));
  const double x = __dadd_rn(m, __dmul_rn(__dsqrt_rn(rn), z));
  return (int32_t)fmax(floor(__dadd_rn(x, 0.5)), 0.0);
}

// Counts of every subsample (noise 0: Poisson by inversion, noise 1: Gaussian),
// one voxel per thread, the subsamples in the inner loop so that the field is
// read once.  FP64 issue bounds any FP64 work here: 13.8 ms at 256^3 with six
// subsamples with every voxel searched in FP64, 1.72 ms with lambda in FP64 and
// the search in FP32 at the observed voxels only (FP64 pipe 77% busy), and
// 0.55 ms with lambda in FP32 pairs as well, 0.42 ms with the registers cut from 64 to
// 32 (56 bytes of spills) for seven blocks per SM instead of four (0.45 ms with six or
// eight): latency.
// Four voxels per thread hold 124 registers and two blocks per SM (0.92 ms); one
// response in flight per thread instead of four takes 0.70 ms.
// EXACT: the definition at every voxel.
template <int NOISE, bool EXACT>
__global__ void __launch_bounds__(256, 7) k_mock_counts(const float* __restrict__ delta, const float* __restrict__ R,
                                                        long long nv, int nsub, MockSub sub, uint64_t seed,
                                                        int32_t* __restrict__ out) {
  constexpr int G = 4;   // responses in flight per thread: most voxels only pass through
  const long long i = blockIdx.x * 256LL + threadIdx.x;
  if (i >= nv) return;
  const float d = delta[i];
  for (int l0 = 0; l0 < nsub; l0 += G) {
    float r[G];
#pragma unroll
    for (int g = 0; g < G; ++g) r[g] = l0 + g < nsub ? R[(l0 + g) * nv + i] : 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int l = l0 + g;
      if (l >= nsub) break;
      int c = 0;
      if constexpr (NOISE) c = gauss_count(r[g], d, sub.b[l], sub.nbar[l], i, l, seed);
      else if constexpr (EXACT) c = poisson_exact(r[g], d, sub.b[l], sub.nbar[l], i, l, seed);
      else if (!(r[g] == 0.f && isfinite(d)))   // lambda = 0 there
        c = poisson_count(r[g], d, sub.b2[l], sub.nbar2[l], sub.b[l], sub.nbar[l], i, l, seed);
      out[l * nv + i] = c;
    }
  }
}

struct RespArgs {
  int N, n_r, n_sub;
  double dx, half_box, thr_cos, r_max;
  double ax, ay, az;   // axis as given; normalised in the kernel
};

// R[l][i] = [cos(theta_i) >= 1 - 2 f_sky and r_i <= r_max] * table_l(r_i),
// the table sampled at r_j = j r_max / (n_r - 1) and interpolated linearly.
// V consecutive voxels of one z line per thread.  In half voxels the coordinates
// are odd integers, so 4 r^2 = S is an exact integer in FP32, S = N^2 mod 8 never
// holds (three odd squares are 3 mod 8) and r <= r_max is S < N^2; the FP32
// cosine is off by less than 1e-6 and decides the cap outside a margin of 1e-5.
// Values are computed as FP32 pairs (t = sqrt(S) (n_r - 1) / N, table entries split
// in two), off by less than 2^-41 of the larger table entry and 2^-43 t of the step
// between the two (in the segment that holds t: the next one's slope is another),
// and kept where that cannot change their rounding to FP32; the rest takes the FP64
// steps that define the response.  With every voxel in FP64 the kernel was bound by FP64 issue: 2.59
// ms at 256^3 with six subsamples, 0.76 ms with FP64 inside the survey only, now
// 0.146 ms.
__device__ __noinline__ float response_exact(const RespArgs& a, int ix, int iy, int iz, double ux, double uy, double uz,
                                             const double* __restrict__ tl) {
  const double nr1 = (double)(a.n_r - 1);
  const double x = __dsub_rn(__dmul_rn((double)ix + 0.5, a.dx), a.half_box);
  const double y = __dsub_rn(__dmul_rn((double)iy + 0.5, a.dx), a.half_box);
  const double z = __dsub_rn(__dmul_rn((double)iz + 0.5, a.dx), a.half_box);
  const double r = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z)));
  const double proj = __dadd_rn(__dadd_rn(__dmul_rn(ux, x), __dmul_rn(uy, y)), __dmul_rn(uz, z));
  const double cos_t = r > 0.0 ? __ddiv_rn(proj, r) : 1.0;
  if (!(cos_t >= a.thr_cos && r <= a.r_max)) return 0.f;
  const double t = fmin(__dmul_rn(__ddiv_rn(r, a.r_max), nr1), nr1);
  const double jf = fmin(floor(t), nr1 - 1.0);
  const int j = (int)jf;
  const double w = __dsub_rn(t, jf);
  return __double2float_rn(__dadd_rn(__dmul_rn(tl[j], __dsub_rn(1.0, w)), __dmul_rn(tl[j + 1], w)));
}

// the table as FP32 pairs, and the unit axis
__global__ void k_mock_table(RespArgs a, const double* __restrict__ table, long long n, float2* __restrict__ out,
                             double* __restrict__ axis) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i == 0) {
    const double nrm = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(a.ax, a.ax), __dmul_rn(a.ay, a.ay)),
                                            __dmul_rn(a.az, a.az)));
    axis[0] = __ddiv_rn(a.ax, nrm);
    axis[1] = __ddiv_rn(a.ay, nrm);
    axis[2] = __ddiv_rn(a.az, nrm);
  }
  if (i >= n) return;
  const float h = (float)table[i];
  out[i] = make_float2(h, (float)(table[i] - (double)h));
}

// EXACT: the FP64 steps for every voxel (boxes whose squared lengths overflow FP64 or
// lose bits there, which decides the radius cut).
template <int V, bool EXACT>
__global__ void __launch_bounds__(256, 4) k_mock_response(RespArgs a, float2 c2, const double* __restrict__ axis,
                                                          const double* __restrict__ table,
                                                          const float2* __restrict__ table2, float* __restrict__ R) {
  const float uxf = (float)axis[0], uyf = (float)axis[1], uzf = (float)axis[2];
  const float cos_out = (float)a.thr_cos - 1e-5f, cos_in = (float)a.thr_cos + 1e-5f;
  const float jmax = (float)(a.n_r - 2);
  // the pair and the FP64 t, each within 2^-44 t, may lie on two sides of a radius: undecided
  const float w_lo = 0x1p-42f * (float)a.n_r, w_hi = 1.f - w_lo;
  const long long nv = (long long)a.N * a.N * a.N;
  const long long i = (blockIdx.x * 256LL + threadIdx.x) * V;
  if (i < nv) {
    const int iz0 = (int)(i % a.N);
    const int iy = (int)((i / a.N) % a.N);
    const int ix = (int)(i / ((long long)a.N * a.N));
    const int x = 2 * ix + 1 - a.N, y = 2 * iy + 1 - a.N;
    const float pxy = uxf * (float)x + uyf * (float)y;
    int state[V];            // 0 outside, 1 inside, 2 undecided
    int jt[V];
    float2 w[V];
    bool any = false;
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const int z = 2 * (iz0 + e) + 1 - a.N;
      const int S = x * x + y * y + z * z;
      const float Sf = (float)S;
      const float cf = (pxy + uzf * (float)z) * rsqrtf(Sf);
      state[e] = 0;
      jt[e] = 0;
      w[e] = make_float2(0.f, 0.f);
      if constexpr (EXACT) {
        any = true;
        state[e] = 2;
        continue;
      }
      if (S >= a.N * a.N || cf < cos_out) continue;
      any = true;
      if (!(cf > cos_in)) {
        state[e] = 2;
        continue;
      }
      state[e] = 1;
      const float s = sqrtf(Sf);
      const float2 s2 = pair_quick(s, __fdividef(__fmaf_rn(-s, s, Sf), 2.f * s));
      const float2 t = pair_mul(s2, c2);
      // the first part may have been rounded up to a radius of the table that t does not reach
      const float fl = floorf(t.x);
      const float j = fminf(fmaxf(t.y < 0.f && t.x == fl ? fl - 1.f : fl, 0.f), jmax);
      jt[e] = (int)j;
      w[e] = pair_sum(t.x - j, t.y);   // t.x - j is exact
      if (w[e].x < w_lo || w[e].x >= w_hi) state[e] = 2;
    }
    for (int l = 0; l < a.n_sub; ++l) {
      float v[V];
#pragma unroll
      for (int e = 0; e < V; ++e) v[e] = 0.f;
      if (any) {
        const double* tl = table + (long long)l * a.n_r;
        const float2* tl2 = table2 + (long long)l * a.n_r;
#pragma unroll
        for (int e = 0; e < V; ++e) {
          if (state[e] == 0) continue;
          bool ok = false;
          if (state[e] == 1) {
            const float2 t0 = __ldg(tl2 + jt[e]), t1 = __ldg(tl2 + jt[e] + 1);
            const float2 f = pair_add(t0, pair_mul(w[e], pair_add(t1, make_float2(-t0.x, -t0.y))));
            const float big = fmaxf(t0.x, t1.x);
            const float tol = 0x1p-41f * big + 0x1p-43f * ((float)(jt[e] + 1) * fabsf(t1.x - t0.x));
            // far from FP32's smallest and largest values, and rounded the same anywhere within tol
            ok = (big == 0.f || (big > 1e-20f && big < 1e30f)) && __fadd_rn(f.x, f.y + tol) == f.x &&
                 __fadd_rn(f.x, f.y - tol) == f.x;
            v[e] = f.x;
          }
          if (!ok) v[e] = response_exact(a, ix, iy, iz0 + e, axis[0], axis[1], axis[2], tl);
        }
      }
      float* Rl = R + (long long)l * nv + i;
      if constexpr (V == 4) *reinterpret_cast<float4*>(Rl) = make_float4(v[0], v[1], v[2], v[3]);
      else *Rl = v[0];
    }
  }
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// ---------------------------------------------------------------- host: Schechter tables
// Gauss-Legendre nodes and weights on [-1, 1] (Newton iteration on P_n from
// the usual cosine starting points)
struct Gauss {
  static constexpr int n = 16;
  double x[n], w[n];
  Gauss() {
    for (int i = 0; i < (n + 1) / 2; ++i) {
      double z = std::cos(M_PI * (i + 0.75) / (n + 0.5)), pp = 1.0;
      for (int it = 0; it < 100; ++it) {
        double p1 = 1.0, p2 = 0.0;
        for (int j = 1; j <= n; ++j) {
          const double p3 = p2;
          p2 = p1;
          p1 = ((2.0 * j - 1.0) * z * p2 - (j - 1.0) * p3) / j;
        }
        pp = n * (z * p1 - p2) / (z * z - 1.0);
        const double dz = p1 / pp;
        z -= dz;
        if (std::fabs(dz) < 1e-16) break;
      }
      x[i] = -z;
      x[n - 1 - i] = z;
      w[i] = w[n - 1 - i] = 2.0 / ((1.0 - z * z) * pp * pp);
    }
  }
  // composite rule over [a, b] with pieces no wider than h
  template <class F>
  double integrate(F f, double a, double b, double h) const {
    if (!(b > a)) return 0.0;
    const int m = std::max(1, (int)std::ceil((b - a) / h));
    const double step = (b - a) / m;
    double s = 0.0;
    for (int k = 0; k < m; ++k) {
      const double c = a + (k + 0.5) * step, hw = 0.5 * step;
      for (int i = 0; i < n; ++i) s += hw * w[i] * f(c + hw * x[i]);
    }
    return s;
  }
};

struct Schechter {
  double M_star, alpha, m_bright, m_faint, omega_m;
  const Gauss& g;
  double phi(double M) const {
    const double x = std::pow(10.0, 0.4 * (M_star - M));
    return 0.4 * std::log(10.0) * std::pow(x, alpha + 1.0) * std::exp(-x);
  }
  double integral(double lo, double hi) const {
    return g.integrate([this](double M) { return phi(M); }, lo, hi, 0.05);
  }
  double hubble(double z) const { return std::sqrt(omega_m * (1.0 + z) * (1.0 + z) * (1.0 + z) + 1.0 - omega_m); }
  double comoving(double z) const {
    return 2997.92458 * g.integrate([this](double t) { return 1.0 / hubble(t); }, 0.0, z, 0.01);
  }
  double redshift(double r) const {   // Newton on D_C(z) = r
    double z = r / 2997.92458;
    for (int it = 0; it < 30; ++it) {
      const double dz = (comoving(z) - r) * hubble(z) / 2997.92458;
      z -= dz;
      if (std::fabs(dz) < 1e-15 * (1.0 + z)) break;
    }
    return z;
  }
};

}  // namespace
}  // namespace bps

using namespace bps;

extern "C" {

bps_status bps_schechter_tables(const bps_schechter* s, int n_sub, const double* M_edges, double r_max, int n_r,
                                double* table, double* nbar_rel) {
  if (!s || !M_edges || !table || n_sub < 1 || n_sub > MAXS || n_r < 2 || !(r_max > 0.0)) {
    set_last_error("bps_schechter_tables: bad arguments");
    return BPS_EINVAL;
  }
  for (int l = 0; l < n_sub; ++l)
    if (!(M_edges[l + 1] > M_edges[l])) {
      set_last_error("bps_schechter_tables: magnitude edges must increase (brightest first)");
      return BPS_EINVAL;
    }
  if (!(s->omega_m > 0.0 && s->omega_m <= 1.0) || !(s->m_faint > s->m_bright)) {
    set_last_error("bps_schechter_tables: need 0 < omega_m <= 1 and m_faint > m_bright");
    return BPS_EINVAL;
  }
  static const Gauss g;
  const Schechter sc{s->M_star, s->alpha, s->m_bright, s->m_faint, s->omega_m, g};
  // distance moduli of the sample radii (shared by all subsamples)
  std::vector<double> mu(n_r, 0.0);
  for (int j = 1; j < n_r; ++j) {
    const double r = j * (r_max / (n_r - 1));
    mu[j] = 5.0 * std::log10((1.0 + sc.redshift(r)) * r) + 25.0;
  }
  for (int l = 0; l < n_sub; ++l) {
    const double norm = sc.integral(M_edges[l], M_edges[l + 1]);
    if (nbar_rel) nbar_rel[l] = norm;
    table[(size_t)l * n_r] = 0.0;
    for (int j = 1; j < n_r; ++j) {
      const double lo = std::max(M_edges[l], s->m_bright - mu[j]);
      const double hi = std::min(M_edges[l + 1], s->m_faint - mu[j]);
      table[(size_t)l * n_r + j] = hi > lo ? sc.integral(lo, hi) / norm : 0.0;
    }
  }
  return BPS_OK;
}

bps_status bps_bias_law(int n, const double* M, double b_star, double M_star, double a, double b, double c,
                        double* b_out) {
  if (n < 0 || (n > 0 && (!M || !b_out))) {
    set_last_error("bps_bias_law: bad arguments");
    return BPS_EINVAL;
  }
  for (int l = 0; l < n; ++l) b_out[l] = b_star * (a + b * std::pow(10.0, 0.4 * (M_star - M[l])) + c * (M[l] - M_star));
  return BPS_OK;
}

}  // extern "C"

// ---- context-bound mock calls (they use the context's transforms and buffers)
namespace bps {

bps_status mock_field(const MockView& v, uint64_t seed, const double* P_n2, float* delta_dev) {
  const int N = v.N;
  const size_t nt = (size_t)3 * (N / 2) * (N / 2) + 1;
  const double vc = std::pow(v.box / N, 3);
  const std::vector<double> P(P_n2, P_n2 + nt);   // pageable: the copy below has left it when it returns
  for (size_t i = 1; i < nt; ++i)
    if (!(P[i] >= 0.0) || !std::isfinite(P[i])) {
      set_last_error("bps_mock_field: the spectrum must be finite and non-negative");
      return BPS_EINVAL;
    }
  double* dP = nullptr;   // the spectrum, then the FP32 amplitudes
  bps_status st = v.get_scratch(nt * (sizeof(double) + sizeof(float)), (void**)&dP);
  if (st != BPS_OK) return st;
  float* damp = reinterpret_cast<float*>(dP + nt);
  cudaStream_t s = v.stream;
  if (cudaMemcpyAsync(dP, P.data(), nt * sizeof(double), cudaMemcpyHostToDevice, s) != cudaSuccess) {
    set_last_error("bps_mock_field: copy of the spectrum failed");
    return BPS_ECUDA;
  }
  // the normals are drawn inside the first z pass, and the amplitudes applied
  // between the two x transforms of one x pass
  k_mock_amp<<<(unsigned)((nt + 255) / 256), 256, 0, s>>>(dP, (int)nt, vc, damp);
  v.pt->z_mock(*v.f, seed, ST_MOCK_FIELD, v.f->W, s);
  v.pt->y_fwd(*v.f, BUF_W, 1, s);
  v.pt->x_amp(*v.f, damp, s);
  v.pt->y_inv(*v.f, BUF_W, 1, s);
  v.pt->z_c2r(*v.f, v.f->W, delta_dev, s);
  *v.launches += 6;
  if (cudaGetLastError() != cudaSuccess) {
    set_last_error("bps_mock_field: kernel launch failed");
    return BPS_ECUDA;
  }
  return BPS_OK;
}

bps_status mock_counts(const MockView& v, uint64_t seed, const float* delta_dev, const float* R_dev, const double* b,
                       const double* nbar, int noise, int32_t* counts_dev) {
  MockSub sub{};
  // whether the FP32 parts of every b and Nbar hold 46 bits, and b delta cannot overflow FP64
  bool plain = true;
  auto ordinary = [](double x) { return x == 0.0 || (std::fabs(x) > 1e-20 && std::fabs(x) < 1e20); };
  for (int l = 0; l < v.n_sub; ++l) {
    if (!std::isfinite(b[l]) || !(nbar[l] >= 0.0) || !std::isfinite(nbar[l])) {
      set_last_error("bps_mock_counts: b must be finite and nbar non-negative");
      return BPS_EINVAL;
    }
    sub.b[l] = b[l];
    sub.nbar[l] = nbar[l];
    plain = plain && ordinary(b[l]) && ordinary(nbar[l]);
    auto split = [](double x) {
      const float h = (float)x;
      return make_float2(h, (float)(x - (double)h));
    };
    sub.b2[l] = split(b[l]);
    sub.nbar2[l] = split(nbar[l]);
  }
  const long long nv = (long long)v.N * v.N * v.N;
  // one block per 256 voxels: the hardware's block order balances the observed
  // region, which a fixed stride over few blocks leaves to some of them
  const unsigned blocks = (unsigned)((nv + 255) / 256);
  auto* k = noise ? k_mock_counts<1, false> : plain ? k_mock_counts<0, false> : k_mock_counts<0, true>;
  k<<<blocks, 256, 0, v.stream>>>(delta_dev, R_dev, nv, v.n_sub, sub, seed, counts_dev);
  *v.launches += 1;
  if (cudaGetLastError() != cudaSuccess) {
    set_last_error("bps_mock_counts: kernel launch failed");
    return BPS_ECUDA;
  }
  return BPS_OK;
}

bps_status mock_response(const MockView& v, double f_sky, const double* axis, int n_r, const double* table,
                         float* R_dev) {
  if (!(f_sky > 0.0 && f_sky <= 1.0) || n_r < 2 || n_r > (1 << 20) || !axis ||
      !(axis[0] * axis[0] + axis[1] * axis[1] + axis[2] * axis[2] > 0.0)) {
    set_last_error("bps_mock_response: need 0 < f_sky <= 1, 2 <= n_r <= 2^20 and a nonzero axis");
    return BPS_EINVAL;
  }
  const size_t tn = (size_t)v.n_sub * n_r;
  for (size_t i = 0; i < tn; ++i)
    if (!(table[i] >= 0.0) || !std::isfinite(table[i])) {
      set_last_error("bps_mock_response: the selection table must be finite and non-negative");
      return BPS_EINVAL;
    }
  double* dt = nullptr;
  bps_status st = v.get_scratch((tn + 3) * sizeof(double) + tn * sizeof(float2), (void**)&dt);
  if (st != BPS_OK) return st;
  if (cudaMemcpyAsync(dt, table, tn * sizeof(double), cudaMemcpyHostToDevice, v.stream) != cudaSuccess) {
    set_last_error("bps_mock_response: copy of the selection table failed");
    return BPS_ECUDA;
  }
  RespArgs a;
  a.N = v.N;
  a.n_r = n_r;
  a.n_sub = v.n_sub;
  a.dx = v.box / v.N;
  a.half_box = v.box / 2.0;
  a.thr_cos = 1.0 - 2.0 * f_sky;
  a.r_max = v.box / 2.0;
  a.ax = axis[0];
  a.ay = axis[1];
  a.az = axis[2];
  double* axis_dev = dt + tn;
  float2* dt2 = reinterpret_cast<float2*>(dt + tn + 3);
  k_mock_table<<<(unsigned)((tn + 255) / 256), 256, 0, v.stream>>>(a, dt, (long long)tn, dt2, axis_dev);
  const double c = (double)(n_r - 1) / (double)v.N;
  const float2 c2 = make_float2((float)c, (float)(c - (double)(float)c));
  const long long nv = (long long)v.N * v.N * v.N;
  // 16-byte stores where R starts on a 16-byte boundary (every subsample then
  // does: N^3 is a multiple of 4); one block per 1024 voxels, so that the
  // hardware's block order balances the observed region
  const unsigned blocks = (unsigned)((nv + 255) / 256), blocks4 = (unsigned)((nv / 4 + 255) / 256);
  cudaStream_t s = v.stream;
  if (!(v.box > 1e-120 && v.box < 1e120))
    k_mock_response<1, true><<<blocks, 256, 0, s>>>(a, c2, axis_dev, dt, dt2, R_dev);
  else if (aligned16(R_dev))
    k_mock_response<4, false><<<blocks4, 256, 0, s>>>(a, c2, axis_dev, dt, dt2, R_dev);
  else
    k_mock_response<1, false><<<blocks, 256, 0, s>>>(a, c2, axis_dev, dt, dt2, R_dev);
  *v.launches += 2;
  if (cudaGetLastError() != cudaSuccess) {
    set_last_error("bps_mock_response: kernel launch failed");
    return BPS_ECUDA;
  }
  return BPS_OK;
}

}  // namespace bps
