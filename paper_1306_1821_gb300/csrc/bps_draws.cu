// Scalar stages of the multiple-block scan, run on the device so that a Gibbs
// iteration needs no host round trip: step size and Metropolis decisions of the
// HMC moves (Sec. 4.1, Eq. acceptance_rule), the chi^2 draw of the power
// spectrum (Sec. 4.2), the normal bias draw (Sec. 3.5, App. B), the GIG draw of
// the normalisations (Sec. 3.6, App. A) and the HMC in ln P of the jump
// (Sec. 4.3, App. C).  All decisions are taken in FP64 from Philox4x64-10
// words at fixed counters.
#include <math.h>

#include "bps_internal.h"
#include "bps_passes.cuh"

namespace bps {

constexpr int MAX_ATTEMPTS = 64;

// the scalar arguments of chain `ch` of a batch (blockIdx.y)
__device__ __forceinline__ ScalarArgs chain_args(ScalarArgs a, int ch) {
  a.ds += ch;
  a.part += ch * a.cstride;
  return a;
}

// Deterministic sum of n partials (stride 1) by one block of 256 threads;
// the value is valid in thread 0.
__device__ double sum_partials(const double* p, int n, double* sh) {
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) v += p[i];
  return block_sum<256>(v, sh);
}

// ------------------------------------------------------------------ HMC move
// The scalar kernels of a Gibbs iteration are chains of FP64 operations on a part
// whose FP64 pipe is 1/64 of the FP32 one: a division or square root takes most
// of a microsecond, a logarithm or exponential more.  So independent ones go to
// different warps, variates that wait for nothing are drawn while the sums are
// read, and small kernels that only consume what another one finishes are that
// one's last block.

// H = (1/2N^3) sum w (|p|^2/M + |delta|^2/lambda) + (1/2) sum (a delta^2 - 2 c delta)
// The eight sums of a move, one block each (on different SMs: each sum is a
// chain of FP64 additions), into the chain state's scratch: K0, E0, L0, K1, E1,
// L1, G0, G1 (the kinetic, prior and likelihood energies at the start and the
// end, and the two force norms of the leapfrog energy identity).  The last block
// to finish takes the Metropolis decision.
__global__ void k_move_end(ScalarArgs a0, int r_init, int r_lik0, int r_final, int r_lik1, int nx, int nz,
                           int advance) {
  await_previous();
  const ScalarArgs a = chain_args(a0, blockIdx.y);
  __shared__ double sh[32];
  DevState* ds = a.ds;
  const double h = 0.5 * a.inv_nv;
  const double* p = nullptr;
  int n = nx;
  double scale = h;
  switch (blockIdx.x) {
    case 0: p = a.part + r_init; break;
    case 1: p = a.part + r_init + a.stride; break;
    case 2: p = a.part + r_lik0; n = nz; scale = 1.0; break;
    case 3: p = a.part + r_final; break;
    case 4: p = a.part + r_final + a.stride; break;
    case 5: p = a.part + r_lik1; n = nz; scale = 1.0; break;
    case 6: p = a.part + r_init + 2 * a.stride; scale = a.inv_nv; break;
    default: p = a.part + r_final + 2 * a.stride; scale = a.inv_nv; break;
  }
  const double s = sum_partials(p, n, sh);
  if (threadIdx.x == 0) {
    ds->scratch[blockIdx.x] = s * scale;
    __threadfence();
    if (atomicAdd(&ds->mdone, 1) != (int)gridDim.x - 1) return;
    __threadfence();
    ds->mdone = 0;
    const double K0 = __ldcg(ds->scratch + 0), E0 = __ldcg(ds->scratch + 1), L0 = __ldcg(ds->scratch + 2);
    const double K1 = __ldcg(ds->scratch + 3), E1 = __ldcg(ds->scratch + 4), L1 = __ldcg(ds->scratch + 5);
    const double G0 = __ldcg(ds->scratch + 6), G1 = __ldcg(ds->scratch + 7);
    const double H0 = K0 + E0 + L0, H1 = K1 + E1 + L1;
    // H(end) - H(start) of Eq. acceptance_rule.  The potential of the density
    // move (Eq. Wiener_Posterior_psi with fixed P, b, Nbar) is exactly quadratic
    // in delta, and for kick-drift-kick leapfrog on a quadratic potential the
    // energy change telescopes exactly: each step changes H by
    // (eps^2/8)(g_{n+1}^T M^-1 g_{n+1} - g_n^T M^-1 g_n), so over the whole
    // trajectory dH = (eps^2/8)(g_L^T M^-1 g_L - g_0^T M^-1 g_0).  Both norms are
    // O(N^3) and their difference is multiplied by eps^2/8, so the FP32 terms
    // carry ~1e-8 into dH, where the difference H1 - H0 of two ~1e7-sized
    // energies carries the FP32 error of the transformed field (~1e-3 at
    // 256^3).  eps is the FP32 step the passes applied.  H0 and H1 are kept
    // for the finiteness check and for inspection.
    const double e32 = (double)(float)ds->eps;
    const double dH = 0.125 * e32 * e32 * (G1 - G0);
    ds->H0 = H0;
    ds->H1 = H1;
    ds->dH = dH;
    ds->lik0 = L0;
    ds->lik1 = L1;
    int acc = 0;
    if (!isfinite(dH) || !isfinite(H0) || !isfinite(H1)) {
      ds->status |= ST_NONFINITE;
    } else {
      acc = ds->log_u < -dH;        // Eq. acceptance_rule, FP64
    }
    ds->accepted = acc;
    if (acc) {
      ds->cur = 1 - ds->cur;
      ds->n_accepted += 1;
    }
    ds->n_moves += 1;
    if (advance) ds->iteration += 1;
  }
}

// ------------------------------------------------------------------ P draw
// Gamma(shape) by Marsaglia & Tsang (ACM TOMS 2000); attempt j of bin m reads
// Philox block (m, iteration, ST_POWER, j): words 0,1 -> normal, word 2 -> uniform;
// shape < 1 uses Gamma(shape + 1) U^(1/shape) with U from word 3 of attempt 0.
// Called by all 32 lanes of one warp (identical arguments): lane q makes the
// attempts q and 32 + q, the first accepted one counts; every lane returns it.
__device__ double gamma_mt(double shape, uint64_t seed, uint64_t it, int m, int* fail) {
  const bool boost = shape < 1.0;
  const double aa = boost ? shape + 1.0 : shape;
  const double d = aa - 1.0 / 3.0;
  const double c = 1.0 / sqrt(9.0 * d);
  const int lane = threadIdx.x & 31;
  double val = d;
  bool ok = false;
  for (int j0 = 0; j0 < MAX_ATTEMPTS && !ok; j0 += 32) {
    P4 r = philox((uint64_t)m, it, ST_POWER, (uint64_t)(j0 + lane), seed);
    const double z = normal64(r.w[0], r.w[1]);
    const double t = 1.0 + c * z;
    bool acc = false;
    double mine = 0.0;
    if (t > 0.0) {
      const double v = t * t * t;
      const double u = u52(r.w[2]);
      acc = log(u) < 0.5 * z * z + d - d * v + d * log(v);
      mine = d * v;
    }
    const unsigned who = __ballot_sync(0xffffffffu, acc);
    if (who) {
      val = __shfl_sync(0xffffffffu, mine, __ffs((int)who) - 1);
      ok = true;
    }
  }
  if (!ok) *fail = 1;
  if (boost) {
    P4 r = philox((uint64_t)m, it, ST_POWER, 0, seed);
    val *= exp(log(u52(r.w[3])) / shape);
  }
  return val;
}

// block m: sigma_m = (V_cell/N^3) sum_{k in m} w |delta_k|^2; then (draw) P_m = sigma_m / x,
// x ~ chi^2_beta = 2 Gamma(beta/2), beta = n_m + 2 alpha - 2 (Sec. 4.2, Eq. XI_SQUARE); then
// (jump) the start of the jump's HMC in theta = ln P with the whitened field fixed
// (Sec. 4.3, App. C), whose mass mu_m = max(1, abar P_ref_m sigma_m / (4 V_cell P_m)) is
// built from the whitened field and a fixed reference spectrum, never from the current P.
// Eight warps sum; a ninth draws the Gamma variate and a tenth the jump's normal
// meanwhile (neither depends on the sum).
// jump = 2: the jump directly follows this iteration's HMC move, so after an accepted
// move its first gradient can take the move's last force.
__global__ void __launch_bounds__(320) k_power(ScalarArgs a0, int region, int nx, int draw, int jump) {
  await_previous();
  const ScalarArgs a = chain_args(a0, blockIdx.y);
  __shared__ double sh[32];
  __shared__ double s_gamma, s_z, s_sigma, s_P;
  __shared__ int s_fail;
  DevState* ds = a.ds;
  const int m = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  double v = 0.0;
  if (warp < 8) {
    const double* p = a.part + region + (size_t)m * a.stride;
    for (int i = t; i < nx; i += 256) v += p[i];
    v = warp_sum(v);
    if (lane == 0) sh[warp] = v;
  } else if (warp == 8) {
    if (draw) {
      int fail = 0;
      const double g = gamma_mt(0.5 * (ds->nmodes[m] + 2.0 * a.alpha - 2.0), ds->seed, ds->iteration, m, &fail);
      if (lane == 0) {
        s_gamma = g;
        s_fail = fail;
      }
    }
  } else if (jump) {
    const P4 r = philox((uint64_t)m, ds->iteration, ST_JUMP_MOM, 0, ds->seed);
    const double z = normal64(r.w[0], r.w[1]);
    if (lane == 0) s_z = z;
  }
  __syncthreads();
  if (t == 0) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += sh[i];
    const double sigma = s * ds->vc * a.inv_nv;
    ds->sigma[m] = sigma;
    double P = ds->P[m];
    if (draw) {
      if (s_fail || !(sigma > 0.0)) {
        atomicOr(&ds->status, ST_DRAW_FAIL);
      } else {
        P = sigma / (2.0 * s_gamma);
        ds->P[m] = P;
      }
    }
    s_sigma = sigma;
    s_P = P;
  }
  if (!jump) return;
  __syncthreads();
  if (lane == 0) {
    if (warp == 0 || warp == 1) {
      const double mu = fmax(1.0, ds->abar * ds->P_ref[m] * s_sigma / (4.0 * ds->vc * s_P));
      if (warp == 0) ds->rho[m] = sqrt(mu) * s_z;
      else ds->inv_mu[m] = 1.0 / mu;
    } else if (warp == 2) {
      const double th = log(s_P);
      ds->th[m] = th;
      ds->th0[m] = th;
      ds->js[m] = 1.f;
    } else if (warp == 3 && m == 0) {
      ds->jreuse = jump == 2 && ds->accepted;
      const P4 r = philox(0, ds->iteration, ST_JUMP, 0, ds->seed);
      ds->jeps = a.jeps_max * u52(r.w[0]);
      ds->jlog_u = log(u52(r.w[1]));
      ds->jaccepted = 0;
    }
  }
}

// ------------------------------------------------------------------ GIG draw
// Density ~ x^(p-1) exp(-(A x + B/x)/2) (Eq. GIG_post).  With eta = sqrt(B/A),
// omega = sqrt(A B), y = x/eta (p >= 0) or eta/x (p < 0) has density
// h(y) ~ y^(lam-1) exp(-omega (y + 1/y)/2), lam = |p|; sampled by the
// ratio-of-uniforms method with mode shift (Kinderman & Monahan 1977), the
// bounding rectangle from the extremes of (y - m) sqrt(h(y)), everything in log
// space about the mode m.  ln h(m + d) - ln h(m):
__device__ double gig_logh(double d, double lam, double om, double m) {
  return (lam - 1.0) * log1p(d / m) - 0.5 * om * d * (1.0 - 1.0 / ((m + d) * m));
}

// Called by all 32 lanes of one warp (identical arguments); every lane returns
// the same draw.  lu, u, w: ln u, u and the second uniform of each of the 64
// attempts (shared memory).
//
// The extremes: d/dy ln((y - m) sqrt(h)) = 0, with the mode's equation
// (lam - 1) m = (omega / 2)(m^2 - 1), is (omega / 4)(y - m)^2 (y + 1/m) = y^2, or
// G(d) = d -+ 2 y / sqrt(omega (y + 1/m)) = 0 with y = m + d, one root on either
// side of the mode.  G rises through its root, nearly linearly for the peaked
// densities of a survey: Newton's method within a bracket, the upper root in the
// lower half of the warp and the lower root in the upper half.  (y - m) sqrt(h) is
// stationary there, so a relative step of 1e-9 leaves it exact to FP64.  A search
// by 32-point section took 12 to 16 rounds for each root, two thirds of the 66 to
// 75 us of this kernel.
__device__ double gig_draw(double p, double A, double B, const double* lu, const double* u, const double* w,
                           int* fail) {
  const int lane = threadIdx.x & 31;
  const double lam = fabs(p);
  const double om = sqrt(A * B);
  const double eta = sqrt(B / A);
  const double q = lam - 1.0;
  const double sq = sqrt(q * q + om * om);
  const double m = q >= 0.0 ? (q + sq) / om : om / (sq - q);
  const double im = 1.0 / m;
  const bool up = lane < 16;
  double lo = up ? 0.0 : -m, hi = up ? 1.7e308 : 0.0;
  double d = 2.0 * m * rsqrt(om * (m + im));
  if (!up) d = d < m ? -d : -0.5 * m;
  for (int i = 0; i < 200; ++i) {
    const double y = m + d;
    const double r = rsqrt(om * (y + im));
    const double f = 2.0 * y * r;
    const double G = up ? d - f : d + f;
    const double df = 2.0 * r - y * om * r * r * r;
    if (G < 0.0) lo = d;
    else hi = d;
    double nd = d - G / (up ? 1.0 - df : 1.0 + df);
    if (!(nd > lo && nd < hi)) nd = up && hi > 1e308 ? 2.0 * d : 0.5 * (lo + hi);
    const bool done = !(fabs(nd - d) > 1e-9 * fabs(d));
    d = nd;
    if (__all_sync(0xffffffffu, done)) break;
  }
  const double ext = m + d > 0.0 ? d * exp(0.5 * gig_logh(d, lam, om, m)) : -m;
  const double vp = __shfl_sync(0xffffffffu, ext, 0), vm = __shfl_sync(0xffffffffu, ext, 16);
  double y = m;
  bool ok = false;
  for (int j0 = 0; j0 < MAX_ATTEMPTS && !ok; j0 += 32) {   // lane q makes the attempts q and 32 + q
    const int j = j0 + lane;
    const double dd = (vm + (vp - vm) * w[j]) / u[j];
    const bool acc = dd + m > 0.0 && 2.0 * lu[j] <= gig_logh(dd, lam, om, m);
    const unsigned who = __ballot_sync(0xffffffffu, acc);
    if (who) {
      y = m + __shfl_sync(0xffffffffu, dd, __ffs((int)who) - 1);
      ok = true;
    }
  }
  if (!ok) *fail = 1;
  return p >= 0.0 ? eta * y : eta / y;
}

// block l: S1 = sum N delta, S2 = sum R delta, S3 = sum R delta^2; then
// b_l ~ N(D/C, 1/C), C = Nbar S3, D = S1 - Nbar S2 (Sec. 3.5, App. B; skipped for
// the fixed index) and Nbar_l ~ GIG(1 - N_obs/2, sum R + 2 b S2 + b^2 S3, sum N^2/R).
// Eight warps sum the three quantities together; a ninth draws the bias normal and
// two more the uniforms of the GIG attempts (attempt j reads Philox block (l,
// iteration, ST_NBAR, j): word 0 gives u, word 1 the second uniform).
// 66-75 us a launch with the section search and serial attempts, now 17-20 us.
__global__ void __launch_bounds__(352) k_bias_nbar(ScalarArgs a0, int region, int nz) {
  await_previous();
  const ScalarArgs a = chain_args(a0, blockIdx.y);
  __shared__ double sh[3][8];
  __shared__ double s_S[3], s_z, s_lu[MAX_ATTEMPTS], s_u[MAX_ATTEMPTS], s_w[MAX_ATTEMPTS];
  DevState* ds = a.ds;
  const int l = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  if (l >= ds->nsub) return;
  const uint64_t it = ds->iteration;
  if (warp < 8) {
    const double* p = a.part + region + (size_t)3 * l * a.stride;
    double v0 = 0.0, v1 = 0.0, v2 = 0.0;
    for (int i = t; i < nz; i += 256) {
      v0 += p[i];
      v1 += p[a.stride + i];
      v2 += p[2 * (size_t)a.stride + i];
    }
    v0 = warp_sum(v0);
    v1 = warp_sum(v1);
    v2 = warp_sum(v2);
    if (lane == 0) {
      sh[0][warp] = v0;
      sh[1][warp] = v1;
      sh[2][warp] = v2;
    }
  } else if (warp == 8) {
    const P4 r = philox((uint64_t)l, it, ST_BIAS, 0, ds->seed);
    const double z = normal64(r.w[0], r.w[1]);
    if (lane == 0) s_z = z;
  } else {
    const int j = (warp - 9) * 32 + lane;
    const P4 r = philox((uint64_t)l, it, ST_NBAR, (uint64_t)j, ds->seed);
    const double u = u52(r.w[0]);
    s_u[j] = u;
    s_w[j] = u52(r.w[1]);
    s_lu[j] = log(u);
  }
  __syncthreads();
  if (warp != 0) return;
  if (lane < 3) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += sh[lane][i];
    s_S[lane] = s;
    ds->sums[l][lane] = s;
  }
  __syncwarp();
  const double S0 = s_S[0], S1 = s_S[1], S2 = s_S[2];
  double b = ds->b[l];
  const double nb = ds->nbar[l];
  int fail = 0;
  if (l != a.fixed_bias) {
    const double C = nb * S2;
    const double D = S0 - nb * S1;
    if (C > 0.0) b = D / C + s_z / sqrt(C);
    else fail = 1;
  }
  const double A = ds->sumR[l] + 2.0 * b * S1 + b * b * S2;
  const double p = 1.0 - 0.5 * ds->nobs[l];
  double x = nb;
  if (A > 0.0 && ds->sumB[l] > 0.0) x = gig_draw(p, A, ds->sumB[l], s_lu, s_u, s_w, &fail);
  else fail = 1;
  if (lane == 0) {
    if (fail || !isfinite(b) || !isfinite(x)) {
      atomicOr(&ds->status, ST_DRAW_FAIL);
    } else {
      ds->b[l] = b;
      ds->nbar[l] = x;
    }
  }
}

// ------------------------------------------------------------------ survey commit
// Activates a survey uploaded into data slot `slot`: sums the data kernel's
// per-block partials of each subsample (sum R, sum N^2/R, observed voxels,
// invalid voxels; 4 x nblk doubles per subsample) in a fixed order, and either
// writes the data constants of Secs. 3.5-3.6 and makes the slot active, or, for
// invalid data or a subsample without observed voxels, flags ST_BADDATA and
// keeps the previous slot.  One block per chain.
__global__ void k_commit_data(DevState* ds0, const double* part0, long long cstride, int nblk, int slot) {
  DevState* ds = ds0 + blockIdx.x;
  const double* part = part0 + blockIdx.x * cstride;
  __shared__ double s_v[MAXS][4];
  const int nsub = ds->nsub;
  // one warp per quantity (4 per subsample), lanes strided over the partials
  const int lane = threadIdx.x & 31;
  for (int q = threadIdx.x >> 5; q < 4 * nsub; q += blockDim.x >> 5) {
    double v = 0.0;
    for (int i = lane; i < nblk; i += 32) v += part[(size_t)q * nblk + i];
    v = warp_sum(v);
    if (lane == 0) s_v[q >> 2][q & 3] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    bool ok = true;
    for (int l = 0; l < nsub; ++l) ok = ok && s_v[l][3] == 0.0 && s_v[l][2] > 0.0;
    if (!ok) {
      atomicOr(&ds->status, ST_BADDATA);
    } else {
      for (int l = 0; l < nsub; ++l) {
        ds->sumR[l] = s_v[l][0];
        ds->sumB[l] = s_v[l][1];
        ds->nobs[l] = s_v[l][2];
      }
      ds->dslot = slot;
    }
  }
}

// ------------------------------------------------------------------ jump move
// HMC in theta = ln P with the whitened field fixed (Sec. 4.3, App. C), started by k_power.
//
// One leapfrog step after its gradient evaluation.  Block m < n_bins reduces the
// gradient d psi_J / d theta_m = (alpha - 1) + (1/2N^3) sum_{k in m} w Re(conj(g) delta)
// and updates bin m, which needs no other bin: J_FIRST half kick and drift (keeping
// the bin's starting energy), J_MID kick and drift, J_LAST half kick and final
// energy.  Block n_bins (J_FIRST and J_LAST) reduces the likelihood energy at theta.
// Only J_LAST joins the bins: its last block to finish sums the energies and takes
// the Metropolis decision.  The field scale sqrt(exp(theta) / P) is
// exp((theta - theta_0) / 2), one FP64 exponential instead of an exponential, a
// division and a square root.  9.0 us a launch at 128^3 with every step joined in
// its last block, now 5.9 us.
__global__ void __launch_bounds__(256) k_jump_step(ScalarArgs a0, int r_grad, int nx, int r_lik, int r_lik_move, int nz,
                                                   int kind) {
  await_previous();
  const ScalarArgs a = chain_args(a0, blockIdx.y);
  __shared__ double sh[32];
  __shared__ int s_last, s_acc;
  DevState* ds = a.ds;
  const int m = blockIdx.x, t = threadIdx.x;
  if (m < a.n_bins) {
    double rho = 0.0, th = 0.0, im = 0.0, th0 = 0.0, eps = 0.0;
    if (t == 0) {                 // in flight with the partial sums
      rho = ds->rho[m];
      th = ds->th[m];
      im = ds->inv_mu[m];
      th0 = ds->th0[m];
      eps = ds->jeps;
    }
    const double s = sum_partials(a.part + r_grad + (size_t)m * a.stride, nx, sh);
    if (t == 0) {
      const double g = (a.alpha - 1.0) + 0.5 * a.inv_nv * s;
      if (kind == J_FIRST) ds->je0[m] = 0.5 * rho * rho * im + (a.alpha - 1.0) * th;
      rho -= (kind == J_MID ? eps : 0.5 * eps) * g;
      ds->rho[m] = rho;
      if (kind == J_LAST) {
        ds->je1[m] = 0.5 * rho * rho * im + (a.alpha - 1.0) * th;
      } else {
        th += eps * rho * im;
        ds->th[m] = th;
        ds->js[m] = (float)exp(0.5 * (th - th0));
      }
    }
  } else {
    // a reused force stage left its likelihood partials where the move's last one wrote them
    const double s = sum_partials(a.part + (ds->jreuse ? r_lik_move : r_lik), nz, sh);
    if (t == 0) {
      if (kind == J_FIRST) {
        ds->jlik0 = s;
        ds->jreuse = 0;           // only the first gradient can reuse the move's force
      } else {
        ds->jlik1 = s;
      }
    }
  }
  if (kind != J_LAST) return;
  if (t == 0) {
    __threadfence();
    s_last = atomicAdd(&ds->jdone, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (t < 32) {
    double e0 = 0.0, e1 = 0.0;
    for (int i = t; i < a.n_bins; i += 32) {
      e0 += ds->je0[i];
      e1 += __ldcg(ds->je1 + i);
    }
    e0 = warp_sum(e0);
    e1 = warp_sum(e1);
    if (t == 0) {
      ds->jdone = 0;
      const double H0 = e0 + ds->jlik0, H1 = e1 + __ldcg(&ds->jlik1);
      const double dH = H1 - H0;
      ds->jH0 = H0;
      ds->jH1 = H1;
      ds->jdH = dH;
      int acc = 0;
      if (!isfinite(dH)) ds->status |= ST_NONFINITE;
      else acc = ds->jlog_u < -dH;
      ds->jaccepted = acc;
      s_acc = acc;
    }
  }
  __syncthreads();
  if (s_acc && t < a.n_bins) ds->P[t] = exp(ds->th[t]);
}

// ------------------------------------------------------------------ misc
// block 0: prior energy, block 1: likelihood energy of a gradient evaluation
__global__ void k_gradient_energies(ScalarArgs a, int r_prior, int nx, int r_lik, int nz) {
  await_previous();
  __shared__ double sh[32];
  const bool prior = blockIdx.x == 0;
  const double s = sum_partials(a.part + (prior ? r_prior : r_lik), prior ? nx : nz, sh);
  if (threadIdx.x == 0) a.ds->scratch[blockIdx.x] = prior ? s * (0.5 * a.inv_nv) : s;
}

// End of a Gibbs iteration: the chain record P[n_bins], b[n_sub], nbar[n_sub], dH, accepted, and
// the iteration counter.  Slot rec_idx
// of chain (chain0 + blockIdx.y) in a buffer laid out [slot][chain][rec_len]
__global__ void k_record(ScalarArgs a0, double* rec0, int rec_len, long long iter_stride, int chain0) {
  await_previous();
  const ScalarArgs a = chain_args(a0, blockIdx.y);
  DevState* ds = a.ds;
  const int t = threadIdx.x;
  const int ns = ds->nsub;
  double* rec = rec0 + (long long)ds->rec_idx * iter_stride + (long long)(chain0 + blockIdx.y) * rec_len;
  if (t < a.n_bins) rec[t] = ds->P[t];
  if (t < ns) {
    rec[a.n_bins + t] = ds->b[t];
    rec[a.n_bins + ns + t] = ds->nbar[t];
  }
  if (t == 0) {
    rec[a.n_bins + 2 * ns] = ds->dH;
    rec[a.n_bins + 2 * ns + 1] = (double)ds->accepted;
  }
  __syncthreads();
  if (t == 0) {
    ds->rec_idx += 1;
    ds->iteration += 1;
  }
}

__global__ void k_advance(DevState* ds) {
  await_previous();
  ds[blockIdx.x].iteration += 1;
}

__global__ void k_reset_rec(DevState* ds) {
  await_previous();
  ds[blockIdx.x].rec_idx = 0;
}

__global__ void k_zero_dc(float2* spec) { spec[0] = make_float2(0.f, 0.f); }

// block j of chain blockIdx.y: sum of the per-tile partials of mass bin j
__global__ void k_mstat(ScalarArgs a0, int region, int nblk, int final_) {
  await_previous();
  const ScalarArgs a = chain_args(a0, blockIdx.y);
  __shared__ double sh[32];
  const int j = blockIdx.x;
  const double s = sum_partials(a.part + region + (size_t)j * a.stride, nblk, sh);
  if (threadIdx.x == 0) {
    if (final_) a.ds->mstat2[j] = s;
    else a.ds->mstat[j] += s;
  }
}

void launch_move_end(const ScalarArgs& a, int r_init, int r_lik0, int r_final, int r_lik1, int nx, int nz, int advance,
                     int nch, cudaStream_t s) {
  launch_dep(k_move_end, dim3(8, nch), dim3(256), 0, s, a, r_init, r_lik0, r_final, r_lik1, nx, nz, advance);
}
void launch_power(const ScalarArgs& a, int region, int nx, int draw, int jump, int nch, cudaStream_t s) {
  launch_dep(k_power, dim3(a.n_bins, nch), dim3(320), 0, s, a, region, nx, draw, jump);
}
void launch_bias_nbar(const ScalarArgs& a, int region, int nz, int nch, cudaStream_t s) {
  launch_dep(k_bias_nbar, dim3(a.max_sub, nch), dim3(352), 0, s, a, region, nz);
}
void launch_jump_step(const ScalarArgs& a, int r_grad, int nx, int r_lik, int r_lik_move, int nz, int kind,
                      int nch, cudaStream_t s) {
  launch_dep(k_jump_step, dim3(a.n_bins + (kind == J_MID ? 0 : 1), nch), dim3(256), 0, s, a, r_grad, nx, r_lik,
             r_lik_move, nz, kind);
}
void launch_gradient_energies(const ScalarArgs& a, int r_prior, int nx, int r_lik, int nz, cudaStream_t s) {
  launch_dep(k_gradient_energies, dim3(2), dim3(256), 0, s, a, r_prior, nx, r_lik, nz);
}
void launch_record(const ScalarArgs& a, double* rec_dev, int rec_len, long long iter_stride, int chain0, int nch,
                   cudaStream_t s) {
  launch_dep(k_record, dim3(1, nch), dim3(MAXB), 0, s, a, rec_dev, rec_len, iter_stride, chain0);
}
void launch_advance(DevState* ds, int nch, cudaStream_t s) { launch_dep(k_advance, dim3(nch), dim3(1), 0, s, ds); }
void launch_commit_data(DevState* ds, const double* part, long long cstride, int nblk, int slot, int nch,
                        cudaStream_t s) {
  k_commit_data<<<nch, 1024, 0, s>>>(ds, part, cstride, nblk, slot);
}
void launch_reset_rec(DevState* ds, int nch, cudaStream_t s) { launch_dep(k_reset_rec, dim3(nch), dim3(1), 0, s, ds); }
void launch_zero_dc(float2* spec, cudaStream_t s) { k_zero_dc<<<1, 1, 0, s>>>(spec); }
void launch_mstat(const ScalarArgs& a, int region, int nblk, int n_mass, int final_, int nch, cudaStream_t s) {
  launch_dep(k_mstat, dim3(n_mass, nch), dim3(256), 0, s, a, region, nblk, final_);
}


// ------------------------------------------------------------------ posterior moments
// Running sums of the chain parameters of one chain (Secs. 6.2 and 7: the
// correlation matrices of P, b and Nbar), one FP64 accumulation per Gibbs
// iteration, in a fixed order.
__global__ void k_param_moments(ScalarArgs a, double* acc) {
  await_previous();
  const DevState* ds = a.ds;
  const int nb = a.n_bins, ns = ds->nsub, D = nb + 2 * ns;
  __shared__ double x[MAXB + 2 * MAXS];
  for (int i = threadIdx.x; i < D; i += blockDim.x)
    x[i] = i < nb ? ds->P[i] : i < nb + ns ? ds->b[i - nb] : ds->nbar[i - nb - ns];
  __syncthreads();
  if (threadIdx.x == 0) acc[0] += 1.0;
  for (int i = threadIdx.x; i < D; i += blockDim.x) acc[1 + i] += x[i];
  for (int q = threadIdx.x; q < D * D; q += blockDim.x) acc[1 + D + q] += x[q / D] * x[q % D];
}

// mean = S1 / n, var = S2 / n - mean^2 per voxel (population moments)
__global__ void k_moments_finish(const double* __restrict__ mom, long long nv, double n, double* mean, double* var) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nv; i += (long long)gridDim.x * blockDim.x) {
    const double m = mom[i] / n;
    if (mean) mean[i] = m;
    if (var) var[i] = mom[nv + i] / n - m * m;
  }
}

void launch_moments_finish(const double* mom, long long nv, double n, double* mean, double* var, int blocks,
                           cudaStream_t s) {
  k_moments_finish<<<blocks, 256, 0, s>>>(mom, nv, n, mean, var);
}

void launch_param_moments(const ScalarArgs& a, double* acc, cudaStream_t s) {
  launch_dep(k_param_moments, dim3(1), dim3(256), 0, s, a, acc);
}

// ------------------------------------------------------------------ failure detection
// Self-test of the bounded device waits: one thread announces 16 bytes on a
// shared-memory mbarrier and waits for them, but no copy is ever issued, so the
// phase never completes.  The wait gives up after limit_ns and records the
// timeout in the chain's status word exactly as a field pass does when a tile
// copy does not land; nothing is in flight when the block exits.
__global__ void k_wait_probe(DevState* ds, unsigned long long limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    mbar_expect_tx(&bar, 16);
    if (!mbar_wait(&bar, 0, limit_ns)) atomicOr(&ds->status, (int)ST_TIMEOUT);
  }
}

void launch_wait_probe(DevState* ds, unsigned long long limit_ns, cudaStream_t s) {
  k_wait_probe<<<1, 32, 0, s>>>(ds, limit_ns);
}

}  // namespace bps
