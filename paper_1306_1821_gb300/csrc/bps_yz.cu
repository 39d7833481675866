// Fused y^-1 / z / y stage of the force evaluation (Eq. Wiener_Posterior_force) on
// grids whose x plane of the work spectrum W(x, ky, kz) fits one block's shared
// memory: one block per plane, W read and written once (2 S_c + 2 S_r of HBM
// traffic where the three separate passes take 6 S_c + 2 S_r).
//
// What bounds it is the shared-memory pipe and the latency of its phases, so the
// plane makes few trips and few barriers:
//   - the first half of the inverse y transform reads W from global memory and the
//     second half of the forward one writes it, both straight from registers;
//   - the y transforms exchange in place.  With N = B A, the inverse reads
//     x[j + A b], transforms over b and leaves t[j][c] in row j + A c; its second
//     half transforms rows j + A c over j and leaves y = c + B d in row d + A c.
//     The forward transform walks back the same way (first over d within the rows
//     d + A c, then over c), so it ends in natural order, and neither needs a
//     second buffer: one block barrier between the halves of each;
//   - a warp owns eight consecutive z lines (four pairs, each one complex
//     transform) from C2R through the local force to R2C: the exchanges go through
//     the pair's own two rows with warp barriers only, and a warp whose lines
//     carry no survey data writes zeros.
// Rows are SP = N/2 + 1 (odd) complex apart, so that consecutive tasks of a first y half
// touch consecutive elements across rows, and the exchange within a pair is
// swizzled (zpos), which keeps the 8-byte accesses of a half warp on distinct banks.
//
// Measured per launch under ncu against the form with a block-wide exchange buffer
// (256 threads or fewer, 151 registers, 18% of the warp slots): 128^3 20.7 -> 13.0 us;
// 32 chains of 96^3 162 -> 103 us, of 64^3 54 -> 33 us, of 32^3 10.8 -> 9.4 us.  At 96^3
// the shared-memory pipe is 64-69% busy, with 40% of the warp slots filled.
#include "bps_internal.h"
#include "bps_passes.cuh"

namespace bps {
namespace {

template <int N, int NWARPS>
struct YZ {
  static constexpr int B = Cfg<N>::R1, A = Cfg<N>::R2;   // N = B A, B >= A
  static constexpr int ZP = Cfg<N>::ZP, H = N / 2, COLS = H + 1;
  static constexpr int SP = COLS;                        // row pitch in shared memory (complex)
  static constexpr int T1 = A * COLS, T2 = B * COLS;     // tasks of the two halves of a y transform
  static constexpr int PAIRS = 4, LINES = 2 * PAIRS;     // z lines of one warp unit
  static constexpr int UNITS = N / LINES;
  static constexpr int NW = NWARPS;
  static constexpr int NT = 32 * NW;
  static constexpr int ZT = PAIRS * B, ZR = (ZT + 31) / 32;   // second-half z tasks of a unit, rounds of them
  static constexpr size_t OFF_TW = (size_t)N * SP * sizeof(float2);
  static constexpr size_t OFF_TA = OFF_TW + (size_t)N * sizeof(float2);   // W^(a c) at c A + a
  static constexpr size_t OFF_TB = OFF_TA + (size_t)N * sizeof(float2);   // W^(c e) at e B + c
  static constexpr size_t BYTES = OFF_TB + (size_t)N * sizeof(float2);
  static_assert(PAIRS * A <= 32, "a unit's first z half is one round");
  static_assert(SP % 2 == 1 && UNITS * LINES == N, "layout");
  // blocks per SM that the registers allow with at most 12 bytes of spills (the narrow block at
  // 64^3, capped at 72 registers; the others have none)
  static constexpr int MIN_BLOCKS = 65536 / (NT * (N == 96 ? 73 : 80)) > 0 ? 65536 / (NT * (N == 96 ? 73 : 80)) : 1;
};

// Slot (c, j), c < B, j < A, of the exchange of pair f: in [0, H) in the pair's
// first row, in [H, N) in its second.
template <int N>
__device__ __forceinline__ int zpos(int c, int j, int f) {
  constexpr int A = Cfg<N>::R2;
  const int s = A == 8 ? (c ^ (c >> 3)) & 7 : ((c >> 2) | ((f & 1) << 1)) & (A - 1);
  return c * A + (j ^ s);
}

template <int N, int NW>
__global__ void __launch_bounds__(YZ<N, NW>::NT, YZ<N, NW>::MIN_BLOCKS) k_yzpass(Fields fp0, int region) {
  using Y = YZ<N, NW>;
  constexpr int A = Y::A, B = Y::B, ZP = Y::ZP, SP = Y::SP, H = Y::H, NT = Y::NT, COLS = Y::COLS;
  const Fields fp = at_chain(fp0, blockIdx.y);
  extern __shared__ __align__(128) unsigned char smem[];
  float2* blk = reinterpret_cast<float2*>(smem);
  float2* tw = reinterpret_cast<float2*>(smem + Y::OFF_TW);
  float2* twa = reinterpret_cast<float2*>(smem + Y::OFF_TA);
  float2* twb = reinterpret_cast<float2*>(smem + Y::OFF_TB);
  __shared__ int s_lo[N], s_hi[N];
  __shared__ float s_red[2 * Y::NW];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int plane = (int)blockIdx.x;
  float2* Wp = fp.W + (long long)plane * N * ZP;
  for (int i = t; i < N; i += NT) {
    tw[i] = fp.tw[i];
    twa[i] = fp.tw[(i / A) * (i % A)];
    twb[i] = fp.tw[(i / B) * (i % B)];
  }
  await_previous();
  // the first task's loads of the inverse y transform go out before anything waits
  // (a plane without support, which does not need them, is rare)
  float2 v0[B];
  if (t < Y::T1) {
#pragma unroll
    for (int b = 0; b < B; ++b) v0[b] = Wp[(t / COLS + A * b) * ZP + t % COLS];
  }
  if (fp.ds->jreuse) return;      // force stage reused by the jump (uniform)

  // ---- supports [lo, hi) of a and c on the z lines; outside them g = 0
  bool mine = false;
  const int2* span = survey(fp).span;
  for (int i = t; i < N; i += NT) {
    int lo = 0, hi = N;
    if (span) {
      const int2 sp = span[(long long)plane * N + i];
      lo = N - sp.x;
      hi = sp.y;
    }
    s_lo[i] = lo;
    s_hi[i] = hi;
    mine |= hi > lo;
  }
  if (!__syncthreads_or(mine)) {
    // a plane without support has g = 0 on every line: a zero force, W not read
    for (int e = t; e < N * ZP; e += NT)
      if (e % ZP <= H) Wp[e] = make_float2(0.f, 0.f);
    if (region >= 0 && t == 0) fp.part[region + plane] = 0.0;
    return;
  }

  // ---- inverse y transform, first half: rows j + A b of W -> t[j][c] in row j + A c
  for (int q = t; q < Y::T1; q += NT) {
    const int j = q / COLS, col = q - j * COLS;
    if (q != t) {
#pragma unroll
      for (int b = 0; b < B; ++b) v0[b] = Wp[(j + A * b) * ZP + col];
    }
    Dft<B, INV>::run(v0);
    blk[j * SP + col] = v0[0];
#pragma unroll
    for (int c = 1; c < B; ++c) {
      float2 w = tw[j * c];
      w.y = -w.y;
      blk[(j + A * c) * SP + col] = cmul(v0[c], w);
    }
  }
  __syncthreads();
  // second half: y = c + B d into row d + A c
  for (int q = t; q < Y::T2; q += NT) {
    const int c = q / COLS, col = q - c * COLS;
    float2* p = blk + A * c * SP + col;
    float2 v[A];
#pragma unroll
    for (int j = 0; j < A; ++j) v[j] = p[j * SP];
    Dft<A, INV>::run(v);
#pragma unroll
    for (int d = 0; d < A; ++d) p[d * SP] = v[d];
  }
  __syncthreads();

  // ---- z lines [y0, y0 + 8) of this warp; pair i is (y0 + i, y0 + i + 4)
  TwoSumAcc en;
  const bool want_e = region >= 0;
  for (int u = warp; u < Y::UNITS; u += NW) {
    const int y0 = u * Y::LINES;
    auto row = [&](int y) { return blk + (y / B + A * (y % B)) * SP; };
    bool some = false;
    if (lane < Y::LINES) some = s_hi[y0 + lane] > s_lo[y0 + lane];
    if (!__any_sync(0xffffffffu, some)) {
      for (int l = 0; l < Y::LINES; ++l) {
        float2* r = row(y0 + l);
        for (int k = lane; k <= H; k += 32) r[k] = make_float2(0.f, 0.f);
      }
    } else {
      const int f1 = lane / A, a1 = lane % A;            // first inverse half and second forward half
      const bool act1 = f1 < Y::PAIRS;
      float2* ra = row(y0 + (act1 ? f1 : 0));
      float2* rb = row(y0 + (act1 ? f1 : 0) + Y::PAIRS);
      auto slot = [&](float2* pa, float2* pb, int pos) -> float2& { return pos < H ? pa[pos] : pb[pos - H]; };
      {
        float2 v[B];
        if (act1) {
#pragma unroll
          for (int b = 0; b < B; ++b) {
            const int k = a1 + A * b;
            float2 xa, xb;
            if (k <= H) {
              xa = ra[k];
              xb = rb[k];
              if (k == 0 || k == H) { xa.y = 0.f; xb.y = 0.f; }
            } else {
              xa = cconj(ra[N - k]);
              xb = cconj(rb[N - k]);
            }
            v[b] = make_float2(xa.x - xb.y, xa.y + xb.x);
          }
          Dft<B, INV>::run(v);
        }
        __syncwarp();
        if (act1) {
#pragma unroll
          for (int c = 0; c < B; ++c) {
            if (c) {
              float2 w = twa[c * A + a1];
              w.y = -w.y;
              v[c] = cmul(v[c], w);
            }
            slot(ra, rb, zpos<N>(c, a1, f1)) = v[c];
          }
        }
      }
      __syncwarp();
#pragma unroll
      for (int r = 0; r < Y::ZR; ++r) {
        const int q = lane + 32 * r;
        const int f = q / B, c = q - f * B;
        const bool act = Y::ZT % 32 == 0 || q < Y::ZT;
        const int ya = y0 + (act ? f : 0), yb = ya + Y::PAIRS;
        float2* pa = row(ya);
        float2* pb = row(yb);
        float2 v[A];
        if (act) {
          const int loa = s_lo[ya], hia = s_hi[ya], lob = s_lo[yb], hib = s_hi[yb];
          const long long la = ((long long)plane * N + ya) * N, lb = la + (long long)Y::PAIRS * N;
          float aa[A], ca[A], ab[A], cb[A];
#pragma unroll
          for (int d = 0; d < A; ++d) {
            const int n = c + B * d;
            const bool ina = n >= loa && n < hia, inb = n >= lob && n < hib;
            aa[d] = ina ? __ldg(fp.a + la + n) : 0.f;
            ca[d] = ina ? __ldg(fp.c + la + n) : 0.f;
            ab[d] = inb ? __ldg(fp.a + lb + n) : 0.f;
            cb[d] = inb ? __ldg(fp.c + lb + n) : 0.f;
          }
#pragma unroll
          for (int j = 0; j < A; ++j) v[j] = slot(pa, pb, zpos<N>(c, j, f));
          Dft<A, INV>::run(v);
          // here v[d] = y[c + B d]: real part line ya, imaginary part line yb
#pragma unroll
          for (int d = 0; d < A; ++d) {
            const float da = v[d].x * fp.inv_nv, db = v[d].y * fp.inv_nv;
            const float ga = fmaf(aa[d], da, -ca[d]), gb = fmaf(ab[d], db, -cb[d]);
            if (want_e) {                               // a d^2 - 2 c d
              en.add(da * (ga - ca[d]));
              en.add(db * (gb - cb[d]));
            }
            v[d] = make_float2(ga, gb);
          }
          Dft<A, FWD>::run(v);
        }
        __syncwarp();
        if (act) {
#pragma unroll
          for (int e = 0; e < A; ++e) slot(pa, pb, zpos<N>(c, e, f)) = e ? cmul(v[e], twb[e * B + c]) : v[e];
        }
      }
      __syncwarp();
      {
        // second forward half, then the split into the two half spectra:
        // G_a[k] = (Y[k] + conj Y[N-k]) / 2, G_b[k] = -i (Y[k] - conj Y[N-k]) / 2; Y[N - k]
        // of k = e + A d sits in the pair's lane A - e as element B - 1 - d (or in the
        // own element (B - d) mod B for e = 0)
        float2 v[B];
        if (act1) {
#pragma unroll
          for (int c = 0; c < B; ++c) v[c] = slot(ra, rb, zpos<N>(c, a1, f1));
          Dft<B, FWD>::run(v);
        }
        __syncwarp();
        const int src = act1 ? lane - a1 + (A - a1) % A : lane;
#pragma unroll
        for (int d = 0; d <= B / 2; ++d) {
          const float2 snd = v[B - 1 - d];
          float2 rcv;
          rcv.x = __shfl_sync(0xffffffffu, snd.x, src);
          rcv.y = __shfl_sync(0xffffffffu, snd.y, src);
          const int k = a1 + A * d;
          if (act1 && k <= H) {
            const float2 yk = v[d];
            const float2 ym = cconj(a1 == 0 ? v[(B - d) % B] : rcv);
            ra[k] = make_float2(0.5f * (yk.x + ym.x), 0.5f * (yk.y + ym.y));
            rb[k] = make_float2(0.5f * (yk.y - ym.y), -0.5f * (yk.x - ym.x));
          }
        }
      }
    }
  }
  __syncthreads();

  // ---- forward y transform, first half: rows d + A c (y = c + B d) -> t[c][e] in row e + A c
  for (int q = t; q < Y::T2; q += NT) {
    const int c = q / COLS, col = q - c * COLS;
    float2* p = blk + A * c * SP + col;
    float2 v[A];
#pragma unroll
    for (int d = 0; d < A; ++d) v[d] = p[d * SP];
    Dft<A, FWD>::run(v);
    p[0] = v[0];
#pragma unroll
    for (int e = 1; e < A; ++e) p[e * SP] = cmul(v[e], tw[c * e]);
  }
  __syncthreads();
  // second half: ky = e + A f straight to W
  for (int q = t; q < Y::T1; q += NT) {
    const int e = q / COLS, col = q - e * COLS;
    float2 v[B];
#pragma unroll
    for (int c = 0; c < B; ++c) v[c] = blk[(e + A * c) * SP + col];
    Dft<B, FWD>::run(v);
#pragma unroll
    for (int f = 0; f < B; ++f) Wp[(e + A * f) * ZP + col] = v[f];
  }
  if (want_e) {
    TwoSumAcc h;                  // halving is exact
    h.s = 0.5f * en.s;
    h.c = 0.5f * en.c;
    const double s = block_sum2<NT>(h, s_red);
    if (t == 0) fp.part[region + plane] = s;
  }
}

template <int N, int NW>
void launch_yz(const Fields& f, int region, int nch, cudaStream_t s) {
  launch_dep(k_yzpass<N, NW>, dim3(N, nch), dim3(YZ<N, NW>::NT), YZ<N, NW>::BYTES, s, f, region);
}

template <int N, int NW>
bool set_yz(YzEntry* out) {
  if (cudaFuncSetAttribute(k_yzpass<N, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)YZ<N, NW>::BYTES) !=
      cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  out->run = launch_yz<N, NW>;
  out->tiles = N;
  return true;
}

}  // namespace

// Two block widths.  With no more planes than SMs each SM holds one block, and a
// block wide enough for one round of first-half y tasks (at 32^3: second-half) is
// fastest.  With more planes narrower blocks, several to an SM, waste fewer lanes
// in their last rounds and wait less at barriers: a Gibbs iteration of 32 chains
// each of 32^3, 64^3 and 96^3 takes 8.83 ms with the wide blocks everywhere, 8.63 ms
// with the narrow ones; of 24 chains of 128^3 9.09 ms with three narrow blocks per
// SM (which spill) and 8.76 ms with two.
bool yz_table(int N, int nch, int n_sm, YzEntry* out) {
  const bool few = N * nch <= n_sm;
  switch (N) {
    case 32: return few ? set_yz<32, 5>(out) : set_yz<32, 3>(out);
    case 64: return few ? set_yz<64, 9>(out) : set_yz<64, 5>(out);
    case 96: return few ? set_yz<96, 13>(out) : set_yz<96, 7>(out);
    case 128: return few ? set_yz<128, 17>(out) : set_yz<128, 9>(out);
    default: return false;
  }
}

}  // namespace bps
