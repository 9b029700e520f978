// passesx.cuh -- the five passes of S^-1 (Sec. 2.2) for FP64 fields, with the
// line transforms in 64-bit block fixed point (fx.cuh).
//
// The pipeline, layouts and register four-step line transforms are those of
// passes4.cuh.  The spectra A and B hold pairs of 64-bit integers in place of
// pairs of doubles, and every block (tile) of a pass writes one exponent: its
// values are q 2^E.  A pass reads the exponents of the tiles its lines cross,
// bounds the L1 norm of its lines from the high words, picks its own exponent
// from the largest, and shifts its values to it before it transforms:
//
//   XF  doubles from the prologue -> A, EA[z][yb]        (yb = y / 32)
//   YF  A, EA -> B, EB[kx][zb]                           (zb = z / 16)
//   Z   B, EB, times the multipliers (each a 53-bit significand and its own
//       exponent) -> B, EZ[kx][kyb]
//   YI  B, EZ -> A, EC[zb][kx]
//   XI  A, EC -> doubles for the epilogue
//
// A tile that meets a NaN or an infinity marks its exponent (kFxNaN), which
// every later tile it reaches inherits, and the epilogue then sees NaN in every
// cell: a transform spreads such a value over the whole grid in any arithmetic
// (the FP64 passes give a mixture of NaNs and infinities).  Multipliers must not
// be negative (kx_z reads a sign bit as part of the exponent; the prior's, the
// bias's and the smoothing's are not), and subnormal ones count as zero.
//
// What bounds them: the FP64 Stockham passes they replace ran at 0.74-0.8 of
// the FP64 pipe (2 per SM and clock).  These issue on half of all cycles with
// 16 warps per SM (128 registers), the integer adders 45-60% busy.  S^-1 at
// 128^3 / 192^3 / 256^3 went from 327 / 1170 / 3450 us to 88 / 264 / 470.
#pragma once

#include <cmath>
#include <vector>

#include "ctx.h"
#include "fx.cuh"
#include "passes4.cuh"

namespace plc {

// Tile exponents of the four intermediate spectra.
struct FxExps {
  int *a, *b, *z, *c;
};
// Ints that FxExps needs for an n^3 grid.
inline size_t fx_exps_ints(int n) {
  const size_t h = n / 2 + 1, t = (n + 15) / 16;
  return (size_t)n * ((n + 31) / 32) + 3 * h * t;
}
inline FxExps fx_exps(int* p, int n) {
  const size_t h = n / 2 + 1, t = (n + 15) / 16;
  int* b = p + (size_t)n * ((n + 31) / 32);
  return FxExps{p, b, b + h * t, b + 2 * h * t};
}

// Twiddles W_n^m of the fixed-point passes; empty for lengths without them.
// long double (at least 64 significant bits on the hosts in use) is software
// arithmetic on AArch64, so only the first octant is evaluated: creating a
// context of 256^3 takes 338 us (310 without this table), 490 with all of the
// circle evaluated, and one of 512^3, which has no such passes, 420 (778).
inline std::vector<fxw> fx_twiddles(int n) {
  if (!fixed_length(n)) return {};
  const int o = n / 8;   // every fixed length is a multiple of 8
  const long double step = 2.0L * std::acos(-1.0L) / (long double)n;
  const long double one = (long double)(1ll << kFxOne);
  std::vector<long long> c(o + 1), s(o + 1);
  for (int j = 0; j <= o; ++j) {
    c[j] = std::llrint(std::cos(step * (long double)j) * one);
    s[j] = std::llrint(std::sin(step * (long double)j) * one);
  }
  auto cosine = [&](int m) {   // cos(2 pi m / n) 2^61
    m = m <= n / 2 ? m : n - m;
    const int r = m <= n / 4 ? m : n / 2 - m;
    const long long v = r <= o ? c[r] : s[n / 4 - r];
    return m <= n / 4 ? v : -v;
  };
  std::vector<fxw> tw(n);
  for (int m = 0; m < n; ++m) tw[m] = fx_factor(cosine(m), -cosine((m + n - n / 4) % n));
  return tw;
}

// Resident blocks per SM asked of the compiler: two (up to 128 registers).
// S^-1 in us at 128^3 / 192^3 / 256^3: 92 / 314 / 545 without a bound (the z
// pass takes 190 registers), 88 / 269 / 504 at two, 90 / 281 / 616 at three
// (spills), taken together.
constexpr int kFxBlocks = 2;

template <int N1_, int N2_> struct GeoX : Geo4<fx, N1_, N2_> {
  static_assert(N1_ / 2 <= kThreads / 32, "one warp per pair of x-pass tasks");
  static_assert(fixed_length(N1_ * N2_), "listed as a fixed-point length");
  using G = Geo4<fx, N1_, N2_>;
  static constexpr int NM = N1_ > N2_ ? N1_ : N2_;
  static constexpr size_t tw_bytes = sizeof(fxw) * N1_ * N2_;
  static constexpr size_t smem_y = tw_bytes + G::x_bytes;
  static constexpr size_t smem_z = smem_y + G::m_bytes;
  static constexpr size_t smem_x = tw_bytes + (G::x_bytes > G::r_bytes ? G::x_bytes : G::r_bytes);
  static_assert(tw_bytes % 16 == 0, "the exchange buffer follows the twiddles");
  // per-thread L1 parts: line c at [c * (NM + 1)]
  static constexpr int red_words = G::L * (NM + 1) + 8;
};

// Twiddles W_N^{k1 n2} as split factors, from the natural table.
template <int N1, int N2>
__device__ __forceinline__ void load_twx(fxw* tw, const fxw* __restrict__ twg) {
  for (int i = threadIdx.x; i < N1 * N2; i += blockDim.x) tw[i] = twg[(i / N2) * (i % N2)];
}

template <int N1, int N2, int SIGN>
__device__ __forceinline__ void phase_a_x(fxc* v, const fxw* tw, int n2) {
  dft_small<fx, SIGN, N1>(v);
#pragma unroll
  for (int k1 = 1; k1 < N1; ++k1) v[k1] = cmulx<SIGN>(v[k1], tw[k1 * N2 + n2]);
}
template <int N1, int N2>
__device__ __forceinline__ void phase_b_inv_x(fxc* v, const fxw* tw, int k1) {
  dft_small<fx, +1, N2>(v);
#pragma unroll
  for (int n2 = 1; n2 < N2; ++n2) v[n2] = cmulx<+1>(v[n2], tw[k1 * N2 + n2]);
}

// The largest L1 norm over the block's 16 lines from the parts of the tasks
// (line c, task j < CNT): the same order of additions in every warp, so all
// threads get the same value.  Publishes with one barrier.
template <int CNT, int NM>
__device__ __forceinline__ float block_l1(float* red, bool task, int c, int j, float part) {
  if (task) red[c * (NM + 1) + j] = part;
  __syncthreads();
  const int l = threadIdx.x & 15;
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < CNT; ++i) s += red[l * (NM + 1) + i];
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(s)));
}

// Largest of cnt exponents e[0], e[stride], ..., in every thread of a warp.
__device__ __forceinline__ int warp_max_exp(const int* __restrict__ e, int cnt, int stride) {
  int m = kFxNone;
  for (int i = threadIdx.x & 31; i < cnt; i += 32) m = max(m, __ldg(e + (size_t)i * stride));
  return __reduce_max_sync(0xffffffffu, m);
}

#define PLC_PASSX_SETUP                                                  \
  using Gm = GeoX<N1, N2>;                                               \
  using C = fxc;                                                         \
  constexpr int N = Gm::N, L = Gm::L;                                    \
  if (done && *done) return;                                             \
  extern __shared__ __align__(16) unsigned char smem_raw[];              \
  fxw* tw = reinterpret_cast<fxw*>(smem_raw);                            \
  C* X = reinterpret_cast<C*>(tw + N);                                   \
  __shared__ float red[Gm::red_words]

// Exponent of a tile whose values come in with exponents up to ref and whose
// lines have L1 norms up to l1 units of 2^(ref + 32) (fx_mag, low by at most
// one unit for each of 2 N values).
__device__ __forceinline__ int tile_exp(int ref, float l1, int n) {
  return ref + max(0, l1_bits(l1 + 2.f * (float)n) + 32 - kFxBits);
}

// ---------------------------------------------------------------------------
// XF: r2c along x + prologue (see k4_xf).
// ---------------------------------------------------------------------------
template <int N1, int N2, typename Pro>
__global__ void __launch_bounds__(kThreads, kFxBlocks)
kx_xf(Pro pro, fxc* __restrict__ A, FxExps ex, const fxw* __restrict__ twg,
      const int* __restrict__ done) {
  PLC_PASSX_SETUP;
  double* R = reinterpret_cast<double*>(tw + N);
  load_twx<N1, N2>(tw, twg);
  pro.prepare();
  const int h = N / 2 + 1, z = blockIdx.y, y0 = blockIdx.x * Gm::RY;
  constexpr int Q = N / 4, TOT = Gm::RY * Q, B4 = 4;
  const size_t row0 = ((size_t)z * N + y0) * N;
  if (threadIdx.x == 0) pro.prefetch(row0, Gm::RY * N);
  int top = 0;   // largest high word of |x|
  for (int base = threadIdx.x; base < TOT; base += B4 * kThreads) {
    V4<double> u[B4];
#pragma unroll
    for (int q = 0; q < B4; ++q) {
      const int e = base + q * kThreads;
      if (e < TOT) u[q] = pro.vec4(row0 + (size_t)(e / Q) * N + 4 * (e % Q));
    }
#pragma unroll
    for (int q = 0; q < B4; ++q) {
      const int e = base + q * kThreads;
      if (e >= TOT) continue;
#pragma unroll
      for (int j = 0; j < 4; ++j) top = max(top, __double2hiint(u[q].v[j]) & 0x7fffffff);
      st4(&R[(e / Q) * Gm::SR + 4 * (e % Q)], u[q]);
    }
  }
  top = __reduce_max_sync(0xffffffffu, top);
  int* tops = reinterpret_cast<int*>(red + L * (Gm::NM + 1));
  if ((threadIdx.x & 31) == 0) tops[threadIdx.x >> 5] = top;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kThreads / 32; ++i) top = max(top, tops[i]);
  const int exm = top >> 20;   // exponent field of the largest |x|
  // phase A on (c, n2), n2 on consecutive lanes
  const bool task_a = threadIdx.x < L * N2;
  const int n2a = threadIdx.x % N2, ca = threadIdx.x / N2;
  const double *ra = R + (2 * ca) * Gm::SR + n2a, *rb = ra + Gm::SR;
  float part = 0.f;
  if (task_a) {
    // |x| in units of 2^(exm - 1023), cut to 20 bits
    const int off = (exm - 127) << 20;
    auto mag = [&](double x) {
      return __uint_as_float((unsigned)max((__double2hiint(x) & 0x7fffffff) - off, 0) << 3);
    };
    if (exm != 0) {
#pragma unroll
      for (int n1 = 0; n1 < N1; ++n1) part += mag(ra[N2 * n1]) + mag(rb[N2 * n1]);
    } else {   // zeros and subnormals, in units of 2^-1042
#pragma unroll 1
      for (int n1 = 0; n1 < N1; ++n1)
        part += (float)((__double2hiint(ra[N2 * n1]) & 0x7fffffff) +
                        (__double2hiint(rb[N2 * n1]) & 0x7fffffff) + 2);
    }
  }
  const float l1 = block_l1<N2, Gm::NM>(red, task_a, ca, n2a, part);
  // (-1083: the finest quantum fx_from converts subnormals to)
  const int E = exm == 2047 ? kFxNaN
                : exm == 0  ? max(-1042 + l1_bits(l1) - kFxBits, -1083)
                            : exm - 1023 + l1_bits(l1) - kFxBits;
  C v[Gm::NM];
  if (task_a) {
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1)
      v[n1] = C{fx_from(ra[N2 * n1], E), fx_from(rb[N2 * n1], E)};
    phase_a_x<N1, N2, -1>(v, tw, n2a);
  }
  __syncthreads();   // X overlays R
  if (task_a) {
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) X[ca * Gm::S + k1 * N2 + n2a] = v[k1];
  }
  if (threadIdx.x == 0) ex.a[z * (N / Gm::RY) + blockIdx.x] = E;
  __syncthreads();
  // phase B in pairs k1, N1 - k1 (one warp per pair), split into X_a, X_b
  const int g = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (g < N1 / 2) {
    const int c = lane & 15, member = lane >> 4;
    const int k1 = pair_k1<N1>(g, member);
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = X[c * Gm::S + k1 * N2 + n2];
    dft_small<fx, -1, N2>(v);
    C* dst = A + ((size_t)z * h + k1) * N + y0 + 2 * c;
    auto put = [&](int k2, C zk, C zm) {   // zm = Z[N - k]
      const C zc = cconj(zm);
      const C s = cadd(zk, zc), d = csub(zk, zc);
      C* p = dst + (size_t)N1 * k2 * N;
      p[0] = C{halve(s.x), halve(s.y)};
      p[1] = C{halve(d.y), -halve(d.x)};
    };
    if (g != 0) {
      C pz[N2 / 2];
#pragma unroll
      for (int j = 0; j < N2 / 2; ++j) pz[j] = shfl_xor16(v[N2 - 1 - j]);
#pragma unroll
      for (int k2 = 0; k2 < N2 / 2; ++k2) put(k2, v[k2], pz[k2]);
    } else if (member == 0) {
#pragma unroll
      for (int k2 = 0; k2 <= N2 / 2; ++k2) put(k2, v[k2], v[(N2 - k2) % N2]);
    } else {
#pragma unroll
      for (int k2 = 0; k2 < N2 / 2; ++k2) put(k2, v[k2], v[N2 - 1 - k2]);
    }
  }
}

// ---------------------------------------------------------------------------
// YF: c2c along y (see k4_yf).
// ---------------------------------------------------------------------------
template <int N1, int N2>
__global__ void __launch_bounds__(kThreads, kFxBlocks)
kx_yf(const fxc* __restrict__ A, fxc* __restrict__ B, FxExps ex, const fxw* __restrict__ twg,
      const int* __restrict__ done) {
  PLC_PASSX_SETUP;
  const int h = N / 2 + 1, z0 = blockIdx.x * L, kx = blockIdx.y;
  constexpr int NB = N / Gm::RY;
  const bool task_a = L * N2 == kThreads || threadIdx.x < L * N2;
  const int n2 = threadIdx.x % N2, c = threadIdx.x / N2;
  C v[N1];
  if (task_a) {
    const C* src = A + ((size_t)(z0 + c) * h + kx) * N + n2;
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) v[n1] = src[N2 * n1];
  }
  load_twx<N1, N2>(tw, twg);
  const int ref = warp_max_exp(ex.a + z0 * NB, L * NB, 1);
  const int* el = ex.a + (z0 + c) * NB;
  float part = 0.f;
  if (task_a) {
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1)
      part = fmaf(fx_mag(v[n1]), exp2_le0(__ldg(el + (N2 * n1 + n2) / Gm::RY) - ref), part);
  }
  const int E = tile_exp(ref, block_l1<N2, Gm::NM>(red, task_a, c, n2, part), N);
  if (task_a) {
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1)
      v[n1] = FxShift(E - __ldg(el + (N2 * n1 + n2) / Gm::RY))(v[n1]);
    phase_a_x<N1, N2, -1>(v, tw, n2);
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) X[c * Gm::S + k1 * N2 + n2] = v[k1];
  }
  if (threadIdx.x == 0) ex.b[kx * (N / L) + blockIdx.x] = E;
  __syncthreads();
  auto task_b = [&](int t) {
    const int c = t % L, k1 = t / L;
    C v[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = X[c * Gm::S + k1 * N2 + n2];
    dft_small<fx, -1, N2>(v);
    C* dst = B + ((size_t)kx * N + k1) * N + z0 + c;
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) dst[(size_t)N1 * k2 * N] = v[k2];
  };
  if constexpr (L * N1 == kThreads) {
    task_b(threadIdx.x);
  } else {
    for (int t = threadIdx.x; t < L * N1; t += kThreads) task_b(t);
  }
}

// ---------------------------------------------------------------------------
// Z: forward c2c along z, times M[|m|^2], inverse c2c, in place (see k4_z).
// A multiplier M = m 2^-61 2^x, m in [2^60, 2^61), multiplies q by m 2^-61
// and adds x to the exponent, so that its 53 bits count whatever the range of
// the multipliers in the tile.
// ---------------------------------------------------------------------------
template <int N1, int N2>
__global__ void __launch_bounds__(kThreads, kFxBlocks)
kx_z(fxc* __restrict__ B, FxExps ex, const double* __restrict__ M, int zero_dc,
     const fxw* __restrict__ twg, const int* __restrict__ done) {
  PLC_PASSX_SETUP;
  double* Ms = reinterpret_cast<double*>(X + L * Gm::S);
  const int ky0 = blockIdx.x * L, kx = N / 2 - blockIdx.y;
  C* line0 = B + ((size_t)kx * N + ky0) * N;
  constexpr bool kOneA = L * N2 == kThreads;
  const bool task_a = kOneA || threadIdx.x < L * N2;
  const int n2a = threadIdx.x % N2, ca = threadIdx.x / N2;
  constexpr int NZ = N / L;
  C v[Gm::NM];
  if (task_a) {
    const C* src = line0 + (size_t)ca * N + n2a;
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) v[n1] = src[N2 * n1];
  }
  load_twx<N1, N2>(tw, twg);
  // the block's multipliers Ms[c][|mz|] and their largest exponent
  constexpr int HM = N / 2 + 1, MP = Gm::MP;
  int xm = 0;
  for (int i = threadIdx.x; i < L * HM; i += kThreads) {
    const int c = i / HM, mz = i - c * HM;
    const int ky = ky0 + c, my = min(ky, N - ky);
    const int m2 = kx * kx + my * my + mz * mz;
    const double m = (zero_dc && m2 == 0) ? 0.0 : __ldg(M + m2);
    xm = max(xm, __double2hiint(m) >> 20);
    Ms[c * MP + mz] = m;
  }
  xm = __reduce_max_sync(0xffffffffu, xm);
  int* tops = reinterpret_cast<int*>(red + L * (Gm::NM + 1));
  if ((threadIdx.x & 31) == 0) tops[threadIdx.x >> 5] = xm;
  const int* eb = ex.b + kx * NZ;
  const int ref = warp_max_exp(eb, NZ, 1);
  float part = 0.f;
  if (task_a) {
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1)
      part = fmaf(fx_mag(v[n1]), exp2_le0(__ldg(eb + (N2 * n1 + n2a) / L) - ref), part);
  }
  const int E1 = tile_exp(ref, block_l1<N2, Gm::NM>(red, task_a, ca, n2a, part), N);
#pragma unroll
  for (int i = 0; i < kThreads / 32; ++i) xm = max(xm, tops[i]);
  if (task_a) {
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1)
      v[n1] = FxShift(E1 - __ldg(eb + (N2 * n1 + n2a) / L))(v[n1]);
    phase_a_x<N1, N2, -1>(v, tw, n2a);
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) X[ca * Gm::S + k1 * N2 + n2a] = v[k1];
  }
  __syncthreads();
  const int xref = xm == 2047 ? kFxNaN : xm - 1022;
  // the tile of the DC mode, whose multiplier is set apart from the others':
  // its magnitudes are taken from all 64 bits
  const bool dc = kx == 0 && ky0 == 0;
  static_assert(L * N1 <= kThreads, "one phase-B task per thread at most");
  const bool task_b = L * N1 == kThreads || threadIdx.x < L * N1;
  const int cb = threadIdx.x % L, k1 = threadIdx.x / L;
  part = 0.f;
  if (task_b) {
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = X[cb * Gm::S + k1 * N2 + n2];
    dft_small<fx, -1, N2>(v);
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) {
      const int kz = k1 + N1 * k2, mz = min(kz, N - kz);
      const long long mb = __double_as_longlong(Ms[cb * MP + mz]);
      const int xe = (int)(mb >> 52);
      const long long mm = xe == 0 ? 0ll : ((mb & 0xFFFFFFFFFFFFFll) | (1ll << 52)) << 8;
      const fxk w{fx_hi(mm), fx_lo(mm)};
      v[k2] = C{v[k2].x * w, v[k2].y * w};
      part = fmaf(fx_mag(v[k2]), exp2_le0(xe - xm), part);
    }
    if (dc) {
      part = 0.f;
#pragma unroll 1
      for (int k2 = 0; k2 < N2; ++k2) {
        const int kz = k1 + N1 * k2, mz = min(kz, N - kz);
        C u = v[0];
#pragma unroll
        for (int j = 1; j < N2; ++j)
          if (j == k2) u = v[j];
        part = fmaf((fabsf((float)u.x.v) + fabsf((float)u.y.v)) * 0x1p-32f,
                    exp2_le0((__double2hiint(Ms[cb * MP + mz]) >> 20) - xm), part);
      }
    }
  }
  // (the parts of the forward transform were read before the last barrier)
  const float l1 = block_l1<N1, Gm::NM>(red, task_b, cb, k1, part);
  // all multipliers zero (xm = 0): E stays far below any exponent in use
  const int E = E1 + xref + l1_bits(l1 + (dc ? 2.f * (float)N * 0x1p-32f : 2.f * (float)N)) + 32 -
                kFxBits;
  if (task_b) {
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) {
      const int kz = k1 + N1 * k2, mz = min(kz, N - kz);
      const int s = E - (E1 + (__double2hiint(Ms[cb * MP + mz]) >> 20) - 1022);
      if (s >= 0) {
        v[k2] = FxShift(s)(v[k2]);
      } else {
        const int t = min(-s, 63);
        v[k2] = C{fx{v[k2].x.v << t}, fx{v[k2].y.v << t}};
      }
    }
    phase_b_inv_x<N1, N2>(v, tw, k1);
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) X[cb * Gm::S + k1 * N2 + n2] = v[n2];
  }
  if (threadIdx.x == 0) ex.z[kx * NZ + blockIdx.x] = E;
  __syncthreads();
  if (task_a) {
#pragma unroll
    for (int k = 0; k < N1; ++k) v[k] = X[ca * Gm::S + k * N2 + n2a];
    dft_small<fx, +1, N1>(v);
    C* dst = line0 + (size_t)ca * N + n2a;
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) dst[N2 * n1] = v[n1];
  }
}

// ---------------------------------------------------------------------------
// YI: inverse c2c along y (see k4_yi).
// ---------------------------------------------------------------------------
template <int N1, int N2>
__global__ void __launch_bounds__(kThreads, kFxBlocks)
kx_yi(const fxc* __restrict__ B, fxc* __restrict__ A, FxExps ex, const fxw* __restrict__ twg,
      const int* __restrict__ done) {
  PLC_PASSX_SETUP;
  const int h = N / 2 + 1, z0 = blockIdx.x * L, kx = blockIdx.y;
  constexpr int NZ = N / L;
  static_assert(L * N1 <= kThreads, "one phase-B task per thread at most");
  const bool task_b = L * N1 == kThreads || threadIdx.x < L * N1;
  const int cb = threadIdx.x % L, k1 = threadIdx.x / L;
  C v[Gm::NM];
  if (task_b) {
    const C* src = B + ((size_t)kx * N + k1) * N + z0 + cb;
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) v[k2] = src[(size_t)N1 * k2 * N];
  }
  load_twx<N1, N2>(tw, twg);
  const int* ez = ex.z + kx * NZ;
  const int ref = warp_max_exp(ez, NZ, 1);
  float part = 0.f;
  if (task_b) {
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2)
      part = fmaf(fx_mag(v[k2]), exp2_le0(__ldg(ez + (k1 + N1 * k2) / L) - ref), part);
  }
  const int E = tile_exp(ref, block_l1<N1, Gm::NM>(red, task_b, cb, k1, part), N);
  if (task_b) {
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2)
      v[k2] = FxShift(E - __ldg(ez + (k1 + N1 * k2) / L))(v[k2]);
    phase_b_inv_x<N1, N2>(v, tw, k1);
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) X[cb * Gm::S + k1 * N2 + n2] = v[n2];
  }
  if (threadIdx.x == 0) ex.c[blockIdx.x * h + kx] = E;
  __syncthreads();
  if (L * N2 == kThreads || threadIdx.x < L * N2) {
    const int n2 = threadIdx.x % N2, c = threadIdx.x / N2;
#pragma unroll
    for (int k = 0; k < N1; ++k) v[k] = X[c * Gm::S + k * N2 + n2];
    dft_small<fx, +1, N1>(v);
    C* dst = A + ((size_t)(z0 + c) * h + kx) * N + n2;
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) dst[N2 * n1] = v[n1];
  }
}

// ---------------------------------------------------------------------------
// XI: c2r along x + epilogue (see k4_xi).  Z[k] = X_a[k] + i X_b[k] and the
// form for N - k have L1 norms of at most |X_a| + |X_b| each, so a line's is
// bounded by twice the sum over k <= n/2.
// ---------------------------------------------------------------------------
// Epilogues that take the transform's integers and exponent (Epi::kRaw).
template <typename Epi, typename = void> struct EpiRaw {
  static constexpr bool value = false;
};
template <typename Epi> struct EpiRaw<Epi, decltype((void)Epi::kRaw)> {
  static constexpr bool value = Epi::kRaw;
};

template <int N1, int N2, typename Epi, typename Fin>
__global__ void __launch_bounds__(kThreads, kFxBlocks)
kx_xi(const fxc* __restrict__ A, FxExps ex, Epi epi, Fin fin, RedArgs ra,
      const fxw* __restrict__ twg, const int* __restrict__ done) {
  PLC_PASSX_SETUP;
  fx* R = reinterpret_cast<fx*>(tw + N);
  const int h = N / 2 + 1, nh = N / 2, z = blockIdx.y, y0 = blockIdx.x * Gm::RY;
  const size_t row0 = ((size_t)z * N + y0) * N;
  if (threadIdx.x == 0) epi.prefetch(row0, Gm::RY * N);
  const int g = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cb = lane & 15, member = lane >> 4;
  const bool task_b = g < N1 / 2;
  const int k1 = task_b ? pair_k1<N1>(g, member) : 0;
  constexpr int NL = N2 / 2 + 1;
  C za[NL], zb[NL];
  const int nload = (g == 0 && member == 0) ? N2 / 2 + 1 : N2 / 2;
  if (task_b) {
    const C* src = A + ((size_t)z * h + k1) * N + y0 + 2 * cb;
#pragma unroll
    for (int k2 = 0; k2 < NL; ++k2)
      if (k2 < nload) {
        za[k2] = src[(size_t)N1 * k2 * N];
        zb[k2] = src[(size_t)N1 * k2 * N + 1];
      }
  }
  load_twx<N1, N2>(tw, twg);
  const int* ec = ex.c + (z / L) * h;
  const int ref = warp_max_exp(ec, h, 1);
  float part = 0.f;
  if (task_b) {
#pragma unroll
    for (int k2 = 0; k2 < NL; ++k2)
      if (k2 < nload)
        part = fmaf(fx_mag(za[k2]) + fx_mag(zb[k2]), exp2_le0(__ldg(ec + k1 + N1 * k2) - ref), part);
  }
  const int E = tile_exp(ref, 2.f * block_l1<N1, Gm::NM>(red, task_b, cb, task_b ? 2 * g + member : 0,
                                                         part), 2 * N);
  C v[Gm::NM];
  if (task_b) {
    C zc[NL];
#pragma unroll
    for (int k2 = 0; k2 < NL; ++k2) {
      if (k2 >= nload) continue;
      const int k = k1 + N1 * k2;
      const FxShift sh(E - __ldg(ec + k));
      C xa = sh(za[k2]), xb = sh(zb[k2]);
      if (k == 0 || k == nh) { xa.y = fx{0}; xb.y = fx{0}; }
      v[k2] = C{xa.x - xb.y, xa.y + xb.x};
      zc[k2] = C{xa.x + xb.y, xb.x - xa.y};
    }
    if (g != 0) {
#pragma unroll
      for (int j = 0; j < N2 / 2; ++j) v[N2 - 1 - j] = shfl_xor16(zc[j]);
    } else if (member == 0) {
#pragma unroll
      for (int k2 = N2 / 2 + 1; k2 < N2; ++k2) v[k2] = zc[N2 - k2];
    } else {
#pragma unroll
      for (int k2 = N2 / 2; k2 < N2; ++k2) v[k2] = zc[N2 - 1 - k2];
    }
    phase_b_inv_x<N1, N2>(v, tw, k1);
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) X[cb * Gm::S + k1 * N2 + n2] = v[n2];
  }
  __syncthreads();
  const bool task_a = threadIdx.x < L * N2;
  const int n2a = threadIdx.x % N2, ca = threadIdx.x / N2;
  if (task_a) {
#pragma unroll
    for (int k = 0; k < N1; ++k) v[k] = X[ca * Gm::S + k * N2 + n2a];
    dft_small<fx, +1, N1>(v);
  }
  __syncthreads();   // R overlays X
  if (task_a) {
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) {
      R[(2 * ca) * Gm::SR + N2 * n1 + n2a] = v[n1].x;
      R[(2 * ca + 1) * Gm::SR + N2 * n1 + n2a] = v[n1].y;
    }
  }
  __syncthreads();
  const bool plain = E > -900 && E < 900;
  auto value = [&](long long q) { return plain ? fx_to_double(fx{q}, E) : fx_to_double_far(q, E); };
  typename Epi::Acc acc[Epi::NV > 0 ? Epi::NV : 1];
#pragma unroll
  for (int j = 0; j < Epi::NV; ++j) acc[j].init((Epi::MAXMASK >> j) & 1u);
  constexpr int Q = N / 4, TOT = Gm::RY * Q;
// one step at a time: unrolled by 2 or 4, with e^s in the loop, it outgrows
// the instruction cache (public H v at 256^3: 254, 260 and 276 us)
#pragma unroll 1
  for (int e = threadIdx.x; e < TOT; e += kThreads) {
    const int row = e / Q, x = 4 * (e % Q);
    const longlong2 a = reinterpret_cast<const longlong2*>(&R[row * Gm::SR + x])[0];
    const longlong2 b = reinterpret_cast<const longlong2*>(&R[row * Gm::SR + x])[1];
    if constexpr (EpiRaw<Epi>::value)
      epi.vec4(row0 + (size_t)row * N + x, V4<fx>{{fx{a.x}, fx{a.y}, fx{b.x}, fx{b.y}}}, E, acc);
    else
      epi.vec4(row0 + (size_t)row * N + x,
             V4<double>{{value(a.x), value(a.y), value(b.x), value(b.y)}}, acc);
  }
  if constexpr (Epi::NV > 0) block_reduce_finish_acc<Epi::NV, Epi::MAXMASK>(acc, ra, fin);
}

#undef PLC_PASSX_SETUP

}  // namespace plc
