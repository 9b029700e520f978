// launch.cuh -- host launchers for the spectral pipeline and element-wise
// kernels.  Included by the per-type translation units, which instantiate
// the templates for their field types.
#pragma once

#include "ctx.h"
#include "limits.cuh"
#include "ops.cuh"
#include <type_traits>

#include "passes.cuh"
#include "passes4.cuh"
#include "passesx.cuh"

namespace plc {

template <typename T> inline const cpx<T>* twiddles(const plc_ctx* c);
template <> inline const cpx<float>* twiddles<float>(const plc_ctx* c) { return c->tw32; }
template <> inline const cpx<double>* twiddles<double>(const plc_ctx* c) { return c->tw64; }
template <typename T> inline const T* multiplier(const plc_ctx* c);
template <> inline const float* multiplier<float>(const plc_ctx* c) { return c->M32; }
template <> inline const double* multiplier<double>(const plc_ctx* c) { return c->M64; }

// Dynamic shared memory of the Stockham passes: what the largest grid (n = 512)
// needs.
template <typename T, auto Kernel> inline void set_smem(int dev) {
  set_smem4<Kernel>(dev, PassGeom<T>::smem_bytes_max(512));
}

inline RedArgs red_args(plc_ctx* c) { return RedArgs{c->partials, c->sc}; }

// The passes with register four-step line transforms (passes4.cuh) in FP32.
template <typename T, int N1, int N2, typename Pro, typename Epi, typename Fin>
void run_pipeline4(plc_ctx* c, Pro pro, Epi epi, Fin fin, int zero_dc, const int* done, int s0,
                   const T* m_override = nullptr) {
  using Gm = Geo4<T, N1, N2>;
  using C = cpx<T>;
  constexpr int n = Gm::N, h = n / 2 + 1;
  C* A = static_cast<C*>(c->specA);
  C* B = static_cast<C*>(c->specB);
  const C* tw = twiddles<T>(c);
  const T* M = m_override ? m_override : multiplier<T>(c);
  const dim3 gx(n / Gm::RY, n), gy(n / Gm::L, h);
  const int dev = current_device();
  set_smem4<k4_xf<T, N1, N2, Pro>>(dev, Gm::smem_x);
  set_smem4<k4_xi<T, N1, N2, Epi, Fin>>(dev, Gm::smem_x);
  {
    LaunchScope ls(c, Site(s0 + 0));
    k4_xf<T, N1, N2, Pro><<<gx, kThreads, Gm::smem_x, c->stream>>>(pro, A, tw, done);
  }
  // The y and z passes of a plane in one block (k4_yzy) up to 96^3: mixed MAP
  // at 32^3 904 -> 835 us, 64^3 867 -> 832, 96^3 1240 -> 1237.  At 128^3 its 65
  // planes leave half the chip idle, and a solve by itself is slower (1601 ->
  // 1645 us), but solves that share the chip gain from the traffic saved, two
  // of them already: batches of 2, 4, 8 and 16 MAPs of 128^3 2233 -> 2157, 3618
  // -> 3447, 7567 -> 7038 and 15020 -> 14110 us; 64 mocks up to 128^3 37.8 ->
  // 36.2 ms.
  auto fused = [&]() {
    if constexpr (n <= 128) {
      using Gp = GeoP<N1, N2>;
      constexpr size_t bytes = Gp::template smem<C>();
      set_smem4<k4_yzy<T, N1, N2>>(dev, bytes);
      LaunchScope ls(c, Site(s0 + 2));
      k4_yzy<T, N1, N2><<<h, Gp::kT, bytes, c->stream>>>(A, M, zero_dc, tw, done);
    }
  };
  auto three_passes = [&]() {
    if constexpr (n > 96) {
      set_smem4<k4_yf<T, N1, N2>>(dev, Gm::smem_y);
      set_smem4<k4_z<T, N1, N2>>(dev, Gm::smem_z);
      set_smem4<k4_yi<T, N1, N2>>(dev, Gm::smem_y);
      {
        LaunchScope ls(c, Site(s0 + 1));
        k4_yf<T, N1, N2><<<gy, kThreads, Gm::smem_y, c->stream>>>(A, B, tw, done);
      }
      {
        LaunchScope ls(c, Site(s0 + 2));
        k4_z<T, N1, N2><<<gy, kThreads, Gm::smem_z, c->stream>>>(B, M, zero_dc, tw, done);
      }
      {
        LaunchScope ls(c, Site(s0 + 3));
        k4_yi<T, N1, N2><<<gy, kThreads, Gm::smem_y, c->stream>>>(B, A, tw, done);
      }
    }
  };
  if (n <= 96 || (n <= 128 && c->shared_chip)) fused();
  else three_passes();
  {
    LaunchScope ls(c, Site(s0 + 4));
    k4_xi<T, N1, N2, Epi, Fin><<<gx, kThreads, Gm::smem_x, c->stream>>>(A, epi, fin, red_args(c),
                                                                        tw, done);
  }
  check(cudaGetLastError(), "spectral pipeline launch");
}

// Dispatch on the context's four-step schedule (every entry of kFourStep,
// ctx.h); false when the plan has none (Stockham stages).
template <typename T, typename Pro, typename Epi, typename Fin>
bool run_four_step(plc_ctx* c, Pro pro, Epi epi, Fin fin, int zero_dc, const int* done, int s0,
                   const T* m_override = nullptr) {
  switch (c->plan.f1 * 64 + c->plan.f2) {
    case 32 * 64 + 16: run_pipeline4<T, 32, 16>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 16 * 64 + 16: run_pipeline4<T, 16, 16>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 16 * 64 + 12: run_pipeline4<T, 16, 12>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 12 * 64 + 16: run_pipeline4<T, 12, 16>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 16 * 64 + 8: run_pipeline4<T, 16, 8>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 8 * 64 + 16: run_pipeline4<T, 8, 16>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 12 * 64 + 8: run_pipeline4<T, 12, 8>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 8 * 64 + 12: run_pipeline4<T, 8, 12>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 8 * 64 + 8: run_pipeline4<T, 8, 8>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 8 * 64 + 4: run_pipeline4<T, 8, 4>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    default: return false;
  }
}

// The FP64 passes in block fixed point (passesx.cuh).
template <int N1, int N2, typename Pro, typename Epi, typename Fin>
void run_pipelinex(plc_ctx* c, Pro pro, Epi epi, Fin fin, int zero_dc, const int* done, int s0,
                   const double* m_override) {
  using Gm = GeoX<N1, N2>;
  constexpr int n = Gm::N, h = n / 2 + 1;
  fxc* A = static_cast<fxc*>(c->specA);
  fxc* B = static_cast<fxc*>(c->specB);
  const fxw* tw = static_cast<const fxw*>(c->twfx);
  const double* M = m_override ? m_override : c->M64;
  const FxExps ex = fx_exps(c->fxexp, n);
  const dim3 gx(n / Gm::RY, n), gy(n / Gm::L, h);
  const int dev = current_device();
  set_smem4<kx_xf<N1, N2, Pro>>(dev, Gm::smem_x);
  set_smem4<kx_yf<N1, N2>>(dev, Gm::smem_y);
  set_smem4<kx_z<N1, N2>>(dev, Gm::smem_z);
  set_smem4<kx_yi<N1, N2>>(dev, Gm::smem_y);
  set_smem4<kx_xi<N1, N2, Epi, Fin>>(dev, Gm::smem_x);
  {
    LaunchScope ls(c, Site(s0 + 0));
    kx_xf<N1, N2, Pro><<<gx, kThreads, Gm::smem_x, c->stream>>>(pro, A, ex, tw, done);
  }
  {
    LaunchScope ls(c, Site(s0 + 1));
    kx_yf<N1, N2><<<gy, kThreads, Gm::smem_y, c->stream>>>(A, B, ex, tw, done);
  }
  {
    LaunchScope ls(c, Site(s0 + 2));
    kx_z<N1, N2><<<gy, kThreads, Gm::smem_z, c->stream>>>(B, ex, M, zero_dc, tw, done);
  }
  {
    LaunchScope ls(c, Site(s0 + 3));
    kx_yi<N1, N2><<<gy, kThreads, Gm::smem_y, c->stream>>>(B, A, ex, tw, done);
  }
  {
    LaunchScope ls(c, Site(s0 + 4));
    kx_xi<N1, N2, Epi, Fin><<<gx, kThreads, Gm::smem_x, c->stream>>>(A, ex, epi, fin, red_args(c),
                                                                     tw, done);
  }
  check(cudaGetLastError(), "spectral pipeline launch");
}

// False when the length has no fixed-point passes or the context's schedule is
// the Stockham stages (run_pipeline then takes the FP64 Stockham passes); any
// four-step schedule of the others runs the default factors of its length.
template <typename Pro, typename Epi, typename Fin>
bool run_fixed(plc_ctx* c, Pro pro, Epi epi, Fin fin, int zero_dc, const int* done, int s0,
               const double* m_override) {
  if (!c->plan.f1 || !fixed_length(c->n)) return false;
  switch (c->n) {
    case 256: run_pipelinex<16, 16>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 192: run_pipelinex<16, 12>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 128: run_pipelinex<16, 8>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 96: run_pipelinex<12, 8>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 64: run_pipelinex<8, 8>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    case 32: run_pipelinex<8, 4>(c, pro, epi, fin, zero_dc, done, s0, m_override); return true;
    default: return false;
  }
}

// Shared memory of the Stockham plane kernel: two planes of up to 108^2 FP32
// modes.  FP64 planes stay apart: n/2+1 blocks would leave most FP64 pipes idle.
constexpr size_t kPlaneSmem = 200 * 1024;
// Sides that take it in a solve or call by itself: public H v 33.3 -> 30.5 us at
// 72^3, 26.0 -> 21.5 at 48^3.  At 96^3 (where the Stockham schedule has to be
// asked for) 35.3 -> 37.2, and at 108^3, whose 55 blocks, one to an SM, leave two
// thirds of the chip idle, 47.5 -> 51.4, a mixed MAP 1847 -> 2000; it pays there
// beside other solves: two MAPs of 108^3 in a batch 2852 -> 2707 us, sixteen
// 16.35 -> 15.72 ms.
constexpr int kPlaneAlone = 72;

// The five passes XF -> YF -> Z -> YI -> XI on the context's stream.
template <typename T, typename Pro, typename Epi, typename Fin>
void run_pipeline(plc_ctx* c, Pro pro, Epi epi, Fin fin, int zero_dc, const int* done,
                  int sites = 0, const T* m_override = nullptr) {
  using G = PassGeom<T>;
  // site group: 0 the Hessian-vector product and public operators, 1 the
  // Newton gradient, 2 the linear-bias model
  constexpr bool k64 = sizeof(T) == 8;
  const int s0 = sites == 2   ? (k64 ? S_BXF64 : S_BXF32)
                 : sites == 1 ? (k64 ? S_GXF64 : S_GXF32)
                              : (k64 ? S_XF64 : S_XF32);
  if constexpr (sizeof(T) == 4) {
    if (run_four_step<float>(c, pro, epi, fin, zero_dc, done, s0, m_override)) return;
  } else {
    if (run_fixed(c, pro, epi, fin, zero_dc, done, s0, m_override)) return;
  }
  const int n = c->n, h = n / 2 + 1;
  const size_t sm = G::smem_bytes(c->plan);
  cpx<T>* A = static_cast<cpx<T>*>(c->specA);
  cpx<T>* B = static_cast<cpx<T>*>(c->specB);
  const cpx<T>* tw = twiddles<T>(c);
  const dim3 gx((n + G::RY - 1) / G::RY, n), gy((n + G::L - 1) / G::L, h);
  const int dev = current_device();
  set_smem<T, k_xf<T, Pro>>(dev);
  set_smem<T, k_yf<T>>(dev);
  set_smem<T, k_z<T>>(dev);
  set_smem<T, k_yi<T>>(dev);
  set_smem<T, k_xi<T, Epi, Fin>>(dev);
  {
    LaunchScope ls(c, Site(s0 + 0));
    k_xf<T, Pro><<<gx, kThreads, sm, c->stream>>>(pro, A, c->plan, tw, done);
  }
  bool plane = false;
  if constexpr (sizeof(T) == 4) {
    plane = plane_smem<T>(n) <= kPlaneSmem && (n <= kPlaneAlone || c->shared_chip);
    if (plane) {
      set_smem4<k_yzy<T>>(dev, kPlaneSmem);
      LaunchScope ls(c, Site(s0 + 2));
      k_yzy<T><<<h, kPlaneThreads, plane_smem<T>(n), c->stream>>>(
          A, m_override ? m_override : multiplier<T>(c), zero_dc, c->plan, tw, done);
    }
  }
  if (!plane) {
    {
      LaunchScope ls(c, Site(s0 + 1));
      k_yf<T><<<gy, kThreads, sm, c->stream>>>(A, B, c->plan, tw, done);
    }
    {
      LaunchScope ls(c, Site(s0 + 2));
      k_z<T><<<gy, kThreads, sm, c->stream>>>(B, m_override ? m_override : multiplier<T>(c), zero_dc,
                                              c->plan, tw, done);
    }
    {
      LaunchScope ls(c, Site(s0 + 3));
      k_yi<T><<<gy, kThreads, sm, c->stream>>>(B, A, c->plan, tw, done);
    }
  }
  {
    LaunchScope ls(c, Site(s0 + 4));
    k_xi<T, Epi, Fin><<<gx, kThreads, sm, c->stream>>>(A, epi, fin, red_args(c), c->plan, tw, done);
  }
  check(cudaGetLastError(), "spectral pipeline launch");
}

template <typename T> void prior_apply(plc_ctx* c, const T* x, T* y) {
  run_pipeline<T>(c, ProLoad<T>{x}, EpiStore<T>{y}, FinNone{}, 0, nullptr);
}

template <typename T> void hessvec_s(plc_ctx* c, const T* s, const T* w, double nbar,
                                     const T* v, T* out) {
  run_pipeline<T>(c, ProLoad<T>{v}, EpiHessS<T>{s, w, (T)nbar, v, out}, FinNone{}, 0, nullptr);
}

template <typename T> void grad_public(plc_ctx* c, const T* s, const T* w, const int32_t* N,
                                       double nbar, T* g) {
  run_pipeline<T>(c, ProShift<T, T>{s, c->mu},
                  EpiGrad<T, T, T, T, 2>{s, w, N, nbar, c->mu, nullptr, g, nullptr, nullptr,
                                         c->jac_c, 0},
                  FinStore<2>{}, 0, nullptr, true);
}

template <typename T, typename TS, typename TC>
void grad_newton(plc_ctx* c, const TS* s, const double* w, const int32_t* N, double nbar, T* y,
                 T* g, TC* D, TC* r, bool jac) {
  if constexpr (std::is_same<T, double>::value && std::is_same<TC, float>::value) {
    // the FP64 gradient of the mixed solve: fixed-point transforms and a
    // float-float epilogue where the length has fixed-point passes
    const EpiGradFF<true> epi{s, w, N, ff(nbar), ff(c->mu), y, g, D, r, (float)c->jac_c,
                              jac ? 1 : 0, static_cast<const ff*>(c->expff)};
    if (run_fixed(c, ProShift<double, double>{s, c->mu}, epi, FinGrad<6>{}, 0, nullptr, S_GXFF,
                  nullptr))
      return;
  }
  constexpr int NS = sizeof(TC) == 8 ? 5 : 6;
  run_pipeline<T>(c, ProShift<T, TS>{s, c->mu},
                  EpiGrad<T, TS, double, TC, NS>{s, w, N, nbar, c->mu, y, g, D, r, c->jac_c,
                                                 jac ? 1 : 0},
                  FinGrad<NS>{}, 0, nullptr, true);
}

// The sums of the FP64 gradient of the mixed solve at an FP64 s (the
// same pipeline with nothing stored: the sums of -ln P and ||g||^2 into
// sc->red, FinGrad), for a stopping test that may end the solve before the
// gradient's fields are needed.  False (nothing run)
// where run_fixed has none.
inline bool grad_sums_ff_impl(plc_ctx* c, const double* s, const double* w, const int32_t* N,
                              double nbar, bool jac) {
  const EpiGradFF<false> epi{s, w, N, ff(nbar), ff(c->mu), nullptr, nullptr, nullptr, nullptr,
                             (float)c->jac_c, jac ? 1 : 0, static_cast<const ff*>(c->expff)};
  return run_fixed(c, ProShift<double, double>{s, c->mu}, epi, FinGrad<3>{}, 0, nullptr, S_GXFF,
                   nullptr);
}

template <typename T, typename TS, typename TC>
void grad_newton_g(plc_ctx* c, const TS* delta, const double* w, const int32_t* N, double nbar,
                   T* y, T* g, TC* D, TC* r, bool jac) {
  run_pipeline<T>(c, ProShift<T, TS>{delta, 0.0},
                  EpiGradG<T, TS, TC>{delta, w, N, nbar, y, g, D, r, c->jac_c, jac ? 1 : 0},
                  FinGrad<6>{}, 0, nullptr, true);
}

// The field the CG's Jacobi products read: D for FP32, the stored M^-1
// (precond) for FP64.
template <typename T> inline const T* precond_field(const plc_ctx* c, const T* D) {
  if constexpr (sizeof(T) == 8) return static_cast<const T*>(c->wf[plc_ctx::kPrecondField]);
  else return D;
}

template <typename T> void cg_hv(plc_ctx* c, const T* r, const T* D, T* p, T* Hp, bool jac) {
  const int* done = &c->sc->done;
  if (jac)
    run_pipeline<T>(c, ProCgDir<T, true>{r, precond_field<T>(c, D), (T)c->jac_c, p, c->sc},
                    EpiHessD<T>{D, p, Hp}, FinAlpha{}, 0, done);
  else
    run_pipeline<T>(c, ProCgDir<T, false>{r, D, (T)c->jac_c, p, c->sc},
                    EpiHessD<T>{D, p, Hp}, FinAlpha{}, 0, done);
}

template <typename TL> void vjp_amplitude(plc_ctx* c, const double* s, const TL* lam) {
  run_pipeline<double>(c, ProShift<double, double>{s, c->mu}, EpiDot<double, TL>{lam},
                       FinStore<1>{}, 1, nullptr);
}

inline int pw_blocks(plc_ctx* c) { return pointwise_blocks((long long)c->n3(), c->sms); }

template <typename T, typename TC>
void newton_update_g(plc_ctx* c, const T* s, const T* y, const T* g, const TC* r, const TC* xi,
                     const TC* D, const int32_t* N, const double* w, double nbar, double tau,
                     bool jac, T* s2, T* y2, T* g2, TC* D2, TC* r2) {
  LaunchScope ls(c, sizeof(T) == 4 ? S_NEWTON_UPDATE32 : S_NEWTON_UPDATE64);
  k_newton_update_g<T, TC><<<pw_blocks(c), kThreads, 0, c->stream>>>(
      s, y, g, r, xi, D, N, w, nbar, tau, c->jac_c, jac ? 1 : 0, s2, y2, g2, D2, r2, c->n3(),
      red_args(c));
  check(cudaGetLastError(), "k_newton_update_g");
}

template <typename T, typename TC>
void boundary_step(plc_ctx* c, const T* delta, const TC* xi, const int32_t* N) {
  LaunchScope ls(c, S_BOUNDARY);
  k_boundary<T, TC><<<pw_blocks(c), kThreads, 0, c->stream>>>(delta, xi, N, c->n3(), red_args(c));
  check(cudaGetLastError(), "k_boundary");
}


template <typename TC> void cg_init(plc_ctx* c, const double* b, const TC* D, TC* r, bool jac) {
  const int nb = pw_blocks(c);
  LaunchScope ls(c, S_CG_INIT);
  if (jac)
    k_cg_init<TC, double, true><<<nb, kThreads, 0, c->stream>>>(b, D, (TC)c->jac_c, r, c->n3(),
                                                                 red_args(c));
  else
    k_cg_init<TC, double, false><<<nb, kThreads, 0, c->stream>>>(b, D, (TC)c->jac_c, r, c->n3(),
                                                                  red_args(c));
  check(cudaGetLastError(), "k_cg_init");
}

template <typename TC> void lsq_init(plc_ctx* c, const int32_t* N, const double* w, double nbar,
                                     TC* D, TC* r, bool jac) {
  const int nb = pw_blocks(c);
  LaunchScope ls(c, S_CG_INIT);
  if (jac)
    k_lsq_init<TC, true><<<nb, kThreads, 0, c->stream>>>(N, w, nbar, (TC)c->jac_c, D, r,
                                                         c->n3(), red_args(c));
  else
    k_lsq_init<TC, false><<<nb, kThreads, 0, c->stream>>>(N, w, nbar, (TC)c->jac_c, D, r,
                                                          c->n3(), red_args(c));
  check(cudaGetLastError(), "k_lsq_init");
}

template <typename TC> void precond(plc_ctx* c, const TC* D, const TC* r, bool jac) {
  if constexpr (sizeof(TC) == 8) {
    if (!jac) return;
    LaunchScope ls(c, S_CG_INIT);
    k_precond<TC><<<pw_blocks(c), kThreads, 0, c->stream>>>(
        D, r, (TC)c->jac_c, static_cast<TC*>(c->wf[plc_ctx::kPrecondField]), c->n3(), red_args(c));
    check(cudaGetLastError(), "k_precond");
  }
}

template <typename TC> void cg_update(plc_ctx* c, TC* x, TC* r, const TC* p, const TC* Hp,
                                      const TC* D, bool jac, double rtol2, int max_iter,
                                      const LoopCtl& loop) {
  // one wave (FP32: 4 blocks of 256 per SM at its 56 registers, 73.8 us
  // against 77.1 with two waves at 256^3)
  const int nb = pointwise_blocks((long long)c->n3(), c->sms, sizeof(TC) == 8 ? 3 : 4);
  LaunchScope ls(c, sizeof(TC) == 4 ? S_CG_UPDATE32 : S_CG_UPDATE64);
  if (jac)
    k_cg_update<TC, true><<<nb, kThreads, 0, c->stream>>>(x, r, p, Hp, precond_field<TC>(c, D),
                                                           (TC)c->jac_c, c->n3(), red_args(c),
                                                           rtol2, max_iter, loop);
  else
    k_cg_update<TC, false><<<nb, kThreads, 0, c->stream>>>(x, r, p, Hp, D, (TC)c->jac_c, c->n3(),
                                                            red_args(c), rtol2, max_iter, loop);
  check(cudaGetLastError(), "k_cg_update");
}

template <typename T, typename TC>
void newton_update(plc_ctx* c, const T* s, const T* y, const T* g, const TC* r, const TC* xi,
                   const TC* D, const int32_t* N, const double* w, double nbar, double tau,
                   bool jac, T* s2, T* y2, T* g2, TC* D2, TC* r2, const double* tau_dev,
                   const LoopCtl& loop) {
  // g may be left out only where forming it again from y, D and N is exact
  if (!g && !std::is_same<T, TC>::value) check(cudaErrorInvalidValue, "newton_update without g");
  LaunchScope ls(c, sizeof(T) == 4 ? S_NEWTON_UPDATE32 : S_NEWTON_UPDATE64);
  k_newton_update<T, TC><<<pw_blocks(c), kThreads, 0, c->stream>>>(
      s, y, g, r, xi, D, N, w, nbar, c->mu, tau, tau_dev, c->jac_c, jac ? 1 : 0, s2, y2, g2, D2, r2,
      c->n3(), red_args(c), loop);
  check(cudaGetLastError(), "k_newton_update");
}

template <typename TS> void diag_start(plc_ctx* c, TS* s, const int32_t* N, const double* w,
                                       double nbar) {
  LaunchScope ls(c, S_SETUP);
  k_diag_start<TS><<<pw_blocks(c), kThreads, 0, c->stream>>>(
      s, N, w, (float)nbar, (float)c->mu, (float)c->prior_var, c->n3());
  check(cudaGetLastError(), "k_diag_start");
}

template <typename TS> void diag_start_g(plc_ctx* c, TS* delta, const int32_t* N, const double* w,
                                         double nbar) {
  LaunchScope ls(c, S_SETUP);
  k_diag_start_g<TS><<<pw_blocks(c), kThreads, 0, c->stream>>>(delta, N, w, (float)nbar,
                                                              (float)c->prior_var, c->n3());
  check(cudaGetLastError(), "k_diag_start_g");
}

template <typename TC> void diag(plc_ctx* c, const double* s, const double* w, double nbar, TC* D) {
  LaunchScope ls(c, S_DIAG);
  k_diag<TC><<<pw_blocks(c), kThreads, 0, c->stream>>>(s, w, nbar, D, c->n3());
  check(cudaGetLastError(), "k_diag");
}

template <typename TD, typename TS> void convert(plc_ctx* c, const TS* src, TD* dst) {
  LaunchScope ls(c, S_CONVERT);
  k_convert<TD, TS><<<pw_blocks(c), kThreads, 0, c->stream>>>(src, dst, c->n3());
  check(cudaGetLastError(), "k_convert");
}

}  // namespace plc
