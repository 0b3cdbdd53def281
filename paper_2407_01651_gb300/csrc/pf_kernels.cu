// pf_kernels.cu -- sm_103a support kernels of the coupled lattice Boltzmann step
// of the gas-liquid-dendrite phase-field model (arXiv 2407.01651); the step
// itself is in pf_step.cu:
//   k_init_spec initial fields from seeds and bubbles, equilibrium populations
//   k_set_fields equilibrium populations from given macroscopic fields
//   k_reduce, k_reduce_thermal, k_rho_bar  FP64 sums (conservation, centroid,
//               Laplace probe, mean density)
//   k_*_state   raw state to / from FP64
//
// Layout: structure of arrays, one plane per population / scalar, x fastest,
// periodic domains concatenated in every plane.
#include "pf_internal.h"
#include "pf_site.cuh"
#include "pf_reduce.cuh"

#include <cuda_fp16.h>
#include <cuda_bf16.h>

#include <algorithm>

namespace pf {

// ---------------------------------------------------------------------------
// Initialisation
// ---------------------------------------------------------------------------
// Minimum-image offset; fmod(d, L) == d whenever |d| < L, so it is only taken
// for offsets of a whole period or more.
__device__ __forceinline__ double min_image(double d, double L) {
  if (d <= -L || d >= L) d = fmod(d, L);
  if (d < -0.5 * L) d += L;
  if (d >= 0.5 * L) d -= L;
  return d;
}

// Temperature lattice of one site at equilibrium (thermal mode): H =
// c_p [theta - (c_p^s/c_p) h(psi)], e = g^eq(rho H, theta, rho H v) of
// Appendix B (axis base rounded as in the collision), and the lagged dendrite
// source at its pointwise part Q_psi(theta) / F(U).
template <typename S, typename R>
__device__ void write_thermal(S* out, R* aout, R* fields, long long ps, long long site, R phi,
                              R psi, R U, R vx, R vy, R theta, const KParams<R>& kp) {
  const R rho = kp.rho_g + phi * kp.drho;
  const R H = kp.th_cp * (theta - kp.th_lh * (R(1) + psi));
  const R m0 = rho * H;
  const R b = th_base(m0, theta);
  st<S, R>(out + (P_E + 0) * ps, site, m0);
  st<S, R>(out + (P_E + 1) * ps, site, b);
  st<S, R>(out + (P_E + 2) * ps, site, b + R(0.5) * (m0 * vx));
  st<S, R>(out + (P_E + 3) * ps, site, b + R(0.5) * (m0 * vy));
  const R omp2 = R(1) - psi * psi, ophi = R(1) - phi;
  const R Q = kp.four_bpsi * psi * omp2 - kp.two_bint * ophi * ophi * (R(1) + psi) -
              kp.lam * omp2 * omp2 * (theta + kp.Mcinf * U);
  const R F = kp.th_iLe + kp.Mcinf * (R(1) + (R(1) - kp.k) * U);
  aout[A_QO * ps + site] = Q / F;
  if (fields) fields[FLD_THETA * ps + site] = theta;
}

// Offset along an axis: minimum image on a periodic axis, plain otherwise.
__device__ __forceinline__ double axis_offset(double d, double L, bool periodic) {
  return periodic ? min_image(d, L) : d;
}

// Write the equilibrium state and the fields of one site.
template <typename S, typename R>
__device__ void write_equilibrium(S* out, R* aout, R* fields, long long ps, long long site,
                                  double phi_d, double psi_d, double C_d, double vx_d,
                                  double vy_d, double p_d, const KParams<R>& kp, int thermal,
                                  double theta_d) {
  const R phi = static_cast<R>(phi_d), psi = static_cast<R>(psi_d), C = static_cast<R>(C_d);
  const R vx = static_cast<R>(vx_d), vy = static_cast<R>(vy_d), p = static_cast<R>(p_d);
  const R omk = R(1) - kp.k;
  const R U = (R(2) * C / (R(1) + kp.k - omk * psi) - R(1)) / omk;
  const R omp2 = R(1) - psi * psi;
  const R ophi = R(1) - phi;
  SiteOut<R> o;
  feq_ns(p, kp.rho_g + phi * kp.drho, vx, vy, o.f);
  // CAC h_eq = w_i phi (1 + 3 c.v); dendrite w_i psi; solute w_i C (1 + 3 c.v)
  o.hA = (w9<R>(1) * phi * R(3)) * vec2(vx, vy);
  o.hD = (w9<R>(5) * phi * R(3)) * vec2(vx + vy, vy - vx);
  o.g = vec2(R(0), R(0));
  o.F = R(0);
  o.s = (w5<R>(1) * C * R(3)) * vec2(vx, vy);
  R g[5];
  for (int i = 0; i < 5; ++i) g[i] = w5<R>(i) * psi;
  o.ias2 = R(1);
  o.phi = phi;
  o.psi = psi;
  o.C = C;
  o.vx = vx;
  o.vy = vy;
  o.Q = kp.four_bpsi * psi * omp2 - kp.two_bint * ophi * ophi * (R(1) + psi) -
        kp.lam * omp2 * omp2 * (kp.theta + kp.Mcinf * U);
  StepArgs<S, R> to{};
  to.out = out;
  to.aout = aout;
  to.plane_stride = ps;
  store_state<S, R>(to, (unsigned)site, o, g);
  if (fields) {
    fields[FLD_PHI * ps + site] = phi;
    fields[FLD_PSI * ps + site] = psi;
    fields[FLD_C * ps + site] = C;
    fields[FLD_U * ps + site] = U;
    fields[FLD_P * ps + site] = p;
    fields[FLD_VX * ps + site] = vx;
    fields[FLD_VY * ps + site] = vy;
    fields[FLD_MU * ps + site] = R(0);
    fields[FLD_THETA * ps + site] = kp.theta;
  }
  if (thermal) write_thermal<S, R>(out, aout, fields, ps, site, phi, psi, U, vx, vy,
                                   static_cast<R>(theta_d), kp);
}

template <typename S, typename R>
__global__ void k_init_spec(InitArgs<S, R> a) {
  const DomDesc d = a.dom;
  const long long n = (long long)d.nx * d.ny;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % d.nx), y = (int)(i / d.nx);
    // tanh of an argument beyond +-30 is exactly +-1 in FP64, so objects that
    // far away are not evaluated (identical result, ~100x fewer tanh).
    const double seed_far = a.R_s + 30.0 * a.W0 / a.sq2bpsi;
    double psi = -1.0, best = 0.0;
    int gid = 0;
    for (int s = 0; s < a.n_seeds; ++s) {
      const double dx = axis_offset((double)x - a.seeds[3 * s], (double)d.nx, d.bc[0] == 0);
      const double dy = axis_offset((double)y - a.seeds[3 * s + 1], (double)d.ny, d.bc[2] == 0);
      const double r2 = dx * dx + dy * dy;
      const double v = r2 > seed_far * seed_far
                           ? -1.0
                           : tanh(a.sq2bpsi * (a.R_s - sqrt(r2)) / a.W0);
      if (s == 0 || v > psi) psi = v;
      if (s == 0 || r2 < best) {
        best = r2;
        gid = s;
      }
    }
    double phi = 1.0;
    for (int b = 0; b < a.n_bub; ++b) {
      const double dx = axis_offset((double)x - a.bubbles[3 * b], (double)d.nx, d.bc[0] == 0);
      const double dy = axis_offset((double)y - a.bubbles[3 * b + 1], (double)d.ny, d.bc[2] == 0);
      const double r2 = dx * dx + dy * dy;
      const double far = a.bubbles[3 * b + 2] + 60.0 * a.Wphi / a.sq2bphi;
      const double v =
          r2 > far * far ? 1.0
                         : 0.5 + 0.5 * tanh(a.sq2bphi * (sqrt(r2) - a.bubbles[3 * b + 2]) /
                                            (2.0 * a.Wphi));
      if (b == 0 || v < phi) phi = v;
    }
    const double C = phi * (1.0 - (1.0 - a.k) * 0.5 * (1.0 + psi));
    const long long site = d.off + i;
    a.grain[site] = (uint8_t)gid;
    write_equilibrium<S, R>(a.out, a.aout, a.fields, a.plane_stride, site, phi, psi, C, 0.0,
                            0.0, 0.0, a.kp, a.thermal, a.theta0);
  }
}

template <typename S, typename R>
__global__ void k_set_fields(SetFieldsArgs<S, R> a) {
  const DomDesc d = a.dom;
  const long long n = (long long)d.nx * d.ny;
  const long long hi = a.i1 > 0 ? a.i1 : n;
  for (long long i = a.i0 + blockIdx.x * (long long)blockDim.x + threadIdx.x; i < hi;
       i += (long long)gridDim.x * blockDim.x) {
    const long long site = d.off + i;
    const double* F = a.f6;
    const double v0 = F[i], v1 = F[n + i], v2 = F[2 * n + i], v3 = F[3 * n + i],
                 v4 = F[4 * n + i], v5 = F[5 * n + i];
    // the host reads this bit after the launch and rejects the fields
    if (!isfinite(v0) || !isfinite(v1) || !isfinite(v2) || !isfinite(v3) || !isfinite(v4) ||
        !isfinite(v5))
      atomicOr(a.err, ERR_NONFINITE_INPUT);
    write_equilibrium<S, R>(a.out, a.aout, a.fields, a.plane_stride, site, v0, v1, v2, v3, v4,
                            v5, a.kp, a.thermal, a.theta0);
    a.grain[site] = a.grain_ids ? a.grain_ids[i] : (uint8_t)0;
  }
}

// Thermal mode: the temperature lattice of a domain at equilibrium for a given
// theta field, with phi, psi, U and v taken from the field planes (the state
// written by the last initialisation).
template <typename S, typename R>
__global__ void k_set_temperature(S* out, R* aout, R* fields, long long ps, DomDesc d,
                                  const double* __restrict__ theta, KParams<R> kp) {
  const long long n = (long long)d.nx * d.ny;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const long long site = d.off + i;
    write_thermal<S, R>(out, aout, fields, ps, site, fields[FLD_PHI * ps + site],
                        fields[FLD_PSI * ps + site], fields[FLD_U * ps + site],
                        fields[FLD_VX * ps + site], fields[FLD_VY * ps + site],
                        static_cast<R>(theta[i]), kp);
  }
}

// ---------------------------------------------------------------------------
// Raw state / fields conversion to and from FP64.
// ---------------------------------------------------------------------------
// Raw state of one site <-> the 39 physical planes (f, h, g_pre, g_post, r,
// s, phi, C, vx, vy, Q_psi), every population of a pair, in FP64.  In the
// offset forms a population stored at site x is relative to the lagged moment
// of x itself.  Thermal mode adds planes 39..43 (e_0..e_4) and 44 (H of the last
// step).  A state taken out and put back gives the same stored values: the
// stored populations and the densities pass through unchanged, and the density
// of a lattice without a plane of its own (g_post, e) is the FP64 sum of its
// populations in sum5's order, of which the rest one is written as density
// minus the others (exact).
__device__ __forceinline__ double sum_pairs5(const double (&v)[5]) {
  return (v[1] + v[3]) + (v[2] + v[4]);
}
__device__ __forceinline__ double sum5(const double (&v)[5]) { return sum_pairs5(v) + v[0]; }

// tied: the populations of the pair-stored lattices are those of the tied planes
// (a raw state), else those the pairs stand for.
template <typename S, typename R>
__global__ void k_state_to_f64(const S* __restrict__ pin, const R* __restrict__ ain, long long ps,
                               long long off, long long n, double* __restrict__ out,
                               int thermal, double rho_g, double drho, const S* __restrict__ tied) {
  constexpr bool offs = Codec<S>::kOffset;
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x) {
    const long long s = off + j;
    auto pop = [&](int k) { return pin[k * ps + s]; };
    // stored and opposite population of a pair with this base
    auto plus = [&](S v, R base) {
      return offs ? (double)base + (double)dec_off<S, R>(v, R(0)) : (double)pair_p<S, R>(v, base);
    };
    auto minus = [&](S v, R base) {
      return offs ? (double)base - (double)dec_off<S, R>(v, R(0)) : (double)pair_m<S, R>(v, base);
    };
    const R phio = ain[A_PHIO * ps + s], Co = ain[A_CO * ps + s];
    const R psio = offs ? ain[A_PSIO * ps + s] : R(0);
    for (int i = 0; i < 9; ++i) out[(X_F + i) * n + j] = (double)pop_ns<S, R>(pin + (P_F + i) * ps, s);
    for (int i = 0; i < 5; ++i)
      out[(X_GPRE + i) * n + j] = (double)pop_off<S, R>(pin + (P_GPRE + i) * ps, s, w5<R>(i) * psio);
    out[X_RR * n + j] = (double)ain[A_RR * ps + s];
    out[X_PHI * n + j] = (double)phio;
    out[X_C * n + j] = (double)Co;
    out[X_VX * n + j] = (double)ain[A_VXO * ps + s];
    out[X_VY * n + j] = (double)ain[A_VYO * ps + s];
    out[X_Q * n + j] = (double)ain[A_QO * ps + s];
    if (tied) {
      auto off_of = [&](int k, R wm) { return (double)dec_off<S, R>(tied[k * n + j], wm); };
      for (int i = 0; i < 9; ++i) out[(X_H + i) * n + j] = off_of(T_H + i, w9<R>(i) * phio);
      for (int i = 0; i < 5; ++i) {
        out[(X_GPOST + i) * n + j] = off_of(T_GPOST + i, w5<R>(i) * psio);
        out[(X_S + i) * n + j] = off_of(T_S + i, w5<R>(i) * Co);
      }
      if (thermal) {
        for (int i = 0; i < 5; ++i) out[(X_E + i) * n + j] = (double)(R)tied[(T_E + i) * n + j];
        out[X_HO * n + j] = (double)(R)tied[T_HO * n + j];
      }
      continue;
    }
    const CacBase<R> b(phio);
    out[X_H * n + j] = (double)b.rest(phio);
    for (int i = 1; i < 9; ++i) {
      const R base = i < 5 ? b.axis : b.diag();
      const S v = pop(P_H + pair9(i));
      out[(X_H + i) * n + j] = minus9(i) ? minus(v, base) : plus(v, base);
    }
    {
      // density m; in the offset forms psi_o + F with F/6 in the first plane
      const double f6 = offs ? (double)dec_off<S, R>(pop(P_GPOST), R(0)) : 0.0;
      const R m = offs ? psio : (R)Codec<S>::template dec<R>(pop(P_GPOST));
      const R base = q5_base(m);
      double g[5];
      for (int i = 1; i < 3; ++i) {
        const S v = pop(P_GPOST + i);
        g[i] = plus(v, base);
        g[i + 2] = minus(v, base) + 2.0 * f6;
      }
      g[0] = ((double)m + 6.0 * f6) - sum_pairs5(g);
      for (int i = 0; i < 5; ++i) out[(X_GPOST + i) * n + j] = g[i];
    }
    {
      const R base = q5_base(Co);
      out[X_S * n + j] = (double)q5_rest(Co, base);
      for (int i = 1; i < 3; ++i) {
        const S v = pop(P_S + i - 1);
        out[(X_S + i) * n + j] = plus(v, base);
        out[(X_S + i + 2) * n + j] = minus(v, base);
      }
    }
    if (thermal) {
      const R m = Codec<S>::template dec<R>(pop(P_E)), base = Codec<S>::template dec<R>(pop(P_E + 1));
      double e[5];
      for (int i = 1; i < 3; ++i) {
        e[i] = plus(pop(P_E + 1 + i), base);
        e[i + 2] = minus(pop(P_E + 1 + i), base);
      }
      e[0] = (double)m - sum_pairs5(e);
      for (int i = 0; i < 5; ++i) out[(X_E + i) * n + j] = e[i];
      out[X_HO * n + j] = (double)m / (rho_g + (double)phio * drho);
    }
  }
}

// Sets *flag where the populations are not a collision's output to rounding (4
// ulp of the pair's size in FP32 arithmetic, 16 in FP64): the state is then kept
// with all of them (pf_raw.cuh).
template <typename R>
__global__ void k_state_general(long long n, const double* __restrict__ in, int thermal,
                                double rho_g, double drho, unsigned int* flag) {
  constexpr double tol = sizeof(R) == 8 ? 16.0 * 2.220446049250313e-16 : 4.0 * 1.1920928955078125e-7;
  bool general = false;
  // a and b are equal to rounding on the scale of their parts
  auto same = [&](double a, double b, double size) {
    if (!(fabs(a - b) <= tol * size)) general = true;
  };
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x) {
    auto x = [&](int k) { return in[k * n + j]; };
    const R phio = (R)x(X_PHI), Co = (R)x(X_C);
    {
      const CacBase<R> b(phio);
      double size = fabs(x(X_PHI));
      for (int i = 0; i < 9; ++i) size = fmax(size, fabs(x(X_H + i)));
      same(x(X_H), (double)b.rest(phio), size);
      for (int i : {1, 2, 5, 6})
        same(x(X_H + i) + x(X_H + i + 2), 2.0 * (double)(i < 5 ? b.axis : b.diag()), size);
    }
    {
      double g[5], size = 0.0;
      for (int i = 0; i < 5; ++i) {
        g[i] = x(X_GPOST + i);
        size = fmax(size, fabs(g[i]));
      }
      const double m = sum5(g);
      same(g[1] + g[3], m / 3.0, 2.0 * size);
      same(g[2] + g[4], m / 3.0, 2.0 * size);
    }
    {
      const R base = q5_base(Co);
      double size = fabs(x(X_C));
      for (int i = 0; i < 5; ++i) size = fmax(size, fabs(x(X_S + i)));
      same(x(X_S), (double)q5_rest(Co, base), size);
      for (int i = 1; i < 3; ++i) same(x(X_S + i) + x(X_S + i + 2), 2.0 * (double)base, size);
    }
    if (thermal) {
      double e[5], size = 0.0;
      for (int i = 0; i < 5; ++i) {
        e[i] = x(X_E + i);
        size = fmax(size, fabs(e[i]));
      }
      const double md = sum5(e), rhoH = (rho_g + x(X_PHI) * drho) * x(X_HO);
      const R m = (R)md, b = round_to_multiple((R)(0.5 * (e[1] + e[3])), quantum_quarter_ulp(m));
      same(e[1] + e[3], 2.0 * (double)b, 2.0 * size);
      same(e[2] + e[4], 2.0 * (double)b, 2.0 * size);
      same(md, rhoH, 2.0 * size);
    }
  }
  if (general) atomicOr(flag, 1u);
}

// tied: also the tied planes of a raw state.
template <typename S, typename R>
__global__ void k_state_from_f64(S* __restrict__ pout, R* __restrict__ aout, long long ps,
                                 long long off, long long n, const double* __restrict__ in,
                                 int thermal, S* __restrict__ tied) {
  constexpr bool offs = Codec<S>::kOffset;
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x) {
    const long long s = off + j;
    auto x = [&](int k) { return in[k * n + j]; };
    auto put = [&](int k, double v, R base) {
      if constexpr (offs) pout[k * ps + s] = enc_off<S, R>((R)(v - (double)base), R(0));
      else pout[k * ps + s] = Codec<S>::template enc<R>((R)v);
    };
    const R phio = (R)x(X_PHI), Co = (R)x(X_C);
    R psio = R(0);  // psi of the last step = sum of g_pre
    for (int i = 0; i < 5; ++i) psio += (R)x(X_GPRE + i);
    for (int i = 0; i < 9; ++i) st_ns<S, R>(pout + (P_F + i) * ps, s, (R)x(X_F + i));
    {
      const CacBase<R> b(phio);
      for (int i : {1, 2, 5, 6}) put(P_H + pair9(i), x(X_H + i), i < 5 ? b.axis : b.diag());
    }
    for (int i = 0; i < 5; ++i)
      st_off<S, R>(pout + (P_GPRE + i) * ps, s, (R)x(X_GPRE + i), w5<R>(i) * psio);
    {
      double g[5];
      for (int i = 0; i < 5; ++i) g[i] = x(X_GPOST + i);
      const double m = sum5(g);
      if constexpr (offs) {
        const R base = q5_base(psio);
        pout[P_GPOST * ps + s] = enc_off<S, R>((R)((m - (double)psio) / 6.0), R(0));
        put(P_GPOST + 1, g[1], base);
        put(P_GPOST + 2, g[2], base);
      } else {
        put(P_GPOST, m, R(0));
        put(P_GPOST + 1, g[1], R(0));
        put(P_GPOST + 2, g[2], R(0));
      }
    }
    for (int i = 1; i < 3; ++i) put(P_S + i - 1, x(X_S + i), q5_base(Co));
    aout[A_RR * ps + s] = (R)x(X_RR);
    aout[A_PHIO * ps + s] = phio;
    aout[A_CO * ps + s] = Co;
    aout[A_VXO * ps + s] = (R)x(X_VX);
    aout[A_VYO * ps + s] = (R)x(X_VY);
    aout[A_QO * ps + s] = (R)x(X_Q);
    if constexpr (offs) aout[A_PSIO * ps + s] = psio;
    if (thermal) {
      double e[5];
      for (int i = 0; i < 5; ++i) e[i] = x(X_E + i);
      const R m = (R)sum5(e);
      st<S, R>(pout + (P_E + 0) * ps, s, m);
      st<S, R>(pout + (P_E + 1) * ps, s,
               round_to_multiple((R)(0.5 * (e[1] + e[3])), quantum_quarter_ulp(m)));
      st<S, R>(pout + (P_E + 2) * ps, s, (R)e[1]);
      st<S, R>(pout + (P_E + 3) * ps, s, (R)e[2]);
    }
    if (!tied) continue;
    for (int i = 0; i < 9; ++i) tied[(T_H + i) * n + j] = enc_off<S, R>((R)x(X_H + i), w9<R>(i) * phio);
    for (int i = 0; i < 5; ++i) {
      tied[(T_GPOST + i) * n + j] = enc_off<S, R>((R)x(X_GPOST + i), w5<R>(i) * psio);
      tied[(T_S + i) * n + j] = enc_off<S, R>((R)x(X_S + i), w5<R>(i) * Co);
    }
    if (thermal) {
      for (int i = 0; i < 5; ++i) st<S, R>(tied + (T_E + i) * n, j, (R)x(X_E + i));
      st<S, R>(tied + T_HO * n, j, (R)x(X_HO));
    }
  }
}

// The temperature planes of the tied ones from the stored state (after
// pf_set_temperature rewrote that).
template <typename S, typename R>
__global__ void k_tied_temperature(const S* __restrict__ pin, const R* __restrict__ ain,
                                   long long ps, long long off, long long n,
                                   S* __restrict__ tied, double rho_g, double drho) {
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x) {
    const long long s = off + j;
    const R m = ld<R>(pin + P_E * ps, s), b = ld<R>(pin + (P_E + 1) * ps, s);
    const R e1 = ld<R>(pin + (P_E + 2) * ps, s), e2 = ld<R>(pin + (P_E + 3) * ps, s);
    st<S, R>(tied + T_E * n, j, q5_rest(m, b));
    st<S, R>(tied + (T_E + 1) * n, j, e1);
    st<S, R>(tied + (T_E + 2) * n, j, e2);
    st<S, R>(tied + (T_E + 3) * n, j, fma(R(2), b, -e1));
    st<S, R>(tied + (T_E + 4) * n, j, fma(R(2), b, -e2));
    st<S, R>(tied + T_HO * n, j, (R)((double)m / (rho_g + (double)ain[A_PHIO * ps + s] * drho)));
  }
}

template <typename R>
__global__ void k_fields_to_f64(const R* __restrict__ fields, long long ps, long long off,
                                long long n, uint32_t mask, double* __restrict__ out) {
  int sel[N_FIELDS];
  int ns = 0;
  for (int f = 0; f < N_FIELDS; ++f)
    if (mask & (1u << f)) sel[ns++] = f;
  const long long tot = n * ns;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot;
       i += (long long)gridDim.x * blockDim.x) {
    const long long q = i / n, j = i % n;
    out[i] = static_cast<double>(fields[sel[q] * ps + off + j]);
  }
}

// ---------------------------------------------------------------------------
// FP64 reductions: each block writes one record of partial sums, the block
// that finishes last adds them in a fixed order (pf_reduce.cuh), so that a
// reduction is one launch.
// ---------------------------------------------------------------------------
// out: NDIAG diagnostics, then the device error bits.  Diagnostics cost FP64
// instructions, of which this GPU retires few: the site's row and column come
// from one 32-bit division, and the speed's square root is taken once, of the
// largest square (the square root is monotone and correctly rounded).
template <typename R>
__global__ void __launch_bounds__(RED_THREADS) k_reduce(ReduceArgs<R> a, double* __restrict__ partial,
                                                        double* __restrict__ out,
                                                        unsigned int* __restrict__ ctr,
                                                        const unsigned int* __restrict__ err) {
  double acc[NDIAG];
#pragma unroll
  for (int q = 0; q < NDIAG; ++q) acc[q] = 0.0;
  const DomDesc d = a.dom;
  const long long n = (long long)d.nx * d.ny;   // at most 2^32
  const long long ps = a.plane_stride;
  const double Rin = a.Rp - 2.0 * a.W, Rout = a.Rp + 4.0 * a.W;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const long long site = d.off + i;
    const double phi = (double)a.fields[FLD_PHI * ps + site];
    const double psi = (double)a.fields[FLD_PSI * ps + site];
    const double C = (double)a.fields[FLD_C * ps + site];
    const double p = (double)a.fields[FLD_P * ps + site];
    const double vx = (double)a.fields[FLD_VX * ps + site];
    const double vy = (double)a.fields[FLD_VY * ps + site];
    const unsigned row = (unsigned)i / (unsigned)d.nx, col = (unsigned)i - row * (unsigned)d.nx;
    const double x = (double)col, y = (double)row, gas = 1.0 - phi;
    acc[0] += phi;
    acc[1] += C;
    acc[2] += 0.5 * (1.0 + psi);
    acc[3] += gas;
    acc[4] += x * gas;
    acc[5] += y * gas;
    if (a.probe) {
      const double dx = min_image(x - a.xc, (double)d.nx), dy = min_image(y - a.yc, (double)d.ny);
      const double r = sqrt(dx * dx + dy * dy);
      if (r < Rin) { acc[6] += p; acc[7] += 1.0; }
      if (r > Rout) { acc[8] += p; acc[9] += 1.0; }
    }
    const double vm = vx * vx + vy * vy;
    if (vm > acc[10]) acc[10] = vm;
    if (!isfinite(phi) || !isfinite(psi) || !isfinite(C) || !isfinite(p) || !isfinite(vx) ||
        !isfinite(vy))
      acc[11] += 1.0;
  }
  const double r = block_sum256<NDIAG, 10>(acc);
  if (threadIdx.x < NDIAG) partial[blockIdx.x * NDIAG + threadIdx.x] = r;
  if (!last_block(ctr)) return;
  const double t = sum_records256<NDIAG, 10>(partial, gridDim.x);
  if (threadIdx.x < NDIAG) out[threadIdx.x] = threadIdx.x == 10 ? sqrt(t) : t;
  if (threadIdx.x == 0) out[NDIAG] = (double)*err;
}

// Thermal totals (FP64): sum over sites of the five temperature populations
// (the total of rho H: their density plane, or the tied populations),
// sum theta, sum psi; then the device error bits.
template <typename S, typename R>
__global__ void __launch_bounds__(RED_THREADS) k_reduce_thermal(
    const S* __restrict__ pop, const R* __restrict__ fields, long long ps, DomDesc d,
    const S* __restrict__ tied, double* __restrict__ partial, double* __restrict__ out, unsigned int* __restrict__ ctr,
    const unsigned int* __restrict__ err) {
  double acc[3] = {0.0, 0.0, 0.0};
  const long long n = (long long)d.nx * d.ny;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const long long site = d.off + i;
    if (tied) {
      double se = 0.0;
      for (int q = 0; q < 5; ++q) se += (double)ld<R>(tied + (T_E + q) * n, i);
      acc[0] += se;
    } else {
      acc[0] += (double)ld<R>(pop + P_E * ps, site);
    }
    acc[1] += (double)fields[FLD_THETA * ps + site];
    acc[2] += (double)fields[FLD_PSI * ps + site];
  }
  const double r = block_sum256<3>(acc);
  if (threadIdx.x < 3) partial[blockIdx.x * 3 + threadIdx.x] = r;
  if (!last_block(ctr)) return;
  const double t = sum_records256<3>(partial, gridDim.x);
  if (threadIdx.x < 3) out[threadIdx.x] = t;
  if (threadIdx.x == 0) out[3] = (double)*err;
}

// Fields [j0, j1) of a domain to FP64 (the band form of k_fields_to_f64).
template <typename R>
__global__ void k_fields_to_f64_range(const R* __restrict__ fields, long long ps, long long off,
                                      long long n, long long j0, long long j1, uint32_t mask,
                                      double* __restrict__ out) {
  int sel[N_FIELDS];
  int ns = 0;
  for (int f = 0; f < N_FIELDS; ++f)
    if (mask & (1u << f)) sel[ns++] = f;
  const long long m = j1 - j0, tot = m * ns;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot;
       i += (long long)gridDim.x * blockDim.x) {
    const long long q = i / m, j = j0 + i % m;
    out[q * n + j] = static_cast<double>(fields[sel[q] * ps + off + j]);
  }
}

// Buoyancy reference of a domain from its n values of phi rounded to R: the
// sum with the thread order and block tree of the phi sum in k_reduce, then
// doms[dom].rho_bar = fma(sum / n, drho, rho_g) in the device descriptor.
template <typename R>
__global__ void __launch_bounds__(RED_THREADS) k_rho_bar(const double* __restrict__ v, long long n,
                                                         double* __restrict__ partial,
                                                         unsigned int* __restrict__ ctr,
                                                         DomDesc* doms, int dom, double rho_g,
                                                         double drho) {
  double acc[1] = {0.0};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    acc[0] += (double)static_cast<R>(v[i]);
  const double r = block_sum256<1>(acc);
  if (threadIdx.x == 0) partial[blockIdx.x] = r;
  if (!last_block(ctr)) return;
  const double t = sum_records256<1>(partial, gridDim.x);
  if (threadIdx.x == 0) doms[dom].rho_bar = fma(t / (double)n, drho, rho_g);
}

// ---------------------------------------------------------------------------
// Host-side launchers (explicit instantiations for FP64 and FP32).
// ---------------------------------------------------------------------------
template <typename S, typename R>
cudaError_t launch_init_spec(const InitArgs<S, R>& a, cudaStream_t st) {
  const long long n = (long long)a.dom.nx * a.dom.ny;
  const int grid = (int)((n + 255) / 256 < 65535 ? (n + 255) / 256 : 65535);
  k_init_spec<S, R><<<grid, 256, 0, st>>>(a);
  return cudaGetLastError();
}

// Sets *flag when any of n staged host values is not finite; run before the
// values reach the state.
__global__ void k_flag_nonfinite(const double* __restrict__ p, long long n,
                                 unsigned int* flag) {
  bool bad = false;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    bad |= !isfinite(p[i]);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1u);
}

cudaError_t launch_flag_nonfinite(const double* p, long long n, unsigned int* flag,
                                  cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(unsigned int), st);
  if (e != cudaSuccess) return e;
  const int grid = (int)std::min<long long>((n + 255) / 256, 1024);
  k_flag_nonfinite<<<std::max(grid, 1), 256, 0, st>>>(p, n, flag);
  return cudaGetLastError();
}

template <typename S, typename R>
cudaError_t launch_set_fields(const SetFieldsArgs<S, R>& a, cudaStream_t st) {
  const long long n = (a.i1 > 0 ? a.i1 : (long long)a.dom.nx * a.dom.ny) - a.i0;
  if (n <= 0) return cudaSuccess;
  const int grid = (int)((n + 255) / 256 < 65535 ? (n + 255) / 256 : 65535);
  k_set_fields<S, R><<<grid, 256, 0, st>>>(a);
  return cudaGetLastError();
}

template <typename S, typename R>
cudaError_t launch_state_to_f64(const S* pin, const R* ain, long long ps, long long off,
                                long long n, double* out, int thermal, double rho_g, double drho,
                                const S* tied, cudaStream_t st) {
  k_state_to_f64<S, R><<<1024, 256, 0, st>>>(pin, ain, ps, off, n, out, thermal, rho_g, drho, tied);
  return cudaGetLastError();
}

template <typename S, typename R>
cudaError_t launch_state_from_f64(S* pout, R* aout, long long ps, long long off, long long n,
                                  const double* in, int thermal, S* tied, cudaStream_t st) {
  k_state_from_f64<S, R><<<1024, 256, 0, st>>>(pout, aout, ps, off, n, in, thermal, tied);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_state_general(long long n, const double* in, int thermal, double rho_g,
                                 double drho, unsigned int* general, cudaStream_t st) {
  k_state_general<R><<<1024, 256, 0, st>>>(n, in, thermal, rho_g, drho, general);
  return cudaGetLastError();
}

template <typename S, typename R>
cudaError_t launch_tied_temperature(const S* pin, const R* ain, long long ps, long long off,
                                    long long n, S* tied, double rho_g, double drho,
                                    cudaStream_t st) {
  k_tied_temperature<S, R><<<1024, 256, 0, st>>>(pin, ain, ps, off, n, tied, rho_g, drho);
  return cudaGetLastError();
}

template <typename S, typename R>
cudaError_t launch_set_temperature(S* out, R* aout, R* fields, long long ps, const DomDesc& d,
                                   const double* theta, const KParams<R>& kp, cudaStream_t st) {
  const long long n = (long long)d.nx * d.ny;
  const int grid = (int)((n + 255) / 256 < 65535 ? (n + 255) / 256 : 65535);
  k_set_temperature<S, R><<<grid, 256, 0, st>>>(out, aout, fields, ps, d, theta, kp);
  return cudaGetLastError();
}

// Blocks of a reduction over n sites (a record each; the phi sums of k_reduce
// and k_rho_bar agree bit for bit because both take this grid).
static int reduce_grid(long long n) {
  return (int)std::min<long long>((n + RED_THREADS - 1) / RED_THREADS, REDUCE_BLOCKS);
}

template <typename S, typename R>
cudaError_t launch_reduce_thermal(const S* pop, const R* fields, long long ps, const DomDesc& d,
                                  const S* tied, double* partial, double* out, unsigned int* ctr,
                                  const unsigned int* err, cudaStream_t st) {
  k_reduce_thermal<S, R><<<reduce_grid((long long)d.nx * d.ny), RED_THREADS, 0, st>>>(
      pop, fields, ps, d, tied, partial, out, ctr, err);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_fields_to_f64(const R* fields, long long ps, long long off, long long n,
                                 uint32_t mask, double* out, cudaStream_t st) {
  k_fields_to_f64<R><<<1024, 256, 0, st>>>(fields, ps, off, n, mask, out);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_fields_to_f64_range(const R* fields, long long ps, long long off, long long n,
                                       long long j0, long long j1, uint32_t mask, double* out,
                                       cudaStream_t st) {
  if (j1 <= j0) return cudaSuccess;
  k_fields_to_f64_range<R><<<1024, 256, 0, st>>>(fields, ps, off, n, j0, j1, mask, out);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_rho_bar(const double* phi, long long n, double* partial, unsigned int* ctr,
                           DomDesc* doms, int dom, double rho_g, double drho, cudaStream_t st) {
  k_rho_bar<R><<<reduce_grid(n), RED_THREADS, 0, st>>>(phi, n, partial, ctr, doms, dom, rho_g,
                                                       drho);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_reduce(const ReduceArgs<R>& a, double* partial, double* out, unsigned int* ctr,
                          const unsigned int* err, cudaStream_t st) {
  k_reduce<R><<<reduce_grid((long long)a.dom.nx * a.dom.ny), RED_THREADS, 0, st>>>(a, partial, out,
                                                                                   ctr, err);
  return cudaGetLastError();
}

#define PF_INST(S, R)                                                                      \
  template cudaError_t launch_init_spec<S, R>(const InitArgs<S, R>&, cudaStream_t);          \
  template cudaError_t launch_set_fields<S, R>(const SetFieldsArgs<S, R>&, cudaStream_t);    \
  template cudaError_t launch_state_to_f64<S, R>(const S*, const R*, long long, long long,   \
                                                 long long, double*, int, double, double,    \
                                                 const S*, cudaStream_t);                    \
  template cudaError_t launch_state_from_f64<S, R>(S*, R*, long long, long long, long long,  \
                                                   const double*, int, S*, cudaStream_t);    \
  template cudaError_t launch_tied_temperature<S, R>(const S*, const R*, long long, long long, \
                                                     long long, S*, double, double,          \
                                                     cudaStream_t);                          \
  template cudaError_t launch_set_temperature<S, R>(S*, R*, R*, long long, const DomDesc&,   \
                                                    const double*, const KParams<R>&,        \
                                                    cudaStream_t);                           \
  template cudaError_t launch_reduce_thermal<S, R>(const S*, const R*, long long,            \
                                                   const DomDesc&, const S*, double*,        \
                                                   double*, unsigned int*,                   \
                                                   const unsigned int*,                      \
                                                   cudaStream_t);

PF_INST(double, double)
PF_INST(float, float)
PF_INST(__half, float)
PF_INST(__nv_bfloat16, float)

template cudaError_t launch_fields_to_f64<double>(const double*, long long, long long,
                                                  long long, uint32_t, double*, cudaStream_t);
template cudaError_t launch_fields_to_f64<float>(const float*, long long, long long, long long,
                                                 uint32_t, double*, cudaStream_t);
template cudaError_t launch_fields_to_f64_range<double>(const double*, long long, long long,
                                                        long long, long long, long long, uint32_t,
                                                        double*, cudaStream_t);
template cudaError_t launch_fields_to_f64_range<float>(const float*, long long, long long,
                                                       long long, long long, long long, uint32_t,
                                                       double*, cudaStream_t);
template cudaError_t launch_state_general<double>(long long, const double*, int, double, double,
                                                  unsigned int*, cudaStream_t);
template cudaError_t launch_state_general<float>(long long, const double*, int, double, double,
                                                 unsigned int*, cudaStream_t);
template cudaError_t launch_rho_bar<double>(const double*, long long, double*, unsigned int*,
                                            DomDesc*, int, double, double, cudaStream_t);
template cudaError_t launch_rho_bar<float>(const double*, long long, double*, unsigned int*,
                                           DomDesc*, int, double, double, cudaStream_t);
template cudaError_t launch_reduce<double>(const ReduceArgs<double>&, double*, double*,
                                           unsigned int*, const unsigned int*, cudaStream_t);
template cudaError_t launch_reduce<float>(const ReduceArgs<float>&, double*, double*,
                                          unsigned int*, const unsigned int*, cudaStream_t);

}  // namespace pf
