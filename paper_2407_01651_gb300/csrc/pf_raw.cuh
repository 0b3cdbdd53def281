// pf_raw.cuh -- pulls from a raw state: the FP64 planes of pf_set_state, with
// every population of a pair (pf_step_general.cu says when they are used).
#pragma once

#include "pf_sides.cuh"

namespace pf {

// One population or scalar of the raw state, rounded to the storage form; j is
// the site within its domain.
template <typename S, typename R>
struct RawState {
  const double* w;
  long long n;
  __device__ __forceinline__ R x(int plane, unsigned j) const { return (R)w[plane * n + j]; }
  __device__ __forceinline__ R ns(int q, unsigned j) const {
    if constexpr (Codec<S>::kOffset) {
      return Codec<S>::template dec<R>(Codec<S>::template enc<R>(x(X_F + q, j) * R(kNSScale))) *
             R(kNSInvScale);
    } else {
      return x(X_F + q, j);
    }
  }
  __device__ __forceinline__ R off(int plane, unsigned j, R wm) const {
    return dec_off<S, R>(enc_off<S, R>(x(plane, j), wm), wm);
  }
  __device__ __forceinline__ R psio(unsigned j) const {
    R p = R(0);
#pragma unroll
    for (int i = 0; i < 5; ++i) p += x(X_GPRE + i, j);
    return p;
  }
};

template <typename S, typename R, bool TH>
struct GeneralPull {
  const RawState<S, R>& s;
  const StepArgs<S, R>& a;
  const DomDesc& d;
  __device__ __forceinline__ unsigned local(unsigned site) const { return site - (unsigned)d.off; }

  __device__ __forceinline__ void hg(int x, int y, V2<R>& J, R (&g)[5], R& phi, R& psi,
                                     R& psio) const {
    const unsigned own = local(site_at(d, x, y));
    R h[9];
    CSum<R> sh;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const PullSrc p = scalar_src<true>(d, x, y, i);
      const unsigned j = local(p.site);
      h[i] = s.off(X_H + p.q, j, w9<R>(p.q) * s.x(X_PHI, j));
      if (p.mode == 3) h[i] = -h[i] + R(2) * w9<R>(i) * R(1);
      sh.add(h[i]);
    }
    phi = sh.value();
    const V2<R> U = vec2(h[5], h[6]) - vec2(h[7], h[8]);
    J = (vec2(h[1], h[2]) - vec2(h[3], h[4])) + vec2(U.x - U.y, U.x + U.y);
    CSum<R> sg;
    R po = R(0);
    const R mo = s.psio(own);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const PullSrc p = scalar_src<true>(d, x, y, i);
      const unsigned j = local(p.site);
      const R gold = s.off(X_GPRE + i, own, w5<R>(i) * mo);
      R gpo = s.off(X_GPOST + p.q, j, w5<R>(p.q) * s.psio(j));
      if (p.mode == 2 || p.mode == 3) gpo = -gpo + R(2) * w5<R>(i) * R(-1);
      g[i] = gold + (gpo - gold) * s.x(X_RR, j);
      sg.add(g[i]);
      po += gold;
    }
    psi = sg.value();
    psio = Codec<S>::kOffset ? mo : po;
  }

  __device__ __forceinline__ void solute(int x, int y, R (&v)[5]) const {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const PullSrc p = scalar_src<true>(d, x, y, i);
      const unsigned j = local(p.site);
      v[i] = s.off(X_S + p.q, j, w5<R>(p.q) * s.x(X_C, j));
      if (p.mode == 2 || p.mode == 3) v[i] = -v[i] + R(2) * w5<R>(i) * R(1);
    }
  }

  __device__ __forceinline__ void site(int x, int y, SiteIn<R>& in) const {
    const unsigned own = local(site_at(d, x, y));
    in.phio = s.x(X_PHI, own);
    in.Co = s.x(X_C, own);
    in.Qo = s.x(X_Q, own);
    in.gid = a.grain[site_at(d, x, y)];
    const R rho_o = a.kp.rho_g + in.phio * a.kp.drho;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const PullSrc p = pull_src<true>(d, x, y, i);
      const bool outlet = p.mode == 4;
      const R v = s.ns(outlet ? opp9(i) : p.q, outlet ? own : local(p.site));
      in.f[i] = side_ns<R>(a.kp, p, i, v, rho_o, s.x(X_VX, own), s.x(X_VY, own),
                           [&](R& fx, R& fy, R& fphi) {
                             const unsigned j = local(p.site);
                             fx = s.x(X_VX, j);
                             fy = s.x(X_VY, j);
                             fphi = s.x(X_PHI, j);
                           });
    }
    solute(x, y, in.s);
    if constexpr (TH) {
      in.mo = rho_o * s.x(X_HO, own);
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        const PullSrc p = scalar_src<true>(d, x, y, i);
        in.e[i] = s.x(X_E + p.q, local(p.site));
        if (p.mode == 2 || p.mode == 3) in.e[i] = -in.e[i] + R(2) * w5<R>(i) * a.kp.th_far;
      }
    }
  }
};

}  // namespace pf
