// pf_raw.cuh -- pulls from a raw state: the stored state and beside it the tied
// planes (T_*, pf_model.cuh), with every population of a pair, that pf_set_state
// kept for it (pf_step_general.cu says when they are used).
//
// The tied planes are in the storage form, as every other plane of the state is:
// 19 values a site (thermal 25) against the 20 (24) that the pairs save on the
// two copies, so a handle whose every domain is raw holds no more than one with
// all populations in its state would (thermal: one value a site more).
#pragma once

#include "pf_sides.cuh"

namespace pf {

template <typename S, typename R, bool TH>
struct GeneralPull {
  const S* w;      // tied planes of the domain
  const StepArgs<S, R>& a;
  const DomDesc& d;
  __device__ __forceinline__ S tied(int k, unsigned site) const {
    return w[k * ((long long)d.nx * d.ny) + (site - (unsigned)d.off)];
  }
  __device__ __forceinline__ R pop(int k, unsigned site) const {
    return ld<R>(plane(a.in, k, (unsigned)a.plane_stride), site);
  }
  __device__ __forceinline__ R aux(int k, unsigned site) const {
    return ldp(plane(a.ain, k, (unsigned)a.plane_stride) + site);
  }
  // a tied population whose offset is from weight x moment (16-bit forms)
  __device__ __forceinline__ R off(int k, unsigned site, R wm) const {
    return dec_off<S, R>(tied(k, site), wm);
  }
  __device__ __forceinline__ R psio_of(unsigned site) const {
    return Codec<S>::kOffset ? aux(A_PSIO, site) : R(0);
  }

  __device__ __forceinline__ void hg(int x, int y, V2<R>& J, R (&g)[5], R& phi, R& psi,
                                     R& psio) const {
    const unsigned own = site_at(d, x, y);
    R h[9];
    CSum<R> sh;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const PullSrc p = scalar_src<true>(d, x, y, i);
      h[i] = off(T_H + p.q, p.site, w9<R>(p.q) * aux(A_PHIO, p.site));
      if (p.mode == 3) h[i] = -h[i] + R(2) * w9<R>(i) * R(1);
      sh.add(h[i]);
    }
    phi = sh.value();
    const V2<R> U = vec2(h[5], h[6]) - vec2(h[7], h[8]);
    J = (vec2(h[1], h[2]) - vec2(h[3], h[4])) + vec2(U.x - U.y, U.x + U.y);
    CSum<R> sg;
    R po = R(0);
    const R mo = psio_of(own);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const PullSrc p = scalar_src<true>(d, x, y, i);
      const R gold = pop_off<S, R>(plane(a.in, P_GPRE + i, (unsigned)a.plane_stride), own,
                                   w5<R>(i) * mo);
      R gpo = off(T_GPOST + p.q, p.site, w5<R>(p.q) * psio_of(p.site));
      if (p.mode == 2 || p.mode == 3) gpo = -gpo + R(2) * w5<R>(i) * R(-1);
      g[i] = gold + (gpo - gold) * aux(A_RR, p.site);
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
      v[i] = off(T_S + p.q, p.site, w5<R>(p.q) * aux(A_CO, p.site));
      if (p.mode == 2 || p.mode == 3) v[i] = -v[i] + R(2) * w5<R>(i) * R(1);
    }
  }

  __device__ __forceinline__ void site(int x, int y, SiteIn<R>& in) const {
    const unsigned own = site_at(d, x, y);
    in.phio = aux(A_PHIO, own);
    in.Co = aux(A_CO, own);
    in.Qo = aux(A_QO, own);
    in.gid = a.grain[own];
    const R rho_o = a.kp.rho_g + in.phio * a.kp.drho;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const PullSrc p = pull_src<true>(d, x, y, i);
      const bool outlet = p.mode == 4;
      const int q = outlet ? opp9(i) : p.q;
      const R v = pop_ns<S, R>(plane(a.in, P_F + q, (unsigned)a.plane_stride), outlet ? own : p.site);
      in.f[i] = side_ns<R>(a.kp, p, i, v, rho_o, aux(A_VXO, own), aux(A_VYO, own),
                           [&](R& fx, R& fy, R& fphi) {
                             fx = aux(A_VXO, p.site);
                             fy = aux(A_VYO, p.site);
                             fphi = aux(A_PHIO, p.site);
                           });
    }
    solute(x, y, in.s);
    if constexpr (TH) {
      in.mo = rho_o * (R)tied(T_HO, own);
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        const PullSrc p = scalar_src<true>(d, x, y, i);
        in.e[i] = (R)tied(T_E + p.q, p.site);
        if (p.mode == 2 || p.mode == 3) in.e[i] = -in.e[i] + R(2) * w5<R>(i) * a.kp.th_far;
      }
    }
  }
};

}  // namespace pf
