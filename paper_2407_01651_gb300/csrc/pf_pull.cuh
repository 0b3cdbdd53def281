// pf_pull.cuh -- streaming (pull) helpers shared by the step kernel and the
// adjoint kernels: source sites of the D2Q9 / D2Q5 pull, the streamed CAC and
// dendrite populations with the a_s^2 time stretch, and the per-site inputs
// that no neighbour needs.
#pragma once

#include "pf_device.cuh"

namespace pf {

// The state pointers of a step as values the compiler has not seen: loads of the
// step (ldp) can neither be merged with those before this point nor move above it.
template <typename S, typename R>
__device__ __forceinline__ void fresh_state(StepArgs<S, R>& a) {
  asm volatile("" : "+l"(a.in), "+l"(a.ain)::"memory");
}

// A step launched behind another (StepArgs::chained): its CTAs are placed while
// the last ones of that step run and wait here until it is complete and its
// writes are visible; then the next step's CTAs may be placed.  The launch of a
// step, about 2 us, is so hidden behind the step before; us per step without and
// with it: FP32 128^2 6.2 -> 4.4, 512^2 18.5 -> 16.4, FP64 128^2 38.9 -> 35.3.
// The state pointers go through the statement behind the wait, so no load moves
// above it.  Every thread calls it, once, before its first load of the state.
template <typename S, typename R>
__device__ __forceinline__ void chain_step(StepArgs<S, R>& a) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" : "+l"(a.in), "+l"(a.ain)::"memory");
}

// Source sites of the pull for the 9 D2Q9 directions at (x, y):
// src[i] = (x - cx_i, y - cy_i), periodic.
struct Src9 {
  unsigned s[9];   // element offsets (a handle holds < 2^32 elements per buffer)
};

__device__ __forceinline__ Src9 sources(const DomDesc& d, int x, int y) {
  const int nx = d.nx, ny = d.ny;
  const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
  const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
  const unsigned off = (unsigned)d.off;
  const unsigned unx = (unsigned)nx;
  const unsigned r0 = off + (unsigned)y * unx, rm = off + (unsigned)ym * unx,
                 rp = off + (unsigned)yp * unx;
  Src9 o;
  o.s[0] = r0 + x; o.s[1] = r0 + xm; o.s[2] = rm + x; o.s[3] = r0 + xp; o.s[4] = rp + x;
  o.s[5] = rm + xm; o.s[6] = rm + xp; o.s[7] = rp + xp; o.s[8] = rp + xm;
  return o;
}

// Element offsets of plane k at site index s.  A handle whose buffers hold
// fewer than 2^32 elements addresses them with one 32-bit offset k*ps + s from
// the buffer base (the fast form); a larger one (BIG) takes a 64-bit base per
// plane and the 32-bit site index (a handle holds fewer than 2^32 sites).
template <bool BIG, typename T>
__device__ __forceinline__ const T* pbase(const T* p, int k, unsigned ps) {
  if constexpr (BIG) return plane(p, k, ps);
  else return p;
}
template <bool BIG>
__device__ __forceinline__ unsigned pidx(int k, unsigned ps, unsigned s) {
  if constexpr (BIG) return s;
  else return (unsigned)k * ps + s;
}

// Plane of the pair of a D2Q9 (or D2Q5) direction within its lattice's pairs,
// and whether the pair stores the opposite direction.
__device__ __forceinline__ constexpr int pair9(int i) { return ((i - 1) & 1) + (i >= 5 ? 2 : 0); }
__device__ __forceinline__ constexpr bool minus9(int i) { return ((i - 1) & 2) != 0; }

// phi and the flux J = sum c h of the streamed CAC populations: v the stored
// population of each direction's pair at its source, ph the sources' phi_o (own
// in ph[0]; 16-bit forms: of every direction, else of 3, 4, 7, 8).
template <typename S, typename R>
__device__ __forceinline__ void cac_moments(const S (&v)[9], const R (&ph)[9], R& phi, V2<R>& J) {
  R h[9];
  h[0] = CacBase<R>(ph[0]).rest(ph[0]);
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    R base = R(0);
    if (Codec<S>::kOffset || minus9(i)) {
      const CacBase<R> b(ph[i]);
      base = i < 5 ? b.axis : b.diag();
    }
    h[i] = minus9(i) ? pair_m<S, R>(v[i], base) : pair_p<S, R>(v[i], base);
  }
  CSum<R> sh;
#pragma unroll
  for (int i = 0; i < 9; ++i) sh.add(h[i]);
  phi = sh.value();
  const V2<R> U = vec2(h[5], h[6]) - vec2(h[7], h[8]);
  J = (vec2(h[1], h[2]) - vec2(h[3], h[4])) + vec2(U.x - U.y, U.x + U.y);
}

// Streamed CAC moments (phi and the flux J) and dendrite populations g (with
// the a_s^2 time stretch g = g_pre + r_src (g_post,src - g_pre)) at (x, y);
// phi and psi are compensated sums, psi_o is the psi of the previous step (sum
// of g_pre, or the stored lagged psi in the offset forms).  In two parts, so
// that a traversal may issue the loads of a row well before it combines them.
template <typename S, typename R>
struct HgLoads {
  S h[9], gpre[5], gp[5], gm[5];   // h and g_post of each direction's pair at its source, the
                                   // sources' g_post density (or F/6)
  R ph[9], po[5], rr[5];           // phi_o, psi_o (offset forms) and r of the sources
};

template <typename S, typename R, bool BIG = false>
__device__ __forceinline__ void load_hg(const StepArgs<S, R>& a, const Src9& src,
                                        HgLoads<S, R>& l) {
  const unsigned ps = (unsigned)a.plane_stride;
  constexpr bool off = Codec<S>::kOffset;
  auto pop = [&](int k, unsigned s) { return ldp(pbase<BIG>(a.in, k, ps) + pidx<BIG>(k, ps, s)); };
  auto aux = [&](int k, unsigned s) { return ldp(pbase<BIG>(a.ain, k, ps) + pidx<BIG>(k, ps, s)); };
  l.ph[0] = aux(A_PHIO, src.s[0]);
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    l.h[i] = pop(P_H + pair9(i), src.s[i]);
    if (off || minus9(i)) l.ph[i] = aux(A_PHIO, src.s[i]);
  }
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    l.gpre[i] = pop(P_GPRE + i, src.s[0]);
    if (i > 0) l.gp[i] = pop(P_GPOST + 1 + pair9(i), src.s[i]);
    if (i == 0 || minus9(i)) l.gm[i] = pop(P_GPOST, src.s[i]);
    if (off) l.po[i] = aux(A_PSIO, src.s[i]);
    l.rr[i] = aux(A_RR, src.s[i]);
  }
}

template <typename S, typename R>
__device__ __forceinline__ void finish_hg(const HgLoads<S, R>& l, V2<R>& J, R g[5], R& phi, R& psi,
                                          R& psio) {
  constexpr bool off = Codec<S>::kOffset;
  cac_moments<S, R>(l.h, l.ph, phi, J);
  CSum<R> sg;
  R po = R(0);
  const R psio_own = off ? l.po[0] : R(0);
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const R gold = dec_off<S, R>(l.gpre[i], w5<R>(i) * psio_own);
    R gpo;
    if constexpr (off) {
      // density psi_o + F of the source; its planes: F/6 and the offsets of g_1, g_2
      const R base = q5_base(l.po[i]);
      if (i == 0) gpo = fma(R(2), dec_off<S, R>(l.gm[0], R(0)), q5_rest(l.po[0], base));
      else if (!minus9(i)) gpo = pair_p<S, R>(l.gp[i], base);
      else gpo = pair_m<S, R>(l.gp[i], fma(R(2), dec_off<S, R>(l.gm[i], R(0)), base));
    } else {
      if (i == 0) gpo = q5_rest((R)l.gm[0], q5_base((R)l.gm[0]));
      else if (!minus9(i)) gpo = (R)l.gp[i];
      else gpo = pair_m<S, R>(l.gp[i], q5_base((R)l.gm[i]));
    }
    g[i] = gold + (gpo - gold) * l.rr[i];
    sg.add(g[i]);
    po += gold;
  }
  psi = sg.value();
  psio = off ? psio_own : po;
}

template <typename S, typename R, bool BIG = false>
__device__ __forceinline__ void pull_hg(const StepArgs<S, R>& a, const Src9& src, V2<R>& J,
                                        R g[5], R& phi, R& psi, R& psio) {
  HgLoads<S, R> l;
  load_hg<S, R, BIG>(a, src, l);
  finish_hg<S, R>(l, J, g, phi, psi, psio);
}

// Three rows of a shared-memory field around a site: row y-1, y, y+1.
template <typename R>
struct Rows3 {
  const R* m;
  const R* c;
  const R* p;
};

// Per-site inputs that do not feed the neighbours' stencils: streamed NS and
// solute populations and the lagged scalars of the site.
template <typename R>
struct SiteIn {
  R f[9], s[5];
  R phio, Co, Qo;
  uint8_t gid;
  GrainCS<R> cs;  // of that grain: load_grain, once gid has arrived
  R e[5], mo;     // thermal mode: streamed temperature populations, lagged rho H
};

// What a tile's sites take from their domain, in the type of the arithmetic:
// converted once per tile, since FP64 conversions run on units that this GPU
// has few of.
template <typename R>
struct SiteDom {
  R rho_bar, eps;
  int grain_off;
  __device__ __forceinline__ explicit SiteDom(const DomDesc& d)
      : rho_bar(static_cast<R>(d.rho_bar)), eps(static_cast<R>(d.eps_s)), grain_off(d.grain_off) {}
};

// The grain rotation of a site.  Issued before the barrier that ends a row's
// streaming: it depends on the grain id, and in the middle of the update every
// warp waited for it.
template <typename S, typename R>
__device__ __forceinline__ void load_grain(const StepArgs<S, R>& a, const SiteDom<R>& sd,
                                           SiteIn<R>& in) {
  in.cs = a.grain_cs[sd.grain_off + in.gid];
}

// Streamed solute populations; Co is C of the last step at the site itself.
template <typename S, typename R, bool BIG = false>
__device__ __forceinline__ void pull_s(const StepArgs<S, R>& a, const Src9& src, R Co, R (&s)[5]) {
  const unsigned ps = (unsigned)a.plane_stride;
  constexpr bool off = Codec<S>::kOffset;
  s[0] = q5_rest(Co, q5_base(Co));
#pragma unroll
  for (int i = 1; i < 5; ++i) {
    const int k = P_S + pair9(i);
    const S v = ldp(pbase<BIG>(a.in, k, ps) + pidx<BIG>(k, ps, src.s[i]));
    R base = R(0);
    if (off || minus9(i))
      base = q5_base(ldp(pbase<BIG>(a.ain, A_CO, ps) + pidx<BIG>(A_CO, ps, src.s[i])));
    s[i] = minus9(i) ? pair_m<S, R>(v, base) : pair_p<S, R>(v, base);
  }
}

template <typename S, typename R, bool BIG = false, bool TH = false>
__device__ __forceinline__ void load_site(const StepArgs<S, R>& a, const Src9& src,
                                          SiteIn<R>& in) {
  const unsigned ps = (unsigned)a.plane_stride;
#pragma unroll
  for (int i = 0; i < 9; ++i) in.f[i] = pop_ns<S, R>(pbase<BIG>(a.in, P_F + i, ps), pidx<BIG>(P_F + i, ps, src.s[i]));
  in.phio = ld<R>(pbase<BIG>(a.ain, A_PHIO, ps), pidx<BIG>(A_PHIO, ps, src.s[0]));
  in.Co = ld<R>(pbase<BIG>(a.ain, A_CO, ps), pidx<BIG>(A_CO, ps, src.s[0]));
  pull_s<S, R, BIG>(a, src, in.Co, in.s);
  in.Qo = ld<R>(pbase<BIG>(a.ain, A_QO, ps), pidx<BIG>(A_QO, ps, src.s[0]));
  in.gid = a.grain[src.s[0]];
  if constexpr (TH) {
    auto pop = [&](int k, unsigned s) { return ld<R>(pbase<BIG>(a.in, k, ps), pidx<BIG>(k, ps, s)); };
    in.mo = pop(P_E, src.s[0]);
    in.e[0] = q5_rest(in.mo, pop(P_E + 1, src.s[0]));
    in.e[1] = pop(P_E + 2, src.s[1]);
    in.e[2] = pop(P_E + 3, src.s[2]);
    in.e[3] = fma(R(2), pop(P_E + 1, src.s[3]), -pop(P_E + 2, src.s[3]));
    in.e[4] = fma(R(2), pop(P_E + 1, src.s[4]), -pop(P_E + 3, src.s[4]));
  }
}

// Supersaturation U of a site from its streamed solute populations (thermal
// mode: U on the stencil neighbourhood feeds grad F), with the arithmetic of
// the site update's own C and U.
template <typename R>
__device__ __forceinline__ R supersat(const KParams<R>& kp, const R (&s)[5], R psi) {
  CSum<R> cs;
#pragma unroll
  for (int i = 0; i < 5; ++i) cs.add(s[i]);
  const R C = cs.value();
  const R omk = R(1) - kp.k;
  const R A = (R(1) + kp.k) - omk * psi;
  return (R(2) * C * frcp(A) - R(1)) * kp.inv_omk;
}
template <typename S, typename R, bool BIG = false>
__device__ __forceinline__ R pull_U(const StepArgs<S, R>& a, const Src9& src, R psi) {
  const unsigned ps = (unsigned)a.plane_stride;
  R s[5];
  pull_s<S, R, BIG>(a, src, ldp(pbase<BIG>(a.ain, A_CO, ps) + pidx<BIG>(A_CO, ps, src.s[0])), s);
  return supersat(a.kp, s, psi);
}

}  // namespace pf
