// pf_sides.cuh -- where the streamed populations and the stencil values of a
// site next to a non-periodic side come from (the rules are stated in
// pf_step_bc.cu), shared by the kernels that meet such sides.
#pragma once

#include "pf_site.cuh"

namespace pf {

__device__ __forceinline__ constexpr int cx9(int i) {
  return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
}
__device__ __forceinline__ constexpr int cy9(int i) {
  return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
}
__device__ __forceinline__ constexpr int opp9(int i) {
  return i == 0 ? 0 : (i <= 4 ? (i + 1) % 4 + 1 : (i + 1) % 4 + 5);
}
// reflections that flip c_x / c_y
__device__ __forceinline__ int mirx9(int i) {
  switch (i) {
    case 1: return 3; case 3: return 1; case 5: return 6; case 6: return 5;
    case 7: return 8; case 8: return 7; default: return i;
  }
}
__device__ __forceinline__ int miry9(int i) {
  switch (i) {
    case 2: return 4; case 4: return 2; case 5: return 8; case 8: return 5;
    case 6: return 7; case 7: return 6; default: return i;
  }
}

__device__ __forceinline__ unsigned site_at(const DomDesc& d, int x, int y) {
  return (unsigned)d.off + (unsigned)y * (unsigned)d.nx + (unsigned)x;
}

// Source of the population of direction i pulled by (x, y): site, direction
// to read and mode (0 plain or reflected, 1 wall bounce, 2 far-field bounce,
// 3 inlet bounce, 4 outlet: source clamped to the last site, 5 extrapolation
// inlet: the source is the ghost node beyond the side, whose NS population is
// built from the fluid site next to it, the one returned).
struct PullSrc {
  unsigned site;
  int q, mode;
};
// IO: some side of the launch is an inlet or an outlet; without them the
// compiler drops those branches from the boundary pulls
template <bool IO>
__device__ __forceinline__ int bounce_rank(int t) {
  return t == BC_WALL ? 1 : (t == BC_FARFIELD ? 2 : (IO && t == BC_INLET ? 3 : 0));
}
template <bool IO>
__device__ __forceinline__ PullSrc pull_src(const DomDesc& d, int x, int y, int i) {
  const int nx = d.nx, ny = d.ny;
  int sx = x - cx9(i), sy = y - cy9(i), q = i, bounce = 0, outlet = 0, nee = 0;
  if (sx < 0 || sx >= nx) {
    const int t = d.bc[sx < 0 ? 0 : 1];
    if (t == BC_PERIODIC) sx += sx < 0 ? nx : -nx;
    else if (t == BC_SYMMETRIC) { sx = sx < 0 ? -1 - sx : 2 * nx - 1 - sx; q = mirx9(q); }
    else if (IO && t == BC_OUTLET) { sx = sx < 0 ? 0 : nx - 1; outlet = 1; }
    else if (IO && t == BC_INLET_NEE) { sx = sx < 0 ? 0 : nx - 1; nee = 1; }
    else bounce = bounce_rank<IO>(t);
  }
  if (sy < 0 || sy >= ny) {
    const int t = d.bc[sy < 0 ? 2 : 3];
    if (t == BC_PERIODIC) sy += sy < 0 ? ny : -ny;
    else if (t == BC_SYMMETRIC) { sy = sy < 0 ? -1 - sy : 2 * ny - 1 - sy; q = miry9(q); }
    else if (IO && t == BC_OUTLET) { sy = sy < 0 ? 0 : ny - 1; outlet = 1; }
    else if (IO && t == BC_INLET_NEE) { sy = sy < 0 ? 0 : ny - 1; nee = 1; }
    else bounce = max(bounce, bounce_rank<IO>(t));
  }
  if (bounce) return {site_at(d, x, y), opp9(i), bounce};
  return {site_at(d, sx, sy), q, nee ? 5 : (outlet ? 4 : 0)};
}

// The lattices other than NS see an extrapolation inlet as an inlet:
// anti-bounce-back at the site itself.
template <bool IO>
__device__ __forceinline__ PullSrc scalar_src(const DomDesc& d, int x, int y, int i) {
  PullSrc p = pull_src<IO>(d, x, y, i);
  if (IO && p.mode == 5) p = {site_at(d, x, y), opp9(i), 3};
  return p;
}

// Ring fields: 0 phi, 1 psi, 2 vx_o, 3 vy_o, 4 U.  Ghost value across one side
// of type t on axis (0: x, 1: y) from the mirror site's value v.
template <typename R, bool IO>
__device__ __forceinline__ R ghost_map(const KParams<R>& kp, int t, int axis, int field, R v) {
  if (IO && t == BC_OUTLET) return v;
  if (field == 2 || field == 3) {
    const bool normal = (field == 2) == (axis == 0);
    if (t == BC_SYMMETRIC) return normal ? -v : v;
    if (IO && t == BC_INLET) return R(2) * (field == 2 ? kp.vin_x : kp.vin_y) - v;
    if (IO && t == BC_INLET_NEE) return field == 2 ? kp.vin_x : kp.vin_y;   // the ghost is the node
    return -v;
  }
  if (t == BC_FARFIELD || (IO && (t == BC_INLET || t == BC_INLET_NEE))) {
    if (field == 1) return R(-2) - v;   // 2 psi_far - psi, psi_far = -1
    if (field == 4) return -v;          // 2 U_far - U, U_far = 0
    if (IO && field == 0 && t != BC_FARFIELD) return R(2) - v;   // liquid inflow, phi = 1
  }
  return v;
}

// NS population of direction i at an outlet or inlet, from the loaded one: the
// site's own opposite population at a pressure outlet (p = 0), the bounced
// one at a moving-wall inlet, the ghost node's at an extrapolation inlet, whose
// velocity and phi of the last step `fluid` loads.
template <typename R, typename F>
__device__ __forceinline__ R side_ns(const KParams<R>& kp, const PullSrc& p, int i, R v, R rho_o,
                                     R vxo, R vyo, F&& fluid) {
  if (p.mode == 4) {
    // -f*_opp(own) + 2 rho_o w_i [(c.v_o)^2 / (2 cs^4) - v_o^2 / (2 cs^2)]
    const R cu = R(cx9(i)) * vxo + R(cy9(i)) * vyo;
    return -v + R(2) * rho_o * w9<R>(i) * (R(4.5) * cu * cu - R(1.5) * (vxo * vxo + vyo * vyo));
  }
  if (p.mode == 3)   // moving-wall bounce-back
    return v + R(2) * (kp.rho_g + kp.drho) * w9<R>(i) * R(3) *
                   (R(cx9(i)) * kp.vin_x + R(cy9(i)) * kp.vin_y);
  if (p.mode == 5) {
    // the ghost node's post-collision population is f_q^eq(p_b, rho_l, u_in) +
    // f*_q(x_f) - f_q^eq(p_f, rho_f, v_f) with p_b = p_f, i.e. f*_q(x_f) +
    // rho_l s_q(u_in) - rho_f s_q(v_f), with s_q(v) = w_q [3 c.v + 4.5 (c.v)^2
    // - 1.5 v^2] and the fluid site's last-step rho and v
    R fx, fy, fphi;
    fluid(fx, fy, fphi);
    const R cb = R(cx9(p.q)) * kp.vin_x + R(cy9(p.q)) * kp.vin_y;
    const R cf = R(cx9(p.q)) * fx + R(cy9(p.q)) * fy;
    const R sb = R(3) * cb + R(4.5) * cb * cb - R(1.5) * (kp.vin_x * kp.vin_x + kp.vin_y * kp.vin_y);
    const R sf = R(3) * cf + R(4.5) * cf * cf - R(1.5) * (fx * fx + fy * fy);
    return v + w9<R>(p.q) * ((kp.rho_g + kp.drho) * sb - (kp.rho_g + fphi * kp.drho) * sf);
  }
  return v;
}

}  // namespace pf
