// pf_step_bc.cu -- the y-march step kernel for domains with non-periodic
// sides (arXiv 2407.01651, Section 3: half-way bounce-back for no-slip walls
// and no-flux scalars, the symmetric scheme for symmetry planes; Section 4:
// far-field Dirichlet values psi = psi_l, C = 1, theta = -Omega).
//
// Same traversal and per-site arithmetic as k_step_ymarch (pf_step.cu); what
// differs is where values come from at a non-periodic side:
//   - pull streaming: a symmetric side reflects the source site and the
//     direction; a wall returns the site's own post-collision population of
//     the opposite direction; a far-field side does the same for NS and CAC
//     and an anti-bounce-back -f*_opp + 2 w_i X_far for psi, C and theta; an
//     inlet adds the moving-wall term 2 rho_l w_i c_i.u_in / c_s^2 for NS and
//     anti-bounces CAC to phi = 1; an outlet anti-bounces NS to p = 0 and
//     clamps the other lattices' source to the last site; an extrapolation
//     inlet gives NS the ghost node's populations f*(x_f) + rho_l s(u_in) -
//     rho_f s(v_f) from the fluid site x_f next to it and treats the other
//     lattices as an inlet; a bounce wins where two sides are crossed, then
//     the extrapolation, then the clamp, then the reflection;
//   - stencils: ghost rows and columns of the shared-memory ring hold the
//     mirror site's values mapped per side (phi, psi, U unchanged, or
//     2 X_far - X for psi and U at a far-field side or inlet, 2 - phi at an
//     inlet; the velocity's normal component flipped at a symmetric side, both
//     components at a wall or far field, 2 u_in - v at an inlet, u_in at an
//     extrapolation inlet; everything
//     copied at an outlet; corners: the y side's map, then the x side's).
// Sites away from a non-periodic side take the periodic pulls of pf_pull.cuh.
// FP32 and FP64 storage only.
#include <type_traits>

#include "pf_sides.cuh"

namespace pf {

namespace {

// Populations of the pair-stored lattices with the direction known at run time
// only: plane of the pair and whether the opposite one is stored.
__device__ __forceinline__ int pair_rt(int q) { return ((q - 1) & 1) + (q >= 5 ? 2 : 0); }
__device__ __forceinline__ bool minus_rt(int q) { return ((q - 1) & 2) != 0; }

// The pulls at a side first issue every load and then combine the values: with
// the source of each direction decided and used one after the other, each
// load's latency was waited for in turn (4.6 us a row of tiles, 1.5 us in the
// periodic kernel).
template <typename S, typename R, bool BIG, bool IO>
__device__ __forceinline__ void pull_hg_b(const StepArgs<S, R>& a, const DomDesc& d, int x,
                                          int y, V2<R>& J, R g[5], R& phi, R& psi, R& psio) {
  const unsigned ps = (unsigned)a.plane_stride;
  const unsigned own = site_at(d, x, y);
  auto pop = [&](int k, unsigned s) { return ld<R>(pbase<BIG>(a.in, k, ps), pidx<BIG>(k, ps, s)); };
  auto aux = [&](int k, unsigned s) { return ld<R>(pbase<BIG>(a.ain, k, ps), pidx<BIG>(k, ps, s)); };
  R v[9], ph[9], gv[5], m[5], rr[5], gold[5];
  int how[9];       // 4 q + class of the mode (0 as is, 2 far field, 3 inlet)
  ph[0] = aux(A_PHIO, own);
  m[0] = pop(P_GPOST, own);
  rr[0] = aux(A_RR, own);
#pragma unroll
  for (int i = 0; i < 5; ++i) gold[i] = pop(P_GPRE + i, own);
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const PullSrc p = scalar_src<IO>(d, x, y, i);
    how[i] = 4 * p.q + (p.mode == 2 || p.mode == 3 ? p.mode : 0);
    v[i] = pop(P_H + pair_rt(p.q), p.site);
    ph[i] = aux(A_PHIO, p.site);
    if (i < 5) {
      gv[i] = pop(P_GPOST + 1 + pair_rt(p.q), p.site);
      m[i] = pop(P_GPOST, p.site);
      rr[i] = aux(A_RR, p.site);
    }
  }
  R h[9];
  h[0] = CacBase<R>(ph[0]).rest(ph[0]);
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const CacBase<R> b(ph[i]);
    const R base = i < 5 ? b.axis : b.diag();   // a reflection keeps axes and diagonals apart
    h[i] = minus_rt(how[i] >> 2) ? fma(R(2), base, -v[i]) : v[i];
    if (IO && (how[i] & 3) == 3) h[i] = -h[i] + R(2) * w9<R>(i) * R(1);   // inlet: phi = 1
  }
  CSum<R> sh;
#pragma unroll
  for (int i = 0; i < 9; ++i) sh.add(h[i]);
  phi = sh.value();
  const V2<R> U = vec2(h[5], h[6]) - vec2(h[7], h[8]);
  J = (vec2(h[1], h[2]) - vec2(h[3], h[4])) + vec2(U.x - U.y, U.x + U.y);
  CSum<R> sg;
  R po = R(0);
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const R base = q5_base(m[i]);
    R gpo;
    if (i == 0) gpo = q5_rest(m[0], base);
    else {
      gpo = minus_rt(how[i] >> 2) ? fma(R(2), base, -gv[i]) : gv[i];
      if (how[i] & 3) gpo = -gpo + R(2) * w5<R>(i) * R(-1);
    }
    g[i] = gold[i] + (gpo - gold[i]) * rr[i];
    sg.add(g[i]);
    po += gold[i];
  }
  psi = sg.value();
  psio = po;
}

// Streamed solute populations next to a side (C_far = 1).
template <typename S, typename R, bool BIG, bool IO>
__device__ __forceinline__ void pull_s_b(const StepArgs<S, R>& a, const DomDesc& d, int x, int y,
                                         R Co, R (&s)[5]) {
  const unsigned ps = (unsigned)a.plane_stride;
  R v[5], c[5];
  int how[5];
#pragma unroll
  for (int i = 1; i < 5; ++i) {
    const PullSrc p = scalar_src<IO>(d, x, y, i);
    how[i] = 2 * p.q + (p.mode == 2 || p.mode == 3);
    const int k = P_S + pair_rt(p.q);
    v[i] = ld<R>(pbase<BIG>(a.in, k, ps), pidx<BIG>(k, ps, p.site));
    c[i] = ld<R>(pbase<BIG>(a.ain, A_CO, ps), pidx<BIG>(A_CO, ps, p.site));
  }
  s[0] = q5_rest(Co, q5_base(Co));
#pragma unroll
  for (int i = 1; i < 5; ++i) {
    s[i] = minus_rt(how[i] >> 1) ? fma(R(2), q5_base(c[i]), -v[i]) : v[i];
    if (how[i] & 1) s[i] = -s[i] + R(2) * w5<R>(i) * R(1);
  }
}

template <typename S, typename R, bool BIG, bool TH, bool IO>
__device__ __forceinline__ void load_site_b(const StepArgs<S, R>& a, const DomDesc& d, int x,
                                            int y, SiteIn<R>& in) {
  const unsigned ps = (unsigned)a.plane_stride;
  const unsigned own = site_at(d, x, y);
  auto pop = [&](int k, unsigned s) { return ld<R>(pbase<BIG>(a.in, k, ps), pidx<BIG>(k, ps, s)); };
  auto aux = [&](int k, unsigned s) { return ld<R>(pbase<BIG>(a.ain, k, ps), pidx<BIG>(k, ps, s)); };
  in.phio = aux(A_PHIO, own);
  in.Co = aux(A_CO, own);
  in.Qo = aux(A_QO, own);
  in.gid = a.grain[own];
  R vxo = R(0), vyo = R(0);
  if constexpr (IO) {
    vxo = aux(A_VXO, own);
    vyo = aux(A_VYO, own);
  }
  PullSrc p[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    p[i] = pull_src<IO>(d, x, y, i);
    // a pressure outlet takes the site's own opposite population
    const bool outlet = IO && p[i].mode == 4;
    in.f[i] = pop(P_F + (outlet ? opp9(i) : p[i].q), outlet ? own : p[i].site);
  }
  pull_s_b<S, R, BIG, IO>(a, d, x, y, in.Co, in.s);
  if constexpr (TH) {
    R v[5], b[5];
    int how[5];
    in.mo = pop(P_E, own);
    b[0] = pop(P_E + 1, own);
#pragma unroll
    for (int i = 1; i < 5; ++i) {
      const PullSrc q = scalar_src<IO>(d, x, y, i);
      how[i] = 2 * q.q + (q.mode == 2 || q.mode == 3);
      v[i] = pop(P_E + 2 + pair_rt(q.q), q.site);
      b[i] = pop(P_E + 1, q.site);
    }
    in.e[0] = q5_rest(in.mo, b[0]);
#pragma unroll
    for (int i = 1; i < 5; ++i) {
      in.e[i] = minus_rt(how[i] >> 1) ? fma(R(2), b[i], -v[i]) : v[i];
      if (how[i] & 1) in.e[i] = -in.e[i] + R(2) * w5<R>(i) * a.kp.th_far;
    }
  }
  if constexpr (IO) {
    const R rho_o = a.kp.rho_g + in.phio * a.kp.drho;
#pragma unroll
    for (int i = 0; i < 9; ++i)
      in.f[i] = side_ns<R>(a.kp, p[i], i, in.f[i], rho_o, vxo, vyo, [&](R& fx, R& fy, R& fphi) {
        fx = aux(A_VXO, p[i].site);
        fy = aux(A_VYO, p[i].site);
        fphi = aux(A_PHIO, p[i].site);
      });
  }
}

template <typename S, typename R, bool BIG, bool IO>
__device__ __forceinline__ R pull_U_b(const StepArgs<S, R>& a, const DomDesc& d, int x, int y,
                                      R psi) {
  const unsigned ps = (unsigned)a.plane_stride;
  R s[5];
  pull_s_b<S, R, BIG, IO>(a, d, x, y, ld<R>(pbase<BIG>(a.ain, A_CO, ps),
                                            pidx<BIG>(A_CO, ps, site_at(d, x, y))), s);
  return supersat(a.kp, s, psi);
}

}  // namespace

template <typename S, typename R, bool BIG, bool TH, bool IO>
__global__ void __launch_bounds__(YM_THREADS, sizeof(R) == 4 ? 3 : 2)
    k_step_ymarch_bc(StepArgs<S, R> a) {
  constexpr int RW = YM_W + 2;
  constexpr int NF = TH ? 5 : 4;
  __shared__ R ring[NF][4][RW];
  const int t = threadIdx.x;
  const unsigned ps = (unsigned)a.plane_stride;
  chain_step(a);

  for (int tile = a.tile_base + blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    const DomDesc d = a.doms[a.tile_dom[tile]];
    const int lt = tile - d.tile0;
    const int nx = d.nx, ny = d.ny;
    const int x0 = (lt % d.tiles_x) * YM_W;
    const int ya = (lt / d.tiles_x) * a.chunk;
    const int yb = min(ya + a.chunk, ny);
    const int w = min(YM_W, nx - x0);
    bool interior = false, active = false;
    int col = 0, sc = 0, tx = -1;   // column of the values, ring column, x ghost side type
    if (t < YM_W) {
      interior = active = t < w;
      col = x0 + t;
      sc = t + 1;
    } else if (t == YM_W) {
      active = true;
      sc = 0;
      if (x0 == 0 && d.bc[0]) { col = 0; tx = d.bc[0]; }
      else col = x0 == 0 ? nx - 1 : x0 - 1;
    } else if (t == YM_W + 1) {
      active = true;
      sc = w + 1;
      if (x0 + w >= nx && d.bc[1]) { col = nx - 1; tx = d.bc[1]; }
      else col = x0 + w >= nx ? x0 + w - nx : x0 + w;
    }

    // Whether the warp's columns in row y are pulled as next to a side: one path
    // per warp, the same for the same tile whatever the scheduling (every lane takes
    // part in the vote, once a tile; those without a column say no); away from the
    // side both paths pull the same values.
    const bool side_col = (col == 0 && d.bc[0]) || (col == nx - 1 && d.bc[1]);
    const bool near_col = __any_sync(0xffffffffu, active && side_col) != 0;
    const bool near_in = __any_sync(0xffffffffu, interior && side_col) != 0;
    auto side_row = [&](int y) { return (y == 0 && d.bc[2]) || (y == ny - 1 && d.bc[3]); };
    // row of the lattice that row yr of the ring comes from
    auto inside_row = [&](int yr) {
      return yr < 0 ? (d.bc[2] ? 0 : yr + ny) : (yr >= ny ? (d.bc[3] ? ny - 1 : yr - ny) : yr);
    };
    // ring values of row yr (ya-1 .. yb, possibly a ghost row) and the
    // streamed h, g of the site (col, row) they were computed at
    auto fill = [&](int yr, bool near, V2<R>& J, R (&g)[5], R& po) {
      int ey = yr, ty = -1;
      if (yr < 0) {
        if (d.bc[2]) { ey = 0; ty = d.bc[2]; } else ey = yr + ny;
      } else if (yr >= ny) {
        if (d.bc[3]) { ey = ny - 1; ty = d.bc[3]; } else ey = yr - ny;
      }
      R v[NF];
      if (near) pull_hg_b<S, R, BIG, IO>(a, d, col, ey, J, g, v[0], v[1], po);
      else pull_hg<S, R, BIG>(a, sources(d, col, ey), J, g, v[0], v[1], po);
      const unsigned s0 = site_at(d, col, ey);
      v[2] = ld<R>(pbase<BIG>(a.ain, A_VXO, ps), pidx<BIG>(A_VXO, ps, s0));
      v[3] = ld<R>(pbase<BIG>(a.ain, A_VYO, ps), pidx<BIG>(A_VYO, ps, s0));
      if constexpr (TH)
        v[4] = near ? pull_U_b<S, R, BIG, IO>(a, d, col, ey, v[1])
                    : pull_U<S, R, BIG>(a, sources(d, col, ey), v[1]);
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        R u = v[f];
        if (ty >= 0) u = ghost_map<R, IO>(a.kp, ty, 1, f, u);
        if (tx >= 0) u = ghost_map<R, IO>(a.kp, tx, 0, f, u);
        ring[f][yr & 3][sc] = u;
      }
    };

    const SiteDom<R> sd(d);
    V2<R> JC = vec2(R(0), R(0));
    R gC[5], poC = R(0);
    for (int k = 0; k < 2; ++k) {
      const bool near = near_col || side_row(inside_row(ya - 1 + k));
      if (active) {
        V2<R> J;
        R g[5], po;
        fill(ya - 1 + k, near, J, g, po);
        if (k == 1) {
          JC = J;
#pragma unroll
          for (int i = 0; i < 5; ++i) gC[i] = g[i];
          poC = po;
        }
      }
    }

    for (int j = ya; j < yb; ++j) {
      SiteIn<R> in;
      Src9 srcj;
      if (interior) {
        if (near_in || side_row(j)) {
          load_site_b<S, R, BIG, TH, IO>(a, d, col, j, in);
          srcj.s[0] = site_at(d, col, j);
        } else {
          srcj = sources(d, col, j);
          load_site<S, R, BIG, TH>(a, srcj, in);
        }
      }
      V2<R> JL = vec2(R(0), R(0));
      R gL[5], poL = R(0);
      if (active) fill(j + 1, near_col || side_row(inside_row(j + 1)), JL, gL, poL);
      if (interior) load_grain(a, sd, in);
      __syncthreads();
      if (interior) {
        const int m = (j - 1) & 3, c0 = j & 3, pp = (j + 1) & 3;
        auto rows = [&](int f) { return Rows3<R>{ring[f][m], ring[f][c0], ring[f][pp]}; };
        site_update<S, R, TH>(a, sd, srcj, in, JC, gC, poC, rows(0), rows(1), rows(2), rows(3),
                              sc, rows(NF - 1));
      }
      JC = JL;
#pragma unroll
      for (int i = 0; i < 5; ++i) gC[i] = gL[i];
      poC = poL;
    }
    __syncthreads();
  }
}

template <typename S, typename R>
cudaError_t launch_ymarch_bc(const StepArgs<S, R>& a, bool big, int grid, cudaStream_t st) {
  if constexpr (sizeof(S) == sizeof(R)) {
    // a.bc: 1 boundary sides, 2 among them an inlet or an outlet
    cudaError_t e = cudaSuccess;
    auto go = [&](auto io) {
      constexpr bool IO = decltype(io)::value;
      if (big) {
        if (a.thermal) e = launch_chained(k_step_ymarch_bc<S, R, true, true, IO>, a, grid, 0, st);
        else e = launch_chained(k_step_ymarch_bc<S, R, true, false, IO>, a, grid, 0, st);
      } else {
        if (a.thermal) e = launch_chained(k_step_ymarch_bc<S, R, false, true, IO>, a, grid, 0, st);
        else e = launch_chained(k_step_ymarch_bc<S, R, false, false, IO>, a, grid, 0, st);
      }
    };
    if (a.bc == 2) go(std::true_type{});
    else go(std::false_type{});
    return e;
  } else {
    return cudaErrorInvalidValue;   // boundaries need FP32 or FP64 storage (checked on the host)
  }
}

template <typename S, typename R>
int ymarch_bc_blocks_per_sm(bool big, bool thermal) {
  int n = 0;
  if constexpr (sizeof(S) == sizeof(R)) {
    if (big) {
      if (thermal)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step_ymarch_bc<S, R, true, true, true>, YM_THREADS, 0);
      else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step_ymarch_bc<S, R, true, false, true>, YM_THREADS, 0);
    } else {
      if (thermal)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step_ymarch_bc<S, R, false, true, true>, YM_THREADS, 0);
      else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step_ymarch_bc<S, R, false, false, true>, YM_THREADS, 0);
    }
  }
  return n > 0 ? n : 1;
}

#define PF_BC_INST(S, R)                                                                  \
  template cudaError_t launch_ymarch_bc<S, R>(const StepArgs<S, R>&, bool, int, cudaStream_t); \
  template int ymarch_bc_blocks_per_sm<S, R>(bool, bool);
PF_BC_INST(double, double)
PF_BC_INST(float, float)
PF_BC_INST(__half, float)
PF_BC_INST(__nv_bfloat16, float)

}  // namespace pf
