// pf_step_general.cu -- k_step_general: one coupled step from a raw state whose
// populations are arbitrary.
//
// The step kernels keep one population of each opposite pair where a collision
// fixes the other (pf_model.cuh).  A state that came out of a step or of an
// initialisation has that form; one written by pf_set_state need not.  Such a
// state keeps every population of those lattices in planes beside the stored
// ones (pf_raw.cuh), this kernel takes the first step from them with the
// pulls, sides and per-site arithmetic of the other kernels, and what it
// writes is a collision's output again.  It runs once after such a call, so it
// is written for any lattice rather than for speed: 32 x 8 tiles with a halo
// of the stencil fields in shared memory.
#include "pf_raw.cuh"

namespace pf {

constexpr int GX = 32, GY = 8;

template <typename S, typename R, bool TH>
__global__ void __launch_bounds__(GX * GY) k_step_general(StepArgs<S, R> a, DomDesc d,
                                                          const S* tied) {
  constexpr int NF = TH ? 5 : 4;
  __shared__ R ring[NF][GY + 2][GX + 2];
  const GeneralPull<S, R, TH> pull{tied, a, d};
  const int tiles_x = (d.nx + GX - 1) / GX;
  const int x0 = (int)(blockIdx.x % tiles_x) * GX, y0 = (int)(blockIdx.x / tiles_x) * GY;
  const int tid = threadIdx.y * GX + threadIdx.x;
  for (int i = tid; i < (GX + 2) * (GY + 2); i += GX * GY) {
    const int lx = i % (GX + 2), ly = i / (GX + 2);
    int ex = x0 + lx - 1, ey = y0 + ly - 1, tx = -1, ty = -1;
    if (ex > d.nx || ey > d.ny) continue;   // beyond a ragged tile's own ghosts
    if (ex < 0 || ex >= d.nx) {
      const int t = d.bc[ex < 0 ? 0 : 1];
      if (t) { ex = ex < 0 ? 0 : d.nx - 1; tx = t; }
      else ex += ex < 0 ? d.nx : -d.nx;
    }
    if (ey < 0 || ey >= d.ny) {
      const int t = d.bc[ey < 0 ? 2 : 3];
      if (t) { ey = ey < 0 ? 0 : d.ny - 1; ty = t; }
      else ey += ey < 0 ? d.ny : -d.ny;
    }
    R v[NF], g[5], po;
    V2<R> J;
    pull.hg(ex, ey, J, g, v[0], v[1], po);
    v[2] = pull.aux(A_VXO, site_at(d, ex, ey));
    v[3] = pull.aux(A_VYO, site_at(d, ex, ey));
    if constexpr (TH) {
      R sv[5];
      pull.solute(ex, ey, sv);
      v[4] = supersat(a.kp, sv, v[1]);
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      R u = v[f];
      if (ty >= 0) u = ghost_map<R, true>(a.kp, ty, 1, f, u);
      if (tx >= 0) u = ghost_map<R, true>(a.kp, tx, 0, f, u);
      ring[f][ly][lx] = u;
    }
  }
  __syncthreads();
  const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
  if (x >= d.nx || y >= d.ny) return;
  V2<R> J;
  R g[5], phi, psi, po;
  pull.hg(x, y, J, g, phi, psi, po);
  SiteIn<R> in;
  pull.site(x, y, in);
  const SiteDom<R> sd(d);
  load_grain(a, sd, in);
  Src9 src;
  src.s[0] = site_at(d, x, y);
  const int r = threadIdx.y;
  auto rows = [&](int f) { return Rows3<R>{ring[f][r], ring[f][r + 1], ring[f][r + 2]}; };
  site_update<S, R, TH>(a, sd, src, in, J, g, po, rows(0), rows(1), rows(2), rows(3),
                        threadIdx.x + 1, rows(NF - 1));
}

template <typename S, typename R>
cudaError_t launch_step_general(const StepArgs<S, R>& a, const DomDesc& d, const S* tied,
                                cudaStream_t st) {
  const unsigned tiles = (unsigned)((d.nx + GX - 1) / GX) * (unsigned)((d.ny + GY - 1) / GY);
  if constexpr (sizeof(S) == sizeof(R)) {
    if (a.thermal) {
      k_step_general<S, R, true><<<tiles, dim3(GX, GY), 0, st>>>(a, d, tied);
      return cudaGetLastError();
    }
  }
  k_step_general<S, R, false><<<tiles, dim3(GX, GY), 0, st>>>(a, d, tied);
  return cudaGetLastError();
}

#define PF_GENERAL_INST(S, R)                                                             \
  template cudaError_t launch_step_general<S, R>(const StepArgs<S, R>&, const DomDesc&,   \
                                                 const S*, cudaStream_t);
PF_GENERAL_INST(double, double)
PF_GENERAL_INST(float, float)
PF_GENERAL_INST(__half, float)
PF_GENERAL_INST(__nv_bfloat16, float)

}  // namespace pf
