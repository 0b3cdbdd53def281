// pf_step_general.cu -- one coupled step from a raw state whose populations are
// arbitrary.
//
// The step kernels keep one population of each opposite pair where a collision
// fixes the other (pf_model.cuh).  A state that came out of a step or of an
// initialisation has that form; one written by pf_set_state need not.  Such a
// state keeps every population of those lattices in planes beside the stored
// ones (pf_raw.cuh), these kernels take the first step from them with the
// pulls, sides and per-site arithmetic of the other kernels (k_step_tied for
// pf_step, k_step_general for the adjoint's sweeps), and what they write is a
// collision's output again.  They run once after such a call, so they are
// written for any lattice rather than for speed: 32 x 8 tiles with a halo of
// the stencil fields in shared memory.
#include "pf_raw.cuh"
#include "pf_reduce.cuh"

namespace pf {

constexpr int GX = 32, GY = 8;

// One 32 x 8 tile of a raw domain, by the 256 threads of a block.
template <typename S, typename R, bool TH>
__device__ __forceinline__ void general_tile(const StepArgs<S, R>& a, const DomDesc& d,
                                             const S* tied, int tile,
                                             R (*ring)[GY + 2][GX + 2]) {
  constexpr int NF = TH ? 5 : 4;
  const GeneralPull<S, R, TH> pull{tied, a, d};
  const int tiles_x = (d.nx + GX - 1) / GX;
  const int x0 = (tile % tiles_x) * GX, y0 = (tile / tiles_x) * GY;
  const int tid = threadIdx.x, tx = tid % GX, ty = tid / GX;
  for (int i = tid; i < (GX + 2) * (GY + 2); i += GX * GY) {
    const int lx = i % (GX + 2), ly = i / (GX + 2);
    int ex = x0 + lx - 1, ey = y0 + ly - 1, gx = -1, gy = -1;
    if (ex > d.nx || ey > d.ny) continue;   // beyond a ragged tile's own ghosts
    if (ex < 0 || ex >= d.nx) {
      const int t = d.bc[ex < 0 ? 0 : 1];
      if (t) { ex = ex < 0 ? 0 : d.nx - 1; gx = t; }
      else ex += ex < 0 ? d.nx : -d.nx;
    }
    if (ey < 0 || ey >= d.ny) {
      const int t = d.bc[ey < 0 ? 2 : 3];
      if (t) { ey = ey < 0 ? 0 : d.ny - 1; gy = t; }
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
      if (gy >= 0) u = ghost_map<R, true>(a.kp, gy, 1, f, u);
      if (gx >= 0) u = ghost_map<R, true>(a.kp, gx, 0, f, u);
      ring[f][ly][lx] = u;
    }
  }
  __syncthreads();
  const int x = x0 + tx, y = y0 + ty;
  if (x < d.nx && y < d.ny) {
    V2<R> J;
    R g[5], phi, psi, po;
    pull.hg(x, y, J, g, phi, psi, po);
    SiteIn<R> in;
    pull.site(x, y, in);
    const SiteDom<R> sd(d);
    load_grain(a, sd, in);
    Src9 src;
    src.s[0] = site_at(d, x, y);
    auto rows = [&](int f) { return Rows3<R>{ring[f][ty], ring[f][ty + 1], ring[f][ty + 2]}; };
    site_update<S, R, TH>(a, sd, src, in, J, g, po, rows(0), rows(1), rows(2), rows(3), tx + 1,
                          rows(NF - 1));
  }
  __syncthreads();   // the ring is the next tile's
}

static inline int tiles_of(const DomDesc& d) {
  return ((d.nx + GX - 1) / GX) * ((d.ny + GY - 1) / GY);
}

template <typename S, typename R, bool TH>
__global__ void __launch_bounds__(GX * GY) k_step_general(StepArgs<S, R> a, DomDesc d,
                                                          const S* tied) {
  __shared__ R ring[TH ? 5 : 4][GY + 2][GX + 2];
  general_tile<S, R, TH>(a, d, tied, (int)blockIdx.x, ring);
}

template <typename S, typename R>
cudaError_t launch_step_general(const StepArgs<S, R>& a, const DomDesc& d, const S* tied,
                                cudaStream_t st) {
  if constexpr (sizeof(S) == sizeof(R)) {
    if (a.thermal) {
      k_step_general<S, R, true><<<tiles_of(d), GX * GY, 0, st>>>(a, d, tied);
      return cudaGetLastError();
    }
  }
  k_step_general<S, R, false><<<tiles_of(d), GX * GY, 0, st>>>(a, d, tied);
  return cudaGetLastError();
}

// The raw domains of a pf_step call's first step.  Which they are is known when
// the kernel runs, from the table of tied planes: the step may be in a caller's
// graph.  Row b of the table holds, for state buffer b, whether any domain is raw
// and then each domain's tied planes (0: none); `row` is the buffer the step read.
// The step's own kernels have updated every domain; the raw ones are written
// again from their tied planes.  Then the entries of the buffers that the call
// overwrites go: the other one, and with `both` (calls of two steps and more) this
// one.  In a graph nothing to do is the common case, and costs the launch.
template <typename S, typename R, bool TH>
__global__ void __launch_bounds__(GX * GY) k_step_tied(StepArgs<S, R> a,
                                                       const DomDesc* __restrict__ doms, int n_doms,
                                                       unsigned long long* table, int row, int both,
                                                       unsigned int* ctr) {
  __shared__ R ring[TH ? 5 : 4][GY + 2][GX + 2];
  unsigned long long* mine = table + (size_t)row * (n_doms + 1);
  unsigned long long* other = table + (size_t)(row ^ 1) * (n_doms + 1);
  if (!mine[0] && !other[0]) return;   // in every block: only the last one changes them
  if (mine[0]) {
    for (int k = 0; k < n_doms; ++k) {
      const S* tied = reinterpret_cast<const S*>(mine[1 + k]);
      if (!tied) continue;
      const DomDesc d = doms[k];
      const int tiles = ((d.nx + GX - 1) / GX) * ((d.ny + GY - 1) / GY);
      for (int t = blockIdx.x; t < tiles; t += gridDim.x) general_tile<S, R, TH>(a, d, tied, t, ring);
    }
  }
  if (!last_block(ctr)) return;
  for (int k = threadIdx.x; k <= n_doms; k += GX * GY) {
    other[k] = 0;
    if (both) mine[k] = 0;
  }
}

template <typename S, typename R>
cudaError_t launch_step_tied(const StepArgs<S, R>& a, const DomDesc* doms, int n_doms,
                             unsigned long long* table, int row, int both, unsigned int* ctr,
                             int grid, cudaStream_t st) {
  if constexpr (sizeof(S) == sizeof(R)) {
    if (a.thermal) {
      k_step_tied<S, R, true><<<grid, GX * GY, 0, st>>>(a, doms, n_doms, table, row, both, ctr);
      return cudaGetLastError();
    }
  }
  k_step_tied<S, R, false><<<grid, GX * GY, 0, st>>>(a, doms, n_doms, table, row, both, ctr);
  return cudaGetLastError();
}

#define PF_GENERAL_INST(S, R)                                                             \
  template cudaError_t launch_step_general<S, R>(const StepArgs<S, R>&, const DomDesc&,   \
                                                 const S*, cudaStream_t);                 \
  template cudaError_t launch_step_tied<S, R>(const StepArgs<S, R>&, const DomDesc*, int, \
                                              unsigned long long*, int, int,              \
                                              unsigned int*, int, cudaStream_t);
PF_GENERAL_INST(double, double)
PF_GENERAL_INST(float, float)
PF_GENERAL_INST(__half, float)
PF_GENERAL_INST(__nv_bfloat16, float)

}  // namespace pf
