// pf_step_staged.cu -- k_step_staged: the coupled LB step (arXiv 2407.01651)
// as a y-marched column strip whose input rows are staged in shared memory by
// the bulk-copy (TMA) engine D rows ahead of the arithmetic.
//
// The arithmetic per site is the one of every other traversal (pf_site.cuh);
// what differs is how the inputs reach it.  Every plane that a site reads at
// its neighbours (f, h, g_post, s, r = 1/a_s^2 and the lagged phi and C that
// give the opposite populations of the stored pairs; in the 16-bit forms also
// the lagged psi) is copied row by row with cp.async.bulk into rings of row
// slots, each stage completing on its own mbarrier.  Planes that only the site
// itself reads (g_pre, the lagged velocity, Q_psi, the grain id) are loaded
// into registers one row ahead of their use.  So no warp waits on HBM inside the
// arithmetic of a row.  Bound by instruction issue (65 % of the slots in FP32, 72 %
// in FP16) and HBM together; us per step, direct loads and staged: FP32 4096^2 828
// and 676; six-slot rings and these: FP16 8192x4096 1663 and 1322.
//
// Shared memory.  Iteration j streams row j+1 and updates row j; stage r is what
// arrives for the streaming of row r - 1 and the update of row r - 2, D stages
// are on their way while a row is updated.  Each group of planes keeps the rows
// that are still to be read, no more:
//   H  h, g_post, r, phi_o (psi_o)  rows j .. j+2, free after the streaming
//   S  s, C_o                       rows j-1 .. j+1 (thermal: .. j+2, for U)
//   E  temperature pairs            rows j-1 .. j+1
//   F  the nine NS rows of one update (f_i at row j - cy_i)
// With every plane in six slots (103 KB in FP32) two CTAs fitted an SM; now four
// do (51 KB, D = 2).  Both matter: at D = 1 every row waited for its copies (FP32
// 832 us a step at 4096^2, against 796 with D = 2 and three CTAs).
//
// Each slot row holds, per staged plane, the strip's interior columns plus
// 16 bytes of halo on each side (the two copies of the halo wrap around the
// periodic x boundary on their own).  Requirements (checked on the host):
// nx a multiple of 16 / sizeof(storage) and of 16 / sizeof(compute), and
// 16-byte aligned plane bases.
#include "pf_site.cuh"

namespace pf {

namespace {

template <typename S, typename R, bool TH>
struct Stage {
  static constexpr int HS = 16 / (int)sizeof(S);   // halo columns of a storage plane
  static constexpr int HR = 16 / (int)sizeof(R);   // halo columns of a compute plane
  static constexpr int PWS = YM_W + 2 * HS;        // staged width, storage planes
  static constexpr int PWR = YM_W + 2 * HR;        // staged width, compute planes
  static constexpr int BS = PWS * (int)sizeof(S), BR = PWR * (int)sizeof(R);   // bytes of a row
  static constexpr bool OFF = Codec<S>::kOffset;
  static constexpr int D = OFF ? 3 : 2;
  // planes of a row: storage type, then compute type
  static constexpr int HP = 7, HA = OFF ? 3 : 2, SP = 2, SA = 1, EP = TH ? 3 : 0, FP = 9;
  static constexpr int H_BYTES = HP * BS + HA * BR, S_BYTES = SP * BS + SA * BR, E_BYTES = EP * BS,
                       F_BYTES = FP * BS;
  static constexpr int NH = 2 + D, NSR = (TH ? 4 : 3) + D, NE = 3 + D, NFR = 1 + D;   // rows held
  static constexpr int S_AT = NH * H_BYTES, E_AT = S_AT + NSR * S_BYTES,
                       F_AT = E_AT + NE * E_BYTES, RING_AT = F_AT + NFR * F_BYTES;
  static constexpr int NF = TH ? 5 : 4;
  static constexpr int RW = YM_W + 2;
  static constexpr int RING_BYTES = NF * 4 * RW * (int)sizeof(R);
  static constexpr int BAR_AT = RING_AT + RING_BYTES;
  static constexpr int SMEM = BAR_AT + NH * 8;
  static constexpr int MIN_BLOCKS = sizeof(S) == 8 ? 2 : (TH ? 3 : 4);
  static_assert(BS % 16 == 0 && BR % 16 == 0 && RING_BYTES % 8 == 0,
                "16-byte staged rows, 8-byte barriers");
  static_assert(HS >= 2 && HR >= 2, "the halo streaming reaches two columns out");
};

// ---- mbarrier and bulk copy (PTX) ----
__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void bar_init(unsigned bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool bar_try(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Wait for the phase of `bar` with parity `parity`; gives up after about one
// second (or 2^24 polls) and returns false.
__device__ __forceinline__ bool bar_wait(unsigned bar, unsigned parity) {
  if (bar_try(bar, parity)) return true;
  const unsigned long long t0 = globaltimer();
  for (unsigned it = 0; it < (1u << 24); ++it) {
    if (bar_try(bar, parity)) return true;
    if ((it & 255u) == 255u && globaltimer() - t0 > 1000000000ull) break;
  }
  return false;
}
__device__ __forceinline__ void bulk_g2s(unsigned dst, const void* src, unsigned bytes,
                                         unsigned bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

// Copy one staged plane row: columns [x0 - H, x0 + w + H) of the strip, the
// halos wrapping around the periodic x boundary.  A strip away from both x
// boundaries is one contiguous piece.
template <typename E>
__device__ __forceinline__ void copy_plane_row(unsigned dst, const E* src, int x0, int w, int nx,
                                               int H, unsigned bar) {
  const bool wl = x0 == 0, wr = x0 + w == nx;
  const unsigned hb = (unsigned)(H * sizeof(E)), wb = (unsigned)(w * sizeof(E));
  if (!wl && !wr) {
    bulk_g2s(dst, src + x0 - H, wb + 2 * hb, bar);
  } else if (!wr) {
    bulk_g2s(dst, src + nx - H, hb, bar);
    bulk_g2s(dst + hb, src + x0, wb + hb, bar);
  } else if (!wl) {
    bulk_g2s(dst, src + x0 - H, hb + wb, bar);
    bulk_g2s(dst + hb + wb, src, hb, bar);
  } else {
    bulk_g2s(dst, src + nx - H, hb, bar);
    bulk_g2s(dst + hb, src + x0, wb, bar);
    bulk_g2s(dst + hb + wb, src, hb, bar);
  }
}

// Source row of D2Q9 direction i: row - cy_i, as 0 (row-1), 1 (row), 2 (row+1).
__device__ __forceinline__ constexpr int src_row(int i) {
  return (i == 2 || i == 5 || i == 6) ? 0 : ((i == 4 || i == 7 || i == 8) ? 2 : 1);
}
// Source column offset of direction i: -cx_i.
__device__ __forceinline__ constexpr int src_dx(int i) {
  return (i == 1 || i == 5 || i == 8) ? -1 : ((i == 3 || i == 6 || i == 7) ? 1 : 0);
}

// Row of the periodic lattice for a row at most two beyond it (ny >= 4).
__device__ __forceinline__ int wrap2(int row, int ny) {
  return row < 0 ? row + ny : (row >= ny ? row - ny : row);
}

// Slots of a stage's rows; a group that the stage does not carry has none (-1).
struct Slots {
  int h, s, e, f;
};

// Issue the copies of stage r.  Called by the last warp (whose other lanes own
// no column): lane 0 announces the byte count on the stage's mbarrier, each lane
// copies one plane row.
template <typename S, typename R, bool TH>
__device__ __forceinline__ void issue_stage(const StepArgs<S, R>& a, const DomDesc& d, int r,
                                            Slots sl, int x0, int w, unsigned char* smem,
                                            unsigned bar, int lane) {
  using G = Stage<S, R, TH>;
  if (a.drop_copies) return;   // testing only: the waits on this stage time out
  const bool hs = sl.s >= 0, he = TH && sl.e >= 0, hf = sl.f >= 0;
  if (lane == 0) {
    const unsigned pw = (w + 2 * G::HS) * sizeof(S), aw = (w + 2 * G::HR) * sizeof(R);
    bar_expect(bar, (G::HP + (hs ? G::SP : 0) + (he ? G::EP : 0) + (hf ? G::FP : 0)) * pw +
                        (G::HA + (hs ? G::SA : 0)) * aw);
  }
  // lanes: H storage, H compute, S storage, C_o, E, F
  constexpr int L1 = G::HP, L2 = L1 + G::HA, L3 = L2 + G::SP, L4 = L3 + 1, L5 = L4 + G::EP,
                L6 = L5 + G::FP;
  static_assert(L6 <= 32, "a lane per plane row");
  int k, row = r, off;
  bool go = true, aux = false;
  if (lane < L1) {
    k = lane < 4 ? P_H + lane : P_GPOST + lane - 4;
    off = sl.h * G::H_BYTES + lane * G::BS;
  } else if (lane < L2) {
    const int u = lane - L1;
    k = u == 0 ? A_RR : (u == 1 ? A_PHIO : A_PSIO);
    off = sl.h * G::H_BYTES + G::HP * G::BS + u * G::BR;
    aux = true;
  } else if (lane < L4) {
    row = TH ? r : r - 1;
    aux = lane == L3;
    k = aux ? A_CO : P_S + lane - L2;
    off = G::S_AT + sl.s * G::S_BYTES + (lane - L2) * G::BS;
    go = hs;
  } else if (lane < L5) {
    row = r - 1;
    k = P_E + 1 + lane - L4;
    off = G::E_AT + sl.e * G::E_BYTES + (lane - L4) * G::BS;
    go = he;
  } else {
    const int i = lane - L5;
    row = r - 2 - ((i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0));
    k = P_F + i;
    off = G::F_AT + sl.f * G::F_BYTES + i * G::BS;
    go = hf && lane < L6;
  }
  if (!go) return;
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  const unsigned ps = (unsigned)a.plane_stride;
  const unsigned at = (unsigned)d.off + (unsigned)wrap2(row, d.ny) * (unsigned)d.nx;
  const unsigned dst = smem_u32(smem + off);
  if (aux) copy_plane_row<R>(dst, plane(a.ain, k, ps) + at, x0, w, d.nx, G::HR, bar);
  else copy_plane_row<S>(dst, plane(a.in, k, ps) + at, x0, w, d.nx, G::HS, bar);
}

// A staged row seen from a thread's column: planes of the storage type, then NP
// of them on of the compute type.
template <typename S, typename R, bool TH, int NP>
struct RowView {
  using G = Stage<S, R, TH>;
  const S* pop;
  const R* aux;
  __device__ __forceinline__ RowView(const unsigned char* row, int dx)
      : pop(reinterpret_cast<const S*>(row) + dx + G::HS),
        aux(reinterpret_cast<const R*>(row + NP * G::BS) + dx + G::HR) {}
  __device__ __forceinline__ S p(int q, int dx) const { return pop[q * G::PWS + dx]; }
  __device__ __forceinline__ R x(int u, int dx) const { return aux[u * G::PWR + dx]; }
};
constexpr int U_RR = 0, U_PHIO = 1, U_PSIO = 2;   // compute planes of an H row

template <typename S, typename R>
__device__ __forceinline__ R dec(S v) {
  return Codec<S>::template dec<R>(v);
}
template <typename S, typename R>
__device__ __forceinline__ R dec_ns(S v) {
  if constexpr (Codec<S>::kOffset) return dec<S, R>(v) * R(kNSInvScale);
  else return dec<S, R>(v);
}

// Own-site inputs of the streaming of one row (loaded a row ahead).
template <typename S, typename R>
struct OwnHG {
  S gpre[5];
  R vxo, vyo;
};
// Own-site inputs of the update of one row (loaded a row ahead).
template <typename R>
struct OwnSite {
  R Qo, mo;      // mo: lagged rho H (thermal mode)
  uint8_t gid;
};

template <typename S, typename R>
__device__ __forceinline__ void load_own_hg(const StepArgs<S, R>& a, unsigned site, OwnHG<S, R>& o) {
  const unsigned ps = (unsigned)a.plane_stride;
#pragma unroll
  for (int i = 0; i < 5; ++i) o.gpre[i] = ldp(plane(a.in, P_GPRE + i, ps) + site);
  o.vxo = ldp(plane(a.ain, A_VXO, ps) + site);
  o.vyo = ldp(plane(a.ain, A_VYO, ps) + site);
}
template <typename S, typename R, bool TH>
__device__ __forceinline__ void load_own_site(const StepArgs<S, R>& a, unsigned site,
                                              OwnSite<R>& o) {
  const unsigned ps = (unsigned)a.plane_stride;
  o.Qo = ldp(plane(a.ain, A_QO, ps) + site);
  o.gid = __ldg(a.grain + site);
  if constexpr (TH) o.mo = ld<R>(plane(a.in, P_E, ps), site);
}

// Streamed CAC moments and g of the thread's site in the middle of the rows, and
// its phi_o; same arithmetic as pull_hg.
template <typename S, typename R, typename View>
__device__ __forceinline__ void stream_hg(const View (&rows)[3], const OwnHG<S, R>& own,
                                          V2<R>& J, R g[5], R& phi, R& psi, R& psio, R& phio) {
  constexpr bool off = Codec<S>::kOffset;
  HgLoads<S, R> l;
  l.ph[0] = phio = rows[1].x(U_PHIO, 0);
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    l.h[i] = rows[src_row(i)].p(pair9(i), src_dx(i));
    if (off || minus9(i)) l.ph[i] = rows[src_row(i)].x(U_PHIO, src_dx(i));
  }
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const View& r = rows[src_row(i)];
    l.gpre[i] = own.gpre[i];
    if (i > 0) l.gp[i] = r.p(5 + pair9(i), src_dx(i));
    if (i == 0 || minus9(i)) l.gm[i] = r.p(4, src_dx(i));
    if (off) l.po[i] = r.x(U_PSIO, src_dx(i));
    l.rr[i] = r.x(U_RR, src_dx(i));
  }
  finish_hg<S, R>(l, J, g, phi, psi, psio);
}

// Streamed s of the thread's site.
template <typename S, typename R, typename View>
__device__ __forceinline__ void stream_s(const View (&rows)[3], R Co, R (&s)[5]) {
  constexpr bool off = Codec<S>::kOffset;
  s[0] = q5_rest(Co, q5_base(Co));
#pragma unroll
  for (int i = 1; i < 5; ++i) {
    const View& r = rows[src_row(i)];
    const S v = r.p(pair9(i), src_dx(i));
    const R base = off || minus9(i) ? q5_base(r.x(0, src_dx(i))) : R(0);
    s[i] = minus9(i) ? pair_m<S, R>(v, base) : pair_p<S, R>(v, base);
  }
}

}  // namespace

template <typename S, typename R, bool TH>
__global__ void __launch_bounds__(YM_THREADS, (Stage<S, R, TH>::MIN_BLOCKS))
    k_step_staged(StepArgs<S, R> a) {
  using G = Stage<S, R, TH>;
  using HView = RowView<S, R, TH, G::HP>;
  using SView = RowView<S, R, TH, G::SP>;
  using EView = RowView<S, R, TH, G::EP>;
  extern __shared__ __align__(128) unsigned char smem[];
  R(*ring)[4][G::RW] = reinterpret_cast<R(*)[4][G::RW]>(smem + G::RING_AT);
  const unsigned bar0 = smem_u32(smem + G::BAR_AT);
  const int t = threadIdx.x;

  if (t < G::NH) bar_init(bar0 + 8 * t);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  chain_step(a);

  unsigned phase = 0;   // bit s: parity of the next completion of barrier s
  bool bad = false;     // a copy did not arrive within the time limit
  auto next = [](int s, int n) { return s + 1 == n ? 0 : s + 1; };
  auto prev = [](int s, int n) { return s == 0 ? n - 1 : s - 1; };
  // stage r completes on barrier (r - first stage) mod NH, the slot of its H row
  auto wait = [&](int s) {
    if (!bar_wait(bar0 + 8 * s, (phase >> s) & 1u)) bad = true;
    phase ^= 1u << s;
  };

  for (int tile = a.tile_base + blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    const DomDesc d = a.doms[a.tile_dom[tile]];
    const int lt = tile - d.tile0;
    const int nx = d.nx, ny = d.ny;
    const int x0 = (lt % d.tiles_x) * YM_W;
    const int ya = (lt / d.tiles_x) * a.chunk;
    const int yb = min(ya + a.chunk, ny);
    const int w = min(YM_W, nx - x0);
    const int rlast = yb + 1;        // last stage of the tile
    bool interior = false, active = false;
    int col = 0, dx = 0;
    if (t < YM_W) {
      interior = active = t < w;
      col = x0 + t;
      dx = t;
    } else if (t == YM_W) {
      active = true;
      col = x0 == 0 ? nx - 1 : x0 - 1;
      dx = -1;
    } else if (t == YM_W + 1) {
      active = true;
      col = x0 + w >= nx ? x0 + w - nx : x0 + w;
      dx = w;
    }
    const int sc = dx + 1;   // ring column
    auto site_of = [&](int row) {
      return (unsigned)d.off + (unsigned)wrap2(row, ny) * (unsigned)nx + (unsigned)col;
    };
    auto issue = [&](int r, Slots sl) {
      if (t >= YM_W) issue_stage<S, R, TH>(a, d, r, sl, x0, w, smem, bar0 + 8 * sl.h, t - YM_W);
    };
    // the first NH stages; S rows start at ya - 1 (TH: ya - 2), E rows at ya - 1,
    // F at the update of ya
    int issued = ya - 3;
    for (int k = 0; k < G::NH && ya - 2 + k <= rlast; ++k) {
      issued = ya - 2 + k;
      issue(issued, Slots{k, TH ? k : k - 2, k - 2, k - 4});
    }
    const SiteDom<R> sd(d);
    OwnHG<S, R> ohg;
    OwnSite<R> osC{};
    V2<R> JC = vec2(R(0), R(0));
    R gC[5], poC = R(0), phC = R(0);
    if (active) load_own_hg(a, site_of(ya - 1), ohg);
    wait(0);
    wait(1);

    // slots: H row j, S and E row j - 1, F of the update of row j
    int h0 = 0, sm = TH ? G::NSR - 1 : G::NSR - 2, em = G::NE - 2, fu = G::NFR - 2;
    for (int j = ya - 2; j < yb; ++j) {
      const int h1 = next(h0, G::NH), h2 = next(h1, G::NH);
      const int s0 = next(sm, G::NSR), s1 = next(s0, G::NSR);
      wait(h2);
      // streaming of row j+1 into the stencil ring
      V2<R> JL = vec2(R(0), R(0));
      R gL[5], poL = R(0), phL = R(0);
      if (active) {
        const HView rows[3] = {HView(smem + h0 * G::H_BYTES, dx), HView(smem + h1 * G::H_BYTES, dx),
                               HView(smem + h2 * G::H_BYTES, dx)};
        const int y = (j + 1) & 3;
        R phi, psi;
        stream_hg<S, R>(rows, ohg, JL, gL, phi, psi, poL, phL);
        ring[0][y][sc] = phi;
        ring[1][y][sc] = psi;
        ring[2][y][sc] = ohg.vxo;
        ring[3][y][sc] = ohg.vyo;
        if constexpr (TH) {
          const int s2 = next(s1, G::NSR);
          const unsigned char* sb = smem + G::S_AT;
          const SView sr[3] = {SView(sb + s0 * G::S_BYTES, dx), SView(sb + s1 * G::S_BYTES, dx),
                               SView(sb + s2 * G::S_BYTES, dx)};
          R sv[5];
          stream_s<S, R>(sr, sr[1].x(0, 0), sv);
          ring[G::NF - 1][y][sc] = supersat(a.kp, sv, psi);
        }
        if (j + 1 < yb) load_own_hg(a, site_of(j + 2), ohg);
      }
      SiteIn<R> in;
      in.gid = osC.gid;
      const bool update = interior && j >= ya;
      if (update) load_grain(a, sd, in);
      OwnSite<R> osN{};
      if (interior && j + 1 >= ya && j + 1 < yb) load_own_site<S, R, TH>(a, site_of(j + 1), osN);
      if (__syncthreads_or(bad)) {
        // drain the stages still in flight (bounded), report, stop
        for (int r = j + 3, q = next(h2, G::NH); r <= issued; ++r, q = next(q, G::NH)) wait(q);
        if (t == 0 && a.err) atomicOr(a.err, 1u);
        return;
      }
      // stage j + 2 + D into the slots whose last readers ran before this barrier:
      // H row j, S and E row j - 2, F of the update of row j - 1
      if (j + 2 + G::D <= rlast) {
        issued = j + 2 + G::D;
        issue(issued, Slots{h0, prev(sm, G::NSR), prev(em, G::NE), prev(fu, G::NFR)});
      }
      if (update) {
        {
          const S* f = reinterpret_cast<const S*>(smem + G::F_AT + fu * G::F_BYTES) + dx + G::HS;
#pragma unroll
          for (int i = 0; i < 9; ++i) in.f[i] = dec_ns<S, R>(f[i * G::PWS + src_dx(i)]);
          const unsigned char* sb = smem + G::S_AT;
          const SView rows[3] = {SView(sb + sm * G::S_BYTES, dx), SView(sb + s0 * G::S_BYTES, dx),
                                 SView(sb + s1 * G::S_BYTES, dx)};
          in.phio = phC;
          in.Co = rows[1].x(0, 0);
          stream_s<S, R>(rows, in.Co, in.s);
          in.Qo = osC.Qo;
          if constexpr (TH) {
            const int e0 = next(em, G::NE), e1 = next(e0, G::NE);
            const unsigned char* eb = smem + G::E_AT;
            const EView m(eb + em * G::E_BYTES, dx), c(eb + e0 * G::E_BYTES, dx),
                p(eb + e1 * G::E_BYTES, dx);
            in.mo = osC.mo;
            in.e[0] = q5_rest(in.mo, (R)c.p(0, 0));
            in.e[1] = (R)c.p(1, -1);
            in.e[2] = (R)m.p(2, 0);
            in.e[3] = fma(R(2), (R)c.p(0, 1), -(R)c.p(1, 1));
            in.e[4] = fma(R(2), (R)p.p(0, 0), -(R)p.p(2, 0));
          }
        }
        Src9 src;
        src.s[0] = site_of(j);
        const int m = (j - 1) & 3, c0 = j & 3, pp = (j + 1) & 3;
        auto rws = [&](int f) { return Rows3<R>{ring[f][m], ring[f][c0], ring[f][pp]}; };
        site_update<S, R, TH>(a, sd, src, in, JC, gC, poC, rws(0), rws(1), rws(2), rws(3), sc,
                              rws(G::NF - 1));
      }
      JC = JL;
#pragma unroll
      for (int i = 0; i < 5; ++i) gC[i] = gL[i];
      poC = poL;
      phC = phL;
      osC = osN;
      h0 = h1;
      sm = s0;
      em = next(em, G::NE);
      fu = next(fu, G::NFR);
    }
    __syncthreads();
  }
}

template <typename S, typename R>
int staged_halo_columns() {
  using G = Stage<S, R, false>;
  return G::HS > G::HR ? G::HS : G::HR;
}

template <typename S, typename R, bool TH>
static cudaError_t launch_staged_t(const StepArgs<S, R>& a, int grid, cudaStream_t st) {
  constexpr int smem = Stage<S, R, TH>::SMEM;
  static int configured[64] = {0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    e = cudaFuncSetAttribute(k_step_staged<S, R, TH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem);
    if (e != cudaSuccess) return e;
    configured[dev] = 1;
  }
  return launch_chained(k_step_staged<S, R, TH>, a, grid, smem, st);
}

template <typename S, typename R>
cudaError_t launch_step_staged(const StepArgs<S, R>& a, int grid, cudaStream_t st) {
  if constexpr (sizeof(S) == sizeof(R))
    if (a.thermal) return launch_staged_t<S, R, true>(a, grid, st);
  return launch_staged_t<S, R, false>(a, grid, st);
}

template <typename S, typename R, bool TH>
static int staged_blocks_t() {
  constexpr int smem = Stage<S, R, TH>::SMEM;
  int n = 0;
  cudaFuncSetAttribute(k_step_staged<S, R, TH>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step_staged<S, R, TH>, YM_THREADS, smem);
  return n > 0 ? n : 1;
}

template <typename S, typename R>
int staged_blocks_per_sm(bool thermal) {
  if constexpr (sizeof(S) == sizeof(R))
    if (thermal) return staged_blocks_t<S, R, true>();
  return staged_blocks_t<S, R, false>();
}

#define PF_STAGED_INST(S, R)                                                          \
  template cudaError_t launch_step_staged<S, R>(const StepArgs<S, R>&, int, cudaStream_t); \
  template int staged_halo_columns<S, R>();                                           \
  template int staged_blocks_per_sm<S, R>(bool);
PF_STAGED_INST(double, double)
PF_STAGED_INST(float, float)
PF_STAGED_INST(__half, float)
PF_STAGED_INST(__nv_bfloat16, float)

}  // namespace pf
