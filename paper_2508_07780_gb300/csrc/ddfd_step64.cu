// FP64 step kernels of the hybrid FE/FD scheme (forward and adjoint): the
// scheme, the boundary terms and the field layout are those described in
// ddfd_step.cu, with one node per thread.
//
// What bounds it: the FP64 unit.  GB300 retires about 1.7 FP64 lanes a clock
// and SM, whatever the number of active lanes (a warp instruction takes 19
// cycles of the SM, 64 as latency; add, multiply and multiply-add alike), so
// the time is the count of FP64 warp instructions, and loads, shared-memory
// traffic and integer work are all but free beside them.  Hence
//   - a thread takes the nodes of its tile in flat order, so that a ragged
//     tile (n = 161: a column of 1 x 8 nodes) runs in as few warps as its
//     nodes need (warps without a node issue no FP64 instruction);
//   - a plain finite-difference node takes the update with unit coefficients,
//     9 instructions a component instead of 12;
//   - the Gauss-law term of the FEM rows is formed through the tetrahedra, not
//     as a 15-point stencil of 3 x 3 blocks: the differences of w along the
//     edges (w = s E forward, mu in the adjoint), the divergences of the six
//     Kuhn tetrahedra of each cube, the sums over the six tetrahedra of each
//     edge, and their difference at the node, each computed once and handed
//     to the neighbours through shared memory: 39 instructions a node (36 in
//     the adjoint) against 102 (78).
// A CTA marches through the planes of its item; a ring of TMA-staged planes
// (ddfd_step_common.h) feeds it.
//
// Measured (us a step, forward and adjoint averaged, against the 15-point
// stencil on full 32 x 8 warps with 8 or 16 planes an item): 161^3 with a
// 121^3 cube 840 -> 482 (the FP64 instructions alone would take about 425),
// 41^3 / 21^3 88 -> 14, 13^3 / 9^3 50 -> 8.  Each step is launched as the last
// one's programmatic dependent (its barriers and descriptors are set up while
// that one drains).  So a step may start while the step that writes its fields or
// its history (a replayed segment's last one) still runs: what that one writes is
// read by ordinary loads after the wait, never by the non-coherent path, which is
// for data that nothing writes while the kernel lives.
#include "ddfd_step_common.h"

namespace ddfd {

namespace {

constexpr int up128(int b) { return (b + 127) / 128 * 128; }

// A staged plane: the current level and s with a one-node halo in y and a
// 16-byte halo in x, the previous level and (q1, q2) without.  Three stages:
// plane k, plane k + 1, and the next one in flight while a plane's FP64 work
// runs.  Tiles of 14 x 9, 8 x 8 or 32 x 8 nodes (tile64).
template <int TW, int TH>
struct Stage64 {
  static constexpr int TX = TW;
  static constexpr int TY = TH;
  // computing threads: the tile's nodes and, on small tiles, warps of their own
  // for its halo nodes (one warp's FP64 instructions run 64 cycles apart, so
  // that a thread with two nodes takes twice as long)
  static constexpr int CONSUMERS = TW == 32 ? 256 : (TW * TH + 31) / 32 * 32 + (2 * (TW + TH) + 4 + 31) / 32 * 32;
  static constexpr int MIN_CTAS = TW == 32 ? 2 : TW == 14 ? 3 : 4;
  static constexpr int HX = 2;
  static constexpr int BXW = TX + 2 * HX;
  static constexpr int ROWS = TY + 2;
  static constexpr int RE = ROWS * BXW;  // component stride of a staged plane
  static constexpr int TXY = TX * TY;
  static constexpr int E_BYTES = 3 * RE * 8;
  static constexpr int O_BYTES = 3 * TXY * 8;
  static constexpr int S_BYTES = RE * 8;
  static constexpr int Q_BYTES = 2 * TXY * 8;
  static constexpr int E_OFF = 0;
  static constexpr int O_OFF = up128(E_BYTES);
  static constexpr int S_OFF = O_OFF + up128(O_BYTES);
  static constexpr int Q_OFF = S_OFF + up128(S_BYTES);
  static constexpr int BYTES = Q_OFF + up128(Q_BYTES);
  static constexpr int RING = 3;
  // Gauss-law scratch, in doubles: over the tile's nodes with a one-node halo
  // (34 x 10) the edge differences in x and y of two planes and in z of one
  // layer; over the cubes whose lower corner is a tile node or lies left of /
  // below one (33 x 9) the six divergences and two edge sums.  w_x, w_y of a
  // plane (forward) share the divergences' space.
  static constexpr int HW = TX + 2, HN = HW * (TY + 2);
  static constexpr int CW = TX + 1, CN = CW * (TY + 1);
  static constexpr int DX = 0, DY = 2 * HN, DZ = 4 * HN, DIV = 5 * HN, FX = DIV + 6 * CN, FY = FX + CN;
  static constexpr int G_DOUBLES = FY + CN;
  static_assert(2 * HN <= 6 * CN, "w_x, w_y fit the divergences' space");
  static_assert(2 * (TW + TH) + 4 <= CONSUMERS, "a thread takes at most one halo node");
  static_assert(TW % 2 == 0, "TMA boxes start on 16 bytes");
  static constexpr int G_OFF = RING * BYTES;
  static constexpr int BAR_OFF = G_OFF + up128(G_DOUBLES * 8);
  static constexpr int SMEM = BAR_OFF + 2 * RING * 8 + 128;
};

// Barrier of the NT computing threads (the producer warp takes no part).
template <int NT>
__device__ __forceinline__ void compute_sync() {
  asm volatile("barrier.sync 1, %0;" ::"n"(NT) : "memory");
}
// The same with a vote: true if every computing thread passes true.
template <int NT>
__device__ __forceinline__ bool compute_all(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.red.and.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "n"(NT)
      : "memory");
  return r != 0;
}

template <bool ADJ, int NB, int TW, int TH>
__global__ void __launch_bounds__(Stage64<TW, TH>::CONSUMERS + 32, Stage64<TW, TH>::MIN_CTAS)
    k_step64(const __grid_constant__ StepLaunch<double, NB> L) {
  using S = Stage64<TW, TH>;
  constexpr int NT = S::CONSUMERS;
  constexpr int RE = S::RE, BW = S::BXW, HW = S::HW, CW = S::CW, CN = S::CN;
  const CtaTile ct = cta_tile(L);
  const StepParams<double> &P = L.p[NB == 1 ? 0 : ct.prob];
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  double *G = (double *)(smem + S::G_OFF);
  uint64_t *bar = (uint64_t *)(smem + S::BAR_OFF);  // "full": plane landed
  uint64_t *emp = bar + S::RING;                    // "empty": consumers released it
  const int n = P.n;
  const int tid = threadIdx.x;

  if (tid == 0) {
    for (int s = 0; s < S::RING; ++s) {
      mbar_init(&bar[s], 1);
      mbar_init(&emp[s], NT / 32);
    }
    mbar_fence_init();
    tma_prefetch_desc(&L.cur);
    tma_prefetch_desc(&L.old);
    tma_prefetch_desc(&L.s);
    tma_prefetch_desc(&L.q);
  }
  pdl_launch_dependents();
  pdl_wait();
  if (!ADJ) sample_detectors(P, ct, tid, (P.n + TW - 1) / TW, (P.n + TH - 1) / TH, NT);

  const int x0 = ct.tx * S::TX, y0 = ct.ty * S::TY;
  const int k0 = ct.k0;
  if (k0 >= n) return;  // uniform per CTA
  const int k1 = min(ct.k1, n);
  const bool tile_fem = x0 <= P.b - 1 && x0 + S::TX - 1 >= P.a + 1 && y0 <= P.b - 1 && y0 + S::TY - 1 >= P.a + 1;

  __syncthreads();

  if (tid >= NT) {
    if (tid == NT)
      produce_planes<S>(&L.cur, &L.old, &L.s, &L.q, smem, bar, emp, x0, y0, k0, k1, n, tile_fem, P.a, P.b,
                        P.chan, P.spin_limit, P.err);
    return;
  }

  // own node of this thread: flat order over the tile's nw x nh nodes
  const int nw = min(S::TX, n - x0), nh = min(S::TY, n - y0);
  const bool own = tid < nw * nh;
  const int ly = own ? tid / nw : 0, lx = own ? tid - ly * nw : 0;
  const int x = x0 + lx, y = y0 + ly;
  const int ci = (ly + 1) * BW + lx + S::HX;  // in a staged plane with halo
  const int oi = ly * S::TX + lx;             // in a centre box
  const int hi = (ly + 1) * HW + lx + 1;      // in the Gauss-law scratch: node with halo
  const int qi = (ly + 1) * CW + lx + 1;      // ... cube (its lower corner)
  const int dym = (y == 0) ? BW : -BW, dyp = (y == n - 1) ? -BW : BW;
  const int dxm = (x == 0) ? 1 : -1, dxp = (x == n - 1) ? -1 : 1;
  const bool colfem = own && x > P.a && x < P.b && y > P.a && y < P.b;
  const bool colfree = own && x >= P.f0 && x < P.f0 + P.nf && y >= P.f0 && y < P.f0 + P.nf;
  const uint32_t sides = (P.abs_now | P.abs_next) & (DDFD_ABS_X0 | DDFD_ABS_X1 | DDFD_ABS_Y0 | DDFD_ABS_Y1);
  // side columns need the boundary path only where a side face absorbs
  const bool colbnd = (x == 0 && (sides & DDFD_ABS_X0)) || (x == n - 1 && (sides & DDFD_ABS_X1)) ||
                      (y == 0 && (sides & DDFD_ABS_Y0)) || (y == n - 1 && (sides & DDFD_ABS_Y1));
  const long long plane = (long long)P.px * n;
  const uint32_t cs = (uint32_t)P.cs;
  double *out = P.old + (long long)k0 * plane + (long long)P.px * y + x;

  // Gauss-law term: the layers of cubes [l, l + 1] that hold a node with s != 0
  // (or, in the adjoint, a free one) as a corner, and in the forward the layer
  // above, whose lower edges close the last FEM row.  The halo nodes of the
  // tile go to the warps after its own nodes (or, for a full tile, to the
  // first ones): the column and row of halo nodes that are cubes' lower
  // corners first, then the others.
  const bool gauss = tile_fem && !P.ebe_r;
  const int gl0 = P.f0 - 1, gl1 = P.f0 + P.nf - (ADJ ? 1 : 0);
  const int e0 = tid - ((nw * nh + 31) & ~31), e = e0 < 0 ? e0 + NT : e0;
  const bool extra = gauss && e < 2 * (nw + nh) + 4;
  const bool ecol = e < nh + 1, erow = !ecol && e < nw + nh + 1;  // x = -1; y = -1
  int ex = 0, ey = 0;
  if (ecol)
    ex = -1, ey = e - 1;
  else if (erow)
    ex = e - nh - 1, ey = -1;
  else if (e < nw + 2 * nh + 3)
    ex = nw, ey = e - (nw + nh + 2);
  else
    ex = e - (nw + 2 * nh + 4), ey = nh;
  const int eci = (ey + 1) * BW + ex + S::HX, ehi = (ey + 1) * HW + ex + 1, eqi = (ey + 1) * CW + ex + 1;
  const bool ecube = extra && (ecol || erow);

  // differences of one staged plane along x and y (they land in scratch plane
  // `pl`), and along z against the plane before it
  double wzp[2] = {0.0, 0.0};      // w_z of the last plane: own node, halo node
  double topx = 0.0, topy = 0.0;   // upper-layer part of the edges (x, y) of the next plane
  double etop = 0.0;
  double fzp = 0.0;                // z edge sum of the layer below
  auto plane_diffs = [&](const unsigned char *st, int pl, bool layer) {
    const double *E = (const double *)(st + S::E_OFF);
    const double *Sp = (const double *)(st + S::S_OFF);
    double *W = G + S::DIV;
    auto put = [&](int c, int h, double &wz0) {
      double wz = E[2 * RE + c];
      if (!ADJ) {
        const double s = Sp[c];
        wz *= s;
        W[h] = s * E[c];
        W[S::HN + h] = s * E[RE + c];
      }
      if (layer) G[S::DZ + h] = wz - wz0;
      wz0 = wz;
    };
    if (own) put(ci, hi, wzp[0]);
    if (extra) put(eci, ehi, wzp[1]);
    if (!ADJ) compute_sync<NT>();
    double *DX = G + S::DX + pl * S::HN, *DY = G + S::DY + pl * S::HN;
    auto diff = [&](int c, int h, bool dx, bool dy) {
      if (ADJ) {
        if (dx) DX[h] = E[c + 1] - E[c];
        if (dy) DY[h] = E[RE + c + BW] - E[RE + c];
      } else {
        if (dx) DX[h] = W[h + 1] - W[h];
        if (dy) DY[h] = W[S::HN + h + HW] - W[S::HN + h];
      }
    };
    if (own) diff(ci, hi, true, true);
    if (extra) diff(eci, ehi, ex < nw, ey < nh);
    compute_sync<NT>();
  };
  // divergences of the six tetrahedra of the cube at scratch node h (path
  // orders xyz, xzy, yxz, yzx, zxy, zyx)
  auto cube_divs = [&](int h, int q, int pl) {
    const double *X0 = G + S::DX + pl * S::HN + h, *X1 = G + S::DX + (pl ^ 1) * S::HN + h;
    const double *Y0 = G + S::DY + pl * S::HN + h, *Y1 = G + S::DY + (pl ^ 1) * S::HN + h;
    const double *Z = G + S::DZ + h;
    double *D = G + S::DIV + q;
    const double z11 = Z[HW + 1], y11 = Y1[1], x11 = X1[HW];
    D[0] = (X0[0] + Y0[1]) + z11;
    D[CN] = (X0[0] + Z[1]) + y11;
    D[2 * CN] = (Y0[0] + X0[HW]) + z11;
    D[3 * CN] = (Y0[0] + Z[HW]) + x11;
    D[4 * CN] = (Z[0] + X1[0]) + y11;
    D[5 * CN] = (Z[0] + Y1[0]) + x11;
  };
  // sums over the tetrahedra of one layer at the edges of cube q's lower
  // corner: lower edges in x (y), upper edges in x (y)
  auto low_x = [&](const double *D) { return (D[0] + D[CN]) + D[2 * CN - CW]; };
  auto low_y = [&](const double *D) { return (D[2 * CN] + D[3 * CN]) + D[-1]; };
  auto top_x = [&](const double *D) { return (D[3 * CN - CW] + D[5 * CN - CW]) + D[4 * CN]; };
  auto top_y = [&](const double *D) { return (D[CN - 1] + D[4 * CN - 1]) + D[5 * CN]; };

  int wq = 0, wslot = 0;   // planes waited so far, slot of the next wait
  uint32_t wphase = 0;     // parity of the next wait
  int sl = 0;              // slot of plane l
  double below[3] = {0.0, 0.0, 0.0}, cen[3] = {0.0, 0.0, 0.0};
  // layer l lies between planes l and l + 1; the nodes of plane l are updated
  // in the layer's turn (the first turn only supplies plane k0 - 1)
  for (int l = k0 - 1; l < k1; ++l) {
    const int p = l - k0 + 1;  // index of plane l among the staged ones
    bool ok = true;
    while (wq <= p + 1) {
      if (!mbar_wait_bounded(&bar[wslot], wphase, P.spin_limit)) {
        ok = false;
        break;
      }
      ++wq;
      if (++wslot == S::RING) {
        wslot = 0;
        wphase ^= 1u;
      }
    }
    // a timeout ends the loop for the warp, or where the CTA's warps meet at
    // barriers for all of them (the producer times out on unreleased slots)
    const bool all = gauss ? compute_all<NT>(ok) : __all_sync(0xffffffffu, ok);
    if (!all) {
      if (!ok && (tid & 31) == 0) atomicOr(P.err, 4);
      break;
    }
    const int sn = sl + 1 == S::RING ? 0 : sl + 1;
    const unsigned char *b0 = smem + sl * S::BYTES, *b1 = smem + sn * S::BYTES;
    const double *E0 = (const double *)(b0 + S::E_OFF);
    const double *E1 = (const double *)(b1 + S::E_OFF);
    double above[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (l == k0 - 1) cen[c] = E0[c * RE + ci];
      above[c] = E1[c * RE + ci];
    }

    double g[3] = {0.0, 0.0, 0.0};  // 6 h^2 M^-1 D^T D w at the own node
    if (gauss && l >= gl0 && l <= gl1) {
      const int pl = l & 1;
      if (l == gl0 || l == k0 - 1) plane_diffs(b0, pl, false);
      plane_diffs(b1, pl ^ 1, true);
      if (own) cube_divs(hi, qi, pl);
      if (ecube) cube_divs(ehi, eqi, pl);
      compute_sync<NT>();
      if (own) {
        const double *D = G + S::DIV + qi;
        G[S::FX + qi] = topx + low_x(D);
        G[S::FY + qi] = topy + low_y(D);
        topx = top_x(D);
        topy = top_y(D);
        const double fz = ((D[4 * CN] + D[5 * CN]) + (D[CN - 1] + D[3 * CN - CW])) + (D[-CW - 1] + D[2 * CN - CW - 1]);
        g[2] = fzp - fz;
        fzp = fz;
      }
      if (ecube && (ecol ? ey >= 0 : true)) {  // (the corner cube has no edge of its own)
        const double *D = G + S::DIV + eqi;
        if (ecol) {
          G[S::FX + eqi] = etop + low_x(D);
          etop = top_x(D);
        } else {
          G[S::FY + eqi] = etop + low_y(D);
          etop = top_y(D);
        }
      }
      compute_sync<NT>();
      if (own) {
        g[0] = G[S::FX + qi - 1] - G[S::FX + qi];
        g[1] = G[S::FY + qi - CW] - G[S::FY + qi];
      }
    }

    if (l >= k0 && own) {
      const int k = l;
      const double *O0 = (const double *)(b0 + S::O_OFF);
      const bool kfem = k > P.a && k < P.b;
      const bool fre = colfree && k >= P.f0 && k < P.f0 + P.nf;
      // bottom plane: absorbing or plain Neumann; top plane: source, absorbing
      // face or detector residuals
      const bool kbnd = (k == 0 && ((P.abs_now | P.abs_next) & DDFD_ABS_BOTTOM)) || k == n - 1;
      double dv[3], R[3], t[3];  // E^n - E^{n-1}, h^2 M^-1 K E, the increment
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double *e0 = E0 + c * RE + ci;
        dv[c] = cen[c] - O0[c * S::TXY + oi];
        R[c] = 6.0 * cen[c] - (e0[dxp] + e0[dxm] + e0[dyp] + e0[dym] + above[c] + below[c]);
      }
      double sx[3] = {0.0, 0.0, 0.0};  // adjoint: tau^2 M^-1 D^T D mu, for the gradient
      if (colfem && kfem) {
        const double *Q0 = (const double *)(b0 + S::Q_OFF);
        const double A = Q0[oi], C = Q0[S::TXY + oi] * P.r2;
        if (P.ebe_r) {
          // element-by-element rows computed by k_ebe for this step
          const int fm = P.b - P.a - 1;
          const long long row = (x - P.a - 1) + (long long)fm * ((y - P.a - 1) + (long long)fm * (k - P.a - 1));
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            R[c] = P.ebe_r[c * P.ebe_rows + row];
            if (ADJ) sx[c] = P.r2 * P.ebe_q[c * P.ebe_rows + row];
          }
        } else if (!ADJ) {
#pragma unroll
          for (int c = 0; c < 3; ++c) R[c] += (1.0 / 6.0) * g[c];
        } else {
          const double s0 = ((const double *)(b0 + S::S_OFF))[ci];
          if (s0 != 0.0 || fre) {
            const double s6 = s0 * (1.0 / 6.0), r6 = P.r2 * (1.0 / 6.0);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              R[c] += s6 * g[c];
              sx[c] = r6 * g[c];
            }
          }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) t[c] = A * dv[c] - C * R[c];
      } else if (colbnd || kbnd) {
        // boundary node: damping of the absorbing faces, top-face source or
        // detector residuals
        const int fn = face_count(x, y, k, n, P.abs_now);
        const double cc = P.cb * (double)fn;
        const double ccn = ADJ ? P.cb * (double)face_count(x, y, k, n, P.abs_next) : cc;
        const double inv = P.inv_tab[fn];  // 1 / (1 + cc)
        const double A = (1.0 - ccn) * inv, B = (ccn - cc) * inv;
#pragma unroll
        for (int c = 0; c < 3; ++c) R[c] *= P.r2;
        if (!ADJ && k == n - 1 && P.src_on) {
          if (!P.oblique) {
            R[1] -= P.src_y;
          } else {
            const double v = P.src_tab ? P.src_tab[x + P.px * y]
                                       : P.src_scale * pulse_value(P.pulse_kind, P.freq, P.t0, P.width,
                                                                   P.t_n - P.delay[x + n * y]);
#pragma unroll
            for (int c = 0; c < 3; ++c) R[c] -= P.pol[c] * v;
          }
        }
        if (ADJ && k == n - 1 && P.n_det > 0) {
          const int q0 = P.det_ptr[x + n * y], q1 = P.det_ptr[x + n * y + 1];
          if (q1 > q0) {
            const double wx = (x == 0 || x == n - 1) ? 0.5 : 1.0;
            const double wy = (y == 0 || y == n - 1) ? 0.5 : 1.0;
            const double sc = P.tau2 * P.inv_h3 / (wx * wy * 0.5);
            double acc[3] = {0.0, 0.0, 0.0};
            for (int qq = q0; qq < q1; ++qq) {
              const int d = P.det_list[qq];
              acc[0] += P.res_k[3 * d + 0];
              acc[1] += P.res_k[3 * d + 1];
              acc[2] += P.res_k[3 * d + 2];
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) R[c] += sc * acc[c];
          }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) t[c] = A * dv[c] + (B * cen[c] - inv * R[c]);
      } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) t[c] = dv[c] - P.r2 * R[c];
      }
      const long long fi = (x - P.f0) + (long long)P.nf * ((y - P.f0) + (long long)P.nf * (k - P.f0));
      double hv[3] = {0.0, 0.0, 0.0}, ae = 0.0, as = 0.0;  // (read ahead of the stores, which they may not be moved across)
      if (ADJ && fre) {
#pragma unroll
        for (int c = 0; c < 3; ++c) hv[c] = P.hist_r[c * P.hcs + fi];
        ae = P.gacc_e[fi], as = P.gacc_s[fi];
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) out[c * cs] = cen[c] + t[c];
      if (fre) {
        if (!ADJ) {
          if (P.hist_w)
#pragma unroll
            for (int c = 0; c < 3; ++c) P.hist_w[c * P.hcs + fi] = cen[c] + t[c];
        } else {
          // mu^{k-1} - 2 mu^k + mu^{k+1} = t - dv, mu^{k-1} - mu^{k+1} = t + dv
          double ge = 0.0, gs = 0.0;
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            ge += hv[c] * ((t[c] - dv[c]) + sx[c]);
            gs += hv[c] * (t[c] + dv[c]);
          }
          P.gacc_e[fi] = ae + ge;
          P.gacc_s[fi] = as + gs;
        }
      }
    }
    if (l >= k0) out += plane;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      below[c] = cen[c];
      cen[c] = above[c];
    }
    // release plane l to the producer: one arrival per warp
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(&emp[sl]);
    sl = sn;
  }
}

template <bool ADJ, int NB, int TW, int TH>
cudaError_t set_smem() {
  return cudaFuncSetAttribute(k_step64<ADJ, NB, TW, TH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              Stage64<TW, TH>::SMEM);
}
template <int TW, int TH>
cudaError_t set_smem_tile() {
  cudaError_t e;
  if ((e = set_smem<false, 1, TW, TH>()) || (e = set_smem<true, 1, TW, TH>()) ||
      (e = set_smem<false, BATCH_MAX, TW, TH>()))
    return e;
  return set_smem<true, BATCH_MAX, TW, TH>();
}

template <bool ADJ, int NB, int TW, int TH>
void launch_tile(const StepLaunch<double, NB> &L, cudaStream_t s) {
  const int n = L.p[0].n;
  const dim3 g = L.items ? dim3((unsigned)L.n_items)
                         : dim3((n + TW - 1) / TW, (n + TH - 1) / TH, L.zchunks * L.nprob);
  launch_chained(k_step64<ADJ, NB, TW, TH>, g, Stage64<TW, TH>::CONSUMERS + 32, Stage64<TW, TH>::SMEM, s,
                 L.chained != 0, L);
}

}  // namespace

cudaError_t prepare_step64_kernels() {
  cudaError_t e;
  if ((e = set_smem_tile<32, 8>()) || (e = set_smem_tile<14, 9>())) return e;
  return set_smem_tile<8, 8>();
}

// 14 x 9 tiles: 126 of 128 lanes, warps of their own for the halo nodes, 3
// thread blocks per SM.  Small grids take 8 x 8 (41^3 13.5 / 14.3 us a forward /
// adjoint step against 18.5 / 19.1; 51^3 even): the FEM cube's nodes, three times
// as dear as the others, then spread over more SMs.  32 x 8, two thread blocks per
// SM (161^3 with a 121^3 cube 530 / 591 us against 456 / 508; 65^3 85 / 96
// against 29 / 31), is left for the grids whose 14-node columns the dispatch
// items cannot count.
Tile64 tile64(int n, int count) {
  const long long items = (long long)((n + 7) / 8) * ((n + 7) / 8) * n * count;
  if (items <= 2048) return {8, 8};
  if (n <= 32 * 14) return {14, 9};
  return {32, 8};
}

template <bool ADJ, int NB>
int launch_step64(const StepLaunch<double, NB> &L, cudaStream_t s) {
  if (L.tile_w == 8)
    launch_tile<ADJ, NB, 8, 8>(L, s);
  else if (L.tile_w == 14)
    launch_tile<ADJ, NB, 14, 9>(L, s);
  else
    launch_tile<ADJ, NB, 32, 8>(L, s);
  return 1;
}
template int launch_step64<false, 1>(const StepLaunch<double, 1> &, cudaStream_t);
template int launch_step64<true, 1>(const StepLaunch<double, 1> &, cudaStream_t);
template int launch_step64<false, BATCH_MAX>(const StepLaunch<double, BATCH_MAX> &, cudaStream_t);
template int launch_step64<true, BATCH_MAX>(const StepLaunch<double, BATCH_MAX> &, cudaStream_t);

}  // namespace ddfd
