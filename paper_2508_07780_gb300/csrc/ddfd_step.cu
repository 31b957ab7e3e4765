// Explicit step kernels of the hybrid FE/FD scheme (forward and adjoint).
//
// Work decomposition: one CTA owns an (x, y) tile and a range of consecutive
// z planes (a dispatch item, or a z chunk of the 3-D grid), which it marches
// through plane by plane.
//   - FP32 (k_step_quad): 32 x 16 tiles, 4 compute warps and a producer warp;
//     each thread owns four x-adjacent nodes, whose arithmetic runs in packed
//     FP32 (one instruction for two nodes) on rows read as float4; on a grid of
//     n = 32 m + 1 nodes the last tile also updates the column x = n - 1.  An
//     item without FEM-cube or free nodes takes a loop of its own, without the
//     block stencil, the gradient or the coefficients.
//   - FP64: ddfd_step64.cu, one node a thread, tiles by grid size, every item alike.
// The planes of the current field (with a one-node halo in y and a
// 16-byte-aligned halo in x), the centre tile of the previous level, and (on
// items that touch the FEM cube) the coefficient planes are staged into
// shared memory by TMA tile loads through rings of slots guarded by
// mbarriers, so that several planes are in flight per CTA while the previous
// ones are computed.  A launch may carry a dispatch order (StepLaunch::items),
// and starts as the programmatic dependent of the step before it.
//
// What bounds the FP32 step: DRAM on large grids (301^3 without a cube 152 us,
// 0.96 of the copy bandwidth on its algorithmic bytes), latency elsewhere -- the
// first planes of an item and the last items of a step -- and the instructions of
// the FEM rows.  us a step, forward / adjoint, against two launches side by side
// (two nodes a thread, a kernel for the FEM items and one for the others):
// 201^3 / 101^3 66 / 71 -> 58 / 64, 301^3 / 151^3 190 / 197 -> 181 / 192,
// 16 x 161^3 (oblique) 597 / 650 -> 527 / 568, 100^3 / 63^3 18 / 19 -> 13.0 / 13.0,
// 41^3 / 21^3 10.5 / 11.5 -> 5.0 / 4.7.  Tried and dropped: the last warp to
// release a slot staging the next plane instead of a producer warp (301^3
// without a cube 156 -> 180), two nodes a thread (173), carrying the stencil's
// lower plane in registers (no gain), s = eps - 1 held for all three components
// (spills), full and lean items mixed by problem and z (batch 583 -> 642: the two
// loops share the instruction cache badly).
//
// Per node and step:
//   FD part (every node): 7-point Laplacian with ghost-node (mirror) Neumann
//     closure, i.e. h^2 M^-1 L of the hexahedral FD scheme;
//   FEM part (nodes strictly inside the FEM cube): the P1 Gauss-law term of
//     eq. forward_prob / eq. model1 on the Kuhn mesh as a 15-point block
//     stencil: forward h^2 M^-1 (D^T D S E)_i = sum_o B_o (s E)_{i+o},
//     adjoint h^2 M^-1 (S D^T D mu)_i = s_i sum_o B_o mu_{i+o};
//   boundary: damping tau/h per absorbing face (first-order absorbing
//     condition of eq. model1 with lumped surface mass), Neumann flux on the
//     top face during the source phase;
//   update in the divided, difference form (V = E^n - E^{n-1}, c = tau C/(2M)):
//     E^{n+1} = E^n + ((eps - c) V - tau^2 (M^-1 K E^n - f^n)) / (eps + c),
//   algebraically the central scheme M E'' + C E' + K E = F, written so that
//   FP32 storage does not cancel 2 E^n - E^{n-1};
//   adjoint: the transposed recursion of the same scheme with the damping of
//     steps k-1 and k+1, detector residuals j^k / m as sources, and the
//     gradient time sums (eq. gradeps, summation-by-parts form) accumulated in
//     FP64 at the free nodes.
//
// Field layout: component-major, x pitch px (a multiple of 8 elements, so
// TMA row strides are 16-byte multiples), offset i + px (j + n k).
#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>

#include "ddfd_step_common.h"

namespace ddfd {

// The Kuhn P1 div-div blocks of an interior node in integer form: (D^T D)_{i,i+o}
// = (h/6) kb(o, .), B_{-o} = B_o = B_o^T, offsets 0, (1,0,0), (0,1,0), (0,0,1),
// (1,1,0), (1,0,1), (0,1,1), (1,1,1).  Compiled in so that zero and unit
// weights cost nothing; ddfd_create checks them against the blocks it
// assembles from the 24 Kuhn tetrahedra (csrc/ddfd_kuhn.cpp) and refuses to
// run if they differ.
__host__ __device__ constexpr int kb(int o, int e) {
  constexpr int t[8][9] = {
      {12, -4, -4, -4, 12, -4, -4, -4, 12},  // 0
      {-6, 2, 2, 2, 0, -1, 2, -1, 0},        // (1,0,0)
      {0, 2, -1, 2, -6, 2, -1, 2, 0},        // (0,1,0)
      {0, -1, 2, -1, 0, 2, 2, 2, -6},        // (0,0,1)
      {0, -2, 1, -2, 0, 1, 1, 1, 0},         // (1,1,0)
      {0, 1, -2, 1, 0, 1, -2, 1, 0},         // (1,0,1)
      {0, 1, 1, 1, 0, -2, 1, -2, 0},         // (0,1,1)
      {0, -1, -1, -1, 0, -1, -1, -1, 0}};    // (1,1,1)
  return t[o][e];
}

static int kb_int(int o, int e) { return kb(o, e); }

cudaError_t check_kuhn_blocks(const KuhnBlocks &kb, cudaStream_t) {
  for (int o = 0; o < 8; ++o)
    for (int e = 0; e < 9; ++e)
      if (std::fabs(kb.B[o][e] * 6.0 - kb_int(o, e)) > 1e-12)
        return cudaErrorInvalidValue;
  return cudaSuccess;
}

// sum_o B_o v_{i+o} for one node (B = kb / 6), with B_{-o} = B_o; v given as
// the centre value and the 7 (+o, -o) neighbour pairs already summed.
template <typename T>
__device__ __forceinline__ void block_apply(const T v0[3], const T vp[7][3], T out[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    T acc = T(kb(0, c * 3 + 0)) * v0[0] + T(kb(0, c * 3 + 1)) * v0[1] + T(kb(0, c * 3 + 2)) * v0[2];
#pragma unroll
    for (int p = 0; p < 7; ++p) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int w = kb(p + 1, c * 3 + d);
        if (w == 1)
          acc += vp[p][d];
        else if (w == -1)
          acc -= vp[p][d];
        else if (w != 0)
          acc += T(w) * vp[p][d];
      }
    }
    out[c] = acc * T(1.0 / 6.0);
  }
}

// FP32 staging: 32 x 16 tile, each of the 128 computing threads owns four
// x-adjacent nodes (so every staged row is read as float4).  Two rings of
// slots: "halo" slots (the current level with its halo and, on full items --
// those with FEM-cube or free nodes -- s), and "centre" slots (the previous
// level and, on full items, (q1, q2)).  The Laplacian and the Gauss-law term
// of plane k hold the halo planes k - 1, k and k + 1, but only the centre plane
// k, so that the rings' sizes differ: 6 and 4 slots (full), 8 and 6 (lean),
// 111 KB a CTA, 2 CTAs per SM, three to six planes in flight.
constexpr int round128(int b) { return (b + 127) / 128 * 128; }
struct QuadStage {
  static constexpr int TX = STEP_TX;
  static constexpr int TY = STEP_TY;
  static constexpr int HX = 4;                     // x halo: one 16-byte unit
  static constexpr int BXW = TX + 2 * HX;          // staged row length (40)
  static constexpr int ROWS = TY + 2;
  static constexpr int RE = ROWS * BXW;            // component stride of a staged plane
  static constexpr int TXY = TX * TY;
  static constexpr int E_BYTES = 3 * RE * 4;
  static constexpr int O_BYTES = 3 * TXY * 4;
  static constexpr int S_BYTES = RE * 4;
  static constexpr int Q_BYTES = 2 * TXY * 4;
  static constexpr int S_OFF = round128(E_BYTES);  // in a halo slot
  static constexpr int Q_OFF = round128(O_BYTES);  // in a centre slot
  static constexpr int FULL_E = S_OFF + round128(S_BYTES), FULL_O = Q_OFF + round128(Q_BYTES);
  static constexpr int LEAN_E = S_OFF, LEAN_O = Q_OFF;
  static constexpr int FULL_NE = 6, FULL_NO = 4, LEAN_NE = 8, LEAN_NO = 6;
  static constexpr int NB = 8;  // barriers of each kind
  static constexpr int BAR_OFF = FULL_NE * FULL_E + FULL_NO * FULL_O;
  static_assert(LEAN_NE * LEAN_E + LEAN_NO * LEAN_O <= BAR_OFF, "the lean slots fit the full ones' space");
  static_assert(NB >= LEAN_NE && NB >= FULL_NE, "a barrier per plane in flight");
  static constexpr int SMEM = BAR_OFF + 2 * NB * 8 + 128;
};
// Warp roles: warps 0..3 compute, warp 4 stages planes (it measured 156
// against 180 us a step on 301^3 without a cube when the last warp to release a
// slot staged the next plane instead).
constexpr int QUAD_CONSUMERS = 128;
constexpr int QUAD_THREADS = QUAD_CONSUMERS + 32;

// ---------------------------------------------------------------------------
// FP32 step kernel, four x-adjacent nodes per thread
// ---------------------------------------------------------------------------

// Moves the line holding p into L2 (no register result, no wait).
__device__ __forceinline__ void prefetch_l2(const void *p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(__cvta_generic_to_global(p)));
}

// Packed FP32 (sm_100+): one instruction for two nodes.  These round exactly
// like the scalar operations; a - b is written fma(b, -1, a), which is exact
// in its negation.
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// The four nodes of a thread: l holds nodes 0 and 1, h nodes 2 and 3.
struct Quad {
  float2 l, h;
};
__device__ __forceinline__ Quad ld4(const float *p) {
  const float4 v = *reinterpret_cast<const float4 *>(p);
  return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ void st4(float *p, const Quad &q) {
  *reinterpret_cast<float4 *>(p) = make_float4(q.l.x, q.l.y, q.h.x, q.h.y);
}
__device__ __forceinline__ Quad add4(const Quad &a, const Quad &b) { return {add2(a.l, b.l), add2(a.h, b.h)}; }
__device__ __forceinline__ Quad mul4(const Quad &a, const Quad &b) { return {mul2(a.l, b.l), mul2(a.h, b.h)}; }
__device__ __forceinline__ Quad mul4(const Quad &a, float2 b) { return {mul2(a.l, b), mul2(a.h, b)}; }
__device__ __forceinline__ Quad fma4(const Quad &a, const Quad &b, const Quad &c) {
  return {fma2(a.l, b.l, c.l), fma2(a.h, b.h, c.h)};
}
__device__ __forceinline__ Quad fma4(const Quad &a, float2 b, const Quad &c) {
  return {fma2(a.l, b, c.l), fma2(a.h, b, c.h)};
}
__device__ __forceinline__ float get(const Quad &q, int j) { return j == 0 ? q.l.x : j == 1 ? q.l.y : j == 2 ? q.h.x : q.h.y; }
__device__ __forceinline__ void set(Quad &q, int j, float v) {
  (j == 0 ? q.l.x : j == 1 ? q.l.y : j == 2 ? q.h.x : q.h.y) = v;
}

// acc + w v for a compile-time weight (0 and +-1 cost no multiply).
__device__ __forceinline__ float2 wacc2(float2 acc, int w, float2 v) {
  if (w == 0) return acc;
  if (w == 1) return add2(acc, v);
  if (w == -1) return fma2(v, f2(-1.f), acc);
  return fma2(f2((float)w), v, acc);
}

// Input component d of a pair's two 15-point block stencils (a at x, b at
// x+1): the centre values and the 7 (+o, -o) pair sums, added as
// out_c += B_o[c][d] * (...), B = kb / 6 applied by the caller; both nodes
// share the weights.
__device__ __forceinline__ void block_acc2(int d, float2 v0, const float2 ps[7], float2 out[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float2 u = wacc2(out[c], kb(0, c * 3 + d), v0);
#pragma unroll
    for (int p = 0; p < 7; ++p) u = wacc2(u, kb(p + 1, c * 3 + d), ps[p]);
    out[c] = u;
  }
}

// The 36 values that the 15-point stencils of a thread's four nodes touch, of
// one component (or of s): plane k (row y: x-1..x+4; row y+1: x..x+4; row
// y-1: x-1..x+3), plane k+1 (rows y, y+1: x..x+4), plane k-1 (rows y, y-1:
// x-1..x+3).
struct Hood {
  Quad c, yp, ym, pc, py, mc, my;
  float cm, cp, ypp, ymm, pcp, pyp, mcm, mym;  // the values at x-1 (m) and x+4 (p)
};

// Adds the block stencils of input component d for both pairs: pair sums of
// the offsets (1,0,0) (0,1,0) (0,0,1) (1,1,0) (1,0,1) (0,1,1) (1,1,1).
__device__ __forceinline__ void hood_acc(int d, const Hood &v, Quad out[3]) {
  float2 ps[7], o[3];
  ps[0] = add2(make_float2(v.c.l.y, v.c.h.x), make_float2(v.cm, v.c.l.x));
  ps[1] = add2(v.yp.l, v.ym.l);
  ps[2] = add2(v.pc.l, v.mc.l);
  ps[3] = add2(make_float2(v.yp.l.y, v.yp.h.x), make_float2(v.ymm, v.ym.l.x));
  ps[4] = add2(make_float2(v.pc.l.y, v.pc.h.x), make_float2(v.mcm, v.mc.l.x));
  ps[5] = add2(v.py.l, v.my.l);
  ps[6] = add2(make_float2(v.py.l.y, v.py.h.x), make_float2(v.mym, v.my.l.x));
#pragma unroll
  for (int c = 0; c < 3; ++c) o[c] = out[c].l;
  block_acc2(d, v.c.l, ps, o);
#pragma unroll
  for (int c = 0; c < 3; ++c) out[c].l = o[c], o[c] = out[c].h;
  ps[0] = add2(make_float2(v.c.h.y, v.cp), make_float2(v.c.l.y, v.c.h.x));
  ps[1] = add2(v.yp.h, v.ym.h);
  ps[2] = add2(v.pc.h, v.mc.h);
  ps[3] = add2(make_float2(v.yp.h.y, v.ypp), make_float2(v.ym.l.y, v.ym.h.x));
  ps[4] = add2(make_float2(v.pc.h.y, v.pcp), make_float2(v.mc.l.y, v.mc.h.x));
  ps[5] = add2(v.py.h, v.my.h);
  ps[6] = add2(make_float2(v.py.h.y, v.pyp), make_float2(v.my.l.y, v.my.h.x));
  block_acc2(d, v.c.h, ps, o);
#pragma unroll
  for (int c = 0; c < 3; ++c) out[c].h = o[c];
}

// The rings of an item, and the staging of its planes (one thread, the producer
// warp).  Plane p = kk - (k0 - 1), p = 0 .. nplanes - 1: its halo box (mirrored
// ghost planes at kk = -1 and kk = n) goes to halo slot p % ne, its centre box
// (computed planes, 1 .. nplanes - 2) to centre slot p % no; coefficients on
// full items, planes a..b.  Turn j (plane j is updated) needs halo plane j + 1
// and centre plane j on top of the turns before it: these two complete barrier
// j % NB (two arrivals; barrier 0: halo planes 0 and 1).  The end of turn j
// (emp, j >= 1, in barrier (j - 1) % NB) frees halo plane j - 1 and centre plane j.  Every wait is bounded; on
// give-up error bit 4 is set and the issued copies are still waited for
// (bounded).
struct QuadRing {
  int ne, no, ebytes, obytes;
};
template <class S, class LT>
__device__ __forceinline__ void produce_quads(const LT &L, const QuadRing R, unsigned char *smem, uint64_t *bar,
                                              uint64_t *emp, int x0, int y0, int k0, int k1, int n, bool full, int a,
                                              int b, int ch, uint32_t spin, int *err) {
  const int nplanes = k1 - k0 + 2;
  int es = 0, os = 1 % R.no;  // next slots
  auto halo = [&](int p) {
    const int kk = k0 - 1 + p;
    const int ksrc = kk < 0 ? 1 : (kk >= n ? n - 2 : kk);  // mirror ghost planes
    const bool coef = full && kk >= a && kk <= b;
    unsigned char *st = smem + es * R.ebytes;
    uint64_t *bb = &bar[(p == 0 ? 0 : p - 1) % S::NB];
    mbar_expect_tx(bb, S::E_BYTES + (coef ? S::S_BYTES : 0));
    tma_load_4d(st, &L.cur, x0 - S::HX, y0 - 1, ksrc, ch, bb);
    if (coef) tma_load_4d(st + S::S_OFF, &L.s, x0 - S::HX, y0 - 1, kk, ch, bb);
    if (++es == R.ne) es = 0;
  };
  auto centre = [&](int p) {
    const int kk = k0 - 1 + p;
    const bool coef = full && kk >= a && kk <= b;
    unsigned char *st = smem + R.ne * R.ebytes + os * R.obytes;
    uint64_t *bb = &bar[p % S::NB];
    mbar_expect_tx(bb, S::O_BYTES + (coef ? S::Q_BYTES : 0));
    tma_load_4d(st, &L.old, x0, y0, kk, ch, bb);
    if (coef) tma_load_4d(st + S::Q_OFF, &L.q, x0, y0, kk, ch + 1, bb);
    if (++os == R.no) os = 0;
  };
  int pe = 0, po = 1;  // next planes
  halo(pe++);
  halo(pe++);
  while (pe < R.ne || po <= R.no) {
    if (pe < R.ne && pe < nplanes) halo(pe);
    if (po <= R.no && po <= nplanes - 2) centre(po);
    ++pe, ++po;
  }
  pe = R.ne, po = R.no + 1;
  bool ok = true;
  for (int j = 1; pe < nplanes || po <= nplanes - 2; ++j, ++pe, ++po) {
    if (!mbar_wait_bounded(&emp[(j - 1) % S::NB], (uint32_t)(((j - 1) / S::NB) & 1), spin)) {
      ok = false;
      break;
    }
    if (pe < nplanes) halo(pe);
    if (po <= nplanes - 2) centre(po);
  }
  if (!ok) atomicOr(err, 4);
  // every issued plane must land before the CTA can retire (bounded)
  for (int q = nplanes > S::NB + 1 ? nplanes - 1 - S::NB : 0; q < nplanes - 1; ++q)
    if (!mbar_wait_bounded(&bar[q % S::NB], (uint32_t)((q / S::NB) & 1), spin)) break;
}

// Oblique flux of one node where no table holds it (a function of its own: the
// sine and exponential inlined at each use crowd the instruction cache).
__device__ __noinline__ float3 oblique_flux(double scale, int kind, double f, double t0, double w, double t, double px,
                                            double py, double pz) {
  const double v = scale * pulse_value(kind, f, t0, w, t);
  return make_float3((float)(px * v), (float)(py * v), (float)(pz * v));
}

// (neighbour sum) - 6 E of a quad, one component: the 7-point Laplacian
// -h^2 M^-1 L E with mirrored ghost nodes, summed as right + left, y + 1, y - 1,
// above, below.  cm, cp: the values at x - 1 and x + 4.
__device__ __forceinline__ Quad neg_lap(const Quad &cen, float cm, float cp, const Quad &yp, const Quad &ym, const Quad &ab,
                                        const Quad &below, bool edge, int x, int n) {
  float s0 = cen.l.y + cm, s1 = cen.h.x + cen.l.x, s2 = cen.h.y + cen.l.y, s3 = cp + cen.h.x;
  if (edge) {  // mirror columns: ghost x-1 = x+1 at x = 0, x+1 = x-1 at x = n-1
    if (x == 0) s0 = cen.l.y + cen.l.y;
    if (x == n - 1) s0 = cm + cm;
    if (x + 1 == n - 1) s1 = cen.l.x + cen.l.x;
    if (x + 2 == n - 1) s2 = cen.l.y + cen.l.y;
    if (x + 3 == n - 1) s3 = cen.h.x + cen.h.x;
  }
  const Quad sn = {make_float2(s0, s1), make_float2(s2, s3)};
  return fma4(cen, f2(-6.f), add4(add4(add4(add4(sn, yp), ym), ab), below));
}

// E^{n+1} = E^n + A (E^n - E^{n-1}) + B E^n - C R, with Q = -R already scaled by
// tau^2 / h^2 and rounded.  The scaling stays apart from this sum, behind a
// branch: contracted with it (as the compiler does within a block, the packed
// intrinsics notwithstanding), vacuum nodes would round one way here and
// another there, and the error of a 201^3 run against FP64 grew from 2.3e-6 to
// 8e-6.
__device__ __forceinline__ Quad update(const Quad &cen, const Quad &od, const Quad &Q, const Quad &A, const Quad &B,
                                       const Quad &C) {
  return add4(cen, add4(mul4(A, fma4(od, f2(-1.f), cen)), fma4(C, Q, mul4(B, cen))));
}
__device__ __forceinline__ Quad update(const Quad &cen, const Quad &od, const Quad &Q) {  // A = 1, B = 0, C = 1
  return add4(cen, add4(fma4(od, f2(-1.f), cen), Q));
}

// GEN: the launch may hold problems with element-gather rows, unpadded history
// rows or an oblique source without a table; without it, that code is left out
// (it crowds registers and the instruction cache: 16 x 161^3 583 -> 545 us a
// forward step, 587 -> 578 an adjoint one).
template <bool ADJ, int NB, bool GEN>
__global__ void __launch_bounds__(QUAD_THREADS, 2) k_step_quad(const __grid_constant__ StepLaunch<float, NB> L) {
  using S = QuadStage;
  constexpr int RE = S::RE, BW = S::BXW, TXY = S::TXY;
  const CtaTile ct = cta_tile(L);
  const StepParams<float> &P = L.p[NB == 1 ? 0 : ct.prob];
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  uint64_t *bar = (uint64_t *)(smem + S::BAR_OFF);  // a turn's planes have landed
  uint64_t *emp = bar + S::NB;                      // a turn has ended
  const int n = P.n;
  const int tid = threadIdx.x;
  const int x0 = ct.tx * S::TX, y0 = ct.ty * S::TY;
  const int k0 = ct.k0, k1 = min(ct.k1, n);
  // does the item hold nodes of FEM rows or free nodes
  const bool full = x0 <= P.b - 1 && x0 + S::TX - 1 >= P.a + 1 && y0 <= P.b - 1 && y0 + S::TY - 1 >= P.a + 1 &&
                    k0 <= P.b - 1 && k1 > P.a + 1;
  const QuadRing R = full ? QuadRing{S::FULL_NE, S::FULL_NO, S::FULL_E, S::FULL_O}
                          : QuadRing{S::LEAN_NE, S::LEAN_NO, S::LEAN_E, S::LEAN_O};
  if (tid == 0) {
    for (int s = 0; s < S::NB; ++s) {
      mbar_init(&bar[s], 2);
      mbar_init(&emp[s], QUAD_CONSUMERS / 32);
    }
    mbar_fence_init();
    tma_prefetch_desc(&L.cur);
    tma_prefetch_desc(&L.old);
    tma_prefetch_desc(&L.s);
    tma_prefetch_desc(&L.q);
  }
  pdl_launch_dependents();
  pdl_wait();
  if (!ADJ) sample_detectors(P, ct, tid, tiles_pair_x(n), (n + S::TY - 1) / S::TY, QUAD_CONSUMERS);
  if (k0 >= n) return;  // uniform per CTA
  __syncthreads();

  if (tid >= QUAD_CONSUMERS) {
    if (tid == QUAD_CONSUMERS)
      produce_quads<S>(L, R, smem, bar, emp, x0, y0, k0, k1, n, full, P.a, P.b, P.chan, P.spin_limit, P.err);
    return;
  }

  // nodes x .. x + 3 of row y of every plane; a warp takes four rows
  const int lane = tid & 31;
  const int yy = 4 * (tid >> 5) + (lane >> 3);
  const int xl = 4 * (lane & 7);
  const int x = x0 + xl, y = y0 + yy;
  const int ci = (yy + 1) * BW + S::HX + xl;  // node 0 in a staged plane (16-byte aligned)
  const int oi = yy * S::TX + xl;             // node 0 in a centre box
  // (a quad that reaches beyond x = n - 1 also writes the row's padding: px is a multiple of 8)
  const bool live = x < n && y < n;
  const int dym = (y == 0) ? BW : -BW, dyp = (y == n - 1) ? -BW : BW;  // mirror rows
  const bool edge = x0 == 0 || x0 + S::TX >= n;                        // the tile holds a mirror column
  const uint32_t sides = (P.abs_now | P.abs_next) & (DDFD_ABS_X0 | DDFD_ABS_X1 | DDFD_ABS_Y0 | DDFD_ABS_Y1);
  const bool ybnd = (y == 0 && (sides & DDFD_ABS_Y0)) || (y == n - 1 && (sides & DDFD_ABS_Y1));
  const bool colbnd = ybnd || (x == 0 && (sides & DDFD_ABS_X0)) || (x + 3 >= n - 1 && (sides & DDFD_ABS_X1));
  const bool tail = x0 + S::TX == n - 1 && xl == S::TX - 4;
  const uint32_t plane = (uint32_t)P.px * (uint32_t)n;
  const uint32_t cs = (uint32_t)P.cs;
  float *out = P.old + (long long)k0 * plane + (long long)P.px * y + x;

  // update coefficients of a node with fn absorbing faces (at step k - 1 in the
  // adjoint) and fnn (at step k + 1): damping tau/h per face (explicit roundings,
  // here and in the x tail: every copy of this code rounds alike)
  auto damping = [&](int fn, int fnn, float &A, float &Bc, float &Cq) {
    const float cc = __fmul_rn(P.cb, (float)fn);
    const float ccn = ADJ ? __fmul_rn(P.cb, (float)fnn) : cc;
    const float inv = fn == 0 ? P.inv_tab[0] : fn == 1 ? P.inv_tab[1] : fn == 2 ? P.inv_tab[2] : P.inv_tab[3];  // 1 / (1 + cc)
    A = __fmul_rn(__fsub_rn(1.f, ccn), inv);
    Bc = __fmul_rn(__fsub_rn(ccn, cc), inv);
    Cq = inv;
  };
  // flux (forward) or detector residuals (adjoint) of top node (xn, y), added to R
  auto top_node = [&](int xn, float Rn[3]) {
    if (!ADJ && P.src_on) {
      if (!P.oblique) {
        Rn[1] -= P.src_y;
      } else if (!GEN || P.src_tab) {
#pragma unroll
        for (int c = 0; c < 3; ++c) Rn[c] -= P.src_tab[xn + P.px * (y + n * c)];
      } else {
        const float3 v = oblique_flux(P.src_scale, P.pulse_kind, P.freq, P.t0, P.width, P.t_n - P.delay[xn + n * y],
                                      P.pol[0], P.pol[1], P.pol[2]);
        Rn[0] -= v.x, Rn[1] -= v.y, Rn[2] -= v.z;
      }
    }
    if (ADJ && P.n_det > 0) {
      // detector residual sources of this node at step k, summed and scaled
      // by k_det_sources
      const int u = P.det_slot[xn + n * y];
      if (u >= 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) Rn[c] += P.src_k[3 * u + c];
      }
    }
  };
  // the boundary form of the update of a quad with boundary nodes in plane k
  // (Q: -tau^2 h^2 M^-1 K E)
  const int fy = face_count(1, y, 1, n, P.abs_now), fyn = ADJ ? face_count(1, y, 1, n, P.abs_next) : 0;
  auto boundary_quad = [&](int k, Quad Q[3], Quad &A, Quad &B, Quad &C) {
    const int fk = fy + face_count(1, 1, k, n, P.abs_now), fkn = ADJ ? fyn + face_count(1, 1, k, n, P.abs_next) : 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int fn = fk + face_count(x + j, 1, 1, n, P.abs_now), fnn = ADJ ? fkn + face_count(x + j, 1, 1, n, P.abs_next) : 0;
      if (fn | fnn) {  // (a FEM node of the quad keeps its coefficients)
        float An, Bn, Cn;
        damping(fn, fnn, An, Bn, Cn);
        set(A, j, An), set(B, j, Bn), set(C, j, Cn);
      }
    }
    if (k == n - 1) {
      if (!ADJ && P.src_on && (GEN ? P.src_tab != nullptr : P.oblique != 0)) {
#pragma unroll
        for (int c = 0; c < 3; ++c) Q[c] = add4(Q[c], ld4(P.src_tab + x + P.px * (y + n * c)));
      } else if (ADJ || P.src_on) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (x + j < n) {
            float Rn[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) Rn[c] = -get(Q[c], j);
            top_node(x + j, Rn);
#pragma unroll
            for (int c = 0; c < 3; ++c) set(Q[c], j, -Rn[c]);
          }
      }
    }
  };
  // x tail: with n = 32 m + 1 the launch has m tiles in x, the last ending at
  // x = n - 2, and its lanes owning columns 28..31 also update the boundary
  // node (n - 1, y), in the staged x halo (an FD node, never FEM or free):
  // 7-point row with the mirror ghost x + 1 = x - 1, summed like the others.
  // e0, e1: the node in planes k, k + 1; tb: its values in plane k - 1; tov:
  // its previous level in plane k, read a plane ahead (only this thread writes it)
  float tb[3] = {0.f, 0.f, 0.f}, tov[3] = {0.f, 0.f, 0.f};
  if (tail && y < n) {
#pragma unroll
    for (int c = 0; c < 3; ++c) tov[c] = out[c * cs + 4];
  }
  auto update_tail = [&](int k, bool kbnd, const float *e0, const float *e1) {
    float Re[3], Ae = 1.f, Be = 0.f, Ce = 1.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float *e = e0 + c * RE;
      const float xme = e[-1];
      Re[c] = __fmaf_rn(6.f, e[0], -(((((xme + xme) + e[dyp]) + e[dym]) + e1[c * RE]) + tb[c]));
      Re[c] = __fmul_rn(Re[c], P.r2);
      tb[c] = e[0];
    }
    if (ybnd || (sides & DDFD_ABS_X1) || kbnd) {
      damping(face_count(n - 1, y, k, n, P.abs_now), ADJ ? face_count(n - 1, y, k, n, P.abs_next) : 0, Ae, Be, Ce);
      if (k == n - 1) top_node(n - 1, Re);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float ce = e0[c * RE], ov = tov[c];
      if (k + 1 < k1) tov[c] = out[c * cs + plane + 4];
      const float m = __fmaf_rn(Be, ce, -__fmul_rn(Ce, Re[c]));
      out[c * cs + 4] = __fadd_rn(ce, __fmaf_rn(Ae, __fsub_rn(ce, ov), m));
    }
  };

  const float2 R2 = f2(P.r2);
  int turn = 0;  // the turn whose planes are waited for next
  auto wait_next = [&]() {
    const bool ok = mbar_wait_bounded(&bar[turn % S::NB], (uint32_t)((turn / S::NB) & 1), P.spin_limit);
    ++turn;
    return ok;
  };
  // gives up after a timeout, for the warp as a whole (so __syncwarp stays safe)
  auto all_ok = [&](bool ok) {
    if (__all_sync(0xffffffffu, ok)) return true;
    if (lane == 0) atomicOr(P.err, 4);
    return false;  // the producer times out on the slots we no longer release
  };
  auto end_turn = [&](int j) {  // one arrival per warp (turns 1, 2, ...)
    __syncwarp();
    if (lane == 0) mbar_arrive(&emp[(j - 1) % S::NB]);
  };
  const int klo = (P.abs_now | P.abs_next) & DDFD_ABS_BOTTOM ? 0 : -1;
  auto boundary_plane = [&](int k) { return k == klo || k == n - 1; };
  const float *T = (const float *)smem + ci;                             // the thread's nodes in halo slot 0
  const float *TC = (const float *)(smem + R.ne * R.ebytes) + oi;  // ... in centre slot 0
  if (!all_ok(wait_next())) return;

  Quad q0[3], q1[3], q2[3];  // three successive planes, their roles rotating
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    q0[c] = ld4(T + c * RE);
    q1[c] = ld4(T + R.ebytes / 4 + c * RE);
    if (tail) tb[c] = T[c * RE + 4];
  }

  if (!full) {
    // finite-difference nodes only
    // side faces: the coefficients of every plane but the first and last
    Quad SA = {f2(1.f), f2(1.f)}, SB = {f2(0.f), f2(0.f)}, SC = {f2(1.f), f2(1.f)};
    if (colbnd) {
      Quad none[3];
      boundary_quad(1, none, SA, SB, SC);
    }
    int es = 1, os = 1, k = k0;  // slots of plane k
    auto step = [&](const Quad (&below)[3], const Quad (&cen)[3], Quad (&ab)[3]) {
      if (k >= k1 || !all_ok(wait_next())) return false;
      const int es1 = es + 1 == S::LEAN_NE ? 0 : es + 1;
      const float *E0 = T + es * (S::LEAN_E / 4), *E1 = T + es1 * (S::LEAN_E / 4);
      const float *O0 = TC + os * (S::LEAN_O / 4);
#pragma unroll
      for (int c = 0; c < 3; ++c) ab[c] = ld4(E1 + c * RE);
      if (live) {
        Quad Q[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float *e = E0 + c * RE;
          Q[c] = mul4(neg_lap(cen[c], e[-1], e[4], ld4(e + dyp), ld4(e + dym), ab[c], below[c], edge, x, n), R2);
        }
        const bool kbnd = boundary_plane(k);
        if (colbnd || kbnd) {
          Quad A = SA, B = SB, C = SC;
          if (kbnd) boundary_quad(k, Q, A, B, C);
#pragma unroll
          for (int c = 0; c < 3; ++c) st4(out + c * cs, update(cen[c], ld4(O0 + c * TXY), Q[c], A, B, C));
        } else {
#pragma unroll
          for (int c = 0; c < 3; ++c) st4(out + c * cs, update(cen[c], ld4(O0 + c * TXY), Q[c]));
        }
        if (tail) update_tail(k, kbnd, E0 + 4, E1 + 4);
      }
      out += plane;
      end_turn(k - k0 + 1);
      es = es1;
      if (++os == S::LEAN_NO) os = 0;
      ++k;
      return true;
    };
#pragma unroll 1
    while (step(q0, q1, q2) && step(q1, q2, q0) && step(q2, q0, q1)) {
    }
    return;
  }

  const bool colfem = y > P.a && y < P.b && x + 3 > P.a && x < P.b;  // some node strictly inside the cube
  const bool colfree = y >= P.f0 && y < P.f0 + P.nf && x + 3 >= P.f0 && x < P.f0 + P.nf;
  bool fnode[4];  // node j's column lies in the free box
#pragma unroll
  for (int j = 0; j < 4; ++j) fnode[j] = colfree && x + j >= P.f0 && x + j < P.f0 + P.nf;
  const int fcol = (x - P.f0) + P.nf * (y - P.f0);  // node 0 among the free nodes of plane f0
  const int hcol = (x - P.hx) + P.hp * (y - P.f0);  // ... in the history's layout
  int em = 0, os = 1, k = k0;                       // halo slot of plane k - 1, centre slot of plane k
  auto step = [&](const Quad (&below)[3], const Quad (&cen)[3], Quad (&ab)[3]) {
    if (k >= k1 || !all_ok(wait_next())) return false;
    const int e0s = em + 1 == S::FULL_NE ? 0 : em + 1, ep = e0s + 1 == S::FULL_NE ? 0 : e0s + 1;
    const float *Em = T + em * (S::FULL_E / 4), *E0 = T + e0s * (S::FULL_E / 4), *Ep = T + ep * (S::FULL_E / 4);
    const float *C0 = TC + os * (S::FULL_O / 4);  // + Q_OFF / 4
    const bool fem = colfem && k > P.a && k < P.b;
    const bool fre = colfree && k >= P.f0 && k < P.f0 + P.nf;
    const bool kbnd = boundary_plane(k);
#pragma unroll
    for (int c = 0; c < 3; ++c) ab[c] = ld4(Ep + c * RE);
    if (live) {
      // the gradient operands of this plane's free nodes (E^k history, block
      // sums), asked for now and used after the stencil
      const int fp = fcol + P.nf * P.nf * (k - P.f0), hq = hcol + P.hp * P.nf * (k - P.f0);
      Quad hv[3], gp[2];  // gp: (g_eps, g_sig) of nodes 0, 1 and of nodes 2, 3
      if (ADJ) {
        const float *hr = P.hist_r + hq, *g = P.gpart + 2 * (long long)hq;
        const bool sums = fre && !(P.gmode & GM_FIRST);
#pragma unroll
        for (int c = 0; c < 3; ++c) hv[c] = {f2(0.f), f2(0.f)};
        gp[0] = gp[1] = {f2(0.f), f2(0.f)};
        if (!GEN || P.hvec) {
          if (fre) {
#pragma unroll
            for (int c = 0; c < 3; ++c) hv[c] = ld4(hr + c * P.hcs);
          }
          if (sums) gp[0] = ld4(g), gp[1] = ld4(g + 4);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
              if (fre && fnode[j]) set(hv[c], j, hr[c * P.hcs + j]);
            if (sums && fnode[j]) (j & 1 ? gp[j >> 1].h : gp[j >> 1].l) = reinterpret_cast<const float2 *>(g)[j];
          }
        }
        if (fre && (P.gmode & GM_FOLD)) {
#pragma unroll
          for (int j = 0; j < 4; j += 3)
            if (fnode[j]) {
              prefetch_l2(P.gacc_e + fp + j);
              prefetch_l2(P.gacc_s + fp + j);
            }
        }
      }
      // s where the Gauss-law term is taken: the forward at the 36 nodes (read
      // for each component: 36 registers more would spill), the adjoint at the
      // quad's own
      const float *Sm = Em + S::S_OFF / 4, *S0 = E0 + S::S_OFF / 4, *Sp = Ep + S::S_OFF / 4;
      bool gauss = fem && !(GEN && P.ebe_r);
      Quad sc;
      if (ADJ && gauss) {
        sc = ld4(S0);
        gauss = fre || sc.l.x != 0.f || sc.l.y != 0.f || sc.h.x != 0.f || sc.h.y != 0.f;
      }
      // Q holds -R, so that every subtraction is a multiply-add with a constant
      // (exact negations); a boundary node converts to R for the scalar
      // boundary terms.
      Quad Q[3], O[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) O[c] = {f2(0.f), f2(0.f)};
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float *e = E0 + c * RE;
        Hood v;
        v.mc = ADJ ? below[c] : ld4(Em + c * RE);  // (forward: plane k - 1 is still staged, and registers are short)
        v.ym = ld4(e + dym);
        v.yp = ld4(e + dyp);
        v.cm = e[-1];
        v.cp = e[4];
        Q[c] = neg_lap(cen[c], v.cm, v.cp, v.yp, v.ym, ab[c], v.mc, edge, x, n);
        if (gauss) {
          // sum_o B_o w_{i+o}, w = s E forward, mu in the adjoint
          v.c = cen[c], v.pc = ab[c];
          v.py = ld4(Ep + c * RE + BW), v.my = ld4(Em + c * RE - BW);
          v.ypp = e[BW + 4], v.ymm = e[-BW - 1];
          v.pcp = Ep[c * RE + 4], v.pyp = Ep[c * RE + BW + 4];
          v.mcm = Em[c * RE - 1], v.mym = Em[c * RE - BW - 1];
          if (!ADJ) {
            if (c > 0) asm volatile("" ::: "memory");
            v.c = mul4(v.c, ld4(S0)), v.yp = mul4(v.yp, ld4(S0 + BW)), v.ym = mul4(v.ym, ld4(S0 - BW));
            v.pc = mul4(v.pc, ld4(Sp)), v.py = mul4(v.py, ld4(Sp + BW));
            v.mc = mul4(v.mc, ld4(Sm)), v.my = mul4(v.my, ld4(Sm - BW));
            v.cm *= S0[-1], v.cp *= S0[4], v.ypp *= S0[BW + 4], v.ymm *= S0[-BW - 1];
            v.pcp *= Sp[4], v.pyp *= Sp[BW + 4], v.mcm *= Sm[-1], v.mym *= Sm[-BW - 1];
          }
          hood_acc(c, v, O);
        }
      }
      Quad od[3], nw[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) od[c] = ld4(C0 + c * TXY);
      Quad A = {f2(1.f), f2(1.f)}, B = {f2(0.f), f2(0.f)}, C = {f2(1.f), f2(1.f)};
      if (fem) {
        A = ld4(C0 + S::Q_OFF / 4);
        C = ld4(C0 + S::Q_OFF / 4 + TXY);
        if (GEN && P.ebe_r) {
          // element-by-element rows computed by k_ebe for this step
          const int fm = P.b - P.a - 1;
          const long long row = (x - P.a - 1) + (long long)fm * ((y - P.a - 1) + (long long)fm * (k - P.a - 1));
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (x + j > P.a && x + j < P.b) {
#pragma unroll
              for (int c = 0; c < 3; ++c) {
                set(Q[c], j, -P.ebe_r[c * P.ebe_rows + row + j]);
                if (ADJ) set(O[c], j, P.ebe_q[c * P.ebe_rows + row + j]);
              }
            }
        } else if (!ADJ) {
#pragma unroll
          for (int c = 0; c < 3; ++c) Q[c] = fma4(O[c], f2(-1.f / 6.f), Q[c]);
        } else if (gauss) {
          const Quad ns0 = mul4(sc, f2(-1.f));
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            O[c] = mul4(O[c], f2(1.f / 6.f));  // kept for the gradient
            Q[c] = fma4(ns0, O[c], Q[c]);
          }
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) Q[c] = mul4(Q[c], R2);
      if (colbnd || kbnd) boundary_quad(k, Q, A, B, C);
      if (fem || colbnd || kbnd) {
#pragma unroll
        for (int c = 0; c < 3; ++c) nw[c] = update(cen[c], od[c], Q[c], A, B, C);
      } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) nw[c] = update(cen[c], od[c], Q[c]);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) st4(out + c * cs, nw[c]);
      if (fre) {
        if (!ADJ) {
          if (P.hist_w) {
            float *hw = P.hist_w + hq;
            if (!GEN || P.hvec) {
#pragma unroll
              for (int c = 0; c < 3; ++c) st4(hw + c * P.hcs, nw[c]);
            } else {
#pragma unroll
              for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                  if (fnode[j]) hw[c * P.hcs + j] = get(nw[c], j);
            }
          }
        } else {
          // the nodes' gradient terms in packed FP32 (at a node that is not free
          // they land in the rows' padding, or are not stored)
          Quad ge = {f2(0.f), f2(0.f)}, gs = {f2(0.f), f2(0.f)};
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const Quad te = fma4(O[c], R2, add4(fma4(cen[c], f2(-2.f), nw[c]), od[c]));
            ge = fma4(hv[c], te, ge);
            gs = fma4(hv[c], fma4(od[c], f2(-1.f), nw[c]), gs);
          }
          // block sums in FP32, folded into the FP64 accumulators
          const Quad g0 = {make_float2(ge.l.x, gs.l.x), make_float2(ge.l.y, gs.l.y)};
          const Quad g1 = {make_float2(ge.h.x, gs.h.x), make_float2(ge.h.y, gs.h.y)};
          gp[0] = P.gmode & GM_FIRST ? g0 : add4(gp[0], g0);
          gp[1] = P.gmode & GM_FIRST ? g1 : add4(gp[1], g1);
          if (P.gmode & GM_FOLD) {
            double ae[4], as[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (fnode[j]) ae[j] = P.gacc_e[fp + j], as[j] = P.gacc_s[fp + j];
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (fnode[j]) {
                const float2 g = j & 1 ? gp[j >> 1].h : gp[j >> 1].l;
                P.gacc_e[fp + j] = ae[j] + (double)g.x;
                P.gacc_s[fp + j] = as[j] + (double)g.y;
              }
          } else {
            float *g = P.gpart + 2 * (long long)hq;
            if (!GEN || P.hvec) {
              st4(g, gp[0]), st4(g + 4, gp[1]);
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (fnode[j]) reinterpret_cast<float2 *>(g)[j] = j & 1 ? gp[j >> 1].h : gp[j >> 1].l;
            }
          }
        }
      }
      if (tail) update_tail(k, kbnd, E0 + 4, Ep + 4);
    }
    out += plane;
    end_turn(k - k0 + 1);
    em = e0s;
    if (++os == S::FULL_NO) os = 0;
    ++k;
    return true;
  };
  if (ADJ || !GEN) {  // (two copies of the turn spill in the adjoint, one with register moves in the general forward)
#pragma unroll 1
    while (step(q0, q1, q2)) {
#pragma unroll
      for (int c = 0; c < 3; ++c) q0[c] = q1[c], q1[c] = q2[c];
    }
  } else {
#pragma unroll 1
    while (step(q0, q1, q2) && step(q0, q2, q1)) {
    }
  }
}

template <bool ADJ, int NB>
static cudaError_t set_smem_f32() {
  const cudaError_t e =
      cudaFuncSetAttribute(k_step_quad<ADJ, NB, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, QuadStage::SMEM);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_step_quad<ADJ, NB, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, QuadStage::SMEM);
}

cudaError_t prepare_step_kernels() {
  cudaError_t e;
  if ((e = set_smem_f32<false, 1>()) != cudaSuccess || (e = set_smem_f32<true, 1>()) != cudaSuccess ||
      (e = set_smem_f32<false, BATCH_MAX>()) != cudaSuccess || (e = set_smem_f32<true, BATCH_MAX>()) != cudaSuccess)
    return e;
  return prepare_step64_kernels();
}

int step_tiles_x(int n) { return tiles_pair_x(n); }
int step_tiles_y(int n) { return (n + STEP_TY - 1) / STEP_TY; }

// Launch grid: 1-D over the dispatch items, or the 3-D tile grid.
template <int NB>
static dim3 step_grid(const StepLaunch<float, NB> &L) {
  if (L.items) return dim3((unsigned)L.n_items);
  return dim3(step_tiles_x(L.p[0].n), step_tiles_y(L.p[0].n), L.zchunks * L.nprob);
}

template <bool ADJ, int NB>
static int launch_step(const StepLaunch<double, NB> &L, cudaStream_t s) {
  return launch_step64<ADJ, NB>(L, s);
}
// The oblique flux of SRC_ROWS steps of the problems that ask for it, one node and step a
// thread.  In the step kernel the 512 FP64 sines and exponentials of a top tile hold one
// SM up for 12 us; here they spread over all SMs, and what a thread waits for, 8 us of
// FP64 latency, is paid once in SRC_ROWS steps (us a forward step, 41^3 / 81^3 / 121^3:
// 13.7 / 19.9 / 34.9 -> 6.5 / 12.0 / 25.2; one step at a time 6.2 / 17.5 / 26.1; a table
// of every step 5.0 / 8.2 / 19.9).
template <int NB>
__global__ void __launch_bounds__(128) k_source_rows(const __grid_constant__ StepLaunch<float, NB> L, int st, double tau) {
  pdl_launch_dependents();
  const StepParams<float> &P = L.p[NB == 1 ? 0 : blockIdx.y];
  const int n = P.n, q = (int)(blockIdx.x * 128 + threadIdx.x), j = q / (n * n), d = q - j * n * n, y = d / n, x = d - n * y;
  const bool mine = j < SRC_ROWS && P.src_fill;
  double v = 0.0;
  if (mine) v = P.src_scale * pulse_value(P.pulse_kind, P.freq, P.t0, P.width, __dmul_rn((double)(st + j), tau) - P.delay[d]);
  pdl_wait();  // (the step before reads the table)
  if (mine)
    for (int c = 0; c < 3; ++c) const_cast<float *>(P.src_tab)[x + P.px * (y + (long long)n * (3 * j + c))] = (float)(P.pol[c] * v);
}

template <bool ADJ, int NB>
static int launch_step(const StepLaunch<float, NB> &L, cudaStream_t s) {
  bool rows = false;
  for (int q = 0; q < L.nprob && !ADJ; ++q) rows |= L.p[q].src_fill != 0;
  if (rows) {
    const int total = L.p[0].n * L.p[0].n * SRC_ROWS;
    const double tau = std::sqrt(L.p[0].tau2);  // (exactly: the root of a rounded square)
    launch_chained(k_source_rows<NB>, dim3((unsigned)((total + 127) / 128), (unsigned)L.nprob), 128, 0, s, L.chained != 0, L,
                   (int)std::lround(L.p[0].t_n / tau), tau);
    StepLaunch<float, NB> M = L;
    for (int q = 0; q < L.nprob; ++q) M.p[q].src_fill = 0;
    M.chained = 1;
    return 1 + launch_step<ADJ, NB>(M, s);
  }
  bool gen = false;
  for (int q = 0; q < L.nprob; ++q) {
    const StepParams<float> &P = L.p[q];
    gen |= P.ebe_r || !P.hvec || (!ADJ && P.src_on && P.oblique && !P.src_tab);
  }
  launch_chained(gen ? k_step_quad<ADJ, NB, true> : k_step_quad<ADJ, NB, false>, step_grid(L), QUAD_THREADS,
                 QuadStage::SMEM, s, L.chained != 0, L);
  return 1;
}

template <typename T, int NB>
int launch_forward_step(const StepLaunch<T, NB> &L, cudaStream_t s) {
  return launch_step<false, NB>(L, s);
}
template <typename T, int NB>
int launch_adjoint_step(const StepLaunch<T, NB> &L, cudaStream_t s) {
  return launch_step<true, NB>(L, s);
}

#define DDFD_STEP_INST(T, NB)                                                                           \
  template int launch_forward_step<T, NB>(const StepLaunch<T, NB> &, cudaStream_t); \
  template int launch_adjoint_step<T, NB>(const StepLaunch<T, NB> &, cudaStream_t);
DDFD_STEP_INST(float, 1)
DDFD_STEP_INST(double, 1)
DDFD_STEP_INST(float, BATCH_MAX)
DDFD_STEP_INST(double, BATCH_MAX)
#undef DDFD_STEP_INST

// Oblique flux of every step of the source phase over the top face, evaluated
// once: it depends on the configuration alone, and in the step kernels its FP64
// sine, exponential and division held the thread blocks of the top planes back
// (16 x 161^3: 587 -> 547 us a forward step; two waves on 41^3: 9.4 -> 5.1).
template <typename T>
__global__ void k_source_table(const __grid_constant__ StepParams<T> P, int steps, double tau, T *out) {
  constexpr int NC = sizeof(T) == 4 ? 3 : 1;
  const long long per = (long long)P.n * P.n, total = per * steps;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total; q += (long long)gridDim.x * blockDim.x) {
    const int st = (int)(q / per), d = (int)(q - per * st), y = d / P.n, x = d - P.n * y;
    // (the product rounded as the step kernels' t_n is: the same flux to the bit)
    const double v = P.src_scale * pulse_value(P.pulse_kind, P.freq, P.t0, P.width, __dmul_rn((double)st, tau) - P.delay[d]);
    T *o = out + (long long)st * NC * P.n * P.px + x + P.px * y;
    if (NC == 1)
      o[0] = (T)v;
    else
      for (int c = 0; c < NC; ++c) o[(long long)c * P.n * P.px] = (T)(P.pol[c] * v);
  }
}
template <typename T>
static void source_table(const StepParams<T> &P, int steps, double tau, T *out, cudaStream_t s) {
  const long long nb = ((long long)P.n * P.n * steps + 255) / 256;
  k_source_table<T><<<(int)(nb < 8192 ? nb : 8192), 256, 0, s>>>(P, steps, tau, out);
}
void launch_source_table(const StepParams<float> &P, int steps, double tau, float *out, cudaStream_t s) {
  source_table(P, steps, tau, out, s);
}
void launch_source_table(const StepParams<double> &P, int steps, double tau, double *out, cudaStream_t s) {
  source_table(P, steps, tau, out, s);
}

// y = h^2 M_eps^-1 K x in FP64 on every node (no damping, no source): the
// operator whose largest eigenvalue bounds the stable time step.  One thread
// per node; x, y unpadded (3 n^3); s read from the padded coefficient field.
template <typename T>
__global__ void k_apply_op(const double *x, double *y, int n, int px, int a, int b, const T *coef_s) {
  const long long nn = (long long)n * n * n;
  const long long nn2 = (long long)n * n;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nn;
       q += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(q % n), j = (int)((q / n) % n), k = (int)(q / nn2);
    const int ip = (i + 1 < n) ? i + 1 : n - 2, im = (i > 0) ? i - 1 : 1;
    const int jp = (j + 1 < n) ? j + 1 : n - 2, jm = (j > 0) ? j - 1 : 1;
    const int kp = (k + 1 < n) ? k + 1 : n - 2, km = (k > 0) ? k - 1 : 1;
    const long long pk = nn2 * k, rj = (long long)n * j;
    double out[3];
    for (int c = 0; c < 3; ++c) {
      const double *xc = x + c * nn;
      out[c] = 6.0 * xc[q] - xc[pk + rj + ip] - xc[pk + rj + im] - xc[pk + (long long)n * jp + i] -
               xc[pk + (long long)n * jm + i] - xc[nn2 * kp + rj + i] - xc[nn2 * km + rj + i];
    }
    double eps = 1.0;
    if (i > a && i < b && j > a && j < b && k > a && k < b) {
      auto sv = [&](int di, int dj, int dk) {
        return (double)coef_s[(i + di) + (long long)px * ((j + dj) + (long long)n * (k + dk))];
      };
      const double s0 = sv(0, 0, 0);
      eps = 1.0 + s0;
      const int dx[7] = {1, 0, 0, 1, 1, 0, 1}, dy[7] = {0, 1, 0, 1, 0, 1, 1}, dz[7] = {0, 0, 1, 0, 1, 1, 1};
      double v0[3], vp[7][3], st[3];
      for (int c = 0; c < 3; ++c) v0[c] = s0 * x[c * nn + q];
      for (int p = 0; p < 7; ++p) {
        const long long og = dx[p] + n * (dy[p] + (long long)n * dz[p]);
        for (int c = 0; c < 3; ++c)
          vp[p][c] = sv(dx[p], dy[p], dz[p]) * x[c * nn + q + og] +
                     sv(-dx[p], -dy[p], -dz[p]) * x[c * nn + q - og];
      }
      block_apply<double>(v0, vp, st);
      for (int c = 0; c < 3; ++c) out[c] += st[c];
    }
    for (int c = 0; c < 3; ++c) y[c * nn + q] = out[c] / eps;
  }
}

void launch_apply_op(const double *x, double *y, int n, int px, int a, int b, const void *coef_s, int fp32,
                     cudaStream_t s) {
  const long long nn = (long long)n * n * n;
  const long long nb = (nn + 255) / 256;
  const int blocks = (int)(nb < 8192 ? nb : 8192);
  if (fp32)
    k_apply_op<float><<<blocks, 256, 0, s>>>(x, y, n, px, a, b, (const float *)coef_s);
  else
    k_apply_op<double><<<blocks, 256, 0, s>>>(x, y, n, px, a, b, (const double *)coef_s);
}

}  // namespace ddfd
