// Device helpers shared by the FP32 and FP64 step kernels (ddfd_step.cu,
// ddfd_step64.cu): the source pulse, the absorbing faces of a node, plane
// staging by TMA, the tile of a CTA and the detector sampling.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "ddfd_internal.h"
#include "ddfd_tma.h"

namespace ddfd {

__device__ __forceinline__ double pulse_value(int kind, double f, double t0, double w, double t) {
  if (kind == DDFD_SRC_GAUSS) {
    const double s = t - t0;
    const double q = s / w;
    return sin(2.0 * 3.141592653589793 * f * s) * exp(-q * q);
  }
  return (t > 0.0 && t < 1.0 / f) ? sin(2.0 * 3.141592653589793 * f * t) : 0.0;
}

__device__ __forceinline__ int face_count(int i, int j, int k, int n, uint32_t abs) {
  int f = 0;
  if (i == 0 && (abs & DDFD_ABS_X0)) ++f;
  if (i == n - 1 && (abs & DDFD_ABS_X1)) ++f;
  if (j == 0 && (abs & DDFD_ABS_Y0)) ++f;
  if (j == n - 1 && (abs & DDFD_ABS_Y1)) ++f;
  if (k == 0 && (abs & DDFD_ABS_BOTTOM)) ++f;
  if (k == n - 1 && (abs & DDFD_ABS_TOP)) ++f;
  return f;
}

// FP64 (the FP32 kernel stages its two rings itself): starts the copies of plane p of
// produce_planes and arms its slot's "full" barrier with their bytes.
template <class S>
__device__ __forceinline__ void stage_plane(int p, const CUtensorMap *mcur, const CUtensorMap *mold,
                                            const CUtensorMap *ms, const CUtensorMap *mq, unsigned char *smem,
                                            uint64_t *bar, int x0, int y0, int k0, int k1, int n, bool tile_fem,
                                            int a, int b, int ch) {
  const int slot = p % S::RING;
  const int kk = k0 - 1 + p;
  const int ksrc = kk < 0 ? 1 : (kk >= n ? n - 2 : kk);  // mirror ghost planes
  unsigned char *st = smem + slot * S::BYTES;
  const bool interior = kk >= k0 && kk < k1;
  const bool coef = tile_fem && kk >= a && kk <= b;
  const bool qc = coef && interior;
  const uint32_t bytes = S::E_BYTES + (interior ? S::O_BYTES : 0) + (coef ? S::S_BYTES : 0) +
                         (qc ? S::Q_BYTES : 0);
  uint64_t *bb = &bar[slot];
  mbar_expect_tx(bb, bytes);
  tma_load_4d(st + S::E_OFF, mcur, x0 - S::HX, y0 - 1, ksrc, ch, bb);
  if (interior) tma_load_4d(st + S::O_OFF, mold, x0, y0, kk, ch, bb);
  if (coef) tma_load_4d(st + S::S_OFF, ms, x0 - S::HX, y0 - 1, kk, ch, bb);
  if (qc) tma_load_4d(st + S::Q_OFF, mq, x0, y0, kk, ch + 1, bb);
}

// Producer (one thread): stages plane p = kk - (k0 - 1) of the chunk into
// slot p % RING once the consumers have released the slot's previous plane
// (p - RING): the current level (halo box; mirrored ghost planes at kk = -1
// and kk = n), the previous level (centre box, computed planes only) and, on
// tiles touching the FEM cube, s (halo box, planes a..b) and (q1, q2)
// (centre box, computed planes a..b).  Every wait is bounded; on give-up it
// sets error bit 4 and still waits (bounded) for its issued copies.
template <class S>
__device__ __forceinline__ void produce_planes(const CUtensorMap *mcur, const CUtensorMap *mold,
                                               const CUtensorMap *ms, const CUtensorMap *mq,
                                               unsigned char *smem, uint64_t *bar, uint64_t *emp, int x0,
                                               int y0, int k0, int k1, int n, bool tile_fem, int a, int b,
                                               int ch, uint32_t spin, int *err) {
  const int nplanes = k1 - k0 + 2;
  int p = 0;
  bool ok = true;
  for (; p < nplanes; ++p) {
    const int slot = p % S::RING;
    // plane p reuses the slot of plane p - RING, whose release is completion
    // number p/RING - 1 of that slot's empty barrier
    if (p >= S::RING && !mbar_wait_bounded(&emp[slot], (uint32_t)((p / S::RING - 1) & 1), spin)) {
      ok = false;
      break;
    }
    stage_plane<S>(p, mcur, mold, ms, mq, smem, bar, x0, y0, k0, k1, n, tile_fem, a, b, ch);
  }
  if (!ok) atomicOr(err, 4);
  // every issued plane must land before the CTA can retire (bounded)
  const int first = p > S::RING ? p - S::RING : 0;
  for (int q = first; q < p; ++q)
    mbar_wait_bounded(&bar[q % S::RING], (uint32_t)((q / S::RING) & 1), spin);
}

// x tiles of the FP32 step kernel: with n = 32 m + 1 the last column is updated
// by the last of m tiles (the kernel's x tail) instead of by a tile of its own.
__host__ __device__ constexpr int tiles_pair_x(int n) { return n % STEP_TX == 1 ? n / STEP_TX : (n + STEP_TX - 1) / STEP_TX; }
// Tile of this CTA: (problem of the launch, tile x, tile y) and its planes
// [k0, k1), from the launch's dispatch order if it has one, else from the 3-D
// grid (z chunks of kz planes).
struct CtaTile {
  int prob, tx, ty, k0, k1;
};
template <typename LT>
__device__ __forceinline__ CtaTile cta_tile(const LT &L) {
  CtaTile t;
  if (L.items) {
    const uint32_t it = L.items[blockIdx.x];
    t.tx = (int)(it & 31u);
    t.ty = (int)((it >> 5) & 127u);
    t.k0 = (int)((it >> 12) & 1023u);
    t.k1 = t.k0 + (int)((it >> 22) & 63u) + 1;
    t.prob = (int)(it >> 28);
  } else {
    t.tx = (int)blockIdx.x;
    t.ty = (int)blockIdx.y;
    t.prob = (int)blockIdx.z / L.zchunks;
    const int zc = (int)blockIdx.z - t.prob * L.zchunks;
    const int kz = L.p[sizeof(L.p) == sizeof(L.p[0]) ? 0 : t.prob].kz;
    t.k0 = zc * kz;
    t.k1 = t.k0 + kz;
  }
  return t;
}

// Forward detector sampling of E^n (read-only in the step kernels): the CTAs
// that own the bottom planes (k0 = 0) of a tile column, one per column
// whatever the z chunking, share the 3 n_det values by their computing
// threads' index within the gx x gy columns.
template <typename T>
__device__ __forceinline__ void sample_detectors(const StepParams<T> &P, const CtaTile &ct, int tid, int gx, int gy,
                                                 int threads) {
  if (P.n_det <= 0 || ct.k0 != 0 || tid >= threads) return;
  const long long nb = (long long)gx * gy * threads;
  for (long long t = ((long long)ct.tx + (long long)gx * ct.ty) * threads + tid; t < 3LL * P.n_det; t += nb) {
    const int d = (int)(t / 3), c = (int)(t - 3LL * d);
    P.trace_n[t] = (double)P.cur[c * P.cs + P.det_node[d]];
  }
}

}  // namespace ddfd
