// step_common.cuh -- device helpers shared by the step kernels of both
// lattices: the bounds checks of the debug build, periodic edge stores, the
// rest-population update and the collisions.
#pragma once

#include "kernels.h"
#include "physics.cuh"
#include "tma.cuh"

namespace mlsw {

// ---------------------------------------------------------------------------
// Bounds checks of the debug build (physics.cuh): a shared-memory pointer
// must lie in the CTA's dynamic shared memory, an index in its array, a
// global store in its buffer or plane. Out of range, the access is counted
// and goes to the first element instead. Release builds pass through.
// ---------------------------------------------------------------------------
#ifdef MLSW_DEBUG
extern __shared__ __align__(128) unsigned char dyn_smem_base[];
__device__ __forceinline__ bool dyn_smem_ok(const void* p, int bytes) {
  if (!__isShared(p)) return false;
  uint32_t size;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(size));
  const uint32_t a = smem_addr(p), lo = smem_addr(dyn_smem_base);
  return a >= lo && a + (uint32_t)bytes <= lo + size;
}
#endif
template <class P>
__device__ __forceinline__ P* chk_smem(P* p) {
#ifdef MLSW_DEBUG
  if (!dyn_smem_ok(p, (int)sizeof(P))) {
    note_bounds_violation();
    return reinterpret_cast<P*>(dyn_smem_base);
  }
#endif
  return p;
}
__device__ __forceinline__ int chk_index(int i, int n) {
#ifdef MLSW_DEBUG
  if (i < 0 || i >= n) {
    note_bounds_violation();
    return 0;
  }
#endif
  return i;
}
// offset of a global store inside its buffer or plane: i in [0, len)
__device__ __forceinline__ long chk_offset(long i, long len) {
#ifdef MLSW_DEBUG
  if (i < 0 || i >= len) {
    note_bounds_violation();
    return 0;
  }
#endif
  return i;
}
// global store target: p[0 .. count) inside [base, base + len), aligned for
// one access
__device__ __forceinline__ float* chk_global(float* base, float* p, long len, int count = 1) {
#ifdef MLSW_DEBUG
  const long i = p - base;
  if (i < 0 || i + count > len || (reinterpret_cast<uintptr_t>(p) & (4 * count - 1)) != 0) {
    note_bounds_violation();
    return base;
  }
#endif
  return p;
}

// ---------------------------------------------------------------------------
// Stores of one post-collision population to its streamed destination
// (dx, dy) (already periodic) and to the ghost cells that image it.
// ---------------------------------------------------------------------------
// Lattices with both sides >= 4 cells: a real column d has at most one
// ghost image (d + n for d < 2, d - n for d >= n - 2), likewise rows, so a
// population near an edge needs at most three extra stores.
constexpr int kNoImage = -(1 << 28);

__device__ __forceinline__ int image_of(int d, int n) {
  return d < 2 ? d + n : (d >= n - 2 ? d - n : kNoImage);
}

__device__ __forceinline__ void store_edge(float* __restrict__ plane_base, const Layout& L,
                                           int dx, int dy, int xi, int yi, float v) {
  // indices into the plane (not derived pointers), so that the stores keep
  // the base pointer's no-alias guarantee
  const long r0 = (long)dy * L.pitch;
  plane_base[chk_offset(r0 + dx + L.gx, L.plane)] = v;
  if (xi != kNoImage) plane_base[chk_offset(r0 + xi + L.gx, L.plane)] = v;
  if (yi != kNoImage) {
    const long r1 = (long)yi * L.pitch;
    plane_base[chk_offset(r1 + dx + L.gx, L.plane)] = v;
    if (xi != kNoImage) plane_base[chk_offset(r1 + xi + L.gx, L.plane)] = v;
  }
}

// ---------------------------------------------------------------------------
// The rest population after the collision, g0* = g0 + delta: the stored rest
// population g0 (shifted by H, O(h - H)) plus a small change (the incoming
// moving populations less the outgoing equilibria, times omega when tau !=
// 1). Rounding g0 + delta to FP32 loses up to half an ulp of g0 per cell
// and step, and in a slowly changing film (a dewetted precursor far from H)
// that loss has the same sign step after step. The exact rounding error
// (Fast2Sum, |g0| >= |delta| in the cells where it matters) is passed on
// instead, half to each of two opposite moving populations: their ulp is
// orders of magnitude finer, the momentum they carry is unchanged, and the
// cell's populations sum to the incoming mass to their rounding.
// ---------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ T rest_update(T g0, T delta, T& fa, T& fb) {
  const T out = g0 + delta;
  const T r = delta - (out - g0);  // exact: the part of delta the sum dropped
  fa = fmav(r, 0.5f, fa);
  fb = fmav(r, 0.5f, fb);
  return out;
}

// Equilibrium, BGK with forcing (Eqs. equilibrium_distribution, BGK) for one
// layer at one cell; fs[k] receives the post-collision populations (rest one
// stored shifted by H). g0: the stored rest population; small: the sum of
// the stored moving ones (h - H = g0 + small); J the flux, U = J / h the mean
// velocity, F the force; f_old (read only when !TAU1) the stored
// pre-collision populations.
//
// For opposite directions c and -c the equilibria share
//   w h (4.5 (c.U)^2 - 1.5 U^2) = w (4.5 (c.J)(c.U) - 1.5 J.U)
// and differ in the sign of 3 w c.J, and the forcing terms 3 w c.F are odd, so
// each pair costs one symmetric and one antisymmetric part; with tau = 1
// flux and force enter the latter only through J + F.
//
// D1Q3 (one component): w = 1/6, the pair is J U / 2 +- (J + F) / 2.
template <bool TAU1>
__device__ __forceinline__ void collide_d1q3(const KParams& P, float g0, float small, float j,
                                             float u, float F, const float* f_old,
                                             float (&fs)[3]) {
  const float sym = 0.5f * (j * u);
  if constexpr (TAU1) {
    const float anti = 0.5f * (j + F);
    fs[1] = sym + anti;
    fs[2] = sym - anti;
  } else {
    const float aeq = 0.5f * j, afr = 0.5f * F;
    fs[1] = fmaf(P.omega, (sym + aeq) - f_old[1], f_old[1]) + afr;
    fs[2] = fmaf(P.omega, (sym - aeq) - f_old[2], f_old[2]) - afr;
  }
  // rest population: h less the moving equilibria, g0 + (small - 2 sym),
  // relaxed by omega when tau != 1 (see rest_update)
  const float d = fmaf(-2.f, sym, small);
  fs[0] = rest_update(g0, TAU1 ? d : P.omega * d, fs[1], fs[2]);
}

// D2Q9: the products p_ab = J_a U_b give the symmetric parts
//   axes       p_xx / 3 - p_yy / 6,  p_yy / 3 - p_xx / 6
//   diagonals  (p_xx + p_yy) / 12 +- p_xy / 4,
// whose sum is (p_xx + p_yy) / 3. Directions: 1 (1,0), 2 (1,1), 3 (0,1),
// 4 (-1,1); 5..8 are their opposites.
template <bool TAU1, class T>
__device__ __forceinline__ void collide_d2q9(const KParams& P, T g0, T small, T jx, T jy, T ux,
                                             T uy, T Fx, T Fy, const T* f_old, T (&fs)[9]) {
  const T pxx = jx * ux, pyy = jy * uy, pxy = jx * uy;
  const T e = (pxx + pyy) * (1.f / 12.f);
  const T sym[4] = {fmav(pyy, -1.f / 6.f, pxx * (1.f / 3.f)), fmav(pxy, 0.25f, e),
                    fmav(pxx, -1.f / 6.f, pyy * (1.f / 3.f)), fmav(pxy, -0.25f, e)};
  if constexpr (TAU1) {
    const T mx = jx + Fx, my = jy + Fy;
    const T anti[4] = {mx * (1.f / 3.f), (mx + my) * (1.f / 12.f), my * (1.f / 3.f),
                       (my - mx) * (1.f / 12.f)};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      fs[q + 1] = sym[q] + anti[q];
      fs[q + 5] = sym[q] - anti[q];
    }
  } else {
    const T cj[4] = {jx, jx + jy, jy, jy - jx}, cf[4] = {Fx, Fx + Fy, Fy, Fy - Fx};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float w3 = (q & 1) ? 1.f / 12.f : 1.f / 3.f;
      const T aeq = cj[q] * w3, afr = cf[q] * w3;
      fs[q + 1] = fmav(P.omega, (sym[q] + aeq) - f_old[q + 1], f_old[q + 1]) + afr;
      fs[q + 5] = fmav(P.omega, (sym[q] - aeq) - f_old[q + 5], f_old[q + 5]) - afr;
    }
  }
  // rest population: h less the moving equilibria, g0 + (small - 8 e),
  // relaxed by omega when tau != 1 (see rest_update)
  const T d = fmav(e, -8.f, small);
  fs[0] = rest_update(g0, TAU1 ? d : d * P.omega, fs[1], fs[5]);
}

// Sum of the eight stored moving populations of one layer at a cell: the
// opposite directions first (their moving parts nearly cancel), then the
// diagonals with the axes. The layer's h - H is the rest population plus
// this sum, added last: adding the small populations to the O(h - H) rest
// population one by one would drop their low bits one direction at a time.
template <class T>
__device__ __forceinline__ T moving_sum(const T (&v)[9]) {
  return ((v[1] + v[5]) + (v[3] + v[7])) + ((v[2] + v[6]) + (v[4] + v[8]));
}

// moments of the nine populations of one layer at a cell (or a pair): the
// rest population, the sum of the moving ones, the flux
template <class T>
struct Moments {
  T g0, s, jx, jy;
};
template <class T>
__device__ __forceinline__ Moments<T> moments_of(const T (&v)[9]) {
  return {v[0], moving_sum(v), ((v[1] + v[2]) + v[8]) - ((v[4] + v[5]) + v[6]),
          ((v[2] + v[3]) + v[4]) - ((v[6] + v[7]) + v[8])};
}

}  // namespace mlsw
