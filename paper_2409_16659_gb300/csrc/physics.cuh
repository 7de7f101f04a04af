// physics.cuh -- per-cell device routines of the multilayer shallow-water
// LBM step (FP32): lattice tables, layer pressures, friction coupling,
// equilibrium/collision. Used by the step kernels and by
// mlswlbm_friction_eval.
#pragma once

#include <cuda_runtime.h>

namespace mlsw {

constexpr int kMaxLayers = 5;

// ---------------------------------------------------------------------------
// Bounds-checked build (compiled with -DMLSW_DEBUG). Index helpers check
// every padded-layout index, shared-memory access and global store of the
// step kernels; an access out of range is counted and redirected to a
// harmless cell (index 0 of a population buffer is the padding cell
// x = -4 of the first row, which no real cell reads) instead of faulting.
// Each translation unit keeps its own counter; the host reads and clears
// them through mlswlbm_debug_bounds_violations. Release builds compile
// none of this.
// ---------------------------------------------------------------------------
#define MLSW_CAT2(a, b) a##b
#define MLSW_CAT(a, b) MLSW_CAT2(a, b)
#ifdef MLSW_DEBUG
static __device__ unsigned int g_bounds_violations;
__device__ __forceinline__ void note_bounds_violation() { atomicAdd(&g_bounds_violations, 1u); }
#define MLSW_DEFINE_BOUNDS_READER(fn)                                                  \
  unsigned fn() {                                                                      \
    unsigned v = 0, z = 0;                                                             \
    if (cudaMemcpyFromSymbol(&v, g_bounds_violations, sizeof v) != cudaSuccess) return ~0u; \
    if (cudaMemcpyToSymbol(g_bounds_violations, &z, sizeof z) != cudaSuccess) return ~0u;   \
    return v;                                                                          \
  }
#else
#define MLSW_DEFINE_BOUNDS_READER(fn) \
  unsigned fn() { return 0; }
#endif

// Kernel-side copy of the problem statement, rounded to FP32 once.
//
// Shifted rest population: the device stores g_0 = f_0 - H_i for the rest
// population of layer i (H_i a per-layer constant near the film thickness)
// and g_k = f_k otherwise. Moments are then formed as deviations
// dh_i = sum_k g_k (h_i = H_i + dh_i), so the interface stencils work on
// O(1e-3) numbers instead of O(1) ones. In FP32 the long-wave curvature of
// an O(1) height field is comparable to its rounding (ulp(1) = 1.2e-7), so
// storing f_0 itself loses the capillary signal; the shift keeps ~1e-10.
// The arithmetic of the scheme is unchanged: only the representation of
// f_0 moves by a constant.
// Device layout of a state buffer: every plane (layer i, direction k: plane
// i * Q + k; or moment q: plane 4 i + q) is a padded 2-D array of `rows` rows
// of `pitch` floats; the real cell (x, y) sits at row y, column x + gx. The
// ghost columns [-4, 0) and [nx, nx + 4) hold the periodic images of the real
// ones, so the step kernels read a strip plus its halo without any
// wrap-around arithmetic; rows are wrapped by the reader. gx keeps every row
// copy 16-byte aligned for the tensor-memory-access unit and, on D2Q9, every
// strip's stores on whole 32-byte sectors.
struct Layout {
  int nx, ny;    // real lattice
  int gx;        // padded column of the real cell (0, 0)
  int pitch;     // floats per padded row (multiple of 4)
  int rows;      // padded rows per plane
  long plane;    // pitch * rows
  int nplanes;   // planes of a buffer (0: not known, planes are then not checked)
  __host__ __device__ long at(int p, int x, int y) const {
#if defined(MLSW_DEBUG) && defined(__CUDA_ARCH__)
    if (x + gx < 0 || x + gx >= pitch || y < 0 || y >= rows || p < 0 ||
        (nplanes > 0 && p >= nplanes)) {
      note_bounds_violation();
      return 0;
    }
#endif
    return (long)p * plane + (long)y * pitch + (x + gx);
  }
  // floats of one buffer (0 when the plane count is not known)
  __host__ __device__ long length() const { return (long)nplanes * plane; }
};

struct KParams {
  int n;
  int nx, ny;
  float omega;                       // 1 / tau
  float gamma[kMaxLayers];           // gamma_{i,i+1}
  float S[kMaxLayers][kMaxLayers];   // S[l][k-1] = S_{lk}
  float Sd[kMaxLayers];              // S_{l1} nw mw / (nw - mw)
  int far_pairs;                     // 1: some S_{lk} with k >= 2 is not zero
  // friction (see friction()): -1 / (6 mu_i), beta_i / mu_i, beta_i^2 / (2 mu_i)
  float fr_visc[kMaxLayers], fr_slip[kMaxLayers], fr_slip2[kMaxLayers];
  float hstar;
  int nw, mw;
  float c_phi;                       // 1 / (nw - mw)
  float c_dphi;                      // nw mw / (nw - mw)
  float H[kMaxLayers];               // rest-population shift of each layer
  // Hsum[l][m] = H_{l+1} + ... + H_m (1-based layers, 0 <= l < m <= n): the
  // reference part of the thickness z_m - z_l between interfaces l and m
  float Hsum[kMaxLayers + 1][kMaxLayers + 1];
  Layout L;                          // padded layout of the state buffers
  // 1 when the lattice has fewer than 4 columns: a real column can then have
  // several ghost images
  int tiny;
  // substrate z_0(x, y) = sub_amp cos(2 pi (sub_kx x / nx + sub_ky y / ny));
  // sub_amp = 0 is the flat substrate
  float sub_amp;
  int sub_kx, sub_ky;
  // wetting potential: 0 the power law (nw, mw), 1 the charged-surface form
  // phi_k(d) = 2 a - a^2, a = e^{-kappa (d - k h*)}
  int wet_kind;
  float kappa;
  // 1: zero coefficients among the pairs that have a part in the pressures
  // (all of them with far_pairs, else k = 1)
  int zero_pairs;
};

// Substrate height at phase 2 pi m / nc, 0 <= m < nc
__device__ __forceinline__ float substrate_height(const KParams& P, long m, long nc) {
  float s, c;
  sincospif(2.f * (float)((double)m / (double)nc), &s, &c);
  return __fmul_rn(P.sub_amp, c);  // not fused into the sum it starts
}

// Substrate height at lattice cell (x, y) (any integers: the cosine is
// periodic); the phase is reduced exactly in integers.
__device__ __forceinline__ float substrate_at(const KParams& P, int x, int y) {
  const long nx = P.nx, ny = P.ny, nc = nx * ny;
  long m = ((long)P.sub_kx * x % nx) * ny + ((long)P.sub_ky * y % ny) * nx;
  m %= nc;
  if (m < 0) m += nc;
  return substrate_height(P, m, nc);
}

// ---------------------------------------------------------------------------
// lattices (section LBM): c_0 = 0, then the paper's order
// ---------------------------------------------------------------------------
template <int LAT> struct Lattice;

template <> struct Lattice<1> {  // D1Q3
  static constexpr int Q = 3;
  __host__ __device__ static constexpr int cx(int k) { return k == 1 ? 1 : (k == 2 ? -1 : 0); }
  __host__ __device__ static constexpr int cy(int) { return 0; }
  __host__ __device__ static constexpr float w(int k) { return k == 0 ? 2.f / 3.f : 1.f / 6.f; }
};

template <> struct Lattice<2> {  // D2Q9, counter-clockwise from +x
  static constexpr int Q = 9;
  __host__ __device__ static constexpr int cx(int k) {
    return (k == 1 || k == 2 || k == 8) ? 1 : ((k == 4 || k == 5 || k == 6) ? -1 : 0);
  }
  __host__ __device__ static constexpr int cy(int k) {
    return (k == 2 || k == 3 || k == 4) ? 1 : ((k == 6 || k == 7 || k == 8) ? -1 : 0);
  }
  __host__ __device__ static constexpr float w(int k) {
    return k == 0 ? 4.f / 9.f : ((k & 1) ? 1.f / 9.f : 1.f / 36.f);
  }
};

// ---------------------------------------------------------------------------
// Arithmetic on one cell (float) or on two cells at once (f2, a packed pair
// evaluated with the FP32x2 instructions of sm_100-class GPUs: one FFMA2 /
// FADD2 / FMUL2 does the work of two scalar ones). The per-cell routines
// below are written once over T in {float, f2}.
// ---------------------------------------------------------------------------
struct f2 {
  float2 v;
};
__device__ __forceinline__ f2 mk2(float a, float b) { return {make_float2(a, b)}; }
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return {__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return {__fmul2_rn(a.v, b.v)}; }
// a - b as one FFMA2: b * (-1) + a (exact product, one rounding)
__device__ __forceinline__ f2 operator-(f2 a, f2 b) {
  return {__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v)};
}
__device__ __forceinline__ f2 operator-(f2 a) { return {make_float2(-a.v.x, -a.v.y)}; }
__device__ __forceinline__ f2 operator+(f2 a, float b) { return a + mk2(b, b); }
__device__ __forceinline__ f2 operator+(float a, f2 b) { return mk2(a, a) + b; }
__device__ __forceinline__ f2 operator-(f2 a, float b) { return a - mk2(b, b); }
__device__ __forceinline__ f2 operator-(float a, f2 b) { return mk2(a, a) - b; }
__device__ __forceinline__ f2 operator*(f2 a, float b) { return a * mk2(b, b); }
__device__ __forceinline__ f2 operator*(float a, f2 b) { return mk2(a, a) * b; }
__device__ __forceinline__ f2& operator+=(f2& a, f2 b) { return a = a + b; }
__device__ __forceinline__ f2& operator-=(f2& a, f2 b) { return a = a - b; }

// One cell in the arithmetic of a pair: every operation rounds by itself, and
// the compiler contracts nothing, so a cell gets the bits it has in a pair.
struct f1 {
  float v;
};
__device__ __forceinline__ f1 operator+(f1 a, f1 b) { return {__fadd_rn(a.v, b.v)}; }
__device__ __forceinline__ f1 operator-(f1 a, f1 b) { return {__fsub_rn(a.v, b.v)}; }
__device__ __forceinline__ f1 operator*(f1 a, f1 b) { return {__fmul_rn(a.v, b.v)}; }
__device__ __forceinline__ f1 operator+(f1 a, float b) { return {__fadd_rn(a.v, b)}; }
__device__ __forceinline__ f1 operator-(f1 a, float b) { return {__fsub_rn(a.v, b)}; }
__device__ __forceinline__ f1 operator-(float a, f1 b) { return {__fsub_rn(a, b.v)}; }
__device__ __forceinline__ f1 operator*(f1 a, float b) { return {__fmul_rn(a.v, b)}; }
__device__ __forceinline__ f1 operator*(float a, f1 b) { return {__fmul_rn(a, b.v)}; }

template <class T> struct Num;
template <> struct Num<f1> {
  __device__ static f1 splat(float a) { return {a}; }
};
template <> struct Num<float> {
  __device__ static float splat(float a) { return a; }
};
template <> struct Num<f2> {
  __device__ static f2 splat(float a) { return mk2(a, a); }
};

__device__ __forceinline__ float fmav(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ f2 fmav(f2 a, f2 b, f2 c) { return {__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ f2 fmav(f2 a, float b, f2 c) { return fmav(a, mk2(b, b), c); }
__device__ __forceinline__ f2 fmav(float a, f2 b, f2 c) { return fmav(mk2(a, a), b, c); }
__device__ __forceinline__ f2 fmav(f2 a, f2 b, float c) { return fmav(a, b, mk2(c, c)); }
__device__ __forceinline__ f2 fmav(f2 a, float b, float c) { return fmav(a, mk2(b, b), mk2(c, c)); }
__device__ __forceinline__ f1 fmav(f1 a, f1 b, f1 c) { return {__fmaf_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ f1 fmav(f1 a, float b, f1 c) { return {__fmaf_rn(a.v, b, c.v)}; }
__device__ __forceinline__ f1 fmav(float a, f1 b, f1 c) { return {__fmaf_rn(a, b.v, c.v)}; }
__device__ __forceinline__ f1 fmav(f1 a, f1 b, float c) { return {__fmaf_rn(a.v, b.v, c)}; }
__device__ __forceinline__ f1 fmav(f1 a, float b, float c) { return {__fmaf_rn(a.v, b, c)}; }

// a product that is rounded by itself: the compiler fuses a scalar product
// into an addition where it likes, differently from kernel to kernel, and a
// packed one never. Products that feed additions go through this, so that
// scalar and packed cells, and all kernels, round identically.
__device__ __forceinline__ float mulr(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ f2 mulr(f2 a, f2 b) { return a * b; }
__device__ __forceinline__ f2 mulr(f2 a, float b) { return a * b; }
__device__ __forceinline__ f1 mulr(f1 a, f1 b) { return a * b; }
__device__ __forceinline__ f1 mulr(f1 a, float b) { return a * b; }

// fast reciprocal: the hardware's approximation, at most 1 ulp for normal
// arguments (here layer thicknesses and friction pivots, far from the ends
// of the FP32 range). Division intrinsics also scale the range of their
// arguments, which none here needs.
__device__ __forceinline__ float rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ f2 rcp(f2 x) { return mk2(rcp(x.v.x), rcp(x.v.y)); }
__device__ __forceinline__ f1 rcp(f1 x) { return {rcp(x.v)}; }
__device__ __forceinline__ f1 expv(f1 x) { return {expf(x.v)}; }
__device__ __forceinline__ float expv(float x) { return expf(x); }
__device__ __forceinline__ f2 expv(f2 x) { return mk2(expf(x.v.x), expf(x.v.y)); }

// v or exactly 0
__device__ __forceinline__ float keep_if(bool c, float v) { return c ? v : 0.f; }
__device__ __forceinline__ f2 keep_if(bool c, f2 v) {
  return mk2(c ? v.v.x : 0.f, c ? v.v.y : 0.f);
}

__device__ __forceinline__ f1 keep_if(bool c, f1 v) { return {c ? v.v : 0.f}; }

// r^e, e >= 0 a uniform run-time exponent: squares, with the factors of the
// low three bits chosen by selects (exponents in use are small) and a loop
// for the rest
template <class T>
__device__ __forceinline__ T ipow(T r, int e) {
  const T one = Num<T>::splat(1.f), r2 = r * r, r4 = r2 * r2;
  T a = ((e & 1) ? r : one) * ((e & 2) ? r2 : one);
  a = a * ((e & 4) ? r4 : one);
  if (e >= 8) {
    T s = r4 * r4;
#pragma unroll 1
    for (e >>= 3;; s = s * s) {
      if (e & 1) a = a * s;
      if ((e >>= 1) == 0) break;
    }
  }
  return a;
}

// ---------------------------------------------------------------------------
// Layer pressures at one cell, with the sign turned: q_i = p_atm - p_i (Eqs.
// Laplace_pressure, disjoining_pressure; p_i = sum_{j>=i} (Lambda_j + Pi_j)),
// so that the force of the next phase is F_i = R_i + h_i grad q_i without a
// negation (a packed pair has no sign modifier on its operands).
// Every interface pair (l, m = l + k), 0 <= l < m <= N, enters once with
// the thickness d = z_m - z_l between them: E = S_lk phi'_k(d)
// (1 + |grad z_l|^2 / 2) is subtracted from Pi_l and added to Pi_m, and
// S_lk phi_k(d) raises the tension of interface l. l = 0 is the substrate
// (height z0, slope factor sg0; no pressure of its own).
// The inputs are the deviations of the interface heights, zd[i - 1] =
// z_i - (H_1 + ... + H_i), so d = Hsum[l][m] + (zd_m - zd_l) (zd_0 = 0): the
// deviations are O(1e-3) numbers and their differences carry the FP32
// round-off of the deviations, not of the O(1) heights.
// ---------------------------------------------------------------------------
// NN: only nearest-neighbour pairs (k = 1) carry a spreading coefficient
// (S_{lk} = 0 for k >= 2, as in the paper's three-layer runs); the pair loop
// is then branch-free. With W32 (exponents 3, 2) the power law is evaluated
// as phi = r^2 (3 - 2 r), phi' = 6 r^2 (r - 1) / d.
// z0, sg0: the substrate height z_0 (on the scale of zd) and 1 + |grad z_0|^2 / 2
// at the cell; null for the flat substrate (0 and 1).
// G: the parameters that hold the reference thicknesses Hsum (P itself, but
// for alike lattices of a batch, which share the rest).
//
// Without NN or W32 the options are run-time values, but uniform ones: the
// pairs are evaluated in straight-line code for one combination (with or
// without far pairs, either potential), chosen once, so that the latencies
// of the pairs overlap. With SKIP a pair without a coefficient contributes
// exactly nothing, whatever its potential evaluates to (r^3 of a thin layer
// overflows, and 0 * inf is NaN). SKIP false: the host knows that every pair
// evaluated has one (zero_pairs).
enum PairForm { kPower32, kPower, kExponential };

template <int N, bool FAR, int FORM, bool SKIP, class T>
__device__ __forceinline__ void interface_pairs(const KParams& P, const KParams& G,
                                                const T (&zd)[N],
                                                const T (&sg)[N], const T* z0, const T* sg0,
                                                T (&ten)[N], T (&pi)[N]) {
#pragma unroll
  for (int l = 0; l < N; ++l) {
    const int i = l > 0 ? l - 1 : 0;
#pragma unroll
    for (int m = l + 1; m <= (FAR ? N : l + 1); ++m) {
      const int k = m - l;
      const float s = P.S[l][k - 1];
      T d;
      if (l > 0)
        d = (zd[m - 1] - zd[i]) + G.Hsum[l][m];
      else if (z0)
        d = (zd[m - 1] - *z0) + G.Hsum[l][m];
      else
        d = zd[m - 1] + G.Hsum[l][m];
      T phi, e;  // phi_k, S phi_k'
      if constexpr (FORM == kExponential) {
        // charged surfaces: a = e^{-kappa (d - k h*)}, phi = 2 a - a^2,
        // phi' = 2 kappa a (a - 1)
        const T a = expv(fmav(d, -P.kappa, P.kappa * ((float)k * P.hstar)));
        phi = a * (2.f - a);
        e = mulr(a * (a - 1.f), s * (2.f * P.kappa));
      } else {
        const T inv_d = rcp(d);
        const T r = ((float)k * P.hstar) * inv_d;
        if constexpr (FORM == kPower32) {
          const T r2 = r * r;
          phi = r2 * fmav(r, -2.f, 3.f);
          e = mulr((r2 * (r - 1.f)) * inv_d, k == 1 ? P.Sd[l] : s * P.c_dphi);
        } else {
          const T rm = ipow(r, P.mw), rn = mulr(rm, ipow(r, P.nw - P.mw));
          phi = fmav(rm, (float)P.nw, rn * (-(float)P.mw)) * P.c_phi;
          e = mulr((rn - rm) * inv_d, s * P.c_dphi);
        }
      }
      if (l > 0)
        e = mulr(e, sg[i]);
      else if (sg0)
        e = mulr(e, *sg0);
      if constexpr (SKIP) {
        phi = keep_if(s != 0.f, phi);
        e = keep_if(s != 0.f, e);
      }
      if (l > 0) {
        ten[i] = fmav(s, phi, ten[i]);
        pi[i] = pi[i] + e;
      }
      pi[m - 1] = pi[m - 1] - e;
    }
  }
}

template <int N, bool W32, class T, bool NN = false, bool SKIP = true>
__device__ __forceinline__ void neg_pressures(const KParams& P, const KParams& G,
                                              const T (&zd)[N], const T (&gx)[N],
                                              const T (&gy)[N], const T (&lz)[N], T (&q)[N],
                                              const T* z0 = nullptr, const T* sg0 = nullptr) {
  T ten[N], pi[N], sg[N];  // tension of the interface; -Pi of the layer; slope factor
#pragma unroll
  for (int i = 0; i < N; ++i) {
    ten[i] = Num<T>::splat(P.gamma[i]);
    pi[i] = Num<T>::splat(0.f);
    sg[i] = fmav(0.5f, fmav(gx[i], gx[i], gy[i] * gy[i]), Num<T>::splat(1.f));
  }
  if constexpr (NN && W32) {
    interface_pairs<N, false, kPower32, false>(P, G, zd, sg, z0, sg0, ten, pi);
  } else if constexpr (W32) {
    if (P.far_pairs)
      interface_pairs<N, true, kPower32, SKIP>(P, G, zd, sg, z0, sg0, ten, pi);
    else
      interface_pairs<N, false, kPower32, SKIP>(P, G, zd, sg, z0, sg0, ten, pi);
  } else if (P.wet_kind == 1) {
    interface_pairs<N, true, kExponential, true>(P, G, zd, sg, z0, sg0, ten, pi);
  } else if (P.far_pairs) {
    interface_pairs<N, true, kPower, true>(P, G, zd, sg, z0, sg0, ten, pi);
  } else {
    interface_pairs<N, false, kPower, true>(P, G, zd, sg, z0, sg0, ten, pi);
  }
  T acc = Num<T>::splat(0.f);
#pragma unroll
  for (int i = N - 1; i >= 0; --i) {
    const T own = fmav(ten[i], lz[i], pi[i]);
    acc = i == N - 1 ? own : acc + own;
    q[i] = acc;
  }
}

// ---------------------------------------------------------------------------
// Friction R_i = 2 mu_i h_i a_i (Eq. friction_force) from the thicknesses
// and the layers' mean velocities U_i = J_i / h_i.
//
// In Stokes layers with pressure gradient G_i, mu_i u'' = G_i; the force
// balance 0 = -h_i G_i + 2 mu_i h_i a_i makes R_i = h_i G_i. Integrating the
// stress down from the stress-free top (Eq. viscous_boundary with mu_{n+1} =
// 0), the interface above layer i carries -T_{i+1} and the one below it
// -T_i, with T_i = sum_{j>=i} R_j (T_{n+1} = 0). Integrating u upward through
// layer i from the velocity w_i of the interface below it, with the slip
// condition of Eq. (no_slip) (the parabola continued a distance beta_i below
// the interface meets w_i),
//   mean velocity  U_i = w_i - (b_i + c_i / h_i) T_i + (c_i / h_i) T_{i+1}
//                          - (h_i / mu_i) (T_i / 3 + T_{i+1} / 6)
//   next interface w_{i+1} - U_i = -(h_i / mu_i) (T_i / 6 + T_{i+1} / 3)
// with b_i = beta_i / mu_i, c_i = beta_i^2 / (2 mu_i). Subtracting
// neighbouring layers eliminates the w_i (w_1 = 0) and leaves a tridiagonal
// system for T: with a_i = h_i / (6 mu_i), s_i = c_i / h_i,
//   a_{i-1} T_{i-1} + (2 a_{i-1} + 2 a_i + b_i + s_i) T_i + (a_i - s_i) T_{i+1}
//     = U_{i-1} - U_i        (a_0 = U_0 = 0).
// Its rows are strictly diagonally dominant (a, b, s >= 0, a > 0), so
// elimination needs no pivoting for any n, thicknesses and slips. Solving
// the full n x n flux-gradient matrix took 2.5 times the arithmetic at n = 3
// (adjugate), and a pivoted elimination on single cells at n = 4, 5.
//
// Back substitution gives T_i = (r_i + (s_i - a_i) T_{i+1}) / d_i from the
// eliminated right-hand side r_i and pivot d_i. R_i = T_i - T_{i+1} is formed as
// (r_i - e_i T_{i+1}) / d_i, with e_i = d_i - (s_i - a_i) = 2 a_{i-1} + 3 a_i + b_i
// less the eliminated term: with slip, a thin layer's s_i = c_i / h_i exceeds
// the rest of its row, T_i and T_{i+1} then agree to h_i / c_i, and their
// difference lost as many digits (relative to the forces that the layers'
// fluxes make one by one: 1e-3 at h = 1e-4 and 1e-1 at 1e-6, 5e-5 at h = 0.05
// with a slip of 30; now 5e-7 throughout). T_i keeps a formula of its own
// because it can be the small one. One more addition and two more
// multiply-adds a layer.
// ih: 1 / h. TWO: both components (else the y ones are left alone).
// ---------------------------------------------------------------------------
template <int N, bool TWO, class T>
__device__ __forceinline__ void friction(const KParams& P, const T (&h)[N], const T (&ih)[N],
                                         const T (&Ux)[N], const T (&Uy)[N], T (&Rx)[N],
                                         T (&Ry)[N]) {
  T piv[N], nsup[N], ne[N], bx[N], by[N];  // ne: -e_i
  T na_prev;                               // -a_{i-1}
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const T na = mulr(h[i], P.fr_visc[i]);
    T rest = fmav(na, -2.f, Num<T>::splat(P.fr_slip[i]));  // d_i - s_i
    nsup[i] = fmav(ih[i], P.fr_slip2[i], na);
    if (i == 0) {
      bx[0] = Ux[0] * -1.f;
      if constexpr (TWO) by[0] = Uy[0] * -1.f;
    } else {
      const int j = i > 0 ? i - 1 : 0;
      const T nf = na_prev * piv[j];
      rest = fmav(nf, nsup[j] * -1.f, fmav(na_prev, -2.f, rest));
      bx[i] = fmav(nf, bx[j], Ux[j] - Ux[i]);
      if constexpr (TWO) by[i] = fmav(nf, by[j], Uy[j] - Uy[i]);
    }
    piv[i] = rcp(fmav(ih[i], P.fr_slip2[i], rest));
    ne[i] = na - rest;
    na_prev = na;
  }
  T tx, ty;  // T_{i+1}
#pragma unroll
  for (int i = N - 1; i >= 0; --i) {
    const T ox = tx, oy = ty;
    tx = mulr(i == N - 1 ? bx[i] : fmav(nsup[i], ox, bx[i]), piv[i]);
    Rx[i] = i == N - 1 ? tx : mulr(fmav(ne[i], ox, bx[i]), piv[i]);
    if constexpr (TWO) {
      ty = mulr(i == N - 1 ? by[i] : fmav(nsup[i], oy, by[i]), piv[i]);
      Ry[i] = i == N - 1 ? ty : mulr(fmav(ne[i], oy, by[i]), piv[i]);
    }
  }
}

}  // namespace mlsw
