// march.cuh -- the fused D2Q9 step (section LBM: moments, interfaces and
// pressures, force, BGK with forcing, streaming) as one warp marching down
// the rows of a strip of 64 columns, shared by the single-lattice kernels
// (step_d2q9.cu) and the batch kernels (batch_kernels.cu).
//
// A lane holds two neighbouring columns as one FP32x2 pair. Column
// neighbours come by warp shuffles, row neighbours from registers carried
// from row to row, so a unit of work needs no barrier with any other warp
// and no field goes through shared memory; only the input rows do, copied
// by TMA into a ring a few rows ahead. Of the 64 columns 56 are written: the
// 4 on each side feed the stencils (z three columns out, p two, the streamed
// populations one), and 56 columns are whole 32-byte sectors. Narrow lattices
// of four and five layers take one column a lane instead (march_solo): 26 of
// 32 columns, the same code and the same bits with half the registers.
//
// With row r arriving:
//   z(r)                 interface deviations z_i - sum_{j<=i} H_j
//   p(r - 1)             needs z of rows r - 2 .. r
//   collision(r - 2)     needs p of rows r - 3 .. r - 1
//   output(r - 3)        needs the populations of rows r - 4 .. r - 2
//
// State. With tau = 1 the collision forgets the populations: a step reads,
// per layer and cell, only the rest population g_0, the sum s of the moving
// ones (h - H = g_0 + s, kept apart because adding them would round s to the
// resolution of g_0) and the flux J = (J_x, J_y). These four moments are the
// state a lattice with tau = 1 is stored in ("moment form", 16 bytes instead
// of 36 per layer and cell, a quarter of the planes to write being whole
// rows); its populations at a time follow from the moments one step earlier
// by the same kernel with populations as its output (OP). Another tau keeps
// populations.
#pragma once

#include "kernels.h"
#include "physics.cuh"
#include "step_common.cuh"
#include "tma.cuh"

namespace mlsw {

constexpr unsigned kFullWarp = 0xffffffffu;

// T: the columns of a lane, a pair (f2) or one (f1)
template <class T> struct MarchLane;
template <> struct MarchLane<f2> {
  static constexpr int kBox = kMarchCols, kOut = kMarchOut, kHalo = kMarchHalo, kPer = 2;
};
template <> struct MarchLane<f1> {
  static constexpr int kBox = kSoloBox, kOut = kSoloOut, kHalo = kSoloHalo, kPer = 1;
};

template <int N, int MODE, bool OP, class T>
struct MarchShape {
  static constexpr bool TAU1 = MODE != kGeneral;
  static_assert(TAU1 || OP, "tau != 1 steps from populations to populations");
  static constexpr int PL = (TAU1 ? kMomPlanes : 9) * N;  // planes of an input row
  static constexpr int BOX = PL * MarchLane<T>::kBox;     // floats of a row's copy
  static constexpr int ROW = (BOX + 31) / 32 * 32;        // of a ring row (128-byte aligned)
  // Ring rows: three are live (the newest down to the one collided) and one
  // is in flight, which a row's time (about 2000 cycles) covers.
  static constexpr int RS = 4;
  // five layers: the older row of upward populations is parked in shared
  // memory (in registers it spills: 90 against 47 us a step at 1024^2)
  static constexpr bool PARK = N >= 5 && !OP && sizeof(T) == sizeof(f2);
  static constexpr size_t kOffPark = (size_t)RS * ROW * 4;
  static constexpr size_t kOffBar = kOffPark + (PARK ? (size_t)3 * N * kMarchCols * 4 : 0);
  static constexpr size_t kSmem = (kOffBar + 8 * RS + 127) / 128 * 128;
};

template <class T> __device__ __forceinline__ T ld_lane(const float* a);
template <> __device__ __forceinline__ f1 ld_lane<f1>(const float* a) { return {*chk_smem(a)}; }
template <> __device__ __forceinline__ f2 ld_lane<f2>(const float* a) {
  const float2 v = *reinterpret_cast<const float2*>(chk_smem(reinterpret_cast<const float2*>(a)));
  return mk2(v.x, v.y);
}
__device__ __forceinline__ void st_lane(float* a, f1 v) { *chk_smem(a) = v.v; }
__device__ __forceinline__ void st_lane(float* a, f2 v) {
  *chk_smem(reinterpret_cast<float2*>(a)) = v.v;
}

// the columns left and right of a pair: .x the column before v.x, .y the one
// after v.y (garbage in the outermost lanes, which feed no output)
__device__ __forceinline__ float2 beside(f2 v) {
  return make_float2(__shfl_up_sync(kFullWarp, v.v.y, 1), __shfl_down_sync(kFullWarp, v.v.x, 1));
}

// what streams in from the column to the left (right)
__device__ __forceinline__ f2 from_left(f2 v) {
  return mk2(__shfl_up_sync(kFullWarp, v.v.y, 1), v.v.x);
}
__device__ __forceinline__ f2 from_right(f2 v) {
  return mk2(v.v.y, __shfl_down_sync(kFullWarp, v.v.x, 1));
}
__device__ __forceinline__ f1 from_left(f1 v) { return {__shfl_up_sync(kFullWarp, v.v, 1)}; }
__device__ __forceinline__ f1 from_right(f1 v) { return {__shfl_down_sync(kFullWarp, v.v, 1)}; }

// Lattice derivatives of a field at the centre row of three, from the centre
// values c and the differences A = north - c and B = c - south:
// with V = north + south - 2 c = A - B and D = north - south = A + B,
//   d/dx = (c_E - c_W) / 2 + (V_E - V_W) / 12
//   d/dy = D / 3 + (D_E + D_W) / 12
//   lap  = (c_E + c_W - 2 c) + 2/3 V + (V_E + V_W) / 6,
// the isotropic stencils (weights 1/3, 1/12 and 2/3, 1/6) written in
// differences of neighbours, so no large values cancel and a constant field
// gives exact zeros.
template <bool LAP>
__device__ __forceinline__ void lattice_derivatives(f2 c, f2 A, f2 B, f2& gx, f2& gy, f2& lap) {
  const f2 V = A - B, D = A + B;
  const float2 cb = beside(c), vb = beside(V), db = beside(D);
  const f2 vd = mk2(V.v.y - vb.x, vb.y - V.v.x);
  const f2 ds = mk2(D.v.y + db.x, db.y + D.v.x);
  gy = fmav(D, 1.f / 3.f, ds * (1.f / 12.f));
  if constexpr (LAP) {
    const f2 fwd = mk2(c.v.y - c.v.x, cb.y - c.v.y), back = mk2(c.v.x - cb.x, c.v.y - c.v.x);
    const f2 vs = mk2(V.v.y + vb.x, vb.y + V.v.x);
    gx = fmav(fwd + back, 0.5f, vd * (1.f / 12.f));
    lap = fmav(V, 2.f / 3.f, fmav(vs, 1.f / 6.f, fwd - back));
  } else {
    gx = fmav(mk2(c.v.y - cb.x, cb.y - c.v.x), 0.5f, vd * (1.f / 12.f));
  }
}

template <bool LAP>
__device__ __forceinline__ void lattice_derivatives(f1 c, f1 A, f1 B, f1& gx, f1& gy, f1& lap) {
  const f1 V = A - B, D = A + B;
  const f1 cw = from_left(c), ce = from_right(c), vw = from_left(V), ve = from_right(V);
  const f1 vd = ve - vw, ds = from_right(D) + from_left(D);
  gy = fmav(D, 1.f / 3.f, ds * (1.f / 12.f));
  if constexpr (LAP) {
    const f1 fwd = ce - c, back = c - cw;
    gx = fmav(fwd + back, 0.5f, vd * (1.f / 12.f));
    lap = fmav(V, 2.f / 3.f, fmav(ve + vw, 1.f / 6.f, fwd - back));
  } else {
    gx = fmav(ce - cw, 0.5f, vd * (1.f / 12.f));
  }
}

// Stores of a pair of output values (columns ca, ca + 1 of a row that starts
// at `row`) and of their periodic images in the ghost columns [-4, 0) and
// [nx, nx + 4). With an even nx >= 8 a pair belongs to the lattice as a whole
// and has at most one image, as a whole: one predicated 8-byte store each,
// at 32-bit lane offsets from a warp-uniform address. Other lattices store
// the strips at their edges column by column. (A strip per lattice edge is
// most of a small lattice: 16 films of 256^2, in the kernel of all kinds, step in
// 38 us instead of 44.)
struct PairStore {
  bool own;       // the pair's first column belongs to the lattice (pairs: both)
  bool image;     // pairs: this lane's pair has an image
  bool pairs;     // (warp-uniform) even nx >= 8
  bool edge;      // (warp-uniform) columns with images, or beyond the lattice
  int nx;
  unsigned off;   // bytes from the row's start to the pair
  // pairs: bytes to its image. Else the stores beside the first column's, one
  // bit each: the second column, then + nx and - nx of each column. (One
  // register for both: with flags of their own the pairs' path lost 1 to 4 %,
  // formed at every store the other one 20 %.)
  unsigned alt;
  __device__ __forceinline__ PairStore(int x0, int lane, int nx_, int gx) {
    nx = nx_;
    const int ca = x0 - kMarchHalo + 2 * lane;
    const bool in = lane >= kMarchHalo / 2 && lane < 32 - kMarchHalo / 2;
    own = in && ca < nx;
    const bool own2 = in && ca + 1 < nx;
    pairs = nx % 2 == 0 && nx >= 8;
    edge = x0 < 4 || x0 + kMarchOut > nx - 4;
    image = own2 && (ca < 4 || ca >= nx - 4);
    off = (unsigned)(gx + ca) * 4u;
    alt = pairs ? (unsigned)(gx + (ca < 4 ? ca + nx : ca - nx)) * 4u
                : (own2 ? 1u : 0u) | (own && ca < 4 ? 2u : 0u) | (own2 && ca + 1 < 4 ? 4u : 0u) |
                      (own && ca >= nx - 4 ? 8u : 0u) | (own2 && ca + 1 >= nx - 4 ? 16u : 0u);
  }
  // the pair's second column belongs to the lattice
  __device__ __forceinline__ bool own2() const { return pairs ? own : (alt & 1u) != 0u; }
  __device__ __forceinline__ void pair(float* buf, long len, float* row, unsigned at, f2 v) const {
    *reinterpret_cast<float2*>(chk_global(
        buf, reinterpret_cast<float*>(reinterpret_cast<char*>(row) + at), len, 2)) = v.v;
  }
  __device__ __forceinline__ void fast(float* buf, long len, float* row, f2 v) const {
    if (own) pair(buf, len, row, off, v);
  }
  __device__ __forceinline__ void with_image(float* buf, long len, float* row, f2 v) const {
    if (own) pair(buf, len, row, off, v);
    if (image) pair(buf, len, row, alt, v);
  }
  __device__ __forceinline__ void slow(float* buf, long len, float* row, f2 v) const {
    float* p = reinterpret_cast<float*>(reinterpret_cast<char*>(row) + off);
    if (own) *chk_global(buf, p, len) = v.v.x;
    if (alt & 1u) *chk_global(buf, p + 1, len) = v.v.y;
    if (alt & 2u) *chk_global(buf, p + nx, len) = v.v.x;
    if (alt & 4u) *chk_global(buf, p + 1 + nx, len) = v.v.y;
    if (alt & 8u) *chk_global(buf, p - nx, len) = v.v.x;
    if (alt & 16u) *chk_global(buf, p + 1 - nx, len) = v.v.y;
  }
  // one store per plane, by the strip's kind
  // (row(k): its row's start, v(k): its values)
  template <int K, class Row, class Val>
  __device__ __forceinline__ void all(float* buf, long len, Row row, Val v) const {
    if (!edge) {
#pragma unroll
      for (int k = 0; k < K; ++k) fast(buf, len, row(k), v(k));
    } else if (pairs) {
#pragma unroll
      for (int k = 0; k < K; ++k) with_image(buf, len, row(k), v(k));
    } else {
#pragma unroll
      for (int k = 0; k < K; ++k) slow(buf, len, row(k), v(k));
    }
  }
  // a height that is not positive, or a force that is not finite, in the
  // lattice (see hlow and fall in march_unit)
  __device__ __forceinline__ bool bad(f2 hlow, f2 fall) const {
    return (own && (!(hlow.v.x > 0.f) || isnan(fall.v.x))) ||
           (own2() && (!(hlow.v.y > 0.f) || isnan(fall.v.y)));
  }
};

// The same with one column a lane: one 4-byte store, and the image that a
// column beside the lattice's edge has; below eight columns it can have two.
struct ColStore {
  bool own;
  bool edge;       // (warp-uniform) columns with images, or beyond the lattice
  bool left, right;  // the column has an image at + nx, at - nx
  int nx;
  unsigned off;    // bytes from the row's start to the column
  __device__ __forceinline__ ColStore(int x0, int lane, int nx_, int gx) {
    nx = nx_;
    const int c = x0 - kSoloHalo + lane;
    own = lane >= kSoloHalo && lane < kSoloCols - kSoloHalo && c < nx;
    edge = x0 < 4 || x0 + kSoloOut > nx - 4;
    left = own && c < 4;
    right = own && c >= nx - 4;
    off = (unsigned)(gx + c) * 4u;
  }
  template <int K, class Row, class Val>
  __device__ __forceinline__ void all(float* buf, long len, Row row, Val v) const {
    if (!edge) {
#pragma unroll
      for (int k = 0; k < K; ++k) {
        float* p = reinterpret_cast<float*>(reinterpret_cast<char*>(row(k)) + off);
        if (own) *chk_global(buf, p, len) = v(k).v;
      }
    } else {
#pragma unroll
      for (int k = 0; k < K; ++k) {
        float* p = reinterpret_cast<float*>(reinterpret_cast<char*>(row(k)) + off);
        if (own) *chk_global(buf, p, len) = v(k).v;
        if (left) *chk_global(buf, p + nx, len) = v(k).v;
        if (right) *chk_global(buf, p - nx, len) = v(k).v;
      }
    }
  }
  __device__ __forceinline__ bool bad(f1 hlow, f1 fall) const {
    return own && (!(hlow.v > 0.f) || isnan(fall.v));
  }
};
template <class T> struct StoreOf { using type = PairStore; };
template <> struct StoreOf<f1> { using type = ColStore; };

__device__ __forceinline__ f2 lower(f2 a, f2 b) {
  return mk2(fminf(a.v.x, b.v.x), fminf(a.v.y, b.v.y));
}
__device__ __forceinline__ f1 lower(f1 a, f1 b) { return {fminf(a.v, b.v)}; }

// The phase of the substrate at a pair of columns, in whole units of
// 1 / (nx ny), carried from row to row; height() gives substrate_at's values.
struct SubstratePhase {
  long col[2], row;
  __device__ SubstratePhase() {}
  __device__ SubstratePhase(const KParams& P, int x, int y) {
    const long nx = P.nx, ny = P.ny, nc = nx * ny;
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      long m = ((long)P.sub_kx * (x + c) % nx) * ny;
      if (m < 0) m += nc;
      (c ? col[1] : col[0]) = m;
    }
    row = ((long)P.sub_ky * y % ny) * nx;
    if (row < 0) row += nc;
  }
  __device__ float height(const KParams& P, int c) const {
    const long nc = (long)P.nx * P.ny;
    long m = col[c] + row;
    if (m >= nc) m -= nc;
    return substrate_height(P, m, nc);
  }
  __device__ __forceinline__ void heights(const KParams& P, f2& z) const {
    z = mk2(height(P, 0), height(P, 1));
  }
  __device__ __forceinline__ void heights(const KParams& P, f1& z) const { z.v = height(P, 0); }
  __device__ void next_row(const KParams& P) {
    const long nc = (long)P.nx * P.ny;
    row += (long)(P.sub_ky % P.ny) * P.nx;
    if (row >= nc) row -= nc;
    if (row < 0) row += nc;
  }
};

// Warps per SM that the registers must allow, in moment form without spills:
// three layers 12 (168 registers; 16 warps at 128 spill into the 15 KB of L1
// that the rings leave: 76 us a step against 29 at 1024^2; 8 warps: 97
// against 89 us at 2048^2), two layers 14 (the registers of 16), one layer 20,
// four and five 8. The other modes carry their options besides: 8 from three
// layers on.
__host__ __device__ constexpr int march_warps(int n, int mode) {
  return n == 1 ? 20 : (n == 2 ? 14 : (n == 3 && mode == kFast ? 12 : 8));
}

// The same with one column a lane (four and five layers; no spills).
__host__ __device__ constexpr int solo_warps(int n) { return n == 4 ? 16 : 12; }
template <class T>
__host__ __device__ constexpr int lane_warps(int n, int mode) {
  return MarchLane<T>::kPer == 2 ? march_warps(n, mode) : solo_warps(n);
}

// A batch instance's parameters, copied to the start of the warp's shared
// memory (kParBytes).
constexpr size_t kParBytes = (sizeof(KParams) + 127) / 128 * 128;
static_assert(sizeof(KParams) % 4 == 0, "parameters are copied as words");
__device__ __forceinline__ const KParams& stage_params(const BatchInst& b, unsigned char* sm) {
  int* dst = reinterpret_cast<int*>(sm);
  const int* src = reinterpret_cast<const int*>(&b.P);
  for (int w = threadIdx.x; w < (int)(sizeof(KParams) / 4); w += 32) *chk_smem(dst + w) = src[w];
  __syncwarp();
  return *reinterpret_cast<const KParams*>(sm);
}

// One unit of work: the output rows [ya, yb) of the strip that starts at
// column x0, by one warp. sm: MarchShape::kSmem bytes, 128-byte aligned.
// wait: the programmatic-launch wait for the previous grid (every global
// access comes after it).
// TWO: two rows a turn of the main loop. G: the parameters that hold the
// rest-population shifts H and Hsum (P itself, or see neg_pressures).
template <int N, int MODE, bool OP, bool TWO, class T>
__device__ __forceinline__ void march_unit(const KParams& P, const KParams& G,
                                           const CUtensorMap* map,
                                           float* __restrict__ fout, int x0, int ya, int yb,
                                           unsigned char* sm, int* __restrict__ status) {
  using S = MarchShape<N, MODE, OP, T>;
  using Lane = MarchLane<T>;
  constexpr bool TAU1 = S::TAU1, W32 = MODE == kFast, NN = MODE == kFast;
  constexpr int Q = 9, RS = S::RS, CW = Lane::kBox;
  constexpr int kRows = TWO ? 2 : 1;
  float* ring = reinterpret_cast<float*>(sm);
  float* park = reinterpret_cast<float*>(sm + S::kOffPark) + Lane::kPer * (threadIdx.x & 31);
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + S::kOffBar);
  const int lane = threadIdx.x & 31;
  const Layout& L = P.L;
  const int nx = P.nx, ny = P.ny;
  // collision rows: the output rows, and one more on each side when the
  // output gathers its populations from them
  const int cA = OP ? ya : ya - 1, cB = OP ? yb : yb + 1;
  const int r0 = cA - 2, nr = cB - cA + 4;  // input rows r0 .. r0 + nr - 1

  // this lane's place in a row of the ring: the copies start at the strip's first
  // column, with one column a lane rounded down to 16 bytes
  const int at = Lane::kPer * lane + (Lane::kPer == 2 ? 0 : (x0 + L.gx - Lane::kHalo) & 3);

  auto wrap_row = [&](int y) {
    y %= ny;
    return y < 0 ? y + ny : y;
  };
  auto issue = [&](int t) {  // lane 0
    uint64_t* b = bar + t % RS;
    const int xs = x0 + L.gx - Lane::kHalo, x = Lane::kPer == 2 ? xs : xs & ~3;
    const int y = wrap_row(r0 + t);
#ifdef MLSW_DEBUG
    // the copy must start on a 16-byte boundary inside the buffer (columns
    // beyond the row's end read as zeros); a bad one is not issued (the
    // barrier completes without data)
    if (x % 4 != 0 || x < 0 || x >= L.pitch || y < 0 || y >= L.rows) {
      note_bounds_violation();
      mbar_arrive_expect_tx(b, 0u);
      return;
    }
#endif
    mbar_arrive_expect_tx(b, (uint32_t)(S::BOX * 4));
    tma_load_3d(ring + (t % RS) * S::ROW, map, b, x, y, 0);
  };
  if (lane == 0) {
    for (int s = 0; s < RS; ++s) mbar_init(bar + s, 1);
    mbar_init_fence();
  }
  // Programmatic dependent launch: the next step's warps are scheduled as
  // this grid's exit, and wait here. They are not let in earlier (no
  // launch_dependents): warps that arrive while an SM still runs its share
  // crowd onto the SMs that finish first (three layers, 128^2: 8.2 us a step
  // with an early trigger, 5.2 without; 1024^2: 30.2 and 28.7). Nor after the
  // wait, when at most one grid is ahead: 128^2 5.30 against 5.00, two layers
  // of 64^2 4.07 against 3.97.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncwarp();
  int issued = RS < nr ? RS : nr;  // input rows whose copies were started
  if (lane == 0)
    for (int t = 0; t < issued; ++t) issue(t);
  // starts the copy of the next row, into the slot of the oldest one, which
  // every lane has read
  auto refill = [&]() {
    if (issued < nr) {
      __syncwarp();
      if (lane == 0) {
        fence_proxy_async_smem();
        issue(issued);
      }
      ++issued;
    }
  };

  const bool sub = MODE != kFast && P.sub_amp != 0.f;
  SubstratePhase sub_phase;
  if (sub) sub_phase = SubstratePhase(P, x0 - Lane::kHalo + Lane::kPer * lane, r0);
  const typename StoreOf<T>::type put(x0, lane, nx, L.gx);
  const T zero = Num<T>::splat(0.f);
  T zc[N], zB[N], pc[N], pB[N];  // previous row, and its difference to the row before
  T sc = zero, sB = zero;        // the same of the substrate
  T up1[N][3], up2[S::PARK ? 1 : N][3], mid[N][3];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    zc[i] = zB[i] = pc[i] = pB[i] = zero;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      up1[i][k] = mid[i][k] = zero;
      if constexpr (S::PARK)
        st_lane(park + (3 * i + k) * CW, zero);
      else
        up2[i][k] = zero;
    }
  }
  // smallest height so far; 0, or NaN once a force was not finite (0 * inf and
  // 0 * NaN are NaN): looked at once, at the end
  T hlow = Num<T>::splat(1.f), fall = zero;
  int slot = 0;  // of the next input row
  uint32_t parity = 0;

  // Row t arrives: its z; returns false when the bounded wait ran out.
  auto arrive = [&](int t, T (&zn)[N], T& sn) {
    if (!mbar_wait_bounded_warp(bar + slot, parity)) return false;
    const float* src = ring + slot * S::ROW + at;
    T z = zero;
    if (sub) {
      sub_phase.heights(P, sn);
      z = sn;
      sub_phase.next_row(P);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if constexpr (!TAU1) {
        T v[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) v[k] = ld_lane<T>(src + (i * Q + k) * CW);
        z = z + (v[0] + moving_sum(v));
      } else {
        z = z + (ld_lane<T>(src + 4 * i * CW) + ld_lane<T>(src + (4 * i + 1) * CW));
      }
      zn[i] = z;
    }
    if (++slot == RS) {
      slot = 0;
      parity ^= 1u;
    }
    return true;
  };
  // Pressures at the centre row (the previous z) from the new row's z.
  auto pressures = [&](const T (&zn)[N], T sn, T (&pn)[N]) {
    T gx[N], gy[N], lz[N], zd[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const T A = zn[i] - zc[i];
      lattice_derivatives<true>(zc[i], A, zB[i], gx[i], gy[i], lz[i]);
      zd[i] = zc[i];
    }
    if (sub) {
      T g0x, g0y, l0;
      lattice_derivatives<true>(sc, sn - sc, sB, g0x, g0y, l0);
      const T sg0 = fmav(0.5f, fmav(g0x, g0x, g0y * g0y), Num<T>::splat(1.f));
      neg_pressures<N, W32, T, NN>(P, G, zd, gx, gy, lz, pn, &sc, &sg0);
    } else {
      neg_pressures<N, W32, T, NN>(P, G, zd, gx, gy, lz, pn);
    }
  };
  auto roll_z = [&](const T (&zn)[N], T sn) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      zB[i] = zn[i] - zc[i];
      zc[i] = zn[i];
    }
    sB = sn - sc;
    sc = sn;
  };
  auto roll_p = [&](const T (&pn)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      pB[i] = pn[i] - pc[i];
      pc[i] = pn[i];
    }
  };

  // Collision of row r0 + t - 2, between the pressures of the two rows before
  // and pn, and the output it completes.
  auto collision = [&](int t, const T (&pn)[N]) {
    const int tc = t - 2, y = r0 + tc;
    T g0[N], sm_[N], jx[N], jy[N], hh[N], ih[N], ux[N], uy[N], Rx[N], Ry[N];
    const int cslot = tc % RS;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if constexpr (!TAU1) {
        const float* src = ring + cslot * S::ROW + i * Q * CW + at;
        T v[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) v[k] = ld_lane<T>(src + k * CW);
        const Moments<T> m = moments_of(v);
        g0[i] = m.g0;
        sm_[i] = m.s;
        jx[i] = m.jx;
        jy[i] = m.jy;
      } else {
        const float* src = ring + cslot * S::ROW + 4 * i * CW + at;
        g0[i] = ld_lane<T>(src);
        sm_[i] = ld_lane<T>(src + CW);
        jx[i] = ld_lane<T>(src + 2 * CW);
        jy[i] = ld_lane<T>(src + 3 * CW);
      }
      hh[i] = (g0[i] + sm_[i]) + G.H[i];
      ih[i] = rcp(hh[i]);
      ux[i] = jx[i] * ih[i];
      uy[i] = jy[i] * ih[i];
    }
    friction<N, true>(P, hh, ih, ux, uy, Rx, Ry);
    // rows of the output
    float* rowp[3];
    float* mrow = nullptr;
    const bool write = OP || t >= 6;
    if constexpr (OP) {
#pragma unroll
      for (int d = 0; d < 3; ++d)
        rowp[d] = fout + (long)wrap_row(y + d - 1) * L.pitch;
    } else {
      mrow = fout + (long)(y - 1) * L.pitch;
    }
    Moments<T> om[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      T gqx, gqy, none;
      lattice_derivatives<false>(pc[i], pn[i] - pc[i], pB[i], gqx, gqy, none);
      const T Fx = fmav(hh[i], gqx, Rx[i]), Fy = fmav(hh[i], gqy, Ry[i]);
      hlow = lower(hlow, hh[i]);
      fall = fmav(Fx + Fy, 0.f, fall);
      T fo[Q], fs[Q];
      if constexpr (!TAU1) {
        const float* src = ring + cslot * S::ROW + i * Q * CW + at;
#pragma unroll
        for (int k = 0; k < Q; ++k) fo[k] = ld_lane<T>(src + k * CW);
      }
      collide_d2q9<TAU1>(P, g0[i], sm_[i], jx[i], jy[i], ux[i], uy[i], Fx, Fy, fo, fs);
      // streaming along x: the pair takes what arrives at its columns
      T v[Q];
      v[0] = fs[0];
      v[3] = fs[3];
      v[7] = fs[7];
#pragma unroll
      for (int k = 1; k < Q; ++k) {
        if (Lattice<2>::cx(k) > 0)
          v[k] = from_left(fs[k]);
        else if (Lattice<2>::cx(k) < 0)
          v[k] = from_right(fs[k]);
      }
      if constexpr (OP) {
        put.all<Q>(
            fout, (long)Q * N * L.plane,
            [&](int k) { return rowp[Lattice<2>::cy(k) + 1] + (long)(i * Q + k) * L.plane; },
            [&](int k) { return v[k]; });
      } else {
        T below[3];  // moving up, from the row below the output row
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if constexpr (S::PARK)
            below[k] = ld_lane<T>(park + (3 * i + k) * CW);
          else
            below[k] = up2[i][k];
        }
        const T w[Q] = {mid[i][0], mid[i][1], below[0], below[1], below[2],
                         mid[i][2], v[6],      v[7],     v[8]};
        om[i] = moments_of(w);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if constexpr (S::PARK)
            st_lane(park + (3 * i + k) * CW, up1[i][k]);
          else
            up2[i][k] = up1[i][k];
          up1[i][k] = v[2 + k];
        }
        mid[i][0] = v[0];
        mid[i][1] = v[1];
        mid[i][2] = v[5];
      }
    }
    if constexpr (!OP) {
      if (write) {
        put.all<kMomPlanes * N>(
            fout, (long)kMomPlanes * N * L.plane, [&](int k) { return mrow + k * L.plane; },
            [&](int k) {
              const Moments<T>& q = om[k / kMomPlanes];
              return k % kMomPlanes == 0 ? q.g0
                                         : (k % kMomPlanes == 1 ? q.s
                                                                : (k % kMomPlanes == 2 ? q.jx : q.jy));
            });
      }
    }
  };

  bool ok = true;
  int t = 0;
  if constexpr (MODE == kFast && !OP) {
    // the steps of a long call: the warm-up rows apart, so that a full row is
    // one block of straight-line code, two rows at a time (the carried rows
    // then change names instead of moving; 31.2 -> 30.3 us a step at 1024^2)
#pragma unroll 1
    for (; t < 4; ++t) {
      T zn[N], pn[N], sn = zero;
      ok = arrive(t, zn, sn);
      if (!ok) break;
      if (t >= 2) {
        refill();  // row t - 2 gave its z and is not collided
        pressures(zn, sn, pn);
        roll_p(pn);
      }
      roll_z(zn, sn);
    }
#pragma unroll kRows
    for (; t < nr && ok; ++t) {
      T zn[N], pn[N], sn = zero;
      ok = arrive(t, zn, sn);
      if (!ok) break;
      pressures(zn, sn, pn);
      roll_z(zn, sn);
      collision(t, pn);
      roll_p(pn);
      refill();
    }
  } else {
#pragma unroll 1
    for (; t < nr; ++t) {
      T zn[N], pn[N], sn = zero;
      ok = arrive(t, zn, sn);
      if (!ok) break;
      if (t >= 2) {
        pressures(zn, sn, pn);
        if (t >= 4) collision(t, pn);
        roll_p(pn);
        refill();  // row t - 2 is used up
      }
      roll_z(zn, sn);
    }
  }
  if (!ok) {
    // a bounded wait ran out: report, and let this warp's copies land
    if (lane == 0) atomicOr(status, kStatusTimeout);
    for (; t < issued; ++t) {
      mbar_wait_bounded(bar + slot, parity, 1u << 16);
      if (++slot == RS) {
        slot = 0;
        parity ^= 1u;
      }
    }
  }
  const bool bad = put.bad(hlow, fall);
  if (bad) atomicOr(status, kStatusNonfinite);
}

}  // namespace mlsw
