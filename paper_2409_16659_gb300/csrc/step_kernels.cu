// step_kernels.cu -- the fused multilayer shallow-water LBM time step of one
// lattice. One launch = one time step over the whole periodic lattice, in
// one pass over its state:
//   * moments: h_i = H_i + g_0 + sum of the moving populations (rest
//     population stored shifted by H_i, see physics.cuh), J_i -- section LBM;
//   * interfaces z_i, their lattice gradient and Laplacian, and the layer
//     pressures p_i (Eqs. Laplace_pressure, disjoining_pressure, p_i =
//     sum_{j>=i} (Lambda_j + Pi_j));
//   * grad p_i, friction (Eq. friction_force), force (Eq. force), equilibrium
//     (Eq. equilibrium_distribution), BGK with forcing (Eq. BGK) and
//     streaming into the other buffer, including the periodic ghost columns
//     the next step reads.
//
// Discrete derivatives are the isotropic lattice stencils, written as sums
// of differences so a constant field gives exactly zero:
//   grad phi = (1/c_s^2) sum_k w_k c_k (phi(x + c_k) - phi(x))
//   lap  phi = (2/c_s^2) sum_k w_k (phi(x + c_k) - phi(x)).
//
// D2Q9: one warp per unit of work, marching down a strip of 64 columns
// (march.cuh, step_d2q9.cu). D1Q3 (small 1-D lattices): plain kernels, here.

#include "kernels.h"
#include "physics.cuh"
#include "step_common.cuh"

namespace mlsw {

// ---------------------------------------------------------------------------
// D1Q3 cell arithmetic shared by the tiled and the persistent kernels, so
// both give the same bits.
// ---------------------------------------------------------------------------
// q_i = p_atm - p_i of one cell from z deviations at x - 1, x, x + 1
// z0w, z0c, z0e: the substrate at x - 1, x, x + 1 (all 0 when flat).
// FORM: kFull32 exponents (3, 2) and a coefficient on every pair that has a
// part, kAny32 exponents (3, 2), kAny any potential; chosen by the host. The
// selects of the second form cost 2 to 4 % from two layers on (us a step, 512
// cells, two layers 0.635 and 0.662; 420 cells, four 1.525 and 1.585); one layer
// takes the second form always (500 cells, 0.407, without its selects 0.495).
enum D1Form { kFull32, kAny32, kAny };
template <int N, int FORM>
__device__ __forceinline__ void d1q3_pressures(const KParams& P, const float (&zw)[N],
                                               const float (&zc)[N], const float (&ze)[N],
                                               float (&p)[N], float z0w = 0.f, float z0c = 0.f,
                                               float z0e = 0.f) {
  constexpr bool W32 = FORM != kAny, SKIP = FORM != kFull32;
  float zd[N], gxz[N], gyz[N], lz[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float e = ze[i] - zc[i], wv = zw[i] - zc[i];
    zd[i] = zc[i];
    gxz[i] = 0.5f * (e - wv);  // (1/cs^2) w_1 = 1/2
    gyz[i] = 0.f;
    lz[i] = e + wv;            // (2/cs^2) w_1 = 1
  }
  if (P.sub_amp != 0.f) {
    const float g0 = 0.5f * (z0e - z0w);
    const float sg0 = fmaf(0.5f, g0 * g0, 1.f);
    neg_pressures<N, W32, float, false, SKIP>(P, P, zd, gxz, gyz, lz, p, &z0c, &sg0);
  } else {
    neg_pressures<N, W32, float, false, SKIP>(P, P, zd, gxz, gyz, lz, p);
  }
}

// Force, collision with forcing, for one cell: fs[i][k] receives the
// post-collision populations; f_old is read only when !TAU1. hlow: the smallest
// height so far; fall: 0, or NaN once a force was not finite (0 * inf and 0 * NaN
// are NaN; a flux that is not finite makes the force so). Both are looked at once,
// at the end.
template <int N, bool TAU1>
__device__ __forceinline__ void d1q3_collide_cell(const KParams& P, const float (&g0)[N],
                                                  const float (&sm)[N],
                                                  const float (&hh)[N], const float (&jx)[N],
                                                  const float (&pw)[N], const float (&pc)[N],
                                                  const float (&pe)[N], const float (&f_old)[N][3],
                                                  float (&fs)[N][3], float& hlow, float& fall) {
  float ih[N], ux[N], Rx[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    ih[i] = rcp(hh[i]);
    ux[i] = mulr(jx[i], ih[i]);
  }
  friction<N, false>(P, hh, ih, ux, ux, Rx, Rx);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float gqx = 0.5f * ((pe[i] - pc[i]) - (pw[i] - pc[i]));
    const float h = hh[i];
    const float Fx = fmav(h, gqx, Rx[i]);
    hlow = fminf(hlow, h);
    fall = fmaf(Fx, 0.f, fall);
    collide_d1q3<TAU1>(P, g0[i], sm[i], jx[i], ux[i], Fx, f_old[i], fs[i]);
  }
}
__device__ __forceinline__ bool d1q3_bad(float hlow, float fall) {
  return !(hlow > 0.f) || isnan(fall);
}

// ---------------------------------------------------------------------------
// D1Q3: tile of TX cells, one cell per thread, plain loads (the padded
// layout supplies the periodic images in x).
// ---------------------------------------------------------------------------
template <int N, int TX, bool TAU1, int FORM>
__global__ void __launch_bounds__(TX)
    step_d1q3_kernel(const float* __restrict__ fin, float* __restrict__ fout, const KParams P,
                     int* __restrict__ status) {
  constexpr int Q = 3;
  constexpr int RW = TX + 4, PW = TX + 2;
  __shared__ float zs[N][RW];  // interface-height deviations, see D2Q9
  __shared__ float ps[N][PW];
  const Layout& L = P.L;
  const int nx = P.nx;
  const int x0 = blockIdx.x * TX, tx = threadIdx.x;

  const bool sub = P.sub_amp != 0.f;
  float hh[N], g0[N], sm[N], jx[N];
  {
    float z = sub ? substrate_at(P, x0 + tx, 0) : 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float f0 = __ldg(fin + L.at(i * Q + 0, x0 + tx, 0));
      const float f1 = __ldg(fin + L.at(i * Q + 1, x0 + tx, 0));
      const float f2 = __ldg(fin + L.at(i * Q + 2, x0 + tx, 0));
      const float s = f0 + (f1 + f2);
      g0[i] = f0;
      sm[i] = f1 + f2;
      hh[i] = P.H[i] + s;
      jx[i] = f1 - f2;
      z += s;
      zs[i][tx + 2] = z;
    }
  }
  if (tx < 4) {
    const int rc = tx < 2 ? tx : RW - 4 + tx;  // columns x0 - 2, x0 - 1, x0 + TX, x0 + TX + 1
    const int x = x0 - 2 + rc;
    float z = sub ? substrate_at(P, x, 0) : 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float f0 = __ldg(fin + L.at(i * Q + 0, x, 0));
      const float f1 = __ldg(fin + L.at(i * Q + 1, x, 0));
      const float f2 = __ldg(fin + L.at(i * Q + 2, x, 0));
      z += f0 + (f1 + f2);
      zs[i][chk_index(rc, RW)] = z;
    }
  }
  __syncthreads();
  for (int pc = tx; pc < PW; pc += TX) {
    const int rc = pc + 1;
    float zw[N], zc[N], ze[N], p[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      zw[i] = zs[i][chk_index(rc - 1, RW)];
      zc[i] = zs[i][chk_index(rc, RW)];
      ze[i] = zs[i][chk_index(rc + 1, RW)];
    }
    if (sub) {
      const int x = x0 - 1 + pc;
      d1q3_pressures<N, FORM>(P, zw, zc, ze, p, substrate_at(P, x - 1, 0), substrate_at(P, x, 0),
                             substrate_at(P, x + 1, 0));
    } else {
      d1q3_pressures<N, FORM>(P, zw, zc, ze, p);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) ps[i][chk_index(pc, PW)] = p[i];
  }
  __syncthreads();
  const int gx = x0 + tx;
  if (gx >= nx) return;
  float pw[N], pc[N], pe[N], fo[N][Q], fs[N][Q];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    pw[i] = ps[i][tx];
    pc[i] = ps[i][tx + 1];
    pe[i] = ps[i][tx + 2];
#pragma unroll
    for (int k = 0; k < Q; ++k) fo[i][k] = TAU1 ? 0.f : fin[L.at(i * Q + k, gx, 0)];
  }
  float hlow = 1.f, fall = 0.f;
  d1q3_collide_cell<N, TAU1>(P, g0, sm, hh, jx, pw, pc, pe, fo, fs, hlow, fall);
  int dxs[3], xis[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    int dx = gx + c - 1;
    dx += (dx < 0) ? nx : 0;
    dx -= (dx >= nx) ? nx : 0;
    dxs[c] = dx;
    xis[c] = P.tiny ? kNoImage : image_of(dx, nx);  // tiny lattices refresh ghosts apart
  }
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const int cxi = Lattice<1>::cx(k) + 1;
      store_edge(fout + (long)(i * Q + k) * L.plane, L, dxs[cxi], 0, xis[cxi], kNoImage,
                 fs[i][k]);
    }
  if (d1q3_bad(hlow, fall)) atomicOr(status, kStatusNonfinite);
}

// ---------------------------------------------------------------------------
// D1Q3, persistent: one CTA holds the whole lattice in shared memory and
// runs nsteps steps in one launch. A warp takes 32 neighbouring cells at a
// time and writes the inner 26: z, the pressures and the streamed populations
// pass between cells by shuffles, the three cells on each side are computed
// again by the neighbours, and a step needs one barrier instead of three
// (512 cells, two layers: 0.88 -> 0.67 us a step; it is bound by the issue of
// 20 warps on one SM). Shared memory (floats): two population
// buffers [3N][nx], the substrate [nx]. The lattice is read from fin and the
// final state written to fout (which may be fin), ghost images included.
// Same cell arithmetic as step_d1q3_kernel.
// ---------------------------------------------------------------------------
constexpr int kD1Out = 26;  // cells a warp writes
// threads: 20 warps cover 520 cells at once; more layers need the registers
constexpr int d1_threads(int n) { return n <= 3 ? 640 : 512; }

template <int N, bool TAU1, int FORM>
__global__ void __launch_bounds__(d1_threads(N), 1)
    step_d1q3_persistent(const float* fin, float* fout, const KParams P, int nsteps,
                         int* __restrict__ status) {
  constexpr int Q = 3;
  constexpr unsigned kAll = 0xffffffffu;
  extern __shared__ __align__(16) float sm[];
  const Layout& L = P.L;
  const int nx = P.nx, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  float* fa = sm;                     // current populations [i * Q + k][x]
  float* fb = fa + 3 * N * nx;        // next populations
  float* z0s = fb + 3 * N * nx;       // [x]
  for (int t = tid; t < Q * N * nx; t += nt) {
    const int pl = t / nx, x = t - pl * nx;
    *chk_smem(fa + t) = fin[L.at(pl, x, 0)];
  }
  const bool sub = P.sub_amp != 0.f;
  if (sub)
    for (int x = tid; x < nx; x += nt) *chk_smem(z0s + x) = substrate_at(P, x, 0);
  __syncthreads();
  float hlow = 1.f, fall = 0.f;
  const bool inner = lane >= 3 && lane < 3 + kD1Out;
  // the warp's first cells, and this lane's one wrapped (kept for one and two
  // layers, whose steps it shortens; three and five layers lose 5 and 10 % to the
  // register)
  const int first = (tid >> 5) * kD1Out;
  int x_first = (first - 3 + lane) % nx;
  if (x_first < 0) x_first += nx;
  for (int s = 0; s < nsteps; ++s) {
    for (int c0 = first; c0 < nx; c0 += (nt >> 5) * kD1Out) {
      const int xo = c0 - 3 + lane;  // this lane's cell before wrapping
      int x = xo;
      if constexpr (N <= 2) {
        x = x_first + (c0 - first);  // below 2 nx
        if (x >= nx) x -= nx;
      } else if (x < 0 || x >= nx) {
        x %= nx;
        x += x < 0 ? nx : 0;
      }
      const float z0 = sub ? *chk_smem(z0s + x) : 0.f;
      float g0[N], sm_[N], hh[N], jx[N], fo[N][Q], fs[N][Q];
      float zw[N], zc[N], ze[N], pw[N], pc[N], pe[N];
      float z = z0;
#pragma unroll
      for (int i = 0; i < N; ++i) {
#pragma unroll
        for (int k = 0; k < Q; ++k) fo[i][k] = *chk_smem(fa + (i * Q + k) * nx + x);
        g0[i] = fo[i][0];
        sm_[i] = fo[i][1] + fo[i][2];
        const float sum = fo[i][0] + (fo[i][1] + fo[i][2]);
        hh[i] = P.H[i] + sum;
        jx[i] = fo[i][1] - fo[i][2];
        z += sum;
        zc[i] = z;
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        zw[i] = __shfl_up_sync(kAll, zc[i], 1);
        ze[i] = __shfl_down_sync(kAll, zc[i], 1);
      }
      if (sub) {
        const float z0w = __shfl_up_sync(kAll, z0, 1), z0e = __shfl_down_sync(kAll, z0, 1);
        d1q3_pressures<N, FORM>(P, zw, zc, ze, pc, z0w, z0, z0e);
      } else {
        d1q3_pressures<N, FORM>(P, zw, zc, ze, pc);
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        pw[i] = __shfl_up_sync(kAll, pc[i], 1);
        pe[i] = __shfl_down_sync(kAll, pc[i], 1);
      }
      d1q3_collide_cell<N, TAU1>(P, g0, sm_, hh, jx, pw, pc, pe, fo, fs, hlow, fall);
      const bool own = inner && xo < nx;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const float right = __shfl_up_sync(kAll, fs[i][1], 1);   // c = +1, from x - 1
        const float left = __shfl_down_sync(kAll, fs[i][2], 1);  // c = -1, from x + 1
        if (own) {
          *chk_smem(fb + (i * Q + 0) * nx + x) = fs[i][0];
          *chk_smem(fb + (i * Q + 1) * nx + x) = right;
          *chk_smem(fb + (i * Q + 2) * nx + x) = left;
        }
      }
    }
    __syncthreads();
    float* t = fa;
    fa = fb;
    fb = t;
  }
  // final state, real cells and the ghost images x in [-2, nx + 2)
  for (int t = tid; t < Q * N * (nx + 4); t += nt) {
    const int pl = t / (nx + 4), x = t - pl * (nx + 4) - 2;
    int sx = x % nx;
    sx += sx < 0 ? nx : 0;
    fout[L.at(pl, x, 0)] = *chk_smem(fa + pl * nx + sx);
  }
  // (the outer lanes' neighbours are not the lattice's; beyond nx it repeats)
  if (inner && d1q3_bad(hlow, fall)) atomicOr(status, kStatusNonfinite);
}

// ---------------------------------------------------------------------------
// dispatch
// ---------------------------------------------------------------------------
constexpr int kD1TX = 128;

int step_mode(const KParams& P) {
  // the general kernel also takes the lattices whose ghosts need a pass of
  // their own after every step
  if (P.omega != 1.f || P.tiny) return kGeneral;
  const bool w32 = (P.wet_kind == 0 && P.nw == 3 && P.mw == 2);
  return (w32 && !P.far_pairs && P.sub_amp == 0.f) ? kFast : kTau1;
}

bool step_dear(const KParams& P) {
  return step_mode(P) == kGeneral || P.far_pairs || P.sub_amp != 0.f || P.wet_kind != 0;
}

bool step_moments(const KParams& P) { return step_mode(P) != kGeneral; }

static D1Form d1_form(const KParams& P) {
  if (P.wet_kind != 0 || P.nw != 3 || P.mw != 2) return kAny;
  return P.zero_pairs || P.n == 1 ? kAny32 : kFull32;
}

// (tau != 1 runs the general form only)
template <int N>
static cudaError_t launch_n(const StepLaunch& a, cudaStream_t st) {
  if (a.lattice == 2) {
    return launch_step_d2q9<N>(a, st);
  }
  auto kern = step_d1q3_kernel<N, kD1TX, false, kAny>;
  if (a.P.omega == 1.f) {
    switch (d1_form(a.P)) {
      case kFull32: kern = step_d1q3_kernel<N, kD1TX, true, kFull32>; break;
      case kAny32: kern = step_d1q3_kernel<N, kD1TX, true, kAny32>; break;
      default: kern = step_d1q3_kernel<N, kD1TX, true, kAny>; break;
    }
  }
  kern<<<(a.P.nx + kD1TX - 1) / kD1TX, kD1TX, 0, st>>>(a.fin, a.fout, a.P, a.status);
  return cudaGetLastError();
}

size_t step_persistent_smem(int n, int lattice, int nx) {
  if (lattice != 1 || n < 1 || n > kMaxLayers || nx < 1) return 0;
  return (size_t)8 * n * nx * sizeof(float);
}

template <int N, bool TAU1, int FORM>
static cudaError_t launch_d1p(const StepLaunch& a, int nsteps, cudaStream_t st) {
  auto kern = step_d1q3_persistent<N, TAU1, FORM>;
  const size_t smem = step_persistent_smem(N, 1, a.P.nx);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int warps = (a.P.nx + kD1Out - 1) / kD1Out;
  const int threads = 32 * warps < d1_threads(N) ? 32 * warps : d1_threads(N);
  kern<<<1, threads, smem, st>>>(a.fin, a.fout, a.P, nsteps, a.status);
  return cudaGetLastError();
}

template <int N>
static cudaError_t launch_d1p_n(const StepLaunch& a, int nsteps, cudaStream_t st) {
  if (a.P.omega != 1.f) return launch_d1p<N, false, kAny>(a, nsteps, st);
  switch (d1_form(a.P)) {
    case kFull32: return launch_d1p<N, true, kFull32>(a, nsteps, st);
    case kAny32: return launch_d1p<N, true, kAny32>(a, nsteps, st);
    default: return launch_d1p<N, true, kAny>(a, nsteps, st);
  }
}

cudaError_t launch_batch_alike(const BatchLaunch& a, int n, int mode, cudaStream_t st) {
  switch (n) {
    case 1: return launch_alike_d2q9<1>(a, mode, st);
    case 2: return launch_alike_d2q9<2>(a, mode, st);
    case 3: return launch_alike_d2q9<3>(a, mode, st);
    case 4: return launch_alike_d2q9<4>(a, mode, st);
    case 5: return launch_alike_d2q9<5>(a, mode, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_step_persistent(const StepLaunch& a, int nsteps, cudaStream_t st) {
  switch (a.P.n) {
    case 1: return launch_d1p_n<1>(a, nsteps, st);
    case 2: return launch_d1p_n<2>(a, nsteps, st);
    case 3: return launch_d1p_n<3>(a, nsteps, st);
    case 4: return launch_d1p_n<4>(a, nsteps, st);
    case 5: return launch_d1p_n<5>(a, nsteps, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_step(const StepLaunch& a, cudaStream_t st) {
  switch (a.P.n) {
    case 1: return launch_n<1>(a, st);
    case 2: return launch_n<2>(a, st);
    case 3: return launch_n<3>(a, st);
    case 4: return launch_n<4>(a, st);
    case 5: return launch_n<5>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

int step_d1q3_cols() { return kD1TX; }

MLSW_DEFINE_BOUNDS_READER(bounds_violations_step)

}  // namespace mlsw
