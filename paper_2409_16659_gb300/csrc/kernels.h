// kernels.h -- internal launch interface between the host library
// (mlswlbm.cu, noalloc.cu) and the kernel translation units. Not part of
// the C ABI.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "physics.cuh"

namespace mlsw {

// status word bits (device int OR-ed by the kernels)
constexpr int kStatusNonfinite = 1;  // h <= 0 or a non-finite value
constexpr int kStatusTimeout = 2;    // a bounded mbarrier wait ran out

// D2Q9 step: a warp marches down a strip of kMarchCols columns, of which the
// kMarchHalo on each side only feed the stencils (march.cuh).
constexpr int kMarchCols = 64, kMarchHalo = 4, kMarchOut = kMarchCols - 2 * kMarchHalo;
// With one column a lane (march_solo) the strip has 32 columns, and a row's
// copy 36, from the 16-byte boundary at or before the strip's first column.
constexpr int kSoloCols = 32, kSoloHalo = 3, kSoloOut = kSoloCols - 2 * kSoloHalo, kSoloBox = 36;
inline int march_strips(int nx, bool solo) {
  const int out = solo ? kSoloOut : kMarchOut;
  return (nx + out - 1) / out;
}
inline int march_box(bool solo) { return solo ? kSoloBox : kMarchCols; }
// A D2Q9 state with tau = 1 is stored as moments: plane 4 i + q holds g_0, s,
// J_x, J_y (q = 0..3) of layer i; another tau (and a lattice whose ghosts need
// a pass of their own) as populations, plane 9 i + k. Both in the layout of
// KParams::L.
constexpr int kMomPlanes = 4;

// Kernel modes of the D2Q9 step: the general step for tau != 1 and for
// tau = 1, and a fast step for the case the paper runs (tau = 1, wetting
// exponents (3, 2), spreading coefficients only between neighbouring
// interfaces).
enum StepMode { kGeneral = 0, kTau1 = 1, kFast = 2 };

// Per-layer rest-population shift (see KParams).
struct KShift {
  float H[kMaxLayers];
};

// One fused time step fin -> fout (distinct buffers, layout P.L).
struct StepLaunch {
  int lattice;                  // 1 = D1Q3, 2 = D2Q9
  const float* fin;
  float* fout;
  const CUtensorMap* fin_map;   // D2Q9: row map of fin (see mlsw_host::make_row_map)
  KParams P;
  int solo;                     // D2Q9: one column a lane (fin_map then has that box)
  int to_populations;           // D2Q9, moments in: write the populations after the step
  int* status;
  int num_sms;
};
cudaError_t launch_step(const StepLaunch& a, cudaStream_t st);
// the D2Q9 step of n = N layers (step_d2q9.cu)
template <int N>
cudaError_t launch_step_d2q9(const StepLaunch& a, cudaStream_t st);
template <> cudaError_t launch_step_d2q9<1>(const StepLaunch& a, cudaStream_t st);
template <> cudaError_t launch_step_d2q9<2>(const StepLaunch& a, cudaStream_t st);
template <> cudaError_t launch_step_d2q9<3>(const StepLaunch& a, cudaStream_t st);
template <> cudaError_t launch_step_d2q9<4>(const StepLaunch& a, cudaStream_t st);
template <> cudaError_t launch_step_d2q9<5>(const StepLaunch& a, cudaStream_t st);
// Cells of a D1Q3 tile (the padded layout covers whole tiles).
int step_d1q3_cols();

// D1Q3 lattices small enough for one CTA's shared memory run many steps in
// one persistent launch: bytes of shared memory it needs (0: not possible
// for this lattice type), and the launch, which reads a.fin and leaves the
// state after nsteps steps in a.fout (ghost images included).
size_t step_persistent_smem(int n, int lattice, int nx);
cudaError_t launch_step_persistent(const StepLaunch& a, int nsteps, cudaStream_t st);

// ---------------------------------------------------------------------------
// Batches: many independent D2Q9 lattices stepped by one launch over one
// table of units, in which the units of instances that share n, kernel mode
// and nominal tile height form a contiguous range (batch_kernels.cu).
// ---------------------------------------------------------------------------
// Nominal tile heights (batch_rows in unit_rows.h): variant 0 = 16 rows (n <= 3
// only), the height of the model, variant 1 = 8 rows, for n <= 3 half of it.
constexpr int kBatchVariants = 2;
constexpr int batch_tile_rows(int variant) { return variant == 0 ? 16 : 8; }

// Device descriptor of one instance (aligned as its tensor maps require).
struct BatchInst {
  CUtensorMap map[2];  // row maps of the two buffers
  KParams P;
  float* f[2];  // buffers, moments or populations
  int kind;     // batch_kind
  int strips;   // strips of its columns
  int rows;     // rows of a unit
};

// Kernel mode of a parameter set.
int step_mode(const KParams& P);
// Whether a cell has many terms: tau != 1, far pairs, a substrate or the
// exponential potential.
bool step_dear(const KParams& P);
// Whether a D2Q9 state is stored as moments (else populations).
bool step_moments(const KParams& P);

// Kernel of an instance: layer count n (1..5) and kernel mode.
constexpr int kBatchKinds = 5 * 3;
__host__ __device__ constexpr int batch_kind(int n, int mode) { return (n - 1) * 3 + mode; }

// One batch step, buffers cur -> cur ^ 1, of every instance in a table of
// (instance, unit) entries, one warp each: one launch.
struct BatchLaunch {
  const BatchInst* inst;
  const int2* table;
  int nunits;
  unsigned kinds;  // bit k: instances of kind k are in the table
  int same_params; // the instances' parameters are P's but for H and Hsum
  KParams P;
  int cur;
  int* status;
};
// warps of a batch step resident on one SM
int batch_warps_per_sm(unsigned kinds);
// Whether the kernel for at most three layers takes a table of these kinds.
constexpr bool batch_small(unsigned kinds) {
  return kinds < 1u << batch_kind(4, 0) && !((kinds >> batch_kind(3, kGeneral)) & 1u);
}
// Whether instances of a kind march with one column a lane in a table of these
// kinds. Its ring is the launch's: with pairs, five layers in the general mode
// take 46 KB a warp and leave four warps an SM for every instance (32 lattices
// of 2 to 5 layers, all modes: 282 us a step with pairs, 226 with single columns).
constexpr bool batch_solo(unsigned kinds, int kind) {
  return kinds != 1u << kind && kind % 3 == kGeneral && kind / 3 + 1 >= 4;
}
cudaError_t launch_batch_step(const BatchLaunch& a, cudaStream_t st);
// all of one kind (step_d2q9.cu)
cudaError_t launch_batch_alike(const BatchLaunch& a, int n, int mode, cudaStream_t st);
template <int N>
cudaError_t launch_alike_d2q9(const BatchLaunch& a, int mode, cudaStream_t st);
template <> cudaError_t launch_alike_d2q9<1>(const BatchLaunch& a, int mode, cudaStream_t st);
template <> cudaError_t launch_alike_d2q9<2>(const BatchLaunch& a, int mode, cudaStream_t st);
template <> cudaError_t launch_alike_d2q9<3>(const BatchLaunch& a, int mode, cudaStream_t st);
template <> cudaError_t launch_alike_d2q9<4>(const BatchLaunch& a, int mode, cudaStream_t st);
template <> cudaError_t launch_alike_d2q9<5>(const BatchLaunch& a, int mode, cudaStream_t st);
// the kernel for at most NMAX layers (3: more warps fit an SM; 5)
template <int NMAX>
cudaError_t launch_batch_step_n(const BatchLaunch& a, cudaStream_t st);
template <> cudaError_t launch_batch_step_n<3>(const BatchLaunch& a, cudaStream_t st);
template <> cudaError_t launch_batch_step_n<5>(const BatchLaunch& a, cudaStream_t st);

// out[2 (j kMaxLayers + i) + {0, 1}] = real and imaginary part of
// sum_x h_i(x) exp(-2 pi i (kx[j] x / nx + ky[j] y / ny)) for every instance
// j < count and layer i (zero for i >= n_j); kx, ky device arrays.
cudaError_t launch_batch_modes(const BatchInst* inst, int count, int cur, const int* kx,
                               const int* ky, double* out, cudaStream_t st);

// Heights [n][ny][nx] of one instance (its host descriptor) from buffer cur.
cudaError_t launch_batch_heights(const BatchInst* inst_host, int cur, float* h, cudaStream_t st);

// Radially averaged power spectra of the layer heights (analysis.cu): the
// row and column FFT passes into work (n nx ny complex values), bin sums
// bins[n][nbins] and wavevector counts counts[nbins], both zeroed by the
// caller. Power-of-two sides up to kSpectrumMaxSide, 1 <= nbins <=
// kSpectrumMaxBins.
constexpr int kSpectrumMaxSide = 8192;
constexpr int kSpectrumMaxBins = 8192;
bool spectrum_supported(int nx, int ny, int nbins);
cudaError_t launch_spectrum(int Q, int n, const Layout& L, const float* f, int nbins,
                            float2* work, double* bins, unsigned long long* counts,
                            cudaStream_t st);

// Azimuthal averages of the interfaces around (cx, cy) (analysis.cu):
// sums[m][nbins] of z_m and counts[nbins] of cells per unit-width ring,
// both zeroed by the caller; z_0 the substrate of the given parameters.
struct ProfileParams {
  double cx, cy;
  int nbins;
  double sub_amp;
  int sub_kx, sub_ky;
};
cudaError_t launch_radial_profile(int Q, int n, const Layout& L, const float* f, const KShift& sh,
                                  const ProfileParams& A, double* sums,
                                  unsigned long long* counts, cudaStream_t st);

// The launches below take a state's planes per layer as Q: 9 (D2Q9) or 3
// (D1Q3) populations, or kMomPlanes for moments.

// f = f_eq(h, U = 0) on the real cells and their ghost images: rest
// population h - H_i, everything else 0; h dense [n][ny][nx]. status |=
// kStatusNonfinite where h <= 0 or h is not finite.
cudaError_t launch_init(int Q, int n, const Layout& L, const float* h, float* f, const KShift& sh,
                        int* status, cudaStream_t st);

// Periodic images: every ghost cell within four columns of the real domain
// copies its real cell, for all nplanes planes.
cudaError_t launch_fill_ghosts(int nplanes, const Layout& L, float* f, cudaStream_t st);

// Moments m (ghosts included) of D2Q9 populations f; the populations f (real
// cells) of a D2Q9 state at rest with moments m.
cudaError_t launch_moments(int n, const Layout& L, const float* f, float* m, cudaStream_t st);
cudaError_t launch_rest_populations(int n, const Layout& L, const float* m, float* f,
                                    cudaStream_t st);

// h dense [n][ny][nx] = H_i + sum_k g[i][k]
// With st_out (a device view of page-locked host memory), the first thread
// also copies the status word *st_in there, so that the host reads it after
// the synchronisation it needs anyway.
cudaError_t launch_heights(int Q, int n, const Layout& L, const float* f, const KShift& sh,
                           float* h, cudaStream_t st, const int* st_in = nullptr,
                           int* st_out = nullptr);

// real cells of the rest planes: f[i][0] += sign * H_i
cudaError_t launch_shift(int Q, int n, const Layout& L, float* f, const KShift& sh, float sign,
                         cudaStream_t st);

// out dense [n][ny][nx] = H_i + g[i][0], the true rest population
cudaError_t launch_rest_planes(int Q, int n, const Layout& L, const float* f, const KShift& sh,
                               float* out, cudaStream_t st);

// Two-pass deterministic reduction of per-layer mass, kinetic energy and
// min h over the real cells. partials: nblk * (n + 2) doubles; out: n + 2
// doubles (mass[0..n-1], kinetic, hmin).
cudaError_t launch_diagnostics(int Q, int n, const Layout& L, const float* f,
                               const KShift& sh, double* partials, int nblk, double* out,
                               cudaStream_t st);

// Free energy of Eq. (free_energy_n_layer) from dense heights [n][ny][nx],
// FP64, with the parameters in double precision. partials: nblk doubles.
struct FreeEnergyParams {
  int n, lattice, nx, ny;
  double gamma[kMaxLayers];
  double S[kMaxLayers][kMaxLayers];
  double hstar;
  int nw, mw;
  double sub_amp;  // substrate z_0 = sub_amp cos(2 pi (kx x / nx + ky y / ny))
  int sub_kx, sub_ky;
  int wet_kind;    // 0 power law (nw, mw), 1 exponential (kappa)
  double kappa;
  double c_phi;    // 1 / (nw - mw)
};
cudaError_t launch_free_energy(const FreeEnergyParams& E, const float* h, double* partials,
                               int nblk, double* out, cudaStream_t st);

// Friction of independent cells (layout [i][cell]); Jy / Ry may be null.
cudaError_t launch_friction_eval(const KParams& P, long ncell, const float* h, const float* Jx,
                                 const float* Jy, float* Rx, float* Ry, cudaStream_t st);

// One CTA waits on an mbarrier with the step kernels' bounded wait (limit
// iterations); the barrier gets its arrival only when arrive != 0. A wait
// that runs out ORs kStatusTimeout into *status.
cudaError_t launch_wait_selftest(int arrive, unsigned limit, int* status, cudaStream_t st);
// One warp's wait, whose lanes in short_lanes run out at once: *went_on the
// lanes that go on (all or none), kStatusTimeout when none does.
cudaError_t launch_warp_wait_selftest(unsigned short_lanes, unsigned limit, unsigned* went_on,
                                      int* status, cudaStream_t st);

// Dense layout of a caller-owned population array (no ghosts).
inline Layout dense_layout(int nx, int ny, int nplanes = 0) {
  Layout L;
  L.nx = nx;
  L.ny = ny;
  L.gx = 0;
  L.pitch = nx;
  L.rows = ny;
  L.plane = (long)nx * ny;
  L.nplanes = nplanes;
  return L;
}

// Bounds-checked build: accesses out of range since the last call, per
// translation unit with device code (0 in release builds; ~0u if the
// counter could not be read).
unsigned bounds_violations_step();
unsigned bounds_violations_aux();
unsigned bounds_violations_analysis();
unsigned bounds_violations_d2q9_1();
unsigned bounds_violations_d2q9_2();
unsigned bounds_violations_d2q9_3();
unsigned bounds_violations_d2q9_4();
unsigned bounds_violations_d2q9_5();
unsigned bounds_violations_batch_3();
unsigned bounds_violations_batch_5();

}  // namespace mlsw
