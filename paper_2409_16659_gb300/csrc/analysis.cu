// analysis.cu -- analysis of a solver's state on the device:
//   * radially averaged power spectra of the layer heights, the quantity the
//     paper's spinodal-dewetting section follows in time and compares with
//     the growth rates of its linear stability analysis;
//   * azimuthal averages of the interface heights around a drop or lens
//     centre, the profiles its droplet-equilibrium section fits circular
//     arcs to.
//
// Spectra.
// S_i(b) = mean of |H_i(k)|^2 over the integer wavevectors k = (kx, ky),
// kx in (-nx/2, nx/2] and likewise ky, with round(|k|) = b, where H_i is the
// unnormalised 2-D DFT of h_i with its mean removed (the k = 0 term is set
// to zero). Two passes of radix-2 FFTs in shared memory (power-of-two
// sides): rows, which also form the height deviations h_i - H_i from the
// stored populations, then columns, which bin |H|^2 in FP64.
#include <cstdint>

#include "kernels.h"
#include "physics.cuh"
#include "ring_plan.h"

namespace mlsw {

namespace {

__device__ __forceinline__ int bitrev(int v, int bits) {
  return bits == 0 ? 0 : (int)(__brev((unsigned)v) >> (32 - bits));
}

// Twiddles e^{-pi i j / half}, j < half: the last stage's, of which stage s
// uses every (half >> s)-th (j / 2^s is the same number). One table per CTA
// instead of a sine and cosine per butterfly.
__device__ void make_twiddles(float2* tw, int half) {
  for (int j = threadIdx.x; j < half; j += blockDim.x) {
    float sn, cs;
    sincospif(-(float)j / (float)half, &sn, &cs);  // exact quotient: half a power of two
    tw[j] = make_float2(cs, sn);
  }
}

// In-place radix-2 decimation-in-time FFT (forward, e^{-2 pi i j k / len}) of
// `count` contiguous arrays of length len = 2^bits, each loaded in
// bit-reversed order; leaves them in natural order. All threads of the CTA
// take part; starts with a barrier.
__device__ void fft_inplace(float2* a, const float2* tw, int bits, int count) {
  const int half = (1 << bits) >> 1;
  for (int s = 0; s < bits; ++s) {
    __syncthreads();
    const int m = 1 << s, lgstep = bits - 1 - s;
    for (int t = threadIdx.x; t < count * half; t += blockDim.x) {
      const int arr = t >> (bits - 1), u = t & (half - 1);
      const int j = u & (m - 1);
      const int i0 = (arr << bits) + ((u >> s) << (s + 1)) + j, i1 = i0 + m;
      const float2 w = tw[j << lgstep];
      const float cs = w.x, sn = w.y;
      const float2 b = a[i1], u0 = a[i0];
      const float2 wb = make_float2(b.x * cs - b.y * sn, b.x * sn + b.y * cs);
      a[i0] = make_float2(u0.x + wb.x, u0.y + wb.y);
      a[i1] = make_float2(u0.x - wb.x, u0.y - wb.y);
    }
  }
  __syncthreads();
}

// One CTA per (row y, layer i): the row of h_i - H_i (the sum of the stored
// planes, PL per layer of which the first Q add up to it), transformed.
template <int Q, int PL>
__global__ void __launch_bounds__(256)
    spectrum_rows_kernel(Layout L, const float* __restrict__ f, int bits_x,
                         float2* __restrict__ work) {
  extern __shared__ float2 row[];  // [nx], then the twiddles [nx / 2]
  const int nx = L.nx, ny = L.ny;
  const int y = blockIdx.x, i = blockIdx.y;
  const float* src = f + L.at(i * PL, 0, y);
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    float d = 0.f;
#pragma unroll
    for (int k = 0; k < Q; ++k) d += src[(long)k * L.plane + x];
    row[bitrev(x, bits_x)] = make_float2(d, 0.f);
  }
  make_twiddles(row + nx, nx / 2);
  fft_inplace(row, row + nx, bits_x, 1);
  float2* dst = work + ((long)i * ny + y) * nx;
  for (int x = threadIdx.x; x < nx; x += blockDim.x) dst[x] = row[x];
}

// round(sqrt(q)) of an integer 0 <= q <= 2 * 4096^2, exactly: the FP32 root
// rounded, corrected by (2 b - 1)^2 <= 4 q < (2 b + 1)^2 (no integer is
// halfway). An FP64 root per wavevector took half of the column pass.
__device__ __forceinline__ int rounded_root(long q) {
  int b = (int)rintf(sqrtf((float)q));
  if (4 * q >= (long)(2 * b + 1) * (2 * b + 1)) ++b;
  if (b > 0 && 4 * q < (long)(2 * b - 1) * (2 * b - 1)) --b;
  return b;
}

// One CTA per (cb columns, layer i): the column transforms, then |H|^2 into
// the radial bins (FP64 sums in shared memory, then global atomics). Layer 0
// also counts the wavevectors per bin.
__global__ void __launch_bounds__(256)
    spectrum_cols_kernel(int nx, int ny, int bits_y, int cb, const float2* __restrict__ work,
                         int nbins, double* __restrict__ bins,
                         unsigned long long* __restrict__ counts) {
  extern __shared__ unsigned char sm[];
  float2* col = reinterpret_cast<float2*>(sm);                      // [cb][ny]
  float2* tw = col + (size_t)cb * ny;                               // [max(1, ny / 2)]
  double* sb = reinterpret_cast<double*>(tw + (ny > 1 ? ny / 2 : 1));  // [nbins]
  unsigned* sc = reinterpret_cast<unsigned*>(sb + nbins);           // [nbins]
  const int c0 = blockIdx.x * cb, i = blockIdx.y;
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
    sb[b] = 0.0;
    sc[b] = 0u;
  }
  const float2* src = work + (long)i * ny * nx;
  for (int e = threadIdx.x; e < cb * ny; e += blockDim.x) {
    const int y = e / cb, c = e - y * cb;  // neighbouring threads read neighbouring columns
    col[c * ny + bitrev(y, bits_y)] = src[(long)y * nx + c0 + c];
  }
  make_twiddles(tw, ny / 2);
  fft_inplace(col, tw, bits_y, cb);
  for (int e = threadIdx.x; e < cb * ny; e += blockDim.x) {
    const int c = e >> bits_y, yy = e & (ny - 1);
    const int kxi = c0 + c;
    const int kx = kxi <= nx / 2 ? kxi : kxi - nx, ky = yy <= ny / 2 ? yy : yy - ny;
    const int b = rounded_root((long)kx * kx + (long)ky * ky);
    if (b < nbins) {
      const float2 v = col[e];
      const double p = (kx == 0 && ky == 0) ? 0.0 : (double)v.x * v.x + (double)v.y * v.y;
      atomicAdd(sb + b, p);
      if (i == 0) atomicAdd(sc + b, 1u);
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
    if (sb[b] != 0.0) atomicAdd(bins + (long)i * nbins + b, sb[b]);
    if (i == 0 && sc[b] != 0u) atomicAdd(counts + b, (unsigned long long)sc[b]);
  }
}

int log2_exact(int v) {
  if (v < 1 || (v & (v - 1)) != 0) return -1;
  int b = 0;
  while ((1 << b) < v) ++b;
  return b;
}

}  // namespace

bool spectrum_supported(int nx, int ny, int nbins) {
  return log2_exact(nx) >= 0 && log2_exact(ny) >= 0 && nx <= kSpectrumMaxSide &&
         ny <= kSpectrumMaxSide && nbins >= 1 && nbins <= kSpectrumMaxBins;
}

cudaError_t launch_spectrum(int Q, int n, const Layout& L, const float* f, int nbins,
                            float2* work, double* bins, unsigned long long* counts,
                            cudaStream_t st) {
  const int nx = L.nx, ny = L.ny;
  if (!spectrum_supported(nx, ny, nbins) || n < 1) return cudaErrorInvalidValue;
  const int bx = log2_exact(nx), by = log2_exact(ny);
  const size_t row_smem = (size_t)(nx + nx / 2) * sizeof(float2);
  const int rthreads = nx / 2 < 32 ? 32 : (nx / 2 > 256 ? 256 : nx / 2);
  cudaError_t e;
  auto rows = Q == 9 ? spectrum_rows_kernel<9, 9>
                     : (Q == 3 ? spectrum_rows_kernel<3, 3> : spectrum_rows_kernel<2, kMomPlanes>);
  if (Q != 9 && Q != 3 && Q != kMomPlanes) return cudaErrorInvalidValue;
  e = cudaFuncSetAttribute(rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)row_smem);
  if (e != cudaSuccess) return e;
  rows<<<dim3(ny, n), rthreads, row_smem, st>>>(L, f, bx, work);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // columns per CTA: up to 8, at most 8192 complex values in shared memory
  int cb = 8192 / ny;
  if (cb > 8) cb = 8;
  if (cb < 1) cb = 1;
  if (cb > nx) cb = nx;
  const size_t col_smem = ((size_t)cb * ny + (ny > 1 ? ny / 2 : 1)) * sizeof(float2) +
                          (size_t)nbins * (sizeof(double) + 4);
  e = cudaFuncSetAttribute(spectrum_cols_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)col_smem);
  if (e != cudaSuccess) return e;
  spectrum_cols_kernel<<<dim3(nx / cb, n), 256, col_smem, st>>>(nx, ny, by, cb, work, nbins, bins,
                                                                counts);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Azimuthal averages of the interface heights z_0 .. z_n (z_0 the substrate)
// in unit-width rings b = floor(r) around (cx, cy), r the periodic
// (minimum-image) distance; per-cell heights as the read-out gives them
// (h_i = H_i + sum of the stored populations, in FP32), interfaces and sums
// in FP64. A CTA adds its cells (ring_plan.h) into rings in shared memory (SHARED: when
// they fit) and those into sums[m][nbins] and counts[nbins]; every cell
// adding to the global rings directly put 300 addresses under a million
// atomics.
// ---------------------------------------------------------------------------
constexpr size_t kProfileShared = 96 * 1024;

__device__ __forceinline__ int ring_of(double q) {  // floor(sqrt(q))
  const float rf = sqrtf((float)q);
  int b = (int)rf;
  // the FP32 root decides unless it is within its error of a ring's edge
  const float edge = rintf(rf);
  if (fabsf(rf - edge) <= 1e-6f * rf + 1e-6f) b = (int)floor(sqrt(q));
  return b;
}

template <int Q, int PL, bool SHARED>
__global__ void __launch_bounds__(256)
    radial_profile_kernel(int n, Layout L, const float* __restrict__ f, KShift sh,
                          ProfileParams A, RingPlan pl, double* __restrict__ sums,
                          unsigned long long* __restrict__ counts) {
  extern __shared__ double rings[];  // [n + 1][nbins], then counts [nbins]
  const int nx = L.nx, ny = L.ny, nb = A.nbins;
  unsigned* rc = reinterpret_cast<unsigned*>(rings + (size_t)(n + 1) * nb);
  if (SHARED) {
    for (int t = threadIdx.x; t < (n + 1) * nb; t += blockDim.x) rings[t] = 0.0;
    for (int t = threadIdx.x; t < nb; t += blockDim.x) rc[t] = 0u;
    __syncthreads();
  }
  const bool sub = A.sub_amp != 0.0;
  const double inx = 1.0 / nx, iny = 1.0 / ny;
  const int tx = 1 << pl.lgx, items = pl.groups * pl.segs;
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    const int group = item / pl.segs, first = (item - group * pl.segs) * pl.seg;
    const int y = group * pl.tr + (int)(threadIdx.x >> pl.lgx), last = min(nx, first + pl.seg);
    if (y >= ny) continue;
    double dy = y - A.cy;
    dy -= ny * rint(dy * iny);
    if (!(fabs(dy) < (double)nb)) continue;  // no cell of this row is in a ring
    for (int x = first + (int)(threadIdx.x & (tx - 1)); x < last; x += tx) {
      double dx = x - A.cx;
      dx -= nx * rint(dx * inx);
      const double q = fma(dx, dx, dy * dy);
      if (!(q < (double)nb * (double)nb)) continue;
      const int b = ring_of(q);
      if (b >= nb) continue;
      double z = 0.0;
      if (sub) {
        // z_0 = a cos(2 pi (kx x / nx + ky y / ny)), phase reduced in integers
        const long nc = (long)nx * ny;
        long m = (((long)A.sub_kx * x) % nx) * ny + (((long)A.sub_ky * y) % ny) * nx;
        m %= nc;
        if (m < 0) m += nc;
        z = A.sub_amp * cospi(2.0 * (double)m / (double)nc);
        atomicAdd((SHARED ? rings : sums) + b, z);
      }
      for (int i = 0; i < n; ++i) {
        const float* src = f + L.at(i * PL, x, y);
        float d = 0.f;
#pragma unroll
        for (int k = 0; k < Q; ++k) d += src[(long)k * L.plane];
        z += (double)(sh.H[i] + d);
        atomicAdd((SHARED ? rings : sums) + (long)(i + 1) * nb + b, z);
      }
      if (SHARED)
        atomicAdd(rc + b, 1u);
      else
        atomicAdd(counts + b, 1ull);
    }
  }
  if (SHARED) {
    __syncthreads();
    for (int t = threadIdx.x; t < nb; t += blockDim.x) {
      if (rc[t] == 0u) continue;
      atomicAdd(counts + t, (unsigned long long)rc[t]);
      for (int m = sub ? 0 : 1; m <= n; ++m) atomicAdd(sums + (long)m * nb + t, rings[(size_t)m * nb + t]);
    }
  }
}

template <int Q, int PL>
static cudaError_t profile_q(int n, const Layout& L, const float* f, const KShift& sh,
                             const ProfileParams& A, double* sums, unsigned long long* counts,
                             cudaStream_t st) {
  const size_t smem = (size_t)A.nbins * ((n + 1) * sizeof(double) + sizeof(unsigned));
  const RingPlan pl = ring_plan(L.nx, L.ny);
  if (smem > kProfileShared) {
    radial_profile_kernel<Q, PL, false><<<pl.blocks, 256, 0, st>>>(n, L, f, sh, A, pl, sums, counts);
    return cudaGetLastError();
  }
  auto kern = radial_profile_kernel<Q, PL, true>;
  const cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kProfileShared);
  if (e != cudaSuccess) return e;
  kern<<<pl.blocks, 256, smem, st>>>(n, L, f, sh, A, pl, sums, counts);
  return cudaGetLastError();
}

cudaError_t launch_radial_profile(int Q, int n, const Layout& L, const float* f, const KShift& sh,
                                  const ProfileParams& A, double* sums,
                                  unsigned long long* counts, cudaStream_t st) {
  const long cells = (long)L.nx * L.ny;
  if (A.nbins < 1 || n < 1 || cells < 1) return cudaErrorInvalidValue;
  switch (Q) {
    case 9: return profile_q<9, 9>(n, L, f, sh, A, sums, counts, st);
    case 3: return profile_q<3, 3>(n, L, f, sh, A, sums, counts, st);
    case kMomPlanes: return profile_q<2, kMomPlanes>(n, L, f, sh, A, sums, counts, st);
    default: return cudaErrorInvalidValue;
  }
}

MLSW_DEFINE_BOUNDS_READER(bounds_violations_analysis)

}  // namespace mlsw
