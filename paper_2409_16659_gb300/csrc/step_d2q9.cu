// step_d2q9.cu -- the D2Q9 step of one lattice: one warp (one CTA) per unit of
// work, marching down a strip of 64 columns (march.cuh). This file is
// compiled once per layer count MLSW_N.
#include "device_once.h"
#include "march.cuh"
#include "unit_rows.h"

#ifndef MLSW_N
#error "MLSW_N: the layer count of the kernels"
#endif

namespace mlsw {

template <int N, int MODE, bool OP, class T>
__global__ void __launch_bounds__(32, lane_warps<T>(N, MODE))
    step_d2q9(const __grid_constant__ CUtensorMap map, float* __restrict__ fout,
              const __grid_constant__ KParams P, int strips, int rows, int* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int strip = (int)(blockIdx.x % strips), ya = (int)(blockIdx.x / strips) * rows;
  // (two rows a turn spill from four layers on)
  march_unit<N, MODE, OP, N <= 3, T>(P, P, &map, fout, strip * MarchLane<T>::kOut, ya,
                                     min(ya + rows, P.ny), smem_raw, status);
}

// A step of a batch whose instances are all of this kind (batch_kernels.cu):
// registers and instructions of one kind only. SAME: they also share every
// parameter but H and Hsum (the films of a trajectory set), which are then the
// kernel's, in the constant bank; two rows a turn pay again. 16 films of 256^2:
// 38.9 us a step in the kernel of all kinds, 35.1 here (33.6 with the present
// friction).
template <int N, int MODE, bool SAME>
__global__ void __launch_bounds__(32, march_warps(N, MODE))
    step_d2q9_alike(const BatchInst* __restrict__ inst, const int2* __restrict__ table,
                    const __grid_constant__ KParams P, int cur, int* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int2 e = table[blockIdx.x];
  const BatchInst& b = inst[e.x];
  const KParams& G = stage_params(b, smem_raw);
  float* fout = b.f[cur ^ 1];
  __builtin_assume(__isGlobal(fout));
  const int strip = e.y % b.strips, ya = e.y / b.strips * b.rows;
  const KParams& Q = SAME ? P : G;
  march_unit<N, MODE, MODE == kGeneral, SAME && N <= 3, f2>(Q, G, &b.map[cur], fout,
                                                        strip * kMarchOut, ya,
                                                        min(ya + b.rows, Q.ny),
                                                        smem_raw + kParBytes, status);
}

template <int N, int MODE, bool SAME>
static cudaError_t launch_alike(const BatchLaunch& a, cudaStream_t st) {
  constexpr size_t smem = kParBytes + MarchShape<N, MODE, MODE == kGeneral, f2>::kSmem;
  auto kern = step_d2q9_alike<N, MODE, SAME>;
  static DeviceOnce configured;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64) return cudaErrorInvalidDevice;
  e = configured(dev, [&] {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (e != cudaSuccess) return e;
  if (a.nunits <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)a.nunits);
  cfg.blockDim = dim3(32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a.inst, a.table, a.P, a.cur, a.status);
}

template <>
cudaError_t launch_alike_d2q9<MLSW_N>(const BatchLaunch& a, int mode, cudaStream_t st) {
  switch (mode) {
    case kGeneral: return launch_alike<MLSW_N, kGeneral, false>(a, st);
    case kFast:
      return a.same_params ? launch_alike<MLSW_N, kFast, true>(a, st)
                           : launch_alike<MLSW_N, kFast, false>(a, st);
    default: return launch_alike<MLSW_N, kTau1, false>(a, st);
  }
}

template <int N, int MODE, bool OP, class T>
static cudaError_t launch_march_t(const StepLaunch& a, cudaStream_t st) {
  using S = MarchShape<N, MODE, OP, T>;
  auto kern = step_d2q9<N, MODE, OP, T>;
  // raise the dynamic shared-memory limit and count the resident warps once
  // per device and instantiation
  static DeviceOnce configured;
  static int per_sm[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64) return cudaErrorInvalidDevice;
  e = configured(dev, [&] {
    cudaError_t e1 =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kSmem);
    if (e1 != cudaSuccess) return e1;
    int nb = 0;
    e1 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, 32, S::kSmem);
    per_sm[dev] = nb > 0 ? nb : 1;
    return e1;
  });
  if (e != cudaSuccess) return e;
  constexpr bool solo = MarchLane<T>::kPer == 1;
  const int strips = march_strips(a.P.nx, solo), slots = a.num_sms * per_sm[dev];
  const bool heavy = N >= (MODE == kGeneral ? 4 : 5) && step_dear(a.P);
  const int rows =
      solo ? solo_rows(MODE == kGeneral, a.P.ny, strips, a.num_sms, slots)
           : march_rows(N, heavy, a.P.ny, strips, a.num_sms, slots);
  const long units = (long)strips * ((a.P.ny + rows - 1) / rows);
  // launched as a programmatic dependent of the previous kernel on the
  // stream (see march_unit)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)units);
  cfg.blockDim = dim3(32);
  cfg.dynamicSmemBytes = S::kSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, *a.fin_map, a.fout, a.P, strips, rows, a.status);
}

template <int N, int MODE, bool OP>
static cudaError_t launch_march(const StepLaunch& a, cudaStream_t st) {
  if constexpr (N >= 4)  // (march_solo)
    if (a.solo) return launch_march_t<N, MODE, OP, f1>(a, st);
  return launch_march_t<N, MODE, OP, f2>(a, st);
}

template <>
cudaError_t launch_step_d2q9<MLSW_N>(const StepLaunch& a, cudaStream_t st) {
  switch (step_mode(a.P)) {
    case kGeneral: return launch_march<MLSW_N, kGeneral, true>(a, st);
    case kFast:
      return a.to_populations ? launch_march<MLSW_N, kFast, true>(a, st)
                              : launch_march<MLSW_N, kFast, false>(a, st);
    default:
      return a.to_populations ? launch_march<MLSW_N, kTau1, true>(a, st)
                              : launch_march<MLSW_N, kTau1, false>(a, st);
  }
}

MLSW_DEFINE_BOUNDS_READER(MLSW_CAT(bounds_violations_d2q9_, MLSW_N))

}  // namespace mlsw
