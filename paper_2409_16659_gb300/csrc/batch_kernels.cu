// batch_kernels.cu -- one D2Q9 step of every instance of a batch in one
// launch. This file is compiled once per MLSW_BATCH_N, the largest layer
// count its kernel holds.
//
// The unit table lists (instance, unit) pairs sorted by kind (layer count,
// kernel mode); a CTA is one warp that marches down one unit (section LBM,
// the same code as the single-lattice step, march.cuh). Neighbouring CTAs
// run the same kind, so the warps of an SM share its instructions.
#include <algorithm>

#include "device_once.h"
#include "march.cuh"

#ifndef MLSW_BATCH_N
#error "MLSW_BATCH_N: the largest layer count of the kernel"
#endif

namespace mlsw {

namespace {

// Warps per SM, as for the single lattice.
constexpr int kWarps = march_warps(MLSW_BATCH_N, kFast);

// The unit, if its kind is K, else the next kinds. Straight-line code: as
// separate functions the kinds would lose the registers that carry rows.
template <int K>
__device__ __forceinline__ void run_kind(int kind, const KParams& P, const BatchInst& b, int cur,
                                         int x0, int ya, int yb, unsigned char* sm,
                                         int* __restrict__ status) {
  constexpr int N = K / 3 + 1, M = K % 3;
  if (kind == K) {
    float* fout = b.f[cur ^ 1];
    __builtin_assume(__isGlobal(fout));
    march_unit<N, M, M == kGeneral, false, f2>(P, P, &b.map[cur], fout, x0, ya, yb, sm, status);
  } else if constexpr (K + 1 < 3 * MLSW_BATCH_N) {
    run_kind<K + 1>(kind, P, b, cur, x0, ya, yb, sm, status);
  }
}

// dynamic shared memory of a launch over the given kinds
template <int K>
size_t smem_from(unsigned kinds) {
  constexpr int N = K / 3 + 1, M = K % 3;
  size_t s = (kinds >> K) & 1u ? MarchShape<N, M, M == kGeneral, f2>::kSmem : 0;
  if constexpr (K + 1 < 3 * MLSW_BATCH_N) s = std::max(s, smem_from<K + 1>(kinds));
  return s;
}

}  // namespace

// The instance's parameters are read from a copy in shared memory: in global
// memory every use after a store would load them again. One row a turn: the
// kinds' code is long, and the warps of an SM wait for instructions (48 lattices
// of 2 to 5 layers: 198 us a step with two rows, 182 with one).
template <int NMAX>
__global__ void __launch_bounds__(32, kWarps)
    step_d2q9_batch(const BatchInst* __restrict__ inst, const int2* __restrict__ table, int cur,
                    int* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int2 e = table[blockIdx.x];
  const BatchInst& b = inst[e.x];
  const KParams& P = stage_params(b, smem_raw);
  const int strip = e.y % b.strips, ya = e.y / b.strips * b.rows;
  run_kind<0>(b.kind, P, b, cur, strip * kMarchOut, ya, min(ya + b.rows, P.ny),
                      smem_raw + kParBytes, status);
}

template <>
cudaError_t launch_batch_step_n<MLSW_BATCH_N>(const BatchLaunch& a, cudaStream_t st) {
  if (a.nunits <= 0) return cudaSuccess;
  auto kern = step_d2q9_batch<MLSW_BATCH_N>;
  // once per device: the largest shared memory any kind can need
  static DeviceOnce configured;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64) return cudaErrorInvalidDevice;
  e = configured(dev, [&] {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(kParBytes + smem_from<0>(~0u)));
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)a.nunits);
  cfg.blockDim = dim3(32);
  cfg.dynamicSmemBytes = kParBytes + smem_from<0>(a.kinds);
  cfg.stream = st;
  // a programmatic dependent of the previous kernel (see march_unit)
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a.inst, a.table, a.cur, a.status);
}

#if MLSW_BATCH_N == 5
cudaError_t launch_batch_step(const BatchLaunch& a, cudaStream_t st) {
  // instances of one kind have a kernel of their own
  for (int k = 0; k < kBatchKinds; ++k)
    if (a.kinds == 1u << k) return launch_batch_alike(a, k / 3 + 1, k % 3, st);
  return a.nmax <= 3 ? launch_batch_step_n<3>(a, st) : launch_batch_step_n<5>(a, st);
}

int batch_warps_per_sm(unsigned kinds) {
  int nmax = 0, alike = 0;
  for (int k = 0; k < kBatchKinds; ++k) {
    if (kinds == 1u << k) alike = march_warps(k / 3 + 1, k % 3);
    if ((kinds >> k) & 1u) nmax = k / 3 + 1;
  }
  // (the same number on each of the four schedulers)
  return (alike ? alike + 3 : march_warps(nmax <= 3 ? 3 : 5, kFast)) / 4 * 4;
}
#endif

MLSW_DEFINE_BOUNDS_READER(MLSW_CAT(bounds_violations_batch_, MLSW_BATCH_N))

}  // namespace mlsw
