// batch_kernels.cu -- one D2Q9 step of every instance of a batch in one
// launch. This file is compiled once per MLSW_BATCH_N, the largest layer
// count its kernel holds.
//
// The unit table lists (instance, unit) pairs sorted by kind (layer count,
// kernel mode); a CTA is one warp that marches down one unit (section LBM,
// the same code as the single-lattice step, march.cuh). Neighbouring CTAs
// run the same kind, so the warps of an SM share its instructions.
#include <algorithm>
#include <type_traits>

#include "device_once.h"
#include "march.cuh"

#ifndef MLSW_BATCH_N
#error "MLSW_BATCH_N: the largest layer count of the kernel"
#endif

namespace mlsw {

namespace {

// The kernel for at most three layers leaves out three layers of the general
// mode (batch_small): 12 warps an SM have no registers for that. 32 lattices of 1
// to 3 layers, all modes: 100 us a step with it (and one height for all), 64 in
// the kernel for five layers. Three layers at tau = 1 stay, although they spill
// (180 bytes): 53 lattices of the fast mode and those take 69 us here, 85 there.
constexpr bool in_kernel(int kind) {
  return MLSW_BATCH_N > 3 ? kind < 3 * MLSW_BATCH_N : batch_small(1u << kind);
}
constexpr int next_kind(int kind) {
  while (kind < kBatchKinds && !in_kernel(kind)) ++kind;
  return kind;
}
template <int K>
constexpr int kNextKind = next_kind(K + 1);
constexpr int kWarps = MLSW_BATCH_N > 3 ? 8 : march_warps(3, kFast);

template <int K>
struct KindOf {
  static constexpr int N = K / 3 + 1, M = K % 3;
  static constexpr bool OP = M == kGeneral;
  using T = typename std::conditional<batch_solo(~0u, K), f1, f2>::type;
  static constexpr size_t kSmem = MarchShape<N, M, OP, T>::kSmem;
};

// The unit, if its kind is K, else the next kinds. Straight-line code: as
// separate functions the kinds would lose the registers that carry rows.
template <int K>
__device__ __forceinline__ void run_kind(int kind, const KParams& P, const BatchInst& b, int cur,
                                         int strip, int ya, int yb, unsigned char* sm,
                                         int* __restrict__ status) {
  using X = KindOf<K>;
  if (kind == K) {
    float* fout = b.f[cur ^ 1];
    __builtin_assume(__isGlobal(fout));
    march_unit<X::N, X::M, X::OP, false, typename X::T>(
        P, P, &b.map[cur], fout, strip * MarchLane<typename X::T>::kOut, ya, yb, sm, status);
  } else if constexpr (kNextKind<K> < kBatchKinds) {
    run_kind<kNextKind<K>>(kind, P, b, cur, strip, ya, yb, sm, status);
  }
}

// dynamic shared memory of a launch over the given kinds
template <int K>
size_t smem_from(unsigned kinds) {
  size_t s = (kinds >> K) & 1u ? KindOf<K>::kSmem : 0;
  if constexpr (kNextKind<K> < kBatchKinds) s = std::max(s, smem_from<kNextKind<K>>(kinds));
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
  run_kind<0>(b.kind, P, b, cur, strip, ya, min(ya + b.rows, P.ny), smem_raw + kParBytes,
                   status);
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
namespace {

// shared memory of a warp of the alike kernels, by kind
template <int K>
size_t alike_smem(int kind) {
  if (kind == K) return kParBytes + MarchShape<K / 3 + 1, K % 3, K % 3 == kGeneral, f2>::kSmem;
  if constexpr (K + 1 < kBatchKinds) return alike_smem<K + 1>(kind);
  return 0;
}

}  // namespace

cudaError_t launch_batch_step(const BatchLaunch& a, cudaStream_t st) {
  // instances of one kind have a kernel of their own
  for (int k = 0; k < kBatchKinds; ++k)
    if (a.kinds == 1u << k) return launch_batch_alike(a, k / 3 + 1, k % 3, st);
  return batch_small(a.kinds) ? launch_batch_step_n<3>(a, st) : launch_batch_step_n<5>(a, st);
}

int batch_warps_per_sm(unsigned kinds) {
  int warps = batch_small(kinds) ? march_warps(3, kFast) : 8;
  size_t smem = kParBytes + smem_from<0>(kinds);
  for (int k = 0; k < kBatchKinds; ++k)
    if (kinds == 1u << k) {
      warps = march_warps(k / 3 + 1, k % 3) + 3;
      smem = alike_smem<0>(k);
    }
  warps = warps / 4 * 4;  // (the same number on each of the four schedulers)
  // 228 KB of shared memory, 1 KB of it taken by each CTA
  return std::min(warps, (int)(233472 / (smem + 1024)));
}
#endif

MLSW_DEFINE_BOUNDS_READER(MLSW_CAT(bounds_violations_batch_, MLSW_BATCH_N))

}  // namespace mlsw
