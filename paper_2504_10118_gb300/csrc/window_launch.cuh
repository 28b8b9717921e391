// window_launch.cuh -- the per-window-side launch entry points declared in
// core.cuh; included by the window_*.cu files, each of which instantiates
// them for its window sides.
#pragma once

namespace magpie_impl {

template <int MS, int MODE>
cudaError_t launch_window(const StepArgs& a, int windows, cudaStream_t st) {
  using Gm = Geo<MS>;
  // minibatch steps overlap their launch with the previous kernel's tail
  constexpr bool pdl = MODE == kStep || MODE == kStepAtomic || MODE == kStepRecycle;
  return launch_ex(window_kernel<MS, MODE>, dim3((unsigned)windows * Gm::CL), dim3(Gm::T), Gm::SMEM, st, Gm::CL, pdl,
                   a);
}

// The objective pass, which fills every SM: three 256-thread blocks per SM
// where a step's window kernel keeps two (900 windows of 128 x 128: 152 us
// against 170).
template <int MS>
__global__ void __launch_bounds__(Geo<MS>::T, Geo<MS>::T == 256 ? 3 : Geo<MS>::MIN_BLOCKS)
    window_eval_kernel(const __grid_constant__ StepArgs A) {
  constexpr int MODE = kEval;
  const int win = blockIdx.x / Geo<MS>::CL;
#include "window_body.inc"
}
template <int MS>
cudaError_t launch_eval(const StepArgs& a, int windows, cudaStream_t st) {
  using Gm = Geo<MS>;
  return launch_ex(window_eval_kernel<MS>, dim3((unsigned)windows * Gm::CL), dim3(Gm::T), Gm::SMEM, st, Gm::CL, false,
                   a);
}

// A sweep's minibatch step of small windows (one block each, m <= 32): lets
// the update be set up, and list its windows, while the windows run.  Larger
// windows fill the SMs, whose slots the update's blocks would hold (0.343
// against 0.324 ms per sweep at m = 128).  8 x 8 raster of m = 32, minibatch
// 16: 30.7 us per sweep, 33.5 without.
template <int MS>
__global__ void __launch_bounds__(Geo<MS>::T, Geo<MS>::MIN_BLOCKS)
    window_early_kernel(const __grid_constant__ StepArgs A) {
  constexpr int MODE = kStep;
  const int win = blockIdx.x / Geo<MS>::CL;
  grid_dep_wait();
  grid_dep_launch();
#include "window_body.inc"
}
template <int MS>
cudaError_t window_early_launch(const StepArgs& a, int windows, cudaStream_t st) {
  using Gm = Geo<MS>;
  static_assert(Gm::CL == 1 && Gm::SMEM <= 48 * 1024, "small windows");
  return launch_ex(window_early_kernel<MS>, dim3((unsigned)windows), dim3(Gm::T), Gm::SMEM, st, 1, true, a);
}

template <int MS>
cudaError_t window_launch(int mode, const StepArgs& a, int windows, cudaStream_t st) {
  switch (mode) {
    case kStep: return launch_window<MS, kStep>(a, windows, st);
    case kEval: return launch_eval<MS>(a, windows, st);
    case kStepRecycle: return launch_window<MS, kStepRecycle>(a, windows, st);
    case kStepAtomic: return launch_window<MS, kStepAtomic>(a, windows, st);
    default: return cudaErrorInvalidValue;
  }
}

// Candidate register bounds of the batched window kernel: blocks per SM.
// The default (Geo::MIN_BLOCKS), an alternative, and a third, denser one:
// three 256-thread blocks (80 registers; three of the m = 128 kernel's
// 72 KB of shared memory fit an SM), or four of 128 threads or fewer.
template <int MS>
constexpr int alt_minb() {
  return Geo<MS>::T >= 512 ? 1 : (Geo<MS>::MIN_BLOCKS == 1 ? 2 : 1);
}
template <int MS>
constexpr int third_minb() {
  return Geo<MS>::T >= 512 ? 1 : (Geo<MS>::T == 256 ? 3 : 4);
}

template <int MS>
cudaError_t window_launch_batched(const StepArgs* table, const int2* map, int windows, cudaStream_t st, int minb) {
  using Gm = Geo<MS>;
  const dim3 grid((unsigned)windows * Gm::CL);
  if (minb == third_minb<MS>() && minb != Gm::MIN_BLOCKS && minb != alt_minb<MS>())
    return launch_ex(window_kernel_batched<MS, kStep, third_minb<MS>()>, grid, dim3(Gm::T), Gm::SMEM, st, Gm::CL,
                     false, table, map);
  if (minb == alt_minb<MS>() && minb != Gm::MIN_BLOCKS)
    return launch_ex(window_kernel_batched<MS, kStep, alt_minb<MS>()>, grid, dim3(Gm::T), Gm::SMEM, st, Gm::CL,
                     false, table, map);
  return launch_ex(window_kernel_batched<MS, kStep, Gm::MIN_BLOCKS>, grid, dim3(Gm::T), Gm::SMEM, st, Gm::CL, false,
                   table, map);
}

template <int MS>
void window_minb_candidates(int* c) {
  c[0] = Geo<MS>::MIN_BLOCKS;
  c[1] = alt_minb<MS>();
  c[2] = third_minb<MS>();
}

template <int MS>
size_t persistent_smem(int max_count) {
  return std::max(Geo<MS>::SMEM, sizeof(ApplyEntry) * (size_t)max_count);
}

template <int MS>
cudaError_t window_launch_persistent(const PersistArgs& P, int clusters, int max_count, cudaStream_t st, int minb) {
  using Gm = Geo<MS>;
  const dim3 grid((unsigned)clusters * Gm::CL);
  const size_t smem = persistent_smem<MS>(max_count);
  if (minb == alt_minb<MS>() && minb != Gm::MIN_BLOCKS)
    return launch_ex(window_kernel_persistent<MS, alt_minb<MS>()>, grid, dim3(Gm::T), smem, st, Gm::CL, false, P);
  return launch_ex(window_kernel_persistent<MS, Gm::MIN_BLOCKS>, grid, dim3(Gm::T), smem, st, Gm::CL, false, P);
}

template <int MS>
int window_persistent_capacity(int max_count, int minb) {
  using Gm = Geo<MS>;
  void (*k)(PersistArgs) = (minb == alt_minb<MS>() && minb != Gm::MIN_BLOCKS)
                               ? window_kernel_persistent<MS, alt_minb<MS>()>
                               : window_kernel_persistent<MS, Gm::MIN_BLOCKS>;
  const size_t smem = persistent_smem<MS>(max_count);
  int dev = 0, sms = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  if constexpr (Gm::CL == 1) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, Gm::T, smem) != cudaSuccess) return 0;
    return n * sms;
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(Gm::CL * sms));
    cfg.blockDim = dim3(Gm::T);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = Gm::CL;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, (void*)k, &cfg) != cudaSuccess) return 0;
    return n;
  }
}

template <int MS>
cudaError_t window_prepare() {
  const int bytes = (int)Geo<MS>::SMEM;
  cudaError_t e = cudaFuncSetAttribute(window_kernel<MS, kStep>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(window_kernel_batched<MS, kStep, Geo<MS>::MIN_BLOCKS>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(window_kernel_batched<MS, kStep, alt_minb<MS>()>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(window_kernel_batched<MS, kStep, third_minb<MS>()>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)  // the densest bound needs the whole shared-memory carve-out
    e = cudaFuncSetAttribute(window_kernel_batched<MS, kStep, third_minb<MS>()>,
                             cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(window_kernel<MS, kStepRecycle>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(window_kernel<MS, kStepAtomic>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(window_eval_kernel<MS>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  const int pbytes = (int)persistent_smem<MS>(kMaxMinibatch);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(window_kernel_persistent<MS, Geo<MS>::MIN_BLOCKS>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, pbytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(window_kernel_persistent<MS, alt_minb<MS>()>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             pbytes);
  return e;
}

// Forward intensities (mode kSim) of windows 0 .. n - 1 without any device
// memory of the call's own: the twiddles travel as a kernel argument and a
// cluster's window index is its number.  The call is bound by the host around
// it: with a twiddle table and an index list allocated, filled and freed on
// every call, 900 windows of 128 x 128 took 0.326 ms, 0.09 of them the kernel;
// 0.149 now, and 0.134 with three 256-thread blocks per SM instead of two.
template <int MS>
struct TwArg {
  float2 t[MS];
};
template <int MS>
__global__ void __launch_bounds__(Geo<MS>::T, Geo<MS>::T == 256 ? 3 : Geo<MS>::MIN_BLOCKS)
    window_sim_kernel(const __grid_constant__ StepArgs P, const __grid_constant__ TwArg<MS> W) {
  __shared__ StepArgs args;
  __shared__ float2 table[MS];
  __shared__ int32_t self;
  for (int i = threadIdx.x; i < MS; i += Geo<MS>::T) table[i] = W.t[i];
  if (threadIdx.x == 0) {
    args = P;
    args.tw = table;
    args.idx = &self;
    self = (int32_t)(blockIdx.x / Geo<MS>::CL);
  }
  __syncthreads();
  const StepArgs& A = args;
  constexpr int win = 0, MODE = kSim;
#include "window_body.inc"
}
template <int MS>
cudaError_t window_sim_launch(const StepArgs& a, const float2* tw, int windows, cudaStream_t st) {
  using Gm = Geo<MS>;
  const cudaError_t e =
      cudaFuncSetAttribute(window_sim_kernel<MS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::SMEM);
  if (e != cudaSuccess) return e;
  TwArg<MS> W;
  std::copy(tw, tw + MS, W.t);
  return launch_ex(window_sim_kernel<MS>, dim3((unsigned)windows * Gm::CL), dim3(Gm::T), Gm::SMEM, st, Gm::CL, false,
                   a, W);
}

// The three kernels of the split form, each a programmatic dependent of the
// one before (the exit kernel of the stream's previous kernel).
template <int MS>
cudaError_t split_launch(bool atomic, bool early, const StepArgs& a, int windows, cudaStream_t st) {
  using S = Split<MS>;
  if (atomic && MS != 64) return cudaErrorInvalidValue;  // atomic_form: no other side uses the float atomics
  const dim3 grid((unsigned)windows * S::TILES), block(S::T);
  cudaError_t e = launch_ex(split_exit_kernel<MS>, grid, block, 0, st, 1, true, a, early);
  if (e == cudaSuccess) e = launch_ex(split_project_kernel<MS>, grid, block, 0, st, 1, true, a);
  if (e == cudaSuccess)
    e = launch_ex(atomic ? split_grad_kernel<MS, MS == 64> : split_grad_kernel<MS, false>, grid, block, 0, st, 1, true, a);
  return e;
}

template <int MS>
cudaError_t split_launch_batched(const StepArgs* table, const int2* map, int windows, cudaStream_t st) {
  using S = Split<MS>;
  const dim3 grid((unsigned)windows * S::TILES), block(S::T);
  cudaError_t e = launch_ex(split_kernel_batched<MS, 0>, grid, block, 0, st, 1, true, table, map);
  if (e == cudaSuccess) e = launch_ex(split_kernel_batched<MS, 1>, grid, block, 0, st, 1, true, table, map);
  if (e == cudaSuccess) e = launch_ex(split_kernel_batched<MS, 2>, grid, block, 0, st, 1, true, table, map);
  return e;
}

#define MAGPIE_INSTANTIATE_EARLY(S) template cudaError_t window_early_launch<S>(const StepArgs&, int, cudaStream_t);

#define MAGPIE_INSTANTIATE_SPLIT(S)                                                     \
  template cudaError_t split_launch<S>(bool, bool, const StepArgs&, int, cudaStream_t); \
  template cudaError_t split_launch_batched<S>(const StepArgs*, const int2*, int, cudaStream_t);

#define MAGPIE_INSTANTIATE_WINDOW(S)                                                                       \
  template cudaError_t window_launch<S>(int, const StepArgs&, int, cudaStream_t);                          \
  template cudaError_t window_sim_launch<S>(const StepArgs&, const float2*, int, cudaStream_t);            \
  template cudaError_t window_launch_batched<S>(const StepArgs*, const int2*, int, cudaStream_t, int);     \
  template cudaError_t window_prepare<S>();                                                                \
  template void window_minb_candidates<S>(int*);                                                            \
  template cudaError_t window_launch_persistent<S>(const PersistArgs&, int, int, cudaStream_t, int);      \
  template int window_persistent_capacity<S>(int, int);

}  // namespace magpie_impl
