// launch_impl.cuh -- bodies of the launchers declared in launch.h; included once per
// storage precision by launch_f32.cu / launch_f64.cu with KSS_T defined.
#pragma once

#include <algorithm>
#include <atomic>

#include "launch.h"

namespace kss {

// (column blocks of 256) x (rows, strided beyond 65535) for the auxiliary kernels.
inline dim3 helper_grid(int nx, long long rows) {
  return dim3((unsigned)((nx + 255) / 256), (unsigned)(rows < 65535 ? rows : 65535));
}

// Columns per thread of the kernels between pitched planes and a dense FP64 array: two
// where every pair of columns of every row is 16-byte aligned there.  (Rows of the planes
// always are: their pitch is a multiple of 128 bytes.)
inline int dense_vec(const void* dense, int nx) {
  return (nx % 2 == 0 && reinterpret_cast<uintptr_t>(dense) % 16 == 0) ? 2 : 1;
}

// Let `kernel` take DYN bytes of dynamic shared memory on the current device (beyond the
// default 48 KB of static plus dynamic memory an opt-in is needed), once per device.
// Threads that race here at most repeat the (idempotent) attribute call.
template <auto kernel, int DYN>
cudaError_t allow_dynamic_smem() {
  if constexpr (DYN == 0) {
    return cudaSuccess;
  } else {
    constexpr int kMaxDev = 64;
    static std::atomic<bool> done[kMaxDev] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDev) return cudaErrorInvalidDevice;
    if (!done[dev].load(std::memory_order_acquire)) {
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DYN);
      if (e != cudaSuccess) return e;
      done[dev].store(true, std::memory_order_release);
    }
    return cudaSuccess;
  }
}

// kernel<<<grid, threads, dyn, stream>>>(args...), launched while the stream's previous kernel
// still runs if that one allows it (see previous_done), in clusters of `cluster` CTAs along z.
template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int threads, int dyn,
                           cudaStream_t stream, int cluster, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = size_t(dyn);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = unsigned(cluster);
  // (FP64: a split step launched into SMs that its predecessor still occupies has its
  // clusters doubled up on the free ones; FP64 128^2 with outputs every 10 steps 7.5 -> 11.3 us)
  const int first = std::is_same<KSS_T, double>::value ? 1 : 0;
  cfg.attrs = attr + first;
  cfg.numAttrs = (cluster > 1 ? 2 : 1) - first;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Let `kernel` run in clusters of more than eight CTAs on the current device, once per
// device (as above).
template <auto kernel>
cudaError_t allow_large_clusters() {
  constexpr int kMaxDev = 64;
  static std::atomic<bool> done[kMaxDev] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDev) return cudaErrorInvalidDevice;
  if (!done[dev].load(std::memory_order_acquire)) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    done[dev].store(true, std::memory_order_release);
  }
  return cudaSuccess;
}

// CTAs of `kernel` (with DYN bytes of dynamic shared memory) resident on the current
// device at once (its occupancy times the SM count), looked up once per device (racing
// threads at most repeat the query).
template <auto kernel, int DYN = 0>
int resident_ctas() {
  constexpr int kMaxDev = 64;
  static std::atomic<int> cache[kMaxDev] = {};  // one per kernel: a template argument
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return 0;
  int n = cache[dev].load(std::memory_order_acquire);
  if (!n) {
    int nsm = 0, per = 0;
    if (allow_dynamic_smem<kernel, DYN>() != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, kThreads, DYN) != cudaSuccess)
      return 0;
    n = nsm * per;
    cache[dev].store(n, std::memory_order_release);
  }
  return n;
}

// Persistent steps: when the step grid exceeds one wave of resident CTAs, one wave that
// strides over the blocks (step_kernel_persistent).  Measured on GB300 (4096^2 / 8192^2):
// slower than one CTA per block for FP32 (fused 0.257 vs 0.243 ms, plain 0.199 vs 0.179 ms)
// and for fused FP16 deviations, faster only for plain FP16-deviation steps (0.113 vs
// 0.123 ms), so that is the one case that takes it (KSS_PERSISTENT=1 forces it everywhere).
#ifndef KSS_PERSISTENT
#define KSS_PERSISTENT 0
#endif
// Eight cells per lane for the FP16 {Kn, KL, neq} step (step_block<..., VC = 8>); 0 keeps
// four.
#ifndef KSS_F16_CELLS8
#define KSS_F16_CELLS8 1
#endif

// SMs of the current device, looked up once per device (0 on error).
inline int sm_count() {
  constexpr int kMaxDev = 64;
  static std::atomic<int> cache[kMaxDev] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return 0;
  int n = cache[dev].load(std::memory_order_acquire);
  if (!n) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    cache[dev].store(n, std::memory_order_release);
  }
  return n;
}

template <>
int split_ranks<KSS_T>(long long nblocks, int rows) {
  const long long slots = 2LL * sm_count();
  int ranks = std::min(rows / split_rows<KSS_T>(), 16);
  if (std::is_same<KSS_T, double>::value) {
    if (7 * nblocks * (rows / kWarps) > 10 * slots) return 0;
  } else if (nblocks * (rows / kWarps) > slots) {
    // (two rows per warp where one each would not fit)
    if (nblocks * (rows / (2 * kWarps)) > slots) return 0;
    ranks /= 2;
  }
  return ranks >= 2 && ranks * split_rows<KSS_T>() * kSplitTurns >= rows ? ranks : 0;
}

template <>
int step_split_ranks<KSS_T>(const StepParams<KSS_T>& p, int mode, bool aar, bool* cells8) {
  bool eight = false;
  dim3 g = step_grid<KSS_T>(p.nx, p.ny, p.tile, p.bands);
  if (std::is_same<KSS_T, __half>::value && mode == MODE_STD && !aar && KSS_F16_PREFETCH &&
      KSS_F16_CELLS8) {
    // (the sums of an FP16 lattice's steps are those of its eight-cell blocks)
    dim3 g8;
    int bands8 = 0;
    if (step_grid8(p.nx, p.ny, p.tile, p.bands, KSS_H8_WARPS, g8, bands8)) {
      if (bands8 != p.bands) return 0;
      eight = true;
      g = g8;
    }
  }
  if (cells8) *cells8 = eight;
  return mode == MODE_PLAIN ? 0 : split_ranks<KSS_T>((long long)g.x * g.y, p.tile * p.bands);
}

// One split step: a cluster of `ranks` CTAs per block of `grid` (the clusters of more than
// eight CTAs of FP64 steps need an opt-in, once per device).
template <int MODE, bool PULL, bool STORE, bool AAR, int VC>
cudaError_t launch_split(const StepParams<KSS_T>& p, dim3 grid, int ranks, cudaStream_t stream) {
  constexpr auto kern = step_kernel_split<KSS_T, MODE, PULL, STORE, AAR, VC>;
  const int dyn = split_smem<KSS_T, MODE, VC>(p.tile * p.bands);
  cudaError_t e = allow_dynamic_smem<kern, split_smem<KSS_T, MODE, VC>(64)>();  // any height
  if (e == cudaSuccess && ranks > 8) e = allow_large_clusters<kern>();
  if (e != cudaSuccess) return e;
  return launch_chained(kern, dim3(grid.x, grid.y, unsigned(ranks)), 32 * split_warps<KSS_T>(),
                        dyn, stream, ranks, p);
}

// A plain FP64 step of a lattice whose 8-row CTAs leave SMs idle (step_plain_f64_kernel:
// 128^2 13.0 -> 5.1 us); true if launched.
template <bool AAR>
bool launch_plain_f64(const StepParams<KSS_T>& p, dim3 grid, cudaStream_t stream,
                      cudaError_t& e) {
  if constexpr (std::is_same<KSS_T, double>::value) {
    if (p.tile * p.bands != 8 || (long long)grid.x * grid.y >= sm_count()) return false;
    const dim3 g((p.nx + 63) / 64, (p.ny + 1) / 2);
    if (g.y > 65535) return false;
    step_plain_f64_kernel<AAR><<<g, 128, 0, stream>>>(p);
    e = cudaGetLastError();
    return true;
  }
  return false;
}

template <int MODE>
cudaError_t launch_step_mode(const StepParams<KSS_T>& p, dim3 grid, cudaStream_t stream) {
  const int nblocks = int(grid.x * grid.y);
  if constexpr (MODE == MODE_PLAIN) {
    cudaError_t e = cudaSuccess;
    if (launch_plain_f64<false>(p, grid, stream, e)) return e;
  }
  if constexpr (MODE != MODE_PLAIN) {
    bool cells8 = false;
    if (const int ranks = step_split_ranks<KSS_T>(p, MODE, false, &cells8)) {
      if constexpr (std::is_same<KSS_T, __half>::value && MODE == MODE_STD) {
        if (cells8)
          return launch_split<MODE, true, true, false, 8>(
              p, dim3(unsigned((p.nx + 255) / 256), grid.y), ranks, stream);
      }
      return launch_split<MODE, true, true, false, Vec<KSS_T>::N>(p, grid, ranks, stream);
    }
  }
  constexpr bool kHalfPlain = std::is_same<KSS_T, __half>::value && MODE == MODE_PLAIN;
  if (KSS_PERSISTENT || kHalfPlain) {
    const int wave = resident_ctas<step_kernel_persistent<KSS_T, MODE, true, true>>();
    if (wave > 0 && nblocks > wave) {
      step_kernel_persistent<KSS_T, MODE, true, true><<<wave, kThreads, 0, stream>>>(
          p, int(grid.x), nblocks);
      return cudaGetLastError();
    }
  }
  if constexpr (std::is_same<KSS_T, float>::value &&
                step_prefetch_smem<KSS_T, MODE, true>() > 0) {
    // FP32 {Kn, KL, neq} with the row prefetch (KSS_F32_ONESTEP_PREFETCH)
    constexpr int dyn = step_prefetch_smem<KSS_T, MODE, true>();
    const cudaError_t e = allow_dynamic_smem<step_kernel<KSS_T, MODE, true, true, false, true>, dyn>();
    if (e != cudaSuccess) return e;
    return launch_chained(step_kernel<KSS_T, MODE, true, true, false, true>, grid, kThreads, dyn,
                          stream, 1, p);
  }
  if constexpr (std::is_same<KSS_T, __half>::value && KSS_F16_PREFETCH &&
                step_prefetch_smem<KSS_T, MODE, true>() > 0) {
    // FP16 deviations, {Kn, KL, neq}: the row prefetch, with its dynamic shared memory.
    // Eight cells per lane: CTA blocks of 256 columns and at most 8 rows per warp, where
    // that grid has no more blocks than the four-cell one (whose count sized the partial
    // sums)
    if constexpr (KSS_F16_CELLS8) {
      constexpr int NW = KSS_H8_WARPS;
      dim3 g8;
      int bands8 = 0;
      if (step_grid8(p.nx, p.ny, p.tile, p.bands, NW, g8, bands8)) {
        StepParams<KSS_T> q = p;
        q.bands = bands8;
        constexpr auto kern = step_kernel<KSS_T, MODE, true, true, false, true, 8, NW>;
        constexpr int dyn8 = step_prefetch_smem<KSS_T, MODE, true, 8, NW>();
        const cudaError_t e = allow_dynamic_smem<kern, dyn8>();
        if (e != cudaSuccess) return e;
        return launch_chained(kern, g8, 32 * NW, dyn8, stream, 1, q);
      }
    }
    constexpr int dyn = step_prefetch_smem<KSS_T, MODE, true>();
    const cudaError_t e = allow_dynamic_smem<step_kernel<KSS_T, MODE, true, true, false, true>, dyn>();
    if (e != cudaSuccess) return e;
    return launch_chained(step_kernel<KSS_T, MODE, true, true, false, true>, grid, kThreads, dyn,
                          stream, 1, p);
  }
  if constexpr (MODE == MODE_PLAIN) {
    step_kernel<KSS_T, MODE, true, true><<<grid, kThreads, 0, stream>>>(p);
    return cudaGetLastError();
  } else {
    return launch_chained(step_kernel<KSS_T, MODE, true, true>, grid, kThreads, 0, stream, 1, p);
  }
}

template <>
cudaError_t launch_step<KSS_T>(const StepParams<KSS_T>& p, int mode, bool pull, bool store,
                               cudaStream_t stream) {
  const dim3 grid = step_grid<KSS_T>(p.nx, p.ny, p.tile, p.bands);
  const dim3 block(kThreads);
  if (store && pull) {
    switch (mode) {
      case MODE_PLAIN: return launch_step_mode<MODE_PLAIN>(p, grid, stream);
      case MODE_STD: return launch_step_mode<MODE_STD>(p, grid, stream);
      case MODE_FULL: return launch_step_mode<MODE_FULL>(p, grid, stream);
      default: return cudaErrorInvalidValue;
    }
  } else if (!store) {
    if (const int ranks = split_ranks<KSS_T>((long long)grid.x * grid.y, p.tile * p.bands)) {
      constexpr int V = Vec<KSS_T>::N;
      if (mode == MODE_STD)
        return pull ? launch_split<MODE_STD, true, false, false, V>(p, grid, ranks, stream)
                    : launch_split<MODE_STD, false, false, false, V>(p, grid, ranks, stream);
      return pull ? launch_split<MODE_FULL, true, false, false, V>(p, grid, ranks, stream)
                  : launch_split<MODE_FULL, false, false, false, V>(p, grid, ranks, stream);
    }
    if (mode == MODE_STD && pull) step_kernel<KSS_T, MODE_STD, true, false><<<grid, block, 0, stream>>>(p);
    else if (mode == MODE_STD) step_kernel<KSS_T, MODE_STD, false, false><<<grid, block, 0, stream>>>(p);
    else if (mode == MODE_FULL && pull) step_kernel<KSS_T, MODE_FULL, true, false><<<grid, block, 0, stream>>>(p);
    else if (mode == MODE_FULL) step_kernel<KSS_T, MODE_FULL, false, false><<<grid, block, 0, stream>>>(p);
    else return cudaErrorInvalidValue;
  } else {
    return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <>
bool can_step_twice<KSS_T>(int nx, int ny) {
  return KSS_STEP_TWICE && std::is_same<KSS_T, float>::value &&
         (ny + kTwiceRows - 1) / kTwiceRows <= 65535 && nx > 0;
}

template <class S>
cudaError_t launch_twice(const StepParams<S>& p, S* mid, cudaStream_t stream) {
#if KSS_STEP_TWICE
  if constexpr (std::is_same<S, float>::value) {
    constexpr auto kern = step_plain_twice_kernel<kTwiceRows>;
    constexpr int dyn = 9 * (kTwiceRows + 2) * kTwicePitch * int(sizeof(float));
    const cudaError_t e = allow_dynamic_smem<kern, dyn>();
    if (e != cudaSuccess) return e;
    const dim3 g((p.nx + 127) / 128, (p.ny + kTwiceRows - 1) / kTwiceRows);
    kern<<<g, 32 * (kTwiceRows + 3), dyn, stream>>>(p, mid);
    return cudaGetLastError();
  }
#endif
  return cudaErrorInvalidValue;
}

template <>
cudaError_t launch_plain_twice<KSS_T>(const StepParams<KSS_T>& p, KSS_T* mid,
                                      cudaStream_t stream) {
  return launch_twice<KSS_T>(p, mid, stream);
}

template <>
cudaError_t launch_step_aar<KSS_T>(const StepParams<KSS_T>& p, int mode, cudaStream_t stream) {
  const dim3 grid = step_grid<KSS_T>(p.nx, p.ny, p.tile, p.bands);
  if (const int ranks = step_split_ranks<KSS_T>(p, mode, true, nullptr)) {
    constexpr int V = Vec<KSS_T>::N;
    return mode == MODE_STD ? launch_split<MODE_STD, true, true, true, V>(p, grid, ranks, stream)
                            : launch_split<MODE_FULL, true, true, true, V>(p, grid, ranks, stream);
  }
  cudaError_t e = cudaSuccess;
  if (mode == MODE_PLAIN && launch_plain_f64<true>(p, grid, stream, e)) return e;
  switch (mode) {
    case MODE_PLAIN:
      step_kernel<KSS_T, MODE_PLAIN, true, true, true><<<grid, kThreads, 0, stream>>>(p);
      return cudaGetLastError();
    case MODE_STD:
      return launch_chained(step_kernel<KSS_T, MODE_STD, true, true, true>, grid, kThreads, 0,
                            stream, 1, p);
    case MODE_FULL:
      return launch_chained(step_kernel<KSS_T, MODE_FULL, true, true, true>, grid, kThreads, 0,
                            stream, 1, p);
    default: return cudaErrorInvalidValue;
  }
}

template <>
int multi_resident_ctas<KSS_T>(int mode, bool aar) {
  if (mode != MODE_STD) return 0;
  return aar ? resident_ctas<step_kernel_multi<KSS_T, MODE_STD, true>,
                             multi_prefetch_smem<KSS_T, MODE_STD, true>()>()
             : resident_ctas<step_kernel_multi<KSS_T, MODE_STD>,
                             multi_prefetch_smem<KSS_T, MODE_STD, false>()>();
}

template <>
cudaError_t launch_step_multi<KSS_T>(const StepParams<KSS_T>& pa, const StepParams<KSS_T>& pb,
                                     const MultiState& m, int mode, int ctas,
                                     cudaStream_t stream, bool aar) {
  StepParams<KSS_T> a = pa, b = pb;
  MultiState ms = m;
  void* args[] = {&a, &b, &ms};
  if (mode != MODE_STD) return cudaErrorInvalidValue;
  constexpr int dyn_aar = multi_prefetch_smem<KSS_T, MODE_STD, true>();
  constexpr int dyn_bgk = multi_prefetch_smem<KSS_T, MODE_STD, false>();
  const int dyn = aar ? dyn_aar : dyn_bgk;
  const cudaError_t e =
      aar ? allow_dynamic_smem<step_kernel_multi<KSS_T, MODE_STD, true>, dyn_aar>()
          : allow_dynamic_smem<step_kernel_multi<KSS_T, MODE_STD>, dyn_bgk>();
  if (e != cudaSuccess) return e;
  const void* fn = aar ? reinterpret_cast<const void*>(step_kernel_multi<KSS_T, MODE_STD, true>)
                       : reinterpret_cast<const void*>(step_kernel_multi<KSS_T, MODE_STD>);
  return cudaLaunchCooperativeKernel(fn, dim3(ctas), dim3(kThreads), args, dyn, stream);
}

template <>
int batch_multi_resident_ctas<KSS_T>(int mode) {
  return mode == MODE_STD ? resident_ctas<batch_kernel_multi<KSS_T, MODE_STD>,
                                         multi_prefetch_smem<KSS_T, MODE_STD, false>()>()
                          : 0;
}

template <>
cudaError_t launch_batch_multi<KSS_T>(const StepParams<KSS_T>* ta, const StepParams<KSS_T>* tb,
                                      const MultiState* mtab, const BatchItem* items,
                                      int nitems, int nsteps, uint32_t* work, int mode,
                                      int ctas, cudaStream_t stream) {
  if (mode != MODE_STD || nitems < 1 || nsteps < 1 || ctas < 1) return cudaErrorInvalidValue;
  const StepParams<KSS_T>* a = ta;
  const StepParams<KSS_T>* b = tb;
  const MultiState* m = mtab;
  const BatchItem* it = items;
  int ni = nitems, ns = nsteps;
  uint32_t* w = work;
  void* args[] = {&a, &b, &m, &it, &ni, &ns, &w};
  constexpr int dyn = multi_prefetch_smem<KSS_T, MODE_STD, false>();
  const cudaError_t e = allow_dynamic_smem<batch_kernel_multi<KSS_T, MODE_STD>, dyn>();
  if (e != cudaSuccess) return e;
  const void* fn = reinterpret_cast<const void*>(batch_kernel_multi<KSS_T, MODE_STD>);
  return cudaLaunchCooperativeKernel(fn, dim3(ctas), dim3(kThreads), args, dyn, stream);
}

template <>
cudaError_t launch_batch_split<KSS_T>(const StepParams<KSS_T>* table, const BatchItem* items,
                                      int nitems, int rows, int ranks, bool defer, bool prev,
                                      cudaStream_t stream) {
  constexpr auto kern = batch_step_kernel_split<KSS_T>;
  constexpr int V = Vec<KSS_T>::N;
  cudaError_t e = allow_dynamic_smem<kern, split_smem<KSS_T, MODE_STD, V>(64)>();
  if (e == cudaSuccess && ranks > 8) e = allow_large_clusters<kern>();
  if (e != cudaSuccess) return e;
  return launch_chained(kern, dim3(unsigned(nitems), 1u, unsigned(ranks)),
                        32 * split_warps<KSS_T>(), split_smem<KSS_T, MODE_STD, V>(rows), stream,
                        ranks, table, items, defer, prev);
}

template <>
cudaError_t launch_batch_step<KSS_T>(const StepParams<KSS_T>* table, const BatchItem* items,
                                     int nitems, int ctas, int mode, cudaStream_t stream,
                                     bool aar) {
  if (nitems < 1 || ctas < 1) return cudaErrorInvalidValue;
  const dim3 grid(unsigned(ctas < nitems ? ctas : nitems)), block(kThreads);
  if (aar) {
    switch (mode) {
      case MODE_PLAIN: batch_step_kernel<KSS_T, MODE_PLAIN, true><<<grid, block, 0, stream>>>(table, items, nitems); break;
      case MODE_STD: batch_step_kernel<KSS_T, MODE_STD, true><<<grid, block, 0, stream>>>(table, items, nitems); break;
      case MODE_FULL: batch_step_kernel<KSS_T, MODE_FULL, true><<<grid, block, 0, stream>>>(table, items, nitems); break;
      default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
  }
  switch (mode) {
    case MODE_PLAIN: batch_step_kernel<KSS_T, MODE_PLAIN><<<grid, block, 0, stream>>>(table, items, nitems); break;
    case MODE_STD: batch_step_kernel<KSS_T, MODE_STD><<<grid, block, 0, stream>>>(table, items, nitems); break;
    case MODE_FULL: batch_step_kernel<KSS_T, MODE_FULL><<<grid, block, 0, stream>>>(table, items, nitems); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

#ifndef KSS_STORAGE_HALF
template <>
cudaError_t launch_adj_objective<KSS_T>(const AdjParams<KSS_T>& p, cudaStream_t stream) {
  adj_objective_kernel<KSS_T><<<adj_grid(p.nx, p.ny, p.rows), kThreads, 0, stream>>>(p);
  return cudaGetLastError();
}

template <>
cudaError_t launch_adj_reverse<KSS_T>(const AdjParams<KSS_T>& p, bool chained,
                                      cudaStream_t stream) {
  const dim3 g = adj_reverse_grid(p.nx, p.ny, p.rows);
  if (chained)
    return launch_chained(adj_reverse_kernel<KSS_T>, g, 32 * kAdjWarps, 0, stream, 1, p);
  adj_reverse_kernel<KSS_T><<<g, 32 * kAdjWarps, 0, stream>>>(p);
  return cudaGetLastError();
}

template <>
cudaError_t launch_adj_totals<KSS_T>(const double* part, int n, int nit, double* totals,
                                     uint32_t* count, double* acc, cudaStream_t stream) {
  adj_iteration_totals<KSS_T><<<nit, kThreads, 0, stream>>>(part, n, nit, totals, count, acc);
  return cudaGetLastError();
}

template <>
cudaError_t launch_adj_final<KSS_T>(const AdjParams<KSS_T>& p, cudaStream_t stream) {
  adj_final_kernel<KSS_T><<<adj_grid(p.nx, p.ny, p.rows), kThreads, 0, stream>>>(p);
  return cudaGetLastError();
}

template <int MODE>
cudaError_t launch_tma_mode(const StepParams<KSS_T>& p, TmaPlan plan, int ctas,
                            cudaStream_t stream) {
  static bool configured = false;  // the dynamic shared-memory opt-in, once per process
  if (!configured) {
    const cudaError_t e = cudaFuncSetAttribute(step_tma_kernel<KSS_T, MODE>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               int(kTmaSmemBytes));
    if (e != cudaSuccess) return e;
    configured = true;
  }
  step_tma_kernel<KSS_T, MODE><<<ctas, kTmaThreads, kTmaSmemBytes, stream>>>(p, plan);
  return cudaGetLastError();
}

template <>
cudaError_t launch_step_tma<KSS_T>(const StepParams<KSS_T>& p, int mode, TmaPlan plan, int ctas,
                                   cudaStream_t stream) {
  switch (mode) {
    case MODE_PLAIN: return launch_tma_mode<MODE_PLAIN>(p, plan, ctas, stream);
    case MODE_STD: return launch_tma_mode<MODE_STD>(p, plan, ctas, stream);
    default: return cudaErrorInvalidValue;
  }
}

template <>
cudaError_t launch_fixup<KSS_T>(const StepParams<KSS_T>& p, bool pull, int ctas,
                                cudaStream_t stream) {
  if (pull)
    fixup_kernel<KSS_T, true><<<ctas, 256, 0, stream>>>(p);
  else
    fixup_kernel<KSS_T, false><<<ctas, 256, 0, stream>>>(p);
  return cudaGetLastError();
}

#endif  // KSS_STORAGE_HALF

template <>
cudaError_t launch_init_equilibrium<KSS_T>(const double* rho, const double* ux, const double* uy,
                                           KSS_T* f, long long plane, int pitch, int nx, int ny,
                                           const codec_t<KSS_T>& codec, cudaStream_t stream) {
  init_equilibrium_kernel<KSS_T, double><<<helper_grid(nx, ny), 256, 0, stream>>>(
      rho, ux, uy, f, plane, pitch, nx, ny, codec);
  return cudaGetLastError();
}

template <>
cudaError_t launch_init_equilibrium_f32<KSS_T>(const float* rho, const float* ux,
                                               const float* uy, KSS_T* f, long long plane,
                                               int pitch, int nx, int ny,
                                               const codec_t<KSS_T>& codec, cudaStream_t stream) {
  init_equilibrium_kernel<KSS_T, float><<<helper_grid(nx, ny), 256, 0, stream>>>(
      rho, ux, uy, f, plane, pitch, nx, ny, codec);
  return cudaGetLastError();
}

template <>
cudaError_t launch_moments<KSS_T>(const KSS_T* f, long long plane, int pitch, int nx, int ny,
                                  double* rho, double* ux, double* uy,
                                  const codec_t<KSS_T>& codec, cudaStream_t stream) {
  moments_kernel<KSS_T><<<helper_grid(nx, ny), 256, 0, stream>>>(
      f, plane, pitch, nx, ny, rho, ux, uy, codec);
  return cudaGetLastError();
}

template <>
cudaError_t launch_pops_to_dense<KSS_T>(const KSS_T* src, long long plane, int pitch, int nx,
                                        int ny, double* dst, const codec_t<KSS_T>& codec,
                                        cudaStream_t stream) {
  if (dense_vec(dst, nx) == 2)
    pops_to_dense_kernel<KSS_T, 2><<<helper_grid((nx + 1) / 2, ny), 256, 0, stream>>>(src, plane, pitch, nx, ny, dst, codec);
  else
    pops_to_dense_kernel<KSS_T, 1><<<helper_grid(nx, ny), 256, 0, stream>>>(src, plane, pitch, nx, ny, dst, codec);
  return cudaGetLastError();
}

template <>
cudaError_t launch_dense_to_pops<KSS_T>(const double* src, long long plane, int pitch, int nx,
                                        int ny, KSS_T* dst, const codec_t<KSS_T>& codec,
                                        cudaStream_t stream) {
  if (dense_vec(src, nx) == 2)
    dense_to_pops_kernel<KSS_T, 2><<<helper_grid((nx + 1) / 2, ny), 256, 0, stream>>>(src, plane, pitch, nx, ny, dst, codec);
  else
    dense_to_pops_kernel<KSS_T, 1><<<helper_grid(nx, ny), 256, 0, stream>>>(src, plane, pitch, nx, ny, dst, codec);
  return cudaGetLastError();
}

#ifndef KSS_STORAGE_HALF
template <>
cudaError_t launch_pitched_to_dense<KSS_T>(const KSS_T* src, long long plane, int pitch, int nx,
                                           int ny, int nplanes, double* dst, cudaStream_t stream) {
  if (dense_vec(dst, nx) == 2)
    pitched_to_dense_kernel<KSS_T, 2><<<helper_grid((nx + 1) / 2, ny), 256, 0, stream>>>(src, plane, pitch, nx, ny, nplanes, dst);
  else
    pitched_to_dense_kernel<KSS_T, 1><<<helper_grid(nx, ny), 256, 0, stream>>>(src, plane, pitch, nx, ny, nplanes, dst);
  return cudaGetLastError();
}

template <>
cudaError_t launch_dense_to_pitched<KSS_T>(const double* src, long long plane, int pitch, int nx,
                                           int ny, int nplanes, KSS_T* dst, cudaStream_t stream) {
  if (dense_vec(src, nx) == 2)
    dense_to_pitched_kernel<KSS_T, 2><<<helper_grid((nx + 1) / 2, ny), 256, 0, stream>>>(src, plane, pitch, nx, ny, nplanes, dst);
  else
    dense_to_pitched_kernel<KSS_T, 1><<<helper_grid(nx, ny), 256, 0, stream>>>(src, plane, pitch, nx, ny, nplanes, dst);
  return cudaGetLastError();
}
#endif  // KSS_STORAGE_HALF

}  // namespace kss
