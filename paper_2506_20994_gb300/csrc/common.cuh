// Shared helpers of the CUDA library: status codes, argument checks, the
// element-field loaders for each storage type, and launch bookkeeping.
#pragma once

#include <algorithm>
#include <atomic>
#include <mutex>

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "../../include/axhelm.h"

#define AX_HD __host__ __device__ __forceinline__
#define AX_D __device__ __forceinline__

namespace ax {

// Converts a CUDA launch status into an AX code (never aborts).
inline int launch_status() {
  cudaError_t e = cudaPeekAtLastError();
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return AX_ELAUNCH;
  }
  return AX_OK;
}

inline bool lx_ok(int lx) { return lx >= AX_LX_MIN && lx <= AX_LX_MAX; }

template <typename... P>
inline bool all_nonnull(P... p) {
  bool ok = true;
  ((ok = ok && (p != nullptr)), ...);
  return ok;
}

// Storage -> compute conversion of one element-field value (read past L1: the
// kernels are launched chained, see grid_wait).
template <typename T>
AX_D T ld_cvt(const double *p) { return (T)__ldcg(p); }
template <typename T>
AX_D T ld_cvt(const float *p) { return (T)__ldcg(p); }
template <typename T>
AX_D T ld_cvt(const __nv_bfloat16 *p) { return (T)__bfloat162float(__ldcg(p)); }

// Raises a kernel's dynamic shared-memory limit to `bytes` on the current
// device when that is above the 48 KB default and above what this kernel was
// granted on this device before (the attribute is per device, so a process
// driving several GPUs raises it on each).  `granted` is the caller's table
// for one kernel, zero-initialised; raises are serialised so the recorded
// size only grows.  False if the device refuses or its index is out of range.
constexpr int kMaxDevices = 64;
inline std::mutex &smem_grant_mutex() {
  static std::mutex m;
  return m;
}
// Static shared memory of the kernels (guard record, reduction buffers) stays
// below this; the 48 KB default covers static and dynamic bytes together.
constexpr size_t kStaticSmemMargin = 4 * 1024;
template <typename K>
inline bool grant_smem(K kernel, size_t bytes, std::atomic<size_t> (&granted)[kMaxDevices]) {
  if (bytes + kStaticSmemMargin <= 48 * 1024) return true;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    (void)cudaGetLastError();
    return false;
  }
  if (bytes <= granted[dev].load(std::memory_order_acquire)) return true;
  std::lock_guard<std::mutex> lock(smem_grant_mutex());
  if (bytes <= granted[dev].load(std::memory_order_relaxed)) return true;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) !=
      cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  granted[dev].store(bytes, std::memory_order_release);
  return true;
}

// Launches that may begin while the kernel before them in the stream is still
// running (programmatic dependent launch): what remains of a launch between
// two kernels is then hidden, 2-3 us of a 10 us apply.  Such a kernel calls
// grid_wait() before it reads or writes anything another kernel may touch;
// the wait returns when every earlier kernel of the stream has finished and
// its writes are visible (each of them has waited in turn).  Behind the wait
// it calls grid_go(), which lets the next launch begin: so at most one kernel
// waits behind the running one, and its blocks take only what is free.
// Behind the wait, data that other kernels write is read past L1 (__ldcg, the
// bulk-copy engine): L1 is emptied when a kernel is launched, which here is
// before the kernel in front of it is done, and read-only loads (const
// __restrict__, __ldg) would return lines that kernel's neighbours have
// rewritten since (EopUpd's vectors are the exception).  In front of the wait
// stands only what no kernel of the stream can be writing: the operator
// handle's coefficients, written once, and its prepared geometry (see
// eop_prepare_lx).
AX_D void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
AX_D void grid_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
inline int launch_chained(bool chained, void (*kern)(P...), dim3 grid, unsigned block, size_t smem,
                          cudaStream_t st, A &&...args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = chained ? 1 : 0;  // without: after everything before it in the stream
  if (cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...) != cudaSuccess) {
    (void)cudaGetLastError();
    return AX_ELAUNCH;
  }
  return AX_OK;
}

// Dynamic shared memory for a chained launch of `grid` blocks that need `smem`
// each: raised to an even share of an SM where the grid is less than one full
// wave of two or more blocks per SM, so that no SM takes more than its part.
// Launched early, the blocks otherwise crowd onto the SMs that the kernel in
// front has left free first, and those then run for longer than the rest (fp32
// at lx 13, 400 blocks: 21.0 us unchained, 29.7 chained and crowded, 20.6 so;
// bf16 at lx 9, 440 blocks, 15.0 / 19.8 / 13.5; fp64 at lx 7, 267 blocks, 20.9 /
// 25.1 / 18.7).  occ: this kernel's
// resident blocks per SM, with the block size they hold for.
template <typename K>
inline size_t spread_smem(K kernel, unsigned grid, unsigned block, size_t smem,
                          std::atomic<unsigned> (&occ)[kMaxDevices]) {
  static std::atomic<int> sm_count[kMaxDevices], sm_bytes[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    (void)cudaGetLastError();
    return smem;
  }
  int sms = sm_count[dev].load(std::memory_order_acquire);
  int bytes = sm_bytes[dev].load(std::memory_order_acquire);
  if (sms <= 0 || bytes <= 0) {
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
            cudaSuccess) {
      (void)cudaGetLastError();
      return smem;
    }
    sm_bytes[dev].store(bytes, std::memory_order_release);
    sm_count[dev].store(sms, std::memory_order_release);
  }
  const unsigned part = (grid + sms - 1) / sms;  // blocks per SM if spread evenly
  if (part < 2) return smem;
  unsigned v = occ[dev].load(std::memory_order_acquire);
  if ((v >> 8) != block) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, (int)block, smem) != cudaSuccess) {
      (void)cudaGetLastError();
      return smem;
    }
    v = (block << 8) | (unsigned)std::min(n, 255);
    occ[dev].store(v, std::memory_order_release);
  }
  if (part >= (v & 255u)) return smem;
  // 1 KB a block is the system's, 2 KB covers the kernels' static arrays; what
  // is left over stays below another block's share for up to ten parts
  const size_t share = ((size_t)bytes / part - 3072) / 128 * 128;
  return std::max(smem, share);
}

// Asks the memory system to bring [p, p + bytes) into L2 (bulk copy engine).
// No data is returned.  The bulk unit needs a 16-byte aligned address and
// size; anything else (a caller's offset view) is skipped, since a prefetch
// is only a hint.
AX_D void prefetch_l2(const void *p, unsigned bytes) {
  if (((reinterpret_cast<uintptr_t>(p) | bytes) & 15u) != 0) return;
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// The whole 16-byte granules inside f[first, first + count) towards L2 (at odd
// lx an element's run is not made of them, a block's almost is).
template <typename S>
AX_D void prefetch_span(const S *f, long long first, long long count) {
  const uintptr_t a = (reinterpret_cast<uintptr_t>(f + first) + 15u) & ~(uintptr_t)15u;
  const uintptr_t b = reinterpret_cast<uintptr_t>(f + first + count) & ~(uintptr_t)15u;
  if (b > a) prefetch_l2(reinterpret_cast<const void *>(a), (unsigned)(b - a));
}
// Thread t < 8 of a block: field t (u, then the geometry) of the elements
// [e0, e0 + nel).
template <typename SU, typename S>
AX_D void prefetch_elements(const SU *u, const S *h1, const S *g11, const S *g22, const S *g33,
                            const S *g12, const S *g13, const S *g23, long long e0, long long nel,
                            int n3) {
  const int t = threadIdx.x;
  if (t >= 8 || nel <= 0) return;
  if (t == 0) {
    prefetch_span(u, e0 * n3, nel * n3);
    return;
  }
  const S *f = t == 1 ? g11 : t == 2 ? g22 : t == 3 ? g33 : t == 4 ? g12 : t == 5 ? g13
             : t == 6 ? g23 : h1;
  prefetch_span(f, e0 * n3, nel * n3);
}
// Explicitly rounded arithmetic (never contracted by the compiler).
AX_D double mul_rn(double a, double b) { return __dmul_rn(a, b); }
AX_D float mul_rn(float a, float b) { return __fmul_rn(a, b); }
AX_D double add_rn(double a, double b) { return __dadd_rn(a, b); }
AX_D float add_rn(float a, float b) { return __fadd_rn(a, b); }
AX_D double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
AX_D float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }

}  // namespace ax
