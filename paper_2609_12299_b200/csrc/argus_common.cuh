// argus_common.cuh — device helpers shared by the kernels of the CUDA library (sm_100a).
#ifndef ARGUS_COMMON_CUH_
#define ARGUS_COMMON_CUH_

#include <cuda_runtime.h>
#include <stdint.h>

#include "argus.h"
#include "argus_testing.h"

typedef unsigned long long u64;
typedef unsigned int u32;

static_assert(sizeof(argus_event_t) == 16, "event layout");
static_assert(sizeof(argus_interval_t) == 48, "interval layout");
static_assert(sizeof(argus_ambiguity_t) == 32, "ambiguity layout");
static_assert(sizeof(argus_agg_t) == 576, "aggregate layout");
static_assert(sizeof(argus_overlap_t) == 32, "overlap layout");
static_assert(sizeof(argus_status_t) == 64, "status layout");

#define ARGUS_CUDA_TRY(expr)                          \
  do {                                                \
    cudaError_t e__ = (expr);                         \
    if (e__ != cudaSuccess) return ARGUS_ERR_CUDA;    \
  } while (0)

// host-side bookkeeping implemented in argus_api.cu
void argus_count_launch();                                      // one more kernel launched by this library
void argus_count_limit_request();                               // one more call that needed argus_allow_smem
void argus_prof_mark(int slot, cudaStream_t stream, int end);   // CUDA events around a dominant kernel (if enabled)
void argus_prof_suppress(int delta);                            // +1 / -1: event recording off while > 0 (it creates events)
enum { ARGUS_PROF_PAIR = 0, ARGUS_PROF_AGGREGATE = 1, ARGUS_PROF_OVERLAP = 2, ARGUS_PROF_SLOTS = 4 };

// Every kernel of the library is launched so that it may start while the one before it on the stream runs out
// (programmatic dependent launch), and begins with argus_kernel_begin(): nothing is read or written before everything
// earlier on the stream is complete. Short kernels let the next one be set up as soon as all their blocks run, long ones
// (argus_kernel_begin_long) only when their blocks are done: blocks that wait beside them cost them time (a 2.4 ms pairing
// kernel on 96 streams took 3.2 ms with the next kernels' blocks resident). A call is a chain of short kernels around one or
// two long ones; this takes the set-up of each out of the chain (10 K events: 88 -> 56 us together with 17 -> 8 launches).
template <class... P, class... A>
inline cudaError_t argus_launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A&&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cfg.attrs = attr; cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
  if (e == cudaSuccess) argus_count_launch();
  return e;
}
#define ARGUS_LAUNCH(...) ARGUS_CUDA_TRY(argus_launch(__VA_ARGS__))

// A kernel gets 48 KB of shared memory without asking, its static arrays included (4 KB at most where the size of the dynamic part
// depends on the call). More has to be asked for, and the limit belongs to the kernel and the device, not to a launch: it is
// always set to the same, the most that any call needs, since another host thread may launch the kernel at the same time.
constexpr size_t kPlainDynamicSmem = 43 * 1024;
template <class K>
inline cudaError_t argus_allow_smem(K* kernel, size_t dynamic, size_t most) {
  if (dynamic <= kPlainDynamicSmem) return cudaSuccess;
  argus_count_limit_request();
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

__device__ __forceinline__ void argus_kernel_begin_long() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void argus_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void argus_kernel_begin() {
  argus_launch_next();
  argus_kernel_begin_long();
}

static inline size_t argus_align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// First device-side error wins; the winner also records where it happened.
__device__ __forceinline__ void argus_set_error(argus_status_t* st, u32 code, u32 stream, u64 event) {
  if (atomicCAS(&st->code, 0u, code) == 0u) {
    st->bad_stream = stream;
    st->bad_event = event;
  }
}

// For whoever meets a CTA that is mapped to an SM that does not exist (CTA `met`): names the first such CTA's first stream, so that
// the answer is the same whoever comes first.
static __device__ __noinline__ void argus_report_bad_sm(argus_status_t* st, const u32* cta_sm, u32 num_sms, u32 warps_per_cta, u32 met) {
  if (*reinterpret_cast<volatile u32*>(&st->code)) return;
  u32 c = 0;
  while (c < met && cta_sm[c] < num_sms) ++c;
  argus_set_error(st, ARGUS_ERR_INVALID_ARG, c * warps_per_cta, cta_sm[c]);
}

// Exclusive prefix sum over the threads of a block (blockDim.x <= 1024, multiple of 32).
// `warp_sums` is shared scratch of 33 elements whatever the block's size (the first warp writes a full warp of them). Returns the
// exclusive prefix of `v`; *total receives the block total. Contains __syncthreads().
template <typename T, int N>
__device__ __forceinline__ T argus_block_exclusive_scan(T v, T (&warp_sums)[N], T* total) {
  static_assert(N >= 33, "a full warp's sums and the total");
  const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = (blockDim.x + 31) >> 5;
  T incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    T o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= (u32)d) incl += o;
  }
  if (lane == 31) warp_sums[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    T w = lane < nwarps ? warp_sums[lane] : T(0);
    T wi = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      T o = __shfl_up_sync(0xffffffffu, wi, d);
      if (lane >= (u32)d) wi += o;
    }
    warp_sums[lane] = wi - w;  // exclusive prefix of warp sums
    if (lane == 31) warp_sums[32] = wi;
  }
  __syncthreads();
  const T base = warp_sums[warp];
  *total = warp_sums[32];
  __syncthreads();
  return base + incl - v;
}

#endif  // ARGUS_COMMON_CUH_
