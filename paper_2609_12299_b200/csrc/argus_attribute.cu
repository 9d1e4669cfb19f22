// argus_attribute.cu — PC-to-region mapping counts and ambiguity-aware attribution.
//
//   k_map_counts   : exec records of a mapping-run trace arrive as intervals of the extra region id R whose
//                    parent_region is the innermost active region (pairing did the stack work); this pass adds
//                    their execution counts into counts[owner][pc] (integer atomics: order does not matter).
//   k_attr_tile    : one block per 32 PCs and all rows: column totals, alpha, entropy, and the block's share of the lifted
//                    metric of every row;
//   k_attr_finish  : mhat[row] = sum of the blocks' shares, in a fixed order.
#include "argus_common.cuh"

namespace {

constexpr int kAttrThreads = 256;
constexpr u32 kAttrWarps = kAttrThreads / 32;
constexpr u32 kAttrRows = 400;        // rows of 32 counts a block keeps in shared memory (100 KB)
constexpr u32 kMapSlots = 2048;       // shared-memory cache of (owner, pc) cells per block
constexpr u32 kMapEmpty = 0xffffffffu;
constexpr u32 kMapSmall = 1u << 12;   // executions a cache slot takes at a time ...
constexpr u32 kMapFlush = 1u << 19;   // ... and records after which the cache is emptied: their product stays below 2^32

// A mapping run touches few of the (R + 1) x P cells and touches them very often, so each block gathers
// its additions in a small direct-mapped table in shared memory (cell index -> 32-bit sum) and adds the table
// to the global counts at the end; a cell whose slot is taken by another cell, or a count of kMapSmall and more, goes to the
// global counts directly. A slot's key is looked at before it is claimed and the add returns nothing: a warp's lanes hit few
// cells, and what they do to one is done one lane after the other. 57.6 M intervals, 808 cells: 682 us with a compare-and-swap
// and a returning 64-bit add per record, 433 us this way (6.4 TB/s of records).
__global__ void __launch_bounds__(256) k_map_counts(const argus_interval_t* intervals, const u64* interval_offsets,
                                                    u32 num_streams, u32 exec_region, u32 num_pcs, u64* counts,
                                                    argus_status_t* status, int use_cache) {
  argus_kernel_begin_long();
  __shared__ u32 keys[kMapSlots];
  __shared__ u32 sums[kMapSlots];
  for (u32 i = threadIdx.x; i < kMapSlots; i += blockDim.x) { keys[i] = kMapEmpty; sums[i] = 0; }
  __syncthreads();
  const u64 lo = interval_offsets[0], hi = interval_offsets[num_streams];
  u32 seen = 0;  // records of this block since the cache was emptied
  for (u64 base = lo + (u64)blockIdx.x * blockDim.x; base < hi; base += (u64)gridDim.x * blockDim.x) {
    const u64 i = base + threadIdx.x;
    if (i < hi) {
      const uint4* p = reinterpret_cast<const uint4*>(intervals + i);
      const uint2 k2 = __ldg(reinterpret_cast<const uint2*>(p) + 1), rc = __ldg(reinterpret_cast<const uint2*>(p + 1) + 1);
      const u32 parent = __ldg(reinterpret_cast<const u32*>(p + 2) + 1);
      const u64 k = (u64)k2.x | ((u64)k2.y << 32);
      const u32 pc = rc.y;
      if (rc.x != exec_region) {
      } else if (pc >= num_pcs) {
        argus_set_error(status, ARGUS_ERR_INVALID_ARG, 0, i);
      } else if (k) {
        const u32 owner = parent < exec_region ? parent : exec_region;  // no parent, or a malformed nesting of exec records
        const u64 cell = (u64)owner * num_pcs + pc;
        bool cached = false;
        if (use_cache && k < kMapSmall) {
          const u32 key = (u32)cell;
          const u32 slot = (key * 2654435761u) >> 21;  // 11 bits
          u32 have = *reinterpret_cast<volatile u32*>(&keys[slot]);
          if (have == kMapEmpty) { have = atomicCAS(&keys[slot], kMapEmpty, key); if (have == kMapEmpty) have = key; }
          cached = have == key;
          if (cached) atomicAdd(&sums[slot], (u32)k);
        }
        if (!cached) atomicAdd(counts + cell, k);
      }
    }
    seen += blockDim.x;
    if (seen >= kMapFlush) {  // uniform
      __syncthreads();
      for (u32 j = threadIdx.x; j < kMapSlots; j += blockDim.x)
        if (sums[j]) { atomicAdd(counts + keys[j], (u64)sums[j]); sums[j] = 0; }
      seen = 0;
      __syncthreads();
    }
  }
  __syncthreads();
  for (u32 i = threadIdx.x; i < kMapSlots; i += blockDim.x)
    if (sums[i]) atomicAdd(counts + keys[i], (u64)sums[i]);
}

// One lane per PC, rows shared out among the warps. The block's counts are read once and kept (kAttrRows rows at most, else read
// again): bound by HBM, counts in and alpha out (203 rows x 70,560 PCs: 63 us with the sums, 222 us in three kernels that read the
// counts three times). Sums over rows and over PCs are taken in an order that the shape alone fixes, so the
// same bits come out every run.
__global__ void __launch_bounds__(kAttrThreads) k_attr_tile(const u64* counts, u32 num_rows, u32 num_pcs, const double* metric,
                                                            double* entropy, double* alpha, u32 num_blocks, double* partial) {
  argus_kernel_begin_long();
  extern __shared__ __align__(16) u64 held[];  // [num_rows][32]
  __shared__ u64 total_of[kAttrWarps][32];
  __shared__ double entropy_of[kAttrWarps][32];
  const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5, p = blockIdx.x * 32 + lane;
  const bool in = p < num_pcs, keep = num_rows <= kAttrRows;
  u64 total = 0;
#pragma unroll 8
  for (u32 r = warp; r < num_rows; r += kAttrWarps) {
    const u64 n = in ? __ldg(counts + (size_t)r * num_pcs + p) : 0ull;
    if (keep) held[r * 32 + lane] = n;
    total += n;
  }
  total_of[warp][lane] = total;
  __syncthreads();
  total = 0;
#pragma unroll
  for (u32 w = 0; w < kAttrWarps; ++w) total += total_of[w][lane];
  const double m = in ? metric[p] : 0.0;
  double h = 0.0;
#pragma unroll 4
  for (u32 r = warp; r < num_rows; r += kAttrWarps) {
    const u64 n = keep ? held[r * 32 + lane] : in ? __ldg(counts + (size_t)r * num_pcs + p) : 0ull;
    const bool some = n != 0 && total != 0;
    double a = 0.0, part = 0.0;
    if (some) {
      a = (double)n / (double)total;
      if (a > 0.0) h -= a * log(a);
      part = a * m;
    }
    if (alpha && in) __stcs(alpha + (size_t)r * num_pcs + p, a);
    if (__any_sync(0xffffffffu, some)) {
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) part += __shfl_down_sync(0xffffffffu, part, d);
    }
    if (lane == 0) partial[(size_t)r * num_blocks + blockIdx.x] = part;
  }
  entropy_of[warp][lane] = h;
  __syncthreads();
  if (warp == 0 && in) {
    h = 0.0;
#pragma unroll
    for (u32 w = 0; w < kAttrWarps; ++w) h += entropy_of[w][lane];
    entropy[p] = h;
  }
}

__global__ void __launch_bounds__(kAttrThreads) k_attr_finish(const double* partial, u32 num_blocks, double* mhat) {
  argus_kernel_begin_long();
  __shared__ double sh[kAttrWarps];
  const u32 r = blockIdx.x;
  double s = 0.0;
  for (u32 b = threadIdx.x; b < num_blocks; b += kAttrThreads) s += partial[(size_t)r * num_blocks + b];
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    s = 0.0;
    for (u32 w = 0; w < kAttrWarps; ++w) s += sh[w];
    mhat[r] = s;
  }
}

struct AttrLayout { size_t total; u32 blocks; };

AttrLayout attr_layout(uint32_t num_rows, uint32_t num_pcs) {
  AttrLayout L;
  L.blocks = (num_pcs + 31) / 32;
  L.total = argus_align_up((size_t)num_rows * L.blocks * 8 + 8, 256);
  return L;
}

}  // namespace

extern "C" int argus_map_pc_counts(const argus_interval_t* intervals, const uint64_t* interval_offsets,
                                   uint32_t num_streams, uint32_t exec_region, uint32_t num_pcs, uint64_t* counts,
                                   argus_status_t* status, void* cuda_stream) {
  if (!interval_offsets || !counts || !status || num_pcs == 0 || exec_region >= ARGUS_MAX_REGIONS) return ARGUS_ERR_INVALID_ARG;
  if (((uintptr_t)intervals & 15) || ((uintptr_t)counts & 7)) return ARGUS_ERR_INVALID_ARG;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  ARGUS_CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(argus_status_t), stream));
  ARGUS_CUDA_TRY(cudaMemsetAsync(counts, 0, ((size_t)exec_region + 1) * num_pcs * sizeof(uint64_t), stream));
  if (num_streams == 0) return ARGUS_OK;
  const int use_cache = ((uint64_t)exec_region + 1) * num_pcs < 0xffffffffull;  // cell indices must fit the 32-bit keys
  ARGUS_LAUNCH(k_map_counts, 148 * 8, 256, 0, stream, intervals, (const u64*)interval_offsets, num_streams, exec_region,
               num_pcs, (u64*)counts, status, use_cache);
  return ARGUS_OK;
}

extern "C" size_t argus_attribute_workspace_bytes(uint32_t num_rows, uint32_t num_pcs) {
  return attr_layout(num_rows, num_pcs).total;
}

extern "C" int argus_attribute(const uint64_t* counts, uint32_t num_rows, uint32_t num_pcs, const double* metric,
                               double* mhat, double* entropy, double* alpha, void* workspace, size_t workspace_bytes,
                               void* cuda_stream) {
  if (!counts || !metric || !mhat || !entropy || !workspace || num_rows == 0 || num_pcs == 0) return ARGUS_ERR_INVALID_ARG;
  if (num_rows > 65535) return ARGUS_ERR_INVALID_ARG;
  if (((uintptr_t)workspace & 255) || ((uintptr_t)counts & 7) || ((uintptr_t)metric & 7) || ((uintptr_t)mhat & 7) ||
      ((uintptr_t)entropy & 7) || ((uintptr_t)alpha & 7))
    return ARGUS_ERR_INVALID_ARG;
  const AttrLayout L = attr_layout(num_rows, num_pcs);
  if (workspace_bytes < L.total) return ARGUS_ERR_WORKSPACE;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  double* partial = (double*)workspace;
  const size_t smem = num_rows <= kAttrRows ? (size_t)num_rows * 32 * 8 : 0;
  ARGUS_CUDA_TRY(argus_allow_smem(k_attr_tile, smem, (size_t)kAttrRows * 32 * 8));
  ARGUS_LAUNCH(k_attr_tile, L.blocks, kAttrThreads, smem, stream, (const u64*)counts, num_rows, num_pcs, metric, entropy, alpha, L.blocks,
               partial);
  ARGUS_LAUNCH(k_attr_finish, num_rows, kAttrThreads, 0, stream, (const double*)partial, L.blocks, mhat);
  return ARGUS_OK;
}
