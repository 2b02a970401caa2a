// Device-wide primitives: exclusive scan (u32) and stable LSD radix sort.
#pragma once
#include "common.cuh"

namespace fmm {
int exclusive_scan_u32(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* total_dev, DBuf& tmp,
                       cudaStream_t s);
constexpr int kSortPasses = 8;  // 8-bit digits of a 64-bit key
struct SortState {
  uint32_t hist[kSortPasses][256], base[kSortPasses][256];
  uint32_t ticket[kSortPasses];
  int active[kSortPasses], sel[kSortPasses + 1];  // pass q reads buffer sel[q]; the result is in sel[npass]
};
// Scratch of the sort: one per stream that sorts.  A look-back wait polls at
// most `spins` times, to the next 1024 (not at all if negative).  When one runs out, *error
// becomes FMM_E_TIMEOUT and *failed 1: that pass and all later sorts with the
// same *failed leave their output unwritten, so whoever uses it looks there
// first (the words are cleared at the start of an evaluation).
constexpr long long kSweepSpin = 1ll << 24;
struct SortScratch {
  DBuf state, look;
  unsigned epoch = 0;
  int *error = nullptr, *failed = nullptr;
  long long spins = kSweepSpin;
};
// A sort in two halves, for a kernel that makes the keys and counts their
// digits (SortState::hist) itself: sort_begin clears the state; sort_passes
// sorts by npass digits.  all: every pass runs, so the result is in buffer
// npass & 1; else passes over a constant digit are left out and the result is
// in buffer SortState::sel[npass], known on the device alone.
int sort_begin(SortScratch& b, int64_t n, cudaStream_t s);
int sort_passes(SortScratch& b, uint64_t* k0, uint32_t* v0, uint64_t* k1, uint32_t* v1, int64_t n, int npass, bool all,
                cudaStream_t s);
int radix_sort_u64(SortScratch& b, uint64_t* k0, uint32_t* v0, uint64_t* k1, uint32_t* v1, int64_t n, int bits,
                   int* in_second, cudaStream_t s);

// A barrier over the blocks of a cooperative launch.  A wait polls at most
// `spins` times (not at all if negative); on expiry the blocks give up together
// and the barrier returns false.  A block may leave the barrier just before
// another gives up, so what the launch wrote is good only if abort is still 0
// when it has ended: whoever uses it looks there first.
struct GridBar {
  uint32_t count, gen, abort;
};
constexpr long long kGridSpin = 1ll << 24;

#ifdef __CUDACC__
// Adds the warp's keys to the block's digit counts h[npass][256] (all lanes
// call it; a digit that is the same in every lane takes one atomic).
__device__ __forceinline__ void count_digits(uint32_t* h, uint64_t key, bool live, int npass) {
  const unsigned m = __ballot_sync(0xffffffffu, live);
  if (!m) return;
  const int lead = __ffs(m) - 1;
  for (int q = 0; q < npass; ++q) {
    const int d = (int)((key >> (8 * q)) & 0xff);
    const int d0 = __shfl_sync(0xffffffffu, d, lead);
    if (__all_sync(0xffffffffu, !live || d == d0)) {
      if ((int)(threadIdx.x & 31) == lead) atomicAdd(&h[q * 256 + d0], (uint32_t)__popc(m));
    } else if (live) {
      atomicAdd(&h[q * 256 + d], 1u);
    }
  }
}
__device__ __forceinline__ void clear_digits(uint32_t* h, int npass) {
  for (int i = threadIdx.x; i < npass * 256; i += blockDim.x) h[i] = 0u;
  __syncthreads();
}
__device__ __forceinline__ void flush_digits(const uint32_t* h, int npass, uint32_t* hist) {
  __syncthreads();
  for (int i = threadIdx.x; i < npass * 256; i += blockDim.x)
    if (h[i]) atomicAdd(&hist[i], h[i]);
}

__device__ __forceinline__ bool grid_barrier(GridBar* st, unsigned nblocks, long long spins) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile uint32_t* gen = &st->gen;
    volatile uint32_t* ab = &st->abort;
    const uint32_t g = *gen;
    __threadfence();
    if (atomicAdd(&st->count, 1u) == nblocks - 1) {
      atomicExch(&st->count, 0u);
      __threadfence();
      atomicAdd(&st->gen, 1u);
    } else {
      for (long long i = 0; spins < 0 || *gen == g; ++i) {
        if (*ab) break;
        if (i > spins) {
          atomicExch(&st->abort, 1u);
          break;
        }
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ((volatile uint32_t*)&st->abort)[0] == 0u;
}
#endif
}  // namespace fmm
