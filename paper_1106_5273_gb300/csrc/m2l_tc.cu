// M2L on the 5th-generation tensor cores (tcgen05), BF16x3 split products
// with FP32 accumulation in tensor memory (Sec. 3.1 M2L, batched per
// translation vector).
//
// A step applies one translation operator T (P x P, P = p^2) to the
// multipoles of the source cells paired with a tile of target cells.  Cells as
// MMA rows (k_m2l_cells), 42 to a tile:
//   D[128 x N] += B[128 x K] . T^T[K x N],  row (slot, comp) of B = M~ of the
// slot's source for that potential component (zero if the slot has no source
// under this translation; rows 126 and 127 are unused), N = P rounded up to 16.
// The cells are the rows and the coefficients the columns: P need not fill the
// 128 rows of an MMA (with the operator as the 128-row operand half of them
// were idle at p = 8, and P = 144 took a second block of 128 rows for its last
// 16).  T = T_hi + T_lo and B = B_hi + B_lo in BF16; D accumulates T_hi B_hi +
// T_hi B_lo + T_lo B_hi (the lo.lo term is below FP32 resolution of the sum).
// The K chunks from m2l_split_chunks on (source degrees 8 and up) take
// T_hi B_hi only: under the MAC their terms are at most theta^8 / (1 - theta)
// of the leading one, which keeps the 2^-8 error of one BF16 product there
// under 7e-6 for theta <= 0.42.  D lives in TMEM for all steps of an item.
//
// A stage is one step and one 64-wide K chunk: the operator (rows pre-swizzled
// in global memory in the 128-byte-swizzle K-major layout) arrives by 1-D bulk
// copies on mbarrier fullA, issued by a warp of their own; 8 producer warps
// load the rows of B (128 B each) into registers, store them in the same swizzle
// once the buffer is free and arrive on fullB; one thread issues the MMAs and
// commits them to the empty barrier.  Every wait is bounded; on expiry the kernel records
// FMM_E_TIMEOUT, waits (bounded) for its own copies, frees its tensor memory
// and returns.
//
// With 64 < P <= 128 the roles are the other way round (k_m2l_rows: operator
// rows as MMA rows, 64 cells x 3 components as 192 columns): P fills most of
// the 128 rows, and an MMA costs about 20-40 cycles on top of N / 2, so fewer
// and wider MMAs win (Taylor-Green 128^3, p = 10: 4.09 ms against 4.74 with the
// cells as rows).  Elsewhere the cells win: Plummer 1,000,000 at p = 12 38.3 ->
// 26.3 ms, Plummer 30,011 at p = 8 0.89 -> 0.56 ms (one stage of cp.async gathers; with the
// gathers in registers while the buffer is still read, 23.9 -> 20.1 and 0.54).
#include <cuda_bf16.h>

#include <algorithm>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

constexpr int kRows = 128;                  // rows of D: (slot, component), 3 kTileCells of them used
constexpr int kProducerWarps = 8;
constexpr int kThreads = (kProducerWarps + 2) * 32;  // + MMA warp, + operator copy warp
constexpr int kMmaWarp = kProducerWarps, kCopyWarp = kProducerWarps + 1;
constexpr uint32_t kBBytes = kRows * 128;   // one K chunk of the gathered rows, hi or lo
constexpr long long kSpin = 1ll << 24;
static_assert(3 * kTileCells <= kRows, "a tile's rows fit one MMA");
// operator-row form
constexpr int kColsB = 3 * kTileRows;                       // 192 columns
constexpr int kRowStages = 1;                               // pipeline stages per CTA (the loop also runs with 2)
constexpr int kProducers = kProducerWarps * 32;
constexpr int kRowThreads = kProducers + 32;                // + control warp
constexpr uint32_t kRowABytes = 128 * 128;                  // 128 rows x 64 bf16
constexpr uint32_t kColBytes = kColsB * 128;                // 192 rows x 64 bf16
constexpr uint32_t kRowStageBytes = 2 * kRowABytes + 2 * kColBytes;  // 80 KB
constexpr uint32_t kBarOff = kRowStages * kRowStageBytes;
constexpr int kRowTmemCols = 256;
constexpr int kRowLd = 128;                                 // coefficients per row of its partial sums
constexpr int kGather = (2 * kColsB * 8) / kProducers;      // 16-byte items per producer thread (12)
// Work items of one-problem plans: S = steps / kItemTarget (about four items
// per concurrent CTA, 2 per SM x 152 SMs) clamped to [kItemMinSteps,
// kItemMaxSteps], then raised if needed so that there are at most kItemsMax
// items.  The upper clamp is for accuracy as much as for balance: the FP32
// accumulation of the tensor memory over a whole tile's steps (thousands of
// MMAs into one sum) measured 4x the M2L error of sums over at most a few
// hundred steps added in FP32 afterwards.
constexpr int64_t kItemMinSteps = 64;
constexpr int64_t kItemMaxSteps = 128;
constexpr int64_t kItemTarget = 4 * 2 * 152;
constexpr int64_t kItemsMax = 1 << 15;
constexpr int64_t kItemSortSteps = 1 << 18;  // the sort costs 0.04 ms: below, it is not worth it

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint32_t bar, uint32_t tx) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(bar),
               "r"(tx)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: false when the limit is reached (the caller aborts).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort,
                                          long long limit = kSpin) {
  for (long long i = 0; i < limit; ++i) {
    if (mbar_try(bar, parity)) return true;
    if ((i & 1023) == 1023 && *abort) return false;
  }
  *abort = 1;
  return false;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 B apart (SBO), descriptor version 1.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
// Instruction descriptor: D f32, both operands K-major, M = 128, N columns;
// kind::f16 with A and B BF16 (format 1), kind::tf32 with A and B TF32 (format 2).
__device__ __forceinline__ uint32_t idesc(int kind, int N) {
  const uint32_t fmt = kind ? 2u : 1u;
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
}

__device__ __forceinline__ uint32_t kRowIdesc(int kind) { return idesc(kind, kColsB); }

template <int KIND>
__device__ __forceinline__ void umma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  if (KIND == 0)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
            tmem),
        "l"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(
            tmem),
        "l"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void store16(uint32_t dst, const uint4& v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

// ---- Cell rows (P <= 64 or P > 128).
// KIND 0: BF16 operands (64 per 128-byte row, K step 16); KIND 1: TF32 (32
// per row, K step 8).  Tb / Mb hold 128-byte rows: a K chunk of one operator
// row or one (cell, hi/lo, component) multipole row.  Operators: [slot][hi/lo]
// [K chunk][N rows].
// CTA x runs work item x (tile, first step, end step, partial slot) of *nitems:
// a tile's steps in runs of at most S; an item that is its tile's only one
// writes the local expansions (slot -1), the others write D to their partial
// slot, summed by k_m2l_combine.  items == nullptr (batches): CTA x runs the
// steps of range range0 + x, i.e. of one key bucket of one tile, into slot x.
// CTAS per SM: three up to N = 64; two with N > 128, whose 256 tensor-memory
// columns admit no more, which leaves the gathers 78 registers a thread instead
// of 64 (Plummer 1,000,000 at p = 12 22.9 -> 20.1 ms; at p = 8 two CTAs are 20%
// slower than three).
template <int KIND, int CTAS>
__global__ void __launch_bounds__(kThreads, CTAS)
    k_m2l_cells(const int2* __restrict__ tile_range, int range0, const int4* __restrict__ items,
             const uint32_t* __restrict__ nitems, const uint32_t* __restrict__ order, const int* __restrict__ tfirst, const int* __restrict__ st_slot,
             const int* __restrict__ st_src, const uint8_t* __restrict__ Tb, const uint8_t* __restrict__ Mb, int P,
             int N, int nkc, int nkc3, int ksteps_last, uint32_t tmem_cols,
             const int* __restrict__ tcell, float* __restrict__ L, float* __restrict__ partial,
             int* __restrict__ flag) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  int tile, pslot;
  int2 rg;
  if (items) {
    if (blockIdx.x >= *nitems) return;  // beyond the items of this evaluation
    const int4 w = items[order ? order[blockIdx.x] : blockIdx.x];
    tile = w.x;
    rg = make_int2(w.y, w.z);
    pslot = w.w;
  } else {
    rg = tile_range[range0 + blockIdx.x];
    tile = (range0 + (int)blockIdx.x) / kKeyBuckets;
    pslot = (int)blockIdx.x;
  }
  if (rg.y <= rg.x) return;  // no M2L here: the whole CTA leaves before any barrier
  constexpr int NB = 2;  // blocks of each operand per stage: hi and lo
  const uint32_t abytes = (uint32_t)N * 128u;
  const uint32_t stage_bytes = (uint32_t)NB * (kBBytes + abytes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + stage_bytes);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 4);
  volatile int* abort = reinterpret_cast<volatile int*>(bars + 5);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t fullA = smem_u32(bars), fullB = fullA + 8u, empty = fullA + 16u, done = fullA + 24u;
  if (threadIdx.x == 0) {
    mbar_init(fullA, 1);
    mbar_init(fullB, kProducerWarps);
    mbar_init(empty, 1);
    mbar_init(done, 1);
    *abort = 0;
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int niter = (rg.y - rg.x) * nkc;

  if (warp < kProducerWarps) {
    // ---- producers: thread t moves 16-byte chunk j = t % 8 of rows t/8 + 32 q
    // (q = 0..3), i.e. of component row % 3 of the source in slot row / 3, hi and
    // lo; a step's rows are loaded before its buffer is waited for
    const int j = threadIdx.x & 7, r0 = threadIdx.x >> 3;
    int nxt[4];
    // pieces of the buffer that hold a source's values: a piece without a source
    // is cleared only if it does (adaptive trees pair few of a tile's cells
    // under one translation)
    uint32_t held = 0xffu;
    auto sources = [&](int st) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = r0 + 32 * q;
        nxt[q] = r < 3 * kTileCells ? __ldg(st_src + (size_t)st * kTileCells + r / 3) : -1;
      }
    };
    sources(rg.x);
    const uint32_t dst = sbase + (uint32_t)r0 * 128u + (uint32_t)((j ^ (r0 & 7)) << 4);
    int st = rg.x, kc = 0;
    uint32_t ph = 0u;
    for (int it = 0; it < niter; ++it) {
      const bool need = j < 2 * (kc == nkc - 1 ? ksteps_last : 4), lo = kc < nkc3;
      uint4 v[8];
      uint32_t live = 0u;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (!need || nxt[q] < 0) continue;
        const uint8_t* p = Mb + ((((size_t)nxt[q] * 2) * 3 + (r0 + 32 * q) % 3) * nkc + kc) * 128 + j * 16;
        v[q] = __ldg(reinterpret_cast<const uint4*>(p));
        if (lo) v[4 + q] = __ldg(reinterpret_cast<const uint4*>(p + (size_t)3 * nkc * 128));
        live |= (lo ? 0x11u : 0x1u) << q;
      }
      if (++kc == nkc) {
        kc = 0;
        if (++st < rg.y) sources(st);
      }
      // the warp goes on or gives up as one
      if (!__all_sync(0xffffffffu, mbar_wait(empty, ph ^ 1u, abort))) break;
      ph ^= 1u;
      const uint32_t clear = need ? held & ~live & (lo ? 0xffu : 0x0fu) : 0u;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const uint32_t at = dst + (uint32_t)(q >> 2) * kBBytes + (uint32_t)(q & 3) * 4096u;
        if (live & (1u << q)) store16(at, v[q]);
        else if (clear & (1u << q)) store16(at, make_uint4(0u, 0u, 0u, 0u));
      }
      held = (held & ~clear) | live;
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(fullB);
    }
  } else if (warp == kCopyWarp) {
    // ---- operator copies
    if (lane == 0) {
      int issued = 0, st = rg.x, kc = 0;
      bool ok = true;
      for (int it = 0; it < niter; ++it) {
        if (!mbar_wait(empty, ((uint32_t)it & 1u) ^ 1u, abort)) {
          ok = false;
          break;
        }
        const uint8_t* T = Tb + (size_t)st_slot[st] * 2 * nkc * abytes;
        const uint32_t a0 = sbase + (uint32_t)NB * kBBytes;
        const bool lo = kc < nkc3;  // chunks from nkc3 on take the hi.hi product only
        mbar_arrive_tx(fullA, lo ? 2u * abytes : abytes);
        bulk_g2s(a0, T + (size_t)kc * abytes, abytes, fullA);
        if (lo) bulk_g2s(a0 + abytes, T + (size_t)(nkc + kc) * abytes, abytes, fullA);
        issued = it + 1;
        if (++kc == nkc) {
          kc = 0;
          ++st;
        }
      }
      if (!ok && issued) {  // let the copies in flight land before the CTA exits
        volatile int never = 0;
        mbar_wait(fullA, (uint32_t)(issued - 1) & 1u, &never);
      }
    }
  } else if (lane == 0) {
    // ---- MMA issue
    const uint32_t id = idesc(KIND, N);
    int kc = 0;
    bool ok = true;
    for (int it = 0; it < niter; ++it) {
      const uint32_t ph = (uint32_t)it & 1u;
      if (!mbar_wait(fullA, ph, abort) || !mbar_wait(fullB, ph, abort)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t b_hi = sbase, b_lo = b_hi + kBBytes;
      const uint32_t a_hi = b_hi + (uint32_t)NB * kBBytes, a_lo = a_hi + abytes;
      const int ks = (kc == nkc - 1) ? ksteps_last : 4;
      const bool three = kc < nkc3;
      for (int kk = 0; kk < ks; ++kk) {
        const uint32_t off = (uint32_t)kk * 32u;
        umma<KIND>(tmem, sw128_desc(b_hi + off), sw128_desc(a_hi + off), id, (it > 0 || kk > 0) ? 1u : 0u);
        if (three) {
          umma<KIND>(tmem, sw128_desc(b_lo + off), sw128_desc(a_hi + off), id, 1u);
          umma<KIND>(tmem, sw128_desc(b_hi + off), sw128_desc(a_lo + off), id, 1u);
        }
      }
      if (++kc == nkc) kc = 0;
      umma_commit(empty);
    }
    umma_commit(done);
    if (!ok) {
      // our MMAs finish before the tensor memory is freed
      *abort = 1;
      volatile int never = 0;
      mbar_wait(done, 0u, &never);
      atomicExch(flag, FMM_E_TIMEOUT);
    }
  }
  // ---- epilogue: warps 0-3 own TMEM lanes 0-127 (row = slot, component)
  if (warp < 4) {
    if (__all_sync(0xffffffffu, mbar_wait(done, 0u, abort))) {
      tc_fence_after();
      const int first = tfirst[tile];
      const int ncell = tfirst[tile + 1] - first;
      const int row = warp * 32 + lane;
      const bool live = row < 3 * ncell;
      float* dst = pslot >= 0 ? partial + ((size_t)pslot * kRows + row) * N
                              : L + ((size_t)(live ? tcell[first + row / 3] : 0) * 3 + row % 3) * P;
      const int cols = pslot >= 0 ? N : P;
      const bool vec = (cols & 3) == 0;  // rows of whole 16-byte groups
#pragma unroll 1
      for (int cb = 0; cb < N; cb += 16) {
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)cb, v);
        if (!live) continue;
        if (vec) {
#pragma unroll
          for (int i = 0; i < 16; i += 4)
            if (cb + i < cols) *reinterpret_cast<float4*>(dst + cb + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (cb + i < cols) dst[cb + i] = v[i];
        }
      }
    } else {
      atomicExch(flag, FMM_E_TIMEOUT);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
  }
}

// ---- Operator rows (64 < P <= 128): D[128 x 192] += T[128 x K] . B[K x 192],
// column (comp, slot) = M~ of the slot's source.  One stage per CTA and two
// CTAs per SM (81 KB, a whole step 111 KB at p = 10, and 256 TMEM columns each):
// while one CTA waits on its gathers and barriers the other's MMAs keep the
// tensor pipe busy.  The producers load a stage's rows into registers before
// they wait for its buffer.
template <int KIND, bool M2>
__global__ void __launch_bounds__(kRowThreads, 2)
    k_m2l_rows(const int2* __restrict__ tile_range, int range0, const int4* __restrict__ items,
             const uint32_t* __restrict__ nitems, const uint32_t* __restrict__ order, const int* __restrict__ tfirst, const int* __restrict__ st_slot, const int* __restrict__ st_src,
             const uint8_t* __restrict__ Tb, const uint8_t* __restrict__ Mb, int P, int N, int nkc, int nkc3,
             int ksteps_last, const int* __restrict__ tcell, float* __restrict__ L, float* __restrict__ partial,
             int* __restrict__ flag) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  int tile, pslot;
  int2 rg;
  if (items) {
    if (blockIdx.x >= *nitems) return;  // beyond the items of this evaluation
    const int4 w = items[order ? order[blockIdx.x] : blockIdx.x];
    tile = w.x;
    rg = make_int2(w.y, w.z);
    pslot = w.w;
  } else {
    rg = tile_range[range0 + blockIdx.x];
    tile = (range0 + (int)blockIdx.x) / kKeyBuckets;
    pslot = (int)blockIdx.x;
  }
  if (rg.y <= rg.x) return;  // no M2L here: the whole CTA leaves before any barrier
  // Only the operator rows below P are copied (whole 8-row swizzle groups):
  // the rows above feed only output rows that the epilogue never stores.
  const uint32_t abytes = (uint32_t)((P + 7) & ~7) * 128u;
  const size_t chunk = (size_t)N * 128;  // bytes of one (operator, hi/lo, K chunk) block
  // M2 (two K chunks, the second with one product, P <= 128): the stage holds
  // a whole step, A buffers of abytes (chunk 0 hi, chunk 0 lo, chunk 1 hi;
  // the MMA's rows past arows read the next buffer and feed discarded output
  // rows) followed by the B buffers (chunk 0 hi, chunk 0 lo, chunk 1 hi).
  const uint32_t abuf = M2 ? abytes : kRowABytes;
  const uint32_t stage_bytes = M2 ? 3u * abuf + 3u * kColBytes : kRowStageBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + stage_bytes);
  // bars: fullA[2], fullB[2], empty[2], done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 8);
  volatile int* abort = reinterpret_cast<volatile int*>(bars + 9);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = smem_u32(bars);
  auto fullA = [&](int s) { return bar0 + 8u * (uint32_t)s; };
  auto fullB = [&](int s) { return bar0 + 8u * (uint32_t)(2 + s); };
  auto empty = [&](int s) { return bar0 + 8u * (uint32_t)(4 + s); };
  const uint32_t done = bar0 + 8u * 6u;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRowStages; ++s) {
      mbar_init(fullA(s), 1);
      mbar_init(fullB(s), kProducers);
      mbar_init(empty(s), 1);
    }
    mbar_init(done, 1);
    *abort = 0;
    fence_mbar_init();
  }
  if (warp == kProducerWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kRowTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int niter = M2 ? (rg.y - rg.x) : (rg.y - rg.x) * nkc;

  if (M2 && warp < kProducerWarps) {
    // ---- producers, whole step per stage: 16-byte chunk j = t % 8 of rows
    // n = t/8 + 32k (k = 0..5) of the three B buffers
    const int j = threadIdx.x & 7, r0 = threadIdx.x >> 3;
    constexpr int G = 18;
    for (int it = 0; it < niter; ++it) {
      const uint32_t ph = (uint32_t)it & 1u;
      const int st = rg.x + it;
      const int srcA = __ldg(st_src + (size_t)st * kTileRows + r0), srcB = __ldg(st_src + (size_t)st * kTileRows + r0 + 32);
      uint4 v[G];
#pragma unroll
      for (int q = 0; q < G; ++q) {
        const int bsel = q / 6, k = q % 6;  // buffer: chunk 0 hi, chunk 0 lo, chunk 1 hi
        const int h = bsel == 1 ? 1 : 0, kc = bsel == 2 ? 1 : 0;
        const int src = (k & 1) ? srcB : srcA;
        v[q] = make_uint4(0u, 0u, 0u, 0u);
        if (src >= 0)
          v[q] = __ldg(reinterpret_cast<const uint4*>(Mb + ((((size_t)src * 2 + h) * 3 + (k >> 1)) * nkc + kc) * 128) +
                       j);
      }
      if (!mbar_wait(empty(0), ph ^ 1u, abort)) break;
#pragma unroll
      for (int q = 0; q < G; ++q) {
        const int bsel = q / 6, n = r0 + 32 * (q % 6);
        *reinterpret_cast<uint4*>(smem + 3 * abuf + bsel * kColBytes + n * 128 + ((j ^ (n & 7)) << 4)) = v[q];
      }
      fence_proxy_async();
      mbar_arrive(fullB(0));
    }
  } else if (M2 && lane == 0 && warp == kProducerWarps) {
    // ---- control thread, whole step per stage: three operator copies, then
    // 12 MMAs for chunk 0 (three products) and ksteps_last for chunk 1 (hi x hi)
    int issued = 0, consumed = 0;
    bool ok = true;
    for (int it = 0; it < niter; ++it) {
      const uint32_t ph = (uint32_t)it & 1u;
      if (!mbar_wait(empty(0), ph ^ 1u, abort)) {
        ok = false;
        break;
      }
      const size_t key = (size_t)st_slot[rg.x + it];
      const uint32_t a0 = sbase;
      mbar_arrive_tx(fullA(0), 3u * abytes);
      bulk_g2s(a0, Tb + ((key * 2 + 0) * nkc + 0) * chunk, abytes, fullA(0));
      bulk_g2s(a0 + abuf, Tb + ((key * 2 + 1) * nkc + 0) * chunk, abytes, fullA(0));
      bulk_g2s(a0 + 2 * abuf, Tb + ((key * 2 + 0) * nkc + 1) * chunk, abytes, fullA(0));
      issued = it + 1;
      if (!mbar_wait(fullA(0), ph, abort)) {
        ok = false;
        break;
      }
      consumed = it + 1;
      if (!mbar_wait(fullB(0), ph, abort)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t b0 = a0 + 3 * abuf;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const uint32_t off = (uint32_t)kk * 32u;
        umma<KIND>(tmem, sw128_desc(a0 + off), sw128_desc(b0 + off), kRowIdesc(KIND), (it > 0 || kk > 0) ? 1u : 0u);
        umma<KIND>(tmem, sw128_desc(a0 + off), sw128_desc(b0 + kColBytes + off), kRowIdesc(KIND), 1u);
        umma<KIND>(tmem, sw128_desc(a0 + abuf + off), sw128_desc(b0 + off), kRowIdesc(KIND), 1u);
      }
      for (int kk = 0; kk < ksteps_last; ++kk) {
        const uint32_t off = (uint32_t)kk * 32u;
        umma<KIND>(tmem, sw128_desc(a0 + 2 * abuf + off), sw128_desc(b0 + 2 * kColBytes + off), kRowIdesc(KIND), 1u);
      }
      umma_commit(empty(0));
    }
    if (ok) {
      umma_commit(done);
    } else {
      *abort = 1;
      volatile int never = 0;
      for (int it = consumed; it < issued; ++it) mbar_wait(fullA(0), (uint32_t)it & 1u, &never);
      umma_commit(done);
      mbar_wait(done, 0u, &never);
      atomicExch(flag, FMM_E_TIMEOUT);
    }
  } else if (M2) {
    // the other lanes of the control warp go straight to the teardown
  } else if (warp < kProducerWarps) {
    // ---- producers: thread t stores 16-byte chunk j = t % 8 of rows n = t/8 + 32k
    // (k = 0..5) of both halves, i.e. of the sources in slots t/8 and t/8 + 32;
    // the rows are loaded before the stage's buffer is waited for.
    static_assert(kGather == 12 && kProducers == 256 && kColsB == 192, "producer row mapping");
    const int j = threadIdx.x & 7, r0 = threadIdx.x >> 3;
    for (int it = 0; it < niter; ++it) {
      const int stage = it % kRowStages;
      const uint32_t ph = (uint32_t)(it / kRowStages) & 1u;
      const int st = rg.x + it / nkc, kc = it % nkc;
      const bool lo = kc < nkc3;  // chunks from nkc3 on take the hi.hi product only
      const int srcA = __ldg(st_src + (size_t)st * kTileRows + r0), srcB = __ldg(st_src + (size_t)st * kTileRows + r0 + 32);
      uint4 v[kGather];
#pragma unroll
      for (int q = 0; q < kGather; ++q) {
        const int h = q / 6, k = q % 6;
        const int src = (k & 1) ? srcB : srcA;
        v[q] = make_uint4(0u, 0u, 0u, 0u);
        if (src >= 0 && (h == 0 || lo))
          v[q] = __ldg(reinterpret_cast<const uint4*>(Mb + ((((size_t)src * 2 + h) * 3 + (k >> 1)) * nkc + kc) * 128) +
                       j);
      }
      if (!mbar_wait(empty(stage), ph ^ 1u, abort)) break;
#pragma unroll
      for (int q = 0; q < kGather; ++q) {
        const int h = q / 6, n = r0 + 32 * (q % 6);
        if (h == 0 || lo)
          *reinterpret_cast<uint4*>(smem + stage * kRowStageBytes + 2 * kRowABytes + h * kColBytes + n * 128 +
                                    ((j ^ (n & 7)) << 4)) = v[q];
      }
      fence_proxy_async();
      mbar_arrive(fullB(stage));
    }
  } else if (lane == 0) {
    // ---- control thread: operator copies and MMAs
    int issued = 0;  // A copies issued for iterations [0, issued)
    auto issue_A = [&](int it) -> bool {
      const int stage = it % kRowStages;
      const uint32_t ph = (uint32_t)(it / kRowStages) & 1u;
      if (!mbar_wait(empty(stage), ph ^ 1u, abort)) return false;
      const int st = rg.x + it / nkc, kc = it % nkc;
      const size_t key = (size_t)st_slot[st];
      const uint8_t* hi = Tb + ((key * 2 + 0) * nkc + kc) * chunk;
      const uint8_t* lo = Tb + ((key * 2 + 1) * nkc + kc) * chunk;
      const uint32_t a0 = sbase + stage * kRowStageBytes;
      const bool with_lo = kc < nkc3;
      mbar_arrive_tx(fullA(stage), with_lo ? 2 * abytes : abytes);
      bulk_g2s(a0, hi, abytes, fullA(stage));
      if (with_lo) bulk_g2s(a0 + kRowABytes, lo, abytes, fullA(stage));
      issued = it + 1;
      return true;
    };
    // operator copies run kRowStages - 1 iterations ahead of the MMAs
    constexpr int kAhead = kRowStages - 1;
    bool ok = true;
    for (int k = 0; ok && k < kAhead && k < niter; ++k) ok = issue_A(k);
    int consumed = 0;  // iterations whose A copy was observed complete
    for (int it = 0; ok && it < niter; ++it) {
      const int stage = it % kRowStages;
      const uint32_t ph = (uint32_t)(it / kRowStages) & 1u;
      if (it + kAhead < niter && !issue_A(it + kAhead)) {
        ok = false;
        break;
      }
      if (!mbar_wait(fullA(stage), ph, abort)) {
        ok = false;
        break;
      }
      consumed = it + 1;
      if (!mbar_wait(fullB(stage), ph, abort)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const int kc = it % nkc;
      const int ks = (kc == nkc - 1) ? ksteps_last : 4;
      const uint32_t a_hi = sbase + stage * kRowStageBytes, a_lo = a_hi + kRowABytes;
      const uint32_t b_hi = a_hi + 2 * kRowABytes, b_lo = b_hi + kColBytes;
      const bool three = kc < nkc3;
      for (int kk = 0; kk < ks; ++kk) {
        const uint32_t off = (uint32_t)kk * 32u;
        umma<KIND>(tmem, sw128_desc(a_hi + off), sw128_desc(b_hi + off), kRowIdesc(KIND), (it > 0 || kk > 0) ? 1u : 0u);
        if (three) {
          umma<KIND>(tmem, sw128_desc(a_hi + off), sw128_desc(b_lo + off), kRowIdesc(KIND), 1u);
          umma<KIND>(tmem, sw128_desc(a_lo + off), sw128_desc(b_hi + off), kRowIdesc(KIND), 1u);
        }
      }
      umma_commit(empty(stage));
    }
    if (ok) {
      umma_commit(done);
    } else {
      *abort = 1;
      // let our own in-flight bulk copies land and our MMAs finish before
      // the tensor memory is freed and the CTA exits
      volatile int never = 0;
      for (int it = consumed; it < issued; ++it)
        mbar_wait(fullA(it % kRowStages), (uint32_t)(it / kRowStages) & 1u, &never);
      umma_commit(done);
      mbar_wait(done, 0u, &never);
      atomicExch(flag, FMM_E_TIMEOUT);
    }
  }
  // ---- epilogue: warps 0-3 own TMEM lanes 0-127 (rows = output coefficients)
  if (warp < 4) {
    // the warp reads the tensor memory or gives up as one
    if (__all_sync(0xffffffffu, mbar_wait(done, 0u, abort))) {
      tc_fence_after();
      const int first = tfirst[tile];
      const int ncell = tfirst[tile + 1] - first;
      const int r = warp * 32 + lane;  // output coefficient of this TMEM lane
      float* pdst = pslot >= 0 ? partial + (size_t)pslot * kColsB * kRowLd : nullptr;
#pragma unroll 1
      for (int cb = 0; cb < kColsB / 16; ++cb) {
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(cb * 16), v);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int n = cb * 16 + i;
          const int comp = n / kTileRows, slot = n % kTileRows;
          if (r >= P || slot >= ncell) continue;
          if (pdst) pdst[(size_t)(slot * 3 + comp) * kRowLd + r] = v[i];
          else L[((size_t)tcell[first + slot] * 3 + comp) * P + r] = v[i];
        }
      }
    } else {
      atomicExch(flag, FMM_E_TIMEOUT);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kProducerWarps) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kRowTmemCols) : "memory");
  }
}

// ---- work items (one-problem plans): runs of at most S steps per CTA

__global__ void k_m2l_item_count(const int2* __restrict__ tr, int ntiles, int S, uint32_t* __restrict__ cnt,
                                 uint32_t* __restrict__ pcnt) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ntiles) return;
  const int c = tr[t].y - tr[t].x;
  const uint32_t k = c > 0 ? (uint32_t)((c + S - 1) / S) : 0u;
  cnt[t] = k;
  pcnt[t] = k > 1 ? k : 0u;
}

// Items in the order of their first operator, for CTAs that run side by side to
// read the same operators out of L2: with 10^5 steps and more the operators a
// problem touches outgrow it (Plummer 1,000,000 at p = 12: 49,141 operators,
// 5.4 GB; M2L 26.3 -> 24.2 ms, Taylor-Green 128^3 4.09 -> 3.86 ms).
__global__ void k_m2l_item_keys(const int4* __restrict__ items, const uint32_t* __restrict__ nitems, int cap,
                                const int* __restrict__ st_slot, uint64_t* __restrict__ keys,
                                uint32_t* __restrict__ vals) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= cap) return;
  keys[i] = i < (int)*nitems ? (uint64_t)st_slot[items[i].y] : 0xffffffffull;
  vals[i] = (uint32_t)i;
}

// The sorted items (in their own order if the sort failed, so that the M2L stays
// within them; the evaluation then ends with FMM_E_TIMEOUT).
__global__ void k_m2l_item_order(const uint32_t* __restrict__ sorted, const int* __restrict__ failed, int n,
                                 uint32_t* __restrict__ order) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) order[i] = *failed ? (uint32_t)i : sorted[i];
}

__global__ void k_m2l_item_fill(const int2* __restrict__ tr, int ntiles, int S, const uint32_t* __restrict__ cnt,
                                const uint32_t* __restrict__ ioff, const uint32_t* __restrict__ poff,
                                int4* __restrict__ items) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ntiles) return;
  const uint32_t k = cnt[t];
  for (uint32_t q = 0; q < k; ++q) {
    const int s0 = tr[t].x + (int)q * S;
    items[ioff[t] + q] = make_int4(t, s0, min(s0 + S, tr[t].y), k > 1 ? (int)(poff[t] + q) : -1);
  }
}

// Local expansions of the split tiles: the partial sums of their items, added
// in item order (a fixed order, so the result is deterministic).  Partial
// sums: [slot][row = cell slot, component][N coefficients].
__global__ void k_m2l_combine(const uint32_t* __restrict__ cnt, const uint32_t* __restrict__ poff,
                              const int* __restrict__ tfirst, const int* __restrict__ tcell, int P, int rows, int N,
                              const float* __restrict__ partial, float* __restrict__ L) {
  const int t = blockIdx.x;
  const uint32_t k = cnt[t];
  if (k <= 1) return;
  const int first = tfirst[t], ncell = tfirst[t + 1] - first;
  for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < 3 * ncell * P; e += gridDim.y * blockDim.x) {
    const int row = e / P, c = e % P;
    float acc = 0.f;
    for (uint32_t q = 0; q < k; ++q) acc += partial[((size_t)(poff[t] + q) * rows + row) * N + c];
    L[((size_t)tcell[first + row / 3] * 3 + row % 3) * P + c] = acc;
  }
}

// The same for the tiles [t0, t0 + gridDim.x) of a batch: the sums of the
// tile's key buckets, in bucket order (empty buckets add nothing, so a problem's
// sums are those it has alone).
__global__ void k_m2l_combine_buckets(const int2* __restrict__ ranges, int t0, const int* __restrict__ tfirst,
                                      const int* __restrict__ tcell, int P, int rows, int N,
                                      const float* __restrict__ partial, float* __restrict__ L) {
  const int t = t0 + blockIdx.x;
  bool some[kKeyBuckets], any = false;
#pragma unroll
  for (int q = 0; q < kKeyBuckets; ++q) {
    const int2 r = ranges[t * kKeyBuckets + q];
    some[q] = r.y > r.x;
    any = any || some[q];
  }
  if (!any) return;
  const int first = tfirst[t], ncell = tfirst[t + 1] - first;
  for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < 3 * ncell * P; e += gridDim.y * blockDim.x) {
    const int row = e / P, c = e % P;
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < kKeyBuckets; ++q)
      if (some[q]) acc += partial[((size_t)(blockIdx.x * kKeyBuckets + q) * rows + row) * N + c];
    L[((size_t)tcell[first + row / 3] * 3 + row % 3) * P + c] = acc;
  }
}

// Self-test of the bounded wait above: one thread waits on a barrier that
// either completes (arrive = 1: it arrives first) or that nothing completes
// (arrive = 0), polling at most `spins` times; FMM_OK or FMM_E_TIMEOUT.
__global__ void k_wait_selftest(long long spins, int arrive, int* status) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    const uint32_t b = smem_u32(&bar);
    abort_flag = 0;
    mbar_init(b, 1);
    if (arrive) mbar_arrive(b);
    *status = mbar_wait(b, 0u, &abort_flag, spins) ? FMM_OK : FMM_E_TIMEOUT;
  }
}

}  // namespace

// Kernel, launch shape and partial-sum layout of a plan's tensor-core M2L.
struct M2lForm {
  const void* kern;
  size_t smem;
  int threads, rows, ld;
  uint32_t tmem_cols;
  bool m2;
};

static M2lForm m2l_form(fmm_plan p, int nkc, int nkc3) {
  const int kind = p->tc_kind;
  const int N = m2l_cols(p->P);
  M2lForm f{};
  if (m2l_tile(p) == kTileRows) {
    // A whole step per stage when it has two BF16 K chunks, the second with one
    // product, and two such CTAs still fit an SM (p = 9 and 10 at theta <= 0.42):
    // one operator-copy latency per step instead of one per chunk.  At p = 11 the
    // stage takes 121 KB, one CTA would run where two do with a chunk per stage
    // (M2L of Plummer 30,011 at theta = 0.4 2.86 ms against 2.56, of Taylor-Green
    // 64^3 1.14 against 1.05).
    const size_t step = 3 * (size_t)((p->P + 7) & ~7) * 128 + 3 * (size_t)kColBytes + 128 + 1024;
    int smem_sm = 0, reserve = 0;
    f.m2 = kind == 0 && nkc == 2 && nkc3 == 1 && !(p->prm.m2l_mode & FMM_M2L_CHUNK_STAGES) &&
           cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, p->device) == cudaSuccess &&
           cudaDeviceGetAttribute(&reserve, cudaDevAttrReservedSharedMemoryPerBlock, p->device) == cudaSuccess &&
           2 * (step + (size_t)reserve) <= (size_t)smem_sm;
    f.kern = f.m2 ? (const void*)k_m2l_rows<0, true>
                  : (kind ? (const void*)k_m2l_rows<1, false> : (const void*)k_m2l_rows<0, false>);
    f.smem = f.m2 ? step : (size_t)kBarOff + 128 + 1024;
    f.threads = kRowThreads;
    f.rows = kColsB;
    f.ld = kRowLd;
    return f;
  }
  const bool two = N > 128;
  f.kern = kind ? (two ? (const void*)k_m2l_cells<1, 2> : (const void*)k_m2l_cells<1, 3>)
                : (two ? (const void*)k_m2l_cells<0, 2> : (const void*)k_m2l_cells<0, 3>);
  f.tmem_cols = 32;
  while ((int)f.tmem_cols < N) f.tmem_cols *= 2;
  // One stage per CTA and as many CTAs per SM as registers, TMEM and the stage
  // memory allow: the CTAs hide each other's gathers, and more gathering threads
  // run.  Rings of 2 and 3 stages of cp.async gathers in fewer CTAs were slower:
  // Plummer 1,000,000 at p = 12 26.3 / 34.1 / 34.4 ms for 1 / 2 / 3 stages, the
  // batch of 32 at p = 8 1.17 / 1.42 / 2.39 ms.
  f.smem = 2 * (kBBytes + (size_t)N * 128) + 64 + 1024;
  f.threads = kThreads;
  f.rows = kRows;
  f.ld = N;
  return f;
}

// The work items of a one-problem plan and their place in p->m2l_items.
struct M2lItems {
  int64_t S, max_items, max_split;
  int4* items;
  uint32_t *order, *cnt, *pcnt, *ioff, *poff, *totals;  // totals: items, partial slots
  size_t bytes;
};

static M2lItems m2l_items(fmm_plan p) {
  const int64_t nt = p->ntiles;
  M2lItems w{};
  w.S = std::min(kItemMaxSteps, std::max(kItemMinSteps, (p->n_steps + kItemTarget - 1) / kItemTarget));
  w.S = std::max(w.S, (p->n_steps + kItemsMax - 1) / kItemsMax);
  w.max_items = nt + p->n_steps / w.S + 1;
  w.max_split = 2 * (p->n_steps / w.S) + 1;
  uint8_t* base = p->m2l_items.as<uint8_t>();
  w.items = reinterpret_cast<int4*>(base);
  uint32_t* u = reinterpret_cast<uint32_t*>(base + (size_t)w.max_items * sizeof(int4));
  w.cnt = u;
  w.pcnt = w.cnt + (nt + 1);
  w.ioff = w.pcnt + (nt + 1);
  w.poff = w.ioff + (nt + 1);
  w.totals = w.poff + (nt + 1);
  uint32_t* order = w.totals + 2;
  w.bytes = (size_t)w.max_items * (sizeof(int4) + sizeof(uint32_t)) + (4 * (size_t)(nt + 1) + 2) * sizeof(uint32_t);
  w.order = p->n_steps >= kItemSortSteps ? order : nullptr;
  return w;
}

// One-problem plans split the tiles into work items of at most S steps:
// with Alg. 1's printed rule the coarse target tiles collect many more steps
// than the rest, and one CTA per tile left a long tail (and long tensor-memory
// sums).  Built once per tree.
int m2l_build_items(fmm_plan p, cudaStream_t s) {
  if (p->n_steps == 0 || p->batched || !p->last_tc) return FMM_OK;
  const int nt = (int)p->ntiles, T = 256;
  FMM_TRY(p->m2l_items.ensure(m2l_items(p).bytes));
  const M2lItems w = m2l_items(p);
  const int2* ranges = p->tile_range.as<int2>();
  const unsigned gt = (unsigned)((nt + T - 1) / T);
  ++g_launches;
  k_m2l_item_count<<<gt, T, 0, s>>>(ranges, nt, (int)w.S, w.cnt, w.pcnt);
  FMM_TRY(exclusive_scan_u32(w.cnt, w.ioff, nt, w.totals, p->scan_tmp, s));
  FMM_TRY(exclusive_scan_u32(w.pcnt, w.poff, nt, w.totals + 1, p->scan_tmp, s));
  ++g_launches;
  k_m2l_item_fill<<<gt, T, 0, s>>>(ranges, nt, (int)w.S, w.cnt, w.ioff, w.poff, w.items);
  if (w.order) {
    const size_t k = (size_t)w.max_items;
    FMM_TRY(p->lk0.ensure(k * sizeof(uint64_t)));
    FMM_TRY(p->lk1.ensure(k * sizeof(uint64_t)));
    FMM_TRY(p->lv0.ensure(k * sizeof(uint32_t)));
    FMM_TRY(p->lv1.ensure(k * sizeof(uint32_t)));
    ++g_launches;
    k_m2l_item_keys<<<(unsigned)((k + T - 1) / T), T, 0, s>>>(w.items, w.totals, (int)k, p->st_slot.as<int>(),
                                                              p->lk0.as<uint64_t>(), p->lv0.as<uint32_t>());
    int second = 0;
    FMM_TRY(radix_sort_u64(p->sort, p->lk0.as<uint64_t>(), p->lv0.as<uint32_t>(), p->lk1.as<uint64_t>(),
                           p->lv1.as<uint32_t>(), (int64_t)k, 32, &second, s));
    ++g_launches;
    k_m2l_item_order<<<(unsigned)((k + T - 1) / T), T, 0, s>>>(
        second ? p->lv1.as<uint32_t>() : p->lv0.as<uint32_t>(), p->sort.failed, (int)k, w.order);
  }
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

int m2l_tensor(fmm_plan p, cudaStream_t s) {
  if (p->n_steps == 0) return FMM_OK;
  const int kind = p->tc_kind;
  const int ksteps = (p->P + m2l_kstep(kind) - 1) / m2l_kstep(kind);
  const int nkc = m2l_kchunks(p->P, kind);
  const int last = ksteps - 4 * (nkc - 1);
  const int nkc3 = m2l_split_chunks(p->P, kind, p->prm.theta, p->prm.m2l_mode & FMM_M2L_FULL_SPLIT);
  const int N = m2l_cols(p->P);
  const M2lForm f = m2l_form(p, nkc, nkc3);
  p->m2l_stage_chunks = f.m2 ? 2 : 1;
  static std::atomic<bool> done[kMaxDevices];
  FMM_TRY(once_per_device(done, [] {
    const void* k[7] = {(const void*)k_m2l_cells<1, 2>, (const void*)k_m2l_cells<1, 3>,
                        (const void*)k_m2l_cells<0, 2>, (const void*)k_m2l_cells<0, 3>,
                        (const void*)k_m2l_rows<0, true>, (const void*)k_m2l_rows<1, false>,
                        (const void*)k_m2l_rows<0, false>};
    for (const void* q : k)
      if (cudaFuncSetAttribute(q, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024) != cudaSuccess ||
          cudaFuncSetAttribute(q, cudaFuncAttributePreferredSharedMemoryCarveout, 100) != cudaSuccess)
        return false;
    return true;
  }));
  const int nt = (int)p->ntiles;
  const int T = 256;
  const int2* ranges = p->tile_range.as<int2>();
  const int* tfirst = p->tile_first.as<int>();
  const int* tcell = p->tile_cells.as<int>();
  float* L = p->L.as<float>();
  const uint32_t* order = nullptr;
  auto launch = [&](unsigned grid, int range0, const int4* items, const uint32_t* nitems) -> int {
    const int* slot = p->st_slot.as<int>();
    const int* src = p->st_src.as<int>();
    const uint8_t* Tb = p->Tbf.as<uint8_t>();
    const uint8_t* Mb = p->Mbf.as<uint8_t>();
    float* partial = p->m2l_partial.as<float>();
    int* flag = p->flags.as<int>();
    int P = p->P, NN = N, a = nkc, b = nkc3, c = last;
    uint32_t e = f.tmem_cols;
    void* cells[] = {&ranges, &range0, &items, &nitems, &order, &tfirst, &slot, &src, &Tb, &Mb, &P, &NN,
                     &a, &b, &c, &e, &tcell, &L, &partial, &flag};
    void* rows[] = {&ranges, &range0, &items, &nitems, &order, &tfirst, &slot, &src, &Tb, &Mb, &P, &NN,
                    &a, &b, &c, &tcell, &L, &partial, &flag};
    ++g_launches;
    FMM_CUDA_TRY(cudaLaunchKernel(f.kern, dim3(grid), dim3(f.threads), f.rows == kRows ? cells : rows, f.smem, s));
    return FMM_OK;
  };
  if (p->batched) {
    // Batches: one CTA per (tile, key bucket), in rounds that bound the partial
    // sums; a tile's buckets are cut by the translation alone, so a problem's
    // sums do not depend on the rest of the batch.  One CTA per tile made the
    // longest tile the time of the phase (32 problems: 4.7 ms, now 1.17).
    const int round = std::min(nt, 1024);
    FMM_TRY(p->m2l_partial.ensure((size_t)round * kKeyBuckets * f.rows * f.ld * sizeof(float)));
    for (int t0 = 0; t0 < nt; t0 += round) {
      const int k = std::min(round, nt - t0);
      FMM_TRY(launch((unsigned)(k * kKeyBuckets), t0 * kKeyBuckets, nullptr, nullptr));
      ++g_launches;
      k_m2l_combine_buckets<<<dim3((unsigned)k, 4), T, 0, s>>>(ranges, t0, tfirst, tcell, p->P, f.rows, f.ld,
                                                               p->m2l_partial.as<float>(), L);
    }
    FMM_CUDA_TRY(cudaGetLastError());
    return FMM_OK;
  }
  const M2lItems w = m2l_items(p);
  order = w.order;
  FMM_TRY(p->m2l_partial.ensure((size_t)w.max_split * f.rows * f.ld * sizeof(float)));
  FMM_TRY(launch((unsigned)w.max_items, 0, w.items, w.totals));
  ++g_launches;
  // a tile's rows over 8 CTAs (the split tiles are a few hundred)
  k_m2l_combine<<<dim3((unsigned)nt, 8), T, 0, s>>>(w.cnt, w.poff, tfirst, tcell, p->P, f.rows, f.ld,
                                                    p->m2l_partial.as<float>(), L);
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

}  // namespace fmm

extern "C" int fmm_selftest_bounded_wait(int64_t spins, int arrive, void* stream) {
  if (spins < 1 || spins > fmm::kSpin || (arrive != 0 && arrive != 1)) return FMM_E_INVAL;
  cudaStream_t s = (cudaStream_t)stream;
  int* d = nullptr;
  int h = FMM_E_CUDA;
  if (cudaMalloc(&d, sizeof(int)) != cudaSuccess) return FMM_E_NOMEM;
  ++fmm::g_launches;
  fmm::k_wait_selftest<<<1, 32, 0, s>>>((long long)spins, arrive, d);
  if (cudaGetLastError() == cudaSuccess && cudaMemcpyAsync(&h, d, sizeof(int), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
      cudaStreamSynchronize(s) == cudaSuccess) {
  } else {
    h = FMM_E_CUDA;
  }
  cudaFree(d);
  return h;
}
