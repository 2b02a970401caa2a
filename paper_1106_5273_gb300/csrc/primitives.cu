// Device-wide exclusive scan and stable LSD radix sort (keys u64, values u32).
// k_sort_hist / k_sort_scatter serve the caller that provides all scratch.
//
// Used by the Morton sort (Sec. 3.2), the tree build, the traversal output
// compaction and the grouping of P2P / M2L lists.  Both are deterministic:
// the scan is a fixed-order reduction, the sort is stable.
#include <algorithm>

#include "primitives.cuh"

namespace fmm {

namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ inline uint32_t warp_incl_scan(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Block-wide exclusive scan of one value per thread; returns the block total.
__device__ inline uint32_t block_excl_scan(uint32_t v, uint32_t* s_warp, uint32_t& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t inc = warp_incl_scan(v);
  if (lane == 31) s_warp[w] = inc;
  __syncthreads();
  if (w == 0) {
    uint32_t x = (lane < (int)(blockDim.x >> 5)) ? s_warp[lane] : 0u;
    uint32_t xi = warp_incl_scan(x);
    s_warp[lane] = xi - x;
    if (lane == 31) s_warp[32] = xi;
  }
  __syncthreads();
  uint32_t r = inc - v + s_warp[w];
  total = s_warp[32];
  __syncthreads();
  return r;
}

__global__ void k_scan_reduce(const uint32_t* __restrict__ in, int64_t n, uint32_t* __restrict__ sums) {
  __shared__ uint32_t s_warp[33];
  int64_t base = (int64_t)blockIdx.x * kScanTile;
  uint32_t acc = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    int64_t idx = base + (int64_t)threadIdx.x * kScanItems + i;
    if (idx < n) acc += in[idx];
  }
  uint32_t total;
  block_excl_scan(acc, s_warp, total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void k_scan_apply(const uint32_t* in, int64_t n, uint32_t* out,
                             const uint32_t* __restrict__ offs, uint32_t* __restrict__ total_out) {
  __shared__ uint32_t s_warp[33];
  int64_t base = (int64_t)blockIdx.x * kScanTile;
  uint32_t v[kScanItems];
  uint32_t acc = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    int64_t idx = base + (int64_t)threadIdx.x * kScanItems + i;
    v[i] = idx < n ? in[idx] : 0u;
    acc += v[i];
  }
  uint32_t total;
  uint32_t pre = block_excl_scan(acc, s_warp, total);
  uint32_t off = offs ? offs[blockIdx.x] : 0u;
  pre += off;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    int64_t idx = base + (int64_t)threadIdx.x * kScanItems + i;
    if (idx < n) out[idx] = pre;
    pre += v[i];
  }
  if (total_out && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total_out = off + total;
}

}  // namespace

static void scan_rec(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* total_dev, uint32_t* tmp,
                     cudaStream_t s) {
  int64_t nb = (n + kScanTile - 1) / kScanTile;
  if (nb <= 1) {
    ++g_launches;
    k_scan_apply<<<1, kScanThreads, 0, s>>>(in, n, out, nullptr, total_dev);
    return;
  }
  uint32_t* sums = tmp;
  ++g_launches;
  k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, sums);
  scan_rec(sums, sums, nb, nullptr, tmp + nb + 1, s);
  ++g_launches;
  k_scan_apply<<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, out, sums, total_dev);
}

// Exclusive scan of n u32 values (in may equal out).  If total_dev is given,
// the sum of all values is written there.  tmp is grown as needed.
int exclusive_scan_u32(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* total_dev, DBuf& tmp,
                       cudaStream_t s) {
  if (n <= 0) {
    if (total_dev) FMM_CUDA_TRY(cudaMemsetAsync(total_dev, 0, sizeof(uint32_t), s));
    return FMM_OK;
  }
  size_t need = 0;
  for (int64_t m = n;;) {
    int64_t nb = (m + kScanTile - 1) / kScanTile;
    if (nb <= 1) break;
    need += (size_t)(nb + 1);
    m = nb;
  }
  FMM_TRY(tmp.ensure((need + 1) * sizeof(uint32_t)));
  scan_rec(in, out, n, total_dev, tmp.as<uint32_t>(), s);
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

// ------------------------------------------------------------------ sort ---

namespace {

constexpr int kSortThreads = 256;
constexpr int kSortRows = 16;
constexpr int kSortTile = kSortThreads * kSortRows;  // 4096 keys per tile

__global__ void k_sort_hist(const uint64_t* __restrict__ keys, int64_t n, int shift, int ntiles,
                            uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  int64_t base = (int64_t)blockIdx.x * kSortTile;
  for (int r = 0; r < kSortRows; ++r) {
    int64_t i = base + r * kSortThreads + threadIdx.x;
    if (i < n) atomicAdd(&h[(keys[i] >> shift) & 0xff], 1u);
  }
  __syncthreads();
  hist[(size_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter: rows of 256 keys in order; within a row, warps in order;
// within a warp, lanes in order.  Element order = (row, warp, lane).
__global__ void k_sort_scatter(const uint64_t* __restrict__ kin, const uint32_t* __restrict__ vin,
                               uint64_t* __restrict__ kout, uint32_t* __restrict__ vout, int64_t n,
                               int shift, int ntiles, const uint32_t* __restrict__ offs) {
  __shared__ uint32_t s_run[256];
  __shared__ uint32_t s_w[8][256];
  __shared__ uint32_t s_base[256];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  s_run[tid] = 0;
  s_base[tid] = offs[(size_t)tid * ntiles + blockIdx.x];
  const uint32_t lt_mask = (1u << lane) - 1u;
  int64_t base = (int64_t)blockIdx.x * kSortTile;
  for (int r = 0; r < kSortRows; ++r) {
    int64_t i = base + r * kSortThreads + tid;
    bool valid = i < n;
    uint64_t key = valid ? kin[i] : 0ull;
    uint32_t val = valid ? vin[i] : 0u;
    int d = valid ? (int)((key >> shift) & 0xff) : 256;
#pragma unroll
    for (int q = 0; q < 8; ++q) s_w[q][tid] = 0;
    __syncthreads();
    uint32_t peers = __match_any_sync(0xffffffffu, d);
    uint32_t rank = __popc(peers & lt_mask);
    if (valid && rank == 0) s_w[w][d] = __popc(peers);
    __syncthreads();
    {
      uint32_t acc = s_run[tid];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        uint32_t c = s_w[q][tid];
        s_w[q][tid] = acc;
        acc += c;
      }
      s_run[tid] = acc;
    }
    __syncthreads();
    if (valid) {
      uint32_t pos = s_base[d] + s_w[w][d] + rank;
      kout[pos] = key;
      vout[pos] = val;
    }
    __syncthreads();
  }
}

// ---- Sort passes with one kernel each: the one-sweep radix sort (Adinets and
// Merrill, arXiv:2206.01784) over decoupled look-back (Merrill and Garland,
// NVIDIA NVR-2016-002).  The digit counts of all passes are
// taken at once (k_digit_hist, or by the kernel that makes the keys), scanned by
// one CTA (k_digit_scan), and a pass (k_onesweep) ranks its tile, learns the
// counts of the tiles before it by looking back over their published counts,
// and scatters.  Tiles are numbered by a ticket in the order the CTAs start, so
// every tile that a CTA waits for has started; the waits are bounded.  Three
// kernels per pass and a host read of the varying digits before: the tree phase
// of 1000 blobs took 0.23 ms, now 0.14, of 100,003 0.44 -> 0.24, of 1,000,000
// 0.82 -> 0.67.

// Counts of digit q (8 bits from bit 8 q) of every key, q < npass.
__global__ void __launch_bounds__(256) k_digit_hist(const uint64_t* __restrict__ keys, int64_t n, int npass,
                                                    uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[kSortPasses * 256];
  clear_digits(h, npass);
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x; b < n; b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = b + threadIdx.x;
    count_digits(h, i < n ? keys[i] : 0ull, i < n, npass);
  }
  flush_digits(h, npass, hist);
}

// First output position of every digit of every pass, and which passes do
// anything: one over a digit that is the same in every key is the identity, and
// is left out unless `all` (the caller then knows where the result is); none
// after a sort that failed.
__global__ void __launch_bounds__(256) k_digit_scan(SortState* __restrict__ st, int64_t n, int npass, int all,
                                                    const int* __restrict__ failed) {
  __shared__ uint32_t ws[8];
  __shared__ int act[kSortPasses];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, bad = *failed;
  for (int q = 0; q < npass; ++q) {
    const uint32_t c = st->hist[q][t];
    if (t == 0) act[q] = all;
    uint32_t inc = warp_incl_scan(c);
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    uint32_t pre = 0;
    for (int i = 0; i < w; ++i) pre += ws[i];
    st->base[q][t] = pre + inc - c;
    if (c != 0u && (int64_t)c < n) act[q] = 1;
    __syncthreads();
  }
  if (t == 0) {
    int sel = 0;
    for (int q = 0; q < npass; ++q) {
      st->active[q] = bad ? 0 : act[q];
      st->sel[q] = sel;
      sel ^= act[q];
    }
    st->sel[npass] = sel;
  }
}

// look: one 64-bit word per (tile, digit): epoch << 34 | state << 32 | count,
// state 1 the tile's own count, 2 the count of it and all before; words of
// earlier passes carry an earlier epoch.
// R keys per thread.  The tile's keys are put in order in shared memory first, so
// that a digit's run is written by consecutive threads.
template <int R>
__global__ void __launch_bounds__(kSortThreads) k_onesweep(uint64_t* __restrict__ k0, uint32_t* __restrict__ v0,
                                                           uint64_t* __restrict__ k1, uint32_t* __restrict__ v1,
                                                           int64_t n, int pass, SortState* __restrict__ st,
                                                           unsigned long long* look, unsigned epoch,
                                                           int spins, int* error, volatile int* failed) {
  // a wait that runs out clears the passes behind, whose input is then not all
  // there (the tiles of its own pass may go on); the word is read here anyway
  if (!st->active[pass]) return;
  const bool swap = st->sel[pass] != 0;
  const uint64_t* kin = swap ? k1 : k0;
  const uint32_t* vin = swap ? v1 : v0;
  uint64_t* kout = swap ? k0 : k1;
  uint32_t* vout = swap ? v0 : v1;
  constexpr int kTileKeys = kSortThreads * R;
  extern __shared__ uint64_t sk[];  // [kTileKeys] keys, then [kTileKeys] values
  uint32_t* sv = reinterpret_cast<uint32_t*>(sk + kTileKeys);
  __shared__ uint32_t cnt[kSortThreads / 32][256];
  __shared__ uint32_t shift_to[256];  // output position minus position in the tile
  __shared__ uint32_t ws[kSortThreads / 32];
  __shared__ int s_tile, s_bad;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) {
    s_tile = (int)atomicAdd(&st->ticket[pass], 1u);
    s_bad = 0;
  }
  for (int q = 0; q < kSortThreads / 32; ++q) cnt[q][tid] = 0u;
  __syncthreads();
  const int tile = s_tile, shift = 8 * pass;
  const int64_t t0 = (int64_t)tile * kTileKeys;
  const int have = (int)min((int64_t)kTileKeys, n - t0);
  // the warp's 32 R keys in order: row r holds keys 32 r + lane
  const int base = w * (32 * R) + lane;
  uint64_t key[R];
  uint32_t val[R], rank[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const bool live = base + 32 * r < have;
    key[r] = live ? kin[t0 + base + 32 * r] : 0ull;
    val[r] = live ? vin[t0 + base + 32 * r] : 0u;
  }
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (w * (32 * R) + 32 * r >= have) break;
    const bool live = base + 32 * r < have;
    const int d = live ? (int)((key[r] >> shift) & 0xff) : 256;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    const int leader = __ffs(peers) - 1;
    uint32_t before = 0;
    if (live && lane == leader) {
      before = cnt[w][d];
      cnt[w][d] = before + (uint32_t)__popc(peers);
    }
    before = __shfl_sync(0xffffffffu, before, leader);
    rank[r] = before + (uint32_t)__popc(peers & lt);
    __syncwarp();
  }
  __syncthreads();
  {  // thread = digit: the tile's count, the warps' first ranks, the tiles before
    uint32_t total = 0;
#pragma unroll
    for (int q = 0; q < kSortThreads / 32; ++q) {
      const uint32_t c = cnt[q][tid];
      cnt[q][tid] = total;
      total += c;
    }
    volatile unsigned long long* lk = look;
    const unsigned long long tag = (unsigned long long)epoch << 34;
    lk[(size_t)tile * 256 + tid] = tag | ((tile == 0 ? 2ull : 1ull) << 32) | total;
    // first position of the digit in the tile
    const uint32_t inc = warp_incl_scan(total);
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    uint32_t local = inc - total;
    for (int q = 0; q < w; ++q) local += ws[q];
#pragma unroll
    for (int q = 0; q < kSortThreads / 32; ++q) cnt[q][tid] += local;
    uint32_t pre = 0;
    bool ok = tile == 0 || spins >= 0;
    for (int t = tile - 1; ok && t >= 0; --t) {
      unsigned long long x = 0;
      int spin = 0;
      while (((x = lk[(size_t)t * 256 + tid]) >> 34) != epoch)
        if ((++spin & 1023) == 0 && (spin >= spins || *failed)) {
          ok = false;
          break;
        }
      pre += (uint32_t)x;
      if ((x >> 32) & 2ull) break;
    }
    if (!ok) s_bad = 1;
    else if (tile > 0) lk[(size_t)tile * 256 + tid] = tag | (2ull << 32) | (pre + total);
    shift_to[tid] = st->base[pass][tid] + pre - local;
  }
  __syncthreads();
  if (s_bad) {  // gave up: write nothing
    if (tid == 0) {
      for (int q = pass + 1; q < kSortPasses; ++q) st->active[q] = 0;
      *failed = 1;
      atomicExch(error, FMM_E_TIMEOUT);
    }
    return;
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (base + 32 * r >= have) break;
    const uint32_t o = cnt[w][(int)((key[r] >> shift) & 0xff)] + rank[r];
    sk[o] = key[r];
    sv[o] = val[r];
  }
  __syncthreads();
  for (int i = tid; i < have; i += kSortThreads) {
    const uint64_t k = sk[i];
    const uint32_t o = shift_to[(int)((k >> shift) & 0xff)] + (uint32_t)i;
    kout[o] = k;
    vout[o] = sv[i];
  }
}

// Keys per thread: small tiles while they are few (a tile is one CTA's serial
// work), large ones for throughput.
int sweep_rows(int64_t n) { return n <= 65536 ? 4 : (n <= (1 << 20) ? 8 : 16); }

}  // namespace

int sort_begin(SortScratch& b, int64_t n, cudaStream_t s) {
  const int64_t tile = (int64_t)kSortThreads * sweep_rows(n);
  const size_t tiles = (size_t)((n + tile - 1) / tile);
  FMM_TRY(b.state.ensure(sizeof(SortState)));
  if (b.look.bytes < tiles * 256 * sizeof(unsigned long long) || b.epoch > (1u << 29)) {
    FMM_TRY(b.look.ensure(tiles * 256 * sizeof(unsigned long long)));
    FMM_CUDA_TRY(cudaMemsetAsync(b.look.ptr, 0, b.look.bytes, s));  // epoch 0: never published
    b.epoch = 0;
  }
  FMM_CUDA_TRY(cudaMemsetAsync(b.state.ptr, 0, sizeof(SortState), s));
  return FMM_OK;
}

int sort_passes(SortScratch& b, uint64_t* k0, uint32_t* v0, uint64_t* k1, uint32_t* v1, int64_t n, int npass, bool all,
                cudaStream_t s) {
  SortState* st = b.state.as<SortState>();
  ++g_launches;
  k_digit_scan<<<1, 256, 0, s>>>(st, n, npass, all ? 1 : 0, b.failed);
  const int R = sweep_rows(n);
  const int64_t tile = (int64_t)kSortThreads * R;
  const unsigned g = (unsigned)((n + tile - 1) / tile);
  const size_t sh = (size_t)tile * (sizeof(uint64_t) + sizeof(uint32_t));
  auto kern = R == 4 ? k_onesweep<4> : (R == 8 ? k_onesweep<8> : k_onesweep<16>);
  static std::atomic<bool> done[kMaxDevices];
  FMM_TRY(once_per_device(done, [] {
    return cudaFuncSetAttribute(k_onesweep<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSortThreads * 16 * 12) ==
           cudaSuccess;
  }));
  unsigned long long* look = b.look.as<unsigned long long>();
  for (int q = 0; q < npass; ++q) {
    ++g_launches;
    kern<<<g, kSortThreads, sh, s>>>(k0, v0, k1, v1, n, q, st, look, ++b.epoch, (int)b.spins, b.error, b.failed);
  }
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

// Sort (keys, vals) by the lowest `bits` key bits, stable; the result is in
// (k1, v1) if *in_second.
int radix_sort_u64(SortScratch& b, uint64_t* k0, uint32_t* v0, uint64_t* k1, uint32_t* v1, int64_t n, int bits,
                   int* in_second, cudaStream_t s) {
  *in_second = 0;
  if (n <= 1 || bits <= 0) return FMM_OK;
  const int npass = (bits + 7) / 8;
  FMM_TRY(sort_begin(b, n, s));
  ++g_launches;
  k_digit_hist<<<(unsigned)std::min<int64_t>(608, (n + 2047) / 2048), 256, 0, s>>>(k0, n, npass,
                                                                                   &b.state.as<SortState>()->hist[0][0]);
  FMM_TRY(sort_passes(b, k0, v0, k1, v1, n, npass, true, s));
  *in_second = npass & 1;
  return FMM_OK;
}

}  // namespace fmm

namespace fmm {

// Variants of the scan and sort above that take their scratch as raw device
// pointers (for callers that provide all memory): scan_tmp must hold
// scan_scratch_words(n) words, hist 256 * ceil(n/4096) words.
size_t scan_scratch_words(int64_t n) {
  size_t need = 0;
  for (int64_t m = n;;) {
    int64_t nb = (m + kScanTile - 1) / kScanTile;
    if (nb <= 1) break;
    need += (size_t)(nb + 1);
    m = nb;
  }
  return need + 1;
}

int radix_sort_u64_raw(uint64_t* k0, uint32_t* v0, uint64_t* k1, uint32_t* v1, int64_t n, int bit_begin,
                       int bit_end, int* in_second, uint32_t* hist, uint32_t* scan_tmp, cudaStream_t s) {
  *in_second = 0;
  if (n <= 1) return FMM_OK;
  int ntiles = (int)((n + kSortTile - 1) / kSortTile);
  uint64_t* ka = k0;
  uint64_t* kb = k1;
  uint32_t* va = v0;
  uint32_t* vb = v1;
  for (int shift = bit_begin; shift < bit_end; shift += 8) {
    ++g_launches;
    k_sort_hist<<<ntiles, kSortThreads, 0, s>>>(ka, n, shift, ntiles, hist);
    scan_rec(hist, hist, (int64_t)256 * ntiles, nullptr, scan_tmp, s);
    ++g_launches;
    k_sort_scatter<<<ntiles, kSortThreads, 0, s>>>(ka, va, kb, vb, n, shift, ntiles, hist);
    FMM_CUDA_TRY(cudaGetLastError());
    std::swap(ka, kb);
    std::swap(va, vb);
    *in_second ^= 1;
  }
  return FMM_OK;
}

}  // namespace fmm
