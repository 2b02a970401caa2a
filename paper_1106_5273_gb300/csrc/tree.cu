// Morton keys, sort, octree build, cell centres and radii (Sec. 3.2).
//
// Keys: positions normalised into the cube in FP64, 21 bits per axis
// interleaved (bit b of x, y, z at 3b+2, 3b+1, 3b), stable LSD radix sort of
// (key, index).  Cells: level by level, a cell splits while it holds more than
// ncrit particles and its level is below 21; children are the non-empty
// octants in digit order, so every level is stored in Morton order.
// Expansion centre = geometric cube centre, radius = largest FP64 distance
// from the centre to a particle of the cell.  Every FP64 expression uses
// explicitly rounded operations (no contraction) in a fixed order, so the MAC
// decisions built on them are reproducible.
#include <cstring>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

// Bounding box; min and max of the FP32 coordinates are exact.
__device__ __forceinline__ void block_min_max(float lo[3], float hi[3], float (*sh)[8]) {
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
      hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
    }
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      sh[a][threadIdx.x >> 5] = lo[a];
      sh[3 + a][threadIdx.x >> 5] = hi[a];
    }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
      for (int a = 0; a < 3; ++a) {
        lo[a] = fminf(lo[a], sh[a][w]);
        hi[a] = fmaxf(hi[a], sh[3 + a][w]);
      }
}

__global__ void __launch_bounds__(256) k_bbox_partial(const float* __restrict__ pos, int64_t n,
                                                      double* __restrict__ part) {
  __shared__ float sh[6][8];
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float v = pos[3 * i + a];
      lo[a] = fminf(lo[a], v);
      hi[a] = fmaxf(hi[a], v);
    }
  }
  block_min_max(lo, hi, sh);
  if (threadIdx.x == 0)
    for (int a = 0; a < 3; ++a) {
      part[blockIdx.x * 6 + a] = (double)lo[a];
      part[blockIdx.x * 6 + 3 + a] = (double)hi[a];
    }
}

// Free-space cube: centre of the bounding box, half side = longest extent/2
// times (1 + 2^-10) (0.5 if all points coincide).
__device__ inline void cube_from_bounds(const double lo[3], const double hi[3], double* box) {
  double ext = 0.0;
  for (int a = 0; a < 3; ++a) ext = fmax(ext, __dsub_rn(hi[a], lo[a]));
  double half = __dmul_rn(__dmul_rn(ext, 0.5), 1.0 + 0.0009765625);
  if (half == 0.0) half = 0.5;
  for (int a = 0; a < 3; ++a) box[a] = __dsub_rn(__dmul_rn(__dadd_rn(lo[a], hi[a]), 0.5), half);
  box[3] = __dmul_rn(half, 2.0);
}

__global__ void __launch_bounds__(256) k_bbox_final(const double* __restrict__ part, int nb,
                                                    double* __restrict__ box) {
  __shared__ float sh[6][8];
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int b = threadIdx.x; b < nb; b += blockDim.x)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      lo[a] = fminf(lo[a], (float)part[b * 6 + a]);
      hi[a] = fmaxf(hi[a], (float)part[b * 6 + 3 + a]);
    }
  block_min_max(lo, hi, sh);
  if (threadIdx.x != 0) return;
  const double l[3] = {lo[0], lo[1], lo[2]}, h[3] = {hi[0], hi[1], hi[2]};
  cube_from_bounds(l, h, box);
}

// One CTA per problem of a batch: its cube (same arithmetic as above; min and
// max are exact, so the cube equals the one of the problem on its own).
__global__ void __launch_bounds__(256) k_bbox_seg(const float* __restrict__ pos, const int* __restrict__ off,
                                                  double* __restrict__ box) {
  const int sg = blockIdx.x;
  const int b = off[sg], e = off[sg + 1];
  __shared__ float sh[6][8];
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int i = b + threadIdx.x; i < e; i += blockDim.x) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float v = pos[3 * (int64_t)i + a];
      lo[a] = fminf(lo[a], v);
      hi[a] = fmaxf(hi[a], v);
    }
  }
  block_min_max(lo, hi, sh);
  if (threadIdx.x == 0) {
    const double l[3] = {lo[0], lo[1], lo[2]}, h[3] = {hi[0], hi[1], hi[2]};
    cube_from_bounds(l, h, box + 4 * sg);
  }
}

// Largest sigma of each problem (float bits; sigma > 0 orders like its bits).
__global__ void __launch_bounds__(256) k_sigma_max_seg(const float* __restrict__ sig, const int* __restrict__ off,
                                                       unsigned int* __restrict__ out) {
  const int sg = blockIdx.x;
  float m = 0.f;
  for (int i = off[sg] + threadIdx.x; i < off[sg + 1]; i += blockDim.x) m = fmaxf(m, sig[i]);
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ float sh[8];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, sh[w]);
    out[sg] = __float_as_uint(fmaxf(m, sh[0]));
  }
}

// Problem of particle i: the largest s with off[s] <= i.
__device__ inline int seg_of(const int* __restrict__ off, int nseg, int64_t i) {
  int lo = 0, hi = nseg;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if ((int64_t)off[mid] <= i) lo = mid;
    else hi = mid;
  }
  return lo;
}

__global__ void k_set_box(double x, double y, double z, double len, double* box) {
  box[0] = x;
  box[1] = y;
  box[2] = z;
  box[3] = len;
}

__device__ inline uint64_t spread3(uint64_t x) {
  x &= 0x1fffffull;
  x = (x | x << 32) & 0x1f00000000ffffull;
  x = (x | x << 16) & 0x1f0000ff0000ffull;
  x = (x | x << 8) & 0x100f00f00f00f00full;
  x = (x | x << 4) & 0x10c30c30c30c30c3ull;
  x = (x | x << 2) & 0x1249249249249249ull;
  return x;
}

__device__ inline uint32_t compact3(uint64_t x) {
  x &= 0x1249249249249249ull;
  x = (x ^ (x >> 2)) & 0x10c30c30c30c30c3ull;
  x = (x ^ (x >> 4)) & 0x100f00f00f00f00full;
  x = (x ^ (x >> 8)) & 0x1f0000ff0000ffull;
  x = (x ^ (x >> 16)) & 0x1f00000000ffffull;
  x = (x ^ (x >> 32)) & 0x1fffffull;
  return (uint32_t)x;
}

// Cell coordinate floor((x - bmin) f) with f = 2^kbits / L rounded once (one
// FP64 division per particle rather than one per coordinate), clamped.
__device__ inline uint64_t quantize_axis(float x, double bmin, double f, double scale) {
  double k = floor(__dmul_rn(__dsub_rn((double)x, bmin), f));
  if (!(k >= 0.0)) k = 0.0;
  if (k > scale - 1.0) k = scale - 1.0;
  return (uint64_t)k;
}

// kbits Morton bits per axis; a batch puts the problem index above them.
// hist (if given): the digit counts of the sort.
__global__ void __launch_bounds__(256) k_keys(const float* __restrict__ pos, int64_t n, const double* __restrict__ box,
                                              const int* __restrict__ off, int nseg, int kbits,
                                              uint64_t* __restrict__ keys, uint32_t* __restrict__ idx, int npass,
                                              uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[kSortPasses * 256];
  __shared__ double f0;
  const double scale = ldexp(1.0, kbits);
  // one problem: f once per block (FP64 division is slow)
  if (!off && threadIdx.x == 0) f0 = __ddiv_rn(scale, box[3]);
  clear_digits(h, npass);
  for (int64_t b0 = (int64_t)blockIdx.x * blockDim.x; b0 < n; b0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = b0 + threadIdx.x;
    uint64_t k = 0ull;
    if (i < n) {
      const int sg = off ? seg_of(off, nseg, i) : 0;
      const double* b = box + 4 * sg;
      const double f = off ? __ddiv_rn(scale, b[3]) : f0;
      const uint64_t kx = quantize_axis(pos[3 * i + 0], b[0], f, scale);
      const uint64_t ky = quantize_axis(pos[3 * i + 1], b[1], f, scale);
      const uint64_t kz = quantize_axis(pos[3 * i + 2], b[2], f, scale);
      k = ((uint64_t)sg << (3 * kbits)) | (spread3(kx) << 2) | (spread3(ky) << 1) | spread3(kz);
      keys[i] = k;
      idx[i] = (uint32_t)i;
    }
    if (hist) count_digits(h, k, i < n, npass);
  }
  if (hist) flush_digits(h, npass, hist);
}

// Sorted position i of a batch lies in its problem's input range.  The sort
// left its result in one of two buffers (sel, known on the device); the keys
// and indices end up in the first.  Nothing if the sort failed.
__global__ void k_permute(const float* __restrict__ pos, const float* __restrict__ gam,
                          const float* __restrict__ sig, float sig_u, const float* __restrict__ seg_sig,
                          const int* __restrict__ off, int nseg, uint64_t* __restrict__ k0, uint32_t* __restrict__ v0,
                          const uint64_t* __restrict__ k1, const uint32_t* __restrict__ v1,
                          const int* __restrict__ sel, const int* __restrict__ failed, int64_t n,
                          float4* __restrict__ A, float4* __restrict__ B) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int second = *sel, bad = *failed;  // both loads in flight
  if (i >= n || bad) return;
  uint32_t j;
  if (second) {
    j = v1[i];
    v0[i] = j;
    k0[i] = k1[i];
  } else {
    j = v0[i];
  }
  const size_t q = 3 * (size_t)j;
  float s = sig ? sig[j] : (seg_sig ? seg_sig[seg_of(off, nseg, i)] : sig_u);
  A[i] = make_float4(pos[q], pos[q + 1], pos[q + 2], s);
  B[i] = make_float4(gam[q], gam[q + 1], gam[q + 2], 0.f);
}

__global__ void k_sigma_max(const float* __restrict__ sig, int64_t n, unsigned int* __restrict__ out) {
  float m = 0.f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    m = fmaxf(m, sig[i]);
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));  // sigma > 0: order of bits = order of values
}

__device__ inline int lower_bound_u64(const uint64_t* a, int lo, int hi, uint64_t v) {
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (a[mid] < v) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// ---- The octree as one cooperative kernel (like the traversal's frontier
// loop): per level the blocks own contiguous ranges of its cells, find the
// children (phase A), meet at a bounded grid barrier, take their output offsets
// from the block totals and write the children in digit order (phase B), and
// meet again; then the centres and the leaf list.  One launch and one host
// read instead of four launches and a read per level: 1000 blobs 0.29 -> 0.23
// ms, Plummer 30,011 (10 levels) 0.61 -> 0.39 ms for the tree phase.  When a
// level outgrows the cell arrays the blocks stop together before writing it;
// the host grows the arrays, keeping their contents, and the launch resumes.

constexpr int kTreeThreads = 256;

struct TreeState {
  int lb, le, level, nlevels, ncells, nleaves, overflow, need, done;
  int level_begin[kMaxLevel + 3];
  GridBar bar;
};

struct TreeArrays {
  int *begin, *end, *level, *parent, *child, *nchild;
  uint64_t* key;
  double* center;
  float4 *cf, *clo;  // the centre as a sum of two FP32 numbers (cf.w: the radius, later)
  unsigned long long* r2;
  uint32_t* r2f;     // bits of the largest FP32 squared distance
  int *leaves, *cseg, *bnd;
  uint32_t* cnt;
};

// Sum over the block; every thread gets it.
__device__ __forceinline__ uint32_t block_sum(uint32_t v, uint32_t* ws) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  uint32_t t = 0;
  for (int w = 0; w < kTreeThreads / 32; ++w) t += ws[w];
  __syncthreads();
  return t;
}

// Sum of the earlier blocks' totals, and of all.
__device__ __forceinline__ void block_offsets(const uint32_t* blk, unsigned G, unsigned b, uint32_t* ws, uint32_t& pre,
                                              uint32_t& all) {
  uint32_t p = 0, t = 0;
  for (unsigned j = threadIdx.x; j < G; j += kTreeThreads) {
    const uint32_t x = ((volatile const uint32_t*)blk)[j];
    t += x;
    if (j < b) p += x;
  }
  pre = block_sum(p, ws);
  all = block_sum(t, ws);
}

// Exclusive scan of one value per thread, with the block total.
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* ws, uint32_t& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) ws[w] = inc;
  __syncthreads();
  uint32_t before = 0;
  total = 0;
  for (int i = 0; i < kTreeThreads / 32; ++i) {
    const uint32_t x = ws[i];
    if (i < w) before += x;
    total += x;
  }
  __syncthreads();
  return before + inc - v;
}

__global__ void __launch_bounds__(kTreeThreads) k_tree_loop(const uint64_t* __restrict__ skeys, TreeArrays t, int n,
                                                            int nroot, const int* __restrict__ off,
                                                            const double* __restrict__ box, int kbits, int ncrit,
                                                            int cap, TreeState* st, uint32_t* __restrict__ blk,
                                                            int resume, long long spins,
                                                            const int* __restrict__ sort_failed) {
  __shared__ uint32_t ws[kTreeThreads / 32];
  const unsigned G = gridDim.x, b = blockIdx.x;
  const int lane = threadIdx.x & 31, d = threadIdx.x & 7;
  int lb = 0, le = nroot, l = 0;
  const int unsorted = *sort_failed;
  if (resume) {
    lb = st->lb;
    le = st->le;
    l = st->level;
  } else {  // root cells: one per problem (key = problem index)
    for (int r = (int)(b * kTreeThreads + threadIdx.x); r < nroot; r += (int)(G * kTreeThreads)) {
      t.begin[r] = off ? off[r] : 0;
      t.end[r] = off ? off[r + 1] : n;
      t.level[r] = 0;
      t.parent[r] = -1;
      t.key[r] = (uint64_t)r;
    }
    if (b == 0 && threadIdx.x == 0) {
      st->level_begin[0] = 0;
      st->level_begin[1] = nroot;
    }
    if (!grid_barrier(&st->bar, G, spins)) return;
  }
  if (unsorted) {  // give up as after an expired wait (the same in every block)
    if (b == 0 && threadIdx.x == 0) st->bar.abort = 1u;
    return;
  }
  for (;; ++l) {
    // phase A: 8 lanes per cell; lane d finds the first particle of child digit
    // d (a binary search in the cell's sorted keys; lane 0 holds the cell's begin)
    const int ncl = le - lb, chunk = (ncl + (int)G - 1) / (int)G;
    const int i0 = min(ncl, (int)b * chunk), i1 = min(ncl, i0 + chunk);
    uint32_t sum = 0;
    for (int base = i0; base < i1; base += kTreeThreads / 8) {
      const int i = base + (threadIdx.x >> 3), c = lb + i;
      const bool live = i < i1;
      int cb = 0, ce = 0;
      bool split = false;
      if (live) {
        cb = t.begin[c];
        ce = t.end[c];
        split = ce - cb > ncrit && l < kbits;
      }
      int bd = cb;
      if (split && d > 0)
        bd = lower_bound_u64(skeys, cb, ce, ((t.key[c] << 3) | (uint64_t)d) << (3 * (kbits - 1 - l)));
      // lane d's child is non-empty when the next bound (lane d + 1, or the end) is larger
      const int nb = __shfl_down_sync(0xffffffffu, bd, 1, 8);
      const int next = d == 7 ? ce : nb;
      const unsigned m = __ballot_sync(0xffffffffu, split && next > bd) >> (lane & ~7);
      if (live) {
        t.bnd[8 * (size_t)i + d] = bd;
        if (d == 0) {
          const uint32_t k = (uint32_t)__popc(m & 0xffu);
          t.cnt[i] = k;
          sum += k;
        }
      }
    }
    sum = block_sum(sum, ws);
    if (threadIdx.x == 0) blk[b] = sum;
    if (!grid_barrier(&st->bar, G, spins)) return;
    uint32_t pre, total;
    block_offsets(blk, G, b, ws, pre, total);
    if ((int64_t)le + total > (int64_t)cap) {  // every block sees the same totals
      if (b == 0 && threadIdx.x == 0) {
        st->overflow = 1;
        st->need = le + (int)total;
        st->lb = lb;
        st->le = le;
        st->level = l;
      }
      return;
    }
    // phase B: the children, in cell and digit order
    uint32_t run = (uint32_t)le + pre;
    for (int base = i0; base < i1; base += kTreeThreads / 8) {
      const int i = base + (threadIdx.x >> 3), c = lb + i;
      const bool live = i < i1;
      const uint32_t k = live ? t.cnt[i] : 0u;
      const int bd = live ? t.bnd[8 * (size_t)i + d] : 0, ce = live ? t.end[c] : 0;
      const int nb = __shfl_down_sync(0xffffffffu, bd, 1, 8);
      const int next = d == 7 ? ce : nb;
      const bool mine = live && k > 0 && next > bd;
      uint32_t tot;
      const uint32_t o = run + block_scan(mine ? 1u : 0u, ws, tot);
      // the cell's first child: the position of its first non-empty digit
      const unsigned m = (__ballot_sync(0xffffffffu, mine) >> (lane & ~7)) & 0xffu;
      const uint32_t first = __shfl_sync(0xffffffffu, o, (lane & ~7) | (m ? __ffs(m) - 1 : 0));
      if (live && d == 0) {
        t.nchild[c] = (int)k;
        t.child[c] = k ? (int)first : -1;
      }
      if (mine) {
        t.begin[o] = bd;
        t.end[o] = next;
        t.level[o] = l + 1;
        t.parent[o] = c;
        t.key[o] = (t.key[c] << 3) | (uint64_t)d;
      }
      run += tot;
    }
    if (!grid_barrier(&st->bar, G, spins)) return;
    if (total == 0) break;
    lb = le;
    le += (int)total;
    if (b == 0 && threadIdx.x == 0) st->level_begin[l + 2] = le;
  }
  // centres, and the leaves in cell order
  const int nc = le, chunk = (nc + (int)G - 1) / (int)G;
  const int i0 = min(nc, (int)b * chunk), i1 = min(nc, i0 + chunk);
  uint32_t sum = 0;
  for (int c = i0 + threadIdx.x; c < i1; c += kTreeThreads) {
    // cell key = problem index above the 3 l level-local Morton bits
    const int lv = t.level[c];
    const uint64_t kf = t.key[c];
    const int sg = (int)(kf >> (3 * lv));
    const uint64_t k = kf & ((1ull << (3 * lv)) - 1ull);
    const double* bx = box + 4 * sg;
    const double a = __dmul_rn(bx[3], ldexp(1.0, -lv));
    const uint32_t ijk[3] = {compact3(k >> 2), compact3(k >> 1), compact3(k)};
    double x[3];
    float hi[3], lo[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      x[q] = __dadd_rn(bx[q], __dmul_rn((double)ijk[q] + 0.5, a));
      t.center[3 * (size_t)c + q] = x[q];
      hi[q] = (float)x[q];
      lo[q] = (float)(x[q] - (double)hi[q]);
    }
    t.cf[c] = make_float4(hi[0], hi[1], hi[2], 0.f);
    t.clo[c] = make_float4(lo[0], lo[1], lo[2], 0.f);
    t.r2[c] = 0ull;
    t.r2f[c] = 0u;
    if (t.cseg) t.cseg[c] = sg;
    sum += t.nchild[c] == 0 ? 1u : 0u;
  }
  sum = block_sum(sum, ws);
  if (threadIdx.x == 0) blk[b] = sum;
  if (!grid_barrier(&st->bar, G, spins)) return;
  uint32_t pre, total;
  block_offsets(blk, G, b, ws, pre, total);
  for (int base = i0; base < i1; base += kTreeThreads) {
    const int c = base + threadIdx.x;
    const bool leaf = c < i1 && t.nchild[c] == 0;
    uint32_t tot;
    const uint32_t o = pre + block_scan(leaf ? 1u : 0u, ws, tot);
    if (leaf) t.leaves[o] = c;
    pre += tot;
  }
  if (b == 0 && threadIdx.x == 0) {
    st->overflow = 0;
    st->nlevels = l + 1;
    st->ncells = nc;
    st->nleaves = (int)total;
    st->done = 1;
  }
}

// Radius of a cell: the largest FP64 distance (explicitly rounded, fixed order)
// of its particles from its centre.  FP64 runs at a 64th of the FP32 rate here,
// so one warp per leaf walks the leaf's ancestors twice: the first pass takes
// the largest FP32 squared distance of each cell (the centre as a sum of two
// FP32 numbers, so the differences are good to 2^-23), the second the FP64
// distance of those particles alone that reach it up to the FP32 rounding;
// their maximum is the maximum of all.  Non-negative numbers order like their
// bit patterns, so both maxima are atomics.  One FP64 distance per particle and
// ancestor took 222 us at Taylor-Green 128^3, the two passes 184 us; at 1,000,000
// Plummer blobs the tree phase went from 1.44 to 0.84 ms with them.
__device__ __forceinline__ float dist2_f(const float4& a, const float4& h, const float4& l) {
  const float dx = (a.x - h.x) - l.x, dy = (a.y - h.y) - l.y, dz = (a.z - h.z) - l.z;
  return dx * dx + dy * dy + dz * dz;
}

template <bool EXACT>
__global__ void __launch_bounds__(256) k_radius(const float4* __restrict__ A, const TreeState* __restrict__ st,
                                                TreeArrays t) {
  const int lane = threadIdx.x & 31, nl = st->nleaves, done = st->done, bad = st->bar.abort;
  if (!done || bad) return;  // the cell arrays are being grown, or are not all there
  for (int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); w < nl; w += (int)((gridDim.x * blockDim.x) >> 5)) {
    const int leaf = t.leaves[w], b = t.begin[leaf], e = t.end[leaf];
    for (int c = leaf; c >= 0; c = t.parent[c]) {
      const float4 h = t.cf[c], l = t.clo[c];
      float m = 0.f;
      for (int i = b + lane; i < e; i += 32) m = fmaxf(m, dist2_f(A[i], h, l));
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (!EXACT) {
        const uint32_t bits = __float_as_uint(m);
        if (lane == 0 && bits > ((volatile uint32_t*)t.r2f)[c]) atomicMax(&t.r2f[c], bits);
        continue;
      }
      // twice the rounding of dist2_f: 8 2^-24 relative, and the 2^-48 |c| of the centre;
      // squares near the end of the FP32 range screen nothing
      const float top = __uint_as_float(t.r2f[c]);
      const float cm = fmaxf(fmaxf(fabsf(h.x), fabsf(h.y)), fabsf(h.z));
      const float low = top < 1e-30f ? 0.f : top - (4e-6f * top + sqrtf(top) * (2e-13f * cm));
      if (m < low) continue;
      const double cx = t.center[3 * (size_t)c], cy = t.center[3 * (size_t)c + 1], cz = t.center[3 * (size_t)c + 2];
      unsigned long long v = 0ull;
      for (int i = b + lane; i < e; i += 32) {
        const float4 a = A[i];
        if (dist2_f(a, h, l) < low) continue;
        const double dx = __dsub_rn((double)a.x, cx), dy = __dsub_rn((double)a.y, cy), dz = __dsub_rn((double)a.z, cz);
        const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
        const unsigned long long bits = (unsigned long long)__double_as_longlong(d2);
        v = v > bits ? v : bits;
      }
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, v, o);
        v = v > x ? v : x;
      }
      if (lane == 0) atomicMax(&t.r2[c], v);
    }
  }
}

__global__ void k_radius_final(const TreeState* __restrict__ st, TreeArrays t, double* __restrict__ R) {
  const int nc = st->ncells, done = st->done, bad = st->bar.abort;
  if (!done || bad) return;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
    const double r = __dsqrt_rn(__longlong_as_double((long long)t.r2[c]));
    R[c] = r;
    t.cf[c].w = (float)r;
  }
}

}  // namespace

int grow_cells(fmm_plan p, int64_t need, cudaStream_t s) {
  size_t ni = (size_t)need;
  FMM_TRY(p->c_begin.grow_copy(ni * sizeof(int), s));
  FMM_TRY(p->c_end.grow_copy(ni * sizeof(int), s));
  FMM_TRY(p->c_level.grow_copy(ni * sizeof(int), s));
  FMM_TRY(p->c_parent.grow_copy(ni * sizeof(int), s));
  FMM_TRY(p->c_child.grow_copy(ni * sizeof(int), s));
  FMM_TRY(p->c_nchild.grow_copy(ni * sizeof(int), s));
  FMM_TRY(p->c_key.grow_copy(ni * sizeof(uint64_t), s));
  return FMM_OK;
}

// Octree over the sorted keys (one root per problem), centres, leaves, radii.
static int tree_from_sorted(fmm_plan p, int64_t n, int nroot, const int* off, const double* box, int kbits,
                            bool with_seg, cudaStream_t s) {
  // at most 2^27 to begin with: more cells are not traversed
  int64_t cap = std::max<int64_t>(
      std::min<int64_t>(64 + 4 * n / std::max(1, p->prm.ncrit) + 2 * (int64_t)nroot, 1ll << 27), p->cell_cap);
  static int grid_blocks[64] = {0};
  const int dev = p->device >= 0 && p->device < 64 ? p->device : 0;
  if (!grid_blocks[dev]) {
    int sms = 0, per_sm = 0;
    FMM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device));
    FMM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tree_loop, kTreeThreads, 0));
    grid_blocks[dev] = std::max(1, sms * std::min(per_sm, 2));
  }
  // a block per 64 cells or so of the widest level; few blocks keep the
  // barriers of a small tree cheap
  const int64_t width = std::max<int64_t>(n / std::max(1, p->prm.ncrit), nroot);
  const unsigned G = (unsigned)std::min<int64_t>(grid_blocks[dev], std::max<int64_t>(1, width / 64));
  FMM_TRY(p->tree_state.ensure(sizeof(TreeState) + (size_t)grid_blocks[dev] * sizeof(uint32_t)));
  TreeState* st = p->tree_state.as<TreeState>();
  uint32_t* blk = reinterpret_cast<uint32_t*>(st + 1);
  FMM_CUDA_TRY(cudaMemsetAsync(st, 0, sizeof(TreeState), s));
  TreeState* hs = reinterpret_cast<TreeState*>(reinterpret_cast<char*>(p->pinned) + 3072);
  static_assert(sizeof(TreeState) <= 1024, "the tree state fits the pinned scratch");
  for (int launch = 0;; ++launch) {
    if (launch > 64 || cap > 0x7fffffff) return FMM_E_CAPACITY;
    FMM_TRY(grow_cells(p, cap, s));
    p->cell_cap = cap;
    FMM_TRY(p->c_center.ensure((size_t)cap * 3 * sizeof(double)));
    FMM_TRY(p->c_radius2.ensure((size_t)cap * sizeof(unsigned long long)));
    FMM_TRY(p->c_radius.ensure((size_t)cap * sizeof(double)));
    FMM_TRY(p->c_cf.ensure((size_t)cap * sizeof(float4)));
    FMM_TRY(p->c_clo.ensure((size_t)cap * (sizeof(float4) + sizeof(uint32_t))));
    FMM_TRY(p->leaves.ensure((size_t)(cap + 1) * sizeof(int)));
    FMM_TRY(p->tcount.ensure((size_t)(cap + 1) * sizeof(uint32_t)));
    FMM_TRY(p->tscan1.ensure((size_t)(8 * cap + 8) * sizeof(int)));  // child bounds (free until the traversal)
    if (with_seg) FMM_TRY(p->c_seg.ensure((size_t)cap * sizeof(int)));
    TreeArrays t;
    t.begin = p->c_begin.as<int>();
    t.end = p->c_end.as<int>();
    t.level = p->c_level.as<int>();
    t.parent = p->c_parent.as<int>();
    t.child = p->c_child.as<int>();
    t.nchild = p->c_nchild.as<int>();
    t.key = p->c_key.as<uint64_t>();
    t.center = p->c_center.as<double>();
    t.cf = p->c_cf.as<float4>();
    t.clo = p->c_clo.as<float4>();
    t.r2 = p->c_radius2.as<unsigned long long>();
    t.r2f = reinterpret_cast<uint32_t*>(t.clo + cap);
    t.leaves = p->leaves.as<int>();
    t.cseg = with_seg ? p->c_seg.as<int>() : nullptr;
    t.bnd = p->tscan1.as<int>();
    t.cnt = p->tcount.as<uint32_t>();
    const uint64_t* sk = p->skeys;
    int ni = (int)n, ncrit = p->prm.ncrit, icap = (int)cap, resume = launch > 0 ? 1 : 0;
    long long spins = p->wait_limit[FMM_WAIT_TREE];
    void* args[] = {&sk, &t, &ni, &nroot, &off, &box, &kbits, &ncrit, &icap, &st, &blk, &resume, &spins, &p->sort.failed};
    ++g_launches;
    FMM_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)k_tree_loop, dim3(G), dim3(kTreeThreads), args, 0, s));
    FMM_CUDA_TRY(cudaMemcpyAsync(hs, st, sizeof(TreeState), cudaMemcpyDeviceToHost, s));
    FMM_CUDA_TRY(cudaEventRecord(p->ev_read, s));
    // the radii run while the host reads the sizes (and at once if the tree is not done)
    const unsigned gr = (unsigned)std::min<int64_t>(8 * 152, cap / 8 + 1);
    g_launches += 3;
    k_radius<false><<<gr, 256, 0, s>>>(p->sortA.as<float4>(), st, t);
    k_radius<true><<<gr, 256, 0, s>>>(p->sortA.as<float4>(), st, t);
    k_radius_final<<<(unsigned)std::min<int64_t>(4 * 152, cap / 256 + 1), 256, 0, s>>>(st, t,
                                                                                      p->c_radius.as<double>());
    FMM_CUDA_TRY(cudaGetLastError());
    FMM_CUDA_TRY(cudaEventSynchronize(p->ev_read));
    if (hs->bar.abort) return FMM_E_TIMEOUT;
    if (hs->done) break;
    if (!hs->overflow) return FMM_E_CUDA;
    cap = 2 * (int64_t)hs->need;
  }
  p->ncells = hs->ncells;
  p->nleaves = hs->nleaves;
  p->nlevels = hs->nlevels;
  p->level_begin.assign(hs->level_begin, hs->level_begin + hs->nlevels + 1);
  return FMM_OK;
}

// Keys and their sort; passes over digits that no key changes are left out (a
// lattice leaves its low bits constant).
static int sort_particles(fmm_plan p, const float* pos, int64_t n, const double* box, const int* off, int nseg,
                          int kbits, int bits, cudaStream_t s) {
  const int npass = (bits + 7) / 8;
  p->skeys = p->keys0.as<uint64_t>();
  p->sidx = p->vals0.as<uint32_t>();
  FMM_TRY(sort_begin(p->sort, n, s));
  ++g_launches;
  k_keys<<<(unsigned)std::min<int64_t>(608, (n + 255) / 256), 256, 0, s>>>(
      pos, n, box, off, nseg, kbits, p->skeys, p->sidx, npass, &p->sort.state.as<SortState>()->hist[0][0]);
  FMM_CUDA_TRY(cudaGetLastError());
  if (n == 1) return FMM_OK;  // in order, in the first buffer (sel is 0)
  return sort_passes(p->sort, p->keys0.as<uint64_t>(), p->vals0.as<uint32_t>(), p->keys1.as<uint64_t>(),
                     p->vals1.as<uint32_t>(), n, npass, false, s);
}

static const int* sorted_sel(fmm_plan p, int bits) { return &p->sort.state.as<SortState>()->sel[(bits + 7) / 8]; }

// Keys, sort, permutation into sorted SoA, octree, centres, radii.
int build_tree(fmm_plan p, int64_t n, const float* pos, const float* gam, const float* sig, float sig_u,
               cudaStream_t s) {
  const int T = 256;
  unsigned nb = (unsigned)((n + T - 1) / T);
  double* box = p->scal.as<double>();
  p->batched = 0;
  p->nseg = 1;
  p->kbits = kMaxLevel;
  if (p->prm.periodic) {
    ++g_launches;
    k_set_box<<<1, 1, 0, s>>>(p->prm.box_min[0], p->prm.box_min[1], p->prm.box_min[2], p->prm.box_len, box);
  } else {
    int parts = (int)std::min<int64_t>(1024, (n + 255) / 256);
    FMM_TRY(p->scan_tmp.ensure((size_t)parts * 6 * sizeof(double)));
    ++g_launches;
    k_bbox_partial<<<parts, 256, 0, s>>>(pos, n, p->scan_tmp.as<double>());
    ++g_launches;
    k_bbox_final<<<1, 256, 0, s>>>(p->scan_tmp.as<double>(), parts, box);
  }
  // sigma max (uniform: the value itself)
  unsigned int* smax = reinterpret_cast<unsigned int*>(box + 8);
  if (sig) {
    FMM_CUDA_TRY(cudaMemsetAsync(smax, 0, sizeof(unsigned int), s));
    int parts = (int)std::min<int64_t>(1024, (n + 255) / 256);
    ++g_launches;
    k_sigma_max<<<parts, 256, 0, s>>>(sig, n, smax);
  }
  FMM_TRY(sort_particles(p, pos, n, box, nullptr, 1, kMaxLevel, 3 * kMaxLevel, s));
  ++g_launches;
  k_permute<<<nb, T, 0, s>>>(pos, gam, sig, sig_u, nullptr, nullptr, 1, p->keys0.as<uint64_t>(),
                             p->vals0.as<uint32_t>(), p->keys1.as<uint64_t>(), p->vals1.as<uint32_t>(),
                             sorted_sel(p, 3 * kMaxLevel), p->sort.failed, n, p->sortA.as<float4>(), p->sortB.as<float4>());
  FMM_CUDA_TRY(cudaGetLastError());
  return tree_from_sorted(p, n, 1, nullptr, box, kMaxLevel, false, s);
}

// Problem tables of a batch to the device (ranges, sigma, periodic cubes).
int upload_segments(fmm_plan p, const SegSpec& sg, cudaStream_t s) {
  const int S = sg.nseg;
  const size_t b_off = (size_t)(S + 1) * sizeof(int), b_sig = (size_t)S * sizeof(float),
               b_box = (size_t)S * 4 * sizeof(double);
  const size_t need = b_box + b_off + 2 * b_sig + 64;
  if (p->seg_pinned_bytes < need) {
    if (p->seg_pinned) cudaFreeHost(p->seg_pinned);
    p->seg_pinned = nullptr;
    p->seg_pinned_bytes = 0;
    if (cudaMallocHost(&p->seg_pinned, need) != cudaSuccess) return FMM_E_NOMEM;
    p->seg_pinned_bytes = need;
  }
  char* h = reinterpret_cast<char*>(p->seg_pinned);
  double* hbox = reinterpret_cast<double*>(h);
  int* hoff = reinterpret_cast<int*>(h + b_box);
  float* hsig = reinterpret_cast<float*>(h + b_box + b_off);
  unsigned int* hsm = reinterpret_cast<unsigned int*>(h + b_box + b_off + b_sig);
  memcpy(hoff, sg.h_off, b_off);
  FMM_TRY(p->seg_off.ensure(b_off));
  FMM_TRY(p->seg_box.ensure(b_box));
  FMM_TRY(p->seg_smax.ensure((size_t)S * sizeof(unsigned int)));
  FMM_TRY(p->seg_mac.ensure((size_t)S * sizeof(SegMac)));
  FMM_TRY(p->seg_p2p.ensure((size_t)S * sizeof(SegP2P)));
  FMM_CUDA_TRY(cudaMemcpyAsync(p->seg_off.ptr, hoff, b_off, cudaMemcpyHostToDevice, s));
  if (sg.h_box) {
    memcpy(hbox, sg.h_box, b_box);
    FMM_CUDA_TRY(cudaMemcpyAsync(p->seg_box.ptr, hbox, b_box, cudaMemcpyHostToDevice, s));
  }
  if (sg.h_sigma) {
    memcpy(hsig, sg.h_sigma, b_sig);
    memcpy(hsm, sg.h_sigma, b_sig);  // sigma > 0: its bits are the max of one value
    FMM_TRY(p->seg_sig.ensure(b_sig));
    FMM_CUDA_TRY(cudaMemcpyAsync(p->seg_sig.ptr, hsig, b_sig, cudaMemcpyHostToDevice, s));
    FMM_CUDA_TRY(cudaMemcpyAsync(p->seg_smax.ptr, hsm, b_sig, cudaMemcpyHostToDevice, s));
  }
  return FMM_OK;
}

// A forest of independent problems: problem index above kBatchBits Morton
// bits per axis, one root per problem, each problem its own cube and sigma.
int build_forest(fmm_plan p, int64_t n, const float* pos, const float* gam, const float* sig, const SegSpec& sg,
                 cudaStream_t s) {
  const int T = 256;
  const int S = sg.nseg;
  unsigned nb = (unsigned)((n + T - 1) / T);
  p->batched = 1;
  p->nseg = S;
  p->kbits = kBatchBits;
  FMM_TRY(upload_segments(p, sg, s));
  const int* off = p->seg_off.as<int>();
  double* box = p->seg_box.as<double>();
  if (!sg.h_box) {
    ++g_launches;
    k_bbox_seg<<<S, 256, 0, s>>>(pos, off, box);
  }
  if (sig) {
    ++g_launches;
    k_sigma_max_seg<<<S, 256, 0, s>>>(sig, off, p->seg_smax.as<unsigned int>());
  }
  int sbits = 0;
  while ((1 << sbits) < S) ++sbits;
  const int bits = 3 * kBatchBits + sbits;
  FMM_TRY(sort_particles(p, pos, n, box, off, S, kBatchBits, bits, s));
  ++g_launches;
  k_permute<<<nb, T, 0, s>>>(pos, gam, sig, 0.f, sig ? nullptr : p->seg_sig.as<float>(), off, S,
                             p->keys0.as<uint64_t>(), p->vals0.as<uint32_t>(), p->keys1.as<uint64_t>(),
                             p->vals1.as<uint32_t>(), sorted_sel(p, bits), p->sort.failed, n, p->sortA.as<float4>(),
                             p->sortB.as<float4>());
  FMM_CUDA_TRY(cudaGetLastError());
  return tree_from_sorted(p, n, S, off, box, kBatchBits, true, s);
}

}  // namespace fmm

namespace fmm {

// Cube and Morton keys into caller-provided memory (same arithmetic as
// build_tree): partials holds 1024*6 doubles, box 4 doubles.
int morton_keys_raw(int64_t n, const float* pos, int periodic, const double* box_min, double box_len,
                    uint64_t* keys, uint32_t* idx, double* partials, double* box, cudaStream_t s) {
  if (periodic) {
    ++g_launches;
    k_set_box<<<1, 1, 0, s>>>(box_min[0], box_min[1], box_min[2], box_len, box);
  } else {
    int parts = (int)std::min<int64_t>(1024, (n + 255) / 256);
    ++g_launches;
    k_bbox_partial<<<parts, 256, 0, s>>>(pos, n, partials);
    ++g_launches;
    k_bbox_final<<<1, 256, 0, s>>>(partials, parts, box);
  }
  ++g_launches;
  k_keys<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pos, n, box, nullptr, 1, kMaxLevel, keys, idx, 0, nullptr);
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

}  // namespace fmm
