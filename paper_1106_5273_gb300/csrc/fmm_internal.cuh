// Plan structure and the host-side entry points of each translation unit.
#pragma once

#include <algorithm>
#include <functional>
#include <vector>

#include "common.cuh"
#include "harmonics.cuh"
#include "primitives.cuh"

// Layout of the small device scalar block (doubles).
namespace fmm {
constexpr int kScalBox = 0;     // box_min[3], box_len
constexpr int kScalDipole = 4;  // dipole velocity correction [3] (double)
constexpr int kScalSigma = 8;   // float bits of max sigma (per-particle sigma)
constexpr int kScalCount = 16;  // u32 counters area
constexpr int kBarriers = 3;    // grid barriers with a limit of their own (the first of FMM_WAIT_*)
constexpr int kBatchBits = 16;  // Morton bits per axis of a batched evaluation (depth cap 16)
constexpr int kMaxBatch = 1 << (63 - 3 * kBatchBits);  // problems per batched evaluation

// Per-problem tables of a batched evaluation (one entry per non-empty problem).
struct SegMac {  // traversal: image shift and regularisation MAC (Sec. 3.3)
  double blen, smax;
  float blenf, ksf, slack0, pad;
};
// erfcx(1/y) ~ sum c_k y^k on [1/4.6, 1] (gen_cutoff_fit.py, degree 3)
constexpr float kE0 = -1.202012900e-02f, kE1 = 6.541014877e-01f, kE2 = -2.626216807e-01f,
                kE3 = 4.812366022e-02f;

// Constants of one core width sigma.  The polynomial H is stored negated
// (hn = -H) so that S = 1/r^3 + q (hn / r^2) is one FMA.
struct SigK {
  float kq;   // -log2(e) / (2 sigma^2)
  float kc;   // -sqrt(2/pi) / (3 sigma^3)   (T' = (S + kc q) / r^2)
  float ku;   // 1 / sigma^2
  float is3;  // 1 / sigma^3
  float is5;  // -2 / (3 sigma^5)            (near series: T' = f'(u) is5)
  float hn0;  // -sqrt(2/pi) / sigma          (constant term of -H)
  float hn1, hn2, hn3, hn4;  // -e_0 .. -e_3,  e_k = c_k (sqrt2 sigma)^k
};

__host__ __device__ inline SigK make_sigk(float sigma) {
  SigK k;
  // one FP64 division (k_sigk and k_direct evaluate this per particle)
  const double s = (double)sigma, ky = 1.4142135623730951 * s, i = 1.0 / s, i2 = i * i, i3 = i2 * i;
  k.kq = (float)(-0.72134752044448170 * i2);
  k.kc = (float)(-0.79788456080286535588 / 3.0 * i3);
  k.ku = (float)i2;
  k.is3 = (float)i3;
  k.is5 = (float)(-2.0 / 3.0 * (i3 * i2));
  k.hn0 = (float)(-0.79788456080286535588 * i);
  k.hn1 = (float)(-(double)kE0);
  k.hn2 = (float)(-(double)kE1 * ky);
  k.hn3 = (float)(-(double)kE2 * ky * ky);
  k.hn4 = (float)(-(double)kE3 * ky * ky * ky);
  return k;
}

struct SegP2P {  // near field: core width and its constants, class bounds, dipole correction
  SigK k;
  float smax, blen, margin;
  float dip[3];
};
// Error words and counts of an evaluation: one block on the device (fmm_plan_s::
// flags), copied whole whenever the host reads one of them.  The first four words
// are cleared at the start.
struct EvalStatus {
  int error;              // FMM_E_* raised by a kernel
  int failed, p_failed;   // a sort with fmm_plan_s::sort / p_sort failed
  uint32_t wide_tiles;    // M2L tiles if they took 64 cells
  uint32_t tiles, keys, steps, missing;  // M2L tiles, translations, steps, operators to build
  int rng[8];             // min and max of each field of the translation keys
};
// Barrier of the kernel that cuts the P2P lists into work items, and its counts
// (read by the host together).
struct ItemState {
  GridBar bar;
  uint32_t items, slots;
};
// Host description of a batch (problems concatenated; nullptr = one problem).
struct SegSpec {
  int nseg;
  const int* h_off;      // [nseg+1] particle ranges of the problems
  const float* h_sigma;  // [nseg] uniform sigma per problem, or nullptr (per-particle sigma)
  const double* h_box;   // [nseg][4] periodic cubes (min xyz, side), or nullptr (free space)
};
}  // namespace fmm

// Plan: parameters, constant operator tables, and the grow-only workspace.
struct fmm_plan_s {
  fmm_params prm;
  int64_t n_max = 0;
  int P = 0;      // p^2 real coefficients per potential
  int device = 0;
  int timing = 0;
  int tc_ok = 0;  // tensor-core M2L usable for this p
  int tc_kind = 0;  // tensor-core element kind: 0 BF16x3, 1 TF32x3 (FMM_M2L_TENSOR_TF32)
  // batched evaluation (several independent problems in one tree forest)
  int batched = 0;         // 1 while the last evaluation was a batch
  int nseg = 1;            // problems (non-empty) of the last evaluation
  int kbits = fmm::kMaxLevel;  // Morton bits per axis
  fmm::DBuf seg_off;       // int32 [nseg+1]
  fmm::DBuf seg_box;       // double [nseg][4]
  fmm::DBuf seg_sig;       // float [nseg] uniform sigma (batch with uniform sigma)
  fmm::DBuf seg_smax;      // u32 float bits [nseg] largest sigma
  fmm::DBuf seg_mac;       // SegMac [nseg]
  fmm::DBuf seg_p2p;       // SegP2P [nseg]
  fmm::DBuf c_seg;         // int32 problem of each cell
  void* seg_pinned = nullptr;  // host staging of the problem tables
  size_t seg_pinned_bytes = 0;
  // constant operator tables (device)
  fmm::DBuf m2m_T;    // [8][P(k)][P(r)] FP32 transposed M2M matrices by child octant
  fmm::DBuf l2l_T;    // [8][P(k)][P(r)] FP32 transposed L2L matrices by child octant
  fmm::DBuf l2p_tab;  // [5][P] int4 L2P gather table (indices into L~, signed weights)
  fmm::DBuf m2l_inu;  // [P] FP64 1 / nu of every coefficient (M2L operators)
  fmm::DBuf lattice;  // [P][P] FP64 periodic lattice operator (row = output)
  // particles
  fmm::DBuf keys0, keys1, vals0, vals1;  // radix sort ping-pong
  uint64_t* skeys = nullptr;             // sorted keys (points into keys0/keys1)
  uint32_t* sidx = nullptr;              // sorted position -> input index
  fmm::DBuf sortA, sortB;                // float4 (x,y,z,sigma), (gx,gy,gz,0) in sorted order
  fmm::DBuf far_u, far_s;                // [n][3] far field, sorted order
  fmm::DBuf near_u, near_s;              // [n][3] near field, sorted order
  fmm::DBuf c_clo;                       // float4 low part of the centre, then u32 FP32 squared radius
  fmm::DBuf tree_state;                  // state and block totals of the octree kernel
  fmm::DBuf in_pos, in_gam, in_sig, out_vel, out_dg;  // staging of the _host entry point
  fmm::DBuf t_pos, t_gam, t_sig, t_vel;                // sources + zero-strength targets (fmm_eval_targets)
  // cells
  fmm::DBuf c_begin, c_end, c_level, c_parent, c_child, c_nchild;  // int32
  fmm::DBuf c_key;                                                  // u64 level-local Morton index
  fmm::DBuf c_center, c_radius2, c_radius;                          // double[3], u64 bits, double
  fmm::DBuf c_cf;                                                   // float4 (centre, radius) rounded to FP32
  fmm::DBuf c_tile;                                                 // int32 tile*64+slot of each cell
  fmm::DBuf tile_cells;                                             // cell of each (tile, slot) position
  fmm::DBuf c_ijk;       // uint64 integer cell coordinates, 21 bits per axis
  fmm::DBuf tile_first;  // int32 [ntiles+1]: tile t = tile_cells[tile_first[t] .. tile_first[t+1])
  fmm::DBuf tile_groups; // int32 (level, octant) cell counts, then cell and tile offsets of the groups
  fmm::DBuf leaves;                                                 // leaf cell ids
  fmm::DBuf M, L;                                                   // [cells][3][P] FP32
  fmm::DBuf Mbf;  // [cells][hi/lo][3][K chunks x 128 bytes] BF16 or TF32 hi/lo
  // traversal
  fmm::DBuf fr0, fr1;                                 // frontier int4 (a,b,o,0)
  fmm::DBuf tcount, tmask, tscan0, tscan1, tscan2;    // per-item scratch
  fmm::DBuf p2p_raw, m2l_raw;                         // int4 (a,b,o,0)
  fmm::DBuf lk0, lk1, lv0, lv1;                       // list sort ping-pong
  fmm::DBuf p2p_sorted, p2p_off;                      // int2 (first source, image) by leaf, CSR offsets per leaf
  fmm::DBuf p2p_pre;                                  // u32 scanned source counts of the list entries
  fmm::DBuf p2p_items, p2p_islot, p2p_plan;           // pair kernel work items, their partial slots, per-leaf split
  fmm::DBuf p2p_bar, p2p_partial, p2p_sigk;                    // partial sums of split lists; per-particle core constants
  fmm::DBuf m2l_key, m2l_slot, ukeys;                 // per pair key, slot; unique keys
  fmm::DBuf T32, Tbf;                                 // M2L operator cache [slot]: FP32, BF16 hi/lo
  fmm::DBuf tc_key, tc_slot;                          // operator cache: open-addressing table key -> slot
  int64_t tc_cap = 0, tc_size = 0;                    // table entries; operators in it
  int64_t tcache_cap = 0;                             // operators T32 / Tbf have room for
  fmm::DBuf tmiss_keys, tmiss_slots, tslot_map;       // keys to build, their slots; unique key -> slot
  int64_t n_built = 0;                                // operators built by the last evaluation
  fmm::DBuf st_tile, st_slot, st_src, tile_range;     // M2L steps
  fmm::DBuf bin_flag, bin_scan, bin_flag2, bin_scan2;  // binned step build: key and bin tables
  fmm::DBuf st_ckey, st_fkey;                         // compact / full translation key per step
  fmm::DBuf m2l_items, m2l_partial;                   // M2L work items (+ split list); partial sums
  // scratch
  fmm::DBuf scan_tmp;
  fmm::SortScratch sort;
  fmm::DBuf pk0, pk1, pv0, pv1, p_scan;  // the P2P grouping's own list sort and scan (it runs beside the M2L lists)
  fmm::SortScratch p_sort;
  fmm::DBuf scal;   // small scalars (see kScal*)
  fmm::DBuf flags;  // EvalStatus
  void* pinned = nullptr;  // host pinned scratch (counts)
  // host mirror of the last tree / lists
  std::vector<int> level_begin;  // cells of level l: [level_begin[l], level_begin[l+1])
  int64_t cell_cap = 0;          // cells the arrays were asked to hold
  int64_t ncells = 0, nleaves = 0, ntiles = 0;
  int nlevels = 0;
  double cf_margin = 0.0;  // rounding margin of the FP32 cell copies (2e-6 x largest coordinate)
  int64_t n_p2p = 0, n_m2l = 0, n_keys = 0, n_steps = 0, p2p_pairs = 0;
  int64_t n_p2p_items = 0, n_p2p_slots = 0;  // pair kernel work items and partial slots
  int64_t last_n = 0;
  int last_tc = 0;
  int m2l_stage_chunks = 0;  // K chunks per stage of the last tensor-core M2L
  fmm::DBuf dip_part;        // partial sums of the dipole term (written beside the traversal)
  // tree reuse (fmm_eval_strengths): set by a successful full evaluation of
  // the plan's own particles; epoch counts full evaluations (a captured graph
  // is valid only within the epoch it was captured in)
  int reuse_ok = 0;
  int reuse_ps = 0;         // the last evaluation had a per-particle sigma array
  float reuse_sig_u = 0.f;  // its uniform sigma
  double reuse_smax = 0.0;  // its largest sigma
  int64_t epoch = 0;
  // list capacities the next traversal starts from (0: from the cell count);
  // a traversal whose lists outgrow them grows them and runs again
  int64_t cap_fr0 = 0, cap_m0 = 0, cap_p0 = 0;
  int64_t trav_runs = 0;  // traversal launches of the last evaluation
  int64_t hw_fr = 0, hw_m = 0, hw_p = 0;  // list sizes the plan's evaluations needed (+1/8)
  fmm_stats stats;
  cudaEvent_t ev[8];
  int have_events = 0;
  // the upward pass runs on this plan stream while the traversal runs on the
  // caller's stream (both read only the tree); fork / join by events
  cudaStream_t s_up = nullptr;
  // the M2L lists, the M2L and the downward pass run on this one (highest
  // priority) while the near field runs on the caller's
  cudaStream_t s_far = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr, ev_up = nullptr, ev_near = nullptr;
  cudaEvent_t ev_read = nullptr;  // the host's reads of list sizes
  long long wait_limit[fmm::kBarriers] = {fmm::kGridSpin, fmm::kGridSpin, fmm::kGridSpin};  // polls (fmm_plan_set_wait_limit)
};

namespace fmm {
// tree.cu
int grow_cells(fmm_plan p, int64_t need, cudaStream_t s);
int build_tree(fmm_plan p, int64_t n, const float* pos, const float* gam, const float* sig, float sig_u,
               cudaStream_t s);
int upload_segments(fmm_plan p, const SegSpec& sg, cudaStream_t s);
int build_forest(fmm_plan p, int64_t n, const float* pos, const float* gam, const float* sig, const SegSpec& sg,
                 cudaStream_t s);
// operators.cu
int build_constant_operators(fmm_plan p);
int find_m2l_operators(fmm_plan p, uint32_t* miss, uint32_t* rank, uint32_t* nmiss, cudaStream_t s);
int build_m2l_operators(fmm_plan p, int64_t nmiss, uint32_t* miss, uint32_t* rank, uint32_t* nmiss_dev,
                        cudaStream_t s);
int remap_step_slots(fmm_plan p, cudaStream_t s);
int apply_lattice(fmm_plan p, cudaStream_t s);
int lattice_operator_host(int p, int images, double* out);
// lattice.cu
int lattice_operator_device(int p, int images, double* A, cudaStream_t s);
// upward.cu
int upward_pass(fmm_plan p, cudaStream_t s);
int dipole_pass(fmm_plan p, int64_t n, cudaStream_t s);
// traverse.cu
// lists of both fields: the P2P lists on s, the M2L lists on f (which may be s);
// near() launches the near field on s as soon as its lists are ready
int traverse(fmm_plan p, double sigma_max_host, cudaStream_t s, cudaStream_t f, const std::function<int()>& near);
// per-problem MAC and near-field tables of a batch (after the forest is built)
int segment_tables(fmm_plan p, int per_particle_sigma, cudaStream_t s);
// m2l.cu
int m2l_simt(fmm_plan p, cudaStream_t s);
int m2l_build_items(fmm_plan p, cudaStream_t s);  // once per tree
int m2l_tensor(fmm_plan p, cudaStream_t s);
// downward.cu
int downward_pass(fmm_plan p, int64_t n, cudaStream_t s);
// fmm_api.cu
int far_field(fmm_plan p, int64_t n, cudaStream_t s, const std::function<void()>& after_m2l);
// reuse.cu
int eval_strengths(fmm_plan p, const float* gam, float* vel, float* dg, cudaStream_t s);
// p2p.cu
int p2p_near(fmm_plan p, int64_t n, float sig_u, int per_particle_sigma, double smax, bool stretching,
             cudaStream_t s);
int p2p_finish(fmm_plan p, int64_t n, float* vel, float* dg, cudaStream_t s);
// work items of the pair kernel, counted in *p->p2p_bar (ItemState)
int p2p_tile(fmm_plan p);
int p2p_build_items(fmm_plan p, int64_t n, int64_t tile_sources, cudaStream_t s);
int p2p_direct_all(int64_t n, const float* pos, const float* gam, const float* sig, float sig_u, float* vel,
                   float* dg, cudaStream_t s);
}  // namespace fmm

namespace fmm {
// M2L translation key (level-independent thanks to the cell-size scaling):
// delta = level(target) - level(source); t = 2 (c_t - c_s - o L) / a_f with
// a_f the side of the finer of the two cells (an integer vector).
// Bits: [57,63) delta+32, [38,57) tx, [19,38) ty, [0,19) tz (two's complement).
constexpr int kKeyBits = 19;
constexpr long long kKeyLim = (1ll << (kKeyBits - 1)) - 1;

__host__ __device__ inline uint64_t m2l_key_encode(int delta, long long tx, long long ty, long long tz) {
  const uint64_t mask = (1ull << kKeyBits) - 1ull;
  return ((uint64_t)(delta + 32) << 57) | (((uint64_t)tx & mask) << 38) | (((uint64_t)ty & mask) << 19) |
         ((uint64_t)tz & mask);
}

__host__ __device__ inline long long key_field(uint64_t key, int shift) {
  long long v = (long long)((key >> shift) & ((1ull << kKeyBits) - 1ull));
  if (v >= (1ll << (kKeyBits - 1))) v -= (1ll << kKeyBits);
  return v;
}

// delta and tau = (c_t - c_s)/a_t (target-cell units); a_s/a_t = 2^delta.
__host__ __device__ inline void m2l_key_decode(uint64_t key, int* delta, double tau[3]) {
  int d = (int)(key >> 57) - 32;
  *delta = d;
  double f = 0.5 * (d < 0 ? ldexp(1.0, d) : 1.0);
  tau[0] = (double)key_field(key, 38) * f;
  tau[1] = (double)key_field(key, 19) * f;
  tau[2] = (double)key_field(key, 0) * f;
}

// K chunks of 64 coefficients (4 MMA K-steps of 16) covering P inputs.
// Tensor-core M2L element kinds: 0 = BF16 (kind::f16, K step 16), 1 = TF32
// (kind::tf32, K step 8).  A K chunk is one 128-byte row of either: 64 BF16 or
// 32 TF32 values, 4 K steps.
__host__ __device__ inline int m2l_kstep(int kind) { return kind ? 8 : 16; }
__host__ __device__ inline int m2l_kchunks(int P, int kind = 0) {
  return ((P + m2l_kstep(kind) - 1) / m2l_kstep(kind) + 3) / 4;
}
// K chunks of the BF16 tensor-core M2L that take all three split products.
// Under the MAC (R_A + R_B < theta |X_A - X_B|) the M2L terms of source
// degree j sum to at most theta^j / (1 - theta) of the leading 1/|X_A - X_B|
// term.  BF16 chunks from the second on hold degrees >= 8 (64 coefficients
// per chunk), so one hi x hi product there (relative error <= 2^-8) adds at
// most 2^-8 theta^8 / (1 - theta) of the leading term: <= 7e-6 for
// theta <= 0.42, whose theta^8 <= 2^-10.  Otherwise, and for TF32, every
// chunk takes three products.
__host__ __device__ inline int m2l_split_chunks(int P, int kind, float theta, bool full) {
  const int nkc = m2l_kchunks(P, kind);
  const float t2 = theta * theta, t8 = t2 * t2 * t2 * t2;
  return (kind == 0 && !full && t8 <= 1.0f / 1024.0f) ? 1 : nkc;
}
// Output coefficients padded to the columns of an MMA (N a multiple of 16).
__host__ __device__ inline int m2l_cols(int P) { return (P + 15) & ~15; }
// Target cells per M2L tile.  With 64 < P <= 128 the operator's P rows are the
// MMA's 128 rows (64 cells x 3 components as columns); otherwise the cells are
// the rows and the P coefficients the columns, which fits any P (both forms
// measured: m2l_tc.cu).  The SIMT M2L reads an operator once per tile and takes
// the wide tiles at any P (Plummer 30,011 at p = 12: 465 ms, 518 with 42 cells), but
// in a batch, where one CTA per tile waits for the longest, the same as the other
// (32 problems of 20,000 at p = 6: 96 ms, 117 with 64 cells).
inline int m2l_tile(fmm_plan p) {
  return (p->last_tc || p->batched) && (p->P <= 64 || p->P > 128) ? kTileCells : kTileRows;
}
// Bucket of a translation: a hash of its key, so that it depends on nothing else.
__host__ __device__ inline int m2l_bucket(uint64_t key) {
  return (int)((key * 0x9E3779B97F4A7C15ull) >> 61) & (kKeyBuckets - 1);
}
}  // namespace fmm
