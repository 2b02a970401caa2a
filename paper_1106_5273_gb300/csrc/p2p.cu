// Near field: the P2P kernel (Sec. 3.1, 3.6; Table 1 counts its flops) and
// the final combine / un-permute.
//
// Per pair (d = x_i - x_j, r = |d|, rho = r/sigma_j, x = rho/sqrt2, c = sqrt(2/pi)):
//   q = exp(-x^2)                       (one ex2)
//   g = 1 - q (erfcx(x) + 2x/sqrt(pi))  (Eq. 2; erfcx by a degree-3 fit in
//                                         y = 1/x = sqrt2 sigma / r, gen_cutoff_fit.py;
//                                         rho^2 < 2 uses the Taylor series of g/rho^3)
//   S = g / r^3 = 1/r^3 - q H / r^2 with H = (erfcx fit + 2x/sqrt(pi)) / r, i.e.
//       H = sqrt(2/pi)/sigma + e_0/r + e_1/r^2 + e_2/r^3 + e_3/r^4,  e_k = c_k (sqrt2 sigma)^k
//       (one Horner polynomial in 1/r: 2x/sqrt(pi) / r is the constant term)
//   T = (c q / sigma^3 - 3 S) / r^2 = S'(r)/r; the kernels carry T' = -T/3 =
//       (S - c q / (3 sigma^3)) / r^2 (no multiply by -3 per pair) and scale the
//       stretching sums by -3 once per target
//   u_i += S (gamma_j x d)                                            (Eq. 1)
//   s_i += S (gamma_j x gamma_i) + T (gamma_i . d)(gamma_j x d)       (Eq. 3)
//   or, transpose scheme (grad u)^T gamma_i:
//   s_i += S (gamma_i x gamma_j) + T (gamma_i . (gamma_j x d)) d
// The gamma_j x gamma_i part is summed as (sum_j S gamma_j) x gamma_i.  The
// self pair is skipped explicitly (its exact value is zero).  Periodic image
// pairs form the exact FP32 difference first and then add the image shift.
//
// A CTA of one warp takes a tile of at most 64 targets of a leaf and a range of
// the leaf's sources; the sources are staged through shared memory in chunks of
// 64.  Each staged source is classified by a lower
// bound on its distance to every target of the tile (its distance to the
// targets' bounding box, rounding margin off): the singular kernel where
// g = 1 to FP32 precision (rho >= 6.5), the cutoff without the series test
// (rho^2 >= 2), or the full form; a chunk is staged grouped by class, so each
// group runs its own branch-free loop.
#include <cooperative_groups.h>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

constexpr float kInv4Pi = 0.0795774715459476679f;
constexpr float kM3 = -3.f;  // T = -3 T': scales the stretching sums built from T'
// Source-leaf classes by a lower bound d_min on the pair distance:
//   kFar : d_min >= 6.5 sigma_max: 1 - g < 4e-9 and exp(-rho^2/2) < 1e-9, so
//          S = 1/r^3 and T = -3/r^5 exactly in FP32 (singular kernel);
//   kMid : d_min >= sqrt2 sigma_max: rho^2 >= 2, no series branch needed;
//   kNear: anything closer (series branch when rho^2 < 2).
constexpr int kNear = 0, kMid = 1, kFar = 2;
constexpr double kFarRho = 6.5, kMidRho = 1.4142135623730951;

constexpr double ser_coef(int k) {  // c (-1)^k / (2^k k! (2k+3))
  double d = 2.0 * k + 3.0;
  for (int i = 1; i <= k; ++i) d *= 2.0 * i;
  return ((k & 1) ? -1.0 : 1.0) * 0.79788456080286535588 / d;
}
constexpr int kSerTerms = 12;
__constant__ float cSer[kSerTerms] = {
    (float)ser_coef(0), (float)ser_coef(1), (float)ser_coef(2),  (float)ser_coef(3),
    (float)ser_coef(4), (float)ser_coef(5), (float)ser_coef(6),  (float)ser_coef(7),
    (float)ser_coef(8), (float)ser_coef(9), (float)ser_coef(10), (float)ser_coef(11)};

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The constants of make_sigk for the mixed core width of a pair,
// sigma_ij^2 = (sigma_i^2 + sigma_j^2) / 2, in FP32 (one division and one
// rsqrt per pair).
__device__ __forceinline__ SigK sigk_mixed(float si, float sj) {
  const float s2 = 0.5f * fmaf(si, si, sj * sj);
  const float iu = 1.f / s2;        // 1 / sigma^2
  const float is = rsqrtf(s2);      // 1 / sigma
  const float sg = s2 * is;         // sigma
  const float is3 = iu * is;        // 1 / sigma^3
  SigK k;
  k.kq = -0.72134752044448170f * iu;  // -log2(e) / 2
  k.kc = -0.26596152026762179f * is3;  // -sqrt(2/pi) / 3
  k.ku = iu;
  k.is3 = is3;
  k.is5 = (-2.f / 3.f) * is3 * iu;
  k.hn0 = -0.79788456080286535588f * is;
  k.hn1 = -kE0;
  k.hn2 = -kE1 * 1.41421356237309515f * sg;
  k.hn3 = -kE2 * 2.f * s2;
  k.hn4 = -kE3 * 2.82842712474619030f * s2 * sg;
  return k;
}

// Axis-aligned bounding box of the targets of one tile, relative to the leaf
// centre (the coordinates the targets carry).
struct TileBox {
  float lx, ly, lz, hx, hy, hz;
};

// Box of the target coordinates x[q], y[q], z[q] (q < TPT) over the warp;
// lanes flag the targets that exist (valid[q]).
template <int TPT>
__device__ __forceinline__ TileBox tile_box(const float* x, const float* y, const float* z, const bool* valid) {
  TileBox b{INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
  for (int q = 0; q < TPT; ++q)
    if (valid[q]) {
      b.lx = fminf(b.lx, x[q]);
      b.ly = fminf(b.ly, y[q]);
      b.lz = fminf(b.lz, z[q]);
      b.hx = fmaxf(b.hx, x[q]);
      b.hy = fmaxf(b.hy, y[q]);
      b.hz = fmaxf(b.hz, z[q]);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    b.lx = fminf(b.lx, __shfl_xor_sync(0xffffffffu, b.lx, o));
    b.ly = fminf(b.ly, __shfl_xor_sync(0xffffffffu, b.ly, o));
    b.lz = fminf(b.lz, __shfl_xor_sync(0xffffffffu, b.lz, o));
    b.hx = fmaxf(b.hx, __shfl_xor_sync(0xffffffffu, b.hx, o));
    b.hy = fmaxf(b.hy, __shfl_xor_sync(0xffffffffu, b.hy, o));
    b.hz = fmaxf(b.hz, __shfl_xor_sync(0xffffffffu, b.hz, o));
  }
  return b;
}

// Class of a staged source at X (relative to the target leaf centre, image
// shift included) for the targets of a tile inside box b of a leaf of radius
// Rt: the distance from X to the box bounds its distance to every target from
// below; the bound is lowered by a margin covering the FP32 rounding of the
// coordinates (which are at most d + 2 Rt in size), so the class is never
// more optimistic than exact arithmetic would give.
__device__ __forceinline__ int source_class(float X, float Y, float Z, const TileBox& b, float Rt, float smax,
                                            float margin0) {
  const float ex = fmaxf(fmaxf(b.lx - X, X - b.hx), 0.f);
  const float ey = fmaxf(fmaxf(b.ly - Y, Y - b.hy), 0.f);
  const float ez = fmaxf(fmaxf(b.lz - Z, Z - b.hz), 0.f);
  const float d = sqrtf(ex * ex + ey * ey + ez * ez);
  const float dmin = d - (margin0 + 1e-6f * (d + 2.f * Rt));
  if (dmin >= (float)kFarRho * smax) return kFar;
  if (dmin >= (float)kMidRho * smax) return kMid;
  return kNear;
}

// Staging slots of this lane's sources j = lane + 32 q (class cls[q], -1 if
// j >= cnt): far sources first, then mid, then near, each group in source
// order.  nf and nm (the far and mid counts) come out equal in every lane.
// When every source is near the slot of source j is j.
template <int TPT>
__device__ __forceinline__ void group_slots(const int* cls, int lane, int* slot, int& nf, int& nm) {
  unsigned bf[TPT], bm[TPT], bn[TPT];
#pragma unroll
  for (int q = 0; q < TPT; ++q) {
    bf[q] = __ballot_sync(0xffffffffu, cls[q] == kFar);
    bm[q] = __ballot_sync(0xffffffffu, cls[q] == kMid);
    bn[q] = __ballot_sync(0xffffffffu, cls[q] == kNear);
  }
  nf = 0;
  nm = 0;
#pragma unroll
  for (int q = 0; q < TPT; ++q) {
    nf += __popc(bf[q]);
    nm += __popc(bm[q]);
  }
  const unsigned lt = (1u << lane) - 1u;
  int ef = 0, em = 0, en = 0;  // members of each class among the earlier q
#pragma unroll
  for (int q = 0; q < TPT; ++q) {
    if (cls[q] == kFar) slot[q] = ef + __popc(bf[q] & lt);
    else if (cls[q] == kMid) slot[q] = nf + em + __popc(bm[q] & lt);
    else if (cls[q] == kNear) slot[q] = nf + nm + en + __popc(bn[q] & lt);
    else slot[q] = -1;
    ef += __popc(bf[q]);
    em += __popc(bm[q]);
    en += __popc(bn[q]);
  }
}

// ---- The pair kernel.  Two pairs at a time run as the two lanes of the
// FP32x2 instructions (fma/mul/add .f32x2): the FMA pipe does the same work
// per clock as with scalars, in half the issue slots.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

// The constants of two pairs.
struct SigK2 {
  float2 kq, kc, ku, is3, is5, hn0, hn1, hn2, hn3, hn4;
};

__device__ __forceinline__ SigK2 make_sigk2(const SigK& a, const SigK& b) {
  SigK2 k;
  k.kq = make_float2(a.kq, b.kq);
  k.kc = make_float2(a.kc, b.kc);
  k.ku = make_float2(a.ku, b.ku);
  k.is3 = make_float2(a.is3, b.is3);
  k.is5 = make_float2(a.is5, b.is5);
  k.hn0 = make_float2(a.hn0, b.hn0);
  k.hn1 = make_float2(a.hn1, b.hn1);
  k.hn2 = make_float2(a.hn2, b.hn2);
  k.hn3 = make_float2(a.hn3, b.hn3);
  k.hn4 = make_float2(a.hn4, b.hn4);
  return k;
}

// Sums of two chains in the leaf-relative form: with X = x - c (c the target
// leaf's centre, image shifts folded into the source's X) and k_j =
// gamma_j x X_j staged per source,  sum_j S (gamma_j x d) = A x X_i - B  and
// sum_j T (gamma_i . d)(gamma_j x d) = C x X_i - D, where A = sum S gamma_j,
// B = sum S k_j, C = sum td gamma_j, D = sum td k_j, td = T' (gamma_i . d)
// (T' = -T/3, so the stretching is s = A x gamma_i - 3 (C x X_i - D)).
// Transpose scheme: with m_i = X_i x gamma_i, w = T' gamma_i . (gamma_j x d) =
// T' (gamma_j . m_i - gamma_i . k_j); cx holds W = sum w and D = sum w (-X_j)
// (the staged coordinates are negated); s = gamma_i x A - 3 (W X_i + D).
struct AccR2 {
  float2 ax, ay, az, bx, by, bz, cx, cy, cz, dx, dy, dz;
};

// S = g/r^3 and T' = -S'(r)/(3r) of two pairs (see the file header); ST = 0: S
// only (velocity without stretching).
template <int MODE, int ST>
__device__ __forceinline__ void pair_ST2(float2 r2, const SigK2& K, float2& S, float2& T) {
  const float2 rinv = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
  const float2 rinv2 = mul2(rinv, rinv);
  T = dup2(0.f);
  if (MODE == kFar) {
    S = mul2(rinv2, rinv);
    if (ST) T = mul2(S, rinv2);
    return;
  }
  const float2 rinv3 = mul2(rinv2, rinv);
  const float2 qa = mul2(r2, K.kq);
  const float2 q = make_float2(ex2_approx(qa.x), ex2_approx(qa.y));
  // beyond the fit range (x > 4.6) exp(-x^2) < 8e-10 multiplies a bounded
  // polynomial, so g = 1 to FP32 precision without clamping
  const float2 hn = fma2(fma2(fma2(fma2(K.hn4, rinv, K.hn3), rinv, K.hn2), rinv, K.hn1), rinv, K.hn0);
  S = fma2(q, mul2(rinv2, hn), rinv3);
  if (ST) T = mul2(fma2(K.kc, q, S), rinv2);
  if (MODE == kNear) {
    const float2 u = mul2(r2, K.ku);
    if (u.x < 2.f || u.y < 2.f) {
      float2 sS = dup2(cSer[kSerTerms - 1]), sT = dup2((float)(kSerTerms - 1) * cSer[kSerTerms - 1]);
#pragma unroll
      for (int k = kSerTerms - 2; k >= 0; --k) {
        sS = fma2(sS, u, dup2(cSer[k]));
        if (ST && k >= 1) sT = fma2(sT, u, dup2((float)k * cSer[k]));
      }
      const float2 Ss = mul2(sS, K.is3), Ts = mul2(sT, K.is5);
      if (u.x < 2.f) {
        S.x = Ss.x;
        T.x = Ts.x;
      }
      if (u.y < 2.f) {
        S.y = Ss.y;
        T.y = Ts.y;
      }
    }
  }
}

// The targets of a lane's two chains (narrow tiles: the same target twice).
struct Tgt2 {
  float2 x, y, z, gx, gy, gz;    // X_i and gamma_i
  float2 mx, my, mz, ngx, ngy, ngz;  // m_i = X_i x gamma_i and -gamma_i (transpose scheme)
  float2 sg;                     // sigma_i (mixed core width)
  int id0, id1;                  // their sorted positions
};

constexpr int kCh = 64;        // sources staged at a time
constexpr int kChPad = 72;     // slots of a staged narrow chunk (padded to a whole unit of 2, 4 or 8)

// The staged sources, every value once.  PAIR (narrow tiles): rows of kChPad
// floats (-X, -Y, -Z, gamma, k), read as float2 = two sources.  Wide tiles:
// (-X, -Y, -Z, gamma_x), (gamma_y, gamma_z, k_x, k_y), k_z per source, each
// value copied to both halves of its register pair after the load: the loop
// is bound by the FMA pipe and the shared-memory reads together, and storing
// every value twice (two and a half times the wavefronts) measured 73 instead
// of 66 cycles per 64 far pairs and warp scheduler, 92 instead of 87 mid.
// id = the source's sorted position (-1 for an image: never the target
// itself).  k (PS = 1): the constants of SigK, PAIR as rows kq kc hn0 hn2 hn3
// hn4 ku is3 is5, wide as two float4 rows and is5; (PS = 2): sigma_j.  The
// next chunk's loads go through shared memory (cp.async) and the targets' box
// is kept there, which leaves the registers to the pair loops.
template <int PS>
struct Stage {
  float4 v[9 * kChPad / 4];
  float4 k[PS == 1 ? 9 * kChPad / 4 : (PS == 2 ? kChPad / 4 : 1)];
  int id[kChPad];
  // the next chunk on its way (each lane reads back its own two sources)
  float4 raw[PS == 1 ? 5 : 2][kCh];
  int rid[kCh], rimg[kCh];
  TileBox box;
  float4 centre;
};

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Sources [jb, je) of a staged chunk in form MODE (PAIR: units of two sources,
// in steps of `step` units).  The near form skips the self pair.
// PS: 0 one core width, 1 sigma_j of the source, 2 the mixed width sigma_ij.
// ST: 0 velocity only, 1 classical stretching, 2 transpose stretching.
template <int MODE, bool PAIR, int PS, int ST>
__device__ __forceinline__ void run_group(const Stage<PS>& sm, int jb, int je, int step, const Tgt2& t,
                                          const SigK2& K0, AccR2& a) {
#pragma unroll(MODE == kNear ? 2 : 4)
  for (int j = jb; j < je; j += PAIR ? step : 1) {
    float2 nx, ny, nz, gjx, gjy, gjz, kjx, kjy, kjz;
    if (PAIR) {
      const float2* r = reinterpret_cast<const float2*>(sm.v) + j;
      constexpr int S = kChPad / 2;
      nx = r[0];
      ny = r[S];
      nz = r[2 * S];
      gjx = r[3 * S];
      gjy = r[4 * S];
      gjz = r[5 * S];
      kjx = r[6 * S];
      kjy = r[7 * S];
      kjz = r[8 * S];
    } else {
      const float4 v0 = sm.v[j], v1 = sm.v[kCh + j];
      nx = dup2(v0.x);
      ny = dup2(v0.y);
      nz = dup2(v0.z);
      gjx = dup2(v0.w);
      gjy = dup2(v1.x);
      gjz = dup2(v1.y);
      kjx = dup2(v1.z);
      kjy = dup2(v1.w);
      kjz = dup2(reinterpret_cast<const float*>(sm.v + 2 * kCh)[j]);
    }
    SigK2 K = K0;
    if constexpr (PS == 1 && MODE != kFar) {
      if constexpr (PAIR) {
        const float2* r = reinterpret_cast<const float2*>(sm.k) + j;
        constexpr int S = kChPad / 2;
        K.kq = r[0];
        K.kc = r[S];
        K.hn0 = r[2 * S];
        K.hn2 = r[3 * S];
        K.hn3 = r[4 * S];
        K.hn4 = r[5 * S];
        if (MODE == kNear) {
          K.ku = r[6 * S];
          K.is3 = r[7 * S];
          K.is5 = r[8 * S];
        }
      } else {
        const float4 a0 = sm.k[j], a1 = sm.k[kChPad + j];
        K.kq = dup2(a0.x);
        K.kc = dup2(a0.y);
        K.hn0 = dup2(a0.z);
        K.hn2 = dup2(a0.w);
        K.hn3 = dup2(a1.x);
        K.hn4 = dup2(a1.y);
        if (MODE == kNear) {
          K.ku = dup2(a1.z);
          K.is3 = dup2(a1.w);
          K.is5 = dup2(reinterpret_cast<const float*>(sm.k + 2 * kChPad)[j]);
        }
      }
    }
    if constexpr (PS == 2 && MODE != kFar) {
      float s0, s1;
      if (PAIR) {
        const float2 s = reinterpret_cast<const float2*>(sm.k)[j];
        s0 = s.x;
        s1 = s.y;
      } else {
        s0 = s1 = reinterpret_cast<const float*>(sm.k)[j];
      }
      K = make_sigk2(sigk_mixed(t.sg.x, s0), sigk_mixed(t.sg.y, s1));
    }
    const float2 dx = add2(t.x, nx), dy = add2(t.y, ny), dz = add2(t.z, nz);
    const float2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
    float2 S, T;
    pair_ST2<MODE, ST>(r2, K, S, T);
    float2 td = dup2(0.f);
    if (ST == 1) td = mul2(T, fma2(t.gx, dx, fma2(t.gy, dy, mul2(t.gz, dz))));
    if (ST == 2)
      td = mul2(T, fma2(t.ngz, kjz,
                        fma2(t.ngy, kjy, fma2(t.ngx, kjx, fma2(gjx, t.mx, fma2(gjy, t.my, mul2(gjz, t.mz)))))));
    if (MODE == kNear) {
      const int i0 = PAIR ? sm.id[2 * j] : sm.id[j], i1 = PAIR ? sm.id[2 * j + 1] : i0;
      if (i0 == t.id0) {
        S.x = 0.f;
        td.x = 0.f;
      }
      if (i1 == t.id1) {
        S.y = 0.f;
        td.y = 0.f;
      }
    }
    a.ax = fma2(S, gjx, a.ax);
    a.ay = fma2(S, gjy, a.ay);
    a.az = fma2(S, gjz, a.az);
    a.bx = fma2(S, kjx, a.bx);
    a.by = fma2(S, kjy, a.by);
    a.bz = fma2(S, kjz, a.bz);
    if (ST == 1) {
      a.cx = fma2(td, gjx, a.cx);
      a.cy = fma2(td, gjy, a.cy);
      a.cz = fma2(td, gjz, a.cz);
      a.dx = fma2(td, kjx, a.dx);
      a.dy = fma2(td, kjy, a.dy);
      a.dz = fma2(td, kjz, a.dz);
    }
    if (ST == 2) {
      a.cx = add2(a.cx, td);
      a.dx = fma2(td, nx, a.dx);
      a.dy = fma2(td, ny, a.dy);
      a.dz = fma2(td, nz, a.dz);
    }
  }
}

// What the pair kernel and the combine kernel write: the near field of every
// particle in sorted order.
struct P2POut {
  float* u;
  float* s;
};

// Near field of target i (sorted position) from its 12 sums.
template <int ST>
__device__ __forceinline__ void write_target(const P2POut& out, int i, float X, float Y, float Z, const float4& g,
                                             const float v[12]) {
  const size_t f = (size_t)3 * i;
  const float ax = v[0], ay = v[1], az = v[2];
  // u = A x X_i - B
  out.u[f] = kInv4Pi * ((ay * Z - az * Y) - v[3]);
  out.u[f + 1] = kInv4Pi * ((az * X - ax * Z) - v[4]);
  out.u[f + 2] = kInv4Pi * ((ax * Y - ay * X) - v[5]);
  if (ST == 1) {  // s = A x gamma_i - 3 (C x X_i - D)
    const float cx = v[6], cy = v[7], cz = v[8];
    out.s[f] = kInv4Pi * ((ay * g.z - az * g.y) + kM3 * ((cy * Z - cz * Y) - v[9]));
    out.s[f + 1] = kInv4Pi * ((az * g.x - ax * g.z) + kM3 * ((cz * X - cx * Z) - v[10]));
    out.s[f + 2] = kInv4Pi * ((ax * g.y - ay * g.x) + kM3 * ((cx * Y - cy * X) - v[11]));
  }
  if (ST == 2) {  // s = gamma_i x A - 3 (W X_i + D)
    out.s[f] = kInv4Pi * ((g.y * az - g.z * ay) + kM3 * (v[6] * X + v[9]));
    out.s[f + 1] = kInv4Pi * ((g.z * ax - g.x * az) + kM3 * (v[6] * Y + v[10]));
    out.s[f + 2] = kInv4Pi * ((g.x * ay - g.y * ax) + kM3 * (v[6] * Z + v[11]));
  }
}

constexpr int kTileMax = 64;  // targets of a work item
// One-warp CTAs asked for per SM (80 registers): Taylor-Green 128^3 took 19.08,
// 18.90, 19.04 and 18.56 ms at 16, 18, 20 and 24, a 100,003-blob ball 1.154,
// 1.125, 1.129 and 1.113 ms.
constexpr int kP2PPerSm = 24;

// One warp per work item: a tile of at most 64 targets of one leaf against a
// range [f0, f1) of the leaf's sources, numbered through the leaf's list
// (epre: the scanned source counts of the list entries).  The sources are
// loaded 64 at a time, one chunk ahead, and staged grouped by class.  Staging
// runs across entry boundaries, so small source leaves fill a chunk.  A tile
// of more than 32 targets is wide: two targets per lane, one source at a
// time.  A tile of at most 32 targets is narrow: one target per lane and two
// sources at a time, and with at most 16 (8) targets 2 (4) lane groups take
// every 2nd (4th) pair of sources, so the lanes stay filled.  The sums of a
// range that is not the whole list go to a partial slot, added in range order
// by k_p2p_combine.  One-warp CTAs keep the chunk bookkeeping warp-uniform
// (four warps per CTA on quarters of an item cost 5% at Taylor-Green 128^3).
// Bound by the FMA pipe: 78 cycles per 64 pairs and warp scheduler at
// Taylor-Green 128^3, where the pair loops alone (microbenchmark) take 66 (far)
// and 87 (mid).  Measured P2P, before (one warp per leaf, whole lists, source
// leaves staged one by one) and after: Taylor-Green 128^3 19.34 -> 18.7 ms,
// Plummer 1,000,000 22.3 -> 9.9 ms, Plummer 30,011 2.52 -> 0.45 ms, ball
// 100,003 1.74 -> 1.11 ms.
template <int PS, int ST>
__global__ void __launch_bounds__(32, kP2PPerSm)
    k_p2p(const int4* __restrict__ items, const int* __restrict__ islot, int tile, const int* __restrict__ leaves,
          const int2* __restrict__ off, const int2* __restrict__ list, const uint32_t* __restrict__ epre,
          const int* __restrict__ begin, const int* __restrict__ end, const float4* __restrict__ cf,
          const float4* __restrict__ A, const float4* __restrict__ B, const float4* __restrict__ sigk, float blen,
          float smax, float margin0, SigK K0, const int* __restrict__ cseg, const SegP2P* __restrict__ sp,
          P2POut out, float* __restrict__ partial, unsigned long long* __restrict__ ccount) {
  __shared__ Stage<PS> sm;
  const int lane = threadIdx.x;
  const int4 item = items[blockIdx.x];
  const int leaf = leaves[item.x];
  const int t0 = item.y, nt = min(tile, end[leaf] - t0);
  const int2 rg = off[item.x];
  const float4 lc = cf[leaf];
  if (cseg) {
    const SegP2P& q = sp[cseg[leaf]];
    K0 = q.k;
    blen = q.blen;
    smax = q.smax;
    margin0 = q.margin;
  }
  const bool wide = nt > 32;
  const int groups = nt > 16 ? 1 : (nt > 8 ? 2 : 4);
  const int width = 32 / groups, grp = lane / width, tl = lane & (width - 1);
  Tgt2 t;
  {
    float xs[2], ys[2], zs[2], gx[2], gy[2], gz[2], sg[2];
    bool valid[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int k = wide ? lane + 32 * q : tl;
      valid[q] = k < nt;
      const float4 xi = valid[q] ? A[t0 + k] : lc;
      const float4 gi = valid[q] ? B[t0 + k] : make_float4(0.f, 0.f, 0.f, 0.f);
      xs[q] = xi.x - lc.x;
      ys[q] = xi.y - lc.y;
      zs[q] = xi.z - lc.z;
      gx[q] = gi.x;
      gy[q] = gi.y;
      gz[q] = gi.z;
      sg[q] = valid[q] ? xi.w : smax;
      (q ? t.id1 : t.id0) = valid[q] ? t0 + k : -2;
    }
    const TileBox b = tile_box<2>(xs, ys, zs, valid);
    if (lane == 0) {
      sm.box = b;
      sm.centre = lc;
    }
    __syncwarp();  // every lane reads them when it classifies its sources
    t.x = make_float2(xs[0], xs[1]);
    t.y = make_float2(ys[0], ys[1]);
    t.z = make_float2(zs[0], zs[1]);
    t.gx = make_float2(gx[0], gx[1]);
    t.gy = make_float2(gy[0], gy[1]);
    t.gz = make_float2(gz[0], gz[1]);
    if (PS == 2) t.sg = make_float2(sg[0], sg[1]);
    if (ST == 2) {
      t.mx = make_float2(ys[0] * gz[0] - zs[0] * gy[0], ys[1] * gz[1] - zs[1] * gy[1]);
      t.my = make_float2(zs[0] * gx[0] - xs[0] * gz[0], zs[1] * gx[1] - xs[1] * gz[1]);
      t.mz = make_float2(xs[0] * gy[0] - ys[0] * gx[0], xs[1] * gy[1] - ys[1] * gx[1]);
      t.ngx = make_float2(-gx[0], -gx[1]);
      t.ngy = make_float2(-gy[0], -gy[1]);
      t.ngz = make_float2(-gz[0], -gz[1]);
    }
  }
  const SigK2 K = make_sigk2(K0, K0);
  AccR2 a;
  a.ax = a.ay = a.az = a.bx = a.by = a.bz = a.cx = a.cy = a.cz = a.dx = a.dy = a.dz = dup2(0.f);
  unsigned c_near = 0, c_mid = 0, c_far = 0;

  const uint32_t base = epre[rg.x], fe = (uint32_t)item.w;
  uint32_t f = (uint32_t)item.z;
  if (f < fe) {
    // the entry that holds source f: the last one whose prefix is <= f
    int e0 = rg.x, hi = rg.y;
    while (hi - e0 > 1) {
      const int st = (hi - e0 + 31) / 32, c = e0 + lane * st;
      const bool le = c < hi && epre[c] - base <= f;
      const int k = __popc(__ballot_sync(0xffffffffu, le)) - 1;
      e0 += k * st;
      hi = min(hi, e0 + st);
    }
    // window of 32 entries from e0: their prefixes, source ranges and images
    uint32_t wp, wend;
    int2 wl;
    auto load_window = [&](int e) {
      const int c = e + lane;
      wp = c < rg.y ? epre[c] - base : 0xffffffffu;
      wl = c < rg.y ? list[c] : make_int2(0, 0);
      wend = epre[min(e + 32, rg.y)] - base;
    };
    int cnt = 0;
    // the next chunk's loads: the sources from f on, within the window; then
    // the window of the chunk after it
    auto load_chunk = [&]() {
      cnt = (int)min(min(fe, wend) - f, (uint32_t)kCh);
      const bool one = __shfl_sync(0xffffffffu, wp, 1) >= f + (uint32_t)cnt;  // all in the first entry
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const uint32_t s = f + (uint32_t)(lane + 32 * q);
        int k = 0;
        if (!one) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            const uint32_t v = __shfl_sync(0xffffffffu, wp, k + o);
            if (v <= s) k += o;
          }
        }
        const uint32_t pk = __shfl_sync(0xffffffffu, wp, k);
        const int bk = __shfl_sync(0xffffffffu, wl.x, k);
        const int ik = __shfl_sync(0xffffffffu, wl.y, k);
        if (lane + 32 * q < cnt) {
          const int j = bk + (int)(s - pk), r = lane + 32 * q;
          copy16(&sm.raw[0][r], A + j);
          copy16(&sm.raw[1][r], B + j);
          if constexpr (PS == 1) {
#pragma unroll
            for (int i = 0; i < 3; ++i) copy16(&sm.raw[2 + i][r], sigk + 3 * (size_t)j + i);
          }
          sm.rid[r] = ik == kImageZero ? j : -1;
          sm.rimg[r] = ik;
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      f += (uint32_t)cnt;
      if (f < fe) {
        e0 += f >= wend ? 32 : __popc(__ballot_sync(0xffffffffu, wp <= f)) - 1;
        load_window(e0);
      }
    };
    load_window(e0);
    load_chunk();
    while (cnt > 0) {
      // stage the loaded chunk: X_j = (x_j - c) - shift, gamma_j, k_j =
      // gamma_j x X_j, grouped far, mid, near (in source order each);
      // sources of zero strength (the separate targets of
      // fmm_eval_targets) add nothing and are left out
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      const TileBox box = sm.box;
      const float4 c = sm.centre;
      float X[2], Y[2], Z[2];
      float4 ra[2], rb[2];
      int cls[2], slot[2], nf, nm;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int r = lane + 32 * q, img = r < cnt ? sm.rimg[r] : kImageZero;
        ra[q] = r < cnt ? sm.raw[0][r] : c;
        rb[q] = r < cnt ? sm.raw[1][r] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float shx = -(float)(img / 9 - 1) * blen, shy = -(float)((img / 3) % 3 - 1) * blen,
                    shz = -(float)(img % 3 - 1) * blen;
        X[q] = (ra[q].x - c.x) - shx;
        Y[q] = (ra[q].y - c.y) - shy;
        Z[q] = (ra[q].z - c.z) - shz;
        const bool live = rb[q].x != 0.f || rb[q].y != 0.f || rb[q].z != 0.f;
        cls[q] = live ? source_class(X[q], Y[q], Z[q], box, c.w, smax, margin0) : -1;
      }
      group_slots<2>(cls, lane, slot, nf, nm);
      const int used = __popc(__ballot_sync(0xffffffffu, cls[0] >= 0)) + __popc(__ballot_sync(0xffffffffu, cls[1] >= 0));
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int k = slot[q];
        if (k < 0) continue;
        const float4 g = rb[q];
        const float kx = g.y * Z[q] - g.z * Y[q], ky = g.z * X[q] - g.x * Z[q], kz = g.x * Y[q] - g.y * X[q];
        sm.id[k] = sm.rid[lane + 32 * q];
        float* sk = reinterpret_cast<float*>(sm.k);
        if (wide) {
          sm.v[k] = make_float4(-X[q], -Y[q], -Z[q], g.x);
          sm.v[kCh + k] = make_float4(g.y, g.z, kx, ky);
          reinterpret_cast<float*>(sm.v + 2 * kCh)[k] = kz;
          if constexpr (PS == 1) {
            sm.k[k] = sm.raw[2][lane + 32 * q];
            sm.k[kChPad + k] = sm.raw[3][lane + 32 * q];
            sk[8 * kChPad + k] = sm.raw[4][lane + 32 * q].x;
          }
        } else {
          float* r = reinterpret_cast<float*>(sm.v) + k;
          r[0] = -X[q];
          r[kChPad] = -Y[q];
          r[2 * kChPad] = -Z[q];
          r[3 * kChPad] = g.x;
          r[4 * kChPad] = g.y;
          r[5 * kChPad] = g.z;
          r[6 * kChPad] = kx;
          r[7 * kChPad] = ky;
          r[8 * kChPad] = kz;
          if constexpr (PS == 1) {
            const float4 k0 = sm.raw[2][lane + 32 * q], k1 = sm.raw[3][lane + 32 * q];
            sk[k] = k0.x;
            sk[kChPad + k] = k0.y;
            sk[2 * kChPad + k] = k0.z;
            sk[3 * kChPad + k] = k0.w;
            sk[4 * kChPad + k] = k1.x;
            sk[5 * kChPad + k] = k1.y;
            sk[6 * kChPad + k] = k1.z;
            sk[7 * kChPad + k] = k1.w;
            sk[8 * kChPad + k] = sm.raw[4][lane + 32 * q].x;
          }
        }
        if (PS == 2) sk[k] = ra[q].w;
      }
      int n0 = nf, n1 = nf + nm, n2 = used;
      if (!wide) {
        // whole units: a class's remainder runs in the next nearer form, the
        // last unit is filled with sources of zero strength away from the targets
        const int unit = 2 * groups;
        n0 &= ~(unit - 1);
        n1 &= ~(unit - 1);
        n2 = (used + unit - 1) & ~(unit - 1);
        if (lane < n2 - used) {
          float* r = reinterpret_cast<float*>(sm.v) + used + lane;
          r[0] = -(box.hx + 4.f * smax + 1.f);
          r[kChPad] = -box.hy;
          r[2 * kChPad] = -box.hz;
#pragma unroll
          for (int q = 3; q < 9; ++q) r[q * kChPad] = 0.f;
          sm.id[used + lane] = -1;
          float* sk = reinterpret_cast<float*>(sm.k) + used + lane;
          if (PS == 1) {
            sk[0] = -1.f;
#pragma unroll
            for (int q = 1; q < 9; ++q) sk[q * kChPad] = 0.f;
            sk[6 * kChPad] = 4.f;
          }
          if (PS == 2) sk[0] = smax;
        }
      }
      c_far += (unsigned)n0;
      c_mid += (unsigned)(n1 - n0);
      c_near += (unsigned)(used - n1);
      __syncwarp();
      const bool more = f < fe;
      if (more) load_chunk();
      else cnt = 0;
      if (wide) {
        if (n0 > 0) run_group<kFar, false, PS, ST>(sm, 0, n0, 1, t, K, a);
        if (n1 > n0) run_group<kMid, false, PS, ST>(sm, n0, n1, 1, t, K, a);
        if (n2 > n1) run_group<kNear, false, PS, ST>(sm, n1, n2, 1, t, K, a);
      } else {
        if (n0 > 0) run_group<kFar, true, PS, ST>(sm, grp, n0 / 2, groups, t, K, a);
        if (n1 > n0) run_group<kMid, true, PS, ST>(sm, n0 / 2 + grp, n1 / 2, groups, t, K, a);
        if (n2 > n1) run_group<kNear, true, PS, ST>(sm, n1 / 2 + grp, n2 / 2, groups, t, K, a);
      }
      __syncwarp();
    }
  }
  constexpr int NV = ST == 0 ? 6 : 12;
  const float2 va[12] = {a.ax, a.ay, a.az, a.bx, a.by, a.bz, a.cx, a.cy, a.cz, a.dx, a.dy, a.dz};
  const int ps = islot[blockIdx.x];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    float v[12];
    const int k = wide ? lane + 32 * q : tl;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      v[i] = q ? va[i].y : va[i].x;
      if (!wide) {  // the two chains and the lane groups hold sums of the same target
        v[i] += q ? va[i].x : va[i].y;
        for (int o = width; o < 32; o <<= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
      }
    }
    if (k >= nt || (!wide && (q || grp))) continue;
    if (ps >= 0) {
#pragma unroll
      for (int i = 0; i < NV; ++i) partial[((size_t)ps * 12 + i) * kTileMax + k] = v[i];
    } else {
      const float4 g = make_float4(q ? t.gx.y : t.gx.x, q ? t.gy.y : t.gy.x, q ? t.gz.y : t.gz.x, 0.f);
      write_target<ST>(out, t0 + k, q ? t.x.y : t.x.x, q ? t.y.y : t.y.x, q ? t.z.y : t.z.x, g, v);
    }
  }
  if (lane == 0) {
    const unsigned long long m = (unsigned long long)nt;
    if (c_near) atomicAdd(&ccount[0], m * c_near);
    if (c_mid) atomicAdd(&ccount[1], m * c_mid);
    if (c_far) atomicAdd(&ccount[2], m * c_far);
  }
}

// Targets of the tiles whose list was split: the partial sums of the ranges,
// added in range order.  One CTA per leaf; plan[leaf] = (first partial slot,
// ranges per tile).
template <int ST>
__global__ void __launch_bounds__(kTileMax) k_p2p_combine(const int2* __restrict__ plan, int tile,
                                                          const int* __restrict__ leaves,
                                                          const int* __restrict__ begin, const int* __restrict__ end,
                                                          const float4* __restrict__ cf,
                                                          const float4* __restrict__ A, const float4* __restrict__ B,
                                                          P2POut out, const float* __restrict__ partial) {
  constexpr int NV = ST == 0 ? 6 : 12;
  const int2 pl = plan[blockIdx.x];
  if (pl.y <= 1) return;
  const int leaf = leaves[blockIdx.x];
  const float4 lc = cf[leaf];
  int slot = pl.x;
  for (int t0 = begin[leaf]; t0 < end[leaf]; t0 += tile, slot += pl.y) {
    const int i = t0 + threadIdx.x;
    if ((int)threadIdx.x >= tile || i >= end[leaf]) continue;
    float v[12];
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = 0.f;
    for (int k = 0; k < pl.y; ++k) {
      const float* src = partial + (size_t)(slot + k) * 12 * kTileMax + threadIdx.x;
#pragma unroll
      for (int q = 0; q < NV; ++q) v[q] += src[q * kTileMax];
    }
    const float4 xi = A[i];
    write_target<ST>(out, i, xi.x - lc.x, xi.y - lc.y, xi.z - lc.z, B[i], v);
  }
}

// The outputs in the caller's order: near + far field, and the uniform velocity of
// the periodic dipole term (dip; in a batch the problem's).
__global__ void k_finish(const float* __restrict__ near_u, const float* __restrict__ near_s,
                         const float* __restrict__ far_u, const float* __restrict__ far_s,
                         const uint32_t* __restrict__ sidx, int64_t n, const double* __restrict__ dip,
                         const SegP2P* __restrict__ sp, const int* __restrict__ off, int nseg,
                         float* __restrict__ vel, float* __restrict__ dg) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float d[3] = {0.f, 0.f, 0.f};
  if (dip)
    for (int a = 0; a < 3; ++a) d[a] = (float)dip[a];
  if (sp) {
    int lo = 0, hi = nseg;  // the problem of sorted position i
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if ((int64_t)off[mid] <= i) lo = mid;
      else hi = mid;
    }
    for (int a = 0; a < 3; ++a) d[a] = sp[lo].dip[a];
  }
  const size_t o = 3 * (size_t)sidx[i], f = 3 * (size_t)i;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (vel) vel[o + a] = far_u[f + a] + near_u[f + a] + d[a];
    if (dg) dg[o + a] = far_s[f + a] + near_s[f + a];
  }
}

// ---- work items: per leaf, tiles x ranges, the longest ranges first (four
// length classes, leaf order within each), so that the last warps to start
// are short: in leaf order the batch of 32 problems waited for its longest
// lists (cut at 2048 sources: P2P 5.56 ms, 5.23 longest first).  One cooperative
// launch: the blocks own contiguous ranges of the leaves, take their class
// totals, meet at a bounded grid barrier and write (one CTA over all leaves took
// 153 us at Taylor-Green 128^3).  The host reads the counts with the barrier's
// abort word and launches the pair kernel only if that is 0.
constexpr int kItemClasses = 4, kItemThreads = 256, kItemBlocks = 128;

__global__ void __launch_bounds__(kItemThreads) k_p2p_items(const int* __restrict__ leaves, int nl,
                                                            const int* __restrict__ begin,
                                                            const int* __restrict__ end,
                                                            const int2* __restrict__ off,
                                                            const uint32_t* __restrict__ epre, int tile, uint32_t range,
                                                            int4* __restrict__ items, int* __restrict__ islot,
                                                            int2* __restrict__ plan, ItemState* st, uint32_t* blk,
                                                            long long spins, const int* __restrict__ sort_failed) {
  constexpr int NC = kItemClasses + 1;  // item classes, then partial slots
  __shared__ uint32_t ws[NC][kItemThreads / 32];
  __shared__ uint32_t carry[NC];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int G = (int)gridDim.x, b = (int)blockIdx.x;
  const int unsorted = *sort_failed;
  const int chunk = (nl + G - 1) / G, l0 = min(nl, b * chunk), l1 = min(nl, l0 + chunk);
  struct Leaf {
    uint32_t nit, nsp, F;
    int cls, tb, te;
  };
  auto read = [&](int i) {
    Leaf q{0u, 0u, 0u, kItemClasses - 1, 0, 0};
    if (i < l1) {
      const int leaf = leaves[i];
      const int2 rg = off[i];
      q.tb = begin[leaf];
      q.te = end[leaf];
      q.F = epre[rg.y] - epre[rg.x];
      q.nsp = q.F <= range ? 1u : (q.F + range - 1) / range;
      q.nit = q.nsp * (uint32_t)((q.te - q.tb + tile - 1) / tile);
      const uint32_t len = q.F / q.nsp;
      q.cls = len >= 8192u ? 0 : (len >= 4096u ? 1 : (len >= 2048u ? 2 : 3));
    }
    return q;
  };
  uint32_t sum[NC] = {0u, 0u, 0u, 0u, 0u};
  for (int i = l0 + threadIdx.x; i < l1; i += kItemThreads) {
    const Leaf q = read(i);
#pragma unroll
    for (int k = 0; k < NC; ++k) sum[k] += (k < kItemClasses ? k == q.cls : q.nsp > 1) ? q.nit : 0u;
  }
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    for (int o = 16; o > 0; o >>= 1) sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], o);
    if (lane == 0) ws[k][w] = sum[k];
  }
  __syncthreads();
  if (threadIdx.x < NC) {
    uint32_t x = 0;
    for (int i = 0; i < kItemThreads / 32; ++i) x += ws[threadIdx.x][i];
    blk[b * NC + threadIdx.x] = x;
  }
  if (!grid_barrier(&st->bar, (unsigned)G, spins)) return;
  if (unsorted) {  // the counts above mean nothing: give up as after an expired wait
    if (b == 0 && threadIdx.x == 0) st->bar.abort = 1u;
    return;
  }
  if (threadIdx.x < NC) {  // this block's first item of each class, and its first slot
    uint32_t pre = 0, all = 0;
    for (int j = 0; j < G; ++j) {
      const uint32_t x = ((volatile uint32_t*)blk)[j * NC + threadIdx.x];
      if (j < b) pre += x;
      all += x;
    }
    carry[threadIdx.x] = pre;
    ws[threadIdx.x][0] = all;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t acc = 0;
    for (int k = 0; k < kItemClasses; ++k) {
      carry[k] += acc;
      acc += ws[k][0];
    }
    if (b == 0) {
      st->items = acc;
      st->slots = ws[kItemClasses][0];
    }
  }
  __syncthreads();
  for (int c0 = l0; c0 < l1; c0 += kItemThreads) {
    const int i = c0 + threadIdx.x;
    const Leaf q = read(i);
    uint32_t at[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const uint32_t own = (k < kItemClasses ? k == q.cls : q.nsp > 1) ? q.nit : 0u;
      uint32_t inc = own;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) ws[k][w] = inc;
      at[k] = inc - own;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      at[k] += carry[k];
      for (int j = 0; j < w; ++j) at[k] += ws[k][j];
    }
    __syncthreads();
    if (threadIdx.x < NC)
      for (int j = 0; j < kItemThreads / 32; ++j) carry[threadIdx.x] += ws[threadIdx.x][j];
    if (i < l1) {
      uint32_t io = 0, slot = at[kItemClasses];
#pragma unroll
      for (int k = 0; k < kItemClasses; ++k)
        if (k == q.cls) io = at[k];
      plan[i] = make_int2((int)slot, (int)q.nsp);
      // equal ranges, so that no range is a short remainder
      const uint32_t len = (q.F + q.nsp - 1) / q.nsp;
      for (int t0 = q.tb; t0 < q.te; t0 += tile)
        for (uint32_t k = 0; k < q.nsp; ++k, ++io, ++slot) {
          items[io] = make_int4(i, t0, (int)min(q.F, k * len), (int)min(q.F, (k + 1) * len));
          islot[io] = q.nsp > 1 ? (int)slot : -1;
        }
    }
    __syncthreads();
  }
}

// The constants of every particle's own core width, in the order the pair
// kernel stages them: (kq, kc, hn0, hn2), (hn3, hn4, ku, is3), (is5).  Once per
// particle: computed in the pair kernel for every staged source, their FP64
// divisions were most of its time (ball of 60,000 own widths: P2P 4.74 ms,
// 1.09 with the table and the packed pairs).
__global__ void k_sigk(const float4* __restrict__ A, int64_t n, float4* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const SigK k = make_sigk(A[i].w);
  out[3 * i] = make_float4(k.kq, k.kc, k.hn0, k.hn2);
  out[3 * i + 1] = make_float4(k.hn3, k.hn4, k.ku, k.is3);
  out[3 * i + 2] = make_float4(k.is5, 0.f, 0.f, 0.f);
}

// All pairs of one array, free space, self pair skipped.  A cluster of eight
// CTAs of four warps takes 64 targets (two per lane, as the two halves of the
// FP32x2 operations); each of its 32 warps sums a contiguous 32nd of the
// sources, staged 32 at a time in its own shared memory, and the partial sums
// meet in distributed shared memory, added in source order.  The split keeps
// the chip filled at any n without a workspace: 20,000 blobs took 1.75 ms as
// 157 CTAs of 128 targets with scalar pairs, 0.67 ms now (100,000: 19.3 ->
// 14.1 ms; the error against FP64 2.5e-6 -> 5.2e-7).  Bound by the FMA
// pipe (38 operations per pair).  The targets keep absolute coordinates, so a
// pair takes gamma_j x d of the exact difference.
constexpr int kDirCluster = 8, kDirWarps = 4, kDirTile = 64;

struct DirStage {
  float4 a[32];  // -x, -y, -z, gamma_x
  float2 b[32];  // gamma_y, gamma_z
};
struct DirStageK {  // constants of the source's own core width
  float4 k0[32], k1[32];  // kq kc hn0 hn2, hn3 hn4 ku is3
  float is5[32];
};

template <bool PS>
__global__ void __cluster_dims__(kDirCluster, 1, 1) __launch_bounds__(32 * kDirWarps, 6)
    k_direct(int64_t n, const float* __restrict__ pos, const float* __restrict__ gam, const float* __restrict__ sig,
             SigK K0, float* __restrict__ vel, float* __restrict__ dg) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ DirStage st[kDirWarps];
  __shared__ DirStageK stk[PS ? kDirWarps : 1];
  __shared__ float red[kDirWarps][9][kDirTile];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = (int)cluster.block_rank();
  const int64_t i0 = (int64_t)(blockIdx.x / kDirCluster) * kDirTile;
  float2 tx, ty, tz, gx, gy, gz;
  {
    float v[2][6];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int64_t i = min(i0 + lane + 32 * q, n - 1);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        v[q][a] = pos[3 * i + a];
        v[q][3 + a] = gam[3 * i + a];
      }
    }
    tx = make_float2(v[0][0], v[1][0]);
    ty = make_float2(v[0][1], v[1][1]);
    tz = make_float2(v[0][2], v[1][2]);
    gx = make_float2(v[0][3], v[1][3]);
    gy = make_float2(v[0][4], v[1][4]);
    gz = make_float2(v[0][5], v[1][5]);
  }
  const SigK2 K1 = make_sigk2(K0, K0);
  float2 acc[9];  // sum S gamma_j x d, sum T' (gamma_i . d) gamma_j x d, sum S gamma_j
#pragma unroll
  for (int q = 0; q < 9; ++q) acc[q] = dup2(0.f);
  const int64_t per = (n + kDirCluster * kDirWarps - 1) / (kDirCluster * kDirWarps);
  const int64_t j0 = min(n, (int64_t)(rank * kDirWarps + warp) * per), j1 = min(n, j0 + per);
  float r[7];
  auto load = [&](int64_t c) {
    const int64_t j = c + lane;
    if (j < j1) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        r[a] = pos[3 * j + a];
        r[3 + a] = gam[3 * j + a];
      }
      r[6] = PS ? sig[j] : 0.f;
    }
  };
  load(j0);
  for (int64_t c = j0; c < j1; c += 32) {
    const int cnt = (int)min((int64_t)32, j1 - c);
    if (lane < cnt) {
      st[warp].a[lane] = make_float4(-r[0], -r[1], -r[2], r[3]);
      st[warp].b[lane] = make_float2(r[4], r[5]);
      if (PS) {
        const SigK k = make_sigk(r[6]);
        stk[PS ? warp : 0].k0[lane] = make_float4(k.kq, k.kc, k.hn0, k.hn2);
        stk[PS ? warp : 0].k1[lane] = make_float4(k.hn3, k.hn4, k.ku, k.is3);
        stk[PS ? warp : 0].is5[lane] = k.is5;
      }
    }
    __syncwarp();
    load(c + 32);
    // staged index of each target itself, if any
    const int64_t d = i0 + lane - c;
    const int self0 = d >= 0 && d < 32 ? (int)d : -1, self1 = d + 32 >= 0 && d < 0 ? (int)d + 32 : -1;
#pragma unroll 2
    for (int j = 0; j < cnt; ++j) {
      const float4 a = st[warp].a[j];
      const float2 b = st[warp].b[j];
      SigK2 K = K1;
      if (PS) {
        const float4 a0 = stk[PS ? warp : 0].k0[j], a1 = stk[PS ? warp : 0].k1[j];
        K.kq = dup2(a0.x);
        K.kc = dup2(a0.y);
        K.hn0 = dup2(a0.z);
        K.hn2 = dup2(a0.w);
        K.hn3 = dup2(a1.x);
        K.hn4 = dup2(a1.y);
        K.ku = dup2(a1.z);
        K.is3 = dup2(a1.w);
        K.is5 = dup2(stk[PS ? warp : 0].is5[j]);
      }
      const float2 dx = add2(tx, dup2(a.x)), dy = add2(ty, dup2(a.y)), dz = add2(tz, dup2(a.z));
      const float2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
      float2 S, T;
      pair_ST2<kNear, 1>(r2, K, S, T);
      if (j == self0) S.x = T.x = 0.f;
      if (j == self1) S.y = T.y = 0.f;
      const float2 jx = dup2(a.w), jy = dup2(b.x), jz = dup2(b.y);
      const float2 cx = fma2(jy, dz, mul2(dup2(-b.y), dy));
      const float2 cy = fma2(jz, dx, mul2(dup2(-a.w), dz));
      const float2 cz = fma2(jx, dy, mul2(dup2(-b.x), dx));
      const float2 td = mul2(T, fma2(gx, dx, fma2(gy, dy, mul2(gz, dz))));
      acc[0] = fma2(S, cx, acc[0]);
      acc[1] = fma2(S, cy, acc[1]);
      acc[2] = fma2(S, cz, acc[2]);
      acc[3] = fma2(td, cx, acc[3]);
      acc[4] = fma2(td, cy, acc[4]);
      acc[5] = fma2(td, cz, acc[5]);
      acc[6] = fma2(S, jx, acc[6]);
      acc[7] = fma2(S, jy, acc[7]);
      acc[8] = fma2(S, jz, acc[8]);
    }
    __syncwarp();
  }
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    red[warp][q][lane] = acc[q].x;
    red[warp][q][lane + 32] = acc[q].y;
  }
  cluster.sync();
  // each CTA finishes eight of the targets: the 32 partial sums of each value
  // in source order
  const int t = threadIdx.x / 9, q = threadIdx.x % 9;
  const int k = rank * (kDirTile / kDirCluster) + t;
  __shared__ float fin[kDirTile / kDirCluster][9];
  if (t < kDirTile / kDirCluster) {
    float v = 0.f;
    for (int b = 0; b < kDirCluster; ++b) {
      const float* src = cluster.map_shared_rank(&red[0][q][k], b);
      for (int w = 0; w < kDirWarps; ++w) v += src[w * 9 * kDirTile];
    }
    fin[t][q] = v;
  }
  cluster.sync();  // the other CTAs' sums have been read
  if (threadIdx.x < kDirTile / kDirCluster) {
    const int64_t i = i0 + rank * (kDirTile / kDirCluster) + threadIdx.x;
    const float* v = fin[threadIdx.x];
    if (i < n) {
      if (vel)
        for (int a = 0; a < 3; ++a) vel[3 * i + a] = kInv4Pi * v[a];
      if (dg) {
        const float x = gam[3 * i], y = gam[3 * i + 1], z = gam[3 * i + 2];
        dg[3 * i] = kInv4Pi * (kM3 * v[3] + (v[7] * z - v[8] * y));
        dg[3 * i + 1] = kInv4Pi * (kM3 * v[4] + (v[8] * x - v[6] * z));
        dg[3 * i + 2] = kInv4Pi * (kM3 * v[5] + (v[6] * y - v[7] * x));
      }
    }
  }
}

// Dipole term of the periodic lattice sum (Sec. 3.5): the cubic-order lattice
// sum exceeds the zero-mean (Ewald) field by (1/(3V)) sum_j (x_j - c0) x gamma_j;
// its negative is added to every velocity.  Two-stage fixed-order FP64 sum.
__global__ void k_dipole_partial(const float4* __restrict__ A, const float4* __restrict__ B, int64_t n,
                                 const double* __restrict__ box, double* __restrict__ part) {
  const double L = box[3];
  const double c0x = box[0] + 0.5 * L, c0y = box[1] + 0.5 * L, c0z = box[2] + 0.5 * L;
  double s[3] = {0.0, 0.0, 0.0};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float4 x = A[i], g = B[i];
    double X = (double)x.x - c0x, Y = (double)x.y - c0y, Z = (double)x.z - c0z;
    s[0] += Y * g.z - Z * g.y;
    s[1] += Z * g.x - X * g.z;
    s[2] += X * g.y - Y * g.x;
  }
  __shared__ double sh[3][256];
  for (int q = 0; q < 3; ++q) sh[q][threadIdx.x] = s[q];
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o)
      for (int q = 0; q < 3; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x < 3) part[blockIdx.x * 3 + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void k_dipole_final(const double* __restrict__ part, int nb, const double* __restrict__ box,
                               double* __restrict__ dip) {
  if (threadIdx.x >= 3) return;
  double s = 0.0;
  for (int b = 0; b < nb; ++b) s += part[b * 3 + threadIdx.x];
  const double L = box[3];
  dip[threadIdx.x] = -s / (3.0 * L * L * L);
}

// The same correction for each problem of a batch (one CTA per problem over
// its sorted particle range), stored with the problem's near-field constants.
__global__ void __launch_bounds__(256) k_dipole_seg(const float4* __restrict__ A, const float4* __restrict__ B,
                                                    const int* __restrict__ off, const double* __restrict__ box,
                                                    SegP2P* __restrict__ sp) {
  const int sg = blockIdx.x;
  const double* bx = box + 4 * sg;
  const double L = bx[3];
  const double c0x = bx[0] + 0.5 * L, c0y = bx[1] + 0.5 * L, c0z = bx[2] + 0.5 * L;
  double s[3] = {0.0, 0.0, 0.0};
  for (int i = off[sg] + threadIdx.x; i < off[sg + 1]; i += blockDim.x) {
    float4 x = A[i], g = B[i];
    double X = (double)x.x - c0x, Y = (double)x.y - c0y, Z = (double)x.z - c0z;
    s[0] += Y * g.z - Z * g.y;
    s[1] += Z * g.x - X * g.z;
    s[2] += X * g.y - Y * g.x;
  }
  __shared__ double sh[3][256];
  for (int q = 0; q < 3; ++q) sh[q][threadIdx.x] = s[q];
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o)
      for (int q = 0; q < 3; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x < 3) sp[sg].dip[threadIdx.x] = (float)(-sh[threadIdx.x][0] / (3.0 * L * L * L));
}

}  // namespace

// The uniform dipole velocity of a periodic one-problem evaluation (the
// zero-mean convention, subtracted in the P2P epilogue).  It needs only the
// sorted particles, so it runs on the upward pass's stream beside the
// traversal, into its own partial-sum buffer.
int dipole_pass(fmm_plan p, int64_t n, cudaStream_t s) {
  if (!p->prm.periodic || n == 0) return FMM_OK;
  if (p->batched) {  // after the problem tables, which hold the result
    ++g_launches;
    k_dipole_seg<<<p->nseg, 256, 0, s>>>(p->sortA.as<float4>(), p->sortB.as<float4>(), p->seg_off.as<int>(),
                                         p->seg_box.as<double>(), p->seg_p2p.as<SegP2P>());
    FMM_CUDA_TRY(cudaGetLastError());
    return FMM_OK;
  }
  const int parts = 256;
  double* scal = p->scal.as<double>();
  FMM_TRY(p->dip_part.ensure((size_t)parts * 3 * sizeof(double)));
  ++g_launches;
  k_dipole_partial<<<parts, 256, 0, s>>>(p->sortA.as<float4>(), p->sortB.as<float4>(), n, scal,
                                         p->dip_part.as<double>());
  ++g_launches;
  k_dipole_final<<<1, 32, 0, s>>>(p->dip_part.as<double>(), parts, scal, scal + kScalDipole);
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

// Work items of the pair kernel (after the list is grouped by leaf): one warp
// per (tile of a leaf, range of its sources).  Ranges bound the longest warp:
// the big outer leaves of a clustered cloud meet thousands of small ones, and
// one warp per leaf left the chip waiting for them (Plummer, 30,011 blobs:
// P2P 2.5 ms; 0.45 ms with ranges), and with it how long the far field's
// kernels wait for room.  One-problem plans take the range that gives kItemTarget
// items, at least 128 sources (two chunks);
// the partial slots are then bounded by twice that many items (3 KB each).  A
// batch keeps whole lists: a problem's sums may not depend on the rest of the
// batch, its many problems fill the chip, and the long lists start first.
// Ranges of 2048 sources for lists above 8192 give 2 to 5% (batch of 32 problems,
// 477,044 blobs: 7.66 ms instead of 7.84) but move single values by up to 1.6e-3
// of the largest component from those of one running sum (whole lists 5.6e-4 at
// most over 18 inputs).  Against the FP64 pair sum both err the same: rel-L2 u
// 3.24e-5 and 3.25e-5, s 9.66e-5 both, largest s 2.3e-4 both.
constexpr int64_t kItemTarget = 8 * 32 * 152;  // items aimed at (half as many: ball 100,003 2.15 instead of 2.09 ms in all)
constexpr uint32_t kItemSrcMin = 128;

int p2p_tile(fmm_plan p) { return p->prm.p2p_tpl == 1 ? 32 : kTileMax; }

int p2p_build_items(fmm_plan p, int64_t n, int64_t tile_sources, cudaStream_t s) {
  const int tile = p2p_tile(p);
  uint32_t range = 0xffffffffu;
  if (!p->batched) {
    const int64_t q = (tile_sources / kItemTarget + kCh - 1) / kCh * kCh;
    range = (uint32_t)std::min<int64_t>(0xffffffffll - kCh, std::max<int64_t>(kItemSrcMin, q));
  }
  // at most one partly filled range and one partly filled tile per leaf
  const int64_t tiles = p->nleaves + n / tile + 1;
  const int64_t items = tiles + tile_sources / range + 1;
  FMM_TRY(p->p2p_items.ensure((size_t)items * sizeof(int4)));
  FMM_TRY(p->p2p_islot.ensure((size_t)items * sizeof(int)));
  FMM_TRY(p->p2p_plan.ensure((size_t)(p->nleaves + 1) * sizeof(int2)));
  FMM_TRY(p->p2p_bar.ensure(sizeof(ItemState) + (size_t)kItemBlocks * (kItemClasses + 1) * sizeof(uint32_t)));
  ItemState* st = p->p2p_bar.as<ItemState>();
  uint32_t* blk = reinterpret_cast<uint32_t*>(st + 1);
  FMM_CUDA_TRY(cudaMemsetAsync(st, 0, sizeof(ItemState), s));
  const int* leaves = p->leaves.as<int>();
  const int* cb = p->c_begin.as<int>();
  const int* ce = p->c_end.as<int>();
  const int2* off = p->p2p_off.as<int2>();
  const uint32_t* pre = p->p2p_pre.as<uint32_t>();
  int4* it = p->p2p_items.as<int4>();
  int* is = p->p2p_islot.as<int>();
  int2* plan = p->p2p_plan.as<int2>();
  int nl = (int)p->nleaves, tl = tile;
  const unsigned G = (unsigned)std::min<int64_t>(kItemBlocks, (nl + kItemThreads - 1) / kItemThreads);
  long long spins = p->wait_limit[FMM_WAIT_ITEMS];
  void* args[] = {&leaves, &nl, &cb, &ce, &off, &pre, &tl, &range, &it, &is, &plan, &st, &blk, &spins, &p->p_sort.failed};
  ++g_launches;
  FMM_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)k_p2p_items, dim3(G), dim3(kItemThreads), args, 0, s));
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

// The staging memory needs the largest shared-memory carveout: 5.4 KB a warp with
// one core width, 5.6 with the mixed rule (24 warps fit an SM), 10.9 with a width
// per particle (19 do).
static_assert(sizeof(Stage<0>) == 5504 && sizeof(Stage<2>) == 5776 && sizeof(Stage<1>) == 11152, "as stated");
static int p2p_attributes() {
  static std::atomic<bool> done[kMaxDevices];
  return once_per_device(done, [] {
    const void* k[9] = {(const void*)k_p2p<0, 0>, (const void*)k_p2p<0, 1>, (const void*)k_p2p<0, 2>,
                        (const void*)k_p2p<1, 0>, (const void*)k_p2p<1, 1>, (const void*)k_p2p<1, 2>,
                        (const void*)k_p2p<2, 0>, (const void*)k_p2p<2, 1>, (const void*)k_p2p<2, 2>};
    for (const void* f : k)
      if (cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 100) != cudaSuccess) return false;
    return true;
  });
}

// The near field of every particle, in sorted order (near_u, near_s).
int p2p_near(fmm_plan p, int64_t n, float sig_u, int ps, double smax, bool stretching, cudaStream_t s) {
  double* scal = p->scal.as<double>();
  const int* cseg = p->batched ? p->c_seg.as<int>() : nullptr;
  SegP2P* sp = p->batched ? p->seg_p2p.as<SegP2P>() : nullptr;
  // both whatever the outputs: fmm_eval_strengths may ask for others and must not allocate
  FMM_TRY(p->near_u.ensure((size_t)n * 3 * sizeof(float)));
  FMM_TRY(p->near_s.ensure((size_t)n * 3 * sizeof(float)));
  const P2POut out{p->near_u.as<float>(), p->near_s.as<float>()};
  const float blen = p->prm.periodic ? (float)p->prm.box_len : 0.f;
  const SigK K0 = make_sigk(ps ? 1.f : sig_u);
  const int mode = ps ? (p->prm.sigma_rule == FMM_SIGMA_MIXED ? 2 : 1) : 0;
  const int tile = p2p_tile(p);
  const float4* A = p->sortA.as<float4>();
  const float4* B = p->sortB.as<float4>();
  const float4* sigk = nullptr;
  if (mode == 1) {
    FMM_TRY(p->p2p_sigk.ensure((size_t)n * 3 * sizeof(float4)));
    ++g_launches;
    k_sigk<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(A, n, p->p2p_sigk.as<float4>());
    sigk = p->p2p_sigk.as<float4>();
  }
  FMM_TRY(p->p2p_partial.ensure((size_t)std::max<int64_t>(p->n_p2p_slots, 1) * 12 * kTileMax * sizeof(float)));
  float* partial = p->p2p_partial.as<float>();
  unsigned long long* cnt = reinterpret_cast<unsigned long long*>(scal + kScalCount + 4);
  FMM_CUDA_TRY(cudaMemsetAsync(cnt, 0, 3 * sizeof(unsigned long long), s));
  const int* leaves = p->leaves.as<int>();
  const int* cb = p->c_begin.as<int>();
  const int* ce = p->c_end.as<int>();
  const float4* cf = p->c_cf.as<float4>();
  const unsigned items = (unsigned)p->n_p2p_items;
  const float smaxf = (float)smax, margin0 = (float)p->cf_margin;
  FMM_TRY(p2p_attributes());
#define FMM_P2P(PS_, ST_)                                                                                             \
  k_p2p<PS_, ST_><<<items, 32, 0, s>>>(p->p2p_items.as<int4>(), p->p2p_islot.as<int>(), tile, leaves,     \
                                                   p->p2p_off.as<int2>(), p->p2p_sorted.as<int2>(),                   \
                                                   p->p2p_pre.as<uint32_t>(), cb, ce, cf, A, B, sigk, blen, smaxf,    \
                                                   margin0, K0, cseg, sp, out, partial, cnt)
#define FMM_P2P_ST(ST_)                \
  do {                                 \
    if (mode == 0) FMM_P2P(0, ST_);    \
    else if (mode == 1) FMM_P2P(1, ST_); \
    else FMM_P2P(2, ST_);              \
    if (p->n_p2p_slots > 0) {          \
      ++g_launches;                    \
      k_p2p_combine<ST_><<<(unsigned)p->nleaves, kTileMax, 0, s>>>(p->p2p_plan.as<int2>(), tile, leaves, cb, ce, cf, \
                                                                   A, B, out, partial);                              \
    }                                  \
  } while (0)
  ++g_launches;
  // without a stretching output the kernels skip T and the stretching sums
  if (!stretching) FMM_P2P_ST(0);
  else if (p->prm.outputs & FMM_OUT_STRETCHING_TRANSPOSE) FMM_P2P_ST(2);
  else FMM_P2P_ST(1);
#undef FMM_P2P_ST
#undef FMM_P2P
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

// Outputs from the near and the far field.
int p2p_finish(fmm_plan p, int64_t n, float* vel, float* dg, cudaStream_t s) {
  if (!vel && !dg) return FMM_OK;
  const bool seg = p->prm.periodic && p->batched;
  SegP2P* sp = seg ? p->seg_p2p.as<SegP2P>() : nullptr;
  const double* dip = p->prm.periodic && !p->batched ? p->scal.as<double>() + kScalDipole : nullptr;
  ++g_launches;
  k_finish<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p->near_u.as<float>(), p->near_s.as<float>(),
                                                       p->far_u.as<float>(), p->far_s.as<float>(), p->sidx, n, dip, sp,
                                                       seg ? p->seg_off.as<int>() : nullptr, p->nseg, vel, dg);
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

int p2p_direct_all(int64_t n, const float* pos, const float* gam, const float* sig, float sig_u, float* vel, float* dg,
                   cudaStream_t s) {
  const int64_t tiles = (n + kDirTile - 1) / kDirTile;
  if (tiles * kDirCluster > 0x7fffffffll) return FMM_E_INVAL;
  const unsigned g = (unsigned)(tiles * kDirCluster);
  const SigK K0 = make_sigk(sig ? 1.f : sig_u);
  ++g_launches;
  if (sig) k_direct<true><<<g, 32 * kDirWarps, 0, s>>>(n, pos, gam, sig, K0, vel, dg);
  else k_direct<false><<<g, 32 * kDirWarps, 0, s>>>(n, pos, gam, sig, K0, vel, dg);
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

}  // namespace fmm
