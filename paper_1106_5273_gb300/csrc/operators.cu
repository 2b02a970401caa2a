// Translation operators as real matrices on the real-packed coefficients.
//
// Sec. 3.1: M2M, M2L, L2L of the spherical-harmonic Laplace expansions
// (formulas in harmonics.cuh).  Octree children sit at beta = (+-1/2)^3 in
// child units with scale ratio 1/2, so M2M and L2L reduce to 8 fixed matrices
// per p, built here once in FP64 on the host.  Each distinct M2L translation
// (level difference, offset: m2l_key_encode) becomes one P x P matrix built in
// FP64 on the device, once per plan (the cache below).  The periodic far field
// (Sec. 3.5) is one FP64 P x P operator on the root multipole: images-1
// rings of 702 super-cells, each ring the M2L sum from offsets
// {-4..4}^3 \ {-1..1}^3, the next super-cell the M2M sum of 27 copies.
#include <complex>
#include <cstring>

#include "fmm_internal.cuh"
#include <cuda_bf16.h>

namespace fmm {

namespace {

using Mat = std::vector<double>;

// Y_n^m (m >= 0) += c * X_j^k  (conj_in: c * conj(X_j^k)), X_j^{-k} = (-1)^k conj(X_j^k).
void add_term(Mat& A, int P, int n, int m, int j, int k, cd c, bool conj_in) {
  int ak = k < 0 ? -k : k;
  double sgn = (k < 0 && (ak & 1)) ? -1.0 : 1.0;
  bool conj_total = (k < 0) != conj_in;
  double br = conj_total ? -1.0 : 1.0;
  cd ca = {c.re * sgn, c.im * sgn};
  cd cb = {-c.im * sgn * br, c.re * sgn * br};
  int row_re = ridx(n, m, 0);
  int col_a = ridx(j, ak, 0);
  A[(size_t)row_re * P + col_a] += ca.re;
  if (m > 0) A[(size_t)ridx(n, m, 1) * P + col_a] += ca.im;
  if (ak > 0) {
    int col_b = ridx(j, ak, 1);
    A[(size_t)row_re * P + col_b] += cb.re;
    if (m > 0) A[(size_t)ridx(n, m, 1) * P + col_b] += cb.im;
  }
}

Mat m2m_matrix(int p, const double beta[3], double ratio) {
  const int P = p * p;
  Mat A((size_t)P * P, 0.0);
  std::vector<cd> R(kPMax * (kPMax + 1) / 2);
  regular_table_d(beta[0], beta[1], beta[2], p, R.data());
  for (int n = 0; n < p; ++n)
    for (int m = 0; m <= n; ++m)
      for (int k = 0; k <= n; ++k)
        for (int l = -k; l <= k; ++l) {
          if (std::abs(m - l) > n - k) continue;
          double w = pow(ratio, n) * nu_d(n, m) / (nu_d(k, l) * nu_d(n - k, m - l));
          cd c = cscale(cconj(harm_get(R.data(), k, l)), w);
          add_term(A, P, n, m, n - k, m - l, c, false);
        }
  return A;
}

Mat l2l_matrix(int p, const double beta[3], double ratio) {
  const int P = p * p;
  Mat A((size_t)P * P, 0.0);
  std::vector<cd> R(kPMax * (kPMax + 1) / 2);
  regular_table_d(beta[0], beta[1], beta[2], p, R.data());
  for (int n = 0; n < p; ++n)
    for (int m = 0; m <= n; ++m)
      for (int k = 0; k < p - n; ++k)
        for (int l = -k; l <= k; ++l) {
          if (std::abs(m + l) > n + k) continue;
          double w = pow(ratio, n + k + 1) * nu_d(n + k, m + l) / (nu_d(n, m) * nu_d(k, l));
          cd c = cscale(harm_get(R.data(), k, l), w);
          add_term(A, P, n, m, n + k, m + l, c, false);
        }
  return A;
}

Mat m2l_matrix(int p, const double tau[3], double ratio) {
  const int P = p * p;
  Mat A((size_t)P * P, 0.0);
  const int D = 2 * p - 1;
  std::vector<cd> I(D * (D + 1) / 2);
  irregular_table_d(tau[0], tau[1], tau[2], D, I.data());
  for (int n = 0; n < p; ++n)
    for (int m = 0; m <= n; ++m)
      for (int j = 0; j < p; ++j)
        for (int k = -j; k <= j; ++k) {
          double w = ((n & 1) ? -1.0 : 1.0) * pow(ratio, j) / (nu_d(n, m) * nu_d(j, k));
          cd c = cscale(cconj(harm_get(I.data(), j + n, k + m)), w);
          add_term(A, P, n, m, j, k, c, true);
        }
  return A;
}

Mat matmul(const Mat& A, const Mat& B, int P) {
  Mat C((size_t)P * P, 0.0);
  for (int i = 0; i < P; ++i)
    for (int k = 0; k < P; ++k) {
      double a = A[(size_t)i * P + k];
      if (a == 0.0) continue;
      for (int j = 0; j < P; ++j) C[(size_t)i * P + j] += a * B[(size_t)k * P + j];
    }
  return C;
}

// Lattice operator: L~_root += A_lat M~_root (root side = box length).
Mat lattice_matrix(int p, int images) {
  const int P = p * p;
  Mat A((size_t)P * P, 0.0);
  Mat S((size_t)P * P, 0.0);  // M2M of level-(lev-1) super-cell from the root
  for (int i = 0; i < P; ++i) S[(size_t)i * P + i] = 1.0;
  // one-level super-cell M2M: 27 copies at offsets o (child units), ratio 1/3
  Mat S3((size_t)P * P, 0.0);
  for (int ox = -1; ox <= 1; ++ox)
    for (int oy = -1; oy <= 1; ++oy)
      for (int oz = -1; oz <= 1; ++oz) {
        double b[3] = {(double)ox, (double)oy, (double)oz};
        Mat T = m2m_matrix(p, b, 1.0 / 3.0);
        for (size_t q = 0; q < T.size(); ++q) S3[q] += T[q];
      }
  double scale = 1.0;  // super-cell side / root side
  for (int lev = 1; lev < images; ++lev) {
    Mat ring((size_t)P * P, 0.0);
    for (int ox = -4; ox <= 4; ++ox)
      for (int oy = -4; oy <= 4; ++oy)
        for (int oz = -4; oz <= 4; ++oz) {
          if (std::max(std::abs(ox), std::max(std::abs(oy), std::abs(oz))) <= 1) continue;
          double tau[3] = {-ox * scale, -oy * scale, -oz * scale};
          Mat T = m2l_matrix(p, tau, scale);
          for (size_t q = 0; q < T.size(); ++q) ring[q] += T[q];
        }
    Mat contrib = matmul(ring, S, P);
    for (size_t q = 0; q < A.size(); ++q) A[q] += contrib[q];
    S = matmul(S3, S, P);
    scale *= 3.0;
  }
  return A;
}

// ---- device: M2L operator per translation key

// Round an FP32 value to TF32 (10 stored mantissa bits, to nearest, ties to
// even) in its 32-bit container; the low 13 bits end up zero.
__device__ __forceinline__ float round_tf32(float x) {
  uint32_t u = __float_as_uint(x);
  if ((u & 0x7f800000u) == 0x7f800000u) return x;  // inf / nan
  u += 0x0FFFu + ((u >> 13) & 1u);
  return __uint_as_float(u & 0xFFFFE000u);
}

// v or -v, by its sign bit.
__device__ __forceinline__ double flip(double v, bool neg) {
  return __longlong_as_double(__double_as_longlong(v) ^ ((long long)neg << 63));
}

// v rounded once to BF16 (to nearest, ties to even): its bits, and in r the
// rounded value.  On the upper word of the pattern, since an FP64 conversion costs
// what 64 FP32 operations do; bad is set where the result is neither zero nor
// normal in BF16 (round_bf16_any serves those).
__device__ __forceinline__ uint32_t round_bf16(double v, double& r, bool& bad) {
  const uint32_t hi = (uint32_t)__double2hiint(v);
  const uint32_t up = ((hi >> 13) | min((uint32_t)__double2loint(v), 1u)) & 1u;  // odd, or beyond the half
  const uint32_t h = (hi + 0xfffu + up) & 0xffffe000u;                           // 7 of 52 mantissa bits stay
  const uint32_t x = (h & 0x7fffffffu) >> 13;                                    // exponent and mantissa
  constexpr uint32_t bias = (1023 - 127) << 7;
  bad = bad || (x != 0u && x - (bias + 128u) >= (254u << 7));
  r = __hiloint2double((int)h, 0);
  return (h >> 16 & 0x8000u) | (uint32_t)max((int)(x - bias), 0);
}
__device__ __noinline__ uint32_t round_bf16_any(double v) { return (uint32_t)__bfloat16_as_ushort(__double2bfloat16(v)); }

// M2L operators of new translations, one CTA each, in FP64; both BF16 halves come
// from the FP64 entry.
// kind 0: BF16 tiles [key][hi/lo][nkc K chunks of 64][rows][64];
// kind 1: TF32 tiles [key][hi/lo][nkc K chunks of 32][rows][32]; both 128-byte
// rows with 16-byte groups in the 128-byte swizzle order (group j at j ^ (row & 7)),
// padding rows and columns zero; nkc = 0: FP32 [key][P][P].
// FP64 runs at a 64th of the FP32 rate, so a BF16 entry takes two additions and two
// multiplications: the factors 1 / nu come from a table, the
// irregular harmonics are built by one thread per order m, and a thread writes
// 16 bytes of a row at a time.  The first evaluation of Plummer 1,000,000 (49,141
// operators, p = 12) spent 57.4 ms here with a division and the conversions per
// entry and one thread for the harmonics, now 12.1 (11.7 with the entry rounded to
// FP32 before the split).
__global__ void __launch_bounds__(256) k_build_m2l(const uint64_t* __restrict__ keys, const int* __restrict__ slots,
                                                   int nkeys, int p, const double* __restrict__ inu,
                                                   float* __restrict__ T32, uint8_t* __restrict__ Tb, int nkc,
                                                   int kind) {
  __shared__ cd I[(2 * kPMax - 1) * (2 * kPMax) / 2];
  __shared__ double ar[kNCoefMax], bc[kNCoefMax];  // (-1)^n / nu of a row, ratio^j / nu of a column
  __shared__ int nmp[kNCoefMax];                   // real index -> (n, m, part) packed
  const int kid = blockIdx.x;
  if (kid >= nkeys) return;
  const int key_id = slots[kid];  // cache slot written by this block
  const int P = p * p, D = 2 * p - 1;
  int delta;
  double tau[3];
  m2l_key_decode(keys[kid], &delta, tau);
  if ((int)threadIdx.x < D) {
    // thread = order m: the diagonal I_m^m, then up the column (the recurrences
    // and their order of irregular_table_d)
    const int m = threadIdx.x;
    const double x = tau[0], y = tau[1], z = tau[2], r2 = x * x + y * y + z * z, inv_r2 = 1.0 / r2;
    cd d = {1.0 / sqrt(r2), 0.0};
    for (int q = 1; q <= m; ++q) d = cscale(cmul(d, cd{x, y}), (2.0 * q - 1.0) * inv_r2);
    I[cidx(m, m)] = d;
    cd b1 = {0.0, 0.0}, b0 = d;  // I_{n-2}^m, I_{n-1}^m
    for (int n = m + 1; n < D; ++n) {
      cd a = cscale(b0, (2.0 * n - 1.0) * z);
      if (n - 2 >= m) {
        const cd b = cscale(b1, (double)((n - 1) * (n - 1) - m * m));
        a.re -= b.re;
        a.im -= b.im;
      }
      b1 = b0;
      b0 = cscale(a, inv_r2);
      I[cidx(n, m)] = b0;
    }
  }
  for (int r = threadIdx.x; r < P; r += blockDim.x) {
    int n = (int)sqrtf((float)r);
    while (n * n > r) --n;
    while ((n + 1) * (n + 1) <= r) ++n;
    int o = r - n * n;
    int m = (o + 1) / 2, part = (o == 0) ? 0 : ((o - 1) & 1);
    nmp[r] = (n << 16) | (m << 8) | part;
    const double v = inu[r];
    ar[r] = (n & 1) ? -v : v;
    bc[r] = ldexp(v, delta * n);
  }
  __syncthreads();
  // entry (r, c): output (n, m, po), input (j, k, pi); A = conj I_{j+n}^{k+m},
  // B = (-1)^k conj I_{j+n}^{m-k} (0 for k = 0); the real parts of
  // s [a (A + B) + i b (B - A)]
  auto entry = [&](int r, int c) -> double {
    if (r >= P || c >= P) return 0.0;
    const int a = nmp[r], b = nmp[c];
    const int n = a >> 16, m = (a >> 8) & 0xff, po = a & 1;
    const int j = b >> 16, k = (b >> 8) & 0xff, pi = b & 1;
    const bool im = po != pi;  // the imaginary parts enter
    const cd* Ia = &I[cidx(j + n, k + m)];
    const double va = flip(im ? Ia->im : Ia->re, im);
    const int q = m - k;
    const cd* Ib = &I[cidx(j + n, q < 0 ? -q : q)];
    // (-1)^k, and for q < 0 I^{q} = (-1)^q conj I^{-q}
    const bool neg = ((k & 1) != 0) != (q < 0 && (((q & 1) != 0) != im));
    const double vb = k > 0 ? flip(im ? Ib->im : Ib->re, neg != im) : 0.0;
    // one form for all parts (signs flipped, no divergence): pi = 0 takes va + vb,
    // pi = 1 va - vb (po = 0) or vb - va
    return ar[r] * bc[c] * (flip(va, pi && po) + flip(vb, pi && !po));
  };
  if (!nkc) {  // the SIMT path's FP32 copy
    for (int e = threadIdx.x; e < P * P; e += blockDim.x) T32[(size_t)key_id * P * P + e] = (float)entry(e / P, e % P);
    return;
  }
  const int rows = m2l_cols(P);  // output rows of the operator tiles
  const size_t chunk_bytes = (size_t)rows * 128;
  uint8_t* T = Tb + (size_t)key_id * 2 * nkc * chunk_bytes;
  for (int u = threadIdx.x; u < rows * nkc * 8; u += blockDim.x) {
    const int r = u / (nkc * 8), kc = (u >> 3) % nkc, g = u & 7;
    uint32_t hi[4], lo[4];
    if (kind == 0) {
      const int c = kc * 64 + g * 8;
      bool bad = false;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        hi[q] = lo[q] = 0u;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const double v = entry(r, c + 2 * q + e);
          double h, l;
          hi[q] |= round_bf16(v, h, bad) << (16 * e);
          lo[q] |= round_bf16(v - h, l, bad) << (16 * e);
        }
      }
      if (bad) {
#pragma unroll 1
        for (int q = 0; q < 8; ++q) {
          const double v = entry(r, c + q);
          const uint32_t h = round_bf16_any(v), sh = 16 * (q & 1);
          const uint32_t l = round_bf16_any(v - (double)__uint_as_float(h << 16));
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i == q >> 1) {
              hi[i] = (hi[i] & ~(0xffffu << sh)) | h << sh;
              lo[i] = (lo[i] & ~(0xffffu << sh)) | l << sh;
            }
        }
      }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double v = entry(r, kc * 32 + g * 4 + q);
        const float h = round_tf32((float)v);
        hi[q] = __float_as_uint(h);
        lo[q] = __float_as_uint(round_tf32((float)(v - (double)h)));
      }
    }
    uint8_t* dst = T + (size_t)kc * chunk_bytes + (size_t)r * 128 + (size_t)((g ^ (r & 7)) << 4);
    *reinterpret_cast<uint4*>(dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dst + (size_t)nkc * chunk_bytes) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

// One CTA per root cell (one per problem; the normalised operator does not
// depend on the cube size): L[root][c][r] += sum_k A[r][k] M[root][c][k]
__global__ void k_apply_lattice(const double* __restrict__ A, int P, float* __restrict__ L, const float* __restrict__ M) {
  const size_t root = (size_t)blockIdx.x * 3 * P;
  for (int e = threadIdx.x; e < 3 * P; e += blockDim.x) {
    int c = e / P, r = e % P;
    double acc = 0.0;
    for (int k = 0; k < P; ++k) acc += A[(size_t)r * P + k] * (double)M[root + c * P + k];
    L[root + c * P + r] += (float)acc;
  }
}

}  // namespace

int build_constant_operators(fmm_plan p) {
  const int pp = p->prm.p, P = pp * pp;
  std::vector<float> m2mT((size_t)8 * P * P), l2lT((size_t)8 * P * P);
  for (int oct = 0; oct < 8; ++oct) {
    double beta[3] = {(oct & 4) ? 0.5 : -0.5, (oct & 2) ? 0.5 : -0.5, (oct & 1) ? 0.5 : -0.5};
    Mat A = m2m_matrix(pp, beta, 0.5);
    Mat B = l2l_matrix(pp, beta, 0.5);
    for (int r = 0; r < P; ++r)
      for (int k = 0; k < P; ++k) {
        m2mT[(size_t)oct * P * P + (size_t)k * P + r] = (float)A[(size_t)r * P + k];
        l2lT[(size_t)oct * P * P + (size_t)k * P + r] = (float)B[(size_t)r * P + k];
      }
  }
  FMM_TRY(p->m2m_T.ensure(m2mT.size() * sizeof(float)));
  FMM_TRY(p->l2l_T.ensure(l2lT.size() * sizeof(float)));
  FMM_CUDA_TRY(cudaMemcpy(p->m2m_T.ptr, m2mT.data(), m2mT.size() * sizeof(float), cudaMemcpyHostToDevice));
  FMM_CUDA_TRY(cudaMemcpy(p->l2l_T.ptr, l2lT.data(), l2lT.size() * sizeof(float), cudaMemcpyHostToDevice));
  // L2P weights for the 5 outputs (n',m') in {(1,0),(1,1),(2,0),(2,1),(2,2)}
  // over inputs (k,l), |l| <= k, index k^2 + k + l:  nu_{n'+k}^{m'+l} / nu_k^l
  const int outs[5][2] = {{1, 0}, {1, 1}, {2, 0}, {2, 1}, {2, 2}};
  std::vector<float> w((size_t)5 * P, 0.f);
  for (int o = 0; o < 5; ++o)
    for (int k = 0; k < pp; ++k)
      for (int l = -k; l <= k; ++l) {
        int n2 = outs[o][0], m2 = outs[o][1];
        if (n2 + k > pp - 1 || std::abs(m2 + l) > n2 + k) continue;
        w[(size_t)o * P + k * k + k + l] = (float)(nu_d(n2 + k, m2 + l) / nu_d(k, l));
      }
  // The L2P gather table: entry o P + (k^2 + k + mm) of the leaf's derivative
  // coefficients D_o(k, mm) = c_re L~(i_re) + i c_im L~(i_im) (per potential),
  // with L~_N^M, N = n'_o + k, M = m'_o + mm read from the real-packed
  // storage (re at N^2 + (|M| ? 2|M| - 1 : 0), im at N^2 + 2|M|), the signs
  // of M < 0, the weight, and (-1)^m for mm = -m < 0 folded into
  // c_re, c_im (zero where N > p - 1 or the term has no imaginary part).
  std::vector<int4> tab((size_t)5 * P);
  for (int o = 0; o < 5; ++o)
    for (int k = 0; k < pp; ++k)
      for (int mm = -k; mm <= k; ++mm) {
        const int kk = k * k + k + mm, m = std::abs(mm);
        const int N = outs[o][0] + k, M = outs[o][1] + mm;
        int4 t = make_int4(0, 0, 0, 0);
        if (N <= pp - 1) {
          const float wv = w[(size_t)o * P + kk];
          const float sg = (mm < 0 && (m & 1)) ? -wv : wv;
          const int am = std::abs(M);
          float sre = 1.f, sim = am == 0 ? 0.f : 1.f;
          if (M < 0) {  // L~_N^{-|M|} = (-1)^|M| conj(L~_N^{|M|})
            sim = -sim;
            if (am & 1) {
              sre = -sre;
              sim = -sim;
            }
          }
          const float cre = sg * sre, cim = sg * sim;
          t.x = N * N + (am == 0 ? 0 : 2 * am - 1);
          t.y = am == 0 ? 0 : N * N + 2 * am;
          std::memcpy(&t.z, &cre, sizeof(float));
          std::memcpy(&t.w, &cim, sizeof(float));
        }
        tab[(size_t)o * P + kk] = t;
      }
  FMM_TRY(p->l2p_tab.ensure(tab.size() * sizeof(int4)));
  FMM_CUDA_TRY(cudaMemcpy(p->l2p_tab.ptr, tab.data(), tab.size() * sizeof(int4), cudaMemcpyHostToDevice));
  std::vector<double> inu(P);
  for (int n = 0; n < pp; ++n)
    for (int m = 0; m <= n; ++m)
      for (int part = 0; part < (m ? 2 : 1); ++part) inu[ridx(n, m, part)] = 1.0 / nu_d(n, m);
  FMM_TRY(p->m2l_inu.ensure(inu.size() * sizeof(double)));
  FMM_CUDA_TRY(cudaMemcpy(p->m2l_inu.ptr, inu.data(), inu.size() * sizeof(double), cudaMemcpyHostToDevice));
  if (p->prm.periodic) {  // the lattice operator, in FP64 on the device
    FMM_TRY(p->lattice.ensure((size_t)P * P * sizeof(double)));
    FMM_TRY(lattice_operator_device(pp, p->prm.images, p->lattice.as<double>(), 0));
  }
  return FMM_OK;
}

// The lattice operator built on the host (the same sums in FP64 C++), kept to
// cross-check the device build (fmm_lattice_operator).
int lattice_operator_host(int p, int images, double* out) {
  Mat A = lattice_matrix(p, images);
  for (size_t q = 0; q < A.size(); ++q) out[q] = A[q];
  return FMM_OK;
}

__global__ void k_remap_slots(int* __restrict__ st_slot, int64_t ns, const int* __restrict__ map) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < ns) st_slot[i] = map[st_slot[i]];
}

// ---- The operator cache.  M2L operators are constants of (translation key,
// p): a plan keeps those it has built, found through an open-addressing table
// in device memory (key -> operator slot).  One thread per distinct key of the
// evaluation looks it up; the missing keys are numbered in key order by a
// scan, inserted and built.  The host reads only the number of missing keys,
// with the step count it reads anyway.  A host map, with its two copies and two
// synchronisations, was most of what separated 1.73 from 0.98 ms in the
// traversal of a Plummer cloud of 30,011 blobs (29,043 translations).
constexpr uint64_t kNoKey = ~0ull;  // no key has all its level bits set
constexpr int64_t kCacheSlots = 1 << 16;  // operators kept (more only if one evaluation needs more)

// The public-domain 64-bit finaliser of MurmurHash3 (A. Appleby).
__device__ __forceinline__ uint64_t key_hash(uint64_t k) {
  k ^= k >> 33;
  k *= 0xff51afd7ed558ccdull;
  k ^= k >> 33;
  k *= 0xc4ceb9fe1a85ec53ull;
  k ^= k >> 33;
  return k;
}

__global__ void k_cache_find(const uint64_t* __restrict__ ukeys, int64_t nk, const uint64_t* __restrict__ tkey,
                             const int* __restrict__ tslot, uint64_t mask, int* __restrict__ map,
                             uint32_t* __restrict__ miss) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nk) return;
  const uint64_t k = ukeys[i];
  uint64_t h = key_hash(k) & mask;
  int slot = -1;
  for (uint64_t q = 0; q <= mask; ++q, h = (h + 1) & mask) {
    const uint64_t v = tkey[h];
    if (v == k) slot = tslot[h];
    if (v == k || v == kNoKey) break;
  }
  map[i] = slot;
  miss[i] = slot < 0 ? 1u : 0u;
}

// The missing keys take the slots from `base` on, in key order.  The keys of
// one evaluation are distinct, and the table is at most half full.
__global__ void k_cache_insert(const uint64_t* __restrict__ ukeys, int64_t nk, const uint32_t* __restrict__ miss,
                               const uint32_t* __restrict__ rank, int base, unsigned long long* __restrict__ tkey,
                               int* __restrict__ tslot, uint64_t mask, int* __restrict__ map,
                               uint64_t* __restrict__ mkeys, int* __restrict__ mslots) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nk || !miss[i]) return;
  const uint64_t k = ukeys[i];
  const int slot = base + (int)rank[i];
  uint64_t h = key_hash(k) & mask;
  for (uint64_t q = 0; q <= mask; ++q, h = (h + 1) & mask)
    if (atomicCAS(&tkey[h], kNoKey, k) == kNoKey) {
      tslot[h] = slot;
      break;
    }
  map[i] = slot;
  mkeys[rank[i]] = k;
  mslots[rank[i]] = slot;
}

// Empty table for at least nk keys.  Until it is all there the plan has none
// (tc_cap 0): an allocation may fail with the old arrays already released.
static int cache_clear(fmm_plan p, int64_t nk, cudaStream_t s) {
  int64_t cap = 2 * kCacheSlots;
  while (cap < 2 * nk) cap *= 2;
  p->tc_cap = 0;
  p->tc_size = 0;
  FMM_TRY(p->tc_key.ensure((size_t)cap * sizeof(uint64_t)));
  FMM_TRY(p->tc_slot.ensure((size_t)cap * sizeof(int)));
  FMM_CUDA_TRY(cudaMemsetAsync(p->tc_key.ptr, 0xff, (size_t)cap * sizeof(uint64_t), s));
  p->tc_cap = cap;
  return FMM_OK;
}

static int cache_find(fmm_plan p, uint32_t* miss, uint32_t* rank, uint32_t* nmiss, cudaStream_t s) {
  const int64_t nk = p->n_keys;
  ++g_launches;
  k_cache_find<<<(unsigned)((nk + 255) / 256), 256, 0, s>>>(p->ukeys.as<uint64_t>(), nk, p->tc_key.as<uint64_t>(),
                                                            p->tc_slot.as<int>(), (uint64_t)p->tc_cap - 1,
                                                            p->tslot_map.as<int>(), miss);
  FMM_CUDA_TRY(cudaGetLastError());
  return exclusive_scan_u32(miss, rank, nk, nmiss, p->scan_tmp, s);
}

// Looks up the n_keys translations of this evaluation (ukeys, distinct): the
// operator slot of each found key to tslot_map, the missing ones flagged and
// ranked; *nmiss (device) = their number.
int find_m2l_operators(fmm_plan p, uint32_t* miss, uint32_t* rank, uint32_t* nmiss, cudaStream_t s) {
  FMM_TRY(p->tslot_map.ensure((size_t)std::max<int64_t>(p->n_keys, 1) * sizeof(int)));
  if (!p->tc_cap) FMM_TRY(cache_clear(p, p->n_keys, s));
  return cache_find(p, miss, rank, nmiss, s);
}

// Builds the nmiss missing operators (in FP64, on the device); afterwards
// tslot_map holds the slot of every key.
int build_m2l_operators(fmm_plan p, int64_t nmiss, uint32_t* miss, uint32_t* rank, uint32_t* nmiss_dev,
                        cudaStream_t s) {
  const int P = p->P;
  p->n_built = 0;
  if (nmiss == 0) return FMM_OK;
  const int64_t nk = p->n_keys;
  // BF16 tiles only for the tensor-core path (the plan's M2L mode does not
  // change between evaluations)
  const int tc = p->last_tc;
  // bound the cache: start over when this evaluation's new operators would
  // take it past kCacheSlots (a cleared cache then holds exactly this evaluation's)
  if (p->tc_size + nmiss > std::max<int64_t>(kCacheSlots, p->tc_size)) {
    FMM_TRY(cache_clear(p, nk, s));
    FMM_TRY(cache_find(p, miss, rank, nmiss_dev, s));
    nmiss = nk;
  }
  const int64_t need = p->tc_size + nmiss;
  if (need > p->tcache_cap) {
    int64_t cap = std::max<int64_t>(need, p->tcache_cap * 2);
    if (!tc) FMM_TRY(p->T32.grow_copy((size_t)cap * P * P * sizeof(float), s));
    if (tc)
      FMM_TRY(p->Tbf.grow_copy((size_t)cap * 2 * m2l_kchunks(P, p->tc_kind) * m2l_cols(P) * 128, s));
    p->tcache_cap = cap;
  }
  FMM_TRY(p->tmiss_keys.ensure((size_t)nmiss * sizeof(uint64_t)));
  FMM_TRY(p->tmiss_slots.ensure((size_t)nmiss * sizeof(int)));
  ++g_launches;
  k_cache_insert<<<(unsigned)((nk + 255) / 256), 256, 0, s>>>(
      p->ukeys.as<uint64_t>(), nk, miss, rank, (int)p->tc_size, p->tc_key.as<unsigned long long>(),
      p->tc_slot.as<int>(), (uint64_t)p->tc_cap - 1, p->tslot_map.as<int>(), p->tmiss_keys.as<uint64_t>(),
      p->tmiss_slots.as<int>());
  ++g_launches;
  k_build_m2l<<<(unsigned)nmiss, 256, 0, s>>>(p->tmiss_keys.as<uint64_t>(), p->tmiss_slots.as<int>(), (int)nmiss,
                                              p->prm.p, p->m2l_inu.as<double>(), p->T32.as<float>(),
                                              p->Tbf.as<uint8_t>(),
                                              tc ? m2l_kchunks(P, p->tc_kind) : 0, p->tc_kind);
  FMM_CUDA_TRY(cudaGetLastError());
  p->tc_size = need;
  p->n_built = nmiss;
  return FMM_OK;
}

// Step list from unique-key index to operator slot.
int remap_step_slots(fmm_plan p, cudaStream_t s) {
  ++g_launches;
  k_remap_slots<<<(unsigned)((p->n_steps + 255) / 256), 256, 0, s>>>(p->st_slot.as<int>(), p->n_steps,
                                                                    p->tslot_map.as<int>());
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

int apply_lattice(fmm_plan p, cudaStream_t s) {
  if (!p->prm.periodic || p->prm.images <= 1) return FMM_OK;
  ++g_launches;
  k_apply_lattice<<<p->batched ? p->nseg : 1, 512, 0, s>>>(p->lattice.as<double>(), p->P, p->L.as<float>(),
                                                           p->M.as<float>());
  FMM_CUDA_TRY(cudaGetLastError());
  return FMM_OK;
}

}  // namespace fmm
