// ve_fx16.cuh -- PSD projection of one 16 x 16 matrix (real symmetric or complex Hermitian) by one
// warp, to float64 accuracy without float64 arithmetic: the products run on the tensor cores in
// sliced fixed point, the eigensolve in float32, and the eigenvectors are corrected until the
// first-order reconstruction is exact to float64 rounding.
//
// Why.  A float64 warp instruction costs 16-19 SM cycles here (64 for a warp alone on its
// sub-partition) and a warm complex Jacobi projection took ~6900 of them, 5100 in its two float64
// sweeps.  Nothing in it needs float64 arithmetic, only float64 accuracy of A = V^H C V, of V's
// orthonormality and of V M V^H.
//
// Products ("Ozaki scheme": Ozaki, Ogita, Oishi & Rump 2012; on tensor cores Mukunoki, Ozaki,
// Ogita & Imamura 2020).  A matrix is held as integers |X| <= 2^53 with one common exponent, and X as
// six balanced base-512 digits, exact in float16.  mma.sync m16n8k16 multiplies digit planes; all
// 16-term sums of the planes s + t = q together stay below 2^24 (12 x 16 x 256^2), so the float32
// accumulation is exact; planes with q <= 6 are kept (without q = 6 a product's error is 2^-52 of
// max|X| max|Y| and the X step's 1.5 times that of float64 arithmetic; with it, 2^-56).  One complex
// 16 x 16 product: 208 MMAs and ~1000 integer instructions for the 512 float64 ones.  The warp-level mma.sync is the right size here: one matrix is one 16 x 16
// tile, a tcgen05 tile (128 rows) would hold eight matrices' unrelated products.
//
// Layout.  Every matrix lives in registers in the A-fragment layout of m16n8k16: element i of a
// lane (g = lane / 4, t = lane % 4) is row g + 8 (i / 2 % 2), column 2 t + i % 2 + 8 (i / 4).  A
// product X Y^T of two matrices so laid out (Y's fragments are then the B operand) comes back in the
// same layout, so chains need no shuffles; transposes go through shared memory.
//
// Eigenvectors.  A is diagonalised in float32 (Jacobi); its rotations Q are float32-accurate and
// unitary to ~1e-6.  V1 = V Q, its Gram matrix I + G formed exactly, V <- V1 (I - G/2 + 3 G^2/8)
// (orthonormal to ~1e-17), and A is formed again.  Its off-diagonal part is now ~1e-10 of the one
// before (float32 is relative to the entries), and the first-order (Daleckii-Krein) rule of
// dk_stop ends the projection; otherwise the cycle repeats.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "ve_device.cuh"

namespace ve {
namespace fx16 {

constexpr int kD = 6;                                              // base-512 digits of an integer
constexpr int kLd = 17;
constexpr long long kBias = 256LL * (((1LL << 54) - 1) / 511);     // 256 in every digit
constexpr int kMaxCycles = 6;

using Frag = long long[8];  // one real 16 x 16 matrix, A-fragment layout

// Shared memory of a warp: two regions of digit fragments (region 0 also holds, at other times, the
// float32 Jacobi's matrices and transposes) and the eigenvalues.
template <bool CPLX>
struct Smem {
  static constexpr size_t region = (CPLX ? 2 : 1) * (size_t)kD * 512;
  static constexpr size_t lam = 2 * region;  // 16 eigenvalues as float32 pairs: high parts, low parts
  static constexpr size_t bytes = lam + 128;
  static constexpr size_t vectors = (CPLX ? 2 : 1) * 256 * 8;  // an eigenvector store of 8-byte words
  static_assert((CPLX ? 2 : 1) * 16 * kLd * 8 <= region && (CPLX ? 4 : 2) * 16 * kLd * 4 <= region, "regions");
};

__device__ __forceinline__ int frag_row(int i, int lane) { return (lane >> 2) + 8 * ((i >> 1) & 1); }
__device__ __forceinline__ int frag_col(int i, int lane) { return 2 * (lane & 3) + (i & 1) + 8 * (i >> 2); }

// x / 2^k rounded (k > 0), or x 2^-k; k uniform or not.
__device__ __forceinline__ long long shift_round(long long x, int k) {
  if (k > 62) return 0;
  if (k > 0) return (x + (1LL << (k - 1))) >> k;
  return x << (k < -62 ? 62 : -k);
}

// Integer <-> float32 without 64-bit conversion instructions (those run at the float64 rate).
// x 2^-53 as a float32, and a float32 |f| <= ~1 as an integer in units of 2^-53.
__device__ __forceinline__ float unit_float(long long x) {
  const int hi = (int)((x + (1 << 29)) >> 30), lo = (int)(x - (long long)hi * (1 << 30));  // |lo| <= 2^29
  return fmaf((float)hi, 1.1920929e-07f, (float)lo * 1.1102230246251565e-16f);
}
__device__ __forceinline__ long long unit_fix(float f) {
  const float t = f * 8388608.f;
  const int hi = __float2int_rn(t);
  const int lo = __float2int_rn((t - (float)hi) * 1073741824.f);
  return (long long)hi * (1 << 30) + lo;
}

// ---- float64 <-> fixed point -----------------------------------------------------------------
// The exponent field E of the largest entry scales a matrix: an entry of that binade becomes
// 2^52 <= |X| < 2^53 and X stands for X 2^(E - 1075).  Integer instructions only.
__device__ __forceinline__ int exponent_field(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ long long fix(double v, int E) {
  const long long b = __double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  long long m = b & 0xfffffffffffffLL;
  if (e) m |= 1LL << 52;
  m = shift_round(m, E - (e ? e : 1));
  return b < 0 ? -m : m;
}
// x 2^e, |x| < 2^62, rounded to nearest (halves away from zero).
__device__ __forceinline__ double word(long long x, int e) {
  unsigned long long a = (unsigned long long)(x < 0 ? -x : x);
  if (a == 0) return 0.0;
  int lz = __clzll((long long)a);
  if (lz < 11) {
    const int k = 11 - lz;
    a = (a + (1ULL << (k - 1))) >> k;
    e += k;
    if (a >> 53) {
      a >>= 1;
      ++e;
    }
    lz = 11;
  }
  const int sh = lz - 11, ex = e - sh + 1075;
  const unsigned long long sign = x < 0 ? 1ULL << 63 : 0;
  if (ex <= 0) {  // subnormal
    if (ex < -52) return 0.0;
    return __longlong_as_double((long long)(sign | (((a << sh) + (1ULL << -ex)) >> (1 - ex))));
  }
  if (ex >= 0x7ff) return __longlong_as_double((long long)(sign | (0x7ffULL << 52)));
  return __longlong_as_double((long long)(sign | ((unsigned long long)ex << 52) | ((a << sh) & 0xfffffffffffffULL)));
}

// Common power of two out of a matrix: |X| < 2^53 with the largest entry in the top binade.
template <bool CPLX>
__device__ __forceinline__ void normalise(Frag& r, Frag& i, int& e) {
  unsigned long long m = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    m |= (unsigned long long)(r[k] ^ (r[k] >> 63));
    if constexpr (CPLX) m |= (unsigned long long)(i[k] ^ (i[k] >> 63));
  }
  const unsigned hi = __reduce_or_sync(0xffffffffu, (unsigned)(m >> 32));
  const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)m);
  const int top = hi ? 63 - __clz((int)hi) : 31 - __clz((int)lo);  // -1 for a zero matrix
  const int k = top < 0 ? 0 : top - 52;
  if (k > 0) {
    const long long h = 1LL << (k - 1);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      r[j] = (r[j] + h) >> k;
      if constexpr (CPLX) i[j] = (i[j] + h) >> k;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      r[j] <<= -k;
      if constexpr (CPLX) i[j] <<= -k;
    }
  }
  e += k;
}

// ---- digits ------------------------------------------------------------------------------------
// The top N balanced base-512 digits as float16 A fragments.  Adding 256 in every digit makes them
// plain bit fields n = d + 256; 0x6400 | n is the float16 1024 + n, and 1280 is taken off again.
template <int N>
__device__ __forceinline__ void digits(const Frag& x, uint32_t (&d)[N][4]) {
  const __half2 off = __halves2half2(__ushort_as_half(0x6500), __ushort_as_half(0x6500));
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const unsigned long long b0 = (unsigned long long)(x[2 * r] + kBias);
    const unsigned long long b1 = (unsigned long long)(x[2 * r + 1] + kBias);
    const uint32_t l0 = (uint32_t)b0, m0 = (uint32_t)(b0 >> 27);
    const uint32_t l1 = (uint32_t)b1, m1 = (uint32_t)(b1 >> 27);
#pragma unroll
    for (int s = 0; s < N; ++s) {
      const uint32_t w0 = s < 3 ? m0 >> (18 - 9 * s) : l0 >> (45 - 9 * s);
      const uint32_t w1 = s < 3 ? m1 >> (18 - 9 * s) : l1 >> (45 - 9 * s);
      const uint32_t mask = s == 0 ? 0x3ffu : 0x1ffu;  // the top digit may reach +256
      const uint32_t n = (w0 & mask) | ((w1 & mask) << 16) | 0x64006400u;
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&n), off);
      d[s][r] = *reinterpret_cast<const uint32_t*>(&h);
    }
  }
}

// Right-operand fragments in shared memory: [digit][n-tile][lane] words of two registers.
template <int N>
__device__ __forceinline__ void put(const uint32_t (&d)[N][4], uint2* f, int lane) {
#pragma unroll
  for (int s = 0; s < N; ++s) {
    f[(2 * s) * 32 + lane] = make_uint2(d[s][0], d[s][2]);
    f[(2 * s + 1) * 32 + lane] = make_uint2(d[s][1], d[s][3]);
  }
}

__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Sum over q of S_q 512^-q as an integer; the product of X 2^ex and Y 2^ey is that integer times
// 2^(ex + ey + product_exp<Q>).
template <int Q>
constexpr int product_exp() {
  return Q == 6 ? 50 : Q == 3 ? 63 : 81;
}
template <int Q>
__device__ __forceinline__ long long combine(const float (&acc)[Q + 1][4], int i) {
  int s[Q + 1];
#pragma unroll
  for (int q = 0; q <= Q; ++q) s[q] = __float2int_rn(acc[q][i]);
  if constexpr (Q == 6) {
    const long long top = (long long)s[0] * 512 + s[1];
    return (top << 31) + (long long)s[2] * (1 << 22) + (long long)s[3] * (1 << 13) + (long long)(s[4] * 16) +
           ((s[5] + ((s[6] + 256) >> 9) + 16) >> 5);
  } else if constexpr (Q == 3) {
    return (((long long)s[0] * 512 + s[1]) << 18) + (long long)s[2] * 512 + s[3];
  } else {
    static_assert(Q == 1, "digit ranges in use");
    return (long long)s[0] * 512 + s[1];
  }
}

// Z = X Y^T, X = Lr + i SL Li (registers), Y = Rr + i SR Ri (shared-memory fragments), SL, SR = +-1
// (-1 takes the conjugate); the digit planes s + t <= Q.  The loop over the real and the imaginary
// part of Z stays rolled: the kernels' code is larger than the instruction caches otherwise.
template <int NL, int NR, int Q, bool CPLX, int SL, int SR>
__device__ __forceinline__ void product(const uint32_t (&Lr)[NL][4], const uint32_t (&Li)[NL][4], const uint2* R,
                                        Frag& zr, Frag& zi, int lane) {
  // part 0: Rr with Lr, -SL SR Ri with Li;  part 1: SR Ri with Lr, SL Rr with Li
  const uint2* b_of = R + lane;
  const uint2* c_of = R + NR * 64 + lane;
  uint32_t bm = 0, cm = SL * SR > 0 ? 0x80008000u : 0u;
#pragma unroll 1
  for (int part = 0; part < (CPLX ? 2 : 1); ++part) {
    Frag z;
#pragma unroll
    for (int tile = 0; tile < 2; ++tile) {
      float acc[Q + 1][4] = {};
#pragma unroll
      for (int t = 0; t < NR; ++t) {
        uint2 b = b_of[(2 * t + tile) * 32];
        if constexpr (CPLX && SR < 0) {
          b.x ^= bm;
          b.y ^= bm;
        }
#pragma unroll
        for (int s = 0; s < NL; ++s)
          if (s + t <= Q) mma(acc[s + t], Lr[s], b.x, b.y);
        if constexpr (CPLX) {
          uint2 c = c_of[(2 * t + tile) * 32];
          c.x ^= cm;
          c.y ^= cm;
#pragma unroll
          for (int s = 0; s < NL; ++s)
            if (s + t <= Q) mma(acc[s + t], Li[s], c.x, c.y);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) z[4 * tile + i] = combine<Q>(acc, i);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      zr[i] = CPLX ? zi[i] : z[i];  // after two parts: zr the first, zi the second
      zi[i] = z[i];
    }
    if constexpr (CPLX) {
      const uint2* x = b_of;
      b_of = c_of;
      c_of = x;
      bm = 0x80008000u;
      cm = SL < 0 ? 0x80008000u : 0u;
    }
  }
}

// Transpose through `buf` (16 x 17 words per part; free before and after).
template <bool CPLX>
__device__ __forceinline__ void transpose(const Frag& r, const Frag& i, Frag& tr, Frag& ti, long long* buf, int lane) {
  long long* bi = buf + 16 * kLd;
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int o = frag_row(k, lane) * kLd + frag_col(k, lane);
    buf[o] = r[k];
    if constexpr (CPLX) bi[o] = i[k];
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int o = frag_col(k, lane) * kLd + frag_row(k, lane);
    tr[k] = buf[o];
    if constexpr (CPLX) ti[k] = bi[o];
  }
  __syncwarp();
}

// ---- the stopping rules -----------------------------------------------------------------------------
// Squared norms of A = diag + E (A scaled to entries of at most 1), summed over the warp: E, the
// part B of E between diagonal entries of opposite sign, and the diagonal's distance d from zero.
struct Off {
  float off = 0.f, cross = 0.f, dg = 0.f, d = 1e30f;
  __device__ __forceinline__ void add(int i, int j, float re, float im, float li, float lj) {
    if (i == j) {
      dg = fmaf(li, li, dg);
      d = fminf(d, fabsf(li));
    } else {
      const float a = fmaf(re, re, im * im);
      off += a;
      if ((li < 0.f) != (lj < 0.f)) cross += a;
    }
  }
  __device__ __forceinline__ void reduce() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      off += shfl_xor(off, o);
      cross += shfl_xor(cross, o);
      dg += shfl_xor(dg, o);
      d = fminf(d, shfl_xor(d, o));
    }
  }
  __device__ __forceinline__ float nrm2() const { return dg + off; }
  // First-order rule.  With f = max(., 0) linear on either side of zero, f(A) = f(Lambda) + L o E +
  // R where R needs the two signs to mix: R vanishes with B, and ||R|| <= c ||B|| ||E|| / d while
  // ||E|| <= d / 4 (c <= 0.25 over random and clustered spectra, tests/test_fx16.py).  So E between
  // eigenvalues of one sign need not be rotated away, and ||B|| ||E|| <= n u ||A|| d / margin stops
  // as accurately as the exact rule (n u: jacobi_sym).
  __device__ __forceinline__ bool first_order(float margin) const {
    return margin * sqrtf(cross) * sqrtf(off) <= 16.f * 1.1102230246251565e-16f * sqrtf(nrm2()) * d &&
           16.f * off <= d * d;
  }
};

// ---- float32 Jacobi on a 16 x 16 matrix in shared memory, one warp ------------------------------
// The method of jacobi_sym / jacobi_herm; every lane keeps the rotation of pair lane % 8 (computed
// redundantly, passed on by shuffles) and its own indices, so a round is two warp barriers.
// Stops when off(A) <= 1e-10 ||A|| or when the float64 first-order rule holds with a margin of 4 on
// this matrix, after min_sw sweeps at least.  Returns the sweeps.
// An entry that this call need not remove is dropped, not rotated away (off0: the squared norm of E at
// the start; float32 angles leave 1e-7 of it, the stop 1e-10 ||A||, rounding 1e-17): with the two diagonal
// entries equal in float32, as in every multiplet of a symmetric model, it would turn the pair by 45
// degrees every sweep and E would only halve (XXZ chain, Delta = 0.9: 18 sweeps a wavevector block in place
// of 2; the projection step 361 and 82 us for 24 clusters, 587 and 154 us for 4096).
// EIG (eigenvalues): until off(A) has fallen by 1e7 (what float32 angles can give), and the diagonal
// is held as float32 pairs (low parts in dl): differences of nearly equal eigenvalues decide the angles there, and float32 alone would leave
// 1e-8 of them on the off-diagonal however often the cycle ran (a projection does not care about
// the basis within one sign).
__device__ __forceinline__ int next15(int a) { return a == 14 ? 0 : a + 1; }

template <bool CPLX, bool EIG>
__device__ int jacobi(float* Ar, float* Ai, float* Qr, float* Qi, float* dl, float off0, int lane, int min_sw,
                      int max_sw) {
  constexpr int LD = kLd;
  const float rel = fmaxf(6e-9f * sqrtf(off0), 4e-17f), negligible = EIG ? rel : fminf(rel, 2e-12f);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int e = lane + 32 * j, o = (e >> 4) * LD + (e & 15);
    Qr[o] = (e >> 4) == (e & 15) ? 1.f : 0.f;
    if constexpr (CPLX) Qi[o] = 0.f;
  }
  __syncwarp();
  int k1 = 0, k2 = 0;
  if (lane < 28) rr_pair(8, lane >> 2, lane & 3, k1, k2);
  const int k = lane & 7;
  [[maybe_unused]] float start = 0.f;
  int sw = 0;
  for (; sw < max_sw; ++sw) {
    if (EIG || sw >= min_sw) {
      Off f;
      const int j = lane & 15;
      const float lj = Ar[j * LD + j];
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        const int i = (lane >> 4) + 2 * h;
        f.add(i, j, Ar[i * LD + j], CPLX ? Ai[i * LD + j] : 0.f, Ar[i * LD + i], lj);
      }
      f.reduce();
      if constexpr (EIG) {
        if (sw == 0) start = f.off;
        else if (f.off <= 1e-14f * start) break;
      } else if (f.off <= 1e-20f * f.nrm2() || f.first_order(4.f)) {
        break;
      }
    }
    // indices of the pair this lane rotates and of its block's two pairs, advanced every round
    int a = k == 0 ? 15 : k, b = k == 0 ? 0 : 15 - k;
    int a1 = k1 == 0 ? 15 : k1, b1 = k1 == 0 ? 0 : 15 - k1;
    int a2 = k2 == 0 ? 15 : k2, b2 = k2 == 0 ? 0 : 15 - k2;
    for (int r = 0; r < 15; ++r) {
      const int p = min(a, b), q = max(a, b);
      const float app = Ar[p * LD + p], aqq = Ar[q * LD + q], br = Ar[p * LD + q];
      float c, s, t, mag, wr = 1.f, wi = 0.f;
      if constexpr (CPLX) {
        const float bi = Ai[p * LD + q];
        mag = 0.f;
        if (br != 0.f || bi != 0.f) unit_phase<float>(br, bi, mag, wr, wi);
      } else {
        mag = br;
      }
      if (fabsf(mag) <= negligible) mag = 0.f;
      float npp, nqq, lpp = 0.f, lqq = 0.f;
      if constexpr (EIG) {
        const float dp = dl[p], dq = dl[q];
        sym_schur2<float>(0.f, (aqq - app) + (dq - dp), mag, c, s, t);
        float e;
        two_sum(app, -t * mag, npp, e);
        fast_two_sum(npp, dp + e, npp, lpp);
        two_sum(aqq, t * mag, nqq, e);
        fast_two_sum(nqq, dq + e, nqq, lqq);
      } else {
        sym_schur2<float>(app, aqq, mag, c, s, t);
        npp = app - t * mag;
        nqq = aqq + t * mag;
      }
      __syncwarp();
      if (lane < 8) {
        Ar[p * LD + p] = npp;
        Ar[q * LD + q] = nqq;
        if constexpr (EIG) {
          dl[p] = lpp;
          dl[q] = lqq;
        }
        Ar[p * LD + q] = 0.f;
        Ar[q * LD + p] = 0.f;
        if constexpr (CPLX) {
          Ai[p * LD + q] = 0.f;
          Ai[q * LD + p] = 0.f;
        }
      }
      const unsigned all = 0xffffffffu;
      const float c1 = __shfl_sync(all, c, k1), s1 = __shfl_sync(all, s, k1);
      const float c2 = __shfl_sync(all, c, k2), s2 = __shfl_sync(all, s, k2);
      float w1r = 1.f, w1i = 0.f, w2r = 1.f, w2i = 0.f;
      if constexpr (CPLX) {
        w1r = __shfl_sync(all, wr, k1);
        w1i = __shfl_sync(all, wi, k1);
        w2r = __shfl_sync(all, wr, k2);
        w2i = __shfl_sync(all, wi, k2);
      }
      if (lane < 28) {
        const int p1 = min(a1, b1), q1 = max(a1, b1), p2 = min(a2, b2), q2 = max(a2, b2);
        const int opp = p1 * LD + p2, opq = p1 * LD + q2, oqp = q1 * LD + p2, oqq = q1 * LD + q2;
        const int tpp = p2 * LD + p1, tpq = q2 * LD + p1, tqp = p2 * LD + q1, tqq = q2 * LD + q1;
        const float m11r = Ar[opp], m12r = Ar[opq], m21r = Ar[oqp], m22r = Ar[oqq];
        if constexpr (CPLX) {
          const float m11i = Ai[opp], m12i = Ai[opq], m21i = Ai[oqp], m22i = Ai[oqq];
          const float sw2r = s2 * w2r, sw2i = s2 * w2i, cw2r = c2 * w2r, cw2i = c2 * w2i;
          const float x11r = c2 * m11r - (sw2r * m12r - sw2i * m12i);
          const float x11i = c2 * m11i - (sw2r * m12i + sw2i * m12r);
          const float x12r = s2 * m11r + (cw2r * m12r - cw2i * m12i);
          const float x12i = s2 * m11i + (cw2r * m12i + cw2i * m12r);
          const float x21r = c2 * m21r - (sw2r * m22r - sw2i * m22i);
          const float x21i = c2 * m21i - (sw2r * m22i + sw2i * m22r);
          const float x22r = s2 * m21r + (cw2r * m22r - cw2i * m22i);
          const float x22i = s2 * m21i + (cw2r * m22i + cw2i * m22r);
          const float sw1r = s1 * w1r, sw1i = -s1 * w1i, cw1r = c1 * w1r, cw1i = -c1 * w1i;
          const float y11r = c1 * x11r - (sw1r * x21r - sw1i * x21i);
          const float y11i = c1 * x11i - (sw1r * x21i + sw1i * x21r);
          const float y22r = s1 * x12r + (cw1r * x22r - cw1i * x22i);
          const float y22i = s1 * x12i + (cw1r * x22i + cw1i * x22r);
          const float y12r = c1 * x12r - (sw1r * x22r - sw1i * x22i);
          const float y12i = c1 * x12i - (sw1r * x22i + sw1i * x22r);
          const float y21r = s1 * x11r + (cw1r * x21r - cw1i * x21i);
          const float y21i = s1 * x11i + (cw1r * x21i + cw1i * x21r);
          Ar[opp] = y11r;
          Ai[opp] = y11i;
          Ar[tpp] = y11r;
          Ai[tpp] = -y11i;
          Ar[opq] = y12r;
          Ai[opq] = y12i;
          Ar[tpq] = y12r;
          Ai[tpq] = -y12i;
          Ar[oqp] = y21r;
          Ai[oqp] = y21i;
          Ar[tqp] = y21r;
          Ai[tqp] = -y21i;
          Ar[oqq] = y22r;
          Ai[oqq] = y22i;
          Ar[tqq] = y22r;
          Ai[tqq] = -y22i;
        } else {
          const float x11 = c2 * m11r - s2 * m12r, x12 = s2 * m11r + c2 * m12r;
          const float x21 = c2 * m21r - s2 * m22r, x22 = s2 * m21r + c2 * m22r;
          const float y11 = c1 * x11 - s1 * x21, y12 = c1 * x12 - s1 * x22;
          const float y21 = s1 * x11 + c1 * x21, y22 = s1 * x12 + c1 * x22;
          Ar[opp] = y11;
          Ar[tpp] = y11;
          Ar[opq] = y12;
          Ar[tpq] = y12;
          Ar[oqp] = y21;
          Ar[tqp] = y21;
          Ar[oqq] = y22;
          Ar[tqq] = y22;
        }
      }
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        const int row = ((lane >> 3) + 4 * it) * LD;
        const float vpr = Qr[row + p], vqr = Qr[row + q];
        if constexpr (CPLX) {
          const float vpi = Qi[row + p], vqi = Qi[row + q];
          const float wvr = wr * vqr - wi * vqi, wvi = wr * vqi + wi * vqr;
          Qr[row + p] = c * vpr - s * wvr;
          Qi[row + p] = c * vpi - s * wvi;
          Qr[row + q] = s * vpr + c * wvr;
          Qi[row + q] = s * vpi + c * wvi;
        } else {
          Qr[row + p] = c * vpr - s * vqr;
          Qr[row + q] = s * vpr + c * vqr;
        }
      }
      __syncwarp();
      a = a == 15 ? 15 : next15(a);
      b = next15(b);
      a1 = a1 == 15 ? 15 : next15(a1);
      b1 = next15(b1);
      a2 = a2 == 15 ? 15 : next15(a2);
      b2 = next15(b2);
    }
  }
  return sw;
}

// The eigenvector store: V, row-major 16 x 16 integers in units of 2^-53 (re, then im).
template <bool CPLX>
__device__ __forceinline__ void load_vectors(const long long* v, bool transposed, Frag& r, Frag& i, int lane) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int row = frag_row(k, lane), col = frag_col(k, lane);
    const int o = transposed ? col * 16 + row : row * 16 + col;
    r[k] = v[o];
    if constexpr (CPLX) i[k] = v[256 + o];
  }
}

template <bool CPLX>
__device__ __forceinline__ void store_vectors(long long* v, const Frag& r, const Frag& i, int lane) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int o = frag_row(k, lane) * 16 + frag_col(k, lane);
    v[o] = r[k];
    if constexpr (CPLX) v[256 + o] = i[k];
  }
}

template <bool CPLX>
__device__ __forceinline__ void identity_vectors(long long* v, int lane) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int row = frag_row(k, lane), col = frag_col(k, lane);
    v[row * 16 + col] = row == col ? 1LL << 53 : 0;
    if constexpr (CPLX) v[256 + row * 16 + col] = 0;
  }
}

// V <- the orthonormal factor of V Q in the store; Q: float32 rotations in region 0, of which NQ digits
// are used (four leave ~1e-11 on the off-diagonal of A, six 1e-16).
template <bool CPLX, int NQ>
__device__ void update_vectors(long long* v, const float* Qr, const float* Qi, unsigned char* s0, int lane) {
  uint2* f0 = reinterpret_cast<uint2*>(s0);
  Frag xr, xi;
  // V1 = V Q = V (Q^T)^T
  {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int o = frag_col(k, lane) * kLd + frag_row(k, lane);
      xr[k] = unit_fix(Qr[o]);
      if constexpr (CPLX) xi[k] = unit_fix(Qi[o]);
    }
    uint32_t q[NQ][4], dr[kD][4], di[kD][4];
    __syncwarp();
    digits<NQ>(xr, q);
    put<NQ>(q, f0, lane);
    if constexpr (CPLX) {
      digits<NQ>(xi, q);
      put<NQ>(q, f0 + NQ * 64, lane);
    }
    load_vectors<CPLX>(v, false, xr, xi, lane);
    digits<kD>(xr, dr);
    if constexpr (CPLX) digits<kD>(xi, di);
    __syncwarp();
    product<kD, NQ, 6, CPLX, 1, 1>(dr, di, f0, xr, xi, lane);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      xr[k] = (xr[k] + 4) >> 3;
      if constexpr (CPLX) xi[k] = (xi[k] + 4) >> 3;
    }
    store_vectors<CPLX>(v, xr, xi, lane);
    __syncwarp();
  }
  // I + G = V1^H V1 = conj(U) U^T with U = V1^T, in units of 2^-56
  {
    load_vectors<CPLX>(v, true, xr, xi, lane);
    uint32_t dr[kD][4], di[kD][4];
    digits<kD>(xr, dr);
    put<kD>(dr, f0, lane);
    if constexpr (CPLX) {
      digits<kD>(xi, di);
      put<kD>(di, f0 + kD * 64, lane);
    }
    __syncwarp();
    product<kD, kD, 6, CPLX, -1, 1>(dr, di, f0, xr, xi, lane);
    __syncwarp();
  }
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (frag_row(k, lane) == frag_col(k, lane)) xr[k] -= 1LL << 56;
  // T = -G / 2 + 3 G^2 / 8 (G^2 = G conj(G)^T from its two top digits: it is ~1e-6 of G)
  int et = -56;
  {
    Frag gr, gi;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      gr[k] = xr[k];
      if constexpr (CPLX) gi[k] = xi[k];
    }
    int eg = -56;
    normalise<CPLX>(gr, gi, eg);
    uint32_t dr[2][4], di[2][4];
    digits<2>(gr, dr);
    put<2>(dr, f0, lane);
    if constexpr (CPLX) {
      digits<2>(gi, di);
      put<2>(di, f0 + 2 * 64, lane);
    }
    __syncwarp();
    product<2, 2, 1, CPLX, 1, -1>(dr, di, f0, gr, gi, lane);
    __syncwarp();
    const int sh = -56 - (2 * eg + product_exp<1>()) + 3;  // to units of 2^-56, over 8
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      xr[k] = shift_round(3 * gr[k], sh) - ((xr[k] + 1) >> 1);
      if constexpr (CPLX) xi[k] = shift_round(3 * gi[k], sh) - ((xi[k] + 1) >> 1);
    }
  }
  normalise<CPLX>(xr, xi, et);
  // V <- V1 + V1 T (T Hermitian: T^T = conj(T))
  {
    uint32_t dr[4][4], di[4][4];
    digits<4>(xr, dr);
    put<4>(dr, f0, lane);
    if constexpr (CPLX) {
      digits<4>(xi, di);
      put<4>(di, f0 + 4 * 64, lane);
    }
    Frag vr, vi;
    load_vectors<CPLX>(v, false, vr, vi, lane);
    digits<4>(vr, dr);
    if constexpr (CPLX) digits<4>(vi, di);
    __syncwarp();
    product<4, 4, 3, CPLX, 1, -1>(dr, di, f0, xr, xi, lane);
    const int sh = -(et + product_exp<3>());  // units 2^(-53 + et + 63) -> 2^-53
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      vr[k] += shift_round(xr[k], sh);
      if constexpr (CPLX) vi[k] += shift_round(xi[k], sh);
    }
    store_vectors<CPLX>(v, vr, vi, lane);
    __syncwarp();
  }
}

// x times the divided difference of max(., 0) between p = ph + pl >= 0 and -q, q = qh + ql > 0, which is
// w = p / (p + q).  x is at most 6e-8 of the matrix where the first-order rule has just been met, so w to
// 2^-31 leaves less than a rounding of x; float32 alone (1e-7) left up to 5 u ||A|| there.
__device__ __forceinline__ int cross_weight(float ph, float pl, float qh, float ql) {  // units of 2^-30
  float dh, dl;
  two_sum(ph, qh, dh, dl);
  dl += pl + ql;
  const float inv = __fdividef(1.f, dh), w = ph * inv;
  const float r = fmaf(-w, dh, ph) + fmaf(-w, dl, pl);
  return __float2int_rn(w * 1073741824.f) + __float2int_rn(r * inv * 1073741824.f);
}
__device__ __forceinline__ long long weighted(long long x, int w) {
  const long long hi = (long long)(int)(x >> 32) * w;
  const unsigned long long lo = (unsigned long long)(uint32_t)x * (uint32_t)w;
  return (hi << 2) + (long long)((lo + (1ULL << 29)) >> 30);
}

// Y is in the fragments; Y = C; Y = 0; (EIG) A = V^H C V is in the fragments
enum Result { kProduct, kSame, kZero, kDiagonal };

// A matrix as fixed point, |X| < 2^53, in the fragment layout.  false when an entry is not finite.
template <bool CPLX>
__device__ __forceinline__ bool fix_matrix(const double (&cr)[8], const double (&ci)[8], Frag& ar, Frag& ai, int& e) {
  int E = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    E = max(E, exponent_field(cr[k]));
    if constexpr (CPLX) E = max(E, exponent_field(ci[k]));
  }
  E = (int)__reduce_max_sync(0xffffffffu, (unsigned)E);
  if (E == 0x7ff) return false;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    ar[k] = fix(cr[k], E);
    if constexpr (CPLX) ai[k] = fix(ci[k], E);
  }
  e = E - 1075;
  return true;
}

// x + x^H (of any matrix in the fragment layout), through region 0.
template <bool CPLX>
__device__ __forceinline__ void add_adjoint(Frag& r, Frag& i, unsigned char* s0, int lane) {
  Frag tr, ti;
  transpose<CPLX>(r, i, tr, ti, reinterpret_cast<long long*>(s0), lane);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    r[k] += tr[k];
    if constexpr (CPLX) i[k] -= ti[k];
  }
}

// Projection of a Hermitian matrix C by one warp.  (ar, ai), ea: C as integers (|X| < 2^53) times
// 2^ea, in the fragment layout; on kProduct they hold Y = Pi_{>=0}(C), exactly Hermitian (|X| <
// 2^60).  v: eigenvector store (global or shared memory): the starting vectors when `warm`, the
// final ones on return.  *dk: the first-order reconstruction ended
// it.  *nsw: the float32 Jacobi sweeps taken.  A definite C (found so by the first-order rule)
// needs no reconstruction: kSame or kZero.
// EIG: no projection; the cycle goes on to the exact rule and leaves A = V^H C V, diagonal but for
// *off2 = ||E||_F^2 (in units of 2^(2 (53 + ea))).
template <bool CPLX, bool EIG = false>
__device__ Result project(Frag& ar, Frag& ai, int& ea, long long* v, bool warm, unsigned char* sm, int lane, bool* dk,
                          int* nsw, float* off2 = nullptr) {
  unsigned char* s0 = sm;
  uint2* f0 = reinterpret_cast<uint2*>(s0);
  uint2* f1 = reinterpret_cast<uint2*>(sm + Smem<CPLX>::region);
  float* lam = reinterpret_cast<float*>(sm + Smem<CPLX>::lam);
  float* Jr = reinterpret_cast<float*>(s0);
  float* Qr = Jr + 16 * kLd;
  float* Ji = Qr + 16 * kLd;
  float* Qi = Ji + 16 * kLd;
  *dk = false;
  *nsw = 0;
  int e1 = ea;  // exponent of the matrix whose fragments are in region 1: C, and M at the end
  {
    uint32_t d[kD][4];
    digits<kD>(ar, d);
    put<kD>(d, f1, lane);
    if constexpr (CPLX) {
      digits<kD>(ai, d);
      put<kD>(d, f1 + kD * 64, lane);
    }
  }
  if (!warm) identity_vectors<CPLX>(v, lane);
  __syncwarp();
  bool last = false;
#pragma unroll 1
  for (int cyc = 0;; ++cyc) {
    if (cyc > 0 || warm) {
      // With X = U = V^T and C in region 1: W^T = U C^T, A = V^H C V = conj(U) W.  At the end, with
      // X = V and conj(M): Z = V M and conj(V) Z^T = Y^T.
      uint32_t dr[kD][4], di[kD][4];
      load_vectors<CPLX>(v, !last, ar, ai, lane);
      digits<kD>(ar, dr);
      if constexpr (CPLX) digits<kD>(ai, di);
      product<kD, kD, 6, CPLX, 1, 1>(dr, di, f1, ar, ai, lane);
      ea = -53 + e1 + product_exp<6>();
      normalise<CPLX>(ar, ai, ea);
      {
        uint32_t d[kD][4];
        digits<kD>(ar, d);
        put<kD>(d, f0, lane);
        if constexpr (CPLX) {
          digits<kD>(ai, d);
          put<kD>(d, f0 + kD * 64, lane);
        }
      }
      __syncwarp();
      product<kD, kD, 6, CPLX, -1, 1>(dr, di, f0, ar, ai, lane);
      ea += -53 + product_exp<6>();
      __syncwarp();
      if (last) break;
      normalise<CPLX>(ar, ai, ea);
    }
    // A in float32, scaled to max 1
    float xf[8], yf[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      xf[k] = unit_float(ar[k]);
      yf[k] = CPLX ? unit_float(ai[k]) : 0.f;
      if (frag_row(k, lane) == frag_col(k, lane)) lam[frag_row(k, lane)] = xf[k];
    }
    __syncwarp();
    Off f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = frag_row(k, lane), j = frag_col(k, lane);
      f.add(i, j, xf[k], yf[k], lam[i], lam[j]);
    }
    f.reduce();
    if constexpr (EIG) {
      if (f.off <= 3.1554436e-30f * f.nrm2() || cyc == kMaxCycles) {
        *off2 = f.off;
        return kDiagonal;
      }
    }
    *dk = !EIG && f.first_order(1.f);
    if (*dk) {
      const unsigned neg = __ballot_sync(0xffffffffu, lam[lane & 15] < 0.f);
      if (neg == 0u || neg == 0xffffffffu) return neg ? kZero : kSame;
    }
    if (!EIG && (*dk || f.off <= 3.1554436e-30f * f.nrm2() /* (n u)^2 */ || cyc == kMaxCycles)) {
      // M = f(Lambda) + L o E, conjugated, into region 1
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (frag_row(k, lane) == frag_col(k, lane)) lam[16 + frag_row(k, lane)] = unit_float(ar[k] - unit_fix(xf[k]));
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int i = frag_row(k, lane), j = frag_col(k, lane);
        const float li = lam[i], lj = lam[j];
        if (i == j) {
          ar[k] = ar[k] > 0 ? ar[k] : 0;
          if constexpr (CPLX) ai[k] = 0;
        } else if (li < 0.f || lj < 0.f) {
          const bool up = li >= lj;
          const float pl = lam[16 + (up ? i : j)], ql = -lam[16 + (up ? j : i)];
          const int w = (li < 0.f) != (lj < 0.f) ? cross_weight(fmaxf(li, lj), pl, -fminf(li, lj), ql) : 0;
          ar[k] = weighted(ar[k], w);
          if constexpr (CPLX) ai[k] = weighted(ai[k], w);
        }
        if constexpr (CPLX) ai[k] = -ai[k];
      }
      uint32_t d[kD][4];
      digits<kD>(ar, d);
      put<kD>(d, f1, lane);
      if constexpr (CPLX) {
        digits<kD>(ai, d);
        put<kD>(d, f1 + kD * 64, lane);
      }
      e1 = ea;
      last = true;
      warm = true;  // a cold start that needed no rotation: V = I is in the store
      __syncwarp();
      continue;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = frag_row(k, lane), j = frag_col(k, lane);
      if (i <= j) {
        Jr[i * kLd + j] = xf[k];
        Jr[j * kLd + i] = xf[k];
        if (EIG && i == j) lam[16 + i] = unit_float(ar[k] - unit_fix(xf[k]));
        if constexpr (CPLX) {
          Ji[i * kLd + j] = i == j ? 0.f : yf[k];
          Ji[j * kLd + i] = i == j ? 0.f : -yf[k];
        }
      }
    }
    __syncwarp();
    *nsw += jacobi<CPLX, EIG>(Jr, Ji, Qr, Qi, lam + 16, f.off, lane, 1, 10);
    update_vectors<CPLX, EIG ? kD : 4>(v, Qr, Qi, s0, lane);
  }
  // Y = (conj(Y^T) + Y^T's transpose) / 2
  if constexpr (CPLX) {
#pragma unroll
    for (int k = 0; k < 8; ++k) ai[k] = -ai[k];
  }
  add_adjoint<CPLX>(ar, ai, s0, lane);
  ea -= 1;
  return kProduct;
}

// A lower bound, up to rounding, on the smallest eigenvalue of C (as in project) by one warp: the smallest
// diagonal entry of A = V^H C V less ||E||_F (Weyl), whether or not the cycle converged.  Rounding, which
// nothing is taken off for: 2^-54 of the largest entry in every entry of C, and both products.  `sm` holds Smem and
// Smem::vectors bytes after it.
template <bool CPLX>
__device__ double lowest(Frag& ar, Frag& ai, int ea, unsigned char* sm, int lane) {
  bool dk;
  int nsw;
  float off2 = 0.f;
  project<CPLX, true>(ar, ai, ea, reinterpret_cast<long long*>(sm + Smem<CPLX>::bytes), false, sm, lane, &dk, &nsw,
                      &off2);
  double w = INFINITY;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (frag_row(k, lane) == frag_col(k, lane)) w = nan_min(w, word(ar[k], ea));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) w = nan_min(w, shfl_xor(w, o));
  __syncwarp();
  // the sum was taken in float32: rounded up by more than its error
  return w - 2.0 * (double)(sqrtf(off2) * 1.0001f) * word(1LL << 52, ea);
}

}  // namespace fx16
}  // namespace ve
