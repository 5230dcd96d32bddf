// ve_fx64.cuh -- PSD projection of one 64 x 64 matrix (real symmetric or complex Hermitian) by one
// CTA, to float64 accuracy without float64 products: Pi(C) = P C P, P = (I + sign(C)) / 2, with the matrix
// sign iteration of ve_fxstep.cuh and the sliced fixed-point products of ve_fx16.cuh (P from both sides:
// ve_fxsign.cu).
//
// Why the sign and not eigenvectors, as at 16 x 16: a float32 Jacobi sweep of a 64 x 64 matrix is 63
// rounds of CTA barriers, so the eigensolve would cost more than the 38 products of the projection,
// which need no starting vectors and no store either.
//
// Ten warps own the ten 16 x 16 blocks on and above the diagonal (the others are their conjugate
// transposes), so a product is 4 x 52 MMAs a warp (complex: 4 x 208).  The iterate and the second
// operand live in shared memory as digit fragments (96 KB each when complex); a block of X^2 stays
// in its warp's registers for the polynomial.  ~18 us a complex product, ~6 us a real one:
// the tensor pipe is 48 and 30 % busy, the rest is ten warps waiting for their MMAs and at the barriers of
// the dependent steps.
#pragma once

#include "ve_fxstep.cuh"

namespace ve {
namespace fx64 {

using fx16::Frag;
using fx16::kD;

constexpr int kThreads = 320, kWarps = 10;
constexpr int kPart = 16 * kD * 32;  // uint4 of one real 64 x 64 matrix

static __constant__ fxstep::Coef kCoef[fxstep::kSteps] = {
    fxstep::coef(0), fxstep::coef(1), fxstep::coef(2), fxstep::coef(3), fxstep::coef(4),  fxstep::coef(5),
    fxstep::coef(6), fxstep::coef(7), fxstep::coef(8), fxstep::coef(9), fxstep::coef(10), fxstep::coef(11)};

template <bool CPLX>
struct Smem {
  static constexpr size_t matrix = (CPLX ? 2 : 1) * kPart * sizeof(uint4);
  static constexpr size_t red = 2 * matrix;  // kWarps doubles, kWarps ints
  static constexpr size_t bytes = red + 128;
};

// The digits of block (I, J) of a Hermitian matrix, and conjugate-transposed as block (J, I); of a
// diagonal block the upper triangle counts.
template <bool CPLX>
__device__ __forceinline__ void write_block(const Frag& zr, const Frag& zi, uint4* out, int I, int J, int lane) {
  const int row = lane >> 2, col = 2 * (lane & 3);
  const uint32_t below = (col < row ? 0xffffu : 0u) | (col + 1 < row ? 0xffff0000u : 0u);
#pragma unroll
  for (int part = 0; part < (CPLX ? 2 : 1); ++part) {
    uint32_t d[kD][4];
    fx16::digits<kD>(part ? zi : zr, d);
    const uint32_t neg = part ? 0x80008000u : 0u;
    uint4* o = out + part * kPart + (I * 4 + J) * (kD * 32) + lane;
    uint4* t = out + part * kPart + (J * 4 + I) * (kD * 32) + lane;
#pragma unroll
    for (int s = 0; s < kD; ++s) {
      const uint4 v = make_uint4(d[s][0], d[s][1], d[s][2], d[s][3]);
      const uint4 w = make_uint4(fxstep::transpose8(v.x) ^ neg, fxstep::transpose8(v.z) ^ neg,
                                 fxstep::transpose8(v.y) ^ neg, fxstep::transpose8(v.w) ^ neg);
      if (I == J) {
        o[s * 32] = make_uint4((v.x & ~below) | (w.x & below), w.y, v.z, (v.w & ~below) | (w.w & below));
      } else {
        o[s * 32] = v;
        t[s * 32] = w;
      }
    }
  }
}

// The digits of block (I, J) of any matrix.
template <bool CPLX>
__device__ __forceinline__ void write_one(const Frag& zr, const Frag& zi, uint4* out, int I, int J, int lane) {
#pragma unroll
  for (int part = 0; part < (CPLX ? 2 : 1); ++part) {
    uint32_t d[kD][4];
    fx16::digits<kD>(part ? zi : zr, d);
    uint4* o = out + part * kPart + (I * 4 + J) * (kD * 32) + lane;
#pragma unroll
    for (int s = 0; s < kD; ++s) o[s * 32] = make_uint4(d[s][0], d[s][1], d[s][2], d[s][3]);
  }
}

// x += the transpose of t, 16 bits of its words at a time.
__device__ __forceinline__ void add_transpose(Frag& x, const Frag& t, bool negative) {
#pragma unroll
  for (int a = 0; a < 2; ++a)  // row half a, column half b of t
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const unsigned long long t0 = (unsigned long long)t[2 * a + 4 * b], t1 = (unsigned long long)t[2 * a + 4 * b + 1];
      unsigned long long v0 = 0, v1 = 0;
#pragma unroll
      for (int s = 0; s < 64; s += 16) {
        const uint32_t u = (uint32_t)((t0 >> s) & 0xffff) | ((uint32_t)((t1 >> s) & 0xffff) << 16);
        const uint32_t v = fxstep::transpose8(u);
        v0 |= (unsigned long long)(v & 0xffff) << s;
        v1 |= (unsigned long long)(v >> 16) << s;
      }
      long long &x0 = x[2 * b + 4 * a], &x1 = x[2 * b + 4 * a + 1];
      x0 += negative ? -(long long)v0 : (long long)v0;
      x1 += negative ? -(long long)v1 : (long long)v1;
    }
}

// Block (I, J) of A B, B Hermitian: sum_k A_Ik conj(B_Jk)^T.
template <bool CPLX>
__device__ __forceinline__ void product(const uint4* A, const uint4* B, int I, int J, Frag& zr, Frag& zi, int lane) {
#pragma unroll 1
  for (int part = 0; part < (CPLX ? 2 : 1); ++part) {
    Frag h = {};
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
      float acc[2][7][4] = {};
      // real part: Ar Br^T + Ai Bi^T; imaginary part: Ai Br^T - Ar Bi^T
#pragma unroll 1
      for (int u = 0; u < (CPLX ? 2 : 1); ++u) {
        const uint4* a = A + (CPLX ? (part ^ u) * kPart : 0) + (I * 4 + k) * (kD * 32) + lane;
        const uint4* b = B + (CPLX ? u * kPart : 0) + (J * 4 + k) * (kD * 32) + lane;
        const uint32_t neg = part & u ? 0x80008000u : 0u;
        uint32_t l[kD][4];
#pragma unroll
        for (int s = 0; s < kD; ++s) {
          const uint4 v = a[s * 32];
          l[s][0] = v.x;
          l[s][1] = v.y;
          l[s][2] = v.z;
          l[s][3] = v.w;
        }
#pragma unroll
        for (int t = 0; t < kD; ++t) {
          uint4 r = b[t * 32];
          if constexpr (CPLX) {
            r.x ^= neg;
            r.y ^= neg;
            r.z ^= neg;
            r.w ^= neg;
          }
#pragma unroll
          for (int s = 0; s < kD; ++s)
            if (s + t <= 6) {
              fx16::mma(acc[0][s + t], l[s], r.x, r.z);
              fx16::mma(acc[1][s + t], l[s], r.y, r.w);
            }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        h[i] += fx16::combine<6>(acc[0], i);
        h[4 + i] += fx16::combine<6>(acc[1], i);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      zr[i] = CPLX ? zi[i] : h[i];  // after two parts: zr the first, zi the second
      zi[i] = h[i];
    }
  }
}

// Sum, and largest value, over the CTA.
__device__ __forceinline__ double reduce_sum(double v, unsigned char* red, int tid) {
  double* rv = reinterpret_cast<double*>(red);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += shfl_xor(v, o);
  __syncthreads();
  if ((tid & 31) == 0) rv[tid >> 5] = v;
  __syncthreads();
  v = 0.0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) v += rv[w];
  return v;
}
__device__ __forceinline__ int reduce_max(int m, unsigned char* red, int tid) {
  int* rm = reinterpret_cast<int*>(red + kWarps * 8);
  m = (int)__reduce_max_sync(0xffffffffu, (unsigned)m);
  __syncthreads();
  if ((tid & 31) == 0) rm[tid >> 5] = m;
  __syncthreads();
  m = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) m = max(m, rm[w]);
  return m;
}

// load(row, col, re, im): entry of the matrix C, Hermitian when taken on and above the diagonal
// (called five times an entry); store(row, col, re, im): entry of the result, all of them (after a
// barrier: it may overwrite what load reads and the first Smem::matrix bytes of sm).  All threads
// call; ends with a barrier.  Returns the passes; a non-finite C gives NaN throughout.
template <bool CPLX, class Load, class Store>
__device__ int project(unsigned char* sm, int tid, Load load, Store store) {
  uint4* X = reinterpret_cast<uint4*>(sm);
  uint4* Z = reinterpret_cast<uint4*>(sm + Smem<CPLX>::matrix);  // X^2, then the polynomial in it
  unsigned char* red = sm + Smem<CPLX>::red;
  const int lane = tid & 31;
  int I, J;
  tri_index(4, tid >> 5, I, J);
  auto row = [&](int i) { return 16 * I + fx16::frag_row(i, lane); };
  auto col = [&](int i) { return 16 * J + fx16::frag_col(i, lane); };
  auto entry = [&](int i, double& re, double& im) {  // Hermitian throughout
    const int r = row(i), c = col(i);
    im = 0.0;
    if (r <= c) {
      load(r, c, re, im);
      if (r == c) im = 0.0;
    } else {
      load(c, r, re, im);
      im = -im;
    }
  };
  Frag hr, hi;
  // ||C||_F of the entries scaled by the largest one's binade: squares that neither overflow nor vanish
  int E = 0;
#pragma unroll 1
  for (int i = 0; i < 8; ++i) {
    double re, im;
    entry(i, re, im);
    E = max(E, fx16::exponent_field(re));
    if constexpr (CPLX) E = max(E, fx16::exponent_field(im));
  }
  E = reduce_max(E, red, tid);
  const bool finite = E != 0x7ff;
  const double unit = fxstep::binade_scale(E);
  double nrm = 0.0;
#pragma unroll 1
  for (int i = 0; i < 8; ++i) {
    double re, im;
    entry(i, re, im);
    re *= unit;
    im *= unit;
    nrm += (I == J ? 1.0 : 2.0) * fma(re, re, CPLX ? im * im : 0.0);
  }
  nrm = reduce_sum(nrm, red, tid);
  int pass = 0;
  if (finite && nrm > 0.0) {
    const double inv = (1.0 - 1e-9) * 9007199254740992.0 / sqrt(nrm);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      double re, im;
      entry(i, re, im);
      hr[i] = __double2ll_rn(re * unit * inv);
      if constexpr (CPLX) hi[i] = __double2ll_rn(im * unit * inv);
    }
    write_block<CPLX>(hr, hi, X, I, J, lane);
    __syncthreads();
    for (bool done = false; !done && pass < fxstep::kMaxPasses; ++pass) {
#pragma unroll 1
      for (int k = 0; k < fxstep::kSteps; ++k) {
        // X^2, units of 2^-56 -> 2^-53
        Frag yr, yi;
        product<CPLX>(X, X, I, J, yr, yi, lane);
        float res = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const bool diag = row(i) == col(i);
          yr[i] = (yr[i] + 4) >> 3;
          const float e = fx16::unit_float(diag ? (1LL << 53) - yr[i] : yr[i]);
          res = fmaf(e, e, res);
          if constexpr (CPLX) {
            yi[i] = diag ? 0 : (yi[i] + 4) >> 3;
            const float f = fx16::unit_float(yi[i]);
            res = fmaf(f, f, res);
          }
        }
        write_block<CPLX>(yr, yi, Z, I, J, lane);
        __syncthreads();
        if (k == fxstep::kSteps - 1) {
          done = reduce_sum((I == J ? 1.0 : 2.0) * (double)res, red, tid) <= fxstep::kResid;
        }
        // a I + b X^2 + c X^4, units of 2^-50
        product<CPLX>(Z, Z, I, J, hr, hi, lane);
        const fxstep::Coef q = kCoef[k];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          long long v = fxstep::scale((hr[i] + 4) >> 3, q.c) + fxstep::scale(yr[i], q.b);
          if (row(i) == col(i)) v += q.a;
          hr[i] = (v + 4) >> 3;
          if constexpr (CPLX) {
            v = fxstep::scale((hi[i] + 4) >> 3, q.c) + fxstep::scale(yi[i], q.b);
            hi[i] = row(i) == col(i) ? 0 : (v + 4) >> 3;
          }
        }
        __syncthreads();
        write_block<CPLX>(hr, hi, Z, I, J, lane);
        __syncthreads();
        product<CPLX>(X, Z, I, J, hr, hi, lane);
        if constexpr (CPLX) {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (row(i) == col(i)) hi[i] = 0;
        }
        __syncthreads();
        write_block<CPLX>(hr, hi, X, I, J, lane);
        __syncthreads();
      }
    }
    // Z = sign(C) C, all blocks (its rounding is not Hermitian), C scaled by its largest entry's binade:
    // units of 2^-3 times C's
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      double re, im;
      entry(i, re, im);
      hr[i] = fx16::fix(re, E);
      if constexpr (CPLX) hi[i] = fx16::fix(im, E);
    }
    write_block<CPLX>(hr, hi, Z, I, J, lane);
    __syncthreads();
    Frag tr, ti;
    product<CPLX>(X, Z, I, J, hr, hi, lane);
    if (I != J) product<CPLX>(X, Z, J, I, tr, ti, lane);
    int top = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (I == J) {
        tr[i] = hr[i];
        if constexpr (CPLX) ti[i] = hi[i];
      }
      unsigned long long m = (unsigned long long)(hr[i] ^ (hr[i] >> 63)) | (unsigned long long)(tr[i] ^ (tr[i] >> 63));
      if constexpr (CPLX)
        m |= (unsigned long long)(hi[i] ^ (hi[i] >> 63)) | (unsigned long long)(ti[i] ^ (ti[i] >> 63));
      top = max(top, 64 - __clzll((long long)m));
    }
    const int k = max(0, reduce_max(top, red, tid) - 53);  // digits hold 53 bits
    {
      Frag qr, qi;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        qr[i] = fx16::shift_round(hr[i], k);
        if constexpr (CPLX) qi[i] = fx16::shift_round(hi[i], k);
      }
      write_one<CPLX>(qr, qi, Z, I, J, lane);
      if (I != J) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          qr[i] = fx16::shift_round(tr[i], k);
          if constexpr (CPLX) qi[i] = fx16::shift_round(ti[i], k);
        }
        write_one<CPLX>(qr, qi, Z, J, I, lane);
      }
    }
    add_transpose(hr, tr, false);
    if constexpr (CPLX) add_transpose(hi, ti, true);
    __syncthreads();
    // C + Z + Z^H + Z sign(C), four times the result, in Z's units
    product<CPLX>(Z, X, I, J, tr, ti, lane);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      double re, im;
      entry(i, re, im);
      hr[i] += fx16::fix(re, E - 3) + fx16::shift_round(tr[i], 3 - k);
      if constexpr (CPLX) hi[i] += fx16::fix(im, E - 3) + fx16::shift_round(ti[i], 3 - k);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) hr[i] = hi[i] = 0;
  }
  const int e = E - 1075 - 53 + fx16::product_exp<6>() - 2;
  double re[8], im[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    re[i] = finite ? fx16::word(hr[i], e) : NAN;
    im[i] = !CPLX || row(i) == col(i) ? 0.0 : finite ? fx16::word(hi[i], e) : NAN;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = row(i), c = col(i);
    if (r <= c) store(r, c, re[i], im[i]);
    if (r < c) store(c, r, re[i], -im[i]);
  }
  __syncthreads();
  return pass;
}

}  // namespace fx64
}  // namespace ve
