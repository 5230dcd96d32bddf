// ve_fxsign.cu -- the dense X step of Algorithm 5 (Khoo & Lindsey, arXiv:2106.02682, Sec. 3.2),
// X <- Pi_{>=0}(X - eps G) for one (N D) x (N D) matrix, as Pi(Y) = P Y P, P = (I + sign(Y)) / 2, with
// the matrix sign from a polynomial iteration: nothing but products, to float64 accuracy, on the tensor
// cores.
//
// Why.  The cyclic Jacobi it replaces is a chain of n - 1 dependent round launches a sweep (7.3 us
// each at n = 512, 6.8 sweeps warm: 27 ms of a 28 ms sweep), and its work is float64.  Here a
// projection is 38 products (of one of them all blocks), each one launch that fills the chip.
//
// P Y P and not P Y = (Y + sign(Y) Y) / 2, which takes two products less: an error d of the sign leaves
// d mu of a negative eigenvalue -mu in the latter, and Y has them up to hundreds of times ||X|| (eps G has
// one of the order of N).  Squared it vanishes.  Smallest eigenvalue of X after the first sweep, P Y and
// P Y P: n = 256 -1.6e-12 and -1.0e-15, n = 1024 -7.5e-11 and -3.8e-15 (by eigenvectors -1e-15); a sweep
// 787 and 816 us at n = 512, 249 at n = 160.
//
// Iteration: ve_fxstep.cuh.
//
// Products.  As in ve_fx16.cuh (integers as six base-512 float16 digits; planes s + t <= 6, whose
// error is 2^-56 of max|X| max|Y|), in 16 x 16 blocks stored as the A fragments of mma.sync
// m16n8k16: a product's output block comes back in that very layout, so each kernel writes the
// next one's operand digits itself.  32 terms of a plane sum stay below 2^24 (at most 6 x 32 x
// 256^2), after which the float32 sums go to int64.  All matrices of the iteration commute and are
// symmetric: only blocks on and above the diagonal are computed, the others are their transposes
// (movmatrix).  Of Z = sign(Y) Y, whose rounding is not symmetric, all blocks are.
// mma.sync rather than tcgen05: the digit planes s + t = q of one output accumulate in registers
// (seven planes x 128 columns would fill tensor memory with one 128 x 128 tile, and n = 160 .. 512
// has 2 .. 16 of those for 152 SMs).
#include "ve_fxsign.h"

#include "ve_fx16.cuh"
#include "ve_fxstep.cuh"

namespace ve {

namespace {

using fx16::Frag;
using fx16::kD;
using namespace fxstep;

constexpr int kBlk = kD * 32;   // uint4 of one 16 x 16 block
constexpr int kWarps = 8;       // warps of a product CTA
constexpr int kNormCtas = 128;
enum Mode { kSquare, kSquareLast, kPoly, kMul, kSide, kFinal };

struct Args {
  int n, nb;
  const uint4* A;
  const uint4* B;
  uint4* out;
  long long* y2;
  long long a, b, c;    // kPoly: the step's coefficients
  double* partial;      // kSquareLast: per-block residuals
  FxSignCtl* ctl;
  const double* Yd;
  double* Xd;
  int sg;               // kFinal: 1 for P Y P, -1 for (I - P) Y (I - P)
};

// Digits of the integers z as block (I, J), and transposed as block (J, I).  Of a diagonal block the
// upper triangle counts: the iteration takes every matrix for exactly symmetric, and would grow an
// antisymmetric rounding error by its growth factor at every step.
__device__ __forceinline__ void write_block(const Frag& z, uint4* out, int nb, int I, int J, int lane) {
  uint32_t d[kD][4];
  fx16::digits<kD>(z, d);
  uint4* o = out + ((size_t)I * nb + J) * kBlk + lane;
  uint4* t = out + ((size_t)J * nb + I) * kBlk + lane;
  // of a lane's two entries (row, 2 t), (row, 2 t + 1) of an 8 x 8 tile, those below the diagonal
  const int row = lane >> 2, col = 2 * (lane & 3);
  const uint32_t below = (col < row ? 0xffffu : 0u) | (col + 1 < row ? 0xffff0000u : 0u);
#pragma unroll
  for (int s = 0; s < kD; ++s) {
    const uint4 v = make_uint4(d[s][0], d[s][1], d[s][2], d[s][3]);
    const uint4 w = make_uint4(transpose8(v.x), transpose8(v.z), transpose8(v.y), transpose8(v.w));
    if (I == J) {
      o[s * 32] = make_uint4((v.x & ~below) | (w.x & below), w.y, v.z, (v.w & ~below) | (w.w & below));
    } else {
      o[s * 32] = v;
      t[s * 32] = w;
    }
  }
}

// Each kernel of the chain lets the next one's CTAs start beside it (they wait here until it has
// finished and its writes are visible, before their first access to global memory).  Every kernel
// waits here, so whatever is two launches back has finished as well.  Measured a sweep, without / with:
// n = 512 810 / 783 us, n = 160 252 / 248 us.
__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The bits that Z has above 2^53 (bits: all of its entries' magnitudes, or-ed).
__device__ __forceinline__ int side_shift(unsigned long long bits) { return max(0, 11 - __clzll((long long)bits)); }

// One product.  A CTA holds TB x TB output blocks of 16 x 16 (blocks TB bi .., TB bj .., bi <= bj),
// KW warps a block sharing its K range.
template <int MODE, int TB>
__global__ void __launch_bounds__(32 * kWarps, 1) k_fx_product(const Args p) {
  constexpr int KW = kWarps / (TB * TB);
  __shared__ long long sum[TB * TB][KW > 1 ? KW - 1 : 1][8][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int blk = warp / KW, kw = warp % KW;
  // tile (bi, bj), row by row: of the upper triangle, or (kSide) of all
  const int T = (p.nb + TB - 1) / TB;
  int bi = blockIdx.x / T, bj = blockIdx.x % T;
  if constexpr (MODE != kSide) tri_index(T, blockIdx.x, bi, bj);
  const int I = bi * TB + blk / TB, J = bj * TB + blk % TB;
  after_previous();
  const bool live = (MODE == kSide ? I < p.nb : I <= J) && J < p.nb;
  Frag h = {};
  if (live) {
    const uint4* a = p.A + (size_t)I * p.nb * kBlk + lane;
    const uint4* b = p.B + (size_t)J * p.nb * kBlk + lane;
    const int per = ((p.nb + KW - 1) / KW + 1) & ~1;  // even: the sums are emptied every 2 steps
    const int k0 = kw * per, k1 = min(p.nb, k0 + per);
    float acc[2][7][4] = {};
    uint4 an[kD], bn[kD];
    if (k0 < k1) {
#pragma unroll
      for (int s = 0; s < kD; ++s) {
        an[s] = a[(size_t)k0 * kBlk + s * 32];
        bn[s] = b[(size_t)k0 * kBlk + s * 32];
      }
    }
    for (int k = k0; k < k1; ++k) {
      uint32_t l[kD][4];
      uint4 r[kD];
#pragma unroll
      for (int s = 0; s < kD; ++s) {
        l[s][0] = an[s].x;
        l[s][1] = an[s].y;
        l[s][2] = an[s].z;
        l[s][3] = an[s].w;
        r[s] = bn[s];
      }
      if (k + 1 < k1) {
#pragma unroll
        for (int s = 0; s < kD; ++s) {
          an[s] = a[(size_t)(k + 1) * kBlk + s * 32];
          bn[s] = b[(size_t)(k + 1) * kBlk + s * 32];
        }
      }
#pragma unroll
      for (int t = 0; t < kD; ++t)
#pragma unroll
        for (int s = 0; s < kD; ++s)
          if (s + t <= 6) {
            fx16::mma(acc[0][s + t], l[s], r[t].x, r[t].z);
            fx16::mma(acc[1][s + t], l[s], r[t].y, r[t].w);
          }
      if (((k - k0) & 1) || k + 1 == k1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          h[i] += fx16::combine<6>(acc[0], i);
          h[4 + i] += fx16::combine<6>(acc[1], i);
        }
#pragma unroll
        for (int q = 0; q < 7; ++q)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[0][q][i] = acc[1][q][i] = 0.f;
      }
    }
  }
  if constexpr (KW > 1) {
    if (kw > 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) sum[blk][kw - 1][i][lane] = h[i];
    }
    __syncthreads();
    if (kw > 0) return;
#pragma unroll
    for (int w = 0; w < KW - 1; ++w)
#pragma unroll
      for (int i = 0; i < 8; ++i) h[i] += sum[blk][w][i][lane];
  }
  if (!live) return;
  // h: the product in units of 2^50 times the operands' (X, X^2: 2^-53; B: 2^-50)
  if constexpr (MODE == kSquare || MODE == kSquareLast) {
    long long* y2 = p.y2 + ((size_t)I * p.nb + J) * 256 + lane;
    float res = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      h[i] = (h[i] + 4) >> 3;
      y2[i * 32] = h[i];
      if constexpr (MODE == kSquareLast) {
        const int row = fx16::frag_row(i, lane), col = fx16::frag_col(i, lane);
        const bool diag = I == J && row == col;
        float e = fx16::unit_float(diag ? (1LL << 53) - h[i] : h[i]);
        if (diag && 16 * I + row >= p.n) e = 0.f;  // padding
        res = fmaf(e, e, res);
      }
    }
    write_block(h, p.out, p.nb, I, J, lane);
    if constexpr (MODE == kSquareLast) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) res += shfl_xor(res, o);
      if (lane == 0) p.partial[(size_t)I * p.nb + J] = (I == J ? 1.0 : 2.0) * (double)res;
    }
  } else if constexpr (MODE == kPoly) {
    const long long* y2 = p.y2 + ((size_t)I * p.nb + J) * 256 + lane;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      long long v = scale((h[i] + 4) >> 3, p.c) + scale(y2[i * 32], p.b);
      if (I == J && fx16::frag_row(i, lane) == fx16::frag_col(i, lane)) v += p.a;
      h[i] = (v + 4) >> 3;  // |B| < 8: units of 2^-50
    }
    write_block(h, p.out, p.nb, I, J, lane);
  } else if constexpr (MODE == kMul) {
    write_block(h, p.out, p.nb, I, J, lane);
  } else if constexpr (MODE == kSide) {
    // Z, in units of 2^-3 times Yq's; its top bit scales the digits (k_fx_side)
    long long* z = p.y2 + ((size_t)I * p.nb + J) * 256 + lane;
    unsigned long long m = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      z[i * 32] = h[i];
      m |= (unsigned long long)(h[i] ^ (h[i] >> 63));
    }
    const unsigned hi = __reduce_or_sync(0xffffffffu, (unsigned)(m >> 32));
    const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)m);
    if (lane == 0) atomicOr(&p.ctl->side, (unsigned long long)hi << 32 | lo);
  } else {
    // X = (Y +- (Z + Z^T) + Z sign(Y)) / 4, added as integers in Z's unit (h: 2^(shift - 3) of it)
    const int E = p.ctl->ey + 1075, e = p.ctl->ey - 3, up = side_shift(p.ctl->side) - 3;
    const bool finite = p.ctl->finite != 0;
    const long long* z = p.y2 + ((size_t)I * p.nb + J) * 256;
    const long long* zt = p.y2 + ((size_t)J * p.nb + I) * 256;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = fx16::frag_row(i, lane), c = fx16::frag_col(i, lane);
      const int row = 16 * I + r, col = 16 * J + c;
      if (row <= col && col < p.n) {
        const double y = 0.5 * (p.Yd[(size_t)row * p.n + col] + p.Yd[(size_t)col * p.n + row]);
        const long long t = zt[((r & 1) + 2 * (c >> 3) + 4 * (r >> 3)) * 32 + (c & 7) * 4 + ((r & 7) >> 1)];
        const long long x = fx16::fix(y, E - 3) + p.sg * (z[i * 32 + lane] + t) + fx16::shift_round(h[i], -up);
        const double v = finite ? fx16::word(x, e - 2) : NAN;
        p.Xd[(size_t)row * p.n + col] = v;
        p.Xd[(size_t)col * p.n + row] = v;
      }
    }
  }
}

// Z as digits (block (I, J) in its own place, one warp a block).
__global__ void __launch_bounds__(256) k_fx_side(const long long* __restrict__ y2, int nb, uint4* out,
                                                 const FxSignCtl* ctl) {
  const int lane = threadIdx.x & 31;
  after_previous();
  const int w = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (w >= nb * nb) return;
  const int k = side_shift(ctl->side);
  Frag z;
#pragma unroll
  for (int i = 0; i < 8; ++i) z[i] = fx16::shift_round(y2[(size_t)w * 256 + i * 32 + lane], k);
  uint32_t d[kD][4];
  fx16::digits<kD>(z, d);
#pragma unroll
  for (int s = 0; s < kD; ++s)
    out[(size_t)w * kBlk + s * 32 + lane] = make_uint4(d[s][0], d[s][1], d[s][2], d[s][3]);
}

// Per-CTA largest entries of Y, and sums of squares of the entries scaled by the CTA's largest one's
// binade: in one pass (the power of two applied to the sum) where the squares stay in range, else in two.
__global__ void __launch_bounds__(256) k_fx_norm(const double* __restrict__ Y, int n, double* partial) {
  __shared__ double red[8];
  const size_t nn = (size_t)n * n;
  double v = 0.0, m = 0.0;
  for (size_t e = blockIdx.x * (size_t)256 + threadIdx.x; e < nn; e += (size_t)gridDim.x * 256) {
    v = fma(Y[e], Y[e], v);
    m = fmax(m, fabs(Y[e]));
  }
  m = -gmin<256>(-m, red);
  const int E = fx16::exponent_field(m);
  const double unit = binade_scale(E);
  if (E > 623 && E < 1423) {
    v = v * unit * unit;
  } else {
    v = 0.0;
    for (size_t e = blockIdx.x * (size_t)256 + threadIdx.x; e < nn; e += (size_t)gridDim.x * 256)
      v = fma(Y[e] * unit, Y[e] * unit, v);
  }
  v = gsum<256>(v, red);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = v;
    partial[kNormCtas + blockIdx.x] = m;
  }
}

// X_0 = Y / ||Y||_F and Y scaled by its largest entry, as digits; one warp a block on or above the
// diagonal.  Every warp adds the norms up itself, in one order.
__global__ void __launch_bounds__(256) k_fx_slice(const double* __restrict__ Y, int n, int nb, const double* partial,
                                                  uint4* X, uint4* Yq, FxSignCtl* ctl) {
  const int lane = threadIdx.x & 31;
  after_previous();
  double v = 0.0, m = 0.0;
  for (int k = lane; k < kNormCtas; k += 32) m = fmax(m, partial[kNormCtas + k]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, shfl_xor(m, o));
  const int E = fx16::exponent_field(m);  // Yq: an entry of the largest one's binade is 2^52 .. 2^53
  for (int k = lane; k < kNormCtas; k += 32) {  // from the CTA's scale to the matrix's
    const int d = binade_field(E) - binade_field(fx16::exponent_field(partial[kNormCtas + k]));  // <= 0
    const double c = d > -1023 ? __hiloint2double((1023 + d) << 20, 0) : 0.0;
    v += partial[k] * c * c;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += shfl_xor(v, o);
  const bool finite = isfinite(v) != 0;
  const double unit = binade_scale(E);
  const double inv = finite && v > 0.0 ? (1.0 - 1e-9) * 9007199254740992.0 / sqrt(v) : 0.0;
  const long w = (long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (w == 0 && lane == 0) {
    ctl->fro2 = v;
    ctl->finite = finite ? 1 : 0;
    ctl->side = 0;
    ctl->ey = E - 1075;
  }
  if (w >= (long)nb * (nb + 1) / 2) return;
  int I, J;
  tri_index(nb, (int)w, I, J);
  Frag x, q;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = 16 * I + fx16::frag_row(i, lane), col = 16 * J + fx16::frag_col(i, lane);
    double y = 0.0;
    if (finite && row < n && col < n) y = 0.5 * (Y[(size_t)row * n + col] + Y[(size_t)col * n + row]);
    x[i] = __double2ll_rn(y * unit * inv);
    q[i] = fx16::fix(y, E);
  }
  write_block(x, X, nb, I, J, lane);
  write_block(q, Yq, nb, I, J, lane);
}

// The convergence test: block residuals added in a fixed order.
__global__ void __launch_bounds__(256) k_fx_check(const double* partial, int nb, FxSignCtl* ctl) {
  __shared__ double red[8];
  after_previous();
  double v = 0.0;
  for (int e = threadIdx.x; e < nb * nb; e += 256)
    if (e / nb <= e % nb) v += partial[e];
  v = gsum<256>(v, red);
  if (threadIdx.x == 0) {
    ctl->resid = v;
    ctl->side = 0;  // for the next pass
    ctl->done = v <= kResid || ctl->fro2 == 0.0 || !ctl->finite;
  }
}

// ||X^2||_F^2 of the integers of X^2 (upper blocks), in a fixed order.
__global__ void __launch_bounds__(1024) k_fx_fro(const long long* __restrict__ y2, int nb, FxSignCtl* ctl) {
  __shared__ double red[32];
  after_previous();
  double v = 0.0;
  for (int b = threadIdx.x >> 8; b < nb * nb; b += 4) {
    const int I = b / nb, J = b % nb;
    if (I > J) continue;
    const double x = (double)y2[(size_t)b * 256 + (threadIdx.x & 255)] * 1.1102230246251565e-16;
    v = fma(I == J ? x : 2.0 * x, x, v);
  }
  v = gsum<1024>(v, red);
  if (threadIdx.x == 0) ctl->resid = v;
}

// A matrix of up to 16 rows by one warp (ve_fx16.cuh, from V = I; rows past n decoupled, with the largest
// entry on their diagonal, which is no smaller than its lowest eigenvalue): its projection into X, or (X
// null) its smallest eigenvalue into ctl->resid.
__global__ void __launch_bounds__(32) k_fx_small(const double* __restrict__ Y, int n, double* X, FxSignCtl* ctl) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x;
  double c[8], m = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = fx16::frag_row(i, lane), col = fx16::frag_col(i, lane);
    c[i] = row < n && col < n ? 0.5 * (Y[row * n + col] + Y[col * n + row]) : 0.0;
    m = fmax(m, fabs(c[i]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, shfl_xor(m, o));
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (fx16::frag_row(i, lane) == fx16::frag_col(i, lane) && fx16::frag_row(i, lane) >= n) c[i] = m;
  Frag q, none;
  int e = 0;
  const bool finite = fx16::fix_matrix<false>(c, c, q, none, e);
  if (!X) {
    const double v = finite ? fx16::lowest<false>(q, none, e, smem_raw, lane) : NAN;
    if (lane == 0) ctl->resid = v;
    return;
  }
  fx16::Result res = fx16::kProduct;
  if (finite) {
    bool dk;
    int nsw;
    long long* v = reinterpret_cast<long long*>(smem_raw + fx16::Smem<false>::bytes);
    res = fx16::project<false>(q, none, e, v, false, smem_raw, lane, &dk, &nsw);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = fx16::frag_row(i, lane), col = fx16::frag_col(i, lane);
    if (row < n && col < n)
      X[row * n + col] = !finite                  ? NAN
                         : res == fx16::kProduct ? fx16::word(q[i], e)
                         : res == fx16::kSame    ? c[i]
                                                 : 0.0;
  }
}

// n <= 16.  One launch and no test on the host, for 42 launches and a copy: a general sweep at n = 8 79 to
// 106 us and not 157 (eigensolve over the whole GPU: 122 to 188), at n = 16 96 to 104 and not 159.
cudaError_t small(const double* Y, int n, double* X, FxSignCtl* ctl, cudaStream_t s) {
  k_fx_small<<<1, 32, fx16::Smem<false>::bytes + fx16::Smem<false>::vectors, s>>>(Y, n, X, ctl);
  return cudaGetLastError();
}

// A launch that need not wait for the one before it on the stream to finish (after_previous).
template <class... P, class... A>
cudaError_t launch_after(void (*f)(P...), int grid, int threads, cudaStream_t s, A... args) {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)grid);
  c.blockDim = dim3((unsigned)threads);
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, f, P(args)...);
}

// 32 x 32 tiles where they fill the chip; else one block a CTA with its K range shared by all the
// warps (n = 160: 55 CTAs instead of 15).
template <int MODE>
cudaError_t launch(const Args& a, cudaStream_t s) {
  const int T = (a.nb + 1) / 2, nb = a.nb;
  auto tiles = [](int t) { return MODE == kSide ? t * t : t * (t + 1) / 2; };
  if (T * (T + 1) / 2 >= 100) return launch_after(k_fx_product<MODE, 2>, tiles(T), 32 * kWarps, s, a);
  return launch_after(k_fx_product<MODE, 1>, tiles(nb), 32 * kWarps, s, a);
}

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// One pass from X[0] to X[0] (kSteps is even), the final products and the test.
cudaError_t issue_pass(FxSignWs& w, const double* Y, double* X, int sg, cudaStream_t s) {
  Args a;
  a.sg = sg;
  a.n = w.n;
  a.nb = w.nb;
  a.y2 = w.y2;
  a.partial = w.partial + 2 * kNormCtas;
  a.ctl = w.ctl;
  a.Yd = Y;
  a.Xd = X;
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < kSteps && e == cudaSuccess; ++k) {
    a.A = a.B = w.X[k & 1];
    a.out = w.Y2;
    e = k == kSteps - 1 ? launch<kSquareLast>(a, s) : launch<kSquare>(a, s);
    if (e != cudaSuccess) return e;
    a.A = a.B = w.Y2;
    a.out = w.B;
    a.a = coef(k).a;
    a.b = coef(k).b;
    a.c = coef(k).c;
    if ((e = launch<kPoly>(a, s)) != cudaSuccess) return e;
    a.A = w.X[k & 1];
    a.B = w.B;
    a.out = w.X[(k + 1) & 1];
    e = launch<kMul>(a, s);
  }
  if (e != cudaSuccess) return e;
  a.A = w.X[0];
  a.B = w.Yq;
  if ((e = launch<kSide>(a, s)) != cudaSuccess) return e;
  if ((e = launch_after(k_fx_side, (w.nb * w.nb + 7) / 8, 256, s, w.y2, w.nb, w.B, w.ctl)) != cudaSuccess) return e;
  a.A = w.B;
  a.B = w.X[0];
  if ((e = launch<kFinal>(a, s)) != cudaSuccess) return e;
  return launch_after(k_fx_check, 1, 256, s, a.partial, w.nb, w.ctl);
}

cudaError_t build_graph(FxSignWs& w, const double* Y, double* X, bool first, cudaGraphExec_t* out) {
  cudaStream_t cs = nullptr;
  cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
  if (e != cudaSuccess) return e;
  e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    if (first) {
      k_fx_norm<<<kNormCtas, 256, 0, cs>>>(Y, w.n, w.partial);
      const int blocks = w.nb * (w.nb + 1) / 2;
      e = cudaGetLastError();
      if (e == cudaSuccess)
        e = launch_after(k_fx_slice, (blocks + 7) / 8, 256, cs, Y, w.n, w.nb, w.partial, w.X[0], w.Yq, w.ctl);
    }
    if (e == cudaSuccess) e = issue_pass(w, Y, X, 1, cs);
    cudaGraph_t g = nullptr;
    const cudaError_t e2 = cudaStreamEndCapture(cs, &g);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(out, g, 0);
    if (g) cudaGraphDestroy(g);
  }
  cudaStreamDestroy(cs);
  return e;
}

cudaError_t host_ctl(FxSignWs& w) {
  return w.hctl ? cudaSuccess : cudaMallocHost((void**)&w.hctl, 2 * sizeof(FxSignCtl));
}

// The root of a scaled sum of squares (FxSignCtl::fro2).
double unscaled(double sum, int ey) {
  const int E = ey + 1075;
  return ldexp(sqrt(sum), E < 2045 ? E - 1023 : 1022);
}

}  // namespace

size_t fxsign_ws_bytes(int n) {
  if (n < 2 || (n & 1)) return 0;
  const size_t nb = (n + 15) / 16;
  return 5 * al256(nb * nb * kBlk * sizeof(uint4)) + al256(nb * nb * 256 * sizeof(long long)) +
         al256((2 * kNormCtas + nb * nb) * sizeof(double)) + al256(2 * sizeof(FxSignCtl));
}

int fxsign_ws_init(FxSignWs& w, int n, void* mem, size_t bytes) {
  const size_t need = fxsign_ws_bytes(n);
  if (need == 0 || !mem || bytes < need || ((uintptr_t)mem & 255)) return -1;
  w = FxSignWs();
  w.n = n;
  w.nb = (n + 15) / 16;
  unsigned char* p = (unsigned char*)mem;
  const size_t nb2 = (size_t)w.nb * w.nb;
  uint4** bufs[5] = {&w.X[0], &w.X[1], &w.Y2, &w.B, &w.Yq};
  for (auto b : bufs) {
    *b = (uint4*)p;
    p += al256(nb2 * kBlk * sizeof(uint4));
  }
  w.y2 = (long long*)p;
  p += al256(nb2 * 256 * sizeof(long long));
  w.partial = (double*)p;
  p += al256((2 * kNormCtas + nb2) * sizeof(double));
  w.ctl = (FxSignCtl*)p;
  return 0;
}

void fxsign_ws_release(FxSignWs& w) {
  if (w.first) cudaGraphExecDestroy(w.first);
  if (w.again) cudaGraphExecDestroy(w.again);
  if (w.hctl) cudaFreeHost(w.hctl);
  w.first = w.again = nullptr;
  w.hctl = nullptr;
}

cudaError_t fxsign_project(FxSignWs& w, const double* Y, double* X, cudaStream_t s) {
  if (w.n <= 16) {
    w.passes = 1;
    w.launches += 1;
    return small(Y, w.n, X, w.ctl, s);
  }
  cudaError_t e;
  if ((e = host_ctl(w)) != cudaSuccess) return e;
  if (w.first && (w.Yd != Y || w.Xd != X)) {
    cudaGraphExecDestroy(w.first);
    if (w.again) cudaGraphExecDestroy(w.again);
    w.first = w.again = nullptr;
  }
  if (!w.first) {
    if ((e = build_graph(w, Y, X, true, &w.first)) != cudaSuccess) return e;
    w.Yd = Y;
    w.Xd = X;
  }
  for (w.passes = 1;; ++w.passes) {
    if (w.passes > 1 && !w.again && (e = build_graph(w, Y, X, false, &w.again)) != cudaSuccess) return e;
    if ((e = cudaGraphLaunch(w.passes == 1 ? w.first : w.again, s)) != cudaSuccess) return e;
    w.launches += 3 * kSteps + 4 + (w.passes == 1 ? 2 : 0);
    if ((e = cudaMemcpyAsync(w.hctl, w.ctl, sizeof(FxSignCtl), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    if (w.hctl->done || w.passes == kMaxPasses) return cudaSuccess;
  }
}

// M = N Y N, N = (I - sign(Y)) / 2, is zero but for rounding and the eigenvalues whose sign is not
// resolved (s near 0: M has a quarter of them) or is negative (all of them), so lmin(Y) >= -4 ||M||_2 up to
// rounding; ||M||_2 <= ||M^2||_F^(1/2), four to five times less than ||M||_F where M is rounding.  One
// pass is enough where Y has no eigenvalue between rounding and 3e-6 ||Y||_F.  An unresolved sign
// (||I - S^2||_F^2 >= 1/2) and a small bound say that lmin(Y) is zero to rounding.
// Measured, a general bound after 60 sweeps (eigensolve of X warm from the X step's own eigenvectors / from
// the last bound's / here): n = 24 767 / 1198 / 228 us, n = 160 3.4 / 8.6 / 0.45 ms, n = 512 8.7 / 60 /
// 1.26 ms, n = 1024 42 / 309 / 6.5 ms; the bounds -1.1e-14 / -1.5e-12 / -1.1e-14 at n = 512.
cudaError_t fxsign_lmin(FxSignWs& w, const double* Y, double* scratch, cudaStream_t s, double* lmin, bool* found) {
  cudaError_t e;
  if ((e = host_ctl(w)) != cudaSuccess) return e;
  FxSignCtl* h = w.hctl;
  auto read = [&]() {
    const cudaError_t r = cudaMemcpyAsync(h, w.ctl, 2 * sizeof(FxSignCtl), cudaMemcpyDeviceToHost, s);
    return r != cudaSuccess ? r : cudaStreamSynchronize(s);
  };
  *found = true;
  if (w.n <= 16) {  // by eigenvalues: one launch, not 47 (a bound at n = 8: 105 to 145 us)
    if ((e = small(Y, w.n, nullptr, w.ctl, s)) != cudaSuccess || (e = read()) != cudaSuccess) return e;
    *lmin = h[0].resid;
    return cudaSuccess;
  }
  const int slices = (w.nb * (w.nb + 1) / 2 + 7) / 8;
  auto slice = [&](const double* from, uint4* x, uint4* q, FxSignCtl* ctl) {
    k_fx_norm<<<kNormCtas, 256, 0, s>>>(from, w.n, w.partial);
    const cudaError_t r = cudaGetLastError();
    return r != cudaSuccess ? r : launch_after(k_fx_slice, slices, 256, s, from, w.n, w.nb, w.partial, x, q, ctl);
  };
  if ((e = slice(Y, w.X[0], w.Yq, w.ctl)) != cudaSuccess) return e;
  for (int pass = 1;; ++pass) {
    if ((e = issue_pass(w, Y, scratch, -1, s)) != cudaSuccess) return e;
    if ((e = slice(scratch, w.Y2, w.B, w.ctl + 1)) != cudaSuccess) return e;
    Args a = {};
    a.n = w.n;
    a.nb = w.nb;
    a.A = a.B = w.Y2;
    a.out = w.B;
    a.y2 = w.y2;
    if ((e = launch<kSquare>(a, s)) != cudaSuccess) return e;
    if ((e = launch_after(k_fx_fro, 1, 1024, s, w.y2, w.nb, w.ctl + 1)) != cudaSuccess) return e;
    if ((e = read()) != cudaSuccess) return e;
    if (!h[0].finite) {
      *lmin = NAN;
      return cudaSuccess;
    }
    const double b = 4.0001 * unscaled(h[1].fro2 * sqrt(h[1].resid), h[1].ey);
    if (h[0].resid >= 0.5 && b <= w.n * 1.1102230246251565e-16 * unscaled(h[0].fro2, h[0].ey)) {
      *lmin = 0.0 - b;
      return cudaSuccess;
    }
    if (h[0].done || pass == kMaxPasses) {
      *found = false;
      return cudaSuccess;
    }
  }
}

}  // namespace ve
