// ve_fxstep.cuh -- the matrix sign iteration of the fixed-point projections (ve_fxsign.cu for one
// dense matrix on the whole GPU, ve_fx64.cuh for a 64 x 64 matrix in one CTA): its steps and the
// integer helpers they share.
//
// Iteration.  X_0 = Y / ||Y||_F; X <- X (a I + b X^2 + c X^4): ten growth steps with odd quintics
// (kStep below) that map [l, 1] into [l', 1] with the largest possible l' (found by a linear
// program; the idea of Chen & Chow 2014's scaled Newton-Schulz iterations), from l = 3e-6 to 0.9841,
// then two Newton-Schulz steps of order three (15/8, -10/8, 3/8), the first centred on that
// interval.  The quintics are held to p(x) >= 0.3 x: one that maps a large eigenvalue to a tiny one
// (the unconstrained optimum sends 1 to l') turns the rounding of the former's eigenvector into a
// relative error of the latter (the stability condition of Nakatsukasa & Higham 2012).  Eigenvalues
// below 3e-6 ||Y||_F (rare; measured 1e-5 .. 1e-2 over the general solver's runs) show in
// ||I - X^2||_F and cost another pass, which starts from the grown X: three passes reach 2.7e-17
// ||Y||_F, below rounding.  An eigenvalue whose sign has not converged then contributes at most its
// own size.
#pragma once

#include <stdint.h>

#include "ve_fx16.cuh"

namespace ve {
namespace fxstep {

constexpr int kSteps = 12;
constexpr int kMaxPasses = 3;
constexpr double kResid = 1e-6;  // ||I - X^2||_F^2 before the last step: ||s| - 1| < 3e-10 after it

// x (a + b x^2 + c x^4) of the steps; the eleventh is the order-three Newton-Schulz step on x / m, m
// the middle of [0.98409, 0.999].  The growth steps stop at 0.999: their slope at 1 is ~10, so a
// quintic with p(1) = 1 would carry rounding above 1 out of its interval within a few steps.
struct Step {
  double a, b, c;
};
constexpr double kM = 0.9915432323472013;
constexpr Step kGrow = {4.0002895, -10.6185218, 7.6172323};
constexpr Step kStep[kSteps] = {
    kGrow, kGrow, kGrow, kGrow, kGrow, kGrow, kGrow, kGrow,
    {3.487584135, -7.220454778, 4.731870643}, {2.352196917, -2.408104863, 1.054907947},
    {1.875 / kM, -1.25 / (kM * kM * kM), 0.375 / (kM * kM * kM * kM * kM)},
    {1.875, -1.25, 0.375}};

// The step's coefficients as integers: a in units of 2^-53, b and c of 2^-56.
struct Coef {
  long long a, b, c;
};
constexpr Coef coef(int k) {
  return Coef{(long long)(kStep[k].a * 9007199254740992.0), (long long)(kStep[k].b * 72057594037927936.0),
              (long long)(kStep[k].c * 72057594037927936.0)};
}

// x c for |c| < 64 given in units of 2^-56, |x| < 2^55.
__device__ __forceinline__ long long scale(long long x, long long c) { return __mul64hi(x << 8, c); }

// The power of two that brings a number of exponent field E into [1, 4); a subnormal one (E = 0) to
// 2^-51 at least.  A product with it is exact.
__device__ __forceinline__ int binade_field(int E) { return E < 2045 ? 2046 - E : 1; }
__device__ __forceinline__ double binade_scale(int E) { return __hiloint2double(binade_field(E) << 20, 0); }

__device__ __forceinline__ uint32_t transpose8(uint32_t v) {
  uint32_t r;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}

}  // namespace fxstep
}  // namespace ve
