// ve_fxsign.h -- PSD projection of a dense real symmetric matrix through its matrix sign, in
// fixed point on the tensor cores (ve_fxsign.cu; not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace ve {

struct FxSignCtl {
  double fro2;     // ||Y||_F^2, Y scaled by its largest entry's binade
  double resid;    // ||I - X^2||_F^2 before the last step; of a null part (fxsign_lmin) ||X^2||_F^2
  int done;        // the sign has converged (or Y is zero or not finite)
  int finite;
  unsigned long long side;  // the magnitudes of sign(Y) Y, or-ed
  int ey;          // exponent of Yq's unit
  int pad;
};

// Device workspace of one n x n projection (carved from caller memory).  The matrices are stored as
// digit fragments: 16 x 16 blocks (nb x nb of them), each 6 digits of 32 lanes x 16 bytes.
struct FxSignWs {
  int n = 0, nb = 0;
  uint4* X[2] = {nullptr, nullptr};  // the iterate (ping-pong)
  uint4* Y2 = nullptr;               // X^2
  uint4* B = nullptr;                // a I + b X^2 + c X^4; at the end sign(Y) Y
  uint4* Yq = nullptr;               // Y, scaled by its largest entry
  long long* y2 = nullptr;           // X^2 as integers (upper blocks, fragment order); at the end sign(Y) Y
  double* partial = nullptr;         // per-CTA norms, per-block residuals
  FxSignCtl* ctl = nullptr;          // two: of Y, and of its null part
  FxSignCtl* hctl = nullptr;         // pinned (allocated on first use)
  cudaGraphExec_t first = nullptr, again = nullptr;  // a whole projection; one more pass
  const double* Yd = nullptr;        // the matrices the graphs were captured for
  double* Xd = nullptr;
  int passes = 0;                    // of the last projection
  long launches = 0;
};

size_t fxsign_ws_bytes(int n);
int fxsign_ws_init(FxSignWs& w, int n, void* mem, size_t bytes);
void fxsign_ws_release(FxSignWs& w);
// X <- Pi_{>=0}((Y + Y^T) / 2) (device, n x n row-major, n even; X and Y distinct).  Issues
// everything on `s` and synchronises it once a pass (the convergence test is read on the host; up to 16
// rows there is none).  A non-finite Y gives NaN throughout.  Not to be called during stream capture.
cudaError_t fxsign_project(FxSignWs& w, const double* Y, double* X, cudaStream_t s);
// A lower bound on the smallest eigenvalue of (Y + Y^T) / 2 where that eigenvalue is zero to rounding, as
// after a projection: *lmin = -4 ||N Y N||_2 at most, N = (I - sign(Y)) / 2.  *found says whether it is
// within n 2^-53 ||Y||_F of the eigenvalue; where it is not (Y definite, or with an eigenvalue well below
// zero) the caller needs an eigensolve.  A non-finite Y gives NaN, found.  scratch: n x n, overwritten.
// Synchronises `s` once a pass.
cudaError_t fxsign_lmin(FxSignWs& w, const double* Y, double* scratch, cudaStream_t s, double* lmin, bool* found);

}  // namespace ve
