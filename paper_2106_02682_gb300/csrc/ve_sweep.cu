// ve_sweep.cu -- the pair pass and the small reductions of one sweep of Algorithm 6
// (Khoo & Lindsey, arXiv:2106.02682, Sec. 3.3).
//
// k_pair     : one thread group per pair offset delta != 0.  Fuses the effective pair
//              Hamiltonian (Eq. (effHam)), the closed-form pair update (Eq. (rhoijUpdate)),
//              the PSD projection (Eq. (rhoijTildeUpdate)), the Lambda update, the X' = X - eps G
//              step for the block (Algorithm 6), the partial traces A1 rho, A2 rho and the
//              per-delta terms of Eq. (feasErr) and of the energy.
//              The offsets delta and -delta describe the same pairs of clusters seen from
//              either end, and the update commutes with exchanging the two clusters (S): from a
//              state with rho~_{-delta} = S rho~_delta S, Lambda likewise, Lambda1_{-delta} =
//              Lambda2_delta and X_{0,-delta} = X_{0,delta}^T, the -delta results are the swap
//              images of the delta ones.  So one group updates the canonical member of each
//              pair {delta, -delta} and writes the images for the other: half the eigensolves.
// k_rho0     : rho_0 update (Eq. (rhoiUpdate), translation-invariant form) with the trace
//              shift, and X'_00 = X_00 - eps G_00[rho_0]: every CTA sums a chunk of offsets, the
//              last CTA to finish adds the chunk sums and updates rho_0.
// k_dual_status : Lambda1/Lambda2 updates (they need the new rho_0); energy per spin, Eq. (feasErr),
//              |energy change|, residual (CTA sums, then the last CTA).
// All reductions run in a fixed order, so a sweep is bitwise reproducible.
#include "ve_device.cuh"
#include "ve_fx16.cuh"
#include "ve_fx64.cuh"
#include "ve_internal.h"

namespace ve {

namespace {

// D = 64 in float64 and double-float (one code for both): the projection in fixed point on the tensor
// cores (ve_fx64.cuh), by ten warps.
template <int D, typename T>
constexpr bool FX64 = D == 64 && std::is_same<T, double>::value;

template <int D, typename T>
struct PairShape {
  static constexpr int m = ClusterDim<D>::m;
  static constexpr int NT = FX64<D, T> ? fx64::kThreads : group_threads<D, T>();
  static constexpr int LD = GroupShape<D>::LD;
  static constexpr int GPC = GroupShape<D>::GPC;  // groups per CTA
};

template <int D, typename T>
struct PairSmem {
  static constexpr int m = PairShape<D, T>::m, LD = PairShape<D, T>::LD;
  static constexpr size_t al(size_t x) { return ((x + 15) / 16) * 16; }
  // per group, in bytes; every array 16-byte aligned
  static constexpr size_t R = 0;                                   // T D*D  (rhs, then rho)
  static constexpr size_t Xs = R + al(sizeof(T) * D * D);          // T D*D  (X_{0,delta})
  static constexpr size_t A = Xs + al(sizeof(T) * D * D);          // T D*LD
  static constexpr size_t V = A + al(sizeof(T) * D * LD);          // T D*LD, or fx64::Smem
  static constexpr size_t WT = V + (FX64<D, T> ? al(fx64::Smem<false>::bytes) : al(sizeof(T) * D * LD));  // T D*LD
  static constexpr size_t CS = WT + (FX64<D, T> ? 0 : al(sizeof(T) * D * LD));  // T D
  static constexpr size_t W = CS + al(sizeof(T) * D);              // T D
  static constexpr size_t TR = W + al(sizeof(T) * D);              // T 2*m*m + 2
  static constexpr size_t RED = TR + al(sizeof(T) * (2 * m * m + 2));
  static constexpr size_t bytes = RED + al(sizeof(T) * 32);
};

// Arithmetic in T (double, or float in the mixed-precision sweep); the state stays float64.
template <int D, typename T>
__global__ void __launch_bounds__(PairShape<D, T>::NT * PairShape<D, T>::GPC, D == 64 ? 1 : GroupShape<D>::MINB)
    k_pair(const PairArgs a) {
  constexpr int m = PairShape<D, T>::m, NT = PairShape<D, T>::NT, LD = PairShape<D, T>::LD;
  constexpr int GPC = PairShape<D, T>::GPC;
  // register-tiled warp products (rgemm16) in float32 only: they compute whole 16 x 16 results
  // where the loops below compute triangles, and float64 / double-float issue is the bound there
  constexpr bool TILE16 = D == 16 && NT == 32 && std::is_same<T, float>::value;
  using S = PairSmem<D, T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int g = threadIdx.x / NT, tid = threadIdx.x % NT;
  unsigned char* base = GroupShape<D>::GLOBAL ? a.gws + (size_t)blockIdx.x * S::bytes
                                              : smem_raw + (size_t)g * S::bytes;
  T* R = reinterpret_cast<T*>(base + S::R);
  T* Xs = reinterpret_cast<T*>(base + S::Xs);
  T* A = reinterpret_cast<T*>(base + S::A);
  T* V = reinterpret_cast<T*>(base + S::V);
  T* Wt = reinterpret_cast<T*>(base + S::WT);
  T* cs = reinterpret_cast<T*>(base + S::CS);
  T* W = reinterpret_cast<T*>(base + S::W);
  T* t1 = reinterpret_cast<T*>(base + S::TR);
  T* t2 = t1 + m * m;
  T* red = reinterpret_cast<T*>(base + S::RED);

  const T mu = (T)a.mu, nu = (T)a.nu, eps = (T)a.eps;
  T c0, c1, c2;
  if constexpr (std::is_same<T, double>::value) {
    c0 = a.k.c0;
    c1 = a.k.c1;
    c2 = a.k.c2;
  } else {
    const T alpha = nu * m;
    c0 = T(1) / mu;
    c1 = T(1) / (mu + alpha);
    c2 = T(1) / (mu + T(2) * alpha);
  }
  const T imu = c0;

  for (long it = (long)blockIdx.x * GPC + g; it < a.Pc; it += (long)gridDim.x * GPC) {
    const long p = a.pidx ? a.pidx[it] : it;
    const long pm = a.pidx ? a.pmir[it] : -1;  // pair index of -delta, or -1
    const long dl = p + 1;  // linear cluster offset delta
    const double* rt = a.rt + p * D * D;
    const double* lam = a.lam + p * D * D;
    const double* l1 = a.lam1 + p * m * m;
    const double* l2 = a.lam2 + p * m * m;
    double* Xb = a.X + dl * D * D;
    const int hs = a.hslot[dl];
    const double* Hb = hs >= 0 ? a.hb + (long)hs * D * D : nullptr;

    for (int e = tid; e < D * D; e += NT) Xs[e] = (T)Xb[e];
    if (pm >= 0) {
      // the multipliers of -delta as images of these, before the rho_0 reduction reads them
      for (int idx = tid; idx < m * m; idx += NT) {
        a.lam1[pm * m * m + idx] = l2[idx];
        a.lam2[pm * m * m + idx] = l1[idx];
      }
    }
    gsync<NT>();
    // right-hand side of Eq. (rhoijUpdate) with H' of Eq. (effHam)
    for (int e = tid; e < D * D; e += NT) {
      const int i = e / D, j = e % D;
      const int pa = i / m, pb = i % m, pc = j / m, pd = j % m;
      const T h = Hb ? (T)Hb[e] : T(0);
      // (R^* X)_{(a,b),(c,d)} = X_{(a,c),(d,b)} and its transpose X_{(c,a),(b,d)}
      const T hp = h - Xs[(pa * m + pc) * D + (pd * m + pb)] - Xs[(pc * m + pa) * D + (pb * m + pd)];
      T y = mu * (T)rt[e] + (T)lam[e] - hp;
      if (pb == pd) y += nu * (T)a.rho0[pa * m + pc] - (T)l1[pa * m + pc];
      if (pa == pc) y += nu * (T)a.rho0[pb * m + pd] - (T)l2[pb * m + pd];
      R[e] = y;
    }
    gsync<NT>();
    // partial traces of the right-hand side
    for (int idx = tid; idx < m * m; idx += NT) {
      const int x = idx / m, z = idx % m;
      T s1 = T(0), s2 = T(0);
      for (int k = 0; k < m; ++k) {
        s1 += R[(x * m + k) * D + (z * m + k)];
        s2 += R[(k * m + x) * D + (k * m + z)];
      }
      t1[idx] = s1;
      t2[idx] = s2;
    }
    gsync<NT>();
    T tr = T(0);
    for (int k = 0; k < m; ++k) tr += t1[k * m + k];
    // rho = (mu + nu A1^*A1 + nu A2^*A2)^{-1} rhs, closed form on the projectors P1, P2, Q
    for (int e = tid; e < D * D; e += NT) {
      const int i = e / D, j = e % D;
      const int pa = i / m, pb = i % m, pc = j / m, pd = j % m;
      const T y = R[e];
      const T P1 = (pb == pd) ? t1[pa * m + pc] / m : T(0);
      const T P2 = (pa == pc) ? t2[pb * m + pd] / m : T(0);
      const T Q = (i == j) ? tr / D : T(0);
      R[e] = (y - P1 - P2 + Q) * c0 + (P1 + P2 - T(2) * Q) * c1 + Q * c2;
    }
    gsync<NT>();
    T* vs = reinterpret_cast<T*>(a.vstore) + p * D * D;
    int nsw = 0;
    bool dk = false;  // the eigensolve stopped early: reconstruct with the first-order correction
    if (!FX64<D, T> && a.warm) {
      for (int e = tid; e < D * D; e += NT) V[(e / D) * LD + (e % D)] = vs[e];
      gsync<NT>();
      if (ns_due<T>(a.iter) && TILE16) {
        // as below, register-tiled warp products
        T acc[2][4];
        rgemm16<T, true, false>(V, LD, V, LD, acc, tid);
        const int r0 = 2 * (tid >> 2), c0 = 4 * (tid & 3);
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
          for (int u = 0; u < 4; ++u) acc[x][u] = ((r0 + x == c0 + u) ? T(1.5) : T(0)) - T(0.5) * acc[x][u];
        store16(Wt, LD, acc, tid);
        __syncwarp();
        rgemm16<T, false, false>(V, LD, Wt, LD, acc, tid);
        __syncwarp();
        store16(V, LD, acc, tid);
        __syncwarp();
      } else if (ns_due<T>(a.iter)) {
        // rotations erode V's orthogonality over many sweeps; one Newton-Schulz step
        // V <- V (3 I - V^T V) / 2 squares the error before V is used (A and Wt as scratch)
        for (int e = tid; e < D * D; e += NT) {
          const int i = e / D, j = e % D;
          T acc = T(0);
          for (int k = 0; k < D; ++k) acc += V[k * LD + i] * V[k * LD + j];
          Wt[i * LD + j] = ((i == j) ? T(1.5) : T(0)) - T(0.5) * acc;
        }
        gsync<NT>();
        for (int e = tid; e < D * D; e += NT) {
          const int i = e / D, j = e % D;
          T acc = T(0);
          for (int k = 0; k < D; ++k) acc += V[i * LD + k] * Wt[k * LD + j];
          A[i * LD + j] = acc;
        }
        gsync<NT>();
        for (int e = tid; e < D * D; e += NT) V[(e / D) * LD + (e % D)] = A[(e / D) * LD + (e % D)];
        gsync<NT>();
      }
    }
    // C = rho - Lambda / mu, symmetrised, into A
    for (int t = tid; t < D * (D + 1) / 2; t += NT) {
      int i, j;
      tri_index(D, t, i, j);
      const T v = T(0.5) * (R[i * D + j] + R[j * D + i]) -
                  T(0.5) * ((T)lam[i * D + j] + (T)lam[j * D + i]) * imu;
      A[i * LD + j] = v;
      A[j * LD + i] = v;
    }
    gsync<NT>();
    if constexpr (FX64<D, T>) {
      fx64::project<false>(
          base + S::V, tid, [&](int i, int j, double& re, double&) { re = A[i * LD + j]; },
          [&](int i, int j, double re, double) { A[i * LD + j] = re; });
    } else if (a.warm && TILE16) {
      // A <- V^T C V with register-tiled warp products (upper triangle mirrored)
      T acc[2][4];
      rgemm16<T, false, false>(A, LD, V, LD, acc, tid);
      store16(Wt, LD, acc, tid);
      __syncwarp();
      rgemm16<T, true, false>(V, LD, Wt, LD, acc, tid);
      store16(A, LD, acc, tid);
      mirror16<T>(A, nullptr, LD, tid);
      nsw = jacobi_sym<T, D, LD, NT, true, false, true>(A, V, cs, red, tid, &dk);
    } else if (a.warm) {
      // start from the previous eigenvectors: A <- V^T C V
      for (int e = tid; e < D * D; e += NT) {
        const int i = e / D, j = e % D;
        T acc = T(0);
#pragma unroll 4
        for (int k = 0; k < D; ++k) acc += A[i * LD + k] * V[k * LD + j];
        Wt[i * LD + j] = acc;
      }
      gsync<NT>();
      for (int t = tid; t < D * (D + 1) / 2; t += NT) {
        int i, j;
        tri_index(D, t, i, j);
        T acc = T(0);
#pragma unroll 4
        for (int k = 0; k < D; ++k) acc += V[k * LD + i] * Wt[k * LD + j];
        A[i * LD + j] = acc;
        A[j * LD + i] = acc;
      }
      gsync<NT>();
      nsw = jacobi_sym<T, D, LD, NT, true, false, true>(A, V, cs, red, tid, &dk);
    } else {
      nsw = jacobi_sym<T, D, LD, NT, true, true, true>(A, V, cs, red, tid, &dk);
    }
    if (a.stats && tid == 0) {
      atomicAdd(a.stats, (unsigned long long)nsw);
      atomicAdd(a.stats + 1, 1ull);
      if (dk) atomicAdd(a.stats + 2, 1ull);
    }
    if constexpr (!FX64<D, T>) {
      for (int e = tid; e < D * D; e += NT) vs[e] = V[(e / D) * LD + (e % D)];
      if (TILE16) {
        // rho~ = V M V^T (M = f(Lambda) + L o E after a first-order stop, else diag(max(l, 0)))
        // with register-tiled warp products; the upper triangle is mirrored
        T acc[2][4];
        if (dk) {
          dk_matrix_sym<T, D, LD, NT>(A, cs, tid);
          rgemm16<T, false, false>(V, LD, A, LD, acc, tid);
          store16(Wt, LD, acc, tid);
          __syncwarp();
          rgemm16<T, false, true>(Wt, LD, V, LD, acc, tid);
        } else {
          for (int k = tid; k < D; k += NT) {
            const T w = A[k * LD + k];
            W[k] = w > T(0) ? w : T(0);
          }
          __syncwarp();
          rgemm16<T, false, true>(V, LD, V, LD, acc, tid, W);
        }
        __syncwarp();
        store16(A, LD, acc, tid);
        mirror16<T>(A, nullptr, LD, tid);
      } else if (dk) {
        // rho~ = V M V^T with M = f(Lambda) + L o E (dk_stop): Wt = V M, then Wt V^T
        dk_matrix_sym<T, D, LD, NT>(A, cs, tid);
        for (int e = tid; e < D * D; e += NT) {
          const int i = e / D, j = e % D;
          T acc = T(0);
  #pragma unroll 4
          for (int k = 0; k < D; ++k) acc += V[i * LD + k] * A[k * LD + j];
          Wt[i * LD + j] = acc;
        }
        gsync<NT>();
        for (int t = tid; t < D * (D + 1) / 2; t += NT) {
          int i, j;
          tri_index(D, t, i, j);
          T s = T(0);
  #pragma unroll 4
          for (int k = 0; k < D; ++k) s += Wt[i * LD + k] * V[j * LD + k];
          A[i * LD + j] = s;
          A[j * LD + i] = s;
        }
      } else {
        for (int k = tid; k < D; k += NT) {
          const T w = A[k * LD + k];
          W[k] = w > T(0) ? w : T(0);
        }
        gsync<NT>();
        // rho~ = V diag(max(w, 0)) V^T
        for (int t = tid; t < D * (D + 1) / 2; t += NT) {
          int i, j;
          tri_index(D, t, i, j);
          T s = T(0);
  #pragma unroll 4
          for (int k = 0; k < D; ++k) s += W[k] * V[i * LD + k] * V[j * LD + k];
          A[i * LD + j] = s;
          A[j * LD + i] = s;
        }
      }
    }
    gsync<NT>();
    T rr = T(0), en = T(0);
    double* rtw = a.rt + p * D * D;
    double* lamw = a.lam + p * D * D;
    // swap images for -delta: rho~ and Lambda conjugated by S, X' transposed
    double* rtm = pm >= 0 ? a.rt + pm * D * D : nullptr;
    double* lamm = pm >= 0 ? a.lam + pm * D * D : nullptr;
    double* Xm = pm >= 0 ? a.X + (pm + 1) * D * D : nullptr;
    for (int e = tid; e < D * D; e += NT) {
      const int i = e / D, j = e % D;
      const int pa = i / m, pb = i % m, pc = j / m, pd = j % m;
      const T rho = R[e];
      const T rtn = A[i * LD + j];
      const T h = Hb ? (T)Hb[e] : T(0);
      const double lamn = (double)((T)lam[e] + mu * (rtn - rho));
      // X'_{0,delta} = X_{0,delta} - eps G_{0,delta}[rho], G entry (a,b),(c,d) = rho_{(a,d),(b,c)}
      const double xn = (double)(Xs[e] - eps * R[(pa * m + pd) * D + (pb * m + pc)]);
      lamw[e] = lamn;
      rtw[e] = (double)rtn;
      Xb[e] = xn;
      if (pm >= 0) {
        const int es = (pb * m + pa) * D + (pd * m + pc);
        lamm[es] = lamn;
        rtm[es] = (double)rtn;
        Xm[j * D + i] = xn;
      }
      rr += (rho - rtn) * (rho - rtn);
      en += h * R[j * D + i];
    }
    for (int idx = tid; idx < m * m; idx += NT) {
      const int x = idx / m, z = idx % m;
      T s1 = T(0), s2 = T(0);
      for (int k = 0; k < m; ++k) {
        s1 += R[(x * m + k) * D + (z * m + k)];
        s2 += R[(k * m + x) * D + (k * m + z)];
      }
      a.a1r[p * m * m + idx] = (double)s1;
      a.a2r[p * m * m + idx] = (double)s2;
      if (pm >= 0) {
        a.a1r[pm * m * m + idx] = (double)s2;
        a.a2r[pm * m * m + idx] = (double)s1;
      }
    }
    rr = gsum<NT>(rr, red);
    en = gsum<NT>(en, red);
    if (tid == 0) {
      a.part[p * 2 + 0] = (double)rr;
      a.part[p * 2 + 1] = (double)en;
      if (pm >= 0) {
        a.part[pm * 2 + 0] = (double)rr;
        a.part[pm * 2 + 1] = (double)en;
      }
    }
    gsync<NT>();
  }
}

// ---- D = 16 in float64 and double-float: the same pass with the projection in fixed point on the
// tensor cores (ve_fx16.cuh), one warp per item; one code serves both arithmetics (float64 words
// need no conversions, and the projection is float64-accurate).  The float64 pipe bounds what is
// left, the elementwise part, so that part is kept to ~200 float64 instructions a matrix: the
// constants of the closed-form solve come from the host, and its projector terms are tables of
// m x m entries (rho = c0 y + [b = d] u1 + [a = c] u2 + [i = j] q).  A lane owns the eight entries
// of the fragment layout, so Lambda, y and rho stay in registers between the steps.
// Measured (4096 clusters, 2048 items): 57 us; 272 us as float64 Jacobi sweeps.
struct Pair16Smem {
  static constexpr size_t R = 0, Xs = 2048, W = 4096, fx = W + 256;
  static constexpr size_t bytes = fx + fx16::Smem<false>::bytes;
};

__global__ void __launch_bounds__(32, 16) k_pair16(const PairArgs a, const double c0, const double e1, const double e2) {
  using namespace fx16;
  constexpr int D = 16, m = 4, mm = 16;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* R = reinterpret_cast<double*>(smem_raw + Pair16Smem::R);
  double* Xs = reinterpret_cast<double*>(smem_raw + Pair16Smem::Xs);
  double* w = reinterpret_cast<double*>(smem_raw + Pair16Smem::W);  // two m x m tables
  unsigned char* fx = smem_raw + Pair16Smem::fx;
  const int lane = threadIdx.x;
  const double mu = a.mu, nu = a.nu, eps = a.eps;
  for (long it = blockIdx.x; it < a.Pc; it += gridDim.x) {
    const long p = a.pidx ? a.pidx[it] : it;
    const long pm = a.pidx ? a.pmir[it] : -1;  // pair index of -delta, or -1
    const long dl = p + 1;
    double* rt = a.rt + p * D * D;
    double* lam = a.lam + p * D * D;
    double* Xb = a.X + dl * D * D;
    const int hs = a.hslot[dl];
    const double* Hb = hs >= 0 ? a.hb + (long)hs * D * D : nullptr;
    long long* vs = reinterpret_cast<long long*>(a.vstore) + p * D * D;

    double lv[8], y[8];
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
      const int o = frag_row(k, lane) * D + frag_col(k, lane);
      *reinterpret_cast<double2*>(Xs + o) = *reinterpret_cast<const double2*>(Xb + o);
      const double2 l = *reinterpret_cast<const double2*>(lam + o), r = *reinterpret_cast<const double2*>(rt + o);
      lv[k] = l.x;
      lv[k + 1] = l.y;
      y[k] = fma(mu, r.x, l.x);
      y[k + 1] = fma(mu, r.y, l.y);
      if (Hb) {
        const double2 h = *reinterpret_cast<const double2*>(Hb + o);
        y[k] -= h.x;
        y[k + 1] -= h.y;
      }
    }
    // lanes 0-15: entry (x, z) of the first cluster's m x m matrices, lanes 16-31: the second's
    const int id = lane & 15, tx = id >> 2, tz = id & 3;
    const bool second = lane >= 16;
    {
      const double l1 = a.lam1[p * mm + id], l2 = a.lam2[p * mm + id];
      if (pm >= 0) {  // the multipliers of -delta as images of these, before the rho_0 reduction reads them
        if (second) a.lam1[pm * mm + id] = l2;
        else a.lam2[pm * mm + id] = l1;
      }
      w[lane] = fma(nu, a.rho0[id], second ? -l2 : -l1);
    }
    __syncwarp();
    // right-hand side of Eq. (rhoijUpdate) with H' of Eq. (effHam)
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = frag_row(k, lane), j = frag_col(k, lane);
      const int pa = i / m, pb = i % m, pc = j / m, pd = j % m;
      y[k] += Xs[(pa * m + pc) * D + (pd * m + pb)] + Xs[(pc * m + pa) * D + (pb * m + pd)];
      if (pb == pd) y[k] += w[pa * m + pc];
      if (pa == pc) y[k] += w[16 + pb * m + pd];
      R[i * D + j] = y[k];
    }
    // partial traces of the matrix in R: (lane < 16) Tr_2, entry (x, z); else Tr_1
    auto trace = [&]() {
      const int st = second ? m * D + m : D + 1, o = second ? tx * D + tz : (tx * D + tz) * m;
      return (R[o] + R[o + st]) + (R[o + 2 * st] + R[o + 3 * st]);
    };
    __syncwarp();
    {
      const double t = trace();
      const unsigned all = 0xffffffffu;
      const double tr = (__shfl_sync(all, t, 0) + __shfl_sync(all, t, 5)) +
                        (__shfl_sync(all, t, 10) + __shfl_sync(all, t, 15));
      __syncwarp();
      w[lane] = e1 * t;
      __syncwarp();
      // rho = (mu + nu A1^*A1 + nu A2^*A2)^{-1} rhs, closed form on the projectors P1, P2, Q
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int i = frag_row(k, lane), j = frag_col(k, lane);
        const int pa = i / m, pb = i % m, pc = j / m, pd = j % m;
        y[k] *= c0;
        if (pb == pd) y[k] += w[pa * m + pc];
        if (pa == pc) y[k] += w[16 + pb * m + pd];
        if (i == j) y[k] = fma(e2, tr, y[k]);
        R[i * D + j] = y[k];
      }
    }
    // C = rho - Lambda / mu, symmetrised in fixed point, and its projection
    Frag yq, none;
    int ye = 0, nsw = 0;
    bool dk = false;
    double c[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) c[k] = fma(-c0, lv[k], y[k]);
    const bool finite = fix_matrix<false>(c, c, yq, none, ye);
    if (finite) {
      add_adjoint<false>(yq, none, fx, lane);
      ye -= 1;
      normalise<false>(yq, none, ye);
      const int ce = ye;
      Frag cq;
#pragma unroll
      for (int k = 0; k < 8; ++k) cq[k] = yq[k];
      const Result res = project<false>(yq, none, ye, vs, a.warm != 0, fx, lane, &dk, &nsw);
      if (res != kProduct) {
        ye = ce;
#pragma unroll
        for (int k = 0; k < 8; ++k) yq[k] = res == kSame ? cq[k] : 0;
      }
    } else if (!a.warm) {  // nothing to diagonalise: the store starts from V = I
      identity_vectors<false>(vs, lane);
    }
    if (a.stats && lane == 0) {
      atomicAdd(a.stats, (unsigned long long)nsw);
      atomicAdd(a.stats + 1, 1ull);
      if (dk) atomicAdd(a.stats + 2, 1ull);
    }
    __syncwarp();
    double rr = 0.0, en = 0.0;
    // swap images for -delta: rho~ and Lambda conjugated by S, X' transposed
    double* rtm = pm >= 0 ? a.rt + pm * D * D : nullptr;
    double* lamm = pm >= 0 ? a.lam + pm * D * D : nullptr;
    double* Xm = pm >= 0 ? a.X + (pm + 1) * D * D : nullptr;
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
      const int i = frag_row(k, lane), j = frag_col(k, lane), o = i * D + j;
      double rn[2], ln[2], xn[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int pa = i / m, pb = i % m, pc = (j + u) / m, pd = (j + u) % m;
        rn[u] = finite ? word(yq[k + u], ye) : NAN;
        const double diff = rn[u] - y[k + u];
        ln[u] = fma(mu, diff, lv[k + u]);
        // X'_{0,delta} = X_{0,delta} - eps G_{0,delta}[rho], G entry (a,b),(c,d) = rho_{(a,d),(b,c)}
        xn[u] = fma(-eps, R[(pa * m + pd) * D + (pb * m + pc)], Xs[o + u]);
        rr = fma(diff, diff, rr);
        if (Hb) en = fma(Hb[o + u], R[(j + u) * D + i], en);
        if (pm >= 0) {
          const int es = (pb * m + pa) * D + (pd * m + pc);
          lamm[es] = ln[u];
          rtm[es] = rn[u];
          Xm[(j + u) * D + i] = xn[u];
        }
      }
      *reinterpret_cast<double2*>(lam + o) = make_double2(ln[0], ln[1]);
      *reinterpret_cast<double2*>(rt + o) = make_double2(rn[0], rn[1]);
      *reinterpret_cast<double2*>(Xb + o) = make_double2(xn[0], xn[1]);
    }
    {
      const double t = trace();
      (second ? a.a2r : a.a1r)[p * mm + id] = t;
      if (pm >= 0) (second ? a.a1r : a.a2r)[pm * mm + id] = t;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rr += shfl_xor(rr, o);
    if (Hb) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) en += shfl_xor(en, o);
    }
    if (lane == 0) {
      a.part[p * 2 + 0] = rr;
      a.part[p * 2 + 1] = en;
      if (pm >= 0) {
        a.part[pm * 2 + 0] = rr;
        a.part[pm * 2 + 1] = en;
      }
    }
    __syncwarp();
  }
}

cudaError_t launch_pair16(const PairArgs& a, cudaStream_t s) {
  static unsigned long long mask = 0;
  cudaError_t e = smem_once(k_pair16, Pair16Smem::bytes, mask);
  if (e != cudaSuccess) return e;
  long blocks = resident_grid((const void*)k_pair16, 32, Pair16Smem::bytes);
  if (blocks > a.Pc) blocks = a.Pc;
  if (blocks < 1) blocks = 1;
  k_pair16<<<(unsigned)blocks, 32, Pair16Smem::bytes, s>>>(a, a.k.c0, (a.k.c1 - a.k.c0) / 4,
                                                        (a.k.c0 - 2.0 * a.k.c1 + a.k.c2) / 16);
  return cudaGetLastError();
}

// ---- D = 256 in float32 with the projection on the tensor cores (ve_tcproj.cu): the pair
// pass splits around one batched projection.  k_pair256_pre forms rho (Eq. (rhoijUpdate)) into
// rbuf and C = rho - Lambda / mu (symmetrised) into the projection's split input; after
// tc_project256, k_pair256_post does what k_pair does after its eigensolve.  Arithmetic in
// float32, as k_pair<256, float>.
constexpr int P256_NT = 512;

__device__ __forceinline__ float tf32_part(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }

__global__ void __launch_bounds__(P256_NT) k_pair256_pre(const PairArgs a, float* __restrict__ Cout) {
  constexpr int D = 256, m = 16, NT = P256_NT, PL = D * D;
  __shared__ float t1[m * m], t2[m * m];
  __shared__ float rho0[m * m];
  const int tid = threadIdx.x;
  const float mu = (float)a.mu, nu = (float)a.nu;
  const float alpha = nu * m;
  const float c0 = 1.f / mu, c1 = 1.f / (mu + alpha), c2 = 1.f / (mu + 2.f * alpha);
  const float imu = 1.f / mu;
  for (int k = tid; k < m * m; k += NT) rho0[k] = (float)a.rho0[k];
  for (long it = blockIdx.x; it < a.Pc; it += gridDim.x) {
    const long p = a.pidx ? a.pidx[it] : it;
    const long pm = a.pidx ? a.pmir[it] : -1;
    const long dl = p + 1;
    const double* rt = a.rt + p * PL;
    const double* lam = a.lam + p * PL;
    const double* l1 = a.lam1 + p * m * m;
    const double* l2 = a.lam2 + p * m * m;
    const double* Xb = a.X + dl * PL;
    const int hs = a.hslot[dl];
    const double* Hb = hs >= 0 ? a.hb + (long)hs * PL : nullptr;
    float* R = a.rbuf + it * PL;
    if (pm >= 0) {
      for (int idx = tid; idx < m * m; idx += NT) {
        a.lam1[pm * m * m + idx] = l2[idx];
        a.lam2[pm * m * m + idx] = l1[idx];
      }
    }
    __syncthreads();
    // right-hand side of Eq. (rhoijUpdate) with H' of Eq. (effHam)
    for (int e = tid; e < PL; e += NT) {
      const int i = e / D, j = e % D;
      const int pa = i / m, pb = i % m, pc = j / m, pd = j % m;
      const float h = Hb ? (float)Hb[e] : 0.f;
      const float hp = h - (float)Xb[(pa * m + pc) * D + (pd * m + pb)] - (float)Xb[(pc * m + pa) * D + (pb * m + pd)];
      float y = mu * (float)rt[e] + (float)lam[e] - hp;
      if (pb == pd) y += nu * rho0[pa * m + pc] - (float)l1[pa * m + pc];
      if (pa == pc) y += nu * rho0[pb * m + pd] - (float)l2[pb * m + pd];
      R[e] = y;
    }
    __syncthreads();
    for (int idx = tid; idx < m * m; idx += NT) {
      const int x = idx / m, z = idx % m;
      float s1 = 0.f, s2 = 0.f;
      for (int k = 0; k < m; ++k) {
        s1 += R[(x * m + k) * D + (z * m + k)];
        s2 += R[(k * m + x) * D + (k * m + z)];
      }
      t1[idx] = s1;
      t2[idx] = s2;
    }
    __syncthreads();
    float tr = 0.f;
    for (int k = 0; k < m; ++k) tr += t1[k * m + k];
    for (int e = tid; e < PL; e += NT) {
      const int i = e / D, j = e % D;
      const int pa = i / m, pb = i % m, pc = j / m, pd = j % m;
      const float y = R[e];
      const float P1 = (pb == pd) ? t1[pa * m + pc] / m : 0.f;
      const float P2 = (pa == pc) ? t2[pb * m + pd] / m : 0.f;
      const float Q = (i == j) ? tr / D : 0.f;
      R[e] = (y - P1 - P2 + Q) * c0 + (P1 + P2 - 2.f * Q) * c1 + Q * c2;
    }
    __syncthreads();
    // C = rho - Lambda / mu, symmetrised, split into the KC4 input of the projection
    float* C = Cout + it * 2 * PL;
    for (int q = tid; q < PL / 4; q += NT) {
      const int r = q % D, k0 = (q / D) * 4;
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = k0 + u;
        v[u] = 0.5f * (R[r * D + j] + R[j * D + r]) - 0.5f * ((float)lam[r * D + j] + (float)lam[j * D + r]) * imu;
      }
      float4 hi, lo;
      hi = make_float4(tf32_part(v[0]), tf32_part(v[1]), tf32_part(v[2]), tf32_part(v[3]));
      lo = make_float4(v[0] - hi.x, v[1] - hi.y, v[2] - hi.z, v[3] - hi.w);
      *reinterpret_cast<float4*>(C + 4 * q) = hi;
      *reinterpret_cast<float4*>(C + PL + 4 * q) = lo;
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(P256_NT) k_pair256_post(const PairArgs a, const float* __restrict__ Y) {
  constexpr int D = 256, m = 16, NT = P256_NT, PL = D * D;
  __shared__ float red[NT / 32];
  const int tid = threadIdx.x;
  const float mu = (float)a.mu, eps = (float)a.eps;
  for (long it = blockIdx.x; it < a.Pc; it += gridDim.x) {
    const long p = a.pidx ? a.pidx[it] : it;
    const long pm = a.pidx ? a.pmir[it] : -1;
    const long dl = p + 1;
    const float* R = a.rbuf + it * PL;
    const float* y = Y + it * 2 * PL;
    double* Xb = a.X + dl * PL;
    const int hs = a.hslot[dl];
    const double* Hb = hs >= 0 ? a.hb + (long)hs * PL : nullptr;
    double* rtw = a.rt + p * PL;
    double* lamw = a.lam + p * PL;
    double* rtm = pm >= 0 ? a.rt + pm * PL : nullptr;
    double* lamm = pm >= 0 ? a.lam + pm * PL : nullptr;
    double* Xm = pm >= 0 ? a.X + (pm + 1) * PL : nullptr;
    float rr = 0.f, en = 0.f;
    // X' reads X_{0,delta} before this item overwrites it: each thread rewrites only entries
    // it has read (e), and the transposed image goes to another block (-delta)
    for (int e = tid; e < PL; e += NT) {
      const int i = e / D, j = e % D;
      const int pa = i / m, pb = i % m, pc = j / m, pd = j % m;
      const float rho = R[e];
      const int o = ((j >> 2) * D + i) * 4 + (j & 3);
      const float rtn = y[o] + y[PL + o];
      const float h = Hb ? (float)Hb[e] : 0.f;
      const double lamn = (double)((float)a.lam[p * PL + e] + mu * (rtn - rho));
      const double xn = (double)((float)Xb[e] - eps * R[(pa * m + pd) * D + (pb * m + pc)]);
      lamw[e] = lamn;
      rtw[e] = (double)rtn;
      Xb[e] = xn;
      if (pm >= 0) {
        const int es = (pb * m + pa) * D + (pd * m + pc);
        lamm[es] = lamn;
        rtm[es] = (double)rtn;
        Xm[j * D + i] = xn;
      }
      rr += (rho - rtn) * (rho - rtn);
      en += h * R[j * D + i];
    }
    for (int idx = tid; idx < m * m; idx += NT) {
      const int x = idx / m, z = idx % m;
      float s1 = 0.f, s2 = 0.f;
      for (int k = 0; k < m; ++k) {
        s1 += R[(x * m + k) * D + (z * m + k)];
        s2 += R[(k * m + x) * D + (k * m + z)];
      }
      a.a1r[p * m * m + idx] = (double)s1;
      a.a2r[p * m * m + idx] = (double)s2;
      if (pm >= 0) {
        a.a1r[pm * m * m + idx] = (double)s2;
        a.a2r[pm * m * m + idx] = (double)s1;
      }
    }
    rr = gsum<NT>(rr, red);
    en = gsum<NT>(en, red);
    if (tid == 0) {
      a.part[p * 2 + 0] = (double)rr;
      a.part[p * 2 + 1] = (double)en;
      if (pm >= 0) {
        a.part[pm * 2 + 0] = (double)rr;
        a.part[pm * 2 + 1] = (double)en;
      }
    }
    __syncthreads();
  }
}

cudaError_t launch_pair_tc(const PairArgs& a, cudaStream_t s) {
  TcProjWs& w = *a.tcw;
  const int grid = (int)(a.Pc < 2 * big_grid() ? a.Pc : 2 * big_grid());
  k_pair256_pre<<<grid, P256_NT, 0, s>>>(a, w.C);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if ((e = tc_project256(w, a.Pc, a.warm != 0, a.stats, s)) != cudaSuccess) return e;
  k_pair256_post<<<grid, P256_NT, 0, s>>>(a, w.Wt);
  return cudaGetLastError();
}

template <int D, typename T>
cudaError_t launch_pair_t(const PairArgs& a, cudaStream_t s) {
  constexpr int NT = PairShape<D, T>::NT, GPC = PairShape<D, T>::GPC;
  constexpr bool G = GroupShape<D>::GLOBAL;
  const size_t smem = G ? 0 : PairSmem<D, T>::bytes * GPC;
  cudaError_t e = cudaSuccess;
  if (!G) {
    static unsigned long long mask = 0;
    e = smem_once(k_pair<D, T>, smem, mask);
    if (e != cudaSuccess) return e;
  }
  long blocks = (a.Pc + GPC - 1) / GPC;
  const long res = G ? (long)big_grid() : resident_grid((const void*)k_pair<D, T>, NT * GPC, smem);
  if (blocks > res) blocks = res;
  if (blocks < 1) blocks = 1;
  k_pair<D, T><<<(unsigned)blocks, NT * GPC, smem, s>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- rho_0 and X'_00
// RHO0_CHUNKS CTAs each sum a contiguous range of offsets delta of nu A1[rho_{0,delta}] +
// Lambda1_{0,delta} (m*m entries); the last CTA to finish (a counter in the status block) adds
// the chunk sums in order.  Both orders are fixed, so the result is reproducible bit for bit.
// Latency bounds it (a float64 add of a lone warp takes 64 cycles), and the X step waits for it: up
// to RHO0_CHUNKS offsets one CTA forms the chunks' terms itself, added in the same order, without
// the counter's round trip; what does not depend on the sums is read before them.
constexpr int RHO0_CHUNKS = 128;

__global__ void __launch_bounds__(256) k_rho0(const SmallArgs a, double* partial) {
  const int m = a.m, mm = m * m, D = a.D;
  // threads: (entry, sub-range) with 256 / mm sub-ranges per chunk
  const int subs = 256 / mm;
  __shared__ double S[256];
  const int t = threadIdx.x;
  const int idx = t % mm, c = t / mm;
  auto term = [&](long p) { return a.nu * a.a1r[p * mm + idx] + a.lam1[p * mm + idx]; };
  // H'_0 = H_0 - sum_a X_{(a,b),(a,d)}  (Eq. (effHam) with matrix units)
  double h0 = 0.0, h0p = 0.0;
  if (t < mm) {
    const int b = t / m, d = t % m;
    double hx = 0.0;
    for (int x = 0; x < m; ++x) hx += a.X[(x * m + b) * D + (x * m + d)];
    h0 = a.H0[t];
    h0p = h0 - hx;
  }
  double acc = 0.0;
  if (gridDim.x == 1) {
    for (long p = c; p < a.P; p += subs) acc += term(p);
  } else {
    const long per = (a.P + RHO0_CHUNKS - 1) / RHO0_CHUNKS;
    const long lo = blockIdx.x * per, hi = min((long)a.P, lo + per);
    for (long p = lo + c; p < hi; p += subs) acc += term(p);
    S[t] = acc;
    __syncthreads();
    if (t < mm) {
      double s = 0.0;
      for (int k = 0; k < subs; ++k) s += S[k * mm + t];
      partial[blockIdx.x * mm + t] = s;
    }
    __threadfence();
    __shared__ bool last;
    __syncthreads();
    if (t == 0) last = atomicAdd(&a.st->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // the last CTA: rho_0 from the chunk sums (read past L1: other CTAs wrote them), each entry
    // summed by subs threads over interleaved chunks, then in order over the threads
    acc = 0.0;
    for (int k = c; k < RHO0_CHUNKS; k += subs) acc += __ldcg(partial + k * mm + idx);
  }
  S[t] = acc;
  __syncthreads();
  __shared__ double rp[256];
  __shared__ double red[8];
  if (t < mm) {
    const int live = gridDim.x == 1 && a.P < subs ? a.P : subs;  // the others hold zeros
    double s = 0.0;
    for (int k = 0; k < live; ++k) s += S[k * mm + t];
    rp[t] = (s - h0p) / (a.nu * (a.N - 1));
  }
  __syncthreads();
  double tr = 0.0;
  for (int k = 0; k < m; ++k) tr += rp[k * m + k];
  const double z = (1.0 - tr) / m;
  __syncthreads();
  if (t < mm) {
    const double r = rp[t] + (t / m == t % m ? z : 0.0);
    rp[t] = r;
    a.rho0[t] = r;
  }
  __syncthreads();
  // X'_00 = X_00 - eps G_00[rho_0], G_00 entry (a,b),(c,d) = delta_ac rho0_{d,b}
  for (int u = t; u < m * mm; u += 256) {
    const int pa = u / mm, pb = (u / m) % m, pd = u % m;
    a.X[(pa * m + pb) * D + (pa * m + pd)] -= a.eps * rp[pd * m + pb];
  }
  // Tr[H_0 rho_0]
  double h = 0.0;
  if (t < mm) h = h0 * rp[(t % m) * m + (t / m)];
  h = gsum<256>(h, red);
  if (t == 0) {
    a.st->h0rho0 = h;
    a.st->done = 0u;  // ready for the next sweep
    a.st->sweep = a.st->iter + 1;
  }
}

// ---------------------------------------------------------------- Lambda1, Lambda2, status
// One warp per pair offset.  With ties (see k_pair) the canonical member of {delta, -delta}
// also writes the other's multipliers, Lambda1_{-delta} = Lambda2_delta and Lambda2_{-delta} =
// Lambda1_delta, so the two stay exact swap images (and the offset counts twice in the sums).  Every
// CTA adds up its offsets' residual and energy terms; the last one to finish adds the CTA sums in
// order and writes the status block: one launch for what were two (8 + 13 us, latency).
constexpr int DUAL_CTAS = 128, DUAL_THREADS = 256;

__global__ void __launch_bounds__(DUAL_THREADS) k_dual_status(const SmallArgs a, double* partial) {
  __shared__ double red[DUAL_THREADS / 32][3];
  const int lane = threadIdx.x & 31, wc = threadIdx.x >> 5;
  const int mm = a.m * a.m;
  const long warps = (long)gridDim.x * (DUAL_THREADS / 32);
  double rr = 0.0, en = 0.0, ff = 0.0;
  for (long w = (long)blockIdx.x * (DUAL_THREADS / 32) + wc; w < a.P; w += warps) {
    const long tie = a.ptie ? a.ptie[w] : -1;
    if (tie == -2) continue;  // uniform over the warp
    double s = 0.0;
    for (int idx = lane; idx < mm; idx += 32) {
      const double r0 = a.rho0[idx];
      const double d1 = a.a1r[w * mm + idx] - r0;
      const double d2 = a.a2r[w * mm + idx] - r0;
      const double n1 = a.lam1[w * mm + idx] + a.nu * d1;
      const double n2 = a.lam2[w * mm + idx] + a.nu * d2;
      a.lam1[w * mm + idx] = n1;
      a.lam2[w * mm + idx] = n2;
      if (tie >= 0) {
        a.lam1[tie * mm + idx] = n2;
        a.lam2[tie * mm + idx] = n1;
      }
      s += d1 * d1 + d2 * d2;
    }
    const double c = tie >= 0 ? 2.0 : 1.0;
    ff = fma(c, s, ff);
    if (lane == 0) {
      rr = fma(c, a.part[w * 2 + 0], rr);
      en = fma(c, a.part[w * 2 + 1], en);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ff += __shfl_xor_sync(0xffffffffu, ff, o);
  if (lane == 0) {
    red[wc][0] = rr;
    red[wc][1] = en;
    red[wc][2] = ff;
  }
  __syncthreads();
  const int t = threadIdx.x;
  if (t < 3) {
    double v = 0.0;
    for (int k = 0; k < DUAL_THREADS / 32; ++k) v += red[k][t];
    partial[blockIdx.x * 3 + t] = v;
  }
  __threadfence();
  __shared__ bool last;
  __syncthreads();
  if (t == 0) last = atomicAdd(&a.st->done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (t >= 32) return;
  rr = en = ff = 0.0;
  for (int k = t; k < (int)gridDim.x; k += 32) {
    rr += __ldcg(partial + k * 3 + 0);
    en += __ldcg(partial + k * 3 + 1);
    ff += __ldcg(partial + k * 3 + 2);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rr += __shfl_xor_sync(0xffffffffu, rr, o);
    en += __shfl_xor_sync(0xffffffffu, en, o);
    ff += __shfl_xor_sync(0xffffffffu, ff, o);
  }
  if (t == 0) {
    DevStatus* st = a.st;
    st->done = 0u;
    const double E = (st->h0rho0 + 0.5 * en) / a.L;
    const double feas = sqrt((rr + ff) / a.P);
    const double dE = isfinite(st->e_prev) ? fabs(E - st->e_prev) : INFINITY;
    st->energy = E;
    st->feas = feas;
    st->d_energy = dE;
    st->residual = fmax(feas, dE);
    st->e_prev = E;
    st->iter += 1;
  }
}

}  // namespace

int resident_grid(const void* kernel, int threads, size_t smem) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem);
  if (sms < 1) sms = 1;
  if (per < 1) per = 1;
  return sms * per;
}

template <int D>
cudaError_t launch_pair_d(const PairArgs& a, int arith, cudaStream_t s) {
  if constexpr (D == 16) {
    return arith == ARITH_FP32 ? launch_pair_t<D, float>(a, s)
           : arith == ARITH_FP64 || arith == ARITH_DF64 ? launch_pair16(a, s) : cudaErrorInvalidValue;
  } else if constexpr (D == 64) {
    return arith == ARITH_FP32 ? launch_pair_t<D, float>(a, s)
           : arith == ARITH_FP64 || arith == ARITH_DF64 ? launch_pair_t<D, double>(a, s) : cudaErrorInvalidValue;
  } else {
    switch (arith) {
      case ARITH_FP64: return launch_pair_t<D, double>(a, s);
      case ARITH_FP32: return launch_pair_t<D, float>(a, s);
      case ARITH_DF64: return launch_pair_t<D, df64>(a, s);
      default: return cudaErrorInvalidValue;
    }
  }
}

cudaError_t launch_pair(const PairArgs& a, int arith, cudaStream_t s) {
  if (a.D == 256 && arith == ARITH_FP32 && a.tcw && a.rbuf) return launch_pair_tc(a, s);
  switch (a.D) {
    case 4: return launch_pair_d<4>(a, arith, s);
    case 16: return launch_pair_d<16>(a, arith, s);
    case 64: return launch_pair_d<64>(a, arith, s);
    case 256: return launch_pair_d<256>(a, arith, s);
    default: return cudaErrorInvalidValue;
  }
}

size_t pair_ws_bytes(int D) {
  if (D != 256) return 0;
  size_t a = PairSmem<256, double>::bytes;
  if (PairSmem<256, df64>::bytes > a) a = PairSmem<256, df64>::bytes;
  return a * (size_t)big_grid();
}

int big_grid() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

cudaError_t launch_rho0(const SmallArgs& a, cudaStream_t s) {
  k_rho0<<<a.P <= RHO0_CHUNKS ? 1 : RHO0_CHUNKS, 256, 0, s>>>(a, a.rho0_partial);
  return cudaGetLastError();
}

cudaError_t launch_dual_status(const SmallArgs& a, cudaStream_t s) {
  const long need = ((long)a.P + DUAL_THREADS / 32 - 1) / (DUAL_THREADS / 32);
  k_dual_status<<<(unsigned)(need < DUAL_CTAS ? need : DUAL_CTAS), DUAL_THREADS, 0, s>>>(a, a.rho0_partial);
  return cudaGetLastError();
}

}  // namespace ve
