// Batched Hermitian eigensolver and the pole (pseudo-Hamiltonian) path (sm_103a).
//
// When Sigma has the pole form of Sec. 3.2.4 (Eq. se_pole),
//   Sigma(i w) = Sigma_inf + sum_i V_i^+ V_i / (i w - p_i),   V_i a 1 x m row,
// the band block of the resolvent of the pseudo-Hamiltonian of Sec. 3.3
// (Eq. pseudo_H_k), here with the pole energies shifted by mu,
//   H_ps = [[H_k + P^+ Sigma_inf P, W^+], [W, diag(p + mu)]],  W_i = V_i P_k,
// is G(k, i w_n) of Eq. dmftloop1 exactly.  With H_ps = Psi diag(E) Psi^+ the
// lattice sums follow in closed form (Eqs. rho_LDA+DMFT_componet_final, fix_mu):
//   rho_k = Psi_b diag(n_F(E - mu)) Psi_b^+,  N_k = sum_l |Psi_b,l|^2 n_F(E_l - mu),
//   G_loc(i w_n) = sum_k w_k sum_l phi_l phi_l^+ / (i w_n + mu - E_l),  phi_l = P Psi_b,l,
// where Psi_b is the band block (first N_b rows) of the eigenvectors.
//
// Two eigensolvers, one CTA per matrix, the matrix and the eigenvectors in shared memory when
// 2 N (N|1) 16-byte elements fit, else in a per-CTA slice of a global workspace (L2-resident):
//  * heev_tri: Householder tridiagonalisation, the tridiagonal eigenpairs in parallel (QR steps
//    where levels are too close for that), back-transformation.  The pole path, the block form's
//    setup and the Lowdin projectors.  N(mu) from pseudo-Hamiltonians of 68 rows takes 1.4 ms for
//    125 k-points (FP64 pipe 73 % busy) and 9.6 ms for 1000, by Jacobi 16.9 and 105 ms.
//  * cyclic Jacobi with the round-robin (circle) ordering of disjoint pairs, so that one step
//    applies N/2 independent rotations: gf_heev_batched, whose caller sets the sweep limit, and
//    the low-rank kernel's setup.
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "gf_block.cuh"
#include "gf_complex.cuh"
#include "gf_internal.cuh"
#include "gf_series.cuh"

namespace gf {

namespace {

using namespace cx;

constexpr int kEigThreads = 256;
// tri_eig: largest entry of Z^T Z - I, largest residual |T z - lambda z| of the norm
// (others 3e-16); nearest levels, of the norm
constexpr float kTriOrth = 3e-8f, kTriRes = 3e-15f, kTriNear = 3e-8f;

__device__ __forceinline__ double eig_block_sum(double v, double* red) {
  // Deterministic: fixed xor tree inside each warp, then warp 0 over the warps.
  for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double r = 0.0;
  for (int w = 0; w < kEigThreads / 32; ++w) r += red[w];
  __syncthreads();
  return r;  // the same value in every thread
}

// Fermi function n_F(x) = 1 / (e^{beta x} + 1) without overflow.
__device__ __forceinline__ double fermi(double x, double beta) {
  return 0.5 * (1.0 - tanh(0.5 * beta * x));
}

// Divided difference (n_F(x) - n_F(y)) / (x - y), n_F'(x) at x = y, from
// fx = n_F(x) and chx = cosh(beta x / 2): with u = beta (x - y) / 2 it is
// -(beta/4) (sinh u / u) / (cosh(beta x/2) cosh(beta y/2)) (tanh difference
// formula), used for |u| <= 1 where the plain quotient would cancel; an
// infinite cosh gives the correct limit 0.  For |u| > 1 the plain quotient
// loses at most 2^-52 / |x - y| <= 2^-53 beta in absolute terms.
__device__ __forceinline__ double fermi_divdiff(double x, double y, double fx, double fy,
                                                double chx, double chy, double beta) {
  const double u = 0.5 * beta * (x - y);
  if (fabs(u) > 1.0) return (fx - fy) / (x - y);
  const double su = fabs(u) < 1e-4 ? fma(u * u, 1.0 / 6.0, 1.0) : sinh(u) / u;
  return -0.25 * beta * su / (chx * chy);
}

// Pair k of round-robin step r over np2 (even) indices: the last index stays,
// the others rotate.  Every unordered pair occurs once in np2 - 1 steps.
__device__ __forceinline__ void rr_pair(int r, int k, int np2, int& p, int& q) {
  const int m = np2 - 1;
  int a, b;
  if (k == 0) {
    a = m;
    b = r;
  } else {
    a = (r + k) % m;
    b = (r - k + m) % m;
  }
  p = min(a, b);
  q = max(a, b);
}

// Cyclic Jacobi on the Hermitian N x N matrix A (row-major, leading dimension
// ld, full storage); V receives the eigenvectors as columns (V = I on entry is
// set here).  On return the diagonal of A holds the eigenvalues.  Scratch:
// rot[4 * npair] doubles and ph[npair] complex in shared memory.  Returns the
// number of sweeps, or -1 when max_sweeps did not reach the threshold
// off(A) <= 1e-30 ||A||_F^2.
__device__ int jacobi_heev(double2* A, double2* V, int N, int ld, int max_sweeps, double* rot,
                           double2* ph, double* red) {
  const int tid = threadIdx.x;
  for (int e = tid; e < N * N; e += kEigThreads) {
    const int i = e / N, j = e - (e / N) * N;
    V[i * ld + j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
  }
  const int np2 = N + (N & 1);
  const int npair = np2 / 2;
  __syncthreads();
  for (int sweep = 0;; ++sweep) {
    double off = 0.0, all = 0.0;
    for (int e = tid; e < N * N; e += kEigThreads) {
      const int i = e / N, j = e - (e / N) * N;
      const double2 a = A[i * ld + j];
      const double s = a.x * a.x + a.y * a.y;
      all += s;
      if (i != j) off += s;
    }
    off = eig_block_sum(off, red);
    all = eig_block_sum(all, red);
    if (off <= 1e-30 * all || off == 0.0) return sweep;
    if (sweep >= max_sweeps) return -1;
    for (int r = 0; r < np2 - 1; ++r) {
      // rotation of each pair: J = [[c, s], [-s e, c e]] with e = conj(b)/|b|
      for (int k = tid; k < npair; k += kEigThreads) {
        int p, q;
        rr_pair(r, k, np2, p, q);
        double c = 1.0, s = 0.0, dp = 0.0, dq = 0.0;
        double2 e = make_double2(1.0, 0.0);
        if (q < N) {
          const double2 b = A[p * ld + q];
          const double ab = hypot(b.x, b.y);
          const double a = A[p * ld + p].x, d = A[q * ld + q].x;
          if (ab > 0.0) {
            const double zeta = (d - a) / (2.0 * ab);
            const double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(fma(zeta, zeta, 1.0)));
            c = 1.0 / sqrt(fma(t, t, 1.0));
            s = t * c;
            e = make_double2(b.x / ab, -b.y / ab);
            dp = a - t * ab;
            dq = d + t * ab;
          } else {
            dp = a;
            dq = d;
          }
        }
        rot[4 * k + 0] = c;
        rot[4 * k + 1] = s;
        rot[4 * k + 2] = dp;
        rot[4 * k + 3] = dq;
        ph[k] = e;
      }
      __syncthreads();
      // columns: M[:, p] <- c M[:, p] - s e M[:, q];  M[:, q] <- s M[:, p] + c e M[:, q]
      for (int x = tid; x < 2 * N * npair; x += kEigThreads) {
        const int which = x >= N * npair;  // 0: A, 1: V
        const int y = x - which * N * npair;
        const int k = y / N, i = y - (y / N) * N;
        int p, q;
        rr_pair(r, k, np2, p, q);
        if (q >= N) continue;
        const double c = rot[4 * k + 0], s = rot[4 * k + 1];
        if (s == 0.0 && ph[k].x == 1.0 && ph[k].y == 0.0) continue;
        double2* M = which ? V : A;
        const double2 xp = M[i * ld + p], xq = M[i * ld + q];
        const double2 eq = cmul(ph[k], xq);
        M[i * ld + p] = make_double2(c * xp.x - s * eq.x, c * xp.y - s * eq.y);
        M[i * ld + q] = make_double2(s * xp.x + c * eq.x, s * xp.y + c * eq.y);
      }
      __syncthreads();
      // rows of A: A[p, :] <- c A[p, :] - s conj(e) A[q, :];  A[q, :] <- s A[p, :] + c conj(e) A[q, :]
      for (int y = tid; y < N * npair; y += kEigThreads) {
        const int k = y / N, j = y - (y / N) * N;
        int p, q;
        rr_pair(r, k, np2, p, q);
        if (q >= N) continue;
        const double c = rot[4 * k + 0], s = rot[4 * k + 1];
        if (j == p) {
          A[p * ld + p] = make_double2(rot[4 * k + 2], 0.0);
          A[q * ld + p] = make_double2(0.0, 0.0);
          continue;
        }
        if (j == q) {
          A[q * ld + q] = make_double2(rot[4 * k + 3], 0.0);
          A[p * ld + q] = make_double2(0.0, 0.0);
          continue;
        }
        if (s == 0.0 && ph[k].x == 1.0 && ph[k].y == 0.0) continue;
        const double2 ec = make_double2(ph[k].x, -ph[k].y);
        const double2 xp = A[p * ld + j], xq = A[q * ld + j];
        const double2 eq = cmul(ec, xq);
        A[p * ld + j] = make_double2(c * xp.x - s * eq.x, c * xp.y - s * eq.y);
        A[q * ld + j] = make_double2(s * xp.x + c * eq.x, s * xp.y + c * eq.y);
      }
      __syncthreads();
    }
  }
}

// Entry (l, l2), l <= l2, of a packed triangle.
__device__ __forceinline__ void tri_pair(int e, int& l, int& l2) {
  l2 = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
  while (l2 * (l2 + 1) / 2 > e) --l2;
  while ((l2 + 1) * (l2 + 2) / 2 <= e) ++l2;
  l = e - l2 * (l2 + 1) / 2;
}

// Scratch of heev_tri in shared memory, for matrices up to 256.
struct QlScratch {
  double d[256], e[256];          // the tridiagonal matrix
  double tau[256];                // reflector scales
  double2 ph[256];                // phases that make the off-diagonal real
  union {
    struct {
      double2 v[256], p[256];     // the current reflector and A v
    };
    double2 rot[2][256];          // QR steps: (c, s) of two sweeps
    struct {
      double lam[256];            // eigenvalues, ascending
      float fd[256], fe[256];     // FP32 copies of d and e^2 for the bisection
      float red[kEigThreads / 32];
    };
  };
  int lo[2], hi[2];
  int more, failed;
};

// Largest of v over the CTA; NaN counts as infinite.
__device__ __forceinline__ float block_max(float v, float* red) {
  v = v == v ? v : INFINITY;
  for (int off = 16; off; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  for (int w = 0; w < kEigThreads / 32; ++w) v = fmaxf(v, red[w]);
  return v;
}

// Eigenpairs of the real symmetric tridiagonal matrix (q.d, q.e), one thread per eigenvalue:
// bisection on Sturm counts in FP32, then three Rayleigh quotient steps in FP64 whose vector comes
// from the twisted factorization at the row of the smallest pivot (Dhillon and Parlett, Linear
// Algebra Appl. 387, 2004), and one step Z <- Z (3 I - Z^T Z) / 2 that restores the orthogonality
// which nearby eigenvalues lose.  Returns false, with d and e unchanged, when an eigenvalue pair
// is closer than that step can mend (degenerate levels, a split matrix, non-finite input): the
// caller then takes QR steps.  The step leaves Z^T Z = I - (3/4) G^2, 7e-16 at the largest G taken, and
// a pair that three quotient steps did not separate keeps a residual; without the residual's limit and
// with G up to 1e-5, levels 1e-6 of the norm apart (two or five, of 26 and 68) came out with
// |T Z - Z L| 4e-12 and |Z^T Z - I| 9e-11.  An FP64 instruction holds its scheduler for 64 clocks for one
// lane as for 32, so this does in about 170 N of them, side by side, what QR steps do in 24 per rotation
// (5,400 rotations for N = 68), one after the other.
__device__ bool tri_eig(double* Z, int zr, int zs, double* G, int gr, int gs, int N, QlScratch& q) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float tn = 0.f;
  for (int i = tid; i < N; i += kEigThreads) {
    const float d = (float)q.d[i], e = (float)q.e[i], ep = i ? (float)q.e[i - 1] : 0.f;
    q.fd[i] = d;
    q.fe[i] = e * e;
    tn = fmaxf(tn, fabsf(d) + fabsf(e) + fabsf(ep));
    if (!(fabsf(d) + fabsf(e) < 1e15f)) tn = INFINITY;
  }
  tn = block_max(tn, q.red);
  if (!(tn > 1e-15f && tn < 1e15f)) return false;
  float gmax = 0.f;
  double lam = 0.0;
  if (tid < N) {
    float lo = -1.001f * tn, hi = 1.001f * tn;
    const float tiny = 1e-12f * tn;
    for (int it = 0; it < 27; ++it) {
      const float x = 0.5f * (lo + hi);
      int below = 0;
      float t = q.fd[0] - x;
      for (int i = 1;; ++i) {
        if (fabsf(t) < tiny) t = -tiny;
        below += t < 0.f;
        if (i == N) break;
        t = (q.fd[i] - x) - __fdividef(q.fe[i - 1], t);
      }
      if (below > tid) hi = x;
      else lo = x;
    }
    q.lam[tid] = lam = 0.5 * ((double)lo + (double)hi);
  }
  __syncthreads();
  // Levels that FP32 does not tell apart come out with one vector (none passed the limits): the QR steps at
  // once.  Pole N(mu) of 300 k-points of 16 spin-degenerate bands 0.82 -> 0.75 ms, 125 of 20 0.95 -> 0.86.
  if (__syncthreads_or(tid > 0 && tid < N && (float)(lam - q.lam[max(tid, 1) - 1]) < kTriNear * tn)) return false;
  if (tid < N) {
    const double small = 1e-18 * (double)tn;
    double* z = Z + tid * zs;
    double* g = G + tid * gs;
    const long long small_bits = __double_as_longlong(small), mask = 0x7fffffffffffffffLL;
    for (int it = 0; it < 3; ++it) {
      // multipliers from above, l_i = e_i / t_i, and from below, m_i = e_i / u_{i+1}, side by side
      double t = q.d[0] - lam, u = q.d[N - 1] - lam;
      for (int i = 0; i + 1 < N; ++i) {
        const int j = N - 2 - i;
        if ((__double_as_longlong(t) & mask) < small_bits) t = small;
        if ((__double_as_longlong(u) & mask) < small_bits) u = small;
        const double l = q.e[i] * rcp_newton(t), m = q.e[j] * rcp_newton(u);
        z[i * zr] = l;
        g[j * gr] = m;
        t = fma(-q.e[i], l, q.d[i + 1] - lam);
        u = fma(-q.e[j], m, q.d[j] - lam);
      }
      // the twist: the row of the smallest gamma_i = t_i - e_i m_i
      double gam = t, el = 0.0;
      int r = N - 1;
      long long best = __double_as_longlong(t) & mask;
      for (int i = 0; i + 1 < N; ++i) {
        const double v = fma(-q.e[i], g[i * gr], (q.d[i] - lam) - el);
        el = q.e[i] * z[i * zr];
        const long long key = __double_as_longlong(v) & mask;
        if (key < best) {
          best = key;
          gam = v;
          r = i;
        }
      }
      // the vector, from the twist in both directions
      double n0 = 1.0, n1 = 0.0, x = 1.0, y = 1.0;
      z[r * zr] = 1.0;
      for (int s = 1; s < N; ++s) {
        const int iu = r - s, id = r + s;
        if (iu < 0 && id >= N) break;
        if (iu >= 0) {
          x *= -z[iu * zr];
          z[iu * zr] = x;
          n0 = fma(x, x, n0);
        }
        if (id < N) {
          y *= -g[(id - 1) * gr];
          z[id * zr] = y;
          n1 = fma(y, y, n1);
        }
      }
      const double nrm = n0 + n1;
      lam += gam / nrm;
      if (it == 2) {
        const double s = rsqrt(nrm);
        gmax = (kTriOrth / kTriRes) * (float)(fabs(gam) * s) / tn;
        for (int i = 0; i < N; ++i) z[i * zr] *= s;
      }
    }
    q.lam[tid] = lam;
  }
  __syncthreads();
  // G = Z^T Z - I (lower triangle and its mirror), its largest entry
  gmax = gmax == gmax ? gmax : INFINITY;
  for (int x = tid; x < N * (N + 1) / 2; x += kEigThreads) {
    int a, b;
    tri_pair(x, a, b);
    double s0 = a == b ? -1.0 : 0.0, s1 = 0.0;
    int i = 0;
    for (; i + 1 < N; i += 2) {
      s0 = fma(Z[i * zr + a * zs], Z[i * zr + b * zs], s0);
      s1 = fma(Z[(i + 1) * zr + a * zs], Z[(i + 1) * zr + b * zs], s1);
    }
    if (i < N) s0 = fma(Z[i * zr + a * zs], Z[i * zr + b * zs], s0);
    s0 += s1;
    G[a * gr + b * gs] = s0;
    G[b * gr + a * gs] = s0;
    const float f = fabsf((float)s0);
    gmax = fmaxf(gmax, f == f ? f : INFINITY);
  }
  gmax = block_max(gmax, q.red);
  if (!(gmax < kTriOrth)) return false;
  // Z -= Z G / 2, one row per warp
  for (int r = warp; r < N; r += kEigThreads / 32) {
    double* zp = Z + r * zr;
    double out[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int c = lane + 32 * t;
      if (c - lane >= N) break;
      double s0 = 0.0, s1 = 0.0;
      if (c < N) {
        int k = 0;
        for (; k + 1 < N; k += 2) {
          s0 = fma(zp[k * zs], G[k * gr + c * gs], s0);
          s1 = fma(zp[(k + 1) * zs], G[(k + 1) * gr + c * gs], s1);
        }
        if (k < N) s0 = fma(zp[k * zs], G[k * gr + c * gs], s0);
        out[t] = fma(-0.5, s0 + s1, zp[c * zs]);
      }
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int c = lane + 32 * t;
      if (c < N) zp[c * zs] = out[t];
    }
  }
  __syncthreads();
  for (int i = tid; i < N; i += kEigThreads) q.d[i] = q.lam[i];
  __syncthreads();
  return true;
}

// Implicit QR steps with Wilkinson's shift on the tridiagonal matrix (Golub and Van Loan, Matrix
// Computations, section 8.3), rotations applied to Z (the identity on entry).  One lane of warp 0
// forms the rotations of a sweep while the other warps apply the previous sweep's.  An off-diagonal entry
// below the rounding of the norm is dropped, since the reduction to tridiagonal form loses as much: with
// two or three distinct levels whole blocks of T lie below it, and compared with their own entries the last
// level waits for all others (of 68 up to 39 steps, of 138 up to 74; like this at most 12 of 250).  Returns false
// when an eigenvalue takes more than 100 steps (non-finite input does).
__device__ bool tri_qr(double* Z, int zr, int zs, int N, QlScratch& q) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int x = tid; x < N * N; x += kEigThreads) {
    const int i = x / N, l = x - i * N;
    Z[i * zr + l * zs] = i == l ? 1.0 : 0.0;
  }
  if (tid == 0) {
    q.more = 1;
    q.failed = 0;
    q.lo[1] = q.hi[1] = 0;  // no sweep to apply yet
  }
  __syncthreads();
  int hi = N - 1, steps = 0;  // warp 0: end of the active block, steps spent on its eigenvalue
  double tiny = 0.0;          // and the rounding of the norm
  if (warp == 0) {
    for (int i = lane; i < N; i += 32)
      tiny = fmax(tiny, fabs(q.d[i]) + fabs(q.e[i]) + (i ? fabs(q.e[i - 1]) : 0.0));
    for (int off = 16; off; off >>= 1) tiny = fmax(tiny, __shfl_xor_sync(0xffffffffu, tiny, off));
    tiny *= 1.2e-16;
  }
  for (int t = 0;; ++t) {
    const int b = t & 1;
    if (warp == 0) {
      // deflate: the largest unreduced block that ends at hi
      int lo = 0;
      for (;;) {
        int last = -1;  // last negligible off-diagonal entry below hi
        for (int i = lane; i < hi; i += 32)
          if (fabs(q.e[i]) <= tiny) last = i;
        last = __reduce_max_sync(0xffffffffu, last);
        lo = last + 1;
        if (lo < hi || hi <= 0) break;
        --hi;
        steps = 0;
      }
      if (lane == 0) {
        q.lo[b] = q.hi[b] = 0;
        if (hi <= 0) {
          q.more = 0;
        } else if (++steps > 100) {
          q.failed = 1;
          q.more = 0;
        } else {
          q.lo[b] = lo;
          q.hi[b] = hi;
          double* d = q.d;
          double* e = q.e;
          const double dl = 0.5 * (d[hi - 1] - d[hi]), eb = e[hi - 1];
          const double den = dl + copysign(sqrt(fma(dl, dl, eb * eb)), dl);
          double x = d[lo] - (d[hi] - (den != 0.0 ? eb * eb / den : 0.0)), z = e[lo];
          double a = d[lo], ek = e[lo];
          for (int k = lo; k < hi; ++k) {
            const double g = d[k + 1], en = e[k + 1];
            const double r2 = fma(x, x, z * z);
            double c = 1.0, s = 0.0;
            if (r2 > 0.0) {
              const double ir = rsqrt(r2);
              c = x * ir;
              s = z * ir;
              if (k > lo) e[k - 1] = r2 * ir;
            } else if (k > lo) {
              e[k - 1] = 0.0;
            }
            // [a ek; ek g] under the rotation, with h = s (g - a) + 2 c ek
            const double h = fma(s, g - a, 2.0 * c * ek), pp = s * h;
            d[k] = a + pp;
            x = fma(c, h, -ek);
            z = s * en;
            a = g - pp;
            ek = c * en;
            e[k] = x;
            q.rot[b][k] = make_double2(c, s);
          }
          d[hi] = a;
        }
      }
      __syncwarp();
    } else {
      // apply the previous sweep to the columns of Z, one row per thread
      const int l0 = q.lo[b ^ 1], h0 = q.hi[b ^ 1];
      for (int r = tid - 32; r < N && l0 < h0; r += kEigThreads - 32) {
        double* zp = Z + r * zr;
        double z0 = zp[l0 * zs];
        for (int k = l0; k < h0; ++k) {
          const double2 cs = q.rot[b ^ 1][k];
          const double z1 = zp[(k + 1) * zs];
          zp[k * zs] = fma(cs.x, z0, cs.y * z1);
          z0 = fma(cs.x, z1, -cs.y * z0);
        }
        zp[h0 * zs] = z0;
      }
    }
    __syncthreads();
    if (!q.more && q.lo[b] >= q.hi[b]) break;
  }
  return !q.failed;
}

// Eigenpairs of the Hermitian N x N matrix A (row-major, leading dimension ld, both triangles):
// Householder reduction to tridiagonal form, the eigenpairs of that, and the back-transformation.
// On return the diagonal of A holds the eigenvalues (as complex numbers) and V the eigenvectors as
// columns.  Z: real N x N scratch (row stride zr, element step zs), G another; both may lie over V
// (its real and its imaginary parts).  Returns false when the QR steps fail.
//
// With nr >= 0 only the rows [r0, r0 + nr) of the eigenvectors are wanted (2 nr <= N): they are left
// in the first nr rows of A, the eigenvalues in q.d, and V is scratch.  The reflectors are then
// applied to those rows of the identity, and the result to Z: 6 nr N^2 FMAs instead of 4 N^3.
//
// About 12 N^3 FP64 FMAs against 18 N^3 per sweep and eight sweeps of cyclic Jacobi.
__device__ bool heev_tri(double2* A, double2* V, double* Z, int zr, int zs, double* G, int gr, int gs, int N, int ld,
                         QlScratch& q, int r0 = 0, int nr = -1) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kW = kEigThreads / 32;
  // a matrix that is diagonal already (to 1e-15 of its norm): no work
  double off = 0.0, dia = 0.0;
  for (int x = tid; x < N * N; x += kEigThreads) {
    const int i = x / N, j = x - i * N;
    const double2 a = A[i * ld + j];
    const double s = fma(a.x, a.x, a.y * a.y);
    if (i == j) dia += s;
    else off += s;
  }
  off = eig_block_sum(off, &q.tau[0]);
  dia = eig_block_sum(dia, &q.tau[0]);
  if (off <= 1e-30 * (off + dia)) {
    for (int i = tid; i < N; i += kEigThreads) q.d[i] = A[i * ld + i].x;
    __syncthreads();
    for (int x = tid; x < nr * N; x += kEigThreads) {
      const int r = x / N, l = x - r * N;
      A[r * ld + l] = make_double2(r0 + r == l ? 1.0 : 0.0, 0.0);
    }
    for (int x = tid; x < N * N && nr < 0; x += kEigThreads) {
      const int i = x / N, l = x - i * N;
      V[i * ld + l] = make_double2(i == l ? 1.0 : 0.0, 0.0);
    }
    __syncthreads();
    return true;
  }
  for (int k = 0; k + 2 < N; ++k) {
    const int len = N - 1 - k;
    // tl lanes per row, consecutive rows per warp: as many lanes as the rows leave
    const int rpw = (len + kW - 1) / kW, tl = 32 / rpw;
    const int sub = lane % tl, rw = lane / tl < rpw ? warp * rpw + lane / tl : len;
    if (warp == 0) {
      double s = 0.0;
      for (int i = lane; i < len; i += 32) {
        const double2 x = A[(k + 1 + i) * ld + k];
        q.v[i] = x;
        s = fma(x.x, x.x, fma(x.y, x.y, s));
      }
      for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      __syncwarp();
      // (every lane the same: an FP64 instruction costs a lane as much as a warp)
      const double2 x0 = q.v[0];
      const double a2 = fma(x0.x, x0.x, x0.y * x0.y);
      const double inx = s > 0.0 ? rsqrt(s) : 0.0, iax = a2 > 0.0 ? rsqrt(a2) : 0.0;
      const double nx = s * inx, ax = a2 * iax;
      const double2 ph = a2 > 0.0 ? make_double2(x0.x * iax, x0.y * iax) : make_double2(1.0, 0.0);
      const double tau = s > 0.0 ? 1.0 / fma(nx, ax, s) : 0.0;
      __syncwarp();
      if (lane == 0) {
        q.v[0] = make_double2(fma(ph.x, nx, x0.x), fma(ph.y, nx, x0.y));
        q.tau[k] = tau;
        q.e[k] = nx;
        q.ph[k + 1] = make_double2(-ph.x, -ph.y);  // phase of the off-diagonal entry
      }
    }
    __syncthreads();
    const double tau = q.tau[k];
    // p = tau A v from the lower triangle
    {
      const int i = rw;
      double2 a0 = make_double2(0.0, 0.0), a1 = a0;
      if (i < len) {
        const double2* Ar = A + (k + 1 + i) * ld + k + 1;
        int c = sub;
        for (; c + tl <= i; c += 2 * tl) {
          cmac(a0, Ar[c], q.v[c]);
          cmac(a1, Ar[c + tl], q.v[c + tl]);
        }
        for (; c <= i; c += tl) cmac(a0, Ar[c], q.v[c]);
        const double2* Ac = A + (k + 1) * ld + k + 1 + i;
        for (; c < len; c += tl) cmac_ca(a1, Ac[c * ld], q.v[c]);
      }
      a0.x += a1.x;
      a0.y += a1.y;
      for (int off = 1; off < tl; off <<= 1) {
        const double bx = __shfl_down_sync(0xffffffffu, a0.x, off), by = __shfl_down_sync(0xffffffffu, a0.y, off);
        if (sub + off < tl) {
          a0.x += bx;
          a0.y += by;
        }
      }
      if (sub == 0 && i < len) q.p[i] = make_double2(tau * a0.x, tau * a0.y);
    }
    __syncthreads();
    // w = p - (tau / 2) (v^+ p) v
    if (warp == 0) {
      double s = 0.0;
      for (int i = lane; i < len; i += 32) s = fma(q.v[i].x, q.p[i].x, fma(q.v[i].y, q.p[i].y, s));
      for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      s *= -0.5 * tau;
      for (int i = lane; i < len; i += 32) {
        const double2 v = q.v[i];
        q.p[i].x = fma(s, v.x, q.p[i].x);
        q.p[i].y = fma(s, v.y, q.p[i].y);
      }
    }
    __syncthreads();
    // lower triangle: A -= v w^+ + w v^+, rows i and len - 1 - i together, so that all lanes have
    // len + 1 entries; column k keeps v for the back-transformation
    {
      const int half = (len + 1) / 2, ppw = (half + kW - 1) / kW, tp = 32 / ppw;
      const int i = warp * ppw + lane / tp, i2 = len - 1 - i, sp = lane % tp;
      if (lane / tp < ppw && i < half) {
        const double2 va = q.v[i], wa = q.p[i], vb = q.v[i2], wb = q.p[i2];
        double2* Ar = A + (k + 1 + i) * ld + k + 1;
        double2* Br = A + (k + 1 + i2) * ld + k + 1;
        if (sp == 0) {
          Ar[-1] = va;
          Br[-1] = vb;
        }
        const int end = i == i2 ? i + 1 : len + 1;
        for (int x = sp; x < end; x += tp) {
          const bool first = x <= i;
          const int c = first ? x : x - i - 1;
          const double2 vi = first ? va : vb, wi = first ? wa : wb;
          double2* at = (first ? Ar : Br) + c;
          const double2 v = q.v[c], w = q.p[c];
          double2 a = *at;
          a.x = fma(-vi.x, w.x, fma(-vi.y, w.y, fma(-wi.x, v.x, fma(-wi.y, v.y, a.x))));
          a.y = fma(-vi.y, w.x, fma(vi.x, w.y, fma(-wi.y, v.x, fma(wi.x, v.y, a.y))));
          *at = a;
        }
      }
    }
    __syncthreads();
  }
  for (int i = tid; i < N; i += kEigThreads) q.d[i] = A[i * ld + i].x;
  if (tid == 0) {
    if (N > 1) {
      const double2 x = A[(N - 1) * ld + N - 2];
      const double ax = sqrt(fma(x.x, x.x, x.y * x.y));
      q.e[N - 2] = ax;
      q.ph[N - 1] = ax > 0.0 ? make_double2(x.x / ax, x.y / ax) : make_double2(1.0, 0.0);
    }
    q.e[N - 1] = 0.0;
    // T = D T_real D^+: running products of the phases
    q.ph[0] = make_double2(1.0, 0.0);
    for (int i = 1; i < N; ++i) q.ph[i] = cmul(q.ph[i], q.ph[i - 1]);
  }
  __syncthreads();
  bool ok = N > 3 && tri_eig(Z, zr, zs, G, gr, gs, N, q);
  if (!ok) ok = tri_qr(Z, zr, zs, N, q);
  __syncthreads();
  if (nr >= 0) {
    // L = (rows of the identity) H_0 H_1 ..., its parts in the first 2 nr rows of G, tl lanes per row
    for (int x = tid; x < nr * N; x += kEigThreads) {
      const int r = x / N, c = x - r * N;
      G[r * gr + c * gs] = r0 + r == c ? 1.0 : 0.0;
      G[(nr + r) * gr + c * gs] = 0.0;
    }
    __syncthreads();
    const int rpw = max(1, (nr + kW - 1) / kW), tl = 32 / rpw;
    const int sub = lane % tl, base = lane - sub, r = warp * rpw + lane / tl;
    const bool on = lane / tl < rpw && r < nr;
    double* Lr = G + (on ? r : 0) * gr;
    double* Li = Lr + nr * gr;
    for (int k = 0; k + 2 < N; ++k) {
      const double2* v = A + (k + 1) * ld + k;
      const int len = N - 1 - k;
      double2 s0 = make_double2(0.0, 0.0), s1 = s0;
      if (on) {
        int i = sub;
        for (; i + tl < len; i += 2 * tl) {
          cmac(s0, make_double2(Lr[(k + 1 + i) * gs], Li[(k + 1 + i) * gs]), v[i * ld]);
          cmac(s1, make_double2(Lr[(k + 1 + i + tl) * gs], Li[(k + 1 + i + tl) * gs]), v[(i + tl) * ld]);
        }
        for (; i < len; i += tl) cmac(s0, make_double2(Lr[(k + 1 + i) * gs], Li[(k + 1 + i) * gs]), v[i * ld]);
      }
      s0.x += s1.x;
      s0.y += s1.y;
      for (int off = 1; off < tl; off <<= 1) {
        const double bx = __shfl_down_sync(0xffffffffu, s0.x, off), by = __shfl_down_sync(0xffffffffu, s0.y, off);
        if (sub + off < tl) {
          s0.x += bx;
          s0.y += by;
        }
      }
      const double tau = q.tau[k];
      s0.x = tau * __shfl_sync(0xffffffffu, s0.x, base);
      s0.y = tau * __shfl_sync(0xffffffffu, s0.y, base);
      if (on)
        for (int i = sub; i < len; i += tl) {  // L -= s v^+
          const double2 vv = v[i * ld];
          double* lr = Lr + (k + 1 + i) * gs;
          double* li = Li + (k + 1 + i) * gs;
          *lr = fma(-s0.x, vv.x, fma(-s0.y, vv.y, *lr));
          *li = fma(-s0.y, vv.x, fma(s0.x, vv.y, *li));
        }
      __syncwarp();
    }
    if (on)
      for (int c = sub; c < N; c += tl) {
        const double2 x = cmul(make_double2(Lr[c * gs], Li[c * gs]), q.ph[c]);
        Lr[c * gs] = x.x;
        Li[c * gs] = x.y;
      }
    __syncthreads();
    for (int x = tid; x < nr * N; x += kEigThreads) {
      const int a = x / N, l = x - a * N;
      const double *ar = G + a * gr, *ai = ar + nr * gr;
      double2 s0 = make_double2(0.0, 0.0), s1 = s0;
      int c = 0;
      for (; c + 1 < N; c += 2) {
        const double z0 = Z[c * zr + l * zs], z1 = Z[(c + 1) * zr + l * zs];
        s0.x = fma(ar[c * gs], z0, s0.x);
        s0.y = fma(ai[c * gs], z0, s0.y);
        s1.x = fma(ar[(c + 1) * gs], z1, s1.x);
        s1.y = fma(ai[(c + 1) * gs], z1, s1.y);
      }
      if (c < N) {
        const double z0 = Z[c * zr + l * zs];
        s0.x = fma(ar[c * gs], z0, s0.x);
        s0.y = fma(ai[c * gs], z0, s0.y);
      }
      A[a * ld + l] = make_double2(s0.x + s1.x, s0.y + s1.y);
    }
    __syncthreads();
    return ok;
  }
  // V = H_0 H_1 ... D Z: phases, then the reflectors in reverse order, tl lanes per column
  for (int x = tid; x < N * N; x += kEigThreads) {
    const int i = x / N, l = x - i * N;
    const double z = Z[i * zr + l * zs];
    V[i * ld + l] = make_double2(q.ph[i].x * z, q.ph[i].y * z);
  }
  __syncthreads();
  const int cpw = (N + kW - 1) / kW, tl = 32 / cpw;  // consecutive columns per warp (N <= 256)
  const int sub = lane % tl, base = lane - sub;
  const int l = warp * cpw + lane / tl;
  const bool on = lane / tl < cpw && l < N;
  for (int k = N - 3; k >= 0; --k) {
    const double2* v = A + (k + 1) * ld + k;
    const int len = N - 1 - k;
    double2 s0 = make_double2(0.0, 0.0), s1 = s0;
    if (on) {
      int i = sub;
      for (; i + tl < len; i += 2 * tl) {
        cmac_ca(s0, v[i * ld], V[(k + 1 + i) * ld + l]);
        cmac_ca(s1, v[(i + tl) * ld], V[(k + 1 + i + tl) * ld + l]);
      }
      for (; i < len; i += tl) cmac_ca(s0, v[i * ld], V[(k + 1 + i) * ld + l]);
    }
    s0.x += s1.x;
    s0.y += s1.y;
    for (int off = 1; off < tl; off <<= 1) {
      const double bx = __shfl_down_sync(0xffffffffu, s0.x, off), by = __shfl_down_sync(0xffffffffu, s0.y, off);
      if (sub + off < tl) {
        s0.x += bx;
        s0.y += by;
      }
    }
    const double tau = q.tau[k];
    s0.x = tau * __shfl_sync(0xffffffffu, s0.x, base);
    s0.y = tau * __shfl_sync(0xffffffffu, s0.y, base);
    if (on)
      for (int i = sub; i < len; i += tl) {
        const double2 vv = v[i * ld];
        double2 u = V[(k + 1 + i) * ld + l];
        u.x = fma(-vv.x, s0.x, fma(vv.y, s0.y, u.x));
        u.y = fma(-vv.x, s0.y, fma(-vv.y, s0.x, u.y));
        V[(k + 1 + i) * ld + l] = u;
      }
    __syncwarp();
  }
  __syncthreads();
  for (int i = tid; i < N; i += kEigThreads) A[i * ld + i] = make_double2(q.d[i], 0.0);
  __syncthreads();
  return ok;
}

// heev_tri with Z and G over V's real and imaginary parts when the matrices are in shared memory;
// with the matrices in a global slice Z has shared memory of its own when that fits (z_smem).
__device__ __forceinline__ bool heev_tri(double2* A, double2* V, int n, int ld, int in_smem, int z_smem,
                                         unsigned char* smem, QlScratch& q, int r0 = 0, int nr = -1) {
  double* v = reinterpret_cast<double*>(V);
  if (!in_smem && z_smem)
    return heev_tri(A, V, reinterpret_cast<double*>(smem), n | 1, 1, v, n | 1, 1, n, ld, q, r0, nr);
  return heev_tri(A, V, v, 2 * ld, 2, v + 1, 2 * ld, 2, n, ld, q, r0, nr);
}

__device__ __forceinline__ size_t eig_ws_elems(int n) { return (size_t)2 * n * (n | 1); }

// Standalone batched eigensolver: A [mat][n][n] -> w [mat][n] ascending,
// V [mat][n][n] with eigenvector l in column l.
__global__ void __launch_bounds__(kEigThreads)
    k_heev_batched(const double2* __restrict__ Ain, int n_mat, int n, int max_sweeps,
                   double* __restrict__ w_out, double2* __restrict__ v_out, double2* gws,
                   int in_smem, int* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double rot[4 * 128];
  __shared__ double2 ph[128];
  __shared__ double red[kEigThreads / 32];
  const int ld = n | 1;
  double2* A = in_smem ? reinterpret_cast<double2*>(smem_raw) : gws + blockIdx.x * eig_ws_elems(n);
  double2* V = A + (size_t)n * ld;
  for (int mat = blockIdx.x; mat < n_mat; mat += gridDim.x) {
    const double2* src = Ain + (size_t)mat * n * n;
    for (int e = threadIdx.x; e < n * n; e += kEigThreads) {
      const int i = e / n, j = e - (e / n) * n;
      // Hermitian part of the input: (A + A^+)/2
      const double2 a = src[i * n + j], b = src[j * n + i];
      A[i * ld + j] = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
    }
    __syncthreads();
    const int sw = jacobi_heev(A, V, n, ld, max_sweeps, rot, ph, red);
    if (sw < 0 && threadIdx.x == 0) atomicOr(status, 2);
    // ascending order; equal values keep their index order
    for (int i = threadIdx.x; i < n; i += kEigThreads) {
      const double li = A[i * ld + i].x;
      int rank = 0;
      for (int j = 0; j < n; ++j) {
        const double lj = A[j * ld + j].x;
        rank += (lj < li) || (lj == li && j < i);
      }
      w_out[(size_t)mat * n + rank] = li;
      for (int r = 0; r < n; ++r) v_out[(size_t)mat * n * n + (size_t)r * n + rank] = V[r * ld + i];
    }
    __syncthreads();
  }
}

// Pole path, one CTA per k (grid-stride over k): build H_ps(mu), diagonalise,
// and reduce in the epilogue selected by mode:
//   kOcc:  kN[k] = sum_l |Psi_b,l|^2 n_F(E_l - mu),
//          kdN[k] = dN_k/dmu = -sum_{l,l'} |(Psi_b^+ Psi_b)_{l l'}|^2 n_F[1](E_l - mu, E_l' - mu)
//          (the derivative of Tr[Pi_b n_F(H_0 - mu Pi_b)] with the pole block of
//          H_0 unshifted; n_F[1] is the divided difference);
//   kRho:  rho_k = Psi_b diag(n_F) Psi_b^+ and kNc[k] = sum_l |phi_l|^2 n_F;
//   kGloc: E_l and phi_l = P Psi_b,l to eout / phiout for k_pole_gloc.
__global__ void __launch_bounds__(kEigThreads) k_pole_eig(const PoleParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double s_x[256], s_f[256], s_ch[256];
  __shared__ QlScratch ql;
  __shared__ double red[kEigThreads / 32];
  const int tid = threadIdx.x;
  bool all = false;  // a second pass over k with every row of the eigenvectors
  for (int k = blockIdx.x; k < p.n_k;) {
    const KInfo ki = p.kinfo[k];
    const SInfo si = p.sinfo[ki.sys];
    const PInfo pi = p.pinfo[ki.sys];
    const int nb = ki.nb, m = si.m, npl = pi.np, n = nb + npl, ld = n | 1;
    const double mu = p.mu[ki.sys];
    double2* A = p.in_smem ? reinterpret_cast<double2*>(smem_raw) : p.ws + blockIdx.x * p.ws_stride;
    double2* V = A + (size_t)n * ld;
    const double2* H = p.H + ki.offH;
    const double2* P = p.P + ki.offP;
    const double2* Sinf = p.Sinf + si.offSinf;
    const double2* Vp = p.Vp + pi.offV;
    // band block H + P^+ (Sigma_inf P), the product in V (m nb <= n ld when m <= n, else recomputed)
    const bool staged = m <= n;
    if (staged) {
      for (int e = tid; e < m * nb; e += kEigThreads) {
        const int a = e / nb, j = e - a * nb;
        double2 t = make_double2(0.0, 0.0);
        for (int b = 0; b < m; ++b) cmac(t, Sinf[a * m + b], P[b * nb + j]);
        V[e] = t;
      }
      __syncthreads();
    }
    for (int e = tid; e < nb * nb; e += kEigThreads) {
      const int i = e / nb, j = e - (e / nb) * nb;
      double2 acc = H[i * nb + j];
      for (int a = 0; a < m; ++a) {
        double2 t = make_double2(0.0, 0.0);
        if (staged) t = V[a * nb + j];
        else
          for (int b = 0; b < m; ++b) cmac(t, Sinf[a * m + b], P[b * nb + j]);
        cmac_ca(acc, P[a * nb + i], t);
      }
      A[i * ld + j] = acc;
    }
    // pole rows/columns W_i = V_i P and the pole diagonal p_i + mu
    for (int e = tid; e < npl * nb; e += kEigThreads) {
      const int i = e / nb, b = e - (e / nb) * nb;
      double2 w = make_double2(0.0, 0.0);
      for (int a = 0; a < m; ++a) cmac(w, Vp[i * m + a], P[a * nb + b]);
      A[(nb + i) * ld + b] = w;
      A[b * ld + nb + i] = make_double2(w.x, -w.y);
    }
    for (int e = tid; e < npl * npl; e += kEigThreads) {
      const int i = e / npl, j = e - (e / npl) * npl;
      A[(nb + i) * ld + nb + j] = make_double2(i == j ? p.poles[pi.offp + i] + mu : 0.0, 0.0);
    }
    __syncthreads();
    // N(mu) needs Psi_b^+ Psi_b = 1 - Psi_p^+ Psi_p only: the pole rows, where they are the fewer
    // (125 k-points of 40 bands and 28 poles 1.42 ms, all rows 1.64 ms), unless the difference loses
    // digits: N_k far below the number of occupied pole levels (at N_k = 5e-5 of it 5e-12, all rows 2e-14)
    const bool few = p.mode == kOcc && npl <= nb && !all;
    const bool ok = heev_tri(A, V, n, ld, p.in_smem, p.z_smem, smem_raw, ql, nb, few ? npl : -1);
    if (!ok && tid == 0) atomicOr(p.status, 2);
    // per eigenpair: x_l = E_l - mu, n_F(x_l), cosh(beta x_l / 2)
    for (int l = tid; l < n; l += kEigThreads) {
      const double x = (few ? ql.d[l] : A[l * ld + l].x) - mu;
      s_x[l] = x;
      s_f[l] = fermi(x, si.beta);
      s_ch[l] = cosh(0.5 * si.beta * x);
    }
    __syncthreads();
    if (p.mode & kOcc) {
      const double2* W = few ? A : V;
      const int nw = few ? npl : nb;
      double nk = 0.0;
      for (int l = tid; l < n; l += kEigThreads) {
        double wb = 0.0;
        for (int b = 0; b < nw; ++b) {
          const double2 v = W[b * ld + l];
          wb = fma(v.x, v.x, fma(v.y, v.y, wb));
        }
        nk = fma(few ? 1.0 - wb : wb, s_f[l], nk);
      }
      nk = eig_block_sum(nk, red);
      if (few && !(nk >= 0.0625 * npl)) {
        all = true;
        continue;
      }
      double dk = 0.0;
      for (int e = tid; e < n * (n + 1) / 2; e += kEigThreads) {
        int l, l2;
        tri_pair(e, l, l2);
        double2 o = make_double2(few && l == l2 ? -1.0 : 0.0, 0.0);  // (its modulus is wanted)
        for (int b = 0; b < nw; ++b) cmac_ca(o, W[b * ld + l], W[b * ld + l2]);
        const double f1 =
            fermi_divdiff(s_x[l], s_x[l2], s_f[l], s_f[l2], s_ch[l], s_ch[l2], si.beta);
        dk = fma((l == l2 ? -1.0 : -2.0) * (o.x * o.x + o.y * o.y), f1, dk);
      }
      dk = eig_block_sum(dk, red);
      if (tid == 0) {
        p.kN[k] = nk;
        p.kdN[k] = dk;
      }
    }
    if (p.mode & kRho) {
      double2* rho = p.rho + ki.offH;
      double hks = 0.0;  // Re Tr(H_k rho_k)
      for (int e = tid; e < nb * (nb + 1) / 2; e += kEigThreads) {
        int i, j;
        tri_pair(e, i, j);
        double2 acc = make_double2(0.0, 0.0);
        for (int l = 0; l < n; ++l) {
          const double f = s_f[l];
          double2 vi = V[i * ld + l];
          vi.x *= f;
          vi.y *= f;
          cmac_cb(acc, vi, V[j * ld + l]);
        }
        if (i == j) acc.y = 0.0;
        rho[i * nb + j] = acc;
        const double2 h = H[j * nb + i];
        hks = fma(h.x, acc.x, fma(-h.y, acc.y, hks));
        if (i != j) {
          rho[j * nb + i] = make_double2(acc.x, -acc.y);
          const double2 h2 = H[i * nb + j];
          hks = fma(h2.x, acc.x, fma(h2.y, acc.y, hks));
        }
      }
      double nc = 0.0;
      for (int e = tid; e < m * n; e += kEigThreads) {
        const int a = e / n, l = e - (e / n) * n;
        double2 f = make_double2(0.0, 0.0);
        for (int b = 0; b < nb; ++b) cmac(f, P[a * nb + b], V[b * ld + l]);
        nc = fma(f.x * f.x + f.y * f.y, s_f[l], nc);
      }
      // sum_l (E_l - mu) |Psi_b,l|^2 n_F(E_l - mu)
      double eps = 0.0;
      for (int l = tid; l < n; l += kEigThreads) {
        double wb = 0.0;
        for (int b = 0; b < nb; ++b) {
          const double2 v = V[b * ld + l];
          wb = fma(v.x, v.x, fma(v.y, v.y, wb));
        }
        eps = fma(s_x[l] * wb, s_f[l], eps);
      }
      nc = eig_block_sum(nc, red);
      hks = eig_block_sum(hks, red);
      eps = eig_block_sum(eps, red);
      if (tid == 0) {
        p.kNc[k] = nc;
        if (p.kHks) p.kHks[k] = hks;
        if (p.kEps) p.kEps[k] = eps;
      }
    }
    if (p.mode & kGloc) {
      double* E = p.eout + p.eoff[k];
      double2* phi = p.phiout + p.phioff[k];
      for (int l = tid; l < n; l += kEigThreads) {
        E[l] = A[l * ld + l].x;
        if (p.wbout) {
          double wb = 0.0;
          for (int b = 0; b < nb; ++b) {
            const double2 v = V[b * ld + l];
            wb = fma(v.x, v.x, fma(v.y, v.y, wb));
          }
          p.wbout[p.eoff[k] + l] = wb;
        }
      }
      for (int e = tid; e < m * n; e += kEigThreads) {
        const int a = e / n, l = e - (e / n) * n;
        double2 f = make_double2(0.0, 0.0);
        for (int b = 0; b < nb; ++b) cmac(f, P[a * nb + b], V[b * ld + l]);
        phi[a * n + l] = f;
      }
    }
    __syncthreads();
    all = false;
    k += gridDim.x;
  }
}

// G_loc(i w_n) = sum_k w_k sum_l t_l / (i w_n + mu - E_l), t = phi_a conj(phi_b), of one system.
// Frequencies below nd are summed as they stand: with g = w_k / (i w + mu - E) = gr + i gi,
// G_ab = Xr + i Xi and G_ba = conj(Xr) + i conj(Xi) with Xr = sum t gr, Xi = sum t gi.  From nd
// on 1 / (z - E) is a Chebyshev series in E over the interval of the levels, whose moments
// sum_k w_k sum_l t_l T_j(x_l), j < J, serve all of them: a moment costs half a frequency's sum.
// A tile is F frequencies or 2 F moments of all pairs a <= b, QP pairs per thread; a CTA sums one
// tile over a share of the system's levels (the tiles times their splits fill the chip), phi and
// the factors staged in shared memory kCh levels at a time, in increasing order.
// J is the multiple of 2 F with the fewest tiles: the frequencies whose series of J terms leaves
// less than e^-37 are those with J asinh(w / r) >= 37, r half the width of the interval (a
// frequency's ellipse of convergence is smallest above the middle of the interval).
// Bound: the FP64 pipe.  125 k-points of 68 levels, 14 orbitals, 512 frequencies: 1.1 ms, 6.2 ms by
// sums alone.
constexpr int kCh = 32;
constexpr int kGlocTerms = 256;  // moments kept at most

struct GlocPlan {
  double c, r;         // middle and half width of the levels' interval
  int nd, J, tiles;    // frequencies summed directly, moments, tiles of both
};

__global__ void __launch_bounds__(kEigThreads) k_pole_span(const PoleParams p, int F, GlocPlan* plan) {
  __shared__ double s_lo[kEigThreads], s_hi[kEigThreads];
  const SInfo si = p.sinfo[blockIdx.x];
  const int tid = threadIdx.x;
  const int64_t e0 = p.eoff[si.k0], e1 = p.eoff[si.k1 - 1] + p.kinfo[si.k1 - 1].nb + p.pinfo[blockIdx.x].np;
  double lo = INFINITY, hi = -INFINITY;
  for (int64_t e = e0 + tid; e < e1; e += kEigThreads) {
    const double v = p.eout[e];
    lo = fmin(lo, v);
    hi = fmax(hi, v);
  }
  s_lo[tid] = lo;
  s_hi[tid] = hi;
  __syncthreads();
  for (int w = kEigThreads / 2; w; w >>= 1) {
    if (tid < w) {
      s_lo[tid] = fmin(s_lo[tid], s_lo[tid + w]);
      s_hi[tid] = fmax(s_hi[tid], s_hi[tid + w]);
    }
    __syncthreads();
  }
  if (tid >= 32) return;
  lo = s_lo[0];
  hi = s_hi[0];
  const double r = fmax(0.5 * (hi - lo) * (1.0 + 1e-12), 1e-6);
  // one candidate J per lane, J = 0 (every frequency as it stands) in lane 0
  int best = (p.n_iw + F - 1) / F, nd = p.n_iw, J = 0;
  for (int j = 2 * F * (tid + 1); j <= kGlocTerms; j += 2 * F * 32) {
    const double n = ceil(0.5 * (r * sinh(37.0 / j) * si.beta / M_PI - 1.0));
    if (!(n < (double)p.n_iw)) continue;  // (also an interval that is not finite)
    const int d = (int)fmax(n, 0.0), t = (d + F - 1) / F + j / (2 * F);
    if (t < best) {
      best = t;
      nd = d;
      J = j;
    }
  }
  for (int off = 16; off; off >>= 1) {
    const int ot = __shfl_xor_sync(0xffffffffu, best, off), on = __shfl_xor_sync(0xffffffffu, nd, off);
    const int oj = __shfl_xor_sync(0xffffffffu, J, off);
    if (ot < best || (ot == best && oj < J)) {
      best = ot;
      nd = on;
      J = oj;
    }
  }
  if (tid == 0) plan[blockIdx.x] = GlocPlan{0.5 * (hi + lo), r, nd, J, best};
}

// Sums of one (tile, split): part[blockIdx.x 2 F + slot][pair], slot 2 f of Xr and
// 2 f + 1 of Xi, or the moment of the tile.
template <int QP, int F>
__global__ void __launch_bounds__(kEigThreads)
    k_pole_gloc(const PoleParams p, const GlocPlan* plan, int per_sys, int nps_max, int npairs_max, double2* part) {
  __shared__ double2 s_phi[32 * kCh];  // m <= 32
  __shared__ double2 s_g[F * kCh];     // w_k / (i w + mu - E), or w_k T_j: [2 F][kCh]
  __shared__ double s_th[kCh];
  const int s = blockIdx.x / per_sys, item = blockIdx.x % per_sys;
  const GlocPlan pl = plan[s];
  const int splits = max(1, per_sys / pl.tiles);
  if (item >= pl.tiles * splits) return;
  const int tile = item % pl.tiles, split = item / pl.tiles;
  const int td = (pl.nd + F - 1) / F;
  const bool mom = tile >= td;
  const int f0 = tile * F, j0 = (tile - td) * 2 * F;
  const SInfo si = p.sinfo[s];
  const int m = si.m, np = p.pinfo[s].np;
  const int npairs = m * (m + 1) / 2;
  const double mu = p.mu[s], ir = 1.0 / pl.r;
  const int tid = threadIdx.x, nt = blockDim.x;
  int pa[QP], pb[QP];
#pragma unroll
  for (int q = 0; q < QP; ++q) {
    int rem = tid + q * nt, a = 0;
    if (rem >= npairs) rem = 0;
    while (rem >= m - a) { rem -= m - a; ++a; }
    pa[q] = a;
    pb[q] = a + rem;
  }
  double2 x[QP][2 * F];
#pragma unroll
  for (int q = 0; q < QP; ++q)
#pragma unroll
    for (int f = 0; f < 2 * F; ++f) x[q][f] = make_double2(0.0, 0.0);
  // chunks of levels, nch per k-point, [ca, cb) of this split
  const int nch = (nps_max + kCh - 1) / kCh;
  const int64_t tot = (int64_t)(si.k1 - si.k0) * nch;
  const int64_t ca = tot * split / splits, cb = tot * (split + 1) / splits;
  for (int64_t ch = ca; ch < cb; ++ch) {
    const int k = si.k0 + (int)(ch / nch), i = (int)(ch % nch);
    const int n = p.kinfo[k].nb + np;
    const int l0 = n * i / nch, cl = n * (i + 1) / nch - l0;
    const double wk = p.kinfo[k].w;
    const double* E = p.eout + p.eoff[k] + l0;
    const double2* phi = p.phiout + p.phioff[k] + l0;
    __syncthreads();
    for (int e = tid; e < m * cl; e += nt) {
      const int a = e / cl, l = e - (e / cl) * cl;
      s_phi[a * kCh + l] = phi[a * n + l];
    }
    if (mom) {
      if (tid < cl) {
        const double t = (E[tid] - pl.c) * ir;
        s_th[tid] = acos(t > 1.0 ? 1.0 : (t < -1.0 ? -1.0 : t));
      }
      __syncthreads();
      double* T = reinterpret_cast<double*>(s_g);
      for (int e = tid; e < 2 * F * cl; e += nt) {
        const int j = e / cl, l = e - (e / cl) * cl;
        T[j * kCh + l] = wk * cos((j0 + j) * s_th[l]);
      }
    } else {
      for (int e = tid; e < F * cl; e += nt) {
        const int f = e / cl, l = e - (e / cl) * cl;
        const double wn = (2.0 * (f0 + f) + 1.0) * 3.14159265358979323846 / si.beta;
        // w_k / (mu - E + i w) = w_k (x - i w) / (x^2 + w^2), x = mu - E
        const double xe = mu - E[l];
        const double d = wk / fma(xe, xe, wn * wn);
        s_g[f * kCh + l] = make_double2(xe * d, -wn * d);
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < QP; ++q) {
      if (tid + q * nt >= npairs) continue;
      const int a = pa[q], b = pb[q];
      const double* T = reinterpret_cast<const double*>(s_g);
      for (int l = 0; l < cl; ++l) {
        double2 t = make_double2(0.0, 0.0);
        cmac_cb(t, s_phi[a * kCh + l], s_phi[b * kCh + l]);
        if (mom) {
#pragma unroll
          for (int j = 0; j < 2 * F; ++j) {
            const double g = T[j * kCh + l];
            x[q][j].x = fma(t.x, g, x[q][j].x);
            x[q][j].y = fma(t.y, g, x[q][j].y);
          }
        } else {
#pragma unroll
          for (int f = 0; f < F; ++f) {
            const double2 g = s_g[f * kCh + l];
            x[q][2 * f].x = fma(t.x, g.x, x[q][2 * f].x);
            x[q][2 * f].y = fma(t.y, g.x, x[q][2 * f].y);
            x[q][2 * f + 1].x = fma(t.x, g.y, x[q][2 * f + 1].x);
            x[q][2 * f + 1].y = fma(t.y, g.y, x[q][2 * f + 1].y);
          }
        }
      }
    }
  }
  double2* out = part + (int64_t)blockIdx.x * 2 * F * npairs_max;
#pragma unroll
  for (int q = 0; q < QP; ++q) {
    const int pr = tid + q * nt;
    if (pr >= npairs) continue;
#pragma unroll
    for (int f = 0; f < 2 * F; ++f) out[f * npairs_max + pr] = x[q][f];
  }
}

// part of the first split = sum over the splits, in order.
__global__ void k_gloc_splits(const GlocPlan* __restrict__ plan, int blocks_per_sys, int per_sys, int64_t per_tile,
                              double2* part) {
  const int s = blockIdx.x / blocks_per_sys, blk = blockIdx.x % blocks_per_sys;
  const GlocPlan pl = plan[s];
  const int splits = max(1, per_sys / pl.tiles);
  double2* v = part + (int64_t)s * per_sys * per_tile;
  const int64_t tot = pl.tiles * per_tile;
  for (int64_t e = blk * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)blocks_per_sys * blockDim.x) {
    double2 acc = v[e];
    for (int sp = 1; sp < splits; ++sp) {
      const double2 u = v[sp * tot + e];
      acc.x += u.x;
      acc.y += u.y;
    }
    v[e] = acc;
  }
}

// G_loc of one frequency and system from the sums: Xr and Xi as they stand, or
// Xr + i Xi = sum_j c_j M_j with complex c_j and M_ba = conj(M_ab).
__global__ void __launch_bounds__(128) k_gloc_write(const PoleParams p, const GlocPlan* __restrict__ plan, int per_sys,
                                                    int F, int npairs_max, const double2* __restrict__ part) {
  __shared__ double2 s_c[kGlocTerms];
  const int s = blockIdx.x / p.n_iw, n = blockIdx.x % p.n_iw, tid = threadIdx.x;
  const GlocPlan pl = plan[s];
  const SInfo si = p.sinfo[s];
  const int m = si.m, td = (pl.nd + F - 1) / F;
  const double2* v = part + (int64_t)s * per_sys * 2 * F * npairs_max;
  if (n >= pl.nd) {
    const double wn = (2.0 * n + 1.0) * 3.14159265358979323846 / si.beta;
    const series::SeriesZ z = series::series_z(p.mu[s] - pl.c, wn, pl.r, false);
    for (int j = tid; j < pl.J; j += 128) {
      const double2 c = cmul(series::cpow_int<8>(z.xi, j), z.c1);
      s_c[j] = j ? make_double2(2.0 * c.x, 2.0 * c.y) : c;
    }
  }
  __syncthreads();
  double2* out = p.gloc + si.offSig + (int64_t)n * m * m;
  for (int pr = tid; pr < m * (m + 1) / 2; pr += 128) {
    int b = pr, a = 0;
    while (b >= m - a) { b -= m - a; ++a; }
    b += a;
    double2 xr = make_double2(0.0, 0.0), xi = xr;  // sums of t with the real and imaginary parts
    if (n < pl.nd) {
      const double2* u = v + ((int64_t)(n / F) * 2 * F + 2 * (n % F)) * npairs_max + pr;
      xr = u[0];
      xi = u[npairs_max];
    } else {
      const double2* u = v + (int64_t)td * 2 * F * npairs_max + pr;
#pragma unroll 4
      for (int j = 0; j < pl.J; ++j) {
        const double2 t = u[(int64_t)j * npairs_max], c = s_c[j];
        xr.x = fma(t.x, c.x, xr.x);
        xr.y = fma(t.y, c.x, xr.y);
        xi.x = fma(t.x, c.y, xi.x);
        xi.y = fma(t.y, c.y, xi.y);
      }
    }
    out[a * m + b] = make_double2(xr.x - xi.y, xr.y + xi.x);
    out[b * m + a] = make_double2(xr.x + xi.y, xi.x - xr.y);
  }
}

// Low-rank path setup, one CTA per k (grid-stride): H_k = U diag(eps) U^+ by
// Jacobi, then Pt = P_k U.
__global__ void __launch_bounds__(kEigThreads)
    k_lr_setup(const double2* __restrict__ H, const double2* __restrict__ P,
               const KInfo* __restrict__ kinfo, const SInfo* __restrict__ sinfo,
               const int64_t* __restrict__ offD, int n_k, int nbmax, double* __restrict__ eps,
               double2* __restrict__ U, double2* __restrict__ Pt, double2* gws, int in_smem,
               int* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double rot[4 * 128];
  __shared__ double2 ph[128];
  __shared__ double red[kEigThreads / 32];
  double2* A = in_smem ? reinterpret_cast<double2*>(smem_raw) : gws + blockIdx.x * eig_ws_elems(nbmax);
  for (int k = blockIdx.x; k < n_k; k += gridDim.x) {
    const KInfo ki = kinfo[k];
    const int n = ki.nb, m = sinfo[ki.sys].m, ld = n | 1;
    double2* V = A + (size_t)n * ld;
    const double2* Hk = H + ki.offH;
    for (int e = threadIdx.x; e < n * n; e += kEigThreads) {
      const int i = e / n, j = e - (e / n) * n;
      const double2 a = Hk[i * n + j], b = Hk[j * n + i];
      A[i * ld + j] = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
    }
    __syncthreads();
    const int sw = jacobi_heev(A, V, n, ld, 40, rot, ph, red);
    if (sw < 0 && threadIdx.x == 0) atomicOr(status, 2);
    for (int l = threadIdx.x; l < n; l += kEigThreads) eps[offD[k] + l] = A[l * ld + l].x;
    for (int e = threadIdx.x; e < n * n; e += kEigThreads) {
      const int i = e / n, l = e - (e / n) * n;
      U[ki.offH + e] = V[i * ld + l];
    }
    const double2* Pk = P + ki.offP;
    for (int e = threadIdx.x; e < m * n; e += kEigThreads) {
      const int a = e / n, l = e - (e / n) * n;
      double2 acc = make_double2(0.0, 0.0);
      for (int b = 0; b < n; ++b) cmac(acc, Pk[a * n + b], V[b * ld + l]);
      Pt[ki.offP + e] = acc;
    }
    __syncthreads();
  }
}

// Block form: eigenpairs of the n2 x n2 block of every k (D22, replaced by its eigenvectors).
__global__ void __launch_bounds__(kEigThreads)
    k_block_eig(const BlockSetup b, double2* gws, int in_smem, int z_smem) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ QlScratch ql;
  if (*b.flags & ~kBlkNoConvergence) return;  // (other CTAs set that bit meanwhile)
  double2* A = in_smem ? reinterpret_cast<double2*>(smem_raw) : gws + blockIdx.x * eig_ws_elems(b.n2max);
  for (int k = blockIdx.x; k < b.n_k; k += gridDim.x) {
    const KInfo ki = b.kinfo[k];
    const int n = ki.nb - b.sinfo[ki.sys].m, ld = n | 1;
    double2* V = A + (size_t)n * ld;
    double2* D = b.D22 + ki.offH;
    for (int e = threadIdx.x; e < n * n; e += kEigThreads) {
      const int i = e / n, j = e - i * n;
      const double2 x = D[i * n + j], y = D[j * n + i];
      A[i * ld + j] = make_double2(0.5 * (x.x + y.x), 0.5 * (x.y - y.y));
    }
    __syncthreads();
    const bool ok = heev_tri(A, V, n, ld, in_smem, z_smem, smem_raw, ql);
    if (!ok && threadIdx.x == 0) atomicOr(b.flags, kBlkNoConvergence);
    for (int l = threadIdx.x; l < n; l += kEigThreads) b.e[b.offD[k] + l] = A[l * ld + l].x;
    for (int e = threadIdx.x; e < n * n; e += kEigThreads) {
      const int i = e / n, l = e - i * n;
      D[e] = V[i * ld + l];
    }
    __syncthreads();
  }
}

// DOS and PDOS on the real axis from the pseudo-Hamiltonian eigenpairs
// (Eqs. DOS and PDOS) with a Lorentzian of half width eta:
//   D(e)       = sum_k w_k sum_l |Psi_b,l|^2 L(e + mu - E_l),
//   D_alpha(e) = sum_k w_k sum_l |phi_l(alpha)|^2 L(e + mu - E_l),
//   L(x) = (eta / pi) / (x^2 + eta^2) = -(1/pi) Im 1/(x + i eta).
// One thread per energy, kDosT channels (the DOS, then the orbitals) per CTA in registers, the
// weights of 32 eigenpairs staged at a time, the k-points in gridDim.z splits (a grid of 201
// energies alone is two CTAs); part [split][system][energy][1 + mmax], k then l increasing.
constexpr int kDosT = 8, kDosL = 32;
__global__ void __launch_bounds__(128)
    k_pole_dos(const PoleParams p, const double* __restrict__ eps_grid, int n_eps, double eta, int n_ch, int mmax,
               double* __restrict__ part) {
  __shared__ double s_w[kDosL][kDosT], s_e[kDosL];
  const int tiles = (n_eps + 127) / 128;
  const int s = blockIdx.y, ie = (blockIdx.x % tiles) * 128 + threadIdx.x, c0 = (blockIdx.x / tiles) * kDosT;
  const SInfo si = p.sinfo[s];
  const int m = si.m, npl = p.pinfo[s].np, nks = si.k1 - si.k0;
  const int ka = si.k0 + (int)((int64_t)nks * blockIdx.z / gridDim.z);
  const int kb = si.k0 + (int)((int64_t)nks * (blockIdx.z + 1) / gridDim.z);
  const double z = eps_grid[min(ie, n_eps - 1)] + p.mu[s], e2 = eta * eta;
  double acc[kDosT];
#pragma unroll
  for (int t = 0; t < kDosT; ++t) acc[t] = 0.0;
  for (int k = ka; k < kb; ++k) {
    const int n = p.kinfo[k].nb + npl;
    const double wk = p.kinfo[k].w * (eta * 0.31830988618379067);
    const double* E = p.eout + p.eoff[k];
    const double* wb = p.wbout + p.eoff[k];
    const double2* phi = p.phiout + p.phioff[k];
    for (int l0 = 0; l0 < n; l0 += kDosL) {
      const int cl = min(kDosL, n - l0);
      __syncthreads();
      for (int i = threadIdx.x; i < cl * kDosT; i += 128) {
        const int t = i / cl, l = i - t * cl, c = c0 + t;
        double w = 0.0;
        if (c == 0) {
          w = wb[l0 + l];
        } else if (c <= m) {
          const double2 f = phi[(c - 1) * n + l0 + l];
          w = fma(f.x, f.x, f.y * f.y);
        }
        s_w[l][t] = wk * w;
        if (t == 0) s_e[l] = E[l0 + l];
      }
      __syncthreads();
      for (int l = 0; l < cl; ++l) {
        const double x = z - s_e[l], lor = 1.0 / fma(x, x, e2);
#pragma unroll
        for (int t = 0; t < kDosT; ++t) acc[t] = fma(s_w[l][t], lor, acc[t]);
      }
    }
  }
  if (ie >= n_eps) return;
  double* out = part + (((int64_t)blockIdx.z * gridDim.y + s) * n_eps + ie) * (1 + mmax);
#pragma unroll
  for (int t = 0; t < kDosT; ++t)
    if (c0 + t < n_ch && c0 + t <= m) out[c0 + t] = acc[t];
}

// Sums of the splits, in order, to dos [system][energy] and pdos (per system [energy][m], or null).
__global__ void k_dos_reduce(const SInfo* __restrict__ sinfo, const double* __restrict__ part, int n_split, int n_sys,
                             int n_eps, int mmax, const int64_t* __restrict__ pdos_off, double* __restrict__ dos,
                             double* __restrict__ pdos) {
  const int s = blockIdx.y, m = sinfo[s].m, ch = 1 + (pdos ? m : 0);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_eps * ch; i += gridDim.x * blockDim.x) {
    const int ie = i / ch, c = i - ie * ch;
    double v = 0.0;
    for (int z = 0; z < n_split; ++z) v += part[(((int64_t)z * n_sys + s) * n_eps + ie) * (1 + mmax) + c];
    if (c == 0) dos[(int64_t)s * n_eps + ie] = v;
    else pdos[pdos_off[s] + (int64_t)ie * m + c - 1] = v;
  }
}

// Orthonormal projectors of Eqs. 6 and 7 (Lowdin):
// P_k = O^{-1/2} W_k, O = W_k W_k^+ (m x m), one CTA per k.  O's eigenpairs by
// heev_tri; eigenvalues <= tol * max eigenvalue flag the k-point
// (linearly dependent projections).
__global__ void __launch_bounds__(kEigThreads)
    k_lowdin(const KInfo* __restrict__ kinfo, const SInfo* __restrict__ sinfo,
             const double2* __restrict__ Wraw, double2* __restrict__ Pout, int mmax, int* status) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ QlScratch ql;
  __shared__ double s_isq[32];
  const int k = blockIdx.x;
  const KInfo ki = kinfo[k];
  const int N = ki.nb, M = sinfo[ki.sys].m, ld = M | 1;
  double2* O = reinterpret_cast<double2*>(smraw);
  double2* V = O + M * ld;
  double2* T = V + M * ld;  // O^{-1/2}
  const double2* Wk = Wraw + ki.offP;
  for (int e = threadIdx.x; e < M * (M + 1) / 2; e += kEigThreads) {
    int a, b;
    tri_pair(e, a, b);
    double2 acc = make_double2(0.0, 0.0);
    for (int j = 0; j < N; ++j) cmac_cb(acc, Wk[a * N + j], Wk[b * N + j]);
    if (a == b) acc.y = 0.0;
    O[a * ld + b] = acc;
    O[b * ld + a] = make_double2(acc.x, -acc.y);
  }
  __syncthreads();
  const bool ok = heev_tri(O, V, M, ld, 1, 0, smraw, ql);
  if (!ok && threadIdx.x == 0) atomicOr(status, 2);
  if (threadIdx.x < 32) {
    double lmax = 0.0;
    for (int l = 0; l < M; ++l) lmax = fmax(lmax, O[l * ld + l].x);
    for (int l = threadIdx.x; l < M; l += 32) {
      const double lam = O[l * ld + l].x;
      if (!(lam > 1e-12 * lmax)) {
        atomicOr(status, kFlagSingular);
        s_isq[l] = 0.0;
      } else {
        s_isq[l] = 1.0 / sqrt(lam);
      }
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < M * (M + 1) / 2; e += kEigThreads) {
    int a, b;
    tri_pair(e, a, b);
    double2 acc = make_double2(0.0, 0.0);
    for (int l = 0; l < M; ++l) {
      double2 v = V[a * ld + l];
      v.x *= s_isq[l];
      v.y *= s_isq[l];
      cmac_cb(acc, v, V[b * ld + l]);
    }
    T[a * ld + b] = acc;
    T[b * ld + a] = make_double2(acc.x, -acc.y);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < M * N; e += kEigThreads) {
    const int a = e / N, j = e - (e / N) * N;
    double2 acc = make_double2(0.0, 0.0);
    for (int b = 0; b < M; ++b) cmac(acc, T[a * ld + b], Wk[b * N + j]);
    Pout[ki.offP + e] = acc;
  }
}

}  // namespace

// Dynamic shared memory of the real scratch of heev_tri when the matrices are in a global slice
// (0: it takes V's place there); heev_tri's static arrays leave 200 KB.
size_t ql_z_bytes(int n) {
  const size_t z = sizeof(double) * (size_t)n * (n | 1);
  return z <= (200u << 10) ? z : 0;
}

cudaError_t launch_lr_setup(const double2* H, const double2* P, const KInfo* kinfo,
                            const SInfo* sinfo, const int64_t* offD, int n_k, int nbmax,
                            double* eps, double2* U, double2* Pt, double2* ws, int grid,
                            int in_smem, int* status, cudaStream_t s) {
  const size_t smem = in_smem ? heev_smem(nbmax) : 0;
  cudaError_t e =
      cudaFuncSetAttribute(k_lr_setup, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_lr_setup<<<grid, kEigThreads, smem, s>>>(H, P, kinfo, sinfo, offD, n_k, nbmax, eps, U, Pt, ws,
                                             in_smem, status);
  return cudaGetLastError();
}

cudaError_t launch_block_eig(const BlockSetup& b, double2* ws, int grid, int in_smem, cudaStream_t s) {
  const size_t zb = in_smem ? 0 : ql_z_bytes(b.n2max);
  const size_t smem = in_smem ? heev_smem(b.n2max) : zb;
  cudaError_t e = cudaFuncSetAttribute(k_block_eig, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_block_eig<<<grid, kEigThreads, smem, s>>>(b, ws, in_smem, zb > 0);
  return cudaGetLastError();
}

cudaError_t launch_lowdin(const KInfo* kinfo, const SInfo* sinfo, int n_k, int mmax,
                          const double2* Wraw, double2* Pout, int* status, cudaStream_t s) {
  const size_t smem = (size_t)3 * mmax * (mmax | 1) * sizeof(double2);
  cudaError_t e = cudaFuncSetAttribute(k_lowdin, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_lowdin<<<n_k, kEigThreads, smem, s>>>(kinfo, sinfo, Wraw, Pout, mmax, status);
  return cudaGetLastError();
}

// k-splits of k_pole_dos: about four CTAs per SM, and at least one k-point each.
int pole_dos_splits(int n_sys, int n_eps, int n_ch, int n_k, int sm_count) {
  const int blocks = n_sys * ((n_eps + 127) / 128) * ((n_ch + kDosT - 1) / kDosT);
  return std::max(1, std::min({64, n_k, (4 * sm_count + blocks - 1) / blocks}));
}

cudaError_t launch_pole_dos(const PoleParams& p, int n_sys, const double* eps_grid, int n_eps, double eta, int mmax,
                            int n_split, double* part, const int64_t* pdos_off, double* dos, double* pdos,
                            cudaStream_t s) {
  const int n_ch = 1 + (pdos ? mmax : 0);
  const dim3 grid(((n_eps + 127) / 128) * ((n_ch + kDosT - 1) / kDosT), n_sys, n_split);
  k_pole_dos<<<grid, 128, 0, s>>>(p, eps_grid, n_eps, eta, n_ch, mmax, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_dos_reduce<<<dim3(std::min(1024, (n_eps * n_ch + 127) / 128), n_sys), 128, 0, s>>>(p.sinfo, part, n_split, n_sys,
                                                                                   n_eps, mmax, pdos_off, dos, pdos);
  return cudaGetLastError();
}

size_t heev_smem(int n) { return (size_t)2 * n * (n | 1) * sizeof(double2); }
size_t heev_ws_elems(int n) { return (size_t)2 * n * (n | 1); }
int heev_max_n() { return 2 * 128; }  // rotation scratch holds 128 pairs

cudaError_t launch_heev_batched(const double2* A, int n_mat, int n, int max_sweeps, double* w,
                                double2* V, double2* gws, int grid, int in_smem, int* status,
                                cudaStream_t s) {
  const size_t smem = in_smem ? heev_smem(n) : 0;
  cudaError_t e = cudaFuncSetAttribute(k_heev_batched, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  k_heev_batched<<<grid, kEigThreads, smem, s>>>(A, n_mat, n, max_sweeps, w, V, gws, in_smem, status);
  return cudaGetLastError();
}

cudaError_t launch_pole_eig(const PoleParams& p, int grid, size_t smem, cudaStream_t s) {
  cudaError_t e =
      cudaFuncSetAttribute(k_pole_eig, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_pole_eig<<<grid, kEigThreads, smem, s>>>(p);
  return cudaGetLastError();
}

namespace {
// pairs per thread and frequencies per tile of k_pole_gloc (32 sums per thread, 48 with three pairs)
int gloc_qp(int mmax) { return (mmax * (mmax + 1) / 2 + kEigThreads - 1) / kEigThreads; }  // 1..3 for m <= 32
int gloc_f(int mmax) { return gloc_qp(mmax) == 1 ? 8 : 4; }
// (tile, split) pairs per system: four CTAs per SM, but at least every frequency's tile
int gloc_per_sys(int n_sys, int n_iw, int mmax, int sm_count) {
  const int F = gloc_f(mmax);
  return std::max((n_iw + F - 1) / F, (4 * sm_count + n_sys - 1) / n_sys);
}
size_t gloc_plan_elems(int n_sys) { return (sizeof(GlocPlan) * n_sys + sizeof(double2) - 1) / sizeof(double2); }
}  // namespace

size_t pole_gloc_ws_elems(int n_sys, int n_iw, int mmax, int sm_count) {
  return gloc_plan_elems(n_sys) +
         (size_t)n_sys * gloc_per_sys(n_sys, n_iw, mmax, sm_count) * gloc_f(mmax) * mmax * (mmax + 1);
}

cudaError_t launch_pole_gloc(const PoleParams& p, int n_sys, int mmax, int nps_max, int sm_count, double2* ws,
                             cudaStream_t s) {
  const int F = gloc_f(mmax), qp = gloc_qp(mmax), npairs = mmax * (mmax + 1) / 2;
  const int per_sys = gloc_per_sys(n_sys, p.n_iw, mmax, sm_count);
  const int threads = ((npairs + qp - 1) / qp + 31) / 32 * 32;
  GlocPlan* plan = reinterpret_cast<GlocPlan*>(ws);
  double2* part = ws + gloc_plan_elems(n_sys);
  k_pole_span<<<n_sys, kEigThreads, 0, s>>>(p, F, plan);
  const int grid = per_sys * n_sys;
  if (qp == 1) k_pole_gloc<1, 8><<<grid, threads, 0, s>>>(p, plan, per_sys, nps_max, npairs, part);
  else if (qp == 2) k_pole_gloc<2, 4><<<grid, threads, 0, s>>>(p, plan, per_sys, nps_max, npairs, part);
  else k_pole_gloc<3, 4><<<grid, threads, 0, s>>>(p, plan, per_sys, nps_max, npairs, part);
  const int64_t per_tile = (int64_t)2 * F * npairs;
  const int64_t most = per_tile * ((p.n_iw + F - 1) / F);
  const int bps = (int)std::min<int64_t>(std::max(1, 4096 / n_sys), (most + 127) / 128);
  k_gloc_splits<<<bps * n_sys, 128, 0, s>>>(plan, bps, per_sys, per_tile, part);
  k_gloc_write<<<p.n_iw * n_sys, 128, 0, s>>>(p, plan, per_sys, F, npairs, part);
  return cudaGetLastError();
}

}  // namespace gf
