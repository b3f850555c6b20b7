// Block form of the lattice points (gf_block.cuh): setup kernels, and the point kernel in FP64 and,
// for the higher frequencies of mixed precision (LOW), in FP32 and FP32 pairs.
//
// FP64 on GB300 issues two DFMAs per clock and SM, so a warp-wide FP64 instruction occupies
// its SM sub-partition for 64 clocks and everything else (shared-memory and L2 loads, index
// arithmetic, FP32) runs in its shadow.  The point kernel is therefore laid out for the
// fewest FP64 warp instructions with full lanes: a warp takes 32 / LW frequencies of one
// k-point (LW = 8, 16 or 32 lanes per m x m matrix), the band sums run over the flattened
// (frequency, pair) list, the elimination over the flattened entries, and the pair table
// B_a conj(B_c) of the k-point is formed once per uploaded H_k instead of per frequency.
//
// Bound: the FP64 pipe, 96-97 % busy.  Per point of a 40-band window with 14 orbitals: 56 k FP64
// FMAs for N(mu) and dN/dmu (band sums 33 k, S^{-1} 11 k, S^{-1} F 11 k) where the inverse of the
// window takes 281 k; 135 k with G_loc and rho_k.  Measured (GB300, 216 k-points x 1024
// frequencies): every output in 58.7 ms, 210 ms by the inverse; mu search and G_loc of 64 k-points
// 50 ms, 340 ms.
// LOW is bound by latency (issue slots 50-65 % busy at 11 to 14 warps an SM, FMA pipe 37-44 %):
// every output of 256 k-points in 9.7 ms, 20.8 ms with S and its inverse in FP64.
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "gf_block.cuh"
#include "gf_complex.cuh"
#include "gf_gj64.cuh"
#include "gf_series.cuh"

namespace gf {

namespace {

using namespace cx;
using gj64::crcp_scaled;
using series::cpow_int;
using series::series_z;
using series::SeriesZ;

constexpr int kSetupThreads = 256;

__device__ __forceinline__ double setup_sum(double v, double* red) {
  for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double r = 0.0;
  for (int w = 0; w < kSetupThreads / 32; ++w) r += red[w];
  return r;  // the same value in every thread
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Whether H_k and P_k allow the block form, and P_k^+ = Q [R; 0] by Householder reflections H_j = I -
// tau v v^+ (real tau, so H_j is Hermitian and unitary; the phases stay in R).  One CTA per k-point,
// ahead of the other kernels, which return at once when any k-point set a flag: the first mixed N(mu) (16
// frequencies) after a refused upload of 256 k-points of 40 bands takes 0.65 ms, 1.81 with the whole set-up.
__global__ void __launch_bounds__(kSetupThreads) k_block_check(const BlockSetup b) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double red[kSetupThreads / 32];
  double2* X = reinterpret_cast<double2*>(smraw);      // [m][N]: columns of P^+, then the vectors v_j
  double2* R = X + (size_t)b.mmax * b.nbmax;           // [m][m]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kSetupThreads / 32;
  const int k = blockIdx.x;
  const KInfo ki = b.kinfo[k];
  const int N = ki.nb, M = b.sinfo[ki.sys].m;
  const double2* H = b.H + ki.offH;
  const double2* P = b.P + ki.offP;
  // the norm of H_k and its distance from a Hermitian matrix
  double nrm = 0.0, anti = 0.0, big = 0.0;
  for (int e = tid; e < N * N; e += kSetupThreads) {
    const int i = e / N, j = e - i * N;
    const double2 h = H[e], t = H[j * N + i];
    nrm += h.x * h.x + h.y * h.y;
    anti = fmax(anti, fmax(fabs(h.x - t.x), fabs(h.y + t.y)));
    big = fmax(big, fmax(fabs(h.x), fabs(h.y)));
  }
  nrm = setup_sum(nrm, red);
  for (int off = 16; off; off >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, off));
  __syncthreads();
  if (lane == 0) red[warp] = big;
  __syncthreads();
  big = red[0];
  for (int w = 1; w < kWarps; ++w) big = fmax(big, red[w]);
  if (tid == 0) b.hnorm[k] = sqrt(nrm / N);
  // (NaN and infinity fail the comparison and take the general path)
  if (__syncthreads_or(!(anti <= 8.9e-16 * big) || !isfinite(nrm))) {
    if (tid == 0) atomicOr(b.flags, kBlkNonHermitian);
    return;
  }
  for (int e = tid; e < M * N; e += kSetupThreads) {
    const double2 p = P[e];
    X[e] = make_double2(p.x, -p.y);
  }
  __syncthreads();
  for (int j = 0; j < M; ++j) {
    double2* x = X + j * N;
    double s = 0.0;
    for (int i = j + tid; i < N; i += kSetupThreads) s += x[i].x * x[i].x + x[i].y * x[i].y;
    s = setup_sum(s, red);
    const double nx = sqrt(s);
    const double2 x0 = x[j];
    const double ax = sqrt(x0.x * x0.x + x0.y * x0.y);
    const double2 ph = ax > 0.0 ? make_double2(x0.x / ax, x0.y / ax) : make_double2(1.0, 0.0);
    const double tau = nx > 0.0 ? 1.0 / (nx * (nx + ax)) : 0.0;
    __syncthreads();
    if (tid == 0) {
      x[j] = make_double2(x0.x + ph.x * nx, x0.y + ph.y * nx);
      R[j * M + j] = make_double2(-ph.x * nx, -ph.y * nx);
      b.tau[(size_t)k * b.mmax + j] = tau;
    }
    __syncthreads();
    // the later columns: x_c -= tau v (v^+ x_c)
    for (int c = j + 1 + warp; c < M; c += kWarps) {
      double2* y = X + c * N;
      double2 d = make_double2(0.0, 0.0);
      for (int i = j + lane; i < N; i += 32) cmac_ca(d, x[i], y[i]);
      d.x = tau * warp_sum(d.x);
      d.y = tau * warp_sum(d.y);
      for (int i = j + lane; i < N; i += 32) {
        const double2 v = x[i];
        y[i].x -= fma(v.x, d.x, -v.y * d.y);
        y[i].y -= fma(v.x, d.y, v.y * d.x);
      }
      __syncwarp();
      if (lane == 0) R[j * M + c] = y[j];
    }
    __syncthreads();
  }
  for (int e = tid; e < M * N; e += kSetupThreads) {
    const int j = e / N, i = e - j * N;
    b.V[ki.offP + e] = i < j ? make_double2(0.0, 0.0) : X[e];
  }
  __syncthreads();
  // R^{-1} over X (M < N), column c by back substitution, and the conditioning of P: B, H11 and O carry
  // R^{-1}, so the errors of the form grow with the condition number of O = (P P^+)^{-1}, which
  // |R|^2 |R^{-1}|^2 / m - (m - 1) estimates (Frobenius norms; 1 for orthonormal rows, exact for one
  // small singular value beside equal ones).
  double r2 = 0.0, ri2 = 0.0;
  for (int c = tid; c < M; c += kSetupThreads) {
    for (int i = M - 1; i >= 0; --i) {
      double2 s = make_double2(i == c ? 1.0 : 0.0, 0.0), x = make_double2(0.0, 0.0);
      if (i <= c) {
        for (int j = i + 1; j <= c; ++j) {
          const double2 r = R[i * M + j], y = X[j * M + c];
          s.x -= fma(r.x, y.x, -r.y * y.y);
          s.y -= fma(r.x, y.y, r.y * y.x);
        }
        const double2 r = R[i * M + c];
        x = cmul(s, crcp(R[i * M + i]));
        r2 = fma(r.x, r.x, fma(r.y, r.y, r2));
        ri2 = fma(x.x, x.x, fma(x.y, x.y, ri2));
      }
      X[i * M + c] = x;
    }
  }
  r2 = setup_sum(r2, red);
  ri2 = setup_sum(ri2, red);
  // (rows that are zero, infinite or NaN fail the comparisons)
  if (tid == 0 && !(r2 * ri2 <= M * (b.cond + (M - 1)) && r2 < b.range && ri2 < b.range))
    atomicOr(b.flags, kBlkIllConditioned);
  for (int e = tid; e < M * M; e += kSetupThreads) b.Ri[(size_t)k * b.mmax * b.mmax + e] = X[e];
}

// Q^+ H_k Q by one rank-2 update per reflection.  One CTA per k-point (grid-stride).
__global__ void __launch_bounds__(kSetupThreads) k_block_reduce(const BlockSetup b, int in_smem) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double red[kSetupThreads / 32];
  if (*b.flags) return;
  double2* X = reinterpret_cast<double2*>(smraw);      // [m][N]: the vectors v_j
  double2* pv = X + (size_t)b.mmax * b.nbmax;          // [N]
  double2* A = in_smem ? pv + b.nbmax : b.ws + (size_t)blockIdx.x * b.nbmax * b.nbmax;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kSetupThreads / 32;
  for (int k = blockIdx.x; k < b.n_k; k += gridDim.x) {
    const KInfo ki = b.kinfo[k];
    const int N = ki.nb, M = b.sinfo[ki.sys].m, n2 = N - M;
    __syncthreads();
    for (int e = tid; e < N * N; e += kSetupThreads) A[e] = b.H[ki.offH + e];
    for (int e = tid; e < M * N; e += kSetupThreads) X[e] = b.V[ki.offP + e];
    __syncthreads();
    for (int j = 0; j < M; ++j) {
      const double2* x = X + j * N;
      const double tau = b.tau[(size_t)k * b.mmax + j];
      // A <- H_j A H_j: p = tau A v, w = p - (tau / 2) (v^+ p) v, A -= v w^+ + w v^+
      for (int i = warp; i < N; i += kWarps) {
        double2 d = make_double2(0.0, 0.0);
        for (int c = j + lane; c < N; c += 32) cmac(d, A[i * N + c], x[c]);
        d.x = warp_sum(d.x);
        d.y = warp_sum(d.y);
        if (lane == 0) pv[i] = make_double2(tau * d.x, tau * d.y);
      }
      __syncthreads();
      double vp = 0.0;
      for (int i = j + tid; i < N; i += kSetupThreads) vp += x[i].x * pv[i].x + x[i].y * pv[i].y;
      vp = 0.5 * tau * setup_sum(vp, red);
      __syncthreads();
      for (int i = j + tid; i < N; i += kSetupThreads) {
        pv[i].x = fma(-vp, x[i].x, pv[i].x);
        pv[i].y = fma(-vp, x[i].y, pv[i].y);
      }
      __syncthreads();
      for (int e = tid; e < N * N; e += kSetupThreads) {
        const int i = e / N, c = e - i * N;
        double2 a = A[e];
        if (i >= j) {
          const double2 v = x[i], w = pv[c];  // v_i conj(w_c)
          a.x -= fma(v.x, w.x, v.y * w.y);
          a.y -= fma(v.y, w.x, -v.x * w.y);
        }
        if (c >= j) {
          const double2 w = pv[i], v = x[c];
          a.x -= fma(w.x, v.x, w.y * v.y);
          a.y -= fma(w.y, v.x, -w.x * v.y);
        }
        A[e] = a;
      }
      __syncthreads();
    }
    for (int e = tid; e < M * M; e += kSetupThreads) {
      const int i = e / M, c = e - i * M;
      b.H11[(size_t)k * b.mmax * b.mmax + e] = A[i * N + c];
    }
    for (int e = tid; e < M * n2; e += kSetupThreads) {
      const int i = e / n2, c = e - i * n2;
      b.B[ki.offP + e] = A[i * N + M + c];
    }
    for (int e = tid; e < n2 * n2; e += kSetupThreads) {
      const int i = e / n2, c = e - i * n2;
      b.D22[ki.offH + e] = A[(M + i) * N + M + c];
    }
  }
}

// B, H11, O, the pair table and U of one k-point per CTA (gf_block.cuh).
__global__ void __launch_bounds__(kSetupThreads) k_block_finish(const BlockSetup b) {
  extern __shared__ __align__(16) unsigned char smraw[];
  if (*b.flags) return;
  const int k = blockIdx.x;
  const KInfo ki = b.kinfo[k];
  const int N = ki.nb, M = b.sinfo[ki.sys].m, n2 = N - M, np = M * (M + 1) / 2;
  const int tid = threadIdx.x;
  double2* Ri = reinterpret_cast<double2*>(smraw);        // R^{-1}
  double2* W = Ri + (size_t)b.mmax * b.mmax;              // m x m
  double2* Bs = W + (size_t)b.mmax * b.mmax;              // m x n2: H12 V, then B
  const double2* V2 = b.D22 + ki.offH;
  for (int e = tid; e < M * M; e += kSetupThreads) Ri[e] = b.Ri[(size_t)k * b.mmax * b.mmax + e];
  for (int e = tid; e < M * n2; e += kSetupThreads) {
    const int a = e / n2, c = e - a * n2;
    double2 s = make_double2(0.0, 0.0);
    for (int x = 0; x < n2; ++x) cmac(s, b.B[ki.offP + a * n2 + x], V2[x * n2 + c]);
    Bs[e] = s;
  }
  __syncthreads();
  // B = R^{-1} (H12 V), column by column in place (row a takes the rows from a on)
  for (int c = tid; c < n2; c += kSetupThreads) {
    for (int a = 0; a < M; ++a) {
      double2 s = make_double2(0.0, 0.0);
      for (int x = a; x < M; ++x) cmac(s, Ri[a * M + x], Bs[x * n2 + c]);
      Bs[a * n2 + c] = s;
    }
  }
  // W = R^{-1} H11
  for (int e = tid; e < M * M; e += kSetupThreads) {
    const int a = e / M, c = e - a * M;
    double2 s = make_double2(0.0, 0.0);
    for (int x = a; x < M; ++x) cmac(s, Ri[a * M + x], b.H11[(size_t)k * b.mmax * b.mmax + x * M + c]);
    W[e] = s;
  }
  __syncthreads();
  for (int e = tid; e < M * n2; e += kSetupThreads) {
    b.B[ki.offP + e] = Bs[e];
    if (b.Bs) b.Bs[ki.offP + e] = make_float2((float)Bs[e].x, (float)Bs[e].y);
  }
  double2* HO = b.HO + (size_t)k * 2 * b.npmax;
  for (int pr = tid; pr < np; pr += kSetupThreads) {
    int a = 0, rem = pr;
    while (rem >= M - a) { rem -= M - a; ++a; }
    const int c = a + rem;
    double2 h = make_double2(0.0, 0.0), o = make_double2(0.0, 0.0);
    for (int x = c; x < M; ++x) {
      cmac_cb(h, W[a * M + x], Ri[c * M + x]);
      cmac_cb(o, Ri[a * M + x], Ri[c * M + x]);
    }
    if (a == c) h.y = o.y = 0.0;
    HO[pr] = h;
    HO[b.npmax + pr] = o;
  }
  for (int e = tid; e < np * n2; e += kSetupThreads) {
    const int l = e / np, pr = e - l * np;
    int a = 0, rem = pr;
    while (rem >= M - a) { rem -= M - a; ++a; }
    const int c = a + rem;
    double2 t = make_double2(0.0, 0.0);
    cmac_cb(t, Bs[a * n2 + l], Bs[c * n2 + l]);
    if (a == c) t.y = 0.0;
    b.T[b.offT[k] + e] = t;
    if (b.Ts) {
      const cf v = from_d2(t);
      b.Ts[b.offT[k] + e] = make_float2(v.rh, v.ih);
      b.Tp[b.offT[k] + e] = st4(v);
    }
  }
  // U = Q diag(R^{-+}, V2): one column per thread, the reflections in reverse order
  double2* U = b.U + ki.offH;
  const double2* Vh = b.V + ki.offP;
  const double* tau = b.tau + (size_t)k * b.mmax;
  for (int c = tid; c < N; c += kSetupThreads) {
    for (int i = 0; i < N; ++i) {
      double2 v = make_double2(0.0, 0.0);
      if (c < M) {
        if (i < M) v = make_double2(Ri[c * M + i].x, -Ri[c * M + i].y);
      } else if (i >= M) {
        v = V2[(i - M) * n2 + c - M];
      }
      U[i * N + c] = v;
    }
    for (int j = M - 1; j >= 0; --j) {
      const double2* v = Vh + j * N;
      double2 s0 = make_double2(0.0, 0.0), s1 = s0;
      int i = j;
      for (; i + 1 < N; i += 2) {
        cmac_ca(s0, v[i], U[i * N + c]);
        cmac_ca(s1, v[i + 1], U[(i + 1) * N + c]);
      }
      if (i < N) cmac_ca(s0, v[i], U[i * N + c]);
      const double2 s = make_double2(tau[j] * (s0.x + s1.x), tau[j] * (s0.y + s1.y));
      for (i = j; i < N; ++i) {
        double2 u = U[i * N + c];
        u.x -= fma(v[i].x, s.x, -v[i].y * s.y);
        u.y -= fma(v[i].x, s.y, v[i].y * s.x);
        U[i * N + c] = u;
      }
    }
  }
}

// Chebyshev moments of one k-point per CTA: C_j by pairs and tau_j.
__global__ void __launch_bounds__(kSetupThreads) k_block_series(const BlockSetup b) {
  extern __shared__ __align__(16) unsigned char smraw[];
  double* Tj = reinterpret_cast<double*>(smraw);  // [jt][n2]
  __shared__ double s_cr[2];
  if (*b.flags) return;
  const int k = blockIdx.x;
  const KInfo ki = b.kinfo[k];
  const int M = b.sinfo[ki.sys].m, n2 = ki.nb - M, np = M * (M + 1) / 2, jt = min(n2, kBlkSeries);
  const int tid = threadIdx.x;
  const double* e = b.e + b.offD[k];
  if (tid < 32) {
    double lo = INFINITY, hi = -INFINITY;
    for (int l = tid; l < n2; l += 32) {
      lo = fmin(lo, e[l]);
      hi = fmax(hi, e[l]);
    }
    for (int off = 16; off; off >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, off));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, off));
    }
    if (tid == 0) {
      s_cr[0] = 0.5 * (lo + hi);
      s_cr[1] = fmax(0.5 * (hi - lo), 1e-3);
      double* cr = b.series + (size_t)kBlkSeries * b.n_k + 2 * (size_t)k;
      cr[0] = s_cr[0];
      cr[1] = s_cr[1];
    }
  }
  __syncthreads();
  for (int l = tid; l < n2; l += kSetupThreads) {
    const double x = (e[l] - s_cr[0]) / s_cr[1];
    double t0 = 1.0, t1 = x;
    for (int j = 0; j < jt; ++j) {
      Tj[j * n2 + l] = t0;
      const double t2 = fma(2.0 * x, t1, -t0);
      t0 = t1;
      t1 = t2;
    }
  }
  __syncthreads();
  for (int j = tid; j < jt; j += kSetupThreads) {
    double s = 0.0;
    for (int l = 0; l < n2; ++l) s += Tj[j * n2 + l];
    b.series[(size_t)kBlkSeries * k + j] = s;
  }
  const double2* T = b.T + b.offT[k];
  for (int i = tid; i < jt * np; i += kSetupThreads) {
    const int j = i / np, pr = i - j * np;
    double2 v = make_double2(0.0, 0.0);
    for (int l = 0; l < n2; ++l) {
      const double2 t = T[(size_t)l * np + pr];
      const double c = Tj[j * n2 + l];
      v.x = fma(c, t.x, v.x);
      v.y = fma(c, t.y, v.y);
    }
    b.C[b.offC[k] + i] = v;
    if (b.Cs) {
      const cf c = from_d2(v);
      b.Cs[b.offC[k] + i] = make_float2(c.rh, c.ih);
      b.Cp[b.offC[k] + i] = st4(c);
    }
  }
}

// ------------------------------------------------------------------ point kernel

template <bool LOW>
struct Rest {  // type of the parts that mixed precision takes from an FP32 inverse
  using c = double2;
  using r = double;
};
template <>
struct Rest<true> {
  using c = float2;
  using r = float;
};
__device__ __forceinline__ float2 to_rest(double2 v, float2) { return make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ void rmac(double2& a, double2 x, double2 y) { cmac(a, x, y); }
__device__ __forceinline__ void rmac(float2& a, float2 x, float2 y) { fmac(a, x, y); }
__device__ __forceinline__ double2 rzero(double2) { return make_double2(0.0, 0.0); }
__device__ __forceinline__ float2 rzero(float2) { return make_float2(0.f, 0.f); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// Shared memory of the point kernel in bytes; every array holds the CTA's W F frequencies, warp
// after warp.  First what is dead once the warps have S^{-1}: F, d^2 / d^3, the pivot row and
// column, Gbar A^+ (adjoint), and with LOW also S and the refinement's residual (rho_k then reads
// S^{-1} in FP32); with LOW B, and the columns S^{-1} B D of rho_k are staged over it, yf frequencies
// at a time.  Then S, with LOW S^{-1} in FP32, d (or the series coefficients), the pivot tables, w_n,
// the pair list and mu O - H11 by pairs.
struct LayoutB {
  size_t oS, oF, od2, orc, oM, oY, oG, od, op, oW, oPair, oHz, oX, oB, bytes;
  size_t sS, sF, sd2, src, sG, sd, sp;  // bytes per warp (sS also of M)
  size_t fG;  // bytes of S^{-1} in FP32 per frequency
  int nf;   // frequencies per warp
  int yf;   // frequencies of the rho_k columns staged at once
};

__host__ __device__ inline LayoutB make_layout_b(int mmax, int n2max, int mode, int low) {
  LayoutB L;
  L.nf = 32 / gj64::lanes(mmax);
  const size_t f = L.nf, mm = (size_t)mmax * mmax, r = low ? 8 : 16, W = kBlkWarps;
  const bool adj = (mode & kAdj) != 0, needF = (mode & kOcc) != 0 || adj, rho = (mode & kRho) != 0;
  auto al = [](size_t x) { return (x + 15) & ~(size_t)15; };
  L.sS = 16 * f * mm;
  // (the adjoint's F and d^2 are pairs with LOW)
  L.sF = needF ? al((adj ? 16 : r) * f * mm) : 0;
  L.sd2 = needF ? al((low && adj ? 24 : 2 * r) * f * n2max) : 0;
  L.src = (low ? 8 : 16) * f * 2 * mmax;
  const size_t kp = (mmax + 1) / 2, pb = ((size_t)n2max + 3) & ~(size_t)3;
  L.fG = low ? (rho ? 16 * kp * mmax : 8 * mm) : 0;  // (rho_k reads it by pairs of rows)
  L.sG = al(f * L.fG);
  L.sd = 16 * f * n2max;
  L.sp = al(4 * f * 2 * mmax);
  size_t o = 0;
  if (!low) { L.oS = o; o += W * L.sS; }
  L.oY = o;
  if (low) { L.oS = o; o += W * L.sS; }
  L.oF = o; o += W * L.sF;
  L.od2 = o; o += W * L.sd2;
  L.orc = o; o += W * L.src;
  L.oM = o; o += adj ? W * L.sS : 0;
  const size_t np = (size_t)mmax * (mmax + 1) / 2;
  const size_t fixed = W * (L.sG + L.sd + L.sp + (low ? 16 : 8) * f) + al(2 * np) + (low ? 32 : 16) * np +
                       (low && rho ? al(4 * (size_t)n2max) : 0);
  const size_t sB = low && rho ? 16 * kp * pb : 0;
  L.oB = L.oY;
  L.oY += sB;
  L.yf = 0;
  if (rho) {
    // as many frequencies as fit over the dead arrays, or as leave three CTAs on an SM, or two:
    // the chunk's sum is read and written once per stage
    const size_t one = 16 * (low ? kp : mmax) * (size_t)n2max;
    const size_t all = f * W;
    size_t room = o > L.oY ? o - L.oY : 0;
    for (size_t lim = (75u << 10) - 128; lim < (113u << 10); lim += 38u << 10)  // (and 128 B of static arrays)
      if (room < all * one && L.oY + fixed + (room > one ? room : one) <= lim) {
        room = lim - L.oY - fixed;
        break;
      }
    const size_t fit = room >= one ? room / one : 1, stages = fit < all ? (all + fit - 1) / fit : 1;
    L.yf = (int)((all + stages - 1) / stages);
    if (L.oY + one * L.yf > o) o = al(L.oY + one * L.yf);
  }
  L.oG = o; o += W * L.sG;
  L.od = o; o += W * L.sd;
  L.op = o; o += W * L.sp;
  L.oW = o; o = al(o + (low ? 16 : 8) * W * f);  // w_n (low: and in pairs)
  L.oPair = o; o += al(2 * np);
  L.oHz = o; o += (low ? 32 : 16) * np;  // (low: pairs of mu O - H11, then of O)
  L.oX = o; o = al(o + (low && rho ? 4 * (size_t)n2max : 0));
  L.bytes = o;
  return L;
}

__device__ __forceinline__ double2 ld_cg(const double2* p) { return __ldg(p); }
__device__ __forceinline__ float2 ld_cg(const float2* p) { return __ldg(p); }

// What an instance of the kernel holds beside S^{-1}: the traces, and rho_k or the adjoint.  G_loc
// alone in FP32 pairs runs in 128 registers and less shared memory, four CTAs on an SM: 5.4 ms
// instead of 6.2 (256 k-points x 1024 frequencies, 40 bands, 14 orbitals); with the traces the
// shared memory leaves three, and fewer registers cost 9 %.  Eight lanes a matrix run in 128 registers but
// for rho_k in FP32, whose pairs spill there: 64 k-points x 1024 frequencies, 96 bands, 7 orbitals 3.8 ms, 3.4
// in 168.
enum { kGlocOnly, kPlain, kWithRho, kWithAdj };

template <int LW, bool LOW, int PART>
__global__ void __launch_bounds__(32 * kBlkWarps,
                                  PART == kGlocOnly || (LW == 8 && !(LOW && PART == kWithRho)) ? 4 : 3)
    k_point_block(const PointParams p, const BlockForm bf, const BlockLaunch bl) {
  using rc_t = typename Rest<LOW>::c;
  using rr_t = typename Rest<LOW>::r;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double s_part[kBlkWarps][3];
  constexpr int F = 32 / LW;
  constexpr int W = kBlkWarps;
  const LayoutB L = make_layout_b(p.mmax, bl.n2max, p.mode, LOW ? 1 : 0);
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, sl = lane % LW, mf = lane / LW;
  double2* sS = reinterpret_cast<double2*>(smraw + L.oS + wp * L.sS);
  rc_t* sF = reinterpret_cast<rc_t*>(smraw + L.oF + wp * L.sF);
  double2* sd = reinterpret_cast<double2*>(smraw + L.od + wp * L.sd);
  rc_t* sd2 = reinterpret_cast<rc_t*>(smraw + L.od2 + wp * L.sd2);
  double2* sM = reinterpret_cast<double2*>(smraw + L.oM + wp * L.sS);
  constexpr bool low_adj = LOW && PART == kWithAdj;  // F and d^2 in pairs
  float2* sG = reinterpret_cast<float2*>(smraw + L.oG + wp * L.sG);
  int* sPv = reinterpret_cast<int*>(smraw + L.op + wp * L.sp);
  double* sW = reinterpret_cast<double*>(smraw + L.oW) + wp * F;
  float2* sWp = reinterpret_cast<float2*>(smraw + L.oW + 8 * W * F) + wp * F;
  uchar2* pair = reinterpret_cast<uchar2*>(smraw + L.oPair);
  double2* hz = reinterpret_cast<double2*>(smraw + L.oHz);
  float* xs = reinterpret_cast<float*>(smraw + L.oX);  // x_b = mu - e_b
  const int unit = bl.unit0 + blockIdx.x / bl.n_chunks, ch = blockIdx.x % bl.n_chunks;
  const int2 un = bl.units[unit];
  const int n0 = bl.n_begin + ch * bl.chunk_w, n1 = min(bl.n_end, n0 + bl.chunk_w);
  const int chunk = bl.chunk0 + ch;
  const bool occ = PART != kGlocOnly && (p.mode & kOcc) != 0;
  constexpr bool adj = PART == kWithAdj, rho = PART == kWithRho;

  for (int q = 0; q < un.y; ++q) {
    const int kk = bl.kperm[un.x + q];
    const KInfo ki = p.kinfo[kk];
    const SInfo si = p.sinfo[ki.sys];
    const int M = si.m, n2 = ki.nb - M, NP = M * (M + 1) / 2, MM = M * M;
    const double mu = p.mu[ki.sys], pib = M_PI / si.beta, wk = ki.w;
    const double* e_k = bf.e + bf.offD[kk];
    const double2* T = bf.T + bf.offT[kk];
    const double2* HO = bf.HO + (size_t)kk * 2 * bf.npmax;
    const double cb = (adj && p.nbar) ? p.nbar[ki.sys] * 2.0 / si.beta : 0.0;
    const bool have_gbar = adj && (LOW ? (const void*)p.Gbd : (const void*)p.gbar) != nullptr;
    double2* A = sS + mf * MM;  // this lane group's matrix
    rc_t* sd3 = sd2 + (low_adj ? 2 : 1) * F * n2;
    rc_t* rcb = reinterpret_cast<rc_t*>(smraw + L.orc + wp * L.src) + mf * 2 * M;
    int* sp = sPv + mf * 2 * M;
    __syncthreads();
    for (int pr = tid; pr < NP; pr += 32 * W) {
      int a = 0, rem = pr;
      while (rem >= M - a) { rem -= M - a; ++a; }
      pair[pr] = make_uchar2((unsigned char)a, (unsigned char)(a + rem));
      const double2 h = HO[pr], o = HO[bf.npmax + pr];
      const double2 z0 = make_double2(fma(mu, o.x, -h.x), fma(mu, o.y, -h.y));
      if constexpr (LOW) {
        reinterpret_cast<float4*>(hz)[pr] = st4(from_d2(z0));
        reinterpret_cast<float4*>(hz)[NP + pr] = st4(from_d2(o));
      } else {
        hz[pr] = z0;
      }
    }
    if constexpr (LOW) {
      if (rho) {
        for (int i = tid; i < n2; i += 32 * W) xs[i] = __double2float_rn(mu - e_k[i]);
      }
    }
    __syncthreads();
    double acc_tr = 0.0, acc_g2 = 0.0, acc_mu = 0.0;
    for (int base = n0; base < n1; base += W * F) {
      const int n = base + wp * F;
      const int nv = min(F, n1 - n);  // frequencies of this warp (<= 0: none)
      if (nv > 0) {
        __syncwarp();
        // the sums over the n2 bands, or over fewer Chebyshev moments where those converge sooner
        // (44.8 = 56 ln 2 + 6; the series' own overhead is about 150 FP64 instructions per warp, so
        // it has to save this many terms x pairs.  FP64, 1600: at 5000 N(mu) of 216 k-points takes
        // 25.1 ms instead of 24.7, at 0 N(mu) of 75 k-points x 333 frequencies 1.60 instead of 1.56.
        // LOW, 5000: at 12000 G_loc of 96 k-points at 88 bands 2.5 ms instead of 1.7, at 0 G_loc of 256
        // at 40 bands 5.5 instead of 5.3)
        int nt = n2;
        const double2* Tt = T;
        const float2* Tst = nullptr;
        const float4* Tpt = nullptr;
        if constexpr (LOW) {
          Tst = bf.Ts + bf.offT[kk];
          Tpt = bf.Tp + bf.offT[kk];
        }
        bool series = false;
        // d (or the series' coefficients) for the sums: in FP32 pairs with LOW
        auto put_d = [&](int i, double2 d) {
          if constexpr (LOW) reinterpret_cast<float4*>(sd)[i] = st4(from_d2(d));
          else sd[i] = d;
        };
        if (lane < F) {
          const double wn = (2.0 * min(n + lane, n1 - 1) + 1.0) * pib;
          sW[lane] = wn;
          if constexpr (LOW) split(wn, sWp[lane].x, sWp[lane].y);
        }
        __syncwarp();
        {
          const double2 cr = bf.cr[kk];
          const int J = series_terms((float)(mu - cr.x), (float)((2.0 * n + 1.0) * pib), (float)cr.y, 44.8f);
          // (LOW: the sums cost a sixth, in FP32 pairs)
          const int sums = occ ? 3 : (adj ? 2 : 1);
          if (J <= min(n2, kBlkSeries) && (LOW ? (n2 - J) * NP * F > 5000 : (n2 - J) * NP * F * sums > 1600)) {
            nt = J;
            Tt = bf.C + bf.offC[kk];
            if constexpr (LOW) {
              Tst = bf.Cs + bf.offC[kk];
              Tpt = bf.Cp + bf.offC[kk];
            }
            series = true;
            const double* tau = bf.tau + (size_t)kBlkSeries * kk;
            int fz = -1;
            SeriesZ z;
            float2 zf[5];
            for (int i = lane; i < F * J; i += 32) {
              const int f = i / J, j = i - f * J;
              if (f != fz) {
                z = series_z(mu - cr.x, sW[f], cr.y, occ || adj);
                fz = f;
                if constexpr (LOW) {
                  zf[0] = to_rest(z.c2a, float2{});
                  zf[1] = to_rest(z.c2b, float2{});
                  zf[2] = to_rest(z.c3a, float2{});
                  zf[3] = to_rest(z.c3b, float2{});
                  zf[4] = to_rest(z.c3c, float2{});
                }
              }
              double2 pw = cpow_int<6>(z.xi, j);
              if (j) pw = make_double2(2.0 * pw.x, 2.0 * pw.y);
              const double2 d = cmul(pw, z.c1);
              put_d(i, d);
              if constexpr (LOW) {
                if (adj) {
                  const double fj = j;
                  reinterpret_cast<float4*>(sd2)[i] =
                      st4(from_d2(cmul(pw, make_double2(fma(fj, z.c2a.x, z.c2b.x), fma(fj, z.c2a.y, z.c2b.y)))));
                }
                if (occ) {
                  const float2 pf = make_float2((float)pw.x, (float)pw.y);
                  const float fj = (float)j, j2 = fj * fj - 1.f;
                  const float2 d2 = fmul(pf, make_float2(fmaf(fj, zf[0].x, zf[1].x), fmaf(fj, zf[0].y, zf[1].y)));
                  if (!adj) sd2[i] = d2;
                  sd3[i] = fmul(pf, make_float2(fmaf(j2, zf[2].x, fmaf(fj, zf[3].x, zf[4].x)),
                                                         fmaf(j2, zf[2].y, fmaf(fj, zf[3].y, zf[4].y))));
                  if (f < nv) {
                    acc_tr = fma(tau[j], d.x, acc_tr);
                    acc_g2 = fma(tau[j], widen(d2.x), acc_g2);
                  }
                }
              } else if (occ || adj) {
                const double fj = j;
                const double2 d2 = cmul(pw, make_double2(fma(fj, z.c2a.x, z.c2b.x), fma(fj, z.c2a.y, z.c2b.y)));
                sd2[i] = d2;
                if (occ) {
                  const double j2 = fma(fj, fj, -1.0);
                  sd3[i] = cmul(pw, make_double2(fma(j2, z.c3a.x, fma(fj, z.c3b.x, z.c3c.x)),
                                                          fma(j2, z.c3a.y, fma(fj, z.c3b.y, z.c3c.y))));
                  if (f < nv) {
                    acc_tr = fma(tau[j], d.x, acc_tr);
                    acc_g2 = fma(tau[j], d2.x, acc_g2);
                  }
                }
              }
            }
          }
        }
        auto bands = [&](bool sums) {  // d_b, and with sums its powers and traces
          for (int i = lane; i < F * n2; i += 32) {
            const int f = i / n2, bb = i - f * n2;
            const double wn = sW[f];
            const double x = mu - e_k[bb];
            const double xw = fma(x, x, wn * wn);
            const double s = rcp_newton(xw);
            const double2 d = make_double2(x * s, -wn * s);
            if constexpr (LOW) {
              const cf dp = from_d2(d);
              reinterpret_cast<float4*>(sd)[i] = st4(dp);
              if (adj) {
                cf d2 = czero();
                cacc(d2, dp, dp);
                cnorm(d2);
                reinterpret_cast<float4*>(sd2)[i] = st4(d2);
              }
              if (occ) {
                const float2 df = make_float2(dp.rh, dp.ih), d2 = fmul(df, df);
                if (!adj) sd2[i] = d2;
                sd3[i] = fmul(d2, df);
                if (f < nv) {
                  acc_tr += d.x;
                  acc_g2 += widen(d2.x);
                }
              }
            } else if (sd[i] = d; sums && (occ || adj)) {
              const double2 d2 = cmul(d, d);
              sd2[i] = d2;
              if (occ) {
                sd3[i] = cmul(d2, d);
                if (f < nv) {
                  acc_tr += d.x;
                  acc_g2 += d2.x;
                }
              }
            }
          }
        };
        if (!series) bands(true);
        __syncwarp();
        // S and F, pair by pair: with t = B_a conj(B_c), sum t Re d and sum t Im d give both
        // (a, c) and (c, a)
        for (int i = lane; i < F * NP; i += 32) {
          const int f = i / NP, pr = i - f * NP;
          const int a = pair[pr].x, c = pair[pr].y;
          const int nn = min(n + f, n1 - 1);
          if constexpr (LOW) {
            // S in FP32 pairs, F in FP32
            const float4* t = Tpt + pr;
            const float4* df = reinterpret_cast<const float4*>(sd) + f * nt;
            float xrr[2] = {0.f, 0.f}, xri[2] = {0.f, 0.f}, xir[2] = {0.f, 0.f}, xii[2] = {0.f, 0.f};
            float2 yr = make_float2(0.f, 0.f), yi = yr;
            auto plus = [](float& sh, float& sl_, float vh, float vl) {  // (sh, sl_) += (vh, vl)
              float s, e;
              two_sum(sh, vh, s, e);
              sh = s;
              sl_ = __fadd_rn(sl_, __fadd_rn(vl, e));
            };
            auto add = [&](float4 tv, float4 d) {
              acc_prod(tv.x, tv.y, d.x, d.y, xrr[0], xrr[1]);
              acc_prod(tv.z, tv.w, d.x, d.y, xri[0], xri[1]);
              acc_prod(tv.x, tv.y, d.z, d.w, xir[0], xir[1]);
              acc_prod(tv.z, tv.w, d.z, d.w, xii[0], xii[1]);
            };
            if (adj) {
              const float4* d2f = reinterpret_cast<const float4*>(sd2) + f * nt;
              cf v1 = czero(), v2 = czero();  // sum t Re d^2 and sum t Im d^2
#pragma unroll 2
              for (int bb = 0; bb < nt; ++bb) {
                const float4 tv = __ldg(t + (size_t)bb * NP), d2 = d2f[bb];
                add(tv, df[bb]);
                acc_prod(tv.x, tv.y, d2.x, d2.y, v1.rh, v1.rl);
                acc_prod(tv.z, tv.w, d2.x, d2.y, v1.ih, v1.il);
                acc_prod(tv.x, tv.y, d2.z, d2.w, v2.rh, v2.rl);
                acc_prod(tv.z, tv.w, d2.z, d2.w, v2.ih, v2.il);
              }
              const float4 o = reinterpret_cast<const float4*>(hz)[NP + pr];
              float4* Fm = reinterpret_cast<float4*>(sF) + f * MM;
              cf g{o.x, o.y, o.z, o.w};
              plus(g.rh, g.rl, v1.rh, v1.rl);
              plus(g.rh, g.rl, -v2.ih, -v2.il);
              plus(g.ih, g.il, v1.ih, v1.il);
              plus(g.ih, g.il, v2.rh, v2.rl);
              cnorm(g);
              Fm[a * M + c] = st4(g);
              if (a != c) {
                cf h{o.x, o.y, -o.z, -o.w};
                plus(h.rh, h.rl, v1.rh, v1.rl);
                plus(h.rh, h.rl, v2.ih, v2.il);
                plus(h.ih, h.il, -v1.ih, -v1.il);
                plus(h.ih, h.il, v2.rh, v2.rl);
                cnorm(h);
                Fm[c * M + a] = st4(h);
              }
            } else if (occ) {
              const float2* d2f = sd2 + f * nt;
#pragma unroll 2
              for (int bb = 0; bb < nt; ++bb) {
                const float4 tv = __ldg(t + (size_t)bb * NP);
                const float2 d2 = d2f[bb];
                add(tv, df[bb]);
                yr.x = fmaf(tv.x, d2.x, yr.x); yr.y = fmaf(tv.z, d2.x, yr.y);
                yi.x = fmaf(tv.x, d2.y, yi.x); yi.y = fmaf(tv.z, d2.y, yi.y);
              }
              const float4 o = reinterpret_cast<const float4*>(hz)[NP + pr];
              float2* Fm = sF + f * MM;
              Fm[a * M + c] = make_float2(o.x + (yr.x - yi.y), o.z + (yr.y + yi.x));
              if (a != c) Fm[c * M + a] = make_float2(o.x + (yr.x + yi.y), (yi.x - yr.y) - o.z);
            } else {
#pragma unroll 2
              for (int bb = 0; bb < nt; ++bb) add(__ldg(t + (size_t)bb * NP), df[bb]);
            }
            // (a, c): h + i w o - Sigma_ac - g_ac; (c, a): conj(h) + i w conj(o) - Sigma_ca - g_ca
            const float4 h = reinterpret_cast<const float4*>(hz)[pr], o = reinterpret_cast<const float4*>(hz)[NP + pr];
            const float2 w = sWp[f];
            const float4* Sg = p.Sd + si.offSig + (int64_t)nn * MM;
            float4* Sm = reinterpret_cast<float4*>(sS) + f * MM;
            {
              const float4 sg = Sg[a * M + c];
              cf v{h.x, h.y, h.z, h.w};
              acc_prod(-w.x, -w.y, o.z, o.w, v.rh, v.rl);
              acc_prod(w.x, w.y, o.x, o.y, v.ih, v.il);
              plus(v.rh, v.rl, -sg.x, -sg.y);
              plus(v.ih, v.il, -sg.z, -sg.w);
              plus(v.rh, v.rl, -xrr[0], -xrr[1]);
              plus(v.rh, v.rl, xii[0], xii[1]);
              plus(v.ih, v.il, -xri[0], -xri[1]);
              plus(v.ih, v.il, -xir[0], -xir[1]);
              cnorm(v);
              Sm[a * M + c] = st4(v);
            }
            if (a != c) {
              const float4 sg = Sg[c * M + a];
              cf v{h.x, h.y, -h.z, -h.w};
              acc_prod(w.x, w.y, o.z, o.w, v.rh, v.rl);
              acc_prod(w.x, w.y, o.x, o.y, v.ih, v.il);
              plus(v.rh, v.rl, -sg.x, -sg.y);
              plus(v.ih, v.il, -sg.z, -sg.w);
              plus(v.rh, v.rl, -xrr[0], -xrr[1]);
              plus(v.rh, v.rl, -xii[0], -xii[1]);
              plus(v.ih, v.il, xri[0], xri[1]);
              plus(v.ih, v.il, -xir[0], -xir[1]);
              cnorm(v);
              Sm[c * M + a] = st4(v);
            }
          } else {
            const double2* t = Tt + pr;
            const double2* df = sd + f * nt;
            double2 xr = make_double2(0.0, 0.0), xi = xr;
            const double2 o = HO[bf.npmax + pr];
            if (occ || adj) {
              double2 yr = make_double2(0.0, 0.0), yi = yr;
              const double2* d2f = sd2 + f * nt;
#pragma unroll 4
              for (int bb = 0; bb < nt; ++bb) {
                const double2 tv = __ldg(t + (size_t)bb * NP), d = df[bb], d2 = d2f[bb];
                xr.x = fma(tv.x, d.x, xr.x); xr.y = fma(tv.y, d.x, xr.y);
                xi.x = fma(tv.x, d.y, xi.x); xi.y = fma(tv.y, d.y, xi.y);
                yr.x = fma(tv.x, d2.x, yr.x); yr.y = fma(tv.y, d2.x, yr.y);
                yi.x = fma(tv.x, d2.y, yi.x); yi.y = fma(tv.y, d2.y, yi.y);
              }
              double2* Fm = sF + f * MM;
              Fm[a * M + c] = make_double2(o.x + (yr.x - yi.y), o.y + (yr.y + yi.x));
              if (a != c) Fm[c * M + a] = make_double2(o.x + (yr.x + yi.y), (yi.x - yr.y) - o.y);
            } else {
#pragma unroll 4
              for (int bb = 0; bb < nt; ++bb) {
                const double2 tv = __ldg(t + (size_t)bb * NP), d = df[bb];
                xr.x = fma(tv.x, d.x, xr.x); xr.y = fma(tv.y, d.x, xr.y);
                xi.x = fma(tv.x, d.y, xi.x); xi.y = fma(tv.y, d.y, xi.y);
              }
            }
            const double2 h = hz[pr];
            const double wn = sW[f];
            const double2* Sg = p.Sig + si.offSig + (int64_t)nn * MM;
            // (a, c): h + i w o - Sigma_ac - g_ac; (c, a): conj(h) + i w conj(o) - Sigma_ca - g_ca
            const double2 s1 = Sg[a * M + c], s2 = Sg[c * M + a];
            double2* Sm = sS + f * MM;
            Sm[a * M + c] = make_double2((fma(-wn, o.y, h.x) - s1.x) - (xr.x - xi.y),
                                         (fma(wn, o.x, h.y) - s1.y) - (xr.y + xi.x));
            if (a != c)
              Sm[c * M + a] = make_double2((fma(wn, o.y, h.x) - s2.x) - (xr.x + xi.y),
                                           (fma(wn, o.x, -h.y) - s2.y) - (xi.x - xr.y));
          }
        }
        __syncwarp();
        // rho_k reads d_b (its barrier comes first): in FP32 with LOW
        if constexpr (LOW) {
          if (rho)
            for (int i = lane; i < F * n2; i += 32) {
              const int f = i / n2;
              const float x = xs[i - f * n2], w = sWp[f].x, q = __frcp_rn(fmaf(x, x, w * w));
              reinterpret_cast<float2*>(sd)[i] = make_float2(x * q, -w * q);
            }
        } else if (rho && series) {
          bands(false);
        }
        const int* sq = sp + M;
        const bool mine = mf < nv;
        double2* out = (p.mode & (kGloc | kAdj))
                           ? p.gq + ((int64_t)(unit - p.gb0) * p.n_iw + min(n + mf, n1 - 1)) * p.mmax * p.mmax
                           : nullptr;
        const rc_t* inv;  // the warp's inverses, A[p_i][q_c] (LOW: FP32)
        if constexpr (LOW) {
          const float4* Sp = reinterpret_cast<const float4*>(A);
          float2* X0 = sG + mf * (L.fG / sizeof(float2));
          for (int i = sl; i < MM; i += LW) X0[i] = make_float2(Sp[i].x, Sp[i].z);
          __syncwarp();
          gj64::invert<LW>(X0, M, rcb, sp, sl, p.status);
          inv = sG;
        } else {
          gj64::invert<LW>(A, M, rcb, sp, sl, p.status);
          inv = sS;
          if ((p.mode & kGloc) && mine)
            for (int i = sl; i < MM; i += LW) {
              const int a = i / M, c = i - a * M;
              const double2 g = A[sp[a] * M + sq[c]];
              gq_put(&out[i], q, make_double2(wk * g.x, wk * g.y));
            }
        }
        if (occ) {
          // LOW: this lane's sums of (Tr X, Tr G^2) and Tr X^2 over the warp's frequencies, in pairs
          float2 low_h = make_float2(0.f, 0.f), low_l = low_h, low_xh = low_h, low_xl = low_h;
          for (int i = lane; i < F * NP; i += 32) {
            const int f = i / NP, pr = i - f * NP;
            const int a = pair[pr].x, c = pair[pr].y;
            const rc_t* Fm = sF + f * MM;
            rc_t x1 = rzero(rc_t{}), x2 = x1;
            const int* pf = sPv + f * 2 * M;
            const int* qf = pf + M;
            const rc_t* Af = inv + f * (LOW ? (int)(L.fG / sizeof(float2)) : MM);
            const int pa = pf[a] * M, pc = pf[c] * M;
            for (int j = 0; j < M; ++j) {
              const int fj = pf[j] * M;
              if (low_adj) {
                const float4* Fp = reinterpret_cast<const float4*>(sF) + f * MM;
                const float4 u = Fp[fj + c], v = Fp[fj + a];
                rmac(x1, Af[pa + j], rc_t{u.x, u.z});
                rmac(x2, Af[pc + j], rc_t{v.x, v.z});
              } else {
                rmac(x1, Af[pa + j], Fm[fj + c]);
                if (LOW || a != c) rmac(x2, Af[pc + j], Fm[fj + a]);
              }
            }
            const rc_t g1 = Af[pa + qf[c]], g2 = Af[pc + qf[a]];
            rc_t zr = rzero(rc_t{}), zi = zr;
            const rc_t* d3f = sd3 + f * nt;
            if constexpr (LOW) {
              const float2* ts = Tst + pr;
#pragma unroll 4
              for (int bb = 0; bb < nt; ++bb) {
                const float2 tv = ld_cg(ts + (size_t)bb * NP), d = d3f[bb];
                zr.x = rfma(tv.x, d.x, zr.x); zr.y = rfma(tv.y, d.x, zr.y);
                zi.x = rfma(tv.x, d.y, zi.x); zi.y = rfma(tv.y, d.y, zi.y);
              }
            } else {
              const double2* t = Tt + pr;
#pragma unroll 4
              for (int bb = 0; bb < nt; ++bb) {
                const double2 tv = ld_cg(t + (size_t)bb * NP);
                const rc_t d = d3f[bb];
                zr.x = rfma(tv.x, d.x, zr.x); zr.y = rfma(tv.y, d.x, zr.y);
                zi.x = rfma(tv.x, d.y, zi.x); zi.y = rfma(tv.y, d.y, zi.y);
              }
            }
            if (f < nv) {
              // Tr X^2 and 2 Tr(S^{-1} B D^3 B^+): the pair's (a, c) and (c, a) terms
              const rr_t z1x = zr.x - zi.y, z1y = zr.y + zi.x;  // (a, c)
              const rr_t z2x = zr.x + zi.y, z2y = zi.x - zr.y;  // (c, a)
              const rr_t xx = a == c ? rfma(x1.x, x1.x, -x1.y * x1.y)
                                     : rr_t(2) * rfma(x1.x, x2.x, -x1.y * x2.y);
              rr_t s = rfma(g1.x, z2x, -g1.y * z2y);
              if (a != c) s = rfma(g2.x, z1x, rfma(-g2.y, z1y, s));
              s = rfma(rr_t(2), s, xx);
              if constexpr (LOW) {
                pair2_add(low_h, low_l, make_float2(a == c ? x1.x : 0.f, s));
                if (have_gbar) pair2_add(low_xh, low_xl, make_float2(xx, 0.f));
              } else {
                if (a == c) acc_tr += x1.x;
                acc_g2 += s;
                if (have_gbar) acc_mu += cb * wk * xx;
              }
            }
          }
          if constexpr (LOW) {
            acc_tr += widen(low_h.x) + widen(low_l.x);
            acc_g2 += widen(low_h.y) + widen(low_l.y);
            if (have_gbar) acc_mu += cb * wk * (widen(low_xh.x) + widen(low_xl.x));
          }
          __syncwarp();
        }
        if constexpr (LOW) {
          // S^{-1} in the orbitals' order for rho_k, and for G_loc and the adjoint one step of
          // refinement, S^{-1} = X0 + X0 R with R = I - S X0 from S in FP32 pairs: 1e-15 of the FP64 inverse at
          // these frequencies, where the FP64 elimination takes 1,500 FP64 instructions a matrix
          // at m = 20.
          const float4* Sp = reinterpret_cast<const float4*>(A);
          float2* X0 = sG + mf * (L.fG / sizeof(float2));
          float2* R = reinterpret_cast<float2*>(A);  // over the rows of S that are done with
          const bool refine = (p.mode & (kGloc | kAdj)) != 0;
          if (refine) {
            // (LW entries of R take as many bytes as LW / 2 of S, and a round finishes more than that)
            for (int i0 = 0; i0 < MM; i0 += LW) {
              const int i = i0 + sl, a = i / M, c = i - a * M;
              cf acc = czero();
              if (i < MM) {
                const int qc = sq[c];
                if (a == c) acc.rh = 1.f;
                for (int x = 0; x < M; ++x) cacc1(acc, cneg(ld4(Sp[a * M + x])), X0[sp[x] * M + qc]);
              }
              __syncwarp();
              if (i < MM) R[i] = make_float2(__fadd_rn(acc.rh, acc.rl), __fadd_rn(acc.ih, acc.il));
            }
            __syncwarp();
          }
          float2* Gn = R + MM;
          float4* Ap = reinterpret_cast<float4*>(sM) + mf * MM;  // (adjoint)
          for (int i = sl; i < MM; i += LW) {
            const int a = i / M, c = i - a * M, pa = sp[a] * M;
            const float2 g = X0[pa + sq[c]];
            float2 h = g;
            if (refine) {
              float2 d = make_float2(0.f, 0.f), l;
              for (int x = 0; x < M; ++x) fmac(d, X0[pa + sq[x]], R[x * M + c]);
              two_sum(g.x, d.x, h.x, l.x);
              two_sum(g.y, d.y, h.y, l.y);
              if (adj) Ap[i] = make_float4(h.x, l.x, h.y, l.y);
              else if (mine)
                gq_put(&out[i], q, make_double2(wk * (widen(h.x) + widen(l.x)), wk * (widen(h.y) + widen(l.y))));
            }
            if (!adj) Gn[i] = h;
          }
          __syncwarp();
          if (rho)  // by pairs of rows, {Re, Re, Im, Im}
            for (int i = sl; i < (M + 1) / 2 * M; i += LW) {
              const int a = i / M * 2, c = i - a / 2 * M;
              const float2 u = Gn[a * M + c], v = a + 1 < M ? Gn[(a + 1) * M + c] : make_float2(0.f, 0.f);
              reinterpret_cast<float4*>(X0)[i] = make_float4(u.x, v.x, u.y, v.y);
            }
          __syncwarp();
        }
        if (adj) {
          // Sigma_bar = A^+ Ghat A^+ with Ghat = Gbar + c F^+ (c = n_bar 2 / beta), A = S^{-1}: Ghat,
          // then Ghat A^+ over it (whole rows, so that a row is read before it is written), then
          // A^+ (Ghat A^+); Re<Gbar, A F A> = Re Tr(F^+ Sigma_bar) - c Re Tr (A F)^2.  With LOW the
          // matrices and products are FP32 pairs (1e-13 of the FP64 kernel, which is bound by the FP64
          // pipe: 256 k-points x 1024 frequencies of 40 bands, 14 orbitals 44 ms, in pairs 15 ms).
          const int rows = LW / M, ra = sl / M, rb = sl - ra * M;  // (rows >= 1: m <= LW)
          const int64_t gb0 = si.offSig + (int64_t)min(n + mf, n1 - 1) * MM;
          if constexpr (LOW) {
            float4* Gh = reinterpret_cast<float4*>(A);  // (S is dead)
            const float4* Fm = reinterpret_cast<const float4*>(sF) + mf * MM;
            const float4* Ap = reinterpret_cast<const float4*>(sM) + mf * MM;
            float ch, cl;
            split(cb, ch, cl);
            for (int i = sl; i < MM; i += LW) {
              const int a = i / M, c = i - a * M;
              const float4 fv = Fm[c * M + a];
              cf g = have_gbar ? ld4(__ldg(p.Gbd + gb0 + i)) : czero();
              acc_prod(ch, cl, fv.x, fv.y, g.rh, g.rl);
              acc_prod(-ch, -cl, fv.z, fv.w, g.ih, g.il);
              cnorm(g);
              Gh[i] = st4(g);
            }
            __syncwarp();
            for (int a0 = 0; a0 < M; a0 += rows) {
              const int a = a0 + ra;
              const bool in = ra < rows && a < M;
              cf acc = czero();
              if (in)
                for (int x = 0; x < M; ++x) cacc_cb(acc, ld4(Gh[a * M + x]), ld4(Ap[rb * M + x]));
              cnorm(acc);
              __syncwarp();
              if (in) Gh[a * M + rb] = st4(acc);
            }
            __syncwarp();
            for (int i = sl; i < MM; i += LW) {
              const int a = i / M, c = i - a * M;
              cf acc = czero();
              for (int x = 0; x < M; ++x) cacc_ca(acc, ld4(Ap[x * M + a]), ld4(Gh[x * M + c]));
              if (mine) {
                const double2 v = make_double2(widen(acc.rh) + widen(acc.rl), widen(acc.ih) + widen(acc.il));
                gq_put(&out[i], q, make_double2(wk * v.x, wk * v.y));
                if (have_gbar) {
                  const float4 fv = Fm[i];
                  acc_mu -= wk * fma(widen(fv.x) + widen(fv.y), v.x, (widen(fv.z) + widen(fv.w)) * v.y);
                }
              }
            }
          } else {
            double2* Gh = sM + mf * MM;
            const double2* Fm = reinterpret_cast<const double2*>(sF) + mf * MM;
            for (int i = sl; i < MM; i += LW) {
              const int a = i / M, c = i - a * M;
              const double2 fv = Fm[c * M + a];
              double2 g = make_double2(cb * fv.x, -cb * fv.y);
              if (have_gbar) {
                const double2 gb = __ldg(p.gbar + gb0 + i);
                g.x += gb.x;
                g.y += gb.y;
              }
              Gh[i] = g;
            }
            __syncwarp();
            for (int a0 = 0; a0 < M; a0 += rows) {
              const int a = a0 + ra;
              const bool in = ra < rows && a < M;
              double2 acc = make_double2(0.0, 0.0);
              if (in) {
                const int pc = sp[rb] * M;  // A[c][p_x] at column x of row p_c
                for (int x = 0; x < M; ++x) cmac_cb(acc, Gh[a * M + sp[x]], A[pc + x]);
              }
              __syncwarp();
              if (in) Gh[a * M + rb] = acc;
            }
            __syncwarp();
            for (int i = sl; i < MM; i += LW) {
              const int a = i / M, c = i - a * M;
              double2 acc = make_double2(0.0, 0.0);
              const int qa = sq[a];
              // conj(A[x][a]) Mt[x][c], A[x][a] at row p_x, column q_a
              for (int x = 0; x < M; ++x) cmac_ca(acc, A[sp[x] * M + qa], Gh[x * M + c]);
              if (mine) {
                gq_put(&out[i], q, make_double2(wk * acc.x, wk * acc.y));
                if (have_gbar) {
                  const double2 fv = Fm[i];
                  acc_mu -= wk * fma(fv.x, acc.x, fv.y * acc.y);
                }
              }
            }
          }
        }
      }
      if (rho) {
        // S_k of the whole CTA's frequencies: columns S^{-1} B D staged in sY for yf
        // frequencies at a time, then the blocks of G are added to the chunk's sum
        const int nb = ki.nb, tot = min(W * F, n1 - base);
        double2* Sk = p.rho_part + (int64_t)chunk * p.rho_chunk_stride + ki.offH;
        auto mat = [&](int f) { return reinterpret_cast<const double2*>(smraw + L.oS + (f / F) * L.sS) + (f % F) * MM; };
        auto piv = [&](int f) { return reinterpret_cast<const int*>(smraw + L.op + (f / F) * L.sp) + (f % F) * 2 * M; };
        auto dof = [&](int f) { return reinterpret_cast<const double2*>(smraw + L.od + (f / F) * L.sd) + (f % F) * n2; };
        const bool first = (base == n0);
        __syncthreads();
        if constexpr (LOW) {
          // B by pairs of rows, {Re, Re, Im, Im}, 0 beyond M and n2: over the dead arrays like Y, anew
          // for each batch (12 KB from L2 for 4 frequencies at 76 levels and 20 orbitals), since the
          // room it would hold costs the third CTA on an SM: 14.1 -> 12.7 ms for every output of 48
          // k-points x 2048 frequencies at 96 bands (13.2 with the frequency sums in pairs)
          float4* sB = reinterpret_cast<float4*>(smraw + L.oB);
          const int pb = (n2 + 3) & ~3;
          const float2* Bk = bf.Bs + ki.offP;
          for (int i = tid; i < (M + 1) / 2 * pb; i += 32 * W) {
            const int x = i / pb * 2, b = i % pb;
            const float2 zero = make_float2(0.f, 0.f);
            const float2 u = b < n2 ? __ldg(Bk + x * n2 + b) : zero;
            const float2 v = b < n2 && x + 1 < M ? __ldg(Bk + (x + 1) * n2 + b) : zero;
            sB[i] = make_float4(u.x, v.x, u.y, v.y);
          }
          __syncthreads();
        }
        for (int f0 = 0; f0 < tot; f0 += L.yf) {
          const int nf = min(L.yf, tot - f0);
          const bool put = first && f0 == 0;
          // the chunk's sum: the old values are loaded before a thread's products and added after
          // them, so that the L2 latency passes under the arithmetic
          auto old = [&](int at) { return put ? make_double2(0.0, 0.0) : Sk[at]; };
          auto add = [&](int at, double2 o, double2 v) { Sk[at] = make_double2(o.x + v.x, o.y + v.y); };
          if constexpr (LOW) {
            // FP32 products, summed over the nf frequencies in pairs (in FP32 the sums would be off by 1e-8 and
            // the pass 7 % faster) and added to the chunk's FP64 sum once (each FP64 add takes the SM 16
            // clocks).  Rows 1 of G_k are [A, Y], Y = A B D, rows 2 are D B^+ [A, Y] + D: orbitals lie in
            // pairs of rows, {Re, Re, Im, Im}, so that the packed FMAs take two terms of the contraction over
            // them, and columns of a thread lie a third of the matrix apart, so that a warp's loads are
            // consecutive.
            const int KP = (M + 1) / 2, CT = M + n2, pb = (n2 + 3) & ~3;
            const float4* sB = reinterpret_cast<const float4*>(smraw + L.oB);
            const float4* sA = reinterpret_cast<const float4*>(smraw + L.oG);  // [frequency][KP][M]
            const int fA = (int)(L.fG / sizeof(float4));
            float4* sY = reinterpret_cast<float4*>(smraw + L.oY);  // [yf][KP][n2]
            auto dlow = [&](int f, int b) {
              return reinterpret_cast<const float2*>(smraw + L.od + (f / F) * L.sd)[(f % F) * n2 + b];
            };
            // Y: four pairs of orbitals of one band a thread
            const int at = (KP + 3) / 4;
            for (int i = tid; i < nf * at * n2; i += 32 * W) {
              const int r = i / n2, c = i - r * n2, f = r / at, p0 = (r - f * at) * 4;
              const float4* ga[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) ga[u] = sA + (size_t)(f0 + f) * fA + min(p0 + u, KP - 1) * M;
              float2 re[4], im[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) re[u] = im[u] = make_float2(0.f, 0.f);
              auto mac = [&](int x, float br, float bi) {
                const float2 r2 = make_float2(br, br), i2 = make_float2(bi, bi), n2i = make_float2(-bi, -bi);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  const float4 g = ga[u][x];
                  const float2 gr = make_float2(g.x, g.y), gi = make_float2(g.z, g.w);
                  re[u] = __ffma2_rn(gr, r2, re[u]);
                  im[u] = __ffma2_rn(gr, i2, im[u]);
                  re[u] = __ffma2_rn(gi, n2i, re[u]);
                  im[u] = __ffma2_rn(gi, r2, im[u]);
                }
              };
              int x = 0;
              for (; x + 1 < M; x += 2) {
                const float4 b = sB[(x >> 1) * pb + c];
                mac(x, b.x, b.z);
                mac(x + 1, b.y, b.w);
              }
              if (x < M) {
                const float4 b = sB[(x >> 1) * pb + c];
                mac(x, b.x, b.z);
              }
              const float2 d = dlow(f0 + f, c);
#pragma unroll
              for (int u = 0; u < 4; ++u)
                if (p0 + u < KP)
                  sY[(size_t)(f * KP + p0 + u) * n2 + c] =
                      make_float4(fmaf(re[u].x, d.x, -im[u].x * d.y), fmaf(re[u].y, d.x, -im[u].y * d.y),
                                  fmaf(re[u].x, d.y, im[u].x * d.x), fmaf(re[u].y, d.y, im[u].y * d.x));
            }
            __syncthreads();
            // (1,1) and (1,2): the sum over the frequencies
            for (int i = tid; i < KP * CT; i += 32 * W) {
              const int pr = i / CT, c = i - pr * CT, a = 2 * pr;
              const bool two = a + 1 < M;
              const double2 o0 = old(a * nb + c), o1 = two ? old((a + 1) * nb + c) : make_double2(0.0, 0.0);
              const float4* v = c < M ? sA + (size_t)f0 * fA + pr * M + c : sY + pr * n2 + (c - M);
              const int fs = c < M ? fA : KP * n2;
              float2 re = make_float2(v[0].x, v[0].y), im = make_float2(v[0].z, v[0].w);
              float2 rl = make_float2(0.f, 0.f), il = rl;
              for (int f = 1; f < nf; ++f) {
                const float4 w = v[(size_t)f * fs];
                pair2_add(re, rl, make_float2(w.x, w.y));
                pair2_add(im, il, make_float2(w.z, w.w));
              }
              add(a * nb + c, o0, make_double2(widen(re.x) + widen(rl.x), widen(im.x) + widen(il.x)));
              if (two) add((a + 1) * nb + c, o1, make_double2(widen(re.y) + widen(rl.y), widen(im.y) + widen(il.y)));
            }
            // (2,1) and (2,2) in tiles of four rows and CW columns
            constexpr int CW = 3;
            const int ctl = (CT + CW - 1) / CW, ntl = pb / 4 * ctl;
            for (int i = tid; i < ntl; i += 32 * W) {
              const int b0 = (i / ctl) * 4, c0 = i - (i / ctl) * ctl;
              const float4* src[CW];
              int ks[CW], fs[CW];  // steps of a pair of orbitals and of a frequency
#pragma unroll
              for (int w = 0; w < CW; ++w) {
                const int c = min(c0 + w * ctl, CT - 1);
                src[w] = c < M ? sA + (size_t)f0 * fA + c : sY + (c - M);
                ks[w] = c < M ? M : n2;
                fs[w] = c < M ? fA : KP * n2;
              }
              float2 v[4][CW], vl[4][CW];
#pragma unroll
              for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int w = 0; w < CW; ++w) v[u][w] = vl[u][w] = make_float2(0.f, 0.f);
              for (int f = 0; f < nf; ++f) {
                float2 re[4][CW], im[4][CW];
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                  for (int w = 0; w < CW; ++w) re[u][w] = im[u][w] = make_float2(0.f, 0.f);
                for (int k = 0; k < KP; ++k) {
                  float2 yr[CW], yi[CW];
#pragma unroll
                  for (int w = 0; w < CW; ++w) {
                    const float4 y = src[w][(size_t)f * fs[w] + k * ks[w]];
                    yr[w] = make_float2(y.x, y.y);
                    yi[w] = make_float2(y.z, y.w);
                  }
#pragma unroll
                  for (int u = 0; u < 4; ++u) {
                    const float4 b = sB[k * pb + b0 + u];
                    const float2 br = make_float2(b.x, b.y), bi = make_float2(b.z, b.w);
                    const float2 nbi = make_float2(-b.z, -b.w);
#pragma unroll
                    for (int w = 0; w < CW; ++w) {  // conj(b) y
                      re[u][w] = __ffma2_rn(br, yr[w], re[u][w]);
                      im[u][w] = __ffma2_rn(br, yi[w], im[u][w]);
                      re[u][w] = __ffma2_rn(bi, yi[w], re[u][w]);
                      im[u][w] = __ffma2_rn(nbi, yr[w], im[u][w]);
                    }
                  }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  const float2 d = dlow(f0 + f, min(b0 + u, n2 - 1));
#pragma unroll
                  for (int w = 0; w < CW; ++w)
                    pair2_add(v[u][w], vl[u][w],
                              fmul(make_float2(re[u][w].x + re[u][w].y, im[u][w].x + im[u][w].y), d));
                }
              }
              double2 o[4][CW];  // (all loads before the first store)
#pragma unroll
              for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int w = 0; w < CW; ++w)
                  o[u][w] = old((M + min(b0 + u, n2 - 1)) * nb + min(c0 + w * ctl, CT - 1));
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const int bb = b0 + u;
                if (bb >= n2) break;
#pragma unroll
                for (int w = 0; w < CW; ++w) {
                  const int c = c0 + w * ctl;
                  if (c >= CT) break;
                  float2 t = v[u][w], tl = vl[u][w];
                  if (M + bb == c)
                    for (int f = f0; f < f0 + nf; ++f) pair2_add(t, tl, dlow(f, bb));
                  add((M + bb) * nb + c, o[u][w], make_double2(widen(t.x) + widen(tl.x), widen(t.y) + widen(tl.y)));
                }
              }
            }
            __syncthreads();
          } else {
            // (1,1) block
            for (int i = tid; i < MM; i += 32 * W) {
              const int a = i / M, c = i - a * M;
              const double2 o = old(a * nb + c);
              double2 v = make_double2(0.0, 0.0);
              for (int f = f0; f < f0 + nf; ++f) {
                const int* pf = piv(f);
                const double2 g = mat(f)[pf[a] * M + pf[M + c]];
                v.x += g.x;
                v.y += g.y;
              }
              add(a * nb + c, o, v);
            }
            const double2* Bk = bf.B + ki.offP;
            double2* sY = reinterpret_cast<double2*>(smraw + L.oY);
            // (1,2) and (2,1): Y = S^{-1} B D, Z = D B^+ S^{-1}
            for (int i = tid; i < M * n2; i += 32 * W) {
              const int a = i / n2, bb = i - a * n2;
              const double2 o12 = old(a * nb + M + bb), o21 = old((M + bb) * nb + a);
              double2 v12 = make_double2(0.0, 0.0), v21 = v12;
              for (int f = f0; f < f0 + nf; ++f) {
                const int* pf = piv(f);
                const int* qf = pf + M;
                const double2* Af = mat(f);
                double2 y = make_double2(0.0, 0.0), z = y;
                const int pa = pf[a] * M, qa = qf[a];
                for (int x = 0; x < M; ++x) {
                  const int xx = pf[x];  // orbital of column x; also the row of orbital x
                  cmac(y, Af[pa + x], ld_cg(Bk + xx * n2 + bb));
                  cmac_ca(z, ld_cg(Bk + x * n2 + bb), Af[xx * M + qa]);
                }
                const double2 d = dof(f)[bb];
                y = cmul(y, d);
                z = cmul(z, d);
                sY[(size_t)(f - f0) * M * n2 + i] = y;
                v12.x += y.x; v12.y += y.y;
                v21.x += z.x; v21.y += z.y;
              }
              add(a * nb + M + bb, o12, v12);
              add((M + bb) * nb + a, o21, v21);
            }
            __syncthreads();
            // (2,2): d_b (delta_bc + sum_a conj(B_ab) Y_ac)
            for (int i = tid; i < n2 * n2; i += 32 * W) {
              const int bb = i / n2, c = i - bb * n2;
              const double2 o = old((M + bb) * nb + M + c);
              double2 v = make_double2(0.0, 0.0);
              for (int f = f0; f < f0 + nf; ++f) {
                double2 w = make_double2(0.0, 0.0);
                const double2* Y = sY + (size_t)(f - f0) * M * n2 + c;
                for (int a = 0; a < M; ++a) cmac_ca(w, ld_cg(Bk + a * n2 + bb), Y[a * n2]);
                const double2 d = dof(f)[bb];
                if (bb == c) w.x += 1.0;
                cmac(v, d, w);
              }
              add((M + bb) * nb + M + c, o, v);
            }
            __syncthreads();
          }
        }
      }
    }
    // deterministic: xor tree in each warp, then the warps in order
    if (p.mode & (kOcc | kAdj)) {
      acc_tr = warp_sum(acc_tr);
      acc_g2 = warp_sum(acc_g2);
      acc_mu = warp_sum(acc_mu);
      if (lane == 0) {
        s_part[wp][0] = acc_tr;
        s_part[wp][1] = acc_g2;
        s_part[wp][2] = acc_mu;
      }
      __syncthreads();
      if (tid == 0) {
        double v[3] = {0.0, 0.0, 0.0};
        for (int w = 0; w < W; ++w)
          for (int x = 0; x < 3; ++x) v[x] += s_part[w][x];
        if (occ) {
          double* o = p.occ_part + ((int64_t)kk * p.n_chunks + chunk) * 2;
          o[0] = v[0];
          o[1] = v[1];
        }
        if (adj) p.mubar_part[(int64_t)kk * p.n_chunks + chunk] = v[2];
      }
    }
  }
}

// rho_part chunk 0 <- U (sum_c S_c) U^+ in two launches over (k, block of rows), so that a few
// k-points fill the chip: T = (sum_c S_c) U^+ (a row of T needs its row of S alone), then U T.
constexpr int kRotRows = 16;
__global__ void __launch_bounds__(kSetupThreads)
    k_block_rotate1(const KInfo* __restrict__ kinfo, const double2* __restrict__ U,
                    const double2* __restrict__ rho_part, int64_t stride, int n_chunks, double2* __restrict__ T) {
  extern __shared__ __align__(16) unsigned char smraw[];
  double2* sS = reinterpret_cast<double2*>(smraw);  // kRotRows x N
  const KInfo ki = kinfo[blockIdx.x];
  const int N = ki.nb, r0 = blockIdx.y * kRotRows, nr = min(kRotRows, N - r0);
  if (nr <= 0) return;
  const double2* Uk = U + ki.offH;
  for (int e = threadIdx.x; e < nr * N; e += kSetupThreads) {
    const int64_t at = ki.offH + (int64_t)r0 * N + e;
    double2 s = rho_part[at];
    for (int c = 1; c < n_chunks; ++c) {
      const double2 v = rho_part[(int64_t)c * stride + at];
      s.x += v.x;
      s.y += v.y;
    }
    sS[e] = s;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nr * N; e += kSetupThreads) {
    const int i = e / N, j = e - i * N;
    double2 acc = make_double2(0.0, 0.0);
    for (int l = 0; l < N; ++l) cmac_cb(acc, sS[i * N + l], Uk[j * N + l]);
    T[ki.offH + (int64_t)r0 * N + e] = acc;
  }
}

__global__ void __launch_bounds__(kSetupThreads)
    k_block_rotate2(const KInfo* __restrict__ kinfo, const double2* __restrict__ U,
                    const double2* __restrict__ T, double2* __restrict__ out) {
  const KInfo ki = kinfo[blockIdx.x];
  const int N = ki.nb, r0 = blockIdx.y * kRotRows, nr = min(kRotRows, N - r0);
  const double2* Uk = U + ki.offH;
  const double2* Tk = T + ki.offH;
  for (int e = threadIdx.x; e < nr * N; e += kSetupThreads) {
    const int i = r0 + e / N, j = e % N;
    double2 acc = make_double2(0.0, 0.0);
    for (int l = 0; l < N; ++l) cmac(acc, Uk[i * N + l], Tk[l * N + j]);
    out[ki.offH + i * N + j] = acc;
  }
}

size_t reduce_smem(int nbmax, int mmax, bool matrix) {
  return sizeof(double2) * ((size_t)mmax * nbmax + nbmax + (matrix ? (size_t)nbmax * nbmax : 0));
}
bool reduce_in_smem(int nbmax, int mmax, int smem_optin) {
  return reduce_smem(nbmax, mmax, true) <= (size_t)smem_optin - 1024;
}
int reduce_grid(int nbmax, int mmax, int n_k, int smem_optin, int sm_count) {
  const bool in = reduce_in_smem(nbmax, mmax, smem_optin);
  const int per_sm = in ? std::max(1, (int)((size_t)smem_optin / reduce_smem(nbmax, mmax, true))) : 2;
  return std::max(1, std::min(n_k, sm_count * std::min(per_sm, 8)));
}

template <int LW, bool LOW, int PART>
cudaError_t launch_part(const PointParams& p, const BlockForm& b, const BlockLaunch& l, size_t smem, cudaStream_t s) {
  cudaError_t e =
      cudaFuncSetAttribute(k_point_block<LW, LOW, PART>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_point_block<LW, LOW, PART>, cudaFuncAttributePreferredSharedMemoryCarveout,
                           (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  k_point_block<LW, LOW, PART><<<l.n_units * l.n_chunks, 32 * kBlkWarps, smem, s>>>(p, b, l);
  return cudaGetLastError();
}

template <int LW, bool LOW>
cudaError_t launch_lw(const PointParams& p, const BlockForm& b, const BlockLaunch& l, size_t smem, cudaStream_t s) {
  if (p.mode & kAdj) return launch_part<LW, LOW, kWithAdj>(p, b, l, smem, s);
  if (p.mode & kRho) return launch_part<LW, LOW, kWithRho>(p, b, l, smem, s);
  if (LOW && !(p.mode & kOcc)) return launch_part<LW, LOW, LOW ? kGlocOnly : kPlain>(p, b, l, smem, s);
  return launch_part<LW, LOW, kPlain>(p, b, l, smem, s);
}

}  // namespace

size_t block_reduce_ws_elems(int nbmax, int mmax, int smem_optin, int sm_count) {
  if (reduce_in_smem(nbmax, mmax, smem_optin)) return 0;
  return (size_t)nbmax * nbmax * 2 * sm_count;
}

cudaError_t launch_block_reduce(const BlockSetup& b, int smem_optin, int sm_count, cudaStream_t s) {
  const size_t chk = sizeof(double2) * ((size_t)b.mmax * b.nbmax + (size_t)b.mmax * b.mmax);
  cudaError_t e = cudaFuncSetAttribute(k_block_check, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)chk);
  if (e != cudaSuccess) return e;
  k_block_check<<<b.n_k, kSetupThreads, chk, s>>>(b);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const bool in = reduce_in_smem(b.nbmax, b.mmax, smem_optin);
  const size_t smem = reduce_smem(b.nbmax, b.mmax, in);
  e = cudaFuncSetAttribute(k_block_reduce, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_block_reduce<<<reduce_grid(b.nbmax, b.mmax, b.n_k, smem_optin, sm_count), kSetupThreads, smem, s>>>(b, in ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_block_finish(const BlockSetup& b, cudaStream_t s) {
  const size_t ser = sizeof(double) * kBlkSeries * (size_t)b.n2max;
  const size_t smem = sizeof(double2) * (2 * (size_t)b.mmax * b.mmax + (size_t)b.mmax * b.n2max);
  cudaError_t e = cudaFuncSetAttribute(k_block_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_block_finish<<<b.n_k, kSetupThreads, smem, s>>>(b);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_block_series, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ser);
  if (e != cudaSuccess) return e;
  k_block_series<<<b.n_k, kSetupThreads, ser, s>>>(b);
  return cudaGetLastError();
}

int block_batch(int mmax) { return kBlkWarps * (32 / gj64::lanes(mmax)); }

size_t block_smem(int mmax, int n2max, int mode, int low) { return make_layout_b(mmax, n2max, mode, low).bytes; }

cudaError_t launch_point_block(const PointParams& p, const BlockForm& b, const BlockLaunch& l, int low,
                               cudaStream_t s) {
  const size_t smem = block_smem(p.mmax, l.n2max, p.mode, low);
  switch (gj64::lanes(p.mmax) + (low ? 1 : 0)) {
    case 8: return launch_lw<8, false>(p, b, l, smem, s);
    case 9: return launch_lw<8, true>(p, b, l, smem, s);
    case 16: return launch_lw<16, false>(p, b, l, smem, s);
    case 17: return launch_lw<16, true>(p, b, l, smem, s);
    case 32: return launch_lw<32, false>(p, b, l, smem, s);
    default: return launch_lw<32, true>(p, b, l, smem, s);
  }
}

cudaError_t launch_block_rotate(const KInfo* kinfo, int n_k, int nbmax, const double2* U, double2* rho_part,
                                int64_t stride, int n_chunks, double2* T, cudaStream_t s) {
  const dim3 grid(n_k, (nbmax + kRotRows - 1) / kRotRows);
  const size_t smem = sizeof(double2) * kRotRows * nbmax;
  cudaError_t e = cudaFuncSetAttribute(k_block_rotate1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_block_rotate1<<<grid, kSetupThreads, smem, s>>>(kinfo, U, rho_part, stride, n_chunks, T);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_block_rotate2<<<grid, kSetupThreads, 0, s>>>(kinfo, U, T, rho_part);
  return cudaGetLastError();
}

}  // namespace gf
