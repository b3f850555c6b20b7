// Block form of the lattice points: declarations shared by gf_block.cu (the kernels) and the
// C-ABI translation units.
//
// With P_k^+ = Q [R; 0] (Householder QR, Q unitary N_b x N_b, R upper triangular m x m) the
// frequency-dependent part of A = (i w_n + mu) - H_k - P_k^+ Sigma P_k lives in the first m
// rows and columns of Q^+ A Q.  The other n2 = N_b - m rows hold H_k alone, so one Hermitian
// eigenproblem of that n2 x n2 block per uploaded H_k makes them diagonal for every frequency:
//   z = i w_n + mu,   D = diag(d_b),  d_b = 1 / (z - e_b),
//   S(z) = z O - H11 - Sigma(i w_n) - B D B^+                        (m x m)
//   P G P^+ = S^{-1},  F = dS/dz = O + B D^2 B^+,  P G^2 P^+ = S^{-1} F S^{-1},
//   Tr G   = sum_b d_b + Tr(S^{-1} F),
//   Tr G^2 = sum_b d_b^2 + Tr((S^{-1} F)^2) + 2 Tr(S^{-1} B D^3 B^+),
//   G = U [[S^{-1}, S^{-1} B D], [D B^+ S^{-1}, D + D B^+ S^{-1} B D]] U^+,
// exactly, with O = (P P^+)^{-1}, H11 = R^{-1} Q1^+ H Q1 R^{-+}, B = R^{-1} Q1^+ H Q2 V and
// U = [Q1 R^{-+} | Q2 V] (V: eigenvectors of the n2 x n2 block).  A point costs
// (N_b - m) m^2 + O(m^3) complex multiply-adds instead of N_b^3.
#pragma once

#include "gf_internal.cuh"

namespace gf {

constexpr int kBlkMaxM = 32;    // orbitals: one lane per row of S
constexpr int kBlkWarps = 4;    // warps per CTA of the point kernels

// Device arrays of the block form of every k-point.
struct BlockForm {
  const double* e;        // [n2] at offD[k]
  const int64_t* offD;
  const double2* T;       // [n2][np] at offT[k]: B_ab conj(B_cb) over the pairs a <= c, np = m(m+1)/2
  const float2* Ts;       // its FP32 rounding and FP32 pairs (GF_PREC_MIXED), or null
  const float4* Tp;
  const int64_t* offT;
  const double2* B;       // [m][n2] at KInfo::offP
  const float2* Bs;
  const double2* HO;      // [2][np] per k at k * 2 * npmax: H11 pairs, then O pairs
  int npmax;
  // Chebyshev moments of the n2 block: with e_b in [c - r, c + r] and x_b = (e_b - c) / r,
  // sum_b t_b / (z - e_b)^p = sum_j a_j^(p)(z) C_j, C_j = sum_b t_b T_j(x_b), whose terms fall
  // off like R^-j, R the sum of the half axes of the ellipse with foci c -+ r through z.
  const double2* C;       // [min(n2, kBlkSeries)][np] at offC[k]
  const float2* Cs;       // its FP32 rounding and FP32 pairs (GF_PREC_MIXED), or null
  const float4* Cp;
  const int64_t* offC;
  const double* tau;      // [kBlkSeries] per k: sum_b T_j(x_b)
  const double2* cr;      // (c, r) per k
};
constexpr int kBlkSeries = 40;  // moments kept

// Terms of the series that leave a remainder of e^-bits for every frequency from w on, bits with a
// margin for the j^2 of the third powers (FP32: only the count depends on it).
__device__ __forceinline__ int series_terms(float dx, float w, float r, float bits) {
  const float xr = dx / r, xi = w / r;
  if (!(fabsf(xr) < 1e9f && xi < 1e9f)) return 1 << 20;  // (x^4 leaves the FP32 range)
  const float ur = xr * xr - xi * xi - 1.f, ui = 2.f * xr * xi, au = sqrtf(ur * ur + ui * ui);
  const float p = sqrtf(0.5f * (au + fabsf(ur))), h = p > 0.f ? 0.5f * fabsf(ui) / p : 0.f;
  const float sr = ur >= 0.f ? p : h, si = ur >= 0.f ? h : p;
  const float R = sqrtf((fabsf(xr) + sr) * (fabsf(xr) + sr) + (fabsf(xi) + si) * (fabsf(xi) + si));
  const float lr = logf(R);
  return lr > 0.02f ? (int)(bits / lr) + 2 : 1 << 20;
}

// One launch over units (k-points, or k-groups for the k-reductions) x frequency chunks.
struct BlockLaunch {
  int n_units, unit0;     // units [unit0, unit0 + n_units)
  const int2* units;      // {first entry of kperm, count} per unit
  const int* kperm;
  int n_begin, n_end;     // frequencies [n_begin, n_end)
  int chunk_w, n_chunks;  // chunks of this launch
  int chunk0;             // index of the first one in the per-chunk partial sums
  int n2max;
};

// Setup over the k-points: check and QR, Q^+ H Q, eigenpairs of the n2 block, and the
// tables above.  flags (device int): kBlkNonHermitian, kBlkIllConditioned,
// kBlkNoConvergence; hnorm (device, n_k): ||H_k||_F / sqrt(N_b).
constexpr int kBlkNonHermitian = 1, kBlkIllConditioned = 2, kBlkNoConvergence = 4;
struct BlockSetup {
  const double2* H;
  const double2* P;
  const KInfo* kinfo;
  const SInfo* sinfo;
  int n_k, nbmax, mmax, n2max, npmax;
  double cond, range;     // largest condition number of O, and of |R|^2 and |R^{-1}|^2
  double2* D22;           // [n2][n2] at offH: the n2 block, then its eigenvectors
  double2* V;             // [m][N_b] at offP: Householder vectors (row j: vector j)
  double2* Ri;            // [m][m] at k * mmax^2: R^{-1}
  double* tau;            // [m] at k * mmax
  double2* H11;           // [m][m] at k * mmax^2
  double2* B;             // [m][n2] at offP: Q1^+ H Q2, then B
  double* e;              // [n2] at offD
  const int64_t* offD;
  double2* T;
  float2* Ts;
  float4* Tp;
  const int64_t* offT;
  float2* Bs;
  double2* HO;
  double2* U;             // [N_b][N_b] at offH
  double2* C;             // Chebyshev moments, as in BlockForm
  float2* Cs;
  float4* Cp;
  const int64_t* offC;
  double* series;         // tau, then (c, r) pairs
  double2* ws;            // per-CTA slices of nbmax^2 elements when the matrix exceeds shared memory
  int* flags;
  double* hnorm;
};
cudaError_t launch_block_reduce(const BlockSetup& b, int smem_optin, int sm_count, cudaStream_t s);  // (two kernels)
cudaError_t launch_block_eig(const BlockSetup& b, double2* ws, int grid, int in_smem, cudaStream_t s);
cudaError_t launch_block_finish(const BlockSetup& b, cudaStream_t s);  // (two kernels)
size_t block_reduce_ws_elems(int nbmax, int mmax, int smem_optin, int sm_count);

// Frequencies a CTA takes at once.
int block_batch(int mmax);
// low = 1 (the higher frequencies of mixed precision): traces and rho_k in FP32, S, G_loc and the
// adjoint in FP32 pairs, S^{-1} in FP32 with one refinement step.
size_t block_smem(int mmax, int n2max, int mode, int low);
cudaError_t launch_point_block(const PointParams& p, const BlockForm& b, const BlockLaunch& l, int low,
                               cudaStream_t s);
// Mixed-precision N(mu) passes: the FP32 kernel (gf_block32.cu), frequencies of a CTA batch and
// shared memory.
int block32_batch(int mmax);
size_t block32_smem(int mmax, int n2max);
cudaError_t launch_occ_block32(const PointParams& p, const BlockForm& b, const BlockLaunch& l, cudaStream_t s);
// rho_part chunk 0 <- U (sum_c S_c) U^+ for every k; T: scratch of the size of H.
cudaError_t launch_block_rotate(const KInfo* kinfo, int n_k, int nbmax, const double2* U, double2* rho_part,
                                int64_t stride, int n_chunks, double2* T, cudaStream_t s);

}  // namespace gf
