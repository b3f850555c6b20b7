// The DMFT self-consistency step around the lattice sums (sm_103a).
//
//   k_eimp_part, k_eimp_reduce E_imp = sum_k w_k P_k H_k P_k^+ - V_DC I   (Eq. E^imp)
//   k_hybridization            Delta(i w_n) = (i w_n + mu) I - E_imp - Sigma(i w_n)
//                                             - G_loc(i w_n)^{-1}          (Eq. dmftloop2)
//                              one to four frequencies per warp, the m x m inverses
//                              in shared memory (gf_gj64.cuh)
// (The orthonormal projectors of Eqs. 6 and 7, k_lowdin, live in gf_eig.cu
// beside the eigensolver they use.)
#include <math.h>
#include <stdint.h>

#include "gf_complex.cuh"
#include "gf_gj64.cuh"
#include "gf_internal.cuh"

namespace gf {

namespace {

using namespace cx;


// part[k][a][b] = w_k (P_k H_k P_k^+)_{ab}, one CTA per k: T = H P^+ (N x m)
// in shared memory, then P T.
__global__ void __launch_bounds__(kThreads)
    k_eimp_part(const KInfo* __restrict__ kinfo, const SInfo* __restrict__ sinfo,
                const double2* __restrict__ H, const double2* __restrict__ P, int mmax,
                double2* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smraw[];
  double2* T = reinterpret_cast<double2*>(smraw);
  const int k = blockIdx.x;
  const KInfo ki = kinfo[k];
  const int N = ki.nb, M = sinfo[ki.sys].m;
  const double2* Hk = H + ki.offH;
  const double2* Pk = P + ki.offP;
  for (int e = threadIdx.x; e < N * M; e += kThreads) {
    const int j = e / M, b = e - (e / M) * M;
    double2 acc = make_double2(0.0, 0.0);
    for (int i = 0; i < N; ++i) cmac_cb(acc, Hk[j * N + i], Pk[b * N + i]);
    T[e] = acc;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < M * M; e += kThreads) {
    const int a = e / M, b = e - (e / M) * M;
    double2 acc = make_double2(0.0, 0.0);
    for (int j = 0; j < N; ++j) cmac(acc, Pk[a * N + j], T[j * M + b]);
    part[(int64_t)k * mmax * mmax + e] = make_double2(ki.w * acc.x, ki.w * acc.y);
  }
}

// out[s][e] = sum over the k of system s of part[k][e] (m_s^2 entries), minus v_dc[s] on the
// diagonal.  kRedE consecutive entries per CTA and 32 k-strides each, summed in a fixed tree: one
// CTA per system left a chain of n_k loads per entry (0.25 -> 0.02 ms at 1000 k-points).
constexpr int kRedE = 8;
__global__ void __launch_bounds__(32 * kRedE)
    k_eimp_reduce(const SInfo* __restrict__ sinfo, const double2* __restrict__ part, int mmax,
                  const double* __restrict__ v_dc, double2* __restrict__ out) {
  __shared__ double2 s_v[32][kRedE];
  const SInfo si = sinfo[blockIdx.y];
  const int M = si.m, t = threadIdx.x % kRedE, r = threadIdx.x / kRedE, e = blockIdx.x * kRedE + t;
  double2 acc = make_double2(0.0, 0.0);
  if (e < M * M)
    for (int k = si.k0 + r; k < si.k1; k += 32) {
      const double2 v = part[(int64_t)k * mmax * mmax + e];
      acc.x += v.x;
      acc.y += v.y;
    }
  s_v[r][t] = acc;
  for (int h = 16; h; h >>= 1) {
    __syncthreads();
    if (r < h) {
      s_v[r][t].x += s_v[r + h][t].x;
      s_v[r][t].y += s_v[r + h][t].y;
    }
  }
  if (r == 0 && e < M * M) {
    acc = s_v[0][t];
    if (e / M == e % M && v_dc) acc.x -= v_dc[blockIdx.y];
    out[si.offSinf + e] = acc;
  }
}

constexpr int kHybWarps = 4;

// Delta for 32 / LW frequencies of one system per warp.  Bound by the FP64 pipe: in place with
// LW lanes per matrix the elimination keeps 94 % of the lanes at m = 14, where one row per lane of
// [G | I] kept 44 % and took twice the columns (0.17 -> 0.04 ms at 1024 frequencies, m = 14).
template <int LW>
__global__ void __launch_bounds__(32 * kHybWarps)
    k_hybridization(const SInfo* __restrict__ sinfo, int n_iw, int mmax, const double* __restrict__ mu,
                    const double2* __restrict__ eimp, const double2* __restrict__ Sig,
                    const double2* __restrict__ gloc, double2* __restrict__ delta, int* status) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int F = 32 / LW;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sl = lane % LW, mf = lane / LW;
  const int n0 = (blockIdx.x * kHybWarps + warp) * F, s = blockIdx.y;
  if (n0 >= n_iw) return;
  const SInfo si = sinfo[s];
  const int M = si.m, MM = M * M, n = min(n0 + mf, n_iw - 1);  // the last warp repeats its last one
  const size_t wstride = 16 * (size_t)F * (mmax * mmax + 2 * mmax) + 8 * (size_t)F * mmax;
  unsigned char* wb = smraw + warp * ((wstride + 15) & ~(size_t)15);
  double2* A = reinterpret_cast<double2*>(wb) + mf * MM;
  double2* rc = reinterpret_cast<double2*>(wb) + F * mmax * mmax + mf * 2 * M;
  int* sp = reinterpret_cast<int*>(wb + 16 * (size_t)F * (mmax * mmax + 2 * mmax)) + mf * 2 * M;
  const int64_t off = si.offSig + (int64_t)n * MM;
  for (int e = sl; e < MM; e += LW) A[e] = gloc[off + e];
  __syncwarp();
  gj64::invert<LW>(A, M, rc, sp, sl, status);
  const int* sq = sp + M;
  const double wn = (2.0 * n + 1.0) * 3.14159265358979323846 / si.beta;
  if (n0 + mf >= n_iw) return;
  for (int e = sl; e < MM; e += LW) {
    const int i = e / M, c = e - i * M;
    const double2 g = A[sp[i] * M + sq[c]], sg = Sig[off + e], ei = eimp[si.offSinf + e];
    double2 v = make_double2(-ei.x - sg.x - g.x, -ei.y - sg.y - g.y);
    if (i == c) {
      v.x += mu[s];
      v.y += wn;
    }
    delta[off + e] = v;
  }
}

template <int LW>
cudaError_t launch_hyb(const SInfo* sinfo, int n_sys, int n_iw, int mmax, const double* mu, const double2* eimp,
                       const double2* Sig, const double2* gloc, double2* delta, int* status, cudaStream_t s) {
  constexpr int F = 32 / LW;
  const size_t w = 16 * (size_t)F * (mmax * mmax + 2 * mmax) + 8 * (size_t)F * mmax;
  const size_t smem = kHybWarps * ((w + 15) & ~(size_t)15);
  cudaError_t e = cudaFuncSetAttribute(k_hybridization<LW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_hybridization<LW><<<dim3((n_iw + kHybWarps * F - 1) / (kHybWarps * F), n_sys), 32 * kHybWarps, smem, s>>>(
      sinfo, n_iw, mmax, mu, eimp, Sig, gloc, delta, status);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_eimp(const KInfo* kinfo, const SInfo* sinfo, int n_k, int n_sys, const double2* H,
                        const double2* P, int nbmax, int mmax, double2* part, const double* v_dc,
                        double2* out, cudaStream_t s) {
  const size_t smem = (size_t)nbmax * mmax * sizeof(double2);
  cudaError_t e0 = cudaFuncSetAttribute(k_eimp_part, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e0 != cudaSuccess) return e0;
  k_eimp_part<<<n_k, kThreads, smem, s>>>(kinfo, sinfo, H, P, mmax, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_eimp_reduce<<<dim3((mmax * mmax + kRedE - 1) / kRedE, n_sys), 32 * kRedE, 0, s>>>(sinfo, part, mmax, v_dc, out);
  return cudaGetLastError();
}

cudaError_t launch_hybridization(const SInfo* sinfo, int n_sys, int n_iw, int mmax, const double* mu,
                                 const double2* eimp, const double2* Sig, const double2* gloc,
                                 double2* delta, int* status, cudaStream_t s) {
  switch (gj64::lanes(mmax)) {
    case 8: return launch_hyb<8>(sinfo, n_sys, n_iw, mmax, mu, eimp, Sig, gloc, delta, status, s);
    case 16: return launch_hyb<16>(sinfo, n_sys, n_iw, mmax, mu, eimp, Sig, gloc, delta, status, s);
    default: return launch_hyb<32>(sinfo, n_sys, n_iw, mmax, mu, eimp, Sig, gloc, delta, status, s);
  }
}

}  // namespace gf
