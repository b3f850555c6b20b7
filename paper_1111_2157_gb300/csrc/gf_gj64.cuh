// FP64 Gauss-Jordan inverses of small matrices, several per warp (device code only): the block
// form's S and the hybridization step's G_loc.
#pragma once

#include "gf_complex.cuh"
#include "gf_internal.cuh"

namespace gf {
namespace gj64 {

using namespace cx;

// Lanes per matrix for m orbitals (m <= 32).
__host__ __device__ inline int lanes(int m) { return m <= 8 ? 8 : (m <= 16 ? 16 : 32); }

// x 2^k by integer arithmetic on the exponent (a product would hold the FP64 pipe); results below the
// normal range become 0, infinity and NaN stay.
__device__ __forceinline__ double scale2(double x, int k) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff, n = e + k;
  if (e == 0x7ff) return x;
  if (e == 0 || n <= 0) return __hiloint2double(hi & (int)0x80000000, 0);
  if (n >= 0x7ff) return __hiloint2double((hi & (int)0x80000000) | 0x7ff00000, 0);
  return __hiloint2double(hi + k * 0x100000, __double2loint(x));
}

// 1 / a with one reciprocal: scaled by a power of two near 1 / max(|Re|, |Im|), so that the squared
// modulus, of [1, 8), neither overflows nor underflows.
__device__ __forceinline__ double2 crcp_scaled(double2 a, unsigned long long key) {
  const int k = 1023 - max((int)(key >> 52), 1);
  const double x = scale2(a.x, k), y = scale2(a.y, k);
  const double q = scale2(rcp_newton(fma(x, x, y * y)), k);
  return make_double2(x * q, -y * q);
}

// Inverses in place of the warp's m x m matrices (m <= LW): LW lanes each, Gauss-Jordan in exchange form with
// partial pivoting and no row interchanges (X[i][c] = A[p_i][q_c], q = p^{-1}).  Every lane
// group holds a valid matrix, so no lane diverges.
template <int LW>
__device__ __forceinline__ void invert(double2* A, int M, double2* rc, int* sp, int sl, int* status) {
  double2* su = rc;
  double2* sc = rc + M;
  int* sq = sp + M;
  bool used = sl >= M;
  for (int j = 0; j < M; ++j) {
    unsigned long long best = used ? 0ULL : pivot_key(A[sl * M + j]);
    int bi = used ? 0x7fffffff : sl;
    for (int off = LW / 2; off; off >>= 1) {
      const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, off);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
      if (ob > best || (ob == best && oi < bi)) {
        best = ob;
        bi = oi;
      }
    }
    if (sl == 0 && (best == 0ULL || best >= 0x7ff0000000000000ULL)) atomicOr(status, kFlagSingular);
    const double2 r = crcp_scaled(A[bi * M + j], best);
    if (sl < M) {
      const double2 u = A[bi * M + sl], l = A[sl * M + j];
      su[sl] = (sl == j) ? r : cmul(u, r);
      sc[sl] = (sl == bi) ? make_double2(-1.0, 0.0) : l;
    }
    if (sl == bi) used = true;
    if (sl == 0) {
      sp[j] = bi;
      sq[bi] = j;
    }
    __syncwarp();
    int i = sl / M, c = sl - (sl / M) * M;
    const int di = LW / M, dc = LW - (LW / M) * M;
    for (int e = sl; e < M * M; e += LW) {
      const double2 l = sc[i], u = su[c];
      double2 v = (i == bi || c == j) ? make_double2(0.0, 0.0) : A[e];
      v.x = fma(-l.x, u.x, fma(l.y, u.y, v.x));
      v.y = fma(-l.x, u.y, fma(-l.y, u.x, v.y));
      A[e] = v;
      i += di;
      c += dc;
      if (c >= M) {
        c -= M;
        ++i;
      }
    }
    __syncwarp();
  }
}

// The same in FP32.
template <int LW>
__device__ __forceinline__ void invert(float2* A, int M, float2* rc, int* sp, int sl, int* status) {
  float2* su = rc;
  float2* sc = rc + M;
  int* sq = sp + M;
  bool used = sl >= M;
  for (int j = 0; j < M; ++j) {
    // key with the row in its low bits: the largest wins, ties go to the lowest row
    unsigned best = used ? 0u : ((pivot_key_s(A[sl * M + j]) & ~31u) | (unsigned)(31 - sl));
    if constexpr (LW == 32) {
      best = __reduce_max_sync(0xffffffffu, best);
    } else {
#pragma unroll
      for (int off = LW / 2; off; off >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, off));
    }
    const int bi = min(31 - (int)(best & 31u), M - 1);
    if (sl == 0 && ((best >> 5) == 0u || (best & ~31u) >= 0x7f800000u)) atomicOr(status, kFlagSingular);
    const float2 r = frcp(A[bi * M + j]);
    if (sl < M) {
      const float2 u = A[bi * M + sl], l = A[sl * M + j];
      su[sl] = (sl == j) ? r : fmul(u, r);
      sc[sl] = (sl == bi) ? make_float2(-1.f, 0.f) : l;
    }
    if (sl == bi) used = true;
    if (sl == 0) {
      sp[j] = bi;
      sq[bi] = j;
    }
    __syncwarp();
    int i = sl / M, c = sl - (sl / M) * M;
    const int di = LW / M, dc = LW - (LW / M) * M;
    for (int e = sl; e < M * M; e += LW) {
      float2 v = (i == bi || c == j) ? make_float2(0.f, 0.f) : A[e];
      fsub_prod(v, sc[i], su[c]);
      A[e] = v;
      i += di;
      c += dc;
      if (c >= M) {
        c -= M;
        ++i;
      }
    }
    __syncwarp();
  }
}

}  // namespace gj64
}  // namespace gf
