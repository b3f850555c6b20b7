// Block form of the lattice points (gf_block.cuh): the FP32 kernel of mixed-precision N(mu)
// passes, for the frequencies whose FP32 rounding stays below that of an FP32 inverse of the
// window (w_n above a fraction of H's scale; k_point_block takes the others in FP64).
//
// A warp takes FW frequencies of one k-point and runs without block barriers:
//   1. d_b = 1 / (z - e_b) and its powers, one (band, frequency) per lane, or the coefficients of
//      the Chebyshev series where that has fewer terms to 2^-24 (the traces of D stay direct: the
//      series' real parts carry the rounding of its moduli);
//   2. band sums of S and F = dS/dz, one orbital pair a <= c per lane and FW frequencies in
//      registers, so that one load of the pair table feeds 8 FW FMAs;
//   3. S^{-1} with LW lanes per matrix, one row per lane in registers (Gauss-Jordan in exchange
//      form, rows rotated one column per pivot, lazy row scales, as warp_invert of
//      gf_warp_gj.cuh), then X = S^{-1} F row by row from the same registers;
//   4. Tr X, Tr X^2, and 2 Tr(S^{-1} B D^3 B^+) from a second sweep over the pair table.
// The sums over frequencies are FP32 pairs within a warp's batch of FW, FP64 over the batches.
//
// Bound by latency: issue slots 46 % and FMA pipe 32 % busy at 11 warps an SM.  N(mu) of 256
// k-points x 1024 frequencies at 40 bands, 14 orbitals: 1.4 ms with the FP64 frequencies beside it;
// the one-warp elimination of the whole window (25 M points/s) takes 10.4 ms.
#include <math.h>
#include <stdint.h>

#include "gf_block.cuh"
#include "gf_complex.cuh"

namespace gf {

namespace {

using namespace cx;

__device__ __forceinline__ float2 z2() { return make_float2(0.f, 0.f); }

// Shared memory (bytes): per CTA x_b = mu - e_b, mu O - H11 and O by pairs and the pair list;
// per warp d, d^2, d^3 as [band][FW], S and F with rows of NMAX entries, the pivot rows and tables.
struct Layout32 {
  size_t oX, oHz, oO, oPair, warp0, wd, ww, wS, wF, wbuf, wp, wstride, bytes;
};

__host__ __device__ inline Layout32 make_layout32(int mmax, int n2max, int nmax, int lw, int fw) {
  Layout32 L;
  auto al = [](size_t x) { return (x + 15) & ~(size_t)15; };
  const size_t np = (size_t)mmax * (mmax + 1) / 2;
  size_t o = 0;
  L.oX = o; o = al(o + 4 * (size_t)n2max);
  L.oHz = o; o = al(o + 8 * np);
  L.oO = o; o = al(o + 8 * np);
  L.oPair = o; o = al(o + 2 * np);
  L.warp0 = o;
  size_t g = 0;
  L.wd = g; g = al(g + 24 * (size_t)fw * n2max);
  L.ww = g; g = al(g + 4 * (size_t)fw);
  L.wS = g; g = al(g + 8 * (size_t)fw * mmax * nmax);
  L.wF = g; g = al(g + 8 * (size_t)fw * mmax * nmax);
  L.wbuf = g; g = al(g + 8 * (size_t)(32 / lw) * nmax);
  L.wp = g; g = al(g + 8 * (size_t)(32 / lw) * nmax);
  L.wstride = g;
  L.bytes = o + kBlkWarps * g;
  return L;
}

template <int NMAX, int LW, int FW>
__global__ void __launch_bounds__(32 * kBlkWarps, NMAX > 24 ? 2 : 3)
    k_occ_block32(const PointParams p, const BlockForm bf, const BlockLaunch bl) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double s_part[kBlkWarps][2];
  constexpr int G = 32 / LW;  // matrices inverted together
  static_assert(FW % G == 0 && FW % 2 == 0 && NMAX % 2 == 0, "batch shape");
  const Layout32 L = make_layout32(p.mmax, bl.n2max, NMAX, LW, FW);
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, sl = lane % LW, mf = lane / LW;
  float* xs = reinterpret_cast<float*>(smraw + L.oX);
  float2* hz = reinterpret_cast<float2*>(smraw + L.oHz);
  float2* oo = reinterpret_cast<float2*>(smraw + L.oO);
  uchar2* pair = reinterpret_cast<uchar2*>(smraw + L.oPair);
  unsigned char* wb = smraw + L.warp0 + (size_t)wp * L.wstride;
  const int unit = bl.unit0 + blockIdx.x / bl.n_chunks, ch = blockIdx.x % bl.n_chunks;
  const int kk = bl.kperm[bl.units[unit].x];  // N(mu) units hold one k-point
  const int n0 = bl.n_begin + ch * bl.chunk_w, n1 = min(bl.n_end, n0 + bl.chunk_w);
  const KInfo ki = p.kinfo[kk];
  const SInfo si = p.sinfo[ki.sys];
  const int M = si.m, n2 = ki.nb - M, NP = M * (M + 1) / 2;
  const double mu = p.mu[ki.sys], pib = M_PI / si.beta;
  const float2* Ts = bf.Ts + bf.offT[kk];
  const float2* Cs = bf.Cs + bf.offC[kk];
  const float cdx = __double2float_rn(mu - bf.cr[kk].x), cr = __double2float_rn(bf.cr[kk].y);
  // the series where it saves four terms, its own cost
  const int jmax = min(min(n2, kBlkSeries), n2 - 4);
  float* sw = reinterpret_cast<float*>(wb + L.ww);
  float2* sd = reinterpret_cast<float2*>(wb + L.wd);
  float2* sd2 = sd + FW * n2;
  float2* sd3 = sd2 + FW * n2;
  float2* sS = reinterpret_cast<float2*>(wb + L.wS);
  float2* sF = reinterpret_cast<float2*>(wb + L.wF);
  float2* sBuf = reinterpret_cast<float2*>(wb + L.wbuf) + mf * NMAX;
  int* sp = reinterpret_cast<int*>(wb + L.wp) + mf * 2 * NMAX;
  int* sq = sp + NMAX;
  for (int b = tid; b < n2; b += 32 * kBlkWarps) xs[b] = __double2float_rn(mu - bf.e[bf.offD[kk] + b]);
  const double2* HO = bf.HO + (size_t)kk * 2 * bf.npmax;
  for (int pr = tid; pr < NP; pr += 32 * kBlkWarps) {
    int a = 0, rem = pr;
    while (rem >= M - a) { rem -= M - a; ++a; }
    pair[pr] = make_uchar2((unsigned char)a, (unsigned char)(a + rem));
    const double2 h = HO[pr], o = HO[bf.npmax + pr];
    hz[pr] = make_float2(__double2float_rn(fma(mu, o.x, -h.x)), __double2float_rn(fma(mu, o.y, -h.y)));
    oo[pr] = make_float2(__double2float_rn(o.x), __double2float_rn(o.y));
  }
  // the padding columns of F (and of X, which takes its place) stay zero
  for (int i = lane; i < FW * M * NMAX; i += 32) sF[i] = z2();
  __syncthreads();
  double acc_tr = 0.0, acc_g2 = 0.0;

  for (int n = n0 + wp * FW; n < n1; n += kBlkWarps * FW) {
    float2 th = z2(), tl = th;  // this lane's sums of (Tr G, Tr G^2) over the warp's frequencies, in pairs
    // 22.6 = 24 ln 2 + 6
    const int J = series_terms(cdx, __double2float_rn((2.0 * n + 1.0) * pib), cr, 22.6f);
    const bool series = J <= jmax;
    const int nt = series ? J : n2;
    const float2* Tt = series ? Cs : Ts;
    if (lane < FW) sw[lane] = __double2float_rn((2.0 * min(n + lane, n1 - 1) + 1.0) * pib);
    __syncwarp();
    for (int i = lane; i < FW * n2; i += 32) {
      const int b = i / FW, f = i - b * FW;
      const float w = sw[f], x = xs[b];
      const float q = __frcp_rn(__fmaf_rn(x, x, __fmul_rn(w, w)));
      const float2 d = make_float2(__fmul_rn(x, q), -__fmul_rn(w, q)), d2 = fmul(d, d);
      if (!series) {
        sd[i] = d;
        sd2[i] = d2;
        sd3[i] = fmul(d2, d);
      }
      if (n + f < n1) {
        pair2_add(th, tl, make_float2(d.x, d2.x));
      }
    }
    if (series) {
      // as series_z of gf_block.cu, with x = (z - c) / r, s = sqrt(x^2 - 1), xi = 1 / (x + s)
      for (int i = lane; i < FW * J; i += 32) {
        const int j = i / FW, f = i - j * FW;
        const float ir = __frcp_rn(cr);
        const float2 x = make_float2(cdx * ir, sw[f] * ir);
        const float2 u = make_float2(fmaf(x.x, x.x, -fmaf(x.y, x.y, 1.f)), 2.f * x.x * x.y);
        const float pr = sqrtf(0.5f * (sqrtf(fmaf(u.x, u.x, u.y * u.y)) + fabsf(u.x))), h = 0.5f * u.y / pr;
        float2 s = u.x >= 0.f ? make_float2(pr, h) : make_float2(h, pr);
        if (s.y < 0.f) s = make_float2(-s.x, -s.y);
        float2 bs = frcp(make_float2(x.x + s.x, x.y + s.y)), pw = make_float2(j ? 2.f : 1.f, 0.f);
#pragma unroll
        for (int t = 0; t < 6; ++t) {
          if ((j >> t) & 1) pw = fmul(pw, bs);
          bs = fmul(bs, bs);
        }
        const float2 is = frcp(s), isr = make_float2(is.x * ir, is.y * ir), t = fmul(x, is);
        const float fj = (float)j;
        const float2 d1 = fmul(pw, isr);
        const float2 c2 = fmul(isr, isr);  // 1 / (s^2 r^2)
        // [j + t] / (s^2 r^2), then [(j^2 - 1) + 3 j t + 3 t^2] / (2 s^3 r^3), t = x / s
        const float2 d2 = fmul(fmul(pw, c2), make_float2(fj + t.x, t.y));
        const float2 t2 = fmul(t, t);
        const float2 d3 = fmul(fmul(fmul(pw, c2), isr),
                               make_float2(0.5f * (fmaf(fj, fj, -1.f) + 3.f * fmaf(fj, t.x, t2.x)),
                                           1.5f * fmaf(fj, t.y, t2.y)));
        sd[i] = d1;
        sd2[i] = d2;
        sd3[i] = d3;
      }
    }
    __syncwarp();
    for (int pr = lane; pr < NP; pr += 32) {
      const int a = pair[pr].x, c = pair[pr].y;
      // packed FMAs: u = sum t.x d and v = sum t.y d, so that xr = (u.x, v.x), xi = (u.y, v.y)
      float2 u[FW], v[FW], yu[FW], yv[FW];
#pragma unroll
      for (int f = 0; f < FW; ++f) u[f] = v[f] = yu[f] = yv[f] = z2();
      const float2* t = Tt + pr;
#pragma unroll 4
      for (int b = 0; b < nt; ++b) {
        const float2 tv = __ldg(t + (size_t)b * NP);
        const float2 tx = make_float2(tv.x, tv.x), ty = make_float2(tv.y, tv.y);
        const float4* d4 = reinterpret_cast<const float4*>(sd + b * FW);
        const float4* e4 = reinterpret_cast<const float4*>(sd2 + b * FW);
#pragma unroll
        for (int f = 0; f < FW; f += 2) {
          const float4 d = d4[f / 2], e = e4[f / 2];
          const float2 d0 = make_float2(d.x, d.y), d1 = make_float2(d.z, d.w);
          const float2 e0 = make_float2(e.x, e.y), e1 = make_float2(e.z, e.w);
          u[f] = __ffma2_rn(tx, d0, u[f]);
          v[f] = __ffma2_rn(ty, d0, v[f]);
          u[f + 1] = __ffma2_rn(tx, d1, u[f + 1]);
          v[f + 1] = __ffma2_rn(ty, d1, v[f + 1]);
          yu[f] = __ffma2_rn(tx, e0, yu[f]);
          yv[f] = __ffma2_rn(ty, e0, yv[f]);
          yu[f + 1] = __ffma2_rn(tx, e1, yu[f + 1]);
          yv[f + 1] = __ffma2_rn(ty, e1, yv[f + 1]);
        }
      }
      const float2 h = hz[pr], o = oo[pr];
#pragma unroll
      for (int f = 0; f < FW; ++f) {
        const int nn = min(n + f, n1 - 1);
        const float w = sw[f];
        const float2* Sg = p.Ss + si.offSig + (int64_t)nn * M * M;
        const float2 s1 = __ldg(Sg + a * M + c), s2 = __ldg(Sg + c * M + a);
        float2* Sm = sS + f * M * NMAX;
        float2* Fm = sF + f * M * NMAX;
        // z o_ac - h_ac - Sigma_ac - g_ac and, with conj(o) and conj(h), (c, a)
        Sm[a * NMAX + c] = make_float2(__fmaf_rn(-w, o.y, h.x) - s1.x - (u[f].x - v[f].y),
                                       __fmaf_rn(w, o.x, h.y) - s1.y - (v[f].x + u[f].y));
        Fm[a * NMAX + c] = make_float2(o.x + (yu[f].x - yv[f].y), o.y + (yv[f].x + yu[f].y));
        if (a != c) {
          Sm[c * NMAX + a] = make_float2(__fmaf_rn(w, o.y, h.x) - s2.x - (u[f].x + v[f].y),
                                         __fmaf_rn(w, o.x, -h.y) - s2.y - (u[f].y - v[f].x));
          Fm[c * NMAX + a] = make_float2(o.x + (yu[f].x + yv[f].y), (yu[f].y - yv[f].x) - o.y);
        }
      }
    }
    __syncwarp();
#pragma unroll 1
    for (int f0 = 0; f0 < FW; f0 += G) {
      const int f = f0 + mf;
      const bool valid = n + f < n1;
      float2* Sm = sS + f * M * NMAX;
      float2* Fm = sF + f * M * NMAX;
      float2 a[NMAX];
#pragma unroll
      for (int c = 0; c < NMAX; c += 2) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (sl < M) {
          const float2 v0 = (c < M) ? Sm[sl * NMAX + c] : z2(), v1 = (c + 1 < M) ? Sm[sl * NMAX + c + 1] : z2();
          v = make_float4(v0.x, v0.y, v1.x, v1.y);
        }
        a[c] = make_float2(v.x, v.y);
        a[c + 1] = make_float2(v.z, v.w);
      }
      bool used = sl >= M;
      float2 sc = make_float2(1.f, 0.f);
#pragma unroll 1
      for (int j = 0; j < M; ++j) {
        unsigned best = used ? 0u : ((pivot_key_s(a[0]) & ~31u) | (unsigned)(31 - sl));
        if constexpr (LW == 32) {
          best = __reduce_max_sync(0xffffffffu, best);
        } else {
#pragma unroll
          for (int off = LW / 2; off; off >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, off));
        }
        const int prow = min(31 - (int)(best & 31u), M - 1);
        if (sl == 0 && valid && ((best >> 5) == 0u || (best & ~31u) >= 0x7f800000u)) atomicOr(p.status, kFlagSingular);
        if (sl == prow) {
#pragma unroll
          for (int c = 0; c < NMAX; c += 2)
            *reinterpret_cast<float4*>(sBuf + c) = make_float4(a[c].x, a[c].y, a[c + 1].x, a[c + 1].y);
          sp[j] = sl;
          sq[sl] = j;
        }
        __syncwarp();
        const float4* b4 = reinterpret_cast<const float4*>(sBuf);
        const float4 u0 = b4[0];
        const float2 r = frcp(make_float2(u0.x, u0.y));
        const bool isp = sl == prow;
        const float2 lq = isp ? z2() : fmul(a[0], r);
        // a_c -= l u_c, each entry moving one register down
        a[0] = a[1];
        fsub_prod(a[0], lq, make_float2(u0.z, u0.w));
#pragma unroll
        for (int c = 2; c < NMAX; c += 2) {
          const float4 u = b4[c / 2];
          a[c - 1] = a[c];
          fsub_prod(a[c - 1], lq, make_float2(u.x, u.y));
          a[c] = a[c + 1];
          fsub_prod(a[c], lq, make_float2(u.z, u.w));
        }
        a[NMAX - 1] = isp ? make_float2(1.f, 0.f) : make_float2(-lq.x, -lq.y);
        if (isp) {
          used = true;
          sc = r;
        }
        __syncwarp();  // the buffer is rewritten by the next pivot
      }
      // this lane: row i = q_sl of S^{-1}; register x holds the stored column (x + M) mod NMAX,
      // which is column p_c of the inverse.  X = S^{-1} F, row i.
      const int row = sl < M ? sq[sl] : 0;
      float2 x[NMAX], xt[NMAX];  // sum g.x F and sum g.y F (packed FMAs)
#pragma unroll
      for (int c = 0; c < NMAX; ++c) x[c] = xt[c] = z2();
#pragma unroll
      for (int y = 0; y < NMAX; ++y) {
        int c = y + M;
        if (c >= NMAX) c -= NMAX;
        if (c < M) {
          const float2 g = fmul(sc, a[y]), gx = make_float2(g.x, g.x), gy = make_float2(g.y, g.y);
          const int pc = sp[c];
          if (sl < M) Sm[row * NMAX + pc] = g;
          const float4* f4 = reinterpret_cast<const float4*>(Fm + pc * NMAX);
#pragma unroll
          for (int z = 0; z < NMAX; z += 2) {
            const float4 v = f4[z / 2];
            const float2 v0 = make_float2(v.x, v.y), v1 = make_float2(v.z, v.w);
            x[z] = __ffma2_rn(gx, v0, x[z]);
            xt[z] = __ffma2_rn(gy, v0, xt[z]);
            x[z + 1] = __ffma2_rn(gx, v1, x[z + 1]);
            xt[z + 1] = __ffma2_rn(gy, v1, xt[z + 1]);
          }
        }
      }
#pragma unroll
      for (int z = 0; z < NMAX; ++z) x[z] = make_float2(x[z].x - xt[z].y, x[z].y + xt[z].x);
      __syncwarp();  // every lane is done with F
      if (sl < M) {
#pragma unroll
        for (int z = 0; z < NMAX; z += 2)
          *reinterpret_cast<float4*>(Fm + row * NMAX + z) = make_float4(x[z].x, x[z].y, x[z + 1].x, x[z + 1].y);
      }
      __syncwarp();
      if (valid && sl < M) {
        float g2 = 0.f;
#pragma unroll
        for (int z = 0; z < NMAX; ++z)
          if (z < M) {
            const float2 y = Fm[z * NMAX + row];
            g2 = __fmaf_rn(x[z].x, y.x, __fmaf_rn(-x[z].y, y.y, g2));
          }
        pair2_add(th, tl, make_float2(Fm[row * NMAX + row].x, g2));
      }
      __syncwarp();
    }
    // 2 Tr(S^{-1} B D^3 B^+)
    for (int pr = lane; pr < NP; pr += 32) {
      const int a = pair[pr].x, c = pair[pr].y;
      float2 u[FW], v[FW];
#pragma unroll
      for (int f = 0; f < FW; ++f) u[f] = v[f] = z2();
      const float2* t = Tt + pr;
#pragma unroll 4
      for (int b = 0; b < nt; ++b) {
        const float2 tv = __ldg(t + (size_t)b * NP);
        const float2 tx = make_float2(tv.x, tv.x), ty = make_float2(tv.y, tv.y);
        const float4* d4 = reinterpret_cast<const float4*>(sd3 + b * FW);
#pragma unroll
        for (int f = 0; f < FW; f += 2) {
          const float4 d = d4[f / 2];
          const float2 d0 = make_float2(d.x, d.y), d1 = make_float2(d.z, d.w);
          u[f] = __ffma2_rn(tx, d0, u[f]);
          v[f] = __ffma2_rn(ty, d0, v[f]);
          u[f + 1] = __ffma2_rn(tx, d1, u[f + 1]);
          v[f + 1] = __ffma2_rn(ty, d1, v[f + 1]);
        }
      }
#pragma unroll
      for (int f = 0; f < FW; ++f) {
        if (n + f >= n1) continue;
        const float2* Sm = sS + f * M * NMAX;
        const float2 g1 = Sm[a * NMAX + c];
        const float z2x = u[f].x + v[f].y, z2y = u[f].y - v[f].x;  // (c, a)
        float s = __fmaf_rn(g1.x, z2x, -__fmul_rn(g1.y, z2y));
        if (a != c) {
          const float2 gt = Sm[c * NMAX + a];
          const float z1x = u[f].x - v[f].y, z1y = v[f].x + u[f].y;  // (a, c)
          s = __fmaf_rn(gt.x, z1x, __fmaf_rn(-gt.y, z1y, s));
        }
        pair2_add(th, tl, make_float2(0.f, 2.f * s));
      }
    }
    __syncwarp();  // d, S and F are rewritten by the next batch
    acc_tr += widen(th.x) + widen(tl.x);
    acc_g2 += widen(th.y) + widen(tl.y);
  }
  // deterministic: xor tree in each warp, then the warps in order
  for (int off = 16; off; off >>= 1) {
    acc_tr += __shfl_xor_sync(0xffffffffu, acc_tr, off);
    acc_g2 += __shfl_xor_sync(0xffffffffu, acc_g2, off);
  }
  if (lane == 0) {
    s_part[wp][0] = acc_tr;
    s_part[wp][1] = acc_g2;
  }
  __syncthreads();
  if (tid == 0) {
    double t = 0.0, u = 0.0;
    for (int w = 0; w < kBlkWarps; ++w) {
      t += s_part[w][0];
      u += s_part[w][1];
    }
    double* o = p.occ_part + ((int64_t)kk * p.n_chunks + bl.chunk0 + ch) * 2;
    o[0] = t;
    o[1] = u;
  }
}

// Shapes by the number of orbitals: columns (registers) per row, lanes per matrix, frequencies
// per warp.
struct Shape32 {
  int nmax, lw, fw;
};
__host__ Shape32 shape32(int m) {
  if (m <= 8) return {8, 8, 4};
  if (m <= 16) return {(m + 1) & ~1, 16, 4};
  if (m <= 20) return {20, 32, 2};
  if (m <= 24) return {24, 32, 2};
  return {32, 32, 2};
}

template <int NMAX, int LW, int FW>
cudaError_t launch32(const PointParams& p, const BlockForm& b, const BlockLaunch& l, size_t smem, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_occ_block32<NMAX, LW, FW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  k_occ_block32<NMAX, LW, FW><<<l.n_units * l.n_chunks, 32 * kBlkWarps, smem, s>>>(p, b, l);
  return cudaGetLastError();
}

}  // namespace

int block32_batch(int mmax) { return kBlkWarps * shape32(mmax).fw; }

size_t block32_smem(int mmax, int n2max) {
  const Shape32 sh = shape32(mmax);
  return make_layout32(mmax, n2max, sh.nmax, sh.lw, sh.fw).bytes;
}

cudaError_t launch_occ_block32(const PointParams& p, const BlockForm& b, const BlockLaunch& l, cudaStream_t s) {
  const size_t smem = block32_smem(p.mmax, l.n2max);
  switch (shape32(p.mmax).nmax) {
    case 8: return launch32<8, 8, 4>(p, b, l, smem, s);
    case 10: return launch32<10, 16, 4>(p, b, l, smem, s);
    case 12: return launch32<12, 16, 4>(p, b, l, smem, s);
    case 14: return launch32<14, 16, 4>(p, b, l, smem, s);
    case 16: return launch32<16, 16, 4>(p, b, l, smem, s);
    case 20: return launch32<20, 32, 2>(p, b, l, smem, s);
    case 24: return launch32<24, 32, 2>(p, b, l, smem, s);
    default: return launch32<32, 32, 2>(p, b, l, smem, s);
  }
}

}  // namespace gf
