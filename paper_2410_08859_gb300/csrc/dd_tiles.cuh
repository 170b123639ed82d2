// Row passes of a separable log-sum-exp in double, by tiles of targets.
#pragma once
#include <algorithm>
#include <cmath>

#include "dd_common.cuh"

namespace {

constexpr int kSepBlock = 16;    // sources per block maximum
constexpr int kTile = 8;         // consecutive targets of one line per group of lanes
// Four lanes: the whole adjoint at eps = 4 h^2, four | eight lanes: N = 192 467 | 469 us, 256 576 | 587,
// 320 655 | 686, 384 730 | 815, 512 964 | 1102, 1024 3151 | 3750 (eight halve a lane's share of a window
// but double the searches for maxima).
constexpr int kTileLanes = 4;
constexpr int kTileMinN = 192;   // smallest grid of the tile passes (few tiles below: their FP64 latency shows)

// One row pass in double: line k = blockIdx.x, L(j) = log2 sum_m 2^{f(k, m) - q2 (j - m)^2}
// for the targets blockIdx.y * per + [0, per), a tile of kTile consecutive targets
// per group of kTileLanes lanes.
// With the tile's anchor a and a centre c of its sources,
//   2^{f(m) - q2 (m - a - k)^2} = G(m) 2^{2 q2 (m - c) k} 2^{2 q2 (c - a) k - q2 k^2},
//   G(m) = 2^{f(m) - q2 (m - a)^2}:
// one exponential per source and tile, then one multiply-add per term with a
// power from a table of 2^{2 q2 n}; the last factor does not depend on m and is
// added to the logarithm.  Per term 1 + 11/8 FP64 operations (two lanes a clock)
// instead of 12.  Only sources within 2^-65 of some target's shift are used
// (maxima of blocks of 16, then a float test).  The powers cover
// |n| <= D4 and 2^{+-400}, so that G stays a normal number for every term that
// counts; a tile whose window is wider, and a target whose sum leaves
// [2^-29, 2^59] of its float maximum, is summed term by term.  The rounding of a
// power's exponent (|2 q2 n| <= 400: below 1e-13) is that of f - q2 d^2 itself at
// |f| ~ 1000.
// MOM >= 1 also carries the mean of m - j under the terms, MOM == 2 that of mom(k, m):
// one and two more multiply-adds a term.
// out(j, L, mean1, mean2) is called once per target by consecutive threads.
// One pass without moments at eps = 4 h^2, against one exponential per term (12
// operations): 1024 x 1024 1093 -> 344 us, 512 x 512 283 -> 96, 256 x 256 81 -> 43.
template <int MOM, typename Out>
__device__ __forceinline__ void tile_rows(unsigned char* sm, const double* __restrict__ src,
                                          const float* __restrict__ srcf, const double* __restrict__ mom,
                                          int N, double q2, int per, int D4, Out out) {
  double2* qd = reinterpret_cast<double2*>(sm);          // (q2 d, d)
  double* row = reinterpret_cast<double*>(qd + N + kTile);   // an anchor may lie kTile / 2 beyond the line
  double* pw = row + N;                                  // 2^{2 q2 n}, n = -D4..D4
  double* accS = pw + 2 * D4 + 1;
  double* sigS = accS + per;
  double* a1S = sigS + per;                              // MOM >= 1
  double* a2S = a1S + (MOM >= 1 ? per : 0);              // MOM == 2
  double* momr = a2S + (MOM == 2 ? per : 0);             // MOM == 2: mom(k, .)
  float* rowf = reinterpret_cast<float*>(momr + (MOM == 2 ? N : 0));
  float* bm = rowf + N;
  __shared__ double pa[2 * 256 + 1], pb[16];             // 2^{2 q2 16 i}, |i| <= 256, and 2^{2 q2 j}, j < 16
  const int k = blockIdx.x, nb = (N + kSepBlock - 1) / kSepBlock;
  const int j_lo = blockIdx.y * per, j_n = min(per, N - j_lo);
  for (int l = threadIdx.x; l < N; l += blockDim.x) {
    row[l] = src[(long long)k * N + l];
    rowf[l] = srcf[(long long)k * N + l];
    if (MOM == 2) momr[l] = mom[(long long)k * N + l];
  }
  for (int l = threadIdx.x; l < N + kTile; l += blockDim.x) qd[l] = make_double2(q2 * (double)l, (double)l);
  const int na = D4 / 16 + 1;
  if (D4 <= 128) {
    for (int i = threadIdx.x; i < 2 * D4 + 1; i += blockDim.x) pw[i] = dd_ex2(2.0 * q2 * (double)(i - D4));
  } else {   // products of a coarse and a fine power (D4 <= 4095; 2 q2 (D4 + 32) < 1022)
    for (int i = threadIdx.x; i < 2 * na + 1; i += blockDim.x) pa[i] = dd_ex2(2.0 * q2 * (double)(16 * (i - na)));
    for (int i = threadIdx.x; i < 16; i += blockDim.x) pb[i] = dd_ex2(2.0 * q2 * (double)i);
  }
  __syncthreads();   // the line (block maxima) and the coarse and fine powers
  if (D4 > 128) {
    for (int i = threadIdx.x; i < 2 * D4 + 1; i += blockDim.x) {
      const int n = i - D4 + 16 * na;                    // >= 0
      pw[i] = pa[n >> 4] * pb[n & 15];
    }
  }
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    float m = -INFINITY;
    for (int l = b * kSepBlock; l < min(N, (b + 1) * kSepBlock); ++l) m = fmaxf(m, rowf[l]);
    bm[b] = m;
  }
  __syncthreads();
  const float q2f = (float)q2, cutf = 65.0f;
  auto bound = [&](int b, int j) {
    const float d = (float)(j - min(max(j, b * kSepBlock), b * kSepBlock + kSepBlock - 1));
    const float u = fmaf(-q2f * d, d, bm[b]);
    return fmaf(1e-6f, fabsf(bm[b]) + fabsf(u), u);
  };
  auto term_f = [&](int m, int j) {
    const float d = (float)(j - m);
    return fmaf(-(q2f * d), d, rowf[m]);
  };
  // the largest float term of target j (the lanes of a group)
  constexpr int P = kTileLanes;
  const int part = threadIdx.x & (P - 1);
  auto maximum = [&](int j) {
    float ub = -INFINITY, mx = -INFINITY;
    int best = 0;
    for (int b = part; b < nb; b += P) {
      const float u = bound(b, j);
      if (u > ub) { ub = u; best = b; }
    }
    for (int o = 1; o < P; o <<= 1) {
      const float u = __shfl_xor_sync(0xffffffffu, ub, o);
      const int b = __shfl_xor_sync(0xffffffffu, best, o);
      if (u > ub || (u == ub && b < best)) { ub = u; best = b; }
    }
    for (int m = best * kSepBlock + part; m < min(N, (best + 1) * kSepBlock); m += P) mx = fmaxf(mx, term_f(m, j));
    for (int o = 1; o < P; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    for (int b = part; b < nb; b += P)
      if (bound(b, j) >= mx)
        for (int m = b * kSepBlock; m < min(N, (b + 1) * kSepBlock); ++m) mx = fmaxf(mx, term_f(m, j));
    for (int o = 1; o < P; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    return mx;
  };
  const int ntile = (j_n + kTile - 1) / kTile, nt = (ntile * P + 31) & ~31;
  for (int i = threadIdx.x; i < nt; i += blockDim.x) {
    const int t0 = min(i / P, ntile - 1) * kTile, n = min(kTile, j_n - t0), j0 = j_lo + t0, a = j0 + kTile / 2;
    const bool own = i / P < ntile;
    float S[kTile];
    bool usable = true;
#pragma unroll
    for (int e = 0; e < kTile; ++e) {
      const float mx = maximum(min(j0 + e, N - 1));
      S[e] = e < n ? mx : INFINITY;
      usable &= e >= n || mx > -INFINITY;
    }
    float Sr = S[0];
#pragma unroll
    for (int e = 1; e < kTile; ++e)
      if (e < n && e <= kTile / 2) Sr = S[e];
    int lo = N, hi = 0;
    if (usable)
      for (int b = part; b < nb; b += P) {
        bool rel = false;
#pragma unroll
        for (int e = 0; e < kTile; ++e) rel |= bound(b, j0 + e) - S[e] > -cutf - 1.0f;
        if (rel) {
          lo = min(lo, b * kSepBlock);
          hi = max(hi, min(N, (b + 1) * kSepBlock));
        }
      }
    for (int o = 1; o < P; o <<= 1) {
      lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    auto covered = [&] { return ((hi - lo) / 2 + 1) * (kTile / 2) <= D4; };
    if (__any_sync(0xffffffffu, usable && !covered())) {   // the exact window instead of whole blocks
      int l2 = N, h2 = 0;
      for (int m = lo + part; m < hi; m += P) {
        float v = -INFINITY;
#pragma unroll
        for (int e = 0; e < kTile; ++e) v = fmaxf(v, term_f(m, j0 + e) - S[e]);
        if (v > -cutf) { l2 = min(l2, m); h2 = max(h2, m + 1); }
      }
      for (int o = 1; o < P; o <<= 1) {
        l2 = min(l2, __shfl_xor_sync(0xffffffffu, l2, o));
        h2 = max(h2, __shfl_xor_sync(0xffffffffu, h2, o));
      }
      lo = l2;
      hi = h2;
    }
    const int c = (lo + hi) / 2;   // |m - c| <= (hi - lo) / 2 + 1
    usable &= hi > lo && covered();
    const double sref = (double)Sr;
    double acc[kTile], a1[MOM >= 1 ? kTile : 1], a2[MOM == 2 ? kTile : 1];
#pragma unroll
    for (int e = 0; e < kTile; ++e) {
      acc[e] = 0.0;
      if (MOM >= 1) a1[e] = 0.0;
      if (MOM == 2) a2[e] = 0.0;
    }
    if (usable)
      for (int m = lo + part; m < hi; m += P) {
        float v = -INFINITY;   // S holds the maxima of these terms: v <= 0
#pragma unroll
        for (int e = 0; e < kTile; ++e) v = fmaxf(v, term_f(m, j0 + e) - S[e]);
        if (v > -cutf) {
          const double2 t = qd[abs(m - a)];
          const double G = dd_ex2(fma(-t.x, t.y, row[m]) - sref);
          const double* w = pw + D4;
          const int dm = m - c;
          double G1 = 0.0, G2 = 0.0;
          if (MOM >= 1) G1 = G * (dm < 0 ? -qd[-dm].y : qd[dm].y);
          if (MOM == 2) G2 = G * momr[m];
#pragma unroll
          for (int e = 0; e < kTile; ++e) {
            const double pe = w[dm * (e - kTile / 2)];
            acc[e] = fma(G, pe, acc[e]);
            if (MOM >= 1) a1[e] = fma(G1, pe, a1[e]);
            if (MOM == 2) a2[e] = fma(G2, pe, a2[e]);
          }
        }
      }
#pragma unroll
    for (int e = 0; e < kTile; ++e)
      for (int o = 1; o < P; o <<= 1) {
        acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
        if (MOM >= 1) a1[e] += __shfl_xor_sync(0xffffffffu, a1[e], o);
        if (MOM == 2) a2[e] += __shfl_xor_sync(0xffffffffu, a2[e], o);
      }
    // lane `part` keeps targets part, part + P, ...
    bool bad = !usable;
#pragma unroll
    for (int e = 0; e < kTile; ++e)
      if (e < n && (e & (P - 1)) == part) {
        const double kk = (double)(e - kTile / 2);
        const double sig = sref + kk * (2.0 * q2 * (double)(c - a) - q2 * kk);
        const int hx = __double2hiint(acc[e]);
        // log2 of the sum against the target's own shift, to a bit
        const float r = (float)((hx >> 20) - 1023) + ((float)(sig - sref) + (Sr - S[e]));
        if (hx < 0x00100000 || hx >= 0x7ff00000 || !(r >= -29.0f && r <= 58.0f)) bad = true;
        if (own) {
          accS[t0 + e] = acc[e];
          sigS[t0 + e] = sig;
          // sum of w (m - j) = sum of w (m - c) + (c - j) sum of w
          if (MOM >= 1) a1S[t0 + e] = fma((double)(c - a) - kk, acc[e], a1[e]);
          if (MOM == 2) a2S[t0 + e] = a2[e];
        }
      }
    for (int o = 1; o < P; o <<= 1) bad |= __shfl_xor_sync(0xffffffffu, (int)bad, o) != 0;
    if (__any_sync(0xffffffffu, bad)) {
      __syncwarp();   // lane 0 of a group replaces what the group's lanes have stored above
      // term by term against each target's maximum
      for (int e = 0; e < kTile; ++e) {
        const int j = min(j0 + e, N - 1);
        const float mx = maximum(j);
        const double mxd = (double)mx;
        double b2 = mx > -INFINITY ? 0.0 : 1.0, b1 = 0.0, b3 = 0.0;
        if (mx > -INFINITY)
          for (int m = part; m < N; m += P)
            if (term_f(m, j) - mx > -cutf) {
              const double2 t = qd[abs(m - j)];
              const double w = dd_ex2(fma(-t.x, t.y, row[m]) - mxd);
              b2 += w;
              if (MOM >= 1) b1 += w * (m < j ? -t.y : t.y);
              if (MOM == 2) b3 += w * momr[m];
            }
        for (int o = 1; o < P; o <<= 1) {
          const double other = __shfl_xor_sync(0xffffffffu, b2, o);
          if (mx > -INFINITY) b2 += other;
          if (MOM >= 1) b1 += __shfl_xor_sync(0xffffffffu, b1, o);
          if (MOM == 2) b3 += __shfl_xor_sync(0xffffffffu, b3, o);
        }
        if (bad && own && part == 0 && e < n) {
          accS[t0 + e] = b2;
          sigS[t0 + e] = mxd;
          if (MOM >= 1) a1S[t0 + e] = b1;
          if (MOM == 2) a2S[t0 + e] = b3;
        }
      }
    }
    __syncwarp();
  }
  __syncthreads();
  for (int t = threadIdx.x; t < j_n; t += blockDim.x) {
    double m1 = 0.0, m2 = 0.0;
    if (MOM >= 1) {
      const double ia = 1.0 / accS[t];
      m1 = a1S[t] * ia;
      if (MOM == 2) m2 = a2S[t] * ia;
    }
    out(j_lo + t, sigS[t] + dd_lg2(accS[t]), m1, m2);
  }
}

// Launch shape of a tile pass.  A row is split over several CTAs (at least 64 targets each) where
// the rows alone are fewer than four per SM: the whole adjoint at eps = 4 h^2, split | one CTA a
// row (eight lanes a tile): N = 192 461 | 506 us, 320 675 | 740, 384 809 | 842, 512 961 | 1023; at 256 and 448 the
// split costs 5 % (575 | 546, 855 | 813); from 608 on it is the same.
struct TileShape {
  int per, threads, D4;
  size_t smem;
  dim3 grid;
};
inline TileShape tile_shape(int N, double q2, int mom) {
  TileShape t;
  const int gy = std::max((N + 1023) / 1024, std::min((N + 63) / 64, (608 + N - 1) / N));
  t.per = ((N + gy - 1) / gy + kTile - 1) / kTile * kTile;
  t.threads = std::min(512, ((t.per / kTile * kTileLanes + 31) / 32) * 32);
  // table: twice the reach of a term within the cut plus the blocks' width, within the exponent range
  const double reach = 2.0 * std::sqrt(66.0 / q2) + 48.0;
  const int D = (int)std::min({(double)N, reach, 1023.0});
  t.D4 = std::max(0, std::min(D * (kTile / 2), (int)std::min(4092.0, 200.0 / q2)));   // |2 q2 n| <= 400
  const int nb = (N + kSepBlock - 1) / kSepBlock;
  t.smem = sizeof(double) * ((3 + (mom == 2)) * (size_t)N + 2 * kTile + 1 + (2 + mom) * (size_t)t.per) +
           sizeof(float) * ((size_t)N + nb) + 16;
  const size_t budget = 216 * 1024;   // of 227 KB, beside the static arrays
  t.D4 = std::min(t.D4, t.smem < budget ? (int)((budget - t.smem) / 16) : 0);
  t.smem += 2 * sizeof(double) * (size_t)t.D4;
  t.grid = dim3(N, (N + t.per - 1) / t.per);
  return t;
}

}  // namespace
