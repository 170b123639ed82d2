// Cell subproblem kernel: one CTA per composite cell of a sub-batch.
//
// For cell J with X box X_J (nx1 x nx2 pixels) and Y box B_J (H x W pixels):
//  a1  rho = max(0, P_Y pi - nu_J)/nu on B_J             (Section 5.1, "Computing and handling nu_{-J}")
//  a2  X-half  alpha = -(eps lam/(eps+lam)) log int exp((beta-c)/eps) dnu   (Eq. sinkhorn-X-iteration)
//  a3  Y-half  per y the root of log(rho + e^{beta/eps + z}) + beta/lam = 0 (Eq. proxdiv-problem)
//  a4  stop when PD/lam = KL(P_X pi | e^{-alpha/lam} mu_J) <= err |mu_J|   (Eq. PD-gap-KL)
//  a5  nu~_i(y), C~_i = <c, pi~_i>, H~_i = KL(pi~_i | mu_i x nu) of the new cell plan per
//      member basic cell i, P_X pi~ and the KL_X change for the step-size decision.
//
// GB300 design:
//  * Everything a cell iterates on lives in shared memory; the cost is never stored: c/eps is
//    q |xi - eta|^2 with integer pixel offsets and q = h^2/eps.
//  * |x - y|^2 separates over the two axes, so every log-sum-exp over a rectangle is computed as
//    two 1-D passes (rows, then columns): (nx1 nx2 W + nx1 H W) terms instead of nx1 nx2 H W.
//  * Cell-local frames keep float arithmetic accurate: with x_c, y_c the box centres and
//    D = x_c - y_c (integer), alpha/eps = A + a(xi) + 2 q D.xi and beta/eps = B + b(eta) - 2 q D.eta
//    with A, B per-cell doubles and B = q|D|^2 - A, so that (alpha + beta - c)/eps =
//    a(xi) + b(eta) - q |xi - eta|^2 exactly; a and b stay moderate while alpha/eps is ~1e4-1e5.
//  * exp/log are ex2.approx/lg2.approx in log2 units; each 1-D log-sum-exp is shifted by the
//    previous iteration's value (one pass), with an exact max-shifted fallback.
#include <cooperative_groups.h>

#include <algorithm>

#include "dd_common.cuh"

// Threads per CTA of the cell kernels (the cell body works with any multiple
// of 32 up to 1024; the block reductions assume at most 32 warps).
#ifndef DD_CELL_THREADS
#define DD_CELL_THREADS 512
#endif
constexpr int kCellThreads = DD_CELL_THREADS;

namespace {

template <typename R, typename F>
__device__ __forceinline__ R lse2_1d(F src, int M, R ctr, R q2, R shift, bool use_shift) {
  // log2 sum_m 2^{src(m) - q2 (m - ctr)^2}
  if (use_shift) {
    R a0 = R(0), a1 = R(0);
    R d = -ctr;
    int m = 0;
    for (; m + 1 < M; m += 2) {
      R v0 = src(m) - q2 * d * d - shift;
      d += R(1);
      R v1 = src(m + 1) - q2 * d * d - shift;
      d += R(1);
      a0 += dd_ex2(v0);
      a1 += dd_ex2(v1);
    }
    if (m < M) a0 += dd_ex2(src(m) - q2 * d * d - shift);
    R acc = a0 + a1;
    if (acc > R(1e-25) && acc < R(1e25)) return shift + dd_lg2(acc);
  }
  R mx = -dd_inf<R>();
  R d = -ctr;
  for (int m = 0; m < M; ++m, d += R(1)) mx = max(mx, src(m) - q2 * d * d);
  if (!(mx > -dd_inf<R>())) return mx;
  R acc = R(0);
  d = -ctr;
  for (int m = 0; m < M; ++m, d += R(1)) acc += dd_ex2(src(m) - q2 * d * d - mx);
  return mx + dd_lg2(acc);
}

// One pass of the epilogue statistics against the shift sh: over m in [b, e),
// with d = m - ctr and w = 2^{src(m) - q2 d^2 - sh}, the sums of w,
// w (A(m) - qR d^2) and w ((d + D)^2 + B(m)).
template <typename R, typename F, typename GA, typename GB>
__device__ __forceinline__ void moments_pass(F src, GA A, GB B, R qR, R D, int b, int e, R ctr, R q2, R sh, R& sw,
                                             R& sa, R& sd) {
  sw = sa = sd = R(0);
  R d = R(b) - ctr;
  for (int m = b; m < e; ++m, d += R(1)) {
    const R w = dd_ex2(src(m) - q2 * d * d - sh);
    sw += w;
    sa += w * (A(m) - qR * d * d);
    sd += w * ((d + D) * (d + D) + B(m));
  }
}

// Epilogue statistics of one target over the sources m in [b, e): with
// v_m = src(m) - q2 (m - ctr)^2 (log2 units) returns L = log2 sum_m 2^{v_m} and
// the means m1 = <A(m) - qR d^2>, m2 = <(d + D)^2 + B(m)> under the weights
// 2^{v_m - L} (d = m - ctr).  With use_shift, `shift` is an upper bound of L
// (the full-range log-sum-exp of the same terms): one pass of exponentials
// against it, and only if that sum leaves [1e-30, 1e30] (the sub-range holds a
// negligible share) the exact pass against the maximum.  Without a shift the
// maximum is found first.
template <typename R, typename F, typename GA, typename GB>
__device__ __forceinline__ R lse_moments(F src, GA A, GB B, R qR, R D, int b, int e, R ctr, R q2, R shift,
                                         bool use_shift, R& m1, R& m2) {
  auto maxpass = [&]() {
    R mx = -dd_inf<R>();
    R d = R(b) - ctr;
    for (int m = b; m < e; ++m, d += R(1)) mx = max(mx, src(m) - q2 * d * d);
    return mx;
  };
  R sh = shift;
  if (!use_shift) {
    sh = maxpass();
    if (!(sh > -dd_inf<R>())) {
      m1 = m2 = R(0);
      return sh;
    }
  }
  for (int pass = 0;; ++pass) {
    R sw, sa, sd;
    moments_pass<R>(src, A, B, qR, D, b, e, ctr, q2, sh, sw, sa, sd);
    if (!use_shift || pass == 1 || (sw >= R(1e-30) && sw <= R(1e30))) {
      const R isw = R(1) / sw;
      m1 = sa * isw;
      m2 = sd * isw;
      return sh + dd_lg2(sw);
    }
    // the shift was far from L: the exact pass against the maximum
    sh = maxpass();
    if (!(sh > -dd_inf<R>())) {
      m1 = m2 = R(0);
      return sh;
    }
  }
}

// Partial sum of 2^{src(m) - q2 (m - ctr)^2 - shift} over m = part, part + P, ...
// (eight independent accumulators to keep several ex2 in flight).
template <typename R, typename F>
__device__ __forceinline__ R psum2(F src, int M, R ctr, R q2, R shift, int part, int P) {
  R a[8] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};
  const R dP = R(P);
  R d = R(part) - ctr;
  int m = part;
  for (; m + 7 * P < M; m += 8 * P) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const R dk = d + R(k) * dP;
      a[k] += dd_ex2(src(m + k * P) - q2 * dk * dk - shift);
    }
    d += R(8) * dP;
  }
  for (; m < M; m += P, d += dP) a[0] += dd_ex2(src(m) - q2 * d * d - shift);
  return ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
}

template <typename R, typename F>
__device__ __forceinline__ R pmax2(F src, int M, R ctr, R q2, int part, int P) {
  R mx = -dd_inf<R>();
  const R dP = R(P);
  R d = R(part) - ctr;
  for (int m = part; m < M; m += P, d += dP) mx = max(mx, src(m) - q2 * d * d);
  return mx;
}

// log2 sum_m 2^{src(m) - q2 (m - ctr)^2} computed by the P lanes of an aligned
// lane group (P a power of two dividing 32).  Must be called by all 32 lanes of
// the warp.  With use_shift the sum is taken against `shift` (the previous
// iteration's value) in one pass; if the group's sum leaves the safe range, or
// without a shift, the warp falls back to the exact max-shifted two passes.
template <typename R, typename F>
__device__ __forceinline__ R lse2_group(F src, int M, R ctr, R q2, R shift, bool use_shift, int part, int P) {
  R acc = R(0);
  bool bad = true;
  if (use_shift) {
    acc = psum2<R>(src, M, ctr, q2, shift, part, P);
    for (int o = 1; o < P; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    bad = !(acc > R(1e-25) && acc < R(1e25));
  }
  if (__any_sync(0xffffffffu, bad)) {
    R mx = pmax2<R>(src, M, ctr, q2, part, P);
    for (int o = 1; o < P; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const bool fin = mx > -dd_inf<R>();
    R s2 = psum2<R>(src, M, ctr, q2, fin ? mx : R(0), part, P);
    for (int o = 1; o < P; o <<= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    if (bad) return fin ? mx + dd_lg2(s2) : mx;
  }
  return shift + dd_lg2(acc);
}

// Lanes per target for a pass with `nt` targets of `M` sources on `nthr` threads.
__device__ __forceinline__ int lanes_per_target(int nt, int M, int nthr) {
  int P = 1;
  while (P < 32 && nt * P * 2 <= nthr && P * 2 <= M) P *= 2;
  return P;
}

// Quotient u / w of non-negative integers by a multiplication with iw ~ 1/w.
__device__ __forceinline__ int quot(int u, int w, float iw) {
  int q = (int)((float)u * iw);
  const int r = u - q * w;
  q += r >= w ? 1 : 0;
  q -= r < 0 ? 1 : 0;
  return q;
}

// A rounded product that is not contracted into a later sum.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// Maximum that is NaN if either argument is.
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// ---- float passes: a tile of B consecutive targets of one line per thread.
// Chunks of kChunk sources whose terms all lie more than kCut (log2 units) below
// their targets' shifts are left out.  A sum made that way is accepted between
// kAccLo and 1e25, so what is left out of M sources is below M 2^-60 / 2^-12 = M 2^-48
// of it: it vanishes in the float sum.  (The floats are summed in one fixed order,
// eight partial sums by the source index modulo eight: where the background
// dominates, the Newton root amplifies a rounding of its argument by lam/eps, so
// a value must not depend on the tile it was computed in.)
constexpr float kCut = 60.0f, kAccLo = 2.44140625e-4f;
constexpr int kChunk = 8;

// acc[k] = sum_m 2^{src[m sm] - q2 (m - ctr0 - k)^2 - S[k]}, k < B.  The distances
// of a chunk are formed once for the whole tile (kChunk + B - 1 of them); a
// term is then an FFMA, a subtraction, an ex2 and an addition.
template <int B>
__device__ __forceinline__ void tile_sum(const float* src, int sm, int M, int ctr0, float q2, const float (&S)[B],
                                         bool cull, float (&acc)[B]) {
  float a[B][kChunk];
#pragma unroll
  for (int k = 0; k < B; ++k)
#pragma unroll
    for (int i = 0; i < kChunk; ++i) a[k][i] = 0.0f;
  int m0 = 0;
  for (; m0 + kChunk <= M; m0 += kChunk) {
    float s[kChunk];
#pragma unroll
    for (int i = 0; i < kChunk; ++i) s[i] = src[(m0 + i) * sm];
    if (cull) {
      float cm = s[0];
#pragma unroll
      for (int i = 1; i < kChunk; ++i) cm = max_nan(cm, s[i]);
      bool need = false;   // a NaN keeps the chunk
#pragma unroll
      for (int k = 0; k < B; ++k) {
        const int j = ctr0 + k;
        const float d = (float)(j - min(max(j, m0), m0 + kChunk - 1));
        need |= !(fmaf(-q2 * d, d, cm) - S[k] < -kCut);
      }
      if (!need) continue;
    }
    float d[kChunk + B - 1], t[kChunk + B - 1];
    const float d0 = (float)(m0 - ctr0 - (B - 1));
#pragma unroll
    for (int i = 0; i < kChunk + B - 1; ++i) {
      d[i] = d0 + (float)i;
      t[i] = q2 * d[i];
    }
#pragma unroll
    for (int i = 0; i < kChunk; ++i)
#pragma unroll
      for (int k = 0; k < B; ++k)
        a[k][i] += dd_ex2(fmaf(-t[i - k + B - 1], d[i - k + B - 1], s[i]) - S[k]);
  }
  for (; m0 < M; ++m0) {
    const float s = src[m0 * sm], d0 = (float)(m0 - ctr0);
#pragma unroll
    for (int k = 0; k < B; ++k) {
      const float d = d0 - (float)k;
      a[k][0] += dd_ex2(fmaf(-(q2 * d), d, s) - S[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < B; ++k)
    acc[k] = ((a[k][0] + a[k][1]) + (a[k][2] + a[k][3])) + ((a[k][4] + a[k][5]) + (a[k][6] + a[k][7]));
}

// out[k] = log2 sum_m 2^{src[m sm] - q2 (m - ctr0 - k)^2} for the first n targets
// of the tile.  With `have`, S holds a previous value of each target as its
// shift (one pass); a target whose sum leaves the accepted range is summed again
// in full, and against its exact maximum if that does not help; so are all
// targets without a previous value.
template <int B>
__device__ __forceinline__ void lse_tile(const float* src, int sm, int M, int ctr0, float q2, float (&S)[B],
                                         bool have, int n, float (&out)[B]) {
  const bool long_line = M > 4 * kChunk;   // shorter ones gain less than the test costs
  bool need[B];
#pragma unroll
  for (int k = 0; k < B; ++k) {
    need[k] = k < n;
    if (k >= n) S[k] = INFINITY;   // no term of a target beyond the line's end
  }
  for (int level = have ? (long_line ? 0 : 1) : 2;; ++level) {
    if (level == 2) {
      float mx[B];
#pragma unroll
      for (int k = 0; k < B; ++k) mx[k] = -INFINITY;
      for (int m = 0; m < M; ++m) {
        const float s = src[m * sm], d = (float)(m - ctr0);
#pragma unroll
        for (int k = 0; k < B; ++k) mx[k] = fmaxf(mx[k], fmaf(-(q2 * (d - (float)k)), d - (float)k, s));
      }
#pragma unroll
      for (int k = 0; k < B; ++k)
        if (need[k]) S[k] = mx[k] > -INFINITY ? mx[k] : 0.0f;
    }
    float acc[B];
    tile_sum<B>(src, sm, M, ctr0, q2, S, long_line && level != 1, acc);
    const float lo = level == 0 ? kAccLo : 1e-25f;
    bool bad = false;
#pragma unroll
    for (int k = 0; k < B; ++k) {
      if (!need[k]) continue;
      out[k] = S[k] + dd_lg2(acc[k]);
      need[k] = !(acc[k] > lo && acc[k] < 1e25f);
      bad |= need[k];
    }
    if (level == 2 || !bad) return;
  }
}

// One 1-D log-sum-exp pass: lines l < L, targets j < J (source m at distance
// m - j - off of target j), sources src[l sl + m sm], m < M.  `prev` holds the
// previous iteration's values at [l ol + j oj] (unless `first`).  put(l, j, n, v)
// receives n <= B consecutive values v[0..n).  Threads tid, tid + nthr, ... of
// the pass; consecutive threads take consecutive lines.
template <int B, typename Put>
__device__ __forceinline__ void pass_tiles(const float* src, int sl, int sm, const float* prev, int ol, int oj, int L,
                                           int J, int M, int off, float q2, bool first, int tid, int nthr, Put put) {
  const int nitem = L * ((J + B - 1) / B);
  const float iL = 1.0f / (float)L;
  for (int it = tid; it < nitem; it += nthr) {
    const int t = quot(it, L, iL), l = it - t * L, j0 = t * B, n = min(B, J - j0);
    float S[B], v[B];
#pragma unroll
    for (int k = 0; k < B; ++k) S[k] = first ? 0.0f : prev[l * ol + min(j0 + k, J - 1) * oj];
    lse_tile<B>(src + l * sl, sm, M, j0 + off, q2, S, !first, n, v);
    put(l, j0, n, v);
  }
}

// One target at a time on a group of P lanes (P a power of two), target j L + l.
template <typename R, typename Put>
__device__ __forceinline__ void pass_lanes(const R* src, int sl, int sm, const R* prev, int ol, int oj, int L, int J,
                                           int M, int off, R q2, bool first, int P, int tid, int nthr, Put put) {
  const int nt = L * J, ni = (nt * P + 31) & ~31, lp = 31 - __clz(P);
  const float iL = 1.0f / (float)L;
  for (int i = tid; i < ni; i += nthr) {
    const int tg0 = i >> lp, part = i & (P - 1), tg = min(tg0, nt - 1);
    const int j = quot(tg, L, iL), l = tg - j * L;
    const R* row = src + l * sl;
    R v[1];
    v[0] = lse2_group<R>([&](int m) { return row[m * sm]; }, M, R(j + off), q2, prev[l * ol + j * oj], !first, part, P);
    __syncwarp();
    if (part == 0 && tg0 < nt) put(l, j, 1, v);
  }
}

// Few targets: a group of lanes each.  Otherwise tiles of two targets when
// those occupy a quarter of the threads, else single targets: the larger tile
// spends fewer instructions per term (about 7.5 against 10), the smaller one
// keeps more warps busy on the small cells.  (Tiles of four spilled registers.)
// `linear`: target j L + l on thread (j L + l) mod nthr in any case (for sums
// over a thread's targets whose order must not depend on the tile).
template <typename Put>
__device__ __forceinline__ void run_pass(const float* src, int sl, int sm, const float* prev, int ol, int oj, int L,
                                         int J, int M, int off, float q2, bool first, int tid, int nthr, Put put,
                                         bool linear = false) {
  const int P = lanes_per_target(L * J, M, nthr);
  if (P > 1)
    pass_lanes<float>(src, sl, sm, prev, ol, oj, L, J, M, off, q2, first, P, tid, nthr, put);
  else if (!linear && 4 * L * ((J + 1) / 2) >= nthr)
    pass_tiles<2>(src, sl, sm, prev, ol, oj, L, J, M, off, q2, first, tid, nthr, put);
  else
    pass_tiles<1>(src, sl, sm, prev, ol, oj, L, J, M, off, q2, first, tid, nthr, put);
}

// ---- double passes: one target on a group of P lanes.  The FP64 pipe gives two
// lanes a clock, so a term (12 operations) is evaluated only if a float test
// finds it within 2^-65 of the target's shift (at eps = h^2: 13 of 32 sources);
// narrowing and widening run on the integer pipe.  The test allows for its own
// rounding: a term that counts is formed from magnitudes below |source| + |shift| + 65,
// so its float value errs by less than 4e-7 (|source| + |shift|) + 0.001.  A sum below 2^-4
// of its shift, and a target without a previous value, is taken against its
// maximum, so what is left out is below M 2^-61 of the sum.  The maximum is the float
// one (any value near it serves) unless it or a source is beyond 1e6, where a float
// one could be off by more than a unit (eps below about 1e-3 h^2).
__device__ __forceinline__ double lse_lanes_f64(const double* row, int sm, int M, int ctr, double q2, double shift,
                                                bool have, int part, int P) {
  const float q2f = (float)q2;
  double acc = 0.0;
  bool todo = true;
  for (int pass = have ? 0 : 1; pass < 2; ++pass) {
    if (pass == 1) {
      float mx = -INFINITY, big = 0.0f;
      for (int m = part; m < M; m += P) {
        const float d = (float)(m - ctr), v = narrow_any(row[m * sm]);
        mx = fmaxf(mx, fmaf(-q2f * d, d, v));
        big = fmaxf(big, fabsf(v));
      }
      for (int o = 1; o < P; o <<= 1) {
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
      }
      double mxd = (double)mx;
      if (__any_sync(0xffffffffu, big > 1e6f || (mx < -1e6f && mx > -INFINITY))) {
        mxd = -INFINITY;
        for (int m = part; m < M; m += P) {
          const double d = (double)(m - ctr);
          mxd = fmax(mxd, fma(-q2, d * d, row[m * sm]));
        }
        for (int o = 1; o < P; o <<= 1) mxd = fmax(mxd, __shfl_xor_sync(0xffffffffu, mxd, o));
      }
      if (todo) shift = mxd > -INFINITY ? mxd : 0.0;
    }
    const float sf = (float)shift, lo = fmaf(-4e-7f, fabsf(sf), -65.001f);
    double a = 0.0;
    for (int m = part; m < M; m += P) {
      const float d = (float)(m - ctr);
      const double v = row[m * sm];
      const float vf = narrow_any(v);
      if (!(fmaf(-q2f * d, d, vf) - sf < fmaf(-4e-7f, fabsf(vf), lo)))
        a += dd_ex2(fma(-q2, widen_pos(d * d), v) - shift);
    }
    for (int o = 1; o < P; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (todo) acc = a;
    if (pass == 0) {
      todo = !(acc > 0.0625 && acc < 1e25);
      if (!__any_sync(0xffffffffu, todo)) break;
    }
  }
  return shift + dd_lg2(acc);
}

template <typename Put>
__device__ __forceinline__ void run_pass(const double* src, int sl, int sm, const double* prev, int ol, int oj, int L,
                                         int J, int M, int off, double q2, bool first, int tid, int nthr, Put put,
                                         bool = false) {
  const int nt = L * J, P = lanes_per_target(nt, M, nthr), ni = (nt * P + 31) & ~31, lp = 31 - __clz(P);
  const float iL = 1.0f / (float)L;
  for (int i = tid; i < ni; i += nthr) {
    const int tg0 = i >> lp, part = i & (P - 1), tg = min(tg0, nt - 1);
    const int j = quot(tg, L, iL), l = tg - j * L;
    double v[1];
    v[0] = lse_lanes_f64(src + l * sl, sm, M, j + off, q2, prev[l * ol + j * oj], !first, part, P);
    __syncwarp();
    if (part == 0 && tg0 < nt) put(l, j, 1, v);
  }
}

// Roots u of g(u) = (1+s) u + c0 + softplus(lr - u) = 0, i.e. of
// log(rho + e^u) + s u + c0 = 0 with lr = log rho (Eq. proxdiv-problem with
// u = beta/eps + z).  g is convex and increasing (g' = 1 + s - sigmoid(lr - u) >= s).
// Both lines (1+s)u + c0 and s u + c0 + lr lie below g, so g >= 0 at
// min(u0, u1), their roots; Newton from there decreases monotonically to the root.
// The Newton iterate after w, and its step *du (the same operations wherever a
// target is advanced).
template <typename R>
__device__ __forceinline__ R newton_next(R lr, R c0, R w, R one_s, R* du = nullptr) {
  const R L2E = R(DD_LOG2E), LN2 = R(DD_LN2);
  R t = lr - w;
  R e = dd_ex2(-fabs(t) * L2E);
  R ie = dd_rcp(R(1) + e);
  R sp = max(t, R(0)) + dd_lg2(R(1) + e) * LN2;
  R sig = t >= R(0) ? ie : e * ie;
  R g = one_s * w + c0 + sp;
  R r = dd_rcp(one_s - sig);
  if (!du) return fma(-g, r, w);
  *du = mul_rn(g, r);
  return w - *du;
}
template <typename R> __device__ __forceinline__ R newton_tol() { return sizeof(R) == 4 ? R(2e-6) : R(1e-14); }

// A tile of B targets advances in lock-step (their dependency chains interleave;
// each stops on its own tolerance).  `uw` holds a previous root per target (or
// +inf: none): one Newton step from it lands right of the root (g is convex and
// increasing), and the start is the smaller of that point and the bound
// min(u0, u1), so the iteration still descends monotonically.
// At most `steps` steps are made; act[k] tells which targets are still short of
// the tolerance.  Where the background dominates, g' is close to s and the
// rounding of g moves u by more than the tolerance, so a few targets (2-5 %) run
// to the cap of 30 while the mean is 2.2: the caller finishes those from a list,
// packed into full warps, instead of holding every warp for them.
template <typename R, int B>
__device__ __forceinline__ void newton_tile(const R (&lr)[B], const R (&c0)[B], const R (&uw)[B], R s, int steps,
                                            R (&u)[B], bool (&act)[B]) {
  const R one_s = R(1) + s, tol = newton_tol<R>();
  bool any = false;
#pragma unroll
  for (int k = 0; k < B; ++k) {
    u[k] = -c0[k] / one_s;
    act[k] = lr[k] > -dd_inf<R>();   // rho = 0: closed form (Eq. sinkhorn-iters-ot)
    if (act[k] && s > R(0)) u[k] = min(u[k], -(lr[k] + c0[k]) / s);
    any |= act[k];
  }
  // probe step from the previous roots
#pragma unroll
  for (int k = 0; k < B; ++k) {
    R wn = newton_next(lr[k], c0[k], uw[k], one_s);
    if (act[k] && wn == wn && wn < u[k]) u[k] = wn;
  }
  for (int it = 0; it < steps && any; ++it) {
    any = false;
#pragma unroll
    for (int k = 0; k < B; ++k) {
      R du = R(0);
      const R un = newton_next(lr[k], c0[k], u[k], one_s, &du);
      if (act[k]) {
        u[k] = un;
        act[k] = !(fabs(du) <= tol * max(R(1), fabs(un)));
        any |= act[k];
      }
    }
  }
}

// At most `steps` further steps of one target.
template <typename R>
__device__ __forceinline__ R newton_rest(R lr, R c0, R u, R s, int steps) {
  const R one_s = R(1) + s, tol = newton_tol<R>();
  for (int it = 0; it < steps; ++it) {
    R du;
    u = newton_next(lr, c0, u, one_s, &du);
    if (fabs(du) <= tol * max(R(1), fabs(u))) break;
  }
  return u;
}

// The root in double.  A float solve gives the start (or the previous root, if it
// lies within 0.05 of it); double steps with the second-order correction
// du (1 + du g''/(2 g')) follow, whose error is below |du|^3 / 2, so a step of at
// most 1e-5 is the last: two steps as a rule (six to eight first-order ones
// before).  About 40 FP64 operations a step: table-driven 2^x and logarithm, the
// reciprocal from the float one, one division-free slope.
__device__ __forceinline__ double newton_f64(double lr, double c0, double uw, double s, double is, double i1s,
                                             int maxit) {
  double u = -c0 * i1s;
  if (!(lr > -dd_inf<double>())) return u;   // rho = 0: closed form (Eq. sinkhorn-iters-ot)
  if (s > 0.0) u = fmin(u, -(lr + c0) * is);
  const double bound = u;                    // right of the root
  const float lrf = (float)lr, c0f = (float)c0, sf = (float)s;
  float uf = (float)u;
  {
    const float w = (float)uw;
    float du;
    const float wn = newton_next(lrf, c0f, w, 1.0f + sf, &du);
    if (wn == wn && wn < uf) uf = wn;
    for (int it = 0; it < 8; ++it) {
      uf = newton_next(lrf, c0f, uf, 1.0f + sf, &du);
      if (fabsf(du) <= 1e-3f * fmaxf(1.0f, fabsf(uf))) break;
    }
    if (fabsf(uf) < 1e6f) u = fmin(u, (double)uf);
    if (fabsf(w - uf) < 0.05f) u = fmin(bound, uw);
  }
  const double one_s = 1.0 + s;
  for (int it = 0; it < maxit; ++it) {
    const double t = lr - u;
    const double e = dd_ex2(-fabs(t) * DD_LOG2E), op = 1.0 + e;
    const double g = fma(one_s, u, c0) + (fmax(t, 0.0) + dd_lg2(op) * DD_LN2);
    const double den = fma(s, op, t >= 0.0 ? e : 1.0);
    const double du0 = g * op * dd_rcp(den);
    // g''/(2 g') in float: it only corrects a small step
    const float h = 0.5f * narrow(e) * dd_rcp(narrow(op) * narrow(den));
    const float d0 = narrow(du0);
    double du = du0;
    if (fabsf(d0) < 0.1f) du = fma(du0, (double)(h * d0), du0);
    u = fmin(u - du, bound);
    if (fabsf(d0) <= 1e-5f) break;
  }
  return u;
}

constexpr int kLock = 4;     // Newton steps made in lock-step by every warp (float cells)
constexpr int kPend = 512;   // targets listed for the remaining steps (more are finished in place)

// mu phi((p0 + d)/mu) - mu phi(p0/mu) with phi(s) = s log s - s + 1, written as
//   d (log(p0/mu) - 1) + (p0 + d) log1p(d/p0),
// an identity whose float evaluation errs by ~1e-7 |d| (both logarithms enter
// multiplied by the change), unlike the difference of the two terms (~1e-7 p0).
// log_mu: natural log of mu.  The result is returned in double for summation.
__device__ __forceinline__ double kl_change_f(double p0, double d, float log_mu) {
  const double p1 = p0 + d;
  if (p0 <= 0.0) {   // mu phi(0) = mu
    if (p1 <= 0.0) return 0.0;
    const float p1f = (float)p1;
    return (double)(p1f * (dd_lg2(p1f) * (float)DD_LN2 - log_mu - 1.0f));
  }
  const float p0f = (float)p0, df = (float)d;
  const float l0 = dd_lg2(p0f) * (float)DD_LN2 - log_mu;
  const float l1p = log1pf(df / p0f);
  if (p1 <= 0.0) return (double)(df * (l0 - 1.0f));   // limit p1 log(p1/p0) -> 0
  return (double)(df * (l0 - 1.0f)) + p1 * (double)l1p;
}

// v[k] for a run-time k in 0..3 without indexing a local array (keeps it in registers).
__device__ __forceinline__ double pick4(const double (&v)[4], int k) {
  return k == 0 ? v[0] : (k == 1 ? v[1] : (k == 2 ? v[2] : v[3]));
}

__device__ __forceinline__ double box_value(const BoxRec& b, const double* arena, int y1, int y2) {
  int a = y1 - b.k0, c = y2 - b.l0;
  if (a < 0 || c < 0 || a >= b.H || c >= b.W) return 0.0;
  return arena[b.off + (long long)a * b.W + c];
}

}  // namespace

// Block sums of a cell (in double; the orders of the double cells' sums are those of block_sum).
template <typename R, int K>
__device__ __forceinline__ void cell_sum(double (&v)[K], double* scratch) {
  if constexpr (sizeof(R) == 4) block_sum_split<K>(v, scratch);
  else block_sum<K>(v, scratch);
}

// Scalars of one cell in the working precision.  One thread computes them from
// the doubles and the CTA reads them from shared memory: the same dozen
// double operations on every thread took 20 k clocks a cell (the FP64 pipe
// gives two lanes a clock), a tenth of a small cell's solve.
template <typename R>
struct CellScalars {
  double A, qD2;   // alpha/eps = A + a + 2 q D.xi; beta/eps = q|D|^2 - A + b - 2 q D.eta
  double bound;    // err |mu_J|
  R q2, qR, sR, rR, sB, cEta1, cEta2, cA, gA, cD1, cD2, tol, is, i1s;
  __device__ __forceinline__ void set_A(const DevState& S, double a) {
    A = a;
    sB = R(S.sl * (qD2 - A));   // s B
    cA = R(-(1.0 - S.rr) * A);
    gA = R(-S.sl * A);          // -s A: the A part of -alpha/lam
  }
  // translation step: alpha += t*, e^{t*/lam} = (a + sqrt(a^2 + 4 A_s B_s)) / (2 B_s) with A_s =
  // <e^{-alpha/lam}, mu_J>, B_s = <e^{-beta/lam}, nu>, a = |nu_{-J}|; it moves A by t*/eps
  __device__ __forceinline__ void translate(const DevState& S, double a0, double a, double As, double Bs) {
    const double uu = (a + sqrt(a * a + 4.0 * As * Bs)) / (2.0 * Bs);
    if (uu > 0.0 && uu < INFINITY) set_A(S, a0 + log(uu) / S.sl);
  }
  __device__ __forceinline__ void set(const DevState& S, int D1, int D2, double a, double muJ) {
    qD2 = S.q * (double)(D1 * D1 + D2 * D2);
    q2 = R(S.q * DD_LOG2E); qR = R(S.q); sR = R(S.sl); rR = R(S.rr);
    cEta1 = R(S.sl * 2.0 * S.q * D1); cEta2 = R(S.sl * 2.0 * S.q * D2);
    cD1 = R(2.0 * (1.0 - S.rr) * S.q * D1); cD2 = R(2.0 * (1.0 - S.rr) * S.q * D2);
    // gap <= err |mu_J| in the working precision: the largest value not above the bound
    is = R(1) / sR;
    i1s = R(1) / (R(1) + sR);
    bound = S.err * muJ;
    if constexpr (sizeof(R) == 4) tol = __double2float_rd(bound);
    else tol = bound;
    set_A(S, a);
  }
};

// What a CTA shares of the cell it works on, one object for both ways of solving it (a
// cell's barriers end before the next one's begin): static shared memory is taken from
// the Y-box capacity.
template <typename R>
struct CellShared {
  CellScalars<R> sk;
  BoxRec box[4];
  int geo[8];
  int npend;
  bool stop;
};

// One composite cell on one CTA: cell `cd` at position `cidx` of a sub-batch
// of `nbatch` cells.
// BAL: with the balancing step (an instance of its own: its registers cost the plain
// solve spills).
template <typename R, bool BAL>
__device__ __forceinline__ void cell_solve_body(const DevState& S, const CellDesc cd, int cidx, int nbatch,
                                                CellShared<R>& sh, unsigned char* smem_raw) {
  namespace cg = cooperative_groups;
  double* red = reinterpret_cast<double*>(smem_raw);  // 32 * 16 doubles (block reductions)
  BoxRec* sbox = sh.box;
  int* sgeo = sh.geo;
  CellScalars<R>& sk = sh.sk;
  int& npend = sh.npend;
  CellOut* out = S.cout + cidx;
  const unsigned long long t_start = dd_global_ns();
  const double* __restrict__ arena = S.arena[*S.cur];
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int N = S.N, s = S.s;
  const int nx1 = cd.nx1, nx2 = cd.nx2, nx = nx1 * nx2;
  auto csync = [&]() { __syncthreads(); };

  // ---------------------------------------------------------------- B_J
  if (tid == 0) {
    int k0 = 1 << 30, l0 = 1 << 30, k1 = -1, l1 = -1, slot = -1;
    for (int q = 0; q < 4; ++q) {
      BoxRec b = {0, 0, 0, 0, 0};
      if (cd.mem[q] >= 0) b = S.box[cd.mem[q]];
      sbox[q] = b;
      if (cd.mem[q] < 0 || b.H * b.W == 0) continue;
      k0 = min(k0, b.k0); l0 = min(l0, b.l0);
      k1 = max(k1, b.k0 + b.H); l1 = max(l1, b.l0 + b.W);
    }
    int st = CELL_OK;
    if (k1 < 0) {
      st = CELL_EMPTY;
      k0 = l0 = k1 = l1 = 0;
    } else {
      k0 = max(0, k0 - S.margin); l0 = max(0, l0 - S.margin);
      k1 = min(N, k1 + S.margin); l1 = min(N, l1 + S.margin);
      int H = k1 - k0, W = l1 - l0;
      // boxes beyond the shared-memory capacity run from a global spill slot
      if (H * W > S.cap_ny || H > S.cap_side || W > S.cap_side) {
        int sl = S.spill_slots > 0 ? (int)atomicAdd(S.spill_count, 1u) : S.spill_slots;
        if (sl >= S.spill_slots) st = CELL_TOOBIG;
        else slot = sl;
      }
    }
    sgeo[0] = k0; sgeo[1] = l0; sgeo[2] = k1 - k0; sgeo[3] = l1 - l0;
    sgeo[4] = st; sgeo[7] = slot;
  }
  csync();
  const int k0 = sgeo[0], l0 = sgeo[1], H = sgeo[2], W = sgeo[3];
  if (sgeo[4] != CELL_OK) {
    if (tid == 0) {
      CellOut o;
      o.k0 = k0; o.l0 = l0; o.H = H; o.W = W; o.iters = 0; o.status = sgeo[4];
      o.D1 = o.D2 = 0; o.gap = 0.0; o.dKX[0] = o.dKX[1] = 0.0; o.slot = -1; o.usec = 0;
      for (int q = 0; q < 4; ++q) {
        int bi = cd.mem[q];
        o.Ct[q] = bi >= 0 ? S.Cc[bi] : 0.0;
        o.Ht[q] = bi >= 0 ? S.Hh[bi] : 0.0;
        o.mass[q] = 0.0;
      }
      *out = o;
      atomicOr(S.status, sgeo[4] == CELL_EMPTY ? ST_EMPTY : ST_TOOBIG);
    }
    return;
  }
  const int ny = H * W;

  // ------------------------------------------------------- shared layout
  // X-side arrays always live in shared memory; the Y-side arrays too unless
  // the box exceeds the shared capacity, then in the cell's spill slot
  // (global memory, L2-resident) sized for an N x N box.
  // Rows of X, of T and U and of the Y-side arrays have odd pitches where those
  // fit (xp, Wp, Up), so that both a line of consecutive elements and a column
  // of consecutive lines are read without bank conflicts.
  const int cap_nx = 4 * s * s, cap_xp = cap_nx + 2 * s, xp = nx2 | 1;
  const int slot = sgeo[7];
  const bool spilled = slot >= 0;
  const int tsz = spilled ? 2 * s * N : 2 * s * S.cap_side;
  const int cap_ny = spilled ? N * N : S.cap_ny;
  const int Wo = W | 1, Uo = nx2 | 1;
  // A spilled box keeps T, U and beta + log nu, which the passes read many times,
  // in shared memory if those fit; the arrays that each y touches once an
  // iteration stay in the slot (143 x 81 at s = 8: 2.15 -> 1.94 ms a solve).
  const int rsz = 4 * s * S.cap_side + 5 * S.cap_ny;
  const bool hyb = spilled && nx1 * Wo + H * Uo + H * Wo <= rsz && 3 * nx1 * W <= rsz && H * Wo <= N * N;
  const int Wp = hyb || (!spilled && nx1 * Wo <= tsz && H * Wo <= cap_ny && 3 * nx1 * Wo <= rsz) ? Wo : W;
  const int Up = hyb || (!spilled && H * Uo <= tsz) ? Uo : nx2;
  R* xa = reinterpret_cast<R*>(smem_raw + 32 * 16 * sizeof(double));
  R* av = xa + cap_xp;
  R* g0 = av + cap_nx;
  R* Wv = g0 + cap_nx;
  R* lm = Wv + cap_nx;
  R* xa_nx = lm + cap_nx;    // next iterate of xa / a (double buffer of the X-update)
  R* av_nx = xa_nx + cap_xp;
  R* gslot = spilled ? reinterpret_cast<R*>(S.spill + (long long)slot * S.spill_stride) : nullptr;
  R* T = spilled && !hyb ? gslot : av_nx + cap_nx;
  R* U = T + (hyb ? nx1 * Wp : tsz);
  R* bl = U + (hyb ? H * Up : tsz);
  R* lrho = hyb ? gslot : bl + cap_ny;
  R* Zv = lrho + cap_ny;
  R* bv = Zv + cap_ny;
  R* lnu = bv + cap_ny;

  // ------------------------------------------------------- load Y side (a1)
  // rho = max(0, P_Y - nu_J)/nu and log nu on B_J; the same pass accumulates
  // the barycentre of nu_J, whose nearest pixel is the Y frame origin (so
  // that 2 q D.xi carries the cell's mean displacement).
  const float iW = 1.0f / (float)W, inx2 = 1.0f / (float)nx2;
  double a_tot = 0.0;   // |nu_{-J}| on B_J (translation step)
  {
    double m3[4] = {0.0, 0.0, 0.0, 0.0};
    for (int u = tid; u < ny; u += nthr) {
      const int kk = quot(u, W, iW), ll = u - kk * W, v = kk * Wp + ll;
      int y1 = k0 + kk, y2 = l0 + ll, y = y1 * N + y2;
      double nuJ = 0.0;
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) nuJ += box_value(sbox[q4], arena, y1, y2);
      double nuy = S.nu[y];
      const double num = fmax(0.0, S.PY[y] - nuJ);
      R rho = R(num) / R(nuy);
      lrho[v] = rho > R(0) ? dd_lg2(rho) * R(DD_LN2) : -dd_inf<R>();
      lnu[v] = R(S.lognu[y]);
      m3[0] += nuJ; m3[1] += nuJ * kk; m3[2] += nuJ * ll;
      if (S.ti) m3[3] += num;
    }
    cell_sum<R, 4>(m3, red);
    a_tot = m3[3];
    if (tid == 0) {
      int c1 = H / 2, c2 = W / 2;
      if (m3[0] > 0.0) {
        c1 = min(H - 1, max(0, (int)lrint(m3[1] / m3[0])));
        c2 = min(W - 1, max(0, (int)lrint(m3[2] / m3[0])));
      }
      sgeo[5] = c1; sgeo[6] = c2;
    }
    __syncthreads();
  }
  const int xc1 = cd.i0 + nx1 / 2, xc2 = cd.j0 + nx2 / 2;
  const int yc1 = k0 + sgeo[5], yc2 = l0 + sgeo[6];
  const int D1 = xc1 - yc1, D2 = xc2 - yc2;
  const int offr = (k0 - cd.i0) + D1, offc = (l0 - cd.j0) + D2;
  const double eps = S.eps, q = S.q, sl = S.sl;   // q = h^2/eps, s = eps/lam

  // ------------------------------------------------------- load X side
  const double inv_eps = S.inv_eps;
  double acc2[2] = {0.0, 0.0};
  for (int t = tid; t < nx; t += nthr) {
    const int r = quot(t, nx2, inx2), c = t - r * nx2;
    int x = (cd.i0 + r) * N + cd.j0 + c;
    int xi1 = cd.i0 + r - xc1, xi2 = cd.j0 + c - xc2;
    acc2[0] += S.alpha[x] * inv_eps - 2.0 * q * (double)(D1 * xi1 + D2 * xi2);
    acc2[1] += S.mu[x];
  }
  block_sum<2>(acc2, red);
  if (tid == 0) sk.set(S, D1, D2, acc2[0] / nx, acc2[1]);
  __syncthreads();
  double A = sk.A;
  const R q2 = sk.q2, qR = sk.qR, sR = sk.sR, rR = sk.rR, cEta1 = sk.cEta1, cEta2 = sk.cEta2, cD1 = sk.cD1,
          cD2 = sk.cD2, tol = sk.tol;
  R sB = sk.sB, cA = sk.cA, gA = sk.gA;
  for (int t = tid; t < nx; t += nthr) {
    const int r = quot(t, nx2, inx2), c = t - r * nx2;
    int x = (cd.i0 + r) * N + cd.j0 + c;
    int xi1 = cd.i0 + r - xc1, xi2 = cd.j0 + c - xc2;
    double lin = 2.0 * q * (double)(D1 * xi1 + D2 * xi2);
    R a = R(S.alpha[x] * inv_eps - lin - A);
    R l = R(S.logmu[x]);
    av[t] = a;
    lm[t] = l;
    g0[t] = R(-sl * lin);
    xa[r * xp + c] = (a + l) * R(DD_LOG2E);
  }
  csync();

  // ------------------------------------------------------- Sinkhorn loop
  // Barriers per iteration: after each of the five passes.  The X-update is
  // computed speculatively inside the last pass into the second buffer, and
  // the gap is reduced from per-warp partials after that pass's barrier.
  const R LN2 = R(DD_LN2), L2E = R(DD_LOG2E);
  const bool stops = S.err >= 0.0;
  const R is = sk.is, i1s = sk.i1s;   // 1/s, 1/(1 + s) (double cells)
  (void)is;
  (void)i1s;
  R* gpart = reinterpret_cast<R*>(red) + 32 * 12;   // per-warp gap partials
  R* apart = gpart + 32;                             // per-warp <e^{-alpha/lam}, mu> (translation step)
  R* bpart = gpart + 64;                             // per-warp <e^{-beta/lam}, nu>
  int* pend = reinterpret_cast<int*>(red + 256);    // kPend list entries (the last 2 KB of red)
  const bool ti = S.ti && sl > 0.0;
  const int lane = tid & 31, wid = tid >> 5, nwarp = nthr >> 5;
  int it = 0;
  R gap = R(0);
  bool first = true;
  // translation step: nu e^{-beta/lam} per y, in the cell's buffer of new marginals (written by the epilogue only)
  R* tib;
  {
    CellOut tmp;
    tmp.slot = slot;
    int st;
    tib = reinterpret_cast<R*>(cell_nut(S, tmp, cidx, &st));
  }
  R *xa_c = xa, *av_c = av;          // current iterate
  R *xa_n = xa_nx, *av_n = av_nx;    // next iterate
  for (;;) {
    ++it;
    if (tid == 0) npend = 0;
    // Y-half, pass over columns of X: T(r, ll) = log2 sum_c 2^{xa(r,c) - q2 (c - ll - offc)^2}
    run_pass(xa_c, xp, 1, T, Wp, 1, nx1, W, nx2, offc, q2, first, tid, nthr, [&](int r, int ll, int n, const auto& v) {
      for (int k = 0; k < n; ++k) T[r * Wp + ll + k] = v[k];
    });
    csync();
    // Y-half, pass over rows of X: Z(kk, ll), then the Newton roots of the tile (a3)
    R bsum = R(0);
    const bool fused_y = sizeof(R) == 4 && ny * 2 > nthr;
    // root u of one y: Z, beta and beta + log nu (Zx: Z in natural units, or, for
    // the small boxes that are not fused, in log2 units)
    auto y_store = [&](int v, int y, R u, R Zx, R Zn, R c0) {
      const R b = fused_y ? u - Zx : fma(-Zx, LN2, u);
      Zv[v] = fused_y ? mul_rn(Zx, L2E) : Zx;
      bv[v] = b;
      bl[v] = (b + lnu[v]) * L2E;
      // nu e^{-beta/lam}: -s beta/eps = -(s root + c0)
      if (ti) tib[y] = dd_ex2((lnu[v] - sR * u - c0) * L2E);
    };
    auto y_root = [&](int ll, int kk, int n, const auto& Z2) {
      constexpr int B = sizeof(Z2) / sizeof(R);
      R lr[B], c0[B], uw[B], root[B], Zn[B];
      const R eta2 = R(l0 + ll - yc2);
#pragma unroll
      for (int k = 0; k < B; ++k) {
        const int v = (kk + min(k, n - 1)) * Wp + ll;
        Zn[k] = mul_rn(k < n ? Z2[k] : Z2[0], LN2);
        const R eta1 = R(k0 + kk + min(k, n - 1) - yc1);
        c0[k] = sB - cEta1 * eta1 - cEta2 * eta2 - sR * Zn[k];
        lr[k] = lrho[v];
        uw[k] = first ? dd_inf<R>() : bv[v] + Zn[k];
      }
      [[maybe_unused]] bool open[B];
      if constexpr (sizeof(R) == 8) {
        root[0] = newton_f64(lr[0], c0[0], uw[0], sR, is, i1s, S.newton_maxit);
      } else {
        newton_tile<R, B>(lr, c0, uw, sR, min(S.newton_maxit, kLock), root, open);
      }
#pragma unroll
      for (int k = 0; k < B; ++k) {
        if (k >= n) break;
        if constexpr (sizeof(R) == 4) {
          if (kLock < S.newton_maxit && open[k]) {
            const int v = (kk + k) * Wp + ll, e = atomicAdd(&npend, 1);
            if (e < kPend) {   // finished below from the list
              pend[e] = v;
              bv[v] = root[k];
              Zv[v] = fused_y ? Zn[k] : Z2[k];
              continue;
            }
            root[k] = newton_rest(lr[k], c0[k], root[k], sR, S.newton_maxit - kLock);
          }
        }
        y_store((kk + k) * Wp + ll, (kk + k) * W + ll, root[k], fused_y ? Zn[k] : Z2[k], Zn[k], c0[k]);
      }
    };
    if constexpr (sizeof(R) == 4) {
      run_pass(T, 1, Wp, Zv, 1, Wp, W, H, nx1, offr, q2, first, tid, nthr, y_root);
      __syncthreads();
      const int np = min(npend, kPend);
      const float iWp = 1.0f / (float)Wp;
      for (int e = tid; e < np; e += nthr) {
        const int v = pend[e], kk = quot(v, Wp, iWp), ll = v - kk * Wp;
        const R Zx = Zv[v], Zn = fused_y ? Zx : mul_rn(Zx, LN2);
        const R eta1 = R(k0 + kk - yc1), eta2 = R(l0 + ll - yc2);
        const R c0 = sB - cEta1 * eta1 - cEta2 * eta2 - sR * Zn;
        y_store(v, kk * W + ll, newton_rest(lrho[v], c0, bv[v], sR, S.newton_maxit - kLock), Zx, Zn, c0);
      }
    } else {
      run_pass(T, 1, Wp, Zv, 1, Wp, W, H, nx1, offr, q2, first, tid, nthr,
               [&](int ll, int kk, int, const auto& v) { Zv[kk * Wp + ll] = v[0]; });
      csync();
      for (int u = tid; u < ny; u += nthr) {
        const int kk = quot(u, W, iW), ll = u - kk * W;
        const R z[1] = {Zv[kk * Wp + ll]};
        y_root(ll, kk, 1, z);
      }
    }
    if (ti) {
      csync();
      for (int u = tid; u < ny; u += nthr) bsum += tib[u];
    }
    if (ti) {
      bsum = warp_sum(bsum);
      if (lane == 0) bpart[wid] = bsum;
    }
    csync();
    // X-half, pass over columns of B_J: U(kk, c) = log2 sum_ll 2^{bl(kk,ll) - q2 (ll - (c - offc))^2}
    run_pass(bl, Wp, 1, U, Up, 1, H, nx2, W, -offc, q2, first, tid, nthr, [&](int kk, int c, int n, const auto& v) {
      for (int k = 0; k < n; ++k) U[kk * Up + c + k] = v[k];
    });
    csync();
    // X-half, pass over rows of B_J: W, the gap terms (a4) and the next a (a2)
    {
      R gl = R(0), asum = R(0);
      run_pass(U, 1, Up, Wv, 1, nx2, nx2, nx1, H, -offr, q2, first, tid, nthr,
               [&](int c, int r0, int n, const auto& v) {
        for (int k = 0; k < n; ++k) {
          const int r = r0 + k, t = r * nx2 + c;
          const R W2 = v[k];
          Wv[t] = W2;
          R a = av_c[t];
          R tt = a + W2 * LN2;         // log(P_X pi / mu)
          R g = gA + g0[t] - sR * a;   // -alpha/lam
          gl += dd_ex2((lm[t] + g) * L2E) * dd_psi<R>(tt - g);
          R xi1 = R(cd.i0 + r - xc1), xi2 = R(cd.j0 + c - xc2);
          R an = cA - rR * W2 * LN2 - cD1 * xi1 - cD2 * xi2;
          av_n[t] = an;
          xa_n[r * xp + c] = (an + lm[t]) * L2E;
          if (ti) asum += dd_ex2((lm[t] + gA + g0[t] - sR * an) * L2E);   // mu e^{-alpha_new/lam}
        }
      }, ti);
      gl = warp_sum(gl);
      if (lane == 0) gpart[wid] = gl;
      if (ti) {
        asum = warp_sum(asum);
        if (lane == 0) apart[wid] = asum;
      }
    }
    csync();
    {
      R gs = R(0);
      for (int w = 0; w < nwarp; ++w) gs += gpart[w];
      gap = gs;
    }
    first = false;
    if ((stops && gap <= tol) || it >= S.maxit || !(gap == gap)) break;
    if (ti) {
      // translation step: alpha += t*, e^{t*/lam} = (a + sqrt(a^2 + 4 A_s B_s)) / (2 B_s); in the
      // cell frame alpha/eps = A + a(xi) + 2qD.xi it moves A by t*/eps = log(u)/s.  One thread
      // computes it: the double root and logarithm on every thread kept the narrow FP64 pipe busy
      // for most of the iteration.
      if (tid == 0) {
        double As = 0.0, Bs = 0.0;
        for (int w = 0; w < nwarp; ++w) {
          As += (double)apart[w];
          Bs += (double)bpart[w];
        }
        sk.translate(S, A, a_tot, As, Bs);
      }
      __syncthreads();
      A = sk.A; sB = sk.sB; cA = sk.cA; gA = sk.gA;
    }
    // accept the X-update: swap the buffers
    R* tp = av_c; av_c = av_n; av_n = tp;
    tp = xa_c; xa_c = xa_n; xa_n = tp;
  }
  const bool nonfinite = !(gap == gap);

  // ------------------------------------------------------- epilogue (a5)
  // alpha, P_X of the new plan and the KL_X change: first CTA only.  With
  // balancing (one CTA per cell) P_X and the KL_X change follow the balancing.
  constexpr bool bal = BAL;
  const double th_s = 1.0 / nbatch;
  double dk[2] = {0.0, 0.0};
  double mubar[4] = {0.0, 0.0, 0.0, 0.0};   // balancing: mu_bar(X_q), X-marginal after one more X-half
  {
    for (int t = tid; t < nx; t += nthr) {
      const int r = quot(t, nx2, inx2), c = t - r * nx2;
      int x = (cd.i0 + r) * N + cd.j0 + c;
      int xi1 = cd.i0 + r - xc1, xi2 = cd.j0 + c - xc2;
      double a = (double)av_c[t];
      S.alphanew[x] = eps * (A + a + 2.0 * q * (double)(D1 * xi1 + D2 * xi2));
      if (bal) {
        // av_n holds the X-half of the final beta (computed before the loop stopped)
        const int qd = 2 * (r >= s) + (c >= s);
        const double mb = exp(((double)lm[t] + (double)gA + (double)g0[t] - sl * (double)av_n[t]));
#pragma unroll
        for (int k = 0; k < 4; ++k) mubar[k] += k == qd ? mb : 0.0;   // static indices (no local memory)
        continue;
      }
      double p1 = (double)dd_ex2((lm[t] + av_c[t]) * L2E + Wv[t]);
      S.PXnew[x] = p1;
      double p0 = S.PX[x];
      if (sizeof(R) == 8) {
        double m = S.mu[x];
        double ps = (1.0 - th_s) * p0 + th_s * p1;
        double k0v = dd_kl_term(p0, m);
        dk[0] += dd_kl_term(p1, m) - k0v;
        dk[1] += dd_kl_term(ps, m) - k0v;
      } else {
        // float cell solve: the KL_X changes from the cancellation-free form
        // (the error scales with the change p1 - p0, not with p)
        dk[0] += kl_change_f(p0, p1 - p0, lm[t]);
        dk[1] += kl_change_f(p0, th_s * (p1 - p0), lm[t]);
      }
    }
    if (bal) block_sum<4>(mubar, red);
    else cell_sum<R, 2>(dk, red);
  }

  R hs[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) hs[k] = R(0);
  const int nhr = nx1 > s ? 2 : 1, nhc = nx2 > s ? 2 : 1;
  int nst;
  double* nut;
  {
    CellOut tmp;
    tmp.slot = slot;
    nut = cell_nut(S, tmp, cidx, &nst);
  }
  R* Te = T;                 // epilogue scratch spans T, U, bl, lrho (and Zv for the widest boxes)
  R* Ma = T + nx1 * W;
  R* Md = Ma + nx1 * W;
  // Zv (the final Z) serves as the shift of the quadrant sums unless Md reaches it
  const bool zok = hyb || Md + nx1 * W <= Zv;
  for (int hc = 0; hc < nhc; ++hc) {
    const int cb = hc * s, ce = min(nx2, cb + s);
    // rows of X_J against columns of B_J, restricted to the column half hc
    for (int t = tid; t < nx1 * W; t += nthr) {
      const int r = quot(t, W, iW), ll = t - r * W;
      const R* row = xa_c + r * xp;
      R ma, md;
      const R T2 = lse_moments<R>([&](int m) { return row[m]; }, [&](int m) { return av_c[r * nx2 + m]; },
                                  [&](int) { return R(0); }, qR, R(D2), cb, ce, R(ll + offc), q2, R(0), false, ma,
                                  md);
      Te[t] = T2;
      Ma[t] = ma;
      Md[t] = md;
    }
    csync();
    for (int u = tid; u < ny; u += nthr) {
      const int kk = quot(u, W, iW), ll = u - kk * W, v = kk * Wp + ll;
      int y = (k0 + kk) * N + l0 + ll;
      R ctr = R(kk + offr);
      double nuy = S.nu[y];
      // Z of the last iteration: the log-sum-exp over all rows of the full-row
      // T, an upper bound of every quadrant's sum at this y
      const R zsh = zok ? Zv[v] : R(0);
      for (int hr = 0; hr < nhr; ++hr) {
        const int rb = hr * s, re = min(nx1, rb + s);
        R ma, md;
        const R P2 = lse_moments<R>(
            [&](int m) { return Te[m * W + ll]; }, [&](int m) { return Ma[m * W + ll]; },
            [&](int m) { return Md[m * W + ll]; }, qR, R(D1), rb, re, ctr, q2, zsh, zok, ma, md);
        const int qd = 2 * hr + hc;
        R nt = R(nuy) * dd_ex2(bv[v] * L2E + P2);
        nut[qd * nst + u] = (double)nt;
        hs[qd] += nt * (ma + bv[v]);
        hs[4 + qd] += nt * md;
        hs[8 + qd] += nt;
      }
    }
    __threadfence();
    csync();
  }
  if constexpr (bal) {
    // ---- balancing (Section 5.3, Eq. balancing): targets m_q = mu_bar(X_q) |nu_J| / mu_bar(X_J);
    // donors scale their rows by m_q/|nu_q|, receivers by 1 + D(y) w_q / nu_q(y) with the donated
    // field D(y) = sum_d (|nu_d| - m_d) nu_d(y)/|nu_d| and w_q = deficit_q / total excess.
    double ms[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) ms[k] = (double)hs[8 + k];
    block_sum<4>(ms, red);
    double mJ = 0.0, mbJ = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) { mJ += ms[k]; mbJ += mubar[k]; }
    double fd[4], rd[4], wr[4];   // donor factor, donor weight in D, receiver share
    double Ex = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double mk = mbJ > 0.0 ? mubar[k] * mJ / mbJ : 0.0;
      const double e = ms[k] - mk;
      fd[k] = 1.0; rd[k] = 0.0; wr[k] = 0.0;
      if (e > 0.0 && ms[k] > 0.0) { fd[k] = mk / ms[k]; rd[k] = e / ms[k]; Ex += e; }
      else if (e < 0.0) wr[k] = -e;
    }
    const bool move = Ex > 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) wr[k] = move ? wr[k] / Ex : 0.0;
    // rho_q(u) from the unbalanced marginals in nut
    auto rho_at = [&](int u, double (&rho)[4]) {
      double nv[4], D = 0.0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int hr = k >> 1, hc = k & 1;
        nv[k] = (hr < nhr && hc < nhc) ? nut[k * nst + u] : 0.0;
        D += rd[k] * nv[k];
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        rho[k] = fd[k];
        if (wr[k] > 0.0 && nv[k] > 0.0) rho[k] = 1.0 + D * wr[k] / nv[k];
      }
    };
    // pass B: C and H of the balanced plan from the same per-y sums, weighted by rho
    if (move) {
#pragma unroll
      for (int k = 0; k < 12; ++k) hs[k] = R(0);
      for (int hc = 0; hc < nhc; ++hc) {
        const int cb = hc * s, ce = min(nx2, cb + s);
        for (int t = tid; t < nx1 * W; t += nthr) {
          int r = t / W, ll = t - r * W;
          const R* row = xa_c + r * xp;
          R ctr = R(ll + offc);
          R T2 = lse2_1d<R>([&](int m) { return row[cb + m]; }, ce - cb, ctr - R(cb), q2, R(0), false);
          R sw = 0, sa = 0, sd = 0;
          for (int c = cb; c < ce; ++c) {
            R d = R(c) - ctr;
            R w = dd_ex2(row[c] - q2 * d * d - T2);
            sw += w;
            sa += w * (av_c[r * nx2 + c] - qR * d * d);
            R dt = d + R(D2);
            sd += w * dt * dt;
          }
          R isw = R(1) / sw;
          Te[t] = T2;
          Ma[t] = sa * isw;
          Md[t] = sd * isw;
        }
        __syncthreads();
        for (int u = tid; u < ny; u += nthr) {
          int kk = u / W, ll = u - kk * W;
          R ctr = R(kk + offr);
          double rho[4];
          rho_at(u, rho);
          for (int hr = 0; hr < nhr; ++hr) {
            const int rb = hr * s, re = min(nx1, rb + s);
            R P2 = lse2_1d<R>([&](int m) { return Te[(rb + m) * W + ll]; }, re - rb, ctr - R(rb), q2, R(0), false);
            R sw = 0, sa = 0, sd = 0;
            for (int r = rb; r < re; ++r) {
              R d = R(r) - ctr;
              R w = dd_ex2(Te[r * W + ll] - q2 * d * d - P2);
              sw += w;
              sa += w * (Ma[r * W + ll] - qR * d * d);
              R dt = d + R(D1);
              sd += w * (dt * dt + Md[r * W + ll]);
            }
            R isw = R(1) / sw;
            const int qd = 2 * hr + hc;
            const double nt = nut[qd * nst + u];
            const double rh = pick4(rho, qd);
            const double nh = rh * nt;
            hs[qd] += R(nh * ((double)(sa * isw) + (double)bv[kk * Wp + ll] + (rh > 0.0 ? log(rh) : 0.0)));
            hs[4 + qd] += R(nh * (double)(sd * isw));
            hs[8 + qd] += R(nh);
          }
        }
        __syncthreads();
      }
    }   // nothing moves: the sums of pass A stand
    // P_X of the balanced plan: per quadrant, one more X-pass with log2 rho_q added to b + log nu
    R* Lq = bl;
    for (int qd = 0; qd < 4; ++qd) {
      const int hr = qd >> 1, hc = qd & 1;
      if (hr >= nhr || hc >= nhc) continue;
      const int cb = hc * s, ce = min(nx2, cb + s), rb = hr * s, re = min(nx1, rb + s);
      for (int u = tid; u < ny; u += nthr) {
        double rho[4];
        rho_at(u, rho);
        const double rq = pick4(rho, qd);
        const double lr = rq > 0.0 ? log2(rq) : -INFINITY;
        const int v = u / W * Wp + u % W;
        Lq[u] = R(((double)bv[v] + (double)lnu[v]) * DD_LOG2E + lr);
      }
      __syncthreads();
      for (int t = tid; t < H * (ce - cb); t += nthr) {
        const int kk = t / (ce - cb), c = cb + (t - kk * (ce - cb));
        U[kk * nx2 + c] = lse2_1d<R>([&](int m) { return Lq[kk * W + m]; }, W, R(c - offc), q2, R(0), false);
      }
      __syncthreads();
      for (int t = tid; t < (re - rb) * (ce - cb); t += nthr) {
        const int r = rb + t / (ce - cb), c = cb + (t - (t / (ce - cb)) * (ce - cb));
        const int tx = r * nx2 + c;
        R W2 = lse2_1d<R>([&](int m) { return U[m * nx2 + c]; }, H, R(r - offr), q2, R(0), false);
        const int x = (cd.i0 + r) * N + cd.j0 + c;
        double p1 = (double)dd_ex2((lm[tx] + av_c[tx]) * L2E + W2);
        if (!move) p1 = (double)dd_ex2((lm[tx] + av_c[tx]) * L2E + Wv[tx]);
        S.PXnew[x] = p1;
        double p0 = S.PX[x], m = S.mu[x];
        double ps = (1.0 - th_s) * p0 + th_s * p1;
        double k0v = dd_kl_term(p0, m);
        dk[0] += dd_kl_term(p1, m) - k0v;
        dk[1] += dd_kl_term(ps, m) - k0v;
      }
      __syncthreads();
    }
    block_sum<2>(dk, red);
    // the balanced marginals
    if (move) {
      for (int u = tid; u < ny; u += nthr) {
        double rho[4];
        rho_at(u, rho);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if ((k >> 1) < nhr && (k & 1) < nhc) nut[k * nst + u] *= rho[k];
      }
    }
    __threadfence();
    __syncthreads();
  }
  // change of P_Y pi for the step-size decision
  for (int u = tid; u < ny; u += nthr) {
    const int kk = quot(u, W, iW), ll = u - kk * W;
    int y1 = k0 + kk, y2 = l0 + ll;
    double dlt = 0.0;
#pragma unroll
    for (int q4 = 0; q4 < 4; ++q4) {
      if (cd.mem[q4] < 0) continue;
      int hr = q4 >> 1, hc = q4 & 1;
      if (hr >= nhr || hc >= nhc) continue;
      dlt += nut[q4 * nst + u] - box_value(sbox[q4], arena, y1, y2);
    }
    if (dlt != 0.0) atomicAdd(S.dPY + y1 * N + y2, dlt);
  }
  double hsd[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) hsd[k] = (double)hs[k];
  cell_sum<R, 12>(hsd, red);
  if (tid == 0) {
    CellOut o;
    o.k0 = k0; o.l0 = l0; o.H = H; o.W = W;
    o.iters = it;
    o.status = nonfinite ? CELL_NONFINITE : (stops && gap > tol ? CELL_MAXIT : CELL_OK);
    o.D1 = D1; o.D2 = D2;
    o.slot = slot;
    o.usec = (int)min((dd_global_ns() - t_start) / 1000ull, 2147483647ull);
    o.gap = (double)gap;
    o.dKX[0] = dk[0]; o.dKX[1] = dk[1];
    for (int q4 = 0; q4 < 4; ++q4) {
      int bi = cd.mem[q4];
      o.Ct[q4] = S.h * S.h * hsd[4 + q4];
      o.mass[q4] = hsd[8 + q4];
      o.Ht[q4] = bi >= 0 ? hsd[q4] - hsd[8 + q4] + S.muinu[bi] : 0.0;
    }
    *out = o;   // the decision kernel adds the sub-batch's counters
    if (nonfinite) atomicOr(S.status, ST_NONFINITE);
  }
}

// ---------------------------------------------------------------------------
// One cell solved by a cluster of C <= S.dist_c CTAs (the layout's capacities
// were sized for S.dist_c, a smaller C only leaves more room), split by rows
// of its Y box.
// CTA r owns rows [kb, ke) of B_J: the Y-side arrays (log rho, log nu, Z, beta,
// beta + log nu) of those rows live in its shared memory only, so a cluster
// holds C times the Y points of one CTA and the largest cells of a sub-batch
// spread over C SMs.  Per iteration:
//   T pass  (rows of X against the columns of B_J, the same for every slab):
//           targets split over the cluster, every result written to all CTAs
//           (distributed shared memory); cluster barrier;
//   Z pass and the Newton roots of the Y-half on the own rows;
//   U pass (rows of B_J against the columns of X) on the own rows;
//   W partial: the column log-sum-exp of the X-half over the own rows only,
//           written to the exchange buffer of every CTA; cluster barrier;
//   every CTA combines the C partials of each x in rank order (so all CTAs
//           hold the same W, gap and next alpha) -- no further exchange.
// The epilogue splits the rows-of-X pass the same way and sums the
// per-quadrant terms of the own rows; the first CTA adds the cluster's sums.
// Whether a cell with Y box H x W fits the shared memory of a cluster of C CTAs.
__device__ __forceinline__ bool fits_cluster(const DevState& S, int H, int W, int C) {
  const int hl = (H + C - 1) / C;
  return C > 1 && C <= S.dist_c && H >= C && W <= S.dist_cap_w && hl <= S.dist_cap_hl && hl * W <= S.dist_cap_nyl;
}
// Whether it does with the per-y arrays in a spill slot: T, U and beta + log nu,
// and the epilogue's three rows-of-X arrays, share the cluster layout's space.
// (234 x 257 at s = 16: 4.65 ms on one CTA from its slot, 0.65 to 0.72 ms so on eight.)
__device__ __forceinline__ bool fits_hybrid(const DevState& S, int nx1, int nx2, int H, int W, int C) {
  if (C < 2 || C > S.dist_c || H < C || S.spill_slots <= 0) return false;
  const long long Wo = W | 1, Hc = (H + C - 1) / C;
  const long long room = 2LL * S.s * S.dist_cap_w + 2LL * S.s * S.dist_cap_hl + 5LL * S.dist_cap_nyl;
  return nx1 * Wo + Hc * (nx2 | 1) + Hc * Wo <= room && 3LL * nx1 * W <= room && H * Wo <= (long long)S.N * S.N;
}

constexpr int kDistMaxC = 8, kDx = 12;

template <typename R>
__device__ __forceinline__ void cell_solve_dist(const DevState& S, const CellDesc cd, int cidx, int nbatch,
                                                int crank, int C, CellShared<R>& sh, unsigned char* smem_raw) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  double* red = reinterpret_cast<double*>(smem_raw);   // 32 * 16 doubles (block reductions)
  BoxRec* dbox = sh.box;
  int* dgeo = sh.geo;
  CellScalars<R>& sk = sh.sk;
  int& npend = sh.npend;
  bool& stop = sh.stop;
  // partial sums of every CTA of the cluster, kDx each: in double at the end of the reductions'
  // space, beyond the largest sum's 396 values and the gap's parts; the float cells' list lies there
  double* dx = red + 400;
  if constexpr (sizeof(R) == 4) {
    __shared__ double dx_own[kDistMaxC * kDx];
    dx = dx_own;
  }
  CellOut* out = S.cout + cidx;
  const unsigned long long t_start = dd_global_ns();
  const double* __restrict__ arena = S.arena[*S.cur];
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int gtid = crank * nthr + tid, gthr = C * nthr;
  const int N = S.N, s = S.s;
  const int nx1 = cd.nx1, nx2 = cd.nx2, nx = nx1 * nx2;
  auto csync = [&]() { cl.sync(); };

  // ---------------------------------------------------------------- B_J
  // every CTA computes the same box; the first one takes a spill slot for the
  // new marginals when the box exceeds the per-cell marginal buffer and tells
  // the others (its status decides for the whole cluster)
  if (tid == 0) {
    int k0 = 1 << 30, l0 = 1 << 30, k1 = -1, l1 = -1;
    for (int q = 0; q < 4; ++q) {
      BoxRec b = {0, 0, 0, 0, 0};
      if (cd.mem[q] >= 0) b = S.box[cd.mem[q]];
      dbox[q] = b;
      if (cd.mem[q] < 0 || b.H * b.W == 0) continue;
      k0 = min(k0, b.k0); l0 = min(l0, b.l0);
      k1 = max(k1, b.k0 + b.H); l1 = max(l1, b.l0 + b.W);
    }
    int st = CELL_OK;
    if (k1 < 0) {
      st = CELL_EMPTY;
      k0 = l0 = k1 = l1 = 0;
    } else {
      k0 = max(0, k0 - S.margin); l0 = max(0, l0 - S.margin);
      k1 = min(N, k1 + S.margin); l1 = min(N, l1 + S.margin);
    }
    const int H = k1 - k0, W = l1 - l0;
    dgeo[0] = k0; dgeo[1] = l0; dgeo[2] = H; dgeo[3] = W;
    if (crank == 0) {
      int slot = -1;
      const bool fits = fits_cluster(S, H, W, C);
      if (st == CELL_OK && !fits && !fits_hybrid(S, nx1, nx2, H, W, C))
        st = CELL_TOOBIG;   // excluded by k_cell_order; kept as a guard
      if (st == CELL_OK && (!fits || H * W > S.cap_nut)) {
        const int sl = S.spill_slots > 0 ? (int)atomicAdd(S.spill_count, 1u) : S.spill_slots;
        if (sl >= S.spill_slots) st = CELL_TOOBIG;
        else slot = sl;
      }
      for (int r = 0; r < C; ++r) {
        int* g = cl.map_shared_rank(dgeo, r);
        g[4] = st;
        g[7] = slot;
      }
    }
  }
  csync();
  const int k0 = dgeo[0], l0 = dgeo[1], H = dgeo[2], W = dgeo[3];
  const int slot = dgeo[7];
  if (dgeo[4] != CELL_OK) {
    if (tid == 0 && crank == 0) {
      CellOut o;
      o.k0 = k0; o.l0 = l0; o.H = H; o.W = W; o.iters = 0; o.status = dgeo[4];
      o.D1 = o.D2 = 0; o.gap = 0.0; o.dKX[0] = o.dKX[1] = 0.0; o.slot = -1; o.usec = 0;
      for (int q = 0; q < 4; ++q) {
        const int bi = cd.mem[q];
        o.Ct[q] = bi >= 0 ? S.Cc[bi] : 0.0;
        o.Ht[q] = bi >= 0 ? S.Hh[bi] : 0.0;
        o.mass[q] = 0.0;
      }
      *out = o;
      atomicOr(S.status, dgeo[4] == CELL_EMPTY ? ST_EMPTY : ST_TOOBIG);
    }
    return;
  }
  const int kb = (int)(((long long)H * crank) / C), ke = (int)(((long long)H * (crank + 1)) / C);
  const int Hl = ke - kb, nyl = Hl * W;

  // ------------------------------------------------------- shared layout
  // odd row pitches where they fit, as in cell_solve_body
  const int cap_nx = 4 * s * s, cap_xp = cap_nx + 2 * s, xp = nx2 | 1, Wo = W | 1;
  const int Uo = nx2 | 1, Hc = (H + C - 1) / C;   // the same in every CTA
  const bool hyb = !fits_cluster(S, H, W, C);     // then fits_hybrid
  const int tszT = hyb ? nx1 * Wo : 2 * s * S.dist_cap_w, tszU = hyb ? Hc * Uo : 2 * s * S.dist_cap_hl;
  const int Wp = hyb || (nx1 * Wo <= tszT && Hc * Wo <= S.dist_cap_nyl) ? Wo : W;
  const int Up = hyb || Hc * Uo <= tszU ? Uo : nx2;
  const float iW = 1.0f / (float)W, inx2 = 1.0f / (float)nx2;
  R* xa = reinterpret_cast<R*>(smem_raw + 32 * 16 * sizeof(double));
  R* av = xa + cap_xp;
  R* g0 = av + cap_nx;
  R* Wv = g0 + cap_nx;       // W of the X-half, combined over the cluster
  R* lm = Wv + cap_nx;
  R* xa_nx = lm + cap_nx;
  R* av_nx = xa_nx + cap_xp;
  R* Wl = av_nx + cap_nx;    // own rows' part of W (the shift of the next iteration)
  R* Wx = Wl + cap_nx;       // C x cap_nx: the parts of all CTAs
  R* T = Wx + C * cap_nx;    // nx1 x W
  R* U = T + tszT;           // Hl x nx2
  R* bl = U + tszU;
  // a box beyond the cluster's shared memory: the arrays that each y touches once
  // an iteration lie in the cell's spill slot, the own rows from kb on
  R* lrho = hyb ? reinterpret_cast<R*>(S.spill + (long long)slot * S.spill_stride) + kb * Wp : bl + S.dist_cap_nyl;
  const int capy = hyb ? N * N : S.dist_cap_nyl;
  R* Zv = lrho + capy;
  R* bv = Zv + capy;
  R* lnu = bv + capy;

  // ------------------------------------------------- load Y side (a1), own rows
  // rho = max(0, P_Y - nu_J)/nu and log nu; the barycentre of nu_J (the Y frame
  // origin) is summed over the whole box from every CTA's part
  int c1, c2;
  double a_tot = 0.0;   // |nu_{-J}| on B_J (translation step)
  {
    double m3[4] = {0.0, 0.0, 0.0, 0.0};
    for (int ul = tid; ul < nyl; ul += nthr) {
      const int kl = quot(ul, W, iW), ll = ul - kl * W, kk = kb + kl, v = kl * Wp + ll;
      const int y1 = k0 + kk, y2 = l0 + ll, y = y1 * N + y2;
      double nuJ = 0.0;
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) nuJ += box_value(dbox[q4], arena, y1, y2);
      const double num = fmax(0.0, S.PY[y] - nuJ);
      const R rho = R(num) / R(S.nu[y]);
      lrho[v] = rho > R(0) ? dd_lg2(rho) * R(DD_LN2) : -dd_inf<R>();
      lnu[v] = R(S.lognu[y]);
      m3[0] += nuJ; m3[1] += nuJ * kk; m3[2] += nuJ * ll;
      if (S.ti) m3[3] += num;
    }
    cell_sum<R, 4>(m3, red);
    if (tid == 0)
      for (int r = 0; r < C; ++r) {
        double* px = cl.map_shared_rank(dx, r);
        for (int k = 0; k < 4; ++k) px[crank * kDx + k] = m3[k];
      }
    csync();
    double t0 = 0.0, t1 = 0.0, t2 = 0.0;
    for (int r = 0; r < C; ++r) { t0 += dx[r * kDx]; t1 += dx[r * kDx + 1]; t2 += dx[r * kDx + 2]; a_tot += dx[r * kDx + 3]; }
    c1 = H / 2; c2 = W / 2;
    if (t0 > 0.0) {
      c1 = min(H - 1, max(0, (int)lrint(t1 / t0)));
      c2 = min(W - 1, max(0, (int)lrint(t2 / t0)));
    }
  }
  const int xc1 = cd.i0 + nx1 / 2, xc2 = cd.j0 + nx2 / 2;
  const int yc1 = k0 + c1, yc2 = l0 + c2;
  const int D1 = xc1 - yc1, D2 = xc2 - yc2;
  const int offr = (k0 - cd.i0) + D1, offc = (l0 - cd.j0) + D2;
  const double eps = S.eps, q = S.q, sl = S.sl;

  // ------------------------------------------------------- load X side (every CTA)
  const double inv_eps = S.inv_eps;
  double acc2[2] = {0.0, 0.0};
  for (int t = tid; t < nx; t += nthr) {
    const int r = quot(t, nx2, inx2), c = t - r * nx2;
    const int x = (cd.i0 + r) * N + cd.j0 + c;
    const int xi1 = cd.i0 + r - xc1, xi2 = cd.j0 + c - xc2;
    acc2[0] += S.alpha[x] * inv_eps - 2.0 * q * (double)(D1 * xi1 + D2 * xi2);
    acc2[1] += S.mu[x];
  }
  block_sum<2>(acc2, red);
  if (tid == 0) sk.set(S, D1, D2, acc2[0] / nx, acc2[1]);
  __syncthreads();
  double A = sk.A;
  R sB = sk.sB, cA = sk.cA, gA = sk.gA;   // they move with A (translation step)
  const R q2 = sk.q2, qR = sk.qR, sR = sk.sR, rR = sk.rR, cEta1 = sk.cEta1, cEta2 = sk.cEta2, cD1 = sk.cD1,
          cD2 = sk.cD2;
  for (int t = tid; t < nx; t += nthr) {
    const int r = quot(t, nx2, inx2), c = t - r * nx2;
    const int x = (cd.i0 + r) * N + cd.j0 + c;
    const int xi1 = cd.i0 + r - xc1, xi2 = cd.j0 + c - xc2;
    const double lin = 2.0 * q * (double)(D1 * xi1 + D2 * xi2);
    const R a = R(S.alpha[x] * inv_eps - lin - A);
    const R l = R(S.logmu[x]);
    av[t] = a;
    lm[t] = l;
    g0[t] = R(-sl * lin);
    xa[r * xp + c] = (a + l) * R(DD_LOG2E);
  }
  __syncthreads();

  // ------------------------------------------------------- Sinkhorn loop
  const R LN2 = R(DD_LN2), L2E = R(DD_LOG2E);
  const R is = sk.is, i1s = sk.i1s;   // 1/s, 1/(1 + s) (double cells)
  (void)is;
  (void)i1s;
  int* pend = reinterpret_cast<int*>(red + 256);    // as in cell_solve_body
  // translation step, as in cell_solve_body: nu e^{-beta/lam} of the own rows in the
  // cell's buffer of new marginals, every CTA's sum in dx[kDx rk + 4] of all CTAs.  It
  // travels with the parts of W, so it adds no cluster barrier (such cells ran on one
  // CTA before: 256 x 256, s = 8, largest box 11 583 points 1.94 -> 0.70 ms).
  const bool ti = S.ti && sl > 0.0;
  R* apart = reinterpret_cast<R*>(red) + 32;
  R* bpart = apart + 32;
  R* tib;
  {
    CellOut tmp;
    tmp.slot = slot;
    int st;
    tib = reinterpret_cast<R*>(cell_nut(S, tmp, cidx, &st)) + kb * W;
  }
  int it = 0;
  double gap = 0.0;   // of thread 0
  bool first = true;
  R *xa_c = xa, *av_c = av, *xa_n = xa_nx, *av_n = av_nx;
  for (;;) {
    ++it;
    if (tid == 0) npend = 0;
    // Y-half, T(r, ll) = log2 sum_c 2^{xa(r,c) - q2 (c - ll - offc)^2}: split, to every CTA
    run_pass(xa_c, xp, 1, T, Wp, 1, nx1, W, nx2, offc, q2, first, gtid, gthr,
             [&](int r, int ll, int n, const auto& v) {
      for (int rk = 0; rk < C; ++rk) {
        R* Tr = cl.map_shared_rank(T, rk);
        for (int k = 0; k < n; ++k) Tr[r * Wp + ll + k] = v[k];
      }
    });
    csync();
    // Y-half on the own rows: Z(kk, ll) = log2 sum_r 2^{T(r,ll) - q2 (r - kk - offr)^2}, Newton (a3)
    const bool fused_y = sizeof(R) == 4 && nyl * 2 > nthr;
    auto y_store = [&](int v, int y, R u, R Zx, R c0) {   // as in cell_solve_body
      const R b = fused_y ? u - Zx : fma(-Zx, LN2, u);
      Zv[v] = fused_y ? mul_rn(Zx, L2E) : Zx;
      bv[v] = b;
      bl[v] = (b + lnu[v]) * L2E;
      if (ti) tib[y] = dd_ex2((lnu[v] - sR * u - c0) * L2E);
    };
    auto y_root = [&](int ll, int kl, int n, const auto& Z2) {
      constexpr int B = sizeof(Z2) / sizeof(R);
      R lr[B], c0[B], uw[B], root[B], Zn[B];
      const R eta2 = R(l0 + ll - yc2);
#pragma unroll
      for (int k = 0; k < B; ++k) {
        const int v = (kl + min(k, n - 1)) * Wp + ll;
        Zn[k] = mul_rn(k < n ? Z2[k] : Z2[0], LN2);
        const R eta1 = R(k0 + kb + kl + min(k, n - 1) - yc1);
        c0[k] = sB - cEta1 * eta1 - cEta2 * eta2 - sR * Zn[k];
        lr[k] = lrho[v];
        uw[k] = first ? dd_inf<R>() : bv[v] + Zn[k];
      }
      [[maybe_unused]] bool open[B];
      if constexpr (sizeof(R) == 8) {
        root[0] = newton_f64(lr[0], c0[0], uw[0], sR, is, i1s, S.newton_maxit);
      } else {
        newton_tile<R, B>(lr, c0, uw, sR, min(S.newton_maxit, kLock), root, open);
      }
#pragma unroll
      for (int k = 0; k < B; ++k) {
        if (k >= n) break;
        if constexpr (sizeof(R) == 4) {
          if (kLock < S.newton_maxit && open[k]) {
            const int v = (kl + k) * Wp + ll, e = atomicAdd(&npend, 1);
            if (e < kPend) {   // finished below from the list
              pend[e] = v;
              bv[v] = root[k];
              Zv[v] = fused_y ? Zn[k] : Z2[k];
              continue;
            }
            root[k] = newton_rest(lr[k], c0[k], root[k], sR, S.newton_maxit - kLock);
          }
        }
        y_store((kl + k) * Wp + ll, (kl + k) * W + ll, root[k], fused_y ? Zn[k] : Z2[k], c0[k]);
      }
    };
    if constexpr (sizeof(R) == 4) {
      run_pass(T, 1, Wp, Zv, 1, Wp, W, Hl, nx1, offr + kb, q2, first, tid, nthr, y_root);
      __syncthreads();
      const int np = min(npend, kPend);
      const float iWp = 1.0f / (float)Wp;
      for (int e = tid; e < np; e += nthr) {
        const int v = pend[e], kl = quot(v, Wp, iWp), ll = v - kl * Wp;
        const R Zx = Zv[v], Zn = fused_y ? Zx : mul_rn(Zx, LN2);
        const R eta1 = R(k0 + kb + kl - yc1), eta2 = R(l0 + ll - yc2);
        const R c0 = sB - cEta1 * eta1 - cEta2 * eta2 - sR * Zn;
        y_store(v, kl * W + ll, newton_rest(lrho[v], c0, bv[v], sR, S.newton_maxit - kLock), Zx, c0);
      }
    } else {
      run_pass(T, 1, Wp, Zv, 1, Wp, W, Hl, nx1, offr + kb, q2, first, tid, nthr,
               [&](int ll, int kl, int, const auto& v) { Zv[kl * Wp + ll] = v[0]; });
      __syncthreads();
      for (int ul = tid; ul < nyl; ul += nthr) {
        const int kl = quot(ul, W, iW), ll = ul - kl * W;
        const R z[1] = {Zv[kl * Wp + ll]};
        y_root(ll, kl, 1, z);
      }
    }
    if (ti) {
      __syncthreads();
      R bsum = R(0);
      for (int ul = tid; ul < nyl; ul += nthr) bsum += tib[ul];
      bsum = warp_sum(bsum);
      if ((tid & 31) == 0) bpart[tid >> 5] = bsum;
    }
    __syncthreads();
    if (ti && tid == 0) {
      double bs = 0.0;
      for (int w = 0; w < (nthr >> 5); ++w) bs += (double)bpart[w];
      for (int rk = 0; rk < C; ++rk) cl.map_shared_rank(dx, rk)[crank * kDx + 4] = bs;
    }
    // X-half on the own rows: U(kl, c) = log2 sum_ll 2^{bl(kl,ll) - q2 (ll - (c - offc))^2}
    run_pass(bl, Wp, 1, U, Up, 1, Hl, nx2, W, -offc, q2, first, tid, nthr, [&](int kl, int c, int n, const auto& v) {
      for (int k = 0; k < n; ++k) U[kl * Up + c + k] = v[k];
    });
    __syncthreads();
    // the own rows' part of W(r, c) = log2 sum_kk 2^{U(kk,c) - q2 (kk - (r - offr))^2}, to every CTA
    if (Hl > 0) {
      run_pass(U, 1, Up, Wl, 1, nx2, nx2, nx1, Hl, -offr - kb, q2, first, tid, nthr,
               [&](int c, int r0, int n, const auto& v) {
        for (int k = 0; k < n; ++k) Wl[(r0 + k) * nx2 + c] = v[k];
        for (int rk = 0; rk < C; ++rk) {
          R* Wr = cl.map_shared_rank(Wx + crank * cap_nx, rk);
          for (int k = 0; k < n; ++k) Wr[(r0 + k) * nx2 + c] = v[k];
        }
      });
    } else {
      for (int t = tid; t < nx; t += nthr)
        for (int rk = 0; rk < C; ++rk) *cl.map_shared_rank(Wx + crank * cap_nx + t, rk) = -dd_inf<R>();
    }
    csync();
    // combine the parts (rank order: every CTA gets the same W), gap terms (a4), next alpha (a2)
    R gl = R(0), ge = R(0), asum = R(0);   // gl + ge: the thread's gap terms without rounding
    for (int t = tid; t < nx; t += nthr) {
      R mx = -dd_inf<R>();
      for (int rk = 0; rk < C; ++rk) mx = max(mx, Wx[rk * cap_nx + t]);
      R W2 = mx;
      if (mx > -dd_inf<R>()) {
        R acc = R(0);
        for (int rk = 0; rk < C; ++rk) acc += dd_ex2(Wx[rk * cap_nx + t] - mx);
        W2 = mx + dd_lg2(acc);
      }
      Wv[t] = W2;
      const int r = quot(t, nx2, inx2), c = t - r * nx2;
      const R a = av_c[t];
      const R tt = a + W2 * LN2;         // log(P_X pi / mu)
      const R g = gA + g0[t] - sR * a;   // -alpha/lam
      const R term = mul_rn(dd_ex2((lm[t] + g) * L2E), dd_psi<R>(tt - g));
      if constexpr (sizeof(R) == 4) {   // TwoSum (Knuth); at most two terms a thread
        const R sum = __fadd_rn(gl, term), b = __fsub_rn(sum, gl);
        ge += __fadd_rn(__fsub_rn(gl, __fsub_rn(sum, b)), __fsub_rn(term, b));
        gl = sum;
      } else {
        gl += term;
      }
      const R xi1 = R(cd.i0 + r - xc1), xi2 = R(cd.j0 + c - xc2);
      const R an = cA - rR * W2 * LN2 - cD1 * xi1 - cD2 * xi2;
      av_n[t] = an;
      xa_n[r * xp + c] = (an + lm[t]) * L2E;
      if (ti) asum += dd_ex2((lm[t] + gA + g0[t] - sR * an) * L2E);   // mu e^{-alpha_new/lam}
    }
    {
      // The gap is summed in double, as its terms decide when a cell stops: over the
      // warps that hold any, then by warp 0, and one thread decides, so no two
      // threads of a CTA can disagree (every CTA adds the same values in the same order).
      // Float cells first add in float: a tree of 21 roundings of terms >= 0 is within 1.3e-6 of
      // the sum, so only at or below 1.0001 of the bound (or at the last iteration) can the
      // double sum stop the cell, and only then it is formed -- each iteration it cost 6 % of a
      // solve of a thousand iterations.  The parts lie clear of the scratch of the epilogue's
      // first sum, which a warp may reach before another has read the decision.
      const int nw = nthr >> 5, wid = tid >> 5, lane = tid & 31;
      const bool some = 32 * wid < nx;
      R* gfirst = reinterpret_cast<R*>(red + 384);
      double* gpart = red + 384;
      const R gw = some ? warp_sum(gl) : R(0);
      if (lane == 0) gfirst[wid] = gw;
      if (ti) {
        asum = warp_sum(asum);
        if (lane == 0) apart[wid] = asum;
      }
      __syncthreads();
      bool near = true;
      if constexpr (sizeof(R) == 4) {
        R gf = R(0);
        for (int w = 0; w < nw; ++w) gf += gfirst[w];
        near = (S.err >= 0.0 && gf <= fmaf(sk.tol, 1.0001f, 1e-37f)) || it >= S.maxit || !(gf == gf);
      }
      if (near) {   // the same in every thread
        if constexpr (sizeof(R) == 4) {
          double gd = (double)gl + (double)ge;
          if (some) gd = warp_sum(gd);
          __syncthreads();   // gfirst has been read
          if (lane == 0) gpart[wid] = gd;
          __syncthreads();
        }
        if (wid == 0) {
          gap = warp_sum(lane < nw ? gpart[lane] : 0.0);
          if (lane == 0) stop = (S.err >= 0.0 && gap <= sk.bound) || it >= S.maxit || !(gap == gap);
        }
        __syncthreads();
        if (stop) break;
      }
    }
    first = false;
    if (ti) {   // every CTA the same step
      if (tid == 0) {
        double As = 0.0, Bs = 0.0;
        for (int w = 0; w < (nthr >> 5); ++w) As += (double)apart[w];
        for (int rk = 0; rk < C; ++rk) Bs += dx[rk * kDx + 4];
        sk.translate(S, A, a_tot, As, Bs);
      }
      __syncthreads();
      A = sk.A; sB = sk.sB; cA = sk.cA; gA = sk.gA;
    }
    R* tp = av_c; av_c = av_n; av_n = tp;
    tp = xa_c; xa_c = xa_n; xa_n = tp;
  }

  // ------------------------------------------------------- epilogue (a5)
  const double th_s = 1.0 / nbatch;
  double dk[2] = {0.0, 0.0};
  if (crank == 0) {
    for (int t = tid; t < nx; t += nthr) {
      const int r = quot(t, nx2, inx2), c = t - r * nx2;
      const int x = (cd.i0 + r) * N + cd.j0 + c;
      const int xi1 = cd.i0 + r - xc1, xi2 = cd.j0 + c - xc2;
      S.alphanew[x] = eps * (A + (double)av_c[t] + 2.0 * q * (double)(D1 * xi1 + D2 * xi2));
      const double p1 = (double)dd_ex2((lm[t] + av_c[t]) * L2E + Wv[t]);
      S.PXnew[x] = p1;
      const double p0 = S.PX[x];
      if (sizeof(R) == 8) {
        const double m = S.mu[x];
        const double ps = (1.0 - th_s) * p0 + th_s * p1;
        const double k0v = dd_kl_term(p0, m);
        dk[0] += dd_kl_term(p1, m) - k0v;
        dk[1] += dd_kl_term(ps, m) - k0v;
      } else {
        dk[0] += kl_change_f(p0, p1 - p0, lm[t]);
        dk[1] += kl_change_f(p0, th_s * (p1 - p0), lm[t]);
      }
    }
    cell_sum<R, 2>(dk, red);
  }
  R hs[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) hs[k] = R(0);
  const int nhr = nx1 > s ? 2 : 1, nhc = nx2 > s ? 2 : 1;
  int nst;
  double* nut;
  {
    CellOut tmp;
    tmp.slot = slot;
    nut = cell_nut(S, tmp, cidx, &nst);
  }
  // rows of X against the columns of B_J per column half (split, to every CTA);
  // the region T .. Zv is free after the loop
  R* Te = T;
  R* Ma = T + nx1 * W;
  R* Md = Ma + nx1 * W;
  const bool zok = hyb || Md + nx1 * W <= Zv;   // Zv (the final Z, own rows) is intact: the quadrant sums' shift
  for (int hc = 0; hc < nhc; ++hc) {
    const int cb = hc * s, ce = min(nx2, cb + s);
    for (int t = gtid; t < nx1 * W; t += gthr) {
      const int r = quot(t, W, iW), ll = t - r * W;
      const R* row = xa_c + r * xp;
      R ma, md;
      const R T2 = lse_moments<R>([&](int m) { return row[m]; }, [&](int m) { return av_c[r * nx2 + m]; },
                                  [&](int) { return R(0); }, qR, R(D2), cb, ce, R(ll + offc), q2, R(0), false, ma,
                                  md);
      for (int rk = 0; rk < C; ++rk) {
        *cl.map_shared_rank(Te + t, rk) = T2;
        *cl.map_shared_rank(Ma + t, rk) = ma;
        *cl.map_shared_rank(Md + t, rk) = md;
      }
    }
    csync();
    for (int ul = tid; ul < nyl; ul += nthr) {
      const int kl = quot(ul, W, iW), ll = ul - kl * W, kk = kb + kl, v = kl * Wp + ll;
      const int u = kk * W + ll;
      const int y = (k0 + kk) * N + l0 + ll;
      const R ctr = R(kk + offr);
      const double nuy = S.nu[y];
      const R zsh = zok ? Zv[v] : R(0);   // the final Z: an upper bound of every quadrant's sum
      for (int hr = 0; hr < nhr; ++hr) {
        const int rb = hr * s, re = min(nx1, rb + s);
        R ma, md;
        const R P2 = lse_moments<R>(
            [&](int m) { return Te[m * W + ll]; }, [&](int m) { return Ma[m * W + ll]; },
            [&](int m) { return Md[m * W + ll]; }, qR, R(D1), rb, re, ctr, q2, zsh, zok, ma, md);
        const int qd = 2 * hr + hc;
        const R ntv = R(nuy) * dd_ex2(bv[v] * L2E + P2);
        nut[qd * nst + u] = (double)ntv;
        hs[qd] += ntv * (ma + bv[v]);
        hs[4 + qd] += ntv * md;
        hs[8 + qd] += ntv;
      }
    }
    csync();   // Te/Ma/Md are rewritten by the next column half
  }
  // change of P_Y pi for the step-size decision (own rows)
  for (int ul = tid; ul < nyl; ul += nthr) {
    const int kl = quot(ul, W, iW), ll = ul - kl * W, kk = kb + kl;
    const int u = kk * W + ll;
    const int y1 = k0 + kk, y2 = l0 + ll;
    double dlt = 0.0;
#pragma unroll
    for (int q4 = 0; q4 < 4; ++q4) {
      if (cd.mem[q4] < 0) continue;
      const int hr = q4 >> 1, hc = q4 & 1;
      if (hr >= nhr || hc >= nhc) continue;
      dlt += nut[q4 * nst + u] - box_value(dbox[q4], arena, y1, y2);
    }
    if (dlt != 0.0) atomicAdd(S.dPY + y1 * N + y2, dlt);
  }
  double hsd[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) hsd[k] = (double)hs[k];
  cell_sum<R, 12>(hsd, red);
  if (tid == 0) {
    double* p0 = cl.map_shared_rank(dx, 0);
    for (int k = 0; k < 12; ++k) p0[crank * kDx + k] = hsd[k];
  }
  csync();
  if (crank != 0 || tid != 0) return;
  for (int k = 0; k < 12; ++k) {
    double a = 0.0;
    for (int r = 0; r < C; ++r) a += dx[r * kDx + k];
    hsd[k] = a;
  }
  CellOut o;
  o.k0 = k0; o.l0 = l0; o.H = H; o.W = W;
  o.iters = it;
  o.status = !(gap == gap) ? CELL_NONFINITE : (S.err >= 0.0 && gap > sk.bound ? CELL_MAXIT : CELL_OK);
  o.D1 = D1; o.D2 = D2;
  o.slot = slot;
  o.usec = (int)min((dd_global_ns() - t_start) / 1000ull, 2147483647ull);
  o.gap = gap;
  o.dKX[0] = dk[0]; o.dKX[1] = dk[1];
  for (int q4 = 0; q4 < 4; ++q4) {
    const int bi = cd.mem[q4];
    o.Ct[q4] = S.h * S.h * hsd[4 + q4];
    o.mass[q4] = hsd[8 + q4];
    o.Ht[q4] = bi >= 0 ? hsd[q4] - hsd[8 + q4] + S.muinu[bi] : 0.0;
  }
  *out = o;   // the decision kernel adds the sub-batch's counters
  if (!(gap == gap)) atomicOr(S.status, ST_NONFINITE);
}

// One sub-batch, persistent grid over the resident CTAs in clusters of
// C = crun.  Phase 1 (C > 1): each cluster takes the next of the first
// nbig cells of `order` (the largest) and solves it with all its CTAs
// (cell_solve_dist).  Phase 2: every CTA takes the remaining cells one at a
// time (cell_solve_body on one CTA).  The order (largest estimated work first
// within each phase, k_cell_order) only decides when a cell starts; the
// results do not depend on it.
// `crun`: the cluster size of the sub-batch's main grid (<= S.dist_c; k_cell_order
// classified the cells for it); `cluster`: this launch's -- crun for the main
// grid, 1 for a helper grid that runs phase 2 only on the SMs the clusters
// leave idle (both take phase-2 cells from the same queue).
template <typename R, bool BAL>
__global__ void __launch_bounds__(kCellThreads, 1)
k_cell_solve(DevState S, const CellDesc* __restrict__ cells, const int* __restrict__ order,
             const int* __restrict__ nbig_p, int begin, int nbatch, int crun, int cluster) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ CellShared<R> sh;
  __shared__ int sj;
  if (*(volatile int*)S.status & ST_HALT) {   // halted until the host reruns the sub-batch
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nbatch; j += gridDim.x * blockDim.x)
      S.cout[j].status = CELL_SKIPPED;
    return;
  }
  const int C = cluster;
  const int nbig = (crun > 1 && order) ? *nbig_p : 0;
  if (C > 1) {
    const int crank = (int)cg::this_cluster().block_rank();
    // every CTA of the cluster must have started before one writes another's shared memory
    cg::this_cluster().sync();
    for (;;) {
      if (crank == 0 && threadIdx.x == 0) {
        const int j = (int)atomicAdd(S.queue, 1u);
        for (int r = 0; r < C; ++r) *cg::this_cluster().map_shared_rank(&sj, r) = j;
      }
      cg::this_cluster().sync();
      const int j = sj;
      if (j >= nbig) break;
      const int cidx = order[begin + j];
      cell_solve_dist<R>(S, cells[begin + cidx], cidx, nbatch, crank, C, sh, smem_raw);
      cg::this_cluster().sync();
    }
  }
  // no shared memory of another CTA is touched from here on
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) sj = (int)atomicAdd(S.queue + 1, 1u);
    __syncthreads();
    const int j = nbig + sj;
    if (j >= nbatch) break;
    const int cidx = order ? order[begin + j] : j;
    cell_solve_body<R, BAL>(S, cells[begin + cidx], cidx, nbatch, sh, smem_raw);
  }
}

// Estimated work of one cell solve iteration: the exp terms of the four
// separable passes, nx1 nx2 (W + H) + H W (nx1 + nx2), from the member boxes;
// H, W: the cell's Y box.
__device__ __forceinline__ unsigned int cell_cost(const DevState& S, const CellDesc& cd, int* Hout, int* Wout) {
  int k0 = 1 << 30, l0 = 1 << 30, k1 = -1, l1 = -1;
  for (int q = 0; q < 4; ++q) {
    if (cd.mem[q] < 0) continue;
    const BoxRec b = S.box[cd.mem[q]];
    if (b.H * b.W == 0) continue;
    k0 = min(k0, b.k0); l0 = min(l0, b.l0);
    k1 = max(k1, b.k0 + b.H); l1 = max(l1, b.l0 + b.W);
  }
  if (k1 < 0) {
    *Hout = *Wout = 0;
    return 1u;
  }
  const long long H = min(S.N, k1 + S.margin) - max(0, k0 - S.margin);
  const long long W = min(S.N, l1 + S.margin) - max(0, l0 - S.margin);
  *Hout = (int)H;
  *Wout = (int)W;
  const long long c = (long long)cd.nx1 * cd.nx2 * (W + H) + H * W * (cd.nx1 + cd.nx2);
  return (unsigned int)min(c + 1, 0x7fffffffLL);
}

// Whether it fits a cluster of the layout's largest size.
__device__ __forceinline__ bool fits_layout(const DevState& S, int H, int W) {
  return fits_cluster(S, H, W, S.dist_c);
}

constexpr int kOrderMax = 4096;   // largest batch sorted (larger ones keep their index order)

// Order of the cells of each sub-batch of partition `part` (block b:
// sub-batch b; one block for the whole partition when not staggered) and the
// number of leading cells that a whole cluster of C CTAs solves.  mode 0: a
// cell goes to a cluster if it fits the cluster layout and either does not fit
// one CTA or its work exceeds `factor` times the mean work per CTA (`slots`
// CTAs); mode 1:
// every cell that fits the cluster layout; mode 2: none.  Within each group
// the cells are sorted by decreasing work (bitonic sort of (group, cost,
// index) keys in shared memory; ties keep the index order).
__global__ void __launch_bounds__(1024) k_cell_order(DevState S, int part, int mode, int slots, int C,
                                                     double factor) {
  __shared__ unsigned long long key[kOrderMax];
  __shared__ double red[33];
  const int b = blockIdx.x;
  const int begin = S.staggered ? S.sub_start[part][b] : 0;
  const int end = S.staggered ? S.sub_start[part][b + 1] : S.sub_start[part][4];
  const int n = end - begin;
  int* out = S.order[part] + begin;
  int* nbig = S.nbig + part * 4 + b;
  if (*(volatile int*)S.status & ST_HALT) return;   // the sweep's cell launches solve nothing
  if (n <= 0) {
    if (threadIdx.x == 0) *nbig = 0;
    return;
  }
  int P = 1;
  while (P < n) P <<= 1;
  if (P > kOrderMax) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) out[i] = i;
    if (threadIdx.x == 0) *nbig = 0;
    return;
  }
  const CellDesc* cells = S.cells[part];
  double tot[1] = {0.0};
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int H, W;
    tot[0] += (double)cell_cost(S, cells[begin + i], &H, &W);
  }
  block_sum<1>(tot, red);
  const double thr = factor * tot[0] / (double)max(1, slots);
  for (int i = threadIdx.x; i < P; i += blockDim.x) {
    unsigned long long k = 0ull;
    if (i < n) {
      int H, W;
      const unsigned int cost = cell_cost(S, cells[begin + i], &H, &W);
      const bool fits_one = H <= S.cap_side && W <= S.cap_side && H * W <= S.cap_ny;
      const CellDesc& cd = cells[begin + i];
      // a box that a larger cluster holds without a slot is regrouped, not spilled
      const bool fits_dist = fits_cluster(S, H, W, C) ||
                             (!fits_one && !fits_layout(S, H, W) && fits_hybrid(S, cd.nx1, cd.nx2, H, W, C));
      const bool big = mode != 2 && fits_dist && (mode == 1 || !fits_one || (double)cost > thr);
      if (!fits_one && !big && fits_layout(S, H, W) && (mode == 2 || C < S.dist_c)) atomicOr(S.status, ST_REGROUP);
      k = ((unsigned long long)big << 62) | ((unsigned long long)cost << 30) | (0x3fffffffu - (unsigned)i);
    }
    key[i] = k;
  }
  __syncthreads();
  // descending bitonic sort
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long a = key[i], c = key[ixj];
          const bool first_half = (i & k) == 0;
          if (first_half ? (a < c) : (a > c)) { key[i] = c; key[ixj] = a; }
        }
      }
      __syncthreads();
    }
  int cnt = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    out[i] = (int)(0x3fffffffu - (unsigned)(key[i] & 0x3fffffffull));
    cnt += (int)((key[i] >> 62) & 1ull);
  }
  double cv[1] = {(double)cnt};
  block_sum<1>(cv, red);
  if (threadIdx.x == 0) *nbig = (int)cv[0];
}

cudaError_t launch_cell_order(const DevState& S, int part, int mode, int slots, int C, double factor,
                              cudaStream_t st) {
  k_cell_order<<<S.staggered ? 4 : 1, 1024, 0, st>>>(S, part, mode, slots, C, factor);
  return cudaGetLastError();
}

// Many independent instances, one staggered sub-batch of every instance per
// launch: the same two phases as k_cell_solve over the (instance, cell)
// references in the order of k_ref_order -- clusters of C CTAs take the first
// nbig references (each CTA loads that instance's state), then every CTA takes
// the rest one at a time.  C must not exceed any instance's dist_c (its
// cluster layout was sized for dist_c CTAs).
template <typename R>
__global__ void __launch_bounds__(kCellThreads, 1)
k_cell_solve_multi(const DevState* __restrict__ states, const CellRef* __restrict__ refs,
                   const int* __restrict__ order, const int* __restrict__ nbig_p, int nref, int part,
                   unsigned int* queue, int C) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ DevState sS;
  __shared__ CellShared<R> sh;
  __shared__ int sj;
  auto load_state = [&](int inst) {
    const int* src = reinterpret_cast<const int*>(states + inst);
    int* dst = reinterpret_cast<int*>(&sS);
    for (int w = threadIdx.x; w < (int)(sizeof(DevState) / sizeof(int)); w += blockDim.x) dst[w] = src[w];
    __syncthreads();
  };
  // a halted instance (status read once per reference, the same in every CTA
  // of a cluster) solves nothing: its cell is marked skipped
  auto halted = [&](const CellRef& rf) {
    if (!(*(volatile int*)sS.status & ST_HALT)) return false;
    if (threadIdx.x == 0 && (C == 1 || (int)cg::this_cluster().block_rank() == 0))
      sS.cout[rf.pos].status = CELL_SKIPPED;
    return true;
  };
  const int nbig = C > 1 ? *nbig_p : 0;
  if (C > 1) {
    const int crank = (int)cg::this_cluster().block_rank();
    // every CTA of the cluster must have started before one writes another's shared memory
    cg::this_cluster().sync();
    for (;;) {
      if (crank == 0 && threadIdx.x == 0) {
        const int j = (int)atomicAdd(queue, 1u);
        for (int r = 0; r < C; ++r) *cg::this_cluster().map_shared_rank(&sj, r) = j;
      }
      cg::this_cluster().sync();
      const int j = sj;
      if (j >= nbig) break;
      const CellRef rf = refs[order[j]];
      load_state(rf.inst);
      if (!halted(rf)) cell_solve_dist<R>(sS, sS.cells[part][rf.cell], rf.pos, rf.nbatch, crank, C, sh, smem_raw);
      cg::this_cluster().sync();
    }
  }
  // no shared memory of another CTA is touched from here on
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) sj = (int)atomicAdd(queue + 1, 1u);
    __syncthreads();
    const int j = nbig + sj;
    if (j >= nref) break;
    const CellRef rf = refs[order ? order[j] : j];
    load_state(rf.inst);
    if (!halted(rf)) cell_solve_body<R, false>(sS, sS.cells[part][rf.cell], rf.pos, rf.nbatch, sh, smem_raw);
  }
}

constexpr int kRefOrderMax = 8192;   // largest reference list sorted (longer ones keep their order)

// Order of the nref references of one many-instance launch (one block): cluster
// references first -- those whose box fits the instance's cluster layout for C
// CTAs and whose estimated work exceeds `factor` times the mean work per CTA
// (`slots` CTAs), or that do not fit one CTA -- each group by decreasing
// estimated work (as k_cell_order); *nbig = the number of cluster references.
__global__ void __launch_bounds__(1024)
k_ref_order(const DevState* __restrict__ states, const CellRef* __restrict__ refs, int nref, int part, int C,
            double factor, int slots, int* order, int* nbig) {
  extern __shared__ unsigned long long rkey[];
  __shared__ double red[33];
  int P = 1;
  while (P < nref) P <<= 1;
  if (P > kRefOrderMax) {
    for (int i = threadIdx.x; i < nref; i += blockDim.x) order[i] = i;
    if (threadIdx.x == 0) *nbig = 0;
    return;
  }
  double tot[1] = {0.0};
  for (int i = threadIdx.x; i < nref; i += blockDim.x) {
    const CellRef rf = refs[i];
    int H, W;
    tot[0] += (double)cell_cost(states[rf.inst], states[rf.inst].cells[part][rf.cell], &H, &W);
  }
  block_sum<1>(tot, red);
  const double thr = factor * tot[0] / (double)max(1, slots);
  for (int i = threadIdx.x; i < P; i += blockDim.x) {
    unsigned long long k = 0ull;
    if (i < nref) {
      const CellRef rf = refs[i];
      const DevState& S = states[rf.inst];
      int H, W;
      const unsigned int cost = cell_cost(S, S.cells[part][rf.cell], &H, &W);
      const bool fits_one = H <= S.cap_side && W <= S.cap_side && H * W <= S.cap_ny;
      const CellDesc& cd = S.cells[part][rf.cell];
      // a box that a larger cluster holds without a slot is regrouped, not spilled
      const bool fits_dist = fits_cluster(S, H, W, C) ||
                             (!fits_one && !fits_layout(S, H, W) && fits_hybrid(S, cd.nx1, cd.nx2, H, W, C));
      const bool big = fits_dist && (!fits_one || (double)cost > thr);
      if (!fits_one && !big && fits_layout(S, H, W) && C < S.dist_c) atomicOr(S.status, ST_REGROUP);
      k = ((unsigned long long)big << 62) | ((unsigned long long)cost << 30) | (0x3fffffffu - (unsigned)i);
    }
    rkey[i] = k;
  }
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long a = rkey[i], c = rkey[ixj];
          const bool first_half = (i & k) == 0;
          if (first_half ? (a < c) : (a > c)) { rkey[i] = c; rkey[ixj] = a; }
        }
      }
      __syncthreads();
    }
  int cnt = 0;
  for (int i = threadIdx.x; i < nref; i += blockDim.x) {
    order[i] = (int)(0x3fffffffu - (unsigned)(rkey[i] & 0x3fffffffull));
    cnt += (int)((rkey[i] >> 62) & 1ull);
  }
  double cv[1] = {(double)cnt};
  block_sum<1>(cv, red);
  if (threadIdx.x == 0) *nbig = (int)cv[0];
}

size_t cell_smem_bytes(int s, int cap_side, int cap_ny, int precision) {
  size_t rs = precision ? sizeof(double) : sizeof(float);
  size_t cap_nx = 4 * (size_t)s * s, tsz = 2 * (size_t)s * cap_side;
  return 32 * 16 * sizeof(double) + rs * (7 * cap_nx + 4 * (size_t)s + 2 * tsz + 5 * (size_t)cap_ny);
}

// Shared memory of the cluster-distributed layout (cell_solve_dist).
size_t dist_smem_bytes(int s, int C, int cap_w, int cap_hl, int cap_nyl, int precision) {
  const size_t rs = precision ? sizeof(double) : sizeof(float), cap_nx = 4 * (size_t)s * s;
  return 32 * 16 * sizeof(double) +
         rs * ((8 + (size_t)C) * cap_nx + 4 * (size_t)s + 2 * (size_t)s * cap_w + 2 * (size_t)s * cap_hl + 5 * (size_t)cap_nyl);
}

// Static shared memory of the cell kernels, the larger of the single- and the
// many-instance kernel (the dynamic part must leave room for it).
int cell_static_smem(int precision) {
  cudaFuncAttributes a[3];
  cudaError_t e[3];
  if (precision) {
    e[0] = cudaFuncGetAttributes(&a[0], k_cell_solve<double, false>);
    e[1] = cudaFuncGetAttributes(&a[1], k_cell_solve<double, true>);
    e[2] = cudaFuncGetAttributes(&a[2], k_cell_solve_multi<double>);
  } else {
    e[0] = cudaFuncGetAttributes(&a[0], k_cell_solve<float, false>);
    e[1] = cudaFuncGetAttributes(&a[1], k_cell_solve<float, true>);
    e[2] = cudaFuncGetAttributes(&a[2], k_cell_solve_multi<float>);
  }
  size_t m = 0;
  for (int k = 0; k < 3; ++k) {
    if (e[k] != cudaSuccess) {
      cudaGetLastError();
      return 4096;
    }
    m = std::max(m, a[k].sharedSizeBytes);
  }
  return (int)m;
}

// Resident CTAs of the single-instance cell kernel with `smem` dynamic bytes:
// C == 1 single CTAs, C > 1 the CTAs of the resident C-CTA clusters (0 if such
// clusters cannot be scheduled).
int cell_resident_ctas(size_t smem, int C, int precision) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e;
  if (smem > (precision ? allow_smem(k_cell_solve<double, false>) : allow_smem(k_cell_solve<float, false>))) return 0;
  if (C <= 1) {
    int per = 0;
    e = precision ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cell_solve<double, false>, kCellThreads, smem)
                  : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cell_solve<float, false>, kCellThreads, smem);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return nsm > 0 ? nsm : 1;
    }
    return std::max(1, per * nsm);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(kCellThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  e = precision ? cudaOccupancyMaxActiveClusters(&n, k_cell_solve<double, false>, &cfg)
                : cudaOccupancyMaxActiveClusters(&n, k_cell_solve<float, false>, &cfg);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n * C;
}

// One sub-batch: `nctas` persistent CTAs (a multiple of `cluster`, at most the
// resident ones) in clusters of `cluster` (the main grid: crun), `smem` dynamic
// bytes; cluster = 1 with crun > 1 launches single CTAs that run phase 2 only.
cudaError_t launch_cell_solve(const DevState& S, const CellDesc* cells, const int* order, const int* nbig_p,
                              int begin, int nbatch, int precision, size_t smem, int nctas, int crun, int cluster,
                              cudaStream_t st) {
  const int C = std::max(1, cluster);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(std::max(C, nctas / C * C));
  cfg.blockDim = dim3(kCellThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = C > 1 ? 1 : 0;
  auto run = [&](auto kernel) {
    allow_smem(kernel);
    return cudaLaunchKernelEx(&cfg, kernel, S, cells, order, nbig_p, begin, nbatch, crun, C);
  };
  if (S.balance) return precision ? run(k_cell_solve<double, true>) : run(k_cell_solve<float, true>);
  return precision ? run(k_cell_solve<double, false>) : run(k_cell_solve<float, false>);
}

// One many-instance launch: order the references (k_ref_order), then `nctas`
// persistent CTAs (a multiple of C) in clusters of C; `order` and `nbig` are
// device scratch (nref ints, one int), `queue` two counters.
cudaError_t launch_cell_solve_multi(const DevState* states, const CellRef* refs, int nref, int part, int* order,
                                    int* nbig, unsigned int* queue, size_t smem, int precision, int C,
                                    double factor, int nctas, cudaStream_t st) {
  C = std::max(1, C);
  int P = 1;
  while (P < nref) P <<= 1;
  const size_t osm = (size_t)std::min(P, kRefOrderMax) * sizeof(unsigned long long);
  allow_smem(k_ref_order);
  k_ref_order<<<1, 1024, osm, st>>>(states, refs, nref, part, C, factor, nctas, order, nbig);
  cudaMemsetAsync(queue, 0, 2 * sizeof(unsigned int), st);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(std::max(C, nctas / C * C));
  cfg.blockDim = dim3(kCellThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = C > 1 ? 1 : 0;
  if (precision) {
    allow_smem(k_cell_solve_multi<double>);
    return cudaLaunchKernelEx(&cfg, k_cell_solve_multi<double>, states, refs, (const int*)order, (const int*)nbig,
                              nref, part, queue, C);
  }
  allow_smem(k_cell_solve_multi<float>);
  return cudaLaunchKernelEx(&cfg, k_cell_solve_multi<float>, states, refs, (const int*)order, (const int*)nbig, nref,
                            part, queue, C);
}

// Resident CTAs of the many-instance kernel in clusters of C (0: not schedulable).
int cell_multi_resident_ctas(size_t smem, int C, int precision) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (smem > (precision ? allow_smem(k_cell_solve_multi<double>) : allow_smem(k_cell_solve_multi<float>))) return 0;
  cudaError_t e;
  if (C <= 1) {
    int per = 0;
    e = precision ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cell_solve_multi<double>, kCellThreads, smem)
                  : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cell_solve_multi<float>, kCellThreads, smem);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return nsm;
    }
    return std::max(1, per * nsm);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(kCellThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  e = precision ? cudaOccupancyMaxActiveClusters(&n, k_cell_solve_multi<double>, &cfg)
                : cudaOccupancyMaxActiveClusters(&n, k_cell_solve_multi<float>, &cfg);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n * C;
}
