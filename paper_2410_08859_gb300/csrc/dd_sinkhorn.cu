// Global unbalanced Sinkhorn on the N x N grid (Eq. sinkhorn-iters-ot, nu_- = 0):
// the comparator of Section 5.3, the warm start of DomDec, and the global
// log-sum-exp of the primal-dual certificate.
//
// A half-step needs, for every x, L(x) = log sum_y exp(f(y) - |x-y|^2/eps) with
// f = pot/eps + log m.  Two evaluations:
//  * dense      : all N^2 terms per x (the plain method), f tiled through shared memory;
//  * separable  : |x-y|^2 = (x1-y1)^2 + (x2-y2)^2, so L is a 1-D log-sum-exp along rows
//                 followed by one along columns: 2 N^3 terms instead of N^4.
// Values are kept in log2 units (ex2/lg2); float or double arithmetic.
#include <algorithm>
#include <cmath>

#include "dd_common.cuh"
#include "domdec.h"

namespace {

// Terms more than `cut` (log2 units) below the maximum are skipped: at most N
// of them change the sum by N 2^-cut relative (< 1e-15 in double, < 1e-7 in float).
template <typename R> __device__ __forceinline__ R cut_log2() { return sizeof(R) == 4 ? R(32) : R(64); }

// After a second pass: the half-step's potential and the next pass's input, in
// place of two launches (pot == NULL: none).  For each pixel, pot = -kappa z and
// in2 = (pot/eps + log m) log2 e (and its float shadow).
template <typename R>
struct SepHalf {
  double* pot;
  const double* logm;
  R* in2;
  float* in2f;
  double kappa, inv_eps;
};

constexpr int kSepLanes = 4;    // lanes per target, one residue of the source index modulo 4 each
constexpr int kSepBlock = 16;   // sources per block maximum

// Row pass with a transposed store: dst[j*N + k] = log2 sum_l 2^{src[k*N + l] - q2 (j - l)^2}
// (blockIdx.x = row k; blockIdx.y: a range of targets).  Applied twice it gives the
// 2-D log-sum-exp in the original layout (the second pass runs along the columns
// of the original image), with every source read from shared memory.
//
// With `shifted`, dst holds the previous iteration's values on entry and each
// target is summed against its previous value: terms more than `cut` below the
// shift are left out, so the skipped mass is below N 2^-cut of the sum.  When the
// shift is unusable -- not finite, a term more than 60 above it, or a sum outside
// [2^-30, 2^60] -- and without `shifted`, the target is summed against its
// maximum.  The tests run in float on the shadow values; only kept terms are
// evaluated in R.  FAST (double only): a kept term's exponent is formed in double
// and only its exponential (at most `cut` below the shift) in float (ex2.approx);
// the sums stay double.  The sum's relative error is ~1e-7, i.e. ~1e-7 absolute
// in log2 units, whatever the magnitude of the exponents.
//
// Bound: the FP64 pipe (two lanes a clock): 3 (FAST) or 12 operations per kept
// term.  So a target's window of sources is found first, in float and by the
// maxima of blocks of 16 sources: the lanes of a warp (8 neighbouring targets)
// then run over nearly the same window, where a test of every source held all of
// them for any one's term; the products q2 d come from a table and the
// logarithms are taken by full warps at the end.  Measured, before -> now:
// 256 x 256 FAST at eps = 8 h^2 71 -> 33 us, 32 h^2 103 -> 47; float 12.5 -> 9.5 (128 h^2);
// 1024 x 1024 FAST 802 -> 317 (2 h^2), float 542 -> 127 (128 h^2); 64 x 64 double 27 -> 12 (the
// rows split over several CTAs to reach all SMs).  WIDE: no windows, every source tested
// (see sep_pass).
template <typename R, bool FAST, bool WIDE>
__global__ void __launch_bounds__(1024)
k_sep_rows_t(const R* __restrict__ src, const float* __restrict__ srcf, R* dst, float* __restrict__ dstf, int N,
             double q2, int shifted, int per, SepHalf<R> half) {
  extern __shared__ __align__(16) unsigned char sm[];
  constexpr bool DBL = sizeof(R) == 8;
  R* row = reinterpret_cast<R*>(sm);
  R* accS = row + N;
  R* sigS = accS + per;
  double* qd = reinterpret_cast<double*>(sigS + per + (N & 1));   // double: (q2 d, d), 16-byte aligned
  float* rowf = DBL ? reinterpret_cast<float*>(qd + 2 * N) : reinterpret_cast<float*>(row);
  float* bm = DBL ? rowf + N : reinterpret_cast<float*>(qd);
  const int k = blockIdx.x, nb = (N + kSepBlock - 1) / kSepBlock;
  const int j_lo = blockIdx.y * per, j_n = min(per, N - j_lo);
  for (int l = threadIdx.x; l < N; l += blockDim.x) {
    row[l] = src[(long long)k * N + l];
    if (DBL) {
      rowf[l] = srcf[(long long)k * N + l];
      reinterpret_cast<double2*>(qd)[l] = make_double2(q2 * (double)l, (double)l);
    }
  }
  __syncthreads();
  if (!WIDE) {
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
      float m = -INFINITY;
      for (int l = b * kSepBlock; l < min(N, (b + 1) * kSepBlock); ++l) m = fmaxf(m, rowf[l]);
      bm[b] = m;
    }
    __syncthreads();
  }
  const float q2f = (float)q2, cutf = (float)cut_log2<R>() + 1.0f;
  const int P = kSepLanes, part = threadIdx.x & (P - 1), nt = (j_n * P + 31) & ~31;
  // upper bound of the terms of block b at target j (a few ulp are added for the rounding)
  auto bound = [&](int b, int j) {
    const float d = (float)(j - min(max(j, b * kSepBlock), b * kSepBlock + kSepBlock - 1));
    const float u = fmaf(-q2f * d, d, bm[b]);
    return fmaf(1e-6f, fabsf(bm[b]) + fabsf(u), u);
  };
  auto term_f = [&](int m, int j) {
    const float d = (float)(j - m);
    return fmaf(-(q2f * d), d, rowf[m]);
  };
  auto term = [&](int m, int j) {   // each operation rounded (the float results do not depend on contraction)
    const float d = (float)(j - m);
    return __fsub_rn(rowf[m], __fmul_rn(__fmul_rn(q2f, d), d));
  };
  for (int i = threadIdx.x; i < nt; i += blockDim.x) {
    const int t0 = i / P, j = j_lo + min(t0, j_n - 1);
    R sig = shifted ? dst[(long long)j * N + k] : R(0);
    float sigf = (float)sig;
    R acc = R(0);
    bool todo = shifted ? sigf > -INFINITY && sigf < INFINITY : false;
    for (int pass = shifted ? 0 : 1; pass < 2; ++pass) {
      if (pass == 1) {
        // the maximum, from the block with the largest bound and those that can exceed it
        const bool again = !todo;
        float ub = -INFINITY, mx = -INFINITY;
        if (WIDE) {
          for (int m = part; m < N; m += P) mx = fmaxf(mx, term_f(m, j));
        } else {
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
        }
        for (int o = 1; o < P; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (again) {
          sigf = mx;
          sig = R(mx);
          acc = mx > -INFINITY ? R(0) : R(1);   // no finite term: the value is the maximum itself
          todo = mx > -INFINITY;
        } else {
          todo = false;   // this target's sum stands; its neighbours' are repeated
        }
      }
      // the window: from the first to the last block that can hold a kept term
      int lo = N, hi = 0;
      if (WIDE) {
        if (todo) { lo = 0; hi = N; }
      } else {
        if (todo)
          for (int b = part; b < nb; b += P)
            if (bound(b, j) - sigf > -cutf - 1.0f) {
              lo = min(lo, b * kSepBlock);
              hi = max(hi, min(N, (b + 1) * kSepBlock));
            }
        for (int o = 1; o < P; o <<= 1) {
          lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
          hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
      }
      bool over = false;
      R a = R(0);
      for (int m = lo + part; m < hi; m += P) {   // lo is a multiple of 16: residue `part`, ascending
        const float vf = term(m, j) - sigf;
        if (vf > -cutf) {
          over |= vf > 60.0f;
          if constexpr (DBL) {
            const int d = abs(j - m);
            const double2 t = reinterpret_cast<const double2*>(qd)[d];   // q2 d, d
            const double x = fma(-t.x, t.y, row[m]) - sig;
            if (FAST) a += widen_pos(dd_ex2(narrow(x)));
            else a += dd_ex2(x);
          } else {
            a += dd_ex2(vf);
          }
        }
      }
      for (int o = 1; o < P; o <<= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        over |= __shfl_xor_sync(0xffffffffu, (int)over, o) != 0;
      }
      if (todo) acc = a;
      if (pass == 0) {
        todo = todo && !over && acc >= R(9.313225746154785e-10) && acc <= R(1.152921504606847e18);   // [2^-30, 2^60]
        if (!__any_sync(0xffffffffu, !todo)) break;
      }
    }
    if (part == 0 && t0 < j_n) {
      accS[t0] = acc;
      sigS[t0] = sig;
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < j_n; t += blockDim.x) {
    R lg;
    if constexpr (DBL && FAST) lg = log2(accS[t]);   // a last-bit change here moves float exponents of the mixed mode
    else lg = dd_lg2(accS[t]);
    const R v = sigS[t] + lg;
    const long long o = (long long)(j_lo + t) * N + k;
    dst[o] = v;
    if (dstf) dstf[o] = (float)v;
    if (half.pot) {
      const double pot = -half.kappa * (double)v * DD_LN2;
      half.pot[o] = pot;
      const R in = R(fma(pot, half.inv_eps, half.logm[o])) * R(DD_LOG2E);
      half.in2[o] = in;
      if (DBL) half.in2f[o] = (float)in;
    }
  }
}

// Dense: out[x] = log2 sum_y 2^{in[y] - q2 |x - y|^2}, shifted by the previous
// value out[x] when `use_shift` (one pass), exact max-shifted otherwise.
template <typename R>
__global__ void __launch_bounds__(256) k_dense(const R* __restrict__ in, R* __restrict__ out, int N, R q2,
                                               int use_shift) {
  constexpr int TILE = 1024;
  __shared__ R tile[TILE];
  const int n = N * N;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const R x1 = R(x / N), x2 = R(x % N);
  const bool active = x < n;
  R shift = (active && use_shift) ? out[x] : R(0);
  bool exact = !use_shift;
  R acc = R(0), mx = -dd_inf<R>();
  for (int pass = 0; pass < 3; ++pass) {
    // pass 0: shifted sum (if use_shift); pass 1: max (if exact); pass 2: sum (if exact)
    if (pass == 0 && !use_shift) continue;
    if (pass > 0) {
      int need = __syncthreads_or(active && exact);
      if (!need) break;
    }
    for (int t0 = 0; t0 < n; t0 += TILE) {
      __syncthreads();
      for (int t = threadIdx.x; t < TILE && t0 + t < n; t += blockDim.x) tile[t] = in[t0 + t];
      __syncthreads();
      if (!active || (pass > 0 && !exact)) continue;
      const int cnt = min(TILE, n - t0);
      for (int t = 0; t < cnt; ++t) {
        int y = t0 + t;
        R d1 = x1 - R(y / N), d2 = x2 - R(y % N);
        R v = tile[t] - q2 * (d1 * d1 + d2 * d2);
        if (pass == 0) acc += dd_ex2(v - shift);
        else if (pass == 1) mx = max(mx, v);
        else acc += dd_ex2(v - mx);
      }
    }
    if (pass == 0 && active) {
      if (acc > R(1e-25) && acc < R(1e25)) shift = shift + dd_lg2(acc);
      else { exact = true; acc = R(0); }
    }
  }
  if (active) out[x] = exact ? (mx > -dd_inf<R>() ? mx + dd_lg2(acc) : mx) : shift;
}

template <typename R>
__global__ void k_to_log2(const double* __restrict__ pot, const double* __restrict__ logm, double inv_eps,
                          R* __restrict__ out, int n, float* __restrict__ shadow = nullptr) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    R v = R((pot ? pot[i] * inv_eps : 0.0) + logm[i]) * R(DD_LOG2E);
    out[i] = v;
    if (shadow) shadow[i] = (float)v;
  }
}

template <typename R>
__global__ void k_half(const R* __restrict__ lse2, double kappa, double* __restrict__ pot, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    pot[i] = -kappa * (double)lse2[i] * DD_LN2;
}

template <typename R>
__global__ void k_to_nat(const R* __restrict__ lse2, double* __restrict__ out, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = (double)lse2[i] * DD_LN2;
}

// PD/lam = KL(P_X | e^{-alpha/lam} mu) with P_X = mu e^{alpha/eps + w} (Eq. PD-gap-KL).
// And the dual of Eq. dual-problem: out = [gap, sum_y nu e^{beta/eps + z}, conj terms..., |mu|, |nu|]
template <typename R>
__global__ void __launch_bounds__(512)
k_sk_eval(const double* __restrict__ mu, const double* __restrict__ nu, const double* __restrict__ alpha,
          const double* __restrict__ beta, const R* __restrict__ w2, const R* __restrict__ z2, double eps,
          double lam, int n, double* out) {
  __shared__ double red[33 * 6];
  double v[6] = {0, 0, 0, 0, 0, 0};
  const bool fin = isfinite(lam);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double a = alpha[i], m = mu[i];
    double t = a / eps + (double)w2[i] * DD_LN2;  // log(P_X/mu)
    double g = fin ? -a / lam : 0.0;              // log(e^{-alpha/lam})
    v[0] += m * exp(g) * dd_psi<double>(t - g);
    if (z2) {
      double b = beta[i], z = (double)z2[i] * DD_LN2;
      v[1] += nu[i] * exp(b / eps + z);
      v[2] += fin ? lam * (exp(-a / lam) - 1.0) * m : -a * m;
      v[3] += fin ? lam * (exp(-b / lam) - 1.0) * nu[i] : -b * nu[i];
    }
    v[4] += m;
    v[5] += nu[i];
  }
  block_sum_to<6>(v, red, out);
}

// k_sk_eval over the grid; partials: kRedBlocks * 6 doubles (NULL: one block).
template <typename R>
void sk_eval(const double* mu, const double* nu, const double* alpha, const double* beta, const R* w2,
             const R* z2, double eps, double lam, int n, double* d_eval, double* partials, cudaStream_t st) {
  const int G = red_blocks(n, 512, partials);
  if (G == 1) {
    k_sk_eval<R><<<1, 512, 0, st>>>(mu, nu, alpha, beta, w2, z2, eps, lam, n, d_eval);
  } else {
    k_sk_eval<R><<<G, 512, 0, st>>>(mu, nu, alpha, beta, w2, z2, eps, lam, n, partials);
    k_sum_partials<<<1, 32 * 6, 0, st>>>(partials, G, 6, d_eval);
  }
}

// Translation step (optional, not in the paper): after an X-half,
// alpha += (lam/2) log(<e^{-alpha/lam}, mu> / <e^{-beta/lam}, nu>), the maximiser
// of the dual of Eq. dual-problem along (alpha + t, beta - t).
__global__ void __launch_bounds__(512) k_ti_sums(const double* __restrict__ mu, const double* __restrict__ nu,
                                                 const double* __restrict__ alpha, const double* __restrict__ beta,
                                                 double lam, int n, double* out) {
  __shared__ double red[33 * 2];
  double v[2] = {0.0, 0.0};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    v[0] += mu[i] * exp(-alpha[i] / lam);
    v[1] += nu[i] * exp(-beta[i] / lam);
  }
  block_sum_to<2>(v, red, out);
}

__global__ void k_ti_apply(double* __restrict__ alpha, const double* __restrict__ sums, double lam, int n) {
  const double t = 0.5 * lam * log(sums[0] / sums[1]);
  if (!(t == t) || isinf(t)) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) alpha[i] += t;
}

// sums: 2 doubles of device scratch; partials: kRedBlocks * 2 doubles.
void ti_step(const double* mu, const double* nu, double* alpha, const double* beta, double lam, int n,
             double* sums, double* partials, cudaStream_t st) {
  const int G = red_blocks(n, 512, partials);
  k_ti_sums<<<G, 512, 0, st>>>(mu, nu, alpha, beta, lam, n, partials);
  k_sum_partials<<<1, 32 * 2, 0, st>>>(partials, G, 2, sums);
  k_ti_apply<<<(n + 255) / 256, 256, 0, st>>>(alpha, sums, lam, n);
}

template <typename R>
struct Work {
  R *in2, *tmp, *w2, *z2, *tmpz;
  float *in2f, *tmpf;  // float shadows (double precision only)
};

// One separable pass: a CTA per row, or several where the rows alone are fewer
// than four per SM of a 152-SM GPU or where the targets' values do not fit beside the row
// (double: N > 5250; the row alone fits up to N = 8200 in double, 54000 in float).
template <typename R, bool FAST>
cudaError_t sep_pass(const R* in, const float* inf, R* out, float* outf, int N, double q2, int shifted,
                     const SepHalf<R>& half, cudaStream_t st) {
  const int gy = std::max(1, std::min((N + 15) / 16, (608 + N - 1) / N));
  const int nb = (N + kSepBlock - 1) / kSepBlock;
  const size_t rowb = sizeof(R) * ((size_t)N + 1) + (sizeof(R) == 8 ? 20 * (size_t)N : 0) + 4 * (size_t)nb + 16;
  int per = (N + gy - 1) / gy;
  if (rowb + 2 * sizeof(R) * (size_t)per > 48 * 1024) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (rowb + 2 * sizeof(R) * 16 > (size_t)optin) return cudaErrorInvalidConfiguration;
    per = (int)std::min<size_t>(per, (optin - rowb) / (2 * sizeof(R)));
  }
  const int thr = std::min(1024, ((per * kSepLanes + 31) / 32) * 32);
  const size_t sm = rowb + 2 * sizeof(R) * (size_t)per;
  // Where the distances alone leave no term out (q2 (N - 1)^2 within the cut and a moderate
  // range of the sources) the windows are whole rows, and looking for them only costs: float,
  // us a pass with all its kernels, windows | without: N = 256 at q2 (N - 1)^2 = 11 16.4 | 14.4,
  // 46 16.0 | 14.4, 183 13.5 | 14.4, 1466 10.7 | 14.4; N = 1024 at 46 518 | 493, 184 369 | 491;
  // N = 64 at 11 4.9 | 4.1; double N = 64 at 45 14.4 | 13.3, N = 256 at 46 467 | 467.
  const bool wide = q2 * (double)(N - 1) * (double)(N - 1) <= 64.0;
  auto kernel = wide ? k_sep_rows_t<R, FAST, true> : k_sep_rows_t<R, FAST, false>;
  if (sm > 48 * 1024 && sm > allow_smem(kernel)) return cudaErrorInvalidConfiguration;
  kernel<<<dim3(N, (N + per - 1) / per), thr, sm, st>>>(in, inf, out, outf, N, q2, shifted, per, half);
  return cudaGetLastError();
}

// in2f / tmpf: float shadows (required for R = double; ignored for float).
// use_shift (separable): tmp and out2 hold this evaluation's previous values
// (tmp: the row pass, transposed) and every target is summed against them in
// one pass; otherwise max-shifted.  half (separable only): see SepHalf.
template <typename R>
cudaError_t lse_all(const R* in2, R* tmp, R* out2, int N, double q, int variant, int use_shift, cudaStream_t st,
                    const float* in2f = nullptr, float* tmpf = nullptr, bool fast = false,
                    const SepHalf<R>& half = SepHalf<R>{}) {
  if (variant == 1) {
    const double q2 = q * DD_LOG2E;
    // rows, stored transposed; then the rows of that (the original columns), transposed back
    const int sh = use_shift ? 1 : 0;
    cudaError_t e;
    if constexpr (sizeof(R) == 8) {
      if (fast) {
        e = sep_pass<R, true>(in2, in2f, tmp, tmpf, N, q2, sh, SepHalf<R>{}, st);
        if (e == cudaSuccess) e = sep_pass<R, true>(tmp, tmpf, out2, nullptr, N, q2, sh, half, st);
      } else {
        e = sep_pass<R, false>(in2, in2f, tmp, tmpf, N, q2, sh, SepHalf<R>{}, st);
        if (e == cudaSuccess) e = sep_pass<R, false>(tmp, tmpf, out2, nullptr, N, q2, sh, half, st);
      }
    } else {
      e = sep_pass<R, false>(in2, nullptr, tmp, nullptr, N, q2, sh, SepHalf<R>{}, st);
      if (e == cudaSuccess) e = sep_pass<R, false>(tmp, nullptr, out2, nullptr, N, q2, sh, half, st);
    }
    return e;
  }
  R q2 = R(q * DD_LOG2E);
  int n = N * N;
  k_dense<R><<<(n + 255) / 256, 256, 0, st>>>(in2, out2, N, q2, use_shift);
  return cudaGetLastError();
}

// Iterations of one eps stage of the alternation, from w = the log-sum-exp of
// beta.  Where no check follows, the second pass of a half-step also writes the
// potential and the next input (SepHalf).  check(it) is called every check_every
// iterations and at the last one and returns true to stop.  Returns the
// iterations made, or -1 with the error in *cerr when a pass could not be launched.
template <typename R, typename Check>
int sinkhorn_stage(const double* logmu, const double* lognu, double* alpha, double* beta, R* in2, float* in2f, R* tmp,
                   R* tmpz, float* tmpf, R* w2, R* z2, int N, double e, double kap, int variant, bool fast, int maxit,
                   int check_every, bool fuse, cudaStream_t st, Check check, void (*after_x)(void*), void* ctx, cudaError_t* cerr) {
  const int n = N * N, grid = (n + 255) / 256;
  const double q = (1.0 / N) * (1.0 / N) / e;
  k_to_log2<R><<<grid, 256, 0, st>>>(beta, lognu, 1.0 / e, in2, n, in2f);
  if ((*cerr = lse_all<R>(in2, tmp, w2, N, q, variant, 0, st, in2f, tmpf, fast)) != cudaSuccess) return -1;
  const bool sep = variant == 1;
  bool ready = false;   // alpha and in2 are those of the coming half-step
  int it = 0, shift_ok = 0;
  while (it < maxit) {
    if (!ready) {
      k_half<R><<<grid, 256, 0, st>>>(w2, kap, alpha, n);
      if (after_x) after_x(ctx);
      k_to_log2<R><<<grid, 256, 0, st>>>(alpha, logmu, 1.0 / e, in2, n, in2f);
    }
    if (sep) {
      *cerr = lse_all<R>(in2, tmpz, z2, N, q, variant, shift_ok, st, in2f, tmpf, fast,
                         SepHalf<R>{beta, lognu, in2, in2f, kap, 1.0 / e});
    } else {
      *cerr = lse_all<R>(in2, tmpz, z2, N, q, variant, shift_ok, st, in2f, tmpf, fast);
      k_half<R><<<grid, 256, 0, st>>>(z2, kap, beta, n);
      k_to_log2<R><<<grid, 256, 0, st>>>(beta, lognu, 1.0 / e, in2, n, in2f);
    }
    if (*cerr != cudaSuccess) return -1;
    shift_ok = 1;
    ++it;
    const bool checked = it % check_every == 0 || it == maxit;
    ready = sep && fuse && !checked;
    *cerr = lse_all<R>(in2, tmp, w2, N, q, variant, 1, st, in2f, tmpf, fast,
                       ready ? SepHalf<R>{alpha, logmu, in2, in2f, kap, 1.0 / e} : SepHalf<R>{});
    if (*cerr != cudaSuccess) return -1;
    if (checked && check(it)) break;
  }
  return it;
}

}  // namespace

// Separable FP64 log-sum-exp over the whole grid (natural units):
// out[x] = log sum_y exp(pot[y]/eps + logm[y] - h^2 |x-y|^2/eps).  pot may be NULL.
// buf_a, buf_b, buf_c: N*N doubles of scratch each.
cudaError_t global_lse64(const double* pot, const double* logm, double eps, double h, int N, double* out,
                         double* buf_a, double* buf_b, double* buf_c, cudaStream_t st) {
  int n = N * N;
  float* sh_in = reinterpret_cast<float*>(buf_c);
  float* sh_tmp = sh_in + n;
  k_to_log2<double><<<(n + 255) / 256, 256, 0, st>>>(pot, logm, 1.0 / eps, buf_a, n, sh_in);
  const cudaError_t e = lse_all<double>(buf_a, buf_b, buf_a, N, h * h / eps, 1, 0, st, sh_in, sh_tmp);
  if (e != cudaSuccess) return e;
  k_to_nat<double><<<(n + 255) / 256, 256, 0, st>>>(buf_a, out, n);
  return cudaGetLastError();
}

// Full Sinkhorn driver; all pointers device.  Returns 0, or 1 when the last
// stage hit maxit.  out: [iterations, PD/lam, primal, dual].
template <typename R>
static int full_sinkhorn_impl(const double* mu, const double* nu, const double* logmu, const double* lognu,
                              int N, double eps_start, double eps, double lam, int variant, int maxit,
                              double err, int check_every, double* alpha, double* beta, double* out,
                              double* d_eval, cudaStream_t st, cudaError_t* cerr, bool fast = false) {
  const int n = N * N;
  const bool ti = (variant & DOMDEC_SINKHORN_TI) && std::isfinite(lam);
  variant &= ~DOMDEC_SINKHORN_TI;
  Work<R> w;
  const size_t wbytes = (sizeof(R) * 5 * (size_t)n + sizeof(float) * 2 * (size_t)n + 255) & ~size_t(255);
  *cerr = cudaMallocAsync(&w.in2, wbytes + sizeof(double) * 6 * kRedBlocks, st);
  if (*cerr != cudaSuccess) return -1;
  // row-pass results of the two half-steps kept apart (each is the next shift of its own half-step)
  w.tmp = w.in2 + n; w.w2 = w.tmp + n; w.z2 = w.w2 + n; w.tmpz = w.z2 + n;
  w.in2f = reinterpret_cast<float*>(w.tmpz + n);
  w.tmpf = w.in2f + n;
  double* partials = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(w.in2) + wbytes);
  double evalh[6];
  long long total = 0;
  double gap = INFINITY;
  int rc = 0;
  if (check_every < 1) check_every = 1;
  double e = eps_start > eps ? eps_start : eps;
  for (;;) {
    const double kap = std::isfinite(lam) ? e / (1.0 + e / lam) : e;
    bool conv = false, broke = false;
    struct Ti { const double *mu, *nu; double *alpha; const double* beta; double lam; int n; double *sums, *part; cudaStream_t st; };
    Ti tc{mu, nu, alpha, beta, lam, n, d_eval + 6, partials, st};
    auto ti_run = [](void* p) {
      Ti* t = static_cast<Ti*>(p);
      ti_step(t->mu, t->nu, t->alpha, t->beta, t->lam, t->n, t->sums, t->part, t->st);
    };
    const int it = sinkhorn_stage<R>(
        logmu, lognu, alpha, beta, w.in2, w.in2f, w.tmp, w.tmpz, w.tmpf, w.w2, w.z2, N, e, kap, variant, fast, maxit,
        check_every, !ti, st,
        [&](int) {
          sk_eval<R>(mu, nu, alpha, beta, w.w2, nullptr, e, lam, n, d_eval, partials, st);
          cudaMemcpyAsync(evalh, d_eval, 6 * sizeof(double), cudaMemcpyDeviceToHost, st);
          *cerr = cudaStreamSynchronize(st);
          if (*cerr != cudaSuccess) return broke = true;
          gap = evalh[0];
          conv = err >= 0.0 && gap <= err * evalh[4];
          return conv || !(gap == gap);
        },
        ti ? +ti_run : nullptr, &tc, cerr);
    if (broke || it < 0) { cudaFreeAsync(w.in2, st); return -1; }
    total += it;
    if (e <= eps) { rc = conv || err < 0.0 ? 0 : 1; break; }
    e = fmax(eps, 0.5 * e);
  }
  // primal / dual at the final eps (z from the last Y-half of the final iterate)
  const double kap = std::isfinite(lam) ? eps / (1.0 + eps / lam) : eps;
  (void)kap;
  sk_eval<R>(mu, nu, alpha, beta, w.w2, w.z2, eps, lam, n, d_eval, partials, st);
  cudaMemcpyAsync(evalh, d_eval, 6 * sizeof(double), cudaMemcpyDeviceToHost, st);
  *cerr = cudaStreamSynchronize(st);
  cudaFreeAsync(w.in2, st);
  if (*cerr != cudaSuccess) return -1;
  const double D = eps * evalh[4] * evalh[5] - eps * evalh[1] - evalh[2] - evalh[3];
  const double pd = std::isfinite(lam) ? lam * evalh[0] : evalh[0];
  out[0] = (double)total;
  out[1] = evalh[0];
  out[2] = D + pd;
  out[3] = D;
  return rc;
}

int full_sinkhorn_dev(const double* mu, const double* nu, const double* logmu, const double* lognu, int N,
                      double eps_start, double eps, double lam, int variant, int precision, int maxit,
                      double err, int check_every, double* alpha, double* beta, double* out, double* d_eval,
                      cudaStream_t st, cudaError_t* cerr) {
  if (precision == 2) {
    // float stages while eps >= 64 h^2 (|pot|/eps small enough for float), then double
    const double h = 1.0 / N, e_sw = 64.0 * h * h;
    double o1[4] = {0, 0, 0, 0};
    long long its = 0;
    if (eps_start > e_sw && eps < e_sw) {
      double e_end = e_sw;
      // last float stage is the first eps of the halving sequence below e_sw's bound
      double e = eps_start;
      while (e * 0.5 >= e_sw) e *= 0.5;
      e_end = e;
      int r = full_sinkhorn_impl<float>(mu, nu, logmu, lognu, N, eps_start, e_end, lam, variant, maxit, err,
                                        check_every, alpha, beta, o1, d_eval, st, cerr);
      if (r < 0) return r;
      its += (long long)o1[0];
      int r2 = full_sinkhorn_impl<double>(mu, nu, logmu, lognu, N, 0.5 * e_end, eps, lam, variant, maxit, err,
                                          check_every, alpha, beta, out, d_eval, st, cerr, true);
      out[0] += (double)its;
      return r2;
    }
    precision = eps < e_sw ? 1 : 0;
    if (precision)   // mixed: the double stages take float exponentials of double exponents
      return full_sinkhorn_impl<double>(mu, nu, logmu, lognu, N, eps_start, eps, lam, variant, maxit, err,
                                        check_every, alpha, beta, out, d_eval, st, cerr, true);
  }
  if (precision)
    return full_sinkhorn_impl<double>(mu, nu, logmu, lognu, N, eps_start, eps, lam, variant, maxit, err,
                                      check_every, alpha, beta, out, d_eval, st, cerr);
  return full_sinkhorn_impl<float>(mu, nu, logmu, lognu, N, eps_start, eps, lam, variant, maxit, err,
                                   check_every, alpha, beta, out, d_eval, st, cerr);
}

// ------------------------------------------------------------------------
// Allocation-free variant of the global Sinkhorn.
//
// Some callers cannot allocate device memory while they run this solver: a
// process that has handed all device memory to its own pool at start-up (a
// cudaMalloc would fail or fragment that pool), or a latency-sensitive loop
// that must not pay the implicit device-wide synchronisation of
// cudaMalloc/cudaFree.  For them the working arrays live in one file-scope
// device array of fixed size, reserved on every GPU that loads the library
// for the life of the process.
namespace {
constexpr int kNoAllocMaxN2 = 256 * 256;  // largest grid: N*N <= 65536 (N <= 256)
// log mu, log nu (N*N doubles each), five N*N work arrays of the log-sum-exp
// (double-sized slots, also used for float), one N*N double slot holding two
// float shadow arrays, 8 doubles of reductions and the input-status word.
constexpr long long kNoAllocDoubles = 8LL * kNoAllocMaxN2 + 16;
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocDoubles];

// Device address of the scratch array in the current device's context (host
// code must not use the symbol itself: it is only a host-side stand-in).  It
// is looked up on every call (no allocation, no cache), so it stays right
// after a cudaDeviceReset or under another context of the same device.
cudaError_t noalloc_scratch(double** out) {
  void* p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (e != cudaSuccess) return e;
  *out = static_cast<double*>(p);
  return cudaSuccess;
}

// True if p is device (or managed) memory that the current device can use
// directly; host memory, pinned or pageable, is rejected.
bool is_current_device_ptr(const void* p) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (at.type == cudaMemoryTypeManaged) return true;
  return at.type == cudaMemoryTypeDevice && at.device == dev;
}

template <typename R>
int full_sinkhorn_noalloc_impl(const double* mu, const double* nu, const double* logmu, const double* lognu,
                               int N, double eps_start, double eps, double lam, int variant, int maxit,
                               double err, int check_every, double* alpha, double* beta, double* out,
                               double* work, double* d_eval, cudaStream_t st, cudaError_t* cerr) {
  const int n = N * N;
  // five work arrays in double-sized slots (float arrays use the first half of each)
  R* in2 = reinterpret_cast<R*>(work);
  R* tmp = reinterpret_cast<R*>(work + n);
  R* w2 = reinterpret_cast<R*>(work + 2 * (long long)n);
  R* z2 = reinterpret_cast<R*>(work + 3 * (long long)n);
  R* tmpz = reinterpret_cast<R*>(work + 4 * (long long)n);
  float* in2f = reinterpret_cast<float*>(work + 5 * (long long)n);
  float* tmpf = in2f + n;
  double evalh[6];
  long long total = 0;
  int rc = 0;
  if (check_every < 1) check_every = 1;
  double e = eps_start > eps ? eps_start : eps;
  for (;;) {
    const double kap = std::isfinite(lam) ? e / (1.0 + e / lam) : e;
    bool conv = false, broke = false;
    const int it = sinkhorn_stage<R>(
        logmu, lognu, alpha, beta, in2, in2f, tmp, tmpz, tmpf, w2, z2, N, e, kap, variant, false, maxit, check_every,
        true, st,
        [&](int) {
          k_sk_eval<R><<<1, 512, 0, st>>>(mu, nu, alpha, beta, w2, nullptr, e, lam, n, d_eval);
          cudaMemcpyAsync(evalh, d_eval, 6 * sizeof(double), cudaMemcpyDeviceToHost, st);
          *cerr = cudaStreamSynchronize(st);
          if (*cerr != cudaSuccess) return broke = true;
          conv = err >= 0.0 && evalh[0] <= err * evalh[4];
          return conv || !(evalh[0] == evalh[0]);
        },
        nullptr, nullptr, cerr);
    if (broke || it < 0) return -1;
    total += it;
    if (e <= eps) { rc = conv || err < 0.0 ? 0 : 1; break; }
    e = fmax(eps, 0.5 * e);
  }
  k_sk_eval<R><<<1, 512, 0, st>>>(mu, nu, alpha, beta, w2, z2, eps, lam, n, d_eval);
  cudaMemcpyAsync(evalh, d_eval, 6 * sizeof(double), cudaMemcpyDeviceToHost, st);
  *cerr = cudaStreamSynchronize(st);
  if (*cerr != cudaSuccess) return -1;
  const double D = eps * evalh[4] * evalh[5] - eps * evalh[1] - evalh[2] - evalh[3];
  const double pd = std::isfinite(lam) ? lam * evalh[0] : evalh[0];
  out[0] = (double)total;
  out[1] = evalh[0];
  out[2] = D + pd;
  out[3] = D;
  return rc;
}
}  // namespace

cudaError_t launch_prepare_inputs(const double* mu, const double* nu, double* logmu, double* lognu, int n,
                                  int* status, cudaStream_t st);

int domdec_full_sinkhorn_noalloc(const double* mu, const double* nu, int N, double eps_start,
                                            double eps, double lambda, int variant, int precision, int maxit,
                                            double err, int check_every, const double* beta_in, double* alpha,
                                            double* beta, double out[4], void* stream) {
  if (!mu || !nu || !alpha || !beta || !out || N <= 0) return DOMDEC_EINVAL;
  if (!(eps > 0.0) || !(lambda > 0.0) || (variant != 0 && variant != 1) || (precision != 0 && precision != 1) ||
      maxit < 1)
    return DOMDEC_EINVAL;
  if ((long long)N * N > kNoAllocMaxN2) return DOMDEC_ETOOBIG;
  // the kernels read mu, nu, beta_in and write alpha, beta directly: each must be
  // memory of the current device (a host array would fault or, where the GPU can
  // reach host memory, be used silently)
  if (!is_current_device_ptr(mu) || !is_current_device_ptr(nu) || !is_current_device_ptr(alpha) ||
      !is_current_device_ptr(beta) || (beta_in && !is_current_device_ptr(beta_in)))
    return DOMDEC_EINVAL;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  double* base = nullptr;
  if (noalloc_scratch(&base) != cudaSuccess) return DOMDEC_ECUDA;
  const int n = N * N;
  double* logmu = base;
  double* lognu = base + n;
  double* work = base + 2 * (long long)n;
  double* d_eval = base + 8LL * kNoAllocMaxN2;
  int* d_status = reinterpret_cast<int*>(d_eval + 8);
  // every call starts from a cleared status word and its own beta
  cudaError_t e = cudaMemsetAsync(d_status, 0, sizeof(int), st);
  if (e == cudaSuccess) {
    if (beta_in) {
      if (beta_in != beta) e = cudaMemcpyAsync(beta, beta_in, n * sizeof(double), cudaMemcpyDefault, st);
    } else {
      e = cudaMemsetAsync(beta, 0, n * sizeof(double), st);
    }
  }
  if (e == cudaSuccess) e = launch_prepare_inputs(mu, nu, logmu, lognu, n, d_status, st);
  int hstat = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hstat, d_status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return DOMDEC_ECUDA;
  if (hstat) return DOMDEC_EINVAL;
  cudaError_t ce = cudaSuccess;
  int r = precision ? full_sinkhorn_noalloc_impl<double>(mu, nu, logmu, lognu, N, eps_start, eps, lambda,
                                                         variant, maxit, err, check_every, alpha, beta, out,
                                                         work, d_eval, st, &ce)
                    : full_sinkhorn_noalloc_impl<float>(mu, nu, logmu, lognu, N, eps_start, eps, lambda,
                                                        variant, maxit, err, check_every, alpha, beta, out,
                                                        work, d_eval, st, &ce);
  if (r < 0) return DOMDEC_ECUDA;
  return r ? 1 : 0;
}
