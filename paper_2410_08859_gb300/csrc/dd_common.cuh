// Shared device definitions of the domain-decomposition library (sm_103a).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "dd_log_table.cuh"

#define DD_LOG2E 1.4426950408889634
#define DD_LN2 0.6931471805599453

// ---------------------------------------------------------------- status codes
// Per-cell status written by the cell kernel (CELL_SKIPPED: the launch found
// the handle halted and solved nothing).
enum { CELL_OK = 0, CELL_MAXIT = 1, CELL_EMPTY = 2, CELL_TOOBIG = 3, CELL_NONFINITE = 4, CELL_SKIPPED = 5 };
// Bits of the handle's device status word.  Two of them halt the enqueued
// sweeps (ST_HALT): every later sweep kernel leaves the state untouched until
// the host has handled the cause and re-enqueued the sub-batches that did not
// run.  ST_ARENA: a sub-batch's new boxes would not fit the arena (set by the
// decision kernel before any state changed; the host grows the arena).
// ST_REGROUP: a cell fits neither one CTA nor a cluster of the launch's size
// but does fit the layout's largest cluster (set by the ordering kernel before
// the sub-batch's cell solve; the host switches to that cluster size).
// ST_ARENA_LOST: the allocation guard of the mixing kernel fired (state lost).
enum { ST_TOOBIG = 1, ST_ARENA = 2, ST_EMPTY = 4, ST_NONFINITE = 8, ST_BADINPUT = 16, ST_ARENA_LOST = 32,
       ST_REGROUP = 64, ST_HALT = ST_ARENA | ST_REGROUP };

// ------------------------------------------------------------------ geometry
// One composite cell: its X box [i0, i0+nx1) x [j0, j0+nx2) (always a
// rectangle of real pixels, also for the clipped boundary cells of partition
// B) and the basic cell of each quadrant (row half, column half) relative to
// the X box origin; -1 where the quadrant does not exist.
struct CellDesc {
  int i0, j0, nx1, nx2;
  int mem[4];
};

// Output record of one cell solve.
struct CellOut {
  int k0, l0, H, W;      // the cell's Y box B_J
  int iters, status, D1, D2;
  int slot, usec;        // spill slot of an oversized box (-1: none); duration of the solve (microseconds)
  double Ct[4], Ht[4], mass[4];  // per quadrant: <c, pi~_i>, KL(pi~_i | mu_i x nu), |nu~_i|
  double dKX[2];         // sum_{x in X_J} [mu phi(P'/mu) - mu phi(P/mu)] for theta = 1 and theta_safe
  double gap;            // last PD/lam of the cell
};

// Basic-cell box: Y rows [k0, k0+H), columns [l0, l0+W), values at arena[off..].
struct BoxRec {
  int k0, l0, H, W;
  long long off;
};

// Everything the sweep kernels need; passed by value.
struct DevState {
  int N, s, nb, nbasic;
  double h, eps, lam, thr, err, tau;
  double inv_eps, q, sl, rr;    // 1/eps, h^2/eps, eps/lam, lam/(eps+lam): set with eps (set_eps_scalars)
  int maxit, newton_maxit, strategy, margin;
  int ti;                       // translation step after each cell X-half (0/1)
  double* line;                 // GetWeights_line state (16 doubles)
  int balance;                  // balancing step after each cell solve (0/1; one CTA per cell)
  int cap_ny, cap_side;
  int cap_nut;                  // new marginals per quadrant in a cell position's buffer (>= cap_ny, and the
                                //   cluster capacity dist_c * dist_cap_nyl)
  unsigned char* spill;         // spill slots: Y-side arrays and new marginals of cells too large
  long long spill_stride;       //   for shared memory (bytes per slot)
  long long spill_nut_off;      //   byte offset of the new marginals (4 N^2 doubles) inside a slot
  int spill_slots;              //   number of slots
  unsigned int* spill_count;    //   slots taken in the current launch (reset by k_decide)
  const double *mu, *nu, *logmu, *lognu;
  double* muinu;                // muinu[i] = |mu_i| |nu|
  double *alpha, *PX, *PY, *PXnew, *dPY;
  double* alphanew;             // the cell solves' new alpha on X_J, committed by the mixing kernel
                                // (so a halted sub-batch is solved again from the same alpha)
  double *Cc, *Hh;
  BoxRec* box;
  double* arena[2];
  int* cur;                     // index of the live arena
  unsigned long long* head;     // bump allocator of the live arena
  long long cap;                // capacity of each arena (doubles)
  CellOut* cout;
  double* nut;                  // per cell position: 4 * cap_nut new marginals
  double* theta;                // device scalar: last theta
  double* declog;               // per sub-batch: E0, E(1), E(safe), theta
  unsigned long long* counters; // 0 cell_iters, 1 cell_solves, 2 maxit cells, 3 greedy, 4 safe, 5 max iters,
                                // 6 max ny, 7 lse terms, 8 Y-box points of the cell solves
  int* status;
  double* red;                  // reduction scratch
  unsigned int* red_count;
  // partitions (for kernels that locate their own sub-batch)
  const CellDesc* cells[2];     // cells of partitions A and B, sorted by sub-batch
  int sub_start[2][5];          // sub-batch b of partition p: cells [sub_start[p][b], sub_start[p][b+1])
  int staggered;                // 1: four sub-batches per sweep, 0: one batch of all cells
  unsigned long long* slotctr;  // decision-log records written so far
  long long* newoff;            // compaction scratch: nbasic + 1 offsets
  unsigned int* queue;          // work queues of the persistent cell kernel: [0] cluster phase,
                                //   [1] single-CTA phase (reset by k_decide)
  int* order[2];                // per partition: cells of each sub-batch, cluster cells first, each
                                //   group by decreasing estimated work (k_cell_order)
  int* nbig;                    // [part * 4 + sub]: leading cells of the order solved by a whole cluster
  // capacities of the cluster-distributed cell solve (one cell over dist_c CTAs, split by Y rows)
  int dist_c;                   // CTAs per cluster (1: no cluster phase)
  int dist_cap_w;               // largest Y-box width
  int dist_cap_hl;              // largest number of Y rows per CTA
  int dist_cap_nyl;             // largest number of Y points per CTA
};

inline void set_eps_scalars(DevState& S, double eps) {
  S.eps = eps;
  S.inv_eps = 1.0 / eps;
  S.q = S.h * S.h / eps;
  S.sl = eps / S.lam;
  S.rr = S.lam / (eps + S.lam);
}

#define DD_LOGCAP 4096          // decision-log records kept per instance

// One cell of a many-instance launch: instance, cell index in its partition
// list, and its position within the instance's sub-batch.
struct CellRef {
  int inst, cell, pos, nbatch;
};

// Global nanosecond timer (the same on every SM).
__device__ __forceinline__ unsigned long long dd_global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// ------------------------------------------------------------------ math
__device__ __forceinline__ float dd_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float dd_lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float dd_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 2^x in double by Tang's table-driven method (ACM TOMS 15, 1989): x = k/64 + r,
// |r| <= 1/128, 2^x = 2^(k div 64) T[k mod 64] (1 + expm1(r log 2)) with the Taylor
// polynomial to degree 5 (remainder below 2^-54).  Nine FP64 operations (the FP64
// pipe gives two lanes a clock; CUDA's exp2 takes about twice as many).  At
// |x| >= 1022 (results outside the normal range) and NaN: CUDA's exp2.
__device__ __forceinline__ double dd_ex2(double x) {
  if ((__double2hiint(x) & 0x7fffffff) >= 0x408ff000) return exp2(x);
  const double big = 6755399441055744.0;   // 1.5 2^52: the sum's low word is round(64 x)
  const double t = fma(x, 64.0, big);
  const int k = __double2loint(t);
  const double r = fma(t - big, -0.015625, x);
  double p = fma(r, 1.3333558146428443e-03, 9.6181291076284772e-03);
  p = fma(p, r, 5.5504108664821580e-02);
  p = fma(p, r, 2.4022650695910072e-01);
  p = fma(p, r, 6.9314718055994531e-01);
  const double T = kExp2T[k & 63];
  const double y = fma(T, p * r, T);
  return __hiloint2double(__double2hiint(y) + (int)((unsigned)(k >> 6) << 20), __double2loint(y));
}
__device__ __forceinline__ double dd_log(double x);
__device__ __forceinline__ double dd_lg2(double x) {
  // positive finite: the table logarithm; 0, negative, infinite, NaN: CUDA's
  const unsigned hi = (unsigned)__double2hiint(x);
  if (hi >= 0x7ff00000u || x == 0.0) return log2(x);
  return dd_log(x) * DD_LOG2E;
}
// 1/x from the float reciprocal by two Newton steps (2^-23 -> 2^-46 -> rounding).
__device__ __forceinline__ double dd_rcp(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  if (e < 1023 - 120 || e > 1023 + 120) return 1.0 / x;
  double r = (double)dd_rcp((float)x);
  r = fma(fma(-x, r, 1.0), r, r);
  return fma(fma(-x, r, 1.0), r, r);
}

// float(x) rounded to nearest, for finite |x| < 2^128 (what is below 2^-126 gives 0), on
// the integer pipe: conversions to and from double share the two-lane FP64 path.
__device__ __forceinline__ float narrow(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  if ((hi & 0x7fffffffu) < 0x38100000u) return 0.0f;   // below 2^-126
  unsigned f = __funnelshift_l(lo, hi, 3) - (896u << 23);
  f += (lo & 0x1fffffffu) + (f & 1u) > 0x10000000u ? 1u : 0u;
  return __uint_as_float((f & 0x7fffffffu) | (hi & 0x80000000u));
}
// (float)x for every x (the conversion itself for zeros, subnormals, what exceeds
// the float range, infinities and NaN).
__device__ __forceinline__ float narrow_any(double x) {
  const unsigned a = (unsigned)__double2hiint(x) & 0x7fffffffu;
  return a - 0x38100000u < 0x47e00000u - 0x38100000u ? narrow(x) : (float)x;
}
// double(f) for positive normal f.  0 gives 2^-127, which changes no exponent that a
// squared distance of 0 is multiplied into.
__device__ __forceinline__ double widen_pos(float f) {
  const unsigned u = __float_as_uint(f);
  return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}

template <typename R> __device__ __forceinline__ R dd_inf() { return R(INFINITY); }

// psi(d) = d e^d - e^d + 1 = e^{-g} KL-term ratio (phi(e^d) with phi(s) = s log s - s + 1),
// evaluated by its Taylor series sum_{k>=2} (k-1)/k! d^k near 0 to avoid cancellation.
template <typename R> __device__ __forceinline__ R dd_psi(R d) {
  const R lim = sizeof(R) == 4 ? R(0.25) : R(0.05);
  if (fabs(d) < lim) {
    R d2 = d * d;
    R poly = R(1.0 / 2) + d * (R(1.0 / 3) + d * (R(1.0 / 8) + d * (R(1.0 / 30) + d * (R(1.0 / 144)
             + d * (R(1.0 / 840) + d * (R(1.0 / 5760) + d * (R(1.0 / 45360) + d * R(1.0 / 403200))))))));
    return d2 * poly;
  }
  R e = dd_ex2(d * R(DD_LOG2E));
  return e * (d - R(1)) + R(1);
}

// Natural logarithm of a positive finite double by Tang's table-driven method
// (ACM TOMS 16, 1990): x = 2^e m with m in [0.75, 1.5) (so e = 0 on all of
// [0.75, 1.5) and no cancellation between e log 2 and log c near x = 1);
// c_j = 1 + j/128 is the nearest to m (j = -32..64); f = m - c_j is exact;
// r = f / c_j as f times the rounded reciprocal (|r| <= 2^-7.6); log1p(r) by
// its Taylor polynomial up to r^7 (remainder below 2^-56 relative);
// log x = e log 2 + log c_j + log1p(r).  About 12 FP64 operations against the
// library logarithm's longer sequence; the GPU test compares it with CUDA's
// log (a few ulp).  The tables are generated by gen_log_table.py.
__device__ __forceinline__ void log_parts(double x, double& ed, double& log_c, double& l1p) {
  int hi = __double2hiint(x);
  int lo = __double2loint(x);
  int e = 0;
  if (hi < 0x00100000) {   // subnormal: scale into the normal range
    x *= 18014398509481984.0;   // 2^54
    hi = __double2hiint(x);
    lo = __double2loint(x);
    e = -54;
  }
  e += (hi >> 20) - 1023;
  // m in [1, 2); from 1.5 on the nearest c with spacing 1/64, both halved: index,
  // c_j and e as a double come from integer operations (conversions to and from
  // double share the FP64 path)
  const int mh = hi & 0x000fffff;
  const double m = __hiloint2double(mh | 0x3ff00000, lo);
  const bool up = mh >= 0x00080000;
  const int kk = up ? (mh + 0x2000) >> 14 : (mh + 0x1000) >> 13;
  const double f = m - __hiloint2double(0x3ff00000 + (up ? kk << 14 : kk << 13), 0);   // exact
  const int j = up ? kk - 64 : kk;   // -32..64
  e += up ? 1 : 0;
  ed = __hiloint2double(0x43300000, (int)((unsigned)e ^ 0x80000000u)) - 4503601774854144.0;   // 2^52 + 2^31
  const double inv = kInvC[j + 32];   // halved in place of f
  const double r = f * __hiloint2double(__double2hiint(inv) - (up ? 0x00100000 : 0), __double2loint(inv));
  double p = fma(r, 1.0 / 7.0, -1.0 / 6.0);
  p = fma(p, r, 0.2);
  p = fma(p, r, -0.25);
  p = fma(p, r, 1.0 / 3.0);
  p = fma(p, r, -0.5);
  l1p = fma(p, r * r, r);
  log_c = kLogC[j + 32];
}
__device__ __forceinline__ double dd_log(double x) {
  double ed, log_c, l1p;
  log_parts(x, ed, log_c, l1p);
  return fma(ed, 0.6931471805599453, log_c + l1p);
}

// 1/b for 2^-120 < b < 2^120 to about 2^-44: the float reciprocal and one Newton step.
__device__ __forceinline__ double rcp_short(double b) {
  const double r = widen_pos(dd_rcp(narrow(b)));
  return fma(fma(-b, r, 1.0), r, r);
}
__device__ __forceinline__ bool mid_range(double x, unsigned e = 120u) {   // 2^-e <= x < 2^(e + 1)
  return ((unsigned)__double2hiint(x) >> 20) - (1023u - e) <= 2u * e;
}
// a/b for a >= 0, b > 0: q = a (1/b), corrected by its remainder a - q b (q and 1/b are
// short of their values by 2^-44, so what the correction leaves is 2^-88: a rounding).
__device__ __forceinline__ double dd_div(double a, double b) {
  if (!mid_range(b) || !mid_range(a, 800u)) return a / b;
  const double r = rcp_short(b), q = a * r;
  return fma(fma(-q, b, a), r, q);
}
// log(a/b) for a, b > 0.  With q near a/b as above, log(a/b) = log q + (a - q b)/a up to the
// square of that (2^-88), so the quotient's rounding, the largest part of the error of
// log(a/b) near a = b, drops out; the second part of log 2 leaves one rounding of the
// result and two of the table's value.  Largest error against long arithmetic (a/b in
// 1 +- 0.1 | 0.5..2 | 1e-6..1e6): 1.4e-17 | 8.2e-17 | 9.4e-16; CUDA's log of CUDA's quotient 1.1e-16 |
// 1.6e-16 | 9.8e-16, at 9.53 against 9.11 ms for a 256 x 256 solve with line searches (log a - log b:
// 4e-15 in all three, 8.97).
__device__ __forceinline__ double dd_log_quotient(double a, double b) {
  if (!mid_range(a) || !mid_range(b)) return log(a / b);
  const double r = rcp_short(b), q = a * r;
  const double corr = fma(-q, b, a) * widen_pos(dd_rcp(narrow(a)));
  double ed, log_c, l1p;
  log_parts(q, ed, log_c, l1p);
  return fma(ed, 0.6931471805599453, log_c + (l1p + fma(ed, 2.3190468138462996e-17, corr)));
}

// mu phi(p/mu) with phi(s) = s log s - s + 1 (phi(0) = 1), in double.
__device__ __forceinline__ double dd_kl_term(double p, double m) {
  if (p <= 0.0) return m;
  return p * log(p / m) - p + m;
}

// Allows a kernel all the dynamic shared memory that the device has beside the kernel's
// static one, and returns how much that is (0: an error).  Always that much, never one
// call's need: the limit belongs to the function, and another host thread may be between its
// own call of this and its launch.
inline size_t allow_smem_of(const void* kernel) {
  int dev = 0, optin = 0;
  cudaFuncAttributes a;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, kernel);
  const int room = e == cudaSuccess ? optin - (int)a.sharedSizeBytes : 0;
  if (e == cudaSuccess && a.maxDynamicSharedSizeBytes < room)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, room);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return (size_t)room;
}
template <typename... A> inline size_t allow_smem(void (*kernel)(A...)) {
  return allow_smem_of(reinterpret_cast<const void*>(kernel));
}

// ------------------------------------------------------------- reductions
template <typename T> __device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <typename T> __device__ __forceinline__ T warp_min(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
template <typename T> __device__ __forceinline__ T warp_max(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Block-wide sum of K values per thread; result valid in every thread.
// Warp k (modulo the number of warps) adds the per-warp partials of value k in a
// fixed order (deterministic).  `scratch` must hold 33*K values of type T; ends with a barrier.
template <int K, typename T>
__device__ __forceinline__ void block_sum(T (&v)[K], T* scratch) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = warp_sum(v[k]);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) scratch[wid * K + k] = v[k];
  __syncthreads();
  // warp k (mod the number of warps) combines the partials of value k in a fixed order
  for (int k = wid; k < K; k += nw) {
    T a = lane < nw ? scratch[lane * K + k] : T(0);
    a = warp_sum(a);
    if (lane == 0) scratch[32 * K + k] = a;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = scratch[32 * K + k];
  __syncthreads();
}

// block_sum through shared memory: the np first threads store their K values, warp
// k mod (number of warps) adds value k (np / 32 additions a lane, then five
// shuffles).  On the two-lane FP64 pipe this is K (np / 32 + 5) warp additions
// where the shuffles of every warp are 5 K np / 32 (14 values of 512 threads:
// 18 k clocks; 14 of 128: 2 k).  sm: K * np + K doubles; ends with a barrier.
template <int K>
__device__ __forceinline__ void block_sum_wide(double (&v)[K], double* sm, int np) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  if ((int)threadIdx.x < np)
#pragma unroll
    for (int k = 0; k < K; ++k) sm[k * np + threadIdx.x] = v[k];
  __syncthreads();
  for (int k = wid; k < K; k += nw) {
    double a = 0.0;
    for (int i = lane; i < np; i += 32) a += sm[k * np + i];
    a = warp_sum(a);
    if (lane == 0) sm[K * np + k] = a;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = sm[K * np + k];
  __syncthreads();
}

// block_sum of K doubles whose warp sums split the values over the lanes: at the
// first steps a lane passes half of its values on and keeps the sums of the other
// half, so K values take about K + 4 shuffled additions a warp where K warp sums take
// 5 K (K = 12: 16 against 60; the FP64 pipe gives two lanes a clock, so 16 warps
// of 60 additions are 15 k clocks).  Same precision: every addition is a double one.
// scratch: 33 K doubles.
template <int K>
__device__ __forceinline__ void block_sum_split(double (&v)[K], double* scratch) {
  constexpr int KP = K > 16 ? 32 : K > 8 ? 16 : K > 4 ? 8 : K > 2 ? 4 : K;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  double u[KP];
#pragma unroll
  for (int k = 0; k < KP; ++k) u[k] = k < K ? v[k] : 0.0;
  int idx = 0, o = 1;   // the value that the lane ends with
#pragma unroll
  for (int h = KP / 2; h > 0; h >>= 1, o <<= 1) {
    const bool up = lane & o;
    idx += up ? h : 0;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const double give = up ? u[k] : u[k + h], keep = up ? u[k + h] : u[k];
      u[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  for (; o < 32; o <<= 1) u[0] += __shfl_xor_sync(0xffffffffu, u[0], o);
  if (lane < KP && idx < K) scratch[wid * K + idx] = u[0];
  __syncthreads();
  for (int k = wid; k < K; k += nw) {
    double a = lane < nw ? scratch[lane * K + k] : 0.0;
    a = warp_sum(a);
    if (lane == 0) scratch[32 * K + k] = a;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = scratch[32 * K + k];
  __syncthreads();
}

// Two-stage grid reduction (deterministic): each of G blocks writes its K
// block sums to partials[blockIdx.x * K + k]; k_sum_partials then adds the G
// rows in block order.  With G = 1 the single block writes the result itself.
// G is at most kRedBlocks, a fixed grid (two blocks per SM of GB300's 152 SMs)
// that sizes the partial buffers; it is not a device query and any SM count works.
constexpr int kRedBlocks = 304;
inline int red_blocks(long long n, int threads, const double* partials) {
  if (!partials) return 1;
  long long g = (n + threads - 1) / threads;
  return (int)(g < 1 ? 1 : (g > kRedBlocks ? kRedBlocks : g));
}
template <int K>
__device__ __forceinline__ void block_sum_to(double (&v)[K], double* scratch, double* dst) {
  block_sum<K>(v, scratch);
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) dst[blockIdx.x * K + k] = v[k];
}
__global__ void k_sum_partials(const double* partials, int G, int K, double* out);

// New marginals of cell position j of the current launch (quadrant stride in *stride).
__device__ __forceinline__ double* cell_nut(const DevState& S, const CellOut& o, int j, int* stride) {
  if (o.slot >= 0) {
    *stride = S.N * S.N;
    return reinterpret_cast<double*>(S.spill + (long long)o.slot * S.spill_stride + S.spill_nut_off);
  }
  *stride = S.cap_nut;
  return S.nut + (long long)j * 4 * S.cap_nut;
}
