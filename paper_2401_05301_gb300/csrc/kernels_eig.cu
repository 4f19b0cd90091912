// FP64 Hermitian eigen-solver for batches of Gram matrices H = theta' theta'^+.
//
// The truncated SVD of every local update (Sec. II B) is taken through the
// Gram matrix: its eigenvectors are the left singular vectors of theta'.
// Stages (each batched over all triples of a layer):
//   1. Householder reduction H = Q T Q^+ with T real symmetric tridiagonal
//      (reflectors H(k) = I - tau_k v_k v_k^+ with real beta_k, so the
//      sub-diagonal is real), blocked: one cooperative launch per panel of 32
//      columns plus a Hermitian rank-64 update of the trailing matrix.
//   2. Multisection on (division-free) Sturm counts for the kmax largest eigenvalues of T.
//   3. Inverse iteration for the K kept eigenvalues (one thread per
//      eigenvector, LU with partial pivoting of T - lambda I), with
//      Gram-Schmidt inside groups of nearly equal eigenvalues.
//   4. Newton-Schulz orthonormalisation Z <- Z (3I - Z^T Z)/2, three rounds.
//   5. Back-transformation U = Q Z: in blocks of 64 reflectors (compact WY form) in the tensor-core
//      paths, reflector by reflector with a warp per eigenvector in the FP64 path.
// All reductions use a fixed order, so results are bitwise reproducible.
#include "ptebd_internal.h"

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <vector>

namespace ptebd {

namespace {

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {  // a*b + c
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(-a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(a.y, b.x, c.y);
  return c;
}
__device__ __forceinline__ double2 cfma_conj(double2 a, double2 b, double2 c) {  // conj(a)*b + c
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(-a.y, b.x, c.y);
  return c;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return __shfl_sync(0xffffffffu, v, 0);
}
__device__ __forceinline__ double2 warp_sum2(double2 v) { return make_double2(warp_sum(v.x), warp_sum(v.y)); }

// Sum over the block (blockDim.x a multiple of 32, <= 1024); every thread gets the result.
__device__ double block_sum(double v, double* sh) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    double t = (l < nw) ? sh[l] : 0.0;
    t = warp_sum(t);
    if (l == 0) sh[32] = t;
  }
  __syncthreads();
  return sh[32];
}

__device__ double block_min(double v, double* sh) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    double t = (l < nw) ? sh[l] : DBL_MAX;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t = fmin(t, __shfl_xor_sync(0xffffffffu, t, o));
    if (l == 0) sh[32] = t;
  }
  __syncthreads();
  return sh[32];
}

__device__ __forceinline__ double pow2i(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }  // |e| <= 1022

constexpr int NT = 256;

// ---- trace and range ------------------------------------------------------------
// The reduction forms A u and u^+ A u with unnormalised rows u and multiplies by the reflector's scale
// and its square later, so what it holds grows and shrinks like the cube of the entries.  Doubles
// carry that while the trace lies within 2^+-200 (a normalised state's is about 1) and every reflector's
// row reaches 2^-340: |scale|^2 stays below 2^680, u^+ A u above 2^-680 |A|, and what is rounded
// away lies below 2^-394.  The exact-digit trailing update holds v (of order 1) and w (of order A) in one row
// with one exponent, so there the trace has to be near 1: its rounding is 2^-57 of the larger of the two.
// A matrix outside is scaled by a power of two (exact) to a trace of [1, 2), and T is scaled back; eight
// CTAs do it, one cluster per matrix.  Charge blocks of little weight pay that (one pass over them), the
// matrices of a normalised state's dense form do not.
constexpr int RANGE_FP64 = 200, RANGE_DIGITS = 8;
constexpr int TRACE_CTAS = 8;
// Exponent taken out of a matrix of trace tr (0: none, also for a trace that is zero or not finite).
__device__ __forceinline__ int range_shift(double tr, int range) {
  const int ef = (__double2hiint(tr) >> 20) & 0x7FF, e = ef - 1023;
  if (!(tr > 0.0) || ef == 0x7FF || (e >= -range && e <= range)) return 0;
  return max(-1022, min(1022, e));  // (pow2i takes no more; a subnormal trace ends in [2^-52, 1))
}

__global__ void __cluster_dims__(TRACE_CTAS, 1, 1) k_trace(const __grid_constant__ EigBatch b) {
  const EigMat& M = b.a[blockIdx.y];
  __shared__ double sh[33];
  double s = 0.0;
  for (int r = threadIdx.x; r < M.m; r += blockDim.x) s += M.H[(size_t)r * M.m + r].x;
  s = block_sum(s, sh);
  if (threadIdx.x == 0 && blockIdx.x == 0) *M.trace = s;
  const int shift = range_shift(s, b.range);  // the same in all CTAs: each has summed the whole diagonal
  if (shift == 0) return;
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
  const double f = pow2i(-shift);
  const size_t n = (size_t)M.m * M.m;
#pragma unroll 4
  for (size_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += TRACE_CTAS * blockDim.x) {
    const double2 x = M.H[i];
    M.H[i] = make_double2(x.x * f, x.y * f);
  }
}

// ---- bisection --------------------------------------------------------------------
// The tridiagonals for the Sturm counts, in the inverse-iteration scratch (free until the
// eigenvectors are computed): T scaled by a power of two (exact) so that its Gershgorin bound lies in
// [1, 2), as pairs (d_i, e_{i-1}^2), after a header of the scale and the Gershgorin interval.
struct SturmHead {
  double gl, gu;  // Gershgorin interval of the scaled T
  double up, dn;  // scaled = x * up, x = scaled * dn
};
__device__ __forceinline__ SturmHead* sturm_head(const EigMat& M) { return reinterpret_cast<SturmHead*>(M.work); }
__device__ __forceinline__ double2* sturm_pairs(const EigMat& M) { return reinterpret_cast<double2*>(M.work + 4); }

__global__ void __launch_bounds__(256) k_sturm_prep(const __grid_constant__ EigBatch b) {
  const EigMat& M = b.a[blockIdx.x];
  const int m = M.m;
  __shared__ double sh[33];
  if (const int shift = range_shift(*M.trace, b.range)) {  // T back to the matrix's own scale
    const double f = pow2i(shift);
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
      M.d[i] *= f;
      M.e[i] *= f;
    }
    __syncthreads();
  }
  double lo = DBL_MAX, hi = DBL_MAX;  // hi stored negated for a min-reduction
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    double r = 0.0;
    if (i > 0) r += fabs(M.e[i - 1]);
    if (i < m - 1) r += fabs(M.e[i]);
    lo = fmin(lo, M.d[i] - r);
    hi = fmin(hi, -(M.d[i] + r));
  }
  const double gl = block_min(lo, sh), gu = -block_min(hi, sh);
  const double bn = fmax(fabs(gl), fabs(gu));
  int e = 0;
  if (bn > 0.0 && bn < DBL_MAX) e = max(-1020, min(1020, ((__double2hiint(bn) >> 20) & 0x7FF) - 1023));
  const double up = __longlong_as_double((long long)(1023 - e) << 52), dn = __longlong_as_double((long long)(1023 + e) << 52);
  if (threadIdx.x == 0) *sturm_head(M) = SturmHead{gl * up, gu * up, up, dn};
  double2* P = sturm_pairs(M);
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const double ei = (i > 0) ? M.e[i - 1] * up : 0.0;
    P[i] = make_double2(M.d[i] * up, ei * ei);
  }
}

// Number of eigenvalues of the scaled T below x: sign changes of the leading principal
// minors p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (Sturm's theorem), with
// a zero minor counted as a change.  Bound: the FP64 pipe, three dependent instructions of 64 clocks
// a step for a warp alone on its scheduler, so only the recurrence runs there: signs and zeros are
// read from the upper words, and the range is checked every fourth step only, by exact rescaling: a step
// raises the magnitude by less than 2^3 (x and d_i are below 4), and lowers it by more than the 2^60 of a rounded
// difference only beside a minor that vanishes, whose size the count does not use.
__device__ __forceinline__ int sturm_count(const double2* __restrict__ P, int m, double x) {
  double pm = 0.0, p = 1.0;
  int hp = 0x3FF00000, cnt = 0;  // upper word of p
  int i = 0;
  auto step = [&](double2 t) {
    double pn = fma(t.x - x, p, -(t.y * pm));
    int hn = __double2hiint(pn);
    if (((hn << 1) | __double2loint(pn)) == 0) {  // a zero minor takes the sign opposite to the previous one
      hn = 0x20B00000 | (~hp & 0x80000000);       // 2^-500
      pn = __hiloint2double(hn, 0);
    }
    cnt += (int)((unsigned)(hn ^ hp) >> 31);
    pm = p;
    p = pn;
    hp = hn;
  };
  for (; i + 4 <= m; i += 4) {
    const double2 t0 = P[i], t1 = P[i + 1], t2 = P[i + 2], t3 = P[i + 3];
    step(t0);
    step(t1);
    step(t2);
    step(t3);
    const int ex = (hp >> 20) & 0x7FF;
    if (ex > 1023 + 300 || ex < 1023 - 300) {
      const double f = (ex > 1023) ? 0x1p-300 : 0x1p300;
      p *= f;
      pm *= f;
      hp = __double2hiint(p);
    }
  }
  for (; i < m; ++i) step(P[i]);
  return cnt;
}

// Multisection: G lanes per eigenvalue count the eigenvalues below G interior points of its
// interval, which shrinks it by G + 1 per iteration (23 iterations to machine precision with 4 lanes,
// 13 with 16, 11 with 32).  A count is a serial chain of m steps, so more lanes are faster while the
// warps do not outnumber the schedulers, and 4 lanes do the least FP64 work (1.7 counts per bit against
// 3.9 with 16), which is what counts for the hundreds of charge blocks of the blocked form.
// Measured against 4 lanes for all and a range check every step: 256 values of 4 matrices of 1024 5.45 -> 1.9
// ms, 61 of 244 1.29 -> 0.46 ms, 8 of 24 90 -> 35 us; the charge blocks of a chi = 1024, d = 5 cut (4 lanes,
// and the threshold below) 5.4 -> 2.8 ms.
__host__ __device__ __forceinline__ int bisect_lanes(int kmax, int few) {
  return kmax <= 32 ? 32 : few && kmax <= 256 ? 16 : few && kmax <= 512 ? 8 : 4;
}

template <int G>
__device__ void bisect_warp(const EigMat& M, int w) {
  const int m = M.m, lane = threadIdx.x & 31, g = lane / G, sub = lane % G;
  const int j = w * (32 / G) + g;
  const SturmHead H = *sturm_head(M);
  const double2* P = sturm_pairs(M);
  const bool active = j < M.kmax && j < m;
  const double bnorm = fmax(fabs(H.gl), fabs(H.gu));
  const double eps = DBL_EPSILON, tiny = DBL_MIN * fmax(1.0, bnorm * bnorm);
  double lo = H.gl - 2.0 * eps * bnorm * m - 4.0 * tiny;
  double hi = H.gu + 2.0 * eps * bnorm * m + 4.0 * tiny;
  const double atol = 2.0 * eps * bnorm + 4.0 * tiny, frac = (double)(sub + 1) * (1.0 / (G + 1));
  const int target = m - 1 - j;  // ascending index of the j-th largest
  for (int it = 0; it < 64; ++it) {
    const bool conv = !(hi - lo > atol);
    if (__all_sync(0xffffffffu, conv || !active)) break;
    const double x = fma(hi - lo, frac, lo);
    const bool above = active && !conv && sturm_count(P, m, x) > target;  // eigenvalue below x
    const unsigned gb = (__ballot_sync(0xffffffffu, above) >> (G * g)) & (unsigned)((1ull << G) - 1);
    const int l0 = gb ? (__ffs(gb) - 1) : G;  // first point above the eigenvalue (G: none)
    const double xa = __shfl_sync(0xffffffffu, x, G * g + (l0 > 0 ? l0 - 1 : 0));
    const double xb = __shfl_sync(0xffffffffu, x, G * g + (l0 < G ? l0 : G - 1));
    if (active && !conv) {
      if (l0 > 0) lo = xa;
      if (l0 < G) hi = xb;
    }
  }
  if (active && sub == 0) M.evals[j] = 0.5 * (lo + hi) * H.dn;
}

__global__ void __launch_bounds__(128) k_bisect(const __grid_constant__ EigBatch b) {
  const EigMat& M = b.a[blockIdx.y];
  const int km = min(M.kmax, M.m), G = bisect_lanes(M.kmax, b.few);
  // warps of a matrix spread over the blocks first
  const int w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  if (w * (32 / G) >= km) return;
  if (G == 32) bisect_warp<32>(M, w);
  else if (G == 16) bisect_warp<16>(M, w);
  else if (G == 8) bisect_warp<8>(M, w);
  else bisect_warp<4>(M, w);
}

// ---- eigenvalue counts of a cut -------------------------------------------------------
// A cut's spectrum is the union of its matrices' (the charge blocks of one truncated
// SVD).  Rule T keeps at most `target` values of the cut, so each matrix needs only
// its eigenvalues above the cut's target-th largest one (and above the floor
// floor_rel x the cut's trace).  One block per cut finds a threshold by
// multisection on the summed Sturm counts, P points per matrix per iteration, then writes per matrix the
// number of its eigenvalues at or above it (capped by kmax).  The search ends at a point that leaves
// at most 1/32 too many: bisecting those costs less than the iterations that would exclude them (each
// a chain of m steps on one SM), and the vectors are chosen from the eigenvalues themselves later.
__device__ __forceinline__ int count_at_or_above(const EigMat& M, double x) {
  const double xs = x * sturm_head(M)->up;
  if (!(xs < 4.0)) return 0;  // beyond the spectrum's bound (2 in the scaled matrix)
  if (xs < -4.0) return M.m;
  return M.m - sturm_count(sturm_pairs(M), M.m, xs);
}

__global__ void __launch_bounds__(1024) k_cut_counts(const ThrCut* __restrict__ cuts) {
  const ThrCut C = cuts[blockIdx.x];
  __shared__ double sh[33];
  __shared__ int cnt[64];
  __shared__ double lo_sh, hi_sh;
  __shared__ int go_sh;
  // the cut's trace and an upper bound of its spectrum (Gershgorin)
  double tr = 0.0, up = 0.0;
  for (int i = threadIdx.x; i < C.n; i += blockDim.x) {
    tr += *C.mats[i].trace;
    const SturmHead* H = sturm_head(C.mats[i]);
    up = fmax(up, H->gu * H->dn);
  }
  tr = block_sum(tr, sh);
  up = -block_min(-up, sh);
  const double floor_v = C.floor_rel * tr;
  // how many eigenvalues lie at or above the floor
  if (threadIdx.x == 0) cnt[0] = 0;
  __syncthreads();
  {
    int mine = 0;
    for (int i = threadIdx.x; i < C.n; i += blockDim.x) mine += min(C.mats[i].kmax, count_at_or_above(C.mats[i], floor_v));
    atomicAdd(&cnt[0], mine);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    lo_sh = floor_v;
    hi_sh = fmax(up, floor_v) * (1.0 + 4.0 * DBL_EPSILON) + DBL_MIN;
    go_sh = cnt[0] > C.target + C.target / 32;
  }
  __syncthreads();
  const int P = max(1, min(7, (int)blockDim.x / max(C.n, 1)));
  for (int it = 0; it < 80 && go_sh; ++it) {
    const double lo = lo_sh, hi = hi_sh;
    if (threadIdx.x < P) cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int pidx = threadIdx.x; pidx < C.n * P; pidx += blockDim.x) {
      const int i = pidx / P, j = pidx - i * P;
      const double x = lo + (hi - lo) * (double)(j + 1) / (double)(P + 1);
      atomicAdd(&cnt[j], min(C.mats[i].kmax, count_at_or_above(C.mats[i], x)));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int jb = -1;  // the last point still holding at least `target` values
      for (int j = 0; j < P; ++j)
        if (cnt[j] >= C.target) jb = j;
      const double nlo = (jb >= 0) ? lo + (hi - lo) * (double)(jb + 1) / (double)(P + 1) : lo;
      const double nhi = (jb + 1 < P) ? lo + (hi - lo) * (double)(jb + 2) / (double)(P + 1) : hi;
      lo_sh = nlo;
      hi_sh = nhi;
      go_sh = (jb < 0 || cnt[jb] > C.target + C.target / 32) && (nhi - nlo) > 4.0 * DBL_EPSILON * fmax(fabs(nhi), DBL_MIN);
    }
    __syncthreads();
  }
  const double x = lo_sh;
  for (int i = threadIdx.x; i < C.n; i += blockDim.x)
    C.kmax_out[i] = min(C.mats[i].kmax, count_at_or_above(C.mats[i], x));
}

// ---- inverse iteration ----------------------------------------------------------------
__device__ __forceinline__ double hash_uniform(unsigned long long a, unsigned long long b) {
  unsigned long long z = a * 0x9E3779B97F4A7C15ull + b * 0xBF58476D1CE4E5B9ull + 0x94D049BB133111EBull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (double)(z >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
}

// Inverse iteration with T - sigma I = P L U (partial pivoting of a tridiagonal: one fill-in diagonal),
// a thread per eigenvector.  Bound: the FP64 pipe and the serial chain of each thread (64 clocks an
// instruction of a warp alone on its scheduler), so a row costs one division for all three solves
// (the reciprocal of its pivot is kept), the first solve starts from L^-1 P z random (back substitution
// only), magnitudes are compared as integers, vectors are rescaled only when their range asks for it,
// and rows are fetched eight ahead of the chain.
// Scratch, row i of vector q at [i * K + q]: 1/U0, U1, U2, multiplier, and a byte for "rows swapped".
// Measured against divisions in every solve, four passes of scaling per iteration and row-by-row loads: 256
// vectors of 4 matrices of 1024 4.1 -> 1.7 ms, 61 of 244 0.98 -> 0.42 ms.
constexpr int IV_AHEAD = 8;

struct TriFactor {
  double *r0, *u1, *u2, *lm;
  unsigned char* sw;
};
__device__ __forceinline__ TriFactor tri_factor(const EigMat& M, int q) {
  const size_t n = (size_t)M.m * M.K;
  return TriFactor{M.work + q, M.work + n + q, M.work + 2 * n + q, M.work + 3 * n + q,
                   reinterpret_cast<unsigned char*>(M.work + 4 * n) + q};
}

__device__ __forceinline__ double floor_pivot(double u, double tiny) { return fabs(u) < tiny ? copysign(tiny, u) : u; }

__device__ void tri_lu(const double* __restrict__ d, const double* __restrict__ e, int m, double sigma, double tiny,
                       const TriFactor& F, int ld) {
  double u = d[0] - sigma, v = (m > 1) ? e[0] : 0.0;
  for (int i0 = 0; i0 < m - 1; i0 += IV_AHEAD) {
    double ec[IV_AHEAD + 1], dc[IV_AHEAD];
#pragma unroll
    for (int t = 0; t <= IV_AHEAD; ++t) ec[t] = (i0 + t < m - 1) ? e[i0 + t] : 0.0;
#pragma unroll
    for (int t = 0; t < IV_AHEAD; ++t) dc[t] = (i0 + t < m - 1) ? d[i0 + t + 1] : 0.0;
#pragma unroll
    for (int t = 0; t < IV_AHEAD; ++t) {
      const int i = i0 + t;
      if (i >= m - 1) break;
      const double c = ec[t], a = dc[t] - sigma, bb = ec[t + 1];  // row i+1: (c, a, bb)
      const bool swap = fabs(c) > fabs(u);
      const double piv = floor_pivot(swap ? c : u, tiny);
      const double r = 1.0 / piv, l = (swap ? u : c) * r;
      const size_t at = (size_t)i * ld;
      F.r0[at] = r;
      F.u1[at] = swap ? a : v;
      F.u2[at] = swap ? bb : 0.0;
      F.lm[at] = l;
      F.sw[at] = swap ? 1 : 0;
      u = swap ? fma(-l, a, v) : fma(-l, v, a);
      v = swap ? -l * bb : bb;
    }
  }
  const size_t at = (size_t)(m - 1) * ld;
  F.r0[at] = 1.0 / floor_pivot(u, tiny);
  F.u1[at] = 0.0;
  F.u2[at] = 0.0;
}

// z <- L^-1 P (f z), f a power of two.
__device__ void tri_forward(int m, const TriFactor& F, int ld, double f, double* __restrict__ z) {
  double cur = z[0] * f;
  for (int i0 = 0; i0 < m - 1; i0 += IV_AHEAD) {
    double zn[IV_AHEAD], l[IV_AHEAD];
    unsigned char s[IV_AHEAD];
#pragma unroll
    for (int t = 0; t < IV_AHEAD; ++t) {
      const bool in = i0 + t < m - 1;
      const size_t at = (size_t)(i0 + t) * ld;
      zn[t] = in ? z[at + ld] : 0.0;
      l[t] = in ? F.lm[at] : 0.0;
      s[t] = in ? F.sw[at] : 0;
    }
#pragma unroll
    for (int t = 0; t < IV_AHEAD; ++t) {
      if (i0 + t >= m - 1) break;
      const double nxt = zn[t] * f;
      z[(size_t)(i0 + t) * ld] = s[t] ? nxt : cur;
      cur = s[t] ? fma(-l[t], nxt, cur) : fma(-l[t], cur, nxt);
    }
  }
  z[(size_t)(m - 1) * ld] = cur;
}

// z <- U^-1 z; returns the largest upper word of |z|.  rnd != 0: z starts as hash_uniform(rnd, i + 1).
__device__ int tri_back(int m, const TriFactor& F, int ld, unsigned long long rnd, double* __restrict__ z) {
  double z1 = 0.0, z2 = 0.0;  // z[i+1], z[i+2]
  int big = 0;
  for (int i0 = m - 1; i0 >= 0; i0 -= IV_AHEAD) {
    double zz[IV_AHEAD], r[IV_AHEAD], a[IV_AHEAD], c[IV_AHEAD];
#pragma unroll
    for (int t = 0; t < IV_AHEAD; ++t) {
      const bool in = i0 - t >= 0;
      const size_t at = (size_t)(in ? i0 - t : 0) * ld;
      zz[t] = rnd ? hash_uniform(rnd, i0 - t + 1) : z[at];
      r[t] = F.r0[at];
      a[t] = F.u1[at];
      c[t] = F.u2[at];
    }
#pragma unroll
    for (int t = 0; t < IV_AHEAD; ++t) {
      if (i0 - t < 0) break;
      const double zi = fma(-a[t], z1, fma(-c[t], z2, zz[t])) * r[t];
      z[(size_t)(i0 - t) * ld] = zi;
      big = max(big, __double2hiint(zi) & 0x7FFFFFFF);
      z2 = z1;
      z1 = zi;
    }
  }
  return big;
}

__global__ void __launch_bounds__(32) k_inviter(const __grid_constant__ EigBatch b) {
  const EigMat& M = b.a[blockIdx.y];
  const int m = M.m, K = M.K;
  if (blockIdx.x * 32 >= K) return;
  double tnorm = 0.0;  // largest row sum: the warp's lanes take rows in turn
  for (int i = threadIdx.x; i < m; i += 32) {
    double r = fabs(M.d[i]);
    if (i > 0) r += fabs(M.e[i - 1]);
    if (i < m - 1) r += fabs(M.e[i]);
    tnorm = fmax(tnorm, r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tnorm = fmax(tnorm, __shfl_xor_sync(0xffffffffu, tnorm, o));
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= K) return;
  const double* ev = M.evals;
  if (tnorm == 0.0) tnorm = 1.0;
  // Bisection places each shift within ~2 eps tnorm of its eigenvalue; eigenvalues
  // closer than 100x that are treated as one group and orthogonalised explicitly.
  const double gtol = 200.0 * DBL_EPSILON * tnorm;
  if (j > 0 && ev[j - 1] - ev[j] <= gtol) return;  // not the first of its group
  int g = j + 1;
  while (g < K && ev[g - 1] - ev[g] <= gtol) ++g;
  const double tiny = DBL_EPSILON * tnorm;
  const int ld = K;
  for (int q = j; q < g; ++q) {
    const TriFactor F = tri_factor(M, q);
    tri_lu(M.d, M.e, m, ev[q], tiny, F, ld);
    double* z = M.Z + q;
    double f = 1.0;  // brings the last solve's vector to order one, applied when it is next read
    for (int it = 0; it < 3; ++it) {
      if (it > 0) tri_forward(m, F, ld, f, z);
      const int big = tri_back(m, F, ld, it == 0 ? (unsigned long long)q + 1 : 0ull, z);
      const int ex = (big >> 20) - 1023;
      f = (big > 0 && big < 0x7FF00000) ? pow2i(max(-1022, min(1022, -ex))) : 1.0;
      for (int p = j; p < q; ++p) {  // Gram-Schmidt against earlier group members (normalised)
        const double* y = M.Z + p;
        double dot = 0.0;
        for (int i = 0; i < m; ++i) dot = fma(y[(size_t)i * ld], z[(size_t)i * ld] * f, dot);
        for (int i = 0; i < m; ++i) z[(size_t)i * ld] = fma(z[(size_t)i * ld], f, -dot * y[(size_t)i * ld]);
        f = 1.0;
      }
    }
    double nrm = 0.0;
#pragma unroll 8
    for (int i = 0; i < m; ++i) {
      const double x = z[(size_t)i * ld] * f;
      nrm = fma(x, x, nrm);
    }
    nrm = sqrt(nrm);
    const double s = (nrm > 0.0) ? f / nrm : 0.0;
#pragma unroll 8
    for (int i = 0; i < m; ++i) z[(size_t)i * ld] *= s;
  }
}

constexpr int NSS_WORK = 8192;   // K^2 m
constexpr int NSS_SIZE = 2048;   // m K
__host__ __device__ __forceinline__ bool ns_small(int m, int K) {
  return (long long)K * K * m <= NSS_WORK && m * K <= NSS_SIZE;
}
// S <- 1.5 I - 0.5 S
__global__ void k_ns_form(const __grid_constant__ EigBatch b) {
  const EigMat& M = b.a[blockIdx.y];
  const int K = M.K;
  if (ns_small(M.m, K)) return;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < K * K; idx += gridDim.x * blockDim.x) {
    const int r = idx / K, c = idx % K;
    M.S[idx] = (r == c ? 1.5 : 0.0) - 0.5 * M.S[idx];
  }
}

// The three Newton-Schulz rounds of a small matrix in one block, with Z, its successor and S in shared
// memory (result in Z2, as after three rounds of the products).  The limit is where nine launches (4 to 5 us
// each) cost as much as the products on one SM (K^2 m / 16 FP64 warp instructions a round).  Measured, with
// the back-transformation reading Z itself: six small blocked simulations 61.3 -> 56.3 ms a step, blocked L = 41
// quench 34.4 -> 32.1 ms, super sites 9.9 -> 8.0 ms.
__global__ void __launch_bounds__(256) k_ns_small(const __grid_constant__ EigBatch b) {
  const EigMat& M = b.a[blockIdx.x];
  const int m = M.m, K = M.K;
  if (K == 0 || !ns_small(m, K)) return;
  __shared__ double za[NSS_SIZE], zb[NSS_SIZE], S[NSS_WORK / 8];  // K^2 <= K^2 m / m, and m >= K
  double *z = za, *zn = zb;
  for (int e = threadIdx.x; e < m * K; e += blockDim.x) z[e] = M.Z[e];
  __syncthreads();
  for (int it = 0; it < 3; ++it) {
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
      const int r = e / K, c = e - r * K;
      double acc = 0.0;
      for (int i = 0; i < m; ++i) acc = fma(z[i * K + r], z[i * K + c], acc);
      S[e] = (r == c ? 1.5 : 0.0) - 0.5 * acc;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < m * K; e += blockDim.x) {
      const int r = e / K, c = e - r * K;
      double acc = 0.0;
      for (int i = 0; i < K; ++i) acc = fma(z[r * K + i], S[i * K + c], acc);
      zn[e] = acc;
    }
    __syncthreads();
    double* t = z;
    z = zn;
    zn = t;
  }
  for (int e = threadIdx.x; e < m * K; e += blockDim.x) M.Z2[e] = z[e];
}

// U[j][r] = Z[r][j] (real -> complex, transposed).
__global__ void k_z_to_u(const __grid_constant__ EigBatch b, int use_z2) {
  const EigMat& M = b.a[blockIdx.z];
  const int m = M.m, K = M.K;
  __shared__ double tile[32][33];
  const double* Z = use_z2 ? M.Z2 : M.Z;
  const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  if (r0 >= m || c0 >= K) return;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    tile[i][threadIdx.x] = (r < m && c < K) ? Z[(size_t)r * K + c] : 0.0;
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (c < K && r < m) M.U[(size_t)c * m + r] = make_double2(tile[threadIdx.x][i], 0.0);
  }
}

// ---- back-transformation, reflector by reflector (FP64 path) ------------------------------
// U <- H(0) H(1) ... H(m-2) Z, a warp per eigenvector, which it keeps in registers (m <= 256) or shared memory.  The Gram
// matrices are graded (rows scaled by lambda), and applying the reflectors one at a time keeps the small
// leading components of the eigenvectors of small singular values to their own relative accuracy; a
// compact-WY block of 64 in FP64 loses a digit of them (rows u^+ theta' of a graded 24 to 60 row matrix:
// 4e-15 against 2e-14 of s_k).
// Bound: the FP64 pipe, 8 instructions per 32 rows and reflector and 14 for the dot product's sum.
// Measured: 61 vectors of 4 matrices of 244 1.9 ms (8 vectors per block with block-wide sums 2.7 ms), 8 vectors
// of matrices of 4 to 24 35 us (167 us).
constexpr int BTS_SMEM = 12288 * 16;  // one vector of the largest matrix (m <= 12288), four of BTS_WARP
constexpr int BTS_WARP = 3072;        // largest matrix for a warp per vector
// Larger matrices: two vectors fit a block, or one, and the FP64 pipe of an SM is four quarters that one warp cannot
// fill, so four or eight warps share a vector (rows dealt in turn, partial dots added in a fixed order).
// Measured, eigenvector stage of an FP64 layer, against a warp per vector: chi = 1024, d = 4 (m = 4096) 750 -> 462 ms,
// chi = 1536 (m = 6144) 3290 -> 1450 ms.
__host__ __device__ __forceinline__ int btw_vectors(int m) { return m <= 6144 ? 2 : 1; }  // per block of 8 warps
template <int NW>
__device__ __forceinline__ void btw_vector(const EigMat& M, const double* Z, double2* u, double2* out, double2* slots,
                                           int vec, int part) {
  constexpr int STEP = 32 * NW;  // rows keep their warp and lane
  const int m = M.m, lane = threadIdx.x & 31, first = 32 * part + lane;
  int phase = 0;
  for (int r = first; r < m; r += STEP) u[r] = make_double2(Z[(size_t)r * M.K], 0.0);
  for (int k = m - 2; k >= 0; --k) {
    const double2 tau = M.tau[k];
    if (tau.x == 0.0 && tau.y == 0.0) continue;
    const double2* v = M.H + (size_t)k * m;
    const int r0 = ((k + 1) & ~(STEP - 1)) + first;
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int r = r0; r < m; r += STEP)
      if (r > k) acc = cfma_conj(v[r], u[r], acc);
    acc = warp_sum2(acc);
    // two sets of sums in turn: one is written again only after the barrier that follows its reading
    double2* sums = slots + 8 * phase;
    phase ^= 1;
    if (lane == 0) sums[part] = acc;
    asm volatile("bar.sync %0, %1;" ::"r"(1 + vec), "r"(STEP) : "memory");
    acc = sums[0];
#pragma unroll
    for (int q = 1; q < NW; ++q) acc = cadd(acc, sums[q]);
    double2 w = cmul(tau, acc);
    w = make_double2(-w.x, -w.y);
#pragma unroll 4
    for (int r = r0; r < m; r += STEP)
      if (r > k) u[r] = cfma(w, v[r], u[r]);
  }
  for (int r = first; r < m; r += STEP) out[r] = u[r];
}

// WIDE: 8 warps a block, for a batch that holds such matrices (the others take four of the warps).
template <bool WIDE>
__global__ void k_backtransform(const __grid_constant__ EigBatch b, int stride, int use_z2) {
  extern __shared__ double2 bts_sh[];
  const EigMat& M = b.a[blockIdx.y];
  const int m = M.m, K = M.K, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (WIDE && m > BTS_WARP) {
    __shared__ double2 slots[16];  // two sets of a sum per warp
    const int nv = btw_vectors(m), nw = 8 / nv, vec = warp / nw, part = warp - vec * nw, j = blockIdx.x * nv + vec;
    if (j >= K) return;
    const double* Z = (use_z2 ? M.Z2 : M.Z) + j;
    double2* u = bts_sh + (size_t)vec * ((m + 31) & ~31);
    double2* out = M.U + (size_t)j * m;
    if (nw == 4) btw_vector<4>(M, Z, u, out, slots + 4 * vec, vec, part);
    else btw_vector<8>(M, Z, u, out, slots, vec, part);
    return;
  }
  const int j = blockIdx.x * 4 + warp;
  if (j >= K || (WIDE && warp >= 4)) return;
  const double* Z = (use_z2 ? M.Z2 : M.Z) + j;
  double2* out = M.U + (size_t)j * m;
  constexpr int R = 8;
  if (m <= 32 * R) {  // the vector in registers, the next reflector's entries on their way during a reflector
    double2 u[R], vn[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int r = 32 * q + lane;
      u[q] = make_double2(r < m ? Z[(size_t)r * K] : 0.0, 0.0);
      vn[q] = (r > m - 2 && r < m && m > 1) ? M.H[(size_t)(m - 2) * m + r] : make_double2(0.0, 0.0);
    }
    for (int k = m - 2; k >= 0; --k) {
      const double2 tau = M.tau[k];
      double2 v[R];
#pragma unroll
      for (int q = 0; q < R; ++q) {
        v[q] = vn[q];
        const int r = 32 * q + lane;
        if (32 * q + 31 >= k) vn[q] = (k > 0 && r > k - 1 && r < m) ? M.H[(size_t)(k - 1) * m + r] : make_double2(0.0, 0.0);
      }
      if (tau.x == 0.0 && tau.y == 0.0) continue;
      double2 a0 = make_double2(0.0, 0.0), a1 = a0;
#pragma unroll
      for (int q = 0; q < R; q += 2) {
        if (32 * q + 31 > k && 32 * q < m) a0 = cfma_conj(v[q], u[q], a0);
        if (32 * q + 63 > k && 32 * q + 32 < m) a1 = cfma_conj(v[q + 1], u[q + 1], a1);
      }
      double2 w = cmul(tau, warp_sum2(cadd(a0, a1)));
      w = make_double2(-w.x, -w.y);
#pragma unroll
      for (int q = 0; q < R; ++q)
        if (32 * q + 31 > k && 32 * q < m) u[q] = cfma(w, v[q], u[q]);
    }
#pragma unroll
    for (int q = 0; q < R; ++q)
      if (32 * q + lane < m) out[32 * q + lane] = u[q];
    return;
  }
  double2* u = bts_sh + (size_t)warp * stride;
  for (int r = lane; r < m; r += 32) u[r] = make_double2(Z[(size_t)r * K], 0.0);
  for (int k = m - 2; k >= 0; --k) {
    const double2 tau = M.tau[k];
    if (tau.x == 0.0 && tau.y == 0.0) continue;
    const double2* v = M.H + (size_t)k * m;
    const int r0 = ((k + 1) & ~31) + lane;  // rows keep their lane
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int r = r0; r < m; r += 32)
      if (r > k) acc = cfma_conj(v[r], u[r], acc);
    double2 w = cmul(tau, warp_sum2(acc));
    w = make_double2(-w.x, -w.y);
#pragma unroll 4
    for (int r = r0; r < m; r += 32)
      if (r > k) u[r] = cfma(w, v[r], u[r]);
  }
  for (int r = lane; r < m; r += 32) out[r] = u[r];
}

// ---- blocked back-transformation (tensor-core paths) ----------------------------------------
// U <- Q Z with Q = H(0) H(1) ... H(m-2) is applied as blocks of BT reflectors,
// Q_p = H(k0) ... H(k0+BT-1) = I - V T V^+ (compact WY form, T upper triangular:
// T[i][i] = tau_i, T[0:i, i] = -tau_i T[0:i, 0:i] (V^+ V)[0:i, i]), last block first:
// U^T <- U^T - V T (V^+ U^T), i.e. three matrix products per block on the rows of U.
// V is read from where the reduction left it: row k of H is v_k, once its part up to the diagonal is
// cleared.  V^+ V and T do not depend on U, so those of all blocks of all matrices are formed at
// once (one block each), and only the three products run one block after the other.
// Measured against T of one block after the other on the chain (165 us each): eigenvectors of 4 matrices of
// 1024 (K = 256) 14.8 -> 10.1 ms, of the chi = 1024, d = 5 charge blocks of 7 triples 11.8 -> 9.7 ms.
constexpr int BT = 64;  // reflectors per block

__host__ __device__ size_t td_panel_size(int m);  // panel arrays of the reduction (complex elements)
__host__ __device__ __forceinline__ int bt_blocks(int m) { return (m - 1 + BT - 1) / BT; }
// After the panel arrays: conj(V^+ V) of every block, then T^T of every block, then S and S T^T (m x BT each).
__host__ __device__ __forceinline__ double2* bt_G(const EigMat& M, int p) {
  return M.pan + td_panel_size(M.m) + (size_t)p * BT * BT;
}
__host__ __device__ __forceinline__ double2* bt_Tt(const EigMat& M, int p) { return bt_G(M, bt_blocks(M.m) + p); }
__host__ __device__ __forceinline__ double2* bt_S(const EigMat& M) { return bt_G(M, 2 * bt_blocks(M.m)); }

// H[k][c] = 0 for c <= k: what is left of row k is v_k.
__global__ void k_bt_clear(const __grid_constant__ EigBatch b) {
  const EigMat& M = b.a[blockIdx.y];
  if (M.K == 0) return;
  for (int k = blockIdx.x; k < M.m; k += gridDim.x)
    for (int c = threadIdx.x; c <= k; c += blockDim.x) M.H[(size_t)k * M.m + c] = make_double2(0.0, 0.0);
}

// T of block p from conj(V^+ V) and tau (one block per matrix and p; four threads per
// row of T share each column's sum), written transposed.
__global__ void __launch_bounds__(4 * BT) k_bt_T(const __grid_constant__ EigBatch b) {
  const EigMat& M = b.a[blockIdx.y];
  const int m = M.m, p = blockIdx.x, k0 = p * BT;
  if (M.K == 0 || k0 >= m - 1) return;
  const int nb = min(BT, m - 1 - k0);
  extern __shared__ double2 Tsh[];  // BT x (BT + 1)
  const double2* G = bt_G(M, p);    // nb x nb
  for (int idx = threadIdx.x; idx < BT * (BT + 1); idx += blockDim.x) Tsh[idx] = make_double2(0.0, 0.0);
  __syncthreads();
  const int l = threadIdx.x >> 2, part = threadIdx.x & 3;
  for (int i = 0; i < nb; ++i) {
    const double2 ti = M.tau[k0 + i];
    double2 acc = make_double2(0.0, 0.0);
    if (l < i)
      for (int q = l + part; q < i; q += 4) acc = cfma(Tsh[l * (BT + 1) + q], G[i * nb + q], acc);
    if ((threadIdx.x & ~31) < 4 * i) {  // warps without a row of this column add nothing
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 1);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 1);
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 2);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 2);
      if (part == 0 && l < i)
        Tsh[l * (BT + 1) + i] = make_double2(-(ti.x * acc.x - ti.y * acc.y), -(ti.x * acc.y + ti.y * acc.x));
    }
    if (part == 0 && l == i) Tsh[l * (BT + 1) + i] = ti;
    __syncthreads();
  }
  double2* Tt = bt_Tt(M, p);
  for (int idx = threadIdx.x; idx < nb * nb; idx += blockDim.x) {
    const int r = idx / nb, c = idx - r * nb;  // Tt[r][c] = T[c][r]
    Tt[idx] = Tsh[c * (BT + 1) + r];
  }
}

// ---- blocked Householder reduction ---------------------------------------------------------
// Panels of TD_NB columns.  Within a panel the trailing matrix is left as it was at the panel
// start; each column's Hermitian product runs on that stored upper triangle and is corrected with
// the panel's earlier (v_i, w_i).  After the panel the trailing matrix takes the whole
// rank-2*TD_NB update as one Hermitian matrix product (tensor cores in the mixed path).
//
// Bound: the FP64 pipe (a warp-wide FP64 instruction every 16 to 19 clocks per SM, however many
// lanes are active) and, for few or small matrices, the latency of a column.  So a column takes
// two grid barriers (1.4 us each), every phase is cut into pieces of 64 to 128 FP64 warp
// instructions spread over all SMs, and nothing but the two products per stored element runs at
// n^2: a tile's row sums come from a transposed read of shared memory instead of shuffled
// reductions, magnitudes are compared as integers, and the reflector's scalars (norm, divisions)
// are one warp's work beside the product, which therefore runs on the unnormalised row.
// Against three barriers per column with a reflector per block, shuffled row sums and 32 x 256 slabs,
// the reduction of 4 matrices of 1024 (with its trailing updates and tail) takes 26 instead of 59 ms,
// of 4 matrices of 244 3.5 instead of 10.8 ms, of the 94 charge blocks (up to 600) of a chi = 1024, d = 5
// cut of 7 triples 16.5 instead of 38 ms.  A column of 4 x 244 spends 9k clocks in phase A, 12k in phase B and
// 8k in the barriers.

constexpr int TD_THREADS = 256;
constexpr int TD_WARPS = TD_THREADS / 32;
constexpr int TD_NB = 32;      // columns per panel of the blocked reduction
// A column whose largest off-diagonal entry lies below 2^-340 is taken as already
// reduced (tau = 0): with a trace of at least 2^-200 (k_trace) such entries are 2^-140 of it, far
// below the matrix's rounding.  They do arise, as rounding noise that each Gram product
// squares, in empty regions of the chain, and the squares and cubes that a column's scalars
// hold would leave the range of a double (NaN below 2^-512).
constexpr int REFL_FLUSH_EXP = 340;
// The last TD_TAIL or fewer columns of every matrix are reduced by one block per
// matrix with the trailing matrix in shared memory (k_tridiag_tail): there the
// cooperative kernel would pay two grid barriers per column for very little work.
// A matrix takes part in the panels k0 < tail_start(m) (a multiple of TD_NB), so the
// split depends on its own size only and each result is independent of its batch.
constexpr int TD_TAIL = 64;
__host__ __device__ __forceinline__ int tail_start(int m) {
  return m <= TD_TAIL ? 0 : ((m - TD_TAIL + TD_NB - 1) / TD_NB) * TD_NB;
}


// Grid barrier for a cooperative launch.  st = {arrival count, unused, error}.
// Every block adds 1 to the count with a fire-and-forget release reduction
// (no serialised round trips) and polls it with acquire loads until it reaches
// the next multiple of the grid size (`target`, advanced by each call).  Waits
// at most `limit` clocks (2e9, ~1 s, unless the handle's "wait_limit_clocks"
// says otherwise); on timeout it records the failure in st[2] and returns
// false so every block can leave.  The count starts at 0 per launch.
// `beside` is run by warp 1 while thread 0 waits (it must not touch what other blocks write).
template <class F>
__device__ bool grid_sync(unsigned int* st, unsigned int& target, long long limit, F beside) {
  __shared__ int ok_sh;
  __syncthreads();
  target += gridDim.x;
  if (threadIdx.x == 0) {
    volatile unsigned int* verr = st + 2;
    int ok = 1;
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(st) : "memory");
    const long long t0 = clock64();
    while (true) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(st) : "memory");
      if ((int)(v - target) >= 0) break;
      if (*verr) { ok = 0; break; }
      if (clock64() - t0 > limit) { atomicExch(st + 2, 1u); ok = 0; break; }
    }
    __threadfence();
    ok_sh = ok && (*verr == 0);
  } else if ((threadIdx.x >> 5) == 1) {
    beside();
  }
  __syncthreads();
  return ok_sh != 0;
}

// Panel arrays of a matrix, in this order:
//   VW[r] = (v_0..v_{NB-1}, w_0..w_{NB-1})(r) and WV[r] the same with the halves swapped (the second
//   operand of the trailing update); the partial dots of the panel corrections (TD_DOTS x 2 NB); the
//   partial sums of the Hermitian product, per strip of 32 columns from row blocks (hc) and from
//   tiles to its right (hr); the partials of u^+ A u, one per tile; the column's scalars.
// The piece sizes (as shifts) follow the trailing size n only, never the batch: the sums keep their order.
__host__ __device__ __forceinline__ int td_rows(int n) { return n <= 256 ? 3 : n <= 2048 ? 4 : 5; }   // rows per tile
__host__ __device__ __forceinline__ int td_cols(int n) { return n <= 256 ? 3 : n <= 1024 ? 4 : 5; }   // columns per phase-B piece
__host__ __device__ __forceinline__ int td_dot(int n) { return n <= 256 ? 4 : n <= 512 ? 5 : 6; }     // rows per partial dot
constexpr int TD_DOTS = 200;  // partial dots: at most ceil(12288 / 64) = 192
// Strips and row blocks that a trailing set of n can touch (its start is not aligned to them).
__host__ __device__ __forceinline__ size_t td_strips(int n) { return (size_t)(n + 31) / 32 + 1; }
__host__ __device__ __forceinline__ size_t td_blocks(int n) { return (size_t)(n >> td_rows(n)) + 2; }
__host__ __device__ __forceinline__ size_t td_tiles(int n) { return td_strips(n) * td_blocks(n); }
__host__ __device__ inline size_t td_max3(size_t a, size_t b, size_t c) { return a > b ? (a > c ? a : c) : (b > c ? b : c); }
__host__ __device__ inline size_t td_hc_tiles(int m) {  // the largest of the three piece sizes' needs
  return td_max3(td_tiles(m), td_tiles(m < 2048 ? m : 2048), td_tiles(m < 256 ? m : 256));
}
__host__ __device__ __forceinline__ size_t td_hr_tiles(int m) { return td_strips(m) * td_strips(m); }
__host__ __device__ size_t td_panel_size(int m) {
  return (size_t)m * 4 * TD_NB + (size_t)TD_DOTS * 2 * TD_NB + 32 * (td_hc_tiles(m) + td_hr_tiles(m)) +
         (td_hc_tiles(m) + 1) / 2 + 8;  // the host lays td_hr, td_q and td_sc out the same way
}
__device__ __forceinline__ double2* pan_vw(const EigMat& M) { return M.pan; }
__device__ __forceinline__ double2* pan_wv(const EigMat& M) { return M.pan + (size_t)M.m * 2 * TD_NB; }
__device__ __forceinline__ double2* pan_xy(const EigMat& M) { return M.pan + (size_t)M.m * 4 * TD_NB; }
__device__ __forceinline__ double2* pan_hc(const EigMat& M) { return pan_xy(M) + (size_t)TD_DOTS * 2 * TD_NB; }
__device__ __forceinline__ double2* pan_hr(const EigMat& M) { return M.td_hr; }
__device__ __forceinline__ double* pan_q(const EigMat& M) { return M.td_q; }
__device__ __forceinline__ double2* pan_scal(const EigMat& M) { return M.td_sc; }  // [0] sc, [1] (A(k+1, k+1), 0)

// What a column's pieces are, from m and k alone.
struct TdGeo {
  int m, k, n;          // trailing set: indices k+1 .. m-1, n of them
  int rows, cols, dot;  // piece sizes (shifts)
  int s0, ns;           // first strip, strips
  int b0, nb;           // first row block, row blocks
  int g0, ng;           // first phase-B piece, pieces
  int nd;               // partial dots
  __device__ TdGeo(int m_, int k_) : m(m_), k(k_), n(m_ - k_ - 1) {
    rows = td_rows(n); cols = td_cols(n); dot = td_dot(n);
    s0 = (k + 1) >> 5; ns = ((m - 1) >> 5) - s0 + 1;
    b0 = (k + 1) >> rows; nb = ((m - 1) >> rows) - b0 + 1;
    g0 = (k + 1) >> cols; ng = ((m - 1) >> cols) - g0 + 1;
    nd = (n + (1 << dot) - 1) >> dot;
  }
  // tiles: row block b of strip S meets the strips S .. end; counted as if the last strip were full
  __device__ int per() const { return 32 >> rows; }
  __device__ int first_blocks() const { return (s0 + 1) * per() - b0; }  // row blocks of the first strip
  __device__ int tiles() const { return first_blocks() * ns + per() * (ns * (ns - 1) / 2); }
  __device__ int items_a(int j) const { return 1 + (j > 0 ? 2 * nd : 0) + tiles(); }
  // tile t -> row block b (relative to b0) and strip T (relative to s0)
  __device__ void tile(int t, int& b, int& T) const {
    const int f = first_blocks() * ns;
    if (t < f) {
      b = t / ns;
      T = t - b * ns;
      return;
    }
    t -= f;
    const int last = per() * (ns * (ns - 1) / 2) - 1 - t;  // counted from the end: strips of 1, 2, ... tiles per row block
    int D = (int)((sqrtf(8.0f * (float)(last >> (5 - rows)) + 1.0f) + 1.0f) * 0.5f);
    while (per() * (D * (D - 1) / 2) > last) --D;
    while (per() * (D * (D + 1) / 2) <= last) ++D;
    const int rem = last - per() * (D * (D - 1) / 2);  // within the strip that has D strips from itself on
    const int sb = rem / D;
    b = first_blocks() + (ns - 1 - D) * per() + (per() - 1 - sb);
    T = ns - 1 - (rem - sb * D);
  }
};

// Exponent field of the larger of |re|, |im| (2047: not finite), read as integers.
__device__ __forceinline__ int expo2(double2 x) {
  return max((__double2hiint(x.x) >> 20) & 0x7FF, (__double2hiint(x.y) >> 20) & 0x7FF);
}

// Partial norm of row k over one piece: lanes hold its entries (zero where there is none; `in`: counted
// in the sum, i.e. not the first entry).  {sum |x|^2, largest exponent field}: a row that is not
// flushed has its largest entry within 2^-340 .. 2^200, so the squares that count stay in range.
__device__ __forceinline__ void put_norm(const EigMat& M, int g, double2 x, bool in) {
  const int ef = __reduce_max_sync(0xffffffffu, expo2(x));
  double s = 0.0;
  if (ef != 0) {
    s = in ? fma(x.x, x.x, x.y * x.y) : 0.0;
    s = warp_sum(s);
  }
  if ((threadIdx.x & 31) == 0) M.part[g] = make_double2(s, __longlong_as_double(ef));
}

// The scalars of column k's reflector from the partial norms of row k (one warp):
// H(k) = I - tau v v^+, v = e_0 + sc (0, conj(x_1), conj(x_2), ...).
__device__ void td_scalars(const EigMat& M, int k) {
  const int m = M.m, lane = threadIdx.x & 31;
  const TdGeo P(m, k - 1);  // the pieces that wrote the partials of row k
  const double2* row = M.H + (size_t)k * m;
  const double2 x0 = row[k + 1];
  const double dk = row[k].x, a00 = M.H[(size_t)(k + 1) * m + k + 1].x;
  int emax = 0;
  double s = 0.0;
  for (int g = lane; g < P.ng; g += 32) {
    const double2 t = M.part[g];
    emax = max(emax, (int)__double_as_longlong(t.y));
    s += t.x;
  }
  emax = __reduce_max_sync(0xffffffffu, emax);
  const double xnorm2 = warp_sum(s);
  const bool flush = emax < 1023 - REFL_FLUSH_EXP;  // every entry below 2^-340
  const double ar = x0.x, ai = -x0.y;
  double beta = x0.x;
  double2 tau = make_double2(0.0, 0.0), sc = tau;
  if (!flush && !(xnorm2 == 0.0 && ai == 0.0)) {
    const double bs = -copysign(sqrt(ar * ar + ai * ai + xnorm2), ar), zr = ar - bs;
    // lane 0: 1 / beta, lane 1: 1 / |alpha - beta|^2
    const double r = 1.0 / ((lane & 1) ? fma(zr, zr, ai * ai) : bs);
    const double inv = __shfl_sync(0xffffffffu, r, 0), iden = __shfl_sync(0xffffffffu, r, 1);
    tau = make_double2(-zr * inv, -ai * inv);
    sc = make_double2(zr * iden, -ai * iden);
    beta = bs;
  }
  if (lane == 0) {
    M.d[k] = dk;
    M.e[k] = beta;
    M.tau[k] = tau;
    pan_scal(M)[0] = sc;
    pan_scal(M)[1] = make_double2(a00, 0.0);
  }
}

// u_r = conj(x_r) of row k for r > k+1, 0 for r = k+1 (the reflector's unit entry is added later).
__device__ __forceinline__ double2 td_u(const EigMat& M, int k, int r) {
  return (r > k + 1 && r < M.m) ? cconj(M.H[(size_t)k * M.m + r]) : make_double2(0.0, 0.0);
}

// One tile of hraw = A u (one warp): row block b against strip T.  The lanes hold the strip's
// columns: each row of A is read once, gives its term of the column sums conj(A[r][c]) u_r from
// registers and, off the diagonal, the row sums A[r][c] u_c through a transposed read of shared
// memory (st: 16 x 33, us: 64).  Diagonal tiles need only the column sums.
template <int SUB>
__device__ void td_tile(const EigMat& M, const TdGeo& G, int t, double2* st, double2* us) {
  const int lane = threadIdx.x & 31, m = G.m, k = G.k;
  int b, T;
  G.tile(t, b, T);
  const int r0 = (G.b0 + b) << G.rows;
  if (r0 >= m) {  // the last strip's missing row blocks
    if (lane == 0) pan_q(M)[t] = 0.0;
    return;
  }
  const int S = r0 / 32 - G.s0;
  const bool diag = (S == T);
  const int c = 32 * (G.s0 + T) + lane;
  const double2 uc = td_u(M, k, c), ur = td_u(M, k, r0 + lane);  // (lanes beyond the row block: not used)
  us[lane] = uc;
  us[32 + lane] = ur;
  double2 acc = make_double2(0.0, 0.0);
  double2* hr = pan_hr(M) + ((size_t)S * G.ns + T) * 32;
  const bool okc = c < m && c > k;
  __syncwarp();
  for (int sub = r0; sub < r0 + (1 << G.rows); sub += SUB) {
    if (sub + SUB <= k + 1 || sub >= m) continue;
#pragma unroll
    for (int h = 0; h < SUB; h += 8) {
      double2 a[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = sub + h + u;
        a[u] = (okc && r > k && r < m) ? M.H[(size_t)r * m + c] : make_double2(0.0, 0.0);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (!diag) st[(h + u) * 33 + lane] = a[u];
        if (sub + h + u > k + 1) acc = cfma_conj(a[u], us[32 + sub - r0 + h + u], acc);  // (rows beyond m hold zeros)
      }
    }
    if (!diag) {
      __syncwarp();
      const int row = lane & (SUB - 1), c0 = (lane / SUB) * SUB;
      double2 ra = make_double2(0.0, 0.0);
#pragma unroll 4
      for (int q = 0; q < SUB; ++q) ra = cfma(st[row * 33 + c0 + q], us[c0 + q], ra);
#pragma unroll
      for (int o = SUB; o < 32; o <<= 1) {
        ra.x += __shfl_xor_sync(0xffffffffu, ra.x, o);
        ra.y += __shfl_xor_sync(0xffffffffu, ra.y, o);
      }
      if (lane < SUB && sub + lane > k && sub + lane < m) hr[(sub + lane) & 31] = ra;
      __syncwarp();
    }
  }
  pan_hc(M)[((size_t)T * G.nb + b) * 32 + lane] = acc;
  // u^+ A u: the two halves of an off-diagonal tile are conjugate
  double q = fma(uc.x, acc.x, uc.y * acc.y);
  q = warp_sum(q);
  if (lane == 0) pan_q(M)[t] = diag ? q : 2.0 * q;
}

// Partial dots of the panel corrections over the rows of piece p (one warp, a lane per i < j):
// which = 0: v_i^+ u, 1: w_i^+ u.
__device__ void td_dots(const EigMat& M, const TdGeo& G, int j, int p, int which) {
  const int lane = threadIdx.x & 31;
  if (lane >= j) return;
  const int r0 = max(G.k + 2, G.k + 1 + (p << G.dot)), r1 = min(G.m, G.k + 1 + ((p + 1) << G.dot));
  const double2* col = pan_vw(M) + which * TD_NB + lane;
  const double2* x = M.H + (size_t)G.k * G.m;
  double2 t = make_double2(0.0, 0.0);
#pragma unroll 8
  for (int r = r0; r < r1; ++r) t = cfma_conj(col[(size_t)r * 2 * TD_NB], cconj(x[r]), t);
  pan_xy(M)[(size_t)p * 2 * TD_NB + which * TD_NB + lane] = t;
}

// The matrix that holds item `it` of a batch with prefix sums pre[0..n].
__device__ __forceinline__ int td_find(const int* pre, int n, int it) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= it) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Item counts of every matrix as prefix sums (one warp; a lane takes EIG_MAXP / 32 neighbours).
template <class F>
__device__ __forceinline__ void td_prefix(int* pre, int n, F count) {
  constexpr int W = EIG_MAXP / 32;
  const int lane = threadIdx.x & 31;
  int v[W], sum = 0;
#pragma unroll
  for (int q = 0; q < W; ++q) {
    const int i = lane * W + q;
    v[q] = i < n ? count(i) : 0;
    sum += v[q];
  }
  int ex = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, ex, o);
    if (lane >= o) ex += t;
  }
  ex -= sum;
#pragma unroll
  for (int q = 0; q < W; ++q) {
    const int i = lane * W + q;
    if (i <= n) pre[i] = ex;
    ex += v[q];
  }
  if (lane == 31 && n == EIG_MAXP) pre[n] = ex;
}

// Blocked Householder tridiagonalisation, one panel of columns [k0, k1) per
// cooperative launch (the trailing matrix from k0 on is current when it starts).
// Column k (panel index j) is reduced against A(k) = A(k0) - sum_{i<j} (v_i w_i^+ +
// w_i v_i^+) without forming A(k).  Row k is A(k)'s when its turn comes.
//   phase A (warps): the reflector's scalars; partial dots v_i^+ u, w_i^+ u; tiles of
//           hraw = A(k0) u and of u^+ A(k0) u, with u = conj(row k) unnormalised, u(k+1) = 0.
//   phase B (blocks, pieces of td_cols columns): v = e_0 + sc u, h = A(k0) v = A(k0) e_0 + sc hraw,
//           p = tau (h - sum_i (v_i (w_i^+ v) + w_i (v_i^+ v))), alpha = -|tau|^2 v^+ A(k) v / 2 with
//           v^+ A(k) v = v^+ h - 2 Re sum_i conj(v_i^+ v) (w_i^+ v) (so no further barrier is
//           needed for it), w = p + alpha v; row k+1 brought to A(k+1), and its partial norms.
// After the panel, the caller applies A -= V W^+ + W V^+ to rows and columns >= k1
// as one Hermitian rank-2*NB matrix product.
constexpr int TD_ST = 16 * 33 + 64;  // shared memory of one warp's tile (complex)
constexpr int TD_SMEM = TD_WARPS * TD_ST * (int)sizeof(double2);
__global__ void __launch_bounds__(TD_THREADS, 2) k_tridiag_panel(const __grid_constant__ EigBatch b, int k0, int k1) {
  extern __shared__ double2 td_sh[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ int pre_a[EIG_MAXP + 1], pre_b[EIG_MAXP + 1];  // items before each matrix, phase A / B
  __shared__ double2 xy_sh[2 * TD_NB];                      // Y_i = v_i^+ v, then X_i = w_i^+ v
  __shared__ double2 vk_sh[2 * TD_NB];                      // v_i(k+1), then w_i(k+1)
  __shared__ double2 pv_sh[TD_WARPS][32], rv_sh[TD_WARPS][32];
  __shared__ double q_sh[4];
  __shared__ double2 h0_sh, p0_sh;
  __shared__ double alpha_sh;
  unsigned int target = 0;  // barrier count expected at the next grid_sync
  auto items_a = [&](int k) {
    td_prefix(pre_a, b.n, [&](int i) { return k0 < tail_start(b.a[i].m) ? TdGeo(b.a[i].m, k).items_a(k - k0) : 0; });
  };
  auto items_b = [&](int k) {
    td_prefix(pre_b, b.n, [&](int i) { return k0 < tail_start(b.a[i].m) ? TdGeo(b.a[i].m, k).ng : 0; });
  };
  // the partial norms of the panel's first row
  if (warp == 0) items_b(k0 - 1);
  __syncthreads();
  for (int it = warp * gridDim.x + blockIdx.x; it < pre_b[b.n]; it += TD_WARPS * gridDim.x) {
    const int mi = td_find(pre_b, b.n, it);
    const EigMat& M = b.a[mi];
    const TdGeo P(M.m, k0 - 1);
    const int g = it - pre_b[mi], c = ((P.g0 + g) << P.cols) + lane;
    const bool ok = lane < (1 << P.cols) && c < M.m && c > k0;
    put_norm(M, g, ok ? M.H[(size_t)k0 * M.m + c] : make_double2(0.0, 0.0), c > k0 + 1);
  }
  if (!grid_sync(b.bar, target, b.wait_clocks, [&] { items_a(k0); })) return;
  for (int k = k0; k < k1; ++k) {
    const int j = k - k0;
    // ---- phase A
    for (int it = warp * gridDim.x + blockIdx.x; it < pre_a[b.n]; it += TD_WARPS * gridDim.x) {
      const int mi = td_find(pre_a, b.n, it);
      const EigMat& M = b.a[mi];
      const TdGeo G(M.m, k);
      int rem = it - pre_a[mi];
      if (rem == 0) {
        td_scalars(M, k);
        continue;
      }
      rem -= 1;
      const int nd2 = j > 0 ? 2 * G.nd : 0;
      if (rem < nd2) {
        td_dots(M, G, j, rem >> 1, rem & 1);
        __syncwarp();
        continue;
      }
      double2* st = td_sh + warp * TD_ST;
      if (G.rows == 3) td_tile<8>(M, G, rem - nd2, st, st + 16 * 33);
      else td_tile<16>(M, G, rem - nd2, st, st + 16 * 33);
      __syncwarp();
    }
    if (!grid_sync(b.bar, target, b.wait_clocks, [&] { items_b(k); })) return;
    // ---- phase B
    for (int it = blockIdx.x; it < pre_b[b.n]; it += gridDim.x) {
      const int mi = td_find(pre_b, b.n, it);
      const EigMat& M = b.a[mi];
      const TdGeo G(M.m, k);
      const int m = M.m, g = it - pre_b[mi];
      const bool nextrow = (k + 1 < k1);
      const double2 sc = pan_scal(M)[0], tau = M.tau[k];
      const int nc_ = 1 << G.cols, grp = 32 >> G.cols;  // columns of the piece, lane groups
      const int cl = lane & (nc_ - 1), c = ((G.g0 + g) << G.cols) + cl;
      const bool ok = c > k && c < m;
      double2 h = make_double2(0.0, 0.0);
      if (warp < 2) {  // X_i = w_i^+ v, Y_i = v_i^+ v over the whole trailing set
        const int v = threadIdx.x;
        double2 x = make_double2(0.0, 0.0), vk = x;
        if ((v & (TD_NB - 1)) < j) {
          vk = pan_vw(M)[(size_t)(k + 1) * 2 * TD_NB + v];
          const double2* xy = pan_xy(M) + v;
          double2 t = make_double2(0.0, 0.0);
#pragma unroll 8
          for (int p = 0; p < G.nd; ++p) t = cadd(t, xy[(size_t)p * 2 * TD_NB]);
          x = cfma(sc, t, cconj(vk));
        }
        xy_sh[v] = x;
        vk_sh[v] = vk;
      } else {
        // hraw of the piece's columns: row blocks down to the strip's own, then the strips to its right
        const int slots = (TD_WARPS - 2) * grp, slot = (warp - 2) * grp + (lane >> G.cols);
        if (ok) {
          const int S = (c >> 5) - G.s0, e = c & 31, n1 = min(G.nb, G.first_blocks() + S * G.per());
          const double2* hc = pan_hc(M) + (size_t)S * G.nb * 32 + e;
          const double2* hr = pan_hr(M) + (size_t)S * G.ns * 32 + e;
#pragma unroll 4
          for (int i = slot; i < n1; i += slots) h = cadd(h, hc[(size_t)i * 32]);
#pragma unroll 4
          for (int T = S + 1 + slot; T < G.ns; T += slots) h = cadd(h, hr[(size_t)T * 32]);
          h = cmul(sc, h);
        }
        if (warp < 6) {  // u^+ A u
          double q = 0.0;
          const int nt = G.tiles();
#pragma unroll 4
          for (int t = (warp - 2) * 32 + lane; t < nt; t += 128) q += pan_q(M)[t];
          q = warp_sum(q);
          if (lane == 0) q_sh[warp - 2] = q;
        } else if (warp == 6) {  // hraw(k+1)
          const int e = (k + 1) & 31, nc = min(G.first_blocks(), G.nb);
          double2 t = make_double2(0.0, 0.0);
          for (int i = lane; i < nc + G.ns - 1; i += 32)
            t = cadd(t, i < nc ? pan_hc(M)[(size_t)i * 32 + e] : pan_hr(M)[(size_t)(i - nc + 1) * 32 + e]);
          t = warp_sum2(t);
          if (lane == 0) h0_sh = t;
        }
      }
      __syncthreads();
      double2 a = make_double2(0.0, 0.0), v = a;
      if (warp == 0) {  // alpha, and v of the piece
        if (ok && lane < nc_) {
          a = M.H[(size_t)(k + 1) * m + c];  // A(k0)(k+1, c): its conjugate is (A e_0)(c)
          v = M.H[(size_t)k * m + c];
        }
        const double2 X = xy_sh[TD_NB + lane], Y = xy_sh[lane], h0 = h0_sh;
        double gx = fma(Y.x, X.x, Y.y * X.y);
        if (j > 0) gx = warp_sum(gx);
        const double q = (q_sh[0] + q_sh[1]) + (q_sh[2] + q_sh[3]);
        // v^+ A(k) v = A00 + 2 Re(sc hraw_0) + |sc|^2 u^+ A u - 2 Re sum_i conj(Y_i) X_i
        const double s0 = fma(sc.x, h0.x, -sc.y * h0.y);
        const double va = fma(fma(sc.x, sc.x, sc.y * sc.y), q, fma(2.0, s0 - gx, pan_scal(M)[1].x));
        if (lane == 0) alpha_sh = -0.5 * fma(tau.x, tau.x, tau.y * tau.y) * va;
        v = (c == k + 1) ? make_double2(1.0, 0.0) : cmul(sc, cconj(v));
      } else if (warp == 1) {  // p(k+1), w(k+1) = p(k+1) + alpha
        const double2 X = xy_sh[TD_NB + lane], Y = xy_sh[lane], vi = vk_sh[lane], wi = vk_sh[TD_NB + lane];
        double2 c0 = cfma(wi, Y, cmul(vi, X));
        if (j > 0) c0 = warp_sum2(c0);
        const double2 h0 = cfma(sc, h0_sh, pan_scal(M)[1]);
        if (lane == 0) p0_sh = cmul(tau, csub(h0, c0));
      } else {  // - corrections of the product, and the corrections of row k+1
        const int slots = (TD_WARPS - 2) * grp, slot = (warp - 2) * grp + (lane >> G.cols);
        double2 rc = make_double2(0.0, 0.0);
        if (ok) {
          const double2* row = pan_vw(M) + (size_t)c * 2 * TD_NB;
          for (int i = slot; i < j; i += slots) {
            const double2 vc = row[i], wc = row[TD_NB + i];
            double2 X = xy_sh[TD_NB + i], Y = xy_sh[i];
            X = make_double2(-X.x, -X.y);
            Y = make_double2(-Y.x, -Y.y);
            h = cfma(vc, X, h);  // - v_i(c) (w_i^+ v) - w_i(c) (v_i^+ v)
            h = cfma(wc, Y, h);
            if (nextrow) {       // v_i(k+1) conj(w_i(c)) + w_i(k+1) conj(v_i(c))
              rc = cfma_conj(wc, vk_sh[i], rc);
              rc = cfma_conj(vc, vk_sh[TD_NB + i], rc);
            }
          }
        }
        for (int o = nc_; o < 32; o <<= 1) {
          h.x += __shfl_xor_sync(0xffffffffu, h.x, o);
          h.y += __shfl_xor_sync(0xffffffffu, h.y, o);
          if (j > 0 && nextrow) {
            rc.x += __shfl_xor_sync(0xffffffffu, rc.x, o);
            rc.y += __shfl_xor_sync(0xffffffffu, rc.y, o);
          }
        }
        if (lane < nc_) {
          pv_sh[warp][lane] = h;
          rv_sh[warp][lane] = rc;
        }
      }
      __syncthreads();
      if (warp == 1 && lane < nc_) {  // the row corrections, beside warp 0's product
        double2 rs = make_double2(0.0, 0.0);
        if (j > 0 && nextrow)
          rs = cadd(cadd(cadd(rv_sh[2][lane], rv_sh[3][lane]), cadd(rv_sh[4][lane], rv_sh[5][lane])),
                    cadd(rv_sh[6][lane], rv_sh[7][lane]));
        rv_sh[0][lane] = rs;
      }
      double2 w = make_double2(0.0, 0.0);
      if (warp == 0 && ok && lane < nc_) {
        const double2 h1 = cadd(cadd(pv_sh[2][lane], pv_sh[3][lane]), cadd(pv_sh[4][lane], pv_sh[5][lane]));
        const double2 h2 = cadd(cconj(a), cadd(pv_sh[6][lane], pv_sh[7][lane]));
        const double alpha = alpha_sh;
        w = cmul(tau, cadd(h1, h2));
        w = make_double2(fma(alpha, v.x, w.x), fma(alpha, v.y, w.y));
        double2* VW = pan_vw(M) + (size_t)c * 2 * TD_NB;
        double2* WV = pan_wv(M) + (size_t)c * 2 * TD_NB;
        VW[j] = v;
        VW[TD_NB + j] = w;
        WV[j] = w;
        WV[TD_NB + j] = v;
        M.H[(size_t)k * m + c] = v;
      }
      __syncthreads();
      if (warp == 0 && nextrow) {  // row k+1 of A(k+1) = A(k0) - corrections - conj(w) - w(k+1) conj(v)
        double2 x = make_double2(0.0, 0.0);
        if (ok && lane < nc_) {
          a = csub(csub(a, rv_sh[0][lane]), cconj(w));
          x = cfma_conj(v, make_double2(-p0_sh.x - alpha_sh, -p0_sh.y), a);
          M.H[(size_t)(k + 1) * m + c] = x;
        }
        const bool off = c > k + 1 && lane < nc_;  // the diagonal is not part of the next reflector
        put_norm(M, g, off ? x : make_double2(0.0, 0.0), c > k + 2);
      }
      if (it + (int)gridDim.x < pre_b[b.n]) __syncthreads();  // the shared arrays are free for the next piece
    }
    if (k + 1 < k1)
      if (!grid_sync(b.bar, target, b.wait_clocks, [&] { items_a(k + 1); })) return;
  }
}

// The columns [tail_start(m), m) of one matrix per block, unblocked, with the
// trailing matrix (n <= TD_TAIL, current when the kernel starts) in shared memory
// as a full Hermitian matrix.  The reflectors are those of the panel kernel, stored the same way
// in the rows of H; each column then applies A <- A - v w^+ - w v^+ with p = tau A v,
// w = p - (|tau|^2 v^+ A v / 2) v.  One fixed order per reduction.
// Bound: one SM's FP64 pipe (8 n^2 / 32 warp instructions a column: the product, and the update of one
// triangle, mirrored) and the chain from a row to its w.  The reflector's scalars are a ninth warp's
// work beside the product, which runs on the unnormalised row as in the panel kernel.
// Measured against 8 + 8 instructions per element of the full square and block-wide reductions: the last 64
// columns of 4 matrices 0.84 -> 0.40 ms, whole matrices of 4 to 24 128 -> 68 us.
constexpr int TL_LD = TD_TAIL + 1;
constexpr int TL_WARPS = 8;                       // warps of the product and the update
constexpr int TL_THREADS = 32 * (TL_WARPS + 1);
__global__ void __launch_bounds__(TL_THREADS) k_tridiag_tail(const __grid_constant__ EigBatch b) {
  extern __shared__ double2 tl_sh[];
  double2* As = tl_sh;                      // TD_TAIL x TL_LD
  double2* vs = As + TD_TAIL * TL_LD;       // v of the current column
  double2* ws = vs + TD_TAIL;               // A u, then w
  __shared__ double2 sc_sh, tau_sh;
  __shared__ double q_sh[2];
  const EigMat& M = b.a[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = M.m, k0 = tail_start(m), nt = m - k0;
  if (nt <= 0) return;
  for (int r = warp; r < nt; r += TL_WARPS + 1)
    for (int c = r + lane; c < nt; c += 32) {
      const double2 x = M.H[(size_t)(k0 + r) * m + k0 + c];
      As[r * TL_LD + c] = x;
      As[c * TL_LD + r] = cconj(x);
    }
  __syncthreads();
  for (int j = 0; j + 1 < nt; ++j) {
    const int k = k0 + j, n = nt - j - 1;  // trailing indices r = 0..n-1 <-> rows/columns j+1+r
    const double2* x = As + j * TL_LD + j + 1;                // row j beyond its diagonal
    double2* At = As + (j + 1) * TL_LD + (j + 1);
    if (warp == TL_WARPS) {  // the reflector's scalars (td_scalars' arithmetic)
      const double2 xa = lane < n ? x[lane] : make_double2(0.0, 0.0);
      const double2 xb = lane + 32 < n ? x[lane + 32] : make_double2(0.0, 0.0);
      const int ef = __reduce_max_sync(0xffffffffu, max(expo2(xa), expo2(xb)));
      double s = 0.0;
      if (lane > 0) s = fma(xa.x, xa.x, xa.y * xa.y);
      s = fma(xb.x, xb.x, fma(xb.y, xb.y, s));
      const double xnorm2 = warp_sum(s);
      if (lane == 0) {
        const double ar = xa.x, ai = -xa.y;
        double beta;
        double2 tau, sc;
        if (ef < 1023 - REFL_FLUSH_EXP || (xnorm2 == 0.0 && ai == 0.0)) {
          beta = xa.x;
          tau = make_double2(0.0, 0.0);
          sc = make_double2(0.0, 0.0);
        } else {
          const double bs = -copysign(sqrt(ar * ar + ai * ai + xnorm2), ar);
          const double zr = ar - bs, inv = 1.0 / bs, iden = 1.0 / (zr * zr + ai * ai);
          tau = make_double2(-zr * inv, -ai * inv);
          sc = make_double2(zr * iden, -ai * iden);
          beta = bs;
        }
        M.d[k] = As[j * TL_LD + j].x;
        M.e[k] = beta;
        M.tau[k] = tau;
        tau_sh = tau;
        sc_sh = sc;
      }
    } else {  // A u with u = (0, conj(x_1), ...), four threads per row
      const int r = threadIdx.x >> 2, part = threadIdx.x & 3;
      if (8 * warp < n) {
        double2 acc = make_double2(0.0, 0.0);
        if (r < n)
          for (int c = 1 + part; c < n; c += 4) acc = cfma(At[r * TL_LD + c], cconj(x[c]), acc);
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 1);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 1);
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 2);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 2);
        if (part == 0 && r < n) ws[r] = acc;
      }
    }
    __syncthreads();
    if (warp < 2) {  // v, g = A v = A e_0 + sc A u, w = tau g - (|tau|^2 Re v^+ g / 2) v
      const int r = threadIdx.x;
      const double2 sc = sc_sh, tau = tau_sh;
      double2 v = make_double2(0.0, 0.0), g = v;
      if (r < n) {
        v = (r == 0) ? make_double2(1.0, 0.0) : cmul(sc, cconj(x[r]));
        g = cfma(sc, ws[r], At[r * TL_LD]);
        vs[r] = v;
        M.H[(size_t)k * m + k + 1 + r] = v;
      }
      double q = warp_sum(fma(v.x, g.x, v.y * g.y));
      if (lane == 0) q_sh[warp] = q;
      asm volatile("bar.sync 1, 64;" ::: "memory");
      const double alpha = -0.5 * fma(tau.x, tau.x, tau.y * tau.y) * (q_sh[0] + q_sh[1]);
      if (r < n) {
        const double2 w = cmul(tau, g);
        ws[r] = make_double2(fma(alpha, v.x, w.x), fma(alpha, v.y, w.y));
      }
    }
    __syncthreads();
    for (int r = warp; r < n; r += TL_WARPS + 1) {
      const double2 vr = vs[r], wr = ws[r];
      for (int c = r + lane; c < n; c += 32) {
        const double2 vc = vs[c], wc = ws[c];
        double2 a = At[r * TL_LD + c];  // - v_r conj(w_c) - w_r conj(v_c)
        a.x = fma(-vr.x, wc.x, a.x);
        a.x = fma(-vr.y, wc.y, a.x);
        a.y = fma(-vr.y, wc.x, a.y);
        a.y = fma(vr.x, wc.y, a.y);
        a.x = fma(-wr.x, vc.x, a.x);
        a.x = fma(-wr.y, vc.y, a.x);
        a.y = fma(-wr.y, vc.x, a.y);
        a.y = fma(wr.x, vc.y, a.y);
        At[r * TL_LD + c] = a;
        At[c * TL_LD + r] = cconj(a);
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    M.d[m - 1] = As[(nt - 1) * TL_LD + nt - 1].x;
    M.e[m - 1] = 0.0;
    M.tau[m - 1] = make_double2(0.0, 0.0);
  }
}

int max_m(const EigBatch& b) {
  int mm = 0;
  for (int i = 0; i < b.n; ++i) mm = std::max(mm, b.a[i].m);
  return mm;
}

}  // namespace

static_assert(sizeof(EigBatch) < 32000, "kernel parameter block too large (32 KB on sm_70 and later)");

int eig_tridiagonalize(const EigBatch& b0, bool mixed, void* const* oz_ws, int* status, cudaStream_t s) {
  if (b0.n == 0) return 0;
  EigBatch b = b0;
  b.range = mixed ? RANGE_DIGITS : RANGE_FP64;
  for (int i = 0; i < b.n; ++i) {  // where the panel arrays' sized parts start
    EigMat& M = b.a[i];
    M.td_hr = M.pan + (size_t)M.m * 4 * TD_NB + (size_t)TD_DOTS * 2 * TD_NB + 32 * td_hc_tiles(M.m);
    M.td_q = reinterpret_cast<double*>(M.td_hr + 32 * td_hr_tiles(M.m));
    M.td_sc = M.td_hr + 32 * td_hr_tiles(M.m) + (td_hc_tiles(M.m) + 1) / 2;
  }
  const int mm = max_m(b);
  static PerDevice panel_shape;  // SMs, and blocks of the panel kernel that fit one (low byte)
  const int shape = panel_shape([] {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (!allow_smem(k_tridiag_panel, TD_SMEM) ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tridiag_panel, TD_THREADS, TD_SMEM) != cudaSuccess)
      return 0;
    return sms << 8 | per_sm;
  });
  const int sms = shape >> 8, per_sm = shape & 255;
  const int grid = std::max(1, sms * std::min(per_sm, b.panel_blocks > 0 ? b.panel_blocks : 3));
  k_trace<<<dim3(TRACE_CTAS, b.n), NT, 0, s>>>(b);
  int launches = 1;
  int kend = 0;  // panels run while any matrix has columns before its tail
  for (int i = 0; i < b.n; ++i) kend = std::max(kend, tail_start(b.a[i].m));
  for (int k0 = 0; k0 < kend; k0 += TD_NB) {
    int k1 = std::min(mm, k0 + TD_NB);
    // a block per tile or piece while SMs are free: the FP64 pipe is per SM, so a tile is faster alone
    long long tiles = 0, pieces = 0;
    for (int i = 0; i < b.n; ++i) {
      if (k0 >= tail_start(b.a[i].m)) continue;
      const int n = b.a[i].m - k0 - 1;
      tiles += (long long)td_tiles(n) / 2 + 1;
      pieces += (n >> td_cols(n)) + 2;
    }
    const int gsz = (int)std::min<long long>(grid, std::max(pieces, tiles));
    cudaMemsetAsync(b.bar, 0, sizeof(unsigned int), s);  // arrival count of the grid barrier
    void* args[] = {&b, &k0, &k1};
    if (cudaLaunchCooperativeKernel((const void*)k_tridiag_panel, dim3(gsz), dim3(TD_THREADS), args, TD_SMEM,
                                    s) != cudaSuccess)
      return -1;
    ++launches;
    // trailing update A[k1:, k1:] -= V W^+ + W V^+ (Hermitian, lower tiles mirrored)
    Gemm g(true, OP_N, OP_C);
    std::vector<OzProb> oz;
    for (int i = 0; i < b.n; ++i) {
      const EigMat& M = b.a[i];
      const int n = M.m - k1;
      if (n <= 0 || k0 >= tail_start(M.m)) continue;
      double2* C = M.H + (size_t)k1 * M.m + k1;
      const double2* VW = M.pan + (size_t)k1 * 2 * TD_NB;
      const double2* WV = M.pan + (size_t)M.m * 2 * TD_NB + (size_t)k1 * 2 * TD_NB;
      if (mixed) {
        OzProb q{};
        q.a = OzOperand{VW, 2 * TD_NB, 1, nullptr, 1, 0};
        q.b = OzOperand{WV, 2 * TD_NB, 1, nullptr, 1, 1};
        q.M = q.N = n;
        q.K = 2 * TD_NB;
        q.C = C;
        q.ldc = M.m;
        q.alpha = -1.0;
        q.beta = 1;
        q.row_div = q.col_div = 1;
        q.herm = 1;
        q.ws = oz_ws[i];
        oz.push_back(q);
      } else {
        GemmProb& p = g.add(n, n, 2 * TD_NB, VW, 2 * TD_NB, WV, 2 * TD_NB, C, M.m);
        p.alpha_re = -1.0;
        p.accumulate = 1;
        p.herm = 1;
      }
    }
    launches += mixed ? oz_gemm_launch(oz, status, s) : g.launch(s);
  }
  {
    constexpr int TL_SMEM = (TD_TAIL * TL_LD + 2 * TD_TAIL) * (int)sizeof(double2);
    static PerDevice smem;
    smem([] { return allow_smem(k_tridiag_tail, TL_SMEM); });
    k_tridiag_tail<<<b.n, TL_THREADS, TL_SMEM, s>>>(b);
    ++launches;
  }
  k_sturm_prep<<<b.n, 256, 0, s>>>(b);
  return launches + 1;
}

size_t eig_panel_doubles2(int m) {
  // panel arrays, then the back-transformation's V^+ V, T^T, S and S T^T
  return td_panel_size(m) + (size_t)2 * bt_blocks(m) * BT * BT + (size_t)2 * m * BT;
}

int eig_cut_counts(const ThrCut* cuts_dev, int ncuts, cudaStream_t s) {
  if (ncuts <= 0) return 0;
  k_cut_counts<<<ncuts, 1024, 0, s>>>(cuts_dev);
  return 1;
}

int eig_bisect(const EigBatch& b, cudaStream_t s) {
  if (b.n == 0) return 0;
  int warps = 0;
  for (int i = 0; i < b.n; ++i) {
    const int per = 32 / bisect_lanes(b.a[i].kmax, b.few), km = std::min(b.a[i].kmax, b.a[i].m);
    warps = std::max(warps, (km + per - 1) / per);
  }
  if (warps == 0) return 0;
  k_bisect<<<dim3((warps + 3) / 4, b.n), 128, 0, s>>>(b);  // up to four warps per block
  return 1;
}

int eig_vectors(const EigBatch& b0, bool mixed, void* const* oz_ws, int* status, cudaStream_t s) {
  if (b0.n == 0) return 0;
  EigBatch b = b0;
  int Kmax = 0, launches = 0;
  for (int i = 0; i < b.n; ++i) Kmax = std::max(Kmax, b.a[i].K);
  if (Kmax == 0) return 0;
  k_inviter<<<dim3((Kmax + 31) / 32, b.n), 32, 0, s>>>(b);
  ++launches;
  // Newton-Schulz: Z <- Z (1.5 I - 0.5 Z^T Z)
  int n_small = 0, n_large = 0;
  for (int i = 0; i < b.n; ++i)
    if (b.a[i].K > 0) ++(ns_small(b.a[i].m, b.a[i].K) ? n_small : n_large);
  if (n_small > 0) {
    k_ns_small<<<b.n, 256, 0, s>>>(b);
    ++launches;
  }
  bool in_z2 = true;  // three rounds end in Z2
  if (n_large > 0) in_z2 = false;
  for (int it = 0; it < 3 && n_large > 0; ++it) {
    Gemm g1(false, OP_C, OP_N), g2(false, OP_N, OP_N);
    std::vector<OzProb> o1, o2;  // the mixed path: the same real products on the exact-digit engine
    for (int i = 0; i < b.n; ++i) {
      const EigMat& M = b.a[i];
      if (M.K == 0 || ns_small(M.m, M.K)) continue;
      const double* Zc = in_z2 ? M.Z2 : M.Z;
      double* Zn = in_z2 ? M.Z : M.Z2;
      if (mixed) {
        OzProb q{};
        q.row_div = q.col_div = 1;
        q.alpha = 1.0;
        q.ws = oz_ws[i];
        OzProb g = q;  // S = Z^T Z
        g.a = OzOperand{reinterpret_cast<const double2*>(Zc), 1, M.K, nullptr, 1, 0, 1};
        g.M = g.N = M.K; g.K = M.m; g.Creal = M.S; g.ldc = M.K; g.gram = g.herm = 1;
        o1.push_back(g);
        OzProb z = q;  // Z' = Z S
        z.a = OzOperand{reinterpret_cast<const double2*>(Zc), M.K, 1, nullptr, 1, 0, 1};
        z.b = OzOperand{reinterpret_cast<const double2*>(M.S), 1, M.K, nullptr, 1, 0, 1};
        z.M = M.m; z.N = M.K; z.K = M.K; z.Creal = Zn; z.ldc = M.K;
        o2.push_back(z);
      } else {
        g1.add(M.K, M.K, M.m, Zc, M.K, Zc, M.K, M.S, M.K);
      }
    }
    launches += mixed ? oz_gemm_launch(o1, status, s) : g1.launch(s);
    k_ns_form<<<dim3(std::max(1, std::min(64, (Kmax * Kmax + 255) / 256)), b.n), 256, 0, s>>>(b);
    ++launches;
    if (mixed) {
      launches += oz_gemm_launch(o2, status, s);
    } else {
      for (int i = 0; i < b.n; ++i) {
        const EigMat& M = b.a[i];
        if (M.K == 0 || ns_small(M.m, M.K)) continue;
        const double* Zc = in_z2 ? M.Z2 : M.Z;
        double* Zn = in_z2 ? M.Z : M.Z2;
        g2.add(M.m, M.K, M.K, Zc, M.K, M.S, M.K, Zn, M.K);
      }
      launches += g2.launch(s);
    }
    in_z2 = !in_z2;
  }
  const int mm = max_m(b);
  const int nblk = bt_blocks(mm);
  static PerDevice smem;
  smem([] {
    return allow_smem(k_backtransform<false>, BTS_SMEM) & allow_smem(k_backtransform<true>, BTS_SMEM) &
           allow_smem(k_bt_T, BT * (BT + 1) * 16);
  });
  if (!mixed) {  // four vectors per block: few of them spread over the SMs
    int m1 = 0, blocks = 1;  // the largest matrix of a warp per vector
    size_t bytes = 0;
    for (int i = 0; i < b.n; ++i) {
      const int m = b.a[i].m, nv = m <= BTS_WARP ? 4 : btw_vectors(m);
      blocks = std::max(blocks, (b.a[i].K + nv - 1) / nv);
      if (m <= BTS_WARP) m1 = std::max(m1, m);
      if (m > 256) bytes = std::max(bytes, (size_t)nv * ((m + 31) & ~31) * 16);
    }
    const dim3 grid(blocks, b.n);
    const int stride = (m1 + 31) & ~31, z2 = in_z2 ? 1 : 0;
    if (mm > BTS_WARP) k_backtransform<true><<<grid, 256, bytes, s>>>(b, stride, z2);
    else k_backtransform<false><<<grid, 128, bytes, s>>>(b, stride, z2);
    return launches + 1;
  }
  k_z_to_u<<<dim3((mm + 31) / 32, (Kmax + 31) / 32, b.n), dim3(32, 8), 0, s>>>(b, in_z2 ? 1 : 0);
  ++launches;
  if (nblk == 0) return launches;  // 1 x 1 matrices only
  k_bt_clear<<<dim3(std::min(mm, 152), b.n), 128, 0, s>>>(b);
  Gemm gG(true, OP_N, OP_C);  // conj(V^+ V): FP64 on the CUDA cores (64 rows per block: too few for a tensor tile's cost)
  for (int i = 0; i < b.n; ++i) {
    const EigMat& M = b.a[i];
    if (M.K == 0) continue;
    for (int p = 0; p < bt_blocks(M.m); ++p) {
      const int k0 = p * BT, nb = std::min(BT, M.m - 1 - k0);
      const double2* V = M.H + (size_t)k0 * M.m + k0 + 1;
      gG.add(nb, nb, M.m - k0 - 1, V, M.m, V, M.m, bt_G(M, p), nb).herm = 1;
    }
  }
  launches += gG.launch(s);
  k_bt_T<<<dim3(nblk, b.n), 4 * BT, BT * (BT + 1) * 16, s>>>(b);
  launches += 2;
  for (int p = nblk - 1; p >= 0; --p) {
    const int k0 = p * BT;
    std::vector<OzProb> oS, oS2, oU;
    for (int i = 0; i < b.n; ++i) {
      const EigMat& M = b.a[i];
      const int m = M.m, K = M.K, mr = m - k0 - 1, nb = std::min(BT, mr);
      if (K == 0 || mr <= 0) continue;
      const double2* V = M.H + (size_t)k0 * m + k0 + 1;  // row i: v_{k0+i} from index k0 + 1 on
      const double2* Tt = bt_Tt(M, p);
      double2* S = bt_S(M);
      double2* S2 = S + (size_t)m * BT;
      double2* U = M.U + k0 + 1;
      OzProb q{};
      q.row_div = q.col_div = 1;
      q.alpha = 1.0;
      q.ws = oz_ws[i];
      OzProb t = q;  // S = U conj(V): S[j][i] = sum_r U[j][r] conj(V[r][i])
      t.a = OzOperand{U, m, 1, nullptr, 1, 0};
      t.b = OzOperand{V, m, 1, nullptr, 1, 1};
      t.M = K; t.N = nb; t.K = mr; t.C = S; t.ldc = nb;
      oS.push_back(t);
      OzProb t2 = q;  // S2 = S T^T
      t2.a = OzOperand{S, nb, 1, nullptr, 1, 0};
      t2.b = OzOperand{Tt, 1, nb, nullptr, 1, 0};
      t2.M = K; t2.N = nb; t2.K = nb; t2.C = S2; t2.ldc = nb;
      oS2.push_back(t2);
      OzProb u = q;  // U -= S2 V^T
      u.a = OzOperand{S2, nb, 1, nullptr, 1, 0};
      u.b = OzOperand{V, 1, m, nullptr, 1, 0};
      u.M = K; u.N = mr; u.K = nb; u.C = U; u.ldc = m; u.alpha = -1.0; u.beta = 1;
      oU.push_back(u);
    }
    launches += oz_gemm_launch(oS, status, s);
    launches += oz_gemm_launch(oS2, status, s);
    launches += oz_gemm_launch(oU, status, s);
  }
  return launches;
}

}  // namespace ptebd
