// Grouped FP64 GEMM for the TEBD contractions (complex) and the eigenvector
// orthonormalisation (real).
//
// Bound: the FP64 pipe, which takes a warp-wide DFMA every 16 to 19 clocks per SM (1.7 to 2
// lanes per clock, measured) however many of its lanes are active.  A tile needs no depth to
// keep it busy (a 16 x 16 complex tile loads under 1 byte per clock from L2), so what counts is
// that no lane computes padding and that every SM has a tile:
//   * tiles are at most 16 x 16 outputs, one per thread, of balanced height and width
//     (24 rows make two tiles of 12), and the threads number a tile's outputs
//     consecutively, so a ragged tile costs only the warps that it fills;
//   * a problem with few tiles splits its reduction over 2, 4 or 8 CTAs of a cluster, which add
//     their partial sums through distributed shared memory in a fixed order.  The split
//     depends on the problem's own shape only, so a result never depends on its batch.
// One launch serves up to GEMM_MAXP independent problems (all triples of a Trotter layer), each
// optionally strided-batched.
// Measured against 64 x 64 tiles with padded outputs: 1000 x 250 x 3990 complex 16.8 -> 7.2 ms (1.11
// TFLOP/s), a bond correlator of chi = 24, d = 4 (two 24 x 24 x 96 products) 806 -> 31 us, a four-step
// quench of L = 8 60.6 -> 23.2 ms, of the blocked L = 41, d = 5 chain 153 -> 45.7 ms.
#include "ptebd_internal.h"

#include <algorithm>
#include <stdexcept>

namespace ptebd {

namespace {

constexpr int TB = 16;        // largest tile height and width
constexpr int BK = 16;        // reduction slab
constexpr int NT = TB * TB;   // one output per thread
constexpr int CLUSTER = 8;    // CTAs per cluster of a launch that holds a split problem
// A problem whose tiles do not fill the 152 SMs twice is split as long as a slice keeps 8
// reduction indices: with two tiles or more per SM the slices' exchange is the larger part.
constexpr long long FILL = 2 * 152;

__host__ __device__ __forceinline__ int tile_count(int n) { return (n + TB - 1) / TB; }
__host__ __device__ __forceinline__ int tile_size(int n) {  // balanced: the tiles differ by the last one only
  const int t = tile_count(n);
  return (n + t - 1) / t;
}
__host__ __device__ __forceinline__ long long tiles_of(const GemmProb& p) {
  const long long tm = tile_count(p.M), tn = tile_count(p.N);
  return p.batch * (p.herm ? tm * (tm + 1) / 2 : tm * tn);
}
int split_of(const GemmProb& p) {
  int s = 1;
  while (s < CLUSTER && tiles_of(p) * s < FILL && p.K >= 16 * s) s *= 2;
  return s;
}

struct R {  // real arithmetic
  using T = double;
  static __device__ __forceinline__ T zero() { return 0.0; }
  static __device__ __forceinline__ T cj(T x) { return x; }
  static __device__ __forceinline__ T scale(T x, double s) { return x * s; }
  static __device__ __forceinline__ void mac(T& acc, T a, T b) { acc = fma(a, b, acc); }
  static __device__ __forceinline__ T mul_alpha(T x, double ar, double) { return x * ar; }
  static __device__ __forceinline__ T add(T a, T b) { return a + b; }
};

struct C {  // complex arithmetic, interleaved (re, im)
  using T = double2;
  static __device__ __forceinline__ T zero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ T cj(T x) { return make_double2(x.x, -x.y); }
  static __device__ __forceinline__ T scale(T x, double s) { return make_double2(x.x * s, x.y * s); }
  static __device__ __forceinline__ void mac(T& acc, T a, T b) {
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
  }
  static __device__ __forceinline__ T mul_alpha(T x, double ar, double ai) {
    return make_double2(x.x * ar - x.y * ai, x.x * ai + x.y * ar);
  }
  static __device__ __forceinline__ T add(T a, T b) { return make_double2(a.x + b.x, a.y + b.y); }
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A shared-memory double of another CTA of the cluster.
__device__ __forceinline__ double peer_load(const double* mine, unsigned rank) {
  double v;
  asm volatile("{\n .reg .u32 a;\n mapa.shared::cluster.u32 a, %1, %2;\n ld.shared::cluster.f64 %0, [a];\n}\n"
               : "=d"(v)
               : "r"((unsigned)__cvta_generic_to_shared(mine)), "r"(rank)
               : "memory");
  return v;
}
__device__ __forceinline__ double peer_value(const double* mine, unsigned rank) { return peer_load(mine, rank); }
__device__ __forceinline__ double2 peer_value(const double2* mine, unsigned rank) {
  const double* m = reinterpret_cast<const double*>(mine);
  return make_double2(peer_load(m, rank), peer_load(m + 1, rank));
}

template <class A_, int OPA, int OPB, int CAP>
__global__ void __launch_bounds__(NT) gemm_kernel(const __grid_constant__ GemmBatch<CAP> gb) {
  using T = typename A_::T;
  __shared__ T As[BK][TB + 1];
  __shared__ T Bs[BK][TB + 1];
  __shared__ T part[NT];

  // the problem of this CTA: tile_start counts CTAs, a multiple of the cluster size per problem
  int pi = 0, hi = gb.nprob - 1;
  while (pi < hi) {
    const int mid = (pi + hi + 1) >> 1;
    if (gb.tile_start[mid] <= (int)blockIdx.x) pi = mid; else hi = mid - 1;
  }
  const GemmProb& P = gb.p[pi];
  const int split = P.split, local = blockIdx.x - gb.tile_start[pi];
  const unsigned rank = split > 1 ? cluster_rank() : 0;
  const int slice = (int)rank & (split - 1);
  const long long unit = local / split;  // the CTAs of a tile are neighbours in their cluster
  const int tn = tile_count(P.N), tm = tile_count(P.M), hm = tile_size(P.M), hn = tile_size(P.N);
  const int per_batch = P.herm ? tm * (tm + 1) / 2 : tm * tn;
  const bool live = unit < (long long)per_batch * P.batch;  // the last cluster may hold idle CTAs
  const int bidx = live ? (int)(unit / per_batch) : 0, r = live ? (int)(unit % per_batch) : 0;
  int bm, bn;
  if (P.herm) {  // r enumerates the lower-triangular tiles row by row
    bm = (int)((sqrtf(8.0f * (float)r + 1.0f) - 1.0f) * 0.5f);
    while (bm * (bm + 1) / 2 > r) --bm;
    while ((bm + 1) * (bm + 2) / 2 <= r) ++bm;
    bn = r - bm * (bm + 1) / 2;
  } else {
    bm = r / tn;
    bn = r % tn;
  }
  const int m0 = bm * hm, n0 = bn * hn;
  const int mt = live ? min(hm, P.M - m0) : 0, nt = live ? min(hn, P.N - n0) : 0;
  const T* __restrict__ A = static_cast<const T*>(P.A) + (long long)bidx * P.sA;
  const T* __restrict__ B = static_cast<const T*>(P.B) + (long long)bidx * P.sB;
  T* __restrict__ Cm = static_cast<T*>(P.C) + (long long)bidx * P.sC;
  // this CTA's share of the reduction
  const int ks = (P.K + split - 1) / split;
  const int kb = min(P.K, slice * ks), ke = live ? min(P.K, kb + ks) : kb;

  // the element of each operand's slab that this thread loads
  const int ai = (OPA == OP_C) ? threadIdx.x % TB : threadIdx.x / BK;
  const int ak = (OPA == OP_C) ? threadIdx.x / TB : threadIdx.x % BK;
  const int bj = (OPB == OP_C) ? threadIdx.x / BK : threadIdx.x % TB;
  const int bk = (OPB == OP_C) ? threadIdx.x % BK : threadIdx.x / TB;
  auto load_a = [&](int k0) {
    T v = A_::zero();
    const int gi = m0 + ai, gk = k0 + ak;
    if (ai < mt && gk < ke) {
      const int kr = P.red_grp > 0 ? gk + gk / P.red_grp : gk;
      if (OPA == OP_N) v = A[(long long)gi * P.lda + kr];
      else if (OPA == OP_C) v = A_::cj(A[(long long)kr * P.lda + gi]);
      else v = A_::cj(A[(long long)gi * P.lda + kr]);
      if (P.s_red) v = A_::scale(v, P.s_red[gk / P.red_div]);
    }
    return v;
  };
  auto load_b = [&](int k0) {
    T v = A_::zero();
    const int gj = n0 + bj, gk = k0 + bk;
    if (bj < nt && gk < ke) {
      const int kr = P.red_grp > 0 ? gk + gk / P.red_grp : gk;
      if (OPB == OP_N) v = B[(long long)kr * P.ldb + gj];
      else if (OPB == OP_C) v = A_::cj(B[(long long)gj * P.ldb + kr]);
      else v = A_::cj(B[(long long)kr * P.ldb + gj]);
      if (P.s_red_b) v = A_::scale(v, P.s_red_b[gk / P.red_div]);
    }
    return v;
  };

  const int outs = mt * nt, e = threadIdx.x;
  const int oi = (e < outs) ? e / nt : 0, oj = (e < outs) ? e - oi * nt : 0;
  const bool busy = (int)(threadIdx.x & ~31u) < outs;  // the warp holds an output
  T acc = A_::zero();
  T va = load_a(kb), vb = load_b(kb);
  for (int k0 = kb; k0 < ke; k0 += BK) {
    As[ak][ai] = va;
    Bs[bk][bj] = vb;
    __syncthreads();
    if (k0 + BK < ke) {  // the next slab is on its way while this one multiplies
      va = load_a(k0 + BK);
      vb = load_b(k0 + BK);
    }
    if (busy) {
      const int kn = min(BK, ke - k0);
      if (kn == BK) {
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) A_::mac(acc, As[kk][oi], Bs[kk][oj]);
      } else {
        for (int kk = 0; kk < kn; ++kk) A_::mac(acc, As[kk][oi], Bs[kk][oj]);
      }
    }
    __syncthreads();
  }

  int e0 = 0, e1 = outs;
  if (split > 1) {  // add the slices' partial sums; each CTA finishes its share of the outputs
    part[e] = acc;
    cluster_sync();
    const int per = (NT / split);  // at least one warp of outputs each
    e0 = slice * per;
    e1 = min(outs, e0 + per);
    if (e >= e0 && e < e1) {
      const unsigned first = rank - (unsigned)slice;
      acc = peer_value(&part[e], first);
      for (int q = 1; q < split; ++q) acc = A_::add(acc, peer_value(&part[e], first + q));
    }
    cluster_sync();  // no CTA leaves while another reads its sums
  }
  if (e < e0 || e >= e1) return;
  const int gi = m0 + oi, gj = n0 + oj;
  T v = acc;  // (a factor of one is not multiplied: 4 of 4 K + 4 instructions, 5 % of 8192 x 8192 x 16)
  if (P.alpha_im != 0.0) v = A_::mul_alpha(v, P.alpha_re, P.alpha_im);
  else if (P.alpha_re != 1.0) v = A_::scale(v, P.alpha_re);
  if (P.s_row || P.s_col)
    v = A_::scale(v, (P.s_row ? P.s_row[gi / P.row_div] : 1.0) * (P.s_col ? P.s_col[gj / P.col_div] : 1.0));
  T* dst = Cm + (long long)gi * P.ldc + gj;
  *dst = P.accumulate ? A_::add(*dst, v) : v;
  if (P.herm && bn < bm) {  // mirror an off-diagonal tile into the upper triangle
    T* mir = Cm + (long long)gj * P.ldc + gi;
    const T cv = A_::cj(v);
    *mir = P.accumulate ? A_::add(*mir, cv) : cv;
  }
}

template <class A_, int OPA, int OPB, int CAP>
void launch_one(const GemmBatch<CAP>& gb, int ctas, bool clustered, cudaStream_t s) {
  if (!clustered) {
    gemm_kernel<A_, OPA, OPB, CAP><<<ctas, NT, 0, s>>>(gb);
    return;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(NT);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = CLUSTER;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, gemm_kernel<A_, OPA, OPB, CAP>, gb);  // a failure stays pending for the caller's check
}

template <class A_, int CAP>
void dispatch(int opA, int opB, const GemmBatch<CAP>& gb, int ctas, bool clustered, cudaStream_t s) {
  const int key = opA * 3 + opB;
  switch (key) {
#define CASE(a, b) \
  case a * 3 + b: launch_one<A_, a, b, CAP>(gb, ctas, clustered, s); break;
    CASE(0, 0) CASE(0, 1) CASE(0, 2) CASE(1, 0) CASE(1, 1) CASE(1, 2) CASE(2, 0) CASE(2, 1) CASE(2, 2)
#undef CASE
    default: throw std::runtime_error("bad gemm op");
  }
}

// Launches the problems [i, n) that fit one batch; returns the index after the last one taken.
template <int CAP>
size_t launch_some(bool cplx, int opA, int opB, const GemmProb* p, size_t i, size_t n, int& launches, cudaStream_t s) {
  GemmBatch<CAP> gb;
  gb.nprob = 0;
  long long ctas = 0;
  bool clustered = false;
  const size_t first = i;
  for (; i < n && gb.nprob < CAP; ++i) {
    const GemmProb& q = p[i];
    if (q.M <= 0 || q.N <= 0 || q.batch <= 0) continue;
    const int split = split_of(q);
    long long c = tiles_of(q) * split;
    c = (c + CLUSTER - 1) / CLUSTER * CLUSTER;
    if (gb.nprob > 0 && ctas + c > 0x7fffffffLL) break;  // the rest goes to the next launch
    gb.p[gb.nprob] = q;
    gb.p[gb.nprob].split = split;
    clustered = clustered || split > 1;
    gb.tile_start[gb.nprob++] = (int)ctas;
    ctas += c;
  }
  if (ctas == 0) return std::max(i, first + 1);
  gb.tile_start[gb.nprob] = (int)ctas;
  if (cplx) dispatch<C, CAP>(opA, opB, gb, (int)ctas, clustered, s);
  else dispatch<R, CAP>(opA, opB, gb, (int)ctas, clustered, s);
  ++launches;
  return i;
}

size_t launch_batch(bool cplx, int opA, int opB, const GemmProb* p, size_t i, size_t n, int& launches, cudaStream_t s) {
  return n - i <= (size_t)FEW_MAXP ? launch_some<FEW_MAXP>(cplx, opA, opB, p, i, n, launches, s)
                                   : launch_some<GEMM_MAXP>(cplx, opA, opB, p, i, n, launches, s);
}

}  // namespace

static_assert(sizeof(GemmBatch<GEMM_MAXP>) < 32000, "kernel parameter block too large (32 KB on sm_70 and later)");

GemmProb& Gemm::add(int M, int N, int K, const void* A, long long lda, const void* B, long long ldb, void* C,
                    long long ldc) {
  GemmProb p{};
  p.A = A; p.B = B; p.C = C;
  p.lda = lda; p.ldb = ldb; p.ldc = ldc;
  p.M = M; p.N = N; p.K = K; p.batch = 1;
  p.red_div = p.row_div = p.col_div = 1;
  p.alpha_re = 1.0; p.alpha_im = 0.0;
  probs_.push_back(p);
  return probs_.back();
}

int gemm_launch_single(bool complex_, int opA, int opB, const GemmProb& p, cudaStream_t s) {
  int launches = 0;
  launch_batch(complex_, opA, opB, &p, 0, 1, launches, s);
  return launches;
}

int Gemm::launch_tf32(cudaStream_t s, int* status, void* const* ws) {
  std::vector<TcGemmProb> tp;
  for (size_t i = 0; i < probs_.size(); ++i) {
    const GemmProb& p = probs_[i];
    if (!cplx_ || opA_ != OP_N || opB_ == OP_CJ || p.s_red || p.s_red_b || p.s_row || p.s_col || p.accumulate || p.herm ||
        p.alpha_im != 0.0 || (p.batch > 1 && p.sA != 0))
      throw std::runtime_error("not a 3xTF32 product");
    TcGemmProb q{};
    q.A = static_cast<const double2*>(p.A);
    q.B = static_cast<const double2*>(p.B);
    q.C = static_cast<double2*>(p.C);
    q.lda = p.lda; q.ldb = p.ldb; q.ldc = p.ldc;
    q.sB = p.sB; q.sC = p.sC;
    q.alpha = p.alpha_re;
    q.M = p.M; q.N = p.N; q.K = p.K; q.batch = p.batch; q.opB = opB_;
    q.ws = ws[i];
    tp.push_back(q);
  }
  probs_.clear();
  return tc_gemm_launch(tp, status, s);
}

int Gemm::launch(cudaStream_t s) {
  int launches = 0;
  for (size_t i = 0; i < probs_.size();)
    i = launch_batch(cplx_, opA_, opB_, probs_.data(), i, probs_.size(), launches, s);
  probs_.clear();
  return launches;
}

}  // namespace ptebd
