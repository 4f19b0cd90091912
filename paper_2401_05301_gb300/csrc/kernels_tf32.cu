// Complex GEMM on the 5th-generation tensor cores as split 3xTF32 products
// with FP32 accumulation (the mixed-precision contractions: theta = B B B,
// the gate, and the rebuild of B).
//
// C (complex, FP64 in memory) = alpha * A * op(B), op(B) in {B, B^+}.
// Real embedding: A is used as stored (re/im interleaved along K, so as a real
// M x 2K matrix) and B is expanded to the real 2K x 2N matrix with 2x2 blocks
// [[br, bi], [-bi, br]]; the real product then holds (Re C, Im C) interleaved
// along its columns, i.e. exactly the complex C.
//
// Split: every FP64 operand element x is cut into tf32 hi + lo by integer
// operations on its IEEE-754 fields, both rounded to nearest, so that
// |x - hi - lo| <= 2^-23 |x| without bias.  The product keeps
// hi*hi + hi*lo + lo*hi (three MMAs per k-step) and drops lo*lo.  No FP64
// arithmetic happens in the loop: on this part FP64 runs at 1/64 of the FP32 rate.
//
// Accumulation: the tensor core's FP32 accumulation rounds towards zero, which
// over a long K becomes a bias growing linearly with K (measured -1e-4 relative
// at K = 4096 with same-sign data).  Every k-step of 8 reals therefore gets a
// fresh accumulator in tensor memory (hi*lo, lo*hi, then hi*hi: one large
// product per chain), and after each slab the threads add the four
// accumulators into FP32 registers with round-to-nearest adds (measured bias
// ~4e-8 relative, independent of K).
//
// Data path.  A packing kernel cuts every operand element once and writes the hi and lo planes in
// the 128-byte-swizzled K-major image that the tensor core reads (blocks of 32 rows x 32 reals, 4 KB,
// ordered [plane][slab][row block]), so a tile of a slab is one contiguous bulk copy per plane.  The
// product kernel (one 128 x 128 real tile per CTA) is warp-specialised: one thread issues the
// copies into a ring of three slabs, one thread issues tcgen05.mma.kind::tf32 (M = 128, N = 128,
// K = 8), and eight warps drain each accumulator as soon as its three products are done and hand
// it back, so the products of the next slab overlap the drains.  Tiles leave through shared memory
// in whole rows.
// Bound: the drains (64 KB of tensor memory and 128 x 128 adds per k-step).  Measured against
// splitting both operands again in every CTA (same bits): 4096 x 1024 x 256 complex 683 -> 132 us.
// Every mbarrier wait is bounded (~1 s); on timeout the CTA flags an error, drains its issued
// copies and MMAs (bounded), frees its tensor memory and returns.
#include "ptebd_internal.h"

#include <algorithm>
#include <cstdint>

namespace ptebd {

namespace {

constexpr int TM = TC_TILE_M;         // rows of the real product per CTA (UMMA M)
constexpr int TN = 2 * TC_TILE_N;     // columns of the real product per CTA (UMMA N) = 64 complex
constexpr int TK = 32;                // reals of K per slab (one 128-byte swizzle row of fp32)
constexpr int DW = 8;                 // drain warps: 4 lane groups x 2 column halves
constexpr int NT = 32 * (DW + 2);     // + one copy warp + one MMA warp
constexpr int BLK = 4096;             // one packed block: 32 rows x 32 fp32
constexpr int A_BYTES = TM * TK * 4;  // 16 KB per plane
constexpr int B_BYTES = TN * TK * 4;  // 16 KB per plane
constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;  // hi and lo planes of A and B: 64 KB
constexpr int NACC = TK / 8;          // one accumulator per k-step of a slab
constexpr int TMEM_COLS = NACC * TN;  // 512: the whole tensor memory of the SM
constexpr int STAGES = 3;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
constexpr int OUT_LD = TN / 2 + 1;    // staged output row (complex), padded
constexpr long long WAIT_CLOCKS = 2000000000LL;  // ~1 s at 2 GHz
static_assert(TM * OUT_LD * 16 <= STAGES * STAGE_BYTES, "the staged tile must fit the stages");

// ---- small PTX wrappers ---------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

// Bounded wait for the phase with the given parity; false on timeout or once another role failed.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* fail) {
  const uint32_t a = smem_u32(bar);
  const long long t0 = clock64();
  for (int it = 0;; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if ((it & 63) == 63) {
      if (fail && *fail) return false;
      if (clock64() - t0 > WAIT_CLOCKS) return false;
    }
  }
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// Bulk copy global -> shared (TMA engine), completion counted on bar.
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);  // start address
  d |= (uint64_t)1 << 16;                  // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;        // stride byte offset
  d |= (uint64_t)1 << 46;                  // version
  d |= (uint64_t)2 << 61;                  // 128-byte swizzle
  return d;
}

// Instruction descriptor for kind::tf32: D = f32, A = B = tf32, both K-major, M x N.
__host__ __device__ constexpr uint32_t tf32_idesc(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// x -> (hi, lo) tf32 bit patterns from the IEEE-754 fields of the double:
// hi = x rounded to 11 significant bits, lo = the remainder rounded to 11 bits.
__device__ __forceinline__ void split_tf32(double x, uint32_t& hi, uint32_t& lo) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const uint32_t s = (uint32_t)(b >> 63) << 31;
  const int e = (int)((b >> 52) & 0x7FF);
  const int E = e - 1023;
  hi = 0u;
  lo = 0u;
  if (e == 0 || E < -126) return;  // zero, subnormal or below fp32 range: 0
  const long long M53 = (long long)((b & 0xFFFFFFFFFFFFFull) | (1ull << 52));
  long long hs = (M53 + (1ll << 41)) >> 42;  // 11-bit significand, rounded
  const long long rem = M53 - (hs << 42);    // |rem| <= 2^41
  int He = E;
  if (hs == 2048) { hs = 1024; He = E + 1; }
  if (He > 127) { hi = s | 0x7F800000u; return; }
  hi = s | ((uint32_t)(He + 127) << 23) | ((uint32_t)(hs & 0x3FF) << 13);
  if (rem == 0) return;
  const unsigned long long a = (unsigned long long)(rem < 0 ? -rem : rem);
  const int p = 63 - __clzll((long long)a);  // leading one, 0..41
  int le = E - 52 + p;
  const int sh = p - 10;
  unsigned long long ls;
  if (sh > 0) {
    ls = (a + (1ull << (sh - 1))) >> sh;
    if (ls == 2048) { ls = 1024; ++le; }
  } else {
    ls = a << (-sh);
  }
  if (le < -126) return;
  lo = (s ^ (rem < 0 ? 0x80000000u : 0u)) | ((uint32_t)(le + 127) << 23) | ((uint32_t)(ls & 0x3FF) << 13);
}

// byte offset of fp32 element (row, k) of a 128-byte-swizzled K-major tile
__device__ __forceinline__ uint32_t swz(int row, int k) {
  return (uint32_t)(row * 128 + ((((k >> 2) ^ (row & 7)) & 7) << 4) + ((k & 3) << 2));
}

// ---- packing ----------------------------------------------------------------------

// One operand's planes: rows x K complex; A: element (r, k) at X[r * rs + k]; B: row r is column r of
// op(B), element (k, r) at X[(r / per) * sb + (r % per) * rs + k * ks] (conjugated for op = C).  A row of A is one row of
// reals (re, im); a column of B is two: (br, -bi) and (bi, br).
struct TfPackJob {
  const double2* X;
  long long rs, ks, sb;
  uint8_t* P;      // hi plane, then lo plane
  size_t plane;    // bytes of a plane
  int rows, K, per, b, conj, nrb, nkt;
};
template <int CAP>
struct TfPackBatch {
  TfPackJob job[2 * CAP];
  int block_start[2 * CAP + 1];
  int njob;
};

// Element (local row r, local k q) of packed block (rb, kt) of A into the two planes.
__device__ __forceinline__ void put_a(const TfPackJob& J, int gr, int gk, uint8_t* hi_p, uint8_t* lo_p, uint32_t at) {
  double2 v = make_double2(0.0, 0.0);
  if (gr < J.rows && gk < J.K) v = __ldg(J.X + (long long)gr * J.rs + gk);
  uint32_t h0, l0, h1, l1;
  split_tf32(v.x, h0, l0);
  split_tf32(v.y, h1, l1);
  *reinterpret_cast<uint2*>(hi_p + at) = make_uint2(h0, h1);  // an even k: both words in one 8-byte slot
  *reinterpret_cast<uint2*>(lo_p + at) = make_uint2(l0, l1);
}
// Column gj, element gk of op(B): rows 2 jj and 2 jj + 1 of the block, words 2 q and 2 q + 1.
__device__ __forceinline__ void put_b(const TfPackJob& J, int gj, int gk, uint8_t* hi_p, uint8_t* lo_p, int jj, int q) {
  double2 v = make_double2(0.0, 0.0);
  if (gj < J.rows && gk < J.K) {
    v = __ldg(J.X + (long long)(gj / J.per) * J.sb + (long long)(gj % J.per) * J.rs + (long long)gk * J.ks);
    if (J.conj) v.y = -v.y;
  }
  uint32_t hr, lr, hm, lm;
  split_tf32(v.x, hr, lr);
  split_tf32(v.y, hm, lm);
  const uint32_t sign = 0x80000000u;
  const uint32_t a0 = swz(2 * jj, 2 * q), a1 = swz(2 * jj + 1, 2 * q);
  *reinterpret_cast<uint2*>(hi_p + a0) = make_uint2(hr, hm ^ (hm ? sign : 0u));
  *reinterpret_cast<uint2*>(lo_p + a0) = make_uint2(lr, lm ^ (lm ? sign : 0u));
  *reinterpret_cast<uint2*>(hi_p + a1) = make_uint2(hm, hr);
  *reinterpret_cast<uint2*>(lo_p + a1) = make_uint2(lm, lr);
}

// One block per packed block: 32 rows x 16 complex (A) or 16 columns x 16 complex (B).
template <int CAP>
__global__ void __launch_bounds__(256) k_tf_pack(const __grid_constant__ TfPackBatch<CAP> pb) {
  int j = 0;
  for (int hi = pb.njob - 1; j < hi;) {
    const int mid = (j + hi + 1) >> 1;
    if (pb.block_start[mid] <= (int)blockIdx.x) j = mid; else hi = mid - 1;
  }
  const TfPackJob& J = pb.job[j];
  const int local = blockIdx.x - pb.block_start[j];
  const int rb = local % J.nrb, kt = local / J.nrb;
  uint8_t* hi_p = J.P + ((size_t)kt * J.nrb + rb) * BLK;
  uint8_t* lo_p = hi_p + J.plane;
  if (!J.b) {
    for (int idx = threadIdx.x; idx < 32 * 16; idx += 256) {
      const int r = idx >> 4, q = idx & 15;
      put_a(J, rb * 32 + r, kt * 16 + q, hi_p, lo_p, swz(r, 2 * q));
    }
  } else {
    const bool k_first = J.ks == 1;  // lanes along the contiguous index
    const int q = k_first ? threadIdx.x & 15 : threadIdx.x >> 4, jj = k_first ? threadIdx.x >> 4 : threadIdx.x & 15;
    put_b(J, rb * 16 + jj, kt * 16 + q, hi_p, lo_p, jj, q);
  }
}

// A direct tile's slabs (at most STAGES) by the drain warps themselves.
__device__ void fill_direct(const TfPackJob& A, const TfPackJob& B, int mt, int nt, int nk, uint8_t* smem) {
  for (int kt = 0; kt < nk; ++kt) {
    uint8_t* st = smem + kt * STAGE_BYTES;
    for (int idx = threadIdx.x; idx < TM * 16; idx += 32 * DW) {
      const int r = idx >> 4, q = idx & 15;
      put_a(A, mt * TM + r, kt * 16 + q, st, st + A_BYTES, swz(r, 2 * q));
    }
    for (int idx = threadIdx.x; idx < (TN / 2) * 16; idx += 32 * DW) {
      const bool k_first = B.ks == 1;
      const int q = k_first ? idx & 15 : idx / (TN / 2), jj = k_first ? idx >> 4 : idx % (TN / 2);
      put_b(B, nt * (TN / 2) + jj, kt * 16 + q, st + 2 * A_BYTES, st + 2 * A_BYTES + B_BYTES, jj, q);
    }
  }
}

// ---- the product ------------------------------------------------------------------

struct TfTile {
  const uint8_t* A;   // hi plane, lo plane planeA further
  const uint8_t* B;
  size_t planeA, planeB;
  double2* C;
  long long ldc, sC;
  double alpha;
  int M, N, per, nkt, nrbA, nrbB, tiles_n;
  TfPackJob da, db;   // direct: the operands, cut by the CTA itself (no planes)
  int direct;
};
template <int CAP>
struct TfBatch {
  TfTile p[CAP];
  int tile_start[CAP + 1];
  int nprob;
  int* status;
};

// An FP32 value as FP64, on the integer pipe (the FP64 pipe takes a warp-wide conversion every 16 to 19 clocks).
__device__ __forceinline__ double widen(float f) {
  const uint32_t b = __float_as_uint(f), e = (b >> 23) & 0xFF;
  if (e == 0 || e == 0xFF) return (double)f;  // zero, subnormal, Inf, NaN
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20))), (int)(b << 29));
}

template <int CAP>
__global__ void __launch_bounds__(NT, 1) k_tf32x3(const __grid_constant__ TfBatch<CAP> gb) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* full = bars;                     // [STAGES] a slab has arrived
  uint64_t* empty = bars + STAGES;           // [STAGES] its products are done
  uint64_t* accfull = bars + 2 * STAGES;     // [NACC]
  uint64_t* accempty = accfull + NACC;       // [NACC]
  uint64_t* done = accempty + NACC;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* fail_sh = reinterpret_cast<volatile int*>(tmem_slot + 1);

  int pi = 0;
  for (int hi = gb.nprob - 1; pi < hi;) {
    const int mid = (pi + hi + 1) >> 1;
    if (gb.tile_start[mid] <= (int)blockIdx.x) pi = mid; else hi = mid - 1;
  }
  const TfTile& P = gb.p[pi];
  const int local = blockIdx.x - gb.tile_start[pi];
  const int mt = local / P.tiles_n, nt = local - mt * P.tiles_n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == DW + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < NACC; ++i) { mbar_init(&accfull[i], 1); mbar_init(&accempty[i], DW); }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *fail_sh = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int nk = P.nkt;

  if (warp == DW) {
    // ---- copies: the four planes of a slab
    if (lane == 0 && !P.direct) {
      int issued = 0;
      bool ok = true;
      for (int kt = 0; kt < nk; ++kt) {
        const int st = kt % STAGES;
        if (kt >= STAGES && !mbar_wait(&empty[st], (uint32_t)((kt / STAGES - 1) & 1), fail_sh)) { ok = false; break; }
        uint8_t* dst = smem + st * STAGE_BYTES;
        const uint8_t* a = P.A + ((size_t)kt * P.nrbA + 4 * mt) * BLK;
        const uint8_t* b = P.B + ((size_t)kt * P.nrbB + 4 * nt) * BLK;
        mbar_expect_tx(&full[st], STAGE_BYTES);
        ++issued;
        bulk_copy(dst, a, A_BYTES, &full[st]);
        bulk_copy(dst + A_BYTES, a + P.planeA, A_BYTES, &full[st]);
        bulk_copy(dst + 2 * A_BYTES, b, B_BYTES, &full[st]);
        bulk_copy(dst + 2 * A_BYTES + B_BYTES, b + P.planeB, B_BYTES, &full[st]);
      }
      if (!ok) {  // let the copies already issued land before the CTA's shared memory is released
        *fail_sh = 1;
        for (int kt = max(0, issued - STAGES); kt < issued; ++kt)
          mbar_wait(&full[kt % STAGES], (uint32_t)((kt / STAGES) & 1), nullptr);
      }
    }
  } else if (warp == DW + 1) {
    // ---- products: k-step kk of every slab into accumulator kk, from a fresh start
    if (lane == 0) {
      const uint32_t idesc = tf32_idesc(TM, TN);
      bool ok = true;
      for (int kt = 0; kt < nk && ok; ++kt) {
        const int st = kt % STAGES;
        if (!mbar_wait(&full[st], (uint32_t)((kt / STAGES) & 1), fail_sh)) { ok = false; break; }
        const uint32_t base = smem_u32(smem + st * STAGE_BYTES);
        const uint32_t a_hi = base, a_lo = base + A_BYTES, b_hi = base + 2 * A_BYTES, b_lo = b_hi + B_BYTES;
        for (int kk = 0; kk < NACC; ++kk) {
          if (kt > 0 && !mbar_wait(&accempty[kk], (uint32_t)((kt - 1) & 1), fail_sh)) { ok = false; break; }
          tc_fence_after();
          const uint32_t off = kk * 32;  // 8 tf32 = 32 bytes along K inside the swizzled row
          const uint32_t d = tmem + (uint32_t)(kk * TN);
          mma_tf32(d, smem_desc(a_hi + off), smem_desc(b_lo + off), idesc, 0u);
          mma_tf32(d, smem_desc(a_lo + off), smem_desc(b_hi + off), idesc, 1u);
          mma_tf32(d, smem_desc(a_hi + off), smem_desc(b_hi + off), idesc, 1u);
          mma_commit(&accfull[kk]);
        }
        // (no copy waits for the last stages: an arrival there could outlive the CTA)
        if (ok && kt + STAGES < nk) mma_commit(&empty[st]);
      }
      if (!ok) {
        *fail_sh = 1;
        mma_commit(done);  // all MMAs issued so far complete before tensor memory is freed
        mbar_wait(done, 0, nullptr);
      }
    }
  } else {
    // ---- drain: warp (g, h) owns TMEM lanes 32g.. and columns 64h.. of every accumulator, which it adds
    // into FP32 registers with round-to-nearest adds, k-step by k-step
    const int g = warp & 3, h = warp >> 2;
    if (P.direct) {
      fill_direct(P.da, P.db, mt, nt, nk, smem);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("bar.sync 1, %0;" ::"r"(32 * DW) : "memory");
      if (threadIdx.x == 0)
        for (int kt = 0; kt < nk; ++kt) mbar_arrive(&full[kt]);
    }
    float acc[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) acc[i] = 0.0f;
    bool ok = true;
    for (int kt = 0; kt < nk && ok; ++kt) {
      for (int q = 0; q < NACC; ++q) {
        if (!mbar_wait(&accfull[q], (uint32_t)(kt & 1), fail_sh)) { ok = false; break; }
        tc_fence_after();
        uint32_t v[64];
        const uint32_t taddr = tmem + ((uint32_t)(32 * g) << 16) + (uint32_t)(q * TN + h * 64);
#pragma unroll
        for (int c0 = 0; c0 < 64; c0 += 16)
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
              "[%16];"
              : "=r"(v[c0]), "=r"(v[c0 + 1]), "=r"(v[c0 + 2]), "=r"(v[c0 + 3]), "=r"(v[c0 + 4]), "=r"(v[c0 + 5]),
                "=r"(v[c0 + 6]), "=r"(v[c0 + 7]), "=r"(v[c0 + 8]), "=r"(v[c0 + 9]), "=r"(v[c0 + 10]),
                "=r"(v[c0 + 11]), "=r"(v[c0 + 12]), "=r"(v[c0 + 13]), "=r"(v[c0 + 14]), "=r"(v[c0 + 15])
              : "r"(taddr + c0));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&accempty[q]);  // the values are in registers
#pragma unroll
        for (int i = 0; i < 64; ++i) acc[i] = __fadd_rn(acc[i], __uint_as_float(v[i]));
      }
    }
    if (!ok) *fail_sh = 1;
    // every drain warp takes the same branch; when all drained everything, all copies and MMAs are done
    int any_bad;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.s32 %0, 1, 0, q;\n}\n"
        : "=r"(any_bad)
        : "r"(ok ? 0 : 1), "r"(32 * DW)
        : "memory");
    if (!any_bad && P.direct) {  // few rows: straight from the registers
      const int row = mt * TM + 32 * g + lane;
      if (row < P.M) {
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const int jj = nt * (TN / 2) + 32 * h + i;
          if (jj < P.N)
            P.C[(long long)(jj / P.per) * P.sC + (long long)row * P.ldc + jj % P.per] =
                make_double2(widen(acc[2 * i]) * P.alpha, widen(acc[2 * i + 1]) * P.alpha);
        }
      }
    } else if (!any_bad) {
      double2* out = reinterpret_cast<double2*>(smem);
      double2* mine = out + (size_t)(32 * g + lane) * OUT_LD + 32 * h;
      const double al = P.alpha;
      if (al == 1.0) {
#pragma unroll
        for (int i = 0; i < 32; ++i) mine[i] = make_double2(widen(acc[2 * i]), widen(acc[2 * i + 1]));
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) mine[i] = make_double2(widen(acc[2 * i]) * al, widen(acc[2 * i + 1]) * al);
      }
      asm volatile("bar.sync 1, %0;" ::"r"(32 * DW) : "memory");
      const int cc = threadIdx.x & (TN / 2 - 1), jj = nt * (TN / 2) + cc;  // a thread keeps its column
      if (jj < P.N) {
        double2* dst = P.C + (long long)(jj / P.per) * P.sC + jj % P.per;
        const int rows = min(TM, P.M - mt * TM);
        for (int r = threadIdx.x / (TN / 2); r < rows; r += 32 * DW / (TN / 2))
          dst[(long long)(mt * TM + r) * P.ldc] = out[(size_t)r * OUT_LD + cc];
      }
    }
  }
  __syncthreads();
  if (*fail_sh && threadIdx.x == 0 && gb.status) atomicExch(gb.status, -6);  // TEBD_ERR_TIMEOUT: a bounded wait ran out
  if (warp == DW + 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
  }
}

struct Geo {
  int nkt, nrbA, nrbB;
  size_t planeA, planeB;
};
Geo geometry(int M, long long N, int K) {
  Geo g{};
  g.nkt = (K + 15) / 16;
  g.nrbA = 4 * ((M + TM - 1) / TM);
  g.nrbB = (int)(4 * ((N + TN / 2 - 1) / (TN / 2)));
  g.planeA = (size_t)g.nkt * g.nrbA * BLK;
  g.planeB = (size_t)g.nkt * g.nrbB * BLK;
  return g;
}

}  // namespace

static_assert(sizeof(TfBatch<TC_MAXP>) < 32000 && sizeof(TfPackBatch<TC_MAXP>) < 32000, "kernel parameter block too large (32 KB on sm_70 and later)");
static_assert(tf32_idesc(128, 128) == ((1u << 4) | (2u << 7) | (2u << 10) | (16u << 17) | (8u << 24)), "idesc");

namespace {
// One slab and one wave of tiles: each CTA cuts its own operands, which is cheaper than a launch and a
// workspace for the planes (32 x 16 x 16 complex 15 us a call against 24 with planes; with two slabs,
// 250 x 100 x 30, 31 against 24).
bool tc_direct(int M, long long N, int K) {
  return K <= 16 && (long long)((M + TM - 1) / TM) * ((N + TN / 2 - 1) / (TN / 2)) <= 152;
}
}  // namespace

size_t tc_workspace_bytes(int M, int N, int K, int batch) {
  if (M <= 0 || N <= 0 || K <= 0 || batch <= 0) return 0;
  if (tc_direct(M, (long long)N * batch, K)) return 0;
  const Geo g = geometry(M, (long long)N * batch, K);
  return 2 * (g.planeA + g.planeB);
}

namespace {
template <int CAP>
int launch_all(const std::vector<TcGemmProb>& probs, int* status, cudaStream_t s) {
  static PerDevice smem;
  smem([] { return allow_smem(k_tf32x3<CAP>, SMEM_BYTES); });
  int launches = 0;
  for (size_t i = 0; i < probs.size();) {
    TfBatch<CAP> gb;
    gb.nprob = 0;
    TfPackBatch<CAP> pk;
    pk.njob = 0;
    gb.status = status;
    int tiles = 0, blocks = 0;
    for (; i < probs.size() && gb.nprob < CAP; ++i) {
      const TcGemmProb& p = probs[i];
      if (p.M <= 0 || p.N <= 0 || p.batch <= 0) continue;
      // the columns of all batch entries side by side: A is shared (sA = 0) or there is one entry
      const int N = p.N * p.batch;
      const Geo g = geometry(p.M, N, p.K);
      uint8_t* ws = static_cast<uint8_t*>(p.ws);
      auto job = [&](const TfPackJob& J) {
        pk.job[pk.njob] = J;
        pk.block_start[pk.njob++] = blocks;
        blocks += J.nrb * J.nkt;
      };
      const bool c = p.opB == OP_C;
      const TfPackJob ja{p.A, p.lda, 1, 0, ws, g.planeA, p.M, p.K, 1, 0, 0, g.nrbA, g.nkt};
      const TfPackJob jb{p.B, c ? p.ldb : 1, c ? 1 : p.ldb, p.sB, ws + 2 * g.planeA, g.planeB, N, p.K, p.N, 1,
                         c ? 1 : 0, g.nrbB, g.nkt};
      TfTile& t = gb.p[gb.nprob];
      t = TfTile{};
      t.direct = tc_direct(p.M, N, p.K);
      if (t.direct) {
        t.da = ja;
        t.db = jb;
      } else {
        job(ja);
        job(jb);
      }
      t.A = ws; t.B = ws + 2 * g.planeA; t.planeA = g.planeA; t.planeB = g.planeB;
      t.C = p.C; t.ldc = p.ldc; t.sC = p.sC; t.alpha = p.alpha; t.M = p.M; t.N = N; t.per = p.N;
      t.nkt = g.nkt; t.nrbA = g.nrbA; t.nrbB = g.nrbB; t.tiles_n = g.nrbB / 4;
      gb.tile_start[gb.nprob++] = tiles;
      tiles += (g.nrbA / 4) * t.tiles_n;
    }
    gb.tile_start[gb.nprob] = tiles;
    pk.block_start[pk.njob] = blocks;
    if (tiles == 0) continue;
    if (blocks > 0) {
      k_tf_pack<CAP><<<blocks, 256, 0, s>>>(pk);
      ++launches;
    }
    k_tf32x3<CAP><<<tiles, NT, SMEM_BYTES, s>>>(gb);
    ++launches;
  }
  return launches;
}
}  // namespace

int tc_gemm_launch(const std::vector<TcGemmProb>& probs, int* status, cudaStream_t s) {
  return probs.size() <= (size_t)FEW_MAXP ? launch_all<FEW_MAXP>(probs, status, s) : launch_all<TC_MAXP>(probs, status, s);
}

int tc_gemm_pooled(std::vector<TcGemmProb>& probs, void* pool, size_t bytes, int* status, cudaStream_t s) {
  int launches = 0;
  std::vector<TcGemmProb> group;
  size_t used = 0;
  for (TcGemmProb& q : probs) {
    const size_t need = tc_workspace_bytes(q.M, q.N, q.K, q.batch);
    if (group.size() == (size_t)TC_MAXP || used + need > bytes) {
      launches += tc_gemm_launch(group, status, s);
      group.clear();
      used = 0;
    }
    q.ws = static_cast<char*>(pool) + used;
    used += need;
    group.push_back(q);
  }
  return launches + tc_gemm_launch(group, status, s);
}

}  // namespace ptebd
