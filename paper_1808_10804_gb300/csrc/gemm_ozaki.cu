// FP64-accurate grouped GEMM on the BF16 tensor cores (tcgen05, sm_103a).
//
// Every FP64 row of an operand gets a power-of-two scale 2^e with
// |x| < 2^e; the scaled row is written, with integer arithmetic on the IEEE
// bit pattern, as a signed-digit expansion
//     x / 2^e = 2^-8 (a0 + 2^-9 (a1 + 2^-9 (a2 + 2^-9 (a3 + 2^-9 a4))))
// with integer digits |a_i| <= 256, which BF16 holds exactly (44 bits kept).
// A product of two digits is an integer below 2^16 in magnitude, exact in
// FP32.  The GEMM sums the 15 digit products with i + j <= 4 by diagonal
// d = i + j (weight 2^-16-9d) in tensor memory:
//   * d = 0, 1, 2 are read out every 64 K (two pipeline stages), where their
//     FP32 sums are exact integers of magnitude <= 3 * 2^22 < 2^24, and
//     added into one 64-bit integer per output (K <= kMaxK keeps it from
//     overflowing);
//   * d = 3, 4 carry weights <= 2^-27 of the leading term and accumulate in
//     FP32 over the whole K.
// The epilogue forms the result with 64-bit integer arithmetic and one
// conversion to FP64.  Relative error ~2^-40 against the row/column scales.
//
// Kernel: persistent, one CTA per SM walking the plan's 128 x 64 (or
// 128 x 32) output tiles; warp 0 drives TMA (64-byte swizzled K-major tiles,
// a ring of 3 stages for five slices, up to 6 for three), warp 1 issues
// tcgen05.mma from one thread (the 15 digit products of a 16-K step as 8
// products, each an A slice times a run of stacked B slices), warps 2..17
// drain tensor memory.
//
// What bounds it: a 32-K chunk's 16 products take the tensor core 960 cycles at
// its peak rate, a chunk of a running tile about 1900 (2432 x 2432 x 2432: five
// tiles of 76 chunks a CTA in 352 us at 2070 MHz; 1450 with the epilogue
// idle); over a batch of 8 corners the tensor pipe is active 49 % of the time.
// The rest is the issuing thread, whose products queue only a few deep: whatever it does between the last product
// of a chunk and the first of the next leaves the tensor core idle, and it
// shares its issue slots with the epilogue.  Hence counters in place of
// divisions, tile tables that hold all a role needs, one copy per operand and
// chunk, barriers looked at ahead of time, and no conversion instruction in
// the epilogue that an addition replaces.  2432 x 2432 x 2432, five digits:
// 430 -> 352 us (1.23 PFLOP/s of digit products); four of 2048 x 2048 x 512:
// 347 -> 253 us; 2432^3 with three digits: 292 -> 233 us.  A tile of one or
// two chunks is bound by the instructions of its output instead (about 100 an
// element for four warps a scheduler): 200000 x 192 x 16, 307 MB out, 243 ->
// 199 us with sums that need no shift or sign extension, 32-bit halves in the
// conversion and four rows side by side.  The launch is programmatic behind
// the split or pack: 1.6 us less per contraction.
//
// Every wait of the pipeline is bounded by the launch's spin limit: on expiry
// the kernel records BST_E_TIMEOUT in the context's error word, the copying
// and the issuing role leave their loops, and the output stage stores nothing
// more; before tensor memory is freed and the CTA exits, the TMA copies it
// has issued and the products it has issued are waited for (they always
// complete; those waits carry a separate, much larger bound).
#include <cuda.h>
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "bst_internal.h"
#include "relayout_dev.cuh"

namespace bst {

namespace oz {

namespace cg = cooperative_groups;

constexpr int kTM = 128;           // tile rows (M)
constexpr int kTK = 32;            // K per stage (64 bytes of BF16)
constexpr int kMaxK = 10000;       // longest sum of a plan (at most 2^43 K < 2^57 in the accumulators)
constexpr int kABytes = kTM * kTK * 2;   // 8 KB per slice
constexpr int kEpiWarps = 16;            // four per quarter of the 128 tensor-memory lanes
constexpr int kThreads = 32 * (2 + kEpiWarps);  // TMA, MMA and epilogue warps
constexpr long long kSpinLimit = 1ll << 28;   // default bound of a pipeline wait (tries)
constexpr long long kDrainLimit = 1ll << 30;  // bound of the waits for issued copies and products

// Shape of one instantiation: S digit slices per operand (5: the FP64-
// accurate split; 3: 26 bits, the cheaper arithmetic), output tiles of
// 128 x TN (TN = 64, or 32 for narrow problems: twice the tiles).
//   tensor memory: d0, d1, d2 side by side, double-buffered (buffer b at
//   columns 3 TN b), then for S = 5 the whole-K diagonals d3 and d4 (2 TN
//   more, from 6 TN); allocated as the next power of two.
template <int S, int TN>
struct Cfg {
  static_assert(S == 5 || S == 3, "digit slices");
  static_assert(TN == 64 || TN == 32, "tile width");
  static constexpr int kBBytes = TN * kTK * 2;
  static constexpr int kStageBytes = S * (kABytes + kBBytes);
  static constexpr int kStages = (196608 / kStageBytes) < 6 ? (196608 / kStageBytes) : 6;
  static constexpr int kColD3 = 6 * TN;
  static constexpr int kCols = 6 * TN + (S - 3) * TN;
  static constexpr int kTmemCols = kCols <= 256 ? 256 : 512;
  // C = T 2^(ea + eb - kShift): T = S0 2^27 + S1 2^18 + S2 2^9 + S3 + S4 2^-9
  // (S = 5) or S0 2^18 + S1 2^9 + S2 (S = 3)
  static constexpr int kShift = S == 5 ? 43 : 34;
  static constexpr int kTopBits = 9 * S - 1;  // bits of the scaled integer (44 or 26)
};

struct Prob {
  int32_t M, N, K, pad;
  int32_t arow, brow;  // first row of this problem in the split A / B buffers
  int64_t c_off, c_m, c_n;
  // output scatter (plans with tables, see Scatter): element (m, n) of the
  // problem goes to C[bbase[bb_off + r ncc + c] + mi w + ni] with (r, mi) = rowtab[rt_off + m]
  // and (c, ni, w) = coltab[ct_off + n]: the canonical block (r, c) of the
  // output tensor, row-major [rows of config r x w], instead of a strided
  // sector matrix
  int32_t ncc;
  int64_t rt_off, ct_off, bb_off;
};

// Output scatter tables of a plan (device pointers; all null for a plain
// strided output) and the epilogue's C = alpha * A B + beta * C.
struct Scatter {
  const int2* rowtab;
  const int4* coltab;
  const long long* bbase;
  double alpha, beta;
};

struct Tile {
  int32_t prob;
  int32_t m0, n0;      // first row and column; their low bits (m0: 7, n0: those of TN - 1) hold the
                       // tile's rows and columns inside the problem, less one
  int32_t nk;          // K chunks of kTK
  int32_t arow, brow;  // the tile's first rows in the split A / B buffers
  int32_t rt, ct;      // its first entries in the scatter's row and column tables
};

struct SplitTask {
  int32_t rows, K;
  int32_t row0, pad;  // first row in the split buffer
  int64_t base, s_r, s_k;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// The same look without the time slice that try_wait may spend asleep.
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait; returns false (and raises the abort flag) on expiry or when
// another role already aborted.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag, int* err,
                                          long long limit) {
  for (long long i = 0; i < limit; ++i) {
    if (mbar_try(b, parity)) return true;
    if (*abort_flag) return false;
  }
  *abort_flag = 1;
  atomicExch(err, int(BST_E_TIMEOUT));
  return false;
}

// All S slices of a tile's rows for one K chunk: box {kTK, rows, S}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          smem_u32(dst)),
      "l"(map), "r"(c0), "r"(c1), "r"(0), "r"(smem_u32(bar))
      : "memory");
}

// Shared-memory matrix descriptor: K-major, 64-byte swizzle, 8-row groups
// 512 bytes apart.  Low word: address / 16 (14 bits; the tiles lie below 227
// KB, so offsets are added without a carry out) and the leading byte offset
// (unused with swizzle); high word: stride, descriptor version, SWIZZLE_64B.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr >> 4) & 0x3FFF) | (1u << 16); }
constexpr uint32_t kDescHi = (512u >> 4) | (1u << 14) | (4u << 29);

// kind::f16 instruction descriptor: BF16 x BF16 -> F32, both K-major.
template <int TN>
__host__ __device__ constexpr uint32_t instr_desc() {
  return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(TN >> 3) << 17) | (uint32_t(kTM >> 4) << 24);
}

// D[128 x N] (+)= A[128 x 16] B[N x 16]^T; N a multiple of 16, at most 256;
// a, b: low words of the operands' descriptors.
template <int N>
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint32_t a, uint32_t b, uint32_t acc) {
  static_assert(N % 16 == 0 && N >= 16 && N <= 256, "tcgen05.mma kind::f16 with M = 128");
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %4, 0;\n"
      " mov.b64 da, {%1, %5};\n mov.b64 db, {%2, %5};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a), "r"(b), "r"(instr_desc<N>()), "r"(acc), "r"(kDescHi));
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// X 2^e rounded to nearest even, built from the IEEE fields: the FP64 pipe
// of this part issues about two operations per clock and SM, so a conversion
// and two products per output cost a 128 x 64 tile ~12000 cycles, more than
// the products of a K = 128 tile.  In 32-bit halves (half the instructions of
// 64-bit shifts and counts).  Results outside the normal range take the FP64
// route.
// (out: such a result, the value returned is not it)
__device__ __forceinline__ double scaled_double(long long X, int e, bool& out) {
  const long long sg = X >> 63;
  const unsigned long long u = (unsigned long long)((X ^ sg) - sg);
  const uint32_t uh = uint32_t(u >> 32), ul = uint32_t(u);
  const bool narrow = uh == 0;
  const uint32_t h = narrow ? ul : uh, l = narrow ? 0u : ul;
  const int lz = __clz(int(h));
  // normalised: leading bit at bit 63 (X = 0: no matter, 0 is returned)
  const uint32_t nh = __funnelshift_l(l, h, lz), nl = l << (lz & 31);
  const int ex = (narrow ? 1053 : 1085) - lz + e;  // biased exponent less one of the leading bit's weight
  const uint32_t tie = (nl >> 11) & 1u;
  const uint32_t up = (nl & 0x7ffu) + tie > 0x400u ? 1u : 0u;  // round to nearest, ties to even
  const unsigned long long m =
      ((unsigned long long)((uint32_t(ex) << 20) + (nh >> 11)) << 32 | __funnelshift_r(nl, nh, 11)) + up;
  out = u != 0 && (ex < 1 || ex > 2043);
  return u == 0 ? 0.0 : __longlong_as_double((long long)(m | ((unsigned long long)sg & 0x8000000000000000ull)));
}

__device__ __noinline__ double scaled_double_far(long long X, int e) {
  const int eh = max(-1022, min(1023, e >> 1)), el = max(-1022, min(1023, e - (e >> 1)));
  return double(X) * __longlong_as_double((long long)(eh + 1023) << 52) *
         __longlong_as_double((long long)(el + 1023) << 52);
}

// a b + c, 64 bits wide (modulo 2^64: the accumulators carry the patterns of
// the rounding constants below until their sum is taken off)
__device__ __forceinline__ unsigned long long mad_wide(int a, int b, unsigned long long c) {
  return (unsigned long long)((long long)a * b) + c;
}
// Adding 3 2^22 to an FP32 number of magnitude up to 2^22 rounds it to an
// integer and puts that in the low bits of the pattern: the conversion
// without the slow conversion instructions.
constexpr float kMagic = 12582912.0f;
constexpr int kMagicBits = 0x4B400000;

constexpr int kOutLd = 9;  // 8 columns (odd stride: rows fall on different banks)
template <int S, int TN>
struct Smem {
  alignas(1024) uint8_t stage[Cfg<S, TN>::kStages][Cfg<S, TN>::kStageBytes];
  long long out[kEpiWarps][32][kOutLd];  // per epilogue warp: 8 columns of its rows
  uint64_t full[Cfg<S, TN>::kStages], empty[Cfg<S, TN>::kStages];
  uint64_t acc_full[2], acc_empty[2];
  uint64_t acc34_empty;  // the epilogue has read d3, d4 of the previous tile
  uint64_t mma_drain;    // abort path: every product issued so far has completed
  uint32_t tmem_base;
  int abort_flag;
};

// Persistent: CTA b processes tiles b, b + gridDim.x, ... in the plan's tile
// order.  Every tile has at least one K chunk (the plan writes K == 0
// problems separately): the epilogue of a tile always waits for that tile's
// products, so no role runs two mbarrier phases ahead of another.  The three roles walk the same sequence of K chunks, counted across
// tiles (stage ring and mbarrier phases continue from tile to tile), and the
// epilogue of one tile overlaps the copies and products of the next: d0..d2
// are double-buffered per pair of chunks, d3 and d4 are released as soon as
// the epilogue has folded them into its integer accumulators.
template <int S, int TN>
__global__ void __launch_bounds__(kThreads, 1)
    ozaki_gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                      const Prob* __restrict__ probs, const Tile* __restrict__ tiles, int ntiles,
                      const int* __restrict__ expA, const int* __restrict__ expB, double* __restrict__ C, const Scatter sc, int* err, long long spin) {
  using CF = Cfg<S, TN>;
  constexpr int kStages = CF::kStages;
  constexpr int kStageBytes = CF::kStageBytes;
  constexpr int kBBytes = CF::kBBytes;
  constexpr int kColD3 = CF::kColD3;
  extern __shared__ uint8_t smem_raw[];
  Smem<S, TN>& sm = *reinterpret_cast<Smem<S, TN>*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sm.acc_full[b], 1);
      mbar_init(&sm.acc_empty[b], 32 * kEpiWarps);
    }
    mbar_init(&sm.acc34_empty, 32 * kEpiWarps);
    mbar_init(&sm.mma_drain, 1);
    sm.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)),
                 "r"(CF::kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // everything before this overlaps the end of the split or pack launch
  grid_wait();
  const uint32_t tmem = sm.tmem_base;
  volatile int* abort_flag = &sm.abort_flag;

  // Ring positions are counted as (stage, phase) and (buffer, phase) pairs:
  // the roles run one instruction stream each, so a 64-bit division by the
  // stage count per chunk is time the tensor core waits for.
  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      uint32_t s = 0, ph = 0;
      int issued = 0;  // chunks issued so far, up to kStages
      bool ok = true;
      Tile t = tiles[blockIdx.x];  // (the grid has at most ntiles CTAs)
      for (int ti = blockIdx.x; ti < ntiles && ok;) {
        ti += gridDim.x;
        const Tile nxt = ti < ntiles ? tiles[ti] : t;  // in flight during this tile
        for (int c = 0; c < t.nk; ++c) {
          if (issued == kStages && !mbar_wait(&sm.empty[s], ph ^ 1u, abort_flag, err, spin)) {
            ok = false;
            break;
          }
          issued += issued < kStages;
          mbar_expect_tx(&sm.full[s], kStageBytes);
          uint8_t* base = sm.stage[s];
          tma_load_3d(base, &mapA, c * kTK, t.arow, &sm.full[s]);
          tma_load_3d(base + S * kABytes, &mapB, c * kTK, t.brow, &sm.full[s]);
          if (++s == kStages) s = 0, ph ^= 1u;
        }
        t = nxt;
      }
      // every copy issued has landed before the CTA may exit, whichever
      // role aborted and when (after a normal run these phases are already
      // complete: the products consumed them)
      for (int i = 0; i < issued; ++i) {
        if (s == 0) s = kStages, ph ^= 1u;
        --s;
        for (long long w = 0; w < kDrainLimit && !mbar_try(&sm.full[s], ph); ++w) {
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    // d0..d2 are drained every pair of K chunks (64 K): their FP32 sums stay
    // exact integers below 2^24 (at most 3 * 64 products of magnitude
    // <= 2^16 per diagonal entry)
    if (lane == 0) {
    uint32_t s = 0, ph = 0;          // stage ring
    uint32_t buf = 0, bph = 0;       // d0..d2 buffers
    int pairs = 0;                   // pairs begun so far, up to 2
    uint32_t tph = 0;                // phase of acc34_empty
    bool ok = true, first_tile = true;
    bool have_full = false, have_buf = false;  // this chunk's waits found done ahead of time
    int nk = tiles[blockIdx.x].nk;
    for (int ti = blockIdx.x; ti < ntiles && ok;) {
      ti += gridDim.x;
      const int nk_next = ti < ntiles ? tiles[ti].nk : 0;
      for (int c = 0; c < nk; ++c) {
        const bool first = (c & 1) == 0;
        if (!have_full && !mbar_wait(&sm.full[s], ph, abort_flag, err, spin)) {
          ok = false;
          break;
        }
        if (first) {
          if (pairs == 2 && !have_buf && !mbar_wait(&sm.acc_empty[buf], bph ^ 1u, abort_flag, err, spin)) {
            ok = false;
            break;
          }
          if (S == 5 && c == 0 && !first_tile && !mbar_wait(&sm.acc34_empty, tph ^ 1u, abort_flag, err, spin)) {
            ok = false;
            break;
          }
          tc_fence_after();
        }
        const uint32_t sn = s + 1 == kStages ? 0u : s + 1, phn = s + 1 == kStages ? ph ^ 1u : ph;
        const uint32_t a0 = desc_lo(smem_u32(sm.stage[s]));
        const uint32_t b0 = a0 + ((S * kABytes) >> 4);
        // The slices of B are stacked in the stage (slice j: rows
        // j TN .. j TN + TN - 1), so B slices j .. j + n - 1 form one
        // operand of n TN rows; in tensor memory the diagonals of a
        // buffer lie side by side (d at buf 3 TN + d TN; d3, d4 at
        // kColD3).  A slice i times B slices j .. j + n - 1 thus adds into
        // diagonals i + j .. i + j + n - 1 with one product: 8 products
        // of width TN .. 3 TN per 16 K instead of 15 of width TN (S = 5),
        // 3 instead of 6 (S = 3), each reading its A slice once.
        const uint32_t cb = tmem + uint32_t(buf * 3 * TN);
        const uint32_t c3 = tmem + uint32_t(kColD3);
#pragma unroll
        for (int ks = 0; ks < kTK / 16; ++ks) {
          const uint32_t acc_b = (!first || ks > 0) ? 1u : 0u;  // first writer of d0..d2 in this pair
          const uint32_t acc_3 = (c > 0 || ks > 0) ? 1u : 0u;   // first writer of d3, d4 in this tile
          auto ad = [&](int i) { return a0 + uint32_t((i * kABytes + ks * 32) >> 4); };
          auto bd = [&](int j) { return b0 + uint32_t((j * kBBytes + ks * 32) >> 4); };
          // (d3, d4 accumulate with rounding: their products keep this
          // order; d0..d2 are exact.  The widest product goes first or last
          // so that the tensor core is busy longest around the waits.)
          if (ks == 0) mma_bf16<3 * TN>(cb, ad(0), bd(0), acc_b);           // d0 d1 d2 += A0 [B0 B1 B2]
          if constexpr (S == 5) mma_bf16<2 * TN>(c3, ad(0), bd(3), acc_3);  // d3 d4 += A0 [B3 B4]
          mma_bf16<2 * TN>(cb + TN, ad(1), bd(0), 1u);                      // d1 d2 += A1 [B0 B1]
          if constexpr (S == 5) mma_bf16<2 * TN>(c3, ad(1), bd(2), 1u);     // d3 d4 += A1 [B2 B3]
          mma_bf16<TN>(cb + 2 * TN, ad(2), bd(0), 1u);                      // d2 += A2 B0
          if (ks == 1) {
            // the next chunk's barriers, looked at while this one's products
            // queue: a wait that starts after the last product leaves the
            // tensor core idle for its latency
            have_full = mbar_test(&sm.full[sn], phn);
            have_buf = mbar_test(&sm.acc_empty[buf ^ 1u], buf ? bph : bph ^ 1u);
          }
          if constexpr (S == 5) {
            mma_bf16<2 * TN>(c3, ad(2), bd(1), 1u);            // d3 d4 += A2 [B1 B2]
            mma_bf16<2 * TN>(c3, ad(3), bd(0), 1u);            // d3 d4 += A3 [B0 B1]
            mma_bf16<TN>(c3 + TN, ad(4), bd(0), 1u);           // d4 += A4 B0
          }
          if (ks == 1) mma_bf16<3 * TN>(cb, ad(0), bd(0), 1u);
        }
        mma_commit(&sm.empty[s]);
        s = sn;
        ph = phn;
        if (!first || c == nk - 1) {
          mma_commit(&sm.acc_full[buf]);
          pairs += pairs < 2;
          buf ^= 1u;
          if (buf == 0) bph ^= 1u;
        }
      }
      first_tile = false;
      tph ^= 1u;
      nk = nk_next;
    }
    // every product issued has written tensor memory before it is freed,
    // whichever role aborted and when (the commit arrives once they have
    // all completed; with none issued, at once)
    mma_commit(&sm.mma_drain);
    for (long long i = 0; i < kDrainLimit && !mbar_try(&sm.mma_drain, 0); ++i) {
    }
    }
  } else {
    // ---------------- epilogue: warps 2..17 ----------------
    // warp w may access tensor-memory lanes 32*(w%4)..+31; the four warps of
    // a lane quarter split the TN columns (with two of them and twice the
    // columns each, a tile's waits, conversions and stores left the tensor
    // core waiting for its accumulators)
    constexpr int kCols = TN / 4;
    const int q = warp & 3;
    const int c0 = ((warp - 2) >> 2) * kCols;
    const int row = q * 32 + lane;
    const uint32_t lane_base = tmem + (uint32_t(q * 32) << 16);
    uint32_t buf = 0, bph = 0;
    // Each lane polls for itself, so when a wait expires, or another role has
    // aborted, some lanes of a warp may have seen the phase complete and
    // others not.  A lane that gave up does not leave its warp, whose loads,
    // shuffles and barriers need it: it walks on to the last tile, with no
    // more waits and nothing stored (a vote per wait instead cost an SU(2)
    // corner 2 %, 607 -> 620 us).
    bool ok = true;
    Tile t = tiles[blockIdx.x];
    for (int ti = blockIdx.x; ti < ntiles;) {
      ti += gridDim.x;
      const Tile nxt = ti < ntiles ? tiles[ti] : t;
      // the tile's rows and columns, loaded while its products run: lane l
      // holds row l's exponent and scatter entry, and those of the columns
      // that it writes, c0 + (l & 7) (+ 8).  Everything hangs on the tile
      // alone, which came with the one before: of a tile of one chunk the
      // chain tile - problem - tables was a good part.
      const int mrows = (t.m0 & (kTM - 1)) + 1 - q * 32, ncols = (t.n0 & (TN - 1)) + 1 - c0;
      const bool idle = mrows <= 0 || ncols <= 0;  // this warp's part lies past the problem
      const bool scatter = sc.rowtab != nullptr;
      const Prob* p = probs + t.prob;
      const int ea = lane < mrows ? expA[t.arow + row] - CF::kShift : 0;
      int2 ri = make_int2(0, 0);
      int ncc = 0;
      long long bb_off = 0;
      if (scatter) {
        if (!idle) ri = sc.rowtab[t.rt + q * 32 + min(lane, mrows - 1)];
        ncc = p->ncc;
        bb_off = p->bb_off;
      }
      // (the output block of this lane's first row in every 8 columns: offset
      // of the column's first row there, and the block's row length)
      const bool one_blk = __all_sync(0xffffffffu, ri.x == __shfl_sync(0xffffffffu, ri.x, 0));
      const int rx0 = __shfl_sync(0xffffffffu, ri.x, lane >> 3);
      int eb[kCols / 8], cw[kCols / 8];
      long long cb[kCols / 8];
#pragma unroll
      for (int h = 0; h < kCols / 8; ++h) {
        const int col = h * 8 + (lane & 7);
        eb[h] = cw[h] = 0;
        cb[h] = 0;
        if (col < ncols) {
          eb[h] = expB[t.brow + c0 + col];
          if (scatter) {
            const int4 ci = sc.coltab[t.ct + c0 + col];
            cw[h] = ci.z;
            cb[h] = sc.bbase[bb_off + (long long)rx0 * ncc + ci.x] + ci.y;
          }
        }
      }
      // X = sum over chunk pairs of (S0 2^18 + S1 2^9 + S2) 2^(9 if S = 5), plus
      // S3 + S4 2^-9: integers below 2^63, summed modulo 2^64
      constexpr int kUp = S == 5 ? 9 : 0;
      unsigned long long T[kCols];
#pragma unroll
      for (int j = 0; j < kCols; ++j) T[j] = 0;
      const int npair = (t.nk + 1) >> 1;
      for (int pp = 0; pp < npair; ++pp) {
        if (ok) ok = mbar_wait(&sm.acc_full[buf], bph, abort_flag, err, spin);
        tc_fence_after();
        if (idle) {
          mbar_arrive(&sm.acc_empty[buf]);
          buf ^= 1u;
          if (buf == 0) bph ^= 1u;
          continue;
        }
        // The three diagonals of 8 columns per wait; the buffer goes back
        // to the products as soon as its last load has landed, before the
        // conversions.  |S0| <= 64 2^16 = 2^22: adding 3 2^22 puts it in the
        // low bits of the FP32 pattern, so the patterns stand for S0 (npair
        // times the constant's pattern is taken off at the end) without the
        // slow conversion that S1 and S2 (up to 3 2^22) need.
#pragma unroll
        for (int h = 0; h < kCols; h += 8) {
          uint32_t v0[8], v1[8], v2[8];
          tmem_ld8(lane_base + buf * 3 * TN + 0 * TN + c0 + h, v0);
          tmem_ld8(lane_base + buf * 3 * TN + 1 * TN + c0 + h, v1);
          tmem_ld8(lane_base + buf * 3 * TN + 2 * TN + c0 + h, v2);
          tmem_wait_ld();
          if (h + 8 == kCols) {
            tc_fence_before();
            mbar_arrive(&sm.acc_empty[buf]);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            T[h + j] = mad_wide(__float_as_int(__uint_as_float(v0[j]) + kMagic), 1 << (18 + kUp), T[h + j]);
            T[h + j] = mad_wide(__float2int_rn(__uint_as_float(v1[j])), 1 << (9 + kUp), T[h + j]);
            T[h + j] = mad_wide(__float2int_rn(__uint_as_float(v2[j])), 1 << kUp, T[h + j]);
          }
        }
        buf ^= 1u;
        if (buf == 0) bph ^= 1u;
      }
      if (idle) {
        if constexpr (S == 5) mbar_arrive(&sm.acc34_empty);
        t = nxt;
        continue;
      }
      // d3 and d4 go back to the next tile's products, which wait for them,
      // before any output is written.  S3 + S4 2^-9 to the nearest integer as
      // 2^12 H + R, both by the constant (|S3| <= 4 K 2^16 < 2^32 for K up to
      // kMaxK, S4 2^-9 is at most 1/400 of that: |H| stays far below 2^22)
      const unsigned long long off = (((unsigned long long)npair * kMagicBits) << (18 + kUp)) +
                                     (S == 5 ? (unsigned long long)kMagicBits * 4097 : 0);
#pragma unroll
      for (int h = 0; h < kCols; h += 8) {
        if constexpr (S == 5) {
          uint32_t w3[8], w4[8];
          tmem_ld8(lane_base + kColD3 + 0 * TN + c0 + h, w3);
          tmem_ld8(lane_base + kColD3 + 1 * TN + c0 + h, w4);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float x = fmaf(__uint_as_float(w4[j]), 1.0f / 512.0f, __uint_as_float(w3[j]));
            const float hc = fmaf(x, 1.0f / 4096.0f, kMagic);
            const float r = fmaf(hc - kMagic, -4096.0f, x);  // exact, at most 2^11
            T[h + j] = mad_wide(__float_as_int(hc), 4096, T[h + j]);
            T[h + j] = mad_wide(__float_as_int(r + kMagic), 1, T[h + j]);
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) T[h + j] -= off;
      }
      if constexpr (S == 5) {
        tc_fence_before();
        mbar_arrive(&sm.acc34_empty);
      }
      // C = X 2^(ea + eb - shift).  A lane holds a row of 8 or 16 columns,
      // which written by itself would touch 32 lines per store: 8 columns at
      // a time go through shared memory, and a store writes 8 columns of
      // four rows.  Scatter: straight into the output tensor's canonical
      // blocks, row (ri.x, ri.y) and column (ci.x, ci.y) of the block (ri.x,
      // ci.x) of width ci.z; else the sector matrix.
      long long(*st)[kOutLd] = sm.out[warp - 2];
      const bool plain = !scatter || (sc.alpha == 1.0 && sc.beta == 0.0);
#pragma unroll
      for (int h = 0; h < kCols / 8; ++h) {
        if (h * 8 >= ncols) break;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j) st[lane][j] = (long long)T[h * 8 + j];
        __syncwarp();
        const int col = h * 8 + (lane & 7);
        const bool col_ok = col < ncols && ok;
        double* cbase;
        int rstride;  // between output rows of a block
        if (scatter) {
          cbase = C + cb[h];
          rstride = cw[h];
        } else {
          rstride = int(p->c_m);
          cbase = C + p->c_off + (long long)((t.m0 & ~(kTM - 1)) + q * 32) * rstride +
                  (long long)((t.n0 & ~(TN - 1)) + c0 + col) * p->c_n;
        }
        // (the values of four rows side by side: the shared load, shuffle and
        // conversion of one are a chain that four warps a scheduler do not
        // hide)
        constexpr int kRows = 4;
#pragma unroll
        for (int g = 0; g < 8 / kRows; ++g) {
          if (4 * kRows * g >= mrows) break;
          const int r0 = 4 * kRows * g + (lane >> 3);  // rows r0, r0 + 4, ..
          double v[kRows];
          double* dst[kRows];
          bool far = false, out[kRows];
#pragma unroll
          for (int i = 0; i < kRows; ++i) {
            const int r = r0 + 4 * i;
            dst[i] = cbase + (long long)(scatter ? __shfl_sync(0xffffffffu, ri.y, r) : r) * rstride;
            v[i] = scaled_double(st[r][lane & 7], __shfl_sync(0xffffffffu, ea, r) + eb[h], out[i]);
            far = far || out[i];
          }
          if (__any_sync(0xffffffffu, far)) {
#pragma unroll 1
            for (int i = 0; i < kRows; ++i) {
              const int r = r0 + 4 * i;
              const double x = scaled_double_far(st[r][lane & 7], __shfl_sync(0xffffffffu, ea, r) + eb[h]);
#pragma unroll
              for (int k = 0; k < kRows; ++k)
                if (k == i && out[k]) v[k] = x;
            }
          }
          if (!one_blk) {  // (rows of several blocks: the columns' table entries again)
            const int4 ci = col_ok ? sc.coltab[t.ct + c0 + col] : make_int4(0, 0, 0, 0);
            const long long* bb = sc.bbase + p->bb_off + ci.x;
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
              const int rx = __shfl_sync(0xffffffffu, ri.x, r0 + 4 * i), my = __shfl_sync(0xffffffffu, ri.y, r0 + 4 * i);
              if (col_ok) dst[i] = C + bb[(long long)rx * p->ncc] + ci.y + (long long)my * rstride;
            }
          }
#pragma unroll
          for (int i = 0; i < kRows; ++i) {
            if (col_ok && r0 + 4 * i < mrows) {
              if (plain) *dst[i] = v[i];
              else *dst[i] = sc.beta == 0.0 ? sc.alpha * v[i] : fma(sc.alpha, v[i], sc.beta * *dst[i]);
            }
          }
        }
      }
      t = nxt;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(CF::kTmemCols));
  }
}

// The outputs of problems with no matched block pair (K == 0), written by
// the last CTAs of the split or pack launch: beta * C through the scatter
// tables, or zeros into the sector matrices of a plain plan.  Single-layer
// moves leave hundreds of MB of them (charges that the contracted
// legs do not reach), so a CTA takes whole rows of about 4096
// elements and their number follows the size: with 8 CTAs a problem the D=8,
// chi=192 absorption (60 M such elements beside 20 M to pack) took 3.5 ms,
// now 0.28 ms, and the whole left move 84 -> 66 ms.
constexpr int kZeroElems = 4096;  // elements of a CTA
struct ZeroCta {
  int prob, m0, m1;       // rows [m0, m1) of a problem (an index into zidx or zp)
};
struct ZeroJob {
  int n;                  // CTAs
  const ZeroCta* ctas;
  const Prob* probs;      // scatter form: problems listed by zidx
  const int* zidx;
  Scatter sc;
  const GemmProb* zp;     // plain form (probs == nullptr)
  double* C;
};

__device__ __forceinline__ void zero_part(const ZeroJob& z, int cta) {
  const ZeroCta zc = z.ctas[cta];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  // lanes along a row; several rows a warp where they are short
  auto each = [&](int N, auto&& row) {
    const int lpr = N > 16 ? 32 : N > 8 ? 16 : N > 4 ? 8 : 4;
    for (int m = zc.m0 + warp * (32 / lpr) + lane / lpr; m < zc.m1; m += nw * (32 / lpr)) row(m, lane % lpr, lpr);
  };
  if (z.probs) {
    const Prob p = z.probs[z.zidx[zc.prob]];
    each(p.N, [&](int m, int c0, int step) {
      const int2 ri = z.sc.rowtab[p.rt_off + m];
      const long long* base = z.sc.bbase + p.bb_off + (long long)ri.x * p.ncc;
      for (int c = c0; c < p.N; c += step) {
        const int4 ci = z.sc.coltab[p.ct_off + c];
        const long long dst = base[ci.x] + (long long)ri.y * ci.z + ci.y;
        z.C[dst] = z.sc.beta == 0.0 ? 0.0 : z.sc.beta * z.C[dst];
      }
    });
  } else {
    const GemmProb p = z.zp[zc.prob];
    each(p.N, [&](int m, int c0, int step) {
      for (int c = c0; c < p.N; c += step) z.C[p.c_off + m * p.c_m + c * p.c_n] = 0.0;
    });
  }
}

// Split FP64 rows into S BF16 digit slices (integer arithmetic on the bit
// pattern); digits for k in [K, roundup(K, 32)) are 0.  One launch splits
// both operands: CTAs [0, ga) take the tasks of A, the next gb those of B;
// a table gives every CTA its task (a search over hundreds of tasks is a
// chain of that many loads, longer than the CTA's work).
//
// The kernel moves 8 bytes in and 2 S out per element (80 registers for three
// CTAs an SM, as the pack below), so what bounds it is how the rows lie in
// memory:
//   * rows contiguous along k (s_k = 1): four consecutive k per lane (two
//     16-byte loads where the row is 16-byte aligned, 8-byte stores).  Rows
//     up to 512 long stay in registers between the maximum and the digits;
//     longer ones are read again;
//   * rows interleaved (s_r = 1, the columns of a row-major block, as every
//     product with the iterated block has them): lanes along the rows, 16
//     consecutive k per thread, so the loads of a warp are 256 contiguous
//     bytes and every thread stores whole 32-byte sectors.  A cluster of up
//     to 8 CTAs shares the k range of 32 rows and exchanges the row maxima
//     through distributed shared memory: one launch, no atomics.  With lanes
//     along k instead, as for contiguous rows, every load of a warp touched
//     32 sectors of which 8 bytes each were used.
struct SplitJob {
  const SplitTask* tasks;
  const int2* ctas;  // per CTA: its task and its number inside it
  int rows_total;
  const double* X;
  __nv_bfloat16* S;
  int* ex;
};

constexpr int kSplitThreads = 256;
constexpr int kSplitRowMax = 512;  // longest contiguous row kept in registers (4 x 4 per lane)

// The digits of the value with bit pattern b against the row exponent e
// (|x| < 2^e), as the bit patterns of the FP32 numbers (BF16 in the upper
// half): X = round(|x| 2^(9 S - 1 - e)) with the sign of x, X = sum_i a_i
// 2^(9 (S - 1 - i)) with a_i in [-256, 255] for i > 0.  Adding 256 at every
// digit but the first makes those bit fields; a field under the pattern of
// 1.5 2^23 is that number plus the field, so one subtraction gives the digit.
template <int S>
__device__ __forceinline__ void split_digits(unsigned long long b, int e, uint32_t (&f)[S]) {
  const uint32_t hi = uint32_t(b >> 32);
  const int E = int(hi >> 20) & 0x7FF;
  // E <= e + 1022 and 9 S - 1 <= 44: the shift is to the right by 9 or more
  const int rs = 1074 + e - (9 * S - 1) - E;
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  long long X = (long long)(((m >> (rs & 63)) + 1) >> 1);  // half a unit up: round to nearest
  if (rs > 62 || E == 0) X = 0;  // (subnormals of a row with a normal maximum are below 2^-44 of it)
  if (int(hi) < 0) X = -X;
  long long bias = 0;
#pragma unroll
  for (int i = 0; i < S - 1; ++i) bias |= 256ll << (9 * i);
  X += bias;
#pragma unroll
  for (int i = S - 1; i >= 1; --i)
    f[i] = __float_as_uint(__uint_as_float((uint32_t(X >> (9 * (S - 1 - i))) & 511u) | 0x4B400000u) - 12583168.0f);
  f[0] = __float_as_uint(__uint_as_float(0x4B400000u + uint32_t(int(X >> (9 * (S - 1))))) - 12582912.0f);
}

// two BF16 numbers (the upper halves of their FP32 patterns), lower k first
__device__ __forceinline__ uint32_t pack_bf16(uint32_t lo, uint32_t hi) { return __byte_perm(lo, hi, 0x7632); }

// |x|'s upper word: enough for a row's exponent
__device__ __forceinline__ uint32_t abs_hi(unsigned long long b) { return uint32_t(b >> 32) & 0x7FFFFFFFu; }
__device__ __forceinline__ int row_exp(uint32_t mx) { return int(mx >> 20) - 1022; }  // |x| < 2^e

// The digits of 16 consecutive k of one row.
template <int S>
__device__ __forceinline__ void store16(__nv_bfloat16* Sd, int rows_total, long long grow, int kpitch, int k, int e,
                                        const unsigned long long (&x)[16]) {
#pragma unroll
  for (int h = 0; h < 16; h += 8) {
    uint32_t w[4][S];
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      uint32_t f[S], g[S];
      split_digits<S>(x[h + j], e, f);
      split_digits<S>(x[h + j + 1], e, g);
#pragma unroll
      for (int i = 0; i < S; ++i) w[j / 2][i] = pack_bf16(f[i], g[i]);
    }
#pragma unroll
    for (int i = 0; i < S; ++i)
      *reinterpret_cast<uint4*>(Sd + ((long long)i * rows_total + grow) * kpitch + k + h) =
          make_uint4(w[0][i], w[1][i], w[2][i], w[3][i]);
  }
}

// Rows contiguous along k: how many a CTA takes.  Four k per lane: rows up
// to 32 (64, 128) long take 8 (16, 32) lanes and a warp does four passes of
// 4 (2, 1) rows, all loads first; longer rows take a warp each.
__host__ __device__ inline int split_cta_rows(int K) {
  const int per_warp = K <= 32 ? 16 : K <= 64 ? 8 : K <= 128 ? 4 : 1;
  return per_warp * (kSplitThreads / 32);
}

template <int S>
__device__ __forceinline__ void split_rows(const SplitJob& J, const SplitTask& tk, int cta, int kpitch) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kend = (tk.K + 31) & ~31;
  auto load4 = [&](const double* xr, int k, unsigned long long (&v)[4]) {
    if (k + 3 < tk.K && (reinterpret_cast<uintptr_t>(xr) & 15) == 0) {
      const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(xr + k);
      const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(xr + k + 2);
      v[0] = p.x, v[1] = p.y, v[2] = q.x, v[3] = q.y;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        v[j] = k + j < tk.K ? (unsigned long long)__double_as_longlong(xr[k + j]) : 0ull;
    }
  };
  auto store4 = [&](long long grow, int k, int e, const unsigned long long (&v)[4]) {
    uint32_t f[4][S];
#pragma unroll
    for (int j = 0; j < 4; ++j) split_digits<S>(v[j], e, f[j]);
#pragma unroll
    for (int i = 0; i < S; ++i)
      *reinterpret_cast<uint2*>(J.S + ((long long)i * J.rows_total + grow) * kpitch + k) =
          make_uint2(pack_bf16(f[0][i], f[1][i]), pack_bf16(f[2][i], f[3][i]));
  };
  unsigned long long x[4][4];
  if (tk.K <= 128) {
    const int lpr = tk.K <= 32 ? 8 : tk.K <= 64 ? 16 : 32;  // lanes per row
    const int rpw = 32 / lpr, k = (lane % lpr) * 4;
    const int r0 = (cta * (kSplitThreads / 32) + warp) * 4 * rpw + lane / lpr;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int r = r0 + it * rpw;
      if (r < tk.rows) load4(J.X + tk.base + (long long)r * tk.s_r, k, x[it]);
      else x[it][0] = x[it][1] = x[it][2] = x[it][3] = 0;
    }
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      uint32_t mx = max(max(abs_hi(x[it][0]), abs_hi(x[it][1])),
                                  max(abs_hi(x[it][2]), abs_hi(x[it][3])));
      for (int o = lpr >> 1; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      // |x| < 2^e for every entry of the row (e from the largest exponent field)
      const int e = row_exp(mx);
      const int r = r0 + it * rpw;
      if (r >= tk.rows) continue;
      if (k == 0) J.ex[tk.row0 + r] = e;
      if (k < kend) store4(tk.row0 + r, k, e, x[it]);
    }
    return;
  }
  const int r = cta * (kSplitThreads / 32) + warp;
  if (r >= tk.rows) return;
  const double* xr = J.X + tk.base + (long long)r * tk.s_r;
  uint32_t mx = 0;
  const bool keep = tk.K <= kSplitRowMax;
  if (keep) {
#pragma unroll
    for (int g = 0; g < 4; ++g) load4(xr, g * 128 + lane * 4, x[g]);
#pragma unroll
    for (int g = 0; g < 4; ++g)
#pragma unroll
      for (int j = 0; j < 4; ++j) mx = max(mx, abs_hi(x[g][j]));
  } else {
#pragma unroll 4
    for (int k = lane; k < tk.K; k += 32) mx = max(mx, abs_hi(__double_as_longlong(xr[k])));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int e = row_exp(mx);
  const long long grow = tk.row0 + r;
  if (lane == 0) J.ex[grow] = e;
  if (keep) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int k = g * 128 + lane * 4;
      if (k < kend) store4(grow, k, e, x[g]);
    }
  } else {
    for (int k = lane * 4; k < kend; k += 128) {
      unsigned long long v[4];
      load4(xr, k, v);
      store4(grow, k, e, v);
    }
  }
}

// One cluster, 32 interleaved rows (lane l: row r0 + l at xr[k s_k]).
template <int S>
__device__ __forceinline__ void split_cols(const SplitJob& J, const SplitTask& tk, int r0, int crank, int csize,
                                           int kpitch) {
  __shared__ uint32_t wmax[kSplitThreads / 32][32];
  __shared__ uint32_t cmax[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = r0 + lane;
  const bool live = r < tk.rows;
  const double* xr = J.X + tk.base + (live ? r : tk.rows - 1);
  const int step = csize * (kSplitThreads / 32) * 16;        // k per pass of the cluster
  const int k0 = (crank * (kSplitThreads / 32) + warp) * 16;  // this thread's first 16
  auto load16 = [&](int k, unsigned long long (&v)[16]) {
#pragma unroll
    for (int j = 0; j < 16; ++j)
      v[j] = k + j < tk.K ? (unsigned long long)__double_as_longlong(xr[(long long)(k + j) * tk.s_k]) : 0ull;
  };
  unsigned long long x[16];
  uint32_t mx = 0;
  // the first pass's values stay in registers (the only pass when the
  // cluster covers K), the others are read again below
  load16(k0, x);
#pragma unroll
  for (int j = 0; j < 16; ++j) mx = max(mx, abs_hi(x[j]));
  for (int k = k0 + step; k < tk.K; k += step) {
    unsigned long long v[16];
    load16(k, v);
#pragma unroll
    for (int j = 0; j < 16; ++j) mx = max(mx, abs_hi(v[j]));
  }
  wmax[warp][lane] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kSplitThreads / 32; ++w) mx = max(mx, wmax[w][lane]);
  if (csize > 1) {
    cg::cluster_group cl = cg::this_cluster();
    if (warp == 0) cmax[lane] = mx;
    cl.sync();
    for (int c = 0; c < csize; ++c) mx = max(mx, cl.map_shared_rank(cmax, c)[lane]);
    cl.sync();  // no CTA leaves while another still reads its maxima
  }
  const int e = row_exp(mx);
  const long long grow = tk.row0 + r;
  if (live && crank == 0 && warp == 0) J.ex[grow] = e;
  if (!live) return;
  const int kend = (tk.K + 31) & ~31;
  for (int k = k0; k < kend; k += step) {
    if (k != k0) load16(k, x);
    store16<S>(J.S, J.rows_total, grow, kpitch, k, e, x);
  }
}

template <int S>
__global__ void __launch_bounds__(kSplitThreads, 3) ozaki_split_kernel(SplitJob ja, SplitJob jb, int ga, int gab,
                                                                    int csize, int kpitch, ZeroJob zj) {
  grid_trigger();
  if (int(blockIdx.x) >= gab) {
    const int z = int(blockIdx.x) - gab;
    if (z < zj.n) zero_part(zj, z);
    return;
  }
  const bool is_a = int(blockIdx.x) < ga;
  const SplitJob& J = is_a ? ja : jb;
  const int2 tc = J.ctas[int(blockIdx.x) - (is_a ? 0 : ga)];
  const SplitTask tk = J.tasks[tc.x];
  const int c = tc.y;
  if (tk.s_k != 1 && tk.s_r == 1) {
    // (a task's CTAs are whole clusters: the branch is the same for all of one)
    const int r0 = (c / csize) * 32;
    if (r0 < tk.rows) split_cols<S>(J, tk, r0, c % csize, csize, kpitch);
    return;
  }
  if (tk.s_k == 1) {
    split_rows<S>(J, tk, c, kpitch);
    return;
  }
  const int r = c * (kSplitThreads / 32) + int(threadIdx.x >> 5);
  if (r >= tk.rows) return;
  // any other strides: one warp per row, lanes along k
  const int lane = threadIdx.x & 31;
  const double* xr = J.X + tk.base + (long long)r * tk.s_r;
  uint32_t mx = 0;
  for (int k = lane; k < tk.K; k += 32) mx = max(mx, abs_hi(__double_as_longlong(xr[(long long)k * tk.s_k])));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int e = row_exp(mx);
  const long long grow = tk.row0 + r;
  if (lane == 0) J.ex[grow] = e;
  for (int k = lane; k < ((tk.K + 31) & ~31); k += 32) {
    uint32_t f[S];
    split_digits<S>(k < tk.K ? (unsigned long long)__double_as_longlong(xr[(long long)k * tk.s_k]) : 0ull, e, f);
#pragma unroll
    for (int i = 0; i < S; ++i)
      J.S[((long long)i * J.rows_total + grow) * kpitch + k] = __ushort_as_bfloat16((unsigned short)(f[i] >> 16));
  }
}

// Gather and split in one pass: the rows of an operand's sector matrices are
// read straight from the tensor's canonical blocks, and only their digits
// are written (8 bytes in, 2 S out per element; a gather followed by a split
// moves 16 + 8 + 2 S).  A row of sector s and row configuration r meets one
// block per column configuration c (a segment [k0, k0 + w) of the row);
// inside block (r, c) the element of row mi and column kk sits at  off +
// sum_rowlegs idx * str + sum_collegs idx * str, the indices from mi and kk
// row-major over the legs in matrix order.
//
// The loads coalesce when the lanes run along the tensor's innermost leg, so
// a group (one sector and row configuration) is read in one of two ways:
//   * innermost leg contracted: lanes along k, four k per lane (as
//     split_rows, several short rows per warp);
//   * innermost leg open: lanes along the rows of the group, 16 consecutive
//     k per thread (as split_cols).  Up to 128 k, the 8 warps of a CTA take
//     8, 4, 2 or 1 blocks of 32 rows; a block of more k is shared by up to 8
//     CTAs of a cluster, which exchange the row maxima, so that values wait
//     for them in registers.  Past 1024 k a thread's later passes are read
//     again (from cache).
// An element's address is that of its row in the segment's block plus an
// offset of k alone: a CTA tabulates both in shared memory (up to 1024 k and
// 4096 rows x segments at a time), so the index arithmetic over the legs is
// paid once per row and segment and once per k, not per element.
//
// What bounds it: the latency of the loads (9 of 16 cycles that a warp waits per issue),
// with 24 warps an SM (80 registers: the five-digit form spills some 90 bytes;
// with two CTAs and none of it the D=8, chi=192 move takes 3 % longer, a half
// system in three digits 49 us instead of 44, the batch as long), at a third of
// the memory's rate.  Against the gather and split it replaced:
// the batch of 64 corners 3.30 -> 2.05 ms, the D=6 corner (22 MB) 0.045 ->
// 0.029 ms, the D=8, chi=192 single-layer move's contractions 44 -> 28 ms;
// with the innermost leg contracted, 2432 x 2432 twice, 200 -> 90 us.
struct PackGroup {
  int32_t row0;         // its first row in the split buffer
  int32_t h, K;         // rows of this (sector, row configuration), columns
  int64_t seg0;         // its segments (one per column configuration), k0 ascending
  int32_t nseg, along;  // along: 0 lanes along k, 1 lanes along the rows
  int32_t pad;
};

struct alignas(16) PackLeg {
  int32_t dim, str;     // extent, stride inside the block
  uint32_t fm, fl;      // FastDiv of dim
};

struct PackSeg {
  int64_t off;          // block offset in its tensor (elements)
  int32_t k0;           // its first column of the row
  int32_t nr, nc;       // row legs, column legs
  int32_t src;          // index of the tensor in the job's pointer table
  PackLeg leg[kMaxRank];  // row legs then column legs, matrix order
};

struct PackJob {
  const PackGroup* groups;
  const PackSeg* segs;
  const int2* ctas;            // per CTA: its group and its number inside it
  int rows_total;              // rows of the split buffer (slice stride)
  const double* src;           // the operand tensor (tab == nullptr)
  const double* const* tab;    // per-segment tensors (batched contractions)
  __nv_bfloat16* S;
  int* ex;
};

__device__ __forceinline__ uint32_t fdiv(uint32_t n, uint32_t m, uint32_t l) { return (__umulhi(n, m) + n) >> l; }

// CTAs of a group
__host__ __device__ inline int pack_col_warps(int K) { return K <= 16 ? 1 : K <= 32 ? 2 : K <= 64 ? 4 : 8; }
// CTAs along k of one block of rows: enough for one pass of 128 k each, as
// far as the cluster goes (powers of two)
__host__ __device__ inline int pack_col_ctas(int K, int csize) {
  int c = 1;
  while (c < csize && c * 128 < K) c *= 2;
  return c;
}
inline int pack_ctas(int h, int K, int along, int csize) {
  if (!along) return ((h + split_cta_rows(K) - 1) / split_cta_rows(K) + csize - 1) / csize * csize;
  const int blocks = (h + 31) / 32, per = 8 / pack_col_warps(K);
  return ((blocks + per - 1) / per * pack_col_ctas(K, csize) + csize - 1) / csize * csize;
}

constexpr int kPackTab = 1024;   // k per table
constexpr int kPackRows = 4096;  // rows x segments per table
constexpr int kPackSegs = 128;   // segments searched on chip

struct PackShared {
  int2 k[kPackTab];                 // element offset inside the block, segment of the table
  const double* row[kPackRows];     // [segment][row]: the row's first element in the segment's block
  uint32_t wmax[kSplitThreads / 32][32];
  uint32_t cmax[32];
  int k0[kPackSegs];
};

// Tables of R rows from r0 for k in [kc, kb); returns the end of their k
// range (kb, or a multiple of 32 past kc).
__device__ __forceinline__ int pack_table(PackShared& sm, const PackJob& J, const PackGroup& G, int r0, int R, int kc,
                                          int kb) {
  const PackSeg* segs = J.segs + G.seg0;
  // the segments' first k, so that the searches below stay on chip (groups
  // of more than kPackSegs segments search the rest in memory)
  for (int i = int(threadIdx.x); i < min(G.nseg, kPackSegs); i += kSplitThreads) sm.k0[i] = segs[i].k0;
  __syncthreads();
  auto seg_of = [&](int k) {
    int lo = 0, hi = G.nseg - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if ((mid < kPackSegs ? sm.k0[mid] : segs[mid].k0) <= k) lo = mid;
      else hi = mid - 1;
    }
    return lo;
  };
  const int s0 = seg_of(kc), smax = s0 + kPackRows / R;
  int ke = min(kb, kc + kPackTab);
  if (smax < G.nseg) ke = min(ke, segs[smax].k0);
  if (ke < kb) ke = kc + ((ke - kc) & ~31);
  const int s1 = seg_of(ke - 1) + 1;
  for (int k = kc + int(threadIdx.x); k < ke; k += kSplitThreads) {
    const int si = seg_of(k);
    const PackSeg& sg = segs[si];
    uint32_t rem = uint32_t(k - sg.k0);
    int o = 0;
    for (int j = sg.nr + sg.nc - 1; j >= sg.nr; --j) {
      const PackLeg l = sg.leg[j];
      const uint32_t q = fdiv(rem, l.fm, l.fl);
      o += int(rem - q * uint32_t(l.dim)) * l.str;
      rem = q;
    }
    sm.k[k - kc] = make_int2(o, si - s0);
  }
  for (int t = int(threadIdx.x); t < (s1 - s0) * R; t += kSplitThreads) {
    const int si = t / R;
    const PackSeg& sg = segs[s0 + si];
    uint32_t rem = uint32_t(min(r0 + t - si * R, G.h - 1));
    long long o = sg.off;
    for (int j = sg.nr - 1; j >= 0; --j) {
      const PackLeg l = sg.leg[j];
      const uint32_t q = fdiv(rem, l.fm, l.fl);
      o += (long long)(rem - q * uint32_t(l.dim)) * l.str;
      rem = q;
    }
    sm.row[t] = (J.tab ? J.tab[sg.src] : J.src) + o;
  }
  __syncthreads();
  return ke;
}

// n consecutive elements of table row r from k on (zeros from ke on)
template <int n>
__device__ __forceinline__ void pack_load(const PackShared& sm, int r, int R, int k, int kc, int ke,
                                          unsigned long long (&v)[n]) {
#pragma unroll
  for (int j = 0; j < n; ++j) {
    v[j] = 0ull;
    if (k + j < ke) {
      const int2 t = sm.k[k + j - kc];
      v[j] = (unsigned long long)__double_as_longlong(__ldg(sm.row[t.y * R + r] + t.x));
    }
  }
}

template <int S>
__device__ __forceinline__ void pack_rows(PackShared& sm, const PackJob& J, const PackGroup& G, int cta, int kpitch) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int R = split_cta_rows(G.K), r0 = cta * R;
  const int kend = (G.K + 31) & ~31;
  auto store4 = [&](int mi, int k, int e, const unsigned long long (&v)[4]) {
    uint32_t f[4][S];
#pragma unroll
    for (int j = 0; j < 4; ++j) split_digits<S>(v[j], e, f[j]);
#pragma unroll
    for (int i = 0; i < S; ++i)
      *reinterpret_cast<uint2*>(J.S + ((long long)i * J.rows_total + G.row0 + mi) * kpitch + k) =
          make_uint2(pack_bf16(f[0][i], f[1][i]), pack_bf16(f[2][i], f[3][i]));
  };
  int ke = pack_table(sm, J, G, r0, R, 0, G.K);
  unsigned long long x[4][4];
  if (G.K <= 128) {  // (at most 128 segments: one table)
    const int lpr = G.K <= 32 ? 8 : G.K <= 64 ? 16 : 32;  // lanes per row
    const int rpw = 32 / lpr, k = (lane % lpr) * 4;
    const int lr = warp * 4 * rpw + lane / lpr;
#pragma unroll
    for (int it = 0; it < 4; ++it) pack_load(sm, lr + it * rpw, R, k, 0, ke, x[it]);
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      uint32_t mx = max(max(abs_hi(x[it][0]), abs_hi(x[it][1])), max(abs_hi(x[it][2]), abs_hi(x[it][3])));
      for (int o = lpr >> 1; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const int e = row_exp(mx);
      const int r = r0 + lr + it * rpw;
      if (r >= G.h) continue;
      if (k == 0) J.ex[G.row0 + r] = e;
      if (k < kend) store4(r, k, e, x[it]);
    }
    return;
  }
  const int r = r0 + warp;
  uint32_t mx = 0;
  const bool one = ke == G.K, keep = one && G.K <= kSplitRowMax;
  if (keep) {
#pragma unroll
    for (int g = 0; g < 4; ++g) pack_load(sm, warp, R, g * 128 + lane * 4, 0, ke, x[g]);
#pragma unroll
    for (int g = 0; g < 4; ++g)
#pragma unroll
      for (int j = 0; j < 4; ++j) mx = max(mx, abs_hi(x[g][j]));
  } else {
    for (int kc = 0;;) {
      for (int k = kc + lane * 4; k < ke; k += 512) {
#pragma unroll
        for (int g = 0; g < 4; ++g) pack_load(sm, warp, R, k + g * 128, kc, ke, x[g]);
#pragma unroll
        for (int g = 0; g < 4; ++g)
#pragma unroll
          for (int j = 0; j < 4; ++j) mx = max(mx, abs_hi(x[g][j]));
      }
      if (ke == G.K) break;
      __syncthreads();
      kc = ke;
      ke = pack_table(sm, J, G, r0, R, kc, G.K);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int e = row_exp(mx);
  if (lane == 0 && r < G.h) J.ex[G.row0 + r] = e;
  if (keep) {
    if (r >= G.h) return;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int k = g * 128 + lane * 4;
      if (k < kend) store4(r, k, e, x[g]);
    }
    return;
  }
  for (int kc = 0; kc < G.K; kc = ke) {
    if (!one) {
      __syncthreads();
      ke = pack_table(sm, J, G, r0, R, kc, G.K);
    }
    if (r >= G.h) continue;
    for (int k = kc + lane * 4; k < ((ke + 31) & ~31); k += 512) {
#pragma unroll
      for (int g = 0; g < 4; ++g) pack_load(sm, warp, R, k + g * 128, kc, ke, x[g]);
#pragma unroll
      for (int g = 0; g < 4; ++g)
        if (k + g * 128 < ((ke + 31) & ~31)) store4(r, k + g * 128, e, x[g]);
    }
  }
}

template <int S>
__device__ __forceinline__ void pack_cols(PackShared& sm, const PackJob& J, const PackGroup& G, int cta, int csize,
                                          int kpitch) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wk = pack_col_warps(G.K);       // warps along k of one block of 32 rows
  const int cpb = pack_col_ctas(G.K, csize);  // CTAs along k of one block
  const int first = warp - warp % wk;
  const int R = 8 / wk * 32, r0 = cta / cpb * R;
  const int lr = warp / wk * 32 + lane, mi = r0 + lr;
  const bool live = mi < G.h;
  // this CTA's k: one pass of 128 (or of all, below) where cpb covers K
  const int kr = (G.K + 128 * cpb - 1) / (128 * cpb) * 128;
  const int ka = cta % cpb * kr, kb = min(G.K, ka + kr);
  const int k0 = (warp % wk) * 16, step = wk * 16;
  unsigned long long x[16];
  uint32_t mx = 0;
  int ke = kb;
  bool one = true;  // one table holds the CTA's k
  if (ka < kb) {
    ke = pack_table(sm, J, G, r0, R, ka, kb);
    one = ke == kb;
    pack_load(sm, lr, R, ka + k0, ka, ke, x);
#pragma unroll
    for (int j = 0; j < 16; ++j) mx = max(mx, abs_hi(x[j]));
    for (int kc = ka;;) {
      for (int k = kc + k0 + (kc == ka ? step : 0); k < ke; k += step) {
        unsigned long long v[16];
        pack_load(sm, lr, R, k, kc, ke, v);
#pragma unroll
        for (int j = 0; j < 16; ++j) mx = max(mx, abs_hi(v[j]));
      }
      if (ke == kb) break;
      __syncthreads();
      kc = ke;
      ke = pack_table(sm, J, G, r0, R, kc, kb);
    }
  }
  sm.wmax[warp][lane] = mx;
  __syncthreads();
  for (int c = 0; c < wk; ++c) mx = max(mx, sm.wmax[first + c][lane]);
  if (cpb > 1) {
    // (wk is 8: the CTA holds one block; all of a cluster take this branch)
    cg::cluster_group cl = cg::this_cluster();
    if (warp == 0) sm.cmax[lane] = mx;
    cl.sync();
    const int base = int(cl.block_rank()) - cta % cpb;
    for (int c = 0; c < cpb; ++c) mx = max(mx, cl.map_shared_rank(sm.cmax, base + c)[lane]);
    cl.sync();  // no CTA leaves while another still reads its maxima
  }
  const int e = row_exp(mx);
  const long long grow = G.row0 + mi;
  if (live && warp == first && ka == 0) J.ex[grow] = e;
  for (int kc = ka; kc < kb; kc = ke) {
    if (!one) {
      __syncthreads();
      ke = pack_table(sm, J, G, r0, R, kc, kb);
    }
    if (!live) continue;
    for (int k = kc + k0; k < ((ke + 31) & ~31); k += step) {
      if (k != ka + k0) pack_load(sm, lr, R, k, kc, ke, x);
      store16<S>(J.S, J.rows_total, grow, kpitch, k, e, x);
    }
  }
}

template <int S>
__global__ void __launch_bounds__(kSplitThreads, 3) pack_split_kernel(PackJob ja, PackJob jb, int ga, int gab,
                                                                      int csize, int kpitch, ZeroJob zj) {
  grid_trigger();
  if (int(blockIdx.x) >= gab) {
    const int z = int(blockIdx.x) - gab;
    if (z < zj.n) zero_part(zj, z);
    return;
  }
  const bool is_a = int(blockIdx.x) < ga;
  const PackJob& J = is_a ? ja : jb;
  const int2 c = J.ctas[int(blockIdx.x) - (is_a ? 0 : ga)];
  const PackGroup G = J.groups[c.x];
  __shared__ PackShared sm;
  if (G.along) pack_cols<S>(sm, J, G, c.y, csize, kpitch);
  else if (c.y * split_cta_rows(G.K) < G.h) pack_rows<S>(sm, J, G, c.y, kpitch);
}

}  // namespace oz

// ---------------------------------------------------------------------------------
// host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    BST_CUDA(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q));
    BST_REQUIRE(p && q == cudaDriverEntryPointSuccess, BST_E_CUDA, "cuTensorMapEncodeTiled unavailable");
    fn = (EncodeTiledFn)p;
  }
  return fn;
}

// Map of a split buffer (S slices of `rows` rows of kpitch): one box is all
// slices of box_rows rows of a K chunk.  Rows past a slice's end are filled
// with zeros; with fewer rows than a box the map reaches into the next slice
// (past the last one into the buffer's spare rows), and what a tile reads
// there goes to rows or columns that are not stored.
static CUtensorMap make_map(void* base, int kpitch, int rows, int box_rows, int S) {
  CUtensorMap m;
  std::memset(&m, 0, sizeof(m));
  cuuint64_t dims[3] = {cuuint64_t(kpitch), cuuint64_t(std::max(rows, box_rows)), cuuint64_t(S)};
  cuuint64_t strides[2] = {cuuint64_t(kpitch) * 2, cuuint64_t(rows) * kpitch * 2};
  cuuint32_t box[3] = {cuuint32_t(oz::kTK), cuuint32_t(box_rows), cuuint32_t(S)};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  BST_REQUIRE(r == CUDA_SUCCESS, BST_E_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string(int(r)));
  return m;
}

struct OzakiPlan {
  int S = 5, TN = 64;  // digit slices per operand, output tile width
  int nprobs = 0, ntiles = 0;
  int rowsA = 0, rowsB = 0, kpitch = 32;
  oz::Prob* d_probs = nullptr;
  oz::Tile* d_tiles = nullptr;
  oz::SplitTask *d_sa = nullptr, *d_sb = nullptr;
  int2 *d_ca = nullptr, *d_cb = nullptr;  // the split's CTA tables
  int split_ca = 0, split_cb = 0;  // CTAs of the split of A and of B
  int split_cluster = 1;           // CTAs that share 32 interleaved rows of an operand
  __nv_bfloat16 *SA = nullptr, *SB = nullptr;
  int *eA = nullptr, *eB = nullptr;
  CUtensorMap mapA, mapB;
  // every problem reads B as it reads A (a Gram matrix X^T X): with the same
  // pointer for both, B's split is skipped and its tiles come from A's
  // digits through mapBA
  bool ab_same = false;
  CUtensorMap mapBA;
  double flops = 0;
  double split_bytes = 0;  // FP64 read + S BF16 digits written per element, exponent per row
  // K == 0 problems (no matched block pair): written as zeros by a separate
  // launch, so every tile of the persistent GEMM has at least one K chunk
  // (its epilogue then always waits for products of that tile, which keeps
  // the CTA's mbarrier phases in step)
  GemmProb* d_zprobs = nullptr;
  oz::ZeroCta* d_zctas = nullptr;
  int nzctas = 0;
  // output scatter into canonical blocks (plans built by
  // ozaki_prepare_scatter): tables on the device, K == 0 problems listed
  // by index for the beta-only pass
  int2* d_rowtab = nullptr;
  int4* d_coltab = nullptr;
  long long* d_bbase = nullptr;
  int* d_zidx = nullptr;
  bool scatter = false;
  // packed operands (pack_split_kernel reads the tensors' blocks; no
  // sector matrices, no separate split)
  bool packed = false;
  void* d_pack = nullptr;  // holds the following tables
  oz::PackGroup *d_pgA = nullptr, *d_pgB = nullptr;
  oz::PackSeg *d_psA = nullptr, *d_psB = nullptr;
  int2 *d_pcA = nullptr, *d_pcB = nullptr;
  int ncA = 0, ncB = 0;                    // CTAs of each operand
  bool pack_apart = false;                 // one launch per operand
  int pack_cluster = 1;                    // CTAs that share the k of a block of rows
  ~OzakiPlan() {
    cudaFree(d_pack);
    cudaFree(d_ca);
    cudaFree(d_cb);
    cudaFree(d_rowtab);
    cudaFree(d_coltab);
    cudaFree(d_bbase);
    cudaFree(d_zidx);
    cudaFree(d_zctas);
    cudaFree(d_probs);
    cudaFree(d_tiles);
    cudaFree(d_sa);
    cudaFree(d_sb);
    cudaFree(SA);
    cudaFree(SB);
    cudaFree(eA);
    cudaFree(eB);
    cudaFree(d_zprobs);
  }
};

template <int S, int TN>
static size_t smem_bytes() { return sizeof(oz::Smem<S, TN>) + 1024; }

template <int S, int TN>
static void set_kernel_attrs() {
  static bool done = false;
  if (done) return;
  BST_CUDA(cudaFuncSetAttribute(oz::ozaki_gemm_kernel<S, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(smem_bytes<S, TN>())));
  done = true;
}

// streaming multiprocessors of the current device (one persistent CTA each)
static int num_sms() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 152;
  return n > 0 ? n : 152;
}

struct PackTables {
  std::vector<oz::PackGroup> g;
  std::vector<oz::PackSeg> sg;
  std::vector<int2> ctas;
  int kcol = 0;    // longest k read with the lanes along the rows
  int blocks = 0;  // CTAs without sharing of k
  void place(int csize) {
    ctas.clear();
    for (size_t i = 0; i < g.size(); ++i) {
      const int n = oz::pack_ctas(g[i].h, g[i].K, g[i].along, csize);
      for (int c = 0; c < n; ++c) ctas.push_back(make_int2(int(i), c));
    }
  }
};

// Appends the pack groups and segments of one operand of one contraction:
// v is the operand's sector-matrix view of layout L (rows: its open legs,
// columns: its contracted legs), probs the contraction's problems in GEMM
// order (their operand sectors at a_off / b_off), `row` the split-buffer
// row of the first problem (advanced by M or N per problem), `src` the
// operand's index in a pointer table (0 for a single contraction).
static void append_pack(PackTables& T, const Layout* L, const MatView& v, const std::vector<GemmProb>& probs,
                        bool b_side, int& row, int src) {
  std::map<int64_t, const MatSector*> by_off;
  for (auto& sec : v.secs)
    if (sec.rows > 0 && sec.cols > 0) by_off[sec.off] = &sec;
  const int r = L->rank;
  const int nr = int(v.rowlegs.size()), nc = int(v.collegs.size());
  BST_REQUIRE(nr + nc == r && r <= kMaxRank, BST_E_ARG, "pack: view does not cover the tensor");

  std::vector<int32_t> tup(r);
  for (auto& g : probs) {
    const int rows = b_side ? g.N : g.M;
    if (g.K > 0) {
      auto it = by_off.find(b_side ? g.b_off : g.a_off);
      BST_REQUIRE(it != by_off.end() && it->second->rows == rows && it->second->cols == g.K, BST_E_SHAPE,
                  "pack: problem does not match its operand sector");
      const MatSector& sec = *it->second;
      for (size_t rc = 0; rc < sec.rcfg.size(); ++rc) {
        const int64_t h = (rc + 1 < sec.rcfg.size() ? sec.roff[rc + 1] : sec.rows) - sec.roff[rc];
        oz::PackGroup pg{};
        pg.along = nc > 0 && v.collegs.back() == r - 1 ? 0 : 1;
        pg.row0 = int32_t(row + sec.roff[rc]);
        pg.h = int32_t(h);
        pg.K = g.K;
        pg.seg0 = int64_t(T.sg.size());
        pg.nseg = int32_t(sec.ccfg.size());
        int64_t kcov = 0;
        for (size_t cc = 0; cc < sec.ccfg.size(); ++cc) {
          for (int j = 0; j < nr; ++j) tup[v.rowlegs[j]] = sec.rcfg[rc][j];
          for (int j = 0; j < nc; ++j) tup[v.collegs[j]] = sec.ccfg[cc][j];
          const int64_t b = L->block_of(tup.data());
          BST_REQUIRE(b >= 0, BST_E_SHAPE, "pack: missing operand block");
          const int64_t* sh = &L->shape[b * r];
          std::vector<int64_t> bst(r, 1);
          for (int i = r - 2; i >= 0; --i) bst[i] = bst[i + 1] * sh[i + 1];
          oz::PackSeg sg{};
          sg.off = L->offset[b];
          sg.k0 = int32_t(sec.coff[cc]);
          sg.nr = nr;
          sg.nc = nc;
          sg.src = src;
          int64_t hh = 1, w = 1;
          for (int j = 0; j < nr + nc; ++j) {
            const int leg = j < nr ? v.rowlegs[j] : v.collegs[j - nr];
            FastDiv f;
            f.init(uint32_t(sh[leg]));
            sg.leg[j] = {int32_t(sh[leg]), int32_t(bst[leg]), f.m, f.l};
            (j < nr ? hh : w) *= sh[leg];
          }
          BST_REQUIRE(hh == h && sg.k0 == kcov, BST_E_SHAPE, "pack: segment does not tile the row");
          kcov += w;
          T.sg.push_back(sg);
        }
        BST_REQUIRE(kcov == g.K, BST_E_SHAPE, "pack: segments do not cover K");
        if (pg.along) T.kcol = std::max(T.kcol, pg.K);
        T.blocks += oz::pack_ctas(pg.h, pg.K, pg.along, 1);
        T.g.push_back(pg);
      }
    }
    row += rows;
  }
}

// Tile schedule of a plan (the order in which CTAs pick up output tiles):
// 0 problem order, row tiles outer; 1 longest K first (the tiles that take
// longest start first, so the last wave is short); 2 problem order, column
// tiles outer (CTAs that run together share B slices in L2).
struct ScatterSpec {
  std::vector<int2> rowtab;
  std::vector<int4> coltab;
  std::vector<long long> bbase;
  std::vector<int64_t> rt_off, ct_off, bb_off;  // per problem
  std::vector<int32_t> ncc;                     // per problem
};

static OzakiPlan* build_plan(Ctx* ctx, const std::vector<GemmProb>& probs, int order = 0,
                             const ScatterSpec* sc = nullptr, int S = 5, int TN = 64) {
  BST_REQUIRE((S == 5 || S == 3) && (TN == 64 || TN == 32), BST_E_ARG, "Ozaki GEMM: unsupported shape");
  auto* P = new OzakiPlan();
  P->S = S;
  P->TN = TN;
  std::vector<oz::Prob> hp;
  std::vector<oz::Tile> ht;
  std::vector<oz::SplitTask> sa, sb;
  std::vector<GemmProb> zp;
  int maxk = 1;
  P->ab_same = !probs.empty();
  for (auto& g : probs) {
    BST_REQUIRE(g.K <= oz::kMaxK, BST_E_UNSUPPORTED, "Ozaki GEMM: K above 10000");
    maxk = std::max(maxk, g.K);
    P->ab_same = P->ab_same && g.M == g.N && g.a_off == g.b_off && g.a_m == g.b_n && g.a_k == g.b_k;
  }
  P->kpitch = (maxk + oz::kTK - 1) / oz::kTK * oz::kTK;
  for (auto& g : probs) {
    oz::Prob q{};
    q.M = g.M;
    q.N = g.N;
    q.K = g.K;
    q.arow = P->rowsA;
    q.brow = P->rowsB;
    q.c_off = g.c_off;
    q.c_m = g.c_m;
    q.c_n = g.c_n;
    if (sc) {
      const size_t pi = hp.size();
      q.ncc = sc->ncc[pi];
      q.rt_off = sc->rt_off[pi];
      q.ct_off = sc->ct_off[pi];
      q.bb_off = sc->bb_off[pi];
    }
    // (a one-column or one-row operand counts as contiguous)
    sa.push_back({g.M, g.K, P->rowsA, 0, g.a_off, g.a_m, g.K <= 1 ? 1 : g.a_k});
    sb.push_back({g.N, g.K, P->rowsB, 0, g.b_off, g.b_n, g.K <= 1 ? 1 : g.b_k});
    P->rowsA += g.M;
    P->rowsB += g.N;
    const int pi = int(hp.size());
    hp.push_back(q);
    auto add_tile = [&](int i, const oz::Prob& o, int m0, int n0) {
      ht.push_back({i, m0 | (std::min(oz::kTM, o.M - m0) - 1), n0 | (std::min(TN, o.N - n0) - 1),
                    (o.K + oz::kTK - 1) / oz::kTK, o.arow + m0, o.brow + n0, int32_t(o.rt_off + m0),
                    int32_t(o.ct_off + n0)});
    };
    if (g.K == 0) {
      zp.push_back(g);
    } else if (order == 2) {
      for (int n0 = 0; n0 < g.N; n0 += TN)
        for (int m0 = 0; m0 < g.M; m0 += oz::kTM) add_tile(pi, q, m0, n0);
    } else {
      for (int m0 = 0; m0 < g.M; m0 += oz::kTM)
        for (int n0 = 0; n0 < g.N; n0 += TN) add_tile(pi, q, m0, n0);
    }
    P->flops += 2.0 * double(g.M) * g.N * g.K;
    P->split_bytes += double(g.M + g.N) * g.K * (8.0 + 2.0 * S) + 4.0 * (g.M + g.N);
  }
  if (order == 1)
    std::stable_sort(ht.begin(), ht.end(),
                     [&](const oz::Tile& x, const oz::Tile& y) { return hp[x.prob].K > hp[y.prob].K; });
  P->nprobs = int(hp.size());
  P->ntiles = int(ht.size());
  // CTAs of the split (a scattering plan's operands are packed, see
  // attach_pack): split_cta_rows contiguous rows each, or a cluster per 32
  // interleaved rows (128 k per CTA and pass: one pass up to K = 1024)
  if (sc) sa.clear(), sb.clear();
  int kcol = 0;
  for (auto* v : {&sa, &sb})
    for (auto& t : *v)
      if (t.s_k != 1 && t.s_r == 1) kcol = std::max(kcol, t.K);
  while (P->split_cluster < 8 && P->split_cluster * 128 < kcol) P->split_cluster *= 2;
  const int sc_ = P->split_cluster;
  auto place = [&](const std::vector<oz::SplitTask>& v) {
    std::vector<int2> ctas;
    for (size_t i = 0; i < v.size(); ++i) {
      const oz::SplitTask& t = v[i];
      const int per = t.s_k == 1 ? oz::split_cta_rows(t.K) : 8;
      int n = t.s_k != 1 && t.s_r == 1 ? (t.rows + 31) / 32 * sc_ : (t.rows + per - 1) / per;
      n = (n + sc_ - 1) / sc_ * sc_;
      for (int c = 0; c < n; ++c) ctas.push_back(make_int2(int(i), c));
    }
    return ctas;
  };
  const std::vector<int2> ca = place(sa), cb = place(sb);
  P->split_ca = int(ca.size());
  P->split_cb = int(cb.size());
  BST_REQUIRE(int64_t(P->rowsA) * S < (1ll << 31) && int64_t(P->rowsB) * S < (1ll << 31),
              BST_E_UNSUPPORTED, "Ozaki GEMM: too many rows");
  auto up = [](auto** dst, const auto& v) {
    using T = typename std::remove_reference<decltype(v)>::type::value_type;
    if (v.empty()) return;
    BST_CUDA(cudaMalloc((void**)dst, sizeof(T) * v.size()));
    BST_CUDA(cudaMemcpy(*dst, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice));
  };
  up(&P->d_probs, hp);
  up(&P->d_tiles, ht);
  up(&P->d_zprobs, zp);
  std::vector<oz::ZeroCta> zc;
  for (size_t i = 0; i < zp.size(); ++i) {
    const int rows = std::max(1, oz::kZeroElems / std::max(zp[i].N, 1));
    for (int m = 0; m < zp[i].M; m += rows) zc.push_back({int(i), m, std::min(zp[i].M, m + rows)});
  }
  up(&P->d_zctas, zc);
  P->nzctas = int(zc.size());
  up(&P->d_sa, sa);
  up(&P->d_sb, sb);
  up(&P->d_ca, ca);
  up(&P->d_cb, cb);
  if (sc) {
    P->scatter = true;
    up(&P->d_rowtab, sc->rowtab);
    up(&P->d_coltab, sc->coltab);
    up(&P->d_bbase, sc->bbase);
    std::vector<int> zi;
    for (int i = 0; i < int(hp.size()); ++i)
      if (hp[i].K == 0) zi.push_back(i);
    up(&P->d_zidx, zi);
  }
  // split buffers: S slices x rows x kpitch BF16, with room for a full tile
  // past the end so TMA boxes of the last rows stay inside the allocation
  const int64_t ra = int64_t(S) * std::max(P->rowsA, 1) + oz::kTM;
  const int64_t rb = int64_t(S) * std::max(P->rowsB, 1) + std::max(TN, oz::kTM);
  BST_CUDA(cudaMalloc(&P->SA, sizeof(__nv_bfloat16) * ra * P->kpitch));
  BST_CUDA(cudaMalloc(&P->SB, sizeof(__nv_bfloat16) * rb * P->kpitch));
  BST_CUDA(cudaMemset(P->SA, 0, sizeof(__nv_bfloat16) * ra * P->kpitch));
  BST_CUDA(cudaMemset(P->SB, 0, sizeof(__nv_bfloat16) * rb * P->kpitch));
  BST_CUDA(cudaMalloc(&P->eA, sizeof(int) * std::max(P->rowsA, 1)));
  BST_CUDA(cudaMalloc(&P->eB, sizeof(int) * std::max(P->rowsB, 1)));
  P->mapA = make_map(P->SA, P->kpitch, std::max(P->rowsA, 1), oz::kTM, S);
  P->mapB = make_map(P->SB, P->kpitch, std::max(P->rowsB, 1), TN, S);
  if (P->ab_same) P->mapBA = make_map(P->SA, P->kpitch, std::max(P->rowsA, 1), TN, S);
  return P;
}

// Launch of `grid` CTAs in clusters of csize (grid a multiple of it).
template <class... P, class... A>
static void launch_clusters(void (*kern)(P...), int grid, int threads, int csize, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = unsigned(csize);
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = csize > 1 ? 1 : 0;
  BST_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
}

// A, B: the operands' sector matrices, or for a packed plan the operand
// tensors themselves (tabA / tabB: per-segment tensor tables of a batch).
// zeros_last: C overlaps an operand, so no output is written before a packed
// plan has read both.
static void run_plan(Ctx* ctx, OzakiPlan* P, const double* A, const double* B, double* C, cudaStream_t s,
                     bool split_a = true, double alpha = 1.0, double beta = 0.0,
                     const double* const* tabA = nullptr, const double* const* tabB = nullptr,
                     const long long* bbase = nullptr, bool zeros_last = false) {
  const oz::Scatter sc{P->d_rowtab, P->d_coltab, bbase ? bbase : P->d_bbase, alpha, beta};
  const bool b_from_a = P->ab_same && A == B && split_a;
  if (P->packed) {
    // gather + split: FP64 read once per element (rows of more than 128 or
    // 512 once more from cache), S digits written; the byte count is that of
    // the split of gathered rows without the FP64 row write and read of a
    // separate gather.  The K == 0 problems' outputs are written by the same
    // launch, or by one behind it.
    ProfScope ps(ctx, s, "pack_bf16", 0.0, P->split_bytes);
    const oz::PackJob ja{P->d_pgA, P->d_psA, P->d_pcA, P->rowsA, A, tabA, P->SA, P->eA};
    const oz::PackJob jb{P->d_pgB, P->d_psB, P->d_pcB, P->rowsB, B, tabB, P->SB, P->eB};
    const oz::ZeroJob zj{P->nzctas, P->d_zctas, P->scatter ? P->d_probs : nullptr, P->d_zidx, sc, P->d_zprobs, C};
    const int cs = P->pack_cluster;
    const int gz = (P->nzctas + cs - 1) / cs * cs;
    auto pack = [&](int ga, int gb, int z) {
      if (ga + gb + z == 0) return;
      launch_clusters(P->S == 5 ? oz::pack_split_kernel<5> : oz::pack_split_kernel<3>, ga + gb + z, oz::kSplitThreads,
                      cs, s, ja, jb, ga, ga + gb, cs, P->kpitch, zj);
      count_launch(ctx);
    };
    const int gz0 = zeros_last ? 0 : gz;
    if (P->pack_apart) {
      pack(P->ncA, 0, 0);
      pack(0, P->ncB, gz0);
    } else {
      pack(P->ncA, P->ncB, gz0);
    }
    if (zeros_last) pack(0, 0, gz);
    if (P->ntiles == 0) return;
  } else {
    // the split of both operands; the K == 0 problems' outputs are written
    // by the same launch
    ProfScope ps(ctx, s, "split_bf16", 0.0, b_from_a ? 0.5 * P->split_bytes : P->split_bytes);
    const int cs = P->split_cluster;
    const int ga = (split_a && P->ntiles) ? P->split_ca : 0, gb = (b_from_a || !P->ntiles) ? 0 : P->split_cb;
    const int gz = (P->nzctas + cs - 1) / cs * cs;
    const oz::ZeroJob zj{P->nzctas, P->d_zctas, P->scatter ? P->d_probs : nullptr, P->d_zidx, sc, P->d_zprobs, C};
    if (ga + gb + gz > 0) {
      const oz::SplitJob ja{P->d_sa, P->d_ca, P->rowsA, A, P->SA, P->eA};
      const oz::SplitJob jb{P->d_sb, P->d_cb, P->rowsB, B, P->SB, P->eB};
      launch_clusters(P->S == 5 ? oz::ozaki_split_kernel<5> : oz::ozaki_split_kernel<3>, ga + gb + gz,
                      oz::kSplitThreads, cs, s, ja, jb, ga, ga + gb, cs, P->kpitch, zj);
      count_launch(ctx);
    }
    if (P->ntiles == 0) return;
  }
  ProfScope ps(ctx, s, "gemm_ozaki", P->flops, 0.0);
  const int grid = std::min(P->ntiles, num_sms());
  const long long spin = ctx->spin_limit > 0 ? ctx->spin_limit : oz::kSpinLimit;
  const CUtensorMap& mB = b_from_a ? P->mapBA : P->mapB;
  const int* eB = b_from_a ? P->eA : P->eB;
  auto launch = [&](auto kern, size_t smem) {
    // (behind the split or pack, whose last blocks its prologue overlaps)
    launch_behind(true, kern, dim3(unsigned(grid)), oz::kThreads, smem, s, P->mapA, mB, (const oz::Prob*)P->d_probs,
                  (const oz::Tile*)P->d_tiles, P->ntiles, (const int*)P->eA, eB, C, sc, ctx->d_err, spin);
  };
  if (P->S == 5 && P->TN == 64) {
    set_kernel_attrs<5, 64>();
    launch(oz::ozaki_gemm_kernel<5, 64>, smem_bytes<5, 64>());
  } else if (P->S == 5) {
    set_kernel_attrs<5, 32>();
    launch(oz::ozaki_gemm_kernel<5, 32>, smem_bytes<5, 32>());
  } else if (P->TN == 64) {
    set_kernel_attrs<3, 64>();
    launch(oz::ozaki_gemm_kernel<3, 64>, smem_bytes<3, 64>());
  } else {
    set_kernel_attrs<3, 32>();
    launch(oz::ozaki_gemm_kernel<3, 32>, smem_bytes<3, 32>());
  }
  BST_CUDA(cudaGetLastError());
  count_launch(ctx);
}

int ozaki_slices(bst_prec prec) { return prec == BST_BF16X3 ? 3 : 5; }

int ozaki_pick_tn(const std::vector<GemmProb>& probs) {
  int64_t tiles64 = 0;
  double cols = 0, cols64 = 0;
  for (auto& g : probs) {
    if (g.K == 0) continue;
    tiles64 += int64_t((g.M + oz::kTM - 1) / oz::kTM) * ((g.N + 63) / 64);
    cols += double(g.N);
    cols64 += double((g.N + 63) / 64 * 64);
  }
  if (tiles64 == 0) return 64;
  return (tiles64 < num_sms() || cols < 0.5 * cols64) ? 32 : 64;
}

// Plan whose epilogue writes every product element into the output
// tensor's canonical block (Sec. 2: the reduced pair products land in the
// output block of their output quantum numbers).  C's legs are A's open
// legs then B's, so the block of (row config r, column config c) is a
// row-major [rows of r x columns of c] matrix: element (m, n) of a sector
// goes to offset(r, c) + mi * width(c) + ni.
// Appends the scatter tables of one contraction's problems (block offsets
// relative to its own output; bsrc, when given, records the contraction
// index `src` of every entry of bbase).
static void append_scatter(ScatterSpec& sc, ContractPlan* p, std::vector<int32_t>* bsrc, int src) {
  const Layout* C = p->C;
  std::vector<int32_t> tup(C->rank);
  size_t pi = 0;
  for (auto& cs : p->vc.secs) {
    if (!(cs.rows > 0 && cs.cols > 0)) continue;
    BST_REQUIRE(pi < p->probs.size() && p->probs[pi].M == cs.rows && p->probs[pi].N == cs.cols, BST_E_SHAPE,
                "scatter plan: problem list does not follow the output sectors");
    sc.rt_off.push_back(int64_t(sc.rowtab.size()));
    sc.ct_off.push_back(int64_t(sc.coltab.size()));
    sc.bb_off.push_back(int64_t(sc.bbase.size()));
    sc.ncc.push_back(int32_t(cs.ccfg.size()));
    std::vector<int64_t> width(cs.ccfg.size());
    for (size_t c = 0; c < cs.ccfg.size(); ++c) {
      const int64_t w = (c + 1 < cs.ccfg.size() ? cs.coff[c + 1] : cs.cols) - cs.coff[c];
      width[c] = w;
      for (int64_t ni = 0; ni < w; ++ni) sc.coltab.push_back(make_int4(int(c), int(ni), int(w), 0));
    }
    for (size_t r = 0; r < cs.rcfg.size(); ++r) {
      const int64_t h = (r + 1 < cs.rcfg.size() ? cs.roff[r + 1] : cs.rows) - cs.roff[r];
      for (int64_t mi = 0; mi < h; ++mi) sc.rowtab.push_back(make_int2(int(r), int(mi)));
      for (size_t c = 0; c < cs.ccfg.size(); ++c) {
        size_t k = 0;
        for (int32_t x : cs.rcfg[r]) tup[k++] = x;
        for (int32_t x : cs.ccfg[c]) tup[k++] = x;
        const int64_t b = C->block_of(tup.data());
        BST_REQUIRE(b >= 0, BST_E_SHAPE, "scatter plan: missing output block");
        sc.bbase.push_back((long long)C->offset[b]);
        if (bsrc) bsrc->push_back(src);
      }
    }
    ++pi;
  }
  BST_REQUIRE(pi == p->probs.size(), BST_E_SHAPE, "scatter plan: problem count mismatch");
  BST_REQUIRE(sc.rowtab.size() < (size_t(1) << 31) && sc.coltab.size() < (size_t(1) << 31), BST_E_UNSUPPORTED,
              "scatter plan: too many rows");
}

static OzakiPlan* prepare_scatter(Ctx* ctx, ContractPlan* p, int S) {
  ScatterSpec sc;
  append_scatter(sc, p, nullptr, 0);
  return build_plan(ctx, p->probs, 0, &sc, S, ozaki_pick_tn(p->probs));
}

// Device tables of the packed operands of a contraction plan.
static void attach_pack(OzakiPlan* P, PackTables& ta, PackTables& tb) {
  // CTAs along k only while the blocks of rows alone leave SMs idle: a CTA
  // pays for its tables whatever its share (the batch of 64 corners takes
  // 3.3 ms with clusters of 8 and 2.05 without, the D=6 corner 28 us with
  // clusters and 31 without)
  P->pack_cluster = oz::pack_col_ctas(std::max(ta.kcol, tb.kcol), 8);
  while (P->pack_cluster > 1 && (ta.blocks + tb.blocks) * P->pack_cluster > 4 * num_sms()) P->pack_cluster /= 2;
  ta.place(P->pack_cluster);
  tb.place(P->pack_cluster);
  // one allocation and one copy: the first pass over a new structure pays for
  // each (768 -> 700 us for five sectors a leg)
  std::vector<char> host;
  auto place = [&](const auto& v) {
    const size_t at = host.size();
    host.resize(at + (v.size() * sizeof(v[0]) + 255) / 256 * 256);
    if (!v.empty()) std::memcpy(host.data() + at, v.data(), v.size() * sizeof(v[0]));
    return at;
  };
  const size_t at[] = {place(ta.g), place(ta.sg), place(tb.g), place(tb.sg), place(ta.ctas), place(tb.ctas)};
  if (!host.empty()) {
    BST_CUDA(cudaMalloc(&P->d_pack, host.size()));
    BST_CUDA(cudaMemcpy(P->d_pack, host.data(), host.size(), cudaMemcpyHostToDevice));
  }
  char* base = static_cast<char*>(P->d_pack);
  P->d_pgA = reinterpret_cast<oz::PackGroup*>(base + at[0]);
  P->d_psA = reinterpret_cast<oz::PackSeg*>(base + at[1]);
  P->d_pgB = reinterpret_cast<oz::PackGroup*>(base + at[2]);
  P->d_psB = reinterpret_cast<oz::PackSeg*>(base + at[3]);
  P->d_pcA = reinterpret_cast<int2*>(base + at[4]);
  P->d_pcB = reinterpret_cast<int2*>(base + at[5]);
  P->ncA = int(ta.ctas.size());
  P->ncB = int(tb.ctas.size());
  P->packed = true;
  P->ab_same = false;
}

static void attach_pack(OzakiPlan* P, ContractPlan* p) {
  PackTables ta, tb;
  int ra = 0, rb = 0;
  append_pack(ta, p->A, p->va, p->probs, false, ra, 0);
  append_pack(tb, p->B, p->vb, p->probs, true, rb, 0);
  BST_REQUIRE(ra == P->rowsA && rb == P->rowsB, BST_E_SHAPE, "pack: row count mismatch");
  attach_pack(P, ta, tb);
}

// Both operands' innermost legs are contracted (in the last pair): the pack
// reads both with its lanes along k.
bool ozaki_k_inner(const ContractPlan* p) {
  return !p->va.collegs.empty() && p->va.collegs.back() == p->A->rank - 1 && !p->vb.collegs.empty() &&
         p->vb.collegs.back() == p->B->rank - 1;
}

void run_gemm_ozaki_scatter(Ctx* ctx, ContractPlan* p, int S, const double* a, const double* b, double* c,
                            double alpha, double beta, cudaStream_t s) {
  OzakiPlan*& P = p->oz[S == 3 ? 1 : 0][1];
  if (!P) {
    P = prepare_scatter(ctx, p, S);
    attach_pack(P, p);
  }
  auto meets = [&](const double* x, const Layout* X) {
    const uintptr_t x0 = uintptr_t(x), c0 = uintptr_t(c);
    return x0 < c0 + sizeof(double) * p->C->nnz && c0 < x0 + sizeof(double) * X->nnz;
  };
  run_plan(ctx, P, a, b, c, s, true, alpha, beta, nullptr, nullptr, nullptr, meets(a, p->A) || meets(b, p->B));
}

void run_gemm_ozaki(Ctx* ctx, ContractPlan* p, int S, const double* Am, const double* Bm, double* Cmat,
                    cudaStream_t s) {
  OzakiPlan*& P = p->oz[S == 3 ? 1 : 0][0];
  if (!P) P = build_plan(ctx, p->probs, 0, nullptr, S, ozaki_pick_tn(p->probs));
  run_plan(ctx, P, Am, Bm, Cmat, s);
}

void ozaki_free(OzakiPlan* oz) { delete oz; }

// Batched contractions: one packed, scattering plan over the problems of
// every contraction (probs: their concatenation, in plan order).  The
// output blocks of contraction i are addressed relative to the first
// output's pointer: bbase_rel holds each entry's offset inside its own
// output and bbase_src its contraction, and ozaki_batch_bbase turns them
// into element offsets from c[0] for one set of output pointers.
OzakiPlan* ozaki_batch_plan(Ctx* ctx, const std::vector<ContractPlan*>& plans, const std::vector<GemmProb>& probs,
                            int order, int S, int TN, std::vector<long long>* bbase_rel,
                            std::vector<int32_t>* bbase_src) {
  ScatterSpec sc;
  bbase_src->clear();
  PackTables ta, tb;
  int ra = 0, rb = 0;
  bool apart = false;
  for (size_t i = 0; i < plans.size(); ++i) {
    append_scatter(sc, plans[i], bbase_src, int(i));
    append_pack(ta, plans[i]->A, plans[i]->va, plans[i]->probs, false, ra, int(i));
    append_pack(tb, plans[i]->B, plans[i]->vb, plans[i]->probs, true, rb, int(i));
    apart = apart || !ozaki_k_inner(plans[i]);
  }
  BST_REQUIRE(sc.rt_off.size() == probs.size(), BST_E_SHAPE, "batch plan: problem count mismatch");
  *bbase_rel = sc.bbase;
  OzakiPlan* P = build_plan(ctx, probs, order, &sc, S, TN == 0 ? ozaki_pick_tn(probs) : TN);
  BST_REQUIRE(ra == P->rowsA && rb == P->rowsB, BST_E_SHAPE, "batch plan: row count mismatch");
  attach_pack(P, ta, tb);
  P->pack_apart = apart;
  return P;
}

void ozaki_batch_bbase(const std::vector<long long>& rel, const std::vector<int32_t>& src,
                       const std::vector<double*>& c, std::vector<long long>* out) {
  std::vector<long long> delta(c.size());
  const uintptr_t c0 = uintptr_t(c[0]);
  for (size_t i = 0; i < c.size(); ++i) {
    const long long d = (long long)(uintptr_t(c[i]) - c0);
    BST_REQUIRE(d % (long long)sizeof(double) == 0, BST_E_ARG, "output pointers must be 8-byte aligned");
    delta[i] = d / (long long)sizeof(double);
  }
  out->resize(rel.size());
  for (size_t j = 0; j < rel.size(); ++j) (*out)[j] = rel[j] + delta[src[j]];
}

void run_ozaki_batch(Ctx* ctx, OzakiPlan* P, double* const* bases, int n, double* c0, const long long* bbase,
                     double alpha, double beta, cudaStream_t s) {
  run_plan(ctx, P, nullptr, nullptr, c0, s, true, alpha, beta, bases, bases + n, bbase);
}

void run_gemm_ozaki_probs(Ctx* ctx, const std::string& tag, const std::vector<GemmProb>& probs, const double* A,
                          const double* B, double* C, cudaStream_t s, int order, bool split_a, int S, int TN) {
  if (TN == 0) TN = ozaki_pick_tn(probs);
  // plans live in the context (freed with it), keyed by caller tag, problem
  // list, tile schedule, digit count and tile width
  const std::string key = tag + "/" + std::to_string(probs_hash(probs)) + "/" + std::to_string(order) + "/" +
                          std::to_string(S) + "x" + std::to_string(TN);
  OzakiPlan* P;
  {
    std::lock_guard<std::mutex> g(ctx->mu);
    auto it = ctx->ozplans.find(key);
    P = it == ctx->ozplans.end() ? nullptr : it->second.get();
  }
  if (!P) {
    std::shared_ptr<OzakiPlan> np(build_plan(ctx, probs, order, nullptr, S, TN));
    P = np.get();
    std::lock_guard<std::mutex> g(ctx->mu);
    ctx->ozplans[key] = std::move(np);
  }
  run_plan(ctx, P, A, B, C, s, split_a);
}

}  // namespace bst
