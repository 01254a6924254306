// Device helpers of the relayout kernels (block <-> strided region copies).
#pragma once

#include <algorithm>

#include "bst_internal.h"

namespace bst {

// A grid launched behind another (launch_behind) may start when every block
// of the first has called grid_trigger (or left), and must call grid_wait,
// which returns when the first has finished and its writes are visible,
// before it touches what that grid reads or writes, and in every block before
// it ends (so that a third grid that waits for it waits for both).
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch with programmatic serialisation behind the previous kernel of the
// stream (behind: that kernel is this library's, launched by the same call),
// else an ordinary one.
template <class... P, class... A>
void launch_behind(bool behind, void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = behind ? 1 : 0;
  BST_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
}

// Division by a runtime constant d >= 1 for numerators below 2^31 with one
// high multiply, an add and a shift (Granlund and Montgomery's round-up
// method): l = ceil(log2 d), m = floor(2^32 (2^l - d) / d) + 1,
// n / d = (umulhi(n, m) + n) >> l.
struct FastDiv {
  uint32_t d, m, l;
  __host__ __device__ void init(uint32_t dd) {
    d = dd;
    l = 0;
    while ((1u << l) < d) ++l;
    m = uint32_t(((uint64_t(1) << 32) * ((uint64_t(1) << l) - d)) / d + 1);
  }
  __device__ __forceinline__ uint32_t div(uint32_t n) const { return (__umulhi(n, m) + n) >> l; }
};

// Copy the elements [begin, end) of one task (row-major over its shape on
// the contiguous side) between blk and the strided side mat.  Each thread
// handles four elements per pass (indices first, then all loads, then all
// stores), so a warp keeps four loads in flight.
//   dir 0: mat[strided] = blk[contiguous]
//   dir 1: blk[contiguous] = alpha * mat[strided] + beta * blk (beta == 0: overwrite)
template <int kThreads>
__device__ __forceinline__ void relayout_range(const RelTask& t, int begin, int end, double* blk, double* mat,
                                               int dir, double alpha, double beta) {
  const int r = t.rank;
  FastDiv fd[kMaxRank];
  long long ms[kMaxRank];
#pragma unroll
  for (int i = 0; i < kMaxRank; ++i) {
    fd[i].init(i < r ? uint32_t(t.shape[i]) : 1u);
    ms[i] = i < r ? t.mstride[i] : 0;
  }
  constexpr int kU = 4;
  for (int e0 = begin + int(threadIdx.x); e0 < end; e0 += kU * kThreads) {
    long long mo[kU];
    bool ok[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int e = e0 + u * kThreads;
      ok[u] = e < end;
      uint32_t rem = uint32_t(ok[u] ? e : 0);
      long long o = t.mat_base;
#pragma unroll
      for (int i = kMaxRank - 1; i >= 0; --i) {
        if (i < r) {
          const uint32_t q = fd[i].div(rem);
          o += (long long)(rem - q * fd[i].d) * ms[i];
          rem = q;
        }
      }
      mo[u] = o;
    }
    double v[kU];
    if (dir == 0) {
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (ok[u]) v[u] = blk[t.blk_off + e0 + u * kThreads];
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (ok[u]) mat[mo[u]] = v[u];
    } else if (alpha == 1.0 && beta == 0.0) {
      // plain gather: no FP64 arithmetic (the FP64 pipe is narrow enough
      // that one multiply per element would cost about as much as its
      // 16 bytes of traffic)
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (ok[u]) v[u] = mat[mo[u]];
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (ok[u]) blk[t.blk_off + e0 + u * kThreads] = v[u];
    } else {
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (ok[u]) {
          v[u] = alpha * mat[mo[u]];
          if (beta != 0.0) v[u] += beta * blk[t.blk_off + e0 + u * kThreads];
        }
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (ok[u]) blk[t.blk_off + e0 + u * kThreads] = v[u];
    }
  }
}

// ---- copies by boxes ------------------------------------------------------------
//
// A tile of the copy is a box of the block that holds a run of up to about
// 64 elements along the innermost legs of either side (all of a short leg, an
// even part of a long one), widened by the next legs to about 2000 elements:
// it is read in one side's order and written in the other's through shared
// memory, so both sides move whole 32-byte sectors whatever the permutation.
// What a task's boxes look like is worked out once, with the task list, and a
// box tabulates the offsets of its runs on either side, to which a lane adds
// that of its place in a run: with the whole index arithmetic in every thread
// the copy was bound by its instructions.
constexpr int kRelBox = 2560;  // elements of a box
constexpr int kRelRows = 256;  // runs of a box
// shared memory shifts by one element every 16, so that the strided side's
// order spreads over the banks
__host__ __device__ constexpr int rel_pos(int i) { return i + (i >> 4); }

// A leg of more than one element (legs that follow each other on both sides
// are one).
struct alignas(16) RelBoxLeg {
  FastDiv outer, nt;   // boxes along the legs outside this one; along this one
  FastDiv full, last;  // extent in a box, in the last box along the leg
  int32_t lin;         // stride inside a box, row-major in the contiguous side's order
  int32_t slot;        // its place (innermost first) in the strided side's order
  int32_t sb, sm;      // element strides of the two sides
  int32_t run;         // bit s: a run of side s goes along it
};

struct alignas(16) RelBox {
  long long blk_off, mat_base;
  int32_t n, ntiles;   // legs; boxes (0: none, copied by relayout_range)
  int32_t nrun[2];     // legs of a run (the innermost ones) on either side
  RelBoxLeg leg[kMaxRank];  // contiguous side's order, innermost first
};

// The legs of a task of more than one element, contiguous side's order,
// innermost first (those that follow each other on both sides as one):
// extents and strides of the contiguous and the strided side; their number.
__host__ __device__ inline int rel_task_legs(const RelTask& t, int* L, long long* sb, long long* sm) {
  int n = 0;
  long long bs = 1;
  for (int k = t.rank - 1; k >= 0; --k) {
    if (t.shape[k] > 1) {
      if (n > 0 && t.mstride[k] == sm[n - 1] * L[n - 1]) {
        L[n - 1] *= t.shape[k];
      } else {
        L[n] = t.shape[k];
        sb[n] = bs;
        sm[n] = t.mstride[k];
        ++n;
      }
    }
    bs *= t.shape[k];
  }
  return n;
}

__host__ __device__ inline void rel_make_box(const RelTask& t, RelBox& b) {
  int L[kMaxRank];
  long long sb[kMaxRank], sm[kMaxRank], inm[kMaxRank];
  const int n = rel_task_legs(t, L, sb, sm);
  b.blk_off = t.blk_off;
  b.mat_base = t.mat_base;
  b.n = n;
  b.ntiles = 0;
  b.nrun[0] = b.nrun[1] = 0;
  int e[kMaxRank];
  long long span = 0;
  for (int j = 0; j < n; ++j) span += (L[j] - 1) * sm[j];
  if (span >= (1ll << 31)) return;
  for (int j = 0; j < n; ++j) {
    // (equal strides: legs of a diagonal, in either order)
    inm[j] = 1;
    int slot = 0;
    for (int k = 0; k < n; ++k)
      if (sm[k] < sm[j] || (sm[k] == sm[j] && k < j)) inm[j] *= L[k], ++slot;
    b.leg[j].slot = slot;
    b.leg[j].sb = int32_t(sb[j]);
    b.leg[j].sm = int32_t(sm[j]);
    b.leg[j].run = (sb[j] < 16 ? 1 : 0) | (inm[j] < 16 ? 2 : 0);
    b.nrun[0] += sb[j] < 16;
    b.nrun[1] += inm[j] < 16;
  }
  // extents: an even part of about `cap` elements of the legs that a run of
  // 16 elements reaches
  long long V = 1;
  for (int cap = 64; cap >= 32; cap /= 2) {
    V = 1;
    for (int j = 0; j < n; ++j) {
      e[j] = 1;
      for (int side = 0; side < 2; ++side) {
        const long long in = side ? inm[j] : sb[j];
        if (in < 16) {
          const int c = (cap + int(in) - 1) / int(in), nt = (L[j] + c - 1) / c, x = (L[j] + nt - 1) / nt;
          e[j] = x > e[j] ? x : e[j];
        }
      }
      V *= e[j];
    }
    if (V <= kRelBox) break;
  }
  // the contiguous side's next legs while the box stays below 2048
  for (int j = 0; j < n; ++j) {
    if (e[j] == L[j] || 2 * V > 2048) continue;
    const long long f = 2048 / V;
    const long long x = f * e[j] < L[j] ? f * e[j] : L[j];
    const int nt = int((L[j] + x - 1) / x), y = (L[j] + nt - 1) / nt;
    if (y <= e[j]) continue;
    V = V / e[j] * y;
    e[j] = y;
  }
  long long rows[2] = {1, 1};
  for (int j = 0; j < n; ++j) {
    if (!(b.leg[j].run & 1)) rows[0] *= e[j];
    if (!(b.leg[j].run & 2)) rows[1] *= e[j];
  }
  if (V > kRelBox || rows[0] > kRelRows || rows[1] > kRelRows) return;  // (does not happen: runs reach 16 elements)
  int lin = 1;
  for (int j = 0; j < n; ++j) {
    const int nt = (L[j] + e[j] - 1) / e[j];
    b.leg[j].lin = lin;
    b.leg[j].nt.init(uint32_t(nt));
    b.leg[j].full.init(uint32_t(e[j]));
    b.leg[j].last.init(uint32_t(L[j] - (nt - 1) * e[j]));
    lin *= e[j];
  }
  // neighbouring tiles are neighbours on the contiguous side: the innermost
  // leg's boxes run fastest
  uint32_t inner = 1;
  for (int j = 0; j < n; ++j) {
    b.leg[j].outer.init(inner);
    inner *= b.leg[j].nt.d;
  }
  b.ntiles = int32_t(inner);
}

// Whether a task is copied faster by boxes than straight, 2048 elements a CTA
// (see launch_relayout): a warp's 32 elements lie on 12 or more 128-byte lines
// of the strided side, and the box has at least eight runs on either side for
// the threads, or the elements lie on 24 or more sectors of 32 bytes and the
// block is so large that the parts of a sector no longer meet in the cache.
// b: its box.
inline bool rel_box_pays(const RelTask& t, const RelBox& b) {
  if (t.n < 1024 || b.n < 2 || b.leg[0].slot == 0) return false;
  int L[kMaxRank], at[kMaxRank] = {}, count[2] = {0, 0};
  long long sb[kMaxRank], sm[kMaxRank], seen[2][32], off = 0;
  const int n = rel_task_legs(t, L, sb, sm);
  for (int e = 0; e < 32; ++e) {
    for (int u = 0; u < 2; ++u) {  // lines, sectors
      const long long at_u = off / (u ? 4 : 16);
      if (std::find(seen[u], seen[u] + count[u], at_u) == seen[u] + count[u]) seen[u][count[u]++] = at_u;
    }
    for (int j = 0; j < n; ++j) {
      off += sm[j];
      if (++at[j] < L[j]) break;
      off -= sm[j] * L[j];
      at[j] = 0;
    }
  }
  int rows[2] = {1, 1};
  for (int j = 0; j < n; ++j)
    for (int side = 0; side < 2; ++side)
      if (!(b.leg[j].run >> side & 1)) rows[side] *= int(b.leg[j].full.d);
  return count[0] >= 12 && ((rows[0] >= 8 && rows[1] >= 8) || (count[1] >= 24 && t.n >= 1 << 24));
}

// A leg of the box at hand, on one side's list.
struct alignas(16) RelLeg {
  uint32_t d, m, l;  // extent and its FastDiv
  int32_t lin, st, pad[3];
};

struct RelShared {
  RelLeg leg[2][kMaxRank];  // contiguous side's order, strided side's order
  long long base[2];        // the box's first element on either side
  int run[2], rows[2];      // elements of a run, runs
  int2 row[2][kRelRows];    // (offset, position) of the runs
  double buf[rel_pos(kRelBox) + 1];
};

// The box `tile` of a task: a lane of the first warp per leg.
__device__ __forceinline__ void rel_box(RelShared& sh, const RelBox& b, int tile) {
  const unsigned all = 0xffffffffu;
  const int lane = int(threadIdx.x);
  long long b0 = 0, m0 = 0;
  int a[4] = {1, 1, 1, 1};  // run and runs of side 0, of side 1
  if (lane < b.n) {
    const RelBoxLeg g = b.leg[lane];
    const uint32_t o = g.outer.div(uint32_t(tile)), q = g.nt.div(o), at = o - q * g.nt.d;
    const FastDiv f = at + 1 == g.nt.d ? g.last : g.full;
    b0 = (long long)(at * g.full.d) * g.sb;
    m0 = (long long)(at * g.full.d) * g.sm;
    a[g.run & 1 ? 0 : 1] = int(f.d);
    a[g.run & 2 ? 2 : 3] = int(f.d);
    sh.leg[0][lane] = RelLeg{f.d, f.m, f.l, g.lin, g.sb, {0, 0, 0}};
    sh.leg[1][g.slot] = RelLeg{f.d, f.m, f.l, g.lin, g.sm, {0, 0, 0}};
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    b0 += __shfl_xor_sync(all, b0, o);
    m0 += __shfl_xor_sync(all, m0, o);
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] *= __shfl_xor_sync(all, a[i], o);
  }
  if (lane == 0) {
    sh.base[0] = b.blk_off + b0;
    sh.base[1] = b.mat_base + m0;
    sh.run[0] = a[0];
    sh.rows[0] = a[1];
    sh.run[1] = a[2];
    sh.rows[1] = a[3];
  }
}

// Box `tile` of one task, a plain copy in either direction (as
// relayout_range).
template <int kThreads, int kU>
__device__ __forceinline__ void relayout_box(RelShared& sh, const RelBox& b, int tile, double* blk, double* mat, int dir) {
  if (threadIdx.x < 32) rel_box(sh, b, tile);
  __syncthreads();
  // (offset, position) of index i over the legs [j, je) of one side's list
  auto place = [&](int side, int j, int je, int i) {
    uint32_t rem = uint32_t(i);
    int2 v = make_int2(0, 0);
    for (; j < je; ++j) {
      const RelLeg g = sh.leg[side][j];
      const uint32_t q = (__umulhi(rem, g.m) + rem) >> g.l;
      const int x = int(rem - q * g.d);
      v.x += x * g.st;
      v.y += x * g.lin;
      rem = q;
    }
    return v;
  };
  const int n0 = sh.rows[0], n1 = n0 + sh.rows[1];
  for (int i = int(threadIdx.x); i < n1; i += kThreads) {
    const int side = i >= n0, at = side ? i - n0 : i;
    sh.row[side][at] = place(side, b.nrun[side], b.n, at);
  }
  __syncthreads();
  // one side's runs, threads along a run, kU runs at a time
  auto each = [&](int side, auto&& body) {
    const int run = sh.run[side], rows = sh.rows[side];
    int sl = run > 32 ? 6 : run > 16 ? 5 : run > 8 ? 4 : run > 4 ? 3 : 2;
    while ((kThreads >> sl) > rows && (1 << sl) < run) ++sl;  // (few long runs: all threads along them)
    const int step = kThreads >> sl;
    for (int x = int(threadIdx.x) & ((1 << sl) - 1); x < run; x += 1 << sl) {
      const int2 t = place(side, 0, b.nrun[side], x);
      for (int k = int(threadIdx.x) >> sl; k < rows; k += kU * step) {
        int off[kU], pos[kU];
        bool ok[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          ok[u] = k + u * step < rows;
          const int2 r = sh.row[side][ok[u] ? k + u * step : 0];
          off[u] = r.x + t.x;
          pos[u] = rel_pos(r.y + t.y);
        }
        body(off, pos, ok);
      }
    }
  };
  const int from = dir == 0 ? 0 : 1;
  const double* src = (dir == 0 ? blk : mat) + sh.base[from];
  double* dst = (dir == 0 ? mat : blk) + sh.base[from ^ 1];
  each(from, [&](const int(&off)[kU], const int(&pos)[kU], const bool(&ok)[kU]) {
    double v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (ok[u]) v[u] = src[off[u]];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (ok[u]) sh.buf[pos[u]] = v[u];
  });
  __syncthreads();
  each(from ^ 1, [&](const int(&off)[kU], const int(&pos)[kU], const bool(&ok)[kU]) {
    double v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (ok[u]) v[u] = sh.buf[pos[u]];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (ok[u]) dst[off[u]] = v[u];
  });
}

// ---- copies by leg tables --------------------------------------------------------

// A task's legs with their divisions prepared: extent, its FastDiv's m and l,
// stride of the strided side.
struct alignas(16) RelLegTab {
  long long blk_off, mat_base;
  int32_t n, pad[3];
  int4 leg[kMaxRank];  // contiguous side's order, innermost first
};

__host__ __device__ inline void rel_make_legs(const RelTask& t, RelLegTab& b) {
  int L[kMaxRank];
  long long sb[kMaxRank], sm[kMaxRank];
  b.blk_off = t.blk_off;
  b.mat_base = t.mat_base;
  b.n = rel_task_legs(t, L, sb, sm);
  for (int j = 0; j < b.n; ++j) {
    FastDiv f;
    f.init(uint32_t(L[j]));
    b.leg[j] = make_int4(int(f.d), int(f.m), int(f.l), int(sm[j]));
  }
}

// Whether a task's offsets on the strided side fit 32 bits.
inline bool rel_narrow(const RelTask& t) {
  long long span = 0;
  for (int i = 0; i < t.rank; ++i) span += (t.shape[i] - 1) * (long long)t.mstride[i];
  return span < (1ll << 31);
}

struct RelLegs {
  int4 leg[kMaxRank];
};

// Elements [begin, end) of one task by the leg table (32-bit offsets), eight
// a thread: a chunk of 2048 in one pass, the loads of all before the stores.
template <int kThreads>
__device__ __forceinline__ void relayout_legs(RelLegs& sh, const RelLegTab& b, int begin, int end, double* blk,
                                              double* mat, int dir, double alpha, double beta) {
  constexpr int kU = 8;
  const int n = b.n;
  if (int(threadIdx.x) < n) sh.leg[threadIdx.x] = b.leg[threadIdx.x];
  blk += b.blk_off;
  mat += b.mat_base;
  __syncthreads();
  for (int e0 = begin + int(threadIdx.x); e0 < end; e0 += kU * kThreads) {
    uint32_t rem[kU];
    int mo[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int e = e0 + u * kThreads;
      rem[u] = uint32_t(e < end ? e : e0);
      mo[u] = 0;
    }
    for (int j = 0; j < n; ++j) {
      const int4 g = sh.leg[j];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const uint32_t q = (__umulhi(rem[u], uint32_t(g.y)) + rem[u]) >> g.z;
        mo[u] += int(rem[u] - q * uint32_t(g.x)) * g.w;
        rem[u] = q;
      }
    }
    double v[kU];
    if (dir == 0) {
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (e0 + u * kThreads < end) v[u] = blk[e0 + u * kThreads];
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (e0 + u * kThreads < end) mat[mo[u]] = v[u];
    } else {
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (e0 + u * kThreads < end) v[u] = mat[mo[u]];
      // (no FP64 arithmetic in a plain copy, see relayout_range)
      if (alpha != 1.0 || beta != 0.0) {
#pragma unroll
        for (int u = 0; u < kU; ++u)
          if (e0 + u * kThreads < end) {
            v[u] = alpha * v[u];
            if (beta != 0.0) v[u] += beta * blk[e0 + u * kThreads];
          }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (e0 + u * kThreads < end) blk[e0 + u * kThreads] = v[u];
    }
  }
}

}  // namespace bst
