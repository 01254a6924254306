// Relayout kernel (block permute / fuse / sector-matrix gather and scatter)
// and small helper kernels.
//
// Every relayout is a list of tasks; a task moves one contiguous block,
// row-major over its own leg order, to or from a strided region of another
// buffer.  The work is split into chunks of kChunk elements, one CTA per
// chunk, so uneven block sizes load-balance across the 152 SMs; large
// transposing copies go by boxes instead, one CTA per box.
//
// What bounds it: small copies, their latency (table loads, then the
// elements; eight of them in flight a thread).  With the divisions by the
// legs' extents prepared in every thread, and four elements in flight, the
// three copies of an FP64 corner contraction (odd sizes, 18 MB) took 39 us,
// now 32, the 78 of a D = 4, chi = 16 move 640 us, now 495.  Large ones whose
// innermost legs differ: each 8-byte store of a warp went to another sector,
// 2.0 TB/s; through boxes 3.7 TB/s (permutation 2031 of a D = 8, chi = 256
// tensor, 289 MB: 269 -> 155 us), bound by the instructions of the two passes.
#include <algorithm>

#include "bst_internal.h"
#include "relayout_dev.cuh"

namespace bst {

ProfScope::ProfScope(Ctx* ctx, cudaStream_t st, const char* cls, double flops, double bytes) : c(ctx), s(st) {
  if (!c->prof) return;
  while (c->evpool.size() < c->evused + 2) {
    cudaEvent_t e;
    BST_CUDA(cudaEventCreate(&e));
    c->evpool.push_back(e);
  }
  ProfRec r{cls, c->evpool[c->evused], c->evpool[c->evused + 1], flops, bytes};
  c->evused += 2;
  BST_CUDA(cudaEventRecord(r.a, s));
  idx = long(c->recs.size());
  c->recs.push_back(r);
}

ProfScope::~ProfScope() {
  if (idx >= 0) cudaEventRecord(c->recs[idx].b, s);
}

constexpr int kChunk = 2048;
constexpr int kRelThreads = 256;
// Copies through boxes: four runs a thread, six CTAs an SM (a few spilled
// registers included: 155 us for the D = 8, chi = 256 permutation below, with
// four CTAs 180, with two runs and eight CTAs 172).
constexpr int kBoxU = 4, kBoxCtas = 6;
constexpr double kBoxElems = 4e6;  // copies of fewer elements stay in the L2 cache, see launch_relayout

std::vector<int2> relayout_chunks(const std::vector<RelTask>& t) {
  std::vector<int2> ch;
  for (int i = 0; i < int(t.size()); ++i)
    for (int s = 0; s < t[i].n; s += kChunk) ch.push_back(make_int2(i, s));
  return ch;
}

void DevRelayout::alloc(int64_t max_tasks, int64_t max_chunks) {
  const size_t nt = size_t(std::max<int64_t>(max_tasks, 1)), nc = size_t(std::max<int64_t>(max_chunks, 1));
  const size_t olegs = (sizeof(RelTask) * nt + 255) / 256 * 256, ochunks = olegs + sizeof(RelLegTab) * nt;
  BST_CUDA(cudaMalloc(&mem, ochunks + sizeof(int2) * nc));
  tasks = reinterpret_cast<RelTask*>(mem);
  legs = reinterpret_cast<RelLegTab*>(static_cast<char*>(mem) + olegs);
  chunks = reinterpret_cast<int2*>(static_cast<char*>(mem) + ochunks);
}

struct RelLists {
  const RelTask* tasks[3];
  RelLegTab* legs[3];
  int n[3];
};
__global__ void rel_legs_kernel(RelLists l) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y;
  if (i < l.n[r]) rel_make_legs(l.tasks[r][i], l.legs[r][i]);
}

// Beside a capture they are made at once, on a stream aside: a graph that
// copies without them is slower for as long as it lives.
void prepare_legs(Ctx* ctx, std::initializer_list<DevRelayout*> rels, cudaStream_t s) {
  DevRelayout* todo[3];
  int k = 0, longest = 0;
  for (DevRelayout* r : rels)
    if (r->narrow && !r->legs_made && r->ntasks > 0) todo[k++] = r, longest = std::max(longest, r->ntasks);
  if (k == 0) return;
  RelLists l{};
  for (int i = 0; i < k; ++i) l.tasks[i] = todo[i]->tasks, l.legs[i] = todo[i]->legs, l.n[i] = todo[i]->ntasks;
  auto make = [&](cudaStream_t t) {
    rel_legs_kernel<<<dim3(unsigned((longest + 63) / 64), unsigned(k)), 64, 0, t>>>(l);
    BST_CUDA(cudaGetLastError());
    count_launch(ctx);
    BST_CUDA(cudaStreamSynchronize(t));  // (the next launch may be on another stream)
  };
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  BST_CUDA(cudaStreamIsCapturing(s, &cap));
  if (cap == cudaStreamCaptureStatusNone) {
    make(s);
  } else {
    Aside aside;
    make(aside.s);
  }
  for (int i = 0; i < k; ++i) todo[i]->legs_made = true;
}

void DevRelayout::upload(Ctx* ctx, const std::vector<RelTask>& t) {
  free_all();
  ntasks = int(t.size());
  elems = 0;
  narrow = true;
  for (auto& x : t) elems += x.n, narrow = narrow && rel_narrow(x);
  std::vector<int2> ch;
  std::vector<RelBox> hb;
  if (narrow && elems >= kBoxElems) {
    // a sample of the blocks decides: up to 64, by their elements
    double in = 0, of = 0;
    for (int i = 0; i < ntasks; i += (ntasks + 63) / 64) {
      RelBox b;
      rel_make_box(t[i], b);
      of += t[i].n;
      if (rel_box_pays(t[i], b)) in += t[i].n;
    }
    if (in > 0.5 * of) {
      hb.resize(ntasks);
      for (int i = 0; i < ntasks; ++i) rel_make_box(t[i], hb[i]);
    }
  }
  if (!hb.empty()) {  // a CTA per box
    for (int i = 0; i < ntasks; ++i)
      for (int k = 0; k < (t[i].n > 0 ? hb[i].ntiles : 0); ++k) ch.push_back(make_int2(i, k));
    BST_CUDA(cudaMalloc(&boxes, sizeof(RelBox) * ntasks));
    BST_CUDA(cudaMemcpy(boxes, hb.data(), sizeof(RelBox) * ntasks, cudaMemcpyHostToDevice));
  } else {
    ch = relayout_chunks(t);
  }
  nchunks = int(ch.size());
  if (nchunks == 0) return;
  alloc(ntasks, nchunks);
  BST_CUDA(cudaMemcpy(tasks, t.data(), sizeof(RelTask) * ntasks, cudaMemcpyHostToDevice));
  BST_CUDA(cudaMemcpy(chunks, ch.data(), sizeof(int2) * nchunks, cudaMemcpyHostToDevice));
  if (!boxes) prepare_legs(ctx, {this}, 0);
}

void DevRelayout::free_all() {
  if (mem) cudaFree(mem);
  if (boxes) cudaFree(boxes);
  *this = DevRelayout{};
}

void* DevBuf::get(size_t need, cudaStream_t s) {
  if (need <= bytes) return p;
  if (p) {
    // the stream may still read the old buffer
    BST_CUDA(cudaStreamSynchronize(s));
    BST_CUDA(cudaFree(p));
    p = nullptr;
    bytes = 0;
  }
  size_t nb = std::max(need, size_t(256));
  if (cudaMalloc(&p, nb) != cudaSuccess) {
    cudaGetLastError();
    p = nullptr;
    throw Error(BST_E_OOM, "device workspace allocation failed");
  }
  bytes = nb;
  return p;
}

void DevBuf::free_all() {
  if (p) cudaFree(p);
  p = nullptr;
  bytes = 0;
}

// dir 0: mat[strided] = blk[contiguous]
// dir 1: blk[contiguous] = alpha * mat[strided] + beta * blk   (beta == 0: overwrite)
__global__ void __launch_bounds__(kRelThreads) relayout_kernel(const RelTask* __restrict__ tasks,
                                                               const int2* __restrict__ chunks,
                                                               double* blk, double* mat, int dir,
                                                               double alpha, double beta) {
  const int2 c = chunks[blockIdx.x];
  const RelTask& t = tasks[c.x];
  relayout_range<kRelThreads>(t, c.y, min(t.n, c.y + kChunk), blk, mat, dir, alpha, beta);
}

__global__ void __launch_bounds__(kRelThreads) relayout_legs_kernel(const RelTask* __restrict__ tasks,
                                                                    const RelLegTab* __restrict__ legs,
                                                                    const int2* __restrict__ chunks, double* blk,
                                                                    double* mat, int dir, double alpha, double beta) {
  __shared__ RelLegs sh;
  grid_trigger();
  const int2 c = chunks[blockIdx.x];
  const int end = min(tasks[c.x].n, c.y + kChunk);
  grid_wait();
  relayout_legs<kRelThreads>(sh, legs[c.x], c.y, end, blk, mat, dir, alpha, beta);
}

// Both operands' gathers of a contraction in one launch.
struct RelPart {
  const RelTask* tasks;
  const RelLegTab* legs;
  const int2* chunks;
  double *blk, *mat;
};
__global__ void __launch_bounds__(kRelThreads) relayout_pair_kernel(RelPart a, RelPart b, int na) {
  __shared__ RelLegs sh;
  grid_trigger();
  const bool first = int(blockIdx.x) < na;
  const RelPart p = first ? a : b;
  const int2 c = p.chunks[int(blockIdx.x) - (first ? 0 : na)];
  relayout_legs<kRelThreads>(sh, p.legs[c.x], c.y, min(p.tasks[c.x].n, c.y + kChunk), p.blk, p.mat, 0, 1.0, 0.0);
}

__global__ void __launch_bounds__(kRelThreads, kBoxCtas) relayout_box_kernel(const RelBox* __restrict__ boxes,
                                                                             const int2* __restrict__ tiles, double* blk,
                                                                             double* mat, int dir) {
  __shared__ RelShared sh;
  const int2 c = tiles[blockIdx.x];
  relayout_box<kRelThreads, kBoxU>(sh, boxes[c.x], c.y, blk, mat, dir);
}

// Boxes only where rel_box_pays.  A straight copy reaches 5.8 TB/s when a
// warp's elements stay on a few lines of the strided side, and what it
// scatters is merged in the L2 cache while both sides fit there; a box pays
// for its tables and two more barriers, and more when few runs, or a small
// block, leave its threads idle.  Microseconds straight / by boxes:
//   by the lines of a warp, blocks (n, a, b) -> (n, b, a) of 40 M elements:
//     b a = 16 x 2 (2 lines) 107 / 132, 5 x 16 (5) 111 / 186, 6 x 16 (6)
//     111 / 148, 16 x 16 (16) 188 / 132; rank 6, legs of 5 to 9, 15.5 M
//     elements: 7 or 8 lines 62 / 83, 32 lines 135 / 75 and 91 / 81;
//   by the runs, (m, n) -> (n, m): 5 M elements, m = 2 (4 lines) 29 / 50, 5
//     (10) 42 / 48, 12 (24, one run) 49 / 41, 16 (32, 16 runs) 55 / 31; 40 M
//     elements 240 / 321, 432 / 299, 603 / 244, 722 / 179;
//   by the size, 18.8 M elements in blocks of 900: 145 / 136, 5.1 M in blocks
//     of 73 k 43 / 30, 60 M in blocks of 0.7 M 429 / 221.
// Below 4 M elements: a D = 4, chi = 64 permutation takes 14 us by boxes, 10
// straight, the odd-sized FP64 corner's copies 89 and 32.
// behind: the previous kernel of the stream is this call's, launch_behind.
void launch_relayout(Ctx* ctx, const DevRelayout& r, const double* blk, double* mat, int dir, double alpha,
                     double beta, cudaStream_t s, bool behind) {
  if (r.nchunks == 0) return;
  ProfScope ps(ctx, s, "relayout", 0.0, 16.0 * r.elems);
  if (r.boxes) {
    // (only uploaded lists have boxes, and those are permutations, fusions and
    // gathers: plain copies)
    BST_REQUIRE(dir == 0 || (alpha == 1.0 && beta == 0.0), BST_E_UNSUPPORTED, "copies by boxes are plain ones");
    relayout_box_kernel<<<r.nchunks, kRelThreads, 0, s>>>(r.boxes, r.chunks, const_cast<double*>(blk), mat, dir);
  } else if (r.legs_made)
    launch_behind(behind, relayout_legs_kernel, dim3(unsigned(r.nchunks)), kRelThreads, 0, s, (const RelTask*)r.tasks,
                  (const RelLegTab*)r.legs, (const int2*)r.chunks, const_cast<double*>(blk), mat, dir, alpha, beta);
  else
    relayout_kernel<<<r.nchunks, kRelThreads, 0, s>>>(r.tasks, r.chunks, const_cast<double*>(blk), mat, dir, alpha,
                                                      beta);
  BST_CUDA(cudaGetLastError());
  count_launch(ctx);
}

void launch_gathers(Ctx* ctx, const DevRelayout& ra, const double* a, double* Am, const DevRelayout& rb,
                    const double* b, double* Bm, cudaStream_t s) {
  if (ra.nchunks == 0 || rb.nchunks == 0 || !ra.legs_made || !rb.legs_made) {
    launch_relayout(ctx, ra, a, Am, 0, 1.0, 0.0, s);
    launch_relayout(ctx, rb, b, Bm, 0, 1.0, 0.0, s);
    return;
  }
  ProfScope ps(ctx, s, "relayout", 0.0, 16.0 * (ra.elems + rb.elems));
  relayout_pair_kernel<<<ra.nchunks + rb.nchunks, kRelThreads, 0, s>>>(
      RelPart{ra.tasks, ra.legs, ra.chunks, const_cast<double*>(a), Am},
      RelPart{rb.tasks, rb.legs, rb.chunks, const_cast<double*>(b), Bm}, ra.nchunks);
  BST_CUDA(cudaGetLastError());
  count_launch(ctx);
}

__global__ void scale_kernel(double* x, long long n, const double* inv) {
  const double f = 1.0 / sqrt(*inv);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    x[i] *= f;
}

// x /= sqrt(*sumsq)
void launch_scale(Ctx* ctx, double* x, int64_t n, const double* dev_sumsq, cudaStream_t s) {
  if (n == 0) return;
  int grid = int(std::min<int64_t>((n + 255) / 256, 152 * 8));
  scale_kernel<<<grid, 256, 0, s>>>(x, n, dev_sumsq);
  BST_CUDA(cudaGetLastError());
  count_launch(ctx);
}

// Sum of squares in FP64: per-CTA partial sums, then one CTA adds them in a
// fixed order (deterministic result).
__global__ void sumsq_partial(const double* x, long long n, double* part) {
  __shared__ double sh[256];
  double acc = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    acc += x[i] * x[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void sumsq_final(const double* part, int np, double* out) {
  __shared__ double sh[256];
  double acc = 0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) acc += part[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

// Weighted sum of squares sum_i w_i x_i^2 (per-CTA partials, then one CTA in
// a fixed order): the Frobenius norm of an SU(2) tensor from its reduced
// blocks, w = 2J+1 of the element's block.
__global__ void sumsq_w_partial(const double* x, const double* w, long long n, double* part) {
  __shared__ double sh[256];
  double acc = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    acc += w[i] * x[i] * x[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int k = 128; k > 0; k >>= 1) {
    if (threadIdx.x < k) sh[threadIdx.x] += sh[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

void launch_sumsq_w(Ctx* ctx, const double* x, const double* w, int64_t n, double* dev_out, cudaStream_t s) {
  int grid = int(std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 304)));
  double* part = (double*)ctx->buf("sumsq.part", sizeof(double) * 304, s);
  sumsq_w_partial<<<grid, 256, 0, s>>>(x, w, n, part);
  sumsq_final<<<1, 256, 0, s>>>(part, grid, dev_out);
  BST_CUDA(cudaGetLastError());
  count_launch(ctx, 2);
}

void launch_sumsq(Ctx* ctx, const double* x, int64_t n, double* dev_out, cudaStream_t s) {
  int grid = int(std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 304)));
  double* part = (double*)ctx->buf("sumsq.part", sizeof(double) * 304, s);
  sumsq_partial<<<grid, 256, 0, s>>>(x, n, part);
  sumsq_final<<<1, 256, 0, s>>>(part, grid, dev_out);
  BST_CUDA(cudaGetLastError());
  count_launch(ctx, 2);
}

__global__ void fill_kernel(double* x, long long n, double v) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    x[i] = v;
}

void launch_fill(Ctx* ctx, double* x, int64_t n, double v, cudaStream_t s) {
  if (n == 0) return;
  int grid = int(std::min<int64_t>((n + 255) / 256, 152 * 8));
  fill_kernel<<<grid, 256, 0, s>>>(x, n, v);
  BST_CUDA(cudaGetLastError());
  count_launch(ctx);
}

}  // namespace bst
