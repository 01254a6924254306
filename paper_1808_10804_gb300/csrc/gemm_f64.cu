// Plain FP64 grouped GEMM on the FP64 tensor path (DMMA, mma.sync m8n8k4).
//
// This is the "plain FP64 GPU path": every matched sector GEMM of a
// contraction in one launch, one 64x64 output tile per CTA, operands read
// through generic element strides so transposed views need no copy.
#include <algorithm>

#include "bst_internal.h"
#include "relayout_dev.cuh"

namespace bst {

const int kF64TileM = 64;
const int kF64TileN = 64;
constexpr int kBK = 16;
constexpr int kPad = 2;
constexpr int kSms = 152;

// CTAs an SM: two, or three for lists of nearly equal tiles (85 % cost three
// quarters of the dearest or more), more than two would take at once.  Two CTAs
// that start together end together, so that equal tiles go to the SMs in
// pairs: 450 tiles of depth 256 1.17 ms against 0.88 with three, 1024 of 512
// 4.64 against 4.07, 360 of 300 1.20 against 1.03.  Unequal ones are spread
// better by two, which leave more of them to the SMs that are free first: the
// D=8, chi=256 FP64 move's products of 2976 x 160 x 2976 12.7 s against 14.2,
// a D=6, chi=128 corner 2.50 ms against 2.67, the odd-sized corner 0.44 against
// 0.52, the products of 40 eigenproblems of 133 values 4.3 against 5.8 (Gram
// matrices, whose tiles are whole, half and empty by turns, always take two).
int f64_ctas(const std::vector<GemmProb>& p) {
  // 8x8 products of a problem's tiles, times K: in whole tiles, along its last
  // column and row of tiles, in the corner
  struct Kind {
    long long n, cost;
  };
  auto kinds = [](const GemmProb& x, Kind (&k)[4]) {
    const long long m = x.M / kF64TileM, n = x.N / kF64TileN;
    const int r = (x.M % kF64TileM + 7) / 8, c = (x.N % kF64TileN + 7) / 8;
    k[0] = {m * n, 64ll * x.K};
    k[1] = {c ? m : 0, 8ll * c * x.K};
    k[2] = {r ? n : 0, 8ll * r * x.K};
    k[3] = {r && c ? 1 : 0, (long long)r * c * x.K};
  };
  Kind k[4];
  long long dearest = 0, tiles = 0, dear = 0;
  for (auto& x : p) {
    kinds(x, k);
    for (auto& y : k) dearest = y.n ? std::max(dearest, y.cost) : dearest, tiles += y.n;
  }
  for (auto& x : p) {
    kinds(x, k);
    for (auto& y : k) dear += 4 * y.cost >= 3 * dearest ? y.n : 0;
  }
  return tiles > 2 * kSms && 20 * dear >= 17 * tiles ? 3 : 2;
}

void DevGemm::upload(const std::vector<GemmProb>& p, int tm, int tn, int order, cudaStream_t s) {
  free_all();
  auto copy = [&](void* dst, const void* src, size_t n) {
    BST_CUDA(cudaMemcpyAsync(dst, src, n, cudaMemcpyHostToDevice, s));
  };
  nprobs = int(p.size());
  flops = 0;
  for (auto& x : p) flops += 2.0 * double(x.M) * x.N * x.K;
  std::vector<int32_t> tp, ti;
  for (int i = 0; i < nprobs; ++i) {
    int mt = (p[i].M + tm - 1) / tm, nt = (p[i].N + tn - 1) / tn;
    for (int t = 0; t < mt * nt; ++t) {
      tp.push_back(i);
      ti.push_back(t);
    }
  }
  ntiles = int(tp.size());
  ctas = f64_ctas(p);
  std::vector<int64_t> wo(std::max(nprobs, 1), 0);
  wtot = 0;
  maxK = 0;
  for (int i = 0; i < nprobs; ++i) {
    wo[i] = wtot;
    wtot += int64_t(p[i].M) * p[i].N;
    maxK = std::max(maxK, p[i].K);
  }
  hw_off.assign(wo.begin(), wo.begin() + nprobs);
  if (order == 1) {
    std::vector<int> idx(ntiles);
    for (int i = 0; i < ntiles; ++i) idx[i] = i;
    std::stable_sort(idx.begin(), idx.end(), [&](int x, int y) { return p[tp[x]].K > p[tp[y]].K; });
    std::vector<int32_t> tp2(ntiles), ti2(ntiles);
    for (int i = 0; i < ntiles; ++i) {
      tp2[i] = tp[idx[i]];
      ti2[i] = ti[idx[i]];
    }
    tp.swap(tp2);
    ti.swap(ti2);
  }
  if (nprobs) {
    BST_CUDA(cudaMalloc(&probs, sizeof(GemmProb) * nprobs));
    copy(probs, p.data(), sizeof(GemmProb) * nprobs);
  }
  if (nprobs) {
    BST_CUDA(cudaMalloc(&w_off, sizeof(int64_t) * nprobs));
    copy(w_off, wo.data(), sizeof(int64_t) * nprobs);
  }
  if (ntiles) {
    BST_CUDA(cudaMalloc(&tile_prob, sizeof(int32_t) * ntiles));
    BST_CUDA(cudaMalloc(&tile_idx, sizeof(int32_t) * ntiles));
    copy(tile_prob, tp.data(), sizeof(int32_t) * ntiles);
    copy(tile_idx, ti.data(), sizeof(int32_t) * ntiles);
  }
  BST_CUDA(cudaStreamSynchronize(s));
}

void DevGemm::free_all() {
  if (probs) cudaFree(probs);
  if (tile_prob) cudaFree(tile_prob);
  if (tile_idx) cudaFree(tile_idx);
  if (w_off) cudaFree(w_off);
  w_off = nullptr;
  probs = nullptr;
  tile_prob = tile_idx = nullptr;
  ntiles = nprobs = 0;
}

__device__ __forceinline__ void dmma(double& c0, double& c1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
               : "+d"(c0), "+d"(c1)
               : "d"(a), "d"(b));
}

// One 64x64 output tile of problem p over the K range [kb, ke), written to
// out[m * om + n * on].  128 threads = 4 warps, up to 4x4 DMMA tiles of 8x8
// each.  The operand tiles are double-buffered in shared memory: the next K
// block's loads are in flight (in registers) while the current block is
// multiplied.
//
// What bounds it: the DMMA units, one a scheduler (an 8x8x4 product takes one
// about 600 cycles: 2048 x 2048 x 512 in 4.07 ms at 2070 MHz), so a product is
// issued only where it counts:
//   * whole tiles: a warp takes a quarter, 4x4 products from 4 + 4 fragments;
//   * tiles at an edge: the 8x8 tiles inside M and N are dealt to the warps one
//     by one (an odd-sized FP64 corner, 0.33 GFLOP: 594 -> 439 us).  Whole tiles
//     dealt likewise need 16 + 16 fragments, and registers that leave room for
//     two CTAs an SM only: 4096 x 4096 x 4 180 -> 132 us, 2048 x 2048 x 512 4.65
//     -> 4.07 ms with quarters and three (f64_ctas);
//   * of a Gram matrix (both operands the same) only those on and above its
//     diagonal; the sums below are the same products in the same order, so
//     they are mirrored.
constexpr int kLd = (kF64TileM * kBK) / 128;  // elements of a 64 x 16 tile per thread
__device__ __forceinline__ void f64_tile(const GemmProb& p, int m0, int n0, int kb, int ke,
                                         const double* __restrict__ A, const double* __restrict__ B,
                                         double* __restrict__ out, long long om, long long on,
                                         double (*sA)[kBK][kF64TileM + kPad], double (*sB)[kBK][kF64TileN + kPad],
                                         int turn) {
  const int tid = threadIdx.x, lane = tid & 31, part = ((tid >> 5) + turn) & 3;
  const int g = lane >> 2, tg = lane & 3;
  const bool sym = A == B && p.a_off == p.b_off && p.M == p.N && p.a_m == p.b_n && p.a_k == p.b_k;
  if (sym && m0 > n0) return;  // (uniform) below the diagonal
  // this warp's 8x8 tiles: every fourth of the tile's, row by row (in a Gram
  // matrix's diagonal tile the columns from the row's own on)
  const int r8 = min(8, (p.M - m0 + 7) >> 3), c8 = min(8, (p.N - n0 + 7) >> 3);
  const bool tri = sym && m0 == n0;
  const int total = tri ? r8 * (r8 + 1) / 2 : r8 * c8, cnt = (total - part + 3) >> 2;
  const bool whole = total == 64;
  const int wi = (part >> 1) * 4, wj = (part & 1) * 4;
  // row and column of the t-th (in 8s), a byte each four to a register
  uint32_t at[4] = {};
  auto row8 = [&](int t) { return int(at[t / 4] >> (t % 4 * 8 + 3) & 7u) * 8; };
  auto col8 = [&](int t) { return int(at[t / 4] >> (t % 4 * 8) & 7u) * 8; };
  if (whole) {
#pragma unroll
    for (int t = 0; t < 16; ++t) at[t / 4] |= uint32_t((wi + t / 4) << 3 | (wj + t % 4)) << (t % 4 * 8);
  } else {
    int i = 0, j = part;  // (counted in a row that starts at column 0, then moved)
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      while (i < r8 && j >= c8) ++i, j -= c8 - (tri ? i : 0);
      if (t < cnt) at[t / 4] |= uint32_t(i << 3 | j) << (t % 4 * 8);
      j += 4;
    }
  }
  double acc[16][2];
#pragma unroll
  for (int t = 0; t < 16; ++t) acc[t][0] = acc[t][1] = 0.0;
  const double* Ap = A + p.a_off;
  const double* Bp = B + p.b_off;
  double ra[kLd], rb[kLd];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < kLd; ++u) {
      const int e = tid + u * 128;
      const int m = e / kBK, k = e % kBK;
      const int gm = m0 + m, gn = n0 + m, gk = k0 + k;
      ra[u] = (gm < p.M && gk < ke) ? Ap[(long long)gm * p.a_m + (long long)gk * p.a_k] : 0.0;
      rb[u] = (gn < p.N && gk < ke) ? Bp[(long long)gn * p.b_n + (long long)gk * p.b_k] : 0.0;
    }
  };
  if (kb < ke) fetch(kb);
  int buf = 0;
  for (int k0 = kb; k0 < ke; k0 += kBK, buf ^= 1) {
#pragma unroll
    for (int u = 0; u < kLd; ++u) {
      const int e = tid + u * 128;
      sA[buf][e % kBK][e / kBK] = ra[u];
      sB[buf][e % kBK][e / kBK] = rb[u];
    }
    __syncthreads();
    if (k0 + kBK < ke) fetch(k0 + kBK);
    // (k steps past the end of the range hold only zero padding)
    const int kn = min(kBK, ke - k0);
#pragma unroll
    for (int kk = 0; kk < kBK; kk += 4) {
      if (kk >= kn) break;
      const double* a = &sA[buf][kk + tg][g];
      const double* b = &sB[buf][kk + tg][g];
      if (whole) {
        double af[4], bf[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) af[t] = a[(wi + t) * 8], bf[t] = b[(wj + t) * 8];
#pragma unroll
        for (int t = 0; t < 16; ++t) dmma(acc[t][0], acc[t][1], af[t / 4], bf[t % 4]);
      } else {
#pragma unroll
        for (int t = 0; t < 16; ++t) {
          if (t >= cnt) break;
          dmma(acc[t][0], acc[t][1], a[row8(t)], b[col8(t)]);
        }
      }
    }
  }
#pragma unroll
  for (int t = 0; t < 16; ++t) {
    if (t >= cnt) break;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int gm = m0 + row8(t) + g;
      const int gn = n0 + col8(t) + tg * 2 + h;
      if (gm >= p.M || gn >= p.N) continue;
      out[(long long)gm * om + (long long)gn * on] = acc[t][h];
      if (sym && row8(t) + m0 < col8(t) + n0) out[(long long)gn * om + (long long)gm * on] = acc[t][h];
    }
  }
}

template <int kCtas>  // an SM
__global__ void __launch_bounds__(128, kCtas) gemm_f64_kernel(const GemmProb* __restrict__ probs,
                                                       const int32_t* __restrict__ tile_prob,
                                                       const int32_t* __restrict__ tile_idx,
                                                       const double* __restrict__ A,
                                                       const double* __restrict__ B, double* __restrict__ C) {
  __shared__ double sA[2][kBK][kF64TileM + kPad];
  __shared__ double sB[2][kBK][kF64TileN + kPad];
  grid_trigger();
  const GemmProb p = probs[tile_prob[blockIdx.x]];
  const int nt = (p.N + kF64TileN - 1) / kF64TileN;
  const int m0 = (tile_idx[blockIdx.x] / nt) * kF64TileM;
  const int n0 = (tile_idx[blockIdx.x] % nt) * kF64TileN;
  grid_wait();
  f64_tile(p, m0, n0, 0, p.K, A, B, C + p.c_off, p.c_m, p.c_n, sA, sB, int(blockIdx.x));
}

// Split-K: CTA (tile, s) computes the partial product over the s-th K slice
// (slices of a multiple of 16) into W[s][problem][m][n]; the reduction adds
// the slices in a fixed order (deterministic result).
__global__ void __launch_bounds__(128, 2) gemm_f64_splitk_kernel(const GemmProb* __restrict__ probs,
                                                              const int32_t* __restrict__ tile_prob,
                                                              const int32_t* __restrict__ tile_idx,
                                                              const double* __restrict__ A,
                                                              const double* __restrict__ B, double* __restrict__ W,
                                                              const int64_t* __restrict__ w_off, long long wtot,
                                                              int ksplit) {
  __shared__ double sA[2][kBK][kF64TileM + kPad];
  __shared__ double sB[2][kBK][kF64TileN + kPad];
  const int pi = tile_prob[blockIdx.x];
  const GemmProb p = probs[pi];
  const int nt = (p.N + kF64TileN - 1) / kF64TileN;
  const int m0 = (tile_idx[blockIdx.x] / nt) * kF64TileM;
  const int n0 = (tile_idx[blockIdx.x] % nt) * kF64TileN;
  const int kc = ((p.K + ksplit - 1) / ksplit + kBK - 1) / kBK * kBK;
  const int kb = min(p.K, int(blockIdx.y) * kc), ke = min(p.K, kb + kc);
  f64_tile(p, m0, n0, kb, ke, A, B, W + blockIdx.y * wtot + w_off[pi], p.N, 1, sA, sB,
           int(blockIdx.x + blockIdx.y));
}

__global__ void gemm_f64_reduce_kernel(const GemmProb* __restrict__ probs, const double* __restrict__ W,
                                       const int64_t* __restrict__ w_off, long long wtot, int ksplit,
                                       double* __restrict__ C) {
  const GemmProb p = probs[blockIdx.y];
  const long long n = (long long)p.M * p.N;
  const double* w = W + w_off[blockIdx.y];
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int s = 0; s < ksplit; ++s) v += w[s * wtot + e];
    const long long m = e / p.N, c = e - m * p.N;
    C[p.c_off + m * p.c_m + c * p.c_n] = v;
  }
}

DevGemm* get_dev_gemm(Ctx* ctx, const std::string& key, const std::vector<GemmProb>& probs) {
  std::lock_guard<std::mutex> lk(ctx->mu);
  auto it = ctx->gplans.find(key);
  if (it != ctx->gplans.end()) return it->second.get();
  auto g = std::make_unique<DevGemm>();
  g->upload(probs, kF64TileM, kF64TileN);
  DevGemm* raw = g.get();
  ctx->gplans[key] = std::move(g);
  return raw;
}

void launch_gemm_f64_splitk(Ctx* ctx, const DevGemm& g, int ksplit, const double* A, const double* B, double* C,
                            cudaStream_t s, const char* ws) {
  if (g.ntiles == 0) return;
  if (ksplit <= 1) {
    launch_gemm_f64(ctx, g, A, B, C, s);
    return;
  }
  double* W = (double*)ctx->buf(ws, sizeof(double) * std::max<int64_t>(1, g.wtot * ksplit), s);
  ProfScope ps(ctx, s, "gemm_f64", g.flops, 0.0);
  gemm_f64_splitk_kernel<<<dim3(unsigned(g.ntiles), unsigned(ksplit)), 128, 0, s>>>(
      g.probs, g.tile_prob, g.tile_idx, A, B, W, g.w_off, g.wtot, ksplit);
  gemm_f64_reduce_kernel<<<dim3(64, unsigned(g.nprobs)), 256, 0, s>>>(g.probs, W, g.w_off, g.wtot, ksplit, C);
  BST_CUDA(cudaGetLastError());
  count_launch(ctx, 2);
}

void launch_ksplit_reduce(Ctx* ctx, const DevGemm& g, const double* W, int ksplit, double* C, cudaStream_t s) {
  if (g.nprobs == 0) return;
  gemm_f64_reduce_kernel<<<dim3(64, unsigned(g.nprobs)), 256, 0, s>>>(g.probs, W, g.w_off, g.wtot, ksplit, C);
  BST_CUDA(cudaGetLastError());
  count_launch(ctx);
}

void launch_gemm_f64(Ctx* ctx, const DevGemm& g, const double* A, const double* B, double* C, cudaStream_t s,
                     bool behind) {
  if (g.ntiles == 0) return;
  ProfScope ps(ctx, s, "gemm_f64", g.flops, 0.0);
  const bool three = g.ctas == 3 && A != B;  // (equal operands: Gram matrices)
  launch_behind(behind, three ? gemm_f64_kernel<3> : gemm_f64_kernel<2>, dim3(unsigned(g.ntiles)), 128, 0, s,
                (const GemmProb*)g.probs, (const int32_t*)g.tile_prob, (const int32_t*)g.tile_idx, A, B, C);
  BST_CUDA(cudaGetLastError());
  count_launch(ctx);
}

}  // namespace bst
