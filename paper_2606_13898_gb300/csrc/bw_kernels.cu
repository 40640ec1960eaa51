// Bandwidth- and latency-bound kernels of the HiLo-Token hot path:
//   score  (per-token high-frequency energy, Sec. 2.3 frequency map)
//   split  (top-k select with index tie-break, mask union, compaction;
//          Sec. 2.3: high-frequency and mask tokens kept, the rest pooled)
//   pack / unpack / unpack_update (gather + pooling, scatter + broadcast;
//          Sec. 2.3: the packed sequence and its restoration to the grid)
//   layernorm (the block's pre-norm: bf16 or fp16 operand for the next GEMM)
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "internal.h"

namespace hilo {

// ============================================================== score =====
//
// One 128-thread CTA per aligned 2x2 window: thread j owns partial sums j of
// the four members (channel groups j, j+128, ... of 8 channels), so the whole
// window is read in one round trip; the window mean is formed once per
// channel. The 128 partials are combined by the fixed halving tree documented
// in hilo.h (64 and 32 through shared memory, then warp shuffles). Every
// add/mul is an explicit round-to-nearest intrinsic so the compiler cannot
// contract to FMA.

__device__ __forceinline__ void bf16x8_to_f32(const uint4& v, float* f) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}

constexpr int SCORE_THREADS = 128;

// ITERS: groups of 8 channels per thread (d <= 4096: at most 4). Bound by HBM, so by
// the loads that the resident CTAs have in flight: with registers for four groups
// whatever the width, 128x128 tokens of 3072 channels took 18.5 us, 16.8 so (6.0
// TB/s), 64x64 6.8 and 6.3, 128x128 of 1024 10.8 and 8.8. Seven CTAs per SM for three
// groups (6.7 us for 64x64 without the limit), eight for two (64x64 of 2048, in L2, 4.2
// us without, 3.7 so, 3.9 with four groups' registers; 16 images of 1536 34.6 and 35.9);
// for the others the compiler's own count (128x128 of 4096: 21.5 us, 22.3 with five, 26.2
// with a limit of one).
template <int ITERS>
__global__ void __launch_bounds__(SCORE_THREADS, ITERS == 3 ? 7 : ITERS == 2 ? 8 : 0) score_kernel(const __nv_bfloat16* __restrict__ x,
                                                              float* __restrict__ s, int B, int H,
                                                              int W, int d) {
  pdl_wait();
  pdl_trigger();
  __shared__ float part[4][SCORE_THREADS];
  const int j = threadIdx.x;
  const int lane = j & 31;
  const int Hw = H >> 1, Ww = W >> 1;
  const long long nwin = static_cast<long long>(B) * Hw * Ww;
  const int G = d >> 3;
  for (long long w = blockIdx.x; w < nwin; w += gridDim.x) {
    const int b = static_cast<int>(w / (Hw * Ww));
    const int r = static_cast<int>(w % (Hw * Ww));
    const int P = r / Ww, Q = r % Ww;
    const long long t0 = (static_cast<long long>(b) * H + 2 * P) * W + 2 * Q;
    const uint4* ra = reinterpret_cast<const uint4*>(x + t0 * d);
    const uint4* rb = reinterpret_cast<const uint4*>(x + (t0 + 1) * d);
    const uint4* rc = reinterpret_cast<const uint4*>(x + (t0 + W) * d);
    const uint4* rd = reinterpret_cast<const uint4*>(x + (t0 + W + 1) * d);
    uint4 va[ITERS], vb[ITERS], vc[ITERS], vd[ITERS];
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {
      const int g = j + SCORE_THREADS * i;
      if (g < G) {
        va[i] = __ldg(ra + g);
        vb[i] = __ldg(rb + g);
        vc[i] = __ldg(rc + g);
        vd[i] = __ldg(rd + g);
      }
    }
    float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f, acc3 = 0.f;
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {
      if (j + SCORE_THREADS * i >= G) break;
      float fa[8], fb[8], fc[8], fd[8];
      bf16x8_to_f32(va[i], fa);
      bf16x8_to_f32(vb[i], fb);
      bf16x8_to_f32(vc[i], fc);
      bf16x8_to_f32(vd[i], fd);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float m = __fmul_rn(__fadd_rn(__fadd_rn(fa[u], fb[u]), __fadd_rn(fc[u], fd[u])), 0.25f);
        const float ea = __fsub_rn(fa[u], m), eb = __fsub_rn(fb[u], m);
        const float ec = __fsub_rn(fc[u], m), ed = __fsub_rn(fd[u], m);
        acc0 = __fadd_rn(acc0, __fmul_rn(ea, ea));
        acc1 = __fadd_rn(acc1, __fmul_rn(eb, eb));
        acc2 = __fadd_rn(acc2, __fmul_rn(ec, ec));
        acc3 = __fadd_rn(acc3, __fmul_rn(ed, ed));
      }
    }
    part[0][j] = acc0;
    part[1][j] = acc1;
    part[2][j] = acc2;
    part[3][j] = acc3;
    __syncthreads();
    if (j < 32) {
      float v[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        // h = 64: p[j] += p[j+64] (j < 64); h = 32: p[j] += p[j+32] (j < 32)
        const float lo = __fadd_rn(part[m][lane], part[m][lane + 64]);
        const float hi = __fadd_rn(part[m][lane + 32], part[m][lane + 96]);
        v[m] = __fadd_rn(lo, hi);
      }
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
        for (int m = 0; m < 4; ++m) v[m] = __fadd_rn(v[m], __shfl_down_sync(0xffffffffu, v[m], off));
      if (lane == 0) {
        float* sb = s + t0;  // score index equals the token index (b*N + p*W + q)
        *reinterpret_cast<float2*>(sb) = make_float2(v[0], v[1]);
        *reinterpret_cast<float2*>(sb + W) = make_float2(v[2], v[3]);
      }
    }
    __syncthreads();
  }
}

// ============================================================== split =====

constexpr int SPLIT_THREADS = 1024;

// Exclusive scan of one int per thread over a 1024-thread block.
__device__ __forceinline__ int block_excl_scan(int v, int* warp_tot, int* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += n;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    int t = lane < static_cast<int>(blockDim.x >> 5) ? warp_tot[lane] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, t, off);
      if (lane >= off) t += n;
    }
    warp_tot[lane] = t;
  }
  __syncthreads();
  const int res = incl - v + (wid > 0 ? warp_tot[wid - 1] : 0);
  if (total) *total = warp_tot[(blockDim.x >> 5) - 1];
  __syncthreads();
  return res;
}

__device__ __forceinline__ int block_sum(int v, int* warp_tot) {
  int tot;
  block_excl_scan(v, warp_tot, &tot);
  return tot;
}

struct SelectShared {
  int hist[2][256];  // radix passes alternate between the two
  int warp_tot[32];
  int warp_tot3[3][32];
  int sel_digit;
  int sel_k;
  int sel_all;
  int rows[SPLIT_CLUSTER];  // packed rows of each image of the cluster
};

// Exclusive scans of three ints per thread at once (one pass of barriers).
__device__ __forceinline__ void block_excl_scan3(int& a, int& b, int& c, int (*wt)[32], int& ta, int& tb,
                                                 int& tc) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int v[3] = {a, b, c}, incl[3] = {a, b, c};
#pragma unroll
  for (int off = 1; off < 32; off <<= 1)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int n = __shfl_up_sync(0xffffffffu, incl[q], off);
      if (lane >= off) incl[q] += n;
    }
  if (lane == 31)
#pragma unroll
    for (int q = 0; q < 3; ++q) wt[q][wid] = incl[q];
  __syncthreads();
  if (wid < 3) {
    int t = lane < static_cast<int>(blockDim.x >> 5) ? wt[wid][lane] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, t, off);
      if (lane >= off) t += n;
    }
    wt[wid][lane] = t;
  }
  __syncthreads();
  a = incl[0] - v[0] + (wid > 0 ? wt[0][wid - 1] : 0);
  b = incl[1] - v[1] + (wid > 0 ? wt[1][wid - 1] : 0);
  c = incl[2] - v[2] + (wid > 0 ? wt[2][wid - 1] : 0);
  const int lw = (blockDim.x >> 5) - 1;
  ta = wt[0][lw];
  tb = wt[1][lw];
  tc = wt[2][lw];
  __syncthreads();
}

// MSB-first radix select over the candidates (bit i of cand: key[i] of this
// thread): the key of the k-th largest candidate of the block (1 <= k <=
// #candidates) and how many candidates with exactly that key belong to the top k
// (those with the lowest token ids). The passes alternate between two
// histograms, so clearing the next one needs no barrier of its own. A pass whose
// digit is taken whole ends the search: every candidate with the prefix so far
// ranks in the top k, so the prefix is the threshold, with all its equals.
template <int CH>
__device__ __forceinline__ void radix_select(const uint32_t (&key)[CH], uint32_t cand, int k, SelectShared& sh,
                                             uint32_t& thr, int& take) {
  uint32_t prefix = 0, pmask = 0;
  int kk = k;
  if (threadIdx.x < 256) sh.hist[0][threadIdx.x] = 0;
  __syncthreads();
  int h = 0;
#pragma unroll 1
  for (int shift = 24; shift >= 0; shift -= 8, h ^= 1) {
    int* hist = sh.hist[h];
#pragma unroll
    for (int i = 0; i < CH; ++i)
      if (((cand >> i) & 1u) && (key[i] & pmask) == prefix) atomicAdd(&hist[(key[i] >> shift) & 255u], 1);
    if (threadIdx.x >= blockDim.x - 256) sh.hist[h ^ 1][threadIdx.x - (blockDim.x - 256)] = 0;
    __syncthreads();
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      // lane L covers digits 255-8L .. 248-8L (descending)
      const int4 lo = *reinterpret_cast<const int4*>(hist + 248 - 8 * lane);
      const int4 hi = *reinterpret_cast<const int4*>(hist + 252 - 8 * lane);
      const int cnt[8] = {hi.w, hi.z, hi.y, hi.x, lo.w, lo.z, lo.y, lo.x};
      int lsum = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) lsum += cnt[j];
      int incl = lsum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += n;
      }
      const int excl = incl - lsum;
      if (excl < kk && kk <= incl) {
        int c = excl, dig = 0, left = 0, all = 0;
        bool found = false;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (!found && c + cnt[j] >= kk) {
            found = true;
            dig = 255 - 8 * lane - j;
            left = kk - c;
            all = left == cnt[j];
          }
          c += cnt[j];
        }
        sh.sel_digit = dig;
        sh.sel_k = left;
        sh.sel_all = all;
      }
    }
    __syncthreads();
    // sel_* are rewritten only after the next pass's barrier, which every
    // thread reaches after these reads
    prefix |= static_cast<uint32_t>(sh.sel_digit) << shift;
    pmask |= 255u << shift;
    kk = sh.sel_k;
    if (sh.sel_all) break;
  }
  thr = prefix;
  take = kk;
}

// Bits of this thread's top-k candidates under (key desc, index asc); thread t
// holds the tokens t CH .. t CH + CH - 1.
template <int CH>
__device__ __forceinline__ uint32_t topk_bits(const uint32_t (&key)[CH], uint32_t cand, int ncand, int k,
                                              SelectShared& sh) {
  if (k <= 0) return 0u;
  if (k >= ncand) return cand;
  uint32_t thr;
  int take;
  radix_select<CH>(key, cand, k, sh, thr, take);
  uint32_t gt = 0, eq = 0;
#pragma unroll
  for (int i = 0; i < CH; ++i) {
    gt |= (key[i] > thr ? 1u : 0u) << i;
    eq |= (key[i] == thr ? 1u : 0u) << i;
  }
  gt &= cand;
  eq &= cand;
  int rank = block_excl_scan(__popc(eq), sh.warp_tot, nullptr);
  // the equals of lowest index, as many as are left to take
  while (eq && rank < take) {
    gt |= eq & (0u - eq);
    eq &= eq - 1;
    ++rank;
  }
  return gt;
}

// Packed rows of one image from its labels (in shared memory): row_src and
// the token -> row map, kept tokens first (raster order), then 2x2 windows,
// then 4x4 windows (window-raster order). `base` is the image's first packed
// row. Called by all threads of the CTA.
__device__ void compact_image(const uint8_t* lab, int b, int H, int W, int levels, int lf, int base, int nk,
                              int n2, int32_t* row_src, int32_t* tok_row, int* warp_tot) {
  const int N = H * W;
  int32_t* trow = tok_row + static_cast<long long>(b) * N;
  // kept tokens in raster order
  {
    const int chunk = (N + blockDim.x - 1) / blockDim.x;
    const int i0 = threadIdx.x * chunk, i1 = min(N, i0 + chunk);
    int c = 0;
    for (int i = i0; i < i1; ++i) c += lab[i] == HILO_LABEL_KEEP ? 1 : 0;
    int r = base + block_excl_scan(c, warp_tot, nullptr);
    for (int i = i0; i < i1; ++i)
      if (lab[i] == HILO_LABEL_KEEP) {
        row_src[r] = i;
        trow[i] = r;
        ++r;
      }
  }
  // low-frequency mode: every lf x lf window of the grid, in window-raster
  // order; its non-kept members read it back
  if (lf) {
    const int Wl = W / lf, nw = (H / lf) * Wl;
    for (int w = threadIdx.x; w < nw; w += blockDim.x) {
      const int r = base + nk + w;
      row_src[r] = w;
      const int t0 = (lf * (w / Wl)) * W + lf * (w % Wl);
      for (int i = 0; i < lf; ++i)
        for (int j = 0; j < lf; ++j)
          if (lab[t0 + i * W + j] != HILO_LABEL_KEEP) trow[t0 + i * W + j] = r;
    }
    return;
  }
  // 2x2 windows in window-raster order
  {
    const int W2 = W >> 1, nw = (H >> 1) * W2;
    const int chunk = (nw + blockDim.x - 1) / blockDim.x;
    const int w0 = threadIdx.x * chunk, w1 = min(nw, w0 + chunk);
    int c = 0;
    for (int w = w0; w < w1; ++w) {
      const int t = (2 * (w / W2)) * W + 2 * (w % W2);
      c += (lab[t] == HILO_LABEL_POOL2 || lab[t + 1] == HILO_LABEL_POOL2 ||
            lab[t + W] == HILO_LABEL_POOL2 || lab[t + W + 1] == HILO_LABEL_POOL2)
               ? 1
               : 0;
    }
    int r = base + nk + block_excl_scan(c, warp_tot, nullptr);
    for (int w = w0; w < w1; ++w) {
      const int t = (2 * (w / W2)) * W + 2 * (w % W2);
      const int mem[4] = {t, t + 1, t + W, t + W + 1};
      bool any = false;
#pragma unroll
      for (int j = 0; j < 4; ++j) any |= lab[mem[j]] == HILO_LABEL_POOL2;
      if (!any) continue;
      row_src[r] = w;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (lab[mem[j]] == HILO_LABEL_POOL2) trow[mem[j]] = r;
      ++r;
    }
  }
  if (levels == 2) {
    const int W4 = W >> 2, nw = (H >> 2) * W4;
    const int chunk = (nw + blockDim.x - 1) / blockDim.x;
    const int w0 = threadIdx.x * chunk, w1 = min(nw, w0 + chunk);
    int c = 0;
    for (int w = w0; w < w1; ++w) {
      const int t = (4 * (w / W4)) * W + 4 * (w % W4);
      bool any = false;
      for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) any |= lab[t + i * W + j] == HILO_LABEL_POOL4;
      c += any ? 1 : 0;
    }
    int r = base + nk + n2 + block_excl_scan(c, warp_tot, nullptr);
    for (int w = w0; w < w1; ++w) {
      const int t = (4 * (w / W4)) * W + 4 * (w % W4);
      bool any = false;
      for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) any |= lab[t + i * W + j] == HILO_LABEL_POOL4;
      if (!any) continue;
      row_src[r] = w;
      for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j)
          if (lab[t + i * W + j] == HILO_LABEL_POOL4) trow[t + i * W + j] = r;
      ++r;
    }
  }
}

// Labels and per-image counts. One CTA per image; thread t owns the tokens
// t CH .. t CH + CH - 1, whose scores stay in its registers (CH is the smallest of
// 4, 8, 16, 32 for which 1024 threads cover the image, and no more threads are
// launched than own tokens, but at least 256). With fused != 0 the same CTA also
// writes cu_img and the packed rows: with 1 the image is the only one and its rows
// begin at 0; above that it is the size of the one cluster that all images' CTAs
// form, in which each CTA tells the others its row count. (Three images of 46x30 took
// 7.2 us with a second kernel for the rows, 5.1 so; four of 64x64 10.0 and 7.4.)
// granular != 0 is the window-granular split: every pooling window
// takes the finest class of its members (an aligned 2x2 window with a kept member
// is kept whole; with two levels an aligned 4x4 block is pooled 4x4 only when all
// its members rank below the k_mid cut, else its non-kept members are pooled 2x2).
// Bound by one SM's latency: barriers, shared atomics and dependent loads. (With
// the keys in shared memory and re-read by each pass, in contiguous chunks per
// thread with up to 16-way bank conflicts, random scores, a quarter kept: 64x64 9.0 us,
// 6.8 so, 128x128 36.7 and 21.6, with two levels 55.0 and 26.9, of four score values
// 56.3 and 31.6.)
template <int CH, bool GRANULAR, bool LFMODE>
__global__ void __launch_bounds__(SPLIT_THREADS) split_select_kernel(
    const float* __restrict__ score, const uint8_t* __restrict__ mask,
    const int32_t* __restrict__ k_keep, const int32_t* __restrict__ k_mid, uint8_t* labels_out,
    int32_t* counts, int B, int H, int W, int levels, int lf_arg, int fused, int32_t* cu_img,
    int32_t* row_src, int32_t* tok_row) {
  // the modes are template parameters, so the plain split carries none of
  // their code (this CTA has up to 1024 threads and at most 64 registers each)
  constexpr bool granular = GRANULAR;
  const int lf = LFMODE ? lf_arg : 0;
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) SelectShared sh;
  const int N = H * W;
  const int b = blockIdx.x;
  if (fused > 1) {
    cluster_arrive_relaxed();
    if (b >= B) {  // the cluster is a power of two
      cluster_wait();
      cluster_sync();
      return;
    }
  }
  uint8_t* lab = smem_raw;  // the labels, N bytes
  const long long base = static_cast<long long>(b) * N;
  const int k = min(max(k_keep[b], 0), N);
  const int km = levels == 2 ? min(max(k_mid[b], 0), N) : 0;
  const int i0 = static_cast<int>(threadIdx.x) * CH;
  // N is a multiple of 4 (H and W are even), so four tokens at a time are all
  // inside or all outside the image; wide loads only where the arrays allow them
  const bool wide = ((reinterpret_cast<uintptr_t>(score + base) & 15) == 0) &&
                    ((reinterpret_cast<uintptr_t>(mask + base) & 3) == 0);
  uint32_t key[CH];
  uint32_t keep = 0, every = 0;  // bit i: token i0 + i is masked (then: kept) / exists
#pragma unroll
  for (int q = 0; q < CH / 4; ++q) {
    const int i = i0 + 4 * q;
    uint32_t m = 0;
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < N) {
      every |= 15u << (4 * q);
      if (wide) {
        f = __ldg(reinterpret_cast<const float4*>(score + base + i));
        m = __ldg(reinterpret_cast<const uint32_t*>(mask + base + i));
      } else {
        f = make_float4(score[base + i], score[base + i + 1], score[base + i + 2], score[base + i + 3]);
#pragma unroll
        for (int j = 0; j < 4; ++j) m |= static_cast<uint32_t>(mask[base + i + j]) << (8 * j);
      }
    }
    // scores are >= +0, so their IEEE bit patterns order like the values
    key[4 * q] = __float_as_uint(f.x);
    key[4 * q + 1] = __float_as_uint(f.y);
    key[4 * q + 2] = __float_as_uint(f.z);
    key[4 * q + 3] = __float_as_uint(f.w);
#pragma unroll
    for (int j = 0; j < 4; ++j) keep |= ((m >> (8 * j)) & 255u ? 1u : 0u) << (4 * q + j);
  }
  keep |= topk_bits<CH>(key, every, N, k, sh);
  // labels of this thread's tokens: a byte each, low = the tokens of `coarse`
  auto put_labels = [&](uint32_t kept, uint32_t coarse) {
#pragma unroll
    for (int q = 0; q < CH / 4; ++q) {
      uint32_t v = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = 4 * q + j;
        const uint32_t l = (kept >> i) & 1u ? HILO_LABEL_KEEP
                                            : (lf ? HILO_LABEL_LF
                                                  : ((coarse >> i) & 1u ? HILO_LABEL_POOL4 : HILO_LABEL_POOL2));
        v |= l << (8 * j);
      }
      if (i0 + 4 * q < N) *reinterpret_cast<uint32_t*>(lab + i0 + 4 * q) = v;
    }
  };
  if (granular) {
    // one thread per 2x2 window: a window with a kept member is kept whole
    put_labels(keep, 0u);
    __syncthreads();
    const int W2 = W >> 1, nw = (H >> 1) * W2;
    for (int w = threadIdx.x; w < nw; w += blockDim.x) {
      const int t = (2 * (w / W2)) * W + 2 * (w % W2);
      uint16_t* l0 = reinterpret_cast<uint16_t*>(lab + t);
      uint16_t* l1 = reinterpret_cast<uint16_t*>(lab + t + W);
      // labels are 0 (kept) or 1 here, so a window is all pooled or has a kept member
      if ((*l0 & *l1) != 0x0101u) *l0 = *l1 = 0;
    }
    __syncthreads();
    keep = 0;
#pragma unroll
    for (int i = 0; i < CH; ++i)
      if (i0 + i < N && lab[i0 + i] == HILO_LABEL_KEEP) keep |= 1u << i;
  }
  uint32_t coarse = 0;
  if (levels == 2) {
    const uint32_t cand = every & ~keep;
    const int ncand = block_sum(__popc(cand), sh.warp_tot);
    coarse = cand & ~topk_bits<CH>(key, cand, ncand, km, sh);
  }
  if (!granular || levels == 2) put_labels(keep, coarse);
  __syncthreads();
  if (granular && levels == 2) {
    // one thread per 4x4 block: pooled 4x4 only when every member is
    const int W4 = W >> 2, nb = (H >> 2) * W4;
    for (int v = threadIdx.x; v < nb; v += blockDim.x) {
      const int t = (4 * (v / W4)) * W + 4 * (v % W4);
      bool all4 = true;
#pragma unroll
      for (int i = 0; i < 4; ++i) all4 &= *reinterpret_cast<const uint32_t*>(lab + t + i * W) == 0x02020202u;
      if (all4) continue;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (lab[t + i * W + j] == HILO_LABEL_POOL4) lab[t + i * W + j] = HILO_LABEL_POOL2;
    }
    __syncthreads();
  }
  // labels out
  const bool wide_out = (reinterpret_cast<uintptr_t>(labels_out + base) & 3) == 0;
#pragma unroll
  for (int q = 0; q < CH / 4; ++q) {
    const int i = i0 + 4 * q;
    if (i >= N) continue;
    const uint32_t v = *reinterpret_cast<const uint32_t*>(lab + i);
    if (wide_out) {
      *reinterpret_cast<uint32_t*>(labels_out + base + i) = v;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) labels_out[base + i + j] = static_cast<uint8_t>(v >> (8 * j));
    }
  }
  // Per thread, its tokens and a contiguous chunk of 2x2 windows and of 4x4
  // windows: kept tokens, and windows holding at least one member of their
  // class, are counted, and one three-way block scan gives both the image's
  // counts and each thread's first packed row.
  // (low-frequency mode: the "2x2 windows" below are the lf x lf windows,
  // every one of which has a row)
  const int W2 = lf ? W / lf : W >> 1, nw2 = (lf ? H / lf : H >> 1) * W2;
  const int wch = (nw2 + blockDim.x - 1) / blockDim.x;  // at most 32
  const int w0 = min(nw2, static_cast<int>(threadIdx.x) * wch), w1 = min(nw2, w0 + wch);
  const int W4 = W >> 2, nw4 = levels == 2 ? (H >> 2) * W4 : 0;
  const int vch = (nw4 + blockDim.x - 1) / blockDim.x;
  const int v0 = min(nw4, static_cast<int>(threadIdx.x) * vch), v1 = min(nw4, v0 + vch);
  // bit j of a label pair / quad: the member has the class
  auto any2 = [&](int t) {  // a 2x2 window's POOL2 members, bits 0..3 in raster order
    const uint32_t a = *reinterpret_cast<const uint16_t*>(lab + t), c = *reinterpret_cast<const uint16_t*>(lab + t + W);
    return ((a & 255u) == HILO_LABEL_POOL2 ? 1u : 0u) | ((a >> 8) == HILO_LABEL_POOL2 ? 2u : 0u) |
           ((c & 255u) == HILO_LABEL_POOL2 ? 4u : 0u) | ((c >> 8) == HILO_LABEL_POOL2 ? 8u : 0u);
  };
  auto any4 = [&](int t) {  // any POOL4 member (label 2: bit 1 of a byte, and not 3 in this mode)
    uint32_t o = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) o |= *reinterpret_cast<const uint32_t*>(lab + t + i * W);
    return (o & 0x02020202u) != 0;
  };
  int rk = __popc(keep), r2 = 0, r4 = 0;
  uint32_t has2 = 0, has4 = 0;
  if (lf) {
    r2 = w1 - w0;
  } else {
    int row = w0 / W2, col = w0 - row * W2;
    for (int w = w0; w < w1; ++w) {
      if (any2(2 * row * W + 2 * col)) has2 |= 1u << (w - w0);
      if (++col == W2) col = 0, ++row;
    }
    r2 = __popc(has2);
  }
  for (int v = v0; v < v1; ++v)
    if (any4((4 * (v / W4)) * W + 4 * (v % W4))) has4 |= 1u << (v - v0);
  r4 = __popc(has4);
  int nk, n2, n4;
  block_excl_scan3(rk, r2, r4, sh.warp_tot3, nk, n2, n4);
  // the image's first packed row
  int row0 = 0;
  if (fused > 1) {
    cluster_wait();  // every CTA has begun: its shared memory may be written
    if (static_cast<int>(threadIdx.x) < fused)
      st_shared_cluster(mapa_shared(smem_u32(&sh.rows[b]), threadIdx.x), nk + n2 + n4);
    __syncwarp();
    cluster_sync();
    for (int j = 0; j < b; ++j) row0 += sh.rows[j];
    rk += row0, r2 += row0, r4 += row0;
  }
  if (threadIdx.x == 0) {
    counts[3 * b + 0] = nk;
    counts[3 * b + 1] = n2;
    counts[3 * b + 2] = n4;
    if (fused) {
      if (b == 0) cu_img[0] = 0;
      cu_img[b + 1] = row0 + nk + n2 + n4;
    }
  }
  if (!fused) return;
  // packed rows: kept tokens (raster order), then 2x2, then 4x4 windows
  int32_t* trow = tok_row + base;
  for (uint32_t m = keep; m; m &= m - 1) {
    const int i = i0 + __ffs(m) - 1;
    row_src[rk] = i;
    trow[i] = rk;
    ++rk;
  }
  r2 += nk;
  if (lf) {
    for (int w = w0; w < w1; ++w, ++r2) {
      row_src[r2] = w;
      const int t0 = (lf * (w / W2)) * W + lf * (w % W2);
      for (int i = 0; i < lf; ++i)
        for (int j = 0; j < lf; ++j)
          if (lab[t0 + i * W + j] != HILO_LABEL_KEEP) trow[t0 + i * W + j] = r2;
    }
  } else {
    for (uint32_t m = has2; m; m &= m - 1) {
      const int w = w0 + __ffs(m) - 1;
      const int t = (2 * (w / W2)) * W + 2 * (w % W2);
      const uint32_t mem = any2(t);
      row_src[r2] = w;
      if (mem & 1u) trow[t] = r2;
      if (mem & 2u) trow[t + 1] = r2;
      if (mem & 4u) trow[t + W] = r2;
      if (mem & 8u) trow[t + W + 1] = r2;
      ++r2;
    }
  }
  r4 += nk + n2;
  for (uint32_t m = has4; m; m &= m - 1) {
    const int v = v0 + __ffs(m) - 1;
    const int t = (4 * (v / W4)) * W + 4 * (v % W4);
    row_src[r4] = v;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (lab[t + i * W + j] == HILO_LABEL_POOL4) trow[t + i * W + j] = r4;
    ++r4;
  }
}

// Packed offsets, row sources and token -> row map. One CTA per image.
__global__ void __launch_bounds__(SPLIT_THREADS) split_compact_kernel(
    const uint8_t* __restrict__ labels, const int32_t* __restrict__ counts, int32_t* cu_img,
    int32_t* row_src, int32_t* tok_row, int H, int W, int levels, int lf) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int warp_tot[32];
  const int N = H * W;
  const int b = blockIdx.x;
  uint8_t* lab = smem_raw;
  const uint8_t* src = labels + static_cast<long long>(b) * N;
  if ((reinterpret_cast<uintptr_t>(src) & 3) == 0) {  // N is a multiple of 4
    for (int i = threadIdx.x; i < N / 4; i += blockDim.x)
      reinterpret_cast<uint32_t*>(lab)[i] = __ldg(reinterpret_cast<const uint32_t*>(src) + i);
  } else {
    for (int i = threadIdx.x; i < N; i += blockDim.x) lab[i] = src[i];
  }
  int base = 0;
  for (int j = 0; j < b; ++j) base += counts[3 * j] + counts[3 * j + 1] + counts[3 * j + 2];
  const int nk = counts[3 * b], n2 = counts[3 * b + 1], n4 = counts[3 * b + 2];
  if (threadIdx.x == 0) {
    if (b == 0) cu_img[0] = 0;
    cu_img[b + 1] = base + nk + n2 + n4;
  }
  __syncthreads();
  compact_image(lab, b, H, W, levels, lf, base, nk, n2, row_src, tok_row, warp_tot);
}

// =============================================================== pack =====
//
// One to four warps per packed image row, each owning every first to fourth
// 8-channel chunk of its lanes, so a row needs one memory round trip. A kept row is a
// 16-byte-vector copy; a pooled row sums the window's members of its class
// in raster order (the first member initialises the sum), divides once with
// correct rounding and rounds to bf16 (nearest even). Bound by each row's chain of
// dependent reads (offsets, counts, row source, labels, data), so by the rows in
// flight: from 513 channels on a CTA per row (two rows per CTA, at 3072 channels and a
// quarter kept: 128x128 with two levels 31.2 us, 27.3 so; four images of 64x64 32.4 and
// 28.7).

constexpr int PACK_WARPS = 4;
constexpr int PACK_THREADS = 32 * PACK_WARPS;
constexpr int PACK_THREADS_SHORT = 256;  // rows of up to 512 channels, several to a CTA

// Warps per row (or slice of a window row): as many as have a chunk of eight channels per
// lane. (A CTA of four warps per row at every width, of 128 channels a quarter kept and
// the rest pooled 2x2: 64x64 tokens 3.7 us, 2.8 so, 128x128 9.1 and 4.0; low-frequency
// rows of 2x2 windows, none kept, 64x64 4.3 and 2.4, of 512 channels 4.3 and 2.8.)
static int pack_warps(int d) { return d <= 256 ? 1 : d <= 512 ? 2 : 4; }

// CTAs per low-frequency row: a slice of 128 chunks of eight channels each, but the
// rows of 2x2 windows, of which there are many, whole (a quarter kept: 128x128 of 3072
// channels 24.9 us whole and 34.1 in slices, of 1152 9.3 and 15.5, 64x64 of 2048 5.3 and
// 7.1; 4x4 windows of 3072 27.6 and 23.5, 8x8 62.7 and 23.8).
__host__ __device__ constexpr int lf_slices(int lf, int d) {
  return lf == 2 ? 1 : (d / 8 + PACK_THREADS - 1) / PACK_THREADS;
}

// (volatile: a batch's loads stay together)
__device__ __forceinline__ uint4 ldg16(const uint4* p) {
  uint4 r;
  asm volatile("ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

// Eight channels (c) of a low-frequency row: the mean of all LF x LF members of the
// window whose first member is w0 (raster order, the first initialising the sum), one
// correctly rounded division.
template <int LF>
__device__ __forceinline__ void pack_lf_chunk(const __nv_bfloat16* __restrict__ w0, int W, int d, int c,
                                              uint4* __restrict__ dst) {
  constexpr int NM = LF * LF, LOADS = NM < 16 ? NM : 16;
  const float cnt = static_cast<float>(NM);
  float acc[8];
#pragma unroll 1
  for (int g = 0; g < NM; g += LOADS) {
    uint4 v[LOADS];
#pragma unroll
    for (int q = 0; q < LOADS; ++q) {
      const int m = g + q;
      v[q] = ldg16(reinterpret_cast<const uint4*>(w0 + static_cast<long long>((m / LF) * W + (m % LF)) * d) + c);
    }
#pragma unroll
    for (int q = 0; q < LOADS; ++q) {
      float f[8];
      bf16x8_to_f32(v[q], f);
#pragma unroll
      for (int u = 0; u < 8; ++u) acc[u] = (g == 0 && q == 0) ? f[u] : __fadd_rn(acc[u], f[u]);
    }
  }
  uint4 o;
  o.x = pack_bf16x2(__fdiv_rn(acc[0], cnt), __fdiv_rn(acc[1], cnt));
  o.y = pack_bf16x2(__fdiv_rn(acc[2], cnt), __fdiv_rn(acc[3], cnt));
  o.z = pack_bf16x2(__fdiv_rn(acc[4], cnt), __fdiv_rn(acc[5], cnt));
  o.w = pack_bf16x2(__fdiv_rn(acc[6], cnt), __fdiv_rn(acc[7], cnt));
  dst[c] = o;
}

// CHUNKS: chunks of a kept row that a lane has in flight, no more than it has (three at
// every width: 16 images of 32x32 tokens of 4096 channels, all kept, 45.8 us, 42.1 with
// four; 128x128 of 1024 10.7, 9.9 with one; 3072 channels with four 39.2, 34.6 with three)
template <int WPR, int THREADS, int CHUNKS>
__global__ void __launch_bounds__(THREADS) pack_kernel(const __nv_bfloat16* __restrict__ x,
                                                   const uint8_t* __restrict__ labels,
                                                   const int32_t* __restrict__ row_src,
                                                   const int32_t* __restrict__ counts,
                                                   const int32_t* __restrict__ cu_img,
                                                   __nv_bfloat16* __restrict__ packed, int B,
                                                   int H, int W, int d, int cap) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int N = H * W;
  const int G = d >> 3;
  const int total = min(cu_img[B], cap);
  const long long nwarps = static_cast<long long>(gridDim.x) * (blockDim.x >> 5);
  for (long long gw = static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
       gw < static_cast<long long>(total) * WPR; gw += nwarps) {
    // from the last row down: an image's pooled rows, 4x4 last, take the longest
    // (5% less at 128x128 with two levels of 3072 channels, 9% at 64x64)
    const int r = total - 1 - static_cast<int>(gw / WPR);
    const int c0 = lane + 32 * static_cast<int>(gw % WPR);
    constexpr int CSTEP = 32 * WPR;
    int b = 0;
    while (b + 1 < B && cu_img[b + 1] <= r) ++b;
    const int local = r - cu_img[b];
    const int nk = counts[3 * b], n2 = counts[3 * b + 1];
    const int src = row_src[r];
    const __nv_bfloat16* xb = x + static_cast<long long>(b) * N * d;
    uint4* dst = reinterpret_cast<uint4*>(packed + static_cast<long long>(r) * d);
    const int size = local < nk ? 1 : local < nk + n2 ? 2 : 4;
    // the row source: a token of the image, or a window of its size
    if (!HILO_DCHECK(local >= 0 && src >= 0 && src < (H / size) * (W / size), DCHECK_PACK_SRC)) continue;
    if (local < nk) {
      const uint4* sp = reinterpret_cast<const uint4*>(xb + static_cast<long long>(src) * d);
#pragma unroll(CHUNKS)
      for (int c = c0; c < G; c += CSTEP) dst[c] = __ldg(sp + c);
      continue;
    }
    const uint8_t cls = size == 2 ? HILO_LABEL_POOL2 : HILO_LABEL_POOL4;
    const int Wn = W / size;
    const int t0 = (size * (src / Wn)) * W + size * (src % Wn);
    // member m = i*size + j  <->  token t0 + i*W + j (raster order within the window)
    bool is_member = false;
    if (lane < size * size) {
      const int t = t0 + (lane / size) * W + (lane % size);
      is_member = labels[static_cast<long long>(b) * N + t] == cls;
    }
    const uint32_t mm = __ballot_sync(0xffffffffu, is_member);
    const float cnt = static_cast<float>(__popc(mm));
    const int ngroups = size * size / 4;
#pragma unroll 3
    for (int c = c0; c < G; c += CSTEP) {
      float acc[8];
      bool first = true;
      for (int gi = 0; gi < ngroups; ++gi) {
        uint4 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int m = 4 * gi + q;
          if (mm & (1u << m)) {
            const int t = t0 + (m / size) * W + (m % size);
            v[q] = __ldg(reinterpret_cast<const uint4*>(xb + static_cast<long long>(t) * d) + c);
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int m = 4 * gi + q;
          if (!(mm & (1u << m))) continue;
          float f[8];
          bf16x8_to_f32(v[q], f);
          if (first) {
#pragma unroll
            for (int u = 0; u < 8; ++u) acc[u] = f[u];
            first = false;
          } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) acc[u] = __fadd_rn(acc[u], f[u]);
          }
        }
      }
      uint4 o;
      o.x = pack_bf16x2(__fdiv_rn(acc[0], cnt), __fdiv_rn(acc[1], cnt));
      o.y = pack_bf16x2(__fdiv_rn(acc[2], cnt), __fdiv_rn(acc[3], cnt));
      o.z = pack_bf16x2(__fdiv_rn(acc[4], cnt), __fdiv_rn(acc[5], cnt));
      o.w = pack_bf16x2(__fdiv_rn(acc[6], cnt), __fdiv_rn(acc[7], cnt));
      dst[c] = o;
    }
  }
}

// Low-frequency mode: per image, the kept rows (copies) and then one row per
// LF x LF window of the grid (the mean of all its members). Rows of 2x2 windows are many
// and short: all rows in one go, from the last down. Larger windows first, in slices of
// 128 chunks of eight channels, with 16 of a lane's loads in flight; then the kept rows.
// Bound by the chain of a window's loads and sums. (With four loads in flight and a
// lane's chunks one after another, 64x64 tokens of 3072 channels took 17.2 us for 4x4
// windows, 7.5 so, and 51 for 8x8, 12.3. The 2x2 windows first, too: 4x 64x64 tokens of
// 1152 channels 11.1 us, 10.1 so. 4x4 windows not first: 128x128 of 512, none kept, 5.4
// and 4.2.)
template <int LF, int WPR, int THREADS>
__global__ void __launch_bounds__(THREADS) pack_lf_kernel(const __nv_bfloat16* __restrict__ x,
                                                               const int32_t* __restrict__ row_src,
                                                               const int32_t* __restrict__ counts,
                                                               const int32_t* __restrict__ cu_img,
                                                               __nv_bfloat16* __restrict__ packed, int B, int H,
                                                               int W, int d, int cap) {
  pdl_wait();
  pdl_trigger();
  const int N = H * W;
  const int G = d >> 3;
  const int total = min(cu_img[B], cap);
  const int slices = lf_slices(LF, d);
  const int nw = (H / LF) * (W / LF);  // window rows of an image
  const long long nwin = LF > 2 ? static_cast<long long>(B) * nw * slices : 0;
  constexpr int STEP = 32 * WPR, ROWS = THREADS / STEP;  // rows per CTA and turn, chunks of a row per turn
  for (long long i = static_cast<long long>(blockIdx.x) * ROWS + threadIdx.x / STEP; i < nwin + total;
       i += static_cast<long long>(gridDim.x) * ROWS) {
    int b = 0, r;
    int c = threadIdx.x % STEP;
    bool window = i < nwin;
    if (window) {
      const int w = static_cast<int>(i / slices);
      c += static_cast<int>(i - static_cast<long long>(w) * slices) * STEP;
      b = w / nw;
      r = cu_img[b] + counts[3 * b] + (w - b * nw);
      if (r >= total) continue;
    } else {
      r = static_cast<int>(nwin + total - 1 - i);
      while (b + 1 < B && cu_img[b + 1] <= r) ++b;
      window = r - cu_img[b] >= counts[3 * b];
      if (LF > 2 && window) continue;
    }
    const int src = row_src[r];
    const __nv_bfloat16* xb = x + static_cast<long long>(b) * N * d;
    uint4* dst = reinterpret_cast<uint4*>(packed + static_cast<long long>(r) * d);
    const int size = window ? LF : 1;
    if (!HILO_DCHECK(r >= cu_img[b] && src >= 0 && src < (H / size) * (W / size), DCHECK_PACK_LF_SRC)) continue;
    if (window) {
      const int t0 = (LF * (src / (W / LF))) * W + LF * (src % (W / LF));
      const __nv_bfloat16* w0 = xb + static_cast<long long>(t0) * d;
      if constexpr (LF == 2) {  // not in slices
        for (; c < G; c += STEP) pack_lf_chunk<LF>(w0, W, d, c, dst);
      } else {
        if (c < G) pack_lf_chunk<LF>(w0, W, d, c, dst);
      }
    } else {
      const uint4* sp = reinterpret_cast<const uint4*>(xb + static_cast<long long>(src) * d);
#pragma unroll 3
      for (; c < G; c += STEP) dst[c] = __ldg(sp + c);
    }
  }
}

// Number of grid tokens each packed image row stands for: 1 for a kept
// token, the count of its class members for a pooled window (the weights of
// proportional attention). One thread per row of the capacity.
__global__ void __launch_bounds__(256) row_sizes_kernel(const uint8_t* __restrict__ labels,
                                                        const int32_t* __restrict__ row_src,
                                                        const int32_t* __restrict__ counts,
                                                        const int32_t* __restrict__ cu_img,
                                                        float* __restrict__ n_img, int B, int H, int W,
                                                        int cap, int lf) {
  pdl_wait();
  pdl_trigger();
  const int N = H * W;
  const int total = min(cu_img[B], cap);
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < total; r += gridDim.x * blockDim.x) {
    int b = 0;
    while (b + 1 < B && cu_img[b + 1] <= r) ++b;
    const int local = r - cu_img[b];
    const int nk = counts[3 * b], n2 = counts[3 * b + 1];
    if (local < nk) {
      n_img[r] = 1.0f;
      continue;
    }
    const int size = lf ? lf : (local < nk + n2 ? 2 : 4);
    const uint8_t cls = lf ? HILO_LABEL_LF : (size == 2 ? HILO_LABEL_POOL2 : HILO_LABEL_POOL4);
    const int src = row_src[r];
    const int Wn = W / size;
    if (!HILO_DCHECK(local >= 0 && src >= 0 && src < (H / size) * Wn, DCHECK_ROW_SIZES_SRC)) continue;
    const uint8_t* lab = labels + static_cast<long long>(b) * N + (size * (src / Wn)) * W + size * (src % Wn);
    int c = 0;
    for (int i = 0; i < size; ++i)
      for (int j = 0; j < size; ++j) c += lab[i * W + j] == cls ? 1 : 0;
    n_img[r] = static_cast<float>(c);
  }
}

// ============================================================= unpack =====
//
// One warp per token, bound by HBM. Where the fp32 arrays begin on 32 bytes (WIDE) a
// lane moves eight channels at a time, 32 bytes of fp32 in one access, and issues all
// loads of a batch of two or four such pieces before the first store; else 16 bytes
// at a time as the compiler unrolls it, which is the better order for those.
// (128x128 tokens of 3072 channels: nearest 45.3 us wide and 47.5 narrow, delta 59.9
// and 67.2, whose 16-byte stores each write half of every 32-byte sector; 64x64: 14.5
// and 15.6, 17.9 and 19.0. Batches of 16-byte accesses took 57.7 and 64.2 us at
// 128x128 and 20.5 for delta at 64x64.)

struct F8 {
  float v[8];
};

// (volatile: the loads of a batch stay ahead of its stores)
__device__ __forceinline__ F8 ldg8(const float* p) {
  F8 r;
  asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]), "=f"(r.v[4]), "=f"(r.v[5]), "=f"(r.v[6]),
                 "=f"(r.v[7])
               : "l"(p));
  return r;
}

__device__ __forceinline__ void stcs8(float* p, const F8& r) {
  asm volatile("st.global.cs.v8.f32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"f"(r.v[0]), "f"(r.v[1]), "f"(r.v[2]),
               "f"(r.v[3]), "f"(r.v[4]), "f"(r.v[5]), "f"(r.v[6]), "f"(r.v[7]), "l"(p)
               : "memory");
}

// One row of d channels; U pieces per lane in flight.
template <bool WIDE, int U>
__device__ __forceinline__ void copy_row(const float* __restrict__ s, float* __restrict__ o, int d, int lane) {
  if constexpr (!WIDE) {
#pragma unroll(2 * U)
    for (int c = lane; c < (d >> 2); c += 32)
      __stcs(reinterpret_cast<float4*>(o) + c, __ldg(reinterpret_cast<const float4*>(s) + c));
  } else {
    for (int c = lane; c < (d >> 3); c += 32 * U) {
      F8 v[U];
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (c + 32 * k < (d >> 3)) v[k] = ldg8(s + 8 * (c + 32 * k));
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (c + 32 * k < (d >> 3)) stcs8(o + 8 * (c + 32 * k), v[k]);
    }
  }
}

template <bool WIDE, int U>
__global__ void __launch_bounds__(256) unpack_kernel(const float* __restrict__ out_img,
                                                     const int32_t* __restrict__ tok_row,
                                                     float* __restrict__ y, long long ntok,
                                                     int d, long long rows_max) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const long long wstep = static_cast<long long>(gridDim.x) * (blockDim.x >> 5);
  for (long long t = static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
       t < ntok; t += wstep) {
    const int r = __ldg(tok_row + t);
    if (!HILO_DCHECK(r >= 0 && r < rows_max, DCHECK_UNPACK_ROW)) continue;
    copy_row<WIDE, U>(out_img + static_cast<long long>(r) * d, y + t * d, d, lane);
  }
}

// Delta unpool: a kept token copies its output row; a pooled member keeps
// its own value plus its window's update, y = x + (out - packed), one fp32
// subtract then one fp32 add (x and packed widened from bf16). Four CTAs per SM:
// small grids need the warps (46x30 tokens of 1152 channels, batch of three: 9.2 us
// with 94 registers and three pieces in flight).
template <bool WIDE, int U>
__global__ void __launch_bounds__(256, WIDE && U > 1 ? 4 : 0) unpack_delta_kernel(const float* __restrict__ out_img,
                                                              const __nv_bfloat16* __restrict__ packed,
                                                              const __nv_bfloat16* __restrict__ x,
                                                              const uint8_t* __restrict__ labels,
                                                              const int32_t* __restrict__ tok_row,
                                                              float* __restrict__ y, long long ntok, int d,
                                                              long long rows_max) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int G = d >> 3;
  const long long wstep = static_cast<long long>(gridDim.x) * (blockDim.x >> 5);
  for (long long t = static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
       t < ntok; t += wstep) {
    const int r = __ldg(tok_row + t);
    if (!HILO_DCHECK(r >= 0 && r < rows_max, DCHECK_UNPACK_DELTA_ROW)) continue;
    const float* s = out_img + static_cast<long long>(r) * d;
    float* o = y + t * d;
    if (__ldg(labels + t) == HILO_LABEL_KEEP) {
      copy_row<WIDE, U>(s, o, d, lane);
      continue;
    }
    const uint4* xr = reinterpret_cast<const uint4*>(x + t * d);
    const uint4* pr = reinterpret_cast<const uint4*>(packed + static_cast<long long>(r) * d);
    if constexpr (!WIDE) {
      for (int c = lane; c < G; c += 32) {
        float xf[8], pf[8];
        bf16x8_to_f32(__ldg(xr + c), xf);
        bf16x8_to_f32(__ldg(pr + c), pf);
        const float4 o0 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c);
        const float4 o1 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c + 1);
        const float ov[8] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y, o1.z, o1.w};
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __fadd_rn(xf[u], __fsub_rn(ov[u], pf[u]));
        __stcs(reinterpret_cast<float4*>(o) + 2 * c, make_float4(v[0], v[1], v[2], v[3]));
        __stcs(reinterpret_cast<float4*>(o) + 2 * c + 1, make_float4(v[4], v[5], v[6], v[7]));
      }
    } else {
      for (int c = lane; c < G; c += 32 * U) {
        uint4 xv[U], pv[U];
        F8 v[U];
#pragma unroll
        for (int k = 0; k < U; ++k)
          if (c + 32 * k < G) {
            xv[k] = __ldg(xr + c + 32 * k);
            pv[k] = __ldg(pr + c + 32 * k);
            v[k] = ldg8(s + 8 * (c + 32 * k));
          }
#pragma unroll
        for (int k = 0; k < U; ++k)
          if (c + 32 * k < G) {
            float xf[8], pf[8];
            bf16x8_to_f32(xv[k], xf);
            bf16x8_to_f32(pv[k], pf);
#pragma unroll
            for (int u = 0; u < 8; ++u) v[k].v[u] = __fadd_rn(xf[u], __fsub_rn(v[k].v[u], pf[u]));
            stcs8(o + 8 * (c + 32 * k), v[k]);
          }
      }
    }
  }
}

template <bool WIDE, int U>
__global__ void __launch_bounds__(256) unpack_update_kernel(const float* __restrict__ out_img,
                                                            const int32_t* __restrict__ tok_row,
                                                            __nv_bfloat16* __restrict__ x,
                                                            long long ntok, int d, float alpha,
                                                            long long rows_max) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int G = d >> 3;
  const long long wstep = static_cast<long long>(gridDim.x) * (blockDim.x >> 5);
  for (long long t = static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
       t < ntok; t += wstep) {
    const int r = __ldg(tok_row + t);
    if (!HILO_DCHECK(r >= 0 && r < rows_max, DCHECK_UNPACK_UPDATE_ROW)) continue;
    const float* s = out_img + static_cast<long long>(r) * d;
    uint4* xr = reinterpret_cast<uint4*>(x + t * d);
    for (int c = lane; c < G; c += 32 * U) {
      uint4 xv[U];
      F8 yv[U];
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (c + 32 * k < G) {
          xv[k] = xr[c + 32 * k];
          if (WIDE) {
            yv[k] = ldg8(s + 8 * (c + 32 * k));
          } else {
            const float4* s4 = reinterpret_cast<const float4*>(s) + 2 * (c + 32 * k);
            const float4 lo = __ldg(s4), hi = __ldg(s4 + 1);
            yv[k] = {{lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w}};
          }
        }
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (c + 32 * k < G) {
          float f[8], o[8];
          bf16x8_to_f32(xv[k], f);
#pragma unroll
          for (int u = 0; u < 8; ++u) o[u] = __fsub_rn(f[u], __fmul_rn(alpha, yv[k].v[u]));
          uint4 v;
          v.x = pack_bf16x2(o[0], o[1]);
          v.y = pack_bf16x2(o[2], o[3]);
          v.z = pack_bf16x2(o[4], o[5]);
          v.w = pack_bf16x2(o[6], o[7]);
          xr[c + 32 * k] = v;
        }
    }
  }
}

// ========================================================== layernorm =====
//
// A row of the row space per group of 128 threads (64 up to 256 elements, a warp up to
// 128), 384 threads per CTA, two CTAs per SM looping over the rows. Rows [0, n_txt) come
// from in_txt, rows [n_txt, n_txt + cu_img[B]) from in_img (bf16 or fp32). Thread t of a
// group of G holds elements 4t + 4G k. Writes the normalised row (no affine, eps 1e-6,
// biased variance) as bf16, fp16 or e4m3.
// Bound by memory latency: a row is one load round trip, two dependent
// reductions and a store, so each group loads its next row before it reduces the
// present one, and every row of a 2400-row block is asked for within two trips.
// (One CTA per row took 6 us until the last had started: 2389 bf16 rows of 3072
// elements 14.2 us, 5.7 so; fp32 rows 10 and 7; 10600 bf16 rows 45 and 25. 128 threads
// for a row of 128 elements: 10000 rows 7.6 us, 2.8 so; of 256 7.0 and 5.3.)

constexpr int LN_THREADS = 384;
constexpr int ln_group(int d) { return d <= 128 ? 32 : d <= 256 ? 64 : 128; }

// Over one group: `red` is 4 floats of its own, used by no other reduction
// until the group has met at two further barriers or ends its row.
template <int GROUP>
__device__ __forceinline__ void ln_group_sync() {
  named_bar_sync(1 + static_cast<int>(threadIdx.x) / GROUP, GROUP);
}

template <int GROUP>
__device__ __forceinline__ float ln_group_sum(float v, float* red) {
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if (GROUP == 32) return v;
  if ((threadIdx.x & 31) == 0) red[(threadIdx.x >> 5) % (GROUP / 32)] = v;
  ln_group_sync<GROUP>();
  return GROUP == 64 ? red[0] + red[1] : (red[0] + red[1]) + (red[2] + red[3]);
}

template <int GROUP>
__device__ __forceinline__ float ln_group_max(float v, float* red) {
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
  if (GROUP == 32) return v;
  if ((threadIdx.x & 31) == 0) red[(threadIdx.x >> 5) % (GROUP / 32)] = v;
  ln_group_sync<GROUP>();
  return GROUP == 64 ? fmaxf(red[0], red[1]) : fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3]));
}

// e4m3 row quantisation constants from the row's largest magnitude: inv =
// 448 / amax and scale = amax / 448, each one correctly rounded division
// (1 and 1 for an all-zero row)
__device__ __forceinline__ void e4m3_row_scale(float amax, float& inv, float& scale) {
  inv = amax > 0.f ? __fdiv_rn(448.0f, amax) : 1.0f;
  scale = amax > 0.f ? __fdiv_rn(amax, 448.0f) : 1.0f;
}

// ln_mode: 0 bf16, 1 fp16 (saturating), 2 e4m3 per row (ln_scale[r] = the
// row's dequantisation scale)
template <int NCH, bool F32, int GROUP>
__global__ void __launch_bounds__(LN_THREADS, 2) layernorm_kernel(const void* __restrict__ in_txt,
                                                                  const void* __restrict__ in_img,
                                                                  void* __restrict__ ln, int ln_mode,
                                                                  float* __restrict__ ln_scale,
                                                                  const int32_t* __restrict__ cu_img, int B,
                                                                  int n_txt, int cap, int d) {
  pdl_wait();
  pdl_trigger();
  constexpr int GROUPS = LN_THREADS / GROUP;
  __shared__ float red_s[GROUPS][3][4];
  const int group = threadIdx.x / GROUP, tid = threadIdx.x % GROUP;
  float(*red)[4] = red_s[group];
  const int rows = n_txt + min(cu_img[B], cap);
  const int step = gridDim.x * GROUPS;
  const float inv_d = 1.0f / static_cast<float>(d);
  uint4 raw[NCH];  // the next row as it is in memory (bf16: .x and .y)
  auto load = [&](int r) {
    const long long off = static_cast<long long>(r < n_txt ? r : r - n_txt) * d;
    const void* base = r < n_txt ? in_txt : in_img;
#pragma unroll
    for (int t = 0; t < NCH; ++t) {
      const int c = 4 * GROUP * t + 4 * tid;
      raw[t] = make_uint4(0u, 0u, 0u, 0u);
      if (c < d) {
        if (F32) {
          raw[t] = __ldg(reinterpret_cast<const uint4*>(static_cast<const float*>(base) + off + c));
        } else {
          const uint2 u = __ldg(reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(base) + off + c));
          raw[t].x = u.x;
          raw[t].y = u.y;
        }
      }
    }
  };
  int r = blockIdx.x + gridDim.x * group;
  if (r < rows) load(r);
  for (; r < rows; r += step) {
    float v[NCH * 4];
#pragma unroll
    for (int t = 0; t < NCH; ++t) {
      if (F32) {
        v[4 * t] = __uint_as_float(raw[t].x);
        v[4 * t + 1] = __uint_as_float(raw[t].y);
        v[4 * t + 2] = __uint_as_float(raw[t].z);
        v[4 * t + 3] = __uint_as_float(raw[t].w);
      } else {
        v[4 * t] = __uint_as_float(raw[t].x << 16);
        v[4 * t + 1] = __uint_as_float(raw[t].x & 0xFFFF0000u);
        v[4 * t + 2] = __uint_as_float(raw[t].y << 16);
        v[4 * t + 3] = __uint_as_float(raw[t].y & 0xFFFF0000u);
      }
    }
    if (r + step < rows) load(r + step);
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < NCH * 4; ++i) sum += v[i];
    const float mean = ln_group_sum<GROUP>(sum, red[0]) * inv_d;
    float sq = 0.f;
#pragma unroll
    for (int t = 0; t < NCH; ++t) {
      if (4 * GROUP * t + 4 * tid < d) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float e = v[4 * t + i] - mean;
          sq += e * e;
        }
      }
    }
    const float rstd = rsqrtf(ln_group_sum<GROUP>(sq, red[1]) * inv_d + 1e-6f);
    if (ln_mode == 2) {
      float am = 0.f;
#pragma unroll
      for (int t = 0; t < NCH; ++t)
        if (4 * GROUP * t + 4 * tid < d) {
#pragma unroll
          for (int i = 0; i < 4; ++i) am = fmaxf(am, fabsf((v[4 * t + i] - mean) * rstd));
        }
      float inv, scale;
      e4m3_row_scale(ln_group_max<GROUP>(am, red[2]), inv, scale);
      uint8_t* q = static_cast<uint8_t*>(ln) + static_cast<long long>(r) * d;
#pragma unroll
      for (int t = 0; t < NCH; ++t) {
        const int c = 4 * GROUP * t + 4 * tid;
        if (c >= d) continue;
        *reinterpret_cast<uint32_t*>(q + c) =
            pack_e4m3x4(__fmul_rn((v[4 * t] - mean) * rstd, inv), __fmul_rn((v[4 * t + 1] - mean) * rstd, inv),
                        __fmul_rn((v[4 * t + 2] - mean) * rstd, inv), __fmul_rn((v[4 * t + 3] - mean) * rstd, inv));
      }
      if (tid == 0) ln_scale[r] = scale;
      continue;
    }
    uint16_t* lo = static_cast<uint16_t*>(ln) + static_cast<long long>(r) * d;
#pragma unroll
    for (int t = 0; t < NCH; ++t) {
      const int c = 4 * GROUP * t + 4 * tid;
      if (c >= d) continue;
      const float y0 = (v[4 * t] - mean) * rstd, y1 = (v[4 * t + 1] - mean) * rstd;
      const float y2 = (v[4 * t + 2] - mean) * rstd, y3 = (v[4 * t + 3] - mean) * rstd;
      uint2 o;
      if (ln_mode == 1) {
        o.x = pack_f16x2_sat(y0, y1);
        o.y = pack_f16x2_sat(y2, y3);
      } else {
        o.x = pack_bf16x2(y0, y1);
        o.y = pack_bf16x2(y2, y3);
      }
      *reinterpret_cast<uint2*>(lo + c) = o;
    }
  }
}

// ==================================================== e4m3 rows =====
// Per-row e4m3 quantisation by persistent 256-thread CTAs. The row's largest
// magnitude, then each element times 448 / amax (fp32) rounded to e4m3; the
// dequantisation scale amax / 448 per row. TYPE 0 bf16, 1 fp16, 2 fp32; cols a
// multiple of 8. Rows: rows_static, or n_txt + min(cu_img[B], cap) when cu_img is
// given (the row space of the block). Bound by memory: 16-bit rows of up to 2048 NP
// elements (NP > 0) are read once and stay in registers while the next row is on its
// way; longer or fp32 rows (NP = 0) are read a second time, from L1 / L2. (The block
// of 2389 rows with e4m3 operands, which has two such passes, takes 6 us less than
// with all rows read twice. 12288 elements are what a thread can hold with three CTAs
// per SM: 80 registers. NP is the least that holds the row: with two pieces for all up to
// 4096 elements and six above, 2400 rows of 5120 took 7.5 us, 5.7 so; 10000 of 512 11.7
// and 8.7. The loops over fp32 rows are not unrolled, so that eight CTAs fit: 10000 rows
// of 2048 19.4 us unrolled, 25.3 with at most 42 registers, 16.2 so; longer 16-bit rows
// are, one row of 16384 3.3 us not unrolled and 2.3 so.)

constexpr int QR_THREADS = 256;

__device__ __forceinline__ void widen8(const uint4& u, int type, float* f) {
  if (type == 0) {
    bf16x8_to_f32(u, f);
    return;
  }
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __half2 h = *reinterpret_cast<const __half2*>(&w[j]);
    const float2 t = __half22float2(h);
    f[2 * j] = t.x;
    f[2 * j + 1] = t.y;
  }
}

__device__ __forceinline__ void load8(const void* src, int type, long long i8, float* f) {
  if (type == 2) {
    const float4* p = static_cast<const float4*>(src) + 2 * i8;
    const float4 a = __ldg(p), b = __ldg(p + 1);
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
    return;
  }
  widen8(__ldg(static_cast<const uint4*>(src) + i8), type, f);
}

__device__ __forceinline__ uint2 quant8(const float* f, float inv) {
  uint2 o;
  o.x = pack_e4m3x4(__fmul_rn(f[0], inv), __fmul_rn(f[1], inv), __fmul_rn(f[2], inv), __fmul_rn(f[3], inv));
  o.y = pack_e4m3x4(__fmul_rn(f[4], inv), __fmul_rn(f[5], inv), __fmul_rn(f[6], inv), __fmul_rn(f[7], inv));
  return o;
}

// The row's largest magnitude over the CTA; `red` is rewritten only after the
// CTA has met again.
__device__ __forceinline__ float quant_amax(float am, float* red) {
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, off));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = am;
  __syncthreads();
  am = red[0];
#pragma unroll
  for (int w = 1; w < QR_THREADS / 32; ++w) am = fmaxf(am, red[w]);
  return am;
}

// CTAs per SM
__host__ __device__ constexpr int quant_ctas(int np) { return np == 6 ? 3 : np == 3 ? 5 : np == 2 ? 6 : 8; }

template <int TYPE, int NP>
__global__ void __launch_bounds__(QR_THREADS, NP ? quant_ctas(NP) : TYPE == 2 ? 0 : 6)
    quant_rows_kernel(const void* __restrict__ src, int cols, int rows_static, const int32_t* __restrict__ cu_img,
                      int B, int n_txt, int cap, uint8_t* __restrict__ dst, float* __restrict__ scale) {
  constexpr bool REG = NP > 0;
  pdl_wait();
  pdl_trigger();
  __shared__ float red[2][QR_THREADS / 32];  // rows alternate
  const int rows = cu_img ? n_txt + min(cu_img[B], cap) : rows_static;
  const int g8 = cols >> 3;
  uint4 raw[REG ? NP : 1];
  auto load = [&](int r) {
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int g = threadIdx.x + k * QR_THREADS;
      raw[k] = make_uint4(0u, 0u, 0u, 0u);
      if (g < g8) raw[k] = __ldg(static_cast<const uint4*>(src) + static_cast<long long>(r) * g8 + g);
    }
  };
  if (REG && blockIdx.x < rows) load(blockIdx.x);
  int h = 0;
  for (int r = blockIdx.x; r < rows; r += gridDim.x, h ^= 1) {
    const long long base8 = static_cast<long long>(r) * g8;
    float am = 0.f, inv, sc;
    if constexpr (REG) {
      uint4 cur[NP];
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        cur[k] = raw[k];
        float f[8];
        widen8(cur[k], TYPE, f);
#pragma unroll
        for (int i = 0; i < 8; ++i) am = fmaxf(am, fabsf(f[i]));
      }
      if (r + static_cast<long long>(gridDim.x) < rows) load(r + gridDim.x);
      e4m3_row_scale(quant_amax(am, red[h]), inv, sc);
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        const int g = threadIdx.x + k * QR_THREADS;
        float f[8];
        widen8(cur[k], TYPE, f);
        if (g < g8) reinterpret_cast<uint2*>(dst)[base8 + g] = quant8(f, inv);
      }
    } else {
#pragma unroll(TYPE == 2 ? 1 : 4)
      for (int g = threadIdx.x; g < g8; g += QR_THREADS) {
        float f[8];
        load8(src, TYPE, base8 + g, f);
#pragma unroll
        for (int i = 0; i < 8; ++i) am = fmaxf(am, fabsf(f[i]));
      }
      e4m3_row_scale(quant_amax(am, red[h]), inv, sc);
      // second pass: the row is in L1 / L2 from the first
#pragma unroll(TYPE == 2 ? 1 : 4)
      for (int g = threadIdx.x; g < g8; g += QR_THREADS) {
        float f[8];
        load8(src, TYPE, base8 + g, f);
        reinterpret_cast<uint2*>(dst)[base8 + g] = quant8(f, inv);
      }
    }
    if (threadIdx.x == 0) scale[r] = sc;
  }
}

// ===================================================== bf16 -> fp16 =====
// Weight conversion at load time (exact for bf16 values in the fp16 normal
// range; saturating at +-65504).

__global__ void __launch_bounds__(256) bf16_to_f16_kernel(const uint4* __restrict__ src,
                                                          uint4* __restrict__ dst, long long n8) {
  pdl_wait();
  pdl_trigger();
  for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < n8;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    float f[8];
    bf16x8_to_f32(__ldg(src + i), f);
    uint4 o;
    o.x = pack_f16x2_sat(f[0], f[1]);
    o.y = pack_f16x2_sat(f[2], f[3]);
    o.z = pack_f16x2_sat(f[4], f[5]);
    o.w = pack_f16x2_sat(f[6], f[7]);
    dst[i] = o;
  }
}

// ============================================================ launchers ===

static int grid_for(long long work_items, int per_block, int num_sms, int blocks_per_sm) {
  long long g = (work_items + per_block - 1) / per_block;
  const long long cap = static_cast<long long>(num_sms) * blocks_per_sm;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return static_cast<int>(g);
}

cudaError_t launch_score(const void* x, float* s, int B, int H, int W, int d, int num_sms,
                         cudaStream_t st) {
  const long long nwin = static_cast<long long>(B) * (H / 2) * (W / 2);
  const int iters = (d + 8 * SCORE_THREADS - 1) / (8 * SCORE_THREADS);
  auto* kern = iters == 1 ? score_kernel<1> : iters == 2 ? score_kernel<2> : iters == 3 ? score_kernel<3> : score_kernel<4>;
  return launch_pdl(kern, dim3(grid_for(nwin, 1, num_sms, 16)), dim3(SCORE_THREADS), 0, st,
                    static_cast<const __nv_bfloat16*>(x), s, B, H, W, d);
}

template <bool GRANULAR, bool LFMODE>
static auto split_kernel_for(int ch) {
  switch (ch) {
    case 4: return split_select_kernel<4, GRANULAR, LFMODE>;
    case 8: return split_select_kernel<8, GRANULAR, LFMODE>;
    case 16: return split_select_kernel<16, GRANULAR, LFMODE>;
    default: return split_select_kernel<32, GRANULAR, LFMODE>;
  }
}

cudaError_t launch_split(const float* score, const uint8_t* mask, const int32_t* k_keep,
                         const int32_t* k_mid, uint8_t* labels, int32_t* row_src, int32_t* counts,
                         int32_t* cu_img, int32_t* tok_row, int B, int H, int W, int levels,
                         int granular, int lf, cudaStream_t st) {
  const int N = H * W;
  // tokens per thread: as few as 1024 threads allow (one level, half as many threads: 17.2
  // instead of 13.4 us for 96x96 and 25.5 instead of 21.7 for 128x128)
  int ch = 4;
  while (ch < 32 && N > ch * SPLIT_THREADS) ch *= 2;
  int threads = (((N + ch - 1) / ch + 31) / 32) * 32;
  threads = threads < 256 ? 256 : threads;
  auto* kern = lf ? split_kernel_for<false, true>(ch)
                  : (granular ? split_kernel_for<true, false>(ch) : split_kernel_for<false, false>(ch));
  // One image: its rows begin at 0. Up to SPLIT_CLUSTER (8, the largest cluster every
  // device takes): the images' CTAs are one cluster, padded to a power of two, and tell
  // one another their row counts. More: a second kernel, once all counts are written
  // (eight images of 64x64 took 10.3 us that way, 7.6 as a cluster).
  int fused = 1;
  while (fused < B && fused <= SPLIT_CLUSTER) fused *= 2;
  if (fused > SPLIT_CLUSTER) fused = 0;
  // at most 32 KB of labels: no larger shared-memory limit to ask for
  const cudaError_t e =
      launch_pdl_cluster(kern, fused > 1 ? fused : 1, dim3(fused > 1 ? fused : B), dim3(threads), N, st, score, mask,
                         k_keep, k_mid, labels, counts, B, H, W, levels, lf, fused, cu_img, row_src, tok_row);
  if (e != cudaSuccess || fused) return e;
  return launch_pdl(split_compact_kernel, dim3(B), dim3(SPLIT_THREADS), N, st,
                    static_cast<const uint8_t*>(labels), static_cast<const int32_t*>(counts), cu_img,
                    row_src, tok_row, H, W, levels, lf);
}

// CTAs per SM on pack_kernel's grid of a row per CTA and turn. The hardware deals further
// CTAs as others end, which evens out rows of one to sixteen members, but one without a
// row still costs its launch, and the capacity is several times the rows: 24 per SM
// from about 5000 rows of capacity on, else 16 (4096 rows of 2048 channels: 5.1 us with
// 16, 6.2 with 24; 16384 of 3072 with two levels 28.6 and 26.4; 5120 rows 10.4 and 10.2;
// four images of 64x64, a quarter kept, of 640 channels 12.3 and 10.9, of 1152 16.9 and
// 14.1, of 4096 40.5 and 36.6; one image of 128x128 of 2048 20.2 and 21.2).
static int pack_ctas(long long items, int num_sms) { return items <= 32LL * num_sms ? 16 : 24; }

cudaError_t launch_pack(const void* x, const uint8_t* labels, const int32_t* row_src,
                        const int32_t* counts, const int32_t* cu_img, void* packed, int B, int H,
                        int W, int d, int cap, int lf, int num_sms, cudaStream_t st) {
  const auto* xs = static_cast<const __nv_bfloat16*>(x);
  auto* ps = static_cast<__nv_bfloat16*>(packed);
  const int wpr = pack_warps(d);
  const bool small = wpr < 4;
  const int threads = small ? PACK_THREADS_SHORT : PACK_THREADS, rows = threads / (32 * wpr);  // rows per CTA and turn
  if (lf == 2 || lf == 4 || lf == 8) {
    // rows of 8x8 windows: 64 loads per lane whatever the width, so one to a CTA
    const bool few = small && lf < 8;
    auto* kern = lf == 8   ? pack_lf_kernel<8, 4, PACK_THREADS>
                 : lf == 4 ? (!few       ? pack_lf_kernel<4, 4, PACK_THREADS>
                              : wpr == 1 ? pack_lf_kernel<4, 1, PACK_THREADS_SHORT>
                                         : pack_lf_kernel<4, 2, PACK_THREADS_SHORT>)
                           : (!few       ? pack_lf_kernel<2, 4, PACK_THREADS>
                              : wpr == 1 ? pack_lf_kernel<2, 1, PACK_THREADS_SHORT>
                                         : pack_lf_kernel<2, 2, PACK_THREADS_SHORT>);
    const long long items = cap + (lf > 2 ? static_cast<long long>(B) * (H / lf) * (W / lf) * lf_slices(lf, d) : 0);
    // 24 CTAs per SM, but 16 where that many hold most of the rows and the rows are short
    // (64x64 tokens, 2x2 windows, a quarter kept: of 1152 channels 5.2 us with 24, 3.8 so, of
    // 2048 5.3 and 4.2, none kept of 3072 4.7 and 6.1; 4x4 windows of 1024 4.3 and 3.3, of 2048
    // 4.6 and 4.9; 8x8 of 3072, four images, 12.3 and 12.7)
    const int ctas = few ? 8 : items <= 40LL * num_sms && d <= (lf == 2 ? 2048 : 1152) ? 16 : 24;
    return launch_pdl(kern, dim3(grid_for(items, few ? rows : 1, num_sms, ctas)),
                      dim3(few ? PACK_THREADS_SHORT : PACK_THREADS), 0, st, xs, row_src, counts, cu_img, ps, B, H, W, d,
                      cap);
  }
  if (lf) return cudaErrorInvalidValue;
  auto* kern = wpr == 1     ? pack_kernel<1, PACK_THREADS_SHORT, 1>
               : wpr == 2   ? pack_kernel<2, PACK_THREADS_SHORT, 1>
               : d <= 1024  ? pack_kernel<4, PACK_THREADS, 1>
               : d <= 3072  ? pack_kernel<4, PACK_THREADS, 3>
                            : pack_kernel<4, PACK_THREADS, 4>;
  return launch_pdl(kern, dim3(grid_for(cap, rows, num_sms, small ? 8 : pack_ctas(cap, num_sms))), dim3(threads), 0, st,
                    xs, labels, row_src, counts, cu_img, ps, B, H, W, d, cap);
}

// CTAs per SM on the unpacks' grids: more than are resident, so that the hardware deals
// them as others end (128x128 of 3072 channels, delta: 60.8 us with 8, 59.9 with 32;
// small grids alike). Rows of up to 256 channels are one piece per lane: no batches, so
// as many warps as the registers allow, and with little to do per token a grid of what
// is resident (128x128 of 128 channels, buffers not in L2: nearest 5.5 us, 4.0 so, delta
// 6.8 and 5.8, update 5.1 and 4.2; of 256 channels 6.3 and 5.4, 8.2 and 7.5, 5.6 and 5.1).
constexpr int UNPACK_CTAS = 32, UNPACK_CTAS_SHORT = 8;
static bool short_row(int d) { return d <= 256; }
static dim3 unpack_grid(long long ntok, int d, int num_sms) {
  return dim3(grid_for(ntok, 8, num_sms, short_row(d) ? UNPACK_CTAS_SHORT : UNPACK_CTAS));
}

// 32-byte accesses on fp32 rows, where a row keeps a whole warp busy with them: it is a
// multiple of 512 bytes, so beyond that the arrays' addresses decide.
static bool wide(const float* a, const float* b, int d) {
  return d >= 256 && ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 31) == 0;
}

cudaError_t launch_unpack(const float* out_img, const int32_t* tok_row, float* y, long long ntok,
                          int d, long long rows_max, int num_sms, cudaStream_t st) {
  const bool w = wide(out_img, y, d), one = short_row(d);
  auto* kern = w ? (one ? unpack_kernel<true, 1> : unpack_kernel<true, 4>) : (one ? unpack_kernel<false, 1> : unpack_kernel<false, 4>);
  return launch_pdl(kern, unpack_grid(ntok, d, num_sms), dim3(256), 0, st, out_img,
                    tok_row, y, ntok, d, rows_max);
}

cudaError_t launch_row_sizes(const uint8_t* labels, const int32_t* row_src, const int32_t* counts,
                             const int32_t* cu_img, float* n_img, int B, int H, int W, int cap, int lf,
                             int num_sms, cudaStream_t st) {
  if (cap <= 0) return cudaSuccess;
  return launch_pdl(row_sizes_kernel, dim3(grid_for(cap, 256, num_sms, 4)), dim3(256), 0, st, labels, row_src,
                    counts, cu_img, n_img, B, H, W, cap, lf);
}

cudaError_t launch_unpack_delta(const float* out_img, const void* packed, const void* x,
                                const uint8_t* labels, const int32_t* tok_row, float* y, long long ntok,
                                int d, long long rows_max, int num_sms, cudaStream_t st) {
  const bool w = wide(out_img, y, d), one = short_row(d);
  auto* kern = w ? (one ? unpack_delta_kernel<true, 1> : unpack_delta_kernel<true, 2>) : (one ? unpack_delta_kernel<false, 1> : unpack_delta_kernel<false, 2>);
  return launch_pdl(kern, unpack_grid(ntok, d, num_sms), dim3(256), 0, st, out_img,
                    static_cast<const __nv_bfloat16*>(packed), static_cast<const __nv_bfloat16*>(x), labels,
                    tok_row, y, ntok, d, rows_max);
}

cudaError_t launch_unpack_update(const float* out_img, const int32_t* tok_row, void* x,
                                 long long ntok, int d, float alpha, long long rows_max, int num_sms,
                                 cudaStream_t st) {
  const bool w = wide(out_img, out_img, d), one = short_row(d);
  auto* kern = w ? (one ? unpack_update_kernel<true, 1> : unpack_update_kernel<true, 2>) : (one ? unpack_update_kernel<false, 1> : unpack_update_kernel<false, 2>);
  return launch_pdl(kern, unpack_grid(ntok, d, num_sms), dim3(256), 0, st,
                    out_img, tok_row, static_cast<__nv_bfloat16*>(x), ntok, d, alpha, rows_max);
}

cudaError_t launch_quant_rows(const void* src, int type, int cols, int rows_static, const int32_t* cu_img,
                              int B, int n_txt, int cap, uint8_t* dst, float* scale, int num_sms,
                              cudaStream_t st) {
  const long long rmax = cu_img ? static_cast<long long>(n_txt) + cap : rows_static;
  if (rmax <= 0) return cudaSuccess;
  const int np = type == 2 || cols > 6 * 2048 ? 0 : cols > 3 * 2048 ? 6 : (cols + 2047) / 2048;
#define HILO_QUANT(T) \
  (np == 1 ? quant_rows_kernel<T, 1> : np == 2 ? quant_rows_kernel<T, 2> : np == 3 ? quant_rows_kernel<T, 3> \
   : np == 6 ? quant_rows_kernel<T, 6> : quant_rows_kernel<T, 0>)
  auto* kern = type == 2 ? quant_rows_kernel<2, 0> : type == 0 ? HILO_QUANT(0) : HILO_QUANT(1);
#undef HILO_QUANT
  return launch_pdl(kern, dim3(grid_for(rmax, 1, num_sms, quant_ctas(np))), dim3(QR_THREADS), 0, st,
                    src, cols, rows_static, cu_img, B, n_txt, cap, dst, scale);
}

cudaError_t launch_bf16_to_f16(const void* src, void* dst, long long n, int num_sms,
                               cudaStream_t st) {
  if (n % 8) return cudaErrorInvalidValue;
  const long long n8 = n / 8;
  return launch_pdl(bf16_to_f16_kernel, dim3(grid_for(n8, 256, num_sms, 8)), dim3(256), 0, st,
                    static_cast<const uint4*>(src), static_cast<uint4*>(dst), n8);
}

cudaError_t launch_layernorm(const void* in_txt, const void* in_img, int in_f32, void* ln, int ln_mode,
                             float* ln_scale, const int32_t* cu_img, int B, int n_txt, int cap, int d, int num_sms,
                             cudaStream_t st) {
  const int group = ln_group(d);
  const dim3 grid(grid_for(static_cast<long long>(n_txt) + cap, LN_THREADS / group, num_sms, 2));
#define HILO_LN(NC, G)                                                                                            \
  (in_f32 ? launch_pdl(layernorm_kernel<NC, true, G>, grid, dim3(LN_THREADS), 0, st, in_txt, in_img, ln, ln_mode, \
                       ln_scale, cu_img, B, n_txt, cap, d)                                                        \
          : launch_pdl(layernorm_kernel<NC, false, G>, grid, dim3(LN_THREADS), 0, st, in_txt, in_img, ln, ln_mode, \
                       ln_scale, cu_img, B, n_txt, cap, d))
  if (group == 32) return HILO_LN(1, 32);
  if (group == 64) return HILO_LN(1, 64);
  switch ((d + 511) / 512) {
#define HILO_LN_CASE(NC) \
  case NC:               \
    return HILO_LN(NC, 128);
    HILO_LN_CASE(1)
    HILO_LN_CASE(2)
    HILO_LN_CASE(3)
    HILO_LN_CASE(4)
    HILO_LN_CASE(5)
    HILO_LN_CASE(6)
    HILO_LN_CASE(7)
    HILO_LN_CASE(8)
#undef HILO_LN_CASE
#undef HILO_LN
    default:
      return cudaErrorInvalidValue;
  }
}

// ================================================== wait-timeout probe =====
// One thread waits on an mbarrier that nothing arrives at, with the bounded
// wait of the tcgen05 kernels; when the limit passes, the wait latches
// DEV_TIMEOUT_PROBE in g_probe_err and the kernel returns.

__device__ int g_probe_err;

__global__ void wait_probe_kernel() {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  abort_flag = 0;
  fence_mbar_init();
  mbar_wait(&bar, 0, &abort_flag, &g_probe_err, DEV_TIMEOUT_PROBE);
}

cudaError_t launch_wait_probe(cudaStream_t st) {
  wait_probe_kernel<<<1, 32, 0, st>>>();
  return cudaGetLastError();
}

int probe_take_device_error() {
  int v = 0;
  const int z = 0;
  if (cudaMemcpyFromSymbol(&v, g_probe_err, sizeof(int)) != cudaSuccess) return -1;
  if (v) cudaMemcpyToSymbol(g_probe_err, &z, sizeof(int));
  return v;
}

int dcheck_take_bw() {
#ifdef HILO_DEVICE_CHECKS
  int v = 0;
  const int z = 0;
  if (cudaMemcpyFromSymbol(&v, g_dcheck, sizeof(int)) != cudaSuccess) return -1;
  if (v) cudaMemcpyToSymbol(g_dcheck, &z, sizeof(int));
  return v;
#else
  return 0;
#endif
}

}  // namespace hilo
