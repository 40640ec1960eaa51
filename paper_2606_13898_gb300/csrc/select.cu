// The paper's token selector (Sec. 2.3 "HiLo-Token Selection"): a Sobel
// frequency map of the input image, normalised by its per-image maximum,
// thresholded and regionalised onto the token grid (each token covers P x P
// pixels), united with the user mask dilated by R tokens.
//
// Two kernels:
//   sobel_tokmax_kernel  one CTA per 32 x 64 pixel tile (plus a one-pixel
//                        halo, replicate borders) in shared memory, pixels as
//                        in the image; full-width tiles load and store their
//                        interior as 16-byte vectors. Each thread walks 8
//                        consecutive pixel rows of one column, so the
//                        horizontal sums of a row serve as the bottom term of
//                        one pixel and the top term of the pixel two rows
//                        below (the same value, not a re-association). The
//                        largest squared magnitude of each token comes from
//                        per-thread maxima, a warp reduction over the lanes
//                        of one token and one shared atomic per token and
//                        warp, on the float bits (squares are >= +0, so their
//                        bit patterns order like the values); the square root
//                        is taken once per token (it keeps the order). The
//                        tile's maximum goes to its own slot (no global
//                        atomics, nothing to clear). Bound by instruction
//                        issue: 1024x1024 pixels of 3 channels 7.4 us with the
//                        keep kernel, 8.9 with channel planes and a root per
//                        pixel; 2048x2048 20.2 and 24.1.
//   sobel_keep_kernel    one CTA per 16 x 16 tokens: the mask tile and a halo
//                        of R tokens as bits in shared memory, the image
//                        maximum from the tile slots; per token: any mask
//                        token within R tokens (square window), or tokmax /
//                        imgmax (one correctly rounded division) > threshold.
// Order of the magnitude, per channel c (P the replicate-padded pixels):
//   gx = ((P(y-1,x+1) + 2 P(y,x+1)) + P(y+1,x+1)) - ((P(y-1,x-1) + 2 P(y,x-1)) + P(y+1,x-1))
//   gy = ((P(y+1,x-1) + 2 P(y+1,x)) + P(y+1,x+1)) - ((P(y-1,x-1) + 2 P(y-1,x)) + P(y-1,x+1))
//   acc = acc + (gx gx + gy gy) over c ascending from 0;  g = sqrt(acc)
// with every operation an explicitly rounded fp32 add, mul or sqrt, so the
// keep map equals a CPU evaluation of the same definition bit for bit.
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "internal.h"

namespace hilo {

namespace {

constexpr int TILE_Y = 32;
constexpr int TILE_X = 64;
constexpr int SOBEL_THREADS = 256;
constexpr int ROWS = TILE_Y / (SOBEL_THREADS / TILE_X);  // consecutive pixel rows per thread

// (a + 2 b) + c, each step rounded to fp32
__device__ __forceinline__ float sobel_sum3(float a, float b, float c) {
  return __fadd_rn(__fadd_rn(a, __fmul_rn(2.0f, b)), c);
}

// The C channels of one pixel of the tile. (Lanes are C floats apart: one float at a
// time meets no bank conflict for odd C, and even C takes one vector.)
template <int C>
__device__ __forceinline__ void load_pixel(const float* p, float (&v)[C]) {
  if constexpr (C == 4) {
    const float4 f = *reinterpret_cast<const float4*>(p);
    v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
  } else if constexpr (C == 2) {
    const float2 f = *reinterpret_cast<const float2*>(p);
    v[0] = f.x, v[1] = f.y;
  } else {
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] = p[c];
  }
}

// Tiles of the tokmax grid for an H x W-token image at `patch` pixels per
// token: one maximum slot each.
inline int sobel_tiles(int H, int W, int patch) {
  return ((W * patch + TILE_X - 1) / TILE_X) * ((H * patch + TILE_Y - 1) / TILE_Y);
}

// Five CTAs per SM, as far as registers and tiles allow (six spill and are slower).
template <int P, int C>
__global__ void __launch_bounds__(SOBEL_THREADS, C == 4 ? 4 : 5) sobel_tokmax_kernel(const float* __restrict__ img,
                                                                     float* __restrict__ tokmax,
                                                                     uint32_t* __restrict__ tilemax, int H,
                                                                     int W, int vec_ok) {
  pdl_wait();
  pdl_trigger();
  constexpr int TOK_Y = TILE_Y / P, TOK_X = TILE_X / P;
  static_assert(TOK_Y * TOK_X <= 32, "token maxima of a tile fit one warp");
  // a row: the left halo pixel ends at FIRST, where the 64 pixels begin
  constexpr int FIRST = 4, STRIDE = TILE_X * C + 2 * FIRST;
  __shared__ __align__(16) float tile[TILE_Y + 2][STRIDE];
  __shared__ uint32_t tmax[TOK_Y * TOK_X];
  const int Hp = H * P, Wp = W * P;
  const int b = blockIdx.z;
  const int y0 = blockIdx.y * TILE_Y, x0 = blockIdx.x * TILE_X;
  const float* base = img + static_cast<long long>(b) * Hp * Wp * C;
  if (threadIdx.x < TOK_Y * TOK_X) tmax[threadIdx.x] = 0u;
  if (vec_ok && x0 + TILE_X <= Wp) {
    // Interior columns x0 .. x0 + 63 of each (row-clamped) tile row are
    // 64 C contiguous floats starting at a multiple of 4 floats (x0 is a
    // multiple of 64, Wp of 8, the image 16-byte aligned): 16 C vectors. The
    // two halo columns are single floats. Every load is issued before the
    // first shared store, so the whole tile is in flight at once.
    constexpr int V = TILE_X * C / 4;
    constexpr int NV = (TILE_Y + 2) * V;
    constexpr int PERV = (NV + SOBEL_THREADS - 1) / SOBEL_THREADS;
    constexpr int NH = (TILE_Y + 2) * 2 * C;
    constexpr int PERH = (NH + SOBEL_THREADS - 1) / SOBEL_THREADS;
    float4 v[PERV];
    float h[PERH];
#pragma unroll
    for (int k = 0; k < PERV; ++k) {
      const int e = threadIdx.x + k * SOBEL_THREADS;
      if (e < NV) {
        const int yy = e / V, m = e - yy * V;
        const int gy = min(max(y0 + yy - 1, 0), Hp - 1);
        v[k] = __ldg(reinterpret_cast<const float4*>(base + (static_cast<long long>(gy) * Wp + x0) * C) + m);
      }
    }
#pragma unroll
    for (int k = 0; k < PERH; ++k) {
      const int e = threadIdx.x + k * SOBEL_THREADS;
      if (e < NH) {
        const int yy = e / (2 * C), w = e - yy * (2 * C);
        const int side = w / C, c = w - side * C;
        const int gy = min(max(y0 + yy - 1, 0), Hp - 1);
        const int gx = side ? min(x0 + TILE_X, Wp - 1) : max(x0 - 1, 0);
        h[k] = __ldg(base + (static_cast<long long>(gy) * Wp + gx) * C + c);
      }
    }
#pragma unroll
    for (int k = 0; k < PERV; ++k) {
      const int e = threadIdx.x + k * SOBEL_THREADS;
      if (e < NV) {
        const int yy = e / V, m = e - yy * V;
        *reinterpret_cast<float4*>(&tile[yy][FIRST + 4 * m]) = v[k];
      }
    }
#pragma unroll
    for (int k = 0; k < PERH; ++k) {
      const int e = threadIdx.x + k * SOBEL_THREADS;
      if (e < NH) {
        const int yy = e / (2 * C), w = e - yy * (2 * C);
        const int side = w / C, c = w - side * C;
        tile[yy][(side ? FIRST + TILE_X * C : FIRST - C) + c] = h[k];
      }
    }
  } else {
    // partial tiles (right image edge) and unaligned images: one clamped
    // float per element
    constexpr int ROW = (TILE_X + 2) * C;
    constexpr int TOTAL = (TILE_Y + 2) * ROW;
    for (int e = threadIdx.x; e < TOTAL; e += SOBEL_THREADS) {
      const int yy = e / ROW, w = e - yy * ROW;
      const int xx = w / C, c = w - xx * C;
      const int gy = min(max(y0 + yy - 1, 0), Hp - 1);
      const int gx = min(max(x0 + xx - 1, 0), Wp - 1);
      tile[yy][FIRST - C + w] = __ldg(base + (static_cast<long long>(gy) * Wp + gx) * C + c);
    }
  }
  __syncthreads();
  // Thread t takes pixel column tx = t % 64 and the ROWS consecutive rows
  // from ty0 = (t / 64) ROWS; ROWS divides P, so they all lie in token row
  // ty0 / P. A warp covers 32 consecutive columns (32 / P tokens).
  static_assert(SOBEL_THREADS % TILE_X == 0 && 32 % P == 0 && P % ROWS == 0, "tile mapping");
  const int tx = threadIdx.x % TILE_X, ty0 = (threadIdx.x / TILE_X) * ROWS;
  const int q = tx + 1;  // column in the padded tile
  // sliding 3-row window per channel: up/mid/dn rows at columns q-1, q, q+1,
  // and the horizontal sums of the up and mid rows
  float up[C][3], mid[C][3], hup[C], hmid[C];
  const int q0 = FIRST - C + (q - 1) * C;  // its left neighbour
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    float u[C], v[C];
    load_pixel<C>(&tile[ty0][q0 + i * C], u);
    load_pixel<C>(&tile[ty0 + 1][q0 + i * C], v);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      up[c][i] = u[c];
      mid[c][i] = v[c];
    }
  }
#pragma unroll
  for (int c = 0; c < C; ++c) {
    hup[c] = sobel_sum3(up[c][0], up[c][1], up[c][2]);
    hmid[c] = sobel_sum3(mid[c][0], mid[c][1], mid[c][2]);
  }
  const bool col_ok = x0 + tx < Wp;
  uint32_t mx = 0u;
#pragma unroll
  for (int j = 0; j < ROWS; ++j) {
    const int r = ty0 + 1 + j;  // row in the padded tile
    float acc = 0.0f;
    float px[3][C];
#pragma unroll
    for (int i = 0; i < 3; ++i) load_pixel<C>(&tile[r + 1][q0 + i * C], px[i]);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const float dn[3] = {px[0][c], px[1][c], px[2][c]};
      const float hdn = sobel_sum3(dn[0], dn[1], dn[2]);                  // bottom
      const float right = sobel_sum3(up[c][2], mid[c][2], dn[2]);
      const float left = sobel_sum3(up[c][0], mid[c][0], dn[0]);
      const float gx = __fsub_rn(right, left);
      const float gy = __fsub_rn(hdn, hup[c]);                            // bottom - top
      acc = __fadd_rn(acc, __fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy)));
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        up[c][i] = mid[c][i];
        mid[c][i] = dn[i];
      }
      hup[c] = hmid[c];
      hmid[c] = hdn;
    }
    if (col_ok && y0 + ty0 + j < Hp) mx = max(mx, __float_as_uint(acc));
  }
  const int lane = threadIdx.x & 31;
  const uint32_t seg = (P >= 32 ? 0xffffffffu : ((1u << P) - 1u)) << (lane & ~(P - 1));
  const uint32_t m = __reduce_max_sync(seg, mx);
  if ((lane & (P - 1)) == 0) atomicMax(&tmax[(ty0 / P) * TOK_X + tx / P], m);
  __syncthreads();
  if (threadIdx.x < 32) {
    uint32_t t = 0u;
    if (threadIdx.x < TOK_Y * TOK_X) {
      const int ti = blockIdx.y * TOK_Y + threadIdx.x / TOK_X;
      const int tj = blockIdx.x * TOK_X + threadIdx.x % TOK_X;
      if (ti < H && tj < W) {
        // a correctly rounded square root keeps the order, so one per token will do
        t = __float_as_uint(__fsqrt_rn(__uint_as_float(tmax[threadIdx.x])));
        tokmax[(static_cast<long long>(b) * H + ti) * W + tj] = __uint_as_float(t);
      }
    }
    t = __reduce_max_sync(0xffffffffu, t);
    if (threadIdx.x == 0) tilemax[(static_cast<long long>(b) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
  }
}

// One CTA per 16 x 16 tokens: the mask tile with a halo of `radius` tokens as bits, the
// tokens' dilation windows (radius <= MAX_RADIUS) from them, then the image maximum from
// the tile slots and the token's normalised maximum. A chain of short waits, no unit is
// busy. The mask was complete before the magnitude kernel, which waits for its own
// predecessor, let this one start, so the dilation runs beside that kernel, ahead of the
// wait. A warp reads a row of the halo at a time; its first lanes find which of the 16
// columns have a mask token within reach in that row, and a token looks at one such
// word per row. (Every token walking its whole window of bytes here, selected by its
// magnitude or not, took 991 us at 64x64 tokens of 16 pixels and radius 64, 13.5 so;
// radius 16 74.6 and 7.6, radius 4 12.3 and 7.3, radius 1 6.9 and 7.0.)
constexpr int KEEP_T = 16;
constexpr int MAX_RADIUS = 64;
constexpr int KEEP_WARPS = KEEP_T * KEEP_T / 32;
constexpr int KEEP_WORDS = (KEEP_T + 2 * MAX_RADIUS + 31) / 32;  // of a row of the halo

// Unused shared memory that spreads these CTAs over the SMs: without it many share one
// SM, the next magnitude kernel's CTAs find the others fuller, and three images of 46x30
// tokens, one selection after another, take 13.0 us instead of 10.2.
constexpr int KEEP_SMEM = 20480;

// WORDS: 32-bit words of a row of the halo (1 up to radius 8)
template <int WORDS>
__global__ void __launch_bounds__(KEEP_T * KEEP_T) sobel_keep_kernel(const float* __restrict__ tokmax,
                                                                   const uint32_t* __restrict__ tilemax,
                                                                   int ntiles, const uint8_t* __restrict__ mask,
                                                                   uint8_t* __restrict__ keep, int H, int W,
                                                                   int radius, float threshold) {
  __shared__ uint32_t near[KEEP_T + 2 * MAX_RADIUS];  // bit c: a mask token within reach of column c
  __shared__ uint32_t wred[KEEP_WARPS];
  const int b = blockIdx.z;
  const int i0 = blockIdx.y * KEEP_T - radius, j0 = blockIdx.x * KEEP_T - radius;
  const int S = KEEP_T + 2 * radius;
  const int lane = threadIdx.x & 31;
  const uint8_t* mb = mask + static_cast<long long>(b) * H * W;
  // four rows of each warp at a time, all their loads in flight
  for (int r0 = threadIdx.x >> 5; r0 < S; r0 += 4 * KEEP_WARPS) {
    uint32_t v[4][WORDS];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = r0 + q * KEEP_WARPS, ii = i0 + r;
#pragma unroll
      for (int w = 0; w < WORDS; ++w) {
        const int c = 32 * w + lane, jj = j0 + c;
        v[q][w] = 0u;
        if (r < S && c < S && ii >= 0 && ii < H && jj >= 0 && jj < W) v[q][w] = __ldcg(mb + ii * W + jj);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      bool any = false;  // column `lane` reaches the bits lane .. lane + 2 radius of the row
#pragma unroll
      for (int w = 0; w < WORDS; ++w) {
        if (w > 0 && 32 * w >= S) break;
        const uint32_t m = __ballot_sync(0xffffffffu, v[q][w] != 0u);
        const int lo = lane - 32 * w, hi = lane + 2 * radius - 32 * w;
        if (hi >= 0) any |= (m & (0xffffffffu << max(lo, 0)) & (0xffffffffu >> (31 - min(hi, 31)))) != 0u;
      }
      const uint32_t cols = __ballot_sync(0xffffffffu, any && lane < KEEP_T);
      const int r = r0 + q * KEEP_WARPS;
      if (lane == 0 && r < S) near[r] = cols;
    }
  }
  __syncthreads();
  const int ti = threadIdx.x / KEEP_T, tj = threadIdx.x % KEEP_T;
  uint32_t reach = 0u;
#pragma unroll 8
  for (int di = 0; di <= 2 * radius; ++di) reach |= near[ti + di];
  const bool k = (reach >> tj) & 1u;
  pdl_wait();
  pdl_trigger();
  uint32_t gm = 0u;
  const uint32_t* tb = tilemax + static_cast<long long>(b) * ntiles;
  for (int e = threadIdx.x; e < ntiles; e += blockDim.x) gm = max(gm, tb[e]);
  gm = __reduce_max_sync(0xffffffffu, gm);
  if ((threadIdx.x & 31) == 0) wred[threadIdx.x >> 5] = gm;
  __syncthreads();
  gm = wred[0];
#pragma unroll
  for (int w = 1; w < KEEP_WARPS; ++w) gm = max(gm, wred[w]);
  const int i = blockIdx.y * KEEP_T + ti, j = blockIdx.x * KEEP_T + tj;
  if (i >= H || j >= W) return;
  const long long t = (static_cast<long long>(b) * H + i) * W + j;
  // 0 / 0 (an image without any gradient) is NaN and selects nothing
  const float f = __fdiv_rn(tokmax[t], __uint_as_float(gm));
  keep[t] = k || f > threshold ? 1 : 0;
}

}  // namespace

size_t sobel_workspace_bytes(int B, int H, int W) {
  // token maxima, then one slot per tokmax tile at the larger tile count of
  // the two patch sizes (16 pixels per token)
  return static_cast<size_t>(B) * H * W * sizeof(float) + 256 +
         static_cast<size_t>(B) * sobel_tiles(H, W, 16) * sizeof(uint32_t);
}

cudaError_t launch_sobel_select(const float* img, int B, int H, int W, int C, int patch,
                                const uint8_t* mask, int radius, float threshold, uint8_t* keep, void* ws,
                                int num_sms, cudaStream_t st) {
  (void)num_sms;
  if (radius > MAX_RADIUS) return cudaErrorInvalidValue;
  float* tokmax = static_cast<float*>(ws);
  uint32_t* tilemax = reinterpret_cast<uint32_t*>(
      (reinterpret_cast<uintptr_t>(tokmax + static_cast<size_t>(B) * H * W) + 255) & ~static_cast<uintptr_t>(255));
  const int vec_ok = (reinterpret_cast<uintptr_t>(img) & 15) == 0;
  const dim3 grid((W * patch + TILE_X - 1) / TILE_X, (H * patch + TILE_Y - 1) / TILE_Y, B);
  cudaError_t e = cudaErrorInvalidValue;
#define HILO_SOBEL_CASE(PP, CC)                                                                         \
  if (patch == PP && C == CC)                                                                           \
    e = launch_pdl(sobel_tokmax_kernel<PP, CC>, grid, dim3(SOBEL_THREADS), 0, st, img, tokmax, tilemax, H, W, \
                   vec_ok);
  HILO_SOBEL_CASE(16, 1) HILO_SOBEL_CASE(16, 2) HILO_SOBEL_CASE(16, 3) HILO_SOBEL_CASE(16, 4)
  HILO_SOBEL_CASE(8, 1) HILO_SOBEL_CASE(8, 2) HILO_SOBEL_CASE(8, 3) HILO_SOBEL_CASE(8, 4)
#undef HILO_SOBEL_CASE
  if (e != cudaSuccess) return e;
  const dim3 kgrid((W + KEEP_T - 1) / KEEP_T, (H + KEEP_T - 1) / KEEP_T, B);
  auto* keep_kernel = KEEP_T + 2 * radius <= 32 ? sobel_keep_kernel<1> : sobel_keep_kernel<KEEP_WORDS>;
  return launch_pdl(keep_kernel, kgrid, dim3(KEEP_T * KEEP_T), KEEP_SMEM, st, static_cast<const float*>(tokmax),
                    static_cast<const uint32_t*>(tilemax), sobel_tiles(H, W, patch), mask, keep, H, W, radius,
                    threshold);
}

}  // namespace hilo
