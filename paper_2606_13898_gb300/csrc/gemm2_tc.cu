// Grouped GEMM of the MMDiT block's linear layers (paper Sec. 2.1, the DiT's
// QKV, output and MLP projections) on the 5th-generation tensor cores:
//   C[r, n] = sum_k X[r, k] * W_g[n, k] + b_g[n]
// with the text rows (group 0) and the packed image rows (group 1) of the row
// space using their own weights. The image row count is read on the device,
// so no host synchronisation is needed between split and block.
//
// CTA pairs (tcgen05 cta_group::2), transposed tiles: the MMA's 256 rows (M)
// are output features and its columns (N) are rows of the row space, 32 to 256
// of them in steps of 32. Features come in multiples of 128, so M wastes
// little, while the row counts are whatever the selection left: with the rows
// on N a group is cut into tiles of nearly equal height, and the tiles of the
// last, partial round are cut again, so that they reach every pair (Plan).
// Bound by the tensor pipe at the chip's power limit for large row counts, by
// fill, last epilogue and partial rounds for small ones. (With rows on M, 256 to
// a tile, and one-CTA tiles for widths that 256 does not divide, a block of 1662
// rows of 1152 took 127 us, 91 so; 2389 rows of 3072 458 and 440, with e4m3
// operands 323 and 295; 10600 rows 2023 and 1969.)
//
// Each CTA of a pair stages 128 rows of W (half of the tile's features) and
// half of the tile's X rows at identical shared-memory offsets; the even CTA
// issues the MMAs, which read both CTAs' halves.
//
// Per CTA, 320 threads:
//   warp 0     TMA producer: W half, X half (as up to three boxes of 128, 64,
//              32 and 16 rows); the completion of both CTAs' copies is counted
//              on the even CTA's "full" barrier
//   warp 1     TMEM allocation (both CTAs); MMA issue (even CTA only): the
//              whole warp walks the schedule and waits, one elected lane issues
//   warps 2-9  epilogue over this CTA's 128 features x the tile's rows, two
//              warps per TMEM lane quarter, 32-row chunks alternating
// "empty" and "accumulator ready" barriers are signalled in both CTAs by a
// multicast commit; "accumulator free" collects 16 arrivals (8 epilogue warps
// x 2 CTAs) in the even CTA. Every wait is bounded.
//
// FP8 (e4m3 X and W, kind::f8f6f4): a k-block is the same 128-byte swizzled
// row of shared memory holding 128 elements instead of 64, and each MMA
// consumes 32 of them; the epilogue multiplies each accumulator by its row's
// X scale and its feature's W scale before the bias.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "gemm_epi.cuh"
#include "internal.h"

namespace hilo {

__device__ int g_gemm_err;

namespace {

constexpr int PF = 256;   // features per pair tile (128 of W staged per CTA)
constexpr int UNIT = 32;  // rows of a tile come in units of 32 ...
constexpr int MAXU = 8;   // ... at most 256
constexpr int BK = 64;
constexpr int STAGES = 7;
constexpr int HALF_BYTES = 128 * BK * 2;    // 16 KB: one CTA's W slice, or its largest X slice
constexpr int STAGE_BYTES = 2 * HALF_BYTES; // W + X slices of this CTA
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 32 * (2 + EPI_WARPS);
constexpr uint32_t TMEM_COLS = 512;         // two 128 x 256 fp32 accumulators
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
constexpr int SPLIT_MIN_KB = 16;            // shortest piece of a tile cut along K
// the plan's costs in SM cycles beside those of the k-blocks
constexpr float TILE_CYC = 400.f;           // going from one tile to the next
constexpr float EPI_CYC = 700.f;            // the last epilogue, per 32 rows
constexpr float EPI_RESID_CYC = 1200.f;     // the same with a residual to load
// where K is short (up to SHORT_K) and epilogues follow one another: a latency per tile
constexpr int SHORT_K = 512;
constexpr float SHORT_CYC = 2800.f;
constexpr float SHORT_RESID_CYC = 3500.f;
constexpr float PIECE_CYC = 300.f;           // a K piece's reductions, per 32 rows

struct Maps {
  CUtensorMap x[4];  // boxes of 128, 64, 32, 16 rows
  CUtensorMap w[2];
};

struct Params {
  int N, K;
  uint32_t idesc;           // without the N field
  const float* a_scale;     // FP8: dequantisation scale per row of X (row space)
  const float* b_scale[2];  // FP8: per output feature, per weight group
  int row_base[2];
  int rows_static[2];
  const int32_t* rows_dev[2];
  const __nv_bfloat16* bias[2];
  int epilogue;
  void* out;
  const void* resid_src[2];
  int resid_f32;
  // for the plan, by epilogue and K: cycles of 32 rows in the last epilogue; with short
  // K the latency of an epilogue and its 32 rows, else 0 and 0; 0 with short K, else far
  // more than any main loop takes
  float epi_cyc, short_cyc, short_epi_cyc, long_k;
};

// One unit of a pair's work: k-blocks [k0, k1) of piece `part` of `parts` (cut by
// rows) of tile t.
struct Work {
  int t, k0, k1, part, parts;
};

// Rows [r0, r0 + 32 units) of group g (of `rows` valid ones), feature block f.
struct Tile {
  int g, f, r0, units, rows, row_base;
};

// How the rows are cut and the tiles dealt; every role of every CTA computes
// the same plan from the same row counts.
struct Plan {
  int rows0, rows1, U0, U1;  // rows and 32-row units per group
  int t0, t1;                // row tiles per group
  int total;                 // tiles
  int whole;                 // tiles dealt whole; the rest are cut
  int nsplit;                // pieces per cut tile
  int kcut;                  // cut along K (else by rows)

  // Cycles of one k-block of a tile of x units. The MMAs take 64 x, but every
  // byte of W and X is written to shared memory once and read once, at 128 bytes
  // a cycle: 2 (16 KB + 2 KB x) / 128 = 256 + 32 x, plus 6% as measured (520,
  // 511, 480 and 427 cycles at x = 8, 7, 6 and 4). So a tile of 256 rows runs at
  // the MMA rate and a lower one loses what it saves in columns.
  __device__ static float kblock(float x) { return 272.0f + 34.0f * x; }

  // Chosen by cost: lane l tries image tiles of at most u1 = 8 - l % 8 units (and
  // text tiles of at most two more), whole or with the tiles left over after the last
  // full round cut into 2 to 8 pieces, by rows or (see below) along K, of which
  // lane l takes the counts 1 + l / 8 and 5 + l / 8; the cheapest wins, the higher
  // tile and the fewer pieces among equals. The cost is that of pair 0, which has the
  // most tiles: its rounds of whole tiles, its pieces, and the epilogue that nothing
  // hides. Up to K = 512 the epilogues take longer than the main loops: a round costs
  // the longer of the two, and the epilogue has a latency of its own per tile. (Priced
  // like longer K, short K was cut into many small pieces: at K = 128, 384 features of
  // 2389 rows took 7.8 us, 5.8 so, of 4096 rows 7.2 and 6.1; at K = 512, 1536 features
  // of 2389 rows 10.5 and 8.9. At 640 and 768 that price was 27% worse for some shapes
  // and 11% better for others.) Called by whole warps. Every cycle here is one before
  // the first product wherever the previous kernel held the SM to its end.
  //
  // A K cut costs the call its bitwise repeatability: the pieces' partial sums meet
  // in whatever order they come. So only calls of many tiles make one, as hilo.h
  // says: widths that are a multiple of 256 from 1024 on, more tiles of 256 x 256
  // than pairs, and the last round of those a partial one. (K cuts at fewer rows are
  // faster: a block of 777 rows of 1024 channels took 60.4 us, 66.4 without; of 300 rows
  // 46.8 and 54.6. Added up in order, through scratch and a counter per tile, they
  // took 61 to 72 and 53.)
  __device__ void init(const Params& p, int dev0, int dev1, int ncl, int kb) {
    const float EPI = p.epi_cyc;
    // a device row count is bounded by the group's capacity (rows_static)
    rows0 = max(0, p.rows_dev[0] ? min(dev0, p.rows_static[0]) : p.rows_static[0]);
    rows1 = max(0, p.rows_dev[1] ? min(dev1, p.rows_static[1]) : p.rows_static[1]);
    U0 = (rows0 + UNIT - 1) / UNIT;
    U1 = (rows1 + UNIT - 1) / UNIT;
    const int F = (p.N + PF - 1) / PF;
    const int full = F * ((U0 + MAXU - 1) / MAXU + (U1 + MAXU - 1) / MAXU);  // tiles of 256 x 256
    const bool split = p.epilogue == EPI_BIAS_RESID_F32 && p.N >= 1024 && p.N % PF == 0 && full > ncl && full % ncl != 0;
    const int lane = lane_id();
    const int u1 = MAXU - (lane & 7), u0 = min(MAXU, u1 + 2);
    const int a0 = (U0 + u0 - 1) / u0, a1 = (U1 + u1 - 1) / u1;
    const int T0 = F * a0, T = F * (a0 + a1);
    const float x0 = a0 ? __fdividef(U0, a0) : 0.f, x1 = a1 ? __fdividef(U1, a1) : 0.f;
    const float xm = fmaxf(x0, x1);
    // no tile has fewer units than its group's floor(U / a), so it can be cut into as
    // many pieces (the quotient is checked: a piece must not be empty)
    auto least_of = [](int U, int a, float x) {
      const int q = static_cast<int>(x + 1e-3f);
      return a == 0 ? MAXU : (q * a <= U ? q : q - 1);
    };
    const int least = min(least_of(U0, a0, x0), least_of(U1, a1, x1));
    const float kbf = static_cast<float>(kb);
    auto loop_of = [&](float x) { return kbf * kblock(x) + TILE_CYC; };
    auto tile_of = [&](float x) { return fmaxf(loop_of(x), p.short_cyc + p.short_epi_cyc * x); };
    auto tail_of = [&](float x) { return fminf(loop_of(x) + p.long_k, p.short_cyc + EPI * x); };
    const float c0 = tile_of(x0), c1 = tile_of(x1);
    // ceil(n / ncl) for the small counts here (n + 0.5 keeps the product away
    // from the whole numbers)
    const float inv = __fdividef(1.0f, static_cast<float>(ncl));
    auto rounds_of = [&](int n) { return static_cast<int>((static_cast<float>(n + ncl - 1) + 0.5f) * inv); };
    const int g_max = rounds_of(T0), rounds = rounds_of(T);
    auto rounds_cost = [&](int n) {
      const int g0 = min(n, g_max);
      return g0 * c0 + (n - g0) * c1;
    };
    const int rem = T > 0 && rounds * ncl != T ? T - (rounds - 1) * ncl : 0;  // of a partial last round
    float best = rounds_cost(rounds) + tail_of(xm);
    int best_s = 1, best_k = 0;
    const float c_full = rounds_cost(rounds - 1);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int s = 1 + (lane >> 3) + 4 * j;
      if (s == 1 || rem == 0) continue;
      const float n = static_cast<float>(rounds_of(rem * s)), sf = static_cast<float>(s);
      const float xs = ceilf(__fdividef(xm, sf) - 1e-3f), ks = ceilf(__fdividef(kbf, sf) - 1e-3f);
      const float cr = c_full + n * tile_of(xs) + tail_of(xs);
      if (s <= least && cr < best) best = cr, best_s = s, best_k = 0;
      const float ck = c_full + n * (ks * kblock(xm) + TILE_CYC + PIECE_CYC * xm) + EPI * xm;
      if (split && kb >= s * SPLIT_MIN_KB && ck < best) best = ck, best_s = s, best_k = 1;
    }
    // costs are positive, so their bit patterns order like the values
    const uint32_t key = __float_as_uint(best);
    const uint32_t lo = __reduce_min_sync(0xffffffffu, key);
    const int win = __ffs(__ballot_sync(0xffffffffu, key == lo)) - 1;
    t0 = __shfl_sync(0xffffffffu, a0, win);
    t1 = __shfl_sync(0xffffffffu, a1, win);
    nsplit = __shfl_sync(0xffffffffu, best_s, win);
    kcut = __shfl_sync(0xffffffffu, best_k, win);
    total = F * (t0 + t1);
    // exact, whatever the estimates above were rounded to
    whole = nsplit > 1 ? total - total % ncl : total;
  }

  // (i U + o) / n, the first unit of row tile i of n
  __device__ static int cut(int i, int U, int n, int o) {
    const int base = U / n, more = U - base * n;
    return i * base + (n <= 32768 ? (i * more + o) / n
                                  : static_cast<int>((static_cast<long long>(i) * more + o) / n));
  }

  // Row tiles vary fastest, so that the pairs running at one time share W. A
  // group's units are dealt to its row tiles as evenly as they go; which tiles
  // get the odd unit turns with the feature block, so that no pair collects
  // only the higher ones.
  __device__ Tile get(const Params& p, const Work& w) const {
    int t = w.t;
    const int T0 = total / (t0 + t1) * t0;
    Tile r;
    r.g = t < T0 ? 0 : 1;
    if (r.g) t -= T0;
    const int n = r.g ? t1 : t0, U = r.g ? U1 : U0;
    r.f = t / n;
    const int i = t - r.f * n;
    int b0 = cut(i, U, n, r.f % n), b1 = cut(i + 1, U, n, r.f % n);
    if (w.parts > 1) {
      const int x = b1 - b0;
      b1 = b0 + (w.part + 1) * x / w.parts;
      b0 += w.part * x / w.parts;
    }
    r.r0 = b0 * UNIT;
    r.units = b1 - b0;
    r.rows = r.g ? rows1 : rows0;
    r.row_base = r.g ? p.row_base[1] : p.row_base[0];
    return r;
  }
};

// The work of pair `cid` of `ncl`: whole tiles round-robin, then the pieces of
// the remaining ones, dealt piece-major: K pieces that run at the same time
// cover one or two K ranges, so the pairs share those slices of X and W in L2
// even when X and W together exceed it. Each K piece adds its partial sum to
// the output (fp32 += only); the one that starts at k = 0 adds the bias.
struct WorkIter {
  int t, whole, rem, nsplit, kcut, ncl, kb, u;
  __device__ WorkIter(const Plan& pl, int cid, int ncl_, int kblocks)
      : t(cid), whole(pl.whole), rem(pl.total - pl.whole), nsplit(pl.nsplit), kcut(pl.kcut), ncl(ncl_), kb(kblocks),
        u(cid) {}
  __device__ bool next(Work& w) {
    w.k0 = 0;
    w.k1 = kb;
    w.part = 0;
    w.parts = 1;
    if (t < whole) {
      w.t = t;
      t += ncl;
      return true;
    }
    if (u >= rem * nsplit) return false;
    const int s = u / rem;  // piece index
    w.t = whole + (u - s * rem);
    if (kcut) {
      w.k0 = s * kb / nsplit;
      w.k1 = (s + 1) * kb / nsplit;
    } else {
      w.part = s;
      w.parts = nsplit;
    }
    u += ncl;
    return true;
  }
};

template <bool FP8>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    gemm2_kernel(const __grid_constant__ Maps tm, const __grid_constant__ Params p) {
  // elements per k-block: one 128-byte swizzled row of X / W
  constexpr int BKE = FP8 ? 128 : BK;
  extern __shared__ unsigned char smem_raw[];
  // (an offset from smem_raw, so that accesses stay 32-bit shared-memory ones)
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* err = &g_gemm_err;

  const int warp = warp_id(), lane = lane_id();
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int cid = blockIdx.x >> 1;
  const int ncl = gridDim.x >> 1;

  // The row counts and the weights were there before the previous kernel
  // started: the plan is made, and this pair's first W slices are on their way,
  // while that kernel finishes. Only X, the residual and the outputs wait for it.
  const int dev0 = p.rows_dev[0] ? ld_l2(p.rows_dev[0]) : 0, dev1 = p.rows_dev[1] ? ld_l2(p.rows_dev[1]) : 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], 2 * EPI_WARPS);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane < 6) tma_prefetch_desc(lane < 4 ? &tm.x[lane] : &tm.w[lane - 4]);
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, TMEM_COLS);
    tmem_relinquish_pair();
  }
  const int kblocks = p.K / BKE;
  Plan pl;
  pl.init(p, dev0, dev1, ncl, kblocks);
  WorkIter it(pl, cid, ncl, kblocks);
  Work w;
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers are initialised before any remote use
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    // ---------------- TMA producer (both CTAs): the whole warp walks the
    // schedule, one elected lane issues
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    uint32_t armed = 0, armed_par = 0;  // per stage: armed at least once, parity of the last arming
    bool ok = true;
    const uint32_t full0 = mapa_shared(smem_u32(full), 0);
    bool first = true;
    while (ok && it.next(w)) {
      const Tile tl = pl.get(p, w);
      const CUtensorMap* mw = tl.g ? &tm.w[1] : &tm.w[0];
      const int yw = tl.f * PF + 128 * static_cast<int>(rank);
      const int yx = tl.row_base + tl.r0 + static_cast<int>(rank) * tl.units * 16;
      const uint32_t bytes = 2u * (HALF_BYTES + static_cast<uint32_t>(tl.units) * 16 * 128);
      auto load_w = [&](int st, int kb) {
        if (leader) mbar_arrive_expect_tx(&full[st], bytes);
        tma_load_2d_pair(smem + st * STAGE_BYTES, mw, full0 + 8u * static_cast<uint32_t>(st), kb * BKE, yw);
      };
      auto load_x = [&](int st, int kb) {
        unsigned char* dst = smem + st * STAGE_BYTES + HALF_BYTES;
        int y = yx;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (tl.units & (8 >> i)) {
            tma_load_2d_pair(dst, &tm.x[i], full0 + 8u * static_cast<uint32_t>(st), kb * BKE, y);
            dst += (128 >> i) * 128;
            y += 128 >> i;
          }
      };
      int kb = w.k0;
      if (first) {
        // the ring is empty: W of its first stages before the wait, X after it
        first = false;
        const int n = min(STAGES, w.k1 - w.k0);
        if (issuer)
          for (int i = 0; i < n; ++i) load_w(i, w.k0 + i);
        pdl_wait();
        if (issuer)
          for (int i = 0; i < n; ++i) load_x(i, w.k0 + i);
        __syncwarp();
        armed = (1u << n) - 1u;  // every parity is still 0
        kb += n;
        stage = n == STAGES ? 0 : n;
        phase = n == STAGES ? 1u : 0u;
      }
      for (; kb < w.k1; ++kb) {
        if (!mbar_wait_warp(&empty[stage], phase ^ 1u, abort_flag, err, DEV_TIMEOUT_GEMM + 256 * 1)) {
          ok = false;
          break;
        }
        if (issuer) {
          load_w(stage, kb);
          load_x(stage, kb);
        }
        __syncwarp();
        armed |= 1u << stage;
        armed_par = (armed_par & ~(1u << stage)) | (phase << stage);
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok) {
      // let the bulk copies already issued land before the CTA can exit
      const uint64_t tw = globaltimer_ns();
      if (leader) {
        for (int s = 0; s < STAGES; ++s) {
          if (!((armed >> s) & 1u)) continue;
          while (!mbar_try_wait(smem_u32(&full[s]), (armed_par >> s) & 1u) &&
                 globaltimer_ns() - tw < HILO_WAIT_LIMIT_NS / 4) {
          }
        }
      } else {
        while (globaltimer_ns() - tw < 50000ull) {
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (leader) {
      // ---------------- MMA issuer (even CTA)
      const bool issuer = elect_one();
      const uint32_t w_lo = (smem_u32(smem) >> 4) + sw128_lo_lbo(16);
      constexpr uint32_t hi = sw128_hi(1024);
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      // X comes after the previous kernel's end anyway; the limit of the waits
      // below is for this kernel's own work
      pdl_wait();
      while (ok && it.next(w)) {
        const uint32_t idesc = p.idesc | (static_cast<uint32_t>(pl.get(p, w).units * (UNIT / 8)) << 17);
        if (!mbar_wait_warp(&tempty[acc], acc_phase ^ 1u, abort_flag, err, DEV_TIMEOUT_GEMM + 256 * 2)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem + static_cast<uint32_t>(acc * UNIT * MAXU);
        for (int kb = w.k0; kb < w.k1; ++kb) {
          if (!mbar_wait_warp(&full[stage], phase, abort_flag, err, DEV_TIMEOUT_GEMM + 256 * 3)) {
            ok = false;
            break;
          }
          tc_fence_after();
          if (issuer) {
            const uint32_t a = w_lo + static_cast<uint32_t>(stage) * (STAGE_BYTES >> 4);
            const uint32_t b = a + (HALF_BYTES >> 4);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              umma_pair_w<FP8>(d_tmem, a + 2 * k, b + 2 * k, hi, idesc, (kb > w.k0 || k > 0) ? 1u : 0u);
            umma_commit_pair(&empty[stage], 0x3);
          }
          __syncwarp();
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        if (issuer) umma_commit_pair(&tfull[acc], 0x3);
        __syncwarp();
        acc ^= 1;
        if (acc == 0) acc_phase ^= 1u;
      }
      if (issuer) umma_commit_pair(drain, 0x1);
      __syncwarp();
      const uint64_t tw = globaltimer_ns();
      while (!mbar_try_wait(smem_u32(drain), 0u)) {
        if (globaltimer_ns() - tw > HILO_WAIT_LIMIT_NS) {
          if (issuer) atomicExch(err, DEV_TIMEOUT_GEMM + 256 * 4);
          break;
        }
      }
      __syncwarp();
    }
  } else {
    // ---------------- epilogue, both CTAs: TMEM lane quarter warp % 4, the
    // even or the odd 32-row chunks
    const int q = warp & 3, half = (warp - 2) >> 2;
    const int N = p.N, epi = p.epilogue;
    const bool resid_f32 = p.resid_f32 != 0;
    int acc = 0;
    uint32_t acc_phase = 0;
    pdl_wait();
    pdl_trigger();
    while (it.next(w)) {
      const Tile tl = pl.get(p, w);
      EpiChunk ch;
      ch.feat = tl.f * PF + 128 * static_cast<int>(rank) + q * 32 + lane;
      const bool on = ch.feat < N;  // N is a multiple of 128: the same for the whole warp
      // the bias is added once per tile, by the piece that starts at k = 0
      const float bias = on && w.k0 == 0 ? __bfloat162float(__ldg((tl.g ? p.bias[1] : p.bias[0]) + ch.feat)) : 0.f;
      const float wscale = FP8 && on ? __ldg((tl.g ? p.b_scale[1] : p.b_scale[0]) + ch.feat) : 1.f;
      const void* resid = tl.g ? p.resid_src[1] : p.resid_src[0];
      uint32_t rn[32];
      const bool with_resid = epi == EPI_BIAS_RESIDIN_F32 && on;
      if (with_resid) {
        // this warp's residual rows into L2 while the accumulator is still
        // being computed, and the first chunk of them into registers
        const int esz = resid_f32 ? 4 : 2;
        for (int c = half + 2; c < tl.units; c += 2) {
          const int r = tl.r0 + c * UNIT + lane;
          if (r < tl.rows)
            prefetch_l2(static_cast<const char*>(resid) + (static_cast<long long>(r) * N + (ch.feat - lane)) * esz);
        }
        const int r = tl.r0 + half * UNIT;
        epi_load_resid(resid, resid_f32, r, half < tl.units ? tl.rows - r : 0, ch.feat, N, rn);
      }
      // FP8: lane r's row scale of each of this warp's chunks
      float rscale[MAXU / 2];
      if (FP8) {
#pragma unroll
        for (int k = 0; k < MAXU / 2; ++k) {
          const int r = tl.r0 + (half + 2 * k) * UNIT + lane;
          rscale[k] = half + 2 * k < tl.units && r < tl.rows ? __ldg(p.a_scale + tl.row_base + r) : 0.f;
        }
      }
      if (!mbar_wait_warp(&tfull[acc], acc_phase, abort_flag, err, DEV_TIMEOUT_GEMM + 256 * 5)) break;
      tc_fence_after();
      const uint32_t taddr =
          tmem + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(acc * UNIT * MAXU);
#pragma unroll 1
      for (int c = half; c < tl.units; c += 2) {
        float v[32];
        tmem_ld32(taddr + c * UNIT, v);
        const int r = tl.r0 + c * UNIT;
        uint32_t rc[32];
        if (with_resid) {
#pragma unroll
          for (int j = 0; j < 32; ++j) rc[j] = rn[j];
          if (c + 2 < tl.units)
            epi_load_resid(resid, resid_f32, r + 2 * UNIT, tl.rows - (r + 2 * UNIT), ch.feat, N, rn);
          __syncwarp();  // a ragged chunk is loaded by some lanes only; the TMEM wait below is for all
        }
        ch.nvalid = min(UNIT, tl.rows - r);
        ch.row = tl.row_base + r;
        tmem_ld_wait_regs(v);
        if (c + 2 >= tl.units) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(mapa_shared(smem_u32(&tempty[acc]), 0));
        }
        if (!on) continue;
        if (FP8) {
          float rs = rscale[0];  // of this chunk (selected: no runtime-indexed array)
#pragma unroll
          for (int k = 1; k < MAXU / 2; ++k) rs = c == half + 2 * k ? rscale[k] : rs;
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] *= __shfl_sync(0xffffffffu, rs, j) * wscale;
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] += bias;
        if (epi == EPI_BIAS_GELU_F16) {
          epi_store16<true>(p.out, N, ch, v);
        } else if (epi == EPI_BIAS_BF16) {
          epi_store16<false>(p.out, N, ch, v);
        } else if (epi == EPI_BIAS_RESID_F32) {
          epi_store32<true>(p.out, N, ch, v);
        } else {
          epi_add_resid(resid_f32, rc, v);
          epi_store32<false>(p.out, N, ch, v);
        }
      }
      if (half >= tl.units) {  // a one-unit tile has no chunk for this warp
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(mapa_shared(smem_u32(&tempty[acc]), 0));
      }
      acc ^= 1;
      if (acc == 0) acc_phase ^= 1u;
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();  // no remote arrivals / copies into the peer after this point
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, TMEM_COLS);
  }
}

}  // namespace

// CTA pairs of one kernel that the current device holds at a time.
template <bool FP8>
static int resident_pairs(int device, int num_sms) {
  static PerDevice pairs;
  const int n = pairs.get(device, [&] {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (num_sms / 2), 1, 1);
    cfg.blockDim = dim3(THREADS, 1, 1);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int found = 0;
    if (cudaOccupancyMaxActiveClusters(&found, gemm2_kernel<FP8>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      found = 0;
    }
    return found;
  });
  return n > 0 ? n : num_sms / 2;
}

cudaError_t launch_gemm(const GemmArgs& a, int device, int num_sms, cudaStream_t st) {
  // FP8: bytes are the elements, 128 per swizzled row
  const TmapType tt = a.fp8 ? TMAP_U8 : TMAP_BF16;
  const uint32_t bk = a.fp8 ? 128 : BK;
  if (a.K % bk != 0 || a.N % 128 != 0) return cudaErrorInvalidValue;
  Maps m;
  for (int i = 0; i < 4; ++i)
    if (!encode_tmap_2d(&m.x[i], tt, a.A, a.K, a.R, a.K, bk, 128u >> i)) return cudaErrorInvalidValue;
  for (int g = 0; g < 2; ++g) {
    const void* wg = a.g[g].weight ? a.g[g].weight : a.g[1 - g].weight;
    if (!encode_tmap_2d(&m.w[g], tt, wg, a.K, a.N, a.K, bk, 128)) return cudaErrorInvalidValue;
  }
  Params p;
  p.N = a.N;
  p.K = a.K;
  // format code 0: fp16 for kind::f16, E4M3 for kind::f8f6f4; the N field is set per tile
  p.idesc = idesc_kind_f16(PF, 0, 0, 0, (a.op_f16 || a.fp8) ? 0 : 1);
  p.a_scale = a.a_scale;
  long long units = 0;
  for (int g = 0; g < 2; ++g) {
    p.b_scale[g] = a.g[g].w_scale;
    p.row_base[g] = a.g[g].row_base;
    p.rows_static[g] = a.g[g].rows_dev ? a.g[g].rows_cap : a.g[g].rows_static;
    p.rows_dev[g] = a.g[g].rows_dev;
    p.bias[g] = static_cast<const __nv_bfloat16*>(a.g[g].bias);
    p.resid_src[g] = a.resid_src[g];
    units += (a.g[g].rows_cap + UNIT - 1) / UNIT;
  }
  p.epilogue = a.epilogue;
  p.out = a.out;
  p.resid_f32 = a.resid_f32;
  const bool resid = a.epilogue == EPI_BIAS_RESIDIN_F32, short_k = a.K <= SHORT_K;
  p.epi_cyc = resid ? EPI_RESID_CYC : EPI_CYC;
  p.short_cyc = short_k ? (resid ? SHORT_RESID_CYC : SHORT_CYC) : 0.f;
  p.short_epi_cyc = short_k ? p.epi_cyc : 0.f;
  p.long_k = short_k ? 0.f : 1e30f;
  if (units <= 0) return cudaSuccess;
  auto* kern = a.fp8 ? gemm2_kernel<true> : gemm2_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
  if (e != cudaSuccess) return e;
  // persistent grid: as many co-resident CTA pairs as the device holds
  const int pairs = a.fp8 ? resident_pairs<true>(device, num_sms) : resident_pairs<false>(device, num_sms);
  return launch_pdl(kern, dim3(2 * pairs), dim3(THREADS), SMEM_BYTES, st, m, p);
}

int gemm_take_device_error() {
  int v = 0, z = 0;
  if (cudaMemcpyFromSymbol(&v, g_gemm_err, sizeof(int)) != cudaSuccess) return -1;
  if (v) cudaMemcpyToSymbol(g_gemm_err, &z, sizeof(int));
  return v;
}

}  // namespace hilo
