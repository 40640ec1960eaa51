// Epilogue of the tcgen05 GEMM (gemm2_tc.cu): one warp turns accumulator
// columns of its TMEM lane quarter into output rows.
//
// The accumulator holds the tile transposed: its TMEM lanes are output
// features and its columns are rows of the row space. A warp's 32 lanes are
// therefore 32 consecutive features of one row at a time, the bias and the
// FP8 weight scale are one value per lane, and fp32 rows leave as whole
// 128-byte lines straight from registers: no staging in shared memory, which
// goes to a seventh ring stage instead.
//   fp32 += ...          one coalesced reduction per row (partial sums of a
//                        tile cut along K add up in whatever order they come)
//   fp32 = resid + ...   the residual rows are loaded one chunk ahead
//   bf16 / fp16          neighbouring lanes exchange one value of two rows, so
//                        that each lane stores two features of one row (a
//                        store instruction writes 64 bytes of two rows)
// A chunk of 32 rows takes a warp pair about 700 cycles, with a residual to load
// 1200, which the next tile's main loop hides except at the end of a launch.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"

namespace hilo {

// GELU in its tanh form, 0.5 z (1 + tanh(u)) with u = sqrt(2/pi) (z + 0.044715 z^3).
// Since 0.5 (1 + tanh(u)) = 1 / (1 + e^(-2u)), it is evaluated as
// z / (1 + 2^(-2u log2 e)): one exp2 and one division.
__device__ __forceinline__ float gelu_tanh(float z) {
  constexpr float k = 2.0f * 0.7978845608028654f * 1.4426950408889634f;  // 2 sqrt(2/pi) log2(e)
  const float t = z * fmaf(0.044715f * z, z, 1.0f);
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(-k * t));
  return __fdividef(z, 1.0f + e);
}

// One warp's 32 rows x 32 features of a tile.
struct EpiChunk {
  long long row;  // first row in the row space
  int nvalid;     // rows of the chunk inside the group: <= 32, may be <= 0
  int feat;       // this lane's output feature
};

// The residual of a chunk as it is in memory: fp32, rn[j] is this lane's
// feature of row j; bf16, rn[j] (even j) holds two neighbouring features of row
// j + (lane & 1), the even one in the low half.
__device__ __forceinline__ void epi_load_resid(const void* resid, bool f32, long long row, int nvalid, int feat,
                                               int N, uint32_t (&rn)[32]) {
  if (f32) {
    const uint32_t* src = static_cast<const uint32_t*>(resid) + row * N + feat;
    if (nvalid >= 32) {
#pragma unroll
      for (int j = 0; j < 32; ++j) rn[j] = __ldg(src + static_cast<long long>(j) * N);
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j) rn[j] = j < nvalid ? __ldg(src + static_cast<long long>(j) * N) : 0u;
    }
  } else {
    const int odd = lane_id() & 1;
    const uint32_t* src =
        reinterpret_cast<const uint32_t*>(static_cast<const uint16_t*>(resid) + (row + odd) * N + (feat & ~1));
    if (nvalid >= 32) {
#pragma unroll
      for (int j = 0; j < 32; j += 2) rn[j] = __ldg(src + static_cast<long long>(j >> 1) * N);
    } else {
#pragma unroll
      for (int j = 0; j < 32; j += 2) rn[j] = j + odd < nvalid ? __ldg(src + static_cast<long long>(j >> 1) * N) : 0u;
    }
  }
}

// v[j] = residual + v[j]
__device__ __forceinline__ void epi_add_resid(bool f32, const uint32_t (&rn)[32], float (&v)[32]) {
  if (f32) {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(rn[j]) + v[j];
  } else {
    const bool odd = lane_id() & 1;
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
      // own: (even, odd feature) of row j + odd; other: of row j + 1 - odd
      const uint32_t own = rn[j], other = __shfl_xor_sync(0xffffffffu, own, 1);
      const uint32_t r0 = odd ? other : own, r1 = odd ? own : other;
      v[j] = __uint_as_float(odd ? r0 & 0xFFFF0000u : r0 << 16) + v[j];
      v[j + 1] = __uint_as_float(odd ? r1 & 0xFFFF0000u : r1 << 16) + v[j + 1];
    }
  }
}

// 16-bit output rows: v[j] is feature c.feat of row j.
template <bool GELU>
__device__ __forceinline__ void epi_store16(void* out, int N, const EpiChunk& c, const float (&v)[32]) {
  const uint32_t odd = lane_id() & 1;
  const uint32_t sel = odd ? 0x3276u : 0x5410u;  // odd: (other.hi, own.hi); even: (own.lo, other.lo)
  uint32_t* dst = reinterpret_cast<uint32_t*>(static_cast<uint16_t*>(out) + (c.row + odd) * N + (c.feat & ~1));
  auto row2 = [&](int j) {
    const uint32_t own = GELU ? pack_f16x2_sat(gelu_tanh(v[j]), gelu_tanh(v[j + 1])) : pack_bf16x2(v[j], v[j + 1]);
    return __byte_perm(own, __shfl_xor_sync(0xffffffffu, own, 1), sel);
  };
  if (c.nvalid >= 32) {
#pragma unroll
    for (int j = 0; j < 32; j += 2) dst[static_cast<long long>(j >> 1) * N] = row2(j);
  } else {
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
      const uint32_t o = row2(j);
      if (j + static_cast<int>(odd) < c.nvalid) dst[static_cast<long long>(j >> 1) * N] = o;
    }
  }
}

// fp32 output rows: += (INPLACE) or =.
template <bool INPLACE>
__device__ __forceinline__ void epi_store32(void* out, int N, const EpiChunk& c, const float (&v)[32]) {
  float* dst = static_cast<float*>(out) + c.row * N + c.feat;
  auto put = [&](int j) {
    if (INPLACE)
      atomicAdd(dst + static_cast<long long>(j) * N, v[j]);
    else
      dst[static_cast<long long>(j) * N] = v[j];
  };
  if (c.nvalid >= 32) {
#pragma unroll
    for (int j = 0; j < 32; ++j) put(j);
  } else {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < c.nvalid) put(j);
  }
}

}  // namespace hilo
