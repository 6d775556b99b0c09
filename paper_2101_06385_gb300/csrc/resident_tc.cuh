// Tile geometry and the warp-level pieces that the resident tensor-core kernels
// share (csrc/resident.cu, csrc/resident_net.cu).
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace sp2 {
namespace res {

using namespace sp2::tc;

constexpr int TB = kResTile;                 // 128
constexpr int HALF_BYTES = TB * BK * 2;      // 16 KB: one plane of one operand
constexpr int T_BOX = 64 * 64 * 2;           // one 64 x 64 box of a transposed read
constexpr int STAGE_SPLIT = 4 * HALF_BYTES;  // hpA loA hpB loB
constexpr int STAGE_PLAIN = 2 * HALF_BYTES;  // hiA hiB
constexpr int STAGES_SPLIT = 3;
constexpr int STAGES_PLAIN = 6;
constexpr int OPERAND_BYTES = STAGES_SPLIT * STAGE_SPLIT;
static_assert(OPERAND_BYTES == STAGES_PLAIN * STAGE_PLAIN, "both precisions use the same shared memory");
constexpr int EPI_WARPS = 16;               // one 32 x 32 chunk each
constexpr int TR_BYTES = EPI_WARPS * 16 * 32 * 4;  // half a chunk per warp
constexpr int CTL_WARP = 2 + EPI_WARPS;
constexpr int THREADS = 32 * (CTL_WARP + 2);
constexpr uint32_t TMEM_COLS = 512;  // two slots of an accumulator and an iterate
constexpr uint32_t SLOT_COLS = 256, Y_COL = 128;
constexpr uint32_t IDESC_T = (1u << 4) | ((uint32_t)(TB >> 3) << 17) | ((uint32_t)(TB >> 4) << 24);
// Work queue entries.  A slot's next entry follows once all its epilogue warps have
// read the one before (they have stored its planes), so a slot has at most one entry
// that some warp has not read: two with both slots, a third in work, the end mark.
constexpr int WQ = 4;
constexpr int WQ_END = 255;

// Loads one 128-row operand of K block k0: K-major, or the stored block left
// of the diagonal transposed (two 64 x 64 boxes).
__device__ __forceinline__ void load_half(uint8_t* dst, const CUtensorMap* tmK, const CUtensorMap* tmT, bool trans,
                                          int row, int k0, int b, uint64_t* bar) {
  if (!trans) {
    tma_load_3d(dst, tmK, k0, row, b, bar);
  } else {
    tma_load_3d(dst, tmT, row, k0, b, bar);
    tma_load_3d(dst + T_BOX, tmT, row + 64, k0, b, bar);
  }
}

// Turns the warp's 32 x 32 chunk from one row per lane (v) to four consecutive
// columns of eight rows (p: register 4 i + e = row 4 i + lane / 8, column
// 4 (lane mod 8) + e), sixteen rows at a time through the warp's 2 KB.
template <class Sink>
__device__ __forceinline__ void turn(float* trb, const uint32_t (&v)[32], int lane, Sink sink) {
  const int r4 = lane >> 3, c4 = lane & 7;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if ((lane >> 4) == h) {
#pragma unroll
      for (int m = 0; m < 8; ++m)
        *epi::tr_at(trb, lane & 15, m) = make_float4(__uint_as_float(v[4 * m]), __uint_as_float(v[4 * m + 1]),
                                                     __uint_as_float(v[4 * m + 2]), __uint_as_float(v[4 * m + 3]));
    }
    __syncwarp();
#pragma unroll
    for (int i = 4 * h; i < 4 * h + 4; ++i) sink(i, *epi::tr_at(trb, 4 * (i - 4 * h) + r4, c4));
    __syncwarp();
  }
}

// The same from the accumulator's tensor memory, sixteen columns at a time: no
// more than sixteen registers of it at once (with all 32 a network's epilogue
// spilled, and the spills' stores, as many bytes as its planes, cost a fifth of
// a layer); before(h) runs ahead of the sinks of half h's rows.
template <class Before, class Sink>
__device__ __forceinline__ void turn_tmem(float* trb, uint32_t taddr, int lane, Before before, Sink sink) {
  const int r4 = lane >> 3, c4 = lane & 7;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      uint32_t v[16];
      __syncwarp();
      tmem_ld16(taddr + 16 * g, v);
      tmem_ld_wait();
      if ((lane >> 4) == h) {
#pragma unroll
        for (int m = 0; m < 4; ++m)
          *epi::tr_at(trb, lane & 15, 4 * g + m) =
              make_float4(__uint_as_float(v[4 * m]), __uint_as_float(v[4 * m + 1]), __uint_as_float(v[4 * m + 2]),
                          __uint_as_float(v[4 * m + 3]));
      }
    }
    before(h);
    __syncwarp();
#pragma unroll
    for (int i = 4 * h; i < 4 * h + 4; ++i) sink(i, *epi::tr_at(trb, 4 * (i - 4 * h) + r4, c4));
    __syncwarp();
  }
}

// (a - b) s by components, as two packed operations.
__device__ __forceinline__ float2 scaled_difference(float2 a, float2 b, float s) {
  float2 r;
  asm("{\n\t.reg .b64 x, y, z;\n\t"
      "mov.b64 x, {%2, %3};\n\t"
      "mov.b64 y, {%4, %5};\n\t"
      "mov.b64 z, {%6, %6};\n\t"
      "sub.rn.f32x2 x, x, y;\n\t"
      "mul.rn.f32x2 x, x, z;\n\t"
      "mov.b64 {%0, %1}, x;\n\t}\n"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(s));
  return r;
}

// Stores the operand planes of the chunk (Eq. 12: hp = 2^s fp16(x) and lo' =
// fp16(2^s (x - fp16(x))), finite where hp is not; plain FP16 keeps hi alone), four
// halves per plane and row; p0, p1 at the lane's first row and column, rows
// 4 i < rows_left.
template <bool SPLIT, class Put>
__device__ __forceinline__ void split_chunk(const float (&y)[32], float lo_scale, Put put) {
  const __half2 s2 = __float2half2_rn(lo_scale);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    uint32_t pa[2], pl[2] = {0u, 0u};
#pragma unroll
    for (int e2 = 0; e2 < 2; ++e2) {
      const float x0 = y[4 * i + 2 * e2], x1 = y[4 * i + 2 * e2 + 1];
      __half2 p2 = __floats2half2_rn(x0, x1);
      if (SPLIT) {
        const float2 hf = __half22float2(p2);
        const float2 lf = scaled_difference(make_float2(x0, x1), hf, lo_scale);
        const __half2 l2 = __floats2half2_rn(lf.x, lf.y);
        pl[e2] = *reinterpret_cast<const uint32_t*>(&l2);
        p2 = __hmul2(p2, s2);
      }
      pa[e2] = *reinterpret_cast<const uint32_t*>(&p2);
    }
    put(i, make_uint2(pa[0], pa[1]), make_uint2(pl[0], pl[1]));
  }
}

template <bool SPLIT>
__device__ __forceinline__ void store_planes(const float (&y)[32], __half* p0, __half* p1, long long ld_h,
                                             int rows_left, float lo_scale) {
  split_chunk<SPLIT>(y, lo_scale, [&](int i, uint2 a, uint2 l) {
    if (4 * i < rows_left) {
      *reinterpret_cast<uint2*>(p0) = a;
      if (SPLIT) *reinterpret_cast<uint2*>(p1) = l;
    }
    p0 += 4 * ld_h;
    if (SPLIT) p1 += 4 * ld_h;
  });
}

// The same into operand tiles in shared memory (128 rows of 128 bytes, 16-byte
// groups XOR-swizzled by row as a TMA load leaves them): t0 the tile of the
// chunk's K block, the second plane's HALF_BYTES after it; row, col: the lane's
// first row and column in the tile.
template <bool SPLIT>
__device__ __forceinline__ void store_planes_shared(const float (&y)[32], uint8_t* t0, int row, int col, int rows_left,
                                                    float lo_scale) {
  split_chunk<SPLIT>(y, lo_scale, [&](int i, uint2 a, uint2 l) {
    if (4 * i < rows_left) {
      const int r = row + 4 * i;
      uint8_t* p = t0 + r * 128 + ((((col >> 3) ^ r) & 7) << 4) + ((col & 4) << 1);
      *reinterpret_cast<uint2*>(p) = a;
      if (SPLIT) *reinterpret_cast<uint2*>(p + HALF_BYTES) = l;
    }
  });
}

// One row of an input matrix by one warp: y = y0(value, column) for each
// element, its operand planes (p0, p1 at the row's start) from column cs on up
// to the padded row length, and put(column, y) for every four columns.
// Returns the lane's part of the row's sum of squares in rownorm_kernel's order
// (vec_norm: its float4 form).
template <class Y0, class Put>
__device__ __forceinline__ double plane_row(const float* row, int N, bool vec_h, int vec_norm, Y0 y0, int cs,
                                            __half* p0, __half* p1, float lo_scale, int lane, Put put) {
  const int n4 = N >> 2, kpad = (N + 63) & ~63;
  double acc = 0.0;
  for (int j0 = 0; j0 < (kpad >> 2); j0 += 32 * 8) {
    float f = 0.f;
    float4 hv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int col = (j0 + u * 32 + lane) * 4;
      hv[u] = col < N ? epi::ld4(row + col, col, N, vec_h) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = j0 + u * 32 + lane, col = 4 * j;
      if (col < kpad) {
        float y[4] = {hv[u].x, hv[u].y, hv[u].z, hv[u].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) y[e] = col + e < N ? y0(y[e], col + e) : 0.f;
        if (j < n4) {
          f = fmaf(y[0], y[0], f);
          f = fmaf(y[1], y[1], f);
          f = fmaf(y[2], y[2], f);
          f = fmaf(y[3], y[3], f);
        }
        put(col, y);
        if (col >= cs) {
          uint32_t pa[2], pl[2];
          const __half2 s2 = __float2half2_rn(lo_scale);
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const __half2 h2 = __floats2half2_rn(y[2 * e], y[2 * e + 1]);
            const float2 hf = __half22float2(h2);
            const __half2 l2 = __floats2half2_rn((y[2 * e] - hf.x) * lo_scale, (y[2 * e + 1] - hf.y) * lo_scale);
            const __half2 q2 = p1 ? __hmul2(h2, s2) : h2;
            pa[e] = *reinterpret_cast<const uint32_t*>(&q2);
            pl[e] = *reinterpret_cast<const uint32_t*>(&l2);
          }
          *reinterpret_cast<uint2*>(p0 + col) = make_uint2(pa[0], pa[1]);
          if (p1) *reinterpret_cast<uint2*>(p1 + col) = make_uint2(pl[0], pl[1]);
        }
      }
    }
    if (vec_norm && j0 < n4) acc += (double)f;
  }
  // columns past the last float4, or every column in FP64 (rownorm_kernel's two tails)
  for (int j = (vec_norm ? n4 << 2 : 0) + lane; j < N; j += 32) {
    const double yv = (double)y0(row[j], j);
    acc += yv * yv;
  }
  return acc;
}

}  // namespace res
}  // namespace sp2
