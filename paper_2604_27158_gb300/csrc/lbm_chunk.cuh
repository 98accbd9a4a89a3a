// Four cells a lane: the gather of the pull for kernels that read a state once (moments, state
// copies, the adjoint seed, vorticity).  A warp owns a row segment of 128 columns, a lane one aligned
// chunk of four cells; the +-1 column shifts are shuffles, the solid bits of a chunk and its
// neighbours one 6-bit window a row.  Against one cell a thread (nine 4-byte loads and nine mask
// words, each with its own 64-bit address) the moments of 64 grids of 512 x 256 took 198 us, and
// HBM needs 59.
#pragma once

#include "common.cuh"
#include "lbm_cell.cuh"

namespace lbmfno {

constexpr int kChunkRows = 4;  // rows (warps) of a block: a tile of the step-kernel table

// This lane's chunk: grid, first column, row; false for lanes beyond the row (they still take
// part in the shuffles) and warps beyond the tile.
struct ChunkAt {
  int grid, x, y;
  bool row, active;
};
__device__ __forceinline__ ChunkAt chunk_of_lane(const GridDev* __restrict__ grids,
                                                 const int4* __restrict__ tiles) {
  const int4 t = __ldg(&tiles[blockIdx.x]);  // (grid, x0, y0, rows)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  ChunkAt c;
  c.grid = t.x;
  c.x = t.y + 4 * lane;
  c.y = t.z + warp;
  c.row = warp < t.w;
  c.active = c.row && c.x < __ldg(&grids[t.x].nx);
  return c;
}

// Solid bits of cells x - 1 .. x + 4 of mask row mr (bit b: cell x - 1 + b); wrapped for periodic
// rows, 0 beyond an open end.
__device__ __forceinline__ uint32_t chunk_window(const uint32_t* __restrict__ mr, const GridDev& G,
                                                 int x) {
  const int wi = x >> 5, sh = x & 31;
  uint64_t v = (uint64_t)__ldg(mr + wi) << 1;
  if (sh == 0 && wi > 0) v |= __ldg(mr + wi - 1) >> 31;
  if (sh == 28 && wi + 1 < G.wpr) v |= (uint64_t)(__ldg(mr + wi + 1) & 1u) << 33;
  uint32_t win = (uint32_t)(v >> sh) & 0x3fu;
  if (x == 0) {
    win &= ~1u;
    if (G.periodic_x) win |= (__ldg(mr + ((G.nx - 1) >> 5)) >> ((G.nx - 1) & 31)) & 1u;
  }
  const int jw = G.nx - 1 - x;
  if (jw < 4) {
    win &= ~(1u << (jw + 2));
    if (G.periodic_x) win |= (__ldg(mr) & 1u) << (jw + 2);
  }
  return win;
}
// Windows of rows y - 1, y, y + 1.
__device__ __forceinline__ void chunk_windows(const uint32_t* __restrict__ m, const GridDev& G,
                                              const ChunkAt& at, uint32_t win[3]) {
  const int ym = at.y == 0 ? G.ny - 1 : at.y - 1, yp = at.y == G.ny - 1 ? 0 : at.y + 1;
  win[0] = win[1] = win[2] = 0u;
  if (at.active) {
    win[0] = chunk_window(m + (size_t)ym * G.wpr, G, at.x);
    win[1] = chunk_window(m + (size_t)at.y * G.wpr, G, at.x);
    win[2] = chunk_window(m + (size_t)yp * G.wpr, G, at.x);
  }
}

__device__ __forceinline__ float4 ld4(const float* p) {
  return __ldg(reinterpret_cast<const float4*>(p));
}
// Cells x + s .. x + s + 3 of a row (s = -1, 0 or 1), wrapped for periodic rows, 0 beyond an open
// end.  Called by every lane of the warp; row + x is 16-byte aligned.
template <int S>
__device__ __forceinline__ void chunk_shifted(const float* __restrict__ row, const GridDev& G,
                                              const ChunkAt& at, float v[4]) {
  const int lane = threadIdx.x & 31;
  const float4 c = at.active ? ld4(row + at.x) : make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (S == 0) {
    v[0] = c.x;
    v[1] = c.y;
    v[2] = c.z;
    v[3] = c.w;
  } else if constexpr (S < 0) {
    float l = __shfl_up_sync(0xffffffffu, c.w, 1);
    if (at.active && at.x == 0)
      l = G.periodic_x ? __ldg(row + G.nx - 1) : 0.0f;
    else if (at.active && lane == 0)
      l = __ldg(row + at.x - 1);
    v[0] = l;
    v[1] = c.x;
    v[2] = c.y;
    v[3] = c.z;
  } else {
    float r = __shfl_down_sync(0xffffffffu, c.x, 1);
    if (at.active && lane == 31 && at.x + 4 < G.nx) r = __ldg(row + at.x + 4);
    v[0] = c.y;
    v[1] = c.z;
    v[2] = c.w;
    v[3] = r;
    const int jw = G.nx - 1 - at.x;
    if (at.active && jw < 4) {
      const float w = G.periodic_x ? __ldg(row) : 0.0f;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j == jw) v[j] = w;
    }
  }
}
__device__ __forceinline__ void chunk_shifted(int s, const float* row, const GridDev& G,
                                              const ChunkAt& at, float v[4]) {
  if (s < 0)
    chunk_shifted<-1>(row, G, at, v);
  else if (s == 0)
    chunk_shifted<0>(row, G, at, v);
  else
    chunk_shifted<1>(row, G, at, v);
}
// where bit j of `bits` is set, v[j] = own[j] (a chunk at a 16-byte aligned address)
__device__ __forceinline__ void chunk_select(uint32_t bits, const float* __restrict__ own,
                                             float v[4]) {
  if (!bits) return;
  const float4 o = ld4(own);
  if (bits & 1u) v[0] = o.x;
  if (bits & 2u) v[1] = o.y;
  if (bits & 4u) v[2] = o.z;
  if (bits & 8u) v[3] = o.w;
}

// pull_cell for the lane's four cells: post-stream populations with halfway bounce-back; the
// Zou-He completion is per cell (complete_cell).  b: the state at the grid's first row.
__device__ __forceinline__ void pull_chunk(const GridDev& G, const float* __restrict__ b,
                                           const ChunkAt& at, const uint32_t win[3],
                                           float g[kQ][4]) {
  const int ym = at.y == 0 ? G.ny - 1 : at.y - 1, yp = at.y == G.ny - 1 ? 0 : at.y + 1;
  const uint32_t own = (win[1] >> 1) & 0xfu;
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const int ys = cy_of(i) > 0 ? ym : (cy_of(i) == 0 ? at.y : yp);
    chunk_shifted(-cx_of(i), b + (size_t)i * G.plane + (size_t)ys * G.pitch, G, at, g[i]);
    if (i > 0) {
      const uint32_t w = cy_of(i) > 0 ? win[0] : (cy_of(i) == 0 ? win[1] : win[2]);
      chunk_select((w >> (1 - cx_of(i))) & 0xfu & ~own,
                   b + (size_t)opp_of(i) * G.plane + (size_t)at.y * G.pitch + at.x, g[i]);
    }
  }
}
// Zou-He completion of one cell (pull_cell's formulas).
__device__ __forceinline__ void complete_cell(const GridDev& G, int x, float g[kQ]) {
  if (G.periodic_x) return;
  if (x == 0) {
    const float G0 = g[0] + g[2] + g[4] + 2.0f * (g[3] + g[6] + g[7]);
    float ru;
    if (G.bc_west == LBM_BC_PRESSURE) {
      ru = G.west_d - G0;
    } else {
      const float U = G.west_d;
      ru = (1.0f + G0) / (1.0f - U) * U;
    }
    const float t = 0.5f * (g[2] - g[4]);
    g[1] = g[3] + (2.0f / 3.0f) * ru;
    g[5] = g[7] - t + (1.0f / 6.0f) * ru;
    g[8] = g[6] + t + (1.0f / 6.0f) * ru;
  }
  if (x == G.nx - 1) {
    const float G0 = g[0] + g[2] + g[4] + 2.0f * (g[1] + g[5] + g[8]);
    float ru;
    if (G.bc_east == LBM_BC_PRESSURE) {
      ru = G0 - G.east_d;
    } else {
      const float U = G.east_d;
      ru = (1.0f + G0) / (1.0f + U) * U;
    }
    const float t = 0.5f * (g[2] - g[4]);
    g[3] = g[1] - (2.0f / 3.0f) * ru;
    g[7] = g[5] + t - (1.0f / 6.0f) * ru;
    g[6] = g[8] - t - (1.0f / 6.0f) * ru;
  }
}
// Four values to dense cells x .. x + 3 of a row: one 16-byte store where `vec` says it is
// aligned, else those inside the row.
__device__ __forceinline__ void store_chunk(float* row, int x, int nx, bool vec, const float v[4]) {
  if (vec) {
    *reinterpret_cast<float4*>(row + x) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (x + j < nx) row[x + j] = v[j];
  }
}
__host__ __device__ __forceinline__ bool aligned16(const void* p) {
  return (reinterpret_cast<uintptr_t>(p) & 15) == 0;
}

}  // namespace lbmfno
