// Reverse-mode (adjoint) kernels of the LBM part of the hybrid pipeline and their
// C ABI: the vector-Jacobian products of the moments (Sec. 2.1), of one fused
// time step (pull streaming with halfway bounce-back, Zou-He completion, BGK
// collision with the Guo source, Sec. 2.1), and of the re-initialisation of the
// populations from macroscopic fields (f^eq + Chapman-Enskog f^neq, Sec. 2.3).
//
// Notation.  s_n is the stored state of the library (shifted post-collision
// populations of time level n-1), P the pull that turns it into the populations
// f_n of level n (gather with bounce-back, then Zou-He completion of the unknown
// populations of open end columns), C the per-cell collision, M the moments:
//   lbm_step:  s_{n+1} = C(P(s_n)),   lbm_macro: (rho, u)_n = M(P(s_n)).
// The adjoint variable mu_n is the gradient of the loss with respect to the
// *pulled known* populations of every fluid cell at level n, i.e. to the values
// gathered by P before the Zou-He completion (unknown slots hold 0, solid cells
// hold 0).  Then
//   mu_N     = Z^T (dM/df)^T (drho, du)                 lbm_adjoint_macro
//   mu_{n-1} = Z^T J_C(f_{n-1})^T G^T mu_n               lbm_adjoint_step
//   (drho, du)_0 = R^T mu_0                              lbm_adjoint_reinit
// with Z the Zou-He completion (linear in the known populations), J_C the 9x9
// collision Jacobian of each cell at f_{n-1} = P(s_{n-1}), G the gather of the
// pull (a permutation of the fluid slots with bounce-back), and R the
// re-initialisation followed by the pull, whose known populations are exactly
// f^eq + f^neq of each cell.
//
// Every buffer here is in the canonical state layout of lbm_get_state: per grid,
// 9 planes of ny x nx floats at 9 * cell offset.  All kernels are per-cell and
// read only the cell's own stencil, so there are no atomics and the results are
// deterministic.
#include <math.h>

#include "common.cuh"
#include "lbm_cell.cuh"
#include "lbm_chunk.cuh"
#include "lbm_internal.cuh"

namespace lbmfno {

namespace {

inline cudaStream_t AS(void* s) { return reinterpret_cast<cudaStream_t>(s); }

// A copy of the grid descriptor that addresses the canonical layout.
__device__ __forceinline__ GridDev canonical(const GridDev& G) {
  GridDev C = G;
  C.pitch = G.nx;
  C.plane = (long long)G.nx * G.ny;
  C.f_off = 9LL * G.cell_off;
  return C;
}

// Transpose of the Zou-He completion at an open end cell: the gradients of the
// completed unknown populations are distributed onto the known ones they were
// computed from, and the unknown slots are cleared.  rho u_x = a + beta * G0
// with G0 the sum of the known populations (2x those pointing outwards).
__device__ __forceinline__ void zou_he_transpose(const GridDev& G, bool west, bool east,
                                                 float m[kQ]) {
  if (west) {  // unknown 1, 5, 8
    const float beta = (G.bc_west == LBM_BC_PRESSURE) ? -1.0f : G.west_d / (1.0f - G.west_d);
    const float bs = beta * ((2.0f / 3.0f) * m[1] + (1.0f / 6.0f) * (m[5] + m[8]));
    m[0] += bs;
    m[2] += bs - 0.5f * m[5] + 0.5f * m[8];
    m[4] += bs + 0.5f * m[5] - 0.5f * m[8];
    m[3] += m[1] + 2.0f * bs;
    m[7] += m[5] + 2.0f * bs;
    m[6] += m[8] + 2.0f * bs;
    m[1] = m[5] = m[8] = 0.0f;
  }
  if (east) {  // unknown 3, 6, 7
    const float beta = (G.bc_east == LBM_BC_PRESSURE) ? 1.0f : G.east_d / (1.0f + G.east_d);
    const float bs = -beta * ((2.0f / 3.0f) * m[3] + (1.0f / 6.0f) * (m[7] + m[6]));
    m[0] += bs;
    m[2] += bs + 0.5f * m[7] - 0.5f * m[6];
    m[4] += bs - 0.5f * m[7] + 0.5f * m[6];
    m[1] += m[3] + 2.0f * bs;
    m[5] += m[7] + 2.0f * bs;
    m[8] += m[6] + 2.0f * bs;
    m[3] = m[6] = m[7] = 0.0f;
  }
}

// lam <- J_C(f)^T lam for the BGK collision with the Guo source:
//   (J^T l)_j = (1 - om) l_j + om [A + V.(c_j - u)] + Gv.(c_j - u) / rho
//   A   = sum_i l_i f^eq_i / rho
//   V_a = sum_i l_i w_i (3 c_ia + 9 (c_i.u) c_ia - 3 u_a)
//   Gv_b = (1 - om/2) sum_i l_i w_i (-3 F_b + 9 c_ib (c_i.F))
__device__ __forceinline__ void collision_transpose(const GridDev& G, const float f[kQ],
                                                    float l[kQ]) {
  float drho, rho, ux, uy;
  moments(G, f, drho, rho, ux, uy);
  const float usq = 1.5f * (ux * ux + uy * uy);
  const float om = G.omega;
  float A = 0.f, Vx = 0.f, Vy = 0.f, Gx = 0.f, Gy = 0.f;
  const bool forced = (G.fx != 0.0f || G.fy != 0.0f);
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const float cx = (float)cx_of(i), cy = (float)cy_of(i);
    const float cu = cx * ux + cy * uy;
    const float wl = w_of(i) * l[i];
    A += wl * (1.0f + 3.0f * cu + 4.5f * cu * cu - usq);
    const float t = 3.0f + 9.0f * cu;
    Vx += wl * (t * cx - 3.0f * ux);
    Vy += wl * (t * cy - 3.0f * uy);
    if (forced) {
      const float cf = 9.0f * (cx * G.fx + cy * G.fy);
      Gx += wl * (cf * cx - 3.0f * G.fx);
      Gy += wl * (cf * cy - 3.0f * G.fy);
    }
  }
  const float ginv = G.guo / rho;  // guo = 1 - om / 2
#pragma unroll
  for (int j = 0; j < kQ; ++j) {
    const float dx = (float)cx_of(j) - ux, dy = (float)cy_of(j) - uy;
    l[j] = (1.0f - om) * l[j] + om * (A + Vx * dx + Vy * dy) + ginv * (Gx * dx + Gy * dy);
  }
}

__device__ __forceinline__ void store9(const GridDev& Gc, float* buf, int x, int y,
                                       const float v[kQ]) {
  float* o = buf + Gc.f_off + (long long)y * Gc.pitch + x;
#pragma unroll
  for (int i = 0; i < kQ; ++i) o[i * Gc.plane] = v[i];
}

__global__ void __launch_bounds__(kBlock) k_adj_macro(const GridDev* __restrict__ grids,
                                                      int ngrids, const uint32_t* __restrict__ mask,
                                                      const float* __restrict__ state,
                                                      const float* __restrict__ drho_i,
                                                      const float* __restrict__ dux_i,
                                                      const float* __restrict__ duy_i,
                                                      float* __restrict__ mu) {
  int gidx, x, y;
  if (!cell_of_thread(grids, ngrids, gidx, x, y)) return;
  const GridDev Gc = canonical(grids[gidx]);
  float f[kQ], m[kQ];
  if (!pull_cell(Gc, mask, state, x, y, f)) {
#pragma unroll
    for (int i = 0; i < kQ; ++i) m[i] = 0.0f;
    store9(Gc, mu, x, y, m);
    return;
  }
  float drho, rho, ux, uy;
  moments(Gc, f, drho, rho, ux, uy);
  const long long c = Gc.cell_off + (long long)y * Gc.nx + x;
  const float dr = drho_i[c], inv = 1.0f / rho;
  const float ax = dux_i[c] * inv, ay = duy_i[c] * inv;
#pragma unroll
  for (int j = 0; j < kQ; ++j)
    m[j] = dr + ax * ((float)cx_of(j) - ux) + ay * ((float)cy_of(j) - uy);
  zou_he_transpose(Gc, !Gc.periodic_x && x == 0, !Gc.periodic_x && x == Gc.nx - 1, m);
  store9(Gc, mu, x, y, m);
}

// Solid bits of cells x - 1, x, x + 1 of mask row mr (bits 0, 1, 2), wrapped for periodic rows, 0
// beyond an open end.  The cells of a warp share their word, so these are broadcast loads.
__device__ __forceinline__ uint32_t cell_window(const uint32_t* __restrict__ mr, const GridDev& G,
                                                int x) {
  const int wi = x >> 5;
  uint64_t v = (uint64_t)__ldg(mr + wi) << 1;
  if (wi > 0) v |= __ldg(mr + wi - 1) >> 31;
  if (wi + 1 < G.wpr) v |= (uint64_t)(__ldg(mr + wi + 1) & 1u) << 33;
  uint32_t win = (uint32_t)(v >> (x & 31)) & 7u;
  if (x == 0) {
    win &= 6u;
    if (G.periodic_x) win |= (uint32_t)mask_bit(mr, 0, G.nx - 1, 0);
  }
  if (x == G.nx - 1) {
    win &= 3u;
    if (G.periodic_x) win |= (uint32_t)mask_bit(mr, 0, 0, 0) << 2;
  }
  return win;
}

// One cell a thread, both gathers from three 3-bit windows of the mask and one selected address a
// population, all eighteen loads in flight at once (with a mask word and an address of its own for
// every neighbour, as pull_cell does it: 74 us on 2.1 M cells, now 62; HBM needs 33, and the 750
// instructions a cell keep the issue slots 68% busy).
__global__ void __launch_bounds__(kBlock) k_adj_step(const GridDev* __restrict__ grids,
                                                     int ngrids, const uint32_t* __restrict__ mask,
                                                     const float* __restrict__ state_prev,
                                                     const float* __restrict__ mu_in,
                                                     float* __restrict__ mu_out) {
  int gidx, x, y;
  if (!cell_of_thread(grids, ngrids, gidx, x, y)) return;
  const GridDev Gc = canonical(grids[gidx]);
  const int ym = (y == 0) ? Gc.ny - 1 : y - 1, yp = (y == Gc.ny - 1) ? 0 : y + 1;
  const uint32_t* m = mask + Gc.mask_off;
  const uint32_t win[3] = {cell_window(m + (size_t)ym * Gc.wpr, Gc, x),
                           cell_window(m + (size_t)y * Gc.wpr, Gc, x),
                           cell_window(m + (size_t)yp * Gc.wpr, Gc, x)};
  float f[kQ], l[kQ];
  if (win[1] & 2u) {
#pragma unroll
    for (int i = 0; i < kQ; ++i) l[i] = 0.0f;
    store9(Gc, mu_out, x, y, l);
    return;
  }
  const bool west_end = x == 0, east_end = x == Gc.nx - 1;
  const bool open_w = !Gc.periodic_x && west_end, open_e = !Gc.periodic_x && east_end;
  // 32-bit indexes from the grid's first value (a batch holds fewer than 2^31)
  const unsigned xm = west_end ? Gc.nx - 1 : x - 1, xp = east_end ? 0 : x + 1;
  const unsigned P = (unsigned)Gc.plane, pitch = (unsigned)Gc.pitch;
  const unsigned row[3] = {(unsigned)ym * pitch, (unsigned)y * pitch, (unsigned)yp * pitch};
  const unsigned here = row[1] + (unsigned)x;
  const float* bs = state_prev + Gc.f_off;
  const float* bm = mu_in + Gc.f_off;
  // population i of f comes from x - c_i; slot (j, x) of the stored state was read by cell x + c_j
  // when that is a fluid cell of the domain, by this cell's population opp(j) (bounce-back) when
  // it is solid, and by nobody when it lies beyond an open end
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const int dx = cx_of(i), dy = cy_of(i);
    const bool from_out = dx > 0 ? open_w : (dx < 0 && open_e);
    const bool to_out = dx > 0 ? open_e : (dx < 0 && open_w);
    const bool from_solid = i > 0 && ((win[1 - dy] >> (1 - dx)) & 1u);
    const bool to_solid = i > 0 && ((win[1 + dy] >> (1 + dx)) & 1u);
    const unsigned from = i * P + row[1 - dy] + (dx > 0 ? xm : (dx < 0 ? xp : (unsigned)x));
    const unsigned to = i * P + row[1 + dy] + (dx > 0 ? xp : (dx < 0 ? xm : (unsigned)x));
    const unsigned own = opp_of(i) * P + here;
    f[i] = from_out ? 0.0f : __ldg(bs + (from_solid ? own : from));
    l[i] = to_out ? 0.0f : __ldg(bm + (to_solid ? own : to));
  }
  complete_cell(Gc, x, f);
  collision_transpose(Gc, f, l);
  zou_he_transpose(Gc, open_w, open_e, l);
  float* o = mu_out + Gc.f_off;
#pragma unroll
  for (int i = 0; i < kQ; ++i) o[i * P + here] = l[i];
}

// k_adj_macro with a chunk of four cells a lane, for batches that fill the chip (chunk_pays) and
// whose canonical and dense rows are 16-byte aligned (2.1 M cells: 64 -> 38 us).  The adjoint step in this form took 86 us: both
// gathers of four cells leave too few warps, so it stays one cell a thread.
__device__ __forceinline__ void store9_chunk(const GridDev& Gc, float* buf, const ChunkAt& at,
                                             const float v[kQ][4]) {
  float* o = buf + Gc.f_off + (size_t)at.y * Gc.pitch + at.x;
#pragma unroll
  for (int i = 0; i < kQ; ++i)
    *reinterpret_cast<float4*>(o + (size_t)i * Gc.plane) =
        make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
}

__global__ void __launch_bounds__(32 * kChunkRows) k_adj_macro_chunk(
    const GridDev* __restrict__ grids, const int4* __restrict__ tiles,
    const uint32_t* __restrict__ mask, const float* __restrict__ state,
    const float* __restrict__ drho_i, const float* __restrict__ dux_i,
    const float* __restrict__ duy_i, float* __restrict__ mu) {
  const ChunkAt at = chunk_of_lane(grids, tiles);
  if (!at.row) return;
  const GridDev Gc = canonical(grids[at.grid]);
  uint32_t win[3];
  chunk_windows(mask + Gc.mask_off, Gc, at, win);
  float f[kQ][4];
  pull_chunk(Gc, state + Gc.f_off, at, win, f);
  if (!at.active) return;
  const size_t c0 = (size_t)Gc.cell_off + (size_t)at.y * Gc.nx + at.x;
  const float4 r4 = ld4(drho_i + c0), x4 = ld4(dux_i + c0), y4 = ld4(duy_i + c0);
  const float dr[4] = {r4.x, r4.y, r4.z, r4.w}, dx[4] = {x4.x, x4.y, x4.z, x4.w},
              dy[4] = {y4.x, y4.y, y4.z, y4.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float c[kQ], m[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) c[i] = f[i][k];
    complete_cell(Gc, at.x + k, c);
    float drho, rho, ux, uy;
    moments(Gc, c, drho, rho, ux, uy);
    const float inv = 1.0f / rho, ax = dx[k] * inv, ay = dy[k] * inv;
#pragma unroll
    for (int j = 0; j < kQ; ++j)
      m[j] = dr[k] + ax * ((float)cx_of(j) - ux) + ay * ((float)cy_of(j) - uy);
    zou_he_transpose(Gc, !Gc.periodic_x && at.x + k == 0, !Gc.periodic_x && at.x + k == Gc.nx - 1,
                     m);
    const bool solid = (win[1] >> (k + 1)) & 1u;
#pragma unroll
    for (int i = 0; i < kQ; ++i) f[i][k] = solid ? 0.0f : m[i];
  }
  store9_chunk(Gc, mu, at, f);
}

// R^T, local part: per fluid cell the gradient with respect to rho and u of the
// cell's own f^eq + f^neq, and the gradients with respect to the four velocity
// derivatives (d_x u_x, d_y u_y, and the shared coefficient of d_x u_y and d_y u_x)
// that the stencil kernel below distributes to the neighbours.
__global__ void __launch_bounds__(kBlock) k_adj_reinit_local(
    const GridDev* __restrict__ grids, int ngrids, const uint32_t* __restrict__ mask,
    const float* __restrict__ mu, const float* __restrict__ rho_i,
    const float* __restrict__ ux_i, const float* __restrict__ uy_i, int neq_mode,
    float* __restrict__ drho_o, float* __restrict__ dux_o, float* __restrict__ duy_o,
    float* __restrict__ dgrad) {
  int gidx, x, y;
  if (!cell_of_thread(grids, ngrids, gidx, x, y)) return;
  const GridDev G = grids[gidx];
  const GridDev Gc = canonical(G);
  const long long cells = (long long)G.nx * G.ny;
  const long long c = G.cell_off + (long long)y * G.nx + x;
  const uint32_t* m = mask + G.mask_off;
  float* dg = dgrad + 3LL * G.cell_off + (long long)y * G.nx + x;
  if (mask_bit(m, G.wpr, x, y)) {
    drho_o[c] = dux_o[c] = duy_o[c] = 0.0f;
    dg[0] = dg[cells] = dg[2 * cells] = 0.0f;
    return;
  }
  float l[kQ];
  const float* b = mu + Gc.f_off + (long long)y * Gc.pitch + x;
#pragma unroll
  for (int i = 0; i < kQ; ++i) l[i] = b[i * Gc.plane];
  // unknown populations of open end cells are not taken from the reinit
  if (!G.periodic_x && x == 0) l[1] = l[5] = l[8] = 0.0f;
  if (!G.periodic_x && x == G.nx - 1) l[3] = l[6] = l[7] = 0.0f;
  const float rho = rho_i[c], ux = ux_i[c], uy = uy_i[c];
  float dxux = 0.f, dxuy = 0.f, dyux = 0.f, dyuy = 0.f;
  if (neq_mode) {
    const float* UX = ux_i + G.cell_off;
    const float* UY = uy_i + G.cell_off;
    dxux = dfield(G, m, UX, x, y, 0);
    dxuy = dfield(G, m, UY, x, y, 0);
    dyux = dfield(G, m, UX, x, y, 1);
    dyuy = dfield(G, m, UY, x, y, 1);
  }
  const float usq = 1.5f * (ux * ux + uy * uy);
  const float div = dxux + dyuy;
  const float k3 = -3.0f * G.tau;
  float gr = 0.f, gx = 0.f, gy = 0.f, sxx = 0.f, syy = 0.f, sxy = 0.f;
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const float cx = (float)cx_of(i), cy = (float)cy_of(i);
    const float cu = cx * ux + cy * uy;
    const float wl = w_of(i) * l[i];
    const float qd = cx * cx * dxux + cx * cy * (dxuy + dyux) + cy * cy * dyuy - div / 3.0f;
    gr += wl * (1.0f + 3.0f * cu + 4.5f * cu * cu - usq + k3 * qd);
    const float t = 3.0f + 9.0f * cu;
    gx += wl * (t * cx - 3.0f * ux);
    gy += wl * (t * cy - 3.0f * uy);
    sxx += wl * (cx * cx - 1.0f / 3.0f);
    syy += wl * (cy * cy - 1.0f / 3.0f);
    sxy += wl * (cx * cy);
  }
  drho_o[c] = gr;
  dux_o[c] = rho * gx;
  duy_o[c] = rho * gy;
  const float kr = k3 * rho;
  dg[0] = kr * sxx;          // d loss / d (d_x u_x)
  dg[cells] = kr * syy;      // d loss / d (d_y u_y)
  dg[2 * cells] = kr * sxy;  // d loss / d (d_x u_y) = d loss / d (d_y u_x)
}

// Stencil of the derivative of a field at fluid cell (x, y) along `axis`: flags for
// the + and - neighbours (fluid cells of the domain), mirroring dfield.
__device__ __forceinline__ void stencil_flags(const GridDev& G, const uint32_t* m, int x, int y,
                                              int axis, bool& okp, bool& okm) {
  int xp = x, xm = x, yp = y, ym = y;
  okp = okm = true;
  if (axis == 0) {
    xp = x + 1;
    xm = x - 1;
    if (G.periodic_x) {
      if (xp >= G.nx) xp = 0;
      if (xm < 0) xm = G.nx - 1;
    } else {
      okp = xp < G.nx;
      okm = xm >= 0;
    }
  } else {
    yp = (y == G.ny - 1) ? 0 : y + 1;
    ym = (y == 0) ? G.ny - 1 : y - 1;
  }
  if (okp && mask_bit(m, G.wpr, xp, yp)) okp = false;
  if (okm && mask_bit(m, G.wpr, xm, ym)) okm = false;
}

// Transpose of the derivative stencil along `axis` applied to the field D (the
// gradient with respect to that derivative), gathered at fluid cell (x, y).
__device__ __forceinline__ float stencil_transpose(const GridDev& G, const uint32_t* m,
                                                   const float* D, int x, int y, int axis) {
  float acc = 0.0f;
  bool okp, okm;
  stencil_flags(G, m, x, y, axis, okp, okm);  // the cell's own derivative
  if (okp != okm) acc += (okp ? -1.0f : 1.0f) * D[(long long)y * G.nx + x];
  // the - neighbour uses this cell as its + neighbour, the + neighbour as its -
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    int nx_ = x, ny_ = y;
    if (axis == 0) {
      nx_ = side == 0 ? x - 1 : x + 1;
      if (nx_ < 0 || nx_ >= G.nx) {
        if (!G.periodic_x) continue;
        nx_ = nx_ < 0 ? G.nx - 1 : 0;
      }
    } else {
      ny_ = side == 0 ? (y == 0 ? G.ny - 1 : y - 1) : (y == G.ny - 1 ? 0 : y + 1);
    }
    if (mask_bit(m, G.wpr, nx_, ny_)) continue;
    bool np, nm;
    stencil_flags(G, m, nx_, ny_, axis, np, nm);
    const float d = D[(long long)ny_ * G.nx + nx_];
    if (side == 0)  // this cell is the + neighbour of (nx_, ny_): np is true
      acc += (nm ? 0.5f : 1.0f) * d;
    else  // this cell is the - neighbour of (nx_, ny_): nm is true
      acc -= (np ? 0.5f : 1.0f) * d;
  }
  return acc;
}

__global__ void __launch_bounds__(kBlock) k_adj_reinit_stencil(
    const GridDev* __restrict__ grids, int ngrids, const uint32_t* __restrict__ mask,
    const float* __restrict__ dgrad, float* __restrict__ dux_o, float* __restrict__ duy_o) {
  int gidx, x, y;
  if (!cell_of_thread(grids, ngrids, gidx, x, y)) return;
  const GridDev G = grids[gidx];
  const uint32_t* m = mask + G.mask_off;
  if (mask_bit(m, G.wpr, x, y)) return;
  const long long cells = (long long)G.nx * G.ny;
  const float* Dxx = dgrad + 3LL * G.cell_off;
  const float* Dyy = Dxx + cells;
  const float* Dxy = Dxx + 2 * cells;
  const long long c = G.cell_off + (long long)y * G.nx + x;
  // u_x enters d_x u_x (axis 0) and d_y u_x (axis 1); u_y enters d_x u_y and d_y u_y
  dux_o[c] += stencil_transpose(G, m, Dxx, x, y, 0) + stencil_transpose(G, m, Dxy, x, y, 1);
  duy_o[c] += stencil_transpose(G, m, Dxy, x, y, 0) + stencil_transpose(G, m, Dyy, x, y, 1);
}

}  // namespace

}  // namespace lbmfno

using namespace lbmfno;

extern "C" {

int lbm_adjoint_macro(lbm_handle* h, const float* gstar_d, const float* drho_d,
                      const float* dux_d, const float* duy_d, float* mu_d, void* stream) {
  LBM_REQUIRE(h != nullptr && gstar_d != nullptr && drho_d != nullptr && dux_d != nullptr &&
                  duy_d != nullptr && mu_d != nullptr,
              "lbm_adjoint_macro: null argument");
  if (h->dense4 && chunk_pays(h) && aligned16(gstar_d) && aligned16(drho_d) &&
      aligned16(dux_d) && aligned16(duy_d) && aligned16(mu_d))
    k_adj_macro_chunk<<<h->ntiles_v[kChunkVariant], 32 * kChunkRows, 0, AS(stream)>>>(
        h->gd_d, h->tiles_d[kChunkVariant], h->mask, gstar_d, drho_d, dux_d, duy_d, mu_d);
  else
    k_adj_macro<<<h->nblk_total, kBlock, 0, AS(stream)>>>(h->gd_d, h->ngrids, h->mask, gstar_d,
                                                          drho_d, dux_d, duy_d, mu_d);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}

int lbm_adjoint_step(lbm_handle* h, const float* gstar_prev_d, const float* mu_d,
                     float* mu_prev_d, void* stream) {
  LBM_REQUIRE(h != nullptr && gstar_prev_d != nullptr && mu_d != nullptr && mu_prev_d != nullptr,
              "lbm_adjoint_step: null argument");
  LBM_REQUIRE(mu_d != mu_prev_d, "lbm_adjoint_step: mu and mu_prev must not alias");
  k_adj_step<<<h->nblk_total, kBlock, 0, AS(stream)>>>(h->gd_d, h->ngrids, h->mask,
                                                       gstar_prev_d, mu_d, mu_prev_d);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}

int lbm_adjoint_reinit(lbm_handle* h, const float* mu_d, const float* rho_d, const float* ux_d,
                       const float* uy_d, int neq_mode, float* scratch_d, float* drho_d,
                       float* dux_d, float* duy_d, void* stream) {
  LBM_REQUIRE(h != nullptr && mu_d != nullptr && rho_d != nullptr && ux_d != nullptr &&
                  uy_d != nullptr && scratch_d != nullptr && drho_d != nullptr &&
                  dux_d != nullptr && duy_d != nullptr,
              "lbm_adjoint_reinit: null argument");
  k_adj_reinit_local<<<h->nblk_total, kBlock, 0, AS(stream)>>>(
      h->gd_d, h->ngrids, h->mask, mu_d, rho_d, ux_d, uy_d, neq_mode, drho_d, dux_d, duy_d,
      scratch_d);
  LBM_CHECK_LAUNCH();
  if (neq_mode) {
    k_adj_reinit_stencil<<<h->nblk_total, kBlock, 0, AS(stream)>>>(h->gd_d, h->ngrids,
                                                                   h->mask, scratch_d, dux_d,
                                                                   duy_d);
    LBM_CHECK_LAUNCH();
  }
  return LBM_OK;
}

}  // extern "C"
