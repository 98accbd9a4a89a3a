// Two time steps of the D2Q9 lattice in one pass over memory (Sec. 2.1 loop: streaming with
// halfway bounce-back, Zou-He completion, moments, BGK collision), for GB300 (sm_103a).
//
// A single step moves 72 B a cell and is bound by HBM (98.7 us on 64 grids of 512 x 256, 0.90
// of the copy bandwidth).  A pass of two steps moves the same 72 B for both.
//
// Decomposition.  A warp owns 128 columns (four cells a lane) and sweeps down the rows of its
// task.  Level 0 are the stored populations, level 1 and 2 the states after one and two steps;
// in iteration k the warp computes one row of level 2 from three rows of level 1, then one row
// of level 1 from three rows of level 0, two rows further on.  Every population of a row is
// pulled by exactly one row of the next level (and by its own row, for bounce-back), so a
// level keeps 21 (level 0: 15) rows of single populations in shared memory, private to the
// lane that wrote them: no barrier orders them.  Level 0 arrives by cp.async, a lane copying
// its own 16 bytes: the slots of an iteration are refilled for the next as soon as they are
// read.  The x-shift takes the neighbouring lane's cell by shuffle.
//
// Rows of up to four warps are split over warps of a group, which hand each other their edge
// columns (six values a row and level) through shared memory, one barrier of the group an
// iteration; wider rows are cut into strips that overlap by one chunk of four columns on each
// side, whose lanes compute but do not store (a level spoils one more column inwards).  Tasks
// overlap in y the same way: a task of l rows computes l + 2 rows of level 1.
//
// Rounding.  The collision runs on packed pairs with the operations of the single-step kernel in
// the same order; the file is compiled without multiply-add contraction.  States are bitwise
// those of single steps.
//
// What bounds it (64 grids of 512 x 256): 57 us a step.  The pass moves 5.3 TB/s; issue
// slots are 47% busy with the eleven to twelve warps a multiprocessor that the shared memory of the
// kept rows allows, and their fixed-latency chains are what is left.  Measured and not kept:
// two cells a lane and 24 warps (89 us: the per-lane work is not halved), the kept rows in
// registers (79 us with 8 warps, or spills), three steps a pass (132 us: 8 warps).
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "lbm_cell.cuh"
#include "lbm_internal.cuh"
#include "lbm_sweep.cuh"

namespace lbmfno {

namespace {

constexpr int kWarps = kSweepWarps;
constexpr int kRing = 4;                   // rows of the edge ring
constexpr int kV = 4;                      // cells of a lane
constexpr int kH = 2;                      // packed pairs of a lane
constexpr int kT = kSweepSteps;
constexpr int kCtas = 3;                   // CTAs a multiprocessor (shared memory, registers)
constexpr int kHalo = (kT + kV - 1) / kV;  // halo chunks
constexpr int kRowFloats = 32 * kV;        // columns of a warp
constexpr uint32_t kOwn = (1u << kV) - 1u;
constexpr int kEdge = 6;                   // edge values of a warp, level and row
// Rows of one population that a warp keeps in shared memory.  Level 0 (input rows): the
// populations moving up (2, 5, 6) and down (4, 7, 8) of two rows, the others of one; every
// further level: three, two and two rows.
constexpr int kRows0 = 2 * 3 + 3 + 2 * 3;
constexpr int kRows1 = 3 * 3 + 2 * 3 + 2 * 3;
constexpr int kEdge0 = 2 * 8;              // level-0 edge columns: two rows, west and east
constexpr int kWarpFloats = (kRows0 + (kT - 1) * kRows1) * kRowFloats + kEdge0;
__host__ __device__ constexpr int cls_of(int i) { return cy_of(i) > 0 ? 0 : (cy_of(i) == 0 ? 1 : 2); }
__host__ __device__ constexpr int in_cls(int i) {  // 2 5 6 | 0 1 3 | 4 7 8
  return i == 2 || i == 0 || i == 4 ? 0 : (i == 5 || i == 1 || i == 7 ? 1 : 2);
}

// cp.async: this lane's own 16 (or 4) bytes, read back by the lane that copied them
__device__ __forceinline__ void cpa16(uint32_t s, const float* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(g) : "memory");
}
// A lane's chunk of a row in shared memory.  volatile: the loads are for values that a
// select may drop, and the compiler would otherwise turn them into branches around them.
__device__ __forceinline__ void ld_chunk(uint32_t p, float2 v[kH]) {
  asm volatile("ld.volatile.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y)
               : "r"(p));
}
__device__ __forceinline__ void st_chunk_s(uint32_t p, const float2 v[kH]) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p), "f"(v[0].x), "f"(v[0].y),
               "f"(v[1].x), "f"(v[1].y));
}
__device__ __forceinline__ float ld_s(uint32_t p) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(p));
  return v;
}
__device__ __forceinline__ void st_s(uint32_t p, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(p), "f"(v));
}
// ... and of a row in global memory
__device__ __forceinline__ void st_chunk(float* p, const float2 v[kH]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
}
__device__ __forceinline__ void cpa4(uint32_t s, const float* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(g) : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Packed FP32: the same rounding per lane as the scalar operation (a - b is the one
// rounding of b * (-1) + a).
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
// a * b as the fused a * b - 0, which cannot be contracted with an addition that follows
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return fma2(a, b, dup(-0.0f)); }
// A constant times a pair as two scalar products: they take the constant as an immediate, which
// packed instructions do not (58.3 -> 57.0 us a step on 64 grids of 512 x 256).
__device__ __forceinline__ float2 mulc(float c, float2 a) {
  return make_float2(__fmul_rn(c, a.x), __fmul_rn(c, a.y));
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, dup(-1.0f), a); }

// Correctly rounded reciprocals of a lane's values, all in [0.5, 2): the approximate
// reciprocal (within one ulp) and one fused Newton step, which rounds correctly (Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor", 1990); if one
// is outside, __frcp_rn.  Equal to the correctly rounded quotient for every float in the range:
// tests/test_gpu_reciprocal.py takes all 2^24.
__device__ __forceinline__ void rcp_lane(const float2 rho[kH], float2 inv[kH]) {
  uint32_t far = 0;
#pragma unroll
  for (int h = 0; h < kH; ++h)
    far |= (__float_as_uint(rho[h].x) ^ 0x3f000000u) | (__float_as_uint(rho[h].y) ^ 0x3f000000u);
  if (far & 0xff000000u) {
#pragma unroll
    for (int h = 0; h < kH; ++h) inv[h] = make_float2(__frcp_rn(rho[h].x), __frcp_rn(rho[h].y));
    return;
  }
#pragma unroll
  for (int h = 0; h < kH; ++h) {
    float2 y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(rho[h].x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(rho[h].y));
    const float2 e = fma2(make_float2(-rho[h].x, -rho[h].y), y, dup(1.0f));
    inv[h] = fma2(y, e, y);
  }
}

__device__ __forceinline__ void relax_pair2(float2& gi, float2& go, float2 wr3, float2 nwr3,
                                            float2 w45, float2 cu, float2 base, float2 om) {
  const float2 even = fma2(mul2(w45, cu), cu, base);
  gi = fma2(om, sub2(fma2(wr3, cu, even), gi), gi);
  go = fma2(om, sub2(fma2(nwr3, cu, even), go), go);
}
// collide() of lbm_cell.cuh on two cells at once: the same operations in the same order,
// so every value is bitwise the value of the single-step kernel.
__device__ __forceinline__ float2 drho2(const float2 g[kQ]) {
  return add2(
      add2(add2(add2(g[0], g[1]), add2(g[2], g[3])), add2(add2(g[4], g[5]), add2(g[6], g[7]))),
      g[8]);
}
__device__ __forceinline__ void collide2(float om1, float2 drho, float2 rho, float2 inv,
                                         float2 g[kQ]) {
  const float2 om = dup(om1);
  const float2 jx = add2(add2(sub2(g[1], g[3]), sub2(g[5], g[6])), sub2(g[8], g[7]));
  const float2 jy = add2(add2(sub2(g[2], g[4]), sub2(g[5], g[8])), sub2(g[6], g[7]));
  const float2 ux = mul2(jx, inv), uy = mul2(jy, inv);
  const float2 rusq = mul2(mulc(1.5f, rho), fma2(ux, ux, mul2(uy, uy)));
  const float2 d = sub2(drho, rusq);
  const float2 e1 = mulc(kW1, d), e2 = mulc(kW2, d);
  const float2 r1 = mulc(kW1, rho), r2 = mulc(kW2, rho);
  const float2 a1 = mulc(3.0f, r1), a2 = mulc(3.0f, r2);
  const float2 n1 = mulc(-1.0f, a1), n2 = mulc(-1.0f, a2);
  const float2 b1 = mulc(4.5f, r1), b2 = mulc(4.5f, r2);
  g[0] = fma2(om, fma2(dup(kW0), d, mulc(-1.0f, g[0])), g[0]);
  relax_pair2(g[1], g[3], a1, n1, b1, ux, e1, om);
  relax_pair2(g[2], g[4], a1, n1, b1, uy, e1, om);
  relax_pair2(g[5], g[7], a2, n2, b2, add2(ux, uy), e2, om);
  relax_pair2(g[6], g[8], a2, n2, b2, sub2(uy, ux), e2, om);
}

// The forced collision (Guo source) on two cells, in the order of collide().  Its products feed
// sums; the assembler contracts a packed product and sum that are separate instructions, so the
// sums here are multiply-adds with `one`, a 1 it cannot see (a run-time value).
__device__ __forceinline__ void forced_pair2(float2& gi, float2& go, float w, float2 cu, float cf,
                                             float2 drho, float2 rho, float2 usq, float2 om,
                                             float2 sym_f, float guo, float2 one) {
  auto add = [&](float2 a, float2 b) { return fma2(a, one, b); };
  const float2 q = mul2(mul2(dup(4.5f), cu), cu);
  const float2 even = mul2(dup(w), add(mul2(rho, sub2(q, usq)), drho));
  const float2 odd = mul2(mul2(mul2(dup(w), rho), dup(3.0f)), cu);
  const float2 s_even = mul2(dup(guo * w), add(mul2(mul2(dup(9.0f), cu), dup(cf)), sym_f));
  const float2 s_odd = dup(guo * w * 3.0f * cf);
  gi = add(add(mul2(om, sub2(add(even, odd), gi)), gi), add(s_even, s_odd));
  go = add(add(mul2(om, sub2(sub2(even, odd), go)), go), sub2(s_even, s_odd));
}
__device__ __forceinline__ void collide2_forced(float om1, float guo, float fx, float fy,
                                                float one1, float2 drho, float2 rho, float2 inv,
                                                float2 g[kQ]) {
  const float2 om = dup(om1), one = dup(one1);
  auto add = [&](float2 a, float2 b) { return fma2(a, one, b); };
  const float2 jx = add2(add2(add2(sub2(g[1], g[3]), sub2(g[5], g[6])), sub2(g[8], g[7])), dup(0.5f * fx));
  const float2 jy = add2(add2(add2(sub2(g[2], g[4]), sub2(g[5], g[8])), sub2(g[6], g[7])), dup(0.5f * fy));
  const float2 ux = mul2(jx, inv), uy = mul2(jy, inv);
  const float2 usq = mul2(dup(1.5f), add(mul2(ux, ux), mul2(uy, uy)));
  const float2 sym_f = mul2(dup(-3.0f), add(mul2(ux, dup(fx)), mul2(uy, dup(fy))));
  g[0] = add(add(mul2(om, sub2(mul2(dup(kW0), sub2(drho, mul2(rho, usq))), g[0])), g[0]),
             mul2(dup(guo * kW0), sym_f));
  forced_pair2(g[1], g[3], kW1, ux, fx, drho, rho, usq, om, sym_f, guo, one);
  forced_pair2(g[2], g[4], kW1, uy, fy, drho, rho, usq, om, sym_f, guo, one);
  forced_pair2(g[5], g[7], kW2, add(ux, uy), fx + fy, drho, rho, usq, om, sym_f, guo, one);
  forced_pair2(g[6], g[8], kW2, sub2(uy, ux), fy - fx, drho, rho, usq, om, sym_f, guo, one);
}

__device__ __forceinline__ float get2(const float2 v[kH], int j) {
  return j == 0 ? v[0].x : (j == 1 ? v[0].y : (j == 2 ? v[1].x : v[1].y));
}
__device__ __forceinline__ void set2(float2 v[kH], int j, float a) {
  if (j == 0) v[0].x = a;
  else if (j == 1) v[0].y = a;
  else if (j == 2) v[1].x = a;
  else v[1].y = a;
}

// Zou-He completion of the open end columns (the single-step kernel's formulas).  west: the
// lane's first cell is x = 0 of an open grid; je: index of the cell x = nx - 1 of an open
// grid, out of range if the lane has none.
__device__ __forceinline__ void complete_ends(float dw, float de, int kinds, bool west,
                                              unsigned je, float2 g[kQ][kH]) {
#pragma unroll
  for (int j = 0; j < kV; ++j) {
    if ((j == 0 && west) || j == (int)je) {
      float c[kQ];
#pragma unroll
      for (int i = 0; i < kQ; ++i) c[i] = get2(g[i], j);
      if (j == 0 && west) {
        const float G0 = c[0] + c[2] + c[4] + 2.0f * (c[3] + c[6] + c[7]);
        const float ru = (kinds & 1) ? dw - G0 : (1.0f + G0) / (1.0f - dw) * dw;
        const float tt = 0.5f * (c[2] - c[4]);
        c[1] = c[3] + (2.0f / 3.0f) * ru;
        c[5] = c[7] - tt + (1.0f / 6.0f) * ru;
        c[8] = c[6] + tt + (1.0f / 6.0f) * ru;
      }
      if (j == (int)je) {
        const float G0 = c[0] + c[2] + c[4] + 2.0f * (c[1] + c[5] + c[8]);
        const float ru = (kinds & 2) ? G0 - de : (1.0f + G0) / (1.0f + de) * de;
        const float tt = 0.5f * (c[2] - c[4]);
        c[3] = c[1] - (2.0f / 3.0f) * ru;
        c[7] = c[5] + tt - (1.0f / 6.0f) * ru;
        c[6] = c[8] - tt - (1.0f / 6.0f) * ru;
      }
#pragma unroll
      for (int i = 1; i < kQ; ++i) set2(g[i], j, c[i]);
    }
  }
}

template <bool FORCED>
__device__ __forceinline__ void collide_lane(const GridDev* __restrict__ G, float om, float one,
                                             float2 g[kQ][kH]) {
  bool forced = false;
  float guo = 0.0f, fx = 0.0f, fy = 0.0f;
  if constexpr (FORCED) {
    fx = __ldg(&G->fx);
    fy = __ldg(&G->fy);
    guo = __ldg(&G->guo);
    forced = fx != 0.0f || fy != 0.0f;
  }
  float2 drho[kH], rho[kH], inv[kH];
#pragma unroll
  for (int h = 0; h < kH; ++h) {
    float2 c[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) c[i] = g[i][h];
    drho[h] = drho2(c);
    rho[h] = make_float2(__fadd_rn(1.0f, drho[h].x), __fadd_rn(1.0f, drho[h].y));
  }
  rcp_lane(rho, inv);
#pragma unroll
  for (int h = 0; h < kH; ++h) {
    float2 c[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) c[i] = g[i][h];
    if (!FORCED || !forced)
      collide2(om, drho[h], rho[h], inv[h], c);
    else
      collide2_forced(om, guo, fx, fy, one, drho[h], rho[h], inv[h], c);
#pragma unroll
    for (int i = 0; i < kQ; ++i) g[i][h] = c[i];
  }
}

// The pulled values of the three populations with c_iy = CY (east-going, straight,
// west-going), from their source row's chunks s and the neighbouring lanes' cells (l: west of
// the first, r: east of the last cell).  With SOLID, halfway bounce-back: cells whose source
// (in the row whose window is w: bit b <-> cell x - 1 + b) is solid take the own cell's
// opposite population, the class whose rows start at `own`.  Solid cells' own values are
// irrelevant.
template <int CY, bool SOLID>
__device__ __forceinline__ void pull_row(uint32_t w, uint32_t own, const float2 (*s)[kH], float l,
                                         float r, float2 g[kQ][kH]) {
  constexpr int ie = CY > 0 ? 5 : (CY == 0 ? 1 : 8), is = CY > 0 ? 2 : (CY == 0 ? 0 : 4),
                iw = CY > 0 ? 6 : (CY == 0 ? 3 : 7);
  float2 oe[kH], os[kH], ow[kH];
  if constexpr (SOLID) {
    ld_chunk(own + in_cls(opp_of(ie)) * (4 * kRowFloats), oe);
    if constexpr (CY != 0) ld_chunk(own + in_cls(opp_of(is)) * (4 * kRowFloats), os);
    ld_chunk(own + in_cls(opp_of(iw)) * (4 * kRowFloats), ow);
  }
#pragma unroll
  for (int b = 0; b < kV + 2; ++b) {
    const bool solid = SOLID && ((w >> b) & 1u);
    if (b < kV) {
      const float v = b == 0 ? l : get2(s[in_cls(ie)], b - 1);
      set2(g[ie], b, solid ? get2(oe, b) : v);
    }
    if (b >= 1 && b <= kV) {
      const float v = get2(s[in_cls(is)], b - 1);
      set2(g[is], b - 1, CY != 0 && solid ? get2(os, b - 1) : v);
    }
    if (b >= 2) {
      const float v = b == kV + 1 ? r : get2(s[in_cls(iw)], b - 1);
      set2(g[iw], b - 2, solid ? get2(ow, b - 2) : v);
    }
  }
}

// Column of a periodic row: x < nx + kV, without a division (rows shorter than a chunk wrap
// more than once).
__device__ __forceinline__ int wrapped(int x, int nx) {
  while (x >= nx) x -= nx;
  return x;
}

// The bits of three consecutive windows of hist.
constexpr uint32_t kNear = 0x010101u * ((1u << (kV + 2)) - 1u);

template <bool FORCED>
__global__ void __launch_bounds__(kWarps * 32, kCtas)
    k_sweep(const GridDev* __restrict__ grids, const SweepTask* __restrict__ tasks,
            const uint32_t* __restrict__ mask, const float* __restrict__ src,
            float* __restrict__ dst, unsigned P, float one) {
  extern __shared__ __align__(128) float smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const SweepTask* tkp = tasks + (blockIdx.x * kWarps + warp);
  const int rows = __ldg(&tkp->rows);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (rows <= 0) return;  // an unused warp slot: no group counts on it
  const int last_lane = tkp->last;
  const int group = tkp->nwarps > 1 ? (int)tkp->bar << 8 | (int)tkp->nwarps * 32 : 0;
  const int west_warp = tkp->left * kEdge * 4, east_warp = tkp->right * kEdge * 4 + 12;
  const GridDev* __restrict__ G = grids + tkp->grid;
  const float om = __ldg(&G->omega);
  const int x = tkp->v0 + kV * lane;  // virtual column of the lane's first cell
  const unsigned pitch = (unsigned)__ldg(&G->pitch), wpr = (unsigned)__ldg(&G->wpr);
  const bool active = lane <= last_lane, last = lane == last_lane;
  // physical column p of the first cell; the lane's cells are one aligned chunk unless the
  // row wraps inside it (periodic rows whose length is no multiple of kV)
  int p = x, pl, pr;
  bool chunk, west = false;
  unsigned je = kV;
  const int nx = __ldg(&G->nx);
  {
    const bool periodic = __ldg(&G->periodic_x) != 0;
    if (periodic) {
      p %= nx;
      if (p < 0) p += nx;
    } else {
      west = x == 0;
      if (active && x < nx) je = (unsigned)(nx - 1 - x);
    }
    chunk = active && (p & (kV - 1)) == 0 && (p + kV <= nx || !periodic);
    pl = p > 0 ? p - 1 : (periodic ? nx - 1 : 0);
    pr = p + kV < nx ? p + kV : (periodic ? (p + kV) % nx : 0);
  }
  const bool at_end = west || je < (unsigned)kV;
  const float dw = __ldg(&G->west_d), de = __ldg(&G->east_d);
  const int kinds = (__ldg(&G->bc_west) == LBM_BC_PRESSURE ? 1 : 0) |
                    (__ldg(&G->bc_east) == LBM_BC_PRESSURE ? 2 : 0);  // else velocity
  // shared-memory byte addresses: this lane's chunk of row 0, the warp's level-0 edge
  // columns, the published edge columns [kT - 1][kRing][kWarps][kEdge]
  constexpr int R = 4 * kRowFloats;  // bytes of a row
  const uint32_t smem_s = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t own0 = smem_s + warp * (4 * kWarpFloats) + 4 * kV * lane;
  const uint32_t e0 = smem_s + warp * (4 * kWarpFloats) + (kRows0 + (kT - 1) * kRows1) * R;
  const uint32_t edges = smem_s + kWarps * (4 * kWarpFloats);
  const int ny = __ldg(&G->ny);
  int ys = (tkp->y0 - kT) % ny;  // next input row to load
  if (ys < 0) ys += ny;
  // 32-bit byte offsets inside a population plane (nine planes hold fewer than 2^31 floats)
  uint32_t sp = 4u * ((uint32_t)__ldg(&G->f_off) + (uint32_t)p + (uint32_t)ys * pitch);
  const uint32_t* mp = mask + __ldg(&G->mask_off) + (size_t)ys * wpr;
  uint32_t dp = 4u * ((uint32_t)__ldg(&G->f_off) + (uint32_t)tkp->y0 * pitch + (uint32_t)x);
  auto from = [&](int i, uint32_t off) {
    return reinterpret_cast<const float*>(reinterpret_cast<const char*>(src + (size_t)i * P) + off);
  };
  auto to = [&](int i, uint32_t off) {
    return reinterpret_cast<float*>(reinterpret_cast<char*>(dst + (size_t)i * P) + off);
  };
  const int outs = (x >= tkp->xs && x < tkp->xe) ? (tkp->xe - x < kV ? tkp->xe - x : kV) : 0;
  uint32_t mw[4] = {0u, 0u, 0u, 0u};
  // Copies one row's populations of the classes in `which` (bit 0: 2, 5, 6; bit 1: 0, 1, 3;
  // bit 2: 4, 7, 8) into shared memory; slot: of the two-row classes.
  auto load = [&](uint32_t row, int which, int slot) {
    if (chunk) {  // inactive lanes have none
#pragma unroll
      for (int i = 0; i < kQ; ++i) {
        if (!((which >> cls_of(i)) & 1)) continue;
        const int at = cls_of(i) == 1 ? 6 + in_cls(i) : (cls_of(i) == 0 ? 0 : 9) + in_cls(i);
        cpa16(own0 + at * R + (cls_of(i) == 1 ? 0 : slot * 3 * R), from(i, row));
      }
    } else if (active) {
#pragma unroll 1
      for (int j = 0; j < kV; ++j) {
        const uint32_t r = row + 4u * (uint32_t)(wrapped(p + j, nx) - p);
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
          if (!((which >> cls_of(i)) & 1)) continue;
          const int at = cls_of(i) == 1 ? 6 + in_cls(i) : (cls_of(i) == 0 ? 0 : 9) + in_cls(i);
          cpa4(own0 + 4 * j + at * R + (cls_of(i) == 1 ? 0 : slot * 3 * R), from(i, r));
        }
      }
    }
    if (lane == 0 || last) {  // the edge columns beyond the warp
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (!((which >> c) & 1)) continue;
        const uint32_t e = e0 + 4 * ((c == 1 ? 0 : slot * 8) + c);
        if (lane == 0) cpa4(e, from(c == 0 ? 5 : (c == 1 ? 1 : 8), row + 4u * (uint32_t)(pl - p)));
        if (last) cpa4(e + 16, from(c == 0 ? 6 : (c == 1 ? 3 : 7), row + 4u * (uint32_t)(pr - p)));
      }
    }
  };
  auto load_mask = [&]() {
    if (!active) return;
    if (chunk) {
      mw[0] = __ldg(mp + (pl >> 5));
      mw[1] = __ldg(mp + (p >> 5));
      mw[2] = __ldg(mp + (pr >> 5));
    } else {  // the row wraps inside the chunk or it is unaligned: words only, no dependent loads
      mw[0] = __ldg(mp + (pl >> 5));
      mw[1] = __ldg(mp + (p >> 5));
      mw[2] = __ldg(mp + (min(p + kV, nx - 1) >> 5));
      mw[3] = __ldg(mp);
    }
  };
  auto next_row = [&]() {  // advance the input row by one
    sp += 4u * pitch;
    mp += wpr;
    if (++ys == ny) {
      ys = 0;
      sp -= 4u * (uint32_t)ny * pitch;
      mp -= (size_t)ny * wpr;
    }
  };
  // solid bits of the row whose mask words were loaded last (those beyond an open end are
  // bits of other cells: they only reach populations that the completion replaces)
  auto window = [&]() -> uint32_t {
    if (!chunk) {
      uint32_t v = mw[1] >> (p & 31);  // cells p ... of the row
      if ((p & 31) > 32 - (kV + 1)) v |= mw[2] << (32 - (p & 31));
      const int in = nx - p;  // ... those before the wrap, then cells 0 ...
      if (in < kV + 1) {
        uint32_t w = mw[3];
        if (nx < kV) {  // rows that wrap more than once
          w &= (1u << nx) - 1u;
          w |= w << nx;
          w |= w << (2 * nx);
        }
        v = (v & ((1u << in) - 1u)) | (w << in);
      }
      return ((mw[0] >> (pl & 31)) & 1u) | ((v & ((1u << (kV + 1)) - 1u)) << 1);
    }
    return ((mw[0] >> (pl & 31)) & 1u) | (((mw[1] >> (p & 31)) & kOwn) << 1) |
           (((mw[2] >> (pr & 31)) & 1u) << (kV + 1));
  };
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // input row n of the sweep is the grid's row y0 - kT + n; iteration k pulls level 1 from
  // rows k (2, 5, 6), k + 1 (0, 1, 3) and k + 2 (4, 7, 8)
  uint64_t hist = 0;
  load(sp, 1, 0);
  load_mask();
  hist = (hist << 8) | window();
  next_row();
  load(sp, 7, 1);
  load_mask();
  hist = (hist << 8) | window();
  next_row();
  load(sp, 4, 0);
  load_mask();
  cpa_commit();

  const int iters = rows + 3 * kT - 3;
  int o0 = 0, o1 = 3 * R, o2 = 6 * R;  // three-row slots, oldest first
  int m0 = 0;                          // two-row slot of the older row
#pragma unroll 1
  for (int k = 0; k < iters; ++k) {
    hist = (hist << 8) | window();  // row n = k + 2
    const uint32_t sp2 = sp;        // row k + 2
    next_row();                     // -> row k + 3
    const bool more = k < rows + 2 * kT - 3;
    if (more) load_mask();
    if (group)
      asm volatile("bar.sync %0, %1;" ::"r"(group >> 8), "r"(group & 0xff) : "memory");
    else
      __syncwarp();
#pragma unroll 1
    for (int t = kT; t >= 1; --t) {
      if (k < 3 * (t - 1) || k > rows + 2 * kT + t - 4) continue;
      // the level's sources: row y - 1 of the upward populations, row y (and the own cells'
      // populations, for bounce-back), row y + 1 of the downward ones
      uint32_t su, ou, sm, sd, od, eu, em, ed;
      int east;  // edge values: west at e? + 4 class, east `east` bytes further
      const int b = k & 1;  // level 1: slot of rows k (2, 5, 6) and k + 2 (4, 7, 8)
      if (t == 1) {
        su = own0 + b * (3 * R);
        ou = own0 + (b ^ 1) * (3 * R);
        sm = own0 + 6 * R;
        sd = su + 9 * R;
        od = ou + 9 * R;
        eu = ed = e0 + b * 32;
        em = e0;
        east = 16;
        cpa_wait<0>();
        __syncwarp();
      } else {
        const uint32_t lv = own0 + (kRows0 + (t - 2) * kRows1) * R;
        su = lv + o0;
        ou = lv + o1;
        sm = lv + 9 * R + m0;
        od = lv + 15 * R + m0;
        sd = lv + 18 * R - m0;
        const uint32_t eb = edges + (t - 2) * (4 * kRing * kWarps * kEdge) + west_warp;
        eu = eb + ((k - 3) & (kRing - 1)) * (4 * kWarps * kEdge);
        em = eb + ((k - 2) & (kRing - 1)) * (4 * kWarps * kEdge);
        ed = eb + ((k - 1) & (kRing - 1)) * (4 * kWarps * kEdge);
        east = east_warp - west_warp;
      }
      // what the neighbouring warp (or the refill) left for lane 0 or the last lane
      const int side = lane == 0 ? 0 : east;
      const float edge[3] = {ld_s(eu + side), ld_s(em + side + 4), ld_s(ed + side + 8)};
      float2 s[3][3][kH];  // source chunks by class and member
      float l[3], r[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const uint32_t row = c == 0 ? su : (c == 1 ? sm : sd);
#pragma unroll
        for (int q = 0; q < 3; ++q) ld_chunk(row + q * R, s[c][q]);
        // members: straight, then 5 1 7 / 6 3 8
        const float lw = __shfl_up_sync(0xffffffffu, s[c][c == 2 ? 2 : 1][1].y, 1);
        const float rw = __shfl_down_sync(0xffffffffu, s[c][c == 2 ? 1 : 2][0].x, 1);
        l[c] = lane == 0 ? edge[c] : lw;
        r[c] = last ? edge[c] : rw;
      }
      const uint32_t w = (uint32_t)(hist >> (16 * (t - 1)));  // windows of rows y + 1, y, y - 1
      float2 g[kQ][kH];
      if (__any_sync(0xffffffffu, w & kNear)) {
        pull_row<1, true>(w >> 16, od, s[0], l[0], r[0], g);
        pull_row<0, true>(w >> 8, sm, s[1], l[1], r[1], g);
        pull_row<-1, true>(w, ou, s[2], l[2], r[2], g);
      } else {
        pull_row<1, false>(0u, 0u, s[0], l[0], r[0], g);
        pull_row<0, false>(0u, 0u, s[1], l[1], r[1], g);
        pull_row<-1, false>(0u, 0u, s[2], l[2], r[2], g);
      }
      if (t == 1) {
        // the rows this lane no longer needs are refilled: populations 2, 5, 6 and 0, 1, 3
        // of row k + 2, populations 4, 7, 8 of row k + 3
        if (more) {
          load(sp2, 3, b);
          load(sp, 4, b ^ 1);
        }
        cpa_commit();
      }
      if (at_end) complete_ends(dw, de, kinds, west, je, g);
      collide_lane<FORCED>(G, om, one, g);
      if (t == kT) {  // the pass's result: solid cells store 0
        if (outs) {
          const uint32_t own = w >> 9;
          if (own & kOwn) {
#pragma unroll
            for (int j = 0; j < kV; ++j) {
              const bool solid = (own >> j) & 1u;
#pragma unroll
              for (int i = 0; i < kQ; ++i) set2(g[i], j, solid ? 0.0f : get2(g[i], j));
            }
          }
          if (outs == kV) {
#pragma unroll
            for (int i = 0; i < kQ; ++i) st_chunk(to(i, dp), g[i]);
          } else {
#pragma unroll
            for (int j = 0; j < kV - 1; ++j)
              if (j < outs) {
#pragma unroll
                for (int i = 0; i < kQ; ++i) to(i, dp)[j] = get2(g[i], j);
              }
          }
        }
        dp += 4u * pitch;
      } else {  // keep the level's new row, publish its edge columns
        const uint32_t lv = own0 + (kRows0 + (t - 1) * kRows1) * R;
#pragma unroll
        for (int i = 0; i < kQ; ++i)
          st_chunk_s(lv + in_cls(i) * R + (cy_of(i) > 0 ? o0 : (cy_of(i) == 0 ? 9 : 15) * R + m0), g[i]);
        const uint32_t e = edges + (t - 1) * (4 * kRing * kWarps * kEdge) +
                           (k & (kRing - 1)) * (4 * kWarps * kEdge) + warp * (4 * kEdge);
        if (last) {
          st_s(e, g[5][1].y);
          st_s(e + 4, g[1][1].y);
          st_s(e + 8, g[8][1].y);
        }
        if (lane == 0) {
          st_s(e + 12, g[6][0].x);
          st_s(e + 16, g[3][0].x);
          st_s(e + 20, g[7][0].x);
        }
      }
    }
    const int tmp = o0;
    o0 = o1;
    o1 = o2;
    o2 = tmp;
    m0 = 3 * R - m0;
  }
}

// rcp_lane of n values, four (a lane's) a thread; the last thread's missing ones are 1.
__global__ void k_rcp_eval(const float* __restrict__ x, float* __restrict__ y, size_t n) {
  const size_t at = 4 * (blockIdx.x * (size_t)blockDim.x + threadIdx.x);
  if (at >= n) return;
  float v[4];
  for (int j = 0; j < 4; ++j) v[j] = at + j < n ? x[at + j] : 1.0f;
  const float2 rho[kH] = {make_float2(v[0], v[1]), make_float2(v[2], v[3])};
  float2 inv[kH];
  rcp_lane(rho, inv);
  for (int j = 0; j < 4; ++j)
    if (at + j < n) y[at + j] = get2(inv, j);
}

constexpr size_t kSmem =
    sizeof(float) * ((size_t)kWarps * kWarpFloats + (size_t)(kT - 1) * kRing * kWarps * kEdge);

}  // namespace

// Strips of one grid's rows: `slots` warps (1, 2 or 4) a strip, output columns split into
// chunks of four as evenly as they go.
struct Strips {
  int slots, n;
  bool whole;  // the whole row in one group: no halo columns
};
static Strips strips_of(const GridDev& d) {
  const int nc = (d.nx + kV - 1) / kV;
  Strips best{0, 0, false};
  int cost = 1 << 30;
  for (int g = 1; g <= kWarps; g *= 2) {
    const int cap = 32 * g;
    Strips s{g, 0, false};
    if (nc <= cap && (!d.periodic_x || (d.nx % kV == 0 && nc > 1))) {
      s.n = 1;
      s.whole = true;
    } else if (d.periodic_x) {
      s.n = (nc + cap - 2 * kHalo - 1) / (cap - 2 * kHalo);
    } else {
      // the two end strips need a halo on one side only
      const int inner = nc - 2 * (cap - kHalo), c = cap - 2 * kHalo;
      s.n = 2 + (inner > 0 ? (inner + c - 1) / c : 0);
    }
    if (s.n * g < cost) {
      cost = s.n * g;
      best = s;
    }
  }
  return best;
}

void sweep_plan(const std::vector<GridDev>& gd, std::vector<SweepTask>* tasks) {
  // Rows a task advances: the cut whose waves of CTAs take the fewest row steps.  A task of l
  // rows costs l + 3 row iterations of level 2 (l + 2 of level 1) and a start of about two
  // more, so many small cuts lose to one wave of large ones: 64 grids of 512 x 256 at 36 rows
  // (one wave of 448 CTAs) 58 us a step, at 30 rows (1.3 waves) 72, at 64 rows 96.
  int max_ny = 0;
  std::vector<Strips> strips;
  for (const GridDev& d : gd) {
    strips.push_back(strips_of(d));
    max_ny = std::max(max_ny, d.ny);
  }
  const long long cap = kSweepSms * kWarps * kCtas;
  int best_l = max_ny;
  double best = 1e300;
  for (int l = max_ny; l >= 1;) {
    long long w = 0;
    for (size_t k = 0; k < gd.size(); ++k)
      w += (long long)strips[k].n * strips[k].slots * ((gd[k].ny + l - 1) / l);
    const double c = (double)((w + cap - 1) / cap) * (l + 5);
    if (c < best) {
      best = c;
      best_l = l;
    }
    if (l == 1) break;
    const int segs = (max_ny + l - 2) / (l - 1);  // the next cut of the tallest grid
    l = std::min(l - 1, (max_ny + segs - 1) / segs);
  }
  tasks->clear();
  for (int g = kWarps; g >= 1; g /= 2) {  // larger groups first: slots stay aligned
    for (size_t k = 0; k < gd.size(); ++k) {
      const GridDev& d = gd[k];
      const Strips& s = strips[k];
      if (s.slots != g) continue;
      const int nc = (d.nx + kV - 1) / kV;
      const int segs = (d.ny + best_l - 1) / best_l;
      for (int q = 0; q < segs; ++q) {
        const int ya = (int)((long long)d.ny * q / segs), yb = (int)((long long)d.ny * (q + 1) / segs);
        for (int u = 0; u < s.n; ++u) {
          // output chunks [ca, cb) of the strip; the end strips of open grids have one halo
          // chunk less and take one output chunk more
          auto bound = [&](int i) -> int {
            if (i <= 0) return 0;
            if (i >= s.n) return nc;
            if (d.periodic_x) return (int)((long long)nc * i / s.n);
            return (int)(kHalo + (long long)(nc - 2 * kHalo) * i / s.n);
          };
          const int ca = bound(u), cb = bound(u + 1);
          const bool hl = !s.whole && (d.periodic_x || u > 0);
          const bool hr = !s.whole && (d.periodic_x || u + 1 < s.n);
          const int first = ca - (hl ? kHalo : 0), end = cb + (hr ? kHalo : 0);
          const int nw = (end - first + 31) / 32;
          const int base = (int)(tasks->size() % kWarps);
          for (int w = 0; w < g; ++w) {
            SweepTask t{};
            if (w < nw) {
              t.grid = (int)k;
              t.v0 = kV * (first + 32 * w);
              t.xs = kV * ca;
              t.xe = std::min(kV * cb, d.nx);
              t.y0 = ya;
              t.rows = yb - ya;
              t.last = (short)std::min(31, end - first - 32 * w - 1);
              t.nwarps = (short)nw;
              t.bar = (short)(1 + base);
              const bool wrap = s.whole && d.periodic_x;
              const int lw = w > 0 ? w - 1 : (wrap ? nw - 1 : w);
              const int rw = w + 1 < nw ? w + 1 : (wrap ? 0 : w);
              t.left = (short)(base + lw);
              t.right = (short)(base + rw);
            }
            tasks->push_back(t);
          }
        }
      }
    }
  }
  while (tasks->size() % kWarps) tasks->push_back(SweepTask{});
}

// Estimated times in us, fitted to 1,493 batches of 2,000 to 16 M cells (24 to 8,192 columns, 1 to
// 100 grids; periodic rows with and without a force, open rows with sparse and dense disks) with a
// spread of 5% (step, in its fastest shape) and 6% (pass).
//  * A single step costs its launch and then the row segments of 128 columns a multiprocessor
//    steps, more once its tiles need a second wave.
//  * A pass costs its launch and, a wave of CTAs, rows + 2 iterations of both levels, whose
//    length is mostly latency: three CTAs on a multiprocessor take 1.5 times as long as one.  A
//    force makes the collision longer, rows that wrap inside a chunk copy their cells one by one,
//    open rows complete their ends, and rows of up to 40 columns leave three quarters of the
//    lanes idle.
// So passes lose where rows are just too many for one wave of one-row tasks and a single step is
// still one wave (eight forced grids of 180 x 119: 6.4 us a step, 7.2 in passes; 20 grids of 122 x
// 120: 7.3 and 9.3), and on many narrow or ragged rows.  Taken from an estimated gain of 4% on.
// Of 1,000 other batches 879 take passes then, 12 of them at less than 0.98 of the speed of single
// steps (0.91 the least), and 24 of the other 121 would gain more than 10%.  After lbm_autotune,
// which times both, 918 take passes, 6 at less than 0.98 (0.97), and 2 of the others would gain more
// than 2% (8%).  It takes an estimate of 1.2 or more as it is: of 845 such batches the least gain
// was 1.02.
double sweep_gain(const std::vector<GridDev>& gd, const std::vector<SweepTask>& tasks, bool one_wave) {
  double cells = 0, segs = 0, forced = 0, ragged = 0, open = 0, narrow = 0;
  for (const GridDev& d : gd) {
    const double c = (double)d.nx * d.ny;
    cells += c;
    segs += (double)d.nseg * d.ny;
    if (d.fx != 0.0f || d.fy != 0.0f) forced += c;
    if (d.periodic_x && d.nx % kV != 0) ragged += c;
    if (!d.periodic_x) open += c;
    if (d.nx <= 40) narrow += c;
  }
  forced /= cells;  // shares of the cells
  ragged /= cells;
  open /= cells;
  narrow /= cells;
  const double w = segs / kSweepSms;  // row segments a multiprocessor
  const double step = (one_wave ? 4.79 + 0.12 * w : 3.46 + 0.22 * w) + forced * (0.45 + 0.03 * w) +
                      0.31 * ragged;
  int rows = 0;
  for (const SweepTask& t : tasks) rows = std::max(rows, t.rows);
  const int wave = kSweepSms * kCtas, ctas = (int)(tasks.size() / kWarps), full = (ctas - 1) / wave;
  const int last = (ctas - wave * full + kSweepSms - 1) / kSweepSms;  // CTAs a multiprocessor, last wave
  static const double base[4] = {0, 1.71, 2.32, 2.51}, force[4] = {0, 0.44, 0.73, 0.85};
  const double kind = 0.86 * ragged + 0.44 * open + 0.41 * narrow;
  auto iteration = [&](int k) { return base[k] + force[k] * forced + kind; };
  const double pass = 1.56 + (rows + 2) * (full * iteration(kCtas) + iteration(last));
  return kSweepSteps * step / pass;
}

int sweep_init() {
  cudaError_t e = cudaFuncSetAttribute(k_sweep<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_sweep<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kSmem);
  return e == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

int sweep_launch(Handle* h, const float* src, float* dst, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)h->sweep_ctas);
  cfg.blockDim = dim3(kWarps * 32);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  bool forced = false;
  for (const GridDev& d : h->gd) forced = forced || d.fx != 0.0f || d.fy != 0.0f;
  auto kernel = forced ? k_sweep<true> : k_sweep<false>;
  LBM_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kernel, (const GridDev*)h->gd_d,
                                    (const SweepTask*)h->sweep_d, (const uint32_t*)h->mask, src,
                                    dst, (unsigned)h->gd[0].plane, 1.0f));
  return LBM_OK;
}

}  // namespace lbmfno

using namespace lbmfno;

extern "C" int lbm_reciprocal_eval(const float* x_d, float* y_d, size_t n, void* stream) {
  LBM_REQUIRE(n == 0 || (x_d != nullptr && y_d != nullptr), "lbm_reciprocal_eval: null buffer");
  LBM_REQUIRE(n <= (size_t)1 << 32, "lbm_reciprocal_eval: n must be at most 2^32");
  if (n == 0) return LBM_OK;
  k_rcp_eval<<<(unsigned)((n + 1023) / 1024), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(x_d, y_d, n);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}
