// Multi-step passes of the LBM (lbm_sweep.cu): task table and launch, used by lbm.cu.
#pragma once

#include <vector>

#include "common.cuh"

namespace lbmfno {

constexpr int kSweepSteps = 2;   // time steps of one pass
constexpr int kSweepWarps = 4;   // warps a CTA
constexpr int kSweepSms = 152;   // multiprocessors the task table is cut for

// What one warp of a sweep does: rows y0 .. y0 + rows - 1 of a strip of columns.
struct SweepTask {
  int grid;
  int v0;        // virtual column of lane 0's first cell (a multiple of 4)
  int xs, xe;    // columns the strip writes
  int y0, rows;  // rows == 0: unused slot
  short last;    // last active lane
  short nwarps, bar;  // warps of the group; its named barrier
  short left, right;  // neighbouring warps (CTA-relative)
};
static_assert(sizeof(SweepTask) == 36, "task table entry");

struct Handle;
// Tasks of a batch, kSweepWarps a CTA.  Host only, a function of the grids alone.
void sweep_plan(const std::vector<GridDev>& gd, std::vector<SweepTask>* tasks);
// Estimated time of two single steps over that of a pass of these tasks; one_wave: a single step's
// tiles are resident at once in some shape.  Host only.
constexpr double kSweepGain = 1.04;  // from here on lbm_step takes passes
constexpr double kSweepSure = 1.2;   // ... and lbm_autotune does not measure
double sweep_gain(const std::vector<GridDev>& gd, const std::vector<SweepTask>& tasks, bool one_wave);
int sweep_init();
int sweep_launch(Handle* h, const float* src, float* dst, cudaStream_t s);

}  // namespace lbmfno
