// lbm_march.cuh -- declarations of the multi-step collide-stream kernel
// (lbm_march.cu): one pass over the grid advances it by MARCH_STEPS steps.
#pragma once

#include <vector>

#include "lbm_internal.cuh"

namespace gblbm {

constexpr int MARCH_STEPS = GROUP_STEPS;  // steps of one pass
constexpr int MARCH_HALO = 4;             // columns computed but not stored on each side of a strip (>= steps - 1)

struct MarchArgs {
    StepArgs s;                  // src = b(t), dst = b(t + steps); grid, boundary and collision parameters; the counters
    void *mid[MARCH_STEPS - 1];  // b(t + 1) .. b(t + steps - 1), rows keep[2]..keep[3] of the grid
    long long mid_plane;         // elements between two planes of a mid buffer
    int out_w;                   // columns a strip stores
    const int2 *units;           // [n_units] the work of each CTA: strip, first row | rows << 16
    int n_units;
    int bounce[4];               // columns x0..x1, rows y0..y1 with a solid node in them or next to them (x0 > x1: none)
    int keep[4];                 // columns x0..x1, rows y0..y1 whose intermediate states are stored (x0 > x1: none)
};

// Strips of the multi-step kernel for a grid (each stores out_w columns) and
// the rows that a CTA takes, away from the body and the edges.
struct MarchPlan {
    int out_w = 0, strips = 0, rows = 0;
};
// Whether a channel grid of this storage type takes multi-step passes.
bool march_grid(int storage, int nx, int ny);
// Resident CTAs per SM of the multi-step kernel.
int march_slots(int storage);
// units receives the work of every CTA (MarchArgs::units), the longest first.
MarchPlan march_plan(int storage, int nx, int ny, int sm_count, const int *bounce, const int *keep,
                     std::vector<int2> *units);
// map: a tensor map over the source buffer viewed as [9][ny][pitch] whose box
// is march_box_columns(storage) columns of one row of all nine planes
cudaError_t launch_march(int storage, const MarchArgs &a, const void *map, cudaStream_t st);
int march_box_columns(int storage);
// *ctr = t
cudaError_t launch_set_counter(long long *ctr, long long t, cudaStream_t st);

// Control-volume partial rows of the steps of a pass, as the single-step
// kernel would have written them: step j reads state[j] and state[j + 1].
struct CvArgs {
    StepArgs s;                              // grid, boundary, box and tiles (src, dst, partials unused)
    const void *state[GROUP_STEPS + 1];      // post-collision states of the pass
    long long plane[GROUP_STEPS + 1];
    double *partials[GROUP_STEPS];
};
// priority: as launch_link_force
cudaError_t launch_cv_sums(int storage, const CvArgs &a, cudaStream_t st, int priority);

}  // namespace gblbm
