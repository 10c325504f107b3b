// The one-launch build of a tree's levels (hgmm_levels.cu).
#pragma once

#include "hgmm_internal.cuh"

namespace hgmm {

constexpr int LV_CTAS_PER_SM = 3;  // as the level-wide E-step: one CTA per chunk of its grid

// levels with at least this many parents, of at most LOCAL_EM_POINTS points
// on average, run their EM parent by parent
constexpr int LOCAL_EM_PARENTS = 256;
constexpr int64_t LOCAL_EM_POINTS = 2048;

struct LevelsArgs {
    const float4* pts;
    int n;
    int levels;                  // levels 0 .. levels - 1 are built
    int em_iters;
    int stop_level, stop_iters;  // stop after stop_iters EM iterations of level stop_level - 1 (0: off)
    float n_min, lam_c, eps_rel;
    int n_chunks;                // chunks of the level-wide E-step's grid
    NodeEst* est;
    NodeStat* stat;
    float4* rnode;
    int* seg_start;
    int* seg_count;
    RootDev* root;
    float* root_part;
    float4* buf[2];
    int* perm[HGMM_MAX_DEPTH];
    float2* part;                // 2 x part_stride: the runs' partials, by iteration parity
    int64_t part_stride;
    float2* slices;              // 2 x slice_stride
    int64_t slice_stride;
    int* item_cnt;
    unsigned* cnt;               // levels_counters() words
    int* status;
};

int64_t levels_slots(int64_t n);
int levels_counters();
bool levels_smem_attr();
int levels_taken(int64_t n, int depth, int est_grid);
// HGMM_OK, HGMM_ECUDA, or LEVELS_REFUSED: the device cannot hold the launch's
// CTAs at once (a context that owns part of its SMs), nothing has run, and the
// level-wide launches, which need no co-residency, build the tree.  refuse:
// checking aid, asks for more CTAs than any device holds.
constexpr int LEVELS_REFUSED = 1;
int levels_launch(LevelsArgs& a, int est_grid, bool refuse, cudaStream_t s);

}  // namespace hgmm
