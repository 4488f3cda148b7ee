// step.cuh -- everything of a DD step that is O(N): nodal forces and glide
// velocities from the pair stage's parts, the Lp / rho sample of the step-start
// state, the Euler update and the next step's source records.  One network and
// a batch of realisations are the same thing here (one network: R = 1).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "ptadd_internal.cuh"

namespace ptadd {

// What a launch does, in this order.  All of it in one launch needs groups that
// hold whole loops (StepGroups::whole); otherwise a launch per phase orders the
// reads of neighbours in other blocks.
enum : int {
    STEP_NODE = 1,        // forces, lumped velocities of the unpinned nodes (0 at pinned ones)
    STEP_CONSISTENT = 2,  // instead of the lumped velocities, the consistent mobility's
    STEP_EULER = 4,       // sums, Euler update into pos_next
    STEP_PREP = 8,        // records of the moved segments (with STEP_EULER)
    STEP_ROWS = 16,       // STEP_CONSISTENT in parts: only set the rows of the system up
};

struct StepArgs {
    int64_t n = 0;
    const double* pos = nullptr;
    double* pos_next = nullptr;
    const int32_t *nxt = nullptr, *prv = nullptr, *loop_of = nullptr;
    const double *loop_b = nullptr, *loop_n = nullptr;
    const int64_t* loop_off = nullptr;
    const uint8_t* pinned = nullptr;
    const int32_t* grp_off = nullptr;   // [groups + 1] first node of each group
    const int32_t* real_of = nullptr;   // per node; null: one network
    const int64_t* node_off = nullptr;  // [R + 1]
    const int64_t* fp_base = nullptr;   // [R] first value of the realisation's parts
    const int32_t* chunks_of = nullptr; // [R]
    int chunks = 0;                     // one network
    const double* fpart = nullptr;
    double* vel = nullptr;  // written and read in one launch: never through the read-only cache
    double* scr = nullptr;  // [10 n]: rows of the consistent system, two copies
    double* src = nullptr;
    float *src32 = nullptr, *srcdf = nullptr;
    const double* origin = nullptr;     // [3 R]; null: org
    double org[3] = {0.0, 0.0, 0.0};
    double a2 = 0.0, dt = 0.0;
    double* part = nullptr;             // [16 groups] running sums weighted by dt: L b (x) (t x vbar) (9), L,
                                        // L vbar (3); [13] this step's L
    int* flag = nullptr;                // non-finite positions
    unsigned* counter = nullptr;        // the batch's work counter, reset for the next pair launch (or null)
};

// Groups of consecutive nodes, a block each: whole loops of one realisation, up
// to 32 nodes together, as long as no loop has more than STEP_LOOP_MAX nodes (a block walks a
// longer loop 32 nodes at a time); otherwise 32 nodes wherever the loops end, and a launch per
// phase: two a step, eight with the consistent mobility.  us a step in whole loops / split, two loops of n nodes
// in FP64: lumped, n = 64 47 / 38, 128 105 / 54, 256 160 / 84, 400 313 / 135; consistent 64 54 / 64,
// 128 114 / 80, 256 174 / 111, 400 337 / 170.  Eight loops of 256 in mixed precision: lumped 247 / 198,
// consistent 260 / 224.  The line could lie lower: a block's walk of a long loop is the chain.
constexpr int STEP_LOOP_MAX = 256;
struct StepGroups {
    std::vector<int32_t> off;       // [groups + 1]
    std::vector<int32_t> real_grp;  // [R + 1] first group of each realisation
    bool whole = true;
};
StepGroups step_groups(int64_t n_loops, const int64_t* loop_off, int32_t R, const int64_t* node_off);

// The phases of one step that follow the pair stage; junctions (which act on
// the velocities) split it with `what`.  Adds the number of launches.  chained: in a chain of
// kernels that all wait for the one before (chain.cuh).
cudaError_t launch_step(const StepArgs& a, int n_groups, bool whole, int max_chunks, int what, cudaStream_t st,
                        int64_t* launches, bool chained = false);
// Nodal forces of every node (F, SoA [3 n]) from the pair stage's parts; 0 at pinned nodes of a batch,
// whose segments may not have been evaluated.
cudaError_t launch_node_force(const StepArgs& a, double* force, cudaStream_t st);
// Adds the groups' running sums to acc[16 r + ..] (slots 0..8 Lp, 9 rho, 13..15 polar
// velocity); length_only: instead, the step's line length into slot 11 (junction
// jumps weight it).
cudaError_t launch_step_finish(int32_t R, const int32_t* real_grp, const double* part, bool length_only, double* acc,
                               cudaStream_t st);

}  // namespace ptadd
