// On-chip Jacobi-PCG (resident.cu): what the solver entry points need of it.
#pragma once

#include <vector>

#include "solver.cuh"

namespace gb {

constexpr int kResThreads = 512;
constexpr int kResMaxCtas = 160;  // bricks of one problem (GB300 has 152 SMs)
constexpr int kResSlotVals = 4;   // 16-byte slots per CTA and grid sum
constexpr int kResFlagStride = 8;  // words between two CTAs' face flags
// two buffers of slots, then the flags, then a batch's count of CTAs that have come to the problem
constexpr size_t kResSlotBytes =
    (size_t)2 * kResMaxCtas * kResSlotVals * 16 + (size_t)kResMaxCtas * kResFlagStride * 4 + 32;

// How a grid is cut: sx x sy x sz bricks of 4 bx4 x by x bz points, each
// thread of a CTA holding one four-point vector in x over `depth` planes
// (cols = bx4 by vector columns, zseg runs of planes per column).
struct ResPlan {
    int build;  // which instance of the kernel (resident.cu)
    int sx, sy, sz, bx4, by, bz, cols, zseg, depth, G;
    int dplanes;  // planes of d held in shared memory
    size_t smem;
    double cycles;  // estimated SM cycles of one iteration
};

// Whether one solve of this grid runs on chip (constant coefficients), and its plan.
bool resident_fits(const gbpcg_grid &g, ResPlan *plan);

// Instead of a status: nothing has been solved, and the problem is to be streamed (or launched alone).
constexpr int kResNoRoom = -1;

// The whole solve, enqueued on s; its scalars go to *st (DEVICE), or to the workspace's state block.
// kResNoRoom where the context may not use the SMs of the plan.
int resident_launch(const SolveCall &c, const ResPlan &plan, cudaStream_t s, SolveState *st = nullptr);

// The same solve driven from the host, which reads the device's stop flag after every iteration (kResNoRoom
// as above).
int resident_host_loop(const SolveCall &c, const ResPlan &plan, cudaStream_t s);

// Which problems of a batch run here, all in one launch or one by one, and which in the streaming
// kernels (numbers into grids).
struct ResidentChoice {
    std::vector<int> in_batch, alone, rest;
};
ResidentChoice resident_choice(int n, const gbpcg_grid *grids);

// One launch of calls[0 .. n) (ResidentChoice::in_batch) on s.  states: DEVICE, one per problem; tables:
// DEVICE scratch (kResNoRoom if it is too small, or the context may not use every SM).
int resident_batch_launch(int n, const SolveCall *calls, SolveState *states, char *tables, size_t table_bytes, int io,
                          cudaStream_t s);

// The same with the bricks and threads of the standalone solves, whose bits the results have; one launch
// per build of the kernel, problems side by side where they leave each other room.
int resident_standalone_launch(int n, const SolveCall *calls, SolveState *states, char *tables, size_t table_bytes,
                               int io, cudaStream_t s);

struct ResProb {
    int nx, ny, nz, nxp;  // nxp: row pitch of zg and pg, nx rounded up to a multiple of 4
    int sx, sy, sz, bx4, by, bz, zseg, depth, cols, G, dplanes;
    OpConst op;  // times unit
    float unit;  // a power of two
    int maxit, iters;           // iters: iterations this launch may take
    int resume, save, final_x;  // host-driven loop: state from / to the workspace; final x update
    unsigned seq0;              // number of the last grid sum before this launch's
    double cx, cy, cz, tol;
    const void *b;
    void *x;
    float *zg;  // r on brick faces, padded rows (all of r after a residual)
    float *pg;     // p of a host-driven loop between launches
    float4 *dlin;  // d, brick by brick, each thread's vectors a brick's thread count apart
    SolveState *st;
    ulonglong2 *slots;
    unsigned *flags;      // per CTA: number of the sum its face values belong to
    unsigned *arrived, *progress;  // batches: CTAs that have come to this problem; steps of any problem
    ulonglong2 *inbox;    // NULL, or every CTA's own slots of the loop's sums (grid_sum_pair)
};

}  // namespace gb
