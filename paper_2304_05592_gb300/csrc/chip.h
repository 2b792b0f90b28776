// chip.h -- interface of the on-chip 2D time loop (step2d_chip.cu).
#pragma once

#include "internal.h"

namespace wave {

constexpr int kMaxCluster = 16;
constexpr int kChipTable = 4096;  // steps of one launch that may name a buffer each

enum : int { kKeepNone = 0, kKeepTable = 1, kKeepRows = 2 };

// One launch: nsteps consecutive forward or adjoint steps of every shot.
struct ChipArgs {
    const float* kap;     // [cell]
    float* pool;          // buffers of `field` floats ([nshot][cell])
    long long field, cell;
    int Nx, Nz, P, nb, nx, nz;
    float ceps;
    // split of a shot over its cluster (filled by launch_chip)
    int Q, C, NC, Rmax, cap_inj, cap_gat, add_rows;
    int z0[kMaxCluster + 1];
    // time: forward steps first, first + 1, ... (u^n -> u^{n+1}); adjoint steps
    // first, first - 1, ... (-> mu^k)
    int first, nsteps;
    int cur, prev;        // pool buffers of the current and previous level at the start (-1: zero)
    int out_last, out_prev;  // pool buffers of the last two levels made (-1: not kept)
    // forward: which levels are kept: buffer tab[i] after step i, or buffer
    // row0 + n + 1; a BF16 copy of level n + 1 in row n + 1 of st16
    int keep_mode, row0;
    __nv_bfloat16* st16;
    // adjoint with imaging: the forward level of step i in pool buffer tab[i],
    // or that of step k in row k of uf16
    const __nv_bfloat16* uf16;
    int g_buf;            // gradient accumulators, one per shot
    float* tacc;          // the injected taps' imaging terms, summed apart ([taps])
    TapList inj, gat;
    const float *amp_a, *amp_b;
    float* slots;
    int rec_from;         // forward: levels made by steps n >= rec_from are gathered
    long long cps;        // tap cells per shot
    int* err;
    short tab[kChipTable];
};

// Forward steps (levels kept in FP32 or not at all, or every level in BF16),
// adjoint steps (without imaging, or with the forward level in FP32 / BF16).
enum : int { kChipForward = 0, kChipFwdBF16 = 1, kChipAdjoint = 2, kChipAdjF32 = 3, kChipAdjBF16 = 4, kChipModes = 5 };

// How a problem is split, or C = 0 if the on-chip loop cannot take it (grid too
// large for a cluster's shared memory, too many taps in one strip, clusters
// not available).
struct ChipPlan {
    int mode = 0, C = 0, shape = 0, NC = 0, threads = 0, Rmax = 0, cap_inj = 0, cap_gat = 0, add_rows = 0;
    int z0[kMaxCluster + 1] = {};
    size_t smem = 0;
    float step_us = 0.0f;  // estimated time of one step of all shots
};
// (inj and gat keep their taps per strip for the next plan of the call)
ChipPlan chip_plan(const Dims& d, const Tiling& t, int nshot, int mode, HostTaps& inj, HostTaps& gat);
void launch_chip_tap_gradient(const TapList& l, int nt, long long cell, const float* tacc, float* g, cudaStream_t s);
cudaError_t launch_chip(const ChipPlan& p, ChipArgs& a, int nshot, cudaStream_t s);

// Restricts chip_plan to one shape (index into kShapes, -1: any) and one cluster
// size (0: any), so that tests reach every instantiation: the estimate takes one per
// problem.  refuse: launches ask for more shared memory than there is, which the CUDA
// runtime refuses on the host, so that tests see how a failed launch is reported.  Per
// host thread; nothing else sets it.
struct ChipForce {
    int shape = -1, C = 0;
    bool refuse = false;
};

}  // namespace wave

extern "C" int wave_chip_force(int shape, int clusters, int refuse);  // returns the number of shapes
