// Device-resident state of the batched / served CJM engine (shared by engine.cu and
// batch.cpp).  Each admitted problem occupies one slot; every kernel of an engine step
// reads the slots' phases from device memory, so one captured CUDA graph of steps serves
// whatever set of problems is admitted when it is replayed.
#pragma once

#include <vector>

#include "cj_internal.h"

// Engine tile: the unit of work of every engine kernel, kEngTX columns x (per slot) ty rows of
// nodes; ty is 16, 32 (the default) or 64, chosen per stencil and size class by
// cj_autotune_engine.
constexpr int kEngTX = 128, kEngTYDefault = 32;

enum SlotPhase : int {
    PHASE_FREE = 0,     // unused
    PHASE_OUTER = 1,    // next step: correction (after the first cycle) + defect + stop test
    PHASE_SWEEP = 2,    // inner FP32 cycle in progress
    PHASE_DONE = 3,     // stopped; the next step copies u to the caller's buffer
    PHASE_RETIRED = 4   // result delivered; the host may release the slot
};

struct SlotDev {
    // set at admission
    int Nx, Ny, st, mode;          // mode: CJ_FP32_INNER or CJ_FP32_INNER_DD
    int depth, ntx, ntiles, ty;    // depth: sweeps per sweep launch; ty: tile rows
    int plain;                     // 1: one sweep per launch over the tile list
    long long M_in, max_outer;
    double tol, S, h2;
    Grid g64, g32;
    double *u, *ulo, *b;           // padded FP64 (ulo: CJ_FP32_INNER_DD only)
    float *e0, *e1, *rt;           // padded FP32
    const float *w32;              // inner-cycle weights, M_in of them
    double *part;                  // 3 doubles per tile
    double *out;                   // caller's device grid for the result
    long long ld_out;
    // evolving
    int phase, status, cur, stall;
    long long counter, outer, sweeps;
    double prev, rho, rinf, fl, bsq, bmax;
};

// Compact per-slot record the host polls after each replay.
struct SlotStatus {
    int phase, status;
    long long sweeps, outer;
    double rho, rinf, fl;
};

// Register-tile lists of an engine: stencil x shape (short or tall tiles), one kernel each; and the
// list of the slots that were asked to sweep once per launch, which run on the tile list.
constexpr int kEngLists = 6, kEngPlain = 6, kEngBranches = 7;

struct EngineDev {
    SlotDev *slots;        // max_slots entries
    int max_slots;
    int2 *tiles;           // (slot, tile index within the slot)
    int *ntiles;           // device counter of valid entries in tiles
    int4 *items;           // register-tile items (slot, first column, first row, last row), by list
    int *item_off;         // kEngLists + 1 offsets of the lists in items
    SlotStatus *status;    // max_slots entries, refreshed by the advance kernel
    double one;            // 1 (additions as fused multiply-adds)
};

// Streams and events of an engine's step: the lists' sweeps are branches of its graph, forked after
// `decide` and joined before `export`.
struct EngineBranches {
    cudaStream_t side[kEngBranches] = {};
    cudaEvent_t fork = nullptr, join[kEngBranches] = {};
};

// launchers (engine.cu)
// one engine step: correct, defect, decide, `sweeps` sweep launches of every list in `lists` (a bit
// per list; register tiles with rt_blocks blocks), export, advance (the step's sweeps applied at once)
cudaError_t eng_launch_step(const EngineDev &e, int grid_tiles, int grid_slots, unsigned lists, int rt_blocks,
                            const EngineBranches &br, int sweeps, cudaStream_t s);
// The register-tile list of a problem, and its items appended; depth: the slot's sweeps per launch.
int eng_list(int st, int Nx, int Ny);
void eng_rt_items(int slot, int Nx, int Ny, int st, int depth, std::vector<int4> &items);
// The list whose sweep kernel fn is, or -1.
int eng_list_of_kernel(const void *fn);
// Sweeps per launch of a problem that does not name them: 8, or 4 of 17 points.
int eng_default_depth(int st);
cudaError_t eng_launch_import(const EngineDev &e, int slot, int ntiles, const double *f,
                              long long ldf, const double *u0, long long ldu, cudaStream_t s);
// true for the kernels that loop over the tile list (their grid may be any size; the sweep among them)
bool eng_is_tile_kernel(const void *fn);
// the sweep kernels' shared-memory limits on the current device
cudaError_t eng_prepare();
