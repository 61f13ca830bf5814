// kernels.h -- host-side launchers of the libmpcd kernels (internal).
#pragma once
#include <cstddef>
#include <cuda_runtime.h>

#include "mpcd_internal.cuh"

namespace mpcd {

// ---- fused step on cell rows (k_cells.cu) ----
// mode: MODE_P stream + bin, MODE_F collide + stream + bin, MODE_C collide in place.
// variant = (thermostat ? 1 : 0) | (solute beads or walls ? 2 : 0) |
// (Andersen rule ? 16 : 0) | (angular-momentum correction ? 32 : 0); the last
// two without solute or walls.
int cells_blocks_per_sm(bool mixed, int variant, int mode);
void launch_cells(bool mixed, int variant, int mode, const BoxDev* boxes, const int2* spans,
                  int nspans, int grid, int* err, cudaStream_t s);
// The same step for mixed-model boxes without walls, members spread over the
// lanes of a warp (k_cells_warp.cu); valid for row capacities up to
// WARP_MAX_K and boxes below 2^22 cells per axis.  force: nonzero body force;
// beads: the box has solute beads; at: Andersen-thermostat rule (Eq. at)
// instead of the rotation (thermo is then false).
constexpr int WARP_MAX_K = 448;
// Members that a warp of k_srd stages at a time, and the longest row it takes.
constexpr int SRD_SLOTS = 192;
// ang (mixed model, SRD without beads): the angular-momentum correction.
// cpw: cells per warp (32, 16 or 8); a 256-cell span is taken in 32 / cpw parts, one block
// each: grid sizes count parts.
int cells_warp_blocks_per_sm(bool thermo, bool force, bool beads, bool at, bool ang, int mode);
void launch_cells_warp(bool thermo, bool force, bool beads, bool at, bool ang, int mode,
                       const BoxDev* boxes, const int2* spans, int nspans, int grid, int cpw, int* err,
                       cudaStream_t s);
// The same step for mixed SRD boxes (walls: with channel walls, then without
// beads) and, without walls and beads, mixed boxes with the Andersen rule (at) or the
// angular correction (ang), with rows of at most SRD_SLOTS records (k_srd.cu).  cpw: cells per warp (32, 16,
// 8 or 4); a 256-cell span is then taken in srd_parts(cpw) parts, one block
// each: grid sizes count parts.  A large solute box takes a launch without beads, over
// the bead groups that hold none, and one with (cpw 32), over the others; mode P
// only the first; smaller ones stay with k_cells_warp.  SRD_MIN_WARPS: see srd_cpw() in capi.cu.
constexpr int SRD_MIN_WARPS = 16, SRDD_MIN_WARPS = 6;
int srd_blocks_per_sm(bool thermo, bool force, bool beads, bool walls, bool at, bool ang, int mode);
int srd_parts(int cpw);
int srd_bead_items(int nspans);  // most blocks' work of the bead launch
void launch_srd(bool thermo, bool force, bool beads, bool walls, bool at, bool ang, int mode, const BoxDev* boxes,
                const int2* spans, int nspans, int grid, int cpw, AfterPass after, int* err,
                cudaStream_t s);
// The FP64 model's counterpart of k_srd (k_srd_d.cu), for periodic SRD boxes
// without solute and rows of at most SRDD_SLOTS records.
// It pays where the latency of a tile counts and not the FP64 pipe's rate:
// against k_cells_warp_d (us a step, density 10) 16^3 cells 17 to 51, 24^3 27 to
// 52, 40^3 72 to 75, 50^3 114 to 143, 64^3 217 to 230, 100^3 743 to 757, 128^3
// 1551 to 1495.  How full its sub-tiles are tells beyond the line: at 100^3 434 to
// 489 at density 5, but 1045 to 872 at density 12.  The boxes of a batch are taken
// each by itself (16 boxes of 50^3 in a launch: 1452 to 1516, 64 of 16^3 221 to 244).
constexpr int SRDD_SLOTS = 112, SRDD_MAX_CELLS = 200000;
int srdd_blocks_per_sm(bool thermo, bool force, int mode);
void launch_srdd(bool thermo, bool force, int mode, const BoxDev* boxes, const int2* spans,
                 int nspans, int grid, int cpw, AfterPass after, int* err, cudaStream_t s);
// The FP64 model's counterpart of k_cells_warp (k_cells_warp_d.cu), same conditions.
int cells_warpd_blocks_per_sm(bool thermo, bool force, bool beads, bool at, int mode);
void launch_cells_warpd(bool thermo, bool force, bool beads, bool at, int mode, const BoxDev* boxes,
                        const int2* spans, int nspans, int grid, int* err, cudaStream_t s);
// Place n particles (device arrays of float (mixed) or double, n x 3) in the
// current rows of a box whose counts are zero.
void launch_load(bool mixed, const BoxDev* box, const void* pos, const void* vel, int n, int* err,
                 cudaStream_t s);
// Current state (of a box at rest between steps) into device arrays in input
// order (cell_out optional); large outputs go through the row set not in use and
// the box's xcnt.  Outputs up to EXTRACT_DIRECT bytes are scattered directly.
constexpr size_t EXTRACT_DIRECT = size_t(16) << 20;
// Tags per bucket, as a power of two: 96 KB of outputs.
__host__ __device__ constexpr int xbucket_shift(bool mixed) { return mixed ? 12 : 11; }
// Counters 64 bytes apart: 10^7 atomics on 2442 neighbouring words took 0.42 ms.
constexpr int XCNT_STRIDE = 16;
inline int xbuckets(bool mixed, int64_t nsol) {
  return (int)((nsol + (1 << xbucket_shift(mixed)) - 1) >> xbucket_shift(mixed));
}
// Allows k_unbucket its shared memory; returns a cudaError_t.
int extract_prepare();
void launch_extract(bool mixed, const BoxDev* box, void* pos, void* vel, int32_t* cell_out,
                    int ncells, int nsol, uint32_t* xcnt, cudaStream_t s);

// Thermal initial state drawn on the device into pos/vel (n x 3 of the storage
// type); sums: 3 device words of scratch.
void launch_init_thermal(bool mixed, int n, uint64_t seed, const double L[3], double sigma,
                         void* pos, void* vel, unsigned long long* sums, cudaStream_t s);

// Solute MD of one collision step for the boxes with the non-bonded WCA
// repulsion (k_wca.cu): neighbour-list build, then max_substeps velocity-
// Verlet substeps (each box takes its own md_substeps).
// tiles: (box, first of WCA_BEADS beads); sync: four device words, zeroed here;
// max_blocks: blocks that fit on the device together (wca_blocks_per_sm per
// SM; the launch is cooperative).  Returns a cudaError_t.
constexpr int WCA_BEADS = 127;
int wca_blocks_per_sm();
int launch_wca_md(const BoxDev* boxes, const int2* tiles, int ntiles, int max_substeps, int max_blocks,
                  unsigned* sync, int* err, cudaStream_t s);

// ---- solute and pass bookkeeping (k_step.cu) ----
// Allows k_md_bin the shared memory of 1024-thread blocks; returns a cudaError_t.
int md_bin_prepare();
void launch_md_bin(const BoxDev* boxes, const int2* tiles, int ntiles, int chains_per_block,
                   int threads, int* err, cudaStream_t s);
void launch_scan(const ScanSeg* segs, const int2* tiles, int ntiles, uint32_t* tsum,
                 unsigned long long* gscan, uint32_t* toff, int grid, cudaStream_t s);
void launch_bead_scatter(BoxDev* boxes, const int2* tiles, int ntiles, cudaStream_t s);
// flip: the output set becomes current (after modes P and F); advance: step += 1
// (after modes F and C).
void launch_after_pass(BoxDev* boxes, int nboxes, bool flip, bool advance, cudaStream_t s);

// Virtual wall particles of the boxes of the tiles (box, first of VIRT_CELLS
// cells of its two wall-cut layers; mixed boxes on k_srd), of the step in the
// records (fresh) or of the step virt_step; virt_step is then the one after it.
// done: a word at zero, left at zero.
constexpr int VIRT_CELLS = 8;
void launch_virtual(BoxDev* boxes, int nboxes, const int2* tiles, int ntiles, int fresh,
                    unsigned* done, cudaStream_t s);

// ---- observables (k_obs.cu) ----
struct ObsCells {
  uint32_t* cnt;
  long long* mass;   // NULL: the count times mass_one = m 2^32 (no beads)
  double mass_one;
  long long* p;  // 3 per cell, in units of p_unit
  long long* k;
  int ncells;
  double p_unit;  // 2^-32; with v_scale m 2^-32 / v_scale
  float v_scale;  // not 0 (mixed, no beads): p sums rne(v v_scale 2^32), a power of two in [m, 2 m)
};
void launch_obs_particles(bool mixed, const BoxDev* box, const void* pos, const void* vel,
                          ObsCells oc, double* partials, int nblocks, cudaStream_t s);
void launch_obs_cells(ObsCells oc, double* partials, int nblocks, cudaStream_t s);
void launch_profile(bool mixed, const void* pos, const void* vel, int n, int nbins, double* sum,
                    unsigned long long* cnt, double H, cudaStream_t s);
void launch_cell_counts(const BoxDev* box, int ncells, int nbead, int32_t* cell_out,
                        int32_t* count_out, cudaStream_t s);

}  // namespace mpcd
