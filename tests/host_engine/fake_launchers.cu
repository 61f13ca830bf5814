// Stand-ins for the kernels' launchers: lines of a log, with what the engine chose.
#include <cstdio>

#include "../../paper_1801_10187_gb300/csrc/kernels.h"

extern "C" {
void fake_say(const char* line);
int fake_failure(const char* who);
void fake_spend(int cpw);
}

namespace mpcd {

int md_bin_prepare() { return 0; }
int extract_prepare() { return 0; }
int wca_blocks_per_sm() { return 4; }
int srd_blocks_per_sm(bool, bool, bool beads, bool, bool, bool, int) { return beads ? 6 : 7; }
int srdd_blocks_per_sm(bool, bool, int) { return 4; }
int cells_blocks_per_sm(bool, int, int) { return 2; }
int srd_parts(int cpw) { return BLOCK / (4 * cpw); }
int srd_bead_items(int nspans) { return 2 * nspans; }

int launch_wca_md(const BoxDev*, const int2*, int, int, int, unsigned*, int*, cudaStream_t) {
  fake_say("wca");
  return fake_failure("wca");
}
void launch_load(bool, const BoxDev*, const void*, const void*, int, int*, cudaStream_t) {}
void launch_init_thermal(bool, int, uint64_t, const double*, double, void*, void*, unsigned long long*, cudaStream_t) {}
void launch_md_bin(const BoxDev*, const int2*, int, int, int, int*, cudaStream_t) {}
void launch_scan(const ScanSeg*, const int2*, int, uint32_t*, unsigned long long*, uint32_t*, int, cudaStream_t) {}
void launch_bead_scatter(BoxDev*, const int2*, int, cudaStream_t) {}
void launch_after_pass(BoxDev*, int, bool, bool, cudaStream_t) { fake_spend(-1); }
void launch_virtual(BoxDev*, int, const int2*, int, int, unsigned*, cudaStream_t) {}
void launch_obs_particles(bool, const BoxDev*, const void*, const void*, ObsCells, double*, int, cudaStream_t) {}
void launch_obs_cells(ObsCells, double*, int, cudaStream_t) {}
void launch_cell_counts(const BoxDev*, int, int, int32_t*, int32_t*, cudaStream_t) {}
void launch_profile(bool, const void*, const void*, int, int, double*, unsigned long long*, double, cudaStream_t) {}
// puts 1 in every position and 2 in every velocity
void launch_extract(bool mixed, const BoxDev*, void* pos, void* vel, int32_t*, int, int nsol, uint32_t*, cudaStream_t) {
  fake_say("extract");
  for (size_t i = 0; i < 3 * (size_t)nsol; ++i)
    if (mixed) {
      ((float*)pos)[i] = 1.0f;
      ((float*)vel)[i] = 2.0f;
    } else {
      ((double*)pos)[i] = 1.0;
      ((double*)vel)[i] = 2.0;
    }
}
int cells_warp_blocks_per_sm(bool, bool, bool, bool, bool, int) { return 4; }
int cells_warpd_blocks_per_sm(bool, bool, bool, bool, int) { return 4; }
static void fused(const char* who, int mode, int nspans, int grid, int cpw) {
  char line[160];
  std::snprintf(line, sizeof line, "%s mode=%d spans=%d grid=%d cpw=%d", who, mode, nspans, grid, cpw);
  fake_say(line);
  fake_spend(cpw);
}
void launch_srd(bool, bool, bool beads, bool, bool, bool, int mode, const BoxDev*, const int2*, int nspans, int grid,
                int cpw, AfterPass, int*, cudaStream_t) {
  fused(beads ? "srd_beads" : "srd", mode, nspans, grid, cpw);
}
void launch_srdd(bool, bool, int mode, const BoxDev*, const int2*, int nspans, int grid, int cpw, AfterPass, int*,
                 cudaStream_t) {
  fused("srdd", mode, nspans, grid, cpw);
}
void launch_cells_warp(bool, bool, bool, bool, bool, int mode, const BoxDev*, const int2*, int nspans, int grid,
                       int cpw, int*, cudaStream_t) {
  fused("warp", mode, nspans, grid, cpw);
}
void launch_cells_warpd(bool, bool, bool, bool, int mode, const BoxDev*, const int2*, int nspans, int grid, int*,
                        cudaStream_t) {
  fused("warpd", mode, nspans, grid, 32);
}
void launch_cells(bool, int, int mode, const BoxDev*, const int2*, int nspans, int grid, int*, cudaStream_t) {
  fused("cells", mode, nspans, grid, 1);
}
}  // namespace mpcd
