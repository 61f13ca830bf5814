// k_cells_warp.cu -- instances and launch dispatch of the warp-spread SRD step
// of the mixed model (kernel template: k_cells_warp.cuh).
#define MPCD_PHILOX_HALVES  // see philox()
#include "k_cells_warp.cuh"

namespace mpcd {

template <bool TH, int MODE, bool FO, bool BE, bool AT, bool ANG = false>
static void* warp_fn() {
  return (void*)k_cells_warp<TH, MODE, FO, BE, AT, ANG>;
}

template <int MODE, bool BE>
static void* warp_variant_mb(bool thermo, bool force, bool at) {
  if (at) return force ? warp_fn<false, MODE, true, BE, true>() : warp_fn<false, MODE, false, BE, true>();
  if (thermo) return force ? warp_fn<true, MODE, true, BE, false>() : warp_fn<true, MODE, false, BE, false>();
  return force ? warp_fn<false, MODE, true, BE, false>() : warp_fn<false, MODE, false, BE, false>();
}

template <int MODE>
static void* warp_variant_mode(bool thermo, bool force, bool beads, bool at, bool ang) {
  if (ang && thermo) return force ? warp_fn<true, MODE, true, false, false, true>()
                                  : warp_fn<true, MODE, false, false, false, true>();
  if (ang) return force ? warp_fn<false, MODE, true, false, false, true>()
                        : warp_fn<false, MODE, false, false, false, true>();
  return beads ? warp_variant_mb<MODE, true>(thermo, force, at)
               : warp_variant_mb<MODE, false>(thermo, force, at);
}

// ang: the angular-momentum correction (SRD without beads only).
static void* warp_variant(bool thermo, bool force, bool beads, bool at, bool ang, int mode) {
  if (mode == MODE_P) return warp_variant_mode<MODE_P>(thermo, force, beads, at, ang);
  if (mode == MODE_F) return warp_variant_mode<MODE_F>(thermo, force, beads, at, ang);
  return warp_variant_mode<MODE_C>(thermo, force, beads, at, ang);
}

int cells_warp_blocks_per_sm(bool thermo, bool force, bool beads, bool at, bool ang, int mode) {
  const void* fn = warp_variant(thermo, force, beads, at, ang, mode);
  const size_t smem = block_smem(beads, at, ang, thermo);
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, BLOCK, smem);
  return nb;
}

void launch_cells_warp(bool thermo, bool force, bool beads, bool at, bool ang, int mode,
                       const BoxDev* boxes, const int2* spans, int nspans, int grid, int cpw, int* err,
                       cudaStream_t s) {
  if (nspans <= 0) return;
  void* args[] = {(void*)&boxes, (void*)&spans, (void*)&nspans, (void*)&cpw, (void*)&err};
  cudaLaunchKernel(warp_variant(thermo, force, beads, at, ang, mode), dim3(grid), dim3(BLOCK), args,
                   block_smem(beads, at, ang, thermo), s);
}

}  // namespace mpcd
