// k_srd.cu -- instances and launch dispatch of the fused SRD step of the mixed
// model (kernel template: k_srd.cuh).
#include "k_srd.cuh"

namespace mpcd {

template <int MODE, bool TH, bool FO>
static void* srd_fn(bool beads, bool walls) {
  if (walls) return (void*)k_srd<TH, MODE, true, false, true, false, false>;  // always with the force terms
  return beads ? (void*)k_srd<TH, MODE, FO, true, false, false, false>
               : (void*)k_srd<TH, MODE, FO, false, false, false, false>;
}

template <int MODE>
static void* srd_mode(bool thermo, bool force, bool beads, bool walls, bool at, bool ang) {
  if (at && MODE != MODE_P)
    return force ? (void*)k_srd<false, MODE, true, false, false, true, false>
                 : (void*)k_srd<false, MODE, false, false, false, true, false>;
  if (ang && MODE != MODE_P) {
    if (thermo) return force ? (void*)k_srd<true, MODE, true, false, false, false, true>
                             : (void*)k_srd<true, MODE, false, false, false, false, true>;
    return force ? (void*)k_srd<false, MODE, true, false, false, false, true>
                 : (void*)k_srd<false, MODE, false, false, false, false, true>;
  }
  // mode P only streams and bins: nothing in it depends on thermostat or beads
  if (MODE == MODE_P) return force ? srd_fn<MODE, false, true>(false, walls)
                                      : srd_fn<MODE, false, false>(false, walls);
  if (thermo) return force ? srd_fn<MODE, true, true>(beads, walls) : srd_fn<MODE, true, false>(beads, walls);
  return force ? srd_fn<MODE, false, true>(beads, walls) : srd_fn<MODE, false, false>(beads, walls);
}

static void* srd_variant(bool thermo, bool force, bool beads, bool walls, bool at, bool ang, int mode) {
  if (mode == MODE_P) return srd_mode<MODE_P>(thermo, force, beads, walls, at, ang);
  if (mode == MODE_F) return srd_mode<MODE_F>(thermo, force, beads, walls, at, ang);
  return srd_mode<MODE_C>(thermo, force, beads, walls, at, ang);
}

static size_t srd_variant_smem(bool thermo, bool beads, bool ang, int mode) {
  return mode == MODE_P ? srd_smem(false, false, false) : srd_smem(thermo, beads, ang);
}

int srd_blocks_per_sm(bool thermo, bool force, bool beads, bool walls, bool at, bool ang, int mode) {
  const void* fn = srd_variant(thermo, force, beads, walls, at, ang, mode);
  const size_t smem = srd_variant_smem(thermo, beads, ang, mode);
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, SB, smem);
  return nb;
}

int srd_parts(int cpw) { return BLOCK / (SWARPS * cpw); }
int srd_bead_items(int nspans) { return nspans * (BLOCK / (SWARPS * BEAD_TILE)); }

void launch_srd(bool thermo, bool force, bool beads, bool walls, bool at, bool ang, int mode, const BoxDev* boxes,
                const int2* spans, int nspans, int grid, int cpw, AfterPass after, int* err, cudaStream_t s) {
  if (nspans <= 0) return;
  void* args[] = {(void*)&boxes, (void*)&spans, (void*)&nspans, (void*)&cpw, (void*)&after, (void*)&err};
  cudaLaunchKernel(srd_variant(thermo, force, beads, walls, at, ang, mode), dim3(grid), dim3(SB), args,
                   srd_variant_smem(thermo, beads, ang, mode), s);
}

}  // namespace mpcd
