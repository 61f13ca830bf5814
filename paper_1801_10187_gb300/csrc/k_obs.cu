// k_obs.cu -- observables (arXiv:1801.10187, Sec. 3.5 last paragraph: net
// momentum, energy and temperature), the z profile of v_x used for the
// Poiseuille check, and the member counts of the last step.
#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "dev_collide.cuh"
#include "mpcd_internal.cuh"

namespace mpcd {

// Per-particle pass: block partial sums of P and KE (double, fixed block
// decomposition) and fixed-point sums per cell of the unshifted grid.  Taking the
// particles from the rows, where neighbours add to the same words, was slower (0.6
// against 0.33 ms for 5 10^6).  PLAIN (mixed, no beads) finds the cell in float,
// sums scaled velocities from their split parts and multiplies by the mass at the
// end: 12 FP64-pipe instructions a particle (16 cycles an SM each) instead of 33;
// 314 -> 210 us for 5 10^6 particles.
template <bool MIXED, bool PLAIN>
__global__ void __launch_bounds__(256) k_obs_particles(const BoxDev* __restrict__ box,
                                                       const real_t<MIXED>* __restrict__ pos,
                                                       const real_t<MIXED>* __restrict__ vel,
                                                       ObsCells oc, double* __restrict__ partials) {
  const BoxDev& B = *box;
  __shared__ double red[4][256];
  double acc[4] = {0, 0, 0, 0};
  const int ntot = B.nsol + B.nbead;
  if (PLAIN) {
    const double hm = 0.5 * B.m, hm32 = hm * 4294967296.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B.nsol; i += gridDim.x * blockDim.x) {
      float w[3];
      int c[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        c[k] = min(max((int)floorf((float)pos[3 * (size_t)i + k]), 0), B.n[k] - 1);
        w[k] = (float)vel[3 * (size_t)i + k];
      }
      const int cell = c[0] + B.n[0] * (c[1] + B.n[1] * c[2]);
      const double d0 = (double)w[0], d1 = (double)w[1], d2 = (double)w[2];
      const double ww = fma(d2, d2, fma(d1, d1, d0 * d0));
      acc[0] += d0;
      acc[1] += d1;
      acc[2] += d2;
      acc[3] += ww;
      atomicAdd(&oc.cnt[cell], 1u);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float a = w[k] * oc.v_scale;
        int H, L;
        const long long q = split32(a, H, L) ? (((long long)H) << 20) + L
                                             : __double2ll_rn(((double)w[k] * (double)oc.v_scale) * 4294967296.0);
        atomicAdd((unsigned long long*)&oc.p[3 * cell + k], (unsigned long long)q);
      }
      atomicAdd((unsigned long long*)&oc.k[cell], (unsigned long long)__double2ll_rn(ww * hm32));
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) acc[k] *= B.m;
    acc[3] *= hm;
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; !PLAIN && i < ntot; i += gridDim.x * blockDim.x) {
    double x[3], w[3], m;
    if (i < B.nsol) {
      for (int k = 0; k < 3; ++k) {
        x[k] = (double)pos[3 * i + k];
        w[k] = (double)vel[3 * i + k];
      }
      m = B.m;
    } else {
      const int b = i - B.nsol;
      for (int k = 0; k < 3; ++k) {
        x[k] = B.spos[3 * b + k];
        w[k] = B.svel[3 * b + k];
      }
      m = B.Mb;
    }
    const double e = (0.5 * m) * (w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
    for (int k = 0; k < 3; ++k) acc[k] += m * w[k];
    acc[3] += e;
    int c[3];
    for (int k = 0; k < 3; ++k) {
      int q = (int)floor(x[k]);
      if (q < 0) q = 0;
      if (q >= B.n[k]) q = B.n[k] - 1;
      c[k] = q;
    }
    const int cell = c[0] + B.n[0] * (c[1] + B.n[1] * c[2]);
    atomicAdd(&oc.cnt[cell], 1u);
    if (oc.mass)  // (without beads it is the count times one mass)
      atomicAdd((unsigned long long*)&oc.mass[cell], (unsigned long long)__double2ll_rn(m * 4294967296.0));
    for (int k = 0; k < 3; ++k)
      atomicAdd((unsigned long long*)&oc.p[3 * cell + k],
                (unsigned long long)__double2ll_rn((m * w[k]) * 4294967296.0));
    atomicAdd((unsigned long long*)&oc.k[cell], (unsigned long long)__double2ll_rn(e * 4294967296.0));
  }
  for (int q = 0; q < 4; ++q) red[q][threadIdx.x] = acc[q];
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s)
      for (int q = 0; q < 4; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int q = 0; q < 4; ++q) partials[4 * blockIdx.x + q] = red[q][0];
}

// Per-cell pass: sum of cell temperatures over cells with >= 2 members, the
// number of such cells and the number of occupied cells (block partials).  Bound by the
// FP64 pipe: one division a cell and no scaling of the sums, 82 -> 54 us for 10^6 cells.
__global__ void __launch_bounds__(256) k_obs_cells(ObsCells oc, double* __restrict__ partials) {
  __shared__ double red[3][256];
  double a[3] = {0, 0, 0};
  unsigned occ = 0u, warm = 0u;
  const double pu = oc.p_unit * 4294967296.0, pu2 = pu * pu;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < oc.ncells; c += gridDim.x * blockDim.x) {
    const uint32_t n = oc.cnt[c];
    if (n >= 1) ++occ;
    if (n >= 2) {  // 2 (K - P^2 / 2 M) / (3 (n - 1)) with one division
      const double M = oc.mass ? (double)oc.mass[c] : (double)n * oc.mass_one;
      const double P0 = (double)oc.p[3 * (size_t)c], P1 = (double)oc.p[3 * (size_t)c + 1],
                   P2 = (double)oc.p[3 * (size_t)c + 2];
      const double K = (double)oc.k[c];
      const double pp = fma(P2, P2, fma(P1, P1, P0 * P0));
      a[0] += fma(2.0 * M, K, -(pp * pu2)) / (M * (double)(3ll * (n - 1u)));
      ++warm;
    }
  }
  a[0] *= 0x1p-32;
  a[1] = (double)warm;
  a[2] = (double)occ;
  for (int q = 0; q < 3; ++q) red[q][threadIdx.x] = a[q];
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s)
      for (int q = 0; q < 3; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int q = 0; q < 3; ++q) partials[3 * blockIdx.x + q] = red[q][0];
}

// Mean-velocity profile: sums of v_x and member counts per z slab.  With few
// slabs every block adds up its own in shared memory, PROFILE_COPIES of them by
// turns of the warps, and then to the totals; 5 10^5 particles on 40 words of
// global memory took 315 us.
constexpr int PROFILE_SHARED = 512;  // slabs summed in shared memory
constexpr int PROFILE_COPIES = 4;
template <bool MIXED>
__global__ void __launch_bounds__(256) k_profile(const real_t<MIXED>* __restrict__ pos,
                                                 const real_t<MIXED>* __restrict__ vel, int n, int nbins,
                                                 double* sum, unsigned long long* cnt, double H) {
  __shared__ double ss[PROFILE_COPIES * PROFILE_SHARED];
  __shared__ unsigned sc[PROFILE_COPIES * PROFILE_SHARED];
  const bool local = nbins <= PROFILE_SHARED;
  const int copy = (int)((threadIdx.x >> 5) % PROFILE_COPIES) * nbins;
  if (local) {
    for (int i = threadIdx.x; i < PROFILE_COPIES * nbins; i += blockDim.x) {
      ss[i] = 0.0;
      sc[i] = 0u;
    }
    __syncthreads();
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    long long b = (long long)floor((double)pos[3 * (size_t)i + 2] / H * (double)nbins);
    if (b < 0) b = 0;
    if (b >= nbins) b = nbins - 1;
    if (local) {
      atomicAdd(&ss[copy + b], (double)vel[3 * (size_t)i]);
      atomicAdd(&sc[copy + b], 1u);
    } else {
      atomicAdd(&sum[b], (double)vel[3 * (size_t)i]);
      atomicAdd(&cnt[b], 1ull);
    }
  }
  if (local) {
    __syncthreads();
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
      double s = 0.0;
      unsigned c = 0u;
      for (int k = 0; k < PROFILE_COPIES; ++k) {
        s += ss[k * nbins + b];
        c += sc[k * nbins + b];
      }
      if (c) {
        atomicAdd(&sum[b], s);
        atomicAdd(&cnt[b], (unsigned long long)c);
      }
    }
  }
}

// Member counts of the current cells: solvent from the row counts, then the
// beads of the step.
__global__ void k_cell_counts(const BoxDev* __restrict__ box, int32_t* count_out) {
  const BoxDev& B = *box;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < B.ncells; c += gridDim.x * blockDim.x)
    count_out[c] = (int32_t)B.cnt[B.cur][c];
}
__global__ void k_bead_cells(const BoxDev* __restrict__ box, int32_t* cell_out, int32_t* count_out) {
  const BoxDev& B = *box;
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < B.nbead; b += gridDim.x * blockDim.x) {
    const int32_t c = B.bcell[b];
    if (cell_out) cell_out[B.nsol + b] = c;
    if (count_out) atomicAdd(&count_out[c], 1);
  }
}

static int grid_for(int n, int per_block) {
  int g = (n + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > 4096) g = 4096;
  return g;
}

void launch_obs_particles(bool mixed, const BoxDev* box, const void* pos, const void* vel,
                          ObsCells oc, double* partials, int nblocks, cudaStream_t s) {
  if (mixed && oc.v_scale != 0.0f)
    k_obs_particles<true, true><<<nblocks, 256, 0, s>>>(box, (const float*)pos, (const float*)vel, oc,
                                                        partials);
  else if (mixed)
    k_obs_particles<true, false><<<nblocks, 256, 0, s>>>(box, (const float*)pos, (const float*)vel, oc,
                                                         partials);
  else
    k_obs_particles<false, false><<<nblocks, 256, 0, s>>>(box, (const double*)pos, (const double*)vel, oc,
                                                   partials);
}

void launch_obs_cells(ObsCells oc, double* partials, int nblocks, cudaStream_t s) {
  k_obs_cells<<<nblocks, 256, 0, s>>>(oc, partials);
}

void launch_profile(bool mixed, const void* pos, const void* vel, int n, int nbins, double* sum,
                    unsigned long long* cnt, double H, cudaStream_t s) {
  const int g = n > 0 ? std::min((n + 255) / 256, 608) : 1;
  if (mixed) k_profile<true><<<g, 256, 0, s>>>((const float*)pos, (const float*)vel, n, nbins, sum, cnt, H);
  else k_profile<false><<<g, 256, 0, s>>>((const double*)pos, (const double*)vel, n, nbins, sum, cnt, H);
}

void launch_cell_counts(const BoxDev* box, int ncells, int nbead, int32_t* cell_out,
                        int32_t* count_out, cudaStream_t s) {
  if (count_out) k_cell_counts<<<grid_for(ncells, 256), 256, 0, s>>>(box, count_out);
  if (nbead > 0) k_bead_cells<<<grid_for(nbead, 256), 256, 0, s>>>(box, cell_out, count_out);
}

}  // namespace mpcd
