// k_wca.cu -- non-bonded solute forces (arXiv:1801.10187, Sec. 4.3: the
// polymer benchmark integrates a bead-spring model by velocity Verlet with
// non-bonded pair forces from a neighbour list of buffer 0.4 a; the pair
// potential is only cited, and the Weeks-Chandler-Andersen repulsion is the
// reading taken here).
//
// One cooperative launch runs the whole solute MD of a collision step for the
// boxes with the repulsion.  Its blocks walk tiles of WCA_BEADS beads and meet
// at a grid barrier:
//   rebuild  clear, insert: a hash grid of the beads (cells of edge 1, unshifted,
//            two buckets per bead, each a linked list built by atomic exchange of
//            its head); list: each bead's neighbours among the 27 cells around it
//            within cutoff + buffer (minimum image)
//   force    bonds, each computed once, plus WCA over the list
//   drift    closing half kick of the last substep, half kick, drift into the
//            other of two position buffers (so that slower blocks may still read
//            the last positions: one barrier a substep)
// The list holds every pair within the cutoff while no bead has moved more than
// half the buffer since the build; a drift that finds one raises a flag, and the
// list is rebuilt before the forces.  More than NL_MAX listed neighbours raises
// ERR_NLIST.  The later binning of the beads for the collision (k_md_bin) skips
// its own MD for these boxes.
//
// What bounds it: the FP64 pipe (51 % busy; a warp instruction every 16 cycles of an
// SM) and the barriers.  The first form took five launches a substep, of which three
// returned at once in nearly every one, and 45 us of force kernel: distances of
// all listed pairs in double, each bond from both its sides with a square root
// and a division.  Here pairs are sorted out by their distance in float from
// 32-bit fixed-point positions (whose differences wrap to the minimum image by
// themselves), only those within the cutoff cost FP64, and a bond is computed
// once.  Bonds and kicks take the oracle's operations one by one.  A reciprocal
// square root and fused forms in their place saved 4 % (four steps of 1024 chains
// of 50 beads and the read 9.74 against 10.17 ms) and put bead velocities a tenth
// further from 64 bits (7.7 against 6.85 10^-14 after these steps).
#include "dev_stream.cuh"
#include "kernels.h"
#include "mpcd_internal.cuh"

namespace mpcd {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int WT = WCA_BEADS + 1;  // threads per block: one bond more than beads
constexpr int FW = WT / 32;
constexpr int ROUNDS = 4;          // rounds of 32 pairs whose loads are in flight together
constexpr int QCAP = 32 * (ROUNDS + 1);  // queue: fewer than 32 waiting plus those
constexpr unsigned SPIN_LIMIT = 1u << 22;

__device__ __forceinline__ uint32_t bucket_of(int key, int hsize) {
  return ((uint32_t)key * 2654435761u) % (uint32_t)hsize;
}

__device__ __forceinline__ int grid_coord(double x, int n) {
  int c = (int)floor(x);
  if (c < 0) c = 0;
  if (c >= n) c = n - 1;
  return c;
}

// minimum-image difference along one axis for |d| < L (both points in the box):
// the same as d - L rint(d / L), where a difference of just L / 2 stays (ties to
// even).  L / 2 has no low word, so the words of d settle the comparison off the
// FP64 pipe; and in this form the subtraction is branched over, as nearly always,
// and not computed and dropped: four steps of 1024 chains of 50 beads and the read
// 11.35 -> 9.74 ms.
__device__ __forceinline__ double min_image(double d, double L) {
  const int h = __double2hiint(L) - 0x00100000;  // of L / 2
  const int e = __double2hiint(d) & 0x7FFFFFFF;
  if (e >= h && (e > h || __double2loint(d) != 0)) d -= copysign(L, d);
  return d;
}

// Position x in [0, L) as a fraction of the box in 32 bits (f = 2^32 / L).
__device__ __forceinline__ int fraction(double x, double f) {
  return (int)(unsigned)__double2ull_rd(x * f);
}

struct MdWarp {
  int off[33];          // first flat pair index of each bead; off[32] = all pairs
  int qown[QCAP];       // queued pair: the warp-local bead it acts on
  int qj[QCAP];         // and the other bead
  double c[3][32];      // forces of one flush, one per lane
  double F[3][32];      // sum of each bead's pair forces
};
struct MdShared {
  MdWarp w[FW];
  double r[3][WT];      // positions of beads b0 - 1 ... b0 + WCA_BEADS - 1
  double g[3][WT];      // force of the bond from bead b0 - 1 + t to the next, on the former
  int X[3][WT];         // fixed-point positions, as r
};

// Grid barrier of a cooperative launch: *bar counts arrivals.  The wait is
// bounded; a block that gives up raises ERR_BARRIER and waits at no barrier again.
__device__ __forceinline__ void grid_barrier(unsigned* bar, unsigned& target, bool& dead, int* err) {
  __syncthreads();
  target += gridDim.x;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    if (!dead) {
      unsigned spins = 0, seen = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
      } while ((int)(seen - target) < 0 && ++spins < SPIN_LIMIT);
      if ((int)(seen - target) < 0) {
        dead = true;
        atomicOr(err, ERR_BARRIER);
      }
    }
    __threadfence();
  }
  __syncthreads();
}

// Forces of queue entries [q0, q0 + nq), nq <= 32: lane l takes entry q0 + l; each run of entries of
// one bead is summed, in order, by its first lane.
__device__ __forceinline__ void wca_flush(const BoxDev& B, MdShared& S, MdWarp& W, int wbase,
                                          const double* pos, int q0, int nq, int lane) {
  const int* qown = W.qown + q0;
  if (lane < nq) {
    const int own = qown[lane], j = W.qj[q0 + lane];
    double d[3];
#pragma unroll
    for (int q = 0; q < 3; ++q)
      d[q] = min_image(__ldcg(&pos[3 * (size_t)j + q]) - S.r[q][wbase + own], B.L[q]);
    const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    double g = 0.0;
    if (r2 < B.wca_rc2) {
      const double inv = 1.0 / r2;
      const double x = B.lj_sig2 * inv;
      const double x6 = x * x * x;
      g = 24.0 * B.lj_eps * x6 * (2.0 * x6 - 1.0) * inv;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) W.c[q][lane] = -(g * d[q]);
  }
  __syncwarp();
  if (lane < nq) {
    const int own = qown[lane];
    if (lane == 0 || qown[lane - 1] != own) {
      double acc[3] = {W.c[0][lane], W.c[1][lane], W.c[2][lane]};
      for (int l = lane + 1; l < nq && qown[l] == own; ++l) {
#pragma unroll
        for (int q = 0; q < 3; ++q) acc[q] += W.c[q][l];
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) W.F[q][own] += acc[q];
    }
  }
  __syncwarp();
}

}  // namespace

__global__ void __launch_bounds__(WT, 4) k_wca_md(const BoxDev* __restrict__ boxes,
                                               const int2* __restrict__ tiles, int ntiles,
                                               int max_substeps, unsigned* bar, int* stale, int* err) {
  __shared__ MdShared S;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  MdWarp& W = S.w[warp];
  unsigned target = 0u;
  bool dead = false;

  // f(box, bead, first bead of the tile) for every bead of this block's tiles
  auto for_beads = [&](auto&& f) {
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
      const int2 tt = tiles[tile];
      const BoxDev& B = boxes[tt.x];
      if (t < WCA_BEADS && tt.y + t < B.nbead) f(B, tt.y + t);
    }
  };
  // rebuild the lists of the boxes with substeps left, at positions buf
  auto rebuild = [&](int sub, int buf) {
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
      const int2 tt = tiles[tile];
      const BoxDev& B = boxes[tt.x];
      if (sub >= B.md_substeps) continue;
      const int h1 = tt.y + WCA_BEADS >= B.nbead ? B.nl_hsize : 2 * (tt.y + WCA_BEADS);
      for (int h = 2 * tt.y + t; h < h1; h += WT) B.nl_head[h] = -1;
    }
    grid_barrier(bar, target, dead, err);
    for_beads([&](const BoxDev& B, int b) {
      if (sub >= B.md_substeps) return;
      int c[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double x = B.wpos[buf][3 * (size_t)b + k];
        B.nl_rb[3 * (size_t)b + k] = x;
        c[k] = grid_coord(x, B.n[k]);
      }
      const int key = c[0] + B.n[0] * (c[1] + B.n[1] * c[2]);
      B.nl_key[b] = key;
      B.nl_next[b] = atomicExch(&B.nl_head[bucket_of(key, B.nl_hsize)], b);
    });
    grid_barrier(bar, target, dead, err);
    for_beads([&](const BoxDev& B, int b) {
      if (sub >= B.md_substeps) return;
      const int key = B.nl_key[b];
      const int c[3] = {key % B.n[0], (key / B.n[0]) % B.n[1], key / (B.n[0] * B.n[1])};
      const double rb[3] = {B.nl_rb[3 * (size_t)b], B.nl_rb[3 * (size_t)b + 1],
                            B.nl_rb[3 * (size_t)b + 2]};
      int cnt = 0;
      bool over = false;
      // n_k >= 3 on every axis, so the 27 cells are distinct
      for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
          for (int dx = -1; dx <= 1; ++dx) {
            int x = c[0] + dx, y = c[1] + dy, z = c[2] + dz;
            x += x < 0 ? B.n[0] : x >= B.n[0] ? -B.n[0] : 0;
            y += y < 0 ? B.n[1] : y >= B.n[1] ? -B.n[1] : 0;
            z += z < 0 ? B.n[2] : z >= B.n[2] ? -B.n[2] : 0;
            const int k2 = x + B.n[0] * (y + B.n[1] * z);
            // other blocks' heads and links of this very launch: past L1
            int j = __ldcg(&B.nl_head[bucket_of(k2, B.nl_hsize)]);
            // a bucket's list is acyclic and holds at most every bead once
            for (int guard = 0; j >= 0 && guard < B.nbead; ++guard, j = __ldcg(&B.nl_next[j])) {
              if (j == b || __ldcg(&B.nl_key[j]) != k2) continue;
              double r2 = 0.0;
#pragma unroll
              for (int q = 0; q < 3; ++q) {
                const double d = min_image(__ldcg(&B.nl_rb[3 * (size_t)j + q]) - rb[q], B.L[q]);
                r2 = fma(d, d, r2);
              }
              if (!(r2 < B.wca_rl2)) continue;
              if (cnt < NL_MAX) B.nl_nbr[(size_t)b * NL_MAX + cnt] = j;
              else over = true;
              ++cnt;
            }
          }
      B.nl_cnt[b] = min(cnt, NL_MAX);
      if (over) atomicOr(err, ERR_NLIST);
    });
    __syncthreads();  // a bead's list is read by its whole warp
  };
  // bond and WCA forces of this block's beads at positions buf
  auto forces = [&](int sub, int buf) {
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
      const int2 tt = tiles[tile];
      const BoxDev& B = boxes[tt.x];
      if (sub > B.md_substeps) continue;  // the same for the whole block
      const double* pos = B.wpos[buf];
      const int4* fix = B.wfix[buf];
      const int b0 = tt.y, cl = B.chain_len;
      __syncthreads();  // the last tile is done with S
      // thread t: bead b0 - 1 + t and its bond to the next bead of its chain
      const int jb = b0 - 1 + t;
      double rj[3] = {0.0, 0.0, 0.0};
      if (jb >= 0 && jb < B.nbead) {
        const int4 f = __ldcg(&fix[jb]);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          rj[q] = __ldcg(&pos[3 * (size_t)jb + q]);
          S.r[q][t] = rj[q];
        }
        S.X[0][t] = f.x;
        S.X[1][t] = f.y;
        S.X[2][t] = f.z;
      }
      __syncthreads();
      double g[3] = {0.0, 0.0, 0.0};
      if (jb >= 0 && jb + 1 < B.nbead && jb % cl != cl - 1) {
        double d[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const double rn = t + 1 < WT ? S.r[q][t + 1] : __ldcg(&pos[3 * (size_t)(jb + 1) + q]);
          d[q] = min_image(rn - rj[q], B.L[q]);
        }
        const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        if (r2 > 0.0) {  // k (1 - r0 / |d|) d; coincident beads: no force
          const double dist = sqrt(r2);
          const double f = (B.bond_k * (dist - B.bond_r0)) / dist;
#pragma unroll
          for (int q = 0; q < 3; ++q) g[q] = f * d[q];
        }
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) S.g[q][t] = g[q];
      const int b = b0 + t;
      const bool valid = t < WCA_BEADS && b < B.nbead;
      const int cnt = valid ? B.nl_cnt[b] : 0;
      // flat pair offsets: exclusive scan of the list lengths over the warp
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
      }
      W.off[lane] = incl - cnt;
      if (lane == 31) W.off[32] = incl;
#pragma unroll
      for (int q = 0; q < 3; ++q) W.F[q][lane] = 0.0;
      __syncthreads();
      const float sc[3] = {(float)(B.L[0] * 0x1p-32), (float)(B.L[1] * 0x1p-32),
                           (float)(B.L[2] * 0x1p-32)};
      const int wbase = warp * 32 + 1;  // place of the warp's first bead in S.r and S.X
      const int total = W.off[32];      // at most 32 NL_MAX
      int nq = 0;                       // queued pairs (the same in every lane)
      for (int base = 0; base < total; base += 32 * ROUNDS) {
        int own[ROUNDS], j[ROUNDS];
        int4 f[ROUNDS];
#pragma unroll
        for (int u = 0; u < ROUNDS; ++u) {
          const int k = base + 32 * u + lane;
          own[u] = 0;
          j[u] = -1;
          if (k < total) {
            // the bead of pair k: the last with off <= k (offsets do not decrease)
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
              if (W.off[own[u] + step] <= k) own[u] += step;
            j[u] = B.nl_nbr[(size_t)(b0 + warp * 32 + own[u]) * NL_MAX + (k - W.off[own[u]])];
          }
        }
#pragma unroll
        for (int u = 0; u < ROUNDS; ++u)
          if (j[u] >= 0) f[u] = __ldcg(&fix[j[u]]);
#pragma unroll
        for (int u = 0; u < ROUNDS; ++u) {
          bool hit = false;
          if (j[u] >= 0) {
            const float dx = (float)(int)((unsigned)f[u].x - (unsigned)S.X[0][wbase + own[u]]) * sc[0];
            const float dy = (float)(int)((unsigned)f[u].y - (unsigned)S.X[1][wbase + own[u]]) * sc[1];
            const float dz = (float)(int)((unsigned)f[u].z - (unsigned)S.X[2][wbase + own[u]]) * sc[2];
            hit = fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < B.wca_rc2f;
          }
          const unsigned m = __ballot_sync(FULL, hit);
          if (hit) {
            const int at = nq + __popc(m & ((1u << lane) - 1u));  // < QCAP
            W.qown[at] = own[u];
            W.qj[at] = j[u];
          }
          nq += __popc(m);
        }
        __syncwarp();
        int q0 = 0;
        for (; nq - q0 >= 32; q0 += 32) wca_flush(B, S, W, wbase, pos, q0, 32, lane);
        if (q0 > 0) {  // the rest (fewer than 32) to the front
          nq -= q0;
          int e0 = 0, e1 = 0;
          if (lane < nq) {
            e0 = W.qown[q0 + lane];
            e1 = W.qj[q0 + lane];
          }
          __syncwarp();
          if (lane < nq) {
            W.qown[lane] = e0;
            W.qj[lane] = e1;
          }
          __syncwarp();
        }
      }
      if (nq > 0) wca_flush(B, S, W, wbase, pos, 0, nq, lane);
      if (valid) {
        // bond to the left (index t) and to the right (t + 1; b0 + t is bead t + 1 of S)
#pragma unroll
        for (int q = 0; q < 3; ++q)
          B.bF[3 * (size_t)b + q] = (S.g[q][t + 1] - S.g[q][t]) + W.F[q][lane];
      }
    }
  };
  auto put = [&](const BoxDev& B, int buf, int b, const double r[3]) {
    int x[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      B.wpos[buf][3 * (size_t)b + k] = r[k];
      x[k] = fraction(r[k], B.wfrac[k]);
    }
    B.wfix[buf][b] = make_int4(x[0], x[1], x[2], 0);
  };

  for_beads([&](const BoxDev& B, int b) {
    // a given state may lie outside the box; cells, fractions and min_image take it inside
    double r[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) r[k] = wrap_bits(B.spos[3 * (size_t)b + k], B.L[k]);
    put(B, 0, b, r);
  });
  rebuild(0, 0);
  forces(0, 0);
  for (int sub = 0; sub < max_substeps; ++sub) {
    const int nxt = (sub + 1) & 1;
    for_beads([&](const BoxDev& B, int b) {
      if (sub >= B.md_substeps) return;
      double r[3], m2 = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double F = B.bF[3 * (size_t)b + k];
        double v = B.svel[3 * (size_t)b + k];
        if (sub > 0) v = v + B.md_hh * F;  // closes the last substep
        v = v + B.md_hh * F;
        r[k] = wrap_bits(B.wpos[nxt ^ 1][3 * (size_t)b + k] + B.md_h * v, B.L[k]);
        B.svel[3 * (size_t)b + k] = v;
        const double d = min_image(r[k] - B.nl_rb[3 * (size_t)b + k], B.L[k]);
        m2 = fma(d, d, m2);
      }
      put(B, nxt, b, r);
      if (m2 > B.wca_half_skin2) stale[sub % 3] = 1;
    });
    grid_barrier(bar, target, dead, err);
    // the flag of two substeps on: read by all before this barrier, set after the next
    if (blockIdx.x == 0 && t == 0) stale[(sub + 2) % 3] = 0;
    int again;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(again) : "l"(stale + sub % 3) : "memory");
    if (again) rebuild(sub, nxt);
    forces(sub + 1, nxt);
  }
  for_beads([&](const BoxDev& B, int b) {
    if (B.md_substeps <= 0) return;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      B.svel[3 * (size_t)b + k] = B.svel[3 * (size_t)b + k] + B.md_hh * B.bF[3 * (size_t)b + k];
      B.spos[3 * (size_t)b + k] = B.wpos[B.md_substeps & 1][3 * (size_t)b + k];
    }
  });
}

int wca_blocks_per_sm() {
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_wca_md, WT, 0);
  return nb;
}

// sync: four words (the barrier's count and the flags), zeroed here.
int launch_wca_md(const BoxDev* boxes, const int2* tiles, int ntiles, int max_substeps, int max_blocks,
                  unsigned* sync, int* err, cudaStream_t s) {
  if (ntiles <= 0) return 0;
  cudaMemsetAsync(sync, 0, 4 * sizeof(unsigned), s);
  int* stale = (int*)(sync + 1);
  void* args[] = {(void*)&boxes, (void*)&tiles, (void*)&ntiles, (void*)&max_substeps,
                  (void*)&sync, (void*)&stale, (void*)&err};
  return (int)cudaLaunchCooperativeKernel((void*)k_wca_md, dim3(ntiles < max_blocks ? ntiles : max_blocks),
                                          dim3(WT), args, 0, s);
}

}  // namespace mpcd
