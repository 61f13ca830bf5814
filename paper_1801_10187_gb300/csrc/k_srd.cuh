// k_srd.cuh -- the fused SRD step of the mixed model (arXiv:1801.10187: Sec. 2
// Eqs. stream, srd and thermo; Sec. 3.4 cell list; Sec. 3.5 cell properties;
// Sec. 3.6 rotation and thermostat, algorithm "SRD collision rule").
//
// For SRD boxes (body force, thermostat, and solute beads or channel walls
// allowed), and without solute and walls boxes with the Andersen rule (AT; Eq. at,
// Sec. 3.7) or SRD with the angular-momentum correction (ANG), whose rows hold at
// most SRD_SLOTS records; modes, records and results are those of k_cells_warp.
// A warp owns cpw consecutive cells (32, or 16, 8 or 4
// on small boxes) and takes them in sub-tiles of at most subc cells with at
// most SRD_SLOTS members between them.  A map in shared memory gives each
// member, numbered in cell order, its cell and place in the row.
//   stage    the records are copied into shared memory asynchronously, each
//            read from DRAM or L2 once per step; the first sub-tile's copies are
//            in flight while the per-cell draws (axis and Gamma pair, one cell a
//            lane) compute
//   cell     32 / subc lanes add up the members of a cell in registers (exact
//            split fixed point; no atomics); the first of them forms u, E_k, xi
//   members  in chunks of SW windows of 32: collided, streamed and binned in
//            registers and written straight to their rows with one 32-byte store;
//            a chunk's slot requests (one atomic for the lanes of a window bound
//            for one cell) are all out before its first record is stored
//
// Channel walls (WALLS): the virtual particles that fill up the cells a wall cuts
// enter a cell's sums as their number and exact totals, which k_virtual
// (k_step.cu) has left in the box for the pending step; a particle that would
// cross a wall bounces back.  k_cells draws them inside the cell's one thread.
//
// The Andersen rule draws a member's velocity once, in place of the staged one, which
// only the sums needed (k_cells_warp draws those beyond its cache twice).  us a
// step, k_cells_warp -> k_srd: 6.0 10^6 particles at density 10 313 -> 208, at
// density 20 1340 -> 387, 16^3 cells 30 -> 13.
//
// The angular correction adds a pass over the staged members for their angular
// momentum and inertia, added up by the lanes of a cell as the sums are; the members
// then get omega x r as they are collided.  k_cells_warp reads the members of that
// pass by itself, at two blocks an SM.  us a step, k_cells_warp -> k_srd: 64^3 cells
// at density 10 161 -> 111 (thermostat 180 -> 137), 80^3 at density 20 888 -> 355
// (1002 -> 445), 50^3 at density 5 53 -> 42 (61 -> 50), 16^3 37 -> 13 (41 -> 15).
//
// Both run at five blocks an SM and chunks of one window: the registers of their
// longer members' phase would spill at seven.
//
// Large solute boxes (solute_pays in capi.cu; k_cells_warp takes the others) take
// two launches in modes F and C: one over the bead groups without beads, one (BEADS)
// over those with.  In one launch the bead code's
// registers cost every cell: 2.69 ms a step at 7.8 10^7 particles with 2000 chains
// and the thermostat, against 2.14 ms for the same box without beads.
// The second takes its groups from k_bead_scatter's list, one a warp by turns: with
// a span of 256 cells to a warp it lasted as long as the warp with the most groups
// (2.61 against 2.46 ms for the step with its bead MD).
//
// What bounds it: neither DRAM (46 % of its peak at 10^7 particles) nor the
// issue slots (52 %) nor the L1 pipe (64 %), but the chain count -> stage ->
// sums -> slot -> store of global latencies, covered by the 28 warps that
// registers and shared memory leave room for.  A stand-in with the same reads,
// slot atomics and scattered writes and no arithmetic takes 131 us at 10^7
// particles (density 10); this kernel takes 175 us there, k_cells_warp 199 us.
// Per step, k_cells_warp -> k_srd (event-timed, GB300): 10^7 particles 199 ->
// 182 us, with the thermostat 253 -> 236; 2 10^7 at density 20 440 -> 328; 5 10^6
// at density 5 with the thermostat 164 -> 145; 7.8 10^7 likewise 2369 -> 2143;
// 32^3 cells at density 10 with the thermostat 25.1 -> 20.5; 16^3 21.7 -> 10.3.
// Why so: fewer instructions (106 M warp instructions against 128 M at 10^7: one
// threshold a wrap and bin axis, sums without atomics or segment ends, no
// write-back of the records to shared memory) and one read of each record
// instead of two.  Measured and slower at 10^7: all windows in registers
// (128 registers, 16 warps: 219-243 us), a second read of the records instead
// of staging them whole (188-197), chunks of 3 windows (201), 32 warps with
// spills (218): with 30 KB of shared memory a block L1 is small, and a spill
// goes to L2.
//
// Slow cases (|v| >= 1024, an overflowing row, a particle that leaves by more
// than one box length) share one copy of cold code each: the kernel is larger
// than the instruction cache (41 KB; 58 KB with the thermostat, which stalls
// two issues in ten on fetches), so chunks are one window there (SW), which
// measured 236 us against 259 us for two.
#pragma once
#include "dev_angular.cuh"
#include "dev_bin.cuh"
#include "dev_collide.cuh"
#include "dev_rows.cuh"
#include "dev_stream.cuh"
#include "kernels.h"
#include "mpcd_internal.cuh"

namespace mpcd {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int SB = 128;         // threads per block
constexpr int SWARPS = SB / 32;

// Parameters of the box, shared by the block.
struct SrdBox {
  float dt, ca, sa, omc, m;
  float L[3], hg[3], gdt[3], g[2];
  // binning under the next grid shift s: floor(x - s) = floor(x) + bias +
  // [frac(x) >= thr], and the one index outside the grid is out, for in
  float thr[3];
  int bias[3], out[3], in[3];
  int n[3], K;
  RecF* rows_cur;
  RecF* rows_out;
  uint32_t* cnt_out;
  RecF* ovf_out;
  uint32_t* ovf_cell_out;
  uint32_t* ovf_n_out;
  int ovf_cap;
  float sf[3], clo[3], chi[3];  // angular: the collision step's shift (rel_pos_f)
  int zb;  // walls: the bottom layer that the wall can cut in the collision step, -1: none
};

// Shared memory of a warp: sv[SRD_SLOTS], sr[SRD_SLOTS], map[SRD_SLOTS], then this.
struct SrdWarp {
  float4 prm[2][32];     // (u, xi), (axis, 0) per cell
};
struct SrdThermo {
  float2 gdv[32];        // accepted Gamma pair (d, v); d < 0: none
};
// Beads of each cell: count, exact int64 momentum and kinetic-energy sums.
struct SrdBeads {
  unsigned long long X[3][32], E[32];
  int nb[32], pad[4];
};
// Angular correction: centre of mass in the cell's frame and omega per cell.
struct SrdAng {
  float4 rc[32], om[32];
};
constexpr unsigned MAGIC_BITS = 0x4B400000u;  // bits of 1.5 2^23

__host__ __device__ constexpr size_t srd_head() { return (sizeof(SrdBox) + 15) & ~(size_t)15; }
__host__ __device__ constexpr size_t srd_warp(bool thermo, bool beads, bool ang) {
  return (size_t)SRD_SLOTS * 34 + sizeof(SrdWarp) + (thermo ? sizeof(SrdThermo) : 0) +
         (beads ? sizeof(SrdBeads) : 0) + (ang ? sizeof(SrdAng) : 0);
}
constexpr size_t srd_smem(bool thermo, bool beads, bool ang) {
  return srd_head() + SWARPS * srd_warp(thermo, beads, ang);
}

// The two roundings of split32 (rne(x 2^32) = H 2^20 + L) with their magic
// numbers left in: th = 1.5 2^23 + H, tl = 1.5 2^23 + L as float bits.  x 2^12 and
// x 2^32 - H 2^20 are exact, so the fused forms round where split32 does.
__device__ __forceinline__ void split_bits(float x, unsigned& th, unsigned& tl) {
  const float t = __fmaf_rn(x, 4096.0f, 12582912.0f);
  const float h20 = __fmaf_rn(t, 1048576.0f, -13194139533312.0f);  // H 2^20, exact
  const float t2 = __fadd_rn(__fmaf_rn(x, 4294967296.0f, -h20), 12582912.0f);
  th = __float_as_uint(t);
  tl = __float_as_uint(t2);
}

}  // namespace

template <bool THERMO, int MODE, bool FORCE, bool BEADS, bool WALLS, bool AT, bool ANG>
__global__ void __launch_bounds__(SB, AT || ANG ? 5 : BEADS ? 6 : 7)
    k_srd(const BoxDev* __restrict__ boxes, const int2* __restrict__ spans, int nspans, int cpw,
          AfterPass after, int* err) {
  constexpr int SW = THERMO || AT || ANG ? 1 : 2;  // windows of 32 members per chunk
  extern __shared__ __align__(16) unsigned char smem_[];
  SrdBox& H = *reinterpret_cast<SrdBox*>(smem_);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned char* wp = smem_ + srd_head() + wid * srd_warp(THERMO, BEADS, ANG);
  float4* sv = reinterpret_cast<float4*>(wp);                             // staged (v, tag)
  float4* sr = sv + SRD_SLOTS;                                             // staged (r, pad)
  unsigned short* map = reinterpret_cast<unsigned short*>(sr + SRD_SLOTS); // place in the row << 5 | cell
  SrdWarp& W = *reinterpret_cast<SrdWarp*>(wp + (size_t)SRD_SLOTS * 34);
  SrdThermo& TS = *reinterpret_cast<SrdThermo*>(&W + 1);
  SrdBeads& BS = *reinterpret_cast<SrdBeads*>(wp + (size_t)SRD_SLOTS * 34 + sizeof(SrdWarp) + (THERMO ? sizeof(SrdThermo) : 0));
  SrdAng& AG = *reinterpret_cast<SrdAng*>(wp + srd_warp(THERMO, BEADS, false));
  // a block's work: a part of a 256-cell span (its warps next to each other), or,
  // with beads, SWARPS of the groups that hold some, one to a warp
  const int parts = BLOCK / (SWARPS * cpw);
  const int ngroups = BEADS ? min((int)boxes[spans[0].x].nbgroup, boxes[spans[0].x].nbead) : 0;  // (one box)
  const int items = BEADS ? (ngroups + SWARPS - 1) / SWARPS : nspans * parts;
  int box_of_params = -1;
  const unsigned lt = (1u << lane) - 1u;
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const int sp = it / parts, part = it - sp * parts;
    const int2 tt = spans[BEADS ? 0 : sp];
    const BoxDev& B = boxes[tt.x];
    if (tt.x != box_of_params) {  // block-uniform
      __syncthreads();
      if (threadIdx.x < 3) {
        const int q = threadIdx.x;
        H.L[q] = B.L_f[q]; H.hg[q] = B.hg_f[q]; H.gdt[q] = B.gdt_f[q]; H.n[q] = B.n[q];
        if (MODE != MODE_C) {
          long long S[3];
          shift_units(B, B.step + (MODE == MODE_P ? 0ull : 1ull), S);
          const long long s = q == 0 ? S[0] : q == 1 ? S[1] : S[2];
          float lo, hi;
          bin_thresholds(s, lo, hi);
          // s < 0: frac < s never holds; s >= 0: frac >= 1 + s never holds
          H.thr[q] = s < 0 ? hi : lo;
          H.bias[q] = (s < 0 ? 0 : -1) - 0x4B000000;
          H.out[q] = s < 0 ? B.n[q] : -1;
          H.in[q] = s < 0 ? 0 : B.n[q] - 1;
          if (WALLS && q == 2) H.bias[q] += 1;  // layers 0 .. n_z + 1, no wrap
        }
        if (ANG && MODE != MODE_P) {
          long long S[3];
          shift_units(B, B.step, S);
          shift_thresholds(q == 0 ? S[0] : q == 1 ? S[1] : S[2], H.sf[q], H.clo[q], H.chi[q]);
        }
      } else if (threadIdx.x == 32) {
        H.dt = B.dt_f; H.ca = B.ca_f; H.sa = B.sa_f; H.omc = B.omc_f; H.m = B.m_f;
        H.K = B.K;
        if (WALLS) {
          H.g[0] = B.g_f[0];
          H.g[1] = B.g_f[1];
          long long S[3];
          shift_units(B, B.step, S);
          H.zb = S[2] > 0 ? 0 : S[2] < 0 ? 1 : -1;
        }
        const int out = B.cur ^ 1;
        H.rows_cur = (RecF*)B.rows[B.cur];
        H.rows_out = (RecF*)B.rows[out];
        H.cnt_out = B.cnt[out];
        H.ovf_out = (RecF*)B.ovf_rec[out];
        H.ovf_cell_out = B.ovf_cell[out];
        H.ovf_n_out = &B.ovf_n[out];
        H.ovf_cap = B.ovf_cap;
      }
      __syncthreads();
      box_of_params = tt.x;
    }
    // Solute boxes: the groups of 32 cells that hold beads are left to a second
    // launch (BEADS), which takes only them, from k_bead_scatter's list; so the bead
    // code and its registers weigh on no other cell.
    if (BEADS && it * SWARPS + wid >= ngroups) continue;
    const int c0 = BEADS ? BEAD_TILE * (int)B.bgroup[it * SWARPS + wid] : tt.y + (part * SWARPS + wid) * cpw;
    if (c0 >= B.ncells) continue;  // warp-uniform
    if (!BEADS && MODE != MODE_P && B.nbead > 0) {
      const int g = c0 / BEAD_TILE;
      if (B.bstart[g + 1] != B.bstart[g]) continue;
    }
    const int K = H.K;
    uint32_t n = 0u;
    if (lane < cpw && c0 + lane < B.ncells) {
      uint32_t* cn = B.cnt[B.cur] + (c0 + lane);
      n = *cn;
      if (MODE != MODE_C && n) *cn = 0u;  // this set is written two steps on
    }
    int gb0 = 0, gnb = 0;  // the beads of the group
    if (BEADS) {
      gb0 = (int)B.bstart[c0 / BEAD_TILE];
      gnb = (int)B.bstart[c0 / BEAD_TILE + 1] - gb0;
    }
    const int nrow = (int)n < K ? (int)n : K;
    int incl = nrow;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, d);
      if (lane >= d) incl += y;
    }
    const int N = __shfl_sync(FULL, incl, 31);
    if (N == 0 && gnb == 0) continue;
    RecF* rows = H.rows_cur + (size_t)c0 * K;
    // f(record) for the members of cell c in the overflow list (rare)
    auto for_overflow = [&](int c, auto&& f) {
      RecF* ovf = (RecF*)B.ovf_rec[B.cur];
      const uint32_t* oc = B.ovf_cell[B.cur];
      const uint32_t novf = min(B.ovf_n[B.cur], (uint32_t)B.ovf_cap);
      for (uint32_t j = 0; j < novf; ++j)
        if (oc[j] == (uint32_t)c) f(ovf + j);
    };
    // f(slot in the group order, local cell) for the beads of the cells [a, b)
    auto for_beads = [&](int a, int b, auto&& f) {
      for (int j0 = 0; j0 < gnb; j0 += 32) {
        const int j = gb0 + j0 + lane;
        if (j0 + lane < gnb) {
          const int lc = B.bgc[j] - c0;
          if (lc >= a && lc < b) f(j, lc);
        }
      }
    };
    int nb = 0;     // beads of this lane's cell; with walls its virtual particles
    int virt = -1;  // with walls: their place in the box's sums
    const int subc = cpw == 32 ? B.subw : min(B.subc, cpw);  // most cells per sub-tile, a power of two
    const int plog = __clz(subc) - 26;  // 2^plog = 32 / subc lanes add up a cell

    for (int a = 0; a < cpw;) {
      // ---- the sub-tile: cells [a, b), members [first, first + cnt) ----
      const int first = __shfl_sync(FULL, incl - nrow, a);
      const int b = min(__popc(__ballot_sync(FULL, incl - first <= SRD_SLOTS)), min(a + subc, cpw));
      const int cnt = __shfl_sync(FULL, incl, b - 1) - first;
      const bool mine = lane >= a && lane < b;
      const int s0 = incl - nrow - first;  // first member of this lane's cell
      __syncwarp();  // the previous sub-tile is done with shared memory
      if (mine) {
        int e = lane;
        for (int j = 0; j < nrow; ++j, e += 32) map[s0 + j] = (unsigned short)e;
      }
      __syncwarp();
      // records into shared memory, neighbouring lanes copying the two halves
      // of a record
      for (int q = lane; q < 2 * cnt; q += 32) {
        const int m = q >> 1, e = map[m];
        cp_async16(((lane & 1) ? sr : sv) + m,
                   reinterpret_cast<const float4*>(rows + ((e & 31) * K + (e >> 5))) + (lane & 1));
      }
      asm volatile("cp.async.commit_group;" ::: "memory");

      if (MODE != MODE_P && a == 0) {
        // Solute beads join their cell's collision with mass M (Sec. 3.6):
        // count, exact int64 momentum and kinetic sums of the warp's cells
        if (BEADS && gnb > 0) {
#pragma unroll
          for (int q = 0; q < 3; ++q) BS.X[q][lane] = 0ull;
          BS.E[lane] = 0ull;
          BS.nb[lane] = 0;
          __syncwarp();
          for_beads(0, cpw, [&](int j, int lc) {
            const double w0 = B.bgv[3 * j], w1 = B.bgv[3 * j + 1], w2 = B.bgv[3 * j + 2];
            atomicAdd(&BS.nb[lc], 1);
            atomicAdd(&BS.X[0][lc], (unsigned long long)__double2ll_rn((B.Mb * w0) * 4294967296.0));
            atomicAdd(&BS.X[1][lc], (unsigned long long)__double2ll_rn((B.Mb * w1) * 4294967296.0));
            atomicAdd(&BS.X[2][lc], (unsigned long long)__double2ll_rn((B.Mb * w2) * 4294967296.0));
            if (THERMO)  // kinetic term of the one-pass energy (Sec. 3.5)
              atomicAdd(&BS.E[lc], (unsigned long long)__double2ll_rn(
                                       (B.Mb * (w0 * w0 + w1 * w1 + w2 * w2)) * 4294967296.0));
          });
          __syncwarp();
          nb = BS.nb[lane];
        }
        if (WALLS && n > 0 && H.zb >= 0) {  // virtual particles of this lane's cell
          const int nxy = B.n[0] * B.n[1];
          const int cz = (c0 + lane) / nxy;
          const int side = cz == H.zb ? 0 : cz == H.zb + B.n[2] ? 1 : -1;
          if (side >= 0) {
            virt = side * nxy + (c0 + lane - cz * nxy);
            nb = B.virt_n[B.step & 1][virt];  // (walls exclude beads)
          }
        }
        // the per-cell draws need only the member count: the axis (Sec. 3.6)
        // and, with the thermostat, the accepted Gamma pair (d, v), E^ = d v kT
        if (!AT && (n > 0 || nb > 0)) {
          float ax[3];
          axis_of(B, B.step, (uint32_t)(c0 + lane), ax);
          W.prm[1][lane] = make_float4(ax[0], ax[1], ax[2], 0.0f);
          if (THERMO) {
            float d = -1.0f, g = 0.0f;
            if ((int)n + nb >= 2 && !gamma_draw_mixed(B, B.step, (uint32_t)(c0 + lane), (int)n + nb, d, g))
              d = -1.0f;
            TS.gdv[lane] = make_float2(d, g);
          }
        }
      }

      if (MODE != MODE_P) {
        // ---- exact momentum sums per cell (Sec. 3.5) ----
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();  // every lane's copies are in shared memory
        // 2^plog lanes add up a cell; the first of them goes on with it
        const int cc = a + (lane >> plog), part = lane & ((1 << plog) - 1);
        const int src = cc < b ? cc : a;
        const int nC = __shfl_sync(FULL, (int)n, src), s0C = __shfl_sync(FULL, s0, src);
        const int nbC = (BEADS || WALLS) ? __shfl_sync(FULL, nb, src) : 0;
        const int virtC = WALLS ? __shfl_sync(FULL, virt, src) : -1;
        const int nrowC = cc < b ? min(nC, K) : 0;
        int slow = 0;  // beyond |v| < 2^10 (or NaN) the split fails: exact sums below
        unsigned hs[3] = {0u, 0u, 0u}, ls[3] = {0u, 0u, 0u};
        long long Shh = 0, Shl = 0, Sll = 0;  // thermostat: sums of H^2, H L and L^2
        unsigned qh[3] = {0u, 0u, 0u}, ql[3] = {0u, 0u, 0u};  // angular: of the positions
        // angular: position in the cell's frame (|x| < 2: its split never fails)
        auto rel = [&](const float4& y, float x[3]) {
          x[0] = rel_pos_f(y.x, H.sf[0], H.clo[0], H.chi[0]);
          x[1] = rel_pos_f(y.y, H.sf[1], H.clo[1], H.chi[1]);
          x[2] = rel_pos_f(y.z, H.sf[2], H.clo[2], H.chi[2]);
        };
        auto sum_cells = [&] {
#pragma unroll (THERMO ? 1 : 2)
          for (int k = part; k < nrowC; k += 1 << plog) {
            const float4 x = sv[s0C + k];
            const float xv[3] = {x.x, x.y, x.z};
            slow |= !(fabsf(x.x) < 1024.0f && fabsf(x.y) < 1024.0f && fabsf(x.z) < 1024.0f);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              unsigned th, tl;
              split_bits(xv[q], th, tl);
              hs[q] += th;
              ls[q] += tl;
              if (THERMO) {  // Sec. 3.5: the kinetic energy in the same pass, exactly
                const int h = (int)(th - MAGIC_BITS), l = (int)(tl - MAGIC_BITS);
                Shh += (long long)h * h;
                Shl += (long long)h * l;
                Sll += (long long)l * l;
              }
            }
            if (ANG) {
              float x[3];
              rel(sr[s0C + k], x);
#pragma unroll
              for (int q = 0; q < 3; ++q) {
                unsigned th, tl;
                split_bits(x[q], th, tl);
                qh[q] += th;
                ql[q] += tl;
              }
            }
          }
          for (int d = 1; d < (1 << plog); d <<= 1) {
            slow |= __shfl_xor_sync(FULL, slow, d);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              hs[q] += __shfl_xor_sync(FULL, hs[q], d);
              ls[q] += __shfl_xor_sync(FULL, ls[q], d);
              if (ANG) {
                qh[q] += __shfl_xor_sync(FULL, qh[q], d);
                ql[q] += __shfl_xor_sync(FULL, ql[q], d);
              }
            }
            if (THERMO) {
              Shh += __shfl_xor_sync(FULL, Shh, d);
              Shl += __shfl_xor_sync(FULL, Shl, d);
              Sll += __shfl_xor_sync(FULL, Sll, d);
            }
          }
        };
        sum_cells();

        // ---- per cell: u (Sec. 3.5), then E_k and xi ----
        if (part == 0 && cc < b && (nC > 0 || nbC > 0)) {
          const unsigned magic = (unsigned)nrowC * MAGIC_BITS;
          const int hq[3] = {(int)(hs[0] - magic), (int)(hs[1] - magic), (int)(hs[2] - magic)};
          const int lq[3] = {(int)(ls[0] - magic), (int)(ls[1] - magic), (int)(ls[2] - magic)};
          float u[3];        // first the solvent momentum over m 2^-32
          long long Qt[3];   // thermostat: sums of V = rne(v 2^32) and of V^2
          __int128 S2 = 0;
          // one rounding of an exact sum of two exact floats, while both parts
          // are below 2^24 (|sum of v| < 4096 in every component)
          const int most = max(max(abs(hq[0]), abs(lq[0])),
                               max(max(abs(hq[1]), abs(lq[1])), max(abs(hq[2]), abs(lq[2]))));
          if (__builtin_expect(!slow && nC <= K && most < 16777216, 1)) {
#pragma unroll
            for (int q = 0; q < 3; ++q)
              u[q] = __fadd_rn(__int2float_rn(hq[q]) * 1048576.0f, __int2float_rn(lq[q]));
            if (THERMO) {
#pragma unroll
              for (int q = 0; q < 3; ++q) Qt[q] = (long long)hq[q] * 1048576LL + (long long)lq[q];
              S2 = ((__int128)Shh << 40) + ((__int128)Shl << 21) + (__int128)Sll;
            }
          } else {  // |v| >= 1024: every member one by one; then the overflow list's
#pragma unroll
            for (int q = 0; q < 3; ++q)
              Qt[q] = slow ? 0ll : (long long)hq[q] * 1048576LL + (long long)lq[q];
            if (THERMO && !slow) S2 = ((__int128)Shh << 40) + ((__int128)Shl << 21) + (__int128)Sll;
            auto add_v = [&](const RecF* p) {
              float w[3];
              load_v(p, w);
#pragma unroll 1
              for (int q = 0; q < 3; ++q) {
                const long long V = fix32_rne(q == 0 ? w[0] : q == 1 ? w[1] : w[2]);
                Qt[0] += q == 0 ? V : 0ll;
                Qt[1] += q == 1 ? V : 0ll;
                Qt[2] += q == 2 ? V : 0ll;
                if (THERMO) S2 += (__int128)V * V;
              }
            };
            if (slow)
              for (int k = 0; k < nrowC; ++k) add_v(rows + (size_t)cc * K + k);
            if (nC > K) for_overflow(c0 + cc, add_v);
#pragma unroll 1
            for (int q = 0; q < 3; ++q) {  // (one copy of the conversion: the code is cold)
              const float c = i64_to_float(q == 0 ? Qt[0] : q == 1 ? Qt[1] : Qt[2]);
              if (q == 0) u[0] = c;
              else if (q == 1) u[1] = c;
              else u[2] = c;
            }
          }
          const bool bd = BEADS && gnb > 0, vp = WALLS && nbC > 0;
          const long long* vs = vp ? B.virt_sum[B.step & 1] + 4 * (size_t)virtC : nullptr;
          float M = H.m * small_to_float(nC);
          if (BEADS) M = M + (small_to_float(nbC) * B.Mb_f + 0.0f * H.m);
          if (WALLS) M = M + (0.0f * B.Mb_f + small_to_float(nbC) * H.m);
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            float P = H.m * u[q];
            if (BEADS) P = P + (bd ? i64_to_float((long long)BS.X[q][cc]) : 0.0f);
            if (WALLS) P = P + (vp ? i64_to_float(vs[q]) : 0.0f);
            u[q] = (P * 0x1p-32f) / M;
          }
          float xi = 1.0f;
          if (THERMO && nC + nbC >= 2) {
            // Eq. thermo: E_k from the cell's exact sums, xi = sqrt(E^/E_k)
            long long X[3] = {0, 0, 0};
            if (bd) {
#pragma unroll
              for (int q = 0; q < 3; ++q) X[q] = (long long)BS.X[q][cc];
            }
            if (vp) {
#pragma unroll
              for (int q = 0; q < 3; ++q) X[q] = vs[q];
            }
            double Mt;
            const double Ep = mixed_ek_mt(B, nC, WALLS ? 0 : nbC, WALLS ? nbC : 0, Qt, S2, X,
                                          bd ? (long long)BS.E[cc] : vp ? vs[3] : 0ll, Mt);
            const float2 dv = TS.gdv[cc];
            if (!thermo_xi_from_draw(B, dv.x, dv.y, Ep, Mt, xi)) atomicOr(err, ERR_GAMMA_CAP);
          }
          W.prm[0][cc] = make_float4(u[0], u[1], u[2], xi);
        }
        if (ANG) {
          // ---- angular-momentum correction: centre of mass, then Pi omega = dL ----
          if (cc < b && part == 0 && nC > 0) {
            const unsigned magic = (unsigned)nrowC * MAGIC_BITS;
            long long Qo[3] = {0, 0, 0};
            if (nC > K)
              for_overflow(c0 + cc, [&](const RecF* p) {
                float x[3];
                rel(reinterpret_cast<const float4*>(p)[1], x);
#pragma unroll
                for (int q = 0; q < 3; ++q) Qo[q] += fix32_rne(x[q]);
              });
            float rc[3];
#pragma unroll
            for (int q = 0; q < 3; ++q)
              rc[q] = (split_sum_to_float((int)(qh[q] - magic), (int)(ql[q] - magic), Qo[q]) * 0x1p-32f) /
                      small_to_float(nC);
            AG.rc[cc] = make_float4(rc[0], rc[1], rc[2], 0.0f);
          }
          __syncwarp();
          // r_c x (v - v') and the inertia-tensor entries of a member of this
          // lane's cell, v' by the same operations as below
          auto terms = [&](const float4& a4, const float4& b4, float tm[9]) {
            const float4 pa = W.prm[0][cc], pb = W.prm[1][cc], c = AG.rc[cc];
            const float v[3] = {a4.x, a4.y, a4.z}, nn[3] = {pb.x, pb.y, pb.z}, uu[3] = {pa.x, pa.y, pa.z};
            float x[3], d[3], rr[3], dv[3];
            rel(b4, x);
#pragma unroll
            for (int q = 0; q < 3; ++q) d[q] = v[q] - uu[q];
            rotate(nn, H.ca, H.sa, H.omc, d, rr);
#pragma unroll
            for (int q = 0; q < 3; ++q) dv[q] = v[q] - (uu[q] + (THERMO ? pa.w * rr[q] : rr[q]));
            const float rc[3] = {x[0] - c.x, x[1] - c.y, x[2] - c.z};
            tm[0] = rc[1] * dv[2] - rc[2] * dv[1];
            tm[1] = rc[2] * dv[0] - rc[0] * dv[2];
            tm[2] = rc[0] * dv[1] - rc[1] * dv[0];
            tm[3] = rc[1] * rc[1] + rc[2] * rc[2];
            tm[4] = rc[0] * rc[1];
            tm[5] = rc[0] * rc[2];
            tm[6] = rc[0] * rc[0] + rc[2] * rc[2];
            tm[7] = rc[1] * rc[2];
            tm[8] = rc[0] * rc[0] + rc[1] * rc[1];
          };
          unsigned ah[9] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u}, al[9] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
          int far = 0;  // a term of 1024 or more (or NaN): exact sums below
#pragma unroll 1
          for (int k = part; k < nrowC; k += 1 << plog) {
            float tm[9];
            terms(sv[s0C + k], sr[s0C + k], tm);
#pragma unroll
            for (int q = 0; q < 9; ++q) {
              unsigned th, tl;
              far |= !(fabsf(tm[q]) < 1024.0f);
              split_bits(tm[q], th, tl);
              ah[q] += th;
              al[q] += tl;
            }
          }
          for (int d = 1; d < (1 << plog); d <<= 1) {
            far |= __shfl_xor_sync(FULL, far, d);
#pragma unroll
            for (int q = 0; q < 9; ++q) {
              ah[q] += __shfl_xor_sync(FULL, ah[q], d);
              al[q] += __shfl_xor_sync(FULL, al[q], d);
            }
          }
          if (cc < b && part == 0 && nC > 0) {
            const unsigned magic = (unsigned)nrowC * MAGIC_BITS;
            float tot[9];
            if (__builtin_expect(far || nC > K, 0)) {
              long long Lo[9];
#pragma unroll
              for (int q = 0; q < 9; ++q)
                Lo[q] = far ? 0ll : (long long)(int)(ah[q] - magic) * 1048576LL + (int)(al[q] - magic);
              auto add = [&](const float4& a4, const float4& b4) {
                float tm[9];
                terms(a4, b4, tm);
#pragma unroll
                for (int q = 0; q < 9; ++q) Lo[q] += fix32_rne(tm[q]);
              };
              if (far)
                for (int k = 0; k < nrowC; ++k) add(sv[s0C + k], sr[s0C + k]);
              if (nC > K)
                for_overflow(c0 + cc, [&](const RecF* p) {
                  add(reinterpret_cast<const float4*>(p)[0], reinterpret_cast<const float4*>(p)[1]);
                });
#pragma unroll
              for (int q = 0; q < 9; ++q) tot[q] = i64_to_float(Lo[q]);
            } else {
#pragma unroll
              for (int q = 0; q < 9; ++q)
                tot[q] = split_sum_to_float((int)(ah[q] - magic), (int)(al[q] - magic), 0);
            }
            float dL[3], P6[6], om[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) dL[k] = H.m * (tot[k] * 0x1p-32f);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
              const float e = H.m * (tot[3 + k] * 0x1p-32f);
              P6[k] = (k == 1 || k == 2 || k == 4) ? -e : e;
            }
            solve_omega<float>(nC, P6, dL, om);
            AG.om[cc] = make_float4(om[0], om[1], om[2], 0.0f);
          }
        }
        if (AT) {
          // Eq. at: every member's random velocity takes the place of its own,
          // which only the sums needed; dbar = sum dv / n the same way
          __syncwarp();
          for (int m = lane; m < cnt; m += 32) {
            const float tg = sv[m].w;
            float dv[3];
            at_draw(B, B.step, __float_as_uint(tg), 0u, B.sig_f, dv);
            sv[m] = make_float4(dv[0], dv[1], dv[2], tg);
          }
          __syncwarp();
          slow = 0;
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            hs[q] = 0u;
            ls[q] = 0u;
          }
          sum_cells();
          if (cc < b && part == 0 && nC > 0) {
            const unsigned magic = (unsigned)nrowC * MAGIC_BITS;
            const float M = H.m * small_to_float(nC);
            long long Qd[3] = {0, 0, 0};
            auto add_dv = [&](float x, float y, float z) {
              Qd[0] += fix32_rne(x);
              Qd[1] += fix32_rne(y);
              Qd[2] += fix32_rne(z);
            };
            if (slow)
              for (int k = 0; k < nrowC; ++k) add_dv(sv[s0C + k].x, sv[s0C + k].y, sv[s0C + k].z);
            if (nC > K)
              for_overflow(c0 + cc, [&](const RecF* p) {
                float dv[3];
                at_draw(B, B.step, p->tag, 0u, B.sig_f, dv);
                add_dv(dv[0], dv[1], dv[2]);
              });
            float dbar[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const float D = H.m * (slow ? i64_to_float(Qd[q])
                                          : split_sum_to_float((int)(hs[q] - magic),
                                                               (int)(ls[q] - magic), Qd[q]));
              dbar[q] = (D * 0x1p-32f) / M;
            }
            W.prm[1][cc] = make_float4(dbar[0], dbar[1], dbar[2], 0.0f);
          }
        }
        __syncwarp();
        if (BEADS && gnb > 0) {  // collide the beads with their cell's parameters
          for_beads(a, b, [&](int j, int lc) {
            const float4 pa = W.prm[0][lc], pb = W.prm[1][lc];
            CellParams<float> prm;
            prm.u[0] = pa.x; prm.u[1] = pa.y; prm.u[2] = pa.z; prm.xi = pa.w;
            prm.n[0] = pb.x; prm.n[1] = pb.y; prm.n[2] = pb.z;
            double w[3] = {B.bgv[3 * j], B.bgv[3 * j + 1], B.bgv[3 * j + 2]};
            collide_bead<true>(B, prm, w, THERMO);
            const uint32_t bb = B.border[j];
            B.svel[3 * bb] = w[0];
            B.svel[3 * bb + 1] = w[1];
            B.svel[3 * bb + 2] = w[2];
          });
        }
      }

      if (MODE == MODE_P) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
      }
      // ---- collide (Eq. srd), stream (Eq. stream), bin (Sec. 3.4) ----
      auto advance = [&](float x[3], float w[3], int o) -> uint32_t {
        if (MODE != MODE_P) {
          const float4 pa = W.prm[0][o], pb = W.prm[1][o];
          if constexpr (AT) {  // Eq. at; w is the random velocity
            w[0] = (pa.x + w[0]) - pb.x;
            w[1] = (pa.y + w[1]) - pb.y;
            w[2] = (pa.z + w[2]) - pb.z;
          } else {
            const float nn[3] = {pb.x, pb.y, pb.z};
            const float uu[3] = {pa.x, pa.y, pa.z};
            float d[3], rr[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) d[q] = w[q] - uu[q];
            rotate(nn, H.ca, H.sa, H.omc, d, rr);
#pragma unroll
            for (int q = 0; q < 3; ++q) w[q] = uu[q] + (THERMO ? pa.w * rr[q] : rr[q]);
            if (ANG) {  // v'' = v' + omega x r_c
              const float4 c = AG.rc[o], om = AG.om[o];
              const float rc[3] = {rel_pos_f(x[0], H.sf[0], H.clo[0], H.chi[0]) - c.x,
                                   rel_pos_f(x[1], H.sf[1], H.clo[1], H.chi[1]) - c.y,
                                   rel_pos_f(x[2], H.sf[2], H.clo[2], H.chi[2]) - c.z};
              w[0] = w[0] + (om.y * rc[2] - om.z * rc[1]);
              w[1] = w[1] + (om.z * rc[0] - om.x * rc[2]);
              w[2] = w[2] + (om.x * rc[1] - om.y * rc[0]);
            }
          }
        }
        if constexpr (MODE == MODE_C) {
          return 0u;
        } else {
        bool hit = false;
        if (WALLS) {  // no-slip bounce-back at z = 0 and z = n_z (stream_one)
          const float Lz = H.L[2], zn = fmaf(w[2], H.dt, x[2]);
          hit = !(zn >= 0.0f && zn < Lz);
          if (hit) {
            const float wall = (zn < 0.0f) ? 0.0f : Lz;
            float tau = (wall - x[2]) / w[2];
            if (!(tau >= 0.0f)) tau = 0.0f;
            if (tau > H.dt) tau = H.dt;
            const float rem = H.dt - tau;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              x[k] = fmaf(w[k], tau, x[k]) + ((0.5f * H.g[k]) * tau) * tau;
              w[k] = -(w[k] + H.g[k] * tau);
              x[k] = fmaf(w[k], rem, x[k]) + ((0.5f * H.g[k]) * rem) * rem;
              w[k] = w[k] + H.g[k] * rem;
            }
            w[2] = -w[2];
            float z = fmaf(w[2], rem, wall);
            if (z < 0.0f) z = 0.0f;
            if (z >= Lz) z = nextafterf(Lz, 0.0f);
            x[2] = z;
          }
        }
        if (!hit)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          x[q] = fmaf(w[q], H.dt, x[q]);
          if (FORCE) {
            x[q] = x[q] + H.hg[q];
            w[q] = w[q] + H.gdt[q];
          }
        }
        // inside the box the bits of x lie below those of L; -0, NaN and what
        // is outside do not
        if (!(__float_as_uint(x[0]) < __float_as_uint(H.L[0]) &&
              __float_as_uint(x[1]) < __float_as_uint(H.L[1]) &&
              (WALLS || __float_as_uint(x[2]) < __float_as_uint(H.L[2])))) {
          bool far = false;
#pragma unroll
          for (int q = 0; q < (WALLS ? 2 : 3); ++q) {
            x[q] = wrap_fast(x[q] + 0.0f, H.L[q]);
            far |= !(x[q] >= 0.0f && x[q] < H.L[q]);
          }
          if (far) {  // more than one box length out, or non-finite (one copy: it is cold)
#pragma unroll 1
            for (int q = 0; q < (WALLS ? 2 : 3); ++q) {
              float y = q == 0 ? x[0] : q == 1 ? x[1] : x[2];
              y = wrap(y, H.L[q]);
              if (q == 0) x[0] = y;
              else if (q == 1) x[1] = y;
              else x[2] = y;
            }
          }
        }
        int c[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float tf = __fadd_rd(x[q], 8388608.0f);  // 2^23 + floor(x)
          const float f = __fsub_rn(x[q], __fsub_rn(tf, 8388608.0f));
          const int i = __float_as_int(tf) + H.bias[q] + (f >= H.thr[q] ? 1 : 0);
          c[q] = (WALLS && q == 2) ? min(max(i, 0), H.n[2] + 1) : i == H.out[q] ? H.in[q] : i;
        }
        return (uint32_t)(c[0] + H.n[0] * (c[1] + H.n[1] * c[2]));
        }
      };
      // append a record to the row of cell c2 at the slot taken for it (or to
      // the overflow list beyond the row capacity)
      auto emit = [&](const float x[3], const float w[3], uint32_t tg, uint32_t c2, uint32_t slot) {
        if (__builtin_expect(slot < (uint32_t)K, 1)) {
          store_rec(H.rows_out + (c2 * (size_t)(uint32_t)K + slot), x, w, tg);
        } else {
          const uint32_t j = atomicAdd(H.ovf_n_out, 1u);
          if (j < (uint32_t)H.ovf_cap) {
            store_rec(H.ovf_out + j, x, w, tg);
            H.ovf_cell_out[j] = c2;
          } else {
            atomicOr(err, ERR_OVERFLOW_CAP);
          }
        }
      };
      for (int base = 0; base < cnt; base += 32 * SW) {
        float v[SW][3], r[SW][3];
        uint32_t tag[SW], c2[SW];
        int own[SW];
#pragma unroll
        for (int w = 0; w < SW; ++w) {
          const int m = base + 32 * w + lane;
          own[w] = 0;
          if (m < cnt) {
            own[w] = map[m];
            const float4 x = sv[m], y = sr[m];
            v[w][0] = x.x; v[w][1] = x.y; v[w][2] = x.z;
            tag[w] = __float_as_uint(x.w);
            r[w][0] = y.x; r[w][1] = y.y; r[w][2] = y.z;
          }
        }
        if constexpr (MODE == MODE_C) {
#pragma unroll
          for (int w = 0; w < SW; ++w)
            if (base + 32 * w + lane < cnt) {
              advance(r[w], v[w], own[w] & 31);
              store_rec(rows + ((own[w] & 31) * K + (own[w] >> 5)), r[w], v[w], tag[w]);
            }
        } else {
        // Slots: the lanes of a window bound for the same cell share one atomic
        // (made by the first of them) and take consecutive slots, so their
        // records land side by side.  An atomic's result is read only when the
        // whole chunk's requests are out.
        uint32_t slot0[SW];
        int lr[SW];  // leader lane | rank << 8
#pragma unroll
        for (int w = 0; w < SW; ++w) {
          const bool act = base + 32 * w + lane < cnt;
          c2[w] = act ? advance(r[w], v[w], own[w] & 31) : FULL;
          const unsigned peers = __match_any_sync(FULL, c2[w]);
          const int leader = __ffs(peers) - 1;
          slot0[w] = 0u;
          if (act && lane == leader) slot0[w] = atomicAdd(&H.cnt_out[c2[w]], (uint32_t)__popc(peers));
          lr[w] = leader | (__popc(peers & lt) << 8);
        }
#pragma unroll
        for (int w = 0; w < SW; ++w) {
          const uint32_t slot = __shfl_sync(FULL, slot0[w], lr[w] & 255) + (uint32_t)(lr[w] >> 8);
          if (base + 32 * w + lane < cnt) emit(r[w], v[w], tag[w], c2[w], slot);
        }
        }
      }
      if (mine && (int)n > K)
        for_overflow(c0 + lane, [&](RecF* p) {
          float x[3], w[3];
          uint32_t tg;
          load_rec(p, x, w, tg);
          if (AT && MODE != MODE_P) at_draw(B, B.step, tg, 0u, B.sig_f, w);
          const uint32_t c = advance(x, w, lane);
          if constexpr (MODE == MODE_C) store_rec(p, x, w, tg);
          else emit(x, w, tg, c, atomicAdd(&H.cnt_out[c], 1u));
        });
      a = b;
    }
  }
  finish_pass(after);
}

}  // namespace mpcd
