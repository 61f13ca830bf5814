// k_cells.cu -- the fused SRD step on cell rows (arXiv:1801.10187: Sec. 2
// Eqs. stream, srd and thermo; Sec. 3.4 cell list; Sec. 3.5 cell properties;
// Sec. 3.6 rotation and thermostat, algorithm "SRD collision rule").
//
// One thread owns one cell.  Its members are the records of its row (plus,
// rarely, overflow records).  Mode F is one whole step boundary in one pass:
//   collide step t      pass 1 forms the exact cell sums (and, with the
//                       thermostat, a second pass the energy about u); the
//                       thread draws the axis and xi; pass 2 rotates each member
//   stream step t + 1   the rotated velocity streams the position
//   bin step t + 1      with the next grid shift; the record is appended to the
//                       row of its new cell in the other buffer (atomic slot)
// Mode P only streams and bins (the first step after the state was read or
// set), mode C only collides, in place (to complete a step before the state is
// read).  Nothing else touches the particles: no separate sort, scan or
// reorder pass exists, and every record moves as one 32-byte sector.
//
// This kernel also carries the Andersen rule (Eq. at, Sec. 3.7) for rows too
// long for the warp-spread kernel, and the angular-momentum-conserving form
// of either rule (Sec. 2: the constraint the paper cites after Eqs. srd and
// at): a second pass over the cell's members forms dL = sum m r_c x (v - v')
// and the inertia tensor about the cell's centre of mass, and every member
// then receives omega x r_c with Pi omega = dL.
#define MPCD_PHILOX_HALVES  // see philox()
#include <algorithm>

#include "dev_angular.cuh"
#include "dev_collide.cuh"
#include "dev_rows.cuh"
#include "dev_stream.cuh"
#include "kernels.h"
#include "mpcd_internal.cuh"

namespace mpcd {

namespace {

// Coordinate of x relative to the shifted cell whose index along the axis is
// i (in [0, 1); a member wrapped across the box edge is brought back).
__device__ __forceinline__ double rel_pos(double x, double s, int i, double L) {
  double d = (x - s) - (double)i;
  if (d < 0.0) d += L;
  else if (d >= 1.0) d -= L;
  return d;
}

// Per-cell sums of the angular correction: positions (centre of mass), then
// r_c x (v - v') and the inertia tensor entries (|r_c|^2 - r_c r_c^T: xx, xy,
// xz, yy, yz, zz with the off-diagonal products summed positive).  Mixed
// model: int64 sums of rne(term 2^32) of float terms; FP64: double sums.
template <bool MIXED> struct AngAcc;
template <> struct AngAcc<true> {
  long long q[3] = {0, 0, 0}, l[3] = {0, 0, 0}, p[6] = {0, 0, 0, 0, 0, 0};
};
template <> struct AngAcc<false> {
  double q[3] = {0, 0, 0}, l[3] = {0, 0, 0}, p[6] = {0, 0, 0, 0, 0, 0};
};

}  // namespace

template <bool MIXED, bool THERMO, bool EXTRA, int MODE, bool AT, bool ANG>
__global__ void __launch_bounds__(BLOCK) k_cells(const BoxDev* __restrict__ boxes,
                                                 const int2* __restrict__ spans, int nspans,
                                                 int* err) {
  using T = real_t<MIXED>;
  using R = rec_t<MIXED>;
  __shared__ long long sSn[3];  // shift of the step the records are binned for
  __shared__ long long sSz;     // z shift of the collision step (wall-cut cells)
  __shared__ long long sSc[3];  // shift of the collision step (angular correction)
  __shared__ float sCf[3][3];   // its float form and thresholds (mixed model)
  for (int sp = blockIdx.x; sp < nspans; sp += gridDim.x) {
    const int2 tt = spans[sp];
    const BoxDev& B = boxes[tt.x];
    const unsigned long long t = B.step;
    __syncthreads();
    if (threadIdx.x == 0) {
      if (MODE != MODE_C) shift_units(B, MODE == MODE_P ? t : t + 1ull, sSn);
      if (EXTRA && MODE != MODE_P) {
        long long S[3];
        shift_units(B, t, S);
        sSz = S[2];
      }
      if (ANG && MODE != MODE_P) {
        shift_units(B, t, sSc);
        for (int k = 0; k < 3; ++k) shift_thresholds(sSc[k], sCf[0][k], sCf[1][k], sCf[2][k]);
      }
    }
    __syncthreads();
    const int cell = tt.y + (int)threadIdx.x;
    if (cell >= B.ncells) continue;
    const int cur = B.cur, out = cur ^ 1;
    const int K = B.K;
    const uint32_t n = B.cnt[cur][cell];
    if (MODE != MODE_C && n) B.cnt[cur][cell] = 0u;  // this set is written two steps on
    const int nrow = (int)n < K ? (int)n : K;
    const bool has_ovf = (int)n > K;
    R* row = ((R*)B.rows[cur]) + (size_t)cell * K;
    R* ovf = (R*)B.ovf_rec[cur];
    const uint32_t* ovf_cell = B.ovf_cell[cur];
    const uint32_t novf = has_ovf ? min(B.ovf_n[cur], (uint32_t)B.ovf_cap) : 0u;
    int b0 = 0, nbt = 0;
    if (EXTRA && MODE != MODE_P && B.nbead > 0) {
      const int g = cell / B.tc;
      b0 = (int)B.bstart[g];
      nbt = (int)B.bstart[g + 1] - b0;
    }
    auto bead_in = [&](int j, int& b) {
      b = (int)B.border[b0 + j];
      return B.bcell[b] == cell;
    };
    bool any = n > 0;
    if (EXTRA)
      for (int j = 0; j < nbt && !any; ++j) {
        int b;
        any = bead_in(j, b);
      }
    if (!any) continue;

    CellParams<T> prm;  // the Andersen rule keeps the mean random velocity in prm.n
    T om[3] = {(T)0, (T)0, (T)0}, rcm[3] = {(T)0, (T)0, (T)0};
    int ic[3] = {0, 0, 0};
    double sc[3] = {0.0, 0.0, 0.0};
    if (ANG && MODE != MODE_P) {
      ic[0] = cell % B.n[0];
      ic[1] = (cell / B.n[0]) % B.n[1];
      ic[2] = cell / (B.n[0] * B.n[1]);
#pragma unroll
      for (int k = 0; k < 3; ++k) sc[k] = (double)sSc[k] * 0x1p-32;
    }
    // position of a member relative to its cell, in the model's type
    auto rel = [&](const T r[3], T o[3]) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if constexpr (MIXED) o[k] = rel_pos_f(r[k], sCf[0][k], sCf[1][k], sCf[2][k]);
        else o[k] = rel_pos(r[k], sc[k], ic[k], B.L[k]);
      }
    };
    // Eq. at: random velocity of a member
    auto draw_dv = [&](uint32_t tag, T dv[3]) {
      if constexpr (MIXED) at_draw(B, t, tag, 0u, B.sig_f, dv);
      else at_draw(B, t, tag, 0u, B.sig, dv);
    };
    // the collision rule without the angular correction
    auto base_rule = [&](T w[3], uint32_t tag) {
      if (AT) {
        T dv[3];
        draw_dv(tag, dv);
#pragma unroll
        for (int k = 0; k < 3; ++k) w[k] = (prm.u[k] + dv[k]) - prm.n[k];
      } else {
        collide_one<MIXED>(B, prm, w, THERMO);
      }
    };
    if (MODE != MODE_P) {
      // ---- cell properties (Sec. 3.5) ----
      CellAcc<MIXED> a;
      CellAcc<MIXED> ad;  // Andersen rule: sums of the random velocities
      AngAcc<MIXED> g;
      auto add_member = [&](const R* p) {
        if (AT || ANG) {
          T r[3], w[3];
          uint32_t tag;
          load_rec(p, r, w, tag);
          a.add_solvent(B, w);
          if (AT) {
            T dv[3];
            draw_dv(tag, dv);
            ad.add_solvent(B, dv);
          }
          if (ANG) {
            T x[3];
            rel(r, x);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              if constexpr (MIXED) g.q[k] += fix32_rne(x[k]);
              else g.q[k] += x[k];
            }
          }
        } else {
          T w[3];
          load_v(p, w);
          a.add_solvent(B, w);
        }
      };
#pragma unroll 4
      for (int k = 0; k < nrow; ++k) add_member(row + k);
      if (has_ovf)
        for (uint32_t j = 0; j < novf; ++j)
          if (ovf_cell[j] == (uint32_t)cell) add_member(ovf + j);
      // the FP64 model's energy about u (the mixed model has E_k from the
      // exact sums of the first pass)
      auto solvent_energy = [&](const T u[3], CellAcc<MIXED>& acc) {
        if constexpr (!MIXED) {
#pragma unroll 4
          for (int k = 0; k < nrow; ++k) {
            T w[3];
            load_v(row + k, w);
            acc.add_solvent_energy(B, w, u);
          }
          if (has_ovf)
            for (uint32_t j = 0; j < novf; ++j)
              if (ovf_cell[j] == (uint32_t)cell) {
                T w[3];
                load_v(ovf + j, w);
                acc.add_solvent_energy(B, w, u);
              }
        }
      };
      const double sz = EXTRA ? (double)sSz * 0x1p-32 : 0.0;
      T u[3];
      cell_mean<MIXED>(B, t, (uint32_t)cell, sz, a, EXTRA ? nbt : 0, bead_in, EXTRA, u);
      if (AT) {  // Eq. at: u and dbar = sum m dv / sum m
        T dbar[3];
        ad.mean_velocity(B, dbar, false);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          prm.u[k] = u[k];
          prm.n[k] = dbar[k];
        }
        prm.xi = (T)1;
      } else {
        if (THERMO) solvent_energy(u, a);
        cell_finish<MIXED>(B, t, (uint32_t)cell, a, u, EXTRA ? nbt : 0, bead_in, THERMO, EXTRA, prm,
                           err);
      }
      if (ANG) {
        // centre of mass in the cell frame, then dL = sum m r_c x (v - v')
        // and the inertia tensor about it
        const int ns = a.ns;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if constexpr (MIXED) rcm[k] = (i64_to_float(g.q[k]) * 0x1p-32f) / small_to_float(ns);
          else rcm[k] = g.q[k] / (double)ns;
        }
        auto add_moment = [&](const R* p) {
          T r[3], w[3];
          uint32_t tag;
          load_rec(p, r, w, tag);
          T x[3], rc[3], v2[3] = {w[0], w[1], w[2]};
          rel(r, x);
          base_rule(v2, tag);
          T d[3];
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            rc[k] = x[k] - rcm[k];
            d[k] = w[k] - v2[k];
          }
          const T cx[3] = {rc[1] * d[2] - rc[2] * d[1], rc[2] * d[0] - rc[0] * d[2],
                           rc[0] * d[1] - rc[1] * d[0]};
          const T te[6] = {rc[1] * rc[1] + rc[2] * rc[2], rc[0] * rc[1], rc[0] * rc[2],
                           rc[0] * rc[0] + rc[2] * rc[2], rc[1] * rc[2],
                           rc[0] * rc[0] + rc[1] * rc[1]};
          if constexpr (MIXED) {
#pragma unroll
            for (int k = 0; k < 3; ++k) g.l[k] += fix32_rne(cx[k]);
#pragma unroll
            for (int k = 0; k < 6; ++k) g.p[k] += fix32_rne(te[k]);
          } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) g.l[k] += B.m * cx[k];
#pragma unroll
            for (int k = 0; k < 6; ++k) g.p[k] += B.m * te[k];
          }
        };
        for (int k = 0; k < nrow; ++k) add_moment(row + k);
        if (has_ovf)
          for (uint32_t j = 0; j < novf; ++j)
            if (ovf_cell[j] == (uint32_t)cell) add_moment(ovf + j);
        T P[6], dL[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if constexpr (MIXED) dL[k] = B.m_f * (i64_to_float(g.l[k]) * 0x1p-32f);
          else dL[k] = g.l[k];
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          T e;
          if constexpr (MIXED) e = B.m_f * (i64_to_float(g.p[k]) * 0x1p-32f);
          else e = g.p[k];
          P[k] = (k == 1 || k == 2 || k == 4) ? -e : e;
        }
        solve_omega<T>(ns, P, dL, om);
      }
    }

    // ---- members: collide, then stream and bin for the next step ----
    auto process = [&](R* p) {
      T r[3], w[3];
      uint32_t tag;
      load_rec(p, r, w, tag);
      if (MODE != MODE_P) {
        if (AT || ANG) base_rule(w, tag);
        else collide_one<MIXED>(B, prm, w, THERMO);
        if (ANG) {  // v'' = v' + omega x r_c
          T x[3], rc[3];
          rel(r, x);
#pragma unroll
          for (int k = 0; k < 3; ++k) rc[k] = x[k] - rcm[k];
          w[0] = w[0] + (om[1] * rc[2] - om[2] * rc[1]);
          w[1] = w[1] + (om[2] * rc[0] - om[0] * rc[2]);
          w[2] = w[2] + (om[0] * rc[1] - om[1] * rc[0]);
        }
      }
      if (MODE == MODE_C) {
        store_rec(p, r, w, tag);
        return;
      }
      stream_one(B, r, w);
      const uint32_t c2 = cell_of(B, sSn, r, err);
      insert<MIXED>(B, out, c2, r, w, tag, err);
    };
#pragma unroll 2
    for (int k = 0; k < nrow; ++k) process(row + k);
    if (has_ovf)
      for (uint32_t j = 0; j < novf; ++j)
        if (ovf_cell[j] == (uint32_t)cell) process(ovf + j);
    if (EXTRA && MODE != MODE_P) {
      for (int j = 0; j < nbt; ++j) {
        int b;
        if (!bead_in(j, b)) continue;
        double w[3] = {B.svel[3 * b], B.svel[3 * b + 1], B.svel[3 * b + 2]};
        collide_bead<MIXED>(B, prm, w, THERMO);
        B.svel[3 * b] = w[0];
        B.svel[3 * b + 1] = w[1];
        B.svel[3 * b + 2] = w[2];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// State in and out.  The input is placed in the rows of the unshifted grid
// (any placement works: the next step re-bins after streaming).  Positions
// are stored as given; only the placement uses a wrapped copy.
// ---------------------------------------------------------------------------
template <bool MIXED>
__global__ void k_load(const BoxDev* __restrict__ box, const real_t<MIXED>* __restrict__ pos,
                       const real_t<MIXED>* __restrict__ vel, int* err) {
  using T = real_t<MIXED>;
  const BoxDev& B = *box;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B.nsol; i += gridDim.x * blockDim.x) {
    const T r[3] = {pos[3 * i], pos[3 * i + 1], pos[3 * i + 2]};
    const T v[3] = {vel[3 * i], vel[3 * i + 1], vel[3 * i + 2]};
    int c[3];
    for (int k = 0; k < 3; ++k) {
      const double L = B.L[k];
      double x = (double)r[k];
      x = x - L * floor(x / L);
      int q = (x >= 0.0 && x < L) ? (int)x : 0;
      if (q >= B.n[k]) q = B.n[k] - 1;
      c[k] = q;
    }
    if (B.walls) c[2] += 1;  // channel layers are 1 .. n_z of the n_z + 2 layers
    const uint32_t cell = (uint32_t)(c[0] + B.n[0] * (c[1] + B.n[1] * c[2]));
    insert<MIXED>(B, B.cur, cell, r, v, (uint32_t)i, err);
  }
}

// Records of the current set, written in input order; cell_out (optional)
// receives each particle's cell.  The outputs are a scatter by tag: 12-byte
// (FP64: 24-byte) writes all over two arrays.
//
// Small outputs (EXTRACT_DIRECT bytes) are scattered straight from the rows.
// From larger ones that costs six scattered 4-byte stores a particle, and beyond
// L2 partial sectors merged in DRAM as well (10^7 mixed particles: 0.74 ms).
// There the records first move, whole, to buckets of XBUCKET consecutive tags,
// and then a block gathers each bucket's outputs in shared memory and writes
// them out in order.  A bucket holds exactly the records of its tags, so the
// buckets lie end to end in [0, nsol) of the row set that is not in use between
// steps.  (10^7 particles: 0.30 ms; buckets of 2^17 tags scattered
// within L2 instead: 0.68 ms.)
//
// f(act, record, cell) with every record of four consecutive cells, eight lanes a
// cell; called by the whole warp together, act marking the lanes with a record.
template <class R, class F>
__device__ __forceinline__ void for_rows(const BoxDev& B, int cur, int c0, F&& f) {
  const int lane = threadIdx.x & 31, c = c0 + (lane >> 3), K = B.K;
  const int n = c < B.ncells ? min((int)B.cnt[cur][c], K) : 0;
  const R* row = ((const R*)B.rows[cur]) + (size_t)c * K;
  const int most = __reduce_max_sync(0xFFFFFFFFu, n);
  for (int k = lane & 7; k - (lane & 7) < most; k += 8) f(k < n, row + k, c);
}

template <bool MIXED>
__device__ __forceinline__ void put_particle(const rec_t<MIXED>* p, real_t<MIXED>* __restrict__ pos,
                                             real_t<MIXED>* __restrict__ vel,
                                             int32_t* __restrict__ cell_out, int cell) {
  real_t<MIXED> r[3], v[3];
  uint32_t tag;
  load_rec(p, r, v, tag);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    pos[3 * (size_t)tag + q] = r[q];
    vel[3 * (size_t)tag + q] = v[q];
  }
  if (cell_out) cell_out[tag] = cell;
}

template <bool MIXED>
__global__ void __launch_bounds__(BLOCK) k_extract(const BoxDev* __restrict__ box,
                                                   real_t<MIXED>* __restrict__ pos,
                                                   real_t<MIXED>* __restrict__ vel,
                                                   int32_t* __restrict__ cell_out) {
  using R = rec_t<MIXED>;
  const BoxDev& B = *box;
  const int cur = B.cur;
  for (int c0 = (blockIdx.x * BLOCK + threadIdx.x) / 32 * 4; c0 < B.ncells;
       c0 += gridDim.x * (BLOCK / 8))
    for_rows<R>(B, cur, c0, [&](bool act, const R* p, int cell) {
      if (act) put_particle<MIXED>(p, pos, vel, cell_out, cell);
    });
  const uint32_t novf = min(B.ovf_n[cur], (uint32_t)B.ovf_cap);
  for (uint32_t j = blockIdx.x * BLOCK + threadIdx.x; j < novf; j += gridDim.x * BLOCK)
    put_particle<MIXED>(((const R*)B.ovf_rec[cur]) + j, pos, vel, cell_out,
                        (int)B.ovf_cell[cur][j]);
}

__device__ __forceinline__ uint32_t tag_of(const RecF* p) { return p->tag; }
__device__ __forceinline__ uint32_t tag_of(const RecD* p) { return p->tag; }

// Copies a record and notes its cell in the padding.
__device__ __forceinline__ void move_rec(RecF* d, const RecF* p, int cell) {
  const float4 a = reinterpret_cast<const float4*>(p)[0];
  float4 b = reinterpret_cast<const float4*>(p)[1];
  b.w = __int_as_float(cell);
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(d), "f"(a.x), "f"(a.y),
               "f"(a.z), "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
               : "memory");
}
__device__ __forceinline__ void move_rec(RecD* d, const RecD* p, int cell) {
#pragma unroll
  for (int q = 0; q < 3; ++q) reinterpret_cast<float4*>(d)[q] = reinterpret_cast<const float4*>(p)[q];
  reinterpret_cast<uint4*>(d)[3] = make_uint4(p->tag, (uint32_t)cell, 0u, 0u);
}
__device__ __forceinline__ int noted_cell(const RecF* p) { return (int)p->pad; }
__device__ __forceinline__ int noted_cell(const RecD* p) { return (int)p->pad; }

// Records into buckets of tags; the lanes of a warp bound for one bucket share an
// atomic and take consecutive places.
template <bool MIXED>
__global__ void __launch_bounds__(BLOCK) k_bucket(const BoxDev* __restrict__ box) {
  using R = rec_t<MIXED>;
  constexpr int SHIFT = xbucket_shift(MIXED);
  const BoxDev& B = *box;
  const int cur = B.cur, lane = threadIdx.x & 31;
  R* out = (R*)B.rows[cur ^ 1];
  auto place = [&](bool act, const R* p, int cell) {
    const uint32_t bucket = act ? tag_of(p) >> SHIFT : 0xFFFFFFFFu;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, bucket);
    const int leader = __ffs(peers) - 1;
    uint32_t at = 0u;
    if (act && lane == leader) at = atomicAdd(&B.xcnt[(size_t)bucket * XCNT_STRIDE], (uint32_t)__popc(peers));
    at = __shfl_sync(0xFFFFFFFFu, at, leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
    if (act) move_rec(out + (((size_t)bucket << SHIFT) + at), p, cell);
  };
  for (int c0 = (blockIdx.x * BLOCK + threadIdx.x) / 32 * 4; c0 < B.ncells;
       c0 += gridDim.x * (BLOCK / 8))
    for_rows<R>(B, cur, c0, place);
  const uint32_t novf = min(B.ovf_n[cur], (uint32_t)B.ovf_cap);
  for (uint32_t j0 = blockIdx.x * BLOCK + (threadIdx.x & ~31u); j0 < novf; j0 += gridDim.x * BLOCK) {
    const uint32_t j = j0 + lane;
    place(j < novf, ((const R*)B.ovf_rec[cur]) + j, j < novf ? (int)B.ovf_cell[cur][j] : 0);
  }
}

// A bucket's outputs gathered in shared memory and written in order.
constexpr int UT = 512;  // threads per block
template <bool MIXED>
__global__ void __launch_bounds__(UT) k_unbucket(const BoxDev* __restrict__ box,
                                                 real_t<MIXED>* __restrict__ pos,
                                                 real_t<MIXED>* __restrict__ vel,
                                                 int32_t* __restrict__ cell_out) {
  using T = real_t<MIXED>;
  using R = rec_t<MIXED>;
  constexpr int N = 1 << xbucket_shift(MIXED);
  extern __shared__ __align__(16) unsigned char xs_[];
  T* sr = reinterpret_cast<T*>(xs_);
  T* sv = sr + 3 * N;
  int32_t* sc = reinterpret_cast<int32_t*>(sv + 3 * N);
  const BoxDev& B = *box;
  const size_t i0 = (size_t)blockIdx.x * N;
  const int n = (int)min((size_t)N, (size_t)B.nsol - i0);
  const R* in = (const R*)B.rows[B.cur ^ 1] + i0;
  for (int i = threadIdx.x; i < n; i += UT) {
    T r[3], v[3];
    uint32_t tag;
    load_rec(in + i, r, v, tag);
    const int j = (int)(tag & (N - 1));
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      sr[3 * j + q] = r[q];
      sv[3 * j + q] = v[q];
    }
    if (cell_out) sc[j] = noted_cell(in + i);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 3 * n; i += UT) {
    pos[3 * i0 + i] = sr[i];
    vel[3 * i0 + i] = sv[i];
  }
  if (cell_out)
    for (int i = threadIdx.x; i < n; i += UT) cell_out[i0 + i] = sc[i];
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
template <bool M, bool TH, bool EX, int MODE, bool AT, bool ANG>
static void* cells_fn() {
  return (void*)k_cells<M, TH, EX, MODE, AT, ANG>;
}

// variant bits: 1 thermostat, 2 walls or beads, 16 Andersen rule, 32 angular
// correction (the last two without walls or beads; the Andersen rule without
// the thermostat).
template <bool M, int MODE>
static void* cells_variant_m(int variant) {
  const bool th = (variant & 1) != 0, ex = (variant & 2) != 0;
  const bool at = (variant & 16) != 0, ang = (variant & 32) != 0;
  if (at) return ang ? cells_fn<M, false, false, MODE, true, true>()
                     : cells_fn<M, false, false, MODE, true, false>();
  if (ang) return th ? cells_fn<M, true, false, MODE, false, true>()
                     : cells_fn<M, false, false, MODE, false, true>();
  if (th) return ex ? cells_fn<M, true, true, MODE, false, false>()
                    : cells_fn<M, true, false, MODE, false, false>();
  return ex ? cells_fn<M, false, true, MODE, false, false>()
            : cells_fn<M, false, false, MODE, false, false>();
}

template <int MODE>
static void* cells_variant_mode(bool mixed, int variant) {
  return mixed ? cells_variant_m<true, MODE>(variant) : cells_variant_m<false, MODE>(variant);
}

static void* cells_variant(bool mixed, int variant, int mode) {
  if (mode == MODE_P) return cells_variant_mode<MODE_P>(mixed, variant);
  if (mode == MODE_F) return cells_variant_mode<MODE_F>(mixed, variant);
  return cells_variant_mode<MODE_C>(mixed, variant);
}

int cells_blocks_per_sm(bool mixed, int variant, int mode) {
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, cells_variant(mixed, variant, mode), BLOCK, 0);
  return nb;
}

void launch_cells(bool mixed, int variant, int mode, const BoxDev* boxes, const int2* spans,
                  int nspans, int grid, int* err, cudaStream_t s) {
  if (nspans <= 0) return;
  void* args[] = {(void*)&boxes, (void*)&spans, (void*)&nspans, (void*)&err};
  cudaLaunchKernel(cells_variant(mixed, variant, mode), dim3(grid), dim3(BLOCK), args, 0, s);
}

static int grid_for_n(int n) {
  int g = (n + 255) / 256;
  if (g < 1) g = 1;
  if (g > 8192) g = 8192;
  return g;
}

void launch_load(bool mixed, const BoxDev* box, const void* pos, const void* vel, int n, int* err,
                 cudaStream_t s) {
  if (n <= 0) return;
  if (mixed)
    k_load<true><<<grid_for_n(n), 256, 0, s>>>(box, (const float*)pos, (const float*)vel, err);
  else
    k_load<false><<<grid_for_n(n), 256, 0, s>>>(box, (const double*)pos, (const double*)vel, err);
}

template <bool MIXED>
static void extract(const BoxDev* box, real_t<MIXED>* pos, real_t<MIXED>* vel, int32_t* cell_out,
                    int ncells, int nsol, uint32_t* xcnt, cudaStream_t s) {
  const int warps = (ncells + 3) / 4;  // four cells each
  const int g = std::min(std::max((warps + BLOCK / 32 - 1) / (BLOCK / 32), 1), 65536);
  if ((size_t)nsol * 6 * sizeof(real_t<MIXED>) <= EXTRACT_DIRECT) {
    k_extract<MIXED><<<g, BLOCK, 0, s>>>(box, pos, vel, cell_out);
    return;
  }
  constexpr int N = 1 << xbucket_shift(MIXED);
  const int nb = xbuckets(MIXED, nsol);
  const size_t smem = (size_t)N * (6 * sizeof(real_t<MIXED>) + (cell_out ? sizeof(int32_t) : 0));
  cudaMemsetAsync(xcnt, 0, sizeof(uint32_t) * XCNT_STRIDE * nb, s);
  k_bucket<MIXED><<<g, BLOCK, 0, s>>>(box);
  k_unbucket<MIXED><<<nb, UT, smem, s>>>(box, pos, vel, cell_out);
}

int extract_prepare() {
  const int most = (1 << xbucket_shift(true)) * (6 * (int)sizeof(float) + (int)sizeof(int32_t));
  const int mostd = (1 << xbucket_shift(false)) * (6 * (int)sizeof(double) + (int)sizeof(int32_t));
  const cudaError_t e = cudaFuncSetAttribute(k_unbucket<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e != cudaSuccess) return (int)e;
  return (int)cudaFuncSetAttribute(k_unbucket<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mostd);
}

void launch_extract(bool mixed, const BoxDev* box, void* pos, void* vel, int32_t* cell_out,
                    int ncells, int nsol, uint32_t* xcnt, cudaStream_t s) {
  if (mixed) extract<true>(box, (float*)pos, (float*)vel, cell_out, ncells, nsol, xcnt, s);
  else extract<false>(box, (double*)pos, (double*)vel, cell_out, ncells, nsol, xcnt, s);
}

}  // namespace mpcd

namespace mpcd {

// ---------------------------------------------------------------------------
// Thermal initial state drawn on the device (input generation for batched and
// served jobs, not part of a step): positions uniform in the box, velocity
// components Gaussian with variance kT/m (Box-Muller), then the mean velocity
// removed, as the benchmark set-up of Sec. 4 / 4.1 does.  Particle i uses
// counters (i, 0..2) under its own purpose; the mean comes from exact int64
// fixed-point sums, so the state is reproducible.
// ---------------------------------------------------------------------------
constexpr uint32_t PURPOSE_INIT = 0x494E4954u;

struct InitParams {
  uint32_t seed_lo, seed_hi;
  double L[3];
  double sigma;
  int n;
};

__device__ __forceinline__ void init_draw(const InitParams& P, int i, double r[3], double v[3]) {
  const uint2 key = make_uint2(P.seed_lo, P.seed_hi ^ PURPOSE_INIT);
  const uint4 a = philox(make_uint4((uint32_t)i, 0u, 0u, 0u), key);
  const uint4 b = philox(make_uint4((uint32_t)i, 1u, 0u, 0u), key);
  const uint4 c = philox(make_uint4((uint32_t)i, 2u, 0u, 0u), key);
  r[0] = P.L[0] * ((double)a.x * 0x1p-32);
  r[1] = P.L[1] * ((double)a.y * 0x1p-32);
  r[2] = P.L[2] * ((double)a.z * 0x1p-32);
  const double u1 = unit53(b.x, b.y), u2 = unit53(b.z, b.w);
  const double u3 = unit53(c.x, c.y), u4 = unit53(c.z, c.w);
  const double rho1 = sqrt(-2.0 * log(1.0 - u1)), rho2 = sqrt(-2.0 * log(1.0 - u3));
  v[0] = P.sigma * (rho1 * cos(kTwoPi * u2));
  v[1] = P.sigma * (rho1 * sin(kTwoPi * u2));
  v[2] = P.sigma * (rho2 * cos(kTwoPi * u4));
}

__global__ void k_init_sum(InitParams P, unsigned long long* sums) {
  long long s[3] = {0, 0, 0};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
    double r[3], v[3];
    init_draw(P, i, r, v);
    for (int k = 0; k < 3; ++k) s[k] += __double2ll_rn(v[k] * 4294967296.0);
  }
  for (int k = 0; k < 3; ++k) {
    long long x = s[k];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xFFFFFFFFu, x, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&sums[k], (unsigned long long)x);
  }
}

template <bool MIXED>
__global__ void k_init_write(InitParams P, const unsigned long long* sums, real_t<MIXED>* pos,
                             real_t<MIXED>* vel) {
  using T = real_t<MIXED>;
  double mean[3];
  for (int k = 0; k < 3; ++k)
    mean[k] = P.n > 0 ? ((double)(long long)sums[k] * 0x1p-32) / (double)P.n : 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
    double r[3], v[3];
    init_draw(P, i, r, v);
    for (int k = 0; k < 3; ++k) {
      T x = (T)r[k];
      if (!((double)x < P.L[k])) x = (T)0;  // rounding up to L wraps to 0
      pos[3 * i + k] = x;
      vel[3 * i + k] = (T)(v[k] - mean[k]);
    }
  }
}

void launch_init_thermal(bool mixed, int n, uint64_t seed, const double L[3], double sigma,
                         void* pos, void* vel, unsigned long long* sums, cudaStream_t s) {
  if (n <= 0) return;
  InitParams P;
  P.seed_lo = (uint32_t)seed;
  P.seed_hi = (uint32_t)(seed >> 32);
  for (int k = 0; k < 3; ++k) P.L[k] = L[k];
  P.sigma = sigma;
  P.n = n;
  int g = (n + 255) / 256;
  if (g > 4096) g = 4096;
  cudaMemsetAsync(sums, 0, 3 * sizeof(unsigned long long), s);
  k_init_sum<<<g, 256, 0, s>>>(P, sums);
  if (mixed) k_init_write<true><<<g, 256, 0, s>>>(P, sums, (float*)pos, (float*)vel);
  else k_init_write<false><<<g, 256, 0, s>>>(P, sums, (double*)pos, (double*)vel);
}

}  // namespace mpcd
