// k_srd_d.cu -- the fused SRD step of the FP64 model with its per-member
// arithmetic on the integer pipe (arXiv:1801.10187: Sec. 2 Eqs. stream, srd and
// thermo; Sec. 3.4 cell list; Sec. 3.5 cell properties; Sec. 3.6 rotation and
// thermostat, algorithm "SRD collision rule").
//
// For periodic SRD boxes without solute, of at most SRDD_MAX_CELLS cells, whose
// rows hold at most SRDD_SLOTS records; modes, records and results (to rounding)
// are those of k_cells_warp_d.  An FP64 warp instruction holds GB300's FP64 pipe for 16 cycles,
// in which an SM issues 64 others, so k_cells_warp_d (82 % of the pipe busy) is
// bound by its 28 FP64 instructions a particle.  Here a cell has an exponent E
// with |v| < 2^E for all its members, and a velocity becomes the 60-bit integer
// V = v 2^(59 - E), truncated:
//   sums     Sum V per cell, exact (two 64-bit words a component)
//   cell     the axis and the rotation matrix R (in double, then as integers
//            R 2^62) for the warp's cells at once, one a lane, before the sums;
//            u = Sum V / n in double, then as an integer U
//   members  V' = U + R (V - U) in 32 x 32 -> 64 bit products of signed halves;
//            what is dropped (low x low) is below 3 units of 2^(E - 59)
// V resolves the cell's largest component to 2^-59, 64 times finer than a
// double's rounding of it, and a cell's mean, differences and products in double
// carry that rounding to all its members; so the only rounding of the size of the
// FP64 path's is the one of V' back to double.  (An exponent shared by the cells
// of a sub-tile would cost a cell beside a faster one its low bits.)  A lone member
// keeps its velocity, as v - u = 0 leaves it.  Streaming is the same fma.  With the
// thermostat the energy about u and the scaling by xi stay in double.  What bounds
// it now: 16 warps an SM (115 registers, 47 KB a block) that wait on the FP64 pipe
// (44 % busy at 50^3 cells) and the integer pipes (37 % of the issue slots) in turn,
// and on how many of its slots a sub-tile fills; the line beyond which
// k_cells_warp_d is taken is at SRDD_MAX_CELLS (kernels.h).  On small boxes a tile's
// latency is what counts, and 4 to 32 cells a warp spread them over the SMs (us a
// step): 10^3 cells at density 5 35 -> 12, with the thermostat 57 -> 22; 16^3 at
// density 10 51 -> 17; 24^3 52 -> 27; 50^3 143 -> 114.  A cell
// with an overflowing row, a non-finite velocity or an exponent beyond +-900 takes
// the same steps in double.
#include "dev_collide.cuh"
#include "dev_rows.cuh"
#include "dev_stream.cuh"
#include "kernels.h"
#include "mpcd_internal.cuh"

namespace mpcd {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int DB = 128;  // threads per block
constexpr int DWARPS = DB / 32;
constexpr int VBITS = 59;
constexpr int LONE = 1 << 20, DOUBLE = LONE + 1;  // in place of a cell's exponent

struct DBox {
  double dt, ca, sa, omc, m;
  double L[3], hg[3], gdt[3];
  double s[3];
  long long S[3];  // grid shift of the step the records are binned for
  int n[3], K;
  RecD* rows_cur;
  RecD* rows_out;
  uint32_t* cnt_out;
  RecD* ovf_out;
  uint32_t* ovf_cell_out;
  uint32_t* ovf_n_out;
  int ovf_cap, pad;
};

// q: quarters of the staged records, (x, y), (z, v_x), (v_y, v_z), (tag, ..);
// after the conversion v_* hold the integers V.  E: the cell's exponent, or LONE or
// DOUBLE (its members' v_* stay doubles).  R: rotation matrix as signed
// halves (hi, lo) of R 2^62, row by row; U: the cell's mean velocity as an integer;
// u, xi: in double (thermostat and the double path).
struct DWarp {
  float4 q[4][SRDD_SLOTS];
  int2 R[9][32];
  long long U[3][32];
  double u[3][32], xi[32];
  int E[32];
  unsigned short map[SRDD_SLOTS];  // place in the row << 5 | cell
};

__host__ __device__ constexpr size_t dhead() { return (sizeof(DBox) + 15) & ~(size_t)15; }
constexpr size_t DSMEM = dhead() + DWARPS * sizeof(DWarp);

__device__ __forceinline__ void cp_async16d(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}

// v 2^(VBITS - E), truncated, for |v| < 2^E (subnormals count as zero).
__device__ __forceinline__ long long to_fixed(double v, int E) {
  const long long b = __double_as_longlong(v);
  const int e = (int)(b >> 52) & 2047;
  // v = m 2^(e - 1075), so V = (m 2^(VBITS - 53)) 2^-(E + 1022 - e)
  const unsigned long long m = (unsigned long long)((b & 0x000FFFFFFFFFFFFFLL) | 0x0010000000000000LL)
                               << (VBITS - 53);
  const int sh = E + 1022 - e;
  const long long q = (e == 0 || sh > 63) ? 0ll : (long long)(m >> sh);
  return b < 0 ? -q : q;
}

// x truncated, for |x| < 2^62.
__device__ __forceinline__ long long truncate(double x) {
  const long long b = __double_as_longlong(x);
  const int sh = 1075 - ((int)(b >> 52) & 2047);
  const unsigned long long m = (unsigned long long)((b & 0x000FFFFFFFFFFFFFLL) | 0x0010000000000000LL);
  const long long q = sh > 63 ? 0ll : (long long)(sh >= 0 ? m >> sh : m << -sh);
  return b < 0 ? -q : q;
}

// The nearest double (ties to even) of V 2^(E - VBITS).
__device__ __forceinline__ double from_fixed(long long V, int E) {
  const unsigned long long a = V < 0 ? 0ull - (unsigned long long)V : (unsigned long long)V;
  const int lz = __clzll((long long)a);
  const unsigned long long t = a << (lz & 63);
  const unsigned low = (unsigned)t & 0x7FFu;
  const unsigned long long m = (t >> 11) + ((low + ((unsigned)(t >> 11) & 1u)) > 0x400u ? 1ull : 0ull);
  const long long r = (long long)(((unsigned long long)(unsigned)(1023 + E + 62 - VBITS - lz) << 52) + m);
  return __longlong_as_double(V == 0 ? 0ll : (V < 0 ? r | (long long)0x8000000000000000ull : r));
}

// x = hi 2^32 + lo with a signed lo.
__device__ __forceinline__ int2 halves(long long x) {
  return make_int2((int)((x + 0x80000000LL) >> 32), (int)x);
}

}  // namespace

template <bool THERMO, int MODE, bool FORCE>
__global__ void __launch_bounds__(DB, 4) k_srd_d(const BoxDev* __restrict__ boxes,
                                                 const int2* __restrict__ spans, int nspans, int cpw,
                                                 AfterPass after, int* err) {
  extern __shared__ __align__(16) unsigned char smem_[];
  DBox& H = *reinterpret_cast<DBox*>(smem_);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  DWarp& W = reinterpret_cast<DWarp*>(smem_ + dhead())[wid];
  const int parts = BLOCK / (DWARPS * cpw);  // blocks' work per 256-cell span
  int box_of_params = -1;
  const unsigned lt = (1u << lane) - 1u;
  for (int it = blockIdx.x; it < nspans * parts; it += gridDim.x) {
    const int sp = it / parts, part = it - sp * parts;
    const int2 tt = spans[sp];
    const BoxDev& B = boxes[tt.x];
    if (tt.x != box_of_params) {  // block-uniform
      __syncthreads();
      if (threadIdx.x < 3) {
        const int q = threadIdx.x;
        H.L[q] = B.L[q]; H.hg[q] = B.hg[q]; H.gdt[q] = B.gdt[q]; H.n[q] = B.n[q];
        if (MODE != MODE_C) {
          long long S[3];
          shift_units(B, B.step + (MODE == MODE_P ? 0ull : 1ull), S);
          H.S[q] = q == 0 ? S[0] : q == 1 ? S[1] : S[2];
          H.s[q] = (double)H.S[q] * 0x1p-32;
        }
      } else if (threadIdx.x == 32) {
        H.dt = B.dt; H.ca = B.ca; H.sa = B.sa; H.omc = B.omc; H.m = B.m;
        H.K = B.K;
        const int out = B.cur ^ 1;
        H.rows_cur = (RecD*)B.rows[B.cur];
        H.rows_out = (RecD*)B.rows[out];
        H.cnt_out = B.cnt[out];
        H.ovf_out = (RecD*)B.ovf_rec[out];
        H.ovf_cell_out = B.ovf_cell[out];
        H.ovf_n_out = &B.ovf_n[out];
        H.ovf_cap = B.ovf_cap;
      }
      __syncthreads();
      box_of_params = tt.x;
    }
    const int c0 = tt.y + (part * DWARPS + wid) * cpw;
    if (c0 >= B.ncells) continue;  // warp-uniform
    const int K = H.K;
    uint32_t n = 0u;
    if (lane < cpw && c0 + lane < B.ncells) {
      uint32_t* cn = B.cnt[B.cur] + (c0 + lane);
      n = *cn;
      if (MODE != MODE_C && n) *cn = 0u;  // this set is written two steps on
    }
    const int nrow = (int)n < K ? (int)n : K;
    int incl = nrow;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, d);
      if (lane >= d) incl += y;
    }
    if (__shfl_sync(FULL, incl, 31) == 0) continue;
    RecD* rows = H.rows_cur + (size_t)c0 * K;
    // f(record) for the members of cell c in the overflow list (rare)
    auto for_overflow = [&](int c, auto&& f) {
      RecD* ovf = (RecD*)B.ovf_rec[B.cur];
      const uint32_t* oc = B.ovf_cell[B.cur];
      const uint32_t novf = min(B.ovf_n[B.cur], (uint32_t)B.ovf_cap);
      for (uint32_t j = 0; j < novf; ++j)
        if (oc[j] == (uint32_t)c) f(ovf + j);
    };
    const int subc = cpw == 32 ? B.subw : min(B.subc, cpw);  // most cells per sub-tile, a power of two
    const int plog = __clz(subc) - 26;  // 2^plog = 32 / subc lanes add up a cell
    double ehat = -1.0;                 // thermostat: this lane's cell's draw, < 0: none

    for (int a = 0; a < cpw;) {
      // ---- the sub-tile: cells [a, b), members [first, first + cnt) ----
      const int first = __shfl_sync(FULL, incl - nrow, a);
      const int b =
          min(__popc(__ballot_sync(FULL, incl - first <= SRDD_SLOTS)), min(a + subc, cpw));
      const int cnt = __shfl_sync(FULL, incl, b - 1) - first;
      const bool mine = lane >= a && lane < b;
      const int s0 = incl - nrow - first;  // first member of this lane's cell
      __syncwarp();                        // the previous sub-tile is done with W
      if (mine) {
        int e = lane;
        for (int j = 0; j < nrow; ++j, e += 32) W.map[s0 + j] = (unsigned short)e;
      }
      __syncwarp();
      // records into shared memory, four neighbouring lanes copying one
      for (int q = lane; q < 4 * cnt; q += 32) {
        const int m = q >> 2, e = W.map[m];
        cp_async16d(&W.q[lane & 3][m],
                    reinterpret_cast<const float4*>(rows + ((e & 31) * K + (e >> 5))) + (lane & 3));
      }
      asm volatile("cp.async.commit_group;" ::: "memory");

      if (MODE != MODE_P && a == 0 && n > 0) {
        // ---- per cell, no sums needed: the axis (Sec. 3.6), R, the Gamma draw ----
        double nn[3];
        axis_of(B, B.step, (uint32_t)(c0 + lane), nn);
        const double ca = H.ca, sa = H.sa, omc = H.omc;
        // Rodrigues' R = cos I + sin [n]x + (1 - cos) n n^T
        auto put = [&](int k, double x) { W.R[k][lane] = halves(__double2ll_rn(x * 0x1p62)); };
        put(0, fma(omc * nn[0], nn[0], ca));
        put(4, fma(omc * nn[1], nn[1], ca));
        put(8, fma(omc * nn[2], nn[2], ca));
        put(1, fma(omc * nn[0], nn[1], -sa * nn[2]));
        put(3, fma(omc * nn[1], nn[0], sa * nn[2]));
        put(2, fma(omc * nn[0], nn[2], sa * nn[1]));
        put(6, fma(omc * nn[2], nn[0], -sa * nn[1]));
        put(5, fma(omc * nn[1], nn[2], -sa * nn[0]));
        put(7, fma(omc * nn[2], nn[1], sa * nn[0]));
        if (THERMO && (int)n >= 2 && !gamma_draw(B, B.step, (uint32_t)(c0 + lane), (int)n, ehat))
          ehat = -1.0;
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncwarp();  // every lane's copies are in shared memory

      double* const vx = reinterpret_cast<double*>(&W.q[1][0]) + 1;  // member m: vx[2 m]
      double2* const vyz = reinterpret_cast<double2*>(&W.q[2][0]);
      if (MODE != MODE_P) {
        // 2^plog lanes add up a cell; the first of them goes on
        const int cc = a + (lane >> plog), part_ = lane & ((1 << plog) - 1);
        const int src = cc < b ? cc : a;
        const int nC = __shfl_sync(FULL, (int)n, src), s0C = __shfl_sync(FULL, s0, src);
        const int nrowC = cc < b ? min(nC, K) : 0;
        const double ehatC = THERMO ? __shfl_sync(FULL, ehat, src) : 0.0;
        // ---- the cell's exponent ----
        unsigned top = 0u;
        for (int k = part_; k < nrowC; k += 1 << plog) {
          const double2 w = vyz[s0C + k];
          top = max(top, max((unsigned)__double2hiint(vx[2 * (s0C + k)]) & 0x7FFFFFFFu,
                             max((unsigned)__double2hiint(w.x) & 0x7FFFFFFFu,
                                 (unsigned)__double2hiint(w.y) & 0x7FFFFFFFu)));
        }
        for (int d = 1; d < (1 << plog); d <<= 1) top = max(top, __shfl_xor_sync(FULL, top, d));
        int E = (int)(top >> 20) - 1022;
        if (nC < 2 && E < 1025) E = LONE;  // (1025: not finite)
        else if (E <= -900 || E >= 900 || nC > K) E = DOUBLE;
        const bool plain = nrowC > 0 && E < LONE, dbl = nrowC > 0 && E == DOUBLE;

        // ---- velocities to integers in place, and their sums ----
        double u[3] = {0.0, 0.0, 0.0}, Ek = 0.0;
        unsigned long long lo[3] = {0ull, 0ull, 0ull};
        long long hi[3] = {0ll, 0ll, 0ll};
        if (plain)
          for (int k = part_; k < nrowC; k += 1 << plog) {
            const double2 w = vyz[s0C + k];
            const long long V[3] = {to_fixed(vx[2 * (s0C + k)], E), to_fixed(w.x, E),
                                    to_fixed(w.y, E)};
            vx[2 * (s0C + k)] = __longlong_as_double(V[0]);
            vyz[s0C + k] = make_double2(__longlong_as_double(V[1]), __longlong_as_double(V[2]));
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              lo[q] += (unsigned)V[q];
              hi[q] += (int)(V[q] >> 32);
            }
          }
        for (int d = 1; d < (1 << plog); d <<= 1) {
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            lo[q] += __shfl_xor_sync(FULL, lo[q], d);
            hi[q] += __shfl_xor_sync(FULL, hi[q], d);
          }
        }
        if (plain) {
          // u = Sum V / n: the sum (below 2^67) rounded once to double; every
          // lane of the cell forms it
          const double iM = 1.0 / ll2d_exact((long long)nC);
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const __int128 T = ((__int128)hi[q] << 32) + (__int128)lo[q];
            const double D = u128_to_double((unsigned __int128)(T < 0 ? -T : T));
            const double uf = (T < 0 ? -D : D) * iM;  // in units of 2^(E - VBITS)
            const long long U = truncate(uf);
            if (THERMO) u[q] = from_fixed(U, E);
            if (part_ == 0) W.U[q][cc] = U;
            if (THERMO) lo[q] = (unsigned long long)U;
          }
          if (THERMO)  // energy about u, from the exact differences
            for (int k = part_; k < nrowC; k += 1 << plog) {
              const double2 w = vyz[s0C + k];
              const long long V[3] = {__double_as_longlong(vx[2 * (s0C + k)]),
                                      __double_as_longlong(w.x), __double_as_longlong(w.y)};
#pragma unroll
              for (int q = 0; q < 3; ++q) {
                const double d = from_fixed(V[q] - (long long)lo[q], E);
                Ek = fma(d, d, Ek);
              }
            }
        }
        if (__any_sync(FULL, dbl)) {  // cells in double
          auto each = [&](auto&& f) {
            if (!dbl) return;
            for (int k = part_; k < nrowC; k += 1 << plog) f(vx[2 * (s0C + k)], vyz[s0C + k]);
            if (part_ == 0 && nC > K)
              for_overflow(c0 + cc, [&](const RecD* p) {
                double w[3];
                load_v(p, w);
                f(w[0], make_double2(w[1], w[2]));
              });
          };
          double su[3] = {0.0, 0.0, 0.0};
          each([&](double x, double2 y) {
            su[0] += x;
            su[1] += y.x;
            su[2] += y.y;
          });
          for (int d = 1; d < (1 << plog); d <<= 1)
#pragma unroll
            for (int q = 0; q < 3; ++q) su[q] += __shfl_xor_sync(FULL, su[q], d);
          if (dbl) {
            const double iM = 1.0 / ll2d_exact((long long)nC);
#pragma unroll
            for (int q = 0; q < 3; ++q) u[q] = su[q] * iM;
          }
          if (THERMO)
            each([&](double x, double2 y) {
              const double d0 = x - u[0], d1 = y.x - u[1], d2 = y.y - u[2];
              Ek += d0 * d0 + d1 * d1 + d2 * d2;
            });
        }
        double xi = 1.0;
        if (THERMO) {
          for (int d = 1; d < (1 << plog); d <<= 1) Ek += __shfl_xor_sync(FULL, Ek, d);
          Ek = (0.5 * H.m) * Ek;
          if (cc < b && nC >= 2 && Ek > 0.0) {
            if (ehatC >= 0.0) xi = sqrt(ehatC / Ek);
            else atomicOr(err, ERR_GAMMA_CAP);
          }
        }
        if (cc < b && part_ == 0) {
          W.E[cc] = E;
          if (THERMO || dbl) {
#pragma unroll
            for (int q = 0; q < 3; ++q) W.u[q][cc] = u[q];
            W.xi[cc] = xi;
          }
        }
        __syncwarp();
      }

      // ---- collide (Eq. srd), stream (Eq. stream), bin (Sec. 3.4) ----
      auto stream_bin = [&](double x[3], double w[3]) -> uint32_t {
        int c[3];
        bool bad = false;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          x[q] = fma(w[q], H.dt, x[q]);
          if (FORCE) {
            x[q] = x[q] + H.hg[q];
            w[q] = w[q] + H.gdt[q];
          }
          x[q] = wrap_bits(x[q], H.L[q]);
          int i = floor_minus_shift(x[q], H.S[q], H.s[q]);  // in [-1, n]
          if (i < 0) i += H.n[q];
          if (i >= H.n[q]) i -= H.n[q];
          if (i < 0 || i >= H.n[q]) {
            bad = true;
            i = 0;
          }
          c[q] = i;
        }
        if (bad) atomicOr(err, ERR_CELL_RANGE);
        return (uint32_t)(c[0] + H.n[0] * (c[1] + H.n[1] * c[2]));
      };
      // the collision in double (W.u, W.xi), for cell o
      auto collide_double = [&](double w[3], int o) {
        const double d[3] = {w[0] - W.u[0][o], w[1] - W.u[1][o], w[2] - W.u[2][o]};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          double s = 0.0;
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const int2 h = W.R[3 * i + k][o];
            s = fma((double)(((long long)h.x << 32) + h.y) * 0x1p-62, d[k], s);
          }
          w[i] = THERMO ? fma(W.xi[o], s, W.u[i][o]) : W.u[i][o] + s;
        }
      };
      auto emit = [&](const double x[3], const double w[3], uint32_t tg, uint32_t c2, uint32_t slot) {
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
      for (int base = 0; base < cnt; base += 32) {
        const int m = base + lane;
        const bool act = m < cnt;
        double x[3], w[3];
        uint32_t tag = 0u, c2 = FULL;
        if (act) {
          const int e = W.map[m], o = e & 31;
          const double2 xy = *reinterpret_cast<const double2*>(&W.q[0][m]);
          x[0] = xy.x;
          x[1] = xy.y;
          x[2] = vx[2 * m - 1];
          w[0] = vx[2 * m];
          const double2 yz = vyz[m];
          w[1] = yz.x;
          w[2] = yz.y;
          tag = __float_as_uint(W.q[3][m].x);
          if (MODE != MODE_P) {
            const int E = W.E[o];
            if (E < LONE) {
              // V' = U + R (V - U): |V - U| < 2^60, |R 2^62| <= 2^62, so the three
              // high products stay below 2^60 and the six mixed ones below 2^63
              int2 d[3];
#pragma unroll
              for (int k = 0; k < 3; ++k)
                d[k] = halves(__double_as_longlong(w[k]) - W.U[k][o]);
#pragma unroll
              for (int i = 0; i < 3; ++i) {
                long long hh = 0, mid = 0;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                  const int2 r = W.R[3 * i + k][o];
                  hh += (long long)r.x * d[k].x;
                  mid += (long long)r.x * d[k].y;
                  mid += (long long)r.y * d[k].x;
                }
                const long long D = (hh << 2) + (mid >> 30);
                w[i] = THERMO ? fma(W.xi[o], from_fixed(D, E), W.u[i][o])
                              : from_fixed(W.U[i][o] + D, E);
              }
            } else if (E == DOUBLE) {
              collide_double(w, o);
            }
          }
          if (MODE == MODE_C)
            store_rec(rows + (o * K + (e >> 5)), x, w, tag);
          else
            c2 = stream_bin(x, w);
        }
        if (MODE != MODE_C) {
          // the lanes bound for one cell share an atomic and take consecutive slots
          const unsigned peers = __match_any_sync(FULL, c2);
          const int leader = __ffs(peers) - 1;
          uint32_t slot0 = 0u;
          if (act && lane == leader) slot0 = atomicAdd(&H.cnt_out[c2], (uint32_t)__popc(peers));
          const uint32_t slot = __shfl_sync(FULL, slot0, leader) + (uint32_t)__popc(peers & lt);
          if (act) emit(x, w, tag, c2, slot);
        }
      }
      if (mine && (int)n > K)
        for_overflow(c0 + lane, [&](RecD* p) {
          double x[3], w[3];
          uint32_t tg;
          load_rec(p, x, w, tg);
          if (MODE != MODE_P) collide_double(w, lane);
          if (MODE == MODE_C) {
            store_rec(p, x, w, tg);
          } else {
            const uint32_t c = stream_bin(x, w);
            emit(x, w, tg, c, atomicAdd(&H.cnt_out[c], 1u));
          }
        });
      a = b;
    }
  }
  finish_pass(after);
}

template <int MODE>
static void* srdd_mode(bool thermo, bool force) {
  if (thermo && MODE != MODE_P)
    return force ? (void*)k_srd_d<true, MODE, true> : (void*)k_srd_d<true, MODE, false>;
  return force ? (void*)k_srd_d<false, MODE, true> : (void*)k_srd_d<false, MODE, false>;
}

static void* srdd_variant(bool thermo, bool force, int mode) {
  if (mode == MODE_P) return srdd_mode<MODE_P>(thermo, force);
  if (mode == MODE_F) return srdd_mode<MODE_F>(thermo, force);
  return srdd_mode<MODE_C>(thermo, force);
}

int srdd_blocks_per_sm(bool thermo, bool force, int mode) {
  const void* fn = srdd_variant(thermo, force, mode);
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DSMEM);
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, DB, DSMEM);
  return nb;
}

void launch_srdd(bool thermo, bool force, int mode, const BoxDev* boxes, const int2* spans,
                 int nspans, int grid, int cpw, AfterPass after, int* err, cudaStream_t s) {
  if (nspans <= 0) return;
  void* args[] = {(void*)&boxes, (void*)&spans, (void*)&nspans, (void*)&cpw, (void*)&after, (void*)&err};
  cudaLaunchKernel(srdd_variant(thermo, force, mode), dim3(grid), dim3(DB), args, DSMEM, s);
}

}  // namespace mpcd
