// capi.cu -- host engine and C ABI of libmpcd (see include/mpcd.h).
//
// An Engine holds one or more independent boxes of one precision.  Each box
// owns its device arrays (stream-ordered allocations); a host-built table of
// BoxDev records plus span tables (256 cells per span, one list per kernel
// variant) lets every launch cover all boxes.
//
// Stepping.  One fused pass per step (k_cells, mode F) collides step t and
// streams and bins step t + 1.  The state therefore rests "half a step on":
// after mpcd_step the last collision is still pending.  Reading the state (or
// changing the set of boxes) first completes it (mode C, in place); stepping
// from a completed state first streams and bins (mode P).  Consecutive
// mpcd_step calls thus cost exactly one pass per step.  The P, F and C passes
// are each captured once into a CUDA graph and replayed; step counters and the
// buffer flips live in the device records.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <thread>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/mpcd.h"
#include "kernels.h"
#include "mpcd_internal.cuh"

using namespace mpcd;

namespace {

thread_local std::string g_last_error;

int fail(int code, const std::string& msg) {
  g_last_error = msg;
  return code;
}

#define CUDA_TRY(expr)                                                                     \
  do {                                                                                     \
    cudaError_t e_ = (expr);                                                               \
    if (e_ != cudaSuccess) {                                                               \
      if (e_ == cudaErrorMemoryAllocation)                                                 \
        return fail(MPCD_ENOMEM, std::string(#expr) + ": " + cudaGetErrorString(e_));      \
      return fail(MPCD_ECUDA, std::string(#expr) + ": " + cudaGetErrorString(e_));         \
    }                                                                                      \
  } while (0)

size_t elem_size(bool mixed) { return mixed ? sizeof(float) : sizeof(double); }
size_t rec_size(bool mixed) { return mixed ? sizeof(RecF) : sizeof(RecD); }

int64_t cells_of(const mpcd_params& p) {
  return (int64_t)p.n[0] * p.n[1] * (p.n[2] + (p.walls_z ? 2 : 0));
}

// Records per cell row: the mean occupancy plus six standard deviations of a
// Poisson count and a margin, rounded up to a multiple of 4.  Busier cells
// spill into the overflow list, which stays correct for any input.
int row_capacity(const mpcd_params& p, int64_t nsol) {
  const double V = (double)p.n[0] * p.n[1] * p.n[2];
  const double rho = V > 0 ? (double)nsol / V : 0.0;
  int K = (int)std::ceil(rho + 6.0 * std::sqrt(rho) + 4.0);
  if (K < 8) K = 8;
  return (K + 3) & ~3;
}

size_t footprint_bytes(const mpcd_params& p, int64_t nsol, int64_t nbead) {
  const bool mixed = p.precision == MPCD_MIXED;
  const int64_t C = cells_of(p);
  const int K = row_capacity(p, nsol);
  const int64_t ng = (C + BEAD_TILE - 1) / BEAD_TILE;
  size_t b = 0;
  b += 2 * (size_t)C * K * rec_size(mixed);                               // rows
  b += 2 * (size_t)C * sizeof(uint32_t);                                  // counts
  b += 2 * (size_t)std::max<int64_t>(nsol, 1) * (rec_size(mixed) + 4);     // overflow lists
  b += (size_t)nsol * 6 * elem_size(mixed);                               // staging (r, v)
  b += (size_t)xbuckets(mixed, nsol) * XCNT_STRIDE * sizeof(uint32_t);    // read-out buckets
  if (mixed && p.walls_z) b += 4 * (size_t)p.n[0] * p.n[1] * (4 * sizeof(long long) + 4);
  if (nbead > 0) {
    b += (size_t)nbead * (9 * sizeof(double) + 2 * sizeof(int32_t) + sizeof(uint64_t) +
                          2 * sizeof(uint32_t));
    b += (size_t)ng * sizeof(uint32_t) + (size_t)(ng + 1) * sizeof(uint32_t);
    if (p.lj_epsilon > 0.0)  // neighbour list: buckets, next, key, count, list, build r, forces
      b += (size_t)(2 * ((nbead + PTILE - 1) / PTILE) * PTILE) * sizeof(int32_t) +
           (size_t)nbead * (3 * sizeof(int32_t) + NL_MAX * sizeof(int32_t) + 12 * sizeof(double) +
                            2 * sizeof(int4));
  }
  return b;
}

int validate(const mpcd_params* p, int precision_expected) {
  if (!p) return fail(MPCD_EINVAL, "params is NULL");
  for (int k = 0; k < 3; ++k)
    if (p->n[k] < 1) return fail(MPCD_EINVAL, "n[k] must be >= 1");
  if (p->precision != MPCD_FP64 && p->precision != MPCD_MIXED)
    return fail(MPCD_EINVAL, "precision must be MPCD_FP64 or MPCD_MIXED");
  if (precision_expected >= 0 && p->precision != precision_expected)
    return fail(MPCD_EINVAL, "box precision differs from the batch precision");
  if (p->a != 1.0) return fail(MPCD_EINVAL, "cell edge a must be 1 (lengths in units of a)");
  if (!(p->dt > 0.0) || !std::isfinite(p->dt)) return fail(MPCD_EINVAL, "dt must be > 0");
  if (!(p->mass > 0.0)) return fail(MPCD_EINVAL, "mass must be > 0");
  if (!(p->kT >= 0.0)) return fail(MPCD_EINVAL, "kT must be >= 0");
  if (!std::isfinite(p->alpha)) return fail(MPCD_EINVAL, "alpha must be finite");
  if (p->walls_z && p->body_force[2] != 0.0)
    return fail(MPCD_EINVAL, "body_force[2] must be 0 with walls_z");
  if (p->walls_z && p->chain_len > 0) return fail(MPCD_EINVAL, "solute with walls is not supported");
  if (p->collision != MPCD_SRD && p->collision != MPCD_AT)
    return fail(MPCD_EINVAL, "collision must be MPCD_SRD or MPCD_AT");
  if (p->collision == MPCD_AT && (p->thermostat || p->walls_z))
    return fail(MPCD_EINVAL, "the Andersen rule thermostats by itself: no thermostat flag, no walls");
  if (p->angular && (p->walls_z || p->chain_len > 0))
    return fail(MPCD_EINVAL, "angular momentum conservation takes neither walls nor solute");
  if (!(p->lj_epsilon >= 0.0)) return fail(MPCD_EINVAL, "lj_epsilon must be >= 0");
  if (p->lj_epsilon > 0.0) {
    if (!(p->lj_sigma > 0.0) || std::pow(2.0, 1.0 / 6.0) * p->lj_sigma + NL_SKIN > 1.0)
      return fail(MPCD_EINVAL, "WCA repulsion needs 0 < 2^(1/6) lj_sigma <= 0.6 (cutoff plus the "
                               "0.4 neighbour-list buffer within one cell)");
    if (p->n[0] < 3 || p->n[1] < 3 || p->n[2] < 3)
      return fail(MPCD_EINVAL, "WCA repulsion needs at least 3 cells per axis");
  }
  if (p->chain_len < 0 || p->chain_len > 1024) return fail(MPCD_EINVAL, "chain_len in [0, 1024]");
  if (p->chain_len > 0 && (p->md_substeps < 1 || !(p->solute_mass > 0.0)))
    return fail(MPCD_EINVAL, "solute needs md_substeps >= 1 and solute_mass > 0");
  const int64_t C = cells_of(*p);
  if (C > 2000000000LL) return fail(MPCD_EINVAL, "too many cells (max 2e9)");
  return MPCD_OK;
}

// Whether a kernel of this device may store `bytes` bytes of elements of size `es`
// at p: aligned device memory of its own, all of them within one allocation.  A copy
// is checked by the driver, and reaches other devices' memory; a kernel's store is not.
bool own_device_memory(const void* p, size_t bytes, size_t es, int device) {
  using Range = int (*)(unsigned long long*, size_t*, unsigned long long);  // cuMemGetAddressRange
  static const Range range = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &q) !=
            cudaSuccess || q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      f = nullptr;
    }
    return (Range)f;
  }();
  if (!range || (uintptr_t)p % es != 0) return false;
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();  // not this call's failure: the copy will say
    return false;
  }
  if (at.type != cudaMemoryTypeDevice || at.device != device) return false;
  unsigned long long base = 0;
  size_t size = 0;
  if (range(&base, &size, (unsigned long long)(uintptr_t)p) != 0) return false;
  const unsigned long long off = (unsigned long long)(uintptr_t)p - base;
  return off <= size && bytes <= size - off;
}

// ---------------------------------------------------------------------------
// Host <-> device transfer of the solvent state.  The host arrays are double;
// the mixed model keeps float on the device.  The values move in chunks of
// XFER_ELEMS: host threads convert (or copy) each chunk into a page-locked
// slot and queue a cudaMemcpyAsync from it, so conversion, DMA and page
// faults of fresh host buffers proceed in parallel.  Slots come from a
// process-wide pool and are kept for reuse by later transfers and contexts.
// ---------------------------------------------------------------------------
constexpr size_t XFER_ELEMS = size_t(1) << 19;
constexpr size_t XFER_SLOT_BYTES = XFER_ELEMS * sizeof(double);
constexpr int XFER_MAX_THREADS = 16;

std::mutex g_slot_mu;
std::vector<void*> g_free_slots;

void* take_slot() {
  {
    std::lock_guard<std::mutex> lk(g_slot_mu);
    if (!g_free_slots.empty()) {
      void* q = g_free_slots.back();
      g_free_slots.pop_back();
      return q;
    }
  }
  void* q = nullptr;
  return cudaMallocHost(&q, XFER_SLOT_BYTES) == cudaSuccess ? q : nullptr;
}

void give_slot(void* q) {
  if (!q) return;
  std::lock_guard<std::mutex> lk(g_slot_mu);
  g_free_slots.push_back(q);
}

// One host array and its device counterpart (n values each).
struct XferSeg {
  double* host;
  void* dev;
  size_t n;
};

// Moves every segment host -> device (to_dev) or device -> host, converting
// between double and float when mixed.  Returns the first CUDA error.
cudaError_t transfer(bool to_dev, bool mixed, const XferSeg* seg, int nseg, int device,
                     cudaStream_t stream) {
  const size_t es = mixed ? sizeof(float) : sizeof(double);
  std::vector<size_t> first(nseg + 1, 0);  // first chunk of each segment
  for (int i = 0; i < nseg; ++i)
    first[i + 1] = first[i] + (seg[i].n + XFER_ELEMS - 1) / XFER_ELEMS;
  const size_t nchunks = first[nseg];
  if (nchunks == 0) return cudaSuccess;
  std::atomic<size_t> next{0};
  std::atomic<int> err{(int)cudaSuccess};

  auto work = [&](bool set_device) {
    if (set_device) cudaSetDevice(device);
    void* slot[2] = {take_slot(), take_slot()};
    cudaEvent_t ev[2] = {nullptr, nullptr};
    cudaError_t e = (slot[0] && slot[1]) ? cudaSuccess : cudaErrorMemoryAllocation;
    for (int j = 0; j < 2 && e == cudaSuccess; ++j)
      e = cudaEventCreateWithFlags(&ev[j], cudaEventDisableTiming);
    bool used[2] = {false, false};
    for (size_t i = 0; e == cudaSuccess && err.load() == (int)cudaSuccess; ++i) {
      const size_t k = next.fetch_add(1);
      if (k >= nchunks) break;
      int s = 0;
      while (k >= first[s + 1]) ++s;
      const size_t off = (k - first[s]) * XFER_ELEMS;
      const size_t len = std::min(XFER_ELEMS, seg[s].n - off);
      char* dev = (char*)seg[s].dev + off * es;
      const int j = (int)(i & 1);
      if (to_dev) {
        if (used[j] && (e = cudaEventSynchronize(ev[j])) != cudaSuccess) break;
        const double* src = seg[s].host + off;
        if (mixed) {
          float* dst = (float*)slot[j];
          for (size_t q = 0; q < len; ++q) dst[q] = (float)src[q];
        } else {
          std::memcpy(slot[j], src, len * sizeof(double));
        }
        if ((e = cudaMemcpyAsync(dev, slot[j], len * es, cudaMemcpyHostToDevice, stream)) != cudaSuccess)
          break;
      } else {
        if ((e = cudaMemcpyAsync(slot[j], dev, len * es, cudaMemcpyDeviceToHost, stream)) != cudaSuccess)
          break;
      }
      if ((e = cudaEventRecord(ev[j], stream)) != cudaSuccess) break;
      used[j] = true;
      if (!to_dev) {
        if ((e = cudaEventSynchronize(ev[j])) != cudaSuccess) break;
        double* dst = seg[s].host + off;
        if (mixed) {
          const float* src = (const float*)slot[j];
          for (size_t q = 0; q < len; ++q) dst[q] = (double)src[q];
        } else {
          std::memcpy(dst, slot[j], len * sizeof(double));
        }
      }
    }
    // a slot goes back to the pool only once its copy has finished
    for (int j = 0; j < 2; ++j) {
      if (ev[j]) {
        const cudaError_t w = used[j] ? cudaEventSynchronize(ev[j]) : cudaSuccess;
        if (e == cudaSuccess) e = w;
        cudaEventDestroy(ev[j]);
      }
      give_slot(slot[j]);
    }
    if (e != cudaSuccess) {
      int ok = (int)cudaSuccess;
      err.compare_exchange_strong(ok, (int)e);
    }
  };

  unsigned hw = std::thread::hardware_concurrency();
  const size_t nthreads =
      std::min<size_t>(nchunks, std::max<unsigned>(1u, std::min<unsigned>(hw, XFER_MAX_THREADS)));
  std::vector<std::thread> pool;
  for (size_t t = 1; t < nthreads; ++t) pool.emplace_back(work, true);
  work(false);
  for (auto& th : pool) th.join();
  return (cudaError_t)err.load();
}

struct Box {
  mpcd_params p{};
  int64_t nsol = 0, nbead = 0;
  BoxDev d{};                  // host mirror of the device record
  std::vector<void*> allocs;   // device allocations of this box
  size_t bytes = 0;
  bool has_state = false;
  int dev_index = -1;          // index in the device table, -1 if not uploaded
  void* stage_r = nullptr;     // n x 3 staging arrays (input order)
  void* stage_v = nullptr;
  void* obs = nullptr;         // observables scratch (allocated lazily)
  size_t obs_bytes = 0;
};

}  // namespace

struct Engine {
  bool mixed = true;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int device = 0;
  int nsm = 1;
  int64_t max_bytes = 0;
  size_t used_bytes = 0;
  std::vector<Box*> slots;
  std::vector<Box*> live;  // boxes in the device table

  // device tables
  BoxDev* d_boxes = nullptr;
  int n_records = 0;
  // per kernel variant: thermostat (1) | walls or beads (2) | warp-spread members (4);
  // for the warp-spread kernel bit 2 means a nonzero body force, bit 8 beads
  // and bit 16 the Andersen rule
  // per-cell kernel: bit 16 the Andersen rule, bit 32 the angular correction;
  // bit 64: k_srd or k_srd_d (bits 1, 2 and 8 as for the warp-spread kernel; bit 4 walls)
  static constexpr int NVAR = 128;
  int2* d_spans[NVAR] = {};
  int n_spans[NVAR] = {};
  ScanSeg* d_bsegs = nullptr;
  int2* d_bstiles = nullptr;
  int n_bstiles = 0;
  int2* d_btiles = nullptr;
  int n_btiles = 0;
  int2* d_mdtiles = nullptr;
  int n_mdtiles = 0;
  int2* d_vtiles = nullptr;  // wall-cut layers of the boxes with virtual particles
  int n_vtiles = 0;
  int2* d_wtiles = nullptr;  // beads of the boxes with the repulsion
  int n_wtiles = 0;
  unsigned* d_wsync = nullptr;  // their MD's barrier count and flags
  int wca_bps = 1;
  int md_chains_per_block = 1, md_threads = 32;
  uint32_t* d_tsum = nullptr;
  unsigned long long* d_gscan = nullptr;
  uint32_t* d_toff = nullptr;
  int* d_err = nullptr;
  unsigned* d_done = nullptr;  // finished blocks of the launch that ends a pass, of k_virtual
  cudaStream_t side = nullptr;  // k_virtual beside the fused pass, between two events
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  double* d_partials = nullptr;
  bool any_beads = false;
  int wca_substeps = 0;  // most MD substeps of a box with the WCA repulsion (0: none)
  int cells_bps[3][NVAR] = {};
  int srd_bead_bps[3][8] = {};  // k_srd's launch over the groups with beads
  // k_srd: cells per warp chosen by the launch tuner (0: by size)
  int tuned_cpw = 0;

  // MODE_P, MODE_F, MODE_C, and GRAPH_STEPS passes of mode F: a graph takes about
  // 10 us to launch, which is longer than a step of a small box (16^3 cells at
  // density 10: 10.3 us a step with a launch each).
  cudaGraphExec_t gexec[4] = {nullptr, nullptr, nullptr, nullptr};
  static constexpr int GRAPH_MANY = 3, GRAPH_STEPS = 16;
  bool tables_ok = false;
  bool pending = false;  // the last collision of every live box is still to do

  int init(int precision, void* user_stream) {
    mixed = precision == MPCD_MIXED;
    CUDA_TRY(cudaGetDevice(&device));
    cudaDeviceProp prop;
    CUDA_TRY(cudaGetDeviceProperties(&prop, device));
    nsm = prop.multiProcessorCount;
    if (user_stream) {
      stream = (cudaStream_t)user_stream;
    } else {
      CUDA_TRY(cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking));
      own_stream = true;
    }
    CUDA_TRY((cudaError_t)md_bin_prepare());
    CUDA_TRY((cudaError_t)extract_prepare());
    CUDA_TRY(cudaMalloc(&d_err, sizeof(int)));
    CUDA_TRY(cudaMemsetAsync(d_err, 0, sizeof(int), stream));
    CUDA_TRY(cudaMalloc(&d_partials, sizeof(double) * 4 * 4096));
    CUDA_TRY(cudaMalloc(&d_done, 2 * sizeof(unsigned)));
    CUDA_TRY(cudaMemsetAsync(d_done, 0, 2 * sizeof(unsigned), stream));
    CUDA_TRY(cudaMalloc(&d_wsync, sizeof(unsigned) * 4));
    wca_bps = std::max(1, wca_blocks_per_sm());
    // keep freed box memory cached in the pool for quick re-admission
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, device) == cudaSuccess) {
      uint64_t thr = UINT64_MAX;
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
    return MPCD_OK;
  }

  // Blocks per SM of a kernel variant in every mode (asked for when a box first
  // needs the variant: there are too many to ask for all when an engine starts).
  void prepare_variant(int v) {
    for (int m = 0; m < 3 && cells_bps[2][v] == 0; ++m) {
      const bool at = (v & 16) != 0, ang = (v & 32) != 0;
      cells_bps[m][v] = 1;
      if (v & 64) {
        if (!mixed) {
          cells_bps[m][v] = srdd_blocks_per_sm((v & 1) != 0, (v & 2) != 0, m);
        } else {
          cells_bps[m][v] = srd_blocks_per_sm((v & 1) != 0, (v & 2) != 0, false, (v & 4) != 0, at, ang, m);
          if (v & 8)
            srd_bead_bps[m][v & 7] =
                std::max(1, srd_blocks_per_sm((v & 1) != 0, (v & 2) != 0, true, false, false, false, m));
        }
      } else if ((v & 4) && ang) {  // warp-spread angular correction: mixed SRD without beads
        if (mixed && !(v & (8 | 16)))
          cells_bps[m][v] = cells_warp_blocks_per_sm((v & 1) != 0, (v & 2) != 0, false, false, true, m);
      } else if ((v & 4) && !(at && (v & 1))) {
        cells_bps[m][v] =
            mixed ? cells_warp_blocks_per_sm((v & 1) != 0, (v & 2) != 0, (v & 8) != 0, at, false, m)
                  : cells_warpd_blocks_per_sm((v & 1) != 0, (v & 2) != 0, (v & 8) != 0, at, m);
      } else if (!(v & 4)) {
        cells_bps[m][v] = cells_blocks_per_sm(mixed, v, m);
      }
      cells_bps[m][v] = std::max(1, cells_bps[m][v]);
    }
  }

  void free_tables() {
    void* ptrs[] = {d_boxes, d_bsegs, d_bstiles, d_btiles, d_mdtiles, d_vtiles, d_wtiles, d_tsum, d_gscan, d_toff};
    for (void* q : ptrs)
      if (q) cudaFree(q);
    for (int v = 0; v < NVAR; ++v) {
      if (d_spans[v]) cudaFree(d_spans[v]);
      d_spans[v] = nullptr;
      n_spans[v] = 0;
    }
    d_boxes = nullptr; d_bsegs = nullptr; d_bstiles = nullptr; d_btiles = nullptr;
    d_mdtiles = nullptr; d_vtiles = nullptr; d_wtiles = nullptr; d_tsum = nullptr; d_gscan = nullptr; d_toff = nullptr;
    n_records = 0;
    n_vtiles = 0;
    n_wtiles = 0;
  }

  void drop_graphs() {
    for (auto& g : gexec) {
      if (g) cudaGraphExecDestroy(g);
      g = nullptr;
    }
  }

  ~Engine() {
    if (stream) cudaStreamSynchronize(stream);
    drop_graphs();
    if (side) cudaStreamDestroy(side);  // (joined to stream at every pass)
    if (ev_fork) cudaEventDestroy(ev_fork);
    if (ev_join) cudaEventDestroy(ev_join);
    for (Box* b : slots) release_box(b);
    free_tables();
    if (d_err) cudaFree(d_err);
    if (d_partials) cudaFree(d_partials);
    if (d_wsync) cudaFree(d_wsync);
    if (d_done) cudaFree(d_done);
    if (own_stream && stream) cudaStreamDestroy(stream);
  }

  void free_box_arrays(Box* b) {
    for (void* q : b->allocs)
      if (q) cudaFreeAsync(q, stream);
    b->allocs.clear();
    if (b->obs) cudaFreeAsync(b->obs, stream);
    b->obs = nullptr;
    b->obs_bytes = 0;
    b->stage_r = b->stage_v = nullptr;
    used_bytes -= b->bytes;
    b->bytes = 0;
  }

  void release_box(Box* b) {
    if (!b) return;
    free_box_arrays(b);
    delete b;
  }

  int pull_records() {
    if (!d_boxes || live.empty() || n_records == 0) return MPCD_OK;
    std::vector<BoxDev> rec(n_records);
    CUDA_TRY(cudaMemcpyAsync(rec.data(), d_boxes, sizeof(BoxDev) * n_records,
                             cudaMemcpyDeviceToHost, stream));
    CUDA_TRY(cudaStreamSynchronize(stream));
    for (Box* b : live)
      if (b->dev_index >= 0 && b->dev_index < n_records) b->d = rec[b->dev_index];
    return MPCD_OK;
  }

  // Forget a box that is about to be freed or re-set (state must be complete).
  void unlink(Box* b) {
    for (size_t i = 0; i < live.size(); ++i)
      if (live[i] == b) {
        live.erase(live.begin() + i);
        break;
      }
    b->dev_index = -1;
    drop_graphs();
    tables_ok = false;
  }

  int check_err() {
    int h = 0;
    CUDA_TRY(cudaMemcpyAsync(&h, d_err, sizeof(int), cudaMemcpyDeviceToHost, stream));
    CUDA_TRY(cudaStreamSynchronize(stream));
    if (h) {
      CUDA_TRY(cudaMemsetAsync(d_err, 0, sizeof(int), stream));
      std::string m;
      if (h & ERR_GAMMA_CAP) m += "thermostat Gamma sampler rejected 64 draws; ";
      if (h & ERR_CELL_RANGE) m += "a position was not finite (cell id clamped); ";
      if (h & ERR_OVERFLOW_CAP) m += "cell overflow list full; ";
      if (h & ERR_BARRIER) m += "solute MD: the blocks of a launch did not meet; ";
      if (h & ERR_NLIST) m += "solute neighbour list: a bead had more than 64 neighbours; ";
      return fail(MPCD_EDEVICE, m);
    }
    return MPCD_OK;
  }

  int rebuild() {
    int rc = pull_records();
    if (rc) return rc;
    drop_graphs();
    free_tables();
    live.clear();
    for (Box* b : slots)
      if (b) b->dev_index = -1;
    for (Box* b : slots)
      if (b && b->has_state) live.push_back(b);
    tables_ok = true;
    if (live.empty()) return MPCD_OK;
    std::vector<BoxDev> rec;
    std::vector<int2> sp[NVAR], bst, bt, mt, vt, wt;
    std::vector<ScanSeg> bseg;
    any_beads = false;
    wca_substeps = 0;
    int max_cl = 1, total_chains = 0;
    for (Box* b : live)
      if (b->nbead > 0) {
        max_cl = std::max(max_cl, (int)b->p.chain_len);
        total_chains += (int)(b->nbead / b->p.chain_len);
      }
    // A block runs its chains' substeps one after another on the FP64 pipe of
    // one SM: with few chains, put fewer in each block so that they spread
    // over the SMs (two blocks per SM before a block takes a second chain).
    md_chains_per_block = std::max(1, std::min(BLOCK / max_cl, total_chains / (2 * nsm)));
    md_threads = ((md_chains_per_block * max_cl + 31) / 32) * 32;
    for (size_t i = 0; i < live.size(); ++i) {
      Box* b = live[i];
      b->dev_index = (int)i;
      rec.push_back(b->d);
      const BoxDev& d = b->d;
      const bool at = d.collision == RULE_AT;
      int variant = (d.thermostat ? 1 : 0) | ((d.walls || d.nbead > 0) ? 2 : 0) | (at ? 16 : 0) |
                    (d.angular ? 32 : 0);
      const bool warp_ang = mixed && !at && d.nbead == 0;
      if (on_srd(d) && d.walls) variant = 64 | 4 | (d.thermostat ? 1 : 0);
      if ((!d.angular || warp_ang) && !d.walls && d.K <= WARP_MAX_K &&
          std::max(d.n[0], std::max(d.n[1], d.n[2])) < (1 << 22)) {
        const bool force = d.g[0] != 0.0 || d.g[1] != 0.0 || d.g[2] != 0.0;
        variant = (on_srd(d) ? 64 : 4) | (d.thermostat ? 1 : 0) | (force ? 2 : 0) |
                  (d.nbead > 0 ? 8 : 0) | (at ? 16 : 0) | (d.angular ? 32 : 0);
      }
      if (on_srd(d) && d.walls)
        for (int i0 = 0; i0 < 2 * d.n[0] * d.n[1]; i0 += VIRT_CELLS) vt.push_back(make_int2((int)i, i0));
      for (int c0 = 0; c0 < d.ncells; c0 += BLOCK) sp[variant].push_back(make_int2((int)i, c0));
      if (d.nbead > 0) {
        any_beads = true;
        if (d.wca) {
          wca_substeps = std::max(wca_substeps, (int)d.md_substeps);
          for (int b0 = 0; b0 < d.nbead; b0 += WCA_BEADS) wt.push_back(make_int2((int)i, b0));
        }
        bseg.push_back(ScanSeg{d.bcount, d.bstart, d.nctiles, 0});
        for (int c0 = 0; c0 < d.nctiles; c0 += STILE)
          bst.push_back(make_int2((int)bseg.size() - 1, c0));
        for (int b0 = 0; b0 < d.nbead; b0 += PTILE) bt.push_back(make_int2((int)i, b0));
        const int nchains = d.nbead / d.chain_len;
        for (int c0 = 0; c0 < nchains; c0 += md_chains_per_block) mt.push_back(make_int2((int)i, c0));
      }
    }
    auto up = [&](auto& vec, auto*& dptr, int* count) -> int {
      using E = typename std::remove_reference<decltype(vec)>::type::value_type;
      if (count) *count = (int)vec.size();
      if (vec.empty()) return MPCD_OK;
      CUDA_TRY(cudaMalloc((void**)&dptr, sizeof(E) * vec.size()));
      CUDA_TRY(cudaMemcpyAsync(dptr, vec.data(), sizeof(E) * vec.size(), cudaMemcpyHostToDevice,
                               stream));
      return MPCD_OK;
    };
    if ((rc = up(rec, d_boxes, &n_records))) return rc;
    for (int v = 0; v < NVAR; ++v) {
      if ((rc = up(sp[v], d_spans[v], &n_spans[v]))) return rc;
      if (n_spans[v] > 0) prepare_variant(v);
    }
    if ((rc = up(bseg, d_bsegs, nullptr))) return rc;
    if ((rc = up(bst, d_bstiles, &n_bstiles))) return rc;
    if ((rc = up(bt, d_btiles, &n_btiles))) return rc;
    if ((rc = up(mt, d_mdtiles, &n_mdtiles))) return rc;
    if ((rc = up(vt, d_vtiles, &n_vtiles))) return rc;
    if (n_vtiles > 0 && !side) {
      CUDA_TRY(cudaEventCreateWithFlags(&ev_fork, cudaEventDisableTiming));
      CUDA_TRY(cudaEventCreateWithFlags(&ev_join, cudaEventDisableTiming));
      CUDA_TRY(cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking));
    }
    if ((rc = up(wt, d_wtiles, &n_wtiles))) return rc;
    if (n_bstiles > 0) {
      CUDA_TRY(cudaMalloc(&d_tsum, sizeof(uint32_t) * n_bstiles));
      CUDA_TRY(cudaMalloc(&d_gscan, sizeof(unsigned long long) * n_bstiles));
      CUDA_TRY(cudaMalloc(&d_toff, sizeof(uint32_t) * n_bstiles));
    }
    CUDA_TRY(cudaStreamSynchronize(stream));
    return MPCD_OK;
  }

  int grid_for(int n, int per_sm) const {
    const int g = nsm * per_sm;
    return n < g ? std::max(n, 1) : g;
  }

  // Solute boxes (mixed): whether k_srd's two launches, over the bead groups without
  // beads and with, beat k_cells_warp's one.  What they save grows with the cells, more
  // so with long rows and with the thermostat of short ones; what they cost is a
  // launch and dearer bead groups, and with the thermostat sub-tiles whose cells often
  // do not all fit.  Time of k_srd over that of k_cells_warp either side of the lines,
  // with w = 0.2 / 0.7 / 2 beads a group: density 5 to 10, 90^3 cells 1.01 / 1.01 / 1.08,
  // 100^3 0.98 / 1.02 / 1.04, 112^3 0.94 / 0.98 / 1.04, 160^3 0.92 / 0.95 / 0.99; with the
  // thermostat density 5 80^3 1.02 / 0.99 / 1.00, 90^3 0.97 / 0.96 / 0.98, density 12 to 15
  // 100^3 1.02 / 1.08 / 1.11, 128^3 0.97 / 1.03 / 1.09; density 20 64^3 0.94 / 0.94 / 0.97, with
  // the thermostat 64^3 1.03 / 1.02 / 1.05, 80^3 0.91 / 0.91 / 1.01, 100^3 0.82 / 0.88 / 0.96.
  bool solute_pays(const BoxDev& d) const {
    const double rho = (double)d.nsol / (double)d.ncells, mean = rho * d.subw;
    const double w = (double)d.nbead / (double)d.nctiles;
    const bool few = w <= 0.45, many = w > 1.3, fits = mean + std::sqrt(mean) <= SRD_SLOTS;
    double cells;
    if (rho >= 18.0)
      cells = !d.thermostat ? 0.23e6 : !many ? 0.45e6 : fits ? 0.9e6 : 5e6;
    else if (d.thermostat && !fits)
      cells = few ? 1.2e6 : 5e6;
    else if (d.thermostat && rho < 6.0)
      cells = 0.6e6;
    else
      cells = few ? 0.9e6 : many ? 3.5e6 : 1.2e6;
    return (double)d.ncells >= cells;
  }

  // Boxes that k_srd (mixed) or k_srd_d (FP64) steps.
  bool on_srd(const BoxDev& d) const {
    if (!mixed && (d.walls || d.nbead > 0 || d.K > SRDD_SLOTS || d.ncells > SRDD_MAX_CELLS)) return false;
    if (d.collision == RULE_AT && (!mixed || d.nbead > 0 || d.angular)) return false;
    if (d.angular && !mixed) return false;
    if (d.nbead > 0 && !solute_pays(d)) return false;
    return d.K <= SRD_SLOTS &&
           std::max(d.n[0], std::max(d.n[1], d.n[2])) < (1 << 22);
  }

  // Cells per warp of k_srd and k_srd_d: as chosen by the tuner, else the
  // most of 32, 16, 8 and 4 that still gives every SM SRD_MIN_WARPS (FP64:
  // SRDD_MIN_WARPS) warps, that is between half and all of what fits on it.
  int srd_cpw() const {
    if (tuned_cpw) return tuned_cpw;
    int64_t cells = 0;
    for (int v = 64; v < NVAR; ++v) cells += (int64_t)n_spans[v] * BLOCK;
    int cpw = 32;
    while (cpw > 4 && cells < (int64_t)cpw * (mixed ? SRD_MIN_WARPS : SRDD_MIN_WARPS) * nsm) cpw >>= 1;
    return cpw;
  }

  // Mixed SRD variants of k_cells_warp, whose mode F takes the tuner's cells per warp.
  bool narrows(int v) const { return mixed && (v & 4) && !(v & (16 | 32 | 64)); }
  int warp_cpw(int v, int mode) const {
    return narrows(v) && mode == MODE_F && tuned_cpw ? std::max(tuned_cpw, 8) : 32;
  }

  // Grid of the fused pass: tuned_grid 0 = the occupancy limit (blocks per
  // SM that fit), k > 0 = at most k blocks per SM, -1 = one block per span
  // part (a 256-cell span is taken in parts where a warp has fewer than 32 cells).
  int tuned_grid = 0;
  int grid_of(int v, int mode) const {
    const int items = n_spans[v] * ((v & 64) ? srd_parts(srd_cpw()) : 32 / warp_cpw(v, mode));
    if (mode == MODE_F && tuned_grid == -1) return std::max(items, 1);
    const int limit = cells_bps[mode][v];
    return grid_for(items, (mode == MODE_F && tuned_grid > 0) ? std::min(tuned_grid, limit) : limit);
  }

  // One pass over every box.  The record updates that end it are done by the last
  // launch itself where that is k_srd or k_srd_d (they come last), else left to
  // end_pass, by a kernel of their own.
  void launch_cells_all(int mode) {
    const AfterPass none{};
    AfterPass end{d_boxes, (int)live.size(), mode != MODE_C, mode != MODE_P, d_done};
    const int last = last_variant();
    for (int v = 0; v < NVAR; ++v) {
      if (n_spans[v] == 0) continue;
      const int grid = grid_of(v, mode);
      const bool at = (v & 16) != 0;
      const AfterPass after = v == last ? end : none;
      if ((v & 64) && !mixed) {
        launch_srdd((v & 1) != 0, (v & 2) != 0, mode, d_boxes, d_spans[v], n_spans[v], grid,
                    srd_cpw(), after, d_err, stream);
      } else if (v & 64) {
        const bool beads = (v & 8) && mode != MODE_P;  // then a second launch, over their groups
        launch_srd((v & 1) != 0, (v & 2) != 0, false, (v & 4) != 0, at, (v & 32) != 0, mode, d_boxes, d_spans[v],
                   n_spans[v], grid, srd_cpw(), beads ? none : after, d_err, stream);
        if (beads)
          launch_srd((v & 1) != 0, (v & 2) != 0, true, (v & 4) != 0, false, false, mode, d_boxes, d_spans[v],
                     n_spans[v], grid_for(srd_bead_items(n_spans[v]), srd_bead_bps[mode][v & 7]), 32,
                     after, d_err, stream);
      } else if ((v & 4) && mixed) {
        launch_cells_warp((v & 1) != 0, (v & 2) != 0, (v & 8) != 0, at, (v & 32) != 0, mode,
                          d_boxes, d_spans[v], n_spans[v], grid, warp_cpw(v, mode), d_err, stream);
      } else if (v & 4) {
        launch_cells_warpd((v & 1) != 0, (v & 2) != 0, (v & 8) != 0, at, mode, d_boxes,
                           d_spans[v], n_spans[v], grid, d_err, stream);
      } else {
        launch_cells(mixed, v, mode, d_boxes, d_spans[v], n_spans[v], grid, d_err, stream);
      }
    }
  }
  void end_pass(int mode) {
    if (last_variant() < 64)
      launch_after_pass(d_boxes, (int)live.size(), mode != MODE_C, mode != MODE_P, stream);
  }
  int last_variant() const {
    int last = -1;
    for (int v = 0; v < NVAR; ++v)
      if (n_spans[v] > 0) last = v;
    return last;
  }

  // Solute: MD substeps and bead grouping for the step in the records.  Returns the
  // error of the cooperative launch, which a device may refuse where it takes others.
  cudaError_t launch_beads() {
    if (!any_beads) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    if (wca_substeps > 0)
      e = (cudaError_t)launch_wca_md(d_boxes, d_wtiles, n_wtiles, wca_substeps, wca_bps * nsm, d_wsync,
                                     d_err, stream);
    launch_md_bin(d_boxes, d_mdtiles, n_mdtiles, md_chains_per_block, md_threads, d_err, stream);
    launch_scan(d_bsegs, d_bstiles, n_bstiles, d_tsum, d_gscan, d_toff, grid_for(n_bstiles, 8),
                stream);
    launch_bead_scatter(d_boxes, d_btiles, n_btiles, stream);
    return e;
  }

  // One pass over every live box (plain launches; captured into the graphs).
  cudaError_t enqueue_pass(int mode) {
    if (live.empty()) return cudaSuccess;
    // Virtual wall particles: the first pass needs them before its collision can
    // follow; a fused pass draws those of the next step beside itself.
    if (n_vtiles > 0 && mode == MODE_F) {
      cudaEventRecord(ev_fork, stream);
      cudaStreamWaitEvent(side, ev_fork, 0);
      launch_virtual(d_boxes, (int)live.size(), d_vtiles, n_vtiles, 0, d_done + 1, side);
      cudaEventRecord(ev_join, side);
    }
    launch_cells_all(mode);
    end_pass(mode);
    if (n_vtiles > 0 && mode == MODE_F) cudaStreamWaitEvent(stream, ev_join, 0);
    if (n_vtiles > 0 && mode == MODE_P)
      launch_virtual(d_boxes, (int)live.size(), d_vtiles, n_vtiles, 1, d_done + 1, stream);
    return mode != MODE_C ? launch_beads() : cudaSuccess;
  }

  int ensure_tables() {
    if (!tables_ok) return rebuild();
    return MPCD_OK;
  }

  int ensure_graph(int mode) {
    int rc = ensure_tables();
    if (rc) return rc;
    if (gexec[mode]) return MPCD_OK;
    cudaGraph_t g = nullptr;
    CUDA_TRY(cudaStreamBeginCapture(stream, cudaStreamCaptureModeThreadLocal));
    cudaError_t le = cudaSuccess;  // of a launch: the graph would lack it
    for (int i = 0; i < (mode == GRAPH_MANY ? GRAPH_STEPS : 1) && le == cudaSuccess; ++i)
      le = enqueue_pass(mode == GRAPH_MANY ? MODE_F : mode);
    cudaError_t e = cudaStreamEndCapture(stream, &g);
    if (le != cudaSuccess) {
      if (e == cudaSuccess) cudaGraphDestroy(g);
      cudaGetLastError();
      return fail(MPCD_ECUDA, std::string("launch: ") + cudaGetErrorString(le));
    }
    if (e != cudaSuccess) return fail(MPCD_ECUDA, std::string("capture: ") + cudaGetErrorString(e));
    e = cudaGraphInstantiate(&gexec[mode], g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return fail(MPCD_ECUDA, std::string("instantiate: ") + cudaGetErrorString(e));
    return MPCD_OK;
  }

  int run_pass(int mode) {
    int rc = ensure_graph(mode);
    if (rc) return rc;
    if (live.empty()) return MPCD_OK;
    CUDA_TRY(cudaGraphLaunch(gexec[mode], stream));
    return MPCD_OK;
  }

  int step(int64_t n) {
    if (n < 0) return fail(MPCD_EINVAL, "nsteps < 0");
    int rc = ensure_tables();
    if (rc) return rc;
    if (n == 0 || live.empty()) return MPCD_OK;
    if (!pending) {
      if ((rc = run_pass(MODE_P))) return rc;
      pending = true;
      n -= 1;
    }
    if (n >= 2 * GRAPH_STEPS) {
      if ((rc = ensure_graph(GRAPH_MANY))) return rc;
      for (; n >= GRAPH_STEPS; n -= GRAPH_STEPS) CUDA_TRY(cudaGraphLaunch(gexec[GRAPH_MANY], stream));
    }
    if (n > 0) {
      if ((rc = ensure_graph(MODE_F))) return rc;
      for (int64_t i = 0; i < n; ++i) CUDA_TRY(cudaGraphLaunch(gexec[MODE_F], stream));
    }
    CUDA_TRY(cudaGetLastError());
    return MPCD_OK;
  }

  // Launch tuner.  The paper tunes its kernels' launch parameters at run time
  // on real steps (Sec. 3.5, Sec. 4).  Here each candidate of the fused pass
  // -- grid (1 .. occupancy-limit blocks per SM, and one block per span part)
  // times, for k_srd, k_srd_d and the SRD variants of k_cells_warp, the cells per
  // warp (32, 16 or 8, and 4 where that is the width by size) -- runs `reps` real
  // steps, timed with CUDA events on the stream; the fastest is kept and the step
  // graph re-captured.  Results do
  // not depend on the candidate: the mixed model's cell sums are exact, the
  // FP64 ones differ at rounding.
  int tune(int64_t reps, int32_t* chosen, double* best_ms, int64_t* steps_taken,
           int32_t* chosen_chunk, int32_t* chosen_cpw) {
    if (reps < 1) return fail(MPCD_EINVAL, "steps per candidate < 1");
    int rc = ensure_tables();
    if (rc) return rc;
    int64_t taken = 0;
    if (live.empty()) {
      if (steps_taken) *steps_taken = 0;
      return MPCD_OK;
    }
    if (!pending) {
      if ((rc = run_pass(MODE_P))) return rc;
      pending = true;
      taken += 1;
    }
    bool any_srd = false, any_width = false;
    for (int v = 0; v < NVAR; ++v)
      if (n_spans[v] > 0) {
        any_srd |= (v & 64) != 0;
        any_width |= (v & 64) || narrows(v);
      }
    tuned_cpw = 0;
    const int by_size = srd_cpw();
    std::vector<int> widths = {32};  // cells per warp
    if (any_width) widths = {32, 16, 8};
    if (any_srd && by_size < 8) widths.push_back(by_size);  // what the boxes have untuned
    cudaEvent_t e0, e1;
    CUDA_TRY(cudaEventCreate(&e0));
    CUDA_TRY(cudaEventCreate(&e1));
    double best = 1e30;
    int best_c = 0, best_cpw = 32;
    for (int width : widths) {
      tuned_cpw = width;
      int maxbps = 1;
      for (int v = 0; v < NVAR; ++v)
        if (n_spans[v] > 0) maxbps = std::max(maxbps, cells_bps[MODE_F][v]);
      std::vector<int> cand;
      for (int k = 1; k <= maxbps; ++k) cand.push_back(k);
      cand.push_back(-1);
      for (int c : cand) {
        tuned_grid = c;
        CUDA_TRY(cudaEventRecord(e0, stream));
        for (int64_t r = 0; r < reps; ++r) CUDA_TRY(enqueue_pass(MODE_F));
        CUDA_TRY(cudaEventRecord(e1, stream));
        CUDA_TRY(cudaEventSynchronize(e1));
        float ms = 0.f;
        CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
        taken += reps;
        if (ms / (double)reps < best) {
          best = ms / (double)reps;
          best_c = c;
          best_cpw = tuned_cpw;
        }
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    tuned_grid = best_c;
    tuned_cpw = best_cpw;
    drop_graphs();
    CUDA_TRY(cudaGetLastError());
    if (chosen) *chosen = best_c;
    if (chosen_chunk) *chosen_chunk = 3;
    if (chosen_cpw) *chosen_cpw = std::max(best_cpw, 8);  // 8 stands for the narrower too
    if (best_ms) *best_ms = best;
    if (steps_taken) *steps_taken = taken;
    return check_err();
  }

  // Finish the pending collision so the records hold a completed step.
  int complete() {
    int rc = ensure_tables();
    if (rc) return rc;
    if (!pending) return MPCD_OK;
    if ((rc = run_pass(MODE_C))) return rc;
    pending = false;
    return MPCD_OK;
  }

  // Internal profiler: eager steps with an event after each phase.
  static constexpr int kPhases = 3;
  int timed_steps(int64_t n, double* ms) {
    int rc = complete();
    if (rc) return rc;
    for (int i = 0; i < kPhases; ++i) ms[i] = 0.0;
    if (live.empty() || n <= 0) return kPhases;
    // the first pass streams and bins (it is not one of the timed steps)
    CUDA_TRY(enqueue_pass(MODE_P));
    pending = true;
    cudaEvent_t ev[kPhases + 1];
    for (auto& e : ev) CUDA_TRY(cudaEventCreate(&e));
    for (int64_t s = 0; s < n; ++s) {
      CUDA_TRY(cudaEventRecord(ev[0], stream));
      if (n_vtiles > 0)
        launch_virtual(d_boxes, (int)live.size(), d_vtiles, n_vtiles, 0, d_done + 1, stream);
      launch_cells_all(MODE_F);
      CUDA_TRY(cudaEventRecord(ev[1], stream));
      end_pass(MODE_F);
      CUDA_TRY(cudaEventRecord(ev[2], stream));
      CUDA_TRY(launch_beads());
      CUDA_TRY(cudaEventRecord(ev[3], stream));
      CUDA_TRY(cudaEventSynchronize(ev[3]));
      for (int i = 0; i < kPhases; ++i) {
        float t = 0.f;
        CUDA_TRY(cudaEventElapsedTime(&t, ev[i], ev[i + 1]));
        ms[i] += t;
      }
    }
    for (auto& e : ev) cudaEventDestroy(e);
    for (int i = 0; i < kPhases; ++i) ms[i] /= (double)n;
    CUDA_TRY(cudaGetLastError());
    return kPhases;
  }

  template <typename P>
  int alloc(Box* b, P*& ptr, size_t count) {
    ptr = nullptr;
    if (count == 0) return MPCD_OK;
    void* q = nullptr;
    CUDA_TRY(cudaMallocAsync(&q, count * sizeof(P), stream));
    b->allocs.push_back(q);
    ptr = (P*)q;
    return MPCD_OK;
  }
  int alloc_bytes(Box* b, void*& ptr, size_t bytes) {
    ptr = nullptr;
    if (bytes == 0) return MPCD_OK;
    CUDA_TRY(cudaMallocAsync(&ptr, bytes, stream));
    b->allocs.push_back(ptr);
    return MPCD_OK;
  }

  // Allocate a box's arrays and fill its record (no particles placed yet).
  int setup_box(Box* b, int64_t nsol, int64_t nbead) {
    const mpcd_params& p = b->p;
    const int64_t C = cells_of(p);
    if (nsol < 0 || nsol > 2000000000LL || nbead < 0 || nbead > 100000000LL)
      return fail(MPCD_EINVAL, "particle count out of range");
    if (nbead > 0 && (p.chain_len < 1 || nbead % p.chain_len != 0))
      return fail(MPCD_EINVAL, "n_solute must be a positive multiple of chain_len");
    const size_t need = footprint_bytes(p, nsol, nbead);
    if (max_bytes > 0 && used_bytes + need > (size_t)max_bytes)
      return fail(MPCD_ENOMEM, "box does not fit in the memory budget");
    BoxDev& d = b->d;
    std::memset(&d, 0, sizeof(d));
    for (int k = 0; k < 3; ++k) d.n[k] = p.n[k];
    d.walls = p.walls_z ? 1 : 0;
    d.nzl = p.n[2] + (d.walls ? 2 : 0);
    d.ncells = (int32_t)C;
    d.nsol = (int32_t)nsol;
    d.nbead = (int32_t)nbead;
    d.chain_len = p.chain_len;
    d.md_substeps = p.md_substeps;
    d.thermostat = p.thermostat ? 1 : 0;
    d.collision = p.collision;
    d.K = row_capacity(p, nsol);
    d.angular = p.angular ? 1 : 0;
    // k_srd, k_srd_d: cells per sub-tile, as many as rarely have more members than the
    // staging area holds (subc).  With 32 cells a warp the area has to be full in FP64
    // and with the thermostat (subw): there a sub-tile of half its slots costs nearly as
    // much as one of all (us a step: 100^3 cells with the thermostat, density 11 291 ->
    // 257 with 16 cells for 8, 45 1053 -> 839 with 4 for 2; FP64 58^3, density 12 225 ->
    // 192), so a few cells may not fit and wait for the next one.  One lane a cell (32)
    // and one of two cells left over are not worth that; nor are the mixed model's other
    // rules, which would lose 2 to 5 % at 64^3.
    auto widest = [&](auto&& fits) {
      int c = 32;
      while (c > 1 && !fits(c, (double)nsol / (double)C * c)) c >>= 1;
      return c;
    };
    const double slots = mixed ? SRD_SLOTS : SRDD_SLOTS;
    auto rarely = [&](int, double mean) { return mean + 2.5 * std::sqrt(mean) <= slots; };
    auto full = [&](int c, double mean) {
      return c == 32 ? rarely(c, mean) : mean <= (c > 2 ? (mixed ? 1.25 : 1.3) * slots : slots);
    };
    d.subc = d.subw = widest(rarely);
    if (!mixed || (d.thermostat && !d.angular && !d.walls)) d.subw = widest(full);
    if (d.collision == RULE_AT && nbead > 0 &&
        (d.K > WARP_MAX_K || std::max(p.n[0], std::max(p.n[1], p.n[2])) >= (1 << 22)))
      return fail(MPCD_EINVAL, "the Andersen rule with solute needs a row capacity <= 448 "
                               "(density below about 300) and fewer than 2^22 cells per axis");
    d.ovf_cap = (int32_t)std::max<int64_t>(nsol, 1);
    d.tc = BEAD_TILE;
    d.nctiles = (int32_t)((C + BEAD_TILE - 1) / BEAD_TILE);
    d.seed_lo = (uint32_t)p.seed;
    d.seed_hi = (uint32_t)(p.seed >> 32);
    d.dt = p.dt;
    d.kT = p.kT;
    d.m = p.mass;
    d.Mb = p.solute_mass;
    d.bond_k = p.bond_k;
    d.bond_r0 = p.bond_r0;
    const double V = (double)p.n[0] * p.n[1] * p.n[2];
    d.virt_density = p.virt_density > 0.0 ? p.virt_density : (double)nsol / V;
    d.sigma_virt = std::sqrt(p.kT / p.mass);
    d.sig = std::sqrt(p.kT / p.mass);
    d.sigb = p.solute_mass > 0.0 ? std::sqrt(p.kT / p.solute_mass) : 0.0;
    d.sig_f = (float)d.sig;
    d.sigb_f = (float)d.sigb;
    d.ca = std::cos(p.alpha);
    d.sa = std::sin(p.alpha);
    d.omc = 1.0 - d.ca;
    for (int k = 0; k < 3; ++k) {
      d.g[k] = p.body_force[k];
      d.hg[k] = ((0.5 * p.body_force[k]) * p.dt) * p.dt;
      d.gdt[k] = p.body_force[k] * p.dt;
      d.L[k] = (double)p.n[k];
      d.g_f[k] = (float)d.g[k];
      d.hg_f[k] = (float)d.hg[k];
      d.gdt_f[k] = (float)d.gdt[k];
      d.L_f[k] = (float)d.L[k];
    }
    if (p.md_substeps > 0) {
      d.md_h = p.dt / (double)p.md_substeps;
      d.md_hh = (0.5 * d.md_h) / p.solute_mass;
    }
    d.hm2 = ((0.5 * p.mass) * p.mass) * 0x1p-64;
    d.dt_f = (float)p.dt;
    d.kT_f = (float)p.kT;
    d.m_f = (float)p.mass;
    d.Mb_f = (float)p.solute_mass;
    d.ca_f = (float)d.ca;
    d.sa_f = (float)d.sa;
    d.omc_f = (float)d.omc;
    const size_t rs = rec_size(mixed), es = elem_size(mixed);
    int rc;
    for (int s = 0; s < 2; ++s) {
      if ((rc = alloc_bytes(b, d.rows[s], (size_t)C * d.K * rs))) return rc;
      if ((rc = alloc(b, d.cnt[s], (size_t)C))) return rc;
      if ((rc = alloc_bytes(b, d.ovf_rec[s], (size_t)d.ovf_cap * rs))) return rc;
      if ((rc = alloc(b, d.ovf_cell[s], (size_t)d.ovf_cap))) return rc;
      CUDA_TRY(cudaMemsetAsync(d.cnt[s], 0, sizeof(uint32_t) * C, stream));
    }
    if ((rc = alloc(b, d.ovf_n, 2))) return rc;
    CUDA_TRY(cudaMemsetAsync(d.ovf_n, 0, sizeof(uint32_t) * 2, stream));
    if ((rc = alloc(b, d.xcnt, (size_t)xbuckets(mixed, nsol) * XCNT_STRIDE))) return rc;
    if (d.walls && on_srd(d)) {
      const size_t cut = 2 * (size_t)d.n[0] * d.n[1];
      for (int k = 0; k < 2; ++k) {
        if ((rc = alloc(b, d.virt_n[k], cut))) return rc;
        if ((rc = alloc(b, d.virt_sum[k], 4 * cut))) return rc;
      }
    }
    if ((rc = alloc_bytes(b, b->stage_r, (size_t)nsol * 3 * es))) return rc;
    if ((rc = alloc_bytes(b, b->stage_v, (size_t)nsol * 3 * es))) return rc;
    if (nbead > 0) {
      if ((rc = alloc(b, d.spos, (size_t)nbead * 3))) return rc;
      if ((rc = alloc(b, d.svel, (size_t)nbead * 3))) return rc;
      if ((rc = alloc(b, d.bcell, (size_t)nbead))) return rc;
      if ((rc = alloc(b, d.bkey, (size_t)nbead))) return rc;
      if ((rc = alloc(b, d.border, (size_t)nbead))) return rc;
      if ((rc = alloc(b, d.bgc, (size_t)nbead))) return rc;
      if ((rc = alloc(b, d.bgv, (size_t)nbead * 3))) return rc;
      if ((rc = alloc(b, d.bcount, (size_t)d.nctiles))) return rc;
      if ((rc = alloc(b, d.bstart, (size_t)d.nctiles + 1))) return rc;
      d.listed = mixed && on_srd(d) ? 1 : 0;
      if (d.listed && (rc = alloc(b, d.bgroup, (size_t)nbead))) return rc;
      CUDA_TRY(cudaMemsetAsync(d.bcount, 0, sizeof(uint32_t) * d.nctiles, stream));
      CUDA_TRY(cudaMemsetAsync(d.bstart, 0, sizeof(uint32_t) * (d.nctiles + 1), stream));
      if (p.lj_epsilon > 0.0) {  // non-bonded WCA repulsion (Sec. 4.3 reading)
        const double s2 = p.lj_sigma * p.lj_sigma;
        const double rcut = std::pow(2.0, 1.0 / 6.0) * p.lj_sigma;
        d.wca = 1;
        d.lj_eps = p.lj_epsilon;
        d.lj_sig2 = s2;
        d.wca_rc2 = std::pow(2.0, 1.0 / 3.0) * s2;
        d.wca_rl2 = (rcut + NL_SKIN) * (rcut + NL_SKIN);
        d.wca_half_skin2 = 0.25 * NL_SKIN * NL_SKIN;
        d.nl_hsize = (int32_t)(2 * ((nbead + PTILE - 1) / PTILE) * PTILE);
        if ((rc = alloc(b, d.nl_head, (size_t)d.nl_hsize))) return rc;
        if ((rc = alloc(b, d.nl_next, (size_t)nbead))) return rc;
        if ((rc = alloc(b, d.nl_key, (size_t)nbead))) return rc;
        if ((rc = alloc(b, d.nl_cnt, (size_t)nbead))) return rc;
        if ((rc = alloc(b, d.nl_nbr, (size_t)nbead * NL_MAX))) return rc;
        if ((rc = alloc(b, d.nl_rb, (size_t)nbead * 3))) return rc;
        if ((rc = alloc(b, d.bF, (size_t)nbead * 3))) return rc;
        double lmax = 0.0;
        for (int k = 0; k < 3; ++k) {
          d.wfrac[k] = 4294967296.0 / d.L[k];
          lmax = std::max(lmax, d.L[k]);
        }
        // float distances of the fractions: a few units of 2^-24, and at most
        // two fractions' 2^-32 L an axis
        d.wca_rc2f = (float)(d.wca_rc2 * (1.0 + 1e-5) + 16.0 * lmax * 0x1p-32 * rcut);
        for (int k = 0; k < 2; ++k) {
          if ((rc = alloc(b, d.wpos[k], (size_t)nbead * 3))) return rc;
          if ((rc = alloc(b, d.wfix[k], (size_t)nbead))) return rc;
        }
      }
    }
    d.cur = 0;
    b->nsol = nsol;
    b->nbead = nbead;
    b->bytes = need;
    used_bytes += need;
    return MPCD_OK;
  }

  // Place particles (device arrays of the storage type) into a set-up box.
  // The box record goes to a one-entry scratch table for the load.
  int place(Box* b, const void* dpos, const void* dvel, const double* spos, const double* svel,
            uint64_t step) {
    BoxDev& d = b->d;
    d.step = d.virt_step = step;
    d.nbgroup = 0u;
    d.cur = 0;
    BoxDev* tmp = nullptr;
    CUDA_TRY(cudaMallocAsync((void**)&tmp, sizeof(BoxDev), stream));
    CUDA_TRY(cudaMemcpyAsync(tmp, &d, sizeof(BoxDev), cudaMemcpyHostToDevice, stream));
    launch_load(mixed, tmp, dpos, dvel, (int)b->nsol, d_err, stream);
    if (b->nbead > 0) {
      CUDA_TRY(cudaMemcpyAsync(d.spos, spos, sizeof(double) * 3 * b->nbead, cudaMemcpyHostToDevice,
                               stream));
      CUDA_TRY(cudaMemcpyAsync(d.svel, svel, sizeof(double) * 3 * b->nbead, cudaMemcpyHostToDevice,
                               stream));
    }
    CUDA_TRY(cudaFreeAsync(tmp, stream));
    CUDA_TRY(cudaStreamSynchronize(stream));
    CUDA_TRY(cudaGetLastError());
    b->has_state = true;
    return check_err();
  }

  int upload_state(Box* b, const double* pos, const double* vel, const double* spos,
                   const double* svel, uint64_t step) {
    const size_t n3 = (size_t)b->nsol * 3;
    if (b->nsol > 0) {
      const XferSeg seg[2] = {{const_cast<double*>(pos), b->stage_r, n3},
                              {const_cast<double*>(vel), b->stage_v, n3}};
      CUDA_TRY(transfer(true, mixed, seg, 2, device, stream));
    }
    return place(b, b->stage_r, b->stage_v, spos, svel, step);
  }

  // Thermal initial state drawn on the device (see launch_init_thermal).
  int thermal_state(Box* b, uint64_t init_seed, uint64_t step) {
    unsigned long long* sums = nullptr;
    CUDA_TRY(cudaMallocAsync((void**)&sums, 3 * sizeof(unsigned long long), stream));
    const double L[3] = {(double)b->p.n[0], (double)b->p.n[1], (double)b->p.n[2]};
    launch_init_thermal(mixed, (int)b->nsol, init_seed, L, std::sqrt(b->p.kT / b->p.mass),
                        b->stage_r, b->stage_v, sums, stream);
    CUDA_TRY(cudaFreeAsync(sums, stream));
    CUDA_TRY(cudaGetLastError());
    return place(b, b->stage_r, b->stage_v, nullptr, nullptr, step);
  }

  // The last step completed, and the state in input order into the given device
  // arrays or (NULL) the box's staging arrays; reports device errors.  Waits for the
  // state, or (ahead) only for the step before it: then the copies that a caller
  // queues next find the kernels still at work, and what the driver does on the host
  // for a copy to fresh memory (page faults: 2 ms for 40 MB) is done meanwhile.
  int extract(Box* b, int32_t* cell_out, void* pos = nullptr, void* vel = nullptr, bool ahead = false) {
    int rc = complete();
    if (!rc && ahead) rc = check_err();
    if (rc) return rc;
    launch_extract(mixed, d_boxes + b->dev_index, pos ? pos : b->stage_r, vel ? vel : b->stage_v,
                   cell_out, (int)b->d.ncells, (int)b->nsol, b->d.xcnt, stream);
    CUDA_TRY(cudaGetLastError());
    return ahead ? MPCD_OK : check_err();
  }

  int download_state(Box* b, double* pos, double* vel, double* spos, double* svel, uint64_t* step) {
    // a caller that wants only the beads does not pay for the solvent
    const bool solvent = b->nsol > 0 && (pos || vel);
    // (ahead: the threads of a long transfer start while the read-out runs)
    const bool ahead = solvent && 3 * (size_t)b->nsol > XFER_ELEMS;
    int rc = complete();
    if (!rc && ahead && step) rc = pull_records();
    if (!rc) rc = solvent ? extract(b, nullptr, nullptr, nullptr, ahead) : check_err();
    if (!rc && !ahead && step) rc = pull_records();
    if (rc) return rc;
    const size_t n3 = (size_t)b->nsol * 3;
    if (solvent) {
      XferSeg seg[2];
      int nseg = 0;
      if (pos) seg[nseg++] = {pos, b->stage_r, n3};
      if (vel) seg[nseg++] = {vel, b->stage_v, n3};
      CUDA_TRY(transfer(false, mixed, seg, nseg, device, stream));
    }
    if (b->nbead > 0) {
      if (spos) CUDA_TRY(cudaMemcpyAsync(spos, b->d.spos, sizeof(double) * 3 * b->nbead,
                                         cudaMemcpyDeviceToHost, stream));
      if (svel) CUDA_TRY(cudaMemcpyAsync(svel, b->d.svel, sizeof(double) * 3 * b->nbead,
                                         cudaMemcpyDeviceToHost, stream));
    }
    CUDA_TRY(cudaStreamSynchronize(stream));
    if (step) *step = b->d.step;
    return MPCD_OK;
  }

  int observables(Box* b, mpcd_obs* out) {
    if (!out) return fail(MPCD_EINVAL, "out is NULL");
    int rc = extract(b, nullptr);
    if (!rc) rc = pull_records();  // the step counter
    if (rc) return rc;
    const mpcd_params& p = b->p;
    const int nc = p.n[0] * p.n[1] * p.n[2];
    const size_t need = (size_t)nc * (sizeof(uint32_t) + 5 * sizeof(long long)) + 64;
    if (b->obs_bytes < need) {
      if (b->obs) cudaFreeAsync(b->obs, stream);
      b->obs = nullptr;
      CUDA_TRY(cudaMallocAsync(&b->obs, need, stream));
      b->obs_bytes = need;
    }
    ObsCells oc;
    char* base = (char*)b->obs;
    oc.mass = b->nbead > 0 ? (long long*)base : nullptr;
    oc.mass_one = p.mass * 4294967296.0;
    oc.p = (long long*)base + nc;
    oc.k = oc.p + 3 * (size_t)nc;
    oc.cnt = (uint32_t*)(oc.k + nc);
    oc.ncells = nc;
    oc.p_unit = 0x1p-32;
    oc.v_scale = 0.0f;
    if (mixed && b->nbead == 0 && p.mass > 0x1p-100 && p.mass < 0x1p100) {
      int e;
      const double f = std::frexp(p.mass, &e);  // in [1/2, 1)
      oc.v_scale = std::ldexp(1.0f, f == 0.5 ? e - 1 : e);
      oc.p_unit = p.mass / (double)oc.v_scale * 0x1p-32;
    }
    CUDA_TRY(cudaMemsetAsync(b->obs, 0, need, stream));
    const BoxDev* rec = d_boxes + b->dev_index;
    const int ntot = (int)(b->nsol + b->nbead);
    const int nb1 = std::max(1, std::min(1024, (ntot + 255) / 256));
    const int nb2 = std::max(1, std::min(1024, (nc + 255) / 256));
    launch_obs_particles(mixed, rec, b->stage_r, b->stage_v, oc, d_partials, nb1, stream);
    std::vector<double> h1(4 * nb1), h2(3 * nb2);
    CUDA_TRY(cudaMemcpyAsync(h1.data(), d_partials, sizeof(double) * 4 * nb1,
                             cudaMemcpyDeviceToHost, stream));
    CUDA_TRY(cudaStreamSynchronize(stream));
    launch_obs_cells(oc, d_partials, nb2, stream);
    CUDA_TRY(cudaMemcpyAsync(h2.data(), d_partials, sizeof(double) * 3 * nb2,
                             cudaMemcpyDeviceToHost, stream));
    CUDA_TRY(cudaStreamSynchronize(stream));
    CUDA_TRY(cudaGetLastError());
    double P[3] = {0, 0, 0}, KE = 0, Tsum = 0, nT = 0, occ = 0;
    for (int i = 0; i < nb1; ++i) {
      for (int k = 0; k < 3; ++k) P[k] += h1[4 * i + k];
      KE += h1[4 * i + 3];
    }
    for (int i = 0; i < nb2; ++i) {
      Tsum += h2[3 * i];
      nT += h2[3 * i + 1];
      occ += h2[3 * i + 2];
    }
    const double M = (double)b->nsol * p.mass + (double)b->nbead * p.solute_mass;
    for (int k = 0; k < 3; ++k) out->P[k] = P[k];
    out->KE = KE;
    const double pp = P[0] * P[0] + P[1] * P[1] + P[2] * P[2];
    out->T_kin = (ntot > 1 && M > 0) ? 2.0 * (KE - pp / (2.0 * M)) / (3.0 * (double)(ntot - 1)) : 0.0;
    out->T_cell_mean = nT > 0 ? Tsum / nT : 0.0;
    out->mass = M;
    out->n = ntot;
    out->occupied_cells = (int64_t)occ;
    out->step = b->d.step;
    return MPCD_OK;
  }
};

struct mpcd_ctx {
  Engine eng;
  Box* box = nullptr;
};

struct mpcd_batch {
  Engine eng;
};

// ===========================================================================
// C ABI
// ===========================================================================
extern "C" {

const char* mpcd_last_error(void) { return g_last_error.c_str(); }

int mpcd_create(const mpcd_params* params, void* stream, mpcd_ctx** out) {
  g_last_error.clear();
  if (!out) return fail(MPCD_EINVAL, "out is NULL");
  *out = nullptr;
  int rc = validate(params, -1);
  if (rc) return rc;
  int ndev = 0;
  cudaError_t e = cudaGetDeviceCount(&ndev);
  if (e != cudaSuccess || ndev < 1)
    return fail(MPCD_ECUDA, std::string("no CUDA device: ") + cudaGetErrorString(e));
  mpcd_ctx* c = new mpcd_ctx();
  rc = c->eng.init(params->precision, stream);
  if (rc) {
    delete c;
    return rc;
  }
  c->box = new Box();
  c->box->p = *params;
  c->eng.slots.push_back(c->box);
  *out = c;
  return MPCD_OK;
}

static int set_state_common(mpcd_ctx* ctx, int64_t n, int64_t nb) {
  Engine& E = ctx->eng;
  int rc = E.complete();
  if (rc) return rc;
  if ((rc = E.pull_records())) return rc;
  Box* b = ctx->box;
  CUDA_TRY(cudaStreamSynchronize(E.stream));
  E.unlink(b);
  b->has_state = false;
  E.free_box_arrays(b);
  return E.setup_box(b, n, nb);
}

int mpcd_set_state(mpcd_ctx* ctx, int64_t n_solvent, const double* pos, const double* vel,
                   int64_t n_solute, const double* solute_pos, const double* solute_vel,
                   uint64_t step) {
  g_last_error.clear();
  if (!ctx) return fail(MPCD_EINVAL, "ctx is NULL");
  if (n_solvent < 0 || n_solute < 0) return fail(MPCD_EINVAL, "negative particle count");
  if (n_solvent > 0 && (!pos || !vel)) return fail(MPCD_EINVAL, "pos/vel is NULL");
  if (n_solute > 0 && (!solute_pos || !solute_vel)) return fail(MPCD_EINVAL, "solute arrays NULL");
  if (n_solute > 0 && ctx->box->p.chain_len < 1)
    return fail(MPCD_EINVAL, "solute given but chain_len is 0");
  int rc = set_state_common(ctx, n_solvent, n_solute);
  if (rc) return rc;
  return ctx->eng.upload_state(ctx->box, pos, vel, solute_pos, solute_vel, step);
}

int mpcd_set_state_device(mpcd_ctx* ctx, int64_t n_solvent, const void* pos, const void* vel,
                          uint64_t step) {
  g_last_error.clear();
  if (!ctx) return fail(MPCD_EINVAL, "ctx is NULL");
  if (n_solvent < 0) return fail(MPCD_EINVAL, "negative particle count");
  if (n_solvent > 0 && (!pos || !vel)) return fail(MPCD_EINVAL, "pos/vel is NULL");
  if (ctx->box->p.chain_len > 0) return fail(MPCD_EINVAL, "use mpcd_set_state for solute runs");
  int rc = set_state_common(ctx, n_solvent, 0);
  if (rc) return rc;
  return ctx->eng.place(ctx->box, pos, vel, nullptr, nullptr, step);
}

int mpcd_set_state_thermal(mpcd_ctx* ctx, int64_t n_solvent, uint64_t init_seed, uint64_t step) {
  g_last_error.clear();
  if (!ctx) return fail(MPCD_EINVAL, "ctx is NULL");
  if (n_solvent < 0) return fail(MPCD_EINVAL, "negative particle count");
  if (ctx->box->p.chain_len > 0) return fail(MPCD_EINVAL, "use mpcd_set_state for solute runs");
  int rc = set_state_common(ctx, n_solvent, 0);
  if (rc) return rc;
  return ctx->eng.thermal_state(ctx->box, init_seed, step);
}

int mpcd_step(mpcd_ctx* ctx, int64_t nsteps) {
  g_last_error.clear();
  if (!ctx) return fail(MPCD_EINVAL, "ctx is NULL");
  if (!ctx->box->has_state) return fail(MPCD_ESTATE, "no state set");
  return ctx->eng.step(nsteps);
}

int mpcd_tune(mpcd_ctx* ctx, int64_t steps_per_candidate, int32_t* blocks_per_sm,
              double* ms_per_step, int64_t* steps_taken, int32_t* pass2_chunk,
              int32_t* cells_per_warp) {
  g_last_error.clear();
  if (!ctx) return fail(MPCD_EINVAL, "ctx is NULL");
  if (!ctx->box->has_state) return fail(MPCD_ESTATE, "no state set");
  return ctx->eng.tune(steps_per_candidate, blocks_per_sm, ms_per_step, steps_taken, pass2_chunk,
                       cells_per_warp);
}

int mpcd_get_state(mpcd_ctx* ctx, double* pos, double* vel, double* solute_pos, double* solute_vel,
                   uint64_t* step) {
  g_last_error.clear();
  if (!ctx) return fail(MPCD_EINVAL, "ctx is NULL");
  if (!ctx->box->has_state) return fail(MPCD_ESTATE, "no state set");
  return ctx->eng.download_state(ctx->box, pos, vel, solute_pos, solute_vel, step);
}

int mpcd_get_state_device(mpcd_ctx* ctx, void* pos, void* vel) {
  g_last_error.clear();
  if (!ctx) return fail(MPCD_EINVAL, "ctx is NULL");
  if (!ctx->box->has_state) return fail(MPCD_ESTATE, "no state set");
  Engine& E = ctx->eng;
  Box* b = ctx->box;
  // straight into the caller's arrays where a kernel may store there, else (another
  // device's memory, a pointer that may be none, arrays that overlap) through the
  // staging arrays and a copy
  const size_t es = elem_size(E.mixed), bytes = (size_t)b->nsol * 3 * es;
  const bool apart = !pos || !vel || (const char*)pos + bytes <= (const char*)vel ||
                     (const char*)vel + bytes <= (const char*)pos;
  void* dp = pos && apart && own_device_memory(pos, bytes, es, E.device) ? pos : nullptr;
  void* dv = vel && apart && own_device_memory(vel, bytes, es, E.device) ? vel : nullptr;
  int rc = E.extract(b, nullptr, dp, dv);
  if (rc) return rc;
  if (bytes == 0 || (dp == pos && dv == vel)) return MPCD_OK;
  if (dp != pos) CUDA_TRY(cudaMemcpyAsync(pos, b->stage_r, bytes, cudaMemcpyDeviceToDevice, E.stream));
  if (dv != vel) CUDA_TRY(cudaMemcpyAsync(vel, b->stage_v, bytes, cudaMemcpyDeviceToDevice, E.stream));
  CUDA_TRY(cudaStreamSynchronize(E.stream));
  CUDA_TRY(cudaGetLastError());
  return MPCD_OK;
}

int mpcd_observables(mpcd_ctx* ctx, mpcd_obs* out) {
  g_last_error.clear();
  if (!ctx) return fail(MPCD_EINVAL, "ctx is NULL");
  if (!ctx->box->has_state) return fail(MPCD_ESTATE, "no state set");
  return ctx->eng.observables(ctx->box, out);
}

int mpcd_profile(mpcd_ctx* ctx, int32_t nbins, double* out) {
  g_last_error.clear();
  if (!ctx || !out) return fail(MPCD_EINVAL, "NULL argument");
  if (nbins < 1 || nbins > (1 << 20)) return fail(MPCD_EINVAL, "nbins out of range");
  if (!ctx->box->has_state) return fail(MPCD_ESTATE, "no state set");
  Engine& E = ctx->eng;
  Box* b = ctx->box;
  int rc = E.extract(b, nullptr);
  if (rc) return rc;
  double* dsum = nullptr;
  unsigned long long* dcnt = nullptr;
  CUDA_TRY(cudaMallocAsync((void**)&dsum, sizeof(double) * nbins, E.stream));
  CUDA_TRY(cudaMallocAsync((void**)&dcnt, sizeof(unsigned long long) * nbins, E.stream));
  CUDA_TRY(cudaMemsetAsync(dsum, 0, sizeof(double) * nbins, E.stream));
  CUDA_TRY(cudaMemsetAsync(dcnt, 0, sizeof(unsigned long long) * nbins, E.stream));
  launch_profile(E.mixed, b->stage_r, b->stage_v, (int)b->nsol, nbins, dsum, dcnt,
                 (double)b->p.n[2], E.stream);
  std::vector<double> hs(nbins);
  std::vector<unsigned long long> hc(nbins);
  CUDA_TRY(cudaMemcpyAsync(hs.data(), dsum, sizeof(double) * nbins, cudaMemcpyDeviceToHost, E.stream));
  CUDA_TRY(cudaMemcpyAsync(hc.data(), dcnt, sizeof(unsigned long long) * nbins,
                           cudaMemcpyDeviceToHost, E.stream));
  CUDA_TRY(cudaFreeAsync(dsum, E.stream));
  CUDA_TRY(cudaFreeAsync(dcnt, E.stream));
  CUDA_TRY(cudaStreamSynchronize(E.stream));
  CUDA_TRY(cudaGetLastError());
  for (int i = 0; i < nbins; ++i) out[i] = hc[i] ? hs[i] / (double)hc[i] : 0.0;
  return MPCD_OK;
}

int mpcd_last_cells(mpcd_ctx* ctx, int32_t* cell_out, int32_t* count_out) {
  g_last_error.clear();
  if (!ctx) return fail(MPCD_EINVAL, "ctx is NULL");
  if (!ctx->box->has_state) return fail(MPCD_ESTATE, "no state set");
  Engine& E = ctx->eng;
  Box* b = ctx->box;
  const int64_t ntot = b->nsol + b->nbead;
  const int64_t C = cells_of(b->p);
  int32_t *dc = nullptr, *dk = nullptr;
  if (cell_out && ntot > 0) CUDA_TRY(cudaMallocAsync((void**)&dc, sizeof(int32_t) * ntot, E.stream));
  if (count_out) CUDA_TRY(cudaMallocAsync((void**)&dk, sizeof(int32_t) * C, E.stream));
  // (small boxes: one wait less instead)
  int rc = E.extract(b, dc, nullptr, nullptr, 3 * (size_t)b->nsol > XFER_ELEMS);
  if (rc) return rc;
  launch_cell_counts(E.d_boxes + b->dev_index, (int)C, (int)b->nbead, dc, dk, E.stream);
  if (dc) CUDA_TRY(cudaMemcpyAsync(cell_out, dc, sizeof(int32_t) * ntot, cudaMemcpyDeviceToHost, E.stream));
  if (dk) CUDA_TRY(cudaMemcpyAsync(count_out, dk, sizeof(int32_t) * C, cudaMemcpyDeviceToHost, E.stream));
  if (dc) CUDA_TRY(cudaFreeAsync(dc, E.stream));
  if (dk) CUDA_TRY(cudaFreeAsync(dk, E.stream));
  CUDA_TRY(cudaStreamSynchronize(E.stream));
  CUDA_TRY(cudaGetLastError());
  return MPCD_OK;
}

int64_t mpcd_num_cells(const mpcd_ctx* ctx) { return ctx ? cells_of(ctx->box->p) : -1; }

static const char* kPhaseNames[] = {"fused_step", "after_pass", "solute"};

int mpcd_phase_times(mpcd_ctx* ctx, int64_t nsteps, double* ms, int32_t nmax, int32_t* nphases) {
  g_last_error.clear();
  if (!ctx || !ms || nsteps < 0) return fail(MPCD_EINVAL, "bad argument");
  if (!ctx->box->has_state) return fail(MPCD_ESTATE, "no state set");
  if (nmax < Engine::kPhases) return fail(MPCD_EINVAL, "nmax too small");
  const int rc = ctx->eng.timed_steps(nsteps, ms);
  if (rc < 0) return rc;
  if (nphases) *nphases = Engine::kPhases;
  return MPCD_OK;
}

const char* mpcd_phase_name(int32_t i) {
  return (i >= 0 && i < Engine::kPhases) ? kPhaseNames[i] : "";
}

void mpcd_destroy(mpcd_ctx* ctx) { delete ctx; }

// ----------------------------- batches -------------------------------------
int mpcd_batch_create(int32_t precision, void* stream, int64_t max_bytes, mpcd_batch** out) {
  g_last_error.clear();
  if (!out) return fail(MPCD_EINVAL, "out is NULL");
  *out = nullptr;
  if (precision != MPCD_FP64 && precision != MPCD_MIXED) return fail(MPCD_EINVAL, "bad precision");
  if (max_bytes < 0) return fail(MPCD_EINVAL, "max_bytes < 0");
  int ndev = 0;
  cudaError_t e = cudaGetDeviceCount(&ndev);
  if (e != cudaSuccess || ndev < 1)
    return fail(MPCD_ECUDA, std::string("no CUDA device: ") + cudaGetErrorString(e));
  mpcd_batch* b = new mpcd_batch();
  int rc = b->eng.init(precision, stream);
  if (rc) {
    delete b;
    return rc;
  }
  b->eng.max_bytes = max_bytes;
  *out = b;
  return MPCD_OK;
}

int64_t mpcd_box_footprint(const mpcd_params* params, int64_t n_solvent) {
  if (!params || n_solvent < 0) return -1;
  return (int64_t)footprint_bytes(*params, n_solvent, 0);
}

int mpcd_batch_add(mpcd_batch* bt, const mpcd_params* params, int64_t n_solvent, const double* pos,
                   const double* vel, uint64_t step, int32_t* slot) {
  g_last_error.clear();
  if (!bt || !slot) return fail(MPCD_EINVAL, "NULL argument");
  Engine& E = bt->eng;
  int rc = validate(params, E.mixed ? MPCD_MIXED : MPCD_FP64);
  if (rc) return rc;
  if (params->chain_len > 0) return fail(MPCD_EINVAL, "no solute in batches");
  if (n_solvent > 0 && (!pos || !vel)) return fail(MPCD_EINVAL, "pos/vel is NULL");
  if ((rc = E.complete())) return rc;
  if ((rc = E.pull_records())) return rc;
  Box* b = new Box();
  b->p = *params;
  if ((rc = E.setup_box(b, n_solvent, 0))) {
    E.free_box_arrays(b);
    delete b;
    return rc;
  }
  if ((rc = E.upload_state(b, pos, vel, nullptr, nullptr, step))) {
    E.release_box(b);
    return rc;
  }
  int s = -1;
  for (size_t i = 0; i < E.slots.size(); ++i)
    if (!E.slots[i]) {
      s = (int)i;
      break;
    }
  if (s < 0) {
    s = (int)E.slots.size();
    E.slots.push_back(nullptr);
  }
  E.slots[s] = b;
  E.drop_graphs();
  E.tables_ok = false;
  *slot = s;
  return MPCD_OK;
}

int mpcd_batch_add_thermal(mpcd_batch* bt, const mpcd_params* params, int64_t n_solvent,
                           uint64_t init_seed, uint64_t step, int32_t* slot) {
  g_last_error.clear();
  if (!bt || !slot) return fail(MPCD_EINVAL, "NULL argument");
  Engine& E = bt->eng;
  int rc = validate(params, E.mixed ? MPCD_MIXED : MPCD_FP64);
  if (rc) return rc;
  if (params->chain_len > 0) return fail(MPCD_EINVAL, "no solute in batches");
  if (n_solvent < 0) return fail(MPCD_EINVAL, "negative particle count");
  if ((rc = E.complete())) return rc;
  if ((rc = E.pull_records())) return rc;
  Box* b = new Box();
  b->p = *params;
  if ((rc = E.setup_box(b, n_solvent, 0))) {
    E.free_box_arrays(b);
    delete b;
    return rc;
  }
  if ((rc = E.thermal_state(b, init_seed, step))) {
    E.release_box(b);
    return rc;
  }
  int s = -1;
  for (size_t i = 0; i < E.slots.size(); ++i)
    if (!E.slots[i]) {
      s = (int)i;
      break;
    }
  if (s < 0) {
    s = (int)E.slots.size();
    E.slots.push_back(nullptr);
  }
  E.slots[s] = b;
  E.drop_graphs();
  E.tables_ok = false;
  *slot = s;
  return MPCD_OK;
}

static Box* batch_box(mpcd_batch* bt, int32_t slot) {
  if (!bt || slot < 0 || slot >= (int32_t)bt->eng.slots.size()) return nullptr;
  return bt->eng.slots[slot];
}

int mpcd_batch_step(mpcd_batch* bt, int64_t nsteps) {
  g_last_error.clear();
  if (!bt) return fail(MPCD_EINVAL, "batch is NULL");
  return bt->eng.step(nsteps);
}

int mpcd_batch_tune(mpcd_batch* bt, int64_t steps_per_candidate, int32_t* blocks_per_sm,
                    double* ms_per_step, int64_t* steps_taken, int32_t* pass2_chunk,
                    int32_t* cells_per_warp) {
  g_last_error.clear();
  if (!bt) return fail(MPCD_EINVAL, "batch is NULL");
  return bt->eng.tune(steps_per_candidate, blocks_per_sm, ms_per_step, steps_taken, pass2_chunk,
                      cells_per_warp);
}

int mpcd_batch_get_state(mpcd_batch* bt, int32_t slot, double* pos, double* vel, uint64_t* step) {
  g_last_error.clear();
  Box* b = batch_box(bt, slot);
  if (!b) return fail(MPCD_EINVAL, "bad slot");
  return bt->eng.download_state(b, pos, vel, nullptr, nullptr, step);
}

int mpcd_batch_observables(mpcd_batch* bt, int32_t slot, mpcd_obs* out) {
  g_last_error.clear();
  Box* b = batch_box(bt, slot);
  if (!b) return fail(MPCD_EINVAL, "bad slot");
  return bt->eng.observables(b, out);
}

int mpcd_batch_remove(mpcd_batch* bt, int32_t slot) {
  g_last_error.clear();
  Box* b = batch_box(bt, slot);
  if (!b) return fail(MPCD_EINVAL, "bad slot");
  Engine& E = bt->eng;
  int rc = E.complete();
  if (rc) return rc;
  if ((rc = E.pull_records())) return rc;
  CUDA_TRY(cudaStreamSynchronize(E.stream));
  E.slots[slot] = nullptr;
  E.unlink(b);
  E.release_box(b);
  return MPCD_OK;
}

int mpcd_batch_sync(mpcd_batch* bt) {
  g_last_error.clear();
  if (!bt) return fail(MPCD_EINVAL, "batch is NULL");
  CUDA_TRY(cudaStreamSynchronize(bt->eng.stream));
  return bt->eng.check_err();
}

int mpcd_batch_info(const mpcd_batch* bt, int32_t* n_boxes, int64_t* bytes_used) {
  if (!bt) return fail(MPCD_EINVAL, "batch is NULL");
  int n = 0;
  for (Box* b : bt->eng.slots)
    if (b) ++n;
  if (n_boxes) *n_boxes = n;
  if (bytes_used) *bytes_used = (int64_t)bt->eng.used_bytes;
  return MPCD_OK;
}

void mpcd_batch_destroy(mpcd_batch* bt) { delete bt; }

}  // extern "C"

// ===========================================================================
// Allocation-free variant of mpcd_profile.
//
// Some callers cannot allocate device memory at the moment they want a
// profile: services that run inside a fixed, pre-reserved device-memory
// budget where every allocation is accounted for up front, and job servers
// that keep nearly all of the GPU's memory filled with resident boxes, where
// an allocation at query time could fail.  This entry point uses only memory
// that already exists: the box's own arrays and a static per-bin scratch
// array below.  It synchronises the box's stream to read the result back.
// ===========================================================================
namespace {

constexpr int kProfileNoAllocMaxBins = 4096;

// Per-bin scratch shared by every call on a device and held by every GPU that
// loads the library until the process exits: sums of v_x in
// [0, kProfileNoAllocMaxBins), member counts (as doubles) after that, and the
// finished means written back over the sums.
static __device__ __align__(256) double g_profile_scratch[2 * kProfileNoAllocMaxBins];

// Device address of g_profile_scratch per device, looked up once per device.
std::mutex g_profile_scratch_mu;
void* g_profile_scratch_addr[64] = {};

__global__ void k_profile_noalloc_clear(int nbins) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 2 * nbins; i += gridDim.x * blockDim.x) {
    const int j = i < nbins ? i : kProfileNoAllocMaxBins + (i - nbins);
    g_profile_scratch[j] = 0.0;
  }
}

template <bool MIXED>
__global__ void k_profile_noalloc_accumulate(const void* __restrict__ pos_,
                                             const void* __restrict__ vel_, int n, int nbins,
                                             double H, double* __restrict__ scratch) {
  using T = typename std::conditional<MIXED, float, double>::type;
  const T* r = (const T*)pos_;
  const T* v = (const T*)vel_;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    long long b = (long long)floor((double)r[3 * i + 2] / H * (double)nbins);
    if (b < 0) b = 0;
    if (b >= nbins) b = nbins - 1;
    atomicAdd(&scratch[b], (double)v[3 * i]);
    atomicAdd(&scratch[kProfileNoAllocMaxBins + b], 1.0);
  }
}

__global__ void k_profile_noalloc_finish(int nbins, double* __restrict__ scratch) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nbins; b += gridDim.x * blockDim.x) {
    const double c = scratch[kProfileNoAllocMaxBins + b];
    scratch[b] = c > 0.0 ? scratch[b] / c : 0.0;
  }
}

}  // namespace

extern "C" int mpcd_profile_noalloc(mpcd_ctx* ctx, int32_t nbins, double* out) {
  g_last_error.clear();
  if (!ctx || !out) return fail(MPCD_EINVAL, "NULL argument");
  if (nbins < 1 || nbins > kProfileNoAllocMaxBins)
    return fail(MPCD_EINVAL, "nbins must be in [1, 4096] for the allocation-free profile");
  Box* b = ctx->box;
  Engine& E = ctx->eng;
  if (!b->has_state) return fail(MPCD_ESTATE, "no state set");
  if (!E.tables_ok || b->dev_index < 0)
    return fail(MPCD_ESTATE,
                "the box is not on the device yet: call mpcd_step (0 steps is enough) first");
  int dev = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(MPCD_ECUDA, "device index out of range");
  void* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_profile_scratch_mu);
    if (!g_profile_scratch_addr[dev]) {
      void* p = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&p, g_profile_scratch);
      if (e != cudaSuccess || !p)
        return fail(MPCD_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      g_profile_scratch_addr[dev] = p;
    }
    scratch = g_profile_scratch_addr[dev];
  }
  // A pending collision is completed with plain kernel launches, and the state
  // is written in input order into the box's existing staging arrays: no
  // allocation on either path.
  if (E.pending) {
    CUDA_TRY(E.enqueue_pass(MODE_C));
    E.pending = false;
  }
  const int n = (int)b->nsol;
  launch_extract(E.mixed, E.d_boxes + b->dev_index, b->stage_r, b->stage_v, nullptr,
                 (int)cells_of(b->p), n, b->d.xcnt, E.stream);
  int grid = (n + 255) / 256;
  if (grid < 1) grid = 1;
  if (grid > 4096) grid = 4096;
  k_profile_noalloc_clear<<<(2 * nbins + 255) / 256, 256, 0, E.stream>>>(nbins);
  if (E.mixed)
    k_profile_noalloc_accumulate<true><<<grid, 256, 0, E.stream>>>(
        b->stage_r, b->stage_v, n, nbins, (double)b->p.n[2], (double*)scratch);
  else
    k_profile_noalloc_accumulate<false><<<grid, 256, 0, E.stream>>>(
        b->stage_r, b->stage_v, n, nbins, (double)b->p.n[2], (double*)scratch);
  k_profile_noalloc_finish<<<(nbins + 255) / 256, 256, 0, E.stream>>>(nbins, (double*)scratch);
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaMemcpyAsync(out, scratch, sizeof(double) * nbins, cudaMemcpyDeviceToHost, E.stream));
  CUDA_TRY(cudaStreamSynchronize(E.stream));
  return E.check_err();
}
