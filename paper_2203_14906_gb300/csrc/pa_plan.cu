// pa_plan.cu -- host side of the C ABI: descriptor validation, tile
// configuration, the plan-time delay / apodisation table kernel (Section 5:
// delays are computed once and kept resident in device memory), per-tile RF
// windows, post-filter masks, and the launch sequence of pa_beamform.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include <cudaTypedefs.h>

#include "pa_internal.cuh"
#include "pa_schedule.h"

using namespace pa;

// ------------------------------------------------------------------ errors
namespace {
thread_local std::string g_err;

pa_status fail(pa_status s, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_err = buf;
  return s;
}

#define PA_CUDA(call)                                                         \
  do {                                                                        \
    cudaError_t e_ = (call);                                                  \
    if (e_ != cudaSuccess)                                                    \
      return fail(PA_ECUDA, "%s failed: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

int popcount3(uint32_t m) { return (int)((m & 1u) + ((m >> 1) & 1u) + ((m >> 2) & 1u)); }

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
    else prev = -1;
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};
}  // namespace

// ------------------------------------------------------------------- plan
// Buffer sets (and streams) of the host-buffer path.
constexpr int kHostSets = 3;

// Pinned words that a timed-out wait sets, one per plan that takes the host
// path.  The first small cudaHostAlloc of a process costs about 140 us and the
// next 1.5 us, but the last cudaFreeHost gives the memory back, so a plan with a
// word of its own paid 125 us in its first call and as much when it was destroyed.
// The words come from pages of 1024 that stay with the library (4 KiB per 1024
// plans alive at once); a page belongs to the context it was made in, as a reset
// device takes it along.
class HostWords {
 public:
  int* take() {
    std::lock_guard<std::mutex> lk(mu_);
    const unsigned long long ctx = context_id();
    for (Page& pg : pages_)
      if (pg.ctx == ctx && !pg.free.empty()) {
        int* w = pg.free.back();
        pg.free.pop_back();
        return w;
      }
    int* base = nullptr;
    if (cudaHostAlloc((void**)&base, kWords * sizeof(int),
                      cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess)
      return nullptr;
    pages_.push_back({ctx, base, {}});
    for (int i = kWords - 1; i > 0; --i) pages_.back().free.push_back(base + i);
    return base;
  }
  void give(int* w) {
    std::lock_guard<std::mutex> lk(mu_);
    for (Page& pg : pages_)
      if (w >= pg.base && w < pg.base + kWords) {
        pg.free.push_back(w);
        return;
      }
  }

 private:
  static constexpr int kWords = 1024;
  struct Page {
    unsigned long long ctx;
    int* base;
    std::vector<int*> free;
  };
  static unsigned long long context_id() {
    static PFN_cuCtxGetId_v12000 fn = [] {
      void* f = nullptr;
      cudaDriverEntryPointQueryResult q;
      if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) !=
              cudaSuccess ||
          q != cudaDriverEntryPointSuccess)
        f = nullptr;
      return reinterpret_cast<PFN_cuCtxGetId_v12000>(f);
    }();
    unsigned long long id = 0;
    if (fn) fn(nullptr, &id);
    return id;
  }
  std::mutex mu_;
  std::vector<Page> pages_;
};
HostWords g_host_words;

// One form of the fused kernel and the shared-memory geometry that goes with
// it: form 0 runs one frame per work item (pa_bf_kernel.cuh), form 1 two
// frames from prepared slots (pa_bf_pipe.cuh), forms 2 and 3 one and two of a
// thread's four pixels, for small launches (pa_bf_fine.cuh).
struct FusedForm {
  int nf = 0;             // frames per work item (0: the plan has no such form)
  const void* func = nullptr;
  int threads = 0;
  int nc = 32;            // channel steps per staged chunk (multiple of kC)
  int stages = 1;         // chunks in shared memory at once (forms 1-3)
  int rp = 0;             // raw-buffer row pitch in samples (128-byte aligned rows)
  int pairs_off = 0;      // shared-memory offset of the interpolation slots
  size_t smem = 0;
  int blocks_per_sm = 0;
  int tmem_cols = 0;      // TMEM columns per block (compensated sums)
  int splits = 1;         // work items per tile (forms 2, 3)
  int2* vchunks = nullptr;  // chunk range of a work item (forms 2, 3: of a tile),
  size_t chunk_at = 0;      // from this entry of the plan's chunk ranges on
  // prepared slots: a row of zeros, then one row of slot_pitch slots per
  // (frames of an item, channel), for max_frames frames a round (forms 2 and
  // 3: at most that many frames a launch)
  int slots_form = 0;     // this form's index if it reads slots
  int slot_bytes = 0;
  unsigned char* slots = nullptr;
  int max_frames = 0;
};

struct pa_plan_s {
  pa_plan_desc d{};
  int device = 0, num_sms = 0;
  int K = 1;
  bool apod = false, comp = false;
  bool full = false;  // per-pixel delay table (PA_TABLE_FULL) instead of the lattice
  // tiling
  int m = 1, R = 1, slots = 1, warps = 1, ngroups = 1, threads = 32;
  int tile_x = 0, tile_z = 32, nxt = 0, nzt = 0, n_tiles = 0, nx_pad = 0, nz_pad = 0;
  int u0 = 0, u1 = 0, nv = 0, dmin = 0, ndrows = 0, tgroups = 0, window = 0;
  size_t full_entries = 0;  // entries of the full table (n_tiles * (steps + 3) * 32 * slots * kC)
  FusedForm form[4];
  unsigned char* arena = nullptr;     // the plan's device memory but for the slots (plan_arena)
  unsigned char* slot_mem = nullptr;  // prepared slots of forms 1-3 (optional)
  size_t slot_mem_bytes = 0;
  bool slots_joined = false;          // slot_mem is the end of the arena's allocation
  unsigned char* spare = nullptr;     // what that allocation's last page leaves
  size_t spare_bytes = 0;
  size_t slot_limit = kNoSlotLimit;   // most bytes of slots the plan may take
  long long slot_pitch = 0;
  int used_lo = 0, used_hi = 0;  // samples [used_lo, used_hi) lie in some window
  int slot_margin = 0, slot_mode = 0;
  bool use_tma = false;
  int lo_align = 4;   // window starts are multiples of this many samples
  int expect_extra = 0;   // > 0 only under PA_INJECT_TMA_SHORTFALL (tests the bounded wait)
  long long timeouts_seen = 0;  // timed-out waits already reported by pa_beamform_host
  int* host_flag = nullptr;  // pinned word a timed-out wait sets (host path; HostWords)
  int wr = 0;         // raw samples per channel delivered by one TMA box
  int item_frames = 0;  // PA_ITEM_FRAMES: 1-4 picks the form (measurements, tests)
  double steps_per_pixel = 0;  // channel steps evaluated per pixel, mean
  bool pairs_pay = false;  // resident warps and slot reuse of the two-frame form suffice
  // post
  int M = 1, log2M = 0, post_wpb = 1, n_out = 0, n_tw = 0;
  int2 band[3] = {};  // bins each output keeps (PostParams)
  int band_rows = 0;
  int out_id[3] = {-1, -1, -1};  // output slot (0..n_out) of DAS, DMAS, HO
  uint32_t warnings = 0;
  float dyn_range = 60.f;
  // device memory
  int2* table = nullptr;     // lattice table
  int2* ftab = nullptr;      // full table (see k_table_full)
  float* wtab = nullptr;
  int* lo = nullptr;
  int2* urange = nullptr;
  int2* chunks = nullptr;  // chunk ranges of all forms
  unsigned long long* active = nullptr;  // count of active pairs (plan build)
  int4* items = nullptr;   // work-item table (tile, group, tx, tz)
  int2* slot_rg = nullptr; // warp slot -> (column residue, column group)
  float2* tw = nullptr;
  float* mask = nullptr;
  // [err, counter, maxslots..., timeouts]; [0] serves pa_beamform, all three
  // the buffer sets of pa_beamform_host
  int* scratch[kHostSets] = {nullptr, nullptr, nullptr};
  size_t scratch_ints = 0;
  // host-buffer path
  void* h_rf = nullptr;       // staging buffers, one allocation or the arena's spare
  float* h_out = nullptr;
  size_t h_rf_bytes = 0, h_out_bytes = 0;
  cudaStream_t hs[kHostSets] = {nullptr, nullptr, nullptr};
  cudaEvent_t h_ev = nullptr;
  cudaEvent_t h_done[kHostSets] = {nullptr, nullptr, nullptr};
  // chunk schedules of the host path, per (frames, stages): every candidate
  // timed once, the three fastest once more, then the fastest kept
  struct HostTune {
    int nf = 0;
    uint32_t stages = 0;
    std::vector<std::vector<int32_t>> cand;
    std::vector<double> best_ms;  // < 0: not measured yet
    std::vector<int> order;       // candidates in the order they are timed
    size_t pos = 0;
    int attempts = 0;             // uncounted (cold) calls of order[pos]
    bool second_round = false;
    int chosen = -1;              // index into cand once tuned
    std::vector<int32_t> fixed;   // set by pa_plan_set_host_schedule
    const std::vector<int32_t>& current() const {
      return !fixed.empty() ? fixed : cand[chosen >= 0 ? chosen : order[pos]];
    }
  };
  std::vector<HostTune> tunes;
  long long graph_builds = 0;  // executable graphs instantiated so far
  // whole host-path calls as graphs (pinned host buffers): every chunk's
  // upload, launch sequence and download, per (frames, stages, schedule);
  // they name the staging buffers, so growing those drops them
  struct HostGraph {
    int nf = 0;
    uint32_t stages = 0;
    std::vector<int32_t> sched;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    std::vector<cudaGraphNode_t> up, down;  // per chunk
    std::vector<void*> up_dev, down_dev;
    std::vector<size_t> up_off, down_off, up_bytes, down_bytes;
    const void* rf_host = nullptr;
    float* out_host = nullptr;
  };
  std::vector<HostGraph> host_graphs;
  // CUDA graphs of the launch sequence, one per (frames, stages)
  struct GraphEntry {
    int nf = 0;
    uint32_t stages = 0;
    cudaGraph_t graph = nullptr;  // kept alive: exec-node updates name its nodes
    cudaGraphExec_t exec = nullptr;
    uint32_t prof = 0;  // kernel kinds timed (bit per kind)
    std::vector<cudaGraphNode_t> kernels;
    // timing graphs (built while pa_plan_profile is on): an event-record
    // node before and after each timed kernel, given fresh events every launch
    std::vector<cudaGraphNode_t> events;
  };
  std::vector<GraphEntry> graphs;
  bool use_graph = true;
  int lane_rows_log2 = 5;  // depth rows per lane group of the fused kernel (log2)
  // kernel timing (pa_plan_profile): bit k set = kernel kind k is timed
  uint32_t prof = 0;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev_free;
  std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> ev_used;
  // facts
  int64_t active_pairs = 0, executed_pairs = 0;
  size_t device_bytes = 0;
  size_t elt = 4;
};

namespace {

// ---------------------------------------------------------- plan kernels
// Layout of the full table, in the order the fused kernel reads it: per
// tile, channel step u' = u - u0 (steps + 3 of them: the last three are
// padding, so the kernel loads two steps ahead with no bound check), half h
// = c / 2 of a thread's kC = 4 pixels, thread t = (rg * slots + sl) * LR + zl
// of the tile (row group rg of the tile's 32 rows, warp slot sl, row zl
// within the group) and pixel c % 2:
//   (((tile * (steps + 3) + u') * 2 + h) * (32 slots) + t) * 2 + c % 2
// with LR depth rows per lane group and RG = 32 / LR.  A thread loads a step
// as two 16-byte entries pairs; the 32 lanes of a warp read each of them as
// 512 contiguous bytes.
struct FullGeom {
  int nxt, n_tiles, tile_x, tile_z, m, slots, steps, lr_log2, nx, nz, n_elem, u0, nv;
};

static_assert(kC == 4, "the full table splits a thread's step into two entry pairs");

__host__ __device__ __forceinline__ size_t full_index(const FullGeom& f, int tile, int up, int c,
                                                     int sl, int zt) {
  const int lr = 1 << f.lr_log2;
  const int rg = zt >> f.lr_log2, zl = zt & (lr - 1);
  const size_t threads = (size_t)32 * f.slots;
  const size_t t = ((size_t)rg * f.slots + sl) * lr + zl;
  return ((((size_t)tile * (f.steps + 3) + up) * 2 + (c >> 1)) * threads + t) * 2 + (c & 1);
}

// Entries of one tile in the full table.
__host__ __device__ __forceinline__ size_t full_per_tile(const FullGeom& f) {
  return (size_t)(f.steps + 3) * 32 * f.slots * kC;
}

// (step, pixel, slot, row in the tile) of entry e of a tile.
__device__ __forceinline__ void full_decode(const FullGeom& f, size_t e, int* up, int* c, int* sl,
                                            int* zt) {
  const int lr = 1 << f.lr_log2;
  const size_t threads = (size_t)32 * f.slots;
  const int c_lo = (int)(e & 1);
  size_t q = e >> 1;
  const size_t t = q % threads;
  q /= threads;
  *c = (int)(q & 1) * 2 + c_lo;
  *up = (int)(q >> 1);
  const int zl = (int)(t % lr);
  const size_t t2 = t / lr;
  *sl = (int)(t2 % f.slots);
  const int rg = (int)(t2 / f.slots);
  *zt = rg * lr + zl;
}

// Pixel column of pixel c of warp slot sl in tile column tx.
__host__ __device__ __forceinline__ int full_column(const FullGeom& f, int tx, int sl, int c) {
  return tx * f.tile_x + (sl / f.m) * f.m * kC + (sl % f.m) + f.m * c;
}

struct TableGeom {
  int ndrows, nzp, dmin, ns, nearest, m, groups;
  double x_const;  // x0 + (N-1)/2 pitch: dx of lattice offset d is x_const + (d + 1/2) dx
  double dx, z0, dz, fs, c, t0, fnum;
  // full table: element i = v + u0 of N at x_i = (i - (N-1)/2) pitch
  double x0, pitch;
  int n_elem, u0, nv;
};

// The one-way time of flight in samples from a pixel at lateral offset dxv
// from the element and depth zp, tau = fs (r / c - t0), as the integer sample
// n0 = floor(tau) and the fraction a = tau - n0 (nearest-sample delays,
// Eq. 1: n0 = round(tau), a = 0).
__device__ void delay_sample(const TableGeom& g, double dxv, double zp, int* n0_out,
                             double* a_out) {
  const double tau = g.fs * (sqrt(dxv * dxv + zp * zp) / g.c - g.t0);
  double fl = g.nearest ? floor(tau + 0.5) : floor(tau);
  double a = g.nearest ? 0.0 : tau - fl;
  const double lim = 1048576.0;
  if (fl < -lim) { fl = -lim; a = 0.0; }
  if (fl > lim) { fl = lim; a = 0.0; }
  int n0 = (int)fl;
  // A delay whose taps leave the record contributes nothing (s = 0).  Staged
  // samples outside [0, Ns) are zero, so pointing such delays at a slot whose
  // two taps both lie outside the record gives s = 0 with no test per pair:
  // n0 = -1 (taps -1, 0) moves to -2, n0 = Ns-1 (taps Ns-1, Ns) moves to Ns.
  // (With a = 0 the nearest sample reads only the first tap: slots n0 = -1 and
  // n0 = Ns-1 already give 0 and r[Ns-1], so no remapping is needed.)
  if (!g.nearest && n0 == -1) n0 = -2;
  if (!g.nearest && n0 == g.ns - 1) n0 = g.ns;
  *n0_out = n0;
  *a_out = a;
}

// Hann dynamic-aperture weight of an element at lateral offset dxv from a
// pixel at depth zp (0 outside the aperture |dxv| <= zp / (2F)).
__device__ float apod_weight(const TableGeom& g, double dxv, double zp) {
  float w = 0.f;
  const double half = zp / (2.0 * g.fnum);
  if (half > 0.0 && fabs(dxv) <= half) {
    const double cw = cos(3.14159265358979323846 * dxv / (2.0 * half));
    w = (float)(cw * cw);
  }
  return w;
}

// Lateral offset x_j - x_i of pixel column j and virtual channel v (element
// i = v + u0), both positions computed as the grid and the array define them.
__device__ double full_dx(const TableGeom& g, int j, int v) {
  const double xp = g.x0 + ((double)j + 0.5) * g.dx;
  const double xi = ((double)(v + g.u0) - 0.5 * (double)(g.n_elem - 1)) * g.pitch;
  return xp - xi;
}

__device__ double pixel_z(const TableGeom& g, int z) { return g.z0 + ((double)z + 0.5) * g.dz; }

// Lattice table: every lattice offset d = j - m i and depth row, entry
// {n0 * 8 (the byte stride of an interpolation slot), FP32 bits of a}.
__global__ void k_table(TableGeom g, int2* table, float* wtab) {
  const int z = blockIdx.y * blockDim.x + threadIdx.x;
  const int row = blockIdx.x;  // (x: a wide aperture has more than 65535 rows)
  if (z >= g.nzp || row >= g.ndrows) return;
  const double dxv = g.x_const + ((double)(g.dmin + row) + 0.5) * g.dx;
  const double zp = pixel_z(g, z);
  int n0;
  double a;
  delay_sample(g, dxv, zp, &n0, &a);
  const size_t ti = table_index(row, z, g.m, g.groups, g.nzp);
  table[ti] = make_int2(n0 * 8, __float_as_int((float)a));
  if (wtab) wtab[ti] = apod_weight(g, dxv, zp);
}

// Full table: the entry of every (pixel, channel step) pair the fused kernel
// evaluates (pixel c of slot sl pairs with channel u + c at step u), in the
// layout of full_index: {(n0 - lo) * 8, FP32 bits of a}, the sample relative
// to the RF window its tile stages for that channel (lo, from
// k_windows_full) as a byte offset into the window's interpolation slots.
// The padding steps hold zeros.
__global__ void k_table_full(TableGeom g, FullGeom f, const int* lo, int2* table, float* wtab) {
  const int tile = blockIdx.y;
  const size_t per_tile = full_per_tile(f);
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= per_tile) return;
  int up, c, sl, zt;
  full_decode(f, e, &up, &c, &sl, &zt);
  const size_t ti = (size_t)tile * per_tile + e;
  if (up >= f.steps) {
    table[ti] = make_int2(0, 0);
    if (wtab) wtab[ti] = 0.f;
    return;
  }
  const int tx = tile % f.nxt, tz = tile / f.nxt;
  const int j = full_column(f, tx, sl, c);
  const int v = up + c;
  const double dxv = full_dx(g, j, v);
  const double zp = pixel_z(g, tz * f.tile_z + zt);
  int n0;
  double a;
  delay_sample(g, dxv, zp, &n0, &a);
  table[ti] = make_int2((n0 - lo[(size_t)tile * g.nv + v]) * 8, __float_as_int((float)a));
  if (wtab) wtab[ti] = apod_weight(g, dxv, zp);
}

// Pairs with a non-zero apodisation weight in the full table (real pixels
// and elements only).
__global__ void k_count_active_full(FullGeom f, const float* wtab, unsigned long long* count) {
  const int tile = blockIdx.y;
  const size_t per_tile = full_per_tile(f);
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long cnt = 0;
  if (e < per_tile) {
    int up, c, sl, zt;
    full_decode(f, e, &up, &c, &sl, &zt);
    const int j = full_column(f, tile % f.nxt, sl, c);
    const int z = (tile / f.nxt) * f.tile_z + zt;
    const int i = up + c + f.u0;
    if (up < f.steps && j < f.nx && z < f.nz && i >= 0 && i < f.n_elem &&
        wtab[(size_t)tile * per_tile + e] > 0.f)
      cnt = 1;
  }
  for (int s = 16; s >= 1; s >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, s);
  if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(count, cnt);
}

constexpr int kLoBias = 1 << 22;  // window starts + kLoBias > 0 (delays are clamped to +-2^20)

struct TileGeom {
  int nxt, nzt, tile_x, tile_z, m, dmin, nzp, nv, u0, ndrows, groups;
  int full;  // 1: full table (laid out as full_index says)
};

// Lattice-table row of pixel column j and virtual channel v (offset
// d = j - m i, i = v + u0).
__device__ __forceinline__ int tile_row(const TileGeom& g, int j, int v) {
  return j - g.m * (v + g.u0) - g.dmin;
}

// Largest window start and (as the largest negative) the smallest one.
__device__ __forceinline__ void record_starts(int* lomax, int lo) {
  atomicMax(lomax, lo + kLoBias);
  atomicMax(lomax + 1, kLoBias - lo);
}

// First staged sample (rounded down to a multiple of 4) and window width of
// every (tile, virtual channel).  The delay grows with depth for z > 0, so the
// minimum over the tile is on its first row and the maximum on its last.
__global__ void k_windows(TileGeom g, int lo_align, const int2* table, int* lo, int* wmax,
                          int* lomax, int* err) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  const int tile = blockIdx.y;
  if (v >= g.nv) return;
  const int tx = tile % g.nxt, tz = tile / g.nxt;
  const int zf = tz * g.tile_z, zl = zf + g.tile_z - 1;
  int mn = 0x7fffffff, mx = -0x7fffffff;
  for (int jj = 0; jj < g.tile_x; ++jj) {
    const int row = tile_row(g, tx * g.tile_x + jj, v);
    if (row < 0 || row >= g.ndrows) {
      atomicOr(err, 4);
      continue;
    }
    mn = min(mn, table[table_index(row, zf, g.m, g.groups, g.nzp)].x >> 3);
    mx = max(mx, table[table_index(row, zl, g.m, g.groups, g.nzp)].x >> 3);
  }
  const int lo_al = mn & ~(lo_align - 1);  // lo_align is a power of two
  lo[(size_t)tile * g.nv + v] = lo_al;
  atomicMax(wmax, mx - lo_al + 1);
  record_starts(lomax, lo_al);
}

// The same windows for the full table, from the delays themselves (the
// packed table is written relative to them afterwards).
__global__ void k_windows_full(TableGeom tg, TileGeom g, int lo_align, int* lo, int* wmax,
                               int* lomax) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  const int tile = blockIdx.y;
  if (v >= g.nv) return;
  const int tx = tile % g.nxt, tz = tile / g.nxt;
  const int zf = tz * g.tile_z, zl = zf + g.tile_z - 1;
  int mn = 0x7fffffff, mx = -0x7fffffff;
  for (int jj = 0; jj < g.tile_x; ++jj) {
    const double dxv = full_dx(tg, tx * g.tile_x + jj, v);
    int n0;
    double a;
    delay_sample(tg, dxv, pixel_z(tg, zf), &n0, &a);
    mn = min(mn, n0);
    delay_sample(tg, dxv, pixel_z(tg, zl), &n0, &a);
    mx = max(mx, n0);
  }
  const int lo_al = mn & ~(lo_align - 1);
  lo[(size_t)tile * g.nv + v] = lo_al;
  atomicMax(wmax, mx - lo_al + 1);
  record_starts(lomax, lo_al);
}

// Channel-step range of every warp slot.  Without apodisation every step is
// evaluated; with it, only steps whose lattice offset has a non-zero weight on
// the warp's deepest row (the widest aperture of its rows).
__global__ void k_uranges(TileGeom g, FullGeom f, int slots, int u1, int kc, const float* wtab,
                          int2* urange) {
  const int sl = blockIdx.x * blockDim.x + threadIdx.x;
  const int tile = blockIdx.y;
  if (sl >= slots) return;
  int2 r = make_int2(g.u0, u1);
  if (wtab) {
    const int tx = tile % g.nxt, tz = tile / g.nxt;
    const int r_m = sl % g.m, grp = sl / g.m;
    const int jt = tx * g.tile_x + grp * g.m * kc + r_m;
    const int zl = tz * g.tile_z + g.tile_z - 1;
    const int t0 = g.full ? 0 : tile_row(g, jt, 0);  // table row at step u0, m lower at each step
    int ua = u1, ub = g.u0;
    for (int u = g.u0; u < u1; ++u) {
      // lattice: the kC pixels of the slot share one entry at step u; full:
      // pixel c (column jt + m c) pairs with channel u + c, each its own entry
      bool on = false;
      if (g.full) {
        for (int c = 0; c < kc; ++c)
          on |= wtab[full_index(f, tile, u - g.u0, c, sl, g.tile_z - 1)] > 0.f;
      } else {
        on = wtab[table_index_rq(t0 % g.m, t0 / g.m - (u - g.u0), zl, g.groups, g.nzp)] > 0.f;
      }
      if (on) {
        ua = min(ua, u);
        ub = max(ub, u + 1);
      }
    }
    if (ua >= ub) {
      r = make_int2(g.u0, g.u0);
    } else {
      ua = g.u0 + ((ua - g.u0) / kc) * kc;
      ub = g.u0 + ((ub - g.u0 + kc - 1) / kc) * kc;
      r = make_int2(ua, ub);
    }
  }
  urange[(size_t)tile * slots + sl] = r;
}

// Clears the work counter and image maxima before a launch sequence.
__global__ void k_zero_ints(int* p, int n) {
  launch_next();
  wait_previous();
  for (int i = threadIdx.x; i < n; i += blockDim.x) p[i] = 0;
}

// Pairs with a non-zero apodisation weight (for the active-pair rate).
__global__ void k_count_active(TileGeom g, int nx, int nz, int n, const float* wtab,
                               unsigned long long* count) {
  const int z = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  unsigned long long c = 0;
  if (z < nz) {
    const int t0 = tile_row(g, j, -g.u0);  // table row of element 0, m lower at each element
    for (int i = 0; i < n; ++i)
      if (wtab[table_index_rq(t0 % g.m, t0 / g.m - i, z, g.groups, g.nzp)] > 0.f) ++c;
  }
  for (int s = 16; s >= 1; s >>= 1) c += __shfl_xor_sync(0xffffffffu, c, s);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, c);
}

// -------------------------------------------------------- host helpers
double band_weight(double f, double lo, double hi, double roll) {
  if (f >= lo && f <= hi) return 1.0;
  const double u = (f < lo) ? (lo - f) : (f - hi);
  if (u < roll) return 0.5 * (1.0 + std::cos(M_PI * u / roll));
  return 0.0;
}

// Real post-filter mask of one output: raised-cosine band (order-dependent
// default band, or the descriptor's) times the analytic-signal weights.
// Returns true when the band lies wholly above the axial Nyquist rate, in
// which case only DC is removed.
bool build_mask(const pa_plan_desc& d, bool even_order, int M, float* out) {
  const double dz = (d.z1_m - d.z0_m) / d.nz;
  const double f_nyq = d.c_m_s / (2.0 * dz);
  const double f0 = d.f0_hz;
  const double roll = 0.25 * f0;
  const bool off = d.band_hi_hz < 0.0;
  double lo, hi;
  if (d.band_lo_hz > 0.0 && d.band_hi_hz > 0.0) {
    lo = d.band_lo_hz;
    hi = d.band_hi_hz;
  } else if (even_order) {
    lo = 1.5 * f0;
    hi = 2.5 * f0;
  } else {
    lo = 0.5 * f0;
    hi = 1.5 * f0;
  }
  const bool dc_only = !off && lo >= f_nyq;
  hi = std::min(hi, f_nyq);
  for (int b = 0; b < M; ++b) {
    double an = (b == 0 || 2 * b == M) ? 1.0 : (2 * b < M ? 2.0 : 0.0);
    double bp;
    if (an == 0.0) bp = 0.0;
    else if (off) bp = 1.0;
    else if (dc_only) bp = (b == 0) ? 0.0 : 1.0;
    else bp = band_weight(d.c_m_s * b / (M * dz), lo, hi, roll);
    out[b] = (float)(bp * an);
  }
  return dc_only;
}

// pitch / lateral pixel pitch when it is an integer m in 1..32 (the lattice
// table applies), else 0.
int lattice_m(const pa_plan_desc& d) {
  const double dx = (d.x1_m - d.x0_m) / d.nx;
  const double mr = d.pitch_m / dx;
  const double mi = std::round(mr);
  if (mi < 1 || mi > 32 || std::fabs(mr - mi) > 1e-6 * mi) return 0;
  return (int)mi;
}

pa_status validate(const pa_plan_desc* d) {
  if (!d) return fail(PA_EINVAL, "null descriptor");
  if (d->n_elem < 1) return fail(PA_EINVAL, "n_elem must be >= 1 (got %d)", d->n_elem);
  if (d->n_samples < 2) return fail(PA_EINVAL, "n_samples must be >= 2 (got %d)", d->n_samples);
  if (d->nx < 1 || d->nz < 1) return fail(PA_EINVAL, "empty image grid %dx%d", d->nx, d->nz);
  if (d->order_k < 1 || d->order_k > kMaxOrder)
    return fail(PA_EINVAL, "order_k must be in 1..%d (got %d)", kMaxOrder, d->order_k);
  if (d->n_elem < d->order_k)
    return fail(PA_EINVAL, "order_k=%d needs at least as many elements (n_elem=%d)", d->order_k,
                d->n_elem);
  if (!(d->pitch_m > 0) || !(d->c_m_s > 0) || !(d->fs_hz > 0))
    return fail(PA_EINVAL, "pitch, c and fs must be positive");
  if (!(d->x1_m > d->x0_m) || !(d->z1_m > d->z0_m))
    return fail(PA_EINVAL, "grid extents must be increasing");
  if (d->z0_m < 0) return fail(PA_EINVAL, "z0 must be >= 0 (pixels in front of the array)");
  if ((d->outputs & 7u) == 0 || (d->outputs & ~7u))
    return fail(PA_EINVAL, "outputs mask 0x%x invalid", d->outputs);
  if (d->rf_dtype != PA_RF_F32 && d->rf_dtype != PA_RF_BF16 && d->rf_dtype != PA_RF_F16)
    return fail(PA_EINVAL, "rf_dtype %d invalid", (int)d->rf_dtype);
  if (d->f_number < 0) return fail(PA_EINVAL, "f_number must be >= 0");
  if (d->interp != PA_INTERP_LINEAR && d->interp != PA_INTERP_NEAREST)
    return fail(PA_EINVAL, "interp %d invalid", (int)d->interp);
  if (d->f_number > 0 || d->band_hi_hz >= 0) {
    if (!(d->f0_hz > 0) && !(d->band_lo_hz > 0 && d->band_hi_hz > 0) && d->band_hi_hz >= 0)
      return fail(PA_EINVAL, "f0_hz must be positive for the default band");
  }
  if (d->max_batch > 65535) return fail(PA_EINVAL, "max_batch must be <= 65535");
  if (d->delay_table != PA_TABLE_AUTO && d->delay_table != PA_TABLE_LATTICE &&
      d->delay_table != PA_TABLE_FULL)
    return fail(PA_EINVAL, "delay_table %d invalid", (int)d->delay_table);
  if (d->delay_table == PA_TABLE_LATTICE && lattice_m(*d) == 0)
    return fail(PA_EINVAL,
                "pitch / lateral pixel pitch = %.9g is not an integer in 1..32: the lattice "
                "delay table needs (x1-x0)/nx = pitch/m (PA_TABLE_AUTO or PA_TABLE_FULL take "
                "any grid)",
                d->pitch_m * d->nx / (d->x1_m - d->x0_m));
  return PA_OK;
}

// Tiling from the descriptor alone (no device work).
void configure(pa_plan_s* P) {
  const pa_plan_desc& d = P->d;
  P->K = d.order_k;
  P->apod = d.f_number > 0;
  P->comp = d.compensated != 0;
  const double dx = (d.x1_m - d.x0_m) / d.nx;
  const int lm = lattice_m(d);
  P->full = d.delay_table == PA_TABLE_FULL || (d.delay_table == PA_TABLE_AUTO && lm == 0);
  // 32-column tiles halve the staged samples per pair; small images keep
  // 16-column tiles so that there are enough tiles to fill the GPU, unless a
  // full launch (max_batch frames) holds at least 1024 32 x 32 tiles.
  const int64_t wide_tiles =
      (int64_t)((d.nx + 31) / 32) * ((d.nz + 31) / 32) * std::max(1, d.max_batch);
  const bool big = (int64_t)d.nx * d.nz >= 512 * 512 || wide_tiles >= 1024;
  if (P->full) {
    // No table entry is shared, so the column stride m of a thread's pixels
    // is free: 4 (as the lattice has at cfg2) keeps a warp's slots on
    // neighbouring columns, whose delays for one channel differ least, so
    // its shared-memory gathers stay narrow.  The RF window of a tile spans
    // the delays over its lateral extent: tiles stay within ~3.2 mm.
    int cols = big ? 32 : 16;
    while (cols > 8 && cols * dx > 3.2e-3) cols /= 2;
    P->m = cols >= 16 ? 4 : 2;
    P->R = cols / (P->m * kC);
  } else {
    P->m = lm;
    P->R = std::max(1, (big ? 8 : 4) / P->m);
  }
  P->slots = P->m * P->R;
  int B = 1;
  for (int b = 1; b <= 8; ++b)
    if (P->slots % b == 0) B = b;
  if (B == 1) {  // prime m > 8: pair up column groups so a block has two warps
    P->R *= 2;
    P->slots *= 2;
    B = 2;
  }
  P->warps = B;
  P->ngroups = P->slots / B;
  // Lane groups of 8 rows x 4 neighbouring slots (a half-warp's shared
  // gather spans ~18 slots instead of ~32) for orders <= 4 without
  // apodisation, where the block's warps split that way.  Apodised plans
  // keep 32 rows x 1 slot, because a warp iterates over the union of its
  // slots' channel ranges; orders >= 5 are arithmetic-bound and lose to the
  // split table loads of 8-row groups.  Measured on GB300 (fused kernel per
  // launch, 32 -> 8 rows): cfg2 FP32 k = 1, 2 0.594 -> 0.488 ms, k = 3
  // 0.651 -> 0.641 ms, k = 4 0.701 -> 0.692 ms, k = 5 0.831 -> 0.837 ms,
  // k = 7 1.280 -> 1.339 ms; cfg5 (apodised) 2.91 -> 3.06 ms; 16-row groups
  // were never the fastest, and 4-row groups (8 slots per warp) were slower
  // still (k = 2 0.488 -> 0.615 ms, k = 3 0.619 -> 0.671 ms).
  // PA_LANE_ROWS=32|16|8 picks one, for comparisons.
  P->lane_rows_log2 = (B % 4 == 0 && !P->apod && P->K <= 4) ? 3 : 5;
  // Compensated sums keep their Kahan totals in TMEM; its accesses are
  // warp-wide, so every lane of a warp must run the same channel steps:
  // apodised plans (per-slot channel ranges) then keep one slot per warp.
  if (const char* e = getenv("PA_LANE_ROWS")) {
    const int want = atoi(e) == 8 ? 3 : (atoi(e) == 16 ? 4 : 5);
    if (B % (1 << (5 - want)) == 0 && !(P->comp && P->apod)) P->lane_rows_log2 = want;
  }
  P->threads = 32 * B;
  P->tile_x = P->m * kC * P->R;
  P->tile_z = 32;
  P->nxt = (d.nx + P->tile_x - 1) / P->tile_x;
  P->nzt = (d.nz + P->tile_z - 1) / P->tile_z;
  P->n_tiles = P->nxt * P->nzt;
  P->nx_pad = P->nxt * P->tile_x;
  P->nz_pad = P->nzt * P->tile_z;
  P->u0 = -(kC - 1);
  const int steps = ((d.n_elem + kC - 1 + kC - 1) / kC) * kC;  // round N + kC - 1 up
  P->u1 = P->u0 + steps;
  const int i_max = P->u1 - 1 + kC - 1;
  P->nv = i_max - P->u0 + 1;
  if (P->full) {  // one entry per evaluated (pixel, channel step) pair
    P->dmin = 0;
    P->ndrows = 0;
    P->full_entries = (size_t)P->n_tiles * (steps + 3) * 32 * P->slots * kC;
  } else {
    // whole groups of four lattice sequence numbers per residue, from the
    // pair of column 0 and the last virtual channel to that of the last
    // padded column and the first one
    P->dmin = -P->m * steps;
    P->tgroups = (P->nx_pad / P->m + steps) / 4 + 1;
    P->ndrows = 4 * P->m * P->tgroups;
  }
  P->M = 1;
  P->log2M = 0;
  while (P->M < d.nz) {
    P->M <<= 1;
    ++P->log2M;
  }
  // warps per post block: most resident warps per SM for the shared memory
  // they need (post_buffers padded M-point buffers per team of
  // post_team_warps warps, plus the twiddles and mask), in whole teams
  {
    const int tw_warps = post_team_warps(P->M);
    const size_t per_team = (size_t)post_buffers(P->M) * post_padded_len(P->M) * sizeof(float2);
    const size_t tw = (size_t)P->M * (sizeof(float2) + sizeof(float));  // twiddles + mask
    const size_t sm_bytes = 227 * 1024;
    int best = tw_warps;
    size_t best_warps = 0;
    for (int w = tw_warps; w <= 8; w += tw_warps) {
      const size_t blk = (w / tw_warps) * per_team + tw + 1024;
      const size_t warps = (sm_bytes / blk) * w;
      if (blk <= 200 * 1024 && warps > best_warps) {
        best_warps = warps;
        best = w;
      }
    }
    P->post_wpb = best;
  }
  P->n_out = popcount3(d.outputs);
  int s = 0;
  for (int o = 0; o < 3; ++o) P->out_id[o] = (d.outputs >> o & 1u) ? s++ : -1;
  P->dyn_range = d.dyn_range_db > 0 ? (float)d.dyn_range_db : 60.f;
  P->elt = d.rf_dtype == PA_RF_F32 ? 4 : 2;
  // TMA boxes start on 16-byte boundaries: window starts are multiples of
  // 16 / elt samples, and rows must be 16-byte strided.
  P->lo_align = (int)(16 / P->elt);
  // zero slots on either side of a prepared row: at least the widest RF
  // window, i.e. the largest delay difference over a tile plus the rounding
  // of its ends
  {
    const double dz = (d.z1_m - d.z0_m) / d.nz;
    const double span = d.fs_hz / d.c_m_s * std::hypot(P->tile_x * dx, P->tile_z * dz);
    P->slot_margin = ((int)std::min(span, 1e6) + P->lo_align + 8) / 4 * 4;
    P->slot_mode = pipe_slot_mode(P->K, P->apod, d.interp == PA_INTERP_NEAREST);
    // 16-byte rows
    P->slot_pitch = ((long long)d.n_samples + 1) / 2 * 2 + 2ll * P->slot_margin;
  }
  // Measured on GB300: TMA staging wins for 16-bit RF (half-size raw buffer),
  // vectorised loads win for FP32 RF (the FP32 raw buffer costs a resident
  // block per SM).  PA_STAGING=tma|loads overrides the choice.
  P->use_tma = (d.n_samples % P->lo_align) == 0 && P->elt == 2;
  // Failure injection for tests, compiled into the checked build only: every
  // chunk expects 16 bytes more than its boxes deliver, so each block's
  // bounded wait runs out (about a second), sets error flag 8, counts a
  // timeout and ends.  Every box of the chunk has landed by then (only the
  // expected count is short), so no copy is left in flight.
#ifdef PA_CHECK_BOUNDS
  P->expect_extra = getenv("PA_INJECT_TMA_SHORTFALL") ? 16 : 0;
#endif
  const char* staging = getenv("PA_STAGING");
  if (staging && strcmp(staging, "loads") == 0) P->use_tma = false;
  if (staging && strcmp(staging, "tma") == 0) P->use_tma = (d.n_samples % P->lo_align) == 0;
  if (const char* e = getenv("PA_ITEM_FRAMES")) P->item_frames = atoi(e);
  if (P->d.max_batch <= 0) P->d.max_batch = 1;
}

// Resident fused-kernel blocks per SM.  For plans that keep their Kahan
// totals in TMEM the count comes from the kernel's registers, shared memory
// and threads (the occupancy calculator reports one block per SM for a
// kernel that allocates tensor memory) and is capped so that the resident
// blocks' TMEM columns fit the SM's 512.
// (Resident blocks of form f from its kernel's attributes a: what the
// occupancy calculator gives without tensor memory.)
int blocks_by_attributes(const FusedForm& f, const cudaFuncAttributes& a, size_t smem) {
  struct Limits {
    int regs = 0, smem = 0, threads = 0, blocks = 0, reserved = 0;
    Limits() {
      int dev = 0;
      if (cudaGetDevice(&dev) != cudaSuccess) return;
      cudaDeviceGetAttribute(&regs, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
      cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
      cudaDeviceGetAttribute(&threads, cudaDevAttrMaxThreadsPerMultiProcessor, dev);
      cudaDeviceGetAttribute(&blocks, cudaDevAttrMaxBlocksPerMultiprocessor, dev);
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    }
  };
  static const Limits lim;  // (one architecture: the same on every device)
  const int warps = (f.threads + 31) / 32;
  const int regs_warp = ((a.numRegs * 32 + 255) / 256) * 256;  // 256-register units per warp
  int b = std::min(lim.regs / std::max(1, regs_warp * warps), lim.threads / (32 * warps));
  b = std::min(b, (int)((size_t)lim.smem / (smem + a.sharedSizeBytes + (size_t)lim.reserved)));
  b = std::min(b, lim.blocks);
  if (f.tmem_cols) b = std::min(b, kTmemColsPerSm / f.tmem_cols);
  return std::max(0, b);
}

cudaError_t fused_blocks_per_sm(const pa_plan_s* P, const FusedForm& f, size_t smem, int* n) {
  cudaError_t e = bf_occupancy(f.func, f.threads, smem, n);
  if (e != cudaSuccess || !f.tmem_cols) return e;
  cudaFuncAttributes a;
  e = cudaFuncGetAttributes(&a, f.func);
  if (e != cudaSuccess) return e;
  *n = blocks_by_attributes(f, a, smem);
  return cudaSuccess;
}

// The one-frame form stages this plan's RF windows sample by sample (rows off
// 16-byte boundaries).
bool staged_by_samples(const pa_plan_s* P) { return !P->use_tma && P->d.n_samples % 4 != 0; }

// Whether some kernel of the plan waits for copies (and may give up): the
// one-frame form by TMA, the others always.
bool may_wait(const pa_plan_s* P) {
  return P->use_tma || P->form[1].nf || P->form[2].nf || P->form[3].nf;
}

// Largest launch, in warps of 4-pixel threads, for which the fine-grained forms
// (one pixel a thread, and two) are built, and the least mean channel steps per
// pixel; pick_form says which of these launches run them, and why.
struct FineLimits {
  int px1, px2;
};
FineLimits fine_limits(const pa_plan_s* P) {
  // (the variants that have kernels)
  const bool one = !P->full || !P->comp || P->K < 8;
  const bool two = !P->comp && P->K <= 5 && (P->full || P->K >= 3);
  if (P->item_frames == 3) return {one ? 1 << 20 : 0, 0};  // tests
  if (P->item_frames == 4) return {0, two ? 1 << 20 : 0};
  if (P->item_frames != 0 || (!P->full && P->use_tma)) return {0, 0};
  return {one ? 1100 : 0, two && (P->full || staged_by_samples(P)) ? 2400 : 0};
}
double fine_steps(const pa_plan_s* P) { return P->item_frames >= 3 ? 1e9 : P->steps_per_pixel; }
double least_fine_steps(const pa_plan_s* P, int px) {
  const bool loads = !P->full && !staged_by_samples(P);
  return px == 2 || (loads && P->K <= 2) ? 50 : 28;
}
// Warps of 4-pixel threads of one frame.
int64_t frame_warps(const pa_plan_s* P) { return (int64_t)P->n_tiles * P->slots; }

bool fine_pays(const pa_plan_s* P, int px, int nf);  // (with pick_form)
bool pairs_pay(const pa_plan_s* P, int nf);

// Bytes of a row of form i's prepared slots, and of the rows of a work item.
size_t slot_row_bytes(const pa_plan_s* P, int i) {
  return (size_t)P->slot_pitch * (i == 1 ? pipe_slot_bytes(P->slot_mode) : sizeof(float2));
}
size_t slot_item_bytes(const pa_plan_s* P, int i) { return (size_t)P->d.n_elem * slot_row_bytes(P, i); }
// Bound of a round's slots; a plan whose work items are larger has no such form.
constexpr size_t kSlotBytesMax = (size_t)512 << 20;

// Whether some launch of the plan picks the two-frame form (an even one or an
// odd one of the largest; build_form2 may still find that it does not fit).
bool pairs_wanted(const pa_plan_s* P) {
  if (P->d.max_batch <= 1 || P->K > 5 || slot_item_bytes(P, 1) > kSlotBytesMax) return false;
  if (P->item_frames != 0) return P->item_frames == 2;
  return pairs_pay(P, P->d.max_batch) || pairs_pay(P, P->d.max_batch - 1);
}

// Most frames of a launch that picks a fine-grained form of px pixels a thread
// (0: none does).
int fine_wanted(const pa_plan_s* P, int px) {
  const FineLimits lim = fine_limits(P);
  if (slot_item_bytes(P, 2) > kSlotBytesMax || fine_steps(P) < least_fine_steps(P, px)) return 0;
  for (int64_t nf = std::min<int64_t>(P->d.max_batch, (px == 1 ? lim.px1 : lim.px2) / frame_warps(P));
       nf > 0; --nf)
    if (fine_pays(P, px, (int)nf)) return (int)nf;
  return 0;
}

// Frames per round of form 1 (of a launch of forms 2 and 3) and the bytes of
// their slots.  The slots of a round are written by the preparation pass and
// read back by every tile.
size_t slots_size(const pa_plan_s* P, int i, int* frames) {
  const int item = i == 1 ? 2 : 1;
  const size_t want = i == 1 ? ((size_t)P->d.max_batch + 1) / 2
                             : (size_t)std::max(fine_wanted(P, 1), fine_wanted(P, 2));
  const size_t items = std::min(want, kSlotBytesMax / slot_item_bytes(P, i));
  *frames = (int)(item * items);
  return slot_row_bytes(P, i) + items * slot_item_bytes(P, i);
}

// Bytes of the delay table and its apodisation weights.
size_t delay_table_bytes(const pa_plan_s* P) {
  if (P->full) return P->full_entries * (sizeof(int2) + (P->apod ? sizeof(float) : 0));
  return (size_t)P->ndrows * P->nz_pad * (sizeof(int2) + (P->apod ? sizeof(float) : 0));
}

pa_status check_table_size(const pa_plan_s* P) {
  if (P->full && delay_table_bytes(P) > PA_FULL_TABLE_MAX_BYTES)
    return fail(PA_EUNSUPPORTED,
                "the full delay table of %zu entries (%zu bytes) exceeds "
                "PA_FULL_TABLE_MAX_BYTES",
                P->full_entries, delay_table_bytes(P));
  return PA_OK;
}

// The plan's device memory but for the optional prepared slots, one allocation:
// lays the arrays out from `base` on (null: sizes only) and returns the bytes.
// (One cudaMalloc of some megabytes costs 30 us and its cudaFree as much; eleven
// allocations of their own 50-80 us more.)
size_t plan_arena(pa_plan_s* P, unsigned char* base) {
  size_t at = 0;
  auto take = [&](auto** p, size_t n) {
    if (base) *p = reinterpret_cast<std::remove_reference_t<decltype(**p)>*>(base + at);
    at += (n * sizeof(**p) + 255) & ~(size_t)255;
  };
  const size_t tab_n = P->full ? P->full_entries : (size_t)P->ndrows * P->nz_pad;
  take(P->full ? &P->ftab : &P->table, tab_n);
  if (P->apod) take(&P->wtab, tab_n);
  take(&P->items, (size_t)P->n_tiles * P->ngroups);
  take(&P->slot_rg, (size_t)P->slots);
  take(&P->lo, (size_t)P->n_tiles * P->nv);
  take(&P->urange, (size_t)P->n_tiles * P->slots);
  take(&P->chunks, (size_t)P->n_tiles * (2 * P->ngroups + 2));  // of forms 0, 1 and 2, 3
  take(&P->tw, (size_t)3 * P->M);  // n_tw <= 2 M, tw_reg
  take(&P->mask, (size_t)3 * P->M);
  take(&P->active, (size_t)1);
  // [0] error flags, [1] work counter, [2, 2 + 3 max_batch) image maxima,
  // [last] running count of timed-out waits
  P->scratch_ints = 3 + (size_t)P->d.max_batch * 3;
  take(&P->scratch[0], P->scratch_ints);
  return at;
}

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime.
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  }();
  return fn;
}

size_t round256(size_t b) { return (b + 255) & ~(size_t)255; }

template <typename T>
pa_status dalloc(pa_plan_s* P, T** ptr, size_t n) {
  if (n == 0) n = 1;
  cudaError_t e = cudaMalloc((void**)ptr, n * sizeof(T));
  if (e != cudaSuccess) {
    *ptr = nullptr;
    cudaGetLastError();
    return fail(e == cudaErrorMemoryAllocation ? PA_ENOMEM : PA_ECUDA, "cudaMalloc(%zu): %s",
                n * sizeof(T), cudaGetErrorString(e));
  }
  P->device_bytes += n * sizeof(T);
  return PA_OK;
}

void drop_host_graphs(pa_plan_s* P) {
  for (auto& g : P->host_graphs) {
    cudaGraphExecDestroy(g.exec);
    cudaGraphDestroy(g.graph);
  }
  P->host_graphs.clear();
}

// Staging buffers of the host path: one allocation, or what the arena's last
// page leaves if they fit there.
void free_staging(pa_plan_s* P) {
  drop_host_graphs(P);
  if (P->h_rf != P->spare) cudaFree(P->h_rf);
  P->device_bytes -= P->h_rf_bytes + P->h_out_bytes;
  P->h_rf = nullptr;
  P->h_out = nullptr;
  P->h_rf_bytes = P->h_out_bytes = 0;
}
pa_status alloc_staging(pa_plan_s* P, size_t rf, size_t out) {
  free_staging(P);
  const size_t at = round256(rf);
  if (at + out <= P->spare_bytes) P->h_rf = P->spare;
  else PA_CUDA(cudaMalloc(&P->h_rf, at + out));
  P->h_out = reinterpret_cast<float*>((unsigned char*)P->h_rf + at);
  P->h_rf_bytes = rf;
  P->h_out_bytes = out;
  P->device_bytes += rf + out;
  return PA_OK;
}

void free_plan(pa_plan_s* P) {
  if (!P) return;
  DeviceGuard g(P->device);
  for (int s = 0; s < kHostSets; ++s)
    if (P->hs[s]) cudaStreamSynchronize(P->hs[s]);
  free_staging(P);
  if (!P->slots_joined) cudaFree(P->slot_mem);
  cudaFree(P->arena);
  for (int s = 1; s < kHostSets; ++s) cudaFree(P->scratch[s]);
  for (int s = 0; s < kHostSets; ++s)
    if (P->hs[s]) cudaStreamDestroy(P->hs[s]);
  if (P->host_flag) g_host_words.give(P->host_flag);
  if (P->h_ev) cudaEventDestroy(P->h_ev);
  for (int s = 0; s < kHostSets; ++s)
    if (P->h_done[s]) cudaEventDestroy(P->h_done[s]);
  for (auto& g : P->graphs) {
    cudaGraphExecDestroy(g.exec);
    cudaGraphDestroy(g.graph);
  }
  for (auto& e : P->ev_free) {
    cudaEventDestroy(e.first);
    cudaEventDestroy(e.second);
  }
  for (auto& e : P->ev_used) {
    cudaEventSynchronize(e.second.second);
    cudaEventDestroy(e.second.first);
    cudaEventDestroy(e.second.second);
  }
  delete P;
}

// Shared memory of a fused-kernel block of form f with c channel steps per
// chunk; *pairs_off is where its interpolation slots start.
size_t form_smem(const pa_plan_s* P, const FusedForm& f, int c, int* pairs_off) {
  const int ncs = c + kC - 1;
  if (f.slot_bytes) {
    const int off = f.nf == 2 ? kPipeSlotOff : kFineSlotOff;
    if (pairs_off) *pairs_off = off;
    return (size_t)off + (size_t)f.stages * ncs * P->window * f.slot_bytes;
  }
  const size_t raw = P->use_tma ? (size_t)ncs * f.rp * P->elt : 0;
  const size_t off = (size_t)kRawOff + ((raw + 127) & ~size_t(127));
  if (pairs_off) *pairs_off = (int)off;
  return off + (size_t)ncs * P->window * 8;
}

// TMEM-dense: a block can hold more than its register share of an SM's TMEM
// columns (see plan_tmem).
bool form_dense(const pa_plan_s* P, const FusedForm& f) {
  if (!f.tmem_cols) return false;
  cudaFuncAttributes a;
  int regs_sm = 65536;
  cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, P->device);
  if (cudaFuncGetAttributes(&a, f.func) != cudaSuccess) {
    cudaGetLastError();
    return true;  // unknown: treat as dense (serialised with other compensated batches)
  }
  const size_t warps = (size_t)(f.threads + 31) / 32;
  const size_t regs_block = (size_t)((a.numRegs * 32 + 255) / 256) * 256 * warps;
  return (size_t)f.tmem_cols * (size_t)regs_sm > (size_t)kTmemColsPerSm * regs_block;
}

// Chunk range of every (tile, share of its slots) of form f: per residue
// group, or (forms 2, 3) of whole tiles.
std::vector<int2> form_chunks(const pa_plan_s* P, const FusedForm& f, const std::vector<int2>& ur) {
  const int groups = f.slots_form > 1 ? 1 : P->ngroups, per = P->slots / groups;
  std::vector<int2> vk((size_t)P->n_tiles * groups);
  for (int t = 0; t < P->n_tiles; ++t) {
    for (int gr = 0; gr < groups; ++gr) {
      int ua = P->u1, ub = P->u0;
      for (int w = 0; w < per; ++w) {
        const int2 r = ur[(size_t)t * P->slots + gr * per + w];
        if (r.y > r.x) {
          ua = std::min(ua, r.x);
          ub = std::max(ub, r.y);
        }
      }
      int2 c = make_int2(0, 0);
      if (ub > ua) c = make_int2((ua - P->u0) / f.nc, (ub - P->u0 + f.nc - 1) / f.nc);
      vk[(size_t)t * groups + gr] = c;
    }
  }
  return vk;
}

// Prepared slots are extra: a plan runs the one-frame form without them.  They
// are taken within the plan's limit and while an eighth of the device's memory
// stays free beside them.
bool room_for_slots(const pa_plan_s* P, size_t bytes) {
  size_t free_b = 0, total = 0;
  return bytes <= P->slot_limit && cudaMemGetInfo(&free_b, &total) == cudaSuccess &&
         bytes + total / 8 <= free_b;
}

// The arena, and with it the slots that the plan is expected to want: one
// allocation takes half the time of two.  The device maps pages of 2 MiB, so
// such an allocation asks for whole ones; what its last page leaves serves the
// staging buffers of the host path if they fit.
pa_status alloc_arena(pa_plan_s* P, size_t slots) {
  constexpr size_t kPage = (size_t)2 << 20;
  const size_t n = plan_arena(P, nullptr);
  const size_t pages = (n + slots + kPage - 1) / kPage * kPage;
  if (slots && n + slots > kPage && room_for_slots(P, slots) && dalloc(P, &P->arena, pages) == PA_OK) {
    P->slot_mem = P->arena + n;
    P->slot_mem_bytes = slots;
    P->slots_joined = true;
    P->spare = P->slot_mem + slots;
    P->spare_bytes = pages - n - slots;
    P->device_bytes -= P->spare_bytes;
  } else if (const pa_status s = dalloc(P, &P->arena, n)) {
    return s;
  }
  plan_arena(P, P->arena);
  return PA_OK;
}

// Gives the slots' memory back (the device idle, no graph of the plan alive):
// joined with the arena, the arena moves to an allocation of its own.
pa_status drop_slot_memory(pa_plan_s* P) {
  if (P->slots_joined) {
    const size_t n = plan_arena(P, nullptr);
    unsigned char* a = nullptr;
    if (P->h_rf && P->h_rf == P->spare) free_staging(P);
    PA_CUDA(cudaMalloc(&a, n));
    const cudaError_t e = cudaMemcpy(a, P->arena, n, cudaMemcpyDeviceToDevice);
    if (e != cudaSuccess) {
      cudaFree(a);
      return fail(PA_ECUDA, "plan arena: %s", cudaGetErrorString(e));
    }
    cudaFree(P->arena);
    P->spare = nullptr;
    P->spare_bytes = 0;
    P->arena = a;
    plan_arena(P, a);
    for (FusedForm& f : P->form) f.vchunks = P->chunks + f.chunk_at;
  } else {
    cudaFree(P->slot_mem);
  }
  P->slot_mem = nullptr;
  P->device_bytes -= P->slot_mem_bytes;
  P->slot_mem_bytes = 0;
  P->slots_joined = false;
  return PA_OK;
}

// Bytes of slots a plan over the full aperture will want, from its descriptor
// alone, for the arena's allocation.  Stands on estimates that the build then
// replaces; apodised plans, whose channel steps come from the tables, are left
// for later (0).
size_t expected_slots(pa_plan_s* P) {
  if (P->apod) return 0;
  const double steps = P->u1 - P->u0;
  P->steps_per_pixel = steps;
  P->form[0].blocks_per_sm = std::max(1, 24 / P->warps);
  // samples between the nearest delay and the farthest
  const pa_plan_desc& d = P->d;
  const double half = 0.5 * (d.n_elem - 1) * d.pitch_m;
  const double far = std::hypot(d.z1_m, std::max(d.x1_m, -d.x0_m) + half);
  const double used = std::min((double)d.n_samples, d.fs_hz / d.c_m_s * (far - d.z0_m));
  P->pairs_pay = steps * P->nx_pad * P->nz_pad >= 48.0 * d.n_elem * used;
  int frames = 0;
  size_t b = 0;
  if (pairs_wanted(P)) b += round256(slots_size(P, 1, &frames));
  if (fine_wanted(P, 1) || fine_wanted(P, 2)) b += round256(slots_size(P, 2, &frames));
  return b;
}

// Slots of form 1 and those forms 2 and 3 share, in one allocation, and the
// chunk ranges of every form.
pa_status alloc_forms(pa_plan_s* P, const std::vector<int2>& ur, cudaStream_t st) {
  int frames1 = 0, frames2 = 0;
  const size_t s1 = P->form[1].nf ? round256(slots_size(P, 1, &frames1)) : 0;
  const size_t s2 = P->form[2].nf || P->form[3].nf ? round256(slots_size(P, 2, &frames2)) : 0;
  if (P->slot_mem && (P->slot_mem_bytes < s1 + s2 || s1 + s2 == 0)) {  // expected otherwise
    PA_CUDA(cudaStreamSynchronize(st));
    if (const pa_status s = drop_slot_memory(P)) return s;
  }
  if (s1 + s2 && !P->slot_mem) {
    if (room_for_slots(P, s1 + s2) && dalloc(P, &P->slot_mem, s1 + s2) == PA_OK)
      P->slot_mem_bytes = s1 + s2;
    else
      for (int i = 1; i < 4; ++i) P->form[i] = FusedForm();
  }
  if (P->slot_mem) PA_CUDA(cudaMemsetAsync(P->slot_mem, 0, s1 + s2, st));
  std::vector<int2> all;
  for (int i = 0; i < 4; ++i) {
    FusedForm& f = P->form[i];
    if (!f.nf) continue;
    f.chunk_at = all.size();
    f.vchunks = P->chunks + f.chunk_at;
    if (i) f.slots = P->slot_mem + (i == 1 ? 0 : s1);
    f.max_frames = i == 1 ? frames1 : frames2;
    const std::vector<int2> vk = form_chunks(P, f, ur);
    all.insert(all.end(), vk.begin(), vk.end());
  }
  // (pageable: the call returns once `all` has been read)
  PA_CUDA(cudaMemcpyAsync(P->chunks, all.data(), all.size() * sizeof(int2), cudaMemcpyHostToDevice, st));
  return PA_OK;
}

// The one-frame form.
pa_status build_form1(pa_plan_s* P) {
  FusedForm& f = P->form[0];
  f.nf = 1;
  f.func = bf_func(P->K, P->apod, P->comp, P->full);
  f.threads = P->threads;
  f.tmem_cols = P->comp ? tmem_columns(P->warps, P->K <= 2 ? 3 : P->K + 2) : 0;
  f.rp = (int)((((size_t)P->wr * P->elt + 127) & ~size_t(127)) / P->elt);
  // Chunk length: every chunk costs a staging pass and two block barriers,
  // so the channel steps are cut into as few, evenly sized chunks as keep
  // the fused kernel's occupancy at what 32-step chunks give (measured at
  // N = 128: 5 chunks of 28 steps 0.696 ms, 4 of 36 0.692 ms, 3 of 44
  // 0.678 ms).  Limits: the slot buffer (at most 200 KiB), one issuing lane
  // per staged channel under TMA (ncs <= 32 warps), and the multiply-shift
  // division of the staging loops (exact while ncs * (W/4)^2 < 2^20).
  // PA_CHUNK_STEPS caps the chunk length (for measurements).
  const int steps = P->u1 - P->u0;
  auto fits = [&](int c) {
    const int ncs = c + kC - 1;
    const long long w4 = P->window / 4;
    return form_smem(P, f, c, nullptr) <= 200 * 1024 && ncs <= 32 * P->warps &&
           (long long)ncs * w4 * w4 < (1ll << 20);
  };
  auto occupancy = [&](int c) {
    int b = 0;
    if (fused_blocks_per_sm(P, f, form_smem(P, f, c, nullptr), &b) != cudaSuccess) b = 0;
    return b;
  };
  auto even = [&](int nch) { return ((steps + nch - 1) / nch + kC - 1) / kC * kC; };
  int cap = kNCMax;
  if (const char* e = getenv("PA_CHUNK_STEPS")) cap = std::max(kC, std::min(kNCMax, atoi(e)));
  int ref = std::min(32, cap);
  while (ref > kC && !fits(ref)) ref -= kC;
  const int occ_ref = occupancy(ref);
  int nc = ref;
  for (int nch = (steps + cap - 1) / cap; nch <= (steps + ref - 1) / ref; ++nch) {
    const int c = std::min(even(nch), cap);
    if (c > ref && fits(c) && occupancy(c) >= occ_ref) {
      nc = c;
      break;
    }
  }
  if (nc == ref) nc = std::min(ref, even((steps + ref - 1) / ref));
  f.nc = nc;
  cudaGetLastError();

  // shared memory and occupancy of the fused kernel
  f.smem = form_smem(P, f, f.nc, &f.pairs_off);
  const long long w4 = P->window / 4;
  if ((long long)(f.nc + kC - 1) * w4 * w4 >= (1ll << 20))
    return fail(PA_EUNSUPPORTED, "RF window of %d samples per channel is too wide; use a finer "
                "depth grid", P->window);
  if (f.smem > 200 * 1024)
    return fail(PA_EUNSUPPORTED,
                "RF window of %d samples per channel needs %zu B of shared memory; use a finer "
                "depth grid",
                P->window, f.smem);
  // (resident blocks never ask for more TMEM than an SM has, so no block's
  // allocation waits on another block of the same launch)
  PA_CUDA(fused_blocks_per_sm(P, f, f.smem, &f.blocks_per_sm));
  if (f.blocks_per_sm < 1)
    return fail(PA_EUNSUPPORTED, "fused kernel does not fit an SM (%d threads, %zu B smem)",
                P->threads, f.smem);
  return PA_OK;
}

// The two-frame form; a plan it does not fit keeps the one-frame form alone.
pa_status build_form2(pa_plan_s* P) {
  if (P->d.max_batch <= 1 || P->K > 5) return PA_OK;
  FusedForm f;
  f.nf = 2;
  f.slot_bytes = pipe_slot_bytes(P->slot_mode);
  f.func = bf_pipe_func(P->K, P->apod, P->comp, P->full, P->d.interp == PA_INTERP_NEAREST);
  f.threads = P->threads;
  f.stages = 2;
  f.tmem_cols = P->comp ? tmem_columns(P->warps, 2 * (P->K <= 2 ? 3 : P->K + 2)) : 0;
  if (f.tmem_cols > kTmemColsPerSm) return PA_OK;
  const int steps = P->u1 - P->u0;
  cudaFuncAttributes fa;
  PA_CUDA(cudaFuncGetAttributes(&fa, f.func));
  auto occupancy = [&](int c) {
    const size_t smem = form_smem(P, f, c, nullptr);
    return smem > 226 * 1024 ? 0 : blocks_by_attributes(f, fa, smem);
  };
  auto even = [&](int nch) { return ((steps + nch - 1) / nch + kC - 1) / kC * kC; };
  int cap = kNCMax;
  if (const char* e = getenv("PA_CHUNK_STEPS")) cap = std::max(kC, std::min(kNCMax, atoi(e)));
  // the longest evenly cut chunk at the most resident blocks that chunks of
  // at least 12 steps leave
  int best = 0;
  const int most = occupancy(kC);
  for (int b = most; b >= 1 && !best; --b)
    for (int nch = (steps + cap - 1) / cap; nch <= (steps + kC - 1) / kC; ++nch) {
      const int c = std::min(even(nch), cap);
      if (c < std::min(12, cap) && b > 1) break;
      if (occupancy(c) >= b) {
        best = c;
        break;
      }
    }
  if (!best) return PA_OK;
  f.nc = best;
  f.smem = form_smem(P, f, f.nc, &f.pairs_off);
  PA_CUDA(fused_blocks_per_sm(P, f, f.smem, &f.blocks_per_sm));
  if (f.blocks_per_sm < 1 || form_dense(P, f)) return PA_OK;
  // chunks of fewer than 12 steps (RF windows of more than 200 samples) spend
  // their time on the hand-over (0.89 measured at 8 steps)
  if (f.nc < std::min(12, std::min(steps, cap))) return PA_OK;
  // Where pairs_pay asks for it: 12 resident warps (six-warp blocks, wide
  // windows) are enough for orders <= 2 (1.12), not for higher ones (0.92-1.0),
  // and the preparation pass pays where a sample serves enough pairs (a twentieth
  // slower than the one-frame form: 2.5 % of all launches without this line,
  // 1.7 % with it).
  const double reuse = (double)P->executed_pairs /
                       ((double)P->d.n_elem * std::max(1, P->used_hi - P->used_lo));
  P->pairs_pay = reuse >= 48 && f.blocks_per_sm * P->warps >= (P->K <= 2 ? 12 : 14);
  if (!pairs_wanted(P)) return PA_OK;
  if (P->window > P->slot_margin) return PA_OK;  // (the margin bounds it)
  f.slots_form = 1;
  P->form[1] = f;
  return PA_OK;
}

// The fine-grained forms: a tile's pixels at px of a thread's four per thread,
// in blocks of at most 16 warps.
pa_status build_form3(pa_plan_s* P, int px) {
  if (!fine_wanted(P, px) || P->window > P->slot_margin) return PA_OK;
  FusedForm f;
  f.nf = 1;
  f.slot_bytes = sizeof(float2);
  f.stages = kFineStages;
  const int tile_warps = P->slots * kC / px;
  int nw = 1;
  for (int w = 1; w <= 16; ++w)
    if (tile_warps % w == 0) nw = w;
  f.splits = tile_warps / nw;
  f.threads = 32 * nw;
  f.func = bf_fine_func(P->K, P->apod, P->comp, P->full, px);
  const int steps = P->u1 - P->u0;
  cudaFuncAttributes fa;
  PA_CUDA(cudaFuncGetAttributes(&fa, f.func));
  auto occupancy = [&](int c) {
    const size_t smem = form_smem(P, f, c, nullptr);
    return smem > 226 * 1024 ? 0 : blocks_by_attributes(f, fa, smem);
  };
  // the longest evenly cut chunk that leaves 32 warps an SM (or as many as
  // registers allow)
  auto even = [&](int nch) { return ((steps + nch - 1) / nch + kC - 1) / kC * kC; };
  int cap = kNCMax;
  if (const char* e = getenv("PA_CHUNK_STEPS")) cap = std::max(kC, std::min(kNCMax, atoi(e)));
  const int most = occupancy(kC);
  int best = 0;
  for (int nch = (steps + cap - 1) / cap; nch <= (steps + kC - 1) / kC && !best; ++nch) {
    const int c = std::min(even(nch), cap);
    const int b = occupancy(c);
    if (b >= 1 && b * nw >= std::min(most * nw, 32)) best = c;
  }
  if (!best) return PA_OK;
  f.nc = best;
  f.smem = form_smem(P, f, f.nc, &f.pairs_off);
  PA_CUDA(fused_blocks_per_sm(P, f, f.smem, &f.blocks_per_sm));
  if (f.blocks_per_sm < 1) return PA_OK;
  f.slots_form = px + 1;
  P->form[px + 1] = f;
  return PA_OK;
}

pa_status build_plan(pa_plan_s* P, cudaStream_t st) {
  const pa_plan_desc& d = P->d;
  PA_CUDA(cudaGetDevice(&P->device));
  PA_CUDA(cudaDeviceGetAttribute(&P->num_sms, cudaDevAttrMultiProcessorCount, P->device));

  pa_status s;
  if ((s = check_table_size(P)) != PA_OK) return s;
  // (slots that a caller limits may be given back later: an allocation of their own)
  const bool join = P->slot_limit == kNoSlotLimit;
  if ((s = alloc_arena(P, join ? expected_slots(P) : 0)) != PA_OK) return s;
  PA_CUDA(cudaMemsetAsync(P->scratch[0], 0, P->scratch_ints * sizeof(int), st));

  if ((size_t)36 * P->M > (size_t)200 * 1024)
    return fail(PA_EUNSUPPORTED, "nz = %d needs a %d-point envelope FFT; at most 4096 is supported",
                d.nz, P->M);

  // delay / apodisation table
  TableGeom tg;
  tg.ndrows = P->ndrows;
  tg.nzp = P->nz_pad;
  tg.m = P->m;
  tg.groups = P->tgroups;
  tg.dmin = P->dmin;
  tg.ns = d.n_samples;
  tg.nearest = d.interp == PA_INTERP_NEAREST;
  tg.dx = (d.x1_m - d.x0_m) / d.nx;
  tg.x_const = d.x0_m + 0.5 * (d.n_elem - 1) * d.pitch_m;
  tg.z0 = d.z0_m;
  tg.dz = (d.z1_m - d.z0_m) / d.nz;
  tg.fs = d.fs_hz;
  tg.c = d.c_m_s;
  tg.t0 = d.t0_s;
  tg.fnum = d.f_number;
  tg.x0 = d.x0_m;
  tg.pitch = d.pitch_m;
  tg.n_elem = d.n_elem;
  tg.u0 = P->u0;
  tg.nv = P->nv;

  // per-tile windows and warp ranges
  TileGeom g;
  g.nxt = P->nxt;
  g.nzt = P->nzt;
  g.tile_x = P->tile_x;
  g.tile_z = P->tile_z;
  g.m = P->m;
  g.dmin = P->dmin;
  g.nzp = P->nz_pad;
  g.nv = P->nv;
  g.u0 = P->u0;
  g.ndrows = P->ndrows;
  g.groups = P->tgroups;
  g.full = P->full ? 1 : 0;
  FullGeom fg{P->nxt, P->n_tiles, P->tile_x, P->tile_z, P->m, P->slots, P->u1 - P->u0,
              P->lane_rows_log2, d.nx, d.nz, d.n_elem, P->u0, P->nv};
  // borrowed before first use as image maxima: window width, window starts
  int* wmax = P->scratch[0] + 2;
  int* lomax = P->scratch[0] + 3;
  if (P->full) {
    // windows first: the packed entries are written relative to them
    dim3 gw((P->nv + 127) / 128, P->n_tiles);
    k_windows_full<<<gw, 128, 0, st>>>(tg, g, P->lo_align, P->lo, wmax, lomax);
    PA_CUDA(cudaGetLastError());
    const size_t per_tile = P->full_entries / P->n_tiles;
    dim3 gt((unsigned)((per_tile + 255) / 256), P->n_tiles);
    k_table_full<<<gt, 256, 0, st>>>(tg, fg, P->lo, P->ftab, P->wtab);
    PA_CUDA(cudaGetLastError());
  } else {
    dim3 gt(P->ndrows, (P->nz_pad + 127) / 128);
    k_table<<<gt, 128, 0, st>>>(tg, P->table, P->wtab);
    PA_CUDA(cudaGetLastError());
    dim3 gw((P->nv + 127) / 128, P->n_tiles);
    k_windows<<<gw, 128, 0, st>>>(g, P->lo_align, P->table, P->lo, wmax, lomax, P->scratch[0]);
    PA_CUDA(cudaGetLastError());
  }
  {
    dim3 grid((P->slots + 31) / 32, P->n_tiles);
    k_uranges<<<grid, 32, 0, st>>>(g, fg, P->slots, P->u1, kC, P->wtab, P->urange);
    PA_CUDA(cudaGetLastError());
  }
  if (P->apod) {
    unsigned long long* const cnt = P->active;
    PA_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), st));
    if (P->full) {
      const size_t per_tile = P->full_entries / P->n_tiles;
      dim3 grid((unsigned)((per_tile + 255) / 256), P->n_tiles);
      k_count_active_full<<<grid, 256, 0, st>>>(fg, P->wtab, cnt);
    } else {
      dim3 grid((d.nz + 127) / 128, d.nx);
      k_count_active<<<grid, 128, 0, st>>>(g, d.nx, d.nz, d.n_elem, P->wtab, cnt);
    }
    PA_CUDA(cudaGetLastError());
  }

  // what does not wait for the kernels, while they run
  // work items (tile, residue group) deepest tiles first; the frame is the
  // fastest index of a work item, so frames of one tile run back to back
  std::vector<int4> it((size_t)P->n_tiles * P->ngroups);
  for (int t = 0; t < P->n_tiles; ++t) {
    const int tz = P->nzt - 1 - t / P->nxt, tx = t % P->nxt;
    for (int gr = 0; gr < P->ngroups; ++gr)
      it[(size_t)t * P->ngroups + gr] = make_int4(tz * P->nxt + tx, gr, tx, tz);
  }
  std::vector<int2> srg(P->slots);
  for (int sl = 0; sl < P->slots; ++sl) srg[sl] = make_int2(sl % P->m, sl / P->m);
  PA_CUDA(cudaMemcpyAsync(P->items, it.data(), it.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
  PA_CUDA(cudaMemcpyAsync(P->slot_rg, srg.data(), srg.size() * sizeof(int2), cudaMemcpyHostToDevice,
                          st));

  // post-filter tables (host FP64 -> FP32)
  // per-pass twiddle blocks of the Stockham FFT, in the order the passes run
  std::vector<float2> tw;
  {
    int ns = 1, rem = P->log2M;
    if (post_inplace_func(P->M) && post_first_radix(P->M) == 16) {
      ns = 16;  // first pass of radix 16 (sub-transform length 1: no twiddles)
      rem -= 4;
    }
    while (rem > 0) {
      const int lr = rem >= 3 ? 3 : rem;
      const int R = 1 << lr;
      if (ns > 1)
        for (int k = 0; k < ns; ++k)
          for (int r = 1; r < R; ++r) {
            const double ang = -2.0 * M_PI * (double)r * k / (double)(ns * R);
            tw.push_back(make_float2((float)std::cos(ang), (float)std::sin(ang)));
          }
      ns *= R;
      rem -= lr;
    }
    if (tw.empty()) tw.push_back(make_float2(1.f, 0.f));
  }
  P->n_tw = (int)tw.size();
  if (post_reg_func(P->M)) {  // then the twiddles between the two levels of M = 32 L
    const int L = P->M / 32;
    tw.resize((size_t)2 * P->M);
    for (int k = 0; k < 32; ++k)
      for (int l = 0; l < L; ++l) {
        const double ang = -2.0 * M_PI * (double)k * l / P->M;
        tw.push_back(make_float2((float)std::cos(ang), (float)std::sin(ang)));
      }
  }
  std::vector<float> mk((size_t)3 * P->M, 0.f);
  const bool even_of[3] = {false, true, (P->K % 2) == 0};
  for (int o = 0; o < 3; ++o) {
    if (P->out_id[o] < 0) continue;
    if (build_mask(d, even_of[o], P->M, mk.data() + (size_t)P->out_id[o] * P->M))
      P->warnings |= 1u << P->out_id[o];
  }
  // first bin each output's mask keeps and rows of L = M / 32 bins from it on
  if (post_reg_func(P->M)) {
    const int L = P->M / 32;
    for (int o = 0; o < P->n_out; ++o) {
      int first = -1, last = -1;
      for (int b = 0; b < P->M; ++b)
        if (mk[(size_t)o * P->M + b] != 0.f) {
          if (first < 0) first = b;
          last = b;
        }
      P->band[o] = first < 0 ? make_int2(0, 0) : make_int2(first, (last - first) / L + 1);
      P->band_rows = std::max(P->band_rows, P->band[o].y);
    }
  }
  PA_CUDA(cudaMemcpyAsync(P->tw, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice, st));
  PA_CUDA(cudaMemcpyAsync(P->mask, mk.data(), mk.size() * sizeof(float), cudaMemcpyHostToDevice,
                          st));
  // post kernels: at most 200 KiB of shared memory a block
  PA_CUDA(post_configure((size_t)200 * 1024));

  int head[5] = {0, 0, 0, 0, 0};
  std::vector<int2> ur((size_t)P->n_tiles * P->slots);
  PA_CUDA(cudaMemcpyAsync(head, P->scratch[0], sizeof head, cudaMemcpyDeviceToHost, st));
  PA_CUDA(cudaMemcpyAsync(ur.data(), P->urange, ur.size() * sizeof(int2), cudaMemcpyDeviceToHost,
                          st));
  unsigned long long active = 0;
  if (P->apod) PA_CUDA(cudaMemcpyAsync(&active, P->active, sizeof active, cudaMemcpyDeviceToHost, st));
  cudaError_t se = cudaStreamSynchronize(st);
  if (se != cudaSuccess) return fail(PA_ECUDA, "plan build: %s", cudaGetErrorString(se));
  if (head[0] != 0) return fail(PA_ECUDA, "plan build: table row outside range (flag %d)", head[0]);
  const int width = head[2];
  P->window = ((std::max(width, 1) + 3) / 4) * 4;
  // samples any window holds
  P->used_lo = std::max(0, kLoBias - head[4]);
  P->used_hi = std::min(d.n_samples, head[3] - kLoBias + P->window);

  PA_CUDA(cudaMemsetAsync(P->scratch[0], 0, P->scratch_ints * sizeof(int), st));

  // TMA box geometry of one staged channel
  P->wr = ((P->window + 1 + P->lo_align - 1) / P->lo_align) * P->lo_align;
  if (P->wr > 256) P->use_tma = false;  // TMA boxes span at most 256 elements
  if (P->use_tma && !tensor_map_encoder()) P->use_tma = false;
  P->executed_pairs = 0;
  for (int t = 0; t < P->n_tiles * P->slots; ++t)
    if (ur[t].y > ur[t].x) P->executed_pairs += (int64_t)(ur[t].y - ur[t].x) * 32 * kC;
  P->steps_per_pixel = (double)P->executed_pairs / ((double)P->nx_pad * P->nz_pad);
  P->active_pairs = P->apod ? (int64_t)active : (int64_t)d.nx * d.nz * d.n_elem;
  if ((s = build_form1(P)) != PA_OK) return s;
  if ((s = build_form2(P)) != PA_OK) return s;
  if ((s = build_form3(P, 1)) != PA_OK) return s;
  if ((s = build_form3(P, 2)) != PA_OK) return s;
  if ((s = alloc_forms(P, ur, st)) != PA_OK) return s;
  PA_CUDA(cudaStreamSynchronize(st));
  return PA_OK;
}

int stage_index(uint32_t stages, uint32_t stage) { return popcount3(stages & (stage - 1u)); }

// A timing event pair from the plan's free list (created when it is empty).
bool take_events(pa_plan_s* P, std::pair<cudaEvent_t, cudaEvent_t>* ev) {
  if (!P->ev_free.empty()) {
    *ev = P->ev_free.back();
    P->ev_free.pop_back();
    return true;
  }
  *ev = {nullptr, nullptr};
  if (cudaEventCreate(&ev->first) != cudaSuccess) {
    ev->first = nullptr;
    return false;
  }
  if (cudaEventCreate(&ev->second) != cudaSuccess) {
    cudaEventDestroy(ev->first);
    *ev = {nullptr, nullptr};
    return false;
  }
  return true;
}

// The launches of one chunk of nf <= max_batch frames, in order.
struct Step {
  LaunchSpec spec;
  void* args[2] = {nullptr, nullptr};
  int begin = -1, end = -1;  // kernel kind whose timing starts / ends here
  bool chain = true;         // may follow the kernel before by a programmatic edge
};
struct ChunkLaunch {
  struct Round {
    BfParams b;
    PrepParams pp;
  };
  std::vector<Round> rounds;
  PostParams q;
  LogParams l;
  std::vector<Step> steps;
  int* zero = nullptr;  // counter + image maxima, cleared before the kernels
  int zero_ints = 0;
};

bool encode_rf_map(pa_plan_s* P, const void* rf, int nf, CUtensorMap* map) {
  const pa_plan_desc& d = P->d;
  const cuuint64_t dims[3] = {(cuuint64_t)d.n_samples, (cuuint64_t)d.n_elem, (cuuint64_t)nf};
  const cuuint64_t strides[2] = {(cuuint64_t)d.n_samples * P->elt,
                                 (cuuint64_t)d.n_samples * d.n_elem * P->elt};
  const cuuint32_t box[3] = {(cuuint32_t)P->wr, 1, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUtensorMapDataType dt =
      P->elt == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16;
  return tensor_map_encoder()(map, dt, 3, const_cast<void*>(rf), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The form a launch of nf frames runs.  The lines follow 4500 random plans (24-256
// elements, 48-1024 depth rows, 1-48 frames, every option), each form timed
// warm and with the record and tables out of L2; the figures are means of
// one-frame form time / this form's time over a class of them (with these lines
// the choice is 0.957 of the fastest form on average, and a twentieth
// slower than the one-frame form on 1.7 %).  What decides is how many work items
// of the one-frame form an SM gets (a block is an item, so few items leave SMs
// idle or one SM with twice another's work), and how that form stages its
// record: by TMA (16-bit rows on 16-byte boundaries), by vector loads, or, rows
// off 16-byte boundaries, sample by sample.
//
// One pixel a thread, up to two items an SM and 1100 warps of 4-pixel threads:
//   full table: plain sums 1.25-1.75 (orders 6-8: 1.07), Kahan sums 1.2-1.55 at
//     orders up to 5, 1.1 at 6 and 7 up to one item an SM and 0.93-0.99 beyond,
//     0.98 at 8, whose sums spill most;
//   lattice, TMA: never (0.83-1.05);
//   lattice, by samples: 1.2-1.45 up to one item an SM, with 50 steps and more
//     1.05-1.25 up to two (fewer: 0.92-1.03);
//   lattice, vector loads: 1.05-1.1 up to half an item an SM, with 50 steps and
//     more 1.1-1.3 up to one and 1.03-1.2 up to two (fewer: 0.95-1.02); orders 1
//     and 2 1.15 with 50 steps up to half an item, about 1 elsewhere.
//   Fewer than 28 steps do not repay the preparation pass (0.84-1.05).
// Two pixels a thread, plain sums from 50 steps and from two items an SM on, up
// to 2400 warps (at fewer items one pixel is the better one; Kahan sums, TMA and
// vector loads 0.8-1.05):
//   full table, orders up to 5: 1.1-1.5;
//   lattice, by samples: order 3 1.2-1.25 up to four items an SM, 4 and 5
//     1.08-1.13 up to three, 0.95-1.05 elsewhere.
bool fine_pays(const pa_plan_s* P, int px, int nf) {
  const FineLimits lim = fine_limits(P);
  if (frame_warps(P) * nf > (px == 1 ? lim.px1 : lim.px2)) return false;
  if (P->item_frames != 0) return true;
  const double per_sm = (double)P->n_tiles * P->ngroups * nf / P->num_sms;
  if (px == 2) return per_sm > 2 && (P->full || per_sm <= (P->K == 3 ? 4 : 3));
  if (P->full) return per_sm <= (!P->comp || P->K <= 5 ? 2 : 1);
  if (!staged_by_samples(P) && P->K <= 2) return per_sm <= 0.5;
  return per_sm <= (fine_steps(P) >= 50 ? 2 : staged_by_samples(P) ? 1 : 0.5);
}

// Two frames an item (orders up to 5).  An item does twice the work, so the line
// is the number of pairs of items an SM gets, from which the time saved per
// item exceeds the coarser end of the launch:
//   full table 1.25-1.35: plain sums of orders up to 3 at any number, Kahan sums
//     of orders 1 and 2 from 1.5, the others from 3 (0.7-1.0 below);
//   lattice, by samples, from 2.5: 1.15-1.2 (0.75-1.05 below; at order 3, plain,
//     1.05 from 1.5 on);
//   lattice, vector loads, from 3, orders 1 and 2 from 4: 1.08-1.2 (0.8-0.95);
//   lattice, TMA, from 4.5: 1.0-1.13; Kahan sums of orders 1 and 2 and
//     apodised ones from 2.5: 1.06 (0.75-0.9 below either).
// An odd launch's last item does a frame's work twice: 3 and 5 frames 0.85-1.0
// but where the record is staged by samples, from three pairs an SM on; 7 and
// more as even launches.  And where rows come by TMA or vector loads, or the
// full table's plain sums are of orders 4 and 5, their samples have to serve
// pairs enough (build_form2: 0.85-1.0 otherwise).
bool pairs_pay(const pa_plan_s* P, int nf) {
  const double per_sm = (double)P->n_tiles * P->ngroups * ((nf + 1) / 2) / P->num_sms;
  const bool by_samples = !P->full && staged_by_samples(P);
  if (nf % 2 != 0 && nf < 7 && !(by_samples && per_sm >= 3)) return false;
  if (P->full && P->comp) return per_sm >= (P->K <= 2 ? 1.5 : 3);
  if (P->full && P->K <= 3) return true;
  if (by_samples) return per_sm >= 2.5;
  if (!P->pairs_pay) return false;
  if (P->full) return per_sm >= 3;
  if (!P->use_tma) return per_sm >= (P->K <= 2 ? 4 : 3);
  return per_sm >= (P->comp && (P->K <= 2 || P->apod) ? 2.5 : 4.5);
}

const FusedForm& pick_form(const pa_plan_s* P, int nf) {
  for (int px = 1; px <= 2; ++px) {
    const FusedForm& f = P->form[px + 1];
    if (f.nf && nf <= f.max_frames && fine_pays(P, px, nf)) return f;
  }
  const FusedForm& two = P->form[1];
  if (two.nf && nf >= 2 && (P->item_frames == 2 || pairs_pay(P, nf))) return two;
  return P->form[0];
}

// Amplitude sums below this take the two-float e_k (df_in_range says why).
float ek_top(int k, int n_elem) {
  return (float)std::min(std::ldexp(1.0, 40), std::ldexp(1.0, 120) / std::pow((double)n_elem, k - 1));
}

// Launch parameters of one round of the fused kernel in form f: nf frames
// from frame f0 of the chunk on.
pa_status fused_params(pa_plan_s* P, const FusedForm& f, const void* rf, int nf, float* out,
                       uint32_t stages, int* scratch, BfParams* bp) {
  const pa_plan_desc& d = P->d;
  const int planes = popcount3(stages) * P->n_out;
  const uint32_t raw_stage =
      (stages & PA_STAGE_RAW) ? PA_STAGE_RAW : ((stages & PA_STAGE_ENV) ? PA_STAGE_ENV : PA_STAGE_LOG);
  const int s_raw = stage_index(stages, raw_stage);

  BfParams& b = *bp;
  memset(&b.tmap, 0, sizeof b.tmap);
  b.use_tma = !f.slots && P->use_tma ? 1 : 0;
  b.wr = P->wr;
  b.rp = f.rp;
  b.nc = f.nc;
  b.ncs = f.nc + kC - 1;
  b.tmem_cols = f.tmem_cols;
  b.chunk_bytes = f.slots ? b.ncs * P->window * f.slot_bytes : b.ncs * P->wr * (int)P->elt;
  b.pairs_off = f.pairs_off;
  if (b.use_tma && !encode_rf_map(P, rf, nf, &b.tmap))
    return fail(PA_ECUDA, "cuTensorMapEncodeTiled rejected the RF layout");
  b.rf = rf;
  b.rf_dtype = (int)d.rf_dtype;
  b.vec_ok = (d.n_samples % 4) == 0;
  b.nearest = d.interp == PA_INTERP_NEAREST;
  b.lane_rows_log2 = P->lane_rows_log2;
  b.n_elem = d.n_elem;
  b.n_samples = d.n_samples;
  b.frame_elems = (long long)d.n_elem * d.n_samples;
  b.table = P->table;
  b.ftab = P->ftab;
  b.full = P->full ? 1 : 0;
  b.steps = P->u1 - P->u0;
  b.wtab = P->wtab;
  b.tgroups = P->tgroups;
  b.nz_pad = P->nz_pad;
  b.items = P->items;
  b.slot_rg = P->slot_rg;
  b.dmin = P->dmin;
  b.m = P->m;
  b.R = P->R;
  b.nxt = P->nxt;
  b.nzt = P->nzt;
  b.tile_x = P->tile_x;
  b.tile_z = P->tile_z;
  b.warps = P->warps;
  b.slots = P->slots;
  b.ngroups = P->ngroups;
  b.nv = P->nv;
  b.u0 = P->u0;
  b.window = P->window;
  b.w4_inv = (int)(((1u << 20) + (unsigned)(P->window / 4) - 1) / (unsigned)(P->window / 4));
  b.lo = P->lo;
  b.urange = P->urange;
  b.vchunks = f.vchunks;
  b.out = out;
  b.planes = planes;
  b.plane_das = P->out_id[0] >= 0 ? s_raw * P->n_out + P->out_id[0] : -1;
  b.plane_dmas = P->out_id[1] >= 0 ? s_raw * P->n_out + P->out_id[1] : -1;
  b.plane_ho = P->out_id[2] >= 0 ? s_raw * P->n_out + P->out_id[2] : -1;
  b.nx = d.nx;
  b.nz = d.nz;
  b.ek_top = ek_top(P->K, d.n_elem);
  b.n_frames = nf;
  b.n_fgroups = (nf + f.nf - 1) / f.nf;
  b.splits = f.splits;
  b.n_items = P->n_tiles * (f.slots && f.nf == 1 ? f.splits : P->ngroups) * b.n_fgroups;
  b.counter = scratch + 1;
  b.err = scratch;
  b.timeouts = scratch + P->scratch_ints - 1;
  b.host_flag = P->host_flag;
  b.expect_extra = P->expect_extra;
  b.stages = f.stages;
  b.slots_dev = f.slots;
  b.slot_pitch = P->slot_pitch;
  b.slot_margin = P->slot_margin;
  return PA_OK;
}

pa_status prepare_chunk(pa_plan_s* P, const void* rf, int nf, float* out, uint32_t stages,
                        int* scratch, ChunkLaunch* c) {
  const pa_plan_desc& d = P->d;
  const int n_st = popcount3(stages);
  const int planes = n_st * P->n_out;
  const uint32_t raw_stage =
      (stages & PA_STAGE_RAW) ? PA_STAGE_RAW : ((stages & PA_STAGE_ENV) ? PA_STAGE_ENV : PA_STAGE_LOG);
  const uint32_t env_stage = (stages & PA_STAGE_ENV) ? PA_STAGE_ENV : PA_STAGE_LOG;
  const int s_raw = stage_index(stages, raw_stage);
  const int s_env = stage_index(stages, env_stage);
  c->zero = scratch + 1;
  c->zero_ints = 1 + nf * P->n_out;

  const FusedForm& f = pick_form(P, nf);
  const int per_round = f.slots ? f.max_frames : nf;
  const int n_rounds = (nf + per_round - 1) / per_round;
  c->rounds.resize(n_rounds);
  c->steps.clear();
  c->steps.reserve(2 * n_rounds + 2);
  if (!f.slots) {
    Step z;
    z.spec.func = reinterpret_cast<const void*>(k_zero_ints);
    z.spec.grid = dim3(1);
    z.spec.block = dim3(256);
    z.args[0] = &c->zero;
    z.args[1] = &c->zero_ints;
    c->steps.push_back(z);
  }
  for (int r = 0; r < n_rounds; ++r) {
    ChunkLaunch::Round& rd = c->rounds[r];
    const int f0 = r * per_round, n = std::min(per_round, nf - f0);
    const char* rf_r = (const char*)rf + (size_t)f0 * d.n_elem * d.n_samples * P->elt;
    const pa_status s = fused_params(P, f, rf_r, n, out + (size_t)f0 * planes * d.nx * d.nz, stages,
                                     scratch, &rd.b);
    if (s != PA_OK) return s;
    Step sb;
    sb.spec.func = f.func;
    sb.spec.grid = dim3(std::max(1, std::min(rd.b.n_items, f.blocks_per_sm * P->num_sms)));
    sb.spec.block = dim3(f.threads);
    sb.spec.smem = f.smem;
    if (f.slots) {
      PrepParams& pp = rd.pp;
      pp.rf = rf_r;
      pp.slots = f.slots;
      pp.nf = f.nf;
      pp.pitch = P->slot_pitch;
      pp.margin = P->slot_margin;
      pp.rf_dtype = (int)d.rf_dtype;
      pp.n_elem = d.n_elem;
      pp.n_samples = d.n_samples;
      pp.n_frames = n;
      pp.n_lo = P->used_lo;
      pp.n_hi = P->used_hi;
      pp.mode = P->slot_mode;
      pp.order = P->K;
      pp.zero = c->zero;
      pp.n_zero = r == 0 ? c->zero_ints : 1;  // later rounds: the work counter only
      pp.counter0 = (int)sb.spec.grid.x;
      Step sp;
      prep_spec(&pp, &sp.spec);
      sp.args[0] = &pp;
      sp.begin = 0;
      c->steps.push_back(sp);
    }
    sb.args[0] = &rd.b;
    // The kernel before lets its successor come up from its start on, and blocks
    // that are placed while it still runs are not spread evenly.  So a fused
    // kernel has a plain edge unless it has more items than resident blocks, or
    // Kahan sums in the two-frame form (whose blocks allocate tensor memory
    // first).  Measured: after the clearing kernel on buffers other than the last
    // call's, one frame of 512 x 512 41.3 -> 47.8 us, of 880 x 435 70 -> 98 (plain
    // edge 41.3 and 70 on any buffers); fine-grained, one frame of 492 x 62 29.1,
    // plain 21.0, one of 572 x 125 with Kahan sums 39.4, plain 29.3; two frames of
    // 292 x 765 at order 4 74.5, plain 64.3; but six BF16 frames of 256 x 256 with
    // Kahan sums 39.3, plain 41.3.
    sb.chain = f.nf == 2 && (P->comp || rd.b.n_items > (int)sb.spec.grid.x);
    sb.begin = f.slots ? -1 : 0;
    sb.end = 0;
    c->steps.push_back(sb);
  }

  const bool post = (stages & (PA_STAGE_ENV | PA_STAGE_LOG)) != 0;
  const bool log = (stages & PA_STAGE_LOG) != 0;
  PostParams& q = c->q;
  q.out = out;
  q.planes = planes;
  q.n_out = P->n_out;
  q.s_src = s_raw;
  q.s_dst = s_env;
  q.nx = d.nx;
  q.nz = d.nz;
  q.m = P->M;
  q.log2m = P->log2M;
  q.tw = P->tw;
  q.tw_reg = P->tw + (size_t)2 * P->M;
  q.n_tw = P->n_tw;
  q.mask = P->mask;
  for (int o = 0; o < 3; ++o) q.band[o] = P->band[o];
  q.band_rows = P->band_rows;
  q.maxslot = scratch + 2;
  q.n_frames = nf;
  q.warps_per_block = P->post_wpb;
  if (post) {
    Step t;
    post_spec(q, &t.spec);
    // Few blocks, placed while the fused kernel's are leaving, share SMs that
    // need not be shared (24 blocks of one 128 x 128 frame: call 20.6 -> 22 us).
    t.chain = (long long)t.spec.grid.x * t.spec.grid.y * t.spec.grid.z >= P->num_sms;
    t.args[0] = &c->q;
    t.begin = t.end = 1;
    c->steps.push_back(t);
  }
  LogParams& l = c->l;
  l.out = out;
  l.planes = planes;
  l.n_out = P->n_out;
  l.s_src = s_env;
  l.s_dst = stage_index(stages, PA_STAGE_LOG);
  l.plane_elems = (long long)d.nx * d.nz;
  l.maxslot = scratch + 2;
  l.dyn_range_db = P->dyn_range;
  l.n_frames = nf;
  if (log) {
    Step t;
    log_spec(l, P->num_sms, &t.spec);
    t.args[0] = &c->l;
    t.begin = t.end = 2;
    c->steps.push_back(t);
  }
  return PA_OK;
}

pa_status launch_direct(pa_plan_s* P, ChunkLaunch& c, cudaStream_t st) {
  std::pair<cudaEvent_t, cudaEvent_t> ev{nullptr, nullptr};
  for (Step& t : c.steps) {
    if (t.begin >= 0 && (P->prof >> t.begin & 1u) && take_events(P, &ev))
      cudaEventRecord(ev.first, st);
    const cudaError_t e =
        cudaLaunchKernel(t.spec.func, t.spec.grid, t.spec.block, t.args, t.spec.smem, st);
    if (ev.first && (t.end >= 0 || e != cudaSuccess)) {
      cudaEventRecord(ev.second, st);
      if (t.end >= 0) P->ev_used.push_back({t.end, ev});
      else P->ev_free.push_back(ev);
      ev = {nullptr, nullptr};
    }
    if (e != cudaSuccess) return fail(PA_ECUDA, "kernel launch: %s", cudaGetErrorString(e));
  }
  return PA_OK;
}

cudaKernelNodeParams node_params(Step& t) {
  cudaKernelNodeParams k{};
  k.func = const_cast<void*>(t.spec.func);
  k.gridDim = t.spec.grid;
  k.blockDim = t.spec.block;
  k.sharedMemBytes = (unsigned)t.spec.smem;
  k.kernelParams = t.args;
  k.extra = nullptr;
  return k;
}

// Adds kernel t after n_deps nodes, or, chained, after the kernel node deps[0]
// with a programmatic edge (wait_previous).
cudaError_t add_kernel_node(cudaGraph_t graph, Step& t, const cudaGraphNode_t* deps, int n_deps,
                            bool chained, cudaGraphNode_t* n) {
  const cudaKernelNodeParams kp = node_params(t);
  if (!chained || !t.chain)
    return cudaGraphAddKernelNode(n, graph, n_deps ? deps : nullptr, n_deps, &kp);
  cudaError_t e = cudaGraphAddKernelNode(n, graph, nullptr, 0, &kp);
  if (e != cudaSuccess) return e;
  cudaGraphEdgeData edge{};
  edge.from_port = cudaGraphKernelNodePortProgrammatic;
  edge.type = cudaGraphDependencyTypeProgrammatic;
  return cudaGraphAddDependencies(graph, deps, n, &edge, 1);
}

// One chunk as a CUDA graph: the chunk's launches in a row.  An executable
// graph is kept per (frames, stages, timing); later calls only rewrite the
// node parameters (buffer pointers, and the timing events) and launch it.
// While timing is on, each timed kernel sits between two event-record nodes,
// so the kernels are timed on the path that serves.
pa_status launch_graph(pa_plan_s* P, ChunkLaunch& c, int nf, uint32_t stages, cudaStream_t st) {
  const uint32_t prof = P->prof;
  pa_plan_s::GraphEntry* ge = nullptr;
  for (auto& g : P->graphs)
    if (g.nf == nf && g.stages == stages && g.prof == prof) ge = &g;
  std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> ev;  // in step order
  auto give_back = [&]() {
    for (auto& e : ev) P->ev_free.push_back(e.second);
  };
  if (prof) {
    for (const Step& t : c.steps) {
      if (t.begin < 0 || !(prof >> t.begin & 1u)) continue;
      std::pair<cudaEvent_t, cudaEvent_t> e;
      if (!take_events(P, &e)) {
        give_back();
        return fail(PA_ECUDA, "timing events: out of resources");
      }
      ev.push_back({t.begin, e});
    }
  }
  if (!ge) {
    // bounded cache: drop the oldest graph once 32 shapes are held (callers
    // that vary the batch size every call would otherwise grow it forever)
    if (P->graphs.size() >= 32) {
      cudaGraphExecDestroy(P->graphs.front().exec);
      cudaGraphDestroy(P->graphs.front().graph);
      P->graphs.erase(P->graphs.begin());
    }
    pa_plan_s::GraphEntry g;
    g.nf = nf;
    g.stages = stages;
    g.prof = prof;
    cudaGraph_t graph;
    cudaError_t e = cudaGraphCreate(&graph, 0);
    if (e != cudaSuccess) {
      give_back();
      return fail(PA_ECUDA, "graph build: %s", cudaGetErrorString(e));
    }
    cudaGraphNode_t prev = nullptr;
    bool chained = false;  // prev is a kernel
    size_t next_ev = 0;
    for (Step& t : c.steps) {
      if (t.begin >= 0 && (prof >> t.begin & 1u)) {
        cudaGraphNode_t n = nullptr;
        e = cudaGraphAddEventRecordNode(&n, graph, prev ? &prev : nullptr, prev ? 1 : 0,
                                        ev[next_ev].second.first);
        if (e != cudaSuccess) break;
        g.events.push_back(n);
        prev = n;
        chained = false;
      }
      cudaGraphNode_t n = nullptr;
      e = add_kernel_node(graph, t, &prev, prev ? 1 : 0, chained, &n);
      if (e != cudaSuccess) break;
      g.kernels.push_back(n);
      prev = n;
      chained = true;
      if (t.end >= 0 && (prof >> t.end & 1u)) {
        cudaGraphNode_t m = nullptr;
        e = cudaGraphAddEventRecordNode(&m, graph, &prev, 1, ev[next_ev++].second.second);
        if (e != cudaSuccess) break;
        g.events.push_back(m);
        prev = m;
        chained = false;
      }
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&g.exec, graph, 0);
    if (e != cudaSuccess) {
      cudaGraphDestroy(graph);
      give_back();
      return fail(PA_ECUDA, "graph build: %s", cudaGetErrorString(e));
    }
    g.graph = graph;
    ++P->graph_builds;
    P->graphs.push_back(std::move(g));
    ge = &P->graphs.back();
  } else {
    cudaError_t e = cudaSuccess;
    for (size_t i = 0; i < c.steps.size() && e == cudaSuccess; ++i) {
      const cudaKernelNodeParams kp = node_params(c.steps[i]);
      e = cudaGraphExecKernelNodeSetParams(ge->exec, ge->kernels[i], &kp);
    }
    for (size_t i = 0; i < ev.size() && e == cudaSuccess; ++i) {
      e = cudaGraphExecEventRecordNodeSetEvent(ge->exec, ge->events[2 * i], ev[i].second.first);
      if (e == cudaSuccess)
        e = cudaGraphExecEventRecordNodeSetEvent(ge->exec, ge->events[2 * i + 1],
                                                 ev[i].second.second);
    }
    if (e != cudaSuccess) {
      give_back();
      return fail(PA_ECUDA, "graph update: %s", cudaGetErrorString(e));
    }
  }
  const cudaError_t e = cudaGraphLaunch(ge->exec, st);
  if (e != cudaSuccess) {
    give_back();
    return fail(PA_ECUDA, "graph launch: %s", cudaGetErrorString(e));
  }
  for (auto& x : ev) P->ev_used.push_back(x);
  return PA_OK;
}

pa_status run_chunk(pa_plan_s* P, const void* rf, int nf, float* out, uint32_t stages,
                    cudaStream_t st, int* scratch) {
  ChunkLaunch c;
  pa_status ps = prepare_chunk(P, rf, nf, out, stages, scratch, &c);
  if (ps != PA_OK) return ps;
  if (P->use_graph) return launch_graph(P, c, nf, stages, st);
  return launch_direct(P, c, st);
}

// Tapered schedule: short first and last chunks (the first upload and the
// last download overlap no compute), evenly sized middle chunks, none above
// cap frames.
std::vector<int32_t> taper_schedule(int n, int cap) {
  std::vector<int32_t> sched;
  const int edge = std::min(cap, std::max(1, n / 5));
  const int mid = n - 2 * edge;
  if (mid < 0) {  // one or two frames
    for (int f = 0; f < n; ++f) sched.push_back(1);
    return sched;
  }
  sched.push_back(edge);
  const int nm = mid == 0 ? 0 : std::max(2, (mid + cap - 1) / cap);
  for (int q = 0; q < nm; ++q) {
    const int c = (mid * (q + 1)) / nm - (mid * q) / nm;
    if (c > 0) sched.push_back(c);
  }
  sched.push_back(edge);
  return sched;
}

// Host-path link rate assumed by the candidate schedules: about 200 GB/s each
// way between pinned Grace memory and the GPU (measured 206 GB/s up, 192 GB/s
// down on GB300).
constexpr double kLinkBytesPerUs = 2.0e5;

// The tuning state of one (frames, stages) shape, created on first use with
// its candidates: the tapered schedule and the pipeline model's best
// schedules for kernel times of 0.6x to 2.8x the per-frame copy time,
// per-chunk launch costs of 8 and 40 us and wave shares of 0 and 1.  None of
// these is known in advance (measured on GB300: 38 us per chunk and no wave
// effect for 512 x 512 images at k = 3; about 50 us and a full wave effect
// at 1024 x 1024, k = 4); the tuning calls measure the outcome.
pa_plan_s::HostTune* host_tune(pa_plan_s* P, int nf, uint32_t stages) {
  for (auto& t : P->tunes)
    if (t.nf == nf && t.stages == stages) return &t;
  if (P->tunes.size() >= 32) P->tunes.erase(P->tunes.begin());  // bounded, oldest first
  pa_plan_s::HostTune t;
  t.nf = nf;
  t.stages = stages;
  const int cap = std::max(1, P->d.max_batch);
  auto add = [&t](std::vector<int32_t> c) {
    if (!c.empty() && std::find(t.cand.begin(), t.cand.end(), c) == t.cand.end())
      t.cand.push_back(std::move(c));
  };
  add(taper_schedule(nf, cap));
  if (nf > 2) {
    pa_pipe_model m{};
    m.items_per_frame = std::max(1, P->n_tiles * P->ngroups);
    m.resident = std::max(1, P->form[0].blocks_per_sm * P->num_sms);
    m.n_sets = kHostSets;
    const double rf_frame = (double)P->d.n_elem * P->d.n_samples * P->elt;
    const double out_frame = (double)popcount3(stages) * P->n_out * P->d.nx * P->d.nz * 4.0;
    m.upload_us = rf_frame / kLinkBytesPerUs;
    m.download_us = out_frame / kLinkBytesPerUs;
    const double copy_us = std::max(m.upload_us, m.download_us);
    for (double x : {0.6, 0.9, 1.3, 1.9, 2.8})
      for (double launch : {8.0, 40.0})
        for (double q : {0.0, 1.0}) {
          m.kernel_us = x * copy_us;
          m.launch_us = launch;
          m.wave_share = q;
          add(pipe_search(m, nf, cap));
        }
  }
  t.best_ms.assign(t.cand.size(), -1.0);
  for (int i = 0; i < (int)t.cand.size(); ++i) t.order.push_back(i);
  if (t.cand.size() == 1) t.chosen = 0;
  P->tunes.push_back(std::move(t));
  return &P->tunes.back();
}

// One tuning call of candidate `cur` took `ms`.  A cold call (it built a
// graph or grew the staging buffers) is not counted unless the candidate was
// cold three times in a row.
void host_tune_record(pa_plan_s::HostTune* t, int cur, double ms, bool cold) {
  if (cold && ++t->attempts < 3) return;
  t->attempts = 0;
  double& b = t->best_ms[cur];
  b = b < 0 ? ms : std::min(b, ms);
  if (++t->pos < t->order.size()) return;
  if (!t->second_round) {  // time the three fastest once more
    t->second_round = true;
    std::vector<int> idx(t->cand.size());
    for (int i = 0; i < (int)idx.size(); ++i) idx[i] = i;
    std::stable_sort(idx.begin(), idx.end(),
                     [t](int a, int c) { return t->best_ms[a] < t->best_ms[c]; });
    for (int i = 0; i < std::min<int>(3, (int)idx.size()); ++i) t->order.push_back(idx[i]);
    return;
  }
  t->chosen = (int)(std::min_element(t->best_ms.begin(), t->best_ms.end()) - t->best_ms.begin());
}

bool is_pinned(const void* p) {
  cudaPointerAttributes a{};
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeHost;
}

// The graph of one host-path call: per chunk c (buffer set b = c mod sets)
// an upload, the launch sequence (clear, fused kernel, post, log) and a
// download, with the ordering of the stream form: a launch sequence after
// its upload and after the previous chunk's launch sequence, a download
// after its launch sequence, an upload into set b after the download that
// last used set b.
pa_status build_host_graph(pa_plan_s* P, pa_plan_s::HostGraph& hg, const void* rf_host,
                           float* out_host, int chunk, int nsets) {
  const pa_plan_desc& d = P->d;
  const size_t rf_frame = (size_t)d.n_elem * d.n_samples * P->elt;
  const size_t out_frame = (size_t)popcount3(hg.stages) * P->n_out * d.nx * d.nz;
  cudaGraph_t graph;
  PA_CUDA(cudaGraphCreate(&graph, 0));
  cudaError_t e = cudaSuccess;
  cudaGraphNode_t prev_last = nullptr;
  int f0 = 0;
  for (size_t c = 0; c < hg.sched.size() && e == cudaSuccess; ++c) {
    const int nf = hg.sched[c];
    const int b = (int)(c % nsets);
    char* rf_d = (char*)P->h_rf + (size_t)b * chunk * rf_frame;
    float* out_d = P->h_out + (size_t)b * chunk * out_frame;
    const size_t up_off = (size_t)f0 * rf_frame, up_bytes = nf * rf_frame;  // bytes
    const size_t down_off = (size_t)f0 * out_frame;                          // floats
    const size_t down_bytes = nf * out_frame * sizeof(float);
    cudaGraphNode_t up = nullptr, down = nullptr;
    {
      cudaGraphNode_t dep = c >= (size_t)nsets ? hg.down[c - nsets] : nullptr;
      e = cudaGraphAddMemcpyNode1D(&up, graph, dep ? &dep : nullptr, dep ? 1 : 0, rf_d,
                                   (const char*)rf_host + up_off, up_bytes, cudaMemcpyHostToDevice);
    }
    ChunkLaunch cl;
    if (e == cudaSuccess) {
      const pa_status ps = prepare_chunk(P, rf_d, nf, out_d, hg.stages, P->scratch[b], &cl);
      if (ps != PA_OK) {
        cudaGraphDestroy(graph);
        return ps;
      }
    }
    cudaGraphNode_t last = nullptr;
    if (e == cudaSuccess) {
      cudaGraphNode_t deps[2] = {up, prev_last};
      int n_deps = prev_last ? 2 : 1;
      for (Step& t : cl.steps) {
        cudaGraphNode_t n = nullptr;
        // plain edges: next to copy nodes, programmatic ones held the chunks'
        // copies back (two frames of 53 channels, k = 5: 71.7 -> 82.2 us a call)
        e = add_kernel_node(graph, t, deps, n_deps, false, &n);
        if (e != cudaSuccess) break;
        last = deps[0] = n;
        n_deps = 1;
      }
    }
    if (e == cudaSuccess)
      e = cudaGraphAddMemcpyNode1D(&down, graph, &last, 1, out_host + down_off, out_d, down_bytes,
                                   cudaMemcpyDeviceToHost);
    hg.up.push_back(up);
    hg.down.push_back(down);
    hg.up_dev.push_back(rf_d);
    hg.down_dev.push_back(out_d);
    hg.up_off.push_back(up_off);
    hg.down_off.push_back(down_off);
    hg.up_bytes.push_back(up_bytes);
    hg.down_bytes.push_back(down_bytes);
    prev_last = last;
    f0 += nf;
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&hg.exec, graph, 0);
  if (e != cudaSuccess) {
    cudaGraphDestroy(graph);
    return fail(PA_ECUDA, "host-path graph build: %s", cudaGetErrorString(e));
  }
  hg.graph = graph;
  hg.rf_host = rf_host;
  hg.out_host = out_host;
  ++P->graph_builds;
  return PA_OK;
}

// End of a host-path call: the tuning record, then the bounded waits that
// ran out during the call (the kernel stopped early).
pa_status host_call_done(pa_plan_s* P, pa_plan_s::HostTune* tune, bool tuning, int cur,
                         std::chrono::steady_clock::time_point t_start, bool cold) {
  if (tuning)
    host_tune_record(tune, cur,
                     std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() -
                                                               t_start).count(),
                     cold);
  // (the counts are read only after some wait has run out: a blocking copy a
  // buffer set costs about 10 us; an earlier launch of the plan may have run
  // out before the word existed, so it starts out set)
  if (P->host_flag && *reinterpret_cast<volatile int*>(P->host_flag)) {
    *reinterpret_cast<volatile int*>(P->host_flag) = 0;
    long long total = 0;
    for (int b = 0; b < kHostSets; ++b) {
      if (!P->scratch[b]) continue;
      int n = 0;
      PA_CUDA(cudaMemcpy(&n, P->scratch[b] + P->scratch_ints - 1, sizeof n, cudaMemcpyDeviceToHost));
      total += n;
    }
    if (total > P->timeouts_seen) {
      const long long fresh = total - P->timeouts_seen;
      P->timeouts_seen = total;
      return fail(PA_ETIMEOUT, "%lld thread block(s) gave up waiting for their RF staging copies",
                  fresh);
    }
  }
  return PA_OK;
}

}  // namespace

// ------------------------------------------------------------ dispatchers
namespace pa {
void set_error_message(const char* msg) { g_err = msg ? msg : ""; }

int* plan_timeout_counter(pa_plan_s* P) {
  return P && P->scratch[0] ? P->scratch[0] + P->scratch_ints - 1 : nullptr;
}

size_t plan_device_bytes(const pa_plan_s* P) { return P ? P->device_bytes : 0; }

size_t plan_slot_bytes(const pa_plan_s* P) { return P ? P->slot_mem_bytes : 0; }

pa_status plan_create(const pa_plan_desc* desc, cudaStream_t st, size_t slot_limit, pa_plan_s** out) {
  *out = nullptr;
  pa_status s = validate(desc);
  if (s != PA_OK) return s;
  pa_plan_s* P = new (std::nothrow) pa_plan_s();
  if (!P) return fail(PA_ENOMEM, "host allocation failed");
  P->d = *desc;
  P->slot_limit = slot_limit;
  configure(P);
  s = build_plan(P, st);
  if (s != PA_OK) {
    const std::string keep = g_err;
    free_plan(P);
    g_err = keep;
    return s;
  }
  *out = P;
  return PA_OK;
}

pa_status plan_drop_slots(pa_plan_s* P) {
  if (!P->slot_mem) return PA_OK;
  for (int i = 1; i < 4; ++i) P->form[i] = FusedForm();
  return drop_slot_memory(P);
}

pa_status plan_memory(const pa_plan_desc* desc, size_t* bytes, size_t* slots) {
  pa_status s = validate(desc);
  if (s != PA_OK) return s;
  pa_plan_s P;
  P.d = *desc;
  configure(&P);
  if ((s = check_table_size(&P)) != PA_OK) return s;
  *bytes = plan_arena(&P, nullptr);
  // bounds, before the tables say which forms pay: the two-frame form at the
  // largest launch, the fine-grained ones at the most frames they are built for
  *slots = 0;
  int frames = 0;
  if (desc->max_batch > 1 && P.K <= 5 && slot_item_bytes(&P, 1) <= kSlotBytesMax)
    *slots += round256(slots_size(&P, 1, &frames));
  const FineLimits lim = fine_limits(&P);
  const int64_t nf = std::min<int64_t>(desc->max_batch, std::max(lim.px1, lim.px2) / frame_warps(&P));
  if (slot_item_bytes(&P, 2) <= kSlotBytesMax)
    *slots += round256(std::min(kSlotBytesMax, (size_t)nf * slot_item_bytes(&P, 2)) + slot_row_bytes(&P, 2));
  return PA_OK;
}

pa_status plan_bf_params(pa_plan_s* P, const void* rf, int nf, float* out, uint32_t stages,
                         BfParams* b, int* k, bool* lattice_fp32_plain) {
  const pa_status s = fused_params(P, P->form[0], rf, nf, out, stages, P->scratch[0], b);
  if (s != PA_OK) return s;
  *k = P->K;
  *lattice_fp32_plain = !P->full && !P->apod && !P->comp && P->d.rf_dtype == PA_RF_F32 &&
                        P->d.interp == PA_INTERP_LINEAR;
  return PA_OK;
}

// A compensated plan's fused-kernel blocks hold tmem_cols TMEM columns each.
// Whatever blocks share an SM, their registers add up to at most the SM's
// register file, so if every block's columns are within its register share
// of the SM's 512 columns (cols * regs_sm <= 512 * regs_block), blocks of
// any mix of such kernels never ask for more TMEM than the SM has.  A plan
// outside that bound (blocks of 3 or fewer warps) is TMEM-dense: its blocks
// can fill an SM's TMEM while registers remain, so a block of another
// compensated kernel landing there would wait in tcgen05.alloc.
void plan_tmem(const pa_plan_s* P, int* cols, bool* dense) {
  *cols = P ? P->form[0].tmem_cols : 0;
  *dense = P && form_dense(P, P->form[0]);  // the two-frame form is never dense (build_form2)
}

const void* bf_func(int order, bool apod, bool comp, bool full) {
  switch (order) {
    case 1: return bf_func_k1(apod, comp, full);
    case 2: return bf_func_k2(apod, comp, full);
    case 3: return bf_func_k3(apod, comp, full);
    case 4: return bf_func_k4(apod, comp, full);
    case 5: return bf_func_k5(apod, comp, full);
    case 6: return bf_func_k6(apod, comp, full);
    case 7: return bf_func_k7(apod, comp, full);
    case 8: return bf_func_k8(apod, comp, full);
  }
  return nullptr;
}
const void* bf_pipe_func(int order, bool apod, bool comp, bool full, bool nearest) {
  switch (order) {
    case 1: return bf_pipe_func_k1(apod, comp, full, nearest);
    case 2: return bf_pipe_func_k2(apod, comp, full, nearest);
    case 3: return bf_pipe_func_k3(apod, comp, full, nearest);
    case 4: return bf_pipe_func_k4(apod, comp, full, nearest);
    case 5: return bf_pipe_func_k5(apod, comp, full, nearest);
  }
  return nullptr;
}
const void* bf_fine_func(int order, bool apod, bool comp, bool full, int px) {
  switch (order) {
    case 1: return bf_fine_func_k1(apod, comp, full, px);
    case 2: return bf_fine_func_k2(apod, comp, full, px);
    case 3: return bf_fine_func_k3(apod, comp, full, px);
    case 4: return bf_fine_func_k4(apod, comp, full, px);
    case 5: return bf_fine_func_k5(apod, comp, full, px);
    case 6: return bf_fine_func_k6(apod, comp, full, px);
    case 7: return bf_fine_func_k7(apod, comp, full, px);
    case 8: return bf_fine_func_k8(apod, comp, full, px);
  }
  return nullptr;
}
cudaError_t bf_occupancy(const void* func, int block, size_t smem, int* n) {
  cudaError_t e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, func, block, smem);
}
}  // namespace pa

// ------------------------------------------------------------------ C ABI
extern "C" {

pa_status pa_plan(const pa_plan_desc* desc, void* cuda_stream, pa_plan_t* out) {
  if (!out) return fail(PA_EINVAL, "null output handle");
  return plan_create(desc, (cudaStream_t)cuda_stream, kNoSlotLimit, out);
}

pa_status pa_plan_footprint(const pa_plan_desc* desc, int32_t n_frames, size_t* bytes) {
  if (!bytes) return fail(PA_EINVAL, "null bytes pointer");
  if (n_frames < 0) return fail(PA_EINVAL, "n_frames < 0");
  size_t b = 0, slots = 0;
  if (const pa_status s = plan_memory(desc, &b, &slots)) return s;
  const size_t elt = desc->rf_dtype == PA_RF_F32 ? 4 : 2;
  b += (size_t)n_frames * desc->n_elem * desc->n_samples * elt;
  b += (size_t)n_frames * 3 * popcount3(desc->outputs) * desc->nx * desc->nz * sizeof(float);
  *bytes = b;
  return PA_OK;
}

pa_status pa_plan_get_info(pa_plan_t P, pa_plan_info* info) {
  if (!P || !info) return fail(PA_EINVAL, "null argument");
  info->lattice_m = P->full ? 0 : P->m;
  info->tile_x = P->tile_x;
  info->tile_z = P->tile_z;
  info->window = P->window;
  info->n_tiles = P->n_tiles;
  info->threads = P->threads;
  info->blocks_per_sm = P->form[0].blocks_per_sm;
  info->fft_size = P->M;
  info->n_outputs = P->n_out;
  info->warnings = P->warnings;
  info->nominal_pairs = (int64_t)P->d.nx * P->d.nz * P->d.n_elem;
  info->active_pairs = P->active_pairs;
  info->executed_pairs = P->executed_pairs;
  info->device_bytes = P->device_bytes;
  info->tma_staging = P->use_tma ? 1 : 0;
  info->chunk_steps = P->form[0].nc;
  info->lane_rows = 1 << P->lane_rows_log2;
  info->tmem_columns = P->form[0].tmem_cols;
  info->delay_table = P->full ? PA_TABLE_FULL : PA_TABLE_LATTICE;
  info->table_bytes = delay_table_bytes(P);
  {
    int cols = 0;
    bool dense = false;
    plan_tmem(P, &cols, &dense);
    info->tmem_dense = dense ? 1 : 0;
  }
  info->device_error_flags = 0;
  {
    DeviceGuard g(P->device);
    for (int b = 0; b < kHostSets; ++b) {
      if (!P->scratch[b]) continue;
      int flag = 0;
      PA_CUDA(cudaDeviceSynchronize());
      PA_CUDA(cudaMemcpy(&flag, P->scratch[b], sizeof flag, cudaMemcpyDeviceToHost));
      info->device_error_flags |= (uint32_t)flag;
    }
  }
  return PA_OK;
}

pa_status pa_plan_form(pa_plan_t P, int32_t n_frames, int32_t* form) {
  if (!P || !form) return fail(PA_EINVAL, "null argument");
  if (n_frames < 1 || n_frames > P->d.max_batch)
    return fail(PA_EINVAL, "a launch of %d frames is outside 1..max_batch (%d)", n_frames, P->d.max_batch);
  *form = 1 + (int32_t)(&pick_form(P, n_frames) - P->form);
  return PA_OK;
}

pa_status pa_beamform(pa_plan_t P, const void* rf_dev, int32_t n_frames, float* out_dev,
                      uint32_t stages, void* cuda_stream) {
  if (!P) return fail(PA_EINVAL, "null plan");
  if (n_frames < 0) return fail(PA_EINVAL, "n_frames < 0");
  if ((stages & 7u) == 0 || (stages & ~7u)) return fail(PA_EINVAL, "stages mask 0x%x invalid", stages);
  if (n_frames == 0) return PA_OK;
  if (!rf_dev || !out_dev) return fail(PA_EINVAL, "null buffer");
  if (((uintptr_t)rf_dev & 15) || ((uintptr_t)out_dev & 15))
    return fail(PA_EINVAL, "buffers must be 16-byte aligned");
  DeviceGuard g(P->device);
  const pa_plan_desc& d = P->d;
  const size_t rf_frame = (size_t)d.n_elem * d.n_samples * P->elt;
  const size_t out_frame = (size_t)popcount3(stages) * P->n_out * d.nx * d.nz;
  for (int f0 = 0; f0 < n_frames; f0 += d.max_batch) {
    const int nf = std::min(d.max_batch, n_frames - f0);
    pa_status s = run_chunk(P, (const char*)rf_dev + (size_t)f0 * rf_frame, nf,
                            out_dev + (size_t)f0 * out_frame, stages, (cudaStream_t)cuda_stream,
                            P->scratch[0]);
    if (s != PA_OK) return s;
  }
  return PA_OK;
}

pa_status pa_beamform_host(pa_plan_t P, const void* rf_host, int32_t n_frames, float* out_host,
                           uint32_t stages, void* cuda_stream) {
  if (!P) return fail(PA_EINVAL, "null plan");
  if (n_frames < 0) return fail(PA_EINVAL, "n_frames < 0");
  if ((stages & 7u) == 0 || (stages & ~7u)) return fail(PA_EINVAL, "stages mask 0x%x invalid", stages);
  if (n_frames == 0) return PA_OK;
  if (!rf_host || !out_host) return fail(PA_EINVAL, "null buffer");
  DeviceGuard g(P->device);
  const pa_plan_desc& d = P->d;
  cudaStream_t user = (cudaStream_t)cuda_stream;
  pa_plan_s::HostTune* tune = host_tune(P, n_frames, stages);
  const bool tuning = tune->fixed.empty() && tune->chosen < 0;
  const int cur = tuning ? tune->order[tune->pos] : -1;
  const std::vector<int32_t> sched = tune->current();
  const long long builds0 = P->graph_builds;
  bool grew = false;
  const auto t_start = std::chrono::steady_clock::now();
  // buffers sized for the largest chunk of any candidate, so trying
  // candidates does not reallocate
  int chunk = 1, sets_needed = 1;
  for (const auto& c : tune->cand) {
    chunk = std::max(chunk, *std::max_element(c.begin(), c.end()));
    sets_needed = std::max(sets_needed, (int)c.size());
  }
  for (int32_t c : tune->fixed) chunk = std::max(chunk, c);
  sets_needed = std::min(kHostSets, std::max(sets_needed, (int)tune->fixed.size()));
  const int nsets = std::min<int>(kHostSets, (int)sched.size());
  const size_t rf_frame = (size_t)d.n_elem * d.n_samples * P->elt;
  const size_t out_frame = (size_t)popcount3(stages) * P->n_out * d.nx * d.nz;
  const size_t need_rf = (size_t)sets_needed * chunk * rf_frame;
  const size_t need_out = (size_t)sets_needed * chunk * out_frame * sizeof(float);
  if (need_rf > P->h_rf_bytes || need_out > P->h_out_bytes) {
    grew = true;
    const pa_status s = alloc_staging(P, std::max(need_rf, P->h_rf_bytes),
                                      std::max(need_out, P->h_out_bytes));
    if (s != PA_OK) return s;
  }
  if (!P->host_flag && may_wait(P)) {
    P->host_flag = g_host_words.take();
    if (!P->host_flag) return fail(PA_ECUDA, "pinned memory: %s", cudaGetErrorString(cudaGetLastError()));
    *P->host_flag = 1;
  }
  if (!P->h_ev) PA_CUDA(cudaEventCreateWithFlags(&P->h_ev, cudaEventDisableTiming));
  for (int b = 0; b < nsets; ++b) {
    if (!P->hs[b]) PA_CUDA(cudaStreamCreateWithFlags(&P->hs[b], cudaStreamNonBlocking));
    if (!P->h_done[b]) PA_CUDA(cudaEventCreateWithFlags(&P->h_done[b], cudaEventDisableTiming));
    if (!P->scratch[b]) {
      pa_status s = dalloc(P, &P->scratch[b], P->scratch_ints);
      if (s != PA_OK) return s;
      PA_CUDA(cudaMemset(P->scratch[b], 0, P->scratch_ints * sizeof(int)));
    }
  }
  if (P->use_graph && P->prof == 0 && is_pinned(rf_host) && is_pinned(out_host)) {
    // pinned buffers: the whole call is one graph launch on the caller's stream
    pa_plan_s::HostGraph* hg = nullptr;
    for (auto& g : P->host_graphs)
      if (g.nf == n_frames && g.stages == stages && g.sched == sched) hg = &g;
    if (!hg) {
      if (P->host_graphs.size() >= 64) {  // bounded, oldest first
        cudaGraphExecDestroy(P->host_graphs.front().exec);
        cudaGraphDestroy(P->host_graphs.front().graph);
        P->host_graphs.erase(P->host_graphs.begin());
      }
      pa_plan_s::HostGraph g;
      g.nf = n_frames;
      g.stages = stages;
      g.sched = sched;
      pa_status s = build_host_graph(P, g, rf_host, out_host, chunk, nsets);
      if (s != PA_OK) return s;
      P->host_graphs.push_back(std::move(g));
      hg = &P->host_graphs.back();
    } else if (hg->rf_host != rf_host || hg->out_host != out_host) {
      for (size_t c = 0; c < hg->sched.size(); ++c) {
        PA_CUDA(cudaGraphExecMemcpyNodeSetParams1D(hg->exec, hg->up[c], hg->up_dev[c],
                                                   (const char*)rf_host + hg->up_off[c],
                                                   hg->up_bytes[c], cudaMemcpyHostToDevice));
        PA_CUDA(cudaGraphExecMemcpyNodeSetParams1D(hg->exec, hg->down[c],
                                                   out_host + hg->down_off[c], hg->down_dev[c],
                                                   hg->down_bytes[c], cudaMemcpyDeviceToHost));
      }
      hg->rf_host = rf_host;
      hg->out_host = out_host;
    }
    PA_CUDA(cudaGraphLaunch(hg->exec, user));
    PA_CUDA(cudaStreamSynchronize(user));
    return host_call_done(P, tune, tuning, cur, t_start, grew || P->graph_builds != builds0);
  }
  // the internal streams start after work already queued on the caller's stream
  PA_CUDA(cudaEventRecord(P->h_ev, user));
  for (int b = 0; b < nsets; ++b) PA_CUDA(cudaStreamWaitEvent(P->hs[b], P->h_ev, 0));
  int f0 = 0;
  for (size_t c = 0; c < sched.size(); ++c) {
    const int nf = sched[c];
    const int b = (int)(c % nsets);
    cudaStream_t st = P->hs[b];
    char* rf_d = (char*)P->h_rf + (size_t)b * chunk * rf_frame;
    float* out_d = P->h_out + (size_t)b * chunk * out_frame;
    PA_CUDA(cudaMemcpyAsync(rf_d, (const char*)rf_host + (size_t)f0 * rf_frame, nf * rf_frame,
                            cudaMemcpyHostToDevice, st));
    // the launch sequence waits for the previous chunk's (measured on GB300,
    // cfg2, 32 FP32 frames: 1.013 ms per call against 1.097 ms when
    // neighbouring chunks' kernels overlap)
    if (c > 0) PA_CUDA(cudaStreamWaitEvent(st, P->h_done[(c - 1) % nsets], 0));
    pa_status s = run_chunk(P, rf_d, nf, out_d, stages, st, P->scratch[b]);
    if (s != PA_OK) return s;
    PA_CUDA(cudaEventRecord(P->h_done[b], st));
    PA_CUDA(cudaMemcpyAsync(out_host + (size_t)f0 * out_frame, out_d,
                            nf * out_frame * sizeof(float), cudaMemcpyDeviceToHost, st));
    f0 += nf;
  }
  for (int b = 0; b < nsets; ++b) PA_CUDA(cudaStreamSynchronize(P->hs[b]));
  return host_call_done(P, tune, tuning, cur, t_start, grew || P->graph_builds != builds0);
}


pa_status pa_plan_set_host_schedule(pa_plan_t P, int32_t n_frames, uint32_t stages,
                                    const int32_t* chunks, int32_t n_chunks) {
  if (!P) return fail(PA_EINVAL, "null plan");
  if (n_frames < 1) return fail(PA_EINVAL, "n_frames < 1");
  if ((stages & 7u) == 0 || (stages & ~7u)) return fail(PA_EINVAL, "stages mask 0x%x invalid", stages);
  if (n_chunks < 0 || (n_chunks > 0 && !chunks)) return fail(PA_EINVAL, "invalid chunk list");
  std::vector<int32_t> v(chunks, chunks + n_chunks);
  long long sum = 0;
  for (int32_t c : v) {
    if (c < 1 || c > P->d.max_batch)
      return fail(PA_EINVAL, "chunk of %d frames outside 1..max_batch (%d)", c, P->d.max_batch);
    sum += c;
  }
  if (n_chunks > 0 && sum != n_frames)
    return fail(PA_EINVAL, "chunks sum to %lld frames, not %d", sum, n_frames);
  pa_plan_s::HostTune* t = host_tune(P, n_frames, stages);
  t->fixed = v;  // empty: back to tuning (or to the tuned choice)
  return PA_OK;
}

pa_status pa_plan_host_schedule(pa_plan_t P, int32_t n_frames, uint32_t stages, int32_t* chunks,
                                int32_t max_chunks, int32_t* n_chunks, int32_t* state) {
  if (!P || !chunks || !n_chunks || !state) return fail(PA_EINVAL, "null argument");
  if (n_frames < 1) return fail(PA_EINVAL, "n_frames < 1");
  if ((stages & 7u) == 0 || (stages & ~7u)) return fail(PA_EINVAL, "stages mask 0x%x invalid", stages);
  pa_plan_s::HostTune* t = host_tune(P, n_frames, stages);
  const std::vector<int32_t>& s = t->current();
  if ((int)s.size() > max_chunks)
    return fail(PA_EINVAL, "schedule has %d chunks, room for %d", (int)s.size(), max_chunks);
  std::copy(s.begin(), s.end(), chunks);
  *n_chunks = (int32_t)s.size();
  *state = !t->fixed.empty() ? 3 : (t->chosen >= 0 ? 2 : 1);
  return PA_OK;
}

pa_status pa_plan_use_graph(pa_plan_t P, int32_t enable) {
  if (!P) return fail(PA_EINVAL, "null plan");
  P->use_graph = enable != 0;
  return PA_OK;
}

pa_status pa_plan_profile(pa_plan_t P, int32_t enable) {
  if (!P) return fail(PA_EINVAL, "null plan");
  if (enable < 0 || enable > 2) return fail(PA_EINVAL, "profile mode %d not in 0..2", (int)enable);
  P->prof = enable == 0 ? 0u : enable == 1 ? 7u : 1u;
  return PA_OK;
}

pa_status pa_plan_profile_read(pa_plan_t P, double ms[3], int64_t launches[3]) {
  if (!P || !ms || !launches) return fail(PA_EINVAL, "null argument");
  DeviceGuard g(P->device);
  for (int k = 0; k < 3; ++k) {
    ms[k] = 0.0;
    launches[k] = 0;
  }
  for (auto& e : P->ev_used) {
    PA_CUDA(cudaEventSynchronize(e.second.second));
    float t = 0.f;
    PA_CUDA(cudaEventElapsedTime(&t, e.second.first, e.second.second));
    ms[e.first] += t;
    launches[e.first] += 1;
    P->ev_free.push_back(e.second);
  }
  P->ev_used.clear();
  return PA_OK;
}

pa_status pa_destroy(pa_plan_t P) {
  free_plan(P);
  return PA_OK;
}

const char* pa_status_str(pa_status s) {
  switch (s) {
    case PA_OK: return "ok";
    case PA_EINVAL: return "invalid argument";
    case PA_ENOMEM: return "out of device memory";
    case PA_ECUDA: return "CUDA error";
    case PA_ETIMEOUT: return "timed out";
    case PA_EUNSUPPORTED: return "unsupported";
    case PA_EBUSY: return "busy";
  }
  return "unknown status";
}

const char* pa_last_error(void) { return g_err.c_str(); }

int32_t pa_version(void) { return 105; }

}  // extern "C"
