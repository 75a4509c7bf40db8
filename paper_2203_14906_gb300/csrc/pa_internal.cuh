// pa_internal.cuh -- types shared by the kernels and the host plan code of
// the HO-DMAS beamformer (not part of the public ABI).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pa_hodmas.h"

namespace pa {

// Columns handled by one thread.  The thread's pixels sit at columns
// jt, jt+m, ..., jt+(kC-1)m of one depth row, so at channel step u they all
// need the delay of the same lattice offset d = jt - m*u (pixel c pairs with
// channel i = u + c): one table load serves kC pairs.
constexpr int kC = 4;
// Channel steps per shared-memory chunk (chosen per plan, a multiple of kC,
// at most kNCMax) and the virtual channels staged per chunk (steps + kC - 1).
constexpr int kNCMax = 72;
constexpr int kNCSMax = kNCMax + kC - 1;
// Channel steps between Kahan folds of the compensated power sums: plain
// FP32 partial sums over 64 channels, compensated across folds.  Every fold
// loads and stores each accumulator's totals in TMEM (about 100 instructions
// per thread), so its issue cost per pair halves with the interval.
// Measured on GB300 (BF16 RF, 128 channels, k = 3, 32 frames, fused kernel
// per launch): folding every 8 / 16 / 32 steps took 0.937 / 0.894 / 0.877 ms
// in an earlier build with the totals in registers; with the totals in TMEM
// every 32 / 64 steps takes 0.676 / 0.661 ms (cfg3, 256 channels: k = 3
// 1.289 / 1.259 ms, k = 5 1.586 / 1.547 ms).
constexpr int kFoldBlocks = 16;  // blocks of kC steps
constexpr int kMaxOrder = 8;
// Shared-memory layout of the fused kernel: work-item words, the TMA
// mbarrier (8 B at 16) and the TMEM base address (4 B at 24), channel bases
// and window starts (kCbInts ints each,
// >= kNCSMax + 1, multiple of 4), the raw TMA buffer (128-byte aligned, empty
// without TMA), then the interpolation slots.
constexpr int kCbInts = 76;
constexpr int kMbarOff = 16;
constexpr int kTmemOff = 24;
constexpr int kCbOff = 32;
constexpr int kLoOff = kCbOff + kCbInts * 4;
constexpr int kRawOff = 640;  // >= kLoOff + 4 kCbInts, 128-byte aligned
static_assert(kRawOff >= kLoOff + kCbInts * 4 && kRawOff % 128 == 0, "shared layout");
constexpr int kMaxThreads = 1024;
// Shared-memory layout of the two-frame kernel: the stages' mbarriers and
// counts of finished warps, TMEM address, stop flag, the running work item,
// then per stage 32 bytes of work-item words and the channel bases, then the
// stages' slots (128-byte aligned).
constexpr int kPipeStages = 4;  // at most
constexpr int kPipeFullOff = 0, kPipeCountOff = 32, kPipeTmemOff = 48, kPipeStopOff = 52;
constexpr int kPipeProdOff = 64;
constexpr int kPipeMetaOff = 96;
constexpr int kPipeCbOff = kPipeMetaOff + 32 * kPipeStages;
constexpr int kPipeSlotOff = 1536;
static_assert(kPipeSlotOff >= kPipeCbOff + kPipeStages * kCbInts * 4 && kPipeSlotOff % 128 == 0,
              "shared layout");

// A call is a chain of kernels, each on the results of the one before.  The
// graph's edges between them are programmatic, so a kernel's blocks are brought
// up while the one before ends: every kernel of the chain lets its successor
// start (launch_next) and touches nothing of the chain's buffers before its
// predecessor has completed and its writes are visible (wait_previous; after a
// plain edge or launch both do nothing).  A successor's blocks are placed only
// when every block of a kernel has come to launch_next, so they take no room
// from it.  The fused kernels come to it before their last epilogue: from their
// start on, the successor's blocks crowd onto the SMs that are free first
// (one quick-look frame 20.6 -> 22.4 us, five ragged frames 74.0 -> 75.5;
// prepare_chunk says when the post filter keeps a plain edge, and why the one-frame
// form has one after the clearing kernel).
// Loads of the chain's buffers are plain or bulk loads, never the read-only
// path; the proxy fence orders bulk copies of slots that the preparation pass
// stored.  Measured on GB300 (whole calls back to back, every edge plain -> as
// prepare_chunk has them): 42 calls 1.013 times as fast on average, the short ones
// most (21.1 -> 19.8 us, 34.1 -> 32.3), those of 0.5 ms and more by nothing.
__device__ __forceinline__ void launch_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_previous() {
  asm volatile("griddepcontrol.wait;\n fence.proxy.async.global;" ::: "memory");
}

// The fine-grained kernel keeps kC shifted copies of the channel bases.
constexpr int kFineSlotOff = kPipeCbOff + 2 * kC * kCbInts * 4 + 128;
constexpr int kFineStages = 2;
static_assert(kFineSlotOff % 16 == 0, "shared layout");

// TMEM columns a fused-kernel block allocates for compensated totals (a
// power of two >= 32): the warps sharing a 32-lane quarter of TMEM times 8
// columns per accumulator (kC totals and kC compensation terms; na counts the
// accumulators of every frame of a work item).
__host__ __device__ constexpr int tmem_columns(int warps, int na) {
  return ((warps + 3) / 4) * na * 8 <= 32    ? 32
         : ((warps + 3) / 4) * na * 8 <= 64  ? 64
         : ((warps + 3) / 4) * na * 8 <= 128 ? 128
         : ((warps + 3) / 4) * na * 8 <= 256 ? 256
                                              : 512;
}
// TMEM columns of one SM.
constexpr int kTmemColsPerSm = 512;

// Lattice-table layout.  Row t = d - dmin of lattice offset d (dmin = -m
// steps) is residue r = t % m, sequence number q = t / m.  A thread's four
// channel steps u .. u + 3 of one block need q, q - 1, q - 2, q - 3 of one
// residue, and q = 3 (mod 4) at every block's first step (tiles and threads
// start on multiples of 4 m columns, u on -3 + 4 k): the four entries of
// every (residue, group of four q, depth) lie together, in the order of the
// steps, as two 16-byte halves kept apart by eight depth rows:
//   [residue][q / 4][z / 8][half][z % 8][2 entries]
// so a block reads two 16-byte pieces at a fixed distance of 128 bytes (eight
// rows' worth), its neighbours in depth the pieces next to them, and the
// next block's pieces lie a fixed stride below.  Depth rows are padded to a
// multiple of 32.  A block's four entries used to be four 8-byte loads from
// four lattice rows, each with its own address; now they are two loads from
// one.  Measured on GB300 (whole calls, before -> after): 16 frames of 512 x
// 512, nearest k = 2 212.3 -> 202.9 us, 8 frames k = 5 252.2 -> 247.8 us,
// 4 frames of 1024 x 1024, BF16 + Kahan k = 3 699 -> 677 us, 32 frames of
// 512 x 512 k = 3 739 -> 730 us; small single frames unchanged.
__host__ __device__ __forceinline__ size_t table_index_rq(int r, int q, int z, int groups, int nzp) {
  const int step = 3 - (q & 3);
  const size_t block = ((size_t)r * groups + (q >> 2)) * (nzp >> 3) + (z >> 3);
  return block * 32 + (step >> 1) * 16 + (z & 7) * 2 + (step & 1);
}
__host__ __device__ __forceinline__ size_t table_index(int t, int z, int m, int groups, int nzp) {
  return table_index_rq(t % m, t / m, z, groups, nzp);
}

// Parameters of the fused gather + interpolate + root + power-sum kernel.
struct BfParams {  // aligned as CUtensorMap requires
  CUtensorMap tmap;       // 3-D RF map [frames][N][Ns], box {wr, 1, 1} (TMA path)
  int use_tma;            // 1: stage with TMA boxes, 0: vectorised loads
  int wr;                 // raw samples per channel delivered by one TMA box
  int rp;                 // row pitch of the raw buffer in samples (128-byte rows)
  int chunk_bytes;        // bytes one chunk's TMA boxes deliver
  int pairs_off;          // byte offset of the interpolation slots
  const void* rf;         // [frames][N][Ns] in rf_dtype
  int rf_dtype;           // pa_rf_dtype
  int vec_ok;             // rows start 8/16-byte aligned (Ns % 4 == 0)
  int nearest;            // 1: nearest-sample delays (a = 0), one tap per pair
  int lane_rows_log2;     // log2 of the depth rows per lane group: 5, 4 or 3
  int nc, ncs;            // channel steps per chunk, virtual channels staged per chunk
  int tmem_cols;          // TMEM columns a block allocates (compensated sums), else 0
  int n_elem, n_samples;
  long long frame_elems;  // N * Ns
  const int2* table;      // lattice table {n0 * 8, float bits of a} (table_index)
  const int2* ftab;       // full table, in the kernel's read order: per tile,
                          // channel step (steps + 3), pixel half c / 2, thread
                          // of the tile, pixel c % 2: {(n0 - window start) * 8,
                          // float bits of a}
  int full;               // 1: full table (channel bases are window starts)
  int steps;              // channel steps u1 - u0
  const float* wtab;      // apodisation weights, in the table's order (or null)
  const int4* items;      // [n_tiles * ngroups] {tile_id, grp, tx, tz}, deepest first
  const int2* slot_rg;    // [slots] {column residue r_m, column group g}
  int tgroups, nz_pad;    // lattice table: groups of four q per residue, padded depth rows
  int dmin;               // lattice offset of table row 0 (-m steps)
  int m;                  // column stride of a thread's pixels (lattice: pitch / dx)
  int R;                  // column groups per residue in a tile
  int nxt, nzt;           // tiles along x and z
  int tile_x, tile_z;
  int warps;              // warps per block
  int slots;              // warp slots per tile (m * R)
  int ngroups;            // residue groups per tile (slots / warps)
  int nv;                 // virtual channels (zero rows pad both ends)
  int u0;                 // first channel step (= -(kC-1))
  int window;             // float2 slots staged per channel (multiple of 4)
  int w4_inv;             // ceil(2^20 / (window / 4)): exact idx / (window / 4) by multiply-shift
  const int* lo;          // [n_tiles][nv] first staged sample per channel
  const int2* urange;     // [n_tiles][warps] channel-step range of a warp
  const int2* vchunks;    // [n_tiles] chunk range of a tile
  float* out;             // output base
  int planes;             // planes per frame (n_stages * n_outputs)
  int plane_das, plane_dmas, plane_ho;  // raw plane of each output or -1
  int nx, nz;
  float ek_top;           // amplitude sums from here on take the FP64 e_k (df_in_range)
  int n_frames;           // frames in this launch
  int n_items;            // n_tiles * ngroups * n_frames (two-frame kernel: * n_fgroups)
  // two-frame kernel
  int n_fgroups;          // frame pairs (ceil(n_frames / 2)); fine kernel: frames
  int splits;             // fine kernel: items per tile
  int stages;             // chunks of slots in shared memory
  const unsigned char* slots_dev;  // prepared slots (k_prep): a row of zeros,
                                   // then [frame pair][channel] rows of
                                   // slot_pitch slots
  long long slot_pitch;
  int slot_margin;        // zero slots before a row's sample 0
  int* counter;           // work counter (set before launch)
  int* err;               // error flags: 1, 2 index checks (checked builds), 8 a wait ran out
  int* timeouts;          // running count of blocks whose bounded TMA wait ran out
  int* host_flag;         // pinned host word set when one did (null before the
                          // plan's first host-path call, and where no kernel waits)
  int expect_extra;       // bytes added to every chunk's expected transaction
                          // count: 0, or > 0 only to test the bounded wait
};

// A kernel launch described as data (direct launch or CUDA-graph node).
struct LaunchSpec {
  const void* func = nullptr;
  dim3 grid, block;
  size_t smem = 0;
};

// Preparation pass of the two-frame kernel (pa_prep.cu).
struct PrepParams {
  const void* rf;      // [frames][N][Ns]
  unsigned char* slots;  // as BfParams::slots_dev
  long long pitch;
  int margin;
  int rf_dtype, n_elem, n_samples, n_frames;
  int n_lo, n_hi;      // samples the windows hold
  int blocks_per_row;
  int nf;              // frames per slot: 2, or 1 ({r, d} slots of the fine kernel)
  int mode, order;     // slot kind (PipeMode), order of its roots
  int* zero;           // words cleared before the fused kernel (work counter, maxima)
  int n_zero;
  int counter0;        // what the work counter starts at: the fused kernel's blocks
};
void prep_spec(PrepParams* p, LaunchSpec* s);

// Post-filter / envelope parameters.
struct PostParams {
  float* out;
  int planes;          // planes per frame
  int n_out;           // outputs per stage
  int s_src, s_dst;    // stage index holding raw / receiving the envelope
  int nx, nz, m, log2m;
  const float2* tw;    // per-pass twiddle blocks (see twiddles() in pa_post.cu)
  const float2* tw_reg;  // k_post_reg: e^{-2 pi i k l / M} at k L + l, k < 32, l < L = M / 32
  int n_tw;            // entries of tw
  const float* mask;   // [n_out][m] band-pass x analytic mask
  int2 band[3];        // per output: first bin the mask keeps, rows of L bins (k_post_reg)
  int band_rows;       // most rows of any output
  int* maxslot;        // [frames][n_out] float bits of the image maximum
  int n_frames;
  int warps_per_block;
};

struct LogParams {
  float* out;
  int planes, n_out, s_src, s_dst;
  long long plane_elems;  // nx * nz
  const int* maxslot;
  float dyn_range_db;
  int n_frames;
};

const void* bf_func(int order, bool apod, bool comp, bool full);
const void* bf_fine_func(int order, bool apod, bool comp, bool full, int px);
int pipe_slot_mode(int order, bool apod, bool nearest);  // PipeMode
int pipe_slot_bytes(int mode);
const void* bf_pipe_func(int order, bool apod, bool comp, bool full, bool nearest);
void post_spec(const PostParams& p, LaunchSpec* s);
// Radix of the first FFT pass of the in-place post kernel (the passes after
// it are radix 8, then one radix-4 or radix-2 pass for the remainder); the
// host builds the per-pass twiddle tables in the same order.
__host__ __device__ constexpr int post_first_radix(int m) { return m == 1024 ? 16 : 8; }
// Post-kernel buffers keep one padding slot every 2^post_pad_shift(M)
// complex elements (16 from 256 points on, else 8).
__host__ __device__ constexpr int post_pad_shift(int m) { return m >= 256 ? 4 : 3; }
__host__ __device__ constexpr int post_padded_len(int m) { return m + (m >> post_pad_shift(m)); }
int post_buffers(int m);     // M-point complex buffers per team of the post kernel
const void* post_inplace_func(int m);  // in-place kernel for M points, or nullptr
int post_team_warps(int m);  // warps per team (column pair) of the post kernel
const void* post_reg_func(int m);      // register kernel for M points, or nullptr
void log_spec(const LogParams& p, int num_sms, LaunchSpec* s);

cudaError_t bf_occupancy(const void* func, int block, size_t smem, int* blocks_per_sm);

// One translation unit per order keeps the builds parallel.
#define PA_DECLARE_ORDER(K) const void* bf_func_k##K(bool apod, bool comp, bool full);
#define PA_DECLARE_PIPE(K) \
  const void* bf_pipe_func_k##K(bool apod, bool comp, bool full, bool nearest);
PA_DECLARE_ORDER(1)
PA_DECLARE_ORDER(2)
PA_DECLARE_ORDER(3)
PA_DECLARE_ORDER(4)
PA_DECLARE_ORDER(5)
PA_DECLARE_ORDER(6)
PA_DECLARE_ORDER(7)
PA_DECLARE_ORDER(8)
PA_DECLARE_PIPE(1)
PA_DECLARE_PIPE(2)
PA_DECLARE_PIPE(3)
PA_DECLARE_PIPE(4)
PA_DECLARE_PIPE(5)
#define PA_DECLARE_FINE(K) \
  const void* bf_fine_func_k##K(bool apod, bool comp, bool full, int px);
PA_DECLARE_FINE(1)
PA_DECLARE_FINE(2)
PA_DECLARE_FINE(3)
PA_DECLARE_FINE(4)
PA_DECLARE_FINE(5)
PA_DECLARE_FINE(6)
PA_DECLARE_FINE(7)
PA_DECLARE_FINE(8)
#undef PA_DECLARE_FINE
#undef PA_DECLARE_ORDER
#undef PA_DECLARE_PIPE

// Sets the thread-local message returned by pa_last_error().
void set_error_message(const char* msg);
// Device address of the plan's running count of timed-out waits (the word
// pa_beamform's launches update), for the server's completion check.
int* plan_timeout_counter(pa_plan_s* P);
// Device memory the plan owns (without synchronising, unlike pa_plan_get_info).
size_t plan_device_bytes(const pa_plan_s* P);
// Of these, the prepared slots, without which the plan runs its one-frame form.
size_t plan_slot_bytes(const pa_plan_s* P);
// pa_plan with at most slot_limit bytes of slots, which plan_drop_slots can give
// back; and that: nothing of the plan in flight, no graph of it kept
// (pa_plan_use_graph 0).
constexpr size_t kNoSlotLimit = (size_t)-1;
pa_status plan_create(const pa_plan_desc* desc, cudaStream_t st, size_t slot_limit, pa_plan_s** out);
pa_status plan_drop_slots(pa_plan_s* P);
// Device memory a plan for desc cannot do without, and a bound of its slots.
pa_status plan_memory(const pa_plan_desc* desc, size_t* bytes, size_t* slots);
// The fused kernel's parameters for one launch of nf frames (what pa_beamform
// would launch), the plan's order, and whether the plan is the plain FP32
// lattice form with linear interpolation.
pa_status plan_bf_params(pa_plan_s* P, const void* rf, int nf, float* out, uint32_t stages,
                         BfParams* b, int* k, bool* lattice_fp32_plain);
// TMEM columns per fused-kernel block and whether the plan is TMEM-dense
// (its blocks can hold more TMEM than their register share of an SM).
void plan_tmem(const pa_plan_s* P, int* cols, bool* dense);

cudaError_t post_configure(size_t smem);

}  // namespace pa
