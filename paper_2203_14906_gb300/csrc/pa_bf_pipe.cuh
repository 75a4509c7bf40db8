// pa_bf_pipe.cuh -- the two-frame form of the fused beamforming kernel: the
// pairs of pa_bf_kernel.cuh, two frames per work item, from slots prepared
// once per launch (pa_prep.cu).
//
// All frames of a launch share the delays.  A thread works on the same 4
// pixels of two frames: one table entry, one slot address and one 128-bit
// shared load serve a pair of each frame, and products and sums of the two run as
// packed instructions.  Per pair that leaves 11.3 of the one-frame form's 18
// instruction slots (k = 3, counted by ncu).
//
// Staging is gone from the arithmetic warps: the slots of a channel window are
// a contiguous run in global memory (any record length or RF type, zeros past
// the record), brought in by one bulk copy per channel into the free one of
// two chunk buffers.  Warps do not wait for one another: each waits for its
// chunk's bytes (mbarrier) and counts itself out when done; the last warp out
// of a chunk starts the copies of the chunk after next, or of the next work
// item, so a block's warps drift across chunks and items (the epilogue of one
// runs under the channel loop of another) without a block barrier.
//
// Bounds, in slots of 1/128 SM clock per pair at k = 3 (measured rates per SM
// and clock: 128 issue, ex2 32, lg2 / rsqrt / sqrt 16 threads): MUFU 12, issue
// 11.3, shared loads 8 (16 B a pair-of-frames, conflict-free) + table 2.  A loop
// of these roots with 13 instructions a pair takes about 16 by itself; 16 warps a
// SM (128 registers: 40 sums) reach 19 (59 % issue active).
// Measured against the one-frame form on GB300, before the sums were packed
// (packed_sums; whole calls, with the slot
// preparation pass; see pick_form for where the line lies): 32 frames of
// 512 x 512, k = 3 730 -> 679 us; nearest k = 2 203 -> 176; 4 frames of 1024 x
// 1024 BF16 + Kahan 677 -> 644; full table 399 -> 290; 5 frames of 1501 samples
// (rows off 16-byte boundaries) 96 -> 81; apodised 64-frame k = 4 batch 3711 ->
// 3398.
#pragma once

#include "pa_bf_kernel.cuh"

namespace pa {

// How a pair's sample is formed, and the slot it reads: linear interpolation
// {r, r', d, d'}; nearest sample with the root taken once per RF sample
// {r, r', root, root'} (k_prep); nearest sample with the root taken per pair
// {r, r'}, for weighted samples, whose root follows the weight, and for orders
// <= 2, where the shared loads bind and half the bytes are worth a MUFU per
// pair (16 frames of 512 x 512, k = 2: 0.207 ms with 16-byte slots).
enum PipeMode { kLinear = 0, kNearestRoots = 1, kNearest = 2 };
__host__ __device__ constexpr PipeMode pipe_mode(int order, bool apod, bool nearest) {
  return !nearest ? kLinear : apod || order <= 2 ? kNearest : kNearestRoots;
}
__host__ __device__ constexpr int slot_bytes(int mode) { return mode == kNearest ? 8 : 16; }

// Adds 1 to a shared counter, ordered with the warp's earlier shared reads and
// the other warps' adds.
__device__ __forceinline__ int count_arrival(uint32_t addr) {
  int old;
  asm volatile("atom.acq_rel.cta.shared::cta.add.s32 %0, [%1], 1;" : "=r"(old) : "r"(addr) : "memory");
  return old;
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, int bytes, uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(mbar)
      : "memory");
}

// Two FP32 products, sums or multiply-adds, in one instruction if PACK (each
// rounded as the scalar one).  A packed instruction takes the arithmetic pipe as
// long as its two scalar ones and one issue slot instead of two.
template <bool PACK>
__device__ __forceinline__ void mul_pair(float& x, float& y, float a0, float a1, float b0, float b1) {
  if constexpr (!PACK) {
    x = a0 * b0;
    y = a1 * b1;
    return;
  }
  asm("{\n .reg .b64 p, q, r;\n mov.b64 p, {%2, %3};\n mov.b64 q, {%4, %5};\n"
      " mul.rn.f32x2 r, p, q;\n mov.b64 {%0, %1}, r;\n}"
      : "=f"(x), "=f"(y)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}
template <bool PACK>
__device__ __forceinline__ void add_pair(float& x, float& y, float a0, float a1) {
  if constexpr (!PACK) {
    x += a0;
    y += a1;
    return;
  }
  asm("{\n .reg .b64 p, q, r;\n mov.b64 p, {%0, %1};\n mov.b64 q, {%2, %3};\n"
      " add.rn.f32x2 r, p, q;\n mov.b64 {%0, %1}, r;\n}"
      : "+f"(x), "+f"(y)
      : "f"(a0), "f"(a1));
}
template <bool PACK>
__device__ __forceinline__ void fma_pair(float& x, float& y, float a0, float a1, float b0, float b1) {
  if constexpr (!PACK) {
    x = fmaf(a0, b0, x);
    y = fmaf(a1, b1, y);
    return;
  }
  asm("{\n .reg .b64 p, q, r, t;\n mov.b64 p, {%2, %3};\n mov.b64 q, {%4, %5};\n"
      " mov.b64 r, {%0, %1};\n fma.rn.f32x2 t, p, q, r;\n mov.b64 {%0, %1}, t;\n}"
      : "+f"(x), "+f"(y)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// Which sums the two frames' pairs are added to by packed instructions, a bit
// per sum: bit 0 v[0], bit 1 v[1], bit 2 v[3], bit 3 v[4], ...; with the bits,
// kProducts packs the roots' products.  A packed sum saves an issue slot and
// ties its operands to aligned register pairs; which of the two weighs more
// depends on the registers a kernel has left, so every line is measured (RAW
// images of 512 x 512, 16 frames; us of the fused kernel and its
// preparation pass with the products alone packed -> with the sums below, and
// the sets of table entries and blocks per SM below):
//   k <= 2 nearest 175 -> 152, linear 232 -> 205, apodised nearest 96 -> 84,
//     Kahan 238 -> 230; 1024 x 1024, 256 channels 428 -> 379
//   k = 3 linear 287 -> 278, nearest 221 -> 215, apodised 140 -> 135, Kahan
//     305 -> 294, both 147 -> 138
//   k = 4 linear 319 (any sums: 321-328), nearest 240 -> 225, apodised 153 ->
//     145, Kahan 348 -> 334, both 156 -> 150
//   k = 5 linear 188 -> 178 (8 frames), nearest 303 -> 300, apodised 161 -> 157,
//     Kahan 381 -> 371, both 171 -> 165
//   nearest with Kahan sums: k = 3 303 -> 232, k = 4 337 -> 247, k = 5 322 -> 318;
//     apodised nearest: k = 3 119, k = 4 137 -> 132, k = 5 154 -> 142
//   k <= 2 with wider windows (3 samples a row): 277 -> 275
// With the full table, whose loads leave issue slots free, nothing is packed
// (the products alone: 0.257 -> 0.270 ms).
constexpr int kProducts = 64;
__host__ __device__ constexpr int packed_sums(int k, bool apod, bool comp, bool full, int mode) {
  if (full) return 0;
  if (k <= 2) return kProducts | (apod && comp ? 0 : 1);
  if (k == 3) return kProducts | (mode == kNearestRoots ? 1 + 2 + 4 : 1 + 2 + 4 + 8);
  if (k == 4) {
    if (mode == kNearestRoots || (apod && comp)) return kProducts | (1 + 4 + 8);
    return kProducts | (apod || comp ? 1 + 2 + 4 + 8 + 16 : 0);
  }
  if (apod && comp) return kProducts | (1 + 8);
  if (comp) return kProducts | (1 + 4 + 8 + 32);
  if (apod || mode == kNearestRoots) return kProducts | (1 + 4 + 8);
  return kProducts | 63;
}

// Blocks per SM.  Orders <= 2 have 24 sums a thread and run 24 warps a SM on 80
// registers (16 warps: nearest k = 2 174 us instead of 153; 32 warps on 64
// registers: 168), but for Kahan sums over the full aperture: their folds leave
// room for one set of table entries only there, and over 350 plans of 2-48 frames
// 24 warps take 1.04-1.18 of the time of 16, however the launch fills the GPU (one
// full launch of 32 frames took 0.965).  With the full table 80
// registers spill (entries and weights of three steps at once: up to 134 bytes) and
// fewer loads are in flight; over 500 plans of 2-48 frames 24 warps take 1.17-1.20
// of the time of 16 (apodised 1.26-1.37, with Kahan sums 1.16-1.26; nearest samples
// 1.0-1.24).
constexpr int pipe_blocks(int k, bool apod, bool comp, bool full) {
  return k <= 2 && (apod || !comp) && !full ? 3 : 2;
}
// Sets of table entries: with one the next block's entries replace those just
// used, with two they are loaded a block ahead.  Two where registers last for
// them (k = 4 linear 319, with one 350; k <= 2 205, with one 222; apodised plain
// k = 3 135, with one 137); one for k = 5 and apodised plans (k = 5 188, with two
// 225; apodised k = 5 161, with two 179), and with Kahan sums or all the sums of
// k = 3 packed (Kahan k = 4 334, with two 340).
__host__ __device__ constexpr bool one_entry_set(int k, bool apod, bool comp, int mode) {
  if (apod) return !(k == 3 && !comp);
  return k == 5 || (k >= 3 && mode != kNearestRoots && (k == 3 || comp));
}

// The root a sample's power sums start from: sgn sqrt|s| (orders <= 2),
// |s|^(1/6), |s|^(1/4), |s|^(1/10) (orders 3, 4, 5), as pair_update takes it.
template <int K>
__device__ __forceinline__ float base_root(float s) {
  const float as = fabsf(s);
  if constexpr (K <= 2) return copysignf(sqrt_approx(as), s);
  else if constexpr (K == 3) return ex2_approx(lg2_approx(as) * (1.0f / 6.0f));
  else if constexpr (K == 4) return rsqrt_approx(rsqrt_approx(as));
  else return ex2_approx(lg2_approx(as) * 0.1f);
}

// The power sums of one pixel for the samples s, t of two frames with their
// base roots y, z: pair_update's operations in its order, so a frame's sums
// have the bits of the one-frame kernel.  PK: packed_sums.
template <int K, int PK>
__device__ __forceinline__ void sums2(float* v, float* w, float s, float t, float y, float z) {
  constexpr bool kMul = (PK & kProducts) != 0;
  add_pair<(PK & 1) != 0>(v[0], w[0], s, t);
  v[2] += fabsf(s);
  w[2] += fabsf(t);
  if constexpr (K <= 2) {
    add_pair<(PK & 2) != 0>(v[1], w[1], y, z);
  } else {
    float y2, z2;
    mul_pair<kMul>(y2, z2, y, z, y, z);
    if constexpr (K == 3) {
      const float x = copysignf(y2, s), u = copysignf(z2, t);
      fma_pair<(PK & 2) != 0>(v[1], w[1], x, u, y, z);
      add_pair<(PK & 4) != 0>(v[3], w[3], x, u);
      fma_pair<(PK & 8) != 0>(v[4], w[4], y2, z2, y2, z2);
    } else if constexpr (K == 4) {
      const float x = copysignf(y, s), u = copysignf(z, t);
      fma_pair<(PK & 2) != 0>(v[1], w[1], x, u, y, z);
      add_pair<(PK & 4) != 0>(v[3], w[3], x, u);
      add_pair<(PK & 8) != 0>(v[4], w[4], y2, z2);
      fma_pair<(PK & 16) != 0>(v[5], w[5], x, u, y2, z2);
    } else {
      const float x = copysignf(y2, s), u = copysignf(z2, t);
      float x2, u2, y3, z3;
      mul_pair<kMul>(x2, u2, y2, z2, y2, z2);
      mul_pair<kMul>(y3, z3, y2, z2, y, z);
      fma_pair<(PK & 2) != 0>(v[1], w[1], x, u, y3, z3);
      add_pair<(PK & 4) != 0>(v[3], w[3], x, u);
      add_pair<(PK & 8) != 0>(v[4], w[4], x2, u2);
      fma_pair<(PK & 16) != 0>(v[5], w[5], x, u, x2, u2);
      fma_pair<(PK & 32) != 0>(v[6], w[6], x2, u2, x2, u2);
    }
  }
}

// Two table entries, loaded where the code says (the compiler may not sink
// the load to its use).
__device__ __forceinline__ int4 load_entries16(const int2* p) {
  int4 e;
  asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];"
               : "=r"(e.x), "=r"(e.y), "=r"(e.z), "=r"(e.w)
               : "l"(p));
  return e;
}

// One slot of a step: load, form the samples of both frames, add.
template <int K, int MODE, bool APOD, int PK>
__device__ __forceinline__ void slot_pair(float* v, float* w, int addr, float a, float weight) {
  float s, t, y = 0.f, z = 0.f;
  if constexpr (MODE == kNearest) {
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(s), "=f"(t) : "r"(addr));
  } else {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(s), "=f"(t), "=f"(y), "=f"(z)
                 : "r"(addr));
  }
  if constexpr (MODE == kLinear) {
    s = fmaf(a, y, s);
    t = fmaf(a, z, t);
  }
  if constexpr (APOD) {
    s *= weight;
    t *= weight;
  }
  if constexpr (MODE != kNearestRoots) {
    if constexpr (K == 3 || K == 5) {
      constexpr float c = K == 3 ? 1.0f / 6.0f : 0.1f;
      float ls, lt;
      mul_pair<(PK & kProducts) != 0>(ls, lt, lg2_approx(fabsf(s)), lg2_approx(fabsf(t)), c, c);
      y = ex2_approx(ls);
      z = ex2_approx(lt);
    } else {
      y = base_root<K>(s);
      z = base_root<K>(t);
    }
  }
  sums2<K, PK>(v, w, s, t, y, z);
}

// Kahan totals in TMEM as in the one-frame kernel; frame h of the item owns
// columns 8 (2 q + h) .. + 7 of accumulator q.
template <int NA, bool LAZY>
__device__ __forceinline__ void fold_tmem2(float (&acc)[2][kC][NA], uint32_t tmem, bool first) {
  __syncwarp();
#pragma unroll
  for (int qh = 0; qh < 2 * NA; ++qh) {
    const int q = qh >> 1, h = qh & 1;
    float t[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (!LAZY || !first) tmem_ld8(tmem + 8 * qh, t);
#pragma unroll
    for (int c = 0; c < kC; ++c) {
      const float y = acc[h][c][q] - t[4 + c];
      const float s = t[c] + y;
      t[4 + c] = (s - t[c]) - y;
      t[c] = s;
      acc[h][c][q] = 0.f;
    }
    tmem_st8(tmem + 8 * qh, t);
  }
}

template <int NA>
__device__ __forceinline__ void final_tmem2(float (&acc)[2][kC][NA], uint32_t tmem) {
  __syncwarp();
#pragma unroll
  for (int qh = 0; qh < 2 * NA; ++qh) {
    const int q = qh >> 1, h = qh & 1;
    float t[8];
    tmem_ld8(tmem + 8 * qh, t);
#pragma unroll
    for (int c = 0; c < kC; ++c) {
      const float y = acc[h][c][q] - t[4 + c];
      const float s = t[c] + y;
      acc[h][c][q] = s - ((s - t[c]) - y);
    }
  }
}

// Loads the next chunk of the block's work into a free stage (whole warp):
// the item's words, the channel bases and one bulk copy per channel window.
// The running item and chunk live in shared memory; calls follow one another
// (each is made by the last warp to finish the stage's previous chunk, and
// that warp finishes no later chunk before it returns).
// START: the block's first chunk, of the item that is its own (k_bf_fused says
// why); the others come from the counter, which the preparation pass sets to the
// number of blocks.  (Told apart or added here, in the loop, they cost the
// variants at 128 registers spills: four frames of 1024 x 1024 with Kahan sums
// 593 -> 620 us.)
// NF frames per item.  With one (pa_bf_fine.cuh) an item is a share of a tile's
// warps, its chunks cover the whole tile, and the channel bases are written
// kC times, shifted by 0 .. kC - 1 channels, so that a warp whose first pixel
// pairs with channel u + c reads aligned fours.
template <bool FULL, int SB, int NF, bool START>
__device__ __forceinline__ void produce(const BfParams& p, unsigned char* smem, uint32_t sbase,
                                     int stage, int lane) {
  int4* prod = reinterpret_cast<int4*>(smem + kPipeProdOff);
  const uint32_t bar = sbase + kPipeFullOff + 8 * stage;
  int4* meta = reinterpret_cast<int4*>(smem + kPipeMetaOff + 32 * stage);
  int4 it = prod[0], run = prod[1];  // {tile, group, tx, tz}, {frame pair, chunk, end, state}
  __syncwarp();
  if (run.w == 2) return;  // no work left
  bool first = false;
  if (START || run.w == 0) {
    int item = START ? (int)blockIdx.x : 0;
    if constexpr (!START) {
      if (lane == 0) item = atomicAdd(p.counter, 1);
      item = __shfl_sync(0xffffffffu, item, 0);
    }
    if (item >= p.n_items) {
      if (lane == 0) {
        prod[1] = make_int4(0, 0, 0, 2);
        meta[0] = make_int4(-1, 0, 0, 0);
        mbar_arrive(bar);
      }
      return;
    }
    const int tg = item / p.n_fgroups;
    int2 vk;
    if constexpr (NF == 2) {
      it = __ldg(p.items + tg);
      vk = __ldg(p.vchunks + (size_t)it.x * p.ngroups + it.y);
    } else {
      it = __ldg(p.items + (size_t)(tg / p.splits) * p.ngroups);
      it.y = tg % p.splits;
      vk = __ldg(p.vchunks + it.x);
    }
    run = make_int4(item - tg * p.n_fgroups, vk.x, vk.y, 1);
    first = true;
  }
  const bool data = run.z > run.y;  // an item without pairs still stores its zeros
  const bool last = run.y + 1 >= run.z;
  const int W = p.window, k = run.y;
  const uint32_t slots =
      sbase + (NF == 2 ? kPipeSlotOff : kFineSlotOff) + stage * (p.ncs * W * SB);
  constexpr int CB = NF == 2 ? 1 : kC;  // copies of the channel bases
  int* s_cb = reinterpret_cast<int*>(smem + kPipeCbOff + stage * CB * kCbInts * 4);
  if (lane == 0) {
    meta[0] = make_int4(it.x, run.x * NF, it.y, k);
    meta[1] = make_int4(it.z, it.w, (first ? 1 : 0) | (last ? 2 : 0) | (data ? 0 : 4), 0);
    prod[0] = it;
    prod[1] = make_int4(run.x, k + 1, run.z, last ? 0 : 1);
  }
  if (!data) {
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
    return;
  }
  int lo[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int cv = lane + 32 * q, v = k * p.nc + cv;
    lo[q] = cv < p.ncs && v < p.nv ? __ldg(p.lo + (size_t)it.x * p.nv + v) : 0;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int cv = lane + 32 * q;
    if (cv >= p.ncs) continue;
    const int cb = (int)slots + (cv * W - (FULL ? 0 : lo[q])) * SB;
    s_cb[cv] = cb;
#pragma unroll
    for (int c = 1; c < CB; ++c)
      if (cv >= c) s_cb[c * kCbInts + cv - c] = cb;
  }
  __syncwarp();
  if (lane == 0) mbar_expect(bar, p.chunk_bytes + p.expect_extra);
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int cv = lane + 32 * q;
    if (cv < p.ncs) {
      // the slots of virtual channels are the zero row, and a window wholly
      // outside the record lies in the zero margins
      const int i = k * p.nc + cv + p.u0;
      const long long row = i >= 0 && i < p.n_elem ? 1 + (long long)run.x * p.n_elem + i : 0;
      // (even slots: 8-byte slots start on 16-byte boundaries)
      const int x = p.slot_margin + max(-p.slot_margin, min(lo[q], (p.n_samples + 1) & ~1));
      bulk_copy(slots + cv * W * SB, p.slots_dev + (row * p.slot_pitch + x) * SB, W * SB, bar);
    }
  }
}

// Counts the warp out of the stage's chunk; the last warp out loads the chunk
// after next into it.  The arrival count's acquire is lane 0's: a shuffle orders
// no memory, so the warp synchronises before every lane of it reads the running
// item, which another warp wrote.
template <bool FULL, int SB, int NF>
__device__ __forceinline__ void leave_chunk(const BfParams& p, unsigned char* smem, uint32_t sbase,
                                            int stage, int lane, int nwarps) {
  __syncwarp();
  int before = 0;
  if (lane == 0) before = count_arrival(sbase + kPipeCountOff + 4 * stage);
  if (__shfl_sync(0xffffffffu, before, 0) != nwarps - 1) return;
  if (lane == 0) reinterpret_cast<int*>(smem + kPipeCountOff)[stage] = 0;
  __syncwarp();
  produce<FULL, SB, NF, false>(p, smem, sbase, stage, lane);
  __syncwarp();
}

template <int K, bool APOD, bool COMP, bool FULL, int MODE>
__global__ void __launch_bounds__(256, pipe_blocks(K, APOD, COMP, FULL)) k_bf_pipe(const __grid_constant__ BfParams p) {
  constexpr int NA = NAcc<K>::value, SB = slot_bytes(MODE);
  constexpr int PK = packed_sums(K, APOD, COMP, FULL, MODE);
  extern __shared__ __align__(128) unsigned char smem[];
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  auto full_bar = [&](int s) { return sbase + kPipeFullOff + 8 * s; };

  wait_previous();
  if constexpr (COMP) {
    if (warp == 0) {  // the whole warp allocates; the address lands in shared memory
      tmem_alloc(sbase + kPipeTmemOff, p.tmem_cols);
      tc_fence_before_sync();
    }
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(full_bar(s));
      reinterpret_cast<int*>(smem + kPipeCountOff)[s] = 0;
    }
    *reinterpret_cast<int*>(smem + kPipeStopOff) = 0;
    reinterpret_cast<int4*>(smem + kPipeProdOff)[1] = make_int4(0, 0, 0, 0);
  }
  __syncthreads();
  int stage = 0, phase = 0;
  if (warp == 0) {
    produce<FULL, SB, 2, true>(p, smem, sbase, 0, lane);
    __syncwarp();
    for (int s = 1; s < p.stages; ++s) {
      produce<FULL, SB, 2, false>(p, smem, sbase, s, lane);
      __syncwarp();
    }
  }
  {
#ifdef PA_CHECK_BOUNDS
    const int slots_lo = (int)sbase + kPipeSlotOff;
    const int slots_hi = slots_lo + (p.stages * p.ncs * p.window - 1) * SB;
#endif
    uint32_t tmem = 0;
    if constexpr (COMP) {
      tc_fence_after_sync();
      tmem = *reinterpret_cast<const volatile uint32_t*>(smem + kPipeTmemOff) +
             ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * NA * 16);
    }
    constexpr bool LAZY = APOD;
    constexpr bool kRing = one_entry_set(K, APOD, COMP, MODE);
    // Lanes -> (warp slot, depth row), as in the one-frame kernel; a 128-bit
    // shared load is served 8 lanes at a time, so with 8-row groups those are
    // 4 rows of 2 neighbouring slots, whose delays span fewer slots.
    const int lr_log2 = p.lane_rows_log2;
    const int sg = nwarps >> (5 - lr_log2);  // slot groups of the block
    int sw = lane >> lr_log2, zl = lane & ((1 << lr_log2) - 1);
    if (lr_log2 == 3) {
      sw = ((lane >> 2) & 1) | ((lane >> 3) & 2);
      zl = (lane & 3) | ((lane >> 1) & 4);
    }
    const int sl0 = ((warp % sg) << (5 - lr_log2)) + sw;
    const int rgrp = warp / sg;
    const int zr = (rgrp << lr_log2) + zl;
    const size_t fhalf = (size_t)32 * p.slots * 2;
    const size_t fstep = 2 * fhalf;
    const size_t tstep = (size_t)p.nz_pad * 4;

    float acc[2][kC][NA];
    int fold = 0;
    bool tsum_live = false, have = false;
    int jt = 0, z = 0;
    int2 ur = make_int2(p.u0, p.u0 + p.steps);
    size_t tblock = 0;  // next block's entries (table_index), or the full table's base
    int2 ea[kC], eb[kC];
    float wa[kC], wb[kC];
    for (;;) {
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(full_bar(stage), phase))) {
        if (lane == 0) {
          if (atomicExch(reinterpret_cast<int*>(smem + kPipeStopOff), 1) == 0) report_timeout(p);
        }
        break;
      }
      const int4* meta = reinterpret_cast<const int4*>(smem + kPipeMetaOff + 32 * stage);
      const int4 m0 = meta[0], m1 = meta[1];
      if (m0.x < 0) break;
      const int tile_id = m0.x, frame = m0.y, k = m0.w;
      const bool first = m1.z & 1, last = m1.z & 2, data = !(m1.z & 4);
      if (first) {
        const int sl = m0.z * nwarps + sl0;
        const int r_m = sl % p.m, g = sl / p.m;
        jt = m1.x * p.tile_x + g * p.m * kC + r_m;
        z = m1.y * p.tile_z + zr;
        if constexpr (APOD) ur = __ldg(p.urange + (size_t)tile_id * p.slots + sl);
        if constexpr (FULL) {
          tblock = (size_t)tile_id * (p.steps + 3) * fstep +
                   (((size_t)rgrp * p.slots + sl) * (1 << lr_log2) + zl) * 2;
        } else {
          tblock = (((size_t)r_m * p.tgroups + ((jt - r_m) / p.m + p.steps) / 4) * (p.nz_pad >> 3) +
                    (z >> 3)) * 32 + (z & 7) * 2 - (size_t)((ur.x - p.u0) >> 2) * tstep;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int c = 0; c < kC; ++c)
#pragma unroll
            for (int q = 0; q < NA; ++q) acc[h][c][q] = 0.f;
        if constexpr (COMP && !LAZY) {
          const float z8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int q = 0; q < NA * 2; ++q) tmem_st8(tmem + 8 * q, z8);
        }
        fold = 0;
        tsum_live = !LAZY;
        have = false;
      }
      const int* s_cb = reinterpret_cast<const int*>(smem + kPipeCbOff + stage * kCbInts * 4);
      const int cu0 = p.u0 + k * p.nc;
      int u = max(cu0, ur.x);
      const int u_end = data ? min(cu0 + p.nc, ur.y) : u;
      auto load_cb = [&](int (&cb)[2 * kC], int uu) {
        // channel bases of channels uu .. uu + 2kC - 2 (uu - cu0 is a multiple of 4)
        const int4* cbv = reinterpret_cast<const int4*>(s_cb + (uu - cu0));
        const int4 c0 = cbv[0], c1 = cbv[1];
        cb[0] = c0.x; cb[1] = c0.y; cb[2] = c0.z; cb[3] = c0.w;
        cb[4] = c1.x; cb[5] = c1.y; cb[6] = c1.z; cb[7] = c1.w;
      };
      auto checked = [&](int addr) {
#ifdef PA_CHECK_BOUNDS
        if (addr < slots_lo || addr > slots_hi) {
          atomicOr(p.err, 2);
          return slots_lo;
        }
#endif
        return addr;
      };
      auto kahan = [&]() {
        if constexpr (COMP) {
          if (++fold == kFoldBlocks) {
            fold_tmem2<NA, LAZY>(acc, tmem, !tsum_live);
            tsum_live = true;
            fold = 0;
          }
        }
      };
      if constexpr (FULL) {
        // Entries [and weights] of the kC pairs of step uu: two 16-byte loads.
        auto load_step = [&](int2 (&e)[kC], float (&w)[kC], int uu) {
          const size_t o = tblock + (size_t)(uu - p.u0) * fstep;
#ifdef PA_CHECK_BOUNDS
          if (o + fhalf + 2 > (size_t)(tile_id + 1) * (p.steps + 3) * fstep) atomicOr(p.err, 1);
#endif
          const int4 q0 = __ldg(reinterpret_cast<const int4*>(p.ftab + o));
          const int4 q1 = __ldg(reinterpret_cast<const int4*>(p.ftab + o + fhalf));
          e[0] = make_int2(q0.x, q0.y);
          e[1] = make_int2(q0.z, q0.w);
          e[2] = make_int2(q1.x, q1.y);
          e[3] = make_int2(q1.z, q1.w);
          if constexpr (APOD) {
            const float2 w0 = __ldg(reinterpret_cast<const float2*>(p.wtab + o));
            const float2 w1 = __ldg(reinterpret_cast<const float2*>(p.wtab + o + fhalf));
            w[0] = w0.x;
            w[1] = w0.y;
            w[2] = w1.x;
            w[3] = w1.y;
          }
        };
        if (u < u_end && !have) {  // steps run on across chunks, two loaded ahead
          load_step(ea, wa, u);
          load_step(eb, wb, u + 1);
          have = true;
        }
        for (; u < u_end; u += kC) {
          int cb[2 * kC];
          load_cb(cb, u);
#pragma unroll
          for (int tt = 0; tt < kC; ++tt) {
            // entries of the step after next (the padding steps at the end of
            // the tile's table keep these loads in bounds)
            int2 e2[kC];
            float w2[kC];
            load_step(e2, w2, u + tt + 2);
#pragma unroll
            for (int c = 0; c < kC; ++c)
              slot_pair<K, MODE, APOD, PK>(acc[0][c], acc[1][c], checked(cb[tt + c] + ea[c].x * (SB / 8)),
                                       __int_as_float(ea[c].y), APOD ? wa[c] : 0.f);
#pragma unroll
            for (int c = 0; c < kC; ++c) {
              ea[c] = eb[c];
              eb[c] = e2[c];
              if constexpr (APOD) {
                wa[c] = wb[c];
                wb[c] = w2[c];
              }
            }
          }
          kahan();
        }
      } else {
        // Table entries (n0, a) [and weight] of the next block's steps: two
        // halves of two steps (table_index).
        auto load_half = [&](int2 (&ee)[kC], float (&ww)[kC], int h) {
          const size_t o = tblock + 16 * h;
#ifdef PA_CHECK_BOUNDS
          if (o + 2 > (size_t)p.m * p.tgroups * tstep) atomicOr(p.err, 1);
#endif
          const int4 e = load_entries16(p.table + o);
          ee[2 * h] = make_int2(e.x, e.y);
          ee[2 * h + 1] = make_int2(e.z, e.w);
          if constexpr (APOD) {
            const float2 w = __ldg(reinterpret_cast<const float2*>(p.wtab + o));
            ww[2 * h] = w.x;
            ww[2 * h + 1] = w.y;
          }
        };
        auto load_entries = [&](int2 (&ee)[kC], float (&ww)[kC]) {
          load_half(ee, ww, 0);
          load_half(ee, ww, 1);
          tblock -= tstep;
        };
        auto block = [&](const int2 (&ee)[kC], const float (&ww)[kC], int uu) {
          int cb[2 * kC];
          load_cb(cb, uu);
#pragma unroll
          for (int tt = 0; tt < kC; ++tt) {
            const int off = ee[tt].x * (SB / 8);
#pragma unroll
            for (int c = 0; c < kC; ++c)
              slot_pair<K, MODE, APOD, PK>(acc[0][c], acc[1][c], checked(cb[tt + c] + off),
                                       __int_as_float(ee[tt].y), APOD ? ww[tt] : 0.f);
          }
          kahan();
        };
        // The next block's entries are loaded one block ahead, also across
        // chunks of an item: into the registers of the entries just used
        // (kRing), or two blocks per iteration with two register sets.
        if (u < u_end && !have) {
          load_entries(ea, wa);
          have = true;
        }
        if constexpr (kRing) {
          for (; u < u_end; u += kC) {
            int cb[2 * kC];
            load_cb(cb, u);
            const bool more = u + kC < ur.y;
#pragma unroll
            for (int tt = 0; tt < kC; ++tt) {
              const int off = ea[tt].x * (SB / 8);
              const float a = __int_as_float(ea[tt].y), weight = APOD ? wa[tt] : 0.f;
              if ((tt & 1) && more) load_half(ea, wa, tt >> 1);
#pragma unroll
              for (int c = 0; c < kC; ++c)
                slot_pair<K, MODE, APOD, PK>(acc[0][c], acc[1][c], checked(cb[tt + c] + off), a, weight);
            }
            tblock -= tstep;
            kahan();
          }
        } else {
        for (; u < u_end; u += 2 * kC) {
          if (u + kC < ur.y) load_entries(eb, wb);
          block(ea, wa, u);
          if (u + kC >= u_end) {
#pragma unroll
            for (int tt = 0; tt < kC; ++tt) {
              ea[tt] = eb[tt];
              if constexpr (APOD) wa[tt] = wb[tt];
            }
            break;
          }
          if (u + 2 * kC < ur.y) load_entries(ea, wa);
          block(eb, wb, u + kC);
        }
        }
      }
      leave_chunk<FULL, SB, 2>(p, smem, sbase, stage, lane, nwarps);
      if (++stage == p.stages) {
        stage = 0;
        phase ^= 1;
      }
      if (!last) continue;
      if (reinterpret_cast<const volatile int4*>(smem + kPipeProdOff)[1].w == 2) launch_next();

      if constexpr (COMP) {
        if (tsum_live) final_tmem2<NA>(acc, tmem);
      }
      // ---- epilogue and store
      const size_t plane = (size_t)p.nx * p.nz;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (frame + h >= p.n_frames) break;  // an odd launch's last item
        const size_t fbase = (size_t)(frame + h) * p.planes * plane;
#pragma unroll
        for (int c = 0; c < kC; ++c) {
          const int j = jt + p.m * c;
          if (j < p.nx && z < p.nz) {
            float das, dmas, ho;
            combine<K>(acc[h][c], p.ek_top, das, dmas, ho);
            const size_t px = fbase + (size_t)j * p.nz + z;
            if (p.plane_das >= 0) p.out[px + (size_t)p.plane_das * plane] = das;
            if (p.plane_dmas >= 0) p.out[px + (size_t)p.plane_dmas * plane] = dmas;
            if (p.plane_ho >= 0) p.out[px + (size_t)p.plane_ho * plane] = ho;
          }
        }
      }
    }
  }
  if constexpr (COMP) {  // every thread's TMEM accesses completed before the barrier
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) {
      tc_fence_after_sync();
      tmem_dealloc(*reinterpret_cast<const volatile uint32_t*>(smem + kPipeTmemOff), p.tmem_cols);
    }
  }
}

}  // namespace pa

#define PA_DEFINE_PIPE(K)                                                            \
  namespace pa {                                                                     \
  template <bool FULL>                                                               \
  static const void* pick_pipe_k##K(bool apod, bool comp, bool nearest) {            \
    constexpr PipeMode AN = pipe_mode(K, true, true), PN = pipe_mode(K, false, true); \
    void (*f)(BfParams);                                                             \
    if (apod)                                                                        \
      f = nearest ? (comp ? k_bf_pipe<K, true, true, FULL, AN>                       \
                          : k_bf_pipe<K, true, false, FULL, AN>)                     \
                  : (comp ? k_bf_pipe<K, true, true, FULL, kLinear>                  \
                          : k_bf_pipe<K, true, false, FULL, kLinear>);               \
    else                                                                             \
      f = nearest ? (comp ? k_bf_pipe<K, false, true, FULL, PN>                      \
                          : k_bf_pipe<K, false, false, FULL, PN>)                    \
                  : (comp ? k_bf_pipe<K, false, true, FULL, kLinear>                 \
                          : k_bf_pipe<K, false, false, FULL, kLinear>);              \
    return reinterpret_cast<const void*>(f);                                         \
  }                                                                                  \
  const void* bf_pipe_func_k##K(bool apod, bool comp, bool full, bool nearest) {     \
    return full ? pick_pipe_k##K<true>(apod, comp, nearest)                          \
                : pick_pipe_k##K<false>(apod, comp, nearest);                        \
  }                                                                                  \
  }
