// pa_bf_fine.cuh -- the fine-grained form of the fused beamforming kernel, for
// launches too small to fill the GPU with 4-pixel threads.
//
// The one-frame form gives a thread four pixels, so one small frame is a few
// hundred warps: a 128 x 128 image runs in 32 blocks of 4 warps on 152 SMs, each
// warp walking 67 steps x 4 pixels one after the other behind two staging
// passes.  Here a thread takes one (or two) of the four: the same tiles,
// tables, channel steps and per-pixel arithmetic in the same order (the bits
// are the one-frame form's), four (two) times the warps.  Bound by latency: a
// warp's chain of table load, shared load and MUFU per step, so what counts is
// warps in flight, not the table entry that now serves one pair instead of
// four.  Chunks come as in the two-frame form, by bulk copies from slots
// prepared for the launch ({r, d} per sample; the pass takes the place of the
// clearing kernel) into two buffers; a tile's channel windows are copied once
// per block of up to 16 warps.  Kahan totals (one pixel a thread) are kept beside
// the sums (2 x 5 at k = 3), in registers as far as the 64 of two blocks a SM go:
// they spill 6-36 bytes at k = 3 and 250 at k = 8, outside the channel loop's
// inner steps (the totals are touched every 64).  These variants still take
// 0.65-0.9 of the one-frame form's time where pick_form sends them.
// Measured on GB300 (RAW images, one-frame form -> this): one frame of 128 x 128,
// 64 channels, k = 3 16.7 -> 14.6 us; one frame of 400 x 512, 128 channels, full
// table 84.5 -> 67.4, with two pixels a thread 55.8; one frame of 291 x 333, 97
// channels of 1501 samples, k = 4 25.0 -> 20.8.  The lines are in fine_pays.
#pragma once

#include "pa_bf_pipe.cuh"

namespace pa {

// Kahan fold of the partial sums into register totals, as kahan_fold_tmem does.
template <int PX, int NA>
__device__ __forceinline__ void fold_regs(float (&acc)[PX][NA], float (&tot)[PX][NA],
                                          float (&comp)[PX][NA]) {
#pragma unroll
  for (int c = 0; c < PX; ++c)
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const float y = acc[c][q] - comp[c][q];
      const float s = tot[c][q] + y;
      comp[c][q] = (s - tot[c][q]) - y;
      tot[c][q] = s;
      acc[c][q] = 0.f;
    }
}

// PX of a thread's kC pixels per thread: warp (cpart, row group, slot group)
// of a tile takes pixels cpart PX .. + PX - 1 of its slots.
template <int K, bool APOD, bool COMP, bool FULL, int PX>
__global__ void __launch_bounds__(512, 2) k_bf_fine(const __grid_constant__ BfParams p) {
  constexpr int NA = NAcc<K>::value;
  extern __shared__ __align__(128) unsigned char smem[];
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  auto full_bar = [&](int s) { return sbase + kPipeFullOff + 8 * s; };
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(full_bar(s));
      reinterpret_cast<int*>(smem + kPipeCountOff)[s] = 0;
    }
    *reinterpret_cast<int*>(smem + kPipeStopOff) = 0;
    reinterpret_cast<int4*>(smem + kPipeProdOff)[1] = make_int4(0, 0, 0, 0);
  }
  wait_previous();
  __syncthreads();
  int stage = 0, phase = 0;
  if (warp == 0) {
    produce<FULL, 8, 1, true>(p, smem, sbase, 0, lane);
    __syncwarp();
    for (int s = 1; s < p.stages; ++s) {
      produce<FULL, 8, 1, false>(p, smem, sbase, s, lane);
      __syncwarp();
    }
  }
#ifdef PA_CHECK_BOUNDS
  const int slots_lo = (int)sbase + kFineSlotOff;
  const int slots_hi = slots_lo + (p.stages * p.ncs * p.window - 1) * 8;
#endif
  const int lr_log2 = p.lane_rows_log2;
  const int sgn = p.slots >> (5 - lr_log2);  // slot groups of a tile
  const int zl = lane & ((1 << lr_log2) - 1);
  const size_t fhalf = (size_t)32 * p.slots * 2;
  const size_t fstep = 2 * fhalf;
  const size_t tstep = (size_t)p.nz_pad * 4;

  float acc[PX][NA], tot[COMP ? PX : 1][NA], comp[COMP ? PX : 1][NA];
  int fold = 0, cp = 0, jt = 0, z = 0;
  bool have = false, folded = false;
  int2 ur = make_int2(p.u0, p.u0 + p.steps);
  size_t tblock = 0;
  int2 ea[kC];
  float wa[kC];
  for (;;) {
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(full_bar(stage), phase))) {
      if (lane == 0 && atomicExch(reinterpret_cast<int*>(smem + kPipeStopOff), 1) == 0)
        report_timeout(p);
      break;
    }
    const int4* meta = reinterpret_cast<const int4*>(smem + kPipeMetaOff + 32 * stage);
    const int4 m0 = meta[0], m1 = meta[1];
    if (m0.x < 0) break;
    const int tile_id = m0.x, frame = m0.y, k = m0.w;
    const bool first = m1.z & 1, last = m1.z & 2, data = !(m1.z & 4);
    if (first) {
      const int gw = m0.z * nwarps + warp;  // warp of the tile
      const int q = gw / sgn, rows = 32 >> lr_log2;
      const int sl = ((gw - q * sgn) << (5 - lr_log2)) + (lane >> lr_log2);
      const int rgrp = q % rows;
      cp = q / rows;
      const int r_m = sl % p.m, g = sl / p.m;
      jt = m1.x * p.tile_x + g * p.m * kC + r_m;
      z = m1.y * p.tile_z + (rgrp << lr_log2) + zl;
      if constexpr (APOD) ur = __ldg(p.urange + (size_t)tile_id * p.slots + sl);
      if constexpr (FULL) {
        tblock = (size_t)tile_id * (p.steps + 3) * fstep +
                 (((size_t)rgrp * p.slots + sl) * (1 << lr_log2) + zl) * 2 +
                 (size_t)(cp * PX >> 1) * fhalf + (PX == 1 ? cp & 1 : 0);
      } else {
        tblock = (((size_t)r_m * p.tgroups + ((jt - r_m) / p.m + p.steps) / 4) * (p.nz_pad >> 3) +
                  (z >> 3)) * 32 + (z & 7) * 2 - (size_t)((ur.x - p.u0) >> 2) * tstep;
      }
#pragma unroll
      for (int c = 0; c < PX; ++c)
#pragma unroll
        for (int a = 0; a < NA; ++a) {
          acc[c][a] = 0.f;
          if constexpr (COMP) tot[c][a] = comp[c][a] = 0.f;
        }
      fold = 0;
      have = folded = false;
    }
    // channel bases, shifted by the warp's first pixel (see produce)
    const int* s_cb = reinterpret_cast<const int*>(smem + kPipeCbOff + stage * kC * kCbInts * 4) +
                      cp * PX * kCbInts;
    const int cu0 = p.u0 + k * p.nc;
    int u = max(cu0, ur.x);
    const int u_end = data ? min(cu0 + p.nc, ur.y) : u;
    auto checked = [&](int addr) {
#ifdef PA_CHECK_BOUNDS
      if (addr < slots_lo || addr > slots_hi) {
        atomicOr(p.err, 2);
        return slots_lo;
      }
#endif
      return addr;
    };
    auto pair = [&](int c, int addr, float a, float w) {
      float r, d;
      asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r), "=f"(d) : "r"(checked(addr)));
      float s = fmaf(a, d, r);  // nearest-sample plans: a = d = 0
      if constexpr (APOD) s *= w;
      pair_update<K>(acc[c], s);
    };
    // Entries of the block of steps at uu: lattice, one per step; full table,
    // the first pixel's here and the second's in e1.
    auto load_block = [&](int2 (&e)[kC], int2 (&e1)[kC], float (&w)[kC], float (&w1)[kC], int uu) {
      (void)e1;
      (void)w1;
      if constexpr (FULL) {
        const size_t o = tblock + (size_t)(uu - p.u0) * fstep;
#pragma unroll
        for (int tt = 0; tt < kC; ++tt) {
          if constexpr (PX == 2) {
            const int4 v = __ldg(reinterpret_cast<const int4*>(p.ftab + o + tt * fstep));
            e[tt] = make_int2(v.x, v.y);
            e1[tt] = make_int2(v.z, v.w);
            if constexpr (APOD) {
              const float2 x = __ldg(reinterpret_cast<const float2*>(p.wtab + o + tt * fstep));
              w[tt] = x.x;
              w1[tt] = x.y;
            }
          } else {
            e[tt] = __ldg(p.ftab + o + tt * fstep);
            if constexpr (APOD) w[tt] = __ldg(p.wtab + o + tt * fstep);
          }
        }
      } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const size_t o = tblock + 16 * h;
          const int4 v = __ldg(reinterpret_cast<const int4*>(p.table + o));
          e[2 * h] = make_int2(v.x, v.y);
          e[2 * h + 1] = make_int2(v.z, v.w);
          if constexpr (APOD) {
            const float2 x = __ldg(reinterpret_cast<const float2*>(p.wtab + o));
            w[2 * h] = x.x;
            w[2 * h + 1] = x.y;
          }
        }
        tblock -= tstep;
      }
    };
    for (; u < u_end; u += kC) {
      int2 e[kC], e1[kC];
      float w[kC], w1[kC];
      if constexpr (FULL) {
        load_block(e, e1, w, w1, u);
      } else {
        if (!have) {
          load_block(ea, e1, wa, w1, u);
          have = true;
        }
#pragma unroll
        for (int tt = 0; tt < kC; ++tt) {
          e[tt] = ea[tt];
          if constexpr (APOD) w[tt] = wa[tt];
        }
        if (u + kC < ur.y) load_block(ea, e1, wa, w1, u + kC);
      }
      int cb[kC + PX - 1];
      {
        const int4 v = *reinterpret_cast<const int4*>(s_cb + (u - cu0));
        cb[0] = v.x; cb[1] = v.y; cb[2] = v.z; cb[3] = v.w;
        if constexpr (PX == 2) cb[4] = s_cb[u - cu0 + 4];
      }
#pragma unroll
      for (int tt = 0; tt < kC; ++tt)
#pragma unroll
        for (int c = 0; c < PX; ++c) {
          const int2 en = FULL && c ? e1[tt] : e[tt];
          pair(c, cb[tt + c] + en.x, __int_as_float(en.y),
               APOD ? (FULL && c ? w1[tt] : w[tt]) : 0.f);
        }
      if constexpr (COMP) {
        if (++fold == kFoldBlocks) {
          fold_regs<PX, NA>(acc, tot, comp);
          folded = true;
          fold = 0;
        }
      }
    }
    leave_chunk<FULL, 8, 1>(p, smem, sbase, stage, lane, nwarps);
    if (++stage == p.stages) {
      stage = 0;
      phase ^= 1;
    }
    if (!last) continue;
    if (reinterpret_cast<const volatile int4*>(smem + kPipeProdOff)[1].w == 2) launch_next();
    if constexpr (COMP) {
      if (folded) {
#pragma unroll
        for (int c = 0; c < PX; ++c)
#pragma unroll
          for (int a = 0; a < NA; ++a) {
            const float y = acc[c][a] - comp[c][a];
            const float s = tot[c][a] + y;
            acc[c][a] = s - ((s - tot[c][a]) - y);
          }
      }
    }
    const size_t plane = (size_t)p.nx * p.nz;
    const size_t fbase = (size_t)frame * p.planes * plane;
#pragma unroll
    for (int c = 0; c < PX; ++c) {
      const int j = jt + p.m * (cp * PX + c);
      if (j < p.nx && z < p.nz) {
        float das, dmas, ho;
        combine<K>(acc[c], p.ek_top, das, dmas, ho);
        const size_t px = fbase + (size_t)j * p.nz + z;
        if (p.plane_das >= 0) p.out[px + (size_t)p.plane_das * plane] = das;
        if (p.plane_dmas >= 0) p.out[px + (size_t)p.plane_dmas * plane] = dmas;
        if (p.plane_ho >= 0) p.out[px + (size_t)p.plane_ho * plane] = ho;
      }
    }
  }
}

}  // namespace pa

// (Null where no launch takes the form: fine_limits.)
#define PA_DEFINE_FINE(K)                                                          \
  namespace pa {                                                                   \
  template <bool FULL>                                                             \
  static const void* pick_fine_k##K(bool apod, bool comp, int px) {                \
    void (*f)(BfParams) = nullptr;                                                 \
    if (px == 1 && !comp)                                                          \
      f = apod ? k_bf_fine<K, true, false, FULL, 1> : k_bf_fine<K, false, false, FULL, 1>; \
    if constexpr (!FULL || K < 8)                                                  \
      if (px == 1 && comp)                                                         \
        f = apod ? k_bf_fine<K, true, true, FULL, 1> : k_bf_fine<K, false, true, FULL, 1>; \
    if constexpr (K <= 5 && (FULL || K >= 3))                                      \
      if (px == 2 && !comp)                                                        \
        f = apod ? k_bf_fine<K, true, false, FULL, 2> : k_bf_fine<K, false, false, FULL, 2>; \
    return reinterpret_cast<const void*>(f);                                       \
  }                                                                                \
  const void* bf_fine_func_k##K(bool apod, bool comp, bool full, int px) {         \
    return full ? pick_fine_k##K<true>(apod, comp, px) : pick_fine_k##K<false>(apod, comp, px); \
  }                                                                                \
  }
