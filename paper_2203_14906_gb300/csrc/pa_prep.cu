// pa_prep.cu -- slots of the two-frame fused kernel, prepared once per launch.
//
// Every (frame pair, channel) row of RF becomes a row of slots (PipeMode in
// pa_bf_pipe.cuh; primes: the second frame): {r[n], r'[n], r[n+1] - r[n],
// r'[n+1] - r'[n]} for linear interpolation, {r[n], r'[n], y, y'} with the base
// root y of the sample or {r[n], r'[n]} for nearest samples.  Samples past the
// record read as zero; the margins around the record and the row of zeros were
// cleared when the plan was built; samples no window holds are left out.  The
// partner of an odd launch's last frame is the frame itself (its results are not
// stored).  The pass also sets the launch's work counter and clears its maxima.
//
// Bound by the slot writes: 16 bytes per sample and frame pair against 8 read
// (FP32); a thread takes slots a block's width apart, so that a warp's stores are
// contiguous.
#include <algorithm>

#include "pa_bf_pipe.cuh"

namespace pa {
namespace {

__device__ __forceinline__ float prep_root(int order, float s) {
  switch (order) {
    case 3: return base_root<3>(s);
    case 4: return base_root<4>(s);
  }
  return base_root<5>(s);
}

constexpr int kPerThread = 2;

// Slots of one frame each: {r[n], r[n+1] - r[n]}, or {r[n], 0} for nearest
// samples (the same fused multiply-add then gives r[n]).
template <int DT>
__global__ void __launch_bounds__(256) k_prep1(const PrepParams p) {
  launch_next();
  wait_previous();
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < p.n_zero; i += blockDim.x) p.zero[i] = i ? 0 : p.counter0;
  const int row = blockIdx.x / p.blocks_per_row;  // frame * N + channel
  const int part = blockIdx.x - row * p.blocks_per_row;
  const size_t a0 = (size_t)row * (size_t)p.n_samples;
  float2* dst = reinterpret_cast<float2*>(p.slots) + (size_t)(1 + row) * p.pitch + p.margin;
#pragma unroll
  for (int q = 0; q < kPerThread; ++q) {
    const int n = p.n_lo + (part * kPerThread + q) * 256 + threadIdx.x;
    if (n >= p.n_hi) return;
    const float a = rf_load<DT>(p.rf, a0 + n);
    float d = 0.f;
    if (p.mode == kLinear) d = (n + 1 < p.n_samples ? rf_load<DT>(p.rf, a0 + n + 1) : 0.f) - a;
    dst[n] = make_float2(a, d);
  }
}

template <int DT>
__global__ void __launch_bounds__(256) k_prep(const PrepParams p) {
  launch_next();
  wait_previous();
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < p.n_zero; i += blockDim.x) p.zero[i] = i ? 0 : p.counter0;
  const int row = blockIdx.x / p.blocks_per_row;  // frame pair * N + channel
  const int part = blockIdx.x - row * p.blocks_per_row;
  const int fg = row / p.n_elem;
  const int i = row - fg * p.n_elem;
  const size_t a0 = ((size_t)(2 * fg) * p.n_elem + i) * (size_t)p.n_samples;
  const size_t b0 =
      a0 + (2 * fg + 1 < p.n_frames ? (size_t)p.n_elem * (size_t)p.n_samples : (size_t)0);
  const size_t dst = (size_t)(1 + row) * p.pitch + p.margin;
#pragma unroll
  for (int q = 0; q < kPerThread; ++q) {
    const int n = p.n_lo + (part * kPerThread + q) * 256 + threadIdx.x;
    if (n >= p.n_hi) return;
    const float a = rf_load<DT>(p.rf, a0 + n), b = rf_load<DT>(p.rf, b0 + n);
    if (p.mode == kNearest) {
      reinterpret_cast<float2*>(p.slots)[dst + n] = make_float2(a, b);
      continue;
    }
    float4 v;
    if (p.mode == kNearestRoots) {
      v = make_float4(a, b, prep_root(p.order, a), prep_root(p.order, b));
    } else {
      const bool in = n + 1 < p.n_samples;
      v = make_float4(a, b, (in ? rf_load<DT>(p.rf, a0 + n + 1) : 0.f) - a,
                      (in ? rf_load<DT>(p.rf, b0 + n + 1) : 0.f) - b);
    }
    reinterpret_cast<float4*>(p.slots)[dst + n] = v;
  }
}

}  // namespace

int pipe_slot_mode(int order, bool apod, bool nearest) { return pipe_mode(order, apod, nearest); }
int pipe_slot_bytes(int mode) { return slot_bytes(mode); }

void prep_spec(PrepParams* p, LaunchSpec* s) {
  const int per_block = 256 * kPerThread;
  p->blocks_per_row = std::max(1, (p->n_hi - p->n_lo + per_block - 1) / per_block);
  if (p->nf == 1) {
    s->func = p->rf_dtype == PA_RF_F32    ? reinterpret_cast<const void*>(k_prep1<PA_RF_F32>)
              : p->rf_dtype == PA_RF_BF16 ? reinterpret_cast<const void*>(k_prep1<PA_RF_BF16>)
                                          : reinterpret_cast<const void*>(k_prep1<PA_RF_F16>);
    s->grid = dim3((unsigned)((long long)p->n_frames * p->n_elem * p->blocks_per_row));
    s->block = dim3(256);
    s->smem = 0;
    return;
  }
  s->func = p->rf_dtype == PA_RF_F32    ? reinterpret_cast<const void*>(k_prep<PA_RF_F32>)
            : p->rf_dtype == PA_RF_BF16 ? reinterpret_cast<const void*>(k_prep<PA_RF_BF16>)
                                        : reinterpret_cast<const void*>(k_prep<PA_RF_F16>);
  s->grid = dim3((unsigned)((long long)((p->n_frames + 1) / 2) * p->n_elem * p->blocks_per_row));
  s->block = dim3(256);
  s->smem = 0;
}

}  // namespace pa
