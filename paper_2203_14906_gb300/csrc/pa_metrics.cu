// pa_metrics.cu -- image-quality metrics of Section 3 (SNR Eq. 10, CR
// Eq. 11, gCNR Eq. 12, lateral FWHM) on device-resident images.
//
// Region membership is decided once per image column: the pixels of a disc,
// rectangle or annulus in one column form one row interval (minus an inner
// interval for the annulus), found with the exact FP64 test, so the passes
// read member pixels only.  Then one of two paths; results do not depend on
// scheduling in either.
//
// k_m_pair, when the members of every ROI pair fit in shared memory: one
// block per (image, ROI pair) fetches the pair's members once (4 B
// asynchronous copies, all in flight together) and does everything else from
// there: sums, maximum, deviations, histograms, the FWHM walk and the record.
// The pixel indices of a region's members are listed once per call, by
// k_m_members, so no image walks columns.  What bounds it is the chain of its
// phases within a block, not the memory (14 KB a pair).  FP64 instructions run
// at 2 lanes per clock and SM here, 1/64 of FP32, so the sums are kept as
// three floats each by exact additions (72 bits, more than a double) and
// become doubles once per region; the largest error of sigma_out against 64
// bits fell from 3.4e-16 to 1.8e-16 of it.  Device time, this path against the
// general one: 96 images x 10 pairs of 3600 pixels 41 against 180 us, 96 x 16
// of 24000 199 / 604, one image and one pair of 700 pixels 19 / 53.  At the
// limit of 51200 values the two meet for few pairs (45000 values: 50 / 72 us
// for one pair, 127 / 373 for 512).
//
// The general path, for larger regions.  Work is split into "slots": one slot
// is one region (target or background) of one ROI pair on one image.  Each
// slot's bounding box of pixels is cut into G chunks, one thread block per
// chunk, so large regions spread over the whole GPU.  Reductions are written
// per block and summed in block order afterwards.  Launches:
//   pass 1   count, sum and the largest value (with its pixel) per block
//   reduce   per slot: count, mean, maximum
//   pass 2   per block: sum of squared deviations from the slot's mean; the
//            256-bin amplitude histogram (integer counts, exact) per slot
//   final    one thread per ROI pair: Eqs. 10-12, and the FWHM walk along
//            the row of the target maximum
// The bytes moved are 2 x 4 B per member pixel, plus the row walks.
#include <math.h>

#include <cmath>

#include <algorithm>
#include <vector>

#include "pa_internal.cuh"
#include "pa_regions.h"

namespace {

constexpr int kBins = 256;
constexpr int kThreads = 256;
constexpr int kMaxChunks = 64;
// ROI pairs per launch sequence: bounds the histogram scratch to
// 2 x 256 x 4 B x 16384 = 32 MiB.
constexpr long long kPairsPerLaunch = 16384;

struct MRegion {
  int shape;
  int j0, j1, l0, l1;  // bounding box of pixel indices, [j0, j1) x [l0, l1)
  long long col0;      // first entry of this region's columns in the range table
  long long pix0;      // first entry of its members in the member list,
  long long pix1;      // and the end of their room
  double xc, zc, a, b;
};

// Member rows of one column: [lo, hi) without [hlo, hhi).
struct ColRange {
  int lo, hi, hlo, hhi;
  // rows before the hole, first row behind it, rows behind it
  __device__ __forceinline__ int before() const {
    return max(0, (hhi > hlo ? min(hi, hlo) : hi) - lo);
  }
  __device__ __forceinline__ int behind_at() const { return max(lo, hhi); }
  __device__ __forceinline__ int behind() const { return hhi > hlo ? max(0, hi - behind_at()) : 0; }
};

// Regions passed with the launch (32 x 80 B of its 4 KB of parameters), so
// that the usual call needs no upload.
constexpr int kParamRegions = 32;
struct RegTable {
  MRegion r[kParamRegions];
};
static_assert(sizeof(RegTable) == kParamRegions * 80 && sizeof(RegTable) < 3500,
              "launch parameters");

struct MGeom {
  int nx, nz, n_roi, chunks;
  long long pair0;  // first (image, roi) pair of this launch sequence
  double x0, z0, dx, dz;
  float rows_per_m;
};

struct Part1 {
  long long cnt;
  double sum;
  unsigned long long key;  // ordered value bits << 32 | ~(pixel index)
};

struct SlotStat {
  long long cnt;
  double mean;
  unsigned long long key;
};

__device__ __forceinline__ unsigned int ordered_bits(float v) {
  const unsigned int u = __float_as_uint(v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float unorder(unsigned int o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

__device__ __forceinline__ float key_value(unsigned long long key) {
  return unorder((unsigned int)(key >> 32));
}

// Pixel-centre membership, FP64 with explicit round-to-nearest operations
// (no fused multiply-add), so the decision matches a plain IEEE evaluation.
// Within one column every test below is monotone in |z - zc|, so each shape's
// member rows form one interval.
__device__ __forceinline__ double px(const MGeom& g, int j) {
  return __dadd_rn(g.x0, __dmul_rn((double)j + 0.5, g.dx));
}
__device__ __forceinline__ double pz(const MGeom& g, int l) {
  return __dadd_rn(g.z0, __dmul_rn((double)l + 0.5, g.dz));
}
// rect: |ez| <= b (the |ex| <= a part is per column); disc of radius rad:
// ex^2 + ez^2 <= rad^2
__device__ __forceinline__ bool row_in(int shape, double ex2, double zc, double rad, const MGeom& g,
                                       int l) {
  const double ez = __dsub_rn(pz(g, l), zc);
  if (shape == PA_REGION_RECT) return fabs(ez) <= rad;
  return __dadd_rn(ex2, __dmul_rn(ez, ez)) <= __dmul_rn(rad, rad);
}

// Interval of rows l in [0, nz) with row_in true, as [lo, hi) (empty: lo == hi).
__device__ int2 row_interval(int shape, double ex2, double zc, double rad, const MGeom& g) {
  // the test is weakest at the row nearest the centre (or at an end of the
  // column when the centre lies beyond it); rounding may move that by one
  double lc = (zc - g.z0) / g.dz - 0.5;
  const float mid = (float)lc;
  lc = fmin(fmax(lc, 0.0), (double)(g.nz - 1));
  int lm = (int)rint(lc), seed = -1;
  for (int d = 0; d <= 2 && seed < 0; ++d) {
    if (lm - d >= 0 && row_in(shape, ex2, zc, rad, g, lm - d)) seed = lm - d;
    else if (lm + d < g.nz && row_in(shape, ex2, zc, rad, g, lm + d)) seed = lm + d;
  }
  if (seed < 0) return make_int2(0, 0);
  // The ends lie about `half` rows from the centre.  The FP32 estimate decides
  // nothing: the exact test is stepped outwards or inwards from it until it
  // changes, in doubling steps (two tests an end as a rule, where a bisection
  // of the column takes log2 nz).
  const double rr = __dmul_rn(rad, rad);
  const float half = g.rows_per_m *
                     (shape == PA_REGION_RECT ? (float)rad : sqrtf(fmaxf((float)(rr - ex2), 0.f)));
  auto in = [&](int l) { return row_in(shape, ex2, zc, rad, g, l); };
  // first member row in [0, seed]
  int lo = 0, hi = seed, e = (int)ceilf(fminf(fmaxf(mid - half, 0.f), (float)seed));
  e = min(max(e, 0), seed);
  if (in(e)) {
    hi = e;
    for (int step = 1; hi > 0; step = min(2 * step, 1 << 20)) {
      const int t = max(hi - step, 0);
      if (!in(t)) {
        lo = t + 1;
        break;
      }
      hi = t;
    }
  } else {
    lo = e + 1;
    for (int step = 1; lo < hi; step = min(2 * step, 1 << 20)) {
      const int t = lo + min(step - 1, hi - lo);
      if (in(t)) {
        hi = t;
        break;
      }
      lo = t + 1;
    }
  }
  while (lo < hi) {
    const int m = (lo + hi) >> 1;
    if (in(m)) hi = m;
    else lo = m + 1;
  }
  const int first = lo;
  // last member row in [seed, nz - 1]
  lo = seed;
  hi = g.nz - 1;
  e = (int)floorf(fminf(fmaxf(mid + half, (float)seed), (float)(g.nz - 1)));
  e = min(max(e, seed), g.nz - 1);
  if (in(e)) {
    lo = e;
    for (int step = 1; lo < g.nz - 1; step = min(2 * step, 1 << 20)) {
      const int t = min(lo, g.nz - 1 - step) + step;
      if (!in(t)) {
        hi = t - 1;
        break;
      }
      lo = t;
    }
  } else {
    hi = e - 1;
    for (int step = 1; lo < hi; step = min(2 * step, 1 << 20)) {
      const int t = max(hi - step + 1, lo);
      if (in(t)) {
        lo = t;
        break;
      }
      hi = t - 1;
    }
  }
  while (lo < hi) {
    const int m = (lo + hi + 1) >> 1;
    if (in(m)) lo = m;
    else hi = m - 1;
  }
  return make_int2(first, lo + 1);
}

// Member rows of column j in the region, or in an annulus's hole.
__device__ __forceinline__ int2 column_interval(const MRegion& R, bool hole, int j, const MGeom& g) {
  const double ex = __dsub_rn(px(g, j), R.xc);
  if (R.shape == PA_REGION_RECT) {
    if (hole || !(fabs(ex) <= R.a)) return make_int2(0, 0);
    return row_interval(PA_REGION_RECT, 0.0, R.zc, R.b, g);
  }
  if (R.shape == PA_REGION_DISC && hole) return make_int2(0, 0);
  // annulus: disc(b) without disc(a)
  return row_interval(PA_REGION_DISC, __dmul_rn(ex, ex), R.zc,
                      R.shape == PA_REGION_DISC || hole ? R.a : R.b, g);
}

// For the general path: one thread per (column, interval), threadIdx.y 0 the
// region, 1 the hole of an annulus.
__global__ void k_m_ranges(MGeom g, const MRegion* regs, ColRange* ranges) {
  const MRegion R = regs[blockIdx.y];
  const int j = R.j0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= R.j1) return;
  reinterpret_cast<int2*>(ranges + R.col0 + (j - R.j0))[threadIdx.y] =
      column_interval(R, threadIdx.y != 0, j, g);
}

// The member pixels of region blockIdx.x, columns and rows ascending, for
// k_m_pair: their number in counts and their indices j * nz + l in list, from
// the region's place pix0 on.
constexpr int kMemberCols = 1024;  // widest region of the list
__global__ void __launch_bounds__(512) k_m_members(MGeom g, const __grid_constant__ RegTable tab,
                                                   int tab_n, const MRegion* regs,
                                                   long long* pix0, int* counts,
                                                   unsigned int* list) {
  __shared__ int2 iv[2][kMemberCols];
  __shared__ int off[kMemberCols + 1];
  const MRegion R = tab_n > 0 ? tab.r[blockIdx.x] : regs[blockIdx.x];
  const int width = R.j1 - R.j0, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int sides = R.shape == PA_REGION_ANNULUS ? 2 : 1;
  const int room = (int)(R.pix1 - R.pix0);
  for (int i = threadIdx.x; i < sides * width; i += blockDim.x) {
    const int hole = i >= width, c = i - (hole ? width : 0);
    iv[hole][c] = column_interval(R, hole, R.j0 + c, g);
  }
  __syncthreads();
  auto range = [&](int c) {
    const int2 v = iv[0][c], h = sides > 1 ? iv[1][c] : make_int2(0, 0);
    return ColRange{v.x, v.y, h.x, h.y};
  };
  if (w == 0) {
    int run = 0;
    for (int c0 = 0; c0 < width; c0 += 32) {
      const int c = c0 + lane;
      int n = 0;
      if (c < width) {
        const ColRange r = range(c);
        n = r.before() + r.behind();
      }
      int inc = n;
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
      }
      if (c < width) off[c] = run + inc - n;
      run += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) {
      counts[blockIdx.x] = min(run, room);  // entries that the list holds, never more
      pix0[blockIdx.x] = R.pix0;
    }
  }
  __syncthreads();
  for (int c = w; c < width; c += (int)(blockDim.x >> 5)) {
    const ColRange r = range(c);
    const int n1 = r.before(), skip = r.behind_at() - n1;
    const int n = min(n1 + r.behind(), room - off[c]);  // (most_members: never cut)
    const unsigned int q = (unsigned)(R.j0 + c) * (unsigned)g.nz;
    unsigned int* const dst = list + R.pix0 + off[c];
    for (int t = lane; t < n; t += 32) dst[t] = q + (unsigned)(t + (t < n1 ? r.lo : skip));
  }
}

struct SlotRef {
  long long pair;  // global (image, roi) pair index
  int side;        // 0 target, 1 background
  const MRegion* reg;
  const float* img;
};

__device__ __forceinline__ SlotRef slot_ref(const MGeom& g, const MRegion* regs,
                                            const float* images, long long slot) {
  SlotRef s;
  s.pair = g.pair0 + slot / 2;
  s.side = (int)(slot & 1);
  const long long img = s.pair / g.n_roi;
  const int roi = (int)(s.pair % g.n_roi);
  s.reg = regs + 2 * roi + s.side;
  s.img = images + (size_t)img * g.nx * g.nz;
  return s;
}

template <typename T, typename Op>
__device__ __forceinline__ T block_reduce(T v, T* sh, Op op) {
  for (int o = 16; o >= 1; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  T r = sh[0];
  for (int i = 1; i < (int)(blockDim.x >> 5); ++i) r = op(r, sh[i]);  // fixed order
  return r;
}

// Calls f(j, l, q) for every member pixel of the block's share of the
// slot's region: warp w of chunk c takes columns c * warps + w, stepping by
// chunks * warps; lanes walk the column's row interval(s).
template <typename F>
__device__ __forceinline__ void for_members(const MGeom& g, const MRegion& r, const ColRange* ranges,
                                            int chunk, F&& f) {
  const int warps = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int width = r.j1 - r.j0;
  for (int c = chunk * warps + w; c < width; c += g.chunks * warps) {
    const ColRange cr = ranges[r.col0 + c];
    const int j = r.j0 + c;
    const long long qj = (long long)j * g.nz;
    const int e1 = cr.hhi > cr.hlo ? min(cr.hi, cr.hlo) : cr.hi;  // rows before the hole
    for (int l = cr.lo + lane; l < e1; l += 32) f(j, l, qj + l);
    if (cr.hhi > cr.hlo)
      for (int l = max(cr.lo, cr.hhi) + lane; l < cr.hi; l += 32) f(j, l, qj + l);
  }
}

__global__ void __launch_bounds__(kThreads) k_m_pass1(MGeom g, const MRegion* regs,
                                                      const ColRange* ranges, const float* images,
                                                      Part1* part) {
  __shared__ long long sh_c[kThreads / 32];
  __shared__ double sh_s[kThreads / 32];
  __shared__ unsigned long long sh_k[kThreads / 32];
  const long long slot = blockIdx.x / g.chunks;
  const int chunk = blockIdx.x % g.chunks;
  const SlotRef s = slot_ref(g, regs, images, slot);
  const MRegion r = *s.reg;
  long long cnt = 0;
  double sum = 0.0;
  unsigned long long key = 0;
  for_members(g, r, ranges, chunk, [&](int, int, long long q) {
    const float v = __ldg(s.img + q);
    ++cnt;
    sum += (double)v;
    const unsigned long long k = ((unsigned long long)ordered_bits(v) << 32) |
                                 (unsigned long long)(0xffffffffu - (unsigned int)q);
    key = k > key ? k : key;
  });
  cnt = block_reduce(cnt, sh_c, [](long long x, long long y) { return x + y; });
  sum = block_reduce(sum, sh_s, [](double x, double y) { return x + y; });
  key = block_reduce(key, sh_k,
                     [](unsigned long long x, unsigned long long y) { return x > y ? x : y; });
  if (threadIdx.x == 0) part[blockIdx.x] = Part1{cnt, sum, key};
}

__global__ void k_m_reduce(long long n_slots, int chunks, const Part1* part, SlotStat* st) {
  const long long slot = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (slot >= n_slots) return;
  long long cnt = 0;
  double sum = 0.0;
  unsigned long long key = 0;
  for (int c = 0; c < chunks; ++c) {
    const Part1 p = part[slot * chunks + c];
    cnt += p.cnt;
    sum += p.sum;
    key = p.key > key ? p.key : key;
  }
  st[slot] = SlotStat{cnt, cnt > 0 ? sum / (double)cnt : 0.0, key};
}

// Normalised-amplitude bin of Eq. 12: floor(v * 256 / vmax), FP32 with an
// IEEE-rounded division, clamped to [0, 255].
__device__ __forceinline__ int amp_bin(float v, float vmax) {
  if (!(vmax > 0.f) || !(v > 0.f)) return 0;
  const float x = __fdiv_rn(v * 256.0f, vmax);
  return x >= 255.0f ? 255 : (int)x;
}

__global__ void __launch_bounds__(kThreads) k_m_pass2(MGeom g, const MRegion* regs,
                                                      const ColRange* ranges, const float* images,
                                                      const SlotStat* st, double* part2, int* hist) {
  __shared__ int h[kBins];
  __shared__ double sh_s[kThreads / 32];
  const long long slot = blockIdx.x / g.chunks;
  const int chunk = blockIdx.x % g.chunks;
  const SlotRef s = slot_ref(g, regs, images, slot);
  const MRegion r = *s.reg;
  const SlotStat mine = st[slot];
  const SlotStat a = st[slot & ~1ll], b = st[slot | 1ll];
  float vmax = -INFINITY;
  if (a.cnt > 0) vmax = key_value(a.key);
  if (b.cnt > 0) vmax = fmaxf(vmax, key_value(b.key));
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) h[i] = 0;
  __syncthreads();
  double ss = 0.0;
  for_members(g, r, ranges, chunk, [&](int, int, long long q) {
    const float v = __ldg(s.img + q);
    const double e = (double)v - mine.mean;
    ss += e * e;
    atomicAdd(&h[amp_bin(v, vmax)], 1);
  });
  ss = block_reduce(ss, sh_s, [](double x, double y) { return x + y; });
  if (threadIdx.x == 0) part2[blockIdx.x] = ss;
  __syncthreads();
  int* dst = hist + (size_t)slot * kBins;
  for (int i = threadIdx.x; i < kBins; i += blockDim.x)
    if (h[i]) atomicAdd(dst + i, h[i]);
}

__global__ void k_m_final(MGeom g, long long n_pairs, const float* images, const SlotStat* st,
                          const double* part2, const int* hist, pa_metrics* out) {
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_pairs) return;
  const long long pair = g.pair0 + p;
  const float* img = images + (size_t)(pair / g.n_roi) * g.nx * g.nz;
  const SlotStat si = st[2 * p], so = st[2 * p + 1];
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  pa_metrics m;
  m.n_in = si.cnt;
  m.n_out = so.cnt;
  m.mu_in = si.cnt > 0 ? si.mean : nan;
  m.mu_out = so.cnt > 0 ? so.mean : nan;
  double ss = 0.0;
  for (int c = 0; c < g.chunks; ++c) ss += part2[(2 * p + 1) * g.chunks + c];
  m.sigma_out = so.cnt > 0 ? sqrt(ss / (double)so.cnt) : nan;
  m.snr_db = 20.0 * log10(m.mu_in / m.sigma_out);
  m.cr_db = 20.0 * log10(m.mu_in / m.mu_out);
  if (si.cnt > 0 && so.cnt > 0) {
    // sum_b min(c_in / n_in, c_out / n_out) = sum_b min(c_in n_out, c_out n_in) / (n_in n_out)
    const int* hi = hist + (size_t)(2 * p) * kBins;
    const int* ho = hi + kBins;
    long long ov = 0;
    for (int b = 0; b < kBins; ++b) {
      const long long u = (long long)hi[b] * so.cnt, v = (long long)ho[b] * si.cnt;
      ov += u < v ? u : v;
    }
    m.gcnr = 1.0 - (double)ov / ((double)si.cnt * (double)so.cnt);
  } else {
    m.gcnr = nan;
  }
  m.peak = nan;
  m.fwhm_m = nan;
  m.peak_j = m.peak_l = -1;
  if (si.cnt > 0) {
    const unsigned int q = 0xffffffffu - (unsigned int)(si.key & 0xffffffffull);
    const int j0 = (int)(q / (unsigned int)g.nz), l0 = (int)(q % (unsigned int)g.nz);
    const float pk = key_value(si.key);
    m.peak = (double)pk;
    m.peak_j = j0;
    m.peak_l = l0;
    const double half = 0.5 * (double)pk;
    const float* row = img + l0;  // element j of the row at row[j * nz]
    auto at = [&](int j) { return (double)row[(size_t)j * g.nz]; };
    auto xp = [&](int j) { return __dadd_rn(g.x0, __dmul_rn((double)j + 0.5, g.dx)); };
    int jl = j0;
    while (jl > 0 && at(jl - 1) >= half) --jl;
    int jr = j0;
    while (jr < g.nx - 1 && at(jr + 1) >= half) ++jr;
    if (jl > 0 && jr < g.nx - 1) {
      const double pl = at(jl - 1), ql = at(jl);
      const double pr = at(jr + 1), qr = at(jr);
      const double xl = __dadd_rn(xp(jl - 1), __dmul_rn(__ddiv_rn(__dsub_rn(half, pl), __dsub_rn(ql, pl)), g.dx));
      const double xr = __dsub_rn(xp(jr + 1), __dmul_rn(__ddiv_rn(__dsub_rn(half, pr), __dsub_rn(qr, pr)), g.dx));
      m.fwhm_m = __dsub_rn(xr, xl);
    }
  }
  out[pair] = m;
}

// A sum of floats as three floats, by exact additions (Knuth's two-sum): the
// first two parts take no rounding error, the third rounds at 2^-72 of the
// sum.  Not finite where a partial sum leaves FP32's range.
__device__ __forceinline__ float two_sum(float a, float b, float* e) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  *e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
  return s;
}
struct Sum3 {
  float a = 0.f, b = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float v) {
    float e, f;
    a = two_sum(a, v, &e);
    b = two_sum(b, e, &f);
    c = __fadd_rn(c, f);
  }
  __device__ __forceinline__ void add_low(float v) {  // v far below the sum
    float f;
    b = two_sum(b, v, &f);
    c = __fadd_rn(c, f);
  }
  __device__ __forceinline__ void merge(const Sum3& o) {
    float e, f, h;
    a = two_sum(a, o.a, &e);
    b = two_sum(b, o.b, &f);
    b = two_sum(b, e, &h);
    c = __fadd_rn(__fadd_rn(c, o.c), __fadd_rn(f, h));
  }
  __device__ __forceinline__ void merge_lanes(int width) {  // over lane ^ 1, 2, .. width / 2
    for (int o = width / 2; o >= 1; o >>= 1) {
      Sum3 v;
      v.a = __shfl_xor_sync(0xffffffffu, a, o);
      v.b = __shfl_xor_sync(0xffffffffu, b, o);
      v.c = __shfl_xor_sync(0xffffffffu, c, o);
      merge(v);
    }
  }
  __device__ __forceinline__ bool finite() const { return isfinite(a) && isfinite(b) && isfinite(c); }
  __device__ __forceinline__ double value() const { return (double)a + ((double)b + (double)c); }
};

constexpr size_t kPairSmem = 200 * 1024;  // most dynamic shared memory of a block
constexpr long long kListMax = 16 << 20;  // most entries of the member list (64 MiB)

// One (image, ROI pair) per block; header of this file.  The dynamic shared
// memory holds `cap` values: the target's, then the background's.  The
// registers suffice for 2048 / T blocks of T threads (T = 1024) or half as
// many (T = 256: 41 us instead of 44 for 960 pairs of 3600 pixels; with T =
// 1024 it is 289 instead of 198 us for 1536 pairs of 24000).
template <int T>
__global__ void __launch_bounds__(T, T == 1024 ? 2 : 1024 / T)
    k_m_pair(MGeom g, const int* counts, const unsigned int* list, const long long* pix0,
             const float* images, int cap, pa_metrics* out) {
  extern __shared__ float vals[];
  __shared__ int hist[2][kBins];
  __shared__ Sum3 sh_s[2][32];
  __shared__ unsigned int sh_o[2][32], sh_i[2][32];
  __shared__ long long sh_l[32];
  __shared__ double sh_d[32], sh_mean[2], sh_rest, sh_ss;
  __shared__ unsigned int sh_ord[2];
  __shared__ int sh_peak[2], sh_walk[2], sh_bad;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, warps = blockDim.x >> 5;
  const long long pair = g.pair0 + blockIdx.x;
  const int roi = (int)(pair % g.n_roi);
  const float* const img = images + (size_t)(pair / g.n_roi) * g.nx * g.nz;
  // (never above the host's bounds; clamped so that nothing can leave `vals`)
  const int n0 = min(counts[2 * roi], cap), n1 = min(counts[2 * roi + 1], cap - n0);
  const unsigned int* const in0 = list + pix0[2 * roi];
  const unsigned int* const in1 = list + pix0[2 * roi + 1];
  auto fetch = [&](const unsigned int* q, int n, float* dst) {
#pragma unroll 4
    for (int t = tid; t < n; t += blockDim.x)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                       (unsigned)__cvta_generic_to_shared(dst + t)),
                   "l"(img + __ldg(q + t)));
  };
  fetch(in0, n0, vals);
  fetch(in1, n1, vals + n0);
  for (int i = tid; i < 2 * kBins; i += blockDim.x) hist[0][i] = 0;
  if (tid == 0) sh_bad = 0;
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  // pass 1: sums, and the largest value with its first place
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    Sum3 s;
    unsigned int ord = 0, idx = 0xffffffffu;
    for (int t = tid; t < (side ? n1 : n0); t += blockDim.x) {
      const float v = vals[side ? n0 + t : t];
      s.add(v);
      const unsigned int o = ordered_bits(v);
      if (o > ord || idx == 0xffffffffu) {
        ord = o;
        idx = (unsigned)t;
      }
    }
    const unsigned int top = __reduce_max_sync(0xffffffffu, ord);
    const unsigned int first = __reduce_min_sync(0xffffffffu, ord == top ? idx : 0xffffffffu);
    s.merge_lanes(32);
    if (lane == 0) {
      sh_s[side][w] = s;
      sh_o[side][w] = top;
      sh_i[side][w] = first;
    }
  }
  __syncthreads();
  if (w < 2) {
    Sum3 s;
    unsigned int ord = 0, idx = 0xffffffffu;
    if (lane < warps) {
      s = sh_s[w][lane];
      ord = sh_o[w][lane];
      idx = sh_i[w][lane];
    }
    const unsigned int top = __reduce_max_sync(0xffffffffu, ord);
    const unsigned int first = __reduce_min_sync(0xffffffffu, ord == top ? idx : 0xffffffffu);
    s.merge_lanes(32);
    if (lane == 0) {
      sh_ord[w] = top;
      const double nn = (double)(w ? n1 : n0), mean = nn > 0 ? s.value() / nn : 0.0;
      sh_mean[w] = mean;
      // mean - (float)mean from the parts of the sum: n (float)mean is exact
      if (w) sh_rest = nn > 0 ? (((double)s.a - nn * (double)(float)mean) + ((double)s.b + (double)s.c)) / nn : 0.0;
      if (!s.finite()) sh_bad = 1;
      if (w == 0 && n0 > 0) {
        const unsigned int q = in0[first];
        sh_peak[0] = (int)(q / (unsigned)g.nz);
        sh_peak[1] = (int)(q % (unsigned)g.nz);
      }
    }
  }
  __syncthreads();
  if (sh_bad) {  // values beyond FP32's range or not finite: in FP64
    for (int side = 0; side < 2; ++side) {
      const int ns = side ? n1 : n0;
      const float* const v = vals + (side ? n0 : 0);
      double s = 0.0;
      for (int t = tid; t < ns; t += blockDim.x) s += (double)v[t];
      s = block_reduce(s, sh_d, [](double x, double y) { return x + y; });
      if (tid == 0) sh_mean[side] = ns > 0 ? s / (double)ns : 0.0;
    }
    __syncthreads();
  }

  // pass 2: histograms, and the background's squared deviations.  With m the
  // mean rounded to FP32, v - m = d + e exactly, and
  //   sum (v - mean)^2 = sum (d + e)^2 - n (mean - m)^2.
  float vmax = -INFINITY;
  if (n0 > 0) vmax = unorder(sh_ord[0]);
  if (n1 > 0) vmax = fmaxf(vmax, unorder(sh_ord[1]));
  for (int t = tid; t < n0; t += blockDim.x) atomicAdd(&hist[0][amp_bin(vals[t], vmax)], 1);
  const double mean = sh_mean[1];
  const float m = (float)mean;
  Sum3 s;
  for (int t = tid; t < n1; t += blockDim.x) {
    const float v = vals[n0 + t];
    atomicAdd(&hist[1][amp_bin(v, vmax)], 1);
    float e;
    const float d = two_sum(v, -m, &e);
    const float p = __fmul_rn(d, d), pe = __fmaf_rn(d, d, -p);
    const float c = __fmul_rn(2.f * d, e), ce = __fmaf_rn(2.f * d, e, -c);
    s.add(p);
    s.add_low(pe);
    s.add_low(c);
    s.c = __fadd_rn(s.c, __fmaf_rn(e, e, ce));
  }
  s.merge_lanes(32);
  if (lane == 0) sh_s[0][w] = s;
  // the walks along the row of the target's maximum, 32 columns at a time:
  // jl, jr are the last columns before one below half the maximum
  const float pk = unorder(sh_ord[0]);
  const double half = 0.5 * (double)pk;
  if (n0 > 0 && w < 2) {
    const int jp = sh_peak[0];
    const float* const row = img + sh_peak[1];
    int end = w ? g.nx - 1 : 0;
    for (int k = 1; w ? jp + k < g.nx : jp - k >= 0; k += 32) {
      const int j = w ? jp + k + lane : jp - k - lane;
      const bool in = j >= 0 && j < g.nx && (double)row[(size_t)j * g.nz] >= half;
      const unsigned int stop = __ballot_sync(0xffffffffu, !in);
      if (stop) {
        const int f = k + __ffs(stop) - 2;
        end = w ? jp + f : jp - f;
        break;
      }
    }
    if (lane == 0) sh_walk[w] = end;
  }
  __syncthreads();
  // Eq. 12's overlap: sum_b min(c_in / n_in, c_out / n_out)
  //                 = sum_b min(c_in n_out, c_out n_in) / (n_in n_out)
  long long ov = 0;
  for (int b = tid; b < kBins; b += blockDim.x) {
    const long long u = (long long)hist[0][b] * n1, v = (long long)hist[1][b] * n0;
    ov += u < v ? u : v;
  }
  ov = block_reduce(ov, sh_l, [](long long x, long long y) { return x + y; });
  if (w == 0) {
    s = lane < warps ? sh_s[0][lane] : Sum3();
    s.merge_lanes(32);
    if (lane == 0) {
      const double ss = s.value() - (double)n1 * sh_rest * sh_rest;
      sh_ss = ss;
      // the products of tiny deviations lose bits to FP32's underflow
      sh_bad = !(s.finite() && ss >= (double)n1 * 0x1p-70);
    }
  }
  __syncthreads();
  if (sh_bad) {
    double q = 0.0;
    for (int t = tid; t < n1; t += blockDim.x) {
      const double e = (double)vals[n0 + t] - mean;
      q += e * e;
    }
    q = block_reduce(q, sh_d, [](double x, double y) { return x + y; });
    if (tid == 0) sh_ss = q;
    __syncthreads();
  }
  if (w != 0) return;
  // lanes 0 and 1 take the two quotients and the two ends of the FWHM
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  const double mu_in = n0 > 0 ? sh_mean[0] : nan, mu_out = n1 > 0 ? mean : nan;
  const double sigma = n1 > 0 ? sqrt(sh_ss / (double)n1) : nan;
  const double db = 20.0 * log10(mu_in / (lane ? mu_out : sigma));
  const double cr = __shfl_sync(0xffffffffu, db, 1);
  double fwhm = nan;
  if (n0 > 0 && sh_walk[0] > 0 && sh_walk[1] < g.nx - 1) {
    const float* const row = img + sh_peak[1];
    const int step = lane ? 1 : -1, at = sh_walk[lane ? 1 : 0];
    const double p = (double)row[(size_t)(at + step) * g.nz], q = (double)row[(size_t)at * g.nz];
    const double f = __dmul_rn(__ddiv_rn(__dsub_rn(half, p), __dsub_rn(q, p)), g.dx);
    const double x = __dadd_rn(g.x0, __dmul_rn((double)(at + step) + 0.5, g.dx));
    const double end = lane ? __dsub_rn(x, f) : __dadd_rn(x, f);
    fwhm = __dsub_rn(__shfl_sync(0xffffffffu, end, 1), end);
  }
  if (lane == 0) {
    pa_metrics r;
    r.mu_in = mu_in;
    r.mu_out = mu_out;
    r.sigma_out = sigma;
    r.snr_db = db;
    r.cr_db = cr;
    r.gcnr = n0 > 0 && n1 > 0 ? 1.0 - (double)ov / ((double)n0 * (double)n1) : nan;
    r.fwhm_m = fwhm;
    r.peak = n0 > 0 ? (double)pk : nan;
    r.n_in = n0;
    r.n_out = n1;
    r.peak_j = n0 > 0 ? sh_peak[0] : -1;
    r.peak_l = n0 > 0 ? sh_peak[1] : -1;
    out[pair] = r;
  }
}

pa_status mfail(pa_status s, const char* msg) {
  pa::set_error_message(msg);
  return s;
}

bool finite_d(double v) { return std::isfinite(v); }

// Conservative index range of pixel centres in [c - h, c + h] on a grid of n
// cells starting at o with step d; the membership test decides exactly.
void index_range(double c, double h, double o, double d, int n, int* lo, int* hi) {
  const double a = (c - h - o) / d - 0.5, b = (c + h - o) / d - 0.5;
  double l = std::floor(a) - 1.0, u = std::ceil(b) + 2.0;
  l = std::max(0.0, std::min((double)n, l));
  u = std::max(0.0, std::min((double)n, u));
  *lo = (int)l;
  *hi = std::max(*lo, (int)u);
}

}  // namespace

extern "C" pa_status pa_image_metrics(const pa_grid* grid, const float* images_dev,
                                      int32_t n_images, const pa_roi* rois, int32_t n_roi,
                                      pa_metrics* out_dev, void* cuda_stream) {
  if (!grid || !rois) return mfail(PA_EINVAL, "pa_image_metrics: null grid or rois");
  if (n_images < 0) return mfail(PA_EINVAL, "pa_image_metrics: n_images < 0");
  if (n_roi < 1 || n_roi > PA_METRICS_MAX_ROIS)
    return mfail(PA_EINVAL, "pa_image_metrics: n_roi outside 1..PA_METRICS_MAX_ROIS");
  const pa_grid G = *grid;
  if (G.nx < 1 || G.nz < 1 || !finite_d(G.x0_m) || !finite_d(G.x1_m) || !finite_d(G.z0_m) ||
      !finite_d(G.z1_m) || !(G.x1_m > G.x0_m) || !(G.z1_m > G.z0_m))
    return mfail(PA_EINVAL, "pa_image_metrics: bad grid");
  if ((long long)G.nx * G.nz > 0xffffffffll)
    return mfail(PA_EINVAL, "pa_image_metrics: image larger than 2^32 pixels");
  if (n_images == 0) return PA_OK;
  if (!images_dev || !out_dev) return mfail(PA_EINVAL, "pa_image_metrics: null buffer");

  MGeom g{};
  g.nx = G.nx;
  g.nz = G.nz;
  g.n_roi = n_roi;
  g.x0 = G.x0_m;
  g.z0 = G.z0_m;
  g.dx = (G.x1_m - G.x0_m) / G.nx;
  g.dz = (G.z1_m - G.z0_m) / G.nz;
  g.rows_per_m = (float)(1.0 / g.dz);
  std::vector<MRegion> regs(2 * (size_t)n_roi);
  long long max_area = 0, n_cols = 0, n_pix = 0, cap = 0;
  int max_width = 0;
  double reach = std::max(std::max(std::fabs(G.x0_m), std::fabs(G.x1_m)),
                          std::max(std::fabs(G.z0_m), std::fabs(G.z1_m)));
  for (int r = 0; r < n_roi; ++r) {
    long long members = 0;
    for (int side = 0; side < 2; ++side) {
      const pa_region& in = side ? rois[r].background : rois[r].target;
      MRegion& o = regs[2 * r + side];
      if (in.shape != PA_REGION_RECT && in.shape != PA_REGION_DISC && in.shape != PA_REGION_ANNULUS)
        return mfail(PA_EINVAL, "pa_image_metrics: unknown region shape");
      if (!finite_d(in.xc_m) || !finite_d(in.zc_m) || !finite_d(in.a_m) || !finite_d(in.b_m) ||
          in.a_m < 0 || in.b_m < 0)
        return mfail(PA_EINVAL, "pa_image_metrics: region extents must be finite and >= 0");
      o.shape = in.shape;
      o.xc = in.xc_m;
      o.zc = in.zc_m;
      o.a = in.a_m;
      o.b = in.b_m;
      reach = std::max({reach, std::fabs(in.xc_m), std::fabs(in.zc_m), in.a_m, in.b_m});
      const double hx = in.shape == PA_REGION_ANNULUS ? in.b_m : in.a_m;
      const double hz = in.shape == PA_REGION_DISC ? in.a_m : in.b_m;
      index_range(in.xc_m, hx, g.x0, g.dx, g.nx, &o.j0, &o.j1);
      index_range(in.zc_m, hz, g.z0, g.dz, g.nz, &o.l0, &o.l1);
      o.col0 = n_cols;
      n_cols += o.j1 - o.j0;
      const bool inside = o.j0 > 0 && o.l0 > 0 && o.j1 < g.nx && o.l1 < g.nz;
      const long long most =
          pa::most_members(o.shape, o.a, o.b, o.j1 - o.j0, o.l1 - o.l0, inside, g.dx, g.dz);
      o.pix0 = n_pix;
      n_pix += most;
      o.pix1 = n_pix;
      members += most;
      max_width = std::max(max_width, o.j1 - o.j0);
      max_area = std::max(max_area, (long long)(o.j1 - o.j0) * (o.l1 - o.l0));
    }
    cap = std::max(cap, members);
  }
  // k_m_pair where the members of every pair fit.  The bounds hold as long as
  // no coordinate is so far from the image that rounding costs a visible part
  // of a pixel.
  const bool in_block = (size_t)cap * 4 <= kPairSmem && max_width <= kMemberCols &&
                        n_pix <= kListMax && reach <= 0x1p40 * std::min(g.dx, g.dz);
  // blocks per region: about 8192 bounding-box pixels each, at least one
  // column per warp
  const long long by_area = (max_area + 8191) / 8192, by_cols = (max_width + 7) / 8;
  g.chunks = (int)std::max<long long>(1, std::min<long long>({(long long)kMaxChunks, by_area, by_cols}));

  cudaStream_t st = (cudaStream_t)cuda_stream;
  const long long n_pairs = (long long)n_images * n_roi;
  const long long pairs_per = std::min(n_pairs, in_block ? 1ll << 30 : kPairsPerLaunch);
  const long long slots_per = in_block ? 0 : 2 * pairs_per;
  const size_t b_regs = regs.size() * sizeof(MRegion);
  // (in_block: counts, places and members instead of the column ranges)
  const size_t b_cols = in_block ? regs.size() * 12 + (size_t)n_pix * 4
                                 : (size_t)std::max<long long>(n_cols, 1) * sizeof(ColRange);
  const size_t b_p1 = (size_t)slots_per * g.chunks * sizeof(Part1);
  const size_t b_st = (size_t)slots_per * sizeof(SlotStat);
  const size_t b_p2 = (size_t)slots_per * g.chunks * sizeof(double);
  const size_t b_h = (size_t)slots_per * kBins * sizeof(int);
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t total = up(b_regs) + up(b_cols) + up(b_p1) + up(b_st) + up(b_p2) + up(b_h);
  char* base = nullptr;
  cudaError_t e = cudaMallocAsync((void**)&base, total, st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return mfail(e == cudaErrorMemoryAllocation ? PA_ENOMEM : PA_ECUDA, cudaGetErrorString(e));
  }
  MRegion* d_regs = (MRegion*)base;
  ColRange* d_cols = (ColRange*)(base + up(b_regs));
  Part1* d_p1 = (Part1*)((char*)d_cols + up(b_cols));
  SlotStat* d_st = (SlotStat*)((char*)d_p1 + up(b_p1));
  double* d_p2 = (double*)((char*)d_st + up(b_st));
  int* d_h = (int*)((char*)d_p2 + up(b_p2));
  RegTable tab;
  const int tab_n = in_block && regs.size() <= kParamRegions ? (int)regs.size() : 0;
  if (tab_n) std::copy(regs.begin(), regs.end(), tab.r);
  else e = cudaMemcpyAsync(d_regs, regs.data(), b_regs, cudaMemcpyHostToDevice, st);
  if (in_block && e == cudaSuccess) {
    long long* d_pix0 = (long long*)d_cols;
    int* d_counts = (int*)(d_pix0 + regs.size());
    unsigned int* d_list = (unsigned int*)(d_counts + regs.size());
    k_m_members<<<(unsigned)regs.size(), 512, 0, st>>>(g, tab, tab_n, d_regs, d_pix0, d_counts, d_list);
    e = cudaGetLastError();
    // About 32 values a thread: 960 pairs of 4200 take 44, 43 and 49 us with
    // 128, 256 and 512 threads, 1536 pairs of 24000 take 554, 327, 223 and 198
    // with 128, 256, 512 and 1024.
    int threads = 128;
    while (threads < 1024 && cap > 32ll * threads) threads *= 2;
    const size_t smem = (size_t)cap * 4;
    const auto kernel = threads > 256 ? k_m_pair<1024> : k_m_pair<256>;
    if (smem > 40 * 1024 && e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPairSmem);
    for (long long p0 = 0; e == cudaSuccess && p0 < n_pairs; p0 += pairs_per) {
      g.pair0 = p0;
      kernel<<<(unsigned)std::min(pairs_per, n_pairs - p0), threads, smem, st>>>(
          g, d_counts, d_list, d_pix0, images_dev, (int)cap, out_dev);
      e = cudaGetLastError();
    }
  } else if (e == cudaSuccess && max_width > 0) {
    const dim3 grid_r((unsigned)((max_width + 31) / 32), (unsigned)regs.size());
    k_m_ranges<<<grid_r, dim3(32, 2), 0, st>>>(g, d_regs, d_cols);
    e = cudaGetLastError();
  }
  for (long long p0 = 0; !in_block && e == cudaSuccess && p0 < n_pairs; p0 += pairs_per) {
    const long long np = std::min(pairs_per, n_pairs - p0);
    const long long ns = 2 * np;
    g.pair0 = p0;
    const long long blocks = ns * g.chunks;
    e = cudaMemsetAsync(d_h, 0, (size_t)ns * kBins * sizeof(int), st);
    if (e != cudaSuccess) break;
    k_m_pass1<<<(unsigned)blocks, kThreads, 0, st>>>(g, d_regs, d_cols, images_dev, d_p1);
    k_m_reduce<<<(unsigned)((ns + 127) / 128), 128, 0, st>>>(ns, g.chunks, d_p1, d_st);
    k_m_pass2<<<(unsigned)blocks, kThreads, 0, st>>>(g, d_regs, d_cols, images_dev, d_st, d_p2,
                                                     d_h);
    k_m_final<<<(unsigned)((np + 127) / 128), 128, 0, st>>>(g, np, images_dev, d_st, d_p2, d_h,
                                                           out_dev);
    e = cudaGetLastError();
  }
  const cudaError_t ef = cudaFreeAsync(base, st);
  if (e == cudaSuccess) e = ef;
  if (e != cudaSuccess) return mfail(PA_ECUDA, cudaGetErrorString(e));
  return PA_OK;
}
