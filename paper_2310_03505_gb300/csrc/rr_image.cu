// rr_image.cu -- polar image assembly and post pass.
//
// Sec. III-B: every return lands in the pixel of its azimuth column and
// range bin; the pixel sums the energies from 0.  Sec. III-C: measurement
// noise as a Gaussian blur along range, a beam pattern across azimuths,
// additive uniform system and ambient noise.
//
// One CTA owns one image column (one azimuth of one scan of the batch; the
// batch's columns are numbered scan by scan): it finds the column's records in every
// bounce's record list (each list is in azimuth order, so two binary
// searches per bounce), accumulates them into a shared-memory histogram with
// warp-aggregated adds (lanes that hit the same bin are summed with shuffles
// and added once), blurs the column in shared memory, adds the noise and
// writes the column once, coalesced.  No global atomics, no memset.
//
// The sums are compensated (Neumaier's improvement of Kahan summation,
// ZAMM 54, 1974): every bin holds a float pair (sum, correction) updated with
// a 64-bit compare-and-swap, and lanes that share a bin combine their values
// the same way first, so a bin's error stays within a few units in the last
// place of its value however many returns it receives and in whatever order.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>

#include "rr_host.h"

namespace rr {

constexpr int kImgBlock = 256;       // beam pattern pass
constexpr int kMaxTaps = 2 * 768 + 1;   // blur / pattern radius up to 768

__device__ __forceinline__ int gauss_taps(float sigma, float* w) {
  // normalised exp(-j^2 / (2 sigma^2)) for |j| <= ceil(3 sigma); w[0..2R]
  const int R = min((int)ceilf(3.0f * sigma), (kMaxTaps - 1) / 2);
  for (int j = threadIdx.x; j <= 2 * R; j += blockDim.x) {
    const float x = (float)(j - R) / sigma;
    w[j] = expf(-0.5f * x * x);
  }
  __syncthreads();
  __shared__ float s_norm;
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int j = 0; j <= 2 * R; ++j) s += w[j];
    s_norm = 1.0f / s;
  }
  __syncthreads();
  for (int j = threadIdx.x; j <= 2 * R; j += blockDim.x) w[j] *= s_norm;
  __syncthreads();
  return R;
}

// first record in [lo, hi) whose column is >= col (records are in column
// order), found by one warp: its lanes probe 32 places at once, so a list of a
// million records takes 4 dependent loads where halving takes 20
template <bool kRaw>
__device__ __forceinline__ uint32_t lower_col(const ScanArgs& a, uint32_t lo, uint32_t hi, uint32_t col) {
  const uint32_t lane = threadIdx.x & 31u;
  while (lo < hi) {   // the answer lies in [lo, hi]
    const uint32_t step = (hi - lo + 31u) / 32u, at = lo + lane * step;
    const bool below = at < hi && (kRaw ? __ldg(&a.raw_column[at]) : __ldg(&a.recs[at].x) >> kBinBits) < col;
    const uint32_t n = __popc(__ballot_sync(0xFFFFFFFFu, below));   // a prefix of the lanes
    if (n == 0u) return lo;
    hi = min(hi, lo + n * step);
    lo += (n - 1u) * step + 1u;
  }
  return lo;
}

// Sec. III-C Perlin noise (Perlin, "Improving noise", SIGGRAPH 2002) of
// pixel (a, bin): gradient noise over a lattice of P = round(n_az / cell_az)
// cells around the circle (periodic) and cells of cell_bins bins along range;
// lattice point (I, J) has the unit gradient at angle 2 pi u, u the uniform of
// Philox counter (scan_id, I, J, purpose); quintic fade; value 1/2 + n/sqrt(2)
__device__ __forceinline__ float perlin_at(uint4 rng, uint32_t n_az, float cell_az, float cell_bins, uint32_t a,
                                          uint32_t bin, uint32_t purpose) {
  const int P = max(1, (int)roundf((float)n_az / cell_az));
  const float x = (float)a * (float)P / (float)n_az, y = (float)bin / cell_bins;
  const float xf = floorf(x), yf = floorf(y);
  const uint32_t i0 = (uint32_t)xf % (uint32_t)P, i1 = (i0 + 1u) % (uint32_t)P;
  const uint32_t j0 = (uint32_t)yf, j1 = j0 + 1u;
  const float fx = x - xf, fy = y - yf;
  float s00, c00, s10, c10, s01, c01, s11, c11;
  sincospif(2.0f * u01(draw(rng, i0, j0, purpose).x), &s00, &c00);
  sincospif(2.0f * u01(draw(rng, i1, j0, purpose).x), &s10, &c10);
  sincospif(2.0f * u01(draw(rng, i0, j1, purpose).x), &s01, &c01);
  sincospif(2.0f * u01(draw(rng, i1, j1, purpose).x), &s11, &c11);
  const float n00 = c00 * fx + s00 * fy, n10 = c10 * (fx - 1.0f) + s10 * fy;
  const float n01 = c01 * fx + s01 * (fy - 1.0f), n11 = c11 * (fx - 1.0f) + s11 * (fy - 1.0f);
  const float sx = fx * fx * fx * (fx * (6.0f * fx - 15.0f) + 10.0f);
  const float sy = fy * fy * fy * (fy * (6.0f * fy - 15.0f) + 10.0f);
  const float nx0 = n00 + sx * (n10 - n00), nx1 = n01 + sx * (n11 - n01);
  return 0.5f + (nx0 + sy * (nx1 - nx0)) * 0.70710678118654752f;
}

// Sec. III-C: system and ambient noise of one pixel, uniform or Perlin
__device__ __forceinline__ float noise_at(const ScanDesc* sd, uint4 rng, float4 post, uint32_t az, uint32_t bin) {
  if (rng.w & RR_NOISE_PERLIN) {
    const float4 ext = __ldg(&sd->ext);
    const uint32_t n_az = __ldg(&sd->dims.x);
    return post.z * perlin_at(rng, n_az, ext.y, ext.z, az, bin, 4u) +
           post.w * perlin_at(rng, n_az, ext.y, ext.z, az, bin, 5u);
  }
  return post.z * u01(draw(rng, az, bin, 2u).x) + post.w * u01(draw(rng, az, bin, 3u).x);
}

// (s, c) + (x, cx) with the rounding error of s + x carried into c
__device__ __forceinline__ float2 neumaier(float2 acc, float x, float cx) {
  const float t = acc.x + x;
  const float e = fabsf(acc.x) >= fabsf(x) ? (acc.x - t) + x : (x - t) + acc.x;
  return make_float2(t, acc.y + (e + cx));
}

__device__ __forceinline__ void bin_add(unsigned long long* cell, float x, float cx) {
  unsigned long long old = *cell, seen;
  do {
    seen = old;
    const float2 cur = make_float2(__uint_as_float((uint32_t)seen), __uint_as_float((uint32_t)(seen >> 32)));
    const float2 nxt = neumaier(cur, x, cx);
    const unsigned long long v = (unsigned long long)__float_as_uint(nxt.x) |
                                 ((unsigned long long)__float_as_uint(nxt.y) << 32);
    old = atomicCAS(cell, seen, v);
  } while (old != seen);
}

// A column is one block's work: with few columns the chip is filled by wider
// blocks (launch_image).
// kRaw: the returns are the caller's arrays (rr_accumulate_returns).
template <int kBlock, bool kRaw>
__global__ void __launch_bounds__(kBlock) k_bin_column(ScanArgs a) {
  extern __shared__ unsigned long long sm64[];
  unsigned long long* cells = sm64;                             // [n_bins] (sum, correction)
  float* hist = reinterpret_cast<float*>(sm64 + a.max_bins);    // [n_bins] the compensated sums
  float* col = reinterpret_cast<float*>(sm64);                  // [n_bins] after the blur (reuses cells)
  __shared__ float taps[kMaxTaps];
  __shared__ uint32_t s_rng[2 * RR_MAX_BOUNCES];
  const uint32_t c = blockIdx.x;
  const uint32_t scan = owner_of(a.col0, a.n_scans, c);
  const ScanDesc* sd = a.desc + scan;
  const uint32_t az = __ldg(&sd->offs.w) + (c - __ldg(&a.col0[scan]));   // the scan's first azimuth + column
  const uint32_t nb = __ldg(&sd->dims.w);
  const float4 post = __ldg(&sd->post);   // blur sigma, pattern sigma, noise_sys, noise_amb
  const int lane = threadIdx.x & 31;
  for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x) cells[i] = 0ull;
  // record range of this column in every bounce's list, one end a warp at a time
  for (uint32_t q = threadIdx.x >> 5; q < 2u * a.max_bounces; q += kBlock / 32) {
    const uint32_t r = lower_col<kRaw>(a, a.ctr->rec_start[q >> 1], a.ctr->rec_start[(q >> 1) + 1], c + (q & 1u));
    if (lane == 0) s_rng[q] = r;
  }
  __syncthreads();
  // the column's records of all bounces in one run: a bounce's list alone
  // seldom fills the block.  Whole warps iterate together so that the
  // shuffles see every lane.
  auto records = [&](uint32_t b) {   // a failed scan's stale slots need not be in order
    return s_rng[2 * b + 1] > s_rng[2 * b] ? s_rng[2 * b + 1] - s_rng[2 * b] : 0u;
  };
  uint32_t total = 0;
  for (uint32_t b = 0; b < a.max_bounces; ++b) total += records(b);
  for (uint32_t base = 0; base < total; base += kBlock) {
    uint32_t r = base + threadIdx.x;
    bool valid = r < total;
    uint32_t bin = 0;
    float e = 0.0f;
    if (valid) {
      uint32_t b = 0;   // its bounce: r < total, so this ends at the last one
      for (uint32_t n = records(0); r >= n; n = records(++b)) r -= n;
      r += s_rng[2 * b];
      if (kRaw) {
        bin = __ldg(&a.raw_bin[r]);
        e = __ldg(&a.raw_energy[r]);
      } else {
        const uint2 rc = __ldg(&a.recs[r]);
        bin = rc.x & kBinMask;
        e = __uint_as_float(rc.y);
      }
      valid = bin < nb;   // a caller's return past the image adds nothing; records always carry bin < n_bins; a failed scan may leave stale slots
    }
    const uint32_t tag = valid ? bin : 0x10000u + (uint32_t)lane;
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, tag);
    float2 acc = make_float2(0.0f, 0.0f);
    for (uint32_t m = peers; m; m &= m - 1u) acc = neumaier(acc, __shfl_sync(peers, e, __ffs(m) - 1), 0.0f);
    if (valid && lane == __ffs(peers) - 1) bin_add(&cells[bin], acc.x, acc.y);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x) {
    const unsigned long long v = cells[i];
    hist[i] = __uint_as_float((uint32_t)v) + __uint_as_float((uint32_t)(v >> 32));
  }
  __syncthreads();
  const float* src = hist;
  if (post.x > 0.0f) {
    const int R = gauss_taps(post.x, taps);
    for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x) {
      float acc = 0.0f;
      for (int j = -R; j <= R; ++j) {
        const int s = (int)i + j;
        if (s >= 0 && s < (int)nb) acc += taps[j + R] * hist[s];
      }
      col[i] = acc;
    }
    __syncthreads();
    src = col;
  }
  if (post.y > 0.0f) {
    float* out = a.image_tmp + __ldg(&sd->offs.z) + (size_t)az * nb;
    for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x) out[i] = src[i];
  } else {
    float* out = sd->image + (size_t)az * nb;
    const uint4 rng = __ldg(&sd->rng);
    const bool noise = (rng.w & RR_NOISE) != 0u;
    for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x)
      out[i] = src[i] + (noise ? noise_at(sd, rng, post, az, i) : 0.0f);
  }
}

// beam pattern across the azimuths of a scan (circular), then noise; one
// block row per image column, scans without a pattern return at once
__global__ void __launch_bounds__(kImgBlock) k_az_pattern(ScanArgs a) {
  __shared__ float taps[kMaxTaps];
  const uint32_t c = blockIdx.x;   // column on x: a batch may hold more than 65535
  const uint32_t scan = owner_of(a.col0, a.n_scans, c);
  const ScanDesc* sd = a.desc + scan;
  const float4 post = __ldg(&sd->post);
  if (!(post.y > 0.0f)) return;   // uniform over the block
  const int R = gauss_taps(post.y, taps);
  const uint32_t az = __ldg(&sd->offs.w) + (c - __ldg(&a.col0[scan]));   // pattern scans are never split: offs.w = 0
  const uint32_t n_az = __ldg(&sd->dims.x), nb = __ldg(&sd->dims.w);
  const uint32_t i = blockIdx.y * blockDim.x + threadIdx.x;
  if (i >= nb) return;
  const float* tmp = a.image_tmp + __ldg(&sd->offs.z);
  float acc = 0.0f;
  for (int j = -R; j <= R; ++j) {
    int s = ((int)az + j) % (int)n_az;
    if (s < 0) s += (int)n_az;
    acc += taps[j + R] * tmp[(size_t)s * nb + i];
  }
  const uint4 rng = __ldg(&sd->rng);
  if (rng.w & RR_NOISE) acc += noise_at(sd, rng, post, az, i);
  sd->image[(size_t)az * nb + i] = acc;
}

// flags a column of caller-given returns that decreases or lies past the image
__global__ void k_check_returns(const uint32_t* __restrict__ column, uint32_t n, uint32_t n_columns,
                                uint32_t* __restrict__ bad) {
  const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const uint32_t c = column[k];
  if ((k > 0 && column[k - 1] > c) || c >= n_columns) atomicOr(bad, 1u);
}

// Sec. III-B display mapping, one pixel: the reference form (a logarithm, a
// division and the rounding)
__device__ __forceinline__ uint32_t db_pixel(float e, float cutoff_db) {
  float v = 0.0f;
  if (e > 0.0f) v = fminf(fmaxf(255.0f * (10.0f * log10f(e) + cutoff_db) / cutoff_db, 0.0f), 255.0f);
  return (uint32_t)floorf(v + 0.5f);
}

// The same pixel from the hardware's base-2 logarithm: v differs from the
// reference's by less than `band` (DbMap), so unless v + 1/2 lies that close
// to a whole number both round to the same pixel; otherwise (about one pixel
// in a thousand) the reference form decides.
struct DbMap {
  float cutoff, slope, band;   // slope: 255 * 10 log10(2) / cutoff
};
__device__ __forceinline__ uint32_t db_pixel_fast(float e, const DbMap& m) {
  const float v = e > 0.0f ? fminf(fmaxf(fmaf(__log2f(e), m.slope, 255.0f), 0.0f), 255.0f) : 0.0f;
  const float w = v + 0.5f, f = floorf(w);
  const float d = w - f;
  if (!(d >= m.band && d <= 1.0f - m.band)) return db_pixel(e, m.cutoff);
  return (uint32_t)f;
}

// One thread maps kDbRows groups of four pixels, each group a 16-byte load and
// a 4-byte store, the loads issued together.  What a pixel costs is the
// arithmetic: the reference form's log10f and division made the pass run at a
// quarter of the copy bandwidth (256 images of 400 x 2,000 pixels, 1.02 GB:
// 611 us; bytes alone would take 151).
constexpr int kDbBlock = 256, kDbRows = 4;
__global__ void __launch_bounds__(kDbBlock) k_db_u8_vec(const float4* __restrict__ polar, uint64_t n4, DbMap m,
                                                        uint32_t* __restrict__ out) {
  const uint64_t i0 = (uint64_t)blockIdx.x * (kDbBlock * kDbRows) + threadIdx.x;
  float4 e[kDbRows];
#pragma unroll
  for (int r = 0; r < kDbRows; ++r) {
    const uint64_t i = i0 + (uint64_t)r * kDbBlock;
    e[r] = i < n4 ? __ldcs(polar + i) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int r = 0; r < kDbRows; ++r) {
    const uint64_t i = i0 + (uint64_t)r * kDbBlock;
    const uint32_t px = db_pixel_fast(e[r].x, m) | db_pixel_fast(e[r].y, m) << 8 | db_pixel_fast(e[r].z, m) << 16 |
                        db_pixel_fast(e[r].w, m) << 24;
    if (i < n4) __stcs(out + i, px);
  }
}
// pixels that the grouped form cannot take: a remainder, or unaligned buffers
__global__ void __launch_bounds__(kDbBlock) k_db_u8(const float* __restrict__ polar, uint64_t n, DbMap m,
                                                    uint8_t* __restrict__ out) {
  const uint64_t i = (uint64_t)blockIdx.x * kDbBlock + threadIdx.x;
  if (i < n) out[i] = (uint8_t)db_pixel_fast(polar[i], m);
}

}  // namespace rr

namespace rr_host {

using namespace rr;

// dynamic shared memory of k_bin_column: (sum, correction) pairs (later the
// blurred column), sums
static size_t bin_smem(uint32_t n_bins) { return (size_t)n_bins * (sizeof(unsigned long long) + sizeof(float)); }

void init_image_attrs() {
  static bool attr_set = false;
  if (!attr_set) {
    for (const void* k : {(const void*)k_bin_column<256, false>, (const void*)k_bin_column<512, false>,
                          (const void*)k_bin_column<1024, false>, (const void*)k_bin_column<256, true>,
                          (const void*)k_bin_column<512, true>, (const void*)k_bin_column<1024, true>})
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bin_smem(RR_MAX_BINS));
    attr_set = true;
  }
}

cudaError_t launch_image(const ScanArgs& a, bool pattern, cudaStream_t st) {
  init_image_attrs();
  const uint32_t sms = (uint32_t)num_sms();
  const int block = a.n_cols <= 2u * sms ? 1024 : (a.n_cols <= 4u * sms ? 512 : 256);
  auto* bin = a.raw_column ? (block == 1024 ? k_bin_column<1024, true> : block == 512 ? k_bin_column<512, true> : k_bin_column<256, true>)
                           : (block == 1024 ? k_bin_column<1024, false> : block == 512 ? k_bin_column<512, false> : k_bin_column<256, false>);
  bin<<<a.n_cols, block, bin_smem(a.max_bins), st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (pattern) {
    dim3 grid(a.n_cols, (a.max_bins + kImgBlock - 1) / kImgBlock);
    k_az_pattern<<<grid, kImgBlock, 0, st>>>(a);
    e = cudaGetLastError();
  }
  return e;
}

cudaError_t launch_db_u8(const float* polar, uint64_t n, float cutoff_db, uint8_t* out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  DbMap m;
  m.cutoff = cutoff_db;
  m.slope = 255.0f * 3.01029995663981195f / cutoff_db;
  // |v - reference| where neither is clamped, so |10 log10 e| <= cutoff, with
  // u = 2^-24: __log2f errs by 2^-22 max(1, |log2 e|), which is slope 2^-22 +
  // 255 * 4 u of v; the roundings here by 255 * 5 u; log10f (2 ulps) and the
  // reference's four operations by 255 * 8 u.  Twice that and more:
  m.band = fabsf(m.slope) * 0x1p-20f + 255.0f * 0x1p-19f;
  // four pixels at a time where both buffers allow it
  const uint64_t n4 = (reinterpret_cast<uintptr_t>(polar) % 16 == 0 && reinterpret_cast<uintptr_t>(out) % 4 == 0) ? n / 4 : 0;
  if (n4) {
    const uint64_t per = (uint64_t)kDbBlock * kDbRows;
    k_db_u8_vec<<<(unsigned)((n4 + per - 1) / per), kDbBlock, 0, st>>>(reinterpret_cast<const float4*>(polar), n4, m,
                                                                       reinterpret_cast<uint32_t*>(out));
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const uint64_t rest = n - 4 * n4;
  if (rest)
    k_db_u8<<<(unsigned)((rest + kDbBlock - 1) / kDbBlock), kDbBlock, 0, st>>>(polar + 4 * n4, rest, m, out + 4 * n4);
  return cudaGetLastError();
}

}  // namespace rr_host

using namespace rr_host;

// device memory of the current device that a kernel can take as 4-byte elements
static bool usable_here(const void* p) {
  cudaPointerAttributes at;
  int dev = -1;
  if (reinterpret_cast<uintptr_t>(p) % 4 != 0 || cudaGetDevice(&dev) != cudaSuccess ||
      cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice && at.device == dev;
}

// Setup block of a call whose buffers are all used in place: slots compiled
// into the library (an allocation of a few hundred bytes took most of the call,
// the driver maps and unmaps its 2 MiB block around it).  A slot is held for
// one blocking call; with none free the call allocates.
namespace {
struct Setup {
  ScanCounters ctr;
  ScanDesc desc;
  uint32_t pre[4], bad;   // ray prefix (unused) and column prefix; the check's flag
};
constexpr int kSetupSlots = 16, kSetupDevices = 64;
__device__ __align__(256) unsigned char g_setup[kSetupSlots][(sizeof(Setup) + 255) & ~size_t(255)];
std::mutex g_setup_lock;
uint32_t g_setup_used[kSetupDevices];

class SetupSlot {
 public:
  SetupSlot() {
    std::lock_guard<std::mutex> guard(g_setup_lock);
    if (cudaGetDevice(&dev_) != cudaSuccess || dev_ < 0 || dev_ >= kSetupDevices) {
      cudaGetLastError();
      return;
    }
    // asked for on each call: a device reset moves the symbol
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_setup) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    base_ = static_cast<char*>(p);
    for (int k = 0; k < kSetupSlots && slot_ < 0; ++k)
      if (!(g_setup_used[dev_] >> k & 1u)) slot_ = k;
    if (slot_ >= 0) g_setup_used[dev_] |= 1u << slot_;
  }
  ~SetupSlot() {
    std::lock_guard<std::mutex> guard(g_setup_lock);
    if (slot_ >= 0) g_setup_used[dev_] &= ~(1u << slot_);
  }
  SetupSlot(const SetupSlot&) = delete;
  SetupSlot& operator=(const SetupSlot&) = delete;
  void* get() const { return slot_ >= 0 ? base_ + slot_ * sizeof g_setup[0] : nullptr; }

 private:
  char* base_ = nullptr;
  int dev_ = -1, slot_ = -1;
};
}  // namespace

extern "C" int rr_accumulate_returns(const uint32_t* column, const uint32_t* bin, const float* energy, uint64_t n,
                                     uint32_t n_columns, uint32_t n_bins, float* out) {
  if (!out || (n && (!column || !bin || !energy))) return fail(RR_ERR_INVALID_ARG, "NULL buffer");
  if (n_columns < 1 || n_columns > kMaxColumns) return fail(RR_ERR_INVALID_ARG, "n_columns must be in [1, 2^18]");
  if (n_bins < 1 || n_bins > RR_MAX_BINS) return fail(RR_ERR_INVALID_ARG, "n_bins must be in [1, 16384]");
  if (n >= (1ull << 31)) return fail(RR_ERR_INVALID_ARG, "at most 2^31 - 1 returns");
  cudaStream_t st = current_stream();
  const size_t img_bytes = (size_t)n_columns * n_bins * sizeof(float);
  // Buffers of this device are read and written where they are; others (host
  // memory, another device's, or not aligned to their elements) go through
  // the scratch of this call, one allocation (none when all are): [column][bin][energy][image]
  // [setup].  Nine allocations, the copies of device inputs and their packing
  // into records were most of a call (1.5M returns into 400 columns: 679 us).
  const bool own_col = usable_here(column), own_bin = usable_here(bin), own_e = usable_here(energy);
  // an image over its own inputs is made apart
  auto over_out = [&](const void* p) {
    const uintptr_t i0 = reinterpret_cast<uintptr_t>(p), o0 = reinterpret_cast<uintptr_t>(out);
    return i0 < o0 + img_bytes && o0 < i0 + n * 4;
  };
  const bool own_out = usable_here(out) && !over_out(column) && !over_out(bin) && !over_out(energy);
  const size_t nn = n ? n : 1;
  auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
  const size_t in_bytes = up(nn * 4);
  size_t off = 0, o_col = 0, o_bin = 0, o_e = 0, o_img = 0;
  if (!own_col) o_col = off, off += in_bytes;
  if (!own_bin) o_bin = off, off += in_bytes;
  if (!own_e) o_e = off, off += in_bytes;
  if (!own_out) o_img = off, off += up(img_bytes);
  const SetupSlot slot;   // given back after the last wait of every path below
  const size_t o_setup = off;
  if (!slot.get()) off += up(sizeof(Setup));
  char* w = nullptr;
  cudaError_t e = off ? dev_malloc(&w, off) : cudaSuccess;
  if (e != cudaSuccess) {
    cudaGetLastError();
    return cuda_fail(e, "accumulating the returns");
  }
  auto cleanup = [&]() {
    cudaStreamSynchronize(st);
    if (w) cudaFree(w);
  };
  const uint32_t* d_col = own_col ? column : (const uint32_t*)(w + o_col);
  const uint32_t* d_bin = own_bin ? bin : (const uint32_t*)(w + o_bin);
  const float* d_e = own_e ? energy : (const float*)(w + o_e);
  float* d_img = own_out ? out : (float*)(w + o_img);
  Setup* d_setup = (Setup*)(slot.get() ? slot.get() : w + o_setup);
  if (n && !own_col) e = cudaMemcpyAsync(w + o_col, column, n * 4, cudaMemcpyDefault, st);
  if (e == cudaSuccess && n && !own_bin) e = cudaMemcpyAsync(w + o_bin, bin, n * 4, cudaMemcpyDefault, st);
  if (e == cudaSuccess && n && !own_e) e = cudaMemcpyAsync(w + o_e, energy, n * 4, cudaMemcpyDefault, st);
  Setup setup;
  memset(&setup, 0, sizeof setup);
  setup.desc.dims = make_uint4(n_columns, 1u, 1u, n_bins);
  setup.desc.offs = make_uint4(0u, 0u, kNone, 0u);
  setup.desc.image = d_img;
  setup.pre[3] = n_columns;
  setup.ctr.rec_start[1] = (uint32_t)n;
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_setup, &setup, sizeof setup, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && n) {
    k_check_returns<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(d_col, (uint32_t)n, n_columns, &d_setup->bad);
    e = cudaGetLastError();
  }
  // the check's answer before anything is written to the output
  uint32_t bad = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&bad, &d_setup->bad, 4, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    cleanup();
    return cuda_fail(e, "accumulating the returns");
  }
  if (bad) {
    cleanup();
    return fail(RR_ERR_INVALID_ARG, "column must be non-decreasing and below n_columns");
  }
  ScanArgs a;
  memset(&a, 0, sizeof a);
  a.desc = &d_setup->desc;
  a.ray0 = d_setup->pre;
  a.col0 = d_setup->pre + 2;
  a.n_scans = 1;
  a.n_cols = n_columns;
  a.max_bounces = 1;
  a.max_bins = n_bins;
  a.raw_column = d_col;
  a.raw_bin = d_bin;
  a.raw_energy = d_e;
  a.ctr = &d_setup->ctr;
  e = launch_image(a, false, st);
  if (e == cudaSuccess && !own_out) e = cudaMemcpyAsync(out, d_img, img_bytes, cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    cleanup();
    return cuda_fail(e, "accumulating the returns");
  }
  if (w) cudaFree(w);
  return RR_OK;
}
