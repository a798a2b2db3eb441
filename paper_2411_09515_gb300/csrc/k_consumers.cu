// The two consumers of the separated background (Sections 3 and 4):
// sparsification (compact the kept pixels of each frame, ascending index)
// and peak picking (local maxima among kept pixels with enough kept
// neighbours), both driven by a per-frame kept-pixel bitmap (1 bit / pixel).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sep_device.cuh"
#include "sep_internal.h"

namespace sep {
namespace {

// Value of pixel i of launch frame f: a float frame's own word without a norm
// (one read, where the staged copy takes the slot's first), the staged copy
// when the call staged the batch, else recomputed from the frame (the same
// IEEE sequence).
template <int DT, bool NORM>
__device__ __forceinline__ float value_of(const PixArgs& p, const void* frame, int64_t f, int64_t i) {
  if (DT == SEP_DTYPE_F32 && !NORM) return __ldg(reinterpret_cast<const float*>(frame) + i);
  if (p.stage) return __ldg(p.stage + f * p.npos + __ldg(p.pos_of + i));
  return pixel_value<DT, NORM>(frame, i, p.npix, p.ped, p.gain, p.norm);
}

// Exclusive scan of one int per thread over a block of NT threads.
template <int NT>
__device__ __forceinline__ int block_exclusive_scan(int x, int* total, int* sh) {
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) sh[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int v = lane < NW ? sh[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    if (lane < NW) sh[lane] = v;
  }
  __syncthreads();
  const int base = warp > 0 ? sh[warp - 1] : 0;
  *total = sh[NW - 1];
  __syncthreads();
  return base + inc - x;
}

__global__ void k_thresholds(const float* mean, const float* sigma, float k_pick, int64_t n, float* thr) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) thr[i] = __double2float_rd((double)mean[i] + (double)k_pick * (double)sigma[i]);
}

// Level of pixel i in a per-bin profile p (bin level, or the radial
// interpolation between the bins a and a + 1 with weight t on the upper).
__device__ __forceinline__ float profile_at(const float* p, int32_t b, const int32_t* ia, const float* it, int64_t i,
                                            int32_t nbins) {
  if (!ia) return __ldg(p + b);
  const int32_t a = __ldg(ia + i);
  const float t = __ldg(it + i);
  const float hi = a + 1 < nbins ? __ldg(p + a + 1) : 0.0f;
  return __fadd_rn(__fmul_rn(__fsub_rn(1.0f, t), __ldg(p + a)), __fmul_rn(t, hi));
}

// Pixels that a thread of the image-order kernels takes from each frame, 32
// apart: a warp covers 128 consecutive pixels, every access of it is
// coalesced whatever the alignment of the frame, and a ballot is a word of
// the bitmap.
constexpr int kPixPerThread = 4;
constexpr int kImageThreads = 256;
constexpr int kPixPerCta = kImageThreads * kPixPerThread;

// Frames a thread of the image-order kernels walks: the pixels' tables
// (calibration, bins) are read once for all of them, as long as the grid
// still holds four waves of 8 CTAs on every multiprocessor; the groups of a
// batch are even.
int32_t frames_per_thread(int32_t n_frames, int64_t ctas) {
  const int32_t most = (int32_t)std::min<int64_t>(std::max<int64_t>(ctas * n_frames / (152 * 8 * 4), 1), 16);
  const int32_t groups = (n_frames + most - 1) / most;
  return (n_frames + groups - 1) / groups;
}

// A source of pixel values beside the SEP_DTYPE_*: the batch's staged copy
// alone, for calls whose outputs may overwrite the frames (a sector a pixel
// read, against a word of the frame: 1814 against 333 us for 64 corrected raw
// Jungfrau-4M frames).
constexpr int kStaged = -1;

// Four pixels of a warp's 128 (32 apart from i0; VEC: consecutive, one vector
// access, for float images of a multiple of 4 pixels at an aligned address),
// for the frames a thread walks: their tables, and their values frame by
// frame. Pixels past the last read the last one's words, and pixels without a
// bin take no part in the tests of value(): neither costs the loop over the
// frames a branch.
template <int DT, bool NORM, bool VEC = false>
struct PixelColumn {
  static constexpr int kStep = VEC ? 1 : 32;
  Level0 cal[kPixPerThread];
  float nm[kPixPerThread];
  uint32_t i[kPixPerThread];   // the pixels, at most npix - 1 (32-bit offsets: one instruction an address)
  bool valid[kPixPerThread];   // inside the image, and with a bin
  __device__ __forceinline__ PixelColumn(const PixArgs& p, int64_t i0) {
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k) {
      i[k] = (uint32_t)min(i0 + kStep * k, p.npix - 1);
      valid[k] = i0 + kStep * k < p.npix && __ldg(p.bop + i[k]) >= 0;
      nm[k] = 1.0f;
      if (DT == SEP_DTYPE_U16_JF) {
        cal[k].set(__ldg(p.ped + i[k]), __ldg(p.gain + i[k]));
        if (!valid[k]) cal[k].limit = 0xffffffffu;
      }
      if (NORM) nm[k] = __ldg(p.norm + i[k]);
    }
  }
  __device__ __forceinline__ const void* frame(const PixArgs& p, int64_t f) const {
    return p.fptr ? (const void*)p.fptr[f] : frame_ptr<DT>(p.frames, f, p.npix);
  }
  __device__ __forceinline__ void load(const PixArgs& p, int64_t f, uint32_t (&w)[kPixPerThread]) const {
    const void* fr = frame(p, f);
    if (VEC) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(fr) + i[0]));
      w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
      return;
    }
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k) {
      if (DT == SEP_DTYPE_U16_JF) w[k] = __ldg(reinterpret_cast<const uint16_t*>(fr) + i[k]);
      else w[k] = __float_as_uint(__ldg(reinterpret_cast<const float*>(fr) + i[k]));
    }
  }
  // the values of frame f's words u: pixel_value(), bit for bit, for the
  // valid pixels
  __device__ __forceinline__ void values(const PixArgs& p, int64_t f, const uint32_t (&u)[kPixPerThread],
                                         float (&x)[kPixPerThread]) const {
    bool rest = false;
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k) {
      x[k] = DT == SEP_DTYPE_U16_JF ? cal[k].value(u[k]) : __uint_as_float(u[k]);
      if (DT == SEP_DTYPE_U16_JF) rest = rest || u[k] >= cal[k].limit;
      if (NORM) x[k] = __fdiv_rn(x[k], nm[k]);
    }
    if (DT != SEP_DTYPE_U16_JF || !rest) return;
    // another gain level or an unusual calibration
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k)
      if (u[k] >= cal[k].limit)
        x[k] = pixel_value<DT, NORM>(frame(p, f), i[k], p.npix, p.ped, p.gain, p.norm);
  }
  // fn(f, values) for the frames [f0, f1), the next frame's words under way
  template <class F>
  __device__ __forceinline__ void walk(const PixArgs& p, int32_t f0, int32_t f1, F&& fn) const {
    uint32_t w[kPixPerThread];
    load(p, f0, w);
    for (int32_t f = f0; f < f1; ++f) {
      float x[kPixPerThread];
      values(p, f, w, x);
      if (f + 1 < f1) load(p, f + 1, w);
      fn(f, x);
    }
  }
};

// The same from the staged copy.
template <>
struct PixelColumn<kStaged, false, false> {
  uint32_t i[kPixPerThread], slot[kPixPerThread];
  bool valid[kPixPerThread];
  __device__ __forceinline__ PixelColumn(const PixArgs& p, int64_t i0) {
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k) {
      i[k] = (uint32_t)min(i0 + 32 * k, p.npix - 1);
      const int32_t q = __ldg(p.pos_of + i[k]);
      valid[k] = i0 + 32 * k < p.npix && q >= 0;
      slot[k] = (uint32_t)max(q, 0);
    }
  }
  template <class F>
  __device__ __forceinline__ void walk(const PixArgs& p, int32_t f0, int32_t f1, F&& fn) const {
    for (int32_t f = f0; f < f1; ++f) {
      float x[kPixPerThread];
#pragma unroll
      for (int k = 0; k < kPixPerThread; ++k) x[k] = __ldg(p.stage + f * p.npos + slot[k]);
      fn(f, x);
    }
  }
};

// v > RD32(m + k s) with the sum in binary64: for a binary32 v that is
// v > RN64(m + k s). Decided in binary32 when v is further from the sum than
// binary32 can be off it (t is within 2^-24 of the sum, the difference within
// 2^-24 of itself), else, and for NaN and infinities, in binary64, whose
// rate on this GPU is a small fraction of binary32's (out of line, or the
// compiler computes both sides of the choice: 242 us instead of 70 for the
// float frames named below).
static __device__ __noinline__ bool above_threshold64(float v, float m, float s, float k) {
  return v > __double2float_rd((double)m + (double)k * (double)s);
}
__device__ __forceinline__ bool above_threshold(float v, float m, float s, float k) {
  const float t = __fmaf_rn(k, s, m);
  const float d = __fsub_rn(v, t);
  bool above = d > 0.0f;
  if (!(fabsf(d) > __fmaf_rn(0x1p-21f, fabsf(t), 0x1p-120f))) above = above_threshold64(v, m, s, k);
  return above;
}

// Kept-pixel bitmap of a batch in image order (Section 3). The threshold of a
// pixel is its bin's (thr [F][nbins]), or, INTERP, RD(mu(x) + k_pick sigma(x))
// from the frame's profile interpolated at the pixel centre. Values are
// corrected from the frame's words: in image order those are one contiguous
// stream, where the staged copy of a batch would cost a sector a pixel. A
// warp writes four words of the bitmap at once, every word of the row
// (pixels past the last count as dropped).
//
// One pixel a thread and frame was bound by its instructions: an IEEE
// division with its tables, a bin, and with INTERP a binary64 sum a pixel
// (16 raw Jungfrau-4M frames: 314 -> 99 us; INTERP, 29 float frames of 1.1
// Mpixel: 301 -> 70 us). It still is: 73 % of the issue slots are taken. The
// register bound keeps 40 warps on a multiprocessor (76 registers without
// it, 149 us).
template <int DT, bool NORM, bool INTERP>
__global__ void __launch_bounds__(kImageThreads, 5) k_mark(PixArgs p, int32_t n_frames, int32_t frames_per_cta,
                                                        int32_t nbins, const float* thr, const float* mean,
                                                        const float* sigma, float k_pick, uint32_t* bitmap,
                                                        int64_t words) {
  const int lane = threadIdx.x & 31;
  const int64_t w0 = ((int64_t)blockIdx.x * (kImageThreads / 32) + (threadIdx.x >> 5)) * kPixPerThread;
  if (w0 >= words) return;   // (words is a multiple of 8)
  PixelColumn<DT, NORM> px(p, w0 * 32 + lane);
  uint32_t b[kPixPerThread];   // the bin (INTERP: the lower bin)
  float t[kPixPerThread];
  uint32_t valid[kPixPerThread];
#pragma unroll
  for (int k = 0; k < kPixPerThread; ++k) {
    valid[k] = __ballot_sync(0xffffffffu, px.valid[k]);
    t[k] = INTERP ? __ldg(p.it + px.i[k]) : 0.0f;
    b[k] = (uint32_t)(INTERP ? __ldg(p.ia + px.i[k]) : max(__ldg(p.bop + px.i[k]), 0));
  }
  const int32_t f0 = blockIdx.y * frames_per_cta, f1 = min(f0 + frames_per_cta, n_frames);
  px.walk(p, f0, f1, [&](int32_t f, const float (&x)[kPixPerThread]) {
    const int64_t row = INTERP && p.orow ? p.orow[f] : f * (int64_t)nbins;
    const float* mu = INTERP ? mean + row : thr + row;   // the frame's profile, or its thresholds
    const float* sd = INTERP ? sigma + row : nullptr;
    uint32_t m[kPixPerThread];
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k) {
      bool keep;
      if (INTERP) {
        const bool up = (int32_t)b[k] + 1 < nbins;
        const float m0 = __ldg(mu + b[k]), m1 = up ? __ldg(mu + b[k] + 1) : 0.0f;
        const float s0 = __ldg(sd + b[k]), s1 = up ? __ldg(sd + b[k] + 1) : 0.0f;
        const float u = __fsub_rn(1.0f, t[k]);
        keep = above_threshold(x[k], __fadd_rn(__fmul_rn(u, m0), __fmul_rn(t[k], m1)),
                               __fadd_rn(__fmul_rn(u, s0), __fmul_rn(t[k], s1)), k_pick);
      } else {
        keep = x[k] > __ldg(mu + b[k]);
      }
      m[k] = __ballot_sync(0xffffffffu, keep) & valid[k];
    }
    if (lane == 0) *reinterpret_cast<uint4*>(bitmap + f * words + w0) = make_uint4(m[0], m[1], m[2], m[3]);
  });
}
static_assert(kPixPerThread == 4, "a warp writes its four words as one vector");

// Corrected frames in image order, NaN where a pixel has no bin: one pass
// over the frames (through the staged copy and back to image order it was a
// write and a gather of 1.5 values a pixel more: 1814 us for 64 raw
// Jungfrau-4M frames). Float frames, and raw frames that the kernel below
// does not take (387 us for those 64).
template <int DT, bool NORM, bool VEC>
__global__ void __launch_bounds__(kImageThreads, 5) k_correct(PixArgs p, int32_t n_frames, int32_t frames_per_cta,
                                                              float* out) {
  const int64_t i0 = (int64_t)blockIdx.x * kPixPerCta +
                     (VEC ? threadIdx.x * kPixPerThread
                          : (threadIdx.x >> 5) * (32 * kPixPerThread) + (threadIdx.x & 31));
  if (i0 >= p.npix) return;
  PixelColumn<DT, NORM, VEC> px(p, i0);
  const int32_t f0 = blockIdx.y * frames_per_cta, f1 = min(f0 + frames_per_cta, n_frames);
  px.walk(p, f0, f1, [&](int32_t f, const float (&v)[kPixPerThread]) {
    float* o = out + (int64_t)f * p.npix;
    float x[kPixPerThread];
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k) x[k] = px.valid[k] ? v[k] : __int_as_float(0x7fc00000);
    if (VEC) {
      *reinterpret_cast<float4*>(o + px.i[0]) = make_float4(x[0], x[1], x[2], x[3]);
    } else {
#pragma unroll
      for (int k = 0; k < kPixPerThread; ++k)
        if (i0 + 32 * k < p.npix) o[px.i[k]] = x[k];
    }
  });
}

// The same for raw frames of a multiple of 8 pixels at 16-byte aligned
// addresses, eight consecutive pixels a thread: one 16-byte load and two
// 16-byte stores, and one test of the packed words for another gain level.
// Bound by memory (64 raw Jungfrau-4M frames: 333 us, 5.2 TB/s of words read
// and values written; with four pixels a thread 387 us, bound by the
// addresses and tests a pixel).
template <bool NORM>
__global__ void __launch_bounds__(kImageThreads, 4) k_correct_raw8(PixArgs p, int32_t n_frames,
                                                                   int32_t frames_per_cta, float* out) {
  const uint32_t i0 = 8 * (blockIdx.x * kImageThreads + threadIdx.x);
  if (i0 >= p.npix) return;
  Level0 cal[8];
  float nm[8];
  uint32_t valid = 0, usual = 0;   // bit k: pixel i0 + k has a bin; its level-0 words need no division
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    cal[k].set(__ldg(p.ped + i0 + k), __ldg(p.gain + i0 + k));
    nm[k] = NORM ? __ldg(p.norm + i0 + k) : 1.0f;
    if (__ldg(p.bop + i0 + k) >= 0) valid |= 1u << k;
    if (cal[k].limit || !((valid >> k) & 1u)) usual |= 1u << k;
  }
  const int32_t f0 = blockIdx.y * frames_per_cta, f1 = min(f0 + frames_per_cta, n_frames);
  const uint16_t* src = reinterpret_cast<const uint16_t*>(p.frames) + (int64_t)f0 * p.npix + i0;
  float* dst = out + (int64_t)f0 * p.npix + i0;
  uint4 v = __ldg(reinterpret_cast<const uint4*>(src));
  for (int32_t f = f0; f < f1; ++f, dst += p.npix) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    src += p.npix;
    if (f + 1 < f1) v = __ldg(reinterpret_cast<const uint4*>(src));   // under way meanwhile
    float x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      x[k] = cal[k].value(k & 1 ? w[k >> 1] >> 16 : w[k >> 1] & 0xffffu);
      if (NORM) x[k] = __fdiv_rn(x[k], nm[k]);
    }
    if (((w[0] | w[1] | w[2] | w[3]) & 0xc000c000u) || usual != 0xffu) {
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (((k & 1 ? w[k >> 1] >> 16 : w[k >> 1]) & 0xc000u) || !((usual >> k) & 1u))
          x[k] = pixel_value<SEP_DTYPE_U16_JF, NORM>(frame_ptr<SEP_DTYPE_U16_JF>(p.frames, f, p.npix), i0 + k, p.npix,
                                                     p.ped, p.gain, p.norm);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (!((valid >> k) & 1u)) x[k] = __int_as_float(0x7fc00000);
    reinterpret_cast<float4*>(dst)[0] = make_float4(x[0], x[1], x[2], x[3]);
    reinterpret_cast<float4*>(dst)[1] = make_float4(x[4], x[5], x[6], x[7]);
  }
}

// Tiles of the ordered compaction. The emitting CTAs wait for a chain of
// reads (counts, words, slots, values): several of 256 threads on every
// multiprocessor overlap theirs, where one or two of 1024 threads (8192 words
// a tile) left it idle: 48 raw Jungfrau-4M frames 101 -> 97 us, 4 frames 27 ->
// 25 us, one 16M float frame 20 -> 13 us.
constexpr int kCompactThreads = 256;
constexpr int64_t kTileWords = (int64_t)kCompactThreads * 8;   // bitmap words per CTA
// ... and tiles of 1024 threads where there are at most kWideCtas: those of a
// small detector or a few frames do not fill the GPU, and where a threshold
// keeps most pixels of a tile its threads take them 2048 at a time, round
// after round (every pixel of one 300 x 301 frame kept: 183 -> 41 us, of one
// raw Jungfrau-4M frame 227 -> 64, of seven 302 -> 168; few kept: the same).
// Beyond that the rounds of one tile hide behind other tiles', and the wide
// tiles are slower where few pixels are kept (40 frames: 306 against 277 us).
constexpr int kWideThreads = 1024;
constexpr int64_t kWideCtas = 152 * 4;

// Phase 1 of the ordered compaction: kept pixels per tile of the bitmap.
__global__ void __launch_bounds__(256) k_count_bits(const uint32_t* bitmap, int64_t words, int32_t* tile_cnt,
                                                    int32_t n_tiles) {
  const int64_t f = blockIdx.y;
  const int64_t w0 = (int64_t)blockIdx.x * kTileWords;
  const uint32_t* bm = bitmap + f * words;
  int cnt = 0;
  for (int64_t w = w0 + 4 * (int64_t)threadIdx.x; w < w0 + kTileWords && w < words; w += 4 * 256) {
    // words is a multiple of 8, so a 4-word vector never runs past the frame
    const uint4 q = *reinterpret_cast<const uint4*>(bm + w);
    cnt += __popc(q.x) + __popc(q.y) + __popc(q.z) + __popc(q.w);
  }
  __shared__ int sh[8];
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int i = 0; i < 8; ++i) t += sh[i];
    tile_cnt[f * n_tiles + blockIdx.x] = t;
  }
}

// Phase 2: each CTA writes its tile's kept pixels (ascending) after the
// pixels of all earlier tiles of the frame; values are recomputed from the
// frame exactly as the clip kernel computed them.
template <int DT, bool NORM, int NT>
__global__ void __launch_bounds__(NT) k_emit_kept(PixArgs p, const uint32_t* bitmap, int64_t words,
                                                               const int32_t* tile_cnt, int32_t n_tiles, int32_t* idx,
                                                               float* val, int64_t cap, int32_t* n_kept,
                                                               int32_t* status) {
  constexpr int kWordsPerThread = (int)(kTileWords / NT);
  constexpr int kEmitList = 8 * NT;   // kept pixels a CTA lists in shared memory at once
  __shared__ int sh[NT / 32];
  __shared__ int64_t base_s;
  const int64_t f = blockIdx.y;
  const int tile = blockIdx.x;
  if (threadIdx.x < 32) {
    int64_t before = 0, all = 0;
    for (int t = threadIdx.x; t < n_tiles; t += 32) {
      const int c = tile_cnt[f * n_tiles + t];
      all += c;
      if (t < tile) before += c;
    }
    for (int o = 16; o > 0; o >>= 1) {
      before += __shfl_xor_sync(0xffffffffu, before, o);
      all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    if (threadIdx.x == 0) {
      base_s = before;
      if (tile == 0) {
        n_kept[p.fidx ? p.fidx[f] : f] = (int32_t)all;
        if (all > cap) atomicOr(status, SEP_DEV_CAPACITY);
      }
    }
  }
  __syncthreads();
  const int64_t base = base_s;
  if (base >= cap) return;
  const uint32_t* bm = bitmap + f * words;
  const void* frame = p.fptr ? (const void*)p.fptr[f] : frame_ptr<DT>(p.frames, f, p.npix);
  const int64_t g = p.fidx ? p.fidx[f] : f;   // output row of this frame
  const int64_t w0 = (int64_t)tile * kTileWords + (int64_t)threadIdx.x * kWordsPerThread;
  uint32_t wv[kWordsPerThread];
  if (kWordsPerThread == 8 && w0 + kWordsPerThread <= words) {
    const uint4* q = reinterpret_cast<const uint4*>(bm + w0);
    const uint4 a = q[0], b = q[1];
    const uint32_t ab[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int j = 0; j < kWordsPerThread; ++j) wv[j] = ab[j];
  } else {
#pragma unroll
    for (int j = 0; j < kWordsPerThread; ++j) wv[j] = (w0 + j < words) ? bm[w0 + j] : 0u;
  }
  int cnt = 0;
#pragma unroll
  for (int j = 0; j < kWordsPerThread; ++j) cnt += __popc(wv[j]);
  int tile_total;
  const int first = block_exclusive_scan<NT>(cnt, &tile_total, sh);   // this thread's first, in the tile
  // The tile's kept pixels go through a shared list, kEmitList at a time:
  // each thread lists its own pixels at their ranks, then consecutive
  // threads take consecutive entries, so the value loads of the whole list
  // are in flight together and the stores are coalesced.
  __shared__ int32_t lst[kEmitList];
  const int64_t n_tile = (int64_t)tile_total < cap - base ? (int64_t)tile_total : cap - base;
  for (int r0 = 0; r0 < n_tile; r0 += kEmitList) {
    if (first < r0 + kEmitList && first + cnt > r0) {
      int rank = first;
#pragma unroll
      for (int j = 0; j < kWordsPerThread; ++j) {
        uint32_t m = wv[j];
        while (m) {
          const int bit = __ffs(m) - 1;
          m &= m - 1u;
          if (rank >= r0 && rank < r0 + kEmitList) lst[rank - r0] = (int32_t)((w0 + j) * 32 + bit);
          ++rank;
        }
      }
    }
    __syncthreads();
    const int nr = (int)(n_tile - r0 < kEmitList ? n_tile - r0 : kEmitList);
    for (int k = threadIdx.x; k < nr; k += NT) {
      const int64_t pos = base + r0 + k;
      const int32_t i = lst[k];
      idx[g * cap + pos] = i;
      val[g * cap + pos] = value_of<DT, NORM>(p, frame, f, i);
    }
    __syncthreads();
  }
}

// Frames a thread walks from which the dense background is better read in
// columns: by bin without deviates, and interpolated.
constexpr int32_t kDenseFrames = 8;
constexpr int32_t kDenseSmoothFrames = 2;

// A pixel's level in a profile with its table in registers (b: its bin, or
// INTERP the lower one, t the weight on the upper, up: there is one).
template <bool INTERP>
__device__ __forceinline__ float profile_level(const float* p, uint32_t b, float t, bool up) {
  const float lo = __ldg(p + b);
  if (!INTERP) return lo;
  const float hi = up ? __ldg(p + b + 1) : 0.0f;
  return __fadd_rn(__fmul_rn(__fsub_rn(1.0f, t), lo), __fmul_rn(t, hi));
}

// Densification (Section 3): the background level of every binned pixel
// (its bin's mean, or RN(mean + RN(sigma z)) with the caller's deviates z;
// INTERP: both from the profile at the pixel centre), fill where a pixel has
// no bin. Four pixels a thread, 32 apart, for several frames: the bins and
// the interpolation table are read once for all of them, and the gathers of
// 32 neighbouring pixels' levels meet a few cache lines (one frame a thread,
// four consecutive pixels: 66 and, with INTERP and NOISE, 218 us for 16
// Jungfrau-4M frames; now 62 and 144 us, bound by the instructions a pixel).
template <bool NOISE, bool INTERP>
__global__ void __launch_bounds__(kImageThreads, NOISE ? 5 : 6) k_dense_background(
    const int32_t* bop, int64_t npix, int32_t nbins, int32_t n_frames, int32_t frames_per_cta, const float* mean,
    const float* sigma, const float* noise, float fill, const int32_t* ia, const float* it, float* out) {
  const int64_t i0 = (int64_t)blockIdx.x * kPixPerCta + (threadIdx.x >> 5) * (32 * kPixPerThread) + (threadIdx.x & 31);
  if (i0 >= npix) return;
  uint32_t i[kPixPerThread], b[kPixPerThread];   // the pixels (at most npix - 1), their (INTERP: lower) bins
  float t[kPixPerThread];
  bool valid[kPixPerThread], up[kPixPerThread];
#pragma unroll
  for (int k = 0; k < kPixPerThread; ++k) {
    i[k] = (uint32_t)min(i0 + 32 * k, npix - 1);
    const int32_t bk = __ldg(bop + i[k]);
    valid[k] = bk >= 0;
    b[k] = (uint32_t)(INTERP ? __ldg(ia + i[k]) : max(bk, 0));
    t[k] = INTERP ? __ldg(it + i[k]) : 0.0f;
    up[k] = (int32_t)b[k] + 1 < nbins;
  }
  const int32_t f0 = blockIdx.y * frames_per_cta, f1 = min(f0 + frames_per_cta, n_frames);
  float z[kPixPerThread];
  auto load = [&](int32_t f) {
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k) z[k] = NOISE ? __ldg(noise + (int64_t)f * npix + i[k]) : 0.0f;
  };
  load(f0);
  for (int32_t f = f0; f < f1; ++f) {
    const float* mu = mean + (int64_t)f * nbins;
    const float* sd = NOISE ? sigma + (int64_t)f * nbins : nullptr;
    float x[kPixPerThread];
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k) {
      // (profile_at, with the pixel's table in registers)
      auto level = [&](const float* p) {
        const float lo = __ldg(p + b[k]);
        if (!INTERP) return lo;
        const float hi = up[k] ? __ldg(p + b[k] + 1) : 0.0f;
        return __fadd_rn(__fmul_rn(__fsub_rn(1.0f, t[k]), lo), __fmul_rn(t[k], hi));
      };
      x[k] = level(mu);
      if (NOISE) x[k] = __fadd_rn(x[k], __fmul_rn(level(sd), z[k]));
      if (!valid[k]) x[k] = fill;
    }
    if (f + 1 < f1) load(f + 1);   // the next frame's deviates are under way meanwhile
    float* o = out + (int64_t)f * npix;
#pragma unroll
    for (int k = 0; k < kPixPerThread; ++k)
      if (i0 + 32 * k < npix) o[i[k]] = x[k];
  }
}

// The same for images of a multiple of 4 pixels at aligned addresses, four
// consecutive pixels of one frame a thread, one vector access each for bins,
// tables, deviates and output, with registers for every warp an SM holds. By
// bin there is little to keep over frames (whole calls with deviates, 64
// Jungfrau-4M frames: 542 us against 556 with the kernel above, 7 frames: 79
// against 83; without, 7 frames: 59 against 64, 16 frames equal, 64 frames
// 401 against 364); interpolated the tables are worth it from two frames a
// thread on (one frame: 14.4 us against 22.6, with deviates 18.6 against
// 25.8; sixteen: 133 against 120, with deviates 193 against 185).
template <bool NOISE, bool INTERP>
__global__ void __launch_bounds__(256) k_dense_background_vec(const int32_t* bop, int64_t npix, int32_t nbins,
                                                              const float* mean, const float* sigma,
                                                              const float* noise, float fill, const int32_t* ia,
                                                              const float* it, float* out) {
  const int64_t f = blockIdx.y;
  const int64_t i = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= npix) return;
  const int4 b4 = __ldg(reinterpret_cast<const int4*>(bop + i));
  int4 a4 = b4;
  float4 t4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), z4 = t4;
  if (INTERP) {
    a4 = __ldg(reinterpret_cast<const int4*>(ia + i));
    t4 = __ldg(reinterpret_cast<const float4*>(it + i));
  }
  if (NOISE) z4 = __ldg(reinterpret_cast<const float4*>(noise + f * npix + i));
  const int b[4] = {b4.x, b4.y, b4.z, b4.w}, a[4] = {a4.x, a4.y, a4.z, a4.w};
  const float t[4] = {t4.x, t4.y, t4.z, t4.w}, z[4] = {z4.x, z4.y, z4.z, z4.w};
  const float* mu = mean + f * nbins;
  const float* sd = NOISE ? sigma + f * nbins : nullptr;
  float x[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    x[k] = fill;
    if (b[k] >= 0) {
      auto level = [&](const float* p) { return profile_level<INTERP>(p, a[k], t[k], a[k] + 1 < nbins); };
      x[k] = level(mu);
      if (NOISE) x[k] = __fadd_rn(x[k], __fmul_rn(level(sd), z[k]));
    }
  }
  *reinterpret_cast<float4*>(out + f * npix + i) = make_float4(x[0], x[1], x[2], x[3]);
}

// ... then the recorded values of the kept pixels.
__global__ void __launch_bounds__(256) k_dense_scatter(const int32_t* idx, const float* val, int64_t cap,
                                                       const int32_t* n_kept, int64_t npix, float* out) {
  const int64_t f = blockIdx.y;
  int64_t n = n_kept[f];
  n = n < 0 ? 0 : (n > cap ? cap : n);
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = idx[f * cap + k];
    if (i >= 0 && i < npix) out[f * npix + i] = val[f * cap + k];
  }
}

// Veto (Section 4): the frames with at least min_peaks peaks, ascending, by
// one CTA scanning the counts in tiles of its size.
__global__ void __launch_bounds__(1024) k_veto(int32_t n_frames, const int32_t* n_peaks, int32_t min_peaks,
                                               int32_t* list, int32_t* n_pass) {
  __shared__ int sh[32];
  int base = 0;
  for (int f0 = 0; f0 < n_frames; f0 += 1024) {
    const int f = f0 + threadIdx.x;
    const int pass = f < n_frames && n_peaks[f] >= min_peaks;
    int total;
    const int pos = base + block_exclusive_scan<1024>(pass, &total, sh);
    if (pass) list[pos] = f;
    base += total;
  }
  if (threadIdx.x == 0) *n_pass = base;
}

// Row j of dst = row list[j] of src for j < *n_pass (32-bit words; 16-byte
// vectors when rows and bases allow).
template <bool VEC>
__global__ void __launch_bounds__(256) k_compact_rows(const int32_t* list, const int32_t* n_pass, int64_t row_words,
                                                      const uint32_t* src, uint32_t* dst) {
  const int64_t j = blockIdx.y;
  if (j >= *n_pass) return;
  const int64_t r = list[j];
  if (r < 0 || r >= gridDim.y) return;   // (a caller's list is not trusted)
  const uint32_t* s = src + r * row_words;
  uint32_t* d = dst + j * row_words;
  if (VEC) {
    const int64_t n4 = row_words >> 2;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += (int64_t)gridDim.x * blockDim.x)
      reinterpret_cast<uint4*>(d)[q] = __ldg(reinterpret_cast<const uint4*>(s) + q);
  } else {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < row_words;
         q += (int64_t)gridDim.x * blockDim.x)
      d[q] = __ldg(s + q);
  }
}

// Indices outside the detector are ignored (a caller's list is not trusted).
__global__ void k_scatter_list(const int32_t* idx, const int32_t* n_kept, int64_t kcap, int64_t npix,
                               uint32_t* bitmap, int64_t words) {
  const int64_t f = blockIdx.y;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t n = n_kept[f];
  if (n > kcap) n = kcap;
  if (k < n) {
    int32_t i = idx[f * kcap + k];
    if (i >= 0 && i < npix) atomicOr(bitmap + f * words + (i >> 5), 1u << (i & 31));
  }
}

constexpr int kPeakThreads = 256;
constexpr int kPeakChunk = 256;          // kept entries per flag chunk (8 flag words)
constexpr int kPeakList = 2048;          // peaks a record CTA lists in shared memory at once
constexpr int kOwnTest = 4;              // (see k_peak_flags)
constexpr int kPeakSlices = 8;           // slices of a frame's records at least
constexpr int kPeakCtas = 152 * 8;       // CTAs wanted of either peak kernel (8 of 256 threads fit a multiprocessor)

// Bits [j, j + w) of a frame's bitmap, w <= 15 (a second word is read only
// where the run crosses into it, so no word past the run's last bit is read).
__device__ __forceinline__ uint32_t bit_run(const uint32_t* bm, int64_t j, int w) {
  const int sh = (int)(j & 31);
  const uint32_t* q = bm + (j >> 5);
  const uint32_t a = __ldg(q);
  const uint32_t b = sh + w > 32 ? __ldg(q + 1) : 0u;
  return __funnelshift_r(a, b, sh) & ((1u << w) - 1u);
}

// Value of pixel j of launch frame f where the pixel is valid (it has a bin,
// hence a centre entry), else ok = false.
template <int DT, bool NORM>
__device__ __forceinline__ float valid_value(const PixArgs& p, const void* frame, int64_t f, int64_t j, bool& ok) {
  if (p.stage && (DT != SEP_DTYPE_F32 || NORM)) {
    const int32_t q = __ldg(p.pos_of + j);
    ok = q >= 0;
    return ok ? __ldg(p.stage + f * p.npos + q) : 0.0f;
  }
  ok = __ldg(p.bop + j) >= 0;
  return ok ? pixel_value<DT, NORM>(frame, j, p.npix, p.ped, p.gain, p.norm) : 0.0f;
}

// Phase 1 of the peaks: one flag bit per kept-list entry, and peaks per chunk
// of 256. A kept pixel is a peak (Section 4) if its patch holds at least
// min_count kept pixels and it is the maximum of the patch's valid pixels
// (ties: lowest index).
//
// The kernel is bound by the latency of dependent gathers. A thread counts
// its pixel's kept neighbours a patch row at a time (a run of bitmap bits and
// a population count). Where few entries of a warp have enough of them (about
// 1 in 50 at the azimuthal model's thresholds), the warp tests them together,
// one lane per patch pixel and as many candidates at once as fit the 32
// lanes, so all their values are in flight at once instead of one neighbour
// after another on one lane. That costs every candidate its whole patch:
// where its rounds would come to more than 1 / kOwnTest of the patch's pixels
// (many candidates: low thresholds, large patches with a low min_count), each
// lane tests its own candidate and stops at the first larger neighbour. The
// grid fills the GPU whatever the number of frames.
// 48 raw Jungfrau-4M frames, 90,000 kept pixels each: 145 -> 92 us, 4 frames:
// 84 -> 21 us. One pixel in six kept (the whole call): 3 x 3 patches 2497 us
// with every candidate tested by the warp, 1934 with the choice, 5 x 5 10270
// and 3650, 7 x 7 8300 and 5740; 15 x 15 15.2 ms by the warp, 18.1 ms a lane
// each. kOwnTest: 2 gives 7820 us for 7 x 7, 8 gives 17.4 ms for 15 x 15.
template <int DT, bool NORM>
__global__ void __launch_bounds__(kPeakThreads) k_peak_flags(PixArgs p, const uint32_t* bitmap, int64_t words,
                                                             const int32_t* idx, const int32_t* n_kept, int64_t kcap,
                                                             int32_t patch, int32_t min_count, uint32_t* flags,
                                                             int32_t* chunk_cnt, int32_t n_chunks) {
  __shared__ int32_t cpix_s[kPeakThreads];   // per warp: its candidates' pixels
  const int64_t f = blockIdx.y;
  const uint32_t* bm = bitmap + f * words;
  const void* frame = p.fptr ? (const void*)p.fptr[f] : frame_ptr<DT>(p.frames, f, p.npix);
  const int64_t g = p.fidx ? p.fidx[f] : f;
  int64_t n = n_kept[g];
  if (n > kcap) n = kcap;
  const int h = patch >> 1, area = patch * patch, mid = area >> 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = area <= 32 ? 32 / area : 1;   // candidates tested at once
  int32_t* cand = cpix_s + 32 * warp;
  for (int64_t ch = blockIdx.x; ch * kPeakChunk < n; ch += gridDim.x) {
    const int64_t k = ch * kPeakChunk + threadIdx.x;
    const int32_t i = k < n ? idx[g * kcap + k] : -1;
    bool enough = false;
    // (a batch's own list names valid pixels only)
    if (i >= 0 && i < p.npix && (p.stage || __ldg(p.bop + i) >= 0)) {
      const int r0 = i / p.cols, c0 = i - r0 * p.cols;
      const int rlo = max(r0 - h, 0), rhi = min(r0 + h, p.rows - 1);
      const int clo = max(c0 - h, 0), w = min(c0 + h, p.cols - 1) - clo + 1;
      int nk = 0;
      for (int r = rlo; r <= rhi; ++r) nk += __popc(bit_run(bm, (int64_t)r * p.cols + clo, w));
      enough = nk >= min_count;
    }
    const uint32_t em = __ballot_sync(0xffffffffu, enough);
    const int nc = __popc(em);
    bool peak = false;
    if (kOwnTest * ((nc + per - 1) / per) > area) {   // many candidates: each lane its own
      peak = enough;
      if (enough) {
        bool ok;
        const float vi = valid_value<DT, NORM>(p, frame, f, i, ok);
        const int cr = i / p.cols, cc = i - cr * p.cols;
        const int rhi = min(cr + h, p.rows - 1), clo = max(cc - h, 0), chi = min(cc + h, p.cols - 1);
        for (int r = max(cr - h, 0); r <= rhi && peak; ++r)
          for (int q = clo; q <= chi && peak; ++q) {
            const int64_t j = (int64_t)r * p.cols + q;
            if (j == i) continue;
            const float vj = valid_value<DT, NORM>(p, frame, f, j, ok);
            if (ok && !(vi > vj || (vi == vj && i < j))) peak = false;
          }
      }
    } else if (em) {
      const int rank = __popc(em & ((1u << lane) - 1u));
      if (enough) cand[rank] = i;
      __syncwarp();
      for (int c0 = 0; c0 < nc; c0 += per) {
        bool fine = true;   // no patch pixel of this lane beats its candidate
        const int sub = per > 1 ? lane / area : 0;
        const int c = c0 + sub;
        const bool active = sub < per && c < nc;
        const int64_t ci = active ? cand[c] : 0;
        const int cr = (int)(ci / p.cols), cc = (int)(ci - (int64_t)cr * p.cols);
        float vi = 0.0f;
        bool ok;
        if (per == 1 && active) vi = valid_value<DT, NORM>(p, frame, f, ci, ok);   // (the patch exceeds the warp)
        for (int o0 = 0; o0 < area; o0 += 32) {
          const int o = per > 1 ? lane - sub * area : o0 + lane;
          const int r = cr + o / patch - h, q = cc + o % patch - h;
          bool there = active && o < area && r >= 0 && r < p.rows && q >= 0 && q < p.cols;
          const int64_t j = (int64_t)r * p.cols + q;
          float vj = 0.0f;
          if (there) vj = valid_value<DT, NORM>(p, frame, f, j, there);
          if (per > 1) vi = __shfl_sync(0xffffffffu, vj, min(sub * area + mid, 31));
          if (there && j != ci && !(vi > vj || (vi == vj && ci < j))) fine = false;
          if (per > 1) break;
          if (__any_sync(0xffffffffu, !fine)) break;
        }
        const uint32_t b = __ballot_sync(0xffffffffu, fine);
        if (enough && rank >= c0 && rank < c0 + per) {
          const uint32_t want = per > 1 ? ((1u << area) - 1u) << ((rank - c0) * area) : 0xffffffffu;
          peak = (b & want) == want;
        }
      }
      __syncwarp();   // the list is rewritten by the warp's next chunk
    }
    const uint32_t peaks = __ballot_sync(0xffffffffu, peak);
    if (lane == 0) flags[f * ((int64_t)n_chunks * 8) + ch * 8 + warp] = peaks;
    const int c = __syncthreads_count(peak);
    if (threadIdx.x == 0) chunk_cnt[f * n_chunks + ch] = c;
  }
}

// Phase 2: every flagged entry writes its record at its rank in the frame:
// ascending pixel order, since the kept list ascends. The chunks of a frame
// are split over gridDim.x CTAs (a slice each, as many as fill the GPU: one
// CTA a frame left a 4-frame call on 4 multiprocessors); each counts the
// peaks of the chunks before its slice itself (a few hundred integers), lists
// its slice's flagged entries at their ranks in shared memory, kPeakList at a
// time, and writes the records one peak a thread.
// 48 Jungfrau-4M frames (750 peaks each): 54 -> 42 us; 4 frames: 55 -> 22 us;
// one 16M frame: 63 -> 20 us. A frame gets at least eight slices: with one each,
// 512 frames with a min_count of 1 took 7.3 ms in the whole call, now 5.6.
template <int DT, bool NORM, bool INTERP>
__global__ void __launch_bounds__(kPeakThreads) k_peak_emit(PixArgs p, int32_t nbins, const float* mean,
                                                            const float* sigma, const uint32_t* bitmap, int64_t words,
                                                            const int32_t* idx, const int32_t* n_kept, int64_t kcap,
                                                            int32_t patch, const uint32_t* flags,
                                                            const int32_t* chunk_cnt, int32_t n_chunks,
                                                            sep_peak* peaks, int64_t pcap, int32_t* n_peaks,
                                                            int32_t* status) {
  constexpr int kWarps = kPeakThreads / 32;
  __shared__ int sh[kWarps];
  __shared__ int64_t sum_s[2][kWarps];
  __shared__ int32_t base_s[kPeakThreads];
  __shared__ int32_t plist[kPeakList];
  const int64_t f = blockIdx.y;
  const int64_t g = p.fidx ? p.fidx[f] : f;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int64_t n = n_kept[g];
  if (n > kcap) n = kcap;
  const int nch = (int)((n + kPeakChunk - 1) / kPeakChunk);
  const int slice = (nch + (int)gridDim.x - 1) / (int)gridDim.x;
  const int first = min((int)blockIdx.x * slice, nch), last = min(first + slice, nch);
  const int32_t* cnt = chunk_cnt + f * n_chunks;
  int64_t before = 0, total = 0;
  for (int c = tid; c < nch; c += kPeakThreads) {
    const int x = cnt[c];
    total += x;
    if (c < first) before += x;
  }
  for (int o = 16; o > 0; o >>= 1) {
    before += __shfl_xor_sync(0xffffffffu, before, o);
    total += __shfl_xor_sync(0xffffffffu, total, o);
  }
  if (lane == 0) {
    sum_s[0][warp] = before;
    sum_s[1][warp] = total;
  }
  __syncthreads();
  before = total = 0;
#pragma unroll
  for (int w8 = 0; w8 < kWarps; ++w8) {
    before += sum_s[0][w8];
    total += sum_s[1][w8];
  }
  if (blockIdx.x == 0 && tid == 0) {
    n_peaks[g] = (int32_t)total;
    if (total > pcap) atomicOr(status, SEP_DEV_CAPACITY);
  }
  const uint32_t* bm = bitmap + f * words;
  const void* frame = p.fptr ? (const void*)p.fptr[f] : frame_ptr<DT>(p.frames, f, p.npix);
  const int64_t row = p.orow ? p.orow[f] : f * (int64_t)nbins;
  const float* mu = mean + row;
  const float* sd = sigma + row;
  const int h = patch >> 1;
  const uint32_t* fl = flags + f * ((int64_t)n_chunks * 8);
  // the slice's chunks, kPeakThreads at a time: their ranks, then their records
  for (int c0 = first; c0 < last && before < pcap; c0 += kPeakThreads) {
    const int nc = min(last - c0, kPeakThreads);
    int part;
    const int off = block_exclusive_scan<kPeakThreads>(tid < nc ? cnt[c0 + tid] : 0, &part, sh);
    base_s[tid] = off;
    __syncthreads();
    const int64_t room = pcap - before;
    const int n_out = (int64_t)part < room ? part : (int)room;
    for (int r0 = 0; r0 < n_out; r0 += kPeakList) {
      for (int c = warp; c < nc; c += kWarps) {
        int rank = base_s[c];
        if (rank >= r0 + kPeakList) break;   // (ranks ascend with the chunk)
        // a lane per flag word: ranks of the 8 words, then of their bits
        const uint32_t mw = lane < 8 ? __ldg(fl + (int64_t)(c0 + c) * 8 + lane) : 0u;
#pragma unroll
        for (int wd = 0; wd < 8; ++wd) {
          const uint32_t m = __shfl_sync(0xffffffffu, mw, wd);
          const int pos = rank + __popc(m & ((1u << lane) - 1u));
          if (((m >> lane) & 1u) && pos >= r0 && pos < r0 + kPeakList)
            plist[pos - r0] = (c0 + c) * kPeakChunk + wd * 32 + lane;
          rank += __popc(m);
        }
      }
      __syncthreads();
      const int nr = min(n_out - r0, kPeakList);
      for (int t = tid; t < nr; t += kPeakThreads) {
        const int64_t i = idx[g * kcap + plist[t]];
        const int rr0 = (int)(i / p.cols), cc0 = (int)(i - (int64_t)rr0 * p.cols);
        const int rlo = max(rr0 - h, 0), rhi = min(rr0 + h, p.rows - 1);
        const int clo = max(cc0 - h, 0), w = min(cc0 + h, p.cols - 1) - clo + 1;
        float I = 0.f, sy = 0.f, sx = 0.f, s2 = 0.f;
        int nk = 0;
        for (int r = rlo; r <= rhi; ++r) {
          const int64_t j0 = (int64_t)r * p.cols + clo;
          const uint32_t m = bit_run(bm, j0, w);
          // three columns at a time, their reads under way together
          for (int k0 = 0; k0 < w; k0 += 3) {
            float v[3], mb[3], sb[3];
            bool use[3];
#pragma unroll
            for (int u = 0; u < 3; ++u) {
              const int64_t j = j0 + k0 + u;
              const int32_t bj = ((m >> (k0 + u)) & 1u) ? __ldg(p.bop + j) : -1;
              use[u] = bj >= 0;   // (a caller's list may name masked pixels)
              v[u] = mb[u] = sb[u] = 0.0f;
              if (use[u]) {
                v[u] = value_of<DT, NORM>(p, frame, f, j);
                // background of the pixel's bin, or the profile at its centre
                mb[u] = INTERP ? profile_at(mu, bj, p.ia, p.it, j, nbins) : __ldg(mu + bj);
                sb[u] = INTERP ? profile_at(sd, bj, p.ia, p.it, j, nbins) : __ldg(sd + bj);
              }
            }
#pragma unroll
            for (int u = 0; u < 3; ++u) {
              if (!use[u]) continue;
              const float w1 = v[u] - mb[u];
              ++nk;
              I += w1;
              sy += w1 * ((float)r + 0.5f);
              sx += w1 * ((float)(clo + k0 + u) + 0.5f);
              s2 += sb[u] * sb[u];
            }
          }
        }
        sep_peak rec;
        rec.idx = (int32_t)i;
        rec.I = I;
        rec.y = sy / I;
        rec.x = sx / I;
        rec.sigma = sqrtf(s2);
        rec.npix = nk;
        peaks[g * pcap + before + r0 + t] = rec;
      }
      __syncthreads();
    }
    before += part;
  }
}

}  // namespace

cudaError_t launch_thresholds(const float* mean, const float* sigma, float k_pick, int64_t n, float* thr,
                              cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_thresholds<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(mean, sigma, k_pick, n, thr);
  return cudaGetLastError();
}

namespace {
template <int DT, bool NORM>
void launch_correct_t(const PixArgs& p, int32_t n_frames, int32_t fpc, dim3 grid, float* out, cudaStream_t s) {
  if constexpr (DT == SEP_DTYPE_F32) {
    if (p.npix % 4 == 0 && (uintptr_t)out % 16 == 0 && (uintptr_t)p.frames % 16 == 0) {
      k_correct<DT, NORM, true><<<grid, kImageThreads, 0, s>>>(p, n_frames, fpc, out);
      return;
    }
  }
  k_correct<DT, NORM, false><<<grid, kImageThreads, 0, s>>>(p, n_frames, fpc, out);
}
}  // namespace

cudaError_t launch_correct(const PixArgs& p, int32_t n_frames, float* out, cudaStream_t s) {
  if (n_frames <= 0 || p.npix <= 0) return cudaSuccess;
  const bool staged = p.stage != nullptr;   // (image order reads the staged copy only where it has to)
  const bool raw8 = !staged && p.dtype == SEP_DTYPE_U16_JF && p.npix % 8 == 0 && (uintptr_t)out % 16 == 0 &&
                    (uintptr_t)p.frames % 16 == 0;
  const int64_t per = raw8 ? 8 * kImageThreads : kPixPerCta;
  const int64_t ctas = (p.npix + per - 1) / per;
  const int32_t fpc = frames_per_thread(n_frames, ctas);
  dim3 grid((unsigned)ctas, (unsigned)((n_frames + fpc - 1) / fpc));
  if (staged) {
    k_correct<kStaged, false, false><<<grid, kImageThreads, 0, s>>>(p, n_frames, fpc, out);
  } else if (raw8) {
    if (p.norm) k_correct_raw8<true><<<grid, kImageThreads, 0, s>>>(p, n_frames, fpc, out);
    else k_correct_raw8<false><<<grid, kImageThreads, 0, s>>>(p, n_frames, fpc, out);
  } else if (p.dtype == SEP_DTYPE_U16_JF) {
    if (p.norm) launch_correct_t<SEP_DTYPE_U16_JF, true>(p, n_frames, fpc, grid, out, s);
    else launch_correct_t<SEP_DTYPE_U16_JF, false>(p, n_frames, fpc, grid, out, s);
  } else {
    if (p.norm) launch_correct_t<SEP_DTYPE_F32, true>(p, n_frames, fpc, grid, out, s);
    else launch_correct_t<SEP_DTYPE_F32, false>(p, n_frames, fpc, grid, out, s);
  }
  return cudaGetLastError();
}

namespace {
template <bool INTERP>
cudaError_t launch_mark_t(const PixArgs& p, int32_t n_frames, int32_t nbins, const float* thr, const float* mean,
                          const float* sigma, float k_pick, uint32_t* bitmap, int64_t words, cudaStream_t s) {
  if (n_frames <= 0) return cudaSuccess;
  const int64_t ctas = (words * 32 + kPixPerCta - 1) / kPixPerCta;
  const int32_t fpc = frames_per_thread(n_frames, ctas);
  dim3 grid((unsigned)ctas, (unsigned)((n_frames + fpc - 1) / fpc));
#define SEP_MARK_ARGS p, n_frames, fpc, nbins, thr, mean, sigma, k_pick, bitmap, words
  if (p.staged_only) {
    k_mark<kStaged, false, INTERP><<<grid, kImageThreads, 0, s>>>(SEP_MARK_ARGS);
  } else if (p.dtype == SEP_DTYPE_U16_JF) {
    if (p.norm) k_mark<SEP_DTYPE_U16_JF, true, INTERP><<<grid, kImageThreads, 0, s>>>(SEP_MARK_ARGS);
    else k_mark<SEP_DTYPE_U16_JF, false, INTERP><<<grid, kImageThreads, 0, s>>>(SEP_MARK_ARGS);
  } else {
    if (p.norm) k_mark<SEP_DTYPE_F32, true, INTERP><<<grid, kImageThreads, 0, s>>>(SEP_MARK_ARGS);
    else k_mark<SEP_DTYPE_F32, false, INTERP><<<grid, kImageThreads, 0, s>>>(SEP_MARK_ARGS);
  }
#undef SEP_MARK_ARGS
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_mark(const PixArgs& p, int32_t n_frames, int32_t nbins, const float* thr, uint32_t* bitmap,
                        int64_t words, cudaStream_t s) {
  return launch_mark_t<false>(p, n_frames, nbins, thr, nullptr, nullptr, 0.0f, bitmap, words, s);
}

cudaError_t launch_mark_interp(const PixArgs& p, int32_t n_frames, int32_t nbins, const float* mean,
                               const float* sigma, float k_pick, uint32_t* bitmap, int64_t words, cudaStream_t s) {
  return launch_mark_t<true>(p, n_frames, nbins, nullptr, mean, sigma, k_pick, bitmap, words, s);
}

// Type of the kernel instances that read listed pixels' values: those of raw
// frames read nothing but the staged copy where the call staged the batch.
static int32_t listed_source(const PixArgs& p) { return p.staged_only ? SEP_DTYPE_U16_JF : p.dtype; }

int32_t compact_tiles(int64_t words) { return (int32_t)((words + kTileWords - 1) / kTileWords); }
int32_t peak_chunks(int64_t kcap) { return (int32_t)((kcap + kPeakChunk - 1) / kPeakChunk); }

cudaError_t launch_compact(const PixArgs& p, int32_t n_frames, const uint32_t* bitmap, int64_t words, int32_t* idx,
                           float* val, int64_t cap, int32_t* n_kept, int32_t* scratch, int32_t* status,
                           cudaStream_t s) {
  if (n_frames <= 0) return cudaSuccess;
  const int32_t nt = compact_tiles(words);
  dim3 grid((unsigned)nt, (unsigned)n_frames);
  k_count_bits<<<grid, 256, 0, s>>>(bitmap, words, scratch, nt);
  const bool nrm = p.norm != nullptr;
#define SEP_EMIT_ARGS p, bitmap, words, scratch, nt, idx, val, cap, n_kept, status
#define SEP_EMIT(DT, NR)                                                             \
  if ((int64_t)nt * n_frames <= kWideCtas)                                           \
    k_emit_kept<DT, NR, kWideThreads><<<grid, kWideThreads, 0, s>>>(SEP_EMIT_ARGS);   \
  else                                                                                \
    k_emit_kept<DT, NR, kCompactThreads><<<grid, kCompactThreads, 0, s>>>(SEP_EMIT_ARGS)
  if (listed_source(p) == SEP_DTYPE_U16_JF) {
    if (nrm) { SEP_EMIT(SEP_DTYPE_U16_JF, true); } else { SEP_EMIT(SEP_DTYPE_U16_JF, false); }
  } else {
    if (nrm) { SEP_EMIT(SEP_DTYPE_F32, true); } else { SEP_EMIT(SEP_DTYPE_F32, false); }
  }
#undef SEP_EMIT
#undef SEP_EMIT_ARGS
  return cudaGetLastError();
}

cudaError_t launch_densify(const int32_t* bop, int64_t npix, int32_t nbins, int32_t n_frames, const float* mean,
                           const float* sigma, const int32_t* idx, const float* val, int64_t cap,
                           const int32_t* n_kept, const float* noise, float fill, const int32_t* interp_a,
                           const float* interp_t, float* out, cudaStream_t s) {
  if (n_frames <= 0 || npix <= 0) return cudaSuccess;
  const int64_t ctas = (npix + kPixPerCta - 1) / kPixPerCta;
  const int32_t fpc = frames_per_thread(n_frames, ctas);
  dim3 g1((unsigned)ctas, (unsigned)((n_frames + fpc - 1) / fpc));
  // the vector kernel by bin with deviates, and where the other one has few
  // frames to hold its tables over
  const bool vec = npix % 4 == 0 && (uintptr_t)out % 16 == 0 && (uintptr_t)noise % 16 == 0 &&
                   (interp_a ? fpc < kDenseSmoothFrames : noise || fpc < kDenseFrames);
#define SEP_DENSE_ARGS bop, npix, nbins, n_frames, fpc, mean, sigma, noise, fill, interp_a, interp_t, out
#define SEP_DENSE_VEC(NZ, IP) \
  k_dense_background_vec<NZ, IP><<<gv, 256, 0, s>>>(bop, npix, nbins, mean, sigma, noise, fill, interp_a, interp_t, out)
  if (vec) {
    dim3 gv((unsigned)((npix + 1023) / 1024), (unsigned)n_frames);
    if (noise && interp_a) SEP_DENSE_VEC(true, true);
    else if (noise) SEP_DENSE_VEC(true, false);
    else if (interp_a) SEP_DENSE_VEC(false, true);
    else SEP_DENSE_VEC(false, false);
  } else if (noise) {
    if (interp_a) k_dense_background<true, true><<<g1, kImageThreads, 0, s>>>(SEP_DENSE_ARGS);
    else k_dense_background<true, false><<<g1, kImageThreads, 0, s>>>(SEP_DENSE_ARGS);
  } else {
    if (interp_a) k_dense_background<false, true><<<g1, kImageThreads, 0, s>>>(SEP_DENSE_ARGS);
    else k_dense_background<false, false><<<g1, kImageThreads, 0, s>>>(SEP_DENSE_ARGS);
  }
#undef SEP_DENSE_VEC
#undef SEP_DENSE_ARGS
  if (cap > 0) {
    dim3 g2((unsigned)std::min<int64_t>((cap + 255) / 256, 64), (unsigned)n_frames);
    k_dense_scatter<<<g2, 256, 0, s>>>(idx, val, cap, n_kept, npix, out);
  }
  return cudaGetLastError();
}

cudaError_t launch_veto(int32_t n_frames, const int32_t* n_peaks, int32_t min_peaks, int32_t* list, int32_t* n_pass,
                        cudaStream_t s) {
  k_veto<<<1, 1024, 0, s>>>(n_frames, n_peaks, min_peaks, list, n_pass);
  return cudaGetLastError();
}

cudaError_t launch_compact_rows(int32_t n_frames, const int32_t* list, const int32_t* n_pass, int64_t row_bytes,
                                const void* src, void* dst, cudaStream_t s) {
  if (n_frames <= 0 || row_bytes <= 0) return cudaSuccess;
  const int64_t words = row_bytes / 4;
  const bool vec = words % 4 == 0 && (uintptr_t)src % 16 == 0 && (uintptr_t)dst % 16 == 0;
  const int64_t per = vec ? words / 4 : words;
  dim3 grid((unsigned)std::min<int64_t>(std::max<int64_t>((per + 255) / 256, 1), 64), (unsigned)n_frames);
  if (vec)
    k_compact_rows<true><<<grid, 256, 0, s>>>(list, n_pass, words, static_cast<const uint32_t*>(src),
                                               static_cast<uint32_t*>(dst));
  else
    k_compact_rows<false><<<grid, 256, 0, s>>>(list, n_pass, words, static_cast<const uint32_t*>(src),
                                                static_cast<uint32_t*>(dst));
  return cudaGetLastError();
}

cudaError_t launch_scatter_list(int32_t n_frames, const int32_t* idx, const int32_t* n_kept, int64_t kcap,
                                int64_t npix, uint32_t* bitmap, int64_t words, cudaStream_t s) {
  if (n_frames <= 0 || kcap <= 0) return cudaSuccess;
  dim3 grid((unsigned)((kcap + 255) / 256), (unsigned)n_frames);
  k_scatter_list<<<grid, 256, 0, s>>>(idx, n_kept, kcap, npix, bitmap, words);
  return cudaGetLastError();
}

cudaError_t launch_peaks(const PixArgs& p, int32_t n_frames, int32_t nbins, const float* mean, const float* sigma,
                         const uint32_t* bitmap, int64_t words, const int32_t* idx, const int32_t* n_kept, int64_t kcap,
                         int32_t patch, int32_t min_count, sep_peak* peaks, int64_t pcap, int32_t* n_peaks,
                         int32_t* scratch, int32_t* status, cudaStream_t s) {
  if (n_frames <= 0) return cudaSuccess;
  const int32_t nch = peak_chunks(kcap);
  uint32_t* flags = reinterpret_cast<uint32_t*>(scratch);
  int32_t* cnt = scratch + (int64_t)n_frames * nch * 8;
  // either grid: kPeakCtas CTAs over the frames where the lists can use them
  // (a chunk each in phase 1, a slice of at least 8 chunks each in phase 2,
  // where a frame gets 8 slices even if the frames alone fill the GPU: a
  // slice's records are a chain of gathers a thread)
  const int32_t want = std::max(1, (kPeakCtas + n_frames - 1) / n_frames);
  dim3 g1((unsigned)std::min(std::max(nch, 1), std::max(want, 64)), (unsigned)n_frames);
  dim3 g2((unsigned)std::min((nch + 7) / 8 + (nch == 0), std::max(want / 4, kPeakSlices)), (unsigned)n_frames);
  const bool nrm = p.norm != nullptr;
  const bool itp = p.ia != nullptr && p.it != nullptr;
#define SEP_FLAG_ARGS p, bitmap, words, idx, n_kept, kcap, patch, min_count, flags, cnt, nch
#define SEP_PEMIT_ARGS p, nbins, mean, sigma, bitmap, words, idx, n_kept, kcap, patch, flags, cnt, nch, peaks, pcap, n_peaks, status
#define SEP_PEMIT(DT, NR)                                                              \
  if (itp) k_peak_emit<DT, NR, true><<<g2, kPeakThreads, 0, s>>>(SEP_PEMIT_ARGS);      \
  else k_peak_emit<DT, NR, false><<<g2, kPeakThreads, 0, s>>>(SEP_PEMIT_ARGS)
  if (listed_source(p) == SEP_DTYPE_U16_JF) {
    if (nrm) {
      k_peak_flags<SEP_DTYPE_U16_JF, true><<<g1, kPeakThreads, 0, s>>>(SEP_FLAG_ARGS);
      SEP_PEMIT(SEP_DTYPE_U16_JF, true);
    } else {
      k_peak_flags<SEP_DTYPE_U16_JF, false><<<g1, kPeakThreads, 0, s>>>(SEP_FLAG_ARGS);
      SEP_PEMIT(SEP_DTYPE_U16_JF, false);
    }
  } else {
    if (nrm) {
      k_peak_flags<SEP_DTYPE_F32, true><<<g1, kPeakThreads, 0, s>>>(SEP_FLAG_ARGS);
      SEP_PEMIT(SEP_DTYPE_F32, true);
    } else {
      k_peak_flags<SEP_DTYPE_F32, false><<<g1, kPeakThreads, 0, s>>>(SEP_FLAG_ARGS);
      SEP_PEMIT(SEP_DTYPE_F32, false);
    }
  }
#undef SEP_PEMIT
#undef SEP_FLAG_ARGS
#undef SEP_PEMIT_ARGS
  return cudaGetLastError();
}

// scratch words needed by launch_compact and launch_peaks for F frames
int64_t consumer_scratch_words(int32_t n_frames, int64_t words, int64_t kcap) {
  const int64_t a = (int64_t)n_frames * compact_tiles(words);
  const int64_t b = (int64_t)n_frames * peak_chunks(kcap) * 9;
  return a > b ? a : b;
}

}  // namespace sep
