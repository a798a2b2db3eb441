// Staging of a batch: every pixel of the image is corrected once per frame
// (Section 1.2, divided by its norm, Eq. 1) and its value is written to the
// slots of its matrix entries in the frame's staged row (slot e holds entry
// e's value, padding slots NaN), so the clip kernel reads each bin's values
// as one contiguous run.
//
// One CTA per image tile (kTileH x kTileW pixels) and group of frames, four
// frames a step: each thread corrects four consecutive pixels of a tile row
// in the four frames and stores a pixel's four values side by side in shared
// memory; then the tile's list of (slot, pixel) pairs, ascending by slot,
// writes them out (the entries of one bin inside a tile occupy consecutive
// slots), one 16-byte read and four stores a slot. The tile is double
// buffered, so a step costs one barrier and the warps of a CTA correct the
// next frames while others still write the last. The raw words of later
// frames arrive meanwhile in a ring in shared memory (cp.async into the
// thread's own slots: no registers held, no barrier). A call of a few frames
// takes two of them a CTA instead (k_stage_few).
//
// Each value is the same IEEE sequence as pixel_value(): RN32(RN32(adc -
// pedestal) / gain), then RN32(. / norm); level 0 without a division (Level0).
//
// What bounds it: the staged values written (27 MB a Jungfrau-4M frame, all
// of whole sectors) and the words read. With one value a shared-memory access
// and range tests a pixel and frame, the kernel was bound by its instructions
// and shared-memory wavefronts: 48 raw Jungfrau-4M frames 475 -> 411 us (4.6
// TB/s); the write-out is half of it. Float frames that had no ring (a width
// that is not a multiple of 4, or a list of frames): 29 frames of 1031 x 1065
// 80 -> 75 us; 24 frames of 619 x 487, whose 80 CTAs left half of the GPU
// idle: 60 -> 26 us.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sep_device.cuh"
#include "sep_internal.h"

namespace sep {
namespace {

constexpr int kTilePix = kTileH * kTileW;
constexpr int kStageThreads = kTilePix / 4;   // 4 consecutive pixels of one row a thread
constexpr int kRowThreads = kTileW / 4;       // threads covering one tile row
constexpr int kStep = 4;                      // frames a step
static_assert(kTileW % 4 == 0 && kStageThreads % 32 == 0 && kStageThreads <= 1024, "tile shape");

// How a thread's four words of a frame reach the ring: one copy (columns a
// multiple of 4, aligned frames), copies of 4 bytes (aligned to those), or
// not at all (plain loads: raw frames of an odd width or address).
enum { LOAD_VECTOR = 2, LOAD_WORD = 1, LOAD_PLAIN = 0 };

// Frames the ring holds (what shared memory allows beside the two tiles).
template <int DT>
__host__ __device__ constexpr int ring_frames() {
  return DT == SEP_DTYPE_U16_JF ? 8 : 4;
}
template <int DT, int LOAD>
constexpr size_t stage_smem_bytes() {
  return sizeof(float4) * 2 * (kTilePix + 1) +
         (LOAD == LOAD_PLAIN ? 0 : (size_t)ring_frames<DT>() * kStageThreads * (DT == SEP_DTYPE_U16_JF ? 8 : 16));
}

// The tile's pairs a thread writes: pairs tid + kStageThreads k for
// k < kScReg stay in registers for every frame, longer lists read the rest at
// each step (with 7 instead of 8 a 512-frame Jungfrau-4M batch takes 13.3
// instead of 12.4 ms: its tiles near the beam hold up to 8,000 pairs). loc:
// the pixel's place in the tile, four consecutive pixels kStageThreads apart
// (the threads of a warp then store side by side); kTilePix, a NaN, for
// padding.
constexpr int kScReg = 8;
__device__ __forceinline__ int tile_place(int pix) {
  return pix < 0 ? kTilePix : (pix & 3) * kStageThreads + (pix >> 2);
}

// pixel_value() of a pixel's words of a step's frames: the calibration of each
// gain level that occurs is read once for all of them, its reads together.
// (Bright frames have such pixels in every warp. With pixel_value() for the
// thread's four pixels in the four frames, one after another, 64 raw
// Jungfrau-4M frames took 1357 us with one pixel in 10,000 at another level,
// 1537 with one in 1000, 1773 with one in 100 and 1852 with all; now 1125,
// 1159, 1230 and 1457, and 1074 without any.)
template <bool NORM>
__device__ __forceinline__ void level_values(const StageArgs& a, int64_t i, const uint32_t (&u)[kStep],
                                             float (&y)[kStep]) {
  float ped[3], gain[3];
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    bool occurs = false;
#pragma unroll
    for (int h = 0; h < kStep; ++h) occurs = occurs || min(u[h] >> 14, 2u) == (uint32_t)l;
    ped[l] = occurs ? __ldg(a.ped + l * a.npix + i) : 0.0f;
    gain[l] = occurs ? __ldg(a.gain + l * a.npix + i) : 1.0f;
  }
  const float norm = NORM ? __ldg(a.norm + i) : 1.0f;
#pragma unroll
  for (int h = 0; h < kStep; ++h) {
    const uint32_t l = u[h] >> 14;
    const float pd = l == 0 ? ped[0] : (l == 1 ? ped[1] : ped[2]);
    const float gn = l == 0 ? gain[0] : (l == 1 ? gain[1] : gain[2]);
    y[h] = __fdiv_rn(__fsub_rn((float)(u[h] & 0x3fffu), pd), gn);
    if (NORM) y[h] = __fdiv_rn(y[h], norm);
  }
}

template <int DT, bool NORM, int LOAD>
__global__ void __launch_bounds__(kStageThreads) k_stage(StageArgs a) {
  constexpr int kWord = DT == SEP_DTYPE_U16_JF ? 2 : 4;
  constexpr int kRing = ring_frames<DT>();
  extern __shared__ __align__(16) unsigned char stage_smem[];
  float4* tv = reinterpret_cast<float4*>(stage_smem);   // [2][kTilePix + 1]: a pixel's values of the step's frames
  unsigned char* ring = stage_smem + sizeof(float4) * 2 * (kTilePix + 1);
  const int t = blockIdx.x;
  const int tid = threadIdx.x;
  const int eb = __ldg(a.tile_ebase + t), ne = __ldg(a.tile_ebase + t + 1) - eb;
  if (ne == 0) return;
  if (tid < 2) {
    const float nan = __int_as_float(0x7fc00000);
    tv[tid * (kTilePix + 1) + kTilePix] = make_float4(nan, nan, nan, nan);
  }
  uint32_t slot[kScReg];   // the pairs' slots and places
  int loc[kScReg];
#pragma unroll
  for (int k = 0; k < kScReg; ++k) {
    int2 sc = make_int2(0, -1);
    if (tid + kStageThreads * k < ne) sc = __ldg(a.tile_sc + eb + tid + kStageThreads * k);
    slot[k] = (uint32_t)sc.x;
    loc[k] = tile_place(sc.y);
  }
  const int64_t r = (int64_t)(t / a.tiles_x) * kTileH + tid / kRowThreads;
  const int64_t c = (int64_t)(t % a.tiles_x) * kTileW + 4 * (tid % kRowThreads);
  const int64_t p = r * a.cols + c;    // first of this thread's 4 pixels
  const int n_in = r < a.rows ? (int)max((int64_t)0, min((int64_t)4, a.cols - c)) : 0;   // of them inside the image
  Level0 cal[4];
  float nm[4];
  // bit k: pixel p + k has a bin; its level-0 words need a division. (Pixels
  // under the mask count for neither: real calibrations hold gain 0 or NaN
  // there, and words of any level.)
  const uint32_t used = DT == SEP_DTYPE_U16_JF ? __ldg(a.used + (int64_t)t * kStageThreads + tid) : 0u;
  uint32_t odd = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    nm[k] = 1.0f;
    if (k < n_in) {
      if (DT == SEP_DTYPE_U16_JF) {
        cal[k].set(__ldg(a.ped + p + k), __ldg(a.gain + p + k));
        if (cal[k].limit == 0) odd |= 1u << k;
      }
      if (NORM) nm[k] = __ldg(a.norm + p + k);
    }
  }
  odd &= used;
  const int f0 = blockIdx.y * a.frames_per_cta;
  const int nfr = min(f0 + a.frames_per_cta, a.n_frames) - f0;
  const int64_t pitch = a.npix * kWord;   // bytes from a frame to the next
  const unsigned char* first = reinterpret_cast<const unsigned char*>(frame_ptr<DT>(a.frames, f0, a.npix)) + p * kWord;
  auto frame_of = [&](int j) {   // this thread's first word of frame f0 + j
    return a.fptr ? reinterpret_cast<const unsigned char*>((uintptr_t)a.fptr[f0 + j]) + p * kWord : first + j * pitch;
  };
  const unsigned ring0 = (unsigned)__cvta_generic_to_shared(ring) + tid * 4 * kWord;
  // copy of a frame's words from src to ring slot q
  auto copy = [&](int q, const unsigned char* src) {
    const unsigned dst = ring0 + (unsigned)(q * kStageThreads * 4 * kWord);
    if (LOAD == LOAD_VECTOR) {
      if (kWord == 2) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
      else asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
    } else {
      // (raw: the width is even, so a pair of pixels is inside or outside)
#pragma unroll
      for (int k = 0; k < 4; k += 4 / kWord)
        if (k < n_in)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst + k * kWord), "l"(src + k * kWord)
                       : "memory");
    }
  };
  // the step's frames from j0 on into the ring slots from q0 on (one commit
  // group a step, empty past the last frame)
  auto issue = [&](int j0, int q0) {
    if (n_in > 0) {
#pragma unroll
      for (int h = 0; h < kStep; ++h)
        if (j0 + h < nfr) copy(q0 + h, frame_of(j0 + h));
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  if (LOAD != LOAD_PLAIN) {
#pragma unroll
    for (int j = 0; j < kRing; j += kStep) issue(j, j);
  }
  int buf = 0;
  for (int j = 0; j < nfr; j += kStep, buf ^= 1) {
    const int nf = min(kStep, nfr - j);
    const int q0 = j % kRing;   // ring slots of the step's frames
    float4* tile = tv + buf * (kTilePix + 1);
    float x[kStep][4];
    uint32_t all01 = 0, all23 = 0;   // the bits of the step's words of pixels 0, 1 and 2, 3
    if (DT == SEP_DTYPE_U16_JF) {
      uint2 v[kStep];   // a frame's four words
      if (LOAD != LOAD_PLAIN) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kRing / kStep - 1) : "memory");
#pragma unroll
        for (int h = 0; h < kStep; ++h)
          v[h] = *reinterpret_cast<const uint2*>(ring + ((q0 + h) * kStageThreads + tid) * 8);
      } else {
#pragma unroll
        for (int h = 0; h < kStep; ++h) {
          const uint16_t* src = reinterpret_cast<const uint16_t*>(h < nf ? frame_of(j + h) : nullptr);
          uint32_t w[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) w[k] = h < nf && k < n_in ? (uint32_t)__ldg(src + k) : 0u;
          v[h] = make_uint2(w[0] | w[1] << 16, w[2] | w[3] << 16);
        }
      }
#pragma unroll
      for (int h = 0; h < kStep; ++h) {
        if (h < nf) {   // (past the last frame the ring holds older words)
          all01 |= v[h].x;
          all23 |= v[h].y;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          // the word's value as a float without a conversion: its 16 bits
          // below the exponent of 2^23, less 2^23 (exact)
          const uint32_t bits = __byte_perm(k < 2 ? v[h].x : v[h].y, 0x4b000000u, k & 1 ? 0x7432 : 0x7410);
          x[h][k] = cal[k].value_of(__fsub_rn(__uint_as_float(bits), 8388608.0f));
          if (NORM) x[h][k] = __fdiv_rn(x[h][k], nm[k]);
        }
      }
    } else {
      if (LOAD != LOAD_PLAIN) asm volatile("cp.async.wait_group %0;\n" ::"n"(kRing / kStep - 1) : "memory");
#pragma unroll
      for (int h = 0; h < kStep; ++h) {
        const float4 v = *reinterpret_cast<const float4*>(ring + ((q0 + h) * kStageThreads + tid) * 16);
        x[h][0] = v.x; x[h][1] = v.y; x[h][2] = v.z; x[h][3] = v.w;
        if (NORM) {
#pragma unroll
          for (int k = 0; k < 4; ++k) x[h][k] = __fdiv_rn(x[h][k], nm[k]);
        }
      }
    }
    if (DT != SEP_DTYPE_U16_JF) issue(j + kRing, q0);   // the slots just read are refilled (in registers now)
#pragma unroll
    for (int k = 0; k < 4; ++k)
      tile[k * kStageThreads + tid] = make_float4(x[0][k], x[1][k], x[2][k], x[3][k]);
    if (DT == SEP_DTYPE_U16_JF && (((all01 | all23) & 0xc000c000u) || odd)) {
      // pixels with a word of another gain level or an unusual calibration
      // (rare: one copy of the code)
      uint32_t todo = odd;
      if (all01 & 0x0000c000u) todo |= 1u;
      if (all01 & 0xc0000000u) todo |= 2u;
      if (all23 & 0x0000c000u) todo |= 4u;
      if (all23 & 0xc0000000u) todo |= 8u;
#pragma unroll 1
      for (todo &= used; todo; todo &= todo - 1) {
        const int k = __ffs(todo) - 1;
        uint32_t u[kStep];
#pragma unroll
        for (int h = 0; h < kStep; ++h) {
          u[h] = 0;
          if (h < nf)
            u[h] = LOAD != LOAD_PLAIN
                       ? *reinterpret_cast<const uint16_t*>(ring + ((q0 + h) * kStageThreads + tid) * 8 + 2 * k)
                       : __ldg(reinterpret_cast<const uint16_t*>(frame_of(j + h)) + k);
        }
        float y[kStep];
        level_values<NORM>(a, p + k, u, y);
        tile[k * kStageThreads + tid] = make_float4(y[0], y[1], y[2], y[3]);
      }
    }
    if (DT == SEP_DTYPE_U16_JF && LOAD != LOAD_PLAIN) issue(j + kRing, q0);   // refilled (this thread's own words)
    __syncthreads();
    // the step's frames, slot by slot
    float* out = a.stage + (int64_t)(f0 + j) * a.npos;
    if (nf == kStep) {
      float *o1 = out + a.npos, *o2 = o1 + a.npos, *o3 = o2 + a.npos;
      auto put = [&](uint32_t q, const float4& v) {
        out[q] = v.x;
        o1[q] = v.y;
        o2[q] = v.z;
        o3[q] = v.w;
      };
#pragma unroll
      for (int k = 0; k < kScReg; ++k)
        if (tid + kStageThreads * k < ne) put(slot[k], tile[loc[k]]);
      for (int q = tid + kStageThreads * kScReg; q < ne; q += kStageThreads) {
        const int2 sc = __ldg(a.tile_sc + eb + q);
        put((uint32_t)sc.x, tile[tile_place(sc.y)]);
      }
    } else {
      // the last step of a group, from the same registers (with the list read
      // again for every pair, two raw Jungfrau-4M frames staged and clipped
      // without steps took 106 us, three 142; now 86 and 101)
      auto put = [&](uint32_t q, const float4& v) {
        float* o = out + q;
        *o = v.x;
        if (nf > 1) o[a.npos] = v.y;
        if (nf > 2) o[2 * a.npos] = v.z;
      };
#pragma unroll
      for (int k = 0; k < kScReg; ++k)
        if (tid + kStageThreads * k < ne) put(slot[k], tile[loc[k]]);
#pragma unroll 1
      for (int q = tid + kStageThreads * kScReg; q < ne; q += kStageThreads) {
        const int2 sc = __ldg(a.tile_sc + eb + q);
        put((uint32_t)sc.x, tile[tile_place(sc.y)]);
      }
      return;   // (said here: it frees the registers of the loop over the full steps, which spilled otherwise)
    }
  }
}

// The same for few frames: two a CTA, by pixel of the tile. There is no step
// of four frames to fill, nothing to prefetch and no list to hold for later
// frames, so the CTA is small (512 threads, 33 KB) and three of them hide one
// another's waits on a multiprocessor, where k_stage keeps one. Bound by that
// chain of waits (list, words, calibration, write-out). Staging and clip of
// one raw Jungfrau-4M frame: 71 us (82 by k_stage), two 79 (95); one 1M float
// frame 27 (31), six 42 (49).
constexpr int kFewThreads = 512;
constexpr int kFewFrames = 8;
constexpr int64_t kFewCtas = 152 * 8;

template <int DT, bool NORM>
__global__ void __launch_bounds__(kFewThreads, 3) k_stage_few(StageArgs a) {
  __shared__ float tv[2][kTilePix + 1];   // two frames' values, and a NaN (padding)
  const int t = blockIdx.x;
  const int tid = threadIdx.x;
  const int eb = __ldg(a.tile_ebase + t), ne = __ldg(a.tile_ebase + t + 1) - eb;
  if (ne == 0) return;
  if (tid < 2) tv[tid][kTilePix] = __int_as_float(0x7fc00000);
  const int r0 = t / a.tiles_x * kTileH, c0 = t % a.tiles_x * kTileW;
  const int f = 2 * blockIdx.y;
  const bool two = f + 1 < a.n_frames;   // (else the frame's words are read twice)
  const void* fr[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int g = two ? f + h : f;
    fr[h] = a.fptr ? (const void*)a.fptr[g] : frame_ptr<DT>(a.frames, g, a.npix);
  }
  // (a warp reads 32 pixels side by side, at any alignment)
#pragma unroll 4
  for (int k = 0; k < kTilePix / kFewThreads; ++k) {
    const int pix = tid + kFewThreads * k, r = r0 + pix / kTileW, c = c0 + pix % kTileW;
    if (r >= a.rows || c >= a.cols) continue;
    const int64_t p = (int64_t)r * a.cols + c;
    float x[2];
    if (DT == SEP_DTYPE_U16_JF) {
      uint32_t u[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) u[h] = __ldg(reinterpret_cast<const uint16_t*>(fr[h]) + p);
      const float ped = __ldg(a.ped + p), gain = __ldg(a.gain + p);   // level 0, read beside the words
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (u[h] < 0x4000u) {
          x[h] = __fdiv_rn(__fsub_rn((float)u[h], ped), gain);
          if (NORM) x[h] = __fdiv_rn(x[h], __ldg(a.norm + p));
        } else {
          x[h] = pixel_value<DT, NORM>(fr[h], p, a.npix, a.ped, a.gain, a.norm);
        }
      }
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h) x[h] = pixel_value<DT, NORM>(fr[h], p, a.npix, a.ped, a.gain, a.norm);
    }
    tv[0][pix] = x[0];
    if (two) tv[1][pix] = x[1];
  }
  __syncthreads();
  float *o0 = a.stage + (int64_t)f * a.npos, *o1 = o0 + a.npos;
  for (int q = tid; q < ne; q += kFewThreads) {
    const int2 sc = __ldg(a.tile_sc + eb + q);
    const int at = sc.y < 0 ? kTilePix : sc.y;
    o0[(uint32_t)sc.x] = tv[0][at];
    if (two) o1[(uint32_t)sc.x] = tv[1][at];
  }
}

template <int DT, bool NORM, int LOAD>
cudaError_t launch_l(const StageArgs& a, dim3 grid, cudaStream_t s) {
  constexpr size_t smem = stage_smem_bytes<DT, LOAD>();
  // opt in once per device (the attribute only needs to be set before the
  // first launch; later calls find it set)
  static bool set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!set[dev]) {
    cudaError_t e =
        cudaFuncSetAttribute(k_stage<DT, NORM, LOAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    set[dev] = true;
  }
  k_stage<DT, NORM, LOAD><<<grid, kStageThreads, smem, s>>>(a);
  return cudaGetLastError();
}

template <int DT, bool NORM>
cudaError_t launch_v(const StageArgs& a, dim3 grid, cudaStream_t s) {
  // Few frames: as long as three CTAs a multiprocessor take them in less than
  // three waves (eight 1M float frames 55 us, k_stage 58; four raw Jungfrau-4M
  // frames 141 and 131, eight of 1031 x 1065 99 and 97).
  const dim3 few(grid.x, (unsigned)((a.n_frames + 1) / 2));
  if (a.n_frames <= kFewFrames && (int64_t)few.x * few.y <= kFewCtas) {
    k_stage_few<DT, NORM><<<few, kFewThreads, 0, s>>>(a);
    return cudaGetLastError();
  }
  // One copy of a thread's four words: every frame at an address aligned to
  // them and the rows' pixels in groups of 4. Copies of 4 bytes: float frames
  // (their words), raw frames of an even width at 4-byte addresses.
  if (a.align % (DT == SEP_DTYPE_U16_JF ? 8 : 16) == 0 && a.cols % 4 == 0) return launch_l<DT, NORM, LOAD_VECTOR>(a, grid, s);
  if (DT == SEP_DTYPE_F32 || (a.align % 4 == 0 && a.cols % 2 == 0)) return launch_l<DT, NORM, LOAD_WORD>(a, grid, s);
  return launch_l<DT, NORM, DT == SEP_DTYPE_F32 ? LOAD_WORD : LOAD_PLAIN>(a, grid, s);
}

}  // namespace

cudaError_t launch_stage(const StageArgs& args, int32_t dtype, bool has_norm, cudaStream_t s) {
  if (args.n_frames <= 0) return cudaSuccess;
  StageArgs a = args;
  const int n_tiles = a.tiles_x * a.tiles_y;
  // Frames a CTA: 32, which read the tile's calibration and list once for
  // all, fewer (whole steps) where the grid would hold less than four CTAs a
  // multiprocessor; up to 16 frames all in one where the tiles alone fill the
  // GPU (ten 1M float frames 76 us, in groups of four 80; sixteen 106 and 112).
  const int64_t share = (int64_t)n_tiles * a.n_frames / (152 * 4) / kStep * kStep;
  a.frames_per_cta = n_tiles >= 152 && a.n_frames <= 16 ? 16 : (int)std::min<int64_t>(std::max<int64_t>(share, kStep), 32);
  dim3 grid(n_tiles, (a.n_frames + a.frames_per_cta - 1) / a.frames_per_cta);
  if (dtype == SEP_DTYPE_U16_JF)
    return has_norm ? launch_v<SEP_DTYPE_U16_JF, true>(a, grid, s) : launch_v<SEP_DTYPE_U16_JF, false>(a, grid, s);
  return has_norm ? launch_v<SEP_DTYPE_F32, true>(a, grid, s) : launch_v<SEP_DTYPE_F32, false>(a, grid, s);
}

}  // namespace sep
