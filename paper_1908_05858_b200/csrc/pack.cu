// Binarize + bit-pack kernels (Section 2.1.1 of the paper): fp32 (or int32) -> one bit per element, 64 channels
// per word, words of a pixel contiguous (channel-packed NHWC).  Pure HBM streaming: 4 bytes read and
// 1/8 byte written per element.
//
// The paper gathers IEEE sign bits with NEON shift-and-insert instructions spread over several
// registers.  Here the sign test is a compare (so -0.0 and NaN pack as +1), 128-bit loads keep the
// memory system busy, bits are gathered in registers by shift-or, and the words leave through shared
// memory so that global stores are whole, contiguous 16-byte pieces.  The int32 form (the paper packs the sign bit
// of 32-bit integers the same way, e.g. a convolution's raw sums) runs the same kernels with an integer compare.
#include "common.cuh"

namespace dabnn {

namespace {

constexpr int kPackThreads = 128;

// Streaming 16-byte load.  Written as volatile asm so that a batch of them is issued back to back, in program
// order, before the first result is consumed (memory-level parallelism is what an HBM-bound kernel lives on).
__device__ __forceinline__ float4 ld_stream_v4(const float4* p) {
  float4 v;
  asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ int4 ld_stream_v4(const int4* p) {
  int4 v;
  asm volatile("ld.global.cs.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
template <typename T> struct Vec4;
template <> struct Vec4<float> { using type = float4; };
template <> struct Vec4<int32_t> { using type = int4; };
// the bit: 1 where the value is negative (a compare: -0.0 and NaN give 0, i.e. +1)
__device__ __forceinline__ unsigned neg(float v) { return (unsigned)(v < 0.0f); }
__device__ __forceinline__ unsigned neg(int32_t v) { return (unsigned)(v < 0); }

// NCHW, H*W a multiple of 4, 16-byte aligned input.  A CTA covers 128 consecutive pixels of the batch (images follow one
// another in the pixel count: a tile may span two or more images, so small images leave no ragged tile per image) and all
// channels.  Each lane owns 4 consecutive pixels of one image (one float4 per channel); the four warps split every word's
// 64 channels into quarters of 16, so a thread has 16 independent 16-byte loads per word, of which as many are in flight as its
// registers hold, and the 16-bit quarters are placed side by side in shared memory, which assembles the 64-bit words without any
// exchange.
// C2: the words leave in the NC1HWC2 layout instead ([N][C1][H][W][2]: 128-bit vectors of one channel group, pixel after
// pixel; an odd last word gets a zero partner).
// SPLIT: gridDim.y CTAs share the words of 128 pixels, for tensors of few pixels and many channels, whose words one CTA packs one after
// another, a load latency each.  512 channels at 14x14, packs in a row on inputs in turn (HBM floor in brackets): batch 256 26.3 -> 17.8
// us (15.7), 64 22.5 -> 6.0 (3.9), 16 10.8 -> 2.7 (1.0; inputs that L2 holds).  (PER_SM: twelve CTAs with 40 registers; with 42 the large tensors take 5
// us of 68 more.  Split launches that ten per SM hold are 5 to 10 % faster without that limit.)
template <typename T, bool C2, bool SPLIT, int PER_SM = 12>
__global__ void __launch_bounds__(kPackThreads, PER_SM) pack_nchw_vec4(const int room, const T* __restrict__ x, int C, int HW, int Cw, long long npix,
                                                               uint64_t* __restrict__ packed) {
  if (room == 2) chain_trigger();
  x = chain_wait_for(x);
  extern __shared__ __align__(16) uint64_t s_words[];  // [128][CwL]
  const int CwL = SPLIT ? Cw / gridDim.y : Cw, cw0 = SPLIT ? blockIdx.y * CwL : 0;  // this CTA's words of each pixel
  uint16_t* s_q = reinterpret_cast<uint16_t*>(s_words);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long pix0 = (long long)blockIdx.x * 128;  // in pixels of the whole batch
  const long long p = pix0 + lane * 4;                 // first of this lane's 4 pixels
  const bool live = p < npix;                          // HW % 4 == 0, so all 4 pixels are live together and in one image
  using V4 = typename Vec4<T>::type;
  const long long n = live ? p / HW : 0;
  const int hw = live ? (int)(p - n * HW) : 0;
  const T* xn = x + (size_t)n * C * HW + hw;
  const size_t cstride = (size_t)HW / 4;
  for (int cw = 0; cw < CwL; cw++) {
    const int c0 = (cw0 + cw) * 64 + warp * 16;
    unsigned b0 = 0, b1 = 0, b2 = 0, b3 = 0;  // 16 channels of each of the 4 pixels
    if (live && c0 < C) {
      const V4* src = reinterpret_cast<const V4*>(xn + (size_t)c0 * HW);
      if (c0 + 16 <= C) {
        V4 v[16];
#pragma unroll
        for (int u = 0; u < 16; u++) v[u] = ld_stream_v4(src + (size_t)u * cstride);
#pragma unroll
        for (int u = 0; u < 16; u++) {
          b0 |= neg(v[u].x) << u;
          b1 |= neg(v[u].y) << u;
          b2 |= neg(v[u].z) << u;
          b3 |= neg(v[u].w) << u;
        }
      } else {
        for (int u = 0; u < C - c0; u++) {
          const V4 v = __ldcs(src + (size_t)u * cstride);
          b0 |= neg(v.x) << u;
          b1 |= neg(v.y) << u;
          b2 |= neg(v.z) << u;
          b3 |= neg(v.w) << u;
        }
      }
    }
    const int lp = lane * 4;
    s_q[((lp + 0) * CwL + cw) * 4 + warp] = (uint16_t)b0;
    s_q[((lp + 1) * CwL + cw) * 4 + warp] = (uint16_t)b1;
    s_q[((lp + 2) * CwL + cw) * 4 + warp] = (uint16_t)b2;
    s_q[((lp + 3) * CwL + cw) * 4 + warp] = (uint16_t)b3;
  }
  if (room == 1) chain_trigger();
  __syncthreads();
  const int npx = (int)min((long long)128, npix - pix0);
  if (npx <= 0) return;
  if (C2) {
    const int C1 = (Cw + 1) / 2;
    ulonglong2* d2 = reinterpret_cast<ulonglong2*>(packed);  // 16-byte aligned: checked on the host
    for (int i = threadIdx.x; i < C1 * npx; i += kPackThreads) {
      const int grp = i / npx, px = i - grp * npx;  // consecutive threads: consecutive pixels of one channel group
      const long long pp = pix0 + px, nn = pp / HW, hh = pp - nn * HW;
      const uint64_t lo = s_words[px * Cw + 2 * grp], hi = (2 * grp + 1 < Cw) ? s_words[px * Cw + 2 * grp + 1] : 0ull;
      d2[((size_t)nn * C1 + grp) * HW + hh] = make_ulonglong2(lo, hi);
    }
    return;
  }
  if (SPLIT) {  // pieces of CwL words, 16 bytes at a time where they come in pairs and start on 16
    if (CwL % 2 == 0 && Cw % 2 == 0 && (reinterpret_cast<uintptr_t>(packed) & 15) == 0) {
      const int pairs = CwL / 2;
      for (int i = threadIdx.x; i < npx * pairs; i += kPackThreads) {
        const int px = i / pairs, q = i - px * pairs;
        *reinterpret_cast<ulonglong2*>(packed + (size_t)(pix0 + px) * Cw + cw0 + 2 * q) = *reinterpret_cast<const ulonglong2*>(s_words + px * CwL + 2 * q);
      }
    } else {
      for (int i = threadIdx.x; i < npx * CwL; i += kPackThreads) {
        const int px = i / CwL, q = i - px * CwL;
        packed[(size_t)(pix0 + px) * Cw + cw0 + q] = s_words[px * CwL + q];
      }
    }
    return;
  }
  // contiguous in global memory: pixels pix0 .. pix0+npx-1 of the batch, all words
  uint64_t* dst = packed + (size_t)pix0 * Cw;
  const int total = npx * Cw;
  if (((size_t)pix0 * Cw) % 2 == 0 && (reinterpret_cast<uintptr_t>(packed) & 15) == 0) {
    const int pairs = total / 2;
    const ulonglong2* s2 = reinterpret_cast<const ulonglong2*>(s_words);
    ulonglong2* d2 = reinterpret_cast<ulonglong2*>(dst);
    for (int i = threadIdx.x; i < pairs; i += kPackThreads) d2[i] = s2[i];
    if ((total & 1) && threadIdx.x == 0) dst[total - 1] = s_words[total - 1];
  } else {
    for (int i = threadIdx.x; i < total; i += kPackThreads) dst[i] = s_words[i];
  }
}

// NCHW, any H*W and alignment: a CTA takes 128 consecutive pixels of one image and one 64-channel word.  The
// 64 x 128 sign flags are gathered with coalesced scalar loads (lanes along pixels) into shared memory; each
// thread then assembles 32 channel bits of one pixel and stores that half word.
template <typename T>
__global__ void __launch_bounds__(256) pack_nchw_tile(const int room, const T* __restrict__ x, int C, int HW, int Cw,
                                                      uint64_t* __restrict__ packed) {
  if (room == 2) chain_trigger();
  x = chain_wait_for(x);
  __shared__ unsigned char s_sign[64 * 128];
  const int tid = threadIdx.x, lane = tid & 31, ty = tid >> 5;
  const int n = blockIdx.y, p0 = blockIdx.x * 128, cw = blockIdx.z;
  const int npix = min(128, HW - p0);
  const T* xn = x + (size_t)n * C * HW + p0;
  const int c0 = cw * 64, cn = min(64, C - c0);
#pragma unroll
  for (int c = ty; c < 64; c += 8) {
    const T* row = xn + (size_t)(c0 + c) * HW;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int p = lane + 32 * q;
      s_sign[c * 128 + p] = (c < cn && p < npix) ? (unsigned char)neg(__ldcs(row + p)) : (unsigned char)0;
    }
  }
  if (room == 1) chain_trigger();
  __syncthreads();
  const int p = tid & 127, half = tid >> 7;
  if (p < npix) {
    uint32_t bits = 0;
#pragma unroll
    for (int c = 0; c < 32; c++) bits |= (uint32_t)s_sign[(half * 32 + c) * 128 + p] << c;
    reinterpret_cast<uint32_t*>(packed)[(((size_t)n * HW + p0 + p) * Cw + cw) * 2 + half] = bits;
  }
}

// NCHW, small images whose H*W is no multiple of 4 (7 x 7): the 64 channels of a word are one contiguous run of 64 * H*W
// values of an image, which starts on 16 bytes when C * H*W is a multiple of 4.  A CTA takes one (image, word): 128-bit loads
// along the run (a vector may straddle two channels), one sign byte per value into shared memory at the same flat index, then
// each thread gathers 32 channels of one pixel (consecutive lanes: consecutive bytes).  The 128-pixel tiles of the kernel above
// would leave 79 of 128 lanes idle at 7 x 7.
template <typename T>
__global__ void __launch_bounds__(256) pack_nchw_small(const int room, const T* __restrict__ x, int C, int HW, int Cw, uint64_t* __restrict__ packed) {
  if (room == 2) chain_trigger();
  x = chain_wait_for(x);
  extern __shared__ __align__(16) unsigned char s_flag[];  // [64 * HW]
  using V4 = typename Vec4<T>::type;
  const int tid = threadIdx.x, cw = blockIdx.x;
  const long long n = blockIdx.y;
  const int cn = min(64, C - cw * 64), count = cn * HW;
  const T* src = x + (n * C + (long long)cw * 64) * HW;
  for (int i0 = 0; i0 < count / 4; i0 += 4 * 256) {
    V4 v[4];
#pragma unroll
    for (int u = 0; u < 4; u++)
      if (i0 + u * 256 + tid < count / 4) v[u] = ld_stream_v4(reinterpret_cast<const V4*>(src) + i0 + u * 256 + tid);
#pragma unroll
    for (int u = 0; u < 4; u++)
      if (i0 + u * 256 + tid < count / 4)
        reinterpret_cast<uint32_t*>(s_flag)[i0 + u * 256 + tid] = neg(v[u].x) | (neg(v[u].y) << 8) | (neg(v[u].z) << 16) | (neg(v[u].w) << 24);
  }
  if (tid < (count & 3)) s_flag[(count & ~3) + tid] = (unsigned char)neg(src[(count & ~3) + tid]);
  if (room == 1) chain_trigger();
  __syncthreads();
  for (int i = tid; i < 2 * HW; i += 256) {
    const int half = i >= HW ? 1 : 0, p = i - half * HW;
    const int live = cn - 32 * half;  // channels of this half that exist
    uint32_t bits = 0;
    if (live >= 32) {
#pragma unroll
      for (int c = 0; c < 32; c++) bits |= (uint32_t)s_flag[(half * 32 + c) * HW + p] << c;
    } else {
      for (int c = 0; c < live; c++) bits |= (uint32_t)s_flag[(half * 32 + c) * HW + p] << c;
    }
    reinterpret_cast<uint32_t*>(packed)[((n * HW + p) * Cw + cw) * 2 + half] = bits;
  }
}

// NHWC, C not a multiple of 64, 16-byte aligned input: a CTA takes P pixels (a multiple of 32), whose P * C values are one
// contiguous run that starts on 16 bytes.  128-bit loads along the run, four in flight; the four sign bits of a vector join
// those of seven neighbours by an OR-reduction, which makes the run's sign bits one flat bitmap in shared memory.  The 32-bit
// half k of pixel p is then the bit field of 32 (or what is left of C) bits that starts at bit p * C + 32 * k: one funnel
// shift, stored by consecutive threads to consecutive addresses.
template <typename T>
__global__ void __launch_bounds__(256) pack_nhwc_flat(const int room, const T* __restrict__ x, int C, int P, int halves, long long npix,
                                                      uint32_t* __restrict__ packed) {
  if (room == 2) chain_trigger();
  x = chain_wait_for(x);
  extern __shared__ __align__(16) uint32_t s_bits[];  // [P * C / 32 + 1]
  using V4 = typename Vec4<T>::type;
  const int tid = threadIdx.x, lane = tid & 31;
  const long long p0 = (long long)blockIdx.x * P;
  const int np = (int)min((long long)P, npix - p0);
  const int count = np * C, count4 = (count + 3) / 4;
  const T* src = x + p0 * C;
  const unsigned gmask = 0xFFu << (lane & 24);  // this lane's 8-lane group
  for (int i0 = 0; i0 < count4; i0 += 4 * 256) {
    V4 v[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const int i = i0 + u * 256 + tid;
      v[u] = V4{0, 0, 0, 0};
      if (4 * i + 4 <= count) v[u] = ld_stream_v4(reinterpret_cast<const V4*>(src) + i);
      else if (4 * i < count) {  // the last, partial vector of the tensor
        v[u].x = src[4 * i];
        if (4 * i + 1 < count) v[u].y = src[4 * i + 1];
        if (4 * i + 2 < count) v[u].z = src[4 * i + 2];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const int i = i0 + u * 256 + tid;
      const unsigned nib = neg(v[u].x) | (neg(v[u].y) << 1) | (neg(v[u].z) << 2) | (neg(v[u].w) << 3);
      const unsigned word = __reduce_or_sync(gmask, nib << (4 * (lane & 7)));
      if ((lane & 7) == 0 && i < count4) s_bits[i >> 3] = word;
    }
  }
  if (room == 1) chain_trigger();
  __syncthreads();
  uint32_t* dst = packed + p0 * halves;
  for (int i = tid; i < np * halves; i += 256) {
    const int p = i / halves, k = i - p * halves;
    const int len = C - 32 * k;  // channels from this half on
    uint32_t bits = 0;
    if (len > 0) {
      const int b = p * C + 32 * k;
      bits = __funnelshift_r(s_bits[b >> 5], s_bits[(b >> 5) + 1], b & 31);  // (the word after the last is never looked at)
      if (len < 32) bits &= (1u << len) - 1u;
    }
    dst[i] = bits;
  }
}

// Any layout, any shape: one thread per output word (c2: the word goes to its place in the NC1HWC2 layout, and the
// thread of an odd last word also writes the zero partner).
template <typename T>
__global__ void pack_generic(const int room, const T* __restrict__ x, int nhwc, int C, int HW, int Cw, long long total_words,
                             uint64_t* __restrict__ packed, int c2) {
  if (room == 2) chain_trigger();
  x = chain_wait_for(x);
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= total_words) return;
  const int cw = (int)(t % Cw);
  const long long pix = t / Cw;  // n*HW + hw
  const int c0 = cw * 64, cn = min(64, C - c0);
  uint64_t w = 0;
  if (nhwc) {
    const T* src = x + (size_t)pix * C + c0;
    for (int c = 0; c < cn; c++) w |= (uint64_t)neg(src[c]) << c;
  } else {
    const long long n = pix / HW, hw = pix % HW;
    const T* src = x + ((size_t)n * C + c0) * HW + hw;
    for (int c = 0; c < cn; c++) w |= (uint64_t)neg(src[(size_t)c * HW]) << c;
  }
  if (room == 1) chain_trigger();
  if (c2) {
    const long long n = pix / HW, hw = pix % HW;
    const int C1 = (Cw + 1) / 2;
    uint64_t* v = packed + (((size_t)n * C1 + (cw >> 1)) * HW + hw) * 2;
    v[cw & 1] = w;
    if (cw == Cw - 1 && (cw & 1) == 0) v[1] = 0;
  } else {
    packed[t] = w;
  }
}

// NHWC with C a multiple of 64 and 16-byte aligned input: 16 lanes share one word; each lane tests 4
// channels (one float4), places its nibble, and an OR-reduction over 8-lane groups builds each half.
template <typename T>
__global__ void __launch_bounds__(256) pack_nhwc_c64(const int room, const T* __restrict__ x, long long total_words,
                                                     uint64_t* __restrict__ packed) {
  // (nothing is left to do behind the loop's last loads: a trigger there gains nothing and costs the loop, 64 x 28 x 28 x 256 11.1 against 10.7 us)
  if (room == 2) chain_trigger();
  x = chain_wait_for(x);
  const int lane = threadIdx.x & 31;
  const long long warp_global = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const unsigned gmask = 0xFFu << (lane & 24);  // this lane's 8-lane group
  using V4 = typename Vec4<T>::type;
  // a warp handles 2 words (128 floats) per step; 4 steps in flight per iteration
  for (long long w0 = warp_global * 8; w0 < total_words; w0 += nwarps * 8) {
    V4 v[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const long long word = w0 + 2 * u + (lane >> 4);
      v[u] = V4{0, 0, 0, 0};
      if (word < total_words) v[u] = __ldcs(reinterpret_cast<const V4*>(x) + word * 16 + (lane & 15));
    }
#pragma unroll
    for (int u = 0; u < 4; u++) {
      unsigned nib = neg(v[u].x) | (neg(v[u].y) << 1) | (neg(v[u].z) << 2) | (neg(v[u].w) << 3);
      unsigned half = __reduce_or_sync(gmask, nib << (4 * (lane & 7)));  // 32 channels of this 8-lane group
      unsigned other = __shfl_xor_sync(0xFFFFFFFFu, half, 8);            // the other half of the word
      const long long word = w0 + 2 * u + (lane >> 4);
      if ((lane & 15) == 0 && word < total_words) packed[word] = (uint64_t)half | ((uint64_t)other << 32);
    }
  }
}

__global__ void pack_weights_kernel(const float* __restrict__ w, int O, int C, int taps, int Cw,
                                    uint64_t* __restrict__ wp) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long total = (long long)O * taps * Cw;
  if (t >= total) return;
  const int cw = (int)(t % Cw);
  const int tap = (int)((t / Cw) % taps);
  const int o = (int)(t / ((long long)Cw * taps));
  const int c0 = cw * 64, cn = min(64, C - c0);
  const float* src = w + ((size_t)o * C + c0) * taps + tap;  // OIHW: channel stride = kh*kw
  uint64_t word = 0;
  for (int c = 0; c < cn; c++) word |= (uint64_t)(src[(size_t)c * taps] < 0.0f) << c;
  wp[t] = word;
}

}  // namespace

}  // namespace dabnn

using namespace dabnn;

namespace {

// NHWC rows of no whole words: one contiguous run per CTA (pack_nhwc_flat) or one thread per word (pack_generic), which reads each
// lane's row on its own.  The latter stays ahead where a row is short (17 channels, 200704 pixels: 4.27 against 5.44 us) and the pixels
// many (38 channels, 33504 pixels: 3.64 against 4.98) or few (40 channels, 25 pixels: 2.43 / 2.85; 600 pixels of 39 channels: 3.72 /
// 2.98), and where 32 long rows are more than a CTA reads in the time (about 9 us) that 64 loads in a row take, unless there are
// enough such CTAs for their rate to count (1427 channels, 125 pixels: 9.1 / 17.7; 997 channels, 3248 pixels: 15.6 / 12.3).
bool nhwc_flat_pays(long long npix, int C) {
  if (C <= 32) return false;
  if (C <= 48) return npix >= 256 && npix < 16384;
  return (npix < 32 ? npix : 32) * C <= 18000 || npix >= 64 * 32;
}

// When a pack lets the next kernel of the stream in: 0 at its end, 1 behind its loads, 2 at its start.
// Behind the loads: at most four CTAs per SM, half of what it holds, of a pack of a few microseconds, so that the next kernel finds room on
// every SM (of 103 MB in 392 CTAs, packs one after the other: 28 us each, 39 when they let one another in).  At the start only where
// the pack's CTAs are on three SMs in ten at most: CTAs that come in while there are more of them settle unevenly.  With its pack,
// 3x3, let in at the start, behind the loads, at the end: 256 channels at 14x14, batch 8 (52 CTAs; integer pipes) 13.1, 10.1 and 10.3 us,
// at 7x7, batch 40 (160) 12.9, 11.3 and 11.6; 128 channels at 14x14, batch 2 (8; tensor engine) 7.4 and 8.2 at the start and behind
// the loads, 64 -> 256 at 32x32, batch 3 (24) 6.9 and 7.7.  Packs of 73 x 434 x 7 x 7 (511) one after the other 5.0, 3.7 and 3.9 each.
int room(dim3 grid, dabnn_shape s) {
  const long long ctas = (long long)grid.x * grid.y * grid.z, sms = sm_count();
  if ((long long)s.N * s.C * s.H * s.W > 4 << 20 || ctas > 4 * sms) return 0;
  return 10 * ctas <= 3 * sms ? 2 : 1;
}

template <typename T>
dabnn_status pack_any(const T* x, dabnn_layout in_layout, dabnn_shape s, uint64_t* packed, void* stream,
                      dabnn_packed_layout pl = DABNN_PACKED_NHWC) {
  if (!x || !packed) return DABNN_ERR_NULL;
  if (s.N <= 0 || s.C <= 0 || s.H <= 0 || s.W <= 0) return DABNN_ERR_SHAPE;
  if (in_layout != DABNN_NCHW && in_layout != DABNN_NHWC) return DABNN_ERR_SHAPE;
  if (pl != DABNN_PACKED_NHWC && pl != DABNN_PACKED_NC1HWC2) return DABNN_ERR_SHAPE;
  const bool c2 = pl == DABNN_PACKED_NC1HWC2;
  if (!aligned(x, 4) || !aligned(packed, c2 ? 16 : 8)) return DABNN_ERR_ALIGNMENT;
  const long long HW = (long long)s.H * s.W;
  const long long Cw = (s.C + 63) / 64;
  if (HW > 0x7FFFFFFF || (long long)s.N * HW > 0x7FFFFFFFFFFLL) return DABNN_ERR_UNSUPPORTED;
  const long long total_words = (long long)s.N * HW * Cw;
  cudaStream_t st = as_stream(stream);
  if (in_layout == DABNN_NCHW && HW % 4 == 0 && aligned(x, 16) && Cw * 128 * 8 <= 48 * 1024 &&
      (long long)s.N * HW <= 128LL * 0x7FFFFFFF) {
    const long long npix = (long long)s.N * HW;
    const unsigned grid = (unsigned)((npix + 127) / 128);
    if (c2) launch_next(pack_nchw_vec4<T, true, false>, dim3(grid), dim3(kPackThreads), (size_t)128 * Cw * 8, st, room(dim3(grid), s), x, s.C, (int)HW, (int)Cw, npix, packed);
    else {
      // words split among CTAs until there are sixteen of them per SM, in pairs (16-byte stores); to single words only for a launch of
      // few CTAs (128 images of 512 channels at 14x14: 9.5 us in pairs, 10.9 in single words; 64 images 7.4 and 5.8)
      int parts = 1;
      for (int d = 2; d <= Cw; d++)
        if (Cw % d == 0 && (long long)grid * parts <= (Cw / d > 1 ? 16LL : 4LL) * sm_count()) parts = d;
      const dim3 g(grid, parts);
      const size_t smem = (size_t)128 * (Cw / parts) * 8;
      if (parts > 1 && (long long)grid * parts <= 10LL * sm_count())
        launch_next(pack_nchw_vec4<T, false, true, 10>, g, dim3(kPackThreads), smem, st, room(g, s), x, s.C, (int)HW, (int)Cw, npix, packed);
      else if (parts > 1)
        launch_next(pack_nchw_vec4<T, false, true>, g, dim3(kPackThreads), smem, st, room(g, s), x, s.C, (int)HW, (int)Cw, npix, packed);
      else
        launch_next(pack_nchw_vec4<T, false, false>, g, dim3(kPackThreads), smem, st, room(g, s), x, s.C, (int)HW, (int)Cw, npix, packed);
    }
  } else if (!c2 && in_layout == DABNN_NCHW && HW <= 256 && (s.C * HW) % 4 == 0 && aligned(x, 16) && s.N <= 65535) {
    // (up to two 128-pixel tiles per image; from there on the tiles waste little.  7 x 7 x 512, batch 64: 3.95 -> 2.34 us, batch 256 9.30 -> 4.59;
    // 15 x 15 x 512, batch 64: 7.15 -> 5.32)
    launch_next(pack_nchw_small<T>, dim3((unsigned)Cw, s.N), dim3(256), (size_t)64 * HW, st, room(dim3((unsigned)Cw, s.N), s), x, s.C, (int)HW, (int)Cw, packed);
  } else if (!c2 && in_layout == DABNN_NCHW && s.N <= 65535 && Cw <= 65535) {
    dim3 grid(ceil_div(HW, 128), s.N, (unsigned)Cw);
    launch_next(pack_nchw_tile<T>, grid, dim3(256), (size_t)0, st, room(grid, s), x, s.C, (int)HW, (int)Cw, packed);
  } else if (!c2 && in_layout == DABNN_NHWC && s.C % 64 == 0 && aligned(x, 16)) {
    const long long warps_needed = (total_words + 7) / 8;
    long long blocks = (warps_needed + 7) / 8;
    const long long cap = (long long)sm_count() * 16;
    if (blocks > cap) blocks = cap;
    launch_next(pack_nhwc_c64<T>, dim3((unsigned)blocks), dim3(256), (size_t)0, st, room(dim3((unsigned)blocks), s), x, total_words, packed);
  } else if (!c2 && in_layout == DABNN_NHWC && s.C <= 4096 && aligned(x, 16) && nhwc_flat_pays((long long)s.N * HW, s.C)) {
    // about 8192 values per CTA, 2048 where that leaves less than two CTAs per SM.  37 x 27 x 29 x 100: 7.16 -> 5.15 us, 200 x 14 x 14 x 300 23.3 -> 13.7
    // against one thread per word
    const long long npix = (long long)s.N * HW;
    const int target = npix * s.C >= 2LL * 8192 * sm_count() ? 8192 : 2048;
    const int P = target / s.C >= 64 ? target / s.C / 32 * 32 : 32;
    launch_next(pack_nhwc_flat<T>, dim3(ceil_div(npix, P)), dim3(256), ((size_t)P * s.C / 32 + 1) * 4, st, room(dim3(ceil_div(npix, P)), s), x, s.C, P, (int)(2 * Cw), npix,
                                                                                 reinterpret_cast<uint32_t*>(packed));
  } else {
    const long long blocks = (total_words + 255) / 256;
    if (blocks > 0x7FFFFFFF) return DABNN_ERR_UNSUPPORTED;
    launch_next(pack_generic<T>, dim3((unsigned)blocks), dim3(256), (size_t)0, st, room(dim3((unsigned)blocks), s), x, in_layout == DABNN_NHWC, s.C, (int)HW, (int)Cw, total_words,
                                                   packed, c2 ? 1 : 0);
  }
  return launch_status();
}

}  // namespace

extern "C" dabnn_status dabnn_pack(const float* x, dabnn_layout in_layout, dabnn_shape s, uint64_t* packed,
                                   void* stream) {
  return pack_any<float>(x, in_layout, s, packed, stream);
}

extern "C" dabnn_status dabnn_pack_as(const float* x, dabnn_layout in_layout, dabnn_shape s, dabnn_packed_layout packed_layout,
                                      uint64_t* packed, void* stream) {
  return pack_any<float>(x, in_layout, s, packed, stream, packed_layout);
}

extern "C" size_t dabnn_packed_words(dabnn_shape s, dabnn_packed_layout packed_layout) {
  if (s.N <= 0 || s.C <= 0 || s.H <= 0 || s.W <= 0) return 0;
  const size_t pix = (size_t)s.N * s.H * s.W;
  if (packed_layout == DABNN_PACKED_NC1HWC2) return pix * 2 * (size_t)((s.C + 127) / 128);
  return packed_layout == DABNN_PACKED_NHWC ? pix * (size_t)((s.C + 63) / 64) : 0;
}

extern "C" dabnn_status dabnn_pack_i32(const int32_t* x, dabnn_layout in_layout, dabnn_shape s, uint64_t* packed,
                                       void* stream) {
  return pack_any<int32_t>(x, in_layout, s, packed, stream);
}

extern "C" dabnn_status dabnn_pack_weights(const float* w_oihw, int O, int C, int kh, int kw, uint64_t* wpacked,
                                           void* stream) {
  if (!w_oihw || !wpacked) return DABNN_ERR_NULL;
  if (O <= 0 || C <= 0 || kh <= 0 || kw <= 0) return DABNN_ERR_SHAPE;
  if (!aligned(w_oihw, 4) || !aligned(wpacked, 8)) return DABNN_ERR_ALIGNMENT;
  const long long Cw = (C + 63) / 64;
  const long long total = (long long)O * kh * kw * Cw;
  const long long blocks = (total + 255) / 256;
  if (blocks > 0x7FFFFFFF) return DABNN_ERR_UNSUPPORTED;
  pack_weights_kernel<<<(unsigned)blocks, 256, 0, as_stream(stream)>>>(w_oihw, O, C, kh * kw, (int)Cw, wpacked);
  return launch_status();
}
