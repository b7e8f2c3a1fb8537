// The STEM module variant of the Bi-Real Net 18 front end (Section 2.3 of the paper: the 7x7 convolution and the
// max-pool replaced by a STEM module, 30 % faster on the paper's phone).  The module's figure is not part of the
// paper's text; the structure built here follows the stem block of the network the paper cites for it:
//     s1  = relu(BN(conv3x3/2, pad 1, 3 -> 32))(image)        224 -> 112
//     a   = relu(BN(conv1x1, 32 -> 16))(s1)
//     a   = relu(BN(conv3x3/2, pad 1, 16 -> 32))(a)           112 -> 56
//     b   = maxpool2x2/2(s1)                                  112 -> 56
//     out = BN(conv1x1, 64 -> 64)(concat(a, b))               no activation: the binary blocks take its sign
// Every value is produced by single IEEE-rounded fp32 operations in a fixed order (fmaf chains over c, kh, kw ascending),
// like the rest of the network's fp32 parts, so the result does not depend on tiling.
#include "common.cuh"

namespace dabnn {

namespace {

// The module's 112 x 112 part in one kernel: s1 = relu(BN(conv3x3/2(image))), a1 = relu(BN(conv1x1(s1))) and the 2x2 max of s1
// into channels 32..63 of the concatenated tensor, with s1 (a 16 x 16 tile of it) in shared memory only -- written and read
// twice it was 3 x 51 MB of traffic at batch 32, and every kernel of its own a launch.  A thread owns 4 pixels of a row x 8
// channels; the image patch lies with even and odd columns apart, so a row's three taps take three loads for all 4 pixels, and
// the multiply-adds are packed pairs (same rounding as fmaf).  Every chain keeps its order: c, kh, kw (then c) ascending.
// The STEM-variant forward at batch 32: 558 us with three kernels here, 443 with this one (of which some 15 us are the binary
// blocks' own gain).
constexpr int FR_TS = 16, FR_PS = 2 * FR_TS + 1, FR_HALF = 20, FR_PITCH = 36;
constexpr int FR_SMEM = (27 * 32 + 32 * 16 + 3 * FR_PS * 2 * FR_HALF + FR_TS * FR_TS * FR_PITCH) * 4;
__global__ void __launch_bounds__(256, 3) stem_module_front(const float* __restrict__ img, const float* __restrict__ w1,
                                                            const float* __restrict__ scale1, const float* __restrict__ shift1,
                                                            const float* __restrict__ w2, const float* __restrict__ scale2,
                                                            const float* __restrict__ shift2, float* __restrict__ a1 /*[N][112][112][16]*/,
                                                            float* __restrict__ cat /*[N][56][56][64]*/) {
  constexpr int IH = 224, IW = 224, OHW = 112, TILES = OHW / FR_TS;
  extern __shared__ __align__(16) float sm[];
  float* w1_s = sm;                                  // [27][32]
  float* w2_s = w1_s + 27 * 32;                      // [32][16]
  float* x_s = w2_s + 32 * 16;                       // [3][33][2][HALF]: even and odd columns apart
  float* s1_s = x_s + 3 * FR_PS * 2 * FR_HALF;       // [256 pixels][PITCH]
  const int tid = threadIdx.x;
  const int tile = blockIdx.x % (TILES * TILES);
  const long long n = blockIdx.x / (TILES * TILES);
  const int oh0 = tile / TILES * FR_TS, ow0 = tile % TILES * FR_TS;
  for (int t = tid; t < 3 * FR_PS * FR_PS; t += 256) {
    const int lw = t % FR_PS, lh = (t / FR_PS) % FR_PS, c = t / (FR_PS * FR_PS);
    const int ih = 2 * oh0 - 1 + lh, iw = 2 * ow0 - 1 + lw;
    const bool in = ih >= 0 && ih < IH && iw >= 0 && iw < IW;
    const float* src = in ? img + ((n * 3 + c) * IH + ih) * IW + iw : img;
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(x_s + ((c * FR_PS + lh) * 2 + (lw & 1)) * FR_HALF + (lw >> 1));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(in ? 4 : 0) : "memory");
  }
  for (int t = tid; t < 27 * 32; t += 256) w1_s[(t % 27) * 32 + t / 27] = w1[t];
  for (int t = tid; t < 32 * 16; t += 256) w2_s[(t % 32) * 16 + t / 32] = w2[t];
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  {
    const int chg = tid & 3, pg = tid >> 2, row = pg >> 2, x0 = (pg & 3) * 4;
    unsigned long long acc2[4][4];  // 4 pixels x 4 channel pairs
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) acc2[i][j] = 0ull;
#pragma unroll 1
    for (int c = 0; c < 3; c++)
#pragma unroll
      for (int ki = 0; ki < 3; ki++) {
        const float* xr = x_s + ((c * FR_PS + 2 * row + ki) * 2) * FR_HALF + x0;
        const float4 e4 = *reinterpret_cast<const float4*>(xr);
        const float4 o4 = *reinterpret_cast<const float4*>(xr + FR_HALF);
        const float xe[5] = {e4.x, e4.y, e4.z, e4.w, xr[4]}, xo[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
        for (int kj = 0; kj < 3; kj++) {
          const float* wk = w1_s + ((c * 3 + ki) * 3 + kj) * 32 + chg * 8;
          const float4 wa = *reinterpret_cast<const float4*>(wk), wb = *reinterpret_cast<const float4*>(wk + 4);
          const unsigned long long w2v[4] = {pack_f32x2(wa.x, wa.y), pack_f32x2(wa.z, wa.w), pack_f32x2(wb.x, wb.y), pack_f32x2(wb.z, wb.w)};
#pragma unroll
          for (int i = 0; i < 4; i++) {
            const float xv = kj == 1 ? xo[i] : xe[i + (kj >> 1)];
            const unsigned long long x2 = pack_f32x2(xv, xv);
#pragma unroll
            for (int j = 0; j < 4; j++) fma_f32x2(acc2[i][j], x2, w2v[j]);
          }
        }
      }
    float sc[8], sf[8];
#pragma unroll
    for (int j = 0; j < 8; j++) {
      sc[j] = __ldg(scale1 + chg * 8 + j);
      sf[j] = __ldg(shift1 + chg * 8 + j);
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
      float r[8];
#pragma unroll
      for (int j = 0; j < 4; j++) unpack_f32x2(acc2[i][j], r[2 * j], r[2 * j + 1]);
#pragma unroll
      for (int j = 0; j < 8; j++) {
        r[j] = __fmaf_rn(r[j], sc[j], sf[j]);
        r[j] = (r[j] > 0.0f) ? r[j] : 0.0f;
      }
      float* d = s1_s + (row * FR_TS + x0 + i) * FR_PITCH + chg * 8;
      *reinterpret_cast<float4*>(d) = make_float4(r[0], r[1], r[2], r[3]);
      *reinterpret_cast<float4*>(d + 4) = make_float4(r[4], r[5], r[6], r[7]);
    }
  }
  __syncthreads();
  {  // 1x1, 32 -> 16: two pixels (128 apart in the tile) x 8 channels per thread
    const int chg = tid & 1, px = tid >> 1;
    unsigned long long acc2[2][4];
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) acc2[i][j] = 0ull;
#pragma unroll 2
    for (int k = 0; k < 32; k += 4) {
      const float4 v0 = *reinterpret_cast<const float4*>(s1_s + px * FR_PITCH + k);
      const float4 v1 = *reinterpret_cast<const float4*>(s1_s + (px + 128) * FR_PITCH + k);
      const float xa[4] = {v0.x, v0.y, v0.z, v0.w}, xb[4] = {v1.x, v1.y, v1.z, v1.w};
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const float4 wa = *reinterpret_cast<const float4*>(w2_s + (k + u) * 16 + chg * 8);
        const float4 wb = *reinterpret_cast<const float4*>(w2_s + (k + u) * 16 + chg * 8 + 4);
        const unsigned long long w2v[4] = {pack_f32x2(wa.x, wa.y), pack_f32x2(wa.z, wa.w), pack_f32x2(wb.x, wb.y), pack_f32x2(wb.z, wb.w)};
        const unsigned long long p0 = pack_f32x2(xa[u], xa[u]), p1 = pack_f32x2(xb[u], xb[u]);
#pragma unroll
        for (int j = 0; j < 4; j++) {
          fma_f32x2(acc2[0][j], p0, w2v[j]);
          fma_f32x2(acc2[1][j], p1, w2v[j]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 2; i++) {
      const int q = px + 128 * i;
      float r[8];
#pragma unroll
      for (int j = 0; j < 4; j++) unpack_f32x2(acc2[i][j], r[2 * j], r[2 * j + 1]);
#pragma unroll
      for (int j = 0; j < 8; j++) {
        r[j] = __fmaf_rn(r[j], __ldg(scale2 + chg * 8 + j), __ldg(shift2 + chg * 8 + j));
        r[j] = (r[j] > 0.0f) ? r[j] : 0.0f;
      }
      float* d = a1 + ((n * OHW + oh0 + q / FR_TS) * OHW + ow0 + q % FR_TS) * 16 + chg * 8;
      *reinterpret_cast<float4*>(d) = make_float4(r[0], r[1], r[2], r[3]);
      *reinterpret_cast<float4*>(d + 4) = make_float4(r[4], r[5], r[6], r[7]);
    }
  }
  {  // 2x2 max: 64 pooled pixels x 32 channels, 8 channels of one per thread
    const int c8 = (tid & 3) * 8, pp = tid >> 2, pr = pp >> 3, pc = pp & 7;
    const float* q = s1_s + (2 * pr * FR_TS + 2 * pc) * FR_PITCH + c8;
    float* d = cat + ((n * 56 + oh0 / 2 + pr) * 56 + ow0 / 2 + pc) * 64 + 32 + c8;
#pragma unroll
    for (int h = 0; h < 2; h++) {
      float4 m = *reinterpret_cast<const float4*>(q + 4 * h);
      auto take = [&](const float4 v) {
        m.x = (v.x > m.x) ? v.x : m.x; m.y = (v.y > m.y) ? v.y : m.y; m.z = (v.z > m.z) ? v.z : m.z; m.w = (v.w > m.w) ? v.w : m.w;
      };
      take(*reinterpret_cast<const float4*>(q + FR_PITCH + 4 * h));
      take(*reinterpret_cast<const float4*>(q + FR_TS * FR_PITCH + 4 * h));
      take(*reinterpret_cast<const float4*>(q + (FR_TS + 1) * FR_PITCH + 4 * h));
      *reinterpret_cast<float4*>(d + 4 * h) = m;
    }
  }
}

// The 56 x 56 part in one kernel: relu(BN(conv3x3/2(a1))), concatenated with the pooled channels in shared memory, then
// BN(conv1x1) as the fp32 stream and its packed signs.  Persistent CTAs of 8 x 8 output pixels with both filter banks resident;
// the patch of a1 lies channel by channel with even and odd columns apart (a row's three taps: three loads for 4 pixels).  A
// thread owns 4 pixels x 2 channels of the first product and 4 x 4 of the second; chains run over c, kh, kw (then c) ascending.
// The STEM-variant forward at batch 32: 443 us with the three kernels this replaces (two convolutions and the pack), 395 with it.
constexpr int TL_TS = 8, TL_PS = 2 * TL_TS + 1, TL_HALF = 12, TL_PITCH = 68;
constexpr int TL_PATCH = 16 * TL_PS * 2 * TL_HALF;
constexpr int TL_SMEM = (144 * 32 + 64 * 64 + TL_PATCH + TL_TS * TL_TS * TL_PITCH) * 4;
__global__ void __launch_bounds__(256, 2) stem_module_tail(const float* __restrict__ a1 /*[N][112][112][16]*/,
                                                           const float* __restrict__ cat /*[N][56][56][64], channels 32..63*/,
                                                           int ntiles, const float* __restrict__ w3, const float* __restrict__ scale3,
                                                           const float* __restrict__ shift3, const float* __restrict__ w4,
                                                           const float* __restrict__ scale4, const float* __restrict__ shift4,
                                                           float* __restrict__ out /*[N][56][56][64]*/, uint64_t* __restrict__ bits) {
  constexpr int IHW = 112, OHW = 56, TILES = OHW / TL_TS;
  extern __shared__ __align__(16) float sm[];
  float* w3_s = sm;                     // [144][32]
  float* w4_s = w3_s + 144 * 32;        // [64][64]
  float* x_s = w4_s + 64 * 64;          // [16][17][2][HALF]
  float* c_s = x_s + TL_PATCH;          // [64 pixels][PITCH]: the concatenation
  const int tid = threadIdx.x, lane = tid & 31;
  for (int t = tid; t < 144 * 32; t += 256) w3_s[(t % 144) * 32 + t / 144] = w3[t];
  for (int t = tid; t < 64 * 64; t += 256) w4_s[(t % 64) * 64 + t / 64] = w4[t];
  const int chp = tid & 15, pg = tid >> 4;  // 16 channel groups x 16 groups of 4 pixels of a row
  const int row = pg >> 1, x0 = (pg & 1) * 4;
  const float sc3[2] = {__ldg(scale3 + 2 * chp), __ldg(scale3 + 2 * chp + 1)}, sf3[2] = {__ldg(shift3 + 2 * chp), __ldg(shift3 + 2 * chp + 1)};
  float sc4[4], sf4[4];
#pragma unroll
  for (int j = 0; j < 4; j++) {
    sc4[j] = __ldg(scale4 + 4 * chp + j);
    sf4[j] = __ldg(shift4 + 4 * chp + j);
  }
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const long long n = tile / (TILES * TILES);
    const int rem = tile % (TILES * TILES), oh0 = rem / TILES * TL_TS, ow0 = rem % TILES * TL_TS;
    for (int t = tid; t < TL_PS * TL_PS * 4; t += 256) {
      const int q = t & 3, px = t >> 2, lw = px % TL_PS, lh = px / TL_PS;
      const int ih = 2 * oh0 - 1 + lh, iw = 2 * ow0 - 1 + lw;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (ih >= 0 && ih < IHW && iw >= 0 && iw < IHW) v = __ldg(reinterpret_cast<const float4*>(a1 + ((n * IHW + ih) * IHW + iw) * 16) + q);
      float* d = x_s + ((4 * q * TL_PS + lh) * 2 + (lw & 1)) * TL_HALF + (lw >> 1);
      d[0] = v.x;
      d[TL_PS * 2 * TL_HALF] = v.y;
      d[2 * TL_PS * 2 * TL_HALF] = v.z;
      d[3 * TL_PS * 2 * TL_HALF] = v.w;
    }
#pragma unroll
    for (int u = 0; u < 2; u++) {
      const int t = tid + 256 * u, q = t & 7, px = t >> 3;
      const long long pix = (n * OHW + oh0 + px / TL_TS) * OHW + ow0 + px % TL_TS;
      *reinterpret_cast<float4*>(c_s + px * TL_PITCH + 32 + 4 * q) = __ldg(reinterpret_cast<const float4*>(cat + pix * 64 + 32) + q);
    }
    __syncthreads();
    {
      unsigned long long acc2[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 1
      for (int c = 0; c < 16; c++)
#pragma unroll
        for (int ki = 0; ki < 3; ki++) {
          const float* xr = x_s + ((c * TL_PS + 2 * row + ki) * 2) * TL_HALF + x0;
          const float4 e4 = *reinterpret_cast<const float4*>(xr);
          const float4 o4 = *reinterpret_cast<const float4*>(xr + TL_HALF);
          const float xe[5] = {e4.x, e4.y, e4.z, e4.w, xr[4]}, xo[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
          for (int kj = 0; kj < 3; kj++) {
            const float2 w = *reinterpret_cast<const float2*>(w3_s + (c * 9 + ki * 3 + kj) * 32 + 2 * chp);
            const unsigned long long w2 = pack_f32x2(w.x, w.y);
#pragma unroll
            for (int i = 0; i < 4; i++) {
              const float xv = kj == 1 ? xo[i] : xe[i + (kj >> 1)];
              fma_f32x2(acc2[i], pack_f32x2(xv, xv), w2);
            }
          }
        }
#pragma unroll
      for (int i = 0; i < 4; i++) {
        float r0, r1;
        unpack_f32x2(acc2[i], r0, r1);
        r0 = __fmaf_rn(r0, sc3[0], sf3[0]);
        r1 = __fmaf_rn(r1, sc3[1], sf3[1]);
        *reinterpret_cast<float2*>(c_s + (row * TL_TS + x0 + i) * TL_PITCH + 2 * chp) = make_float2((r0 > 0.0f) ? r0 : 0.0f, (r1 > 0.0f) ? r1 : 0.0f);
      }
    }
    __syncthreads();
    {
      const float* cp = c_s + (row * TL_TS + x0) * TL_PITCH;
      unsigned long long acc2[4][2];
#pragma unroll
      for (int i = 0; i < 4; i++) acc2[i][0] = acc2[i][1] = 0ull;
#pragma unroll 2
      for (int k = 0; k < 64; k += 4) {
        float xv[4][4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const float4 v = *reinterpret_cast<const float4*>(cp + i * TL_PITCH + k);
          xv[i][0] = v.x; xv[i][1] = v.y; xv[i][2] = v.z; xv[i][3] = v.w;
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
          const float4 w = *reinterpret_cast<const float4*>(w4_s + (k + u) * 64 + 4 * chp);
          const unsigned long long wa = pack_f32x2(w.x, w.y), wb = pack_f32x2(w.z, w.w);
#pragma unroll
          for (int i = 0; i < 4; i++) {
            const unsigned long long x2 = pack_f32x2(xv[i][u], xv[i][u]);
            fma_f32x2(acc2[i][0], x2, wa);
            fma_f32x2(acc2[i][1], x2, wb);
          }
        }
      }
      const unsigned gmask = 0xFFu << (lane & 24);
#pragma unroll
      for (int i = 0; i < 4; i++) {
        float r[4];
        unpack_f32x2(acc2[i][0], r[0], r[1]);
        unpack_f32x2(acc2[i][1], r[2], r[3]);
        unsigned nib = 0;
#pragma unroll
        for (int j = 0; j < 4; j++) {
          r[j] = __fmaf_rn(r[j], sc4[j], sf4[j]);
          nib |= (unsigned)(r[j] < 0.0f) << j;
        }
        const long long pix = (n * OHW + oh0 + row) * OHW + ow0 + x0 + i;
        *reinterpret_cast<float4*>(out + pix * 64 + 4 * chp) = make_float4(r[0], r[1], r[2], r[3]);
        const unsigned half = __reduce_or_sync(gmask, nib << (4 * (lane & 7)));
        const unsigned other = __shfl_xor_sync(0xFFFFFFFFu, half, 8);
        if (chp == 0) bits[pix] = (uint64_t)half | ((uint64_t)other << 32);
      }
    }
    __syncthreads();
  }
}

}  // namespace

// a1: [N][112][112][16], cat: [N][56][56][64] (scratch); out: [N][56][56][64] fp32, bits: its signs.
dabnn_status launch_stem_module(const dabnn_stem_module_params* sm, const float* images, int N, float* a1, float* cat,
                                float* out, uint64_t* bits, cudaStream_t st) {
  for (int i = 0; i < 4; i++)
    if (!sm->w[i] || !sm->scale[i] || !sm->shift[i]) return DABNN_ERR_NULL;
  {
    static bool configured[kMaxDevices] = {};
    const int dev = current_device();
    if (dev < 0) return DABNN_ERR_CUDA;
    if (!configured[dev]) {
      if (cudaFuncSetAttribute(stem_module_front, cudaFuncAttributeMaxDynamicSharedMemorySize, FR_SMEM) != cudaSuccess ||
          cudaFuncSetAttribute(stem_module_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, TL_SMEM) != cudaSuccess) {
        cudaGetLastError();
        return DABNN_ERR_CUDA;
      }
      configured[dev] = true;
    }
    stem_module_front<<<(unsigned)(N * 49), 256, FR_SMEM, st>>>(images, sm->w[0], sm->scale[0], sm->shift[0], sm->w[1], sm->scale[1],
                                                              sm->shift[1], a1, cat);
  }
  const int ntiles = N * 49, cap = 2 * sm_count();
  stem_module_tail<<<ntiles < cap ? ntiles : cap, 256, TL_SMEM, st>>>(a1, cat, ntiles, sm->w[2], sm->scale[2], sm->shift[2], sm->w[3],
                                                                   sm->scale[3], sm->shift[3], out, bits);
  return launch_status();
}

}  // namespace dabnn
