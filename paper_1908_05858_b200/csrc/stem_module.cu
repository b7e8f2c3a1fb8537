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

// Direct fp32 convolution, zero padding, then y = fmaf(acc, scale, shift) and an optional ReLU, as a register-tiled product
// with a fixed summation order.  A CTA of 256 threads owns 128 consecutive output pixels x BN output channels; K = CIN * k * k
// is walked in chunks of CG channels x all taps (k index = c * taps + tap ascending: the pinned order).  Per chunk the
// im2col values of the CTA's pixels go to shared memory k-major ([k][pixel]: a thread later reads its 4 pixels as one
// 128-bit load) and the filters as [k][channel] (broadcast reads); thread (tx, ty) keeps 4 pixels x TN = BN / 8 channels.
// The loader thread of pixel p fetches CG consecutive channels of a tap with one vector load.  Taps outside the image are
// zeros: fmaf(0, w, acc) = acc.
// x: NHWC with CIN channels per pixel; y: NHWC with y_stride channels per pixel, written at channel y_off.
template <int K, int S, int PAD, int CIN, int BN, int CG, bool RELU>
__global__ void __launch_bounds__(256) conv_fp32_pinned(const float* __restrict__ x, int N, int H, int W, int OH, int OW,
                                                        const float* __restrict__ w_oihw, const float* __restrict__ scale,
                                                        const float* __restrict__ shift, float* __restrict__ y,
                                                        int y_stride, int y_off) {
  constexpr int BM = 128, T = K * K, KC = CG * T, TN = BN / 8, AP = BM + 4, WP = BN + 4;
  static_assert(CIN % CG == 0 && BN % 16 == 0 && (K == 1 ? CG % 8 == 0 : CG == 4), "tile");
  __shared__ __align__(16) float a_s[KC * AP];
  __shared__ __align__(16) float w_s[KC * WP];
  const int tid = threadIdx.x;
  const long long npix = (long long)N * OH * OW;
  const long long p0 = (long long)blockIdx.x * BM;
  const int o0 = blockIdx.y * BN;
  // loader role: pixel lp, and one half of the chunk's taps (or channels, for a single tap)
  const int lp = tid & (BM - 1), lhalf = tid >> 7;
  const long long pl = p0 + lp;
  int ih0 = 0, iw0 = 0;
  long long xn = -1;  // offset of image n in x, or -1 for a pixel beyond the end
  if (pl < npix) {
    const int ow = (int)(pl % OW), oh = (int)((pl / OW) % OH);
    const long long n = pl / ((long long)OW * OH);
    ih0 = oh * S - PAD;
    iw0 = ow * S - PAD;
    xn = n * (long long)CIN * H * W;
  }
  const int tx = tid & 31, ty = tid >> 5;
  float acc[4][TN];
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int j = 0; j < TN; j++) acc[i][j] = 0.0f;

  for (int c0 = 0; c0 < CIN; c0 += CG) {
    // filters of this chunk: w_s[k][o] = w[o0 + o][c0 * T + k]
    for (int idx = tid; idx < KC * BN; idx += 256) {
      const int o = idx / KC, k = idx - o * KC;  // consecutive threads: consecutive k of one filter (contiguous in OIHW)
      w_s[k * WP + o] = w_oihw[(size_t)(o0 + o) * (CIN * T) + c0 * T + k];
    }
    // im2col values of this chunk
    if (T == 1) {
      // one tap: the two loader threads of a pixel take half of the chunk's channels each
#pragma unroll
      for (int q = 0; q < CG / 8; q++) {
        const int cc = lhalf * (CG / 2) + 4 * q;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (xn >= 0) v = __ldg(reinterpret_cast<const float4*>(x + xn + ((long long)ih0 * W + iw0) * CIN + c0 + cc));
        a_s[(cc + 0) * AP + lp] = v.x; a_s[(cc + 1) * AP + lp] = v.y; a_s[(cc + 2) * AP + lp] = v.z; a_s[(cc + 3) * AP + lp] = v.w;
      }
    } else {
#pragma unroll
      for (int t = 0; t < T; t++) {
        if ((t & 1) != lhalf) continue;
        const int ih = ih0 + t / K, iw = iw0 + t % K;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (xn >= 0 && ih >= 0 && ih < H && iw >= 0 && iw < W) v = __ldg(reinterpret_cast<const float4*>(x + xn + ((long long)ih * W + iw) * CIN + c0));
        a_s[(0 * T + t) * AP + lp] = v.x; a_s[(1 * T + t) * AP + lp] = v.y; a_s[(2 * T + t) * AP + lp] = v.z; a_s[(3 * T + t) * AP + lp] = v.w;
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < KC; k++) {
      const float4 a = *reinterpret_cast<const float4*>(a_s + k * AP + 4 * tx);
      float wv[TN];
#pragma unroll
      for (int j = 0; j < TN; j += 2) {
        const float2 w2 = *reinterpret_cast<const float2*>(w_s + k * WP + ty * TN + j);
        wv[j] = w2.x; wv[j + 1] = w2.y;
      }
#pragma unroll
      for (int j = 0; j < TN; j++) {
        acc[0][j] = __fmaf_rn(a.x, wv[j], acc[0][j]);
        acc[1][j] = __fmaf_rn(a.y, wv[j], acc[1][j]);
        acc[2][j] = __fmaf_rn(a.z, wv[j], acc[2][j]);
        acc[3][j] = __fmaf_rn(a.w, wv[j], acc[3][j]);
      }
    }
    __syncthreads();
  }
  const int o = o0 + ty * TN;
  float sc[TN], sf[TN];
#pragma unroll
  for (int j = 0; j < TN; j++) { sc[j] = __ldg(scale + o + j); sf[j] = __ldg(shift + o + j); }
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const long long pp = p0 + 4 * tx + i;
    if (pp >= npix) continue;
    float* dst = y + pp * y_stride + y_off + o;
#pragma unroll
    for (int j = 0; j < TN; j += 2) {
      float r0 = __fmaf_rn(acc[i][j], sc[j], sf[j]), r1 = __fmaf_rn(acc[i][j + 1], sc[j + 1], sf[j + 1]);
      if (RELU) { r0 = (r0 > 0.0f) ? r0 : 0.0f; r1 = (r1 > 0.0f) ? r1 : 0.0f; }
      *reinterpret_cast<float2*>(dst + j) = make_float2(r0, r1);
    }
  }
}

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

}  // namespace

// a1: [N][112][112][16], cat: [N][56][56][64] (scratch); out: [N][56][56][64] fp32, bits: its signs.
dabnn_status launch_stem_module(const dabnn_stem_module_params* sm, const float* images, int N, float* a1, float* cat,
                                float* out, uint64_t* bits, cudaStream_t st) {
  for (int i = 0; i < 4; i++)
    if (!sm->w[i] || !sm->scale[i] || !sm->shift[i]) return DABNN_ERR_NULL;
  const long long p56 = (long long)N * 56 * 56;  // output pixels
  {
    static bool configured[kMaxDevices] = {};
    const int dev = current_device();
    if (dev < 0) return DABNN_ERR_CUDA;
    if (!configured[dev]) {
      if (cudaFuncSetAttribute(stem_module_front, cudaFuncAttributeMaxDynamicSharedMemorySize, FR_SMEM) != cudaSuccess) {
        cudaGetLastError();
        return DABNN_ERR_CUDA;
      }
      configured[dev] = true;
    }
    stem_module_front<<<(unsigned)(N * 49), 256, FR_SMEM, st>>>(images, sm->w[0], sm->scale[0], sm->shift[0], sm->w[1], sm->scale[1],
                                                              sm->shift[1], a1, cat);
  }
  conv_fp32_pinned<3, 2, 1, 16, 32, 4, true><<<dim3(ceil_div(p56, 128), 1), 256, 0, st>>>(
      a1, N, 112, 112, 56, 56, sm->w[2], sm->scale[2], sm->shift[2], cat, 64, 0);
  conv_fp32_pinned<1, 1, 0, 64, 64, 16, false><<<dim3(ceil_div(p56, 128), 1), 256, 0, st>>>(
      cat, N, 56, 56, 56, 56, sm->w[3], sm->scale[3], sm->shift[3], out, 64, 0);
  dabnn_status s = launch_status();
  if (s != DABNN_OK) return s;
  const dabnn_shape sh = {N, 64, 56, 56};
  return dabnn_pack(out, DABNN_NHWC, sh, bits, st);
}

}  // namespace dabnn
