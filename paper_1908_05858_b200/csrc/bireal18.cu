// Bi-Real Net 18 forward (Section 2.3, Table 2 of the paper): fp32 stem and head around sixteen binary
// 3x3 convolutions whose BN + shortcut + sign + re-pack run in the convolution's epilogue.
//
// All activations between layers are NHWC.  Every fp32 value is produced by single IEEE-rounded
// operations in a fixed order (explicit fmaf chains, ascending channel / tap order), never by tensor
// cores or split sums, because the next binary layer takes the SIGN of these values: a different
// rounding order could flip a bit and change integer results downstream.
#include <mutex>

#include "common.cuh"

namespace dabnn {

thread_local bool g_chain_launch = false;  // see launch_chain() in common.cuh

namespace {

// ---- BN fold, in double ---------------------------------------------------------------------------
__global__ void bn_fold_kernel(const float* gamma, const float* beta, const float* mean, const float* var, double eps,
                               int O, float* scale, float* shift) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= O) return;
  const double sd = __ddiv_rn((double)gamma[o], __dsqrt_rn(__dadd_rn((double)var[o], eps)));
  scale[o] = (float)sd;
  shift[o] = (float)__dsub_rn((double)beta[o], __dmul_rn((double)mean[o], sd));
}

// ---- stem: conv 7x7 / 2, 3 -> 64, zero pad 3, then BN ----------------------------------------------
// A CTA computes a TS x TS tile of output pixels for 4 * CPT channels (all 64 with CPT = 16; with CPT = 8 two CTAs
// share a tile, which spreads a single image over twice as many CTAs).  The input patch sits in shared
// memory with even and odd columns apart, so that lanes walking along ow (input stride 2) read
// consecutive words.  A thread owns PPT pixels (rows TS/PPT apart... see below) x CPT channels and runs one fmaf
// chain per output over (c, kh, kw) in that order.  Zero padding is held as zeros in the patch:
// fmaf(0, w, acc) returns acc.
constexpr int STEM_K = 147;
// Columns per parity of the input patch, padded: the lanes of a warp read 8 consecutive columns of 4 patch rows that
// are two rows (4 * half words) apart, which fall on distinct banks when 4 * half is 8 or 24 modulo 32.
__host__ __device__ constexpr int stem_half(int ps) {
  int h = (ps + 1) / 2 + 1;
  while ((4 * h) % 32 != 8 && (4 * h) % 32 != 24) h++;
  return h;
}

template <int TS, int PPT, int CPT>
__global__ void __launch_bounds__((TS * TS / PPT) * 4, 2) stem_conv_bn(const float* __restrict__ img,
                                                                       const float* __restrict__ w,
                                                                       const float* __restrict__ scale,
                                                                       const float* __restrict__ shift, int N,
                                                                       float* __restrict__ out /*[N][112][112][64]*/) {
  // (the head of a forward: what it reads may be the work of the kernel before it, whatever that was)
  w = chain_wait_for(w);
  scale = after_wait(scale);
  shift = after_wait(shift);
  constexpr int IH = 224, IW = 224, OHW = 112;
  constexpr int PS = 2 * TS + 5;         // patch side
  constexpr int HALF = stem_half(PS);
  constexpr int PATCH = 3 * PS * 2 * HALF;  // floats per patch buffer
  constexpr int PGROUPS = TS * TS / PPT; // pixel groups = threads per channel group
  constexpr int THREADS = PGROUPS * 4;
  constexpr int RSTEP = TS / PPT;        // a thread's pixels are RSTEP rows apart
  constexpr int TILES = (OHW + TS - 1) / TS;
  constexpr int CB = 4 * CPT;            // channels per CTA (blockIdx.y picks which): four thread groups of CPT channels
  static_assert(CPT == 16 || CPT == 8, "channels per thread");
  extern __shared__ __align__(16) float sm[];
  float* w_s = sm;                       // [147][CB], filled once per CTA
  float* x_s = sm + STEM_K * CB;         // [2 buffers][3][PS][2][HALF]
  float* w_raw = x_s + 2 * PATCH;        // [CB][147] as in global memory, until it has been transposed into w_s
  const int ch0 = blockIdx.y * CB;
  w += (size_t)ch0 * STEM_K;             // this CTA's rows of the [64][147] weight matrix
  const int tid = threadIdx.x;
  if ((reinterpret_cast<uintptr_t>(w) & 15) == 0) {  // one coalesced asynchronous copy, in flight together with the first patch
    for (int t = tid; t < STEM_K * CB / 4; t += THREADS) {
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(w_raw + 4 * t);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(w + 4 * t) : "memory");
    }
  } else {
    for (int t = tid; t < STEM_K * CB; t += THREADS) w_raw[t] = w[t];
  }
  const long long ntiles = (long long)N * TILES * TILES;
  // asynchronous copy of one tile's zero-padded input patch (even and odd columns apart)
  auto load_patch = [&](long long tile, float* dst) {
    const int n = (int)(tile / (TILES * TILES));
    const int rem = (int)(tile % (TILES * TILES));
    const int ih_base = 2 * (rem / TILES) * TS - 3, iw_base = 2 * (rem % TILES) * TS - 3;
    for (int t = tid; t < 3 * PS * PS; t += THREADS) {
      const int lw = t % PS, lh = (t / PS) % PS, c = t / (PS * PS);
      const int ih = ih_base + lh, iw = iw_base + lw;
      const bool in = ih >= 0 && ih < IH && iw >= 0 && iw < IW;
      const float* src = in ? img + (((size_t)n * 3 + c) * IH + ih) * IW + iw : img;
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + ((c * PS + lh) * 2 + (lw & 1)) * HALF + (lw >> 1));
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(in ? 4 : 0) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int cg = tid / PGROUPS;          // channel group: 16 channels
  const int pg = tid % PGROUPS;
  const int low = pg % TS, lohb = pg / TS;  // pixels (lohb + RSTEP*i, low)
  float sc[CPT], sf[CPT];
#pragma unroll
  for (int j = 0; j < CPT; j++) {
    sc[j] = scale[ch0 + cg * CPT + j];
    sf[j] = shift[ch0 + cg * CPT + j];
  }
  long long tile = blockIdx.x;
  int buf = 0;
  if (tile < ntiles) load_patch(tile, x_s);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  // [CB][147] -> [147][CB]: lanes walk over o, 147 words apart in w_raw (an odd stride: distinct banks) and consecutive in w_s
  for (int t = tid; t < STEM_K * CB; t += THREADS) w_s[t] = w_raw[(t % CB) * STEM_K + t / CB];
  for (; tile < ntiles; tile += gridDim.x, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // this tile's patch (and, the first time, the weights) are in place; the other buffer is free
    if (tile + gridDim.x < ntiles) load_patch(tile + gridDim.x, x_s + (buf ^ 1) * PATCH);
    const float* xb = x_s + buf * PATCH;
    unsigned long long acc2[PPT][CPT / 2];  // channel pairs (packed fp32 FMAs, same rounding as scalar fmaf)
#pragma unroll
    for (int i = 0; i < PPT; i++)
#pragma unroll
      for (int j = 0; j < CPT / 2; j++) acc2[i][j] = 0ull;
#pragma unroll 1
    for (int c = 0; c < 3; c++)
#pragma unroll 1
      for (int ki = 0; ki < 7; ki++) {  // one row of taps per iteration keeps the loop body inside the instruction cache
#pragma unroll
        for (int kj = 0; kj < 7; kj++) {
          const int k = (c * 7 + ki) * 7 + kj;
          unsigned long long w2[CPT / 2];
#pragma unroll
          for (int q = 0; q < CPT / 4; q++) {
            const float4 t4 = *reinterpret_cast<const float4*>(w_s + k * CB + cg * CPT + 4 * q);
            w2[2 * q] = pack_f32x2(t4.x, t4.y);
            w2[2 * q + 1] = pack_f32x2(t4.z, t4.w);
          }
#pragma unroll
          for (int i = 0; i < PPT; i++) {
            const int lh = 2 * (lohb + RSTEP * i) + ki;
            const float xv = xb[((c * PS + lh) * 2 + (kj & 1)) * HALF + low + (kj >> 1)];
            const unsigned long long x2 = pack_f32x2(xv, xv);
#pragma unroll
            for (int j = 0; j < CPT / 2; j++) fma_f32x2(acc2[i][j], x2, w2[j]);
          }
        }
      }
    float acc[PPT][CPT];
#pragma unroll
    for (int i = 0; i < PPT; i++)
#pragma unroll
      for (int j = 0; j < CPT / 2; j++) unpack_f32x2(acc2[i][j], acc[i][2 * j], acc[i][2 * j + 1]);
    if (tile + gridDim.x >= ntiles) chain_trigger();  // the CTA's last tile: the next kernel may start its set-up
    const int n = (int)(tile / (TILES * TILES));
    const int rem = (int)(tile % (TILES * TILES));
    const int oh0 = (rem / TILES) * TS, ow0 = (rem % TILES) * TS;
#pragma unroll
    for (int i = 0; i < PPT; i++) {
      const int oh = oh0 + lohb + RSTEP * i, ow = ow0 + low;
      if (oh >= OHW || ow >= OHW) continue;
      float* dst = out + (((size_t)n * OHW + oh) * OHW + ow) * 64 + ch0 + cg * CPT;
#pragma unroll
      for (int j = 0; j < CPT; j += 4)
        *reinterpret_cast<float4*>(dst + j) =
            make_float4(__fmaf_rn(acc[i][j], sc[j], sf[j]), __fmaf_rn(acc[i][j + 1], sc[j + 1], sf[j + 1]),
                        __fmaf_rn(acc[i][j + 2], sc[j + 2], sf[j + 2]), __fmaf_rn(acc[i][j + 3], sc[j + 3], sf[j + 3]));
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Larger batches: the convolution, its BN and the 3x3 / 2 max-pool in one kernel, so that the 112x112x64 tensor (411 MB at
// batch 128) is never written.  A group of four warps sweeps down the image: a unit is one pooled row, i.e. the convolution
// rows 2p and 2p + 1 at full width (two warps each); row 2p - 1, which the pooling also needs, is the last one of the unit
// before, kept in shared memory.  Only the first unit of a group's range computes that row again.  A CTA has two such groups
// (one warp of each per scheduler), so that one group's pooling, stores and barriers run under the other's multiply-adds,
// and one copy of the weights for both.
// A thread owns 14 pixels (along a row) x CPT channels: per (c, kh) it loads the 33 input values of its pixels once for all
// seven horizontal taps.  The order of every output's fmaf chain is the one above: c, then kh, then kw.
// Bound by the FMA pipe: batch 128 takes 419 us of it with the rows computed twice; measured 528 us (pooling and stores 20 of
// them, the rest the loop, whose bare form reaches 88 % of the pipe), against 557 + 96 for a convolution kernel that wrote the
// tensor and a max-pool kernel that read it.
constexpr int SP_ROWS = 18;    // input rows a group holds: nine of the unit at work, up to nine of the next one
constexpr int SP_PITCH = 232;  // floats per row: columns -4 .. 227 (the image's 224 on a 16-byte boundary)
template <int CPT>
constexpr int stem_pool_smem() { return (STEM_K * 8 * CPT + 2 * SP_ROWS * 3 * SP_PITCH + 2 * 3 * 56 * 8 * CPT + 2 * 2 * 8 * CPT) * 4; }

__device__ __forceinline__ float max3(float a, float b, float c) { return fmaxf(fmaxf(a, b), c); }

template <int CPT>
__global__ void __launch_bounds__(256, 1) stem_pool(const float* __restrict__ img, const float* __restrict__ w,
                                                    const float* __restrict__ scale, const float* __restrict__ shift, int N,
                                                    float* __restrict__ y /*[N][56][56][64]*/,
                                                    uint32_t* __restrict__ bits /*[N][56][56][2]*/) {
  if constexpr (CPT == 4) {  // (the head of a forward: what it reads may be the work of the kernel before it)
    w = chain_wait_for(w);
    scale = after_wait(scale);
    shift = after_wait(shift);
  }
  // A chained successor may set itself up as this grid drains; it waits for all of it before reading activations.  Behind the wait:
  // the successor reads its weights before its own, and they may be the work of the kernel before this one.
  chain_trigger();
  constexpr int IHW = 224, PHW = 56;
  constexpr int CB = 8 * CPT;  // channels per CTA; blockIdx.y picks which
  constexpr int PXT = 14;      // pixels per thread
  static_assert(CPT == 8 || CPT == 4, "channels per thread");
  extern __shared__ __align__(16) float sm[];
  float* w_s = sm;                                         // [147][CB]
  float* x_all = w_s + STEM_K * CB;                        // [2 groups][SP_ROWS][3][SP_PITCH]
  float* pool_all = x_all + 2 * SP_ROWS * 3 * SP_PITCH;    // [2 groups][3][56][CB]: rows pooled along w: 2p; 2p + 1 of this unit
                                                           // and of the one before, in turn
  float* edge_all = pool_all + 2 * 3 * PHW * CB;           // [2 groups][2 rows][CB]: the last pixel of a row's left half
  const int tid = threadIdx.x, lane = tid & 31;
  const int group = tid >> 7, gtid = tid & 127, gwarp = gtid >> 5;
  const int rho = (gwarp >> 1) ^ group, half = gwarp & 1;  // row of the unit, half of the row (the two groups' rows on
                                                           // different schedulers: a range's first unit needs one row only)
  const int chg = lane & 7, pxg = half * 4 + (lane >> 3);
  const int ch0 = blockIdx.y * CB;
  float* xg = x_all + group * SP_ROWS * 3 * SP_PITCH;
  float* pool = pool_all + group * 3 * PHW * CB;
  float* edge = edge_all + group * 2 * CB;

  const long long units = (long long)N * PHW;
  const int u_cta = (int)(units * blockIdx.x / gridDim.x), u_end = (int)(units * (blockIdx.x + 1) / gridDim.x);
  const int u_mid = u_cta + (u_end - u_cta + 1) / 2;
  const int first = group ? u_mid : u_cta, last = group ? u_end : u_mid;  // this group's units
  const bool img_vec = (reinterpret_cast<uintptr_t>(img) & 15) == 0;

  // asynchronous copies of input rows r0 .. 8 of unit u's nine, zeros outside the image, into the ring from `slot` on: two
  // channel rows at a time, 56 threads each
  const int lq = gtid < 56 ? gtid : gtid - 56, lh = gtid < 56 ? 0 : 1;
  auto load_rows = [&](int u, int slot, int r0) {
    if (gtid >= 112) return;
    const int n = u / PHW, ih0 = 4 * (u % PHW) - 3;
    int r = r0, c = lh;
#pragma unroll 1
    while (r < 9) {
      const int ih = ih0 + r;
      const bool in = ih >= 0 && ih < IHW;
      const int s = slot + r >= SP_ROWS ? slot + r - SP_ROWS : slot + r;
      const float* src = img + (((size_t)n * 3 + c) * IHW + (in ? ih : 0)) * IHW;
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(xg + (s * 3 + c) * SP_PITCH + 4);
      if (img_vec) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d + 16 * lq), "l"(src + 4 * lq), "r"(in ? 16 : 0) : "memory");
      } else {
#pragma unroll
        for (int e = 0; e < 4; e++)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d + 4 * (lq + 56 * e)), "l"(src + lq + 56 * e), "r"(in ? 4 : 0) : "memory");
      }
      c += 2;
      if (c >= 3) { c -= 3; r++; }
    }
  };
  auto group_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(1 + group) : "memory"); };
  auto ring_next = [&](int u, int slot) {  // ring slot of unit u + 1's first row: of the same image (five rows shared) or the next
    const int s = slot + ((u + 1) % PHW != 0 ? 4 : 9);
    return s >= SP_ROWS ? s - SP_ROWS : s;
  };

  int u = first < last && first % PHW != 0 ? first - 1 : first;  // (a range that starts inside an image: row 2p - 1 first)
  int slot = 0;
  if (first < last) load_rows(u, slot, 0);
  // columns outside the image, once
  for (int t = gtid; t < SP_ROWS * 3 * 8; t += 128) {
    const int q = t & 7;
    xg[(t >> 3) * SP_PITCH + (q < 4 ? q : SP_PITCH - 8 + q)] = 0.0f;
  }
  {  // weights [CB][147] -> [147][CB] through the pooling rows' space: coalesced in, both steps free of bank conflicts
    static_assert(2 * 3 * PHW * CB >= STEM_K * CB, "room for the weights as they are in global memory");
    for (int t = tid; t < STEM_K * CB; t += 256) pool_all[t] = w[(size_t)ch0 * STEM_K + t];
    __syncthreads();
    for (int t = tid; t < STEM_K * CB; t += 256) w_s[t] = pool_all[(t % CB) * STEM_K + t / CB];
  }
  unsigned long long sc2[CPT / 2], sf2[CPT / 2];
  auto channel = [&](int j) { return j < 4 ? chg * 4 + j : 32 + chg * 4 + (j - 4); };
#pragma unroll
  for (int j = 0; j < CPT / 2; j++) {
    sc2[j] = pack_f32x2(scale[ch0 + channel(2 * j)], scale[ch0 + channel(2 * j + 1)]);
    sf2[j] = pack_f32x2(shift[ch0 + channel(2 * j)], shift[ch0 + channel(2 * j + 1)]);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  if (u + 1 < last) load_rows(u + 1, ring_next(u, slot), (u + 1) % PHW != 0 ? 5 : 0);

  int odd = 0;  // which of the two rows 2p + 1 is this unit's
#pragma unroll 1
  for (; u < last; u++, odd ^= 1) {  // (the unit's rows are in place, the next one's on their way)
    const bool store = u >= first, busy = store || rho == 1;
    float v[PXT][CPT];
    if (busy) {
      unsigned long long acc2[PXT][CPT / 2];  // channel pairs of each pixel
#pragma unroll
      for (int i = 0; i < PXT; i++)
#pragma unroll
        for (int j = 0; j < CPT / 2; j++) acc2[i][j] = 0ull;  // (+0.0, +0.0)
#pragma unroll 1
      for (int c = 0; c < 3; c++)
#pragma unroll 1
        for (int ki = 0; ki < 7; ki++) {
          int s = slot + 2 * rho + ki;
          if (s >= SP_ROWS) s -= SP_ROWS;
          const float* xr = xg + (s * 3 + c) * SP_PITCH + 2 * PXT * pxg;
          float x[36];  // columns 28 * pxg - 4 ..: pixel i's tap kj is x[2 * i + kj + 1]
#pragma unroll
          for (int q = 0; q < 9; q++) {
            const float4 t4 = *reinterpret_cast<const float4*>(xr + 4 * q);
            x[4 * q] = t4.x; x[4 * q + 1] = t4.y; x[4 * q + 2] = t4.z; x[4 * q + 3] = t4.w;
          }
          const float* wk = w_s + (c * 7 + ki) * 7 * CB + chg * 4;
#pragma unroll
          for (int kj = 0; kj < 7; kj++) {
            unsigned long long w2[CPT / 2];
#pragma unroll
            for (int h = 0; h < CPT / 4; h++) {
              const float4 t4 = *reinterpret_cast<const float4*>(wk + kj * CB + 32 * h);
              w2[2 * h] = pack_f32x2(t4.x, t4.y);
              w2[2 * h + 1] = pack_f32x2(t4.z, t4.w);
            }
            // (channel pairs outside, pixels inside, the weights as the first factor; pixels outside: 544 us instead of 528 at batch 128,
            // by the banks of the registers that meet in an instruction, presumably)
#pragma unroll
            for (int j = 0; j < CPT / 2; j++)
#pragma unroll
              for (int i = 0; i < PXT; i++) {
                const float xv = x[2 * i + kj + 1];
                fma_f32x2(acc2[i][j], w2[j], pack_f32x2(xv, xv));
              }
          }
        }
#pragma unroll
      for (int i = 0; i < PXT; i++)
#pragma unroll
        for (int j = 0; j < CPT / 2; j++) {
          unsigned long long t = sf2[j];
          fma_f32x2(t, acc2[i][j], sc2[j]);
          unpack_f32x2(t, v[i][2 * j], v[i][2 * j + 1]);
        }
      if (half == 0 && lane >= 24) {  // what the right half's first pooled pixel needs of this half
#pragma unroll
        for (int j = 0; j < CPT; j++) edge[rho * CB + channel(j)] = v[PXT - 1][j];
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    group_sync();  // the group has left this unit's input rows and the pooling rows of the one before; the next one's rows are here
    slot = ring_next(u, slot);
    if (u + 2 < last) load_rows(u + 2, ring_next(u + 1, slot), (u + 2) % PHW != 0 ? 5 : 0);
    float* row1 = pool + (1 + odd) * PHW * CB;
    if (busy) {  // the maximum over columns 2q - 1, 2q, 2q + 1
      float* dst = rho ? row1 : pool;
      float left[CPT];
#pragma unroll
      for (int j = 0; j < CPT; j++) {
        left[j] = __shfl_up_sync(0xFFFFFFFFu, v[PXT - 1][j], 8);
        if (lane < 8) left[j] = half ? edge[rho * CB + channel(j)] : -INFINITY;
      }
#pragma unroll
      for (int q = 0; q < PXT / 2; q++)
#pragma unroll
        for (int g = 0; g < CPT; g += 4) {
          float h[4];
#pragma unroll
          for (int e = 0; e < 4; e++) h[e] = max3(v[2 * q][g + e], v[2 * q + 1][g + e], q ? v[q ? 2 * q - 1 : 0][g + e] : left[g + e]);
          *reinterpret_cast<float4*>(dst + (PXT / 2 * pxg + q) * CB + 8 * g + chg * 4) = make_float4(h[0], h[1], h[2], h[3]);
        }
    }
    group_sync();
    if (store) {  // the maximum over rows 2p - 1, 2p, 2p + 1: a thread takes four channels of every LPX-th pixel
      constexpr int LANES = CB / 4, LPX = 128 / LANES, NPX = (PHW + LPX - 1) / LPX;
      const float* row_1 = pool + (2 - odd) * PHW * CB;  // row 2p - 1
      const int n = u / PHW, p = u % PHW, c4 = gtid % LANES, px0 = gtid / LANES;
      const float4* r0 = reinterpret_cast<const float4*>(pool) + gtid;
      const float4* r1 = reinterpret_cast<const float4*>(row1) + gtid;
      const float4* rm = reinterpret_cast<const float4*>(row_1) + gtid;
      float* dst = y + (((size_t)n * PHW + p) * PHW + px0) * 64 + ch0 + 4 * c4;
      uint32_t nibs = 0;  // four signs of each of the thread's pixels
#pragma unroll
      for (int i = 0; i < NPX; i++) {
        if (NPX * LPX == PHW || px0 + i * LPX < PHW) {
          const float4 a = r0[128 * i], b = r1[128 * i];
          float4 m = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
          if (p != 0) m = rm[128 * i];
          m.x = fmaxf(max3(a.x, b.x, m.x), -INFINITY); m.y = fmaxf(max3(a.y, b.y, m.y), -INFINITY);
          m.z = fmaxf(max3(a.z, b.z, m.z), -INFINITY); m.w = fmaxf(max3(a.w, b.w, m.w), -INFINITY);
          *reinterpret_cast<float4*>(dst + (size_t)i * LPX * 64) = m;
          nibs |= ((uint32_t)(m.x < 0.0f) | ((uint32_t)(m.y < 0.0f) << 1) | ((uint32_t)(m.z < 0.0f) << 2) | ((uint32_t)(m.w < 0.0f) << 3)) << (4 * i);
        }
      }
      // 8 lanes x 8 nibbles transposed: lane i of each eight gets the 32 signs of pixel i
#pragma unroll
      for (int d = 4; d; d >>= 1) {
        const uint32_t lo = d == 4 ? 0x0000FFFFu : d == 2 ? 0x00FF00FFu : 0x0F0F0F0Fu;
        const uint32_t t = __shfl_xor_sync(0xFFFFFFFFu, nibs, d);
        nibs = lane & d ? (nibs & ~lo) | ((t & ~lo) >> (4 * d)) : (nibs & lo) | ((t & lo) << (4 * d));
      }
      const int px = px0 + (lane & 7) * LPX;
      if ((lane & 7) < NPX && px < PHW) bits[(((size_t)n * PHW + p) * PHW + px) * 2 + (ch0 >> 5) + (c4 >> 3)] = nibs;
    }
  }
}

// In the kernels that take part in chained launches, the pointer to the ACTIVATIONS (what the previous kernel of the stream
// wrote) is deliberately neither __restrict__ nor read with __ldg: such loads count as invariant and the compiler may move
// them above the wait for the previous kernel (seen in a trial that chained the fc kernel: it read pooled values before
// they were written).  Where the read-only path matters, ld_nc_f4 (volatile asm) keeps the load behind the wait.
// ---- maxpool 3x3 / 2, pad 1 (64 channels) -> fp32 residual stream + packed signs -------------------
// A thread handles 4 channels of one output pixel; 16 lanes make one 64-bit word.
__global__ void __launch_bounds__(256) maxpool_pack(const float* x /*[N][112][112][64]*/, long long npix,
                                                    float* __restrict__ y /*[N][56][56][64]*/,
                                                    uint64_t* __restrict__ bits /*[N][56][56][1]*/) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const long long pix = t >> 4;
  const int c4 = (int)(t & 15);
  const bool live = pix < npix;
  float4 m = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  chain_wait();
  chain_trigger();
  if (live) {
    const int ow = (int)(pix % 56), oh = (int)((pix / 56) % 56);
    const long long n = pix / (56 * 56);
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int j = 0; j < 3; j++) {
        const int ih = 2 * oh + i - 1, iw = 2 * ow + j - 1;
        if (ih < 0 || ih >= 112 || iw < 0 || iw >= 112) continue;
        const float4 v = ld_nc_f4(x + ((n * 112 + ih) * 112 + iw) * 64 + c4 * 4);
        m.x = fmaxf(m.x, v.x); m.y = fmaxf(m.y, v.y); m.z = fmaxf(m.z, v.z); m.w = fmaxf(m.w, v.w);
      }
    *reinterpret_cast<float4*>(y + pix * 64 + c4 * 4) = m;
  }
  unsigned nib = 0;
  if (live) nib = (unsigned)(m.x < 0.0f) | ((unsigned)(m.y < 0.0f) << 1) | ((unsigned)(m.z < 0.0f) << 2) | ((unsigned)(m.w < 0.0f) << 3);
  const unsigned gmask = 0xFFu << (lane & 24);
  const unsigned half = __reduce_or_sync(gmask, nib << (4 * (lane & 7)));
  const unsigned other = __shfl_xor_sync(0xFFFFFFFFu, half, 8);
  if (live && (lane & 15) == 0) bits[pix] = (uint64_t)half | ((uint64_t)other << 32);
}

// ---- downsample shortcut: avgpool 2x2 / 2 -> fp32 conv 1x1 (C -> O) -> BN ---------------------------
// Three kernels by the number of outputs, all with one fmaf chain per output over c ascending, as pinned, on pooled activations
// formed on the fly (three adds and one multiply, in that order).  C is 64, 128 or 256 and O = 2 * C.
__device__ __forceinline__ float pool_avg(float a, float b, float c, float d) {
  return __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(a, b), c), d), 0.25f);
}
__device__ __forceinline__ float4 pool_avg4(const float4 (&r)[4]) {
  return make_float4(pool_avg(r[0].x, r[1].x, r[2].x, r[3].x), pool_avg(r[0].y, r[1].y, r[2].y, r[3].y),
                     pool_avg(r[0].z, r[1].z, r[2].z, r[3].z), pool_avg(r[0].w, r[1].w, r[2].w, r[3].w));
}
// The first of the four input pixels of output pixel p; nullptr beyond the last.
__device__ __forceinline__ const float* pool_source(const float* x, long long p, long long npix_out, int HW, int C) {
  if (p >= npix_out) return nullptr;
  const int OHW = HW / 2, ow = (int)(p % OHW), oh = (int)((p / OHW) % OHW);
  const long long n = p / ((long long)OHW * OHW);
  return x + ((n * HW + 2 * oh) * HW + 2 * ow) * C;
}
// (volatile: loads are issued where they stand, all of a batch before the first use, and behind a chained launch's wait)
__device__ __forceinline__ void pool_load(float4 (&r)[4], const float* src, int HW, int C) {
#pragma unroll
  for (int e = 0; e < 4; e++) {
    r[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (src != nullptr)
      asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(r[e].x), "=f"(r[e].y), "=f"(r[e].z), "=f"(r[e].w)
                   : "l"(src + (size_t)((e >> 1) * HW + (e & 1)) * C));
  }
}

// Keeps what is done with a batch's values behind the last of its loads (the first additions would wait for the first of them).
__device__ __forceinline__ void pool_hold(float4 (&r)[4]) {
#pragma unroll
  for (int e = 0; e < 4; e++) asm volatile("" : "+f"(r[e].x), "+f"(r[e].y), "+f"(r[e].z), "+f"(r[e].w));
}

// Many outputs: 64 pixels x 128 channels per CTA, 128 threads of 8 x 8 outputs, K in chunks of 16 through two shared-memory
// stages.  The next chunk's raw inputs wait in registers and are pooled when they are stored, behind the multiply-adds, so that
// nothing waits for them before.  Shared-memory reads (four 128-bit loads per 32 packed multiply-adds) and the short life of a
// CTA hold it at half the FMA pipe: 50, 50 and 48 us at batch 128 (22 of FMA pipe each), against 62, 63 and 61 with 256 threads
// of 4 x 8 outputs; 16 x 8 outputs in persistent CTAs measured 60 to 75.
constexpr int SC_BM = 64, SC_BN = 128, SC_BK = 16;
__global__ void __launch_bounds__(128, 3) shortcut_down(const float* __restrict__ x /*[N][HW][HW][C]*/, int HW, int C,
                                                     const float* __restrict__ w /*[O][C]*/, int O,
                                                     const float* __restrict__ scale, const float* __restrict__ shift,
                                                     long long npix_out, float* __restrict__ y /*[N][HW/2][HW/2][O]*/) {
  chain_trigger();  // (as in the stem: lets a chained tensor-engine block start its set-up under this grid's tail)
  constexpr int XPITCH = SC_BM + 4, WPITCH = SC_BN + 4;
  __shared__ __align__(16) float p_s[2][SC_BK][XPITCH];  // [stage][c][pixel]
  __shared__ __align__(16) float w_s[2][SC_BK][WPITCH];  // [stage][c][channel]
  const int tid = threadIdx.x;
  const long long p0 = (long long)blockIdx.x * SC_BM;
  const int o0 = blockIdx.y * SC_BN;
  // loader roles: four consecutive c of pixels tid / 4 and tid / 4 + 32, and of channels tid / 4 + 32 * v
  const int lc = (tid & 3) * 4, lp = tid >> 2;
  const float* xq[2];
#pragma unroll
  for (int h = 0; h < 2; h++) {
    xq[h] = pool_source(x, p0 + lp + 32 * h, npix_out, HW, C);
    if (xq[h] != nullptr) xq[h] += lc;
  }
  const float* wq = w + (size_t)(o0 + lp) * C + lc;
  const bool w_vec = (reinterpret_cast<uintptr_t>(w) & 15) == 0;
  float4 raw[2][4], wreg[4];
  auto load = [&](int c0) {
#pragma unroll
    for (int h = 0; h < 2; h++) pool_load(raw[h], xq[h] != nullptr ? xq[h] + c0 : nullptr, HW, C);
#pragma unroll
    for (int v = 0; v < 4; v++) {
      const float* q = wq + (size_t)v * 32 * C + c0;
      if (w_vec) wreg[v] = *reinterpret_cast<const float4*>(q);
      else wreg[v] = make_float4(q[0], q[1], q[2], q[3]);
    }
  };
  auto put = [&](int st) {
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const float4 v = pool_avg4(raw[h]);
      float* d = &p_s[st][lc][lp + 32 * h];
      d[0] = v.x; d[XPITCH] = v.y; d[2 * XPITCH] = v.z; d[3 * XPITCH] = v.w;
    }
#pragma unroll
    for (int v = 0; v < 4; v++) {
      float* d = &w_s[st][lc][lp + 32 * v];
      d[0] = wreg[v].x; d[WPITCH] = wreg[v].y; d[2 * WPITCH] = wreg[v].z; d[3 * WPITCH] = wreg[v].w;
    }
  };
  // compute roles: thread (ty, tx) owns pixels ty*8 .. +7 and channels tx*4 .. +3 and 64 + tx*4 .. +3
  const int ty = tid >> 4, tx = tid & 15;
  unsigned long long acc2[8][4];  // channel pairs of each pixel (packed fp32 FMAs, same rounding as scalar fmaf)
#pragma unroll
  for (int i = 0; i < 8; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) acc2[i][j] = 0ull;
  const int nchunks = C / SC_BK;
  load(0);
  put(0);
  __syncthreads();
#pragma unroll 1
  for (int ch = 0; ch < nchunks; ch++) {
    const int st = ch & 1;
    if (ch + 1 < nchunks) load((ch + 1) * SC_BK);
    const float* pb = &p_s[st][0][ty * 8];
    const float* wb = &w_s[st][0][tx * 4];
#pragma unroll
    for (int cc = 0; cc < SC_BK; cc++) {
      float pv[8];
#pragma unroll
      for (int i = 0; i < 8; i += 4) {
        const float4 t = *reinterpret_cast<const float4*>(pb + cc * XPITCH + i);
        pv[i] = t.x; pv[i + 1] = t.y; pv[i + 2] = t.z; pv[i + 3] = t.w;
      }
      unsigned long long w2[4];
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const float4 t = *reinterpret_cast<const float4*>(wb + cc * WPITCH + 64 * h);
        w2[2 * h] = pack_f32x2(t.x, t.y);
        w2[2 * h + 1] = pack_f32x2(t.z, t.w);
      }
#pragma unroll
      for (int j = 0; j < 4; j++)
#pragma unroll
        for (int i = 0; i < 8; i++) fma_f32x2(acc2[i][j], w2[j], pack_f32x2(pv[i], pv[i]));
    }
    asm volatile("" ::: "memory");  // (the pooling stays behind the multiply-adds)
    if (ch + 1 < nchunks) put(st ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int o = o0 + 64 * h + tx * 4;
    float sc[4], sf[4];
#pragma unroll
    for (int j = 0; j < 4; j++) {
      sc[j] = scale[o + j];
      sf[j] = shift[o + j];
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const long long p = p0 + ty * 8 + i;
      if (p >= npix_out) continue;
      float r0, r1, r2, r3;
      unpack_f32x2(acc2[i][2 * h], r0, r1);
      unpack_f32x2(acc2[i][2 * h + 1], r2, r3);
      *reinterpret_cast<float4*>(y + p * O + o) =
          make_float4(__fmaf_rn(r0, sc[0], sf[0]), __fmaf_rn(r1, sc[1], sf[1]), __fmaf_rn(r2, sc[2], sf[2]), __fmaf_rn(r3, sc[3], sf[3]));
    }
  }
}

// Fewer: 32 pixels x 64 channels per CTA with all of K in shared memory, so that it waits for memory once: the weights as
// asynchronous copies in the order they have in global memory, the inputs in batches of 16 loads.  128 threads of 4 pixels x 4
// channels; accumulators are pairs of pixels, a weight both halves of the other factor.  Batch 8, stages 2 to 4: 9.6, 11.0 and
// 11.6 us, against 11.3 with the kernel above and 18.9 and 20.4 with the one below.
constexpr int SW_BM = 32, SW_BN = 64, SW_XP = SW_BM + 4;
constexpr int shortcut_whole_smem(int C) { return (SW_BN * (C + 4) + C * SW_XP) * 4; }
__global__ void __launch_bounds__(128) shortcut_whole(const float* x, int HW, int C, const float* __restrict__ w, int O,
                                                      const float* __restrict__ scale, const float* __restrict__ shift,
                                                      long long npix_out, float* y) {
  extern __shared__ __align__(16) float sm[];
  const int wp = C + 4, tid = threadIdx.x, o0 = blockIdx.y * SW_BN;
  float* w_s = sm;                // [64][C + 4]
  float* x_s = sm + SW_BN * wp;   // [C][36]
  const bool w_vec = (reinterpret_cast<uintptr_t>(w) & 15) == 0;
  for (int t = tid; t < SW_BN * C / 4; t += 128) {
    const int row = t / (C / 4), q = t - row * (C / 4);
    const float* src = w + (size_t)(o0 + row) * C + 4 * q;
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(w_s + row * wp + 4 * q);
    if (w_vec) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    } else {
#pragma unroll
      for (int e = 0; e < 4; e++) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4 * e), "l"(src + e) : "memory");
    }
  }
  chain_wait();  // (the weights above do not depend on the previous kernel)
  const int lq = (tid & 7) * 4, lp = tid >> 3;
  const float* src[2];
#pragma unroll
  for (int h = 0; h < 2; h++) {
    src[h] = pool_source(x, (long long)blockIdx.x * SW_BM + lp + 16 * h, npix_out, HW, C);
    if (src[h] != nullptr) src[h] += lq;
  }
#pragma unroll 1
  for (int c = 0; c < C; c += 64) {
    float4 raw[4][4];
#pragma unroll
    for (int q = 0; q < 4; q++) pool_load(raw[q], src[q & 1] != nullptr ? src[q & 1] + c + 32 * (q >> 1) : nullptr, HW, C);
#pragma unroll
    for (int q = 0; q < 4; q++) pool_hold(raw[q]);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const float4 v = pool_avg4(raw[q]);
      float* d = x_s + (c + 32 * (q >> 1) + lq) * SW_XP + lp + 16 * (q & 1);
      d[0] = v.x; d[SW_XP] = v.y; d[2 * SW_XP] = v.z; d[3 * SW_XP] = v.w;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  chain_trigger();
  const int ty = tid >> 4, tx = tid & 15;
  const float* xs = x_s + ty * 4;
  const float* ws = w_s + tx * wp;
  unsigned long long acc2[2][4];  // pixels 2i, 2i + 1 of the thread's four, channel tx + 16 * j
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) acc2[i][j] = 0ull;
#pragma unroll 8
  for (int c = 0; c < C; c += 4) {
    float4 w4[4];
#pragma unroll
    for (int j = 0; j < 4; j++) w4[j] = *reinterpret_cast<const float4*>(ws + j * 16 * wp + c);
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const float4 t = *reinterpret_cast<const float4*>(xs + (c + u) * SW_XP);
      const unsigned long long x2[2] = {pack_f32x2(t.x, t.y), pack_f32x2(t.z, t.w)};
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const float wv = u == 0 ? w4[j].x : u == 1 ? w4[j].y : u == 2 ? w4[j].z : w4[j].w;
        fma_f32x2(acc2[0][j], x2[0], pack_f32x2(wv, wv));
        fma_f32x2(acc2[1][j], x2[1], pack_f32x2(wv, wv));
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 4; j++) {
    const int o = o0 + tx + 16 * j;
    const float sc = scale[o], sf = shift[o];
#pragma unroll
    for (int i = 0; i < 2; i++) {
      const long long p = (long long)blockIdx.x * SW_BM + ty * 4 + 2 * i;
      float v0, v1;
      unpack_f32x2(acc2[i][j], v0, v1);
      if (p < npix_out) y[p * O + o] = __fmaf_rn(v0, sc, sf);
      if (p + 1 < npix_out) y[(p + 1) * O + o] = __fmaf_rn(v1, sc, sf);
    }
  }
}

// The same for a few images, with every global load issued before the first fmaf: a tile is 16 output pixels x 16
// channels; its 16 weight rows and the pooled inputs of its 16 pixels go through shared memory (coalesced float4 loads,
// all in flight at once), then each thread runs the fmaf chain(s) of its output(s) over c ascending.  C <= 256, C % 4 == 0.
// `sm` holds 2 x 16 x SC16_PITCH floats.  CHAINED: hooks of a kernel launched by launch_chain (see common.cuh).
constexpr int SC16_PITCH = 260;  // floats per row: 16 rows, read as float4, fall on distinct banks
template <int THREADS, bool CHAINED>
__device__ __forceinline__ void shortcut_tile16(const float* x, int HW, int C, const float* __restrict__ w, int O,
                                                const float* __restrict__ scale, const float* __restrict__ shift,
                                                long long npix_out, float* y, const long long bx, const int by, float* sm) {
  constexpr int NOUT = 256 / THREADS;  // outputs per thread, 128 apart in the tile
  float(*pooled)[SC16_PITCH] = reinterpret_cast<float(*)[SC16_PITCH]>(sm);
  float(*ws)[SC16_PITCH] = reinterpret_cast<float(*)[SC16_PITCH]>(sm + 16 * SC16_PITCH);
  const int tid = threadIdx.x;
  const long long p0 = bx * 16;
  const int o0 = by * 16;
  const int OHW = HW / 2, C4 = C / 4;
#pragma unroll 4
  for (int t = tid; t < 16 * C4; t += THREADS) {
    const int row = t / C4, q = t - row * C4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (o0 + row < O) v = __ldg(reinterpret_cast<const float4*>(w + (size_t)(o0 + row) * C) + q);
    *reinterpret_cast<float4*>(&ws[row][4 * q]) = v;
  }
  if (CHAINED) chain_wait();  // (the weights above do not depend on the previous kernel)
#pragma unroll 4
  for (int t = tid; t < 16 * C4; t += THREADS) {
    const int pp = t / C4, q = t - pp * C4;
    const long long p = p0 + pp;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p < npix_out) {
      const int ow = (int)(p % OHW), oh = (int)((p / OHW) % OHW);
      const long long n = p / ((long long)OHW * OHW);
      const float* src = x + ((n * HW + 2 * oh) * HW + 2 * ow) * C + 4 * q;
      const float4 a = *reinterpret_cast<const float4*>(src);
      const float4 b = *reinterpret_cast<const float4*>(src + C);
      const float4 c = *reinterpret_cast<const float4*>(src + (size_t)HW * C);
      const float4 d = *reinterpret_cast<const float4*>(src + (size_t)HW * C + C);
      v.x = __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(a.x, b.x), c.x), d.x), 0.25f);
      v.y = __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(a.y, b.y), c.y), d.y), 0.25f);
      v.z = __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(a.z, b.z), c.z), d.z), 0.25f);
      v.w = __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(a.w, b.w), c.w), d.w), 0.25f);
    }
    *reinterpret_cast<float4*>(&pooled[pp][4 * q]) = v;
  }
  __syncthreads();
  if (CHAINED) chain_trigger();
  const int oo = tid & 15, o = o0 + oo;
  float a[NOUT];
#pragma unroll
  for (int u = 0; u < NOUT; u++) a[u] = 0.0f;
#pragma unroll 4
  for (int c = 0; c < C; c += 4) {
    const float4 wv = *reinterpret_cast<const float4*>(&ws[oo][c]);
#pragma unroll
    for (int u = 0; u < NOUT; u++) {
      const float4 pv = *reinterpret_cast<const float4*>(&pooled[(tid >> 4) + u * (THREADS / 16)][c]);
      a[u] = __fmaf_rn(pv.x, wv.x, a[u]);
      a[u] = __fmaf_rn(pv.y, wv.y, a[u]);
      a[u] = __fmaf_rn(pv.z, wv.z, a[u]);
      a[u] = __fmaf_rn(pv.w, wv.w, a[u]);
    }
  }
  if (o < O) {
    const float sc = scale[o], sf = shift[o];
#pragma unroll
    for (int u = 0; u < NOUT; u++) {
      const long long p = p0 + (tid >> 4) + u * (THREADS / 16);
      if (p < npix_out) y[p * O + o] = __fmaf_rn(a[u], sc, sf);
    }
  }
}
__global__ void __launch_bounds__(256) shortcut_down_tile16(const float* x, int HW, int C, const float* __restrict__ w, int O,
                                                            const float* __restrict__ scale, const float* __restrict__ shift,
                                                            long long npix_out, float* y) {
  __shared__ __align__(16) float sm[2 * 16 * SC16_PITCH];
  shortcut_tile16<256, true>(x, HW, C, w, O, scale, shift, npix_out, y, blockIdx.x, blockIdx.y, sm);
}

// ---- head: global average over 7x7 (sequential sum over (h, w), then /49) into the workspace, then fc 512 -> 1000 as
// one fmaf chain per logit over k ascending, then + bias.  Three forms of the fc, by batch size, below.
__global__ void __launch_bounds__(512) gap_small(const float* x /*[N][7][7][512]*/, float* g) {
  const int n = blockIdx.x, c = threadIdx.x;
  chain_trigger();
  chain_wait();
  float s = 0.0f;
  for (int q = 0; q < 49; q++) s = __fadd_rn(s, x[((size_t)n * 49 + q) * 512 + c]);
  g[(size_t)n * 512 + c] = __fdiv_rn(s, 49.0f);
}
// One to four images: pooling and fc in one launch.  A 512-thread CTA takes 8 logits of one image: it pools the image's
// 7x7x512 map itself (thread c owns channel c; same sum order and division as gap_small) while its 8 weight rows are in
// flight, then 8 threads run the 8 fmaf chains out of shared memory.
__global__ void __launch_bounds__(512) head_small(const float* x /*[N][7][7][512]*/,
                                                  const float* __restrict__ fw, const float* __restrict__ fb,
                                                  float* __restrict__ logits) {
  constexpr int PITCH = 516;
  __shared__ __align__(16) float gs[512];
  __shared__ __align__(16) float ws[8][PITCH];
  const int n = blockIdx.y, tid = threadIdx.x, j0 = blockIdx.x * 8;
  float4 wv[2];
#pragma unroll
  for (int u = 0; u < 2; u++) {
    const int idx = tid + 512 * u, row = idx >> 7, q = idx & 127;
    wv[u] = (j0 + row < 1000) ? __ldg(reinterpret_cast<const float4*>(fw + (size_t)(j0 + row) * 512) + q)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  chain_wait();  // (chained launches: the weight rows above do not depend on the previous kernel)
  float s = 0.0f;
#pragma unroll 7
  for (int q = 0; q < 49; q++) s = __fadd_rn(s, x[((size_t)n * 49 + q) * 512 + tid]);
  gs[tid] = __fdiv_rn(s, 49.0f);
#pragma unroll
  for (int u = 0; u < 2; u++) {
    const int idx = tid + 512 * u, row = idx >> 7, q = idx & 127;
    *reinterpret_cast<float4*>(&ws[row][4 * q]) = wv[u];
  }
  __syncthreads();
  const int j = j0 + tid;
  if (tid >= 8 || j >= 1000) return;
  float a = 0.0f;
#pragma unroll 8
  for (int k = 0; k < 512; k += 4) {
    const float4 w4 = *reinterpret_cast<const float4*>(&ws[tid][k]);
    const float4 g4 = *reinterpret_cast<const float4*>(&gs[k]);
    a = __fmaf_rn(g4.x, w4.x, a);
    a = __fmaf_rn(g4.y, w4.y, a);
    a = __fmaf_rn(g4.z, w4.z, a);
    a = __fmaf_rn(g4.w, w4.w, a);
  }
  logits[(size_t)n * 1000 + j] = __fadd_rn(a, fb[j]);
}

// Five to 63 images: pooled vectors come from gap_small; a 64-thread CTA takes 8 logits of up to 8 images.  Its 8 weight
// rows and the images' pooled vectors are staged in shared memory by coalesced loads, all in flight at once; thread
// (image, logit) then runs its fmaf chain over k ascending.
__global__ void __launch_bounds__(64) fc_mid(const float* g /*[N][512]*/, int N, const float* __restrict__ fw,
                                             const float* __restrict__ fb, float* __restrict__ logits) {
  constexpr int PITCH = 516;
  __shared__ __align__(16) float gs[8][PITCH];
  __shared__ __align__(16) float ws[8][PITCH];
  const int tid = threadIdx.x, j0 = blockIdx.x * 8, n0 = blockIdx.y * 8;
  float4 wv[16], gv[16];
#pragma unroll
  for (int u = 0; u < 16; u++) {  // 8 rows x 128 float4 each
    const int idx = tid + 64 * u, row = idx >> 7, q = idx & 127;
    wv[u] = (j0 + row < 1000) ? __ldg(reinterpret_cast<const float4*>(fw + (size_t)(j0 + row) * 512) + q)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  chain_wait();  // (chained launches: the weight rows above do not depend on the previous kernel)
#pragma unroll
  for (int u = 0; u < 16; u++) {
    const int idx = tid + 64 * u, row = idx >> 7, q = idx & 127;
    gv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n0 + row < N) gv[u] = ld_nc_f4(g + (size_t)(n0 + row) * 512 + 4 * q);
  }
#pragma unroll
  for (int u = 0; u < 16; u++) {
    const int idx = tid + 64 * u, row = idx >> 7, q = idx & 127;
    *reinterpret_cast<float4*>(&ws[row][4 * q]) = wv[u];
    *reinterpret_cast<float4*>(&gs[row][4 * q]) = gv[u];
  }
  __syncthreads();
  const int jj = tid & 7, im = tid >> 3, j = j0 + jj, n = n0 + im;
  float a = 0.0f;
#pragma unroll 8
  for (int k = 0; k < 512; k += 4) {
    const float4 w4 = *reinterpret_cast<const float4*>(&ws[jj][k]);
    const float4 g4 = *reinterpret_cast<const float4*>(&gs[im][k]);
    a = __fmaf_rn(g4.x, w4.x, a);
    a = __fmaf_rn(g4.y, w4.y, a);
    a = __fmaf_rn(g4.z, w4.z, a);
    a = __fmaf_rn(g4.w, w4.w, a);
  }
  if (j < 1000 && n < N) logits[(size_t)n * 1000 + j] = __fadd_rn(a, fb[j]);
}

// Larger batches: pooled vectors come from gap_small; a 64-thread CTA computes 64 logits for 8 images, so every weight
// it loads is used 8 times and there are 16 x N/8 CTAs.  The weight rows of the 64 logits pass through shared memory in
// chunks of 32 inputs (coalesced 128-byte pieces of each row in, conflict-free columns out), the next chunk in flight
// while the current one is multiplied.  Each logit is still one fmaf chain over the inputs in ascending order.
__global__ void __launch_bounds__(64) fc_batched(const float* __restrict__ g /*[N][512]*/, int N, const float* __restrict__ fw,
                                                 const float* __restrict__ fb, float* __restrict__ logits) {
  __shared__ __align__(16) float gs[8][512];
  __shared__ __align__(16) float ws[64][36];  // (pitch 36: 128-bit rows in and 128-bit columns out, both free of bank conflicts)
  const int tid = threadIdx.x;
  const int n0 = blockIdx.y * 8, nimg = min(8, N - n0);
  for (int t = tid; t < 8 * 128; t += 64) {
    const int im = t / 128;
    reinterpret_cast<float4*>(&gs[0][0])[t] =
        im < nimg ? reinterpret_cast<const float4*>(g + (size_t)n0 * 512)[t] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const int j0 = blockIdx.x * 64, j = j0 + tid;
  float4 wreg[8];
  auto w_load = [&](int k0) {  // 64 rows x 32 inputs: piece u of this thread is row (tid + 64u) / 8, float4 (tid + 64u) % 8
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int idx = tid + 64 * u, row = idx >> 3, q = idx & 7;
      wreg[u] = (j0 + row < 1000) ? __ldg(reinterpret_cast<const float4*>(fw + (size_t)(j0 + row) * 512 + k0) + q)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto w_store = [&]() {
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int idx = tid + 64 * u, row = idx >> 3, q = idx & 7;
      *reinterpret_cast<float4*>(&ws[row][4 * q]) = wreg[u];
    }
  };
  float a[8];
#pragma unroll
  for (int im = 0; im < 8; im++) a[im] = 0.0f;
  w_load(0);
  for (int k0 = 0; k0 < 512; k0 += 32) {
    __syncthreads();  // the previous chunk has been read (and, the first time, gs is complete)
    w_store();
    __syncthreads();
    if (k0 + 32 < 512) w_load(k0 + 32);
#pragma unroll 2
    for (int kk = 0; kk < 32; kk += 4) {  // four inputs per 128-bit load; each chain still takes them in ascending order
      const float4 wv = *reinterpret_cast<const float4*>(&ws[tid][kk]);
#pragma unroll
      for (int im = 0; im < 8; im++) {
        const float4 gv = *reinterpret_cast<const float4*>(&gs[im][k0 + kk]);
        a[im] = __fmaf_rn(gv.x, wv.x, a[im]);
        a[im] = __fmaf_rn(gv.y, wv.y, a[im]);
        a[im] = __fmaf_rn(gv.z, wv.z, a[im]);
        a[im] = __fmaf_rn(gv.w, wv.w, a[im]);
      }
    }
  }
  if (j >= 1000) return;
  const float bias = fb[j];
#pragma unroll
  for (int im = 0; im < 8; im++)
    if (im < nimg) logits[(size_t)(n0 + im) * 1000 + j] = __fadd_rn(a[im], bias);
}

constexpr int kStageC[4] = {64, 128, 256, 512};
constexpr int kStageHW[4] = {56, 28, 14, 7};

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct Workspace {
  size_t stem_out, res_a, res_b, bits_a, bits_b, gap, total;
};

// Up to this many images the 7x7 stem may run as two kernels with the 112x112x64 tensor between them in the workspace; from there on
// it is always the fused one, and that space holds no more than the STEM module's two tensors.
constexpr int kTwoKernelStemImages = 3;
constexpr size_t kStemBytes = (size_t)112 * 112 * 64 * 4, kModuleBytes = (size_t)(112 * 112 * 16 + 56 * 56 * 64) * 4;

Workspace plan(int N) {
  Workspace ws;
  size_t off = 0;
  // (the larger of both, so that a workspace for N images also does for fewer)
  const size_t two_kernels = (N < kTwoKernelStemImages ? N : kTwoKernelStemImages) * kStemBytes, module = N * kModuleBytes;
  ws.stem_out = off; off = align_up(off + (two_kernels > module ? two_kernels : module), 256);
  ws.res_a = off;    off = align_up(off + (size_t)N * 56 * 56 * 64 * 4, 256);
  ws.res_b = off;    off = align_up(off + (size_t)N * 28 * 28 * 128 * 4, 256);
  ws.bits_a = off;   off = align_up(off + (size_t)N * 56 * 56 * 8, 256);
  ws.bits_b = off;   off = align_up(off + (size_t)N * 56 * 56 * 8, 256);
  ws.gap = off;      off = align_up(off + (size_t)N * 512 * 4, 256);
  ws.total = off;
  return ws;
}

template <int CPT>
dabnn_status launch_stem_pool(const dabnn_bireal18_params* p, const float* images, int N, float* y, uint64_t* bits, cudaStream_t st) {
  constexpr int SMEM = stem_pool_smem<CPT>();
  static bool configured[kMaxDevices] = {};
  const int dev = current_device();
  if (dev < 0) return DABNN_ERR_CUDA;
  if (!configured[dev]) {
    if (cudaFuncSetAttribute(stem_pool<CPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM) != cudaSuccess) {
      cudaGetLastError();
      return DABNN_ERR_CUDA;
    }
    configured[dev] = true;
  }
  constexpr int PARTS = 8 / CPT;  // CTAs that share a unit's 64 channels
  const long long units = (long long)N * 56, cap = sm_count() / PARTS;
  const dim3 grid((unsigned)(units < cap ? units : cap), PARTS);
  uint32_t* bits32 = reinterpret_cast<uint32_t*>(bits);
  // (64 channels per CTA: an ordinary launch; with the wait in the kernel its loop comes out 10 us slower at batch 128, whose
  // forward has 1.5 us to gain)
  if (CPT == 4) launch_next(stem_pool<CPT>, grid, dim3(256), (size_t)SMEM, st, images, p->stem_w, p->stem_scale, p->stem_shift, N, y, bits32);
  else stem_pool<CPT><<<grid, 256, SMEM, st>>>(images, p->stem_w, p->stem_scale, p->stem_shift, N, y, bits32);
  return launch_status();
}

template <int TS, int PPT, int CPT>
dabnn_status launch_stem(const dabnn_bireal18_params* p, const float* images, int N, float* out, cudaStream_t st) {
  constexpr int PS = 2 * TS + 5, HALF = stem_half(PS);
  constexpr size_t SMEM = (size_t)(2 * STEM_K * 4 * CPT + 2 * 3 * PS * 2 * HALF) * 4;
  auto kern = stem_conv_bn<TS, PPT, CPT>;
  static bool configured[kMaxDevices] = {};
  const int dev = current_device();
  if (dev < 0) return DABNN_ERR_CUDA;
  if (!configured[dev]) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM) != cudaSuccess) {
      cudaGetLastError();
      return DABNN_ERR_CUDA;
    }
    configured[dev] = true;
  }
  const int tiles = (112 + TS - 1) / TS;
  const long long ntiles = (long long)N * tiles * tiles;
  const long long cap = 2LL * sm_count();  // persistent: two CTAs per SM, each walking over tiles
  launch_next(kern, dim3((unsigned)(ntiles < cap ? ntiles : cap), 16 / CPT), dim3((TS * TS / PPT) * 4), SMEM, st, images, p->stem_w,
              p->stem_scale, p->stem_shift, N, out);  // head of a chain
  return launch_status();
}

}  // namespace

}  // namespace dabnn

using namespace dabnn;

extern "C" dabnn_status dabnn_bn_fold(const float* gamma, const float* beta, const float* mean, const float* var,
                                      double eps, int O, float* scale, float* shift, void* stream) {
  if (!gamma || !beta || !mean || !var || !scale || !shift) return DABNN_ERR_NULL;
  if (O <= 0 || !(eps >= 0.0)) return DABNN_ERR_SHAPE;
  bn_fold_kernel<<<ceil_div(O, 128), 128, 0, as_stream(stream)>>>(gamma, beta, mean, var, eps, O, scale, shift);
  return launch_status();
}

extern "C" size_t dabnn_bireal18_workspace_bytes(int N) { return N <= 0 ? 0 : plan(N).total; }

// The kernel of a shortcut by its number of outputs.
static dabnn_status launch_shortcut(const float* x, int HW, int C, const float* w, int O, const float* scale, const float* shift,
                                    long long npo, float* y, cudaStream_t st) {
  const long long sms = sm_count();
  const long long ctas = (long long)ceil_div(npo, SW_BM) * (O / SW_BN);
  // 16 x 16 outputs per CTA for a launch of few of them (one image, stages 2 to 4: 6.8, 7.1 and 9.0 us, 6.6, 8.8 and 11.2 with
  // all of K at once, but its start cannot move forward as far: forward 100.0 and 100.4 us); all of K at once as long as its CTAs are resident together (256 channels: two per SM) or nearly so (32 images, stage 4:
  // 23.4 and 22.5 us; 16 images, stage 2: 15.2 and 13.5).
  if ((long long)ceil_div(npo, 16) * (O / 16) <= 3 * sms && aligned(w, 16)) {
    launch_chain(shortcut_down_tile16, dim3(ceil_div(npo, 16), ceil_div(O, 16)), dim3(256), (size_t)0, st, x, HW, C, w, O, scale, shift, npo, y);
  } else if (ctas <= (C <= 128 ? 4 : 2) * sms) {
    static bool configured[kMaxDevices] = {};
    const int dev = current_device();
    if (dev < 0) return DABNN_ERR_CUDA;
    if (!configured[dev]) {
      if (cudaFuncSetAttribute(shortcut_whole, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448) != cudaSuccess) {
        cudaGetLastError();
        return DABNN_ERR_CUDA;
      }
      configured[dev] = true;
    }
    // (shared memory for as many CTAs per SM as an even deal gives and no more: chained, they come in while the block before them
    // still holds some of the SMs, and would settle on the others.  Forward of 8 images 223 -> 212 us, 215 with ordinary launches)
    const int even = (int)(233472 / ((ctas + sms - 1) / sms) - 1024) / 128 * 128, need = shortcut_whole_smem(C);
    const int smem = ctas <= sms || even <= need ? need : even;
    launch_chain(shortcut_whole, dim3(ceil_div(npo, SW_BM), O / SW_BN), dim3(128), (size_t)smem, st, x, HW, C, w, O, scale, shift, npo, y);
  } else {
    shortcut_down<<<dim3(ceil_div(npo, SC_BM), O / SC_BN), 128, 0, st>>>(x, HW, C, w, O, scale, shift, npo, y);
  }
  return launch_status();
}

// sm == nullptr: the 7x7 stem and the max-pool; else the STEM module in their place.
static dabnn_status forward_impl(const dabnn_bireal18_params* p, const dabnn_stem_module_params* sm, const float* images,
                                 int N, float* logits, void* workspace, size_t workspace_bytes, void* stream) {
  if (!p || !images || !logits || !workspace) return DABNN_ERR_NULL;
  if (N <= 0 || N > 65535) return DABNN_ERR_SHAPE;
  if ((!sm && (!p->stem_w || !p->stem_scale || !p->stem_shift)) || !p->fc_w || !p->fc_b) return DABNN_ERR_NULL;
  for (int b = 0; b < 16; b++)
    if (!p->block_w[b] || !p->block_scale[b] || !p->block_shift[b]) return DABNN_ERR_NULL;
  for (int d = 0; d < 3; d++)
    if (!p->down_w[d] || !p->down_scale[d] || !p->down_shift[d]) return DABNN_ERR_NULL;
  if (!aligned(workspace, 256) || !aligned(images, 4) || !aligned(logits, 4) || !aligned(p->fc_w, 16))
    return DABNN_ERR_ALIGNMENT;
  const Workspace ws = plan(N);
  if (workspace_bytes < ws.total) return DABNN_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  // The launches are chained: each kernel that takes part may start its set-up while its predecessor finishes (see
  // launch_chain; DABNN_NO_CHAIN=1 in the environment keeps the ordinary stream order, for measurements).  For one to four
  // images that is a chain of 22 launches shorter than a launch takes; for large batches it hides the start-up of the
  // persistent tensor-engine kernels (tensor memory, barriers, 144 KB of weights per CTA) under the previous kernel's tail.
  const bool chain_off = !chain_enabled();
  struct ChainScope {
    explicit ChainScope(bool on) { g_chain_launch = on; }
    ~ChainScope() { g_chain_launch = false; }
  } chain_scope(!chain_off);
  char* base = static_cast<char*>(workspace);
  float* stem_out = reinterpret_cast<float*>(base + ws.stem_out);
  float* cur = reinterpret_cast<float*>(base + ws.res_a);
  float* other = reinterpret_cast<float*>(base + ws.res_b);
  uint64_t* bits_in = reinterpret_cast<uint64_t*>(base + ws.bits_a);
  uint64_t* bits_out = reinterpret_cast<uint64_t*>(base + ws.bits_b);

  dabnn_status s;
  if (sm) {
    // the stem output area holds the module's two scratch tensors: a1 and the concatenation
    float* a1 = stem_out;
    float* cat = a1 + (size_t)N * 112 * 112 * 16;
    if ((s = launch_stem_module(sm, images, N, a1, cat, cur, bits_in, st)) != DABNN_OK) return s;
  } else {
    // The fused stem sweeps whole rows, N * 56 of them, and each CTA computes one convolution row twice.  From 1.5 rows per SM
    // on that costs less than the max-pool's launch and the tensor between the two kernels (forward of 3 images 147 us apart,
    // 150 fused; 4: 167 and 166); below 7 rows per SM two CTAs share a row's channels, so that ranges differ by half a row at
    // most (16 images: 298 us with 64 channels per CTA, 295 with 32; 20: 324 and 325; 128: 1133 and 1169, with two kernels 1298).
    const long long rows = (long long)N * 56, sms_here = sm_count();
    if (N > kTwoKernelStemImages || 2 * rows >= 3 * sms_here) {  // (148 SMs: the same bound)
      s = rows >= 7 * sms_here ? launch_stem_pool<8>(p, images, N, cur, bits_in, st) : launch_stem_pool<4>(p, images, N, cur, bits_in, st);
      if (s != DABNN_OK) return s;
    } else {
      s = N == 1 ? launch_stem<8, 2, 8>(p, images, N, stem_out, st)  // one image: 392 half-tile CTAs
                 : launch_stem<8, 2, 16>(p, images, N, stem_out, st);
      if (s != DABNN_OK) return s;
      const long long npix = (long long)N * 56 * 56;
      launch_chain(maxpool_pack, dim3(ceil_div(npix * 16, 256)), dim3(256), (size_t)0, st, stem_out, npix, cur, bits_in);
      if ((s = launch_status()) != DABNN_OK) return s;
    }
  }
  // consecutive tensor-engine blocks are chained (DABNN_NO_CHAIN=1 keeps the ordinary stream order)
  const bool tc_chain = !chain_off;
  const int sms = sm_count();
  int C = 64, HW = 56;
  for (int b = 0; b < 16; b++) {
    const int stage = b / 4, O = kStageC[stage], OHW = kStageHW[stage];
    const bool down = stage > 0 && b % 4 == 0;
    if (down) {
      const long long npo = (long long)N * OHW * OHW;
      s = launch_shortcut(cur, HW, C, p->down_w[stage - 1], O, p->down_scale[stage - 1], p->down_shift[stage - 1], npo, other, st);
      if (s != DABNN_OK) return s;
      float* t = cur; cur = other; other = t;
    }
    const dabnn_shape in = {N, C, HW, HW};
    const int stride = down ? 2 : 1;
    const dabnn_conv cv = {3, 3, stride, stride, 1, 1, -1};
    s = DABNN_ERR_UNSUPPORTED;
    // tensor-core engine where it covers the layer and pays; chained launches hide part of its start-up (measured: a credit
    // of 1.5 us against lone launches; batch 8 240 -> 234 us, batch 12 283 -> 269, batch 16 340 -> 322, batch 4 unchanged;
    // with 3 us batch 2 and 4 lose 3 us each)
    if (p->block_w_tc[b] != nullptr)
      s = tc_bireal_block(bits_in, in, p->block_w_tc[b], O, cv, p->block_scale[b], p->block_shift[b], cur, cur,
                          b == 15 ? nullptr : bits_out, tc_chain, int_pipes_us(in, O, cv, 2, false, true, sms) + (tc_chain ? 1.5 : 0.0), sms, st);
    if (s == DABNN_ERR_UNSUPPORTED)
      s = int_pipes_bn_add_sign_pack(bits_in, in, p->block_w[b], O, cv, p->block_scale[b], p->block_shift[b], cur, cur,
                                     b == 15 ? nullptr : bits_out, st);
    if (s != DABNN_OK) return s;
    uint64_t* tb = bits_in; bits_in = bits_out; bits_out = tb;
    C = O; HW = OHW;
  }
  {
    if (N <= 4) {
      launch_chain(head_small, dim3(125, N), dim3(512), (size_t)0, st, cur, p->fc_w, p->fc_b, logits);
      return launch_status();
    }
    float* gbuf = reinterpret_cast<float*>(base + ws.gap);
    if (N < 64) {
      launch_chain(gap_small, dim3(N), dim3(512), (size_t)0, st, cur, gbuf);
      if ((s = launch_status()) != DABNN_OK) return s;
      launch_chain(fc_mid, dim3(125, ceil_div(N, 8)), dim3(64), (size_t)0, st, gbuf, N, p->fc_w, p->fc_b, logits);
    } else {  // (not chained: let in early their CTAs settle unevenly, forward of 128 images 1096 -> 1125 us)
      gap_small<<<N, 512, 0, st>>>(cur, gbuf);
      if ((s = launch_status()) != DABNN_OK) return s;
      fc_batched<<<dim3(ceil_div(1000, 64), ceil_div(N, 8)), 64, 0, st>>>(gbuf, N, p->fc_w, p->fc_b, logits);
    }
  }
  return launch_status();
}

extern "C" dabnn_status dabnn_bireal18_forward(const dabnn_bireal18_params* p, const float* images, int N,
                                               float* logits, void* workspace, size_t workspace_bytes, void* stream) {
  return forward_impl(p, nullptr, images, N, logits, workspace, workspace_bytes, stream);
}

extern "C" dabnn_status dabnn_bireal18_forward_stem_module(const dabnn_bireal18_params* p, const dabnn_stem_module_params* sm,
                                                           const float* images, int N, float* logits, void* workspace,
                                                           size_t workspace_bytes, void* stream) {
  if (!sm) return DABNN_ERR_NULL;
  return forward_impl(p, sm, images, N, logits, workspace, workspace_bytes, stream);
}

// ---- allocation-free variant ---------------------------------------------------------------------------
// Scratch for dabnn_bireal18_forward_static: part of the library image, present on every device that loads
// it.  In host code the symbol below is only a handle; its device address is looked up per device.
static __device__ __align__(256) unsigned char g_static_scratch[DABNN_STATIC_SCRATCH_BYTES];

namespace {
std::mutex g_static_mutex;
void* g_static_addr[kMaxDevices] = {};  // device address of g_static_scratch, per device ordinal
}  // namespace

extern "C" dabnn_status dabnn_bireal18_forward_static(const dabnn_bireal18_params* p, const float* images, int N,
                                                      float* logits, void* stream) {
  if (N > DABNN_STATIC_MAX_BATCH) return DABNN_ERR_STATIC_LIMIT;
  if (N <= 0) return DABNN_ERR_SHAPE;
  if (dabnn_bireal18_workspace_bytes(N) > (size_t)DABNN_STATIC_SCRATCH_BYTES) return DABNN_ERR_STATIC_LIMIT;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return DABNN_ERR_CUDA;
  }
  if (dev < 0 || dev >= kMaxDevices) return DABNN_ERR_UNSUPPORTED;
  void* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_static_mutex);
    scratch = g_static_addr[dev];
    if (scratch == nullptr) {
      // once per device, with that device current: the symbol's address in this device's memory
      if (cudaGetSymbolAddress(&scratch, g_static_scratch) != cudaSuccess || scratch == nullptr) {
        cudaGetLastError();
        return DABNN_ERR_CUDA;
      }
      g_static_addr[dev] = scratch;
    }
  }
  return dabnn_bireal18_forward(p, images, N, logits, scratch, (size_t)DABNN_STATIC_SCRATCH_BYTES, stream);
}
