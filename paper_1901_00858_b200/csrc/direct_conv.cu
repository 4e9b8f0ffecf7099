// Direct convolution on CUDA cores: the path for any valid layer (and the fallback of the
// planner for shapes the specialised kernels do not take).  NCHW in, NCHW out, fp32
// accumulation, fused bias + ReLU + one round-to-nearest-even conversion to binary16.
//
// Work split: one thread per output pixel, KT output channels of one group per CTA row, so a
// loaded input value feeds KT FMAs.  The CTA's KT weight rows are staged in shared memory in
// chunks of the flattened (c', r, s) tap index; every thread walks the chunk with running
// (c', r, s) counters.
#include "hgc_internal.h"

namespace hgc {
HGC_DEBUG_STATE(direct)
namespace {

constexpr int kThreads = 128;
constexpr int kChunk = 512;  // taps staged per pass

template <int KT>
__global__ void __launch_bounds__(kThreads)
direct_conv_kernel(ConvGeom g, const __half* __restrict__ x, const __half* __restrict__ w,
                   const __half* __restrict__ bias, __half* __restrict__ y, int relu) {
  grid_dependency_wait();
  __shared__ float ws[KT][kChunk];

  // blockIdx.x = (n * ktiles + ktile) * px_tiles + px_tile
  const int ktiles_per_group = (g.kg + KT - 1) / KT;
  const int ktiles = g.group * ktiles_per_group;
  const int64_t pq = (int64_t)g.p * g.q;
  const unsigned px_tiles = (unsigned)((pq + kThreads - 1) / kThreads);
  const unsigned px_tile = blockIdx.x % px_tiles;
  const unsigned nk = blockIdx.x / px_tiles;
  const int ktile = (int)(nk % (unsigned)ktiles);
  const int n = (int)(nk / (unsigned)ktiles);
  const int grp = ktile / ktiles_per_group;
  const int k_in_grp0 = (ktile % ktiles_per_group) * KT;
  const int64_t pix = (int64_t)px_tile * kThreads + threadIdx.x;
  const bool live = pix < pq;
  const int op = live ? (int)(pix / g.q) : 0;
  const int oq = live ? (int)(pix % g.q) : 0;
  const int ih0 = op * g.stride_h - g.pad_h;
  const int iw0 = oq * g.stride_w - g.pad_w;
  const int rs = g.r * g.s;
  const int64_t taps = (int64_t)g.cg * rs;
  const int64_t plane = (int64_t)g.h * g.w;
  const __half* xg = x + ((int64_t)n * g.c + (int64_t)grp * g.cg) * plane;

  float acc[KT];
#pragma unroll
  for (int i = 0; i < KT; ++i) acc[i] = 0.f;

  for (int64_t t0 = 0; t0 < taps; t0 += kChunk) {
    const int len = (int)((taps - t0) < kChunk ? (taps - t0) : kChunk);
    __syncthreads();
    for (int i = threadIdx.x; i < KT * len; i += kThreads) {
      const int kk = i / len, t = i % len;
      const int kin = k_in_grp0 + kk;
      float v = 0.f;
      if (kin < g.kg) v = __half2float(w[((int64_t)grp * g.kg + kin) * taps + t0 + t]);
      ws[kk][t] = v;
    }
    __syncthreads();
    if (live) {
      int cc = (int)(t0 / rs);
      int rem = (int)(t0 % rs);
      int r = rem / g.s, s = rem % g.s;
      for (int t = 0; t < len; ++t) {
        const int ih = ih0 + r * g.dil_h;
        const int iw = iw0 + s * g.dil_w;
        if (ih >= 0 && ih < g.h && iw >= 0 && iw < g.w) {
          float xv = 0.f;
          if (HGC_ADDR_OK(xg + (int64_t)cc * plane + (int64_t)ih * g.w + iw, sizeof(__half)))
            xv = __half2float(__ldg(xg + (int64_t)cc * plane + (int64_t)ih * g.w + iw));
#pragma unroll
          for (int i = 0; i < KT; ++i) acc[i] = fmaf(xv, ws[i][t], acc[i]);
        }
        if (++s == g.s) {
          s = 0;
          if (++r == g.r) {
            r = 0;
            ++cc;
          }
        }
      }
    }
  }

  if (live) {
#pragma unroll
    for (int i = 0; i < KT; ++i) {
      const int kin = k_in_grp0 + i;
      if (kin < g.kg) {
        const int k = grp * g.kg + kin;
        float v = acc[i];
        if (bias != nullptr) v += __half2float(bias[k]);
        if (relu) v = fmaxf(v, 0.f);
        if (HGC_ADDR_OK(y + ((int64_t)n * g.k + k) * pq + pix, sizeof(__half))) y[((int64_t)n * g.k + k) * pq + pix] = __float2half_rn(v);
      }
    }
  }
}

// Image stems (at most 8 channels, one group) of little work.  The tensor-core path takes two launches for them,
// a bordered or expanded copy of x and the layer, and such a layer is over sooner than the host can issue the
// second one.  Here it is one: a block brings the input rows under 128 consecutive output pixels of an image
// into shared memory with their zero border, 8 channels' weights and the taps' offsets, all loads
// under way together; a thread then sums its pixel's taps for the 8 channels with the mixed-precision FMA
// (products of binary16 values are exact, FP32 sums in the order of the taps).  One trip to memory and one barrier:
// 3->16 channels, 3x3 on 32x32, one image, 6.5 -> 4.0 us a call.
constexpr int kStemThreads = 128, kStemK = 8;

struct StemTile {  // of a block, for any of its positions
  int64_t taps, in_w, rows;  // taps per output; columns and (at most) rows of the input tile
  size_t bytes;
};
StemTile stem_tile(const ConvGeom& g) {
  StemTile t;
  t.taps = (int64_t)g.c * g.r * g.s;
  t.in_w = (int64_t)(g.q - 1) * g.stride_w + (int64_t)(g.s - 1) * g.dil_w + 1;
  const int64_t spans = (kStemThreads - 1 + g.q - 1) / g.q;  // output rows that 128 pixels reach beyond their first
  t.rows = (spans < g.p - 1 ? spans : g.p - 1) * g.stride_h + (int64_t)(g.r - 1) * g.dil_h + 1;
  t.bytes = (size_t)t.taps * (kStemK * 2 + 4) + (size_t)(g.c * t.rows * t.in_w) * 2;
  return t;
}

template <bool RELU>
__device__ __forceinline__ uint16_t to_half(float v) {  // (the rounding and ReLU of the tensor-core epilogues: a NaN stays one)
  uint32_t d;
  if (RELU) asm("cvt.rn.relu.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(0.f), "f"(v));
  else asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(0.f), "f"(v));
  return (uint16_t)(d & 0xffffu);
}

template <bool RELU>
__global__ void __launch_bounds__(kStemThreads)
stem_small_kernel(const ConvGeom g, const uint16_t* __restrict__ x, const uint16_t* __restrict__ w, const uint16_t* __restrict__ bias,
                  uint16_t* __restrict__ y, int taps, int in_w) {
  extern __shared__ __align__(16) uint8_t stem_smem[];
  uint16_t* ws = reinterpret_cast<uint16_t*>(stem_smem);          // [tap][8 channels]
  int* offs = reinterpret_cast<int*>(stem_smem + (size_t)taps * kStemK * 2);  // [tap]: from a pixel's first input value
  uint16_t* xs = reinterpret_cast<uint16_t*>(offs + taps);        // [channel][row][in_w]
  const int tid = (int)threadIdx.x;
  const int pq = g.p * g.q;
  const int px0 = (int)blockIdx.x * kStemThreads, k0 = (int)blockIdx.y * kStemK, n = (int)blockIdx.z;
  const int px_last = px0 + kStemThreads - 1 < pq ? px0 + kStemThreads - 1 : pq - 1;
  const int p_first = px0 / g.q;
  const int rows = (px_last / g.q - p_first) * g.stride_h + (g.r - 1) * g.dil_h + 1;
  const int h0 = p_first * g.stride_h - g.pad_h;
  for (int t = tid; t < taps; t += kStemThreads) {
    const int c = t / (g.r * g.s), rs = t - c * g.r * g.s, r = rs / g.s;
    offs[t] = (c * rows + r * g.dil_h) * in_w + (rs - r * g.s) * g.dil_w;
  }
  grid_dependency_wait();
  grid_launch_dependents();
  float b[kStemK];
#pragma unroll
  for (int i = 0; i < kStemK; ++i) {
    b[i] = 0.f;
    if (bias != nullptr && k0 + i < g.k && HGC_ADDR_OK(bias + k0 + i, 2)) b[i] = __half2float(__ushort_as_half(__ldg(bias + k0 + i)));
  }
  // x with its border, then the weights; eight loads of a thread under way at a time
  const int nx = g.c * rows * in_w;
  const uint16_t* xn = x + (int64_t)n * g.c * g.h * g.w;
  for (int i0 = tid; i0 < nx; i0 += 8 * kStemThreads) {
    uint16_t v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int i = i0 + j * kStemThreads;
      v[j] = 0;
      if (i < nx) {
        const int line = i / in_w, c = line / rows;
        const int ih = h0 + line - c * rows, iw = i - line * in_w - g.pad_w;
        if (ih >= 0 && ih < g.h && iw >= 0 && iw < g.w) {
          const uint16_t* src = xn + ((int64_t)c * g.h + ih) * g.w + iw;
          HGC_CHECKED_LOAD(v[j], src, __ldg(src));
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (i0 + j * kStemThreads < nx) xs[i0 + j * kStemThreads] = v[j];
  }
  for (int i = tid; i < taps * kStemK; i += kStemThreads) {
    const int kk = i / taps, t = i - kk * taps;
    uint16_t v = 0;
    if (k0 + kk < g.k) HGC_CHECKED_LOAD(v, w + (int64_t)(k0 + kk) * taps + t, __ldg(w + (int64_t)(k0 + kk) * taps + t));
    ws[t * kStemK + kk] = v;
  }
  __syncthreads();
  const int px = px0 + tid;
  if (px >= pq) return;
  const int op = px / g.q, oq = px - op * g.q;
  const uint16_t* xp = xs + (op - p_first) * g.stride_h * in_w + oq * g.stride_w;
  float acc[kStemK];
#pragma unroll
  for (int i = 0; i < kStemK; ++i) acc[i] = 0.f;
#pragma unroll 8
  for (int t = 0; t < taps; ++t) {
    const uint16_t xv = xp[offs[t]];
    const uint4 wv = *reinterpret_cast<const uint4*>(ws + t * kStemK);
    const uint32_t wp[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint16_t lo, hi;
      asm("mov.b32 {%0, %1}, %2;" : "=h"(lo), "=h"(hi) : "r"(wp[i]));
      asm("fma.rn.f32.f16 %0, %1, %2, %0;" : "+f"(acc[2 * i]) : "h"(xv), "h"(lo));
      asm("fma.rn.f32.f16 %0, %1, %2, %0;" : "+f"(acc[2 * i + 1]) : "h"(xv), "h"(hi));
    }
  }
  uint16_t* yp = y + ((int64_t)n * g.k + k0) * pq + px;
#pragma unroll
  for (int i = 0; i < kStemK; ++i)
    if (k0 + i < g.k) HGC_CHECKED_STORE(yp + (int64_t)i * pq, yp[(int64_t)i * pq] = to_half<RELU>(acc[i] + b[i]));
}

}  // namespace

// Where the one launch is the faster form (us per call as a graph, against the copy and the tensor-core layer):
// an input tile that a thread brings in with one round of eight loads (3->16 3x3 on 32x32 3.6 against 5.7, 3->128
// 3.7 against 6.0, 3->64 on 64x64 4.4 against 6.2, 8 images of 3->64 on 32x32 4.9 against 6.1; with three to five rounds
// 3->32 stride 2 on 112x112 7.5 against 5.5, 8->24 on 40x44 7.4 against 5.4) and few products, which here are
// CUDA-core FMAs (3->64 on 128x128, 28 M products, 9.4 against 6.4).
constexpr int64_t kStemProducts = 8 << 20;
constexpr int64_t kStemLoads = 8 * kStemThreads;

bool stem_small_supported(const ConvGeom& g) {
  if (g.group != 1 || g.c > 8 || g.x_nhwc || g.y_nhwc || g.no_small_stem) return false;
  const int64_t pq = (int64_t)g.p * g.q;
  if ((int64_t)g.c * g.r * g.s > 512 || (int64_t)g.n * pq * g.k * g.c * g.r * g.s > kStemProducts) return false;
  const StemTile t = stem_tile(g);
  return (int64_t)g.c * t.rows * t.in_w <= kStemLoads && t.bytes <= 48 * 1024 && g.n <= 65535 && g.k <= 65535 &&
         (int64_t)g.h * g.w <= 0x7fffffffLL;
}

cudaError_t launch_stem_small(const ConvGeom& g, const __half* x, const __half* w, const __half* bias, __half* y, int relu,
                              cudaStream_t stream) {
  const StemTile t = stem_tile(g);
  const int pq = g.p * g.q;
  const dim3 grid((unsigned)((pq + kStemThreads - 1) / kStemThreads), (unsigned)((g.k + kStemK - 1) / kStemK), (unsigned)g.n);
  const cudaError_t err = launch_kernel_attr(true, 0, relu ? stem_small_kernel<true> : stem_small_kernel<false>, grid, dim3(kStemThreads), t.bytes, stream, g,
                                             reinterpret_cast<const uint16_t*>(x), reinterpret_cast<const uint16_t*>(w),
                                             reinterpret_cast<const uint16_t*>(bias), reinterpret_cast<uint16_t*>(y), (int)t.taps, (int)t.in_w);
  if (err != cudaSuccess) return err;
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_direct_conv(const ConvGeom& g, const __half* x, const __half* w,
                               const __half* bias, __half* y, int relu, cudaStream_t stream) {
  const int64_t pq = (int64_t)g.p * g.q;
  const int64_t px_tiles = (pq + kThreads - 1) / kThreads;
  const int kt = g.kg >= 4 ? 8 : 1;
  const int64_t ktiles = (int64_t)g.group * ((g.kg + kt - 1) / kt);
  const double total = (double)px_tiles * (double)ktiles * (double)g.n;
  if (total > 2147483647.0) return cudaErrorInvalidConfiguration;
  dim3 grid((unsigned)(px_tiles * ktiles * g.n));
  if (kt == 8)
    launch_smem_kernel(direct_conv_kernel<8>, dim3(grid), dim3(kThreads), 0, stream, g, x, w, bias, y, relu);
  else
    launch_smem_kernel(direct_conv_kernel<1>, dim3(grid), dim3(kThreads), 0, stream, g, x, w, bias, y, relu);
  count_launch();
  return cudaGetLastError();
}

}  // namespace hgc
