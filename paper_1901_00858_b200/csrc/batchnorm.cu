// Batch norm forward in the form Section 3.1 of the paper describes for narrow arithmetic:
//   * grouped mean: the N*H*W values of a channel are partitioned into groups (one image, one run
//     of at most 2048 consecutive pixels), the mean of every group is taken separately, then the
//     mean of those means (weighted by the group sizes, which only differ for the last run of a
//     plane);
//   * shifting before squaring: the centred value is multiplied by a power of two (1/32 for data
//     with large values, 32 for data with small values, 1 for neither) before it is squared, and
//     the variance is shifted back by the square of that factor afterwards.
// On this GPU every sum is carried in FP32, so neither step is needed to stay in range: they are
// kept because they cost nothing (a grouped mean is how a parallel reduction is organised anyway,
// and scaling by a power of two is exact), and the result is independent of the shift.
//
//   y = (x - mean_c) / sqrt(var_c + eps),  var_c the biased variance, one rounding to FP16.
//
// Two passes over x, both bound by HBM bandwidth (or L2 for tensors that fit): 6 bytes per element.
// The first holds a group in registers and takes its mean and its mean square about that mean; the
// variance of a channel is the mean of (group square + (group mean - mean)^2), the usual
// decomposition, so the values need not be read again once the mean is known (a pass of its own for
// that made it 8 bytes: 16 x 64 x 224 x 224 79.4 us).  The second pass walks backwards, from what the
// first left in L2, and has its first values under way before it waits for the statistics.
// With stored statistics only the second runs.
// Every reduction has a fixed order: results are deterministic and every block of a channel
// derives bit-identical statistics from the per-group values.
#include "hgc_internal.h"

namespace hgc {
namespace {

constexpr int kBnThreads = 256;
constexpr int kBnWarps = kBnThreads / 32;
constexpr int kBnGroup = 2048;  // elements per group: 64 per lane, eight 16-byte loads

// x * m + acc with one rounding, x and m binary16: the mixed-precision FMA takes x as it is.  (A
// conversion runs at a quarter of the FMA rate; two per value made the first pass instruction bound.)
__device__ __forceinline__ float fma_h(uint16_t x, uint16_t m, float acc) {
  float d;
  asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(d) : "h"(x), "h"(m), "f"(acc));
  return d;
}
constexpr uint16_t kHalfOne = 0x3c00;

// Sum over the L lanes that share a group.
template <int L>
__device__ __forceinline__ float lane_sum(float v) {
#pragma unroll
  for (int off = L / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// A group of at most 64 * L values in the registers of L lanes: the 16-byte vectors that lie inside it
// (up to eight per lane, all loads under way at once) and the up to seven values before the first
// and after the last of them, one per lane.  Planes whose size is not a multiple of 8 start anywhere.
template <int L>
struct Group {
  uint4 q[8];
  uint16_t edge[2];
  int nvec, head, tail;  // vectors; values in front of and behind them
  bool live;
  __device__ __forceinline__ void place(const uint16_t* p, int count, bool exists) {
    live = exists;
    const int off = (int)((reinterpret_cast<uintptr_t>(p) >> 1) & 7u);
    head = (8 - off) & 7;
    if (head > count) head = count;
    nvec = (count - head) >> 3;
    tail = count - head - 8 * nvec;
  }
  template <bool LAST_USE>
  __device__ __forceinline__ void load(const uint16_t* __restrict__ p) {
    const int lane = (int)(threadIdx.x & (L - 1));
    const uint4* pv = reinterpret_cast<const uint4*>(p + head);
    edge[0] = edge[1] = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (live && lane + L * j < nvec) q[j] = LAST_USE ? __ldcs(pv + lane + L * j) : __ldg(pv + lane + L * j);
    if (live && lane < head) edge[0] = __ldg(p + lane);
    if (live && lane < tail) edge[1] = __ldg(p + head + 8 * nvec + lane);
  }
  // f(binary16 bits of a value) over this lane's values
  template <typename F>
  __device__ __forceinline__ void each(F&& f) const {
    const int lane = (int)(threadIdx.x & (L - 1));
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (live && lane + L * j < nvec) {
        const uint32_t w[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint16_t lo, hi;
          asm("mov.b32 {%0, %1}, %2;" : "=h"(lo), "=h"(hi) : "r"(w[i]));
          f(lo);
          f(hi);
        }
      }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (live && lane < (e == 0 ? head : tail)) f(edge[e]);
  }
};

// Sum of v over the block in a fixed order; every thread returns it.  `red` holds kBnWarps floats.
__device__ __forceinline__ float block_sum(float v, float* red) {
  v = lane_sum<32>(v);
  __syncthreads();  // red may still be read from a previous call
  if ((threadIdx.x & 31u) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float total = 0.f;
#pragma unroll
  for (int w = 0; w < kBnWarps; ++w) total += red[w];
  return total;
}

// Pass 1: stats[c][g] = (mean of group g, mean of ((x - that mean) * shift)^2 over it).
template <int L>
__global__ void __launch_bounds__(kBnThreads)
bn_group_kernel(const uint16_t* __restrict__ x, float2* __restrict__ stats, int n_img, int C, int64_t hw, int chunks, float shift) {
  grid_dependency_wait();
  grid_launch_dependents();  // (not before the wait: the second kernel loads x before its own)
  const int c = (int)blockIdx.y;
  const int G = n_img * chunks;
  constexpr int kSlots = kBnThreads / L;  // groups per block and step
  const int slot = (int)threadIdx.x / L;
  const uint16_t shift16 = __half_as_ushort(__float2half_rn(shift));  // (2^-8 .. 2^8: exact)
  for (int g0 = (int)blockIdx.x * kSlots; g0 < G; g0 += (int)gridDim.x * kSlots) {
    const int g = g0 + slot < G ? g0 + slot : G - 1;
    const int img = g / chunks, ch = g - img * chunks;
    const int64_t start = (int64_t)ch * kBnGroup;
    const int count = (int)(hw - start < kBnGroup ? hw - start : kBnGroup);
    const uint16_t* p = x + ((int64_t)img * C + c) * hw + start;
    Group<L> grp;
    grp.place(p, count, g0 + slot < G);
    grp.template load<false>(p);
    float s = 0.f;
    grp.each([&](uint16_t v) { s = fma_h(v, kHalfOne, s); });
    const float mean = lane_sum<L>(s) / (float)count;
    float sq = 0.f;
    const float centre = -mean * shift;
    grp.each([&](uint16_t v) {  // (the shift is a power of two: v * shift - mean * shift is (v - mean) * shift, rounded alike)
      const float d = fma_h(v, shift16, centre);
      sq = fmaf(d, d, sq);
    });
    sq = lane_sum<L>(sq) / (float)count;
    if ((threadIdx.x & (L - 1)) == 0 && grp.live) stats[(int64_t)c * G + g] = make_float2(mean, sq);
  }
}

// Pass 2: statistics of the channel from the per-group values (or the stored ones), then y.  Blocks
// and groups run backwards: the end of x is what pass 1 read last.  The values of the first step are
// loaded before the wait for pass 1: that kernel lets this one start after its own wait, so
// whatever wrote x has completed.
template <int L>
__global__ void __launch_bounds__(kBnThreads)
bn_apply_kernel(const uint16_t* __restrict__ x, uint16_t* __restrict__ y, const float2* __restrict__ stats, float* __restrict__ mean_io,
                float* __restrict__ var_io, int use_stored, int n_img, int C, int64_t hw, int chunks, float eps, float shift) {
  __shared__ float red[kBnWarps];
  if (use_stored) grid_dependency_wait();
  const int c = C - 1 - (int)blockIdx.y;
  const int G = n_img * chunks;
  constexpr int kSlots = kBnThreads / L;
  const int slot = (int)threadIdx.x / L;
  const int first = ((int)gridDim.x - 1 - (int)blockIdx.x) * kSlots;
  const int step = (int)gridDim.x * kSlots;
  auto locate = [&](int g0, int& count) {
    const int g = g0 + slot < G ? g0 + slot : G - 1;
    const int img = g / chunks, ch = g - img * chunks;
    const int64_t start = (int64_t)ch * kBnGroup;
    count = (int)(hw - start < kBnGroup ? hw - start : kBnGroup);
    return ((int64_t)img * C + c) * hw + start;
  };
  Group<L> grp;
  int g0 = first + (G - 1 - first) / step * step;  // this block's last step first
  int count;
  int64_t at = locate(g0, count);
  grp.place(x + at, count, g0 + slot < G);
  grp.template load<true>(x + at);
  float mean, var;
  if (use_stored) {
    mean = mean_io[c];
    var = var_io[c];
  } else {
    grid_dependency_wait();
    const float2* st = stats + (int64_t)c * G;
    const int last = (int)(hw - (int64_t)(chunks - 1) * kBnGroup);  // size of the last group of a plane
    const float total = (float)n_img * (float)hw;
    float acc = 0.f;
    for (int g = (int)threadIdx.x; g < G; g += kBnThreads) acc += st[g].x * (float)((g % chunks) == chunks - 1 ? last : kBnGroup);
    mean = block_sum(acc, red) / total;
    acc = 0.f;
    for (int g = (int)threadIdx.x; g < G; g += kBnThreads) {
      const float2 v = st[g];
      const float d = (v.x - mean) * shift;
      acc += (v.y + d * d) * (float)((g % chunks) == chunks - 1 ? last : kBnGroup);
    }
    var = block_sum(acc, red) / total * (1.0f / (shift * shift));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      mean_io[c] = mean;
      var_io[c] = var;
    }
  }
  const float inv = 1.0f / sqrtf(var + eps);
  const int lane = (int)(threadIdx.x & (L - 1));
  for (;;) {
    uint4* py = reinterpret_cast<uint4*>(y + at + grp.head);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (grp.live && lane + L * j < grp.nvec) {
        const uint32_t w[4] = {grp.q[j].x, grp.q[j].y, grp.q[j].z, grp.q[j].w};
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint16_t lo, hi;
          asm("mov.b32 {%0, %1}, %2;" : "=h"(lo), "=h"(hi) : "r"(w[i]));
          const __half2 h = __floats2half2_rn(fma_h(lo, kHalfOne, -mean) * inv, fma_h(hi, kHalfOne, -mean) * inv);
          o[i] = *reinterpret_cast<const uint32_t*>(&h);
        }
        __stcs(py + lane + L * j, make_uint4(o[0], o[1], o[2], o[3]));
      }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (grp.live && lane < (e == 0 ? grp.head : grp.tail))
        y[at + (e == 0 ? 0 : grp.head + 8 * grp.nvec) + lane] =
            __half_as_ushort(__float2half_rn(fma_h(grp.edge[e], kHalfOne, -mean) * inv));
    g0 -= step;
    if (g0 < 0) break;
    at = locate(g0, count);
    grp.place(x + at, count, true);
    grp.template load<true>(x + at);
  }
}

// Folding stored statistics and an optional scale/shift into the convolution before the batch
// norm: a_k = gamma_k / sqrt(var_k + eps); w'[k][j] = w[k][j] * a_k; b'[k] = (b[k] - mean_k) * a_k
// + beta_k.  One block per output channel.
__global__ void __launch_bounds__(256)
bn_fold_kernel(const uint16_t* __restrict__ w, const uint16_t* __restrict__ bias, const float* __restrict__ mean,
               const float* __restrict__ var, const float* __restrict__ gamma, const float* __restrict__ beta,
               float eps, int64_t per_k, uint16_t* __restrict__ w_out, uint16_t* __restrict__ b_out) {
  grid_dependency_wait();
  const int64_t k = blockIdx.x;
  const float a = (gamma != nullptr ? gamma[k] : 1.0f) / sqrtf(var[k] + eps);
  for (int64_t j = threadIdx.x; j < per_k; j += blockDim.x)
    w_out[k * per_k + j] = __half_as_ushort(__float2half_rn(__half2float(__ushort_as_half(w[k * per_k + j])) * a));
  if (threadIdx.x == 0) {
    const float b = bias != nullptr ? __half2float(__ushort_as_half(bias[k])) : 0.f;
    b_out[k] = __half_as_ushort(__float2half_rn(fmaf(b - mean[k], a, beta != nullptr ? beta[k] : 0.f)));
  }
}

int bn_chunks(int64_t hw) { return (int)((hw + kBnGroup - 1) / kBnGroup); }

}  // namespace

size_t batchnorm_workspace_bytes(int32_t n, int32_t c, int64_t hw) {
  return (size_t)2 * (size_t)c * (size_t)n * (size_t)bn_chunks(hw) * sizeof(float);
}

cudaError_t launch_batchnorm(const __half* x, __half* y, int32_t n, int32_t c, int64_t hw, float eps,
                             int32_t shift_log2, int32_t use_stored, float* mean, float* var, void* ws,
                             cudaStream_t stream) {
  const int chunks = bn_chunks(hw);
  const int64_t G = (int64_t)n * chunks;
  // Planes of at most 512 pixels: eight lanes per group (four groups per warp), so that 7x7 and 14x14
  // planes do not leave most of a warp without a vector.
  const bool small = hw <= 512;
  const int slots = kBnThreads / (small ? 8 : 32);
  // blocks per channel: one group per slot unless that would be far more blocks than the GPU can
  // hold several times over
  int64_t bx = (G + slots - 1) / slots;
  const int64_t cap = ((int64_t)sm_count() * 64 + c - 1) / c;
  if (bx > cap) bx = cap;
  if (bx < 1) bx = 1;
  const dim3 grid((unsigned)bx, (unsigned)c);
  const uint16_t* x16 = reinterpret_cast<const uint16_t*>(x);
  float2* stats = static_cast<float2*>(ws);
  const float shift = ldexpf(1.0f, shift_log2);
  cudaError_t err;
  if (!use_stored) {
    err = launch_kernel(small ? bn_group_kernel<8> : bn_group_kernel<32>, grid, dim3(kBnThreads), 0, stream, x16, stats, (int)n, (int)c,
                        hw, chunks, shift);
    if (err != cudaSuccess) return err;
    count_launch();
  }
  err = launch_kernel_attr(true, kCopyKernelCarveout, small ? bn_apply_kernel<8> : bn_apply_kernel<32>, grid,
                           dim3(kBnThreads), 0, stream, x16, reinterpret_cast<uint16_t*>(y), (const float2*)stats, mean, var,
                           (int)use_stored, (int)n, (int)c, hw, chunks, eps, shift);
  if (err != cudaSuccess) return err;
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_bn_fold(const __half* w, const __half* bias, const float* mean, const float* var,
                           const float* gamma, const float* beta, float eps, int32_t k, int64_t per_k, __half* w_out,
                           __half* b_out, cudaStream_t stream) {
  const cudaError_t err =
      launch_kernel(bn_fold_kernel, dim3((unsigned)k), dim3(256), 0, stream, reinterpret_cast<const uint16_t*>(w),
                    reinterpret_cast<const uint16_t*>(bias), mean, var, gamma, beta, eps, per_k,
                    reinterpret_cast<uint16_t*>(w_out), reinterpret_cast<uint16_t*>(b_out));
  if (err != cudaSuccess) return err;
  count_launch();
  return cudaGetLastError();
}

}  // namespace hgc
