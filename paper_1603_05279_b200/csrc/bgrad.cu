// Backward convolution with a binarised gradient (Section 3.2, "Binary Gradient"): the
// gradient at a convolution's output enters the backward convolution as sign(g) scaled by
// max|g| (of the image), the filters as alpha * sign(W) (Algorithm 1).  The contraction runs
// over the filters co with alpha[co] inside the sum, so it is a convolution of the real-valued
// tensor u = gmax * alpha[co] * sign(g) with +-1 filters: the Binary-Weight form (Eq. 1), run
// on that kernel with the filters transposed and turned by 180 degrees.  This file has the two
// small kernels around it: the per-image maximum and the transposed sign packing.
#include <algorithm>

#include "bgrad.cuh"

namespace xnor {

namespace {

constexpr int kMaxThreads = 256, kMaxCluster = 8;

__device__ __forceinline__ float abs_max4(float4 v) {
  return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
}

// max|g| over the block's share of an image: part `part` of `parts`, four 16-byte loads in flight.  NaN is
// skipped.
__device__ __forceinline__ float block_abs_max(const float *gi, size_t per_image, int vec4, unsigned part, unsigned parts) {
  const size_t step = (size_t)parts * kMaxThreads, first = (size_t)part * kMaxThreads + threadIdx.x;
  float m = 0.0f;
  if (vec4) {
    const float4 *g4 = reinterpret_cast<const float4 *>(gi);
    const size_t n4 = per_image / 4;
    size_t i = first;
    for (; i + 3 * step < n4; i += 4 * step) {
      const float4 a = load_global(g4 + i), b = load_global(g4 + i + step), c = load_global(g4 + i + 2 * step), d = load_global(g4 + i + 3 * step);
      m = fmaxf(m, fmaxf(fmaxf(abs_max4(a), abs_max4(b)), fmaxf(abs_max4(c), abs_max4(d))));
    }
    for (; i < n4; i += step) m = fmaxf(m, abs_max4(load_global(g4 + i)));
  } else {
    for (size_t i = first; i < per_image; i += step) m = fmaxf(m, fabsf(load_global(gi + i)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ float red[kMaxThreads / 32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kMaxThreads / 32; ++i) m = fmaxf(m, red[i]);
  return m;
}

// Blocks of an image meet in its element of gmax, cleared before: non-negative floats order like their bit
// patterns, so an integer atomicMax is exact and independent of the order of arrival.
__global__ void __launch_bounds__(kMaxThreads)
grad_max_kernel(const float *g, size_t per_image, int vec4, float *__restrict__ gmax) {
  stream_order();
  const float m = block_abs_max(g + (size_t)blockIdx.y * per_image, per_image, vec4, blockIdx.x, gridDim.x);
  if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned int *>(gmax) + blockIdx.y, __float_as_uint(m));
}

// The same with the cluster of an image's blocks, which needs neither zeros in gmax (a separate clear of
// the N values cost 1.3 us and the overlap with the kernel before) nor atomics.  Bound by HBM; the whole
// backward call at 128 channels, 28x28, 128 images: 67.7 -> 62.4 us with it and the wider preparation.
__global__ void __launch_bounds__(kMaxThreads)
grad_max_cluster_kernel(const float *g, size_t per_image, int vec4, float *__restrict__ gmax) {
  __shared__ float part[kMaxCluster];
  stream_order();
  const float m = block_abs_max(g + (size_t)blockIdx.y * per_image, per_image, vec4, blockIdx.x, kMaxCluster);
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");   // every block has started
  if (threadIdx.x == 0) {
    uint32_t a;                              // part[blockIdx.x] of the cluster's first block
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(part + blockIdx.x)));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(m) : "memory");
  }
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    float r = part[0];
    for (int i = 1; i < kMaxCluster; ++i) r = fmaxf(r, part[i]);
    gmax[blockIdx.y] = r;
  }
}

// One warp per packed word: lane = channel co of the word, the word is a ballot.
__global__ void __launch_bounds__(256)
binarize_weights_transposed_kernel(const float *w, int Co, int C, int kh, int kw,
                                   int CwT, uint32_t *__restrict__ wT_packed) {
  stream_order();
  const int lane = threadIdx.x & 31;
  const int taps = kh * kw, nwords = taps * CwT, npad = (nwords + 1) & ~1;
  const long long total = (long long)C * npad;
  for (long long id = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); id < total; id += (long long)gridDim.x * 8) {
    const int ci = (int)(id / npad), f = (int)(id - (long long)ci * npad);
    uint32_t word = 0u;
    if (f < nwords) {
      const int tap = f / CwT, cw = f - tap * CwT;
      const int ky = tap / kw, kx = tap - ky * kw;
      const int co = cw * 32 + lane;
      const bool in = co < Co;
      const float v = in ? load_global(w + (((size_t)co * C + ci) * kh + (kh - 1 - ky)) * kw + (kw - 1 - kx)) : -1.0f;
      word = __ballot_sync(0xffffffffu, in && v >= 0.0f);
    }
    if (lane == 0) wT_packed[packed_weight_index(C, ci, f)] = word;
  }
}

}  // namespace

cudaError_t launch_grad_max(const float *g, int N, size_t per_image, float *gmax, cudaStream_t st) {
  if (N > 65535) return cudaErrorInvalidValue;
  const int vec4 = (per_image % 4 == 0) ? 1 : 0;     // then every image starts on a 16-byte boundary
  // a cluster per image where these fill the GPU; fewer images need more blocks each than a cluster has
  if (kMaxCluster * N >= 4 * sm_count_of_current_device())
    return launch_kernel(grad_max_cluster_kernel, dim3(kMaxCluster, (unsigned)N), kMaxThreads, 0, st, (unsigned)kMaxCluster, g,
                         per_image, vec4, gmax);
  cudaError_t e = cudaMemsetAsync(gmax, 0, sizeof(float) * (size_t)N, st);
  if (e != cudaSuccess) return e;
  // enough blocks to fill the GPU whatever the batch, at most one per 4096 values
  const int sms = sm_count_of_current_device();
  const size_t want = (size_t)(8 * sms + N - 1) / (size_t)N;
  const size_t cap = (per_image + 4095) / 4096;
  const unsigned bx = (unsigned)std::max<size_t>(1, std::min(want, cap));
  return launch_kernel(grad_max_kernel, dim3(bx, (unsigned)N), kMaxThreads, 0, st, 1, g, per_image, vec4, gmax);
}

cudaError_t launch_binarize_weights_transposed(const float *w, int Co, int C, int kh, int kw,
                                               uint32_t *wT_packed, cudaStream_t st) {
  const int CwT = (Co + 31) / 32;
  const long long total = (long long)C * ((kh * kw * CwT + 1) & ~1);
  const unsigned grid = (unsigned)std::min<long long>((total + 7) / 8, 4096);
  return launch_kernel(binarize_weights_transposed_kernel, dim3(grid), 256, 0, st, 1, w, Co, C, kh, kw, CwT, wT_packed);
}

}  // namespace xnor
