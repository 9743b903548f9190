// The Pool layer that closes the block (Section 3.2, "Training XNOR-Networks": BatchNorm,
// BinActiv, BinConv, Pool, with an optional ReLU after the binary convolution): max pooling
// of BinConv's fp32 output.  Taps outside the image take no part in the maximum.
#include <algorithm>

#include "common.cuh"
#include "umma_common.cuh"

namespace xnor {

__device__ int g_status_pool = 0;

namespace {

constexpr int kPoolThreads = 256;

// Exact n / d for n < 2^31: q = (n * m) >> (31 + s) with m = ceil(2^(31+s) / d), s = ceil(log2 d).
struct Magic { uint32_t m; int s; };
__device__ __forceinline__ uint32_t fast_div(uint32_t n, Magic g) {
  return (uint32_t)(((uint64_t)n * g.m) >> (31 + g.s));
}

struct PoolParams {
  const float *x;
  float *out;
  long long planes;              // N * C
  int H, W, k, stride, pad, Ho, Wo;
  Magic div_howo, div_wo;
  int per_chunk;                 // planes per chunk: a multiple of 4, so that chunks start on 16 bytes
  uint32_t chunk_bytes;          // shared memory of a chunk's planes
};

// Maximum over the window whose corner is (iy, ix) of plane t in shared memory.
// Windows of KS x KS, wholly inside the plane or (kPad) with every tap moved to the nearest one that is: that
// is one of the window's own (pad < k), so the maximum is the same and nothing branches.  (Loops over the taps
// inside the plane were slower than the kernel below: 64 channels, 39x39, 3x3/2 with a padding of 1, 247
// images 63.4 us, the kernel below 52.3, this 27.2; 2x2 to 7x7, 200 drawn shapes, 0.68 in the median.)
template <int KS, bool kPad>
__device__ __forceinline__ float window_max(const PoolParams &P, const float *t, int iy, int ix) {
  int row[KS], col[KS];
#pragma unroll
  for (int i = 0; i < KS; ++i) {
    row[i] = (kPad ? min(max(iy + i, 0), P.H - 1) : iy + i) * P.W;
    col[i] = kPad ? min(max(ix + i, 0), P.W - 1) : ix + i;
  }
  float m = t[row[0] + col[0]];
#pragma unroll
  for (int ky = 0; ky < KS; ++ky)
#pragma unroll
    for (int kx = 0; kx < KS; ++kx)
      if (ky + kx > 0) m = fmaxf(m, t[row[ky] + col[kx]]);
  return m;
}

// Planes are streamed through shared memory: a chunk is a few whole planes, contiguous in memory and
// 16-byte aligned, and comes in with one bulk copy; kBufs chunks per block in flight.  HBM bounds it.
constexpr int kBufs = 4;
template <bool kRelu, int KS, bool kPad>
__global__ void __launch_bounds__(kPoolThreads) maxpool_stream_kernel(const PoolParams P) {
  using namespace umma;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) uint64_t full[kBufs];
  __shared__ volatile int abort_flag;
  const int tid = threadIdx.x;
  const uint32_t base = smem_u32(smem);
  const int HW = P.H * P.W, HoWo = P.Ho * P.Wo;
  const long long nchunks = (P.planes + P.per_chunk - 1) / P.per_chunk;
  if (tid == 0) {
    for (int i = 0; i < kBufs; ++i) mbar_init(smem_u32(&full[i]), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  stream_order();
  // from the end to the start: the last part of what the convolution wrote is still in the L2
  auto place = [&](long long c) { return nchunks - 1 - c; };
  // thread 0: chunk c into buffer b; the tensor's last floats (its size need not be a multiple of
  // four) by plain loads
  auto fetch = [&](long long c, int b) {
    const long long p0 = place(c) * P.per_chunk, np = min((long long)P.per_chunk, P.planes - p0);
    const uint32_t floats = (uint32_t)np * (uint32_t)HW, bulk = floats & ~3u, dst = base + (uint32_t)b * P.chunk_bytes;
    const float *src = P.x + (size_t)p0 * HW;
    for (uint32_t i = bulk; i < floats; ++i) reinterpret_cast<float *>(smem + (size_t)b * P.chunk_bytes)[i] = load_global(src + i);
    const uint32_t bar = smem_u32(&full[b]);
    if (bulk) {
      mbar_arrive_expect_tx(bar, bulk * 4u);
      bulk_copy_g2s(dst, src, bulk * 4u, bar);
    } else {
      mbar_arrive(bar);
    }
  };
  long long next = blockIdx.x;
  int pending = 0;                       // copies started and not yet waited for
  if (tid == 0)
    for (int b = 0; b < kBufs - 1 && next < nchunks; ++b, next += gridDim.x, ++pending) fetch(next, b);
  int b = 0;
  uint32_t ph = 0u;
  bool ok = true;
  for (long long c = blockIdx.x; c < nchunks; c += gridDim.x) {
    // the buffer filled now is the one every thread left before the last __syncthreads
    if (tid == 0 && next < nchunks) {
      fence_proxy_async();
      fetch(next, b == 0 ? kBufs - 1 : b - 1);
      next += gridDim.x;
      ++pending;
    }
    ok = mbar_wait(smem_u32(&full[b]), ph, &abort_flag, &g_status_pool);
    if (__syncthreads_or(!ok)) break;
    --pending;
    const long long p0 = place(c) * P.per_chunk;
    const uint32_t count = (uint32_t)min((long long)P.per_chunk, P.planes - p0) * (uint32_t)HoWo;
    const float *chunk = reinterpret_cast<const float *>(smem + (size_t)b * P.chunk_bytes);
    float *out = P.out + (size_t)p0 * HoWo;
    for (uint32_t i = tid; i < count; i += kPoolThreads) {
      const uint32_t pl = fast_div(i, P.div_howo), r = i - pl * (uint32_t)HoWo, oy = fast_div(r, P.div_wo), ox = r - oy * (uint32_t)P.Wo;
      const float m = window_max<KS, kPad>(P, chunk + (size_t)pl * HW, (int)oy * P.stride - P.pad, (int)ox * P.stride - P.pad);
      __stcs(out + i, kRelu ? fmaxf(m, 0.0f) : m);
    }
    if (++b == kBufs) { b = 0; ph ^= 1u; }
    __syncthreads();
  }
  // gave up: the copies in flight must land before the block's shared memory is released
  if (tid == 0)
    for (; pending > 0; --pending) {
      for (int i = 0; i < (1 << 20) && !mbar_try(smem_u32(&full[b]), ph); ++i) {}
      if (++b == kBufs) { b = 0; ph ^= 1u; }
    }
}

// A thread per output, its window through the read-only cache: planes too large to stage, and calls
// too small to be worth it.
template <bool kRelu>
__global__ void __launch_bounds__(kPoolThreads)
maxpool_kernel(const float *x, long long total_out, int H, int W, int k, int stride,
               int pad, int Ho, int Wo, Magic div_howo, Magic div_wo, float *__restrict__ out) {
  stream_order();
  const int HoWo = Ho * Wo;
  // chunks of 2^30 outputs keep the index arithmetic in 32 bits
  for (long long base = 0; base < total_out; base += (1ll << 30)) {
    const uint32_t count = (uint32_t)min(total_out - base, 1ll << 30);
    const long long plane0 = base / HoWo;               // base is not a multiple of HoWo in general:
    const uint32_t off0 = (uint32_t)(base - plane0 * HoWo);   // outputs of the chunk start off0 into plane0
    for (uint32_t i = blockIdx.x * kPoolThreads + threadIdx.x; i < count;
         i += gridDim.x * kPoolThreads) {
      const uint32_t o = i + off0;                       // < 2^31
      const uint32_t pl = fast_div(o, div_howo);
      const int r = (int)(o - pl * (uint32_t)HoWo);
      const int oy = (int)fast_div((uint32_t)r, div_wo), ox = r - oy * Wo;
      const int y0 = max(oy * stride - pad, 0), y1 = min(oy * stride - pad + k, H);
      const int x0 = max(ox * stride - pad, 0), x1 = min(ox * stride - pad + k, W);
      const float *t = x + (size_t)(plane0 + pl) * H * W;
      float m = load_global(t + (size_t)y0 * W + x0);
      for (int iy = y0; iy < y1; ++iy)
        for (int ix = x0; ix < x1; ++ix) m = fmaxf(m, load_global(t + (size_t)iy * W + ix));
      out[base + i] = kRelu ? fmaxf(m, 0.0f) : m;
    }
  }
}

template <bool kRelu, int KS, bool kPad>
cudaError_t launch_stream(const PoolParams &P, unsigned grid, size_t smem, cudaStream_t st) {
  static bool attr_flags[64] = {};
  bool &attr_set = attr_done_for_current_device(attr_flags);
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(maxpool_stream_kernel<kRelu, KS, kPad>, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024);
    if (e != cudaSuccess) { (void)cudaGetLastError(); return e; }
    attr_set = true;
  }
  return launch_kernel(maxpool_stream_kernel<kRelu, KS, kPad>, dim3(grid), kPoolThreads, smem, st, 1, P);
}

}  // namespace

cudaError_t launch_maxpool2d(const float *x, int N, int C, int H, int W, int k, int stride, int pad,
                             bool relu, float *out, cudaStream_t st) {
  const int Ho = (H + 2 * pad - k) / stride + 1, Wo = (W + 2 * pad - k) / stride + 1;
  if ((long long)Ho * Wo >= (1ll << 30)) return cudaErrorInvalidValue;
  const long long total = (long long)N * C * Ho * Wo;
  const int sms = sm_count_of_current_device();
  auto magic = [](uint32_t d) {
    Magic g;
    g.s = 0;
    while ((1u << g.s) < d) ++g.s;
    g.m = (uint32_t)((((unsigned long long)1 << (31 + g.s)) + d - 1) / d);
    return g;
  };
  const Magic dh = magic((uint32_t)(Ho * Wo)), dw = magic((uint32_t)Wo);
  // Streamed when chunks of at least four planes and at most 24 KB exist, enough of them for several
  // rounds of every block (as many blocks per SM as fit, four chunks each).  AlexNet's 3x3/2 pool of conv2's
  // output (235 MB): 92 us with a thread per output, bounded by its nine global loads, 47 us streamed (5 TB/s).
  const size_t four = 16 * (size_t)H * W;
  if (four <= 24 * 1024 && (k <= 5 || k == 7)) {
    PoolParams P;
    P.x = x; P.out = out; P.planes = (long long)N * C;
    P.H = H; P.W = W; P.k = k; P.stride = stride; P.pad = pad; P.Ho = Ho; P.Wo = Wo;
    P.div_howo = dh; P.div_wo = dw;
    P.per_chunk = 4 * (int)std::max<size_t>(1, 16 * 1024 / four);
    P.chunk_bytes = (uint32_t)(((size_t)P.per_chunk * H * W * 4 + 127) / 128 * 128);
    const long long nchunks = (P.planes + P.per_chunk - 1) / P.per_chunk;
    if (nchunks >= 4ll * sms) {
      const size_t smem = (size_t)kBufs * P.chunk_bytes;
      const long long per_sm = std::min<long long>(6, (long long)(227 * 1024 / (smem + 2048)));
      const unsigned grid = (unsigned)std::min<long long>(nchunks, per_sm * sms);
#define XNOR_POOL(KS, kPad) (relu ? launch_stream<true, KS, kPad>(P, grid, smem, st) : launch_stream<false, KS, kPad>(P, grid, smem, st))
      if (k == 1) return XNOR_POOL(1, true);
      if (k == 2) return pad ? XNOR_POOL(2, true) : XNOR_POOL(2, false);
      if (k == 3) return pad ? XNOR_POOL(3, true) : XNOR_POOL(3, false);
      if (k == 4) return XNOR_POOL(4, true);
      if (k == 5) return XNOR_POOL(5, true);
      return XNOR_POOL(7, true);
#undef XNOR_POOL
    }
  }
  const unsigned grid = (unsigned)std::min<long long>((total + kPoolThreads - 1) / kPoolThreads,
                                                      16ll * sms);
  return launch_kernel(relu ? maxpool_kernel<true> : maxpool_kernel<false>, dim3(grid), kPoolThreads, 0, st, 1, x, total, H, W,
                       k, stride, pad, Ho, Wo, dh, dw, out);
}

cudaError_t read_status_pool(int *status) {
  cudaError_t e = cudaMemcpyFromSymbol(status, g_status_pool, sizeof(int));
  const int zero = 0;
  if (e == cudaSuccess && *status != 0) e = cudaMemcpyToSymbol(g_status_pool, &zero, sizeof(int));
  return e;
}

}  // namespace xnor
