// Shared declarations of the CUDA translation units of libxnor (internal).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "xnor.h"

namespace xnor {

struct ConvGeom {
  int N, C, H, W, Co, kh, kw, stride, pad, Ho, Wo, Cw;
  int flags;      // XNOR_FLAG_* of the descriptor
};

// What the BinConv epilogues do beyond Eq. 11's D K alpha (+ residual).
struct EpiOpts {
  int relu;          // max(v, 0) on the stored value
  float out_scale;   // v = D K (alpha out_scale); 1: as Eq. 11
  int acc_shift;     // acc_out receives D << acc_shift ...
  int acc_accum;     // ... added to what acc_out holds (1) or stored (0)
};
inline EpiOpts default_epi(const ConvGeom &g) {
  EpiOpts e;
  e.relu = (g.flags & XNOR_FLAG_RELU) ? 1 : 0;
  e.out_scale = 1.0f;
  e.acc_shift = 0;
  e.acc_accum = 0;
  return e;
}

inline ConvGeom make_geom(const xnor_conv_desc &d) {
  ConvGeom g;
  g.N = d.N; g.C = d.C_in; g.H = d.H; g.W = d.W; g.Co = d.C_out;
  g.kh = d.k_h; g.kw = d.k_w; g.stride = d.stride; g.pad = d.pad;
  g.Ho = (d.H + 2 * d.pad - d.k_h) / d.stride + 1;
  g.Wo = (d.W + 2 * d.pad - d.k_w) / d.stride + 1;
  g.Cw = (d.C_in + 31) / 32;
  g.flags = d.flags;
  return g;
}

// Consecutive kernels of a stream overlap their launch and set-up with the end of the kernel before
// (programmatic dependent launch).  Every kernel that reads or writes a caller's memory is launched through
// launch_kernel, calls stream_order() before its first access to global memory and reads that memory
// with load_global, asynchronous copies or ordinary loads: stream_order() returns when the kernels before
// it in the stream have completed and their writes are visible, so a kernel sees everything that
// was launched before it.  A kernel that leaves SMs free then lets the next one start at once (a batch-1
// layer's kernels take 2 to 9 us each, a launch gap with the set-up of the tensor-core kernel 3: the
// 16-layer chain of one image 395 -> 276 us).  A kernel that fills the GPU lets it start as its own
// blocks leave (256 images 1643 -> 1578 us against ordinary launches): started earlier, the next kernel's
// waiting blocks keep other streams' kernels off the SMs (the four AlexNet layers on parallel branches
// 224 -> 238 us) and its own split of L1 and shared memory is the one of the kernel it waits for (a pool
// that reads through L1 92 -> 113 us).
// (Plans and this rule take a B200's SM count for a constant, so that they can be made without a device;
// grids go by the device's.)
constexpr unsigned kSms = 148;
__device__ __forceinline__ void stream_order() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (gridDim.x * gridDim.y < kSms) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A load of global memory that the kernel before may still have been writing when this one started: coherent,
// and volatile, which keeps it behind stream_order().  (__ldg, or an ordinary load through a pointer to
// const that is __restrict__, promises that nobody writes the memory while the kernel lives, and may be
// moved ahead of the wait.)
__device__ __forceinline__ float load_global(const float *p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ float4 load_global(const float4 *p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ uint32_t load_global(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ uint2 load_global(const uint2 *p) {
  uint2 v;
  asm volatile("ld.global.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(__cvta_generic_to_global(p)));
  return v;
}
// The same where `in`, else 0: one predicated instruction.  (A branch around each volatile load made the
// 49 taps of the 7x7 box filter 0.7 us slower.)
__device__ __forceinline__ float load_global_if(const float *p, bool in) {
  float v;
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %2, 0;\n\t"
      "mov.f32 %0, 0f00000000;\n\t"
      "@q ld.global.f32 %0, [%1];\n\t}"
      : "=&f"(v) : "l"(__cvta_generic_to_global(p)), "r"((int)in));
  return v;
}

// `cluster`: CTAs per cluster along x (1: none).
template <class... Params, class... Args>
cudaError_t launch_kernel(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st,
                          unsigned cluster, const Args &...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
  if (e != cudaSuccess) (void)cudaGetLastError();
  return e;
}

// Packed weights are stored word-pair-major so that the convolution kernels read them
// coalesced: with f = tap * Cw + cw the index of a word inside a filter (tap = ky * k_w + kx),
// word f of filter co is element ((f / 2) * C_out + co) * 2 + f % 2.  Words 2j and 2j+1 of all
// filters (one 64-channel step of the contraction) are contiguous.
__host__ __device__ inline size_t packed_weight_index(int Co, int co, int f) {
  return ((size_t)(f >> 1) * Co + co) * 2 + (f & 1);
}

// Launchers: return the cudaError_t of the launch (cudaGetLastError, cleared).
cudaError_t launch_binarize_weights(const float *w, int Co, int C, int kh, int kw,
                                    uint32_t *w_packed, float *alpha, cudaStream_t st);
cudaError_t launch_binactiv(const float *x, const float *scale, const float *shift,
                            const ConvGeom &g, uint32_t *x_packed, float *A, float *K,
                            cudaStream_t st);
// Same, with A in the library's own fixed array (N*H*W <= binactiv_static_max_pixels()).
size_t binactiv_static_max_pixels();
cudaError_t launch_binactiv_static(const float *x, const float *scale, const float *shift,
                                   const ConvGeom &g, uint32_t *x_packed, float *K,
                                   cudaStream_t st);
bool binactiv_supported(const ConvGeom &g, bool has_bn);
// BinActiv with q_k in place of sign(): kbits planes of index bits, [kbits][N][H][W][Cw].
cudaError_t launch_binactiv_kbit(const float *x, const float *scale, const float *shift,
                                 const ConvGeom &g, int kbits, uint32_t *x_planes, float *A, float *K,
                                 cudaStream_t st);
bool binconv_popc_supported(const ConvGeom &g);
cudaError_t launch_binconv_popc(const uint32_t *xp, const uint32_t *wp, const float *alpha,
                                const float *K, const float *residual, const ConvGeom &g,
                                const EpiOpts &epi, float *out, int32_t *acc_out, cudaStream_t st);
// Function attributes (dynamic shared-memory limits) belong to a device: a launcher sets them
// once per device.  Returns the flag of the current device (out-of-range ids share the last).
inline bool &attr_done_for_current_device(bool (&flags)[64]) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); dev = 0; }
  return flags[dev < 0 ? 0 : (dev > 63 ? 63 : dev)];
}

// Number of SMs of the current device, looked up once per device (persistent kernels size
// their grids by it).  148 if the query fails.
inline int sm_count_of_current_device() {
  static int counts[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return 148; }
  const int slot = dev < 0 ? 0 : (dev > 63 ? 63 : dev);
  if (counts[slot] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
      (void)cudaGetLastError();
      n = 148;
    }
    counts[slot] = n;
  }
  return counts[slot];
}

// Persistent tensor-core engine (strides 1 and 2).  Variants: one CTA per SM or CTA pairs
// (one MMA drives two SMs), each with the filters of a slab resident in shared memory when
// they fit or always streamed through a ring (re-expanded per work item).
enum TcVariant { kTcAuto = 0, kTcSingle, kTcSingleStream, kTcPair, kTcPairStream };
// planes: bit planes of the input that one pass takes, 1 or 2
bool umma_tc_supported(const ConvGeom &g, TcVariant v, int planes = 1);
// Fills the tensor-core fields of *out; false: the shape is not covered.
bool tc_plan_info(const ConvGeom &g, TcVariant v, bool fuse, int planes, bool residual, xnor_conv_plan *out);
cudaError_t launch_binconv_tc(const uint32_t *xp, const uint32_t *wp, const float *alpha,
                              const float *K, const float *residual, const ConvGeom &g,
                              const EpiOpts &epi, float *out, int32_t *acc_out, TcVariant v,
                              cudaStream_t st, const uint32_t *xp2 = nullptr);
// BinConv with the next layer's BinActiv fused into its epilogue (sign bits packed along the
// filters, partial sums of |y| per filter slab and chunk of its columns); tc_fused_parts = number of
// partial planes for the shape (0: the fused kernel does not cover it).
int tc_fused_parts(const ConvGeom &g, TcVariant v);
cudaError_t launch_binconv_tc_fused(const uint32_t *xp, const uint32_t *wp, const float *alpha,
                                    const float *K, const float *residual, const ConvGeom &g,
                                    float *out, const float *next_scale, const float *next_shift,
                                    uint32_t *xp_next, float *A_part, TcVariant v, cudaStream_t st);
// A = (sum of the partial planes) / C, then K = box filter of A for geometry g.
cudaError_t launch_binactiv_finish(const float *A_part, int parts, const ConvGeom &g, float *A,
                                   float *K, cudaStream_t st);
// Binary-Weight-Network convolution (Eq. 1) on bf16 activations laid out as a zero-padded pixel
// stream: elements of that stream for a geometry, its preparation from fp32 NCHW, the convolution.
bool bwn_supported(const ConvGeom &g);
size_t bwn_stream_elems(const ConvGeom &g);
cudaError_t launch_bwn_prepare(const float *x, const float *scale, const float *shift,
                               const ConvGeom &g, uint16_t *x_stream, cudaStream_t st);
cudaError_t launch_bwn_conv(const uint16_t *x_stream, const uint32_t *wp, const float *alpha,
                            const float *residual, const ConvGeom &g, float *out, cudaStream_t st);
cudaError_t read_status_bwn(int *status);
// Measured rates of the tensor pipe (1-bit MACs of the mxf4 MMA per clock per SM) and of the
// CUDA-core population count (popc per clock per SM) on the current device.  Synchronises.
cudaError_t measure_pipe_peaks(double *mma_mac_per_clk_per_sm, double *popc_per_clk_per_sm,
                               cudaStream_t st);
// A one-warp kernel whose bounded wait expires (nothing signals its barrier).
cudaError_t launch_wait_timeout_selftest(cudaStream_t st);
// Reads (and clears if set) the device status word of the tensor-core kernel.
cudaError_t read_status_tc(int *status);
// Same for the BinActiv kernel that waits on bulk copies.
cudaError_t read_status_act(int *status);
// Same for the pooling kernel that streams planes.
cudaError_t read_status_pool(int *status);
// Kernels launch_binactiv launches for this shape (1 or 2).
int binactiv_launch_count(const ConvGeom &g, bool has_bn);
cudaError_t launch_maxpool2d(const float *x, int N, int C, int H, int W, int k, int stride, int pad,
                             bool relu, float *out, cudaStream_t st);
cudaError_t launch_shortcut_conv1x1(const float *x, const float *w, int N, int C, int H, int W,
                                    int Co, int stride, float *out, cudaStream_t st);

}  // namespace xnor
