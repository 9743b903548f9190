// Full-precision 1x1 strided convolution without bias (ResNet projection
// shortcut, Section 4.2): out[n][co][oy][ox] = sum_c x[n][c][oy*s][ox*s] w[co][c].
// Every output is one chain of fused multiply-adds over the channels in order, whatever the tiling.
#include "common.cuh"

namespace xnor {

namespace {

constexpr int kThreads = 128, TX = 16, TY = 8;

// (a.x * b.x + c.x, a.y * b.y + c.y), each rounded as by fmaf: one instruction for two values
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long dup(float v) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float2 halves(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
// four bytes global -> shared, zeros where !on
__device__ __forceinline__ void copy4(void *dst, const float *src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
               ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(on ? 4 : 0) : "memory");
}

// Thread (tx, ty) owns PT pixels (groups of 4, 64 apart; PT = 2: a pair) and FT filters; KS channels per
// step, ST steps in flight.  The inner loop is FT / 2 * PT paired multiply-adds for (PT + FT) / 4
// 16-byte shared-memory reads.  What bounds the large tile is the fp32 pipe (128 multiply-adds per
// clock and SM: 44 us for the 64 -> 128 projection of 256 56x56 images); the former kernel, with 8 x 4
// outputs per thread and register staging, spent as long on shared-memory reads (115 us).
template <int PT, int FT, int KS, int ST>
__global__ void __launch_bounds__(kThreads, PT == 8 ? 4 : 8)
shortcut_conv1x1_kernel(const float *__restrict__ x, const float *__restrict__ w, int C, int H,
                        int W, int Co, int stride, int Ho, int Wo, long long total_pix, int fblocks,
                        float *__restrict__ out) {
  constexpr int TPX = TX * PT, TF = TY * FT, WP = TF + 4;       // pitch of a filter row: staggered banks
  extern __shared__ __align__(16) float smem[];
  float *const xs = smem;                                       // [ST][KS][TPX]
  float *const ws = smem + ST * KS * TPX;                       // [ST][KS][WP]
  stream_order();
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const long long op0 = (long long)(blockIdx.x / (unsigned)fblocks) * TPX;
  const int co0 = (int)(blockIdx.x % (unsigned)fblocks) * TF;
  const int HoWo = Ho * Wo;
  const size_t plane = (size_t)H * W;

  // staging: a thread copies channels lk, lk + 128 / TPX, ... of one pixel, and TF KS / 128 weights
  const int lp = tid % TPX, lk = tid / TPX;
  const long long lgp = op0 + lp;
  const bool lp_on = lgp < total_pix;
  const long long ln = lp_on ? lgp / HoWo : 0;
  const int lop = lp_on ? (int)(lgp - ln * HoWo) : 0, loy = lop / Wo, lox = lop - loy * Wo;
  const float *xsrc = x + ((size_t)ln * C * H + (size_t)loy * stride) * W + (size_t)lox * stride;
  auto fetch = [&](int step) {
    if (step * KS < C) {
      float *xd = xs + (step % ST) * (KS * TPX) + lp, *wd = ws + (step % ST) * (KS * WP);
#pragma unroll
      for (int q = 0; q < KS * TPX / kThreads; ++q) {
        const int k = lk + q * (kThreads / TPX), c = step * KS + k;
        const bool on = lp_on && c < C;
        copy4(xd + k * TPX, on ? xsrc + (size_t)c * plane : x, on);
      }
#pragma unroll
      for (int q = 0; q < KS * TF / kThreads; ++q) {
        const int e = tid + q * kThreads, k = e % KS, f = e / KS, c = step * KS + k;
        const bool on = co0 + f < Co && c < C;
        copy4(wd + k * WP + f, on ? w + (size_t)(co0 + f) * C + c : w, on);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  unsigned long long acc[PT / 2][FT];
#pragma unroll
  for (int i = 0; i < PT / 2; ++i)
#pragma unroll
    for (int j = 0; j < FT; ++j) acc[i][j] = 0ull;
#pragma unroll
  for (int s = 0; s < ST - 1; ++s) fetch(s);
  const int nsteps = (C + KS - 1) / KS;
  for (int step = 0; step < nsteps; ++step) {
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
    __syncthreads();                       // the step's operands are here, everybody has left the last one's
    fetch(step + ST - 1);
    const float *xt = xs + (step % ST) * (KS * TPX), *wt = ws + (step % ST) * (KS * WP) + ty * FT;
#pragma unroll 8
    for (int k = 0; k < KS; ++k) {
      unsigned long long xv[PT / 2];
      float wv[FT];
      if constexpr (PT == 8) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(xt + k * TPX + tx * 4);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(xt + k * TPX + 64 + tx * 4);
        xv[0] = a.x; xv[1] = a.y; xv[2] = b.x; xv[3] = b.y;
      } else {
        xv[0] = *reinterpret_cast<const unsigned long long *>(xt + k * TPX + tx * 2);
      }
      if constexpr (FT == 8) {
        const float4 a = *reinterpret_cast<const float4 *>(wt + k * WP), b = *reinterpret_cast<const float4 *>(wt + k * WP + 4);
        wv[0] = a.x; wv[1] = a.y; wv[2] = a.z; wv[3] = a.w;
        wv[4] = b.x; wv[5] = b.y; wv[6] = b.z; wv[7] = b.w;
      } else {
        const float2 a = *reinterpret_cast<const float2 *>(wt + k * WP);
        wv[0] = a.x; wv[1] = a.y;
      }
#pragma unroll
      for (int j = 0; j < FT; ++j) {
        const unsigned long long ww = dup(wv[j]);
#pragma unroll
        for (int i = 0; i < PT / 2; ++i) acc[i][j] = fma2(xv[i], ww, acc[i][j]);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  // runs of 4 (2) consecutive pixels of the flat index: one image and aligned when H_out*W_out is a
  // multiple of their number, else each pixel finds its own image
  constexpr int RUN = PT == 8 ? 4 : 2;
#pragma unroll
  for (int h = 0; h < PT / RUN; ++h) {
    const long long gp = op0 + 64 * h + tx * RUN;
    if (gp >= total_pix) continue;
    const long long n0 = gp / HoWo;
    const int p0 = (int)(gp - n0 * HoWo);
#pragma unroll
    for (int j = 0; j < FT; ++j) {
      const int co = co0 + ty * FT + j;
      if (co >= Co) continue;
      float v[RUN];
#pragma unroll
      for (int i = 0; i < RUN / 2; ++i) {
        const float2 t = halves(acc[h * (RUN / 2) + i][j]);
        v[2 * i] = t.x; v[2 * i + 1] = t.y;
      }
      if (HoWo % RUN == 0) {
        float *dst = out + ((size_t)n0 * Co + co) * HoWo + p0;
        if constexpr (RUN == 4) *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
        else *reinterpret_cast<float2 *>(dst) = make_float2(v[0], v[1]);
      } else {
#pragma unroll
        for (int i = 0; i < RUN; ++i) {
          if (gp + i < total_pix) {
            const long long ni = p0 + i < HoWo ? n0 : (gp + i) / HoWo;
            const int pi = (int)(gp + i - ni * HoWo);
            out[((size_t)ni * Co + co) * HoWo + pi] = v[i];
          }
        }
      }
    }
  }
}

template <int PT, int FT, int KS, int ST>
cudaError_t launch_tiles(const float *x, const float *w, int C, int H, int W, int Co, int stride, int Ho, int Wo,
                         long long total_pix, float *out, cudaStream_t st) {
  constexpr int TPX = TX * PT, TF = TY * FT;
  constexpr size_t smem = (size_t)ST * KS * (TPX + TF + 4) * sizeof(float);
  static_assert(smem <= 48 * 1024, "no opt-in needed");
  const int fblocks = (Co + TF - 1) / TF;
  const long long blocks = (total_pix + TPX - 1) / TPX * fblocks;
  if (blocks > 0x7FFFFFFFll) return cudaErrorInvalidValue;
  return launch_kernel(shortcut_conv1x1_kernel<PT, FT, KS, ST>, dim3((unsigned)blocks), kThreads, smem, st, 1, x, w, C, H, W, Co,
                       stride, Ho, Wo, total_pix, fblocks, out);
}

}  // namespace

cudaError_t launch_shortcut_conv1x1(const float *x, const float *w, int N, int C, int H, int W,
                                    int Co, int stride, float *out, cudaStream_t st) {
  const int Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
  const long long total_pix = (long long)N * Ho * Wo;
  // tiles of 128 pixels x 64 filters where they fill the GPU twice over (four are resident per SM),
  // else 32 x 16: a single image's projection has 7 to 28 large tiles
  if ((total_pix + 127) / 128 * ((Co + 63) / 64) >= 2ll * sm_count_of_current_device())
    return launch_tiles<8, 8, 16, 3>(x, w, C, H, W, Co, stride, Ho, Wo, total_pix, out, st);
  return launch_tiles<2, 2, 32, 4>(x, w, C, H, W, Co, stride, Ho, Wo, total_pix, out, st);
}

}  // namespace xnor
