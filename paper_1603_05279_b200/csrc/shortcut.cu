// Full-precision 1x1 strided convolution without bias (ResNet projection
// shortcut, Section 4.2): out[n][co][oy][ox] = sum_c x[n][c][oy*s][ox*s] w[co][c].
// Every output is one chain of fused multiply-adds over the channels in order, whatever the tiling.
#include <algorithm>

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
__device__ __forceinline__ unsigned long long swapped(unsigned long long v) {
  unsigned long long r;
  asm("{\n\t.reg .b32 a, b;\n\tmov.b64 {a, b}, %1;\n\tmov.b64 %0, {b, a};\n\t}" : "=l"(r) : "l"(v));
  return r;
}
__device__ __forceinline__ float2 halves(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
// `bytes` (4 or 0) bytes global -> shared, zeros for the rest of the four
__device__ __forceinline__ void copy4(uint32_t dst, const float *src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// Thread (tx, ty) owns PT pixels (groups of 4, 64 apart; PT = 2: a pair) and FT filters; KS channels per
// step, ST steps in flight.  The multiply-adds are paired: pixels (x0, x1) with filters (w0, w1) and
// with (w1, w0), so that neither operand has to be duplicated.  What bounds the large tile is the fp32
// pipe (128 multiply-adds per clock and SM measured: 45 us for the 64 -> 128 projection of 256 56x56
// images) and the issue slots beside it (an earlier form spent 38 of 64 M instructions on duplicating
// filters and on staging addresses, 92 us); hence addresses by increments, and clipping of the channels
// only in a last partial step.
template <int PT, int FT, int KS, int ST>
__global__ void __launch_bounds__(kThreads, PT == 8 ? 4 : 8)
shortcut_conv1x1_kernel(const float *x, const float *w, int C, int H,
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

  // staging: a thread copies channels lk, lk + KT, ... of one pixel and channel wk of filters wf, wf + FQ, ...
  constexpr int KT = kThreads / TPX, FQ = kThreads / KS;
  const int lp = tid % TPX, lk = tid / TPX, wk = tid % KS, wf = tid / KS;
  const long long lgp = op0 + lp;
  const bool lp_on = lgp < total_pix;
  const long long ln = lp_on ? lgp / HoWo : 0;
  const int lop = lp_on ? (int)(lgp - ln * HoWo) : 0, loy = lop / Wo, lox = lop - loy * Wo;
  const float *xsrc = x + ((size_t)ln * C * H + (size_t)loy * stride) * W + (size_t)lox * stride + (size_t)lk * plane;
  const float *wsrc = w + (size_t)(co0 + wf) * C + wk;
  const uint32_t xd0 = (uint32_t)__cvta_generic_to_shared(xs) + (uint32_t)(lk * TPX + lp) * 4u;
  const uint32_t wd0 = (uint32_t)__cvta_generic_to_shared(ws) + (uint32_t)(wk * WP + wf) * 4u;
  int fbuf = 0;                                                 // buffer of the next step to fetch
  auto fetch = [&](int step) {
    const int left = C - step * KS;                             // channels from this step on
    if (left > 0) {
      const uint32_t xd = xd0 + (uint32_t)fbuf * (KS * TPX * 4u), wd = wd0 + (uint32_t)fbuf * (KS * WP * 4u);
      const float *s = xsrc;
      if (left >= KS) {
        const int bytes = lp_on ? 4 : 0;
#pragma unroll
        for (int q = 0; q < KS / KT; ++q) {
          copy4(xd + (uint32_t)(q * KT * TPX) * 4u, s, bytes);
          s += KT * plane;
        }
      } else {
#pragma unroll
        for (int q = 0; q < KS / KT; ++q) {
          const bool on = lp_on && lk + q * KT < left;
          copy4(xd + (uint32_t)(q * KT * TPX) * 4u, on ? s : x, on ? 4 : 0);
          s += KT * plane;
        }
      }
      xsrc += KS * plane;
      s = wsrc;
#pragma unroll
      for (int q = 0; q < TF / FQ; ++q) {
        const bool on = co0 + wf + q * FQ < Co && wk < left;
        copy4(wd + (uint32_t)(q * FQ) * 4u, on ? s : w, on ? 4 : 0);
        s += (size_t)FQ * C;
      }
      wsrc += KS;
    }
    if (++fbuf == ST) fbuf = 0;
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // acc[i][j][0] = (x0 w0, x1 w1), acc[i][j][1] = (x0 w1, x1 w0) for pixel pair i and filter pair j
  unsigned long long acc[PT / 2][FT / 2][2];
#pragma unroll
  for (int i = 0; i < PT / 2; ++i)
#pragma unroll
    for (int j = 0; j < FT / 2; ++j) acc[i][j][0] = acc[i][j][1] = 0ull;
#pragma unroll
  for (int s = 0; s < ST - 1; ++s) fetch(s);
  const int nsteps = (C + KS - 1) / KS;
  int cur = 0;
  for (int step = 0; step < nsteps; ++step) {
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
    __syncthreads();                       // the step's operands are here, everybody has left the last one's
    fetch(step + ST - 1);
    const float *xt = xs + cur * (KS * TPX) + tx * (PT >= 4 ? 4 : 2), *wt = ws + cur * (KS * WP) + ty * FT;
    if (++cur == ST) cur = 0;
#pragma unroll
    for (int k = 0; k < KS; ++k) {
      unsigned long long xv[PT / 2], wv[FT / 2];
      if constexpr (PT >= 4) {
#pragma unroll
        for (int h = 0; h < PT / 4; ++h) {
          const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(xt + k * TPX + 64 * h);
          xv[2 * h] = a.x; xv[2 * h + 1] = a.y;
        }
      } else {
        xv[0] = *reinterpret_cast<const unsigned long long *>(xt + k * TPX);
      }
      if constexpr (FT >= 4) {
#pragma unroll
        for (int h = 0; h < FT / 4; ++h) {
          const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(wt + k * WP + 4 * h);
          wv[2 * h] = a.x; wv[2 * h + 1] = a.y;
        }
      } else {
        wv[0] = *reinterpret_cast<const unsigned long long *>(wt + k * WP);
      }
#pragma unroll
      for (int j = 0; j < FT / 2; ++j) {
        const unsigned long long wx = swapped(wv[j]);
#pragma unroll
        for (int i = 0; i < PT / 2; ++i) {
          acc[i][j][0] = fma2(xv[i], wv[j], acc[i][j][0]);
          acc[i][j][1] = fma2(xv[i], wx, acc[i][j][1]);
        }
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  // runs of 4 (2) consecutive pixels of the flat index: one image and aligned when H_out*W_out is a
  // multiple of their number, else each pixel finds its own image
  constexpr int RUN = PT >= 4 ? 4 : 2;
#pragma unroll
  for (int h = 0; h < PT / RUN; ++h) {
    const long long gp = op0 + 64 * h + tx * RUN;
    if (gp >= total_pix) continue;
    const long long n0 = gp / HoWo;
    const int p0 = (int)(gp - n0 * HoWo);
    // the run's pixels in the plane of the thread's first filter, formed once: per filter and pixel these
    // divisions and products were most of an odd plane's time at few channels (4 channels,
    // 37x37, 208 filters, stride 2, 162 images 48.5 -> 23.9 us; 92 drawn shapes 0.49 to 1.02)
    float *const dst0 = out + ((size_t)n0 * Co + co0 + ty * FT) * HoWo + p0;
    const bool whole = HoWo % RUN == 0;
    float *dst[RUN];
    if (!whole) {
#pragma unroll
      for (int i = 0; i < RUN; ++i) {
        const long long ni = p0 + i < HoWo ? n0 : (gp + i) / HoWo;
        dst[i] = gp + i < total_pix ? out + ((size_t)ni * Co + co0 + ty * FT) * HoWo + (gp + i - ni * HoWo) : nullptr;
      }
    }
#pragma unroll
    for (int j = 0; j < FT; ++j) {
      const int co = co0 + ty * FT + j;
      if (co >= Co) continue;
      float v[RUN];
#pragma unroll
      for (int i = 0; i < RUN / 2; ++i) {
        const float2 a = halves(acc[h * (RUN / 2) + i][j / 2][0]), b = halves(acc[h * (RUN / 2) + i][j / 2][1]);
        v[2 * i] = (j & 1) ? b.x : a.x;
        v[2 * i + 1] = (j & 1) ? a.y : b.y;
      }
      const size_t plane_off = (size_t)j * HoWo;
      if (whole) {
        if constexpr (RUN == 4) *reinterpret_cast<float4 *>(dst0 + plane_off) = make_float4(v[0], v[1], v[2], v[3]);
        else *reinterpret_cast<float2 *>(dst0 + plane_off) = make_float2(v[0], v[1]);
      } else {
#pragma unroll
        for (int i = 0; i < RUN; ++i)
          if (dst[i] != nullptr) dst[i][plane_off] = v[i];
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
  // Tiles: 128 pixels x 64 filters use the fp32 pipe best; 64 x 32 and 32 x 16 spread a projection of few
  // pixels over more SMs.  The choice is the shortest time of the SM with the most blocks, from the
  // cycles a channel takes (with the SM to itself, and as one of several blocks).
  const long long sms = sm_count_of_current_device();
  auto cost = [&](int tpx, int tf, double alone, double shared) {
    const long long blocks = (total_pix + tpx - 1) / tpx * ((Co + tf - 1) / tf);
    return std::max(alone, (double)((blocks + sms - 1) / sms) * shared);
  };
  const double big = cost(128, 64, 130, 90), mid = cost(64, 32, 60, 38), small = cost(32, 16, 40, 18);
  if (big <= mid && big <= small) return launch_tiles<8, 8, 16, 3>(x, w, C, H, W, Co, stride, Ho, Wo, total_pix, out, st);
  if (mid <= small) return launch_tiles<4, 4, 32, 3>(x, w, C, H, W, Co, stride, Ho, Wo, total_pix, out, st);
  return launch_tiles<2, 2, 32, 4>(x, w, C, H, W, Co, stride, Ho, Wo, total_pix, out, st);
}

}  // namespace xnor
