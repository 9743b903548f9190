// Binary-Weight-Network convolution (Section 3.1, Eq. 1): I * W ~ (I (+) B) alpha with real
// inputs and B = sign(W), on the 5th-generation tensor cores.
//
// The inputs are rounded once to bfloat16 and laid out as the "pixel stream" the XNOR kernel
// uses (every input row preceded by lead zero pixels, every image by lead zero rows, one
// stream per stride phase), but materialised in memory with the padding written as zeros, one plane
// per eight channels:
//   x_stream  bf16 [phases][Cp / 8][L][8],  L = N*Hq*Wq stream positions, Cp = C rounded up to 32;
// plane 4 w + q holds channels 32 w + 4 q + i and 32 w + 16 + 4 q + i (i = 0..3) at elements 2 i and
// 2 i + 1 (the order in which a packed word of filter signs expands with two operations per register).
// With GEMM row m = stream position of an output pixel, tap (ky,kx) reads position
// m + shift(ky,kx) of one phase: a CTA fetches the ppix = 128 + halo positions a tile touches
// ONCE, one contiguous bulk copy per plane: shared memory then holds [plane][position][16 bytes], the
// no-swizzle K-major operand layout, and every tap's A operand is that patch at a shifted start address.
// (With the channels innermost in memory a patch came in as 16-byte pieces of a tiled tensor copy.)
//
// B operand: the packed sign words of a slab of NT filters, expanded by producer warps into
// +-1 bfloat16 rows in a ring of stages (one K-step of 16 channels = two 16-byte pieces of a
// filter row).  tcgen05.mma kind::f16 (bf16 x bf16, fp32 accumulation in tensor memory): every
// product is +-x exactly; only the fp32 accumulation rounds.
//
// Roles (768 threads, persistent, one CTA per SM, items = (pixel tiles, filter slab) in tile-major
// order, a contiguous range per CTA): warps 0-7 epilogue (D * alpha (+ residual) -> NCHW; two
// warps per quarter of the lanes, taking alternate groups of 16 columns), warps 8 and 16 issue the MMAs,
// warp 12 the bulk copies, and the twelve warps 9-11, 13-15, 17-19, 21-23 expand weights (three groups of
// four, every third stage each).  Warp w runs on scheduler w % 4: the expansion stays off scheduler 0,
// whose instruction cache then holds the loop of the issuing threads, the path everything waits for.
// Every wait is bounded; on expiry the CTA records XNOR_ERR_TIMEOUT, stops, and frees its tensor memory.
#include <cuda_bf16.h>

#include <algorithm>

#include "bgrad.cuh"
#include "umma_common.cuh"

namespace xnor {

__device__ int g_status_bwn = 0;

namespace {

using namespace umma;

constexpr int kEpiWarps = 8;          // two per quarter of the tensor-memory lanes
constexpr int kMmaWarp = 8, kMma2Warp = 16;
constexpr int kTmaWarp = 12;
constexpr int kWgtGroups = 3, kWgtWarps = 4;     // groups of four warps
constexpr int kThreads = 768;                    // 24 warps, 80 registers each
constexpr int kTileM = 128;
constexpr int kTmemCols = 512;
constexpr int kMaxAcc = 4;
constexpr int kMaxStages = 8;
constexpr int kMaxPatchBufs = 3;
constexpr int kMaxTaps = 121;
constexpr size_t kCtrlBytes = 1024;
constexpr size_t kSmemMax = 232448 - 1024;

struct BwnParams {
  const uint8_t *xs;           // x_stream
  const uint32_t *wp;
  const float *alpha, *residual;
  float *out;
  int N, C, H, W, Co, kh, kw, stride, pad, Ho, Wo, Cw;
  int Cp;                      // channels padded to 32
  int Hq, Wq, leadY, leadX;
  long long L;
  int ntiles, nslabs, NT, nacc, ppix, npb, stages, ntaps, phases;
  int nwords, wps;             // packed words per filter row; words per weight stage
  int tpi;                     // pixel tiles per work item (1 or 2): every weight stage then serves
                               // tpi MMAs, so the filter rows are expanded once per tpi * 128 pixels;
                               // ntiles counts items' worth of tiles (groups of tpi stream tiles)
  int rows_mod;
  uint32_t plane_bytes, phase_bytes, patch_bytes, stage_bytes;
  uint32_t off_vec, off_ring, off_patch;
  int vec_len;
  uint32_t idesc;
  int relu;
  uint32_t tap_lo[kMaxTaps + 1];   // per tap: start of its A operand inside a patch, in 16-byte units
  uint32_t div_wq_m, div_hq_m;
  int div_wq_s, div_hq_s;
};

__device__ __forceinline__ uint32_t fast_div(uint32_t n, uint32_t m, int s) {
  return (uint32_t)(((uint64_t)n * m) >> (31 + s));
}

__device__ __forceinline__ uint32_t elect_one() {
  uint32_t pred = 0;
  asm volatile(
      "{\n\t.reg .b32 rx;\n\t.reg .pred px;\n\t"
      "elect.sync rx|px, %1;\n\t"
      "@px mov.s32 %0, 1;\n\t}"
      : "+r"(pred) : "r"(0xFFFFFFFFu));
  return pred;
}

// One MMA of 128 x NT x 16 (bf16).  One elected lane of the issuing warp runs the whole issue
// loop (a predicate per MMA in a converged warp costs a divergence each time).
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi,
                                          uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %2};\n\t"
      "mov.b64 db, {%3, %4};\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void commit_one(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(bar) : "memory");
}

__device__ __forceinline__ float4 lds_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float lds_f(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}

struct Smem {
  uint32_t wfull, wempty, pfull, pempty, afull, aempty;
  uint32_t *tmem_slot;
  volatile int *abort_flag;
  uint32_t ring, patch, alpha;
};

__device__ __forceinline__ Smem carve(uint8_t *smem, const BwnParams &P) {
  Smem s;
  const uint32_t base = smem_u32(smem);
  s.wfull = base;
  s.wempty = s.wfull + 8u * kMaxStages;
  s.pfull = s.wempty + 8u * kMaxStages;
  s.pempty = s.pfull + 8u * kMaxPatchBufs;
  s.afull = s.pempty + 8u * kMaxPatchBufs;
  s.aempty = s.afull + 8u * kMaxAcc;
  s.tmem_slot = reinterpret_cast<uint32_t *>(smem + 8 * (2 * kMaxStages + 2 * kMaxPatchBufs + 2 * kMaxAcc));
  s.abort_flag = reinterpret_cast<volatile int *>(s.tmem_slot + 1);
  s.ring = base + P.off_ring;
  s.patch = base + P.off_patch;
  s.alpha = base + P.off_vec;
  return s;
}

__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
  return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, abort_flag, &g_status_bwn));
}

// ------------------------------------------------------------------ MMA issuer (one thread)
// Issues the MMAs of pixel tile `which` of every item: the items' second tile has a warp of its own (one
// thread issues an MMA in 60 to 85 cycles beside the other roles, the tensor core takes 64; both read the
// same filter rows, into different accumulators).  What can be is kept in registers, a stage's barrier
// is polled before the MMAs of the stage before it, and two words are issued in straight-line code.
__device__ void mma_loop(const BwnParams &P, const Smem &S, long long i0, long long i1,
                         uint32_t tmem_base, uint32_t which) {
  const int wps = P.wps, nwords = P.nwords, Cw = P.Cw, nslabs = P.nslabs;
  const uint32_t NT = (uint32_t)P.NT, idesc = P.idesc, stages = (uint32_t)P.stages;
  const uint32_t b_lbo = NT * 16u;
  const uint32_t hi = (128u >> 4) | (1u << 14);           // 128 B between 8-row groups; version
  const uint32_t a_lbo_hi = (P.plane_bytes >> 4) << 16;    // the K-step's second piece: next plane
  const uint32_t b_lo0 = ((S.ring & 0x3FFFFu) >> 4) | ((b_lbo >> 4) << 16);
  const uint32_t b_step = (2u * b_lbo) >> 4;               // next K-step
  const uint32_t a_step = (2u * P.plane_bytes) >> 4;       // next 16 channels of the same tap
  const uint32_t stage_step = P.stage_bytes >> 4;
  uint32_t ws = 0u, wph = 0u, pph = 0u, aph = 1u;
  int pb = 0, ab = 0;
  int slab = (int)(i0 % nslabs);
  bool new_tile = true, ready = false;
  uint32_t patch_lo = 0;
  const uint32_t nitems = (uint32_t)(i1 - i0);
  for (uint32_t it = 0; it < nitems; ++it) {
    if (new_tile) {
      if (!mbar_wait(S.pfull + 8u * pb, pph, S.abort_flag, &g_status_bwn)) return;
      // the second tile is the same patch 128 positions (128 x 16 bytes) further
      patch_lo = ((((S.patch + (uint32_t)pb * P.patch_bytes) & 0x3FFFFu) >> 4) + which * (uint32_t)kTileM) | a_lbo_hi;
    }
    if (!mbar_wait(S.aempty + 8u * ab, aph, S.abort_flag, &g_status_bwn)) return;
    tc_fence_after();
    const uint32_t d_tmem = tmem_base + ((uint32_t)(ab * P.tpi) + which) * NT;
    // word f = tap * Cw + cw is two K-steps; addresses stay below 2^18: no carry into the offset field
    int tap = 0, cw = 0;
    uint32_t a = patch_lo + P.tap_lo[0], a_next = patch_lo + P.tap_lo[1], acc = 0u;
    auto next_word = [&]() {
      const uint32_t cur = a;
      a += 2u * a_step;
      if (++cw == Cw) { cw = 0; a = a_next; ++tap; a_next = patch_lo + P.tap_lo[min(tap + 1, kMaxTaps)]; }
      return cur;
    };
    auto step = [&](uint32_t av, uint32_t b, uint32_t accumulate) {
      umma_bf16(d_tmem, av, hi, b, hi, idesc, accumulate);
    };
    for (int left = nwords; left > 0; left -= wps) {
      if (!ready && !mbar_wait(S.wfull + 8u * ws, wph, S.abort_flag, &g_status_bwn)) return;
      uint32_t b = b_lo0 + ws * stage_step;
      uint32_t nws = ws + 1u, nph = wph;
      if (nws == stages) { nws = 0u; nph ^= 1u; }
      ready = mbar_try(S.wfull + 8u * nws, nph);
      int n = min(wps, left);
#pragma unroll 1
      for (; n >= 2; n -= 2) {
        const uint32_t a0 = next_word(), a1 = next_word();
        step(a0, b, acc);
        step(a0 + a_step, b + b_step, 1u);
        step(a1, b + 2u * b_step, 1u);
        step(a1 + a_step, b + 3u * b_step, 1u);
        acc = 1u;
        b += 4u * b_step;
      }
      if (n > 0) {
        const uint32_t a0 = next_word();
        step(a0, b, acc);
        step(a0 + a_step, b + b_step, 1u);
        acc = 1u;
      }
      commit_one(S.wempty + 8u * ws);
      ws = nws;
      wph = nph;
    }
    new_tile = false;
    if (++slab == nslabs) { slab = 0; new_tile = true; }
    commit_one(S.afull + 8u * ab);
    if (new_tile || it + 1 == nitems) commit_one(S.pempty + 8u * pb);
    if (new_tile) { if (++pb == P.npb) { pb = 0; pph ^= 1u; } }
    if (++ab == P.nacc) { ab = 0; aph ^= 1u; }
  }
}

__device__ __forceinline__ void mma_role(const BwnParams &P, const Smem &S, long long i0, long long i1,
                                         uint32_t tmem_base, uint32_t which) {
  if (elect_one()) mma_loop(P, S, i0, i1, tmem_base, which);
  __syncwarp();
}

// ------------------------------------------------------------------ patch producer (one warp)
__device__ void tma_role(const BwnParams &P, const Smem &S, long long i0, long long i1, int lane) {
  const int tile0 = (int)(i0 / P.nslabs);
  const uint32_t npatches = (uint32_t)((i1 - 1) / P.nslabs) - (uint32_t)tile0 + 1u;
  const int nplanes = P.phases * (P.Cp / 8);
  bool ok = true;
  uint32_t started = 0;
  for (uint32_t seq = 0; seq < npatches && ok; ++seq) {
    const uint32_t pb = seq % (uint32_t)P.npb, use = seq / (uint32_t)P.npb;
    ok = wait_warp(S.pempty + 8u * pb, (use & 1u) ^ 1u, S.abort_flag);
    if (!ok) break;
    // positions of the patch inside the stream; those beyond it are the padding below and right of the
    // last image: zeros
    const long long pos = (long long)(tile0 + (int)seq) * P.tpi * kTileM;
    const uint32_t bytes = (uint32_t)min((long long)P.ppix, P.L - pos) * 16u;
    const uint32_t bar = S.pfull + 8u * pb, dst = S.patch + pb * P.patch_bytes;
    if (bytes < P.plane_bytes) {
      for (int pl = 0; pl < nplanes; ++pl)
        for (uint32_t b = bytes + (uint32_t)lane * 16u; b < P.plane_bytes; b += 512u)
          sts128(dst + (uint32_t)pl * P.plane_bytes + b, 0u, 0u, 0u, 0u);
      fence_proxy_async();
      __syncwarp();
    }
    if (lane == 0) mbar_arrive_expect_tx(bar, bytes * (uint32_t)nplanes);
    __syncwarp();
    for (int pl = lane; pl < nplanes; pl += 32)
      bulk_copy_g2s(dst + (uint32_t)pl * P.plane_bytes, P.xs + ((size_t)pl * (size_t)P.L + (size_t)pos) * 16u, bytes, bar);
    __syncwarp();
    started = seq + 1u;
  }
  if (!ok && started > 0u) {
    // gave up: the copies started last must land before the CTA's shared memory is released
    for (uint32_t back = 1; back <= (uint32_t)P.npb && back <= started; ++back) {
      const uint32_t c = started - back;
      for (int i = 0; i < (1 << 20) &&
                      !mbar_try(S.pfull + 8u * (c % (uint32_t)P.npb), (c / (uint32_t)P.npb) & 1u); ++i) {}
    }
  }
}

// ------------------------------------------------------------------ weight producers (12 warps)
// A packed word (32 sign bits, a set bit is +1) -> 16 registers of two bfloat16 +-1 (0x3F80 / 0xBF80):
// register r holds channel r in its low half and channel r + 16 in its high one, so that a shift brings
// both signs to their places: two operations per register.  `inv` is the complemented word.
__device__ __forceinline__ uint32_t expand_pair(uint32_t inv, int r) {
  return ((r <= 15 ? inv << (15 - r) : inv) & 0x80008000u) | 0x3F803F80u;
}

// A stage holds wps packed words of NT filter rows: word i in pieces 4 i .. 4 i + 3 of NT x 16 bytes (two
// K-steps).  The groups of four warps take the stages of the sequence over all items in turn; a thread
// expands up to two words of one row per stage.  Its words of the group's next stage are fetched ahead:
// the filters are re-read (from L2) for every work item.
__device__ void weight_role(const BwnParams &P, const Smem &S, long long i0, long long i1, int group, int t, int lane) {
  constexpr int kU = 2;
  const int nst = (P.nwords + P.wps - 1) / P.wps;
  const int row = t % P.rows_mod, sub = t / P.rows_mod, subs = 32 * kWgtWarps / P.rows_mod;   // words sub, sub + subs of a stage
  const uint32_t b_lbo = (uint32_t)P.NT * 16u;
  struct Cursor { long long it; int st, slab; };
  auto advance = [&](Cursor &c, int by) {
    c.st += by;
    while (c.st >= nst) {
      c.st -= nst;
      ++c.it;
      if (++c.slab == P.nslabs) c.slab = 0;
    }
  };
  auto fetch = [&](const Cursor &c, uint32_t w[kU]) {
    const int co = c.slab * P.NT + row;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int wl = sub + u * subs, f = c.st * P.wps + wl;
      w[u] = row < P.NT && wl < P.wps && c.it < i1 && f < P.nwords && co < P.Co ? load_global(P.wp + packed_weight_index(P.Co, co, f)) : 0u;
    }
  };
  Cursor c{i0, 0, (int)(i0 % P.nslabs)};
  advance(c, group);
  uint32_t cur[kU], nxt[kU];
  fetch(c, cur);
  uint32_t ws = (uint32_t)group, wph = 1u;             // stages >= groups (host)
  const uint32_t off = (uint32_t)row * 16u + (uint32_t)(4 * sub) * b_lbo;
#pragma unroll 1
  while (c.it < i1) {
    advance(c, kWgtGroups);
    fetch(c, nxt);
    if (!mbar_wait_relaxed(S.wempty + 8u * ws, wph, S.abort_flag, &g_status_bwn, 50)) return;
    const uint32_t a = S.ring + ws * P.stage_bytes + off;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      if (row < P.NT && sub + u * subs < P.wps) {
        const uint32_t inv = ~cur[u], au = a + (uint32_t)(4 * u * subs) * b_lbo;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          sts128(au + (uint32_t)q * b_lbo, expand_pair(inv, 4 * q), expand_pair(inv, 4 * q + 1), expand_pair(inv, 4 * q + 2),
                 expand_pair(inv, 4 * q + 3));
      }
    }
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) mbar_arrive(S.wfull + 8u * ws);
    ws += kWgtGroups;
    if (ws >= (uint32_t)P.stages) { ws -= (uint32_t)P.stages; wph ^= 1u; }
#pragma unroll
    for (int u = 0; u < kU; ++u) cur[u] = nxt[u];
  }
}

// ------------------------------------------------------------------ epilogue (8 warps)
// A warp reads tensor-memory lanes 32 q .. + 31 (stream positions) of its quarter q and the
// groups of 16 columns (filters) e, e + 2, ...; for one filter a warp stores 32 consecutive
// pixels of the NCHW output.
__device__ void epilogue_role(const BwnParams &P, const Smem &S, long long i0, long long i1,
                              uint32_t tmem_base, int quarter, int e, int lane) {
  const int b_end = P.NT / 16;
  const int nk = (b_end - e + 1) / 2;                 // groups of this warp per item
  const size_t HoWo = (size_t)P.Ho * P.Wo;
  const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
  const bool relu = P.relu != 0;
  int tile = (int)(i0 / P.nslabs), slab = (int)(i0 - (long long)tile * P.nslabs);
  struct Pix { bool valid; size_t obase; };
  auto decode = [&](int t) {
    Pix px{false, 0};
    const uint32_t m = (uint32_t)t * kTileM + (uint32_t)(quarter * 32 + lane);
    if (m < (uint32_t)P.L) {
      const uint32_t r = fast_div(m, P.div_wq_m, P.div_wq_s);
      const int ox = (int)(m - r * (uint32_t)P.Wq);
      const uint32_t n = fast_div(r, P.div_hq_m, P.div_hq_s);
      const int oy = (int)(r - n * (uint32_t)P.Hq);
      if (ox < P.Wo && oy < P.Ho) {
        px.valid = true;
        px.obase = (size_t)n * P.Co * HoWo + (size_t)oy * P.Wo + ox;
      }
    }
    return px;
  };
  int ab = 0;
  uint32_t fph = 0;
  bool ok = true;
  const uint32_t nitems = (uint32_t)(i1 - i0);
  for (uint32_t it = 0; it < nitems && ok; ++it) {
    ok = mbar_wait_relaxed(S.afull + 8u * ab, fph, S.abort_flag, &g_status_bwn, 200);
    if (!ok) break;
    tc_fence_after();
    const int co0 = slab * P.NT;
    if (nk == 0) {                               // a slab of 16 filters: nothing for the second warp
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(S.aempty + 8u * ab);
    }
   for (int tt = 0; tt < P.tpi && nk > 0; ++tt) {   // the item's pixel tiles, one accumulator each
    const Pix px = decode(tile * P.tpi + tt);
    const bool last_tile = tt + 1 == P.tpi;
    const uint32_t t_acc = t_lane + (uint32_t)((ab * P.tpi + tt) * P.NT);
    int32_t cur[16];
#pragma unroll 1
    for (int k = 0; k < nk; ++k) {
      const int b = e + 2 * k;
      __syncwarp();
      tmem_ld16(t_acc + (uint32_t)(b * 16), cur);
      tmem_wait16(cur);
      if (k + 1 == nk && last_tile) {            // last load of the item done: release its accumulators
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(S.aempty + 8u * ab);
      }
      if (!px.valid) continue;
      const int co = co0 + b * 16;
      const size_t o0 = px.obase + (size_t)co * HoWo;
      if (co + 16 <= P.Co && P.residual == nullptr && HoWo < ((size_t)1 << 27)) {
        // whole group, no residual: 32-bit offsets from one pointer
        float *op = P.out + o0;
        const uint32_t howo = (uint32_t)HoWo;
#pragma unroll
        for (int j4 = 0; j4 < 4; ++j4) {
          const float4 al = lds_f4(S.alpha + (uint32_t)(co * 4 + j4 * 16));
          const float a4[4] = {al.x, al.y, al.z, al.w};
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const float v = __fmul_rn(__int_as_float(cur[j4 * 4 + jj]), a4[jj]);
            op[(uint32_t)(j4 * 4 + jj) * howo] = relu ? fmaxf(v, 0.0f) : v;
          }
        }
        continue;
      }
      float res[16];
      if (P.residual != nullptr) {
#pragma unroll
        for (int j = 0; j < 16; ++j) res[j] = co + j < P.Co ? P.residual[o0 + (size_t)j * HoWo] : 0.0f;
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (co + j < P.Co) {
          float v = __fmul_rn(__int_as_float(cur[j]), lds_f(S.alpha + (uint32_t)((co + j) * 4)));
          if (P.residual != nullptr) v += res[j];
          if (relu) v = fmaxf(v, 0.0f);
          P.out[o0 + (size_t)j * HoWo] = v;
        }
      }
    }
   }
    if (++slab == P.nslabs) { slab = 0; ++tile; }
    if (++ab == P.nacc) { ab = 0; fph ^= 1u; }
  }
}

__global__ void __launch_bounds__(kThreads, 1)
bwn_conv_kernel(const __grid_constant__ BwnParams P) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Smem S = carve(smem, P);
  if (tid == 0) {
    for (int i = 0; i < kMaxStages; ++i) {
      mbar_init(S.wfull + 8u * i, kWgtWarps);
      mbar_init(S.wempty + 8u * i, (uint32_t)P.tpi);           // a commit of every issuing warp
    }
    for (int i = 0; i < kMaxPatchBufs; ++i) {
      mbar_init(S.pfull + 8u * i, 1);
      mbar_init(S.pempty + 8u * i, (uint32_t)P.tpi);
    }
    for (int i = 0; i < kMaxAcc; ++i) {
      mbar_init(S.afull + 8u * i, (uint32_t)P.tpi);
      mbar_init(S.aempty + 8u * i, kEpiWarps);
    }
    *S.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(S.tmem_slot)), "r"((uint32_t)kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // the tensor memory is taken before any thread lets the next kernel start: a block of that kernel on this
  // SM could take it first, and then waits for this one
  __syncthreads();
  stream_order();
  for (int i = tid; i < P.vec_len; i += kThreads)
    reinterpret_cast<float *>(smem + P.off_vec)[i] =
        i < P.Co ? (P.alpha != nullptr ? load_global(P.alpha + i) : 1.0f) : 0.0f;   // no alpha: unit scale
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *S.tmem_slot;

  const long long total = (long long)P.ntiles * P.nslabs;
  const long long i0 = total * blockIdx.x / gridDim.x;
  const long long i1 = total * (blockIdx.x + 1) / gridDim.x;
  if (i0 < i1) {
    if (warp < kEpiWarps) epilogue_role(P, S, i0, i1, tmem_base, warp & 3, warp >> 2, lane);
    else if (warp == kMmaWarp) mma_role(P, S, i0, i1, tmem_base, 0u);
    else if (warp == kMma2Warp) { if (P.tpi == 2) mma_role(P, S, i0, i1, tmem_base, 1u); }
    else if (warp == kTmaWarp) tma_role(P, S, i0, i1, lane);
    else if ((warp & 3) != 0) {
      const int wi = ((warp >> 2) - 2) * 3 + (warp & 3) - 1;           // 0 .. 11
      weight_role(P, S, i0, i1, wi / kWgtWarps, 32 * (wi % kWgtWarps) + lane, lane);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 ::"r"(tmem_base), "r"((uint32_t)kTmemCols) : "memory");
}

// ------------------------------------------------------------------ input preparation
// fp32 NCHW (after the optional BatchNorm affine) -> the bf16 stream, zeros at padding positions and in
// channels C .. Cp - 1.  Thread = stream position, kPrepPlanes planes of eight channels: every load of a
// warp runs along consecutive input pixels, every store is 512 contiguous bytes, nothing is transposed.
// HBM bounds it.
constexpr int kPrepPlanes = 4;                // planes per block: one group of 32 channels

// All 32 loads of a thread are in flight before the first is used: 256 channels, 14x14, 256 images
// 15.9 -> 14.5 us (HBM: 11.8), 64 channels, 56x56, 128 images 28.9 -> 25.2 (23.6).
constexpr int kPrepThreads = 128;

template <bool kGrad>
__global__ void __launch_bounds__(kPrepThreads, 6)
bwn_prepare_kernel(const float *x, const float *scale,
                   const float *shift, const float *gmax, int C, int H,
                   int W, int s, int Hq, int Wq, int leadY, int leadX, long long L, int Cp, int ngroups,
                   uint4 *__restrict__ xs) {
  stream_order();
  const int phase = (int)(blockIdx.y / (unsigned)ngroups), grp = (int)blockIdx.y - phase * ngroups;
  __shared__ __align__(16) float factor[2][32];            // scale and shift of the block's channels
  if (threadIdx.x < 32 && scale != nullptr) {
    const int ch = grp * 32 + threadIdx.x;
    factor[0][threadIdx.x] = ch < C ? load_global(scale + ch) : 0.0f;
    factor[1][threadIdx.x] = !kGrad && ch < C ? load_global(shift + ch) : 0.0f;
  }
  __syncthreads();
  const long long m = (long long)blockIdx.x * kPrepThreads + threadIdx.x;
  if (m >= L) return;
  const int py = phase / s, px = phase - py * s;
  const uint32_t mu = (uint32_t)m, r = mu / (uint32_t)Wq, c = mu - r * (uint32_t)Wq, n = r / (uint32_t)Hq;   // L < 2^31
  const int ry = (int)(r - n * (uint32_t)Hq);
  const int iy = (ry - leadY) * s + py, ix = ((int)c - leadX) * s + px;
  const bool real = ry >= leadY && (int)c >= leadX && iy < H && ix < W;
  const size_t plane = (size_t)H * W;
  const int c0 = grp * 32;
  const float *src = x + ((size_t)n * C + c0) * plane + (size_t)iy * W + ix;
  const float gm = kGrad && real ? load_global(gmax + n) : 0.0f;    // the scale of this position's image
  uint4 *dst = xs + ((size_t)(phase * (Cp / 8) + grp * kPrepPlanes) * (size_t)L + (size_t)m);
  const bool whole = c0 + 32 <= C;
  float values[kPrepPlanes][8];
#pragma unroll
  for (int q = 0; q < kPrepPlanes; ++q)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int ch = 4 * q + (j & 3) + 16 * (j >> 2);
      values[q][j] = load_global_if(src + (size_t)ch * plane, real && (whole || c0 + ch < C));
    }
#pragma unroll
  for (int q = 0; q < kPrepPlanes; ++q) {
    float (&v)[8] = values[q];                // channels c0 + 4 q + i, then c0 + 16 + 4 q + i
    float sc[8], sh[8];
    if (scale != nullptr) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 a = *reinterpret_cast<const float4 *>(&factor[0][16 * h + 4 * q]);
        const float4 b = *reinterpret_cast<const float4 *>(&factor[1][16 * h + 4 * q]);
        sc[4 * h] = a.x; sc[4 * h + 1] = a.y; sc[4 * h + 2] = a.z; sc[4 * h + 3] = a.w;
        sh[4 * h] = b.x; sh[4 * h + 1] = b.y; sh[4 * h + 2] = b.z; sh[4 * h + 3] = b.w;
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (!real) continue;                    // padding stays zero
      if (kGrad) {
        // binarised gradient (Section 3.2, "Binary Gradient"): sign(g) scaled by the image's max|g| and,
        // here, by the filter's alpha (`scale`), the product formed in fp32
        const float p = __fmul_rn(gm, sc[j]);
        v[j] = v[j] >= 0.0f ? p : -p;
      } else if (scale != nullptr) {
        v[j] = __fmaf_rn(sc[j], v[j], sh[j]);
      }
    }
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 b = __floats2bfloat162_rn(v[i], v[i + 4]);       // to nearest even
      w[i] = *reinterpret_cast<const uint32_t *>(&b);
    }
    dst[(size_t)q * (size_t)L] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

struct BwnPlan {
  BwnParams P;
  size_t smem;
  bool ok;
};

// Stream geometry shared by the preparation kernel and the convolution.
struct StreamGeom {
  int s, phases, dymin, dxmin, dymax, dxmax, leadY, leadX, Hq, Wq, Cp;
  long long L;
};

StreamGeom stream_geom(const ConvGeom &g) {
  StreamGeom q;
  q.s = g.stride;
  q.phases = q.s * q.s;
  q.dymin = floor_div(-g.pad, q.s); q.dxmin = floor_div(-g.pad, q.s);
  q.dymax = floor_div(g.kh - 1 - g.pad, q.s); q.dxmax = floor_div(g.kw - 1 - g.pad, q.s);
  q.leadY = -q.dymin; q.leadX = -q.dxmin;
  const int Hc = (g.H + q.s - 1) / q.s, Wc = (g.W + q.s - 1) / q.s;
  const int Hd = std::max(std::max(Hc, g.Ho + q.dymax - q.leadY), g.Ho);
  const int Wd = std::max(std::max(Wc, g.Wo + q.dxmax - q.leadX), g.Wo);
  q.Hq = q.leadY + Hd; q.Wq = q.leadX + Wd;
  q.L = (long long)g.N * q.Hq * q.Wq;
  q.Cp = (g.C + 31) / 32 * 32;      // whole packed words: K-step j is half j & 1 of word j >> 1
  return q;
}

BwnPlan make_plan(const ConvGeom &g) {
  BwnPlan pl{};
  pl.ok = false;
  BwnParams &P = pl.P;
  if (g.stride < 1 || g.stride > 2 || g.Ho < 1 || g.Wo < 1 || g.kh * g.kw > kMaxTaps) return pl;
  const StreamGeom q = stream_geom(g);
  P.N = g.N; P.C = g.C; P.H = g.H; P.W = g.W; P.Co = g.Co; P.kh = g.kh; P.kw = g.kw;
  P.stride = g.stride; P.pad = g.pad; P.Ho = g.Ho; P.Wo = g.Wo; P.Cw = g.Cw;
  P.Cp = q.Cp;
  P.Hq = q.Hq; P.Wq = q.Wq; P.leadY = q.leadY; P.leadX = q.leadX; P.L = q.L;
  P.phases = q.phases;
  P.ntaps = g.kh * g.kw;
  P.nwords = P.ntaps * g.Cw;
  const int halo = (q.dymax - q.dymin) * q.Wq + (q.dxmax - q.dxmin);
  // the window of one tile: 256 positions was the most a tiled copy took; the bulk copies do not need the limit,
  // which stays because no wider window has been tested or timed
  if ((kTileM + halo + 7) / 8 * 8 > 256) return pl;
  if (q.L + 4 * kTileM + 256 >= (1ll << 31)) return pl;
  // filter slabs: as few as fit two accumulators into the tensor-memory columns
  const int max_nt = 128;
  P.nslabs = (g.Co + max_nt - 1) / max_nt;
  P.NT = ((g.Co + P.nslabs - 1) / P.nslabs + 15) / 16 * 16;
  // weight stages: rows_mod threads of a group of warps cover the rows of a word
  int ntp = 16;
  while (ntp < P.NT) ntp *= 2;
  P.rows_mod = ntp;
  P.off_vec = (uint32_t)((kCtrlBytes + 127) / 128 * 128);
  P.vec_len = (g.Co + 15) / 16 * 16 + 256;
  P.off_ring = (uint32_t)((P.off_vec + (size_t)P.vec_len * 4 + 127) / 128 * 128);
  // Two pixel tiles per work item when their common window (256 + halo positions) fits beside two
  // weight stages: the expansion of the filter rows, which bounds the kernel, is then shared by
  // two MMAs.
  const int stream_tiles = (int)((q.L + kTileM - 1) / kTileM);
  const int wps_max = std::min(4, 2 * 32 * kWgtWarps / ntp);   // two words per thread: 2 (128 filters) or 4
  auto stage_of = [&](int wps) { P.wps = wps; P.stage_bytes = (uint32_t)wps * (uint32_t)P.NT * 64u; };
  for (P.tpi = (kTmemCols / P.NT >= 2 && stream_tiles >= 2) ? 2 : 1; P.tpi >= 1; --P.tpi) {
    P.ppix = (P.tpi * kTileM + halo + 7) / 8 * 8;
    P.plane_bytes = (uint32_t)P.ppix * 16u;
    P.phase_bytes = P.plane_bytes * (uint32_t)(P.Cp / 8);
    P.patch_bytes = P.phase_bytes * (uint32_t)P.phases;
    // a stage per group of weight warps at least: shorter ones where the patch leaves little room
    stage_of(wps_max);
    while (P.tpi == 1 && P.wps > 1 && P.off_ring + kWgtGroups * (size_t)P.stage_bytes + P.patch_bytes > kSmemMax)
      stage_of(P.wps / 2);
    if (P.off_ring + (P.tpi == 2 ? 4 : kWgtGroups) * (size_t)P.stage_bytes + P.patch_bytes <= kSmemMax) break;
  }
  if (P.tpi < 1) return pl;
  P.ntiles = (stream_tiles + P.tpi - 1) / P.tpi;
  P.nacc = std::max(1, std::min(kMaxAcc, kTmemCols / (P.NT * P.tpi)));
  const size_t avail = kSmemMax - P.off_ring;
  auto fits = [&](int st, int pb) { return (size_t)st * P.stage_bytes + (size_t)pb * P.patch_bytes <= avail; };
  // a second patch buffer hides the patch copies behind the MMAs and comes before more stages than one
  // per group of weight warps
  int stages = kWgtGroups, npb = 1;
  if (!fits(stages, npb)) return pl;
  while (npb < 2 && fits(stages, npb + 1)) ++npb;
  while (stages < kMaxStages && fits(stages + 1, npb)) ++stages;
  while (npb < kMaxPatchBufs && fits(stages, npb + 1)) ++npb;
  P.stages = stages; P.npb = npb;
  P.off_patch = (uint32_t)((P.off_ring + (size_t)stages * P.stage_bytes + 127) / 128 * 128);
  pl.smem = (size_t)P.off_patch + (size_t)npb * P.patch_bytes;
  if (pl.smem > kSmemMax) return pl;
  // instruction descriptor: D fp32, A and B bf16, both K-major, N = NT, M = 128
  P.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(P.NT >> 3) << 17) |
            ((uint32_t)(kTileM >> 4) << 24);
  for (int tap = 0; tap < P.ntaps; ++tap) {
    const int ky = tap / g.kw, kx = tap - ky * g.kw;
    const int ay = ky - g.pad, ax = kx - g.pad;
    const int dy = floor_div(ay, q.s), dx = floor_div(ax, q.s);
    const int py = ay - dy * q.s, px = ax - dx * q.s;
    const int phase = py * q.s + px;
    const int shift = (dy - q.dymin) * q.Wq + (dx - q.dxmin);
    P.tap_lo[tap] = ((uint32_t)phase * P.phase_bytes + (uint32_t)shift * 16u) >> 4;
  }
  auto magic = [](uint32_t d, uint32_t *m, int *sh) {
    int l = 0;
    while ((1u << l) < d) ++l;
    *sh = l;
    *m = (uint32_t)((((unsigned long long)1 << (31 + l)) + d - 1) / d);
  };
  magic((uint32_t)P.Wq, &P.div_wq_m, &P.div_wq_s);
  magic((uint32_t)P.Hq, &P.div_hq_m, &P.div_hq_s);
  pl.ok = true;
  return pl;
}

}  // namespace

bool bwn_supported(const ConvGeom &g) { return make_plan(g).ok; }

size_t bwn_stream_elems(const ConvGeom &g) {
  if (g.stride < 1 || g.Ho < 1 || g.Wo < 1) return 0;
  const StreamGeom q = stream_geom(g);
  return (size_t)q.phases * (size_t)q.L * (size_t)q.Cp;
}

namespace {

template <bool kGrad>
cudaError_t launch_prepare(const float *x, const float *scale, const float *shift, const float *gmax, const ConvGeom &g,
                           uint16_t *x_stream, cudaStream_t st) {
  const StreamGeom q = stream_geom(g);
  const int ngroups = q.Cp / 32;
  if (q.L >= (1ll << 31) || (long long)ngroups * q.phases > 65535) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)((q.L + kPrepThreads - 1) / kPrepThreads), (unsigned)(ngroups * q.phases));
  return launch_kernel(bwn_prepare_kernel<kGrad>, grid, kPrepThreads, 0, st, 1, x, scale, shift, gmax, g.C, g.H, g.W, q.s, q.Hq, q.Wq,
                       q.leadY, q.leadX, q.L, q.Cp, ngroups, reinterpret_cast<uint4 *>(x_stream));
}

}  // namespace

cudaError_t launch_bwn_prepare(const float *x, const float *scale, const float *shift,
                               const ConvGeom &g, uint16_t *x_stream, cudaStream_t st) {
  return launch_prepare<false>(x, scale, shift, nullptr, g, x_stream, st);
}

cudaError_t launch_bwn_prepare_grad(const float *g, const float *alpha, const float *gmax,
                                    const ConvGeom &gb, uint16_t *g_stream, cudaStream_t st) {
  return launch_prepare<true>(g, alpha, nullptr, gmax, gb, g_stream, st);
}

cudaError_t launch_bwn_conv(const uint16_t *x_stream, const uint32_t *wp, const float *alpha,
                            const float *residual, const ConvGeom &g, float *out, cudaStream_t st) {
  BwnPlan pl = make_plan(g);
  if (!pl.ok) return cudaErrorInvalidValue;
  BwnParams &P = pl.P;
  P.xs = reinterpret_cast<const uint8_t *>(x_stream);
  P.wp = wp; P.alpha = alpha; P.residual = residual; P.out = out;
  P.relu = (g.flags & XNOR_FLAG_RELU) ? 1 : 0;
  static bool attr_flags[64] = {};
  bool &attr_set = attr_done_for_current_device(attr_flags);
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(bwn_conv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSmemMax);
    if (e != cudaSuccess) { (void)cudaGetLastError(); return e; }
    attr_set = true;
  }
  const long long total = (long long)P.ntiles * P.nslabs;
  const unsigned grid = (unsigned)std::min<long long>(total, sm_count_of_current_device());
  return launch_kernel(bwn_conv_kernel, dim3(grid), kThreads, pl.smem, st, 1, P);
}

cudaError_t read_status_bwn(int *status) {
  cudaError_t e = cudaMemcpyFromSymbol(status, g_status_bwn, sizeof(int));
  if (e == cudaSuccess && *status != 0) {
    const int zero = 0;
    e = cudaMemcpyToSymbol(g_status_bwn, &zero, sizeof(int));
  }
  return e;
}

}  // namespace xnor
