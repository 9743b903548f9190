// BinConv on the 5th-generation tensor cores (Eq. 11): persistent,
// warp-specialised implicit GEMM on tcgen05.mma kind::mxf4.
//
// sign(I) (*) sign(W) is an exact integer contraction.  Both operands become
// e2m1 (4-bit) numbers whose products are all +-1, block scales are 1, and the
// fp32 accumulators in tensor memory hold exact integers (|sum| < 2^24).  HBM
// only ever sees the 1-bit packed words; a CTA expands what it needs into
// shared memory.
//
//  GEMM roles.  D[pixel][filter] = sum_k X[pixel][k] * Wt[filter][k]:
//    A (M = 128 rows) = 128 consecutive positions of a virtual pixel stream.
//        For stride s the input is split into s*s phase planes (plane (py,px)
//        holds input pixels (s*r+py, s*c+px)); every plane is laid out as one
//        long stream in which each row is preceded by `lead` zero pixels and
//        each image by `leadY` zero rows.  With GEMM row m = stream index of
//        an output pixel, filter tap (ky,kx) reads, in ONE phase plane, stream
//        position m + shift(ky,kx): a pure shift.  So the pixels a tile
//        touches are expanded ONCE into the no-swizzle K-major operand layout
//        (8 pixels x 16 bytes per core matrix, pixels contiguous, one plane
//        per 32 channels) and every tap's A operand is that patch at a shifted
//        start address.  Zero pixels and the channel tail expand to the value
//        0, so padded taps contribute exactly 0 with no mask or correction.
//        Stream positions that are padding give junk rows that are never stored.
//    B (N = NT rows)  = a slab of NT filters, expanded from bits by producer
//        warps into a ring of shared-memory stages.  One MMA (a K-step, K = 64)
//        consumes two 32-channel pieces; a piece is one packed word (tap,
//        channel word) of a filter row, and K-step j takes words 2j and 2j+1
//        of the row in memory order, so a step may straddle two taps and no
//        step is wasted on channel padding.  The host precomputes, per step,
//        the A-operand descriptor (start of the lower-addressed piece, distance
//        to the other one) and whether the two pieces are swapped.
//
//  Encodings.  A packed word holds 32 sign bits; it becomes 32 e2m1 nibbles in
//  four registers, register r holding channels r, r+4, ..., r+28.  Activations
//  are +-{2, 1, 0.5, 0.5} for r = 0..3, weights +-{0.5, 1, 2, 2}: every product
//  is the product of the two signs.
//
//  Roles (one CTA per SM, CTAs loop over work items = (pixel tile, filter slab)): warps 0-3 epilogue
//  (tensor memory -> registers -> coalesced NCHW stores of D * K * alpha (+ residual)), warp 4 issues the
//  MMAs.  Resident schedule (512 threads): warps 5-12 expand weights, warps 13-15 expand activation
//  patches.  Streaming schedule (768 threads): twelve warps expand weights, or eight with four more
//  draining (items of few K-steps, see make_plan), and three patches; neither weights nor patches are on
//  scheduler 0 (warp w runs on scheduler w % 4), whose instruction cache then holds the loop of the
//  issuing thread, the path everything waits for.
//  Accumulators are multi-buffered in tensor memory so the epilogue of one
//  item overlaps the MMAs of the next.  Every wait is bounded: on expiry the
//  CTA records XNOR_ERR_TIMEOUT in a device status word, stops, frees its
//  tensor memory and exits.
//
//  CTA pairs (kPair kernels, clusters of 2).  One tcgen05.mma.cta_group::2
//  drives the tensor cores of two SMs: M = 256 (each CTA's 128-position tile,
//  patch and tensor memory) and each CTA expands and holds half of a slab's
//  filter rows.  The producers of both CTAs arrive on the barriers of rank 0,
//  whose MMA warp issues; its commits reach the consumer barriers of both.
//
//  Fused BinActiv (kFuse kernels).  The epilogue also applies the next layer's
//  BatchNorm affine to its output values, packs their sign bits along the
//  filters (the next layer's channels) and writes partial sums of |y|.
//
//  Two schedules.  "Resident": when the expanded rows of a filter slab fit in
//  shared memory beside two patches, the slab is expanded ONCE per CTA and the
//  CTA then walks the pixel tiles of that slab (items in slab-major order, one
//  patch per item); the weight warps, idle after the fill, join the epilogue
//  (three warps per quarter of the lanes, taking chunks of the items in turn).  "Streaming":
//  otherwise the weights of every item pass through a ring of stages (items in
//  tile-major order, so that a patch serves all slabs of its tile).
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "drain.cuh"
#include "umma_common.cuh"

namespace xnor {

__device__ int g_status_tc = 0;

// Checking build (-DXNOR_BOUNDS_CHECK): every shared-memory address a producer computes and
// every global index the epilogue stores to is compared with the extent of its buffer; the
// first violation is recorded (its site number) and the access is skipped, so nothing traps.
// In the ordinary build in_bounds() is the constant true and its argument is never evaluated.
#ifdef XNOR_BOUNDS_CHECK
__device__ int g_bounds_tc = 0;
#define in_bounds(cond, site) ((cond) ? true : (atomicCAS(&xnor::g_bounds_tc, 0, (site)), false))
#else
#define in_bounds(cond, site) true
#endif

namespace {

using namespace umma;

// nanoseconds a waiting role sleeps between polls of its barrier
#ifndef XNOR_SLEEP_EPI
#define XNOR_SLEEP_EPI 200
#endif
#ifndef XNOR_SLEEP_PAT
#define XNOR_SLEEP_PAT 200
#endif
#ifndef XNOR_SLEEP_WGT
#define XNOR_SLEEP_WGT 50
#endif

constexpr int kEpiWarps = 4;
constexpr int kMmaWarp = 4;
constexpr int kWgtWarp0 = 5, kWgtWarps = 8;
constexpr int kPatWarp0 = 13, kPatWarps = 3;
constexpr int kThreadsRes = 32 * (kPatWarp0 + kPatWarps);   // 512: 16 warps, 128 registers each
// streaming: weight warps in groups of four, patch warps behind them (see the kernel's role table)
constexpr int kLongItem = 64, kLongFused = 96;   // streaming: K-steps of an item that count as many
constexpr int kPairSteps = 32;       // K-steps from which a pair issues them better (see plan_variant_uncached)
constexpr int kGroupWarps = 4, kThreadsStream = 768;   // 24 warps, 80 registers each
constexpr int kTileM = 128;          // stream positions per tile = tensor-memory lanes
constexpr int kTmemCols = 512;
constexpr int kSfCol = 480;          // columns [480, 512): unit block scales
constexpr int kMaxAccCols = 480;
constexpr int kMaxAcc = 4;           // accumulator buffers
constexpr int kMaxStages = 8;         // ring stages of the streaming schedule
constexpr int kMaxBarStages = 32;    // stage barriers (the resident schedule has one stage per mps K-steps of a row)
constexpr int kEpiSplitMax = 3;      // warps per lane quarter in the resident epilogue
constexpr int kMaxPatchBufs = 4;
constexpr int kMaxRaw = 6;            // raw buffers: up to 2 for each of up to 3 subgroups of patch warps
constexpr int kMaxSteps = 800;       // K-steps (MMAs) per work item (< 1024: swap_mask)
constexpr size_t kCtrlBytes = 1024;
constexpr size_t kSmemMax = 232448 - 1024;

struct TcParams {
  const uint32_t *xp, *wp;
  const float *alpha, *K, *residual;
  float *out;
  int32_t *acc_out;
  int relu;                    // max(v, 0) on every stored value
  float out_scale;             // extra factor of D K alpha (1 unless several calls build one output), folded into the staged alpha
  int acc_shift, acc_accum;    // acc_out receives D << acc_shift, stored or added to its content
  int N, C, H, W, Co, kh, kw, stride, pad, Ho, Wo, Cw;
  int Hq, Wq, leadY, leadX;    // stream geometry of every phase plane
  int dymin, dxmin;
  long long L;                 // stream length N*Hq*Wq
  int ntiles, nslabs, NT;      // pixel tiles, filter slabs, filters per slab (multiple of 16)
  int nacc;                    // accumulator buffers in tensor memory (1 .. 4)
  int ppix;                    // stream positions staged per phase plane (128 + halo, rounded to 8)
  int nplanes;                 // stride*stride*Cw operand planes per patch
  int npb;                     // patch buffers
  int nsteps;                  // K-steps per item
  int mps;                     // K-steps per weight stage
  int stages;
  uint32_t patch_bytes, stage_bytes;
  int rows_mod, grp_steps;     // weight-thread mapping (see weight producer)
  uint32_t off_ring, off_patch, off_raw;  // byte offsets in dynamic shared memory
  uint32_t off_tab;            // streaming: descriptor words of the K-steps in shared memory (0: read from here)
  uint32_t off_vec;            // per-filter vectors staged for the epilogue: alpha, then (fused)
  int vec_len;                 // the next layer's scale and shift; vec_len floats each
  uint32_t raw_bytes;          // size of a raw buffer: the packed input rows a patch can touch, of every bit plane
  uint32_t raw_plane;          // the share of one bit plane
  const uint32_t *xp2;         // two bit planes in one pass: the upper one (see patch_role)
  int nraw;                    // raw buffers per subgroup of patch warps (1 or 2)
  int pat_sub;                 // subgroups of the patch warps (each builds whole patches): 3 or 1
  uint32_t idesc;
  uint32_t tail_mask;          // bits of real channels in the last word
  // Low word of the A-operand descriptor of every K-step (start address relative to the
  // patch in bits 0-13, leading-dimension offset in bits 16-29; the high word is the same
  // for all).  It lives in the kernel parameters so that the MMA issuer reads and offsets
  // it on the uniform datapath: an MMA is as short as 32 cycles, and descriptors that pass
  // through per-thread registers cost more than that to issue.
  uint32_t adesc_lo[kMaxSteps];
  uint32_t swap_mask[32];              // bit j: word 2j+1 is the first piece of step j
  int row_words;               // packed words per filter row = k_h*k_w*Cw
  int pair;                    // 1: two CTAs (a cluster) share every MMA: 256 pixels x NT filters
  int NTh;                     // filter rows of a slab that one CTA expands and holds: NT or NT/2
  // Fused BinActiv of the next layer (kFuse kernels): the epilogue also applies the next
  // BatchNorm affine to its output values, packs their signs along the filters (the next
  // layer's channels) and sums |y| over the filters it handles.
  const float *nscale, *nshift;      // [C_out], both null = identity
  uint32_t *xp_next;                 // u32 [N][Ho][Wo][Cw_next]
  float *A_part;                     // fp32 [nslabs * drain.chunks][N][Ho][Wo]: partial sums of |y|
  int Cw_next;                       // ceil(C_out / 32)
  int resident;                // 1: resident schedule (stages = all stages of a slab)
  int wgt_groups;              // streaming: groups of four warps that expand weights, 3 or 2
  Drain drain;                 // how the warps of a lane quarter drain accumulators
  int any_swap;                // some bit of swap_mask is set
  uint32_t div_wq_m, div_hq_m; // multipliers and shifts of the exact divisions by Wq and Hq
  int div_wq_s, div_hq_s;      // (dividends below 2^31)
  uint32_t div_pg_m, div_g_m;  // the same for the patch units: by phases * ngrp and by ngrp
  int div_pg_s, div_g_s;       // (ngrp = patch_groups())
  uint32_t wq_rcp;             // 2^32 / Wq, rounded up: exact quotients of a patch's positions
  int pat_table;               // a patch touches at most 32 rows of the stream
};

// One MMA.  The issuing warp elects one lane, and that lane alone runs the whole issue loop:
// a predicate per MMA inside a converged warp costs a divergence and a reconvergence each
// time (measured: 95 cycles per MMA against 65 for the single-thread loop, the tensor core
// needing 64 for 128 x 128 x 64).  Descriptors are passed as their two 32-bit halves.
__device__ __forceinline__ void umma_mxf4(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi,
                                          uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                          uint32_t sf, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %2};\n\t"
      "mov.b64 db, {%3, %4};\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.block32 [%0], da, db, %5, [%7], [%7], p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate),
        "r"(sf)
      : "memory");
}

__device__ __forceinline__ void umma_commit_one(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(bar) : "memory");
}

// The same for a CTA pair: one instruction drives the tensor cores of both SMs (M = 256: rows
// 0-127 from this CTA's patch into its tensor memory, rows 128-255 the peer's; each CTA
// supplies half of the N filter rows).  Commits signal the barrier at the same offset in both.
__device__ __forceinline__ void umma_mxf4_pair(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi,
                                               uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                               uint32_t sf, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %2};\n\t"
      "mov.b64 db, {%3, %4};\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::mxf4.block_scale.block32 [%0], da, db, %5, [%7], [%7], p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate),
        "r"(sf)
      : "memory");
}

__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .b16 mask;\n\t"
      "mov.b16 mask, 3;\n\t"
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], mask;\n\t}"
      ::"r"(bar) : "memory");
}

template <bool kPair>
__device__ __forceinline__ void umma_issue(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi,
                                           uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t sf,
                                           uint32_t accumulate) {
  if (kPair) umma_mxf4_pair(d_tmem, a_lo, a_hi, b_lo, b_hi, idesc, sf, accumulate);
  else umma_mxf4(d_tmem, a_lo, a_hi, b_lo, b_hi, idesc, sf, accumulate);
}

template <bool kPair>
__device__ __forceinline__ void umma_commit_to(uint32_t bar) {
  if (kPair) umma_commit_pair(bar);
  else umma_commit_one(bar);
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

// 32 sign bits -> 32 e2m1 nibbles (sign in bit 3 of a nibble, magnitude code
// 1 = 0.5, 2 = 1, 4 = 2).  Register r holds channels r, r+4, ...; a set bit is +.
// kAct: magnitudes {2, 1, 0.5, 0.5}; otherwise {0.5, 1, 2, 2}.
template <bool kAct>
__device__ __forceinline__ void expand_signs(uint32_t w, uint32_t v[4]) {
  constexpr uint32_t m0 = kAct ? 0xCCCCCCCCu : 0x99999999u;
  constexpr uint32_t m1 = 0xAAAAAAAAu;
  constexpr uint32_t m2 = kAct ? 0x99999999u : 0xCCCCCCCCu;
  constexpr uint32_t m3 = kAct ? 0x99999999u : 0xCCCCCCCCu;
  v[0] = ((w << 3) & 0x88888888u) ^ m0;
  v[1] = ((w << 2) & 0x88888888u) ^ m1;
  v[2] = ((w << 1) & 0x88888888u) ^ m2;
  v[3] = (w & 0x88888888u) ^ m3;
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

// Shift of a filter tap inside a phase plane, and the plane it reads.
inline void tap_geometry(const TcParams &P, int tap, int &phase, int &shift) {
  const int ky = tap / P.kw, kx = tap - ky * P.kw;
  const int ay = ky - P.pad, ax = kx - P.pad;
  // floor division / non-negative remainder by the stride
  const int dy = (ay >= 0) ? ay / P.stride : -((-ay + P.stride - 1) / P.stride);
  const int dx = (ax >= 0) ? ax / P.stride : -((-ax + P.stride - 1) / P.stride);
  const int py = ay - dy * P.stride, px = ax - dx * P.stride;
  phase = py * P.stride + px;
  shift = (dy - P.dymin) * P.Wq + (dx - P.dxmin);
}

// Piece (tap, w) -> byte offset of its A operand inside a patch.
inline uint32_t piece_offset(const TcParams &P, int tap, int w) {
  int phase, shift;
  tap_geometry(P, tap, phase, shift);
  return (uint32_t)(phase * P.Cw + w) * ((uint32_t)P.ppix * 16u) + (uint32_t)shift * 16u;
}

// K-step j: pieces = words 2j and 2j+1 of a filter row (flat index tap*Cw + w).  Returns
// the low descriptor word of its A operand; *swap tells whether word 2j+1 comes first.
inline uint32_t kstep_desc(const TcParams &P, int j, bool *swap) {
  const int f1 = 2 * j, f2 = 2 * j + 1;
  uint32_t o1 = piece_offset(P, f1 / P.Cw, f1 % P.Cw), lbo = 16u;   // lone piece: any in-bounds
  *swap = false;                                                    // partner, its weights are 0
  if (f2 < P.row_words) {
    uint32_t o2 = piece_offset(P, f2 / P.Cw, f2 % P.Cw);
    if (o2 < o1) { const uint32_t o = o1; o1 = o2; o2 = o; *swap = true; }
    lbo = o2 - o1;
  }
  return (o1 >> 4) | ((lbo >> 4) << 16);
}

// Units of channel words at one position of a patch.  Four words come together where they can be loaded as one, and in
// the resident schedule.  Streaming, with fewer registers, other counts of five words and more go one by one, for
// twice as many positions at a time: guarding each of four words for one position was slower than the two
// divisions per unit before it (218 images, 477 channels, 14x14, 400 filters 1x1 stride 2: 25.1 us with the
// divisions, 26.2 guarded, 20.4 now; over 16 drawn shapes 0.97 to 1.10 of the time with the divisions, now 0.81
// to 0.98).  Resident, one by one takes 0.85 to 1.05 of the time; small problems lose.
__host__ __device__ inline int patch_groups(int Cw, bool resident) {
  return !resident && Cw > 4 && (Cw & 3) != 0 ? Cw : (Cw + 3) / 4;
}

// Exact n / d for n < 2^31: q = (n * m) >> (31 + s) with m = ceil(2^(31+s) / d), s = ceil(log2 d).
__device__ __forceinline__ uint32_t fast_div(uint32_t n, uint32_t m, int s) {
  return (uint32_t)(((uint64_t)n * m) >> (31 + s));
}

// Resident schedule: which pixel tiles a CTA (a pair) takes.  The U units of the grid are
// split into one group per filter slab (so a CTA expands one slab, once); inside its group of
// G units, unit g takes tiles g, g + G, g + 2G, ... of the slab: at any moment the CTAs of a
// group write neighbouring runs of every output plane, so the lines that leave the L2
// together lie together in memory (measured on 27x27 planes: 3.9 TB/s of stores against
// 2.85 TB/s when every CTA owns a contiguous range of tiles).
struct ResSched {
  uint32_t ntiles;
  uint32_t slab, g, G;           // this unit's slab, its index in the slab's group, the group's size
  __device__ __forceinline__ uint32_t total() const { return g < ntiles ? (ntiles - g + G - 1u) / G : 0u; }
  __device__ __forceinline__ uint32_t tile(uint32_t seq) const { return g + seq * G; }    // seq < total()
};

__device__ __forceinline__ ResSched res_sched(int ntiles, int nslabs, bool pair) {
  ResSched R;
  const uint32_t unit = pair ? blockIdx.x >> 1 : blockIdx.x;
  const uint32_t units = pair ? gridDim.x >> 1 : gridDim.x;    // >= nslabs (host)
  const uint32_t ns = (uint32_t)nslabs;
  R.ntiles = (uint32_t)ntiles;
  // group s = units [s U / nslabs, (s + 1) U / nslabs)
  R.slab = unit * ns / units;
  while ((R.slab + 1u) * units / ns <= unit) ++R.slab;
  while (R.slab * units / ns > unit) --R.slab;
  const uint32_t g0 = R.slab * units / ns;
  R.g = unit - g0;
  R.G = (R.slab + 1u) * units / ns - g0;
  return R;
}

struct Smem {
  uint32_t wfull, wempty, pfull, pempty, afull, aempty, rawfull, rawdone;   // shared-space addresses of barrier arrays
  uint32_t *tmem_slot;
  volatile int *abort_flag;
  uint32_t ring, patch, raw;                              // shared-space byte addresses
  uint32_t tab;                                           // descriptor words (streaming)
  uint32_t alpha, nscale, nshift;                         // staged per-filter vectors
  uint32_t rank;                                          // CTA rank in its pair (0 = issues the MMAs)
};

__device__ __forceinline__ Smem carve(uint8_t *smem, const TcParams &P) {
  Smem s;
  const uint32_t base = smem_u32(smem);
  s.wfull = base;
  s.wempty = s.wfull + 8u * kMaxBarStages;
  s.pfull = s.wempty + 8u * kMaxBarStages;
  s.pempty = s.pfull + 8u * kMaxPatchBufs;
  s.afull = s.pempty + 8u * kMaxPatchBufs;
  s.aempty = s.afull + 8u * kMaxAcc;
  s.rawfull = s.aempty + 8u * kMaxAcc;
  s.rawdone = s.rawfull + 8u * kMaxRaw;
  s.tmem_slot = reinterpret_cast<uint32_t *>(
      smem + 8 * (2 * kMaxBarStages + 2 * kMaxPatchBufs + 2 * kMaxAcc + 2 * kMaxRaw));
  s.abort_flag = reinterpret_cast<volatile int *>(s.tmem_slot + 1);
  s.ring = base + P.off_ring;
  s.patch = base + P.off_patch;
  s.raw = base + P.off_raw;
  s.tab = base + P.off_tab;
  s.alpha = base + P.off_vec;
  s.nscale = s.alpha + 4u * (uint32_t)P.vec_len;
  s.nshift = s.nscale + 4u * (uint32_t)P.vec_len;
  s.rank = P.pair ? cluster_ctarank() : 0u;
  return s;
}

// ------------------------------------------------------------------ MMA issuer (one thread)
// The MMAs of one full weight stage, unrolled.
template <int MPS, bool kPair>
__device__ __forceinline__ void issue_stage(const TcParams &P, int j0, uint32_t d_tmem,
                                            uint32_t patch_lo, uint32_t a_hi, uint32_t b_lo,
                                            uint32_t b_hi, uint32_t b_step, uint32_t tmem_sf,
                                            uint32_t first) {
#pragma unroll
  for (int jj = 0; jj < MPS; ++jj)
    umma_issue<kPair>(d_tmem, P.adesc_lo[j0 + jj] + patch_lo, a_hi, b_lo + (uint32_t)jj * b_step,
                      b_hi, P.idesc, tmem_sf, jj == 0 ? first : 1u);
}

// All MMAs of an item whose filter rows are already in shared memory (resident schedule, every
// item but the first).  The stages of the ring are contiguous, so K-step j reads its filter
// rows at b_lo0 + j b_step.  The patch descriptors of a batch of K-steps are fetched together
// and the batch is issued in straight-line code: per MMA two additions and the instruction,
// no load on its path (the stage-by-stage loop below needs ~100 cycles per MMA next to the
// other roles, the tensor core 64).
template <bool kPair>
__device__ __forceinline__ void issue_item_flat(const TcParams &P, uint32_t d_tmem, uint32_t patch_lo,
                                                uint32_t desc_hi, uint32_t b_lo0, uint32_t b_step,
                                                uint32_t tmem_sf) {
  constexpr int kBatch = 16;
  uint32_t b = b_lo0;
  for (int j0 = 0; j0 < P.nsteps; j0 += kBatch) {
    uint32_t a[kBatch];
#pragma unroll
    for (int i = 0; i < kBatch; ++i) a[i] = j0 + i < P.nsteps ? P.adesc_lo[j0 + i] + patch_lo : 0u;
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      if (j0 + i < P.nsteps) {
        umma_issue<kPair>(d_tmem, a[i], desc_hi, b, desc_hi, P.idesc, tmem_sf, (j0 + i) > 0 ? 1u : 0u);
        b += b_step;
      }
    }
  }
}

// Resident schedule.  The stage barriers are waited for only before the first item (the CTA stays on one
// slab, which stays in shared memory) and never released.
template <bool kPair>
__device__ void mma_resident(const TcParams &P, const Smem &S, uint32_t tmem_base) {
  const uint32_t tmem_sf = tmem_base + (uint32_t)kSfCol;
  const int nst = (P.nsteps + P.mps - 1) / P.mps;
  const uint32_t b_lbo = (uint32_t)P.NTh * 16u;
  // descriptor halves: high word = stride between 8-row groups (128 B) and the version bit
  const uint32_t desc_hi = (128u >> 4) | (1u << 14);
  const uint32_t b_lo0 = ((S.ring & 0x3FFFFu) >> 4) | ((b_lbo >> 4) << 16);   // stage 0, K-step 0
  const uint32_t b_step = (2u * b_lbo) >> 4;                                   // next K-step
  const uint32_t stage_step = P.stage_bytes >> 4;
  int pb = 0, ab = 0;
  uint32_t pph = 0;
  uint32_t aph = 1u;                     // parity to wait for on the accumulator's empty barrier
  const uint32_t nitems = res_sched(P.ntiles, P.nslabs, kPair).total();       // one patch per item
  for (uint32_t it = 0; it < nitems; ++it) {
    if (!mbar_wait(S.pfull + 8u * pb, pph, S.abort_flag, &g_status_tc)) return;
    const uint32_t patch_lo = ((S.patch + (uint32_t)pb * P.patch_bytes) & 0x3FFFFu) >> 4;   // in descriptor units
    if (!mbar_wait(S.aempty + 8u * ab, aph, S.abort_flag, &g_status_tc)) return;
    tc_fence_after();
    const uint32_t d_tmem = tmem_base + (uint32_t)(ab * P.NT);
    if (it > 0) {
      issue_item_flat<kPair>(P, d_tmem, patch_lo, desc_hi, b_lo0, b_step, tmem_sf);
    } else {
      for (int st = 0; st < nst; ++st) {
        const int j0 = st * P.mps;
        const int nj = min(P.mps, P.nsteps - j0);
        const uint32_t b_lo = b_lo0 + (uint32_t)st * stage_step;
        const uint32_t first = st == 0 ? 0u : 1u;     // the first MMA of an item overwrites
        if (!mbar_wait(S.wfull + 8u * st, 0u, S.abort_flag, &g_status_tc)) return;
        tc_fence_after();
        if (nj == 4) issue_stage<4, kPair>(P, j0, d_tmem, patch_lo, desc_hi, b_lo, desc_hi, b_step, tmem_sf, first);
        else if (nj == 2) issue_stage<2, kPair>(P, j0, d_tmem, patch_lo, desc_hi, b_lo, desc_hi, b_step, tmem_sf, first);
        else if (nj == 8) issue_stage<8, kPair>(P, j0, d_tmem, patch_lo, desc_hi, b_lo, desc_hi, b_step, tmem_sf, first);
        else {
          int jj = 0;
#pragma unroll 1
          for (; jj + 4 <= nj; jj += 4)              // the large steps of a small problem (see make_plan)
            issue_stage<4, kPair>(P, j0 + jj, d_tmem, patch_lo, desc_hi, b_lo + (uint32_t)jj * b_step, desc_hi, b_step, tmem_sf,
                                  jj == 0 ? first : 1u);
#pragma unroll 1
          for (; jj < nj; ++jj)
            umma_issue<kPair>(d_tmem, P.adesc_lo[j0 + jj] + patch_lo, desc_hi,
                              b_lo + (uint32_t)jj * b_step, desc_hi, P.idesc, tmem_sf,
                              jj == 0 ? first : 1u);
        }
      }
    }
    umma_commit_to<kPair>(S.afull + 8u * ab);
    umma_commit_to<kPair>(S.pempty + 8u * pb);
    if (++pb == P.npb) { pb = 0; pph ^= 1u; }
    if (++ab == P.nacc) { ab = 0; aph ^= 1u; }
  }
}

// Streaming schedule: items [i0, i1), item = tile * nslabs + slab, so that a patch serves all slabs of
// its tile.  The thread's instruction latencies are on the path of everything else (an MMA takes 64
// cycles): constants in registers, the patch descriptors four at a time from shared memory, the next
// stage's barrier polled before this stage's MMAs are issued.
template <bool kPair>
__device__ void mma_stream(const TcParams &P, const Smem &S, long long i0, long long i1, uint32_t tmem_base) {
  const uint32_t sf = tmem_base + (uint32_t)kSfCol, idesc = P.idesc, stages = (uint32_t)P.stages;
  const int nsteps = P.nsteps, mps = P.mps, nslabs = P.nslabs;
  const uint32_t b_lbo = (uint32_t)P.NTh * 16u;
  const uint32_t hi = (128u >> 4) | (1u << 14);
  const uint32_t b_lo0 = ((S.ring & 0x3FFFFu) >> 4) | ((b_lbo >> 4) << 16);
  const uint32_t b_step = (2u * b_lbo) >> 4, stage_step = P.stage_bytes >> 4;
  const bool table = P.off_tab != 0u;
  uint32_t ws = 0u, wph = 0u, pph = 0u, aph = 1u, patch_lo = 0u;
  int pb = 0, ab = 0, slab = (int)(i0 % nslabs);
  bool new_tile = true, ready = false;
  const uint32_t nitems = (uint32_t)(i1 - i0);
  for (uint32_t it = 0; it < nitems; ++it) {
    if (new_tile) {
      if (!mbar_wait(S.pfull + 8u * pb, pph, S.abort_flag, &g_status_tc)) return;
      patch_lo = ((S.patch + (uint32_t)pb * P.patch_bytes) & 0x3FFFFu) >> 4;
    }
    if (!mbar_wait(S.aempty + 8u * ab, aph, S.abort_flag, &g_status_tc)) return;
    tc_fence_after();
    const uint32_t d_tmem = tmem_base + (uint32_t)(ab * P.NT);
    uint32_t acc = 0u;                           // the first MMA of an item overwrites
    for (int j0 = 0; j0 < nsteps; j0 += mps) {
      if (!ready && !mbar_wait(S.wfull + 8u * ws, wph, S.abort_flag, &g_status_tc)) return;
      uint32_t b = b_lo0 + ws * stage_step;
      uint32_t nws = ws + 1u, nph = wph;
      if (nws == stages) { nws = 0u; nph ^= 1u; }
      ready = mbar_try(S.wfull + 8u * nws, nph);
      int n = min(mps, nsteps - j0), j = j0;
#pragma unroll 1
      for (; n >= 4; n -= 4, j += 4) {
        uint32_t x[4];
        if (table) {
          lds128(S.tab + (uint32_t)j * 4u, x);   // mps is 4 or 8 here: 16-byte aligned
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) x[i] = P.adesc_lo[j + i];
        }
        umma_issue<kPair>(d_tmem, x[0] + patch_lo, hi, b, hi, idesc, sf, acc);
        umma_issue<kPair>(d_tmem, x[1] + patch_lo, hi, b + b_step, hi, idesc, sf, 1u);
        umma_issue<kPair>(d_tmem, x[2] + patch_lo, hi, b + 2u * b_step, hi, idesc, sf, 1u);
        umma_issue<kPair>(d_tmem, x[3] + patch_lo, hi, b + 3u * b_step, hi, idesc, sf, 1u);
        acc = 1u;
        b += 4u * b_step;
      }
#pragma unroll 1
      for (; n > 0; --n, ++j) {
        umma_issue<kPair>(d_tmem, P.adesc_lo[j] + patch_lo, hi, b, hi, idesc, sf, acc);
        acc = 1u;
        b += b_step;
      }
      umma_commit_to<kPair>(S.wempty + 8u * ws);
      ws = nws;
      wph = nph;
    }
    // next item: same tile (next slab) or the next tile
    new_tile = false;
    if (++slab == nslabs) { slab = 0; new_tile = true; }
    umma_commit_to<kPair>(S.afull + 8u * ab);
    if (new_tile || it + 1 == nitems) umma_commit_to<kPair>(S.pempty + 8u * pb);
    if (new_tile) { if (++pb == P.npb) { pb = 0; pph ^= 1u; } }
    if (++ab == P.nacc) { ab = 0; aph ^= 1u; }
  }
}

template <bool kRes, bool kPair>
__device__ __forceinline__ void mma_role(const TcParams &P, const Smem &S, long long i0, long long i1,
                                         uint32_t tmem_base) {
  if (elect_one()) {
    if constexpr (kRes) mma_resident<kPair>(P, S, tmem_base);
    else mma_stream<kPair>(P, S, i0, i1, tmem_base);
  }
  __syncwarp();
}

// ------------------------------------------------------------------ weight producers (8 warps)
// A stage holds mps K-steps of NT filter rows: plane (2 jj + piece) of NT x 16 bytes.  K-step
// j consumes words 2j, 2j+1 of every filter row, which the word-pair-major weight layout
// keeps contiguous over the filters: a warp reads 32 rows of one K-step as one 256-byte run.
// Thread mapping: row = wt % rows_mod, and the 256 / rows_mod thread groups split the
// stage's K-steps, gs = grp_steps each (unit u of a thread = K-step grp * gs + u of the stage).
// The packed words of kPrefetch stages are in flight in registers.
constexpr int kPrefetch = 3;

// kUnits = grp_steps: K-steps a thread expands per stage.  kSwap: some K-step has its two
// pieces in descending address order (odd Cw or stride 2); otherwise the swap test is compiled
// out.  The common stage (all its K-steps exist, none is the row's lone last word) takes a
// path without per-step predicates.
// The role fills the ring once: it has one stage per stage of the slab, so nothing is waited for.
template <int kUnits, bool kSwap>
__device__ void weight_role(const TcParams &P, const Smem &S, int slab, int wt, int lane) {
  const int nst = (P.nsteps + P.mps - 1) / P.mps;
  const int row = wt % P.rows_mod, grp = wt / P.rows_mod;
  constexpr int gs = kUnits;
  const bool grp_on = grp * gs < P.mps && row < P.NTh;
  const uint32_t b_lbo = (uint32_t)P.NTh * 16u;
  const int row_co = (int)S.rank * P.NTh + row;          // this thread's filter inside a slab
  const int jj0 = grp * gs;                         // first K-step of this thread inside a stage
  const int nplain = (P.row_words >> 1);            // K-steps j < nplain have both words
  const int co = slab * P.NT + row_co;
  const bool on = grp_on && co < P.Co;
  const uint2 *wp2 = reinterpret_cast<const uint2 *>(P.wp);
  uint2 pf[kPrefetch][kUnits];
  auto fetch = [&](uint2 dst[kUnits], int st) {
    const int j0 = st * P.mps + jj0;                // beyond the last stage every K-step is beyond nsteps
    if (on && j0 + gs <= P.nsteps) {
      const uint2 *src = wp2 + ((size_t)j0 * P.Co + co);
#pragma unroll
      for (int u = 0; u < kUnits; ++u) dst[u] = load_global(src + (size_t)u * P.Co);
    } else {
#pragma unroll
      for (int u = 0; u < kUnits; ++u)
        dst[u] = (on && j0 + u < P.nsteps) ? load_global(wp2 + ((size_t)(j0 + u) * P.Co + co))
                                           : make_uint2(0u, 0u);
    }
  };
#pragma unroll
  for (int d = 0; d < kPrefetch; ++d) fetch(pf[d], d);
  const uint32_t row_off = (uint32_t)row * 16u + (uint32_t)(2 * jj0) * b_lbo;
  const uint32_t ring_end = S.ring + (uint32_t)P.stages * P.stage_bytes;
  (void)ring_end;
#pragma unroll 1
  for (int st = 0; st < nst; ++st) {
    const uint32_t stage = S.ring + (uint32_t)st * P.stage_bytes + row_off;
    const int j0 = st * P.mps + jj0;
    if (on && j0 + gs <= nplain) {
      // plain stage: every K-step of this thread exists and has both of its words
      uint32_t sbits = 0u;                      // swap bits of K-steps j0 .. j0 + gs - 1
      if (kSwap) {
        const int wi = (j0 >> 5) & 31;
        sbits = __funnelshift_r(P.swap_mask[wi], P.swap_mask[(wi + 1) & 31], j0 & 31);
      }
#pragma unroll
      for (int u = 0; u < kUnits; ++u) {
        uint32_t v0[4], v1[4];
        expand_signs<false>(pf[0][u].x, v0);
        expand_signs<false>(pf[0][u].y, v1);
        const uint32_t a = stage + (uint32_t)(2 * u) * b_lbo;
        const uint32_t sw = (kSwap && ((sbits >> u) & 1u)) ? b_lbo : 0u;
        if (in_bounds(a >= S.ring && a + b_lbo + 16u <= ring_end, 1)) {
          sts128(a + sw, v0[0], v0[1], v0[2], v0[3]);
          sts128(a + b_lbo - sw, v1[0], v1[1], v1[2], v1[3]);
        }
      }
    } else if (on) {
#pragma unroll
      for (int u = 0; u < kUnits; ++u) {
        const int j = j0 + u;
        if (j < P.nsteps) {
          const bool swap = (P.swap_mask[(j >> 5) & 31] >> (j & 31)) & 1u;
          const uint32_t keep = j < nplain ? 0xFFFFFFFFu : 0u;   // lone last word: partner is 0
          uint32_t v0[4], v1[4];
          expand_signs<false>(pf[0][u].x, v0);
          expand_signs<false>(pf[0][u].y, v1);
          v1[0] &= keep; v1[1] &= keep; v1[2] &= keep; v1[3] &= keep;
          const uint32_t a = stage + (uint32_t)(2 * u) * b_lbo;
          if (in_bounds(a >= S.ring && a + b_lbo + 16u <= ring_end, 2)) {
            sts128(swap ? a + b_lbo : a, v0[0], v0[1], v0[2], v0[3]);
            sts128(swap ? a : a + b_lbo, v1[0], v1[1], v1[2], v1[3]);
          }
        }
      }
    }
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) { if (P.pair) mbar_arrive_peer_mma(S.wfull + 8u * st, 0u); else mbar_arrive(S.wfull + 8u * st); }
    // the queue of packed words moves up one stage; the freed slot is refilled
#pragma unroll
    for (int d = 0; d + 1 < kPrefetch; ++d)
#pragma unroll
      for (int u = 0; u < kUnits; ++u) pf[d][u] = pf[d + 1][u];
    fetch(pf[kPrefetch - 1], st + kPrefetch);
  }
}

template <int kUnits>
__device__ __forceinline__ void weight_role_swap(const TcParams &P, const Smem &S, int slab, int wt, int lane) {
  if (P.any_swap) weight_role<kUnits, true>(P, S, slab, wt, lane);
  else weight_role<kUnits, false>(P, S, slab, wt, lane);
}

__device__ __forceinline__ void weight_dispatch(const TcParams &P, const Smem &S, int slab, int wt, int lane) {
  if (P.grp_steps == 4) weight_role_swap<4>(P, S, slab, wt, lane);
  else if (P.grp_steps == 2) weight_role_swap<2>(P, S, slab, wt, lane);
  else weight_role_swap<1>(P, S, slab, wt, lane);
}

// ---- streaming schedule: three groups of four warps, or two
// The groups of four warps fill the stages of the sequence over all items in turn: with every warp on
// every stage the expansion was bound by its latency (one instruction in 10 to 15 cycles per warp next
// to the other roles, barriers and bookkeeping per stage).  A thread expands up to four K-steps of one
// row of a stage: row t % rows_mod, every (128 / rows_mod)-th K-step.  What bounds the loop is its number
// of instructions, so nothing in it is predicated: rows beyond C_out and K-steps beyond the last re-read
// an existing word (their columns are never stored, their K-steps never issued), and a word of the next
// stage is loaded into the register of the one just expanded.
template <bool kSpecial>
__device__ void weight_stream(const TcParams &P, const Smem &S, uint32_t nitems, int slab0, int group, int t, int lane) {
  constexpr int kU = 4;
  const int nst = (P.nsteps + P.mps - 1) / P.mps;
  const int subs = 32 * kGroupWarps / P.rows_mod, row = t & (P.rows_mod - 1), sub = t / P.rows_mod;
  const int nu = max(1, P.mps / subs);               // K-steps of this thread in a stage
  const bool on = row < P.NTh && sub < P.mps;
  const uint32_t lbo = (uint32_t)P.NTh * 16u, lstep = (uint32_t)subs * 2u * lbo, gstep = (uint32_t)(subs * P.Co);
  const uint32_t last = (uint32_t)(P.nsteps * P.Co) - 1u;
  const int nplain = P.row_words >> 1;               // K-steps j < nplain have both words
  const int row_co = (int)S.rank * P.NTh + row;
  const uint32_t row_off = (uint32_t)row * 16u + (uint32_t)sub * 2u * lbo;
  const uint2 *wp2 = reinterpret_cast<const uint2 *>(P.wp);
  uint32_t it = 0u;
  int st = group, slab = slab0;
  auto settle = [&]() {
    while (st >= nst) {
      st -= nst;
      ++it;
      if (++slab == P.nslabs) slab = 0;
    }
  };
  auto offset = [&]() { return (uint32_t)((st * P.mps + sub) * P.Co + min(slab * P.NT + row_co, P.Co - 1)); };
  settle();
  uint2 w[kU];
  uint32_t off = offset();
#pragma unroll
  for (int u = 0; u < kU; ++u) w[u] = load_global(wp2 + min(off + (uint32_t)u * gstep, last));
  uint32_t ws = (uint32_t)group, wph = 1u;           // stages >= groups (host)
#pragma unroll 1
  while (it < nitems) {
    const int j0 = st * P.mps + sub;
    st += P.wgt_groups;
    settle();
    off = offset();
    if (!mbar_wait_relaxed(S.wempty + 8u * ws, wph, S.abort_flag, &g_status_tc, XNOR_SLEEP_WGT)) return;
    if (on) {
      uint32_t a = S.ring + ws * P.stage_bytes + row_off;
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        if (u < nu) {
          uint32_t v0[4], v1[4], sw = 0u;
          expand_signs<false>(w[u].x, v0);
          expand_signs<false>(w[u].y, v1);
          w[u] = load_global(wp2 + min(off, last));
          if (kSpecial) {
            const int j = j0 + u * subs;
            if ((P.swap_mask[(j >> 5) & 31] >> (j & 31)) & 1u) sw = lbo;
            if (j >= nplain) v1[0] = v1[1] = v1[2] = v1[3] = 0u;       // the row's lone last word: its partner is 0
          }
          if (in_bounds(a >= S.ring && a + lbo + 16u <= S.ring + (uint32_t)P.stages * P.stage_bytes, 13)) {
            sts128(a + sw, v0[0], v0[1], v0[2], v0[3]);
            sts128(a + lbo - sw, v1[0], v1[1], v1[2], v1[3]);
          }
          a += lstep;
          off += gstep;
        }
      }
    }
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) { if (P.pair) mbar_arrive_peer_mma(S.wfull + 8u * ws, 0u); else mbar_arrive(S.wfull + 8u * ws); }
    ws += (uint32_t)P.wgt_groups;
    if (ws >= (uint32_t)P.stages) { ws -= (uint32_t)P.stages; wph ^= 1u; }
  }
}

// ------------------------------------------------------------------ patch producers
// The group of the three patch warps builds the CTA's patches one after the
// other, all warps on the same patch, or each builds patches of its own.  The
// packed pixels a patch touches are ONE contiguous range of x_packed: input rows
// g0 .. g1 - 1 of the N*H rows (images follow one another in memory, the zero rows and
// columns of the stream exist only in the patch).  Every patch buffer has a raw buffer; the
// group's first warp brings a patch's range into it with one bulk copy (an aligned superset
// inside the tensor; the ragged last words of the tensor, if any, by plain loads) as soon as
// the group is done with the buffer's previous patch, so the rows of the next patches are on
// their way while one is expanded.  Padding and the channel tail become the value 0 through
// masks folded into the sign mask and the magnitude constants.
// Streaming: one patch per tile of the CTA's range.  Resident (kRes): one patch per item.
// kTwo: two bit planes of a k-bit input in one pass.  Their level code b0 + 2 b1 stands for -3, -1, 1, 3,
// all of them e2m1 values beside any of the three magnitudes: the upper plane is the sign, and equal bits
// triple the magnitude.  The convolution then costs what one plane costs.
template <bool kRes, bool kTwo>
__device__ void patch_role(const TcParams &P, const Smem &S, long long i0, long long i1, int pw,
                           int lane) {
  const ResSched R = res_sched(P.ntiles, P.nslabs, P.pair != 0);
  const int tile0 = kRes ? 0 : (int)(i0 / P.nslabs);
  const uint32_t npatches = kRes ? R.total()
                                 : (uint32_t)((i1 - 1) / P.nslabs) - (uint32_t)tile0 + 1u;
  const int s = P.stride, phases = s * s;
  const uint32_t plane_bytes = (uint32_t)P.ppix * 16u;
  // nibble masks of the channel tail, one per expanded register
  uint32_t tm[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) tm[r] = ((P.tail_mask >> r) & 0x11111111u) * 0xFu;
  const bool tail = P.tail_mask != 0xFFFFFFFFu;
  const uint32_t word_bytes = (uint32_t)P.Cw * 4u, row_bytes = (uint32_t)P.W * word_bytes;   // of a pixel, a row
  // pairs: work tile t is stream tiles 2t (rank 0) and 2t + 1 (rank 1)
  const uint32_t tmul = P.pair ? 2u : 1u;
  const int ngrp = patch_groups(P.Cw, kRes);

  auto first_pos = [&](uint32_t seq) {                    // of patch seq, in the stream
    return ((kRes ? R.tile(seq) : (uint32_t)tile0 + seq) * tmul + S.rank) * kTileM;
  };
  // the input row (of the N*H rows of the tensor) that stream row r stands for, clamped to its image;
  // add = 0: the first of its rows, s: the one behind the last
  auto input_row = [&](uint32_t r, int add) {
    const uint32_t n = fast_div(r, P.div_hq_m, P.div_hq_s);
    return (int)n * P.H + min(max(((int)(r - n * (uint32_t)P.Hq) - P.leadY) * s + add, 0), P.H);
  };
  // a subgroup's first warp, lane 0: starts the copy of a patch's rows into raw buffer rb
  auto start_copy = [&](uint32_t seq, uint32_t rb) {
    const uint32_t m0 = first_pos(seq), mlast = min(m0 + (uint32_t)P.ppix - 1u, (uint32_t)P.L - 1u);
    const int g0 = input_row(fast_div(m0, P.div_wq_m, P.div_wq_s), 0);
    const int g1 = input_row(fast_div(mlast, P.div_wq_m, P.div_wq_s), s);
    const uint32_t bar = S.rawfull + 8u * rb;
    const uint32_t dst = S.raw + rb * P.raw_bytes;
    if (g1 <= g0) { mbar_arrive(bar); return; }          // nothing but padding
    const size_t b0 = (size_t)g0 * row_bytes, a0 = b0 & ~(size_t)15, left = (size_t)P.N * P.H * row_bytes - a0;
    const uint32_t need = ((uint32_t)b0 & 15u) + (uint32_t)(g1 - g0) * row_bytes;    // from the 16-byte boundary a0
    uint32_t bulk = (need + 15u) & ~15u;
    if (bulk > left) bulk = (uint32_t)left & ~15u;
    for (uint32_t b = bulk; b < need; b += 4u)           // at most 3 words, at the tensor's end
      if (in_bounds(b + 4u <= P.raw_plane, 3))
      {
        sts32(dst + b, load_global(P.xp + ((a0 + b) >> 2)));
        if (kTwo) sts32(dst + P.raw_plane + b, load_global(P.xp2 + ((a0 + b) >> 2)));
      }
    if (bulk && in_bounds(bulk <= P.raw_plane && bulk <= left, 4)) {
      mbar_arrive_expect_tx(bar, kTwo ? 2u * bulk : bulk);
      bulk_copy_g2s(dst, reinterpret_cast<const uint8_t *>(P.xp) + a0, bulk, bar);
      if (kTwo) bulk_copy_g2s(dst + P.raw_plane, reinterpret_cast<const uint8_t *>(P.xp2) + a0, bulk, bar);
    } else {
      mbar_arrive(bar);
    }
  };

  // The group works as `nsub` subgroups of equal size; subgroup sg builds patches sg,
  // sg + nsub, ... (nsub <= npb: a barrier's parity tells apart only two consecutive uses of
  // a buffer, so no subgroup may run more than one use ahead of the consumer).
  const uint32_t nsub = (uint32_t)P.pat_sub, gsize = (uint32_t)kPatWarps / nsub;
  const uint32_t sg = (uint32_t)pw % nsub, mi = (uint32_t)pw / nsub;

  // Expands this warp's share of a patch: raw buffer rb holds input rows g0 .. from address `raw` on, m0 is the
  // patch's first position.  Units, in this order of nesting: kPos x 32 positions, phase plane, kWords channel
  // words (0: up to four, one after the other); every warp of the subgroup takes a contiguous share.  A lane keeps
  // the address of one row of the patch, so that locating a position costs a multiplication and a shuffle; the
  // work on the kPos positions is independent, and the innermost part does not branch.  What bounds a patch is
  // the latency of its one warp: two divisions per position and unit, as before, took 4500 cycles for the patch of
  // 64 channels, 56x56, where an item takes 2300 and three warps build patches (256 images, 64 filters 3x3: 63.1 ->
  // 55.7 us; stride 2, 128 filters 38.1 -> 32.4; 256 channels, 14x14, stride 2, one image 8.7 -> 7.5).  The same steps with
  // the place of a unit kept by branches in one flat loop were slower than the divisions (67.5).
  auto build = [&](auto kpos_, auto kwords_, uint32_t m0, int g0, uint32_t raw, uint32_t rb, uint32_t patch) {
    constexpr int kPos = decltype(kpos_)::value, kWords = decltype(kwords_)::value, kLoop = kWords ? kWords : 4;
    constexpr int kStep = kWords == 1 ? 1 : 4;            // channel words of a unit
    const uint32_t r0 = fast_div(m0, P.div_wq_m, P.div_wq_s), c0 = m0 - r0 * (uint32_t)P.Wq;
    // addresses of the input rows of stream row r, one per row phase; 0: padding
    auto row_address = [&](uint32_t r, uint32_t &a0, uint32_t &a1) {
      const uint32_t n = fast_div(r, P.div_hq_m, P.div_hq_s);
      const int y = ((int)(r - n * (uint32_t)P.Hq) - P.leadY) * s;
      const uint32_t a = raw + (uint32_t)((int)n * P.H + y - g0) * row_bytes;
      const bool in = n < (uint32_t)P.N && y >= 0;
      a0 = in && y < P.H ? a : 0u;
      a1 = in && y + 1 < P.H ? a + row_bytes : 0u;
    };
    uint32_t tab0, tab1;
    row_address(r0 + (uint32_t)lane, tab0, tab1);
    const int nunits = (P.ppix + 32 * kPos - 1) / (32 * kPos) * phases * ngrp;
    const int share = (nunits + (int)gsize - 1) / (int)gsize;
    int u = (int)mi * share;
    const int u1 = min(u + share, nunits);
    int block = 0, phase = 0, w0 = 0;
    if (u > 0) {
      block = (int)fast_div((uint32_t)u, P.div_pg_m, P.div_pg_s);
      const int rem = u - block * (phases * ngrp);
      phase = (int)fast_div((uint32_t)rem, P.div_g_m, P.div_g_s);
      w0 = (rem - phase * ngrp) * kStep;
    }
#pragma unroll 1
    for (; u < u1; ++block, phase = 0) {
      int col[kPos];
      uint32_t row0[kPos], row1[kPos], pdst[kPos];
      bool on[kPos];
#pragma unroll
      for (int b = 0; b < kPos; ++b) {
        const int q = (block * kPos + b) * 32 + lane;
        const uint32_t x = c0 + (uint32_t)q;
        on[b] = q < P.ppix;
        pdst[b] = patch + (uint32_t)q * 16u;
        if (P.pat_table) {
          const uint32_t i = __umulhi(x, P.wq_rcp);
          col[b] = ((int)(x - i * (uint32_t)P.Wq) - P.leadX) * s;
          row0[b] = __shfl_sync(0xffffffffu, tab0, (int)i);
          row1[b] = s == 2 ? __shfl_sync(0xffffffffu, tab1, (int)i) : 0u;
        } else {
          const uint32_t i = fast_div(x, P.div_wq_m, P.div_wq_s);
          col[b] = ((int)(x - i * (uint32_t)P.Wq) - P.leadX) * s;
          row_address(r0 + i, row0[b], row1[b]);
        }
      }
#pragma unroll 1
      for (; phase < phases && u < u1; ++phase, w0 = 0) {
        const int py = phase >> (s - 1), px = phase & (s - 1);     // stride 1 or 2
        uint32_t src[kPos], dst[kPos], sm[kPos], mc[kPos][3];
#pragma unroll
        for (int b = 0; b < kPos; ++b) {
          const uint32_t row = py ? row1[b] : row0[b];
          const bool real = on[b] && row != 0u && col[b] >= 0 && col[b] + px < P.W;
          const uint32_t keep = real ? 0xFFFFFFFFu : 0u;           // padding expands to 0, whatever its word is
          sm[b] = 0x88888888u & keep;
          mc[b][0] = 0xCCCCCCCCu & keep; mc[b][1] = 0xAAAAAAAAu & keep; mc[b][2] = 0x99999999u & keep;
          src[b] = (real ? row + (uint32_t)(col[b] + px) * word_bytes : S.raw + rb * P.raw_bytes) + (uint32_t)w0 * 4u;
          dst[b] = pdst[b] + (uint32_t)(phase * P.Cw + w0) * plane_bytes;
        }
#pragma unroll 1
        for (; w0 < P.Cw && u < u1; w0 += kStep, ++u) {
          uint32_t wv[kPos][4], wu[kTwo ? kPos : 1][4];
          auto load = [&](uint32_t a, uint32_t (&v)[4]) {
            if constexpr (kWords == 4) lds128(a, v);
            else if constexpr (kWords == 2) lds64(a, v[0], v[1]);
            else {
#pragma unroll
              for (int i = 0; i < kLoop; ++i) v[i] = kWords || w0 + i < P.Cw ? lds32(a + (uint32_t)i * 4u) : 0u;
            }
          };
#pragma unroll
          for (int b = 0; b < kPos; ++b) {
            if (in_bounds(src[b] >= S.raw + rb * P.raw_bytes &&
                          src[b] + 4u * (uint32_t)min(kStep, P.Cw - w0) <= S.raw + rb * P.raw_bytes + P.raw_plane, 6)) {
              load(src[b], wv[b]);
              if constexpr (kTwo) load(src[b] + P.raw_plane, wu[b]);
            }
            src[b] += 4u * kStep;
          }
#pragma unroll
          for (int i = 0; i < kLoop; ++i) {
            if (kWords || w0 + i < P.Cw) {
              const bool cut = tail && w0 + i == P.Cw - 1;       // channels beyond C_in are 0
#pragma unroll
              for (int b = 0; b < kPos; ++b) {
                const uint32_t w = kTwo ? wu[b][i] : wv[b][i];      // signs
                uint32_t v0 = ((w << 3) & sm[b]) ^ mc[b][0];
                uint32_t v1 = ((w << 2) & sm[b]) ^ mc[b][1];
                uint32_t v2 = ((w << 1) & sm[b]) ^ mc[b][2];
                uint32_t v3 = (w & sm[b]) ^ mc[b][2];
                if constexpr (kTwo) {                     // magnitudes 2, 1, 0.5 (100, 010, 001) -> 6, 3, 1.5 (111, 101, 011)
                  const uint32_t e = ~(wv[b][i] ^ wu[b][i]), e0 = (e << 3) & sm[b], e1 = (e << 2) & sm[b];
                  v0 ^= (e0 >> 2) | (e0 >> 3);
                  v1 ^= e1 - (e1 >> 3);
                  v2 ^= ((e << 1) & sm[b]) >> 2;
                  v3 ^= (e & sm[b]) >> 2;
                }
                if (cut) { v0 &= tm[0]; v1 &= tm[1]; v2 &= tm[2]; v3 &= tm[3]; }
                if (on[b] && in_bounds(dst[b] >= patch && dst[b] + 16u <= patch + P.patch_bytes, 5)) sts128(dst[b], v0, v1, v2, v3);
                dst[b] += plane_bytes;
              }
            }
          }
        }
      }
    }
  };

  // The subgroup's k-th patch (patch sg + k nsub of the CTA) expands from the subgroup's raw
  // buffer k % nraw; its rows are fetched as soon as the subgroup is done with patch k - nraw.
  const uint32_t nraw = (uint32_t)P.nraw, rb0 = sg * nraw;
  bool ok = true;
  uint32_t kc = 0;                           // patches of the subgroup whose copy has been started
  if (mi == 0) {
    for (; kc < nraw && sg + kc * nsub < npatches; ++kc)
      if (lane == 0) start_copy(sg + kc * nsub, rb0 + kc);
  }
  uint32_t k = 0;
#pragma unroll 1
  for (uint32_t seq = sg; seq < npatches && ok; seq += nsub, ++k) {
    const uint32_t pb = seq % (uint32_t)P.npb;
    const uint32_t use = seq / (uint32_t)P.npb;
    const uint32_t rb = rb0 + k % nraw, ruse = k / nraw;
    if (mi == 0 && k >= 1u && sg + kc * nsub < npatches) {
      // kc = k - 1 + nraw: the raw buffer of patch k - 1 is free once every warp of the
      // subgroup has expanded that patch
      const uint32_t crb = rb0 + kc % nraw;
      ok = mbar_wait_relaxed(S.rawdone + 8u * crb, (kc / nraw - 1u) & 1u, S.abort_flag,
                             &g_status_tc, XNOR_SLEEP_PAT);
      if (!ok) break;
      fence_proxy_async();
      if (lane == 0) start_copy(sg + kc * nsub, crb);
      ++kc;
    }
    const uint32_t m0 = first_pos(seq);
    const int g0 = input_row(fast_div(m0, P.div_wq_m, P.div_wq_s), 0);
    ok = mbar_wait_relaxed(S.rawfull + 8u * rb, ruse & 1u, S.abort_flag, &g_status_tc, XNOR_SLEEP_PAT);
    if (!ok) break;
    ok = mbar_wait_relaxed(S.pempty + 8u * pb, (use & 1u) ^ 1u, S.abort_flag, &g_status_tc,
                           XNOR_SLEEP_PAT);
    if (!ok) break;
    const uint32_t patch = S.patch + pb * P.patch_bytes;
    const uint32_t raw = S.raw + rb * P.raw_bytes +
                         (uint32_t)(((size_t)g0 * row_bytes) & 15u);   // where row g0 starts
    using std::integral_constant;
    constexpr int kWide = kRes ? 2 : 1;           // (registers)
    const integral_constant<int, kWide> few;
    const integral_constant<int, 2 * kWide> many;
    if ((P.Cw & 3) == 0) build(few, integral_constant<int, 4>{}, m0, g0, raw, rb, patch);
    else if (P.Cw == 1) build(many, integral_constant<int, 1>{}, m0, g0, raw, rb, patch);
    else if (P.Cw == 2) build(many, integral_constant<int, 2>{}, m0, g0, raw, rb, patch);
    else if (P.Cw == 3) build(few, integral_constant<int, 3>{}, m0, g0, raw, rb, patch);
    else if constexpr (kRes) build(few, integral_constant<int, 0>{}, m0, g0, raw, rb, patch);
    else build(many, integral_constant<int, 1>{}, m0, g0, raw, rb, patch);
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(S.rawdone + 8u * rb);
      if (P.pair) mbar_arrive_peer_mma(S.pfull + 8u * pb, 0u); else mbar_arrive(S.pfull + 8u * pb);
    }
  }
  if (!ok && mi == 0) {
    // gave up: the copies this warp started last (one per buffer at most can still be in
    // flight) must land before the CTA's shared memory is released
    for (uint32_t back = 1; back <= nraw && back <= kc; ++back) {
      const uint32_t c = kc - back;
      for (int i = 0; i < (1 << 20) && !mbar_try(S.rawfull + 8u * (rb0 + c % nraw), (c / nraw) & 1u); ++i) {}
    }
  }
}

// ------------------------------------------------------------------ epilogue (4 warps)
// Warp w reads tensor-memory lanes 32 (w % 4) .. +31 (pixels), of every item the columns (filters) of some chunks.
// Lane = pixel, so for one filter a warp stores 32 consecutive stream pixels: a contiguous
// run of the NCHW output row.
// Drains the CTA's `nitems` items: streaming, items i0, i0 + 1, ...
// (item = tile * nslabs + slab); resident, tiles tile0, tile0 + tstep, ... of slab `slab0`.
// An item is cut into chunks, and the chunks of all items in sequence are dealt to the warps that share a quarter
// of the lanes (Drain): a warp's work per item (decoding its pixel, the waits) is then spread over a whole chunk.
// A warp may have no chunk in an item and skips it; plan_drain keeps such steps within what parities can tell.
// kFuse: a chunk is an even number of groups (a pair = 32 consecutive filters = one packed word of the
// next layer's input) and has a plane of partial sums of its own; see the fused emit below.
template <bool kRes, bool kFuse>
__device__ void epilogue_role(const TcParams &P, const Smem &S, long long i0, int slab0, int tile0,
                              int tstep, uint32_t nitems, uint32_t tmem_base, int quarter, int e, int lane) {
  const int b_end = P.NT / 16;
  const Drain D = P.drain;
  const size_t HoWo = (size_t)P.Ho * P.Wo;
  const uint32_t howo = (uint32_t)HoWo;
  const size_t out_elems = (size_t)P.N * P.Co * HoWo;
  (void)out_elems;
  // the fast store paths: offsets of 16 consecutive filters fit 32 bits, no integer output
  const bool small = HoWo < ((size_t)1 << 27) && P.acc_out == nullptr;
  const bool relu = P.relu != 0;
  const bool plain = small && P.residual == nullptr, with_res = small && P.residual != nullptr;
  const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
  // the chunk at hand: chunk c of item it; its accumulator buffer and the parity of that one's full barrier
  struct At { uint32_t it; int c, tile, slab, ab; uint32_t fph; };
  At at{0u, e, 0, 0, 0, 0u};
  if (kRes) { at.slab = slab0; at.tile = tile0; }
  else { at.tile = (int)(i0 / P.nslabs); at.slab = (int)(i0 - (long long)at.tile * P.nslabs); }
  auto settle = [&](At &a) {
    while (a.c >= D.chunks) {
      a.c = D.carry(a.c);
      ++a.it;
      if (++a.ab == P.nacc) { a.ab = 0; a.fph ^= 1u; }
      if (kRes) a.tile += tstep;
      else if (++a.slab == P.nslabs) { a.slab = 0; ++a.tile; }
    }
  };
  settle(at);
  constexpr uint32_t kNoPixel = 0xFFFFFFFFu;
  // this lane's output pixel in a tile: whether it exists, its K, offset of (image, filter 0, pixel)
  struct Pix { float kv; size_t obase; uint32_t gpix; };   // gpix: pixel index over all images (below the stream's length)
  const uint32_t tile_len = P.pair ? 2u * kTileM : kTileM, pos0 = S.rank * kTileM + (uint32_t)(quarter * 32 + lane);
  auto decode = [&](int t) {
    Pix px{0.0f, 0, kNoPixel};
    const uint32_t m = (uint32_t)t * tile_len + pos0;
    if (m < (uint32_t)P.L) {
      const uint32_t r = fast_div(m, P.div_wq_m, P.div_wq_s);
      const int ox = (int)(m - r * (uint32_t)P.Wq);
      const uint32_t n = fast_div(r, P.div_hq_m, P.div_hq_s);
      const int oy = (int)(r - n * (uint32_t)P.Hq);
      if (ox < P.Wo && oy < P.Ho) {
        const size_t pix = (size_t)oy * P.Wo + ox;
        px.kv = load_global(P.K + (size_t)n * HoWo + pix);
        px.obase = (size_t)n * P.Co * HoWo + pix;
        px.gpix = n * howo + (uint32_t)pix;
      }
    }
    return px;
  };
  // The residual of a chunk is pulled into L2 while the warp drains the chunk before: the loads in the
  // drain loop then see L2 latency only, and the bytes in flight are not bounded by registers.  The warp's
  // pixels are one run of a filter's plane (at most 128 bytes: two lines), so a lane takes a filter and touches
  // the two ends of its run: a handful of instructions instead of one prefetch per filter and lane.
  auto prefetch_residual = [&](const At &a, const Pix &px) {
    const unsigned vm = __ballot_sync(0xffffffffu, px.gpix != kNoPixel);
    if (vm == 0u) return;
    const unsigned long long o0 = __shfl_sync(0xffffffffu, (unsigned long long)px.obase, __ffs(vm) - 1);
    const unsigned long long o1 = __shfl_sync(0xffffffffu, (unsigned long long)px.obase, 31 - __clz(vm));
    const int f0 = a.slab * P.NT + a.c * D.chunk * 16, f1 = min(P.Co, min(f0 + D.chunk * 16, (a.slab + 1) * P.NT));
    for (int j = f0 + lane; j < f1; j += 32) {
      const float *rp = P.residual + (size_t)j * HoWo;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(rp + o0));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(rp + o1));
    }
  };
  Pix px{0.0f, 0, kNoPixel};
  if (at.it < nitems) {
    px = decode(at.tile);
    if (P.residual != nullptr) prefetch_residual(at, px);
  }
  while (at.it < nitems) {
    const bool valid = px.gpix != kNoPixel;
    const float kv = px.kv;
    const size_t obase = px.obase;
    const uint32_t obase_pix = px.gpix;
    // the chunk after this one; its pixel is decoded (and its K and residual on their way) while this one drains
    At nx = at;
    nx.c += D.split;
    settle(nx);
    Pix npx = px;
    if (nx.it < nitems) {
      if (nx.tile != at.tile) npx = decode(nx.tile);
      if (P.residual != nullptr) prefetch_residual(nx, npx);
    }
    const int slab = at.slab;
    if (!mbar_wait_relaxed(S.afull + 8u * at.ab, at.fph, S.abort_flag, &g_status_tc, XNOR_SLEEP_EPI)) break;
    tc_fence_after();
    const uint32_t t_acc = t_lane + (uint32_t)(at.ab * P.NT);
    const int co0 = slab * P.NT;

    // Store addresses step from filter to filter by one multiply-add each (forming every
    // address from the group's base takes two instructions per store and measured slower).
    auto emit = [&](int b, const int32_t r[16]) {
      if (!valid) return;
      const int co = co0 + b * 16;
      float *op = P.out + obase + (size_t)co * HoWo;
      if (co + 16 <= P.Co && plain) {
        float4 al[4];
#pragma unroll
        for (int j4 = 0; j4 < 4; ++j4)
          al[j4] = lds_f4(S.alpha + (uint32_t)(co * 4 + j4 * 16));
        // the 16 products first, then the 16 stores (and the ReLU test once per group, not per
        // value): two multiplies, an address and a store per output
        float v[16];
#pragma unroll
        for (int j4 = 0; j4 < 4; ++j4) {
          v[j4 * 4 + 0] = __fmul_rn(__fmul_rn(__int_as_float(r[j4 * 4 + 0]), kv), al[j4].x);
          v[j4 * 4 + 1] = __fmul_rn(__fmul_rn(__int_as_float(r[j4 * 4 + 1]), kv), al[j4].y);
          v[j4 * 4 + 2] = __fmul_rn(__fmul_rn(__int_as_float(r[j4 * 4 + 2]), kv), al[j4].z);
          v[j4 * 4 + 3] = __fmul_rn(__fmul_rn(__int_as_float(r[j4 * 4 + 3]), kv), al[j4].w);
        }
        if (relu) {
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = fmaxf(v[j], 0.0f);
        }
        // one address per store, each one multiply-add from the one before.  (Evict-first stores gain
        // 6-8 % on the ResNet layers run back to back, but the next layer's BinActiv or pool, which
        // starts with what was written last, then finds less of it in the L2.)
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (in_bounds(obase + (size_t)(co + j) * HoWo < out_elems, 7)) *op = v[j];
          op += howo;
        }
      } else if (co + 16 <= P.Co && with_res) {
        const float *rp = P.residual + obase + (size_t)co * HoWo;
        float res[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) { res[j] = *rp; rp += howo; }
#pragma unroll
        for (int j4 = 0; j4 < 4; ++j4) {
          const float4 al = lds_f4(S.alpha + (uint32_t)(co * 4 + j4 * 16));
          const float a4[4] = {al.x, al.y, al.z, al.w};
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const float v = __fmul_rn(__fmul_rn(__int_as_float(r[j4 * 4 + jj]), kv), a4[jj]) + res[j4 * 4 + jj];
            if (in_bounds((size_t)(op - P.out) < out_elems, 8)) *op = relu ? fmaxf(v, 0.0f) : v;
            op += howo;
          }
        }
      } else {
        const size_t o0 = obase + (size_t)co * HoWo;
        float res[16];
        if (P.residual) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            res[j] = co + j < P.Co ? P.residual[o0 + (size_t)j * HoWo] : 0.0f;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (co + j < P.Co) {
            const float d = __int_as_float(r[j]);
            float v = __fmul_rn(__fmul_rn(d, kv), lds_f(S.alpha + (uint32_t)((co + j) * 4)));
            if (P.residual) v += res[j];
            if (relu) v = fmaxf(v, 0.0f);
            if (in_bounds(o0 + (size_t)j * HoWo < out_elems, 9)) P.out[o0 + (size_t)j * HoWo] = v;
            if (P.acc_out) {
              int32_t *ap = P.acc_out + o0 + (size_t)j * HoWo;
              *ap = (P.acc_accum ? *ap : 0) + (__float2int_rn(d) << P.acc_shift);
            }
          }
        }
      }
    };

    // Fused: out = D K alpha (+ residual) as above (stored only if the caller wants the fp32
    // tensor), then y = fmaf(scale, out, shift) of the next layer's BatchNorm, the sign bit of
    // y into the word of this pair of groups, |y| into this warp's partial sum for A.
    uint32_t word = 0u;
    float as0 = 0.0f, as1 = 0.0f, as2 = 0.0f, as3 = 0.0f;     // four chains of the |y| sum
    auto emit_fused = [&](int b, const int32_t r[16]) {
      if (!valid) return;
      const int co = co0 + b * 16;
      uint32_t half = 0u;                     // the 16 sign bits of this group
      float *op = P.out + obase + (size_t)co * HoWo;
      float res[16];                          // all 16 residual loads in flight together
      if (P.residual != nullptr) {
        const float *rp = P.residual + obase + (size_t)co * HoWo;
#pragma unroll
        for (int j = 0; j < 16; ++j) { res[j] = *rp; rp += howo; }
      }
#pragma unroll
      for (int j4 = 0; j4 < 4; ++j4) {
        const float4 al = lds_f4(S.alpha + (uint32_t)(co * 4 + j4 * 16));
        float4 sc = make_float4(1.0f, 1.0f, 1.0f, 1.0f), sh = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (P.nscale != nullptr) {
          sc = lds_f4(S.nscale + (uint32_t)(co * 4 + j4 * 16));
          sh = lds_f4(S.nshift + (uint32_t)(co * 4 + j4 * 16));
        }
        const float a4[4] = {al.x, al.y, al.z, al.w};
        const float s4[4] = {sc.x, sc.y, sc.z, sc.w}, h4[4] = {sh.x, sh.y, sh.z, sh.w};
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const int j = j4 * 4 + jj;
          float v = __fmul_rn(__fmul_rn(__int_as_float(r[j]), kv), a4[jj]);
          if (P.residual != nullptr) v += res[j];
          if (relu) v = fmaxf(v, 0.0f);
          if (P.out != nullptr && in_bounds(obase + (size_t)(co + j) * HoWo < out_elems, 10)) *op = v;
          op += howo;
          const float y = P.nscale != nullptr ? __fmaf_rn(s4[jj], v, h4[jj]) : v;
          half |= (y >= 0.0f ? 1u : 0u) << j;
          if (jj == 0) as0 += fabsf(y);
          else if (jj == 1) as1 += fabsf(y);
          else if (jj == 2) as2 += fabsf(y);
          else as3 += fabsf(y);
        }
      }
      word |= half << (co & 16);              // C_out % 32 == 0: a group is the low or the high half
    };

    // 16 columns at a time: load, wait, scale and store.  (Loading the next 16 during the
    // stores of the current ones saves the ~50 cycles of a tensor-memory load per group but
    // costs 16 register copies, which take longer here.)
    int32_t cur[16];
    const int b1 = min((at.c + 1) * D.chunk, b_end);      // groups of the chunk
#pragma unroll 1
    for (int b = at.c * D.chunk; b < b1; ++b) {
      tmem_ld16(t_acc + (uint32_t)(b * 16), cur);
      tmem_wait16(cur);
      if (b + 1 == b1) {                         // that was the last load: release the buffer
        tc_fence_before();
        __syncwarp();
        if (lane == 0) { if (P.pair) mbar_arrive_peer_mma(S.aempty + 8u * at.ab, 0u); else mbar_arrive(S.aempty + 8u * at.ab); }
      }
      if (kFuse) {
        // C_out is a multiple of 32, so a pair of groups lies inside the filters or (last slab)
        // wholly beyond them
        if (co0 + b * 16 >= P.Co) continue;
        emit_fused(b, cur);
        if ((b & 1) && valid) {                  // the pair is complete: its word of the next input
          if (in_bounds(obase_pix < (size_t)P.N * HoWo && ((co0 + b * 16) >> 5) < P.Cw_next, 11))
            P.xp_next[(size_t)obase_pix * (size_t)P.Cw_next + (size_t)((co0 + b * 16) >> 5)] = word;
          word = 0u;
        }
      } else {
        emit(b, cur);
      }
    }
    if (kFuse && valid && in_bounds(obase_pix < (size_t)P.N * HoWo, 12))
      P.A_part[(size_t)(slab * D.chunks + at.c) * ((size_t)P.N * HoWo) + obase_pix] = (as0 + as1) + (as2 + as3);
    px = npx;
    at = nx;
  }
}

template <bool kRes, bool kPair, bool kFuse, bool kTwo>
__global__ void __launch_bounds__(kRes ? kThreadsRes : kThreadsStream, 1)
binconv_tc_kernel(const __grid_constant__ TcParams P) {
  extern __shared__ __align__(128) uint8_t smem[];
  constexpr int kThreads = kRes ? kThreadsRes : kThreadsStream;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Smem S = carve(smem, P);

  if (tid == 0) {
    // In a pair the producers of both CTAs arrive on the barriers of rank 0 (whose MMA warp
    // waits for them); the MMA warp's commits reach the consumer barriers of both CTAs.
    constexpr uint32_t kCtas = kPair ? 2u : 1u;
    for (int i = 0; i < kMaxBarStages; ++i) {
      mbar_init(S.wfull + 8u * i, (uint32_t)(kRes ? kWgtWarps : kGroupWarps) * kCtas);
      mbar_init(S.wempty + 8u * i, 1);
    }
    for (int i = 0; i < kMaxPatchBufs; ++i) {
      mbar_init(S.pfull + 8u * i, (uint32_t)(kPatWarps / P.pat_sub) * kCtas);
      mbar_init(S.pempty + 8u * i, 1);
    }
    for (int i = 0; i < kMaxRaw; ++i) {
      mbar_init(S.rawfull + 8u * i, 1);
      mbar_init(S.rawdone + 8u * i, (uint32_t)(kPatWarps / P.pat_sub));
    }
    for (int i = 0; i < kMaxAcc; ++i) {
      mbar_init(S.afull + 8u * i, 1);
      mbar_init(S.aempty + 8u * i, (uint32_t)(kEpiWarps * P.drain.chunks) * kCtas);
    }
    *S.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    if (kPair) {
      // the same warp of both CTAs of the pair allocates, at the same shared-memory offset
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(S.tmem_slot)), "r"((uint32_t)kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(S.tmem_slot)), "r"((uint32_t)kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *S.tmem_slot;
  if (warp < 4) {
    // unit block scales (ue8m0 1.0 = 0x7F) in every lane of the scale columns
    const uint32_t taddr = tmem_base + ((uint32_t)(warp * 32) << 16) + (uint32_t)kSfCol;
    const uint32_t one = 0x7F7F7F7Fu;
#pragma unroll
    for (int k = 0; k < (kTmemCols - kSfCol) / 8; ++k)
      asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};"
                   ::"r"(taddr + 8u * k), "r"(one) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  // everything up to here overlaps the end of the kernel before this one
  stream_order();
  // per-filter vectors of the epilogue, zero beyond C_out (one global round trip per CTA
  // instead of one per 16 columns drained); alpha carries the call's extra output factor
  // (1 except in the passes of a k-bit convolution; a product with 1 is exact)
  if (!kRes && P.off_tab != 0u)
    for (int i = tid; i < P.nsteps; i += kThreads) reinterpret_cast<uint32_t *>(smem + P.off_tab)[i] = P.adesc_lo[i];
  for (int i = tid; i < P.vec_len; i += kThreads) {
    reinterpret_cast<float *>(smem + P.off_vec)[i] = i < P.Co ? __fmul_rn(load_global(P.alpha + i), P.out_scale) : 0.0f;
    if (kFuse && P.nscale != nullptr) {
      reinterpret_cast<float *>(smem + P.off_vec)[P.vec_len + i] = i < P.Co ? load_global(P.nscale + i) : 0.0f;
      reinterpret_cast<float *>(smem + P.off_vec)[2 * P.vec_len + i] = i < P.Co ? load_global(P.nshift + i) : 0.0f;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // no CTA of a pair signals a barrier of the other before that one has set it up
  if (kPair) cluster_sync();

  // this CTA's (pair's) contiguous range of work items; item = tile * nslabs + slab
  // (streaming) or slab * ntiles + tile (resident); for a pair a tile is two stream tiles
  const long long total = (long long)P.ntiles * P.nslabs;
  const unsigned unit = kPair ? blockIdx.x >> 1 : blockIdx.x, units = kPair ? gridDim.x >> 1 : gridDim.x;
  const long long i0 = total * unit / units;
  const long long i1 = total * (unit + 1) / units;
  const ResSched R = res_sched(P.ntiles, P.nslabs, kPair);
  if (kRes ? R.total() > 0u : i0 < i1) {
    const int wt = tid - 32 * kWgtWarp0;
    if (warp == kMmaWarp) { if (S.rank == 0) mma_role<kRes, kPair>(P, S, i0, i1, tmem_base); }
    else if constexpr (!kRes) {
      // warps 5-7, 9-11, ... in this order: weight groups, patch warps; the last four warps drain too
      // where the epilogue is split
      const int wi = ((warp >> 2) - 1) * 3 + (warp & 3) - 1 - kGroupWarps * P.wgt_groups;
      const bool last = warp >= kThreadsStream / 32 - kEpiWarps && P.drain.split == 2;
      if (warp < kEpiWarps || last)
        epilogue_role<false, kFuse>(P, S, i0, 0, 0, 0, (uint32_t)(i1 - i0), tmem_base, warp & 3, last ? 1 : 0, lane);
      else if ((warp & 3) == 0) {}
      else if (wi < 0) {
        const int group = (wi >> 2) + P.wgt_groups, t = 32 * (wi & 3) + lane, slab0 = (int)(i0 % P.nslabs);
        if (P.any_swap || (P.row_words & 1)) weight_stream<true>(P, S, (uint32_t)(i1 - i0), slab0, group, t, lane);
        else weight_stream<false>(P, S, (uint32_t)(i1 - i0), slab0, group, t, lane);
      }
      else if (wi < kPatWarps) patch_role<false, kTwo>(P, S, i0, i1, wi, lane);
    }
    else if (warp >= kPatWarp0) patch_role<kRes, kTwo>(P, S, i0, i1, warp - kPatWarp0, lane);
    else {
      // The weight warps expand the slab, then every worker warp drains its share of the items.
      const bool wgt = warp >= kWgtWarp0;
      const int e = wgt ? 1 + (warp - kWgtWarp0) / 4 : 0;
      if (wgt) weight_dispatch(P, S, (int)R.slab, wt, lane);
      if (e < P.drain.split)
        epilogue_role<true, kFuse>(P, S, 0, (int)R.slab, (int)R.g, (int)R.G, R.total(), tmem_base, warp & 3, e, lane);
    }
  }
  tc_fence_before();
  __syncthreads();
  // both CTAs of a pair are done with each other's barriers and tensor memory
  if (kPair) cluster_sync();
  if (warp == kMmaWarp) {
    if (kPair)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;"
                   ::"r"(tmem_base), "r"((uint32_t)kTmemCols) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                   ::"r"(tmem_base), "r"((uint32_t)kTmemCols) : "memory");
  }
}

int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

struct Plan {
  TcParams P;
  size_t smem;
  bool ok;
  bool by_time;                // streaming although the resident schedule would fit: estimated to be faster
};

// Weight-thread mapping and stage size for slabs of NT filters: rows_mod threads cover the
// rows of a K-step, the other thread groups take other K-steps of the stage; a stage is up to
// 32 KB of expanded weights.
void plan_stage(TcParams &P, bool few) {
  int ntp = 16;
  while (ntp < P.NTh) ntp *= 2;                         // 16 .. 256
  P.rows_mod = ntp;
  const int groups = std::max(1, 32 * kWgtWarps / P.rows_mod);   // 1 .. 16
  P.mps = std::max(2, std::min(few ? 32 : 8, 1024 / ntp));
  while (P.mps > 4 && P.nsteps < (few ? 2 : 3) * P.mps) P.mps /= 2;   // short items: smaller stages start sooner
  if (P.mps > 4 * groups) P.mps = 4 * groups;           // a thread expands at most 4 K-steps of a stage
  P.grp_steps = std::max(1, P.mps / groups);            // 4, 4, 2, 1, 1
  P.stage_bytes = (uint32_t)P.mps * (uint32_t)P.NTh * 32u;
}

// Filters per slab for `ns` slabs.  A pair splits the rows of a slab between its two CTAs
// (halves of a multiple of 16 rows each).
int slab_width(int Co, int ns, bool pair) {     // pair: also set for the fused epilogue (32-filter words)
  const int q = pair ? 32 : 16;
  return ((Co + ns - 1) / ns + q - 1) / q * q;
}

// schedule: 0 = resident when the slab fits, 1 = streaming.  pair: CTA pairs (clusters of 2).
Plan make_plan(const ConvGeom &g, int schedule, bool pair, bool fuse, int planes, bool residual) {
  Plan pl{};
  pl.ok = false;
  TcParams &P = pl.P;
  const int s = g.stride;
  if (s < 1 || s > 2 || g.Ho < 1 || g.Wo < 1) return pl;
  P.N = g.N; P.C = g.C; P.H = g.H; P.W = g.W; P.Co = g.Co; P.kh = g.kh; P.kw = g.kw;
  P.stride = s; P.pad = g.pad; P.Ho = g.Ho; P.Wo = g.Wo; P.Cw = g.Cw;
  // stream geometry of a phase plane (see the header comment)
  P.dymin = floor_div(-g.pad, s); P.dxmin = floor_div(-g.pad, s);
  const int dymax = floor_div(g.kh - 1 - g.pad, s), dxmax = floor_div(g.kw - 1 - g.pad, s);
  P.leadY = -P.dymin; P.leadX = -P.dxmin;
  const int Hc = (g.H + s - 1) / s, Wc = (g.W + s - 1) / s;    // rows/columns of the largest plane
  const int Hd = std::max(std::max(Hc, g.Ho + dymax - P.leadY), g.Ho);
  const int Wd = std::max(std::max(Wc, g.Wo + dxmax - P.leadX), g.Wo);
  P.Hq = P.leadY + Hd; P.Wq = P.leadX + Wd;
  P.L = (long long)g.N * P.Hq * P.Wq;
  P.ntiles = (int)((P.L + kTileM - 1) / kTileM);
  P.pair = pair ? 1 : 0;
  if (pair) P.ntiles = (P.ntiles + 1) / 2;               // a work tile is two stream tiles
  const int halo = (dymax - P.dymin) * P.Wq + (dxmax - P.dxmin);
  P.ppix = (kTileM + halo + 1 + 7) / 8 * 8;             // +1: a lone piece reads one pixel further
  if (P.L + P.ppix + 2 * kTileM >= (1ll << 31)) return pl;  // stream positions stay below 2^31
  // packed input rows one patch can touch: its stream rows, `stride` input rows each; the
  // copy is an aligned superset (up to 12 bytes before, 15 after)
  const long long raw_rows = ((long long)(P.ppix - 1) / P.Wq + 2) * s;
  const long long raw_bytes = (raw_rows * g.W * g.Cw * 4 + 12 + 15 + 15) / 16 * 16;
  if (raw_bytes > (long long)kSmemMax) return pl;
  P.raw_plane = (uint32_t)raw_bytes;
  P.raw_bytes = (uint32_t)planes * P.raw_plane;
  P.nplanes = s * s * g.Cw;
  P.patch_bytes = (uint32_t)P.nplanes * (uint32_t)P.ppix * 16u;
  // K-steps
  P.row_words = g.kh * g.kw * g.Cw;
  P.nsteps = (P.row_words + 1) / 2;
  if (P.nsteps > kMaxSteps) return pl;
  // shared memory: control, weight stages, patch buffers
  // per-filter vectors (alpha; fused: also the next scale and shift), padded to whole slabs
  P.off_vec = (uint32_t)((kCtrlBytes + 127) / 128 * 128);
  P.vec_len = (g.Co + 15) / 16 * 16 + 512;          // every slab of any width ends inside it
  P.off_ring = (uint32_t)((P.off_vec + (size_t)(fuse ? 3 : 1) * P.vec_len * 4 + 127) / 128 * 128);
  if (P.off_ring + 4096 > kSmemMax) return pl;
  const size_t avail = kSmemMax - P.off_ring;
  // st weight stages, pb patch buffers, nraw raw buffers for each subgroup of patch warps
  auto subgroups = [&](int pb) { return pb >= kPatWarps ? kPatWarps : 1; };
  auto fits = [&](int st, int pb, int nraw) {
    return (size_t)st * P.stage_bytes + (size_t)pb * P.patch_bytes +
           (size_t)(subgroups(pb) * nraw) * P.raw_bytes <= avail;
  };
  // as few slabs as fit two accumulators in the tensor-memory columns
  const int max_nt = pair ? 224 : 240;
  int min_slabs = (g.Co + max_nt - 1) / max_nt;
  // Items for fewer than half the SMs: narrower slabs on up to half of them, a CTA then expands and
  // drains less (512 channels, 7x7, one image: 15.6 -> 9.4 us; 64 channels, 14x14: 6.7 -> 6.5 us).  With
  // few K-steps the drain counts most and 16 filters win, else 32.  A small problem fills its one item's
  // stages in few, large steps (`few` in plan_stage): the latency per stage is what it waits for.  Fused, 64
  // filters: every slab adds planes of partial sums (352 channels, 9x9, 224 filters 3x3: 21.4 us in slabs of
  // 128, 13.3 of 64, 15.8 of 32; 0.87 of the time in the median of 68 drawn shapes of up to four images).
  // Narrower slabs than those that spread the problem stay one item per SM (480 channels, 51x51, 192 filters
  // 3x3, three images, in 12 resident slabs of 16: 28.7 us, streaming 14.8); with two bit planes, whose patches
  // cost more, two items (256 channels, 23x23, 120 filters 5x5, 12 images, k = 2: 16.3 us, streaming 22.1).
  // Beyond 16 slabs the resident search below gives up and the shape streams, which is the faster there
  // (16 channels, 5x5, 832 filters 3x3, two images: 7.0 us, 9.1 resident; 1.04 to 1.30 over 19 drawn shapes).
  const int spread = (int)kSms / 2 / P.ntiles;
  const bool few = !pair && min_slabs <= spread;
  if (few) {
    const int width = fuse ? 64 : P.nsteps < 16 ? 16 : 32;
    min_slabs = std::max(min_slabs, std::min(spread, (g.Co + width - 1) / width));
  }
  int stages = 0, npb = 0;
  P.resident = 0;
  const int units = (int)kSms / (pair ? 2 : 1);
  const int stream_slabs = std::max(min_slabs, (g.Co + 127) / 128);
  // Several slabs of few K-steps: the resident schedule drains with three warps per quarter of the lanes and
  // builds a patch per item, the streaming one drains with two and builds a patch per tile.  The time of the
  // fullest CTA from what was measured: per 16 columns drained 6 and 9 (with a residual 11 and 16), per plane
  // and 32 positions of a patch 1 (0.055 us).  79 images, 80 channels, 49x49, 912 filters 3x3 stride 2: 98 us
  // streaming, 60 resident; 37 images, 544 channels, 51x47, 256 filters 1x1 with a residual: 70 and 52; 128
  // channels, 28x28, 256 filters 3x3 stride 2, 256 images: 27.0 and 29.5.  Without a residual streaming also
  // wins within a tenth: of 14 drawn shapes where the sides differ by that or the choice was wrong, those up to
  // 1.09 were faster streaming (72 images, 192 channels, 48x48, 400 filters 1x1 stride 2: 29.3 and 32.6 us),
  // those from 1.12 resident (84 images, 720 channels, 17x53, 448 filters 1x1: 70 and 50 us).
  auto streams_faster = [&]() {
    const int snt = slab_width(g.Co, stream_slabs, pair || fuse), sns = (g.Co + snt - 1) / snt;
    const int patch = P.nplanes * ((P.ppix + 31) / 32), group = units / P.nslabs;
    auto time = [&](long long items, int drain, int patch_per_item) {
      return patch + drain + (items - 1) * std::max(drain, patch_per_item);
    };
    const long long res = time((P.ntiles + group - 1) / group, (residual ? 11 : 6) * P.NT / 16, patch);
    const long long str = time(((long long)P.ntiles * sns + units - 1) / units, (residual ? 16 : 9) * snt / 16, (patch + sns - 1) / sns);
    return (residual ? 11 : 10) * str < 11 * res;
  };
  if (schedule == 0) {
    // Resident: the widest slab whose expanded rows fit beside two patches.  Every slab needs its own
    // patch per tile and narrow MMAs re-read the pixel operand more often.  So (measured) several slabs
    // pay only from 128 filters (a pair: 96; 512 channels, 7x7, residual: 45.6 -> 34.1 us) and, with fewer
    // than two K-steps per plane of the patch, where streams_faster() says no.  The fused epilogue, half as long
    // again, outweighs the patches whatever the kernel: resident wherever it fits (16 channels, 34x34, 768
    // filters 1x1, 58 images: 136 us streaming, 64 resident; 0.68 of the time in the median of 68 drawn shapes of
    // several slabs).
    for (int ns = min_slabs; ns <= 16 && !P.resident; ++ns) {
      P.NT = slab_width(g.Co, ns, pair || fuse);
      P.nslabs = (g.Co + P.NT - 1) / P.NT;
      P.NTh = pair ? P.NT / 2 : P.NT;
      if (P.nslabs > 1 && (!few || P.ntiles * ns > (int)kSms * planes)) {
        if (P.NT < (pair ? 96 : 128)) break;
        if (!fuse && P.nsteps < 2 * P.nplanes && (pl.by_time = streams_faster())) break;
      }
      // (Lending four of the weight warps to the patch builders where a pixel has many channel
      // words was the better split while the drain loop was longer; since its trimming twelve
      // draining warps win on every layer measured: conv4 50.4 -> 48.1 us, conv5 39.4 -> 37.3.)
      plan_stage(P, few);
      const int nst = (P.nsteps + P.mps - 1) / P.mps;
      if (nst <= kMaxBarStages && fits(nst, 2, 1)) {
        P.resident = 1;
        stages = nst; npb = 2;
        // With a third buffer each patch warp builds whole patches by itself: of one or two items the first would
        // be built by one warp while the others wait (one: 37 images, 100 channels, 15x17, 77 filters 5x5 10.7 -> 9.9
        // us, 60 images, 40 channels, 30x30, stride 2 8.7 -> 7.4; two: 128 channels, 28x28, 40 images 12.4 -> 11.9).
        const bool many_items = (long long)P.ntiles * P.nslabs > 2 * units;
        if (!few && many_items && fits(stages, 3, 1)) npb = 3;
        if (npb == 3 && fits(stages, 4, 2)) npb = 4;     // a second raw buffer comes first
      }
    }
  }
  if (!P.resident) {
    int ns = stream_slabs;
    if (pair) {
      // Up to 224 filters per slab: the expansion, the longest part of an item, takes the same time for the
      // rows between two powers of two, so wider slabs pay where they save rounds of the pairs over the items
      // (928 channels, 38x38, 912 filters 5x5, two images: 92.6 us in 8 slabs of 128, 60.8 in 5 of 192) and
      // at equal estimates (544 channels, 22x53, 176 filters 3x3, 8 images: 23.5 -> 21.2).  Only where stages
      // of four K-steps still fit.  Of 175 drawn shapes of 64 K-steps and more 29 change, to 0.66 .. 1.07.
      auto rows = [&](int n) {
        int r = 16;
        while (2 * r < slab_width(g.Co, n, true)) r *= 2;
        return r;
      };
      auto time = [&](int n) { return ((long long)P.ntiles * n + units - 1) / units * rows(n); };
      // Up to 256 where every pair has one item: there is then no next item for a second accumulator (1024 channels,
      // 7x7, 256 filters, 64 images 79.7 us in two slabs, 71.0 in one: the MMAs of 256 columns leave shared
      // memory a quarter of its bandwidth, those of 128 none; two rounds: 500 filters, 20x20, 32.3 -> 34.7).
      for (int n = stream_slabs - 1; n >= (g.Co + 255) / 256; --n) {
        if (n < min_slabs && (fuse || P.ntiles * n > units)) break;
        const size_t ring = (size_t)3 * 4 * 32 * (slab_width(g.Co, n, true) / 2);
        if (time(n) <= time(ns) && ring + P.patch_bytes + P.raw_bytes <= avail) ns = n;
      }
    }
    P.NT = slab_width(g.Co, ns, pair || fuse);
    P.nslabs = (g.Co + P.NT - 1) / P.NT;
    P.NTh = pair ? P.NT / 2 : P.NT;
    // stages of four units per thread of a group of warps (see weight_stream), shorter ones where the
    // patch leaves little room; a stage per group at least
    if (P.NTh > 32 * kGroupWarps) return pl;             // a thread expands one row
    P.rows_mod = 16;
    while (P.rows_mod < P.NTh) P.rows_mod *= 2;
    const int subs = 32 * kGroupWarps / P.rows_mod;
    P.mps = std::min(8, 4 * subs);
    while (P.mps > 4 && P.nsteps < 3 * P.mps) P.mps /= 2;   // short items: smaller stages start sooner
    // Long items are bound by the expansion, short ones by the epilogue: two warps per quarter of the
    // lanes in place of a weight group (1024 channels, 1x1: 27.2 -> 25.6 us; 512 channels, 3x3, 72 K-steps:
    // 32.8 -> 34.7 us).  The fused epilogue is the longer one (245 channels, 52x52, 640 filters 3x3 stride 2,
    // 16 images: 49 -> 40 us with two; 976 channels, 192 filters, 140 K-steps: 96 -> 114).
    P.wgt_groups = P.nsteps < (fuse ? kLongFused : kLongItem) ? 2 : 3;
    auto stage = [&](int mps) { P.mps = mps; P.stage_bytes = (uint32_t)mps * (uint32_t)P.NTh * 32u; };
    stage(P.mps);
    while (P.mps > 1 && !fits(P.wgt_groups, 1, 1)) stage(P.mps / 2);
    if (!fits(P.wgt_groups, 1, 1)) return pl;
    // at least 3 stages and 1 patch; then patches up to 3, stages up to 8, one more patch
    stages = P.wgt_groups; npb = 1;
    while (stages < 4 && fits(stages + 1, npb, 1)) ++stages;
    while (npb < 3 && fits(stages, npb + 1, 1)) ++npb;
    while (stages < kMaxStages && fits(stages + 1, npb, 2)) ++stages;
    while (npb < kMaxPatchBufs && fits(stages, npb + 1, 2)) ++npb;
  }
  P.nraw = fits(stages, npb, 2) ? 2 : 1;
  P.nacc = std::max(1, std::min(kMaxAcc, kMaxAccCols / P.NT));
  // warps per quarter of the lanes: resident, the four epilogue warps and the eight weight warps
  const int drain_warps = P.resident ? kEpiSplitMax : P.wgt_groups == 2 ? 2 : 1;
  const long long unit_items = ((long long)P.ntiles * P.nslabs + units - 1) / units;
  P.drain = plan_drain(P.NT / 16, std::min(drain_warps, P.NT / (fuse ? 32 : 16)), unit_items >= 4, fuse, P.nacc);
  if (fuse && (g.Co & 31) != 0) return pl;          // whole words of the next layer's input
  P.stages = stages; P.npb = npb;
  P.off_tab = 0u;
  // small patches: every patch warp builds whole patches on its own, three at a time
  P.pat_sub = subgroups(npb);
  P.off_patch = P.off_ring + (uint32_t)stages * P.stage_bytes;
  P.off_raw = P.off_patch + (uint32_t)npb * P.patch_bytes;
  pl.smem = (size_t)P.off_raw + (size_t)(P.pat_sub * P.nraw) * P.raw_bytes;
  if (!P.resident && pl.smem + (size_t)P.nsteps * 4 + 16 <= kSmemMax) {       // the descriptor table, where it fits
    P.off_tab = (uint32_t)((pl.smem + 15) / 16 * 16);
    pl.smem = (size_t)P.off_tab + (size_t)P.nsteps * 4;
  }
  // block-scaled instruction descriptor: e2m1 x e2m1, ue8m0 scales, M = 128 (256 for a
  // pair), N = NT
  P.idesc = (1u << 7) | (1u << 10) | ((uint32_t)(P.NT >> 3) << 17) | (1u << 23) |
            ((uint32_t)((pair ? 2 * kTileM : kTileM) >> 4) << 24);
  const int crem = g.C - 32 * (g.Cw - 1);
  P.tail_mask = crem == 32 ? 0xFFFFFFFFu : ((1u << crem) - 1u);
  for (int j = 0; j < 32; ++j) P.swap_mask[j] = 0u;
  P.any_swap = 0;
  for (int j = 0; j < P.nsteps; ++j) {
    bool swap;
    P.adesc_lo[j] = kstep_desc(P, j, &swap);
    if (swap) { P.swap_mask[j >> 5] |= 1u << (j & 31); P.any_swap = 1; }
  }
  auto magic = [](uint32_t d, uint32_t *m, int *sh) {
    int l = 0;
    while ((1u << l) < d) ++l;
    *sh = l;
    *m = (uint32_t)((((unsigned long long)1 << (31 + l)) + d - 1) / d);
  };
  magic((uint32_t)P.Wq, &P.div_wq_m, &P.div_wq_s);
  magic((uint32_t)P.Hq, &P.div_hq_m, &P.div_hq_s);
  const uint32_t ngrp = (uint32_t)patch_groups(P.Cw, P.resident != 0);
  magic((uint32_t)(s * s) * ngrp, &P.div_pg_m, &P.div_pg_s);
  magic(ngrp, &P.div_g_m, &P.div_g_s);
  P.wq_rcp = (uint32_t)((((unsigned long long)1 << 32) + P.Wq - 1) / P.Wq);    // (0 for a width of 1: no table then)
  P.pat_table = (P.ppix + P.Wq - 2) / P.Wq + 1 <= 32 && P.Wq > 1;
  pl.ok = true;
  return pl;
}

}  // namespace

namespace {

// The plan of a variant.  kTcAuto: one CTA per SM unless only a pair, each CTA holding half of a slab, can keep
// the filters resident, or the items are long (see below).  Neither resident: pairs where the items are long (each CTA
// expands half the rows of a slab; 1024 channels, 1x1, 16 K-steps: 16.9 -> 17.5 us) and the slabs wide enough to
// fill a pair.  Over 255 drawn shapes the choice takes 1.010 of the time of the best variant (geometric mean;
// 233 of them within 2 %, 245 within 5 %).
Plan plan_variant_uncached(const ConvGeom &g, TcVariant v, bool fuse, int planes, bool residual) {
  switch (v) {
    case kTcSingle: return make_plan(g, 0, false, fuse, planes, residual);
    case kTcSingleStream: return make_plan(g, 1, false, fuse, planes, residual);
    case kTcPair: return make_plan(g, 0, true, fuse, planes, residual);
    case kTcPairStream: return make_plan(g, 1, true, fuse, planes, residual);
    default: break;
  }
  Plan single = make_plan(g, 0, false, fuse, planes, residual);
  // From 32 K-steps on the MMAs bound an item, and one thread of a pair issues those of two SMs at the cost of
  // one's; against that the two CTAs wait for each other's patches and accumulators at every item.  Measured, pair
  // against single CTAs, both resident, 26 to 75 K-steps: two slabs and five items and more per CTA 0.90 from 32
  // K-steps (AlexNet conv2 58.6 -> 54.9 us; 219 channels, 20x20, 256 filters 3x3, 160 images 0.91), 0.96 .. 0.98
  // at 27, with fewer items 0.99 .. 1.29.  One slab, where a single CTA has every filter and each patch is built
  // once, 1.03 over 88 shapes (0.89 .. 1.19; with five items and more from 32 K-steps 0.99 over 20, no size tells
  // the better ones apart); three slabs of 128, which a pair makes two of 192, 0.99 and 1.04, conv3 1.10.
  // Streaming, slabs wider than 64: 0.87 (0.74 .. 1.02) over 9 shapes of 32 to 63 K-steps, 0.82 (0.58 .. 1.02) over 25
  // of more (256 channels, 14x14, 512 filters 3x3 stride 2, 256 images 24.7 -> 22.6 us).
  const bool long_items = !fuse && planes == 1 && single.ok && single.P.nsteps >= kPairSteps;
  if (single.ok && single.P.resident) {
    if (long_items && single.P.nslabs == 2 && single.P.ntiles * 2 >= 5 * (int)kSms) {
      const Plan pair = make_plan(g, 0, true, fuse, planes, residual);
      if (pair.ok && pair.P.resident) return pair;
    }
    return single;
  }
  // a problem of few items is better spread over single CTAs
  if (single.ok && 2 * single.P.ntiles * single.P.nslabs <= (int)kSms) return single;
  Plan pair = make_plan(g, single.by_time ? 1 : 0, true, fuse, planes, residual);
  if (pair.ok && (pair.P.resident || !single.ok || (pair.P.NT > 64 && (long_items || pair.P.nsteps >= kLongItem)))) return pair;
  return single;
}

template <bool kRes, bool kPair, bool kFuse, bool kTwo = false>
cudaError_t launch_variant(const Plan &pl, unsigned units, cudaStream_t st) {
  return launch_kernel(binconv_tc_kernel<kRes, kPair, kFuse, kTwo>, dim3(kPair ? 2 * units : units), kRes ? kThreadsRes : kThreadsStream, pl.smem, st,
                       kPair ? 2u : 1u, pl.P);
}

}  // namespace

// The last plans made, by (geometry, variant, fused, bit planes, residual): one call of the library plans its shape
// two or three times (support check, then launch), and a network repeats a few shapes; planning
// evaluates up to 800 descriptor words.  Plans hold no pointers until a launcher fills them in.
namespace {

struct PlanKey {
  int N, C, H, W, Co, kh, kw, stride, pad, variant, fuse, planes, residual;
  bool operator==(const PlanKey &o) const {
    return N == o.N && C == o.C && H == o.H && W == o.W && Co == o.Co && kh == o.kh && kw == o.kw &&
           stride == o.stride && pad == o.pad && variant == o.variant && fuse == o.fuse && planes == o.planes && residual == o.residual;
  }
};

Plan plan_variant(const ConvGeom &g, TcVariant v, bool fuse, int planes, bool residual) {
  constexpr int kSlots = 16;
  static std::mutex mu;
  static PlanKey keys[kSlots];
  static Plan plans[kSlots];
  static bool used[kSlots] = {};
  static int next = 0;
  const PlanKey key{g.N, g.C, g.H, g.W, g.Co, g.kh, g.kw, g.stride, g.pad, (int)v, fuse ? 1 : 0, planes, residual ? 1 : 0};
  std::lock_guard<std::mutex> lock(mu);
  for (int i = 0; i < kSlots; ++i)
    if (used[i] && keys[i] == key) return plans[i];
  const int slot = next;
  next = (next + 1) % kSlots;
  plans[slot] = plan_variant_uncached(g, v, fuse, planes, residual);
  keys[slot] = key;
  used[slot] = true;
  return plans[slot];
}

}  // namespace

bool umma_tc_supported(const ConvGeom &g, TcVariant v, int planes) { return plan_variant(g, v, false, planes, false).ok; }

bool tc_plan_info(const ConvGeom &g, TcVariant v, bool fuse, int planes, bool residual, xnor_conv_plan *out) {
  const Plan pl = plan_variant(g, v, fuse, planes, residual);
  if (!pl.ok) return false;
  out->tensor_cores = 1;
  out->resident = pl.P.resident; out->pair = pl.P.pair; out->slabs = pl.P.nslabs; out->slab_filters = pl.P.NT;
  return true;
}

namespace {

cudaError_t launch_plan(Plan &pl, cudaStream_t st, bool fuse) {
  TcParams &P = pl.P;
  static bool attr_flags[64] = {};
  bool &attr_set = attr_done_for_current_device(attr_flags);
  if (!attr_set) {
    const void *kernels[12] = {(const void *)binconv_tc_kernel<false, false, false, false>,
                               (const void *)binconv_tc_kernel<true, false, false, false>,
                               (const void *)binconv_tc_kernel<false, true, false, false>,
                               (const void *)binconv_tc_kernel<true, true, false, false>,
                               (const void *)binconv_tc_kernel<false, false, true, false>,
                               (const void *)binconv_tc_kernel<true, false, true, false>,
                               (const void *)binconv_tc_kernel<false, true, true, false>,
                               (const void *)binconv_tc_kernel<true, true, true, false>,
                               (const void *)binconv_tc_kernel<false, false, false, true>,
                               (const void *)binconv_tc_kernel<true, false, false, true>,
                               (const void *)binconv_tc_kernel<false, true, false, true>,
                               (const void *)binconv_tc_kernel<true, true, false, true>};
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 12 && e == cudaSuccess; ++i)
      e = cudaFuncSetAttribute(kernels[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)kSmemMax);
    if (e != cudaSuccess) { (void)cudaGetLastError(); return e; }
    attr_set = true;
  }
  const long long total = (long long)P.ntiles * P.nslabs;
  const int sms = sm_count_of_current_device();
  // one CTA per SM, or one pair per two SMs
  const unsigned units = (unsigned)std::min<long long>(total, P.pair ? sms / 2 : sms);
  cudaError_t e_;
  if (fuse) {
    if (P.pair) e_ = P.resident ? launch_variant<true, true, true>(pl, units, st) : launch_variant<false, true, true>(pl, units, st);
    else e_ = P.resident ? launch_variant<true, false, true>(pl, units, st) : launch_variant<false, false, true>(pl, units, st);
  } else if (P.xp2 != nullptr) {
    if (P.pair) e_ = P.resident ? launch_variant<true, true, false, true>(pl, units, st) : launch_variant<false, true, false, true>(pl, units, st);
    else e_ = P.resident ? launch_variant<true, false, false, true>(pl, units, st) : launch_variant<false, false, false, true>(pl, units, st);
  } else {
    if (P.pair) e_ = P.resident ? launch_variant<true, true, false>(pl, units, st) : launch_variant<false, true, false>(pl, units, st);
    else e_ = P.resident ? launch_variant<true, false, false>(pl, units, st) : launch_variant<false, false, false>(pl, units, st);
  }
  if (e_ != cudaSuccess) (void)cudaGetLastError();
  return e_;
}

}  // namespace

cudaError_t launch_binconv_tc(const uint32_t *xp, const uint32_t *wp, const float *alpha,
                              const float *K, const float *residual, const ConvGeom &g,
                              const EpiOpts &epi, float *out, int32_t *acc_out, TcVariant variant,
                              cudaStream_t st, const uint32_t *xp2) {
  Plan pl = plan_variant(g, variant, false, xp2 != nullptr ? 2 : 1, residual != nullptr);
  if (!pl.ok) return cudaErrorInvalidValue;
  TcParams &P = pl.P;
  P.xp = xp; P.xp2 = xp2; P.wp = wp; P.alpha = alpha; P.K = K; P.residual = residual;
  P.out = out; P.acc_out = acc_out;
  P.relu = epi.relu; P.out_scale = epi.out_scale; P.acc_shift = epi.acc_shift; P.acc_accum = epi.acc_accum;
  P.nscale = nullptr; P.nshift = nullptr; P.xp_next = nullptr; P.A_part = nullptr; P.Cw_next = 0;
  return launch_plan(pl, st, false);
}

// Partial planes of |y| sums that the fused kernel writes for this shape: one per filter slab
// and chunk of its columns.  0: not supported.
int tc_fused_parts(const ConvGeom &g, TcVariant variant) {
  const Plan pl = plan_variant(g, variant, true, 1, false);
  if (!pl.ok) return 0;
  return pl.P.nslabs * pl.P.drain.chunks;
}

cudaError_t launch_binconv_tc_fused(const uint32_t *xp, const uint32_t *wp, const float *alpha,
                                    const float *K, const float *residual, const ConvGeom &g,
                                    float *out, const float *next_scale, const float *next_shift,
                                    uint32_t *xp_next, float *A_part, TcVariant variant,
                                    cudaStream_t st) {
  Plan pl = plan_variant(g, variant, true, 1, false);
  if (!pl.ok) return cudaErrorInvalidValue;
  TcParams &P = pl.P;
  P.xp = xp; P.xp2 = nullptr; P.wp = wp; P.alpha = alpha; P.K = K; P.residual = residual;
  P.out = out; P.acc_out = nullptr;
  P.relu = (g.flags & XNOR_FLAG_RELU) ? 1 : 0; P.out_scale = 1.0f; P.acc_shift = 0; P.acc_accum = 0;
  P.nscale = next_scale; P.nshift = next_shift; P.xp_next = xp_next; P.A_part = A_part;
  P.Cw_next = (g.Co + 31) / 32;
  return launch_plan(pl, st, true);
}


namespace {

// One warp waits, with a limit of about a millisecond, on a barrier that nothing signals: the
// wait must give up, raise the CTA's abort flag and record XNOR_ERR_TIMEOUT.
__global__ void wait_timeout_selftest_kernel() {
  __shared__ __align__(8) uint64_t bar;
  __shared__ volatile int abort_flag;
  stream_order();
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  (void)mbar_wait_slow(smem_u32(&bar), 0u, &abort_flag, &g_status_tc, 1ll << 21);
}

}  // namespace

cudaError_t launch_wait_timeout_selftest(cudaStream_t st) {
  return launch_kernel(wait_timeout_selftest_kernel, dim3(1), 32, 0, st, 1);
}

cudaError_t read_status_tc(int *status) {
  cudaError_t e = cudaMemcpyFromSymbol(status, g_status_tc, sizeof(int));
  if (e == cudaSuccess && *status != 0) {
    const int zero = 0;
    e = cudaMemcpyToSymbol(g_status_tc, &zero, sizeof(int));
  }
#ifdef XNOR_BOUNDS_CHECK
  // checking build: a recorded violation wins over everything else (1000 + its site number)
  int site = 0;
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(&site, g_bounds_tc, sizeof(int));
  if (e == cudaSuccess && site != 0) {
    const int zero = 0;
    e = cudaMemcpyToSymbol(g_bounds_tc, &zero, sizeof(int));
    *status = 1000 + site;
  }
#endif
  return e;
}

}  // namespace xnor
