// How the warps that share a quarter of the tensor-memory lanes divide the accumulators' columns
// (internal; plain arithmetic of the host and of the draining warps).
#pragma once

#ifdef __CUDACC__
#define XNOR_HD __host__ __device__ __forceinline__
#else
#define XNOR_HD inline
#endif

namespace xnor {

// An item's groups of 16 columns are cut into chunks, and the chunks of all items in sequence are dealt
// to the warps in turn: warp e starts with chunk e of item 0 and goes on `split` chunks at a time.
struct Drain {
  int split;             // warps per quarter of the lanes
  int chunk, chunks;     // groups of a chunk (the last has what is left), chunks of an item
  int rotate;            // 1: the turns move on by a warp from item to item

  // the chunk of the next item that a warp comes to when its count runs over the end of an item (c >= chunks)
  XNOR_HD int carry(int c) const {
    c -= chunks + rotate;
    return c < 0 ? c + split : c;
  }
};

// many: four and more items per CTA (pair).  accumulators: buffers that the items take in turn.
//
// A draining warp may have no chunk in some items.  It finds an item's accumulator full by the parity of that
// buffer's barrier, which tells apart two consecutive uses only.  So when it waits for an item it must know that the
// buffer's use before is over, that is, have seen an item no more than `accumulators` back (they are committed
// in order): ceil(split / chunks) <= accumulators.  Beyond that it would take an earlier item's accumulator
// for the one it waits for, with wrong sums and no expired wait.  Fewer warps take turns then.  (No plan needs that
// today: one chunk is at most 64 filters, which leave four accumulators for three warps.)
//
// What a warp does per item (its pixel, K, the waits: some 150 instructions) was a third of all instructions while
// every warp took a share of every item: 64 channels, 56x56, 64 filters 3x3, 256 images 71.8 -> 63.1 us in chunks
// of four groups, with a residual 107.0 -> 90.5; 128 channels, 28x28: 36.2 -> 32.7 and 51.4 -> 49.0; fused, the
// same two layers 102 -> 82 and 50 -> 41.  With fewer items than warps take turns over, all of them share an
// item, whose latency then counts (fused, one image: 7.4 us, in chunks of 64 filters 7.7).
//
// Where the number of chunks is a multiple of the number of warps, a warp would meet the same chunk in every item.
// The turns then move on from item to item if the short last chunk leaves some warp more than an even share of
// whole groups: 64 channels, 56x56, 144 filters 3x3 (4 + 4 + 1 groups over three warps), 128 images 78.5 -> 63.9
// us; 28x28, 200 images with a residual 46.4 -> 41.7, streaming 92.5 -> 69.9.  Chunks of even size instead (3 + 3 +
// 3): 64.3, 42.6 and 76.4, and slower where four groups gain (1x1, 256 images 28.1 fixed, 28.3 in turn, 31.6 even).
// Without need: 160 filters 22.1 -> 22.5, 176 24.0 -> 24.4.
//
// Fused, a chunk is an even number of groups (a pair is a packed word of the next layer's input).
inline Drain plan_drain(int groups, int warps, bool many, bool fused, int accumulators) {
  Drain d{};
  d.split = warps;
  d.chunk = (groups + warps - 1) / warps;
  if (fused) d.chunk = (d.chunk + 1) / 2 * 2;
  if (many && (!fused || d.chunk < 4)) d.chunk = 4;
  d.chunks = (groups + d.chunk - 1) / d.chunk;
  if ((warps + d.chunks - 1) / d.chunks > accumulators) return plan_drain(groups, warps - 1, many, fused, accumulators);
  const int unit = fused ? 2 : 1, share = (groups / unit + warps - 1) / warps * unit;
  d.rotate = d.chunks % warps == 0 && d.chunks / warps * d.chunk > share;
  return d;
}

}  // namespace xnor
