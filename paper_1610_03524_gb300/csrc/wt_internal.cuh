// wt_internal.cuh -- device-side types and helpers shared by the kernels of
// the GB300 wavelet library (not part of the public ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace wtk {

// Levels per partition pass (upper bound; a larger tau runs as passes of 4).
// With four, a thread's 32 elements need six plane moves for their levels and
// one element move, a tile has 15 runs of level bits and 16 of elements, and
// its tables are 64 bytes; eight levels in one pass would halve the passes'
// reads and writes of the elements, which are not what bounds them.
constexpr int TAU_MAX = 4;
constexpr uint32_t FULL = 0xffffffffu;

// device error word bits
// (ERR_INTERNAL: a prefix table disagreed with a tile; never for correct tables)
enum : uint32_t { ERR_SYMBOL = 1u, ERR_INTERNAL = 4u };

// structure shapes handled by the partition pass
enum Shape : int { SHAPE_WM = 0, SHAPE_WT = 1, SHAPE_HUFF = 2 };

// One tile of a pass: `count` consecutive elements of T_a starting at
// `start`, all inside node `node`.
struct TileDesc {
  uint64_t start;
  uint32_t count;
  uint32_t node;
  uint32_t seg0;  // index of the node's first tile
};

// Per-tile digit counts of a pass (the K sub-problems' per-node counts of
// Section 4.2) and their prefix sums across tiles, in chunks of 2^chsh tiles:
// tile ti's counts sit at tcnt[ti * TC_STRIDE + r] (u32, exclusive within its chunk
// after the scan) and chunk c's exclusive counts at tchunk[c * TC_STRIDE + r]
// (u64), the totals after the last chunk.
constexpr int TC_STRIDE = 1 << TAU_MAX;  // row stride of both tables
// Tiles per chunk: 64, which a block of 256 threads holds in one round of
// loads, and more from 2^20 tiles on, so that the cluster that scans the chunks
// walks at most 16384.
constexpr uint64_t MAX_CHUNKS = 16384;
inline int chunk_shift(uint64_t tiles) {
  int s = 6;
  while (((tiles + ((uint64_t)1 << s) - 1) >> s) > MAX_CHUNKS) s++;
  return s;
}

// Chunks of the passes whose counting kernel also scans the counts.
constexpr uint32_t SCAN_CHUNKS = 256;

// Symbols per tile of the partition pass.
#ifndef WT_PASS_T
#define WT_PASS_T 4096
#endif
constexpr int PASS_T = WT_PASS_T;

// Batched builds: the per-sequence part of a pass, one entry per sequence
// taking part in the launch.  Its tiles are tile0 .. tile0 + ceil(n/T) - 1 of
// the launch's tile numbering.
// The pass's class starts (wm_cls) and the sequence's zero counts (zeros) are
// planned on the device from the totals of the pass's own tile counts;
// sigma (first pass only, else 0) is the bound the tile counts check the
// symbols against.
struct SegDesc {
  const void* in;
  void* out;
  uint64_t* bits;
  uint64_t* wm_cls;
  uint64_t* zeros;
  uint32_t* err;
  uint64_t n;
  uint32_t tile0;
  uint32_t sigma;
  int in_w, out_w, L, a, t, rbits;
};

struct PassParams {
  // input sequence T_a (elements hold the rbits = L - a low bits still needed)
  const void* in;
  int in_w;                 // bytes per input element (1, 2, 4)
  // output sequence T_{a+t}, narrowed to rbits - t bits (nullptr on the last pass)
  void* out;
  int out_w;
  // geometry
  int L;                    // total levels (max code length for HUFF)
  int a, t;                 // first level of the pass, levels in the pass
  int rbits;                // bits per input element that matter (L - a)
  int shape;
  // outputs
  uint64_t* bits;           // level bitmaps (or digit levels)
  const uint64_t* lvl_off;  // HUFF: word offset per level (the others' levels, of n_in
  const uint64_t* lvl_len;  // elements each, stand back to back), and its elements
  // class starts
  const uint64_t* wm_cls;   // WM: per level j of the pass, 2^j+1 starts at 2^j-1+j
  const uint64_t* wt_C;     // WT: starts of the nodes of level a + t, 2^(a+t) + 1
  const uint64_t* hf_node;  // HUFF: starts of the internal nodes, per level + sentinel
  const uint64_t* hf_lvl;   // HUFF: per level l: [3l] table offset, [3l+1] first internal prefix, [3l+2] count
  // tiles
  const TileDesc* tiles;    // nullptr: uniform tiles of TILE elements over n_in
  const uint32_t* ntiles_dev;
  uint32_t ntiles;
  uint64_t n_in;
  uint32_t tile0;           // first tile of the sequence (0 unless batched)
  uint32_t sigma;           // first passes: the tile counts check S[i] < sigma (0: no check)
  // batched builds: per-sequence parts, sorted by tile0
  const SegDesc* segs;
  uint32_t nsegs;
  // prefix sums of the tiles' digit counts (see TileDesc)
  const uint32_t* tcnt;
  const uint64_t* tchunk;
  uint32_t chsh;         // log2 of the tiles per chunk
  uint32_t* tick;           // zeroed tickets of the counts' scans, or nullptr
  uint32_t* err;
  // 16-byte units of a later pass's levels to zero, `clear_per` of them per
  // tile (nullptr: none); see clear_share
  uint4* clear;
  uint64_t clear_units, clear_per;
};

// Zero tile ti's share of `units` 16-byte units at `p`: units
// [ti * per, (ti + 1) * per), per = ceil(units / tiles) taken on the host.
__device__ __forceinline__ void clear_share(uint4* p, uint64_t units, uint64_t per, uint64_t ti,
                                            int tid, int nthreads) {
  const uint64_t b = ti * per;
  const uint64_t e = b + per < units ? b + per : units;
  for (uint64_t i = b + (uint64_t)tid; i < e; i += (uint64_t)nthreads)
    __stcs(p + i, make_uint4(0u, 0u, 0u, 0u));
}

__device__ __forceinline__ uint32_t rev_bits(uint32_t k, int j) {
  return j == 0 ? 0u : (__brev(k) >> (32 - j));
}

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

}  // namespace wtk
