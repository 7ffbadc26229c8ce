// dirq.cu -- rank/select directories on every level (Section 5) and the
// batched query kernels (access / rank / select, Section 2 definitions).
//
// Binary levels (Section 5.1, rank of 0 only, Jacobson-style two-level
// counts): one 16-byte record per 2048-bit superblock, {u64 zeros before the
// superblock, 4 x u16 zeros before each 512-bit block inside it}, plus a
// trailing record with the level total.  Select (Section 5.1, positions of
// every k-th bit kept, here k = 4096): the position of the occurrence with
// 0-based index 4096k of each bit value; a query starts at the sample and
// searches superblocks, blocks, words, then the bit inside the word.
// Digit levels of the 4-ary tree (Section 5.2, per-value counts): one
// 64-byte record per 1024 digits, {4 x u64 counts of each value before the
// superblock, 4 blocks x 4 values u16 counts inside it}; select samples per
// digit value (Section 5.2 generalized select: the position of every 4096th
// occurrence of each value), four regions of n/4096 + 1 per level.
#include <algorithm>
#include <cooperative_groups.h>
#include <cstdio>
#include <vector>

#include "wt_host.h"
#include "wt_internal.cuh"

namespace wtk {

constexpr uint64_t NONE = ~0ull;

#define CK(x)                                                   \
  do {                                                          \
    cudaError_t e_ = (x);                                       \
    if (e_ != cudaSuccess) {                                    \
      fprintf(stderr, "wavelet: %s -> %s\n", #x, cudaGetErrorString(e_)); \
      cudaGetLastError(); /* reported here */                   \
      return e_ == cudaErrorMemoryAllocation ? WT_ERR_NO_MEMORY : WT_ERR_CUDA; \
    }                                                           \
  } while (0)

// exclusive u64 scan from build.cu
wt_status scan_excl_u64_pub(const uint64_t* in, uint64_t* out, uint64_t n, uint64_t* scratch,
                            cudaStream_t st);
uint64_t scan_scratch_pub(uint64_t n);

// r-th (0-based) set bit of v, by halving (__fns steps bit by bit)
__device__ __forceinline__ uint32_t sel64(uint64_t v, uint32_t r) {
  uint32_t x = (uint32_t)v, at = 0;
  const uint32_t pl = __popc(x);
  if (r >= pl) {
    r -= pl;
    x = (uint32_t)(v >> 32);
    at = 32;
  }
#pragma unroll
  for (uint32_t w = 16; w > 0; w >>= 1) {
    const uint32_t c = __popc(x & ((1u << w) - 1u));
    if (r >= c) {
      r -= c;
      x >>= w;
      at += w;
    }
  }
  return at;
}

// The eight words of a 64-byte directory block, requested together: one
// round of loads instead of one per word visited.  PADDED as the word count
// marks a level of the library's own (16-byte aligned, padded to 2048 bits);
// of a caller's bitvector the words at or past nw are not read.
constexpr uint64_t PADDED = ~0ull;
__device__ __forceinline__ void load_block(const uint64_t* lbits, uint64_t w0, uint64_t nw,
                                           uint64_t v[8]) {
  if (nw == PADDED) {
    const ulonglong2* p = (const ulonglong2*)(lbits + w0);
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const ulonglong2 q = p[i];
      v[2 * i] = q.x;
      v[2 * i + 1] = q.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = w0 + i < nw ? lbits[w0 + i] : 0ull;
  }
}

// ---------------------------------------------------------------------------
// binary directories
// ---------------------------------------------------------------------------
// Three launches build the directories of any number of levels: the counts
// of every group of DIR_GROUP superblocks of one level with their prefix sums
// inside the group (blk_first[l]: first group of level l), the prefix sums of
// the group totals of each level, and the absolute counts with the select
// samples.  One launch does when no level has more than one group.
#ifndef WT_DIR_SB_PER_WARP
#define WT_DIR_SB_PER_WARP 8
#endif
constexpr int DIR_SB_PER_WARP = WT_DIR_SB_PER_WARP;
constexpr int DIR_SB_PER_BLOCK = 8 * DIR_SB_PER_WARP;  // 256 threads
constexpr int DIR_GROUP = DIR_SB_PER_BLOCK;

// Up to DIR_SMALL levels: their first groups and metadata ride in the kernel
// parameters, so a block finds its level without a dependent load (else the
// tables are searched in global memory).
constexpr int DIR_SMALL = 32;
struct DirLevels {
  int nlev;
  uint64_t blk_first[DIR_SMALL + 1];
  LevelMeta meta[DIR_SMALL];
};

// the last level whose first group is at most b, found by the whole warp: 32
// entries a step (a binary search over the 39000 levels of a batch of 4096
// sequences is 16 dependent loads)
__device__ __forceinline__ int warp_find_level(const uint64_t* first, int nlev, uint64_t b) {
  const int lane = threadIdx.x & 31;
  int lo = 0, hi = nlev - 1;
  while (lo < hi) {
    const int step = (hi - lo + 31) >> 5;
    const int at = lo + (lane + 1) * step;
    const uint32_t c = (uint32_t)__popc(__ballot_sync(FULL, at <= hi && first[at] <= b));
    lo += (int)c * step;
    if (c < 32 && lo + step - 1 < hi) hi = lo + step - 1;
  }
  return lo;
}

// idx-th (0-based) set bit of m
__device__ __forceinline__ int nth_bit(uint32_t m, uint32_t idx) {
  int at = 0;
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) {
    const uint32_t c = __popc(m & ((1u << w) - 1u));
    if (idx >= c) {
      idx -= c;
      m >>= w;
      at += w;
    }
  }
  return at;
}

// position (inside superblock s, relative to its start) of the r-th
// (0-based) bit equal to bv, which lies in s; rel: the second word of its
// record; nw as for load_block
__device__ uint32_t find_in_sb(const uint64_t* lbits, uint64_t rel, uint64_t s, int bv,
                               uint32_t r, uint64_t nw) {
  int b = 3;
  for (; b > 0; b--) {
    const uint32_t z = (uint32_t)((rel >> (16 * b)) & 0xffffu);
    const uint32_t before = bv ? 512u * b - z : z;
    if (before <= r) break;
  }
  const uint32_t z = b ? (uint32_t)((rel >> (16 * b)) & 0xffffu) : 0u;
  r -= bv ? 512u * b - z : z;
  uint64_t v[8];
  load_block(lbits, 32 * s + 8 * (uint64_t)b, nw, v);
  uint64_t word = 0;
  int at = -1;
#pragma unroll
  for (int i = 0; i < 8; i++) {
    const uint64_t x = bv ? v[i] : ~v[i];
    const uint32_t c = (uint32_t)__popcll(x);
    if (at < 0) {
      if (c > r) {
        at = i;
        word = x;
      } else {
        r -= c;
      }
    }
  }
  if (at < 0) return 2047;
  return (uint32_t)((8 * b + at) * 64) + sel64(word, r);
}

// Select samples of a group: every 4096th zero and one of the level's
// superblocks s0 + 2 lane and the next (live; zeros zb before it and zs in it,
// rel the second word of its record).  About half of the superblocks of a dense
// level hold a sample, so a lane has about one search, and the warp's are dealt
// to its lanes instead of the zeros' and the ones' in turn.
__device__ __forceinline__ void warp_samples(const bool live[2], uint64_t s0, const uint64_t zb[2],
                                             const uint32_t zs[2], const uint64_t rel[2],
                                             const LevelMeta& m, const uint64_t* lb, bool aligned,
                                             uint64_t* samp) {
  const int lane = threadIdx.x & 31;
  // lanes with a sample: zeros of the first, of the second superblock; ones
  uint32_t has[4], first[5] = {0u, 0u, 0u, 0u, 0u};
#pragma unroll
  for (int c = 0; c < 4; c++) {
    const int e = c & 1;
    const uint64_t s = s0 + 2 * lane + e;
    bool h;
    if (c < 2) {
      h = live[e] && ((zb[e] + 4095) & ~4095ull) < zb[e] + zs[e];
    } else {
      const uint64_t nvalid = live[e] ? std::min<uint64_t>(2048, m.n - 2048 * s) : 0;
      const uint64_t ob = 2048 * s - zb[e];
      h = live[e] && ((ob + 4095) & ~4095ull) < ob + (nvalid - zs[e]);
    }
    has[c] = __ballot_sync(FULL, h);
    first[c + 1] = first[c] + __popc(has[c]);
  }
  for (uint32_t b = 0; b < first[4]; b += 32) {
    const uint32_t task = b + lane;
    const bool on = task < first[4];
    const int c = task >= first[3] ? 3 : (task >= first[2] ? 2 : (task >= first[1] ? 1 : 0));
    const uint32_t mask = c == 3 ? has[3] : (c == 2 ? has[2] : (c == 1 ? has[1] : has[0]));
    const uint32_t f = c == 3 ? first[3] : (c == 2 ? first[2] : (c == 1 ? first[1] : 0u));
    const int src = on ? nth_bit(mask, task - f) : 0, e = c & 1, bv = c >> 1;
    const uint64_t z0 = __shfl_sync(FULL, zb[0], src), z1 = __shfl_sync(FULL, zb[1], src);
    const uint64_t r0 = __shfl_sync(FULL, rel[0], src), r1 = __shfl_sync(FULL, rel[1], src);
    if (on) {
      const uint64_t ss = s0 + 2 * src + e, z = e ? z1 : z0;
      const uint64_t before = bv ? 2048 * ss - z : z, k = (before + 4095) >> 12;
      // a whole superblock's words can all be read; the last one's, and those
      // of a caller's bitvector off a 16-byte boundary, one by one up to the end
      const uint64_t nw = ss + 1 < m.nsb && aligned ? PADDED : (m.n + 63) / 64;
      samp[(bv ? m.s1_off : m.s0_off) + k] =
          2048 * ss + find_in_sb(lb, e ? r1 : r0, ss, bv, (uint32_t)(4096 * k - before), nw);
    }
  }
}

// Counts of one group: a record per superblock with the zeros before it in
// the group; the group's total into blk_tot.  ONE: the group is the whole
// level (block l = level l): its records are final, and its total record, zero
// count and samples are written too.  DRAM is the bound where all of a group's
// words are there: 2^33 bits in 148 us, 7.7 TB/s with the records, against 194
// us with a prefix sum per superblock and every word's bounds checked (16
// levels of 2^30 bits: 311 and 436 us).
template <bool SMALL, bool ONE>
__global__ void __launch_bounds__(256) k_dir_count(const uint64_t* bits, const LevelMeta* meta,
                                                   int nlev, const uint64_t* blk_first,
                                                   uint64_t* dir, uint64_t* blk_tot, uint64_t* samp,
                                                   uint64_t* zeros,
                                                   const __grid_constant__ DirLevels dl) {
  __shared__ LevelMeta sm;
  __shared__ uint64_t s_sb0;
  __shared__ uint32_t s_z[DIR_GROUP];
  __shared__ uint64_t s_rel[ONE ? DIR_GROUP : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  LevelMeta m;
  uint64_t sb0;
  if (SMALL) {
    int l = 0;
    if (ONE) l = (int)blockIdx.x;
    else
      while (l + 1 < dl.nlev && dl.blk_first[l + 1] <= blockIdx.x) l++;
    m = dl.meta[l];
    sb0 = ONE ? 0 : (blockIdx.x - dl.blk_first[l]) * DIR_GROUP;
  } else {
    if (warp == 0) {
      const int l = warp_find_level(blk_first, nlev, blockIdx.x);
      if (lane == 0) {
        sm = meta[l];
        s_sb0 = (blockIdx.x - blk_first[l]) * DIR_GROUP;
      }
    }
    __syncthreads();
    m = sm;
    sb0 = s_sb0;
  }
  // two superblocks at a time: lanes 0-15 the first, 16-31 the second, each
  // lane two consecutive words (one 16-byte load where aligned)
  const int hl = lane & 15, half = lane >> 4;
  const uint64_t s0 = sb0 + (uint64_t)warp * DIR_SB_PER_WARP;
  const uint64_t* lb = bits + m.bit_off;
  const bool vec = (((uintptr_t)lb) & 15) == 0;
  constexpr int NP = DIR_SB_PER_WARP / 2;
  static_assert(NP == 4, "four counts in two words");
  uint32_t z[NP];  // zeros of the lane's words
  if (vec && 2048 * (sb0 + DIR_GROUP) <= m.n) {
    const ulonglong2* const p = (const ulonglong2*)(lb + 32 * (s0 + half) + 2 * hl);
    ulonglong2 q[NP];
#pragma unroll
    for (int u = 0; u < NP; u++) q[u] = __ldcs(p + 32 * u);
#pragma unroll
    for (int u = 0; u < NP; u++) z[u] = 128 - __popcll(q[u].x) - __popcll(q[u].y);
  } else {
#pragma unroll
    for (int u = 0; u < NP; u++) {
      const uint64_t s = s0 + 2 * u + half;
      const int64_t rem = (int64_t)m.n - (int64_t)(2048 * s + 128 * (uint64_t)hl);
      const bool live = s < m.nsb && rem > 0;
      const int v0 = !live ? 0 : (rem >= 64 ? 64 : (int)rem);
      const int v1 = (!live || rem <= 64) ? 0 : (rem >= 128 ? 64 : (int)(rem - 64));
      const uint64_t* p = lb + 32 * s + 2 * hl;
      // words past the last valid bit are not read (a caller bitvector may end there)
      ulonglong2 q = make_ulonglong2(0ull, 0ull);
      if (v1 && vec) {
        q = __ldcs((const ulonglong2*)p);
      } else {
        if (v0) q.x = __ldcs(p);
        if (v1) q.y = __ldcs(p + 1);
      }
      z[u] = v0 + v1 - __popcll(q.x) - __popcll(q.y);
    }
  }
  // all four superblocks' prefix sums over the half's lanes at once, two 16-bit
  // counts a word; then lane u < 4 of the half has superblock u's record
  uint32_t za = z[0] | (z[1] << 16), zb = z[2] | (z[3] << 16);
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) {
    const uint32_t ya = __shfl_up_sync(FULL, za, o, 16), yb = __shfl_up_sync(FULL, zb, o, 16);
    if (hl >= o) {
      za += ya;
      zb += yb;
    }
  }
  // zeros before 512-bit blocks 1, 2, 3 of the superblock, and in all: lanes 3, 7, 11, 15
  const int u = hl & 3;
  uint32_t at[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const uint32_t xa = __shfl_sync(FULL, za, 4 * k + 3, 16), xb = __shfl_sync(FULL, zb, 4 * k + 3, 16);
    at[k] = ((u & 2 ? xb : xa) >> (16 * (u & 1))) & 0xffffu;
  }
  const uint64_t rel = ((uint64_t)(at[1] | (at[2] << 16)) << 32) | (at[0] << 16);
  const int i = warp * DIR_SB_PER_WARP + 2 * u + half;  // in the group
  if (hl < 4) {
    s_z[i] = at[3];
    if (ONE) s_rel[i] = rel;
  }
  __syncthreads();
  // zeros before each of the warp's superblocks in the group: lane i the sum
  // of the earlier warps' and of the warp's first i
  static_assert(DIR_GROUP == 64, "two superblocks a lane");
  const uint32_t a = s_z[2 * lane], b = s_z[2 * lane + 1];
  uint32_t inc = a + b;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc += y;
  }
  const uint32_t total = __shfl_sync(FULL, inc, 31);
  {
    // lane i / 2 holds the pair of superblock i
    const uint32_t pair = __shfl_sync(FULL, inc - a - b, warp * NP + u);
    const uint32_t prev = __shfl_sync(FULL, a, warp * NP + u);
    const uint64_t s = s0 + 2 * u + half;
    if (hl < 4 && s < m.nsb)
      *(ulonglong2*)(dir + m.dir_off + 2 * s) = make_ulonglong2(pair + (half ? prev : 0u), rel);
  }
  if (!ONE) {
    if (threadIdx.x == 0) blk_tot[blockIdx.x] = total;
  } else {
    if (threadIdx.x == 0) {
      *(ulonglong2*)(dir + m.dir_off + 2 * m.nsb) = make_ulonglong2(total, 0ull);
      if (zeros) zeros[blockIdx.x] = total;
    }
    __syncthreads();
    if (warp == 0) {
      const bool live[2] = {2 * (uint64_t)lane < m.nsb, 2 * (uint64_t)lane + 1 < m.nsb};
      const uint64_t zb[2] = {inc - a - b, inc - b}, rl[2] = {s_rel[2 * lane], s_rel[2 * lane + 1]};
      const uint32_t zs[2] = {a, b};
      warp_samples(live, 0, zb, zs, rl, m, lb, vec, samp);
    }
  }
}

// Exclusive prefix sums of tot[0 .. n) in place by the warps of a cluster of CL
// blocks, each a contiguous range, four values a lane and step; returns the
// grand total (to every thread).  (One block alone takes 36 us for the 65536
// groups of 2^33 bits: an SM's loads in flight bound it; eight take 14.)
template <int CL>
__device__ uint64_t cluster_scan_range(uint64_t* tot, uint64_t n) {
  namespace cg = cooperative_groups;
  __shared__ uint64_t ws[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int rank = CL > 1 ? (int)cg::this_cluster().block_rank() : 0;
  const uint64_t per = ((n + nw * CL - 1) / (nw * CL) + 127) & ~127ull;
  const uint64_t b0 = std::min<uint64_t>(per * (rank * nw + warp), n), b1 = std::min<uint64_t>(b0 + per, n);
  uint64_t sum = 0;
#pragma unroll 8
  for (uint64_t i = b0 + lane; i < b1; i += 32) sum += tot[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
  if (lane == 0) ws[warp] = sum;
  if (CL > 1) cg::this_cluster().sync();
  else __syncthreads();
  // lane w: warp w's sum of each block
  uint64_t carry = 0, all = 0;
  for (int r = 0; r < CL; r++) {
    const uint64_t* rs = CL > 1 ? cg::this_cluster().map_shared_rank(ws, r) : ws;
    const uint64_t x = lane < nw ? rs[lane] : 0ull;
    uint64_t before = r < rank || (r == rank && lane < warp) ? x : 0ull, every = x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      before += __shfl_xor_sync(FULL, before, o);
      every += __shfl_xor_sync(FULL, every, o);
    }
    carry += before;
    all += every;
  }
  if (CL > 1) cg::this_cluster().sync();  // the sums are read before a block ends
  for (uint64_t i0 = b0; i0 < b1; i0 += 128) {
    const uint64_t i = i0 + 4 * lane;
    uint64_t v[4], x = 0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      v[k] = i + k < b1 ? tot[i + k] : 0ull;
      x += v[k];
    }
    const uint64_t mine = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(FULL, x, o);
      if (lane >= o) x += y;
    }
    uint64_t at = carry + x - mine;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (i + k < b1) tot[i + k] = at;
      at += v[k];
    }
    carry += __shfl_sync(FULL, x, 31);
  }
  return all;
}

// The group totals of every level to prefix sums, and the level's total
// record: SMALL a cluster of DIR_CLUSTER blocks per level, else one warp.
constexpr int DIR_CLUSTER = 8;
template <bool SMALL>
__device__ __forceinline__ void dir_groups(int l, int rank, const LevelMeta* meta,
                                           const uint64_t* blk_first, uint64_t* blk_tot,
                                           uint64_t* dir, uint64_t* zeros, const DirLevels& dl) {
  const uint64_t b0 = SMALL ? dl.blk_first[l] : blk_first[l];
  const uint64_t b1 = SMALL ? dl.blk_first[l + 1] : blk_first[l + 1];
  const uint64_t total = cluster_scan_range<SMALL ? DIR_CLUSTER : 1>(blk_tot + b0, b1 - b0);
  if (rank == 0 && threadIdx.x == 0) {
    const uint64_t off = SMALL ? dl.meta[l].dir_off + 2 * dl.meta[l].nsb
                               : meta[l].dir_off + 2 * meta[l].nsb;
    *(ulonglong2*)(dir + off) = make_ulonglong2(total, 0ull);
    if (zeros) zeros[l] = total;
  }
}

__global__ void __cluster_dims__(DIR_CLUSTER, 1, 1) __launch_bounds__(512)
    k_dir_groups_small(uint64_t* blk_tot, uint64_t* dir, uint64_t* zeros,
                       const __grid_constant__ DirLevels dl) {
  dir_groups<true>((int)blockIdx.x / DIR_CLUSTER, (int)blockIdx.x % DIR_CLUSTER, nullptr, nullptr,
                   blk_tot, dir, zeros, dl);
}

__global__ void __launch_bounds__(32) k_dir_groups(const LevelMeta* meta, const uint64_t* blk_first,
                                                   uint64_t* blk_tot, uint64_t* dir, uint64_t* zeros,
                                                   const __grid_constant__ DirLevels dl) {
  dir_groups<false>((int)blockIdx.x, 0, meta, blk_first, blk_tot, dir, zeros, dl);
}

// Absolute counts and select samples: a warp per group, two superblocks a lane.
// (2^33 bits: 62 us; 83 with a superblock a lane, half of whose searches were
// idle, and 93 with only the changed half of each record stored.)
template <bool SMALL>
__global__ void __launch_bounds__(256) k_dir_finish(const uint64_t* bits, const LevelMeta* meta,
                                                    int nlev, const uint64_t* blk_first,
                                                    uint64_t ngroups, const uint64_t* blk,
                                                    uint64_t* dir, uint64_t* samp,
                                                    const __grid_constant__ DirLevels dl) {
  static_assert(DIR_GROUP == 64, "two superblocks a lane");
  const int lane = threadIdx.x & 31;
  const uint64_t g = (uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (g >= ngroups) return;  // a whole warp
  LevelMeta m;
  uint64_t s0;  // the group's first superblock
  if (SMALL) {
    int l = 0;
    while (l + 1 < dl.nlev && dl.blk_first[l + 1] <= g) l++;
    m = dl.meta[l];
    s0 = (g - dl.blk_first[l]) * DIR_GROUP;
  } else {
    const int l = warp_find_level(blk_first, nlev, g);
    m = meta[l];
    s0 = (g - blk_first[l]) * DIR_GROUP;
  }
  const uint64_t s = s0 + 2 * lane;
  const bool live[2] = {s < m.nsb, s + 1 < m.nsb};
  uint64_t* const ld = dir + m.dir_off;
  const uint64_t base = blk[g];
  ulonglong2 r0 = make_ulonglong2(0ull, 0ull), r1 = r0;
  if (live[0]) r0 = *(const ulonglong2*)(ld + 2 * s);
  if (live[1]) r1 = *(const ulonglong2*)(ld + 2 * s + 2);
  r0.x += base;
  r1.x += base;
  // zeros before the next superblock: of the level's last one, its total; after
  // the group's last one, the next group's
  uint64_t end0 = r1.x, end1 = __shfl_down_sync(FULL, r0.x, 1);
  if (live[0] && !live[1]) end0 = ld[2 * m.nsb];
  if (live[1] && s + 2 == m.nsb) end1 = ld[2 * m.nsb];
  else if (live[1] && lane == 31) end1 = blk[g + 1];
  if (live[0]) *(ulonglong2*)(ld + 2 * s) = r0;
  if (live[1]) *(ulonglong2*)(ld + 2 * s + 2) = r1;
  const uint64_t* lb = bits + m.bit_off;
  const uint64_t zb[2] = {r0.x, r1.x}, rel[2] = {r0.y, r1.y};
  const uint32_t zs[2] = {(uint32_t)(end0 - r0.x), (uint32_t)(end1 - r1.x)};
  warp_samples(live, s0, zb, zs, rel, m, lb, (((uintptr_t)lb) & 15) == 0, samp);
}

// ---------------------------------------------------------------------------
// digit-level (4-ary) directories
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t digit_match(uint64_t w, uint32_t d) {
  const uint64_t x = w ^ (0x5555555555555555ull * d);
  return ~(x | (x >> 1)) & 0x5555555555555555ull;
}

// The same three launches for digit levels (there are never more than
// DIR_SMALL): a group's records with the four values' counts before each
// superblock in the group, eight superblocks a warp, two at a time (each
// half-warp one: 16 lanes x two words = 1024 digits).  A lane holds 64 digits,
// counts the values 1 to 3 by their two bit planes (the zeros are the others),
// and the four lanes of a 256-digit block add up; lane (q, j) of a half then
// has block q of superblock j.  The group's totals of value d into blk_tot[d *
// ngroups + group].  (3*10^8 symbols in four levels: 51 us, 7.4 TB/s; a prefix
// sum per superblock and value took 181.)
__global__ void __launch_bounds__(256) k_mdir_count(const uint64_t* bits, uint64_t ngroups,
                                                    uint64_t* dir, uint64_t* blk_tot,
                                                    const __grid_constant__ DirLevels dl) {
  __shared__ uint32_t s_z[4][DIR_GROUP];
  int l = 0;
  while (l + 1 < dl.nlev && dl.blk_first[l + 1] <= blockIdx.x) l++;
  const LevelMeta m = dl.meta[l];
  const uint64_t sb0 = (blockIdx.x - dl.blk_first[l]) * DIR_GROUP;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int hl = lane & 15, half = lane >> 4;
  const uint64_t s0 = sb0 + (uint64_t)warp * DIR_SB_PER_WARP;
  const uint64_t* lb = bits + m.bit_off;
  constexpr int NP = DIR_SB_PER_WARP / 2;
  static_assert(NP == 4, "a block's four lanes take one superblock each");
  ulonglong2 w[NP];
  if (1024 * (sb0 + DIR_GROUP) <= m.n) {
#pragma unroll
    for (int u = 0; u < NP; u++) w[u] = __ldcs((const ulonglong2*)(lb + 32 * (s0 + 2 * u + half) + 2 * hl));
  } else {
#pragma unroll
    for (int u = 0; u < NP; u++) {
      const uint64_t s = s0 + 2 * u + half, first = 1024 * s + 64 * (uint64_t)hl;
      w[u] = make_ulonglong2(0ull, 0ull);
      if (first < m.n) {  // levels are padded to whole superblocks
        w[u] = __ldcs((const ulonglong2*)(lb + 32 * s + 2 * hl));
        const uint64_t rem = m.n - first;  // digits past the end as zeros
        if (rem < 64) w[u].y &= rem > 32 ? (1ull << (2 * (rem - 32))) - 1ull : 0ull;
        if (rem < 32) w[u].x &= (1ull << (2 * rem)) - 1ull;
      }
    }
  }
  uint32_t c12[NP], c3[NP];  // counts of the values 1 and 2 (16 bits each), and 3
#pragma unroll
  for (int u = 0; u < NP; u++) {
    constexpr uint64_t E = 0x5555555555555555ull;
    const uint64_t lo = (w[u].x & E) | ((w[u].y & E) << 1), hi = ((w[u].x >> 1) & E) | (w[u].y & ~E);
    c3[u] = (uint32_t)__popcll(lo & hi);
    c12[u] = ((uint32_t)__popcll(lo) - c3[u]) | (((uint32_t)__popcll(hi) - c3[u]) << 16);
  }
  // the block's sums, the lane's own superblock's kept
  uint32_t e = c3[0] | (c3[1] << 16), f = c3[2] | (c3[3] << 16);
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
#pragma unroll
    for (int u = 0; u < NP; u++) c12[u] += __shfl_xor_sync(FULL, c12[u], o);
    e += __shfl_xor_sync(FULL, e, o);
    f += __shfl_xor_sync(FULL, f, o);
  }
  const int q = hl >> 2, j = hl & 3;
  uint32_t n12 = j & 2 ? (j & 1 ? c12[3] : c12[2]) : (j & 1 ? c12[1] : c12[0]);
  uint32_t n3 = ((j & 2 ? f : e) >> (16 * (j & 1))) & 0xffffu;
  const uint32_t own12 = n12, own3 = n3;
#pragma unroll
  for (int o = 4; o < 16; o <<= 1) {  // up to and with block q
    const uint32_t y12 = __shfl_up_sync(FULL, n12, o, 16), y3 = __shfl_up_sync(FULL, n3, o, 16);
    if (hl >= o) {
      n12 += y12;
      n3 += y3;
    }
  }
  const uint64_t s = s0 + 2 * j + half;
  const int i = warp * DIR_SB_PER_WARP + 2 * j + half;  // in the group
  // digits of the superblock, of its blocks before q
  const uint64_t left = s < m.nsb ? m.n - 1024 * s : 0ull;
  const uint32_t len = left < 1024 ? (uint32_t)left : 1024u, upto = min(256u * q, len);
  if (q == 3) {
    const uint32_t n1 = n12 & 0xffffu, n2 = n12 >> 16;
    s_z[0][i] = len - n1 - n2 - n3;
    s_z[1][i] = n1;
    s_z[2][i] = n2;
    s_z[3][i] = n3;
  }
  n12 -= own12;
  n3 -= own3;
  const uint32_t b1 = n12 & 0xffffu, b2 = n12 >> 16, b0 = upto - b1 - b2 - n3;
  const uint64_t rec = q ? ((uint64_t)(b2 | (n3 << 16)) << 32) | (b0 | (b1 << 16)) : 0ull;
  __syncthreads();
  if (warp < 4) {  // value warp: its counts before each superblock of the group, in place
    const uint32_t a = s_z[warp][2 * lane], b = s_z[warp][2 * lane + 1];
    uint32_t inc = a + b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc += y;
    }
    s_z[warp][2 * lane] = inc - a - b;
    s_z[warp][2 * lane + 1] = inc - b;
    if (lane == 31) blk_tot[(uint64_t)warp * ngroups + blockIdx.x] = inc;
  }
  __syncthreads();
  if (s < m.nsb) {
    uint64_t* const r = dir + m.dir_off + 8 * s;
    r[q] = s_z[q][i];
    r[4 + q] = rec;
  }
}

// The groups' totals of every level and value to prefix sums, and the
// level's total record: a cluster per level and value.
__global__ void __cluster_dims__(DIR_CLUSTER, 1, 1) __launch_bounds__(512)
    k_mdir_groups(uint64_t ngroups, uint64_t* blk_tot, uint64_t* dir,
                  const __grid_constant__ DirLevels dl) {
  const int c = (int)blockIdx.x / DIR_CLUSTER, l = c >> 2, d = c & 3;
  const uint64_t total = cluster_scan_range<DIR_CLUSTER>(
      blk_tot + (uint64_t)d * ngroups + dl.blk_first[l], dl.blk_first[l + 1] - dl.blk_first[l]);
  if (blockIdx.x % DIR_CLUSTER == 0 && threadIdx.x == 0) {
    uint64_t* const r = dir + dl.meta[l].dir_off + 8 * dl.meta[l].nsb;
    r[d] = total;
    r[4 + d] = 0;
  }
}

// position (inside digit superblock s, relative to its start) of the r-th
// (0-based) occurrence of digit value d; the occurrence lies in s
__device__ uint32_t find_in_dsb(const uint64_t* lbits, const uint64_t* ldir, uint64_t s, uint32_t d,
                                uint32_t r) {
  int b = 3;
  for (; b > 0; b--)
    if (((ldir[8 * s + 4 + b] >> (16 * d)) & 0xffffull) <= r) break;
  r -= b ? (uint32_t)((ldir[8 * s + 4 + b] >> (16 * d)) & 0xffffull) : 0u;
  uint64_t v[8];
  load_block(lbits, 32 * s + 8 * (uint64_t)b, PADDED, v);
  uint64_t word = 0;
  int at = -1;
#pragma unroll
  for (int i = 0; i < 8; i++) {
    const uint64_t m = digit_match(v[i], d);
    const uint32_t c = (uint32_t)__popcll(m);
    if (at < 0) {
      if (c > r) {
        at = i;
        word = m;
      } else {
        r -= c;
      }
    }
  }
  if (at < 0) return 1023;
  return (uint32_t)((8 * b + at) * 32) + sel64(word, r) / 2;
}

// Absolute counts and the samples of each value (the position of every
// 4096th occurrence): 64 threads per group, the warp's searches dealt to its
// lanes.
__global__ void __launch_bounds__(256) k_mdir_finish(const uint64_t* bits, uint64_t ngroups,
                                                     const uint64_t* blk, uint64_t* dir,
                                                     uint64_t* samp,
                                                     const __grid_constant__ DirLevels dl) {
  const int lane = threadIdx.x & 31;
  const uint64_t g = (uint64_t)blockIdx.x * (256 / DIR_GROUP) + threadIdx.x / DIR_GROUP;
  const bool in = g < ngroups;
  int l = 0;
  while (l + 1 < dl.nlev && dl.blk_first[l + 1] <= g) l++;
  const LevelMeta m = dl.meta[l];
  const uint64_t s0 = (g - dl.blk_first[l]) * DIR_GROUP + threadIdx.x % DIR_GROUP - lane;
  const uint64_t s = s0 + lane;
  const bool live = in && s < m.nsb;
  uint64_t* const ld = dir + m.dir_off;
  const bool lastsb = s + 1 == m.nsb, lastg = (s + 1) % DIR_GROUP == 0;
  uint64_t at[4], end[4];
  ulonglong2 rec[2] = {make_ulonglong2(0ull, 0ull), make_ulonglong2(0ull, 0ull)};
  if (live) {
    rec[0] = *(const ulonglong2*)(ld + 8 * s);
    rec[1] = *(const ulonglong2*)(ld + 8 * s + 2);
  }
#pragma unroll
  for (int d = 0; d < 4; d++) {
    const uint64_t* const bd = blk + (uint64_t)d * ngroups;
    at[d] = end[d] = 0;
    if (live) {
      at[d] = bd[g] + (d & 1 ? rec[d >> 1].y : rec[d >> 1].x);
      if (lastsb) end[d] = ld[8 * m.nsb + d];
      else if (lastg) end[d] = bd[g + 1];
      else if (lane == 31) end[d] = bd[g] + ld[8 * s + 8 + d];
    }
    const uint64_t next = __shfl_down_sync(FULL, at[d], 1);
    if (live && lane < 31 && !lastsb && !lastg) end[d] = next;
  }
  // the middle of a group is read by one warp and written by the other
  __syncthreads();
  if (live) {
    *(ulonglong2*)(ld + 8 * s) = make_ulonglong2(at[0], at[1]);
    *(ulonglong2*)(ld + 8 * s + 2) = make_ulonglong2(at[2], at[3]);
  }
  uint32_t has[4], first[5] = {0u, 0u, 0u, 0u, 0u};
#pragma unroll
  for (int d = 0; d < 4; d++) {
    has[d] = __ballot_sync(FULL, live && ((at[d] + 4095) & ~4095ull) < end[d]);
    first[d + 1] = first[d] + __popc(has[d]);
  }
  const uint64_t* lb = bits + m.bit_off;
  const uint64_t cap = m.n / 4096 + 1;
  for (uint32_t b = 0; b < first[4]; b += 32) {
    const uint32_t task = b + lane;
    const bool on = task < first[4];
    const int d = task >= first[3] ? 3 : (task >= first[2] ? 2 : (task >= first[1] ? 1 : 0));
    const uint32_t mask = d == 3 ? has[3] : (d == 2 ? has[2] : (d == 1 ? has[1] : has[0]));
    const uint32_t f = d == 3 ? first[3] : (d == 2 ? first[2] : (d == 1 ? first[1] : 0u));
    const int src = on ? nth_bit(mask, task - f) : 0;
    uint64_t before = 0;
#pragma unroll
    for (int e = 0; e < 4; e++) {
      const uint64_t x = __shfl_sync(FULL, at[e], src);
      if (e == d) before = x;
    }
    if (on) {
      const uint64_t ss = s0 + src, k = (before + 4095) >> 12;
      samp[m.s0_off + (uint64_t)d * cap + k] =
          1024 * ss + find_in_dsb(lb, ld, ss, (uint32_t)d, (uint32_t)(4096 * k - before));
    }
  }
}

wt_status upload_meta(wt_struct* h) {
  const size_t nb = std::max<size_t>(h->meta.size(), 1) * sizeof(LevelMeta);
  if (!h->d_meta) CK(dmalloc((void**)&h->d_meta, nb, h->stream));
  if (!h->meta.empty()) return upload(h->d_meta, h->meta.data(), h->meta.size() * sizeof(LevelMeta), h->stream);
  return WT_OK;
}

// Binary directories and select samples of nlev levels described by d_meta
// or, when not null, by h_meta (offsets relative to bits / dir / samp); sb_first: first
// superblock of each level in one numbering, its first nlev + 1 entries used.
// zeros: when not null, each level's zero count is stored in zeros[l].
wt_status dir_build_levels(const uint64_t* bits, const LevelMeta* d_meta, uint32_t nlev,
                           const std::vector<uint64_t>& sb_first, uint64_t* dir, uint64_t* samp,
                           uint64_t* zeros, cudaStream_t st, const LevelMeta* h_meta) {
  if (nlev == 0) return WT_OK;
  // few levels with host metadata: the level tables go in the parameters
  const bool small = h_meta && nlev <= (uint32_t)DIR_SMALL;
  std::vector<uint64_t> blk_first((size_t)nlev + 1, 0);
  bool one = small;
  for (uint32_t l = 0; l < nlev; l++) {
    const uint64_t nsb = sb_first[l + 1] - sb_first[l];
    blk_first[l + 1] = blk_first[l] + (nsb + DIR_GROUP - 1) / DIR_GROUP;
    one = one && nsb <= (uint64_t)DIR_GROUP;
  }
  const uint64_t nblk = blk_first[nlev];
  DirLevels dl;
  memset(&dl, 0, sizeof(dl));
  if (small) {
    dl.nlev = (int)nlev;
    for (uint32_t l = 0; l <= nlev; l++) dl.blk_first[l] = blk_first[l];
    for (uint32_t l = 0; l < nlev; l++) dl.meta[l] = h_meta[l];
  }
  if (one) {
    k_dir_count<true, true><<<nlev, 256, 0, st>>>(bits, nullptr, (int)nlev, nullptr, dir, nullptr,
                                                  samp, zeros, dl);
    count_launch();
    CK(cudaGetLastError());
    return WT_OK;
  }
  Work wk{st};
  uint64_t *d_first = nullptr, *blk;
  TRY(wk.get(&blk, nblk + 1));
  const unsigned fgrid = (unsigned)((nblk + 7) / 8);
  if (small) {
    k_dir_count<true, false><<<(unsigned)nblk, 256, 0, st>>>(bits, nullptr, (int)nlev, nullptr, dir,
                                                            blk, samp, nullptr, dl);
    k_dir_groups_small<<<nlev * DIR_CLUSTER, 512, 0, st>>>(blk, dir, zeros, dl);
    k_dir_finish<true><<<fgrid, 256, 0, st>>>(bits, nullptr, (int)nlev, nullptr, nblk, blk, dir,
                                              samp, dl);
    count_launch(3);
  } else {
    TRY(wk.get(&d_first, (size_t)nlev + 1));
    TRY(upload(d_first, blk_first.data(), blk_first.size() * 8, st));
    if (nblk) {
      k_dir_count<false, false><<<(unsigned)nblk, 256, 0, st>>>(bits, d_meta, (int)nlev, d_first, dir,
                                                               blk, samp, nullptr, dl);
      count_launch();
    }
    k_dir_groups<<<nlev, 32, 0, st>>>(d_meta, d_first, blk, dir, zeros, dl);
    count_launch();
    if (nblk) {
      k_dir_finish<false><<<fgrid, 256, 0, st>>>(bits, d_meta, (int)nlev, d_first, nblk, blk, dir,
                                                 samp, dl);
      count_launch();
    }
  }
  CK(cudaGetLastError());
  return WT_OK;
}

// ---------------------------------------------------------------------------
// constant-time select directory (after Clark, Section 5.1 select)
// ---------------------------------------------------------------------------
constexpr uint64_t CK_HUGE_MIN = 1ull << 32;    // range length that keeps all positions
constexpr uint64_t CK_SPARSE_MIN = 1ull << 16;  // sub-range length that keeps all offsets

// occurrences of value b before superblock s of a level: bit values of a
// binary level (2048-bit superblocks), digit values of a digit level (1024)
template <bool DIG>
__device__ __forceinline__ uint64_t occ_before(const uint64_t* ldir, int b, uint64_t s) {
  if (DIG) return ldir[8 * s + b];
  const uint64_t z = ldir[2 * s];
  return b ? 2048 * s - z : z;
}

// position of occurrence q of value b, known to lie in superblocks [lo, hi]
// of the level (q >= occurrences before lo); nw as for load_block.  Each step
// reads seven evenly spaced records at once: between two samples of a dense
// level lie four or five superblocks, found in one round of loads where a
// binary search takes three dependent ones.
template <bool DIG>
__device__ uint64_t dir_select(const uint64_t* lbits, const uint64_t* ldir, int b, uint64_t q,
                               uint64_t lo, uint64_t hi, uint64_t nw) {
  while (lo < hi) {
    const uint64_t step = (hi - lo + 7) >> 3;
    uint64_t before[7];
#pragma unroll
    for (int i = 0; i < 7; i++) {
      const uint64_t s = lo + (uint64_t)(i + 1) * step;
      before[i] = s <= hi ? occ_before<DIG>(ldir, b, s) : ~0ull;
    }
    uint32_t c = 0;
#pragma unroll
    for (int i = 0; i < 7; i++) c += before[i] <= q ? 1u : 0u;
    lo += c * step;
    if (c < 7 && lo + step - 1 < hi) hi = lo + step - 1;
  }
  const uint32_t r = (uint32_t)(q - occ_before<DIG>(ldir, b, lo));
  if (DIG) return 1024 * lo + find_in_dsb(lbits, ldir, lo, (uint32_t)b, r);
  return 2048 * lo + find_in_sb(lbits, ldir[2 * lo + 1], lo, b, r, nw);
}

// one (level, bit or digit value) of the directory build
struct CkSeg {
  uint64_t g0;        // its first range in the global numbering
  uint64_t cnt;       // occurrences
  uint64_t bit_off, dir_off, samp_off, n, nsb;
  int b;
};

__device__ __forceinline__ uint32_t ck_seg_of(const CkSeg* segs, uint32_t nseg, uint64_t g) {
  uint32_t lo = 0, hi = nseg - 1;
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (segs[mid].g0 <= g) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// per range: kind, sub-sample offsets, mask of long sub-ranges
template <bool DIG>
__global__ void k_ck_ranges(const uint64_t* bits, const uint64_t* dir, const uint64_t* samp,
                            const CkSeg* segs, uint32_t nseg, uint64_t G, uint32_t* sub,
                            uint64_t* mask_or_huge, uint64_t* nh, uint64_t* ns) {
  const uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= G) return;
  const CkSeg sg = segs[ck_seg_of(segs, nseg, g)];
  const uint64_t k = g - sg.g0, R = (sg.cnt + 4095) / 4096;
  const uint64_t* lbits = bits + sg.bit_off;
  const uint64_t* ldir = dir + sg.dir_off;
  const uint64_t* ls = samp + sg.samp_off;
  const uint64_t S1 = ls[k];
  const uint64_t e = (k + 1 < R) ? ls[k + 1] : sg.n;
  const uint64_t M = (sg.cnt + 255) / 256;
  const bool huge = e - S1 >= CK_HUGE_MIN;
  uint32_t mask = 0;
  uint64_t prev = S1;  // start of sub-range i
  constexpr int SBSH = DIG ? 10 : 11;
  const uint64_t lo_sb = S1 >> SBSH, hi_sb = (e - 1) >> SBSH;
  const uint64_t nw = DIG ? PADDED : (sg.n + 63) / 64;
  for (int i = 0; i < 16; i++) {
    const uint64_t m = 16 * k + i;
    uint64_t start = 0;
    if (!huge && m < M) start = i == 0 ? S1 : dir_select<DIG>(lbits, ldir, sg.b, 256 * m, lo_sb, hi_sb, nw);
    sub[16 * g + i] = huge ? 0u : (m < M ? (uint32_t)(start - S1) : 0xffffffffu);
    if (!huge && i > 0 && m - 1 < M && m < M && start - prev >= CK_SPARSE_MIN) mask |= 1u << (i - 1);
    if (!huge && m < M) prev = start;
    if (!huge && m < M && (i == 15 || m + 1 >= M) && e - start >= CK_SPARSE_MIN) mask |= 1u << i;
  }
  mask_or_huge[g] = huge ? (1ull << 63) : (uint64_t)mask;
  nh[g] = huge ? 1 : 0;
  ns[g] = huge ? 0 : (uint64_t)__popc(mask);
}

// descriptors, numbered inside their (level, bit value)
__global__ void k_ck_desc(const CkSeg* segs, uint32_t nseg, uint64_t G, const uint64_t* kind,
                          const uint64_t* gh, const uint64_t* gs, uint64_t* desc) {
  const uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= G) return;
  const CkSeg sg = segs[ck_seg_of(segs, nseg, g)];
  const uint64_t kd = kind[g];
  if (kd >> 63) desc[g] = (1ull << 63) | (4096 * (gh[g] - gh[sg.g0]));
  else desc[g] = (gs[g] - gs[sg.g0]) | (kd << 40);
}

// explicit answers: one block per range that keeps any
template <bool DIG>
__global__ void k_ck_fill(const uint64_t* bits, const uint64_t* dir, const uint64_t* samp,
                          const CkSeg* segs, uint32_t nseg, uint64_t G, const uint64_t* kind,
                          const uint64_t* gh, const uint64_t* gs, const uint32_t* sub,
                          uint64_t* huge_all, uint32_t* sparse_all) {
  for (uint64_t g = blockIdx.x; g < G; g += gridDim.x) {
    const uint64_t kd = kind[g];
    if (kd == 0) continue;
    const CkSeg sg = segs[ck_seg_of(segs, nseg, g)];
    const uint64_t k = g - sg.g0, R = (sg.cnt + 4095) / 4096;
    const uint64_t* lbits = bits + sg.bit_off;
    const uint64_t* ldir = dir + sg.dir_off;
    const uint64_t S1 = samp[sg.samp_off + k];
    const uint64_t e = (k + 1 < R) ? samp[sg.samp_off + k + 1] : sg.n;
    constexpr int SBSH = DIG ? 10 : 11;
    const uint64_t lo_sb = S1 >> SBSH, hi_sb = (e - 1) >> SBSH;
    const uint64_t nw = DIG ? PADDED : (sg.n + 63) / 64;
    if (kd >> 63) {
      for (uint32_t j = threadIdx.x; j < 4096; j += blockDim.x) {
        const uint64_t q = 4096 * k + j;
        huge_all[4096 * gh[g] + j] =
            q < sg.cnt ? dir_select<DIG>(lbits, ldir, sg.b, q, lo_sb, hi_sb, nw) : ~0ull;
      }
    } else {
      uint32_t mask = (uint32_t)kd;
      uint64_t s = gs[g];
      while (mask) {
        const int i = __ffs(mask) - 1;
        mask &= mask - 1;
        for (uint32_t j = threadIdx.x; j < 256; j += blockDim.x) {
          const uint64_t q = 4096 * k + 256 * i + j;
          sparse_all[256 * s + j] =
              q < sg.cnt ? (uint32_t)(dir_select<DIG>(lbits, ldir, sg.b, q, lo_sb, hi_sb, nw) - S1)
                         : 0xffffffffu;
        }
        s++;
      }
    }
  }
}

__global__ void k_gather_u64(const uint64_t* src, const uint64_t* idx, uint64_t n, uint64_t* out) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = src[idx[i]];
}

// dig: digit levels (4 values; occurrence counts from the directory's
// trailing records), else binary levels (2 values; counts from the zeros)
static wt_status build_clark(wt_struct* h) {
  cudaStream_t st = h->stream;
  const uint32_t nlev = h->levels;
  const bool dig = h->bpe == 2;
  const int NV = dig ? 4 : 2;
  // occurrence counts of every value on every level, on the host
  std::vector<uint64_t> occ((size_t)NV * nlev, 0);
  if (nlev) {
    if (dig) {
      std::vector<uint64_t> idx(occ.size());
      for (uint32_t l = 0; l < nlev; l++)
        for (int d = 0; d < 4; d++) idx[4 * l + d] = h->meta[l].dir_off + 8 * h->meta[l].nsb + d;
      Work wk0{st};
      uint64_t *d_idx, *d_got;
      TRY(wk0.get(&d_idx, idx.size()));
      TRY(wk0.get(&d_got, idx.size()));
      TRY(upload(d_idx, idx.data(), idx.size() * 8, st));
      k_gather_u64<<<(unsigned)((idx.size() + 255) / 256), 256, 0, st>>>(h->d_dir, d_idx,
                                                                         idx.size(), d_got);
      count_launch();
      CK(cudaMemcpyAsync(occ.data(), d_got, occ.size() * 8, cudaMemcpyDeviceToHost, st));
      CK(cudaStreamSynchronize(st));
    } else {
      std::vector<uint64_t> zeros(nlev, 0);
      CK(cudaMemcpyAsync(zeros.data(), h->d_zeros, nlev * 8, cudaMemcpyDeviceToHost, st));
      CK(cudaStreamSynchronize(st));
      for (uint32_t l = 0; l < nlev; l++) {
        occ[2 * l] = zeros[l];
        occ[2 * l + 1] = h->meta[l].n - zeros[l];
      }
    }
  }
  std::vector<CkSeg> segs;
  h->cmeta.assign(nlev, ClarkMeta{});
  uint64_t G = 0;
  for (uint32_t l = 0; l < nlev; l++) {
    const LevelMeta& m = h->meta[l];
    for (int b = 0; b < NV; b++) {
      CkSeg sg;
      sg.g0 = G;
      sg.cnt = occ[(size_t)NV * l + b];
      sg.bit_off = m.bit_off;
      sg.dir_off = m.dir_off;
      sg.samp_off = dig ? m.s0_off + (uint64_t)b * (m.n / 4096 + 1) : (b ? m.s1_off : m.s0_off);
      sg.n = m.n;
      sg.nsb = m.nsb;
      sg.b = b;
      const uint64_t R = (sg.cnt + 4095) / 4096;
      h->cmeta[l].nr[b] = R;
      h->cmeta[l].desc[b] = G;
      h->cmeta[l].sub[b] = 16 * G;
      if (R) segs.push_back(sg);
      G += R;
    }
  }
  const uint32_t nseg = (uint32_t)segs.size();
  Work wk{st};
  uint64_t *d_kind, *d_nh, *d_ns, *d_gh, *d_gs, *scr;
  CkSeg* d_segs;
  uint32_t* d_sub;
  TRY(wk.get(&d_sub, std::max<uint64_t>(16 * G, 1)));
  TRY(wk.get(&d_kind, std::max<uint64_t>(G, 1)));
  TRY(wk.get(&d_nh, std::max<uint64_t>(G, 1)));
  TRY(wk.get(&d_ns, std::max<uint64_t>(G, 1)));
  TRY(wk.get(&d_gh, G + 1));
  TRY(wk.get(&d_gs, G + 1));
  TRY(wk.get(&scr, scan_scratch_pub(G)));
  TRY(wk.get(&d_segs, std::max<uint32_t>(nseg, 1)));
  if (nseg) TRY(upload(d_segs, segs.data(), nseg * sizeof(CkSeg), st));
  const unsigned gg = (unsigned)((G + 255) / 256);
  if (G) {
    if (dig)
      k_ck_ranges<true><<<gg, 256, 0, st>>>(h->d_bits_ro, h->d_dir, h->d_samp, d_segs, nseg, G,
                                            d_sub, d_kind, d_nh, d_ns);
    else
      k_ck_ranges<false><<<gg, 256, 0, st>>>(h->d_bits_ro, h->d_dir, h->d_samp, d_segs, nseg, G,
                                             d_sub, d_kind, d_nh, d_ns);
    count_launch();
  }
  wt_status s = scan_excl_u64_pub(d_nh, d_gh, G, scr, st);
  if (s == WT_OK) s = scan_excl_u64_pub(d_ns, d_gs, G, scr, st);
  uint64_t tot[2] = {0, 0};
  if (s == WT_OK) {
    CK(cudaMemcpyAsync(&tot[0], d_gh + G, 8, cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(&tot[1], d_gs + G, 8, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
  }
  const uint64_t H = tot[0], S = tot[1];
  if (s == WT_OK) {
    CK(dmalloc((void**)&h->d_ck64, std::max<uint64_t>(G + 4096 * H, 1) * 8, st));
    CK(dmalloc((void**)&h->d_ck32, std::max<uint64_t>(16 * G + 256 * S, 1) * 4, st));
    if (G) {
      CK(cudaMemcpyAsync(h->d_ck32, d_sub, 16 * G * 4, cudaMemcpyDeviceToDevice, st));
      k_ck_desc<<<gg, 256, 0, st>>>(d_segs, nseg, G, d_kind, d_gh, d_gs, h->d_ck64);
      count_launch();
      const unsigned fg = (unsigned)std::min<uint64_t>(G, (uint64_t)num_sms() * 16);
      if (dig)
        k_ck_fill<true><<<fg, 256, 0, st>>>(h->d_bits_ro, h->d_dir, h->d_samp, d_segs, nseg, G,
                                            d_kind, d_gh, d_gs, d_sub, h->d_ck64 + G,
                                            h->d_ck32 + 16 * G);
      else
        k_ck_fill<false><<<fg, 256, 0, st>>>(h->d_bits_ro, h->d_dir, h->d_samp, d_segs, nseg, G,
                                             d_kind, d_gh, d_gs, d_sub, h->d_ck64 + G,
                                             h->d_ck32 + 16 * G);
      count_launch();
    }
    // per (level, value): the scans at its first and one-past-last range
    const size_t nv = (size_t)NV * nlev;
    std::vector<uint64_t> idx(2 * nv, 0);
    for (uint32_t l = 0; l < nlev; l++)
      for (int b = 0; b < NV; b++) {
        idx[2 * (NV * l + b)] = h->cmeta[l].desc[b];
        idx[2 * (NV * l + b) + 1] = h->cmeta[l].desc[b] + h->cmeta[l].nr[b];
      }
    std::vector<uint64_t> both(2 * idx.size(), 0);
    if (nlev) {
      uint64_t *d_idx, *d_got;
      TRY(wk.get(&d_idx, idx.size()));
      TRY(wk.get(&d_got, both.size()));
      TRY(upload(d_idx, idx.data(), idx.size() * 8, st));
      k_gather_u64<<<(unsigned)((idx.size() + 255) / 256), 256, 0, st>>>(d_gh, d_idx, idx.size(), d_got);
      count_launch();
      k_gather_u64<<<(unsigned)((idx.size() + 255) / 256), 256, 0, st>>>(d_gs, d_idx, idx.size(),
                                                                         d_got + idx.size());
      count_launch();
      CK(cudaMemcpyAsync(both.data(), d_got, both.size() * 8, cudaMemcpyDeviceToHost, st));
      CK(cudaStreamSynchronize(st));
    }
    for (uint32_t l = 0; l < nlev; l++)
      for (int b = 0; b < NV; b++) {
        const size_t i = 2 * ((size_t)NV * l + b);
        ClarkMeta& cm = h->cmeta[l];
        cm.nh[b] = both[i + 1] - both[i];
        cm.ns[b] = both[idx.size() + i + 1] - both[idx.size() + i];
        cm.huge[b] = G + 4096 * both[i];
        cm.sparse[b] = 16 * G + 256 * both[idx.size() + i];
      }
    CK(dmalloc((void**)&h->d_cmeta, std::max<uint32_t>(nlev, 1) * sizeof(ClarkMeta), st));
    if (nlev)
      CK(cudaMemcpyAsync(h->d_cmeta, h->cmeta.data(), nlev * sizeof(ClarkMeta),
                         cudaMemcpyHostToDevice, st));
    CK(cudaStreamSynchronize(st));  // host vectors above are pageable and local
  }
  cudaError_t e = cudaGetLastError();
  if (s != WT_OK) return s;
  return e == cudaSuccess ? WT_OK : WT_ERR_CUDA;
}

// A wavelet matrix keeps its symbols' starts (k_wm_starts) where the sequence
// has at least START_MIN elements per entry, so that their walks (20 us for
// 2^16 symbols) are a small part of a build.
constexpr uint64_t START_MIN = 256;
static wt_status build_starts(wt_struct* h);

wt_status build_directories(wt_struct* h) {
  cudaStream_t st = h->stream;
  const uint32_t nlev = h->levels;
  const bool dig = h->bpe == 2;
  const uint64_t sbsz = dig ? 1024 : 2048;
  const uint64_t rec = dig ? 8 : 2;
  // select samples: per level one region of n/4096 + 1 per value (2 bit
  // values, or 4 digit values)
  const uint32_t NV = dig ? 4 : 2;
  h->meta.assign(nlev, LevelMeta{});
  h->dir_off.assign(nlev + 1, 0);
  h->samp_off.assign(NV * nlev + 1, 0);
  std::vector<uint64_t> sb_first(nlev + 1, 0);
  for (uint32_t l = 0; l < nlev; l++) {
    LevelMeta& m = h->meta[l];
    m.bit_off = h->level_off[l];
    m.n = h->level_len[l];
    m.nsb = (m.n + sbsz - 1) / sbsz;
    m.dir_off = h->dir_off[l];
    h->dir_off[l + 1] = h->dir_off[l] + rec * (m.nsb + 1);
    sb_first[l + 1] = sb_first[l] + m.nsb;
    const uint64_t cap = m.n / 4096 + 1;
    for (uint32_t v = 0; v < NV; v++) h->samp_off[NV * l + v + 1] = h->samp_off[NV * l + v] + cap;
    m.s0_off = h->samp_off[NV * l];
    m.s1_off = h->samp_off[NV * l + 1];
  }
  {
    const uint64_t dir = (h->dir_off[nlev] + 31) / 32 * 32, samp = (h->samp_off[NV * nlev] + 31) / 32 * 32;
    const bool starts = h->kind == WT_KIND_WM && h->L <= 24 && h->n >> h->L >= START_MIN;
    const uint64_t ns = starts ? ((uint64_t)1 << h->L) + 1 : 0;
    CK(dmalloc((void**)&h->d_dir, std::max<uint64_t>(dir + samp + ns, 1) * 8, st));
    h->d_samp = h->d_dir + dir;
    if (starts) h->d_start = h->d_samp + samp;
  }
  // (queries compute the offsets of levels of equal length)
  wt_status s = h->kind == WT_KIND_HUFF ? upload_meta(h) : WT_OK;
  if (s != WT_OK) return s;
  if (nlev == 0) return WT_OK;
  if (!dig) {
    s = dir_build_levels(h->d_bits_ro, h->d_meta, nlev, sb_first, h->d_dir, h->d_samp,
                         h->kind == WT_KIND_RS ? h->d_zeros : nullptr, st, h->meta.data());
    if (s == WT_OK && h->d_start) s = build_starts(h);
    if (s == WT_OK && (h->flags & WT_FLAG_SELECT_O1)) s = build_clark(h);
    return s;
  }
  DirLevels dl;
  memset(&dl, 0, sizeof(dl));
  dl.nlev = (int)nlev;
  for (uint32_t l = 0; l < nlev; l++) {
    dl.blk_first[l + 1] = dl.blk_first[l] + (h->meta[l].nsb + DIR_GROUP - 1) / DIR_GROUP;
    dl.meta[l] = h->meta[l];
  }
  const uint64_t ng = dl.blk_first[nlev];
  Work wk{st};
  uint64_t* blk;
  TRY(wk.get(&blk, 4 * ng + 1));
  if (ng) {
    k_mdir_count<<<(unsigned)ng, 256, 0, st>>>(h->d_bits_ro, ng, h->d_dir, blk, dl);
    count_launch();
  }
  k_mdir_groups<<<nlev * 4 * DIR_CLUSTER, 512, 0, st>>>(ng, blk, h->d_dir, dl);
  count_launch();
  if (ng) {
    constexpr int per = 256 / DIR_GROUP;
    k_mdir_finish<<<(unsigned)((ng + per - 1) / per), 256, 0, st>>>(h->d_bits_ro, ng, blk, h->d_dir,
                                                                    h->d_samp, dl);
    count_launch();
  }
  CK(cudaGetLastError());
  if (h->flags & WT_FLAG_SELECT_O1) return build_clark(h);
  return WT_OK;
}

// ---------------------------------------------------------------------------
// queries
// ---------------------------------------------------------------------------
struct QStruct {
  int kind;
  uint64_t n;
  uint32_t sigma;
  int L;        // binary levels (HUFF: max code length)
  int levels;   // output levels
  const uint64_t* bits;
  const uint64_t* dir;
  const uint64_t* samp;
  const LevelMeta* meta;
  const uint64_t* zeros;
  const uint64_t* start;  // wavelet matrix: see k_wm_starts, or null
  HuffQuery hq;
  const ClarkMeta* cmeta;  // constant-time select directory, or null
  const uint64_t* ck64;
  const uint32_t* ck32;
};

struct BinLevel {
  const uint64_t* bits;
  const uint64_t* dir;
  const uint64_t* s0;
  const uint64_t* s1;
  uint64_t n, nsb, zeros;
  uint64_t nw;  // as for load_block
  const ClarkMeta* cm;
  const uint64_t* ck64;
  const uint32_t* ck32;
};

__device__ __forceinline__ BinLevel bin_level(const QStruct& S, int l) {
  const LevelMeta m = S.meta[l];
  BinLevel v;
  v.bits = S.bits + m.bit_off;
  v.dir = S.dir + m.dir_off;
  v.s0 = S.samp + m.s0_off;
  v.s1 = S.samp + m.s1_off;
  v.n = m.n;
  v.nsb = m.nsb;
  v.zeros = S.zeros[l];
  v.nw = PADDED;
  v.cm = S.cmeta ? S.cmeta + l : nullptr;
  v.ck64 = S.ck64;
  v.ck32 = S.ck32;
  return v;
}

// The same for a wavelet matrix, a balanced tree or a bitvector, whose levels
// all have n bits: the offsets follow from n and l, so that no table read stands before
// a level's first access.
__device__ __forceinline__ BinLevel uniform_level(const QStruct& S, int l) {
  const uint64_t nsb = (S.n + 2047) >> 11, cap = (S.n >> 12) + 1;
  BinLevel v;
  v.bits = S.bits + (uint64_t)l * 32 * nsb;
  v.dir = S.dir + (uint64_t)l * 2 * (nsb + 1);
  v.s0 = S.samp + (uint64_t)(2 * l) * cap;
  v.s1 = v.s0 + cap;
  v.n = S.n;
  v.nsb = nsb;
  v.zeros = S.zeros[l];
  v.nw = PADDED;
  v.cm = S.cmeta ? S.cmeta + l : nullptr;
  v.ck64 = S.ck64;
  v.ck32 = S.ck32;
  return v;
}

__device__ __forceinline__ int get_bit(const BinLevel& v, uint64_t i) {
  return (int)((v.bits[i >> 6] >> (i & 63)) & 1ull);
}

// A level at one position x: its directory record and the words of x's
// 512-bit block that hold bits before x.  All of it is requested at once, and
// the lines of several positions before any of them is used: a query is
// bound by the latency of its chain of levels (and by L2 and DRAM sectors
// when many run), so a level costs one round of loads, where words read one
// after another up to the position cost a round each.  With the searches of
// dir_select and the joint walks below: 2^22 ranks on 2^30 symbols of 16
// levels 2.85 -> 1.79 ms;
// 2^16 mixed queries over 64 matrices of up to 2^22 symbols 270 -> 82 us.
struct Line {
  ulonglong2 rec;
  uint64_t w[8];
};

__device__ __forceinline__ Line load_line(const BinLevel& v, uint64_t x) {
  Line ln;
  const uint32_t in = (uint32_t)(x & 511);
  const uint64_t* p = v.bits + 8 * (x >> 9);
  ln.rec = *(const ulonglong2*)(v.dir + 2 * (x >> 11));
  if (v.nw == PADDED) {
#pragma unroll
    for (int i = 0; i < 4; i++) {
      ulonglong2 q = make_ulonglong2(0, 0);
      if ((uint32_t)(128 * i) < in) q = ((const ulonglong2*)p)[i];
      ln.w[2 * i] = q.x;
      ln.w[2 * i + 1] = q.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; i++) ln.w[i] = (uint32_t)(64 * i) < in ? p[i] : 0ull;
  }
  return ln;
}

// zeros in [0, x), x <= n
__device__ __forceinline__ uint64_t zeros_before(const Line& ln, uint64_t x) {
  const uint32_t b = (uint32_t)((x >> 9) & 3), in = (uint32_t)(x & 511), k = in >> 6;
  const uint64_t part = (1ull << (in & 63)) - 1ull;
  uint32_t ones = 0;
#pragma unroll
  for (uint32_t i = 0; i < 8; i++) {
    const uint64_t m = i < k ? ~0ull : (i == k ? part : 0ull);
    ones += (uint32_t)__popcll(ln.w[i] & m);
  }
  return ln.rec.x + ((ln.rec.y >> (16 * b)) & 0xffffull) + (in - ones);
}

__device__ __forceinline__ uint64_t rank0(const BinLevel& v, uint64_t x) {
  return zeros_before(load_line(v, x), x);
}
__device__ __forceinline__ uint64_t rank1(const BinLevel& v, uint64_t x) { return x - rank0(v, x); }

// position of the k-th (0-based) bit equal to bv; k < count
__device__ uint64_t select_b(const BinLevel& v, int bv, uint64_t k) {
  const uint64_t* samp = bv ? v.s1 : v.s0;
  if (v.cm) {
    // constant-time directory: the range's descriptor gives the stored
    // answer, or a sub-range shorter than 2^16 bits to search
    const uint64_t kk = k >> 12;
    const uint64_t d = v.ck64[v.cm->desc[bv] + kk];
    if (d >> 63) return v.ck64[v.cm->huge[bv] + (d & ((1ull << 63) - 1)) + (k & 4095)];
    const uint32_t mask = (uint32_t)((d >> 40) & 0xffffu);
    const int i = (int)((k >> 8) & 15);
    const uint64_t S1 = samp[kk];
    if ((mask >> i) & 1u) {
      const uint64_t sidx = (d & ((1ull << 40) - 1)) + (uint64_t)__popc(mask & ((1u << i) - 1u));
      return S1 + v.ck32[v.cm->sparse[bv] + 256 * sidx + (k & 255)];
    }
    const uint32_t* sb = v.ck32 + v.cm->sub[bv] + 16 * kk;
    const uint64_t p0 = S1 + sb[i];
    if ((k & 255) == 0) return p0;
    // the sub-range ends at the next sub-sample, or at the range's end
    uint64_t p1 = (i + 1 < 16 && sb[i + 1] != 0xffffffffu) ? S1 + sb[i + 1] : 0;
    if (!p1) {
      const uint64_t ns = ((bv ? v.n - v.zeros : v.zeros) + 4095) / 4096;
      p1 = kk + 1 < ns ? samp[kk + 1] : v.n;
    }
    return dir_select<false>(v.bits, v.dir, bv, k, p0 >> 11, (p1 - 1) >> 11, v.nw);
  }
  const uint64_t cnt = bv ? v.n - v.zeros : v.zeros;
  const uint64_t ns = (cnt + 4095) / 4096;
  const uint64_t idx = k >> 12;
  const uint64_t lo = samp[idx] >> 11;
  const uint64_t hi = (idx + 1 < ns) ? (samp[idx + 1] >> 11) : v.nsb - 1;
  return dir_select<false>(v.bits, v.dir, bv, k, lo, hi, v.nw);
}

// Wavelet matrix.  The three operations walk down together, so that a warp
// with a mixture of them walks once: rank and select carry the start s and
// the end p of the symbol's class, access the position p alone.  Select then
// walks up.  Where the structure keeps the symbols' starts (k_wm_starts),
// rank carries its position alone and select does not walk down: half of the
// lines of a rank (2^22 of them on n = 2^30: 1.79 -> 1.50 ms), and of the
// latency of a select.
__device__ uint64_t q_wm(const QStruct& S, int op, uint32_t c, uint64_t x) {
  const int L = S.L;
  if (op == 2 ? x == 0 : x >= S.n) return NONE;
  if (op != 0 && c >= S.sigma) return NONE;
  uint64_t s = 0, p = op == 0 ? x : (op == 1 ? x + 1 : S.n);
  const bool starts = S.start != nullptr, both = op != 0 && !starts;
  uint32_t sym = 0;
  if (starts && op != 0) {
    const uint32_t r = rev_bits(c, L);
    s = S.start[r];
    if (op == 2) p = S.start[r + 1];
  }
  if (!(starts && op == 2)) {
    for (int l = 0; l < L; l++) {
      const BinLevel v = uniform_level(S, l);
      const Line lp = load_line(v, p);
      Line ls;
      int b = (int)((c >> (L - 1 - l)) & 1u);
      if (op == 0) b = get_bit(v, p);
      if (both) ls = load_line(v, s);
      const uint64_t zp = zeros_before(lp, p);
      p = b ? v.zeros + (p - zp) : zp;
      if (op == 0) sym = (sym << 1) | (uint32_t)b;
      if (both) {
        const uint64_t zs = zeros_before(ls, s);
        s = b ? v.zeros + (s - zs) : zs;
      }
    }
  }
  if (op == 0) return sym;
  if (op == 1) return p - s;
  if (x > p - s) return NONE;
  uint64_t pos = s + x - 1;
  for (int l = L - 1; l >= 0; l--) {
    const BinLevel v = uniform_level(S, l);
    const int b = (int)((c >> (L - 1 - l)) & 1u);
    pos = select_b(v, b, b ? pos - v.zeros : pos);
  }
  return pos;
}

// Wavelet matrix: the start of every symbol's class in the order after the
// last level (ascending in the symbol's L bits reversed), entry r for the
// symbol rev(r), and n at the end: one walk down per symbol.
__global__ void __launch_bounds__(64) k_wm_starts(const QStruct S, uint64_t* start) {
  const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x, nr = 1u << S.L;
  if (r == 0) start[nr] = S.n;
  if (r >= nr) return;
  uint64_t s = 0;
  for (int l = 0; l < S.L; l++) {
    const BinLevel v = uniform_level(S, l);
    const uint64_t z = rank0(v, s);
    s = (r >> l) & 1u ? v.zeros + (s - z) : z;
  }
  start[r] = s;
}

// Balanced tree: the node's start s and end e, and the position p in it
// (access, rank), walked down together; select keeps every level's start and
// the zeros before it for its way up.
__device__ uint64_t q_wt(const QStruct& S, int op, uint32_t c, uint64_t x) {
  const int L = S.L;
  if (op == 2 ? x == 0 : x >= S.n) return NONE;
  if (op != 0 && c >= S.sigma) return NONE;
  uint64_t S0[33], Z0[33];
  uint64_t s = 0, e = S.n, p = op == 1 ? x + 1 : x;
  uint32_t sym = 0;
  for (int l = 0; l < L; l++) {
    const BinLevel v = uniform_level(S, l);
    const Line le = load_line(v, e), ls = load_line(v, s);
    Line lp;
    int b = (int)((c >> (L - 1 - l)) & 1u);
    if (op != 2) lp = load_line(v, p);
    if (op == 0) b = get_bit(v, p);
    const uint64_t zs = zeros_before(ls, s), ze = zeros_before(le, e);
    const uint64_t m = s + (ze - zs);  // end of the zeros' child
    if (op == 2) {
      S0[l] = s;
      Z0[l] = zs;
    } else {
      const uint64_t zp = zeros_before(lp, p);
      p = b ? m + (p - s) - (zp - zs) : s + (zp - zs);
      sym = (sym << 1) | (uint32_t)b;
    }
    if (b) s = m;
    else e = m;
  }
  if (op == 0) return sym;
  if (op == 1) return p - s;
  if (x > e - s) return NONE;
  uint64_t off = x - 1;
  for (int l = L - 1; l >= 0; l--) {
    const BinLevel v = uniform_level(S, l);
    const int b = (int)((c >> (L - 1 - l)) & 1u);
    off = select_b(v, b, (b ? S0[l] - Z0[l] : Z0[l]) + off) - S0[l];
  }
  return off;  // the root starts at 0
}

// Huffman-shaped tree: node (level l, prefix q) -> [start, end) on level l
__device__ __forceinline__ bool huff_node(const QStruct& S, int l, uint64_t q, uint64_t& st,
                                          uint64_t& en) {
  if (l >= S.L) return false;
  const uint64_t off = S.hq.node_lvl[3 * l], first = S.hq.node_lvl[3 * l + 1],
                 num = S.hq.node_lvl[3 * l + 2];
  if (q < first || q >= first + num) return false;
  st = S.hq.node[off + q - first];
  en = S.hq.node[off + q - first + 1];
  return true;
}

__device__ uint64_t q_huff(const QStruct& S, int op, uint32_t c, uint64_t x) {
  if (op == 0) {
    if (x >= S.n) return NONE;
    uint64_t q = 0, s = 0, pos = x;
    for (int l = 0; l < S.L; l++) {
      const BinLevel v = bin_level(S, l);
      const Line lp = load_line(v, pos), ls = load_line(v, s);
      const int b = get_bit(v, pos);
      const uint64_t child = (q << 1) | (uint64_t)b;
      uint64_t cs, ce;
      const bool inner = huff_node(S, l + 1, child, cs, ce);
      if (!inner) {
        // a leaf at depth l+1: canonical code -> symbol
        const int ln = l + 1;
        const uint64_t first = S.hq.len_first[ln], base = S.hq.len_base[ln];
        return S.hq.sym_by_rank[base + (child - first)];
      }
      const uint64_t z = zeros_before(lp, pos) - zeros_before(ls, s);
      q = child;
      pos = cs + (b ? (pos - s) - z : z);
      s = cs;
    }
    return NONE;
  }
  if (c >= S.sigma) return NONE;
  const int ln = S.hq.len[c];
  const uint64_t code = S.hq.code[c];
  if (op == 1) {
    if (x >= S.n) return NONE;
    if (ln == 0) return 0;
    uint64_t q = 0, s = 0, j = x + 1;
    for (int l = 0; l < ln; l++) {
      const BinLevel v = bin_level(S, l);
      const int b = (int)((code >> (ln - 1 - l)) & 1u);
      const Line lj = load_line(v, j), ls = load_line(v, s);
      q = (q << 1) | (uint64_t)b;
      uint64_t cs = 0, ce;
      if (l + 1 < ln) huff_node(S, l + 1, q, cs, ce);
      const uint64_t z = zeros_before(lj, j) - zeros_before(ls, s);
      const uint64_t cb = b ? (j - s) - z : z;
      if (l == ln - 1) return cb;
      s = cs;
      j = cs + cb;
    }
    return NONE;
  }
  if (x == 0 || ln == 0) return NONE;
  // the code's nodes and the zeros before each on the way down; only the
  // last level's count of the code's bit decides whether there are x
  uint64_t S0[33], Z0[33];
  uint64_t q = 0, s = 0, e = S.n;
  for (int l = 0; l < ln; l++) {
    const BinLevel v = bin_level(S, l);
    const int b = (int)((code >> (ln - 1 - l)) & 1u);
    const uint64_t zs = rank0(v, s);
    S0[l] = s;
    Z0[l] = zs;
    if (l == ln - 1) {
      const uint64_t z = rank0(v, e) - zs;
      if (x > (b ? (e - s) - z : z)) return NONE;
      break;
    }
    q = (q << 1) | (uint64_t)b;
    // the child [s, e) of the code's bit, from the node table
    huff_node(S, l + 1, q, s, e);
  }
  // bottom-up: at level l the target is the off-th b-bit of node [S0[l], .)
  uint64_t off = x - 1, pos = 0;
  for (int l = ln - 1; l >= 0; l--) {
    const BinLevel v = bin_level(S, l);
    const int b = (int)((code >> (ln - 1 - l)) & 1u);
    pos = select_b(v, b, (b ? S0[l] - Z0[l] : Z0[l]) + off);
    off = pos - S0[l];
  }
  return pos;
}

// 4-ary tree: digit levels, per-value counts
struct DigLevel {
  const uint64_t* bits;
  const uint64_t* dir;
  const uint64_t* samp;  // 4 regions of n/4096 + 1: samples of values 0..3
  uint64_t n, nsb;
  const ClarkMeta* cm;
  const uint64_t* ck64;
  const uint32_t* ck32;
};

__device__ __forceinline__ DigLevel dig_level(const QStruct& S, int l) {
  const uint64_t nsb = (S.n + 1023) >> 10;  // digit levels all have n digits
  DigLevel v;
  v.bits = S.bits + (uint64_t)l * 32 * nsb;
  v.dir = S.dir + (uint64_t)l * 8 * (nsb + 1);
  v.samp = S.samp + (uint64_t)l * 4 * ((S.n >> 12) + 1);
  v.n = S.n;
  v.nsb = nsb;
  v.cm = S.cmeta ? S.cmeta + l : nullptr;
  v.ck64 = S.ck64;
  v.ck32 = S.ck32;
  return v;
}

// A digit level at one position: the counts before its superblock and its
// 256-digit block, and the block's words with digits before it, all
// requested at once (see Line).
struct DigLine {
  ulonglong2 c01, c23;
  uint64_t rel;
  uint64_t w[8];
};

__device__ __forceinline__ DigLine load_dig(const DigLevel& v, uint64_t x) {
  DigLine ln;
  const uint32_t in = (uint32_t)(x & 255);
  const uint64_t* r = v.dir + 8 * (x >> 10);
  ln.c01 = *(const ulonglong2*)r;
  ln.c23 = *(const ulonglong2*)(r + 2);
  ln.rel = r[4 + ((x >> 8) & 3)];
  const ulonglong2* p = (const ulonglong2*)(v.bits + 8 * (x >> 8));
#pragma unroll
  for (int i = 0; i < 4; i++) {
    ulonglong2 q = make_ulonglong2(0, 0);
    if ((uint32_t)(64 * i) < in) q = p[i];
    ln.w[2 * i] = q.x;
    ln.w[2 * i + 1] = q.y;
  }
  return ln;
}

// digits equal to d (eq) and smaller than d (lt) in [0, x)
__device__ __forceinline__ void dig_counts(const DigLine& ln, uint64_t x, uint32_t d, uint64_t& eq,
                                           uint64_t& lt) {
  const uint32_t in = (uint32_t)(x & 255), k = in >> 5;
  const uint64_t part = (1ull << (2 * (in & 31))) - 1ull;
  auto rel = [&](int v) -> uint64_t { return (ln.rel >> (16 * v)) & 0xffffull; };
  const uint64_t c0 = ln.c01.x + rel(0), c1 = ln.c01.y + rel(1), c2 = ln.c23.x + rel(2),
                 c3 = ln.c23.y + rel(3);
  uint32_t e = 0, s = 0;
#pragma unroll
  for (uint32_t i = 0; i < 8; i++) {
    const uint64_t m = (i < k ? ~0ull : (i == k ? part : 0ull)) & 0x5555555555555555ull;
    const uint64_t lo = ln.w[i], hi = lo >> 1;
    e += (uint32_t)__popcll(digit_match(lo, d) & m);
    const uint64_t less = d == 0 ? 0ull : (d == 1 ? ~(hi | lo) : (d == 2 ? ~hi : ~(hi & lo)));
    s += (uint32_t)__popcll(less & m);
  }
  eq = e + (d == 0 ? c0 : (d == 1 ? c1 : (d == 2 ? c2 : c3)));
  lt = s + (d > 0 ? c0 : 0ull) + (d > 1 ? c1 : 0ull) + (d > 2 ? c2 : 0ull);
}

__device__ __forceinline__ uint32_t get_digit(const DigLevel& v, uint64_t i) {
  return (uint32_t)((v.bits[i >> 5] >> (2 * (i & 31))) & 3ull);
}

// position of the k-th (0-based) occurrence of digit d; k < its count
// (Section 5.2 generalized select: the structures of the binary case per
// digit value)
__device__ uint64_t select_d(const DigLevel& v, uint32_t d, uint64_t k) {
  const uint64_t* samp = v.samp + d * (v.n / 4096 + 1);
  const uint64_t kk = k >> 12;
  if (v.cm) {
    // constant-time directory: stored answer, or a sub-range shorter than
    // 2^16 digits to search
    const uint64_t dsc = v.ck64[v.cm->desc[d] + kk];
    if (dsc >> 63) return v.ck64[v.cm->huge[d] + (dsc & ((1ull << 63) - 1)) + (k & 4095)];
    const uint32_t mask = (uint32_t)((dsc >> 40) & 0xffffu);
    const int i = (int)((k >> 8) & 15);
    const uint64_t S1 = samp[kk];
    if ((mask >> i) & 1u) {
      const uint64_t sidx = (dsc & ((1ull << 40) - 1)) + (uint64_t)__popc(mask & ((1u << i) - 1u));
      return S1 + v.ck32[v.cm->sparse[d] + 256 * sidx + (k & 255)];
    }
    const uint32_t* sb = v.ck32 + v.cm->sub[d] + 16 * kk;
    const uint64_t p0 = S1 + sb[i];
    if ((k & 255) == 0) return p0;
    // the sub-range ends at the next sub-sample, or at the range's end
    uint64_t p1 = (i + 1 < 16 && sb[i + 1] != 0xffffffffu) ? S1 + sb[i + 1] : 0;
    if (!p1) {
      const uint64_t ns = (v.dir[8 * v.nsb + d] + 4095) / 4096;
      p1 = kk + 1 < ns ? samp[kk + 1] : v.n;
    }
    return dir_select<true>(v.bits, v.dir, (int)d, k, p0 >> 10, (p1 - 1) >> 10, PADDED);
  }
  // sampled: the search starts between two samples
  const uint64_t ns = (v.dir[8 * v.nsb + d] + 4095) / 4096;
  const uint64_t lo = samp[kk] >> 10;
  const uint64_t hi = kk + 1 < ns ? samp[kk + 1] >> 10 : v.nsb - 1;
  return dir_select<true>(v.bits, v.dir, (int)d, k, lo, hi, PADDED);
}

// The node's start s and end e, and the position p in it (access, rank),
// walked down together; select keeps for its way up every level's start and
// the occurrences of its digit before it.
__device__ uint64_t q_multi(const QStruct& S, int op, uint32_t c, uint64_t x) {
  const int L = S.L, D = S.levels;
  if (op == 2 ? x == 0 : x >= S.n) return NONE;
  if (op != 0 && c >= S.sigma) return NONE;
  auto dwidth = [&](int be) { return (2 * be + 1 < L) ? 2 : 1; };
  auto cdigit = [&](int be) -> uint32_t {
    const int w = dwidth(be);
    const int sh = L - 2 * be - w;
    return (c >> sh) & ((1u << w) - 1u);
  };
  uint64_t S0[17], R0[17];
  uint64_t s = 0, e = S.n, p = op == 1 ? x + 1 : x;
  uint32_t sym = 0;
  for (int be = 0; be < D; be++) {
    const DigLevel v = dig_level(S, be);
    const DigLine le = load_dig(v, e), ls = load_dig(v, s);
    DigLine lp;
    if (op != 2) lp = load_dig(v, p);
    const uint32_t d = op == 0 ? get_digit(v, p) : cdigit(be);
    uint64_t qs, ts, qe, te;
    dig_counts(ls, s, d, qs, ts);
    dig_counts(le, e, d, qe, te);
    const uint64_t cs = s + (te - ts);
    if (op == 2) {
      S0[be] = s;
      R0[be] = qs;
    } else {
      uint64_t qp, tp;
      dig_counts(lp, p, d, qp, tp);
      p = cs + (qp - qs);
      sym = (sym << dwidth(be)) | d;
    }
    s = cs;
    e = cs + (qe - qs);
  }
  if (op == 0) return sym;
  if (op == 1) return p - s;
  if (x > e - s) return NONE;
  uint64_t off = x - 1;
  for (int be = D - 1; be >= 0; be--) {
    const DigLevel v = dig_level(S, be);
    off = select_d(v, cdigit(be), R0[be] + off) - S0[be];
  }
  return off;  // the root starts at 0
}

__device__ uint64_t q_rs(const QStruct& S, int op, uint32_t c, uint64_t x) {
  BinLevel v = uniform_level(S, 0);
  v.nw = (S.n + 63) / 64;  // the caller's words
  if (op == 0) return x < S.n ? (uint64_t)get_bit(v, x) : NONE;
  if (c > 1) return NONE;
  if (op == 1) {
    if (x >= S.n) return NONE;
    return c ? rank1(v, x + 1) : rank0(v, x + 1);
  }
  const uint64_t cnt = c ? S.n - v.zeros : v.zeros;
  if (x == 0 || x > cnt) return NONE;
  return select_b(v, (int)c, x - 1);
}

__global__ void k_query(QStruct S, int op, const uint32_t* c, const uint64_t* x, uint64_t q,
                        uint64_t* out) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= q) return;
  const uint32_t ci = c ? c[i] : 0u;
  const uint64_t xi = x[i];
  uint64_t r;
  switch (S.kind) {
    case WT_KIND_WM: r = q_wm(S, op, ci, xi); break;
    case WT_KIND_WT: r = q_wt(S, op, ci, xi); break;
    case WT_KIND_HUFF: r = q_huff(S, op, ci, xi); break;
    case WT_KIND_MULTI: r = q_multi(S, op, ci, xi); break;
    default: r = q_rs(S, op, ci, xi); break;
  }
  out[i] = r;
}

static void fill_qstruct(const wt_struct* h, QStruct& S) {
  S.kind = h->kind;
  S.n = h->n;
  S.sigma = h->sigma;
  S.L = (int)h->L;
  S.levels = (int)h->levels;
  S.bits = h->d_bits_ro;
  S.dir = h->d_dir;
  S.samp = h->d_samp;
  S.meta = h->d_meta;
  S.zeros = h->d_zeros;
  S.start = h->d_start;
  S.hq.code = h->d_code;
  S.hq.len = h->d_len;
  S.hq.sym_by_rank = h->d_sym_by_rank;
  S.hq.len_first = h->d_len_tab;
  S.hq.len_base = h->d_len_tab ? h->d_len_tab + 34 : nullptr;
  S.hq.len_count = h->d_len_tab ? h->d_len_tab + 68 : nullptr;
  S.hq.node = h->d_node;
  S.hq.node_lvl = h->d_node_lvl;
  S.cmeta = h->d_cmeta;
  S.ck64 = h->d_ck64;
  S.ck32 = h->d_ck32;
}

// Threads per block: single warps while they all fit on the SMs at once, so
// that a small batch spreads over all of them.
static unsigned query_block(uint64_t q) { return q <= (uint64_t)num_sms() * 512 ? 32u : 128u; }

static wt_status build_starts(wt_struct* h) {
  QStruct S;
  fill_qstruct(h, S);
  k_wm_starts<<<((1u << h->L) + 63) / 64, 64, 0, h->stream>>>(S, h->d_start);
  count_launch();
  CK(cudaGetLastError());
  return WT_OK;
}

wt_status launch_query(wt_struct* h, int op, const uint32_t* c, const uint64_t* x, uint64_t q,
                       uint64_t* out, cudaStream_t st) {
  if (q == 0) return WT_OK;
  QStruct S;
  fill_qstruct(h, S);
  const unsigned bt = query_block(q);
  k_query<<<(unsigned)((q + bt - 1) / bt), bt, 0, st>>>(S, op, c, x, q, out);
  count_launch();
  CK(cudaGetLastError());
  return WT_OK;
}

// Queries over several structures in one launch: query i applies op[i] to
// structure sid[i] of the table.
__global__ void k_query_multi(const QStruct* tab, uint32_t ns, const uint32_t* sid,
                              const uint8_t* op, const uint32_t* c, const uint64_t* x, uint64_t q,
                              uint64_t* out) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= q) return;
  const uint32_t s = sid[i];
  const int o = op[i];
  if (s >= ns || o > 2) {
    out[i] = NONE;
    return;
  }
  const QStruct& S = tab[s];
  const uint32_t ci = c[i];
  const uint64_t xi = x[i];
  uint64_t r;
  switch (S.kind) {
    case WT_KIND_WM: r = q_wm(S, o, ci, xi); break;
    case WT_KIND_WT: r = q_wt(S, o, ci, xi); break;
    case WT_KIND_HUFF: r = q_huff(S, o, ci, xi); break;
    case WT_KIND_MULTI: r = q_multi(S, o, ci, xi); break;
    default: r = q_rs(S, o, ci, xi); break;
  }
  out[i] = r;
}

wt_status launch_query_multi(wt_struct* const* hs, uint32_t nh, const uint32_t* sid,
                             const uint8_t* op, const uint32_t* c, const uint64_t* x, uint64_t q,
                             uint64_t* out, cudaStream_t st) {
  if (q == 0) return WT_OK;
  std::vector<QStruct> tab(std::max<uint32_t>(nh, 1));
  for (uint32_t i = 0; i < nh; i++) fill_qstruct(hs[i], tab[i]);
  Work wk{st};
  QStruct* d_tab = nullptr;
  TRY(wk.get(&d_tab, tab.size()));
  TRY(upload(d_tab, tab.data(), tab.size() * sizeof(QStruct), st));
  const unsigned bt = query_block(q);
  k_query_multi<<<(unsigned)((q + bt - 1) / bt), bt, 0, st>>>(d_tab, nh, sid, op, c, x, q, out);
  count_launch();
  CK(cudaGetLastError());
  return WT_OK;
}

}  // namespace wtk
