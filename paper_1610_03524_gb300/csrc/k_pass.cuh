// k_pass.cuh -- the level-group partition kernel (one pass = t <= 4 levels).
//
// One CTA processes one tile of T_a at a time; no CTA waits on another.  A
// thread holds 32 consecutive elements of the tile as bit planes (bitplane.cuh),
// in which t - 1 stable 1-bit splits (Section 4.1: the descendants'
// sub-sequences are a stable integer sort on the next tau bits; Section 4.3:
// for the wavelet matrix the key is the reversed digit, i.e. the splits run
// from the level-a bit up) give its bits of levels a .. a+t-1, each in the
// order that level has inside the 32 elements, with every class's bits
// together.  The counts of the 2^t keys in the earlier threads (a prefix sum
// over the tile, two 16-bit counts a word) place those pieces in the tile's
// runs, one per (level, class), which are assembled in shared memory at the
// alignment they have in the output's 16-byte units; units that several tiles
// or nodes share (the "boundary" words of Section 4.2) are merged with
// atomicOr into the level buffer, which is zero before the pass
// (in a wavelet-matrix build each tile zeroes its share of the next pass's
// levels).  The same counts give every element's place in the tile's stable
// order by key: each thread walks its elements once with a pointer per key,
// and the runs of T_{a+t} (big nodes, Section 3), narrowed to the bits still
// needed, are again assembled at their output alignment.  One bulk copy takes
// each run out, behind the loads of the next tile; its first and last unit, if
// not the run's alone, are written piecewise.
//
// The digit counts of all earlier tiles of a tile's sequence or node come from
// prefix sums, taken before the pass, of every tile's digit counts: the
// domain decomposition of Section 4.2 with K = number of tiles and per-node
// offsets by prefix sums across the K sub-problems.
//
// What bounds it: instructions, most of them on the integer logic pipe (66% of
// its rate, 2.6 instructions per cycle and SM; DRAM at 10-20%), and the warps'
// waits for each other three times a tile.  Per 32 elements a pass takes 60 to
// 62 warp instructions, 42 the last one: the splits 13, the pieces 10, the move
// 11, loading, planes and prefix sums 15, the runs and their way out the rest.
// 2^30 16-bit symbols of 16 levels: 9.2 ms in four passes.  Moving every element
// through shared memory once per level (a ballot, a rank and a store per 32
// elements) in two passes of eight levels takes 231 and 198 instructions and
// 14.3 ms.  Three choices carry the difference: planes, which move 32 elements'
// bits at once; the first element in a plane's top bit, where half of a split's
// moves are multiplications on an idle pipe (2^28 symbols: 2.53 ms of passes
// against 2.74); and one bulk copy per run instead of a search and a store per
// word (2.44 against 2.53).
#pragma once
#include <type_traits>

#include "bitplane.cuh"
#include "wt_internal.cuh"

namespace wtk {

__device__ __forceinline__ uint32_t load_elem(const void* p, int w, uint64_t i) {
  if (w == 1) return ((const uint8_t*)p)[i];
  if (w == 2) return ((const uint16_t*)p)[i];
  return ((const uint32_t*)p)[i];
}

// Batched builds: tile ti's sequence, the last segment with tile0 <= ti, found
// by a whole warp, 32 segments a step (a binary search over 4096 sequences is
// twelve dependent loads).
__device__ __forceinline__ const SegDesc& seg_of(const PassParams& P0, uint32_t ti) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t lo = 0, hi = P0.nsegs - 1;
  while (lo < hi) {
    const uint32_t step = (hi - lo + 31) >> 5, at = lo + (lane + 1) * step;
    const bool before = at <= hi && P0.segs[at].tile0 <= ti;
    lo += step * (uint32_t)__popc(__ballot_sync(FULL, before));
    hi = min(hi, lo + step - 1);
  }
  return P0.segs[lo];
}

// Batched builds: the part of the parameters that belongs to tile ti's
// sequence into D (a whole warp; its first lane writes).
__device__ __forceinline__ void fill_seg(PassParams& D, const PassParams& P0, uint32_t ti) {
  const SegDesc& d = seg_of(P0, ti);
  if (threadIdx.x & 31) return;
  D.in = d.in;
  D.in_w = d.in_w;
  D.out = d.out;
  D.out_w = d.out_w;
  D.L = d.L;
  D.a = d.a;
  D.t = d.t;
  D.rbits = d.rbits;
  D.bits = d.bits;
  D.wm_cls = d.wm_cls;
  D.err = d.err;
  D.n_in = d.n;
  D.tile0 = d.tile0;
  D.sigma = d.sigma;
}

// A tile: where its elements are and which part of the pass it belongs to.
struct TileInfo {
  const unsigned char* src;
  uint64_t ts;          // its first element's index
  int cnt;
  uint32_t node, seg0;  // node of level a; first tile of its sequence or node
};

__device__ __forceinline__ TileInfo tile_info(const PassParams& P, uint32_t ti, uint32_t tile) {
  TileInfo I;
  if (P.tiles) {
    const TileDesc d = P.tiles[ti];
    I.ts = d.start;
    I.cnt = (int)d.count;
    I.node = d.node;
    I.seg0 = d.seg0;
  } else {
    I.ts = (uint64_t)(ti - P.tile0) * tile;
    const uint64_t rem = P.n_in - I.ts;
    I.cnt = (int)(rem < tile ? rem : tile);
    I.node = 0;
    I.seg0 = P.tile0;
  }
  I.src = (const unsigned char*)P.in + I.ts * (uint64_t)P.in_w;
  return I;
}

// Where the start of class k of level a+j stands (k = the tile-local key whose
// bit i is digit bit i, i.e. the LSD order of the splits), for a tile inside
// node `node` of level a; nullptr for Huffman prefixes that are not internal
// nodes at that level (their elements have left the tree).  hf: the pass's
// rows of hf_lvl.
__device__ __forceinline__ const uint64_t* class_start(const PassParams& P, int j, uint32_t k,
                                                       uint32_t node, const uint64_t* hf) {
  if (P.shape == SHAPE_WM) return P.wm_cls + ((1u << j) - 1u + (uint32_t)j) + k;
  const uint64_t q = ((uint64_t)node << j) | rev_bits(k, j);
  if (P.shape == SHAPE_WT) return P.wt_C + (q << (P.t - j));  // wt_C: node starts of level a + t
  const uint64_t off = hf[3 * j], first = hf[3 * j + 1], num = hf[3 * j + 2];
  return q < first || q >= first + num ? nullptr : P.hf_node + off + (q - first);
}

// 16-byte asynchronous copies into shared memory (each thread's own, complete
// for it after cp_async_wait and for the block after the next barrier)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
template <int B>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {  // 4 or 8 bytes
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(dst)), "l"(src), "n"(B) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Bulk copies from shared to global memory (both 16-byte aligned, a multiple
// of 16 bytes): issued by one thread, which waits until its copies have read
// their source; other threads' writes to the source are fenced before the
// barrier that precedes the copy.
__device__ __forceinline__ void bulk_store(uint64_t dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_addr(src)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ uint32_t ld_shared_u16(uint32_t a) {
  unsigned short v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
  return v;
}
template <int W>
__device__ __forceinline__ void st_shared(uint32_t a, uint32_t v) {
  if (W == 1) asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory");
  else if (W == 2) asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((unsigned short)v) : "memory");
  else asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// set the bits v at shared-memory word a (no access when there are none)
__device__ __forceinline__ void or_shared(uint32_t a, uint32_t v) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p red.shared.or.b32 [%0], %1;\n\t}" ::"r"(a), "r"(v)
               : "memory");
}

__device__ __forceinline__ uint64_t spread32(uint32_t v) {
  uint64_t x = v;
  x = (x | (x << 16)) & 0x0000FFFF0000FFFFull;
  x = (x | (x << 8)) & 0x00FF00FF00FF00FFull;
  x = (x | (x << 4)) & 0x0F0F0F0F0F0F0F0Full;
  x = (x | (x << 2)) & 0x3333333333333333ull;
  x = (x | (x << 1)) & 0x5555555555555555ull;
  return x;
}

// Shared memory of one CTA: the move's pointers, 1 KB a warp (at its own
// alignment, so that addresses are put together by OR); the tile as loaded, a
// row per thread padded by 16 bytes (eight lanes' 16-byte reads of their rows
// then fall on all banks); the elements in key order, each key's run at its
// output's 16-byte alignment (and before that the prefix sums' scratch); the
// level bits, each run at its output's 16-byte alignment too.
template <int EW, int NT>
struct PassSmem {
  static constexpr int T = 32 * NT, RS = 32 * EW + 16;
  static constexpr int KEYS = 1 << TAU_MAX, RUNS = KEYS - 1;
  static constexpr int SCRW = 8 * 32 + 3 * 8;                   // scratch words per warp
  static constexpr int AREA = TAU_MAX * T / 128 + 2 * RUNS + 2;  // 16-byte units
  static constexpr int SRT = T * EW + 32 * KEYS > NT / 32 * SCRW * 4 ? T * EW + 32 * KEYS : NT / 32 * SCRW * 4;
  static constexpr size_t off_ptr = 0;
  static constexpr size_t off_in = off_ptr + (size_t)(NT / 32) * 1024;
  static constexpr size_t off_srt = off_in + (size_t)NT * RS;
  static constexpr size_t off_area = off_srt + (size_t)SRT;
  static constexpr size_t bytes = off_area + (size_t)AREA * 16;
};

// CTAs per SM the register budget is sized for, at 128 threads
#ifndef WT_PASS_CTAS
#define WT_PASS_CTAS 8
#endif
template <int EW, int NT>
struct PassCtas {
  static constexpr int at128 = EW == 4 ? 5 : WT_PASS_CTAS;
  static constexpr int value = NT == 64 ? 2 * at128 : (NT == 128 ? at128 : at128 / 2);
};

// One run of a tile on its way out: the 16-byte units first .. last - 1 of its
// area are the run's alone, its area has n units from unit `at` on; unit i goes
// to address base + 16 i (base == 0: nowhere).
struct __align__(16) Run {
  uint64_t base;
  uint16_t first, last, at, n;
};

template <typename E, bool DIG, bool BATCH, int NT>
__global__ void __launch_bounds__(NT, (PassCtas<sizeof(E), NT>::value)) k_pass(const __grid_constant__ PassParams P0) {
  constexpr int EW = (int)sizeof(E), T = 32 * NT, W = NT / 32;
  using SM = PassSmem<EW, NT>;
  constexpr int RS = SM::RS, KEYS = SM::KEYS;
  static_assert(TAU_MAX == 4, "planes, keys and runs are laid out for four levels");
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* const s_in = smem + SM::off_in;
  unsigned char* const s_srt = smem + SM::off_srt;
  uint64_t* const s_area = (uint64_t*)(smem + SM::off_area);

  __shared__ PassParams s_P[BATCH ? 2 : 1];
  __shared__ TileInfo s_info[2];
  __shared__ __align__(16) uint32_t s_wtot[W][8];  // the warps' key counts, two a word
  // the next tile's table rows (its own, the next tile's and its first
  // tile's, within their chunks; the chunks' and the next chunk's) and class
  // starts, brought in with its elements
  __shared__ uint32_t s_ta[KEYS], s_tn[KEYS], s_tb[KEYS];
  __shared__ uint64_t s_ca[KEYS], s_cn[KEYS], s_cb[KEYS];
  __shared__ uint64_t s_cs[2 * KEYS - 1];
  __shared__ uint64_t s_hf[3 * (TAU_MAX + 1)], s_lo[TAU_MAX], s_ll[TAU_MAX];  // Huffman: rows of the level tables
  __shared__ uint32_t s_own[KEYS];  // the tile's key counts by the tables
  __shared__ bool s_over;           // a run past its level's or the sequence's end
  // the runs of level bits that are not empty, and those of the next
  // sequence; the latter's offset in the first unit, bytes << 8
  __shared__ Run s_run[2][KEYS];
  __shared__ uint32_t s_nr[2];
  __shared__ uint32_t s_edge[KEYS];
  __shared__ __align__(16) uint32_t s_ab[KEYS];  // a run's first bit, from shared memory's start
  __shared__ __align__(16) uint32_t s_sb[8];  // where a key's first element goes in s_srt, two keys a word

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* const ptr = (uint32_t*)(smem + SM::off_ptr) + warp * 256;
  uint32_t* const scr = (uint32_t*)s_srt + warp * SM::SCRW;
  const int bpe = DIG ? 2 : 1;
  const uint32_t ntiles = P0.tiles ? *P0.ntiles_dev : P0.ntiles;

  // tile ti's parameters into buffer b (the last thread; batched builds its warp)
  const bool sets = BATCH ? warp == W - 1 : tid == NT - 1;
  auto set_info = [&](uint32_t ti, int b) {
    if (BATCH) fill_seg(s_P[b], P0, ti);
    if (!BATCH || lane == 0) s_info[b] = tile_info(BATCH ? s_P[b] : P0, ti, T);
  };
  // its elements into s_in (all threads)
  auto load_tile = [&](int b) {
    const PassParams& P = BATCH ? s_P[b] : P0;
    const TileInfo I = s_info[b];
    if (I.cnt == T && ((uintptr_t)I.src & 15) == 0) {
#pragma unroll
      for (int k = 0; k < 2 * EW; k++) {
        const int i = tid + k * NT;
        cp_async16(s_in + 16 * i + 16 * (i / (2 * EW)), I.src + 16 * i);
      }
      return;
    }
    // else 4-byte words put together from the aligned words around them, as
    // far as those lie inside the sequence, and single elements
    int from = 0;
    const unsigned char* const base = (const unsigned char*)((uintptr_t)I.src & ~(uintptr_t)3);
    const uint32_t mis = (uint32_t)((uintptr_t)I.src & 3) * 8;
    if (base >= (const unsigned char*)P.in) {
      const uint64_t left = (uint64_t)((const unsigned char*)P.in + P.n_in * (uint64_t)EW - base) / 4;
      const int have = left > (uint64_t)(T * EW) ? T * EW : (int)left - (mis ? 1 : 0);
      const int nwords = min((I.cnt * EW + 3) / 4, have);
      const uint32_t* src = (const uint32_t*)base;
      for (int j = tid; j < nwords; j += NT) {
        const uint32_t lo = __ldcs(src + j), hi = mis ? __ldcs(src + j + 1) : 0u;
        *(uint32_t*)(s_in + 4 * j + 16 * (j / (8 * EW))) = __funnelshift_r(lo, hi, mis);
      }
      from = max(nwords, 0) * 4 / EW;
    }
    for (int i = from + tid; i < I.cnt; i += NT) {
      ((E*)(s_in + (i >> 5) * RS))[i & 31] = ((const E*)I.src)[i];
    }
  };

  // the control data of the tile ti whose parameters are in buffer b (warp 0)
  auto load_ctl = [&](uint32_t ti, int b) {
    const PassParams& P = BATCH ? s_P[b] : P0;
    const TileInfo I = s_info[b];
    const int nd = 1 << P.t;
    if (lane < nd) {
      const uint64_t* ca = P0.tchunk + (uint64_t)(ti >> P0.chsh) * TC_STRIDE + lane;
      const uint32_t* ta = P0.tcnt + (uint64_t)ti * TC_STRIDE + lane;
      cp_async<8>(s_ca + lane, ca);
      cp_async<8>(s_cn + lane, ca + TC_STRIDE);
      cp_async<8>(s_cb + lane, P0.tchunk + (uint64_t)(I.seg0 >> P0.chsh) * TC_STRIDE + lane);
      cp_async<4>(s_ta + lane, ta);
      cp_async<4>(s_tn + lane, ti + 1 < ntiles ? ta + TC_STRIDE : ta);
      cp_async<4>(s_tb + lane, P0.tcnt + (uint64_t)I.seg0 * TC_STRIDE + lane);
    }
    // lanes 0-14 the classes of levels a .. a+t-1, lanes 16-31 of level a+t
    if (lane < nd - 1 || (lane >= 16 && lane - 16 < nd && P.out != nullptr)) {
      const int ci = lane < 16 ? lane : nd - 1 + lane - 16;
      const int j = 31 - __clz(ci + 1);
      const uint64_t* at = class_start(P, j, (uint32_t)(ci + 1 - (1 << j)), I.node, s_hf);
      if (at) cp_async<8>(s_cs + ci, at);
      else s_cs[ci] = ~0ull;
    }
  };

  if (BATCH && tid < 2) s_P[tid] = P0;
  if (P0.shape == SHAPE_HUFF) {
    if (tid < 3 * (TAU_MAX + 1))
      s_hf[tid] = P0.a + tid / 3 < P0.L ? P0.hf_lvl[3 * P0.a + tid] : 0ull;
    if (tid < P0.t) {
      s_lo[tid] = P0.lvl_off[P0.a + tid];
      s_ll[tid] = P0.lvl_len[P0.a + tid];
    }
  }
  __syncthreads();
  uint32_t ti = blockIdx.x;
  int cur = 0;
  if (ti < ntiles) {
    if (sets) set_info(ti, 0);
    __syncthreads();
    load_tile(0);
    if (warp == 0) load_ctl(ti, 0);
  }
  for (; ti < ntiles; ti += gridDim.x, cur ^= 1) {
    const PassParams& P = BATCH ? s_P[cur] : P0;
    const bool more = ti + gridDim.x < ntiles;
    const int t = P.t, nd = 1 << t;
    const int cnt = s_info[cur].cnt;
    // this tile's share of the zeroing of a later pass's levels (stores that
    // use the DRAM bandwidth the tile's compute leaves idle)
    if (!BATCH && P0.clear && warp) clear_share(P0.clear, P0.clear_units, P0.clear_per, ti, tid - 32, NT - 32);
    cp_async_wait();
    if (warp == 0) bulk_wait_read();  // the last tile's runs have left
    __syncthreads();
    // (this, the zeroing above and the runs' ends are left to the other warps:
    // warp 0 has the runs to lay out, and the others wait for it)
    if (warp)
      for (int i = tid - 32; i < SM::AREA; i += NT - 32) ((uint4*)s_area)[i] = make_uint4(0u, 0u, 0u, 0u);

    // ---- 1. where the runs go (from the tables; warp 0, lanes 0-15 the level
    //      bits', lanes 16-31 the next sequence's), and the next tile ---------
    if (warp == 0) {
      const int half = lane >> 4, l16 = lane & 15;
      // l16 = r < 2^t: key r's count in the tile (a difference of prefixes) and
      // in the earlier tiles of its sequence or node
      uint32_t c = 0;
      uint64_t ex = 0;
      if (l16 < nd) {
        const bool last = ((ti + 1) >> P0.chsh) != (ti >> P0.chsh) || ti + 1 >= ntiles;
        const uint32_t a = s_ta[l16];
        c = last ? (uint32_t)(s_cn[l16] - s_ca[l16]) - a : s_tn[l16] - a;
        ex = (s_ca[l16] + a) - (s_cb[l16] + s_tb[l16]);
      }
      if (half == 0) s_own[l16] = c;
      // lanes 0-15: lane i takes class k of level j, i + 1 = 2^j + k: the keys'
      // counts folded level by level
      int j = 31 - __clz(l16 + 1);
      {
        const int mk = l16 + 1 - (1 << j);
        uint32_t fc = c, rc = 0;
        uint64_t fx = ex, rx = 0;
        for (int l = t - 1; l >= 0; l--) {
          fc += __shfl_down_sync(FULL, fc, 1 << l);
          fx += __shfl_down_sync(FULL, fx, 1 << l);
          const uint32_t yc = __shfl_sync(FULL, fc, mk);
          const uint64_t yx = __shfl_sync(FULL, fx, mk);
          if (j == l) {
            rc = yc;
            rx = yx;
          }
        }
        if (half == 0) {
          c = l16 < nd - 1 && (!DIG || (j & 1) == 0) ? rc : 0u;
          ex = rx;
        } else if (P.out == nullptr) {
          c = 0;
        }
      }
      uint32_t n = 0, len = 0, off = 0;  // 16-byte units; bits or bytes; offset in the first
      uint64_t where = 0;                // address of the first (0: nowhere)
      bool over = false;
      if (c) {
        const uint64_t cs = s_cs[half ? nd - 1 + l16 : l16], b0 = cs + ex;
        const bool dead = cs == ~0ull;
        if (half) {
          over = !dead && b0 + c > P.n_in;  // never for consistent tables
          where = (uint64_t)(uintptr_t)P.out + b0 * (uint64_t)P.out_w;
          off = (uint32_t)(where & 15);
          where -= off;
          len = c * (uint32_t)P.out_w;
          n = (off + len + 15) >> 4;
        } else {
          // levels of n_in elements back to back, or the Huffman tree's
          const uint64_t lv = (uint64_t)(DIG ? (P.a + j) >> 1 : P.a + j);
          const bool hf = P.shape == SHAPE_HUFF;
          const uint64_t lbits = hf ? s_ll[j] : P.n_in * bpe;
          const uint64_t lwords = hf ? s_lo[j] : lv * (((lbits + 2047) >> 11) << 5);
          const uint64_t G0 = b0 * bpe;
          len = c * bpe;
          over = !dead && G0 + len > lbits;  // never for consistent tables
          off = (uint32_t)(G0 & 127);
          n = (off + len + 127) >> 7;
          where = (uint64_t)(uintptr_t)(P.bits + lwords + 2 * (G0 >> 7));
        }
        if (dead) where = 0;
      }
      uint32_t first = n;
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, first, o, 16);
        if (l16 >= o) first += y;
      }
      first -= n;
      const uint32_t some = __ballot_sync(FULL, n != 0u) & (half ? 0xffff0000u : 0xffffu);
      if (n) {
        const int at = __popc(some & lanemask_lt()), sh = half ? 4 : 7;  // a unit's bytes or bits
        Run r;
        r.base = where ? where - 16ull * first : 0ull;
        r.first = (uint16_t)(first + (off ? 1u : 0u));
        r.last = (uint16_t)(where ? first + ((off + len) >> sh) : 0u);
        r.at = (uint16_t)first;
        r.n = (uint16_t)n;
        s_run[half][at] = r;
        if (half) s_edge[at] = where ? off | (len << 8) : 0u;
      }
      if (half) ((uint16_t*)s_sb)[l16] = (uint16_t)(16 * first + off);
      else s_ab[l16] = 8 * smem_addr(s_area) + 128 * first + off;
      if (l16 == 0) s_nr[half] = (uint32_t)__popc(some);
      const bool stop = __any_sync(FULL, over);
      if (lane == 0) s_over = stop;
    }
    if (sets && more) set_info(ti + gridDim.x, cur ^ 1);

    // ---- 2. planes and key counts of the thread's 32 elements -------------
    const unsigned char* const row = s_in + tid * RS;
    const int nv = min(max(cnt - 32 * tid, 0), 32);
    const uint32_t v = low_mask((uint32_t)nv);
    uint32_t p[4], C[8], X[8];
    planes_of<EW>([&](int i, uint32_t* w) {
      const uint4 q = *(const uint4*)(row + 16 * i);
      w[0] = q.x;
      w[1] = q.y;
      w[2] = q.z;
      w[3] = q.w;
    }, P.rbits, p);
    if (t < 2) p[1] = 0u;
    if (t < 3) p[2] = 0u;
    if (t < 4) p[3] = 0u;
    key_counts(p, v, C);
    // prefix sums over the warp: lane (q, k) adds up word k of eight lanes,
    // rows of eight words, eight apart more every eight rows (no bank is hit
    // twice by the four q)
    {
      uint32_t* const mine = scr + lane * 8 + (lane >> 3) * 8;
      *(uint4*)mine = make_uint4(C[0], C[1], C[2], C[3]);
      *(uint4*)(mine + 4) = make_uint4(C[4], C[5], C[6], C[7]);
      __syncwarp();
      const int k = lane & 7, q = lane >> 3;
      uint32_t* const col = scr + q * 72 + k;
      uint32_t c[8], sum = 0;
#pragma unroll
      for (int i = 0; i < 8; i++) {
        c[i] = col[8 * i];
        sum += c[i];
      }
      uint32_t inc = sum;
      uint32_t y = __shfl_up_sync(FULL, inc, 8);
      if (q >= 1) inc += y;
      y = __shfl_up_sync(FULL, inc, 16);
      if (q >= 2) inc += y;
      if (q == 3) s_wtot[warp][k] = inc;
      uint32_t run = inc - sum;
#pragma unroll
      for (int i = 0; i < 8; i++) {
        col[8 * i] = run;
        run += c[i];
      }
      __syncwarp();
      const uint4 a = *(const uint4*)mine, b = *(const uint4*)(mine + 4);
      X[0] = a.x;
      X[1] = a.y;
      X[2] = a.z;
      X[3] = a.w;
      X[4] = b.x;
      X[5] = b.y;
      X[6] = b.z;
      X[7] = b.w;
    }
    __syncthreads();

    // ---- 3. the splits ------------------------------------------------------
    // the tile's key counts against the tables': tables that disagree with the
    // tile would misplace its runs, so the tile is flagged (every warp finds
    // the same) and its outputs are left alone
    bool bad = s_over;
    {
      uint32_t tot = 0;
      if (lane < nd) {
#pragma unroll
        for (int w = 0; w < W; w++) tot += s_wtot[w][lane >> 1];
        tot = (tot >> (16 * (lane & 1))) & 0xffffu;
      }
      bad |= __any_sync(FULL, lane < nd && tot != s_own[lane & (KEYS - 1)]);
      if (bad && tid == 0) atomicOr(P.err, ERR_INTERNAL);
    }
#pragma unroll
    for (int j = 0; j < 4; j++) p[j] |= ~v;  // the bits past the tile's end stay last
    const uint32_t d1 = p[1];  // digit levels: the second bit of the first digit
    // (one copy of the code for every t: the last levels' splits are the same)
    if (t >= 2) {
      uint32_t x[4];  // the first element in the top bit
      if (t == 4) {
#pragma unroll
        for (int j = 0; j < 4; j++) x[j] = reverse32(p[j]);
      } else {
        x[1] = reverse32(p[0]);
        x[2] = t == 3 ? reverse32(p[1]) : x[1];
        x[3] = reverse32(t == 3 ? p[2] : p[1]);
      }
      if (t == 4) split_planes<3>(x[0], x + 1);
      if (t >= 3) split_planes<2>(x[1], x + 2);
      if (!DIG || t == 3) split_planes<1>(x[2], x + 3);
      p[1] = reverse32(t == 4 ? x[1] : (t == 3 ? x[2] : x[3]));
      p[2] = reverse32(t == 4 ? x[2] : x[3]);
      p[3] = reverse32(x[3]);
    }

    if (!bad) {
      // the earlier warps' counts
      for (int w = 0; w < warp; w++) {
        const uint4 a = *(const uint4*)s_wtot[w], b = *(const uint4*)(s_wtot[w] + 4);
        X[0] += a.x;
        X[1] += a.y;
        X[2] += a.z;
        X[3] += a.w;
        X[4] += b.x;
        X[5] += b.y;
        X[6] += b.z;
        X[7] += b.w;
      }
      // ---- 4. the level bits into the runs' areas -------------------------
      // a piece's set bits at bit q of shared memory (pieces of one thread or
      // of several share words)
      auto or_bits = [&](uint32_t q, uint32_t x) {
        const uint32_t w = (q >> 3) & ~3u;
        or_shared(w, __funnelshift_l(0u, x, q));
        or_shared(w + 4, __funnelshift_l(x, 0u, q));
      };
      // level j: its bits b0 (and b1, the digit's second bit), the thread's
      // and the earlier threads' counts of its classes
      auto level = [&](auto jc, uint32_t b0, uint32_t b1, const uint32_t* c, const uint32_t* x) {
        constexpr int j = decltype(jc)::value;
        uint32_t at = 0, below = 0, below1 = 0;  // bits of the classes before k, as masks
        // digits: the thread's 32 in two words, put together once for all classes
        // (for each class apart they cost a 4-ary build of 3*10^8 symbols 1.73
        // ms instead of 1.56)
        const uint64_t d = !DIG ? 0ull : (P.a + j + 1 < P.L ? (spread32(b0) << 1) | spread32(b1) : spread32(b0));
#pragma unroll
        for (int k = 0; k < (1 << j); k++) {
          const uint32_t n = (k & 1) ? c[k >> 1] >> 16 : c[k >> 1] & 0xffffu;
          const uint32_t xk = (k & 1) ? x[k >> 1] >> 16 : x[k >> 1] & 0xffffu;
          const uint32_t q = s_ab[(1 << j) - 1 + k] + xk * bpe - at * bpe;
          at += n;
          // shifted as they stand, from the earlier classes' bits before their place on
          if (!DIG) {
            const uint32_t upto = low_mask(at);
            or_bits(q, b0 & upto & ~below);
            below = upto;
          } else {
            const uint32_t upto = low_mask(2 * at), upto1 = low_mask((uint32_t)max((int)(2 * at) - 32, 0));
            const uint32_t y0 = (uint32_t)d & upto & ~below, y1 = (uint32_t)(d >> 32) & upto1 & ~below1;
            const uint32_t w = (q >> 3) & ~3u;
            or_shared(w, __funnelshift_l(0u, y0, q));
            or_shared(w + 4, __funnelshift_l(y0, y1, q));
            or_shared(w + 8, __funnelshift_l(y1, 0u, q));
            below = upto;
            below1 = upto1;
          }
        }
      };
      uint32_t c2[2], x2[2], c1, x1;
      {
        uint32_t c3[4], x3[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
          c3[k] = C[k] + C[k + 4];
          x3[k] = X[k] + X[k + 4];
        }
        if (!DIG && t > 3) level(std::integral_constant<int, 3>{}, p[3], 0u, c3, x3);
#pragma unroll
        for (int k = 0; k < 2; k++) {
          c2[k] = c3[k] + c3[k + 2];
          x2[k] = x3[k] + x3[k + 2];
        }
      }
      if (t > 2) level(std::integral_constant<int, 2>{}, p[2], p[3], c2, x2);
      c1 = c2[0] + c2[1];
      x1 = x2[0] + x2[1];
      if (!DIG && t > 1) level(std::integral_constant<int, 1>{}, p[1], 0u, &c1, &x1);
      const uint32_t c0 = (uint32_t)nv, x0 = min((uint32_t)(32 * tid), (uint32_t)cnt);
      level(std::integral_constant<int, 0>{}, p[0], d1, &c0, &x0);

      // ---- 5. the elements into key order ----------------------------------
      // a pointer per key and thread, two 16-bit ones a word: word b1 b2 b3
      // (the digit's lower bits as they stand in the element), half b0
      if (P.out != nullptr) {
        const uint32_t ow = (uint32_t)P.out_w;
#pragma unroll
        for (int k = 0; k < 8; k++) {
          const int rk = ((k & 1) << 2) | (k & 2) | (k >> 2);
          ptr[rk * 32 + lane] = s_sb[k] + X[k] * ow;
        }
        // (no other thread reads them)
        const uint32_t ptrs = smem_addr(ptr) + 4 * lane, srt = smem_addr(s_srt);
        const uint32_t m1 = t == 4 ? 0x380u : (t == 3 ? 0x300u : (t == 2 ? 0x200u : 0u));
        const int r1 = P.rbits - 11, r0 = P.rbits - 2;
        auto move = [&](auto wc) {
          constexpr int OW = decltype(wc)::value;
          constexpr int PER = 4 / EW;  // elements a word
          auto one = [&](uint32_t w, int sh) {
            const uint32_t pa = (rotr32(w, r0 + sh) & 2u) | ((rotr32(w, r1 + sh) & m1) | ptrs);
            const uint32_t to = ld_shared_u16(pa);
            st_shared<OW>(srt + to, w >> sh);
            st_shared<2>(pa, to + OW);
          };
          const int whole = nv * EW / 16;
#pragma unroll 1
          for (int i = 0; i < whole; i++) {
            const uint4 q = *(const uint4*)(row + 16 * i);
            const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int k = 0; k < 4; k++)
#pragma unroll
              for (int h = 0; h < PER; h++) one(w[k], 8 * EW * h);
          }
#pragma unroll 1
          for (int i = whole * 16 / EW; i < nv; i++) one((uint32_t)((const E*)row)[i], 0);
        };
        if (ow == 1) move(std::integral_constant<int, 1>{});
        else if (EW >= 2 && ow == 2) move(std::integral_constant<int, 2>{});
        else if (EW == 4) move(std::integral_constant<int, 4>{});
      }
    }
    fence_async_smem();
    __syncthreads();
    if (more) {  // behind the stores below
      load_tile(cur ^ 1);
      if (warp == 0) load_ctl(ti + gridDim.x, cur ^ 1);
    }
    if (bad) continue;  // uniform; nothing was put into the areas

    // ---- 6. the runs out: whole 16-byte units by bulk copies, a lane per run
    if (warp == 0) {
      const int half = lane >> 4;
      if ((uint32_t)(lane & 15) < s_nr[half]) {
        const Run r = s_run[half][lane & 15];
        const unsigned char* const from = half ? s_srt : (const unsigned char*)s_area;
        if (r.last > r.first && r.base)
          bulk_store(r.base + 16ull * r.first, from + 16 * r.first, 16 * (r.last - r.first));
      }
      bulk_commit();
      continue;
    }
    // the units at the runs' ends, shared with other tiles: level words ORed ...
    for (uint32_t e = tid - 32; e < 4 * s_nr[0]; e += NT - 32) {
      const Run r = s_run[0][e >> 2];
      const uint32_t u = r.at + ((e & 2) ? r.n - 1 : 0u);
      if (((e & 2) && r.n == 1) || (u >= r.first && u < r.last)) continue;
      const uint64_t x = s_area[2 * u + (e & 1)];
      if (x && r.base)
        atomicOr((unsigned long long*)(uintptr_t)(r.base + 16ull * u + 8 * (e & 1)), (unsigned long long)x);
    }
    // ... and elements four bytes a thread, one by one where not all are the run's
    if (P.out != nullptr) {
      for (uint32_t e = tid - 32; e < 8 * s_nr[1]; e += NT - 32) {
        const uint32_t at = e >> 3, b = 4 * (e & 3), oe = s_edge[at];
        const uint32_t off = oe & 0xffu, end = off + (oe >> 8);
        const uint32_t k = (e & 4) ? (end - 1) >> 4 : 0u;  // last unit or first
        const uint32_t lo = k ? 0u : off, hi = min(end - 16 * k, 16u);
        // once only, and only if not stored whole above
        if (oe == 0u || ((e & 4) && k == 0u) || hi - lo == 16u) continue;
        const uint32_t i = s_run[1][at].at + k;
        const unsigned char* from = s_srt + 16 * i + b;
        unsigned char* to = (unsigned char*)(uintptr_t)(s_run[1][at].base + 16ull * i) + b;
        if (lo <= b && b + 4 <= hi) {
          *(uint32_t*)to = *(const uint32_t*)from;
        } else if (P.out_w == 2) {
          if (lo <= b && b + 2 <= hi) *(uint16_t*)to = *(const uint16_t*)from;
          if (lo <= b + 2 && b + 4 <= hi) *(uint16_t*)(to + 2) = *(const uint16_t*)(from + 2);
        } else if (P.out_w == 1) {
#pragma unroll
          for (uint32_t q = 0; q < 4; q++)
            if (lo <= b + q && b + q < hi) to[q] = from[q];
        }
      }
    }
  }
  if (warp == 0) bulk_wait();
}

}  // namespace wtk
