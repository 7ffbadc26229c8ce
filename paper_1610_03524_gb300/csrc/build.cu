// build.cu -- construction of wavelet matrices, balanced / Huffman-shaped /
// 4-ary wavelet trees on one GPU.
//
// Pipeline of one build (all on one stream, no host synchronisation except
// for a Huffman code's tables):
//   1. Huffman-shaped trees: symbol counts, code (huffdev.cu, or huffman.cpp
//      for small alphabets) and the symbols' codewords, which the passes read;
//   2. per pass of up to four levels: every tile's digit counts (Section 4.1:
//      counting for the integer sort), the first pass's with the check of the
//      symbols; their prefix sums across the tiles (Section 4.2); from the
//      totals the start offsets of the pass's nodes or classes and its zero
//      counts z_l (Section 4.3): one launch up to SCAN_TILES tiles, else three;
//      then the partition (k_pass.cuh);
//   3. rank/select directories on every level (dirq.cu).
#include <algorithm>
#include <cmath>
#include <cooperative_groups.h>
#include <type_traits>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>

#include "k_pass.cuh"
#include "wt_host.h"

namespace wtk {


#define CK(x)                                                   \
  do {                                                          \
    cudaError_t e_ = (x);                                       \
    if (e_ != cudaSuccess) {                                    \
      fprintf(stderr, "wavelet: %s -> %s\n", #x, cudaGetErrorString(e_)); \
      cudaGetLastError(); /* reported here */                   \
      return e_ == cudaErrorMemoryAllocation ? WT_ERR_NO_MEMORY : WT_ERR_CUDA; \
    }                                                           \
  } while (0)

// Device memory comes from the device's stream-ordered pool.  The pool keeps
// up to POOL_KEEP bytes of freed memory reserved instead of returning it to
// the driver at every synchronisation, so repeated builds do not map and
// unmap their multi-GB buffers each time.  It reuses memory freed on another
// stream only once that free has completed (or the allocating stream already
// waits for it): it never makes one stream wait for another's work to hand
// memory over, which would serialise builds and copies queued on different
// streams; it takes more memory from the device instead.
constexpr uint64_t POOL_KEEP = 32ull << 30;

cudaError_t dmalloc(void** p, size_t bytes, cudaStream_t s) {
  static std::mutex mu;
  static bool done[64] = {false};
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64) {
    std::lock_guard<std::mutex> g(mu);
    if (!done[dev]) {
      cudaMemPool_t pool;
      if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
        uint64_t keep = POOL_KEEP;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        int no = 0;
        cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &no);
      }
      done[dev] = true;
    }
  }
  if (bytes == 0) bytes = 16;
  const cudaError_t e = cudaMallocAsync(p, bytes, s);
  // the caller has the error: the thread's next call does not meet it again
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}
void dfree(void* p, cudaStream_t s) {
  if (p) cudaFreeAsync(p, s);
}

Prof& prof() {
  static Prof p;
  return p;
}

uint32_t num_sms() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  return (uint32_t)sms;
}

static uint32_t levels_of(uint32_t sigma) {
  uint32_t L = 0;
  while (L < 32 && ((uint64_t)1 << L) < (uint64_t)sigma) L++;
  return L == 0 ? 1 : L;
}
static uint64_t level_words(uint64_t nbits) { return ((nbits + 2047) / 2048) * 32; }
static int width_for_bits(int b) { return b <= 8 ? 1 : (b <= 16 ? 2 : 4); }

// ---------------------------------------------------------------------------
// 1. histogram / validation
// ---------------------------------------------------------------------------
template <int WB, typename F>
__device__ __forceinline__ void for_each_symbol(const void* seq, uint64_t n, uint64_t gtid,
                                                uint64_t gstride, F&& f) {
  using T = typename std::conditional<WB == 1, uint8_t,
                                      typename std::conditional<WB == 2, uint16_t, uint32_t>::type>::type;
  const T* s = (const T*)seq;
  constexpr int PER = 16 / WB;
  const bool aligned = (((uintptr_t)seq) & 15) == 0;
  uint64_t nvec = aligned ? n / PER : 0;
  const uint4* v = (const uint4*)seq;
  for (uint64_t i = gtid; i < nvec; i += gstride) {
    const uint4 q = __ldcs(v + i);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (WB == 1) {
#pragma unroll
        for (int b = 0; b < 4; b++) f((w[k] >> (8 * b)) & 0xffu);
      } else if (WB == 2) {
        f(w[k] & 0xffffu);
        f(w[k] >> 16);
      } else {
        f(w[k]);
      }
    }
  }
  for (uint64_t i = nvec * PER + gtid; i < n; i += gstride) f((uint32_t)s[i]);
}

// What a pass's plan gives, from the totals of its tiles' digit counts by key
// (the digit reversed): for the wavelet matrix the class starts of its levels
// a .. a+t (level a+j's classes are the values of the key's low j bits) into
// cls and every level's zero count (the start of class 2^(j-1) after split j);
// for a balanced tree's first pass the starts of the nodes of level t.
enum PlanKind : int { PLAN_NONE = 0, PLAN_WM = 1, PLAN_WT = 2 };
struct PassPlan {
  int kind;
  int a, t;
  uint64_t* cls;    // WM
  uint64_t* C;      // WT: 2^t + 1
  uint64_t* zeros;  // WM
};

// exclusive prefix sums of one value a lane over the first n lanes
__device__ __forceinline__ uint64_t warp_scan_excl(uint64_t v, uint64_t& total) {
  const int lane = threadIdx.x & 31;
  uint64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  total = __shfl_sync(FULL, x, 31);
  return x - v;
}

// One warp: the plan from the totals, lane r < 2^t holding key r's.  Level j's
// counts are folded from level j+1's.  (A thread scanning each level in turn
// took 40-55 us for eight levels, more than any other kernel of a small
// build.)
__device__ void plan_pass(uint64_t tot, const PassPlan& p) {
  const int lane = threadIdx.x & 31, t = p.t;
  uint64_t c = lane < (1 << t) ? tot : 0ull, all;
  if (p.kind == PLAN_WT) {
    // in order of the digit: lane v takes the count of key rev(v)
    const uint64_t d = __shfl_sync(FULL, c, (int)rev_bits((uint32_t)lane & ((1u << t) - 1u), t));
    const uint64_t start = warp_scan_excl(lane < (1 << t) ? d : 0ull, all);
    if (lane <= (1 << t)) p.C[lane] = start;
    return;
  }
  for (int j = t; j >= 0; j--) {
    const int nk = 1 << j;
    const uint64_t start = warp_scan_excl(lane < nk ? c : 0ull, all);
    uint64_t* const out = p.cls + (nk - 1 + j);
    if (lane <= nk) out[lane] = start;  // the lane after the last class: the total
    if (j > 0 && lane == nk / 2) p.zeros[p.a + j - 1] = start;
    const uint64_t up = __shfl_down_sync(FULL, c, nk / 2);
    c += lane < nk / 2 ? up : 0ull;
  }
}

// Prefix sums of the tiles' counts of chunk c (2^chsh tiles), per key, in place,
// and the chunk's totals, by a block of 256: 64 tiles a step, warp (h, q) keys
// 4 q .. 4 q + 3 of tiles 32 h + lane.
__device__ __forceinline__ void scan_chunk(uint32_t* tcnt, uint32_t ntiles, uint32_t c, uint32_t chsh,
                                           uint64_t* tchunk) {
  constexpr int S = TC_STRIDE;
  static_assert(S == 16, "four threads a tile");
  __shared__ uint4 s_half[2][4];
  const int lane = threadIdx.x & 31, q = (threadIdx.x >> 5) & 3, h = threadIdx.x >> 7;
  auto add = [](uint4 a, uint4 b) { return make_uint4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); };
  uint4 carry = make_uint4(0u, 0u, 0u, 0u);
  for (uint32_t g = 0; g < 1u << (chsh - 6); g++) {
    const uint32_t ti = (c << chsh) + 64 * g + 32 * h + lane;
    uint4* const row = (uint4*)(tcnt + (uint64_t)ti * S) + q;
    const uint4 v = ti < ntiles ? __ldcg(row) : make_uint4(0u, 0u, 0u, 0u);
    uint4 x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint4 y = make_uint4(__shfl_up_sync(FULL, x.x, o), __shfl_up_sync(FULL, x.y, o),
                                 __shfl_up_sync(FULL, x.z, o), __shfl_up_sync(FULL, x.w, o));
      if (lane >= o) x = add(x, y);
    }
    if (g) __syncthreads();
    if (lane == 31) s_half[h][q] = x;
    __syncthreads();
    const uint4 lo = s_half[0][q];
    if (h) x = add(x, lo);
    x = add(x, carry);
    if (ti < ntiles) *row = make_uint4(x.x - v.x, x.y - v.y, x.z - v.z, x.w - v.w);
    carry = add(carry, add(lo, s_half[1][q]));
  }
  if (h && lane == 31) {
    uint64_t* const to = tchunk + (uint64_t)c * S + 4 * q;
    *(ulonglong2*)to = make_ulonglong2(carry.x, carry.y);
    *(ulonglong2*)(to + 2) = make_ulonglong2(carry.z, carry.w);
  }
}

// The prefix sums of the tiles' counts and the pass's plan as the tail of the
// counting kernel, for passes of at most SCAN_TILES tiles, which run one tile a
// warp: the block that is the last of its chunk's eight to finish scans the
// chunk's 64 tiles, and the one that finishes the last chunk scans the chunks
// and makes the plan (a block takes a ticket when it is done; no block waits
// for another).  A block's 256 threads hold a chunk's, or the chunks', counts
// in one round of loads.  A wavelet matrix of 12.3 million 32-bit symbols (5
// passes of 3015 tiles) went from 454 to 419 us with two launches less a pass,
// one of 50 million 16-bit ones (4 passes of 12208) from 1290 to 1258 us, a
// tree of 2^20 bytes from 184 to 167 us.  Above that the fence and the ticket
// of every block meet a kernel that DRAM bounds, and the launches no longer
// count.
constexpr uint32_t SCAN_TILES = 64 * SCAN_CHUNKS;
struct TileScan {
  uint32_t* tick;  // finished chunks, then every chunk's finished blocks: zero before and after
  uint32_t nchunk;
  uint64_t* tchunk;
  PassPlan plan;
};

// Whether the block is the last of n to come here; what the others wrote
// before is then visible to all its threads.
__device__ __forceinline__ bool last_block(uint32_t* tick, uint32_t n) {
  __shared__ bool s_last;
  __syncthreads();
  if (n == 1) return true;
  if (threadIdx.x == 0) {
    __threadfence();
    const bool last = atomicAdd(tick, 1u) == n - 1;
    if (last) *tick = 0;
    __threadfence();
    s_last = last;
  }
  __syncthreads();
  return s_last;
}

__device__ __noinline__ void scan_tail(uint32_t* tcnt, uint32_t ntiles, const TileScan& sc) {
  constexpr int S = TC_STRIDE;
  static_assert(S == 16 && SCAN_CHUNKS == 256, "a warp per two keys, eight chunks a lane");
  __shared__ uint64_t s_tot[S];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t c = blockIdx.x >> 3;
  if (!last_block(sc.tick + 1 + c, min(8u, gridDim.x - 8 * c))) return;
  scan_chunk(tcnt, ntiles, c, 6, sc.tchunk);
  if (!last_block(sc.tick, sc.nchunk)) return;
  {
    // warp w: keys 2 w and 2 w + 1, lanes the chunks
    ulonglong2 v[8];
#pragma unroll
    for (int g = 0; g < 8; g++) {
      const uint32_t i = 32 * g + lane;
      v[g] = i < sc.nchunk ? __ldcg((const ulonglong2*)(sc.tchunk + (uint64_t)i * S + 2 * warp))
                           : make_ulonglong2(0ull, 0ull);
    }
    uint64_t a = 0, b = 0;  // before the group
#pragma unroll
    for (int g = 0; g < 8; g++) {
      if (32u * g >= sc.nchunk) break;
      const uint32_t i = 32 * g + lane;
      uint64_t ta, tb;
      const uint64_t xa = warp_scan_excl(v[g].x, ta), xb = warp_scan_excl(v[g].y, tb);
      if (i < sc.nchunk)
        *(ulonglong2*)(sc.tchunk + (uint64_t)i * S + 2 * warp) = make_ulonglong2(a + xa, b + xb);
      a += ta;
      b += tb;
    }
    if (lane == 0) {
      *(ulonglong2*)(sc.tchunk + (uint64_t)sc.nchunk * S + 2 * warp) = make_ulonglong2(a, b);
      s_tot[2 * warp] = a;
      s_tot[2 * warp + 1] = b;
    }
  }
  __syncthreads();
  if (warp == 0 && sc.plan.kind != PLAN_NONE) plan_pass(lane < S ? s_tot[lane] : 0ull, sc.plan);
}

// Digit counts of every tile of a pass (the K sub-problems' per-class counts
// of Section 4.2), by key (the digit reversed): one warp per tile, the same
// tiles and digits as k_pass.  A lane takes 32 elements a step as bit planes
// (bitplane.cuh; their order does not matter) and counts each key's
// indicator word; the lanes' sums, two 16-bit counts a word, by eight warp
// reductions a tile.  No atomics and no barriers: about 4 instructions per
// 32 elements, so that DRAM is the bound, where a shared-memory atomic per
// element was.  First passes also check the symbols against sigma and zero
// their share of the pass's levels.
template <int EW, bool BATCH, bool SCAN>
__global__ void __launch_bounds__(256) k_tile_counts(const __grid_constant__ PassParams P0,
                                                     uint32_t* tcnt, uint32_t tile,
                                                     const __grid_constant__ TileScan sc) {
  __shared__ PassParams s_P[BATCH ? 8 : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t ntiles = P0.tiles ? *P0.ntiles_dev : P0.ntiles;
  const uint32_t nw = gridDim.x * 8;
  if (BATCH && lane == 0) s_P[warp] = P0;
  for (uint32_t ti = blockIdx.x * 8 + warp; ti < ntiles; ti += nw) {
    if (BATCH) {
      __syncwarp();
      fill_seg(s_P[warp], P0, ti);
      __syncwarp();
    }
    const PassParams& P = BATCH ? s_P[warp] : P0;
    if (!BATCH && P.clear) clear_share(P.clear, P.clear_units, P.clear_per, ti, lane, 32);
    const TileInfo I = tile_info(P, ti, tile);
    const int t = P.t;
    const uint32_t sigma = P.sigma;
    // every value of the element's width is below sigma: nothing to check
    const bool check = sigma != 0u && (EW == 4 || sigma < (1u << (8 * (EW & 3))));
    uint32_t acc[8] = {};
    uint32_t top[2] = {0u, 0u};  // running maxima (of 16-bit halves below 4 bytes)
    auto count = [&](uint32_t p[4], uint32_t v) {
      if (t < 2) p[1] = 0u;
      if (t < 3) p[2] = 0u;
      if (t < 4) p[3] = 0u;
      uint32_t c[8];
      key_counts(p, v, c);
#pragma unroll
      for (int k = 0; k < 8; k++) acc[k] += c[k];
    };
    bool bad = false;
    constexpr int PV = 16 / EW;  // elements a vector
    {
      // 16-byte vectors from the aligned one that holds the tile's first
      // element, 2 EW of them a lane and step; the ends' other elements masked
      const int skew = (int)(((uintptr_t)I.src & 15) / EW);
      const uint4* const src = (const uint4*)((uintptr_t)I.src & ~(uintptr_t)15);
      const uint4* const in0 = (const uint4*)(((uintptr_t)P.in + 15) & ~(uintptr_t)15);
      const uint4* const in1 = (const uint4*)(((uintptr_t)P.in + P.n_in * (uint64_t)EW) & ~(uintptr_t)15);
      const int nvec = (skew + I.cnt + PV - 1) / PV;
      const bool inside = skew == 0 && I.cnt == (int)tile;
      for (int i0 = 0; i0 < nvec; i0 += 64 * EW) {
        uint4 q[2 * EW];
        uint32_t v = FULL;
        if (inside) {
#pragma unroll
          for (int i = 0; i < 2 * EW; i++) q[i] = __ldcs(src + i0 + 32 * i + lane);
        } else {
          v = 0u;
#pragma unroll
          for (int i = 0; i < 2 * EW; i++) {
            const int at = i0 + 32 * i + lane;
            q[i] = make_uint4(0u, 0u, 0u, 0u);
            // elements lo .. hi - 1 of the vector are the tile's
            const int lo = max(skew - PV * at, 0), hi = min(skew + I.cnt - PV * at, PV);
            if (lo < hi) {
              if (src + at >= in0 && src + at < in1) {
                q[i] = __ldcs(src + at);
              } else {  // a vector that reaches past the sequence
                for (int e = lo; e < hi; e++) {
                  const uint32_t x = load_elem(src + at, EW, (uint64_t)e);
                  const uint32_t y = x << (8 * ((e * EW) & 3));
                  const int k = (e * EW) >> 2;
                  if (k == 0) q[i].x |= y;
                  else if (k == 1) q[i].y |= y;
                  else if (k == 2) q[i].z |= y;
                  else q[i].w |= y;
                }
              }
              v |= (low_mask((uint32_t)hi) & ~low_mask((uint32_t)lo)) << (PV * i);
              if (check && (lo > 0 || hi < PV)) {
                // the neighbours' elements out of the running maxima
                const uint32_t w[4] = {q[i].x, q[i].y, q[i].z, q[i].w};
                for (int e = lo; e < hi; e++) {
                  uint32_t x = w[0];
                  const int k = (e * EW) >> 2;
                  x = k == 1 ? w[1] : (k == 2 ? w[2] : (k == 3 ? w[3] : x));
                  x >>= 8 * ((e * EW) & 3);
                  if (EW == 1) x &= 0xffu;
                  if (EW == 2) x &= 0xffffu;
                  bad |= x >= sigma;
                }
              }
            }
          }
        }
        if (check) {
#pragma unroll
          for (int i = 0; i < 2 * EW; i++) {
            const uint32_t w[4] = {q[i].x, q[i].y, q[i].z, q[i].w};
            // whole vectors only
            if (!inside && ((v >> (PV * i)) & low_mask(PV)) != low_mask(PV)) continue;
#pragma unroll
            for (int k = 0; k < 4; k++) {
              if (EW == 4) {
                top[0] = max(top[0], w[k]);
              } else if (EW == 2) {
                top[0] = __vmaxu2(top[0], w[k]);
              } else {
                top[0] = __vmaxu2(top[0], w[k] & 0x00FF00FFu);
                top[1] = __vmaxu2(top[1], (w[k] >> 8) & 0x00FF00FFu);
              }
            }
          }
        }
        uint32_t p[4];
        planes_of<EW>([&](int i, uint32_t* w) {
          w[0] = q[i].x;
          w[1] = q[i].y;
          w[2] = q[i].z;
          w[3] = q[i].w;
        }, P.rbits, p);
        count(p, v);
      }
      if (check) {
        if (EW == 4) bad |= top[0] >= sigma;
        else bad |= max(max(top[0] & 0xffffu, top[0] >> 16), max(top[1] & 0xffffu, top[1] >> 16)) >= sigma;
      }
    }
    uint32_t mine = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t sum = __reduce_add_sync(FULL, acc[k]);
      if ((lane >> 1) == k) mine = (sum >> (16 * (lane & 1))) & 0xffffu;
    }
    if (lane < TC_STRIDE) tcnt[(uint64_t)ti * TC_STRIDE + lane] = mine;
    if (__any_sync(FULL, bad) && lane == 0) atomicOr(P.err, ERR_SYMBOL);
  }
  if (SCAN) scan_tail(tcnt, ntiles, sc);
}

// The same counts for bytes over SIG = 2 .. 8 values in a single pass
// (DNA-like text): one warp per tile, sixteen bytes a lane and step as two
// registers of 4-bit symbols, whose bits' three planes give each value's
// indicators by one three-input operation; they are added in 4-bit counters,
// and the lanes' sums by four warp reductions a tile.  No atomics, shared
// memory or barriers: about 3 instructions per 32 symbols, so that DRAM is
// the bound (2^32 symbols over 5 values with the zeroing of three levels:
// 1.0 ms, 5.9 TB/s; shared-memory atomics per symbol took 1.8 ms).  A symbol >=
// SIG is flagged; by which value it is counted does not matter (a single pass
// scatters nothing by these counts).
template <int SIG>
__global__ void __launch_bounds__(256) k_count_tiles_bytes(const uint8_t* seq, uint64_t n,
                                                           uint32_t* err, uint32_t* tcnt,
                                                           uint32_t tile, uint4* clear,
                                                           uint64_t clear_units,
                                                           uint64_t clear_per) {
  constexpr int NV = SIG - 1, T0 = SIG <= 2 ? 1 : (SIG <= 4 ? 2 : 3);
  constexpr uint32_t M = 0x11111111u;
  const int lane = threadIdx.x & 31;
  const uint64_t ntiles = (n + tile - 1) / tile;
  const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const bool vec = (((uintptr_t)seq) & 15) == 0;
  uint32_t bad = 0;
  for (uint64_t ti = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; ti < ntiles; ti += nw) {
    if (clear) clear_share(clear, clear_units, clear_per, ti, lane, 32);
    const uint64_t i0 = ti * tile;
    const uint32_t len = (uint32_t)(i0 + tile < n ? tile : n - i0);
    uint32_t cnt[NV] = {};  // of values 1 .. NV
    if (vec && len == tile) {
      const uint4* v = (const uint4*)(seq + i0) + lane;
      for (uint32_t k0 = 0; k0 < tile / 16; k0 += 128) {  // 4 steps of 32 x 16 bytes
        uint4 q[4];
#pragma unroll
        for (int k = 0; k < 4; k++) q[k] = __ldcs(v + k0 + 32 * k);
        uint32_t acc[NV] = {};
#pragma unroll
        for (int k = 0; k < 4; k++) {
          const uint32_t w[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
          bad |= (w[0] | w[1] | w[2] | w[3]) & 0xF8F8F8F8u;
          const uint32_t x[2] = {(w[0] & 0x07070707u) + 16u * (w[1] & 0x07070707u),
                                 (w[2] & 0x07070707u) + 16u * (w[3] & 0x07070707u)};
#pragma unroll
          for (int h = 0; h < 2; h++) {
            if (SIG < 8) bad |= (x[h] + (8u - SIG) * M) & (8u * M);
            const uint32_t b0 = x[h] & M, b1 = (x[h] >> 1) & M, b2 = (x[h] >> 2) & M;
#pragma unroll
            for (int s = 1; s <= NV; s++)
              acc[s - 1] += ((s & 1) ? b0 : ~b0) & ((s & 2) ? b1 : ~b1) & ((s & 4) ? b2 : ~b2);
          }
        }
#pragma unroll
        for (int s = 0; s < NV; s++)  // 4-bit counters (at most 8 each) to their sum
          cnt[s] += (((acc[s] & 0x0F0F0F0Fu) + ((acc[s] >> 4) & 0x0F0F0F0Fu)) * 0x01010101u) >> 24;
      }
    } else {
      for (uint32_t i = lane; i < len; i += 32) {
        const uint32_t x = seq[i0 + i];
        bad |= x >= SIG ? 1u : 0u;
#pragma unroll
        for (int s = 1; s <= NV; s++) cnt[s - 1] += x == (uint32_t)s ? 1u : 0u;
      }
    }
    // two sums per reduction (a tile has at most 8192 symbols)
    uint32_t rest = len, mine = 0;
#pragma unroll
    for (int s = 0; s < NV; s += 2) {
      const uint32_t two = __reduce_add_sync(FULL, cnt[s] | (s + 1 < NV ? cnt[s + 1] << 16 : 0u));
      const uint32_t lo = two & 0xffffu, hi = two >> 16;
      rest -= lo + hi;
      if (lane == (int)rev_bits((uint32_t)(s + 1), T0)) mine = lo;
      if (s + 1 < NV && lane == (int)rev_bits((uint32_t)(s + 2), T0)) mine = hi;
    }
    if (lane == 0) mine = rest;
    if (lane < TC_STRIDE) tcnt[ti * TC_STRIDE + lane] = mine;
  }
  if (__any_sync(FULL, bad != 0u) && lane == 0) atomicOr(err, ERR_SYMBOL);
}

// counts by k_count_tiles_bytes
static bool byte_counts(const PassParams& P) {
  return P.in_w == 1 && !P.tiles && P.sigma >= 2 && P.sigma <= 8 && P.t == P.L;
}

template <bool BATCH, bool SCAN>
static void launch_tile_counts(const PassParams& P, uint32_t T, unsigned grid, uint32_t* tcnt,
                               const TileScan& sc, cudaStream_t st) {
  if (P.in_w == 1) k_tile_counts<1, BATCH, SCAN><<<grid, 256, 0, st>>>(P, tcnt, T, sc);
  else if (P.in_w == 2) k_tile_counts<2, BATCH, SCAN><<<grid, 256, 0, st>>>(P, tcnt, T, sc);
  else k_tile_counts<4, BATCH, SCAN><<<grid, 256, 0, st>>>(P, tcnt, T, sc);
}

// Launch of a pass's tile counts into tcnt (mt tiles at most); sc: the scans and
// the plan too (at most SCAN_TILES tiles).
template <bool BATCH>
static wt_status launch_counts(const PassParams& P, uint32_t T, uint64_t mt, uint32_t* tcnt,
                               const TileScan* sc, cudaStream_t st) {
  const unsigned grid = (unsigned)std::min<uint64_t>((mt + 7) / 8, (uint64_t)num_sms() * 32);
  if (!BATCH && byte_counts(P)) {
    const uint8_t* sb = (const uint8_t*)P.in;
#define WT_COUNT_BYTES(S)                                                                          \
  case S:                                                                                          \
    k_count_tiles_bytes<S><<<grid, 256, 0, st>>>(sb, P.n_in, P.err, tcnt, T, P.clear,              \
                                                 P.clear_units, P.clear_per);                      \
    break
    switch (P.sigma) {
      WT_COUNT_BYTES(2);
      WT_COUNT_BYTES(3);
      WT_COUNT_BYTES(4);
      WT_COUNT_BYTES(5);
      WT_COUNT_BYTES(6);
      WT_COUNT_BYTES(7);
      WT_COUNT_BYTES(8);
    }
#undef WT_COUNT_BYTES
  } else if (!BATCH && sc) {
    launch_tile_counts<false, true>(P, T, (unsigned)((mt + 7) / 8), tcnt, *sc, st);
  } else {
    launch_tile_counts<BATCH, false>(P, T, grid, tcnt, TileScan{}, st);
  }
  count_launch();
  CK(cudaGetLastError());
  return WT_OK;
}

// Histogram of a byte sequence over sigma = NV + 1 <= 8 values, four bytes
// at a time in a 32-bit word: a byte equals v exactly when w ^ (v x
// 0x01010101) has a zero byte there, which ((t & 0x7F7F7F7F) + 0x7F7F7F7F)
// finds without carries between bytes; the count of the last value is the
// bytes seen minus the others.  No atomics per symbol.
template <int NV>
__device__ __forceinline__ void hist_bytes_swar(const void* seq, uint64_t n, uint64_t* hist,
                                                uint32_t* err) {
  constexpr uint32_t sigma = NV + 1;
  uint32_t cnt[NV > 0 ? NV : 1] = {};
  uint64_t seen = 0;
  bool bad = false;
  constexpr uint32_t ge = (0x80u - sigma) * 0x01010101u;  // + low 7 bits: bit 7 iff byte >= sigma
  auto word = [&](uint32_t w) {
    bad |= ((((w & 0x7F7F7F7Fu) + ge) | w) & 0x80808080u) != 0u;
#pragma unroll
    for (int v = 0; v < NV; v++) {
      const uint32_t t = w ^ ((uint32_t)v * 0x01010101u);
      const uint32_t y = (t & 0x7F7F7F7Fu) + 0x7F7F7F7Fu;
      cnt[v] += __popc(~(y | t) & 0x80808080u);
    }
  };
  const uint8_t* sb = (const uint8_t*)seq;
  const uint64_t gt = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t gs = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t nvec = ((((uintptr_t)seq) & 15) == 0) ? n / 16 : 0;
  const uint4* vp = (const uint4*)seq;
  for (uint64_t i = gt; i < nvec; i += gs) {
    const uint4 q = __ldcs(vp + i);
    word(q.x);
    word(q.y);
    word(q.z);
    word(q.w);
    seen += 16;
  }
  for (uint64_t i = nvec * 16 + gt; i < n; i += gs) {
    const uint32_t x = sb[i];
    bad |= x >= sigma;
#pragma unroll
    for (int v = 0; v < NV; v++) cnt[v] += x == (uint32_t)v ? 1u : 0u;
    seen++;
  }
  if (bad) atomicOr(err, ERR_SYMBOL);
  const int lane = threadIdx.x & 31;
  uint64_t rest = seen;
#pragma unroll
  for (int v = 0; v < NV; v++) rest -= cnt[v];
#pragma unroll
  for (int v = 0; v <= NV; v++) {
    uint64_t c = v < NV ? (uint64_t)cnt[v] : rest;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
    if (lane == 0 && c) atomicAdd((unsigned long long*)&hist[v], (unsigned long long)c);
  }
}

// Full symbol histogram (balanced / Huffman / 4-ary trees).
// (large alphabets: block b adds into copy b % ncopy of the histogram, at
// (b % ncopy) * sigma, so that the frequent symbols of a skewed alphabet
// spread their atomics over several addresses; the copies are summed
// afterwards.  The copies are 32-bit (hist32) while no count can reach
// 2^32, so that 16 copies of a 2^20-symbol alphabet, 64 MB, stay in L2: as
// 64-bit copies they took 128 MB and their atomics went to DRAM)
template <int WB>
__global__ void k_hist_full(const void* seq, uint64_t n, uint32_t sigma, uint64_t* hist,
                            uint32_t* err, int use_smem, uint32_t ncopy = 1,
                            uint32_t* hist32 = nullptr) {
  extern __shared__ uint32_t shh[];
  if (use_smem) {
    for (uint32_t i = threadIdx.x; i < sigma; i += blockDim.x) shh[i] = 0;
    __syncthreads();
  }
  bool bad = false;
  const int lane = threadIdx.x & 31;
  if (WB == 1 && sigma <= 8) {
    // byte sequences over tiny alphabets (DNA-like text)
    switch (sigma) {
      case 1: hist_bytes_swar<0>(seq, n, hist, err); return;
      case 2: hist_bytes_swar<1>(seq, n, hist, err); return;
      case 3: hist_bytes_swar<2>(seq, n, hist, err); return;
      case 4: hist_bytes_swar<3>(seq, n, hist, err); return;
      case 5: hist_bytes_swar<4>(seq, n, hist, err); return;
      case 6: hist_bytes_swar<5>(seq, n, hist, err); return;
      case 7: hist_bytes_swar<6>(seq, n, hist, err); return;
      default: hist_bytes_swar<7>(seq, n, hist, err); return;
    }
  }
  for_each_symbol<WB>(seq, n, (uint64_t)blockIdx.x * blockDim.x + threadIdx.x,
                      (uint64_t)gridDim.x * blockDim.x, [&](uint32_t x) {
                        const bool ok = x < sigma;
                        bad |= !ok;
                        if (use_smem) {
                          if (ok) atomicAdd(&shh[x], 1u);
                        } else {
                          // lanes holding the same symbol add once (skewed
                          // alphabets put many lanes on the frequent ones)
                          const uint32_t act = __activemask();
                          const uint32_t peers = __match_any_sync(act, x);
                          if (ok && lane == __ffs(peers) - 1) {
                            const uint64_t at = (uint64_t)(blockIdx.x % ncopy) * sigma + x;
                            if (hist32) atomicAdd(&hist32[at], (uint32_t)__popc(peers));
                            else atomicAdd((unsigned long long*)&hist[at], (unsigned long long)__popc(peers));
                          }
                        }
                      });
  if (bad) atomicOr(err, ERR_SYMBOL);
  if (use_smem) {
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < sigma; i += blockDim.x)
      if (shh[i]) atomicAdd((unsigned long long*)&hist[i], (unsigned long long)shh[i]);
  }
}

// The histogram of a large alphabet with a table of HIST_SLOTS counters in
// shared memory, one block an SM: a slot belongs to the first of its symbols
// (those equal modulo HIST_SLOTS) that the block meets, which a frequent one
// is likely to be, and its other symbols are added to the global copies.  The
// table is emptied every HIST_ROUNDS steps of the block, so that symbols that
// become frequent later find a slot too.  Lanes that hold the same symbol add
// once where most of a warp misses the table (else the search for them costs
// more than their atomics).  The atomics of a symbol each were the bound: 2^28
// symbols over 2^20 (Zipf) took 1.85 ms, 0.70 here.
constexpr uint32_t HIST_SLOTS = 1u << 14;
constexpr uint32_t HIST_ROUNDS = 64;
template <int WB>
__global__ void __launch_bounds__(1024, 1) k_hist_slots(const void* seq, uint64_t n, uint32_t sigma,
                                                        uint64_t* hist, uint32_t* err, uint32_t ncopy,
                                                        uint32_t* hist32) {
  extern __shared__ uint32_t shh[];
  uint32_t *const tag = shh, *const cnt = shh + HIST_SLOTS;
  for (uint32_t i = threadIdx.x; i < HIST_SLOTS; i += 1024) {
    tag[i] = ~0u;
    cnt[i] = 0u;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const uint64_t copy = (uint64_t)(blockIdx.x % ncopy) * sigma;
  auto add_global = [&](uint32_t x, uint32_t c) {
    if (hist32) atomicAdd(&hist32[copy + x], c);
    else atomicAdd((unsigned long long*)&hist[copy + x], (unsigned long long)c);
  };
  bool bad = false;
  auto one = [&](uint32_t x) {
    if (x >= sigma) {
      bad = true;
      return;
    }
    const uint32_t slot = x & (HIST_SLOTS - 1);
    uint32_t t = ((volatile uint32_t*)tag)[slot];
    if (t == ~0u) {
      t = atomicCAS(&tag[slot], ~0u, x);
      if (t == ~0u) t = x;
    }
    if (t == x) {
      atomicAdd(&cnt[slot], 1u);
    } else {
      const uint32_t act = __activemask();
      if (__popc(act) <= 20) {
        add_global(x, 1u);
      } else {
        const uint32_t peers = __match_any_sync(act, x);
        if (lane == __ffs(peers) - 1) add_global(x, (uint32_t)__popc(peers));
      }
    }
  };
  auto flush = [&]() {
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < HIST_SLOTS; i += 1024) {
      if (cnt[i]) add_global(tag[i], cnt[i]);
      tag[i] = ~0u;
      cnt[i] = 0u;
    }
    __syncthreads();
  };
  constexpr int PER = 16 / WB;
  const uint64_t nvec = (((uintptr_t)seq) & 15) == 0 ? n / PER : 0, stride = (uint64_t)gridDim.x * 1024;
  const uint4* const v = (const uint4*)seq;
  uint64_t i = (uint64_t)blockIdx.x * 1024 + threadIdx.x;
  uint4 q = make_uint4(0u, 0u, 0u, 0u);
  if (i < nvec) q = __ldcs(v + i);
  uint32_t round = 0;
  for (uint64_t b = (uint64_t)blockIdx.x * 1024; b < nvec; b += stride, i += stride) {
    const uint4 w = q;
    if (i + stride < nvec) q = __ldcs(v + i + stride);
    if (i < nvec) {
      const uint32_t e[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int k = 0; k < 4; k++) {
        if (WB == 4) {
          one(e[k]);
        } else {
          one(e[k] & 0xffffu);
          one(e[k] >> 16);
        }
      }
    }
    if (++round % HIST_ROUNDS == 0) flush();
  }
  for (uint64_t k = nvec * PER + (uint64_t)blockIdx.x * 1024 + threadIdx.x; k < n; k += stride)
    one(load_elem(seq, WB, k));
  if (bad) atomicOr(err, ERR_SYMBOL);
  flush();
}

template <typename C>
__global__ void k_hist_sum_copies(const C* copies, uint32_t sigma, uint32_t ncopy, uint64_t* hist) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < sigma;
       i += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t a = 0;
    for (uint32_t c = 0; c < ncopy; c++) a += copies[(uint64_t)c * sigma + i];
    hist[i] += a;
  }
}

#ifndef WT_HIST_COPY_MB
#define WT_HIST_COPY_MB 64
#endif
constexpr uint64_t HIST_COPY_BYTES = (uint64_t)WT_HIST_COPY_MB << 20;

// below this the tables' clearing and emptying outweigh the atomics saved
constexpr uint64_t HIST_SLOTS_MIN = 1ull << 22;
static wt_status launch_hist_full(const void* seq, int w, uint64_t n, uint32_t sigma,
                                  uint64_t* hist, uint32_t* err, cudaStream_t st) {
  if (n == 0) return WT_OK;
  const int use_smem = sigma <= 12288;
  const size_t shb = use_smem ? sigma * 4 : 0;
  const uint32_t blocks = std::min<uint64_t>(num_sms() * 4, (n + 4095) / 4096 + 1);
  // global counters: up to 16 copies (32-bit while no count can reach 2^32),
  // taking at most HIST_COPY_BYTES so that they stay in L2
  uint32_t ncopy = 1;
  uint64_t* dst = hist;
  uint32_t* dst32 = nullptr;
  Work wk{st};
  const bool narrow = n < (1ull << 32);
  if (!use_smem) {
    const uint64_t c32 = HIST_COPY_BYTES / (4ull * sigma);
    if (narrow && c32 >= 2) {
      ncopy = (uint32_t)std::min<uint64_t>(16, c32);
      TRY(wk.get(&dst32, (size_t)ncopy * sigma));
      CK(cudaMemsetAsync(dst32, 0, (size_t)ncopy * sigma * 4, st));
    } else if ((ncopy = (uint32_t)std::max<uint64_t>(
                    1, std::min<uint64_t>(16, HIST_COPY_BYTES / (8ull * sigma)))) > 1) {
      TRY(wk.get(&dst, (size_t)ncopy * sigma));
      CK(cudaMemsetAsync(dst, 0, (size_t)ncopy * sigma * 8, st));
    }
  }
  if (!use_smem && w > 1 && n >= HIST_SLOTS_MIN) {
    constexpr int bytes = 8 * (int)HIST_SLOTS;
    auto kern = w == 2 ? k_hist_slots<2> : k_hist_slots<4>;
    CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    kern<<<(unsigned)num_sms(), 1024, bytes, st>>>(seq, n, sigma, dst, err, ncopy, dst32);
  } else if (w == 1) k_hist_full<1><<<blocks, 512, shb, st>>>(seq, n, sigma, dst, err, use_smem, ncopy, dst32);
  else if (w == 2) k_hist_full<2><<<blocks, 512, shb, st>>>(seq, n, sigma, dst, err, use_smem, ncopy, dst32);
  else k_hist_full<4><<<blocks, 512, shb, st>>>(seq, n, sigma, dst, err, use_smem, ncopy, dst32);
  count_launch();
  CK(cudaGetLastError());
  const unsigned sg = (unsigned)std::min<uint64_t>((sigma + 255) / 256, (uint64_t)num_sms() * 8);
  if (dst32) {
    k_hist_sum_copies<uint32_t><<<sg, 256, 0, st>>>(dst32, sigma, ncopy, hist);
    count_launch();
    CK(cudaGetLastError());
  } else if (ncopy > 1) {
    k_hist_sum_copies<uint64_t><<<sg, 256, 0, st>>>(dst, sigma, ncopy, hist);
    count_launch();
    CK(cudaGetLastError());
  }
  return WT_OK;
}

// ---------------------------------------------------------------------------
// exclusive scan of u64 (n entries -> n+1 outputs); reduce, scan, add
// ---------------------------------------------------------------------------
constexpr int SCAN_BT = 1024, SCAN_PER = 4, SCAN_CH = SCAN_BT * SCAN_PER;

__device__ uint64_t block_scan_excl_u64(uint64_t v, uint64_t* total) {
  __shared__ uint64_t ws[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    uint64_t s = lane < nw ? ws[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(FULL, s, o);
      if (lane >= o) s += y;
    }
    if (lane < nw) ws[lane] = s;
  }
  __syncthreads();
  const uint64_t base = warp ? ws[warp - 1] : 0;
  if (total) *total = ws[(blockDim.x >> 5) - 1];
  __syncthreads();
  return base + x - v;
}

__global__ void k_scan_reduce(const uint64_t* in, uint64_t n, uint64_t* bsum) {
  const uint64_t b0 = (uint64_t)blockIdx.x * SCAN_CH;
  uint64_t s = 0;
  for (int k = 0; k < SCAN_PER; k++) {
    const uint64_t i = b0 + (uint64_t)k * SCAN_BT + threadIdx.x;
    if (i < n) s += in[i];
  }
  uint64_t tot;
  block_scan_excl_u64(s, &tot);
  if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void k_scan_top(uint64_t* bsum, uint64_t nb) {
  __shared__ uint64_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (uint64_t c0 = 0; c0 < nb; c0 += blockDim.x) {
    const uint64_t i = c0 + threadIdx.x;
    const uint64_t v = i < nb ? bsum[i] : 0;
    uint64_t tot;
    const uint64_t ex = block_scan_excl_u64(v, &tot);
    if (i < nb) bsum[i] = carry + ex;
    __syncthreads();
    if (threadIdx.x == 0) carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) bsum[nb] = carry;
}

__global__ void k_scan_down(const uint64_t* in, uint64_t n, const uint64_t* bsum, uint64_t* out) {
  const uint64_t b0 = (uint64_t)blockIdx.x * SCAN_CH;
  const uint64_t i0 = b0 + (uint64_t)threadIdx.x * SCAN_PER;
  uint64_t v[SCAN_PER], s = 0;
  for (int k = 0; k < SCAN_PER; k++) {
    v[k] = (i0 + k < n) ? in[i0 + k] : 0;
    s += v[k];
  }
  uint64_t ex = block_scan_excl_u64(s, nullptr) + bsum[blockIdx.x];
  for (int k = 0; k < SCAN_PER; k++) {
    if (i0 + k < n) out[i0 + k] = ex;
    ex += v[k];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = bsum[gridDim.x];
}

// out[0..n] = exclusive prefix of in[0..n); scratch >= n/4096 + 2 entries
static wt_status scan_excl_u64(const uint64_t* in, uint64_t* out, uint64_t n, uint64_t* scratch,
                               cudaStream_t st) {
  const uint64_t nb = (n + SCAN_CH - 1) / SCAN_CH;
  if (nb == 0) {
    CK(cudaMemsetAsync(out, 0, sizeof(uint64_t), st));
    return WT_OK;
  }
  k_scan_reduce<<<(unsigned)nb, SCAN_BT, 0, st>>>(in, n, scratch);
  count_launch();
  k_scan_top<<<1, SCAN_BT, 0, st>>>(scratch, nb);
  count_launch();
  k_scan_down<<<(unsigned)nb, SCAN_BT, 0, st>>>(in, n, scratch, out);
  count_launch();
  CK(cudaGetLastError());
  return WT_OK;
}
static uint64_t scan_scratch(uint64_t n) { return n / SCAN_CH + 2; }

// ---------------------------------------------------------------------------
// 2. plans
// ---------------------------------------------------------------------------
struct PassGeom {
  int a, t, rbits, in_w, out_w;
};

static std::vector<PassGeom> make_passes(int L, int tau, int first_w) {
  std::vector<PassGeom> ps;
  for (int a = 0; a < L; a += tau) {
    PassGeom p;
    p.a = a;
    p.t = std::min(tau, L - a);
    p.rbits = L - a;
    p.in_w = a == 0 ? first_w : width_for_bits(L - a);
    p.out_w = (a + p.t < L) ? width_for_bits(L - a - p.t) : 0;
    ps.push_back(p);
  }
  return ps;
}

// The sequences between the passes: pass g writes buffer g & 1, which holds the
// largest of the outputs that it gets (count(g): elements that pass g writes).
template <typename Count>
static void want_seqbufs(Work& wk, uint8_t* buf[2], const std::vector<PassGeom>& ps, Count&& count) {
  const int G = (int)ps.size();
  for (int k = 0; k < std::min(G - 1, 2); k++) {
    uint64_t bytes = 0;
    for (int g = k; g + 1 < G; g += 2)
      bytes = std::max<uint64_t>(bytes, count(g) * (uint64_t)ps[g].out_w);
    wk.want(&buf[k], bytes);
  }
}

// Batched builds, one warp per sequence of the launch: the plan of its pass
// from the totals of its own tiles' digit counts, i.e. the difference of the
// scanned tables' prefixes at its last and first tile (tcnt exclusive within
// chunks of 2^chsh tiles, tchunk the chunks' exclusive prefixes with the
// total after the last chunk).
__device__ __forceinline__ uint64_t tile_prefix(const uint32_t* tcnt, const uint64_t* tchunk,
                                                uint32_t ntiles, uint32_t nchunk, uint32_t chsh,
                                                uint32_t ti, uint32_t r) {
  if (ti >= ntiles) return tchunk[(uint64_t)nchunk * TC_STRIDE + r];
  return tchunk[(uint64_t)(ti >> chsh) * TC_STRIDE + r] + tcnt[(uint64_t)ti * TC_STRIDE + r];
}

__global__ void __launch_bounds__(256) k_plan_batch_pass(const SegDesc* segs, uint32_t nsegs,
                                                         const uint32_t* tcnt,
                                                         const uint64_t* tchunk, uint32_t ntiles,
                                                         uint32_t nchunk, uint32_t chsh) {
  const uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, r = threadIdx.x & 31;
  if (i >= nsegs) return;
  const SegDesc& d = segs[i];
  const uint32_t t0 = d.tile0, t1 = t0 + (uint32_t)((d.n + PASS_T - 1) / PASS_T);
  uint64_t tot = 0;
  if (r < (1u << d.t))
    tot = tile_prefix(tcnt, tchunk, ntiles, nchunk, chsh, t1, r) -
          tile_prefix(tcnt, tchunk, ntiles, nchunk, chsh, t0, r);
  plan_pass(tot, PassPlan{PLAN_WM, d.a, d.t, d.wm_cls, nullptr, d.zeros});
}

// Balanced trees, passes after the first, one warp per node q of level a: the
// starts of its descendants on level a + t, C[q 2^t .. (q+1) 2^t), from the
// totals of the node's tiles toff[q] .. toff[q+1] - 1 (and C's last entry, n).
__global__ void __launch_bounds__(256) k_plan_nodes(const uint64_t* Ca, const uint64_t* toff,
                                                    uint64_t nn, int t, uint64_t n,
                                                    const uint32_t* tcnt, const uint64_t* tchunk,
                                                    const uint32_t* ntiles_dev, uint32_t nchunk,
                                                    uint32_t chsh, uint64_t* C) {
  const uint64_t q = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t v = threadIdx.x & 31;
  if (q >= nn) return;
  const uint32_t ntiles = *ntiles_dev;
  const uint32_t t0 = (uint32_t)toff[q], t1 = (uint32_t)toff[q + 1];
  uint64_t tot = 0, all;
  if (v < (1u << t) && t1 > t0) {
    const uint32_t r = rev_bits(v, t);
    tot = tile_prefix(tcnt, tchunk, ntiles, nchunk, chsh, t1, r) -
          tile_prefix(tcnt, tchunk, ntiles, nchunk, chsh, t0, r);
  }
  const uint64_t start = Ca[q] + warp_scan_excl(tot, all);
  if (v < (1u << t)) C[(q << t) + v] = start;
  if (q + 1 == nn && v == 0) C[nn << t] = n;
}

// Balanced-tree helpers over C (C[v] = number of symbols < v, v in [0, 2^L]).
// Zero counts: z_l = sum over nodes q of level l of the size of the left child.
__global__ void k_wt_zeros(const uint64_t* C, int L, uint64_t* zeros) {
  // one block per level
  const int l = blockIdx.x;
  const int sh = L - l - 1;
  uint64_t s = 0;
  for (uint64_t q = threadIdx.x; q < ((uint64_t)1 << l); q += blockDim.x)
    s += C[(2 * q + 1) << sh] - C[(2 * q) << sh];
  uint64_t tot;
  block_scan_excl_u64(s, &tot);
  if (threadIdx.x == 0) zeros[l] = tot;
}

// Node-aligned tiles over T_a: node p spans [bnd[p], bnd[p+1]).
__global__ void k_tiles_count(const uint64_t* bnd, uint64_t nn, uint32_t T, uint64_t* tcnt) {
  const uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nn) return;
  const uint64_t sz = bnd[p + 1] - bnd[p];
  tcnt[p] = (sz + T - 1) / T;
}

// The tile counts' and offsets of up to 4096 nodes by one block (one launch
// instead of four).
__global__ void __launch_bounds__(1024) k_tiles_offsets(const uint64_t* bnd, uint32_t nn, uint32_t T,
                                                        uint64_t* toff) {
  uint64_t c[4], sum = 0;
  const uint32_t p0 = threadIdx.x * 4;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    c[k] = p0 + k < nn ? (bnd[p0 + k + 1] - bnd[p0 + k] + T - 1) / T : 0ull;
    sum += c[k];
  }
  uint64_t tot, ex = block_scan_excl_u64(sum, &tot);
#pragma unroll
  for (int k = 0; k < 4; k++) {
    if (p0 + k < nn) toff[p0 + k] = ex;
    ex += c[k];
  }
  if (threadIdx.x == 0) toff[nn] = tot;
}

// One thread per tile: tile i belongs to the node p with toff[p] <= i <
// toff[p+1] (nodes without tiles share their toff with the next node, so the
// last p with toff[p] <= i is the right one).
__global__ void k_tiles_write(const uint64_t* bnd, uint64_t nn, uint32_t T, uint64_t node_base, const uint64_t* toff, TileDesc* tiles,
                              uint32_t* ntiles, uint64_t max_tiles) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t total = toff[nn];
  if (i == 0) *ntiles = (uint32_t)total;
  if (i >= total || i >= max_tiles) return;
  uint64_t lo = 0, hi = nn - 1;
  while (lo < hi) {
    const uint64_t mid = (lo + hi + 1) >> 1;
    if (toff[mid] <= i) lo = mid;
    else hi = mid - 1;
  }
  const uint64_t p = lo, k = i - toff[p];
  const uint64_t s = bnd[p] + k * T, e = bnd[p + 1];
  TileDesc d;
  d.start = s;
  d.count = (uint32_t)std::min<uint64_t>(T, e - s);
  d.node = (uint32_t)(node_base + p);
  d.seg0 = (uint32_t)toff[p];
  tiles[i] = d;
}

// The node-aligned tiles of a pass: node p of nn spans [bnd[p], bnd[p+1]).
static wt_status launch_node_tiles(const uint64_t* bnd, uint64_t nn, uint32_t T, uint64_t node_base,
                                   uint64_t mt, uint64_t* tcnt, uint64_t* toff, uint64_t* scr,
                                   TileDesc* tiles, uint32_t* d_ntiles, cudaStream_t st) {
  if (nn <= 4096) {
    k_tiles_offsets<<<1, 1024, 0, st>>>(bnd, (uint32_t)nn, T, toff);
    count_launch();
  } else {
    k_tiles_count<<<(unsigned)((nn + 255) / 256), 256, 0, st>>>(bnd, nn, T, tcnt);
    count_launch();
    TRY(scan_excl_u64(tcnt, toff, nn, scr, st));
  }
  k_tiles_write<<<(unsigned)((mt + 255) / 256), 256, 0, st>>>(bnd, nn, T, node_base, toff, tiles,
                                                             d_ntiles, mt);
  count_launch();
  CK(cudaGetLastError());
  return WT_OK;
}

// ---------------------------------------------------------------------------
// 3. pass launch
// ---------------------------------------------------------------------------
constexpr int PT = PASS_T;

// Prefix sums of the tiles' counts, per key: exclusive inside each chunk of
// 2^chsh tiles (in place, u32), and the chunks' totals, a block per chunk.
// (2^18 tiles: 11 us; 50 with a thread per chunk and key, too few loads in
// flight.)
__global__ void __launch_bounds__(256) k_tile_scan_chunk(uint32_t* tcnt, const uint32_t* ntiles_dev,
                                                         uint32_t ntiles_host, uint32_t chsh,
                                                         uint64_t* tchunk) {
  scan_chunk(tcnt, ntiles_dev ? *ntiles_dev : ntiles_host, blockIdx.x, chsh, tchunk);
}

// The whole scan and the pass's plan where there is one chunk: its totals are
// the grand totals (row 1), row 0 is zero.  One warp.
__global__ void __launch_bounds__(32) k_tile_scan_one(uint32_t* tcnt, const uint32_t* ntiles_dev,
                                                      uint32_t ntiles_host, uint64_t* tchunk,
                                                      const PassPlan plan) {
  constexpr int S = TC_STRIDE;
  const uint32_t nt = ntiles_dev ? *ntiles_dev : ntiles_host, r = threadIdx.x % S;
  uint32_t run = 0;
  if (threadIdx.x < S) {
    // sixteen loads in flight before their stores (in place: the stores would
    // otherwise wait for each load in turn)
    constexpr int B = 16;
    for (uint32_t ti = 0; ti < nt; ti += B) {
      uint32_t v[B];
#pragma unroll
      for (int k = 0; k < B; k++) v[k] = ti + k < nt ? tcnt[(uint64_t)(ti + k) * S + r] : 0u;
#pragma unroll
      for (int k = 0; k < B; k++) {
        if (ti + k < nt) tcnt[(uint64_t)(ti + k) * S + r] = run;
        run += v[k];
      }
    }
    tchunk[r] = 0;
    tchunk[S + r] = run;
  }
  __syncwarp();
  if (plan.kind != PLAN_NONE) plan_pass(run, plan);
}

// ... and the exclusive prefix of the chunks' totals (u64), with the grand
// total after the last chunk, and the pass's plan from it: a cluster of blocks,
// 64 runs of chunks side by side in each, whose sums are known before they are
// scanned.  (4096 chunks 8 us, 16384 chunks 14; one block, whose loads in flight
// bound it, 19 and 62.)
constexpr int TOP_CLUSTER = 8;
__global__ void __cluster_dims__(TOP_CLUSTER, 1, 1) __launch_bounds__(1024)
    k_tile_scan_top(uint64_t* tchunk, uint32_t nchunk, const PassPlan plan) {
  namespace cg = cooperative_groups;
  constexpr int S = TC_STRIDE, RUN = 1024 / S;
  __shared__ uint64_t sums[RUN][S];
  __shared__ uint64_t total[S];  // the block's
  const uint32_t rank = cg::this_cluster().block_rank();
  const uint32_t r = threadIdx.x % S, w = threadIdx.x / S;
  const uint32_t per = (nchunk + RUN * TOP_CLUSTER - 1) / (RUN * TOP_CLUSTER);
  const uint32_t c0 = min((rank * RUN + w) * per, nchunk), c1 = min(c0 + per, nchunk);
  constexpr int B = 8;
  uint64_t sum = 0;
  for (uint32_t c = c0; c < c1; c += B) {
    uint64_t v[B];
#pragma unroll
    for (int k = 0; k < B; k++) v[k] = c + k < c1 ? tchunk[(uint64_t)(c + k) * S + r] : 0ull;
#pragma unroll
    for (int k = 0; k < B; k++) sum += v[k];
  }
  sums[w][r] = sum;
  __syncthreads();
  uint64_t run = 0;
#pragma unroll 8
  for (uint32_t k = 0; k < w; k++) run += sums[k][r];
  if (w == RUN - 1) total[r] = run + sum;
  cg::this_cluster().sync();
  uint64_t all = 0;
#pragma unroll
  for (uint32_t q = 0; q < TOP_CLUSTER; q++) {
    const uint64_t x = cg::this_cluster().map_shared_rank(total, q)[r];
    all += x;
    run += q < rank ? x : 0ull;
  }
  cg::this_cluster().sync();  // the totals are read before a block ends
  for (uint32_t c = c0; c < c1; c += B) {
    uint64_t v[B];
#pragma unroll
    for (int k = 0; k < B; k++) v[k] = c + k < c1 ? tchunk[(uint64_t)(c + k) * S + r] : 0ull;
#pragma unroll
    for (int k = 0; k < B; k++) {
      if (c + k < c1) tchunk[(uint64_t)(c + k) * S + r] = run;
      run += v[k];
    }
  }
  if (rank) return;
  if (w == 0) tchunk[(uint64_t)nchunk * S + r] = all;
  if (threadIdx.x < 32 && plan.kind != PLAN_NONE) plan_pass(threadIdx.x < S ? all : 0ull, plan);
}

template <int EW, bool DIG, bool BATCH, int NT>
static wt_status launch_pass_t(const PassParams& Q, uint64_t mt, const wt_build_opts* o,
                               cudaStream_t st) {
  using E = typename std::conditional<EW == 1, uint8_t,
                                      typename std::conditional<EW == 2, uint16_t, uint32_t>::type>::type;
  using SM = PassSmem<EW, NT>;
  auto kern = k_pass<E, DIG, BATCH, NT>;
  static bool attr = false;
  static int occ = 0;
  if (!attr) {
    CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM::bytes));
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, NT, SM::bytes));
    if (occ < 1) occ = 1;
    attr = true;
  }
  int per_sm = occ;
  if (o && o->ctas_per_sm) per_sm = std::min<int>(occ, (int)o->ctas_per_sm);
  const uint64_t grid = std::min<uint64_t>((uint64_t)num_sms() * per_sm, std::max<uint64_t>(mt, 1));
  Prof& pf = prof();
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (pf.on) {
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, st);
  }
  kern<<<(unsigned)grid, NT, SM::bytes, st>>>(Q);
  CK(cudaGetLastError());
  count_launch();
  if (pf.on) {
    cudaEventRecord(e1, st);
    std::lock_guard<std::mutex> g(pf.mu);
    pf.ev.push_back(e0);
    pf.ev.push_back(e1);
    pf.pass_launches++;
  }
  return WT_OK;
}

// Nodes of a tree pass after the first, planned from its own tiles' counts.
struct NodePlan {
  const uint64_t* Ca = nullptr;  // starts of the nodes of level a
  const uint64_t* toff = nullptr;
  uint64_t nn = 0;
  uint64_t* C = nullptr;  // starts of the nodes of level a + t
};

// Count tables of the passes of a build with at most mt tiles each.
struct PassTables {
  uint32_t* tcnt = nullptr;
  uint64_t* tchunk = nullptr;
  void want(Work& wk, uint64_t mt) {
    mt = std::max<uint64_t>(mt, 1);
    wk.want(&tcnt, mt * TC_STRIDE);
    wk.want(&tchunk, (std::min<uint64_t>((mt + 63) / 64, MAX_CHUNKS) + 1) * TC_STRIDE);
  }
};

// One pass over at most mt tiles: every tile's digit counts, their prefix
// sums across the tiles, what is planned from their totals, and the pass.
template <bool BATCH, typename Launch>
static wt_status run_pass(const PassParams& P, uint64_t mt, uint32_t T, const PassTables& tb,
                          const PassPlan& plan, const NodePlan& np, cudaStream_t st,
                          Launch&& launch) {
  mt = std::max<uint64_t>(mt, 1);
  PassParams Q = P;
  Q.chsh = (uint32_t)chunk_shift(mt);
  const uint32_t nchunk = (uint32_t)((mt + (1u << Q.chsh) - 1) >> Q.chsh);
  uint32_t* const tcnt = tb.tcnt;
  uint64_t* const tchunk = tb.tchunk;
  // the zeroing belongs to the counts of a first pass (sigma set), else to
  // the pass
  if (!P.sigma) Q.clear = nullptr;
  // up to SCAN_TILES tiles one launch counts, scans and plans, else three
  const TileScan sc{P.tick, nchunk, tchunk, plan};
  const bool tail = !BATCH && P.tick && mt <= SCAN_TILES && !byte_counts(P);
  TRY(launch_counts<BATCH>(Q, T, mt, tcnt, tail ? &sc : nullptr, st));
  const uint32_t* nt_dev = P.tiles ? P.ntiles_dev : nullptr;
  if (tail) {
  } else if (nchunk == 1) {
    k_tile_scan_one<<<1, 32, 0, st>>>(tcnt, nt_dev, P.ntiles, tchunk, plan);
    count_launch();
  } else {
    k_tile_scan_chunk<<<nchunk, 256, 0, st>>>(tcnt, nt_dev, P.ntiles, Q.chsh, tchunk);
    k_tile_scan_top<<<TOP_CLUSTER, 1024, 0, st>>>(tchunk, nchunk, plan);
    count_launch(2);
  }
  if (BATCH) {
    k_plan_batch_pass<<<(P.nsegs + 7) / 8, 256, 0, st>>>(P.segs, P.nsegs, tcnt, tchunk,
                                                         (uint32_t)mt, nchunk, Q.chsh);
    count_launch();
  }
  if (np.nn) {
    k_plan_nodes<<<(unsigned)((np.nn + 7) / 8), 256, 0, st>>>(np.Ca, np.toff, np.nn, P.t, P.n_in,
                                                              tcnt, tchunk, P.ntiles_dev, nchunk,
                                                              Q.chsh, np.C);
    count_launch();
  }
  CK(cudaGetLastError());
  Q.tcnt = tcnt;
  Q.tchunk = tchunk;
  Q.clear = P.sigma ? nullptr : P.clear;
  return launch(Q, mt);
}

// tile: symbols per tile (PT for the trees; 2048, 4096 or 8192 for the
// wavelet matrix)
template <int EW>
static wt_status launch_pass_w(const PassParams& Q, bool dig, uint64_t mt, const wt_build_opts* o,
                               cudaStream_t st, uint32_t tile) {
  if (dig) return launch_pass_t<EW, true, false, PT / 32>(Q, mt, o, st);
  if (tile == 2048) return launch_pass_t<EW, false, false, 64>(Q, mt, o, st);
  if (tile == 8192) return launch_pass_t<EW, false, false, 256>(Q, mt, o, st);
  return launch_pass_t<EW, false, false, PT / 32>(Q, mt, o, st);
}
static wt_status launch_pass(const PassParams& P, bool dig, uint64_t mt, const PassTables& tb,
                             const wt_build_opts* o, cudaStream_t st,
                             const PassPlan& plan = PassPlan{},
                             const NodePlan& np = NodePlan{}, uint32_t tile = PT) {
  const int ew = P.in_w;
  return run_pass<false>(P, mt, tile, tb, plan, np, st, [&](const PassParams& Q, uint64_t m) {
    if (ew == 1) return launch_pass_w<1>(Q, dig, m, o, st, tile);
    if (ew == 2) return launch_pass_w<2>(Q, dig, m, o, st, tile);
    return launch_pass_w<4>(Q, dig, m, o, st, tile);
  });
}

// Batched wavelet matrices: one launch over the tiles of every sequence in
// P.segs (P.ntiles tiles in total), whose elements all have P.in_w bytes.
wt_status launch_pass_batch(const PassParams& P, const wt_build_opts* o, cudaStream_t st) {
  Work wk{st};
  PassTables tb;
  tb.want(wk, P.ntiles);
  TRY(wk.take());
  return run_pass<true>(P, P.ntiles, PT, tb, PassPlan{}, NodePlan{}, st,
                        [&](const PassParams& Q, uint64_t m) {
                          if (Q.in_w == 1) return launch_pass_t<1, false, true, PT / 32>(Q, m, o, st);
                          if (Q.in_w == 2) return launch_pass_t<2, false, true, PT / 32>(Q, m, o, st);
                          return launch_pass_t<4, false, true, PT / 32>(Q, m, o, st);
                        });
}

static int pick_tau(const wt_build_opts* o, int L, bool even, uint64_t n = 0) {
  int tau = (o && o->tau) ? (int)o->tau : (even ? TAU_MAX : tuned_tau((uint32_t)L, n));
  if (tau < 1) tau = 1;
  if (tau > TAU_MAX) tau = TAU_MAX;
  if (even && (tau & 1)) tau = tau > 1 ? tau - 1 : 2;
  return tau;
}

// zero_bits: false when the build's own kernels zero the level buffer
static wt_status alloc_outputs(wt_struct* h, uint64_t total_words, bool zero_bits = true) {
  CK(dmalloc((void**)&h->d_bits, total_words * 8, h->stream));
  h->d_bits_ro = h->d_bits;
  // the partition passes store whole words and OR the words shared by
  // several tiles or nodes, so the level buffer starts at zero
  if (zero_bits) CK(cudaMemsetAsync(h->d_bits, 0, total_words * 8, h->stream));
  return WT_OK;
}

static void set_uniform_levels(wt_struct* h, uint64_t elems_per_level) {
  h->level_len.assign(h->levels, elems_per_level);
  h->level_off.assign(h->levels + 1, 0);
  for (uint32_t l = 0; l < h->levels; l++)
    h->level_off[l + 1] = h->level_off[l] + level_words(elems_per_level * h->bpe);
}

static PassParams base_params(wt_struct* h) {
  PassParams P;
  memset(&P, 0, sizeof(P));
  P.bits = h->d_bits;
  P.err = h->d_err;
  P.tick = h->d_tick;
  return P;
}

// Host tables reach the device without a copy engine: a host-to-device copy
// would queue behind whatever large copy the caller has in flight (the next
// input, in a pipelined loop) and stall the build.  Tables up to 32 KB go as
// kernel parameters.
constexpr size_t UPLOAD_MAX = 3968, UPLOAD_BIG = 32000;
struct UploadBlock {
  uint8_t b[UPLOAD_MAX];
};
struct UploadBigBlock {
  uint8_t b[UPLOAD_BIG];
};

__global__ void k_upload(uint8_t* dst, const __grid_constant__ UploadBlock blk, uint32_t bytes) {
  for (uint32_t i = threadIdx.x; i < bytes; i += blockDim.x) dst[i] = blk.b[i];
}

__global__ void k_upload_big(uint8_t* dst, const __grid_constant__ UploadBigBlock blk,
                             uint32_t bytes) {
  for (uint32_t i = threadIdx.x; i < bytes; i += blockDim.x) dst[i] = blk.b[i];
}

// Larger tables: a pinned, device-mapped staging buffer that the host fills
// and a kernel copies into device memory, reading it over the host link (no
// copy engine).  Buffers are kept per device and reused once the event
// recorded after their copy kernel has completed.
struct Stage {
  uint8_t* p = nullptr;
  size_t bytes = 0;
  cudaEvent_t ev = nullptr;
};
constexpr size_t STAGE_MIN = 8u << 20;

__global__ void k_gather_host(uint8_t* dst, const uint8_t* src, size_t bytes) {
  const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  if ((((uintptr_t)dst | (uintptr_t)src) & 15) == 0) {
    const size_t nv = bytes / 16;
    for (size_t i = i0; i < nv; i += stride) ((uint4*)dst)[i] = ((const uint4*)src)[i];
    for (size_t i = nv * 16 + i0; i < bytes; i += stride) dst[i] = src[i];
  } else {
    for (size_t i = i0; i < bytes; i += stride) dst[i] = src[i];
  }
}

static wt_status upload_staged(void* d_dst, const void* h_src, size_t bytes, cudaStream_t st) {
  static std::mutex mu;
  static std::vector<Stage> stages[64];
  int dev = 0;
  CK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return WT_ERR_CUDA;
  std::lock_guard<std::mutex> g(mu);
  std::vector<Stage>& v = stages[dev];
  Stage* s = nullptr;
  for (Stage& x : v)
    if (x.bytes >= bytes && cudaEventQuery(x.ev) == cudaSuccess) {
      s = &x;
      break;
    }
  // a busy buffer answers cudaErrorNotReady: a status, not an error to keep
  if (cudaPeekAtLastError() == cudaErrorNotReady) cudaGetLastError();
  if (!s) {
    Stage n;
    n.bytes = std::max(bytes, STAGE_MIN);
    CK(cudaHostAlloc((void**)&n.p, n.bytes, cudaHostAllocMapped | cudaHostAllocPortable));
    if (cudaEventCreateWithFlags(&n.ev, cudaEventDisableTiming) != cudaSuccess) {
      cudaFreeHost(n.p);
      return WT_ERR_CUDA;
    }
    v.push_back(n);
    s = &v.back();
  }
  memcpy(s->p, h_src, bytes);
  const unsigned grid = (unsigned)std::min<size_t>((bytes / 16 + 255) / 256 + 1, 4 * (size_t)num_sms());
  k_gather_host<<<grid, 256, 0, st>>>((uint8_t*)d_dst, s->p, bytes);
  count_launch();
  CK(cudaGetLastError());
  CK(cudaEventRecord(s->ev, st));
  return WT_OK;
}

wt_status upload(void* d_dst, const void* h_src, size_t bytes, cudaStream_t st) {
  if (bytes == 0) return WT_OK;
  if (bytes > UPLOAD_BIG) return upload_staged(d_dst, h_src, bytes, st);
  if (bytes <= UPLOAD_MAX) {
    UploadBlock blk;
    memcpy(blk.b, h_src, bytes);
    k_upload<<<1, 256, 0, st>>>((uint8_t*)d_dst, blk, (uint32_t)bytes);
    count_launch();
    CK(cudaGetLastError());
    return WT_OK;
  }
  static thread_local UploadBigBlock big;
  memcpy(big.b, h_src, bytes);
  k_upload_big<<<1, 1024, 0, st>>>((uint8_t*)d_dst, big, (uint32_t)bytes);
  count_launch();
  CK(cudaGetLastError());
  return WT_OK;
}

// An alphabet can be larger than the sequence's elements can hold; the passes
// read a digit's bits inside the element, so such a sequence is widened first
// (reading zeros past the element's end in the pass itself cost every build 1%).
__global__ void __launch_bounds__(256) k_widen(const void* in, int w, void* out, int ow, uint64_t n) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t x = load_elem(in, w, i);
    if (ow == 2) ((uint16_t*)out)[i] = (uint16_t)x;
    else ((uint32_t*)out)[i] = x;
  }
}

// bytes per element the passes need for L levels
int pass_width(int w, int L) { return L > 8 * w ? width_for_bits(L) : w; }

wt_status widen(const void* d_in, int w, void* d_out, int ow, uint64_t n, cudaStream_t st) {
  const unsigned grid = (unsigned)std::min<uint64_t>((n + 255) / 256, (uint64_t)num_sms() * 16);
  k_widen<<<grid, 256, 0, st>>>(d_in, w, d_out, ow, n);
  count_launch();
  CK(cudaGetLastError());
  return WT_OK;
}

// the sequence as the passes read it
static wt_status widened(const void** d_seq, int* w, int L, uint64_t n, Work& wk) {
  const int ow = pass_width(*w, L);
  if (ow == *w) return WT_OK;
  uint8_t* wide;
  TRY(wk.get(&wide, (size_t)n * ow));
  TRY(widen(*d_seq, *w, wide, ow, n, wk.st));
  *d_seq = wide;
  *w = ow;
  return WT_OK;
}

// ---------------------------------------------------------------------------
// wavelet matrix
// ---------------------------------------------------------------------------
wt_status build_wm(const void* d_seq, uint64_t n, uint32_t sigma, int w, const wt_build_opts* o,
                   wt_struct* h) {
  cudaStream_t st = h->stream;
  const int L = (int)levels_of(sigma);
  h->kind = WT_KIND_WM;
  h->L = h->levels = (uint32_t)L;
  h->bpe = 1;
  set_uniform_levels(h, n);
  const uint64_t W = level_words(n);
  // the level buffer is zeroed by the build's kernels (the first pass's counts
  // the levels of two passes, each later pass the next one's), not by a memset
  TRY(alloc_outputs(h, W * L, n == 0));
  Work wk{st};
  if (n == 0) return build_directories(h);
  TRY(widened(&d_seq, &w, L, n, wk));
  // levels per pass, symbols per tile and CTAs per SM: the caller's, else
  // the autotuner's for (L, ceil(log2 n)), else 4 / 4096 / the occupancy limit
  const TuneConfig tc = tuned_config((uint32_t)L, n);
  wt_build_opts eo = o ? *o : wt_build_opts{};
  if (!eo.tau) eo.tau = (uint32_t)tc.tau;
  if (!eo.tile_symbols) eo.tile_symbols = tc.tile;
  if (!eo.ctas_per_sm) eo.ctas_per_sm = tc.ctas;
  o = &eo;
  const int tau = pick_tau(o, L, false, n);
  std::vector<PassGeom> ps = make_passes(L, tau, w);
  const int G = (int)ps.size();
  const uint32_t T = o->tile_symbols;
  uint64_t* cls;
  int ncls = 0;
  for (auto& p : ps) ncls += (2 << p.t) + p.t + 1;
  const uint64_t ntiles = (n + T - 1) / T;
  PassTables tb;
  uint8_t* seqbuf[2] = {nullptr, nullptr};  // intermediate sequences
  wk.want(&cls, ncls);
  tb.want(wk, ntiles);
  want_seqbufs(wk, seqbuf, ps, [&](int) { return n; });
  TRY(wk.take());
  const void* in = d_seq;
  int coff = 0;
  for (int g = 0; g < G; g++) {
    const PassGeom& pg = ps[g];
    PassParams P = base_params(h);
    P.in = in;
    P.in_w = pg.in_w;
    P.out = (g + 1 < G) ? seqbuf[g & 1] : nullptr;
    P.out_w = pg.out_w;
    P.L = L;
    P.a = pg.a;
    P.t = pg.t;
    P.rbits = pg.rbits;
    P.shape = SHAPE_WM;
    P.wm_cls = cls + coff;
    P.ntiles = (uint32_t)ntiles;
    P.n_in = n;
    // the first pass's counts check the symbols and zero the levels of the
    // first two passes, every later pass zeroes the next pass's
    const int z0 = g == 0 ? 0 : (g + 1 < G ? ps[g + 1].a : L);
    const int z1 = g == 0 ? (G > 1 ? ps[1].a + ps[1].t : L) : (g + 1 < G ? z0 + ps[g + 1].t : L);
    if (g == 0) P.sigma = sigma;
    if (z1 > z0) {
      P.clear = (uint4*)(h->d_bits + W * (uint64_t)z0);
      P.clear_units = W * (uint64_t)(z1 - z0) / 2;
      P.clear_per = (P.clear_units + ntiles - 1) / ntiles;
    }
    // every pass is planned from its own tiles' digit counts
    const PassPlan plan{PLAN_WM, pg.a, pg.t, cls + coff, nullptr, h->d_zeros};
    TRY(launch_pass(P, false, ntiles, tb, o, st, plan, NodePlan{}, T));
    coff += (2 << pg.t) + pg.t + 1;
    in = P.out;
  }
  if (o && (o->flags & WT_FLAG_NO_DIRECTORY)) return WT_OK;
  return build_directories(h);
}

// ---------------------------------------------------------------------------
// balanced wavelet tree and its 4-ary variant
// ---------------------------------------------------------------------------
wt_status build_wt(const void* d_seq, uint64_t n, uint32_t sigma, int w, const wt_build_opts* o,
                   wt_struct* h, bool multiary) {
  cudaStream_t st = h->stream;
  const int L = (int)levels_of(sigma);
  if (L > 24) return WT_ERR_UNSUPPORTED;
  h->kind = multiary ? WT_KIND_MULTI : WT_KIND_WT;
  h->L = (uint32_t)L;
  h->levels = multiary ? (uint32_t)((L + 1) / 2) : (uint32_t)L;
  h->bpe = multiary ? 2 : 1;
  set_uniform_levels(h, n);
  const int tau = pick_tau(o, L, multiary);
  std::vector<PassGeom> ps = make_passes(L, tau, pass_width(w, L));
  const int G = (int)ps.size();
  // a tree of one pass has its level buffer zeroed by the counting kernel
  const bool one = G == 1;
  TRY(alloc_outputs(h, h->level_off.back(), !one || n == 0));
  Work wk{st};
  if (n == 0) return build_directories(h);
  TRY(widened(&d_seq, &w, L, n, wk));
  const uint32_t T = PT;
  const uint64_t ntiles0 = (n + T - 1) / T;
  uint64_t *scr = nullptr, *tcnt = nullptr, *toff = nullptr;
  uint32_t* d_ntiles = nullptr;
  TileDesc* tiles = nullptr;
  PassTables tb;
  uint8_t* seqbuf[2] = {nullptr, nullptr};
  std::vector<uint64_t*> Cs(G, nullptr);
  const uint64_t max_nodes = (uint64_t)1 << ps.back().a;
  for (int g = 0; g < G; g++) wk.want(&Cs[g], ((uint64_t)1 << (ps[g].a + ps[g].t)) + 1);
  tb.want(wk, ntiles0 + (one ? 0 : max_nodes));
  if (!one) {
    wk.want(&scr, scan_scratch(max_nodes));
    wk.want(&tcnt, max_nodes);
    wk.want(&toff, max_nodes + 1);
    wk.want(&tiles, ntiles0 + max_nodes + 1);
    wk.want(&d_ntiles, 1);
  }
  want_seqbufs(wk, seqbuf, ps, [&](int) { return n; });
  TRY(wk.take());
  // Every pass is planned from its own tiles' digit counts (no histogram of
  // the symbols): C holds the starts of the nodes of level a, and the totals
  // of each node's tiles give those of level a + t.
  uint64_t* C = nullptr;
  const void* in = d_seq;
  for (int g = 0; g < G; g++) {
    const PassGeom& pg = ps[g];
    PassParams P = base_params(h);
    const uint64_t nn = (uint64_t)1 << pg.a;
    uint64_t* const Cn = Cs[g];
    uint64_t mt = ntiles0;
    NodePlan np;
    if (g > 0) {
      // tiles inside the nodes of the pass's first level (the first pass has
      // one node, the whole sequence)
      mt = ntiles0 + nn;
      TRY(launch_node_tiles(C, nn, T, 0, mt, tcnt, toff, scr, tiles, d_ntiles, st));
      P.tiles = tiles;
      P.ntiles_dev = d_ntiles;
      np.Ca = C;
      np.toff = toff;
      np.nn = nn;
      np.C = Cn;
    } else {
      P.sigma = sigma;
      if (one) {
        P.clear = (uint4*)h->d_bits;
        P.clear_units = h->level_off.back() / 2;
        P.clear_per = (P.clear_units + ntiles0 - 1) / ntiles0;
      }
    }
    P.in = in;
    P.in_w = pg.in_w;
    P.out = (g + 1 < G) ? seqbuf[g & 1] : nullptr;
    P.out_w = pg.out_w;
    P.L = L;
    P.a = pg.a;
    P.t = pg.t;
    P.rbits = pg.rbits;
    P.shape = SHAPE_WT;
    P.wt_C = Cn;
    P.ntiles = (uint32_t)ntiles0;
    P.n_in = n;
    const PassPlan plan{g == 0 ? PLAN_WT : PLAN_NONE, 0, pg.t, nullptr, Cn, nullptr};
    TRY(launch_pass(P, multiary, mt, tb, o, st, plan, np));
    in = P.out;
    C = Cn;
  }
  if (!multiary) {
    k_wt_zeros<<<L, 1024, 0, st>>>(C, L, h->d_zeros);
    count_launch();
    CK(cudaGetLastError());
  }
  if (o && (o->flags & WT_FLAG_NO_DIRECTORY)) return WT_OK;
  return build_directories(h);
}

// ---------------------------------------------------------------------------
// Huffman-shaped wavelet tree
// ---------------------------------------------------------------------------
// The symbols' left-aligned codewords, four bytes each, which every pass then
// reads as elements (mapping the symbols in the first pass's counts and again
// in the pass itself took two gathers per symbol through their slowest
// loads).  in == out for 4-byte symbols; both 16-byte aligned.
template <int W>
__global__ void __launch_bounds__(256) k_map_codes(const void* in, uint64_t n, const uint32_t* map,
                                                   uint32_t* out) {
  const uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x, nv = n / 4;
  for (uint64_t i = i0; i < nv; i += stride) {
    uint32_t x[4];
    if (W == 4) {
      const uint4 q = ((const uint4*)in)[i];
      x[0] = q.x;
      x[1] = q.y;
      x[2] = q.z;
      x[3] = q.w;
    } else if (W == 2) {
      const uint2 q = ((const uint2*)in)[i];
      x[0] = q.x & 0xffffu;
      x[1] = q.x >> 16;
      x[2] = q.y & 0xffffu;
      x[3] = q.y >> 16;
    } else {
      const uint32_t q = ((const uint32_t*)in)[i];
#pragma unroll
      for (int k = 0; k < 4; k++) x[k] = (q >> (8 * k)) & 0xffu;
    }
    ((uint4*)out)[i] = make_uint4(map[x[0]], map[x[1]], map[x[2]], map[x[3]]);
  }
  for (uint64_t i = nv * 4 + i0; i < n; i += stride) out[i] = map[load_elem(in, W, i)];
}

uint32_t huffman_lengths(const uint64_t* hist, uint32_t sigma, uint32_t cap, uint8_t* len);
void canonical_codes(const uint8_t* len, uint32_t sigma, uint32_t* code);

// The code tables from the symbol counts (or the caller's lengths), on the
// host: codes, node table, zero counts, level lengths.
static wt_status huff_tables_host(const uint64_t* hist, uint32_t sigma, const uint8_t* h_len,
                                  wt_struct* h, uint32_t* d_left, std::vector<uint64_t>& node_lvl) {
  cudaStream_t st = h->stream;
  std::vector<uint64_t> hh(sigma);
  uint32_t err = 0;
  CK(cudaMemcpyAsync(hh.data(), hist, (size_t)sigma * 8, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(&err, h->d_err, 4, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  if (err & ERR_SYMBOL) return WT_ERR_SYMBOL_GE_SIGMA;
  h->code_len.assign(sigma, 0);
  h->code.assign(sigma, 0);
  uint32_t maxlen = 0;
  if (h_len) {
    // caller lengths: every present symbol needs a code, Kraft sum <= 1
    double kraft = 0;
    uint32_t present = 0;
    for (uint32_t s = 0; s < sigma; s++) {
      h->code_len[s] = h_len[s];
      if (h_len[s] > 32) return WT_ERR_INVALID_ARG;
      if (hh[s] && !h_len[s]) return WT_ERR_INVALID_ARG;
      if (h_len[s]) {
        kraft += std::ldexp(1.0, -(int)h_len[s]);
        maxlen = std::max<uint32_t>(maxlen, h_len[s]);
        present++;
      }
    }
    if (kraft > 1.0 + 1e-12) return WT_ERR_INVALID_ARG;
    (void)present;
  } else {
    maxlen = huffman_lengths(hh.data(), sigma, 32, h->code_len.data());
  }
  h->max_code_len = maxlen;
  const int Lm = (int)maxlen;
  h->L = h->levels = (uint32_t)Lm;
  // The sweeps below run on up to 16 host threads, each over a contiguous
  // chunk of symbols (or of `order`), with per-thread partial results
  // combined in a fixed order, so the result does not depend on the thread
  // count.
  const uint32_t hw = std::max(1u, std::thread::hardware_concurrency());
  auto par = [&](uint64_t items, auto&& f) {
    const int nt = (int)std::max<uint64_t>(1, std::min<uint64_t>({16, hw, items / 65536 + 1}));
    std::vector<std::thread> th;
    for (int t = 1; t < nt; t++) th.emplace_back(f, t, nt);
    f(0, nt);
    for (auto& x : th) x.join();
    return nt;
  };
  auto chunk = [](uint64_t items, int t, int nt, uint64_t& b, uint64_t& e) {
    b = items * (uint64_t)t / (uint64_t)nt;
    e = items * (uint64_t)(t + 1) / (uint64_t)nt;
  };
  constexpr int MAXT = 16;
  // symbols in canonical order (= order of the left-aligned codewords):
  // by (length, symbol), a counting sort on the length, stable across the
  // threads' symbol ranges
  std::vector<uint32_t> order;
  uint64_t lcount[34] = {0};
  uint64_t lpos[34] = {0};  // first index in `order` of each length
  {
    uint64_t tc[MAXT][34] = {};
    const int nt = par(sigma, [&](int t, int n_t) {
      uint64_t b, e;
      chunk(sigma, t, n_t, b, e);
      for (uint64_t s = b; s < e; s++) tc[t][h->code_len[s]]++;
    });
    for (int t = 0; t < nt; t++)
      for (int ln = 0; ln <= 33; ln++) lcount[ln] += tc[t][ln];
    for (int ln = 2; ln <= 33; ln++) lpos[ln] = lpos[ln - 1] + (ln - 1 >= 1 ? lcount[ln - 1] : 0);
    // each thread's first slot per length: after the earlier threads'
    uint64_t at[MAXT][34];
    for (int ln = 1; ln <= 33; ln++) {
      uint64_t p0 = lpos[ln];
      for (int t = 0; t < nt; t++) {
        at[t][ln] = p0;
        p0 += tc[t][ln];
      }
    }
    order.resize(lpos[33]);
    par(sigma, [&](int t, int n_t) {
      uint64_t b, e;
      chunk(sigma, t, n_t, b, e);
      uint64_t* w = at[t];
      for (uint64_t s = b; s < e; s++)
        if (h->code_len[s]) order[w[h->code_len[s]]++] = (uint32_t)s;
    });
  }
  // level sizes, internal nodes of every level and their start positions,
  // and zero counts.  `order` is sorted by length, so the elements still on
  // level l (length > l) are a suffix of it, starting at first_gt[l]; their
  // l-bit prefixes (top bits of the left-aligned codewords) never decrease
  // along it and, the codes being canonical, grow by at most one from one
  // symbol to the next (the next codeword adds 2^(Lm - len) to the left-
  // aligned value, len > l).  So symbol i opens a node on level l exactly
  // when l < len(i) and l exceeds the common prefix of codewords i-1 and i
  // (every level below len(0) for i = 0); that node's index on level l is
  // its prefix minus the level's first one, and it starts at the elements
  // before i on that level: S[i] - S[first_gt[l]], S = prefix sums of the
  // symbol counts along `order`.
  const size_t np = order.size();
  const int Lw = std::max(Lm, 1);
  // canonical codes: consecutive values within a length, the first of each
  // length the last of the previous length plus one, shifted left
  uint64_t fcode[34] = {0};
  {
    uint64_t c = 0;
    int prev = 0;
    for (int ln = 1; ln <= 33; ln++) {
      if (!lcount[ln]) continue;
      if (prev) c = (c + lcount[prev]) << (ln - prev);
      fcode[ln] = c;
      prev = ln;
    }
  }
  auto lcode = [&](uint64_t i, int& ln_i) -> uint64_t {  // left-aligned code of order[i]
    ln_i = h->code_len[order[i]];
    return (fcode[ln_i] + (i - lpos[ln_i])) << (Lm - ln_i);
  };
  auto first_open = [&](uint64_t i, uint64_t lci) -> int {  // first level symbol i opens a node on
    if (i == 0) return 0;
    int lp;
    const uint64_t prev = lcode(i - 1, lp);
    return __builtin_clzll((prev ^ lci) << (64 - Lm)) + 1;
  };
  std::vector<uint64_t> S(np + 1, 0);
  std::vector<uint64_t> nn(Lw, 0);
  {
    // chunk sums of the counts, then the prefix sums, the codes and the
    // nodes opened per level
    uint64_t csum[MAXT + 1] = {0};
    uint64_t topen[MAXT][33] = {};
    const int nt = par(np, [&](int t, int n_t) {
      uint64_t b, e, acc = 0;
      chunk(np, t, n_t, b, e);
      for (uint64_t i = b; i < e; i++) acc += hh[order[i]];
      csum[t + 1] = acc;
    });
    for (int t = 0; t < nt; t++) csum[t + 1] += csum[t];
    par(np, [&](int t, int n_t) {
      uint64_t b, e;
      chunk(np, t, n_t, b, e);
      uint64_t acc = csum[t];
      for (uint64_t i = b; i < e; i++) {
        const uint32_t sy = order[i];
        int ln_i;
        const uint64_t lci = lcode(i, ln_i);
        h->code[sy] = (uint32_t)(lci >> (Lm - ln_i));
        S[i] = acc;
        acc += hh[sy];
        for (int l = first_open(i, lci); l < ln_i; l++) topen[t][l]++;
      }
      if (t + 1 == n_t) S[np] = acc;
    });
    for (int t = 0; t < nt; t++)
      for (int l = 0; l < Lm; l++) nn[l] += topen[t][l];
  }
  std::vector<uint64_t> first_gt(Lw + 1, np);
  {
    uint64_t acc = 0;
    for (int l = 0; l <= Lw; l++) {
      first_gt[l] = acc;  // symbols with length <= l come first
      if (l + 1 <= 33) acc += lcount[std::min(l + 1, 33)];
    }
    for (int l = 0; l <= Lw; l++) first_gt[l] = std::min<uint64_t>(first_gt[l], np);
  }
  h->level_len.assign(Lm, 0);
  node_lvl.assign(3 * (size_t)Lw, 0);
  std::vector<uint64_t> zc(Lw, 0);
  std::vector<uint64_t> node;
  {
    uint64_t tot = 0;
    for (int l = 0; l < Lm; l++) {
      int lf;
      node_lvl[3 * l] = tot;
      node_lvl[3 * l + 1] = first_gt[l] < np ? lcode(first_gt[l], lf) >> (Lm - l) : 0;
      node_lvl[3 * l + 2] = nn[l];
      tot += nn[l] + 1;  // with the sentinel
      h->level_len[l] = S[np] - S[first_gt[l]];
    }
    node.resize(tot);
  }
  // node starts at their indices, the ones of every level (the counts of the
  // symbols whose code bit l is 1), and the left-aligned codes the first
  // pass maps the symbols to
  std::vector<uint32_t> left(sigma, 0u);
  std::vector<uint64_t> ones(Lw, 0);
  {
    uint64_t tones[MAXT][33] = {};
    int tbad[MAXT] = {0};
    const int nt = par(np, [&](int t, int n_t) {
      uint64_t b, e;
      chunk(np, t, n_t, b, e);
      for (uint64_t i = b; i < e; i++) {
        const uint32_t sy = order[i];
        int ln_i;
        const uint64_t lci = lcode(i, ln_i);
        left[sy] = (uint32_t)lci;
        const uint64_t w = hh[sy];
        for (int l = first_open(i, lci); l < ln_i; l++) {
          const uint64_t k = (lci >> (Lm - l)) - node_lvl[3 * l + 1];
          if (k >= nn[l]) {  // never for a prefix code
            tbad[t] = 1;
            continue;
          }
          node[node_lvl[3 * l] + k] = S[i] - S[first_gt[l]];
        }
        for (int l = 0; l < ln_i; l++)
          if ((lci >> (Lm - 1 - l)) & 1u) tones[t][l] += w;
      }
    });
    for (int t = 0; t < nt; t++) {
      if (tbad[t]) return WT_ERR_INVALID_ARG;  // not a prefix code
      for (int l = 0; l < Lm; l++) ones[l] += tones[t][l];
    }
  }
  for (int l = 0; l < Lm; l++) {
    zc[l] = h->level_len[l] - ones[l];
    node[node_lvl[3 * l] + nn[l]] = h->level_len[l];  // sentinel = level length
  }
  // zero counts per level: elements whose code bit l is 0
  h->zeros.assign(zc.begin(), zc.begin() + Lm);
  if (Lm) CK(cudaMemcpyAsync(h->d_zeros, h->zeros.data(), Lm * 8, cudaMemcpyHostToDevice, st));
  h->zeros_valid = true;
  // device tables
  // per length: first canonical code, its index in `order`, symbol count
  std::vector<uint64_t> lentab(3 * 34, 0);
  {
    uint64_t idx = 0;
    for (uint32_t ln = 1; ln <= 32; ln++) {
      lentab[34 + ln] = idx;
      lentab[68 + ln] = lcount[ln];
      if (lcount[ln]) lentab[ln] = h->code[order[idx]];
      idx += lcount[ln];
    }
  }
  CK(dmalloc((void**)&h->d_code, (size_t)sigma * 4, st));
  CK(dmalloc((void**)&h->d_len, sigma, st));
  CK(dmalloc((void**)&h->d_sym_by_rank, std::max<size_t>(order.size(), 1) * 4, st));
  CK(dmalloc((void**)&h->d_len_tab, lentab.size() * 8, st));
  CK(dmalloc((void**)&h->d_node, std::max<size_t>(node.size(), 1) * 8, st));
  CK(dmalloc((void**)&h->d_node_lvl, node_lvl.size() * 8, st));
  CK(cudaMemcpyAsync(h->d_code, h->code.data(), (size_t)sigma * 4, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(h->d_len, h->code_len.data(), sigma, cudaMemcpyHostToDevice, st));
  if (!order.empty())
    CK(cudaMemcpyAsync(h->d_sym_by_rank, order.data(), order.size() * 4, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(h->d_len_tab, lentab.data(), lentab.size() * 8, cudaMemcpyHostToDevice, st));
  if (!node.empty())
    CK(cudaMemcpyAsync(h->d_node, node.data(), node.size() * 8, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(h->d_node_lvl, node_lvl.data(), node_lvl.size() * 8, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(d_left, left.data(), (size_t)sigma * 4, cudaMemcpyHostToDevice, st));
  CK(cudaStreamSynchronize(st));  // host vectors above are pageable and local
  return WT_OK;
}

wt_status huff_tables_device(const uint64_t* hist, uint64_t n, uint32_t sigma, wt_struct* h,
                             uint32_t* d_left, std::vector<uint64_t>& node_lvl, bool* done);

// Alphabets from which the code is built on the device.  Whole trees over 2^16
// symbols, with the code built here and on the host: 2^16 elements 0.92 and 1.53
// ms, 2^22 1.13 and 3.55, 2^28 4.9 and 7.5.  Below some tens of thousands of
// symbols the device's launches outweigh the host's work (2^16 elements over
// 4000: 0.57 ms with the host's code).
constexpr uint32_t HUFF_DEVICE_MIN = 1u << 16;

// Copies of h->d_len and h->d_code into the handle's host vectors, ordered after
// what is on its stream at begin(), made by finish() on another stream.
struct HostCopies {
  cudaEvent_t ready = nullptr;
  cudaStream_t xs = nullptr;
  wt_status begin(wt_struct* h) {
    CK(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
    CK(cudaEventRecord(ready, h->stream));
    return WT_OK;
  }
  wt_status finish(wt_struct* h) {
    if (!ready) return WT_OK;
    CK(cudaStreamCreateWithFlags(&xs, cudaStreamNonBlocking));
    CK(cudaStreamWaitEvent(xs, ready, 0));
    h->code_len.resize(h->sigma);
    h->code.resize(h->sigma);
    CK(cudaMemcpyAsync(h->code_len.data(), h->d_len, h->sigma, cudaMemcpyDeviceToHost, xs));
    CK(cudaMemcpyAsync(h->code.data(), h->d_code, (size_t)h->sigma * 4, cudaMemcpyDeviceToHost, xs));
    CK(cudaStreamSynchronize(xs));
    return WT_OK;
  }
  ~HostCopies() {
    if (xs) cudaStreamDestroy(xs);
    if (ready) cudaEventDestroy(ready);
  }
};

// d_seq: the library's own copy of the sequence (16-byte aligned), overwritten
wt_status build_huff(void* d_seq, uint64_t n, uint32_t sigma, int w, const uint8_t* h_len,
                     const wt_build_opts* o, wt_struct* h) {
  cudaStream_t st = h->stream;
  if (sigma > (1u << 24)) return WT_ERR_UNSUPPORTED;
  h->kind = WT_KIND_HUFF;
  h->bpe = 1;
  Work wk{st};
  uint64_t* hist;
  TRY(wk.get(&hist, sigma));
  CK(cudaMemsetAsync(hist, 0, (size_t)sigma * 8, st));
  TRY(launch_hist_full(d_seq, w, n, sigma, hist, h->d_err, st));
  uint32_t* d_left;
  TRY(wk.get(&d_left, sigma));
  std::vector<uint64_t> node_lvl;
  bool dev = false;
  if (!h_len && n && n < (1ull << 32) && sigma >= HUFF_DEVICE_MIN)
    TRY(huff_tables_device(hist, n, sigma, h, d_left, node_lvl, &dev));
  if (!dev) TRY(huff_tables_host(hist, sigma, h_len, h, d_left, node_lvl));
  const int Lm = (int)h->max_code_len;
  h->level_off.assign(Lm + 1, 0);
  for (int l = 0; l < Lm; l++) h->level_off[l + 1] = h->level_off[l] + level_words(h->level_len[l]);
  TRY(alloc_outputs(h, std::max<uint64_t>(h->level_off.back(), 1)));
  // the handle's host copies of device-built codes: by a stream of their own,
  // while the passes run
  HostCopies copies;
  if (dev) TRY(copies.begin(h));
  if (n == 0 || Lm == 0) return build_directories(h);
  // the pass kernel wants hf_lvl as [off, first] pairs plus the count; use a
  // 3-wide table and read [3l], [3l+1], [3l+2]
  const int tau = pick_tau(o, Lm, false);
  std::vector<PassGeom> ps = make_passes(Lm, tau, 4);
  const int G = (int)ps.size();
  const uint32_t T = PT;
  uint64_t *d_off, *d_len, *scr, *tcnt, *toff;
  uint32_t* d_ntiles;
  TileDesc* tiles;
  uint64_t max_nodes = 1;
  for (int l = 0; l < Lm; l++) max_nodes = std::max<uint64_t>(max_nodes, node_lvl[3 * l + 2]);
  const uint64_t max_tiles = (n + T - 1) / T + max_nodes + 1;
  PassTables tb;
  uint8_t* seqbuf[2] = {nullptr, nullptr};
  uint32_t* codes = (uint32_t*)d_seq;
  uint64_t most = 0;  // tiles of a pass: by its elements and nodes
  for (const PassGeom& p : ps)
    most = std::max<uint64_t>(most, (h->level_len[p.a] + T - 1) / T + node_lvl[3 * p.a + 2]);
  wk.want(&d_off, Lm + 1);
  wk.want(&d_len, Lm);
  wk.want(&scr, scan_scratch(max_nodes));
  wk.want(&tcnt, max_nodes);
  wk.want(&toff, max_nodes + 1);
  wk.want(&tiles, max_tiles);
  wk.want(&d_ntiles, 1);
  tb.want(wk, most);
  if (w < 4) wk.want(&codes, n);
  want_seqbufs(wk, seqbuf, ps, [&](int g) { return h->level_len[ps[g + 1].a]; });
  TRY(wk.take());
  TRY(upload(d_off, h->level_off.data(), (Lm + 1) * 8, st));
  TRY(upload(d_len, h->level_len.data(), Lm * 8, st));
  {
    const unsigned grid = (unsigned)std::min<uint64_t>((n / 4 + 255) / 256 + 1, (uint64_t)num_sms() * 16);
    if (w == 1) k_map_codes<1><<<grid, 256, 0, st>>>(d_seq, n, d_left, codes);
    else if (w == 2) k_map_codes<2><<<grid, 256, 0, st>>>(d_seq, n, d_left, codes);
    else k_map_codes<4><<<grid, 256, 0, st>>>(d_seq, n, d_left, codes);
    count_launch();
    CK(cudaGetLastError());
  }
  const void* in = codes;
  for (int g = 0; g < G; g++) {
    const PassGeom& pg = ps[g];
    const uint64_t nn = node_lvl[3 * pg.a + 2];
    PassParams P = base_params(h);
    P.lvl_off = d_off;
    P.lvl_len = d_len;
    P.n_in = h->level_len[pg.a];
    P.ntiles = (uint32_t)((P.n_in + T - 1) / T);
    uint64_t mt = P.ntiles;
    if (g > 0) {
      // tiles inside the nodes of the pass's first level (the first pass has
      // one node, the whole sequence)
      if (nn) {
        const uint64_t* bnd = h->d_node + node_lvl[3 * pg.a];
        mt += nn;
        TRY(launch_node_tiles(bnd, nn, T, node_lvl[3 * pg.a + 1], mt, tcnt, toff, scr, tiles,
                              d_ntiles, st));
      } else {
        CK(cudaMemsetAsync(d_ntiles, 0, 4, st));
      }
      CK(cudaGetLastError());
      P.tiles = tiles;
      P.ntiles_dev = d_ntiles;
    }
    P.in = in;
    P.in_w = pg.in_w;
    P.out = (g + 1 < G) ? seqbuf[g & 1] : nullptr;
    P.out_w = pg.out_w;
    P.L = Lm;
    P.a = pg.a;
    P.t = pg.t;
    P.rbits = pg.rbits;
    P.shape = SHAPE_HUFF;
    P.hf_node = h->d_node;
    P.hf_lvl = h->d_node_lvl;
    TRY(launch_pass(P, false, mt, tb, o, st));
    in = P.out;
  }
  if (!(o && (o->flags & WT_FLAG_NO_DIRECTORY))) TRY(build_directories(h));
  return copies.finish(h);
}


}  // namespace wtk

namespace wtk {
wt_status scan_excl_u64_pub(const uint64_t* in, uint64_t* out, uint64_t n, uint64_t* scratch,
                            cudaStream_t st) {
  return scan_excl_u64(in, out, n, scratch, st);
}
uint64_t scan_scratch_pub(uint64_t n) { return scan_scratch(n); }
}  // namespace wtk
