// huffdev.cu -- Huffman code tables of large alphabets on the device (paper
// Section 4.3, arbitrarily shaped trees: the code the tree is built from).
//
// The result is that of huffman.cpp and the host sweeps of build_huff, bit for
// bit: lengths of the merge that always takes the two lightest nodes, ties by
// (weight, id) with leaf id = symbol and internal id = sigma + creation order;
// canonical codes; the node tables of every level.  The host does nothing per
// symbol.
//
//   1. the symbols sorted by (weight, symbol): a stable LSD radix sort;
//   2. the merge in rounds.  Both queues (sorted leaves, internal nodes in
//      creation order) are sorted; let M be the sum of the two lightest heads.
//      Every node present with weight <= M precedes every node that a merge
//      creates from now on (those weigh at least M, and at M their ids are
//      larger), so these nodes are paired two by two in their merged order at
//      once, each pair placed by a merge-path search.  M at least doubles every
//      second round, so the rounds grow with the logarithm of the total weight;
//      a code that needs more than ROUNDS of them (or lengths past 32, which
//      are limited on the host) is left to the host;
//   3. depths by pointer jumping over the internal nodes' parents;
//   4. the symbols by (length, symbol): one more radix pass; codes, node
//      starts and zero counts from each symbol's place in that order.
//
// What bounds it: launches and L2 latency.  About 110 launches, whose kernels take
// 0.6 ms over 2^20 symbols, half of it the 72 rounds of the merge.  A Huffman-
// shaped tree of 2^28 symbols over 2^20 takes 8.1 ms; the host needs 16 ms for
// that code alone.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "wt_host.h"
#include "wt_internal.cuh"

namespace wtk {

#define CK(x)                                                                   \
  do {                                                                          \
    cudaError_t e_ = (x);                                                       \
    if (e_ != cudaSuccess) {                                                    \
      fprintf(stderr, "wavelet: %s -> %s\n", #x, cudaGetErrorString(e_));      \
      cudaGetLastError(); /* reported here */                                   \
      return e_ == cudaErrorMemoryAllocation ? WT_ERR_NO_MEMORY : WT_ERR_CUDA; \
    }                                                                           \
  } while (0)

wt_status scan_excl_u64_pub(const uint64_t* in, uint64_t* out, uint64_t n, uint64_t* scratch,
                            cudaStream_t st);
uint64_t scan_scratch_pub(uint64_t n);

namespace {

constexpr int ROUNDS = 72;
constexpr uint32_t RS_TILE = 4096;  // items per block of a radix pass: 512 per warp

// the keys of a radix pass: symbol counts (u64, below 2^32), u32 keys, lengths
enum Src : int { SRC_HIST = 0, SRC_U32 = 1, SRC_LEN = 2 };
template <int SRC>
__device__ __forceinline__ uint32_t rs_key(const void* keys, uint32_t i) {
  if (SRC == SRC_HIST) return (uint32_t)((const uint64_t*)keys)[i];
  if (SRC == SRC_LEN) return ((const uint8_t*)keys)[i];
  return ((const uint32_t*)keys)[i];
}

// counts of each block's 8-bit digits, digit by digit: cnt[d * nblk + block]
template <int SRC>
__global__ void __launch_bounds__(256) k_rs_count(const void* keys, uint32_t n, int shift,
                                                  uint64_t* cnt) {
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t i0 = blockIdx.x * RS_TILE;
  for (uint32_t k = threadIdx.x; k < RS_TILE; k += 256)
    if (i0 + k < n) atomicAdd(&h[(rs_key<SRC>(keys, i0 + k) >> shift) & 255u], 1u);
  __syncthreads();
  cnt[(uint64_t)threadIdx.x * gridDim.x + blockIdx.x] = h[threadIdx.x];
}

// stable scatter by the digit, from the scanned counts: a warp's 512 items in
// rows of 32, ranked by the lanes with the same digit
template <int SRC>
__global__ void __launch_bounds__(256) k_rs_scatter(const void* keys, const uint32_t* vals, uint32_t n,
                                                    int shift, const uint64_t* base,
                                                    uint32_t* keys_out, uint32_t* vals_out) {
  __shared__ uint32_t wc[8][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = lane; k < 256; k += 32) wc[warp][k] = 0;
  __syncwarp();
  const uint32_t i0 = blockIdx.x * RS_TILE + warp * 512 + lane;
  constexpr uint32_t NODIGIT = 256;
  for (int row = 0; row < 16; row++) {
    const uint32_t i = i0 + 32 * row;
    const uint32_t d = i < n ? (rs_key<SRC>(keys, i) >> shift) & 255u : NODIGIT;
    const uint32_t peers = __match_any_sync(FULL, d);
    if (d != NODIGIT && lane == __ffs(peers) - 1) wc[warp][d] += __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  {
    uint32_t run = (uint32_t)base[(uint64_t)threadIdx.x * gridDim.x + blockIdx.x];
    for (int w = 0; w < 8; w++) {
      const uint32_t c = wc[w][threadIdx.x];
      wc[w][threadIdx.x] = run;
      run += c;
    }
  }
  __syncthreads();
  for (int row = 0; row < 16; row++) {
    const uint32_t i = i0 + 32 * row;
    const uint32_t key = i < n ? rs_key<SRC>(keys, i) : 0u;
    const uint32_t d = i < n ? (key >> shift) & 255u : NODIGIT;
    const uint32_t peers = __match_any_sync(FULL, d);
    if (d != NODIGIT) {
      const uint32_t at = wc[warp][d] + __popc(peers & lanemask_lt());
      if (keys_out) keys_out[at] = key;
      vals_out[at] = vals ? vals[i] : i;
    }
    __syncwarp();
    if (d != NODIGIT && lane == __ffs(peers) - 1) wc[warp][d] += __popc(peers);
    __syncwarp();
  }
}

// first index in [lo, hi) of the sorted a with a[index] > v, by a whole warp,
// 32 entries a step
__device__ uint32_t warp_upper_bound(const uint32_t* a, uint32_t lo, uint32_t hi, uint32_t v) {
  const uint32_t lane = threadIdx.x & 31;
  while (lo < hi) {
    const uint32_t step = (hi - lo + 31) / 32, at = lo + (lane + 1) * step - 1;
    const uint32_t c = (uint32_t)__popc(__ballot_sync(FULL, at < hi && a[at] <= v));
    const uint32_t next = lo + c * step;
    hi = min(hi, next + step - 1);  // a[next + step - 1] > v, or past the end
    lo = min(next, hi);
    if (step == 1) break;
  }
  return lo;
}

// The merge's state before a round: next leaf, next internal node, internal
// nodes made.
struct Merge {
  uint32_t li, qi, ni;
};

__global__ void k_huff_begin(const uint32_t* w, uint32_t sigma, Merge* st) {
  const uint32_t z = warp_upper_bound(w, 0, sigma, 0u);  // past the absent symbols
  if (threadIdx.x == 0) st[0] = Merge{z, 0u, 0u};
}

// leaves among the first d nodes of the merged order of the leaves wl[0..A)
// and the internal nodes wi[0..B) (equal weights: the leaf first)
__device__ __forceinline__ uint32_t merge_path(const uint32_t* wl, uint32_t A, const uint32_t* wi,
                                               uint32_t B, uint32_t d) {
  uint32_t lo = d > B ? d - B : 0u, hi = d < A ? d : A;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (wl[mid] <= wi[d - 1 - mid]) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(256) k_huff_round(const uint32_t* w, uint32_t sigma, uint32_t* iw,
                                                    uint32_t* pl, uint32_t* pi, Merge* st) {
  __shared__ uint32_t s_end[2];
  const Merge m = st[0];
  const uint32_t leaves = sigma - m.li, inner = m.ni - m.qi;
  if (leaves + inner <= 1) {  // the root is made
    if (blockIdx.x == 0 && threadIdx.x == 0) st[1] = m;
    return;
  }
  const uint64_t none = 1ull << 40;
  const uint64_t a0 = leaves > 0 ? w[m.li] : none, a1 = leaves > 1 ? w[m.li + 1] : none;
  const uint64_t b0 = inner > 0 ? iw[m.qi] : none, b1 = inner > 1 ? iw[m.qi + 1] : none;
  const uint32_t M = (uint32_t)min(a0 + b0, min(a0 + a1, b0 + b1));
  const int warp = threadIdx.x >> 5;
  if (warp < 2) {
    const uint32_t e = warp == 0 ? warp_upper_bound(w, m.li, sigma, M) : warp_upper_bound(iw, m.qi, m.ni, M);
    if ((threadIdx.x & 31) == 0) s_end[warp] = e;
  }
  __syncthreads();
  const uint32_t *wl = w + m.li, *wi = iw + m.qi;
  const uint32_t A = s_end[0] - m.li, B = s_end[1] - m.qi, pairs = (A + B) / 2;
  for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < pairs; p += gridDim.x * blockDim.x) {
    uint32_t a = merge_path(wl, A, wi, B, 2 * p), b = 2 * p - a, sum = 0;
#pragma unroll
    for (int k = 0; k < 2; k++) {
      if (a < A && (b >= B || wl[a] <= wi[b])) {
        sum += wl[a];
        pl[m.li + a++] = m.ni + p;
      } else {
        sum += wi[b];
        pi[m.qi + b++] = m.ni + p;
      }
    }
    iw[m.ni + p] = sum;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const uint32_t a = merge_path(wl, A, wi, B, 2 * pairs);
    st[1] = Merge{m.li + a, m.qi + 2 * pairs - a, m.ni + pairs};
  }
}

// parent and distance to it of every internal node (the root its own)
__global__ void k_huff_parents(const uint32_t* pi, const Merge* st, uint2* up) {
  const uint32_t ni = st->ni;
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < ni; k += gridDim.x * blockDim.x)
    up[k] = k + 1 == ni ? make_uint2(k, 0u) : make_uint2(pi[k], 1u);
}
__global__ void k_huff_jump(const uint2* up, const Merge* st, uint2* out) {
  const uint32_t ni = st->ni;
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < ni; k += gridDim.x * blockDim.x) {
    const uint2 a = up[k], b = up[a.x];
    out[k] = make_uint2(b.x, a.y + b.y);
  }
}

// lengths of the sorted leaves' symbols, and the weight of each length
// (33: longer than 32); neighbours mostly share theirs
__global__ void __launch_bounds__(256) k_huff_lengths(const uint32_t* w, const uint32_t* sym,
                                                      uint32_t sigma, const uint32_t* pl,
                                                      const uint2* up, const Merge* begin,
                                                      uint8_t* len, uint64_t* wlen) {
  const uint32_t z = begin->li, lane = threadIdx.x & 31;
  for (uint32_t b = z + blockIdx.x * blockDim.x + (threadIdx.x & ~31u); b < sigma; b += gridDim.x * blockDim.x) {
    const uint32_t i = b + lane;
    const bool on = i < sigma;
    uint32_t ln = 0, wi = 0;
    if (on) {
      ln = sigma - z == 1 ? 1u : min(up[pl[i]].y + 1u, 33u);
      wi = w[i];
      len[sym[i]] = (uint8_t)ln;
    }
    const uint32_t peers = __match_any_sync(FULL, ln);
    const uint32_t sum = __reduce_add_sync(peers, wi);  // at most n, below 2^32
    if (on && lane == (uint32_t)__ffs(peers) - 1) atomicAdd((unsigned long long*)&wlen[ln], (unsigned long long)sum);
  }
}

// what the host needs: start of each length in the (length, symbol) order, its
// weight, and the merge's last state
struct HuffInfo {
  uint64_t first[35], weight[34];
  Merge end;
  uint32_t err;
};
__global__ void k_huff_info(const uint64_t* base, uint32_t nblk, const uint64_t* wlen, const Merge* end,
                            const uint32_t* err, HuffInfo* info) {
  const int t = threadIdx.x;
  if (t < 35) info->first[t] = base[(uint64_t)t * nblk];
  if (t < 34) info->weight[t] = wlen[t];
  if (t == 0) {
    info->end = *end;
    info->err = *err;
  }
}

__global__ void k_huff_weights(const uint64_t* hist, const uint32_t* order, uint32_t np, uint64_t* w) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x)
    w[i] = hist[order[i]];
}

// per length: first code and index in the order; per level: offset and first
// prefix in the node table, elements before the level's first symbol, nodes,
// elements
struct HuffLevels {
  int Lm;
  uint32_t np;
  uint64_t fcode[33];
  uint32_t lpos[33];
  uint64_t off[32], prefix[32], before[32], nodes[32], elems[32];
};

// codes, left-aligned codes, symbols in order, node starts and zero counts
// (the canonical codes' properties that give a symbol's new nodes are stated
// at the host form of this sweep in build_huff)
__global__ void __launch_bounds__(256) k_huff_tables(const __grid_constant__ HuffLevels t,
                                                     const uint32_t* order, const uint8_t* len,
                                                     const uint64_t* w, const uint64_t* S,
                                                     uint32_t* code, uint32_t* left, uint32_t* by_rank,
                                                     uint64_t* node, uint64_t* zeros) {
  const int Lm = t.Lm;
  const uint32_t lane = threadIdx.x & 31;
  uint64_t mine = 0;  // lane l: the zeros of level l met by this warp
  for (uint32_t b = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); b < t.np; b += gridDim.x * blockDim.x) {
    const uint32_t i = b + lane;
    int ln = 0;
    uint64_t lc = 0;
    uint32_t wi = 0;
    if (i < t.np) {
      const uint32_t sym = order[i];
      ln = len[sym];
      const uint64_t c = t.fcode[ln] + (i - t.lpos[ln]);
      lc = c << (Lm - ln);
      wi = (uint32_t)w[i];
      code[sym] = (uint32_t)c;
      left[sym] = (uint32_t)lc;
      by_rank[i] = sym;
      int open = 0;
      if (i > 0) {
        const int lp = len[order[i - 1]];
        const uint64_t prev = (t.fcode[lp] + (i - 1 - t.lpos[lp])) << (Lm - lp);
        open = __clzll((long long)((prev ^ lc) << (64 - Lm))) + 1;
      }
      for (int l = open; l < ln; l++) {
        const uint64_t k = (lc >> (Lm - l)) - t.prefix[l];
        if (k < t.nodes[l]) node[t.off[l] + k] = S[i] - t.before[l];  // always, for a prefix code
      }
    }
    for (int l = 0; l < Lm; l++) {
      const bool zero = l < ln && !((lc >> (Lm - 1 - l)) & 1u);
      const uint32_t sum = __reduce_add_sync(FULL, zero ? wi : 0u);  // at most n, below 2^32
      if ((int)lane == l) mine += sum;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x < Lm)
    node[t.off[threadIdx.x] + t.nodes[threadIdx.x]] = t.elems[threadIdx.x];  // sentinel
  if ((int)lane < Lm && mine) atomicAdd((unsigned long long*)&zeros[lane], (unsigned long long)mine);
}

template <int SRC>
wt_status radix_pass(const void* keys, const uint32_t* vals, uint32_t n, int shift, uint64_t* cnt,
                     uint64_t* base, uint64_t* scr, uint32_t* keys_out, uint32_t* vals_out,
                     cudaStream_t st) {
  const uint32_t nblk = (n + RS_TILE - 1) / RS_TILE;
  k_rs_count<SRC><<<nblk, 256, 0, st>>>(keys, n, shift, cnt);
  count_launch();
  TRY(scan_excl_u64_pub(cnt, base, (uint64_t)256 * nblk, scr, st));
  k_rs_scatter<SRC><<<nblk, 256, 0, st>>>(keys, vals, n, shift, base, keys_out, vals_out);
  count_launch();
  CK(cudaGetLastError());
  return WT_OK;
}

}  // namespace

// The code tables of h (device arrays, levels, lengths of the levels) from the
// symbol counts; *done = false when the host has to make them.  d_left: the
// left-aligned codes.  Returns WT_ERR_SYMBOL_GE_SIGMA if the counts met one.
wt_status huff_tables_device(const uint64_t* hist, uint64_t n, uint32_t sigma, wt_struct* h,
                             uint32_t* d_left, std::vector<uint64_t>& node_lvl, bool* done) {
  *done = false;
  cudaStream_t st = h->stream;
  const uint32_t nblk = (sigma + RS_TILE - 1) / RS_TILE;
  Work wk{st};
  uint32_t *key[2], *val[2], *pl, *pi, *iw, *order;
  uint64_t *cnt, *base, *scr, *wlen, *wS, *S;
  uint2* up[2];
  Merge* ms;
  HuffInfo* info;
  for (int k = 0; k < 2; k++) {
    wk.want(&key[k], sigma);
    wk.want(&val[k], sigma);
    wk.want(&up[k], sigma);
  }
  wk.want(&pl, sigma);
  wk.want(&pi, sigma);
  wk.want(&iw, sigma);
  wk.want(&order, sigma);
  wk.want(&cnt, (size_t)256 * nblk);
  wk.want(&base, (size_t)256 * nblk + 1);
  wk.want(&scr, scan_scratch_pub(std::max<uint64_t>((uint64_t)256 * nblk, sigma)));
  wk.want(&wlen, 34);
  wk.want(&wS, sigma);
  wk.want(&S, (size_t)sigma + 1);
  wk.want(&ms, ROUNDS + 1);
  wk.want(&info, 1);
  TRY(wk.take());
  CK(dmalloc((void**)&h->d_code, (size_t)sigma * 4, st));
  CK(dmalloc((void**)&h->d_len, sigma, st));
  CK(cudaMemsetAsync(h->d_len, 0, sigma, st));
  CK(cudaMemsetAsync(h->d_code, 0, (size_t)sigma * 4, st));
  CK(cudaMemsetAsync(wlen, 0, 34 * 8, st));
  // 1. symbols by (weight, symbol); a weight is at most n
  int bits = 1;
  while (bits < 32 && (n >> bits)) bits++;
  int c = 0;
  for (int sh = 0; sh < bits; sh += 8, c ^= 1) {
    if (sh == 0) TRY(radix_pass<SRC_HIST>(hist, nullptr, sigma, 0, cnt, base, scr, key[c], val[c], st));
    else TRY(radix_pass<SRC_U32>(key[c ^ 1], val[c ^ 1], sigma, sh, cnt, base, scr, key[c], val[c], st));
  }
  const uint32_t *w = key[c ^ 1], *sym = val[c ^ 1];
  // 2. the merge
  const unsigned grid = (unsigned)std::min<uint64_t>((sigma / 2 + 255) / 256 + 1, (uint64_t)num_sms() * 8);
  k_huff_begin<<<1, 32, 0, st>>>(w, sigma, ms);
  for (int r = 0; r < ROUNDS; r++) k_huff_round<<<grid, 256, 0, st>>>(w, sigma, iw, pl, pi, ms + r);
  // 3. depths below 64
  k_huff_parents<<<grid, 256, 0, st>>>(pi, ms + ROUNDS, up[0]);
  for (int k = 0; k < 6; k++) k_huff_jump<<<grid, 256, 0, st>>>(up[k & 1], ms + ROUNDS, up[(k & 1) ^ 1]);
  k_huff_lengths<<<grid, 256, 0, st>>>(w, sym, sigma, pl, up[0], ms, h->d_len, wlen);
  count_launch(ROUNDS + 9);
  // 4. symbols by (length, symbol), the absent ones first
  TRY(radix_pass<SRC_LEN>(h->d_len, nullptr, sigma, 0, cnt, base, scr, nullptr, order, st));
  k_huff_info<<<1, 64, 0, st>>>(base, nblk, wlen, ms + ROUNDS, h->d_err, info);
  count_launch();
  CK(cudaGetLastError());
  HuffInfo hi;
  CK(cudaMemcpyAsync(&hi, info, sizeof(hi), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  if (hi.err & ERR_SYMBOL) return WT_ERR_SYMBOL_GE_SIGMA;
  const uint64_t absent = hi.first[1], np = sigma - absent;
  // the root not made in time, or lengths past 32: the host's
  const bool root = (sigma - hi.end.li) + (hi.end.ni - hi.end.qi) == 1;
  if (np == 0 || !root || hi.first[33] != sigma) {
    dfree(h->d_code, st);
    dfree(h->d_len, st);
    h->d_code = nullptr;
    h->d_len = nullptr;
    return WT_OK;
  }
  // per length and per level, from the symbols and weights of each length
  HuffLevels t{};
  std::vector<uint64_t> lentab(3 * 34, 0);
  int Lm = 0;
  uint64_t code = 0;
  for (int ln = 1; ln <= 32; ln++) {
    const uint64_t k = hi.first[ln + 1] - hi.first[ln];
    t.lpos[ln] = (uint32_t)(hi.first[ln] - absent);
    lentab[34 + ln] = t.lpos[ln];
    lentab[68 + ln] = k;
    if (!k) continue;
    const uint64_t before = Lm ? lentab[68 + Lm] : 0;
    code = Lm ? (code + before) << (ln - Lm) : 0;
    t.fcode[ln] = lentab[ln] = code;
    Lm = ln;
  }
  t.Lm = Lm;
  t.np = (uint32_t)np;
  h->max_code_len = (uint32_t)Lm;
  h->L = h->levels = (uint32_t)Lm;
  h->level_len.assign(Lm, 0);
  node_lvl.assign(3 * (size_t)Lm, 0);
  uint64_t tot = 0, left_in = n;  // elements with longer codes than l
  const uint64_t last = t.fcode[Lm] + lentab[68 + Lm] - 1;
  for (int l = 0; l < Lm; l++) {
    if (l) left_in -= hi.weight[l];
    int lf = l + 1;  // the first symbol of the level has the next length in use
    while (!lentab[68 + lf]) lf++;
    t.off[l] = tot;
    t.prefix[l] = t.fcode[lf] >> (lf - l);
    t.nodes[l] = (last >> (Lm - l)) - t.prefix[l] + 1;
    t.before[l] = n - left_in;
    t.elems[l] = left_in;
    h->level_len[l] = left_in;
    node_lvl[3 * l] = t.off[l];
    node_lvl[3 * l + 1] = t.prefix[l];
    node_lvl[3 * l + 2] = t.nodes[l];
    tot += t.nodes[l] + 1;
  }
  CK(dmalloc((void**)&h->d_sym_by_rank, np * 4, st));
  CK(dmalloc((void**)&h->d_len_tab, lentab.size() * 8, st));
  CK(dmalloc((void**)&h->d_node, tot * 8, st));
  CK(dmalloc((void**)&h->d_node_lvl, node_lvl.size() * 8, st));
  TRY(upload(h->d_len_tab, lentab.data(), lentab.size() * 8, st));
  TRY(upload(h->d_node_lvl, node_lvl.data(), node_lvl.size() * 8, st));
  order += absent;
  k_huff_weights<<<grid, 256, 0, st>>>(hist, order, (uint32_t)np, wS);
  count_launch();
  TRY(scan_excl_u64_pub(wS, S, np, scr, st));
  k_huff_tables<<<grid, 256, 0, st>>>(t, order, h->d_len, wS, S, h->d_code, d_left, h->d_sym_by_rank,
                                      h->d_node, h->d_zeros);
  count_launch();
  CK(cudaGetLastError());
  *done = true;
  return WT_OK;
}

}  // namespace wtk
