// The bit-plane arithmetic of the partition pass, compiled for the host,
// against element-by-element definitions.  Prints "ok" or the first difference.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "bitplane.cuh"

using namespace wtk;

static uint64_t state = 88172645463325252ull;
static uint32_t rnd() {  // xorshift64
  state ^= state << 13;
  state ^= state >> 7;
  state ^= state << 17;
  return (uint32_t)(state >> 16);
}

static void fail(const char* what, int ew, int rbits, int t, int n) {
  printf("%s: %d-byte elements, %d bits, %d levels, %d elements\n", what, ew, rbits, t, n);
  exit(1);
}

template <int EW>
static void check(int rbits, int t, int n, int fill) {
  // 32 elements, the first n of them the thread's, in memory order
  uint32_t words[8 * EW], el[32];
  for (int i = 0; i < 8 * EW; i++) words[i] = fill == 0 ? rnd() : (fill == 1 ? 0u : ~0u);
  for (int i = 0; i < 32; i++) {
    const int bit = 8 * EW * i;
    el[i] = EW == 4 ? words[i] : (words[bit / 32] >> (bit % 32)) & ((1u << (8 * EW & 31)) - 1u);
  }
  auto digit = [&](uint32_t e, int j) { return (e >> (rbits - 1 - j)) & 1u; };
  uint32_t p[4];
  planes_of<EW>([&](int i, uint32_t* w) {
    for (int k = 0; k < 4; k++) w[k] = words[4 * i + k];
  }, rbits, p);
  for (int j = t; j < 4; j++) p[j] = 0u;
  for (int j = 0; j < t; j++)
    for (int i = 0; i < 32; i++)
      if (((p[j] >> i) & 1u) != digit(el[i], j)) fail("planes", EW, rbits, t, n);
  const uint32_t v = low_mask((uint32_t)n);
  uint32_t c[8], want[16] = {};
  key_counts(p, v, c);
  for (int i = 0; i < n; i++) {
    uint32_t key = 0;
    for (int j = 0; j < t; j++) key |= digit(el[i], j) << j;
    want[key]++;
  }
  for (int k = 0; k < 16; k++)
    if (((c[k / 2] >> (16 * (k & 1))) & 0xffffu) != want[k]) fail("key counts", EW, rbits, t, n);
  // the splits as the pass makes them: the level bits of a .. a + t - 1
  for (int j = 0; j < 4; j++) p[j] |= ~v;
  if (t >= 2) {
    uint32_t x[4];
    if (t == 4) {
      for (int j = 0; j < 4; j++) x[j] = reverse32(p[j]);
    } else {
      x[1] = reverse32(p[0]);
      x[2] = t == 3 ? reverse32(p[1]) : x[1];
      x[3] = reverse32(t == 3 ? p[2] : p[1]);
    }
    if (t == 4) split_planes<3>(x[0], x + 1);
    if (t >= 3) split_planes<2>(x[1], x + 2);
    split_planes<1>(x[2], x + 3);
    p[1] = reverse32(t == 4 ? x[1] : (t == 3 ? x[2] : x[3]));
    p[2] = reverse32(t == 4 ? x[2] : x[3]);
    p[3] = reverse32(x[3]);
  }
  std::vector<uint32_t> cur(el, el + n);
  for (int j = 0; j < t; j++) {
    for (int i = 0; i < n; i++)
      if (((p[j] >> i) & 1u) != digit(cur[i], j)) fail("splits", EW, rbits, t, n);
    std::vector<uint32_t> next;
    for (int b = 0; b < 2; b++)
      for (uint32_t e : cur)
        if ((int)digit(e, j) == b) next.push_back(e);
    cur = next;
  }
}

int main() {
  for (int n = 0; n <= 32; n++)
    for (int t = 1; t <= 4; t++)
      for (int r = 0; r < 8; r++) {
        const int fill = r < 6 ? 0 : r - 5;
        for (int b = t; b <= 8; b++) check<1>(b, t, n, fill);
        for (int b = t; b <= 16; b++) check<2>(b, t, n, fill);
        for (int b = t; b <= 32; b++) check<4>(b, t, n, fill);
      }
  // one split of every pattern of a byte's bits beside the others
  for (uint32_t b = 0; b < 256; b++)
    for (int r = 0; r < 64; r++) {
      const uint32_t by = (b << (8 * (r & 3))) | (rnd() & ~(0xffu << (8 * (r & 3))));
      uint32_t x = rnd(), want = 0, at = 0;
      for (int h = 0; h < 2; h++)
        for (int i = 31; i >= 0; i--)
          if ((int)((by >> i) & 1u) == h) want |= ((x >> i) & 1u) << (31 - at++);
      split_planes<1>(by, &x);
      if (x != want) fail("split", 0, 0, 1, 32);
    }
  printf("ok\n");
  return 0;
}
