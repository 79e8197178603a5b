// Work items of the persistent prefill attention (fp_attn_tc.cu): which query tiles
// make up an item and in which order the CTAs take the items.  Host and device.
#pragma once

#include <algorithm>
#include <numeric>

#ifdef __CUDACC__
#define FP_BOTH __host__ __device__ __forceinline__
#else
#define FP_BOTH inline
#endif

namespace fpk {

constexpr int kPaB = 128;  // query rows per tile = keys per tile

struct PaPlan {
  int pair;   // 0: one query tile an item, its key tiles taken in turn by the two
              // softmax groups; 1: the same rows of two heads; 2: 256 rows of a head
  int units;  // items of one (sequence, head or pair of heads)
  int items;
  int block;  // (sequence, head)s whose items are taken together
};

// The item that CTA c of g takes in round n, plan.items or more: none.  The list holds
// block after block of heads and, within a block, the longest items first; every other
// round takes it backwards, which evens the CTAs' shares out.
FP_BOTH int pa_item(int n, int c, int g) { return n * g + ((n & 1) ? g - 1 - c : c); }

// The (sequence, head) of item i and its place among that head's items, 0 the shortest.
FP_BOTH void pa_place(int i, const PaPlan& p, unsigned* head, int* unit) {
  const unsigned all = (unsigned)p.items / (unsigned)p.units, per = (unsigned)p.block * (unsigned)p.units;
  const unsigned first = (unsigned)i / per * (unsigned)p.block, rem = (unsigned)i % per;  // the block's first head
  const unsigned nh = all - first < (unsigned)p.block ? all - first : (unsigned)p.block;
  *head = first + rem % nh;
  *unit = p.units - 1 - (int)(rem / nh);
}

// A work item: up to two query tiles of sequence b that share KV head kvh.
struct PaItem {
  int b, h[2], q0[2], nt[2], kvh;  // nt: key tiles up to the diagonal (0: no rows in this tile)
  FP_BOTH PaItem(int i, int S, int H, int Hkv, const PaPlan& p) {
    const unsigned heads = p.pair == 1 ? H / 2 : H;
    unsigned hb;
    int u;
    pa_place(i, p, &hb, &u);
    b = hb / heads;
    const int hh = hb % heads;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int j = 0; j < 2; ++j) {
      h[j] = p.pair == 1 ? 2 * hh + j : hh;
      q0[j] = p.pair == 2 ? (2 * u + j) * kPaB : u * kPaB;
      const int end = q0[j] + kPaB < S ? q0[j] + kPaB : S;
      nt[j] = q0[j] < S && (j == 0 || p.pair) ? (end - 1) / kPaB + 1 : 0;
    }
    kvh = (unsigned)h[0] / ((unsigned)H / (unsigned)Hkv);
  }
  FP_BOTH int tiles() const { return nt[0] > nt[1] ? nt[0] : nt[1]; }
  // of tile j (a runtime index into the arrays would put them in local memory)
  FP_BOTH int head(int j) const { return j ? h[1] : h[0]; }
  FP_BOTH int row0(int j) const { return j ? q0[1] : q0[0]; }
  FP_BOTH int key_tiles(int j) const { return j ? nt[1] : nt[0]; }
};

// Pairs of tiles, or, where those leave SMs idle or one CTA's share too long, single
// tiles with their keys cut in two: the smaller of the largest shares that the CTAs draw,
// with 4100 cycles for a step of a pair (a key tile) and 6500 an item, 7200 for a single
// tile's step (two key tiles) and 2500 an item.  Fitted to 18,500 launches of both forms (1
// to 24 sequences, 129 to 4096 tokens, both caches): the form chosen is 0.16 % slower than
// the better one on average, at most 17 %.  (With 3500 / 4100 / 4000 and the mean share it
// was 0.7-5 % and at most 73 %: bf16 3 x 267 tokens, 32 heads 19.2 us against 15.7, 10 x 1645,
// 8 heads 100 against 92.)  Past four rounds pairs, which work 1.75 times as fast.
// Longest first over the whole list leaves the SMs' shares even (largest / mean 1.00-1.03)
// but has them read different heads' keys and values; blocks of heads keep most of the
// sharing in L2.  A block that is a whole even number of rounds of the SMs evens its
// shares out by itself, so four rounds are enough; where eight rounds hold no such
// block, the list is cut into equal blocks of at least eight, whose ends cost up to 15 %
// (2 to 64 tiles, 5 to 110 rounds).  Microseconds, blocks of four whole rounds | eight
// rounds | the whole list | head by head, the tile an item takes rotated from round to
// round (where the rotation's step and the number of tiles had a common divisor, a CTA
// drew the same tile every time):
//   int8  4 x 4000, 32 heads      1093 | 1202 | 1192 | 1163
//         32 x 2048, 64 on 8      4190 | 4338 | 4734 | 4525
//         16 x 1300, 32 heads      749 |  761 |  767 |  815
//         8 x 2304, 32 heads           |  829 |  828 | 1289
//         32 x 2100, 64 on 8           | 4774 | 5302 | 8351
//   bf16  32 x 2048, 32 heads     1053 | 1096 | 1142 | 1071
//         8 x 1024, 40 heads       121 |  125 |  126 |  126
//         32 x 2304, 32 heads          | 1366 | 1380 | 2296
inline PaPlan pa_plan(int B, int S, int H, int G, int sms) {
  const long long tiles = (S + kPaB - 1) / kPaB;
  const int pair = G % 2 == 0 ? 1 : 2;
  auto make = [&](int pr) {
    PaPlan p{};
    p.pair = pr;
    p.units = (int)(pr == 2 ? (tiles + 1) / 2 : tiles);
    const long long heads = (long long)B * (pr == 1 ? H / 2 : H);
    p.items = (int)(heads * p.units);
    const long long whole = 2LL * sms / std::gcd(2LL * sms, (long long)p.units);  // heads of even whole rounds
    const long long blocks = std::max(1LL, p.items / (8LL * sms));
    if (whole * p.units <= 8LL * sms) p.block = (int)std::min(heads, whole * std::max(1LL, 4LL * sms / (whole * p.units)));
    else p.block = (int)((heads + blocks - 1) / blocks);
    return p;
  };
  auto span = [&](const PaPlan& p) {
    double worst = 0;
    const int g = std::min(p.items, sms);
    for (int c = 0; c < g + 7; c += 8) {  // some of the CTAs: neighbours draw alike
      double t = 0;
      for (int n = 0, cta = std::min(c, g - 1), i = cta; i < p.items; i = pa_item(++n, cta, g)) {
        unsigned head;
        int u;
        pa_place(i, p, &head, &u);
        const long long steps = p.pair == 2 ? std::min(tiles, 2LL * u + 2) : p.pair == 1 ? u + 1 : u / 2 + 1;
        t += p.pair ? 4100. * steps + 6500 : 7200. * steps + 2500;
      }
      worst = std::max(worst, t);
    }
    return worst;
  };
  const PaPlan two = make(pair);
  if (two.items > 4LL * sms) return two;
  const PaPlan one = make(0);
  return span(one) < span(two) ? one : two;
}

}  // namespace fpk
