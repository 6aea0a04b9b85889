// How many CTAs (of one thread-block cluster) share a piece of work: the rules of
// the launchers and kernels, in C++ that a host compiler takes too.
#pragma once

#include <algorithm>

#ifdef __CUDACC__
#define TK_HOST_DEVICE __host__ __device__
#else
#define TK_HOST_DEVICE
#endif

namespace tk {

constexpr int kMaxSplit = 8;  // CTAs of a cluster

// Prefill: CTAs, at most `most`, among which the kv tiles of a query tile pair are
// split, for a sequence of kv_tiles 128-key tiles: where the tiles saved (about
// 1 us each) are worth the merge (3 to 4 us), and of all kv tiles every CTA keeps
// three (pairs early in a causal sequence have fewer).  Measured, r = 32, d_v = 128,
// one CTA a pair against split: 32/8 heads, 500 tokens after 8000 82 us -> 51 (two
// CTAs), 23 after 13000 100 -> 35 (four); 16/8 heads, B=2, 500 after 2000, int8
// 35 -> 30; but 500 after 500 (8 kv tiles) 16.8 -> 18.0 and a prompt of 512 (4)
// 9.6 -> 12.0.
TK_HOST_DEVICE inline int prefill_shares(long long kv_tiles, int most) {
  // (without a loop and without branches: the kernel's values stay warp-uniform)
  const int fit = kv_tiles >= 24 ? 8 : (kv_tiles >= 12 ? 4 : (kv_tiles >= 10 ? 2 : 1));
  return fit < most ? fit : most;   // powers of two
}

// Prefill: CTAs of a cluster for `pairs` query tile pairs, so that each finds an SM;
// kv_tiles is the launch's bound.  A sequence of fewer tiles uses as many of them as
// prefill_shares gives its own, so that its result and, but for idle CTAs, its time do
// not depend on the bound.
inline int prefill_cluster(long long pairs, long long kv_tiles, int num_sms) {
  int most = 1;
  while (2 * most <= kMaxSplit && pairs * 2 * most <= num_sms) most *= 2;
  return prefill_shares(kv_tiles, most);
}

}  // namespace tk
