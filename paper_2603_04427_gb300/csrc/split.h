// How many CTAs (of one thread-block cluster) share a piece of work: the rules of
// the launchers and kernels, in C++ that a host compiler takes too.
#pragma once

#include <algorithm>
#include <cmath>

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

// Backward: CTAs of a cluster per 128-key tile: the number with the least estimated
// time, in units of one query tile's (1.6 us at r = 32): a CTA costs 5 for set-up and
// epilogue, 2 more if split; causal launches (CTAs of many sizes, the largest first)
// take the longer of their heaviest CTA and the mean of the SMs, and half a set-up more
// where a split needs a second CTA on an SM; others whole waves.  Every CTA of the
// heaviest key tile keeps at least two query tiles (of a causal sequence's last key
// tiles some CTAs have none).  Measured without and with the split: 16/2 heads, r=64,
// d_v=128, B=3, S=138 41 us -> 16; r=32, B=1, S=2000 206 -> 59; r=128, S=500 117 -> 28;
// 32/8 heads, r=32, S=300 26 -> 16, S=1531 87 -> 53; but 12 heads, r=16, d_v=64, S=1024
// 17.4 -> 21.1 with two CTAs a key tile (192 on 152 SMs), so that one is not split.
inline int backward_split(int batch, int h_q, int h_kv, int seq, bool causal, int num_sms) {
  const int n_qt = (seq + 127) / 128;
  const long long grid = static_cast<long long>(batch) * h_kv * n_qt;
  const double heaviest = static_cast<double>(h_q / h_kv) * n_qt;   // the first key tile's
  const double total = heaviest * grid * (causal ? (n_qt + 1) / (2.0 * n_qt) : 1.0);
  int best = 1;
  double least = 0;
  for (int c = 1; c <= kMaxSplit; c *= 2) {
    if (c > 1 && heaviest < 2 * c) break;
    const double fixed = c > 1 ? 7 : 5, one = heaviest / c + fixed;
    const double mean = (total + grid * c * fixed) / num_sms;
    const double t = causal ? std::max(one, mean) + (c > 1 && grid * c > num_sms ? fixed / 2 : 0)
                            : std::ceil(static_cast<double>(grid) * c / num_sms) * one;
    if (c == 1 || t < 0.95 * least) {
      best = c;
      least = t;
    }
  }
  return best;
}

// Backward: CTAs in key tile order over all heads, the heaviest first, rather than head
// by head: where Q and dO of all heads stay within about 48 MB of L2.
inline bool backward_tile_major(int batch, int h_q, int seq, int r, int d_v) {
  return static_cast<long long>(batch) * h_q * seq * (r + d_v) * 2 <= (48LL << 20);
}

}  // namespace tk
