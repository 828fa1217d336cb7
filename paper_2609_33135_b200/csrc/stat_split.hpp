// How the statistics pass over a head's tokens is split.  Host code without CUDA.
#pragma once
#include <algorithm>

namespace mpfa {

constexpr int STAT_CLUSTER = 16;         // largest cluster; more than eight CTAs have to be allowed
constexpr int STAT_CLUSTER_MIN = 128;    // tokens of a slice: one round of loads
// Tokens of a slice up to which clusters are the faster form.  Stage 1 with slices / clusters whose slices have 400, 512, 640 and 800 tokens: 1 + 1
// heads 13.3 / 10.1, 13.1 / 10.8, 14.0 / 12.0, 15.0 / 13.8 us; 8 + 2 19.6 / 18.0, 20.6 / 18.6, 19.7 / 20.0, 22.6 / 25.1; 16 + 4 19.8 / 17.7,
// 20.0 / 18.6, 20.7 / 19.9, 22.4 / 25.0; 32 + 8 20.1 / 18.1, 20.4 / 18.9, 20.2 / 19.8, 23.1 / 25.0.
constexpr int STAT_CLUSTER_MAX = 640;
constexpr int STAT_MIN = 512;            // tokens of a slice where a launch of its own folds them, which costs about as much

struct StatSplit {
  int slices;
  bool clusters;   // the slices of a head are a cluster
};

// heads: of both tensors and all batch elements; N: tokens of the longer tensor; ctas: resident per SM; placeable(C): whether a cluster of
// C CTAs can be launched.
template <class Placeable>
StatSplit stat_split(long long heads, int N, int max_slices, int ctas, int n_sm, Placeable placeable) {
  // Short passes: a cluster for each head, of a power of two CTAs (clusters of seven leave places free in every GPC: 8 + 2 heads of
  // 4 x 777 tokens 13.7 us of stage 1, with four 11.9), as long as its slices stay short and all clusters fit at once.
  int C = STAT_CLUSTER;
  while (C > 1 && (C > max_slices || (C > 8 && N <= 16 * STAT_CLUSTER_MIN) || C * heads * 8 > 7LL * ctas * n_sm || C / 2 * STAT_CLUSTER_MIN >= N)) C /= 2;
  while (C > 1 && N <= C * STAT_CLUSTER_MAX && !placeable(C)) C /= 2;
  if (C > 1 && N <= C * STAT_CLUSTER_MAX) return {C, true};
  // As many slices as the launch can hold in one wave.
  return {(int)std::max(1LL, std::min({(long long)max_slices, (long long)ctas * n_sm / heads, (long long)N / STAT_MIN})), false};
}

}  // namespace mpfa
