// How many CTAs an RVE gets in FP64 (plain host code; the tests compile it by itself).
//
// The FP64 pipe is 2 operations per clock and SM, so RVEs that leave SMs idle are
// spread over more of them, up to 16 CTAs each as long as a part keeps kSplitNodes
// nodes: below that the latency of an iteration (3.5 us) is no longer the
// work's. One RVE, us per iteration: 512 nodes on 1 CTA 13.0, on 8 5.0, on 16 5.3;
// 700 nodes on 1 CTA 17, on 8 5.6, on 16 5.3 (taken with the sums of before; now 3.5 for
// both on 8 and 16); 5000 nodes on 8 CTAs 15.8, on 16 9.7.
//
// max_cluster is the largest cluster that the device can hold (fp64_max_cluster): a
// larger one could never be placed, and such an RVE runs on fewer CTAs.
#pragma once
#include <stdint.h>

namespace fe2 {

constexpr int kMaxSplit = 16;  // CTAs of one RVE
constexpr int kSplitNodes = 40;

// Largest factor by which an RVE's n_parts parts may be divided, whatever its batch.
// The parts divided so are its leaves: the sums go leaf by leaf, so results are
// the same bits for any split.
inline int fp64_leaf_factor(int n_nodes, int n_parts) {
    int f = 1;
    while (2 * f * n_parts <= kMaxSplit && n_nodes >= 2 * f * n_parts * kSplitNodes) f *= 2;
    return f;
}

// Groups into which a leaf's terms are divided before they are summed: about 64
// nodes each, at most 16 to a CTA that holds a whole part.
inline int fp64_groups(int n_nodes, int n_parts, int leaves) {
    int g = 1;
    while (2 * g * (leaves / n_parts) <= kMaxSplit && n_nodes >= 2 * g * leaves * 64) g *= 2;
    return g;
}

// Factor taken in a batch of `ctas` parts: up to 128 CTAs in all.
inline int fp64_split_factor(int64_t ctas, int n_nodes, int n_parts, int max_cluster) {
    const int most = fp64_leaf_factor(n_nodes, n_parts);
    int f = 1;
    while (2 * f * ctas <= 128 && 2 * f <= most && 2 * f * n_parts <= max_cluster) f *= 2;
    return f;
}

// CTAs of the allocation-free call.
inline int fp64_single_parts(int n_nodes, int max_cluster) {
    int c = 1;
    while (2 * c <= kMaxSplit && 2 * c <= max_cluster && n_nodes >= 2 * c * kSplitNodes) c *= 2;
    return c;
}

}  // namespace fe2
