// blk_fit.h -- whether a bond list fits the slots of the thread-per-row kernels at a split position
// (blk_params.cuh), and the smallest split that holds it.  Host only, no CUDA headers.
#pragma once

#include <map>
#include <utility>

namespace hm {

// HM_BLK_SL low bonds for each class and byte type, HM_BLK_SX cross bonds for each class and byte of their
// low end, HM_BLK_SG distances among the low bonds of a class.  Bonds p[t] < q[t] of class cls[t].
inline bool blk_slots_fit(int nb, const unsigned char *p, const unsigned char *q, const int *cls, int K, int sl, int sx,
                          int sg) {
    if (K > 15) return false;
    std::map<std::pair<int, int>, int> low, cross;      // (class, type) -> bonds
    std::map<int, unsigned> dist;                       // class -> the distances of its low bonds
    for (int t = 0; t < nb; ++t) {
        if (q[t] < K) {
            if (++low[{cls[t], q[t] < 8 ? 0 : p[t] >= 8 ? 1 : 2}] > sl) return false;
            dist[cls[t]] |= 1u << (q[t] - p[t]);
        } else if (p[t] < K) {
            if (++cross[{cls[t], p[t] < 8 ? 0 : 1}] > sx) return false;
        }
    }
    for (const auto &d : dist)
        if (__builtin_popcount(d.second) > sg) return false;
    return true;
}

// The smallest K in k0 .. kmax whose slots hold the list, or k0 when none does.  A smaller K turns low
// bonds into cross bonds, which have half the slots: two-dimensional clusters, ladders and rings with far
// neighbours fit only from some K on.
inline int blk_fitting_K(int nb, const unsigned char *p, const unsigned char *q, const int *cls, int k0, int kmax, int sl,
                         int sx, int sg) {
    for (int K = k0; K <= kmax; ++K)
        if (blk_slots_fit(nb, p, q, cls, K, sl, sx, sg)) return K;
    return k0;
}

}  // namespace hm
