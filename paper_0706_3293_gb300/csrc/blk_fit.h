// blk_fit.h -- whether a bond list fits the slots of the thread-per-row kernels at a split position
// (blk_params.cuh), and the smallest split that holds it.  Host only, no CUDA headers.
#pragma once

namespace hm {

// HM_BLK_SL low bonds for each class and byte type, HM_BLK_SX cross bonds for each class and byte of their
// low end, HM_BLK_SG distances among the low bonds of a class.  Bonds p[t] < q[t] < 32 of class cls[t] < 4.
inline bool blk_slots_fit(int nb, const unsigned char *p, const unsigned char *q, const int *cls, int K, int sl, int sx,
                          int sg) {
    if (K > 15) return false;
    int low[4][3] = {}, cross[4][2] = {};
    unsigned dist[4] = {};                              // the distances of a class's low bonds
    for (int t = 0; t < nb; ++t) {
        const int c = cls[t];
        if (q[t] < K) {
            if (++low[c][q[t] < 8 ? 0 : p[t] >= 8 ? 1 : 2] > sl) return false;
            dist[c] |= 1u << (q[t] - p[t]);
        } else if (p[t] < K) {
            if (++cross[c][p[t] < 8 ? 0 : 1] > sx) return false;
        }
    }
    for (unsigned d : dist)
        if (__builtin_popcount(d) > sg) return false;
    return true;
}

// The smallest K in k0 .. kmax whose slots hold the list, or -1 when none does.  A smaller K turns low
// bonds into cross bonds, which have half the slots: two-dimensional clusters, ladders and rings with far
// neighbours fit only from some K on.
inline int blk_fitting_K(int nb, const unsigned char *p, const unsigned char *q, const int *cls, int k0, int kmax, int sl,
                         int sx, int sg) {
    for (int K = k0; K <= kmax; ++K)
        if (blk_slots_fit(nb, p, q, cls, K, sl, sx, sg)) return K;
    return -1;
}

}  // namespace hm
