// blk_fit.h -- whether a bond list fits the slots of the thread-per-row kernels at a split position
// (blk_params.cuh), and the smallest split that holds it.  Host only, no CUDA headers.
#pragma once

namespace hm {

// how many earlier bonds of the list are the same pair of the same class (a torus two sites wide has its bonds
// twice): the groups of low bonds are masks of their lower ends, so that each repetition takes a group of its own
inline int blk_repetition(const unsigned char *p, const unsigned char *q, const int *cls, int t) {
    int n = 0;
    for (int i = 0; i < t; ++i) n += p[i] == p[t] && q[i] == q[t] && cls[i] == cls[t];
    return n;
}

// HM_BLK_SL low bonds for each class and byte type, HM_BLK_SX cross bonds for each class and byte of their
// low end, HM_BLK_SG distances among the low bonds of a class, those of a repetition counted again
// (own: a coefficient for each bond, whose rows take no groups).  Bonds p[t] < q[t] < 32 of class cls[t] < 4.
inline bool blk_slots_fit(int nb, const unsigned char *p, const unsigned char *q, const int *cls, bool own, int K, int sl,
                          int sx, int sg) {
    if (K > 15) return false;
    int low[4][3] = {}, cross[4][2] = {};
    unsigned dist[4][8] = {}, have[4][32] = {};         // by class: the distances of each repetition; the bonds so far
    for (int t = 0; t < nb; ++t) {
        const int c = cls[t];
        if (q[t] < K) {
            if (++low[c][q[t] < 8 ? 0 : p[t] >= 8 ? 1 : 2] > sl) return false;
            int r = 0;
            if (!own && (have[c][p[t]] >> q[t] & 1u)) r = blk_repetition(p, q, cls, t);
            if (r > 7) return false;
            have[c][p[t]] |= 1u << q[t];
            dist[c][r] |= 1u << (q[t] - p[t]);
        } else if (p[t] < K) {
            if (++cross[c][p[t] < 8 ? 0 : 1] > sx) return false;
        }
    }
    for (auto &d : dist) {
        int n = 0;
        for (unsigned m : d) n += __builtin_popcount(m);
        if (n > sg) return false;
    }
    return true;
}

// The smallest K in k0 .. kmax whose slots hold the list, or -1 when none does.  A smaller K turns low
// bonds into cross bonds, which have half the slots: two-dimensional clusters, ladders and rings with far
// neighbours fit only from some K on.
inline int blk_fitting_K(int nb, const unsigned char *p, const unsigned char *q, const int *cls, bool own, int k0, int kmax,
                         int sl, int sx, int sg) {
    for (int K = k0; K <= kmax; ++K)
        if (blk_slots_fit(nb, p, q, cls, own, K, sl, sx, sg)) return K;
    return -1;
}

}  // namespace hm
