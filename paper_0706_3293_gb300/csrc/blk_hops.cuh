// blk_hops.cuh -- the exchange targets of a row of the block path (blk.cuh) as lists, for kernels
// in which several lanes share a row (one lane or a few a vector: ftlm.cu, blk_multi.cu).
//
// The low part of every block of class k (k ones) runs through the same low words, so the
// ranks that its low exchanges reach stand in a table, once per layout: row g (position in the
// word list BlkParams::lw) has, in 16-bit entries, the number of low targets of each class as four
// bytes and an entry for each of the first HOP_XHEAD low ends of cross bonds (the rank of l ^ 2^p
// among the words of its popcount), then from seg[c] on the low targets of class c in the
// order of the bond groups, padded to a multiple of four with the row's own rank, then from
// xs on the entries of the other low ends.  A target then takes a shift, an address and the gather;
// finding it takes masks, a bit scan, an xor and two table lookups, by all lanes of the row.
// High and cross exchanges are listed once per block (hops_setup_high, hops_setup_cross).
#pragma once

#include "blk.cuh"

namespace hm {

constexpr int HOP_XHEAD = 6;

struct HopTab {
    int stride, seg[HM_BLK_MAXC], xs, nx;
    uint8_t xp[HM_BLK_MAXB], xi[HM_BLK_MAXB];   // the low ends of cross bonds; that of each cross bond
};

inline HopTab hop_layout(const BlkParams &P) {
    HopTab h{};
    int o = 2 + HOP_XHEAD;
    for (int c = 0; c < P.nc; ++c) {
        int m = 0;
        for (int g = P.lg_cs[3 * c]; g < P.lg_cs[3 * c + 3]; ++g) m += __builtin_popcount(P.lg_mask[g]);
        h.seg[c] = o;
        o += (m + 3) & ~3;
    }
    h.xs = o;
    for (int e = 0; e < P.ncb; ++e) {
        int i = 0;
        while (i < h.nx && h.xp[i] != P.cb_p[e]) ++i;
        if (i == h.nx) h.xp[h.nx++] = P.cb_p[e];
        h.xi[e] = (uint8_t)i;
    }
    h.stride = (o + (h.nx > HOP_XHEAD ? h.nx - HOP_XHEAD : 0) + 7) & ~7;
    return h;
}

// row g of the table
__device__ __forceinline__ void hop_fill(const BlkParams &P, const HopTab &H, uint32_t g, uint16_t *table) {
    BlkTabs tb;
    tb.U = (const uint16_t *)((const unsigned char *)P.tab + P.off_U);
    tb.R0 = (const uint8_t *)P.tab + P.off_R0;
    tb.C = (const uint32_t *)((const unsigned char *)P.tab + P.off_C);
    const uint32_t l = P.lw[g];
    const int k = __popc(l);
    const uint32_t r = g - (uint32_t)P.lwoff[k];
    uint16_t *T = table + (size_t)g * H.stride;
    for (int c = 0; c < HM_BLK_MAXC; ++c) {
        int m = 0;
        if (c < P.nc) {
            uint16_t *t = T + H.seg[c];
            blk_low_hops(P, tb, c, l, r, tb.U + k * P.nb1, [&](uint32_t r2) { t[m++] = (uint16_t)r2; });
            for (int i = m; i & 3; ++i) t[i] = (uint16_t)r;
        }
        ((uint8_t *)T)[c] = (uint8_t)m;
    }
    for (int i = 0; i < H.nx; ++i) {
        const uint32_t l2 = l ^ (1u << H.xp[i]);
        T[i < HOP_XHEAD ? 2 + i : H.xs + i - HOP_XHEAD] = (uint16_t)rank_low(P, tb, l2, __popc(l2));
    }
}

// the exchange lists of a block
struct Hops {
    int4 *x;              // [ncb] cross bond: {target block's rows less own, xor | test mask << 16, low end, 0}
    int *hcd;             // [nhb] offsets (target row - own row) of the valid high exchanges
    int *hcs;             // [HM_BLK_MAXC + 1] class c owns hcd[hcs[c] .. hcs[c+1])
};
__host__ __device__ __forceinline__ size_t hops_bytes(const BlkParams &P) {
    return ((size_t)P.ncb * 16 + (size_t)(P.nhb + HM_BLK_MAXC + 1) * 4 + 15) & ~(size_t)15;
}
__device__ __forceinline__ Hops hops_carve(const BlkParams &P, void *p) {
    Hops s;
    s.x = (int4 *)p;
    s.hcd = (int *)(s.x + P.ncb);
    s.hcs = s.hcd + P.nhb;
    return s;
}

// Hop lists of block (h, k), by one warp: the valid high exchanges as row offsets,
// compacted by class (lane e tests bonds e and e + 32, ballots give the positions), and
// the targets of the cross exchanges (hops_setup_cross).  The caller syncs before and after.
__device__ __forceinline__ void hops_setup_high(const BlkParams &P, const BlkTabs &tb, uint32_t h, int k, uint32_t off,
                                                const Hops &sh, int lane) {
    int val[2] = {0, 0}, hoff[2] = {0, 0};
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int e = lane + 32 * half;
        if (e < P.nhb) {
            const int p = P.hb_p[e], q = P.hb_q[e];
            val[half] = (((h >> p) ^ (h >> q)) & 1u) ? 1 : 0;
            if (val[half]) hoff[half] = (int)(blk_off(P, tb, h ^ ((1u << p) | (1u << q)), k) - off);
        }
    }
    const uint32_t b0 = __ballot_sync(0xffffffffu, val[0]), b1 = __ballot_sync(0xffffffffu, val[1]);
    const uint32_t below = (1u << lane) - 1u;
    if (val[0]) sh.hcd[__popc(b0 & below)] = hoff[0];
    if (val[1]) sh.hcd[__popc(b0) + __popc(b1 & below)] = hoff[1];
    if (lane <= HM_BLK_MAXC) {                    // class c starts at the valid ones before hb_start[c]
        const int e = P.hb_start[lane];
        sh.hcs[lane] = e >= 32 ? __popc(b0) + __popc(e >= 64 ? b1 : b1 & ((1u << (e - 32)) - 1u))
                               : __popc(b0 & ((1u << e) - 1u));
    }
}
__device__ __forceinline__ void hops_setup_cross(const BlkParams &P, const HopTab &H, const BlkTabs &tb, uint32_t h, int k,
                                                 uint32_t off, const Hops &sh, int lane) {
    for (int e = lane; e < P.ncb; e += 32) {
        const int p = P.cb_p[e], q = P.cb_q[e];
        const uint32_t bq = (h >> q) & 1u;
        const int k2 = k + (bq ? 1 : -1);
        const bool ok = k2 >= 0 && k2 <= P.K;     // else the test mask is empty
        sh.x[e] = make_int4(ok ? (int)(blk_off(P, tb, h ^ (1u << q), k2) - off) : 0,
                            (int)((bq << p) | (ok ? 1u << (p + 16) : 0u)), H.xi[e], 0);
    }
}

// row offset (target - first row of the own block) of cross exchange x for a row whose table row T
// starts with hd, and whether low word l allows it
__device__ __forceinline__ bool hop_cross(const HopTab &H, const int4 &x, const uint4 &hd, const uint16_t *T, uint32_t l,
                                          int *target) {
    const uint32_t xw = x.z < 2 ? hd.y : x.z < 4 ? hd.z : hd.w;
    int t2 = (int)((x.z & 1) ? xw >> 16 : xw & 0xFFFFu);
    if (x.z >= HOP_XHEAD) t2 = (int)__ldg(T + H.xs + x.z - HOP_XHEAD);
    *target = x.x + t2;
    return ((l ^ (uint32_t)x.y) & ((uint32_t)x.y >> 16)) != 0u;
}

}  // namespace hm
