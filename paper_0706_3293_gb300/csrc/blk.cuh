// blk.cuh -- block-structured row kernel for s = 1/2 sectors (shared by the matvec API,
// the Lanczos step and the batched finite-temperature driver).
//
// The sector states of N spins s = 1/2 with A flipped spins are the N-bit words of
// popcount A in increasing numerical order (Sec. 3: position N most significant).  Split
// a word into its high part h (positions K..N-1) and its low part l (positions 0..K-1).
// The rank of Sec. 3.2 is additive over positions, so
//     index(h, l) = off(h) + rank_K(l),   off(h) = sum over the ones of h of C(t, cnt),
// and all states with the same h form one contiguous block of C(K, A - popc(h)) rows.
// The kernel processes one block per CTA iteration:
//   * off(h) and the offsets of the blocks one exchange away are encoded once per block
//     with the paper's rank formula (D(p, c) = C(p, c) for s = 1/2);
//   * the low part is decoded and re-encoded with byte-chunk rank tables -- the same
//     rank sums of Sec. 3.2 precomputed 8 positions at a time:
//         rank_K(l) = U[popc(l)][l >> 8] + R0[l & 255];
//   * the block's own x values are staged in shared memory, so exchanges among the low
//     positions gather from shared memory; exchanges among the high positions move a
//     whole block to another block at a constant offset (coalesced gathers); exchanges
//     across the split touch one bit on each side.
// Couplings are grouped into classes of equal J (at most HM_BLK_MAXC).  In FP64 the
// hop sums of a class are exact int64 fixed-point sums (ef64.cuh), combined per row
// in double-float arithmetic: no FP64 instruction runs per row.
#pragma once

#include <climits>

#include "blk_params.cuh"
#include "ef64.cuh"
#include "hm_internal.cuh"

namespace hm {

// host: builds the plan; returns 0 if the bond list and sector take the fast path.  use:
// bit t set = bond t is applied (a pass of the two-pass product applies a subset; the
// coupling classes always come from the whole list, so both passes share them)
int blk_plan(hm_basis *b, const BondParams &bp, int K, BlkParams *out, bool bond_corr = false,
             uint64_t use = ~0ull);

// ---- device helpers ----------------------------------------------------------------------
__device__ __forceinline__ BlkTabs stage_blk_tables(const BlkParams &P, unsigned char *smem) {
    const uint32_t *src = (const uint32_t *)P.tab;
    uint32_t *dst = (uint32_t *)smem;
    for (int k = threadIdx.x; k < P.tab_bytes / 4; k += blockDim.x) dst[k] = src[k];
    BlkTabs t;
    t.U = (const uint16_t *)(smem + P.off_U);
    t.R0 = (const uint8_t *)(smem + P.off_R0);
    t.C = (const uint32_t *)(smem + P.off_C);
    return t;
}

__device__ __forceinline__ uint32_t rank_low(const BlkParams &P, const BlkTabs &T, uint32_t l, int k) {
    return (uint32_t)T.U[k * P.nb1 + (l >> 8)] + (uint32_t)T.R0[l & 255u];
}

}  // namespace hm

namespace hm {

// ---- low exchanges ----------------------------------------------------------------------
// f(r2) for every allowed exchange of class c among the low positions (targets in the
// same block); returns their number
template <class F>
__device__ __forceinline__ int blk_low_hops(const BlkParams &P, const BlkTabs &tb, int c, uint32_t l,
                                            uint32_t r, const uint16_t *Uk, F &&f) {
    const uint32_t R0own = tb.R0[l & 255u];
    const uint32_t R1own = r - R0own;
    int mc = 0;
    for (int g = P.lg_cs[3 * c]; g < P.lg_cs[3 * c + 1]; ++g) {        // inside byte 0
        const int d = P.lg_d[g];
        const uint32_t pat = 1u | (1u << d);
        uint32_t m = ((l >> d) ^ l) & P.lg_mask[g];
        while (m) {
            const int p = __ffs(m) - 1;
            m &= m - 1;
            f(R1own + tb.R0[(l ^ (pat << p)) & 255u]);
            ++mc;
        }
    }
    for (int g = P.lg_cs[3 * c + 1]; g < P.lg_cs[3 * c + 2]; ++g) {    // inside byte 1
        const int d = P.lg_d[g];
        const uint32_t pat = 1u | (1u << d);
        uint32_t m = ((l >> d) ^ l) & P.lg_mask[g];
        while (m) {
            const int p = __ffs(m) - 1;
            m &= m - 1;
            f(R0own + Uk[(l ^ (pat << p)) >> 8]);
            ++mc;
        }
    }
    for (int g = P.lg_cs[3 * c + 2]; g < P.lg_cs[3 * c + 3]; ++g) {    // across the bytes
        const int d = P.lg_d[g];
        const uint32_t pat = 1u | (1u << d);
        uint32_t m = ((l >> d) ^ l) & P.lg_mask[g];
        while (m) {
            const int p = __ffs(m) - 1;
            m &= m - 1;
            const uint32_t l2 = l ^ (pat << p);
            f((uint32_t)Uk[l2 >> 8] + tb.R0[l2 & 255u]);
            ++mc;
        }
    }
    return mc;
}

}  // namespace hm
