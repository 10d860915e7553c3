// lz_small.cuh -- whole FP64 Lanczos runs of small s = 1/2 sectors in one cooperative kernel
// (lz_small.cu); used by lanczos_run and e0_grad (lanczos.cu).
#pragma once

#include "blk.cuh"
#include "blk_sweep.cuh"

namespace hm {

constexpr int LZS_MAX_H = 10;    // such a sector has at most 2^10 blocks, of at most 2 BLK_NT rows

struct LzSmall {
    BlkParams P;                 // with its target table (tt)
    int ctas, threads;           // one CTA a block of the sector
    size_t smem;
};

struct LzSmallArgs {
    long long *X;                // fixed-point copy of q_cur (start vector: k_fix_start)
    const float2 *q0;            // start vector as double-float pairs
    LzScalars *S;
    double *alpha, *beta;
    double *pa, *pn, *pd;        // per block h: q.Hq, |w|^2, w.q; zero for absent blocks
    int *pe;                     // per block: largest exponent of w; then two unsigned (barrier, abort)
    double *psi;                 // psi += coef_j v_j, or NULL
    const double *coef;
    int steps;
    double tol;
    unsigned long long limit_ns; // a barrier gives up after this long
};

// bytes of LzSmallArgs::pe and what follows it (zeroed by lz_small_launch)
inline size_t lz_small_bytes(int H) { return ((size_t)4 << H) + 16; }
// The plan for a block plan of an FP64 run, or 1 when such a run goes step by step.  Sectors with a plan
// take their update by blocks also in step-wise runs (k_lz_update_blk), and add as this kernel
// does, so that both forms give the same bits.
int lz_small_plan(const BlkParams &P, LzSmall *out);
int lz_small_launch(const LzSmall &L, const LzSmallArgs &a, cudaStream_t st);

#ifdef __CUDACC__
// one row of w = sigma y - alpha sigma q - gamma q_prev (yb: binary64 bits of (H q)_i) in double-float,
// |w|^2 and w.q added to nn and dq, the exponent field to eh
__device__ __forceinline__ float2 lz_row_update(unsigned long long yb, float2 q2, float2 p2, ef::df sg, ef::df as,
                                                ef::df gm, ef::df &nn, ef::df &dq, uint32_t &eh) {
    const ef::df q = ef::df{q2.x, q2.y};
    const ef::df t1 = ef::df_mul(sg, ef::df_from_bits(yb, 0));
    const ef::df t2 = ef::df_mul(as, q);
    const ef::df t3 = ef::df_mul(gm, ef::df{p2.x, p2.y});
    const ef::df w = ef::df_add(t1, ef::df_neg(ef::df_add(t2, t3)));
    eh = max(eh, (ef::f2u(w.hi) >> 23) & 0xFFu);
    nn = ef::df_add(nn, ef::df_mul(w, w));
    dq = ef::df_add(dq, ef::df_mul(w, q));
    return make_float2(w.hi, w.lo);
}

// a block's |w|^2, w.q and largest exponent from those of its threads (whole warps, at most BLK_NT
// threads), by shuffle trees over the lanes and then over the warps; valid in lanes 0 (tn) and 16 (td)
// of warp 0, *em in all its lanes.  The lower lanes add one sum, the upper the other: a binary64 add
// occupies the pipe for 64 cycles whichever lanes take part.
__device__ __forceinline__ double lz_block_sums(ef::df nn, ef::df dq, uint32_t eh, int *em) {
    __shared__ double red[2][BLK_NT / 32];
    __shared__ uint32_t s_em[BLK_NT / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const double vn = (double)nn.hi + (double)nn.lo, vd = (double)dq.hi + (double)dq.lo;
    // both halves exchange what the other one adds
    const double give = lane < 16 ? vd : vn, got = __shfl_xor_sync(0xffffffffu, give, 16);
    double v = (lane < 16 ? vn : vd) + got;
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    eh = __reduce_max_sync(0xffffffffu, eh);
    if ((lane & 15) == 0) red[lane >> 4][warp] = v;
    if (lane == 0) s_em[warp] = eh;
    __syncthreads();
    v = 0.0;
    if (warp == 0) {
        const int w = lane & 15;
        v = w < nw ? red[lane >> 4][w] : 0.0;
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        *em = (int)__reduce_max_sync(0xffffffffu, w < nw ? s_em[w] : 0u);
    }
    return v;
}
#endif

}  // namespace hm
