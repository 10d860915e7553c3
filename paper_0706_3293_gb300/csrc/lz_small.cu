// lz_small.cu -- whole FP64 Lanczos runs of small s = 1/2 sectors in one cooperative kernel.
//
// A step of a small sector is bound by latency: three launches of 22 us together (N = 16, 12,870
// rows; captured in a graph, whose capture costs the host another 10 us a step), of which the
// arithmetic is under two.  Here every block of the block path (blk.cuh) belongs to one CTA for the
// whole run.  Its rows of q_cur and q_prev stay in registers and the fixed-point copy of q_cur in
// shared memory; the block's exchange targets are set up once; other blocks' values are gathered
// from the global fixed-point copy.  A step has three grid barriers: after the product's dot
// (alpha_j), after the update's norm, dot and largest exponent (beta_j and the next fixed-point
// unit), and after the new fixed-point copy.  Every CTA forms alpha_j and beta_j itself, from the
// same partial sums in the same order.  Rows, sums and their order are those of the step-wise path, so
// both give the same bits.  Measured per step of a run, host included: N = 16 28.5 -> 14 us,
// N = 18 32 -> 14, N = 20 44 -> 22.  From N = 21 the sector has more blocks than CTAs fit.
#include <algorithm>

#include "lz_small.cuh"

namespace hm {

namespace {

constexpr int LZS_R = 2;             // rows of a thread at most: t and t + BLK_NT

struct GFixCg {                      // fixed-point copy, written during the kernel: no read-only path
    __device__ __forceinline__ int64_t operator()(const unsigned char *p) const {
        return (int64_t)__ldcg((const long long *)p);
    }
};

// row sum of a per-bond plan with its target table: low slots, cross slots, high list (A: PbSum or PbSumW)
template <class A>
__device__ __forceinline__ A lzs_row_pb(const BlkParams &P, const BlkMeta &B, const unsigned char *Xsb,
                                        const unsigned char *Xg, uint32_t l, uint32_t r, int64_t xo) {
    const GFixCg gx;
    A a(0);
    const uint32_t g = B.lwo + r;
    const uint4 *tt = P.tt + g;
    for (int e0 = 0; e0 < P.tt_nsgl; e0 += 8, tt += P.tt_stride) {
        const uint4 q = ldg_v4(tt);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (e0 + k >= P.tt_nsgl) break;
            const uint32_t o = k & 1 ? w[k >> 1] >> 16 : w[k >> 1] & 0xFFFFu;
            const int b = P.tt_pb[e0 + k];
            a = pb_mac(P.pb_cl[b], P.pb_ch[b], P.pb_cw[b], xo - *(const int64_t *)(Xsb + o), a);
        }
    }
    for (int t = 0; t < 2; ++t)
        for (int s = 0; s < P.xn[0][t]; ++s) {
            const int d = t * HM_BLK_SX + s;
            const XSlot x_ = B.xs[d];
            if ((l ^ x_.wm) & x_.vm) {
                const int e = P.tt_xe[d], b = P.pb_xb[t][s];
                const uint32_t v_ = __ldg((const uint16_t *)P.tt + ((size_t)(e >> 3) * P.tt_stride + g) * 8 + (e & 7));
                a = pb_mac(P.pb_cl[b], P.pb_ch[b], P.pb_cw[b], xo - gx(x_.base + v_), a);
            }
        }
    return blk_high_pb<int64_t>(P, B, Xg, r, gx, xo, a);
}

// all CTAs past their writes; false when a barrier gave up.  bar[0] counts arrivals (never reset:
// barrier k ends at k ctas), bar[1] is the abort flag.  A limit of 0 waits for nobody: CTAs that
// are not alone give up
__device__ __forceinline__ bool lzs_barrier(unsigned *bar, unsigned target, unsigned long long limit_ns) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        volatile unsigned *v = bar;
        int ok = 1;
        if (limit_ns == 0 && gridDim.x > 1) {
            atomicExch(bar + 1, 1u);
            ok = 0;
        } else if (*v < target) {
            unsigned long long t0, t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
            for (unsigned spin = 1; *v < target; ++spin) {
                if (spin & 31u) continue;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if (v[1] || t - t0 > limit_ns) { atomicExch(bar + 1, 1u); ok = 0; break; }
            }
        }
        __threadfence();
        s_ok = ok && !v[1];
    }
    __syncthreads();
    return s_ok != 0;
}

// NC: coupling classes (1, 2, 4), or 0 for a per-bond plan, -1 for one with low parts (pb_wide)
template <int NC, bool PSI>
__global__ void __launch_bounds__(BLK_NT, 2) k_lz_small(BlkParams P, LzSmallArgs a) {
    if (a.S->done) return;
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr bool PB = NC <= 0;
    constexpr int NCA = PB ? 1 : NC;
    const int tid = threadIdx.x, nt = blockDim.x, ctas = gridDim.x, nh = 1 << P.H;
    int64_t *Xs = (int64_t *)smem;
    BlkMeta &B = *(BlkMeta *)(smem + blk_row_xs_bytes(P, 8, BLK_XPAD));
    BlkMetaX *BX = PB ? (BlkMetaX *)((unsigned char *)&B + 2 * al16(sizeof(BlkMeta))) : nullptr;
    __shared__ uint32_t s_h;
    __shared__ double red[BLK_NT / 32], s_cj;
    __shared__ ef::df s_as, s_sg, s_gm;              // scalars of the update, from warp 0 (s_dq: warp 1)
    __shared__ int s_emax, s_stop;
    const unsigned char *Xg = (const unsigned char *)a.X;
    const GFixCg gx;
    BlkTabs tb;
    tb.U = nullptr; tb.R0 = nullptr;
    tb.C = (const uint32_t *)((const unsigned char *)P.tab + P.off_C);
    // the CTA's block: the blockIdx.x-th high word whose low part holds the rest of the ones
    if (tid == 0) {
        int left = blockIdx.x;
        uint32_t h = 0;
        while (!blk_h_valid(P, h) || left-- > 0) ++h;
        s_h = h;
        B.hv[0] = B.hv[1] = 0u;
    }
    if (tid == 0) Xs[P.max_block + BLK_XPAD - 1] = 0;
    __syncthreads();
    const uint32_t h = s_h;
    const int k = P.A - __popc(h);
    // targets of the high and cross exchanges, as blk_sweep sets them up for each block
    for (int e = tid; e < P.nhb; e += nt)
        if (((h >> P.hb_p[e]) ^ (h >> P.hb_q[e])) & 1u) atomicOr(&B.hv[e >> 5], 1u << (e & 31));
    for (int e = tid; e < P.nxf; e += nt) {
        const int p = P.xf_p[e], q = P.xf_q[e];
        const uint32_t bq = (h >> q) & 1u;
        const int k2 = k + (bq ? 1 : -1);
        const bool ok = k2 >= 0 && k2 <= P.K;
        XSlot xs;
        xs.base = ok ? Xg + (size_t)blk_off(P, tb, h ^ (1u << q), k2) * 8 : Xg;
        xs.wm = (uint16_t)(bq << p);
        xs.vm = (uint16_t)(ok ? 1u << p : 0u);
        xs.kofs2 = 0u;
        B.xs[P.xf_dst[e]] = xs;
    }
    if (tid == 0) {
        B.x = BX;
        B.off = blk_off(P, tb, h, k);
        B.n = tb.C[P.K * (P.A + 1) + k];
        B.kofs = (uint32_t)k << P.kshift;
        B.lwo = (uint32_t)P.lwoff[k];
    }
    __syncthreads();
    const uint64_t hm = ((uint64_t)B.hv[1] << 32) | B.hv[0];
    for (int e = tid; e < max(P.nhb, HM_BLK_MAXC); e += nt) {
        int start = 0;                               // each class's run padded to a multiple of 4 entries
        for (int c = 0; c < HM_BLK_MAXC; ++c) {
            const int b0 = popc_below(hm, P.hb_start[c]), b1 = popc_below(hm, P.hb_start[c + 1]);
            if (e < P.nhb && e >= P.hb_start[c] && e < P.hb_start[c + 1] && ((hm >> e) & 1ull)) {
                const int i = start + popc_below(hm, e) - b0;
                B.hbi[i] = blk_off(P, tb, h ^ ((1u << P.hb_p[e]) | (1u << P.hb_q[e])), k);
                if (PB) {
                    BX->hbc[i] = make_int2(P.pb_cl[P.pb_hbb[e]], P.pb_ch[P.pb_hbb[e]]);
                    BX->hbcf[i] = P.pb_cw[P.pb_hbb[e]];
                }
            }
            if (e == c) {
                B.hs[c] = start;
                B.he[c] = start + (b1 - b0);
                if (PB) BX->fs[c] = BX->fe[c] = 0;
            }
            start += (b1 - b0 + 3) & ~3;
        }
    }
    const uint32_t off = B.off, n = B.n;
    float2 q[LZS_R], p[LZS_R];
    uint32_t low[LZS_R];
#pragma unroll
    for (int j = 0; j < LZS_R; ++j) {
        const uint32_t r = tid + j * BLK_NT;
        q[j] = p[j] = make_float2(0.0f, 0.0f);
        low[j] = 0u;
        if (r < n) {
            q[j] = a.q0[off + r];
            low[j] = P.lw[B.lwo + r];
            Xs[r] = a.X[off + r];
        }
    }
    __syncthreads();
    unsigned *bar = (unsigned *)(a.pe + nh), nbar = 0;
    int E = a.S->emax[0], steps = 0, status = HM_OK;
    // the binary64 scalars live in warp 0 alone: an instruction on them costs every warp of the CTA 64
    // cycles of its quarter of the SM
    double sg = 0.0, gm = 0.0, scale = 0.0, al = 0.0;
    __shared__ double s_dq;
    auto todf = [](double v) { const float f = (float)v; return ef::df{f, (float)(v - (double)f)}; };
    if (tid == 0) {
        sg = a.S->sigma_cur;
        s_sg = todf(sg);
        s_gm = ef::df{0.0f, 0.0f};
        s_dq = 0.0;
    }
    for (int js = 0; js < a.steps; ++js) {
        // product and q.Hq
        const int u = E - 1022 - ef::FIX_BITS;
        unsigned long long yb[LZS_R];
        __int128 d1 = 0;
        ef::df d1f{0.0f, 0.0f};
        const bool exact_dot = !PB && P.iratio;
        const double sy = PB ? ef::pow2d(u - P.pb_s) : 0.0;
#pragma unroll
        for (int j = 0; j < LZS_R; ++j) {
            const uint32_t r = tid + j * BLK_NT;
            yb[j] = 0ull;
            if (r >= n) continue;
            const int64_t xo = Xs[r];
            if constexpr (PB) {
                const auto sv = lzs_row_pb<typename PbAcc<int64_t, NC == -1>::T>(P, B, smem, Xg, low[j], r, xo);
                yb[j] = ef::d2u(i128_to_double(sv.row(P, xo)) * sy);
            } else {
                int64_t acc[NCA], Tc[NCA], ts = 0;
                int cnt[NCA];
                RowTable<NCA>::template sums<int64_t>(P, B, smem, Xg, low[j], r, gx, xo, acc, cnt);
                blk_classes<NCA>(P, acc, cnt, xo, Tc);
                yb[j] = blk_y_bits<NCA>(P, Tc, u, &ts);
                d1 += (__int128)xo * ts;
            }
            if (!exact_dot)
                d1f = ef::df_add(d1f, ef::df_mul(ef::df_from_fix(xo, E, 0, E - 1023), ef::df_from_bits(yb[j], E - 1023)));
        }
        {
            const double t = blk_dot_warp(exact_dot, d1, d1f);
            if (tid < BLK_NT / 32) red[tid] = 0.0;
            __syncthreads();
            if ((tid & 31) == 0) red[tid >> 5] = t;
            __syncthreads();
            if (tid < 32) {
                double v = red[tid & 15];
                for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (tid == 0) a.pa[h] = blk_dot_scaled(P, exact_dot, E, v);
            }
        }
        if (!lzs_barrier(bar, ++nbar * ctas, a.limit_ns)) { status = HM_ETIMEOUT; break; }
        if (tid < 32) {
            const double s1 = warp_sum_of(a.pa, nh);
            if (tid == 0) {
                al = sg * sg * s1 - sg * gm * s_dq;
                scale = fmax(scale, fabs(al));
                s_as = todf(al * sg);
                if constexpr (PSI) s_cj = a.coef[js] * sg;
            }
        }
        __syncthreads();
        // w = sigma y - alpha sigma q - gamma q_prev, |w|^2, w.q and the largest exponent
        const ef::df sg_d = s_sg, as_d = s_as, gm_d = s_gm;
        ef::df nn{0.0f, 0.0f}, dq{0.0f, 0.0f};
        uint32_t eh = 0;
        const double cj = PSI ? s_cj : 0.0;
#pragma unroll
        for (int j = 0; j < LZS_R; ++j) {
            const uint32_t r = tid + j * BLK_NT;
            if (r >= n) continue;
            const float2 w = lz_row_update(yb[j], q[j], p[j], sg_d, as_d, gm_d, nn, dq, eh);
            if constexpr (PSI) a.psi[off + r] += cj * ((double)q[j].x + (double)q[j].y);
            p[j] = q[j];
            q[j] = w;
        }
        {
            int em = 0;
            const double t = lz_block_sums(nn, dq, eh, &em);
            if (tid == 0) {
                a.pn[h] = t;
                a.pe[h] = em;
            } else if (tid == 16) {
                a.pd[h] = t;
                __threadfence();
            }
        }
        if (!lzs_barrier(bar, ++nbar * ctas, a.limit_ns)) { status = HM_ETIMEOUT; break; }
        if (tid < 32) {
            const double s2 = warp_sum_of(a.pn, nh);
            if (tid == 0) {
                const double be = sqrt(s2);
                if (blockIdx.x == 0) { a.alpha[js] = al; a.beta[js] = be; }
                s_stop = be <= a.tol * scale;
                scale = s_stop ? scale : fmax(scale, be);
                gm = be * sg;                        // beta_j sigma_j: the next q_prev is this q
                sg = 1.0 / be;
                s_sg = todf(sg);
                s_gm = todf(gm);
            }
        } else if (tid < 64) {
            const double s3 = warp_sum_of(a.pd, nh);
            int em = 0;
            for (int i = tid & 31; i < nh; i += 32) em = max(em, __ldcg(a.pe + i));
            em = __reduce_max_sync(0xffffffffu, em);
            if (tid == 32) { s_dq = s3; s_emax = em; }
        }
        __syncthreads();
        steps = js + 1;
        if (s_stop) { status = HM_BREAKDOWN; break; }
        E = s_emax ? s_emax - 127 + 1023 : 0;
        if (js + 1 == a.steps) break;
#pragma unroll
        for (int j = 0; j < LZS_R; ++j) {
            const uint32_t r = tid + j * BLK_NT;
            if (r >= n) continue;
            const int64_t x = ef::fix_from_df(ef::df{q[j].x, q[j].y}, E, 0);
            Xs[r] = x;
            __stcg(a.X + off + r, (long long)x);
        }
        if (!lzs_barrier(bar, ++nbar * ctas, a.limit_ns)) { status = HM_ETIMEOUT; break; }
    }
    if (status == HM_ETIMEOUT) {
        if (tid == 0) a.S->status = HM_ETIMEOUT;
    } else if (blockIdx.x == 0 && tid == 0) {
        a.S->j = steps;
        a.S->scale = scale;
        a.S->status = status;
        a.S->done = status == HM_BREAKDOWN;
    }
}

const void *lzs_kernel(const BlkParams &P, bool psi) {
    if (P.perbond && P.pb_wide) return psi ? (const void *)k_lz_small<-1, true> : (const void *)k_lz_small<-1, false>;
    if (P.perbond) return psi ? (const void *)k_lz_small<0, true> : (const void *)k_lz_small<0, false>;
    if (P.nc == 1) return psi ? (const void *)k_lz_small<1, true> : (const void *)k_lz_small<1, false>;
    if (P.nc == 2) return psi ? (const void *)k_lz_small<2, true> : (const void *)k_lz_small<2, false>;
    return psi ? (const void *)k_lz_small<4, true> : (const void *)k_lz_small<4, false>;
}

}  // namespace

int lz_small_plan(const BlkParams &P, LzSmall *out) {
    if (!P.tt || P.split || P.bcmode || P.par || P.H > LZS_MAX_H || P.max_block > LZS_R * BLK_NT) return 1;
    int ctas = 0;
    for (uint32_t h = 0; h < (1u << P.H); ++h) {
        const int k = P.A - __builtin_popcount(h);
        ctas += k >= 0 && k <= P.K;
    }
    if (ctas < 1) return 1;
    out->P = P;
    out->ctas = ctas;
    // whole warps for the rows of the largest block, and two for the sums
    out->threads = std::max(64, std::min(BLK_NT, (P.max_block + 31) & ~31));
    out->smem = blk_row_smem_bytes(P, 8, BLK_XPAD);
    for (bool psi : {false, true}) {
        const void *kern = lzs_kernel(P, psi);
        HM_CUDA(raise_smem_limit(kern, out->smem));
        int per = 0;
        HM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, out->threads, out->smem));
        if (per * sm_count() < ctas) return 1;       // cooperative: all CTAs resident
    }
    return 0;
}

int lz_small_launch(const LzSmall &L, const LzSmallArgs &a, cudaStream_t st) {
    HM_CUDA(cudaMemsetAsync(a.pe, 0, lz_small_bytes(L.P.H), st));
    void *args[] = {(void *)&L.P, (void *)&a};
    HM_CUDA(cudaLaunchCooperativeKernel(lzs_kernel(L.P, a.psi != nullptr), dim3(L.ctas), dim3(L.threads), args, L.smem, st));
    return HM_OK;
}

}  // namespace hm
