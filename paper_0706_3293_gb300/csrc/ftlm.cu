// ftlm.cu -- finite-temperature Lanczos over all sectors of an s = 1/2 system in one
// persistent, cooperative launch (Jaklic and Prelovsek's estimator; the paper cites it
// as an application of the Lanczos machinery, Sec. 1).
//
// For every sector A (digit sum, M = N/2 - A) and start vector r = 0..R-1 a Lanczos run
// of up to `steps` steps starts from the +-1 vector of SplitMix64 stream (seed, A, r).
// All R runs of a sector share one product: a row's R vector entries sit in one
// 128-byte line (row-major [dim][32]), a warp serves VT rows with 32/VT lanes each, lane
// l of a row holding vectors l*VT .. l*VT+VT-1, so the codec of a row runs once per
// warp instruction for all of its vectors.  The rows of all sectors are cut into the
// blocks of blk.cuh (one high word, all low words).  Every warp owns an equal share of
// the rows (a fixed interval of the row order, cut on the host): it walks the blocks its
// rows fall in, builds their exchange lists itself and writes one partial sum per sector
// it touches, so no CTA barrier separates blocks and the sums come out in a fixed order.
// A step is four phases separated by grid barriers with bounded waits:
//   A  u = sigma H q - beta_prev sigma_prev q_prev over q_prev, alpha partials
//   B  alpha per (sector, vector): the sector's warp partials in order
//   C  w = u - alpha sigma q over q_prev, |w|^2 partials
//   D  beta, breakdown, sigma
// Then per (sector, vector) the eigenvalues of the tridiagonal T, the Ritz values theta_j, and
// the squares tau_j of the first components of its eigenvectors are formed on the device.  Finally
//   Z(T) = sum_A (D_A / R) sum_r sum_j tau e^{-(theta - e_ref)/T},
//   E(T) = [same with theta inside] / Z(T)     (Z returned relative to e^{-e_ref/T}).
#include <algorithm>
#include <cstdlib>
#include <climits>
#include <cmath>
#include <cstring>
#include <map>
#include <vector>

#include "blk_hops.cuh"
#include "tridiag.cuh"

namespace hm {

__host__ __device__ __forceinline__ size_t al16f(size_t x) { return (x + 15) & ~(size_t)15; }

constexpr int FT_NT = 512;          // threads per CTA of the persistent kernel
// CTAs per SM the register budget is cut for: with two (64 registers) the widest tiling spills little,
// with three (40) its four gathers in flight and eight sums spill at every row: 463 against 510 us a
// step of the N = 20 run, 151 against 178 at N = 18
#ifndef HM_FT_CTAS
#define HM_FT_CTAS 2
#endif
constexpr int FT_CTAS = HM_FT_CTAS;
constexpr int FT_W = 32;            // row stride in floats (vectors per row, padded)
constexpr int FT_MAXS = 65;         // sectors (N + 1 for s = 1/2, N <= 64)
constexpr double FT_TOL = 1e-5;     // breakdown threshold (above the FP32 noise floor)

struct GridBar {
    unsigned count;
    unsigned gen;
    int abort;
    int pad;
};

// A warp's share of the row phases: global rows [g0, g1) (all sectors' rows in order, which
// is also the order of the blocks in `items`), the first of them in item it0; its partial
// sums go to slots slot0, slot0 + 1, ... one per sector the rows touch, so the slots of a
// sector are consecutive over the warps.
struct FtRange {
    uint64_t g0, g1;
    uint32_t it0, slot0;
};

struct FtDev {
    // per (sector, vector) state, index s * FT_W + v
    double *sig_cur, *sig_prev, *beta_prev, *scale, *as;
    int *done, *nsteps;
    double *alpha, *beta;           // [(s * FT_W + v) * steps + j]
    double *part;                   // [slot][v]: warp partials of the update phase (FtRange)
    double *parta;                  // [sector][warp][v]: warp partials of the product phase
    double *partc;                  // [sector][cta][v]: the sums over each CTA's warps, of either phase
    const uint32_t *ck_it0;         // [chunk]: the block holding the chunk's first row
    const uint32_t *ck_cs;          // [nsec + 1]: sector s owns chunks ck_cs[s] .. ck_cs[s + 1] - 1
    const FtRange *wr;              // [warp]
    const uint32_t *slo;            // [nsec + 1]: sector s owns slots slo[s] .. slo[s + 1] - 1
    const uint2 *cta_rng;           // [nsec]: the CTAs [x, y) whose update rows include rows of sector s
    int *sec_active;                // [s]: four bytes, one for each eight vectors
    GridBar *bar;
    const uint32_t *items;          // (A << 16) | h, sorted by A
    const uint64_t *rowoff;         // first global row of sector A
    const uint32_t *secdim;         // D(N, A)
    uint16_t *hops;                 // [2^K][hop.stride]: targets of each low word (k_ft_hops)
    float *q0, *q1;                 // [rows][FT_W]
    double *theta, *tau;            // [(s * FT_W + v) * steps + j]
    int *mlen;                      // Krylov length per (s, v)
    double *zsum, *esum, *eref;     // thermodynamics (n_t each), e_ref
};

// A sector whose dimension does not exceed the step count would exhaust its Krylov
// space; it is diagonalised exactly instead (dense, FP64, one CTA): the Lanczos
// quadrature sum_j tau_j f(theta_j) of a start vector is then the exact <r|f(H)|r>.
struct ExactSec {
    int A, dim;
    uint32_t cd_off;                // its CD table inside the exact-table buffer
    int cd_rowlen, cd_len;
    uint64_t mat_off;               // ft_exact_bytes(dim)
};
constexpr int FT_MAXEXACT = 40;

struct FtParams {
    BlkParams P;                    // block plan built with A = N (full binomial table)
    FtDev d;
    int nsec, R, steps, nitems;
    uint32_t nchunks, ck_rows;      // product phase: chunks of ck_rows rows (a sector's last is shorter)
    unsigned nctas;
    uint64_t seed;
    unsigned long long barrier_ns;  // a grid barrier gives up after this long (default 5 s)
    uint64_t exact_mask;            // bit A set: sector A is diagonalised exactly
    HopTab hop;
    int nexact;
    ExactSec ex[FT_MAXEXACT];
};

__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// grid-wide barrier of a cooperative launch; gives up after limit_ns (sets abort) so a
// lost CTA can never hang the GPU
__device__ bool grid_sync(GridBar *gb, unsigned nctas, unsigned long long limit_ns) {
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned *vgen = &gb->gen;
        volatile int *vab = &gb->abort;
        const unsigned g = *vgen;
        __threadfence();
        const unsigned arrived = atomicAdd(&gb->count, 1u);
        if (arrived == nctas - 1) {
            atomicExch(&gb->count, 0u);
            __threadfence();
            atomicAdd(&gb->gen, 1u);
        } else {
            const unsigned long long t0 = globaltimer_ns();
            while (*vgen == g) {
                if (*vab) break;
                if (globaltimer_ns() - t0 > limit_ns) { atomicExch(&gb->abort, 1); break; }
                __nanosleep(32);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return *(volatile int *)&gb->abort == 0;
}

// ---- start vectors and state -----------------------------------------------------------
__global__ void k_ft_init(FtParams F) {
    const FtDev &d = F.d;
    const uint64_t nrows = d.rowoff[F.nsec];
    const uint64_t total = nrows * FT_W;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < total;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t row = t / FT_W;
        const int v = (int)(t % FT_W);
        int A = 0;
        while (d.rowoff[A + 1] <= row) ++A;          // few sectors: linear search
        float val = 0.0f;
        if (v < F.R) {
            const uint64_t stream = sm64(F.seed, ((uint64_t)A << 20) + (uint64_t)v);
            val = (sm64(stream, row - d.rowoff[A]) >> 63) ? -1.0f : 1.0f;
        }
        d.q0[t] = val;
        d.q1[t] = 0.0f;
    }
    // product-phase partials: the (sector, warp) pairs no chunk visits stay zero
    const uint64_t npa = (uint64_t)F.nsec * F.nctas * (FT_NT / 32) * FT_W;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < npa; t += (uint64_t)gridDim.x * blockDim.x)
        d.parta[t] = 0.0;
    const int nst = F.nsec * FT_W;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nst; t += gridDim.x * blockDim.x) {
        const int s = t / FT_W, v = t % FT_W;
        const bool on = v < F.R && d.secdim[s] > 0 && !((F.exact_mask >> s) & 1ull);
        d.sig_cur[t] = on ? 1.0 / sqrt((double)d.secdim[s]) : 0.0;   // |+-1 vector| = sqrt(dim)
        d.sig_prev[t] = 0.0;
        d.beta_prev[t] = 0.0;
        d.scale[t] = 0.0;
        d.as[t] = 0.0;
        d.done[t] = on ? 0 : 1;
        d.nsteps[t] = 0;
        d.mlen[t] = 0;
    }
    if (blockIdx.x == 0 && threadIdx.x < FT_MAXS && (int)threadIdx.x < F.nsec)
        d.sec_active[threadIdx.x] = ((F.exact_mask >> threadIdx.x) & 1ull) ? 0 : 0x01010101;
    if (blockIdx.x == 0 && threadIdx.x == 0) { d.bar->count = 0; d.bar->gen = 0; d.bar->abort = 0; }
}

// The warp's partials p[q] (vectors v0 + q of row group grp) summed over its VT row groups
// in a fixed order and written to slot `slot` of part, then cleared.  All 32 lanes call it.
template <int VT>
__device__ __forceinline__ void ft_warp_flush(ef::df *p, double *part, uint32_t slot, int lane, int grp, int v0) {
    constexpr int LPR = 32 / VT;                  // lanes per row group
#pragma unroll
    for (int q = 0; q < VT; ++q) {
        ef::df s = p[q];
#pragma unroll
        for (int g = 1; g < VT; ++g) {
            const float hi = __shfl_sync(0xffffffffu, p[q].hi, lane + g * LPR);
            const float lo = __shfl_sync(0xffffffffu, p[q].lo, lane + g * LPR);
            s = ef::df_add(s, ef::df{hi, lo});
        }
        if (grp == 0) part[(size_t)slot * FT_W + v0 + q] = (double)s.hi + (double)s.lo;
        p[q] = ef::df{0.0f, 0.0f};
    }
}

// The target table (blk_hops.cuh), once per run.  With the targets found by all 32 lanes for the same few
// rows, a row took 429 warp instructions and the product was issue-bound.  Product phase of the
// N = 20 run 382 -> 346 us a step, where the gathers' way through L1 and L2 bounds it, not instructions.
__global__ void k_ft_hops(FtParams F) {
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < 1u << F.P.K) hop_fill(F.P, F.hop, g, F.d.hops);
}

// Per (sector, vector) sums of the CTA partials partc[s][b][v] over the CTAs b in [lo(s), hi(s))
// in a fixed order: eight vectors of a sector to a CTA, thread (chunk, vector) takes every 64th CTA, the
// 64 chunks by shuffles over four lanes and over the warps' sums in order; f(s, v, sum) then runs
// on 8 lanes.  All threads call it.  The sums run over CTAs, not warps, and a binary64 add costs a
// warp 64 cycles: with one CTA and 16 chunks to a sector's 32 vectors the two grid barriers
// around this took 20 us of a step of the N = 20 run, 7 now.
constexpr int FT_OCT = FT_W / 8;                  // CTAs a sector
template <class R, class F>
__device__ __forceinline__ void ft_sector_sums(const FtParams &Fp, double *red, R &&range, F &&f) {
    const FtDev &d = Fp.d;
    constexpr int NCH = FT_NT / 8;
    const int v8 = threadIdx.x & 7, c = threadIdx.x >> 3, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int so = blockIdx.x; so < Fp.nsec * FT_OCT; so += gridDim.x) {
        const int s = so / FT_OCT, v = (so % FT_OCT) * 8 + v8;
        const double *ps = d.partc + (size_t)s * Fp.nctas * FT_W + v;
        const uint2 lh = range(s);
        double a = 0.0;
#pragma unroll 8
        for (unsigned b = lh.x + c; b < lh.y; b += NCH) a += __ldcg(ps + (size_t)b * FT_W);
        a += __shfl_xor_sync(0xffffffffu, a, 8);
        a += __shfl_xor_sync(0xffffffffu, a, 16);
        if (lane < 8) red[warp * 8 + lane] = a;
        __syncthreads();
        if (warp == 0) {
            double t = 0.0;
#pragma unroll
            for (int i = 0; i < FT_NT / 32; i += 4) t += red[(i + (lane >> 3)) * 8 + v8];
            t += __shfl_xor_sync(0xffffffffu, t, 8);
            t += __shfl_xor_sync(0xffffffffu, t, 16);
            if (lane < 8) f(s, v, t);
        }
        __syncthreads();
    }
}

// a += b where on holds, two additions to an instruction and no branch
template <int VT>
__device__ __forceinline__ void ft_add(float *a, const float *b, bool on = true) {
    if constexpr (VT == 1) {
        if (on) a[0] += b[0];
    } else {
#pragma unroll
        for (int q = 0; q < VT; q += 2) {
            unsigned long long s, t;
            asm("mov.b64 %0, {%1, %2};" : "=l"(s) : "f"(a[q]), "f"(a[q + 1]));
            asm("mov.b64 %0, {%1, %2};" : "=l"(t) : "f"(b[q]), "f"(b[q + 1]));
            asm("{\n.reg .pred p;\nsetp.ne.s32 p, %2, 0;\n@p add.rn.f32x2 %0, %0, %1;\n}" : "+l"(s) : "l"(t), "r"((int)on));
            asm("mov.b64 {%0, %1}, %2;" : "=f"(a[q]), "=f"(a[q + 1]) : "l"(s));
        }
    }
}

// VT consecutive floats of one row (16- or 8-byte aligned for VT = 4, 2), read-only path
template <int VT>
__device__ __forceinline__ void ft_ld(const float *p, float *v) {
    if constexpr (VT == 4) {
        const float4 t = __ldg((const float4 *)p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else if constexpr (VT == 2) {
        const float2 t = __ldg((const float2 *)p);
        v[0] = t.x; v[1] = t.y;
    } else {
        v[0] = __ldg(p);
    }
}

// the same of shared memory or the buffer the kernel writes, and the store
template <int VT>
__device__ __forceinline__ void ft_ld_rw(const float *p, float *v) {
    if constexpr (VT == 4) {
        const float4 t = *(const float4 *)p;
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else if constexpr (VT == 2) {
        const float2 t = *(const float2 *)p;
        v[0] = t.x; v[1] = t.y;
    } else {
        v[0] = *p;
    }
}
template <int VT>
__device__ __forceinline__ void ft_st(float *p, const float *v) {
    if constexpr (VT == 4) *(float4 *)p = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (VT == 2) *(float2 *)p = make_float2(v[0], v[1]);
    else *p = v[0];
}

// sector of a global row (few sectors: linear search)
__device__ __forceinline__ int ft_sector_of(const FtDev &d, int nsec, uint64_t g) {
    int A = 0;
    while (A + 1 < nsec && d.rowoff[A + 1] <= g) ++A;
    return A;
}

// per-warp shared slice: hop lists | sigma, gamma of the current sector | alpha sigma
__host__ __device__ __forceinline__ size_t ft_warp_bytes(const BlkParams &P) { return hops_bytes(P) + FT_W * 4 * 3; }

// ---- the persistent kernel ---------------------------------------------------------------
// Every warp owns the global rows [g0, g1) of its FtRange (rows of all sectors in order,
// balanced over the warps) in both row phases, so no CTA barrier separates blocks: a
// warp walks the blocks its rows fall in, builds their hop lists itself, and writes one
// partial per sector it touches.  Shared layout: block tables | per-warp slices | the
// sector-sum scratch.  A block's own rows are read through L1.
template <int NC, int VT>
__global__ void __launch_bounds__(FT_NT, FT_CTAS) k_ftlm(FtParams F) {
    const BlkParams &P = F.P;
    const FtDev &d = F.d;
    extern __shared__ __align__(16) unsigned char smem[];
    const BlkTabs tb = stage_blk_tables(P, smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *ws = smem + al16f(P.tab_bytes) + warp * ft_warp_bytes(P);
    const Hops sh = hops_carve(P, ws);
    float *sgw = (float *)(ws + hops_bytes(P));     // [sigma | gamma | alpha sigma][FT_W]
    double *red = (double *)(smem + al16f(P.tab_bytes) + (FT_NT / 32) * ft_warp_bytes(P));
    constexpr int LPR = 32 / VT;                   // lanes per row
    const int grp = lane / LPR, li = lane % LPR;   // row group in the warp, lane in row
    const int v0 = li * VT;                        // first vector of this lane
    const unsigned nw = gridDim.x * (FT_NT / 32), gw = blockIdx.x * (FT_NT / 32) + warp;
    const FtRange rg = d.wr[gw];
    const unsigned long long LIMIT = F.barrier_ns;
    __syncthreads();

    for (int j = 0; j < F.steps; ++j) {
        const float *qc = (j & 1) ? d.q1 : d.q0;
        float *qp = (j & 1) ? d.q0 : d.q1;
        // ---------------- phase A: products ----------------
        // chunk c of ck_rows rows goes to warp c mod W, so all warps sweep the rows together
        // and the targets of nearby exchanges are still in L2; a warp's partial for sector s
        // sums its chunks of s and goes to parta[s][warp]
        {
            ef::df dot[VT];
#pragma unroll
            for (int q = 0; q < VT; ++q) dot[q] = ef::df{0.0f, 0.0f};
            int curA = -1;
            bool act = false;
            for (uint32_t c = gw; c < F.nchunks; c += nw) {
                int A = curA < 0 ? 0 : curA;
                while (d.ck_cs[A + 1] <= c) ++A;
                const uint64_t g0 = d.rowoff[A] + (uint64_t)(c - d.ck_cs[A]) * F.ck_rows;
                const uint64_t g1 = g0 + F.ck_rows < d.rowoff[A + 1] ? g0 + F.ck_rows : d.rowoff[A + 1];
                if (A != curA) {
                    if (curA >= 0) ft_warp_flush<VT>(dot, d.parta, (uint32_t)curA * nw + gw, lane, grp, v0);
                    curA = A;
                    act = d.sec_active[A] != 0;
                    __syncwarp();
                    if (act) {
                        const int sv = A * FT_W + lane;
                        sgw[lane] = (float)d.sig_cur[sv];
                        sgw[FT_W + lane] = (float)(d.beta_prev[sv] * d.sig_prev[sv]);
                    }
                }
                if (!act) continue;
                const uint64_t base = d.rowoff[A];
                for (uint32_t it = d.ck_it0[c]; it < (uint32_t)F.nitems; ++it) {
                    const uint32_t item = d.items[it];
                    if ((int)(item >> 16) != A) break;     // the chunk ends at the sector's end
                    const uint32_t h = item & 0xFFFFu;
                    const int k = A - __popc(h);
                    const uint32_t off = blk_off(P, tb, h, k);
                    const uint32_t n = tb.C[P.K * (P.A + 1) + k];
                    const uint64_t ig0 = base + off;
                    if (ig0 >= g1) break;
                    const uint32_t ra = ig0 < g0 ? (uint32_t)(g0 - ig0) : 0u;
                    const uint32_t rb = ig0 + n > g1 ? (uint32_t)(g1 - ig0) : n;
                    __syncwarp();                  // the previous block's lists are read no more
                    hops_setup_high(P, tb, h, k, off, sh, lane);
                    hops_setup_cross(P, F.hop, tb, h, k, off, sh, lane);
                    __syncwarp();
                    const float *Xb = qc + ig0 * FT_W + v0;   // the block's rows, this lane's vectors
                    for (uint32_t r = ra + grp; r < rb; r += VT) {
                        const uint32_t g = (uint32_t)P.lwoff[k] + r, l = __ldg(P.lw + g);
                        const uint16_t *T = d.hops + (size_t)g * F.hop.stride;
                        const uint4 hd = __ldg((const uint4 *)T);   // counts, cross entries
                        float acc[NC][VT];
                        int cnt[NC];
#pragma unroll
                        for (int cl = 0; cl < NC; ++cl) {
                            float *ac = acc[cl];
#pragma unroll
                            for (int q = 0; q < VT; ++q) ac[q] = 0.0f;
                            // low exchanges: four gathers in flight, added in the order of the list; the
                            // padding reads the row itself and is not added
                            int mc = (int)((hd.x >> (8 * cl)) & 0xFFu);
                            const uint16_t *t = T + F.hop.seg[cl];
                            for (int e = 0; e < mc; e += 4) {
                                const uint2 w = __ldg((const uint2 *)(t + e));
                                float x0[VT], x1[VT], x2[VT], x3[VT];
                                ft_ld<VT>(Xb + (size_t)(w.x & 0xFFFFu) * FT_W, x0);
                                ft_ld<VT>(Xb + (size_t)(w.x >> 16) * FT_W, x1);
                                ft_ld<VT>(Xb + (size_t)(w.y & 0xFFFFu) * FT_W, x2);
                                ft_ld<VT>(Xb + (size_t)(w.y >> 16) * FT_W, x3);
                                ft_add<VT>(ac, x0);
                                ft_add<VT>(ac, x1, e + 1 < mc);
                                ft_add<VT>(ac, x2, e + 2 < mc);
                                ft_add<VT>(ac, x3, e + 3 < mc);
                            }
                            for (int e = P.cb_start[cl]; e < P.cb_start[cl + 1]; ++e) {
                                const int4 x = sh.x[e];
                                int t2;
                                const bool on = hop_cross(F.hop, x, hd, T, l, &t2);
                                float xv[VT];
                                ft_ld<VT>(Xb + (int64_t)(on ? t2 : (int)r) * FT_W, xv);
                                ft_add<VT>(ac, xv, on);
                                mc += (int)on;
                            }
                            // high exchanges: four independent gathers in flight (the far ones miss L2)
                            const int e1 = sh.hcs[cl + 1];
                            int e = sh.hcs[cl];
                            for (; e + 4 <= e1; e += 4) {
                                float x0[VT], x1[VT], x2[VT], x3[VT];
                                ft_ld<VT>(Xb + (int64_t)((int)r + sh.hcd[e]) * FT_W, x0);
                                ft_ld<VT>(Xb + (int64_t)((int)r + sh.hcd[e + 1]) * FT_W, x1);
                                ft_ld<VT>(Xb + (int64_t)((int)r + sh.hcd[e + 2]) * FT_W, x2);
                                ft_ld<VT>(Xb + (int64_t)((int)r + sh.hcd[e + 3]) * FT_W, x3);
                                ft_add<VT>(x0, x1);
                                ft_add<VT>(x2, x3);
                                ft_add<VT>(x0, x2);
                                ft_add<VT>(ac, x0);
                            }
                            for (; e < e1; ++e) {
                                float xv[VT];
                                ft_ld<VT>(Xb + (int64_t)((int)r + sh.hcd[e]) * FT_W, xv);
                                    ft_add<VT>(ac, xv);
                            }
                            cnt[cl] = mc + (sh.hcs[cl + 1] - sh.hcs[cl]);
                        }
                        float *up = qp + (ig0 + r) * FT_W + v0;
                        float xov[VT], uv[VT], sg[VT], gm[VT];
                        ft_ld<VT>(Xb + (size_t)r * FT_W, xov);
                        ft_ld_rw<VT>(up, uv);
                        ft_ld_rw<VT>(sgw + v0, sg);
                        ft_ld_rw<VT>(sgw + FT_W + v0, gm);
#pragma unroll
                        for (int q = 0; q < VT; ++q) {
                            const float xo = xov[q];
                            float y = 0.0f;
#pragma unroll
                            for (int cl = 0; cl < NC; ++cl)
                                y += P.gq[cl] * (2.0f * acc[cl][q] + (float)(P.ntot[cl] - 2 * cnt[cl]) * xo);
                            const float u = sg[q] * y - gm[q] * uv[q];
                            uv[q] = u;
                            dot[q] = ef::df_add(dot[q], ef::two_prod(sg[q] * xo, u));
                        }
                        ft_st<VT>(up, uv);
                    }
                }
            }
            if (curA >= 0) ft_warp_flush<VT>(dot, d.parta, (uint32_t)curA * nw + gw, lane, grp, v0);
            // the CTA's warp partials, summed in warp order (written by this CTA just now)
            __syncthreads();
            const unsigned w0 = blockIdx.x * (FT_NT / 32);
            for (int t = threadIdx.x; t < F.nsec * FT_W; t += FT_NT) {
                const int s = t / FT_W, v = t % FT_W;
                const double *ps = d.parta + ((size_t)s * nw + w0) * FT_W + v;
                double a = 0.0;
#pragma unroll
                for (int i = 0; i < FT_NT / 32; ++i) a += ps[(size_t)i * FT_W];
                d.partc[((size_t)s * F.nctas + blockIdx.x) * FT_W + v] = a;
            }
        }
        if (!grid_sync(d.bar, F.nctas, LIMIT)) return;
        // ---------------- phase B: alpha ----------------
        ft_sector_sums(F, red, [&](int) { return make_uint2(0u, F.nctas); }, [&](int s, int v, double a) {
            const int t = s * FT_W + v;
            if (d.done[t]) return;
            d.alpha[(size_t)t * F.steps + j] = a;
            d.scale[t] = fmax(d.scale[t], fabs(a));
            d.as[t] = a * d.sig_cur[t];
        });
        if (!grid_sync(d.bar, F.nctas, LIMIT)) return;
        // ---------------- phase C: update (a stream over the warp's rows) ----------------
        // lane: float4 number lane % 8 of a row, i.e. vectors 4 (lane % 8) .. + 3; the four
        // lanes of one float4 position are row groups 0..3 (ft_warp_flush<4> layout)
        if (rg.g0 < rg.g1) {
            ef::df nn[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) nn[q] = ef::df{0.0f, 0.0f};
            const int c4 = lane & 7, g4 = lane >> 3;
            int A = ft_sector_of(d, F.nsec, rg.g0);
            uint32_t slot = rg.slot0;
            for (;; ++A, ++slot) {
                const uint64_t a0 = rg.g0 > d.rowoff[A] ? rg.g0 : d.rowoff[A];
                const uint64_t a1 = rg.g1 < d.rowoff[A + 1] ? rg.g1 : d.rowoff[A + 1];
                if (d.sec_active[A]) {
                    __syncwarp();
                    sgw[2 * FT_W + lane] = (float)d.as[A * FT_W + lane];
                    __syncwarp();
                    float as4[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) as4[q] = sgw[2 * FT_W + 4 * c4 + q];
                    for (uint64_t row = a0 + g4; row < a1; row += 4) {
                        const size_t ix = row * FT_W + 4 * c4;
                        const float4 u = *(const float4 *)(qp + ix);
                        const float4 x = __ldcs((const float4 *)(qc + ix));
                        float4 w;
                        w.x = u.x - as4[0] * x.x; w.y = u.y - as4[1] * x.y;
                        w.z = u.z - as4[2] * x.z; w.w = u.w - as4[3] * x.w;
                        *(float4 *)(qp + ix) = w;
                        nn[0] = ef::df_add(nn[0], ef::two_prod(w.x, w.x));
                        nn[1] = ef::df_add(nn[1], ef::two_prod(w.y, w.y));
                        nn[2] = ef::df_add(nn[2], ef::two_prod(w.z, w.z));
                        nn[3] = ef::df_add(nn[3], ef::two_prod(w.w, w.w));
                    }
                }
                ft_warp_flush<4>(nn, d.part, slot, lane, g4, 4 * c4);
                if (a1 >= rg.g1) break;
            }
        }
        // the CTA's slots of each sector it touches, in order (written by this CTA just now)
        __syncthreads();
        {
            const uint32_t w0 = blockIdx.x * (FT_NT / 32);
            const uint32_t b0 = d.wr[w0].slot0, b1 = w0 + FT_NT / 32 < nw ? d.wr[w0 + FT_NT / 32].slot0 : d.slo[F.nsec];
            for (int t = threadIdx.x; t < F.nsec * FT_W; t += FT_NT) {
                const int s = t / FT_W, v = t % FT_W;
                const uint32_t s0 = max(b0, d.slo[s]), s1 = min(b1, d.slo[s + 1]);
                if (s0 >= s1) continue;
                double a = 0.0;
                for (uint32_t sl = s0; sl < s1; ++sl) a += d.part[(size_t)sl * FT_W + v];
                d.partc[((size_t)s * F.nctas + blockIdx.x) * FT_W + v] = a;
            }
        }
        if (!grid_sync(d.bar, F.nctas, LIMIT)) return;
        // ---------------- phase D: beta ----------------
        ft_sector_sums(F, red, [&](int s) { return d.cta_rng[s]; }, [&](int s, int v, double sum) {
            const int t = s * FT_W + v;
            bool act = false;
            if (!d.done[t]) {
                const double b = sqrt(sum);
                d.beta[(size_t)t * F.steps + j] = b;
                d.nsteps[t] = j + 1;
                // stop when beta is at the noise floor or the sector is exhausted
                if (b <= FT_TOL * d.scale[t] || (uint32_t)(j + 1) >= d.secdim[s]) {
                    d.done[t] = 1;
                    d.sig_cur[t] = 0.0;
                    d.sig_prev[t] = 0.0;
                    d.beta_prev[t] = 0.0;
                    d.as[t] = 0.0;
                } else {
                    d.scale[t] = fmax(d.scale[t], b);
                    d.sig_prev[t] = d.sig_cur[t];
                    d.sig_cur[t] = 1.0 / b;
                    d.beta_prev[t] = b;
                    act = true;
                }
            }
            // a sector stays active while any of its vectors runs: one byte for each eight of them
            const unsigned any = __ballot_sync(0xFFu, act);
            if (v % 8 == 0) ((unsigned char *)(d.sec_active + s))[v / 8] = any != 0u;
        });
        if (!grid_sync(d.bar, F.nctas, LIMIT)) return;
    }
}

// ---- tridiagonal eigenvalues and first components -----------------------------------------
// theta and tau of (sector, vector) blockIdx.x: the eigenvalues lambda_i of T and mu_i of T without its
// first row and column, by bisection with Sturm counts (tridiag.cuh), one eigenvalue a lane, and
//   tau_i = prod_j (lambda_i - mu_j) / prod_{j != i} (lambda_i - lambda_j)
// (the residues of the first diagonal entry of the resolvent; Golub and Meurant, Matrices, Moments and
// Quadrature).  Whatever the rounding of interlacing lambda and mu, they are those of some Jacobi
// matrix close to T, so the tau are positive and sum to one also where ghosts lie an ulp apart.  All m
// values are found at once, where the rotations of the implicit QR algorithm form one chain of
// m^2 times 30 dependent binary64 instructions: N = 20, 672 matrices of 80 rows 9.5 -> 2.2 ms.
// Eigenvalues are cut to the last bit of the norm: binary32 counts to 2^-18 of it, widened by 2^-19
// for their rounding, then binary64.  lambda and mu in dynamic shared memory (2 x steps doubles).
constexpr int FT_EIG_NT = 192;
__global__ void __launch_bounds__(FT_EIG_NT) k_ft_eig(FtParams F) {
    extern __shared__ __align__(16) double ft_eig_sh[];
    const FtDev &d = F.d;
    const int t = blockIdx.x, v = t % FT_W, tid = threadIdx.x, lane = tid & 31;
    if ((F.exact_mask >> (t / FT_W)) & 1ull) return;   // filled by k_ft_exact
    const int m = (v < F.R) ? d.nsteps[t] : 0;
    if (tid == 0) d.mlen[t] = m;
    if (m == 0) return;
    double *lam = ft_eig_sh, *mu = lam + F.steps;
    const double *al = d.alpha + (size_t)t * F.steps, *be = d.beta + (size_t)t * F.steps;
    double *theta = d.theta + (size_t)t * F.steps, *tau = d.tau + (size_t)t * F.steps;
    bool bad = false;
    for (int i = tid; i < m; i += FT_EIG_NT) bad |= !isfinite(al[i]) || (i + 1 < m && !isfinite(be[i]));
    double g0, g1;
    tri_gershgorin(m, al, be, &g0, &g1);
    const double bound = fmax(fabs(g0), fabs(g1));
    if (__syncthreads_or(bad) || !(bound <= 1.7e308)) {
        for (int i = tid; i < m; i += FT_EIG_NT) theta[i] = tau[i] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    if (m == 1 || bound == 0.0) {
        for (int i = tid; i < m; i += FT_EIG_NT) { theta[i] = al[i]; tau[i] = i == 0 ? 1.0 : 0.0; }
        return;
    }
    const int ex = min(max(ilogb(bound), -1000), 1000);
    const double s = tri_pow2(-ex);                    // s T has a norm in [1, 2)
    const double pad = 2.0 * 2.220446049250313e-16 * bound * s;
    const int nw = (m + 31) / 32, nw1 = (m + 30) / 32; // warps' worth of lambda, of mu
    for (int w = tid >> 5; w < nw + nw1; w += FT_EIG_NT / 32) {
        const bool sub = w >= nw;
        const int mm = m - (int)sub, e = (sub ? w - nw : w) * 32 + lane + 1;
        const double *A = al + (int)sub, *B = be + (int)sub;
        const int ec = min(e, mm);                     // idle lanes repeat the last eigenvalue
        float fa = __double2float_rd(g0 * s - pad), fc = __double2float_ru(g1 * s + pad);
        for (int it = 0; it < 21; ++it) {              // 4 2^-21 < 2^-18
            const float x = 0.5f * (fa + fc);
            if (tri_count<float>(mm, A, B, s, x) < ec) fa = x; else fc = x;
        }
        double a = (double)fa - 0x1p-19, c = (double)fc + 0x1p-19;
        for (int it = 0; it < 60; ++it) {
            const double x = 0.5 * (a + c);
            const bool more = c - a > 0x1p-53 && x > a && x < c;
            if (!__any_sync(0xffffffffu, more)) break;
            if (tri_count<double>(mm, A, B, s, x) < ec) a = more ? x : a; else c = more ? x : c;
        }
        if (e <= mm) (sub ? mu : lam)[e - 1] = 0.5 * (a + c);
    }
    __syncthreads();
    // strictly increasing lambda (T is unreduced) at least two units of the norm's last place apart,
    // mu between its neighbours
    bool close = false;
    for (int i = tid; i + 1 < m; i += FT_EIG_NT) close |= lam[i + 1] - lam[i] < 0x1p-51;
    if (__syncthreads_or(close) && tid == 0)
        for (int i = 1; i < m; ++i) lam[i] = fmax(lam[i], lam[i - 1] + 0x1p-51);
    __syncthreads();
    for (int i = tid; i + 1 < m; i += FT_EIG_NT) mu[i] = fmin(fmax(mu[i], lam[i]), lam[i + 1]);
    __syncthreads();
    for (int i = tid; i < m; i += FT_EIG_NT) {
        const double x = lam[i];
        double w = 1.0;
        for (int j0 = 0; j0 + 1 < m; j0 += 8) {        // eight factors to a division
            double nu = 1.0, de = 1.0;
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
                const int j = j0 + jj;
                if (j + 1 < m) {
                    nu *= x - mu[j];
                    de *= x - lam[j < i ? j : j + 1];
                }
            }
            w *= nu / de;
        }
        theta[i] = x * tri_pow2(ex);
        tau[i] = w;
    }
}

// Dense H of one small sector (rows by the paper's decode/encode, Eq. E-4-b), its
// eigen-decomposition by parallel cyclic Jacobi (Brent-Luk round-robin ordering of the
// rotations, each zeroing one off-diagonal pair as in Golub and Van Loan, Sec. 8.5),
// then theta_k = E_k and tau_k = <r^|psi_k>^2 for every start vector r^ = r / |r|.
// One CTA a sector, so what bounds it is the binary64 pipe of one SM and the chain of a round's
// rotation angles.  The rotations are applied to the start vectors (W = V^T r) instead of to an
// n x n V; both sides of H at once, a 2 x 2 block of two rotations a thread and only one of each two
// mirrored blocks; angles by two rsqrt (eighteen dependent instructions, forty before);
// matrices in shared memory where they fit.  N = 12, two sectors of 66 states: 3.4 ms, the run 17.5 -> 8.3 ms.
// n is padded to an even size with a zero row; H has a power of two taken out.
constexpr int FT_X_NT = 1024;
constexpr size_t FT_X_SMEM = 200 * 1024;   // n <= 144
__host__ __device__ __forceinline__ size_t ft_exact_bytes(int n) {
    const size_t m = (size_t)n + (n & 1);
    return m * m * 8 + m * FT_W * 8;
}
__global__ void __launch_bounds__(FT_X_NT) k_ft_exact(FtParams F, BondParams bp, const uint32_t *__restrict__ cdall,
                                                      double *__restrict__ mats, size_t smem_bytes) {
    extern __shared__ __align__(16) double ft_x_sh[];
    const FtDev &d = F.d;
    const ExactSec ex = F.ex[blockIdx.x];
    const int n = ex.dim, m = n + (n & 1), mh = m / 2, tid = threadIdx.x;
    double *H = ft_exact_bytes(n) <= smem_bytes ? ft_x_sh : mats + ex.mat_off, *W = H + (size_t)m * m;
    __shared__ int sp[256], sq[256], s_stop;
    __shared__ double sc[256], ss[256], red[FT_X_NT / 32];
    for (int t = tid; t < m * m; t += FT_X_NT) H[t] = 0.0;
    const double inv = 1.0 / sqrt((double)n);
    for (int t = tid; t < m * FT_W; t += FT_X_NT) {
        const int i = t / FT_W, r = t % FT_W;
        const uint64_t stream = sm64(F.seed, ((uint64_t)ex.A << 20) + (uint64_t)r);
        W[t] = i < n && r < F.R ? ((sm64(stream, (uint64_t)i) >> 63) ? -inv : inv) : 0.0;
    }
    __syncthreads();
    Codec<uint32_t> c{cdall + ex.cd_off, F.P.N, 1, ex.A, 1, 3, ex.cd_rowlen};
    double big = 0.0;
    for (int i = tid; i < n; i += FT_X_NT) {
        const uint64_t w = c.decode((uint32_t)i);
        double dg = 0.0;
        for (int t = 0; t < bp.nb; ++t) {
            const int p = bp.p[t], q = bp.q[t];
            const int ap = dig(w, p, 1), aq = dig(w, q, 1);
            dg += bp.jm[t] * (0.5 - ap) * (0.5 - aq);
            if (ap != aq) {
                const uint32_t j = (uint32_t)i + c.delta(w, p, q, ap ? -1 : +1);
                H[(size_t)i * m + j] += bp.jm[t] * 0.5;
            }
        }
        H[(size_t)i * m + i] += dg;
        for (int k = 0; k < n; ++k) big = fmax(big, fabs(H[(size_t)i * m + k]));
    }
    for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
    if ((tid & 31) == 0) red[tid >> 5] = big;
    __syncthreads();
    for (int w = 0; w < FT_X_NT / 32; ++w) big = fmax(big, red[w]);
    __syncthreads();
    const int e2 = big > 0.0 && big < 1e308 ? min(max(ilogb(big), -1000), 1000) : 0;
    for (int t = tid; t < m * m; t += FT_X_NT) H[t] = ldexp(H[t], -e2);
    __syncthreads();
    const int nblk = mh * (mh / 2 + 1);   // blocks (k, k + o mod mh), o = 0 .. mh / 2 (half of the last o if mh is even)
    for (int sweep = 0; sweep < 40 && n > 1; ++sweep) {
        // stop when the off-diagonal part is negligible
        double off = 0.0, tot = 0.0;
        for (int t = tid; t < m * m; t += FT_X_NT) {
            const double h = H[t];
            tot += h * h;
            if (t / m != t % m) off += h * h;
        }
        off = block_sum<FT_X_NT>(off, red);
        __syncthreads();
        tot = block_sum<FT_X_NT>(tot, red);
        if (tid == 0) s_stop = off <= 1e-30 * tot;
        __syncthreads();
        if (s_stop) break;
        for (int round = 0; round < m - 1; ++round) {
            for (int k = tid; k < mh; k += FT_X_NT) {
                int p, q;
                if (k == 0) { p = m - 1; q = round; }
                else { p = (round + k) % (m - 1); q = (round - k + (m - 1)) % (m - 1); }
                if (p > q) { const int tt = p; p = q; q = tt; }
                // tan 2 theta = 2 apq / (aqq - app), |theta| <= pi / 4.  The largest element is in [1, 2): an apq
                // below 2^-500 counts as zero, as r2 would otherwise leave the normal numbers and c^2 + s^2 one
                const double dd = H[(size_t)q * m + q] - H[(size_t)p * m + p], h2 = 2.0 * H[(size_t)p * m + q];
                const double r2 = dd * dd + h2 * h2, ri = rsqrt(r2);
                const bool on = fabs(h2) > 0x1p-500;
                const double x = fma(0.5 * fabs(dd), ri, 0.5), rx = rsqrt(x);
                sp[k] = p;
                sq[k] = q;
                sc[k] = on ? x * rx : 1.0;
                ss[k] = on ? 0.5 * h2 * (dd < 0.0 ? -ri : ri) * rx : 0.0;
            }
            __syncthreads();
            for (int t = tid; t < nblk + mh * FT_W; t += FT_X_NT) {
                if (t < nblk) {                            // J1^T B J2
                    const int o = t / mh, k1 = t - o * mh, k2 = k1 + o < mh ? k1 + o : k1 + o - mh;
                    if (2 * o == mh && k1 >= o) continue;
                    const size_t p1 = sp[k1], q1 = sq[k1], p2 = sp[k2], q2 = sq[k2];
                    const double c1 = sc[k1], s1 = ss[k1], c2 = sc[k2], s2 = ss[k2];
                    const double a = H[p1 * m + p2], b = H[p1 * m + q2], e = H[q1 * m + p2], f = H[q1 * m + q2];
                    const double ra = c1 * a - s1 * e, rb = c1 * b - s1 * f, re = s1 * a + c1 * e, rf = s1 * b + c1 * f;
                    const double na = c2 * ra - s2 * rb, nf = s2 * re + c2 * rf;
                    double nb = s2 * ra + c2 * rb, ne = c2 * re - s2 * rf;
                    if (o == 0) nb = ne = 0.0;             // the pair that the rotation zeroes
                    H[p1 * m + p2] = na; H[p1 * m + q2] = nb; H[q1 * m + p2] = ne; H[q1 * m + q2] = nf;
                    if (o != 0) { H[p2 * m + p1] = na; H[q2 * m + p1] = nb; H[p2 * m + q1] = ne; H[q2 * m + q1] = nf; }
                } else {                                   // W <- J^T W
                    const int u = t - nblk, k = u / FT_W, r = u % FT_W;
                    double *wp = W + (size_t)sp[k] * FT_W + r, *wq = W + (size_t)sq[k] * FT_W + r;
                    const double a = *wp, b = *wq;
                    *wp = sc[k] * a - ss[k] * b;
                    *wq = ss[k] * a + sc[k] * b;
                }
            }
            __syncthreads();
        }
    }
    // weights of every start vector
    for (int t = tid; t < F.R * n; t += FT_X_NT) {
        const int r = t / n, kk = t % n;
        const double o = W[(size_t)kk * FT_W + r];
        const size_t sv = (size_t)ex.A * FT_W + r;
        d.theta[sv * F.steps + kk] = ldexp(H[(size_t)kk * m + kk], e2);
        d.tau[sv * F.steps + kk] = o * o;
    }
    for (int r = tid; r < FT_W; r += FT_X_NT) d.mlen[(size_t)ex.A * FT_W + r] = r < F.R ? n : 0;
}

// Thermal sums.  Every (temperature, Ritz value) pair costs an exponential, about 25 binary64
// operations on a pipe that takes 1.7 a cycle and SM: on one SM the 1.3 M pairs of 24
// temperatures at N = 20 took 8.9 ms, over all of them 0.09 ms.
// mins[s] = lowest Ritz value of sector s
__global__ void __launch_bounds__(256) k_ft_min(FtParams F, double *__restrict__ mins) {
    const FtDev &d = F.d;
    __shared__ double red[8];
    const int s = blockIdx.x;
    double mn = 1e308;
    for (int p = threadIdx.x; p < F.R * F.steps; p += 256) {
        const int t = s * FT_W + p / F.steps, i = p % F.steps;
        if (i < d.mlen[t]) mn = fmin(mn, d.theta[(size_t)t * F.steps + i]);
    }
    for (int o = 16; o > 0; o >>= 1) mn = fmin(mn, __shfl_down_sync(0xffffffffu, mn, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mn;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) mn = fmin(mn, red[w]);
        mins[s] = mn;
    }
}

// CTA (s, it): the sums of sector s at temperature temps[it], zs / es [it nsec + s]
__global__ void __launch_bounds__(256) k_ft_thermo(FtParams F, const double *__restrict__ temps,
                                                    const double *__restrict__ mins, double *__restrict__ zs,
                                                    double *__restrict__ es) {
    const FtDev &d = F.d;
    __shared__ double red[8];
    const int s = blockIdx.x, it = blockIdx.y;
    double e_ref = 1e308;
    for (int k = 0; k < F.nsec; ++k) e_ref = fmin(e_ref, mins[k]);
    const double T = temps[it], wgt = (double)d.secdim[s] / (double)F.R;
    double z = 0.0, ez = 0.0;
    for (int p = threadIdx.x; p < F.R * F.steps; p += 256) {
        const int t = s * FT_W + p / F.steps, i = p % F.steps;
        if (i < d.mlen[t]) {
            const double th = d.theta[(size_t)t * F.steps + i];
            const double b = d.tau[(size_t)t * F.steps + i] * exp(-(th - e_ref) / T) * wgt;
            z += b;
            ez += b * th;
        }
    }
    z = block_sum<256>(z, red);
    __syncthreads();
    ez = block_sum<256>(ez, red);
    if (threadIdx.x == 0) {
        zs[(size_t)it * F.nsec + s] = z;
        es[(size_t)it * F.nsec + s] = ez;
    }
}

// e_ref, Z and E from the sectors' sums, in sector order
__global__ void __launch_bounds__(256) k_ft_thermo_fin(FtParams F, const double *__restrict__ mins,
                                                        const double *__restrict__ zs, const double *__restrict__ es,
                                                        int n_t) {
    const FtDev &d = F.d;
    const int it = blockIdx.x * 256 + threadIdx.x;
    if (it == 0) {
        double m = 1e308;
        for (int k = 0; k < F.nsec; ++k) m = fmin(m, mins[k]);
        *d.eref = m;
    }
    if (it >= n_t) return;
    double z = 0.0, e = 0.0;
    for (int s = 0; s < F.nsec; ++s) {
        z += zs[(size_t)it * F.nsec + s];
        e += es[(size_t)it * F.nsec + s];
    }
    d.zsum[it] = z;
    d.esum[it] = e / z;
}

// ---- host --------------------------------------------------------------------------------
struct FtLayout {
    size_t q0, q1, st, ab, part, wr, slo, crng, parta, partc, ckit, ckcs, sec, bar, items, rowoff, secdim, hops, theta, tau, mlen, therm, tsum, temps,
        xcd, xmat, total;
};

static int ft_choose_K(int N) {
    // largest K (8..16, K <= N-2) whose biggest block of 32-float rows fits ~75 KB, so
    // two CTAs fit on an SM (K = 11: 462 rows, 59 KB)
    int best = -1;
    for (int K = 8; K <= 16 && K <= N - 2; ++K) {
        uint64_t c = 1;
        for (int i = 0; i < K / 2; ++i) c = c * (K - i) / (i + 1);
        if (c * FT_W * 4 <= 75 * 1024) best = K;
    }
    return best;
}

static FtLayout ft_layout(int N, int nsec, int R, int steps, int nitems, int nctas, int n_t, size_t xcd_words,
                          size_t xmat_doubles, size_t nchunks, size_t hop_entries) {
    (void)R;
    FtLayout L{};
    auto a = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const uint64_t rows = 1ull << N;     // sum of all sector dimensions for s = 1/2
    const size_t nst = (size_t)nsec * FT_W;
    size_t o = 0;
    L.q0 = o; o += a(rows * FT_W * 4);
    L.q1 = o; o += a(rows * FT_W * 4);
    L.st = o; o += a(nst * 8 * 5 + nst * 4 * 2);
    L.ab = o; o += a(nst * (size_t)steps * 8 * 2);
    const size_t nslots = (size_t)nctas * (FT_NT / 32) + nsec + 1;   // bound on the warp-sector pairs
    L.part = o; o += a(nslots * FT_W * 8);
    L.wr = o; o += a((size_t)nctas * (FT_NT / 32) * sizeof(FtRange));
    L.slo = o; o += a((size_t)(nsec + 1) * 4);
    L.crng = o; o += a((size_t)nsec * sizeof(uint2));
    L.parta = o; o += a((size_t)nsec * nctas * (FT_NT / 32) * FT_W * 8);
    L.partc = o; o += a((size_t)nsec * nctas * FT_W * 8);
    L.ckit = o; o += a((nchunks > 0 ? nchunks : 1) * 4);
    L.ckcs = o; o += a((size_t)(nsec + 1) * 4);
    L.sec = o; o += a(FT_MAXS * 4);
    L.bar = o; o += a(sizeof(GridBar));
    L.items = o; o += a((size_t)nitems * 4);
    L.rowoff = o; o += a((size_t)(nsec + 1) * 8);
    L.secdim = o; o += a((size_t)nsec * 4);
    L.hops = o; o += a(hop_entries * 2);
    L.theta = o; o += a(nst * (size_t)steps * 8);
    L.tau = o; o += a(nst * (size_t)steps * 8);
    L.mlen = o; o += a(nst * 4);
    L.therm = o; o += a((size_t)(2 * n_t + 1) * 8);
    L.tsum = o; o += a((size_t)nsec * (2 * (size_t)n_t + 1) * 8);
    L.temps = o; o += a((size_t)(n_t > 0 ? n_t : 1) * 8);
    L.xcd = o; o += a((xcd_words > 0 ? xcd_words : 1) * 4);
    L.xmat = o; o += a((xmat_doubles > 0 ? xmat_doubles : 1) * 8);
    L.total = o;
    return L;
}

template <int NC, int VT>
static const void *ft_kernel() { return (const void *)k_ftlm<NC, VT>; }

static const void *pick_kernel(int nc, int vt) {
    if (nc == 1) return vt == 1 ? ft_kernel<1, 1>() : vt == 2 ? ft_kernel<1, 2>() : ft_kernel<1, 4>();
    if (nc == 2) return vt == 1 ? ft_kernel<2, 1>() : vt == 2 ? ft_kernel<2, 2>() : ft_kernel<2, 4>();
    return vt == 1 ? ft_kernel<4, 1>() : vt == 2 ? ft_kernel<4, 2>() : ft_kernel<4, 4>();
}

static size_t ft_smem(const BlkParams &P, int nsec) {
    (void)nsec;
    size_t o = al16f(P.tab_bytes);
    o += (FT_NT / 32) * ft_warp_bytes(P);
    o += (size_t)(FT_NT / 32) * 8 * 8;    // sector-sum scratch
    return o;
}

// The warps' row ranges (equal shares of all 2^N rows) and their partial-sum slots.
// items: the blocks (A << 16 | h) in row order; C(K, k) rows each.
static void ft_ranges(int n_sites, int K, const hm_basis &full, const std::vector<uint32_t> &items, int W,
                      uint32_t ck_rows, std::vector<FtRange> *wr, std::vector<uint32_t> *slo, std::vector<uint2> *crng,
                      std::vector<uint32_t> *ck_it0, std::vector<uint32_t> *ck_cs) {
    const int N = n_sites, nsec = N + 1, Wd = N + 1;
    std::vector<uint64_t> r0(items.size() + 1, 0);
    for (size_t i = 0; i < items.size(); ++i) {
        const int A = (int)(items[i] >> 16);
        const int k = A - __builtin_popcount(items[i] & 0xFFFFu);
        r0[i + 1] = r0[i] + full.D[(size_t)K * Wd + k];
    }
    std::vector<uint64_t> rowoff(nsec + 1, 0);
    for (int A = 0; A < nsec; ++A) rowoff[A + 1] = rowoff[A] + full.D[(size_t)N * Wd + A];
    const uint64_t T = r0.back();
    auto sector_of = [&](uint64_t g) { return (int)(std::upper_bound(rowoff.begin(), rowoff.end(), g) - rowoff.begin()) - 1; };
    wr->assign(W, FtRange{});
    std::vector<int> slot_sec;
    for (int w = 0; w < W; ++w) {
        FtRange &g = (*wr)[w];
        g.g0 = T * (uint64_t)w / (uint64_t)W;
        g.g1 = T * (uint64_t)(w + 1) / (uint64_t)W;
        g.slot0 = (uint32_t)slot_sec.size();
        if (g.g0 >= g.g1) { g.it0 = (uint32_t)items.size(); continue; }
        g.it0 = (uint32_t)(std::upper_bound(r0.begin(), r0.end(), g.g0) - r0.begin() - 1);
        for (int A = sector_of(g.g0); A <= sector_of(g.g1 - 1); ++A) slot_sec.push_back(A);
    }
    slo->assign(nsec + 1, 0);
    size_t i = 0;
    for (int s = 0; s <= nsec; ++s) {
        while (i < slot_sec.size() && slot_sec[i] < s) ++i;
        (*slo)[s] = (uint32_t)i;
    }
    // the CTAs that own slots of each sector (their first slots increase)
    crng->assign(nsec, make_uint2(0u, 0u));
    const int wpc = FT_NT / 32, nct = W / wpc;
    for (int s2 = 0; s2 < nsec; ++s2) {
        uint2 &r = (*crng)[s2];
        bool any = false;
        for (int c = 0; c < nct; ++c) {
            const uint32_t b0 = (*wr)[(size_t)c * wpc].slot0;
            const uint32_t b1 = c + 1 < nct ? (*wr)[(size_t)(c + 1) * wpc].slot0 : (*slo)[nsec];
            if (std::max(b0, (*slo)[s2]) >= std::min(b1, (*slo)[s2 + 1])) continue;
            if (!any) r.x = (uint32_t)c;
            r.y = (uint32_t)c + 1;
            any = true;
        }
    }
    // product-phase chunks: each sector cut into runs of ck_rows rows
    ck_it0->clear();
    ck_cs->assign(nsec + 1, 0);
    for (int A = 0; A < nsec; ++A) {
        (*ck_cs)[A] = (uint32_t)ck_it0->size();
        for (uint64_t g = rowoff[A]; g < rowoff[A + 1]; g += ck_rows)
            ck_it0->push_back((uint32_t)(std::upper_bound(r0.begin(), r0.end(), g) - r0.begin() - 1));
    }
    (*ck_cs)[nsec] = (uint32_t)ck_it0->size();
}

// rows per product-phase chunk: HM_FT_CHUNK (16..1024), default 64, and fewer below N = 22, where
// chunks of 64 rows are too few for 7296 warps to share evenly (whole runs of 40 steps, 16 / 32 /
// 64 rows: N = 16 9.3 / 10.4 / 13.5 ms, N = 20 29.5 / 31.1 / 32.6, N = 22 111 / 103 / 101)
static uint32_t ft_chunk_rows(int n_sites) {
    const char *e = getenv("HM_FT_CHUNK");
    const int v = e ? atoi(e) : n_sites <= 20 ? 16 : n_sites == 21 ? 32 : 64;
    return (uint32_t)(v < 16 ? 16 : v > 1024 ? 1024 : v);
}

// how long a grid barrier of the persistent kernel waits before it gives up: 5 s, or
// HM_FT_BARRIER_NS (0 .. 5e9 ns; a test sets 0 to make the first wait give up)
static unsigned long long ft_barrier_ns() {
    const unsigned long long dflt = 5000000000ull;
    const char *e = getenv("HM_FT_BARRIER_NS");
    if (!e || !*e) return dflt;
    const long long v = atoll(e);
    return v < 0 ? 0ull : (unsigned long long)v > dflt ? dflt : (unsigned long long)v;
}

// vectors-per-lane tiling chosen by timing each candidate once per (N, bonds) shape
static std::map<std::pair<int, int>, int> g_ft_tuned;

struct FtSetup {
    hm_basis full;                   // tables with the full binomial table (A = N)
    FtParams F;
    BondParams bp;
    FtLayout L;
    size_t smem;
    int nctas;
    std::vector<uint32_t> xcd;       // CD tables of the exactly diagonalised sectors
    std::vector<FtRange> wr;         // per warp
    std::vector<uint32_t> slo;       // per sector, + 1
    std::vector<uint2> crng;         // per sector
    std::vector<uint32_t> ck_it0;    // per product-phase chunk
    std::vector<uint32_t> ck_cs;     // per sector, + 1
};

static int ft_prepare(int n_sites, int two_s, int n_bonds, const int32_t *u, const int32_t *v,
                      const double *J, int R, int steps, int n_t, FtSetup *S, std::vector<uint32_t> *items) {
    if (two_s != 1) return fail(HM_EINVAL, "ftlm_run supports s = 1/2 (two_s = 1)");
    if (R < 1 || R > FT_W) return fail(HM_EINVAL, "R must be in 1..%d", FT_W);
    if (steps < 1 || steps > 2000) return fail(HM_EINVAL, "steps must be in 1..2000");   // k_ft_eig: 2 x steps doubles
    if (n_t < 0 || n_t > 4096) return fail(HM_EINVAL, "n_t must be in 0..4096");
    const int K = ft_choose_K(n_sites);
    if (K < 0 || n_sites > 32) return fail(HM_EINVAL, "ftlm_run needs 10 <= n_sites <= 32");
    HM_TRY(build_tables(n_sites, 1, -n_sites, &S->full));      // A = N: full table
    BondParams &bp = S->bp;
    HM_TRY(make_bonds(&S->full, n_bonds, u, v, J, &bp));
    memset(&S->F, 0, sizeof S->F);
    const int prc = blk_plan(&S->full, bp, K, &S->F.P);
    if (prc < 0) return prc;
    if (prc > 0 || S->F.P.perbond)
        return fail(HM_EINVAL, "ftlm_run: more than %d coupling classes or %d bonds", HM_BLK_MAXC, HM_BLK_MAXB);
    // the plan's block size was taken for A = N; use the largest over all sectors
    uint64_t mb = 1;
    for (int i = 0; i < K / 2; ++i) mb = mb * (K - i) / (i + 1);
    S->F.P.max_block = (int)mb;
    S->F.hop = hop_layout(S->F.P);
    const int nsec = n_sites + 1;
    items->clear();
    const int H = n_sites - K;
    for (int A = 0; A <= n_sites; ++A)
        for (uint32_t h = 0; h < (1u << H); ++h) {
            const int k = A - __builtin_popcount(h);
            if (k >= 0 && k <= K) items->push_back(((uint32_t)A << 16) | h);
        }
    S->F.nsec = nsec;
    S->F.R = R;
    S->F.steps = steps;
    // sectors of dimension <= steps (and <= 512): exact treatment
    S->xcd.clear();
    uint64_t xmat = 0;
    for (int A = 0; A <= n_sites; ++A) {
        const int W = n_sites + 1;
        const uint64_t dimA = S->full.D[(size_t)n_sites * W + A];
        if (dimA > (uint64_t)steps || dimA > 512) continue;
        if (S->F.nexact == FT_MAXEXACT) return fail(HM_EINVAL, "ftlm_run: too many small sectors");
        hm_basis sb;
        HM_TRY(build_tables(n_sites, 1, n_sites - 2 * A, &sb));
        ExactSec &ex = S->F.ex[S->F.nexact++];
        ex.A = A;
        ex.dim = (int)dimA;
        ex.cd_off = (uint32_t)S->xcd.size();
        ex.cd_rowlen = sb.view.cd_rowlen;
        ex.cd_len = sb.view.cd_len;
        for (int k = 0; k < sb.view.cd_len; ++k) S->xcd.push_back((uint32_t)sb.cd[k]);
        ex.mat_off = xmat;
        xmat += ft_exact_bytes((int)dimA) / 8;
        S->F.exact_mask |= 1ull << A;
    }
    S->F.nitems = (int)items->size();
    S->smem = ft_smem(S->F.P, nsec);
    if (S->smem > 227 * 1024) return fail(HM_EINVAL, "ftlm_run: shared memory plan too large");
    // co-resident CTAs per SM: the fewest any tiling allows (at most FT_CTAS)
    int per_sm = FT_CTAS;
    for (int vt : {1, 2, 4}) {
        const void *kfn = pick_kernel(S->F.P.nc, vt);
        int p = 0;
        HM_CUDA(raise_smem_limit(kfn, (int)S->smem));
        HM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, kfn, FT_NT, S->smem));
        per_sm = std::min(per_sm, p);
    }
    if (per_sm < 1) return fail(HM_EINVAL, "ftlm_run: kernel does not fit on an SM");
    S->F.ck_rows = ft_chunk_rows(n_sites);
    // cooperative: all resident.  No more CTAs than their warps have chunks (N <= 16): the grid
    // barriers and the sums over the CTAs are most of a step there; but one for each eight vectors of a
    // sector, so that the sums go in one round (60 steps of 20 vectors, N = 10: 5.4 -> 4.4 ms, N = 12 3.8 -> 3.5)
    const uint64_t nck = ((1ull << n_sites) + S->F.ck_rows - 1) / S->F.ck_rows + (uint64_t)nsec;
    const uint64_t want = std::max<uint64_t>((nck + FT_NT / 32 - 1) / (FT_NT / 32), (uint64_t)nsec * FT_OCT);
    S->nctas = (int)std::min<uint64_t>((uint64_t)sm_count() * per_sm, want);
    S->F.nctas = (unsigned)S->nctas;
    ft_ranges(n_sites, K, S->full, *items, S->nctas * (FT_NT / 32), S->F.ck_rows, &S->wr, &S->slo, &S->crng, &S->ck_it0,
              &S->ck_cs);
    S->F.nchunks = (uint32_t)S->ck_it0.size();
    S->L = ft_layout(n_sites, nsec, R, steps, S->F.nitems, S->nctas, n_t, S->xcd.size(), (size_t)xmat,
                     S->F.nchunks, (size_t)S->F.hop.stride << K);
    return HM_OK;
}

static void ft_bind(FtSetup *S, unsigned char *w) {
    const FtLayout &L = S->L;
    FtDev &d = S->F.d;
    const size_t nst = (size_t)S->F.nsec * FT_W;
    d.q0 = (float *)(w + L.q0);
    d.q1 = (float *)(w + L.q1);
    double *st = (double *)(w + L.st);
    d.sig_cur = st; d.sig_prev = st + nst; d.beta_prev = st + 2 * nst; d.scale = st + 3 * nst; d.as = st + 4 * nst;
    d.done = (int *)(st + 5 * nst);
    d.nsteps = d.done + nst;
    d.alpha = (double *)(w + L.ab);
    d.beta = d.alpha + nst * S->F.steps;
    d.part = (double *)(w + L.part);
    d.wr = (const FtRange *)(w + L.wr);
    d.slo = (const uint32_t *)(w + L.slo);
    d.cta_rng = (const uint2 *)(w + L.crng);
    d.parta = (double *)(w + L.parta);
    d.partc = (double *)(w + L.partc);
    d.ck_it0 = (const uint32_t *)(w + L.ckit);
    d.ck_cs = (const uint32_t *)(w + L.ckcs);
    d.sec_active = (int *)(w + L.sec);
    d.bar = (GridBar *)(w + L.bar);
    d.items = (const uint32_t *)(w + L.items);
    d.rowoff = (const uint64_t *)(w + L.rowoff);
    d.secdim = (const uint32_t *)(w + L.secdim);
    d.hops = (uint16_t *)(w + L.hops);
    d.theta = (double *)(w + L.theta);
    d.tau = (double *)(w + L.tau);
    d.mlen = (int *)(w + L.mlen);
    double *th = (double *)(w + L.therm);
    d.zsum = th;
    d.esum = th + 1;   // reassigned with n_t below
    d.eref = th;
}

static int ft_launch_persistent(FtSetup *S, int vt, cudaStream_t st) {
    const void *kfn = pick_kernel(S->F.P.nc, vt);
    HM_CUDA(raise_smem_limit(kfn, (int)S->smem));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S->nctas);
    cfg.blockDim = dim3(FT_NT);
    cfg.dynamicSmemBytes = S->smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    void *args[] = {(void *)&S->F};
    HM_CUDA(cudaLaunchKernelExC(&cfg, kfn, args));
    return HM_OK;
}

}  // namespace hm

using namespace hm;

extern "C" {

int ftlm_workspace(int n_sites, int two_s, int n_bonds, const int32_t *u, const int32_t *v,
                   const double *J, int R, int steps, int n_t, size_t *bytes) {
    if (!bytes) return fail(HM_EINVAL, "bytes is NULL");
    FtSetup S;
    std::vector<uint32_t> items;
    HM_TRY(ft_prepare(n_sites, two_s, n_bonds, u, v, J, R, steps, n_t, &S, &items));
    *bytes = S.L.total;
    return HM_OK;
}

int ftlm_run(int n_sites, int two_s, int n_bonds, const int32_t *u, const int32_t *v, const double *J,
             int R, int steps, uint64_t seed, const double *temps, int n_t, double *Z, double *E,
             double *e_ref, double *theta, double *tau, int *mlen, int vt, void *work,
             size_t work_bytes, void *stream) {
    if (n_t > 0 && (!temps || !Z || !E)) return fail(HM_EINVAL, "temperature arrays are NULL");
    if (vt != 0 && vt != 1 && vt != 2 && vt != 4) return fail(HM_EINVAL, "vt must be 0 (autotune), 1, 2 or 4");
    FtSetup S;
    std::vector<uint32_t> items;
    HM_TRY(ft_prepare(n_sites, two_s, n_bonds, u, v, J, R, steps, n_t, &S, &items));
    if (!work || work_bytes < S.L.total || ((uintptr_t)work & 255))
        return fail(HM_EWORKSPACE, "ftlm_run needs %zu workspace bytes (256-byte aligned)", S.L.total);
    cudaStream_t st = as_stream(stream);
    unsigned char *w = (unsigned char *)work;
    ft_bind(&S, w);
    S.F.seed = seed;
    S.F.barrier_ns = ft_barrier_ns();
    double *therm = (double *)(w + S.L.therm);
    S.F.d.eref = therm;
    S.F.d.zsum = therm + 1;
    S.F.d.esum = therm + 1 + n_t;
    // host-built inputs: items, sector row offsets and dimensions
    const int nsec = S.F.nsec;
    std::vector<uint64_t> rowoff(nsec + 1, 0);
    std::vector<uint32_t> dims(nsec);
    {
        const int W = S.full.view.S2 * n_sites + 1;
        for (int A = 0; A < nsec; ++A) {
            dims[A] = (uint32_t)S.full.D[(size_t)n_sites * W + A];
            rowoff[A + 1] = rowoff[A] + dims[A];
        }
    }
    HM_CUDA(cudaMemcpyAsync(w + S.L.items, items.data(), items.size() * 4, cudaMemcpyHostToDevice, st));
    HM_CUDA(cudaMemcpyAsync(w + S.L.rowoff, rowoff.data(), rowoff.size() * 8, cudaMemcpyHostToDevice, st));
    HM_CUDA(cudaMemcpyAsync(w + S.L.secdim, dims.data(), dims.size() * 4, cudaMemcpyHostToDevice, st));
    HM_CUDA(cudaMemcpyAsync(w + S.L.wr, S.wr.data(), S.wr.size() * sizeof(FtRange), cudaMemcpyHostToDevice, st));
    HM_CUDA(cudaMemcpyAsync(w + S.L.crng, S.crng.data(), S.crng.size() * sizeof(uint2), cudaMemcpyHostToDevice, st));
    HM_CUDA(cudaMemcpyAsync(w + S.L.slo, S.slo.data(), S.slo.size() * 4, cudaMemcpyHostToDevice, st));
    if (!S.ck_it0.empty())
        HM_CUDA(cudaMemcpyAsync(w + S.L.ckit, S.ck_it0.data(), S.ck_it0.size() * 4, cudaMemcpyHostToDevice, st));
    HM_CUDA(cudaMemcpyAsync(w + S.L.ckcs, S.ck_cs.data(), S.ck_cs.size() * 4, cudaMemcpyHostToDevice, st));
    if (!S.xcd.empty())
        HM_CUDA(cudaMemcpyAsync(w + S.L.xcd, S.xcd.data(), S.xcd.size() * 4, cudaMemcpyHostToDevice, st));
    double *d_temps = (double *)(w + S.L.temps);
    if (n_t > 0) HM_CUDA(cudaMemcpyAsync(d_temps, temps, n_t * 8, cudaMemcpyHostToDevice, st));
    k_ft_hops<<<((1u << S.F.P.K) + 127) / 128, 128, 0, st>>>(S.F);
    HM_CUDA(cudaGetLastError());
    // autotune the vectors-per-lane tiling on a short run (2 steps), once per shape
    int use_vt = vt;
    if (use_vt == 0) {
        auto key = std::make_pair(n_sites, S.F.P.nc * 1000 + S.F.P.nhb * 10 + R);
        auto it = g_ft_tuned.find(key);
        if (it != g_ft_tuned.end()) {
            use_vt = it->second;
        } else {
            float best = 1e30f;
            int bvt = 1;
            FtParams keep = S.F;
            S.F.steps = std::min(steps, 2);
            cudaEvent_t e0, e1;
            HM_CUDA(cudaEventCreate(&e0));
            HM_CUDA(cudaEventCreate(&e1));
            for (int cand : {1, 2, 4}) {
                k_ft_init<<<sm_count() * 4, 256, 0, st>>>(S.F);
                HM_CUDA(cudaGetLastError());
                HM_CUDA(cudaEventRecord(e0, st));
                HM_TRY(ft_launch_persistent(&S, cand, st));
                HM_CUDA(cudaEventRecord(e1, st));
                HM_CUDA(cudaEventSynchronize(e1));
                float ms = 0.0f;
                HM_CUDA(cudaEventElapsedTime(&ms, e0, e1));
                if (ms < best) { best = ms; bvt = cand; }
            }
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            S.F = keep;
            use_vt = bvt;
            g_ft_tuned[key] = bvt;
        }
    }
    // the run: init, persistent steps, eigen-decompositions, sums -- one captured graph
    cudaStream_t cap = nullptr, br = nullptr;
    cudaEvent_t ev = nullptr;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ge = nullptr;
    int rc = HM_OK;
    cudaError_t e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&br, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) rc = cuda_fail(e, "ftlm capture");
    if (rc == HM_OK) {
        k_ft_init<<<sm_count() * 4, 256, 0, cap>>>(S.F);
        if ((e = cudaGetLastError()) != cudaSuccess) rc = cuda_fail(e, "k_ft_init");
        if (rc == HM_OK) rc = ft_launch_persistent(&S, use_vt, cap);
        if (rc == HM_OK) {
            const int nst = nsec * FT_W;
            // the exactly diagonalised sectors on a branch beside the eigen-decompositions
            const bool fork = S.F.nexact > 0;
            if (fork && ((e = cudaEventRecord(ev, cap)) != cudaSuccess || (e = cudaStreamWaitEvent(br, ev, 0)) != cudaSuccess))
                rc = cuda_fail(e, "ftlm fork");
            k_ft_eig<<<nst, FT_EIG_NT, (size_t)2 * S.F.steps * 8, cap>>>(S.F);
            if ((e = cudaGetLastError()) != cudaSuccess) rc = cuda_fail(e, "k_ft_eig");
            if (rc == HM_OK && fork) {
                // shared memory for the largest sector that fits; larger ones work in mats
                size_t xs = 0;
                for (int x = 0; x < S.F.nexact; ++x) {
                    const size_t need = ft_exact_bytes(S.F.ex[x].dim);
                    if (need <= FT_X_SMEM) xs = std::max(xs, need);
                }
                if (xs > 0 && (e = raise_smem_limit((const void *)k_ft_exact, xs)) != cudaSuccess)
                    rc = cuda_fail(e, "k_ft_exact shared memory");
                k_ft_exact<<<S.F.nexact, FT_X_NT, xs, br>>>(S.F, S.bp, (const uint32_t *)(w + S.L.xcd),
                                                            (double *)(w + S.L.xmat), xs);
                if ((e = cudaGetLastError()) != cudaSuccess) rc = cuda_fail(e, "k_ft_exact");
                else if ((e = cudaEventRecord(ev, br)) != cudaSuccess || (e = cudaStreamWaitEvent(cap, ev, 0)) != cudaSuccess)
                    rc = cuda_fail(e, "ftlm join");
            }
        }
        cudaError_t e2 = cudaStreamEndCapture(cap, &g);
        if (rc == HM_OK && e2 != cudaSuccess) rc = cuda_fail(e2, "ftlm end capture");
    }
    if (rc == HM_OK && (e = cudaGraphInstantiate(&ge, g, 0)) != cudaSuccess) rc = cuda_fail(e, "ftlm instantiate");
    if (rc == HM_OK && (e = cudaGraphLaunch(ge, st)) != cudaSuccess) rc = cuda_fail(e, "ftlm graph launch");
    if (ge) cudaGraphExecDestroy(ge);
    if (g) cudaGraphDestroy(g);
    if (ev) cudaEventDestroy(ev);
    if (br) cudaStreamDestroy(br);
    if (cap) cudaStreamDestroy(cap);
    HM_TRY(rc);
    if (n_t > 0) {
        double *mins = (double *)(w + S.L.tsum), *zs = mins + nsec, *es = zs + (size_t)nsec * n_t;
        k_ft_min<<<nsec, 256, 0, st>>>(S.F, mins);
        k_ft_thermo<<<dim3(nsec, n_t), 256, 0, st>>>(S.F, d_temps, mins, zs, es);
        k_ft_thermo_fin<<<(n_t + 255) / 256, 256, 0, st>>>(S.F, mins, zs, es, n_t);
        HM_CUDA(cudaGetLastError());
    }
    GridBar bar;
    HM_CUDA(cudaMemcpyAsync(&bar, S.F.d.bar, sizeof bar, cudaMemcpyDeviceToHost, st));
    std::vector<double> th(1 + 2 * (size_t)n_t);
    HM_CUDA(cudaMemcpyAsync(th.data(), therm, th.size() * 8, cudaMemcpyDeviceToHost, st));
    HM_CUDA(cudaStreamSynchronize(st));
    if (bar.abort) return fail(HM_ETIMEOUT, "ftlm_run: a grid barrier timed out");
    if (e_ref) *e_ref = th[0];
    for (int i = 0; i < n_t; ++i) { Z[i] = th[1 + i]; E[i] = th[1 + n_t + i]; }
    const size_t nst = (size_t)nsec * FT_W;
    if (theta) HM_CUDA(cudaMemcpy(theta, S.F.d.theta, nst * steps * 8, cudaMemcpyDeviceToHost));
    if (tau) HM_CUDA(cudaMemcpy(tau, S.F.d.tau, nst * steps * 8, cudaMemcpyDeviceToHost));
    if (mlen) HM_CUDA(cudaMemcpy(mlen, S.F.d.mlen, nst * 4, cudaMemcpyDeviceToHost));
    return use_vt;   // > 0: the tiling that ran (informational)
}

}  // extern "C"
