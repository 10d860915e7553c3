// hm_row.cuh -- the per-row kernel bodies of Eq. (E-4-b): apply every bond term of
// Eq. (E-2-1) to the row's own basis state, encode each target, gather x there.
//
// Two forms.  The sweep form (RowPlan, row_sweep) decodes the row and forms every exchange
// target in one pass over the positions; it serves every sector whose tables fit in shared
// memory (row_plan).  The table form below it (row_apply) is the general one: it also serves the
// larger tables and the successor-rule row runs (HM_ROW_RUN).
#pragma once

#include <type_traits>

#include "hm_internal.cuh"

namespace hm {

// ---- the sweep form ------------------------------------------------------------------------
// An exchange of p < q by dp (digit at p by dp, at q by -dp) changes the rank terms of
// positions p..q (Sec. 3.2).  With the running digit sums S_r of the row and CD of hm_internal.cuh
//   E_dp = CD[p][S_p + dp][a_p + dp] - CD[p][S_p][a_p]
//   F_dp = CD[q][S_q][a_q - dp] - CD[q][S_q][a_q]
//   G_dp[r] = CD[r][S_r + dp][a_r] - CD[r][S_r][a_r]        (p < r < q)
// the index change is E_dp + sum_{p < r < q} G_dp[r] + F_dp.  The differences are tables beside CD
// (basis_build), so a position costs one lookup.  The sweep goes down from position N - 1: it
// finds the digit (Sec. 3.1), adds G to the suffix sums Q_dp, keeps R_dp = F_dp - Q_dp[q] of a
// site that is the upper end of a bond in one of a few per-thread slots, and, for the bonds whose
// lower end the position is, has the target as i + (E_dp + Q_dp[p + 1]) + R_dp.
// What bounds it in FP64 is the binary64 pipe (64 cycles a warp instruction and SM quarter), so
// the exchange coefficients -J_b f are tables too (one multiply-add an exchange) and the
// diagonal is an exact integer sum, converted once a row.  The gathers of one bond are in flight
// while those of the bond before are added.  Measured (s = 3/2 ring, N = 12, 1.7 M rows, FP64):
// k_matvec, the table form, 362 us; this form 110 us.
// Aligned to a 16-byte shared load at most: the tables start on 16 bytes, behind the coefficients.
template <class I> struct alignas(16) RowEF { I ep, fp, em, fm; };
template <class I> struct alignas(2 * sizeof(I)) RowG { I gp, gm; };

constexpr int ROW_NT = 256;          // threads per CTA of the row kernels
constexpr int ROW_SLOT_NONE = 255;

// Lists of more than ROW_MB bonds take the table form: a kernel's parameters are copied at every
// launch (4.4 KB here)
constexpr int ROW_MB = 128;
struct RowPlan {
    int nslots, nc;
    double dscale, dscale_low;       // 2^-s of dC, 2^-(s+t) of dL
    // per position: first bond whose lower end it is | their number << 10 | slot of its R << 20
    // (ROW_SLOT_NONE: not the upper end of a bond)
    uint32_t pos[HM_MAX_SITES];
    uint32_t bond[ROW_MB];           // bit offset of the upper end's digit | its slot << 8 | class << 16
    double jm[ROW_MB];               // by class (distinct coupling): -J
    long long dC[ROW_MB];            // by class: round(-J / 4 2^s), and the remainder 2^-t dL; dlow: some dL is not zero
    int dL[ROW_MB];
    int dlow;
    long long dsum;                  // sum of dC over the bonds (s = 1/2: the diagonal is dsum - 2 sum over unequal spins)
    double hs_pdn[64], hs_pup[64];   // as in BondParams
};

// the plan of a bond list; 0, or 1 when the table form has to serve: more than ROW_MB bonds, tables
// above the shared memory, couplings so far apart that the integer diagonal does not hold
// them exactly, or row runs (HM_ROW_RUN).  *smem: dynamic shared memory of a CTA for accumulation type size es
int row_plan(const SectorView &sv, const BondParams &bp, int es, RowPlan *P, size_t *smem);

// CTAs of a row kernel: one resident wave at most (every CTA stages the tables), and no more
// than grid_blocks, for which the workspaces' partial sums are sized
template <class F>
inline int row_grid(uint64_t rows, F kern, size_t smem) {
    const int need = grid_blocks(rows, ROW_NT);
    if (need <= sm_count()) return need;             // one CTA an SM always fits: no query (about 1 us of a call's 27)
    int per = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, ROW_NT, smem) != cudaSuccess) {
        cudaGetLastError();
        per = 1;
    }
    const int wave = sm_count() * (per < 1 ? 1 : per);
    return need < wave ? need : wave;
}

__host__ __device__ __forceinline__ size_t row_coef_bytes(const RowPlan &P, int S2, int es) {
    const int n1 = S2 + 1;
    return ((size_t)P.nc * 2 * n1 * n1 * es + 15) & ~(size_t)15;
}

// shared layout: exchange coefficients | E, F | G | CD | slots
template <class I, class Acc>
struct RowTabs {
    const Acc *coef;
    const RowEF<I> *ef;
    const RowG<I> *g;
    const I *cd;
    RowG<I> *slots;                  // this thread's, stride ROW_NT
};
template <class I>
__host__ __device__ __forceinline__ size_t row_tab_bytes(const SectorView &sv) {
    return ((size_t)sv.cd_len * 7 * sizeof(I) + 15) & ~(size_t)15;
}

template <class I, class Acc>
__device__ __forceinline__ RowTabs<I, Acc> row_stage(const SectorView &sv, const RowPlan &P, unsigned char *smem) {
    const int n1 = sv.S2 + 1, n2 = n1 * n1;
    Acc *coef = reinterpret_cast<Acc *>(smem);
    for (int k = threadIdx.x; k < P.nc * 2 * n2; k += ROW_NT) {
        const int c = k / (2 * n2), m = k % (2 * n2), e = m % n2, h = (e / n1) * 8 + e % n1;
        const double f = m < n2 ? P.hs_pdn[h] : P.hs_pup[h];
        coef[k] = (Acc)P.jm[c] * (Acc)f;
    }
    I *cd = reinterpret_cast<I *>(smem + row_coef_bytes(P, sv.S2, sizeof(Acc)));
    // device tables: CD, then E/F, then G (basis_build); in shared memory the wide ones first
    const I *src = (const I *)sv.cd;
    for (int k = threadIdx.x; k < 6 * sv.cd_len; k += ROW_NT) cd[k] = src[sv.cd_len + k];
    for (int k = threadIdx.x; k < sv.cd_len; k += ROW_NT) cd[6 * (size_t)sv.cd_len + k] = src[k];
    RowTabs<I, Acc> t;
    t.coef = coef;
    t.ef = reinterpret_cast<const RowEF<I> *>(cd);
    t.g = reinterpret_cast<const RowG<I> *>(cd + 4 * (size_t)sv.cd_len);
    t.cd = cd + 6 * (size_t)sv.cd_len;
    t.slots = reinterpret_cast<RowG<I> *>(smem + row_coef_bytes(P, sv.S2, sizeof(Acc)) + row_tab_bytes<I>(sv)) + threadIdx.x;
    __syncthreads();
    return t;
}

// every bond of the state of index i: f(class, a_p, a_q, target of s-_p s+_q (dp = +1), target of
// s+_p s-_q (dp = -1)); a target is meaningful only when the exchange is allowed
template <class I, class Acc, class F>
__device__ __forceinline__ void row_sweep(const SectorView &sv, const RowPlan &P, const RowTabs<I, Acc> &T, I i, F &&f) {
    const int bits = sv.bits, S2 = sv.S2;
    const uint32_t mask = (1u << bits) - 1u;
    const int o2 = S2 + 1 < 2 ? S2 + 1 : 2, o3 = S2 + 1 < 3 ? S2 + 1 : 3;   // entry S2 + 1 is above every index
    uint64_t w = 0;
    int S = sv.A, row = (sv.N - 1) * sv.cd_rowlen;
    I res = i, qp = 0, qm = 0;
    for (int r = sv.N - 1; r >= 0; --r, row -= sv.cd_rowlen) {
        const int ix = row + S * sv.cd_w;
        int a = S;
        if (r > 0) {                               // the digit whose cumulative range holds res
            const I *c = T.cd + ix;
            a = (c[1] <= res) + (c[o2] <= res) + (c[o3] <= res);
            for (int k = 4; k <= S2; ++k) a += c[k] <= res;
            res -= c[a];
        }
        w |= (uint64_t)a << (r * bits);
        const RowEF<I> e = T.ef[ix + a];
        const RowG<I> g = T.g[ix + a];
        const I lp = i + e.ep + qp, lm = i + e.em + qm;
        qp += g.gp;
        qm += g.gm;
        const uint32_t pr = P.pos[r];
        const int sl = (int)(pr >> 20);
        if (sl != ROW_SLOT_NONE) T.slots[sl * ROW_NT] = RowG<I>{(I)(e.fp - qp), (I)(e.fm - qm)};
        const int t1 = (int)(pr & 1023u) + (int)((pr >> 10) & 1023u);
        for (int t = (int)(pr & 1023u); t < t1; ++t) {
            const uint32_t br = P.bond[t];
            const int aq = (int)((uint32_t)(w >> (br & 255u)) & mask);
            const RowG<I> R = T.slots[((br >> 8) & 255u) * ROW_NT];
            f((int)(br >> 16), a, aq, (I)(lp + R.gp), (I)(lm + R.gm));
        }
        S -= a;
    }
}

// (H x)_i for NV columns: *dg the diagonal element, acc the exchange sums.  MODE: ROW_ONE one class
// of couplings (a ring, a uniform lattice); ROW_HALF s = 1/2, where a bond allows one direction at
// most, so one gather and one multiply-add serve it; ROW_ANY the rest; ROW_LOW any list whose diagonal has a
// low part (of its own, since a test for it costs the others 5%)
enum { ROW_ANY = 0, ROW_ONE = 1, ROW_HALF = 2, ROW_LOW = 3 };
// f(std::integral_constant<int, MODE>) for the plan's mode
template <class F>
inline auto row_dispatch(const SectorView &sv, const RowPlan &P, F &&f) {
    if (P.nc == 1 && sv.S2 > 1) return f(std::integral_constant<int, ROW_ONE>());
    if (P.dlow) return f(std::integral_constant<int, ROW_LOW>());
    if (sv.S2 == 1) return f(std::integral_constant<int, ROW_HALF>());
    return f(std::integral_constant<int, ROW_ANY>());
}
template <int MODE>
__device__ __forceinline__ double row_diag(const RowPlan &P, long long di, int dl, int k1) {
    if constexpr (MODE == ROW_ONE) return 0.25 * P.jm[0] * (double)k1;
    if constexpr (MODE == ROW_HALF)
        return (double)(long long)((unsigned long long)P.dsum - 2ull * (unsigned long long)di) * P.dscale;
    const double d = (double)di * P.dscale;
    return MODE == ROW_LOW ? fma((double)dl, P.dscale_low, d) : d;
}
template <class I, class T, class Acc, int NV, int MODE>
__device__ __forceinline__ void row_hops(const SectorView &sv, const RowPlan &P, const RowTabs<I, Acc> &Tb, I i,
                                         const T *__restrict__ x, int ld, int c0, Acc *acc, Acc *dg) {
    const int S2 = sv.S2, n1 = S2 + 1, n2 = n1 * n1;
    Acc cp[2] = {Acc(0), Acc(0)};                  // the bond before: coefficients and gathered values
    T vp[2][NV];
    long long di = 0;
    int k1 = 0, dl = 0;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        acc[k] = Acc(0);
        vp[0][k] = vp[1][k] = T(0);
    }
    row_sweep(sv, P, Tb, i, [&](int c, int ap, int aq, I jp, I jm) {
        if constexpr (MODE == ROW_HALF) {
            // a_p = 1: the first digits (1, 0) of the table, -J / 2 as for (0, 1)
            const bool ne = ap != aq;
            if (ne) di += P.dC[c];
            const Acc cn = Tb.coef[c * 8 + 2];
            const T *xr = x + (size_t)(ap ? jm : jp) * ld + c0;
            T vn[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) vn[k] = ne ? __ldg(xr + k) : T(0);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                acc[k] = fma(cp[0], (Acc)vp[0][k], acc[k]);
                vp[0][k] = vn[k];
            }
            cp[0] = cn;
        } else {
            const int kk = (S2 - 2 * ap) * (S2 - 2 * aq);
            if constexpr (MODE == ROW_ONE) k1 += kk;
            else {
                di += P.dC[c] * kk;
                if constexpr (MODE == ROW_LOW) dl += P.dL[c] * kk;
            }
            const Acc *co = Tb.coef + ap * n1 + aq;
            if constexpr (MODE != ROW_ONE) co += c * 2 * n2;
            const bool dn = ap >= 1 && aq < S2, up = ap < S2 && aq >= 1;
            // a coefficient whose exchange is not allowed is zero in the table
            const Acc c1 = co[0], c2 = co[n2];
            const T *x1 = x + (size_t)jm * ld + c0, *x2 = x + (size_t)jp * ld + c0;
            T v1[NV], v2[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                v1[k] = dn ? __ldg(x1 + k) : T(0);
                v2[k] = up ? __ldg(x2 + k) : T(0);
            }
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                acc[k] = fma(cp[0], (Acc)vp[0][k], acc[k]);
                acc[k] = fma(cp[1], (Acc)vp[1][k], acc[k]);
                vp[0][k] = v1[k];
                vp[1][k] = v2[k];
            }
            cp[0] = c1;
            cp[1] = c2;
        }
    });
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        acc[k] = fma(cp[0], (Acc)vp[0][k], acc[k]);
        if constexpr (MODE != ROW_HALF) acc[k] = fma(cp[1], (Acc)vp[1][k], acc[k]);
    }
    *dg = (Acc)row_diag<MODE>(P, di, dl, k1);
}

// ---- the table form ------------------------------------------------------------------------

// Tables one CTA needs in shared memory: the exchange factors, then the rank table CD.
// Layout: double hs[128] | float hsf[128] | CD.  hs[0..64) = pdn, hs[64..128) = pup.
template <class I>
__device__ __forceinline__ I *stage_tables(const SectorView &sv, const BondParams &bp,
                                           unsigned char *smem_raw, const double **pdn,
                                           const double **pup) {
    double *hs = reinterpret_cast<double *>(smem_raw);
    float *hsf = reinterpret_cast<float *>(smem_raw + 128 * sizeof(double));
    I *cd = reinterpret_cast<I *>(smem_raw + 128 * sizeof(double) + 128 * sizeof(float));
    for (int k = threadIdx.x; k < 64; k += blockDim.x) {
        hs[k] = bp.hs_pdn[k];
        hs[64 + k] = bp.hs_pup[k];
        hsf[k] = (float)bp.hs_pdn[k];
        hsf[64 + k] = (float)bp.hs_pup[k];
    }
    for (int k = threadIdx.x; k < sv.cd_len; k += blockDim.x) cd[k] = ((const I *)sv.cd)[k];
    __syncthreads();
    *pdn = hs;
    *pup = hs + 64;
    return cd;
}

// Per-thread scratch of the suffix form of the target encode (row_apply with px): suffix
// sums Q+[r], Q-[r] (r = 1..N, Q[N] = 0) of the rank-term changes a +-1 shift of the
// running digit sum causes at positions r..N-1, and the running digit sums S[r].  Laid
// out [slot][thread]: the threads of a warp visit the same bond together, so they read
// the same slot of consecutive threads (no bank conflict).
template <class I>
__host__ __device__ __forceinline__ size_t row_px_bytes(const SectorView &sv) {
    const size_t a = (size_t)2 * (sv.N + 1) * ROW_NT * sizeof(I);
    return ((a + 15) & ~(size_t)15) + (((size_t)sv.N * ROW_NT + 15) & ~(size_t)15);
}
// the suffix form is used while its scratch stays below this (else the per-hop walk)
constexpr size_t ROW_PX_MAX = 96 * 1024;

template <class I>
__host__ __forceinline__ size_t row_smem_bytes(const SectorView &sv) {
    size_t b = 128 * sizeof(double) + 128 * sizeof(float) + (size_t)sv.cd_len * sizeof(I);
    b = (b + 15) & ~(size_t)15;
    if (row_px_bytes<I>(sv) <= ROW_PX_MAX) b += row_px_bytes<I>(sv);
    return b;
}

// scratch of the prefix form for this thread (nullptr when the walk is used)
template <class I>
__device__ __forceinline__ I *row_px_base(const SectorView &sv, unsigned char *smem_raw) {
    if (row_px_bytes<I>(sv) > ROW_PX_MAX) return nullptr;
    size_t b = 128 * sizeof(double) + 128 * sizeof(float) + (size_t)sv.cd_len * sizeof(I);
    b = (b + 15) & ~(size_t)15;
    return reinterpret_cast<I *>(smem_raw + b) + threadIdx.x;
}

// views of the per-thread scratch (px = row_px_base; nullptr = no scratch)
template <class I>
struct RowPx {
    I *Qp, *Qm;          // [r * ROW_NT], r = 0..N
    uint8_t *S;          // [r * ROW_NT], r = 0..N-1
    __device__ __forceinline__ RowPx(I *px, int N) {
        Qp = px;
        Qm = px ? px + (size_t)(N + 1) * ROW_NT : nullptr;
        S = px ? reinterpret_cast<uint8_t *>(px - threadIdx.x) +
                     (((size_t)2 * (N + 1) * ROW_NT * sizeof(I) + 15) & ~(size_t)15) + threadIdx.x
               : nullptr;
    }
};

// running digit sums and suffix sums of the rank-term changes of positions lo..hi (descending
// from hi, whose running sum S_hi is given; Q[hi + 1] must be current)
template <class I>
__device__ __forceinline__ void px_fill(const Codec<I> &c, uint64_t w, const RowPx<I> &x, int hi, int S) {
    I qp = x.Qp[(size_t)(hi + 1) * ROW_NT], qm = x.Qm[(size_t)(hi + 1) * ROW_NT];
    for (int r = hi; r >= 0; --r) {
        const int a = dig(w, r, c.bits);
        x.S[(size_t)r * ROW_NT] = (uint8_t)S;
        if (r >= 1) {
            const I t0 = c.at(r, S, a);
            qp += (S < c.A ? c.at(r, S + 1, a) : t0) - t0;
            qm += (S > 0 ? c.at(r, S - 1, a) : t0) - t0;
            x.Qp[(size_t)r * ROW_NT] = qp;
            x.Qm[(size_t)r * ROW_NT] = qm;
        }
        S -= a;
    }
}

// scratch for state w (all positions)
template <class I>
__device__ __forceinline__ void px_full(const Codec<I> &c, uint64_t w, const RowPx<I> &x) {
    x.Qp[(size_t)c.N * ROW_NT] = 0;
    x.Qm[(size_t)c.N * ROW_NT] = 0;
    px_fill(c, w, x, c.N - 1, c.A);
}

// Successor rule (Sec. 3.1): the state of the next index.  The lowest position k whose
// digit can give one unit to position k+1 does so, and the units left at positions
// 0..k are refilled from the bottom, at most 2s each.  Returns k (digits 0..k+1 changed;
// the running digit sums above are unchanged), or -1 for the last state of the sector.
__device__ __forceinline__ int successor_word(uint64_t &w, int N, int S2, int bits) {
    const uint64_t m = (1ull << bits) - 1ull;
    int units = 0, k = -1;
    for (int p = 0; p + 1 < N; ++p) {
        const int a = (int)((w >> (p * bits)) & m);
        units += a;
        if (a > 0 && (int)((w >> ((p + 1) * bits)) & m) < S2) { k = p; break; }
    }
    if (k < 0) return -1;
    w += 1ull << ((k + 1) * bits);
    w &= ~((1ull << ((k + 1) * bits)) - 1ull);
    units -= 1;
    for (int p = 0; p <= k && units > 0; ++p) {
        const int t = units < S2 ? units : S2;
        w |= (uint64_t)t << (p * bits);
        units -= t;
    }
    return k;
}

// every row of this thread's share.  run = 1: one row per thread per grid stride, each
// decoded (Sec. 3.1 decode rule; consecutive threads take consecutive rows, so the row
// loads coalesce).  run > 1: runs of `run` consecutive rows per thread, the first decoded
// and the others reached by the successor rule, the scratch (if any) following the state
// incrementally.  f(row, w) sees the scratch of w.
template <class I, class F>
__device__ __forceinline__ void row_runs(const Codec<I> &c, uint64_t dim, I *px, int run, F &&f) {
    const RowPx<I> x(px, c.N);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    if (run <= 1) {
        for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r < dim; r += stride) {
            const uint64_t w = c.decode((I)r);
            if (px) px_full(c, w, x);
            f(r, w);
        }
        return;
    }
    const uint64_t nruns = (dim + run - 1) / run;
    for (uint64_t k0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k0 < nruns; k0 += stride) {
        uint64_t r = k0 * run;
        const uint64_t rend = r + run < dim ? r + run : dim;
        uint64_t w = c.decode((I)r);
        if (px) px_full(c, w, x);
        for (;;) {
            f(r, w);
            if (++r >= rend) break;
            const int k = successor_word(w, c.N, c.S2, c.bits);
            if (px) px_fill(c, w, x, k + 1, x.S[(size_t)(k + 1) * ROW_NT]);
        }
    }
}

// run length of the row kernels: HM_ROW_RUN (1..64, default 1)
int row_run_len();

template <class Acc>
__device__ __forceinline__ Acc jm_of(const BondParams &bp, int t) {
    if constexpr (sizeof(Acc) == 8) return (Acc)bp.jm[t];
    else return (Acc)bp.jmf[t];
}

// (H x)_i for NV vector columns of a row-major [dim][ld] array starting at column c0.
// T is the storage type, Acc the accumulation type.  Returns the diagonal element in
// *diag_out (as Acc) and the off-diagonal sum in acc[]; the caller forms
// y = diag * x_i + acc, the same association as the oracle's row.
//
// Target encode (Sec. 3.2): an exchange moves the digit at p by dp and the one at q > p by
// -dp, so only the rank terms of positions p..q change, and those strictly between p and
// q change only through their running digit sum (S_r -> S_r + dp).  With px (the
// per-thread scratch of row_px_bytes, describing w: px_full / row_runs) every exchange
// costs its two end terms and Q_dp[p+1] - Q_dp[q], the suffix sums
// Q_dp[r] = sum_{t=r..N-1} (CD[t][S_t + dp][a_t] - CD[t][S_t][a_t]); without it each
// exchange walks positions p..q (Codec::delta).
template <class I, class T, class Acc, int NV>
__device__ __forceinline__ void row_apply(const Codec<I> &c, const BondParams &bp,
                                          const double *hs_pdn, const double *hs_pup,
                                          I i, uint64_t w, const T *__restrict__ x, int ld,
                                          int c0, Acc *acc, Acc *diag_out, I *px = nullptr) {
    const int S2 = c.S2, bits = c.bits;
    // coefficients in the accumulation type: an FP32 product never touches the FP64 pipe
    const Acc half = Acc(0.5) * Acc(S2);
    // pdn table base; pup = pdn + 64 (doubles) -- for floats the copy starts 128 doubles in
    const Acc *tpdn, *tpup;
    if constexpr (sizeof(Acc) == 8) {
        tpdn = reinterpret_cast<const Acc *>(hs_pdn);
        tpup = reinterpret_cast<const Acc *>(hs_pup);
    } else {
        tpdn = reinterpret_cast<const Acc *>(hs_pdn + 128);
        tpup = tpdn + 64;
    }
    Acc dg = Acc(0);
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = Acc(0);
    const RowPx<I> sx(px, c.N);
    // index change of the exchange (p, q, dp) from the suffix sums of the scratch
    auto delta_px = [&](int p, int q, int ap, int aq, int dp) -> I {
        const int Sq = sx.S[(size_t)q * ROW_NT];
        const I *Q = dp > 0 ? sx.Qp : sx.Qm;
        I d = Q[(size_t)(p + 1) * ROW_NT] - Q[(size_t)q * ROW_NT] + (c.at(q, Sq, aq - dp) - c.at(q, Sq, aq));
        if (p >= 1) {
            const int Sp = sx.S[(size_t)p * ROW_NT];
            d += c.at(p, Sp + dp, ap + dp) - c.at(p, Sp, ap);
        }
        return d;
    };
    for (int t = 0; t < bp.nb; ++t) {
        const int p = bp.p[t], q = bp.q[t];
        const int ap = dig(w, p, bits), aq = dig(w, q, bits);
        const Acc jm = jm_of<Acc>(bp, t);
        dg += jm * (half - Acc(ap)) * (half - Acc(aq));
        if (ap >= 1 && aq < S2) {          // s+_p s-_q
            const I j = i + (px ? delta_px(p, q, ap, aq, -1) : c.delta(w, p, q, -1));
            const Acc cf = jm * tpdn[ap * 8 + aq];
            const T *xr = x + (size_t)j * ld + c0;
#pragma unroll
            for (int k = 0; k < NV; ++k) acc[k] += cf * (Acc)xr[k];
        }
        if (ap < S2 && aq >= 1) {          // s-_p s+_q
            const I j = i + (px ? delta_px(p, q, ap, aq, +1) : c.delta(w, p, q, +1));
            const Acc cf = jm * tpup[ap * 8 + aq];
            const T *xr = x + (size_t)j * ld + c0;
#pragma unroll
            for (int k = 0; k < NV; ++k) acc[k] += cf * (Acc)xr[k];
        }
    }
    *diag_out = dg;
}

}  // namespace hm
