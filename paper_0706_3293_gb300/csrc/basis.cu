// basis.cu -- sector tables (Sec. 3, Eq. E-3-c), the codec test hooks (Sec. 3.1, 3.2),
// bond preparation, seeded start vectors and error reporting.
#include <stdlib.h>
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>

#include "hm_row.cuh"

namespace hm {

static thread_local std::string g_err;

int fail(int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

int cuda_fail(cudaError_t e, const char *what) {
    return fail(HM_ECUDA, "%s: %s (%s)", what, cudaGetErrorString(e), cudaGetErrorName(e));
}

cudaStream_t as_stream(void *s) { return reinterpret_cast<cudaStream_t>(s); }

int digit_bits(int two_s) { return two_s == 1 ? 1 : (two_s <= 3 ? 2 : 4); }

int check_sector(int n_sites, int two_s, int two_m, int *A) {
    if (two_s < 1 || two_s > 7) return fail(HM_EINVAL, "two_s must be in 1..7 (got %d)", two_s);
    if (n_sites < 1 || n_sites > HM_MAX_SITES)
        return fail(HM_EINVAL, "n_sites must be in 1..%d (got %d)", HM_MAX_SITES, n_sites);
    if (n_sites * digit_bits(two_s) > 64)
        return fail(HM_EINVAL, "n_sites * bits-per-digit exceeds 64 (N=%d, 2s=%d)", n_sites, two_s);
    long t = (long)n_sites * two_s - two_m;
    if (t % 2 != 0 || t < 0 || t > 2L * n_sites * two_s)
        return fail(HM_EPARITY, "2M=%d is not a magnetic quantum number of N=%d spins 2s=%d",
                    two_m, n_sites, two_s);
    *A = (int)(t / 2);
    return HM_OK;
}

// D(k, a) by Eq. (E-3-c) and CD[p][S][a] = sum_{n<a} D(p, S-n); entries of rows
// (p, S) that no sector state reaches are stored as 0.
int build_tables(int n_sites, int two_s, int two_m, hm_basis *b) {
    int A = 0;
    HM_TRY(check_sector(n_sites, two_s, two_m, &A));
    const int N = n_sites, S2 = two_s, W = S2 * N + 1;
    const uint64_t LIM = 1ull << 63;
    b->D.assign((size_t)(N + 1) * W, 0);
    auto D = [&](int k, int a) -> uint64_t {
        if (k < 0 || k > N || a < 0 || a > S2 * k) return 0;
        return b->D[(size_t)k * W + a];
    };
    b->D[0] = 1;
    for (int k = 1; k <= N; ++k)
        for (int a = 0; a <= S2 * k; ++a) {
            uint64_t s = 0;
            for (int n = 0; n <= S2; ++n) {
                s += D(k - 1, a - n);
                if (s >= LIM) return fail(HM_EOVERFLOW, "D(%d,%d) exceeds 2^63", k, a);
            }
            b->D[(size_t)k * W + a] = s;
        }
    const uint64_t dim = D(N, A);
    SectorView &v = b->view;
    v.N = N; v.S2 = S2; v.A = A; v.bits = digit_bits(S2);
    v.cd_w = S2 + 2;
    v.cd_rowlen = (A + 1) * v.cd_w;
    v.cd_len = N * v.cd_rowlen;
    v.dim = dim;
    v.idx64 = dim >= (1ull << 32) ? 1 : 0;
    v.cd = nullptr;
    b->cd.assign((size_t)v.cd_len, 0);
    for (int p = 0; p < N; ++p)
        for (int S = 0; S <= A; ++S) {
            bool reach = S <= S2 * (p + 1) && (A - S) <= S2 * (N - 1 - p);
            if (!reach) continue;
            uint64_t c = 0;
            for (int a = 0; a <= S2 + 1; ++a) {
                b->cd[(size_t)p * v.cd_rowlen + S * v.cd_w + a] = c;
                if (a <= S2) c += D(p, S - a);
            }
            if (c > dim) return fail(HM_EOVERFLOW, "rank table entry above the dimension");
        }
    return HM_OK;
}

int upload_table(const void *host, size_t bytes, void **dev, const char *what) {
    const CaptureRelaxed relaxed;
    HM_CUDA(cudaMalloc(dev, bytes));
    // a copy on the null stream would join the capture of a blocking stream
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(cudaStreamLegacy, &cs);
    if (e == cudaErrorStreamCaptureImplicit) {
        cudaGetLastError();
        cudaStream_t st = nullptr;
        e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaMemcpyAsync(*dev, host, bytes, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (st) cudaStreamDestroy(st);
    } else if (e == cudaSuccess) {
        e = cudaMemcpy(*dev, host, bytes, cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) {
        cudaFree(*dev);
        *dev = nullptr;
        return cuda_fail(e, what);
    }
    return HM_OK;
}

int sm_count() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 1;
    }
    return n;
}

int grid_blocks(uint64_t rows, int threads) {
    uint64_t need = (rows + threads - 1) / threads;
    uint64_t cap = (uint64_t)sm_count() * 8;
    if (need < 1) need = 1;
    return (int)(need < cap ? need : cap);
}

int row_run_len() {
    const char *e = getenv("HM_ROW_RUN");
    const int v = e ? atoi(e) : 1;
    return v < 1 ? 1 : v > 64 ? 64 : v;
}

int make_bonds(const hm_basis *b, int n_bonds, const int32_t *u, const int32_t *v,
               const double *J, BondParams *out) {
    HM_TRY(bonds_check(b->view.N, n_bonds, u, v, J));
    const int S2 = b->view.S2;
    out->nb = n_bonds;
    out->S2 = S2;
    for (int t = 0; t < n_bonds; ++t) {
        int p = u[t], q = v[t];
        if (p > q) { int s = p; p = q; q = s; }   // s_u.s_v is symmetric in u, v
        out->p[t] = (unsigned char)p;
        out->q[t] = (unsigned char)q;
        out->jm[t] = -J[t];
        out->jmf[t] = (float)(-J[t]);
    }
    for (int ap = 0; ap <= S2; ++ap)
        for (int aq = 0; aq <= S2; ++aq) {
            long up_p = (long)ap * (S2 - ap + 1), dn_p = (long)(S2 - ap) * (ap + 1);
            long up_q = (long)aq * (S2 - aq + 1), dn_q = (long)(S2 - aq) * (aq + 1);
            out->hs_pdn[ap * 8 + aq] = 0.5 * std::sqrt((double)(up_p * dn_q));
            out->hs_pup[ap * 8 + aq] = 0.5 * std::sqrt((double)(dn_p * up_q));
        }
    if (b->mom_k >= 0) HM_TRY(mom_check_bonds(b, n_bonds, u, v, J));
    return HM_OK;
}

// the device tables of a basis: CD, then per entry (p, S, a) the rank changes {E+, F+, E-, F-}
// and {G+, G-} of the exchanges that the row sweep reads (hm_row.cuh), zero where there is none
template <class I>
static std::vector<I> row_tables(const hm_basis *b) {
    const SectorView &v = b->view;
    const size_t n = (size_t)v.cd_len, w = (size_t)v.cd_w;
    std::vector<I> t(7 * n, 0);
    for (size_t k = 0; k < n; ++k) t[k] = (I)b->cd[k];
    for (int p = 1; p < v.N; ++p)                    // position 0 has no rank term
        for (int S = std::max(0, v.A - v.S2 * (v.N - 1 - p)); S <= std::min(v.A, v.S2 * (p + 1)); ++S) {
            const size_t k0 = (size_t)p * v.cd_rowlen + (size_t)S * w;
            const I *c = t.data() + k0, *up = S < v.A ? c + w : nullptr, *dn = S >= 1 ? c - w : nullptr;
            I *e = t.data() + n + 4 * k0, *g = t.data() + 5 * n + 2 * k0;
            const int most = std::min(S, v.S2);
            for (int a = 0; a <= most; ++a) {
                if (up) {
                    if (a < v.S2) e[4 * a] = up[a + 1] - c[a];
                    g[2 * a] = up[a] - c[a];
                }
                if (a >= 1) e[4 * a + 1] = c[a - 1] - c[a];
                if (dn) {
                    if (a >= 1) e[4 * a + 2] = dn[a - 1] - c[a];
                    g[2 * a + 1] = dn[a] - c[a];
                }
                if (a < v.S2) e[4 * a + 3] = c[a + 1] - c[a];
            }
        }
    return t;
}

int row_plan(const SectorView &sv, const BondParams &bp, int es, RowPlan *P, size_t *smem) {
    if (row_run_len() > 1 || bp.nb > ROW_MB || bp.nb == 0) return 1;
    const int N = sv.N, S2 = sv.S2;
    P->nc = P->nslots = 0;
    memcpy(P->hs_pdn, bp.hs_pdn, sizeof P->hs_pdn);
    memcpy(P->hs_pup, bp.hs_pup, sizeof P->hs_pup);
    // classes of equal coupling, found by a small hash (bonds of one class mostly follow each other), bonds by
    // lower end.  This runs in every call: 0.4 .. 2 us
    uint16_t bc[ROW_MB];
    unsigned char of[256];                                     // class of a hash value, 255: none
    memset(of, 255, sizeof of);
    int last[HM_MAX_SITES], slot_of[HM_MAX_SITES], freed[HM_MAX_SITES], nf = 0;    // last[q]: lowest partner below q
    int next[HM_MAX_SITES], head[HM_MAX_SITES + 1];            // sites by their lowest partner
    for (int r = 0; r < N; ++r) last[r] = N;
    double most = 0.0;
    int count[HM_MAX_SITES] = {};
    for (int t = 0; t < bp.nb; ++t) {
        int c = t > 0 ? bc[t - 1] : 0;
        if (t == 0 || bp.jm[t] != bp.jm[t - 1]) {
            uint64_t bits;
            memcpy(&bits, &bp.jm[t], sizeof bits);
            unsigned h = (unsigned)((bits * 0x9E3779B97F4A7C15ull) >> 56);
            while (of[h] != 255 && P->jm[of[h]] != bp.jm[t]) h = (h + 1) & 255u;
            if (of[h] == 255) {
                of[h] = (unsigned char)P->nc;
                P->jm[P->nc++] = bp.jm[t];
            }
            c = of[h];
        }
        bc[t] = (uint16_t)c;
        most += std::fabs(bp.jm[t] / 4.0);
        last[bp.q[t]] = std::min(last[bp.q[t]], (int)bp.p[t]);
        ++count[bp.p[t]];
    }
    // slots: a site holds one from its own position down to its lowest partner's
    for (int r = 0; r <= N; ++r) head[r] = -1;
    for (int r = N - 1; r >= 0; --r) {                         // from the highest, so that a list runs upward
        next[r] = head[last[r]];
        head[last[r]] = r;
    }
    for (int r = N - 1; r >= 0; --r) {
        slot_of[r] = ROW_SLOT_NONE;
        if (last[r] < r) {
            if (nf == 0) freed[nf++] = P->nslots++;
            slot_of[r] = freed[--nf];
        }
        for (int q = head[r]; q >= 0; q = next[q]) freed[nf++] = slot_of[q];
    }
    int at[HM_MAX_SITES], n = 0;
    for (int r = 0; r < N; ++r) {
        at[r] = n;
        P->pos[r] = (uint32_t)n | ((uint32_t)count[r] << 10) | ((uint32_t)slot_of[r] << 20);
        n += count[r];
    }
    for (int t = 0; t < bp.nb; ++t)
        P->bond[at[bp.p[t]]++] = (uint32_t)(bp.q[t] * sv.bits) | ((uint32_t)slot_of[bp.q[t]] << 8) | ((uint32_t)bc[t] << 16);
    // diagonal sum_b dC_b k_b with |k_b| <= S2^2 in two parts, dC 2^-s below 2^62 and the remainder dL 2^-(s+t)
    // below 2^30; taken when they hold every coupling as exactly as a binary64 (binary32) term does: a digit can
    // make the term of a large coupling zero (integer spins), and terms of large couplings can cancel
    int ex = 0, kb = 0;
    std::frexp(most * S2 * S2, &ex);                 // sum of |J_b| / 4 S2^2 < 2^ex
    while ((1 << kb) < S2 * S2 * bp.nb) ++kb;
    const int s = 62 - ex, t = 30 - kb;
    if (kb > 10 || s <= -900 || s >= 900) return 1;
    P->dscale = std::ldexp(1.0, -s);
    P->dscale_low = std::ldexp(1.0, -s - t);
    P->dlow = 0;
    const double up = std::ldexp(1.0, s), up2 = std::ldexp(1.0, t), keep = std::ldexp(1.0, t - (es == 8 ? 53 : 29));
    for (int c = 0; c < P->nc; ++c) {
        const double v = P->jm[c] / 4.0 * up;
        P->dC[c] = (long long)v;
        const double rem = (v - (double)P->dC[c]) * up2;
        P->dL[c] = (int)rem;
        // one class at s > 1/2: ROW_ONE, without dC
        if ((std::fabs(rem - (double)P->dL[c]) > std::fabs(v) * keep || v * P->dscale != P->jm[c] / 4.0) && !(P->nc == 1 && S2 > 1))
            return 1;
        P->dlow |= P->dL[c] != 0;
    }
    P->dsum = 0;
    for (int b = 0; b < bp.nb; ++b) P->dsum += P->dC[bc[b]];
    const size_t tabs = sv.idx64 ? row_tab_bytes<uint64_t>(sv) : row_tab_bytes<uint32_t>(sv);
    *smem = row_coef_bytes(*P, S2, es) + tabs + (size_t)P->nslots * ROW_NT * (sv.idx64 ? 16 : 8);
    // at least two CTAs on an SM; more shared memory than that leaves the table form ahead
    return *smem <= 110 * 1024 ? 0 : 1;
}

// ---------------------------------------------------------------------------------------
// codec test hooks
// ---------------------------------------------------------------------------------------
template <class I>
__global__ void k_decode(SectorView sv, const int64_t *__restrict__ idx,
                         uint64_t *__restrict__ out, int64_t n) {
    extern __shared__ unsigned char smem_raw[];
    I *cd = reinterpret_cast<I *>(smem_raw);
    for (int k = threadIdx.x; k < sv.cd_len; k += blockDim.x) cd[k] = ((const I *)sv.cd)[k];
    __syncthreads();
    Codec<I> c{cd, sv.N, sv.S2, sv.A, sv.bits, sv.cd_w, sv.cd_rowlen};
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = idx[t];
        out[t] = (i < 0 || (uint64_t)i >= sv.dim) ? ~0ull : c.decode((I)i);
    }
}

template <class I>
__global__ void k_encode(SectorView sv, const uint64_t *__restrict__ st,
                         int64_t *__restrict__ out, int64_t n) {
    extern __shared__ unsigned char smem_raw[];
    I *cd = reinterpret_cast<I *>(smem_raw);
    for (int k = threadIdx.x; k < sv.cd_len; k += blockDim.x) cd[k] = ((const I *)sv.cd)[k];
    __syncthreads();
    Codec<I> c{cd, sv.N, sv.S2, sv.A, sv.bits, sv.cd_w, sv.cd_rowlen};
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        uint64_t w = st[t];
        // validity: digits <= 2s, no bits above the N positions, digit sum A
        bool ok = (sv.N * sv.bits >= 64) || (w >> (sv.N * sv.bits)) == 0;
        int S = 0;
        for (int p = 0; p < sv.N && ok; ++p) {
            int a = dig(w, p, sv.bits);
            if (a > sv.S2) ok = false;
            S += a;
        }
        ok = ok && S == sv.A;
        const int64_t ix = ok ? (int64_t)c.encode(w) : -1;
        out[t] = ix >= 0 && (uint64_t)ix < sv.dim ? ix : -1;   // spin-flip basis: representatives only
    }
}

template <class I>
static size_t cd_bytes(const SectorView &sv) { return (size_t)sv.cd_len * sizeof(I); }

}  // namespace hm

using namespace hm;

extern "C" {

const char *hm_last_error(void) { return g_err.c_str(); }

int basis_dim_query(int n_sites, int two_s, int two_m, int64_t *dim) {
    if (!dim) return fail(HM_EINVAL, "dim is NULL");
    hm_basis tmp;
    HM_TRY(build_tables(n_sites, two_s, two_m, &tmp));
    *dim = (int64_t)tmp.view.dim;
    return HM_OK;
}

int bonds_check(int n_sites, int n_bonds, const int32_t *u, const int32_t *v, const double *J) {
    if (n_bonds < 0 || n_bonds > HM_MAX_BONDS)
        return fail(HM_EINVAL, "n_bonds must be in 0..%d (got %d)", HM_MAX_BONDS, n_bonds);
    if (n_bonds > 0 && (!u || !v || !J)) return fail(HM_EINVAL, "bond arrays are NULL");
    for (int t = 0; t < n_bonds; ++t) {
        if (u[t] < 0 || u[t] >= n_sites || v[t] < 0 || v[t] >= n_sites)
            return fail(HM_EINVAL, "bond %d (%d,%d) outside 0..%d", t, u[t], v[t], n_sites - 1);
        if (u[t] == v[t]) return fail(HM_EINVAL, "bond %d joins site %d to itself", t, u[t]);
        if (!std::isfinite(J[t])) return fail(HM_EINVAL, "bond %d has a non-finite coupling", t);
    }
    return HM_OK;
}

int basis_build(int n_sites, int two_s, int two_m, hm_basis **out) {
    if (!out) return fail(HM_EINVAL, "out is NULL");
    *out = nullptr;
    hm_basis *b = new (std::nothrow) hm_basis();
    if (!b) return fail(HM_ENOMEM, "host allocation failed");
    int rc = build_tables(n_sites, two_s, two_m, b);
    if (rc < 0) { delete b; return rc; }
    SectorView &v = b->view;
    const std::vector<uint64_t> t64 = v.idx64 ? row_tables<uint64_t>(b) : std::vector<uint64_t>();
    const std::vector<uint32_t> t32 = v.idx64 ? std::vector<uint32_t>() : row_tables<uint32_t>(b);
    const size_t bytes = t64.size() * 8 + t32.size() * 4;
    const void *src = v.idx64 ? (const void *)t64.data() : (const void *)t32.data();
    cudaError_t e = cudaGetDevice(&b->device);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_cd, bytes > 0 ? bytes : 8);
    b->eslots = std::make_shared<ExpSlots>();
    if (e == cudaSuccess) e = cudaMalloc(&b->eslots->dev, (size_t)HM_ESLOTS * HM_EPART * sizeof(int));
    if (e == cudaSuccess) e = cudaMemcpy(b->d_cd, src, bytes, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        if (b->d_cd) cudaFree(b->d_cd);
        if (b->eslots->dev) cudaFree(b->eslots->dev);
        delete b;
        return cuda_fail(e, "basis_build: device tables");
    }
    v.cd = b->d_cd;
    *out = b;
    return HM_OK;
}

int basis_build_flip(int n_sites, int parity, hm_basis **out) {
    if (!out) return fail(HM_EINVAL, "out is NULL");
    *out = nullptr;
    if (parity != 1 && parity != -1) return fail(HM_EINVAL, "parity must be +1 or -1 (got %d)", parity);
    if (n_sites < 10 || n_sites > 32 || (n_sites & 1))
        return fail(HM_EINVAL, "spin-flip basis needs an even n_sites in 10..32 (got %d)", n_sites);
    HM_TRY(basis_build(n_sites, 1, 0, out));
    (*out)->parity = parity;
    (*out)->view.dim /= 2;          // the representatives: the first half of the sector
    return HM_OK;
}

int basis_free(hm_basis *b) {
    if (!b) return HM_OK;
    cudaError_t e = cudaSuccess, e2;
    if (b->d_cd && (e2 = cudaFree(b->d_cd)) != cudaSuccess) e = e2;
    if (b->eslots) {
        std::lock_guard<std::mutex> lk(b->eslots->mu);
        if (b->eslots->dev && (e2 = cudaFree(b->eslots->dev)) != cudaSuccess) e = e2;
        for (int *p : b->eslots->captured)
            if ((e2 = cudaFree(p)) != cudaSuccess) e = e2;
    }
    for (auto &kv : b->blk_tabs)
        if (kv.second.dev && (e2 = cudaFree(kv.second.dev)) != cudaSuccess) e = e2;
    for (auto &kv : b->s1_tabs)
        if (kv.second.dev && (e2 = cudaFree(kv.second.dev)) != cudaSuccess) e = e2;
    for (auto &kv : b->blk_ttabs)
        if (kv.second && (e2 = cudaFree(kv.second)) != cudaSuccess) e = e2;
    if (b->d_mom && (e2 = cudaFree(b->d_mom)) != cudaSuccess) e = e2;
    delete b;
    if (e != cudaSuccess) return cuda_fail(e, "basis_free");
    return HM_OK;
}

int basis_dim(const hm_basis *b, int64_t *dim) {
    if (!b || !dim) return fail(HM_EINVAL, "NULL argument");
    *dim = (int64_t)b->view.dim;
    return HM_OK;
}

int basis_decode(const hm_basis *b, const int64_t *idx, uint64_t *states, int64_t n, void *stream) {
    if (!b || n < 0 || (n > 0 && (!idx || !states))) return fail(HM_EINVAL, "bad argument");
    if (b->mom_k >= 0) return fail(HM_EINVAL, "basis_decode: not available on a momentum basis");
    if (n == 0) return HM_OK;
    const SectorView &sv = b->view;
    int blocks = grid_blocks((uint64_t)n, 256);
    if (sv.idx64) {
        size_t sm = cd_bytes<uint64_t>(sv);
        HM_CUDA(raise_smem_limit(k_decode<uint64_t>, (int)sm));
        k_decode<uint64_t><<<blocks, 256, sm, as_stream(stream)>>>(sv, idx, states, n);
    } else {
        size_t sm = cd_bytes<uint32_t>(sv);
        HM_CUDA(raise_smem_limit(k_decode<uint32_t>, (int)sm));
        k_decode<uint32_t><<<blocks, 256, sm, as_stream(stream)>>>(sv, idx, states, n);
    }
    HM_CUDA(cudaGetLastError());
    return HM_OK;
}

int basis_encode(const hm_basis *b, const uint64_t *states, int64_t *idx, int64_t n, void *stream) {
    if (!b || n < 0 || (n > 0 && (!idx || !states))) return fail(HM_EINVAL, "bad argument");
    if (b->mom_k >= 0) return fail(HM_EINVAL, "basis_encode: not available on a momentum basis");
    if (n == 0) return HM_OK;
    const SectorView &sv = b->view;
    int blocks = grid_blocks((uint64_t)n, 256);
    if (sv.idx64) {
        size_t sm = cd_bytes<uint64_t>(sv);
        HM_CUDA(raise_smem_limit(k_encode<uint64_t>, (int)sm));
        k_encode<uint64_t><<<blocks, 256, sm, as_stream(stream)>>>(sv, states, idx, n);
    } else {
        size_t sm = cd_bytes<uint32_t>(sv);
        HM_CUDA(raise_smem_limit(k_encode<uint32_t>, (int)sm));
        k_encode<uint32_t><<<blocks, 256, sm, as_stream(stream)>>>(sv, states, idx, n);
    }
    HM_CUDA(cudaGetLastError());
    return HM_OK;
}

}  // extern "C"
