// blk_multi.cu -- y = H x for several vectors at once ([dim][nvec], s = 1/2, class plans).
//
// A row is shared by a power of two of lanes, each with 16 bytes of its vectors where the alignment allows
// (wider blocks go 32 columns at a time), so an exchange target, read once for the row from
// its lists (blk_hops.cuh), serves a coalesced gather of all its vectors.  A block of blk.cuh is
// cut into parts, one CTA each, so that every SM has several.
//
// What bounds the FP64 product is arithmetic: a warp's binary64 instruction occupies its quarter of
// an SM for 64 cycles, and a multiply-add for each of the 40 bonds of a J1-J2 ring kept that pipe 72%
// busy (k_row_matvec).  Here the exchange sums are integers: every gathered value is aligned to the
// largest term of its row and column so far, in powers of two of |J_c| |x_j| (the sums move along when a
// larger one comes), with four bits below the last place.  So a value is cut at 2^-55 of the row's largest
// term -J_c/2 x_j, however far apart the couplings lie, where a binary64 sum rounds at every addition.
// A class's low, cross and high sums meet in one integer, and a class takes a conversion, a scaling
// and a multiply-add; the diagonal term is a binary64 product.  Rows with infinities or NaN, and those whose
// largest term is near the ends of binary64's range, are added in binary64; couplings more than 2^MULTI_SPREAD
// apart, or zero, take the general rows.  Adding the high exchanges in binary64 beside the integers was
// slower (100 against 95 us, before the last tuning).
// Measured on GB300, J1-J2 ring, N = 20, against k_matvec (general rows): eight vectors FP64 255 -> 81 us (unit
// vectors, whose rows are nearly all zeros, 255 -> 112), FP32 78 -> 25; 16 vectors FP64 361 -> 142; 33
// vectors (rows of no 16 bytes' alignment) 723 -> 330.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>

#include "blk_hops.cuh"
#include "ef64.cuh"

namespace hm {

namespace {

constexpr int MV_NT = 256;
constexpr int MULTI_SPREAD = 60;   // FP64: binary orders between the largest and the smallest |J_c|

__device__ __forceinline__ int hi32(double v) { return __double2hiint(v); }
__device__ __forceinline__ int lo32(double v) { return __double2loint(v); }

struct MultiArgs {
    const uint16_t *hops;
    double gd[HM_BLK_MAXC];        // -J_c / 4
    int oc[HM_BLK_MAXC];           // binary orders of |J_c| below the largest
    int ld, c0, w, parts;          // columns c0 .. c0 + w - 1 of ld; CTAs a block
    int lsh;                       // 2^lsh lanes a row
};

// V columns of one row (aligned to their size)
template <class T, int V>
__device__ __forceinline__ void multi_ld(const T *p, T *v) {
    if constexpr (V == 1) {
        v[0] = __ldg(p);
    } else if constexpr (sizeof(T) == 8) {
        const double2 t = __ldg((const double2 *)p);
        v[0] = t.x; v[1] = t.y;
    } else if constexpr (V == 2) {
        const float2 t = __ldg((const float2 *)p);
        v[0] = t.x; v[1] = t.y;
    } else {
        const float4 t = __ldg((const float4 *)p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    }
}
template <class T, int V>
__device__ __forceinline__ void multi_st(T *p, const T *v) {
    if constexpr (V == 1) *p = v[0];
    else if constexpr (sizeof(T) == 8) *(double2 *)p = make_double2(v[0], v[1]);
    else if constexpr (V == 2) *(float2 *)p = make_float2(v[0], v[1]);
    else *(float4 *)p = make_float4(v[0], v[1], v[2], v[3]);
}

// f(row offset) for every target of class cl of row r; returns their number
template <class F>
__device__ __forceinline__ int multi_targets(const BlkParams &P, const HopTab &Hp, const Hops &sh, const uint16_t *T,
                                             uint4 hd, uint32_t l, uint32_t r, int cl, F &&f) {
    int cnt = (int)((hd.x >> (8 * cl)) & 0xFFu);
    for (int e = 0; e < cnt; ++e) f((int)__ldg(T + Hp.seg[cl] + e));
    for (int e = P.cb_start[cl]; e < P.cb_start[cl + 1]; ++e) {
        int t2;
        if (!hop_cross(Hp, sh.x[e], hd, T, l, &t2)) continue;
        f(t2);
        ++cnt;
    }
    for (int e = sh.hcs[cl]; e < sh.hcs[cl + 1]; ++e) f((int)r + sh.hcd[e]);
    return cnt + sh.hcs[cl + 1] - sh.hcs[cl];
}

// whether all targets of a row hold zeros in the lane's columns (blocks of unit vectors are made of such rows)
template <int NC, int V>
__device__ __noinline__ bool multi_row_zeros(const BlkParams &P, const HopTab &Hp, const MultiArgs &a, const Hops &sh,
                                             const double *Xb, const uint16_t *T, uint4 hd, uint32_t l, uint32_t r) {
    unsigned bits = 0u;
    for (int cl = 0; cl < NC; ++cl)
        multi_targets(P, Hp, sh, T, hd, l, r, cl, [&](int t) {
            double v[V];
            multi_ld<double, V>(Xb + (ptrdiff_t)t * a.ld, v);
#pragma unroll
            for (int q = 0; q < V; ++q) bits |= (unsigned)hi32(v[q]) << 1 | (unsigned)lo32(v[q]);
        });
    return bits == 0u;
}

// one row and column in binary64, for the rows the integers do not serve; a term at a time, so that large values
// under small couplings do not overflow
template <int NC>
__device__ __noinline__ double multi_row_f64(const BlkParams &P, const HopTab &Hp, const MultiArgs &a, const Hops &sh,
                                             const double *Xb, const uint16_t *T, uint4 hd, uint32_t l, uint32_t r) {
    double y = 0.0, dg = 0.0;
    for (int cl = 0; cl < NC; ++cl) {
        const double g2 = 2.0 * a.gd[cl];
        const int cnt = multi_targets(P, Hp, sh, T, hd, l, r, cl,
                                      [&](int t) { y = fma(g2, __ldg(Xb + (ptrdiff_t)t * a.ld), y); });
        dg += a.gd[cl] * (double)(P.ntot[cl] - 2 * cnt);
    }
    return fma(dg, __ldg(Xb + (ptrdiff_t)r * a.ld), y);
}

// running sums of one row and column: FP32 plainly, FP64 as integers, class c in units of 2^(E + oc - 1079)
template <class T, int NC> struct MultiAcc;
template <int NC> struct MultiAcc<float, NC> {
    float s[NC];
    __device__ __forceinline__ void start() {
#pragma unroll
        for (int c = 0; c < NC; ++c) s[c] = 0.0f;
    }
    __device__ __forceinline__ void to_class(int) {}
    __device__ __forceinline__ void add(int c, float v, bool on) { s[c] += on ? v : 0.0f; }
};
template <int NC> struct MultiAcc<double, NC> {
    // E serves from E_LO + 1 to E_HI: above, all shifts and scales are those of normal numbers, and a value
    // that is not finite has an exponent field above E_HI + oc
    static constexpr int E_LO = 64, E_HI = 2030 - MULTI_SPREAD;
    long long s[NC];
    int E;                         // of the largest term so far; plus oc while a class is added
    __device__ __forceinline__ void start() {
        E = E_LO;
#pragma unroll
        for (int c = 0; c < NC; ++c) s[c] = 0;
    }
    __device__ __forceinline__ void to_class(int d) { E += d; }
    __device__ __forceinline__ static long long fixed(int hi, int lo, int E) {
        const int e = (hi >> 20) & 0x7FF;
        const unsigned long long M = ((unsigned long long)(unsigned)((hi & 0xFFFFF) | 0x100000) << 32 | (unsigned)lo) << 4;
        unsigned long long q;
        asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(M), "r"(E - e));       // zero from 64 on
        const long long m = (long long)q, sg = hi >> 31;
        return (m ^ sg) - sg;
    }
    // a value that is not on counts as zero (exponent field 0: shifted out, as E is at least E_LO)
    __device__ __forceinline__ void add(int c, double v, bool on) {
        const int hi = on ? hi32(v) : 0, lo = lo32(v), e = (hi >> 20) & 0x7FF;
        if (e > E) {
            const int d = min(e - E, 63);
#pragma unroll
            for (int k = 0; k < NC; ++k) s[k] >>= d;
            E = e;
        }
        s[c] += fixed(hi, lo, E);
    }
    __device__ __forceinline__ bool low() const { return E == E_LO; }
    // the integers hold the sums: a largest term in range, or only zeros
    __device__ __forceinline__ bool serves(bool zeros) const { return low() ? zeros : E <= E_HI; }
};

template <class T, int NC, int V>
__global__ void __launch_bounds__(MV_NT, 4) k_blk_multi(BlkParams P, HopTab Hp, MultiArgs a, const T *__restrict__ x,
                                                     T *__restrict__ y) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t h = blockIdx.x / a.parts;
    const int part = blockIdx.x % a.parts, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k = P.A - __popc(h);
    if (k < 0 || k > P.K) return;
    BlkTabs tb;
    tb.U = nullptr; tb.R0 = nullptr;
    tb.C = (const uint32_t *)((const unsigned char *)P.tab + P.off_C);
    const uint32_t off = blk_off(P, tb, h, k), n = tb.C[P.K * (P.A + 1) + k];
    const Hops sh = hops_carve(P, smem);
    if (warp == 0) hops_setup_high(P, tb, h, k, off, sh, lane);
    else if (warp == 1) hops_setup_cross(P, Hp, tb, h, k, off, sh, lane);
    __syncthreads();
    // row of the warp's and the lane's columns; idle lanes repeat the last column group
    const int rpw = 32 >> a.lsh, grp = lane >> a.lsh, li = (lane & ((1 << a.lsh) - 1)) * V;
    const bool on_col = li < a.w;
    const int col = on_col ? li : a.w - V;
    const T *Xb = x + (size_t)off * a.ld + a.c0 + col;
    const int ldb = a.ld * (int)sizeof(T);
    auto row = [&](int r2, T *v) { multi_ld<T, V>((const T *)((const char *)Xb + (int64_t)r2 * ldb), v); };
    const uint32_t ra = (uint32_t)((uint64_t)n * part / a.parts), rb = (uint32_t)((uint64_t)n * (part + 1) / a.parts);
    for (uint32_t r = ra + warp * rpw + grp; r < rb; r += MV_NT / 32 * rpw) {
        const uint32_t g = (uint32_t)P.lwoff[k] + r, l = __ldg(P.lw + g);
        const uint16_t *Tr = a.hops + (size_t)g * Hp.stride;
        const uint4 hd = __ldg((const uint4 *)Tr);
        MultiAcc<T, NC> acc[V];
#pragma unroll
        for (int q = 0; q < V; ++q) acc[q].start();
        int nd[NC];
#pragma unroll
        for (int cl = 0; cl < NC; ++cl) {
            const int oc = a.oc[cl];
#pragma unroll
            for (int q = 0; q < V; ++q) acc[q].to_class(oc);
            auto add = [&](const T *v, bool on) {
#pragma unroll
                for (int q = 0; q < V; ++q) acc[q].add(cl, v[q], on);
            };
            int mc = (int)((hd.x >> (8 * cl)) & 0xFFu);
            const uint16_t *t = Tr + Hp.seg[cl];
            for (int e = 0; e < mc; e += 4) {
                const uint2 w = __ldg((const uint2 *)(t + e));
                T x0[V], x1[V], x2[V], x3[V];
                row((int)(w.x & 0xFFFFu), x0);
                row((int)(w.x >> 16), x1);
                row((int)(w.y & 0xFFFFu), x2);
                row((int)(w.y >> 16), x3);
                add(x0, true);
                add(x1, e + 1 < mc);
                add(x2, e + 2 < mc);
                add(x3, e + 3 < mc);
            }
            for (int e = P.cb_start[cl]; e < P.cb_start[cl + 1]; ++e) {
                int t2;
                const bool on = hop_cross(Hp, sh.x[e], hd, Tr, l, &t2);
                T v[V];
                row(on ? t2 : (int)r, v);
                add(v, on);
                mc += (int)on;
            }
            const int e0 = sh.hcs[cl], e1 = sh.hcs[cl + 1];
            int e = e0;
            for (; e + 4 <= e1; e += 4) {
                T x0[V], x1[V], x2[V], x3[V];
                row((int)r + sh.hcd[e], x0);
                row((int)r + sh.hcd[e + 1], x1);
                row((int)r + sh.hcd[e + 2], x2);
                row((int)r + sh.hcd[e + 3], x3);
                add(x0, true);
                add(x1, true);
                add(x2, true);
                add(x3, true);
            }
            for (; e < e1; ++e) {
                T v[V];
                row((int)r + sh.hcd[e], v);
                add(v, true);
            }
            nd[cl] = P.ntot[cl] - 2 * (mc + e1 - e0);
#pragma unroll
            for (int q = 0; q < V; ++q) acc[q].to_class(-oc);
        }
        T yv[V], own[V], dg = T(0);
        bool zeros = false;
        row((int)r, own);
        if constexpr (sizeof(T) == 8) {
#pragma unroll
            for (int cl = 0; cl < NC; ++cl) dg = fma(a.gd[cl], (double)nd[cl], dg);
            bool low = false;
#pragma unroll
            for (int q = 0; q < V; ++q) low |= acc[q].low();
            if (low) zeros = multi_row_zeros<NC, V>(P, Hp, a, sh, Xb, Tr, hd, l, r);
        }
#pragma unroll
        for (int q = 0; q < V; ++q) {
            if constexpr (sizeof(T) == 4) {
                yv[q] = 0.0f;
#pragma unroll
                for (int cl = 0; cl < NC; ++cl) yv[q] += P.gq[cl] * (2.0f * acc[q].s[cl] + (float)nd[cl] * own[q]);
            } else if (!acc[q].serves(zeros)) {
                yv[q] = multi_row_f64<NC>(P, Hp, a, sh, Xb + q, Tr, hd, l, r);
            } else {
                yv[q] = 0.0;
#pragma unroll
                for (int cl = 0; cl < NC; ++cl) {                // at most 64 values below 2^57; 2 s in the scale
                    const double t = (double)acc[q].s[cl];
                    const int th = hi32(t);
                    yv[q] = fma(a.gd[cl], __hiloint2double(th ? th + ((acc[q].E + a.oc[cl] - 1078) << 20) : 0, lo32(t)), yv[q]);
                }
                yv[q] = fma(dg, own[q], yv[q]);
            }
        }
        if (on_col) multi_st<T, V>(y + ((size_t)off + r) * a.ld + a.c0 + li, yv);
    }
}

template <class T, int V>
const void *multi_kernel(int nc) {
    return nc == 1 ? (const void *)k_blk_multi<T, 1, V> : nc == 2 ? (const void *)k_blk_multi<T, 2, V>
                                                                  : (const void *)k_blk_multi<T, 4, V>;
}

__global__ void k_hop_table(BlkParams P, HopTab H, uint16_t *table) {
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < 1u << P.K) hop_fill(P, H, g, table);
}

}  // namespace

// The target table of a class plan from the basis's layouts, or nullptr at *table when it is not there
// and build is false (no allocation)
int blk_hop_table(hm_basis *b, const BlkParams &P, const HopTab &H, bool build, const uint16_t **table) {
    std::string key = "hops:" + std::to_string(P.K) + ":" + std::to_string(P.nc) + ":";
    for (int g = 0; g < P.nlg; ++g) key += std::to_string(P.lg_mask[g]) + "/" + std::to_string((int)P.lg_d[g]) + ",";
    for (int c = 0; c <= 3 * HM_BLK_MAXC; ++c) key += std::to_string(P.lg_cs[c]) + ";";
    for (int i = 0; i < H.nx; ++i) key += std::to_string((int)H.xp[i]) + ",";
    std::lock_guard<std::mutex> lk(b->tab_mu);
    auto it = b->blk_ttabs.find(key);
    if (it == b->blk_ttabs.end()) {
        *table = nullptr;
        if (!build) return HM_OK;
        void *dev = nullptr;
        HM_CUDA(cudaMalloc(&dev, ((size_t)H.stride * 2) << P.K));
        k_hop_table<<<((1u << P.K) + 127) / 128, 128, 0, cudaStreamPerThread>>>(P, H, (uint16_t *)dev);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamPerThread);   // complete for every stream from here on
        if (e != cudaSuccess) { cudaFree(dev); return cuda_fail(e, "target table"); }
        it = b->blk_ttabs.emplace(key, dev).first;
    }
    *table = (const uint16_t *)it->second;
    return HM_OK;
}

// blocks of the sector: high words that leave 0 .. K ones to the low part
static int blk_multi_blocks(int H, int K, int A) {
    int valid = 0;
    for (int c = std::max(0, A - K); c <= std::min(H, A); ++c) {
        uint64_t b = 1;
        for (int i = 0; i < c; ++i) b = b * (H - i) / (i + 1);
        valid += (int)b;
    }
    return valid;
}

// Whether blocks are the faster form for nvec vectors: a CTA sets a block up and takes 256 / (lanes a row) rows
// at a time, so sectors far from M = 0, whose blocks have few rows, leave it idle.  The line is at
// rows a block times (vectors + 4) = 480.  Measured (J1-J2 ring, FP64, us, blocks / general rows):
//   N = 32, 5 ones (12 rows a block): 2 vectors 1228 / 65, 8 vectors 1253 / 211, 32 vectors 1367 / 903
//   N = 30, 7 ones (49): 610 / 492, 1146 / 1698, 3275 / 7673    N = 28, 7 ones (72): 243 / 269, 592 / 934, 1922 / 4268
//   N = 24, 5 ones (42): 42 / 23, 51 / 59, 117 / 247            N = 26, 8 ones (220): 209 / 324, 683 / 1147, 2490 / 5429
bool blk_multi_serves(uint64_t dim, int H, int K, int A, int nvec) {
    return dim * (uint64_t)(std::min(nvec, 32) + 4) >= 480ull * (uint64_t)blk_multi_blocks(H, K, A);
}

// binary orders of each |J_c| below the largest (gd: the -J_c / 4 of nc classes); false when the integer sums
// do not serve them
bool blk_multi_orders(const double *gd, int nc, int *oc) {
    int most = INT_MIN;
    for (int c = 0; c < nc; ++c) {
        if (gd[c] == 0.0) return false;
        oc[c] = std::ilogb(gd[c]);
        most = std::max(most, oc[c]);
    }
    for (int c = 0; c < HM_BLK_MAXC; ++c) {
        oc[c] = c < nc ? most - oc[c] : 0;
        if (oc[c] > MULTI_SPREAD) return false;
    }
    return true;
}

// y = H x, columns 0 .. nvec - 1 of rows of nvec elements, 32 at a time
int blk_multi_launch(const BlkParams &P, const HopTab &H, const uint16_t *table, const double *gd, const int *oc,
                     const void *x, void *y, int dtype, int nvec, cudaStream_t st) {
    MultiArgs a{};
    a.hops = table;
    memcpy(a.gd, gd, sizeof a.gd);
    memcpy(a.oc, oc, sizeof a.oc);
    a.ld = nvec;
    const int valid = blk_multi_blocks(P.H, P.K, P.A);
    const size_t sm = hops_bytes(P);
    for (a.c0 = 0; a.c0 < nvec; a.c0 += a.w) {
        a.w = std::min(32, nvec - a.c0);
        // columns a lane: 16 bytes where rows, columns and pointers are aligned to them (the work on a target
        // is then done by fewer lanes), else 8, else one
        const size_t es = dtype == HM_F64 ? 8 : 4, align = ((uintptr_t)x | (uintptr_t)y | (size_t)nvec * es | (size_t)a.w * es) & 15;
        const int v = align == 0 ? (int)(16 / es) : align == 8 ? (int)(8 / es) : 1;
        a.lsh = 0;
        while ((v << a.lsh) < a.w) ++a.lsh;
        // 24 CTAs an SM (six: 8 to 15% slower, the last wave is nearly empty), but at least one pass of the CTA's
        // rows each
        const int rows = MV_NT >> a.lsh, most = std::max(1, (P.max_block + rows - 1) / rows);
        a.parts = std::min(most, std::max(1, (24 * sm_count() + valid - 1) / std::max(1, valid)));
        void *args[] = {(void *)&P, (void *)&H, (void *)&a, (void *)&x, (void *)&y};
        const void *kern = dtype == HM_F64 ? (v == 2 ? multi_kernel<double, 2>(P.nc) : multi_kernel<double, 1>(P.nc))
                         : v == 4          ? multi_kernel<float, 4>(P.nc)
                         : v == 2          ? multi_kernel<float, 2>(P.nc)
                                           : multi_kernel<float, 1>(P.nc);
        HM_CUDA(cudaLaunchKernel(kern, dim3((unsigned)a.parts << P.H), dim3(MV_NT), args, sm, st));
    }
    return HM_OK;
}

}  // namespace hm
