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
// largest exponent among those seen so far in its row and column (the sums move along when a larger
// one comes), with two bits below the last place, so a value is cut at 2^-54 of the largest one
// of its row where a binary64 sum rounds at every addition.  Both sums of a class and the diagonal
// meet in one integer, and a class takes a conversion, a scaling and a multiply-add.  Rows with
// infinities or NaN, and those whose largest value is below 2^-959 or above 2^1007, are added in
// binary64.  Adding the high exchanges in binary64 beside the integers was slower (100 against 95 us, before the last tuning).
// Measured on GB300, J1-J2 ring, whole calls: N = 20, eight vectors FP64 135 -> 80 us, FP32 71 -> 41;
// 16 vectors 315 -> 175 and 178 -> 56; 33 vectors (rows of no 16 bytes' alignment) 492 -> 344 and 243 -> 193.
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <string>

#include "blk_hops.cuh"
#include "ef64.cuh"

namespace hm {

namespace {

constexpr int MV_NT = 256;

__device__ __forceinline__ int hi32(double v) { return __double2hiint(v); }
__device__ __forceinline__ int lo32(double v) { return __double2loint(v); }

struct MultiArgs {
    const uint16_t *hops;
    double gd[HM_BLK_MAXC];        // -J_c / 4
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

// one row and column in binary64, for the rows the integers do not serve
template <int NC>
__device__ __noinline__ double multi_row_f64(const BlkParams &P, const HopTab &Hp, const MultiArgs &a, const Hops &sh,
                                             const double *Xb, const uint16_t *T, uint4 hd, uint32_t l, uint32_t r) {
    const double xo = __ldg(Xb + (ptrdiff_t)r * a.ld);
    double y = 0.0, dg = 0.0;
    for (int cl = 0; cl < NC; ++cl) {
        double s = 0.0;
        int cnt = (int)((hd.x >> (8 * cl)) & 0xFFu);
        for (int e = 0; e < cnt; ++e) s += __ldg(Xb + (ptrdiff_t)__ldg(T + Hp.seg[cl] + e) * a.ld);
        for (int e = P.cb_start[cl]; e < P.cb_start[cl + 1]; ++e) {
            int t2;
            if (!hop_cross(Hp, sh.x[e], hd, T, l, &t2)) continue;
            s += __ldg(Xb + (ptrdiff_t)t2 * a.ld);
            ++cnt;
        }
        for (int e = sh.hcs[cl]; e < sh.hcs[cl + 1]; ++e) s += __ldg(Xb + (ptrdiff_t)((int)r + sh.hcd[e]) * a.ld);
        cnt += sh.hcs[cl + 1] - sh.hcs[cl];
        dg += a.gd[cl] * (double)(P.ntot[cl] - 2 * cnt);
        y += 2.0 * a.gd[cl] * s;
    }
    return dg * xo + y;
}

// running sums of one row and column: FP32 plainly, FP64 as integers in units of 2^(E - 1077)
template <class T, int NC> struct MultiAcc;
template <int NC> struct MultiAcc<float, NC> {
    float s[NC], own;
    __device__ __forceinline__ void start(float xo) {
        own = xo;
#pragma unroll
        for (int c = 0; c < NC; ++c) s[c] = 0.0f;
    }
    __device__ __forceinline__ void add(int c, float v, bool on) { s[c] += on ? v : 0.0f; }
};
template <int NC> struct MultiAcc<double, NC> {
    long long s[NC];
    int E;
    double own;
    __device__ __forceinline__ void start(double xo) {
        own = xo;
        E = (hi32(xo) >> 20) & 0x7FF;
#pragma unroll
        for (int c = 0; c < NC; ++c) s[c] = 0;
    }
    __device__ __forceinline__ static long long fixed(int hi, int lo, int E) {
        const int e = (hi >> 20) & 0x7FF;
        const unsigned long long M = ((unsigned long long)(unsigned)((hi & 0xFFFFF) | 0x100000) << 32 | (unsigned)lo) << 2;
        unsigned long long q;
        asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(M), "r"(E - e));       // zero from 64 on
        const long long m = (long long)q, sg = hi >> 31;
        return (m ^ sg) - sg;
    }
    // a value that is not on counts as zero (exponent 0: shifted out whenever E serves)
    __device__ __forceinline__ void add(int c, double v, bool on) {
        const int hi = on ? hi32(v) : 0, e = (hi >> 20) & 0x7FF;
        if (e > E) {
            const int d = min(e - E, 63);
#pragma unroll
            for (int k = 0; k < NC; ++k) s[k] >>= d;
            E = e;
        }
        s[c] += fixed(hi, lo32(v), E);
    }
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
        {
            T v[V];
            row((int)r, v);
#pragma unroll
            for (int q = 0; q < V; ++q) acc[q].start(v[q]);
        }
        int nd[NC];
#pragma unroll
        for (int cl = 0; cl < NC; ++cl) {
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
        }
        T yv[V];
#pragma unroll
        for (int q = 0; q < V; ++q) {
            if constexpr (sizeof(T) == 4) {
                yv[q] = 0.0f;
#pragma unroll
                for (int cl = 0; cl < NC; ++cl) yv[q] += P.gq[cl] * (2.0f * acc[q].s[cl] + (float)nd[cl] * acc[q].own);
            } else if (acc[q].E < 64 || acc[q].E > 2030) {
                yv[q] = multi_row_f64<NC>(P, Hp, a, sh, Xb + q, Tr, hd, l, r);
            } else {
                // |2 s + nd xo| < 3 64 2^55
                const long long xo = MultiAcc<T, NC>::fixed(hi32(acc[q].own), lo32(acc[q].own), acc[q].E);
                const double sc = ef::u2d((uint64_t)(acc[q].E - 1077 + 1023) << 52);
                yv[q] = 0.0;
#pragma unroll
                for (int cl = 0; cl < NC; ++cl) yv[q] = fma(a.gd[cl], (double)(2 * acc[q].s[cl] + nd[cl] * xo) * sc, yv[q]);
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

// y = H x, columns 0 .. nvec - 1 of rows of nvec elements, 32 at a time
int blk_multi_launch(const BlkParams &P, const HopTab &H, const uint16_t *table, const double *gd, const void *x, void *y,
                     int dtype, int nvec, cudaStream_t st) {
    MultiArgs a{};
    a.hops = table;
    memcpy(a.gd, gd, sizeof a.gd);
    a.ld = nvec;
    int valid = 0;
    for (uint32_t h = 0; h < (1u << P.H); ++h) {
        const int k = P.A - __builtin_popcount(h);
        valid += k >= 0 && k <= P.K;
    }
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
