// Shared by the block-algebra translation units: the column partition as the
// kernels see it, runs of whole systems (tiles), element access in the
// RHS-interleaved pair layout and packed complex arithmetic on column pairs.
#pragma once

#include <algorithm>

#include "bk_common.cuh"
#include "bk_kernels.h"

// system owning column pair q (columns 2q, 2q + 1)
__device__ __forceinline__ int sys_of_pair(const SysPart& p, int q) {
    int lo = 0, hi = p.nsys - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (2 * q >= p.col0[mid]) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Runs of whole active systems, at most maxp pairs each (one system may be
// larger): the unit a block or warp takes, so that every column it combines
// is its own.
struct PTiles {
    int n;
    int p0[BK_MAX_SYS];
    int np[BK_MAX_SYS];
};

inline PTiles make_ptiles(const SysPart& p, int maxp) {
    PTiles t;
    t.n = 0;
    bool open = false;
    for (int s = 0; s < p.nsys; ++s) {
        const int q0 = p.col0[s] / 2, nq = (p.col0[s + 1] - p.col0[s]) / 2;
        if (!((p.active >> s) & 1ull) || nq == 0) {
            open = false;
            continue;
        }
        if (open && t.np[t.n - 1] + nq <= maxp) {
            t.np[t.n - 1] += nq;
        } else {
            t.p0[t.n] = q0;
            t.np[t.n] = nq;
            t.n++;
            open = true;
        }
    }
    return t;
}
// Neighbouring tiles joined over the inactive systems between them (the
// kernel skips their lanes), where the wider tile takes no more warp steps per
// row (1 / floor(32 / pairs)) than the two.
inline PTiles join_ptiles(const PTiles& a, int maxp) {
    auto steps = [](int pairs) { return 1.0 / std::max(1, 32 / pairs); };
    PTiles t;
    t.n = 0;
    for (int i = 0; i < a.n; ++i) {
        const int l = t.n - 1, wide = t.n ? a.p0[i] + a.np[i] - t.p0[l] : 0;
        if (t.n && wide <= maxp && steps(wide) <= steps(t.np[l]) + steps(a.np[i]) + 1e-9) {
            t.np[l] = wide;
        } else {
            t.p0[t.n] = a.p0[i];
            t.np[t.n++] = a.np[i];
        }
    }
    return t;
}

inline int max_active_L(const SysPart& p) {
    int m = 0;
    for (int s = 0; s < p.nsys; ++s)
        if ((p.active >> s) & 1ull) m = std::max(m, p.L[s]);
    return m;
}

template <typename R2>
struct CxPair {  // one spinor component of a column pair, arithmetic type
    R2 re, im;
};

template <typename R2>
__device__ __forceinline__ CxPair<R2> cp_zero() {
    CxPair<R2> v;
    v.re = v.im = pzero<R2>();
    return v;
}

template <typename R2>
__device__ __forceinline__ CxPair<R2> shfl_pair(const CxPair<R2>& v, int src) {
    CxPair<R2> o;
    o.re.x = __shfl_sync(0xffffffffu, v.re.x, src);
    o.re.y = __shfl_sync(0xffffffffu, v.re.y, src);
    o.im.x = __shfl_sync(0xffffffffu, v.im.x, src);
    o.im.y = __shfl_sync(0xffffffffu, v.im.y, src);
    return o;
}

__device__ __forceinline__ float2 bcast(float v) { return make_float2(v, v); }
__device__ __forceinline__ double2 bcast(double v) { return make_double2(v, v); }

// acc (pair) += c (complex scalar) * v (pair)
template <typename R, typename R2>
__device__ __forceinline__ void cpair_mac(CxPair<R2>& acc, cx<R> c, const CxPair<R2>& v) {
    const R2 cr = bcast(c.r), ci = bcast(c.i), nci = bcast(-c.i);
    acc.re = pfma(cr, v.re, acc.re);
    acc.re = pfma(nci, v.im, acc.re);
    acc.im = pfma(cr, v.im, acc.im);
    acc.im = pfma(ci, v.re, acc.im);
}

// Element e (row * np + pair) through the read-only data path, FP16 scale
// applied.  Only for operands that no thread of the kernel writes, or that
// the reading thread alone writes after its one read.
template <int P>
__device__ __forceinline__ CxPair<typename Prec<P>::pair> ldg_at(const Field& f, size_t e,
                                                                  typename Prec<P>::pair sc) {
    CxPair<typename Prec<P>::pair> v;
    if constexpr (P == BK_FP64) {
        const double2* q = (const double2*)f.data + 2 * e;
        v.re = __ldg(q);
        v.im = __ldg(q + 1);
    } else if constexpr (P == BK_FP32) {
        const float4 q = __ldg((const float4*)f.data + e);
        v.re = make_float2(q.x, q.y);
        v.im = make_float2(q.z, q.w);
    } else {
        const uint2 q = __ldg((const uint2*)f.data + e);
        v.re = pmul(__half22float2(*reinterpret_cast<const __half2*>(&q.x)), sc);
        v.im = pmul(__half22float2(*reinterpret_cast<const __half2*>(&q.y)), sc);
    }
    return v;
}

template <int P>
__device__ __forceinline__ CxPair<typename Prec<P>::pair> load_at(const Field& f, size_t e) {
    CxPair<typename Prec<P>::pair> v;
    if constexpr (P == BK_FP64) {
        const double2* q = (const double2*)f.data + 2 * e;
        v.re = q[0];
        v.im = q[1];
    } else {
        static_assert(P == BK_FP32, "accumulators are FP32 or FP64");
        const float4 q = ((const float4*)f.data)[e];
        v.re = make_float2(q.x, q.y);
        v.im = make_float2(q.z, q.w);
    }
    return v;
}

template <int P>
__device__ __forceinline__ void store_at(const Field& f, size_t e, typename Prec<P>::pair re,
                                         typename Prec<P>::pair im) {
    if constexpr (P == BK_FP64) {
        double2* q = (double2*)f.data + 2 * e;
        q[0] = re;
        q[1] = im;
    } else {
        static_assert(P == BK_FP32, "element stores are for FP32 / FP64 blocks");
        ((float4*)f.data)[e] = make_float4(re.x, re.y, im.x, im.y);
    }
}

__device__ __forceinline__ float flip_sign(float v) { return __int_as_float(__float_as_int(v) ^ 0x80000000); }
__device__ __forceinline__ double flip_sign(double v) {
    return __hiloint2double(__double2hiint(v) ^ 0x80000000, __double2loint(v));
}
// (a call: general factors are rare, and FP64 arithmetic on either side of a
// select would be paid for by every FP32 kernel)
static __device__ __noinline__ void scale2(double& re, double& im, double mult) {
    re *= mult;
    im *= mult;
}

// complex coefficient mult * (ptr ? ptr[s] : 1); unit: 1 or -1 when mult is that
template <int P>
__device__ __forceinline__ cx<typename Prec<P>::real> coef(const double* ptr, double mult, int unit, int s) {
    using R = typename Prec<P>::real;
    if (!ptr) return mk(d2r<R>(mult), R(0));
    double re = __ldg(ptr + 2 * s), im = __ldg(ptr + 2 * s + 1);
    if (unit == 0) scale2(re, im, mult);
    R r = d2r<R>(re), i = d2r<R>(im);
    return unit < 0 ? mk(flip_sign(r), flip_sign(i)) : mk(r, i);
}

// FP32 products are summed in FP32 over at most this many (site, component)
// rows, the lanes added in FP32 included, then in FP64
constexpr int ROW_FLUSH = 96;

// rows.cu: systems of at most ROWS_MAXL columns
constexpr int ROWS_MAXL = 12;
// Row chunks (grid.y, partial-sum rows) of the row Gram kernel.  FP64: a chunk
// per 4 warp steps, so that a small lattice still fills every SM's FP64 pipe
// (4^4, 12 columns: 615 steps).  FP32 / FP16: a chunk per 64 steps, 8 a warp,
// since there a block's fixed costs (FP64 conversions, the finishing sums)
// outweigh a few more rows.  Up to two tiles (FP64) or four: at most the blocks
// that are resident at once (FP64: 1 an SM, else 2), since a 153rd block would
// double the time; more tiles take several waves anyway, of 76 chunks each.
inline int gram_row_chunks(int prec, int V, const PTiles& t) {
    int spw = 32;
    for (int i = 0; i < t.n; ++i) spw = std::min(spw, 32 / std::max(1, t.np[i]));
    const int steps = (12 * V) / std::max(1, spw);
    const int most = std::max(76, (prec == BK_FP64 ? 152 : 304) / std::max(1, t.n));
    return std::max(1, std::min(steps / (prec == BK_FP64 ? 4 : 64), most));
}
inline int gram_row_chunks_max(int V) { return std::max(1, std::min(12 * V / 4, 304)); }
bk_status rows_gram(int prec, Field A, Field B, Field B2, int NB, const SysPart& p, double2* partial, int nchunk,
                    int V, cudaStream_t st);
PTiles row_tiles(int prec, const SysPart& p);
bk_status rows_update(int prec, const GenOp& g, int V, int nchunk, int np, cudaStream_t st);
// GenOp's unit flags and whether it uses M
inline GenOp with_units(GenOp g) {
    auto unit = [](double x) { return x == 1.0 ? 1 : (x == -1.0 ? -1 : 0); };
    for (int e = 0; e < GENOP_MAXE; ++e) g.ea_unit[e] = unit(g.ea_mult[e]);
    for (int u = 0; u < GENOP_MAXMI; ++u) g.ma_unit[u] = unit(g.ma_mult[u]);
    g.xa_unit = unit(g.xa_mult);
    g.y_unit = unit(g.ym);
    g.x_unit = unit(g.xm);
    g.mat = g.nmi > 0 && g.M != nullptr && ((g.hasY && g.ym != 0.0) || (g.hasX && g.xm != 0.0));
    return g;
}
// wide.cu: systems of any size
int wide_gram_chunks(const SysPart& p, int V);
bk_status wide_gram(int prec, Field A, Field B, const SysPart& p, double2* partial, int nchunk, int V,
                    cudaStream_t st);
bk_status wide_update(int prec, const GenOp& g, int V, int nchunk, cudaStream_t st);
