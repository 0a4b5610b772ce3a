// Multi-RHS O(a)-improved Wilson-Dirac operator, Eq. (wd-op) of arXiv:0903.4936,
// and the layout-conversion kernels around it.
//
//     y = x - kappa_c * ( sum_mu [(1 - gamma_mu) U_mu(n) x(n+mu)
//                                 + (1 + gamma_mu) U_mu(n-mu)^+ x(n-mu)] + C(n) x(n) )
//
// FP32 / FP16 storage (k_dslash_pair): one thread per site and column pair.
// Blocks are RHS-interleaved (all columns of a site in one row), so the
// lanes of a warp read one contiguous line per spinor component and share
// every gauge link and clover entry of their site.  All arithmetic is on pairs
// {column 2p, column 2p + 1} with the packed FP32x2 multiply-add of sm_100+;
// a link or clover entry is loaded as {re, im} (8 bytes for the whole warp)
// and its operands {u_r, u_r}, {u_i, u_i}, {-u_i, -u_i} are formed by moves,
// for which the issue slots are free.  The clover term is applied first (out =
// x - kappa C x needs x(n) only once); each of the eight hops then adds -kappa
// times its term directly.
//
// What bounds it (16^3x32, 30 columns, 281 us): the load pipe of L1, 79 % busy,
// with the 15 warps an SM that registers allow waiting for it 57 % of their
// time; L2 is 46 % busy (2.8 GB to the SMs, the rows about seven times), DRAM 37
// %, issue 34 %.  A row element takes four passes of that pipe per warp and load,
// a link or clover entry one per site in the warp.  Before, links and clover
// were stored as the duplicated pairs (224 and 816 bytes) and took 216 loads a
// thread: 404 us there (24^3x48, 96 columns 5080 us, now 4060; FP16 12x10x14x18,
// 13 columns 51, now 34).  A form with the rows staged by bulk copies
// (cp.async.bulk, a producer warp, 2x2x2 site tiles sharing their rows, 5
// fetches a site instead of 8) took 306 us.
//
// FP64 / double-float (k_dslash_col): one thread per site and column, FP64
// links and clover in [element][site] order (the FP64 pipe, not memory,
// bounds this kernel on GB300).
//
// Each (1 -+ gamma_mu) has rank two: the neighbour spinor is projected to two
// colour vectors, multiplied by the 3x3 link, and expanded again.  With the
// printed gamma matrices, for projector (1 + s gamma_mu) (s = -1 forward,
// +1 backward) and h = (h0, h1):
//   mu=x: h0 = q0 - i s q3, h1 = q1 - i s q2;  out = (h0, h1,  i s h1,  i s h0)
//   mu=y: h0 = q0 -   s q3, h1 = q1 +   s q2;  out = (h0, h1,    s h1,   -s h0)
//   mu=z: h0 = q0 - i s q2, h1 = q1 + i s q3;  out = (h0, h1,  i s h0, -i s h1)
//   mu=t: s=+1: out = (2 q0, 2 q1, 0, 0);  s=-1: out = (0, 0, 2 q2, 2 q3)
#include "bk_common.cuh"
#include "bk_kernels.h"

#include <algorithm>

namespace {

// ================================================================= FP32 / FP16: packed pairs

struct DPairArgs {
    Field x, y, b;
    const float* __restrict__ U;  // compact links, [site][mu] of BK_LINKC floats
    const float* __restrict__ C;  // compact clover, BK_CLOVC floats per site
    int L[4], st[4];
    int V, p0, npl, residual;
    float2 nk[BK_MAX_COLS / 2];  // {-kappa_2p, -kappa_2p+1} of launch pair p - p0
};

struct Hop {
    float2 r[6], i[6];  // projected half spinor: colour a of h0 at a, of h1 at 3 + a
};

// projection (1 + S gamma_mu) x -> h for one column pair and colour a
template <int MU, int S>
__device__ __forceinline__ void project_pair(const float2 (&qr)[12], const float2 (&qi)[12], Hop& h, int a) {
    {
        const int c0 = a, c1 = 3 + a, c2 = 6 + a, c3 = 9 + a;
        if constexpr (MU == 0) {
            if constexpr (S > 0) {  // h0 = q0 - i q3, h1 = q1 - i q2
                h.r[a] = padd(qr[c0], qi[c3]);
                h.i[a] = psub(qi[c0], qr[c3]);
                h.r[3 + a] = padd(qr[c1], qi[c2]);
                h.i[3 + a] = psub(qi[c1], qr[c2]);
            } else {  // h0 = q0 + i q3, h1 = q1 + i q2
                h.r[a] = psub(qr[c0], qi[c3]);
                h.i[a] = padd(qi[c0], qr[c3]);
                h.r[3 + a] = psub(qr[c1], qi[c2]);
                h.i[3 + a] = padd(qi[c1], qr[c2]);
            }
        } else if constexpr (MU == 1) {
            if constexpr (S > 0) {  // h0 = q0 - q3, h1 = q1 + q2
                h.r[a] = psub(qr[c0], qr[c3]);
                h.i[a] = psub(qi[c0], qi[c3]);
                h.r[3 + a] = padd(qr[c1], qr[c2]);
                h.i[3 + a] = padd(qi[c1], qi[c2]);
            } else {  // h0 = q0 + q3, h1 = q1 - q2
                h.r[a] = padd(qr[c0], qr[c3]);
                h.i[a] = padd(qi[c0], qi[c3]);
                h.r[3 + a] = psub(qr[c1], qr[c2]);
                h.i[3 + a] = psub(qi[c1], qi[c2]);
            }
        } else if constexpr (MU == 2) {
            if constexpr (S > 0) {  // h0 = q0 - i q2, h1 = q1 + i q3
                h.r[a] = padd(qr[c0], qi[c2]);
                h.i[a] = psub(qi[c0], qr[c2]);
                h.r[3 + a] = psub(qr[c1], qi[c3]);
                h.i[3 + a] = padd(qi[c1], qr[c3]);
            } else {  // h0 = q0 + i q2, h1 = q1 - i q3
                h.r[a] = psub(qr[c0], qi[c2]);
                h.i[a] = padd(qi[c0], qr[c2]);
                h.r[3 + a] = padd(qr[c1], qi[c3]);
                h.i[3 + a] = psub(qi[c1], qr[c3]);
            }
        } else {
            if constexpr (S > 0) {
                h.r[a] = qr[c0];
                h.i[a] = qi[c0];
                h.r[3 + a] = qr[c1];
                h.i[3 + a] = qi[c1];
            } else {
                h.r[a] = qr[c2];
                h.i[a] = qi[c2];
                h.r[3 + a] = qr[c3];
                h.i[3 + a] = qi[c3];
            }
        }
    }
}

// acc += -kappa * expand(w) for projector (1 + S gamma_mu), colour a of both
// half-spinor vectors (w0, w1); nk = {-kappa}, pk = {+kappa}
template <int MU, int S>
__device__ __forceinline__ void reconstruct_colour(int a, float2 w0r, float2 w0i, float2 w1r, float2 w1i, float2 nk,
                                                   float2 pk, float2 (&ar)[12], float2 (&ai)[12]) {
    const int c0 = a, c1 = 3 + a, c2 = 6 + a, c3 = 9 + a;
    if constexpr (MU == 3) {
        const float2 n2 = padd(nk, nk);
        if constexpr (S > 0) {
            ar[c0] = pfma(n2, w0r, ar[c0]);
            ai[c0] = pfma(n2, w0i, ai[c0]);
            ar[c1] = pfma(n2, w1r, ar[c1]);
            ai[c1] = pfma(n2, w1i, ai[c1]);
        } else {
            ar[c2] = pfma(n2, w0r, ar[c2]);
            ai[c2] = pfma(n2, w0i, ai[c2]);
            ar[c3] = pfma(n2, w1r, ar[c3]);
            ai[c3] = pfma(n2, w1i, ai[c3]);
        }
    } else {
        ar[c0] = pfma(nk, w0r, ar[c0]);
        ai[c0] = pfma(nk, w0i, ai[c0]);
        ar[c1] = pfma(nk, w1r, ar[c1]);
        ai[c1] = pfma(nk, w1i, ai[c1]);
        if constexpr (MU == 0) {
            // lower = (i S w1, i S w0); i w = (-w_i, w_r)
            if constexpr (S > 0) {
                ar[c2] = pfma(pk, w1i, ar[c2]);
                ai[c2] = pfma(nk, w1r, ai[c2]);
                ar[c3] = pfma(pk, w0i, ar[c3]);
                ai[c3] = pfma(nk, w0r, ai[c3]);
            } else {
                ar[c2] = pfma(nk, w1i, ar[c2]);
                ai[c2] = pfma(pk, w1r, ai[c2]);
                ar[c3] = pfma(nk, w0i, ar[c3]);
                ai[c3] = pfma(pk, w0r, ai[c3]);
            }
        } else if constexpr (MU == 1) {
            // lower = (S w1, -S w0)
            if constexpr (S > 0) {
                ar[c2] = pfma(nk, w1r, ar[c2]);
                ai[c2] = pfma(nk, w1i, ai[c2]);
                ar[c3] = pfma(pk, w0r, ar[c3]);
                ai[c3] = pfma(pk, w0i, ai[c3]);
            } else {
                ar[c2] = pfma(pk, w1r, ar[c2]);
                ai[c2] = pfma(pk, w1i, ai[c2]);
                ar[c3] = pfma(nk, w0r, ar[c3]);
                ai[c3] = pfma(nk, w0i, ai[c3]);
            }
        } else {
            // MU == 2: lower = (i S w0, -i S w1)
            if constexpr (S > 0) {
                ar[c2] = pfma(pk, w0i, ar[c2]);
                ai[c2] = pfma(nk, w0r, ai[c2]);
                ar[c3] = pfma(nk, w1i, ar[c3]);
                ai[c3] = pfma(pk, w1r, ai[c3]);
            } else {
                ar[c2] = pfma(nk, w0i, ar[c2]);
                ai[c2] = pfma(pk, w0r, ai[c2]);
                ar[c3] = pfma(pk, w1i, ar[c3]);
                ai[c3] = pfma(nk, w1r, ai[c3]);
            }
        }
    }
}

// Compact complex table entries (gauge.cu).  All lanes of a site read the same
// 8 bytes, and the pairs {u, u} of the packed arithmetic are formed by moves.
struct GTab {
    const float2* p;
    __device__ __forceinline__ float2 at(int e) const { return __ldg(p + e); }
};
__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }

// Product with the link U (forward) or U^+ (backward) and reconstruction, fused
// row by row: output colour i of both half-spinor vectors is formed and added
// at once, so only one row of the link and one colour of w are live.
template <int MU, int S>
__device__ __forceinline__ void link_mul_add(GTab u, const Hop& h, float2 nk, float2 pk, float2 (&ar)[12],
                                             float2 (&ai)[12]) {
    constexpr bool DAG = S > 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        float2 e[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) e[j] = u.at(DAG ? 3 * j + i : 3 * i + j);
        float2 wr[2], wi[2];
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) wr[hh] = wi[hh] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float2 ur = dup(e[j].x), ui = dup(e[j].y), un = dup(-e[j].y);
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const float2 hr = h.r[3 * hh + j], hi = h.i[3 * hh + j];
                wr[hh] = pfma(ur, hr, wr[hh]);
                wr[hh] = pfma(DAG ? ui : un, hi, wr[hh]);
                wi[hh] = pfma(ur, hi, wi[hh]);
                wi[hh] = pfma(DAG ? un : ui, hr, wi[hh]);
            }
        }
        reconstruct_colour<MU, S>(i, wr[0], wi[0], wr[1], wi[1], nk, pk, ar, ai);
    }
}

// y = H_b v for chiral block b (6 diagonal entries, then 15 complex ones below
// the diagonal) of a compact site term
__device__ __forceinline__ void herm6_pair(GTab c, int b, const float2 (&vr)[6], const float2 (&vi)[6], float2 (&yr)[6],
                                           float2 (&yi)[6]) {
#pragma unroll
    for (int i = 0; i < 6; i += 2) {
        const float2 d = c.at(18 * b + i / 2);
        yr[i] = pmul(dup(d.x), vr[i]);
        yi[i] = pmul(dup(d.x), vi[i]);
        yr[i + 1] = pmul(dup(d.y), vr[i + 1]);
        yi[i + 1] = pmul(dup(d.y), vi[i + 1]);
    }
    int q = 0;
#pragma unroll
    for (int i = 1; i < 6; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j, ++q) {
            const float2 A = c.at(18 * b + 3 + q);
            const float2 AR = dup(A.x), AI = dup(A.y), NAI = dup(-A.y);
            // y_i += A v_j, y_j += conj(A) v_i
            yr[i] = pfma(AR, vr[j], yr[i]);
            yr[i] = pfma(NAI, vi[j], yr[i]);
            yi[i] = pfma(AR, vi[j], yi[i]);
            yi[i] = pfma(AI, vr[j], yi[i]);
            yr[j] = pfma(AR, vr[i], yr[j]);
            yr[j] = pfma(AI, vi[i], yr[j]);
            yi[j] = pfma(AR, vi[i], yi[j]);
            yi[j] = pfma(NAI, vr[i], yi[j]);
        }
}

// The site term on (ar, ai) in place: CLOVER: out = q - kappa C q (nk =
// {-kappa}); else out = A^-1 q.  The blocks act on u + l and u - l.
template <bool CLOVER>
__device__ __forceinline__ void site_term(GTab c, float2 nk, float2 (&ar)[12], float2 (&ai)[12]) {
    float2 vr[2][6], vi[2][6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        vr[0][k] = padd(ar[k], ar[k + 6]);
        vi[0][k] = padd(ai[k], ai[k + 6]);
        vr[1][k] = psub(ar[k], ar[k + 6]);
        vi[1][k] = psub(ai[k], ai[k + 6]);
    }
    const float2 pk = make_float2(-nk.x, -nk.y);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        float2 yr[6], yi[6];
        herm6_pair(c, b, vr[b], vi[b], yr, yi);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            if (CLOVER) {  // upper half: -kappa y; lower: -kappa y (b = 0), +kappa y (b = 1)
                ar[k] = pfma(nk, yr[k], ar[k]);
                ai[k] = pfma(nk, yi[k], ai[k]);
                ar[k + 6] = pfma(b == 0 ? nk : pk, yr[k], ar[k + 6]);
                ai[k + 6] = pfma(b == 0 ? nk : pk, yi[k], ai[k + 6]);
            } else if (b == 0) {  // u = y0 + y1, l = y0 - y1
                ar[k] = ar[k + 6] = yr[k];
                ai[k] = ai[k + 6] = yi[k];
            } else {
                ar[k] = padd(ar[k], yr[k]);
                ai[k] = padd(ai[k], yi[k]);
                ar[k + 6] = psub(ar[k + 6], yr[k]);
                ai[k + 6] = psub(ai[k + 6], yi[k]);
            }
        }
    }
}

template <int P, int MU, int S>
__device__ __forceinline__ void hop_pair(const Field& x, int nb, int p, const float* __restrict__ link,
                                         float2 nk, float2 pk, float2 (&ar)[12], float2 (&ai)[12]) {
    Hop h;
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // the four spin components of colour c
        float2 qr[12], qi[12];
#pragma unroll
        for (int sp = 0; sp < 4; ++sp) {
            // the t projector reads only two of the four spins
            if (MU == 3 && ((S > 0) != (sp < 2))) continue;
            load_elem<P>(x, nb, 3 * sp + c, p, qr[3 * sp + c], qi[3 * sp + c]);
        }
        Hop hc;
        project_pair<MU, S>(qr, qi, hc, c);
        h.r[c] = hc.r[c];
        h.i[c] = hc.i[c];
        h.r[3 + c] = hc.r[3 + c];
        h.i[3 + c] = hc.i[3 + c];
    }
    if constexpr (P == BK_FP16) {  // the projection is linear: scale the 12 projected pairs
        const float2 sc = pair_scale<P>(x, nb, p);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            h.r[k] = pmul(h.r[k], sc);
            h.i[k] = pmul(h.i[k], sc);
        }
    }
    link_mul_add<MU, S>(GTab{reinterpret_cast<const float2*>(link)}, h, nk, pk, ar, ai);
}

template <int P, int MU>
__device__ __forceinline__ void hop_dir_pair(const DPairArgs& a, const int (&co)[4], int n, int p, float2 nk,
                                             float2 pk, float2 (&ar)[12], float2 (&ai)[12]) {
    const int Lm = a.L[MU], sm = a.st[MU];
    const int nf = co[MU] == Lm - 1 ? n - (Lm - 1) * sm : n + sm;
    const int nb = co[MU] == 0 ? n + (Lm - 1) * sm : n - sm;
    // forward: (1 - gamma_mu) U_mu(n) x(n + mu)
    hop_pair<P, MU, -1>(a.x, nf, p, a.U + ((size_t)n * 4 + MU) * BK_LINKC, nk, pk, ar, ai);
    // backward: (1 + gamma_mu) U_mu(n - mu)^+ x(n - mu)
    hop_pair<P, MU, +1>(a.x, nb, p, a.U + ((size_t)nb * 4 + MU) * BK_LINKC, nk, pk, ar, ai);
}

// Blocks of 128 threads, MINB of them an SM (3: 168 registers, 4: 128).
template <int P, int MINB>
__global__ void __launch_bounds__(128, MINB) k_dslash_pair(const __grid_constant__ DPairArgs a) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (long long)a.V * a.npl) return;
    const int s = (int)(g / a.npl), pl = (int)(g - (long long)s * a.npl), p = a.p0 + pl;
    int co[4];
    {
        int r = s;
        co[3] = r / a.st[3];
        r -= co[3] * a.st[3];
        co[2] = r / a.st[2];
        r -= co[2] * a.st[2];
        co[1] = r / a.st[1];
        co[0] = r - co[1] * a.st[1];
    }
    // (the site again from its coordinates: s itself would stay in a register
    // throughout, and with it the kernel spills at 128)
    const int n = co[0] + a.st[1] * co[1] + a.st[2] * co[2] + a.st[3] * co[3];
    const float2 nk = a.nk[pl];
    const float2 pk = make_float2(-nk.x, -nk.y);
    float2 ar[12], ai[12];
    load_pair<P>(a.x, n, p, ar, ai);  // out = x - kappa C x
    site_term<true>(GTab{reinterpret_cast<const float2*>(a.C + (size_t)n * BK_CLOVC)}, nk, ar, ai);
    hop_dir_pair<P, 0>(a, co, n, p, nk, pk, ar, ai);
    hop_dir_pair<P, 1>(a, co, n, p, nk, pk, ar, ai);
    hop_dir_pair<P, 2>(a, co, n, p, nk, pk, ar, ai);
    hop_dir_pair<P, 3>(a, co, n, p, nk, pk, ar, ai);
    if (a.residual) {  // b - D x
        float2 br[12], bi[12];
        load_pair<P>(a.b, n, p, br, bi);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            ar[k] = psub(br[k], ar[k]);
            ai[k] = psub(bi[k], ai[k]);
        }
    }
    store_pair<P>(a.y, n, p, ar, ai);
}

// ================================================================= FP64 / double-float: one column per thread

template <int P>
struct DColArgs {
    Field x, y, b;
    const typename Prec<P>::link* __restrict__ U;  // [mu][9][V] double2
    const typename Prec<P>::clov* __restrict__ C;  // [36][V] double2
    int L[4], st[4];
    int V, c0, ncl, residual;
    double kappa[BK_MAX_COLS];
};

template <int MU, int S, typename R>
__device__ __forceinline__ void project(const cx<R> (&q)[12], cx<R> (&h)[6]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const cx<R> q0 = q[a], q1 = q[3 + a], q2 = q[6 + a], q3 = q[9 + a];
        if constexpr (MU == 0) {
            h[a] = S > 0 ? q0 - ti(q3) : q0 + ti(q3);
            h[3 + a] = S > 0 ? q1 - ti(q2) : q1 + ti(q2);
        } else if constexpr (MU == 1) {
            h[a] = S > 0 ? q0 - q3 : q0 + q3;
            h[3 + a] = S > 0 ? q1 + q2 : q1 - q2;
        } else if constexpr (MU == 2) {
            h[a] = S > 0 ? q0 - ti(q2) : q0 + ti(q2);
            h[3 + a] = S > 0 ? q1 + ti(q3) : q1 - ti(q3);
        } else {
            h[a] = S > 0 ? q0 : q2;
            h[3 + a] = S > 0 ? q1 : q3;
        }
    }
}

// FIRST: acc is taken as zero (the first hop sets it, 24 additions saved)
template <int MU, int S, bool FIRST, typename R>
__device__ __forceinline__ void reconstruct(const cx<R> (&w)[6], cx<R> (&acc)[12]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const cx<R> w0 = w[a], w1 = w[3 + a];
        if constexpr (FIRST) {
            static_assert(!FIRST || S < 0, "the first hop is a forward one");
            const R two = R(2), zero = R(0);
            if constexpr (MU == 0) {
                acc[a] = w0;
                acc[3 + a] = w1;
                acc[6 + a] = mk(w1.i, -w1.r);
                acc[9 + a] = mk(w0.i, -w0.r);
            } else if constexpr (MU == 1) {
                acc[a] = w0;
                acc[3 + a] = w1;
                acc[6 + a] = mk(-w1.r, -w1.i);
                acc[9 + a] = w0;
            } else if constexpr (MU == 2) {
                acc[a] = w0;
                acc[3 + a] = w1;
                acc[6 + a] = mk(w0.i, -w0.r);
                acc[9 + a] = mk(-w1.i, w1.r);
            } else {
                acc[a] = mk(zero, zero);
                acc[3 + a] = mk(zero, zero);
                acc[6 + a] = two * w0;
                acc[9 + a] = two * w1;
            }
        } else if constexpr (MU == 0) {
            acc[a] = acc[a] + w0;
            acc[3 + a] = acc[3 + a] + w1;
            acc[6 + a] = S > 0 ? acc[6 + a] + ti(w1) : acc[6 + a] - ti(w1);
            acc[9 + a] = S > 0 ? acc[9 + a] + ti(w0) : acc[9 + a] - ti(w0);
        } else if constexpr (MU == 1) {
            acc[a] = acc[a] + w0;
            acc[3 + a] = acc[3 + a] + w1;
            acc[6 + a] = S > 0 ? acc[6 + a] + w1 : acc[6 + a] - w1;
            acc[9 + a] = S > 0 ? acc[9 + a] - w0 : acc[9 + a] + w0;
        } else if constexpr (MU == 2) {
            acc[a] = acc[a] + w0;
            acc[3 + a] = acc[3 + a] + w1;
            acc[6 + a] = S > 0 ? acc[6 + a] + ti(w0) : acc[6 + a] - ti(w0);
            acc[9 + a] = S > 0 ? acc[9 + a] - ti(w1) : acc[9 + a] + ti(w1);
        } else {
            const R two = R(2);
            if constexpr (S > 0) {
                acc[a] = acc[a] + two * w0;
                acc[3 + a] = acc[3 + a] + two * w1;
            } else {
                acc[6 + a] = acc[6 + a] + two * w0;
                acc[9 + a] = acc[9 + a] + two * w1;
            }
        }
    }
}

template <typename L, typename R>
__device__ __forceinline__ void load_link(const L* __restrict__ U, int mu, int s, int V, cx<R> (&u)[9]) {
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        L q = __ldg(U + (size_t)(mu * 9 + k) * V + s);
        u[k] = mk((R)q.x, (R)q.y);
    }
}

// HALF: the input x is a half-lattice (one parity) block, site n at index n >> 1
template <int P, int MU, bool HALF, bool FIRST, typename Args>
__device__ __forceinline__ void hop_dir_col(const Args& a, const int (&co)[4], int n, int c,
                                            cx<typename Prec<P>::real> (&acc)[12]) {
    using R = typename Prec<P>::real;
    const int Lm = a.L[MU], sm = a.st[MU];
    const int nf = co[MU] == Lm - 1 ? n - (Lm - 1) * sm : n + sm;
    const int nb = co[MU] == 0 ? n + (Lm - 1) * sm : n - sm;
    const int xf = HALF ? nf >> 1 : nf, xb = HALF ? nb >> 1 : nb;
    {   // forward: (1 - gamma_mu) U_mu(n) x(n + mu)
        cx<R> u[9], q[12], h[6], w[6];
        load_link(a.U, MU, n, a.V, u);
        load_col<P>(a.x, xf, c, q);
        project<MU, -1>(q, h);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                cx<R> t = u[3 * i] * h[3 * hh];
                cmac(t, u[3 * i + 1], h[3 * hh + 1]);
                cmac(t, u[3 * i + 2], h[3 * hh + 2]);
                w[3 * hh + i] = t;
            }
        reconstruct<MU, -1, FIRST>(w, acc);
    }
    {   // backward: (1 + gamma_mu) U_mu(n - mu)^+ x(n - mu)
        cx<R> u[9], q[12], h[6], w[6];
        load_link(a.U, MU, nb, a.V, u);
        load_col<P>(a.x, xb, c, q);
        project<MU, +1>(q, h);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                cx<R> t = mk(R(0), R(0));
                cjmac(t, u[i], h[3 * hh]);
                cjmac(t, u[3 + i], h[3 * hh + 1]);
                cjmac(t, u[6 + i], h[3 * hh + 2]);
                w[3 * hh + i] = t;
            }
        reconstruct<MU, +1, false>(w, acc);
    }
}

// y = A x for a packed 6x6 Hermitian block (36 reals: 6 diagonal, 15 complex lower).
template <typename R>
__device__ __forceinline__ void herm6(const R (&m)[36], const cx<R> (&x)[6], cx<R> (&y)[6]) {
#pragma unroll
    for (int i = 0; i < 6; ++i) y[i] = m[i] * x[i];
    int p = 0;
#pragma unroll
    for (int i = 1; i < 6; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j, ++p) {
            const cx<R> A = mk(m[6 + 2 * p], m[7 + 2 * p]);
            cmac(y[i], A, x[j]);
            cjmac(y[j], A, x[i]);
        }
}

template <int P>
__global__ void __launch_bounds__(128) k_dslash_col(const __grid_constant__ DColArgs<P> a) {
    using R = typename Prec<P>::real;
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (long long)a.V * a.ncl) return;
    const int n = (int)(g / a.ncl);
    const int cl = (int)(g - (long long)n * a.ncl);
    const int c = a.c0 + cl;
    int co[4];
    {
        int r = n;
        co[0] = r % a.L[0];
        r /= a.L[0];
        co[1] = r % a.L[1];
        r /= a.L[1];
        co[2] = r % a.L[2];
        co[3] = r / a.L[2];
    }
    cx<R> acc[12];
    hop_dir_col<P, 0, false, true>(a, co, n, c, acc);
    hop_dir_col<P, 1, false, false>(a, co, n, c, acc);
    hop_dir_col<P, 2, false, false>(a, co, n, c, acc);
    hop_dir_col<P, 3, false, false>(a, co, n, c, acc);
    cx<R> q[12];
    load_col<P>(a.x, n, c, q);
    // clover: the chiral blocks act on a = u + l (block 0) and b = u - l (block 1)
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
        R m[36];
#pragma unroll
        for (int e = 0; e < 18; ++e) {
            const double2 v = __ldg(a.C + (size_t)(18 * blk + e) * a.V + n);
            m[2 * e] = (R)v.x;
            m[2 * e + 1] = (R)v.y;
        }
        cx<R> v[6], yv[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = blk == 0 ? q[k] + q[k + 6] : q[k] - q[k + 6];
        herm6(m, v, yv);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            acc[k] = acc[k] + yv[k];
            acc[k + 6] = blk == 0 ? acc[k + 6] + yv[k] : acc[k + 6] - yv[k];
        }
    }
    cx<R> out[12];
    const R kap = (R)a.kappa[cl];
#pragma unroll
    for (int k = 0; k < 12; ++k) out[k] = q[k] - kap * acc[k];
    if (a.residual) {
        cx<R> bb[12];
        load_col<P>(a.b, n, c, bb);
#pragma unroll
        for (int k = 0; k < 12; ++k) out[k] = bb[k] - out[k];
    }
    store_col<P>(a.y, n, c, out);
}

// Rows 3 H .. 3 H + 2 of chiral block BLK times v (Hermitian, packed as herm6).
template <int BLK, int H>
__device__ __forceinline__ void herm6_rows(const double2* __restrict__ C, int V, int n, const cx<double> (&v)[6],
                                           cx<double> (&y)[3]) {
    const double* c = reinterpret_cast<const double*>(C);
    auto real_at = [&](int e) {  // packed real e of this block
        const int q = 36 * BLK + e;
        return __ldg(c + 2 * ((size_t)(q >> 1) * V + n) + (q & 1));
    };
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int i = 3 * H + r;
        y[r] = real_at(i) * v[i];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            if (j == i) continue;
            const int hi = i > j ? i : j, lo = i > j ? j : i, e = 6 + 2 * (hi * (hi - 1) / 2 + lo);
            const cx<double> A = mk(real_at(e), real_at(e + 1));
            if (i > j) cmac(y[r], A, v[j]);
            else cjmac(y[r], A, v[j]);
        }
    }
}

// FP64 operator for few site-columns: four warps share 32 of them, warp t
// takes the two hops of direction t and three rows of one chiral block of the
// clover term, and finishes spin t.  An SM's scheduler starts an FP64
// instruction of a warp every 64 cycles, so one thread per site and column
// takes 40 us however few there are; a quarter of that each, on four times the
// warps, is faster while they do not fill the chip (see split_over_warps).
__global__ void __launch_bounds__(128) k_dslash_col4(const __grid_constant__ DColArgs<BK_FP64> a) {
    __shared__ double hs[4][24][32], ys[4][6][32];
    const int t = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long g = (long long)blockIdx.x * 32 + lane;
    const bool on = g < (long long)a.V * a.ncl;
    const int n = on ? (int)(g / a.ncl) : 0;
    const int cl = on ? (int)(g - (long long)n * a.ncl) : 0;
    const int c = a.c0 + cl;
    int co[4];
    {
        int r = n;
        co[0] = r % a.L[0];
        r /= a.L[0];
        co[1] = r % a.L[1];
        r /= a.L[1];
        co[2] = r % a.L[2];
        co[3] = r / a.L[2];
    }
    if (on) {
        cx<double> acc[12];
        if (t == 0) hop_dir_col<BK_FP64, 0, false, true>(a, co, n, c, acc);
        else if (t == 1) hop_dir_col<BK_FP64, 1, false, true>(a, co, n, c, acc);
        else if (t == 2) hop_dir_col<BK_FP64, 2, false, true>(a, co, n, c, acc);
        else hop_dir_col<BK_FP64, 3, false, true>(a, co, n, c, acc);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            hs[t][2 * k][lane] = acc[k].r;
            hs[t][2 * k + 1][lane] = acc[k].i;
        }
        cx<double> q[12], v[6], y[3];
        load_col<BK_FP64>(a.x, n, c, q);
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = t < 2 ? q[k] + q[k + 6] : q[k] - q[k + 6];
        if (t == 0) herm6_rows<0, 0>(a.C, a.V, n, v, y);
        else if (t == 1) herm6_rows<0, 1>(a.C, a.V, n, v, y);
        else if (t == 2) herm6_rows<1, 0>(a.C, a.V, n, v, y);
        else herm6_rows<1, 1>(a.C, a.V, n, v, y);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            ys[t][2 * r][lane] = y[r].r;
            ys[t][2 * r + 1][lane] = y[r].i;
        }
    }
    __syncthreads();
    if (!on) return;
    const int h = t & 1;  // spin t = h + 2 (t >> 1): row h of u (t < 2) or of l
    const size_t e0 = 4 * (((size_t)n * 12 + 3 * t) * a.x.np + (c >> 1)) + (c & 1), es = 4 * (size_t)a.x.np;
    const double* xq = (const double*)a.x.data + e0;
    const double* bq = (const double*)a.b.data + e0;
    double* yq = (double*)a.y.data + e0;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int k = 2 * (3 * t + r) + p;
            double s = (hs[0][k][lane] + hs[1][k][lane]) + (hs[2][k][lane] + hs[3][k][lane]);
            const double y0 = ys[h][2 * r + p][lane], y1 = ys[2 + h][2 * r + p][lane];
            s += t < 2 ? y0 + y1 : y0 - y1;
            double o = xq[r * es + 2 * p] - a.kappa[cl] * s;
            if (a.residual) o = bq[r * es + 2 * p] - o;
            yq[r * es + 2 * p] = o;
        }
}

void geometry(const int dims[4], int (&L)[4], int (&st)[4]) {
    int stride = 1;
    for (int mu = 0; mu < 4; ++mu) {
        L[mu] = dims[mu];
        st[mu] = stride;
        stride *= dims[mu];
    }
}

// Blocks an SM of the pair kernels.  Measured (us, 3 / 4): FP32 full operator
// 16^3x32, 30 columns 291 / 284, 60 columns 543 / 537, 24^3x48, 96 columns
// 4234 / 4245, 8^3x16, 12 columns (less than one wave) 12.6 / 14.7; FP16
// 16^3x32, 30 columns 279 / 281.
// Below one wave single-warp blocks even out the SMs' shares (192 blocks of 128
// threads give 40 SMs twice the work of the others).
int pair_threads(long long items) { return items <= 152LL * 3 * 128 ? 32 : 128; }
int pair_blocks(int prec, long long items) { return prec == BK_FP32 && items > 152LL * 3 * 128 ? 4 : 3; }

template <int P>
bk_status dslash_pair_impl(const DslashOp& op, cudaStream_t st) {
    // launch over whole pairs [col0 / 2, (col0 + ncol + 1) / 2)
    const int p0 = op.col0 / 2, p1 = (op.col0 + op.ncol + 1) / 2;
    const int maxp = BK_MAX_COLS / 2;
    for (int q0 = p0; q0 < p1; q0 += maxp) {
        const int npl = std::min(maxp, p1 - q0);
        DPairArgs a;
        a.x = op.x;
        a.y = op.y;
        a.b = op.b;
        a.U = (const float*)op.U;
        a.C = (const float*)op.clov;
        geometry(op.dims, a.L, a.st);
        a.V = op.V;
        a.p0 = q0;
        a.npl = npl;
        a.residual = op.residual;
        for (int j = 0; j < npl; ++j) {
            // kappa of columns 2q, 2q + 1 (op.kappa[i] belongs to column col0 + i); a
            // column outside [col0, col0 + ncol) is padding: kappa 0, it is copied through
            const int ca = 2 * (q0 + j) - op.col0, cb = ca + 1;
            const double ka = (ca >= 0 && ca < op.ncol) ? op.kappa[ca] : 0.0;
            const double kb = (cb >= 0 && cb < op.ncol) ? op.kappa[cb] : 0.0;
            a.nk[j] = make_float2((float)-ka, (float)-kb);
        }
        const long long items = (long long)op.V * npl;
        const int T = pair_threads(items);
        const unsigned blocks = (unsigned)((items + T - 1) / T);
        if (pair_blocks(P, items) == 4) k_dslash_pair<P, 4><<<blocks, T, 0, st>>>(a);
        else k_dslash_pair<P, 3><<<blocks, T, 0, st>>>(a);
        BK_CUDA_TRY(cudaGetLastError());
    }
    return BK_OK;
}

// Which FP64 form: n rounds of one 32-item block per SM take the split form 11 us
// each; the other form is as slow as the fullest scheduler, which steps after 4,
// 6 and 8 warps an SM.  Measured (us, split / one thread each): n = 1 14 / 40, 2
// 24 / 40, 3 35 / 42, 4 46 / 42, 5 57 / 63, 6 67 / 63, 7 79 / 80.
bool split_over_warps(long long items) {
    const long long n = ((items + 31) / 32 + 151) / 152;
    return n <= 3 || n == 5 || n == 7;
}

// Threads per block of the one-column-per-thread kernels.  Their FP64 pipe
// works at full rate with few warps, so what matters is that every scheduler
// has the same number: single-warp blocks up to 16 warps a scheduler, two-warp
// blocks above.
int col_threads(long long items) { return items <= 608LL * 16 * 32 ? 32 : 64; }

template <int P>
bk_status dslash_col_impl(const DslashOp& op, cudaStream_t st) {
    for (int c0 = 0; c0 < op.ncol; c0 += BK_MAX_COLS) {
        const int n = std::min(BK_MAX_COLS, op.ncol - c0);
        DColArgs<P> a;
        a.x = op.x;
        a.y = op.y;
        a.b = op.b;
        a.U = (const typename Prec<P>::link*)op.U;
        a.C = (const typename Prec<P>::clov*)op.clov;
        geometry(op.dims, a.L, a.st);
        a.V = op.V;
        a.c0 = op.col0 + c0;
        a.ncl = n;
        a.residual = op.residual;
        for (int j = 0; j < n; ++j) a.kappa[j] = op.kappa[c0 + j];
        const long long items = (long long)op.V * n;
        if constexpr (P == BK_FP64) {
            if (split_over_warps(items) && op.x.np == op.y.np && (!op.residual || op.b.np == op.x.np)) {
                k_dslash_col4<<<(unsigned)((items + 31) / 32), 128, 0, st>>>(a);
                BK_CUDA_TRY(cudaGetLastError());
                continue;
            }
        }
        const int threads = col_threads(items);
        k_dslash_col<P><<<(unsigned)((items + threads - 1) / threads), threads, 0, st>>>(a);
        BK_CUDA_TRY(cudaGetLastError());
    }
    return BK_OK;
}

// ================================================================= conversions

// FP64 / FP32: canonical column j (of a chunk of ncan columns) <-> device column
// dcol[j] (dcol == nullptr: dbase + j), through a shared-memory tile of CT_S
// sites x CT_C columns: a canonical column is contiguous along (site,
// component), a device row along the columns, so one side of a direct copy
// touches a separate line per lane.  Loads issued one by one and half of the
// device-side lanes idle made this slower than the direct copy where L2 holds
// the blocks (8^3x16, 64 columns, FP32: direct 34 us, tile then 42, tile now
// 26; 12^3x24, 24 columns 60, 76, 50; 4^4, 16 columns 3.1, 4.6, 3.2).
constexpr int CT_S = 8, CT_C = 16, CT_R = CT_S * 12;

__device__ __forceinline__ int dev_col(const int* dcol, int dbase, int j) { return dcol ? __ldg(dcol + j) : dbase + j; }

// A thread issues its loads before their first use.  On the device side 16 bytes
// of a pair of the layout are a lane's access (FP32: the pair; FP64: its real or
// its imaginary parts), for the two neighbouring columns of the tile that the
// lane owns, whichever of them the pair starts at.
template <int P, bool PACK>
__global__ void __launch_bounds__(256) k_convert(double2* __restrict__ canon, int ncan, const int* __restrict__ dcol,
                                                 int dbase, Field f) {
    __shared__ double2 tile[CT_R][CT_C + 1];
    const int j0 = blockIdx.y * CT_C, nj = min(CT_C, ncan - j0);
    const int n0 = blockIdx.x * CT_S, nr = 12 * min(CT_S, f.V - n0);
    const int t = threadIdx.x;
    // canonical side, rows fastest
    constexpr int NU = CT_R * CT_C / 256;
    auto canonical = [&](bool load) {
        double2 v[NU];
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            if (256 * u >= nj * CT_R) break;
            const int e = t + 256 * u, j = e / CT_R, r = e - j * CT_R;
            double2* q = canon + ((size_t)(j0 + j) * f.V + n0) * 12 + r;
            if (j < nj && r < nr) {
                if (load) v[u] = *q;
                else *q = tile[r][j];
            }
        }
        if (load)
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                if (256 * u >= nj * CT_R) break;
                const int e = t + 256 * u, j = e / CT_R, r = e - j * CT_R;
                if (j < nj && r < nr) tile[r][j] = v[u];
            }
    };
    if (PACK) canonical(true);
    // device side, columns fastest: a power of two of column pairs side by side
    constexpr int LP = P == BK_FP64 ? 2 : 1;  // lanes a pair
    using R = typename Prec<P>::real;
    int sw = CT_C / 2;
    while (sw > 1 && sw >= nj) sw /= 2;
    const int js = 2 * ((t & (sw * LP - 1)) / LP), part = t & (LP - 1), r0 = t / (sw * LP), rstep = 256 / (sw * LP);
    int col[2], act[2];  // device column; 0: nothing to do here, 1: the column alone, 2: with the next one
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = js + h;
        col[h] = act[h] = 0;
        if (j >= nj) continue;
        col[h] = dev_col(dcol, dbase, j0 + j);
        if (col[h] & 1) act[h] = j > 0 && dev_col(dcol, dbase, j0 + j - 1) == col[h] - 1 ? 0 : 1;
        else act[h] = j + 1 < nj && dev_col(dcol, dbase, j0 + j + 1) == col[h] + 1 ? 2 : 1;
    }
    if (PACK) __syncthreads();
    constexpr int NR = CT_R / (256 / (CT_C / 2 * LP));  // passes over the rows, at most
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!act[h]) continue;
        const int j = js + h, half = col[h] & 1;
        const bool both = act[h] == 2;
        R* base = (R*)f.data + 4 * ((size_t)n0 * 12 * f.np + (col[h] >> 1)) + 2 * part;
        R v[NR][4 / LP];
        if (!PACK)
#pragma unroll
            for (int u = 0; u < NR; ++u) {
                const int r = r0 + u * rstep;
                const R* q = base + 4 * (size_t)r * f.np;
                if (r >= nr) break;
                if constexpr (LP == 2) {
                    if (both) *(double2*)v[u] = *(const double2*)q;
                    else v[u][0] = q[half];
                } else {
                    if (both) *(float4*)v[u] = *(const float4*)q;
                    else v[u][0] = q[half], v[u][2] = q[2 + half];
                }
            }
#pragma unroll
        for (int u = 0; u < NR; ++u) {
            const int r = r0 + u * rstep;
            if (r >= nr) break;
            R* q = base + 4 * (size_t)r * f.np;
            double2 *a = &tile[r][j], *b = both ? a + 1 : a;
            if constexpr (LP == 2) {  // part 0: real parts, 1: imaginary parts
                double *x = (double*)a + part, *y = (double*)b + part;
                if (PACK && both) *(double2*)q = make_double2(*x, *y);
                else if (PACK) q[half] = *x;
                else *x = v[u][0];
                if (!PACK && both) *y = v[u][1];
            } else {
                if (PACK && both) *(float4*)q = make_float4(d2f(a->x), d2f(b->x), d2f(a->y), d2f(b->y));
                else if (PACK) q[half] = d2f(a->x), q[2 + half] = d2f(a->y);
                else *a = make_double2(f2d(v[u][0]), f2d(v[u][2]));
                if (!PACK && both) *b = make_double2(f2d(v[u][1]), f2d(v[u][3]));
            }
        }
    }
    if (!PACK) {
        __syncthreads();
        canonical(false);
    }
}

// FP16: the same with one thread per (canonical column, site), which forms or
// applies the column's scale, its largest component rounded to FP32 first.
__global__ void k_pack16(const double2* __restrict__ canon, int ncan, const int* __restrict__ dcol, int dbase, Field f) {
    const int j = blockIdx.y * blockDim.x + threadIdx.x;
    const int n = blockIdx.x * blockDim.y + threadIdx.y;
    if (j >= ncan || n >= f.V) return;
    const int c = dcol ? dcol[j] : dbase + j;
    const double2* src = canon + ((size_t)j * f.V + n) * 12;
    const size_t e0 = (size_t)n * 12 * f.np + (c >> 1);
    const int half = c & 1;
    double2 v[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = src[k];
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 12; ++k) m = fmaxf(m, fmaxf(fabsf((float)v[k].x), fabsf((float)v[k].y)));
    const float inv = m > 0.f ? 1.0f / m : 0.f;
    __half* q = (__half*)f.data + 4 * e0 + half;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        q[4 * (size_t)k * f.np] = __float2half_rn((float)v[k].x * inv);
        q[4 * (size_t)k * f.np + 2] = __float2half_rn((float)v[k].y * inv);
    }
    float* sc = (float*)(f.norm + (size_t)n * f.np + (c >> 1));
    sc[half] = m;
}
__global__ void k_unpack16(Field f, const int* __restrict__ dcol, int dbase, double2* __restrict__ canon, int ncan) {
    const int j = blockIdx.y * blockDim.x + threadIdx.x;
    const int n = blockIdx.x * blockDim.y + threadIdx.y;
    if (j >= ncan || n >= f.V) return;
    const int c = dcol ? dcol[j] : dbase + j;
    double2* dst = canon + ((size_t)j * f.V + n) * 12;
    const size_t e0 = (size_t)n * 12 * f.np + (c >> 1);
    const int half = c & 1;
    const __half* q = (const __half*)f.data + 4 * e0 + half;
    const float m = ((const float*)(f.norm + (size_t)n * f.np + (c >> 1)))[half];
#pragma unroll
    for (int k = 0; k < 12; ++k)
        dst[k] = make_double2((double)(__half2float(q[4 * (size_t)k * f.np]) * m),
                              (double)(__half2float(q[4 * (size_t)k * f.np + 2]) * m));
}

// zero device column c (both parts, every site and component)
template <int P>
__global__ void k_zero_col(Field f, int c) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)f.V * 12) return;
    const size_t el = (size_t)e * f.np + (c >> 1);
    const int half = c & 1;
    if constexpr (P == BK_FP64 || P == BK_DF64) {
        double* q = (double*)f.data + 4 * el + half;
        q[0] = 0.0;
        q[2] = 0.0;
    } else if constexpr (P == BK_FP32) {
        float* q = (float*)f.data + 4 * el + half;
        q[0] = 0.f;
        q[2] = 0.f;
    } else {
        __half* q = (__half*)f.data + 4 * el + half;
        q[0] = __float2half_rn(0.f);
        q[2] = __float2half_rn(0.f);
        if (e % 12 == 0) ((float*)(f.norm + (size_t)(e / 12) * f.np + (c >> 1)))[half] = 0.f;
    }
}

// precision conversion over pairs [0, np) of in and out (same pair count)
template <int PI, int PO>
__global__ void k_cast(Field in, Field out, int np) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (long long)in.V * np) return;
    const int n = (int)(g / np), p = (int)(g - (long long)n * np);
    typename Prec<PI>::pair r[12], i[12];
    load_pair<PI>(in, n, p, r, i);
    typename Prec<PO>::pair ro[12], io[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        if constexpr (PI == BK_FP64 && PO != BK_FP64) {
            ro[k] = d2f(r[k]);
            io[k] = d2f(i[k]);
        } else if constexpr (PI != BK_FP64 && PO == BK_FP64) {
            ro[k] = f2d(r[k]);
            io[k] = f2d(i[k]);
        } else {
            ro[k] = r[k];
            io[k] = i[k];
        }
    }
    store_pair<PO>(out, n, p, ro, io);
}

__global__ void k_gamma5(const double2* __restrict__ X, double2* __restrict__ Y, long long n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double2 v[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = X[i * 12 + k];
    // gamma_5 of Section 2: spin 0 <-> 2, 1 <-> 3, all entries +1
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Y[i * 12 + a] = v[6 + a];
        Y[i * 12 + 3 + a] = v[9 + a];
        Y[i * 12 + 6 + a] = v[a];
        Y[i * 12 + 9 + a] = v[3 + a];
    }
}

// ================================================================= even-odd (Schur complement) form
//
// Not in the paper: the same system reordered by site parity p(n) = (x + y +
// z + t) mod 2.  With D = A - kappa H (A the site term of Eq. (wd-op), H the
// hopping sum, which only joins sites of opposite parity), the even sites
// solve M x_e = b^_e, M = 1 - kappa^2 A_ee^-1 H_eo A_oo^-1 H_oe.  A
// half-lattice block holds the sites of one parity, site n at index n >> 1
// (with Lx even, n and n + 1 have opposite parities and share n >> 1).  The
// clover-inverse tables (A^-1 per kappa, see k_clover_inverse) and the links
// stay indexed by the full site.

__device__ __forceinline__ int eo_site(int h, int par, const int (&L)[4], int (&co)[4]) {
    int n = 2 * h, r = n;
    co[0] = r % L[0];
    r /= L[0];
    co[1] = r % L[1];
    r /= L[1];
    co[2] = r % L[2];
    co[3] = r / L[2];
    if (((co[0] + co[1] + co[2] + co[3]) & 1) != par) {  // co[0] is even, so co[0] + 1 < Lx
        ++n;
        ++co[0];
    }
    return n;
}

struct EOPairArgs {
    Field in, xs, y;  // in: the other parity; xs: this parity (mode 2); y: the output (this parity)
    const float* __restrict__ U;       // compact links, full-site index
    const float* Ci[BK_MAX_COLS / 2];  // compact A^-1 table of launch pair p - p0 (its kappa)
    int L[4], st[4];
    int V, Vh, p0, npl, par, mode;
    float2 mk2[BK_MAX_COLS / 2];  // mode 2: {-kappa^2} of the pair's columns
};

// mode 1: y = A^-1 H in;  mode 2: y = xs - kappa^2 A^-1 H in  (FP32 / FP16 storage)
template <int P, int MINB>
__global__ void __launch_bounds__(128, MINB) k_eo_pair(const __grid_constant__ EOPairArgs a) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (long long)a.Vh * a.npl) return;
    const int h = (int)(g / a.npl), pl = (int)(g - (long long)h * a.npl), p = a.p0 + pl;
    int co[4];
    const int n = eo_site(h, a.par, a.L, co);
    const float2 one = make_float2(1.f, 1.f), mone = make_float2(-1.f, -1.f);
    float2 ar[12], ai[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) ar[k] = ai[k] = make_float2(0.f, 0.f);
#define BK_EO_DIR(MU)                                                                                          \
    {                                                                                                          \
        const int Lm = a.L[MU], sm = a.st[MU];                                                                 \
        const int nf = co[MU] == Lm - 1 ? n - (Lm - 1) * sm : n + sm;                                          \
        const int nb = co[MU] == 0 ? n + (Lm - 1) * sm : n - sm;                                               \
        hop_pair<P, MU, -1>(a.in, nf >> 1, p, a.U + ((size_t)n * 4 + MU) * BK_LINKC, one, mone, ar, ai); \
        hop_pair<P, MU, +1>(a.in, nb >> 1, p, a.U + ((size_t)nb * 4 + MU) * BK_LINKC, one, mone, ar, ai); \
    }
    BK_EO_DIR(0)
    BK_EO_DIR(1)
    BK_EO_DIR(2)
    BK_EO_DIR(3)
#undef BK_EO_DIR
    site_term<false>(GTab{reinterpret_cast<const float2*>(a.Ci[pl] + (size_t)n * BK_CLOVC)}, one, ar, ai);
    if (a.mode == 2) {
        float2 xr[12], xi[12];
        load_pair<P>(a.xs, h, p, xr, xi);
        const float2 m = a.mk2[pl];
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            ar[k] = pfma(m, ar[k], xr[k]);
            ai[k] = pfma(m, ai[k], xi[k]);
        }
    }
    store_pair<P>(a.y, h, p, ar, ai);
}

template <int P>
struct EOColArgs {
    Field x, xs, y, b;  // x: the other parity (hop input); xs: this parity; y: output; b: residual mode
    const typename Prec<P>::link* __restrict__ U;  // [mu][9][V] double2, full-site index
    const typename Prec<P>::clov* Ci[BK_MAX_COLS];  // [36][V] A^-1 table of launch column c - c0
    int L[4], st[4];
    int V, Vh, c0, ncl, par, mode, hop, residual;
    double kappa[BK_MAX_COLS];
};

// FP64 / double-float, one column per thread:
//   mode 1: y = A^-1 H x
//   mode 2: y = xs - kappa^2 A^-1 H x        (residual: y = b - that)
//   mode 3: y = A^-1 (xs + kappa H x)       (hop = 0: y = A^-1 xs)
template <int P>
__global__ void __launch_bounds__(128) k_eo_col(const __grid_constant__ EOColArgs<P> a) {
    using R = typename Prec<P>::real;
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (long long)a.Vh * a.ncl) return;
    const int h = (int)(g / a.ncl);
    const int cl = (int)(g - (long long)h * a.ncl);
    const int c = a.c0 + cl;
    int co[4];
    const int n = eo_site(h, a.par, a.L, co);
    cx<R> acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = mk(R(0), R(0));
    if (a.hop) {
        hop_dir_col<P, 0, true, true>(a, co, n, c, acc);
        hop_dir_col<P, 1, true, false>(a, co, n, c, acc);
        hop_dir_col<P, 2, true, false>(a, co, n, c, acc);
        hop_dir_col<P, 3, true, false>(a, co, n, c, acc);
    }
    const R kap = (R)a.kappa[cl];
    cx<R> xs[12];
    if (a.mode != 1) load_col<P>(a.xs, h, c, xs);
    if (a.mode == 3) {
#pragma unroll
        for (int k = 0; k < 12; ++k) acc[k] = xs[k] + kap * acc[k];
    }
    cx<R> w[12];
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
        R m[36];
#pragma unroll
        for (int e = 0; e < 18; ++e) {
            const double2 v = __ldg(a.Ci[cl] + (size_t)(18 * blk + e) * a.V + n);
            m[2 * e] = (R)v.x;
            m[2 * e + 1] = (R)v.y;
        }
        cx<R> v[6], yv[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = blk == 0 ? acc[k] + acc[k + 6] : acc[k] - acc[k + 6];
        herm6(m, v, yv);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            if (blk == 0) {
                w[k] = yv[k];
                w[k + 6] = yv[k];
            } else {
                w[k] = w[k] + yv[k];
                w[k + 6] = w[k + 6] - yv[k];
            }
        }
    }
    cx<R> out[12];
    if (a.mode == 2) {
        const R k2 = kap * kap;
#pragma unroll
        for (int k = 0; k < 12; ++k) out[k] = xs[k] - k2 * w[k];
        if (a.residual) {
            cx<R> bb[12];
            load_col<P>(a.b, h, c, bb);
#pragma unroll
            for (int k = 0; k < 12; ++k) out[k] = bb[k] - out[k];
        }
    } else {
#pragma unroll
        for (int k = 0; k < 12; ++k) out[k] = w[k];
    }
    store_col<P>(a.y, h, c, out);
}

// full-lattice FP64 block <-> its two half-lattice blocks (same columns)
__device__ __forceinline__ int site_parity(int n, const int (&L)[4]) {
    int r = n, s = r % L[0];
    r /= L[0];
    s += r % L[1];
    r /= L[1];
    s += r % L[2];
    s += r / L[2];
    return s & 1;
}

struct EOGeo {
    int L[4];
};

template <bool MERGE>
__global__ void k_eo_split_merge(Field full, Field ev, Field od, EOGeo geo) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long row = 12LL * full.np;
    if (g >= (long long)full.V * row) return;
    const int n = (int)(g / row);
    const long long e = g - (long long)n * row;
    const Field& half = site_parity(n, geo.L) ? od : ev;
    double2* f = (double2*)full.data + 2 * g;  // an FP64 element: two double2
    double2* hp = (double2*)half.data + 2 * ((long long)(n >> 1) * row + e);
    if (MERGE) {
        f[0] = hp[0];
        f[1] = hp[1];
    } else {
        hp[0] = f[0];
        hp[1] = f[1];
    }
}

template <int P>
bk_status eo_pair_impl(const EoOp& op, cudaStream_t st) {
    const int p0 = op.col0 / 2, p1 = (op.col0 + op.ncol + 1) / 2;
    const int maxp = BK_MAX_COLS / 2;
    for (int q0 = p0; q0 < p1; q0 += maxp) {
        const int npl = std::min(maxp, p1 - q0);
        EOPairArgs a;
        a.in = op.x;
        a.xs = op.xs;
        a.y = op.y;
        a.U = (const float*)op.U;
        int st4[4];
        geometry(op.dims, a.L, st4);
        for (int mu = 0; mu < 4; ++mu) a.st[mu] = st4[mu];
        a.V = op.V;
        a.Vh = op.V / 2;
        a.p0 = q0;
        a.npl = npl;
        a.par = op.par;
        a.mode = op.mode;
        for (int j = 0; j < npl; ++j) {
            // the pair's columns share one kappa (systems have even widths); a
            // column outside [col0, col0 + ncol) is padding: kappa 0
            const int ca = 2 * (q0 + j) - op.col0, cb = ca + 1;
            const bool ina = ca >= 0 && ca < op.ncol, inb = cb >= 0 && cb < op.ncol;
            const double ka = ina ? op.kappa[ca] : 0.0, kb = inb ? op.kappa[cb] : 0.0;
            a.Ci[j] = (const float*)op.Ci[ina ? ca : cb];
            a.mk2[j] = make_float2((float)(-ka * ka), (float)(-kb * kb));
        }
        const long long items = (long long)a.Vh * npl;
        const int T = pair_threads(items);
        const unsigned blocks = (unsigned)((items + T - 1) / T);
        if (pair_blocks(P, items) == 4) k_eo_pair<P, 4><<<blocks, T, 0, st>>>(a);
        else k_eo_pair<P, 3><<<blocks, T, 0, st>>>(a);
        BK_CUDA_TRY(cudaGetLastError());
    }
    return BK_OK;
}

template <int P>
bk_status eo_col_impl(const EoOp& op, cudaStream_t st) {
    for (int c0 = 0; c0 < op.ncol; c0 += BK_MAX_COLS) {
        const int n = std::min(BK_MAX_COLS, op.ncol - c0);
        EOColArgs<P> a;
        a.x = op.x;
        a.xs = op.xs;
        a.y = op.y;
        a.b = op.b;
        a.U = (const typename Prec<P>::link*)op.U;
        geometry(op.dims, a.L, a.st);
        a.V = op.V;
        a.Vh = op.V / 2;
        a.c0 = op.col0 + c0;
        a.ncl = n;
        a.par = op.par;
        a.mode = op.mode;
        a.hop = op.hop;
        a.residual = op.residual;
        for (int j = 0; j < n; ++j) {
            a.kappa[j] = op.kappa[c0 + j];
            a.Ci[j] = (const typename Prec<P>::clov*)op.Ci[c0 + j];
        }
        const long long items = (long long)a.Vh * n;
        const int threads = col_threads(items);
        k_eo_col<P><<<(unsigned)((items + threads - 1) / threads), threads, 0, st>>>(a);
        BK_CUDA_TRY(cudaGetLastError());
    }
    return BK_OK;
}

}  // namespace

bk_status launch_dslash(int prec, const DslashOp& op, cudaStream_t st) {
    if (op.ncol <= 0) return BK_OK;
    switch (prec) {
        case BK_FP64: return dslash_col_impl<BK_FP64>(op, st);
        case BK_DF64: return dslash_col_impl<BK_DF64>(op, st);
        case BK_FP32: return dslash_pair_impl<BK_FP32>(op, st);
        case BK_FP16: return dslash_pair_impl<BK_FP16>(op, st);
    }
    return BK_ERR_INVALID_ARG;
}

bk_status launch_pack(int prec, const double* canon, int ncan, const int* dcol, int dbase, Field f, cudaStream_t st) {
    if (ncan <= 0) return BK_OK;
    // sites on grid.x (up to 2^31 - 1 blocks), columns on grid.y
    const dim3 tiles((f.V + CT_S - 1) / CT_S, (ncan + CT_C - 1) / CT_C);
    double2* c = (double2*)canon;
    switch (prec) {
        case BK_FP64: k_convert<BK_FP64, true><<<tiles, 256, 0, st>>>(c, ncan, dcol, dbase, f); break;
        case BK_FP32: k_convert<BK_FP32, true><<<tiles, 256, 0, st>>>(c, ncan, dcol, dbase, f); break;
        case BK_FP16:
            k_pack16<<<dim3((f.V + 7) / 8, (ncan + 31) / 32), dim3(32, 8), 0, st>>>(c, ncan, dcol, dbase, f);
            break;
        default: return BK_ERR_INVALID_ARG;
    }
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status launch_unpack(int prec, Field f, const int* dcol, int dbase, double* canon, int ncan, cudaStream_t st) {
    if (ncan <= 0) return BK_OK;
    const dim3 tiles((f.V + CT_S - 1) / CT_S, (ncan + CT_C - 1) / CT_C);
    double2* c = (double2*)canon;
    switch (prec) {
        case BK_FP64: k_convert<BK_FP64, false><<<tiles, 256, 0, st>>>(c, ncan, dcol, dbase, f); break;
        case BK_FP32: k_convert<BK_FP32, false><<<tiles, 256, 0, st>>>(c, ncan, dcol, dbase, f); break;
        case BK_FP16:
            k_unpack16<<<dim3((f.V + 7) / 8, (ncan + 31) / 32), dim3(32, 8), 0, st>>>(f, dcol, dbase, c, ncan);
            break;
        default: return BK_ERR_INVALID_ARG;
    }
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status launch_zero_col(int prec, Field f, int c, cudaStream_t st) {
    const long long n = (long long)f.V * 12;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    switch (prec) {
        case BK_FP64: k_zero_col<BK_FP64><<<blocks, 256, 0, st>>>(f, c); break;
        case BK_FP32: k_zero_col<BK_FP32><<<blocks, 256, 0, st>>>(f, c); break;
        case BK_FP16: k_zero_col<BK_FP16><<<blocks, 256, 0, st>>>(f, c); break;
        default: return BK_ERR_INVALID_ARG;
    }
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status launch_cast(int pin, Field in, int pout, Field out, int np, cudaStream_t st) {
    if (np <= 0) return BK_OK;
    const long long items = (long long)in.V * np;
    const unsigned blocks = (unsigned)((items + 127) / 128);
#define BK_CAST(A, B)                                              \
    if (pin == A && pout == B) {                                   \
        k_cast<A, B><<<blocks, 128, 0, st>>>(in, out, np);         \
        BK_CUDA_TRY(cudaGetLastError());                           \
        return BK_OK;                                              \
    }
    BK_CAST(BK_FP64, BK_FP32)
    BK_CAST(BK_FP64, BK_FP16)
    BK_CAST(BK_FP32, BK_FP64)
    BK_CAST(BK_FP16, BK_FP64)
    BK_CAST(BK_FP32, BK_FP16)
    BK_CAST(BK_FP16, BK_FP32)
    BK_CAST(BK_FP64, BK_FP64)
    BK_CAST(BK_FP32, BK_FP32)
    BK_CAST(BK_FP16, BK_FP16)
#undef BK_CAST
    return BK_ERR_INVALID_ARG;
}

bk_status launch_gamma5_canon(const double* X, double* Y, long long n, cudaStream_t st) {
    if (n <= 0) return BK_OK;
    k_gamma5<<<(unsigned)((n + 127) / 128), 128, 0, st>>>((const double2*)X, (double2*)Y, n);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status launch_eo(int prec, const EoOp& op, cudaStream_t st) {
    if (op.ncol <= 0) return BK_OK;
    if ((op.dims[0] & 1) || (op.V & 1)) {
        bk_set_error("the even-odd form needs an even extent in x");
        return BK_ERR_INVALID_ARG;
    }
    if (op.mode < 1 || op.mode > 3 || ((prec == BK_FP32 || prec == BK_FP16) && op.mode == 3)) {
        bk_set_error("bad even-odd operator mode");
        return BK_ERR_INVALID_ARG;
    }
    switch (prec) {
        case BK_FP64: return eo_col_impl<BK_FP64>(op, st);
        case BK_DF64: return eo_col_impl<BK_DF64>(op, st);
        case BK_FP32: return eo_pair_impl<BK_FP32>(op, st);
        case BK_FP16: return eo_pair_impl<BK_FP16>(op, st);
    }
    return BK_ERR_INVALID_ARG;
}

static bk_status eo_split_merge(bool merge, Field full, Field ev, Field od, const int dims[4], cudaStream_t st) {
    if (ev.np != full.np || od.np != full.np || 2 * ev.V != full.V || 2 * od.V != full.V) {
        bk_set_error("even-odd split: half blocks must have the full block's columns and half its sites");
        return BK_ERR_INVALID_ARG;
    }
    EOGeo geo;
    for (int mu = 0; mu < 4; ++mu) geo.L[mu] = dims[mu];
    const long long items = (long long)full.V * 12 * full.np;
    const unsigned blocks = (unsigned)((items + 255) / 256);
    if (merge) k_eo_split_merge<true><<<blocks, 256, 0, st>>>(full, ev, od, geo);
    else k_eo_split_merge<false><<<blocks, 256, 0, st>>>(full, ev, od, geo);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status launch_eo_split(Field full, Field ev, Field od, const int dims[4], cudaStream_t st) {
    return eo_split_merge(false, full, ev, od, dims, st);
}

bk_status launch_eo_merge(Field ev, Field od, Field full, const int dims[4], cudaStream_t st) {
    return eo_split_merge(true, full, ev, od, dims, st);
}
