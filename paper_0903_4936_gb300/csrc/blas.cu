// Block linear algebra of block BiCGSTAB / block BiCGGR (Section 3 of
// arXiv:0903.4936): column dot products for the traces Tr(W^H R) and the
// residual norms, the finishing sums of every reduction, block updates of
// FP16 blocks, sums into FP64, seeded blocks, the L x L solves of any size
// (FP64), and the launchers.  Gram matrices and the updates of FP64 / FP32
// blocks: rows.cu (systems of up to 12 columns) and wide.cu.
//
// All block kernels are block-diagonal over a partition of the columns into
// independent systems (one system for a plain solve).  Blocks are in the
// RHS-interleaved pair layout of bk_common.cuh.
#include <algorithm>
#include <cstring>

#include "blas_common.cuh"

SysPart make_part(int nsys, const int* Ls) {
    SysPart p;
    p.nsys = nsys;
    p.col0[0] = 0;
    p.coef_off[0] = 0;
    for (int s = 0; s < nsys; ++s) {
        p.L[s] = Ls[s];
        p.col0[s + 1] = p.col0[s] + ((Ls[s] + 1) & ~1);
        p.coef_off[s + 1] = p.coef_off[s] + Ls[s] * Ls[s];
    }
    for (int s = nsys; s < BK_MAX_SYS; ++s) p.L[s] = 0;
    for (int s = nsys + 1; s <= BK_MAX_SYS; ++s) {
        p.col0[s] = p.col0[nsys];
        p.coef_off[s] = p.coef_off[nsys];
    }
    p.active = all_systems(nsys);
    return p;
}

SysPart single_part(int L) { return make_part(1, &L); }

namespace {

// pairs of a tile of the any-size FP16 update
constexpr int TILE_MAXP = 64;

// row chunks (partial-sum rows) of the column dots, at most
constexpr int MAX_CHUNKS = 304;  // 2 per SM of 152

// ---------------------------------------------------------------- warp tiles
//
// The FP16 update of systems of at most 12 columns gives every warp a run of
// whole active systems of at most 32 pairs, one pair per lane, and lets the
// warps of a block take different sites (a site's 12 components stay with one
// lane, which forms the scale of the stored column).  A lane loads only its own
// pair of each operand; the pairs of the other columns of its system come from
// the lanes that hold them by register shuffles.
constexpr int WT_PAIRS = 32;

struct WLane {
    bool live;  // the lane holds a pair of an active system
    int q, s, qs, Ls, i0, nps, base;  // pair, system, its first pair, size, first column, pairs, first lane
};

__device__ __forceinline__ WLane wlane(const SysPart& p, int tp0, int tnp, int lane) {
    WLane w;
    w.live = lane < tnp;
    if (w.live) {
        w.q = tp0 + lane;
        w.s = sys_of_pair(p, w.q);
        w.qs = p.col0[w.s] / 2;
        w.Ls = p.L[w.s];
        w.i0 = 2 * w.q - p.col0[w.s];
        w.nps = (w.Ls + 1) / 2;
        w.base = lane - (w.q - w.qs);
    } else {
        w.q = tp0;
        w.s = 0;
        w.qs = tp0;
        w.Ls = 0;
        w.i0 = 0;
        w.nps = 1;
        w.base = lane;
    }
    return w;
}

constexpr int GW_WARPS = 8;

// ---------------------------------------------------------------- finishing sums

// Sums over the chunks' partial rows: FIN_E entries x FIN_ROWS row slices per
// block (a thread adds every FIN_ROWS-th row), combined in shared memory in a
// fixed order.  Few entries a block, because the FP64 adds of one SM are the
// bound (one thread per entry over all rows: 75 us for 360 entries of 304
// rows; 32 entries a block: 18 us for 144 entries of 608).
constexpr int FIN_E = 8;
constexpr int FIN_ROWS = 32;

template <typename F>
__device__ __forceinline__ double2 sum_rows(int nrows, bool on, F row) {
    __shared__ double2 red[FIN_ROWS][FIN_E];
    double2 v = make_double2(0.0, 0.0);
    if (on) {
#pragma unroll 4
        for (int c = threadIdx.y; c < nrows; c += FIN_ROWS) {
            const double2 x = row(c);
            v.x += x.x;
            v.y += x.y;
        }
    }
    red[threadIdx.y][threadIdx.x] = v;
#pragma unroll
    for (int o = FIN_ROWS / 2; o > 0; o >>= 1) {
        __syncthreads();
        if (threadIdx.y < o) {
            const double2 b = red[threadIdx.y + o][threadIdx.x];
            v.x += b.x;
            v.y += b.y;
            red[threadIdx.y][threadIdx.x] = v;
        }
    }
    return v;  // valid in the threads of row 0
}

// G[e] (and G2) = sum over chunks of the partial sums, for the entries of the
// active systems.
__global__ void __launch_bounds__(FIN_E * FIN_ROWS) k_gram_finish(const double2* __restrict__ partial, int nchunk, int NB,
                                                              SysPart p, double2* __restrict__ G,
                                                              double2* __restrict__ G2) {
    const int ne = p.coef_off[p.nsys];
    const int e = blockIdx.x * FIN_E + threadIdx.x;
    const int b = e / ne, el = e - b * ne;
    bool on = e < NB * ne;
    if (on) {
        int lo = 0, hi = p.nsys - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (el >= p.coef_off[mid]) lo = mid;
            else hi = mid - 1;
        }
        on = (p.active >> lo) & 1ull;
    }
    const double2 v =
        sum_rows(nchunk, on, [&](int c) { return __ldg(partial + (size_t)(b * nchunk + c) * ne + el); });
    if (on && threadIdx.y == 0) (b == 0 ? G : G2)[el] = v;
}

// ---------------------------------------------------------------- column dots
//
// Over pairs [q0, q0 + nq), column by column: MODE 0: out[0] = A^H B, 1:
// out[0] = |A|^2, 2: out[0] = A^H B and out[1] = |A|^2 (one read of A).
// Thread block: TX pair slots x 256 / TX rows (site, component); grid: (pair
// groups, row chunks).  Rows, not sites: 12 times the parallelism, which the
// small lattices need.  UR rows per thread are loaded before any is used.
// Sums as in the Gram kernels.

template <int P, int MODE, int TX>
__global__ void __launch_bounds__(256) k_coldot(Field A, Field B, int q0, int nq, double2* __restrict__ partial,
                                                unsigned rows, int nchunk) {
    using R = typename Prec<P>::real;
    using R2 = typename Prec<P>::pair;
    constexpr int TY = 256 / TX;  // rows: narrow column ranges get more of them per block
    constexpr int NOUT = MODE == 2 ? 2 : 1;
    constexpr int UR = P == BK_FP64 ? 2 : 4;
    __shared__ double2 red[TY][TX][NOUT * 2];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int ql = blockIdx.x * TX + tx, q = q0 + ql;
    const bool on = ql < nq;
    const int chunk = blockIdx.y, np = A.np;
    R2 dr = pzero<R2>(), di = dr, nn = dr;
    double2 d0 = make_double2(0.0, 0.0), d1 = d0, n01 = d0;
    auto flush = [&]() {
        if (MODE != 1) {
            d0 = make_double2(d0.x + f2d(dr.x), d0.y + f2d(di.x));
            d1 = make_double2(d1.x + f2d(dr.y), d1.y + f2d(di.y));
        }
        if (MODE != 0) n01 = make_double2(n01.x + f2d(nn.x), n01.y + f2d(nn.y));
        dr = di = nn = pzero<R2>();
    };
    int since = 0;
    const unsigned step = (unsigned)nchunk * TY;
    for (unsigned r0 = (unsigned)chunk * TY + ty; r0 < rows; r0 += step * UR) {
        CxPair<R2> a[UR], b[UR];
#pragma unroll
        for (int x = 0; x < UR; ++x) {
            const unsigned r = r0 + x * step;
            a[x] = b[x] = cp_zero<R2>();
            if (on && r < rows) {
                R2 sa = pzero<R2>(), sb = sa;
                if constexpr (P == BK_FP16) {
                    sa = pair_scale<P>(A, r / 12, q);
                    if (MODE != 1) sb = pair_scale<P>(B, r / 12, q);
                }
                a[x] = ldg_at<P>(A, (size_t)r * np + q, sa);
                if (MODE != 1) b[x] = ldg_at<P>(B, (size_t)r * np + q, sb);
            }
        }
#pragma unroll
        for (int x = 0; x < UR; ++x) {
            if (MODE != 1) {
                dr = pfma(a[x].re, b[x].re, dr);
                dr = pfma(a[x].im, b[x].im, dr);
                di = pfma(a[x].re, b[x].im, di);
                R2 nai;
                nai.x = -a[x].im.x;
                nai.y = -a[x].im.y;
                di = pfma(nai, b[x].re, di);
            }
            if (MODE != 0) {
                nn = pfma(a[x].re, a[x].re, nn);
                nn = pfma(a[x].im, a[x].im, nn);
            }
        }
        if constexpr (P != BK_FP64) {
            since += UR;
            if (since >= ROW_FLUSH) {
                flush();
                since = 0;
            }
        }
    }
    flush();
    if (MODE != 1) {
        red[ty][tx][0] = d0;
        red[ty][tx][1] = d1;
    }
    if (MODE != 0) {
        red[ty][tx][NOUT * 2 - 2] = make_double2(n01.x, 0.0);
        red[ty][tx][NOUT * 2 - 1] = make_double2(n01.y, 0.0);
    }
    __syncthreads();
    for (int t = ty * TX + tx; t < TX * NOUT * 2; t += 256) {
        const int c = t % (NOUT * 2), x = t / (NOUT * 2), qx = blockIdx.x * TX + x;
        if (qx >= nq) continue;
        double2 v = make_double2(0.0, 0.0);
        for (int y = 0; y < TY; ++y) {
            v.x += red[y][x][c].x;
            v.y += red[y][x][c].y;
        }
        partial[((size_t)chunk * NOUT + (c >> 1)) * (2 * nq) + 2 * qx + (c & 1)] = v;
    }
}

// out[kk * ldo + j] = sum over chunks, columns j < n
__global__ void __launch_bounds__(FIN_E * FIN_ROWS) k_coldot_finish(const double2* __restrict__ partial, int nchunk,
                                                                int npair, int nq, int n, double2* __restrict__ out,
                                                                int ldo) {
    const int e = blockIdx.x * FIN_E + threadIdx.x;
    const bool on = e < npair * n;
    const int kk = e / n, j = e - kk * n;
    const double2 v = sum_rows(
        nchunk, on, [&](int c) { return __ldg(partial + ((size_t)c * npair + kk) * (2 * nq) + j); });
    if (on && threadIdx.y == 0) out[(size_t)kk * ldo + j] = v;
}

// ---------------------------------------------------------------- fused block update
//
//   matpart_j = sum_{i in s} comb_i M_s[i][j],   comb_i = sum_u ma_u Mi_u,i
//   Y_j       = sum_t ea_t E_t,j + ym matpart_j
//   X_j      += xa Xin_j + xm matpart_j          (X in FP64 for FP64 blocks, else FP32)
// coefficient value = mult * (ptr ? ptr[s] : 1), ptr complex FP64 per system.
//
// FP64 and FP32 blocks: k_update_r (rows.cu), k_update_t (wide.cu).  FP16 blocks
// here: systems of at most 12 columns in k_genop_w (warp tiles, below), larger
// ones in k_genop: SR site rows x 64 pair slots over a tile of whole systems,
// grid (tiles, site chunks, 64 pairs of a wider system).  Each thread forms the
// comb columns of its system pair by pair (the system's threads share the reads
// through L1) and combines them with its two columns of M, read through the
// read-only path, then writes its pair of Y and X.  Optionally the squared
// norms of the Y columns are summed per chunk.

// element with its (site, pair) scale applied
__device__ __forceinline__ CxPair<float2> load_scaled(const Field& f, int n, int k, int q, float2 sc) {
    CxPair<float2> v;
    load_elem<BK_FP16>(f, n, k, q, v.re, v.im);
    v.re = pmul(v.re, sc);
    v.im = pmul(v.im, sc);
    return v;
}

template <int SR>
__global__ void __launch_bounds__(256) k_genop(const __grid_constant__ GenOp g, PTiles tl, int V, int nchunk,
                                               int ncols) {
    constexpr int P = BK_FP16, XP = BK_FP32;
    using R = float;
    using R2 = float2;
    __shared__ double2 ynred[SR][TILE_MAXP];
    const int tx = threadIdx.x, t = tx + (int)blockIdx.z * TILE_MAXP, r = threadIdx.y;  // systems wider than a tile: grid.z
    const int tile = blockIdx.x, chunk = blockIdx.y;
    const int tp0 = tl.p0[tile], tnp = tl.np[tile];
    bool on = t < tnp;
    const int q = tp0 + t;
    int s = 0, qs = 0, Ls = 0, i0 = 0;
    if (on) {
        s = sys_of_pair(g.p, q);
        qs = g.p.col0[s] / 2;
        Ls = g.p.L[s];
        i0 = 2 * q - g.p.col0[s];
        if (g.skip && g.skip[s]) on = false;
    }
    const int nps = (Ls + 1) / 2;
    const bool mat = g.nmi > 0 && g.M != nullptr && ((g.hasY && g.ym != 0.0) || (g.hasX && g.xm != 0.0));
    cx<R> ea[GENOP_MAXE], ma[GENOP_MAXMI], xa = mk(R(0), R(0));
#pragma unroll
    for (int e = 0; e < GENOP_MAXE; ++e) ea[e] = e < g.ne ? coef<P>(g.ea[e], g.ea_mult[e], 0, s) : mk(R(0), R(0));
#pragma unroll
    for (int u = 0; u < GENOP_MAXMI; ++u) ma[u] = u < g.nmi ? coef<P>(g.ma[u], g.ma_mult[u], 0, s) : mk(R(0), R(0));
    if (g.hasX) xa = coef<P>(g.xa, g.xa_mult, 0, s);
    const double2* M = reinterpret_cast<const double2*>(g.M) + (on && mat ? g.p.coef_off[s] : 0);
    const bool j1ok = i0 + 1 < Ls;
    R2 ym2;
    ym2.x = (R)g.ym;
    ym2.y = (R)g.ym;
    const R2 xm2 = bcast((R)g.xm);
    double yn[2] = {0.0, 0.0};
    const int iters = (V + SR * nchunk - 1) / (SR * nchunk);
    for (int it = 0; it < iters; ++it) {
        const int n = (it * nchunk + chunk) * SR + r;
        if (!on || n >= V) continue;
        R2 esc[GENOP_MAXE];
#pragma unroll
        for (int e = 0; e < GENOP_MAXE; ++e)
            if (e < g.ne) esc[e] = pair_scale<P>(g.E[e], n, q);
        const R2 xsc = g.hasX ? pair_scale<P>(g.Xin, n, q) : pzero<R2>();
        R2 yr[12], yi[12];
        R sa = R(0), sb = R(0);
#pragma unroll 2
        for (int k = 0; k < 12; ++k) {
            // matpart of the thread's columns j = i0, i0 + 1 (pair over j):
            // comb_i = sum_u ma_u Mi_u,i for every column i of the system, read
            // pair by pair (the system's threads share the rows through L1)
            CxPair<R2> mp;
            mp.re = pzero<R2>();
            mp.im = pzero<R2>();
            if (mat) {
                // one partner pair ip of the system at a time; i = 2 ip + h
                auto accumulate = [&](int ip, const R2 (&mr2)[2], const R2 (&mi2)[2]) {
                    CxPair<R2> c;
                    c.re = pzero<R2>();
                    c.im = pzero<R2>();
#pragma unroll
                    for (int u = 0; u < GENOP_MAXMI; ++u)
                        if (u < g.nmi)
                            cpair_mac<R, R2>(c, ma[u], load_scaled(g.Mi[u], n, k, qs + ip,
                                                                      pair_scale<P>(g.Mi[u], n, qs + ip)));
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const R cr = h ? c.re.y : c.re.x, ci = h ? c.im.y : c.im.x;
                        R2 crr, cii, nmi;
                        crr.x = cr;
                        crr.y = cr;
                        cii.x = ci;
                        cii.y = ci;
                        nmi.x = -mi2[h].x;
                        nmi.y = -mi2[h].y;
                        mp.re = pfma(crr, mr2[h], mp.re);
                        mp.re = pfma(cii, nmi, mp.re);
                        mp.im = pfma(crr, mi2[h], mp.im);
                        mp.im = pfma(cii, mr2[h], mp.im);
                    }
                };
                {
                    for (int ip = 0; ip < nps; ++ip) {
                        R2 mr2[2], mi2[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int i = 2 * ip + h;
                            double2 m0 = make_double2(0.0, 0.0), m1 = make_double2(0.0, 0.0);
                            if (i < Ls) {
                                m0 = __ldg(M + i * Ls + i0);
                                if (j1ok) m1 = __ldg(M + i * Ls + i0 + 1);
                            }
                            mr2[h].x = (R)m0.x;
                            mr2[h].y = (R)m1.x;
                            mi2[h].x = (R)m0.y;
                            mi2[h].y = (R)m1.y;
                        }
                        accumulate(ip, mr2, mi2);
                    }
                }
            }
            if (g.hasY) {
                CxPair<R2> y;
                y.re = pmul(ym2, mp.re);
                y.im = pmul(ym2, mp.im);
#pragma unroll
                for (int e = 0; e < GENOP_MAXE; ++e)
                    if (e < g.ne) cpair_mac<R, R2>(y, ea[e], load_scaled(g.E[e], n, k, q, esc[e]));
                if (g.ynorm) {
                    sa = fma(y.re.x, y.re.x, sa);
                    sa = fma(y.im.x, y.im.x, sa);
                    sb = fma(y.re.y, y.re.y, sb);
                    sb = fma(y.im.y, y.im.y, sb);
                }
                yr[k] = y.re;
                yi[k] = y.im;
            }
            if (g.hasX) {
                const CxPair<R2> v = load_scaled(g.Xin, n, k, q, xsc);
                const size_t e = ((size_t)n * 12 + k) * g.X.np + q;
                CxPair<R2> x = load_at<XP>(g.X, e);
                cpair_mac<R, R2>(x, xa, v);
                store_at<XP>(g.X, e, pfma(xm2, mp.re, x.re), pfma(xm2, mp.im, x.im));
            }
        }
        if (g.hasY) store_pair<P>(g.Y, n, q, yr, yi);
        yn[0] += (double)sa;
        yn[1] += (double)sb;
    }
    if (g.ynorm) {
        ynred[r][tx] = make_double2(yn[0], yn[1]);
        __syncthreads();
        if (on && r == 0) {
            double2 v = make_double2(0.0, 0.0);
            for (int rr = 0; rr < SR; ++rr) {
                v.x += ynred[rr][tx].x;
                v.y += ynred[rr][tx].y;
            }
            g.ynorm[(size_t)chunk * ncols + 2 * q] = v.x;
            g.ynorm[(size_t)chunk * ncols + 2 * q + 1] = v.y;
        }
    }
}

// FP16 update over warp tiles (systems of at most MAXL <= 12 columns).  Each
// lane forms comb = sum_u ma_u Mi_u for its own pair, takes the comb pairs of
// its system's other lanes by shuffles and combines them with its two columns
// of M (registers), then adds the elementwise terms and writes its pair of Y
// and X.  Every operand has the layout's pair count np, so one element offset
// serves them all.  NMI, NE and HX fix the operand counts of the solvers'
// updates at compile time.
template <int MAXL, int NMI, int NE, int HX>
__global__ void __launch_bounds__(GW_WARPS * 32) k_genop_w(const __grid_constant__ GenOp g, PTiles wt, int V,
                                                          int nchunk, int ncols, int np) {
    constexpr int P = BK_FP16, XP = BK_FP32;
    using R = float;
    using R2 = float2;
    constexpr int MMI = NMI >= 0 ? NMI : GENOP_MAXMI, ME = NE >= 0 ? NE : GENOP_MAXE;
    const int nmi = NMI >= 0 ? NMI : g.nmi, ne = NE >= 0 ? NE : g.ne;
    const bool hx = HX >= 0 ? HX != 0 : g.hasX != 0;
    __shared__ double2 ynred[GW_WARPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int chunk = blockIdx.y;
    const WLane L = wlane(g.p, wt.p0[blockIdx.x], wt.np[blockIdx.x], lane);
    const bool act = L.live && !(g.skip && g.skip[L.s]);
    const int s = L.s;
    const bool mat = nmi > 0 && g.M != nullptr && ((g.hasY && g.ym != 0.0) || (hx && g.xm != 0.0));
    cx<R> ea[ME > 0 ? ME : 1], ma[MMI > 0 ? MMI : 1], xa = mk(R(0), R(0));
#pragma unroll
    for (int e = 0; e < ME; ++e) ea[e] = e < ne ? coef<P>(g.ea[e], g.ea_mult[e], 0, s) : mk(R(0), R(0));
#pragma unroll
    for (int u = 0; u < MMI; ++u) ma[u] = u < nmi ? coef<P>(g.ma[u], g.ma_mult[u], 0, s) : mk(R(0), R(0));
    if (hx) xa = coef<P>(g.xa, g.xa_mult, 0, s);
    // the lane's two columns of M; rows and columns past the system's size are zero
    R2 Mr[MAXL], Mi[MAXL];
    {
        const double2* M = reinterpret_cast<const double2*>(g.M) + (act && mat ? g.p.coef_off[s] : 0);
        const bool j1ok = L.i0 + 1 < L.Ls;
#pragma unroll
        for (int i = 0; i < MAXL; ++i) {
            double2 m0 = make_double2(0.0, 0.0), m1 = make_double2(0.0, 0.0);
            if (act && mat && i < L.Ls) {
                m0 = M[i * L.Ls + L.i0];
                if (j1ok) m1 = M[i * L.Ls + L.i0 + 1];
            }
            Mr[i].x = (R)m0.x;
            Mr[i].y = (R)m1.x;
            Mi[i].x = (R)m0.y;
            Mi[i].y = (R)m1.y;
        }
    }
    const R2 ym2 = bcast((R)g.ym);
    const R2 xm2 = bcast((R)g.xm);
    double yn0 = 0.0, yn1 = 0.0;
    const int iters = (V + GW_WARPS * nchunk - 1) / (GW_WARPS * nchunk);
    for (int it = 0; it < iters; ++it) {
        const int n = (it * nchunk + chunk) * GW_WARPS + w;
        if (n >= V) break;  // the same for the whole warp
        R2 msc[MMI > 0 ? MMI : 1], esc[ME > 0 ? ME : 1], xsc = pzero<R2>();
#pragma unroll
        for (int u = 0; u < MMI; ++u) msc[u] = act && u < nmi ? pair_scale<P>(g.Mi[u], n, L.q) : pzero<R2>();
#pragma unroll
        for (int e = 0; e < ME; ++e) esc[e] = act && e < ne ? pair_scale<P>(g.E[e], n, L.q) : pzero<R2>();
        if (act && hx) xsc = pair_scale<P>(g.Xin, n, L.q);
        R2 yr[12], yi[12];
        R sa = R(0), sb = R(0);
        const size_t e0 = (size_t)n * 12 * np + L.q;
        // the site's 12 components stay in registers for the scaled store
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const size_t e = e0 + (size_t)k * np;
            CxPair<R2> vm[MMI > 0 ? MMI : 1], ve[ME > 0 ? ME : 1], vx = cp_zero<R2>(), x = cp_zero<R2>();
#pragma unroll
            for (int u = 0; u < MMI; ++u)
                vm[u] = act && mat && u < nmi ? ldg_at<P>(g.Mi[u], e, msc[u]) : cp_zero<R2>();
#pragma unroll
            for (int t = 0; t < ME; ++t) ve[t] = act && g.hasY && t < ne ? ldg_at<P>(g.E[t], e, esc[t]) : cp_zero<R2>();
            if (act && hx) {
                vx = ldg_at<P>(g.Xin, e, xsc);
                x = load_at<XP>(g.X, e);
            }
            CxPair<R2> mp = cp_zero<R2>();
            if (mat) {
                CxPair<R2> c = cp_zero<R2>();
#pragma unroll
                for (int u = 0; u < MMI; ++u)
                    if (u < nmi) cpair_mac<R, R2>(c, ma[u], vm[u]);
#pragma unroll
                for (int ip = 0; ip < MAXL / 2; ++ip) {
                    const CxPair<R2> cp = shfl_pair(c, L.base + min(ip, L.nps - 1));
                    if (ip < L.nps) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const R2 cr = bcast(h ? cp.re.y : cp.re.x), ci = bcast(h ? cp.im.y : cp.im.x);
                            const R2 nci = bcast(h ? -cp.im.y : -cp.im.x);
                            mp.re = pfma(cr, Mr[2 * ip + h], mp.re);
                            mp.re = pfma(nci, Mi[2 * ip + h], mp.re);
                            mp.im = pfma(cr, Mi[2 * ip + h], mp.im);
                            mp.im = pfma(ci, Mr[2 * ip + h], mp.im);
                        }
                    }
                }
            }
            if (!act) continue;
            if (g.hasY) {
                CxPair<R2> y;
                y.re = pmul(ym2, mp.re);
                y.im = pmul(ym2, mp.im);
#pragma unroll
                for (int t = 0; t < ME; ++t)
                    if (t < ne) cpair_mac<R, R2>(y, ea[t], ve[t]);
                if (g.ynorm) {
                    sa = fma(y.re.x, y.re.x, sa);
                    sa = fma(y.im.x, y.im.x, sa);
                    sb = fma(y.re.y, y.re.y, sb);
                    sb = fma(y.im.y, y.im.y, sb);
                }
                yr[k] = y.re;
                yi[k] = y.im;
            }
            if (hx) {
                cpair_mac<R, R2>(x, xa, vx);
                store_at<XP>(g.X, e, pfma(xm2, mp.re, x.re), pfma(xm2, mp.im, x.im));
            }
        }
        if (act && g.hasY) store_pair<P>(g.Y, n, L.q, yr, yi);
        yn0 += (double)sa;
        yn1 += (double)sb;
    }
    if (g.ynorm) {
        ynred[w][lane] = make_double2(yn0, yn1);
        __syncthreads();
        if (act && w == 0) {
            double2 v = make_double2(0.0, 0.0);
            for (int ww = 0; ww < GW_WARPS; ++ww) {
                v.x += ynred[ww][lane].x;
                v.y += ynred[ww][lane].y;
            }
            g.ynorm[(size_t)chunk * ncols + 2 * L.q] = v.x;
            g.ynorm[(size_t)chunk * ncols + 2 * L.q + 1] = v.y;
        }
    }
}

__global__ void __launch_bounds__(FIN_E * FIN_ROWS) k_norm_finish(const double* __restrict__ part, int nrows, int ncols,
                                                              int c0, int n, double* __restrict__ out) {
    const int j = blockIdx.x * FIN_E + threadIdx.x;
    const bool on = j < n;
    const double2 v = sum_rows(
        nrows, on, [&](int c) { return make_double2(__ldg(part + (size_t)c * ncols + c0 + j), 0.0); });
    if (on && threadIdx.y == 0) {
        out[2 * (c0 + j)] = v.x;
        out[2 * (c0 + j) + 1] = 0.0;
    }
}

// Sums into FP64 by element: a block takes rpb consecutive rows (site,
// component) of np pairs, a thread EL_U of their elements, all loaded before
// the first store.  Memory bounds it.  A thread per (site, pair), holding 12
// components 12 rows apart, kept too few loads in flight (16^3x32 even sites,
// all 60 columns: 704 us, now 528; 6 of 60, where each row's piece is half a
// line: 93, now 83).
constexpr int EL_U = 4, EL_THREADS = 256;
inline unsigned rows_per_block(unsigned rows, int np) {
    return std::max(1u, std::min(EL_U * EL_THREADS / (unsigned)np, rows / 304));
}

// X64 += Xlo (sub: -=) over pairs [p0, p0 + np); zero_lo: then Xlo = 0
__global__ void __launch_bounds__(EL_THREADS) k_accum(Field x64, Field xlo, int p0, int np, int sub, int zero_lo,
                                                      unsigned rows, unsigned rpb) {
    const unsigned r0 = blockIdx.x * rpb, items = min(rpb, rows - r0) * np;
    for (unsigned i0 = threadIdx.x; i0 < items; i0 += EL_U * EL_THREADS) {
        CxPair<double2> x[EL_U];
        CxPair<float2> l[EL_U];
        size_t row[EL_U];
        int q[EL_U];
#pragma unroll
        for (int u = 0; u < EL_U; ++u) {
            const unsigned i = i0 + u * EL_THREADS, r = i / np;
            row[u] = r0 + r;
            q[u] = p0 + (int)(i - r * np);
            if (i < items) {
                x[u] = load_at<BK_FP64>(x64, row[u] * x64.np + q[u]);
                l[u] = load_at<BK_FP32>(xlo, row[u] * xlo.np + q[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < EL_U; ++u) {
            if (i0 + u * EL_THREADS >= items) break;
            const double2 r = f2d(l[u].re), i = f2d(l[u].im);
            store_at<BK_FP64>(x64, row[u] * x64.np + q[u], sub ? psub(x[u].re, r) : padd(x[u].re, r),
                              sub ? psub(x[u].im, i) : padd(x[u].im, i));
            if (zero_lo)
                store_at<BK_FP32>(xlo, row[u] * xlo.np + q[u], make_float2(0.f, 0.f), make_float2(0.f, 0.f));
        }
    }
}

// Seeded Gaussian block: SplitMix64 of (seed, canonical index), Box-Muller.
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
template <int P>
__device__ __forceinline__ void gauss(uint64_t seed, uint64_t idx, typename Prec<P>::real& re,
                                      typename Prec<P>::real& im) {
    const uint64_t a = splitmix64(seed ^ (2 * idx)), b = splitmix64(seed ^ (2 * idx + 1));
    if constexpr (P == BK_FP64) {
        const double u1 = ((a >> 11) + 1) * (1.0 / 9007199254740993.0);
        const double u2 = (b >> 11) * (1.0 / 9007199254740992.0);
        const double rr = sqrt(-log(u1));  // |z| of a complex Gaussian with E|z|^2 = 1
        re = rr * cospi(2 * u2);
        im = rr * sinpi(2 * u2);
    } else {  // a low-precision shadow block needs no FP64 transcendentals
        const float u1 = (float)((a >> 40) + 1) * (1.0f / 16777217.0f);
        const float u2 = (float)(b >> 40) * (1.0f / 16777216.0f);
        const float rr = sqrtf(-logf(u1));
        float sn, cs;
        sincospif(2.0f * u2, &sn, &cs);
        re = rr * cs;
        im = rr * sn;
    }
}
template <int P>
__global__ void k_random(Field f, int L, uint64_t seed) {
    using R2 = typename Prec<P>::pair;
    const int np = (L + 1) / 2;
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (long long)f.V * np) return;
    const int n = (int)(g / np), q = (int)(g - (long long)(g / np) * np);
    R2 vr[12], vi[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = 2 * q + h;
            typename Prec<P>::real re = 0, im = 0;
            if (c < L) gauss<P>(seed, ((uint64_t)c * f.V + n) * 12 + k, re, im);
            if (h == 0) {
                vr[k].x = re;
                vi[k].x = im;
            } else {
                vr[k].y = re;
                vi[k].y = im;
            }
        }
    }
    store_pair<P>(f, n, q, vr, vi);
}

// ---------------------------------------------------------------- small solves

__device__ __forceinline__ cx<double> cdiv(cx<double> a, cx<double> b) {
    const double d = b.r * b.r + b.i * b.i;
    return mk((a.r * b.r + a.i * b.i) / d, (a.i * b.r - a.r * b.i) / d);
}

// ---------------------------------------------------------------- L x L solves: factor, then substitute
//
// k_lu_factor: one thread block per system factors P G = L U (FP64, partial
// pivoting, matrix in shared memory for L <= 96) and stores the factors and
// the pivot rows; info[s] = k + 1 if pivot k is below 1e-14 max|G| or not
// finite.  k_lu_solve: one warp per right-hand-side column computes
// X = G^-1 (scale H) from the factors.

constexpr int LU_THREADS = 256;
constexpr int LU_MAXL_SMEM = 96;

__global__ void __launch_bounds__(LU_THREADS) k_lu_factor(const double2* __restrict__ G, double2* __restrict__ LU,
                                                          int* __restrict__ piv, int* info, SysPart p) {
    extern __shared__ double2 lu_smem_raw[];
    const int s = blockIdx.x;
    if (!((p.active >> s) & 1u)) return;
    const int n = p.L[s];
    const int off = p.coef_off[s];
    cx<double>* A = n <= LU_MAXL_SMEM ? reinterpret_cast<cx<double>*>(lu_smem_raw)
                                      : reinterpret_cast<cx<double>*>(LU) + off;
    __shared__ int pr_s, bad;
    __shared__ double gmax;
    const int tid = threadIdx.x;
    double lmax = 0.0;
    for (int e = tid; e < n * n; e += LU_THREADS) {
        const double2 g = G[off + e];
        A[e] = mk(g.x, g.y);
        lmax = fmax(lmax, fabs(g.x) + fabs(g.y));
        if (!isfinite(g.x) || !isfinite(g.y)) lmax = INFINITY;
    }
    if (tid == 0) {
        gmax = 0.0;
        bad = 0;
    }
    __syncthreads();
    for (int o = 16; o > 0; o >>= 1) lmax = fmax(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
    if ((tid & 31) == 0) atomicMax(reinterpret_cast<unsigned long long*>(&gmax), __double_as_longlong(lmax));
    __syncthreads();
    const double thresh = 1e-14 * gmax;
    if (tid == 0 && !isfinite(gmax)) bad = 1;
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (bad) break;
        if (tid < 32) {
            double best = -1.0;
            int bi = k;
            for (int i = k + tid; i < n; i += 32) {
                const cx<double> v = A[i * n + k];
                const double m = fabs(v.r) + fabs(v.i);
                if (m > best) {
                    best = m;
                    bi = i;
                }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const double ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ob > best || (ob == best && oi < bi)) {
                    best = ob;
                    bi = oi;
                }
            }
            if (tid == 0) {
                pr_s = bi;
                piv[p.col0[s] + k] = bi;
                if (!(best > thresh) || !isfinite(best)) bad = k + 1;
            }
        }
        __syncthreads();
        if (bad) break;
        const int pr = pr_s;
        if (pr != k)
            for (int c = tid; c < n; c += LU_THREADS) {
                const cx<double> t = A[k * n + c];
                A[k * n + c] = A[pr * n + c];
                A[pr * n + c] = t;
            }
        __syncthreads();
        const cx<double> dk = A[k * n + k];
        for (int i = k + 1 + tid; i < n; i += LU_THREADS) A[i * n + k] = cdiv(A[i * n + k], dk);
        __syncthreads();
        const int m = n - k - 1;
        for (int e = tid; e < m * m; e += LU_THREADS) {
            const int i = k + 1 + e / m, j = k + 1 + e % m;
            cx<double> v = A[i * n + j];
            const cx<double> f = A[i * n + k];
            cmac(v, mk(-f.r, -f.i), A[k * n + j]);
            A[i * n + j] = v;
        }
        __syncthreads();
    }
    if (bad) {
        if (tid == 0) info[s] = bad;
        return;
    }
    if (n <= LU_MAXL_SMEM)
        for (int e = tid; e < n * n; e += LU_THREADS) LU[off + e] = make_double2(A[e].r, A[e].i);
}

// grid: (ceil(maxL / 4), nsys); 4 warps per block, one right-hand-side column per warp
__global__ void __launch_bounds__(128) k_lu_solve(const double2* __restrict__ LU, const int* __restrict__ piv,
                                                  const double2* __restrict__ H, const double2* __restrict__ scale,
                                                  double2 hscale, double2* __restrict__ Xs, int* info, SysPart p) {
    const int s = blockIdx.y;
    if (!((p.active >> s) & 1u)) return;
    if (info[s] != 0) return;
    const int n = p.L[s];
    const int j = blockIdx.x * 4 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (j >= n) return;
    const int off = p.coef_off[s];
    const cx<double>* F = reinterpret_cast<const cx<double>*>(LU) + off;
    const int* pv = piv + p.col0[s];
    cx<double> sc = mk(hscale.x, hscale.y);
    if (scale) sc = mk(scale[s].x, scale[s].y);
    // column j of scale * H, rows distributed over the lanes (n <= 4 * 32 handled by 4 slots)
    constexpr int SL = 4;
    cx<double> b[SL];
#pragma unroll
    for (int q = 0; q < SL; ++q) {
        const int i = lane + 32 * q;
        b[q] = mk(0.0, 0.0);
        if (i < n) {
            const double2 h = H[off + i * n + j];
            b[q] = sc * mk(h.x, h.y);
        }
    }
    auto get = [&](int i) -> cx<double> {
        cx<double> v = b[0];
#pragma unroll
        for (int q = 1; q < SL; ++q)
            if (i >= 32 * q) v = b[q];
        const int src = i & 31;
        return mk(__shfl_sync(0xffffffffu, v.r, src), __shfl_sync(0xffffffffu, v.i, src));
    };
    auto put = [&](int i, cx<double> v) {
#pragma unroll
        for (int q = 0; q < SL; ++q)
            if (lane + 32 * q == i) b[q] = v;
    };
    // row interchanges in the order of factorisation
    for (int k = 0; k < n; ++k) {
        const int pk = pv[k];
        if (pk != k) {
            const cx<double> vk = get(k), vp = get(pk);
            put(k, vp);
            put(pk, vk);
        }
    }
    // L y = P b (unit lower triangle)
    for (int k = 0; k < n; ++k) {
        const cx<double> yk = get(k);
#pragma unroll
        for (int q = 0; q < SL; ++q) {
            const int i = lane + 32 * q;
            if (i > k && i < n) {
                const cx<double> l = F[i * n + k];
                cmac(b[q], mk(-l.r, -l.i), yk);
            }
        }
    }
    // U x = y
    for (int k = n - 1; k >= 0; --k) {
        cx<double> xk = cdiv(get(k), F[k * n + k]);
        put(k, xk);
#pragma unroll
        for (int q = 0; q < SL; ++q) {
            const int i = lane + 32 * q;
            if (i < k) {
                const cx<double> u = F[i * n + k];
                cmac(b[q], mk(-u.r, -u.i), xk);
            }
        }
    }
    bool finite = true;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
        const int i = lane + 32 * q;
        if (i < n) {
            Xs[off + i * n + j] = make_double2(b[q].r, b[q].i);
            if (!isfinite(b[q].r) || !isfinite(b[q].i)) finite = false;
        }
    }
    if (!finite) atomicMax(&info[s], n + 1);
}

// ---------------------------------------------------------------- Cholesky basis change
//
// k_chol_inv: one thread block per system.  S = V^H V (Hermitian positive
// definite, FP64) is factored as S = T^H T with T upper triangular, and
// Tinv = T^-1 is written (row-major, zeros below the diagonal).  If S is not
// numerically positive definite, Tinv = identity (the basis is left as it is);
// floor as in bk_kernels.h.

__global__ void __launch_bounds__(256) k_chol_inv(const double2* __restrict__ S, double2* __restrict__ Tinv,
                                                  SysPart p, double shift_rel, double floor) {
    extern __shared__ double2 ch_smem_raw[];
    const int s = blockIdx.x;
    if (!((p.active >> s) & 1u)) return;
    const int n = p.L[s];
    const int off = p.coef_off[s];
    cx<double>* A = reinterpret_cast<cx<double>*>(ch_smem_raw);  // n x n, becomes T (upper)
    cx<double>* X = reinterpret_cast<cx<double>*>(Tinv) + off;   // T^-1, written in place
    __shared__ int bad;
    __shared__ double dmax;
    const int tid = threadIdx.x;
    for (int e = tid; e < n * n; e += blockDim.x) {
        const double2 v = S[off + e];
        A[e] = mk(v.x, v.y);
    }
    __syncthreads();  // the diagonal shift below updates entries other threads loaded
    if (tid == 0) {
        bad = 0;
        dmax = 0.0;
        double tr = 0.0;
        for (int k = 0; k < n; ++k) {
            dmax = fmax(dmax, S[off + k * n + k].x);
            tr += S[off + k * n + k].x;
        }
        // shifted factorisation S + shift_rel trace(S) I (shifted Cholesky QR)
        if (shift_rel > 0.0)
            for (int k = 0; k < n; ++k) A[k * n + k].r += shift_rel * tr;
    }
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (tid == 0) {
            double d = A[k * n + k].r;
            const double low = floor > 0.0 ? floor * n * S[off + k * n + k].x : 1e-14 * dmax;
            if (!(d > low)) {  // with a floor: that, unless the pivot is zero to FP64 rounding
                if (floor > 0.0 && low > 0.0 && fabs(d) > CHOL_EXACT / (floor * n) * low) d = low;
                else bad = 1;
            }
            if (!isfinite(d)) bad = 1;
            else A[k * n + k] = mk(sqrt(d), 0.0);
        }
        __syncthreads();
        if (bad) break;
        const double rd = 1.0 / A[k * n + k].r;
        for (int j = k + 1 + tid; j < n; j += blockDim.x) A[k * n + j] = rd * A[k * n + j];
        __syncthreads();
        const int m = n - k - 1;
        for (int e = tid; e < m * m; e += blockDim.x) {
            const int i = k + 1 + e / m, j = k + 1 + e % m;
            if (j >= i) {
                cx<double> v = A[i * n + j];
                cjmac(v, mk(-A[k * n + i].r, -A[k * n + i].i), A[k * n + j]);  // -= conj(T_ki) T_kj
                A[i * n + j] = v;
            }
        }
        __syncthreads();
    }
    if (bad) {
        for (int e = tid; e < n * n; e += blockDim.x)
            Tinv[off + e] = make_double2((e / n) == (e % n) ? 1.0 : 0.0, 0.0);
        return;
    }
    // T^-1 column by column (back substitution, one thread per column)
    for (int j = tid; j < n; j += blockDim.x) {
        for (int i = n - 1; i >= 0; --i) {
            cx<double> v = mk(i == j ? 1.0 : 0.0, 0.0);
            for (int k = i + 1; k <= j; ++k) cmac(v, mk(-A[i * n + k].r, -A[i * n + k].i), X[k * n + j]);
            X[i * n + j] = i > j ? mk(0.0, 0.0) : (1.0 / A[i * n + i].r) * v;
        }
    }
}

}  // namespace

// ---------------------------------------------------------------- launchers

namespace {

template <int P>
bk_status gram_impl(Field A, Field B, Field B2, int NB, const SysPart& p, double* G, double* G2, double* partial,
                    int nchunk, int V, cudaStream_t st) {
    double2* part = (double2*)partial;
    const int maxL = max_active_L(p);
    if (maxL == 0) return BK_OK;
    const int ne = p.coef_off[p.nsys];
    if (maxL <= ROWS_MAXL) {
        BK_TRY(rows_gram(P, A, B, B2, NB, p, part, nchunk, V, st));
    } else {
        for (int b = 0; b < NB; ++b)
            BK_TRY(wide_gram(P, A, b == 0 ? B : B2, p, part + (size_t)b * nchunk * ne, nchunk, V, st));
    }
    k_gram_finish<<<(NB * ne + FIN_E - 1) / FIN_E, dim3(FIN_E, FIN_ROWS), 0, st>>>(part, nchunk, NB, p, (double2*)G, (double2*)G2);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status gram_dispatch(int prec, Field A, Field B, Field B2, int NB, const SysPart& p, double* G, double* G2,
                        double* partial, int nchunk, int V, cudaStream_t st) {
    switch (prec) {
        case BK_FP64: return gram_impl<BK_FP64>(A, B, B2, NB, p, G, G2, partial, nchunk, V, st);
        case BK_FP32: return gram_impl<BK_FP32>(A, B, B2, NB, p, G, G2, partial, nchunk, V, st);
        case BK_FP16: return gram_impl<BK_FP16>(A, B, B2, NB, p, G, G2, partial, nchunk, V, st);
    }
    return BK_ERR_INVALID_ARG;
}

}  // namespace

// Partial-sum rows a partition may use, whichever of its systems are active: no
// more partial sums than a block has elements.  That binds for wide systems on
// small lattices (4^4, 512 columns: 6 rows and 50 MB; 304 rows of 512^2 sums
// are 2.5 GB).
static int gram_chunk_limit(const SysPart& p, int V) {
    const long long rows = 12LL * V * p.col0[p.nsys] / std::max(1, p.coef_off[p.nsys]);
    return (int)std::max(1LL, std::min<long long>(rows, gram_row_chunks_max(V)));
}

// partial-sum rows of a Gram matrix over the active systems
static int gram_chunks(int prec, const SysPart& p, int V) {
    const int n = max_active_L(p) <= ROWS_MAXL ? gram_row_chunks(prec, V, row_tiles(prec, p)) : wide_gram_chunks(p, V);
    return std::min(n, gram_chunk_limit(p, V));
}

size_t gram_partial_bytes(const SysPart& p, int V) {
    return (size_t)2 * gram_chunk_limit(p, V) * std::max(1, p.coef_off[p.nsys]) * sizeof(double2);
}

bk_status launch_gram(int prec, Field A, Field B, const SysPart& p, double* G, double* partial, int V,
                      cudaStream_t st) {
    return gram_dispatch(prec, A, B, B, 1, p, G, nullptr, partial, gram_chunks(prec, p, V), V, st);
}

bk_status launch_gram2(int prec, Field A, Field B, Field B2, const SysPart& p, double* G, double* G2,
                       double* partial, int V, cudaStream_t st) {
    return gram_dispatch(prec, A, B, B2, 2, p, G, G2, partial, gram_chunks(prec, p, V), V, st);
}

bk_status launch_gram_slots(int prec, Field A, Field B, const SysPart& p, double* G, double* partial,
                            long long slots, int V, cudaStream_t st) {
    const long long ne = p.coef_off[p.nsys];
    if (ne <= 0 || ne > slots) {
        bk_set_error("Gram partial sums need %lld slots per site chunk, %lld available", ne, slots);
        return BK_ERR_INVALID_ARG;
    }
    const int nchunk = (int)std::min<long long>(gram_chunks(prec, p, V), slots / ne);
    return gram_dispatch(prec, A, B, B, 1, p, G, nullptr, partial, nchunk, V, st);
}

// For any range of the L columns: a range of nq pairs takes at most one row
// chunk per 32 rows, and MAX_CHUNKS over its groups of 32 pairs, so at most 64
// MAX_CHUNKS sums in all (one chunk from MAX_CHUNKS groups on).
size_t coldot_partial_bytes(int L, int npair, int V) {
    const size_t cols = 2 * (size_t)npairs(L), chunks = std::max(1, std::min(MAX_CHUNKS, 12 * V / 32));
    return std::max(std::min(chunks * cols, (size_t)64 * MAX_CHUNKS), cols) * npair * sizeof(double2);
}

bk_status launch_coldot(int prec, int npair, const Field* A, const Field* B, int c0, int n, double* out, int ldo,
                        double* partial, int V, cudaStream_t st) {
    if (n <= 0) return BK_OK;
    if (c0 & 1) {
        bk_set_error("column dots start on an even column");
        return BK_ERR_INVALID_ARG;
    }
    // npair 1: A[0]^H B[0]; 2: A[0]^H B[0] and |A[0]|^2 (the only pairs the methods need)
    const bool self = A[0].data == B[0].data;
    if (npair < 1 || npair > 2 || (npair == 2 && (A[1].data != A[0].data || B[1].data != A[0].data))) {
        bk_set_error("unsupported column dots");
        return BK_ERR_INVALID_ARG;
    }
    const int mode = npair == 2 ? 2 : (self ? 1 : 0);
    const int q0 = c0 / 2, nq = (n + 1) / 2;
    double2* part = (double2*)partial;
    // pair slots per block: the smallest of 4, 8, 16, 32 that covers the range
    const int tx = nq <= 4 ? 4 : (nq <= 8 ? 8 : (nq <= 16 ? 16 : 32));
    const unsigned rows = 12u * (unsigned)V;
    // at least 4 rows a thread, at most 2 blocks an SM in all
    const int ngrp = (nq + tx - 1) / tx;
    const int nchunk = (int)std::max(1u, std::min(rows / (256u / tx * 4u), (unsigned)std::max(1, MAX_CHUNKS / ngrp)));
    dim3 grid(ngrp, nchunk);
#define BK_CD1(PP, MD, TX) k_coldot<PP, MD, TX><<<grid, dim3(TX, 256 / TX), 0, st>>>(A[0], B[0], q0, nq, part, rows, nchunk)
#define BK_CD(PP, MD)                       \
    if (tx == 4) BK_CD1(PP, MD, 4);         \
    else if (tx == 8) BK_CD1(PP, MD, 8);    \
    else if (tx == 16) BK_CD1(PP, MD, 16);  \
    else BK_CD1(PP, MD, 32);
#define BK_CDM(PP)                          \
    if (mode == 0) { BK_CD(PP, 0) }         \
    else if (mode == 1) { BK_CD(PP, 1) }    \
    else { BK_CD(PP, 2) }
    switch (prec) {
        case BK_FP64: BK_CDM(BK_FP64) break;
        case BK_FP32: BK_CDM(BK_FP32) break;
        case BK_FP16: BK_CDM(BK_FP16) break;
        default: return BK_ERR_INVALID_ARG;
    }
#undef BK_CDM
#undef BK_CD
#undef BK_CD1
    BK_CUDA_TRY(cudaGetLastError());
    k_coldot_finish<<<(npair * n + FIN_E - 1) / FIN_E, dim3(FIN_E, FIN_ROWS), 0, st>>>(part, nchunk, npair, nq, n,
                                                                         (double2*)out + c0, ldo);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

// grid rows of the updates (a function of the lattice alone: the fused norms
// of a system whose update was skipped stay those of its last residual)
int genop_norm_rows(int V) {
    const int c = std::max(1, (12 * V) / 16);  // 16 rows a block and more
    return c >= 304 ? 304 : (c >= 152 ? 152 : c);  // whole waves of one or two blocks an SM
}

bk_status launch_genop(int prec, const GenOp& g, int V, cudaStream_t st, bool* ynorm_done) {
    if (ynorm_done) *ynorm_done = false;
    const int nchunk = genop_norm_rows(V);
    const int ncols = g.p.col0[g.p.nsys];
    const int maxL = max_active_L(g.p);
    if (maxL == 0) return BK_OK;
    // every operand has the layout's pair count (one element offset serves them all)
    const int np = g.Y.np;
    bool same_np = g.hasY != 0;
    for (int u = 0; u < g.nmi; ++u) same_np &= g.Mi[u].np == np;
    for (int e = 0; e < g.ne; ++e) same_np &= g.E[e].np == np;
    if (g.hasX) same_np &= g.X.np == np && g.Xin.np == np;
    if (!same_np) {
        bk_set_error("block update: an output and operands of one layout expected");
        return BK_ERR_INVALID_ARG;
    }
    if (prec != BK_FP16) {
        BK_TRY(maxL <= ROWS_MAXL ? rows_update(prec, with_units(g), V, nchunk, np, st)
                                 : wide_update(prec, with_units(g), V, nchunk, st));
    } else if (maxL <= ROWS_MAXL) {
        const PTiles wt = make_ptiles(g.p, WT_PAIRS);
        const dim3 grid(wt.n, nchunk);
        const bool h = g.hasX != 0;
#define BK_GW(ML, NM, NE, HX) k_genop_w<ML, NM, NE, HX><<<grid, GW_WARPS * 32, 0, st>>>(g, wt, V, nchunk, ncols, np)
        // the updates of the two methods, then any other combination
#define BK_GWS(ML)                                                \
    if (g.nmi == 1 && g.ne == 0 && !h) BK_GW(ML, 1, 0, 0);        \
    else if (g.nmi == 1 && g.ne == 1 && !h) BK_GW(ML, 1, 1, 0);   \
    else if (g.nmi == 1 && g.ne == 2 && h) BK_GW(ML, 1, 2, 1);    \
    else if (g.nmi == 2 && g.ne == 1 && !h) BK_GW(ML, 2, 1, 0);   \
    else if (g.nmi == 2 && g.ne == 0 && h) BK_GW(ML, 2, 0, 1);    \
    else if (g.nmi == 0 && g.ne == 3 && !h) BK_GW(ML, 0, 3, 0);   \
    else BK_GW(ML, -1, -1, -1);
        if (maxL <= 6) {
            BK_GWS(6)
        } else {
            BK_GWS(12)
        }
#undef BK_GWS
#undef BK_GW
    } else {
        const PTiles tl = make_ptiles(g.p, TILE_MAXP);
        constexpr int SR = 4;
        int widest = 1;
        for (int i = 0; i < tl.n; ++i) widest = std::max(widest, tl.np[i]);
        k_genop<SR><<<dim3(tl.n, nchunk, (widest + TILE_MAXP - 1) / TILE_MAXP), dim3(TILE_MAXP, SR), 0, st>>>(
            g, tl, V, nchunk, ncols);
    }
    BK_CUDA_TRY(cudaGetLastError());
    if (ynorm_done && g.ynorm && g.hasY) *ynorm_done = true;
    return BK_OK;
}

bk_status launch_norm_finish(const double* ynorm, int ncols, int c0, int n, double* out, int V, cudaStream_t st) {
    if (n <= 0) return BK_OK;
    k_norm_finish<<<(n + FIN_E - 1) / FIN_E, dim3(FIN_E, FIN_ROWS), 0, st>>>(ynorm, genop_norm_rows(V), ncols, c0, n, out);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status launch_xmy(int prec, Field X, const double* M, const double* c_dev, Field Z, bool hasZ, Field Y,
                     const SysPart& p, int V, cudaStream_t st) {
    GenOp g;
    memset(&g, 0, sizeof(g));
    g.p = p;
    if (hasZ) {
        g.ne = 1;
        g.E[0] = Z;
        g.ea_mult[0] = 1.0;
    }
    g.nmi = 1;
    g.Mi[0] = X;
    g.ma[0] = c_dev;
    g.ma_mult[0] = 1.0;
    g.M = M;
    g.hasY = 1;
    g.Y = Y;
    g.ym = 1.0;
    return launch_genop(prec, g, V, st);
}

namespace {
bk_status accum(Field X64, Field Xlo, int p0, int np, int sub, int zero_lo, cudaStream_t st) {
    if (np <= 0) return BK_OK;
    const unsigned rows = 12u * (unsigned)X64.V, rpb = rows_per_block(rows, np);
    k_accum<<<(rows + rpb - 1) / rpb, EL_THREADS, 0, st>>>(X64, Xlo, p0, np, sub, zero_lo, rows, rpb);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}
}  // namespace

bk_status launch_accum(Field X64, Field Xlo, int p0, int np, cudaStream_t st) {
    return accum(X64, Xlo, p0, np, 0, 1, st);
}

bk_status launch_sub_lo(Field X64, Field Ylo, int p0, int np, cudaStream_t st) {
    return accum(X64, Ylo, p0, np, 1, 0, st);
}

bk_status launch_random(int prec, Field f, int L, uint64_t seed, cudaStream_t st) {
    const long long items = (long long)f.V * npairs(L);
    const unsigned blocks = (unsigned)((items + 127) / 128);
    switch (prec) {
        case BK_FP64: k_random<BK_FP64><<<blocks, 128, 0, st>>>(f, L, seed); break;
        case BK_FP32: k_random<BK_FP32><<<blocks, 128, 0, st>>>(f, L, seed); break;
        case BK_FP16: k_random<BK_FP16><<<blocks, 128, 0, st>>>(f, L, seed); break;
        default: return BK_ERR_INVALID_ARG;
    }
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status launch_lu_factor(const double* G, double* LU, int* piv, int* info, const SysPart& p, cudaStream_t st) {
    int maxL = 0;
    for (int s = 0; s < p.nsys; ++s) maxL = std::max(maxL, p.L[s]);
    if (maxL > 128) {
        bk_set_error("L x L factorisation supports L <= 128 per system");
        return BK_ERR_INVALID_ARG;
    }
    const int sL = std::min(maxL, LU_MAXL_SMEM);
    const size_t smem = (size_t)sL * sL * sizeof(double2);
    BK_CUDA_TRY(cudaFuncSetAttribute(k_lu_factor, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)((size_t)LU_MAXL_SMEM * LU_MAXL_SMEM * sizeof(double2))));
    BK_CUDA_TRY(cudaMemsetAsync(info, 0, sizeof(int) * p.nsys, st));
    k_lu_factor<<<p.nsys, LU_THREADS, smem, st>>>((const double2*)G, (double2*)LU, piv, info, p);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status launch_lu_solve(const double* LU, const int* piv, const double* H, const double* scale_dev,
                          const double* scale_host, double* Xs, int* info, const SysPart& p, cudaStream_t st) {
    int maxL = 0;
    for (int s = 0; s < p.nsys; ++s) maxL = std::max(maxL, p.L[s]);
    const double2 hs = scale_host ? make_double2(scale_host[0], scale_host[1]) : make_double2(1.0, 0.0);
    dim3 grid((maxL + 3) / 4, p.nsys);
    k_lu_solve<<<grid, 128, 0, st>>>((const double2*)LU, piv, (const double2*)H, (const double2*)scale_dev, hs,
                                     (double2*)Xs, info, p);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status launch_chol_inv(const double* S, double* Tinv, const SysPart& p, cudaStream_t st, double shift_rel,
                          double floor) {
    int maxL = 0;
    for (int s = 0; s < p.nsys; ++s) maxL = std::max(maxL, p.L[s]);
    if (maxL > 118) {
        bk_set_error("basis orthonormalisation supports L <= 118 per system");
        return BK_ERR_INVALID_ARG;
    }
    const size_t smem = (size_t)maxL * maxL * sizeof(double2);
    BK_CUDA_TRY(cudaFuncSetAttribute(k_chol_inv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_chol_inv<<<p.nsys, 256, smem, st>>>((const double2*)S, (double2*)Tinv, p, shift_rel, floor);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

// ---------------------------------------------------------------- no-allocation Gram
//
// bk_block_gram_noalloc: the Gram reduction of bk_block_gram with its
// per-chunk partial sums kept in a fixed, file-scope device array instead of
// library workspace, so the call itself never allocates.  See bkrylov.h.

namespace {

// Partial-sum slots (complex FP64) shared by every bk_block_gram_noalloc call
// in the process: 2 MiB of device memory on every GPU that loads the library.
constexpr int NOALLOC_GRAM_SLOTS = 131072;
static __device__ __align__(256) double2 g_gram_noalloc_scratch[NOALLOC_GRAM_SLOTS];

}  // namespace

extern "C" bk_status bk_block_gram_noalloc(int V, const void* A, const void* B, int L, bk_prec prec, double* G,
                                           void* stream) {
    if (V < 16 || !A || !B || !G || L < 1 || (prec != BK_FP64 && prec != BK_FP32 && prec != BK_FP16)) {
        bk_set_error("bad argument to bk_block_gram_noalloc");
        return BK_ERR_INVALID_ARG;
    }
    // One slot per entry of G and site chunk; at least one chunk must fit.
    // Bounded before any arithmetic in int.
    if (L > 360) {
        bk_set_error("bk_block_gram_noalloc: L = %d needs %lld partial-sum slots, more than the fixed %d "
                     "(L <= 360 fits); use bk_block_gram",
                     L, (long long)L * L, NOALLOC_GRAM_SLOTS);
        return BK_ERR_INVALID_ARG;
    }
    // The array's device address is looked up on every call, with the
    // caller's device current, so that it always belongs to the current
    // context (a cached address would dangle after cudaDeviceReset).  The
    // first lookup on a device loads the library's device code there.
    void* scratch = nullptr;
    {
        cudaError_t e = cudaGetSymbolAddress(&scratch, g_gram_noalloc_scratch);
        if (e != cudaSuccess || !scratch) {
            bk_set_error("bk_block_gram_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
            return BK_ERR_CUDA;
        }
    }
    const SysPart p = single_part(L);
    const Field fa = make_field((void*)A, L, V, prec), fb = make_field((void*)B, L, V, prec);
    return launch_gram_slots(prec, fa, fb, p, G, (double*)scratch, NOALLOC_GRAM_SLOTS, V, (cudaStream_t)stream);
}
