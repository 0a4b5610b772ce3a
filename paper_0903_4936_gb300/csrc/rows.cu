// Block algebra of systems of at most 12 columns (Section 3 of
// arXiv:0903.4936): Gram matrices A_s^H B_s and fused block updates.
//
// A block is a matrix of 12 V rows (site, spinor component) of np column
// pairs.  A warp takes a tile, a run of whole systems of tnp <= 32 pairs, and
// 32 / tnp rows at a time: lane (sub, j) holds pair j of row sub, loads only
// that element of each operand (the warp's rows are consecutive, so it reads
// contiguous lines when the tile is the whole block) and gets the other
// columns of its system from their lanes by register shuffles.
//
// Why rows side by side: GB300's FP64 pipe takes 16 cycles per warp
// instruction whatever its active lanes, so a 12-column system that keeps 6
// of 32 lanes busy (one row per warp) wastes four fifths of it; with five
// rows per warp 30 lanes work.  Why rows and not sites: 4^4 has 256 sites but
// 3072 rows, enough for every SM.
#include "blas_common.cuh"

namespace {

constexpr int GW = 8;  // warps per block

// Consecutive row groups a warp takes at a time: up to 12 (a site's rows when
// one row fills the warp), so that the lines its rows share and their DRAM
// pages are used together (16^3x32, 60 columns, even sites, X and R update: 489
// us with single rows strided over the grid, 470 in runs, both with narrow
// tiles); fewer where the groups do not go round.
__device__ __forceinline__ unsigned row_run(unsigned units, unsigned warps) {
    return min(12u, max(1u, units / warps));
}
// The warp's place among all warps: neighbours in a block take neighbouring
// runs; where there are fewer row groups than warps the blocks share them out.
__device__ __forceinline__ unsigned warp_place(unsigned units, int nchunk, int chunk, int w) {
    return units < (unsigned)nchunk * GW ? (unsigned)w * nchunk + chunk : (unsigned)chunk * GW + w;
}

struct RLane {
    bool live;  // the lane holds a pair of an active system
    int sub, q, s, Ls, i0, nps, base;  // row of the group, pair, system, its size, first column, pairs, first lane
};

__device__ __forceinline__ RLane rlane(const SysPart& p, int tp0, int tnp, int lane) {
    RLane w;
    w.sub = lane / tnp;
    w.q = tp0 + lane - w.sub * tnp;
    w.s = sys_of_pair(p, w.q);
    w.live = w.sub < 32 / tnp && ((p.active >> w.s) & 1ull);
    w.Ls = p.L[w.s];
    w.i0 = 2 * w.q - p.col0[w.s];
    w.nps = (w.Ls + 1) / 2;
    w.base = lane - w.i0 / 2;
    if (!w.live) {
        w.nps = 1;
        w.base = lane;
    }
    return w;
}

// ---------------------------------------------------------------- Gram
//
// G_s = A_s^H B_s (NB = 2: and A_s^H B1_s).  A lane adds conj(A_i) B_j for its
// two columns i and every column j of its system.  UR row groups are loaded
// before the first is used.  The block adds its warps' sums at the end and
// writes one partial row per chunk.
//
// FP32 / FP16 products are summed in FP32 registers (packed pairs over j).
// Every ROW_FLUSH rows these go to FP64 accumulators in shared memory.  With
// several rows side by side (spw > 1) a full warp does that for all lanes of a
// column pair, and where the lanes have few rows each (small lattices: 8) it
// adds them in FP32 first, up to ROW_FLUSH rows to a sum: an FP64 add takes 16
// cycles of the SM's FP64 pipe per warp instruction.
// FP64 sums stay in registers and are added over the rows in the tail.

template <int P, int NB, int MAXL, int UR>
__global__ void __launch_bounds__(GW * 32, P == BK_FP64 ? 1 : 2) k_gram_r(Field A, Field B0, Field B1, SysPart p,
                                                                         PTiles wt, double2* __restrict__ partial,
                                                                         unsigned rows, int nchunk) {
    using R2 = typename Prec<P>::pair;
    constexpr int NACC = NB * 2 * MAXL;
    extern __shared__ double2 gr_acc[];  // [warp][NACC * 32]
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int chunk = blockIdx.y;
    const int tp0 = wt.p0[blockIdx.x], tnp = wt.np[blockIdx.x];
    const int spw = 32 / tnp, np = A.np;
    const RLane L = rlane(p, tp0, tnp, lane);
    double2* my = gr_acc + (size_t)w * NACC * 32;
    float2* stage = reinterpret_cast<float2*>(my + NACC * 16);  // spw > 1: accumulators fill at most the first half
    CxPair<R2> acc[NB][2][MAXL / 2];
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int ii = 0; ii < 2; ++ii)
#pragma unroll
            for (int jp = 0; jp < MAXL / 2; ++jp) acc[b][ii][jp] = cp_zero<R2>();
    const unsigned units = (rows + spw - 1) / spw, nw = (unsigned)nchunk * GW;
    const unsigned wid = warp_place(units, nchunk, chunk, w);
    bool first = true;
    int since = 0;
    auto flush = [&]() {
        const bool staged = P != BK_FP64 && spw > 1;
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int ii = 0; ii < 2; ++ii)
#pragma unroll
                for (int jp = 0; jp < MAXL / 2; ++jp) {
                    CxPair<R2>& c = acc[b][ii][jp];
#pragma unroll
                    for (int jj = 0; jj < 2; ++jj) {
                        const int e = (b * 2 + ii) * MAXL + 2 * jp + jj;
                        const auto re = jj ? c.re.y : c.re.x, im = jj ? c.im.y : c.im.x;
                        if (staged) {
                            stage[e * 32 + lane] = make_float2((float)re, (float)im);
                        } else {
                            double2& v = my[e * 32 + lane];
                            if (first) v = make_double2(f2d(re), f2d(im));
                            else v = make_double2(v.x + f2d(re), v.y + f2d(im));
                        }
                    }
                    c = cp_zero<R2>();
                }
        if (staged) {
            const int lanes = ROW_FLUSH / max(since, 1);  // of an FP32 sum
            __syncwarp();
#pragma unroll 1
            for (int x = lane; x < NACC * tnp; x += 32) {
                const int e = x / tnp, pr = x - e * tnp;
                double2 sum = first ? make_double2(0.0, 0.0) : my[x];
#pragma unroll 1
                for (int s0 = 0; s0 < spw; s0 += lanes) {
                    float2 v = stage[e * 32 + s0 * tnp + pr];
                    for (int sub = s0 + 1; sub < min(s0 + lanes, spw); ++sub)
                        v = padd(v, stage[e * 32 + sub * tnp + pr]);
                    if (first && s0 == 0) sum = f2d(v);
                    else sum = make_double2(sum.x + f2d(v.x), sum.y + f2d(v.y));
                }
                my[x] = sum;
            }
            __syncwarp();
        }
        first = false;
        since = 0;
    };
    const unsigned run = row_run(units, nw);
    for (unsigned u1 = wid * run; u1 < units; u1 += nw * run)
    for (unsigned u0 = u1; u0 < min(u1 + run, units); u0 += UR) {
        CxPair<R2> av[UR], bv[UR][NB];
#pragma unroll
        for (int x = 0; x < UR; ++x) {
            const unsigned u = u0 + x, row = u * spw + L.sub;
            av[x] = cp_zero<R2>();
#pragma unroll
            for (int b = 0; b < NB; ++b) bv[x][b] = cp_zero<R2>();
            if (L.live && u < min(u1 + run, units) && row < rows) {
                const size_t e = (size_t)row * np + L.q;
                R2 sa = pzero<R2>(), sb[NB];
#pragma unroll
                for (int b = 0; b < NB; ++b) sb[b] = sa;
                if constexpr (P == BK_FP16) {
                    const int n = row / 12;
                    sa = pair_scale<P>(A, n, L.q);
#pragma unroll
                    for (int b = 0; b < NB; ++b) sb[b] = pair_scale<P>(b == 0 ? B0 : B1, n, L.q);
                }
                av[x] = ldg_at<P>(A, e, sa);
#pragma unroll
                for (int b = 0; b < NB; ++b) bv[x][b] = ldg_at<P>(b == 0 ? B0 : B1, e, sb[b]);
            }
        }
#pragma unroll
        for (int x = 0; x < UR; ++x)
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int jp = 0; jp < MAXL / 2; ++jp) {
                    const CxPair<R2> bp = shfl_pair(bv[x][b], L.base + min(jp, L.nps - 1));
                    if (jp < L.nps) {
#pragma unroll
                        for (int ii = 0; ii < 2; ++ii) {
                            const R2 ar = bcast(ii ? av[x].re.y : av[x].re.x);
                            const R2 ai = bcast(ii ? av[x].im.y : av[x].im.x);
                            const R2 nai = bcast(ii ? -av[x].im.y : -av[x].im.x);
                            CxPair<R2>& c = acc[b][ii][jp];
                            c.re = pfma(ar, bp.re, c.re);
                            c.re = pfma(ai, bp.im, c.re);
                            c.im = pfma(ar, bp.im, c.im);
                            c.im = pfma(nai, bp.re, c.im);
                        }
                    }
                }
        if constexpr (P != BK_FP64) {
            since += UR;
            if (since >= ROW_FLUSH) flush();
        }
    }
    if (wid * run < units && (first || since > 0)) flush();
    __syncthreads();
    // the block's partial sums: one thread per (operand, column of the pair, column, pair)
    const int ne = p.coef_off[p.nsys];
    int nact = 0;  // warps with rows (the first of the block)
    while (nact < GW && warp_place(units, nchunk, chunk, nact) * run < units) ++nact;
    const int estr = P == BK_FP64 || spw == 1 ? 32 : tnp, nsub = P == BK_FP64 ? spw : 1;
    for (int x = threadIdx.x; x < tnp * NACC; x += GW * 32) {
        const int e = x / tnp, pr = x - e * tnp, j = e % MAXL, ii = (e / MAXL) & 1, b = e / (2 * MAXL);
        const int s = sys_of_pair(p, tp0 + pr), Ls = p.L[s], i = 2 * (tp0 + pr) - p.col0[s] + ii;
        if (i >= Ls || j >= Ls || !((p.active >> s) & 1ull)) continue;
        double2 v = make_double2(0.0, 0.0);
        for (int ww = 0; ww < nact; ++ww)
            for (int sub = 0; sub < nsub; ++sub) {
                const double2 a = gr_acc[(size_t)ww * NACC * 32 + e * estr + sub * tnp + pr];
                v.x += a.x;
                v.y += a.y;
            }
        partial[(size_t)(b * nchunk + chunk) * ne + p.coef_off[s] + i * Ls + j] = v;
    }
}

template <int P, int NB, int MAXL, int UR>
bk_status run_gram_r(Field A, Field B0, Field B1, const SysPart& p, const PTiles& wt, double2* part, int nchunk, int V,
                     cudaStream_t st) {
    const size_t smem = (size_t)GW * NB * 2 * MAXL * 32 * sizeof(double2);
    BK_CUDA_TRY(cudaFuncSetAttribute(k_gram_r<P, NB, MAXL, UR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
    k_gram_r<P, NB, MAXL, UR><<<dim3(wt.n, nchunk), GW * 32, smem, st>>>(A, B0, B1, p, wt, part, 12u * (unsigned)V,
                                                                         nchunk);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

template <int P>
bk_status rows_gram_p(Field A, Field B, Field B2, int NB, const SysPart& p, double2* part, int nchunk, int V,
                      cudaStream_t st) {
    const PTiles wt = row_tiles(P, p);
    const int maxL = max_active_L(p);
    const int ne = p.coef_off[p.nsys];
    constexpr int UR = P == BK_FP64 ? 2 : 4;
    // two operands: 3 row groups (16^3x32 even sites, 60 columns: 4 groups spill 74 bytes and take 320 us, 3 take
    // 238, 2 take 260; the three blocks once are 167 us of memory time)
    if (NB == 2 && maxL <= 6) return run_gram_r<P, 2, 6, P == BK_FP64 ? 2 : 3>(A, B, B2, p, wt, part, nchunk, V, st);
    for (int b = 0; b < NB; ++b) {
        Field Bb = b == 0 ? B : B2;
        double2* pb = part + (size_t)b * nchunk * ne;
        if (maxL <= 6) BK_TRY((run_gram_r<P, 1, 6, UR>(A, Bb, Bb, p, wt, pb, nchunk, V, st)));
        else BK_TRY((run_gram_r<P, 1, 12, P == BK_FP64 ? 1 : 2>(A, Bb, Bb, p, wt, pb, nchunk, V, st)));
    }
    return BK_OK;
}

// ---------------------------------------------------------------- fused block update
//
//   matpart_j = sum_{i in s} comb_i M_s[i][j],   comb = sum_u ma_u Mi_u
//   Y_j       = sum_t ea_t E_t,j + ym matpart_j
//   X_j      += xa Xin_j + xm matpart_j          (X in FP64 for FP64 blocks, else FP32)
//
// A lane keeps its two columns of M in registers (with one Mi operand its
// coefficient is multiplied into them, in FP64), forms comb for its own pair,
// takes its system's other pairs by shuffles, and writes its pair of Y and X.
// UR row groups are loaded before any of their arithmetic and stores.  NMI,
// NE and HX fix the operand counts of the solvers' updates at compile time.
// Unit coefficients cost nothing (FP64 instructions are what bounds the FP64
// updates of wide systems; memory bounds the FP32 ones).

// FP64 coefficients times their factor: a call, so that the FP32 kernels that
// need no FP64 arithmetic do none (8^3x16, 12 columns: with the conversions and
// signs of M in the FP64 pipe it was 40 to 53 % busy, 13 to 18 us an update)
__device__ __noinline__ void scale_coefs(const GenOp& g, int s, cx<double>& m0, cx<double>& m1) {
    const cx<double> f = coef<BK_FP64>(g.ma[0], g.ma_mult[0], g.ma_unit[0], s);
    m0 = f * m0;
    m1 = f * m1;
}
// sign flipped by its bit
__device__ __forceinline__ float flip(float v, bool neg) {
    return __int_as_float(__float_as_int(v) ^ (neg ? 0x80000000 : 0));
}
__device__ __forceinline__ double flip(double v, bool neg) {
    return __hiloint2double(__double2hiint(v) ^ (neg ? 0x80000000 : 0), __double2loint(v));
}

template <int P, int MAXL, int UR, int MINB, int NMI, int NE, int HX>
__global__ void __launch_bounds__(GW * 32, MINB) k_update_r(const __grid_constant__ GenOp g,
                                                            const __grid_constant__ PTiles wt, unsigned rows,
                                                            int nchunk, int ncols, int np) {
    using R = typename Prec<P>::real;
    using R2 = typename Prec<P>::pair;
    constexpr int MMI = NMI >= 0 ? NMI : GENOP_MAXMI;
    constexpr int ME = NE >= 0 ? NE : GENOP_MAXE;
    const int nmi = NMI >= 0 ? NMI : g.nmi;
    const int ne = NE >= 0 ? NE : g.ne;
    const bool hx = HX >= 0 ? HX != 0 : g.hasX != 0;
    __shared__ double2 ynred[GW][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int chunk = blockIdx.y;
    const int tp0 = wt.p0[blockIdx.x], tnp = wt.np[blockIdx.x];
    const int spw = 32 / tnp;
    const unsigned units = (rows + spw - 1) / spw, nw = (unsigned)nchunk * GW;
    const unsigned wid = warp_place(units, nchunk, chunk, w);
    if (wid >= units && !g.ynorm) return;
    const RLane L = rlane(g.p, tp0, tnp, lane);
    const bool act = L.live && !(g.skip && g.skip[L.s]);
    const int s = L.s;
    const bool mat = g.mat != 0;
    cx<R> ea[ME > 0 ? ME : 1], ma[MMI > 0 ? MMI : 1], xa = mk(R(0), R(0));
    int ekind[ME > 0 ? ME : 1];  // coefficient of E_t: 1, -1 (adds) or general
#pragma unroll
    for (int e = 0; e < ME; ++e) {
        ea[e] = e < ne ? coef<P>(g.ea[e], g.ea_mult[e], g.ea_unit[e], s) : mk(R(0), R(0));
        ekind[e] = e < ne && g.ea[e] == nullptr ? g.ea_unit[e] : 0;
    }
#pragma unroll
    for (int u = 0; u < MMI; ++u) ma[u] = u < nmi ? coef<P>(g.ma[u], g.ma_mult[u], g.ma_unit[u], s) : mk(R(0), R(0));
    const bool munit = nmi == 1 || (g.ma[0] == nullptr && g.ma_unit[0] == 1);
    if (hx) xa = coef<P>(g.xa, g.xa_mult, g.xa_unit, s);
    // the lane's two columns of M; rows and columns past the system's size are zero
    R2 Mr[MAXL], Mi[MAXL];
    {
        const double2* M = reinterpret_cast<const double2*>(g.M) + (act && mat ? g.p.coef_off[s] : 0);
        const bool j1ok = L.i0 + 1 < L.Ls;
        // one operand: its coefficient goes into M; 1 and -1 without FP64 arithmetic
        const int unit = nmi != 1 || !mat ? 1 : (g.ma[0] ? 0 : g.ma_unit[0]);
        const bool neg = unit < 0;
#pragma unroll
        for (int i = 0; i < MAXL; ++i) {
            cx<double> m0 = mk(0.0, 0.0), m1 = mk(0.0, 0.0);
            if (act && mat && i < L.Ls) {
                const double2 a = __ldg(M + i * L.Ls + L.i0);
                m0 = mk(a.x, a.y);
                if (j1ok) {
                    const double2 b = __ldg(M + i * L.Ls + L.i0 + 1);
                    m1 = mk(b.x, b.y);
                }
                if (unit == 0) scale_coefs(g, s, m0, m1);
            }
            Mr[i].x = flip(d2r<R>(m0.r), neg);
            Mr[i].y = flip(d2r<R>(m1.r), neg);
            Mi[i].x = flip(d2r<R>(m0.i), neg);
            Mi[i].y = flip(d2r<R>(m1.i), neg);
        }
    }
    const bool yunit = g.y_unit == 1, xunit = g.x_unit == 1;
    const R2 ym2 = bcast(d2r<R>(g.ym)), xm2 = bcast(d2r<R>(g.xm));
    double yn0 = 0.0, yn1 = 0.0;
    R sa = R(0), sb = R(0);
    int since = 0;
    const CxPair<R2> zero = cp_zero<R2>();
    constexpr int XP = P;  // X accumulates in the block's precision (FP32 or FP64)
    const unsigned run = row_run(units, nw);
    for (unsigned u1 = wid * run; u1 < units; u1 += nw * run)
    for (unsigned u0 = u1; u0 < min(u1 + run, units); u0 += UR) {
        CxPair<R2> vm[UR][MMI > 0 ? MMI : 1], ve[UR][ME > 0 ? ME : 1], vx[UR], xo[UR];
        bool on[UR];
        size_t ee[UR];
#pragma unroll
        for (int x = 0; x < UR; ++x) {
            const unsigned u = u0 + x, row = u * spw + L.sub;
            on[x] = act && u < min(u1 + run, units) && row < rows;
            ee[x] = (size_t)row * np + L.q;
            const R2 one = bcast(R(1));
#pragma unroll
            for (int m = 0; m < MMI; ++m)
                vm[x][m] = on[x] && mat && m < nmi ? ldg_at<P>(g.Mi[m], ee[x], one) : zero;
#pragma unroll
            for (int t = 0; t < ME; ++t) ve[x][t] = on[x] && g.hasY && t < ne ? ldg_at<P>(g.E[t], ee[x], one) : zero;
            vx[x] = xo[x] = zero;
            if (on[x] && hx) {
                vx[x] = ldg_at<P>(g.Xin, ee[x], one);
                xo[x] = load_at<XP>(g.X, ee[x]);
            }
        }
#pragma unroll
        for (int x = 0; x < UR; ++x) {
            CxPair<R2> mp = zero;
            if (mat) {
                CxPair<R2> c = zero;
                if (munit) c = vm[x][0];
                else cpair_mac<R, R2>(c, ma[0], vm[x][0]);
#pragma unroll
                for (int m = 1; m < MMI; ++m)
                    if (m < nmi) cpair_mac<R, R2>(c, ma[m], vm[x][m]);
#pragma unroll
                for (int ip = 0; ip < MAXL / 2; ++ip) {
                    const CxPair<R2> cp = shfl_pair(c, L.base + min(ip, L.nps - 1));
                    if (ip < L.nps) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const R2 cr = bcast(h ? cp.re.y : cp.re.x), ci = bcast(h ? cp.im.y : cp.im.x);
                            const R2 nci = bcast(h ? -cp.im.y : -cp.im.x);
                            if (ip == 0 && h == 0) {
                                mp.re = pmul(cr, Mr[0]);
                                mp.im = pmul(cr, Mi[0]);
                            } else {
                                mp.re = pfma(cr, Mr[2 * ip + h], mp.re);
                                mp.im = pfma(cr, Mi[2 * ip + h], mp.im);
                            }
                            mp.re = pfma(nci, Mi[2 * ip + h], mp.re);
                            mp.im = pfma(ci, Mr[2 * ip + h], mp.im);
                        }
                    }
                }
            }
            if (!on[x]) continue;
            if (g.hasY) {
                CxPair<R2> y = mp;
                if (!yunit) {
                    y.re = pmul(ym2, mp.re);
                    y.im = pmul(ym2, mp.im);
                }
#pragma unroll
                for (int t = 0; t < ME; ++t)
                    if (t < ne) {
                        if (t == 0 && !mat && ekind[0] == 1) {
                            y = ve[x][0];
                        } else if (ekind[t] == 1) {
                            y.re = padd(y.re, ve[x][t].re);
                            y.im = padd(y.im, ve[x][t].im);
                        } else if (ekind[t] == -1) {
                            y.re = psub(y.re, ve[x][t].re);
                            y.im = psub(y.im, ve[x][t].im);
                        } else {
                            cpair_mac<R, R2>(y, ea[t], ve[x][t]);
                        }
                    }
                if (g.ynorm) {
                    sa = fma(y.re.x, y.re.x, sa);
                    sa = fma(y.im.x, y.im.x, sa);
                    sb = fma(y.re.y, y.re.y, sb);
                    sb = fma(y.im.y, y.im.y, sb);
                }
                store_at<P>(g.Y, ee[x], y.re, y.im);
            }
            if (hx) {
                CxPair<R2> v = xo[x];
                cpair_mac<R, R2>(v, xa, vx[x]);
                if (xunit) {
                    v.re = padd(v.re, mp.re);
                    v.im = padd(v.im, mp.im);
                } else {
                    v.re = pfma(xm2, mp.re, v.re);
                    v.im = pfma(xm2, mp.im, v.im);
                }
                store_at<XP>(g.X, ee[x], v.re, v.im);
            }
        }
        // FP32 squares of at most 12 rows per FP32 sum, then FP64
        since += UR;
        if (g.ynorm && since >= 12) {
            yn0 += f2d(sa);
            yn1 += f2d(sb);
            sa = sb = R(0);
            since = 0;
        }
    }
    if (g.ynorm) {
        // rows of a column pair: first within each warp, then over the warps (an
        // FP64 add of one warp takes 64 cycles, so few of them in a row)
        ynred[w][lane] = make_double2(yn0 + f2d(sa), yn1 + f2d(sb));
        __syncwarp();
        if (lane < tnp) {
            double2 v = ynred[w][lane];
            for (int sub = 1; sub < spw; ++sub) {
                v.x += ynred[w][sub * tnp + lane].x;
                v.y += ynred[w][sub * tnp + lane].y;
            }
            ynred[w][lane] = v;
        }
        __syncthreads();
        if (act && threadIdx.x < tnp) {
            double2 v = ynred[0][lane];
            for (int ww = 1; ww < GW; ++ww) {
                v.x += ynred[ww][lane].x;
                v.y += ynred[ww][lane].y;
            }
            g.ynorm[(size_t)chunk * ncols + 2 * L.q] = v.x;
            g.ynorm[(size_t)chunk * ncols + 2 * L.q + 1] = v.y;
        }
    }
}

}  // namespace

// Tiles of the row kernels: runs of whole systems, with inactive ones between
// active ones where that saves a tile.  FP32 / FP16: the widest that fit a
// warp, since memory bounds them and a narrow tile reads scattered pieces of
// the rows (16^3x32 even sites, ten systems of 6 columns, X and R update: six
// tiles of 5 pairs 594 us, one of 30 pairs 350; with one system in the middle
// inactive, two tiles 600 us, one over the gap 357).  FP64: the width
// that keeps the most lanes busy (a tile of tnp pairs costs 1 / floor(32 /
// tnp) of a warp step per row; the widest of the cheapest splittings).
PTiles row_tiles(int prec, const SysPart& p) {
    PTiles best = join_ptiles(make_ptiles(p, 32), 32);
    if (prec != BK_FP64) return best;
    double cost = 1e30;
    for (int maxp = 32; maxp >= ROWS_MAXL / 2; --maxp) {
        const PTiles t = join_ptiles(make_ptiles(p, maxp), maxp);
        double c = 0.0;
        for (int i = 0; i < t.n; ++i) c += 1.0 / (32 / t.np[i]);
        if (c < cost - 1e-9) {
            cost = c;
            best = t;
        }
    }
    return best;
}

bk_status rows_gram(int prec, Field A, Field B, Field B2, int NB, const SysPart& p, double2* partial, int nchunk,
                    int V, cudaStream_t st) {
    switch (prec) {
        case BK_FP64: return rows_gram_p<BK_FP64>(A, B, B2, NB, p, partial, nchunk, V, st);
        case BK_FP32: return rows_gram_p<BK_FP32>(A, B, B2, NB, p, partial, nchunk, V, st);
        case BK_FP16: return rows_gram_p<BK_FP16>(A, B, B2, NB, p, partial, nchunk, V, st);
    }
    return BK_ERR_INVALID_ARG;
}

bk_status rows_update(int prec, const GenOp& g, int V, int nchunk, int np, cudaStream_t st) {
    const PTiles wt = row_tiles(prec, g.p);
    const dim3 grid(wt.n, nchunk);
    const int ncols = g.p.col0[g.p.nsys];
    const unsigned rows = 12u * (unsigned)V;
    const bool h = g.hasX != 0;
    const int maxL = max_active_L(g.p);
#define BK_UR(PP, ML, UR, MB, NM, NE, HX) \
    k_update_r<PP, ML, UR, MB, NM, NE, HX><<<grid, GW * 32, 0, st>>>(g, wt, rows, nchunk, ncols, np)
    // the updates of the two methods, then any other combination
#define BK_URS(PP, ML, U, MB)                                                         \
    if (g.nmi == 1 && g.ne == 0 && !h) BK_UR(PP, ML, U, MB, 1, 0, 0);                 \
    else if (g.nmi == 1 && g.ne == 1 && !h) BK_UR(PP, ML, U, MB, 1, 1, 0);            \
    else if (g.nmi == 1 && g.ne == 2 && h) BK_UR(PP, ML, U, MB, 1, 2, 1);             \
    else if (g.nmi == 2 && g.ne == 1 && !h) BK_UR(PP, ML, U, MB, 2, 1, 0);            \
    else if (g.nmi == 2 && g.ne == 0 && h) BK_UR(PP, ML, U, MB, 2, 0, 1);             \
    else if (g.nmi == 0 && g.ne == 3 && !h) BK_UR(PP, ML, U, MB, 0, 3, 0);            \
    else BK_UR(PP, ML, 1, 1, -1, -1, -1);
    if (prec == BK_FP64) {
        if (maxL <= 6) {
            BK_URS(BK_FP64, 6, 1, 2)
        } else {
            BK_URS(BK_FP64, 12, 1, 1)
        }
    } else if (prec == BK_FP32) {
        if (maxL <= 6) {
            BK_URS(BK_FP32, 6, 2, 2)
        } else {
            BK_URS(BK_FP32, 12, 2, 2)
        }
    } else {
        return BK_ERR_INVALID_ARG;
    }
#undef BK_URS
#undef BK_UR
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}
