// Block algebra of systems of more than 12 columns (Section 3 of
// arXiv:0903.4936): Gram matrices and fused block updates as register-tiled
// products through shared memory.
//
// A block is a matrix of 12 V rows (site, spinor component) of np column
// pairs.  Both products are bound by the FP32 (FP64) multiply-adds from about
// 24 columns on (4 L flops per byte of an operand), so what counts is how many
// of them a shared-memory read feeds: a thread owns 4 x 4 columns of a Gram
// matrix, or 4 rows x 4 columns of an update, and needs 4 (8) 16-byte reads
// for 32 (64) packed multiply-adds.
//
// 16^3x32, 48 columns, FP32: Gram 887 us and update 845 us; 1930 and 16100
// before, when the update read M and the partner columns through L1 for every
// product (at the FP32 rate each is 370 us).
#include <cstring>

#include "blas_common.cuh"

namespace {

__device__ __forceinline__ void copy16(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// element (row, pair) of f into shared memory: asynchronously for FP32 / FP64,
// with the site's scale applied for FP16
template <int P>
__device__ __forceinline__ void stage_elem(CxPair<typename Prec<P>::pair>* dst, const Field& f, unsigned row, int q) {
    const size_t e = (size_t)row * f.np + q;
    if constexpr (P == BK_FP16) {
        *dst = ldg_at<P>(f, e, pair_scale<P>(f, row / 12, q));
    } else {
        const char* src = (const char*)f.data + e * Prec<P>::ebytes;
        copy16(dst, src);
        if constexpr (P == BK_FP64) copy16((char*)dst + 16, src + 16);
    }
}

// ---------------------------------------------------------------- Gram
//
// A block takes one system (and at most `threads` of its 4 x 4 column tiles)
// and one chunk of rows; `slices` groups of threads share the rows of a stage.
// FP32 sums of at most ROW_FLUSH rows are added to FP64 sums in shared memory.
// The FP64 pipe needs a third of the multiply-adds' time for that, so a thread
// moves a quarter of its sums at a time and goes on multiplying meanwhile.

struct WideWork {
    int n;
    int sys[256];
    int t0[256];  // Gram: first tile; update: pairs of comb a stage
};

template <int P>
__global__ void __launch_bounds__(320, P == BK_FP64 ? 1 : 2) k_gram_t(Field A, Field B, const __grid_constant__ SysPart p,
                                                const __grid_constant__ WideWork w, double2* __restrict__ partial,
                                                unsigned rows, int nchunk, int KR, int half) {
    using R = typename Prec<P>::real;
    using R2 = typename Prec<P>::pair;
    using E = CxPair<R2>;
    extern __shared__ __align__(16) unsigned char wide_smem[];
    const int s = w.sys[blockIdx.x], chunk = blockIdx.y, T = blockDim.x;
    const int Ls = p.L[s], nps = (Ls + 1) / 2, side = (nps + 1) / 2, qs = p.col0[s] / 2;
    const int ntile = min(T, side * side - w.t0[blockIdx.x]), slices = T / ntile;
    const int slice = threadIdx.x / ntile, tile = w.t0[blockIdx.x] + threadIdx.x - slice * ntile;
    const bool on = slice < slices;
    const int ti = tile / side, tj = tile - ti * side;
    // pairs of the tile: ti, ti + side of A and tj, tj + side of B (neighbouring
    // lanes read neighbouring elements)
    const int ia[2] = {ti, min(ti + side, nps - 1)}, jb[2] = {tj, min(tj + side, nps - 1)};
    E* buf = reinterpret_cast<E*>(wide_smem);  // [2][A, B][half]: KR rows of nps elements
    R2 acr[4][2], aci[4][2];  // [column of A][pair of B]
    // FP32 / FP16: the thread's FP64 sums, [entry][thread] {pair}
    double2* sums = reinterpret_cast<double2*>(buf + (size_t)4 * half) + threadIdx.x;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) acr[a][b] = aci[a][b] = pzero<R2>();
    if constexpr (P != BK_FP64)
#pragma unroll
        for (int k = 0; k < 16; ++k) sums[k * T] = make_double2(0.0, 0.0);
    const unsigned per = (rows + nchunk - 1) / nchunk, r0 = (unsigned)chunk * per;
    const unsigned r1 = min(rows, r0 + per);
    const int nst = r0 < r1 ? (int)((r1 - r0 + KR - 1) / KR) : 0;
    // (row, pair) of the thread's elements of a stage, advanced without a division
    const int rr0 = threadIdx.x / nps, q0 = threadIdx.x - rr0 * nps, rstep = T / nps, qstep = T - rstep * nps;
    auto issue = [&](int st) {
        const unsigned b0 = r0 + (unsigned)st * KR;
        E* As = buf + (st & 1) * 2 * half;
        int rr = rr0, q = q0;
        for (int e = threadIdx.x; e < KR * nps; e += T) {
            if (b0 + rr < r1) {
                stage_elem<P>(As + e, A, b0 + rr, qs + q);
                stage_elem<P>(As + half + e, B, b0 + rr, qs + q);
            }
            rr += rstep;
            q += qstep;
            if (q >= nps) {
                q -= nps;
                ++rr;
            }
        }
        copy_commit();
    };
    // row a of the 4 x 4 columns; all of them for a < 0
    auto flush = [&](int row) {
        if constexpr (P != BK_FP64) {
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                if (row >= 0 && a != row) continue;
#pragma unroll
                for (int b = 0; b < 2; ++b)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        float2& v = c ? aci[a][b] : acr[a][b];
                        double2& t = sums[((a * 2 + b) * 2 + c) * T];
                        t = make_double2(t.x + f2d(v.x), t.y + f2d(v.y));
                        v = make_float2(0.f, 0.f);
                    }
            }
        }
    };
    // rows of a stage that a thread takes; a quarter of the sums after every
    // ROW_FLUSH / 4 rows, or all after ROW_FLUSH where a stage is longer than that
    const int per_stage = (KR + slices - 1) / slices;
    const bool quarters = per_stage <= ROW_FLUSH / 4;
    int since = 0, next = 0;
    if (nst > 0) issue(0);
    for (int st = 0; st < nst; ++st) {
        if (st + 1 < nst) {
            issue(st + 1);
            copy_wait<1>();
        } else {
            copy_wait<0>();
        }
        __syncthreads();
        const int nr = (int)min((unsigned)KR, r1 - (r0 + (unsigned)st * KR));
        const E* As = buf + (st & 1) * 2 * half;
        const E* Bs = As + half;
        if (on) {
            const E *pa0 = As + slice * nps + ia[0], *pa1 = As + slice * nps + ia[1];
            const E *pb0 = Bs + slice * nps + jb[0], *pb1 = Bs + slice * nps + jb[1];
            const int step = slices * nps;
#pragma unroll 2
            for (int rr = slice; rr < nr; rr += slices) {
                const E a2[2] = {*pa0, *pa1}, b2[2] = {*pb0, *pb1};
                pa0 += step;
                pa1 += step;
                pb0 += step;
                pb1 += step;
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const R xr = (a & 1) ? a2[a >> 1].re.y : a2[a >> 1].re.x;
                    const R xi = (a & 1) ? a2[a >> 1].im.y : a2[a >> 1].im.x;
                    const R2 ar = bcast(xr), ai = bcast(xi), nai = bcast(-xi);
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        acr[a][b] = pfma(ar, b2[b].re, acr[a][b]);
                        acr[a][b] = pfma(ai, b2[b].im, acr[a][b]);
                        aci[a][b] = pfma(ar, b2[b].im, aci[a][b]);
                        aci[a][b] = pfma(nai, b2[b].re, aci[a][b]);
                    }
                }
            }
            since += per_stage;
            if (P != BK_FP64 && since + per_stage > (quarters ? ROW_FLUSH / 4 : ROW_FLUSH)) {
                flush(quarters ? next : -1);
                next = (next + 1) & 3;
                since = 0;
            }
        }
        __syncthreads();
    }
    flush(-1);
    // slices in FP64 through shared memory, 8 of the 16 entries at a time
    double2* red = reinterpret_cast<double2*>(wide_smem);  // [slice][8][ntile]
    const int ne = p.coef_off[p.nsys], tl = threadIdx.x - slice * ntile;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        __syncthreads();
        if (on)
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    double re, im;
                    if constexpr (P == BK_FP64) {
                        re = y ? acr[a][b].y : acr[a][b].x;
                        im = y ? aci[a][b].y : aci[a][b].x;
                    } else {
                        const double2 r = sums[(a * 2 + b) * 2 * T], i = sums[((a * 2 + b) * 2 + 1) * T];
                        re = y ? r.y : r.x;
                        im = y ? i.y : i.x;
                    }
                    red[((size_t)slice * 8 + 2 * a + y) * ntile + tl] = make_double2(re, im);
                }
        __syncthreads();
        for (int x = threadIdx.x; x < 8 * ntile; x += T) {
            const int k = x / ntile, t = w.t0[blockIdx.x] + x - k * ntile, a = k >> 1, y = k & 1;
            const int i0 = t / side, j0 = t - i0 * side;
            const int i = 2 * (i0 + (a >> 1) * side) + (a & 1), j = 2 * (j0 + b * side) + y;
            if (i >= Ls || j >= Ls) continue;
            double2 v = make_double2(0.0, 0.0);
            for (int sl = 0; sl < slices; ++sl) {
                const double2 z = red[((size_t)sl * 8 + k) * ntile + x - k * ntile];
                v.x += z.x;
                v.y += z.y;
            }
            partial[(size_t)chunk * ne + p.coef_off[s] + i * Ls + j] = v;
        }
    }
}

WideWork wide_work(const SysPart& p, int T) {
    WideWork w;
    w.n = 0;
    for (int s = 0; s < p.nsys; ++s) {
        if (!((p.active >> s) & 1ull)) continue;
        const int nps = (p.L[s] + 1) / 2, side = (nps + 1) / 2;
        for (int t0 = 0; t0 < side * side; t0 += T) {
            if (w.n >= 256) {
                w.n = -1;
                return w;
            }
            w.sys[w.n] = s;
            w.t0[w.n] = t0;
            w.n++;
        }
    }
    return w;
}

// Threads a block: the count, of those whose blocks fit the work list, that
// leaves the fewest threads idle over the launch; then the one with the fewest
// blocks a row chunk, since each of them stages the system's rows for itself.
// A block with few tiles has its rows shared out over slices and ends early.  Up
// to 8 blocks a chunk all blocks are resident at once, so the longest one is the
// launch's time (64 columns: 192 threads take 192 tiles and 64 in three slices,
// 256 take all in one block).
int wide_threads(const SysPart& p) {
    int best = 256, fewest = 1 << 30;
    double most = 0.0;
    for (int T = 192; T <= 320; T += 32) {
        const int n = wide_work(p, T).n;
        if (n <= 0) continue;
        double use = 0.0, sum = 0.0, longest = 0.0;
        for (int s = 0; s < p.nsys; ++s) {
            if (!((p.active >> s) & 1ull)) continue;
            const int nps = (p.L[s] + 1) / 2, side = (nps + 1) / 2;
            for (int t0 = 0; t0 < side * side; t0 += T) {
                const int nt = std::min(T, side * side - t0);
                const double time = 1.0 / (T / nt);  // slices share it
                use += (double)nt / T;               // work in units of full blocks
                sum += time;
                longest = std::max(longest, time);
            }
        }
        const double u = use / (n <= 8 ? n * longest : sum);
        if (u > most + 1e-9 || (u > most - 1e-9 && n < fewest)) {
            most = std::max(most, u);
            best = T;
            fewest = n;
        }
    }
    return best;
}

template <int P>
bk_status wide_gram_p(Field A, Field B, const SysPart& p, double2* partial, int nchunk, int V, cudaStream_t st) {
    const int T = wide_threads(p);
    const WideWork w = wide_work(p, T);
    if (w.n < 0 || wide_work(p, 256).n < 0) {
        bk_set_error("Gram of this partition needs more than 256 thread-block rows");
        return BK_ERR_INVALID_ARG;
    }
    const int maxnps = (max_active_L(p) + 1) / 2;
    const size_t row = (size_t)2 * maxnps * sizeof(CxPair<typename Prec<P>::pair>);
    if (12 * row > (size_t)200 * 1024) {
        bk_set_error("Gram supports systems of at most 512 columns");
        return BK_ERR_INVALID_ARG;
    }
    // rows a stage: two stages in at most 32 KB beside the FP64 sums (FP64: 96 KB), so that two blocks fit
    const size_t lim = (P == BK_FP64 ? 48 : 16) * 1024, sums = P == BK_FP64 ? 0 : (size_t)T * 16 * sizeof(double2);
    const int KR = (int)std::max<size_t>(1, std::min<size_t>(64, lim / row));
    // (the slices' sums overwrite the stages: 128 bytes a thread)
    const size_t stage = std::max((size_t)2 * KR * row, (size_t)T * 8 * sizeof(double2));
    const size_t smem = stage + sums;
    const int half = (int)(stage / 4 / sizeof(CxPair<typename Prec<P>::pair>));
    BK_CUDA_TRY(cudaFuncSetAttribute(k_gram_t<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_gram_t<P><<<dim3(w.n, nchunk), T, smem, st>>>(A, B, p, w, partial, 12u * (unsigned)V, nchunk, KR, half);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

// ---------------------------------------------------------------- fused block update
//
// The update of rows.cu for systems of any size.  A block of 256 threads takes
// (up to UQ pairs of) one system and strides over tiles of rows; thread (rg,
// cg) owns rows rg, rg + nrg, ... (4 of them) and pairs cg, cg + ng.  comb and
// M, rounded to the arithmetic, are staged KC pairs of comb at a time.

constexpr int UT = 256;
constexpr int UQ = 128;

template <int P>
__global__ void __launch_bounds__(UT, P == BK_FP64 ? 1 : 2) k_update_t(const __grid_constant__ GenOp g,
                                                                      const __grid_constant__ WideWork w,
                                                                      unsigned rows, int nchunk, int ncols) {
    using R = typename Prec<P>::real;
    using R2 = typename Prec<P>::pair;
    using E = CxPair<R2>;
    constexpr int NR = 4;
    extern __shared__ __align__(16) unsigned char wide_smem[];
    const int s = w.sys[blockIdx.x], chunk = blockIdx.y;
    if (g.skip && g.skip[s]) return;
    const int Ls = g.p.L[s], nps = (Ls + 1) / 2, qs = g.p.col0[s] / 2;
    const int q0 = blockIdx.z * UQ, wps = min(UQ, nps - q0);  // the block's pairs [q0, q0 + wps)
    if (wps <= 0) return;
    const int ng = (wps + 1) / 2, nrg = UT / ng;
    const int rt = NR * nrg;  // rows of a tile
    const int rg = threadIdx.x / ng, cg = threadIdx.x - rg * ng;
    const bool on = rg < nrg, has1 = cg + ng < wps;
    const int KC = w.t0[blockIdx.x], cstr = KC | 1;  // odd row stride: rows in different banks
    E* Cs = reinterpret_cast<E*>(wide_smem);  // [rt][cstr]
    E* Ms = Cs + (size_t)rt * cstr;           // [2 KC][wps]: {M_i,2q, M_i,2q+1} real parts, imaginary parts
    const bool mat = g.mat != 0, hx = g.hasX != 0;
    cx<R> ea[GENOP_MAXE], ma[GENOP_MAXMI], xa = mk(R(0), R(0));
    int ekind[GENOP_MAXE];
#pragma unroll
    for (int e = 0; e < GENOP_MAXE; ++e) {
        ea[e] = e < g.ne ? coef<P>(g.ea[e], g.ea_mult[e], g.ea_unit[e], s) : mk(R(0), R(0));
        ekind[e] = e < g.ne && g.ea[e] == nullptr ? g.ea_unit[e] : 0;
    }
#pragma unroll
    for (int u = 0; u < GENOP_MAXMI; ++u)
        ma[u] = u < g.nmi ? coef<P>(g.ma[u], g.ma_mult[u], g.ma_unit[u], s) : mk(R(0), R(0));
    const bool m0unit = g.ma[0] == nullptr && g.ma_unit[0] == 1;
    if (hx) xa = coef<P>(g.xa, g.xa_mult, g.xa_unit, s);
    const R2 ym2 = bcast(d2r<R>(g.ym)), xm2 = bcast(d2r<R>(g.xm));
    const double2* M = reinterpret_cast<const double2*>(g.M) + (mat ? g.p.coef_off[s] : 0);
    double2 yn[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
    const unsigned ntile = (rows + rt - 1) / rt;
    bool m_ready = false;  // M stays when all of it fits
    for (unsigned t = chunk; t < ntile; t += nchunk) {
        const unsigned base = t * rt;
        E acc[NR][2];
#pragma unroll
        for (int x = 0; x < NR; ++x) acc[x][0] = acc[x][1] = cp_zero<R2>();
        if (mat)
            for (int k0 = 0; k0 < nps; k0 += KC) {
                const int kn = min(KC, nps - k0);
                __syncthreads();
                constexpr int UE = 4;  // elements loaded before the first is stored
                int rr = threadIdx.x / kn, q = threadIdx.x - rr * kn;
                const int rstep = UT / kn, qstep = UT - rstep * kn;
                for (int e0 = threadIdx.x; e0 < rt * kn; e0 += UE * UT) {
                    E v0[UE], v1[UE];
                    int at[UE];
#pragma unroll
                    for (int z = 0; z < UE; ++z) {
                        const int e = e0 + z * UT;
                        const size_t el = (size_t)(base + rr) * g.Y.np + qs + k0 + q;
                        const bool in = e < rt * kn && base + rr < rows;
                        at[z] = e < rt * kn ? rr * cstr + q : -1;
                        rr += rstep;
                        q += qstep;
                        if (q >= kn) {
                            q -= kn;
                            ++rr;
                        }
                        v0[z] = in ? ldg_at<P>(g.Mi[0], el, bcast(R(1))) : cp_zero<R2>();
                        v1[z] = in && g.nmi > 1 ? ldg_at<P>(g.Mi[1], el, bcast(R(1))) : cp_zero<R2>();
                    }
#pragma unroll
                    for (int z = 0; z < UE; ++z) {
                        if (at[z] < 0) continue;
                        E c = v0[z];
                        if (!m0unit) {
                            c = cp_zero<R2>();
                            cpair_mac<R, R2>(c, ma[0], v0[z]);
                        }
                        if (g.nmi > 1) cpair_mac<R, R2>(c, ma[1], v1[z]);
                        Cs[at[z]] = c;
                    }
                }
                if (!m_ready) {
                    for (int e = threadIdx.x; e < 2 * kn * wps; e += UT) {
                        const int ii = e / wps, j = 2 * (q0 + e - ii * wps), i = 2 * k0 + ii;
                        double2 m0 = make_double2(0.0, 0.0), m1 = m0;
                        if (i < Ls) {
                            m0 = __ldg(M + (size_t)i * Ls + j);
                            if (j + 1 < Ls) m1 = __ldg(M + (size_t)i * Ls + j + 1);
                        }
                        E v;
                        v.re.x = d2r<R>(m0.x);
                        v.re.y = d2r<R>(m1.x);
                        v.im.x = d2r<R>(m0.y);
                        v.im.y = d2r<R>(m1.y);
                        Ms[e] = v;
                    }
                    m_ready = KC == nps;
                }
                __syncthreads();
                if (on) {
                    const E* cp = Cs + rg * cstr;
                    for (int ip = 0; ip < kn; ++ip) {
                        E c[NR];
#pragma unroll
                        for (int x = 0; x < NR; ++x) c[x] = cp[x * nrg * cstr + ip];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const E* mrow = Ms + (2 * ip + h) * wps;
                            const E m0 = mrow[cg], m1 = mrow[has1 ? cg + ng : cg];
#pragma unroll
                            for (int x = 0; x < NR; ++x) {
                                const R xr = h ? c[x].re.y : c[x].re.x, xi = h ? c[x].im.y : c[x].im.x;
                                const R2 cr = bcast(xr), ci = bcast(xi), nci = bcast(-xi);
                                acc[x][0].re = pfma(cr, m0.re, acc[x][0].re);
                                acc[x][0].re = pfma(nci, m0.im, acc[x][0].re);
                                acc[x][0].im = pfma(cr, m0.im, acc[x][0].im);
                                acc[x][0].im = pfma(ci, m0.re, acc[x][0].im);
                                acc[x][1].re = pfma(cr, m1.re, acc[x][1].re);
                                acc[x][1].re = pfma(nci, m1.im, acc[x][1].re);
                                acc[x][1].im = pfma(cr, m1.im, acc[x][1].im);
                                acc[x][1].im = pfma(ci, m1.re, acc[x][1].im);
                            }
                        }
                    }
                }
            }
        if (!on) continue;
        R sq[2][2] = {{R(0), R(0)}, {R(0), R(0)}};
        // each operand's loads before their use
        auto load_all = [&](const Field& f, E (&v)[NR][2], bool plain) {
#pragma unroll
            for (int x = 0; x < NR; ++x)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const unsigned row = base + rg + x * nrg;
                    const size_t el = (size_t)row * g.Y.np + qs + q0 + cg + u * ng;
                    v[x][u] = cp_zero<R2>();
                    if (row < rows && (!u || has1))
                        v[x][u] = plain ? load_at<P>(f, el) : ldg_at<P>(f, el, bcast(R(1)));
                }
        };
        auto store_all = [&](const Field& f, const E (&v)[NR][2]) {
#pragma unroll
            for (int x = 0; x < NR; ++x)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const unsigned row = base + rg + x * nrg;
                    const size_t el = (size_t)row * g.Y.np + qs + q0 + cg + u * ng;
                    if (row < rows && (!u || has1)) store_at<P>(f, el, v[x][u].re, v[x][u].im);
                }
        };
        if (hx) {
            E xv[NR][2], v[NR][2];
            load_all(g.X, xv, true);
            load_all(g.Xin, v, false);
#pragma unroll
            for (int x = 0; x < NR; ++x)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    cpair_mac<R, R2>(xv[x][u], xa, v[x][u]);
                    const E mp = acc[x][u];
                    if (g.x_unit == 1) {
                        xv[x][u].re = padd(xv[x][u].re, mp.re);
                        xv[x][u].im = padd(xv[x][u].im, mp.im);
                    } else {
                        xv[x][u].re = pfma(xm2, mp.re, xv[x][u].re);
                        xv[x][u].im = pfma(xm2, mp.im, xv[x][u].im);
                    }
                }
            store_all(g.X, xv);
        }
        if (g.y_unit != 1) {
#pragma unroll
            for (int x = 0; x < NR; ++x)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    acc[x][u].re = pmul(ym2, acc[x][u].re);
                    acc[x][u].im = pmul(ym2, acc[x][u].im);
                }
        }
#pragma unroll
        for (int e = 0; e < GENOP_MAXE; ++e) {
            if (e >= g.ne) continue;
            E v[NR][2];
            load_all(g.E[e], v, false);
#pragma unroll
            for (int x = 0; x < NR; ++x)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    E& y = acc[x][u];
                    if (ekind[e] == 1) {
                        y.re = padd(y.re, v[x][u].re);
                        y.im = padd(y.im, v[x][u].im);
                    } else if (ekind[e] == -1) {
                        y.re = psub(y.re, v[x][u].re);
                        y.im = psub(y.im, v[x][u].im);
                    } else {
                        cpair_mac<R, R2>(y, ea[e], v[x][u]);
                    }
                }
        }
        if (g.ynorm) {
#pragma unroll
            for (int x = 0; x < NR; ++x)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const E& y = acc[x][u];
                    if (base + rg + x * nrg >= rows || (u && !has1)) continue;
                    sq[u][0] = fma(y.re.x, y.re.x, fma(y.im.x, y.im.x, sq[u][0]));
                    sq[u][1] = fma(y.re.y, y.re.y, fma(y.im.y, y.im.y, sq[u][1]));
                }
        }
        store_all(g.Y, acc);
        if (g.ynorm)
#pragma unroll
            for (int u = 0; u < 2; ++u)
                yn[u] = make_double2(yn[u].x + f2d(sq[u][0]), yn[u].y + f2d(sq[u][1]));
    }
    if (g.ynorm) {
        double2* red = reinterpret_cast<double2*>(wide_smem);  // [2][UT]
        __syncthreads();
        red[threadIdx.x] = yn[0];
        red[UT + threadIdx.x] = yn[1];
        __syncthreads();
        for (int q = threadIdx.x; q < wps; q += UT) {
            double2 v = make_double2(0.0, 0.0);
            const int u = q >= ng;
            for (int r = 0; r < nrg; ++r) {
                const double2 z = red[u * UT + r * ng + q - u * ng];
                v.x += z.x;
                v.y += z.y;
            }
            g.ynorm[(size_t)chunk * ncols + 2 * (qs + q0 + q)] = v.x;
            g.ynorm[(size_t)chunk * ncols + 2 * (qs + q0 + q) + 1] = v.y;
        }
    }
}

template <int P>
bk_status wide_update_p(const GenOp& g, int V, int nchunk, cudaStream_t st) {
    using E = CxPair<typename Prec<P>::pair>;
    WideWork w;
    w.n = 0;
    int maxnps = 0;
    size_t smem = 2 * UT * sizeof(double2);
    for (int s = 0; s < g.p.nsys; ++s) {
        if (!((g.p.active >> s) & 1ull)) continue;
        // pairs of comb a stage: each system's own, the most that fits 80 KB (two
        // blocks an SM).  Not one number for all: a system of 2 pairs takes tiles
        // of 1024 rows and would put the wide ones to one pair a stage.
        const int nps = (g.p.L[s] + 1) / 2;
        int KC = nps;
        size_t need;
        for (;; KC = (KC + 1) / 2) {
            need = 0;
            for (int q0 = 0; q0 < nps; q0 += UQ) {
                const int wps = std::min(UQ, nps - q0), rt = 4 * (UT / ((wps + 1) / 2));
                need = std::max(need, ((size_t)rt * (KC | 1) + (size_t)2 * KC * wps) * sizeof(E));
            }
            if (need <= (size_t)80 * 1024 || KC == 1) break;
        }
        smem = std::max(smem, need);
        maxnps = std::max(maxnps, nps);
        w.sys[w.n] = s;
        w.t0[w.n++] = KC;
    }
    BK_CUDA_TRY(cudaFuncSetAttribute(k_update_t<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_update_t<P><<<dim3(w.n, nchunk, (maxnps + UQ - 1) / UQ), UT, smem, st>>>(g, w, 12u * (unsigned)V, nchunk, g.p.col0[g.p.nsys]);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

}  // namespace

int wide_gram_chunks(const SysPart& p, int V) {
    const WideWork w = wide_work(p, wide_threads(p));
    return std::max(1, std::min(12 * V / 64, std::max(38, 304 / std::max(1, w.n))));
}

bk_status wide_gram(int prec, Field A, Field B, const SysPart& p, double2* partial, int nchunk, int V,
                    cudaStream_t st) {
    switch (prec) {
        case BK_FP64: return wide_gram_p<BK_FP64>(A, B, p, partial, nchunk, V, st);
        case BK_FP32: return wide_gram_p<BK_FP32>(A, B, p, partial, nchunk, V, st);
        case BK_FP16: return wide_gram_p<BK_FP16>(A, B, p, partial, nchunk, V, st);
    }
    return BK_ERR_INVALID_ARG;
}

bk_status wide_update(int prec, const GenOp& g, int V, int nchunk, cudaStream_t st) {
    if (prec == BK_FP64) return wide_update_p<BK_FP64>(g, V, nchunk, st);
    if (prec == BK_FP32) return wide_update_p<BK_FP32>(g, V, nchunk, st);
    return BK_ERR_INVALID_ARG;
}
