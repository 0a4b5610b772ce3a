// The L x L steps of both methods for systems of at most 12 columns: LU with
// partial pivoting and its right-hand side in one pass, later right-hand sides
// with the stored factors, the scalars zeta of the iteration, and the Cholesky
// basis change.  FP64.
//
// One block of four warps per system, the augmented matrix [G | H] in shared
// memory.  Each of an SM's four schedulers starts one FP64 warp instruction in
// 64 cycles, whatever its active lanes, so the cost is the number of dependent
// FP64 instructions: an elimination step spreads its elements over the 128
// threads, divides once (by the pivot; U keeps a unit diagonal) and compares
// magnitudes as integers.  The general kernels (blas.cu) take 29 + 31 us for a
// 12 x 12 factorisation and solve in two launches, k_small_step 22 us for both
// (6 x 6: 11); larger systems use them.
#include "blas_common.cuh"

namespace {

typedef unsigned long long u64;

constexpr int NT = 128;  // worker threads; one more warp forms the scalars

// barrier of the worker threads
__device__ __forceinline__ void bar() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }

// a - b c
__device__ __forceinline__ cx<double> cnmac(cx<double> a, cx<double> b, cx<double> c) {
    a.r = fma(-b.r, c.r, a.r);
    a.i = fma(-b.r, c.i, a.i);
    a.r = fma(b.i, c.i, a.r);
    a.i = fma(-b.i, c.r, a.i);
    return a;
}
// bits of a non-negative double: ordered like the value, NaN above infinity
__device__ __forceinline__ u64 mag_bits(cx<double> v) {
    return (u64)__double_as_longlong(fabs(v.r) + fabs(v.i));
}
constexpr u64 INF_BITS = 0x7ff0000000000000ull;

// zeta = sum_j d0_j / sum_j d1_j, its negative and its inverse; zbad = 1 when
// zeta is not finite or zero.  dots: d0 at [j], d1 (real) at [Lt + j].
__device__ void zeta_warp(const SmallStep& a, int s, int lane) {
    const double2* dots = reinterpret_cast<const double2*>(a.dots);
    const int j = a.p.col0[s] + lane;
    double2 num = make_double2(0.0, 0.0);
    double den = 0.0;
    if (lane < a.p.L[s]) {
        num = dots[j];
        den = dots[a.Lt + j].x;
    }
    for (int o = 8; o > 0; o >>= 1) {
        num.x += __shfl_xor_sync(0xffffffffu, num.x, o);
        num.y += __shfl_xor_sync(0xffffffffu, num.y, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    if (lane != 0) return;
    const double zr = num.x / den, zi = num.y / den;
    const double m = zr * zr + zi * zi;
    reinterpret_cast<double2*>(a.zeta)[s] = make_double2(zr, zi);
    reinterpret_cast<double2*>(a.mzeta)[s] = make_double2(-zr, -zi);
    reinterpret_cast<double2*>(a.izeta)[s] = make_double2(zr / m, -zi / m);
    a.zbad[s] = (isfinite(zr) && isfinite(zi) && m > 0.0) ? 0 : 1;
}

// scale_s * H into columns [c0, c0 + n) of A (row stride W)
template <int W>
__device__ __forceinline__ void load_rhs(const SmallStep& a, int s, int n, cx<double>* A, int c0) {
    const double2* H = reinterpret_cast<const double2*>(a.H) + a.p.coef_off[s];
    const cx<double> sc = a.hs_dev ? mk(a.hs_dev[2 * s], a.hs_dev[2 * s + 1]) : mk(1.0, 0.0);
    for (int e = threadIdx.x; e < n * n; e += NT) {
        const int i = e / n, j = e - i * n;
        const double2 h = H[e];
        cx<double> v = mk(h.x, h.y);
        if (a.hs_dev) v = sc * v;
        else if (a.hs_neg) v = mk(-h.x, -h.y);
        A[i * W + c0 + j] = v;
    }
}

// columns [c0, c0 + n) of A to X; *bad is set when an entry is not finite
template <int W>
__device__ __forceinline__ void store_rhs(const SmallStep& a, int s, int n, const cx<double>* A, int c0, int* bad) {
    double2* X = reinterpret_cast<double2*>(a.X) + a.p.coef_off[s];
    for (int e = threadIdx.x; e < n * n; e += NT) {
        const int i = e / n, j = e - i * n;
        const cx<double> v = A[i * W + c0 + j];
        X[e] = make_double2(v.r, v.i);
        if (!isfinite(v.r) || !isfinite(v.i)) *bad = 1;
    }
    bar();
}

// U x = y with U's unit upper triangle in columns [0, n) of A
template <int W>
__device__ __forceinline__ void back_substitute(int n, cx<double>* A, const cx<double>* F, int FW, int c0) {
    for (int k = n - 1; k > 0; --k) {
        for (int e = threadIdx.x; e < k * n; e += NT) {
            const int i = e / n, j = c0 + e - i * n;
            A[i * W + j] = cnmac(A[i * W + j], F[i * FW + k], A[k * W + j]);
        }
        bar();
    }
}

// P G = L U by columns: L keeps the pivots (their reciprocals are stored on
// the diagonal), U has a unit diagonal; the right-hand side goes through the
// same steps.
template <int N>
__device__ void factor_block(const SmallStep& a, int s, cx<double>* A, u64* gmax, int* bad) {
    constexpr int W = 2 * N;
    const int n = a.p.L[s], off = a.p.coef_off[s], tid = threadIdx.x, lane = tid & 31;
    const int w = 2 * n;  // columns in use
    u64 gm = 0;
    for (int e = tid; e < n * n; e += NT) {
        const double2 g = reinterpret_cast<const double2*>(a.G)[off + e];
        const cx<double> v = mk(g.x, g.y);
        A[(e / n) * W + e % n] = v;
        gm = max(gm, mag_bits(v));
    }
    load_rhs<W>(a, s, n, A, n);
    for (int o = 16; o > 0; o >>= 1) gm = max(gm, __shfl_xor_sync(0xffffffffu, gm, o));
    if (lane == 0) atomicMax(gmax, gm);
    bar();
    gm = *gmax;
    int info = gm < INF_BITS ? 0 : 1;
    const u64 thresh = (u64)__double_as_longlong(1e-14 * __longlong_as_double((long long)gm));
    int* piv = a.piv + a.p.col0[s];
    for (int k = 0; k < n && !info; ++k) {
        if (tid < 32) {
            // pivot: the largest entry of column k (the four low bits of the
            // magnitude make room for its row)
            u64 best = 0;
            if (tid >= k && tid < n) best = (mag_bits(A[tid * W + k]) & ~15ull) | (u64)(15 - tid);
            for (int o = 8; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o, 16));
            best = __shfl_sync(0xffffffffu, best, 0);
            const int pr = 15 - (int)(best & 15ull);
            best &= ~15ull;
            if (best >= INF_BITS || best <= thresh) {
                if (tid == 0) *bad = k + 1;
            } else {
                // rows k and pr change places, row k divided by the pivot right of the diagonal
                const cx<double> d = A[pr * W + k];
                cx<double> p = mk(0.0, 0.0), t = p;
                if (tid < w) {
                    p = A[pr * W + tid];
                    t = A[k * W + tid];
                }
                const double r = 1.0 / fma(d.r, d.r, d.i * d.i);
                const cx<double> inv = mk(d.r * r, -d.i * r);
                cx<double> q = p * inv;
                if (tid < k) q = p;
                if (tid == k) q = inv;
                __syncwarp();
                if (tid < w) {
                    if (pr != k) A[pr * W + tid] = t;
                    A[k * W + tid] = q;
                }
                if (tid == 0) piv[k] = pr;
            }
        }
        bar();
        if ((info = *bad)) break;
        const int m = w - k - 1;
        for (int e = tid; e < (n - k - 1) * m; e += NT) {
            const int i = k + 1 + e / m, j = k + 1 + e % m;
            A[i * W + j] = cnmac(A[i * W + j], A[i * W + k], A[k * W + j]);
        }
        bar();
    }
    if (!info) {
        for (int e = tid; e < n * n; e += NT) {
            const cx<double> v = A[(e / n) * W + e % n];
            reinterpret_cast<double2*>(a.LU)[off + e] = make_double2(v.r, v.i);
        }
        back_substitute<W>(n, A, A, W, n);
        store_rhs<W>(a, s, n, A, n, bad);
        if (*bad) info = n + 1;
    }
    if (tid == 0) a.info[s] = info;
}

// X = G^-1 (scale H) with the factors of factor_block
template <int N>
__device__ void resolve_block(const SmallStep& a, int s, cx<double>* A, int* bad) {
    constexpr int W = 2 * N;
    const int n = a.p.L[s], off = a.p.coef_off[s], tid = threadIdx.x;
    int info = a.info_in[s];
    if (!info) {
        const int* piv = a.piv + a.p.col0[s];
        for (int e = tid; e < n * n; e += NT) {
            const double2 f = reinterpret_cast<const double2*>(a.LU)[off + e];
            A[(e / n) * W + e % n] = mk(f.x, f.y);
        }
        load_rhs<W>(a, s, n, A, n);
        bar();
        if (tid < n)
            for (int k = 0; k < n; ++k) {
                const int pr = piv[k];
                if (pr != k) {
                    const cx<double> t = A[k * W + n + tid];
                    A[k * W + n + tid] = A[pr * W + n + tid];
                    A[pr * W + n + tid] = t;
                }
            }
        bar();
        for (int k = 0; k < n; ++k) {
            if (tid < n) A[k * W + n + tid] = A[k * W + n + tid] * A[k * W + k];
            bar();
            for (int e = tid; e < (n - k - 1) * n; e += NT) {
                const int i = k + 1 + e / n, j = n + e % n;
                A[i * W + j] = cnmac(A[i * W + j], A[i * W + k], A[k * W + j]);
            }
            bar();
        }
        back_substitute<W>(n, A, A, W, n);
        store_rhs<W>(a, s, n, A, n, bad);
        if (*bad) info = n + 1;
    }
    if (tid == 0) a.info[s] = info;
}

// block = system; the worker warps factor (a.G) or re-solve, the last forms zeta (a.dots)
template <int N>
__global__ void __launch_bounds__(NT + 32) k_small_step(const __grid_constant__ SmallStep a) {
    __shared__ cx<double> A[N * 2 * N];
    __shared__ u64 gmax;
    __shared__ int bad;
    const int s = blockIdx.x;
    if (!((a.p.active >> s) & 1ull)) return;
    if (threadIdx.x == 0) {
        gmax = 0;
        bad = 0;
    }
    __syncthreads();
    if (threadIdx.x >= NT) {
        if (a.dots) zeta_warp(a, s, threadIdx.x & 31);
    } else if (a.G) {
        factor_block<N>(a, s, A, &gmax, &bad);
    } else {
        resolve_block<N>(a, s, A, &bad);
    }
}

// Tinv_s = T^-1 with S_s = T^H T, T upper triangular.  Elimination on [S | 1]
// without pivoting gives S = L D L^H and the rows of L^-1; T^-1 = L^-H D^-1/2.
// One barrier a step: a step writes only rows below k, and column k no more.
// floor as for launch_chol_inv.
template <int N>
__global__ void __launch_bounds__(NT) k_small_chol(const double2* __restrict__ S, double2* __restrict__ Tinv,
                                                  const __grid_constant__ SysPart p, double floor) {
    __shared__ cx<double> A[N][N], R[N][N];
    __shared__ double rs[N], lows[N];
    const int s = blockIdx.x, tid = threadIdx.x;
    if (!((p.active >> s) & 1ull)) return;
    const int n = p.L[s], off = p.coef_off[s];
    for (int e = tid; e < n * n; e += NT) {
        const double2 g = S[off + e];
        A[e / n][e % n] = mk(g.x, g.y);
        R[e / n][e % n] = mk(e / n == e % n ? 1.0 : 0.0, 0.0);
        if (e / n == e % n) lows[e / n] = floor * n * g.x;
    }
    __syncthreads();
    u64 dm = 0;
    for (int k = 0; k < n; ++k) {
        const long long b = __double_as_longlong(A[k][k].r);
        if (b > 0) dm = max(dm, (u64)b);
    }
    const double dmin = 1e-14 * __longlong_as_double((long long)dm);
    __syncthreads();  // every thread has the diagonal before a step changes it
    bool bad = false;
    for (int k = 0; k < n; ++k) {
        const double low = floor > 0.0 ? lows[k] : dmin;
        double d = A[k][k].r;
        if (!(d > low)) {
            if (!(floor > 0.0) || !(low > 0.0) || !(fabs(d) > CHOL_EXACT / (floor * n) * low)) {
                bad = true;
                break;
            }
            d = low;
        }
        if (!isfinite(d)) {
            bad = true;
            break;
        }
        const double q = rsqrt(d), r = q * q;
        if (tid == 0) rs[k] = q;
        // rows below: columns right of k of S, columns up to k of the inverse
        for (int e = tid; e < (n - k - 1) * n; e += NT) {
            const int i = k + 1 + e / n, j = e % n;
            const cx<double> l = r * A[i][k];
            if (j > k) A[i][j] = cnmac(A[i][j], l, A[k][j]);
            else R[i][j] = cnmac(R[i][j], l, R[k][j]);
        }
        __syncthreads();
    }
    __syncthreads();
    for (int e = tid; e < n * n; e += NT) {
        const int j = e / n, k = e % n;
        double2 t = make_double2(j == k ? 1.0 : 0.0, 0.0);
        if (!bad) t = j <= k ? make_double2(rs[k] * R[k][j].r, -rs[k] * R[k][j].i) : make_double2(0.0, 0.0);
        Tinv[off + e] = t;
    }
}

}  // namespace

bk_status launch_small_step(const SmallStep& a, cudaStream_t st) {
    int maxL = 0;
    for (int s = 0; s < a.p.nsys; ++s) maxL = std::max(maxL, a.p.L[s]);
    if (maxL > SMALL_MAXL) {
        bk_set_error("the one-launch L x L step supports L <= %d per system", SMALL_MAXL);
        return BK_ERR_INVALID_ARG;
    }
    if (maxL <= 6) k_small_step<6><<<a.p.nsys, NT + 32, 0, st>>>(a);
    else k_small_step<12><<<a.p.nsys, NT + 32, 0, st>>>(a);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}

bk_status launch_small_chol(const double* S, double* Tinv, const SysPart& p, double floor, cudaStream_t st) {
    int maxL = 0;
    for (int s = 0; s < p.nsys; ++s) maxL = std::max(maxL, p.L[s]);
    if (maxL > SMALL_MAXL) {
        bk_set_error("the one-launch Cholesky supports L <= %d per system", SMALL_MAXL);
        return BK_ERR_INVALID_ARG;
    }
    if (maxL <= 6) k_small_chol<6><<<p.nsys, NT, 0, st>>>((const double2*)S, (double2*)Tinv, p, floor);
    else k_small_chol<12><<<p.nsys, NT, 0, st>>>((const double2*)S, (double2*)Tinv, p, floor);
    BK_CUDA_TRY(cudaGetLastError());
    return BK_OK;
}
