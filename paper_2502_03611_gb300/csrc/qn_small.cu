// Whole-solve persistent kernel for small 2-D FP64 problems (Sec. 4 eq. identity-method
// with the inverse of Sec. 4.1 eq. fin_inverse), n <= kSmallMaxN.
//
// At these sizes every phase of an iteration is a few microseconds of work (the 63^2
// grid has 3969 unknowns; one mode product is 125k FP64 FMAs), so a solve made of
// separate launches is bound by launch and host-check latency. Here one cooperative
// launch runs the whole solve; block b owns row y = b of the grid and mode kx = b (and
// b + grid, ... with fewer blocks than rows).
//
//   iteration k:  wait for the neighbouring rows' updates (one flag word per row)
//                 residual r = A_h U + lam U + b U^3 - f of the row (+ block partials of
//                 ||r||^2, ||f||^2 at k = 0, min / max U^2), and from it
//                 P1  Y1[kx][y] = sum_x S^{-1}[kx][x] r[y][x]          -> grid barrier
//                 every block reduces the partial records in the same order, so all
//                 take the same stop decision and the same beta_n = (min + max)/2 of
//                 3 b U^2; block 0 records the iterate's statistics
//                 P2  Y2[ky] = sum_y S^{-1}[ky][y] Y1[kx][y] / (lam_kx + lam_ky + lam + beta_n)
//                 P3  Z[y][kx] = sum_ky S[y][ky] Y2[ky], in the same block  -> grid barrier
//                 P4  U[y][x] -= step * sum_kx S[x][kx] Z[y][kx]; the row's flag
//
// The backward transform takes y first, so that a mode's column never leaves its block:
// two grid barriers an iteration and a wait for two neighbours, where the order of the
// large solves needs four barriers. The products use the reflection symmetry (half the
// FP64 work, see qn_modeprod_f64tc.cu), with both half matrices transposed in shared
// memory: read from L1 by rows, a warp's 32 lanes touched 32 lines for every term, and
// the four products took most of an iteration. 273 -> 190 us per 63^2 solve of seven iterations
// (the kernel 235 -> 140 us).
//
// Every wait is bounded (2 s of %globaltimer), after which the block sets the error word,
// and all blocks leave at their next wait. The launch is cooperative, so all blocks are
// resident at once.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include "qn_internal.h"
#include "qn_numeric.cuh"

namespace qn {

namespace {

constexpr int kSmallThreads = 128;
constexpr int kBarGen = 32;   // the generation word, a 128-byte line away from the counter
constexpr int kBarFlags = 64; // one word per row: updates applied to it
constexpr unsigned long long kSmallTimeoutNs = 2000000000ull;

__device__ __forceinline__ unsigned long long small_timer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Grid barrier: returns false when a wait gave up (or another block's had), after
// recording QN_ETIMEOUT in *err. Thread 0 arrives with one acquire-release add on the
// counter (after the block's barrier, it releases the block's writes); the last block
// resets the counter and releases the generation word, which the others poll with
// acquire loads.
__device__ bool small_barrier(unsigned *count, unsigned *gen, int *err) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        const unsigned g = ld_acquire(gen);
        unsigned old;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(count) : "memory");
        if (old == gridDim.x - 1) {
            asm volatile("st.relaxed.gpu.global.u32 [%0], 0;" ::"l"(count) : "memory");
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(gen) : "memory");
        } else {
            // the error word and the clock only every 64 polls
            const unsigned long long t0 = small_timer();
            unsigned polls = 0;
            while (ld_acquire(gen) == g) {
                if ((++polls & 63u) == 0 &&
                    (*(volatile int *)err != 0 || small_timer() - t0 > kSmallTimeoutNs)) {
                    atomicExch(err, QN_ETIMEOUT);
                    ok = 0;
                    break;
                }
            }
        }
    }
    __syncthreads();
    return ok != 0;
}

struct SmallArgs {
    double *U;
    const double *f;
    const double *S, *Si, *lam1;   // n x n row-major (S[:, k] eigenvector k), eigenvalues
    double *w0, *w1;               // n^2 work arrays
    double *partials;              // [gridDim][4]
    unsigned *bar;                 // barrier counter, generation, row flags
    DevState *st;                  // it / status / done on return
    qn_stats *hist;
    int hist_cap;
    int *err;
    int n, neumann;
    double inv_h2, lam, b, tol, beta_value, step;
    int beta_fixed, max_it;
};

// Wait (thread 0) until the two neighbouring rows of row y have had `it` updates.
__device__ bool wait_rows(const unsigned *flags, int y, int n, unsigned it, int *err) {
    for (int k = -1; k <= 1; k += 2) {
        const int r = y + k;
        if (r < 0 || r >= n) continue;
        const unsigned long long t0 = small_timer();
        unsigned polls = 0;
        while (ld_acquire(flags + r) < it) {
            if ((++polls & 63u) == 0 && (*(volatile int *)err != 0 || small_timer() - t0 > kSmallTimeoutNs)) {
                atomicExch(err, QN_ETIMEOUT);
                return false;
            }
        }
    }
    return true;
}

// Four chains of the terms 0 .. len - 1 of column t of a table with row stride n.
__device__ __forceinline__ double dot_column(const double *tab, const double *v, int vs, int len, int n, int t) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    int j = 0;
    for (; j + 4 <= len; j += 4) {
        s0 = fma(tab[j * n + t], v[j * vs], s0);
        s1 = fma(tab[(j + 1) * n + t], v[(j + 1) * vs], s1);
        s2 = fma(tab[(j + 2) * n + t], v[(j + 2) * vs], s2);
        s3 = fma(tab[(j + 3) * n + t], v[(j + 3) * vs], s3);
    }
    for (; j < len; ++j) s0 = fma(tab[j * n + t], v[j * vs], s0);
    return (s0 + s1) + (s2 + s3);
}

// Forward product of the row in v (n values, overwritten by its mirror sums and differences):
// thread k < n returns sum_j S^{-1}[k][j] v[j].
__device__ __forceinline__ double small_forward(const double *F, double *v, int n, int t) {
    const int nsym = (n + 1) >> 1, nanti = n >> 1;
    double x = 0.0, y = 0.0;
    if (t < nsym) {
        x = v[t];
        y = (t < nanti) ? v[n - 1 - t] : 0.0;
    }
    __syncthreads();
    if (t < nsym) v[t] = x + y;
    if (t < nanti) v[nsym + t] = x - y;
    __syncthreads();
    if (t >= n) return 0.0;
    // one loop for both parities (a branch would run them one after the other)
    return dot_column(F, v + ((t & 1) ? nsym : 0), 1, (t & 1) ? nanti : nsym, n, t);
}

// Backward product of the modes in v: thread s < n returns sum_k S[s][k] v[k]. q: n doubles.
__device__ __forceinline__ double small_backward(const double *B, const double *v, double *q, int n, int t) {
    const int nsym = (n + 1) >> 1, nanti = n >> 1;
    // p_t over the even modes, q_{t - nsym} over the odd ones
    if (t < n) q[t] = dot_column(B, v + (t < nsym ? 0 : 1), 2, t < nsym ? nsym : nanti, n, t);
    __syncthreads();
    double d = 0.0;
    if (t < nsym)
        d = q[t] + (t < nanti ? q[nsym + t] : 0.0);
    else if (t < n)
        d = q[n - 1 - t] - q[nsym + (n - 1 - t)];
    __syncthreads();
    return d;
}

__global__ void __launch_bounds__(kSmallThreads) k_small2d_fp64(SmallArgs a) {
    // F[j][k] = S^{-1}[k][j], j < ceil(n/2); B[i][t] = S[t][2i] (t < ceil(n/2)), S[t - ceil(n/2)][2i+1];
    // three rows of scratch; the block's rows of U
    extern __shared__ double sm[];
    __shared__ double sh_beta, sh_fn;
    __shared__ int sh_stop, sh_ok;
    const int n = a.n, nsym = (n + 1) >> 1, nanti = n >> 1;
    double *F = sm, *B = F + nsym * n, *row = B + nsym * n, *tmp = row + n, *rc = tmp + n, *Ur = rc + n;
    const bool neu = a.neumann != 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = threadIdx.x;
    unsigned *flags = a.bar + kBarFlags;
    for (int e = t; e < n * nsym; e += kSmallThreads) {
        const int k = e / nsym, j = e - k * nsym;   // rows of the matrices: coalesced reads
        F[j * n + k] = __ldg(a.Si + k * n + j);
        const int sr = k < nsym ? k : k - nsym, md = k < nsym ? 2 * j : 2 * j + 1;
        B[j * n + k] = md < n ? __ldg(a.S + sr * n + md) : 0.0;
    }
    {
        int i = 0;
        for (int y = blockIdx.x; y < n; y += gridDim.x, ++i)
            for (int x = t; x < n; x += kSmallThreads) Ur[i * n + x] = __ldcg(a.U + y * n + x);
    }
    if (t == 0) sh_ok = 1;
    __syncthreads();
    double fn = 0.0;
    int it = 0;
    int status = QN_ENOTCONV;
    // The last warp has no outputs of a product up to n = 96: it takes the reductions and the
    // stop decision while the others run the products.
    constexpr int kRedWarp = kSmallThreads / 32 - 1;
    for (;; ++it) {
        // ---- residual of the rows this block owns, its partial record, and P1
        double r2 = 0.0, f2 = 0.0, mn = INFINITY, mx = 0.0;
        int i = 0;
        for (int y = blockIdx.x; y < n; y += gridDim.x, ++i) {
            if (it > 0 && t == 0 && !wait_rows(flags, y, n, (unsigned)it, a.err)) sh_ok = 0;
            __syncthreads();
            if (!sh_ok) return;
            if (t < n) {
                const double *ur = Ur + i * n;
                const int yu = y > 0 ? y - 1 : (neu ? 1 : -1), yd = y < n - 1 ? y + 1 : (neu ? n - 2 : -1);
                const double up = yu >= 0 ? __ldcg(a.U + yu * n + t) : 0.0;
                const double dn = yd >= 0 ? __ldcg(a.U + yd * n + t) : 0.0;
                const double le = t > 0 ? ur[t - 1] : (neu ? ur[1] : 0.0);
                const double ri = t < n - 1 ? ur[t + 1] : (neu ? ur[n - 2] : 0.0);
                const double u = ur[t];
                const double lap = ((4.0 * u - le) - ri) - (up + dn);
                const double fv = __ldg(a.f + y * n + t);
                double v = fma(a.b, (u * u) * u, -fv);
                v = fma(a.lam, u, v);
                const double r = fma(lap, a.inv_h2, v);
                row[t] = r;
                rc[t] = r;
            }
            __syncthreads();
            const double v = small_forward(F, row, n, t);
            if (t < n) a.w1[t * n + y] = v;   // Y1[kx = t][y]
            if (warp == kRedWarp)
                for (int x = lane; x < n; x += 32) {
                    const double r = rc[x], u = Ur[i * n + x], u2 = u * u;
                    r2 = fma(r, r, r2);
                    if (it == 0) {
                        const double fv = __ldg(a.f + y * n + x);
                        f2 = fma(fv, fv, f2);
                    }
                    mn = fmin(mn, u2);
                    mx = fmax(mx, u2);
                }
        }
        if (warp == kRedWarp) {
            for (int o = 16; o > 0; o >>= 1) {
                r2 += __shfl_xor_sync(0xffffffffu, r2, o);
                if (it == 0) f2 += __shfl_xor_sync(0xffffffffu, f2, o);
                mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
                mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            }
            if (lane == 0) {
                double *q = a.partials + 4 * blockIdx.x;
                q[0] = r2;
                q[1] = f2;
                q[2] = mn;
                q[3] = mx;
            }
        }
        if (!small_barrier(a.bar, a.bar + kBarGen, a.err)) return;
        // ---- every block: the same reduction, the same decision
        auto decide = [&]() {
            double R = 0.0, F2 = 0.0, MN = INFINITY, MX = 0.0;
            for (int i = lane; i < (int)gridDim.x; i += 32) {
                const double *q = a.partials + 4 * i;
                R += __ldcg(q + 0);
                F2 += __ldcg(q + 1);
                MN = fmin(MN, __ldcg(q + 2));
                MX = fmax(MX, __ldcg(q + 3));
            }
            for (int o = 16; o > 0; o >>= 1) {
                R += __shfl_xor_sync(0xffffffffu, R, o);
                F2 += __shfl_xor_sync(0xffffffffu, F2, o);
                MN = fmin(MN, __shfl_xor_sync(0xffffffffu, MN, o));
                MX = fmax(MX, __shfl_xor_sync(0xffffffffu, MX, o));
            }
            if (lane == 0) {
                if (it == 0) sh_fn = sqrt(F2);
                const double res = sqrt(R);
                const double f_norm = sh_fn;
                const double fa = 3.0 * a.b * MN, fb = 3.0 * a.b * MX;
                const double fu_min = fmin(fa, fb), fu_max = fmax(fa, fb);
                const double beta = a.beta_fixed ? a.beta_value : 0.5 * (fu_min + fu_max);
                const double rel = (f_norm > 0.0) ? res / f_norm : ((res == 0.0) ? 0.0 : INFINITY);
                if (blockIdx.x == 0 && it < a.hist_cap) {
                    qn_stats s;
                    s.res_norm = res;
                    s.f_norm = f_norm;
                    s.fu_min = fu_min;
                    s.fu_max = fu_max;
                    s.beta = beta;
                    s.rel = rel;
                    s.lambda = 0.0;
                    a.hist[it] = s;
                }
                int stop = 0;
                if (rel <= a.tol) {
                    stop = 1;
                    status = QN_OK;
                } else if (!isfinite(rel) || rel > 1e8 || !isfinite(beta)) {
                    stop = 1;
                    status = QN_EDIVERGED;
                } else if (it >= a.max_it) {
                    stop = 1;
                    status = QN_ENOTCONV;
                }
                sh_stop = stop;
                sh_beta = a.lam + beta;
            }
        };
        // P2, P3 of the modes kx this block owns; the decision falls during the first P2
        bool stop = false;
        for (int kx = blockIdx.x; kx < n; kx += gridDim.x) {
            __syncthreads();
            if (t < n) row[t] = __ldcg(a.w1 + kx * n + t);
            __syncthreads();
            double v = small_forward(F, row, n, t);
            if (kx == (int)blockIdx.x) {
                if (warp == kRedWarp) decide();
                __syncthreads();
                fn = sh_fn;
                stop = sh_stop != 0;
                if (stop) break;
            }
            const double shift = sh_beta;
            if (t < n) tmp[t] = v / ((__ldg(a.lam1 + kx) + __ldg(a.lam1 + t)) + shift);
            __syncthreads();
            v = small_backward(B, tmp, row, n, t);
            if (t < n) a.w0[t * n + kx] = v;   // Z[y = t][kx]
        }
        if (stop) break;
        if (!small_barrier(a.bar, a.bar + kBarGen, a.err)) return;
        // P4 and the update of the rows
        i = 0;
        for (int y = blockIdx.x; y < n; y += gridDim.x, ++i) {
            if (t < n) tmp[t] = __ldcg(a.w0 + y * n + t);
            __syncthreads();
            const double d = small_backward(B, tmp, row, n, t);
            if (t < n) {
                const double u = Ur[i * n + t];
                const double w = (a.step == 1.0) ? u - d : fma(-a.step, d, u);
                Ur[i * n + t] = w;
                a.U[y * n + t] = w;
            }
            __syncthreads();
            if (t == 0)
                asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(flags + y), "r"((unsigned)(it + 1)) : "memory");
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 32 * kRedWarp) {   // the lane that decided
        a.st->it = it;
        a.st->status = status;
        a.st->done = 1;
        a.st->f_norm = fn;
    }
}

}  // namespace

int small_solve_supported(int dim, int n) { return dim == 2 && n >= 1 && n <= kSmallMaxN; }

// Shared memory for `grid` blocks: both half matrices, three rows of scratch, the block's rows.
static size_t small_smem(int n, int grid) {
    const int nsym = (n + 1) / 2, rows = (n + grid - 1) / grid;
    return sizeof(double) * ((size_t)2 * nsym * n + 3 * n + (size_t)rows * n);
}

int small_solve_set_attributes() {
    QN_CUDA(cudaFuncSetAttribute(k_small2d_fp64, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    return QN_OK;
}

int launch_small_solve(const SmallSolve &q, cudaStream_t s) {
    // one block per SM (the phases are FP64-FMA bound: about 2 FMAs per clock per SM on
    // this GPU) and per row
    const char *eg = getenv("QN_SMALL_GRID");
    int grid = eg ? atoi(eg) : q.n;
    if (grid > q.num_sms) grid = q.num_sms;
    if (grid > q.n) grid = q.n;
    if (grid < 1) grid = 1;
    if (grid > q.partials_cap) grid = q.partials_cap;
    if (grid < 1) grid = 1;
    // a block holds both half matrices and its rows of U: one block's rows do not fit above n = 117
    if (small_smem(q.n, grid) > 220 * 1024 && q.num_sms > 1 && q.partials_cap > 1) grid = 2;
    if (small_smem(q.n, grid) > 220 * 1024) {
        set_error("launch_small_solve: %d rows of n = %d per block do not fit in shared memory", (q.n + grid - 1) / grid,
                  q.n);
        return QN_EINVAL;
    }
    SmallArgs a;
    a.U = q.U;
    a.f = q.f;
    a.S = q.S;
    a.Si = q.Si;
    a.lam1 = q.lam1;
    a.w0 = q.w0;
    a.w1 = q.w1;
    a.partials = q.partials;
    a.bar = q.bar;
    a.st = q.st;
    a.hist = q.hist;
    a.hist_cap = q.hist_cap;
    a.err = q.err;
    a.n = q.n;
    a.neumann = q.neumann;
    a.inv_h2 = q.inv_h2;
    a.lam = q.lam;
    a.b = q.b;
    a.tol = q.tol;
    a.beta_value = q.beta_value;
    a.step = q.step;
    a.beta_fixed = q.beta_fixed;
    a.max_it = q.max_it;
    QN_CUDA(cudaMemsetAsync(q.bar, 0, kSmallBarWords * sizeof(unsigned), s));
    void *params[] = {&a};
    QN_CUDA(cudaLaunchCooperativeKernel((const void *)k_small2d_fp64, dim3(grid), dim3(kSmallThreads), params,
                                        small_smem(q.n, grid), s));
    return QN_OK;
}

}  // namespace qn
