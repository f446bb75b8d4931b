// FP64 mode product on the FP64 pipe (plain-precision path).
//
// One mode product Y = X x_a M of Sec. 4.1 eq. fin_inverse (the paper's
// vec(A X B^T) = (B kron A) vec(X) identity) is written as one GEMM over the
// contiguous axis of X, with the result stored TRANSPOSED:
//
//     out[k][m] = sum_j A[m][j] * M[k][j],   A = X viewed as [Mtot][n].
//
// Storing out[k][m] rotates the tensor's axes by one: a [z][y][x] input
// contracted over x comes out as [k_x][z][y], so the next product again
// contracts the contiguous axis. After dim products the axes are back in
// their original order. Every product is therefore the same K-contiguous
// GEMM, and consecutive threads write consecutive m (coalesced).
//
// Epilogues: EPI_STORE (next product's input), EPI_DIVIDE (pointwise
// division by lambda_k + row eigen-sum + shift, eq. fin_inverse), EPI_UPDATE
// (U -= step * delta; the last backward product's (k, m) is U's own dense
// index k*Mtot + m), EPI_DENSE (plain store to the dense output).
//
// The products of small problems only: larger ones run on the tensor cores
// (qn_modeprod_f64tc.cu, f64tc_pays). 8 x 8 output tiles spread them over the SMs.
#include "qn_internal.h"

namespace qn {

namespace {

// 8 x 8 outputs per 64-thread block: a 63^2 product would be one 64 x 64 tile, i.e. one SM
// bound by its FP64 pipe. The block stages its 8 rows of A and 8 rows of B (all of K <= kSmallK) in
// shared memory; thread (i, j) forms one dot product. Same epilogues.
constexpr int SB = 8, kSmallK = 256;

template <int DIM, int EPI>
__global__ void __launch_bounds__(64) k_modeprod_f64_small(const double *__restrict__ A,
                                                           const double *__restrict__ B,
                                                           double *__restrict__ out, int Mtot, int n,
                                                           EpiArgs e) {
    if (e.done != nullptr && *(volatile const int *)e.done) return;
    __shared__ double As[SB][kSmallK + 1];
    __shared__ double Bs[SB][kSmallK + 1];
    const long long m0 = (long long)blockIdx.x * SB;
    const int k0 = blockIdx.y * SB;
    for (int t = threadIdx.x; t < SB * n; t += 64) {
        const int r = t / n, c = t - r * n;
        const long long gm = m0 + r;
        const int gk = k0 + r;
        As[r][c] = (gm < Mtot) ? __ldg(A + gm * n + c) : 0.0;
        Bs[r][c] = (gk < n) ? __ldg(B + (long long)gk * n + c) : 0.0;
    }
    __syncthreads();
    const int i = threadIdx.x & 7, j = threadIdx.x >> 3;
    const long long m = m0 + i;
    const int k = k0 + j;
    double acc0 = 0.0, acc1 = 0.0;   // two chains: the FP64 pipe's latency
    int c = 0;
    for (; c + 1 < n; c += 2) {
        acc0 = fma(As[i][c], Bs[j][c], acc0);
        acc1 = fma(As[i][c + 1], Bs[j][c + 1], acc1);
    }
    if (c < n) acc0 = fma(As[i][c], Bs[j][c], acc0);
    const double acc = acc0 + acc1;
    if (m >= Mtot || k >= n) return;
    const long long o = (long long)k * Mtot + m;
    if (EPI == EPI_STORE || EPI == EPI_DENSE) {
        out[o] = acc;
    } else if (EPI == EPI_DIVIDE) {
        const double rowlam = (DIM == 3) ? e.lam64[m / n] + e.lam64[m % n] : e.lam64[m];
        out[o] = acc / (e.lam64[k] + rowlam + *e.shift);
    } else {   // EPI_UPDATE
        out[o] = out[o] - e.step * acc;
    }
}

template <int DIM>
void launch_small(const double *A, const double *B, double *out, const GemmShape &g, Epi epi,
                  const EpiArgs &e, cudaStream_t s) {
    dim3 grid((unsigned)((g.Mtot + SB - 1) / SB), (unsigned)((g.n + SB - 1) / SB));
    switch (epi) {
        case EPI_STORE: k_modeprod_f64_small<DIM, EPI_STORE><<<grid, 64, 0, s>>>(A, B, out, g.Mtot, g.n, e); break;
        case EPI_DIVIDE: k_modeprod_f64_small<DIM, EPI_DIVIDE><<<grid, 64, 0, s>>>(A, B, out, g.Mtot, g.n, e); break;
        case EPI_UPDATE: k_modeprod_f64_small<DIM, EPI_UPDATE><<<grid, 64, 0, s>>>(A, B, out, g.Mtot, g.n, e); break;
        case EPI_DENSE: k_modeprod_f64_small<DIM, EPI_DENSE><<<grid, 64, 0, s>>>(A, B, out, g.Mtot, g.n, e); break;
    }
}

}  // namespace

int launch_modeprod_f64(const double *A, const double *B, double *out, const GemmShape &g,
                        Epi epi, const EpiArgs &e, cudaStream_t s) {
    if (g.n > kSmallK) {
        set_error("launch_modeprod_f64: n = %d is beyond the small-problem kernel", g.n);
        return QN_EINVAL;
    }
    if (g.dim == 3)
        launch_small<3>(A, B, out, g, epi, e, s);
    else
        launch_small<2>(A, B, out, g, epi, e, s);
    QN_CUDA(cudaGetLastError());
    return QN_OK;
}

}  // namespace qn
