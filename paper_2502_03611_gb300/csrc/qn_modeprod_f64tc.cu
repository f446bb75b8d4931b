// FP64 mode products on the tensor cores (plain-precision path).
//
// The same product as qn_modeprod_f64.cu (one mode product of Sec. 4.1 eq. fin_inverse, the
// result stored transposed so that the axes rotate):
//
//     out[k][m] = sum_j A[m][j] * M[k][j],   A = X viewed as [Mtot][n], FP64 in and out,
//
// computed from exact integer digits instead of FP64 multiply-adds (the splitting of Ozaki,
// Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication", Numer. Algorithms 59, 2012, in its fixed-point form):
//
//   1. k_slice_rows brings every row of A to one power-of-two scale as 63-bit fixed point and
//      cuts it into seven balanced digits of nine bits in [-256, 255], stored as FP16
//      integers. The mirror sums and differences of the reflection split are formed there,
//      exactly, on the integers.
//   2. k_modeprod_f64tc forms the digit products D_i G_j with i + j <= 6 (28 tcgen05 products,
//      FP16 operands, FP32 accumulation) into one TMEM accumulator per d = i + j. A product of
//      two digits is an integer of at most 2^16, and FP32 sums of integers are exact up to 2^24 =
//      256 products: accumulators 0 and 1 take kSegK = 128 terms at a time, 2 to 4 take
//      BK = 64. So the sums up to d = 3 are exact whatever the digits. Those of d = 4 are while the
//      five products of a term average below 0.8 of their range (a row of B that is constant may have
//      more); a rounding there is 2^-51 of the largest product, within what a chain of FP64
//      multiply-adds may lose on the same terms. Those of d = 5 and 6 are below the last bit kept.
//   3. Its epilogue adds the seven accumulators as one 64-bit integer
//      sum_d C_d 2^(38-9d), forms p +- q of the reflection split on the integers, converts
//      once to FP64, applies the row's and the column's exponents and stores, divides or
//      updates as the FP64 kernels do.
//
// Every output therefore carries two roundings at the end (the 64-bit sum's and the
// conversion's), where a chain of FP64 multiply-adds rounds at every step. GB300's FP64 pipe runs at
// about 2 lanes per clock per SM: a product at 255^3 took it 3.6 ms, where the 28 FP16 products take
// 0.15 to 0.21 ms and the slicing 0.06.
//
// A row that holds a NaN or an infinity has no fixed-point form: its digits are zero, its
// exponent is a mark, and the epilogue forms its outputs with FP64 multiply-adds from the
// row itself, so non-finite values propagate as they do in the FP64 kernels.
#include <cuda_fp16.h>
#include <cudaTypedefs.h>
#include <limits.h>
#include <stdlib.h>
#include <string.h>

#include <new>

#include "qn_internal.h"
#include "qn_ptx.cuh"

namespace qn {

namespace {

constexpr int kDig = 7;                  // digits per value
constexpr int BM = 128, BK = 64;         // tile rows; K per pipeline step (a 128-byte swizzle row)
constexpr int kSlots = 9;                // digit tiles of A and B in shared memory
constexpr int kSegK = 128;               // terms per sum of digit products,
constexpr int kMid0 = 2, kMid1 = 4;      // of which these accumulators take BK at a time
constexpr int kTotal = 256;              // terms whose 64-bit sum fits with full-range digits
constexpr int kEpiWarps = 16;            // four warps per TMEM lane quadrant
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kCtrlBytes = 512;
constexpr int kNonFinite = INT_MAX;      // exponent mark of a row without a fixed-point form
constexpr int kBits = 9;
// 256 in every digit: makes the nine-bit fields of a sum the digits plus 256
constexpr unsigned long long kBias = 0x4020100804020100ull;
constexpr unsigned long long kTop = 1ull << 62;   // digits reach kTop - (kBias without its top field)

// How a row pair of digits is read from FP64 rows.
enum SliceKind : int {
    SL_DENSE = 0,   // one half: x_j
    SL_FWD = 1,     // halves x_j + x_{n-1-j} (the middle x of an odd n alone) and x_j - x_{n-1-j}
    SL_PARITY = 2,  // halves x_{2i} and x_{2i+1}, one common scale
    SL_ROWS = 3,    // halves are the rows 2r and 2r + 1 of the source (their first ceil(n/2), n/2 columns)
};

// Both operands of a product use this: digits[d][row][half * Kp + j], exponents ex[row].{x, y}
// per half, value = integer * 2^ex with the integers scaled as in the file comment.
struct SliceArgs {
    const double *src;
    __half *dig;
    int2 *ex;
    const int *done;
    long long slice_stride;   // elements between digits d and d + 1
    int rows, n, Kp, ld;      // ld = halves * Kp
    int row0;                 // first source row (SL_ROWS: first row pair)
    int extra;                // bits of headroom kept free (B operands of long sums)
};

// Fixed point of one double against the row's largest exponent: 61-bit magnitude.
__device__ __forceinline__ long long to_fixed(double v, int emax) {
    const long long b = __double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    unsigned long long mant = (unsigned long long)b & 0xfffffffffffffull;
    if (e != 0) mant |= 1ull << 52;
    const int sh = emax - max(e, 1);
    const unsigned long long f = (sh < 64) ? (mant << 8) >> sh : 0ull;
    return b < 0 ? -(long long)f : (long long)f;
}

__device__ __forceinline__ int exp_of(double v) { return max((__double2hiint(v) >> 20) & 0x7ff, 1); }

__device__ __forceinline__ unsigned long long abs64(long long v) {
    return v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
}

// Left shift that brings the largest magnitude of a row to the top of the digit range: the
// shifted value plus the bias of the six lower digits stays below 2^62.
__device__ __forceinline__ int norm_shift(unsigned long long mine, bool *zero) {
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(mine >> 32));
    unsigned long long mx = ((unsigned long long)hi << 32) | 0xffffffffull;
    if (hi == 0) mx = __reduce_max_sync(0xffffffffu, (unsigned)mine);
    *zero = (mx == 0);
    if (mx == 0) return 0;
    int sh = __clzll((long long)mx) - 2;
    if ((mx << sh) + (kBias ^ kTop) >= kTop) --sh;
    return sh;
}

__device__ __forceinline__ unsigned long long shifted(long long v, int sh) {
    return (unsigned long long)(sh >= 0 ? v << sh : v >> -sh) + kBias;
}

// Digit d (0 = most significant) of two biased values as an FP16 pair: the nine-bit field is
// the mantissa of 1024 + field.
template <int d>
__device__ __forceinline__ uint32_t digit_pair(unsigned long long t0, unsigned long long t1) {
    constexpr int at = kBits * (kDig - 1 - d);
    const uint32_t two = __byte_perm((uint32_t)(t0 >> at), (uint32_t)(t1 >> at), 0x5410);
    const uint32_t h = (two & 0x01ff01ffu) | 0x64006400u;
    const __half2 r = __hsub2(*reinterpret_cast<const __half2 *>(&h), __float2half2_rn(1280.0f));
    return *reinterpret_cast<const uint32_t *>(&r);
}

template <int d>
__device__ __forceinline__ void put_digits(const SliceArgs &a, long long at, unsigned long long t0,
                                           unsigned long long t1) {
    if constexpr (d < kDig) {
        *reinterpret_cast<uint32_t *>(a.dig + at + d * a.slice_stride) = digit_pair<d>(t0, t1);
        put_digits<d + 1>(a, at, t0, t1);
    }
}

// One warp per row; a lane takes columns 64 s + 2 lane and the next one, NST steps of 64.
template <int KIND, int NST>
__global__ void __launch_bounds__(256) k_slice_rows(const SliceArgs a) {
    if (a.done != nullptr && *(volatile const int *)a.done) return;
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= a.rows) return;
    const int n = a.n, nsym = (n + 1) >> 1, nanti = n >> 1;
    constexpr bool TWO = (KIND != SL_DENSE);
    const double *s0 = a.src + (long long)(KIND == SL_ROWS ? 2 * (a.row0 + row) : a.row0 + row) * n;
    const bool has1 = KIND != SL_ROWS || 2 * (a.row0 + row) + 1 < n;
    const double *s1 = (KIND == SL_ROWS) ? s0 + n : s0;

    double x[NST][2], y[NST][2];
    int e0 = 1, e1 = 1;
#pragma unroll
    for (int s = 0; s < NST; ++s)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int j = 64 * s + 2 * lane + u;
            x[s][u] = y[s][u] = 0.0;
            if (KIND == SL_DENSE) {
                if (j < n) x[s][u] = __ldg(s0 + j);
            } else if (KIND == SL_FWD) {
                if (j < nsym) x[s][u] = __ldg(s0 + j);
                if (j < nanti) y[s][u] = __ldg(s0 + (n - 1 - j));
            } else if (KIND == SL_PARITY) {
                if (2 * j < n) x[s][u] = __ldg(s0 + 2 * j);
                if (2 * j + 1 < n) y[s][u] = __ldg(s0 + 2 * j + 1);
            } else {
                if (j < nsym) x[s][u] = __ldg(s0 + j);
                if (has1 && j < nanti) y[s][u] = __ldg(s1 + j);
            }
            e0 = max(e0, exp_of(x[s][u]));
            if (TWO) e1 = max(e1, exp_of(y[s][u]));
        }
    if (KIND != SL_ROWS) e0 = max(e0, e1);
    e0 = (int)__reduce_max_sync(0xffffffffu, (unsigned)e0);
    if (KIND == SL_ROWS)
        e1 = (int)__reduce_max_sync(0xffffffffu, (unsigned)e1);
    else
        e1 = e0;
    const bool bad0 = e0 == 0x7ff, bad1 = e1 == 0x7ff;

    long long p[NST][2], q[NST][2];
    unsigned long long m0 = 0, m1 = 0;
#pragma unroll
    for (int s = 0; s < NST; ++s)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const long long X = bad0 ? 0 : to_fixed(x[s][u], e0);
            const long long Y = (!TWO || bad1) ? 0 : to_fixed(y[s][u], e1);
            if (KIND == SL_FWD) {
                const int j = 64 * s + 2 * lane + u;
                p[s][u] = X + Y;
                q[s][u] = (j < nanti) ? X - Y : 0;
            } else {
                p[s][u] = X;
                q[s][u] = Y;
            }
            m0 = max(m0, abs64(p[s][u]));
            m1 = max(m1, abs64(q[s][u]));
        }
    if (KIND == SL_PARITY) m0 = m1 = max(m0, m1);
    bool z0, z1 = true;
    int sh0 = norm_shift(m0, &z0) - a.extra, sh1 = 0;
    if (KIND == SL_PARITY) {
        sh1 = sh0;
        z1 = z0;
    } else if (TWO) {
        sh1 = norm_shift(m1, &z1) - a.extra;
    }
    const long long at = (long long)row * a.ld + 2 * lane;
#pragma unroll
    for (int s = 0; s < NST; ++s) {
        if (64 * s + 2 * lane >= a.Kp) break;
        put_digits<0>(a, at + 64 * s, shifted(p[s][0], sh0), shifted(p[s][1], sh0));
        if (TWO) put_digits<0>(a, at + a.Kp + 64 * s, shifted(q[s][0], sh1), shifted(q[s][1], sh1));
    }
    if (lane == 0) {
        // value = integer * 2^(e - 1083 - sh), integer = sum_i D_i 2^(54-9i): half of the 2^70
        // between the product of the integers and the epilogue's 64-bit sum goes to each side
        int2 e;
        e.x = bad0 ? kNonFinite : (z0 ? 0 : e0 - 1083 - sh0 + 35);
        e.y = bad1 ? kNonFinite : (z1 ? 0 : e1 - 1083 - sh1 + 35);
        a.ex[row] = e;
    }
}

// ---------------------------------------------------------------------------------------------
// the digit products
// ---------------------------------------------------------------------------------------------
enum Mode : int { MD_DENSE = 0, MD_FWD = 1, MD_BWD = 2 };

struct ProdArgs {
    const CUtensorMap *amap, *bmap;
    const int2 *ea, *eb;
    const double *A, *B;      // the FP64 operands (rows with non-finite values)
    double *out;              // next product's input, or the dense target
    int rows;                 // rows of this launch
    int m0;                   // the first one's index among all Mtot rows
    int Mtot, n, dim;
    int Kp;                   // padded contraction length of a half
    int Kt;                   // contraction length rounded up to 16 (later columns are zero)
    int nrow;                 // B rows per half that exist (ceil(n/2), or n for the dense product)
    int ntn;                  // column tiles per half
    int ntiles;
    EpiArgs e;
};

// integer * 2^e as a double (one conversion; subnormal and overflowing results take scalbn)
__device__ __noinline__ double scale_slow(double v, int e) { return scalbn(v, e); }

__device__ __forceinline__ double scaled(long long v, int e) {
    const double d = (double)v;
    const int hi = __double2hiint(d), lo = __double2loint(d);
    const int ne = (hi >> 20 & 0x7ff) + e;
    if (v == 0) return 0.0;
    if (ne < 1 || ne > 2046) return scale_slow(d, e);
    return __hiloint2double(hi + (e << 20), lo);
}

__device__ __noinline__ double divided_slow(long long v, int e, double d) { return scalbn((double)v, e) / d; }

// integer * 2^e / d. The FP64 pipe would need about nine of its slow operations per output for
// the division (415 us for a 255^3 product when one without it took 144; now 154 and 213), so the quotient is
// formed on the integer pipe: a reciprocal of the divisor's 64-bit significand from an FP32
// seed and two terms of the series 1/d = x (1 + e + e^2 + ..), e = 1 - d x, |e| < 2^-22, good to
// about 2^-60, times the normalised integer; rounded to 53 bits once.
__device__ __forceinline__ double divided(long long v, int e, double d) {
    const int dhi = __double2hiint(d);
    const int dexp = (dhi >> 20) & 0x7ff;
    if (v == 0 && dexp != 0 && dexp != 0x7ff) return 0.0;
    const unsigned long long D = 1ull << 63 | ((unsigned long long)__double_as_longlong(d) << 11);   // d' = D / 2^64
    const uint32_t dh = (uint32_t)(D >> 32), dl = (uint32_t)D;
    float x;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"((float)(dh >> 8)));   // 2^-24 / d'
    const uint32_t X = __float2uint_rz(x * 0x1p54f);                        // x ~ 2^30 / d', 24 bits
    const long long t = (long long)((unsigned long long)dh * X + __umulhi(dl, X));   // 2^62 d' x
    const long long E = (1ll << 62) - t;                                    // 2^62 e
    const int Es = (int)(E >> 10);
    const long long F = E + (long long)(((unsigned long long)((long long)Es * Es)) >> 42);   // 2^62 (e + e^2)
    const long long xf = ((long long)((unsigned long long)X * (uint32_t)F >> 30)) + (((long long)(int)(F >> 32) * (long long)X) << 2);
    const unsigned long long R = ((unsigned long long)X << 32) + (unsigned long long)xf;      // 2^62 / d'
    const unsigned long long u = abs64(v);
    const int cl = __clzll((long long)u);
    const unsigned long long Q = __umul64hi(u << cl, R);                    // [2^61, 2^63)
    const int sh = 11 - __clzll((long long)Q);
    const unsigned long long q = (Q + (1ull << (sh - 1))) >> sh;            // 53 bits (2^53 after a carry)
    // |v| 2^e / |d| = Q 2^(2 - cl + e - (dexp - 1022)), and a double's exponent field is that of its leading bit + 1075
    const int qe = sh + 2 - cl + e - dexp + 1022 + 1075;
    if (dexp == 0 || dexp == 0x7ff || qe < 1 || qe > 2044) return divided_slow(v, e, d);
    const unsigned long long bits = q + ((unsigned long long)(qe - 1) << 52);
    return __longlong_as_double((long long)(bits | ((unsigned long long)(v ^ __double_as_longlong(d)) & (1ull << 63))));
}

// The product's outputs for one row with non-finite values, as the FP64 kernels form them.
template <int MODE>
__device__ __noinline__ double2 dot_fp64(const double *a, const double *B, int n, int k) {
    const int nsym = (n + 1) >> 1, nanti = n >> 1;
    double p = 0.0, q = 0.0;
    if (MODE == MD_FWD) {
        for (int j = 0; j < nsym; ++j) {
            const double x = a[j], y = (j < nanti) ? a[n - 1 - j] : 0.0;
            const double v = (k & 1) ? (j < nanti ? x - y : 0.0) : x + y;
            p = fma(v, B[(long long)k * n + j], p);
        }
    } else {
        for (int j = 0; j < n; ++j) {
            if (MODE == MD_BWD && (j & 1))
                q = fma(a[j], B[(long long)k * n + j], q);
            else
                p = fma(a[j], B[(long long)k * n + j], p);
        }
    }
    return make_double2(p, q);
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}

template <int NC>
__device__ __forceinline__ void tmem_ld(uint32_t addr, uint32_t (&r)[NC]) {
    if constexpr (NC == 16)
        ptx::tmem_ld_32x32b_x16(addr, r);
    else if constexpr (NC == 8)
        ptx::tmem_ld_32x32b_x8(addr, r);
    else
        ptx::tmem_ld_32x32b_x4(addr, r);
}

template <int BN>
__host__ __device__ constexpr uint32_t slot_bytes() {
    return (BM + BN) * BK * 2;
}

// The order in which the seven digit tiles of a K step are released. Tile t of a step (digit t
// of A and of B) is multiplied with the tiles j <= min(t, 6 - t) that came before it, so tile i
// is last used at t = max(i, 6 - i), and a commit after those MMAs releases its slot. With nine
// slots, tiles 0 and 1 of the next step load into the spare two, its tiles 2..6 into the slots
// released first, and tiles 0 and 6 of this step are the next spare ones. A step's slots are packed
// four bits each.
__device__ __forceinline__ uint32_t next_slots(uint32_t prev2, uint32_t prev1) {
    auto at = [](uint32_t m, int t) { return (m >> (4 * t)) & 15u; };
    return at(prev2, 0) | at(prev2, 6) << 4 | at(prev1, 3) << 8 | at(prev1, 2) << 12 | at(prev1, 4) << 16 |
           at(prev1, 1) << 20 | at(prev1, 5) << 24;
}
constexpr uint32_t kSlots0 = 0x6543210u, kSlotsBefore = 0x8000007u;

// Persistent, one CTA of 576 threads per SM: warp 0 loads the digit tiles by TMA, warp 1 issues
// the MMAs, warps 2..17 are the epilogue. TMEM holds seven accumulators of BN columns (448 of
// 512 at BN = 64), so they are not double-buffered as a whole; each has its own full / empty
// barrier instead. Taking the digits in order makes accumulator d complete with tile d of the
// last K step and first needed again with tile ceil(d/2) of the next sum, so the epilogue
// drains them in order d = 0..6 while the MMAs run on.
//
// A in tensor memory (tcgen05.cp of the seven digits per K = 16 step, where an MMA does not read
// 128 rows of shared memory each time) needs the readers of those columns to be done before the
// next copy: copies are ordered before later MMAs, not after earlier ones. An inverse at 255^3,
// with sums of 128 terms in every accumulator, took 1370 us as it is, with the waits and one set of
// columns in two groups 1419, eight slots in turn 1447, tiles of 48 columns and three sets 1634,
// of 32 and four sets 1899. (Emptying accumulators 2 to 4 every 64 terms takes 1370 to 1448.)
template <int BN, int MODE, int EPI>
__global__ void __maxnreg__(96) k_modeprod_f64tc(const ProdArgs g) {
    if (g.e.done != nullptr && *(volatile const int *)g.e.done) return;
    constexpr uint32_t a_bytes = BM * BK * 2;
    constexpr uint32_t kSlot = slot_bytes<BN>();
    constexpr int NC = BN / (kEpiWarps / 4);   // columns per epilogue thread
    static_assert(kDig * BN <= 512, "TMEM columns");

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t ctrl = base + kSlots * kSlot;
    auto full_bar = [&](uint32_t s) { return ctrl + 8u * s; };
    auto empty_bar = [&](uint32_t s) { return ctrl + 80u + 8u * s; };
    auto tfull_bar = [&](int d) { return ctrl + 160u + 8u * d; };
    auto tempty_bar = [&](int d) { return ctrl + 224u + 8u * d; };
    const uint32_t mma_done_bar = ctrl + 288u;
    const uint32_t tmem_slot = ctrl + 296u;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem_raw + (ctrl + 300u - raw));
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSlots; ++s) {
            ptx::mbar_init(full_bar(s), 1);
            ptx::mbar_init(empty_bar(s), 1);
        }
        for (int d = 0; d < kDig; ++d) {
            ptx::mbar_init(tfull_bar(d), 1);
            ptx::mbar_init(tempty_bar(d), kEpiWarps);
        }
        ptx::mbar_init(mma_done_bar, 1);
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::fence_proxy_async();
        ptx::prefetch_tensormap(g.amap);
        ptx::prefetch_tensormap(g.bmap);
    }
    if (warp == 1) {
        ptx::tmem_alloc(tmem_slot, kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t *>(smem_raw + (tmem_slot - raw));

    auto mid = [](int d) { return d >= kMid0 && d <= kMid1; };   // accumulators emptied every K step
    constexpr int kHalves = (MODE == MD_BWD) ? 2 : 1;   // halves summed by one tile
    const int tpm = (MODE == MD_FWD ? 2 : 1) * g.ntn;   // tiles per 128 rows
    const int steps = g.Kp / BK;                        // K steps of a half
    constexpr int kSegSteps = kSegK / BK;
    static_assert(2 * kSegK <= 256 && (kMid1) * BK <= 256, "digit sums within 2^24 up to d = 3");

    if (warp == 0 && lane == 0) {
        uint32_t phase = 0, armed = 0;   // per slot: the next load's phase; loaded at least once
        uint32_t sl1 = kSlotsBefore, sl = kSlots0;
        bool ok = true;
        for (int t = blockIdx.x; ok && t < g.ntiles; t += gridDim.x) {
            const int mt = t / tpm, r = t % tpm;
            const int n0 = (r % g.ntn) * BN;
            const int x0 = (MODE == MD_FWD) ? (r / g.ntn) * g.Kp : 0;
            for (int k = 0; ok && k < kHalves * steps; ++k) {
                for (int d = 0; d < kDig; ++d) {
                    const uint32_t s = (sl >> (4 * d)) & 15u;
                    if (!ptx::wait_bar(empty_bar(s), ((phase >> s) & 1u) ^ 1u, abort_flag, g.e.err)) {
                        ok = false;
                        break;
                    }
                    const uint32_t st = base + s * kSlot;
                    ptx::mbar_arrive_expect_tx(full_bar(s), kSlot);
                    ptx::tma_load_3d(st, g.amap, full_bar(s), x0 + k * BK, mt * BM, d);
                    ptx::tma_load_3d(st + a_bytes, g.bmap, full_bar(s), x0 + k * BK, n0, d);
                    phase ^= 1u << s;
                    armed |= 1u << s;
                }
                const uint32_t nx = next_slots(sl1, sl);
                sl1 = sl;
                sl = nx;
            }
        }
        if (!ok)
            for (int i = 0; i < kSlots; ++i)
                if (armed & (1u << i)) ptx::drain_bar(full_bar(i), ((phase >> i) & 1u) ^ 1u);
    } else if (warp == 1) {
        constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((BM >> 4) << 24);   // FP16, FP32 sums
        auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
            return __all_sync(0xffffffffu, ptx::wait_bar(bar, parity, abort_flag, g.e.err));
        };
        uint32_t phase = 0, tp = 0, tm = 0;
        uint32_t sl1 = kSlotsBefore, sl = kSlots0;
        bool ok = true;
        for (int t = blockIdx.x; ok && t < g.ntiles; t += gridDim.x) {
            for (int step = 0; ok && step < kHalves * steps; ++step) {
                const int hs = (MODE == MD_BWD && step >= steps) ? step - steps : step;   // step within its half
                const bool first = hs % kSegSteps == 0;
                const bool last = hs % kSegSteps == kSegSteps - 1 || hs == steps - 1;
                const int nk = min(BK, g.Kt - hs * BK) / 16;   // K = 16 MMAs of this step
                uint64_t da[kDig], db[kDig];
#pragma unroll
                for (int i = 0; i < kDig; ++i) {
                    const uint32_t st = base + ((sl >> (4 * i)) & 15u) * kSlot;
                    da[i] = ptx::smem_desc_kmajor(st, BK * 2, 2);
                    db[i] = ptx::smem_desc_kmajor(st + a_bytes, BK * 2, 2);
                }
#pragma unroll
                for (int i = 0; i < kDig; ++i) {
                    const uint32_t s = (sl >> (4 * i)) & 15u;
                    if (ok) ok = wait(full_bar(s), (phase >> s) & 1u);
                    phase ^= 1u << s;
#pragma unroll
                    for (int d = 2 * i - 1; d <= 2 * i && i <= 3; ++d)   // these start with this tile
                        if (ok && d >= 0 && (first || mid(d))) ok = wait(tempty_bar(d), (mid(d) ? tm : tp) ^ 1u);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    constexpr int jmax[kDig] = {0, 1, 2, 3, 2, 1, 0};   // min(i, 6 - i)
                    if (ptx::elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            if (kk >= nk) break;
#pragma unroll
                            for (int j = 0; j <= jmax[i]; ++j) {
                                const uint32_t acc = tmem_base + (uint32_t)((i + j) * BN);
                                // the first product into accumulator i + j overwrites it
                                const uint32_t keep =
                                    (kk == 0 && i == (i + j + 1) / 2) ? (first || mid(i + j) ? 0u : 1u) : 1u;
                                ptx::mma_f16(acc, da[i] + 2 * kk, db[j] + 2 * kk, idesc, keep);
                                if (j != i) ptx::mma_f16(acc, da[j] + 2 * kk, db[i] + 2 * kk, idesc, 1u);
                            }
                        }
                        if (last || mid(i)) ptx::mma_commit(tfull_bar(i));
                        // tiles released by this one (see next_slots)
                        if (i >= 3) ptx::mma_commit(empty_bar(s));
                        if (i > 3) ptx::mma_commit(empty_bar((sl >> (4 * (6 - i))) & 15u));
                    }
                    __syncwarp();
                }
                if (last) tp ^= 1u;
                tm ^= 1u;
                const uint32_t nx = next_slots(sl1, sl);
                sl1 = sl;
                sl = nx;
            }
        }
        if (ptx::elect_one()) ptx::mma_commit(mma_done_bar);
        __syncwarp();
        ptx::drain_bar(mma_done_bar, 0);
    } else if (warp >= 2) {
        const int quad = warp & 3, part = (warp - 2) >> 2;
        const int row = quad * 32 + lane;
        const uint32_t tcol = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(part * NC);
        uint32_t tp = 0, tm = 0;
        bool ok = true;
        // acc += sum_d C_d 2^(38-9d) of the next sum of `sub` K steps; false after a timeout (warp-uniform)
        auto drain_sum = [&](long long(&acc)[NC], int sub) -> bool {
            float c5[NC];
            for (int u = 1; u <= sub; ++u) {
#pragma unroll
                for (int d = 0; d < kDig; ++d) {
                    if (u < sub && !mid(d)) continue;
                    const bool ready = ptx::wait_bar(tfull_bar(d), mid(d) ? tm : tp, abort_flag, g.e.err);
                    if (!__all_sync(0xffffffffu, ready)) return false;
                    ptx::tc_fence_after();
                    uint32_t r[NC];
                    tmem_ld<NC>(tcol + (uint32_t)(d * BN), r);
                    ptx::tmem_ld_wait();
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(tempty_bar(d));
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const float v = __uint_as_float(r[c]);
                        if (d == 0)
                            acc[c] += (long long)((unsigned long long)(unsigned)__float2int_rn(v) << 38);
                        else if (d < 5)
                            acc[c] = mad_wide(__float2int_rn(v), 1 << (38 - kBits * d), acc[c]);
                        else if (d == 5)
                            c5[c] = v;
                        else
                            acc[c] += (long long)__float2int_rn(fmaf(v, 0x1p-9f, c5[c]) * 0x1p-7f);
                    }
                }
                tm ^= 1u;
            }
            tp ^= 1u;
            return true;
        };
        for (int t = blockIdx.x; ok && t < g.ntiles; t += gridDim.x) {
            const int mt = t / tpm, r = t % tpm;
            const int n0 = (r % g.ntn) * BN + part * NC;
            const int h0 = (MODE == MD_FWD) ? r / g.ntn : 0;
            long long p[NC], q[(MODE == MD_BWD) ? NC : 1];
#pragma unroll
            for (int c = 0; c < NC; ++c) p[c] = 0;
            for (int at = 0; ok && at < steps; at += kSegSteps) ok = drain_sum(p, min(kSegSteps, steps - at));
            if constexpr (MODE == MD_BWD) {
#pragma unroll
                for (int c = 0; c < NC; ++c) q[c] = 0;
                for (int at = 0; ok && at < steps; at += kSegSteps) ok = drain_sum(q, min(kSegSteps, steps - at));
            }
            if (!ok) break;
            const int ml = mt * BM + row;
            if (ml < g.rows) {
                const int m = g.m0 + ml;
                const int2 ea2 = g.ea[ml];
                const int ea = h0 ? ea2.y : ea2.x;
                const bool bad = ea2.x == kNonFinite || ea2.y == kNonFinite;
                double rowlam = 0.0;   // the divisor without lambda_k
                if (EPI == EPI_DIVIDE)
                    rowlam = ((g.dim == 3) ? g.e.lam64[m / g.n] + g.e.lam64[m % g.n] : g.e.lam64[m]) + *g.e.shift;
                auto put = [&](int k, double v) {
                    const long long o = (long long)k * g.Mtot + m;
                    if (EPI == EPI_UPDATE)
                        g.out[o] = g.out[o] - g.e.step * v;
                    else
                        g.out[o] = v;
                };
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const int rb = n0 + c;   // B row of this half
                    if (rb >= g.nrow) continue;
                    const int k = (MODE == MD_FWD) ? 2 * rb + h0 : rb;
                    if (MODE == MD_FWD && k >= g.n) continue;
                    const int2 eb2 = __ldg(g.eb + rb);
                    double v, w = 0.0;
                    if (bad) {
                        const double2 pq = dot_fp64<MODE>(g.A + (long long)m * g.n, g.B, g.n, k);
                        v = (MODE == MD_BWD) ? pq.x + pq.y : pq.x;
                        w = pq.x - pq.y;
                        if (EPI == EPI_DIVIDE) v /= __ldg(g.e.lam64 + k) + rowlam;
                    } else if constexpr (MODE == MD_BWD) {
                        v = scaled(p[c] + q[c], ea + eb2.x);
                        w = scaled(p[c] - q[c], ea + eb2.x);
                    } else if constexpr (EPI == EPI_DIVIDE) {
                        v = divided(p[c], ea + (h0 ? eb2.y : eb2.x), __ldg(g.e.lam64 + k) + rowlam);
                    } else {
                        v = scaled(p[c], ea + (h0 ? eb2.y : eb2.x));
                    }
                    put(k, v);
                    if (MODE == MD_BWD && rb < (g.n >> 1)) put(g.n - 1 - rb, w);
                }
            }
            __syncwarp();
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, kTmemCols);
    }
}

size_t smem_for(int BN) { return 1024 + (size_t)kSlots * (BM + BN) * BK * 2 + kCtrlBytes; }

template <int KIND>
int slice_kind(const SliceArgs &a, cudaStream_t s) {
    const int grid = (a.rows + 7) / 8, nst = (a.Kp + 63) / 64;
    if (nst <= 1)
        k_slice_rows<KIND, 1><<<grid, 256, 0, s>>>(a);
    else if (nst <= 2)
        k_slice_rows<KIND, 2><<<grid, 256, 0, s>>>(a);
    else if (nst <= 4)
        k_slice_rows<KIND, 4><<<grid, 256, 0, s>>>(a);
    else if (nst <= 8)
        k_slice_rows<KIND, 8><<<grid, 256, 0, s>>>(a);
    else
        k_slice_rows<KIND, 16><<<grid, 256, 0, s>>>(a);
    QN_CUDA(cudaGetLastError());
    return QN_OK;
}

int slice(int kind, const SliceArgs &a, cudaStream_t s) {
    switch (kind) {
        case SL_DENSE: return slice_kind<SL_DENSE>(a, s);
        case SL_FWD: return slice_kind<SL_FWD>(a, s);
        case SL_PARITY: return slice_kind<SL_PARITY>(a, s);
        default: return slice_kind<SL_ROWS>(a, s);
    }
}

template <int BN, int MODE, int EPI>
int launch_one(const ProdArgs &g, int grid, cudaStream_t s) {
    k_modeprod_f64tc<BN, MODE, EPI><<<grid, kThreads, smem_for(BN), s>>>(g);
    QN_CUDA(cudaGetLastError());
    return QN_OK;
}

template <int BN>
int launch_bn(int mode, Epi epi, const ProdArgs &g, int grid, cudaStream_t s) {
    if (mode == MD_FWD)
        return epi == EPI_DIVIDE ? launch_one<BN, MD_FWD, EPI_DIVIDE>(g, grid, s)
                                 : launch_one<BN, MD_FWD, EPI_STORE>(g, grid, s);
    if (mode == MD_BWD)
        return epi == EPI_UPDATE ? launch_one<BN, MD_BWD, EPI_UPDATE>(g, grid, s)
                                 : launch_one<BN, MD_BWD, EPI_STORE>(g, grid, s);
    if (epi == EPI_DIVIDE) return launch_one<BN, MD_DENSE, EPI_DIVIDE>(g, grid, s);
    if (epi == EPI_UPDATE) return launch_one<BN, MD_DENSE, EPI_UPDATE>(g, grid, s);
    return launch_one<BN, MD_DENSE, EPI_STORE>(g, grid, s);
}

template <int BN, int MODE, int EPI>
int opt_in() {
    QN_CUDA(cudaFuncSetAttribute(k_modeprod_f64tc<BN, MODE, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem_for(BN)));
    return QN_OK;
}

template <int BN>
int opt_in_bn() {
    int rc = opt_in<BN, MD_FWD, EPI_STORE>();
    if (rc == QN_OK) rc = opt_in<BN, MD_FWD, EPI_DIVIDE>();
    if (rc == QN_OK) rc = opt_in<BN, MD_BWD, EPI_STORE>();
    if (rc == QN_OK) rc = opt_in<BN, MD_BWD, EPI_UPDATE>();
    if (rc == QN_OK) rc = opt_in<BN, MD_DENSE, EPI_STORE>();
    if (rc == QN_OK) rc = opt_in<BN, MD_DENSE, EPI_DIVIDE>();
    if (rc == QN_OK) rc = opt_in<BN, MD_DENSE, EPI_UPDATE>();
    return rc;
}

// Digits [kDig][rows][ld] as a 3-D FP16 tensor read in 64 x box_rows boxes of one digit.
int encode_digits(CUtensorMap *m, const __half *ptr, int ld, int rows, int box_rows) {
    cuuint64_t dims[3] = {(cuuint64_t)ld, (cuuint64_t)rows, (cuuint64_t)kDig};
    cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)rows * ld * 2};
    cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1};
    return tc_encode_tiled(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, ptr, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

}  // namespace

// The digits of both matrices, and room for the digits of one chunk of rows of A.
struct F64TcPlan {
    int n, dim, split, Mtot, Kp, ld, nrow, BN, ntn, chunk, num_sms;
    __half *adig, *bdig[2];      // bdig[0]: forward (S^{-1}), [1]: backward (S)
    int2 *ea, *eb[2];
    const double *B[2];
    CUtensorMap *maps;           // device: A, forward B, backward B
};

void f64tc_destroy(F64TcPlan *p) {
    if (p == nullptr) return;
    cudaFree(p->adig);
    cudaFree(p->ea);
    for (int b = 0; b < 2; ++b) {
        cudaFree(p->bdig[b]);
        cudaFree(p->eb[b]);
    }
    cudaFree(p->maps);
    delete p;
}

// Below about 6 million multiply-adds per product (2-D n = 181, 3-D n = 49) the two launches of a
// product cost more than the FP64 pipe: an inverse takes 54 against 85 us at 130^2 and 46 against
// 89 us at 32^3; it is even at 200^2 (98 / 91 us) and 48^3 (104 / 103 us), and 207 / 97 us at
// 255^2, 345 / 111 us at 64^3.
bool f64tc_pays(int n, int dim) {
    double work = n;
    for (int a = 0; a < dim; ++a) work *= n;
    return work > 6.0e6;
}

int f64tc_create(F64TcPlan **out, int n, int dim, int split, const double *S, const double *Si, int num_sms) {
    *out = nullptr;
    F64TcPlan *p = new (std::nothrow) F64TcPlan();
    if (p == nullptr) return QN_ENOMEM;
    memset(p, 0, sizeof(*p));
    p->n = n;
    p->dim = dim;
    p->split = split;
    p->num_sms = num_sms;
    p->Mtot = (dim == 3) ? n * n : n;
    p->nrow = split ? (n + 1) / 2 : n;
    const int kt = split ? (n + 1) / 2 : n;      // contraction length of a half
    p->Kp = (kt + BK - 1) / BK * BK;
    p->ld = (split ? 2 : 1) * p->Kp;
    const int mtiles = (p->Mtot + BM - 1) / BM;
    // 64 columns unless a half has fewer rows, or narrower tiles are needed to occupy the SMs
    p->BN = 64;
    while (p->BN > 16 && (p->nrow <= p->BN / 2 ||
                          (long long)mtiles * (split ? 2 : 1) * ((p->nrow + p->BN - 1) / p->BN) * 2 <= num_sms))
        p->BN /= 2;
    p->ntn = (p->nrow + p->BN - 1) / p->BN;
    // rows per pass: the digits take 14 bytes per padded value, at most 2 GiB of them at a time
    // (QN_DIGIT_MB: another limit; all rows up to 520^3; passes of 96 MB, which would stay in L2,
    // lost more to the tails of their launches than they saved: 1.87 against 1.63 ms per 255^3
    // inverse), and less where the device has no room for that
    const char *em = getenv("QN_DIGIT_MB");
    const long long mb = (em && atoll(em) >= 1 && atoll(em) <= 2048) ? atoll(em) : 2048;
    long long ct = (mb << 20) / ((long long)kDig * p->ld * 2 * BM);
    if (ct < 1) ct = 1;
    if (ct > mtiles) ct = mtiles;

    auto fail = [&](int rc) {
        f64tc_destroy(p);
        return rc;
    };
    int rc = opt_in_bn<64>();
    if (rc == QN_OK) rc = opt_in_bn<32>();
    if (rc == QN_OK) rc = opt_in_bn<16>();
    if (rc != QN_OK) return fail(rc);
    CUtensorMap h[3];
    while (cudaMalloc(&p->adig, (size_t)kDig * ct * BM * p->ld * 2) != cudaSuccess) {
        p->adig = nullptr;
        cudaGetLastError();
        if (ct == 1) {
            set_error("qn_ctx_create: out of device memory for the FP64 products' digits");
            return fail(QN_ENOMEM);
        }
        ct = (ct + 1) / 2;
    }
    p->chunk = (int)ct * BM;
    if (cudaMalloc(&p->ea, sizeof(int2) * p->chunk) != cudaSuccess ||
        cudaMalloc(&p->maps, sizeof(h)) != cudaSuccess) {
        set_error("qn_ctx_create: out of device memory for the FP64 products' digits");
        return fail(QN_ENOMEM);
    }
    rc = encode_digits(&h[0], p->adig, p->ld, p->chunk, BM);
    for (int b = 0; b < 2 && rc == QN_OK; ++b) {
        if (cudaMalloc(&p->bdig[b], (size_t)kDig * p->nrow * p->ld * 2) != cudaSuccess ||
            cudaMalloc(&p->eb[b], sizeof(int2) * p->nrow) != cudaSuccess) {
            set_error("qn_ctx_create: out of device memory for the FP64 products' digits");
            return fail(QN_ENOMEM);
        }
        p->B[b] = b ? S : Si;
        // sums longer than kSegK terms: as much headroom in B as the 64-bit total needs
        const int terms = (split && b == 0) ? kt : n;
        SliceArgs a{};
        a.src = p->B[b];
        a.dig = p->bdig[b];
        a.ex = p->eb[b];
        a.slice_stride = (long long)p->nrow * p->ld;
        a.rows = p->nrow;
        a.n = n;
        a.Kp = p->Kp;
        a.ld = p->ld;
        for (int t = kTotal; t < terms; t *= 2) a.extra++;
        rc = slice(!split ? SL_DENSE : (b == 0 ? SL_ROWS : SL_PARITY), a, nullptr);
        if (rc == QN_OK) rc = encode_digits(&h[1 + b], p->bdig[b], p->ld, p->nrow, p->BN);
    }
    if (rc != QN_OK) return fail(rc);
    if (cudaMemcpy(p->maps, h, sizeof(h), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaStreamSynchronize(nullptr) != cudaSuccess) {
        set_error("qn_ctx_create: preparing the FP64 products' digits failed");
        return fail(QN_ECUDA);
    }
    *out = p;
    return QN_OK;
}

int launch_modeprod_f64tc(const F64TcPlan *p, bool forward, const double *A, double *out, Epi epi, const EpiArgs &e,
                          cudaStream_t s, int *launches) {
    const int b = forward ? 0 : 1;
    const int mode = !p->split ? MD_DENSE : (forward ? MD_FWD : MD_BWD);
    *launches = 0;
    for (int m0 = 0; m0 < p->Mtot; m0 += p->chunk) {
        const int rows = (p->Mtot - m0 < p->chunk) ? p->Mtot - m0 : p->chunk;
        SliceArgs a{};
        a.src = A;
        a.dig = p->adig;
        a.ex = p->ea;
        a.done = e.done;
        a.slice_stride = (long long)p->chunk * p->ld;
        a.rows = rows;
        a.n = p->n;
        a.Kp = p->Kp;
        a.ld = p->ld;
        a.row0 = m0;
        int rc = slice(!p->split ? SL_DENSE : (forward ? SL_FWD : SL_PARITY), a, s);
        if (rc != QN_OK) return rc;
        ProdArgs g{};
        g.amap = p->maps;
        g.bmap = p->maps + 1 + b;
        g.ea = p->ea;
        g.eb = p->eb[b];
        g.A = A;
        g.B = p->B[b];
        g.out = out;
        g.rows = rows;
        g.m0 = m0;
        g.Mtot = p->Mtot;
        g.n = p->n;
        g.dim = p->dim;
        g.Kp = p->Kp;
        g.Kt = (p->split ? (p->n + 1) / 2 : p->n) + 15 & ~15;
        g.nrow = p->nrow;
        g.ntn = p->ntn;
        g.ntiles = (rows + BM - 1) / BM * p->ntn * (mode == MD_FWD ? 2 : 1);
        g.e = e;
        const int grid = g.ntiles < p->num_sms ? g.ntiles : p->num_sms;
        rc = p->BN == 64 ? launch_bn<64>(mode, epi, g, grid, s)
                         : (p->BN == 32 ? launch_bn<32>(mode, epi, g, grid, s) : launch_bn<16>(mode, epi, g, grid, s));
        if (rc != QN_OK) return rc;
        *launches += 2;
    }
    return QN_OK;
}

}  // namespace qn
