// Training kernels of the warm-start network (forward, loss, backward) for up to eight modes per
// axis. Included by qn_net.cu.
//
// An activation of 8 x 64^3 nodes is 134 MB in BF16 and a gradient 268 MB in FP32, so nothing is
// read twice; what is left waits on instruction issue (FP32 multiply-adds of the transforms,
// 43 to 66 %) and shared memory, at 1 to 3 TB/s. Per block l the kernels are
//   k_tr_analysis   one read of h_l (or of dh and z_l): the x and y analysis of a quarter of a z
//                   plane per CTA, which writes M^2 x 32 sums instead of the x-analysed tensor;
//   k_tr_mix        z analysis and channel mixing, one CTA per mode (backward: both gradients);
//   k_tr_fwd        z_l = synthesis(g) + h_l W + b and h_{l+1}; the spectral term is formed in
//                   registers per row. The last block also projects, takes the loss and its
//                   gradient, and sums the projection's gradients;
//   k_tr_bwd        dz = dh gelu'(z) again from dh and z (cheaper than storing dz), dW, db and
//                   dh_prev = dz W^T + synthesis(dhh), in place of dh.
// The lifted input h_0 = f wl + bl is formed where it is read (4 instead of 64 bytes a node), as
// are the last block's dh = dout wp; block 0's dh_prev goes straight into the lift's gradients.
//
// The 32 x 32 channel products run on the tensor cores (mma.sync: register operands, 16 nodes of
// one row per warp step) without losing FP32: a BF16 activation is one operand level, an FP32
// operand three (x = x0 + x1 + x2, 24 bits), and the products down to 2^-24 of the leading one are
// kept (3 for h W and h^T dz, 6 for dz W^T). Sums over nodes are added outside the tensor core,
// in FP32 with rounding to nearest. Lanes own eight channels (8t .. 8t+7, t = lane & 3) of rows
// g and g + 8 (g = lane >> 2): a permutation of the MMA's k and n indices that makes every load
// and store 16 bytes wide.
//
// 10.4 -> 2.26 ms per loss + gradient at 64^3, batch 8.
#pragma once

#include <cuda_bf16.h>

namespace qn {
namespace {

constexpr int kTrRows = 16;   // rows of one z plane per work item

// gelu(x) = x s and gelu'(x) = s + 2 x s (1 - s) u', s = sigmoid(2u) = (1 + tanh u)/2, u = sqrt(2/pi) (x +
// 0.044715 x^3): the tanh form rewritten through the smaller of s and 1 - s, r = 1/(1 + exp 2|u|), so
// that nothing cancels, and for |u| < 0.6 (where r would round 1/2 first) through tanh u as an odd
// polynomial, fitted to it within 9e-8 relative. RMS error against 64 bits, with tanhf and so:
// gelu' 2.15e-8, 2.16e-8 on |x| < 0.5; 5.1e-8, 4.3e-8 on [1.6, 2]; 18.6e-8, 3.8e-8 on [3, 5]; 9.6e-8, 0.7e-8
// on [-4, -2]; gelu 6.6e-9, 6.5e-9; 5.3e-8, 3.6e-8; 14.5e-8, 11.0e-8; 26.5e-9, 3.2e-9 on the same. Two
// values at a time, in packed FP32 arithmetic: 2.26 ms per loss + gradient at 64^3, batch 8, against
// 2.13 with s = 1 / (1 + exp(-2u)), whose gelu' was off by 3.2e-8 and 6.1e-8 on |x| < 0.5 and
// [0.5, 2], and 2.75 with tanhf on [-0.5, 2].
struct TrSigmoid {
    float2 x2, t, r;
    bool small_x, small_y;
    __device__ __forceinline__ explicit TrSigmoid(float2 x) {
        x2 = __fmul2_rn(x, x);
        const float2 u = __fmul2_rn(two(kGeluC), __ffma2_rn(__fmul2_rn(two(0.044715f), x2), x, x)), z = __fmul2_rn(u, u);
        float2 p = __ffma2_rn(two(0.0155801f), z, two(-0.0521884f));
        p = __ffma2_rn(__ffma2_rn(p, z, two(0.13312598f)), z, two(-0.33332564f));
        t = __ffma2_rn(__fmul2_rn(u, z), p, u);
        const float2 w = __fmul2_rn(two(2.8853900818f), u);   // 2 u log2(e)
        r.x = inverse(1.0f + exp_2(fabsf(w.x)));
        r.y = inverse(1.0f + exp_2(fabsf(w.y)));
        small_x = fabsf(u.x) < 0.6f;
        small_y = fabsf(u.y) < 0.6f;
    }
    static __device__ __forceinline__ float exp_2(float v) {   // v >= 0: no subnormal results
        float e;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(v));
        return e;
    }
    static __device__ __forceinline__ float inverse(float v) {
        float e;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(v));
        return e;
    }
    static __device__ __forceinline__ float2 two(float v) { return make_float2(v, v); }
    __device__ __forceinline__ float2 half_plus() const { return __ffma2_rn(two(0.5f), t, two(0.5f)); }   // s, small u
};

__device__ __forceinline__ float2 tr_gelu(float2 x) {
    const TrSigmoid g(x);
    const float2 a = __fmul2_rn(x, g.half_plus()), b = __fmul2_rn(x, g.r);
    // x (1 - r) with one rounding (an infinite x stays infinite)
    return make_float2(g.small_x ? a.x : (x.x < 0.0f ? b.x : fmaf(-fminf(x.x, 1e38f), g.r.x, x.x)),
                       g.small_y ? a.y : (x.y < 0.0f ? b.y : fmaf(-fminf(x.y, 1e38f), g.r.y, x.y)));
}

__device__ __forceinline__ float2 tr_gelu_grad(float2 x) {
    const TrSigmoid g(x);
    const float2 a = g.half_plus(), qa = __ffma2_rn(__fmul2_rn(TrSigmoid::two(-0.25f), g.t), g.t, TrSigmoid::two(0.25f));
    const float2 qb = __ffma2_rn(make_float2(-g.r.x, -g.r.y), g.r, g.r);   // s (1 - s)
    const float2 q = make_float2(g.small_x ? qa.x : qb.x, g.small_y ? qa.y : qb.y);
    const float2 s = make_float2(g.small_x ? a.x : (x.x < 0.0f ? g.r.x : 1.0f - g.r.x),
                                 g.small_y ? a.y : (x.y < 0.0f ? g.r.y : 1.0f - g.r.y));
    const float2 du = __fmul2_rn(TrSigmoid::two(kGeluC), __ffma2_rn(TrSigmoid::two(3.0f * 0.044715f), g.x2, TrSigmoid::two(1.0f)));
    return __ffma2_rn(__fmul2_rn(__fmul2_rn(TrSigmoid::two(2.0f), x), q), du, s);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}
__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// The next BF16 level of a pair; the arguments keep what it leaves.
__device__ __forceinline__ uint32_t take_level(float &a, float &b) {
    const uint32_t v = pack_bf16(a, b);
    a -= bf_lo(v);
    b -= bf_hi(v);
    return v;
}

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t trans8x8(uint32_t v) {
    uint32_t r;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}

// 16 or 4 bytes global -> shared without a register; `ok` false writes zeros.
__device__ __forceinline__ void copy16(void *dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(ok ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void copy4(void *dst, const void *src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(ok ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// What a step of eight nodes reads, eight channels a lane: the block's input (stored BF16, or
// lifted from f), or dz in backward (dh gelu'(z), or the last block's dout wp). One lane's
// pieces go through its own slots of a shared-memory ring (it alone writes and reads them, so no
// barrier is needed), a fixed number of steps ahead: the loads of a register pipeline that deep
// would not fit, and with one step in flight these kernels waited on memory most of the time.
enum TrSrc : int { TR_H = 0, TR_LIFT = 1, TR_DZ = 2, TR_DOUT = 3 };

struct TrIn {
    const __nv_bfloat16 *h, *z;
    const float *f, *wl, *bl;   // lift
    const float *dh;            // gradient of the block's output, or dout (TR_DOUT)
    const float *wp;
};

// 16-byte pieces of one lane and one step in the ring
__host__ __device__ constexpr int tr_pieces(int src) { return src == TR_DZ ? 3 : 1; }

template <int SRC>
struct TrLoad {
    TrIn in;
    float w[8], b[8];
    int t;
    __device__ __forceinline__ TrLoad(const TrIn &i, int t_) : in(i), t(t_) {
        if (SRC == TR_LIFT || SRC == TR_DOUT)
            for (int j = 0; j < 8; ++j) {
                w[j] = (SRC == TR_LIFT ? i.wl : i.wp)[8 * t_ + j];
                b[j] = SRC == TR_LIFT ? i.bl[8 * t_ + j] : 0.0f;
            }
    }
    // slot: this lane's first piece of the step; pieces are 32 lanes apart
    __device__ __forceinline__ void issue(uint4 *slot, long long p, bool ok) const {
        if (!ok) p = 0;
        if (SRC == TR_H) {
            copy16(slot, in.h + p * 32 + 8 * t, ok);
        } else if (SRC == TR_DZ) {
            copy16(slot, in.dh + p * 32 + 8 * t, ok);
            copy16(slot + 32, in.dh + p * 32 + 8 * t + 4, ok);
            copy16(slot + 64, in.z + p * 32 + 8 * t, ok);
        } else {
            copy4(slot, (SRC == TR_LIFT ? in.f : in.dh) + p, ok);
        }
    }
    // BF16 pairs of the input (SRC H, LIFT); nodes past the row's end are zero
    __device__ __forceinline__ uint4 octet(const uint4 *slot, bool ok) const {
        if (SRC == TR_H) return *slot;
        const float x = *reinterpret_cast<const float *>(slot);
        uint4 v;
        v.x = pack_bf16(fmaf(x, w[0], b[0]), fmaf(x, w[1], b[1]));
        v.y = pack_bf16(fmaf(x, w[2], b[2]), fmaf(x, w[3], b[3]));
        v.z = pack_bf16(fmaf(x, w[4], b[4]), fmaf(x, w[5], b[5]));
        v.w = pack_bf16(fmaf(x, w[6], b[6]), fmaf(x, w[7], b[7]));
        return ok ? v : make_uint4(0, 0, 0, 0);
    }
    __device__ __forceinline__ void values(const uint4 *slot, bool ok, float2 (&v)[4]) const {
        if (SRC == TR_H || SRC == TR_LIFT) {
            const uint4 o = octet(slot, ok);
            v[0] = make_float2(bf_lo(o.x), bf_hi(o.x));
            v[1] = make_float2(bf_lo(o.y), bf_hi(o.y));
            v[2] = make_float2(bf_lo(o.z), bf_hi(o.z));
            v[3] = make_float2(bf_lo(o.w), bf_hi(o.w));
        } else if (SRC == TR_DOUT) {
            const float d = *reinterpret_cast<const float *>(slot);
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = make_float2(d * w[2 * j], d * w[2 * j + 1]);
        } else {   // zeros past the row's end: dh is zero there
            const float4 d0 = *reinterpret_cast<const float4 *>(slot), d1 = *reinterpret_cast<const float4 *>(slot + 32);
            const uint4 o = slot[64];
            v[0] = __fmul2_rn(make_float2(d0.x, d0.y), tr_gelu_grad(make_float2(bf_lo(o.x), bf_hi(o.x))));
            v[1] = __fmul2_rn(make_float2(d0.z, d0.w), tr_gelu_grad(make_float2(bf_lo(o.y), bf_hi(o.y))));
            v[2] = __fmul2_rn(make_float2(d1.x, d1.y), tr_gelu_grad(make_float2(bf_lo(o.z), bf_hi(o.z))));
            v[3] = __fmul2_rn(make_float2(d1.z, d1.w), tr_gelu_grad(make_float2(bf_lo(o.w), bf_hi(o.w))));
        }
    }
};

// The steps of one warp: rows y0, y0 + dy, .. below y1 of one plane, `per` x steps each.
struct TrSteps {
    long long plane;   // first row's index of the plane
    int y, x, dy, y1, dx, G;
    __device__ __forceinline__ bool done() const { return y >= y1; }
    __device__ __forceinline__ long long row() const { return (plane + y) * G; }
    __device__ __forceinline__ void next() {
        x += dx;
        if (x >= G) {
            x = 0;
            y += dy;
        }
    }
};

constexpr int kTrDepthA = 8;   // steps of eight nodes in flight per warp (analysis)
constexpr int kTrParts = 4;    // CTAs per plane

template <int MP, int SRC>
__host__ __device__ constexpr int tr_analysis_smem() {
    const int ring = 8 * kTrDepthA * tr_pieces(SRC) * 32 * 16, sums = 8 * MP * MP * 32 * 4;
    return (ring > sums ? ring : sums) + 256 * MP * 8;
}

// t2[plane][part][ky][kx][c] = sum_y sum_x B[y][ky] B[x][kx] v[plane][y][x][c] over the part's
// rows, kTrParts CTAs per plane (b, z). basis: [G][M]; MP = M rounded up to even (the extra mode
// is zero).
template <int MP, int SRC>
__global__ void __launch_bounds__(256, 2) k_tr_analysis(const TrIn in, const float *__restrict__ basis, int G, int M,
                                                        float *__restrict__ t2) {
    extern __shared__ __align__(16) uint8_t tr_smem[];
    float2 *sB = reinterpret_cast<float2 *>(tr_smem);               // (b, b) pairs: packed multiply-adds
    uint4 *ring = reinterpret_cast<uint4 *>(tr_smem + 256 * MP * 8);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    constexpr int kPieces = tr_pieces(SRC);
    uint4 *mine = ring + warp * kTrDepthA * kPieces * 32 + lane;
    const TrLoad<SRC> load(in, t);
    const int plane = blockIdx.x / kTrParts, part = blockIdx.x % kTrParts;
    TrSteps ahead{(long long)plane * G, G * part / kTrParts + warp, 0, 8, G * (part + 1) / kTrParts, 8, G};
    TrSteps at = ahead;
    int slot = 0;
    auto issue = [&](int sl) {
        if (!ahead.done()) load.issue(mine + sl * kPieces * 32, ahead.row() + ahead.x + g, ahead.x + g < G);
        ahead.next();
        copy_commit();
    };
#pragma unroll
    for (int i = 0; i < kTrDepthA - 1; ++i) issue(i);
    for (int e = threadIdx.x; e < MP * G; e += 256) {
        const int x = e / MP, k = e % MP;
        const float v = (k < M) ? basis[x * M + k] : 0.0f;
        sB[e] = make_float2(v, v);
    }
    __syncthreads();
    float Q[MP][MP];
#pragma unroll
    for (int a = 0; a < MP; ++a)
#pragma unroll
        for (int k = 0; k < MP; ++k) Q[a][k] = 0.0f;
    while (!at.done()) {
        const int y = at.y;
        float2 acc[MP][4];
#pragma unroll
        for (int k = 0; k < MP; ++k)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[k][j] = make_float2(0.0f, 0.0f);
        for (int x0 = 0; x0 < G; x0 += 8) {
            copy_wait<kTrDepthA - 2>();
            const int x = x0 + g;
            float2 v[4];
            load.values(mine + slot * kPieces * 32, x < G, v);
            issue(slot == 0 ? kTrDepthA - 1 : slot - 1);
            slot = (slot + 1) & (kTrDepthA - 1);
            const float2 *b = sB + min(x, G - 1) * MP;
#pragma unroll
            for (int k = 0; k < MP; ++k) {
                const float2 bk = b[k];
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[k][j] = __ffma2_rn(bk, v[j], acc[k][j]);
            }
        }
        at.x = 0;
        at.y += 8;
        // sum over the eight g lanes, halving the channels a lane holds each time
        const bool u2 = lane & 16, u1 = lane & 8, u0 = lane & 4;
        float T[MP];
#pragma unroll
        for (int k = 0; k < MP; ++k) {
            const float c8[8] = {acc[k][0].x, acc[k][0].y, acc[k][1].x, acc[k][1].y,
                                 acc[k][2].x, acc[k][2].y, acc[k][3].x, acc[k][3].y};
            float r4[4], r2[2];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                r4[j] = (u2 ? c8[j + 4] : c8[j]) + __shfl_xor_sync(0xffffffffu, u2 ? c8[j] : c8[j + 4], 16);
#pragma unroll
            for (int j = 0; j < 2; ++j)
                r2[j] = (u1 ? r4[j + 2] : r4[j]) + __shfl_xor_sync(0xffffffffu, u1 ? r4[j] : r4[j + 2], 8);
            T[k] = (u0 ? r2[1] : r2[0]) + __shfl_xor_sync(0xffffffffu, u0 ? r2[0] : r2[1], 4);
        }
#pragma unroll
        for (int a = 0; a < MP; ++a) {
            const float b = sB[y * MP + a].x;
#pragma unroll
            for (int k = 0; k < MP; ++k) Q[a][k] = fmaf(b, T[k], Q[a][k]);
        }
    }
    copy_wait<0>();
    __syncthreads();
    // the warps' sums in a fixed order; the ring's memory holds them
    float *sQ = reinterpret_cast<float *>(ring);
    const int c = 8 * t + 4 * ((lane >> 4) & 1) + 2 * ((lane >> 3) & 1) + ((lane >> 2) & 1);   // this lane's channel
#pragma unroll
    for (int a = 0; a < MP; ++a)
#pragma unroll
        for (int k = 0; k < MP; ++k) sQ[(warp * MP * MP + a * MP + k) * 32 + c] = Q[a][k];
    __syncthreads();
    float *o = t2 + (long long)blockIdx.x * MP * MP * 32;
    for (int e = threadIdx.x; e < MP * MP * 32; e += 256) {
        float v = 0.0f;
#pragma unroll
        for (int w = 0; w < 8; ++w) v += sQ[w * MP * MP * 32 + e];
        o[e] = v;
    }
}

// The z analysis of one mode k = (kz, ky, kx) for eight samples b0 .. b0 + 7: the warps take
// every eighth plane (all their loads independent: with one warp walking all planes of a sample
// this waited on memory), lane = channel; warp w returns sample b0 + w.
__device__ __forceinline__ float z_analysis(const float *__restrict__ t2, const float *__restrict__ basis, int b0, int B,
                                            int G, int M, int MP, int k, float (*red)[8][32]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int kz = k / (M * M), ky = k / M % M, kx = k % M;
    const int stride = MP * MP * 32;
    __syncthreads();
#pragma unroll 2
    for (int i = 0; i < 8; ++i) {
        if (b0 + i >= B) break;
        const float *p = t2 + (long long)(b0 + i) * G * kTrParts * stride + (ky * MP + kx) * 32 + lane;
        float a = 0.0f;
#pragma unroll 4
        for (int z = warp; z < G; z += 8) {
            const float *q = p + (long long)z * kTrParts * stride;
            float v = 0.0f;
#pragma unroll
            for (int r = 0; r < kTrParts; ++r) v += __ldg(q + r * stride);
            a = fmaf(__ldg(basis + z * M + kz), v, a);
        }
        red[i][warp][lane] = a;
    }
    __syncthreads();
    float s = 0.0f;
    if (b0 + warp < B)
#pragma unroll
        for (int w = 0; w < 8; ++w) s += red[warp][w][lane];
    return s;
}

// hh[b][k][c], g[b][k][o] = sum_i hh[b][k][i] R[k][i][o]; one CTA per mode.
__global__ void __launch_bounds__(256) k_tr_mix(const float *__restrict__ t2, const float *__restrict__ basis, int B,
                                                int G, int M, int MP, const float *__restrict__ R,
                                                float *__restrict__ hh, float *__restrict__ g) {
    __shared__ float red[8][8][32];
    const int lane = threadIdx.x & 31, k = blockIdx.x, K = gridDim.x;
    float r[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) r[i] = __ldg(R + (long long)k * 1024 + i * 32 + lane);
    for (int b0 = 0; b0 < B; b0 += 8) {
        const float v = z_analysis(t2, basis, b0, B, G, M, MP, k, red);
        const int b = b0 + (threadIdx.x >> 5);
        if (b >= B) continue;
        hh[((long long)b * K + k) * 32 + lane] = v;
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < 32; ++i) s = fmaf(__shfl_sync(0xffffffffu, v, i), r[i], s);
        g[((long long)b * K + k) * 32 + lane] = s;
    }
}

// dg = z analysis of dz's sums; dhh[b][k][i] = sum_o dg[b][k][o] R[k][i][o]; dR[k][i][o] =
// sum_b hh[b][k][i] dg[b][k][o] in order of b. One CTA per mode.
__global__ void __launch_bounds__(256) k_tr_mix_bwd(const float *__restrict__ t2, const float *__restrict__ basis, int B,
                                                    int G, int M, int MP, const float *__restrict__ R,
                                                    const float *__restrict__ hh, float *__restrict__ dhh,
                                                    float *__restrict__ dR) {
    __shared__ float sR[32 * 33], sdg[64 * 32], shh[64 * 32], red[8][8][32];
    const int lane = threadIdx.x & 31, k = blockIdx.x, K = gridDim.x;
    for (int e = threadIdx.x; e < 1024; e += 256) sR[(e >> 5) * 33 + (e & 31)] = R[(long long)k * 1024 + e];
    for (int b0 = 0; b0 < B; b0 += 8) {
        const float v = z_analysis(t2, basis, b0, B, G, M, MP, k, red);
        const int b = b0 + (threadIdx.x >> 5);
        if (b >= B) continue;
        sdg[b * 32 + lane] = v;
        shh[b * 32 + lane] = hh[((long long)b * K + k) * 32 + lane];
    }
    __syncthreads();
    for (int b = threadIdx.x >> 5; b < B; b += 8) {
        float s = 0.0f;
#pragma unroll 8
        for (int o = 0; o < 32; ++o) s = fmaf(sdg[b * 32 + o], sR[lane * 33 + o], s);
        dhh[((long long)b * K + k) * 32 + lane] = s;
    }
    for (int e = threadIdx.x; e < 1024; e += 256) {
        float s = 0.0f;
        for (int b = 0; b < B; ++b) s = fmaf(shh[b * 32 + (e >> 5)], sdg[b * 32 + (e & 31)], s);
        dR[(long long)k * 1024 + e] = s;
    }
}

// MMA fragments of a 32 x 32 matrix X[k][n] in three BF16 levels, k and n permuted as the lanes
// own channels: sW[level][k half][n pair][lane] holds the B operands of two column tiles.
__device__ __forceinline__ void load_fragments(uint4 *sW, const float *X, bool transpose, int threads) {
    for (int e = threadIdx.x; e < 2 * 2 * 32; e += threads) {
        const int lane = e & 31, np = (e >> 5) & 1, ks = e >> 6;
        const int g = lane >> 2, t = lane & 3;
        uint32_t lv[3][4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int n = 8 * (g >> 1) + 2 * (2 * np + q) + (g & 1);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = 8 * t + 4 * ks + 2 * h;
                float a = transpose ? X[n * 32 + k] : X[k * 32 + n];
                float b = transpose ? X[n * 32 + k + 1] : X[(k + 1) * 32 + n];
#pragma unroll
                for (int l = 0; l < 3; ++l) lv[l][2 * q + h] = take_level(a, b);
            }
        }
#pragma unroll
        for (int l = 0; l < 3; ++l)
            sW[((l * 2 + ks) * 2 + np) * 32 + lane] = make_uint4(lv[l][0], lv[l][1], lv[l][2], lv[l][3]);
    }
}

// sS[ky][kx][c] = sum_kz B[z][kz] g[b][kz][ky][kx][c] of one plane.
template <int MP>
__device__ __forceinline__ void z_synthesis(float *sS, const float *sB, const float *__restrict__ g, int b, int z, int M,
                                            int threads) {
    const float *gb = g + (long long)b * M * M * M * 32;
    for (int e = threadIdx.x; e < MP * MP * 32; e += threads) {
        const int kk = e >> 5, ky = kk / MP, kx = kk % MP;
        float a = 0.0f;
        if (ky < M && kx < M)
            for (int k = 0; k < M; ++k) a = fmaf(sB[z * MP + k], __ldg(gb + ((k * M + ky) * M + kx) * 32 + (e & 31)), a);
        sS[e] = a;
    }
}

// sT[kx][c] = sum_ky B[y][ky] sS[ky][kx][c] of one row, by one warp (lane = channel).
template <int MP>
__device__ __forceinline__ void y_synthesis(float *sT, const float *sS, const float *sB, int y, int lane) {
    __syncwarp();
#pragma unroll
    for (int kx = 0; kx < MP; ++kx) {
        float a = 0.0f;
#pragma unroll
        for (int ky = 0; ky < MP; ++ky) a = fmaf(sB[y * MP + ky], sS[(ky * MP + kx) * 32 + lane], a);
        sT[kx * 32 + lane] = a;
    }
    __syncwarp();
}

struct TrFwd {
    TrIn in;
    const float *basis, *g, *W, *bvec;
    __nv_bfloat16 *z, *hnext;
    int B, G, M;
    // last block: projection, and with a target the loss and its gradients
    const float *wp, *bp, *target;
    float *out, *dout, *dwp, *dbp;
    double *loss;
};

constexpr int kTrDepthF = 5, kTrDepthB = 3;   // steps of 16 nodes in flight per warp
constexpr int tr_fwd_smem() { return 8 * kTrDepthF * 2 * 32 * 16; }
constexpr int tr_bwd_smem(bool first, bool last) {
    return 4 * kTrDepthB * 2 * (tr_pieces(last ? TR_DOUT : TR_DZ) + tr_pieces(first ? TR_LIFT : TR_H)) * 32 * 16;
}

template <int MP, bool LIFT, bool LAST>
__global__ void __launch_bounds__(256, 2) k_tr_fwd(const TrFwd a) {
    __shared__ float sB[256 * MP];
    __shared__ __align__(16) float sS[MP * MP * 32];
    __shared__ __align__(16) float sT[8][MP * 32];
    __shared__ uint4 sW[3 * 2 * 2 * 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int G = a.G, M = a.M;
    for (int e = threadIdx.x; e < MP * G; e += 256) {
        const int x = e / MP, k = e % MP;
        sB[e] = (k < M) ? a.basis[x * M + k] : 0.0f;
    }
    load_fragments(sW, a.W, false, 256);
    extern __shared__ __align__(16) uint8_t tr_smem[];
    uint4 *mine = reinterpret_cast<uint4 *>(tr_smem) + warp * kTrDepthF * 2 * 32 + lane;
    const TrLoad<LIFT ? TR_LIFT : TR_H> load(a.in, t);
    float bias[8], wp[LAST ? 8 : 1], gw[LAST ? 8 : 1], gb = 0.0f, bp = 0.0f, inv = 0.0f;
    double loss = 0.0;
#pragma unroll
    for (int j = 0; j < 8; ++j) bias[j] = a.bvec[8 * t + j];
    if constexpr (LAST) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            wp[j] = a.wp[8 * t + j];
            gw[j] = 0.0f;
        }
        bp = a.bp[0];
        inv = 1.0f / (float)((long long)a.B * G * G * G);
    }
    const int chunks = (G + kTrRows - 1) / kTrRows;
    const int items = a.B * G * chunks;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int plane = it / chunks, y0 = (it % chunks) * kTrRows, y1 = min(y0 + kTrRows, G);
        TrSteps ahead{(long long)plane * G, y0 + warp, 0, 8, y1, 16, G};
        int slot = 0;
        auto issue = [&](int sl) {
            if (!ahead.done()) {
                load.issue(mine + sl * 64, ahead.row() + ahead.x + g, ahead.x + g < G);
                load.issue(mine + sl * 64 + 32, ahead.row() + ahead.x + 8 + g, ahead.x + 8 + g < G);
            }
            ahead.next();
            copy_commit();
        };
        for (int i = 0; i < kTrDepthF - 1; ++i) issue(i);
        __syncthreads();
        z_synthesis<MP>(sS, sB, a.g, plane / G, plane % G, M, 256);
        __syncthreads();
        for (int y = y0 + warp; y < y1; y += 8) {
            y_synthesis<MP>(sT[warp], sS, sB, y, lane);
            float2 T[MP][4];
#pragma unroll
            for (int k = 0; k < MP; ++k)
#pragma unroll
                for (int j = 0; j < 4; ++j) T[k][j] = *reinterpret_cast<const float2 *>(sT[warp] + k * 32 + 8 * t + 2 * j);
            const long long row = ((long long)plane * G + y) * G;
            for (int x0 = 0; x0 < G; x0 += 16) {
                copy_wait<kTrDepthF - 2>();
                const uint4 cA = load.octet(mine + slot * 64, x0 + g < G);
                const uint4 cB = load.octet(mine + slot * 64 + 32, x0 + 8 + g < G);
                issue(slot == 0 ? kTrDepthF - 1 : slot - 1);
                slot = slot == kTrDepthF - 1 ? 0 : slot + 1;
                float d[4][4];
#pragma unroll
                for (int n = 0; n < 4; ++n) d[n][0] = d[n][1] = d[n][2] = d[n][3] = 0.0f;
#pragma unroll
                for (int l = 2; l >= 0; --l)
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                        for (int np = 0; np < 2; ++np) {
                            const uint4 w = sW[((l * 2 + ks) * 2 + np) * 32 + lane];
                            const uint32_t a0 = ks ? cA.z : cA.x, a1 = ks ? cB.z : cB.x;
                            const uint32_t a2 = ks ? cA.w : cA.y, a3 = ks ? cB.w : cB.y;
                            mma16816(d[2 * np], a0, a1, a2, a3, w.x, w.y);
                            mma16816(d[2 * np + 1], a0, a1, a2, a3, w.z, w.w);
                        }
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int x = x0 + 8 * r + g;
                    const bool ok = x < G;
                    float2 s2[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) s2[j] = make_float2(bias[2 * j], bias[2 * j + 1]);
                    const float *b = sB + min(x, G - 1) * MP;
#pragma unroll
                    for (int k = 0; k < MP; ++k)
#pragma unroll
                        for (int j = 0; j < 4; ++j) s2[j] = __ffma2_rn(make_float2(b[k], b[k]), T[k][j], s2[j]);
                    float s[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) s[j] = (j & 1 ? s2[j >> 1].y : s2[j >> 1].x) + d[j >> 1][2 * r + (j & 1)];
                    const long long p = row + x;
                    uint4 o;
                    if (LAST || a.z != nullptr) {
                        o = make_uint4(pack_bf16(s[0], s[1]), pack_bf16(s[2], s[3]), pack_bf16(s[4], s[5]),
                                       pack_bf16(s[6], s[7]));
                        if (!LAST && ok) *reinterpret_cast<uint4 *>(a.z + p * 32 + 8 * t) = o;
                    }
                    if constexpr (!LAST) {
#pragma unroll
                        for (int j = 0; j < 8; j += 2) {
                            const float2 v = tr_gelu(make_float2(s[j], s[j + 1]));
                            s[j] = v.x;
                            s[j + 1] = v.y;
                        }
                        o = make_uint4(pack_bf16(s[0], s[1]), pack_bf16(s[2], s[3]), pack_bf16(s[4], s[5]),
                                       pack_bf16(s[6], s[7]));
                        if (ok) *reinterpret_cast<uint4 *>(a.hnext + p * 32 + 8 * t) = o;
                    } else {
                        const float hv[8] = {bf_lo(o.x), bf_hi(o.x), bf_lo(o.y), bf_hi(o.y),
                                             bf_lo(o.z), bf_hi(o.z), bf_lo(o.w), bf_hi(o.w)};
                        float v = 0.0f;
#pragma unroll
                        for (int j = 0; j < 8; ++j) v = fmaf(hv[j], wp[j], v);
                        v += __shfl_xor_sync(0xffffffffu, v, 1);
                        v += __shfl_xor_sync(0xffffffffu, v, 2);
                        v += bp;
                        if (ok) {   // h_L itself is not stored: nothing reads it
                            if (t == 0) a.out[p] = v;
                            if (a.target != nullptr) {
                                const float e = v - a.target[p];
                                const float dd = 2.0f * e * inv;
#pragma unroll
                                for (int j = 0; j < 8; ++j) gw[j] = fmaf(dd, hv[j], gw[j]);
                                if (t == 0) {
                                    a.dout[p] = dd;
                                    gb += dd;
                                    loss += (double)e * e;
                                }
                            }
                        }
                    }
                }
            }
        }
    }
    if constexpr (LAST) {
        copy_wait<0>();
        if (a.target == nullptr) return;
        // the projection's gradients and the loss: lanes of one t, then the warps
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
#pragma unroll
            for (int j = 0; j < 8; ++j) gw[j] += __shfl_xor_sync(0xffffffffu, gw[j], o);
            gb += __shfl_xor_sync(0xffffffffu, gb, o);
            loss += __shfl_xor_sync(0xffffffffu, loss, o);
        }
        __syncthreads();
        if (g == 0)
#pragma unroll
            for (int j = 0; j < 8; ++j) sT[warp][8 * t + j] = gw[j];
        if (lane == 0) {
            sT[warp][32] = gb;
            atomicAdd(a.loss, loss / (double)((long long)a.B * G * G * G));
        }
        __syncthreads();
        if (threadIdx.x < 33) {
            float s = 0.0f;
            for (int w = 0; w < 8; ++w) s += sT[w][threadIdx.x];
            atomicAdd(threadIdx.x < 32 ? a.dwp + threadIdx.x : a.dbp, s);
        }
    }
}

struct TrBwd {
    TrIn in;
    const float *basis, *dhh, *W;
    float *dh_prev;             // block 0: not written, goes into dwl, dbl
    float *dW, *db, *dwl, *dbl;
    int B, G, M;
};

template <int MP, bool FIRST, bool LAST>
__global__ void __launch_bounds__(128, 3) k_tr_bwd(const TrBwd a) {
    __shared__ float sB[256 * MP];
    __shared__ __align__(16) float sS[MP * MP * 32 < 1024 + 96 ? 1024 + 96 : MP * MP * 32];
    __shared__ __align__(16) float sT[4][MP * 32];
    __shared__ uint4 sW[3 * 2 * 2 * 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int G = a.G, M = a.M;
    for (int e = threadIdx.x; e < MP * G; e += 128) {
        const int x = e / MP, k = e % MP;
        sB[e] = (k < M) ? a.basis[x * M + k] : 0.0f;
    }
    load_fragments(sW, a.W, true, 128);
    constexpr int kH = FIRST ? TR_LIFT : TR_H, kZ = LAST ? TR_DOUT : TR_DZ;
    constexpr int kStep = 2 * (tr_pieces(kZ) + tr_pieces(kH)) * 32;   // ring slots of a step
    extern __shared__ __align__(16) uint8_t tr_smem[];
    uint4 *mine = reinterpret_cast<uint4 *>(tr_smem) + warp * kTrDepthB * kStep + lane;
    const TrLoad<kH> load_h(a.in, t);
    const TrLoad<kZ> load_dz(a.in, t);
    float dW[2][4][4], db[8], gl[FIRST ? 8 : 1], gbl[FIRST ? 8 : 1];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int n = 0; n < 4; ++n) dW[m][n][0] = dW[m][n][1] = dW[m][n][2] = dW[m][n][3] = 0.0f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        db[j] = 0.0f;
        if constexpr (FIRST) gl[j] = gbl[j] = 0.0f;
    }
    const int chunks = (G + kTrRows - 1) / kTrRows;
    const int items = a.B * G * chunks;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int plane = it / chunks, y0 = (it % chunks) * kTrRows, y1 = min(y0 + kTrRows, G);
        TrSteps ahead{(long long)plane * G, y0 + warp, 0, 4, y1, 16, G};
        int slot = 0;
        auto issue = [&](int sl) {
            if (!ahead.done()) {
                uint4 *q = mine + sl * kStep;
                const long long p = ahead.row() + ahead.x + g;
                const bool okA = ahead.x + g < G, okB = ahead.x + 8 + g < G;
                load_dz.issue(q, p, okA);
                load_dz.issue(q + tr_pieces(kZ) * 32, p + 8, okB);
                load_h.issue(q + 2 * tr_pieces(kZ) * 32, p, okA);
                load_h.issue(q + 2 * tr_pieces(kZ) * 32 + 32, p + 8, okB);
            }
            ahead.next();
            copy_commit();
        };
        for (int i = 0; i < kTrDepthB - 1; ++i) issue(i);
        __syncthreads();
        z_synthesis<MP>(sS, sB, a.dhh, plane / G, plane % G, M, 128);
        __syncthreads();
        for (int y = y0 + warp; y < y1; y += 4) {
            y_synthesis<MP>(sT[warp], sS, sB, y, lane);
            const long long row = ((long long)plane * G + y) * G;
            for (int x0 = 0; x0 < G; x0 += 16) {
                const int xA = x0 + g, xB = x0 + 8 + g;
                copy_wait<kTrDepthB - 2>();
                const uint4 *q = mine + slot * kStep;
                float2 vA[4], vB[4];
                load_dz.values(q, xA < G, vA);
                load_dz.values(q + tr_pieces(kZ) * 32, xB < G, vB);
                const uint4 oA = load_h.octet(q + 2 * tr_pieces(kZ) * 32, xA < G);
                const uint4 oB = load_h.octet(q + 2 * tr_pieces(kZ) * 32 + 32, xB < G);
                issue(slot == 0 ? kTrDepthB - 1 : slot - 1);
                slot = slot == kTrDepthB - 1 ? 0 : slot + 1;
                uint32_t lA[3][4], lB[3][4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    db[2 * j] += vA[j].x + vB[j].x;
                    db[2 * j + 1] += vA[j].y + vB[j].y;
#pragma unroll
                    for (int l = 0; l < 3; ++l) {
                        lA[l][j] = take_level(vA[j].x, vA[j].y);
                        lB[l][j] = take_level(vB[j].x, vB[j].y);
                    }
                }
                // dW += h^T dz over the 16 nodes
                {
                    const uint32_t hA[4] = {oA.x, oA.y, oA.z, oA.w}, hB[4] = {oB.x, oB.y, oB.z, oB.w};
                    uint32_t tA[4], tB[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        tA[r] = trans8x8(hA[r]);
                        tB[r] = trans8x8(hB[r]);
                    }
#pragma unroll
                    for (int n = 0; n < 4; ++n) {
                        float d[2][4] = {{0.0f, 0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f, 0.0f}};
#pragma unroll
                        for (int l = 2; l >= 0; --l) {
                            const uint32_t b0 = trans8x8(lA[l][n]), b1 = trans8x8(lB[l][n]);
#pragma unroll
                            for (int m = 0; m < 2; ++m)
                                mma16816(d[m], tA[2 * m], tA[2 * m + 1], tB[2 * m], tB[2 * m + 1], b0, b1);
                        }
#pragma unroll
                        for (int m = 0; m < 2; ++m)
#pragma unroll
                            for (int e = 0; e < 4; ++e) dW[m][n][e] += d[m][e];
                    }
                }
                // dh_prev = dz W^T + synthesis
                float d[4][4];
#pragma unroll
                for (int n = 0; n < 4; ++n) d[n][0] = d[n][1] = d[n][2] = d[n][3] = 0.0f;
#pragma unroll
                for (int lw = 2; lw >= 0; --lw)
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                        for (int np = 0; np < 2; ++np) {
                            const uint4 w = sW[((lw * 2 + ks) * 2 + np) * 32 + lane];
#pragma unroll
                            for (int l = 2; l >= 0; --l) {
                                if (l + lw > 2) continue;
                                mma16816(d[2 * np], lA[l][2 * ks], lB[l][2 * ks], lA[l][2 * ks + 1], lB[l][2 * ks + 1],
                                         w.x, w.y);
                                mma16816(d[2 * np + 1], lA[l][2 * ks], lB[l][2 * ks], lA[l][2 * ks + 1],
                                         lB[l][2 * ks + 1], w.z, w.w);
                            }
                        }
                float2 s2[2][4];
                const float *bA = sB + min(xA, G - 1) * MP, *bB = sB + min(xB, G - 1) * MP;
#pragma unroll
                for (int j = 0; j < 4; ++j) s2[0][j] = s2[1][j] = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int k = 0; k < MP; ++k) {
                    const float4 u = *reinterpret_cast<const float4 *>(sT[warp] + k * 32 + 8 * t);
                    const float4 v = *reinterpret_cast<const float4 *>(sT[warp] + k * 32 + 8 * t + 4);
                    const float2 T[4] = {{u.x, u.y}, {u.z, u.w}, {v.x, v.y}, {v.z, v.w}};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        s2[0][j] = __ffma2_rn(make_float2(bA[k], bA[k]), T[j], s2[0][j]);
                        s2[1][j] = __ffma2_rn(make_float2(bB[k], bB[k]), T[j], s2[1][j]);
                    }
                }
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int x = x0 + 8 * r + g;
                    float s[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        s[j] = (j & 1 ? s2[r][j >> 1].y : s2[r][j >> 1].x) + d[j >> 1][2 * r + (j & 1)];
                    if (x >= G) continue;
                    if constexpr (FIRST) {
                        const float fv = a.in.f[row + x];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            gl[j] = fmaf(fv, s[j], gl[j]);
                            gbl[j] += s[j];
                        }
                    } else {
                        float4 *o = reinterpret_cast<float4 *>(a.dh_prev + (row + x) * 32 + 8 * t);
                        o[0] = make_float4(s[0], s[1], s[2], s[3]);
                        o[1] = make_float4(s[4], s[5], s[6], s[7]);
                    }
                }
            }
        }
    }
    // sums over the lanes of one t, then over the warps in a fixed order, then one atomic each
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            db[j] += __shfl_xor_sync(0xffffffffu, db[j], o);
            if constexpr (FIRST) {
                gl[j] += __shfl_xor_sync(0xffffffffu, gl[j], o);
                gbl[j] += __shfl_xor_sync(0xffffffffu, gbl[j], o);
            }
        }
    __syncthreads();
    for (int e = threadIdx.x; e < 1024 + 96; e += 128) sS[e] = 0.0f;
    __syncthreads();
    for (int w = 0; w < 4; ++w) {
        if (warp == w) {
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int n = 0; n < 4; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int i = 8 * (g >> 1) + 2 * (2 * m + (e >> 1)) + (g & 1), o = 8 * t + 2 * n + (e & 1);
                        sS[i * 32 + o] += dW[m][n][e];
                    }
            if (g == 0)
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    sS[1024 + 8 * t + j] += db[j];
                    if constexpr (FIRST) {
                        sS[1056 + 8 * t + j] += gl[j];
                        sS[1088 + 8 * t + j] += gbl[j];
                    }
                }
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < 1024 + (FIRST ? 96 : 32); e += 128) {
        float *o = e < 1024 ? a.dW + e : (e < 1056 ? a.db + (e - 1024) : (e < 1088 ? a.dwl + (e - 1056) : a.dbl + (e - 1088)));
        atomicAdd(o, sS[e]);
    }
}

// Forward pass of B samples (f: [B][G^3]); with a target the loss, dout and the projection's
// gradients too (the gradient array must be zero).
struct TrNet {
    int G, M, L, B;
    const float *f, *target, *basis;
    float *params, *grads, *t2, *g, *dhh, *out, *dout, *dh;
    double *loss;
    __nv_bfloat16 *const *h, *const *z;
    float *const *hh;
    const long long *off_R, *off_W, *off_b;
    long long off_wp;
    int num_sms;   // two (forward) and three (backward) resident CTAs on each
};

template <typename K>
int tr_opt_in(K kernel, int bytes) {
    QN_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    return QN_OK;
}

// More than 48 KB of shared memory for every kernel of one MP (at network creation).
template <int MP>
int tr_set_attributes() {
    int rc = tr_opt_in(k_tr_analysis<MP, TR_H>, tr_analysis_smem<MP, TR_H>());
    if (rc == QN_OK) rc = tr_opt_in(k_tr_analysis<MP, TR_LIFT>, tr_analysis_smem<MP, TR_LIFT>());
    if (rc == QN_OK) rc = tr_opt_in(k_tr_analysis<MP, TR_DZ>, tr_analysis_smem<MP, TR_DZ>());
    if (rc == QN_OK) rc = tr_opt_in(k_tr_analysis<MP, TR_DOUT>, tr_analysis_smem<MP, TR_DOUT>());
    if (rc == QN_OK) rc = tr_opt_in(k_tr_fwd<MP, false, false>, tr_fwd_smem());
    if (rc == QN_OK) rc = tr_opt_in(k_tr_fwd<MP, false, true>, tr_fwd_smem());
    if (rc == QN_OK) rc = tr_opt_in(k_tr_fwd<MP, true, false>, tr_fwd_smem());
    if (rc == QN_OK) rc = tr_opt_in(k_tr_fwd<MP, true, true>, tr_fwd_smem());
    if (rc == QN_OK) rc = tr_opt_in(k_tr_bwd<MP, false, false>, tr_bwd_smem(false, false));
    if (rc == QN_OK) rc = tr_opt_in(k_tr_bwd<MP, false, true>, tr_bwd_smem(false, true));
    if (rc == QN_OK) rc = tr_opt_in(k_tr_bwd<MP, true, false>, tr_bwd_smem(true, false));
    if (rc == QN_OK) rc = tr_opt_in(k_tr_bwd<MP, true, true>, tr_bwd_smem(true, true));
    return rc;
}

template <int MP>
void tr_forward(const TrNet &n, cudaStream_t s) {
    const int planes = n.B * n.G, K = n.M * n.M * n.M;
    const int items = planes * ((n.G + kTrRows - 1) / kTrRows);
    const int grid = items < 2 * n.num_sms ? items : 2 * n.num_sms;
    for (int l = 0; l < n.L; ++l) {
        TrFwd a{};
        a.in.h = n.h[l];
        a.in.f = n.f;
        a.in.wl = n.params;
        a.in.bl = n.params + 32;
        if (l == 0)
            k_tr_analysis<MP, TR_LIFT><<<planes * kTrParts, 256, tr_analysis_smem<MP, TR_LIFT>(), s>>>(a.in, n.basis, n.G, n.M, n.t2);
        else
            k_tr_analysis<MP, TR_H><<<planes * kTrParts, 256, tr_analysis_smem<MP, TR_H>(), s>>>(a.in, n.basis, n.G, n.M, n.t2);
        k_tr_mix<<<K, 256, 0, s>>>(n.t2, n.basis, n.B, n.G, n.M, MP, n.params + n.off_R[l], n.hh[l], n.g);
        a.basis = n.basis;
        a.g = n.g;
        a.W = n.params + n.off_W[l];
        a.bvec = n.params + n.off_b[l];
        a.z = n.target != nullptr ? n.z[l] : nullptr;
        a.hnext = n.h[l + 1];
        a.B = n.B;
        a.G = n.G;
        a.M = n.M;
        a.wp = n.params + n.off_wp;
        a.bp = a.wp + 32;
        a.target = n.target;
        a.out = n.out;
        a.dout = n.dout;
        a.dwp = n.grads + n.off_wp;
        a.dbp = a.dwp + 32;
        a.loss = n.loss;
        const bool last = l == n.L - 1;
        if (l == 0 && last)
            k_tr_fwd<MP, true, true><<<grid, 256, tr_fwd_smem(), s>>>(a);
        else if (l == 0)
            k_tr_fwd<MP, true, false><<<grid, 256, tr_fwd_smem(), s>>>(a);
        else if (last)
            k_tr_fwd<MP, false, true><<<grid, 256, tr_fwd_smem(), s>>>(a);
        else
            k_tr_fwd<MP, false, false><<<grid, 256, tr_fwd_smem(), s>>>(a);
    }
}

template <int MP>
void tr_backward(const TrNet &n, cudaStream_t s) {
    const int planes = n.B * n.G, K = n.M * n.M * n.M;
    const int items = planes * ((n.G + kTrRows - 1) / kTrRows);
    const int grid = items < 3 * n.num_sms ? items : 3 * n.num_sms;
    for (int l = n.L - 1; l >= 0; --l) {
        const bool last = l == n.L - 1;
        TrBwd a{};
        a.in.h = n.h[l];
        a.in.z = n.z[l];
        a.in.f = n.f;
        a.in.wl = n.params;
        a.in.bl = n.params + 32;
        a.in.dh = last ? n.dout : n.dh;
        a.in.wp = n.params + n.off_wp;
        if (last)
            k_tr_analysis<MP, TR_DOUT><<<planes * kTrParts, 256, tr_analysis_smem<MP, TR_DOUT>(), s>>>(a.in, n.basis, n.G, n.M, n.t2);
        else
            k_tr_analysis<MP, TR_DZ><<<planes * kTrParts, 256, tr_analysis_smem<MP, TR_DZ>(), s>>>(a.in, n.basis, n.G, n.M, n.t2);
        k_tr_mix_bwd<<<K, 256, 0, s>>>(n.t2, n.basis, n.B, n.G, n.M, MP, n.params + n.off_R[l], n.hh[l], n.dhh,
                                       n.grads + n.off_R[l]);
        a.basis = n.basis;
        a.dhh = n.dhh;
        a.W = n.params + n.off_W[l];
        a.dh_prev = n.dh;
        a.dW = n.grads + n.off_W[l];
        a.db = n.grads + n.off_b[l];
        a.dwl = n.grads;
        a.dbl = n.grads + 32;
        a.B = n.B;
        a.G = n.G;
        a.M = n.M;
        if (l == 0 && last)
            k_tr_bwd<MP, true, true><<<grid, 128, tr_bwd_smem(true, true), s>>>(a);
        else if (l == 0)
            k_tr_bwd<MP, true, false><<<grid, 128, tr_bwd_smem(true, false), s>>>(a);
        else if (last)
            k_tr_bwd<MP, false, true><<<grid, 128, tr_bwd_smem(false, true), s>>>(a);
        else
            k_tr_bwd<MP, false, false><<<grid, 128, tr_bwd_smem(false, false), s>>>(a);
    }
}

}  // namespace
}  // namespace qn
