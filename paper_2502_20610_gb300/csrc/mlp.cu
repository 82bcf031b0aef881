// Learned absorbing boundary: the network's kernels.
//
// The network (2 hidden layers of 64, FP32, tanh) maps the 3x3x3 stencil of
// the six fields at steps n and n-1 around a cell of the wall layer (324
// inputs) to a correction of that cell's Yee step.  Every cell of the
// domain takes the Yee step with the domain's PEC walls (Yee_D); a layer
// cell then adds the correction, scale-equivariantly: with
// r = sqrt(mean(x^2)) the network sees x / r and
//     S^{n+1}(centre) = Yee_D(S^n)(centre) + r * f(x / r),
// so a wave of any amplitude meets the same boundary operator (the update is
// linear in the fields), and f = 0 is the plain PEC box.  Only the values
// the box's own walls get wrong are corrected: on a cell of a low face the
// two E components tangential to it (PEC holds them), on a cell of a high
// face the two tangential H components (PEC reads E beyond it as 0).  Every
// other value of the box's Yee step is exact, so its correction is zero
// (tangent_mask).  A stencil with r < R_MIN (1e-30, where 1/r would
// leave the FP32 range) counts as zero: the cell keeps its value.  Parameters, in this order: W1 [64][324], b1 [64],
// W2 [64][64], b2 [64], W3 [6][64], b3 [6] (row = output unit).
//
// Training runs on the GPU with these kernels: one that takes 32 samples at
// a time through the whole forward and backward pass in shared memory and
// registers, and one that sums its partial gradients and takes the Adam
// step.  The layer update of
// a simulation step is one fused persistent kernel over patches of the
// domain's faces, the two large contractions on the tensor cores (mma.sync
// TF32, three-term split for FP32 accuracy).
#include "internal.h"
#include "mlp.h"
#include "yee_cell.cuh"

#include <cmath>
#include <cstring>
#include <random>
#include <vector>

namespace {

using namespace mlpnet;

constexpr int NPARAM_PITCH = (NPARAM + 31) / 32 * 32;  // one partial gradient, 128-byte aligned rows

// ------------------------------------------------- forward / backward pass

// One kernel takes a minibatch through the whole network: a CTA holds the
// weights and 32 samples in shared memory, runs the three layers, the loss
// and (training) the backward pass on them, and keeps the weight gradients
// in registers over all its tiles, so activations never leave the SM and a
// minibatch costs two launches (this one, then grad_kernel).  What bounds
// it: FP32 FMA issue (25 k multiply-adds a sample forward, 29 k backward).
// Splitting a minibatch over its samples gives a CTA per 32 of them; the
// sums over samples are then short (32 in sequence, then one partial per
// CTA), where one CTA per weight-gradient tile ran a 4096-long chain.
// Measured (ncu): 29 us + 7 us in grad_kernel for a batch of 4096, against
// 1.38 ms in eleven GEMM and reduction launches; two epochs over 32768
// samples 22.1 ms -> 0.75 ms.
// FP32 multiply-adds, not split TF32 products on the tensor cores: a
// split has no form for infinities (inf - inf), and the sums here round
// as FP32 sums do.  Pairs of multiply-adds go out as one packed f32x2
// instruction, each half rounded as the scalar one is.
constexpr int TS = 32;         // samples per tile
constexpr int NT = 256;        // threads
constexpr int PH = NH + 4;     // pitch of 64-wide rows: 16-byte rows, 8 rows on 8 bank groups
constexpr int KC1 = NI / 4, KC2 = NH / 4;  // 16-byte chunks of a row
static_assert(NI % 4 == 0 && (NI / 4) % 8 == 1 && (PH / 4) % 8 == 1, "row starts of 8 lanes on 8 bank groups");
static_assert(OFF_W2 % 4 == 0, "W2 rows 16-byte aligned when the parameters are");
// shared memory, in floats
constexpr int NS_W1 = 0, NS_X = NS_W1 + NH * NI, NS_W2 = NS_X + TS * NI, NS_W2T = NS_W2 + NH * PH,
              NS_H1 = NS_W2T + NH * PH, NS_H2 = NS_H1 + TS * PH, NS_Z1 = NS_H2 + TS * PH, NS_Z2 = NS_Z1 + TS * PH,
              NS_RED = NS_Z2 + TS * PH, NS_W3 = NS_RED + 3 * TS * NH, NS_B = NS_W3 + NO * NH, NS_DY = NS_B + 136,
              NS_LOSS = NS_DY + TS * 8, NS_END = NS_LOSS + 2 * NT;
static_assert(NS_LOSS % 2 == 0, "FP64 partial sums 8-byte aligned");
constexpr size_t NET_SMEM = sizeof(float) * NS_END;
static_assert(NET_SMEM <= 227 * 1024, "one CTA's shared memory");
// CTAs (and gradient partials) of a minibatch: one per SM of the chip at most
constexpr int MAX_PARTS = 152;

int net_parts(long long B) { return (int)std::min<long long>((B + TS - 1) / TS, MAX_PARTS); }

__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long pair(float lo, float hi)
{
    return (unsigned long long)__float_as_uint(lo) | ((unsigned long long)__float_as_uint(hi) << 32);
}
__device__ __forceinline__ float lo_of(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi_of(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }

// out[s][u] = sum_k A[s][k] W[u][k] for the tile's 32 samples and 64 units
// (CHUNKS 16-byte chunks of k), before bias and activation, left as four
// partial sums to be added by tile_sum: warp w takes samples 16 * (w / 4) ..
// and every fourth chunk from w % 4, a lane units lane and lane + 32.  A's
// loads are broadcasts, W's conflict-free; 16 samples a warp make a chunk 24
// shared-memory wavefronts for 64 packed multiply-adds.
template <int CHUNKS>
__device__ __forceinline__ void tile_product(const float *A, int pa, const float *W, int pw, float *out, float *red)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, kq = w & 3, s0 = 16 * (w >> 2);
    unsigned long long acc[16][2];
#pragma unroll
    for (int s = 0; s < 16; ++s) acc[s][0] = acc[s][1] = 0ull;
#pragma unroll 1
    for (int c = kq; c < CHUNKS; c += 4) {
        const ulonglong2 w0 = *reinterpret_cast<const ulonglong2 *>(W + lane * pw + 4 * c);
        const ulonglong2 w1 = *reinterpret_cast<const ulonglong2 *>(W + (lane + 32) * pw + 4 * c);
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(A + (s0 + s) * pa + 4 * c);
            acc[s][0] = fma2(x.x, w0.x, acc[s][0]);
            acc[s][1] = fma2(x.x, w1.x, acc[s][1]);
            acc[s][0] = fma2(x.y, w0.y, acc[s][0]);
            acc[s][1] = fma2(x.y, w1.y, acc[s][1]);
        }
    }
    float *dst = kq == 0 ? out : red + (kq - 1) * TS * NH;
    const int pd = kq == 0 ? PH : NH;
#pragma unroll
    for (int s = 0; s < 16; ++s)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            dst[(s0 + s) * pd + lane + 32 * h] = __fadd_rn(lo_of(acc[s][h]), hi_of(acc[s][h]));
}

// The four partial sums of element (s, u); called after a block barrier.
__device__ __forceinline__ float tile_sum(const float *out, const float *red, int s, int u)
{
    const int r = s * NH + u;
    return __fadd_rn(__fadd_rn(out[s * PH + u], red[r]), __fadd_rn(red[TS * NH + r], red[2 * TS * NH + r]));
}

// Y = f(X) of B samples X[rows[b]] (rows may be null; FORWARD only: Y is
// written), or (!FORWARD) this CTA's share of the gradient of the mean
// squared error against T into part[blockIdx.x][NPARAM] and of the sum of
// squared errors into loss_part[blockIdx.x].  vec: P and X are 16-byte
// aligned (rows of X then are too), loaded by 16-byte asynchronous copies.
template <bool FORWARD>
__global__ void __launch_bounds__(NT, 1) net_kernel(const float *__restrict__ P, const float *__restrict__ X,
                                                    const int *__restrict__ rows, const float *__restrict__ T,
                                                    long long B, float *__restrict__ Y, float *__restrict__ part,
                                                    double *__restrict__ loss_part, int vec)
{
    extern __shared__ __align__(16) float sm[];
    float *const W1 = sm + NS_W1, *const Xs = sm + NS_X, *const W2 = sm + NS_W2, *const W2t = sm + NS_W2T;
    float *const H1 = sm + NS_H1, *const H2 = sm + NS_H2, *const Z1 = sm + NS_Z1, *const Z2 = sm + NS_Z2;
    float *const red = sm + NS_RED, *const W3 = sm + NS_W3, *const bias = sm + NS_B, *const dY = sm + NS_DY;
    double *const lsum = reinterpret_cast<double *>(sm + NS_LOSS);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const long long ntiles = (B + TS - 1) / TS;
    auto copy16 = [](float *dst, const float *src) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                     : "memory");
    };
    auto load_tile = [&](long long tile) {
        for (int e = tid; e < TS * KC1; e += NT) {
            const int s = e / KC1, c = e - s * KC1;
            const long long b = tile * TS + s;
            float *const dst = Xs + s * NI + 4 * c;
            if (b < B) {
                const float *const src = X + (rows ? (long long)rows[b] : b) * NI + 4 * c;
                if (vec) {
                    copy16(dst, src);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) dst[q] = src[q];
                }
            } else {  // past the batch: zeros, and no share of dY
                *reinterpret_cast<float4 *>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    };
    load_tile(blockIdx.x);
    if (vec) {
        for (int e = tid; e < NH * KC1; e += NT) copy16(W1 + 4 * e, P + OFF_W1 + 4 * e);
        for (int e = tid; e < NH * KC2; e += NT) copy16(W2 + (e / KC2) * PH + 4 * (e % KC2), P + OFF_W2 + 4 * e);
    } else {
        for (int e = tid; e < NH * NI; e += NT) W1[e] = P[OFF_W1 + e];
        for (int e = tid; e < NH * NH; e += NT) W2[(e / NH) * PH + e % NH] = P[OFF_W2 + e];
    }
    if (!FORWARD)
        for (int e = tid; e < NH * NH; e += NT) W2t[(e % NH) * PH + e / NH] = P[OFF_W2 + e];
    for (int e = tid; e < NO * NH; e += NT) W3[e] = P[OFF_W3 + e];
    if (tid < NH) {
        bias[tid] = P[OFF_B1 + tid];
        bias[NH + tid] = P[OFF_B2 + tid];
    }
    if (tid < NO) bias[2 * NH + tid] = P[OFF_B3 + tid];

    // weight gradients of this CTA's tiles: dW1 of units 8w.. and inputs
    // 4 lane + 128 j .. (+3), dW2 of units 8w.. and units 2 lane (+1), dW3 of
    // elements tid, tid + 256, and the bias of unit tid (64..127: of layer 1)
    unsigned long long g1[8][6], g2[8];
    float g3[2] = {0.f, 0.f}, gb = 0.f, gb3 = 0.f;
    double loss = 0.0;
    const float dscale = 2.f / (float)(B * NO);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        g2[u] = 0ull;
#pragma unroll
        for (int j = 0; j < 6; ++j) g1[u][j] = 0ull;
    }
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        if (tile != blockIdx.x) {
            __syncthreads();  // the previous tile's last reads of Xs
            load_tile(tile);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // rows past the batch stay zero in every layer, whatever the weights
        const int live = (int)min((long long)TS, B - tile * TS);
        tile_product<KC1>(Xs, NI, W1, NI, H1, red);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < TS * NH / NT; ++q) {
            const int s = (tid >> 6) + 4 * q, u = tid & 63;
            H1[s * PH + u] = s < live ? tanhf(__fadd_rn(tile_sum(H1, red, s, u), bias[u])) : 0.f;
        }
        __syncthreads();
        tile_product<KC2>(H1, PH, W2, PH, H2, red);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < TS * NH / NT; ++q) {
            const int s = (tid >> 6) + 4 * q, u = tid & 63;
            H2[s * PH + u] = s < live ? tanhf(__fadd_rn(tile_sum(H2, red, s, u), bias[NH + u])) : 0.f;
        }
        __syncthreads();
        if (tid < TS * NO) {  // layer 3: Y, and dY = 2 (Y - T) / (6 B)
            const int s = tid / NO, o = tid - s * NO;
            const long long b = tile * TS + s;
            float f = 0.f;
#pragma unroll
            for (int k = 0; k < NH; k += 4) {
                const float4 h = *reinterpret_cast<const float4 *>(H2 + s * PH + k);
                const float4 v = *reinterpret_cast<const float4 *>(W3 + o * NH + k);
                f = __fmaf_rn(h.x, v.x, f);
                f = __fmaf_rn(h.y, v.y, f);
                f = __fmaf_rn(h.z, v.z, f);
                f = __fmaf_rn(h.w, v.w, f);
            }
            f = __fadd_rn(f, bias[2 * NH + o]);
            if (FORWARD) {
                if (b < B) Y[b * NO + o] = f;
            } else {
                float d = 0.f;
                if (b < B) {
                    d = __fsub_rn(f, T[(rows ? (long long)rows[b] : b) * NO + o]);
                    loss += (double)d * (double)d;
                }
                dY[s * 8 + o] = __fmul_rn(d, dscale);
            }
        }
        if (FORWARD) continue;
        __syncthreads();
        // dZ2 = (dY W3) (1 - H2^2); dW3 and db3
        {
            const int u = tid & 63;
            float v3[NO];
#pragma unroll
            for (int o = 0; o < NO; ++o) v3[o] = W3[o * NH + u];
#pragma unroll
            for (int q = 0; q < TS * NH / NT; ++q) {
                const int s = (tid >> 6) + 4 * q;
                float z = 0.f;
#pragma unroll
                for (int o = 0; o < NO; ++o) z = __fmaf_rn(dY[s * 8 + o], v3[o], z);
                const float h = H2[s * PH + u];
                Z2[s * PH + u] = s < live ? __fmul_rn(z, __fsub_rn(1.f, __fmul_rn(h, h))) : 0.f;
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int e = tid + q * NT;
                if (e < NO * NH)
                    for (int s = 0; s < TS; ++s) g3[q] = __fmaf_rn(dY[s * 8 + (e >> 6)], H2[s * PH + (e & 63)], g3[q]);
            }
            if (tid < NO)
                for (int s = 0; s < TS; ++s) gb3 = __fadd_rn(gb3, dY[s * 8 + tid]);
        }
        __syncthreads();
        // dW2 = dZ2^T H1 and db2; dZ1 = (dZ2 W2) (1 - H1^2)
#pragma unroll 4
        for (int s = 0; s < TS; ++s) {
            const float4 za = *reinterpret_cast<const float4 *>(Z2 + s * PH + 8 * w);
            const float4 zb = *reinterpret_cast<const float4 *>(Z2 + s * PH + 8 * w + 4);
            const unsigned long long h = *reinterpret_cast<const unsigned long long *>(H1 + s * PH + 2 * lane);
            const float z[8] = {za.x, za.y, za.z, za.w, zb.x, zb.y, zb.z, zb.w};
#pragma unroll
            for (int u = 0; u < 8; ++u) g2[u] = fma2(pair(z[u], z[u]), h, g2[u]);
        }
        tile_product<KC2>(Z2, PH, W2t, PH, Z1, red);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < TS * NH / NT; ++q) {
            const int s = (tid >> 6) + 4 * q, u = tid & 63;
            const float h = H1[s * PH + u];
            Z1[s * PH + u] = s < live ? __fmul_rn(tile_sum(Z1, red, s, u), __fsub_rn(1.f, __fmul_rn(h, h))) : 0.f;
        }
        __syncthreads();
        if (tid < 2 * NH) {  // db2 (unit tid), db1 (unit tid - 64)
            const float *const Z = tid < NH ? Z2 + tid : Z1 + tid - NH;
            for (int s = 0; s < TS; ++s) gb = __fadd_rn(gb, Z[s * PH]);
        }
        // dW1 = dZ1^T X
#pragma unroll 1
        for (int s = 0; s < TS; ++s) {
            const float4 za = *reinterpret_cast<const float4 *>(Z1 + s * PH + 8 * w);
            const float4 zb = *reinterpret_cast<const float4 *>(Z1 + s * PH + 8 * w + 4);
            const float z[8] = {za.x, za.y, za.z, za.w, zb.x, zb.y, zb.z, zb.w};
            ulonglong2 x[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int k = 4 * lane + 128 * j;
                x[j] = k < NI ? *reinterpret_cast<const ulonglong2 *>(Xs + s * NI + k) : make_ulonglong2(0ull, 0ull);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const unsigned long long zz = pair(z[u], z[u]);
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    g1[u][2 * j] = fma2(zz, x[j].x, g1[u][2 * j]);
                    g1[u][2 * j + 1] = fma2(zz, x[j].y, g1[u][2 * j + 1]);
                }
            }
        }
    }
    if (FORWARD) return;
    float *const G = part + (long long)blockIdx.x * NPARAM_PITCH;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int k = 4 * lane + 128 * j;
            if (k < NI)
                *reinterpret_cast<float4 *>(G + OFF_W1 + (8 * w + u) * NI + k) =
                    make_float4(lo_of(g1[u][2 * j]), hi_of(g1[u][2 * j]), lo_of(g1[u][2 * j + 1]), hi_of(g1[u][2 * j + 1]));
        }
        *reinterpret_cast<float2 *>(G + OFF_W2 + (8 * w + u) * NH + 2 * lane) = make_float2(lo_of(g2[u]), hi_of(g2[u]));
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
        if (tid + q * NT < NO * NH) G[OFF_W3 + tid + q * NT] = g3[q];
    if (tid < NH) G[OFF_B2 + tid] = gb;
    else if (tid < 2 * NH) G[OFF_B1 + tid - NH] = gb;
    if (tid < NO) G[OFF_B3 + tid] = gb3;
    lsum[tid] = loss;
    __syncthreads();
    for (int n = NT / 2; n > 0; n >>= 1) {
        if (tid < n) lsum[tid] += lsum[tid + n];
        __syncthreads();
    }
    if (tid == 0) loss_part[blockIdx.x] = lsum[0];
}

// The minibatch's gradient from its nparts partials (a thread sums every
// eighth, then the eight sums; the order is fixed), then the Adam step
// (Kingma & Ba): m <- b1 m + (1-b1) g, v <- b2 v + (1-b2) g^2,
// p <- p - lr * (m / (1-b1^t)) / (sqrt(v / (1-b2^t)) + eps); or (!ADAM) the
// gradient into out.  *loss += the sum of squared errors.  Bounded by the
// read of the partials out of L2 (13 MB at a batch of 4096); 32 parameters a
// CTA put 793 CTAs of independent loads on it.
template <bool ADAM>
__global__ void __launch_bounds__(256) grad_kernel(const float *__restrict__ part, const double *__restrict__ loss_part,
                                                   int nparts, float *__restrict__ p, float *__restrict__ m,
                                                   float *__restrict__ v, float lr, float c1, float c2,
                                                   float *__restrict__ out, double *__restrict__ loss)
{
    __shared__ float sum[8][32];
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (i < NPARAM) {
#pragma unroll 4
        for (int j = sl; j < nparts; j += 8) s = __fadd_rn(s, part[(long long)j * NPARAM_PITCH + i]);
    }
    sum[sl][lane] = s;
    __syncthreads();
    if (blockIdx.x == 0 && sl == 1) {
        double l = 0.0;
        for (int j = lane; j < nparts; j += 32) l += loss_part[j];
        for (int d = 16; d > 0; d >>= 1) l += __shfl_down_sync(0xffffffffu, l, d);
        if (lane == 0) *loss += l;
    }
    if (sl || i >= NPARAM) return;
    float gi = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) gi = __fadd_rn(gi, sum[q][lane]);
    if (ADAM) {
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    } else {
        out[i] = gi;
    }
}

struct Scratch {
    float *part, *m, *v;
    double *loss, *loss_part;
    int *rows;  // the training permutation (n entries)
};

size_t scratch_bytes(int batch, long long n)
{
    const size_t parts = (size_t)net_parts(batch);
    return sizeof(float) * (parts * NPARAM_PITCH + 2 * (size_t)NPARAM) + sizeof(double) * (2 + parts) +
           sizeof(int) * (size_t)n + 7 * 256;
}

Scratch carve(void *base, int batch, long long n)
{
    // the caller's block may start anywhere; the partials are written 16 bytes at a time
    char *p = (char *)(((uintptr_t)base + 15) / 16 * 16);
    auto take = [&](size_t bytes) {
        char *q = p;
        p += (bytes + 255) / 256 * 256;
        return q;
    };
    const size_t parts = (size_t)net_parts(batch);
    Scratch s;
    s.loss = (double *)take(sizeof(double) * 2);
    s.loss_part = (double *)take(sizeof(double) * parts);
    s.part = (float *)take(sizeof(float) * parts * NPARAM_PITCH);
    s.m = (float *)take(sizeof(float) * NPARAM);
    s.v = (float *)take(sizeof(float) * NPARAM);
    s.rows = (int *)take(sizeof(int) * (size_t)n);
    return s;
}

#define CKE(x)                                                                 \
    do {                                                                       \
        cudaError_t e_ = (x);                                                  \
        if (e_ != cudaSuccess) return e_;                                      \
    } while (0)

template <bool FORWARD>
cudaError_t net_configure()
{
    return cudaFuncSetAttribute(net_kernel<FORWARD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)NET_SMEM);
}

template <bool FORWARD>
cudaError_t net(const float *P, const float *X, const int *rows, const float *T, long long B, float *Y, float *part,
                double *loss_part, cudaStream_t st)
{
    const int vec = ((uintptr_t)P % 16 == 0) && ((uintptr_t)X % 16 == 0);
    net_kernel<FORWARD><<<net_parts(B), NT, NET_SMEM, st>>>(P, X, rows, T, B, Y, part, loss_part, vec);
    return cudaGetLastError();
}

// Components of cell (x,y,z) that the correction applies to (bit c = Ex..Hz):
// tangential E on the low faces, tangential H on the high faces it lies on.
__device__ __forceinline__ unsigned tangent_mask(int x, int y, int z, int nx, int ny, int nz)
{
    unsigned m = 0;
    if (x == 0) m |= 0x6;         // Ey, Ez
    if (y == 0) m |= 0x5;         // Ex, Ez
    if (z == 0) m |= 0x3;         // Ex, Ey
    if (x == nx - 1) m |= 0x30;   // Hy, Hz
    if (y == ny - 1) m |= 0x28;   // Hx, Hz
    if (z == nz - 1) m |= 0x18;   // Hx, Hy
    return m;
}

// ---------------------------------------------------- sample recording

// Yee step of the centre of a stencil of S^n (v: [c][dz][dy][dx], 0 outside
// the box) in the box standing alone with PEC walls: tangential E on the
// box's low faces stays, E and H beyond it read 0.  Same operations as the
// naive kernels (yee_cell.cuh).
__device__ void yee_centre(const float *v, float ndt, float cb, float ca, bool lossy, bool lo_x, bool lo_y, bool lo_z,
                           float out[6])
{
    auto V = [&](int c, int dx, int dy, int dz) { return v[c * 27 + (dz + 1) * 9 + (dy + 1) * 3 + (dx + 1)]; };
    // H^{n+1/2} at offset o from the E^n and H^{n-1/2} of the stencil
    auto Hx = [&](int dx, int dy, int dz) {
        return h_x(V(3, dx, dy, dz), V(2, dx, dy + 1, dz), V(2, dx, dy, dz), V(1, dx, dy, dz + 1), V(1, dx, dy, dz), ndt);
    };
    auto Hy = [&](int dx, int dy, int dz) {
        return h_y(V(4, dx, dy, dz), V(0, dx, dy, dz + 1), V(0, dx, dy, dz), V(2, dx + 1, dy, dz), V(2, dx, dy, dz), ndt);
    };
    auto Hz = [&](int dx, int dy, int dz) {
        return h_z(V(5, dx, dy, dz), V(1, dx + 1, dy, dz), V(1, dx, dy, dz), V(0, dx, dy + 1, dz), V(0, dx, dy, dz), ndt);
    };
    const float hx = Hx(0, 0, 0), hy = Hy(0, 0, 0), hz = Hz(0, 0, 0);
    const float ex = V(0, 0, 0, 0), ey = V(1, 0, 0, 0), ez = V(2, 0, 0, 0);
    const float dex = lossy ? __fmul_rn(ca, ex) : ex, dey = lossy ? __fmul_rn(ca, ey) : ey,
                dez = lossy ? __fmul_rn(ca, ez) : ez;
    out[0] = (lo_y || lo_z) ? ex : e_x(dex, hz, Hz(0, -1, 0), hy, Hy(0, 0, -1), cb);
    out[1] = (lo_x || lo_z) ? ey : e_y(dey, hx, Hx(0, 0, -1), hz, Hz(-1, 0, 0), cb);
    out[2] = (lo_x || lo_y) ? ez : e_z(dez, hy, Hy(-1, 0, 0), hx, Hx(0, -1, 0), cb);
    out[3] = hx;
    out[4] = hy;
    out[5] = hz;
}

// The six components of the box [lo, hi) into dst [6][box cells] (x fastest).
__global__ void __launch_bounds__(256) record_box_kernel(const float *__restrict__ f, long long fstride, int pitch,
                                                         int ny, int3 lo, int3 hi, float *__restrict__ dst)
{
    const int bx = hi.x - lo.x, by = hi.y - lo.y;
    const long long bc = (long long)bx * by * (hi.z - lo.z);
    const long long q = blockIdx.x * 256ll + threadIdx.x;
    if (q >= bc) return;
    const int i = lo.x + (int)(q % bx), j = lo.y + (int)((q / bx) % by), k = lo.z + (int)(q / ((long long)bx * by));
    const long long p = i + (long long)pitch * (j + (long long)ny * k);
#pragma unroll
    for (int c = 0; c < 6; ++c) dst[c * bc + q] = f[c * fstride + p];
}

// Training pairs from a reference run: for cells (x,y,z) of the layer region
// (inside the box [lo, hi) of the reference grid), the normalised stencil of
// (S^n, S^{n-1}) -- cells outside the box read 0, as they would at a wall --
// and the normalised correction (S^{n+1} - Yee_box(S^n))(centre) / r that
// takes the box's own Yee step to the reference's next state.  cur and prev
// hold the box alone ([6][box cells]), nxt the whole reference state.
// One warp per sample: a thread per sample left 4 CTAs to write 1.3 kB rows
// 32 rows apart (267 us for 1000 samples); a warp writes its row in whole
// lines and sums the squares with shuffles.  Bounded by the latency of the
// gather (the box is in L2).
constexpr int RW = 8;  // samples (warps) per CTA
__global__ void __launch_bounds__(32 * RW) record_kernel(const float *__restrict__ prev, const float *__restrict__ cur,
                                                         const float *__restrict__ nxt, long long fstride, int pitch,
                                                         int ny, int3 lo, int3 hi, const int *__restrict__ cells, int n,
                                                         const float *__restrict__ ce, const float *__restrict__ ca,
                                                         float ndt, float *__restrict__ X, float *__restrict__ Y)
{
    __shared__ float raw[RW][NI];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int q = blockIdx.x * RW + w;
    if (q >= n) return;
    const int x = cells[3 * q], y = cells[3 * q + 1], z = cells[3 * q + 2];
    const int bx = hi.x - lo.x, by = hi.y - lo.y;
    const long long bc = (long long)bx * by * (hi.z - lo.z);
    double ss = 0.0;
#pragma unroll
    for (int u = 0; u < (NI + 31) / 32; ++u) {
        const int k = lane + 32 * u;
        if (k < NI) {
            const int d = k % 27, c = (k / 27) % 6;
            const int xx = x + d % 3 - 1, yy = y + (d / 3) % 3 - 1, zz = z + d / 9 - 1;
            float v = 0.f;
            if (xx >= lo.x && xx < hi.x && yy >= lo.y && yy < hi.y && zz >= lo.z && zz < hi.z)
                v = (k < NI / 2 ? cur : prev)[c * bc + (xx - lo.x) + (long long)bx * ((yy - lo.y) + (long long)by * (zz - lo.z))];
            raw[w][k] = v;
            ss += (double)v * v;
        }
    }
    for (int d = 16; d > 0; d >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, d);
    __syncwarp();
    // r below R_MIN counts as a zero stencil (its reciprocal would overflow
    // FP32): the pair is recorded as zeros
    const double r = sqrt(ss / NI);
    const double ir = r >= (double)R_MIN ? 1.0 / r : 0.0;
    float *xo = X + (long long)q * NI;
#pragma unroll
    for (int u = 0; u < (NI + 31) / 32; ++u) {
        const int k = lane + 32 * u;
        if (k < NI) xo[k] = (float)(raw[w][k] * ir);
    }
    const long long p = x + (long long)pitch * (y + (long long)ny * z);
    float yee[6];  // every lane the same values; lane c writes component c
    yee_centre(raw[w], ndt, ce[p], ca ? ca[p] : 1.f, ca != nullptr, x == lo.x, y == lo.y, z == lo.z, yee);
    const unsigned m = tangent_mask(x - lo.x, y - lo.y, z - lo.z, hi.x - lo.x, hi.y - lo.y, hi.z - lo.z);
#pragma unroll
    for (int c = 0; c < 6; ++c)
        if (lane == c)
            Y[(long long)q * NO + c] = (m >> c) & 1u ? (float)(((double)nxt[c * fstride + p] - (double)yee[c]) * ir) : 0.f;
}

// -------------------------------------------------- layer update (fused)

// Tensor-core contraction of the fused layer kernel: mma.sync m16n8k8 with
// TF32 operands and FP32 accumulation, each operand split in two TF32 terms
// (x = hi + lo, hi = tf32(x), lo = tf32(x - hi)) and the product taken as
// lo*hi + hi*lo + hi*hi ("3xTF32"): ~22 significant bits per operand, the
// dropped lo*lo term below FP32 rounding of the sum, so the layer keeps
// FP32 accuracy.
// x rounded to TF32 (13 bits fewer, to nearest, ties away) as two integer
// operations: cvt.rna.tf32.f32 gives the same for finite values and infinities,
// as a longer sequence on this part.  A NaN comes out as a number (the carry of
// 0x7fffffff, which arithmetic makes, leaves -0), in lo as in hi, and so does the
// inf - inf of an infinity's lo.  split_tf32 is for values whose NaN is found
// elsewhere; split_tf32_nan has one in hi where x is not finite.
__device__ __forceinline__ unsigned tf32_rna(float x)
{
    return (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
}
__device__ __forceinline__ void split_tf32(float x, unsigned &hi, unsigned &lo)
{
    hi = tf32_rna(x);
    lo = tf32_rna(__fsub_rn(x, __uint_as_float(hi)));
}
__device__ __forceinline__ void split_tf32_nan(float x, unsigned &hi, unsigned &lo)
{
    hi = tf32_rna(x);
    const float d = __fsub_rn(x, __uint_as_float(hi));
    lo = tf32_rna(d);
    if (d != d) hi = 0x7fc00000u;
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9},"
                 " {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// acc[n] += A B over one step of k, for the eight unit tiles n: w points at
// this lane's fragment of unit tile 0.  Each of the three products runs over
// all tiles before the next, so an accumulator's next use is eight
// instructions away.
__device__ __forceinline__ void contract(float (&acc)[8][4], const unsigned (&ah)[4], const unsigned (&al)[4], const uint4 *w)
{
    uint4 b[8];
#pragma unroll
    for (int n = 0; n < 8; ++n) b[n] = w[8 * n];
#pragma unroll
    for (int n = 0; n < 8; ++n) mma_tf32(acc[n], al, b[n].x, b[n].y);
#pragma unroll
    for (int n = 0; n < 8; ++n) mma_tf32(acc[n], ah, b[n].z, b[n].w);
#pragma unroll
    for (int n = 0; n < 8; ++n) mma_tf32(acc[n], ah, b[n].x, b[n].y);
}

// The layer is the domain's six faces.  On a face the third of a stencil
// beyond the wall is zero, which leaves 216 of the 324 inputs: 24 planes (the
// face's own and the next one inward, two levels, six components) x 3 x 3
// taps in the face.  A group of four warps takes patches of 16 x 4 cells of a
// face, stages their footprint (24 planes of 18 x 6 cells) and contracts it as an implicit
// convolution: a warp holds one row of 16 cells, k runs over taps and, within
// a tap, over the planes, so an operand fragment is read straight from the
// footprint at the tap's offset.
//
// What bounds it: the tensor pipe (3 x 280 k-rows of 64 units a cell, 8
// cycles an m16n8k8), beside the weights' fragments from shared memory (256
// of 394 cycles a k-step).  The kernel before it gathered each cell's 324
// inputs on their own (81 copies of 4 bytes a thread and tile, six times the
// footprint) and moved the hidden layers through shared memory, with five
// block barriers a tile: 160^3 (152 k cells) 258 us, now 105 (56 % of the
// tensor pipe), a step 329 -> 157.  The
// hidden layers now stay in registers: an accumulator fragment holds units 2q
// and 2q + 1 of a row where an operand fragment wants k = q and q + 4, so the
// second layer's k is taken in that order.
constexpr int PU = 16, PV = 4;             // cells of a patch
constexpr int FROW = 20, FPL = 136;        // footprint: floats of a row (18 used), of a plane (6 rows)
constexpr int NPL = 24, KF = 9 * NPL;      // planes, inputs of a face cell
constexpr int WP = 66;                     // pitch of a row of weight fragments, in fragments of 16 bytes
static_assert((PU + 2) * (PV + 2) > 96 && (PU + 2) * (PV + 2) <= 128 && NPL == 6 * 4, "four elements of six planes a lane");
static_assert(FPL >= (PV + 2) * FROW, "a plane's rows");
static_assert(FPL % 32 == 8, "the four planes of a fragment on disjoint banks");
static_assert(WP % 8 == 2, "the fragments of eight lanes on disjoint banks");
constexpr int LS_W1 = 0, LS_W2 = LS_W1 + 4 * (KF / 2) * WP, LS_F = LS_W2 + 4 * (NH / 2) * WP, LS_W3 = LS_F + 4 * NPL * FPL,
              LS_B = LS_W3 + NO * NH, LS_END = LS_B + 2 * NH + 8;
static_assert(LS_W2 % 4 == 0 && LS_F % 4 == 0 && LS_W3 % 4 == 0, "16-byte copies");
constexpr size_t LAYER_SMEM = sizeof(float) * LS_END;
static_assert(LAYER_SMEM <= 227 * 1024, "one CTA's shared memory");

// Input k of the network that face f (0..5 = x low, x high, y low, ...) reads
// as plane p = (depth * 2 + level) * 6 + component at tap (dv, du).
__device__ __host__ __forceinline__ int face_input(int f, int p, int dv, int du)
{
    const int c = p % 6, lev = (p / 6) % 2, depth = p / 12;
    const int axis = f >> 1, dn = f & 1 ? 1 - depth : 1 + depth;  // offset + 1 along the face's normal
    // u, v: the other two axes, the lower one first
    const int dx = axis == 0 ? dn : du, dy = axis == 1 ? dn : (axis == 0 ? du : dv), dz = axis == 2 ? dn : dv;
    return (lev * 6 + c) * 27 + dz * 9 + dy * 3 + dx;
}

// The first two layers' weights as the layer kernel reads them: fragment (step,
// q, unit) holds the rows k = q and q + 4 of an eight-row step of k, split:
// {hi(q), hi(q + 4), lo(q), lo(q + 4)}, so that one 16-byte load gives the two
// register pairs of an operand.  W1 of each face [6][KF / 8][4][NH] (step tap *
// 3 + p / 8, row p % 8), then W2 [NH / 8][4][NH] (step j, rows q and q + 4:
// inputs 8j + 2q and 8j + 2q + 1).
__global__ void __launch_bounds__(256) weight_image_kernel(const float *__restrict__ P, uint4 *__restrict__ img)
{
    const int e = blockIdx.x * 256 + threadIdx.x;
    constexpr int N1 = 6 * KF / 2 * NH;
    if (e >= N1 + NH / 2 * NH) return;
    float v[2];
    if (e < N1) {
        const int u = e % NH, q = (e / NH) % 4, step = (e / (4 * NH)) % (KF / 8), f = e / (4 * NH * (KF / 8));
        const int tap = step / 3, p = 8 * (step % 3) + q;
        for (int i = 0; i < 2; ++i) v[i] = P[OFF_W1 + u * NI + face_input(f, p + 4 * i, tap / 3, tap % 3)];
        // a weight of the third left out that is not finite makes its unit NaN too
        // (times the zeros beyond the wall), here in the unit's first row
        if (step == 0 && q == 0)
            for (int k = 0; k < NI; ++k)
                if (!isfinite(P[OFF_W1 + u * NI + k])) v[0] = nanf("");
    } else {
        const int r = e - N1, u = r % NH, q = (r / NH) % 4, j = r / (4 * NH);
        for (int i = 0; i < 2; ++i) v[i] = P[OFF_W2 + u * NH + 8 * j + 2 * q + i];
    }
    uint4 o;
    split_tf32_nan(v[0], o.x, o.z);
    split_tf32_nan(v[1], o.y, o.w);
    img[e] = o;
}

// x, y, z of in-plane (u, v) of face f at depth d
__device__ __forceinline__ void face_cell(const LearnedGeo &g, int f, int u, int v, int d, int &x, int &y, int &z)
{
    const int axis = f >> 1, n = axis == 0 ? g.nx : axis == 1 ? g.ny : g.nz, w = f & 1 ? n - 1 - d : d;
    x = axis == 0 ? w : u;
    y = axis == 1 ? w : (axis == 0 ? u : v);
    z = axis == 2 ? w : v;
}

// The two planes of each face of the six components, as they are now: plane
// (face, depth) of component c at face's offset + ((depth * 6 + c) * nv + v) *
// nu + u.  A block takes one face, both depths (neighbours in memory on the x
// faces) and one component.
__global__ void __launch_bounds__(256) snapshot_kernel(const __grid_constant__ LearnedGeo g, const float *__restrict__ fld,
                                                       long long fs, int pitch, float *__restrict__ snap)
{
    const int f = blockIdx.y / 6, c = blockIdx.y % 6;
    const LearnedFace &F = g.face[f];
    const int n = F.nu * F.nv;
    for (int e = blockIdx.x * 256 + threadIdx.x; e < n; e += gridDim.x * 256) {
        const int v = e / F.nu, u = e - v * F.nu;
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            if (d >= F.depth) break;
            int x, y, z;
            face_cell(g, f, u, v, d, x, y, z);
            snap[F.snap + (long long)(d * 6 + c) * n + e] = fld[c * fs + x + (long long)pitch * (y + (long long)g.ny * z)];
        }
    }
}

// tanh without a branch, for the 128 evaluations a thread and patch that the
// tensor cores otherwise wait for.  Below 1 the seventh convergent of
// Lambert's continued fraction x / (1 + x^2 / (3 + x^2 / (5 + ...))) as x less
// x times a quotient of polynomials in x^2 (its truncation error is under 1e-9
// there), above it 1 - 2 / (exp(2 |x|) + 1); one reciprocal for both, refined
// by a Newton step.  Over all floats of [2^-14, 12] on this GPU: 1.25 units in the
// last place at most, near 1 (tanhf: 1.82); odd, NaN for NaN.
__device__ __forceinline__ float tanh_fast(float x)
{
    const float a = fabsf(x) > 10.f ? 10.f : fabsf(x), t = __fmul_rn(a, a);  // (NaN stays)
    float e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(__fmul_rn(a, 2.885390081777927f)));  // 2 log2(e)
    const bool small = a < 1.f;
    const float ns = __fmul_rn(__fmul_rn(a, t), __fmaf_rn(t, __fmaf_rn(t, 27.f, 2772.f), 45045.f));
    const float ds = __fmaf_rn(t, __fmaf_rn(t, __fmaf_rn(t, 28.f, 3150.f), 62370.f), 135135.f);
    const float n = small ? ns : 2.f, d = small ? ds : __fadd_rn(e, 1.f);
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(d));
    r = __fmaf_rn(r, __fmaf_rn(-d, r, 1.f), r);
    const float y = __fmaf_rn(-n, r, small ? a : 1.f);
    return copysignf(y, x);
}

// Footprint of one patch into shared memory by asynchronous 4-byte copies;
// cells beyond the face (and a second plane that does not exist) read 0.  A
// warp takes six planes (`place`: where the lane's four elements of a plane lie,
// row << 8 | column, the same for every plane and patch).
__device__ __forceinline__ void stage_patch(const LearnedGeo &g, int f, int u0, int v0, const float *__restrict__ cur,
                                            const float *__restrict__ prev, const int (&place)[4], float *dst)
{
    const LearnedFace &F = g.face[f];
    const int n = F.nu * F.nv, w = (threadIdx.x >> 5) & 3;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = place[i] >> 8, col = place[i] & 255;
        const int u = u0 + col - 1, v = v0 + row - 1;
        const bool in = (unsigned)u < (unsigned)F.nu && (unsigned)v < (unsigned)F.nv;
        const int o = in ? v * F.nu + u : 0;
        const unsigned a = (unsigned)__cvta_generic_to_shared(dst + w * FPL + row * FROW + col);
        if (i < 3 || row < PV + 2) {
#pragma unroll
            for (int k = 0; k < 6; ++k) {  // planes w + 4 k: depth of plane p is p / 12, level (p / 6) % 2
                const int p = w + 4 * k, d = k / 3, lc = p - 12 * d;
                const bool ok = in && d < F.depth;
                const float *const src = (lc < 6 ? cur : prev) + F.snap + (long long)(ok ? d * 6 + lc % 6 : 0) * n + o;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(a + 16u * k * FPL), "l"(src), "r"(ok ? 4 : 0)
                             : "memory");
            }
        }
    }
}

__device__ __forceinline__ void copy16(float *dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Corrections r f(x / r) of the face cells from the snapshots of S^n (cur) and
// S^{n-1} (prev): component o of cell `id` at out[o * cells + id].  Persistent:
// a CTA takes a run of consecutive patches, so it changes face (and first-layer
// weights) once at most in the usual grids.  Its two groups of four warps (one
// of each on an SM sub-partition) take the run's patches in turn, the second
// half a patch behind: while one evaluates tanh the other has the tensor cores.
__device__ __forceinline__ void bar_group(int grp) { asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory"); }

__global__ void __launch_bounds__(256, 1) layer_kernel(const __grid_constant__ LearnedGeo g, const float *__restrict__ P,
                                                       const uint4 *__restrict__ img, const float *__restrict__ cur,
                                                       const float *__restrict__ prev, float *__restrict__ out)
{
    extern __shared__ __align__(16) float sm[];
    float *const W1 = sm + LS_W1, *const W2 = sm + LS_W2, *const FP = sm + LS_F, *const W3 = sm + LS_W3;
    float *const b1 = sm + LS_B, *const b2 = b1 + NH, *const b3 = b2 + NH;
    const int tid = threadIdx.x, lane = tid & 31, w = (tid >> 5) & 3, grp = tid >> 7, gr = lane >> 2, q = lane & 3;
    const int per = (g.patches + gridDim.x - 1) / gridDim.x;
    const int first = blockIdx.x * per, last = min(first + per, g.patches);
    if (first >= last) return;
    auto face_of = [&](int patch) {
        int f = 0;
        while (patch >= g.face[f].patch0 + g.face[f].pu * g.face[f].pv) ++f;
        return f;
    };
    auto origin = [&](int patch, int f, int &u0, int &v0) {
        const LearnedFace &F = g.face[f];
        const int r = patch - F.patch0;
        u0 = F.u0 + PU * (r % F.pu);
        v0 = F.v0 + PV * (r / F.pu);
    };
    auto load_w1 = [&](int f) {
        const float *const src = reinterpret_cast<const float *>(img + (size_t)f * (KF / 2) * NH);
        for (int e = tid; e < KF / 2 * NH; e += 256) copy16(W1 + 4 * ((e / NH) * WP + e % NH), src + 4 * e);
    };
    int place[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) place[i] = (lane + 32 * i) / (PU + 2) << 8 | (lane + 32 * i) % (PU + 2);
    for (int e = tid; e < NO * NH; e += 256) W3[e] = P[OFF_W3 + e];
    if (tid < NH) {
        b1[tid] = P[OFF_B1 + tid];
        b2[tid] = P[OFF_B2 + tid];
    }
    if (tid < NO) b3[tid] = P[OFF_B3 + tid];
    {
        const float *const src = reinterpret_cast<const float *>(img + (size_t)6 * (KF / 2) * NH);
        for (int e = tid; e < NH / 2 * NH; e += 256) copy16(W2 + 4 * ((e / NH) * WP + e % NH), src + 4 * e);
    }
    float *const fpg = FP + grp * 2 * NPL * FPL;
    for (int seg = first, seg_end; seg < last; seg = seg_end) {  // the run's patches on one face
        const int f = face_of(seg);
        const LearnedFace &F = g.face[f];
        seg_end = min(last, F.patch0 + F.pu * F.pv);
        int u0, v0;
        if (seg != first) __syncthreads();  // everybody is past the previous face's weights
        load_w1(f);
        if (seg + grp < seg_end) {
            origin(seg + grp, f, u0, v0);
            stage_patch(g, f, u0, v0, cur, prev, place, fpg);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    for (int patch = seg + grp, it = 0; patch < seg_end; patch += 2, ++it) {
        if (it) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            bar_group(grp);  // this patch's footprint has landed; the other buffer is free
        }
        origin(patch, f, u0, v0);
        if (patch + 2 < seg_end) {
            int nu0, nv0;
            origin(patch + 2, f, nu0, nv0);
            stage_patch(g, f, nu0, nv0, cur, prev, place, fpg + ((it + 1) & 1) * NPL * FPL);
        }
        // the second group's first patch starts once the first group is through
        // its first layer
        if (it == 0 && grp == 1) asm volatile("bar.sync 3, 256;" ::: "memory");
        const float *const fp = fpg + (it & 1) * NPL * FPL + w * FROW + gr;
        float acc[8][4];
#pragma unroll
        for (int n = 0; n < 8; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
        // layer 1 on the unnormalised inputs, and the sum of their squares (rows
        // gr and gr + 8 of the warp's 16 cells)
        float ss0 = 0.f, ss1 = 0.f;
        const uint4 *wr = reinterpret_cast<const uint4 *>(W1) + q * WP + gr;
#pragma unroll 1
        for (int tap = 0; tap < 9; ++tap) {
            const float *const ft = fp + (tap / 3) * FROW + tap % 3;
#pragma unroll
            for (int j = 0; j < 3; ++j, wr += 4 * WP) {
                const float x0 = ft[(8 * j + q) * FPL], x1 = ft[(8 * j + q) * FPL + 8];
                const float x2 = ft[(8 * j + q + 4) * FPL], x3 = ft[(8 * j + q + 4) * FPL + 8];
                ss0 = __fmaf_rn(x0, x0, __fmaf_rn(x2, x2, ss0));
                ss1 = __fmaf_rn(x1, x1, __fmaf_rn(x3, x3, ss1));
                unsigned ah[4], al[4];
                split_tf32(x0, ah[0], al[0]);
                split_tf32(x1, ah[1], al[1]);
                split_tf32(x2, ah[2], al[2]);
                split_tf32(x3, ah[3], al[3]);
                contract(acc, ah, al, wr);
            }
        }
#pragma unroll
        for (int d = 1; d < 4; d <<= 1) {
            ss0 = __fadd_rn(ss0, __shfl_xor_sync(0xffffffffu, ss0, d));
            ss1 = __fadd_rn(ss1, __shfl_xor_sync(0xffffffffu, ss1, d));
        }
        const float r0 = sqrtf(ss0 / NI), r1 = sqrtf(ss1 / NI);
        // smaller r: the cell keeps its value; a NaN in the stencil is in r, and so in
        // the correction
        const bool live0 = !(r0 < R_MIN), live1 = !(r1 < R_MIN);
        const float ir0 = live0 ? 1.f / r0 : 0.f, ir1 = live1 ? 1.f / r1 : 0.f;
        if (it == 0 && grp == 0 && seg + 1 < seg_end) asm volatile("bar.arrive 3, 256;" ::: "memory");
        // H1 = tanh((W1 x) / r + b1), in place.  A NaN among a row's (a weight's, an
        // overflow's) is the one with bit 30 set, and goes into its sums of layer 3
        unsigned m0 = 0, m1 = 0;
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const float2 b = *reinterpret_cast<const float2 *>(b1 + 8 * n + 2 * q);
            acc[n][0] = tanh_fast(__fmaf_rn(acc[n][0], ir0, b.x));
            acc[n][1] = tanh_fast(__fmaf_rn(acc[n][1], ir0, b.y));
            acc[n][2] = tanh_fast(__fmaf_rn(acc[n][2], ir1, b.x));
            acc[n][3] = tanh_fast(__fmaf_rn(acc[n][3], ir1, b.y));
            m0 |= __float_as_uint(acc[n][0]) | __float_as_uint(acc[n][1]);
            m1 |= __float_as_uint(acc[n][2]) | __float_as_uint(acc[n][3]);
        }
        // layer 2: operand fragment j from accumulator fragment j
        float acc2[8][4];
#pragma unroll
        for (int n = 0; n < 8; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc2[n][e] = 0.f;
        const uint4 *const w2 = reinterpret_cast<const uint4 *>(W2) + q * WP + gr;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            unsigned ah[4], al[4];
            split_tf32(acc[j][0], ah[0], al[0]);
            split_tf32(acc[j][2], ah[1], al[1]);
            split_tf32(acc[j][1], ah[2], al[2]);
            split_tf32(acc[j][3], ah[3], al[3]);
            contract(acc2, ah, al, w2 + 4 * j * WP);
        }
        // layer 3 in FP32: a lane's 16 units of its two rows, then the four lanes of a row
        float y0[NO], y1[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            y0[o] = m0 & 0x40000000u ? nanf("") : 0.f;
            y1[o] = m1 & 0x40000000u ? nanf("") : 0.f;
        }
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const float2 b = *reinterpret_cast<const float2 *>(b2 + 8 * n + 2 * q);
            const float h00 = tanh_fast(__fadd_rn(acc2[n][0], b.x)), h01 = tanh_fast(__fadd_rn(acc2[n][1], b.y));
            const float h10 = tanh_fast(__fadd_rn(acc2[n][2], b.x)), h11 = tanh_fast(__fadd_rn(acc2[n][3], b.y));
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                const float2 c = *reinterpret_cast<const float2 *>(W3 + o * NH + 8 * n + 2 * q);
                y0[o] = __fmaf_rn(h01, c.y, __fmaf_rn(h00, c.x, y0[o]));
                y1[o] = __fmaf_rn(h11, c.y, __fmaf_rn(h10, c.x, y1[o]));
            }
        }
#pragma unroll
        for (int o = 0; o < NO; ++o)
#pragma unroll
            for (int d = 1; d < 4; d <<= 1) {
                y0[o] = __fadd_rn(y0[o], __shfl_xor_sync(0xffffffffu, y0[o], d));
                y1[o] = __fadd_rn(y1[o], __shfl_xor_sync(0xffffffffu, y1[o], d));
            }
        // lane q writes components q and q + 4 of cells (u0 + gr, v0 + w) and (u0 + gr + 8, v0 + w)
        const int v = v0 + w;
        if (v < F.v1) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int u = u0 + gr + 8 * h;
                if (u >= F.u1) continue;
                const long long id = F.cell0 + (long long)(v - F.v0) * (F.u1 - F.u0) + (u - F.u0);
                const float r = h ? (live1 ? r1 : 0.f) : (live0 ? r0 : 0.f);
#pragma unroll
                for (int o = 0; o < NO; ++o)
                    if ((o & 3) == q) out[o * g.cells + id] = __fmul_rn(r, __fadd_rn(h ? y1[o] : y0[o], b3[o]));
            }
        }
    }
    }
}

// The corrections added to the components that the walls get wrong.
__global__ void __launch_bounds__(256) scatter_kernel(const __grid_constant__ LearnedGeo g, float *__restrict__ fld,
                                                      long long fs, int pitch, const float *__restrict__ vals)
{
    const LearnedFace &F = g.face[blockIdx.y];
    const int nu = F.u1 - F.u0, n = nu * (F.v1 - F.v0);
    const int e = blockIdx.x * 256 + threadIdx.x;
    if (e >= n) return;
    const int v = e / nu, u = e - v * nu;
    int x, y, z;
    face_cell(g, blockIdx.y, F.u0 + u, F.v0 + v, 0, x, y, z);
    const unsigned m = tangent_mask(x, y, z, g.nx, g.ny, g.nz);
    const long long p = x + (long long)pitch * (y + (long long)g.ny * z);
#pragma unroll
    for (int c = 0; c < NO; ++c)
        if ((m >> c) & 1u) fld[c * fs + p] = __fadd_rn(fld[c * fs + p], vals[c * g.cells + F.cell0 + e]);
}

} // namespace

// ------------------------------------------------------------ internal API

size_t mlp_scratch_bytes(int batch, long long n) { return scratch_bytes(batch, n); }

cudaError_t mlp_forward(const float *params, const float *X, long long n, float *Y, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    CKE(net_configure<true>());
    return net<true>(params, X, nullptr, nullptr, n, Y, nullptr, nullptr, st);
}

cudaError_t mlp_grad(const float *params, const float *X, const float *T, int n, float *grad, double *loss_host,
                     void *scratch, int batch, cudaStream_t st)
{
    if (n > batch) return cudaErrorInvalidValue;
    Scratch s = carve(scratch, batch, 0);
    CKE(net_configure<false>());
    CKE(cudaMemsetAsync(s.loss, 0, sizeof(double), st));
    CKE(net<false>(params, X, nullptr, T, n, nullptr, s.part, s.loss_part, st));
    grad_kernel<false><<<(NPARAM + 31) / 32, 256, 0, st>>>(s.part, s.loss_part, net_parts(n), nullptr, nullptr, nullptr,
                                                           0.f, 1.f, 1.f, grad, s.loss);
    CKE(cudaGetLastError());
    double l = 0.0;
    CKE(cudaMemcpyAsync(&l, s.loss, sizeof(double), cudaMemcpyDeviceToHost, st));
    CKE(cudaStreamSynchronize(st));
    if (loss_host) *loss_host = l / ((double)n * NO);
    return cudaSuccess;
}

cudaError_t mlp_train(float *params, const float *X, const float *T, long long n, int batch, int epochs, double lr,
                      unsigned long long seed, void *scratch, cudaStream_t st, double *last_epoch_loss)
{
    Scratch s = carve(scratch, batch, n);
    CKE(net_configure<false>());
    CKE(cudaMemsetAsync(s.m, 0, sizeof(float) * NPARAM, st));
    CKE(cudaMemsetAsync(s.v, 0, sizeof(float) * NPARAM, st));
    CKE(cudaMemsetAsync(s.loss, 0, sizeof(double), st));
    std::mt19937_64 rng(seed);
    std::vector<int> perm((size_t)n);
    for (long long i = 0; i < n; ++i) perm[(size_t)i] = (int)i;
    const long long nb = n / batch;  // whole batches only
    const int parts = net_parts(batch);
    long long t = 0;
    // the host shuffles the next epoch's order while the GPU runs this one:
    // an epoch's order is copied from a host buffer of its own, taken again
    // two epochs later, after that copy
    std::vector<int> order[2];
    struct Events {
        cudaEvent_t e[2] = {nullptr, nullptr};
        ~Events()
        {
            for (cudaEvent_t x : e)
                if (x) cudaEventDestroy(x);
        }
    } copied;
    for (int ep = 0; ep < epochs; ++ep) {
        std::shuffle(perm.begin(), perm.end(), rng);
        cudaEvent_t &ev = copied.e[ep & 1];
        if (ev) CKE(cudaEventSynchronize(ev));
        else CKE(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        order[ep & 1] = perm;
        CKE(cudaMemsetAsync(s.loss, 0, sizeof(double), st));
        CKE(cudaMemcpyAsync(s.rows, order[ep & 1].data(), sizeof(int) * (size_t)n, cudaMemcpyHostToDevice, st));
        CKE(cudaEventRecord(ev, st));
        for (long long b = 0; b < nb; ++b) {
            CKE(net<false>(params, X, s.rows + b * batch, T, batch, nullptr, s.part, s.loss_part, st));
            ++t;
            const float c1 = (float)(1.0 - std::pow(0.9, (double)t)), c2 = (float)(1.0 - std::pow(0.999, (double)t));
            grad_kernel<true><<<(NPARAM + 31) / 32, 256, 0, st>>>(s.part, s.loss_part, parts, params, s.m, s.v, (float)lr,
                                                                  c1, c2, nullptr, s.loss);
            CKE(cudaGetLastError());
        }
    }
    double l = 0.0;
    CKE(cudaMemcpyAsync(&l, s.loss, sizeof(double), cudaMemcpyDeviceToHost, st));
    CKE(cudaStreamSynchronize(st));
    if (last_epoch_loss) *last_epoch_loss = epochs > 0 && nb > 0 ? l / ((double)nb * batch * NO) : 0.0;
    return cudaSuccess;
}

cudaError_t mlp_record(const float *prev, const float *cur, const float *nxt, long long fstride, int pitch, int ny,
                       const int lo[3], const int hi[3], const int *cells, int n, const float *ce, const float *ca,
                       float neg_dt, float *X, float *Y, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    record_kernel<<<(n + RW - 1) / RW, 32 * RW, 0, st>>>(prev, cur, nxt, fstride, pitch, ny,
                                                         make_int3(lo[0], lo[1], lo[2]), make_int3(hi[0], hi[1], hi[2]),
                                                         cells, n, ce, ca, neg_dt, X, Y);
    return cudaGetLastError();
}

cudaError_t mlp_record_box(const float *f, long long fstride, int pitch, int ny, const int lo[3], const int hi[3],
                           float *dst, cudaStream_t st)
{
    const long long bc = (long long)(hi[0] - lo[0]) * (hi[1] - lo[1]) * (hi[2] - lo[2]);
    record_box_kernel<<<(unsigned)((bc + 255) / 256), 256, 0, st>>>(f, fstride, pitch, ny, make_int3(lo[0], lo[1], lo[2]),
                                                                     make_int3(hi[0], hi[1], hi[2]), dst);
    return cudaGetLastError();
}

LearnedGeo learned_geometry(int nx, int ny, int nz)
{
    LearnedGeo g = {};
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    const int n[3] = {nx, ny, nz};
    long long snap = 0, cell = 0;
    int patch = 0;
    for (int f = 0; f < 6; ++f) {
        LearnedFace &F = g.face[f];
        const int axis = f >> 1, ua = axis == 0 ? 1 : 0, va = axis == 2 ? 1 : 2;
        F.nu = n[ua];
        F.nv = n[va];
        F.depth = std::min(2, n[axis]);
        // each cell belongs to one face: all of the z faces', of the y faces' those
        // between them, of the x faces' the rest; one face where a domain is one cell thick
        F.u0 = axis == 0 ? std::min(1, ny) : 0;
        F.u1 = axis == 0 ? std::max(F.u0, ny - 1) : F.nu;
        F.v0 = axis == 2 ? 0 : std::min(1, nz);
        F.v1 = axis == 2 ? F.nv : std::max(F.v0, nz - 1);
        if ((f & 1) && n[axis] == 1) F.u1 = F.u0;
        const bool none = F.u1 <= F.u0 || F.v1 <= F.v0;
        F.pu = none ? 0 : (F.u1 - F.u0 + PU - 1) / PU;
        F.pv = none ? 0 : (F.v1 - F.v0 + PV - 1) / PV;
        if (none) F.u1 = F.u0;
        F.snap = snap;
        F.cell0 = cell;
        F.patch0 = patch;
        snap += 12ll * F.nu * F.nv;
        cell += (long long)(F.u1 - F.u0) * (F.v1 - F.v0);
        patch += F.pu * F.pv;
    }
    g.snap_floats = snap;
    g.cells = cell;
    g.patches = patch;
    return g;
}

size_t learned_image_bytes() { return sizeof(uint4) * (6 * (size_t)(KF / 2) * NH + NH / 2 * NH); }

cudaError_t learned_layer_configure(const float *params, void *image, cudaStream_t st)
{
    CKE(cudaFuncSetAttribute(layer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LAYER_SMEM));
    weight_image_kernel<<<((6 * KF + NH) / 2 * NH + 255) / 256, 256, 0, st>>>(params, (uint4 *)image);
    return cudaGetLastError();
}

cudaError_t learned_snapshot(const LearnedGeo &g, const float *f, long long fs, int pitch, float *snap, cudaStream_t st)
{
    const long long n = std::max(std::max((long long)g.nx * g.ny, (long long)g.nx * g.nz), (long long)g.ny * g.nz);
    snapshot_kernel<<<dim3((unsigned)std::min<long long>((n + 255) / 256, 4096), 36), 256, 0, st>>>(g, f, fs, pitch, snap);
    return cudaGetLastError();
}

cudaError_t learned_layer_predict(const LearnedGeo &g, const float *params, const void *image, const float *cur,
                                  const float *prev, float *out, int grid, cudaStream_t st)
{
    layer_kernel<<<std::min(grid, g.patches), 256, LAYER_SMEM, st>>>(g, params, (const uint4 *)image, cur, prev, out);
    return cudaGetLastError();
}

cudaError_t learned_layer_scatter(const LearnedGeo &g, float *f, long long fs, int pitch, const float *vals,
                                  cudaStream_t st)
{
    int most = 0;
    for (const LearnedFace &F : g.face) most = std::max(most, (F.u1 - F.u0) * (F.v1 - F.v0));
    scatter_kernel<<<dim3((unsigned)((most + 255) / 256), 6), 256, 0, st>>>(g, f, fs, pitch, vals);
    return cudaGetLastError();
}
