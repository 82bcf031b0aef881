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
// a simulation step is one fused persistent kernel: it gathers the stencils
// of 64 layer cells into shared memory and runs the three layers on them
// with the weights resident in shared memory, the two large contractions on
// the tensor cores (mma.sync TF32, three-term split for FP32 accuracy).
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
__device__ __forceinline__ unsigned tf32_rna(float x)
{
    unsigned r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ void split_tf32(float x, unsigned &hi, unsigned &lo)
{
    hi = tf32_rna(x);
    lo = tf32_rna(__fsub_rn(x, __uint_as_float(hi)));
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                         unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9},"
                 " {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Shared tiles [k][64] (k = input feature or unit, 64 = cells or units) are
// stored with the column index XOR-swizzled by (k mod 4) * 8, so the
// fragment loads of a warp (rows k .. k+3, eight consecutive columns each)
// hit 32 different banks.
__device__ __forceinline__ int swz(int k, int c) { return c ^ ((k & 3) << 3); }

// D[64 x 64] of this CTA's eight warps (warp w: rows 16*(w%4).., columns
// 32*(w/4).., four m16n8 tiles) = sum_k A[k][row] B[k][col] over K (a
// multiple of 8; A, B swizzled [k][64] tiles in shared memory).
template <int K>
__device__ __forceinline__ void warp_gemm_3xtf32(const float *A, const float *B, float (&acc)[4][4])
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int g = lane >> 2, q = lane & 3;
    const int m0 = 16 * (w & 3), n0 = 32 * (w >> 2);
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
#pragma unroll 2
    for (int k0 = 0; k0 < K; k0 += 8) {
        const int ka = k0 + q, kb = k0 + q + 4;
        unsigned ah[4], al[4];
        split_tf32(A[ka * 64 + swz(ka, m0 + g)], ah[0], al[0]);
        split_tf32(A[ka * 64 + swz(ka, m0 + g + 8)], ah[1], al[1]);
        split_tf32(A[kb * 64 + swz(kb, m0 + g)], ah[2], al[2]);
        split_tf32(A[kb * 64 + swz(kb, m0 + g + 8)], ah[3], al[3]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + 8 * j + g;
            unsigned bh0, bl0, bh1, bl1;
            split_tf32(B[ka * 64 + swz(ka, n)], bh0, bl0);
            split_tf32(B[kb * 64 + swz(kb, n)], bh1, bl1);
            mma_tf32(acc[j], al[0], al[1], al[2], al[3], bh0, bh1);
            mma_tf32(acc[j], ah[0], ah[1], ah[2], ah[3], bl0, bl1);
            mma_tf32(acc[j], ah[0], ah[1], ah[2], ah[3], bh0, bh1);
        }
    }
}

// Shared memory of the fused layer kernel, in floats; the float4-read arrays
// come first, each a multiple of 64 floats, so they stay 16-byte aligned.
constexpr int LC = 64;  // layer cells per tile
constexpr int NIP = 328;  // NI padded to a multiple of 8 (zero rows)
static_assert((NIP - NI) * LC == 256, "one padding float per thread of the layer kernel");
constexpr int SM_W1T = NIP * NH, SM_W2T = NH * NH, SM_W3T = NH * NO, SM_XT = NIP * LC, SM_H = NH * LC;
constexpr size_t LAYER_SMEM =
    sizeof(float) * (SM_W1T + SM_W2T + SM_XT + 2 * SM_H + SM_W3T + 2 * NH + NO + 2 * LC + 4 * LC);

// Asynchronous 4-byte copy, global -> shared (cp.async, cached in L1).  With
// valid == false nothing is read and the shared word is zero-filled; src is
// then still an address inside the field array.
__device__ __forceinline__ void cp_async_4(float *dst, const float *src, bool valid)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Each band snapshot (six components at c * fstride, rows of `pitch`) is
// followed by its x slab: the planes x = 0, 1 (side 0) and x = nx-2, nx-1
// (side 1) of every component, y fastest, [comp][side][xd][z][y], so that
// the stencils of the cells on the two x faces (a full row apart from each
// other in the snapshot) are read with consecutive y across the lanes.
__device__ __host__ __forceinline__ long long xslab_floats(int ny, int nz) { return 24LL * ny * nz; }

// Stage the unnormalised stencils of `tile` into Xt ([k][cell], swizzled)
// with asynchronous copies: thread -> cell q = tid % 64 and three of the
// twelve (level, component) pairs, (tid / 64) * 3 + 0..2, each a 27-cell
// stencil; neighbour offsets are unrolled, validity is per axis, neighbours
// outside the domain and cells past the list are zero.  Cells on an x face
// read the x slab, the others the snapshot itself (same values).
__device__ __forceinline__ void stage_stencils(float *Xt, const float *__restrict__ cur,
                                               const float *__restrict__ prev, long long fstride, int pitch,
                                               int nx, int ny, int nz, const int *__restrict__ cells, int ncells,
                                               int tile)
{
    const int tid = threadIdx.x, q = tid & (LC - 1), p0 = (tid >> 6) * 3;
    const int cell = tile * LC + q;
    if (cell < ncells) {
        const int x = cells[3 * cell], y = cells[3 * cell + 1], z = cells[3 * cell + 2];
        const bool vx[3] = {x > 0, true, x + 1 < nx}, vy[3] = {y > 0, true, y + 1 < ny},
                   vz[3] = {z > 0, true, z + 1 < nz};
        const long long nyz = (long long)ny * nz;
        // address of (x', y', z') of component c: level base + c * cs + o0 + x' sx + y' sy + z' sz
        long long sx = 1, sy = pitch, sz = (long long)pitch * ny, cs = fstride, o0 = 0;
        if (x == 0 || x == nx - 1) {
            const int side = x == 0 ? 0 : 1, base = side ? nx - 2 : 0;
            sx = nyz, sy = 1, sz = ny, cs = 4 * nyz;
            o0 = 6 * fstride + (2 * side - base) * nyz;
        }
        const long long centre = o0 + x * sx + y * sy + z * sz;
        const long long ox[3] = {-sx, 0, sx}, oy[3] = {-sy, 0, sy}, oz[3] = {-sz, 0, sz};
#pragma unroll 1
        for (int pq = 0; pq < 3; ++pq) {
            const int pr = p0 + pq, lev = pr / 6, comp = pr - lev * 6;
            const float *src = (lev == 0 ? cur : prev) + comp * cs + centre;
#pragma unroll
            for (int d = 0; d < 27; ++d) {
                const int dx = d % 3, dy = (d / 3) % 3, dz = d / 9;
                const int k = pr * 27 + d;
                const bool ok = vx[dx] && vy[dy] && vz[dz];
                const float *a = ok ? src + (ox[dx] + oy[dy] + oz[dz]) : src;
                cp_async_4(&Xt[k * LC + swz(k, q)], a, ok);
            }
        }
    } else {
#pragma unroll
        for (int pq = 0; pq < 3; ++pq)
#pragma unroll
            for (int d = 0; d < 27; ++d) {
                const int k = (p0 + pq) * 27 + d;
                Xt[k * LC + swz(k, q)] = 0.f;
            }
    }
}

__global__ void __launch_bounds__(256, 1) layer_kernel(const float *__restrict__ P, const float *__restrict__ cur,
                                                       const float *__restrict__ prev, long long fstride, int pitch,
                                                       int nx, int ny, int nz, const int *__restrict__ cells,
                                                       int ncells, float *__restrict__ out)
{
    extern __shared__ __align__(16) float sm[];
    float *W1t = sm;                  // [k][unit]
    float *W2t = W1t + SM_W1T;        // [k][unit]
    float *Xt = W2t + SM_W2T;         // [k][cell]: the unnormalised stencil
    float *H1t = Xt + SM_XT;          // [unit][cell]
    float *H2t = H1t + SM_H;
    float *W3t = H2t + SM_H;          // [k][out]
    float *b1 = W3t + SM_W3T, *b2 = b1 + NH, *b3 = b2 + NH;
    float *rr = b3 + NO;              // r per cell
    float *ir = rr + LC;              // 1/r per cell (0 if r = 0)
    float *part = ir + LC;            // [4][cell] partial sums of x^2
    const int tid = threadIdx.x;
    const int ntiles = (ncells + LC - 1) / LC;
    // the first tile's stencils are in flight while the weights are loaded
    if ((int)blockIdx.x < ntiles)
        stage_stencils(Xt, cur, prev, fstride, pitch, nx, ny, nz, cells, ncells, blockIdx.x);
    for (int e = tid; e < NH * NI; e += 256) {
        const int u = e / NI, k = e - u * NI;
        W1t[k * NH + swz(k, u)] = P[OFF_W1 + e];
    }
    for (int e = tid; e < (NIP - NI) * NH; e += 256) W1t[NI * NH + e] = 0.f;  // padding rows
    for (int e = tid; e < NH * NH; e += 256) {
        const int u = e / NH, k = e - u * NH;
        W2t[k * NH + swz(k, u)] = P[OFF_W2 + e];
    }
    for (int e = tid; e < NO * NH; e += 256) {
        const int o = e / NH, k = e - o * NH;
        W3t[k * NO + o] = P[OFF_W3 + e];
    }
    if (tid < NH) {
        b1[tid] = P[OFF_B1 + tid];
        b2[tid] = P[OFF_B2 + tid];
    }
    if (tid < NO) b3[tid] = P[OFF_B3 + tid];
    Xt[NI * LC + tid] = 0.f;  // padding rows of the stencil (256 zeros), never staged over
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        cp_async_wait_all();
        __syncthreads();  // this tile's stencils have landed; the previous tile is done with H / rr
        {
            // sum of squares of the thread's own 81 staged values, in staging order
            const int q = tid & (LC - 1), p0 = (tid >> 6) * 3;
            float ss = 0.f;
#pragma unroll
            for (int pq = 0; pq < 3; ++pq)
#pragma unroll
                for (int d = 0; d < 27; ++d) {
                    const int k = (p0 + pq) * 27 + d;
                    const float v = Xt[k * LC + swz(k, q)];
                    ss = __fmaf_rn(v, v, ss);
                }
            part[(tid >> 6) * LC + q] = ss;
        }
        __syncthreads();
        if (tid < LC) {
            const float ss = part[tid] + part[LC + tid] + part[2 * LC + tid] + part[3 * LC + tid];
            const float r = sqrtf(ss / NI);
            const bool live = r >= R_MIN;  // smaller r: the cell keeps its value
            rr[tid] = live ? r : 0.f;
            ir[tid] = live ? 1.f / r : 0.f;
        }
        __syncthreads();
        // layers 1 and 2 on the tensor cores (3xTF32): H1 = tanh((W1 x) / r +
        // b1), H2 = tanh(W2 H1 + b2); warp w holds cells 16*(w%4) + g (+8) and
        // units 32*(w/4) + 8j + 2q (+1) of its accumulator fragments
        {
            const int lane = tid & 31, w = tid >> 5, g = lane >> 2, q = lane & 3;
            const int m0 = 16 * (w & 3), n0 = 32 * (w >> 2);
            float acc[4][4];
            warp_gemm_3xtf32<NIP>(Xt, W1t, acc);
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int cell = m0 + g + 8 * (e >> 1), unit = n0 + 8 * j + 2 * q + (e & 1);
                    H1t[unit * LC + swz(unit, cell)] = tanhf(__fmaf_rn(acc[j][e], ir[cell], b1[unit]));
                }
            __syncthreads();  // every warp is past layer 1's reads of Xt
            // the next tile's stencils fly while layers 2 and 3 run
            const int next = tile + gridDim.x;
            if (next < ntiles) stage_stencils(Xt, cur, prev, fstride, pitch, nx, ny, nz, cells, ncells, next);
            warp_gemm_3xtf32<NH>(H1t, W2t, acc);
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int cell = m0 + g + 8 * (e >> 1), unit = n0 + 8 * j + 2 * q + (e & 1);
                    H2t[unit * LC + swz(unit, cell)] = tanhf(__fadd_rn(acc[j][e], b2[unit]));
                }
        }
        __syncthreads();
        // layer 3: the correction r f added to the Yee step later
        for (int e = tid; e < LC * NO; e += 256) {
            const int q = e / NO, o = e - q * NO;
            const int cell = tile * LC + q;
            if (cell >= ncells) continue;
            float f = b3[o];
            for (int k = 0; k < NH; ++k) f = __fmaf_rn(H2t[k * LC + swz(k, q)], W3t[k * NO + o], f);
            const unsigned m = tangent_mask(cells[3 * cell], cells[3 * cell + 1], cells[3 * cell + 2], nx, ny, nz);
            out[(long long)cell * NO + o] = (m >> o) & 1u ? __fmul_rn(rr[q], f) : 0.f;
        }
    }
    cp_async_wait_all();  // nothing left in flight at exit
}

__global__ void __launch_bounds__(256) scatter_kernel(float *__restrict__ f, long long fstride, int pitch, int ny,
                                                      const int *__restrict__ cells, int ncells,
                                                      const float *__restrict__ vals)
{
    const int q = blockIdx.x * 256 + threadIdx.x;
    if (q >= ncells) return;
    const long long p = cells[3 * q] + (long long)pitch * (cells[3 * q + 1] + (long long)ny * cells[3 * q + 2]);
    for (int c = 0; c < NO; ++c) f[c * fstride + p] = __fadd_rn(f[c * fstride + p], vals[(long long)q * NO + c]);
}

__global__ void __launch_bounds__(256) copy_cells_kernel(float *__restrict__ dst, const float *__restrict__ src,
                                                         long long fstride, int pitch, int ny,
                                                         const int *__restrict__ cells, int ncells)
{
    const int q = blockIdx.x * 256 + threadIdx.x;
    if (q >= ncells) return;
    const long long p = cells[3 * q] + (long long)pitch * (cells[3 * q + 1] + (long long)ny * cells[3 * q + 2]);
    for (int c = 0; c < NO; ++c) dst[c * fstride + p] = src[c * fstride + p];
}

// The x slab of a band snapshot (layout above): element e of the slab is
// (comp, side, xd, z, y) in that order, y fastest; planes outside the grid
// (nx < 2) are zero and never read.
__global__ void __launch_bounds__(256) fill_xslab_kernel(float *__restrict__ snap, const float *__restrict__ f,
                                                         long long fstride, int pitch, int nx, int ny, int nz)
{
    const long long n = xslab_floats(ny, nz);
    float *slab = snap + 6 * fstride;
    for (long long e = blockIdx.x * 256LL + threadIdx.x; e < n; e += (long long)gridDim.x * 256) {
        const int y = (int)(e % ny);
        long long r = e / ny;
        const int z = (int)(r % nz);
        r /= nz;
        const int xd = (int)(r & 1), side = (int)((r >> 1) & 1), comp = (int)(r >> 2);
        const int x = side ? nx - 2 + xd : xd;
        slab[e] = (x >= 0 && x < nx) ? f[comp * fstride + x + (long long)pitch * (y + (long long)ny * z)] : 0.f;
    }
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

size_t learned_layer_smem() { return LAYER_SMEM; }

cudaError_t learned_layer_configure()
{
    return cudaFuncSetAttribute(layer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LAYER_SMEM);
}

cudaError_t learned_layer_predict(const float *params, const float *cur, const float *prev, long long fstride,
                                  int pitch, int nx, int ny, int nz, const int *cells, int ncells, float *out,
                                  int grid, cudaStream_t st)
{
    if (ncells <= 0) return cudaSuccess;
    const int tiles = (ncells + LC - 1) / LC;
    layer_kernel<<<std::min(grid, tiles), 256, LAYER_SMEM, st>>>(params, cur, prev, fstride, pitch, nx, ny, nz, cells,
                                                                 ncells, out);
    return cudaGetLastError();
}

cudaError_t learned_layer_scatter(float *f, long long fstride, int pitch, int ny, const int *cells, int ncells,
                                  const float *vals, cudaStream_t st)
{
    if (ncells <= 0) return cudaSuccess;
    scatter_kernel<<<(ncells + 255) / 256, 256, 0, st>>>(f, fstride, pitch, ny, cells, ncells, vals);
    return cudaGetLastError();
}

cudaError_t learned_copy_cells(float *dst, const float *src, long long fstride, int pitch, int ny, const int *cells,
                               int ncells, cudaStream_t st)
{
    if (ncells <= 0) return cudaSuccess;
    copy_cells_kernel<<<(ncells + 255) / 256, 256, 0, st>>>(dst, src, fstride, pitch, ny, cells, ncells);
    return cudaGetLastError();
}

size_t learned_xslab_bytes(int ny, int nz) { return sizeof(float) * (size_t)xslab_floats(ny, nz); }

cudaError_t learned_fill_xslab(float *snap, const float *f, long long fstride, int pitch, int nx, int ny, int nz,
                               cudaStream_t st)
{
    const long long n = xslab_floats(ny, nz);
    const int blocks = (int)std::min<long long>((n + 255) / 256, 4096);
    fill_xslab_kernel<<<blocks, 256, 0, st>>>(snap, f, fstride, pitch, nx, ny, nz);
    return cudaGetLastError();
}
