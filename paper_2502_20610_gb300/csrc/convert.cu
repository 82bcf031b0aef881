// Fields between the caller's dense FP32 arrays (nx*ny*nz values a component)
// and the simulation's arrays (rows of `pitch` elements in the storage format;
// 16-bit: q = fl_S(v / s), to nearest even, on the way in, v = s * q, exact, on
// the way out), used by fdtd_write_fields / fdtd_read_fields.
//
// All components in one launch.  Bounded by memory on large grids (one read
// and one write of each value), by the launch on small ones, where a copy per
// component cost 2.5 us of host time each.  A block's x threads run along a
// row, four values each where rows and pointers allow, its y threads take
// rows: no division per value (an element-wise kernel with a 64-bit division
// and a launch per component took 142 us to write and read 128^3 FP16, this 31).
#include "internal.h"
#include "storage.cuh"

namespace {

// enc or dec of four values at once: 16-byte FP32, 8-byte 16-bit accesses
template <class S>
__device__ __forceinline__ void put4(typename S::T *p, const float4 v, float is)
{
    if constexpr (sizeof(typename S::T) == 4) {
        *reinterpret_cast<float4 *>(p) = v;
    } else {
        *reinterpret_cast<uint2 *>(p) = make_uint2(S::enc2(v.x, v.y, is), S::enc2(v.z, v.w, is));
    }
}
template <class S>
__device__ __forceinline__ float4 get4(const typename S::T *p, float s)
{
    using T = typename S::T;
    if constexpr (sizeof(T) == 4) {
        return *reinterpret_cast<const float4 *>(p);
    } else {
        const uint2 u = *reinterpret_cast<const uint2 *>(p);
        return make_float4(S::dec((T)(u.x & 0xffffu), s), S::dec((T)(u.x >> 16), s), S::dec((T)(u.y & 0xffffu), s),
                           S::dec((T)(u.y >> 16), s));
    }
}

// comps: the component of each z block, 4 bits each.  IN: dense -> arrays
// (and the nzero words at `zero` cleared); else arrays -> dense, nothing if
// *err is set.
template <class S, bool IN, bool VEC>
__global__ void __launch_bounds__(256)
fields_kernel(typename S::T *arrays, long long fs, float *dense, long long n, int nx, long long rows, int pitch,
              unsigned comps, const Scales sc, int *zero, int nzero, const int *err)
{
    if (!IN && *err != DEV_OK) return;
    if (IN && blockIdx.x == 0 && blockIdx.z == 0 && threadIdx.y == 0)
        for (int q = threadIdx.x; q < nzero; q += blockDim.x) zero[q] = 0;
    const int c = (comps >> (4 * blockIdx.z)) & 15;
    typename S::T *const f = arrays + c * fs;
    float *const d = dense + blockIdx.z * n;
    for (long long r = blockIdx.x * (long long)blockDim.y + threadIdx.y; r < rows; r += (long long)gridDim.x * blockDim.y) {
        typename S::T *const fr = f + r * pitch;
        float *const dr = d + r * nx;
        if (VEC) {
            for (int x = 4 * threadIdx.x; x < nx; x += 4 * blockDim.x) {
                if (IN) put4<S>(fr + x, *reinterpret_cast<const float4 *>(dr + x), sc.is[c]);
                else *reinterpret_cast<float4 *>(dr + x) = get4<S>(fr + x, sc.s[c]);
            }
        } else {
            for (int x = threadIdx.x; x < nx; x += blockDim.x) {
                if (IN) fr[x] = S::enc(dr[x], sc.is[c]);
                else dr[x] = S::dec(fr[x], sc.s[c]);
            }
        }
    }
}

// The same for rows that leave most of such a grid idle.  PARTS: few rows, whose
// parts go over y blocks.  Else: many rows that are not in groups of four values,
// four of them, next to one another, in flight a thread.  (Forms of their own: in
// the one above, four rows a grid apart made 128^3 slower to write, 25 -> 30 us in
// FP32, and a stride over y blocks 23 -> 26 in FP16.)
template <class S, bool IN, bool VEC, bool PARTS>
__global__ void __launch_bounds__(256)
odd_rows_kernel(typename S::T *arrays, long long fs, float *dense, long long n, int nx, long long rows, int pitch,
                unsigned comps, const Scales sc, int *zero, int nzero, const int *err)
{
    static_assert(PARTS || !VEC, "groups of four values need no more rows in flight");
    if (!IN && *err != DEV_OK) return;
    if (IN && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.y == 0)
        for (int q = threadIdx.x; q < nzero; q += blockDim.x) zero[q] = 0;
    const int c = (comps >> (4 * blockIdx.z)) & 15;
    typename S::T *const f = arrays + c * fs;
    float *const d = dense + blockIdx.z * n;
    constexpr int Q = PARTS ? 1 : 4;
    const int x0 = blockIdx.y * blockDim.x + threadIdx.x, dx = gridDim.y * blockDim.x;
    for (long long r = Q * (blockIdx.x * (long long)blockDim.y + threadIdx.y); r < rows;
         r += Q * (long long)gridDim.x * blockDim.y) {
        typename S::T *const fr = f + r * pitch;
        float *const dr = d + r * nx;
        if constexpr (VEC) {
            for (int x = 4 * x0; x < nx; x += 4 * dx) {
                if (IN) put4<S>(fr + x, *reinterpret_cast<const float4 *>(dr + x), sc.is[c]);
                else *reinterpret_cast<float4 *>(dr + x) = get4<S>(fr + x, sc.s[c]);
            }
        } else {
            const int live = (int)min((long long)Q, rows - r);
            for (int x = x0; x < nx; x += dx) {
                float v[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if (q < live) v[q] = IN ? dr[q * nx + x] : S::dec(fr[q * pitch + x], sc.s[c]);
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if (q < live) {
                        if (IN) fr[q * pitch + x] = S::enc(v[q], sc.is[c]);
                        else dr[q * nx + x] = v[q];
                    }
            }
        }
    }
}

template <class S, bool IN>
cudaError_t go(void *arrays, long long fs, float *dense, int nx, int ny, int nz, int pitch, unsigned comps, int ncomp,
               const Scales &sc, int *zero, int nzero, const int *err, cudaStream_t st)
{
    const long long rows = (long long)ny * nz;
    // four values a thread: rows of both sides start on 16 (8) bytes
    const bool vec = nx % 4 == 0 && (uintptr_t)dense % 16 == 0;
    const int per_row = vec ? nx / 4 : nx;
    // (a row of three values by eight threads: 3 x 700 x 700 in FP16 read in 92 us, a
    // launch and a division a value had taken 72; 62 with four)
    int bx = 1;
    while (bx < 256 && bx < per_row) bx *= 2;
    const dim3 block((unsigned)bx, 256u / bx);
    // where rows are few, a row's parts go over blocks too (nine rows of 20000 values in
    // FP16 from pinned memory: 170 us by nine blocks a component, 107 so); where they are
    // many and not in groups of four values, four rows a thread (a component of 30 x 600
    // x 600 in FP16 read in 60 us with one row in flight, 46 so)
    constexpr long long BLOCKS = 152 * 8;
    const long long blocks = (rows + block.y - 1) / block.y;
    const unsigned gx = (unsigned)std::min(blocks, BLOCKS);
    const unsigned parts = std::min((unsigned)((per_row + bx - 1) / bx), (unsigned)(BLOCKS / gx));
    const dim3 grid(gx, parts, (unsigned)ncomp);
    auto launch = [&](auto kernel) {
        kernel<<<grid, block, 0, st>>>((typename S::T *)arrays, fs, dense, (long long)nx * rows, nx, rows, pitch, comps, sc, zero,
                                       nzero, err);
    };
    if (parts > 1) launch(vec ? odd_rows_kernel<S, IN, true, true> : odd_rows_kernel<S, IN, false, true>);
    else if (!vec && blocks >= 4 * BLOCKS) launch(odd_rows_kernel<S, IN, false, false>);
    else launch(vec ? fields_kernel<S, IN, true> : fields_kernel<S, IN, false>);
    return cudaGetLastError();
}

template <bool IN>
cudaError_t dispatch(int storage, void *arrays, long long fs, float *dense, int nx, int ny, int nz, int pitch,
                     unsigned comps, int ncomp, const Scales &sc, int *zero, int nzero, const int *err, cudaStream_t st)
{
    // the host converts with s at the boundary in the uniform formats too
    if (storage == FDTD_STORAGE_F16)
        return go<StoreF16, IN>(arrays, fs, dense, nx, ny, nz, pitch, comps, ncomp, sc, zero, nzero, err, st);
    if (storage == FDTD_STORAGE_BF16)
        return go<StoreBF16, IN>(arrays, fs, dense, nx, ny, nz, pitch, comps, ncomp, sc, zero, nzero, err, st);
    return go<StoreF32, IN>(arrays, fs, dense, nx, ny, nz, pitch, comps, ncomp, sc, zero, nzero, err, st);
}

} // namespace

cudaError_t launch_write_fields(void *arrays, long long fs, const float *dense, int storage, int nx, int ny, int nz,
                                int pitch, unsigned comps, int ncomp, const Scales &sc, int *zero, int nzero,
                                cudaStream_t st)
{
    return dispatch<true>(storage, arrays, fs, const_cast<float *>(dense), nx, ny, nz, pitch, comps, ncomp, sc, zero, nzero,
                          nullptr, st);
}

cudaError_t launch_read_fields(float *dense, const void *arrays, long long fs, int storage, int nx, int ny, int nz,
                               int pitch, unsigned comps, int ncomp, const Scales &sc, const int *err, cudaStream_t st)
{
    return dispatch<false>(storage, const_cast<void *>(arrays), fs, dense, nx, ny, nz, pitch, comps, ncomp, sc, nullptr, 0,
                           err, st);
}
