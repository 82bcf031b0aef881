// Naive schedule: one streaming kernel per half-step over the whole grid
// (the "very straightforward" implementation of Sec. 2 whose cost model is
// 6 memory operations and 6 flops per component).  Every launch boundary is
// a grid-wide synchronisation.  It is the in-library baseline, and the
// systolic kernel must reproduce its results bit for bit.
//
// Layout: 256-thread CTAs of 32 (x) x 8 (y) threads; each thread marches up
// a column of NAIVE_KZ cells in z and carries the z-neighbour in registers,
// so x rows are read coalesced and the z-neighbour plane is read once.
// Fields are stored as FP32, FP16 or BF16 (storage.cuh); arithmetic is FP32.
#include "internal.h"
#include "storage.cuh"
#include "sys_common.cuh"
#include "yee_cell.cuh"

namespace {

constexpr int NAIVE_BX = 32, NAIVE_BY = 8, NAIVE_KZ = 8;
constexpr int NAIVE_BLOCK_CELLS = 1024;

template <class S>
__global__ void __launch_bounds__(NAIVE_BX *NAIVE_BY)
naive_h_kernel(typename S::T *__restrict__ ex_, typename S::T *__restrict__ ey_, typename S::T *__restrict__ ez_,
               typename S::T *__restrict__ hx_, typename S::T *__restrict__ hy_, typename S::T *__restrict__ hz_,
               int nx, int ny, int nz, int pitch, float ndt, const Scales sc)
{
    using T = typename S::T;
    const int i = blockIdx.x * NAIVE_BX + threadIdx.x;
    const int j = blockIdx.y * NAIVE_BY + threadIdx.y;
    const int k0 = blockIdx.z * NAIVE_KZ;
    if (i >= nx || j >= ny || k0 >= nz) return;
    const int k1 = min(k0 + NAIVE_KZ, nz);
    const long long sxy = (long long)pitch * ny;
    const bool ip = i + 1 < nx, jp = j + 1 < ny;
    const T *Ex = ex_, *Ey = ey_, *Ez = ez_;
    const float s0 = sc.s[0], s1 = sc.s[1], s2 = sc.s[2];
    long long p = i + (long long)pitch * (j + (long long)ny * k0);
    float exc = S::dec(__ldg(Ex + p), s0), eyc = S::dec(__ldg(Ey + p), s1);
    for (int k = k0; k < k1; ++k, p += sxy) {
        const bool kp = k + 1 < nz;
        const float exn = kp ? S::dec(__ldg(Ex + p + sxy), s0) : 0.f;
        const float eyn = kp ? S::dec(__ldg(Ey + p + sxy), s1) : 0.f;
        const float ez = S::dec(__ldg(Ez + p), s2);
        const float ez_ip = ip ? S::dec(__ldg(Ez + p + 1), s2) : 0.f;
        const float ey_ip = ip ? S::dec(__ldg(Ey + p + 1), s1) : 0.f;
        const float ez_jp = jp ? S::dec(__ldg(Ez + p + pitch), s2) : 0.f;
        const float ex_jp = jp ? S::dec(__ldg(Ex + p + pitch), s0) : 0.f;
        hx_[p] = S::enc(h_x(S::dec(hx_[p], sc.s[3]), ez_jp, ez, eyn, eyc, ndt), sc.is[3]);
        hy_[p] = S::enc(h_y(S::dec(hy_[p], sc.s[4]), exn, exc, ez_ip, ez, ndt), sc.is[4]);
        hz_[p] = S::enc(h_z(S::dec(hz_[p], sc.s[5]), ey_ip, eyc, ex_jp, exc, ndt), sc.is[5]);
        exc = exn;
        eyc = eyn;
    }
}

// BACK: from the last planes to the first (e_backwards).  A form of its own: the
// choice made here took 0.7 us of a kernel of one plane (1000 x 1000 x 1, 14.4 ->
// 15.8 us a step).
template <class S, bool LOSSY, bool BACK>
__global__ void __launch_bounds__(NAIVE_BX *NAIVE_BY)
naive_e_kernel(typename S::T *__restrict__ ex_, typename S::T *__restrict__ ey_, typename S::T *__restrict__ ez_,
               typename S::T *__restrict__ hx_, typename S::T *__restrict__ hy_, typename S::T *__restrict__ hz_,
               const float *__restrict__ ce_, const float *__restrict__ ca_, int nx, int ny, int nz, int pitch,
               long long step, const SrcSet src, const Scales sc)
{
    using T = typename S::T;
    const int i = blockIdx.x * NAIVE_BX + threadIdx.x;
    const int j = blockIdx.y * NAIVE_BY + threadIdx.y;
    const int k0 = (int)(BACK ? gridDim.z - 1 - blockIdx.z : blockIdx.z) * NAIVE_KZ;
    if (i >= nx || j >= ny || k0 >= nz) return;
    const int k1 = min(k0 + NAIVE_KZ, nz);
    const long long sxy = (long long)pitch * ny;
    const T *Hx = hx_, *Hy = hy_, *Hz = hz_;
    const float s3 = sc.s[3], s4 = sc.s[4], s5 = sc.s[5];
    long long p = i + (long long)pitch * (j + (long long)ny * k0);
    float hxm = k0 > 0 ? S::dec(__ldg(Hx + p - sxy), s3) : 0.f;
    float hym = k0 > 0 ? S::dec(__ldg(Hy + p - sxy), s4) : 0.f;
    for (int k = k0; k < k1; ++k, p += sxy) {
        const float hx = S::dec(__ldg(Hx + p), s3), hy = S::dec(__ldg(Hy + p), s4);
        const float hz = S::dec(__ldg(Hz + p), s5);
        const float ce = __ldg(ce_ + p);
        const float ca = LOSSY ? __ldg(ca_ + p) : 1.f;
        float ex = S::dec(ex_[p], sc.s[0]), ey = S::dec(ey_[p], sc.s[1]), ez = S::dec(ez_[p], sc.s[2]);
        // PEC: tangential E on the low planes is never updated.  Lossy cells:
        // E <- ca E + cb curl H, with cb in place of dt/eps
        if (j > 0 && k > 0) ex = e_x(decay<LOSSY>(ca, ex), hz, S::dec(__ldg(Hz + p - pitch), s5), hy, hym, ce);
        if (i > 0 && k > 0) ey = e_y(decay<LOSSY>(ca, ey), hx, hxm, hz, S::dec(__ldg(Hz + p - 1), s5), ce);
        if (i > 0 && j > 0)
            ez = e_z(decay<LOSSY>(ca, ez), hy, S::dec(__ldg(Hy + p - 1), s4), hx, S::dec(__ldg(Hx + p - pitch), s3), ce);
        for (int q = 0; q < src.n; ++q) {
            const SrcDesc &s = src.s[q];
            if (s.idx == p && step < s.n_amp) {
                const float a = S::src_amp(s.amp[step], sc.src);
                if (s.comp == 0) ex = add_source(ex, a);
                else if (s.comp == 1) ey = add_source(ey, a);
                else ez = add_source(ez, a);
            }
        }
        ex_[p] = S::enc(ex, sc.is[0]);
        ey_[p] = S::enc(ey, sc.is[1]);
        ez_[p] = S::enc(ez, sc.is[2]);
        hxm = hx;
        hym = hy;
    }
}

// Small domains (at most NAIVE_BLOCK_CELLS cells, the largest thread block):
// one CTA, one thread per cell, runs all the steps of a call with block
// barriers between the half-steps instead of kernel boundaries, the regime
// of Fig. 1 in which the update needs no global synchronisation.  A thread's
// own six values stay in registers for the whole call, neighbours go through
// shared memory, so a half-step is a shared-memory round trip and a barrier:
// 8^3, 100 steps 40.0 -> 25.9 us (fields in global memory before).
template <class S, bool LOSSY>
__global__ void __launch_bounds__(NAIVE_BLOCK_CELLS)
naive_block_kernel(typename S::T *__restrict__ ex_, typename S::T *__restrict__ ey_, typename S::T *__restrict__ ez_,
                   typename S::T *__restrict__ hx_, typename S::T *__restrict__ hy_, typename S::T *__restrict__ hz_,
                   const float *__restrict__ ce_, const float *__restrict__ ca_, int nx, int ny, int nz, int pitch, float ndt, long long step0,
                   int nsteps, const SrcSet src, const Scales sc)
{
    __shared__ float sex[NAIVE_BLOCK_CELLS], sey[NAIVE_BLOCK_CELLS], sez[NAIVE_BLOCK_CELLS];
    __shared__ float shx[NAIVE_BLOCK_CELLS], shy[NAIVE_BLOCK_CELLS], shz[NAIVE_BLOCK_CELLS];
    const int q = threadIdx.x, qy = nx, qz = nx * ny;
    const bool own = q < nx * ny * nz;
    const int i = own ? q % nx : 0, j = own ? (q / nx) % ny : 0, k = own ? q / qz : 0;
    const long long p = i + (long long)pitch * (j + (long long)ny * k);
    const bool ip = own && i + 1 < nx, jp = own && j + 1 < ny, kp = own && k + 1 < nz;
    const float ce = own ? ce_[p] : 0.f;
    const float ca = LOSSY && own ? ca_[p] : 1.f;
    float ex = 0.f, ey = 0.f, ez = 0.f, hx = 0.f, hy = 0.f, hz = 0.f;
    if (own) {
        ex = S::dec(ex_[p], sc.s[0]); ey = S::dec(ey_[p], sc.s[1]); ez = S::dec(ez_[p], sc.s[2]);
        hx = S::dec(hx_[p], sc.s[3]); hy = S::dec(hy_[p], sc.s[4]); hz = S::dec(hz_[p], sc.s[5]);
    }
    unsigned mine = 0;  // the sources on this cell
    for (int qq = 0; qq < src.n; ++qq)
        if (own && src.s[qq].idx == p) mine |= 1u << qq;
    sex[q] = ex; sey[q] = ey; sez[q] = ez;
    __syncthreads();
    for (int s = 0; s < nsteps; ++s) {
        if (own) {
            const float ez_jp = jp ? sez[q + qy] : 0.f, ey_kp = kp ? sey[q + qz] : 0.f;
            const float ex_kp = kp ? sex[q + qz] : 0.f, ez_ip = ip ? sez[q + 1] : 0.f;
            const float ey_ip = ip ? sey[q + 1] : 0.f, ex_jp = jp ? sex[q + qy] : 0.f;
            hx = S::rnd(h_x(hx, ez_jp, ez, ey_kp, ey, ndt), sc.s[3], sc.is[3]);
            hy = S::rnd(h_y(hy, ex_kp, ex, ez_ip, ez, ndt), sc.s[4], sc.is[4]);
            hz = S::rnd(h_z(hz, ey_ip, ey, ex_jp, ex, ndt), sc.s[5], sc.is[5]);
            shx[q] = hx; shy[q] = hy; shz[q] = hz;
        }
        __syncthreads();
        if (own) {
            if (j > 0 && k > 0) ex = e_x(decay<LOSSY>(ca, ex), hz, shz[q - qy], hy, shy[q - qz], ce);
            if (i > 0 && k > 0) ey = e_y(decay<LOSSY>(ca, ey), hx, shx[q - qz], hz, shz[q - 1], ce);
            if (i > 0 && j > 0) ez = e_z(decay<LOSSY>(ca, ez), hy, shy[q - 1], hx, shx[q - qy], ce);
            const long long step = step0 + s;
            for (unsigned m = mine; m; m &= m - 1) {
                const SrcDesc &d = src.s[__ffs((int)m) - 1];
                if (step < d.n_amp) {
                    const float a = S::src_amp(d.amp[step], sc.src);
                    if (d.comp == 0) ex = add_source(ex, a);
                    else if (d.comp == 1) ey = add_source(ey, a);
                    else ez = add_source(ez, a);
                }
            }
            ex = S::rnd(ex, sc.s[0], sc.is[0]);
            ey = S::rnd(ey, sc.s[1], sc.is[1]);
            ez = S::rnd(ez, sc.s[2], sc.is[2]);
            sex[q] = ex; sey[q] = ey; sez[q] = ez;
        }
        __syncthreads();
    }
    if (own) {
        ex_[p] = S::enc(ex, sc.is[0]); ey_[p] = S::enc(ey, sc.is[1]); ez_[p] = S::enc(ez, sc.is[2]);
        hx_[p] = S::enc(hx, sc.is[3]); hy_[p] = S::enc(hy, sc.is[4]); hz_[p] = S::enc(hz, sc.is[5]);
    }
}

// Mid-size domains: all the steps of a call in one cooperative launch, one
// CTA per SM, with a grid barrier after each half-step in place of a kernel
// boundary.  Bounded by the barriers (about 2 us each) on small grids and by
// L2 bandwidth on larger ones; a pair of launches a step costs 14 us however
// small the grid.  A warp takes 32 consecutive x of kz rows in z (z neighbours
// in registers), the warps of a CTA consecutive y, so neighbour rows are
// L1 hits.  Loads are plain (coherent): the barrier's acquire orders them
// after the other CTAs' stores.
constexpr int COOP_NT = 1024;

// Grid barrier: count of arrivals in bar[0], generation in bar[4]; the last
// arrival resets the count and bumps the generation, so a launch needs no
// state from the host.  Bounded wait; false (in every thread) past it, with the
// block and -5 behind the error word.
__device__ bool grid_barrier(int *bar, unsigned &gen, int *err, long long timeout_ns)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int good = 1;
        unsigned *const g = reinterpret_cast<unsigned *>(bar + 4);
        __threadfence();
        if (atomicAdd(bar, 1) == (int)gridDim.x - 1) {
            *reinterpret_cast<volatile int *>(bar) = 0;
            sysc::st_release(g, gen + 1u);
        } else {
            const unsigned long long t0 = sysc::globaltimer();
            while (sysc::ld_acquire(g) == gen) {
                if (sysc::ld_volatile(err) != DEV_OK) {
                    good = 0;
                    break;
                }
                if (sysc::globaltimer() - t0 > (unsigned long long)timeout_ns) {
                    if (atomicCAS(err, DEV_OK, DEV_ERR_TIMEOUT) == DEV_OK) {
                        err[1] = (int)blockIdx.x;
                        err[2] = -5;
                    }
                    good = 0;
                    break;
                }
            }
        }
        ok = good;
    }
    ++gen;
    __syncthreads();
    return ok != 0;
}

template <class S, bool LOSSY>
__global__ void __launch_bounds__(COOP_NT, 1)
naive_coop_kernel(typename S::T *f, long long fs, const float *__restrict__ ce_, const float *__restrict__ ca_, int nx,
                  int ny, int nz, int pitch, int kz, float ndt, long long step0, int nsteps, const SrcSet src,
                  const Scales sc, bool back, int *bar, int *err, long long timeout_ns)
{
    using T = typename S::T;
    T *const ex_ = f, *const ey_ = f + fs, *const ez_ = f + 2 * fs, *const hx_ = f + 3 * fs, *const hy_ = f + 4 * fs,
             *const hz_ = f + 5 * fs;
    unsigned gen = 0;
    if (threadIdx.x == 0) gen = sysc::ld_acquire(reinterpret_cast<unsigned *>(bar + 4));
    const int lane = threadIdx.x & 31;
    const int nxc = (nx + 31) / 32, nzc = (nz + kz - 1) / kz;
    const long long items = (long long)nxc * ny * nzc, stride = (long long)gridDim.x * (COOP_NT / 32);
    const long long first = (long long)blockIdx.x * (COOP_NT / 32) + (threadIdx.x >> 5);
    const long long last = first + (items - 1 - first) / stride * stride;  // of this warp (if it has any)
    const long long sxy = (long long)pitch * ny;
    auto place = [&](long long it, int &i, int &j, int &k0) {
        j = (int)(it % ny);
        const int r = (int)(it / ny);
        i = (r % nxc) * 32 + lane;
        k0 = (r / nxc) * kz;
    };
    for (int s = 0; s < nsteps; ++s) {
        for (long long it = first; it < items; it += stride) {
            int i, j, k0;
            place(it, i, j, k0);
            if (i >= nx) continue;
            const int k1 = min(k0 + kz, nz);
            const bool ip = i + 1 < nx, jp = j + 1 < ny;
            long long p = i + (long long)pitch * (j + (long long)ny * k0);
            float exc = S::dec(ex_[p], sc.s[0]), eyc = S::dec(ey_[p], sc.s[1]);
#pragma unroll 2
            for (int k = k0; k < k1; ++k, p += sxy) {
                const bool kp = k + 1 < nz;
                const float exn = kp ? S::dec(ex_[p + sxy], sc.s[0]) : 0.f;
                const float eyn = kp ? S::dec(ey_[p + sxy], sc.s[1]) : 0.f;
                const float ez = S::dec(ez_[p], sc.s[2]);
                const float ez_ip = ip ? S::dec(ez_[p + 1], sc.s[2]) : 0.f;
                const float ey_ip = ip ? S::dec(ey_[p + 1], sc.s[1]) : 0.f;
                const float ez_jp = jp ? S::dec(ez_[p + pitch], sc.s[2]) : 0.f;
                const float ex_jp = jp ? S::dec(ex_[p + pitch], sc.s[0]) : 0.f;
                const float hx = S::dec(hx_[p], sc.s[3]), hy = S::dec(hy_[p], sc.s[4]), hz = S::dec(hz_[p], sc.s[5]);
                hx_[p] = S::enc(h_x(hx, ez_jp, ez, eyn, eyc, ndt), sc.is[3]);
                hy_[p] = S::enc(h_y(hy, exn, exc, ez_ip, ez, ndt), sc.is[4]);
                hz_[p] = S::enc(h_z(hz, ey_ip, eyc, ex_jp, exc, ndt), sc.is[5]);
                exc = exn;
                eyc = eyn;
            }
        }
        if (!grid_barrier(bar, gen, err, timeout_ns)) return;
        const long long step = step0 + s;
        for (long long q = first; q < items; q += stride) {
            const long long it = back ? last - (q - first) : q;
            int i, j, k0;
            place(it, i, j, k0);
            if (i >= nx) continue;
            const int k1 = min(k0 + kz, nz);
            long long p = i + (long long)pitch * (j + (long long)ny * k0);
            float hxm = k0 > 0 ? S::dec(hx_[p - sxy], sc.s[3]) : 0.f;
            float hym = k0 > 0 ? S::dec(hy_[p - sxy], sc.s[4]) : 0.f;
#pragma unroll 2
            for (int k = k0; k < k1; ++k, p += sxy) {
                const float hx = S::dec(hx_[p], sc.s[3]), hy = S::dec(hy_[p], sc.s[4]), hz = S::dec(hz_[p], sc.s[5]);
                const float hz_jm = j > 0 ? S::dec(hz_[p - pitch], sc.s[5]) : 0.f;
                const float hx_jm = j > 0 ? S::dec(hx_[p - pitch], sc.s[3]) : 0.f;
                const float hz_im = i > 0 ? S::dec(hz_[p - 1], sc.s[5]) : 0.f;
                const float hy_im = i > 0 ? S::dec(hy_[p - 1], sc.s[4]) : 0.f;
                const float ce = __ldg(ce_ + p);
                const float ca = LOSSY ? __ldg(ca_ + p) : 1.f;
                float ex = S::dec(ex_[p], sc.s[0]), ey = S::dec(ey_[p], sc.s[1]), ez = S::dec(ez_[p], sc.s[2]);
                if (j > 0 && k > 0) ex = e_x(decay<LOSSY>(ca, ex), hz, hz_jm, hy, hym, ce);
                if (i > 0 && k > 0) ey = e_y(decay<LOSSY>(ca, ey), hx, hxm, hz, hz_im, ce);
                if (i > 0 && j > 0) ez = e_z(decay<LOSSY>(ca, ez), hy, hy_im, hx, hx_jm, ce);
                for (int q = 0; q < src.n; ++q) {
                    const SrcDesc &d = src.s[q];
                    if (d.idx == p && step < d.n_amp) {
                        const float a = S::src_amp(d.amp[step], sc.src);
                        if (d.comp == 0) ex = add_source(ex, a);
                        else if (d.comp == 1) ey = add_source(ey, a);
                        else ez = add_source(ez, a);
                    }
                }
                ex_[p] = S::enc(ex, sc.is[0]);
                ey_[p] = S::enc(ey, sc.is[1]);
                ez_[p] = S::enc(ez, sc.is[2]);
                hxm = hx;
                hym = hy;
            }
        }
        if (s + 1 < nsteps && !grid_barrier(bar, gen, err, timeout_ns)) return;
    }
}

dim3 naive_grid(int nx, int ny, int nz)
{
    return dim3((nx + NAIVE_BX - 1) / NAIVE_BX, (ny + NAIVE_BY - 1) / NAIVE_BY,
                (nz + NAIVE_KZ - 1) / NAIVE_KZ);
}

// Does the E half-step sweep the grid backwards, from what the H half-step
// touched last?  It finds that part in L2 when the state does not fit there:
// measured, FP32 (the pair of kernels) 160^3 64 -> 57 us a step, 256^3
// 232 -> 222, 384^3 742 -> 738; FP16 256^3 197 -> 182.  A state of less than
// 96 MB (six components and dt/eps) is in L2 either way, and the forward
// sweep is then as fast or faster (FP16 160^3 33 us against 37).
bool e_backwards(size_t eb, int nx, int ny, int nz)
{
    return (double)nx * ny * nz * (6.0 * eb + 4.0) > 96e6;
}

template <class S>
cudaError_t launch_h(void *const f[6], int nx, int ny, int nz, int pitch, float neg_dt, const Scales &sc,
                     cudaStream_t st)
{
    using T = typename S::T;
    naive_h_kernel<S><<<naive_grid(nx, ny, nz), dim3(NAIVE_BX, NAIVE_BY), 0, st>>>(
        (T *)f[0], (T *)f[1], (T *)f[2], (T *)f[3], (T *)f[4], (T *)f[5], nx, ny, nz, pitch, neg_dt, sc);
    return cudaGetLastError();
}

template <class S, bool LOSSY, bool BACK>
cudaError_t launch_e_form(void *const f[6], const float *ce, const float *ca, int nx, int ny, int nz, int pitch,
                          long long step, const SrcSet &src, const Scales &sc, cudaStream_t st)
{
    using T = typename S::T;
    naive_e_kernel<S, LOSSY, BACK><<<naive_grid(nx, ny, nz), dim3(NAIVE_BX, NAIVE_BY), 0, st>>>(
        (T *)f[0], (T *)f[1], (T *)f[2], (T *)f[3], (T *)f[4], (T *)f[5], ce, ca, nx, ny, nz, pitch, step, src, sc);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_e(void *const f[6], const float *ce, const float *ca, int nx, int ny, int nz, int pitch,
                     long long step, const SrcSet &src, const Scales &sc, cudaStream_t st)
{
    const bool back = e_backwards(sizeof(typename S::T), nx, ny, nz);
    if (ca)
        return back ? launch_e_form<S, true, true>(f, ce, ca, nx, ny, nz, pitch, step, src, sc, st)
                    : launch_e_form<S, true, false>(f, ce, ca, nx, ny, nz, pitch, step, src, sc, st);
    return back ? launch_e_form<S, false, true>(f, ce, ca, nx, ny, nz, pitch, step, src, sc, st)
                : launch_e_form<S, false, false>(f, ce, ca, nx, ny, nz, pitch, step, src, sc, st);
}

template <class S>
cudaError_t launch_block(void *const f[6], const float *ce, const float *ca, int nx, int ny, int nz, int pitch,
                         float neg_dt, long long step0, int nsteps, const SrcSet &src, const Scales &sc,
                         cudaStream_t st)
{
    using T = typename S::T;
    const int threads = (nx * ny * nz + 31) / 32 * 32;
    if (ca)
        naive_block_kernel<S, true><<<1, threads, 0, st>>>((T *)f[0], (T *)f[1], (T *)f[2], (T *)f[3], (T *)f[4],
                                                            (T *)f[5], ce, ca, nx, ny, nz, pitch, neg_dt, step0,
                                                            nsteps, src, sc);
    else
        naive_block_kernel<S, false><<<1, threads, 0, st>>>((T *)f[0], (T *)f[1], (T *)f[2], (T *)f[3], (T *)f[4],
                                                             (T *)f[5], ce, ca, nx, ny, nz, pitch, neg_dt, step0,
                                                             nsteps, src, sc);
    return cudaGetLastError();
}

// Rows in z per warp of the cooperative launch: the fewest row steps on the
// busiest warp, a column's start (its two z-neighbour loads) counted as half a
// row; a remainder round of full-height columns would double a half-step.
int rows_per_warp(int nx, int ny, int nz, int sms)
{
    const long long rows = (long long)((nx + 31) / 32) * ny, warps = (long long)sms * (COOP_NT / 32);
    int kz = 1;
    double least = 0.0;
    for (int k = 1; k <= std::min(nz, 24); ++k) {
        const double cost = (double)((rows * ((nz + k - 1) / k) + warps - 1) / warps) * (k + 0.5);
        if (k == 1 || cost < least) {
            least = cost;
            kz = k;
        }
    }
    return kz;
}

template <class S, bool LOSSY>
cudaError_t launch_coop(void *f, long long fs, const float *ce, const float *ca, int nx, int ny, int nz, int pitch,
                        float neg_dt, long long step0, int nsteps, const SrcSet &src, const Scales &sc, int *bar, int *err,
                        long long timeout_ns, int sms, cudaStream_t st)
{
    using T = typename S::T;
    const int kz = rows_per_warp(nx, ny, nz, sms);
    const long long rows = (long long)((nx + 31) / 32) * ny;
    const long long items = rows * ((nz + kz - 1) / kz);
    const int grid = (int)std::min<long long>(sms, (items + COOP_NT / 32 - 1) / (COOP_NT / 32));
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(COOP_NT);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, naive_coop_kernel<S, LOSSY>, (T *)f, fs, ce, ca, nx, ny, nz, pitch, kz, neg_dt, step0,
                              nsteps, src, sc, e_backwards(sizeof(T), nx, ny, nz), bar, err, timeout_ns);
}

} // namespace

cudaError_t launch_naive_coop(void *f, long long fs, int fmt, const float *ce, const float *ca, int nx, int ny, int nz,
                              int pitch, float neg_dt, long long step0, int nsteps, const SrcSet &src, const Scales &sc,
                              int *bar, int *err, long long timeout_ns, int sms, cudaStream_t st)
{
    if (ca)
        DISPATCH_FORMAT(fmt, S, launch_coop<S, true>(f, fs, ce, ca, nx, ny, nz, pitch, neg_dt, step0, nsteps, src, sc, bar,
                                                     err, timeout_ns, sms, st));
    DISPATCH_FORMAT(fmt, S, launch_coop<S, false>(f, fs, ce, ca, nx, ny, nz, pitch, neg_dt, step0, nsteps, src, sc, bar, err,
                                                  timeout_ns, sms, st));
}

double naive_coop_row_steps(int nx, int ny, int nz, int sms)
{
    const int kz = rows_per_warp(nx, ny, nz, sms);
    const long long warps = (long long)sms * (COOP_NT / 32), items = (long long)((nx + 31) / 32) * ny * ((nz + kz - 1) / kz);
    return (double)((items + warps - 1) / warps) * (kz + 1);
}

int naive_block_max_cells() { return NAIVE_BLOCK_CELLS; }

cudaError_t launch_naive_block(void *const f[6], int fmt, const float *ce, const float *ca, int nx, int ny, int nz,
                               int pitch, float neg_dt, long long step0, int nsteps, const SrcSet &src,
                               const Scales &sc, cudaStream_t st)
{
    DISPATCH_FORMAT(fmt, S, launch_block<S>(f, ce, ca, nx, ny, nz, pitch, neg_dt, step0, nsteps, src, sc, st));
}

cudaError_t launch_naive_h(void *const f[6], int fmt, int nx, int ny, int nz, int pitch, float neg_dt,
                           const Scales &sc, cudaStream_t st)
{
    DISPATCH_FORMAT(fmt, S, launch_h<S>(f, nx, ny, nz, pitch, neg_dt, sc, st));
}

cudaError_t launch_naive_e(void *const f[6], int fmt, const float *ce, const float *ca, int nx, int ny, int nz,
                           int pitch, long long step, const SrcSet &src, const Scales &sc, cudaStream_t st)
{
    DISPATCH_FORMAT(fmt, S, launch_e<S>(f, ce, ca, nx, ny, nz, pitch, step, src, sc, st));
}
