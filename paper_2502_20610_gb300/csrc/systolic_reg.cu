// Systolic schedule, register-resident form (Sec. 3, Fig. 7; Sec. 4).
//
// Same method as systolic.cu: each CTA owns a tile, a box [A, A+n) of
// skewed space sigma = p + t, scans it down the x-y-z-t diagonal, takes its
// lower shell (level t) from the upwind tiles through global memory and
// leaves its top faces there for the downwind ones, with per-tile progress
// flags and no grid-wide synchronisation.  What differs is where the tile
// lives: in registers instead of shared memory.
//
//   x: lane = physical x mod 32 (a ring, as in shared memory);
//   y: warp = physical y mod 16 (a ring);
//   z: register row r in [-1, NZ) = skewed z, sigma_z = A_z + r.
//
// Because rows are indexed by skewed z, the value a row needs from the
// previous level sits one row below it in the same thread (sigma - 1 is the
// same physical cell one step earlier): the diagonal scan is an implicit
// register shift, H[r] <- f(H[r-1], E[r-1], E[r], ...), applied top-down in
// place.  Row -1 holds the lower z shell.  x neighbours come by warp
// shuffle, y neighbours through a small shared-memory exchange, so one cell
// update costs 4 shared-memory loads/stores, 4 shuffles and 24 FP32
// operations instead of ~27 shared-memory accesses.
//
// The slot that leaves the tile at the top in x (one lane per warp) and in y
// (one warp) is refilled each step with the lower x / y shell, and row -1
// with the lower z shell.  All three shells of level t are fetched into a
// shared staging buffer by bulk tensor copies (TMA): the z shell (with its x
// and y edges) from the field arrays, the y and x shells from two face
// buffers, one copy per shell for the six fields (the field index is a
// dimension of the copy) and one per shell for the coefficients.  Each
// thread waits on the buffer's mbarrier itself.
//
// Face buffers: the top y and x faces of a tile do not go to the field
// arrays but to a y-face and an x-face buffer indexed by physical (x, y) and
// by skewed z modulo a period of whole tile z-extents, in z-blocks: rows
// 1..NZ of a column sit at consecutive addresses (rounded up to 16 bytes), at
// a place that stays fixed for the whole life of the tile.  So the lane
// leaving the box in x and the warp leaving it in y store their whole columns
// with 16-byte stores, and the x lane and the y-shell warp refill theirs
// with 16-byte shared loads.  Columns are stored and read whole, rows outside
// the grid in z included (their E is 0, see below): the period is a tile's z
// extent longer than the grid, so that no tile's rows share a block with
// another's that are still to be read, and a wrapped position is next written
// only by a tile downwind of every reader of the value there (the CPU model
// checks both).
//
// Bookkeeping: two warps of their own.  One polls the upwind tiles and fetches
// the next step's shells as soon as their staging buffer is free, the other
// publishes the tile's levels.  While the warp whose y slot is outside the box
// did this between its refills, its chain of stores, release, poll and copies
// (3100 of 9500 cycles) was as long as the other warps' half-steps and stores.
//
// Code size: the step is some 3500 instructions long, and what lies between
// is fetched with it.  Taking the cold paths out of the loop (row-by-row
// stores and clearing at the grid's ends in z, masks of the H half-step, the
// launch's last step, the capture box, a search for a source's row) gave
// 172.8 -> 193 GCUPS at 256^3 and 180 -> 196 at 512^3 before the bookkeeping
// warp, which gave 201 and 216 (FP16 at 256^3: 163 -> 188).
//
// Top faces: the z face goes to the field arrays and the y and x faces to
// their buffers at the end of each step, each warp then arriving at that step's
// barrier (of four in turn), which the publishing warp watches: a level is
// published as soon as its last face is stored.  A cell's path through time
// crosses into the next tile every 1 / (1/31 + 1/15 + 1/12) = 5.5 steps, so on
// domains that do not fill the chip this delay is a part of every step: with
// the y face stored a step late and a level published after B2 of the step
// after, 64^3 x 200 steps took 1082 us, now 982 (128^3 FP16 146 -> 155 GCUPS,
// 200 x 200 x 100 163 -> 169, 256^3 unchanged at 213).  An arrival costs least:
// a release store a warp instead took 1.5 %, with a look at the abort word 3 %.
//
// Two barriers per step: B1, after the E rows are exchanged for the H
// half-step, and B2, after the H rows are exchanged for the E half-step.  A
// warp arrives as soon as its rows are written (the H rows are written as they
// are computed) and waits only when it needs its neighbour's: its z and x face
// stores lie between arrival and wait of B1, its refills between those of B2.
// With block barriers after the stores and refills: 201 GCUPS at 256^3, 216 at
// 512^3, FP16 188 at 256^3, lossy 162 at 224^3; so 208, 223, 197 and 167.
//
// Masks: none but the low walls'.  A cell outside the domain has dt/eps = 0
// (the coefficient shells are zero-filled there), so its E stays 0; its H is
// only read by such cells and by the tangential E of the low walls, which
// stays as it is (the masked form of the E half-step, on steps whose box
// touches a low wall).  Every arithmetic step is yee_cell.cuh, so the result
// equals the naive schedule bit for bit, but for one case: an infinite H beside
// a high wall makes a NaN of 0 times infinity beyond it, and a value there that
// is infinite in the naive schedule may then be NaN.  (The same values are not
// finite in both.  Masks for the high walls in the masked form, and so in a part
// of the cases only, cost 0.7 % at 256^3, 1.4 % at 128^3 in FP16.)
//
// Storage: fields live in global memory as FP32, FP16 or BF16 (S, see
// storage.cuh); registers hold FP32 values already rounded to the storage
// format, so each new H value is rounded where it is computed and each new
// E value once its point source (if any) has been added, exactly where the
// naive schedule rounds on store.  dt/eps stays FP32.
#include "internal.h"
#include "storage.cuh"
#include "sys_common.cuh"
#include "yee_cell.cuh"

#include <type_traits>

namespace {

using namespace sysc;

template <int NZ_, class S_, bool LOSSY_, int TY_, int CL_ = 1, bool CAP_ = false>
struct RegTile {
    using S = S_;
    static constexpr bool LOSSY = LOSSY_;  // conducting cells: E <- ca E + cb curl H
    static constexpr bool CAP = CAP_;      // the adjoint's launches: store the capture box's E every step
    // CTAs per thread-block cluster along x: 2 = pairs of x-adjacent tiles,
    // the upwind one sending its top x face through distributed shared memory
    static constexpr int CL = CL_;
    static_assert(CL_ == 1 || (CL_ == 2 && !LOSSY_), "clusters of one, or x pairs of lossless tiles");
    using T = typename S_::T;
    static constexpr int NZ = NZ_;        // updated z rows (registers 0..NZ-1)
    static constexpr int NR = NZ_ + 1;    // plus the shell row -1
    static constexpr int RY = 16, NTC = 32 * RY;  // y slots = compute warps
    // and a warpgroup for the bookkeeping (two warps of it work), whose registers
    // the compute warps take over: 640 * 96 = 512 * 112 + 128 * 32
    static constexpr int NT = NTC + 128;
    static constexpr int CREG = 112, BREG = 32;
    static_assert(NTC * CREG + (NT - NTC) * BREG <= NT * 96, "within the launch's registers");
    // TY = RY - 1: one y slot outside the box, the y shell (its warp also
    // holds the previous step's top y row until its refill); TY = RY - 2:
    // the previous top row has a slot (and warp) of its own
    static constexpr int TX = 31, TY = TY_, TZ = NZ_;
    static_assert(TY_ == RY - 1 || TY_ == RY - 2, "one or two y slots outside the box");
    static_assert(NR <= 16 && TY <= 16, "cooperative entries: row < 16, warp offset < 16");
    static_assert(NZ % 4 == 0, "rows move in groups of four (16-byte accesses) and pairs (packed rounding)");
    // shared memory, in floats
    // y-neighbour exchange, one component.  VX (16-bit storage): [warp][lane]
    // [row], rows moved in 16-byte groups of four; a lane's rows start XR
    // floats after the previous lane's, XR / 4 odd, so the 8 lanes of a
    // quarter warp hit disjoint banks.  FP32: [warp][row][lane], one row per
    // access (measured faster there: 176 vs 169 GCUPS at 256^3, while 16-bit
    // storage gains 156 -> 164 from the vector form)
    static constexpr bool VX = S_::narrow;
    static constexpr int XR = (NZ_ / 4) % 2 ? NZ_ : NZ_ + 4;
    // pitch of the coefficient ring's rows: 33 where there is room, so that one
    // lane's column (the x shell's, copied by a lane a row: 2 accesses instead of
    // the 24 of that lane alone; FP32 256^3 207.8 -> 212.3 GCUPS, lossy 224^3 167.2
    // -> 173.7) falls on as many banks
    static constexpr int CP = CL_ == 2 ? 32 : 33;
    static constexpr int XE_F = VX ? RY * 32 * XR : RY * NZ_ * 32;
    // lower-shell staging, filled per step by bulk tensor copies (TMA) of
    // boxes whose x start is rounded down to 16 bytes (XA elements): SW =
    // 32 + XA elements cover the 32-wide x window.  One copy per shell
    // fetches all six fields ([field][...] in shared memory), one more the
    // FP32 coefficients (C-suffixed sizes, [cb, ca][...]); sizes below are
    // per array, in elements, and every shell's region starts on a 128-byte
    // boundary.
    static constexpr int EB = (int)sizeof(T);
    static constexpr int XA = 16 / EB, SW = 32 + XA;
    static constexpr int ZB = RY * SW;        // z shell box {SW,16,1}: [y][x]
    // The top x and y faces go to two face buffers in z-blocks: rows 1..NZ of
    // one (x, y) column of a tile sit at BZ consecutive elements (NZ rounded
    // up to 16 bytes), so shells and faces move with 16-byte accesses.
    static constexpr int BZ = (NZ_ * EB + 15) / 16 * 16 / EB;
    static_assert(BZ % (16 / EB) == 0 && NZ_ % 4 == 0, "z-blocks of whole 16-byte chunks, 4 rows per access");
    static constexpr int YB = 32 * BZ;        // y shell box {BZ,32,1} from the y-face buffer: [x][z]
    static constexpr int XB = 16 * BZ;        // x shell box {BZ,16,1} from the x-face buffer: [y][z]
    static constexpr int XAC = 4, SWC = 36;
    static constexpr int ZBC = RY * SWC, YBC = NR * SWC, XBC = NR * 16 * XAC;
    static constexpr int NCOEF = LOSSY ? 2 : 1;   // FP32 coefficient arrays: cb (dt/eps), ca
    static constexpr size_t r128(size_t b) { return (b + 127) / 128 * 128; }
    // byte offsets of the shells within one staging buffer: of the fields, and of
    // the coefficients
    static constexpr size_t OFF_Y = r128(6 * (size_t)ZB * EB);
    static constexpr size_t OFF_X = OFF_Y + r128(6 * (size_t)YB * EB);
    static constexpr size_t STG_B = OFF_X + r128(6 * (size_t)XB * EB);
    static constexpr size_t OFF_YC = r128(NCOEF * 4 * (size_t)ZBC);
    static constexpr size_t OFF_XC = OFF_YC + r128(NCOEF * 4 * (size_t)YBC);
    static constexpr size_t COF_B = OFF_XC + r128(NCOEF * 4 * (size_t)XBC);
    static constexpr unsigned FIELD_BYTES = 6u * EB * (ZB + YB + XB), COEF_BYTES = NCOEF * 4u * (ZBC + YBC + XBC);
    // staging buffers: two, so that a step's shells are fetched during the step
    // before.  The lossy form's second coefficient leaves room for one buffer of
    // coefficients beside the two of fields, on a barrier of its own: coefficients
    // are read before B2 only, so they are fetched from B2 on, and need no upwind
    // tile.  (One buffer for everything, fetched from B1 on, left the copies'
    // latency in every step: 224^3 FP32, 130 -> 162 GCUPS.)
    static constexpr int NCBUF = LOSSY_ ? 1 : 2;
    // coefficient ring rows: a power of two, or (lossy, for room) just a column
    static constexpr int CR = LOSSY_ ? NR : 16;
    // and, where there is room, its first NZ rows once more behind the others: the
    // E half-step then reads a column at fixed offsets from one address instead
    // of wrapping every row (FP16 256^3 198.4 -> 201.0 GCUPS, FP32 212.2 -> 213.0)
    static constexpr bool MIR = !LOSSY_ && CL_ == 1;
    static constexpr int CRM = MIR ? 16 + NZ_ : CR;
    static constexpr int CE_F = RY * CRM * CP;
    static_assert(CR >= NR, "coefficient ring holds the whole column");
    // x pairs: the downwind tile's receive ring of x faces, NSLOT slots of
    // [field][box row y][z-block] (rows 1..NZ of the x shell of one step)
    static constexpr int NSLOT = 6;
    static constexpr int RXS = 6 * 16 * BZ;  // elements per slot
    static constexpr size_t RX_B = CL_ == 2 ? NSLOT * (size_t)RXS * EB : 0;
    static constexpr size_t smem_bytes()
    {
        return 2 * STG_B + NCBUF * COF_B + sizeof(float) * (4 * (size_t)XE_F + ((size_t)NCOEF * CE_F + 3) / 4 * 4) + RX_B;
    }
};

__device__ __forceinline__ float shfl_from(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// Named barrier of the compute warps with the two bookkeeping warps at a tile's start.
__device__ __forceinline__ void bar_tile() { asm volatile("bar.sync 2, 576;" ::: "memory"); }

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// Four consecutive rows of one field as one 16-byte (FP32) or 8-byte (16-bit)
// access: p must be aligned to it.
template <class S>
__device__ __forceinline__ void ld4(const typename S::T *p, float s, float &a, float &b, float &c, float &d)
{
    if constexpr (sizeof(typename S::T) == 4) {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        a = v.x; b = v.y; c = v.z; d = v.w;
    } else {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        a = S::dec((typename S::T)(v.x & 0xffffu), s); b = S::dec((typename S::T)(v.x >> 16), s);
        c = S::dec((typename S::T)(v.y & 0xffffu), s); d = S::dec((typename S::T)(v.y >> 16), s);
    }
}

template <class S>
__device__ __forceinline__ void st4(typename S::T *p, float is, float a, float b, float c, float d)
{
    if constexpr (sizeof(typename S::T) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
    } else {
        uint2 v;
        v.x = S::enc2(a, b, is);
        v.y = S::enc2(c, d, is);
        *reinterpret_cast<uint2 *>(p) = v;
    }
}

// Rows 1..NZ of one field of a column, loaded from a z-block and stored into one.
template <class S, int NR>
__device__ __forceinline__ void ld_rows(const typename S::T *p, float s, float (&v)[NR])
{
#pragma unroll
    for (int q = 0; q < (NR - 1) / 4; ++q) ld4<S>(p + 4 * q, s, v[4 * q + 1], v[4 * q + 2], v[4 * q + 3], v[4 * q + 4]);
}

template <class S, int NR>
__device__ __forceinline__ void st_rows(typename S::T *p, float is, const float (&v)[NR])
{
#pragma unroll
    for (int q = 0; q < (NR - 1) / 4; ++q)
        st4<S>(p + 4 * q, is, v[4 * q + 1], v[4 * q + 2], v[4 * q + 3], v[4 * q + 4]);
}

// Bulk tensor copy of one box of a 4D map (TMA: x, y, z, array) starting at
// array 0 into shared memory, completing on an mbarrier; elements outside
// the tensor are written as zero.
__device__ __forceinline__ void tma_box(void *dst, const CUtensorMap *map, int x, int y, int z,
                                        unsigned long long *bar)
{
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
                 "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z), "r"(0),
                 "r"(smem_u32(bar))
                 : "memory");
}

// The same for a 5D map (face buffers: z-block rows, y or x, x or y, block,
// field), starting at field 0.
__device__ __forceinline__ void tma_box5(void *dst, const CUtensorMap *map, int r, int a, int b, int kb,
                                         unsigned long long *bar)
{
    asm volatile("cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(smem_u32(dst)),
                 "l"(reinterpret_cast<unsigned long long>(map)), "r"(r), "r"(a), "r"(b), "r"(kb), "r"(0),
                 "r"(smem_u32(bar))
                 : "memory");
}

// Thread-block cluster primitives (x pairs).
__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// the shared::cluster address of local shared address `a` in CTA `rank`
__device__ __forceinline__ unsigned mapa(unsigned a, unsigned rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// every thread of every CTA of the cluster (orders all prior memory accesses,
// distributed shared memory included, before all later ones)
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void st_remote_u32(unsigned a, unsigned v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void arrive_remote(unsigned bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Four rows of one field into another CTA's shared memory (16 bytes FP32,
// 8 bytes 16-bit, packed as st4 does).
template <class S>
__device__ __forceinline__ void st4_remote(unsigned a, float is, float x, float y, float z, float w)
{
    if constexpr (sizeof(typename S::T) == 4) {
        asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w)
                     : "memory");
    } else {
        asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(S::enc2(x, y, is)),
                     "r"(S::enc2(z, w, is))
                     : "memory");
    }
}
template <class S, int NR>
__device__ __forceinline__ void st_rows_remote(unsigned a, float is, const float (&v)[NR])
{
#pragma unroll
    for (int q = 0; q < (NR - 1) / 4; ++q)
        st4_remote<S>(a + 4 * q * (unsigned)sizeof(typename S::T), is, v[4 * q + 1], v[4 * q + 2], v[4 * q + 3],
                      v[4 * q + 4]);
}

// Bounded wait (acquire at cluster scope) for phase `parity` of a local
// mbarrier that a partner CTA of the cluster completes.  Returns false (error
// word set) past the launch's timeout.
__device__ bool wait_cluster_bar(const SysLaunch &P, unsigned long long *bar, unsigned parity, int ticket)
{
    unsigned long long t0 = 0;
    for (int it = 0;; ++it) {
        unsigned done;
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;"
                     " selp.u32 %0, 1, 0, p; }"
                     : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        if (done) return true;
        if (ld_volatile(P.ctrl + 1) != DEV_OK) return false;
        const unsigned long long now = globaltimer();
        if (it == 0) {
            t0 = now;
        } else if (now - t0 > (unsigned long long)P.timeout_ns) {
            if (atomicCAS(P.ctrl + 1, DEV_OK, DEV_ERR_TIMEOUT) == DEV_OK) {
                P.ctrl[2] = ticket;
                P.ctrl[3] = -2;
            }
            return false;
        }
    }
}

// True once the wait that began at t0 (set on the first call) is past `ns`.
__device__ __forceinline__ bool past(unsigned long long &t0, unsigned long long ns)
{
    const unsigned long long now = globaltimer();
    if (t0 == 0) t0 = now;
    return now - t0 > ns;
}

__device__ __noinline__ void timed_out(int *ctrl, int ticket, int what)
{
    if (atomicCAS(ctrl + 1, DEV_OK, DEV_ERR_TIMEOUT) == DEV_OK) {
        ctrl[2] = ticket;
        ctrl[3] = what;
    }
}

// Release / acquire at CTA scope on a shared word: how the compute warps and
// the bookkeeping warps tell each other where they are.
__device__ __forceinline__ void st_rel_cta(unsigned *p, unsigned v)
{
    asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_acq_cta(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}

// Bounded wait for phase `parity` of a staging barrier; gives up at once when
// a bookkeeping warp has (*quit).  False: the error word is set.
__device__ bool wait_stage(const SysLaunch &P, unsigned long long *bar, unsigned parity, const unsigned *quit, int ticket)
{
    unsigned long long t0 = 0;
    for (;;) {
        unsigned done;
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;"
                     " selp.u32 %0, 1, 0, p; }"
                     : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        if (done) return true;
        if (quit && ld_acq_cta(quit)) return false;
        if (past(t0, 2 * (unsigned long long)P.timeout_ns)) {
            timed_out(P.ctrl, ticket, -1);
            return false;
        }
    }
}

// The two barriers of a step, as an arrival of each compute warp (once its
// lanes' shared-memory accesses before it are done) and a wait later: what a
// warp does in between holds nobody up.  The wait is bounded and ends when the
// CTA gives up (*quit); every lane gets the same answer.
__device__ __forceinline__ void half_arrive(unsigned long long *bar)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool half_wait(const SysLaunch &P, unsigned long long *bar, unsigned parity, const int *quit,
                                          int ticket)
{
    unsigned long long t0 = 0;
    for (;;) {
        unsigned done;
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;"
                     " selp.u32 %0, 1, 0, p; }"
                     : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        if (__all_sync(0xffffffffu, done)) return true;
        bool late = past(t0, 4 * (unsigned long long)P.timeout_ns);
        if (late) timed_out(P.ctrl, ticket, -4);
        late |= *(const volatile int *)quit != 0;
        if (__any_sync(0xffffffffu, late)) return false;
    }
}

template <class R>
__global__ void __launch_bounds__(R::NT, 1) systolic_reg_kernel(const __grid_constant__ SysLaunch P)
{
    using S = typename R::S;
    using T = typename R::T;
    constexpr int NZ = R::NZ, NR = R::NR, TX = R::TX, TY = R::TY, TZ = R::TZ;
    constexpr int SW = R::SW, XA = R::XA, SWC = R::SWC;
    extern __shared__ __align__(1024) float4 smem4[];
    // staging buffers first (the dynamic shared memory base is 1024-byte
    // aligned): the lower z, y and x shells of the 6 fields, twice, then those
    // of dt/eps (and ca)
    char *const stg0 = reinterpret_cast<char *>(smem4);
    // y exchange (layout: RegTile::VX): E^t (level t-1) rows i = 0..NZ-1, and
    // the new H rows r = 1..NZ at row r-1
    char *const cof0 = stg0 + 2 * R::STG_B;
    float *const XEx = reinterpret_cast<float *>(cof0 + R::NCBUF * R::COF_B);
    float *const XEz = XEx + R::XE_F;
    float *const XHx = XEz + R::XE_F;
    float *const XHz = XHx + R::XE_F;
    // element (warp, row, lane) of one exchanged component
    auto xe_at = [](int wq, int row, int ln) {
        return R::VX ? (wq * 32 + ln) * R::XR + row : (wq * NZ + row) * 32 + ln;
    };
    // dt/eps of each column, indexed by physical z mod CR: a cell's coefficient
    // stays in place while the skewed register rows move past it
    float *const CEs = XHz + R::XE_F;      // [warp][ring row][lane], pitch CP
    float *const CAs = CEs + R::CE_F;      // the same for ca (lossy only)
    // x pairs: the receive ring of x faces (downwind CTA), after the rings
    T *const RX = reinterpret_cast<T *>(CEs + (R::NCOEF * R::CE_F + 3) / 4 * 4);  // [slot][field][box row][BZ]
    __shared__ int s_ticket, s_abort;
    // x pairs: a slot of the receive ring is full (the upwind CTA arrives
    // once its x lanes have written it) / free again (the downwind CTA arrives)
    __shared__ alignas(8) unsigned long long s_rxf[R::NSLOT], s_rxe[R::NSLOT];
    __shared__ alignas(8) unsigned long long s_bar[3];  // staging barriers, one per buffer (lossy: and the
                                                        // coefficients'): one phase per fill
    // the bookkeeping warps' view of the compute warps: B1 barriers passed over
    // the CTA's life, and a barrier each for four steps in turn, which the compute
    // warps arrive at once a step's faces are stored.  s_told: the steps that the
    // publishing warp has seen there; s_quit: a bookkeeping warp has given up
    __shared__ unsigned s_steps, s_told, s_quit;
    __shared__ alignas(8) unsigned long long s_fin[4];
    __shared__ alignas(8) unsigned long long s_half[3];  // B1 and B2 (lossy: and a step's coefficients read)
    __shared__ int s_pfail;  // ... before the tile's first step
    __shared__ unsigned s_seen[3];

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const float ndt = P.neg_dt;
    const long long sxy = (long long)P.pitch * P.ny;
    // field pointers and scales are read from the kernel parameters where
    // used (they stay in the constant bank instead of taking registers)
#define F0 reinterpret_cast<T *>(P.f[0])
#define F1 reinterpret_cast<T *>(P.f[1])
#define F2 reinterpret_cast<T *>(P.f[2])
#define F3 reinterpret_cast<T *>(P.f[3])
#define F4 reinterpret_cast<T *>(P.f[4])
#define F5 reinterpret_cast<T *>(P.f[5])
#define CE P.ce
#define CA P.ca
#define SC(c) P.sc.s[c]
#define IS(c) P.sc.is[c]
#define RND(v, c) S::rnd(v, SC(c), IS(c))
#define RND2(a, b, c) S::rnd2(a, b, SC(c), IS(c))
#define STORE6(g, i)                                                                          \
    do {                                                                                      \
        F0[g] = S::enc(ex[i], IS(0)); F1[g] = S::enc(ey[i], IS(1)); F2[g] = S::enc(ez[i], IS(2)); \
        F3[g] = S::enc(hx[i], IS(3)); F4[g] = S::enc(hy[i], IS(4)); F5[g] = S::enc(hz[i], IS(5)); \
    } while (0)

    // Face buffers: rows 1..NZ of component f of column (x, y) of a tile in
    // z-block kb are at
    //   x faces: XF + f*fxs + ((kb*nx + x)*ny + y)*BZ + (row - 1),
    //   y faces: YF + f*fys + ((kb*ny + y)*nx + x)*BZ + (row - 1),
    // kb = K mod (number of z-blocks): block kb holds skewed z (sigma_z = z +
    // t) modulo the blocks' period, so a tile's faces and lower x / y shells
    // keep one aligned place for its whole life, and a face (or shell) of one
    // tile step is one contiguous run per field.  A tile's top x face is
    // stored by the lane leaving the box in x, its top y face by the warp
    // leaving it in y, straight from registers.
    T *const XF = reinterpret_cast<T *>(P.xf);
    T *const YF = reinterpret_cast<T *>(P.yf);
    constexpr int BZ = R::BZ;
#define FACE_STORE(dst, fs)                                                              \
    do {                                                                                \
        st_rows<S>((dst), IS(0), ex); st_rows<S>((dst) + (fs), IS(1), ey);               \
        st_rows<S>((dst) + 2 * (fs), IS(2), ez); st_rows<S>((dst) + 3 * (fs), IS(3), hx); \
        st_rows<S>((dst) + 4 * (fs), IS(4), hy); st_rows<S>((dst) + 5 * (fs), IS(5), hz); \
    } while (0)

    constexpr int CR = R::CR, CP = R::CP, CRM = R::CRM;
    if (tid < 4)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_fin[tid])), "r"(R::RY) : "memory");
    if (tid == 0) {
        s_steps = s_told = s_quit = 0u;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_bar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_bar[1])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_bar[2])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_half[0])), "r"(R::RY) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_half[1])), "r"(R::RY) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_half[2])), "r"(R::RY) : "memory");
        if constexpr (R::CL == 2) {
#pragma unroll
            for (int k = 0; k < R::NSLOT; ++k) {
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_rxf[k])) : "memory");
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_rxe[k])) : "memory");
            }
        }
    }
    if (tid < 4) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    // x pairs: rank 0 holds the upwind tile (I even), rank 1 the downwind one;
    // every CTA of the cluster must be running before distributed shared
    // memory is touched
    const unsigned rank = R::CL == 2 ? cluster_rank() : 0u;
    if constexpr (R::CL == 2) cluster_sync_all();
    const unsigned rx_remote = R::CL == 2 ? mapa(smem_u32(RX), 1u) : 0u;        // rank 0 -> rank 1's ring
    const unsigned rxf_remote = R::CL == 2 ? mapa(smem_u32(&s_rxf[0]), 1u) : 0u;
    const unsigned rxe_remote = R::CL == 2 ? mapa(smem_u32(&s_rxe[0]), 0u) : 0u;  // rank 1 -> rank 0
    // the tile of a ticket (x pairs: this CTA's half of it, I may be past the last)
    auto tile_of = [&](int ticket, int &I, int &J, int &K) {
        const int tl = P.tiles[ticket];
        const int gxe = R::CL == 2 ? (P.gx + 1) / 2 : P.gx;
        I = tl % gxe;
        if (R::CL == 2) I = 2 * I + (int)rank;
        J = (tl / gxe) % P.gy;
        K = tl / (gxe * P.gy);
    };
    // messages (x faces) sent / received over this CTA's life: message m
    // uses slot m % NSLOT, its (m / NSLOT)-th use of that slot
    int msg_base = 0;
    // slot to signal after the next block barrier (the y-shell warp does it):
    // rank 0, the slot its x lanes have just filled; rank 1, the slot its x
    // lane has just read
    int sig_slot = -1;
    if (w >= R::RY) {
        // ----------------------------------------------- bookkeeping warps
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R::BREG));
        if (w > R::RY + 1) {
            // (x pairs: cluster barriers count every thread that has not left)
            return;
        }
        // The first polls the upwind tiles' progress and fetches a step's lower
        // shells (six bulk tensor copies; x start rounded down to 16 bytes, zero
        // fill off the domain) as soon as their staging buffer is free.  The
        // second publishes the tile's own levels: the release of a flag waits for
        // the CTA's stores to land (1000 to 1900 cycles), and a poll and the
        // copies take as long again.
        const bool publisher = w == R::RY + 1;
        unsigned steps0 = 0, n0 = 0, n1 = 0, n2 = 0;  // s_steps at the tile's start; fills of each buffer
        unsigned n_fin = 0;  // steps before the tile's (fetch), steps seen finished (publisher)
        auto fetch_coefs = [&](int t, int Ax, int Ay, int Az, char *sb, unsigned long long *bar) {
            const int bx = Ax - t, by = Ay - t, bz = Az - t, x0c = (bx - 1) & ~(R::XAC - 1);
            tma_box(sb, &P.tm[0][1], x0c, by - 1, bz - 1, bar);
            tma_box(sb + R::OFF_YC, &P.tm[1][1], x0c, by - 1, bz - 1, bar);
            tma_box(sb + R::OFF_XC, &P.tm[2][1], x0c, by, bz - 1, bar);
        };
        for (;;) {
            if constexpr (R::CL == 2) cluster_sync_all(); else bar_tile();
            if constexpr (R::CL == 2) cluster_sync_all(); else bar_tile();
            const int ticket = s_ticket;
            if (s_abort || ticket >= P.ntiles) break;
            int I, J, K;
            tile_of(ticket, I, J, K);
            if (R::CL == 2 && I >= P.gx) continue;
            const int tile = I + P.gx * (J + P.gy * K);
            const int Ax = I * TX, Ay = J * TY, Az = K * TZ, kb = K % P.nzblk;
            const Interval iv = tile_interval<TX, TY, TZ>(P, I, J, K);
            Upwind U;
            upwind_of<TX, TY, TZ>(P, I, J, K, U);
            if (publisher) {
                bar_tile();
                if (s_pfail) continue;
                // a tile that starts late (or, start > end, enters the domain only
                // after this launch) carries its upwind tiles' guarantee on
                if (iv.s > 0 && lane == 0) publish(P, tile, ticket, P.epoch + (unsigned)iv.s);
                if (iv.s > iv.e) continue;
                unsigned long long t_own = 0;
                for (int t = iv.s; t <= iv.e;) {
                    unsigned fin;
                    asm volatile("{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;"
                                 " selp.u32 %0, 1, 0, p; }"
                                 : "=r"(fin) : "r"(smem_u32(&s_fin[n_fin & 3u])), "r"((n_fin >> 2) & 1u) : "memory");
                    if (__all_sync(0xffffffffu, fin)) {
                        ++t;
                        ++n_fin;
                        if (lane == 0) {
                            *(volatile unsigned *)&s_told = n_fin;
                            publish(P, tile, ticket, P.epoch + (unsigned)t);
                        }
                        t_own = 0;
                        continue;
                    }
                    __nanosleep(32);
                    bool late = lane == 0 && past(t_own, 8 * (unsigned long long)P.timeout_ns);
                    if (late) {
                        timed_out(P.ctrl, ticket, -3);
                        st_rel_cta(&s_quit, 1u);
                    }
                    late |= *(volatile int *)&s_abort != 0;
                    if (__any_sync(0xffffffffu, late)) break;
                }
                continue;
            }
            if (lane < 3) s_seen[lane] = 0u;
            __syncwarp();
            bool ok = iv.s == 0 || wait_level(P, U, s_seen, iv.s - 1, ticket);
            if (lane == 0) s_pfail = !ok;
            bar_tile();
            if (!ok || iv.s > iv.e) continue;
            int t = iv.s, tc = iv.s;                 // the next step to fetch (tc: lossy, its coefficients)
            unsigned long long t_up = 0, t_own = 0;  // waiting for the upwind tiles, for the compute warps
            while (ok && (t <= iv.e || (R::LOSSY && tc <= iv.e))) {
                bool idle = true;
                if (R::LOSSY && tc <= iv.e) {  // the coefficients' buffer: free once step tc - 1 has read it
                    unsigned read = 1;
                    if (n2 > 0)  // (reads of fill n2 - 1; the compute warps cannot be a phase ahead of it)
                        asm volatile("{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;"
                                     " selp.u32 %0, 1, 0, p; }"
                                     : "=r"(read) : "r"(smem_u32(&s_half[2])), "r"((n2 - 1u) & 1u) : "memory");
                    if (__all_sync(0xffffffffu, read)) {
                        idle = false;
                        if (lane == 0) {
                            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&s_bar[2])),
                                         "r"(R::COEF_BYTES) : "memory");
                            fetch_coefs(tc, Ax, Ay, Az, cof0, &s_bar[2]);
                        }
                        ++tc;
                        ++n2;
                    }
                }
                // step t's buffer: free at the tile's start, else once B1 of step
                // t - 1 has been passed.  (And no step may finish whose barrier has
                // one that the publishing warp has not seen: four steps before it)
                const unsigned passed = __shfl_sync(0xffffffffu, ld_acq_cta(&s_steps), 0);
                const unsigned told = __shfl_sync(0xffffffffu, *(volatile unsigned *)&s_told, 0);
                if (t <= iv.e && (t < iv.s + 2 || ((int)(passed - (steps0 + (unsigned)(t - iv.s))) >= 0 &&
                                                   (int)(told + 3u - (n_fin + (unsigned)(t - iv.s))) >= 0))) {
                    idle = false;
                    if (level_ready(P, U, s_seen, t)) {
                        __syncwarp();  // orders lanes 1, 2's acquires before lane 0's copies
                        if (lane == 0) {
                            const int bx = Ax - t, by = Ay - t, bz = Az - t, b = t & 1;
                            const int x0 = (bx - 1) & ~(XA - 1);
                            char *const sb = stg0 + (size_t)b * R::STG_B;
                            unsigned long long *const bar = &s_bar[b];
                            // order this thread's view of the upwind tiles' global stores
                            // (generic proxy, acquired through their progress flags)
                            // before the bulk copies that read them
                            asm volatile("fence.proxy.async.global;" ::: "memory");
                            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                                         "r"(R::FIELD_BYTES + (R::LOSSY ? 0u : R::COEF_BYTES)) : "memory");
                            tma_box(sb, &P.tm[0][0], x0, by - 1, bz - 1, bar);                 // z shell: field arrays
                            tma_box5(sb + R::OFF_Y, &P.tm[1][0], 0, bx, by - 1, kb, bar);      // y shell: y-face buffer
                            tma_box5(sb + R::OFF_X, &P.tm[2][0], 0, by - 1, bx - 1, kb, bar);  // x shell: x-face buffer
                            if (!R::LOSSY) fetch_coefs(t, Ax, Ay, Az, cof0 + (size_t)b * R::COF_B, bar);
                        }
                        if (t & 1) ++n1;
                        else ++n0;
                        ++t;
                        t_up = t_own = 0;
                    } else {
                        bool late = lane == 0 && past(t_up, (unsigned long long)P.timeout_ns);
                        if (late) timed_out(P.ctrl, ticket, (int)(P.epoch + (unsigned)t + 1u));
                        late |= ld_volatile(P.ctrl + 1) != DEV_OK;
                        ok = !__any_sync(0xffffffffu, late);
                    }
                }
                if (idle) {
                    __nanosleep(32);
                    bool late = lane == 0 && past(t_own, 8 * (unsigned long long)P.timeout_ns);
                    if (late) timed_out(P.ctrl, ticket, -3);
                    late |= *(volatile int *)&s_abort != 0;
                    ok = !__any_sync(0xffffffffu, late);
                }
            }
            if (!ok && lane == 0) st_rel_cta(&s_quit, 1u);
            n_fin += (unsigned)(iv.e - iv.s + 1);
            steps0 += (unsigned)(iv.e - iv.s + 1) + (R::CL == 2 ? 1u : 0u);  // (x pairs: one pass more than steps)
        }
        // no copy may still be writing when the CTA's shared memory goes (after an
        // abort some were never waited for)
        if (lane == 0 && !publisher) {
            if (n0) wait_stage(P, &s_bar[0], (n0 - 1) & 1u, nullptr, -1);
            if (n1) wait_stage(P, &s_bar[1], (n1 - 1) & 1u, nullptr, -1);
            if (n2) wait_stage(P, &s_bar[2], (n2 - 1) & 1u, nullptr, -1);
        }
        __syncwarp();
        if constexpr (R::CL == 2) cluster_sync_all();
        return;
    }

    // ------------------------------------------------------- compute warps
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R::CREG));
    // passes over the step loop (phases of B1 and of B2), and the parities of the
    // next fill of each staging buffer (bits 0, 1; lossy: 2, the coefficients):
    // every thread waits for every phase and keeps the same counts
    unsigned n_half = 0, fills = 0, n_fin = 0;
    // the coefficient ring's row of physical z = bz - 1 + i, with zr the row of
    // bz - 1 (lossless: any number congruent to it)
    auto ring = [](int zr, int i) {
        if (!R::LOSSY) return (zr + i) & (R::CR - 1);
        const int q = zr + i;
        return q >= R::CR ? q - R::CR : q;
    };
    auto put_ce = [&](int row, int ln, float v) {
        CEs[(w * CRM + row) * CP + ln] = v;
        if (R::MIR && row < NZ) CEs[(w * CRM + row + 16) * CP + ln] = v;
    };
    // the tile column of this thread: registers row i <-> r = i-1
    float ex[NR], ey[NR], ez[NR], hx[NR], hy[NR], hz[NR];

    for (;;) {
        if constexpr (R::CL == 2) {
            // the pair takes one ticket: both CTAs have finished their previous
            // tiles (barrier), rank 0 takes the ticket and reads the error
            // word for both, both read them after the second barrier, so the
            // two always stop together
            cluster_sync_all();
            if (rank == 0 && tid == 0) {
                const int tk = atomicAdd(P.ctrl, 1);
                const int ab = ld_volatile(P.ctrl + 1) != DEV_OK;
                s_ticket = tk;
                s_abort = ab;
                st_remote_u32(mapa(smem_u32(&s_ticket), 1u), (unsigned)tk);
                st_remote_u32(mapa(smem_u32(&s_abort), 1u), (unsigned)ab);
            }
            cluster_sync_all();
        } else {
            bar_tile();
            if (tid == 0) {
                s_ticket = atomicAdd(P.ctrl, 1);
                s_abort = ld_volatile(P.ctrl + 1) != DEV_OK;
            }
            bar_tile();
        }
        const int ticket = s_ticket;
        if (s_abort || ticket >= P.ntiles) break;
        bool abort = false;
        int nmsg = 0;
        do {  // one tile (`break` leaves it early: an abort, or a pair member without a tile)
        int I, J, K;
        int m_lo = 1, m_hi = 0;  // x pairs: steps whose x face goes through the ring
        tile_of(ticket, I, J, K);
        if constexpr (R::CL == 2) {
            const int I0 = I - (int)rank;
            if (I0 + 1 < P.gx) {
                const Interval i0 = tile_interval<TX, TY, TZ>(P, I0, J, K);
                const Interval i1 = tile_interval<TX, TY, TZ>(P, I0 + 1, J, K);
                if (i0.s <= i0.e && i1.s <= i1.e) {
                    m_lo = i1.s;
                    m_hi = min(i0.e, i1.e);
                }
            }
            nmsg = max(0, m_hi - m_lo + 1);
            if (I >= P.gx) break;  // the last pair of an odd tile row has one tile
        }
        const int Ax = I * TX, Ay = J * TY, Az = K * TZ;
        const int kb = K % P.nzblk;  // this tile's z-block in the face buffers
        T *const XFk = XF + (long long)kb * P.nx * P.ny * BZ;
        T *const YFk = YF + (long long)kb * P.nx * P.ny * BZ;
        const Interval iv = tile_interval<TX, TY, TZ>(P, I, J, K);
        bar_tile();  // the bookkeeping warp has waited for level start - 1
        if (s_pfail) break;
        if (iv.s > iv.e) continue;  // enters the domain only after this launch: nothing to do

        // ring row of physical z = bz - 1 at the first step
        int zl = R::LOSSY ? (((Az - iv.s - 1) % CR) + CR) % CR : 0;
        const int zr0 = R::LOSSY ? zl : Az - iv.s - 1;
        // initial load: level start-1, rows sigma_z = Az + r at physical Az + r - start + 1
        {
            const int bx = Ax - iv.s, by = Ay - iv.s;
            const int px = bx + ((lane - bx) & 31), py = by + ((w - by) & (R::RY - 1));
            const bool cin = (unsigned)px < (unsigned)P.nx && (unsigned)py < (unsigned)P.ny;
            // rows 1..NZ of the lower x shell column and of the lower y shell
            // row at level start-1: written by the upwind tiles into the face
            // buffers during this launch (start >= 1; the x-face buffer holds
            // the corner column), else the launch's initial state in the
            // field arrays (start = 0); row 0 is the lower z shell
            const bool xshell = px == bx && iv.s > 0;
            const bool yshell = py == by && iv.s > 0 && !xshell;
            const long long col = px + (long long)P.pitch * py;
            const T *const fq = xshell ? XFk + ((long long)px * P.ny + py) * BZ
                                       : YFk + ((long long)py * P.nx + px) * BZ;
            const long long fqs = xshell ? P.fxs : P.fys;
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const int pz = Az + i - 1 - iv.s + 1;
                float c = 0.f, a = 0.f;
                if (cin && (unsigned)pz < (unsigned)P.nz) {
                    const long long g = col + sxy * pz;
                    if (i > 0 && (xshell || yshell)) {  // the upwind tiles' top x / y face of level start-1
                        const T *q = fq + (i - 1);
                        ex[i] = S::dec(S::ld_cg(q), SC(0)); ey[i] = S::dec(S::ld_cg(q + fqs), SC(1));
                        ez[i] = S::dec(S::ld_cg(q + 2 * fqs), SC(2)); hx[i] = S::dec(S::ld_cg(q + 3 * fqs), SC(3));
                        hy[i] = S::dec(S::ld_cg(q + 4 * fqs), SC(4)); hz[i] = S::dec(S::ld_cg(q + 5 * fqs), SC(5));
                    } else {
                        ex[i] = S::dec(S::ld_cg(F0 + g), SC(0)); ey[i] = S::dec(S::ld_cg(F1 + g), SC(1));
                        ez[i] = S::dec(S::ld_cg(F2 + g), SC(2)); hx[i] = S::dec(S::ld_cg(F3 + g), SC(3));
                        hy[i] = S::dec(S::ld_cg(F4 + g), SC(4)); hz[i] = S::dec(S::ld_cg(F5 + g), SC(5));
                    }
                    c = __ldg(CE + g);
                    if (R::LOSSY) a = __ldg(CA + g);
                } else {
                    ex[i] = ey[i] = ez[i] = hx[i] = hy[i] = hz[i] = 0.f;
                }
                put_ce(ring(zr0, i == NR - 1 && R::LOSSY ? 0 : i + 1), lane, c);
                if (R::LOSSY) CAs[(w * CRM + ring(zr0, i == NR - 1 ? 0 : i + 1)) * CP + lane] = a;
            }
        }

        // may a point source lie in the box during this tile's steps?  (per
        // axis, the box holds coordinate c at steps A - c .. A - c + n - 1)
        bool tile_src = false;
        for (int q = 0; q < P.src.n; ++q) {
            const SrcDesc &s = P.src.s[q];
            const int lo = max(max(iv.s, Ax - s.i), max(Ay - s.j, Az - s.k));
            const int hi = min(min(iv.e, Ax - s.i + TX - 1), min(Ay - s.j + TY - 1, Az - s.k + TZ - 1));
            tile_src |= lo <= hi;
        }
        // A. publish E^t (old) rows for the warp below's H half-step, and arrive at
        //    the barrier before it
        auto publish_e = [&]() {
            if constexpr (R::VX) {
                float *const qx = XEx + xe_at(w, 0, lane), *const qz = XEz + xe_at(w, 0, lane);
#pragma unroll
                for (int i = 0; i < NZ; i += 4) {
                    *reinterpret_cast<float4 *>(qx + i) = make_float4(ex[i], ex[i + 1], ex[i + 2], ex[i + 3]);
                    *reinterpret_cast<float4 *>(qz + i) = make_float4(ez[i], ez[i + 1], ez[i + 2], ez[i + 3]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < NZ; ++i) {
                    XEx[xe_at(w, i, lane)] = ex[i];
                    XEz[xe_at(w, i, lane)] = ez[i];
                }
            }
            half_arrive(&s_half[0]);
        };
        publish_e();
        for (int t = iv.s;; ++t, zl = R::LOSSY ? (zl == 0 ? CR - 1 : zl - 1) : 0) {
            // (x pairs: one pass more than steps, for the last slot's signal)
            const int bx = Ax - t, by = Ay - t, bz = Az - t;  // box low corner at step t
            const int zr = R::LOSSY ? zl : bz - 1;
            const int cur = t & 1;
            const char *const sb = stg0 + (size_t)cur * R::STG_B;
            const char *const cb = cof0 + (R::LOSSY ? 0 : (size_t)cur * R::COF_B);
            const T *const ZST = reinterpret_cast<const T *>(sb);
            const T *const YST = reinterpret_cast<const T *>(sb + R::OFF_Y);
            const T *const XST = reinterpret_cast<const T *>(sb + R::OFF_X);
            const float *const ZSC = reinterpret_cast<const float *>(cb), *const ZSA = ZSC + R::ZBC;
            const float *const YSC = reinterpret_cast<const float *>(cb + R::OFF_YC), *const YSA = YSC + R::YBC;
            const float *const XSC = reinterpret_cast<const float *>(cb + R::OFF_XC), *const XSA = XSC + R::XBC;
            const int dx = (lane - bx) & 31, dy = (w - by) & (R::RY - 1);
            const int px = bx + dx, py = by + dy;
            const bool xbox = dx < TX, ybox = dy < TY;
            // a row of cells outside the domain in y stays as it is (E = 0, and its H is
            // read by nobody): its warp skips the half-steps until it becomes the
            // y shell, and leaves its share of the issue slots to the others (FP32
            // 256^3 213.2 -> 216.9 GCUPS, 512^3 228.3 -> 230.5, FP16 256^3 203.0 ->
            // 205.7, 128^3 155.3 -> 158.3).  The same for groups of four z rows
            // cost more, in branches and spills, than it saved (209.0, FP16 173.2).
            const bool act = ybox && (unsigned)py < (unsigned)P.ny;
            const bool colin = xbox && ybox && (unsigned)px < (unsigned)P.nx && (unsigned)py < (unsigned)P.ny;
            const int ey_w = (by - 1) & (R::RY - 1);  // warp holding the y shell this step
            const long long col = px + (long long)P.pitch * py;
            // the box touches a low wall, whose tangential E is left alone.  (No
            // other masks: cells outside the domain have dt/eps (and c_a) 0, as the
            // coefficient shells are zero-filled there, so their E stays 0; their H
            // is only read by such cells and by that tangential E; and the x-shell
            // lane computes values that its refill overwrites.)
            const bool walls = bx < 1 || by < 1 || bz < 1;
            // physical x of this lane's column after the refills (the x-shell
            // lane moves to bx - 1)
            const int xw = (bx - 1) + ((lane - bx + 1) & 31);

            if (!half_wait(P, &s_half[0], n_half & 1u, &s_abort, ticket)) s_abort = 1;  // B1
            // (a wait of the step before may have run out: every warp sees it here)
            if (s_abort) { abort = true; break; }
            ++n_half;
            if (tid == 0) st_rel_cta(&s_steps, n_half);
            // x pairs: this step's x face travels through ring slot `slot`
            const bool msg = R::CL == 2 && t >= m_lo && t <= m_hi;
            const bool rx_msg = msg && rank == 1, tx_msg = msg && rank == 0;
            const int mi = msg_base + (t - m_lo);
            const int slot = mi % R::NSLOT;
            if constexpr (R::CL == 2) {
                // every lane is past last step's ring accesses: rank 0's x
                // lanes have written the slot (the release covers their stores),
                // rank 1's x lane has read it; the y-shell warp, idle in the H
                // half-step, tells the partner
                if (sig_slot >= 0) {
                    if (w == ((by - 1) & (R::RY - 1)) && lane == 0)
                        arrive_remote((rank == 0 ? rxf_remote : rxe_remote) + 8u * (unsigned)sig_slot);
                    sig_slot = -1;
                }
            }
            if (R::CL == 2 && t > iv.e) break;
            // x start of the staged z shell (rounded down to 16 bytes)
            const int x0 = (bx - 1) & ~(XA - 1), x0c = (bx - 1) & ~(R::XAC - 1);

            // C. H half-step, top-down in place: H[i] <- H[i-1] - dt curl_f(E[i-1], E[i], ...)
            if (act) {
                const int wn = (w + 1) & (R::RY - 1);
                const int src = (lane + 1) & 31;
                // rows in pairs (i, i-1), both computed from the old values
                // before either is written, so 16-bit storage rounds two new
                // values with one packed conversion
                const float *const qx = XEx + xe_at(wn, 0, lane), *const qz = XEz + xe_at(wn, 0, lane);
                float *const hxo = XHx + xe_at(w, 0, lane), *const hzo = XHz + xe_at(w, 0, lane);
                {
                    float4 gx, gz;  // VX: the y+1 neighbour's E rows 4q .. 4q+3
#pragma unroll
                    for (int i = NR - 1; i >= 2; i -= 2) {
                        if (R::VX && i % 4 == 0) {  // rows i-4 .. i-1
                            gx = *reinterpret_cast<const float4 *>(qx + i - 4);
                            gz = *reinterpret_cast<const float4 *>(qz + i - 4);
                        }
                        float nh[2][3];
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const int r = i - k;
                            const float ez_xp = shfl_from(ez[r - 1], src);
                            const float ey_xp = shfl_from(ey[r - 1], src);
                            const int m = (r - 1) & 3;
                            const float ez_yp = !R::VX ? qz[(r - 1) * 32]
                                                : m == 0 ? gz.x : m == 1 ? gz.y : m == 2 ? gz.z : gz.w;
                            const float ex_yp = !R::VX ? qx[(r - 1) * 32]
                                                : m == 0 ? gx.x : m == 1 ? gx.y : m == 2 ? gx.z : gx.w;
                            nh[k][0] = h_x(hx[r - 1], ez_yp, ez[r - 1], ey[r], ey[r - 1], ndt);
                            nh[k][1] = h_y(hy[r - 1], ex[r], ex[r - 1], ez_xp, ez[r - 1], ndt);
                            nh[k][2] = h_z(hz[r - 1], ey_xp, ey[r - 1], ex_yp, ex[r - 1], ndt);
                        }
                        RND2(nh[0][0], nh[1][0], 3);
                        RND2(nh[0][1], nh[1][1], 4);
                        RND2(nh[0][2], nh[1][2], 5);
                        hx[i] = nh[0][0]; hy[i] = nh[0][1]; hz[i] = nh[0][2];
                        hx[i - 1] = nh[1][0]; hy[i - 1] = nh[1][1]; hz[i - 1] = nh[1][2];
                        // published for the warp above's E half-step as they come (the
                        // last readers are behind B1; the x-shell lane's are not used)
                        if (!R::VX) {
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                hxo[(i - k - 1) * 32] = hx[i - k];
                                hzo[(i - k - 1) * 32] = hz[i - k];
                            }
                        } else if ((i - 2) % 4 == 0) {
                            *reinterpret_cast<float4 *>(hxo + i - 2) = make_float4(hx[i - 1], hx[i], hx[i + 1], hx[i + 2]);
                            *reinterpret_cast<float4 *>(hzo + i - 2) = make_float4(hz[i - 1], hz[i], hz[i + 1], hz[i + 2]);
                        }
                    }
                }
                half_arrive(&s_half[1]);
            }
            // every thread waits on the staging barrier itself: its completion
            // makes the copied shells visible to that thread, so no block
            // barrier is needed here (a timeout is noticed after B2)
            {
                if (!wait_stage(P, &s_bar[cur], (fills >> cur) & 1u, &s_quit, ticket)) s_abort = 1;
                fills ^= 1u << cur;
                if (R::LOSSY) {
                    if (!wait_stage(P, &s_bar[2], (fills >> 2) & 1u, &s_quit, ticket)) s_abort = 1;
                    fills ^= 4u;
                }
            }

            // D. refills from the staged shells, then publish new H rows for the
            //    warp above's E half-step
            const int xec = (bx - 1) - x0c;  // x offset of the coefficient shell column in its chunk
            if (w == ey_w) {  // the y shell warp takes its whole column set (level t)
                // row 0 from the lower z shell (its row y = by - 1); rows
                // 1..NZ from the y-face shell (x = bx .. bx+30) or, in the
                // corner lane (x = bx - 1), from the x-face shell's row by - 1
                const int xl = xw - x0, xlc = xw - x0c;
                ex[0] = S::dec(ZST[0 * R::ZB + xl], SC(0));
                ey[0] = S::dec(ZST[1 * R::ZB + xl], SC(1));
                ez[0] = S::dec(ZST[2 * R::ZB + xl], SC(2));
                hx[0] = S::dec(ZST[3 * R::ZB + xl], SC(3));
                hy[0] = S::dec(ZST[4 * R::ZB + xl], SC(4));
                hz[0] = S::dec(ZST[5 * R::ZB + xl], SC(5));
                const bool corner = xw == bx - 1;
                const T *src = corner ? XST : YST + (xw - bx) * BZ;
                const int fst = corner ? R::XB : R::YB;
                ld_rows<S>(src, SC(0), ex);
                ld_rows<S>(src + fst, SC(1), ey);
                ld_rows<S>(src + 2 * fst, SC(2), ez);
                ld_rows<S>(src + 3 * fst, SC(3), hx);
                ld_rows<S>(src + 4 * fst, SC(4), hy);
                ld_rows<S>(src + 5 * fst, SC(5), hz);
#pragma unroll
                for (int i = 0; i < NR; ++i) {
                    put_ce(ring(zr, i), lane, YSC[i * SWC + xlc]);
                    if (R::LOSSY) CAs[(w * CRM + ring(zr, i)) * CP + lane] = YSA[i * SWC + xlc];
                }
            } else if (!act) {  // outside the domain, or the previous top y row (two outside slots): kept
            } else {  // every lane's row -1 takes the lower z shell's H and coefficient
                const int o = (dy + 1) * SW + (xw - x0), oc = (dy + 1) * SWC + (xw - x0c);
                hx[0] = S::dec(ZST[3 * R::ZB + o], SC(3));
                hy[0] = S::dec(ZST[4 * R::ZB + o], SC(4));
                hz[0] = S::dec(ZST[5 * R::ZB + o], SC(5));
                put_ce(ring(zr, 0), lane, ZSC[oc]);
                if (R::LOSSY) CAs[(w * CRM + ring(zr, 0)) * CP + lane] = ZSA[oc];
                // the x-shell lane's coefficients, rows 1..NZ: a row a lane
                if (lane >= 1 && lane < NR) {
                    const int o = (w * CRM + ring(zr, lane)) * CP + ((bx - 1) & 31);
                    put_ce(ring(zr, lane), (bx - 1) & 31, XSC[(lane * 16 + dy) * R::XAC + xec]);
                    if (R::LOSSY) CAs[o] = XSA[(lane * 16 + dy) * R::XAC + xec];
                }
                if (!xbox) {  // the lane leaving the tile in x: rows 1..NZ of H from the x-face shell
                    // (x pairs: from the ring, once the upwind CTA's lanes have arrived)
                    const T *xs = XST + (dy + 1) * BZ;
                    int xst = R::XB;
                    if (R::CL == 2 && rx_msg) {
                        if (!wait_cluster_bar(P, &s_rxf[slot], (unsigned)(mi / R::NSLOT) & 1u, ticket)) s_abort = 1;
                        xs = RX + slot * R::RXS + dy * BZ;
                        xst = 16 * BZ;
                    }
                    ld_rows<S>(xs + 3 * xst, SC(3), hx);
                    ld_rows<S>(xs + 4 * xst, SC(4), hy);
                    ld_rows<S>(xs + 5 * xst, SC(5), hz);
                }
            }
            if (!ybox) {  // the y-shell warp's H rows
#pragma unroll
                for (int i = 1; i < NR; ++i) {
                    XHx[xe_at(w, i - 1, lane)] = hx[i];
                    XHz[xe_at(w, i - 1, lane)] = hz[i];
                }
            }
            if (!act) half_arrive(&s_half[1]);
            if (R::LOSSY) half_arrive(&s_half[2]);  // the coefficients are read
            if (!half_wait(P, &s_half[1], (n_half - 1u) & 1u, &s_abort, ticket)) {  // B2
                s_abort = 1;
                abort = true;
                break;
            }

            // does this thread own a point source this step?  (16-bit storage:
            // its E rows are rounded after the source is added, not before)
            const long long step = P.step0 + t;
            bool srcthr = false;
            if (S::narrow && tile_src) {
                for (int q = 0; q < P.src.n; ++q) {
                    const SrcDesc &s = P.src.s[q];
                    srcthr |= step < s.n_amp && s.i >= bx && s.i < bx + TX && s.j >= by && s.j < by + TY &&
                              s.k >= bz && s.k < bz + TZ && lane == (s.i & 31) && w == (s.j & (R::RY - 1));
                }
                srcthr = __any_sync(0xffffffffu, srcthr);  // its whole warp rounds late (shuffles in the E half-step)
            }

            if (act) {
                // F. E half-step, top-down in place: E[i] <- E[i-1] + ce curl_b(H[i], H[i-1], ...)
                const int wm = (w - 1) & (R::RY - 1);
                const int src = (lane - 1) & 31;
                const bool ux = py > 0, uy = px > 0, uz = px > 0 && py > 0;
                const float *const qx = XHx + xe_at(wm, 0, lane), *const qz = XHz + xe_at(wm, 0, lane);
                const float *const ceb = CEs + (w * CRM + ring(zr, 1)) * CP + lane;
                auto e_pass = [&](auto round, auto masked) {
                    float4 gx, gz;  // VX: the y-1 neighbour's new H rows 4q .. 4q+3
#pragma unroll
                    for (int i = NR - 1; i >= 2; i -= 2) {
                        if (R::VX && i % 4 == 0) {  // rows i-4 .. i-1
                            gx = *reinterpret_cast<const float4 *>(qx + i - 4);
                            gz = *reinterpret_cast<const float4 *>(qz + i - 4);
                        }
                        float ne[2][3];
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const int r = i - k;
                            const float hz_xm = shfl_from(hz[r], src);
                            const float hy_xm = shfl_from(hy[r], src);
                            const int m = (r - 1) & 3;
                            const float hx_ym = !R::VX ? qx[(r - 1) * 32]
                                                : m == 0 ? gx.x : m == 1 ? gx.y : m == 2 ? gx.z : gx.w;
                            const float hz_ym = !R::VX ? qz[(r - 1) * 32]
                                                : m == 0 ? gz.x : m == 1 ? gz.y : m == 2 ? gz.z : gz.w;
                            const float c = R::MIR ? ceb[(r - 1) * CP] : CEs[(w * CRM + ring(zr, r)) * CP + lane];
                            const float a = R::LOSSY ? CAs[(w * CRM + ring(zr, r)) * CP + lane] : 1.f;
                            ne[k][0] = e_x(decay<R::LOSSY>(a, ex[r - 1]), hz[r], hz_ym, hy[r], hy[r - 1], c);
                            ne[k][1] = e_y(decay<R::LOSSY>(a, ey[r - 1]), hx[r], hx[r - 1], hz[r], hz_xm, c);
                            ne[k][2] = e_z(decay<R::LOSSY>(a, ez[r - 1]), hy[r], hy_xm, hx[r], hx_ym, c);
                        }
                        if (decltype(round)::value) {
                            RND2(ne[0][0], ne[1][0], 0);
                            RND2(ne[0][1], ne[1][1], 1);
                            RND2(ne[0][2], ne[1][2], 2);
                        }
                        float o[2][3];
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const int r = i - k;
                            if (decltype(masked)::value) {
                                const bool kz = bz + r - 1 > 0;
                                o[k][0] = (ux && kz) ? ne[k][0] : ex[r - 1];
                                o[k][1] = (uy && kz) ? ne[k][1] : ey[r - 1];
                                o[k][2] = uz ? ne[k][2] : ez[r - 1];
                            } else {
                                o[k][0] = ne[k][0];
                                o[k][1] = ne[k][1];
                                o[k][2] = ne[k][2];
                            }
                        }
                        ex[i] = o[0][0]; ey[i] = o[0][1]; ez[i] = o[0][2];
                        ex[i - 1] = o[1][0]; ey[i - 1] = o[1][1]; ez[i - 1] = o[1][2];
                    }
                };
                // 16-bit storage rounds each new E value here, except in the (rare)
                // warp that adds a point source this step: it rounds after the
                // source, below
                if (S::narrow && srcthr)
                    e_pass(std::false_type(), std::true_type());
                else if (walls)
                    e_pass(std::bool_constant<S::narrow>(), std::true_type());
                else
                    e_pass(std::bool_constant<S::narrow>(), std::false_type());
                {  // every lane's row -1 takes the lower z shell's E (level t)
                    const int o = (dy + 1) * SW + (xw - x0);
                    ex[0] = S::dec(ZST[0 * R::ZB + o], SC(0));
                    ey[0] = S::dec(ZST[1 * R::ZB + o], SC(1));
                    ez[0] = S::dec(ZST[2 * R::ZB + o], SC(2));
                }
                if (!xbox) {  // the x lane: rows 1..NZ of E from the x-face shell (or the ring)
                    const bool ring = R::CL == 2 && rx_msg;
                    const T *xs = ring ? RX + slot * R::RXS + dy * BZ : XST + (dy + 1) * BZ;
                    const int xst = ring ? 16 * BZ : R::XB;
                    ld_rows<S>(xs, SC(0), ex);
                    ld_rows<S>(xs + xst, SC(1), ey);
                    ld_rows<S>(xs + 2 * xst, SC(2), ez);
                }
            }

            // point sources inside the box: the owning thread adds them
            for (int q = 0; tile_src && q < P.src.n; ++q) {
                const SrcDesc &s = P.src.s[q];
                if (step < s.n_amp && s.i >= bx && s.i < bx + TX && s.j >= by && s.j < by + TY &&
                    s.k >= bz && s.k < bz + TZ && lane == (s.i & 31) && w == (s.j & (R::RY - 1))) {
                    const float a = S::src_amp(s.amp[step], P.sc.src);
                    // added to the whole column, with -0 (which changes no value) in
                    // the other rows: a select and an add a row is less code than
                    // finding the row
                    const int ri = s.k - bz + 1;
                    auto add = [&](float (&e)[NR]) {
#pragma unroll
                        for (int i = 1; i < NR; ++i) e[i] = add_source(e[i], i == ri ? a : -0.f);
                    };
                    if (s.comp == 0) add(ex);
                    else if (s.comp == 1) add(ey);
                    else add(ez);
                }
            }
            if (S::narrow && srcthr) {  // one rounding per value, as the naive schedule stores it
#pragma unroll
                for (int i = 1; i < NR; i += 2) {
                    RND2(ex[i], ex[i + 1], 0);
                    RND2(ey[i], ey[i + 1], 1);
                    RND2(ez[i], ez[i + 1], 2);
                }
            }

            // what the warp below waits for first, then this warp's stores (x pairs:
            // last, the stores into the partner's ring are signalled after B1)
            if (R::CL == 1 && t < iv.e) publish_e();
            // the adjoint's recompute: this step's E of the cells of the
            // capture box (tiles that meet it only)
            if (R::CAP && colin && bx < P.cap_hi[0] && bx + TX > P.cap_lo[0] && by < P.cap_hi[1] &&
                by + TY > P.cap_lo[1] && bz < P.cap_hi[2] && bz + TZ > P.cap_lo[2] && px >= P.cap_lo[0] &&
                px < P.cap_hi[0] && py >= P.cap_lo[1] && py < P.cap_hi[1]) {
                float *cp = P.cap + 3 * P.cap_bc * (long long)t;
                const int cbx = P.cap_hi[0] - P.cap_lo[0], cby = P.cap_hi[1] - P.cap_lo[1];
                const long long cxy = (long long)(px - P.cap_lo[0]) + (long long)cbx * (py - P.cap_lo[1]);
#pragma unroll
                for (int i = 1; i < NR; ++i) {
                    const int z = bz + i - 1;
                    if (z >= P.cap_lo[2] && z < P.cap_hi[2]) {
                        const long long b = cxy + (long long)cbx * cby * (z - P.cap_lo[2]);
                        cp[b] = ex[i];
                        cp[P.cap_bc + b] = ey[i];
                        cp[2 * P.cap_bc + b] = ez[i];
                    }
                }
            }
            // G. the top faces (of the launch's last step too, which is stored whole
            // below: the downwind tiles need not wait for that).  The top y face: its
            // warp, which is idle in the next H half-step, has the most to store.
            // Last, or with 16-bit storage first (FP32 256^3 213.4 and 211.8 GCUPS,
            // FP16 201.3 and 203.1)
            auto y_face = [&]() {
                if (colin && dy == TY - 1) FACE_STORE(YFk + ((long long)py * P.nx + px) * BZ, P.fys);
            };
            if (S::narrow) y_face();
            if (colin && (unsigned)(bz + NR - 2) < (unsigned)P.nz) {  // top z face
                const long long g = col + sxy * (bz + NR - 2);
                STORE6(g, NR - 1);
            }
            // top x face (all rows of the lane leaving the box in x) into the
            // x-face buffer, where the downwind tile's x shell is fetched.
            // x pairs, rank 0: into rank 1's ring instead (its slot was freed
            // before the second barrier), every box row's lane then arriving
            // on the slot's barrier; the top box row still goes to the x-face
            // buffer too (the corner of the next pair's y shell)
            if (ybox && dx == TX - 1) {
                if (R::CL == 2 && tx_msg) {
                    // the slot's previous message must have been read
                    if (mi >= R::NSLOT &&
                        !wait_cluster_bar(P, &s_rxe[slot], (unsigned)((mi / R::NSLOT) - 1) & 1u, ticket))
                        s_abort = 1;
                    const unsigned a = rx_remote + (unsigned)((slot * R::RXS + dy * BZ) * (int)sizeof(T));
                    constexpr unsigned FS = 16u * BZ * (unsigned)sizeof(T);
                    st_rows_remote<S>(a, IS(0), ex);
                    st_rows_remote<S>(a + FS, IS(1), ey);
                    st_rows_remote<S>(a + 2 * FS, IS(2), ez);
                    st_rows_remote<S>(a + 3 * FS, IS(3), hx);
                    st_rows_remote<S>(a + 4 * FS, IS(4), hy);
                    st_rows_remote<S>(a + 5 * FS, IS(5), hz);
                }
                if ((!(R::CL == 2 && tx_msg) || dy == TY - 1) && (unsigned)px < (unsigned)P.nx &&
                    (unsigned)py < (unsigned)P.ny)
                    FACE_STORE(XFk + ((long long)px * P.ny + py) * BZ, P.fxs);
            }
            if (!S::narrow) y_face();
            // this warp's faces of level t are stored
            half_arrive(&s_fin[n_fin & 3u]);
            ++n_fin;
            if (R::CL == 2) publish_e();
            if (R::CL == 2 && msg) sig_slot = slot;
            if (R::CL == 1 && t == iv.e) break;
        }
        if (abort || *(volatile int *)&s_abort != 0) break;
        if (iv.e == P.T - 1) {  // the launch's last step: the whole box
            const int bx = Ax - iv.e, by = Ay - iv.e, bz = Az - iv.e;
            const int dx = (lane - bx) & 31, dy = (w - by) & (R::RY - 1);
            const int px = bx + dx, py = by + dy;
            if (dx < TX && dy < TY && (unsigned)px < (unsigned)P.nx && (unsigned)py < (unsigned)P.ny) {
                const long long col = px + (long long)P.pitch * py;
#pragma unroll
                for (int i = 1; i < NR; ++i)
                    if ((unsigned)(bz + i - 1) < (unsigned)P.nz) {
                        const long long g = col + sxy * (bz + i - 1);
                        STORE6(g, i);
                    }
            }
        }
        if constexpr (R::CL == 2) {  // B2's phase of the pass more
            half_arrive(&s_half[1]);
            if (!half_wait(P, &s_half[1], (n_half - 1u) & 1u, &s_abort, ticket)) {
                s_abort = 1;
                break;
            }
        }
        } while (false);
        msg_base += nmsg;
        sig_slot = -1;
        // (after an abort the CTA, or a pair together, leaves at the next ticket)
    }
    // x pairs: neither CTA leaves while its partner may still write into its
    // shared memory
    if constexpr (R::CL == 2) cluster_sync_all();
}

#undef F0
#undef F1
#undef F2
#undef F3
#undef F4
#undef F5
#undef CE
#undef CA
#undef SC
#undef IS
#undef RND
#undef RND2
#undef STORE6
#undef FACE_STORE

// 31 x 15 x 12 and 31 x 15 x 8 tiles, each for every kernel format and in the
// lossy (absorber) form
// the box leaves one y slot of the ring outside (TY = 15): as fast as two
// outside slots (TY = 14) and updates more cells per step
constexpr int REG_TY = 15;
template <int NZ>
struct RegShape {
    static constexpr bool HAS_PAIRS = NZ == 12;  // x pairs in thread-block clusters: the 31 x 15 x 12 tile
    static cudaError_t configure(int fmt, bool lossy, int cl)
    {
        if (lossy) {
            if (cl == 1) DISPATCH_FORMAT(fmt, S, set<RegTile<NZ, S, true, REG_TY>>());
            return cudaErrorInvalidValue;
        }
        if (cl == 2) {
            if constexpr (HAS_PAIRS) {
                if (fmt == FDTD_STORAGE_F32) {  // and its capturing form, for the adjoint
                    const cudaError_t e = set<RegTile<NZ, StoreF32, false, REG_TY, 2, true>>();
                    if (e != cudaSuccess) return e;
                }
                DISPATCH_FORMAT(fmt, S, set<RegTile<NZ, S, false, REG_TY, 2>>());
            }
            return cudaErrorInvalidValue;
        }
        if (fmt == FDTD_STORAGE_F32) {  // and its capturing form
            const cudaError_t e = set<RegTile<NZ, StoreF32, false, REG_TY, 1, true>>();
            if (e != cudaSuccess) return e;
        }
        DISPATCH_FORMAT(fmt, S, set<RegTile<NZ, S, false, REG_TY>>());
    }
    static int per_sm(int fmt, bool lossy)
    {
        if (lossy) {
            DISPATCH_FORMAT(fmt, S, occ<RegTile<NZ, S, true, REG_TY>>());
        }
        DISPATCH_FORMAT(fmt, S, occ<RegTile<NZ, S, false, REG_TY>>());
    }
    static int clusters(int fmt)
    {
        if constexpr (HAS_PAIRS) DISPATCH_FORMAT(fmt, S, occ_pairs<RegTile<NZ, S, false, REG_TY, 2>>());
        return 0;
    }
    static cudaError_t launch(const SysLaunch &p, int grid, cudaStream_t st, int fmt, int cl)
    {
        if (p.cap) {  // the capturing forms: lossless FP32 (a launch with no such form stores nothing there: an error)
            if (p.ca || fmt != FDTD_STORAGE_F32) return cudaErrorInvalidValue;
            if (cl == 1) return go<RegTile<NZ, StoreF32, false, REG_TY, 1, true>>(p, grid, st);
            if constexpr (HAS_PAIRS) return go<RegTile<NZ, StoreF32, false, REG_TY, 2, true>>(p, grid, st);
            return cudaErrorInvalidValue;
        }
        if (p.ca) {
            if (cl == 1) DISPATCH_FORMAT(fmt, S, go<RegTile<NZ, S, true, REG_TY>>(p, grid, st));
            return cudaErrorInvalidValue;
        }
        if (cl == 2) {
            if constexpr (HAS_PAIRS) DISPATCH_FORMAT(fmt, S, go<RegTile<NZ, S, false, REG_TY, 2>>(p, grid, st));
            return cudaErrorInvalidValue;
        }
        DISPATCH_FORMAT(fmt, S, go<RegTile<NZ, S, false, REG_TY>>(p, grid, st));
    }
    template <class R>
    static cudaError_t set()
    {
        return cudaFuncSetAttribute(systolic_reg_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)R::smem_bytes());
    }
    template <class R>
    static int occ()
    {
        int n = 0;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, systolic_reg_kernel<R>, R::NT, R::smem_bytes()) ==
                       cudaSuccess
                   ? n
                   : 0;
    }
    template <class R>
    static cudaLaunchConfig_t config(int grid, cudaStream_t st, cudaLaunchAttribute *at)
    {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3((unsigned)R::NT);
        cfg.dynamicSmemBytes = R::smem_bytes();
        cfg.stream = st;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)R::CL;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cfg;
    }
    // co-resident clusters of a pair kernel on this device
    template <class R>
    static int occ_pairs()
    {
        cudaLaunchAttribute at[1];
        cudaLaunchConfig_t cfg = config<R>(2, 0, at);
        int n = 0;
        return cudaOccupancyMaxActiveClusters(&n, systolic_reg_kernel<R>, &cfg) == cudaSuccess ? n : 0;
    }
    template <class R>
    static cudaError_t go(const SysLaunch &p, int grid, cudaStream_t st)
    {
        if constexpr (R::CL == 1) {
            systolic_reg_kernel<R><<<grid, R::NT, R::smem_bytes(), st>>>(p);
            return cudaGetLastError();
        } else {
            cudaLaunchAttribute at[1];
            cudaLaunchConfig_t cfg = config<R>(grid, st, at);
            return cudaLaunchKernelEx(&cfg, systolic_reg_kernel<R>, p);
        }
    }
};

using RegA = RegShape<12>;  // 31 x 15 x 12
using RegB = RegShape<8>;   // 31 x 15 x 8

} // namespace

int systolic_reg_rows(int k) { return (k == 0 ? 12 : 8) + 1; }

SysShape systolic_reg_shape(int k) { return SysShape{31, REG_TY, k == 0 ? 12 : 8}; }

cudaError_t systolic_reg_configure(int k, int fmt, bool lossy, int cl)
{
    return k == 0 ? RegA::configure(fmt, lossy, cl) : RegB::configure(fmt, lossy, cl);
}

int systolic_reg_max_ctas_per_sm(int k, int fmt, bool lossy)
{
    return k == 0 ? RegA::per_sm(fmt, lossy) : RegB::per_sm(fmt, lossy);
}

int systolic_reg_max_pairs(int k, int fmt) { return k == 0 ? RegA::clusters(fmt) : RegB::clusters(fmt); }

cudaError_t launch_systolic_reg(const SysLaunch &p, int grid, cudaStream_t st, int k, int fmt, int cl)
{
    return k == 0 ? RegA::launch(p, grid, st, fmt, cl) : RegB::launch(p, grid, st, fmt, cl);
}
