// Fused single-read path (steps A1-A3): one thread-block cluster walks one draft chain (b,k), one
// CTA of 32 warps per SM, the row resident in TENSOR MEMORY between the two sweeps.
//
// For every position i = 0..gamma-1 of the chain the cluster
//   * streams the target row and the draft row from HBM exactly once.  CTA r of the cluster owns a contiguous slice of the
//     vocabulary, each of its warps one to four 256-entry cells of it.  Every warp runs its own little ring of asynchronous copies
//     (one cell of both tensors per slot): the warp that consumes a slot refills it itself, so the load path needs no block-wide
//     synchronisation and runs ahead across rows and chains;
//   * first sweep: a thread takes 8 (target, draft) pairs of a cell, turns them into exponentials relative to its warp's reference
//     and parks them in tensor memory (tcgen05.st; each warp owns 64 of the 512 columns of its lane quarter, 256 KB per SM in all =
//     32,768 pairs) or, every fifth cell, in shared memory; only their sum stays in registers;
//   * exchanges (reference, sum-exp) partials in two levels: the warps of a CTA leave theirs in shared memory, and the last warp,
//     which has no cells unless there are more than the others can hold, combines them and PUSHES one partial per CTA into
//     every CTA's shared memory with asynchronous distributed-shared-memory stores that complete on the receiver's
//     mbarrier.  The other warps meanwhile sweep the row before for the last time and the row behind for the first;
//   * second sweep: reads the exponentials back and writes one partial sum of the coupling terms per cell.  Shared memory holds
//     a copied cell once and the registers no row data between the sweeps, which is what lets 32 warps share the SM.
// The joint likelihood ratio c_i = p(x^i)/q(x^i) is carried as a running product by the last warp, which works c_{i+1} out
// right after the release of row i.  The finishing kernel (weights, scan, extra token) consumes the cell sums.
//
// What bounds it: the special-function unit (3.1 of its instructions per pair, 63 % of its rate at 16 x 8 x 8 x 151936 float32) and
// the exchange, during which most of the SM waits; up to there float32 rows, HBM.  Whole calls one after the other, us, with references
// per thread and cell / per warp (one B200): 64 x 8 x 8 x 151936 float32 1140 / 951 (bursts of 140 calls, before the power limit counts:
// 820), 256 x 8 x 4 x 32000 float32 437 / 376, 32 x 4 x 5 x 128256 bfloat16 180 / 138, 256 x 1 x 4 x 32000 float32 80 / 68.  Warp
// instructions per 32 pairs 34.1 / 26.3 (16 x 8 x 8 x 151936 float32).
//
// Every wait on an mbarrier or on a word in global memory is bounded; on expiry the warp records
// an error flag and keeps executing the protocol, so a lost copy cannot hang the kernel, and the
// tensor memory is released on every path.
#include <float.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "sgbv_cluster.cuh"
#include "sgbv_common.cuh"

namespace sgbv {

namespace {

constexpr int kCell = kTile;               // 256 contiguous entries: the unit a warp works on
constexpr int kWarps = 32;                 // warps per CTA, one CTA per SM (16 warps of 128 registers, or two CTAs of 16, measured slower)
constexpr int kCtaThreads = kWarps * 32;
constexpr int kCtaCells = 128;             // cells of a row per CTA: 16 tensor-memory columns per cell in each of the 4
                                           // lane quarters, 512 columns per SM: 128 cells = 32,768 entries per SM
constexpr int kSlack = 16;  // extra bytes per cell and tensor in a slot when rows start anywhere: a copy then begins at the
                           // 16-byte boundary before the cell and ends behind it
constexpr int kParkBytes = kCell * 2 * (int)sizeof(float);  // the exponentials of one cell of both tensors, a warp's parked first cell
constexpr int kTmemCols = 512;             // all of the SM's tensor memory
constexpr int kMaxCluster = 8;  // CTAs per cluster (beyond 8 the size is not portable, which sm_100 allows)
constexpr long long kWaitLimitCycles = 2000000000ll;  // about one second of SM clock
constexpr uint32_t kPollNs = 100u;                    // sleep between two tests of a barrier that is not ready
static_assert(kTile == 256, "the fused path writes one partial sum per 256-element cell");

struct FusedParams {
    const void *zq;
    const void *zp;
    const int32_t *tok;
    Shape s;
    Workspace ws;
    int cluster;      // CTAs per cluster
    int slice_cells;  // cells of a row per CTA (at most kCtaCells)
    int nchains;      // B*K
    const double *carry_loga, *carry_logb;  // Algorithm 2: per-chain joint logs carried in (else NULL)
    int *error_flag;  // set to 1 if a bounded wait expired
    long long poll_limit;  // cycles a poll of a published ratio may take (row walk)
    int withhold;     // failure-detection test: the first row of every chain does not publish its ratio
    float rise;       // kRise in units of logits
    int aux_here;     // rows with c < 1 get their two extra sums in this kernel (else: the kernels that follow it)
};

// ---- PTX wrappers ------------------------------------------------------------------------------

// mbarrier operations take the barrier's 32-bit shared-memory address
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: sets `gave_up` if the phase did not complete within about a second.  Between tests the
// warp sleeps, so that a waiting warp leaves the issue slots to the working ones; the clock is read only
// every 64 tests.  A thread that has given up once only tests from then on, so that the time a failing
// kernel takes stays bounded.
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, uint32_t &gave_up) {
    if (mbar_test(bar, parity) || gave_up) return;
    uint32_t tests = 0;
    long long t0 = 0;
    for (;;) {
        __nanosleep(kPollNs);
        if (mbar_test(bar, parity)) return;
        if ((++tests & 63u) == 0u) {
            const long long t = clock64();
            if (t0 == 0) t0 = t;
            else if (t - t0 > kWaitLimitCycles) {
                gave_up = 1u;
                return;
            }
        }
    }
}
// One cell of both tensors into a ring slot (the draft part `half` bytes behind the target part): the lane
// with pred != 0 announces 2 x bytes on the slot's barrier and starts the two bulk copies.  Every lane
// executes the statement (no branch); the copies complete on the barrier.
__device__ __forceinline__ void issue_cell(uint32_t dst, const void *zq, const void *zp, uint32_t bytes, uint32_t bar,
                                           uint32_t pred, uint32_t half) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b32 d2, b2;\n\t"
        "setp.ne.u32 p, %5, 0;\n\t"
        "shl.b32 b2, %3, 1;\n\t"
        "add.u32 d2, %0, %6;\n\t"
        "@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%4], b2;\n\t"
        "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %3, [%4];\n\t"
        "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [d2], [%2], %3, [%4];\n\t}" ::"r"(dst),
        "l"(zq), "l"(zp), "r"(bytes), "r"(bar), "r"(pred), "r"(half)
        : "memory");
}
// Asynchronous store of 16 bytes into the shared memory of CTA `rank` of this cluster, at the
// address that `local` has in this CTA; its completion is counted (16 bytes) on the receiver's
// mbarrier that sits where `local_bar` sits here.
__device__ __forceinline__ void push_f4(void *local, uint32_t local_bar, uint32_t rank, float4 v) {
    uint32_t dst, bar;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(smem_u32(local)), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar) : "r"(local_bar), "r"(rank));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1,%2,%3,%4}, [%5];" ::"r"(dst),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
                 : "memory");
}
// This thread's asynchronous copies of 16 bytes, in groups that complete in order.
template <int kDst, int kSrc>
__device__ __forceinline__ void copy16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global.L2::128B [%0 + %2], [%1 + %3], 16;" ::"r"(dst), "l"(src), "n"(kDst), "n"(kSrc) : "memory");
}
__device__ __forceinline__ void copy_group_end() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// Waits until at most N of this thread's groups are under way.
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// ---- tensor memory --------------------------------------------------------------------------------
// One warp allocates all columns for the CTA (the address lands in shared memory), every warp then
// reads and writes only the lanes of its own quarter (warp index mod 4) and its own columns.
__device__ __forceinline__ void tmem_alloc(uint32_t *dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// 16 consecutive columns of this thread's lane: the 8 target and the 8 draft exponentials of a cell
__device__ __forceinline__ void tmem_st_cell(uint32_t taddr, const float2 (&a)[4], const float2 (&b)[4]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "f"(a[0].x), "f"(a[0].y), "f"(a[1].x), "f"(a[1].y), "f"(a[2].x), "f"(a[2].y), "f"(a[3].x), "f"(a[3].y), "f"(b[0].x),
        "f"(b[0].y), "f"(b[1].x), "f"(b[1].y), "f"(b[2].x), "f"(b[2].y), "f"(b[3].x), "f"(b[3].y)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_cell(uint32_t taddr, float2 (&a)[4], float2 (&b)[4]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=f"(a[0].x), "=f"(a[0].y), "=f"(a[1].x), "=f"(a[1].y), "=f"(a[2].x), "=f"(a[2].y), "=f"(a[3].x), "=f"(a[3].y),
          "=f"(b[0].x), "=f"(b[0].y), "=f"(b[1].x), "=f"(b[1].y), "=f"(b[2].x), "=f"(b[2].y), "=f"(b[3].x), "=f"(b[3].y)
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Waits for this thread's tensor-memory loads; the loaded registers pass through the statement, so that no
// use of them can be scheduled ahead of it.
__device__ __forceinline__ void tmem_wait_ld(float2 (&a)[4], float2 (&b)[4]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0].x), "+f"(a[0].y), "+f"(a[1].x), "+f"(a[1].y), "+f"(a[2].x), "+f"(a[2].y), "+f"(a[3].x), "+f"(a[3].y),
                   "+f"(b[0].x), "+f"(b[0].y), "+f"(b[1].x), "+f"(b[1].y), "+f"(b[2].x), "+f"(b[2].y), "+f"(b[3].x), "+f"(b[3].y)
                 :
                 : "memory");
}

// ---- shared memory layout ------------------------------------------------------------------------
// [rings: 32 warps x slots x (cell of zq, cell of zp)] [full barriers: 32 warps x slots] [Control]
struct Control {
    uint64_t xbar[2];                    // by row parity: "the partials of all CTAs of the cluster are here"
    // partials (reference of zq, sum eq, reference of zp, sum ep): of this CTA's warps, and, double-buffered by
    // row parity, of every CTA of the cluster (pushed by their owners)
    float4 wslots[kWarps];
    float4 slots[2][kMaxCluster];
    float4 low[2][kMaxCluster];          // what the sums in `slots` were rounded by (y, w)
    float4 rs;                           // the row's scalars for the second sweep: rq, rp, kappa, c
    uint32_t tmem_base;                  // address of the allocated tensor memory
};

// Named hardware barriers of the CTA (0 is the one of __syncthreads).
__device__ __forceinline__ void bar_sync(int id, int nthreads) {
    asm volatile("barrier.cta.sync.aligned %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int nthreads) {
    asm volatile("barrier.cta.arrive.aligned %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Reads this lane's 8 elements of one cell of one tensor from the ring.
template <typename T>
__device__ __forceinline__ void read_cell(const unsigned char *cell_base, int lane, float2 (&v)[4]);
template <>
__device__ __forceinline__ void read_cell<float>(const unsigned char *cell_base, int lane, float2 (&v)[4]) {
    const float4 *p = reinterpret_cast<const float4 *>(cell_base) + lane;
    const float4 a = p[0], b = p[32];
    v[0] = make_float2(a.x, a.y); v[1] = make_float2(a.z, a.w);
    v[2] = make_float2(b.x, b.y); v[3] = make_float2(b.z, b.w);
}
template <>
__device__ __forceinline__ void read_cell<uint16_t>(const unsigned char *cell_base, int lane, float2 (&v)[4]) {
    const uint4 a = reinterpret_cast<const uint4 *>(cell_base)[lane];
    v[0] = make_float2(__uint_as_float(a.x << 16), __uint_as_float(a.x & 0xffff0000u));
    v[1] = make_float2(__uint_as_float(a.y << 16), __uint_as_float(a.y & 0xffff0000u));
    v[2] = make_float2(__uint_as_float(a.z << 16), __uint_as_float(a.z & 0xffff0000u));
    v[3] = make_float2(__uint_as_float(a.w << 16), __uint_as_float(a.w & 0xffff0000u));
}
// The same from a slot whose cell begins at any multiple of the element size behind the slot's start: a lane takes every
// 32nd entry, so that the 32 lanes of a load read 32 neighbours.
template <typename T>
__device__ __forceinline__ void read_cell_at(const unsigned char *cell_base, int lane, float2 (&v)[4]) {
    const T *p = reinterpret_cast<const T *>(cell_base) + lane;
    auto at = [&](int e) {
        return sizeof(T) == 4 ? __uint_as_float((uint32_t)reinterpret_cast<const uint32_t *>(p)[32 * e]) : __uint_as_float((uint32_t)p[32 * e] << 16);
    };
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = make_float2(at(2 * e), at(2 * e + 1));
}
// Offset (in elements, within the 256-element cell) of this lane's e-th element.
template <typename T, bool kAny>
__device__ __forceinline__ int cell_offset(int lane, int e) {
    if (kAny) return lane + 32 * e;
    if (sizeof(T) == 4) return (e < 4) ? lane * 4 + e : 128 + lane * 4 + (e - 4);
    return lane * 8 + e;
}

// Maximum over the warp in one instruction (NaN inputs are passed over, as fmaxf does).
__device__ __forceinline__ float warp_max_redux(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
// Sums P values over the 32 lanes of a warp at once ("transposed" butterfly: at every step a lane
// hands half of its values to its partner and keeps the other half).  P is a power of two (<= 8).
// On return v[0] of lane l is the warp total of value number owner_index<P>(l).
template <int P>
__device__ __forceinline__ int owner_index(int lane) {
    int idx = 0;
    if (P >= 2) idx += (lane & 16) ? P / 2 : 0;
    if (P >= 4) idx += (lane & 8) ? P / 4 : 0;
    if (P >= 8) idx += (lane & 4) ? P / 8 : 0;
    return idx;
}
template <int P>
__device__ __forceinline__ void warp_sum_multi(float (&v)[P], int lane) {
    int off = 16;
#pragma unroll
    for (int n = P; n > 1; n >>= 1, off >>= 1) {
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int k = 0; k < n / 2; ++k) {
            const float keep = upper ? v[k + n / 2] : v[k];
            const float send = upper ? v[k] : v[k + n / 2];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
}

// Exponentials are relative to ONE logit per warp and tensor of a row, its reference: the maximum of the warp's first cell.  The
// warp's later cells may reach kRise above it, in units of log2; a logit beyond that becomes the reference from there on (the cells
// before it keep theirs, see FirstSweep::moved): a few warps per row.  So what carries most of a row's mass is a reference or
// within 2^kRise of one, the largest entry of a point-mass row maps to exactly 1, and every factor between units is the same for the
// whole warp.  References per thread and cell, as before, took three exponentials and some 25 instructions per cell.
constexpr float kRise = 6.0f;

// What the second sweep needs of a row, in units of this warp's references.
struct RowScalars {
    float Fq;     // moves sums to units of the row's reference
    float KF;     // kappa * Fp / Fq: c p(x)/q(x) = KF * ep/eq
    float kFp;    // kappa * Fp (rows with c < 1: where the warp's target share underflows)
    float c;      // c_i
};
// What a warp keeps of the row whose first sweep runs.
struct FirstSweep {
    float bq, bp;    // references (-FLT_MAX: no finite logit so far, and -inf against it still gives 0)
    float2 sq, sp;   // this thread's sums of exponentials
    int moved;       // 0, or the first cell whose references are not in shared memory: references have moved, and the cells before
                     // it keep theirs
};

// f(Int<0>()), ..., f(Int<N - 1>()), N <= 4: an unrolled loop whose index is a constant expression.
template <int I>
using Int = std::integral_constant<int, I>;
template <int N, typename F>
__device__ __forceinline__ void for_each_cell(F f) {
    f(Int<0>());
    if constexpr (N > 1) f(Int<1>());
    if constexpr (N > 2) f(Int<2>());
    if constexpr (N > 3) f(Int<3>());
    static_assert(N <= 4, "cells per warp");
}

__device__ __forceinline__ void cell_maxima(const float2 (&eq)[4], const float2 (&ep)[4], float &m1, float &m2) {
    m1 = m2 = -FLT_MAX;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        m1 = max3(m1, eq[e].x, eq[e].y);
        m2 = max3(m2, ep[e].x, ep[e].y);
    }
}
// First sweep of one cell, first half: the lane's 8 target and 8 draft logits from the ring slot (entries past the
// end of the row read as -inf), and their maxima.
template <typename T, bool kAny>
__device__ __forceinline__ void first_sweep_fetch(const unsigned char *slot, uint32_t off_q, uint32_t off_p, int lane, bool is_tail,
                                                  int tail_valid, float2 (&eq)[4], float2 (&ep)[4], float &m1, float &m2) {
    if (kAny) {
        read_cell_at<T>(slot + off_q, lane, eq);
        read_cell_at<T>(slot + kCell * (int)sizeof(T) + kSlack + off_p, lane, ep);
    } else {
        read_cell<T>(slot, lane, eq);
        read_cell<T>(slot + kCell * (int)sizeof(T), lane, ep);
    }
    if (is_tail) {  // the row ends inside this cell
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (cell_offset<T, kAny>(lane, 2 * e) >= tail_valid) eq[e].x = ep[e].x = -INFINITY;
            if (cell_offset<T, kAny>(lane, 2 * e + 1) >= tail_valid) eq[e].y = ep[e].y = -INFINITY;
        }
    }
    cell_maxima(eq, ep, m1, m2);
}
// A cell that no copy can bring (its 16-byte pieces reach past an end of a tensor): straight from global memory.
template <typename T>
__device__ __forceinline__ void first_sweep_direct(const unsigned char *q, const unsigned char *p, int lane, int valid,
                                                   float2 (&eq)[4], float2 (&ep)[4], float &m1, float &m2) {
    auto at = [&](const unsigned char *base, int e) {
        const int x = lane + 32 * e;
        return x < valid ? ld_logit(reinterpret_cast<const T *>(base), x) : -INFINITY;
    };
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        eq[e] = make_float2(at(q, 2 * e), at(q, 2 * e + 1));
        ep[e] = make_float2(at(p, 2 * e), at(p, 2 * e + 1));
    }
    cell_maxima(eq, ep, m1, m2);
}
// Before the exponentials of cell j: the warp's references.  m1, m2: this thread's maxima of the cell; refs: the warp's words in
// shared memory, one pair per cell.
__device__ __forceinline__ void set_references(FirstSweep &f, int j, float m1, float m2, float scale, float rise, float2 *refs) {
    if (j == 0) {
        f.bq = warp_max_redux(m1);
        f.bp = warp_max_redux(m2);
        return;
    }
    // (the difference is what the exponent takes; b + rise would be rounded to a multiple of b's ulp, which may be as much as rise)
    if (!__any_sync(0xffffffffu, m1 - f.bq > rise || m2 - f.bp > rise)) return;
    if ((threadIdx.x & 31) == 0)
        for (int i = f.moved; i < j; ++i) refs[i] = make_float2(f.bq, f.bp);
    f.moved = j;
    auto raise = [&](float m, float &b, float2 &sum) {
        m = warp_max_redux(m);
        if (!(m - b > rise)) return;
        const float move = ex2((b - m) * scale);
        sum.x *= move;
        sum.y *= move;
        b = m;
    };
    raise(m1, f.bq, f.sq);
    raise(m2, f.bp, f.sp);
}
// Second half: the exponentials into tensor memory, or into shared memory (parked), and their sums.
__device__ __forceinline__ void first_sweep_store(uint32_t taddr_cell, bool parked, float4 *park, float scale, float2 (&eq)[4], float2 (&ep)[4], FirstSweep &f) {
    const float2 nbq = splat(-f.bq), nbp = splat(-f.bp), sc2 = splat(scale);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 aq = __fmul2_rn(__fadd2_rn(eq[e], nbq), sc2);
        const float2 ap = __fmul2_rn(__fadd2_rn(ep[e], nbp), sc2);
        eq[e] = make_float2(ex2(aq.x), ex2(aq.y));
        ep[e] = make_float2(ex2(ap.x), ex2(ap.y));
        f.sq = __fadd2_rn(f.sq, eq[e]);
        f.sp = __fadd2_rn(f.sp, ep[e]);
    }
    if (parked) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            park[32 * e] = make_float4(eq[2 * e].x, eq[2 * e].y, eq[2 * e + 1].x, eq[2 * e + 1].y);
            park[32 * e + 64] = make_float4(ep[2 * e].x, ep[2 * e].y, ep[2 * e + 1].x, ep[2 * e + 1].y);
        }
    } else {
        tmem_st_cell(taddr_cell, eq, ep);
    }
}

// Second sweep of one cell, read back from tensor memory (or shared memory: parked), two vocabulary entries per instruction (f32x2).
// eq/ep are exponentials relative to the warp's references; with kt = KF c p(x)/q(x) = kt ep/eq.  Returns this thread's sums
//   w  = sum eq (1 - min{kt ep/eq, 1})^K                    (Eq. 4's weights, Eq. 2's sum)
//   sd = sum max(kt ep - eq, 0)                             (c < 1 only)
//   sm = sum eq (c - t)^2 Q(t)                              (c < 1 only)
// tiny: the warp's share of the target row underflows (or nearly so, which would overflow kt): its q is 0 in row units, its weights
// vanish, and max(c p - q, 0) = c p, in units of the draft (kAux; without the extra sums nothing needs doing: whatever kt is, the
// clamp below leaves a weight in [0, eq]).
template <int KT, bool kAux>
__device__ __forceinline__ void second_sweep_cell(uint32_t taddr_cell, bool parked, const float4 *park, float kt, float c, bool tiny, int K, float &w, float &sd_out,
                                                  float &sm_out) {
    float2 eq[4], ep[4];
    const float v1 = 1.0f - c;
    const float2 nv1 = splat(-v1);
    if (parked) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float4 a = park[32 * e], b = park[32 * e + 64];
            eq[2 * e] = make_float2(a.x, a.y);
            eq[2 * e + 1] = make_float2(a.z, a.w);
            ep[2 * e] = make_float2(b.x, b.y);
            ep[2 * e + 1] = make_float2(b.z, b.w);
        }
    } else {
        tmem_ld_cell(taddr_cell, eq, ep);
        tmem_wait_ld(eq, ep);
    }
    if (kAux) {
        if (tiny) {
#pragma unroll
            for (int e = 0; e < 4; ++e) eq[e] = splat(0.0f);
            kt = 1.0f;
        }
    }
    const float2 nkt = splat(-kt);
    float coef[KT > 2 ? KT - 2 : 1];  // Horner coefficients of Q, (t+1) (1-c)^t, t = 1..K-2
    if (kAux && KT > 2) {
        float vj = 1.0f;
#pragma unroll
        for (int t = 1; t <= KT - 2; ++t) {
            vj *= v1;
            coef[t - 1] = (float)(t + 1) * vj;
        }
    }
    float2 sw = splat(0.0f), sd = splat(0.0f), sm = splat(0.0f);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 q = eq[e];
        const float2 diff = __ffma2_rn(nkt, ep[e], q);  // q - c p, thread units
        if (KT == 1) {  // one draft: Q = 0, the second extra sum vanishes and nothing needs the ratio
            sw = __fadd2_rn(sw, make_float2(fmaxf(diff.x, 0.0f), fmaxf(diff.y, 0.0f)));
            if (kAux) sd = __fadd2_rn(sd, make_float2(fmaxf(-diff.x, 0.0f), fmaxf(-diff.y, 0.0f)));
            continue;
        }
        // r = 1 - min{c p/q, 1}; q = 0 gives -inf or NaN before the clamp to [0, 1], 0 after it
        const float2 r = make_float2(mul_sat(diff.x, rcp(q.x)), mul_sat(diff.y, rcp(q.y)));
        if (KT != 1) sw = __ffma2_rn(q, ipow2<KT>(r, K), sw);
        if (kAux) {
            sd = __fadd2_rn(sd, make_float2(fmaxf(-diff.x, 0.0f), fmaxf(-diff.y, 0.0f)));
            float2 acc = splat(0.0f);
            if (KT > 0) {
                if (KT >= 2) {
                    acc = splat(1.0f);
#pragma unroll
                    for (int u = 0; u < KT - 2; ++u) acc = __ffma2_rn(acc, r, splat(coef[u]));
                }
            } else if (K >= 2) {
                acc = splat(1.0f);
                float vj = 1.0f;
                for (int u = 1; u <= K - 2; ++u) {
                    vj *= v1;
                    acc = __ffma2_rn(acc, r, splat((float)(u + 1) * vj));
                }
            }
            const float2 ct = __fadd2_rn(r, nv1);  // c - t with t = 1 - r
            sm = __ffma2_rn(__fmul2_rn(q, __fmul2_rn(ct, ct)), acc, sm);
        }
    }
    w = sw.x + sw.y;
    if (kAux) {
        sd_out = sd.x + sd.y;
        sm_out = sm.x + sm.y;
    }
}

// 2^((m - row) scale), m <= row: the factor that moves a sum from units of the reference m to units of the row's, in float64.
__device__ __forceinline__ double unit_factor(float m, float row, float scale) {
    // e^(f ln 2), |f| <= 1/2, by its Taylor series to degree 11 (remainder below 7e-15), in pairs and without a branch: behind
    // exp2_short's the lanes ran apart and the shuffles of the sums took 1.1 us more per row
    // (the nearest integer by an addition that leaves no room for a fraction: it also stands in the low word then)
    const double x = fmax(((double)m - (double)row) * (double)scale, -1000.0), y = x + 6755399441055744.0;
    const double t = (x - (y - 6755399441055744.0)) * 0.6931471805599453094, t2 = t * t, t4 = t2 * t2;
    const double c0 = 1.0 + t, c1 = fma(t, 1.0 / 6.0, 0.5), c2 = fma(t, 1.0 / 120.0, 1.0 / 24.0), c3 = fma(t, 1.0 / 5040.0, 1.0 / 720.0);
    const double c4 = fma(t, 1.0 / 362880.0, 1.0 / 40320.0), c5 = fma(t, 1.0 / 39916800.0, 1.0 / 3628800.0);
    const double lo = fma(t2, c1, c0), mid = fma(t2, c3, c2), hi = fma(t2, c5, c4);
    return fma(t4, fma(t4, hi, mid), lo) * __hiloint2double((__double2loint(y) + 1023) << 20, 0);
}
// (m - row) scale in float32, m <= row, and what the difference and the product were rounded by.
__device__ __forceinline__ float unit_exponent(float m, float row, float scale, float &lost) {
    const float d = row - m, x = d * -scale;
    lost = fmaf(d, -scale, -x) - ((row - d) - m) * scale;
    return x;
}
// unit_factor in float32, with what the exponent was rounded by, so that what is left is the error of ex2.approx, 2^-22, in factors
// other than 1.
__device__ __forceinline__ float unit_factor_f32(float m, float row, float scale) {
    float lost;
    const float f = ex2(unit_exponent(m, row, scale, lost));
    return f > 0.0f ? fmaf(f, lost * 0.69314718f, f) : 0.0f;  // (0 x inf where m is -FLT_MAX)
}
// Sum over the warp of values in [0, 2^17), rounded to multiples of 2^-28 (of 32 multiples each, which add up exactly): the parts above
// and below 2^-5 as integers.  NaN if a lane's value is not in the range.
__device__ __forceinline__ double warp_sum_fixed(float v) {
    const float hi0 = 1.5f * 262144.0f, lo0 = 1.5f / 32.0f;  // an addition to these leaves the integer in the low bits
    const float hi = v + hi0, lo = (v - (hi - hi0)) + lo0;
    const int h = __reduce_add_sync(0xffffffffu, __float_as_int(hi) - __float_as_int(hi0));
    const int l = __reduce_add_sync(0xffffffffu, __float_as_int(lo) - __float_as_int(lo0));
    const double sum = fma((double)h, 1.0 / 32.0, (double)l * (1.0 / 268435456.0));
    return __any_sync(0xffffffffu, !(v < 131072.0f)) ? (double)NAN : sum;
}
// 1/x for x in the range of normal float32 numbers: the hardware's float32 reciprocal and one step of Newton's method, which squares
// its error: at most 2^-24 from x's conversion and 2^-23 from rcp.approx, 1.8e-7, so 3.2e-14 is left.  NaN for 0 and inf.
__device__ __forceinline__ double reciprocal(double x) {
    const double r = (double)rcp((float)x);
    return fma(r, fma(-x, r, 1.0), r);
}

// kAny: rows that do not all start on 16-byte boundaries (odd vocabularies, unaligned buffers).  A copy then brings the
// 16-byte pieces that hold the cell, and the reads from shared memory start at the remainder.  The few cells at the ends of the
// tensors whose pieces reach past them are loaded directly.
// Two sweeps over such rows (three scalar reads of every logit, four kernels) take longer, unless the rows are short and many
// (fused_outrun): 16 prompts, K = 4, gamma = 4, V = 50257 bfloat16 93 us against 55 here, one prompt, K = 3, gamma = 12, V = 32001
// float32 104 and 26, 64 prompts, K = 2, gamma = 4, V = 128255 float32 499 and 190.
// Against rows that start on the boundaries it costs 16 loads per lane and cell instead of 2 or 4, and mbarriers for its copies.
// NS: ring slots per warp (the cells per warp and row, kCtaCells / kWarps, are a multiple of it, so
// that cell j of a row always sits in slot j % NS); KT: the number of drafts K when it has a specialised
// second sweep (1, 2, 3, 4, 8), else 0 (any K, loops).
template <typename T, bool kRow, int NS, int KT, bool kAny>
__global__ void __launch_bounds__(kCtaThreads, 1) fused_chain_kernel(const FusedParams p) {
    constexpr int kCellsPerWarp = kCtaCells / kWarps;
    static_assert(kCellsPerWarp % NS == 0, "cell j of a row must always land in slot j % NS");
    extern __shared__ __align__(1024) unsigned char smem[];
    const Shape &s = p.s;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (tells the compiler that it is the same in all lanes)
    const int C = p.cluster;
    const int rank = (int)cluster_ctarank();
    const int cid = blockIdx.x / C;
    const int G = gridDim.x / C;
    constexpr int kHalfBytes = kCell * (int)sizeof(T);  // one tensor's cell
    constexpr int kHalfSlot = kHalfBytes + (kAny ? kSlack : 0);
    constexpr int kSlotBytes = 2 * kHalfSlot;           // the cell of zq, then the same cell of zp
    constexpr int kStride = kAny ? kWarps : 1;  // from one cell of a warp to its next, in a row
    constexpr int kRingBytes = kWarps * NS * kSlotBytes;
    // [rings][full barriers][references of the cells][parked first cells][Control]
    const unsigned char *ring = smem + (size_t)warp * NS * kSlotBytes;
    const uint32_t ring_u32 = smem_u32(ring);
    uint32_t pieces_u32 = ring_u32 + (uint32_t)lane * 16u;
    const uint32_t full_u32 = smem_u32(smem) + (uint32_t)(kRingBytes + warp * NS * 8);
    float2 *refs = reinterpret_cast<float2 *>(smem + kRingBytes + kWarps * NS * 8) + warp * kCellsPerWarp;
    float4 *park = reinterpret_cast<float4 *>(smem + kRingBytes + kWarps * NS * 8 + kCtaCells * (int)sizeof(float2)) + warp * 128 + lane;  // stride 32
    Control *ctl = reinterpret_cast<Control *>(smem + kRingBytes + kWarps * NS * 8 + kCtaCells * (int)sizeof(float2) + kWarps * kParkBytes);
    const uint32_t xbar_u32 = smem_u32(&ctl->xbar[0]);

    // This CTA's slice of the vocabulary, and this warp's cells in it: a few neighbours each.  The last warp, which does the exchange
    // of every row, only has those that the others cannot hold (with its share of the cells it kept the whole CTA waiting).
    const int cell_begin = rank * p.slice_cells;
    const int ncells_cta = max(0, min(s.ntiles, cell_begin + p.slice_cells) - cell_begin);
    // (In the row walk, where one row is all that most clusters have, the cells are shared out evenly.)
    const int most = kRow ? (ncells_cta + kWarps - 1) / kWarps : kCellsPerWarp;
    const int rest = max(0, ncells_cta - most * (kWarps - 1));  // of the last warp
    const int each = (ncells_cta - rest) / (kWarps - 1), more_by_one = (ncells_cta - rest) % (kWarps - 1);
    // (Rows that start anywhere: cells w, w + 32, ... of the slice for warp w; of the last warp's, those that fit go one each to
    // the first warps that would have one cell fewer than others.  Its only cell of a slice of 32 goes to another warp too: all waited for
    // its sweeps on top of the exchange, 4 x 4 x 12 x 32003 float32 81 -> 70 us, bfloat16 85 -> 71, 12 x 4 x 8 x 16001 61 -> 52, 63 -> 52.  With
    // two or three cells each a warp with one more takes as long, 64 x 4 x 4 x 16383 88 and 86, 71 and 70.  The row walk, where one row is
    // all that most clusters have, shares them out evenly.)
    const int columns = ncells_cta / kWarps, odd = ncells_cta % kWarps;
    const int given = odd > 0 ? min(columns, kWarps - 1 - odd) : columns == 1 && !kRow ? 1 : 0;
    const int own_cells = columns + (warp < odd), extra = kAny && warp >= odd && warp < odd + given ? warp - odd : -1;
    int ncw = !kAny ? (warp == kWarps - 1 ? rest : each + (warp < more_by_one))  // cells of this warp per row
                    : warp == kWarps - 1 ? columns - given : own_cells + (extra >= 0);
    const int first_cell = cell_begin + (kAny ? (warp == kWarps - 1 ? warp + given * kWarps : warp) : warp == kWarps - 1 ? ncells_cta - rest : warp * each + min(warp, more_by_one));
    // cell j of this warp, counted from its first one
    const int extra_j = extra >= 0 ? own_cells : -1, extra_at = kWarps - 1 + extra * kWarps - warp;
    auto cell_at = [&](int j) { return kAny && j == extra_j ? extra_at : j * kStride; };
    // the row's last cell may be a partial one: which of this warp's cells it is (-1: none), and its entries
    const int tail_valid = s.V - (s.ntiles - 1) * kCell;
    int tail_j = -1;
    for (int j = 0; j < ncw; ++j)
        if (tail_valid < kCell && first_cell + cell_at(j) == s.ntiles - 1) tail_j = j;

    if (tid == 0) {
        mbar_init(xbar_u32, 1);
        mbar_init(xbar_u32 + 8, 1);
    }
    if (kAny && lane == 0)
        for (int k = 0; k < NS; ++k) mbar_init(full_u32 + 8 * k, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    if (warp == 0) tmem_alloc(&ctl->tmem_base, kTmemCols);
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    // lanes of this warp's quarter, and its columns
    const uint32_t taddr = ctl->tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(warp >> 2) * (16u * kCellsPerWarp);
    cluster_arrive();  // every CTA of the cluster is running before any remote shared-memory access
    cluster_wait();

    // Small batches: this grid is itself launched with programmatic stream serialisation, so all of the above may have run while
    // the kernel ahead of it in the stream was still running (in a sequence of calls that is the previous
    // call's finishing kernel, which reads the scratch that this grid is about to write).  Nothing in global
    // memory has been touched so far; from here on that kernel has completed and its writes are visible.
    if (s.B <= kChainedLaunchMaxB) asm volatile("griddepcontrol.wait;" ::: "memory");
    // The finishing kernel is launched with programmatic stream serialisation: let it be scheduled now
    // (it waits for this grid to complete before it reads anything this grid writes).  Not in row mode:
    // there clusters wait for one another, so no CTA of this grid may find its place on an SM taken by
    // a kernel that in turn waits for this grid.
    if (!kRow) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0 && tid == 0) {
        *p.error_flag = 0;  // set again only by a wait that expires (about a second later)
        if (!kRow && !p.aux_here) p.ws.list[0] = 0;
    }
    // The walk of this cluster: position n = 0, 1, ... is row (bk, i).
    //   chain mode: the list of all rows, u = bk*gamma + i, is cut into G contiguous ranges of equal length (+-1), one
    //               per cluster, so that the clusters finish together whatever the number of chains.  A range may
    //               begin and end inside a chain.  The cluster walks first the HEAD of the chain its range ends in
    //               (rows 0..off_hi-1 of chain_hi) and leaves the ratio c reached there in a word of global memory,
    //               then its whole chains, and last the TAIL of the chain its range begins in (rows off_lo.. of
    //               chain_lo), whose c it picks up from the word the cluster before it wrote at its very start (one word
    //               per cluster).  The words are preset to a NaN pattern; the one wait (bounded) is for something written
    //               long before.
    //   row mode:   rows u = cid, cid+G, ... of the list.  Used when there are few rows: all rows of a chain then run
    //               at the same time on different clusters, and c_i comes from the ratios p_j(tok_j)/q_j(tok_j) that
    //               the clusters of rows j < i publish in global memory.  A row only waits for rows earlier in the
    //               list, which are walked no later by clusters that are all resident, so every wait ends.
    constexpr bool row_mode = kRow;
    const long total_rows = (long)p.nchains * s.gamma;
    const long range_lo = row_mode ? 0 : total_rows * cid / G, range_hi = row_mode ? 0 : total_rows * (cid + 1) / G;
    const int chain_lo = (int)(range_lo / s.gamma), off_lo = (int)(range_lo % s.gamma);
    const int chain_hi = (int)(range_hi / s.gamma), off_hi = (int)(range_hi % s.gamma);
    const int chain_mid = chain_lo + (off_lo > 0 ? 1 : 0);  // first whole chain of the range
    const int nrows = row_mode ? (int)((total_rows - cid + G - 1) / G) : (int)(range_hi - range_lo);  // rows this cluster walks
    // The first row of the walk: its number in the list and its place in its chain; seg_end: where its segment ends
    // (a range of gamma rows or more has a head or a whole chain)
    int r_b = row_mode ? cid : (off_hi > 0 ? chain_hi : chain_mid) * s.gamma;
    int i_b = row_mode ? cid % s.gamma : 0;
    int seg_end = row_mode ? 0 : off_hi > 0 ? r_b + off_hi : chain_hi * s.gamma;
    // From row (r, i) to the row after it in the walk.  Returns the number of chains between them.
    auto walk_next = [&](int &r, int &i) {
        if (row_mode) {
            const int from = r / s.gamma;
            r += G;
            i = r % s.gamma;
            return r / s.gamma - from;
        }
        ++r;
        ++i;
        if (r == seg_end) {
            const int from = (r - 1) / s.gamma;
            if (from == chain_hi && chain_mid < chain_hi) {  // from the head to the whole chains
                r = chain_mid * s.gamma;
                i = 0;
                seg_end = chain_hi * s.gamma;
            } else {  // to the tail
                r = (int)range_lo;
                i = off_lo;
                seg_end = -1;
            }
            return r / s.gamma - from;
        }
        if (i < s.gamma) return 0;
        i = 0;
        return 1;
    };
    const uint32_t xbytes = (uint32_t)(C * 2 * sizeof(float4));  // one partial from every CTA of the cluster
    uint32_t timed_out = 0;

    // ---- this warp's copy ring --------------------------------------------------------------------
    // Cell j of a row lands in slot j % NS.  The warp that has moved a cell from its slot to registers refills the slot at once,
    // with cell j + NS of the same row or, past the last, of the next row of the walk: the schedule is fixed at compile time.
    // Rows on 16-byte boundaries: every thread copies the 16-byte pieces that it will read itself (cp.async), one group of copies
    // per cell, an empty one where the warp has no such cell, and waits for its own groups by their order: no barrier, no
    // elected lane and hardly any address arithmetic.
    // kAny: bulk copies on the slot's mbarrier, which may start and end off the cell's boundaries; `pending` has bit k set
    // while a copy into slot k is under way, `phases` bit k is the parity of slot k's barrier.  A warp that has
    // given up on a wait issues no further loads and, before it leaves, waits for those in flight.
    const size_t row_bytes = (size_t)s.V * sizeof(T);
    const unsigned char *const zq_begin = reinterpret_cast<const unsigned char *>(p.zq), *const zp_begin = reinterpret_cast<const unsigned char *>(p.zp);
    const size_t ahead = (size_t)first_cell * kHalfBytes + (kAny ? 0 : lane * 16);  // from the start of a row to this warp's first cell
    const uint32_t is_lane0 = lane == 0 ? 1u : 0u;
    uint32_t pending = 0, phases = 0;
    // kAny: where a copy starts (the 16-byte boundary at or before the cell) and how long it is (a constant for all full
    // cells: always one piece more)
    auto floor16 = [](const unsigned char *a) {
        return reinterpret_cast<const unsigned char *>(reinterpret_cast<uintptr_t>(a) & ~(uintptr_t)15);
    };
    auto rest16 = [](const unsigned char *a) { return (uint32_t)reinterpret_cast<uintptr_t>(a) & 15u; };
    constexpr uint32_t kCopyBytes = (uint32_t)kHalfSlot;
    const uint32_t tail_bytes = (((uint32_t)(tail_valid * (int)sizeof(T)) + 15u) & ~15u) + kSlack;
    // whether copies of [a, a + bytes) of both tensors would leave them
    auto outside = [&](const unsigned char *q, const unsigned char *pp, size_t bytes) {
        return floor16(q) < zq_begin || floor16(pp) < zp_begin ||
               floor16(q) + bytes > zq_begin + (size_t)p.nchains * s.zq_rows * row_bytes ||
               floor16(pp) + bytes > zp_begin + (size_t)p.nchains * s.gamma * row_bytes;
    };
    // Rows that may hold such cells, by their number: those that begin within 64 bytes of the tensors' starts or end within 64 of their
    // ends (a copy begins at most 14 bytes before its cell and ends at most 31 behind it; row r of zp has at least as many
    // rows before and behind it in zq).  By their addresses it took a warp, with all others at the same place, 1000 cycles per row:
    // 4 x 4 x 12 x 50257 bfloat16 84 -> 76 us, 64 x 4 x 8 x 50257 268 -> 252, float32 259 -> 253.
    const int edge_rows = (int)(64 / row_bytes), edge_end = (int)total_rows - 1 - edge_rows;
    auto edge_row = [&](int r) { return kAny && (r <= edge_rows || r >= edge_end); };
    // cell j of the row whose first cells are q and pp cannot be copied
    auto direct = [&](const unsigned char *q, const unsigned char *pp, int j, bool edge) {
        return kAny && edge && outside(q + (size_t)cell_at(j) * kHalfBytes, pp + (size_t)cell_at(j) * kHalfBytes, j == tail_j ? tail_bytes : kCopyBytes);
    };
    // Starts the copies of cell j of the row whose first cells are q and pp.  whole: not the partial cell.
    auto request = [&](const unsigned char *q, const unsigned char *pp, auto cell, bool edge, auto whole) {
        constexpr bool kWhole = decltype(whole)::value;
        constexpr int j = decltype(cell)::value, slot = j % NS;
        if constexpr (kAny) {
            const unsigned char *qj = q + (size_t)cell_at(j) * kHalfBytes, *pj = pp + (size_t)cell_at(j) * kHalfBytes;
            if (!direct(q, pp, j, edge)) {
                issue_cell(ring_u32 + (uint32_t)(slot * kSlotBytes), floor16(qj), floor16(pj), !kWhole && j == tail_j ? tail_bytes : kCopyBytes,
                           full_u32 + 8u * (uint32_t)slot, is_lane0, kHalfSlot);
                pending |= 1u << slot;
            }
        } else {
            auto pieces = [&](auto part) {  // 32 pieces of 16 bytes at a time
                constexpr int h = decltype(part)::value, to = slot * kSlotBytes + 512 * h, from = j * kHalfBytes + 512 * h;
                if (!kWhole && j == tail_j && (lane + 32 * h) * (16 / (int)sizeof(T)) >= tail_valid) return;  // past the row's end
                copy16<to, from>(pieces_u32, q);
                copy16<to + kHalfSlot, from>(pieces_u32, pp);
            };
            pieces(Int<0>());
            if constexpr (kHalfBytes > 512) pieces(Int<1>());
        }
    };

    // The last warp of this CTA combines the partials, carries c_i and fetches the token logits of a row ahead of its exchange
    // (every lane the same words).
    const bool combiner = warp == kWarps - 1;
    // c at the start of chain bk: 1, or exp(log p(s) - log q(s)) of what Algorithm 2 carries in
#define SGBV_C0(BK) (p.carry_loga ? exp_short(p.carry_logb[BK] - p.carry_loga[BK]) : 1.0)
    double c_carry = 1.0;  // chain walk: c of the row whose exchange comes next (the first row of the walk starts a chain)
    if (combiner && nrows > 0) c_carry = SGBV_C0(r_b / s.gamma);
    // The combining warp: the next row's draft token, fetched a row ahead, and that row's logits of it.
    int tok_b = combiner && nrows > 0 && p.tok ? __ldg(p.tok + r_b) : 0;
    float zq_tok = 0.0f, zp_tok = 0.0f;
    auto prepare_exchange = [&](int pos, int r, int i) {
        if (C > 1 && lane == 0) mbar_expect_tx(xbar_u32 + 8u * (uint32_t)(pos & 1), xbytes);  // the partials of the cluster's CTAs
        const int t = tok_b >= 0 && tok_b < s.V ? tok_b : 0;  // (the finishing kernel flags the batch row)
        zq_tok = ld_logit(reinterpret_cast<const T *>(p.zq) + ((size_t)(r / s.gamma) * s.zq_rows + i) * s.V, t);
        zp_tok = ld_logit(reinterpret_cast<const T *>(p.zp) + (size_t)r * s.V, t);
    };
    // The exchange of row r (position pos of the walk; row nx, at place i_nx of its chain, chains_on chains further, follows if
    // has_next), by the combining warp.
    auto exchange = [&](int pos, int r, int i, bool has_next, int nx, int i_nx, int chains_on) {
        const int par = pos & 1;
        const uint32_t xph = (uint32_t)(pos >> 1) & 1u;
        const uint32_t xbar = xbar_u32 + 8u * (uint32_t)par;
        bar_sync(1, kCtaThreads);
        const float4 v = lane < kWarps ? ctl->wslots[lane] : make_float4(-INFINITY, 0.0f, -INFINITY, 0.0f);
        float bq_row = warp_max_redux(v.x), bp_row = warp_max_redux(v.z);
        float rq_row = (bq_row > -INFINITY) ? bq_row : 0.0f, rp_row = (bp_row > -INFINITY) ? bp_row : 0.0f;
        // The sum over the lanes of z, each moved from units of m to units of `row` (-inf: a lane without a share).  Every cycle from
        // here to the release is one that most of the SM's warps wait.  Sums and factors in float32 made up half of the error of the
        // residual masses; all in float64 (rows that start anywhere) took 500 cycles more per level.
        auto combine = [&](float m, double z, float row) {
            const double moved = z * unit_factor(m, row, s.scale);
            return warp_sum(m > -INFINITY ? moved : 0.0);
        };
        double Zq, Zp;
        if constexpr (kAny) {
            Zq = combine(v.x, v.y, rq_row);
            Zp = combine(v.z, v.w, rp_row);
        } else {
            Zq = warp_sum_fixed(v.x > -INFINITY ? v.y * unit_factor_f32(v.x, rq_row, s.scale) : 0.0f);
            Zp = warp_sum_fixed(v.z > -INFINITY ? v.w * unit_factor_f32(v.z, rp_row, s.scale) : 0.0f);
        }
        if (C > 1) {  // the same once more over the CTAs of the cluster
            const float4 mine = make_float4(bq_row, (float)Zq, bp_row, (float)Zp);
            if (lane < C) push_f4(&ctl->slots[par][rank], xbar, (uint32_t)lane, mine);
            if (lane < C) push_f4(&ctl->low[par][rank], xbar, (uint32_t)lane, make_float4(0.0f, (float)(Zq - (double)mine.y), 0.0f, (float)(Zp - (double)mine.w)));
            mbar_wait(xbar, xph, timed_out);
            timed_out = __any_sync(0xffffffffu, timed_out != 0);
            const float4 cv = lane < C ? ctl->slots[par][lane] : make_float4(-INFINITY, 0.0f, -INFINITY, 0.0f);
            bq_row = warp_max_redux(cv.x);
            bp_row = warp_max_redux(cv.z);
            rq_row = (bq_row > -INFINITY) ? bq_row : 0.0f;
            rp_row = (bp_row > -INFINITY) ? bp_row : 0.0f;
            const float4 low = lane < C ? ctl->low[par][lane] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if constexpr (kAny) {
                Zq = combine(cv.x, (double)cv.y + (double)low.y, rq_row);
                Zp = combine(cv.z, (double)cv.w + (double)low.w, rp_row);
            } else {  // (at most eight CTAs)
                Zq = cv.x > -INFINITY ? ((double)cv.y + (double)low.y) * (double)unit_factor_f32(cv.x, rq_row, s.scale) : 0.0;
                Zp = cv.z > -INFINITY ? ((double)cv.w + (double)low.w) * (double)unit_factor_f32(cv.z, rp_row, s.scale) : 0.0;
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    Zq += __shfl_xor_sync(0xffffffffu, Zq, o);
                    Zp += __shfl_xor_sync(0xffffffffu, Zp, o);
                }
                Zq = __shfl_sync(0xffffffffu, Zq, 0);
                Zp = __shfl_sync(0xffffffffu, Zp, 0);
            }
        }
        // The ratio p_i(tok_i)/q_i(tok_i) of this row: a chain of float64 operations.  In the chain walk only the
        // NEXT row needs it, so it is worked out after the other warps have been released.
        const double Zratio = Zq * reciprocal(Zp);
        auto ratio_of_row = [&]() {
            return exp2_short(((double)zp_tok - (double)rp_row) * (double)s.scale - ((double)zq_tok - (double)rq_row) * (double)s.scale) * Zratio;
        };
        double cd;
        if (row_mode) {
            const double ratio = ratio_of_row();
            // Publish this row's ratio for the clusters that walk the later rows of this chain.  The
            // word itself says "ready": it is preset to a NaN pattern, and a ratio is never stored as
            // NaN (a row that produces one is flagged invalid anyway).
            if (lane == 0 && rank == 0 && i + 1 < s.gamma && !(p.withhold && i == 0))
                *reinterpret_cast<volatile double *>(p.ws.ratio + r) = (ratio != ratio) ? 0.0 : ratio;
            // c_i = product of the published ratios of rows 0..i-1 of this chain (fixed order: a
            // butterfly over the lanes).  Those rows are walked by other clusters at about the same
            // time and publish right after their own statistics, which do not depend on c: no chain of
            // waits forms.  Every lane polls one of them.  Bounded waits.
            cd = SGBV_C0(r / s.gamma);
            const int r0 = r - i;
            for (int j0 = 0; j0 < i; j0 += 32) {
                double w = 1.0;
                if (j0 + lane < i) {
                    const volatile double *word = reinterpret_cast<const volatile double *>(p.ws.ratio + r0 + j0 + lane);
                    w = *word;
                    if (w != w && timed_out) w = 0.0;
                    if (w != w) {
                        const long long t0 = clock64();
                        while ((w = *word) != w) {
                            if (clock64() - t0 > p.poll_limit) {
                                timed_out = 1;
                                w = 0.0;
                                break;
                            }
                        }
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) w *= __shfl_xor_sync(0xffffffffu, w, o);
                cd *= w;
            }
            timed_out = __any_sync(0xffffffffu, timed_out != 0);
        } else {
            cd = c_carry;  // carried along the chain
        }
        const float4 rowv = make_float4(rq_row, rp_row, (float)(cd * Zratio), (float)cd);
        if (lane == 0) ctl->rs = rowv;
        __syncwarp();
        bar_arrive(2, kCtaThreads);
        // off the critical path: c of the next row of the chain walk (c_{i+1} = c_i ratio, and 1 at the start of
        // the next chain), and the row's record for the finishing kernel
        if (!row_mode) {
            const double c_next = cd * ratio_of_row();  // c after this row
            // the head of a chain that another cluster continues: leave c where that cluster looks for it
            if (r == chain_hi * s.gamma + off_hi - 1 && off_hi > 0 && lane == 0 && rank == 0)
                *reinterpret_cast<volatile double *>(p.ws.ratio + cid) = (c_next != c_next) ? 0.0 : c_next;
            if (has_next) {
                if (i_nx == 0) {
                    c_carry = SGBV_C0(nx / s.gamma);
                } else if (chains_on == 0) {
                    c_carry = c_next;
                } else {  // the tail of a chain whose head another cluster walked at its very start
                    const volatile double *word = reinterpret_cast<const volatile double *>(p.ws.ratio + cid - 1);
                    double w = *word;
                    if (w != w && !timed_out) {
                        const long long t0 = clock64();
                        while ((w = *word) != w)
                            if (clock64() - t0 > kWaitLimitCycles) {
                                timed_out = 1;
                                break;
                            }
                    }
                    c_carry = (w != w) ? 0.0 : w;
                }
            }
        }
        if (lane == 0 && rank == 0) {
            // nonfinite logits: NaN poisons Z, +inf shows up as an infinite reference, a row of
            // -inf only has Z = 0
            const bool bad = !(Zq > 0.0f) || !(Zp > 0.0f) || !(Zq < (double)INFINITY) || !(Zp < (double)INFINITY) ||
                             !(bq_row < INFINITY) || !(bp_row < INFINITY);
            RowInfo ri;
            ri.flags = bad ? SGBV_STATUS_NONFINITE_LOGIT : 0;
            ri.pad_ = 0;
            ri.Zq = (double)Zq;
            ri.Zp = (double)Zp;
            ri.mq = bq_row;
            ri.mp = bp_row;
            ri.kappa = rowv.z;
            ri.c = rowv.w;
            p.ws.rows[r] = ri;
        }
        return rowv;
    };
    // Without cells that is all it does.
    const bool exchange_only = combiner && ncw == 0;
    if (exchange_only) {
        if (lane == 0) ctl->wslots[warp] = make_float4(-INFINITY, 0.0f, -INFINITY, 0.0f);
        __syncwarp();
        for (int pos = 0, r = r_b, i = i_b; pos < nrows; ++pos) {
            int nx = r, i_nx = i;
            const int chains_on = walk_next(nx, i_nx);
            prepare_exchange(pos, r, i);
            if (pos + 1 < nrows && p.tok) tok_b = __ldg(p.tok + nx);
            exchange(pos, r, i, pos + 1 < nrows, nx, i_nx, chains_on);
            r = nx;
            i = i_nx;
        }
    }

    // Rows of the walk: A = the row whose second sweep runs, B = the one after it, whose first sweep runs in the same loop, D = the
    // one after B, E = the one after D.  A warp's cells take five places in turn, four in tensor memory and one in shared memory: cell j
    // of the row at position n lies in place (4 n + j) mod 5, so that cell j + 1 of row B goes where cell j of row A has just been
    // read.  Row B's partial is posted before the last cell of row A has its second sweep and the first cell of row D its first
    // one: that work runs while row B's partials are exchanged.
    // this warp's first cells (with cp.async this thread's first pieces) of the row whose cells are requested: the row of a cell
    // that lies NS cells behind the one that is swept
    const unsigned char *q_r = zq_begin + ahead + ((size_t)(r_b / s.gamma) * s.zq_rows + i_b) * row_bytes;
    const unsigned char *p_r = zp_begin + ahead + (size_t)r_b * row_bytes;
    bool edge_r = nrows > 0 && edge_row(r_b);
    const int nwalk = exchange_only ? -1 : nrows;  // rows that this warp sweeps
    if (nwalk > 0) {
        for_each_cell<NS>([&](auto cell) {
            if (cell < ncw) request(q_r, p_r, cell, edge_r, std::false_type());
            if (!kAny) copy_group_end();
        });
    }
    int r_w = r_b, i_w = i_b, chains_w = 0;  // the row that q_r, p_r go to next, and the chains between it and the one before
    auto to_next_row = [&]() {
        const int from = r_w;
        chains_w = walk_next(r_w, i_w);
        const int rows = r_w - from;
        q_r += (long)(rows + chains_w * (s.zq_rows - s.gamma)) * (int)row_bytes;
        p_r += (long)rows * (int)row_bytes;
        if (kAny) edge_r = edge_row(r_w);
    };
    FirstSweep f;  // row B, later row D
    auto fresh_row = [&]() {
        f.bq = f.bp = -FLT_MAX;
        f.sq = f.sp = splat(0.0f);
        f.moved = 0;
    };
    // First sweep of a cell of row r (kAny: its remainders and whether it may touch an end of a tensor); the slot is refilled, if
    // more: the row behind r exists.  steady: more, no partial cell, no end of a tensor.
    auto first_sweep = [&](auto cell, int place, int r, uint32_t rest_q, uint32_t rest_p, bool edge, bool more, auto steady) {
        constexpr bool kSteady = decltype(steady)::value;
        constexpr int j = decltype(cell)::value, slot = j % NS;
        constexpr bool kSameRow = j + NS < kCellsPerWarp;
        if constexpr (j + NS == kCellsPerWarp) to_next_row();  // from here on the next row's cells
        auto refill = [&]() {
            constexpr int next = (j + NS) % kCellsPerWarp;
            if (next < ncw && (kSameRow || kSteady || more) && (!kAny || kSteady || !timed_out)) request(q_r, p_r, Int<next>(), edge_r, steady);
            if (!kAny) copy_group_end();
        };
        if (j >= ncw) {
            refill();
            return;
        }
        float2 eq[4], ep[4];
        float m1, m2;
        if constexpr (kAny) {
            const bool copied = kSteady || (pending & (1u << slot));
            if (copied) {
                mbar_wait(full_u32 + 8u * slot, (phases >> slot) & 1u, timed_out);
                phases ^= 1u << slot;
                pending &= ~(1u << slot);
            }
            if (copied) {
                first_sweep_fetch<T, kAny>(ring + slot * kSlotBytes, rest_q, rest_p, lane, !kSteady && j == tail_j, tail_valid, eq, ep, m1, m2);
            } else {
                const size_t off = ahead + (size_t)cell_at(j) * kHalfBytes;
                first_sweep_direct<T>(zq_begin + off + (size_t)(r + r / s.gamma * (s.zq_rows - s.gamma)) * row_bytes, zp_begin + off + (size_t)r * row_bytes,
                                      lane, j == tail_j ? tail_valid : kCell, eq, ep, m1, m2);
            }
            __syncwarp();  // every lane holds its share of the slot in registers now
        } else {
            copy_wait<NS - 1>();
            first_sweep_fetch<T, kAny>(ring + slot * kSlotBytes, 0, 0, lane, !kSteady && j == tail_j, tail_valid, eq, ep, m1, m2);
        }
        refill();
        set_references(f, j, m1, m2, s.scale, p.rise, refs);
        first_sweep_store(taddr + 16u * (uint32_t)place, place == 4, park, s.scale, eq, ep, f);
    };
    uint32_t rest_qb = rest16(q_r), rest_pb = rest16(p_r);  // (kAny) row B
    bool edge_b = edge_r;
    fresh_row();
    if (nwalk > 0) first_sweep(Int<0>(), 0, r_b, rest_qb, rest_pb, edge_b, nrows > 1, std::false_type());

    RowScalars rs;         // row A
    rs.Fq = rs.KF = rs.kFp = 0.0f;
    rs.c = 1.0f;
    bool moved_a = false;  // row A's cells have references of their own (in this warp)

    int r_a = 0;  // (set when B becomes A)
    int place = 1;  // of row A's first cell (n = -1: -4 mod 5)
    // n = -1: only the first sweep of row 0; n = nrows - 1: only the second sweep of the last row
    for (int n = -1; n < nwalk; ++n) {
        // (what follows from these is worked out where it is needed: hoisted out of the loop it would take more registers than there are)
        asm volatile("" : "+r"(ncw), "+r"(tail_j), "+r"(pieces_u32));
        const bool has_a = n >= 0, has_b = n + 1 < nrows, has_d = n + 2 < nrows, has_e = n + 3 < nrows;
        if (combiner && has_b) prepare_exchange(n + 1, r_b, i_b);

        // ---- second sweep of row A from tensor memory, cell by cell, each followed by the first sweep of the
        //      same cell of row B into the columns just read: the exponentials of the one and the sums of the
        //      other keep different pipes busy --------------------------------------------------------------
        float wsum[kCellsPerWarp];  // row A; the last one is that of the warp's last cell
#pragma unroll
        for (int j = 0; j < kCellsPerWarp; ++j) wsum[j] = 0.0f;
        auto part_of = [&](float *base) { return base + (size_t)r_a * s.ntiles + first_cell; };
        // Rows with c < 1 may need two more sums for Eq. 2.  Small and medium problems work them out here, for all
        // such rows (p.aux_here).  Large ones leave them to two kernels that follow this one and only touch the rows
        // whose plain numerator would cancel, a few per cent: here they slow every row with c < 1, and with it the
        // whole cluster, by more than half, which is worth two more launches only when the step is long.
        const bool aux_row = p.aux_here && rs.c < 1.0f;
        // Second sweep of a cell of row A.  plain: no extra sums, one reference per warp.
        auto second_sweep = [&](int j, float &w, auto plain) {
            float aux[2];
            if constexpr (decltype(plain)::value) {
                second_sweep_cell<KT, false>(taddr + 16u * (uint32_t)place, place == 4, park, rs.KF, rs.c, false, s.K, w, aux[0], aux[1]);
            } else {
                float fq = 1.0f, fp = 1.0f, kt = rs.KF;
                if (moved_a) {  // 2^(this cell's references - the warp's last ones)
                    const float2 d = refs[j];
                    fq = ex2(d.x);
                    fp = ex2(d.y);
                    kt = fminf(kt * ex2(d.y - d.x), FLT_MAX);
                }
                if (aux_row) {  // two more sums per cell, which leave right away
                    const bool tiny = !(fq * rs.Fq > 1e-30f);
                    second_sweep_cell<KT, true>(taddr + 16u * (uint32_t)place, place == 4, park, kt, rs.c, tiny, s.K, w, aux[0], aux[1]);
                    warp_sum_multi<2>(aux, lane);
                    if ((lane & 15) == 0) part_of((lane & 16) ? p.ws.mpart : p.ws.dpart)[cell_at(j)] = aux[0] * (tiny ? ((lane & 16) ? 0.0f : rs.kFp * fp) : fq * rs.Fq);
                    if (tiny) w = 0.0f;
                } else {
                    second_sweep_cell<KT, false>(taddr + 16u * (uint32_t)place, place == 4, park, kt, rs.c, false, s.K, w, aux[0], aux[1]);
                }
                w *= fq;
            }
        };
        auto next_place = [&]() { place = place == 4 ? 0 : place + 1; };
        // The common case by far has next to nothing to decide per cell.
        const bool plain = has_a && !aux_row && !moved_a && ncw > 0;
        if (plain && has_d && tail_j < 0 && !(kAny && (edge_b || timed_out))) {
            for_each_cell<kCellsPerWarp - 1>([&](auto cell) {
                constexpr int j = decltype(cell)::value;
                if (j + 1 < ncw) second_sweep(j, wsum[j], std::true_type());
                first_sweep(Int<j + 1>(), place, r_b, rest_qb, rest_pb, edge_b, true, std::true_type());
                next_place();
            });
        } else {
            for_each_cell<kCellsPerWarp - 1>([&](auto cell) {
                constexpr int j = decltype(cell)::value;
                if (has_a && j + 1 < ncw) second_sweep(j, wsum[j], std::false_type());
                if (has_b) first_sweep(Int<j + 1>(), place, r_b, rest_qb, rest_pb, edge_b, has_d, std::false_type());
                next_place();
            });
        }
        auto last_cell = [&]() {
            const int at = place;  // (of cell kCellsPerWarp - 1, whether or not the warp has it)
            place = at - (kCellsPerWarp - ncw);
            if (place < 0) place += 5;
            if (plain) second_sweep(ncw - 1, wsum[kCellsPerWarp - 1], std::true_type());
            else if (has_a && ncw > 0) second_sweep(ncw - 1, wsum[kCellsPerWarp - 1], std::false_type());
            place = at;
        };
        // row A's cell sums: summed over the warp, stored by the lane that owns value number idx
        auto store_sums = [&]() {
            const int idx = owner_index<kCellsPerWarp>(lane);
            constexpr int kOwnerMask = 32 / kCellsPerWarp - 1;  // lanes that hold the same total
            warp_sum_multi<kCellsPerWarp>(wsum, lane);
            const bool is_last = idx == kCellsPerWarp - 1;
            if ((lane & kOwnerMask) == 0 && (is_last ? ncw > 0 : idx + 1 < ncw)) part_of(p.ws.wpart)[cell_at(is_last ? ncw - 1 : idx)] = wsum[0] * rs.Fq;
        };
        if (!has_b) {
            last_cell();
            store_sums();
            break;
        }
        if (kAny) timed_out = __any_sync(0xffffffffu, timed_out != 0);  // the warp gives up as one
        // (the requests have come to row D)
        const int r_d = r_w, i_d = i_w, chains_on = chains_w;
        if (combiner && has_d && p.tok) tok_b = __ldg(p.tok + r_d);
        const uint32_t rest_qd = rest16(q_r), rest_pd = rest16(p_r);
        const bool edge_d = edge_r;
        float part[2] = {f.sq.x + f.sq.y, f.sp.x + f.sp.y};  // the warp's partial of row B: its references, and its sums relative to them
        warp_sum_multi<2>(part, lane);                       // lanes 0-15: the target's, 16-31: the draft's
        // Exchange.  Every warp leaves its partial in shared memory; the LAST warp of the CTA combines them,
        // trades the CTA's partial with the other CTAs of the cluster (asynchronous distributed-shared-memory
        // stores that complete on the receiver's mbarrier; it alone polls that barrier), works out the row's
        // scalars and hands them to the others.  The others wait on hardware barriers, which costs them no
        // issue slots: barrier 1 = "all partials are in", barrier 2 = "the row's scalars are in".
        // (a store to shared memory followed by an arrival on the barrier is the producer half of the hardware
        // barrier's producer/consumer pattern: the consumer that syncs on it sees the store)
        if ((lane & 15) == 0) reinterpret_cast<float2 *>(&ctl->wslots[warp])[lane >> 4] = make_float2(lane ? f.bp : f.bq, part[0]);
        __syncwarp();
        float4 rowv;  // rq, rp, kappa, c
        if (!combiner) {
            bar_arrive(1, kCtaThreads);
        } else {
            rowv = exchange(n + 1, r_b, i_b, has_d, r_d, i_d, chains_on);
        }
        last_cell();
        moved_a = f.moved != 0;
        if (moved_a) {  // the cells' references against the warp's last ones, in units of log2
            __syncwarp();
            if (lane < ncw) {
                const float2 own = lane < f.moved ? refs[lane] : make_float2(f.bq, f.bp);
                refs[lane] = make_float2((own.x - f.bq) * s.scale, (own.y - f.bp) * s.scale);
            }
            __syncwarp();  // (the combining warp comes to no block barrier before all its lanes read them)
        }
        const float bq_b = f.bq, bp_b = f.bp;
        fresh_row();
        if (has_d) first_sweep(Int<0>(), place, r_d, rest_qd, rest_pd, edge_d, has_e, std::false_type());
        if (has_a) store_sums();
        tmem_wait_st();
        next_place();  // of row B's first cell
        if (!combiner) {
            bar_sync(2, kCtaThreads);
            rowv = ctl->rs;  // (the barrier statement is a compiler barrier for memory)
        }
        // this warp's units -> the row's; row B becomes row A
        // (a factor is common to all of the warp's cells: its exponent's rounding, up to 2^-24 of the exponent, stays in their sums
        // where that of single entries averages out)
        float lost_q, lost_p;
        const float ref_q = unit_exponent(bq_b, rowv.x, s.scale, lost_q), ref_p = unit_exponent(bp_b, rowv.y, s.scale, lost_p);
        const float f_q = ex2_wide(ref_q);  // (not flushed below 2^-126: the warp's exponentials may be up to 2^kRise)
        rs.Fq = f_q > 0.0f ? fmaf(f_q, lost_q * 0.69314718f, f_q) : 0.0f;
        // equal references (identical rows above all) must give kappa itself: p = q everywhere then leaves an
        // exactly zero residual.  Finite: 0 x inf would take the weight of an entry with p = 0
        const float ref_pq = ref_p - ref_q, f_pq = ex2(ref_pq), lost_pq = (ref_p - (ref_q + ref_pq)) + (lost_p - lost_q);
        rs.KF = f_pq > 0.0f ? fminf(rowv.z * fmaf(f_pq, lost_pq * 0.69314718f, f_pq), FLT_MAX) : 0.0f;
        rs.kFp = p.aux_here ? rowv.z * ex2(ref_p) : 0.0f;
        rs.c = rowv.w;
        r_a = r_b;
        r_b = r_d;
        i_b = i_d;
        rest_qb = rest_qd;
        rest_pb = rest_pd;
        edge_b = edge_d;
    }
    if (!kAny) copy_wait<0>();
    // a warp that gave up may still have copies under way: they must land before the shared memory goes
    if (timed_out) {
        uint32_t fresh = 0;
#pragma unroll
        for (int k = 0; k < NS; ++k)
            if (kAny && (pending & (1u << k))) mbar_wait(full_u32 + 8u * k, (phases >> k) & 1u, fresh);
        if (lane == 0) atomicExch(p.error_flag, 1);
    }
    cluster_arrive();  // no CTA leaves while a neighbour may still write into its slots
    cluster_wait();
    tmem_fence_before();
    __syncthreads();  // every warp of this CTA is done with the tensor memory
    if (warp == 0) tmem_dealloc(ctl->tmem_base, kTmemCols);
#undef SGBV_C0
}

// ---- host side ----------------------------------------------------------------------------------------
struct Plan {
    int cluster, slice_cells, row_mode;
};

int g_opt_cluster = 0;     // 0 = automatic
int g_opt_max_clusters = 0;
int g_opt_walk = 0;        // 0 = automatic, 1 = chains, 2 = rows
int g_opt_poll_us = 0;     // 0 = about a second
int g_opt_withhold = 0;
int g_opt_aux = 0;         // 0 = automatic, 1 = the extra sums of rows with c < 1 in the streaming kernel, 2 = in kernels of their own
constexpr double kAuxApartMinBytes = 1024.0 * 1024 * 1024;

constexpr int kSmemPerCta = 227 * 1024;  // largest dynamic shared memory of one CTA
constexpr int kDevices = 64;
std::mutex g_plan_mu;      // guards the options and the per-device caches below

constexpr int kCtaSlots = 148;  // CTAs the device holds
// ring slots per warp: half a row's cells for float32 (128 KB of copies under way per SM), all of them for bfloat16
template <typename T>
constexpr int slots_for() { return sizeof(T) == 4 ? 2 : 4; }
template <typename T, bool kAny>
constexpr size_t smem_bytes() {
    return (size_t)kWarps * slots_for<T>() * (2 * (kCell * sizeof(T) + (kAny ? kSlack : 0)) + 8) + (size_t)kCtaCells * sizeof(float2) + (size_t)kWarps * kParkBytes + sizeof(Control);
}
int slice_cells_of(int cells, int C) { return (cells + C - 1) / C; }

template <typename T, bool kRow, int KT, bool kAny>
cudaError_t prepare(int dev) {
    static bool attr_done[kDevices];
    if (!attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(fused_chain_kernel<T, kRow, slots_for<T>(), KT, kAny>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerCta);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(fused_chain_kernel<T, kRow, slots_for<T>(), KT, kAny>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        attr_done[dev] = true;
    }
    return cudaSuccess;
}

// Clusters of C CTAs of this kernel that the device runs side by side (queried once per configuration).
template <typename T, bool kRow, int KT, bool kAny>
int resident_clusters(int dev, int C) {
    static int cached[kDevices][kMaxCluster + 1];
    int &slot = cached[dev][C];
    if (slot == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.blockDim = dim3(kCtaThreads);
        cfg.dynamicSmemBytes = smem_bytes<T, kAny>();
        cfg.gridDim = dim3(C * (kCtaSlots / C));
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int nmax = 0;
        if (cudaOccupancyMaxActiveClusters(&nmax, fused_chain_kernel<T, kRow, slots_for<T>(), KT, kAny>, &cfg) != cudaSuccess || nmax < 1) {
            cudaGetLastError();
            return 0;
        }
        slot = nmax;
    }
    return slot;
}

template <typename T, bool kRow, int KT, bool kAny>
int launch_as(const Launch &L, const Plan &plan, int *error_flag, int clusters, bool aux_here, int words_used) {
    FusedParams fp;
    fp.zq = L.zq;
    fp.zp = L.zp;
    fp.tok = L.tok;
    fp.s = L.s;
    fp.ws = L.ws;
    fp.cluster = plan.cluster;
    fp.slice_cells = plan.slice_cells;
    fp.nchains = L.s.B * L.s.cpr;
    fp.carry_loga = L.carry_loga;
    fp.carry_logb = L.carry_logb;
    fp.error_flag = error_flag;
    fp.poll_limit = g_opt_poll_us > 0 ? (long long)g_opt_poll_us * 2000ll : kWaitLimitCycles;
    fp.withhold = g_opt_withhold;
    fp.rise = std::min(kRise / L.s.scale, FLT_MAX / 2.0f);  // (-FLT_MAX stands for "no finite logit so far": what follows has to lie above it)
    fp.aux_here = aux_here ? 1 : 0;

    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kCtaThreads);
    cfg.dynamicSmemBytes = smem_bytes<T, kAny>();
    cfg.stream = L.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = plan.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // the kernel may be scheduled before the one ahead of it in the stream has finished (it waits for it
    // itself before it touches global memory): its launch and start-up then overlap that kernel's tail
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // Small batches only (see kChainedLaunchMaxB), and not where the clusters would be packed around the finishing kernel's
    // CTAs, one per batch row: if those do not fit on the SMs that the clusters leave idle, some clusters of an odd size find
    // no room and run behind the others (16 x 8 x 4 x 98304, clusters of three, float32 138 -> 156 us, bfloat16 138 -> 158;
    // clusters of five with 18 idle SMs gain 5 us of 250, those of two, four, six and eight lost nothing).
    const bool early = L.s.B <= kChainedLaunchMaxB &&
                       (kRow || plan.cluster == 1 || plan.cluster % 2 == 0 || clusters * plan.cluster + L.s.B <= kCtaSlots);
    cfg.numAttrs = early ? 2 : 1;
    cfg.gridDim = dim3(clusters * plan.cluster);
    if (words_used > 0 && !L.ratio_preset &&
        cudaMemsetAsync(L.ws.ratio, 0xff, (size_t)words_used * sizeof(double), L.stream) != cudaSuccess)
        return SGBV_ERR_CUDA;
    if (L.ev_begin) cudaEventRecord(L.ev_begin, L.stream);
    cudaError_t e = cudaLaunchKernelEx(&cfg, fused_chain_kernel<T, kRow, slots_for<T>(), KT, kAny>, fp);
    if (L.ev_end) cudaEventRecord(L.ev_end, L.stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return SGBV_ERR_CUDA;
    }
    return 1;
}

// Chooses the cluster size and the walk, then launches.  Returns launches, 0 if declined, or < 0.
template <typename T, int KT, bool kAny>
int plan_and_launch(const Launch &L, int *error_flag, int *words_used, bool *aux_apart) {
    const Shape &s = L.s;
    const int cells = s.ntiles;
    const long nchains = (long)s.B * s.cpr, units = nchains * s.gamma;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return SGBV_ERR_CUDA;
    if (prepare<T, false, KT, kAny>(dev) != cudaSuccess || prepare<T, true, KT, kAny>(dev) != cudaSuccess) {
        cudaGetLastError();
        return SGBV_ERR_CUDA;
    }
    Plan plan;
    int Cmin = (cells + kCtaCells - 1) / kCtaCells;  // smallest cluster whose slices fit the tensor memory
    if (Cmin > kMaxCluster) return 0;
    auto fits = [&](int C) { return C >= Cmin && C <= kMaxCluster; };
    auto resident = [&](int C, bool row) {
        return row ? resident_clusters<T, true, KT, kAny>(dev, C) : resident_clusters<T, false, KT, kAny>(dev, C);
    };
    // Few units of work: spread each over more CTAs (at least half the warps keep a cell) while all of them
    // still run side by side.
    auto widen = [&](long n_units, bool row) {
        int C = Cmin;
        while (2 * C <= kMaxCluster && cells >= C * kWarps && n_units <= resident(2 * C, row)) C *= 2;
        return C;
    };
    int C = g_opt_cluster ? g_opt_cluster : widen(nchains, false);
    // Few rows in all: when every ROW can have a cluster of its own in one wave, share out single rows
    // instead of chains (their only coupling, c_i, is looked up), so that the gamma rows of a chain run
    // side by side instead of one after the other.
    const int Crow = g_opt_cluster ? g_opt_cluster : widen(units, true);
    plan.row_mode = 0;
    if (g_opt_walk == 2 && units > kRatioWords) return SGBV_ERR_SHAPE;  // one ratio word per row, and only so many
    if (s.gamma > 1 && fits(Crow) && units <= kRatioWords &&
        (g_opt_walk == 2 || (g_opt_walk == 0 && units <= resident(Crow, true)))) {
        plan.row_mode = 1;
        C = Crow;
    }
    // A few rounds of rows: what counts is the number of rounds times the time of a row, some 3 us and 48 ns for each of a CTA's
    // cells.  (64 rows of 594 cells: clusters of five 26 at a time, three rounds, of six 24, three shorter ones: 39.6 -> 36.8 us.  Long
    // walks are bound by throughput, and the smallest cluster is best: 64 x 8 x 8 rows of that length 821 us, of six 996.)
    if (!g_opt_cluster && !plan.row_mode && fits(C) && g_opt_max_clusters == 0) {
        auto cost = [&](int c) {
            const long side_by_side = std::min<long>(resident(c, false), nchains);
            return side_by_side < 1 ? 1e30 : (double)((units + side_by_side - 1) / side_by_side) * (62.0 + (double)((cells + c - 1) / c));
        };
        const double base = cost(C);
        if (units <= 4L * std::min<long>(resident(C, false), nchains)) {
            int best = C;
            for (int c = C + 1; c <= kMaxCluster && c < 2 * C; ++c)
                if (cost(c) < 0.95 * base && cost(c) < cost(best)) best = c;
            C = best;
        }
    }
    if (!fits(C)) return g_opt_cluster ? SGBV_ERR_SHAPE : 0;
    plan.cluster = C;
    plan.slice_cells = slice_cells_of(cells, C);
    int clusters = g_opt_max_clusters > 0 ? g_opt_max_clusters : resident(C, plan.row_mode != 0);
    if (clusters < 1) return 0;  // this cluster shape cannot be scheduled here: nothing launched
    const long share = plan.row_mode ? units : nchains;  // what the clusters share out
    if (clusters > share) clusters = (int)share;
    if (clusters > kRatioWords) clusters = kRatioWords;  // (a forced number: one hand-over word per cluster)
    // hand-over words: one per row in the row walk; in the chain walk one per cluster, if a range may end inside a chain
    // (the words are put back by the finishing kernel, so on the library's own scratch no call has to clear them)
    *words_used = plan.row_mode ? (int)units : (s.gamma > 1 && nchains % clusters != 0) ? clusters : 0;
    // the extra sums of rows with c < 1: in this kernel, or for long steps (chain walk, 1 GB of logits or more) in the
    // kernels that the caller queues behind it
    const double bytes = 2.0 * (double)units * (double)s.V * (double)sizeof(T);
    // (with one draft the extra sum costs the kernel next to nothing, and most rows with c < 1 would be listed; rows that start
    // anywhere included: error of the weights against 64 bits with the sums here / apart 4.1e-8 / 5.7e-8 at 64 x 8 x 6 x 50257
    // bfloat16, 5.9e-8 / 1.0e-7 at 64 x 2 x 12 x 100003, where the two-sweep path has 1.6e-7 and 4.0e-7)
    // (Apart, rows whose numerator does not cancel take its plain form, which costs them up to a bit, and some of the error: bfloat16 with
    // many drafts would be faster apart from 100 MB on, 16 x 8 x 4 x 151936 148 / 140 us, 64 x 6 x 8 x 32000 220 / 170, but the 2-norm of the
    // weights' error there is 5.5e-8 / 6.5e-8 and 6.9e-8 / 7.4e-8.)
    const bool apart = bytes >= kAuxApartMinBytes;
    const bool aux_here = plan.row_mode || g_opt_aux == 1 || (g_opt_aux == 0 && (!apart || s.K == 1));
    *aux_apart = !aux_here;
    return plan.row_mode ? launch_as<T, true, KT, kAny>(L, plan, error_flag, clusters, true, *words_used)
                         : launch_as<T, false, KT, kAny>(L, plan, error_flag, clusters, aux_here, *words_used);
}

}  // namespace

void fused_set_options(int cluster, int max_clusters, int walk, int poll_us, int withhold, int aux) {
    std::lock_guard<std::mutex> lock(g_plan_mu);
    g_opt_aux = aux;
    g_opt_withhold = withhold;
    g_opt_walk = walk;
    g_opt_cluster = cluster;
    g_opt_max_clusters = max_clusters;
    g_opt_poll_us = poll_us;
}

// Whether all rows of this call start on 16-byte boundaries.
bool rows_aligned(const Launch &L) {
    const size_t esz = L.dtype == SGBV_DTYPE_BF16 ? 2 : 4;
    return (uintptr_t)L.zq % 16 == 0 && (uintptr_t)L.zp % 16 == 0 && ((size_t)L.s.V * esz) % 16 == 0;
}

// Whether the fused path can take this call: a row must fit the tensor memory of a cluster (8 CTAs x 32,768 entries).
bool fused_supported(const Launch &L) { return L.s.ntiles <= kMaxCluster * kCtaCells; }

// Whether the two-sweep kernels are the faster ones: many short rows that start anywhere.  A row costs a cluster some 2.5 us
// however short it is, and a cluster walks its rows one after the other, where the two-sweep kernels run all rows side by side
// and pay by the entry (three scalar reads, and the power of Eq. 2 in a loop where K has no kernel of its own).  Two sweeps :
// streaming, us, bfloat16 (float32): 1024 rows (64 x 4 x 4) of 4 cells 43 : 49 (44 : 47), of 12 cells 51 : 50 (47 : 48), of 17 cells
// 53 : 51 (51 : 49); 8192 rows (256 x 8 x 4) of 4 cells 85 : 245 (86 : 218), 17 cells 196 : 267 (215 : 252), 24 cells 249 : 274
// (270 : 262), 29 cells 286 : 285 (318 : 276).  One position (1024 x 1 x 1): 4 cells 40 : 51 (40 : 50), 20 cells 54 : 55 (54 : 53), 25
// cells 57 : 56 (59 : 55); 512 rows (64 x 8 x 1) of 4 cells 34 : 36 (34 : 34), of 9 cells 37 : 36 (35 : 34), of 17 cells 41 : 37 (39 : 36).
// K = 5, 3840 rows of 7 cells 69 : 134 (72 : 124), of 13 cells 92 : 138 (138 : 145), of 17 cells 110 : 142 (176 : 152): the line lies at
// 9 cells there, which leaves up to 12 cells of bfloat16 something to gain.  Rows on the boundaries (16-byte reads) stay with the streaming kernel at any
// length, as before.
bool fused_outrun(const Launch &L) {
    const Shape &s = L.s;
    std::lock_guard<std::mutex> lock(g_plan_mu);
    if (rows_aligned(L) || g_opt_cluster || g_opt_max_clusters || g_opt_walk || g_opt_aux) return false;
    const long rows = (long)s.B * s.cpr * s.gamma;
    const bool own_kernel = s.K <= 4 || s.K == 8;
    if (s.gamma == 1 && rows < 6 * 148) return rows >= 3 * 148 && s.ntiles <= 9 && own_kernel;
    if (rows < 6 * 148) return false;
    if (!own_kernel) return s.ntiles <= 9;
    return s.ntiles <= (rows >= 12 * 148 || s.gamma == 1 ? 24 : 12);
}

template <typename T, bool kAny>
int dispatch_k(const Launch &L, int *error_flag, int *words_used, bool *aux_apart) {
    switch (L.s.K) {
        case 1: return plan_and_launch<T, 1, kAny>(L, error_flag, words_used, aux_apart);
        case 2: return plan_and_launch<T, 2, kAny>(L, error_flag, words_used, aux_apart);
        case 3: return plan_and_launch<T, 3, kAny>(L, error_flag, words_used, aux_apart);
        case 4: return plan_and_launch<T, 4, kAny>(L, error_flag, words_used, aux_apart);
        case 8: return plan_and_launch<T, 8, kAny>(L, error_flag, words_used, aux_apart);
        default: return plan_and_launch<T, 0, kAny>(L, error_flag, words_used, aux_apart);
    }
}

int launch_fused(const Launch &L, int *error_flag, int *words_used, bool *aux_apart) {
    *words_used = 0;
    *aux_apart = false;
    std::lock_guard<std::mutex> lock(g_plan_mu);
    const bool any = !rows_aligned(L);
    if (L.dtype == SGBV_DTYPE_BF16)
        return any ? dispatch_k<uint16_t, true>(L, error_flag, words_used, aux_apart)
                   : dispatch_k<uint16_t, false>(L, error_flag, words_used, aux_apart);
    return any ? dispatch_k<float, true>(L, error_flag, words_used, aux_apart)
               : dispatch_k<float, false>(L, error_flag, words_used, aux_apart);
}

}  // namespace sgbv
