// Helpers of the tcgen05 kernels:
// tile constants, mbarrier waits with a time budget, TMA loads, shared-memory
// and instruction descriptors, MMA issue and commit, TMEM loads, and the
// epilogue's named barrier and bitonic sort.  Included by one translation
// unit per kernel; everything is internal to that unit.
#pragma once
#include <cuda.h>
#include <cfloat>
#include "fc_internal.cuh"

namespace fc {
namespace {

constexpr int TC_BM = 128;          // tile rows of a CTA
constexpr int TC_BK = 128;          // K bytes per pipeline stage
constexpr int TC_SCHED = 4;         // depth of the tile-scheduling ring
constexpr uint32_t TC_TMEM_COLS = 512;
constexpr uint32_t TC_A_BYTES = TC_BM * TC_BK;   // 16 KiB
constexpr unsigned FULL = 0xffffffffu;
constexpr long long WAIT_BUDGET = TC_WAIT_TICKS;  // clock64 ticks (~2 s) per wait

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// The same test, letting the hardware suspend the thread until the phase
// completes or about 20 us pass (a waiting warp then issues nothing, which
// leaves the issue slots of its scheduler to the epilogue warps).
__device__ __forceinline__ bool mbar_try_suspend(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(20000u)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of the given parity.  On timeout it raises the
// CTA abort flag and the device error word; every role then leaves its loop.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                          uint32_t *err, long long budget = WAIT_BUDGET)
{
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_suspend(bar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > budget) {
            *abort_flag = 1;
            atomicOr(err, ERR_TIMEOUT);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void tma_load_2d(const CUtensorMap *map, uint64_t *bar, void *dst, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(smem_u32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Shared-memory matrix descriptor for a K-major tile written by TMA with the
// 128-byte swizzle: rows of 128 bytes, 8-row (1024-byte) swizzle atoms.
// Fields: start address >> 4 (bits 0-13), leading byte offset >> 4 (16-29,
// unused for swizzled K-major, set to 1), stride byte offset >> 4 (32-45:
// 1024 bytes between 8-row groups), fixed 0b001 at bits 46-48, swizzle mode
// 2 (128 B) at bits 61-63.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3fff);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// ---- kind::mxf4: packed 4-bit 0/1 operands -----------------------------------
// Indicator rows as e2m1 nibbles (0x2 = 1.0, sample m in nibble m): 128-byte
// K chunks hold 256 samples, four MMAs of K = 64.  A block scale (ue8m0, one
// per 32 samples and row, in TMEM) multiplies the products; here a scale is
// the same for every row and block, so a TMEM column whose bytes are all
// equal serves any scale layout.  Control samples take the A scale 2^12, so
// that one FP32 accumulator holds n_case + 4096 n_ctrl.  Exact: the products
// are 0 or 1 times a power of two, and FP32 accumulation of integers below
// 2^24 was measured exact on GB300 up to 16,777,215 (128 x 240 tiles over
// 8,190 samples with full rows).  Half the bytes per sample of e4m3 and, for
// N = 240, twice its multiply-adds per cycle (120 cycles per K = 64 MMA).
constexpr uint32_t FP4_SCALE_ONE = 0x7F7F7F7Fu;    // ue8m0 2^0
constexpr uint32_t FP4_SCALE_4 = 0x81818181u;      // ue8m0 2^2
constexpr uint32_t FP4_SCALE_4096 = 0x8B8B8B8Bu;   // ue8m0 2^12
constexpr uint32_t FP4_SCALE_COLS = 16;            // TMEM columns per scale (at most 8 are read)

// Instruction descriptor, kind::mxf4: A = B = E2M1 (bits 7-9, 10-11 = 1),
// N >> 3 at bits 17-22, scales ue8m0 (bit 23), M >> 4 at bits 24-28, K = 64
// (bit 31 = 0), scale ids 0 (bits 4-5, 29-30).
__host__ __device__ constexpr uint32_t idesc_mxf4(int M, int N)
{
    return (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | (1u << 23) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_mxf4(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t scale_a, uint32_t scale_b, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.block32 [%0], %1, %2, %3, [%4], [%5], p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(scale_a), "r"(scale_b), "r"(accumulate)
        : "memory");
}

// ---- CTA pairs (cta_group::2) ---------------------------------------------------
// Two CTAs of a cluster (one TPC) work on one M = 256 tile: each holds its
// 128 rows of A, half of the rows of B and its 128 accumulator lanes; the MMAs
// are issued by the leader (rank 0) alone.  Copies of both CTAs complete on
// the leader's barriers, commits arrive on both CTAs' barriers.
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Shared-cluster address of `p` in the CTA of rank `rank`.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}
// Arrive on the barrier at a shared-cluster address.  What crosses the pair
// this way is only "this slot has been read" and "this accumulator has been
// read" (ordered by tcgen05 fences); arrivals and waits of cluster scope would
// add a fence and drop the L1 lines of the waiting SM each time (orders 5 and
// 6 at 2,048 samples: 174 and 168 ms instead of 126 and 130).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// Writes {x, y} to the 8 bytes at a shared-cluster address, completing the
// current phase of the barrier at `bar` there (one arrival and these bytes):
// a waiter on that barrier sees the data.
__device__ __forceinline__ void cluster_post2(uint32_t addr, uint32_t bar, int x, int y)
{
    asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], 8;" ::"r"(bar) : "memory");
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(addr), "r"(x),
                 "r"(y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void cluster_post4(uint32_t addr, uint32_t bar, uint4 v)
{
    asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], 16;" ::"r"(bar) : "memory");
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "r"(v.x),
        "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
        : "memory");
}
// Copy into this CTA's shared memory that completes on barrier `bar` (the
// same offset) of the pair's leader: bit 24 of a shared-cluster address
// selects the CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(const CUtensorMap *map, uint64_t *bar, void *dst, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(smem_u32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar) & 0xFEFFFFFFu)
        : "memory");
}
__device__ __forceinline__ void mma_mxf4_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t scale_a, uint32_t scale_b, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::mxf4.block_scale.block32 [%0], %1, %2, %3, [%4], [%5], p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(scale_a), "r"(scale_b), "r"(accumulate)
        : "memory");
}
// Arrives on `bar` (the same offset) of both CTAs once the MMAs issued so far
// are complete.
__device__ __forceinline__ void mma_commit_pair(uint64_t *bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"((uint16_t)3)
        : "memory");
}

// 16 TMEM columns of this warp's lane quarter, all words v.
__device__ __forceinline__ void tmem_fill16(uint32_t taddr, uint32_t v)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr),
        "r"(v)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 32 sample bits as 32 e2m1 nibbles (16 bytes).
__device__ __forceinline__ uint4 expand_fp4(uint32_t bits)
{
    uint32_t o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t x = (bits >> (8 * q)) & 0xffu;
        x = (x | (x << 12)) & 0x000F000Fu;
        x = (x | (x << 6)) & 0x03030303u;
        x = (x | (x << 3)) & 0x11111111u;
        o[q] = x << 1;
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// True on one lane of a converged warp.  The MMA and TMA issue loops run
// under this predicate rather than under lane == 0: the compiler then knows
// that one thread runs the branch and keeps descriptors and addresses in
// uniform registers, which the tcgen05 and bulk-copy instructions take
// directly.  Under lane == 0 every MMA first moved its operands there one by
// one, and the issue alone took 136 cycles per MMA (128 x 240 x 64 in fp4, 120
// cycles of tensor work; 172 with the waits and copies of the pipeline)
// against 120 (both) under elect.sync, measured on GB300 over 6400 chunks.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

// Position in a ring of n stages: stage s, and the parity of its current
// fill (the pipeline's loops step it instead of dividing a fill count).
struct Ring {
    int s = 0;
    uint32_t par = 0;
    __device__ __forceinline__ void next(int n)
    {
        if (++s == n) {
            s = 0;
            par ^= 1;
        }
    }
};

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Ties registers written by tcgen05.ld to a point after tcgen05.wait::ld:
// the compiler sees them redefined here, so no use can move above the wait.
template <int N>
__device__ __forceinline__ void tmem_regs_after_wait(uint32_t (&v)[N])
{
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("" : "+r"(v[i]));
}

// Named barrier 1 over the NT epilogue threads.
template <int NT>
__device__ __forceinline__ void epi_bar_n() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }

// 28 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld28(uint32_t taddr, uint32_t (&v)[28])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
          "=r"(v[15])
        : "r"(taddr));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23])
                 : "r"(taddr + 16));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27])
                 : "r"(taddr + 24));
}

// A float of shared memory at a shared-space byte address (a table that is
// constant after the kernel's first barrier).
__device__ __forceinline__ float lds_f32(uint32_t addr)
{
    float v;
    asm("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

// Exact integer value of an FP32 accumulator holding an integer in [0, 2^23).
__device__ __forceinline__ uint32_t f2u_exact(uint32_t bits)
{
    return __float_as_uint(__uint_as_float(bits) + 8388608.0f) - 0x4B000000u;
}

__device__ __forceinline__ int ordered_int(float f)
{
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float from_ordered(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

// Descending bitonic sort of n = 2^p (score, rank) pairs by the NT
// epilogue threads (tid in [0, NT)).
template <int NT>
__device__ void epi_bitonic_desc_n(float *s, uint64_t *r, int n, int tid)
{
    for (int size = 2; size <= n; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            epi_bar_n<NT>();
            for (int i = tid; i < (n >> 1); i += NT) {
                const int lo = 2 * i - (i & (stride - 1));
                const int hi = lo + stride;
                const bool desc = (lo & size) == 0;
                const float s1 = s[lo], s2 = s[hi];
                const uint64_t r1 = r[lo], r2 = r[hi];
                const bool sw = desc ? better(s2, r2, s1, r1) : better(s1, r1, s2, r2);
                if (sw) { s[lo] = s2; s[hi] = s1; r[lo] = r2; r[hi] = r1; }
            }
        }
    }
    epi_bar_n<NT>();
}

}  // namespace
}  // namespace fc
