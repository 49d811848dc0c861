// The scoring and candidate helpers shared by the tensor-core epilogues of
// orders 2 and 3: exact integer accumulators as packed counts, FP32 pairs, the
// hardware logarithm, the warps' candidate buffers, the CTA's sorted list, and
// the score threshold over all CTAs.  Included by one translation unit per
// kernel, after fc_tc.cuh.
#pragma once
#include "fc_tc.cuh"

namespace fc {
namespace {

constexpr int TC_WBUF = 64;   // candidates of a warp's buffer

// 8 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr));
}

// Two exact FP32 accumulators (integers below 2^16) packed as lo | hi << 16:
// x + 2^23 has the integer in its low mantissa bits, and the exponent
// field of the high word falls outside 32 bits after the shift.
__device__ __forceinline__ uint32_t pack_exact(uint32_t lo_bits, uint32_t hi_bits)
{
    const uint32_t a = __float_as_uint(__uint_as_float(lo_bits) + 8388608.0f);
    const uint32_t b = __float_as_uint(__uint_as_float(hi_bits) + 8388608.0f);
    return a + (b << 16) - 0x4B000000u;
}

// One encoded accumulator x = 4 (n_case + 4096 n_ctrl) (a multiple of 4 below
// 2^26, n_case < 4096, so exact) as 4 n_case | 4 n_ctrl << 16: v = x as an
// integer, and v + (v >> 14) (2^18 - 2^14) moves n_ctrl from bit 14 to bit 18.
__device__ __forceinline__ uint32_t unpack_enc(uint32_t bits)
{
    const uint32_t v = __float2uint_rz(__uint_as_float(bits));
    return v + (v >> 14) * 245760u;
}

// Two FP32 operations per instruction.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float x, float y)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 f2_split(F2 a)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

constexpr float LN2F = 0.693147180559945309f;

// Hardware base-2 logarithm (MUFU), flush-to-zero; x >= 1 here.
__device__ __forceinline__ float lg2_approx(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// An integer below 2^23 as a float, exactly.
__device__ __forceinline__ float u2f_small(uint32_t n)
{
    return __uint_as_float(n | 0x4B000000u) - 8388608.0f;
}

// (The next three functions are calls, so that the scoring loop keeps its
// registers.)
// Sorts a warp's m <= TC_WBUF candidates (ws, wr) best first, keeping those
// that beat (thr_s, thr_r); returns their number.
__device__ __noinline__ int sort_candidates(float *ws, uint64_t *wr, int m, float thr_s, uint64_t thr_r, int lane)
{
    float cs[2];
    uint64_t cr[2];
    unsigned keep[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int x = lane + 32 * h;
        cs[h] = x < m ? ws[x] : -FLT_MAX;
        cr[h] = x < m ? wr[x] : NO_RANK;
        keep[h] = __ballot_sync(FULL, x < m && better(cs[h], cr[h], thr_s, thr_r));
    }
    const unsigned below = (1u << lane) - 1u;
    bool mine[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        mine[h] = (keep[h] >> lane & 1u) != 0;
        if (mine[h]) {
            const int p = (h ? __popc(keep[0]) : 0) + __popc(keep[h] & below);
            ws[p] = cs[h];
            wr[p] = cr[h];
        }
    }
    m = __popc(keep[0]) + __popc(keep[1]);
    __syncwarp();
    // A candidate's place is the number of better ones.
    int at[2] = {0, 0};
#pragma unroll 4
    for (int y = 0; y < m; ++y) {
        const float s = ws[y];
        const uint64_t r = wr[y];
#pragma unroll
        for (int h = 0; h < 2; ++h) at[h] += better(s, r, cs[h], cr[h]);
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (mine[h]) {
            ws[at[h]] = cs[h];
            wr[at[h]] = cr[h];
        }
    __syncwarp();
    return m;
}

// Number of the n entries (s, r), best first, that are better than (cs, cr).
__device__ __forceinline__ int count_better(const float *s, const uint64_t *r, int n, float cs, uint64_t cr)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (better(s[mid], r[mid], cs, cr)) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Merges m <= TC_WBUF candidates (ws, wr), best first, into the CTA's list (ls,
// lr: `fill` of L entries, best first, the rest -FLT_MAX / NO_RANK); returns the
// entries then.  All lanes of the warp that holds the list's lock.  An entry
// moves down by the candidates placed before it: one number for a chunk of 32
// entries but for the few candidates placed inside it (a search per entry
// took 28 us for a list of 2048, and 2,000 SNPs with top 1,000 2.6 ms instead of
// 0.45).
__device__ __noinline__ int merge_candidates(float *ls, uint64_t *lr, int L, int fill, const float *ws, const uint64_t *wr,
                                             int m, int lane)
{
    // Every candidate's place: its place among the candidates plus the list
    // entries before it.
    int before[2], first = L;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int x = lane + 32 * h;
        before[h] = L;
        if (x < m) {
            before[h] = count_better(ls, lr, fill, ws[x], wr[x]);
            first = min(first, before[h]);
        }
    }
    first = __reduce_min_sync(FULL, first);
    // Entries from `first` on, blocks of 256 from the end.
    constexpr int B = 8;
    for (int base = (fill - 1) / (32 * B) * (32 * B); fill > 0 && base >= 0 && base + 32 * B > first; base -= 32 * B) {
        float s[B];
        uint64_t r[B];
        int p[B];
#pragma unroll
        for (int q = 0; q < B; ++q) {
            const int c = base + 32 * q, x = c + lane;
            const bool in = x >= first && x < fill;
            if (in) {
                s[q] = ls[x];
                r[q] = lr[x];
            }
            int shift = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                shift += __popc(__ballot_sync(FULL, before[h] <= c));
                unsigned inside = __ballot_sync(FULL, before[h] > c && before[h] < min(c + 32, L));
                for (; inside; inside &= inside - 1) shift += __shfl_sync(FULL, before[h], __ffs(inside) - 1) <= x;
            }
            p[q] = in ? x + shift : L;
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < B; ++q)
            if (p[q] < L) {
                ls[p[q]] = s[q];
                lr[p[q]] = r[q];
            }
        __syncwarp();
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int x = lane + 32 * h, to = before[h] + x;
        if (x < m && to < L) {
            ls[to] = ws[x];
            lr[to] = wr[x];
        }
    }
    __syncwarp();
    return min(L, fill + m);
}

// A score that at least L combinations reach, from what the CTAs of the
// launch have published (pub[n]: the score of the list's entry m - 1 as an
// ordered int): the r-th largest, r m >= L, to 20 bits downwards; -FLT_MAX while
// fewer than r have.  All lanes of a warp; n <= 32 TC_PUB_PER_LANE.
constexpr int TC_PUB_PER_LANE = 8;
__device__ __noinline__ float published_threshold(const int *pub, int n, int r, int lane)
{
    uint32_t key[TC_PUB_PER_LANE];
#pragma unroll
    for (int x = 0; x < TC_PUB_PER_LANE; ++x) {
        const int c = lane + 32 * x;
        key[x] = c < n ? (uint32_t)*(volatile const int *)(pub + c) ^ 0x80000000u : 0u;
    }
    uint32_t t = 0;
    for (int b = 31; b >= 12; --b) {
        const uint32_t c = t | 1u << b;
        int cnt = 0;
#pragma unroll
        for (int x = 0; x < TC_PUB_PER_LANE; ++x) cnt += __popc(__ballot_sync(FULL, key[x] >= c));
        if (cnt >= r) t = c;
    }
    // Below r lists t is the key of the value set before the launch, 0x80808080,
    // to 20 bits.
    return t > 0x00808000u ? from_ordered((int)(t ^ 0x80000000u)) : -FLT_MAX;
}

}  // namespace
}  // namespace fc
