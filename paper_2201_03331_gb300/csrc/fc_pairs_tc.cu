// Order-2 all-pairs search on the fifth-generation tensor cores (tcgen05).
//
// For k = 2 the contingency counts of every SNP pair form a dense binary
// contraction (Section "Computing the contingency tables": a cell is the
// population count of the AND of one row of each SNP's genotype table):
//     n_c(g, h)[i, j] = sum_{m in class c} [G_i(m) = g] [G_j(m) = h].
// With the genotype rows g, h in {0, 1} stored as packed 0/1 e2m1 nibbles
// (E[2s + g][m]) one class's counts for all pairs are E_c E_c^T, and
// tcgen05.mma kind::mxf4 computes the four {0,1}x{0,1} cells of every pair
// exactly (fc_tc.cuh).  The five cells that involve genotype 2 follow exactly
// from the per-SNP genotype counts (the rows of each SNP's genotype table
// partition the samples):
//     n(g,2) = n_i(g) - n(g,0) - n(g,1),   n(2,h) = n_j(h) - n(0,h) - n(1,h),
//     n(2,2) = n_i(2) - n(2,0) - n(2,1).
// The epilogue scores each pair with the FP32 mutual information and keeps a
// CTA top list; the count matrix is never written.
//
// Two forms (template ENC), as in the order-3 kernel:
//   ENC = 1: control samples carry the block scale 4096, so one accumulator
//            holds n_case + 4096 n_ctrl (exact while both classes have at
//            most 4095 samples); a tile of 128 SNPs i and 112 SNPs j is worked
//            on by a pair of CTAs (cta_group::2, M = 256, N = 224): each
//            loads 64 SNPs i and 56 SNPs j and scores its SNPs i against all
//            112;
//   ENC = 0: the case and control samples accumulate into two accumulators;
//            a tile of 64 SNPs i and 56 SNPs j per CTA (M = 128, N = 112).
// A tile takes 224 TMEM columns and two tiles are in flight.
//
// The scores are those of the order-3 epilogue over 9 cells: t(a, b) = xl[n] -
// a lg2~(a) - b lg2~(b), counts times a power of two q that brings the samples to Q =
// q N < 8 (4 <= Q from 8 samples on).  |MI32 - MI| <= 28 u, u = 2^-24, whatever the
// samples: with x a scaled count, x |log2 x| <= 0.531 up to 1/2 and <= x max(1, log2 Q)
// above, so that the sum of x max(1, |log2 x|) over the 18 class counts is at most 9.6 +
// Q log2 Q <= 4.4 Q, and that of n |log2 n| over the 9 cells 4.8 + Q log2 Q <= 3.6 Q.
// In units of u Q, in bits, the table entries then err by 3.6, the logarithms (4 u
// max(1, |log2 x|) each) by 17.6, the first multiply-add of every cell by 3.6 + 4.4, the
// second (t <= n) by 1, the four levels of additions by 4; ln 2, its product, 1/N,
// H(Y) and the last multiply-add add 5: 39.2 u ln 2 < 28 u in nats.
//
// What bounds the kernel: with many samples the operands' way from L2 (30 KB a
// chunk and CTA; 12,000 SNPs x 8,192 samples, form 0, move 20 GB at 15 TB/s, the
// tensor pipe 37 % active, 1.6 instructions a cycle), with few the scoring.
// 40,000 SNPs x 8,192 samples, lists of 2048: 12.9 ms, x 2,048 samples: 7.1 ms; a
// search with its tail 13.1 and 7.3.  (The kernel before, byte rows in 128 x 128
// tiles of one CTA and four epilogue warps that met at barriers and sorted a
// shared buffer of candidates, took 37 ms for the first, and 15 of the 16 ms of
// a search of 12,001 SNPs x 2,987 samples met once, now 1.6: it sorted after
// nearly every 16 SNPs while its list filled.)
//
// TMEM lane 2 i + g holds genotype g of SNP i, columns 2 j + h genotype h of SNP
// j.  The two lanes of a SNP i take two SNPs j at a time, one each: they
// exchange the two cells of the other's SNP, and lane g reads its cells with
// the genotypes of i in the order g, 1 - g (its table of i is swapped alike).
//
// Candidates as in the order-3 kernel: a buffer per epilogue warp, merged into
// the CTA's sorted list under a lock, and a score threshold over all CTAs.
//
// Roles (one persistent CTA per SM, 640 threads):
//   warps 0, 1 : TMA producers (128-byte K chunks, 256 samples, of 128 rows of
//                the SNPs i and 112 of the SNPs j), warp w owning the stages
//                s = w (mod 2)
//   warp 2     : schedules the tiles (ENC 1: in the pair's leader), score
//                threshold
//   warp 3     : TMEM allocation; one elected lane (ENC 1: of the pair's
//                leader) issues the MMAs
//   warps 4-19 : epilogue, four warps per TMEM lane quarter, each taking every
//                fourth four SNPs j of a tile
#include <algorithm>

#include "fc_candidates.cuh"
#include "fc_ie.cuh"

namespace fc {

namespace {

constexpr int T2_PRODUCERS = 2;
constexpr int T2_EPI_WARP0 = 4;
constexpr int T2_EPI_WARPS = 16;
constexpr int T2_PARTS = T2_EPI_WARPS / 4;         // epilogue warps per TMEM lane quarter
constexpr int T2_EPI_THREADS = 32 * T2_EPI_WARPS;
constexpr int T2_THREADS = 32 * T2_EPI_WARP0 + T2_EPI_THREADS;
static_assert(T2_EPI_WARP0 % 4 == 0, "epilogue warp w reads TMEM lane quarter w % 4");
constexpr int T2_NJ = 56;                          // SNPs j per stage
constexpr int T2_N = 2 * T2_NJ;                    // their rows
constexpr int T2_IB = 64;                          // SNPs i per CTA and tile
constexpr uint32_t T2_STAGE = TC_A_BYTES + (uint32_t)T2_N * TC_BK;
static_assert(T2_STAGE % 1024 == 0, "swizzled stages");
constexpr int T2_BUF = 2 * T2_N;                   // TMEM columns of a tile
constexpr uint32_t T2_SCALE_COL = 2 * T2_BUF;      // TMEM column of scale 1, then of 4096, then of 4
static_assert(T2_SCALE_COL + 3 * FP4_SCALE_COLS <= TC_TMEM_COLS, "scales behind the accumulators");
constexpr int T2_WARP_SNPS = 4 * ((2 * T2_NJ / 4 + T2_PARTS - 1) / T2_PARTS);   // SNPs j of a tile per warp (ENC 1)
static_assert(T2_WARP_SNPS <= 32, "a lane per SNP record");

// ---- data preparation ------------------------------------------------------

// Per SNP and class, how many samples carry genotype 0, 1, 2:
// marg[s*8 + c*3 + g], c = 0 cases, 1 controls.
__global__ void k_marginals(const uint4 *X, int64_t S, int64_t S_pad, int W0, int Wt, uint16_t *marg)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    uint32_t cnt[2][3] = {{0, 0, 0}, {0, 0, 0}};
    for (int w = 0; w < Wt; ++w) {
        const int c = w < W0 ? 0 : 1;
        for (int g = 0; g < 3; ++g) {
            const uint4 v = X[((size_t)w * 3 + g) * S_pad + s];
            cnt[c][g] += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
        }
    }
    for (int c = 0; c < 2; ++c)
        for (int g = 0; g < 3; ++g) marg[s * 8 + c * 3 + g] = (uint16_t)cnt[c][g];
    marg[s * 8 + 6] = 0;
    marg[s * 8 + 7] = 0;
}

// ---- the fused tensor-core kernel ------------------------------------------

template <int MODE, int ENC>
__global__ void __launch_bounds__(T2_THREADS, 1) k_pairs_tc(const __grid_constant__ CUtensorMap tmapI,
                                                            const __grid_constant__ CUtensorMap tmapJ, PairsArgs a)
{
    constexpr bool PAIR = ENC == 1;                 // a tile per CTA pair
    constexpr int NJT = PAIR ? 2 * T2_NJ : T2_NJ;   // SNPs j per tile
    constexpr int SH = PAIR ? 2 : 0;                // counts come times 2^SH: the block scale of the SNPs j
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_full[TC_MAX_STAGES], bar_empty[TC_MAX_STAGES];
    __shared__ uint64_t bar_tfull[2], bar_tempty[2], bar_done, bar_epi;
    __shared__ uint32_t tmem_base_slot;
    __shared__ uint64_t bar_sfull[TC_SCHED], bar_sempty[TC_SCHED];
    __shared__ int2 sched_tile[TC_SCHED];   // {I << 16 | J, 1}, {0, 0}: no more tiles
    __shared__ int abort_flag_s;
    __shared__ int list_lock, list_fill;
    __shared__ int epi_end;                 // the epilogue has ended
    __shared__ float threshold;             // published_threshold

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int stages = a.stages;
    const uint32_t crank = PAIR ? cluster_rank() : 0;   // CTA of the pair (0: its leader)
    volatile int *abort_flag = &abort_flag_s;

    // The x log2 x table first (a constant base saves an addition per read);
    // then the stages, 1024-byte aligned, the warps' SNP records, the candidate
    // list and the warps' buffers (ranks before scores).
    float *xltab = reinterpret_cast<float *>(smem_raw);
    uint8_t *smem = reinterpret_cast<uint8_t *>(((uintptr_t)(xltab + a.M + 1) + 1023) & ~(uintptr_t)1023);
    uint2 *recs = reinterpret_cast<uint2 *>(smem + (size_t)stages * T2_STAGE);
    uint64_t *lrank = reinterpret_cast<uint64_t *>(recs + T2_EPI_WARPS * T2_WARP_SNPS);
    uint64_t *wrank = lrank + a.L;
    float *lscore = reinterpret_cast<float *>(wrank + T2_EPI_WARPS * TC_WBUF);
    float *wscore = lscore + a.L;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&bar_full[s], 1);
            mbar_init(&bar_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bar_tfull[b], 1);
            mbar_init(&bar_tempty[b], (PAIR ? 2 : 1) * T2_EPI_WARPS);
        }
        mbar_init(&bar_done, 1);
        mbar_init(&bar_epi, T2_EPI_WARPS);
        for (int s = 0; s < TC_SCHED; ++s) {
            mbar_init(&bar_sfull[s], 1);
            // The MMA thread, and the producer and epilogue warps (of both
            // CTAs of a pair).
            mbar_init(&bar_sempty[s], 1 + (PAIR ? 2 : 1) * (T2_PRODUCERS + T2_EPI_WARPS));
        }
        abort_flag_s = 0;
        list_lock = 0;
        list_fill = 0;
        epi_end = 0;
        threshold = -FLT_MAX;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 3) {
        if constexpr (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&tmem_base_slot)),
                         "r"(TC_TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&tmem_base_slot)),
                         "r"(TC_TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    for (int i = threadIdx.x; i <= a.M; i += blockDim.x) xltab[i] = a.xlogx[i];
    if (MODE == MODE_TOPN) {
        for (int i = threadIdx.x; i < a.L; i += blockDim.x) {
            lscore[i] = -FLT_MAX;
            lrank[i] = NO_RANK;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    if (warp >= T2_EPI_WARP0 && warp < T2_EPI_WARP0 + 4) {
        const uint32_t q = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + T2_SCALE_COL;
        tmem_fill16(q, FP4_SCALE_ONE);
        tmem_fill16(q + FP4_SCALE_COLS, FP4_SCALE_4096);
        tmem_fill16(q + 2 * FP4_SCALE_COLS, FP4_SCALE_4);
        tmem_wait_st();
    }
    tc_fence_before();
    // Barriers and scales of both CTAs are ready before either uses them.
    if constexpr (PAIR) cluster_sync(); else __syncthreads();
    tc_fence_after();
    const long long wt = a.wait_ticks;
    const int nk = (a.Wt + 1) / 2;   // K chunks

    // A consumer's word that it has read a slot of the tile ring.
    const uint32_t sempty0 = PAIR ? cluster_addr(&bar_sempty[0], 0) : 0;
    auto slot_read = [&](int slot) {
        if constexpr (PAIR) mbar_arrive_cluster(sempty0 + 8 * slot);
        else mbar_arrive(&bar_sempty[slot]);
    };

    if (warp < T2_PRODUCERS) {
        // ---------------- TMA producers ----------------
        if (elect_one()) {
            Ring ring;
            int owner = 0;   // producer of stage ring.s
            // Parity of the last fill issued into each owned stage (at most
            // three: stages warp, warp + 2, warp + 4), -1 before the first.
            int last[3] = {-1, -1, -1};
            auto step = [&]() {
                ring.next(stages);
                owner = ring.s == 0 || owner + 1 == T2_PRODUCERS ? 0 : owner + 1;
            };
            bool ok = true;
            for (int it = 0; ok; ++it) {
                const int slot = it % TC_SCHED;
                const uint32_t sn = (uint32_t)(it / TC_SCHED);
                if (!mbar_wait(&bar_sfull[slot], sn & 1, abort_flag, a.err, wt)) { ok = false; break; }
                const int2 tile = sched_tile[slot];
                slot_read(slot);
                if (!tile.y) break;
                const int I = (int)((uint32_t)tile.x >> 16), J = tile.x & 0xffff;
                const int rowI = 2 * T2_IB * ((PAIR ? 2 : 1) * I + (int)crank);
                const int rowJ = 2 * NJT * J + T2_N * (int)crank;
                for (int kc = 0; kc < nk; ++kc, step()) {
                    if (owner != warp) continue;
                    const int s = ring.s;
                    uint8_t *st = smem + (size_t)s * T2_STAGE;
                    if (!mbar_wait(&bar_empty[s], ring.par ^ 1, abort_flag, a.err, wt)) { ok = false; break; }
                    const int x = kc * TC_BK;
                    if constexpr (PAIR) {
                        // The leader's barrier counts the bytes of both CTAs.
                        if (crank == 0) mbar_expect_tx(&bar_full[s], 2 * T2_STAGE);
                        tma_load_2d_pair(&tmapI, &bar_full[s], st, x, rowI);
                        tma_load_2d_pair(&tmapJ, &bar_full[s], st + TC_A_BYTES, x, rowJ);
                    } else {
                        mbar_expect_tx(&bar_full[s], T2_STAGE);
                        tma_load_2d(&tmapI, &bar_full[s], st, x, rowI);
                        tma_load_2d(&tmapJ, &bar_full[s], st + TC_A_BYTES, x, rowJ);
                    }
                    last[0] = s == warp ? (int)ring.par : last[0];
                    last[1] = s == warp + T2_PRODUCERS ? (int)ring.par : last[1];
                    last[2] = s == warp + 2 * T2_PRODUCERS ? (int)ring.par : last[2];
                }
            }
            // Let the last copies into the owned stages land before the CTA
            // can exit (earlier ones were consumed).  A pair's copies complete
            // on its leader's barriers, and neither CTA exits before the other
            // (the cluster barrier below); where a wait ran out, the second
            // CTA allows its own copies a millisecond.
            if (crank == 0) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int s = warp + q * T2_PRODUCERS;
                    if (s >= stages || last[q] < 0) continue;
                    const long long t0 = clock64();
                    while (!mbar_try(&bar_full[s], (uint32_t)last[q]) && clock64() - t0 < WAIT_BUDGET) {}
                }
            } else if (!ok) {
                const long long t0 = clock64();
                while (clock64() - t0 < 2000000) {}
            }
        }
    } else if (warp == 2) {
        // ---------------- scheduler, score threshold ----------------
        // Lane 0 hands out the tiles; while the ring is full the warp renews
        // the threshold.
        const uint32_t peer_tile = PAIR ? cluster_addr(&sched_tile[0], 1) : 0;
        const uint32_t peer_sfull = PAIR ? cluster_addr(&bar_sfull[0], 1) : 0;
        unsigned pause = 500;
        bool done = false;   // all tiles are handed out (the threshold is renewed to the epilogue's end)
        long long t0 = clock64();
        for (int it = 0;;) {
            const int slot = it % TC_SCHED;
            const uint32_t sn = (uint32_t)(it / TC_SCHED);
            int ready = 0;   // 1: a tile was handed out, 2: no tile is left
            if (!done && crank == 0 && lane == 0 && mbar_try(&bar_sempty[slot], (sn & 1) ^ 1)) {
                const int t = atomicAdd(a.tile_counter, 1);
                const bool end = t >= a.ntiles;
                const int2 tile = end ? make_int2(0, 0) : make_int2((int)a.tiles[t], 1);
                sched_tile[slot] = tile;
                mbar_arrive(&bar_sfull[slot]);
                if constexpr (PAIR) cluster_post2(peer_tile + 8 * slot, peer_sfull + 8 * slot, tile.x, tile.y);
                ready = end ? 2 : 1;
            }
            ready = __shfl_sync(FULL, ready, 0);
            done = done || ready == 2;
            if (ready == 1) {
                ++it;
                t0 = clock64();
                continue;
            }
            int stop = 0;
            if (lane == 0) {
                if (!done && crank == 0 && clock64() - t0 > wt) {
                    *abort_flag = 1;
                    atomicOr(a.err, ERR_TIMEOUT);
                }
                stop = *abort_flag || *(volatile int *)&epi_end;
            }
            if (__shfl_sync(FULL, stop, 0)) break;
            if (MODE == MODE_TOPN) {
                const float thr = published_threshold(a.pub, (int)gridDim.x, a.pub_r, lane);
                if (lane == 0) *(volatile float *)&threshold = thr;
            }
            __nanosleep(pause);
            pause = min(pause + pause / 2, 4000u);
        }
    } else if (warp == 3) {
        if (crank == 0 && elect_one()) {
            // ---------------- MMA issue ----------------
            const uint32_t idesc = idesc_mxf4(PAIR ? 2 * TC_BM : TC_BM, PAIR ? 2 * T2_N : T2_N);
            const uint64_t descI = smem_desc_sw128(smem_u32(smem)), descJ = smem_desc_sw128(smem_u32(smem + TC_A_BYTES));
            const uint32_t one = tmem_base + T2_SCALE_COL, sj = one + (PAIR ? 2 * FP4_SCALE_COLS : 0);
            Ring ring;
            bool ok = true;
            const int Wt = a.Wt, W0 = a.W0;
            for (int it = 0; ok; ++it) {
                const int slot = it % TC_SCHED;
                const uint32_t sn = (uint32_t)(it / TC_SCHED);
                if (!mbar_wait(&bar_sfull[slot], sn & 1, abort_flag, a.err, wt)) break;
                const int more = sched_tile[slot].y;
                mbar_arrive(&bar_sempty[slot]);
                if (!more) break;
                const int b = it & 1;
                const uint32_t u = (uint32_t)(it >> 1);
                if (!mbar_wait(&bar_tempty[b], (u & 1) ^ 1, abort_flag, a.err, wt)) break;
                tc_fence_after();
                const uint32_t d0 = tmem_base + (uint32_t)(b * T2_BUF);
                for (int kc = 0; kc < nk; ++kc, ring.next(stages)) {
                    const int s = ring.s;
                    if (!mbar_wait(&bar_full[s], ring.par, abort_flag, a.err, wt)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t id = descI + (uint64_t)s * (T2_STAGE >> 4);
                    const uint64_t jd = descJ + (uint64_t)s * (T2_STAGE >> 4);
                    // Two words of 128 samples (K = 64 twice): cases, then
                    // controls (ENC 0: into the second accumulator; ENC 1: with
                    // scale 4096).
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int w = 2 * kc + h;
                        if (w < Wt) {
                            const bool ctrl = w >= W0;
                            const bool first = w == 0 || (!PAIR && w == W0);
                            const uint32_t d = d0 + (!PAIR && ctrl ? T2_N : 0);
                            const uint32_t si = one + (PAIR && ctrl ? FP4_SCALE_COLS : 0);
                            if constexpr (PAIR) {
                                mma_mxf4_pair(d, id + 4 * h, jd + 4 * h, idesc, si, sj, first ? 0u : 1u);
                                mma_mxf4_pair(d, id + 4 * h + 2, jd + 4 * h + 2, idesc, si, sj, 1u);
                            } else {
                                mma_mxf4(d, id + 4 * h, jd + 4 * h, idesc, si, sj, first ? 0u : 1u);
                                mma_mxf4(d, id + 4 * h + 2, jd + 4 * h + 2, idesc, si, sj, 1u);
                            }
                        }
                    }
                    if constexpr (PAIR) mma_commit_pair(&bar_empty[s]); else mma_commit(&bar_empty[s]);
                }
                if (ok) {
                    if constexpr (PAIR) mma_commit_pair(&bar_tfull[b]); else mma_commit(&bar_tfull[b]);
                }
            }
            // All MMAs issued by this thread complete before TMEM is released.
            if constexpr (PAIR) mma_commit_pair(&bar_done); else mma_commit(&bar_done);
            const long long t0 = clock64();
            while (!mbar_try(&bar_done, 0) && clock64() - t0 < WAIT_BUDGET) {}
        }
    } else {
        // ---------------- epilogue ----------------
        const int ew = warp - T2_EPI_WARP0;
        const int quarter = warp & 3;
        const int part = ew >> 2;                          // four SNPs j x = part, part + 4, .. of a tile
        const int g = lane & 1;                            // genotype of this lane's row
        const uint32_t tempty0 = PAIR ? cluster_addr(&bar_tempty[0], 0) : 0;
        const int L = a.L;
        float *ws = wscore + ew * TC_WBUF;
        uint64_t *wr = wrank + ew * TC_WBUF;
        uint2 *rec = recs + ew * T2_WARP_SNPS;
        const int S = (int)a.S;
        const float invN = a.invN * (1.f / a.scale);   // (exact: the scale is a power of two)
        const bool whole = a.rank_begin == 0 && a.rank_end >= a.pair_base;
        uint32_t all[3];   // genotype counts of SNP 0, whose sum is the classes
        unpack_marg(a.marg4[0], all);
        const uint32_t samples = all[0] + all[1] + all[2];
        // This warp's candidates, and the CTA list's last entry when the
        // warp last merged: a candidate has to beat it.
        int cnt = 0;
        float thr_s = -FLT_MAX;
        uint64_t thr_r = NO_RANK;
        // The least score of a candidate by now: that of the list's last entry
        // (which only rises; a racy read is a score it had at some time), and
        // the one that enough pairs of all CTAs are known to reach.
        auto floor_score = [&]() -> float {
            return fmaxf(*(volatile float *)(lscore + L - 1), *(volatile float *)&threshold);
        };
        auto merge = [&]() {
            // Sorted outside the lock, against the list's last score then.
            const float racy = *(volatile float *)(lscore + L - 1);
            const bool later = racy > thr_s;
            int m = sort_candidates(ws, wr, cnt, later ? racy : thr_s, later ? NO_RANK : thr_r, lane);
            cnt = 0;
            if (m == 0) return;
            bool held = true;
            if (lane == 0) {
                const long long t0 = clock64();
                while (atomicCAS(&list_lock, 0, 1) != 0) {
                    __nanosleep(100);
                    if (clock64() - t0 > WAIT_BUDGET) {
                        *abort_flag = 1;
                        atomicOr(a.err, ERR_TIMEOUT);
                        held = false;
                        break;
                    }
                }
                __threadfence_block();
            }
            held = __shfl_sync(FULL, held, 0);
            if (held) {
                // (What the threshold has passed meanwhile is left out.)
                const float now = floor_score();
                m = __popc(__ballot_sync(FULL, lane < m && ws[lane] >= now)) +
                    __popc(__ballot_sync(FULL, lane + 32 < m && ws[lane + 32] >= now));
                const int fill = merge_candidates(lscore, lrank, L, list_fill, ws, wr, m, lane);
                if (lane == 0) list_fill = fill;
                thr_s = lscore[L - 1];
                thr_r = lrank[L - 1];
                __threadfence_block();
                __syncwarp();
                if (lane == 0) {
                    if (lrank[a.pub_m - 1] != NO_RANK)
                        *(volatile int *)(a.pub + blockIdx.x) = ordered_int(lscore[a.pub_m - 1]);
                    __threadfence_block();
                    atomicExch(&list_lock, 0);
                }
            }
            __syncwarp();
        };
        // hs + (t(c), t(d)) for two packed cells c, d (a | b << 16, times 2^SH).
        auto add_terms = [&](F2 hs, uint32_t c, uint32_t d) -> F2 {
            // a 2^SH under the exponent of 2^(23 - SH) is 2^(23 - SH) + a, and -a q
            // = 2^(23 - SH) q minus q times that, exactly (q the scale, a power of
            // two).  The logarithm's argument is a q + 1e-30, that is a q, or
            // 1e-30 at a = 0, whose finite logarithm times 0 adds nothing.
            constexpr uint32_t EXP = SH == 2 ? 0x4A000000u : 0x4B000000u;
            constexpr float BIG = SH == 2 ? 2097152.f : 8388608.f;
            const F2 minus = f2(-1.f, -1.f), tiny = f2(1e-30f, 1e-30f);
            const F2 mscale = f2(-a.scale, -a.scale), big = f2(BIG * a.scale, BIG * a.scale);
            const F2 na = f2_fma(f2(__uint_as_float(__byte_perm(c, EXP, 0x7610)), __uint_as_float(__byte_perm(d, EXP, 0x7610))),
                                 mscale, big);
            const F2 nb = f2_fma(f2(__uint_as_float(__byte_perm(c, EXP, 0x7632)), __uint_as_float(__byte_perm(d, EXP, 0x7632))),
                                 mscale, big);
            const float2 aa = f2_split(f2_fma(na, minus, tiny)), bb = f2_split(f2_fma(nb, minus, tiny));
            // The byte offset of the table entry of n = a + b.
            auto xl = [&](uint32_t x) {
                return *reinterpret_cast<const float *>(reinterpret_cast<const char *>(xltab) +
                                                        __dp2a_lo(x, SH == 2 ? 0x00000101u : 0x00000404u, 0u));
            };
            F2 t = f2_fma(na, f2(lg2_approx(aa.x), lg2_approx(aa.y)), f2(xl(c), xl(d)));
            t = f2_fma(nb, f2(lg2_approx(bb.x), lg2_approx(bb.y)), t);
            return f2_add(hs, t);
        };
        bool ok = true;
        for (int it = 0;; ++it) {
            const int slot = it % TC_SCHED;
            const uint32_t sn = (uint32_t)(it / TC_SCHED);
            ok = mbar_wait(&bar_sfull[slot], sn & 1, abort_flag, a.err, wt);
            ok = __all_sync(FULL, ok);
            if (!ok) break;
            const int2 tile = sched_tile[slot];
            __syncwarp();
            if (lane == 0) slot_read(slot);
            if (!tile.y) break;
            const int b = it & 1;
            const uint32_t u = (uint32_t)(it >> 1);
            // Tile data that does not depend on the accumulators, loaded
            // while the tile's MMAs may still run.
            const int I = (int)((uint32_t)tile.x >> 16), j0 = (tile.x & 0xffff) * NJT;
            const int iw = T2_IB * ((PAIR ? 2 : 1) * I + (int)crank) + quarter * 16;   // this warp's first SNP i
            const int i = iw + (lane >> 1);
            const bool iv = i < S;
            // This warp's fours of SNPs j, x = part + 4 r, r0 <= r < r1, that
            // hold some valid pair: their last j after the warp's first i,
            // their first j before S.
            const int xlo = j0 + 3 > iw ? 0 : (iw - j0 - 3) / 4 + 1;
            const int xhi = iw < S ? min(NJT / 4, (S - j0 + 3) / 4) : 0;
            const int r0 = xlo > part ? (xlo - part + T2_PARTS - 1) / T2_PARTS : 0;
            const int r1 = xhi > part ? (xhi - part + T2_PARTS - 1) / T2_PARTS : 0;
            // Every cell has to be a count (it is a table offset): where i is
            // no SNP its rows are zero, those of a SNP of genotype 2
            // throughout.  Genotypes of i in the order g, 1 - g.
            uint32_t Ti[3] = {0, 0, samples << SH};
            uint64_t rb = 0;   // rank of (i, j) less j
            if (iv) {
                uint32_t T[3];
                unpack_marg(a.marg4[i], T);
                Ti[0] = (g ? T[1] : T[0]) << SH;
                Ti[1] = (g ? T[0] : T[1]) << SH;
                Ti[2] = T[2] << SH;
                const uint64_t si = (uint64_t)(S - i);
                rb = a.pair_base - si * (si - 1) / 2 - (uint64_t)i - 1;
            }
            __syncwarp();
            if (lane < T2_WARP_SNPS) {
                // Counts of genotypes 0 and 1 of SNP j, a lane per SNP; no
                // samples where j is no SNP (its rows are zero).
                const int j = j0 + 4 * (part + T2_PARTS * (lane >> 2)) + (lane & 3);
                uint32_t T[3] = {0, 0, 0};
                if (j < S) unpack_marg(a.marg4[j], T);
                rec[lane] = make_uint2(T[0] << SH, T[1] << SH);
            }
            ok = mbar_wait(&bar_tfull[b], u & 1, abort_flag, a.err, wt);
            ok = __all_sync(FULL, ok);   // (also orders the records)
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * T2_BUF + 8 * part);
            auto release = [&]() {
                // This warp's last read of the buffer.
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if constexpr (PAIR) mbar_arrive_cluster(tempty0 + 8 * b);
                    else mbar_arrive(&bar_tempty[b]);
                }
            };
            // Read again whenever a pair passes what was read before.
            float thr = MODE == MODE_TOPN ? floor_score() : 0.f;
            const uint32_t after = iv ? (uint32_t)(S - 1 - i) : 0u;   // SNPs j after i
            if (r0 >= r1) release();
            for (int r = r0; r < r1; ++r) {
                uint32_t v[8];
                {
                    uint32_t w[8];
                    tmem_ld8(taddr + 8 * T2_PARTS * r, v);
                    if constexpr (!PAIR) tmem_ld8(taddr + T2_N + 8 * T2_PARTS * r, w);
                    tmem_wait_ld();
                    tmem_regs_after_wait(v);
                    if constexpr (!PAIR) tmem_regs_after_wait(w);
#pragma unroll
                    for (int x = 0; x < 8; ++x) {
                        if constexpr (PAIR) v[x] = unpack_enc(v[x]);
                        else v[x] = pack_exact(v[x], w[x]);
                    }
                }
                if (r + 1 == r1) release();
                // SNPs 2 e and 2 e + 1 of the four: this lane's is 2 e + g.
                float score[2];
                const int j = j0 + 4 * (part + T2_PARTS * r) + g;   // (that of e = 0)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const uint2 Tj = rec[4 * r + 2 * e + g];
                    uint32_t R[2][2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        R[0][h] = g ? v[4 * e + 2 + h] : v[4 * e + h];
                        R[1][h] = __shfl_xor_sync(FULL, g ? v[4 * e + h] : v[4 * e + 2 + h], 1);
                    }
                    const uint32_t c02 = Ti[0] - R[0][0] - R[0][1], c12 = Ti[1] - R[1][0] - R[1][1];
                    const uint32_t c20 = Tj.x - R[0][0] - R[1][0], c21 = Tj.y - R[0][1] - R[1][1];
                    const uint32_t c22 = Ti[2] - c20 - c21;
                    F2 hs[2] = {f2(0.f, 0.f), f2(0.f, 0.f)};
                    hs[0] = add_terms(hs[0], R[0][0], R[0][1]);
                    hs[1] = add_terms(hs[1], R[1][0], R[1][1]);
                    hs[0] = add_terms(hs[0], c02, c12);
                    hs[1] = add_terms(hs[1], c20, c21);
                    hs[0] = add_terms(hs[0], c22, 0u);   // (a cell of no sample adds 0)
                    const float2 h2 = f2_split(f2_add(hs[0], hs[1]));
                    score[e] = fmaf(-LN2F * (h2.x + h2.y), invN, a.hy);
                    if (MODE == MODE_DUMP && (uint32_t)(j + 2 * e - i - 1) < after) {
                        const size_t at = (size_t)i * (size_t)S + (size_t)(j + 2 * e);
                        if (a.dump_scores) a.dump_scores[at] = score[e];
                        if (a.dump_tables) {
                            const uint32_t c[9] = {R[g][0], R[g][1], g ? c12 : c02, R[1 - g][0], R[1 - g][1], g ? c02 : c12,
                                                   c20, c21, c22};
                            uint32_t *o = a.dump_tables + at * 18;
#pragma unroll
                            for (int x = 0; x < 9; ++x) {
                                o[2 * x] = (c[x] & 0xffffu) >> SH;
                                o[2 * x + 1] = c[x] >> (16 + SH);
                            }
                        }
                    }
                }
                if (MODE == MODE_TOPN) {
                    // Few pairs reach the threshold: one vote for both scores,
                    // and ranks only after it.
                    bool near[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) near[e] = (uint32_t)(j + 2 * e - i - 1) < after && score[e] >= thr;
                    if (__any_sync(FULL, near[0] || near[1])) {
                        thr = floor_score();
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const uint64_t rank = rb + (uint64_t)(j + 2 * e);
                            const bool cand = near[e] && score[e] >= thr && (whole || (rank >= a.rank_begin && rank < a.rank_end)) &&
                                              better(score[e], rank, thr_s, thr_r);
                            const unsigned mk = __ballot_sync(FULL, cand);
                            if (mk == 0) continue;
                            if (cand) {
                                const int p = cnt + __popc(mk & ((1u << lane) - 1u));
                                ws[p] = score[e];
                                wr[p] = rank;
                            }
                            cnt += __popc(mk);
                            __syncwarp();
                            if (cnt > TC_WBUF - 32) merge();
                        }
                    }
                }
            }
        }
        if (MODE == MODE_TOPN) {
            // The CTA's list (after a wait that ran out, as far as it got: the
            // search fails).
            if (ok) merge();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_epi);
            mbar_wait(&bar_epi, 0, abort_flag, a.err, wt);
            for (int x = threadIdx.x - 32 * T2_EPI_WARP0; x < L; x += T2_EPI_THREADS) {
                a.list_score[(size_t)blockIdx.x * L + x] = lscore[x];
                a.list_rank[(size_t)blockIdx.x * L + x] = lrank[x];
            }
        }
        if (ew == 0 && lane == 0) *(volatile int *)&epi_end = 1;
    }

    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) {
        // Neither CTA of a pair leaves while the other may still signal it or
        // an MMA may read its shared memory (the leader has waited for its
        // last commit above).
        if (crank == 1 && threadIdx.x == 0) {
            const long long t0 = clock64();
            while (!mbar_try(&bar_done, 0) && clock64() - t0 < WAIT_BUDGET) {}
        }
        __syncwarp();
        cluster_sync();
    }
    if (warp == 3) {
        tc_fence_after();
        if constexpr (PAIR)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TC_TMEM_COLS)
                         : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TC_TMEM_COLS)
                         : "memory");
    }
}

}  // namespace

int pairs_rows_i(int enc) { return (enc ? 2 : 1) * T2_IB; }
int pairs_rows_j(int enc) { return (enc ? 2 : 1) * T2_NJ; }
int pairs_block_rows() { return T2_N; }

size_t pairs_smem_bytes(int stages, int M, int L)
{
    // 1 KiB for the alignment of the stages; the list and the warps' buffers
    // where there is a list.
    return 1024 + TC_STATIC_SMEM + (size_t)(M + 1) * 4 + (size_t)stages * T2_STAGE + (size_t)T2_EPI_WARPS * T2_WARP_SNPS * 8 +
           (L > 0 ? (size_t)(L + T2_EPI_WARPS * TC_WBUF) * (8 + 4) : 0);
}

int pairs_stages(int M, int L, size_t smem_cap)
{
    for (int st = TC_MAX_STAGES; st >= 2; --st)
        if (pairs_smem_bytes(st, M, L) <= smem_cap) return st;
    return 0;
}

cudaError_t launch_marginals(const uint4 *X, int64_t S, int64_t S_pad, int W0, int Wt, uint16_t *marg,
                             cudaStream_t st)
{
    k_marginals<<<(unsigned)((S + 127) / 128), 128, 0, st>>>(X, S, S_pad, W0, Wt, marg);
    return cudaGetLastError();
}

cudaError_t launch_pairs_tc(int mode, const CUtensorMap &tmapI, const CUtensorMap &tmapJ, const PairsArgs &a, int grid,
                            cudaStream_t st)
{
    // (The pipeline's arrays and addresses hold for two stages and more.)
    if (a.stages < 2 || a.stages > TC_MAX_STAGES) return cudaErrorInvalidValue;
    const size_t bytes = pairs_smem_bytes(a.stages, a.M, a.L) - TC_STATIC_SMEM;
    void *fn = mode == MODE_TOPN ? (a.enc ? reinterpret_cast<void *>(&k_pairs_tc<MODE_TOPN, 1>)
                                          : reinterpret_cast<void *>(&k_pairs_tc<MODE_TOPN, 0>))
                                 : (a.enc ? reinterpret_cast<void *>(&k_pairs_tc<MODE_DUMP, 1>)
                                          : reinterpret_cast<void *>(&k_pairs_tc<MODE_DUMP, 0>));
    cudaError_t e = allow_dynamic_smem(fn, bytes);
    if (e != cudaSuccess) return e;
    CUtensorMap mI = tmapI, mJ = tmapJ;
    PairsArgs args = a;
    void *params[] = {&mI, &mJ, &args};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(T2_THREADS);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    if (a.enc) {
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
    }
    return cudaLaunchKernelExC(&cfg, fn, params);
}

}  // namespace fc
