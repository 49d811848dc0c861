// Order-3 exhaustive search on the fifth-generation tensor cores (tcgen05).
//
// For a combination (i, j, l) the cells with all three genotypes in {0, 1}
// are, per class c (Section "Computing the contingency tables": a cell is
// the population count of the AND of one row of each SNP's table),
//     n_c(a, b, g) = sum_{m in c} [G_i(m) = a] [G_j(m) = b] [G_l(m) = g]
//                  = < P_c[(i, j), (a, b)], E_c[l, g] >,
// the dot product over the samples of a pair row P = E[i, a] AND E[j, b]
// with a SNP row E[l, g].  Rows are packed 0/1 e2m1 nibbles; for one block of
// SNPs l and one block of pairs (i, j) with a fixed i the dot products are one
// tcgen05.mma kind::mxf4 tile, exact (fc_tc.cuh).  The other 19 cells of the
// 3 x 3 x 3 table follow exactly by inclusion-exclusion from the restricted
// pair table and the per-SNP genotype counts (the three rows of a SNP's
// table partition the samples).  The epilogue scores every combination with
// the FP32 mutual information and keeps a CTA top list; no count is written
// to memory.
//
// Two forms (template ENC):
//   ENC = 1: control samples carry the block scale 4096, so one accumulator
//            holds n_case + 4096 n_ctrl (exact while both classes have at
//            most 4095 samples); a tile of 128 SNPs l and 56 pairs is worked
//            on by a pair of CTAs (cta_group::2, M = 256, N = 224): each
//            loads 64 SNPs and 28 pairs and scores its SNPs against all 56
//            pairs;
//   ENC = 0: the case and control samples accumulate into two accumulators;
//            a tile of 64 SNPs and 28 pairs per CTA (M = 128, N = 112).
// Either way a CTA's stage is 128 + 112 rows, a tile takes 224 TMEM columns,
// and two tiles are in flight.  What bounds the kernel is the scoring, about
// 400 instructions per 32 combinations: 1,000 SNPs x 4,000 samples take 4.56 ms,
// 701 x 9,001 2.49, a search with its tail 4.7 and 2.6 (5.9 and 6.5 with byte rows
// and both genotypes of a SNP from different tiles); at 500 SNPs 1.8 instructions
// are issued a cycle and the tensor pipe is 31 % active.  Parts left out, when the
// first search took 5.3 ms (its selection and merges were slower): the tiles alone
// were 1.9 ms, the logarithms 0.95, the table reads 0.86 and the exchange of the
// cells 0.45.  (One CTA per 128 x 24 tile with both genotypes of a SNP in one lane
// needed no exchange of cells, but 1,000 bytes of shared memory per combination
// against about 530 here: 5.2 ms then, but 3.9 ms instead of 2.9 for the second.
// 12 epilogue warps with more registers: 5.5 and 3.2 ms.)
//
// The pair rows live in a slab in device memory, the paper's `combine` of
// two genotype tables done once per data set (k_pair_rows): for each first
// SNP i, the rows of its pairs (i, j), j = i + 1 + jo, row 4 jo + 2 a + b, zero
// where j >= S.  A tile is (i, the block of SNPs j from j0 = i + 1 + NP J', the
// SNPs l from l0 = j0 + 1 + LB L'): blocks start right after the SNPs before
// them; a warp whose 16 SNPs l are all at or before the SNPs j of two pairs,
// or beyond the last SNP, skips them.  Forming the rows on chip instead (TMA of
// the rows of the SNPs j, AND with the rows of SNP i in shared memory) was
// measured slower: the builder's shared-memory traffic cost more than the
// slab's one-time write.
//
// TMEM lane 2 l + g holds genotype g of SNP l, columns 4 q + 2 a + b the cells of
// pair q.  The two lanes of a SNP take two pairs at a time, one each: they
// exchange the four cells of the other's pair, and lane g reads its cells with
// the genotypes of l in the order g, 1 - g (every table of l is swapped alike),
// so that nothing is put back in order.  Counts come times four (the block
// scale of the pair rows is 4; still exact): a packed count n is then the byte
// offset of its table entry.
//
// The epilogue scores each cell, in bits, as t(a, b) = xl[n] - a lg2~(a) - b
// lg2~(b) = a log2(n/a) + b log2(n/b) (a, b the class counts, n = a + b), and
// MI = H(Y) - ln 2 sum t / N, where xl is a shared-memory table of x log2 x over
// the sample counts (entries correctly rounded) and lg2~ the hardware base-2
// logarithm, with |lg2~(x) - log2 x| <= 2^-22 max(1, |log2 x|) (absolute within
// [1/2, 2], relative elsewhere; a test checks it on the device for every count
// up to 2^17 under every scale below; fc_log2_approx_scaled).  Counts are scored times the power of two
// 2^-s, s = floor(log2 M) - 2 (the sum times 2^s is the same): the logarithms of
// the fullest cells are then near 0, and with them the roundings, while no
// |log2 x| exceeds log2 M.  Errors of 27-cell scores against FP64 (rms, 4,000
// and 8,190 samples): 2.1e-7 and 2.8e-7 unscaled, 0.8e-7 and
// 0.7e-7 scaled.
// One table read per cell instead of two relieves shared memory, and taking
// the two smaller of the three terms from the logarithm instead of the
// largest lowers the error.  With u = 2^-24 (so 2^-22 = 4u) and in bits, a cell
// errs by at most u n log2 M from the table entry, 4u (a + b) (log2 M + 1) from
// the logarithms and 2 u n log2 M from the two fused multiply-subtracts; over
// the 27 cells (sum n = N), the 27 accumulations (partial sums <= N), the
// product with ln 2 and the final scaling this gives, in nats, |MI32 - MI| <= u
// (7 ln M + 37 ln 2), which the FP64 rescoring window of the library covers
// (twice the larger of this and the sweep's bound).
//
// Candidates: each epilogue warp keeps its own buffer of 64; when it cannot
// take another 32 the warp merges it into the CTA's sorted list under a lock.
// No barrier joins the epilogue warps between the first and the last tile (a
// shared buffer took two barriers per tile and two more every third group of
// pairs).  Merging is kept rare by a threshold over all CTAs: each publishes
// the score of one entry m - 1 of its list (m about 2 L / CTAs), and a score
// that the entries of L / m CTAs reach is reached by L combinations, so lower
// ones need no place in any list; the scheduler warp looks for it while it
// waits.  (With each CTA's own list alone, a CTA took about L (1 + ln(n / L))
// of its n combinations, and merging them a third of the time at 500 SNPs.)
//
// Roles (one persistent CTA per SM, 640 threads):
//   warps 0, 1 : TMA producers (128-byte K chunks, 256 samples, of the 128 SNP
//                rows and 112 pair rows), warp w owning the stages s = w (mod 2)
//   warp 2     : schedules the tiles (ENC 1: in the pair's leader), score
//                threshold
//   warp 3     : TMEM allocation; one elected lane (ENC 1: of the pair's
//                leader) issues the MMAs
//   warps 4-19 : epilogue, four warps per TMEM lane quarter, each taking every
//                fourth two pairs of a tile
#include <algorithm>

#include "fc_candidates.cuh"
#include "fc_ie.cuh"

namespace fc {

namespace {

constexpr int T3_PRODUCERS = 2;
constexpr int T3_MAX_STAGES = 6;
constexpr int T3_EPI_WARP0 = 4;
constexpr int T3_EPI_WARPS = 16;
constexpr int T3_PARTS = T3_EPI_WARPS / 4;         // epilogue warps per TMEM lane quarter
constexpr int T3_EPI_THREADS = 32 * T3_EPI_WARPS;
constexpr int T3_THREADS = 32 * T3_EPI_WARP0 + T3_EPI_THREADS;
static_assert(T3_EPI_WARP0 % 4 == 0, "epilogue warp w reads TMEM lane quarter w % 4");
constexpr int T3_NP = 28;                          // pairs (i, j) per stage
constexpr int T3_N = 4 * T3_NP;                    // pair rows per stage
constexpr int T3_LB = 64;                          // SNPs l per CTA and tile
constexpr uint32_t T3_STAGE = TC_A_BYTES + (uint32_t)T3_N * TC_BK;
static_assert(T3_STAGE % 1024 == 0, "swizzled stages");
constexpr int T3_BUF = 2 * T3_N;                   // TMEM columns of a tile
constexpr uint32_t T3_SCALE_COL = 2 * T3_BUF;      // TMEM column of scale 1, then of 4096, then of 4
static_assert(T3_SCALE_COL + 3 * FP4_SCALE_COLS <= TC_TMEM_COLS, "scales behind the accumulators");
__host__ __device__ constexpr int t3_warp_pairs(int enc)   // pairs of a tile per warp, at most
{
    return 2 * (((enc ? 2 : 1) * T3_NP / 2 + T3_PARTS - 1) / T3_PARTS);
}
constexpr int T3_WBUF_SHORT = 40;                  // a warp's buffer where one of TC_WBUF does not fit
static_assert(T3_WBUF_SHORT > 32, "a round's 32 candidates fit after a merge");
constexpr int T3_REC_WORDS = 12;                   // per pair: T01[9], rank base (2 words)
static_assert(T3_REC_WORDS % 4 == 0, "records of uint4");
static_assert(t3_warp_pairs(1) <= 32, "a lane per pair record");

__device__ __forceinline__ uint64_t c3(uint64_t n) { return n * (n - 1) * (n - 2) / 6; }   // 0 for n < 3
__device__ __forceinline__ uint64_t c2(uint64_t n) { return n * (n - 1) / 2; }             // 0 for n < 2

// BATCH: the items of several jobs (T3Job), job-major, in one launch.
template <int MODE, int ENC, bool BATCH>
__global__ void __launch_bounds__(T3_THREADS, 1)
    k_triples_tc(const __grid_constant__ CUtensorMap tmapA, const __grid_constant__ CUtensorMap tmapP, TriplesArgs a)
{
    static_assert(!BATCH || MODE == MODE_TOPN, "the batched launch searches");
    constexpr bool PAIR = ENC == 1;                 // a tile per CTA pair
    constexpr int NPT = PAIR ? 2 * T3_NP : T3_NP;   // pairs per tile
    constexpr int WPAIRS = t3_warp_pairs(ENC);
    const int wbuf = PAIR ? TC_WBUF : a.wbuf;       // candidates of a warp's buffer
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_full[T3_MAX_STAGES], bar_empty[T3_MAX_STAGES];
    __shared__ uint64_t bar_tfull[2], bar_tempty[2], bar_done, bar_epi;
    __shared__ uint32_t tmem_base_slot;
    __shared__ uint64_t bar_sfull[TC_SCHED], bar_sempty[TC_SCHED];
    // Tiles {rowP, i | j0 << 16, l0, job (0 where there are none; -1: no more
    // tiles)}.
    __shared__ uint4 sched_tile[TC_SCHED];
    __shared__ int abort_flag_s;
    __shared__ int list_lock, list_fill;
    __shared__ int epi_job;          // job of the tile that the epilogue's first warp took last, -2 at the end
    // published_threshold: job in the high half, score bits in the low one
    // (read and written as one word).
    __shared__ unsigned long long threshold;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int stages = a.stages;
    const uint32_t crank = PAIR ? cluster_rank() : 0;   // CTA of the pair (0: its leader)
    volatile int *abort_flag = &abort_flag_s;

    // The x log2 x table first (a constant base saves an addition per read);
    // then the stages, 1024-byte aligned, the warps' pair records (16-byte
    // aligned), the candidate list and the warps' buffers (ranks before
    // scores).
    float *xltab = reinterpret_cast<float *>(smem_raw);
    uint8_t *smem = reinterpret_cast<uint8_t *>(((uintptr_t)(xltab + a.M + 1) + 1023) & ~(uintptr_t)1023);
    uint32_t *recs = reinterpret_cast<uint32_t *>(smem + (size_t)stages * T3_STAGE);
    uint64_t *lrank = reinterpret_cast<uint64_t *>(recs + T3_EPI_WARPS * WPAIRS * T3_REC_WORDS);
    uint64_t *wrank = lrank + a.L;
    float *lscore = reinterpret_cast<float *>(wrank + T3_EPI_WARPS * wbuf);
    float *wscore = lscore + a.L;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&bar_full[s], 1);
            mbar_init(&bar_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bar_tfull[b], 1);
            mbar_init(&bar_tempty[b], (PAIR ? 2 : 1) * T3_EPI_WARPS);
        }
        mbar_init(&bar_done, 1);
        mbar_init(&bar_epi, T3_EPI_WARPS);
        for (int s = 0; s < TC_SCHED; ++s) {
            mbar_init(&bar_sfull[s], 1);
            // The MMA thread, and the producer and epilogue warps (of both
            // CTAs of a pair).
            mbar_init(&bar_sempty[s], 1 + (PAIR ? 2 : 1) * (T3_PRODUCERS + T3_EPI_WARPS));
        }
        abort_flag_s = 0;
        list_lock = 0;
        list_fill = 0;
        epi_job = -1;
        threshold = ~0ull << 32;
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
    if (warp >= T3_EPI_WARP0 && warp < T3_EPI_WARP0 + 4) {
        const uint32_t q = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + T3_SCALE_COL;
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

    // A consumer's word that it has read a slot of the tile ring.
    const uint32_t sempty0 = PAIR ? cluster_addr(&bar_sempty[0], 0) : 0;
    auto slot_read = [&](int slot) {
        if constexpr (PAIR) mbar_arrive_cluster(sempty0 + 8 * slot);
        else mbar_arrive(&bar_sempty[slot]);
    };

    if (warp < T3_PRODUCERS) {
        // ---------------- TMA producers ----------------
        if (elect_one()) {
            Ring ring;
            int owner = 0;   // producer of stage ring.s
            // Parity of the last fill issued into each owned stage (at most
            // three: stages warp, warp + 2, warp + 4), -1 before the first.
            int last[3] = {-1, -1, -1};
            auto step = [&]() {
                ring.next(stages);
                owner = ring.s == 0 || owner + 1 == T3_PRODUCERS ? 0 : owner + 1;
            };
            bool ok = true;
            const CUtensorMap *mapA = &tmapA, *mapP = &tmapP;
            int nk = (a.Wt + 1) / 2, cur_job = -1;
            for (int it = 0; ok; ++it) {
                const int slot = it % TC_SCHED;
                const uint32_t sn = (uint32_t)(it / TC_SCHED);
                if (!mbar_wait(&bar_sfull[slot], sn & 1, abort_flag, a.err, wt)) { ok = false; break; }
                const uint4 tile = sched_tile[slot];
                slot_read(slot);
                const int job = (int)tile.w;
                if (job < 0) break;
                if (BATCH && job != cur_job) {
                    cur_job = job;
                    const T3Job *jb = a.jobs + job;
                    mapA = jb->tmapA;
                    mapP = jb->tmapP;
                    nk = (jb->Wt + 1) / 2;
                }
                const int rowA = 2 * ((int)tile.z + T3_LB * (int)crank), rowP = (int)tile.x + T3_N * (int)crank;
                for (int kc = 0; kc < nk; ++kc, step()) {
                    if (owner != warp) continue;
                    const int s = ring.s;
                    uint8_t *st = smem + (size_t)s * T3_STAGE;
                    if (!mbar_wait(&bar_empty[s], ring.par ^ 1, abort_flag, a.err, wt)) { ok = false; break; }
                    const int x = kc * TC_BK;
                    if constexpr (PAIR) {
                        // The leader's barrier counts the bytes of both CTAs.
                        if (crank == 0) mbar_expect_tx(&bar_full[s], 2 * T3_STAGE);
                        tma_load_2d_pair(mapA, &bar_full[s], st, x, rowA);
                        tma_load_2d_pair(mapP, &bar_full[s], st + TC_A_BYTES, x, rowP);
                    } else {
                        mbar_expect_tx(&bar_full[s], T3_STAGE);
                        tma_load_2d(mapA, &bar_full[s], st, x, rowA);
                        tma_load_2d(mapP, &bar_full[s], st + TC_A_BYTES, x, rowP);
                    }
                    last[0] = s == warp ? (int)ring.par : last[0];
                    last[1] = s == warp + T3_PRODUCERS ? (int)ring.par : last[1];
                    last[2] = s == warp + 2 * T3_PRODUCERS ? (int)ring.par : last[2];
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
                    const int s = warp + q * T3_PRODUCERS;
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
        // the threshold of the job that the epilogue works on.  In a batched
        // launch: the job of the last item taken and its items [s_first,
        // s_end); items only grow.
        int s_job = BATCH ? -1 : 0, s_first = 0, s_end = 0;
        const uint4 *tiles = a.tiles;
        const int n_items = BATCH ? a.n_items : a.ntiles;
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
                int t = atomicAdd(a.tile_counter, 1);
                const bool end = t >= n_items;
                if (BATCH && !end) {
                    if (t >= s_end) {
                        // The last job whose first item is at most t.
                        int lo = s_job < 0 ? 0 : s_job, hi = a.n_jobs - 1;
                        while (lo < hi) {
                            const int mid = (lo + hi + 1) >> 1;
                            if (a.jobs[mid].item_first <= t) lo = mid; else hi = mid - 1;
                        }
                        s_job = lo;
                        s_first = a.jobs[lo].item_first;
                        s_end = s_first + a.jobs[lo].ntiles;
                        tiles = a.jobs[lo].tiles;
                    }
                    t -= s_first;
                }
                uint4 tile = end ? make_uint4(0, 0, 0, 0) : tiles[t];
                tile = make_uint4(tile.x, tile.y | tile.z << 16, tile.w, end ? ~0u : (uint32_t)s_job);
                sched_tile[slot] = tile;
                mbar_arrive(&bar_sfull[slot]);
                if constexpr (PAIR) cluster_post4(peer_tile + 16 * slot, peer_sfull + 8 * slot, tile);
                ready = end ? 2 : 1;
            }
            ready = __shfl_sync(FULL, ready, 0);
            done = done || ready == 2;
            if (ready == 1) {
                ++it;
                t0 = clock64();
                continue;
            }
            const int job = __shfl_sync(FULL, *(volatile int *)&epi_job, 0);
            int stop = 0;
            if (lane == 0) {
                if (!done && crank == 0 && clock64() - t0 > wt) {
                    *abort_flag = 1;
                    atomicOr(a.err, ERR_TIMEOUT);
                }
                stop = *abort_flag || job == -2;
            }
            if (__shfl_sync(FULL, stop, 0)) break;
            if (MODE == MODE_TOPN) {
                if (job >= 0) {
                    const int *pub = a.pub + (size_t)(BATCH ? a.jobs[job].slot : 0) * gridDim.x;
                    const float thr = published_threshold(pub, (int)gridDim.x, a.pub_r, lane);
                    if (lane == 0)
                        *(volatile unsigned long long *)&threshold = (unsigned long long)job << 32 | __float_as_uint(thr);
                }
            }
            __nanosleep(pause);
            pause = min(pause + pause / 2, 4000u);
        }
    } else if (warp == 3) {
        if (crank == 0 && elect_one()) {
            // ---------------- MMA issue ----------------
            const uint32_t idesc = idesc_mxf4(PAIR ? 2 * TC_BM : TC_BM, PAIR ? 2 * T3_N : T3_N);
            const uint64_t descA = smem_desc_sw128(smem_u32(smem)), descB = smem_desc_sw128(smem_u32(smem + TC_A_BYTES));
            const uint32_t one = tmem_base + T3_SCALE_COL, four = one + 2 * FP4_SCALE_COLS;
            Ring ring;
            bool ok = true;
            int Wt = a.Wt, W0 = a.W0, cur_job = -1;
            for (int it = 0; ok; ++it) {
                const int slot = it % TC_SCHED;
                const uint32_t sn = (uint32_t)(it / TC_SCHED);
                if (!mbar_wait(&bar_sfull[slot], sn & 1, abort_flag, a.err, wt)) break;
                const int job = (int)sched_tile[slot].w;
                mbar_arrive(&bar_sempty[slot]);
                if (job < 0) break;
                if (BATCH && job != cur_job) {
                    cur_job = job;
                    Wt = a.jobs[job].Wt;
                    W0 = a.jobs[job].W0;
                }
                const int b = it & 1;
                const uint32_t u = (uint32_t)(it >> 1);
                if (!mbar_wait(&bar_tempty[b], (u & 1) ^ 1, abort_flag, a.err, wt)) break;
                tc_fence_after();
                const uint32_t d0 = tmem_base + (uint32_t)(b * T3_BUF);
                for (int kc = 0; 2 * kc < Wt; ++kc, ring.next(stages)) {
                    const int s = ring.s;
                    if (!mbar_wait(&bar_full[s], ring.par, abort_flag, a.err, wt)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t ad = descA + (uint64_t)s * (T3_STAGE >> 4);
                    const uint64_t bd = descB + (uint64_t)s * (T3_STAGE >> 4);
                    // Two words of 128 samples (K = 64 twice): cases, then
                    // controls (ENC 0: into the second accumulator; ENC 1: with
                    // scale 4096).
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int w = 2 * kc + h;
                        if (w < Wt) {
                            const bool ctrl = w >= W0;
                            const bool first = w == 0 || (!PAIR && w == W0);
                            const uint32_t d = d0 + (!PAIR && ctrl ? T3_N : 0);
                            const uint32_t sa = one + (PAIR && ctrl ? FP4_SCALE_COLS : 0);
                            if constexpr (PAIR) {
                                mma_mxf4_pair(d, ad + 4 * h, bd + 4 * h, idesc, sa, four, first ? 0u : 1u);
                                mma_mxf4_pair(d, ad + 4 * h + 2, bd + 4 * h + 2, idesc, sa, four, 1u);
                            } else {
                                mma_mxf4(d, ad + 4 * h, bd + 4 * h, idesc, sa, four, first ? 0u : 1u);
                                mma_mxf4(d, ad + 4 * h + 2, bd + 4 * h + 2, idesc, sa, four, 1u);
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
        const int ew = warp - T3_EPI_WARP0;
        const int quarter = warp & 3;
        const int part = ew >> 2;                          // two pairs dp = part, part + 4, .. of a tile
        const int g = lane & 1;                            // genotype of this lane's row
        const uint32_t tempty0 = PAIR ? cluster_addr(&bar_tempty[0], 0) : 0;
        const int L = a.L;
        float *ws = wscore + ew * wbuf;
        uint64_t *wr = wrank + ew * wbuf;
        uint32_t *rec = recs + ew * (WPAIRS * T3_REC_WORDS);
        // The job of the tile (a batched launch reads the job's data again with
        // each tile: kept, they cost the scoring loop its registers).
        int cur_job = BATCH ? -1 : 0;
        const float unscale = 1.f / a.scale;   // (exact)
        const bool whole = BATCH || (a.rank_begin == 0 && a.rank_end >= a.total);
        // This warp's candidates, and the CTA list's last entry when the
        // warp last merged: a candidate has to beat it.
        int cnt = 0;
        float thr_s = -FLT_MAX;
        uint64_t thr_r = NO_RANK;
        // The least score of a candidate by now: that of the list's last entry
        // (which only rises; a racy read is a score it had at some time), and
        // the one that enough combinations of all CTAs are known to reach.
        auto published = [&]() -> float {
            const unsigned long long t2 = *(volatile unsigned long long *)&threshold;
            return (int)(t2 >> 32) == cur_job ? __uint_as_float((uint32_t)t2) : -FLT_MAX;
        };
        auto floor_score = [&]() -> float { return fmaxf(*(volatile float *)(lscore + L - 1), published()); };
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
                        *(volatile int *)(a.pub + (size_t)(BATCH ? a.jobs[cur_job].slot : 0) * gridDim.x + blockIdx.x) = ordered_int(lscore[a.pub_m - 1]);
                    __threadfence_block();
                    atomicExch(&list_lock, 0);
                }
            }
            __syncwarp();
        };
        // All epilogue warps meet, unless a wait ran out in some role.
        uint32_t epi_par = 0;
        auto meet = [&]() -> bool {
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_epi);
            const bool met = mbar_wait(&bar_epi, epi_par, abort_flag, a.err, wt);
            epi_par ^= 1;
            return __all_sync(FULL, met);
        };
        // The CTA's list of the current job, written out as the list of its
        // slot of
        // this CTA (all epilogue warps).
        auto flush = [&]() -> bool {
            merge();
            if (!meet()) return false;
            const size_t o = ((size_t)(BATCH ? a.jobs[cur_job].slot : 0) * gridDim.x + blockIdx.x) * L;
            for (int x = threadIdx.x - 32 * T3_EPI_WARP0; x < L; x += T3_EPI_THREADS) {
                a.list_score[o + x] = lscore[x];
                a.list_rank[o + x] = lrank[x];
                lscore[x] = -FLT_MAX;
                lrank[x] = NO_RANK;
            }
            if (ew == 0 && lane == 0) list_fill = 0;
            thr_s = -FLT_MAX;
            thr_r = NO_RANK;
            return meet();
        };
        // hs + (t(c), t(d)) for two packed cells c, d (4 a | 4 b << 16).
        auto add_terms = [&](F2 hs, uint32_t c, uint32_t d) -> F2 {
            // 4 a under the exponent of 2^21 is 2^21 + a; -a q = 2^21 q minus q
            // times that, exactly (q the scale, a power of two).  The logarithm's
            // argument is a q + 1e-30, that is a q, or 1e-30 at a = 0, whose
            // finite logarithm times 0 adds nothing.
            const F2 minus = f2(-1.f, -1.f), tiny = f2(1e-30f, 1e-30f);
            const F2 mscale = f2(-a.scale, -a.scale), big = f2(2097152.f * a.scale, 2097152.f * a.scale);
            const F2 na = f2_fma(f2(__uint_as_float(__byte_perm(c, 0x4A000000u, 0x7610)),
                                    __uint_as_float(__byte_perm(d, 0x4A000000u, 0x7610))), mscale, big);
            const F2 nb = f2_fma(f2(__uint_as_float(__byte_perm(c, 0x4A000000u, 0x7632)),
                                    __uint_as_float(__byte_perm(d, 0x4A000000u, 0x7632))), mscale, big);
            const float2 aa = f2_split(f2_fma(na, minus, tiny)), bb = f2_split(f2_fma(nb, minus, tiny));
            // 4 n = 4 a + 4 b is the byte offset of the table entry of n.
            auto xl = [&](uint32_t x) {
                return *reinterpret_cast<const float *>(reinterpret_cast<const char *>(xltab) + __dp2a_lo(x, 0x00000101u, 0u));
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
            const uint4 tile = sched_tile[slot];
            const int job = (int)tile.w;
            __syncwarp();
            if (lane == 0) slot_read(slot);
            if (job < 0) break;
            if (BATCH && job != cur_job) {
                // A new job: the list of the last one goes out, and the list
                // starts empty (every epilogue warp sees the same items).
                if (cur_job >= 0 && !flush()) { ok = false; break; }
                cur_job = job;
            }
            const T3Job *jb = BATCH ? a.jobs + job : nullptr;
            const int S = (int)(BATCH ? jb->S : a.S), Sp = (int)(BATCH ? jb->S_pad : a.S_pad);
            const uint4 *marg4 = BATCH ? jb->marg4 : a.marg4, *PR = BATCH ? jb->PR : a.PR;
            if (MODE == MODE_TOPN && ew == 0 && lane == 0) *(volatile int *)&epi_job = job;
            const int b = it & 1;
            const uint32_t u = (uint32_t)(it >> 1);
            // Tile data that does not depend on the accumulators, loaded
            // while the tile's MMAs may still run.
            const int i = (int)(tile.y & 0xffffu), j0 = (int)(tile.y >> 16);
            const int lw = (int)tile.z + T3_LB * (int)crank + quarter * 16;   // this warp's first third SNP
            const int l = lw + (lane >> 1);
            const bool lv = l < S;
            // This warp's two pairs dp = part + 4 r, r < nr, that hold some
            // valid combination: the first pair's j before S and before the
            // warp's last SNP l.
            const int jn = lw < S ? min(min(S, lw + 15) - j0, NPT) : 0;    // pairs q < jn
            const int nr = jn > 2 * part ? ((jn + 1) / 2 - part + T3_PARTS - 1) / T3_PARTS : 0;
            // Lanes beyond the last SNP count no sample (their rows are
            // zero): zero tables keep every derived cell a count.  Genotypes
            // of l in the order g, 1 - g.
            uint32_t R02[4] = {0, 0, 0, 0}, Tl0 = 0, Tl1 = 0;
            if (lv) {
                uint32_t Tl[3];
                unpack_marg(marg4[l], Tl);
                Tl0 = (g ? Tl[1] : Tl[0]) << 2;
                Tl1 = (g ? Tl[0] : Tl[1]) << 2;
                const uint4 p4 = PR[(size_t)i * Sp + l];
                R02[0] = (g ? p4.y : p4.x) << 2;
                R02[1] = (g ? p4.x : p4.y) << 2;
                R02[2] = (g ? p4.w : p4.z) << 2;
                R02[3] = (g ? p4.z : p4.w) << 2;
            }
            __syncwarp();
            if (lane < 2 * nr) {
                // The table of pair (i, j), one lane per pair.  Every cell has
                // to be a count (it is a table offset): where j is no SNP its
                // rows are zero, those of a SNP of genotype 2 throughout.
                const int j = j0 + 2 * (part + T3_PARTS * (lane >> 1)) + g;
                uint32_t Ti[3], T01[9];
                unpack_marg(marg4[i], Ti);
#pragma unroll
                for (int x = 0; x < 9; ++x) T01[x] = x % 3 == 2 ? Ti[x / 3] : 0;
                uint64_t rb = 0;
                if (j < S) {
                    uint32_t Tj[3];
                    unpack_marg(marg4[j], Tj);
                    const uint4 q4 = PR[(size_t)i * Sp + j];
                    const uint32_t Rq[4] = {q4.x, q4.y, q4.z, q4.w};
                    full2(Rq, Ti, Tj, T01);
                    // rank of (i, j, l) = base_i - C(S - j, 2) + l - j - 1
                    const uint64_t base_i = (BATCH ? jb->total : a.total) - c3((uint64_t)(S - i)) + c2((uint64_t)(S - i - 1));
                    rb = base_i - c2((uint64_t)(S - j)) - (uint64_t)j - 1;
                }
#pragma unroll
                for (int x = 0; x < 9; ++x) T01[x] <<= 2;
                uint4 *o = reinterpret_cast<uint4 *>(rec + lane * T3_REC_WORDS);
                o[0] = make_uint4(T01[0], T01[1], T01[2], T01[3]);
                o[1] = make_uint4(T01[4], T01[5], T01[6], T01[7]);
                o[2] = make_uint4(T01[8], (uint32_t)rb, (uint32_t)(rb >> 32), 0u);
            }
            // PR[j][l] of this lane's next pair.
            int j = j0 + 2 * part + g;
            const uint4 *pr = PR + (size_t)j * Sp + l;
            uint4 pj_next = make_uint4(0, 0, 0, 0);
            if (nr > 0 && lv && j < S) pj_next = *pr;
            ok = mbar_wait(&bar_tfull[b], u & 1, abort_flag, a.err, wt);
            ok = __all_sync(FULL, ok);   // (also orders the records)
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * T3_BUF + 8 * part);
            // Read again whenever a combination passes what was read before.
            float thr = MODE == MODE_TOPN ? floor_score() : 0.f;
            const float hy = BATCH ? jb->hy : a.hy;
            const float invN = (BATCH ? jb->invN : a.invN) * unscale;
            for (int r = 0; r < nr; ++r, j += 2 * T3_PARTS) {
                // The cells of two pairs with this lane's genotype of l; those
                // of the other lane's pair go there.  R[z][2 a + b]: z = 0 this
                // lane's genotype; packed 4 cases | 4 controls << 16 (all cells
                // below are).
                uint32_t R[2][4];
                {
                    uint32_t v[8], w[8];
                    tmem_ld8(taddr + 8 * T3_PARTS * r, v);
                    if constexpr (!PAIR) tmem_ld8(taddr + T3_N + 8 * T3_PARTS * r, w);
                    tmem_wait_ld();
                    tmem_regs_after_wait(v);
                    if constexpr (!PAIR) tmem_regs_after_wait(w);
#pragma unroll
                    for (int x = 0; x < 8; ++x) {
                        if constexpr (PAIR) v[x] = unpack_enc(v[x]);
                        else v[x] = pack_exact(v[x], w[x]);
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        R[0][x] = g ? v[4 + x] : v[x];
                        R[1][x] = __shfl_xor_sync(FULL, g ? v[x] : v[4 + x], 1);
                    }
                }
                const uint4 pj = pj_next;
                if (r + 1 < nr) {
                    pr += (size_t)(2 * T3_PARTS) * Sp;
                    pj_next = make_uint4(0, 0, 0, 0);
                    if (lv && j + 2 * T3_PARTS < S) pj_next = *pr;
                } else {
                    // This warp's last read of the buffer.
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (PAIR) mbar_arrive_cluster(tempty0 + 8 * b);
                        else mbar_arrive(&bar_tempty[b]);
                    }
                }
                const uint4 *rq = reinterpret_cast<const uint4 *>(rec + (2 * r + g) * T3_REC_WORDS);
                const uint4 r0 = rq[0], r1 = rq[1], r2 = rq[2];
                const uint32_t T01[9] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w, r2.x};
                const uint32_t R12[4] = {(g ? pj.y : pj.x) << 2, (g ? pj.x : pj.y) << 2, (g ? pj.w : pj.z) << 2,
                                         (g ? pj.z : pj.w) << 2};
                const uint64_t rank_of_pair = ((uint64_t)r2.z << 32) | r2.y;   // less l
                // Cells (x, y, 0) and (x, y, 1); (x, y, 2) is the rest of
                // T01(x, y).
                F2 hs[2] = {f2(0.f, 0.f), f2(0.f, 0.f)};
                uint32_t c2z[2][2];   // cells (x, 2, z), x in {0, 1}
                uint32_t odd = 0;     // cell (x, y, 2) of the last even (x, y)
#pragma unroll
                for (int x = 0; x < 3; ++x)
#pragma unroll
                    for (int y = 0; y < 3; ++y) {
                        uint32_t c[3];
#pragma unroll
                        for (int z = 0; z < 2; ++z) {
                            if (x < 2 && y < 2) c[z] = R[z][2 * x + y];
                            else if (y < 2) c[z] = R12[2 * y + z] - R[z][y] - R[z][2 + y];
                            else if (x < 2) c[z] = c2z[x][z] = R02[2 * x + z] - R[z][2 * x] - R[z][2 * x + 1];
                            else c[z] = ((z ? Tl1 : Tl0) - R12[z] - R12[2 + z]) - c2z[0][z] - c2z[1][z];
                        }
                        c[2] = T01[3 * x + y] - c[0] - c[1];
                        hs[0] = add_terms(hs[0], c[0], c[1]);
                        if ((3 * x + y) % 2 == 0) odd = c[2];
                        if ((3 * x + y) % 2 == 1 || 3 * x + y == 8)   // (a cell of no sample adds 0)
                            hs[1] = add_terms(hs[1], odd, 3 * x + y == 8 ? 0u : c[2]);
                        if (MODE == MODE_DUMP && a.dump_tables && lv && j < l) {
                            uint32_t *o = a.dump_tables + (size_t)(rank_of_pair + (uint64_t)l) * 54 + 18 * x + 6 * y;
#pragma unroll
                            for (int z = 0; z < 3; ++z) {
                                const int zz = z < 2 ? z ^ g : 2;   // genotype of l
                                o[2 * zz] = (c[z] & 0xffffu) >> 2;
                                o[2 * zz + 1] = c[z] >> 18;
                            }
                        }
                    }
                const float2 h2 = f2_split(f2_add(hs[0], hs[1]));
                const float score = fmaf(-LN2F * (h2.x + h2.y), invN, hy);
                const bool valid = lv && j < l;
                if (MODE == MODE_DUMP && valid && a.dump_scores) a.dump_scores[rank_of_pair + (uint64_t)l] = score;
                if (MODE == MODE_TOPN) {
                    // Few combinations reach the threshold: ranks only after
                    // the vote.
                    const bool near = valid && score >= thr;
                    if (__any_sync(FULL, near)) {
                        thr = floor_score();
                        const uint64_t rank = rank_of_pair + (uint64_t)l;
                        const bool cand = near && score >= thr && (whole || (rank >= a.rank_begin && rank < a.rank_end)) &&
                                          better(score, rank, thr_s, thr_r);
                        const unsigned mk = __ballot_sync(FULL, cand);
                        if (mk) {
                            if (cand) {
                                const int p = cnt + __popc(mk & ((1u << lane) - 1u));
                                ws[p] = score;
                                wr[p] = rank;
                            }
                            cnt += __popc(mk);
                            __syncwarp();
                            if (cnt > wbuf - 32) merge();
                        }
                    }
                }
            }
            if (nr == 0) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if constexpr (PAIR) mbar_arrive_cluster(tempty0 + 8 * b);
                    else mbar_arrive(&bar_tempty[b]);
                }
            }
        }
        // The last list (a batched launch: of the last job this CTA took;
        // its lists of jobs it never took stay as filled before the launch).
        if (MODE == MODE_TOPN && ok && (!BATCH || cur_job >= 0)) flush();
        if (ew == 0 && lane == 0) *(volatile int *)&epi_job = -2;
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

template <int MODE, int ENC, bool BATCH>
void *kernel_ptr()
{
    return reinterpret_cast<void *>(&k_triples_tc<MODE, ENC, BATCH>);
}

// Pair rows of the first SNPs [i0, i1): thread (i - i0, t), t over the
// pairs (i, j), j = i + 1 + jo, jo < 2 NP ceil((S - 1 - i) / (2 NP)), times the
// 16-byte chunks of a row; the row of pair (j, a, b) is
// rowbase[i - i0] + 4 jo + 2 a + b.
__global__ void k_pair_rows(const uint8_t *E, int64_t pitch, int Wt, int64_t S, int64_t i0, const int64_t *rowbase,
                            uint8_t *P)
{
    const int64_t ii = blockIdx.y;
    const int64_t i = i0 + ii;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t npairs = (S - 1 - i + 2 * T3_NP - 1) / (2 * T3_NP) * (2 * T3_NP);
    const int cw = 4 * Wt;                         // 16-byte chunks per row
    if (t >= npairs * cw) return;
    const int64_t jo = t / cw;
    const int ch = (int)(t - jo * cw);
    const int64_t j = i + 1 + jo;
    const uint4 a0 = *(reinterpret_cast<const uint4 *>(E + (2 * i) * pitch) + ch);
    const uint4 a1 = *(reinterpret_cast<const uint4 *>(E + (2 * i + 1) * pitch) + ch);
    uint4 b0 = make_uint4(0, 0, 0, 0), b1 = b0;
    if (j < S) {
        b0 = *(reinterpret_cast<const uint4 *>(E + (2 * j) * pitch) + ch);
        b1 = *(reinterpret_cast<const uint4 *>(E + (2 * j + 1) * pitch) + ch);
    }
    const int64_t row = rowbase[ii] + 4 * jo;
    auto put = [&](int r, const uint4 &x, const uint4 &y) {
        *(reinterpret_cast<uint4 *>(P + (row + r) * pitch) + ch) =
            make_uint4(x.x & y.x, x.y & y.y, x.z & y.z, x.w & y.w);
    };
    put(0, a0, b0);
    put(1, a0, b1);
    put(2, a1, b0);
    put(3, a1, b1);
}

// E[2 s + g]: genotype row g of SNP s as e2m1 nibbles, 64 bytes a word; rows of
// padding SNPs are zero.  Thread (row, word).
__global__ void k_expand_fp4(const uint4 *X, int64_t S, int64_t S_pad, int64_t rows, int Wt, int64_t pitch, uint8_t *E)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= rows * Wt) return;
    const int64_t row = t / Wt;
    const int w = (int)(t % Wt);
    const int64_t s = row >> 1;
    uint4 bits = make_uint4(0, 0, 0, 0);
    if (s < S) bits = X[((size_t)w * 3 + (row & 1)) * S_pad + s];
    uint4 *dst = reinterpret_cast<uint4 *>(E + row * pitch + (int64_t)w * 64);
    dst[0] = expand_fp4(bits.x);
    dst[1] = expand_fp4(bits.y);
    dst[2] = expand_fp4(bits.z);
    dst[3] = expand_fp4(bits.w);
}

__global__ void k_fill_lists(float *s, uint64_t *r, size_t n)
{
    for (size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (size_t)gridDim.x * blockDim.x) {
        s[x] = -FLT_MAX;
        r[x] = NO_RANK;
    }
}

}  // namespace

cudaError_t launch_expand_fp4(const uint4 *X, int64_t S, int64_t S_pad, int Wt, int64_t pitch, uint8_t *E,
                              cudaStream_t st)
{
    const int64_t n = triples_rows(S) * Wt;
    k_expand_fp4<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(X, S, S_pad, triples_rows(S), Wt, pitch, E);
    return cudaGetLastError();
}

cudaError_t launch_fill_lists(float *s, uint64_t *r, size_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    const size_t blocks = std::min<size_t>((n + 255) / 256, 4096);
    k_fill_lists<<<(unsigned)blocks, 256, 0, st>>>(s, r, n);
    return cudaGetLastError();
}

namespace {
__global__ void k_log2_approx(const uint32_t *n, int64_t count, float scale, float *out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const float x = u2f_small(n[i] & 0x7fffffu);
    // (add_terms' argument: the scaled count, 1e-30 for a count of 0)
    out[i] = lg2_approx(scale > 0.f ? fmaf(x, scale, 1e-30f) : fmaxf(x, 1.0f));
}
}  // namespace

cudaError_t launch_log2_approx(const uint32_t *n, int64_t count, float scale, float *out, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    k_log2_approx<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(n, count, scale, out);
    return cudaGetLastError();
}

int triples_pairs_per_tile(int enc) { return enc ? 2 * T3_NP : T3_NP; }
int triples_snps_per_tile(int enc) { return enc ? 2 * T3_LB : T3_LB; }
int triples_block_rows() { return T3_N; }

size_t triples_smem_bytes(int enc, int stages, int wbuf, int M, int L)
{
    // 1 KiB for the alignment of the stages.
    return 1024 + TC_STATIC_SMEM + (size_t)(M + 1) * 4 + (size_t)stages * T3_STAGE +
           (size_t)T3_EPI_WARPS * t3_warp_pairs(enc) * T3_REC_WORDS * 4 + (size_t)(L + T3_EPI_WARPS * wbuf) * (8 + 4);
}

TriplesShape triples_shape(int enc, int M, int L, size_t smem_cap)
{
    for (int st = T3_MAX_STAGES; st >= 2; --st)
        if (triples_smem_bytes(enc, st, TC_WBUF, M, L) <= smem_cap) return {st, TC_WBUF};
    // The longest lists beside the tables of the most samples (form 0 takes
    // 2 x 16,383): shorter buffers.  400 SNPs x 32,766 samples, top 1,000, take 4.2
    // ms (in the sweep 188).
    if (!enc && triples_smem_bytes(0, 2, T3_WBUF_SHORT, M, L) <= smem_cap) return {2, T3_WBUF_SHORT};
    return {0, 0};
}

float triples_scale(int64_t M)
{
    float q = 1.f;
    for (int64_t m = M; m >= 8; m >>= 1) q *= 0.5f;   // 2^-s, s = floor(log2 M) - 2 (8 <= M)
    return q;
}

void triples_publish(int L, int grid, int *pub_m, int *pub_r)
{
    const int half = std::max(1, std::min(grid, 32 * TC_PUB_PER_LANE) / 2);
    *pub_m = std::min(L, (L + half - 1) / half);
    *pub_r = (L + *pub_m - 1) / *pub_m;
}

cudaError_t launch_pair_rows(const uint8_t *E, int64_t pitch, int Wt, int64_t S, int64_t i0, int64_t i1,
                             const int64_t *rowbase, uint8_t *P, cudaStream_t st)
{
    if (i1 <= i0) return cudaSuccess;
    const int64_t blk = 2 * T3_NP;
    const int64_t maxn = (S - 1 - i0 + blk - 1) / blk * blk * 4 * (int64_t)Wt;   // the pairs of i0, the most
    dim3 grid((unsigned)((maxn + 255) / 256), (unsigned)(i1 - i0));
    k_pair_rows<<<grid, 256, 0, st>>>(E, pitch, Wt, S, i0, rowbase, P);
    return cudaGetLastError();
}

cudaError_t prepare_triples_tc_batch(int enc, size_t smem_bytes)
{
    if (enc != 0 && enc != 1) return cudaErrorInvalidValue;
    void *fn = enc == 1 ? kernel_ptr<MODE_TOPN, 1, true>() : kernel_ptr<MODE_TOPN, 0, true>();
    return allow_dynamic_smem(fn, smem_bytes - TC_STATIC_SMEM);
}

cudaError_t launch_triples_tc(int mode, const CUtensorMap &tmapA, const CUtensorMap &tmapP, const TriplesArgs &a,
                              int grid, cudaStream_t st, bool set_attr)
{
    const size_t bytes = triples_smem_bytes(a.enc, a.stages, a.wbuf, a.M, a.L) - TC_STATIC_SMEM;
    if ((a.enc != 0 && a.enc != 1) || a.stages < 2 || a.stages > T3_MAX_STAGES || a.wbuf < T3_WBUF_SHORT ||
        a.wbuf > TC_WBUF || (a.enc && a.wbuf != TC_WBUF))
        return cudaErrorInvalidValue;
    void *fn = nullptr;
    if (a.jobs) {
        if (mode != MODE_TOPN) return cudaErrorInvalidValue;
        fn = a.enc ? kernel_ptr<MODE_TOPN, 1, true>() : kernel_ptr<MODE_TOPN, 0, true>();
    } else {
        fn = mode == MODE_TOPN ? (a.enc ? kernel_ptr<MODE_TOPN, 1, false>() : kernel_ptr<MODE_TOPN, 0, false>())
                               : (a.enc ? kernel_ptr<MODE_DUMP, 1, false>() : kernel_ptr<MODE_DUMP, 0, false>());
    }
    if (set_attr) {
        const cudaError_t e = allow_dynamic_smem(fn, bytes);
        if (e != cudaSuccess) return e;
    }
    if (grid <= 0) return cudaSuccess;   // attributes only
    CUtensorMap mA = tmapA, mP = tmapP;
    TriplesArgs args = a;
    void *params[] = {&mA, &mP, &args};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(T3_THREADS);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = a.enc ? 1 : 0;   // form 1: CTA pairs (an even grid)
    return cudaLaunchKernelExC(&cfg, fn, params);
}

}  // namespace fc
