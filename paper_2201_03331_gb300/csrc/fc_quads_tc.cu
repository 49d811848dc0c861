// Orders 4 to 6 of the exhaustive search on the fifth-generation tensor
// cores (tcgen05).
//
// A k-combination is a left tuple of LT SNPs followed by a right tuple of RT
// SNPs (k = LT + RT: 2 + 2, 2 + 3, 3 + 3).  Every cell of its 3^k table is,
// per class c (Section "Computing the contingency tables": the population
// count of the AND of one row of each SNP's table),
//     n_c(cell_L, cell_R) = < P_c[left, cell_L], P_c[right, cell_R] >,
// the dot product over the samples of two tuple rows P[t, d] = [G_t = d]
// (all SNPs of tuple t at genotypes d).  The rows are stored as 0/1 e2m1
// nibbles; with the left operand a block of left tuples and the right operand
// blocks of right tuples, both with all 3^T genotype rows, one tcgen05.mma
// kind::mxf4 tile yields every cell of every combination of the blocks
// exactly (fc_tc.cuh).  No cell is derived; combinations whose left tuple
// ends before the right tuple starts are the valid ones.
//
// Row layout.  A left block is 128 rows, 27 / 3^LT tuples in each 32-row TMEM
// lane quarter: one triple in rows 0 .. 26, or three pairs p with genotypes
// d < 8 in rows 8 p + d and d = 8 in row 24 + p (so that the sums over a
// pair's rows are three shuffle levels over eight lanes and one row more);
// the other rows are zero.  A right block is 112 rows, four groups of 28:
// 27 / 3^RT tuples with row 3^RT t + d, then one zero row.  A thread owns the
// 3^RT cells of its (left tuple, d) row against each right tuple.
//
// Scoring: MI = H(Y) - (1/N) sum_cells t(a, b), t = x ln x (a + b) - x ln x (a)
// - x ln x (b).  Most cells of a high-order table are small: where both
// class counts are below 128, t comes from one read of a 128 x 128 table
// (correctly rounded; row stride 133 words, which spreads the few frequent
// entries over the banks), three columns at a time where no lane of the warp
// holds a larger count; the others take three reads of a table of x ln x.
// (A 64 x 64 table leaves room for two more load stages, but at 2,048
// samples more cells are above it: order 4, a 64th of 1,001 SNPs, 57.7 ms
// against 46.9; order 5 at 152 SNPs 120 against 112.)  What bounds the kernel is
// the tensor pipe (74 % active at order 4, 120 SNPs x 6,000 samples, operands at
// 14.5 TB/s from L2) and with few samples the epilogue: 300 SNPs x 6,000 samples
// take 53.7 ms, that 64th of 1,001 SNPs 46.0, orders 5 and 6 at 152 and 76 SNPs
// x 2,048 samples 111 and 113.
// The accumulator n_case + 4096 n_ctrl plus 2^21 holds four times the packed
// counts in its mantissa, so the table offset 4 a + 532 b takes a shift and a
// multiply-add.  Each thread sums the terms of its row's cells, the 3^LT lanes
// of a left tuple add their partial sums; every addend is a sum of
// non-negative cell terms bounded by N ln 2, so as for order 3 |MI32 - MI| <=
// u (3 ln M + (3^k + 4) ln 2) (u = 2^-24), within the sweep's bound
// u (2 ln M + (2 3^k + 6) ln 2) for M < 2^(3^k + 2).  The lexicographic rank
// of a combination is the sum of a part that depends on the left tuple only
// and one that depends on the right tuple only, both computed on the host.
//
// Two forms (template ENC):
//   ENC = 0: case and control samples accumulate into two accumulators of 112
//            columns; a tile is (left block, right block), one CTA each;
//   ENC = 1: control samples carry the block scale 4096, so one accumulator
//            holds n_case + 4096 n_ctrl (exact while both classes have at
//            most 4095 samples); a tile is (two left blocks, two right
//            blocks), worked on by a pair of CTAs (cta_group::2, M = 256, N =
//            224): each CTA loads one left and one right block and scores
//            its left block against both right blocks.  With 128-row tiles
//            per CTA the copies of both right blocks set the pace (44 KB a
//            chunk and CTA at 65 bytes a cycle, the same with the scoring
//            left out); the pair loads 30 KB.
//
// Roles (one persistent CTA per SM, 640 threads):
//   warps 0, 1 : TMA producers (128-byte K chunks, 256 samples, of the left and
//                right blocks), warp w owning the stages s = w (mod 2)
//   warp 2     : one lane (ENC 1: of the pair's leader) schedules the tiles
//   warp 3     : TMEM allocation; one elected lane (ENC 1: of the pair's
//                leader) issues the MMAs.  With the scheduling in the same
//                thread, the tensor cores idled about 700 cycles between
//                tiles (3,584 cycles of MMAs at 2,048 samples)
//   warps 4-19 : epilogue (TMEM -> registers -> partial MI over a row's cells
//                -> sum over a left tuple's lanes -> CTA top list), four warps
//                per TMEM lane quarter, each a quarter of the tile's groups of
//                28 columns.  With one warp per quarter the epilogue set the
//                pace: about 18,000 cycles per 128 x 256 tile.
// TMEM: two accumulator buffers of 224 columns and two blocks of columns of
// scales.
#include "fc_tc.cuh"

namespace fc {

namespace {

constexpr int T4_PRODUCERS = 2;
constexpr int T4_EPI_WARP0 = 4;
constexpr int T4_EPI_WARPS = 16;
constexpr int T4_PARTS = T4_EPI_WARPS / 4;         // epilogue warps per TMEM lane quarter
constexpr int T4_EPI_THREADS = 32 * T4_EPI_WARPS;
constexpr int T4_THREADS = 32 * T4_EPI_WARP0 + T4_EPI_THREADS;
constexpr int T4_GROUP = 28;                       // columns of a group of right tuples (27 used)
constexpr int T4_BLOCK = 4 * T4_GROUP;             // columns of a right block
constexpr int T4_BUF = 2 * T4_BLOCK;               // columns of an accumulator buffer
constexpr uint32_t T4_SCALE_COL = 2 * T4_BUF;      // TMEM column of scale 1, then of scale 4096
static_assert(T4_SCALE_COL + 2 * FP4_SCALE_COLS <= TC_TMEM_COLS, "scales behind the accumulators");
// Table of t(a, b) for a, b < 128.
constexpr int T4_SMALL = 128;
constexpr int T4_SMALL_STRIDE = 133;
constexpr int T4_SMALL_FLOATS = (T4_SMALL * T4_SMALL_STRIDE + 3) / 4 * 4;
// x + 2^21 for an integer x = a + 4096 b < 2^21: 4 x in the low mantissa bits.
constexpr uint32_t T4_MAGIC = 0x4A000000u;
// Bits of x + 2^21 that are zero exactly where a, b < 128 (and x is a
// non-negative integer): a's bits 7-11, b's bits 7-8, the exponent's low two
// bits, the two fraction bits.
constexpr uint32_t T4_LARGE_BITS = 0x01E03E03u;
constexpr uint32_t T4_MUL = 16384 - 4 * T4_SMALL_STRIDE;                      // u - (u >> 14) T4_MUL = 4 a + 532 b + T4_OFF
constexpr uint32_t T4_OFF = T4_MAGIC - (T4_MAGIC >> 14) * T4_MUL;

// Tuple-row slab: thread (row, 16-byte chunk); the row is [G_t = d] (every
// SNP of the tuple at its genotype digit, first SNP most significant) over
// the 32 samples of the chunk, one nibble each.
template <int T, bool LEFT>
__global__ void k_tuple_rows(const uint4 *X, int64_t S_pad, int Wt, const uint64_t *tuples, int64_t nblocks,
                             int64_t pitch, uint8_t *Q)
{
    constexpr int R = T == 2 ? 9 : 27;              // rows per tuple
    constexpr int PQ = 27 / R;                      // tuples per quarter (group)
    constexpr int QROWS = LEFT ? 32 : T4_GROUP;     // rows per quarter (group)
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int cw = 4 * Wt;                          // 16-byte chunks per row
    if (t >= nblocks * (4 * QROWS) * cw) return;
    const int64_t row = t / cw;
    const int ch = (int)(t - row * cw);
    const int64_t blk = row / (4 * QROWS);
    const int r = (int)(row - blk * (4 * QROWS));
    const int quarter = r / QROWS, rq = r % QROWS;
    uint32_t bits = 0;
    if (rq < 27) {
        // Tuple of the quarter and genotype digits of this row.
        const int p = LEFT && T == 2 ? (rq < 24 ? rq >> 3 : rq - 24) : rq / R;
        int d = LEFT && T == 2 ? (rq < 24 ? rq & 7 : 8) : rq % R;
        const uint64_t tup = tuples[blk * (4 * PQ) + quarter * PQ + p];
        if (tup != NO_TUPLE) {
            const int w = ch >> 2, q32 = ch & 3;    // 128-sample word, 32-sample part
            bits = ~0u;
#pragma unroll
            for (int u = T - 1; u >= 0; --u) {
                const int g = d % 3;
                d /= 3;
                const uint32_t s = (uint32_t)(tup >> (16 * u)) & 0xffffu;
                bits &= reinterpret_cast<const uint32_t *>(X + ((size_t)w * 3 + g) * S_pad + s)[q32];
            }
        }
    }
    *(reinterpret_cast<uint4 *>(Q + row * pitch) + ch) = expand_fp4(bits);
}

// The class counts of an encoded accumulator x = a + 4096 b (a, b < 4096),
// clamped to the classes so that no index can leave the x ln x table.
__device__ __forceinline__ void split_enc(float x, float xmax, float amax, uint32_t &a, uint32_t &b)
{
    x = fminf(fmaxf(x, 0.f), xmax);
    const float y = __fmaf_rz(x, 1.f / 4096.f, 8388608.f);   // 2^23 + floor(x / 4096)
    const float af = fminf(fmaf(-4096.f, y - 8388608.f, x), amax);
    b = __float_as_uint(y) - 0x4B000000u;
    a = __float_as_uint(af + 8388608.f) - 0x4B000000u;
}

template <int LT, int RT, int MODE, int ENC>
__global__ void __launch_bounds__(T4_THREADS, 1)
    k_quads_tc(const __grid_constant__ CUtensorMap tmapL, const __grid_constant__ CUtensorMap tmapR, QuadsArgs a)
{
    constexpr bool PAIR = ENC == 1;                 // a tile per CTA pair
    constexpr int NB = ENC ? T4_BUF : T4_BLOCK;     // MMA N
    constexpr uint32_t STAGE = TC_A_BYTES + (uint32_t)T4_BLOCK * TC_BK;   // one left and one right block
    constexpr int RL = LT == 2 ? 9 : 27;            // rows (cells) per left tuple
    constexpr int RR = RT == 2 ? 9 : 27;            // columns (cells) per right tuple
    constexpr int LPQ = 27 / RL;                    // left tuples per lane quarter
    constexpr int RPG = 27 / RR;                    // right tuples per group of columns
    constexpr int GROUPS = NB / T4_GROUP;           // groups per tile
    constexpr int GPW = GROUPS / T4_PARTS;          // groups per epilogue warp
    constexpr int V = GPW * RPG;                    // right tuples per epilogue warp
    constexpr int CK = RL * RR;                     // cells of a table (3^k)
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_full[TC_MAX_STAGES], bar_empty[TC_MAX_STAGES];
    __shared__ uint64_t bar_tfull[2], bar_tempty[2], bar_done;
    __shared__ uint32_t tmem_base_slot;
    __shared__ uint64_t bar_sfull[TC_SCHED], bar_sempty[TC_SCHED];
    // Left and right block of each slot of the ring (ENC 1: pairs of blocks;
    // left block -1: no more tiles).
    __shared__ __align__(8) int2 sched_tile[TC_SCHED];
    __shared__ int abort_flag_s;
    __shared__ int buf_count;
    __shared__ int epi_stop;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int stages = a.stages;
    const uint32_t crank = PAIR ? cluster_rank() : 0;   // CTA of the pair (0: its leader)
    volatile int *abort_flag = &abort_flag_s;

    uint8_t *smem = reinterpret_cast<uint8_t *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    float *xltab = reinterpret_cast<float *>(smem + (size_t)stages * STAGE);   // x ln x
    const int lt_floats = (a.M + 1 + 3) & ~3;
    float *small = xltab + lt_floats;                                          // t(a, b), ENC 1
    uint64_t *lrank = reinterpret_cast<uint64_t *>(small + (ENC ? T4_SMALL_FLOATS : 0));
    float *lscore = reinterpret_cast<float *>(lrank + a.P2);

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&bar_full[s], 1);
            mbar_init(&bar_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bar_tfull[b], 1);
            mbar_init(&bar_tempty[b], (PAIR ? 2 : 1) * T4_EPI_WARPS);
        }
        mbar_init(&bar_done, 1);
        for (int s = 0; s < TC_SCHED; ++s) {
            mbar_init(&bar_sfull[s], 1);
            // The MMA thread, and the producers and epilogue warps (of both
            // CTAs of a pair).
            mbar_init(&bar_sempty[s], 1 + (PAIR ? 2 : 1) * (T4_PRODUCERS + T4_EPI_WARPS));
        }
        abort_flag_s = 0;
        buf_count = 0;
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
    if (ENC)
        for (int i = threadIdx.x; i < T4_SMALL_FLOATS; i += blockDim.x) small[i] = a.small_terms[i];
    if (MODE == MODE_TOPN) {
        for (int i = threadIdx.x; i < a.P2; i += blockDim.x) {
            lscore[i] = -FLT_MAX;
            lrank[i] = NO_RANK;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    if (warp >= T4_EPI_WARP0 && warp < T4_EPI_WARP0 + 4) {
        const uint32_t q = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + T4_SCALE_COL;
        tmem_fill16(q, FP4_SCALE_ONE);
        tmem_fill16(q + FP4_SCALE_COLS, FP4_SCALE_4096);
        tmem_wait_st();
    }
    tc_fence_before();
    // Barriers and scales of both CTAs are ready before either uses them.
    if constexpr (PAIR) cluster_sync(); else __syncthreads();
    tc_fence_after();

    // A consumer's word that it has read a slot of the tile ring.
    const uint32_t sempty0 = PAIR ? cluster_addr(&bar_sempty[0], 0) : 0;
    auto slot_read = [&](int slot) {
        if constexpr (PAIR) mbar_arrive_cluster(sempty0 + 8 * slot);
        else mbar_arrive(&bar_sempty[slot]);
    };

    const int nk = (a.Wt + 1) / 2;   // 256-sample chunks (two words; the last may hold one, then zeros)

    if (warp < T4_PRODUCERS) {
        // ---------------- TMA producers ----------------
        if (elect_one()) {
            Ring ring;
            int owner = 0;   // producer of stage ring.s
            // Parity of the last fill issued into each owned stage (at most
            // three: stages warp, warp + 2, warp + 4), -1 before the first.
            int last[3] = {-1, -1, -1};
            auto step = [&]() {
                ring.next(stages);
                owner = ring.s == 0 || owner + 1 == T4_PRODUCERS ? 0 : owner + 1;
            };
            bool ok = true;
            for (int it = 0; ok; ++it) {
                const int slot = it % TC_SCHED;
                const uint32_t sn = (uint32_t)(it / TC_SCHED);
                if (!mbar_wait(&bar_sfull[slot], sn & 1, abort_flag, a.err)) { ok = false; break; }
                const int t = sched_tile[slot].x;
                const int rb = sched_tile[slot].y;
                slot_read(slot);
                if (t < 0) break;
                const int rowL = (PAIR ? 2 * t + (int)crank : t) * TC_BM;
                const int rowR = (PAIR ? 2 * rb + (int)crank : rb) * T4_BLOCK;
                for (int kc = 0; kc < nk; ++kc, step()) {
                    if (owner != warp) continue;
                    const int s = ring.s;
                    uint8_t *st = smem + (size_t)s * STAGE;
                    if (!mbar_wait(&bar_empty[s], ring.par ^ 1, abort_flag, a.err)) { ok = false; break; }
                    if constexpr (PAIR) {
                        // The leader's barrier counts the bytes of both CTAs.
                        if (crank == 0) mbar_expect_tx(&bar_full[s], 2 * STAGE);
                        tma_load_2d_pair(&tmapL, &bar_full[s], st, kc * TC_BK, rowL);
                        tma_load_2d_pair(&tmapR, &bar_full[s], st + TC_A_BYTES, kc * TC_BK, rowR);
                    } else {
                        mbar_expect_tx(&bar_full[s], STAGE);
                        tma_load_2d(&tmapL, &bar_full[s], st, kc * TC_BK, rowL);
                        tma_load_2d(&tmapR, &bar_full[s], st + TC_A_BYTES, kc * TC_BK, rowR);
                    }
                    last[0] = s == warp ? (int)ring.par : last[0];
                    last[1] = s == warp + T4_PRODUCERS ? (int)ring.par : last[1];
                    last[2] = s == warp + 2 * T4_PRODUCERS ? (int)ring.par : last[2];
                }
            }
            // Let the last copies into the stages this producer owns land
            // before the CTA can exit (earlier ones were consumed).  A pair's
            // copies complete on its leader's barriers, and neither CTA exits
            // before the other (the cluster barrier below); where a wait ran
            // out, the second CTA allows its own copies a millisecond.
            if (crank == 0) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int s = warp + q * T4_PRODUCERS;
                    const int par = last[q];
                    if (s >= stages || par < 0) continue;
                    long long t0 = clock64();
                    while (!mbar_try(&bar_full[s], (uint32_t)par) && clock64() - t0 < WAIT_BUDGET) {}
                }
            } else if (!ok) {
                const long long t0 = clock64();
                while (clock64() - t0 < 2000000) {}
            }
        }
    } else if (warp == 2) {
        if (crank == 0 && lane == 0) {
            // ---------------- scheduler ----------------
            const uint32_t peer_tile = PAIR ? cluster_addr(&sched_tile[0], 1) : 0;
            const uint32_t peer_sfull = PAIR ? cluster_addr(&bar_sfull[0], 1) : 0;
            // The strip being handed out: right block s_b, left blocks
            // [s_a, s_aend); the group of the last item taken.
            int s_b = 0, s_a = 0, s_aend = 0;
            int s_first = 0, s_end = 0, s_lo = 0, s_g0 = 0, s_g1 = 0, s_n = 1;
            auto next_tile = [&](int &ta, int &tb) -> bool {
                for (;;) {
                    while (s_a < s_aend) {
                        const int x = s_a++;
                        if (!a.include || a.include[x]) {
                            ta = x;
                            tb = s_b;
                            return true;
                        }
                    }
                    const int q = atomicAdd(a.tile_counter, 1);
                    if (q >= a.n_items) return false;
                    if (q >= s_end) {
                        // Items only grow: the group is this one or a later one.
                        int lo = 0, hi = a.ngroups - 1;
                        while (lo < hi) {
                            const int mid = (lo + hi + 1) >> 1;
                            if (a.groups[mid].w <= q) lo = mid; else hi = mid - 1;
                        }
                        const int4 gr = a.groups[lo];
                        s_g0 = gr.x;
                        s_g1 = gr.y;
                        s_lo = gr.z;
                        s_first = gr.w;
                        s_end = lo + 1 < a.ngroups ? a.groups[lo + 1].w : a.n_items;
                        s_n = (s_g1 - s_g0 + a.sub - 1) / a.sub;
                    }
                    const int r = q - s_first;
                    s_b = s_lo + r / s_n;
                    s_a = s_g0 + (r % s_n) * a.sub;
                    s_aend = min(min(s_a + a.sub, s_g1), a.amax[s_b]);
                }
            };
            for (int it = 0;; ++it) {
                const int slot = it % TC_SCHED;
                const uint32_t sn = (uint32_t)(it / TC_SCHED);
                if (!mbar_wait(&bar_sempty[slot], (sn & 1) ^ 1, abort_flag, a.err)) break;
                int ta = -1, tb = 0;
                if (!next_tile(ta, tb)) ta = -1;
                sched_tile[slot] = make_int2(ta, tb);
                mbar_arrive(&bar_sfull[slot]);
                if constexpr (PAIR) cluster_post2(peer_tile + 8 * slot, peer_sfull + 8 * slot, ta, tb);
                if (ta < 0) break;
            }
        }
    } else if (warp == 3) {
        if (crank == 0 && elect_one()) {
            // ---------------- MMA issue ----------------
            const uint32_t idesc = idesc_mxf4(PAIR ? 2 * TC_BM : TC_BM, NB);
            const uint64_t descA = smem_desc_sw128(smem_u32(smem)), descB = smem_desc_sw128(smem_u32(smem + TC_A_BYTES));
            const uint32_t one = tmem_base + T4_SCALE_COL;
            Ring ring;
            bool ok = true;
            for (int it = 0; ok; ++it) {
                const int slot = it % TC_SCHED;
                const uint32_t sn = (uint32_t)(it / TC_SCHED);
                if (!mbar_wait(&bar_sfull[slot], sn & 1, abort_flag, a.err)) break;
                const int t = sched_tile[slot].x;
                mbar_arrive(&bar_sempty[slot]);
                if (t < 0) break;
                const int b = it & 1;
                const uint32_t u = (uint32_t)(it >> 1);
                if (!mbar_wait(&bar_tempty[b], (u & 1) ^ 1, abort_flag, a.err)) break;
                tc_fence_after();
                const uint32_t d0 = tmem_base + (uint32_t)(b * T4_BUF);
                for (int kc = 0; kc < nk && ok; ++kc, ring.next(stages)) {
                    const int s = ring.s;
                    if (!mbar_wait(&bar_full[s], ring.par, abort_flag, a.err)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t ad = descA + (uint64_t)s * (STAGE >> 4);
                    const uint64_t bd = descB + (uint64_t)s * (STAGE >> 4);
                    // Two words of 128 samples (two MMAs each): cases, then
                    // controls (ENC 0: into the second accumulator; ENC 1:
                    // with scale 4096).
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int w = 2 * kc + h;
                        if (w < a.Wt) {
                            const bool ctrl = w >= a.W0;
                            const bool first = w == 0 || (!ENC && w == a.W0);
                            const uint32_t d = d0 + (!ENC && ctrl ? T4_BLOCK : 0);
                            const uint32_t sa = one + (ENC && ctrl ? FP4_SCALE_COLS : 0);
                            if constexpr (PAIR) {
                                mma_mxf4_pair(d, ad + 4 * h, bd + 4 * h, idesc, sa, one, first ? 0u : 1u);
                                mma_mxf4_pair(d, ad + 4 * h + 2, bd + 4 * h + 2, idesc, sa, one, 1u);
                            } else {
                                mma_mxf4(d, ad + 4 * h, bd + 4 * h, idesc, sa, one, first ? 0u : 1u);
                                mma_mxf4(d, ad + 4 * h + 2, bd + 4 * h + 2, idesc, sa, one, 1u);
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
            long long t0 = clock64();
            while (!mbar_try(&bar_done, 0) && clock64() - t0 < WAIT_BUDGET) {}
        }
    } else {
        // ---------------- epilogue ----------------
        const int tid = threadIdx.x - 32 * T4_EPI_WARP0;   // 0 .. T4_EPI_THREADS - 1
        const int quarter = warp & 3;
        const int part = (warp - T4_EPI_WARP0) >> 2;       // groups [part GPW, (part + 1) GPW)
        // Left tuple of the quarter and genotype digits of this lane's row
        // (p = LPQ: a padding row).
        const int p = LT == 3 ? (lane < 27 ? 0 : 1) : lane < 24 ? lane >> 3 : lane - 24;
        const int cell_l = LT == 3 ? lane : lane < 24 ? lane & 7 : 8;
        // After the sum over a left tuple's rows this lane scores the
        // combination of its left tuple with right tuple `vsel` of the warp
        // (-1: none).
        int vsel = -1;
        if (LT == 3) {
            if (V == 2 ? (lane & 15) == 0 : lane == 0) vsel = V == 2 ? lane >> 4 : 0;
        } else if (lane < 24) {
            if (V == 6 && (lane & 3) < 3) vsel = 3 * ((lane >> 2) & 1) + (lane & 3);
            if (V == 3 && (lane & 7) < 3) vsel = lane & 7;
            if (V == 2 && (lane & 3) == 0) vsel = (lane >> 2) & 1;
            if (V == 1 && (lane & 7) == 0) vsel = 0;
        }
        const int L = a.L;
        const int Bcap = a.Bcap;
        const uint32_t lt = (uint32_t)a.M;
        const uint32_t tempty0 = PAIR ? cluster_addr(&bar_tempty[0], 0) : 0;
        const float xmax = a.acc_max, amax = a.case_max;
        const uint32_t small_off = smem_u32(small) - T4_OFF;
        float thr_s = -FLT_MAX;
        uint64_t thr_r = NO_RANK;
        // A tile inserts at most one candidate per combination.
        constexpr int TILE_CANDS = 4 * LPQ * GROUPS * RPG;
        for (int it = 0;; ++it) {
            const int slot = it % TC_SCHED;
            const uint32_t sn = (uint32_t)(it / TC_SCHED);
            const bool ok = mbar_wait(&bar_sfull[slot], sn & 1, abort_flag, a.err);
            int t = ok ? sched_tile[slot].x : -1;
            const int rb = ok ? sched_tile[slot].y : 0;
            if (ok) {
                __syncwarp();
                if (lane == 0) slot_read(slot);
            }
            if (PAIR && t >= 0) t = 2 * t + (int)crank;   // this CTA's left block
            const int b = it & 1;
            const uint32_t u = (uint32_t)(it >> 1);
            // Tile data that does not depend on the accumulators, loaded while
            // the tile's MMAs may still run: this lane's left tuple and the
            // right tuple it scores, with their parts of the rank.
            uint64_t ltp = NO_TUPLE, lrk = 0, rtp = NO_TUPLE, rrk = 0;
            const size_t ri0 = (size_t)rb * (GROUPS * RPG) + part * V;   // this warp's first right tuple
            float gthr = -FLT_MAX;
            if (t >= 0) {
                if (p < LPQ) {
                    const size_t li = (size_t)t * (4 * LPQ) + quarter * LPQ + p;
                    ltp = a.ltup[li];
                    lrk = a.lrank[li];
                }
                if (vsel >= 0) {
                    rtp = a.rtup[ri0 + vsel];
                    rrk = a.rrank[ri0 + vsel];
                }
                // The global threshold only rises; a value read once per tile
                // admits at most a few more candidates than a fresh one would.
                if (MODE == MODE_TOPN) gthr = from_ordered(*(volatile int *)a.gthr);
                mbar_wait(&bar_tfull[b], u & 1, abort_flag, a.err);
            }
            // One stop decision for all epilogue warps (they meet at named
            // barriers, which have no timeout); t is the same for all.
            // Between the barriers nobody inserts, so the buffer's fill is
            // the same for all.
            epi_bar_n<T4_EPI_THREADS>();
            if (tid == 0) epi_stop = *abort_flag;
            const int fill = buf_count;
            epi_bar_n<T4_EPI_THREADS>();
            if (epi_stop || t < 0) break;
            if (MODE == MODE_TOPN) {
                if (fill > Bcap - TILE_CANDS) {
                    for (int x = L + fill + tid; x < a.P2; x += T4_EPI_THREADS) { lscore[x] = -FLT_MAX; lrank[x] = NO_RANK; }
                    epi_bitonic_desc_n<T4_EPI_THREADS>(lscore, lrank, a.P2, tid);
                    if (tid == 0) {
                        buf_count = 0;
                        if (lrank[L - 1] != NO_RANK) atomicMax(a.gthr, ordered_int(lscore[L - 1]));
                    }
                    epi_bar_n<T4_EPI_THREADS>();
                }
                thr_s = lscore[L - 1];
                thr_r = lrank[L - 1];
            }
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * T4_BUF);
            float val[V];
#pragma unroll
            for (int gi = 0; gi < GPW; ++gi) {
                const uint32_t col = taddr + (uint32_t)((part * GPW + gi) * T4_GROUP);
                uint32_t v0[28];
                uint32_t v1[ENC ? 1 : 28];
                tmem_ld28(col, v0);
                if constexpr (!ENC) tmem_ld28(col + T4_BLOCK, v1);
                tmem_wait_ld();
                tmem_regs_after_wait(v0);
                if constexpr (!ENC) tmem_regs_after_wait(v1);
                if (gi == GPW - 1) {
                    // This warp's last read of the buffer.
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (PAIR) mbar_arrive_cluster(tempty0 + 8 * b);
                        else mbar_arrive(&bar_tempty[b]);
                    }
                }
#pragma unroll
                for (int q = 0; q < RPG; ++q) {
                    // Three partial sums shorten the chain of dependent
                    // additions.
                    float hs[3] = {0.f, 0.f, 0.f};
#pragma unroll
                    for (int c = RR * q; c < RR * q + RR; c += 3) {
                        bool general = true;
                        if constexpr (ENC) {
                            uint32_t w[3];
#pragma unroll
                            for (int e = 0; e < 3; ++e)
                                w[e] = __float_as_uint(__uint_as_float(v0[c + e]) + __uint_as_float(T4_MAGIC));
                            general = __any_sync(FULL, ((w[0] | w[1] | w[2]) & T4_LARGE_BITS) != 0);
                            if (!general) {
#pragma unroll
                                for (int e = 0; e < 3; ++e)
                                    hs[e] += lds_f32(small_off + (w[e] - (w[e] >> 14) * T4_MUL));
                            }
                        }
                        if (general) {
#pragma unroll
                            for (int e = 0; e < 3; ++e) {
                                uint32_t ca, cb;
                                if constexpr (ENC) {
                                    split_enc(__uint_as_float(v0[c + e]), xmax, amax, ca, cb);
                                    hs[e] += (xltab[ca + cb] - xltab[ca]) - xltab[cb];
                                } else {
                                    // Clamped so that no index can leave the table.
                                    ca = min(f2u_exact(v0[c + e]), lt);
                                    cb = min(f2u_exact(v1[c + e]), lt);
                                    hs[e] += (xltab[min(ca + cb, lt)] - xltab[ca]) - xltab[cb];
                                }
                            }
                        }
                    }
                    val[gi * RPG + q] = (hs[0] + hs[1]) + hs[2];
                    if (MODE == MODE_DUMP && a.dump_tables && p < LPQ && ltp != NO_TUPLE) {
                        const size_t ri = ri0 + gi * RPG + q;
                        const uint64_t rq = a.rtup[ri];
                        const uint32_t llast = (uint32_t)(ltp >> (16 * (LT - 1))) & 0xffffu;
                        if (rq != NO_TUPLE && llast < ((uint32_t)rq & 0xffffu)) {
                            uint32_t *o = a.dump_tables + (size_t)(lrk + a.rrank[ri]) * (2 * CK) + (size_t)cell_l * (2 * RR);
#pragma unroll
                            for (int c = 0; c < RR; ++c) {
                                uint32_t ca, cb;
                                if constexpr (ENC) {
                                    split_enc(__uint_as_float(v0[RR * q + c]), xmax, amax, ca, cb);
                                } else {
                                    ca = min(f2u_exact(v0[RR * q + c]), lt);
                                    cb = min(f2u_exact(v1[RR * q + c]), lt);
                                }
                                o[2 * c] = ca;
                                o[2 * c + 1] = cb;
                            }
                        }
                    }
                }
            }
            // Sum over the RL rows of each left tuple; where the warp holds
            // two or six right tuples, the first level also splits them
            // between the halves.
            float tot;
            if constexpr (LT == 3) {
                // Padding rows hold no counts and add 0.
                static_assert(V <= 2, "order 6");
                if constexpr (V == 2) {
                    const bool hi = (lane & 16) != 0;
                    const float send = hi ? val[0] : val[1];
                    tot = (hi ? val[1] : val[0]) + __shfl_xor_sync(FULL, send, 16);
                } else {
                    tot = val[0] + __shfl_xor_sync(FULL, val[0], 16);
                }
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) tot += __shfl_xor_sync(FULL, tot, o);
            } else {
                // Row d = 8 of pair p comes from lane 24 + p.
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const float ninth = __shfl_sync(FULL, val[v], 24 + (lane >> 3));
                    if ((lane & 7) == 0) val[v] += ninth;
                }
                constexpr int H = V % 2 ? V : V / 2;
                float kept[H];
                const bool hi = (lane & 4) != 0;
#pragma unroll
                for (int v = 0; v < H; ++v) {
                    if constexpr (V % 2) {
                        kept[v] = val[v] + __shfl_xor_sync(FULL, val[v], 4);
                    } else {
                        const float send = hi ? val[v] : val[v + H];
                        kept[v] = (hi ? val[v + H] : val[v]) + __shfl_xor_sync(FULL, send, 4);
                    }
                }
#pragma unroll
                for (int o = 2; o > 0; o >>= 1)
#pragma unroll
                    for (int v = 0; v < H; ++v) kept[v] += __shfl_xor_sync(FULL, kept[v], o);
                tot = kept[0];
                if constexpr (H == 3) {
                    const int pick = V == 6 ? lane & 3 : lane & 7;
                    tot = pick == 1 ? kept[1] : pick == 2 ? kept[2] : kept[0];
                }
            }
            const uint32_t llast = (uint32_t)(ltp >> (16 * (LT - 1))) & 0xffffu;
            const uint32_t rfirst = (uint32_t)rtp & 0xffffu;
            const bool real = vsel >= 0 && ltp != NO_TUPLE && rtp != NO_TUPLE && llast < rfirst;
            const uint64_t rank = lrk + rrk;   // modulo 2^64
            const bool valid = real && rank >= a.rank_begin && rank < a.rank_end;
            const float score = fmaf(-tot, a.invN, a.hy);
            if (MODE == MODE_DUMP && valid && a.dump_scores) a.dump_scores[rank] = score;
            if (MODE == MODE_TOPN) {
                const bool cand = valid && score >= gthr && better(score, rank, thr_s, thr_r);
                const unsigned mk = __ballot_sync(FULL, cand);
                if (mk) {
                    int base = 0;
                    if (lane == 0) base = atomicAdd(&buf_count, __popc(mk));
                    base = __shfl_sync(FULL, base, 0);
                    if (cand) {
                        // The check above keeps the slot inside the buffer.
                        const int s2 = min(L + base + __popc(mk & ((1u << lane) - 1u)), a.P2 - 1);
                        lscore[s2] = score;
                        lrank[s2] = rank;
                    }
                }
            }
        }
        if (MODE == MODE_TOPN) {
            epi_bar_n<T4_EPI_THREADS>();
            const int nb = buf_count;
            for (int x = L + nb + tid; x < a.P2; x += T4_EPI_THREADS) { lscore[x] = -FLT_MAX; lrank[x] = NO_RANK; }
            epi_bitonic_desc_n<T4_EPI_THREADS>(lscore, lrank, a.P2, tid);
            for (int x = tid; x < L; x += T4_EPI_THREADS) {
                a.list_score[(size_t)blockIdx.x * L + x] = lscore[x];
                a.list_rank[(size_t)blockIdx.x * L + x] = lrank[x];
            }
        }
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

int tuple_block_rows(bool left) { return left ? TC_BM : T4_BLOCK; }

cudaError_t launch_tuple_rows(int T, bool left, const uint4 *X, int64_t S_pad, int Wt, const uint64_t *tuples,
                              int64_t nblocks, int64_t pitch, uint8_t *Q, cudaStream_t st)
{
    const int64_t n = nblocks * tuple_block_rows(left) * 4 * (int64_t)Wt;
    if (n == 0) return cudaSuccess;
    const unsigned grid = (unsigned)((n + 255) / 256);
    if (T == 2 && left) k_tuple_rows<2, true><<<grid, 256, 0, st>>>(X, S_pad, Wt, tuples, nblocks, pitch, Q);
    else if (T == 2) k_tuple_rows<2, false><<<grid, 256, 0, st>>>(X, S_pad, Wt, tuples, nblocks, pitch, Q);
    else if (left) k_tuple_rows<3, true><<<grid, 256, 0, st>>>(X, S_pad, Wt, tuples, nblocks, pitch, Q);
    else k_tuple_rows<3, false><<<grid, 256, 0, st>>>(X, S_pad, Wt, tuples, nblocks, pitch, Q);
    return cudaGetLastError();
}

int quads_small_floats() { return T4_SMALL_FLOATS; }

cudaError_t launch_quads_small_terms(float *t, cudaStream_t st)
{
    return launch_small_terms(t, T4_SMALL, T4_SMALL_STRIDE, T4_SMALL_FLOATS, st);
}

size_t quads_smem_bytes(int enc, int stages, int M, int P2)
{
    // 1 KiB for the alignment of the stages.
    return 1024 + TC_STATIC_SMEM + (size_t)stages * (TC_A_BYTES + T4_BLOCK * TC_BK) + (size_t)((M + 1 + 3) & ~3) * 4 +
           (enc ? (size_t)T4_SMALL_FLOATS * 4 : 0) + (size_t)P2 * (8 + 4);
}

template <int LT, int RT>
void *quads_kernel(int mode, int enc)
{
    if (mode == MODE_TOPN)
        return enc ? reinterpret_cast<void *>(&k_quads_tc<LT, RT, MODE_TOPN, 1>)
                   : reinterpret_cast<void *>(&k_quads_tc<LT, RT, MODE_TOPN, 0>);
    return enc ? reinterpret_cast<void *>(&k_quads_tc<LT, RT, MODE_DUMP, 1>)
               : reinterpret_cast<void *>(&k_quads_tc<LT, RT, MODE_DUMP, 0>);
}

cudaError_t launch_quads_tc(int k, int mode, const CUtensorMap &tmapL, const CUtensorMap &tmapR, const QuadsArgs &a,
                            int grid, cudaStream_t st)
{
    if (a.stages < 2 || a.stages > TC_MAX_STAGES) return cudaErrorInvalidValue;
    const size_t bytes = quads_smem_bytes(a.enc, a.stages, a.M, a.P2) - TC_STATIC_SMEM;
    void *fn = nullptr;
    if (k == 4) fn = quads_kernel<2, 2>(mode, a.enc);
    if (k == 5) fn = quads_kernel<2, 3>(mode, a.enc);
    if (k == 6) fn = quads_kernel<3, 3>(mode, a.enc);
    if (!fn) return cudaErrorInvalidValue;
    cudaError_t e = allow_dynamic_smem(fn, bytes);
    if (e != cudaSuccess) return e;
    CUtensorMap mL = tmapL, mR = tmapR;
    QuadsArgs args = a;
    void *params[] = {&mL, &mR, &args};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(T4_THREADS);
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
