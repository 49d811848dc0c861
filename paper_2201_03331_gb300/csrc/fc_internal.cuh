// Internal declarations shared by the library's translation units.
//
// Genotype layout in HBM (the "bit table", a GPU form of the genotype
// tables of the paper's Section "Constructing the genotype tables"):
//   X[(w * 3 + g) * S_pad + s]   (uint4 = 128 samples)
// w  : 128-bit word index; words [0, W0) hold the cases, [W0, Wt) the
//      controls (W0 = ceil(M1/128), Wt = W0 + ceil(M0/128));
// g  : genotype row 0/1/2 (rows a_1, a_2, a_3 of a genotype table);
// s  : SNP, innermost, so the 32 lanes of a warp that work on 32 consecutive
//      extension SNPs read 512 contiguous bytes.
// Bit b of word w is sample 128*w' + b of its class in input order (w' the
// word index within the class).  Padding bits are 0 in all three rows, so
// ANDs over padding contribute nothing.
#pragma once

#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

namespace fc {

constexpr int KMAX_SEARCH = 6;   // orders of the fused search kernels
constexpr int KMAX_BATCH = 4;    // orders of the batched kernel
constexpr int KMAX_TABLES = 6;   // orders of the exact-table kernel

__host__ __device__ constexpr int pow3(int k) { return k <= 0 ? 1 : 3 * pow3(k - 1); }

// C(n, r) for the sizes the library accepts (C(S, k) < 2^60, r <= 6): each
// intermediate is i * C(n - r + i, i) <= r * C(n, r) < 2^63.
__host__ __device__ inline uint64_t binom(int64_t n, int r)
{
    if (r < 0 || n < r) return 0;
    // Unrolled, so that each division is by a constant: a division by a
    // variable takes some 70 instructions, and a rank is turned into its
    // combination by up to 30 of these.
    uint64_t c = 1;
    static_assert(KMAX_TABLES <= 6, "r is at most the order");
#pragma unroll
    for (int i = 1; i <= 6; ++i)
        if (i <= r) c = c * (uint64_t)(n - r + i) / (uint64_t)i;
    return c;
}

// Lexicographic unranking of k-subsets of {0..S-1}: rank 0 is (0,1,..,k-1).
// Combinations with first element v: C(S-1-v, k-1).  The count of those
// with c_t in [lo, v) is C(S-lo, m+1) - C(S-v, m+1), m = k-1-t, which lets
// each position be found by binary search.
__host__ __device__ inline void unrank(int64_t S, int k, uint64_t rank, uint32_t *out)
{
    int64_t lo = 0;
    for (int t = 0; t < k; ++t) {
        const int m = k - 1 - t;
        const uint64_t base = binom(S - lo, m + 1);
        // largest v in [lo, S-1-m] with base - C(S - v, m + 1) <= rank
        int64_t a = lo, b = S - 1 - m;
        while (a < b) {
            int64_t mid = a + (b - a + 1) / 2;
            if (base - binom(S - mid, m + 1) <= rank) a = mid; else b = mid - 1;
        }
        rank -= base - binom(S - a, m + 1);
        out[t] = (uint32_t)a;
        lo = a + 1;
    }
}

__host__ __device__ inline uint64_t rank_of(int64_t S, int k, const uint32_t *c)
{
    uint64_t r = 0;
    int64_t lo = 0;
    for (int t = 0; t < k; ++t) {
        const int m = k - 1 - t;
        r += binom(S - lo, m + 1) - binom(S - (int64_t)c[t], m + 1);
        lo = (int64_t)c[t] + 1;
    }
    return r;
}

// Ranking key: larger score first; equal scores by smaller rank (rank order
// is lexicographic order of the index tuple).
__host__ __device__ inline bool better(float s1, uint64_t r1, float s2, uint64_t r2)
{
    return s1 > s2 || (s1 == s2 && r1 < r2);
}
__host__ __device__ inline bool better64(double s1, uint64_t r1, double s2, uint64_t r2)
{
    return s1 > s2 || (s1 == s2 && r1 < r2);
}

constexpr uint64_t NO_RANK = ~0ull;

// Device-side error word bits.
enum : uint32_t {
    ERR_GENOTYPE = 1u,     // genotype value outside {0,1,2}
    ERR_PHENOTYPE = 2u,    // phenotype value outside {0,1}
    ERR_LIST_SHORT = 4u,   // candidate list too short for the FP32 error window
    ERR_TIMEOUT = 8u,      // bounded device wait ran out
};

// ---- kernel launch wrappers (defined in the .cu files) --------------------

struct PackArgs {
    const uint8_t *G;       // [S][M] device (k_pack: the rows of SNPs s_base .. s_base + S - 1)
    const uint8_t *ph;      // [M] device
    int64_t S, M, S_pad;
    int64_t s_base;         // k_pack: first SNP of G within the table
    int W0, Wt;
    uint4 *X;               // [Wt][3][S_pad]
    int32_t *case_idx;      // [M1] sample index of the i-th case
    int32_t *ctrl_idx;      // [M0]
    uint32_t *err;          // error word
    int64_t *class_count;   // [2] cases, controls
};
// Lets launches of kernel fn take `bytes` of dynamic shared memory.  The limit is
// one value per kernel and device, for all threads of the process, and a launch
// above it is refused: it is only ever raised (setting every launch's own size,
// four threads with lists of 64 to 2048 refused each other's launches).
cudaError_t allow_dynamic_smem(const void *fn, size_t bytes);

cudaError_t launch_class_index(const PackArgs &a, cudaStream_t st);
cudaError_t launch_pack(const PackArgs &a, int64_t M1, int64_t M0, cudaStream_t st);
cudaError_t launch_logtab(float *logtab, int64_t M, cudaStream_t st);
// y ln y (base2: y log2 y), y = scale x, for x = 0..M, each the FP64 product
// rounded once.
cudaError_t launch_xlogx(float *t, int64_t M, cudaStream_t st, bool base2 = false, double scale = 1.0);
// t(a, b) = a ln(n/a) + b ln(n/b), n = a + b, for a, b < n_max at b stride + a, each
// rounded once; 0 in the rest of `floats` entries.
cudaError_t launch_small_terms(float *t, int n_max, int stride, int floats, cudaStream_t st);

struct SearchArgs {
    const uint4 *X;
    int64_t S, S_pad;
    int W0, Wt;
    const float *logtab;    // ln(n) for n = 0..M (ln 0 := 0)
    int M;                  // samples (size of logtab - 1)
    float hy, invN;         // H(Y) and 1/N in FP32
    uint64_t rank_begin, rank_end;
    int L;                  // list capacity
    float *list_score;      // [grid][L]
    uint64_t *list_rank;    // [grid][L]
    void *dump;             // MODE_SCORES: float [n]; MODE_TABLES: uint32 [n][3^k][2]
    // Inclusion-exclusion inputs (k <= 3 with cfg.ie).
    const uint4 *marg4;     // per-SNP genotype counts (one uint4 per SNP)
    const uint4 *PR;        // restricted pair counts [S_pad][S_pad] (k = 3), both orders of a pair
    uint32_t nn;            // cases | controls << 16
};

// Counting variants of the sweep (all give the same exact table):
//  VAR_FULL: popcount all 3^k cells (the paper's method);
//  VAR_IE:   popcount the 2^k cells with genotypes in {0,1}; the rest from
//            per-SNP counts and restricted pair tables (k = 2, 3);
//  VAR_JR:   popcount the cells whose extension-SNP genotype is 0 or 1
//            (2 * 3^(k-1)); genotype 2 from the prefix's own table.
//  VAR_PX:   popcount all 3^k cells, with a (k-2)-prefix table extended by
//            a SNP pair whose 9 rows are formed in registers (k = 4..6).
enum SweepVariant { VAR_FULL = 0, VAR_IE = 1, VAR_JR = 2, VAR_PX = 3 };

struct TuneConfig {
    int G;          // lanes per combination
    int NW;         // warps per CTA
    int WT;         // 128-bit words per prefix-table tile
    int grid;       // CTAs
    int var;        // SweepVariant
};

enum SearchMode { MODE_TOPN = 0, MODE_SCORES = 1, MODE_TABLES = 4 };

cudaError_t launch_restricted_pairs(const uint4 *X, int64_t S, int64_t S_pad, int W0, int Wt, uint4 *PR,
                                    cudaStream_t st);

cudaError_t launch_search(int k, const TuneConfig &cfg, int mode, const SearchArgs &a,
                          cudaStream_t st, size_t *smem_out);
// The variant a kernel of (order, requested variant, mode) really runs.
int effective_variant(int k, int var, int mode);
int search_max_blocks_per_sm(int k, const TuneConfig &cfg, int mode, int L, int M, size_t *smem);

cudaError_t launch_merge(const float *in_s, const uint64_t *in_r, int nlists, int L,
                         float *out_s, uint64_t *out_r, int *nout, cudaStream_t st);

struct RescoreArgs {
    const uint4 *X;
    int64_t S, S_pad;
    int W0, Wt;
    int k;
    int N;                  // requested top_n (<= L)
    int L;
    const float *cand_s;    // [L] sorted best first (FP32)
    const uint64_t *cand_r; // [L]
    float eps;              // FP32 score error bound
    uint64_t total;         // C(S, k)
    double *res_s;          // [L] FP64 scores (-inf where skipped)
    uint64_t *res_r;        // [L]
    uint32_t *res_c;        // [L][k] combinations
    uint32_t *err;
    double *out_score;      // [N] the list
    uint32_t *out_idx;      // [N][k]
    uint32_t *out_err;      // *err after the rescoring
};
cudaError_t launch_rescore(const RescoreArgs &a, int sms, cudaStream_t st);
cudaError_t launch_final(const RescoreArgs &a, cudaStream_t st);

// ---- batched persistent search (many data sets / phenotype replicates) -----

enum { MODE_BATCH = 3 };

struct JobDesc {
    const uint4 *X;         // the job's bit table
    int64_t S, S_pad;
    int W0, Wt;
    float hy, invN, eps;    // H(Y), 1/N and the FP32 score error bound
    int N;                  // min(top_n, C(S, k))
    uint64_t total;         // C(S, k)
    int item_first, n_items;
    const uint4 *marg4;     // inclusion-exclusion tables of the job (or null)
    const uint4 *PR;
    uint32_t nn;            // cases | controls << 16
};

struct BatchItem {
    uint32_t job, pad;
    uint64_t r0, r1;        // rank range [r0, r1) of the job
};

struct BatchArgs {
    const JobDesc *jobs;
    const BatchItem *items;
    int n_items;
    int *counter;           // work-queue head, zeroed before the launch
    const float *logtab;    // ln(n), n = 0..M (M = largest sample count)
    int M;
    int L;
    float *item_score;      // [n_items][L]
    uint64_t *item_rank;
};

cudaError_t launch_search_batch(int k, const TuneConfig &cfg, const BatchArgs &b, cudaStream_t st);
cudaError_t prepare_merge_jobs(int n2);
cudaError_t launch_merge_jobs(const JobDesc *jobs, int n_jobs, const float *item_s, const uint64_t *item_r, int L,
                              int n2, float *out_s, uint64_t *out_r, cudaStream_t st);

struct RescoreBatchArgs {
    const JobDesc *jobs;
    int n_jobs, k, L;
    const float *cand_s;    // [jobs][L]
    const uint64_t *cand_r;
    double *res_s;          // [jobs][L]
    uint64_t *res_r;
    uint32_t *res_tab;      // [jobs][L][3^k][2]
    uint32_t *job_err;      // [jobs]
};
cudaError_t launch_rescore_batch(const RescoreBatchArgs &a, cudaStream_t st);
cudaError_t prepare_final_sort_batch(int L);
cudaError_t launch_final_sort_batch(const JobDesc *jobs, int n_jobs, double *res_s, uint64_t *res_r, int L,
                                    int n_out, int k, uint32_t *out_idx, double *out_score, cudaStream_t st);

// ---- order-2 tensor-core path (fc_pairs_tc.cu) -----------------------------

constexpr int TC_MAX_STAGES = 6;
// Static shared memory of a tensor-core kernel, rounded up (256 to 320 bytes).
constexpr size_t TC_STATIC_SMEM = 512;
enum { MODE_DUMP = 2 };
// Time budget of one mbarrier wait in the tensor-core kernels, in clock64
// ticks (about 2 s).  The pipeline waits of the order-2 kernel take theirs
// from PairsArgs::wait_ticks (a test shortens it so that the waits run out);
// the drain waits before the kernel exits always take this one.
constexpr long long TC_WAIT_TICKS = 4000000000ll;

struct PairsArgs {
    const uint32_t *tiles;  // (I << 16 | J): SNPs i from pairs_rows_i I, SNPs j from pairs_rows_j J
    int ntiles;
    int enc;                // 1: one accumulator n_case + 4096 n_ctrl, a tile per CTA pair; 0: one per class
    int64_t S;
    int W0, Wt;             // 128-sample words: cases [0, W0), controls [W0, Wt)
    const uint4 *marg4;     // per-SNP genotype counts (one uint4 per SNP)
    int stages;             // load stages (pairs_stages)
    const float *xlogx;     // y log2 y, y = scale x, for x = 0..M (FP64 rounded once to FP32)
    float scale;            // the power of two the kernel scores counts in (triples_scale)
    int M;
    float hy, invN;
    uint64_t pair_base;     // C(S, 2)
    uint64_t rank_begin, rank_end;   // only pairs with ranks in [rank_begin, rank_end) count
    int L;
    long long wait_ticks;   // budget of each pipeline wait (clock64 ticks)
    float *list_score;      // [grid][L]
    uint64_t *list_rank;
    // Scores of the lists' entries pub_m - 1 as ordered ints, [grid], set below
    // every score before the launch; pub_r of them bound the score of the last
    // of L pairs (triples_publish).
    int *pub;
    int pub_m, pub_r;
    int *tile_counter;      // next tile of the global order, zeroed before launch
    uint32_t *err;
    float *dump_scores;     // MODE_DUMP: [S][S] (i < j)
    uint32_t *dump_tables;  // MODE_DUMP: [S][S][9][2]
};

// SNPs of a tile on either side, and the rows a CTA loads of the SNPs j.
int pairs_rows_i(int enc);
int pairs_rows_j(int enc);
int pairs_block_rows();
// The load stages that fit smem_cap bytes of shared memory beside the table of
// M samples and lists of L (0: a dump, which keeps no candidates); 0 if not
// even two do.
int pairs_stages(int M, int L, size_t smem_cap);
size_t pairs_smem_bytes(int stages, int M, int L);
cudaError_t launch_marginals(const uint4 *X, int64_t S, int64_t S_pad, int W0, int Wt, uint16_t *marg,
                             cudaStream_t st);
cudaError_t launch_pairs_tc(int mode, const CUtensorMap &tmapI, const CUtensorMap &tmapJ, const PairsArgs &a, int grid,
                            cudaStream_t st);

// Order-3 tensor-core search (fc_triples_tc.cu).  A tile pairs the SNPs l0 ..
// l0 + triples_snps_per_tile - 1 (packed 4-bit rows 2 l + g) with the pairs (i,
// j0 + q), q < triples_pairs_per_tile, of slab rows from rowP (pair row (q, a, b)
// at rowP + 4 q + 2 a + b).
int triples_pairs_per_tile(int enc);
int triples_snps_per_tile(int enc);
// Slab rows a CTA loads for a tile (28 pairs).
int triples_block_rows();
// SNP rows, zero beyond SNP S: a tile starts at any SNP and never leaves them.
constexpr int64_t triples_rows(int64_t S) { return 2 * ((S + 63) / 64 * 64 + 128); }
// Bytes from one row of the SNP rows or of the slab to the next.
constexpr int64_t triples_pitch(int Wt) { return (int64_t)Wt * 64 + 128; }
// One job of the batched order-3 launch (a data set with one phenotype
// replicate), with its own operands and lists.
struct T3Job {
    const CUtensorMap *tmapA;   // the job's SNP rows, 128 x 128-byte boxes
    const CUtensorMap *tmapP;   // the job's slab, 112 x 128-byte boxes
    const uint4 *tiles;         // the job's tiles {rowP, i, j0, l0}
    const uint4 *marg4;         // the job's per-SNP genotype counts
    const uint4 *PR;            // the job's restricted pair table [S_pad][S_pad]
    int64_t S, S_pad;
    uint64_t total;             // C(S, 3)
    float hy, invN;
    int W0, Wt;                 // 128-sample words: cases [0, W0), controls [W0, Wt)
    int item_first, ntiles;     // the job's items [item_first, item_first + ntiles) of its launch
    int slot;                   // lists [slot][grid][L], pub[slot][grid]
};

struct TriplesArgs {
    const uint4 *tiles;     // {rowP, i, j0, l0} per tile of this launch
    int ntiles;
    // 1: one accumulator n_case + 4096 n_ctrl, 0: one per class.
    int enc;
    // Batched launch (jobs != null): items of all jobs, job-major; the fields
    // above and below that describe one data set come from the job table,
    // and list_score, list_rank and pub are indexed by the job's slot.
    const T3Job *jobs;
    int n_jobs, n_items;
    int64_t S, S_pad;
    int W0, Wt;             // 128-sample words: cases [0, W0), controls [W0, Wt)
    const uint4 *marg4;     // per-SNP genotype counts (one uint4 per SNP)
    const uint4 *PR;        // restricted pair table [S_pad][S_pad]
    int stages, wbuf;       // load stages, candidates of a warp's buffer (triples_shape)
    const float *xlogx;     // y log2 y, y = scale x, for x = 0..M (FP64 rounded once to FP32)
    float scale;            // the power of two the kernel scores counts in (triples_scale)
    int M;                  // extent of the kernel's table: the samples
    float hy, invN;
    uint64_t total;         // C(S, 3)
    uint64_t rank_begin, rank_end;   // only combinations with ranks in [rank_begin, rank_end) count
    int L;
    long long wait_ticks;   // budget of each pipeline wait (clock64 ticks)
    float *list_score;      // [grid][L] (batched: [slots][grid][L])
    uint64_t *list_rank;
    // Scores of the lists' entries pub_m - 1 as ordered ints, [grid] (batched:
    // [slots][grid]), set below every score before the first launch; pub_r of
    // them bound the score of the last of L combinations (triples_publish).
    int *pub;
    int pub_m, pub_r;
    int *tile_counter;      // next tile (item) of this launch, zeroed before launch
    uint32_t *err;
    float *dump_scores;     // MODE_DUMP: [C(S,3)] by rank
    uint32_t *dump_tables;  // MODE_DUMP: [C(S,3)][27][2]
};

// The base-2 logarithm the tensor-core epilogues of orders 2 and 3 take of a class
// count, for n[0 .. count) (each modulo 2^23): of n times `scale`, a power of two,
// or 1e-30 where n = 0; scale 0: of max(n, 1).
cudaError_t launch_log2_approx(const uint32_t *n, int64_t count, float scale, float *out, cudaStream_t st);
// The load stages and the entries of a warp's candidate buffer that fit smem_cap
// bytes of shared memory beside the x log2 x table of M samples and lists of L;
// no stages if not even two do.
struct TriplesShape {
    int stages, wbuf;
};
TriplesShape triples_shape(int enc, int M, int L, size_t smem_cap);
size_t triples_smem_bytes(int enc, int stages, int wbuf, int M, int L);
// The power of two the kernel scores the counts of M samples in.
float triples_scale(int64_t M);
// pub_m and pub_r for lists of L and `grid` CTAs: pub_m pub_r >= L, pub_r at most
// about half the CTAs.
void triples_publish(int L, int grid, int *pub_m, int *pub_r);
// The SNP rows of a bit table X: row 2 s + g, one nibble a sample.
cudaError_t launch_expand_fp4(const uint4 *X, int64_t S, int64_t S_pad, int Wt, int64_t pitch, uint8_t *E,
                              cudaStream_t st);
// Slab rows of the first SNPs [i0, i1) from the SNP rows E (pitch bytes per
// row); rowbase[i - i0] is the first slab row of SNP i.
cudaError_t launch_pair_rows(const uint8_t *E, int64_t pitch, int Wt, int64_t S, int64_t i0, int64_t i1,
                             const int64_t *rowbase, uint8_t *P, cudaStream_t st);
// tmapA: the SNP rows in 128 x 128-byte boxes; tmapP: the slab in 112 x
// 128-byte boxes (both with the 128-byte swizzle).
// set_attr = false skips setting the kernel's shared-memory attribute (set
// by an earlier call; a graph capture may not set it); grid = 0 only sets it.
cudaError_t launch_triples_tc(int mode, const CUtensorMap &tmapA, const CUtensorMap &tmapP, const TriplesArgs &a,
                              int grid, cudaStream_t st, bool set_attr = true);
// Shared-memory attribute of the batched kernel of form enc: the largest
// launch's bytes (triples_smem_bytes), set before a graph capture.
cudaError_t prepare_triples_tc_batch(int enc, size_t smem_bytes);
// n list entries (-FLT_MAX, NO_RANK).
cudaError_t launch_fill_lists(float *s, uint64_t *r, size_t n, cudaStream_t st);

// Orders 4 to 6 on tensor cores (fc_quads_tc.cu): left tuples of LT SNPs
// x right tuples of RT SNPs, k = LT + RT (2 + 2, 2 + 3, 3 + 3).  Each side is
// a slab of tuple rows (packed 4-bit 0/1, 64 bytes a word) with all 3^T
// genotype combinations, left tuples in order of their last SNP, right tuples
// in order of their first; a left block of 128 rows or right block of 112
// rows holds 4 (27 / 3^T) tuples: 12 pairs or 4 triples.  A tile is one left
// block x one right block (form 0) or two x two (form 1).
constexpr int tc_left_size(int k) { return k == 6 ? 3 : 2; }
constexpr int tc_tuples_per_block(int T) { return 4 * (27 / (T == 2 ? 9 : 27)); }
constexpr uint64_t NO_TUPLE = ~0ull;
// Rows of a left or right block, bytes from one tuple row to the next.
int tuple_block_rows(bool left);
// Blocks that the tiles of a form take together, on either side.
constexpr int tuple_tile_blocks(int enc) { return enc ? 2 : 1; }
constexpr int64_t tuple_pitch(int Wt) { return (int64_t)Wt * 64 + 128; }
struct QuadsArgs {
    // Tiles (left block a, right block b; enc 1: pairs of consecutive left and
    // of right blocks in place of blocks) come in strips of at most `sub` left
    // blocks: with r = q - item_first and n = ceil((g1 - g0) / sub),
    // item q of the launch is (group g, right block b = lo + r / n, strip
    // r % n) of the group {g0, g1, lo, item_first} with the first
    // item_first <= q, and its tiles are the left blocks a in
    // [g0 + sub (r % n), g0 + sub (r % n + 1)) below min(g1, amax[b]) (those
    // with include[a] set, if include is not null).  Within a group the right
    // blocks stream while the group's left blocks stay in L2; consecutive
    // items share a right block, so the CTAs in flight hold few of them.
    const int4 *groups;     // by item_first
    int ngroups;
    int sub;
    int enc;                // 1: one accumulator n_case + 4096 n_ctrl, tiles of CTA pairs
    int n_items;
    const int *amax;        // [right blocks]: left blocks whose smallest last SNP is below the block's largest first SNP
    const uint8_t *include;
    int64_t S;
    int W0, Wt;
    const uint64_t *ltup;   // left tuples: SNP t in bits [16 t, 16 t + 16), NO_TUPLE for padding
    const uint64_t *lrank;  // rank part of a left tuple (the terms of its SNPs and of its last SNP)
    const uint64_t *rtup;   // right tuples
    const uint64_t *rrank;  // rank part of a right tuple (modulo 2^64)
    const float *xlogx;     // x ln x for x = 0..M
    const float *small_terms;   // cell terms t(a, b) of small counts (launch_quads_small_terms)
    int M;
    float acc_max, case_max;    // M1 + 4096 M0 and M1 (enc 1)
    float hy, invN;
    uint64_t rank_begin, rank_end;   // only combinations with ranks in [rank_begin, rank_end) count
    int L, Bcap, P2, stages;    // stages: 2 .. TC_MAX_STAGES
    float *list_score;      // [grid][L]
    uint64_t *list_rank;
    int *gthr;
    int *tile_counter;
    uint32_t *err;
    float *dump_scores;     // MODE_DUMP: [C(S,k)] by rank
    uint32_t *dump_tables;  // MODE_DUMP: [C(S,k)][3^k][2]
};

// Tuple rows of T-SNP tuples (nblocks left or right blocks).
cudaError_t launch_tuple_rows(int T, bool left, const uint4 *X, int64_t S_pad, int Wt, const uint64_t *tuples,
                              int64_t nblocks, int64_t pitch, uint8_t *Q, cudaStream_t st);
// The table of cell terms of small class counts, quads_small_floats() floats.
int quads_small_floats();
cudaError_t launch_quads_small_terms(float *t, cudaStream_t st);
// Shared memory of the orders 4-6 kernel.
size_t quads_smem_bytes(int enc, int stages, int M, int P2);
cudaError_t launch_quads_tc(int k, int mode, const CUtensorMap &tmapL, const CUtensorMap &tmapR, const QuadsArgs &a,
                            int grid, cudaStream_t st);

struct TablesArgs {
    const uint4 *X;
    int64_t S, S_pad;
    int W0, Wt;
    int k;
    const uint32_t *combos; // [n][k] device
    int64_t n;
    uint32_t *out;          // [n][3^k][2] device
};
cudaError_t launch_tables(const TablesArgs &a, cudaStream_t st);

}  // namespace fc
