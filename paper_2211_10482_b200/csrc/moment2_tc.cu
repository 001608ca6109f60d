// st_sym_moment2, tensor-core paths: out[p(i,j)] = sum_n X[n,i] X[n,j], fp32 accumulation (Section 3, M1; the outer
// product summed over samples is a symmetric rank-N update, i.e. a triangular tile GEMM X^T X).  Five forms of X:
//   M2_BF16   bfloat16
//   M2_TF32   fp32, of which the tensor core reads the upper 19 bits
//   M2_CONV   fp32, in the kernel x = hi + lo in bfloat16: hi^T hi + hi^T lo + lo^T hi (M2TC_SYM_SUM: two of the three)
//   M2_SPLIT  the same products of hi and lo that lie in memory (the pair features of moment4.cu)
//   M2_EXACT  fp32, in the kernel of moment2_exact.cuh x = hi + mid + lo, at the error of fp32 arithmetic
//
// A cluster of two blocks owns an output tile of 256 rows (i) x up to 256 columns (j) for a range of the samples.
// Only tiles that contain an entry with i <= j are launched, and a tile of the last column is as wide as the columns
// left, rounded up to 32.  Block r of the pair stages columns 256*TM+128r.. (its 128 rows of the A operand) and its
// half of the columns of the B operand; on full diagonal tiles the two coincide and are loaded once, and where all rows are
// in the first block its A holds its B ([1048576,64] bf16 57 us with both loaded, now 50; [271319,8] 22, now 16).  The leader block
// issues one MMA of M = 256 for the pair; each block keeps the accumulator of its 128 rows in its own tensor memory
// and adds it into an fp32 partial tile; a second kernel adds the partial tiles of all sample ranges in a fixed order
// and writes the packed upper triangle.
//
// Up to 128 columns that are left over after whole tiles of 256 (`ext`) have no tiles of their own, which would load 256 columns
// of A for a few of B: the tiles on the diagonal, whose A is B, load them in the place of A and make a second product of
// their rows with them, and the last of these tiles also the product of the left-over columns with themselves.  Such a tile
// needs the tensor memory of both accumulators, so that its MMAs wait while the epilogue empties them (a tenth of a phase
// with one load from tensor memory at a time and sums that come back from L2; hardly anything with m2tc_add_in_l2).
// us, with tiles of their own / carried along: [262144,520] split 384 / 314 (with M2TC_SYM_SUM 283), TF32 287 / 206, bf16 161 / 119;
// [131072,776] 346 / 286, 229 / 187, 129 / 110; [262144,264] 161 / 109, 137 / 76, 71 / 43; [131072,896] (128 columns) 399 / 327, 250 / 217, 131 / 117.
//
// The tensor core adds into its fp32 accumulator without round-to-nearest, so a chain of
// many thousands of accumulating MMAs drifts low (measured: -7.7e-4 relative on all-positive
// sums of 150k terms).  The chain is therefore cut every FLUSH_CHUNKS stages: the MMAs switch
// to the second accumulator in tensor memory while the epilogue warps add the finished one
// into the block's partial tile with ordinary fp32 additions.
//
// Both operands of X^T X are "MN-major" for the tensor core: X is [N, d] row-major, so the
// output index (i or j) is contiguous and the reduction index n strides by a row.  TMA
// loads boxes of 128 bytes x KROWS rows with the 128-byte swizzle, which is exactly the
// canonical MN-major layout of tcgen05 (8 rows x 128 bytes per swizzle atom).  An MN-major operand of 32-bit elements
// (TF32) has one legal shared-memory form, the 128-byte swizzle of 32-byte units, which the copies write (tensor-map
// swizzle "128B, atom 32B") and the descriptors name.
//
// What bounds it: wide tiles the tensor pipe and the L2 that feeds it; every column panel is read by all tiles of its
// row and column, so clusters that work on the same samples must run in step to share X in L2.  Four stages of 32 KB
// are the measured optimum there: with six or seven the clusters of a sample range drift apart and the kernel gets
// 5-12% slower, with three it starves.  M2_SPLIT makes its three products from one load of both parts (64 instead of
// 96 bytes per sample and column pair).  Few features: the latency of a stage, hence more and smaller stages.
//
// M2_CONV: a pass that wrote hi and lo before moved 8 bytes a value through HBM on top of the 4 read here, and took
// 176 of the 590 us of [262144,520], now 283; [1048576,256] 700, now 285; [1048576,64] 245, now 143.  Copies bring the
// fp32 boxes, converting warps rewrite them in place and arrive at the leader's barrier.  Bound by shared memory: per
// 32 samples of a full tile off the diagonal 256 cycles each for the copy, the reads and the writes and 384 for the
// operands of 768 cycles of MMA.  Loads through registers instead of the copies avoid two of these, but every arrival
// then waits for the loads in flight (760 us).
//
// Warp roles (192 threads, M2_CONV 384 more): warp 0 = TMA producer, warp 1 = MMA issuer and TMEM owner,
// warps 2..5 = epilogue (TMEM -> registers -> global), one per 32-lane quarter of TMEM,
// warps 6.. convert.
#include "tc_common.cuh"
#include "st_index.cuh"
#include "pair_layout.cuh"
#include <cuda_bf16.h>
#include <algorithm>
#include <functional>

namespace st {

enum { M2_BF16 = 0, M2_TF32 = 1, M2_SPLIT = 2, M2_CONV = 3, M2_EXACT = 4 };

namespace m2tc {
constexpr int BM = 256, BN = 256;               // tile of the pair
constexpr int HALF = 128;                       // rows staged per block, and most B columns
constexpr int MAX_STAGES = 24;
constexpr size_t STAGES_BYTES = 131072;         // all stages together
constexpr size_t STAGES_BYTES_1 = 196608;       // a single tile: nobody to keep in step with
constexpr int THREADS = 192;
constexpr int CONV_GROUPS = 3;                  // M2_CONV: groups of four converting warps on successive stages
constexpr int CONV_THREADS = 128 * CONV_GROUPS;
constexpr size_t STAGES_BYTES_CONV = 196608;    // with 131072 [262144,520] ran 552 us instead of 510, [30000,520] 78 instead of 68
constexpr int MAX_TILES = 160;
constexpr int MAX_EXT = 16;                     // 4096 columns in tiles of 256
constexpr uint32_t TMEM_COLS = 512;
template <int MODE> struct Shape {
    static constexpr int ELEM = MODE == M2_TF32 ? 4 : 2;
    static constexpr int PARTS = MODE == M2_EXACT ? 3 : MODE >= M2_SPLIT ? 2 : 1;   // hi (, mid) and lo
    static constexpr int KROWS = MODE == M2_BF16 ? 64 : 32; // sample rows per stage
    static constexpr int KMMA = MODE == M2_TF32 ? 8 : 16;   // sample rows per MMA
    static constexpr int BOXC = 128 / ELEM;                 // columns per TMA box (128 bytes)
    static constexpr int BOX_BYTES = 128 * KROWS;
    static constexpr int NBOX = HALF / BOXC;                // most boxes per operand and part in a block
    // accumulating MMAs per phase: 256 (bf16), 512 (TF32, half the samples each), 252 (split)
    static constexpr int FLUSH_CHUNKS = MODE == M2_BF16 ? 64 : MODE == M2_TF32 ? 128 : 42;
};

struct TileTable {
    int ntiles;
    unsigned char diag[MAX_TILES];                     // on the diagonal: the columns start where the rows do
    unsigned char width[MAX_TILES];                    // columns, units of 32
    unsigned short row[MAX_TILES], col[MAX_TILES];     // first row and column of the result, units of 8
    unsigned short rows[MAX_TILES];                    // at most 256
    unsigned short first[MAX_TILES + 1];               // first cluster: the clusters of a tile share its samples
    unsigned char ext[MAX_TILES];                      // columns that are left over after the whole tiles, units of 16: 0 or, on
                                                       // tiles that carry them, all of them
    unsigned char next, carrier[MAX_EXT];              // those tiles
    unsigned char corner;                              // the last of them also has the left-over columns among themselves
    unsigned short ext_col;                            // first left-over column, units of 8
    unsigned char sym;                                 // M2_CONV: full diagonal tiles hold S, of which (S + S^T) / 2 is the result
};
// A partial tile holds four columns of a row side by side: [BN / 4][HALF][4] for each block, and after the BN columns of the
// tile the left-over ones, and after these the corner.
struct Args {
    float *partials;                                   // [2 * cluster + block][pitch]
    unsigned *status;
    int d;                                             // columns of X
    int chunks_total, stages, nb, na;                  // nb, na: boxes of B and A per part in a stage
    int pitch;                                         // floats of a block's partial tile
    int lo_row0;                                       // M2_SPLIT: first row of the lo part
    const float *X;                                    // M2_EXACT: what the copies read
    int64_t N, ldx;
    TileTable tab;
};
}  // namespace m2tc

// Tile of a cluster.
__device__ __forceinline__ int m2tc_tile_of(const m2tc::TileTable &t, int cluster)
{
    int lo = 0, hi = t.ntiles - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((int)t.first[mid] <= cluster) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Adds 32 columns of a thread's row, those of `mask` (four by four), to the partial tile, in L2 and without an answer;
// the additions of one thread to one place take effect in their order.  L2 takes subnormal numbers for zero.  Where |v| is
// at least 2^-100 no sum is one, and what it lacks is below 2^-25 of v; four columns with a smaller value among them are added here.  But
// a zero changes no sum, and where the others are large they go one by one: padding, and categories that a sample range lacks.
// [262144,520] in rows of calls, us: N(0,1) split 283, bf16 119, TF32 207; with zeros added here, and 32 columns for one of them, / now:
// split, a zero column 447 / 303, 128 categories in sorted order 436 / 287; bf16, 300 of these 159 / 112; TF32, 300 unsorted 241 / 191.
// Sums below 2^-100 wait for L2: split with a third of the columns times 2^-54 500 (tiles of their own 392), bf16 with all 163 (150).
__device__ __forceinline__ void m2tc_add_in_l2(float *p, const uint32_t (&r)[32], uint32_t mask)
{
    constexpr int QUAD = 4 * m2tc::HALF;                   // floats from one group of four columns to the next
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
        if (!(mask >> e & 15u)) continue;
        const float v[4] = {__uint_as_float(r[e]), __uint_as_float(r[e + 1]), __uint_as_float(r[e + 2]), __uint_as_float(r[e + 3])};
        float *q = p + e / 4 * QUAD;
        if (fminf(fminf(fabsf(v[0]), fabsf(v[1])), fminf(fabsf(v[2]), fabsf(v[3]))) >= 0x1p-100f) {
            asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(q), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
            continue;
        }
        bool tiny = false;
#pragma unroll
        for (int i = 0; i < 4; ++i) tiny |= fabsf(v[i]) < 0x1p-100f && v[i] != 0.f;
        if (!tiny) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (v[i] != 0.f) asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(q + i), "f"(v[i]) : "memory");
            continue;
        }
        float4 o;
        asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(o.x), "=f"(o.y), "=f"(o.z), "=f"(o.w) : "l"(q) : "memory");
        asm volatile("st.relaxed.gpu.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(q), "f"(o.x + v[0]), "f"(o.y + v[1]), "f"(o.z + v[2]), "f"(o.w + v[3]) : "memory");
    }
}

}  // namespace st
#include "moment2_exact.cuh"
namespace st {

// EXT: some tiles carry left-over columns (an instance of its own: the registers of their epilogue cost small calls without any 2 to 6 %).
template <int MODE, bool EXT>
__global__ void __launch_bounds__(MODE == M2_CONV ? m2tc::THREADS + m2tc::CONV_THREADS : m2tc::THREADS, 1)
moment2_tc_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ m2tc::Args a)
{
    using namespace m2tc;
    using namespace tc;
    using S = Shape<MODE>;
    constexpr int KROWS = S::KROWS, BOXC = S::BOXC, BOX_BYTES = S::BOX_BYTES, NBOX = S::NBOX;
    constexpr int PARTS = S::PARTS;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = align_smem(smem_raw);
    const uint32_t part_bytes = (uint32_t)((a.nb + a.na) * BOX_BYTES), stage_bytes = PARTS * part_bytes;
    // M2_CONV: a box of fp32 becomes its hi and its lo box in place; else all hi boxes, then all lo boxes
    constexpr int BOX_PITCH = MODE == M2_CONV ? 2 * BOX_BYTES : BOX_BYTES;
    const uint32_t lo_off = MODE == M2_CONV ? BOX_BYTES : part_bytes;
    const int stages = a.stages;
    // an MMA reads 128 columns of A per block, na boxes of which were loaded: behind the last stage there is room for the others
    uint64_t *bars = (uint64_t *)(smem + (size_t)stages * stage_bytes + (size_t)(NBOX - a.na) * BOX_PITCH);
    uint64_t *full = bars, *empty = bars + MAX_STAGES, *acc_full = bars + 2 * MAX_STAGES, *acc_empty = bars + 2 * MAX_STAGES + 2;
    uint64_t *raw = bars + 2 * MAX_STAGES + 4;          // M2_CONV: fp32 boxes have landed
    uint32_t *tmem_slot = (uint32_t *)(raw + MAX_STAGES);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();            // 0 = leader
    const int cluster = blockIdx.x >> 1;
    const int tile = m2tc_tile_of(a.tab, cluster), split = cluster - a.tab.first[tile];
    const int nsplit = a.tab.first[tile + 1] - a.tab.first[tile];
    const int row = 8 * a.tab.row[tile], rows = a.tab.rows[tile], col = 8 * a.tab.col[tile], width = 32 * a.tab.width[tile];
    const bool diag = a.tab.diag[tile] != 0;
    // narrow tiles are cheap to flush: chains half as long, as short as those of twice as many sample ranges
    const int FLUSH_CHUNKS = MODE == M2_BF16 && width <= HALF ? S::FLUSH_CHUNKS / 2 : S::FLUSH_CHUNKS;
    const bool alias = diag && width == BN;             // A columns == B columns in both blocks: one load serves both
    const bool lead = diag && rows <= HALF;             // all rows in the first block, whose A holds its half of B as well
    const bool sym = MODE == M2_CONV && alias && a.tab.sym;
    // (a tile that carries left-over columns is on the diagonal, and full)
    const int ext = EXT ? 16 * a.tab.ext[tile] : 0, ecol = 8 * a.tab.ext_col;
    const bool corner = ext > 0 && a.tab.corner && tile == a.tab.carrier[a.tab.next - 1];
    const int chunks_per_split = (a.chunks_total + nsplit - 1) / nsplit;
    const int c_begin = split * chunks_per_split;
    int c_end = c_begin + chunks_per_split;
    if (c_end > a.chunks_total) c_end = a.chunks_total;
    const int nchunks = c_end > c_begin ? c_end - c_begin : 0;
    const int nphases = (nchunks + FLUSH_CHUNKS - 1) / FLUSH_CHUNKS;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            // leader's producer arrives once and announces the bytes of both blocks; converting warps arrive each
            mbar_init(&full[s], MODE == M2_CONV ? 8 : 1);
            if (MODE == M2_CONV) mbar_init(&raw[s], 1);
            mbar_init(&empty[s], 1);         // one commit per use, delivered to both blocks
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 8);     // four epilogue warps in each of the two blocks (leader's copy is used)
        }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, TMEM_COLS);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                      // both blocks' barriers exist before anything is signalled across
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        // the status words are cleared here instead of by a separate memset; a time-out
        // report can only be written 2^24 failed polls later
        a.status[kWsStatusWord] = 0;
        a.status[kWsDetailWord] = 0;
    }

    // boxes of BU columns that block r loads: of B, and of A the ones that hold rows of the result (and nothing past the
    // last column; what is not loaded makes entries that are never read)
    constexpr int BU = MODE == M2_CONV ? 32 : BOXC;
    auto boxes_b = [&](int r) {
        int n = lead && r == 0 && rows > width / 2 ? rows : width / 2;
        if (n > a.d - col - r * (width / 2)) n = a.d - col - r * (width / 2);
        return n <= 0 ? 0 : (n + BU - 1) / BU;
    };
    auto boxes_a = [&](int r) {
        int n = rows - r * HALF;
        if (ext > 0) n = min(ext / 2, a.d - ecol - r * (ext / 2));      // in the place of A, which B holds there
        else if (alias || lead) n = 0;
        return n <= 0 ? 0 : n >= HALF ? HALF / BU : (n + BU - 1) / BU;
    };
    const int col_a = ext > 0 ? ecol + (int)rank * (ext / 2) : row + (int)rank * HALF, col_b = col + (int)rank * (width / 2);
    if (MODE == M2_CONV && warp == 0) {
        // ---------------- TMA producer (both blocks): own boxes, fp32
        if (elect_one()) {
            prefetch_tmap(&tmap);
            const int nb = boxes_b((int)rank), na = boxes_a((int)rank);
            int s = 0;
            uint32_t parity = 1;
            for (int c = 0; c < nchunks; ++c) {
                if (c >= stages && !mbar_wait(&empty[s], parity, abort_flag, a.status, 1)) break;
                mbar_expect_tx(&raw[s], (uint32_t)((nb + na) * BOX_BYTES));
                unsigned char *base = smem + (size_t)s * stage_bytes;
                const int y = (c_begin + c) * KROWS;
                for (int b = 0; b < nb; ++b) tma_load_2d(base + b * BOX_BYTES, &tmap, &raw[s], col_b + b * BU, y);
                for (int b = 0; b < na; ++b) tma_load_2d(base + (2 * a.nb + b) * BOX_BYTES, &tmap, &raw[s], col_a + b * BU, y);
                if (++s == stages) { s = 0; parity ^= 1u; }
            }
        }
    } else if (warp == 0) {
        // ---------------- TMA producer (both blocks): own boxes, completion counted on the leader's barrier
        if (elect_one()) {
            prefetch_tmap(&tmap);
            const int nb = boxes_b((int)rank), na = boxes_a((int)rank);
            const uint32_t tx = (uint32_t)((boxes_b(0) + boxes_b(1) + boxes_a(0) + boxes_a(1)) * PARTS * BOX_BYTES);
            const uint32_t bar0 = map_to_cta(smem_u32(full), 0);
            int s = 0;
            uint32_t parity = 1;
            for (int c = 0; c < nchunks; ++c) {
                if (c >= stages && !mbar_wait(&empty[s], parity, abort_flag, a.status, 1)) break;
                if (rank == 0) mbar_expect_tx(&full[s], tx);
                const uint32_t bar = bar0 + (uint32_t)(s * sizeof(uint64_t));
                const int sample = (c_begin + c) * KROWS;
#pragma unroll
                for (int p = 0; p < PARTS; ++p) {
                    unsigned char *base = smem + (size_t)s * stage_bytes + (size_t)p * part_bytes;
                    const int y = sample + (p ? a.lo_row0 : 0);
                    for (int b = 0; b < nb; ++b)            // B half (and A on full diagonal tiles)
                        tma_load_2d_pair(base + b * BOX_BYTES, &tmap, bar, col_b + b * BOXC, y);
                    for (int b = 0; b < na; ++b)            // A rows of this block
                        tma_load_2d_pair(base + (a.nb + b) * BOX_BYTES, &tmap, bar, col_a + b * BOXC, y);
                }
                if (++s == stages) { s = 0; parity ^= 1u; }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (leader only)
        if (rank == 0 && elect_one()) {
            const uint32_t idesc = make_idesc(MODE == M2_TF32 ? 2 : 1, 1, 1, BM, (uint32_t)width);
            const uint32_t a_off = alias || lead ? 0u : (uint32_t)(a.nb * BOX_PITCH);
            const uint32_t sb0 = smem_u32(smem);
            // bf16: groups of 8 sample rows, 16-byte swizzle units; fp32 read as TF32: groups of 4, 32-byte units
            const uint64_t adesc_base = make_smem_desc(sb0 + a_off, BOX_PITCH, MODE == M2_TF32 ? 512 : 1024, MODE == M2_TF32 ? 1 : 2);
            const uint64_t bdesc_base = make_smem_desc(sb0, BOX_PITCH, MODE == M2_TF32 ? 512 : 1024, MODE == M2_TF32 ? 1 : 2);
            const uint64_t lo = (uint64_t)(lo_off >> 4), ext_off = (uint64_t)((a.nb * BOX_PITCH) >> 4);
            const uint32_t idesc_ext = make_idesc(MODE == M2_TF32 ? 2 : 1, 1, 1, BM, (uint32_t)ext);
            bool ok = true;
            int c = 0, s = 0;
            uint32_t parity = 0;
            for (int ph = 0; ph < nphases && ok; ++ph) {
                const int buf = ext > 0 ? 0 : ph & 1;
                if (ext > 0) {
                    if (ph >= 1 && !mbar_wait(&acc_empty[0], (uint32_t)((ph - 1) & 1), abort_flag, a.status, 4)) break;
                } else if (ph >= 2 && !mbar_wait(&acc_empty[buf], (uint32_t)(((ph >> 1) - 1) & 1), abort_flag, a.status, 4)) {
                    break;
                }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * BN);
                const int ce = (c + FLUSH_CHUNKS < nchunks) ? c + FLUSH_CHUNKS : nchunks;
                uint32_t accumulate = 0;
                for (; c < ce; ++c) {
                    if (!mbar_wait<MODE == M2_CONV>(&full[s], parity, abort_flag, a.status, 2)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t ad = adesc_base + (uint64_t)((uint32_t)s * (stage_bytes >> 4));
                    const uint64_t bd = bdesc_base + (uint64_t)((uint32_t)s * (stage_bytes >> 4));
                    // sym: lo holds 2 lo, S = hi^T hi + hi^T 2 lo, and the sum of the partial tiles makes (S + S^T) / 2 of it; with 2 lo
                    // the left-over columns take hi / 2, which lies `half` behind hi
                    auto products = [&](uint32_t acc, uint64_t a0, uint64_t b0, uint32_t shape, bool two, uint64_t half) {
                        uint32_t on = accumulate;
#pragma unroll
                        for (int k = 0; k < KROWS / S::KMMA; ++k) {
                            // one MMA spans KMMA sample rows of 128 bytes: 2048 bytes (bf16) or 1024 bytes (TF32) further on
                            constexpr int STEP = S::KMMA * 128 / 16;
                            const uint64_t ak = a0 + (uint64_t)(k * STEP), bk = b0 + (uint64_t)(k * STEP);
                            if (MODE == M2_TF32) mma_tf32_pair(acc, ak, bk, shape, on);
                            else mma_bf16_pair(acc, ak, bk, shape, on);
                            on = 1;
                            if (PARTS == 2) {
                                mma_bf16_pair(acc, ak, bk + lo, shape, 1u);
                                if (!two) mma_bf16_pair(acc, ak + lo, bk + half, shape, 1u);
                            }
                        }
                    };
                    products(d_tmem, ad, bd, idesc, sym, 0);
                    if (ext > 0) {
                        products(tmem_base + BN, ad, bd + ext_off, idesc_ext, false, sym ? (uint64_t)(BOX_PITCH >> 4) : 0);
                        if (corner) products(tmem_base + (uint32_t)(BN + ext), bd + ext_off, bd + ext_off, idesc_ext, false, 0);
                    }
                    accumulate = 1;
                    tc_commit_pair(&empty[s]);
                    if (++s == stages) { s = 0; parity ^= 1u; }
                }
                tc_commit_pair(&acc_full[buf]);
            }
        }
    } else if (MODE == M2_CONV && warp >= THREADS / 32) {
        // ---------------- converting warps (both blocks): x = hi + lo, each in the form that a copy of boxes of 64 columns x
        // 32 rows with the 128-byte swizzle leaves.  A warp takes eight rows of all boxes of a stage.  They are two runs of
        // 1024 bytes of every pair of boxes of 32 columns, the first of which becomes hi and the second lo: in place.
        constexpr int H = 4, PAIRS_B = 2;
        const int cw = warp - THREADS / 32, group = cw >> 2;
        const int r0 = lane >> 4, c4 = (lane & 15) * 4;           // rows r0 + 2h of the eight, columns c4 .. c4+3
        const int nb = boxes_b((int)rank), na = boxes_a((int)rank);
        const uint32_t bar0 = map_to_cta(smem_u32(full), 0);
        uint32_t from[H], to[H];
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int r = r0 + 2 * h;
            from[h] = (uint32_t)((cw & 3) * 1024 + (c4 >> 5) * BOX_BYTES + r * 128 + ((((c4 >> 2) & 7) ^ r) << 4));
            to[h] = (uint32_t)((cw & 3) * 1024 + r * 128 + (((c4 >> 3) ^ r) << 4) + (c4 & 4) * 2);
        }
        int s = group % stages;
        uint32_t parity = (uint32_t)(group / stages) & 1u;
        bool ok = true;
        for (int c = group; c < nchunks; c += CONV_GROUPS) {
            ok = ok && mbar_wait(&raw[s], parity, abort_flag, a.status, 1);
            unsigned char *stage = smem + (size_t)s * stage_bytes;
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const int n = side ? na : nb;
                unsigned char *p = stage + (side ? a.nb * BOX_PITCH : 0);
                const float twice = sym && side == 0 ? 2.f : 1.f;
                float4 v[PAIRS_B][H];
#pragma unroll
                for (int q = 0; q < PAIRS_B; ++q)
                    if (2 * q + (c4 >> 5) < n) {
#pragma unroll
                        for (int h = 0; h < H; ++h) v[q][h] = *reinterpret_cast<const float4 *>(p + q * BOX_PITCH + from[h]);
                    }
                __syncwarp();
#pragma unroll
                for (int q = 0; q < PAIRS_B; ++q)
                    if (2 * q + (c4 >> 5) < n) {
#pragma unroll
                        for (int h = 0; h < H; ++h) {
                            const float4 x = v[q][h];
                            const __nv_bfloat162 h0 = __floats2bfloat162_rn(x.x, x.y), h1 = __floats2bfloat162_rn(x.z, x.w);
                            const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
                            const __nv_bfloat162 l0 = __floats2bfloat162_rn(twice * (x.x - f0.x), twice * (x.y - f0.y)),
                                                 l1 = __floats2bfloat162_rn(twice * (x.z - f1.x), twice * (x.w - f1.y));
                            unsigned char *w = p + q * BOX_PITCH + to[h];
                            *reinterpret_cast<uint2 *>(w) =
                                make_uint2(*reinterpret_cast<const uint32_t *>(&h0), *reinterpret_cast<const uint32_t *>(&h1));
                            *reinterpret_cast<uint2 *>(w + BOX_BYTES) =
                                make_uint2(*reinterpret_cast<const uint32_t *>(&l0), *reinterpret_cast<const uint32_t *>(&l1));
                            if (EXT && side == 1 && sym) {
                                const __nv_bfloat162 g0 = __floats2bfloat162_rn(0.5f * f0.x, 0.5f * f0.y), g1 = __floats2bfloat162_rn(0.5f * f1.x, 0.5f * f1.y);
                                *reinterpret_cast<uint2 *>(w + BOX_PITCH) =
                                    make_uint2(*reinterpret_cast<const uint32_t *>(&g0), *reinterpret_cast<const uint32_t *>(&g1));
                            }
                        }
                    }
            }
            fence_proxy_async();          // generic writes, read by the tensor core
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster_smem(bar0 + (uint32_t)(s * sizeof(uint64_t)));
            s += CONV_GROUPS;
            while (s >= stages) { s -= stages; parity ^= 1u; }
        }
    } else {
        // ---------------- epilogue (both blocks): own 128 rows of the tile; what is past the tile's rows or
        // wholly below the diagonal is not stored (the reduction does not read it)
        const int q = warp & 3;
        const int row0 = (int)rank * HALF + q * 32;
        const bool used = row0 < rows;
        const int c_first = diag && !sym ? row0 : 0;         // row0 is a multiple of 32
        float *dst = a.partials + (size_t)blockIdx.x * (EXT ? a.pitch : HALF * BN) + (q * 32 + lane) * 4;         // columns c .. c+3: + c HALF
        // columns in use: c_first .. width, and where the tile carries left-over columns all in between and after them
        const int c_end = ext > 0 ? BN + (ext * (corner && q * 32 < ext / 2 ? 2 : 1) + 31) / 32 * 32 : width;
        const uint32_t leader_acc_empty0 = map_to_cta(smem_u32(&acc_empty[0]), 0);
        if (nphases == 0 && used) {
            for (int c0 = c_first; c0 < c_end; c0 += 4) *reinterpret_cast<float4 *>(dst + c0 * HALF) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int ph = 0; ph < nphases; ++ph) {
            const int buf = ext > 0 ? 0 : ph & 1;
            if (!mbar_wait(&acc_full[buf], (uint32_t)((ext > 0 ? ph : ph >> 1) & 1), abort_flag, a.status, 3)) break;
            tc_fence_after();
            if (used && ext > 0) {
                // The MMAs wait until the accumulators have been read: 32 columns are on their way from tensor memory while the
                // 32 before them are added to the partial tile, in L2, so that nothing has to come back for it.
                const uint32_t t0 = tmem_base + ((uint32_t)(q * 32) << 16);
                auto add = [&](int c0, const uint32_t (&r)[32]) {
                    if (ph > 0) {
                        if (c0 < BN) {
                            m2tc_add_in_l2(dst + c0 * HALF, r, ~0u);
                        } else {
                            // the left-over columns and those of the corner, without what fills them up
                            const int c = c0 - BN, left = a.d - ecol;
                            auto low = [](int n) { return n <= 0 ? 0u : n >= 32 ? ~0u : (1u << n) - 1; };
                            m2tc_add_in_l2(dst + c0 * HALF, r, low(left - c) | (low(ext - c + left) & ~low(ext - c)));
                        }
                        return;
                    }
#pragma unroll
                    for (int e = 0; e < 32; e += 4)
                        *reinterpret_cast<float4 *>(dst + (c0 + e) * HALF) = make_float4(
                            __uint_as_float(r[e]), __uint_as_float(r[e + 1]), __uint_as_float(r[e + 2]), __uint_as_float(r[e + 3]));
                };
                uint32_t r0[32], r1[32];
                tmem_ld_32x32(t0 + (uint32_t)c_first, r0);
#pragma unroll 1
                for (int c0 = c_first; c0 < c_end; c0 += 64) {
                    tmem_ld_wait();
                    if (c0 + 32 < c_end) tmem_ld_32x32(t0 + (uint32_t)(c0 + 32), r1);
                    add(c0, r0);
                    if (c0 + 32 < c_end) {
                        tmem_ld_wait();
                        if (c0 + 64 < c_end) tmem_ld_32x32(t0 + (uint32_t)(c0 + 64), r0);
                        add(c0 + 32, r1);
                    }
                }
            } else if (used) {
#pragma unroll 1
                for (int c0 = c_first; c0 < width; c0 += 32) {
                    uint32_t r[32];
                    tmem_ld_32x32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * BN + c0), r);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; e += 4) {
                        float4 v = make_float4(__uint_as_float(r[e]), __uint_as_float(r[e + 1]), __uint_as_float(r[e + 2]),
                                               __uint_as_float(r[e + 3]));
                        float4 *p = reinterpret_cast<float4 *>(dst + (c0 + e) * HALF);
                        if (ph > 0) {
                            const float4 o = *p;
                            v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
                        }
                        *p = v;
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_acc_empty0 + (uint32_t)(buf * sizeof(uint64_t)));
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                      // no block leaves while its peer may still signal it
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, TMEM_COLS);
    }
}

// Sums of the partial tiles over the sample ranges, i <= j < d only.  A warp owns 32 rows and four columns, which lie side
// by side in a partial tile as the epilogue's warps wrote them: with whole rows there, a warp's store met 32 lines, and
// the last flush of a 256-wide tile took 4 us.  `wps` warps share a unit: the first adds ranges 0, wps, 2 wps, ..., four
// loads at a time, and so on, then their sums are added in order.  (Ten loads at a time and eight ranges per warp take so
// many registers that the blocks do not all fit beside the next kernel's: [4096,1024] 17.4 us, now 14.2; fourth moment of
// [4096,24] 18.8, now 16.0.)
// PAIRS: X holds pair features in the order of pair_layout.cuh; pairs[column] is the pair of a column, and an entry goes
// to the place of its 4-tuple in the packed 4-simplex, if this is the product that was chosen for that tuple.
__host__ __device__ inline int m2tc_sum_warps(int nsplit) { return nsplit <= 4 ? 1 : nsplit <= 8 ? 2 : nsplit <= 16 ? 4 : 8; }
// EXT: some tiles carry left-over columns (an instance of its own: with them in it the others took 1 to 2 us longer).
// SYM: full diagonal tiles hold S, of which (S + S^T) / 2 is the result.
template <bool PAIRS, bool EXT, bool SYM>
__global__ void __launch_bounds__(256)
moment2_tc_reduce_kernel(const float *partials, float *out, int d, int features, int within, int64_t out_elems,
                         const unsigned *pairs, int pitch, const __grid_constant__ m2tc::TileTable tab)
{
    using namespace m2tc;
    __shared__ float4 part[2][8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the tiles, then the left-over columns of each tile that carries them, then the corner
    const int e = EXT ? (int)blockIdx.x - tab.ntiles : -1;
    const bool corner = EXT && e >= (int)tab.next;
    const int tile = e < 0 ? (int)blockIdx.x : tab.carrier[corner ? (int)tab.next - 1 : e], ext = 16 * tab.ext[tile];
    const int row = 8 * (corner ? tab.ext_col : tab.row[tile]), col = 8 * (e < 0 ? tab.col[tile] : tab.ext_col);
    const int rows = corner ? min(ext, d - row) : tab.rows[tile], block_rows = corner ? ext / 2 : HALF;
    const int at_col = e < 0 ? 0 : corner ? BN + ext : BN;                                    // in the partial tile
    const int quads = (min(e < 0 ? 32 * (int)tab.width[tile] : ext, d - col) + 3) / 4, units = (rows + 31) / 32 * quads;
    const int first = tab.first[tile], nsplit = tab.first[tile + 1] - first;
    const int wps = m2tc_sum_warps(nsplit);
    const int per = 8 / wps, w0 = warp % wps;
    const int block = EXT ? pitch : HALF * BN;           // floats of a block's partial tile
    const size_t stride = (size_t)2 * block;
    constexpr int BATCH = 4;
    pdl_wait();
    pdl_trigger();
    int buf = 0;
    for (int u0 = blockIdx.y * per; u0 < units; u0 += gridDim.y * per) {
        const int u = u0 + warp / wps, r = u / quads * 32 + lane, c = u % quads * 4;      // this thread's row, columns c .. c+3
        const int gi = row + r, gj = col + c;
        // what is loaded does not wait for what has to be looked up
        const bool use = u < units && r < rows && gj + 4 > (PAIRS && gi >= within ? 0 : gi);
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        const int second = EXT ? r >= block_rows ? 1 : 0 : r >> 7, in_block = EXT ? r - second * block_rows : r & 127;
        const float *base = partials + (size_t)(2 * first + second) * block + (at_col + c) * HALF + in_block * 4;
        for (int k0 = w0; k0 < nsplit; k0 += BATCH * wps) {
            float4 v[BATCH];
#pragma unroll
            for (int e = 0; e < BATCH; ++e)
                v[e] = use && k0 + wps * e < nsplit ? __ldcg(reinterpret_cast<const float4 *>(base + (size_t)(k0 + wps * e) * stride))
                                                    : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int e = 0; e < BATCH; ++e) { s.x += v[e].x; s.y += v[e].y; s.z += v[e].z; s.w += v[e].w; }
        }
        if (SYM && e < 0 && tab.diag[tile] && 32 * (int)tab.width[tile] == BN) {
            // S^T of the four columns: rows c .. c+3, column r.  Four lanes read four columns of these rows, 64 bytes in a row, and
            // exchange their sums.  Halved before they are added: their sum may be no fp32 number.
            const int j = lane & 3;
            const bool in = u < units && (r & ~3) < rows && gj + 4 > (gi & ~3);
            const float *t = partials + (size_t)(2 * first + ((c + j) >> 7)) * block + (r & ~3) * HALF + ((c + j) & 127) * 4;
            float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int k0 = w0; k0 < nsplit; k0 += BATCH * wps) {
                float4 v[BATCH];
#pragma unroll
                for (int b = 0; b < BATCH; ++b)
                    v[b] = in && k0 + wps * b < nsplit ? __ldcg(reinterpret_cast<const float4 *>(t + (size_t)(k0 + wps * b) * stride))
                                                       : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int b = 0; b < BATCH; ++b) { y.x += v[b].x; y.y += v[b].y; y.z += v[b].z; y.w += v[b].w; }
            }
            auto exchange = [&](float &lo, float &hi, int bit) {           // of lanes that differ in `bit`
                const float got = __shfl_xor_sync(0xFFFFFFFFu, lane & bit ? lo : hi, bit);
                (lane & bit ? lo : hi) = got;
            };
            exchange(y.x, y.y, 1); exchange(y.z, y.w, 1);
            exchange(y.x, y.z, 2); exchange(y.y, y.w, 2);
            s.x = fmaf(0.5f, y.x, 0.5f * s.x); s.y = fmaf(0.5f, y.y, 0.5f * s.y);
            s.z = fmaf(0.5f, y.z, 0.5f * s.z); s.w = fmaf(0.5f, y.w, 0.5f * s.w);
        }
        int at[4];                                         // where the columns go to, -1: not an output
        const int at0 = PAIRS ? 0 : (int)tri_encode(d, gi, gj);
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            at[x] = -1;
            if (PAIRS) {
                int i, j, k, l;
                if (use && gj + x < d && pair_product(pairs[gi], pairs[gj + x], i, j, k, l)) at[x] = pair_place(features, i, j, k, l);
            } else if (use && gi <= gj + x && gj + x < d) {
                at[x] = at0 + x;
            }
        }
        if (wps > 1) {
            part[buf][warp][lane] = s;
            __syncthreads();
        }
        if (w0 == 0 && use) {
            for (int w = 1; w < wps; ++w) {
                const float4 v = part[buf][warp + w][lane];
                s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
            }
            const float f[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (at[x] >= 0 && ST_BOUNDS_OK(at[x], out_elems, PAIRS ? 7 : 2)) out[at[x]] = f[x];
        }
        buf ^= 1;
    }
}

struct M2TcPlan {
    m2tc::TileTable tab;
    int chunks_total, stages, nb, na, pitch;
    size_t partial_bytes, smem;
    double time;                                       // stages of a full tile that the call takes
    bool ok;
};

// Time per stage, a full tile = 1: the 256 columns of A are loaded whatever the width (the MMA alone would be 43 cycles
// at 64 columns against 128; with 0.35 in place of 0.7 [400000,304] bf16 ran 127 us instead of 111).  ext: left-over columns
// that the tile carries along, times the products that it makes of them (with those for nothing [262144,520] split ran 325 us
// instead of 311, [131072,776] 320 and 288, [131072,896] 412 and 340).
static double m2tc_cost(int width, int ext, int products)
{
    return 0.7 + 0.3 * width / m2tc::BN + (ext > 0 ? products * (0.08 + (double)ext / m2tc::BN) : 0);
}
// M2_EXACT, where a stage takes as long as its values are converted: us per 32 samples 1.36, on the diagonal 1.2, 1.27 at 32
// columns off it, 1.0, 0.73 and 0.65 where all columns are 128, 64 or four.
static double m2tc_exact_cost(int rows, int width, bool diag)
{
    if (!diag) return 0.92 + 0.08 * width / m2tc::BN;
    return rows > m2tc::HALF ? 0.88 : 0.47 + 0.26 * rows / m2tc::HALF;
}

constexpr double m2tc_stage_cycles(int mode) { return mode == M2_CONV ? 1226 : 512; }      // a full tile's
template <int MODE>
static double m2tc_cycles(int64_t N, double cost)          // of a cluster, where tiles of this cost together share the chip
{
    return (double)((N + m2tc::Shape<MODE>::KROWS - 1) / m2tc::Shape<MODE>::KROWS) * cost * m2tc_stage_cycles(MODE) / (sm_count_or_default() / 2);
}
// Columns that are left over after `full` tiles of 256: carried along by the tiles on the diagonal, or tiles of their own.  The
// epilogue of a tile that carries them has up to twice the columns, and the sum more parts: a fixed time that the samples of a
// cluster, in cycles of their stages, have to outweigh.  us, tiles of their own / carried: TF32 [20000,300] 17.9 / 19.1, [60000,300]
// 35.8 / 29.0, [20000,380] 19.7 / 24.1, [60000,380] 39.6 / 36.9; bf16 [20000,264] 13.3 / 15.2, [60000,264] 22.7 / 20.8, [20000,800] 26.3 /
// 27.7, [60000,800] 59 / 53; split [6000,520] 19.5 / 21.7, [20000,520] 39.4 / 36.0, [20000,384] 24.4 / 27.4, [60000,384] 51.5 / 43.8.
// The tiles that carry them are longer, too, which costs more than it saves where a tile has a cluster or two.  M2TC_CARRY_GAIN: the
// longest cluster has to become that much shorter.  1800 features are 36 tiles of two clusters each, or 28 of which those off the
// diagonal have two as well; 3200 are 91, or 78 on 74 pairs of SMs of which the last takes twice as long.  us in rows of calls: TF32
// [81405,1800] 524 / 566, [80567,2568] 1033 / 1098, [80386,3080] 1836 / 2296, [78977,3200] 1702 / 2514, bf16 [63182,3200] 712 / 1087, split
// [52771,3200] 1916 / 2701; a gain where the longest becomes 6 % shorter, TF32 [97053,1152] 292 / 266, 21 %, [81425,2176] 890 / 799, and
// 43 %, bf16 [64795,2056] 463 / 278.
constexpr double M2TC_CARRY_GAIN = 0.97;
template <int MODE>
static bool m2tc_carry(int64_t N, int full, int left_over)
{
    if (MODE == M2_EXACT || full == 0 || left_over == 0 || left_over > m2tc::HALF) return false;
    const int tiles = full * (full + 1) / 2, ext = (left_over + 15) / 16 * 16;
    const double cycles = m2tc_cycles<MODE>(N, tiles + (full + 1) * (m2tc_cost(m2tc::BN, ext, 1) - 1));
    return cycles >= (MODE == M2_CONV ? 1.6 : 1.0) * (6000 + 130 * ext + 3500 * (tiles - 1));
}

// Full diagonal tiles of M2_CONV may make two products instead of three, S = hi^T hi + hi^T 2 lo: C = (S + S^T) / 2 (their error is
// smaller too, as fewer sums are truncated: 2-norm against 64 bits [262144,520] 8.9e-6 with three, 7.5e-6).  M2TC_SYM_*: what a stage of
// such a tile takes less, a full tile = 1, as rows of calls show it (wide tiles run at the power cap, where fewer products are more
// clock): with left-over columns, for a table of one tile, others.  Their clusters have twice the sums to add and the sum has S^T to read,
// M2TC_SYM_SUM cycles for each: the two products are taken where the call is shortened by more, that is where the clusters that
// they free shorten the longest one.  us in rows of calls / alone, three products -> two: taken [50000,512] 53 / 60 -> 49 / 59,
// [160000,512] 159 / 167 -> 149 / 157, [60000,520] 79 / 89 -> 76 / 85, [120000,520] 146 / 153 -> 132 / 142, [60000,776] 137 / 145 -> 129 / 136,
// [10000,1024] 42 / 48 -> 37 / 44, [262144,1024] 990 / 1028 -> 861 / 896, [60000,1280] 358 / 363 -> 290 / 304, [10000,3072] 369 / 378 -> 350 / 359,
// [300000,256] 89 / 93 -> 82 / 94; not taken [120000,256] 41 / 48 -> 44 / 52, [60000,280] 34 / 42 -> 37 / 45, [15000,896] 53 / 60 -> 54 / 62,
// [120000,1536] 949 / 980 -> 966 / 984, [30000,1800] 330 / 339 -> 347 / 356, [60000,2048] 762 / 793 -> 769 / 797.
constexpr double M2TC_SYM_EXT = 0.1, M2TC_SYM_ONE = 0.06, M2TC_SYM_FULL = 0.2, M2TC_SYM_SUM = 110;

// Tiles of a plan while it is made.
struct M2TcTiles {
    M2TcPlan *p;
    int n;
    bool one;                                          // the only tile of its plan
    double cost[m2tc::MAX_TILES];
    template <int MODE>
    bool add(int row, int rows, int col, int width, bool diag, int ext_col = 0, int ext = 0, bool corner = false)
    {
        using namespace m2tc;
        using S = Shape<MODE>;
        if (n >= MAX_TILES) return false;
        p->tab.row[n] = (unsigned short)(row / 8);
        p->tab.rows[n] = (unsigned short)rows;
        p->tab.col[n] = (unsigned short)(col / 8);
        p->tab.width[n] = (unsigned char)(width / 32);
        p->tab.diag[n] = diag ? 1 : 0;
        cost[n] = MODE == M2_EXACT ? m2tc_exact_cost(rows, width, diag) : m2tc_cost(width, ext, corner ? 2 : 1);
        if (p->tab.sym && diag && width == BN) cost[n] -= ext > 0 ? M2TC_SYM_EXT : one ? M2TC_SYM_ONE : M2TC_SYM_FULL;
        const bool lead = diag && rows <= HALF;
        const int cols_b = lead && rows > width / 2 ? rows : width / 2, nb = (cols_b + S::BOXC - 1) / S::BOXC;
        if (nb > p->nb) p->nb = nb;
        if (ext > 0 || (!(diag && width == BN) && !lead)) {
            const int n_a = ext > 0 ? ext / 2 : rows;
            const int na = n_a >= HALF || (MODE == M2_CONV && ext > 0) ? S::NBOX : (n_a + S::BOXC - 1) / S::BOXC;     // (with room for hi / 2)
            if (na > p->na) p->na = na;
        }
        p->tab.ext[n] = (unsigned char)(ext / 16);
        if (ext > 0) {
            if (p->tab.next >= MAX_EXT) return false;
            p->tab.carrier[p->tab.next++] = (unsigned char)n;
            p->tab.ext_col = (unsigned short)(ext_col / 8);
            if (corner) p->tab.corner = 1;
        }
        const int columns = BN + (ext * (corner ? 2 : 1) + 31) / 32 * 32;             // written 32 at a time
        if (columns * HALF > p->pitch) p->pitch = columns * HALF;
        ++n;
        return true;
    }
};

// Sample ranges, stages and sizes of a plan whose tiles are known.
template <int MODE>
static void m2tc_finish(M2TcPlan &p, const M2TcTiles &t, int64_t N)
{
    using namespace m2tc;
    using S = Shape<MODE>;
    const int n = t.n;
    const double *cost = t.cost;
    for (int i = n; i < MAX_TILES; ++i) p.tab.diag[i] = p.tab.width[i] = p.tab.row[i] = p.tab.rows[i] = p.tab.col[i] = 0;
    p.tab.ntiles = n;
    const int64_t chunks = (N + S::KROWS - 1) / S::KROWS;
    if (chunks > (int64_t(1) << 30)) return;
    p.chunks_total = (int)chunks;
    const size_t stage = (size_t)S::PARTS * (p.nb + p.na) * S::BOX_BYTES;
    p.stages = (int)((MODE == M2_CONV ? STAGES_BYTES_CONV : n == 1 ? STAGES_BYTES_1 : STAGES_BYTES) / stage);
    if (p.stages > MAX_STAGES) p.stages = MAX_STAGES;
    // a stage always belongs to the same group of converting warps: a group that came by only every other time could not
    // tell the two apart by the parity of the barrier
    if (MODE == M2_CONV) p.stages -= p.stages % CONV_GROUPS;
    p.smem = MODE == M2_EXACT ? EX_SMEM : (size_t)p.stages * stage + (size_t)(S::NBOX - p.na) * S::BOX_BYTES * (MODE == M2_CONV ? 2 : 1) + 1024 + 1024;
    // Clusters (one per pair of SMs) go to the tiles in proportion to their cost, the remaining ones each to the tile whose
    // share of the samples takes longest; then every tile gives back what it does not need to keep up with the slowest.
    // Tiles of equal width so get equal shares: their clusters run in step and share X in L2 (with unequal shares the wide
    // case was 12-20% slower on more SMs).
    int split[MAX_TILES];
    const int clusters = sm_count_or_default() / 2;
    double sum = 0;
    for (int i = 0; i < n; ++i) sum += cost[i];
    int64_t left = clusters;
    for (int i = 0; i < n; ++i) {
        int64_t k = (int64_t)(cost[i] * clusters / sum);
        k = k < 1 ? 1 : k > chunks ? chunks : k;
        split[i] = (int)k;
        left -= k;
    }
    double longest = 0;
    for (;;) {
        int worst = 0;
        for (int i = 1; i < n; ++i)
            if (cost[i] * split[worst] > cost[worst] * split[i]) worst = i;
        longest = cost[worst] / split[worst];
        if (left <= 0 || split[worst] >= chunks) break;
        ++split[worst];
        --left;
    }
    int first = 0;
    for (int i = 0; i < n; ++i) {
        while (split[i] > 1 && cost[i] / (split[i] - 1) <= longest * (1 + 1e-9)) --split[i];
        p.tab.first[i] = (unsigned short)first;
        first += split[i];
    }
    for (int i = n; i <= MAX_TILES; ++i) p.tab.first[i] = (unsigned short)first;
    p.partial_bytes = (size_t)2 * first * p.pitch * sizeof(float);
    if (first > clusters) {                            // several waves: each cluster in turn on the pair of SMs that is free first
        double busy[MAX_TILES] = {};                   // a heap, that pair in front
        const int pairs = clusters < MAX_TILES ? clusters : MAX_TILES;
        longest = 0;
        for (int i = 0; i < n; ++i)
            for (int k = 0; k < split[i]; ++k) {
                std::pop_heap(busy, busy + pairs, std::greater<double>());
                busy[pairs - 1] += cost[i] / split[i];
                if (busy[pairs - 1] > longest) longest = busy[pairs - 1];
                std::push_heap(busy, busy + pairs, std::greater<double>());
            }
    }
    p.time = (double)chunks * longest;
    p.ok = true;
}

template <int MODE>
static M2TcPlan m2tc_plan_of(int64_t N, int64_t d, bool dense, bool carry, bool sym)
{
    using namespace m2tc;
    M2TcPlan p{};
    const int full = (int)(d / BM), ext = carry ? (int)(d % BM + 15) / 16 * 16 : 0;
    const int nt = carry ? full : (int)((d + BM - 1) / BM);
    M2TcTiles t{&p, 0, nt == 1, {}};
    p.tab.sym = sym;
    for (int tn = 0; tn < nt; ++tn)
        for (int tm = 0; tm < nt; ++tm) {
            if (tm > tn && !dense) continue;
            const int left = (int)d - tn * BN, below = (int)d - tm * BM;
            int width = left >= BN ? BN : (left + 31) / 32 * 32;
            // M2_EXACT: with all 256 columns A holds B, and half as many values are converted ([65536,200] 52 us, now 45)
            if (MODE == M2_EXACT && tm == tn && width > HALF) width = BN;
            const int e = tm == tn ? ext : 0;
            if (!t.add<MODE>(tm * BM, below < BM ? below : BM, tn * BN, width, tm == tn, full * BM, e, tm == nt - 1)) return p;
        }
    m2tc_finish<MODE>(p, t, N);
    return p;
}

template <int MODE>
static M2TcPlan m2tc_plan(int64_t N, int64_t d, unsigned flags)
{
    using namespace m2tc;
    const bool dense = (flags & ST_FLAG_DENSE_CONTROL) != 0;
    M2TcPlan three = m2tc_plan_of<MODE>(N, d, dense, false, false);
    bool carry = !dense && m2tc_carry<MODE>(N, (int)(d / BM), (int)(d % BM));
    if (carry) {
        const M2TcPlan with = m2tc_plan_of<MODE>(N, d, false, true, false);
        carry = with.ok && (!three.ok || with.time < M2TC_CARRY_GAIN * three.time);
        if (carry) three = with;
    }
    if constexpr (MODE == M2_CONV) {
        const double most = M2TC_SYM_FULL * m2tc_stage_cycles(MODE) * three.time;            // that two products can save
        if (dense || d < BN || !three.ok || most < M2TC_SYM_SUM) return three;
        const M2TcPlan two = m2tc_plan_of<MODE>(N, d, dense, carry, true);
        int clusters = 0;
        for (int i = 0; i < two.tab.ntiles; ++i)
            if (two.tab.diag[i] && 32 * (int)two.tab.width[i] == BN) clusters += two.tab.first[i + 1] - two.tab.first[i];
        if (two.ok && (three.time - two.time) * m2tc_stage_cycles(MODE) >= M2TC_SYM_SUM * clusters) return two;
    }
    return three;
}

// Tiles of the products of pair features that pair_layout.cuh names, in turn to f(row, rows, col, width, on the diagonal).
// (Left-over columns carried by the tile on the diagonal: [30011,45] 92 us without, 96 with them.)
template <class F>
static void pair_tiles(const PairLayout &L, F f)
{
    using namespace m2tc;
    auto strip = [&](int row, int rows, int col, int end) {
        for (int c = col; c < end; c += BN) f(row, rows, c, end - c >= BN ? BN : (end - c + 31) / 32 * 32, c == row);
    };
    for (int r = 0; r < L.within; r += BM) strip(r, L.within - r < BM ? L.within - r : BM, r, L.cols);
    for (int r = 0; r < L.rows_n && L.prod_n > 0; r += BM)
        strip(L.rows + r, L.rows_n - r < BM ? L.rows_n - r : BM, L.prod, L.prod + L.prod_n);
}

// Ranges of the features: one, two or three of about equal size, or four and a smaller one, whichever gives the cheapest
// tiles.  (Four and a smaller one: 45 features take 256 rows as 11, 11, 11, 10 and 2, but 261 as five nines.)
// one: a single range.  That is the product (i,j) (k,l) of a 4-tuple i <= j <= k <= l everywhere, which the bf16 form keeps:
// its results depend on the pairing by a rounding of bf16 (at 409 samples up to 1.6 % of the outputs' mean size).
PairLayout pair_layout(int features, bool one)
{
    thread_local PairLayout kept[2] = {};                  // of the last call: the size query and the call itself need it
    PairLayout &best = kept[one ? 1 : 0];
    if (best.features == features) return best;
    double least = 0;
    for (int option = 0; option < (one ? 1 : 4 + features / 4); ++option) {
        const int last = option < 3 ? 0 : option - 3, m = option < 3 ? option + 1 : 4;   // m equal ranges and the last one
        PairLayout L{};
        int n[5] = {0, 0, 0, 0, last}, within = 0;
        for (int g = 0; g < m; ++g) n[g] = (features - last) / m + (g < (features - last) % m ? 1 : 0);
        for (int g = 0; g < 5; ++g) {
            L.lo[g + 1] = L.lo[g] + n[g];
            within += n[g] * (n[g] + 1) / 2;
        }
        L.features = features;
        L.within = within;
        L.rows_n = n[0] * n[1] + (n[0] + n[1]) * n[4];
        L.prod_n = n[2] * n[3] + (n[2] + n[3]) * n[4];
        L.rows = (within + 7) / 8 * 8;
        L.prod = (L.rows + L.rows_n + 7) / 8 * 8;
        L.cols = L.prod + (int)tri_rows(features) - within - L.rows_n;
        double cost = 0;
        pair_tiles(L, [&](int, int, int, int width, bool) { cost += m2tc_cost(width, 0, 0); });
        if (option == 0 || cost < least) {
            best = L;
            least = cost;
        }
    }
    return best;
}

template <int MODE>
static const M2TcPlan &m2tc_plan_pairs(int64_t N, const PairLayout &L)
{
    thread_local M2TcPlan p{};                             // of the last call, as above
    thread_local int64_t of[3] = {0, 0, 0};
    const int64_t now[3] = {N, L.features, sm_count_or_default()};
    if (of[0] == now[0] && of[1] == now[1] && of[2] == now[2]) return p;
    for (int i = 0; i < 3; ++i) of[i] = now[i];
    p = M2TcPlan{};
    M2TcTiles t{&p, 0, false, {}};
    bool ok = true;
    pair_tiles(L, [&](int row, int rows, int col, int width, bool diag) { ok = ok && t.add<MODE>(row, rows, col, width, diag); });
    if (ok) m2tc_finish<MODE>(p, t, N);
    return p;
}

template <int MODE> static auto m2tc_kernel(bool ext)
{
    if constexpr (MODE == M2_EXACT) return moment2_exact_kernel;
    else if constexpr (MODE == M2_SPLIT) return moment2_tc_kernel<MODE, false>;        // products of pairs carry none
    else return ext ? moment2_tc_kernel<MODE, true> : moment2_tc_kernel<MODE, false>;
}

// Launches the tile kernel and the sum of its partial tiles.  rows: rows of X in memory; pairs: X holds the pair features
// of `features` features and the result goes to their packed 4-simplex.
template <int MODE>
static st_status m2tc_launch(const M2TcPlan &q, const void *X, int64_t rows, int64_t d, int64_t ldx, float *out, float *partials,
                             unsigned *status, cudaStream_t stream, int64_t lo_row0 = 0, const unsigned *pairs = nullptr, int features = 0, int within = 0)
{
    using S = m2tc::Shape<MODE>;
    CUtensorMap tmap;
    constexpr bool WORDS = MODE == M2_TF32 || MODE == M2_CONV || MODE == M2_EXACT;
    if (!tc::make_tmap_2d(&tmap, WORDS ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, X, (uint64_t)rows,
                          (uint64_t)d, (uint64_t)ldx * (WORDS ? 4 : 2), WORDS ? 32 : S::BOXC, S::KROWS,
                          MODE == M2_TF32 ? CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B : CU_TENSOR_MAP_SWIZZLE_128B))
        return ST_ERR_CUDA;
    m2tc::Args a;
    a.partials = partials; a.status = status;
    a.chunks_total = q.chunks_total; a.stages = q.stages; a.nb = q.nb; a.na = q.na; a.pitch = q.pitch; a.lo_row0 = (int)lo_row0; a.d = (int)d;
    a.X = (const float *)X; a.N = rows; a.ldx = ldx;
    a.tab = q.tab;
    const auto kernel = m2tc_kernel<MODE>(q.tab.next > 0);
    if (!ensure_dynamic_smem(kernel, q.smem)) return ST_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (unsigned)q.tab.first[q.tab.ntiles]);
    cfg.blockDim = dim3(MODE == M2_EXACT ? m2tc::EX_THREADS : MODE == M2_CONV ? m2tc::THREADS + m2tc::CONV_THREADS : m2tc::THREADS);
    cfg.dynamicSmemBytes = q.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if (cudaLaunchKernelEx(&cfg, kernel, tmap, a) != cudaSuccess) {
        (void)cudaGetLastError();
        return ST_ERR_CUDA;
    }
    // blocks for all units of a tile, up to 16 per SM together: more of them would only be in the way of the next kernel's
    unsigned blocks = 1;
    for (int t = 0; t < q.tab.ntiles; ++t) {
        const unsigned per = 8u / (unsigned)m2tc_sum_warps(q.tab.first[t + 1] - q.tab.first[t]);
        const unsigned n = ((unsigned)((q.tab.rows[t] + 31) / 32 * 8 * q.tab.width[t]) + per - 1) / per;
        if (n > blocks) blocks = n;
    }
    const unsigned most = 16u * (unsigned)sm_count_or_default() / (unsigned)q.tab.ntiles;
    if (blocks > most) blocks = most < 64 ? 64 : most;
    const dim3 rgrid((unsigned)(q.tab.ntiles + q.tab.next + q.tab.corner), blocks);
    constexpr bool CONV = MODE == M2_CONV;
    const auto sum = pairs ? moment2_tc_reduce_kernel<true, false, false>
                   : q.tab.next > 0 ? (q.tab.sym ? moment2_tc_reduce_kernel<false, true, CONV> : moment2_tc_reduce_kernel<false, true, false>)
                                    : (q.tab.sym ? moment2_tc_reduce_kernel<false, false, CONV> : moment2_tc_reduce_kernel<false, false, false>);
    return launch(sum,
                  rgrid, 256, 0, stream, partials, out, (int)d,
                  features, within, pairs ? simp4_rows(features) : tri_rows(d), pairs, q.pitch, q.tab);
}

// One workspace serves the structured call and its dense control, and the same calls of fewer samples too: their plan may be one that
// is not taken for these samples, with tiles of their own for the left-over columns or with another number of products, and may need
// more room.
template <int MODE>
static size_t m2tc_workspace(int64_t N, int64_t d, unsigned flags)
{
    if (N <= 0 || d <= 0 || d > 4096 || N > (int64_t(1) << 31) - 64) return 0;
    const M2TcPlan plain = m2tc_plan<MODE>(N, d, 0u), dense = m2tc_plan<MODE>(N, d, ST_FLAG_DENSE_CONTROL);
    if (!(flags & ST_FLAG_DENSE_CONTROL ? dense : plain).ok) return 0;
    size_t bytes = 0;
    auto fit = [&](const M2TcPlan &q) {
        if (q.ok && q.partial_bytes > bytes) bytes = q.partial_bytes;
    };
    fit(plain);
    fit(dense);
    for (int carry = 0; carry <= (plain.tab.next > 0); ++carry)
        for (int sym = 0; sym <= (MODE == M2_CONV && d >= m2tc::BN); ++sym) fit(m2tc_plan_of<MODE>(N, d, false, carry != 0, sym != 0));
    return kWsHeaderBytes + bytes;
}

template <int MODE>
static st_status m2tc_run(const void *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes, unsigned flags,
                          cudaStream_t stream)
{
    if (d > 4096 || N > (int64_t(1) << 31) - 64) return ST_ERR_UNSUPPORTED;
    const M2TcPlan q = m2tc_plan<MODE>(N, d, flags);
    if (!q.ok) return ST_ERR_UNSUPPORTED;
    if (!ws || ws_bytes < kWsHeaderBytes + q.partial_bytes) return ST_ERR_WORKSPACE;
    if (!aligned256(ws)) return ST_ERR_ALIGN;
    return m2tc_launch<MODE>(q, X, N, d, ldx, out, (float *)((unsigned char *)ws + kWsHeaderBytes), (unsigned *)ws, stream);
}

// fp32 input read as TF32 (any d that is a multiple of 4: tiles beyond d are zero-filled by the copies)
size_t moment2_tf32_tc_workspace(int64_t N, int64_t d, unsigned flags)
{
    return d % 4 != 0 ? 0 : m2tc_workspace<M2_TF32>(N, d, flags);
}

st_status moment2_tf32_tc(const void *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes,
                          unsigned flags, cudaStream_t stream)
{
    if (d % 4 != 0 || ldx % 4 != 0) return ST_ERR_ALIGN;
    return m2tc_run<M2_TF32>(X, N, d, ldx, out, ws, ws_bytes, flags, stream);
}

size_t moment2_bf16_tc_workspace(int64_t N, int64_t d, unsigned flags)
{
    return d % 8 != 0 ? 0 : m2tc_workspace<M2_BF16>(N, d, flags);
}

st_status moment2_bf16_tc(const void *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes,
                          unsigned flags, cudaStream_t stream)
{
    if (d % 8 != 0 || ldx % 8 != 0) return ST_ERR_ALIGN;
    return m2tc_run<M2_BF16>(X, N, d, ldx, out, ws, ws_bytes, flags, stream);
}

// fp32 input at the error of fp32 arithmetic (moment2_exact.cuh); rows of X that a tensor map can name
size_t moment2_exact_tc_workspace(int64_t N, int64_t d, unsigned flags) { return m2tc_workspace<M2_EXACT>(N, d, flags); }

st_status moment2_exact_tc(const float *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes,
                           unsigned flags, cudaStream_t stream)
{
    if (ldx % 4 != 0) return ST_ERR_ALIGN;
    if (!m2tc_exact_fits()) return ST_ERR_UNSUPPORTED;
    return m2tc_run<M2_EXACT>(X, N, d, ldx, out, ws, ws_bytes, flags, stream);
}

// ---------------------------------------------------------------------------------------------
// fp32 input at the fp32 tolerance on the tensor cores (ST_FLAG_TC_SPLIT): x = hi + lo with hi = bf16(x) and
// lo = bf16(x - hi) (what is left is below 2^-16 |x|), and the pair kernel adds hi^T hi + hi^T lo + lo^T hi, or on full diagonal tiles
// hi^T hi + hi^T 2 lo, whose symmetric part that is (M2TC_SYM_SUM); either way lo^T lo, below 2^-16 of the result, is left out.
size_t moment2_split_tc_workspace(int64_t N, int64_t d, unsigned flags)
{
    return d % 8 != 0 || N > (int64_t(1) << 29) ? 0 : m2tc_workspace<M2_CONV>(N, d, flags);
}

st_status moment2_split_tc(const float *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes,
                           unsigned flags, cudaStream_t stream)
{
    if (d % 8 != 0 || ldx % 4 != 0) return ST_ERR_ALIGN;
    if (N > (int64_t(1) << 29)) return ST_ERR_UNSUPPORTED;
    return m2tc_run<M2_CONV>(X, N, d, ldx, out, ws, ws_bytes, flags, stream);
}

// The products of pair features that the caller has written (moment4.cu), straight into the packed 4-simplex.  split:
// P = [hi rows; lo rows], each part N rounded up to 64 rows with zero rows at the end; else N rows of bf16.  ldp: columns
// of P, those of the layout and zeros after them.
int64_t moment2_split_part_rows(int64_t N) { return (N + 63) / 64 * 64; }

size_t moment2_pairs_partial_bytes(int64_t N, const PairLayout &L, bool split)
{
    // the copies' row coordinate has 31 bits, and split features have two rows for a sample
    if (N <= 0 || N > (split ? int64_t(1) << 29 : (int64_t(1) << 31) - 64)) return 0;
    const M2TcPlan &q = split ? m2tc_plan_pairs<M2_SPLIT>(N, L) : m2tc_plan_pairs<M2_BF16>(N, L);
    return q.ok ? q.partial_bytes : 0;
}

st_status moment2_pairs_tc(const void *P, int64_t N, const PairLayout &L, int64_t ldp, bool split, const unsigned *pairs, float *out,
                           float *partials, unsigned *status, cudaStream_t stream)
{
    const int64_t Np = moment2_split_part_rows(N);
    if (split)
        return m2tc_launch<M2_SPLIT>(m2tc_plan_pairs<M2_SPLIT>(N, L), P, 2 * Np, ldp, ldp, out, partials, status, stream, (int)Np, pairs,
                                     L.features, L.within);
    return m2tc_launch<M2_BF16>(m2tc_plan_pairs<M2_BF16>(N, L), P, N, ldp, ldp, out, partials, status, stream, 0, pairs, L.features, L.within);
}

}  // namespace st
