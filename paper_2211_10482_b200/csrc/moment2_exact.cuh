// Second moment of fp32 samples on the tensor cores, at the error of fp32 arithmetic (M2_EXACT of moment2_tc.cu, which includes
// this file; tiles, clusters and the sum of the partial tiles are those of that file).
//
// x = hi + mid + lo in bfloat16, exactly: 24 bits are three times eight.  Of the nine products of the parts the three that lie
// 2^-27 and more below the result are left out, the other six go through the tensor core.  It truncates what it adds to the
// grid of the larger operand, so
//   - the products of 32 samples, the small ones first, are added in tensor memory, and every further addition is an fp32 one
//     in registers: an epilogue thread holds the sums of half a row of the tile, 128 of them;
//   - the sums of squares, whose terms all have one sign, are added by the converting warps with fp32 FMAs; truncation would
//     leave them half a unit in the last place too small (measured -5.8e-8 relative; other sums of both signs have no such drift).
// 2-norm of the error against 64 bits, of the result's, FMA kernels / here: N(0,1) [4096,256] 6.2e-8 / 4.8e-8, [65536,140]
// 5.4e-8 / 5.5e-8, [65536,512] 1.8e-7 / 5.5e-8, [1500,2048] 3.9e-7 / 8.3e-8.  Where all x are positive sums come out 5e-8 (long
// tails 7e-8) too small, which short chains of FMAs do not: uniform [4096,256] 5.3e-8 / 7.1e-8, [5000,520] 5.8e-8 / 6.9e-8,
// [262144,256] 9.2e-8 / 7.3e-8, [65536,512] 1.3e-7 / 7.7e-8, [1500,2048] 2.9e-7 / 7.9e-8.  With the small products in an accumulator
// of their own the first would be 5.9e-8, but lognormal 7.9e-8 where it is 8.1e-8, and the kernel takes 7 to 10 % longer.
// What bounds it: per 32 samples of a full tile 1536 cycles of MMA, 1660 of shared memory (copies 256, loads 256 and stores 384 of
// the converting warps, operands 768), and in the converting warps, which take the 2500 cycles that are measured, about 1400
// of the issue slots of a scheduler, whose loads wait behind the tensor core's; 12 bytes of their registers are spilled.  Calls in a
// row on one table, us: [65536,512] 371 with fp32 FMAs, here 121; [65536,256] 112 and 47; [4096,2048] 376 and 113.  Tried (the kernel
// alone, when it took 122): four converting warps (139 at [65536,512]), two groups of four on
// alternate stages (152), polls by one lane (148), the mixed-precision subtraction (134 instead of 131).
// Infinities, NaN and |x| > 2^127.99 have no parts and make a sum that is no number; of |x| < 2^-102 parts may be lost or subnormal.
// A cluster that meets either looks its samples through, and adds once more, with fp32 FMAs, the sums that are no number though
// neither of their columns has a NaN, and those of which tiny values may have lost more than 2^-25: lines (rows or columns of the
// tile) that hold such sums, or where there are many of them the whole tile.  [65536,512], us, 371 with FMA kernels whatever the
// values: 121 with ordinary ones, 230 with a |x| of 1e-38 or a NaN among them, 364 with infinities in one to four columns, 526 in
// sixteen, 935 where one value in a hundred is one (all samples to 256 threads with a row each: 3640 with any of these).
#pragma once
#include <atomic>
#include <type_traits>

namespace st {

namespace m2tc {
// Warps 0 .. EX_CONV_WARPS - 1 convert, then copies, MMA, two idle ones, eight of the epilogue.
constexpr int EX_CONV_WARPS = 8, EX_COPY_WARP = EX_CONV_WARPS, EX_MMA_WARP = EX_CONV_WARPS + 1, EX_EPI_WARP = EX_CONV_WARPS + 4;
constexpr int EX_EPI_THREADS = 256;
constexpr int EX_THREADS = 32 * EX_EPI_WARP + EX_EPI_THREADS;
// Registers of a thread at launch, and of the warpgroups afterwards: an epilogue thread needs 128 for its sums alone.
constexpr int EX_REGS = 65536 / EX_THREADS / 8 * 8, EX_REGS_MAIN = 32, EX_REGS_EPI = 168, EX_REGS_CONV = 56;
static_assert(EX_CONV_WARPS / 4 * EX_REGS_CONV + EX_REGS_MAIN + 2 * EX_REGS_EPI <= EX_THREADS / 128 * EX_REGS,
              "the warpgroups share what the block was launched with");
static_assert(EX_REGS_CONV <= EX_REGS && EX_REGS_MAIN <= EX_REGS && EX_REGS_EPI >= EX_REGS, "setmaxnreg.dec must not add, .inc not take");
// Stages of operands (3 boxes a unit) and of fp32 (2) in flight for tiles of 1 .. 4 boxes a part
constexpr int EX_MAX_STAGES = 8, EX_BOXES = 52;
__device__ constexpr int EX_STAGES[5] = {0, 8, 5, 3, 3}, EX_RAW_STAGES[5] = {0, 8, 5, 4, 2};
constexpr int EX_LEVEL = 256;                          // phases that are added before the sum goes to the partial tile
constexpr int EX_SQUARES = 2 * EX_CONV_WARPS;          // parts of a column's sum of squares
constexpr uint32_t EX_TINY = 2 * (25u << 23) - 1;      // 2 |x| - 1 of 2^-102, in bits; of zero it is the largest
constexpr float EX_LOST = 0x1p-125f;                   // most that the parts of a number below it can lack
constexpr int EX_LINES = 8, EX_MOST_LINES = 64;        // lines of a pass over the samples; from where the whole tile takes less
constexpr int EX_FEW = 32;                             // sums of half a row that are left to their columns, if no more than half of them
constexpr int EX_AGAIN = 64;                           // samples at a time of the whole tile, two of them in shared memory
constexpr int EX_AGAIN_FLOATS = EX_AGAIN * (HALF + BN);
constexpr size_t EX_SMEM = 1024 + (size_t)EX_BOXES * 4096 + 512 + (size_t)EX_SQUARES * HALF * sizeof(float);
static_assert((2 * (size_t)EX_AGAIN_FLOATS + 2 * (HALF + BN) + 12) * sizeof(float) <= (size_t)EX_BOXES * 4096, "the FMA path reuses the stages");
static_assert(EX_LINES * EX_EPI_THREADS * 4 <= 2 * EX_AGAIN_FLOATS, "the sums of a pass take the place of the samples");
}  // namespace m2tc

template <int REGS> __device__ __forceinline__ void regs_up() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS)); }
template <int REGS> __device__ __forceinline__ void regs_down() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS)); }

// x += y and x -= y for two fp32 numbers at a time (y: their bits).
__device__ __forceinline__ uint64_t ex_pack2(uint32_t lo, uint32_t hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ void ex_add2(float &x0, float &x1, uint32_t y0, uint32_t y1)
{
    uint64_t x = ex_pack2(__float_as_uint(x0), __float_as_uint(x1));
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(x) : "l"(ex_pack2(y0, y1)));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x0), "=f"(x1) : "l"(x));
}
__device__ __forceinline__ void ex_sub2(float &x0, float &x1, uint32_t y0, uint32_t y1)
{
    uint64_t x = ex_pack2(__float_as_uint(x0), __float_as_uint(x1));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(x) : "l"(ex_pack2(y0, y1)), "l"(0xBF800000BF800000ull));      // x + y (-1)
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x0), "=f"(x1) : "l"(x));
}

// Barrier of the epilogue warps of a block; true if any of them says so.
__device__ __forceinline__ bool ex_any(bool x)
{
    uint32_t r = x ? 1u : 0u;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %0, 0;\n\tbar.red.or.pred q, 1, %1, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "+r"(r) : "n"(m2tc::EX_EPI_THREADS) : "memory");
    return r != 0;
}

__global__ void __launch_bounds__(m2tc::EX_THREADS, 1)
moment2_exact_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ m2tc::Args a)
{
    using namespace m2tc;
    using namespace tc;
    using S = Shape<M2_EXACT>;
    constexpr int KROWS = S::KROWS, BOX_BYTES = S::BOX_BYTES;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = align_smem(smem_raw);
    uint64_t *bars = (uint64_t *)(smem + EX_BOXES * BOX_BYTES);
    uint64_t *full = bars, *empty = full + EX_MAX_STAGES, *raw_full = empty + EX_MAX_STAGES, *raw_empty = raw_full + EX_MAX_STAGES,
             *acc_full = raw_empty + EX_MAX_STAGES, *acc_empty = acc_full + 2;
    uint32_t *tmem_slot = (uint32_t *)(acc_empty + 2);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    unsigned *tiny_seen = (unsigned *)(tmem_slot + 2);
    float *squares = reinterpret_cast<float *>(smem + EX_BOXES * BOX_BYTES + 512);       // [EX_SQUARES][HALF]: of this block's rows

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();            // 0 = leader
    const int cluster = blockIdx.x >> 1;
    const int tile = m2tc_tile_of(a.tab, cluster), split = cluster - a.tab.first[tile];
    const int nsplit = a.tab.first[tile + 1] - a.tab.first[tile];
    const int row = 8 * a.tab.row[tile], rows = a.tab.rows[tile], col = 8 * a.tab.col[tile], width = 32 * a.tab.width[tile];
    const bool diag = a.tab.diag[tile] != 0;
    const bool alias = diag && width == BN;             // A columns == B columns in both blocks: one copy serves both
    const bool lead = diag && rows <= HALF;             // all rows in the first block, whose A holds its half of B as well
    // A stage of operands: all hi boxes (64 columns x 32 samples), all mid boxes, all lo boxes; a stage as it was copied: boxes of
    // 32 columns x 32 samples of fp32, two for each of those.  Boxes of B and of A, the most that either block has:
    const int tb = ((lead && rows > width / 2 ? rows : width / 2) + 63) / 64, ta = alias || lead ? 0 : rows >= HALF ? 2 : (rows + 63) / 64;
    const uint32_t part_bytes = (uint32_t)((tb + ta) * BOX_BYTES), stage_bytes = 3 * part_bytes, raw_bytes = 2 * part_bytes;
    const int stages = EX_STAGES[tb + ta], raw_stages = EX_RAW_STAGES[tb + ta];
    // an MMA reads 128 columns of A per block, of which fewer may have been written: behind the operands it meets the fp32 boxes
    unsigned char *raw0 = smem + (size_t)stages * stage_bytes;
    const int chunks_per_split = (a.chunks_total + nsplit - 1) / nsplit;
    const int c_begin = split * chunks_per_split;
    int c_end = c_begin + chunks_per_split;
    if (c_end > a.chunks_total) c_end = a.chunks_total;
    const int nchunks = c_end > c_begin ? c_end - c_begin : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full[s], 2 * EX_CONV_WARPS);     // the converting warps of both blocks (leader's copy is used)
            mbar_init(&empty[s], 1);                    // one commit per use, delivered to both blocks
        }
        for (int s = 0; s < raw_stages; ++s) {
            mbar_init(&raw_full[s], 1);
            mbar_init(&raw_empty[s], EX_CONV_WARPS);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 16);               // eight epilogue warps in each of the two blocks (leader's copy is used)
        }
        *abort_flag = 0;
        *tiny_seen = 0;
        fence_barrier_init();
    }
    if (warp == EX_MMA_WARP) {
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
        a.status[kWsStatusWord] = 0;
        a.status[kWsDetailWord] = 0;
    }

    // boxes of 32 columns that block r copies: of B, and of A the ones that hold rows of the result
    auto boxes_b = [&](int r) {
        int n = lead && r == 0 && rows > width / 2 ? rows : width / 2;
        if (n > a.d - col - r * (width / 2)) n = a.d - col - r * (width / 2);
        return n <= 0 ? 0 : (n + 31) / 32;
    };
    auto boxes_a = [&](int r) {
        const int n = rows - r * HALF;
        return alias || lead || n <= 0 ? 0 : n >= HALF ? HALF / 32 : (n + 31) / 32;
    };
    const int col_a = row + (int)rank * HALF, col_b = col + (int)rank * (width / 2);
    const int nb = boxes_b((int)rank), na = boxes_a((int)rank);

    if (warp < EX_CONV_WARPS) {
        // ---------------- converting warps (both blocks): the parts of x, each in the form that a copy of boxes of 64 columns x 32
        // rows with the 128-byte swizzle leaves.  A warp takes RPW rows of all boxes of a stage.
        regs_down<EX_REGS_CONV>();
        constexpr int RPW = KROWS / EX_CONV_WARPS, H = RPW / 2;
        const int c4 = (lane & 15) * 4, r0 = ((warp * RPW) & 7) + (lane >> 4);    // columns c4 .. c4+3 of 64, rows r0 + 2h of eight
        const uint32_t bar0 = map_to_cta(smem_u32(full), 0);
        // of row r0; row r0 + 2h: 256 h further, and bits 5 and 6, where the swizzle puts bits 1 and 2 of the row, exclusive-or h
        const uint32_t from0 = (uint32_t)(warp * RPW / 8 * 1024 + (c4 >> 5) * BOX_BYTES + r0 * 128 + ((((c4 >> 2) & 7) ^ r0) << 4));
        const uint32_t to0 = (uint32_t)(warp * RPW / 8 * 1024 + r0 * 128 + (((c4 >> 3) ^ r0) << 4) + (c4 & 4) * 2);
        uint32_t least[2] = {~0u, ~0u};                                     // smallest 2 |x| - 1, as bits: zeros come out as the largest
        auto convert = [&](auto diag_tag) {
            constexpr bool DIAG = decltype(diag_tag)::value;
            float square[8] = {};
            // Items of a stage: 64 columns of B, the other 64 of B, of A, of A, whichever this block has.  The loads of an item are
            // issued before the one ahead of it is converted.
            const int qb = (nb + 1) / 2, items = qb + (na + 1) / 2 > 0 ? qb + (na + 1) / 2 : 1;
            int s = 0, rs = 0;
            uint32_t parity = 1, rparity = 0;
            float rest[H][4], next[H][4];
            auto there = [&](int item) { return 2 * (item < qb ? item : item - qb) + (c4 >> 5) < (item < qb ? nb : na); };
            auto load = [&](int item) {
                const unsigned char *p = raw0 + rs * raw_bytes + 2 * (item < qb ? item : tb + item - qb) * BOX_BYTES;
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    const float4 v = there(item) ? *reinterpret_cast<const float4 *>(p + (from0 ^ (h << 5)) + 256 * h) : make_float4(0.f, 0.f, 0.f, 0.f);
                    next[h][0] = v.x; next[h][1] = v.y; next[h][2] = v.z; next[h][3] = v.w;
                }
            };
            bool ok = nchunks > 0 && mbar_wait(&raw_full[0], 0, abort_flag, a.status, 5);
            if (ok) load(0);
            for (int c = 0; c < nchunks && ok; ++c) {
                if (c >= stages && !mbar_wait(&empty[s], parity, abort_flag, a.status, 6)) break;
                bool loaded = false;
                for (int item = 0; item < items; ++item) {
#pragma unroll
                    for (int h = 0; h < H; ++h)
#pragma unroll
                        for (int e = 0; e < 4; ++e) rest[h][e] = next[h][e];
                    if (item + 1 < items) {
                        load(item + 1);
                    } else {
                        __syncwarp();                             // all lanes have the last values of the stage
                        if (lane == 0) mbar_arrive(&raw_empty[rs]);
                        if (++rs == raw_stages) { rs = 0; rparity ^= 1u; }
                        if (c + 1 < nchunks && __all_sync(0xFFFFFFFFu, mbar_try_wait(&raw_full[rs], rparity))) {
                            load(0);
                            loaded = true;
                        }
                    }
                    const bool store = there(item);
                    unsigned char *w = smem + s * stage_bytes + (item < qb ? item : tb + item - qb) * BOX_BYTES;
                    if (DIAG && item < qb) {                          // B holds the columns of a diagonal block's rows
                        const bool upper = item != 0;
#pragma unroll
                        for (int h = 0; h < H; ++h)
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                if (upper) square[4 + e] = fmaf(rest[h][e], rest[h][e], square[4 + e]);
                                else square[e] = fmaf(rest[h][e], rest[h][e], square[e]);
                            }
                    }
                    // all values of the item step by step: one after the other they would be a chain of seven results each
#pragma unroll
                    for (int part = 0; part < 3; ++part) {
                        uint32_t b[H][2];
#pragma unroll
                        for (int h = 0; h < H; ++h)
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const __nv_bfloat162 r = __floats2bfloat162_rn(rest[h][2 * e], rest[h][2 * e + 1]);
                                b[h][e] = *reinterpret_cast<const uint32_t *>(&r);
                            }
                        if (part == 0) {
#pragma unroll
                            for (int h = 0; h < H; ++h)
#pragma unroll
                                for (int e = 0; e < 2; ++e)
                                    least[e] = __vimin3_u32(least[e], 2 * __float_as_uint(rest[h][2 * e]) - 1, 2 * __float_as_uint(rest[h][2 * e + 1]) - 1);
                        }
                        if (store) {
#pragma unroll
                            for (int h = 0; h < H; ++h)
                                *reinterpret_cast<uint2 *>(w + part * part_bytes + (to0 ^ (h << 5)) + 256 * h) = make_uint2(b[h][0], b[h][1]);
                        }
                        if (part < 2) {
#pragma unroll
                            for (int h = 0; h < H; ++h)
#pragma unroll
                                for (int e = 0; e < 2; ++e) {
                                    ex_sub2(rest[h][2 * e], rest[h][2 * e + 1], b[h][e] << 16, b[h][e] & 0xFFFF0000u);
                                }
                        }
                    }
                }
                fence_proxy_async();          // generic writes, read by the tensor core
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster_smem(bar0 + (uint32_t)(s * sizeof(uint64_t)));
                if (++s == stages) { s = 0; parity ^= 1u; }
                if (c + 1 < nchunks && !loaded) {
                    ok = mbar_wait(&raw_full[rs], rparity, abort_flag, a.status, 5);
                    if (ok) load(0);
                }
            }
            if (DIAG) {
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int e = 0; e < 4; ++e) squares[(warp * 2 + (lane >> 4)) * HALF + q * 64 + c4 + e] = square[4 * q + e];
            }
        };
        if (diag) convert(std::integral_constant<bool, true>{});
        else convert(std::integral_constant<bool, false>{});
        if (min(least[0], least[1]) < EX_TINY) atomicOr(tiny_seen, 1u);
    } else if (warp < EX_EPI_WARP) {
        regs_down<EX_REGS_MAIN>();
        if (warp == EX_COPY_WARP && elect_one()) {
            // ---------------- copies (both blocks): own boxes, fp32
            prefetch_tmap(&tmap);
            int s = 0;
            uint32_t parity = 1;
            for (int c = 0; c < nchunks; ++c) {
                if (c >= raw_stages && !mbar_wait(&raw_empty[s], parity, abort_flag, a.status, 1)) break;
                mbar_expect_tx(&raw_full[s], (uint32_t)((nb + na) * BOX_BYTES));
                unsigned char *base = raw0 + s * raw_bytes;
                const int y = (c_begin + c) * KROWS;
                for (int b = 0; b < nb; ++b) tma_load_2d(base + b * BOX_BYTES, &tmap, &raw_full[s], col_b + b * 32, y);
                for (int b = 0; b < na; ++b) tma_load_2d(base + (2 * tb + b) * BOX_BYTES, &tmap, &raw_full[s], col_a + b * 32, y);
                if (++s == raw_stages) { s = 0; parity ^= 1u; }
            }
        } else if (warp == EX_MMA_WARP && rank == 0 && elect_one()) {
            // ---------------- MMA issuer (leader only).  The small products first: only what follows the first hi^T hi is cut at the
            // grid of the result.
            const uint32_t idesc = make_idesc(1, 1, 1, BM, (uint32_t)width);
            const uint32_t a_off = alias || lead ? 0u : (uint32_t)(tb * BOX_BYTES);
            const uint32_t sb0 = smem_u32(smem);
            const uint64_t adesc_base = make_smem_desc(sb0 + a_off, BOX_BYTES, 1024), bdesc_base = make_smem_desc(sb0, BOX_BYTES, 1024);
            const uint64_t part = (uint64_t)(part_bytes >> 4);
            int s = 0;
            uint32_t parity = 0;
            for (int c = 0; c < nchunks; ++c) {
                const int buf = c & 1;
                if (!mbar_wait<true>(&full[s], parity, abort_flag, a.status, 2)) break;
                if (c >= 2 && !mbar_wait(&acc_empty[buf], (uint32_t)(((c >> 1) - 1) & 1), abort_flag, a.status, 4)) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * BN);
                const uint64_t ad = adesc_base + (uint64_t)((uint32_t)s * (stage_bytes >> 4));
                const uint64_t bd = bdesc_base + (uint64_t)((uint32_t)s * (stage_bytes >> 4));
                constexpr int PA[6] = {0, 2, 1, 0, 1, 0}, PB[6] = {2, 0, 1, 1, 0, 0};
#pragma unroll
                for (int p = 0; p < 6; ++p)
#pragma unroll
                    for (int k = 0; k < KROWS / S::KMMA; ++k) {
                        constexpr int STEP = S::KMMA * 128 / 16;
                        mma_bf16_pair(d_tmem, ad + PA[p] * part + (uint64_t)(k * STEP), bd + PB[p] * part + (uint64_t)(k * STEP), idesc,
                                      p > 0 || k > 0 ? 1u : 0u);
                    }
                tc_commit_pair(&empty[s]);
                tc_commit_pair(&acc_full[buf]);
                if (++s == stages) { s = 0; parity ^= 1u; }
            }
        }
        __syncwarp();
    }
    if (warp >= EX_EPI_WARP) {
        // ---------------- epilogue (both blocks): a thread owns row row0 + lane of the tile and half of its columns, c_half ..
        regs_up<EX_REGS_EPI>();
        const int row0 = (int)rank * HALF + (warp & 3) * 32, half = width / 2, c_half = warp >= EX_EPI_WARP + 4 ? half : 0;
        float *dst = a.partials + (size_t)blockIdx.x * HALF * BN + ((warp & 3) * 32 + lane) * 4;      // columns c .. c+3: + c HALF
        // sixteen columns of the half: in the tile, and not wholly below the diagonal?
        auto wanted = [&](int t) { return row0 < rows && 16 * t < half && !(diag && c_half + 16 * t + 15 < row0); };
        float sum[128];
#pragma unroll
        for (int e = 0; e < 128; ++e) sum[e] = 0.f;
        const uint32_t leader_acc_empty0 = map_to_cta(smem_u32(&acc_empty[0]), 0);
        const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c_half;
        auto store = [&](bool add) {
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if (wanted(t)) {
#pragma unroll
                    for (int e = 16 * t; e < 16 * t + 16; e += 4) {
                        float4 v = make_float4(sum[e], sum[e + 1], sum[e + 2], sum[e + 3]);
                        float4 *p = reinterpret_cast<float4 *>(dst + (c_half + e) * HALF);
                        if (add) {
                            const float4 o = *p;
                            v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
                        }
                        *p = v;
                    }
                }
        };
        // infinities, NaN and what rounds to infinity in bfloat16 show in the sums, 0 times a number that is none; looked at
        // whenever the sums leave the registers (columns from d on are zeros there)
        float zero = 0.f;
        auto look = [&]() {
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if (wanted(t) && col + c_half + 16 * t < a.d) {
#pragma unroll
                    for (int e = 16 * t; e < 16 * t + 16; ++e) zero = fmaf(sum[e], 0.f, zero);
                }
        };
        int held = 0;
        bool stored = false;
        for (int c = 0; c < nchunks; ++c) {
            const int buf = c & 1;
            if (!mbar_wait(&acc_full[buf], (uint32_t)((c >> 1) & 1), abort_flag, a.status, 3)) break;
            tc_fence_after();
#pragma unroll
            for (int t = 0; t < 8; t += 2)
                if (wanted(t) || wanted(t + 1)) {
                    uint32_t r[32];
                    tmem_ld_32x32(taddr + (uint32_t)(buf * BN + 16 * t), r);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; e += 2) ex_add2(sum[16 * t + e], sum[16 * t + e + 1], r[e], r[e + 1]);
                }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster_smem(leader_acc_empty0 + (uint32_t)(buf * sizeof(uint64_t)));
            if (++held == EX_LEVEL) {
                look();
                store(stored);
                stored = true;
                held = 0;
#pragma unroll
                for (int e = 0; e < 128; ++e) sum[e] = 0.f;
            }
        }
        look();
        store(stored);
        // every value of the pair's samples has been looked at when the converting warps have arrived here
        __syncthreads();
        cluster_sync_all();
        uint32_t tiny[2];
#pragma unroll
        for (int r = 0; r < 2; ++r)
            asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(tiny[r]) : "r"(map_to_cta(smem_u32(tiny_seen), (uint32_t)r)));
        const int i = row + row0 + lane, t = (int)threadIdx.x - 32 * EX_EPI_WARP;
        const int64_t n0 = (int64_t)c_begin * KROWS, n1 = (int64_t)c_end * KROWS < a.N ? (int64_t)c_end * KROWS : a.N;
        if ((tiny[0] | tiny[1]) != 0 || ex_any(zero != 0.f && row0 < rows && i < a.d)) {
            // two buffers of samples (64 x 128 values of the rows' columns, 64 x 256 of the tile's); of the rows' columns and the
            // tile's the largest |x| and the smallest 2 |x| - 1, as bits; lines
            float *panels = reinterpret_cast<float *>(smem), *block = a.partials + (size_t)blockIdx.x * HALF * BN;
            uint32_t *most = reinterpret_cast<uint32_t *>(panels + 2 * EX_AGAIN_FLOATS), *least = most + HALF + BN, *lines = least + HALF + BN;
            for (int k = t; k < HALF + BN; k += EX_EPI_THREADS) {
                most[k] = 0;
                least[k] = ~0u;
            }
            if (t < 12) lines[t] = 0;
            ex_any(false);
            // Columns of a side (of the tile: 0, of the block's rows: 1, unless the tile's hold them), four to a thread; all samples,
            // `step` at a time.
            auto side_first = [&](int side) { return side ? col_a : col; };
            auto side_quads = [&](int side) {
                const int n = side ? min(HALF, rows - (int)rank * HALF) : width;
                return (min(n, a.d - side_first(side)) + 3) / 4;
            };
            for (int side = 0; side < (diag ? 1 : 2); ++side) {
                const int quads = side_quads(side);
                if (quads <= 0) continue;
                const int step = EX_EPI_THREADS / quads, r = t / quads, q = t % quads;
                uint32_t m[4] = {0, 0, 0, 0}, l[4] = {~0u, ~0u, ~0u, ~0u};
                constexpr int U = 16;
                for (int64_t n = n0 + r; r < step && n < n1; n += U * step) {
                    uint4 v[U];
#pragma unroll
                    for (int k = 0; k < U; ++k)
                        v[k] = n + k * step < n1 ? *reinterpret_cast<const uint4 *>(a.X + (n + k * step) * a.ldx + side_first(side) + 4 * q) : make_uint4(0, 0, 0, 0);
#pragma unroll
                    for (int k = 0; k < U; ++k) {
                        const uint32_t w[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            m[e] = max(m[e], w[e] & 0x7FFFFFFFu);
                            l[e] = min(l[e], 2 * w[e] - 1);
                        }
                    }
                }
                const int at = (side ? 0 : HALF) + 4 * q;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    atomicMax(most + at + e, m[e]);
                    atomicMin(least + at + e, l[e]);
                }
            }
            ex_any(false);
            // Which sums: no number, though neither column has a NaN; or what the parts of a column lack, times the largest value of
            // the other in every sample, is more than 2^-25 of the sum.
            const float lost = (float)(n1 - n0) * (EX_LOST * 0x1p25f);
            const int own = (diag ? HALF + (int)rank * HALF : 0) + (warp & 3) * 32 + lane;
            const uint32_t most_row = most[own];
            const bool tiny_row = least[own] < EX_TINY, nan_row = most_row > 0x7F800000u;
            uint32_t which[4] = {0, 0, 0, 0};
            int count = 0, all = 0;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                float4 v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    v[q] = wanted(2 * w + q / 4) ? *reinterpret_cast<const float4 *>(dst + (c_half + 32 * w + 4 * q) * HALF) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    const int c = 32 * w + e;
                    if (!wanted(c >> 4) || i >= a.d || col + c_half + c >= a.d || i == col + c_half + c) continue;    // squares: below
                    ++all;
                    const float4 f = v[e / 4];
                    const float s = fabsf(e % 4 == 0 ? f.x : e % 4 == 1 ? f.y : e % 4 == 2 ? f.z : f.w);
                    const uint32_t most_col = most[HALF + c_half + c];
                    const bool tiny_col = least[HALF + c_half + c] < EX_TINY;
                    const float may_lack = (tiny_row ? lost : 0.f) * __uint_as_float(most_col) + (tiny_col ? lost : 0.f) * __uint_as_float(most_row);
                    const bool poor = (tiny_row || tiny_col) && !(s >= may_lack);
                    if (!nan_row && most_col <= 0x7F800000u && (poor || !(s <= 0x1.fffffep127f))) {
                        which[w] |= 1u << e;
                        ++count;
                    }
                }
            }
            // Their lines: rows of the block (four words; on the diagonal the columns that they are too), columns of the tile (eight)
            if (count > EX_FEW || 2 * count > all) {
                atomicOr(lines + (diag ? 4 + 4 * (int)rank : 0) + (warp & 3), 1u << lane);
            } else if (count > 0) {
#pragma unroll
                for (int w = 0; w < 4; ++w)
                    if (which[w] != 0) {
                        // columns c_half + 32 w ..: they straddle two words where a half is no multiple of 32
                        const int c = c_half + 32 * w;
                        atomicOr(lines + 4 + c / 32, which[w] << (c & 31));
                        if ((c & 31) != 0) atomicOr(lines + 4 + c / 32 + 1, which[w] >> (32 - (c & 31)));
                    }
            }
            ex_any(false);
            int line_rows = 0, line_cols = 0;
#pragma unroll
            for (int w = 0; w < 12; ++w) (w < 4 ? line_rows : line_cols) += __popc(lines[w]);
            if (line_rows + line_cols <= EX_MOST_LINES) {
                // x of EX_LINES lines times x of the columns across them; on the diagonal across all of the tile's
                for (int side = 0; side < 2; ++side) {
                    const int total = side ? line_cols : line_rows, words = side ? 8 : 4, across = diag ? 0 : side, quads = side_quads(across);
                    if (total == 0 || quads <= 0) continue;
                    const uint32_t *set = side ? lines + 4 : lines;
                    auto line = [&](int k) {                      // the k-th one
                        int w = 0, n = __popc(set[0]);
                        while (k >= n && w + 1 < words) { k -= n; n = __popc(set[++w]); }
                        return k < n ? 32 * w + (int)__fns(set[w], 0, k + 1) : 0;
                    };
                    const int step = EX_EPI_THREADS / quads, r = t / quads, q = t % quads;
                    for (int first = 0; first < total; first += EX_LINES) {
                        int from[EX_LINES];                       // column of a line less the ones across it
                        float acc[EX_LINES][4] = {};
#pragma unroll
                        for (int l = 0; l < EX_LINES; ++l)
                            from[l] = side_first(1 - side) + line(first + l < total ? first + l : first) - side_first(across) - 4 * q;
                        if (r < step) {
                            const float *x = a.X + (n0 + r) * a.ldx + side_first(across) + 4 * q;
#pragma unroll 4
                            for (int64_t n = n0 + r; n < n1; n += step, x += step * a.ldx) {
                                const float4 v = *reinterpret_cast<const float4 *>(x);
#pragma unroll
                                for (int l = 0; l < EX_LINES; ++l) {
                                    const float y = x[from[l]];
                                    acc[l][0] = fmaf(y, v.x, acc[l][0]);
                                    acc[l][1] = fmaf(y, v.y, acc[l][1]);
                                    acc[l][2] = fmaf(y, v.z, acc[l][2]);
                                    acc[l][3] = fmaf(y, v.w, acc[l][3]);
                                }
                            }
#pragma unroll
                            for (int l = 0; l < EX_LINES; ++l)
                                *reinterpret_cast<float4 *>(panels + ((l * step + r) * quads + q) * 4) = make_float4(acc[l][0], acc[l][1], acc[l][2], acc[l][3]);
                        }
                        ex_any(false);
                        for (int k = t; k < EX_LINES * 4 * quads; k += EX_EPI_THREADS) {
                            const int l = k / (4 * quads), o = k % (4 * quads);
                            if (first + l >= total) break;
                            float total_sum = 0.f;
                            for (int p = 0; p < step; ++p) total_sum += panels[(l * step + p) * quads * 4 + o];
                            const int at = line(first + l);
                            auto put = [&](int r, int c) {
                                if (r >= 0 && r < HALF) block[(c & ~3) * HALF + r * 4 + (c & 3)] = total_sum;
                            };
                            if (!diag) {
                                put(side ? o : at, side ? at : o);
                            } else {
                                put(o - (int)rank * HALF, at);
                                put(at - (int)rank * HALF, o);
                            }
                        }
                        ex_any(false);
                    }
                }
            } else {
                // the whole tile: a thread has eight rows and, of each 32 columns of its half of 128, four
                // EX_AGAIN samples at a time (zeros past the end): body(rows' columns, tile's columns)
                auto samples = [&](auto body) {
                    auto fetch = [&](int64_t n, int buf) {
                        const uint32_t xa = smem_u32(panels + buf * EX_AGAIN_FLOATS), xb = xa + EX_AGAIN * HALF * 4;
                        for (int k = t; k < EX_AGAIN * (HALF + BN) / 4; k += EX_EPI_THREADS) {
                            const bool is_a = k < EX_AGAIN * HALF / 4;
                            const int u = is_a ? k : k - EX_AGAIN * HALF / 4, r = is_a ? u / (HALF / 4) : u / (BN / 4), c = 4 * (is_a ? u % (HALF / 4) : u % (BN / 4));
                            const int gc = (is_a ? col_a : col) + c;
                            const bool in = n + r < n1 && gc < a.d && (is_a || c < width);
                            const float *src = in ? a.X + (n + r) * a.ldx + gc : a.X;
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((is_a ? xa : xb) + 16u * (uint32_t)u), "l"(src), "r"(in ? 16 : 0) : "memory");
                        }
                        asm volatile("cp.async.commit_group;" ::: "memory");
                    };
                    int buf = 0;
                    fetch(n0, 0);
                    for (int64_t n = n0; n < n1; n += EX_AGAIN, buf ^= 1) {
                        fetch(n + EX_AGAIN, buf ^ 1);
                        asm volatile("cp.async.wait_group 1;" ::: "memory");
                        ex_any(false);
                        body(panels + buf * EX_AGAIN_FLOATS, panels + buf * EX_AGAIN_FLOATS + EX_AGAIN * HALF);
                        ex_any(false);
                    }
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                };
                const int ra = (warp & 3) * 32 + (lane >> 3) * 8, cb = (warp >= EX_EPI_WARP + 4 ? HALF : 0) + (lane & 7) * 4;
                uint64_t acc[8][8] = {};
                samples([&](const float *xa, const float *xb) {
#pragma unroll 1
                    for (int k = 0; k < EX_AGAIN; ++k) {
                        const float4 a0 = *reinterpret_cast<const float4 *>(xa + k * HALF + ra), a1 = *reinterpret_cast<const float4 *>(xa + k * HALF + ra + 4);
                        const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                        ulonglong2 b[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) b[q] = *reinterpret_cast<const ulonglong2 *>(xb + k * BN + cb + 32 * q);
#pragma unroll
                        for (int r = 0; r < 8; ++r) {
                            const uint64_t aa = ex_pack2(__float_as_uint(av[r]), __float_as_uint(av[r]));
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[r][2 * q]) : "l"(aa), "l"(b[q].x));
                                asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[r][2 * q + 1]) : "l"(aa), "l"(b[q].y));
                            }
                        }
                    }
                });
#pragma unroll
                for (int r = 0; r < 8; ++r)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        *reinterpret_cast<ulonglong2 *>(block + (cb + 32 * q) * HALF + (ra + r) * 4) = make_ulonglong2(acc[r][2 * q], acc[r][2 * q + 1]);
                ex_any(false);
            }
        }
        // the sums of squares take their places on the diagonal
        const int o = i - row;
        if (diag && row0 < rows && i < a.d && o >= c_half && o < c_half + half) {
            float total = 0.f;
#pragma unroll
            for (int p = 0; p < EX_SQUARES; ++p) total += squares[p * HALF + (warp & 3) * 32 + lane];
            dst[(o & ~3) * HALF + (o & 3)] = total;
        }
    } else {
        __syncwarp();
        __syncthreads();
        cluster_sync_all();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                      // no block leaves while its peer may still read its flag
    if (warp == EX_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, TMEM_COLS);
    }
}

// The warpgroups of moment2_exact_kernel pass registers among them: what they end with is what the block must start with, or
// one of them would wait for good.  A kernel that was built with fewer is not launched.
inline bool m2tc_exact_fits()
{
    static std::atomic<int> known{0};
    int regs = known.load(std::memory_order_relaxed);
    if (regs == 0) {
        cudaFuncAttributes f;
        if (cudaFuncGetAttributes(&f, moment2_exact_kernel) != cudaSuccess) {
            (void)cudaGetLastError();
            return false;
        }
        known.store(regs = f.numRegs, std::memory_order_relaxed);
    }
    return (regs + 7) / 8 * 8 >= m2tc::EX_REGS;
}

}  // namespace st
