// st_sym_moment3, tensor-core path (ST_FLAG_TC_TF32 / ST_FLAG_TC_BF16):
//     out[q(i,j,k)] = sum_n X[n,i] X[n,j] X[n,k]   for 0 <= i <= j <= k < d
// (Section 3, M2 = f (x) vec(f (x) f) summed over samples; unique elements i<=j<=k, Section 2
// "Tensor Structures").  With the pair product hoisted out of the k loop (loop-invariant code
// motion, Section 5.5) the sum is a contraction over the samples,
//     out[(i,j), k] = sum_n P[n,(i,j)] X[n,k],      P[n,(i,j)] = X[n,i] X[n,j]   (i <= j),
// that is a GEMM [pairs x samples] x [samples x d] whose left operand exists nowhere in memory.
// This kernel makes P on the fly.  Loader warps fetch slices of 32 (TF32) or 64 (bf16) samples and write X^T,
// rounded, into shared memory in the K-major 128-byte-swizzled form the tensor core reads (lane =
// sample).  Producer warps read their lane's x_i and x_j back from that slice, multiply the
// pairs of one tile (8 values of i x 16 values of j) and store the products, rounded to TF32, in
// the same form as the left operand of the tile's MMA.  A tile with j >= 16*JB needs the
// columns k >= 16*JB only: its MMA has N = d - 16*JB, so the part k < j of the iteration space
// is (up to that granularity) never issued, and tiles with i > j everywhere do not exist.
// Accumulators of all tiles of a block stay in tensor memory for the block's whole sample
// range; two to eight blocks ("groups") share one sample range and its tiles, for fewer partial sums.
//
// What bounds it: shared memory.  A stage takes 465 cycles at [40009,50] in bf16; per tile and slice the producers store 16 KB of
// products (128 cycles) and the tensor core reads them back with the columns of X^T (128 and 33 to 64; an MMA of M = 128, N <= 64 takes
// 39 to 48 cycles), the producers' own operands take 80.  Products straight into tensor memory, a row to a thread, load an x_i
// for each of them: 51 us where this takes 33.
// A warp took 2700 cycles for a whole stage, 1300 of them for 128 products a lane, and eight warps made
// one every 340; sixteen, two to a stage, and copies without a selected address for whole slices: [40009,50] bf16 36.0 us,
// now 35.2, [200000,50] 140 (before generic loads went) and 117, TF32 246 and 183.  Two issuer warps take alternate stages: polls and commits
// between the MMAs cost one alone about 100 cycles per stage.  bf16 halves the number of stages (64 samples per slice
// instead of 32).  Products and x_k rounded to TF32 / bf16, fp32 accumulation: 5e-3 tolerance (bf16: for N >= 1000).
#include "tc_common.cuh"
#include "st_index.cuh"
#include <type_traits>

namespace st {

namespace m3tc {
constexpr int DP = 64;                       // largest d
constexpr int TI = 8, TJ = 16;               // a tile holds the pairs (8 IB + a, 16 JB + b)
constexpr int BM = TI * TJ;                  // 128 pairs = rows of the MMA
constexpr int ROW_BYTES = 128;               // one swizzled row: 32 TF32 or 64 bf16 samples
constexpr int A_STAGE_BYTES = BM * ROW_BYTES; // 16 KiB
constexpr int NA_MAX = 10;                   // A stages in flight (TF32: 10, bf16: 8; even: see the issuers)
constexpr int NB_MAX = 16;                   // slices in flight: as many as fit beside the A stages (4 at d = 64), see ring()
constexpr int PRODUCERS = 16;                // producer warps (also the epilogue warps): two to a stage, half of its rows each
constexpr int MMA_WARPS = 2;                 // issuer w takes the stages q = w (mod 2): while one polls, the other's MMAs run
constexpr int MMA_WARP = PRODUCERS, LOAD_WARP = PRODUCERS + MMA_WARPS;
constexpr int LOAD_WARPS = 4;                // fetch slices of X and turn them into the right operand
constexpr int THREADS = 32 * (PRODUCERS + MMA_WARPS + LOAD_WARPS);
constexpr uint32_t TMEM_COLS = 512;
constexpr int MAX_GROUP_TILES = 12, MAX_TILES = 20, MAX_GROUPS = 8;
// A slice in flight: dcols rows of X^T as the right operand, and the samples as they are in memory, rows of dcols + 1
// floats (an odd pitch: lanes that read one column of consecutive samples touch every bank once).
constexpr size_t FIXED_SMEM = 1024 + 1024;    // alignment of the first stage; barriers
constexpr size_t b_stage_bytes(int dcols) { return (size_t)dcols * ROW_BYTES; }
constexpr size_t x_stage_bytes(int dcols, bool bf16) { return (size_t)(bf16 ? 64 : 32) * (dcols + 1) * 4; }
constexpr size_t a_ring_bytes(bool bf16) { return (size_t)(bf16 ? 8 : 10) * A_STAGE_BYTES; }
constexpr int ring(int dcols, bool bf16)
{
    const size_t n = (227 * 1024 - FIXED_SMEM - a_ring_bytes(bf16)) / (b_stage_bytes(dcols) + x_stage_bytes(dcols, bf16));
    return n > NB_MAX ? NB_MAX : (int)n;
}
static_assert(ring(DP, true) >= 4 && ring(DP, false) >= 4, "four slices in flight at least");
constexpr size_t smem_bytes(int dcols, bool bf16)
{
    return FIXED_SMEM + a_ring_bytes(bf16) + ring(dcols, bf16) * (b_stage_bytes(dcols) + x_stage_bytes(dcols, bf16));
}
// slices whose copies are under way while one is turned into the right operand
__host__ __device__ constexpr int fetch_ahead(int nb) { return nb >= 12 ? 8 : nb >= 8 ? 5 : 2; }

struct Tile {
    unsigned char ib, jb;
    unsigned short col;                      // first tensor-memory column of the tile's accumulator
    int part;                                // first of its partial sums in a slice
};

struct Args {
    const float *X;
    float *partials;
    unsigned *status;
    int64_t N, ldx, rows_per_slice;
    int nb;                                  // slices in flight
    int d, dcols, part_elems;                // part_elems: partial sums per slice; dcols = d rounded up to a multiple of 16
    int first[MAX_GROUPS + 1];               // tiles of group g: first[g] ..
    Tile tiles[MAX_TILES];
};

// byte offset of the 4-byte word `lane` (one TF32 sample, or two bf16 samples) inside a 128-byte row whose
// index has (row & 7) == m
__device__ __forceinline__ uint32_t swz(int lane, int m) { return (uint32_t)((((lane >> 2) ^ m) << 4) + ((lane & 3) << 2)); }

__device__ __forceinline__ uint64_t m3tc_pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

template <bool BF16>
__global__ void __launch_bounds__(THREADS, 1)
moment3_tc_kernel(const __grid_constant__ Args a)
{
    using namespace tc;
    constexpr int KS = BF16 ? 64 : 32;           // samples per slice
    constexpr int NA = BF16 ? 8 : 10;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = align_smem(smem_raw);
    unsigned char *a_stage0 = smem;
    const int NB = a.nb, x_pitch = a.dcols + 1;
    const uint32_t B_STAGE_BYTES = (uint32_t)a.dcols * ROW_BYTES, X_STAGE_FLOATS = (uint32_t)(KS * x_pitch);
    unsigned char *b_stage0 = smem + (size_t)NA * A_STAGE_BYTES;
    uint64_t *bars = (uint64_t *)(b_stage0 + (size_t)NB * (B_STAGE_BYTES + 4 * X_STAGE_FLOATS));
    float *x_stage0 = (float *)(b_stage0 + (size_t)NB * B_STAGE_BYTES);   // slices of X as they are in memory
    uint64_t *a_full = bars, *a_empty = bars + NA_MAX, *b_full = bars + 2 * NA_MAX, *b_empty = bars + 2 * NA_MAX + NB_MAX,
             *acc_full = bars + 2 * NA_MAX + 2 * NB_MAX;
    uint64_t *iss_sync = acc_full + 1;
    uint32_t *tmem_slot = (uint32_t *)(acc_full + 2);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int group = blockIdx.x;
    const int tg = a.first[group + 1] - a.first[group];      // tiles of this block
    const Tile *tiles = a.tiles + a.first[group];

    if (threadIdx.x == 0) {
        for (int s = 0; s < NA; ++s) {
            mbar_init(&a_full[s], 2);
            mbar_init(&a_empty[s], 1);
        }
        for (int s = 0; s < NB; ++s) {
            mbar_init(&b_full[s], LOAD_WARPS);
            mbar_init(&b_empty[s], MMA_WARPS);
        }
        mbar_init(acc_full, MMA_WARPS);
        mbar_init(iss_sync, MMA_WARPS);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == MMA_WARP) {
        tmem_alloc(tmem_slot, TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        a.status[kWsStatusWord] = 0;
        a.status[kWsDetailWord] = 0;
    }

    const int64_t n_begin = (int64_t)blockIdx.y * a.rows_per_slice;
    int64_t n_end = n_begin + a.rows_per_slice;
    if (n_end > a.N) n_end = a.N;
    const int nslices = n_end > n_begin ? (int)((n_end - n_begin + KS - 1) / KS) : 0;
    const int64_t nstages = (int64_t)nslices * tg;

    uint32_t sw[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) sw[m] = swz(lane, m);

    if (warp < PRODUCERS) {
        // ---- producers: A stage q = slice * tg + tile is made by the pair of warps q % (PRODUCERS / 2) -------------
        // A wait names a phase by its parity only, so a waiter must never be two phases ahead of its
        // barrier: with stages dealt round-robin to `nprod` pairs that holds when nprod <= NA (slots of
        // the A ring) and nprod <= NB * tg (stages covered by the slices of the X^T ring).
        const int nprod = min(min(PRODUCERS / 2, NA), NB * tg), pair = warp >> 1;
        const int e0 = (warp & 1) * (TI / 2);                 // values of i of this warp: e0 .. e0 + TI / 2 - 1 of the tile's
        bool ok = true;
        int bs = pair / tg, ti = pair - bs * tg, as = pair, use = 0;           // of stage q; bs: ring position of its slice
        uint32_t b_parity = 0;
        while (bs >= NB) { bs -= NB; b_parity ^= 1u; }
        const int dslice = nprod / tg, dti = nprod - dslice * tg;
        for (int64_t q = pair; q < nstages && ok && pair < nprod; q += nprod) {
            if (!mbar_wait(&b_full[bs], b_parity, abort_flag, a.status, 11)) break;
            // this lane's sample: x_i for the tile's 8 values of i, x_j for its 16 values of j
            const unsigned char *bst = b_stage0 + (size_t)bs * B_STAGE_BYTES;
            const Tile t = tiles[ti];
            // TF32: the rounded values of the MMA's own slice; bf16: the slice of X itself, samples `lane` and
            // `lane` + 32, so that every product is rounded once
            uint64_t xi[TI / 2], xj[TJ];                   // TF32: the low word only
            if (BF16) {
                const float *xst = x_stage0 + (size_t)bs * X_STAGE_FLOATS + lane * x_pitch;
#pragma unroll
                for (int e = 0; e < TI / 2; ++e) xi[e] = m3tc_pack2(xst[TI * t.ib + e0 + e], xst[(BF16 ? 32 : 0) * x_pitch + TI * t.ib + e0 + e]);
#pragma unroll
                for (int e = 0; e < TJ; ++e) xj[e] = m3tc_pack2(xst[TJ * t.jb + e], xst[(BF16 ? 32 : 0) * x_pitch + TJ * t.jb + e]);
            } else {
#pragma unroll
                for (int e = 0; e < TI / 2; ++e) xi[e] = *reinterpret_cast<const uint32_t *>(bst + (TI * t.ib + e0 + e) * 128 + swz(lane, e0 + e));
#pragma unroll
                for (int e = 0; e < TJ; ++e) xj[e] = *reinterpret_cast<const uint32_t *>(bst + (TJ * t.jb + e) * 128 + sw[e & 7]);
            }
            if (use > 0 && !mbar_wait(&a_empty[as], (uint32_t)((use - 1) & 1), abort_flag, a.status, 12)) {
                ok = false;
                break;
            }
            unsigned char *ast = a_stage0 + (size_t)as * A_STAGE_BYTES + e0 * TJ * 128;
#pragma unroll
            for (int e = 0; e < TI / 2; ++e)
#pragma unroll
                for (int f = 0; f < TJ; ++f) {
                    // row (e0 + e) * 16 + f of the tile
                    uint32_t v;
                    if (BF16) {
                        // two samples per word, each product rounded once to bf16 (first sample in the low half)
                        uint64_t p;
                        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(p) : "l"(xi[e]), "l"(xj[f]));
                        asm("{\n\t.reg .f32 a, b;\n\tmov.b64 {a, b}, %1;\n\tcvt.rn.bf16x2.f32 %0, b, a;\n\t}" : "=r"(v) : "l"(p));
                    } else {
                        // round to nearest TF32 (ties away from zero): the tensor core ignores the low 13 bits
                        v = __float_as_uint(__uint_as_float((uint32_t)xi[e]) * __uint_as_float((uint32_t)xj[f])) + 0x1000u;
                    }
                    *reinterpret_cast<uint32_t *>(ast + (e * TJ + f) * 128 + sw[f & 7]) = v;
                }
            fence_proxy_async();      // generic-proxy stores must be visible to the tensor core
            __syncwarp();
            if (lane == 0) mbar_arrive(&a_full[as]);
            bs += dslice;
            ti += dti;
            if (ti >= tg) { ti -= tg; ++bs; }
            while (bs >= NB) { bs -= NB; b_parity ^= 1u; }
            as += nprod;
            if (as >= NA) { as -= NA; ++use; }
        }

        // ---- epilogue: tensor memory -> this slice's partial sums ---------------------------------
        if (nstages > 0 && mbar_wait(acc_full, 0u, abort_flag, a.status, 13)) {
            tc_fence_after();
            // partial sums of a tile: [column][row], so that a warp stores 32 consecutive rows (pairs) of one column k
            // straight from tensor memory; rows with i > j are not outputs and are skipped
            float *__restrict__ mine = a.partials + (size_t)blockIdx.y * a.part_elems;
            const int q4 = warp & 3;                                // lanes 32*q4 .. 32*q4+31 of tensor memory
            for (int ti = warp >> 2; ti < tg; ti += PRODUCERS / 4) {
                const Tile t = tiles[ti];
                const int ncols = a.d - TJ * t.jb;                  // (with the columns that fill up to dcols [40009,50] bf16 35.7 us, without 33.4)
                uint32_t v[DP];
#pragma unroll
                for (int c0 = 0; c0 < DP; c0 += 16)                 // all loads of the tile in flight, one wait
                    if (c0 < ncols)
                        tmem_ld_32x16(tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(t.col + c0), v + c0);
                tmem_ld_wait();
                const int r = q4 * 32 + lane;
                const int i = TI * t.ib + r / TJ, j = TJ * t.jb + r % TJ;
                float *dst = mine + t.part + r;
                if (i <= j && j < a.d) {
#pragma unroll
                    for (int c0 = 0; c0 < DP; c0 += 16)
                        if (c0 < ncols) {
#pragma unroll
                            for (int e = 0; e < 16; ++e)
                                if (c0 + e < ncols && ST_BOUNDS_OK(t.part + r + (c0 + e) * BM, a.part_elems, 4)) dst[(c0 + e) * BM] = __uint_as_float(v[c0 + e]);
                        }
                }
            }
        }
    } else if (warp < LOAD_WARP) {
        // ---- MMA issuers: two warps.  A barrier poll issued behind tcgen05.mma instructions of the same thread
        // returns only as they drain, so one issuer alone leaves the tensor pipe idle while it polls.
        // A ring slot q % NA has the parity of q (NA is even), so every slot has one issuer and its uses are polled in
        // order.  An even number of tiles has one issuer each.  Of an odd number every tile changes issuers from slice to
        // slice, and MMAs of two threads into one accumulator are in no order by themselves: both issuers have then issued
        // all of a slice before either goes on to the next.
        const int iw = warp - MMA_WARP;
        if (elect_one()) {
            bool ok = true;
            int q_slot = 0;                                         // ring slot and phase of stage q = slice * tg + ti
            uint32_t q_parity = 0, b_parity = 0;
            int b_slot = 0;
            for (int slice = 0; slice < nslices && ok; ++slice) {
                const int bs = b_slot;
                if (!mbar_wait(&b_full[bs], b_parity, abort_flag, a.status, 14)) break;
                if (++b_slot == NB) { b_slot = 0; b_parity ^= 1u; }
                const uint32_t sb = smem_u32(b_stage0 + (size_t)bs * B_STAGE_BYTES);
                for (int ti = 0; ti < tg; ++ti) {
                    const int as = q_slot;
                    const uint32_t a_parity = q_parity;
                    const bool mine = (q_slot & 1) == iw;          // NA is even
                    if (++q_slot == NA) { q_slot = 0; q_parity ^= 1u; }
                    if (!mine) continue;
                    const Tile t = tiles[ti];
                    const int kstart = TJ * t.jb, ncols = a.dcols - kstart;
                    if (!mbar_wait(&a_full[as], a_parity, abort_flag, a.status, 15)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(a_stage0 + (size_t)as * A_STAGE_BYTES);
                    const uint32_t idesc = make_idesc(BF16 ? 1 : 2, 0, 0, BM, (uint32_t)ncols);
#pragma unroll
                    for (int kk = 0; kk < ROW_BYTES / 32; ++kk) {             // 32 bytes of K per MMA
                        const uint64_t adesc = make_smem_desc(sa + kk * 32, 16, 1024);
                        const uint64_t bdesc = make_smem_desc(sb + kstart * 128 + kk * 32, 16, 1024);
                        if (BF16) mma_bf16(tmem_base + (uint32_t)t.col, adesc, bdesc, idesc, (slice > 0 || kk > 0) ? 1u : 0u);
                        else mma_tf32(tmem_base + (uint32_t)t.col, adesc, bdesc, idesc, (slice > 0 || kk > 0) ? 1u : 0u);
                    }
                    tc_commit(&a_empty[as]);
                }
                if (!ok) break;
                tc_commit(&b_empty[bs]);
                if (tg % 2 != 0 && slice + 1 < nslices) {
                    tc_fence_before();
                    mbar_arrive(iss_sync);
                    if (!mbar_wait(iss_sync, (uint32_t)(slice & 1), abort_flag, a.status, 17)) break;
                    tc_fence_after();
                }
                if (slice == nslices - 1) tc_commit(acc_full);
            }
        }
    } else {
        // ---- loaders: slices of X by asynchronous copies, consecutive lanes along a row (one warp that read a
        // sample per lane, two round trips to memory per slice, was what the whole kernel waited for), then X^T
        // (row = column c of X) rounded to TF32 or bf16.  A lane owns one 4-byte word of every row of X^T: sample
        // `lane` (TF32) or samples `lane` and `lane` + 32 (bf16; the order of the samples is the one of the products).
        const int lt = (int)threadIdx.x - 32 * LOAD_WARP, lw = warp - LOAD_WARP;
        // the block's rows are asked for in L2 far ahead: PREFETCH slices now, one more with every slice fetched
        constexpr int PREFETCH = 16;
        auto prefetch = [&](int64_t first, int64_t last) {                // rows
            if (last > n_end) last = n_end;
            if (first >= last) return;
            const char *lo = reinterpret_cast<const char *>(a.X + first * a.ldx);
            const int64_t bytes = ((last - 1 - first) * a.ldx + a.d) * 4;
            for (int64_t o = 128 * (int64_t)lt; o < bytes; o += 128 * 32 * LOAD_WARPS) asm volatile("prefetch.global.L2 [%0];" ::"l"(lo + o));
        };
        prefetch(n_begin, n_begin + PREFETCH * KS);
        // a warp copies 32 / W rows at a time, W lanes along each (and a second time for columns 32 and up); lanes past
        // column d and samples past the end write zeros
        auto copy_rows = [&](auto width, int64_t n0, int rows, uint32_t dst) {
            constexpr int W = decltype(width)::value, STEP = 32 * LOAD_WARPS / W;
            const int r0 = lt / W, c = lt % W;
            const float *src = a.X + (n0 + r0) * a.ldx + c;
            const int64_t src_step = STEP * a.ldx;
            const bool c0 = c < a.d, c1 = W == 32 && c + 32 < a.d, wide = W == 32 && a.dcols > 32;
            dst += (uint32_t)(r0 * x_pitch + c) * 4u;
            if (W == 32 && rows == KS) {
                // a whole slice: lanes of columns past d copy nothing (their words are zeros from the start)
                const uint32_t dst_step = (uint32_t)(STEP * x_pitch) * 4u;
#pragma unroll 8
                for (int u = 0; u < KS / STEP; ++u, dst += dst_step, src += src_step) {
                    if (c0) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src));
                    if (c1) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 128u), "l"(src + 32));
                }
                return;
            }
#pragma unroll 8
            for (int r = r0; r < KS; r += STEP, dst += (uint32_t)(STEP * x_pitch) * 4u, src += src_step) {
                const bool p0 = c0 && r < rows, p1 = c1 && r < rows;
                const float *s0 = p0 ? src : a.X, *s1 = p1 ? src + 32 : a.X;
                if (W == 32 || c < a.dcols)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(s0), "r"(p0 ? 4 : 0));
                if (wide && c + 32 < a.dcols)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 128u), "l"(s1), "r"(p1 ? 4 : 0));
            }
        };
        // columns past d: zeros in every buffer before the first copy
        for (int r = a.dcols > 16 ? lt : NB * KS; r < NB * KS; r += 32 * LOAD_WARPS)
            for (int c = a.d; c < a.dcols; ++c) x_stage0[(size_t)(r / KS) * X_STAGE_FLOATS + (r % KS) * x_pitch + c] = 0.f;
        int fetch_slot = 0;
        auto fetch = [&](int slice) {                                     // called with slice = 0, 1, 2, ...
            const int64_t n0 = n_begin + (int64_t)slice * KS;
            const int rows = n_end - n0 < KS ? (int)(n_end - n0) : KS;
            const uint32_t dst = smem_u32(x_stage0 + (size_t)fetch_slot * X_STAGE_FLOATS);
            if (++fetch_slot == NB) fetch_slot = 0;
            if (a.dcols == 16) copy_rows(std::integral_constant<int, 16>{}, n0, rows, dst);
            else copy_rows(std::integral_constant<int, 32>{}, n0, rows, dst);
            prefetch(n0 + PREFETCH * KS, n0 + (PREFETCH + 1) * KS);
        };
        const int ahead = fetch_ahead(NB);
        for (int s = 0; s < ahead; ++s) {
            if (s < nslices) fetch(s);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        int bs = 0;
        uint32_t free_parity = 1;                                         // of the buffers that the next fetch fills
        for (int slice = 0; slice < nslices; ++slice) {
            // a slice's buffers are free once the MMAs of the slice NB before it are complete
            uint32_t failed = 0;
            const int next = slice + ahead;
            if (next < nslices) {
                if (next >= NB && fetch_slot == 0) free_parity ^= 1u;
                if (next >= NB && !mbar_wait(&b_empty[fetch_slot], free_parity, abort_flag, a.status, 16)) failed = 1;
                else fetch(next);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            if (ahead == 8) asm volatile("cp.async.wait_group 8;" ::: "memory");
            else if (ahead == 5) asm volatile("cp.async.wait_group 5;" ::: "memory");
            else asm volatile("cp.async.wait_group 2;" ::: "memory");
            // every loader's copies of the slice have landed; all loaders leave together if one gave up
            asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %0, 0;\n\tbar.red.or.pred q, 1, %1, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                         : "+r"(failed) : "n"(32 * LOAD_WARPS) : "memory");
            if (failed) break;
            unsigned char *bst = b_stage0 + (size_t)bs * B_STAGE_BYTES;
            const float *xst = x_stage0 + (size_t)bs * X_STAGE_FLOATS + lane * x_pitch;
            for (int c8 = 8 * lw; c8 < a.dcols; c8 += 8 * LOAD_WARPS) {
                float x[8], y[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    x[c] = xst[c8 + c];
                    y[c] = BF16 ? xst[(BF16 ? 32 * x_pitch : 0) + c8 + c] : 0.f;
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    uint32_t t;
                    if (BF16) asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(t) : "f"(y[c]), "f"(x[c]));
                    else asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(t) : "f"(x[c]));
                    *reinterpret_cast<uint32_t *>(bst + (c8 + c) * 128 + sw[c]) = t;
                }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&b_full[bs]);
            if (++bs == NB) bs = 0;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

struct SumArgs {
    const float *partials;
    float *out;
    int slices, part_elems, d, ntiles;
    Tile tiles[MAX_TILES];
};

// out[q(i,j,k)] = sum over the slices of the partial sum of row (i, j), column k of a tile: a block owns a column, a lane four of its
// 128 rows, warp w of W adds the slices w, w + W, ... with its loads in flight, then the sums of the warps are added in order.  Eight
// to 32 warps, so that one batch of loads is enough for most.  With a float to a lane and eight warps there were four times
// as many blocks, more than fit at once: [4096,64] bf16 17.7 us the call, now 13.3; [40009,50] 33.4 and 32.3; [256,50] 9.9 and 8.0;
// with eight warps whatever the slices [40009,16] 15.1, now 11.4.
constexpr int SUM_BATCH = 5, MAX_SUM_WARPS = 32;
constexpr int sum_warps(int slices) { return slices <= 8 * SUM_BATCH ? 8 : slices <= 16 * SUM_BATCH ? 16 : MAX_SUM_WARPS; }
__global__ void __launch_bounds__(32 * MAX_SUM_WARPS)
moment3_tc_sum_kernel(const __grid_constant__ SumArgs a)
{
    __shared__ float4 part[MAX_SUM_WARPS][BM / 4];
    const int warps = blockDim.x >> 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int e = blockIdx.x * BM;
    int ti = 0;
    while (ti + 1 < a.ntiles && a.tiles[ti + 1].part <= e) ++ti;
    const Tile t = a.tiles[ti];
    const int k = TJ * t.jb + (e - t.part) / BM;
    // rows 4 lane .. 4 lane + 3 have one i and four j; one of them at least is an output, or none is read
    const bool any = TI * t.ib + 4 * lane / TJ <= min(TJ * t.jb + 4 * lane % TJ + 3, k) && TJ * t.jb + 4 * lane % TJ <= k;
    pdl_wait();
    pdl_trigger();
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (any) {
        const float *p = a.partials + e + 4 * lane;
        for (int k0 = warp; k0 < a.slices; k0 += SUM_BATCH * warps) {
            float4 v[SUM_BATCH];
#pragma unroll
            for (int u = 0; u < SUM_BATCH; ++u)
                v[u] = k0 + u * warps < a.slices ? __ldcg(reinterpret_cast<const float4 *>(p + (size_t)(k0 + u * warps) * a.part_elems))
                                                     : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < SUM_BATCH; ++u) { s.x += v[u].x; s.y += v[u].y; s.z += v[u].z; s.w += v[u].w; }
        }
    }
    part[warp][lane] = s;
    __syncthreads();
    const int r = threadIdx.x, i = TI * t.ib + r / TJ, j = TJ * t.jb + r % TJ;
    if (r >= BM || !(i <= j && j <= k)) return;
    float sum = 0.f;
#pragma unroll 8
    for (int w = 0; w < warps; ++w) sum += reinterpret_cast<const float *>(part[w])[r];
    const int64_t at = tet_encode(a.d, i, j, k);
    if (ST_BOUNDS_OK(at, tet_rows(a.d), 4)) a.out[at] = sum;
}

struct Plan {
    int groups, slices, dcols, ntiles;
    int first[MAX_GROUPS + 1];
    Tile tiles[MAX_TILES];
    int64_t rows_per_slice;
    int part_elems;
    bool ok;
};

static Plan plan(int64_t N, int64_t d, bool bf16)
{
    const int KS = bf16 ? 64 : 32;
    Plan p{};
    p.ok = false;
    if (N <= 0 || d < 1 || d > DP) return p;
    p.dcols = (int)((d + 15) / 16 * 16);
    // tiles in the order (JB, IB); a tile exists when it holds some i <= j < d
    int cols[MAX_TILES], n = 0;
    for (int jb = 0; jb * TJ < d; ++jb)
        for (int ib = 0; ib * TI < d && ib * TI <= jb * TJ + TJ - 1; ++ib) {
            if (n >= MAX_TILES) return p;
            p.tiles[n].ib = (unsigned char)ib;
            p.tiles[n].jb = (unsigned char)jb;
            cols[n] = p.dcols - jb * TJ;
            p.tiles[n].part = p.part_elems;
            p.part_elems += ((int)d - jb * TJ) * BM;      // columns past d are not stored
            ++n;
        }
    p.ntiles = n;
    // Groups: the number for which the longest block and the sum after it take least, in cycles: 230 a stage, but 2000 a slice at
    // least (what fetching and turning it takes), 650 a tile for its partial sums (two at least: one is no faster), 60 a slice in the
    // sum.  With 1, 2, 4 and 8 groups, bf16, us: [256,33] 11.2, 9.3, 8.2, 7.6; [4096,33] 11.9, 10.2, 10.0, 10.8; [40009,33] 23.6,
    // 22.5, 26.1, 40.6; [200000,33] 66, 77, 101, 175.  With 1, 2 and 4: [4096,32] 9.5, 8.5, 8.4, TF32 10.6, 9.5, 9.7; [16384,32]
    // 12.4, 12.4, 12.6, TF32 14.9, 14.8, 16.6; with 1 and 2: [4096,16] 7.4, 7.6, TF32 8.6, 8.3; [40009,16] 11.8, 14.2, TF32 15.7, 19.1.
    // Before, with as few groups as tensor memory allows: [256,50] 15.1, now 11.2; [256,64] 16.1, 12.1.
    const int sms = sm_count_or_default();
    double best = 0;
    for (int groups = 1; groups <= MAX_GROUPS && groups <= n && groups <= sms; ++groups) {
        // equal numbers of tiles: the stores of P are the bound
        int first[MAX_GROUPS + 1], longest = 0;
        bool fits = true;
        for (int g = 0; g <= groups; ++g) first[g] = (int)((int64_t)n * g / groups);
        for (int g = 0; g < groups; ++g) {
            int col = 0;
            for (int t = first[g]; t < first[g + 1]; ++t) col += cols[t];
            if (first[g + 1] - first[g] > longest) longest = first[g + 1] - first[g];
            fits = fits && col <= (int)TMEM_COLS;
        }
        if (!fits || longest > MAX_GROUP_TILES) continue;
        int64_t slices = sms / groups, rps = ((N + slices - 1) / slices + KS - 1) / KS * KS;      // whole MMA slices
        slices = (N + rps - 1) / rps;
        const double cost = (double)(rps / KS) * (longest * 230 > 2000 ? longest * 230 : 2000) + (longest > 2 ? longest : 2) * 650 + (double)slices * 60;
        if (p.ok && cost >= best) continue;
        best = cost;
        p.groups = groups;
        p.slices = (int)slices;
        p.rows_per_slice = rps;
        for (int g = 0; g <= groups; ++g) p.first[g] = first[g];
        p.ok = true;
    }
    for (int g = 0; g < p.groups; ++g)
        for (int t = p.first[g], col = 0; t < p.first[g + 1]; col += cols[t++]) p.tiles[t].col = (unsigned short)col;
    return p;
}

}  // namespace m3tc

size_t moment3_tc_workspace(int64_t N, int64_t d, bool bf16)
{
    const m3tc::Plan p = m3tc::plan(N, d, bf16);
    if (!p.ok) return 0;
    return kWsHeaderBytes + (size_t)p.slices * p.part_elems * sizeof(float);
}

st_status moment3_tc(const float *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes,
                     bool bf16, cudaStream_t stream)
{
    using namespace m3tc;
    const Plan p = plan(N, d, bf16);
    if (!p.ok) return ST_ERR_UNSUPPORTED;
    const size_t need = kWsHeaderBytes + (size_t)p.slices * p.part_elems * sizeof(float);
    if (!ws || ws_bytes < need) return ST_ERR_WORKSPACE;
    if (!aligned256(ws)) return ST_ERR_ALIGN;
    const DeviceInfo di = device_info();
    if (!di.ok) return ST_ERR_CUDA;
    if (smem_bytes(p.dcols, bf16) > (size_t)di.max_smem_optin) return ST_ERR_UNSUPPORTED;
    Args a;
    a.X = X;
    a.partials = (float *)((unsigned char *)ws + kWsHeaderBytes);
    a.status = (unsigned *)ws;
    a.N = N; a.ldx = ldx; a.rows_per_slice = p.rows_per_slice;
    a.nb = ring(p.dcols, bf16);
    a.d = (int)d; a.dcols = p.dcols; a.part_elems = p.part_elems;
    for (int g = 0; g <= MAX_GROUPS; ++g) a.first[g] = p.first[g <= p.groups ? g : p.groups];
    for (int t = 0; t < MAX_TILES; ++t) a.tiles[t] = p.tiles[t];
    auto run = [&](auto kernel) {
        if (!ensure_dynamic_smem(kernel, smem_bytes(p.dcols, bf16))) return ST_ERR_CUDA;
        return launch(kernel, dim3(p.groups, p.slices), THREADS, smem_bytes(p.dcols, bf16), stream, a);
    };
    const st_status rc = bf16 ? run(moment3_tc_kernel<true>) : run(moment3_tc_kernel<false>);
    if (rc != ST_OK) return rc;
    SumArgs m;
    m.partials = a.partials;
    m.out = out;
    m.slices = p.slices;
    m.part_elems = p.part_elems;
    m.d = (int)d;
    m.ntiles = p.ntiles;
    for (int t = 0; t < MAX_TILES; ++t) m.tiles[t] = p.tiles[t];
    return launch(moment3_tc_sum_kernel, (unsigned)(p.part_elems / BM), 32 * sum_warps(p.slices), 0, stream, m);
}

}  // namespace st
