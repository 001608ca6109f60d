// st_ttm_blockdiag, tensor-core path (ST_FLAG_TC_TF32): Ap[m, r] = sum_k Bp[m, k] U[k, r] over
// the fibres of the diagonal blocks only (Table 1, TTM; B is a direct sum of blocks).  In the
// packed layout the whole operation is one tall-skinny GEMM [rows, K] x [K, R]; what the
// structure buys is that the fibres of the zero blocks are never read.  HBM bound.
//
// Persistent blocks walk tiles of 128 packed fibres.  Per tile, K is streamed in slices of 32
// floats by TMA (128-byte swizzle, K-major A operand read as TF32 by the tensor core: the low
// 13 mantissa bits are ignored).  U is rounded to TF32, transposed once per block into the
// same swizzled K-major form and stays in shared memory.  The 128 x R fp32 accumulator lives
// in tensor memory, double buffered so that the epilogue of one tile overlaps the MMAs of the
// next.  Warp roles: warp 0 TMA producer, warp 1 MMA issuer / TMEM owner, warps 2..9 epilogue, two groups
// of four on alternate tiles.
#include "tc_common.cuh"
#include "st_index.cuh"
#include "fibre_epilogue.cuh"

namespace st {

namespace ttmtc {
constexpr int BM = 128;                    // fibres per tile
constexpr int KC = 32;                     // floats per k-slice (128 bytes)
constexpr int STAGE_BYTES = BM * KC * 4;   // 16 KiB
// Groups of four epilogue warps, on alternate tiles.  Short fibres leave an MTTKRP tile's epilogue (two dependent trips to L2)
// as the chain: I = 900, K = 48, R = 64 runs 59 us with one group, 42 with two.
constexpr int EPI_GROUPS = 2;
constexpr int THREADS = 64 + 128 * EPI_GROUPS;
// 96 KB of fibres in flight per SM: a copy loop without arithmetic reads 269 MB at 6.5 TB/s with six stages, 5.9 with ten and
// 5.8 with thirteen (the memory system queues); this kernel 56.4 us with five or six ([64,64,64,256] x [256,64], 269 MB
// read, 67 written), 57.2 with eight, 58.9 with ten, 58.8 with four.
constexpr int MAX_STAGES = 6;
}  // namespace ttmtc

enum { TC_TTM = 0, TC_MTTKRP_PACKED = 1, TC_MTTKRP_DENSE = 2 };

struct TtmTcArgs {
    const float *U;
    const float *C;      // MTTKRP: [I, R]
    int I, mode;
    int64_t div;         // TC_MTTKRP_DENSE: fibre `row` belongs to (i, j) = (row / div, row % div)
    float *out;
    unsigned *status;
    int64_t rows;
    int K, R, kchunks, ntiles, stages;
    int reverse;         // walk the tiles from the last one down (see tc_rows_launch)
    uint32_t tmem_cols;
};

__global__ void __launch_bounds__(ttmtc::THREADS, 1)
ttm_tc_kernel(const __grid_constant__ CUtensorMap tmap, const TtmTcArgs a)
{
    using namespace ttmtc;
    using namespace tc;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int u_region = a.R * 128;                                  // bytes of one k-slice of U^T (multiple of 2048)
    unsigned char *u_smem = smem;                                    // kchunks regions
    unsigned char *stage0 = smem + (size_t)a.kchunks * u_region;
    uint64_t *bars = (uint64_t *)(stage0 + (size_t)a.stages * STAGE_BYTES);
    uint64_t *full = bars, *empty = bars + MAX_STAGES, *acc_full = bars + 2 * MAX_STAGES,
             *acc_empty = bars + 2 * MAX_STAGES + 2;
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * MAX_STAGES + 4);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4);     // one arrival per epilogue warp
        }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, a.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
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

    if (warp != 0) {
        // The other warps build U^T while warp 0 already streams fibres: U rounded to TF32, K-major with the 128-byte
        // swizzle; element (r, k) of slice k/32 goes to byte r*128 + ((k%32/4) ^ (r%8))*16 + (k%4)*4 of that slice's
        // region.  A warp takes (slice, 16 columns r): lane = (4 columns, four of the 32 k); it loads float4 U[k + e, r ..]
        // and stores 16 bytes per column, the eight lanes of a column one row of 128 bytes (single words of
        // neighbouring columns met 16 lanes in one bank: [2080,300] R = 128 18.4 us, now 12.2;
        // [65536,256] blocks R = 64 54.6, now 53.4).
        const int nw = THREADS / 32 - 1, items = a.kchunks * (a.R / 16), q = lane & 7;
        constexpr int UB = 4;
        for (int i0 = warp - 1; i0 < items; i0 += UB * nw) {
            float4 v[UB][4];                                          // sixteen independent loads in flight: U comes from cold memory
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int it = i0 + u * nw, kc = it / (a.R / 16), r0 = (it - kc * (a.R / 16)) * 16 + (lane >> 3) * 4;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int k = kc * KC + 4 * q + e;
                    v[u][e] = it < items && k < a.K ? *reinterpret_cast<const float4 *>(a.U + (size_t)k * a.R + r0)
                                                    : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int it = i0 + u * nw, kc = it / (a.R / 16), r0 = (it - kc * (a.R / 16)) * 16 + (lane >> 3) * 4;
                if (it >= items) break;
                unsigned char *region = u_smem + (size_t)kc * u_region;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int r = r0 + j;
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(w[e]) : "f"(j == 0 ? v[u][e].x : j == 1 ? v[u][e].y : j == 2 ? v[u][e].z : v[u][e].w));
                    *reinterpret_cast<uint4 *>(region + r * 128 + ((q ^ (r & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
        }
        fence_proxy_async();      // make the generic-proxy writes of U visible to the tensor core
        asm volatile("bar.sync 1, %0;" ::"n"(THREADS - 32) : "memory");
    }

    const int my_tiles = (a.ntiles > (int)blockIdx.x) ? (a.ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

    if (warp == 0) {
        if (elect_one()) {
            prefetch_tmap(&tmap);
            // ring position and barrier phase are carried in counters: a 64-bit division per stage would cost
            // this single thread a good part of the time one stage takes to arrive
            int s = 0;
            uint32_t empty_parity = 0;
            bool first_pass = true, ok = true;
            for (int t = 0; t < my_tiles && ok; ++t) {
                int64_t tile = blockIdx.x + (int64_t)t * gridDim.x;
                if (a.reverse) tile = a.ntiles - 1 - tile;
                const int y = (int)(tile * BM);
                for (int kc = 0; kc < a.kchunks; ++kc) {
                    if (!first_pass && !mbar_wait(&empty[s], empty_parity, abort_flag, a.status, 1)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(&full[s], STAGE_BYTES);
                    tma_load_2d(stage0 + (size_t)s * STAGE_BYTES, &tmap, &full[s], kc * KC, y);
                    if (++s == a.stages) {
                        s = 0;
                        if (first_pass) first_pass = false;
                        else empty_parity ^= 1u;
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = make_idesc(2, 0, 0, BM, (uint32_t)a.R);
            int s = 0;
            uint32_t full_parity = 0;
            bool ok = true;
            for (int t = 0; t < my_tiles && ok; ++t) {
                const int buf = t & 1;
                const int use = t >> 1;
                if (use > 0 && !mbar_wait(&acc_empty[buf], (uint32_t)((use - 1) & 1), abort_flag, a.status, 2)) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * a.R);
                for (int kc = 0; kc < a.kchunks; ++kc) {
                    if (!mbar_wait(&full[s], full_parity, abort_flag, a.status, 3)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(stage0 + (size_t)s * STAGE_BYTES);
                    const uint32_t sb = smem_u32(u_smem + (size_t)kc * u_region);
#pragma unroll
                    for (int kk = 0; kk < KC / 8; ++kk) {
                        const uint64_t adesc = make_smem_desc(sa + kk * 32, 16, 1024);
                        const uint64_t bdesc = make_smem_desc(sb + kk * 32, 16, 1024);
                        mma_tf32(d_tmem, adesc, bdesc, idesc, (kc > 0 || kk > 0) ? 1u : 0u);
                    }
                    tc_commit(&empty[s]);
                    if (++s == a.stages) {
                        s = 0;
                        full_parity ^= 1u;
                    }
                }
                tc_commit(&acc_full[buf]);
            }
        }
    } else {
        const int q = warp & 3;
        for (int t = (warp - 2) >> 2; t < my_tiles; t += EPI_GROUPS) {
            const int buf = t & 1;
            int64_t tile = blockIdx.x + (int64_t)t * gridDim.x;
            if (a.reverse) tile = a.ntiles - 1 - tile;
            const int64_t unit = tile * (BM / 32) + q;
            // MTTKRP: the fibres' (i, j) and the first columns of their rows of C are fetched before the accumulator is
            // waited for -- with the memory system saturated by the fibre stream a dependent load costs
            // microseconds
            UnitFibres f;
            float2 cpre[2][4];
            if (a.mode != TC_TTM) {
                f = unit_fibres(unit * 32, a.rows, a.mode == TC_MTTKRP_DENSE, a.I, a.div, lane);
                unit_load_c(f, a.C, a.R, 0, lane, cpre);
            }
            if (!mbar_wait(&acc_full[buf], (uint32_t)((t >> 1) & 1), abort_flag, a.status, 4)) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * a.R);
            if (a.mode == TC_TTM) ttm_epilogue<false>(taddr, a.R, unit * 32, a.rows, a.out, lane);
            else mttkrp_epilogue<false>(taddr, a.R, f, a.C, unit, a.out, mttkrp_slots(a.rows, 32, a.I, 1), lane, cpre);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, a.tmem_cols);
    }
}

struct TtmTcPlan {
    int kchunks, stages;
    uint32_t tmem_cols;
    size_t smem;
    bool ok;
};

static TtmTcPlan ttm_tc_plan(int64_t K, int64_t R)
{
    using namespace ttmtc;
    TtmTcPlan p{};
    p.ok = false;
    if (K <= 0 || R <= 0 || K % 4 != 0 || R % 16 != 0 || R > 256 || K > (1 << 20)) return p;
    p.kchunks = (int)((K + KC - 1) / KC);
    // two accumulators of R columns, which the epilogue reads 16 columns at a time; an allocation is a power of two, at least 32
    uint32_t cols = 32;
    while (cols < 2 * (uint32_t)R) cols *= 2;
    p.tmem_cols = cols;
    const size_t u_bytes = (size_t)p.kchunks * R * 128;
    const size_t fixed = 1024 + u_bytes + 512;
    const size_t budget = 227 * 1024;
    if (fixed + 2 * STAGE_BYTES > budget) return p;
    size_t st = (budget - fixed) / STAGE_BYTES;
    if (st > MAX_STAGES) st = MAX_STAGES;
    p.stages = (int)st;
    p.smem = fixed + st * STAGE_BYTES;
    p.ok = true;
    return p;
}

size_t ttm_tf32_tc_workspace(int64_t rows, int64_t K, int64_t R)
{
    if (rows <= 0) return 0;
    return ttm_tc_plan(K, R).ok ? kWsHeaderBytes : 0;
}

static st_status tc_rows_launch(const float *Bp, int64_t rows, int64_t K, const float *U, int64_t R, float *Ap,
                                const float *C, int64_t I, int mode, void *ws, size_t ws_bytes, cudaStream_t stream,
                                int64_t div = 0);

st_status ttm_tf32_tc(const float *Bp, int64_t rows, int64_t K, const float *U, int64_t R, float *Ap, void *ws,
                      size_t ws_bytes, cudaStream_t stream)
{
    return tc_rows_launch(Bp, rows, K, U, R, Ap, nullptr, 0, TC_TTM, ws, ws_bytes, stream);
}

size_t mttkrp_tf32_tc_workspace(int64_t rows, int64_t I, int64_t K, int64_t R)
{
    if (rows <= 0 || R % 32 != 0 || !ttm_tc_plan(K, R).ok) return 0;
    return kWsHeaderBytes + (size_t)mttkrp_slots(rows, 32, I, 1) * R * sizeof(float);
}

// MTTKRP on tensor cores: the same streaming kernel with W = D; the epilogue scales every fibre's result
// by C[j,:] and writes the sums of the runs of equal i to the workspace, a second kernel adds them in a
// fixed order (mttkrp_common.cuh).  `m` says how a row maps to (i, j); the fibres reach rows
// i_off .. i_off + m.I - 1 of A_full, which has I_full rows.  TF32 operands, 5e-3 tolerance.
st_status mttkrp_tf32_tc(const float *Bp, const MttkrpRows &m, int64_t K, const float *C, const float *D, int64_t R,
                         float *A_full, int64_t I_full, int64_t i_off, void *ws, size_t ws_bytes, cudaStream_t stream)
{
    if (R % 32 != 0) return ST_ERR_UNSUPPORTED;
    const size_t need = mttkrp_tf32_tc_workspace(m.rows, m.I, K, R);
    if (need == 0) return ST_ERR_UNSUPPORTED;
    if (!ws || ws_bytes < need) return ST_ERR_WORKSPACE;
    float *part = (float *)((unsigned char *)ws + kWsHeaderBytes);
    const st_status rc = tc_rows_launch(Bp, m.rows, K, D, R, part, C, m.I, m.mode == MK_PACKED ? TC_MTTKRP_PACKED : TC_MTTKRP_DENSE,
                                        ws, ws_bytes, stream, m.div);
    if (rc != ST_OK) return rc;
    return mttkrp_rowsum_launch(part, A_full, I_full, i_off, m, (int)R, 32, 1, stream);
}

static st_status tc_rows_launch(const float *Bp, int64_t rows, int64_t K, const float *U, int64_t R, float *Ap,
                                const float *C, int64_t I, int mode, void *ws, size_t ws_bytes, cudaStream_t stream,
                                int64_t div)
{
    using namespace ttmtc;
    const TtmTcPlan p = ttm_tc_plan(K, R);
    if (!p.ok) return ST_ERR_UNSUPPORTED;
    if (rows > (int64_t(1) << 31) - BM) return ST_ERR_UNSUPPORTED;
    if (!ws || ws_bytes < kWsHeaderBytes) return ST_ERR_WORKSPACE;
    if (!aligned256(ws)) return ST_ERR_ALIGN;
    const DeviceInfo di = device_info();
    if (!di.ok) return ST_ERR_CUDA;
    if (p.smem > (size_t)di.max_smem_optin) return ST_ERR_UNSUPPORTED;
    CUtensorMap tmap;
    if (!tc::make_tmap_2d(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, Bp, (uint64_t)rows, (uint64_t)K, (uint64_t)K * 4, KC,
                          BM))
        return ST_ERR_CUDA;
    TtmTcArgs a;
    a.U = U; a.C = C; a.I = (int)I; a.mode = mode; a.div = div > 0 ? div : (I > 0 ? I : 1); a.out = Ap; a.status = (unsigned *)ws; a.rows = rows; a.K = (int)K; a.R = (int)R;
    a.kchunks = p.kchunks; a.stages = p.stages; a.tmem_cols = p.tmem_cols;
    a.ntiles = (int)((rows + BM - 1) / BM);
    // MTTKRP usually runs right after the call that produced its packed operand (st_pack, or a kernel
    // that writes packed output).  The end of that operand is then still in L2, so the tiles are walked
    // from the last one down: what was written last is read first, before later fills evict it.
    a.reverse = mode != TC_TTM ? 1 : 0;
    if (!ensure_dynamic_smem(ttm_tc_kernel, p.smem)) return ST_ERR_CUDA;
    const int grid = a.ntiles < di.sm_count ? a.ntiles : di.sm_count;
    return launch(ttm_tc_kernel, grid, THREADS, p.smem, stream, tmap, a);
}

}  // namespace st
