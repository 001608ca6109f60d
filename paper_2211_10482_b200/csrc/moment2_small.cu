// st_sym_moment2, fp32 path for few features (see moment2_use_small in moment2.cu) -- the regime
// of the paper's covariance workloads (Section 7.2; its real datasets have 6 and 13 features).
//
// out[p(i,j)] = sum_n X[n,i] X[n,j], 0 <= i <= j < d  (Section 3, M1; Section 5.5, y_U = i <= j).
//
// The d columns, padded to a multiple of 8, are dealt to "column blocks" of 8; block b owns columns 4b..4b+3 of the first half
// of a row and the same four of the second half (two 16-byte chunks, so that the threads of a warp
// read one contiguous 128-byte segment per load and a row can stay in its natural layout).  Every
// unordered pair of columns lies in exactly one unordered pair of blocks, so the 8x8 tiles {x,y}
// (x <= y) cover the unique set once: 36 tiles for d = 64, not 64.
//
// Shared memory returns 32 words per cycle to the registers of an SM, against 128 FMA lanes: an
// 8x8 register tile (16 operand words per 64 FMAs) saturates both at once.  A work item is
// therefore two tiles with one block in common, {s,p} and {s,q}: 24 operand words per 128 FMAs.
// The host pairs the tiles up (an odd one out computes its tile twice and drops one copy).  The
// rows of a shared-memory stage are dealt to RG "row groups"; one thread owns (item, row group)
// and keeps the 128 sums of its item over its rows in registers.  Blocks own slices of the samples
// (one block per SM), receive them in a 3-buffer pipeline of bulk copies, add their row groups in
// shared memory in a fixed order and write one partial per block; a second kernel adds the
// partials in slice order.  Diagonal tiles compute all 64 products (the 28 below the diagonal are
// dropped): 36*64 = 2304 FMAs issued per sample for 2080 useful.
#include "st_common.cuh"
#include "st_index.cuh"
#include "tc_common.cuh"
#include "moment2_rule.cuh"
#include <tuple>
#include <type_traits>

namespace st {

constexpr int M2S_MAX_THREADS = 256;
constexpr int M2S_MAX_BLOCKS = 31;         // column blocks: one item per thread at most (d <= 248; dense control: 22 blocks)
constexpr int M2S_BUFFERS = 3;
constexpr int M2S_CLUSTER_THREADS = 128;   // half the threads: half the sums to add ([4096,64] 7.1 us, with 256 threads 7.9)
constexpr int M2S_CLUSTER_ITEMS = 5;       // at most, per cluster ([4096,100]: five 9.3 us, three 15.2; [4096,64]: 7.1, nine 8.1)
constexpr int M2S_STAGE_BYTES = 57344;     // upper bound of one stage (3 stages + slack fit in 227 KB)

// bulk copy global -> shared of `bytes` (a multiple of 16, both addresses 16-byte aligned),
// completion counted in bytes on `bar`
__device__ __forceinline__ void m2s_bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     tc::smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(tc::smem_u32(bar))
                 : "memory");
}

// Number of work items, and item t: tiles {s,p} and {s,q} of column blocks (q = -1: one tile only).  Structured:
// for every block y the tiles {x,y}, x <= y, are paired along x with y as the common block (floor(y^2/4) items come
// before those of y); when their number is odd, tile {0,y} is held back, and the held-back tiles (y even) are paired
// with block 0 in common.  Dense control: all ordered tiles (x,y), paired along y with x in common.
__host__ __device__ inline int m2s_nitems(int nbk, bool dense)
{
    return dense ? nbk * ((nbk + 1) / 2) : (nbk * (nbk + 1) / 2 + 1) / 2;
}
__device__ __forceinline__ void m2s_item(int t, int nbk, bool dense, int &s, int &p, int &q)
{
    if (dense) {
        const int per = (nbk + 1) / 2;
        s = t / per;
        p = 2 * (t - s * per);
        q = p + 1 < nbk ? p + 1 : -1;
        return;
    }
    const int paired = nbk * nbk / 4;
    if (t < paired) {
        int y = (int)(2.f * sqrtf((float)t));
        while (y * y / 4 > t) --y;
        while ((y + 1) * (y + 1) / 4 <= t) ++y;
        s = y;
        p = ((y + 1) & 1) + 2 * (t - y * y / 4);
        q = p + 1;
    } else {
        s = 0;
        p = 4 * (t - paired);
        q = p + 2 < nbk ? p + 2 : -1;
    }
}

// Pitch, in words, of the block-level sum's buffer: at least rg * nitems, and nitems modulo 32.
__host__ __device__ inline int m2s_red_pitch(int rg, int nitems)
{
    const int cells = rg * nitems;
    return cells + ((nitems - cells) & 31);
}

struct M2SmallArgs {
    const float *X;
    float *partials;      // [slices][128][nitems]
    unsigned *status;     // workspace header (status and detail words)
    int64_t N, ldx, rows_per_slice;
    int d, pitch, nbk, nitems, rg, rpg, dense, bar_floats;
    float *out;           // CLUSTER: the result
    int items_all;        // CLUSTER: nitems counts those of a cluster
};

// column of element e (0..7) of column block b
__device__ __forceinline__ int m2s_column(int b, int e, int half) { return (e < 4) ? 4 * b + e : half + 4 * b + (e - 4); }

// Whether element k of an item is an output, and which: not the second tile of the odd item out; not the lower half of a
// diagonal tile (the dense control also computes the tiles below the diagonal and discards them here); not the padding of
// the last column blocks.
__device__ __forceinline__ bool m2s_output(int k, int item, int nbk, bool dense, int d, int64_t &at)
{
    const int i8 = (k >> 3) & 7, j8 = k & 7;
    int x, p, q;
    m2s_item(item, nbk, dense, x, p, q);
    const int y = (k < 64) ? p : q;
    const int ci = m2s_column(x, i8, 4 * nbk), cj = m2s_column(y, j8, 4 * nbk);
    at = tri_encode(d, ci < cj ? ci : cj, ci < cj ? cj : ci);
    return y >= 0 && !((x == y && i8 > j8) || (dense && x > y)) && ci < d && cj < d;
}

// BULK: rows start on 16-byte boundaries and arrive by bulk copies, in shared memory at their own pitch; otherwise
// they are copied word by word to a pitch rounded up to 16 bytes (one copy instruction per 32 words, against more
// than 64 FMA instructions).  Either way a tile that reaches past column d reads whatever follows the row: only
// sums that are dropped contain it.  [50021,75]: 18 us the call, 71 with the plain 64 x 64 tiles that served it before.
// What bounds it: two warps to a scheduler issue in 68 % of the cycles ([300000,64]; FMA pipe 59 %), the rest waits for operands.
// Packed FMAs (two to an instruction) are slower here, [1000000,64] 109 us instead of 102, and so is the next row's operands loaded
// ahead of this one's FMAs, 107: both take registers from what the compiler overlaps by itself.
// CLUSTER: few samples, one launch.  A cluster of M2S_CLUSTER blocks (gridDim.x) owns nitems work items (gridDim.y clusters),
// its blocks own slices of the samples, and the sums of the blocks are added through distributed shared memory instead of
// partials and a second launch.
template <bool BULK, bool CLUSTER>
__global__ void __launch_bounds__(M2S_MAX_THREADS, 1) moment2_small_kernel(const M2SmallArgs a)
{
    extern __shared__ __align__(16) float smem[];
    const int stage_rows = a.rg * a.rpg;
    const int stage_floats = stage_rows * a.pitch;
    const int tid = threadIdx.x, nthreads = blockDim.x;
    const int nitems = a.nitems;
    const int item_rg = tid / nitems, item = tid - item_rg * nitems;
    const bool active = item_rg < a.rg;
    const int half = 4 * a.nbk;
    int bs, bp, bq;
    const int item0 = CLUSTER ? (int)blockIdx.y * nitems : 0;
    m2s_item(CLUSTER ? (item0 + item < a.items_all ? item0 + item : 0) : item, a.nbk, a.dense != 0, bs, bp, bq);
    const int os = 4 * bs, op = 4 * bp, oq = bq < 0 ? op : 4 * bq;

    float accp[8][8], accq[8][8];                      // tiles {s,p} and {s,q}
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) accp[i][j] = accq[i][j] = 0.f;

    const int64_t n_begin = (int64_t)blockIdx.x * a.rows_per_slice;
    int64_t n_end = n_begin + a.rows_per_slice;
    if (n_end > a.N) n_end = a.N;

    uint64_t *full = reinterpret_cast<uint64_t *>(smem + a.bar_floats);      // one barrier per buffer
    volatile int *abort_flag = reinterpret_cast<volatile int *>(full + M2S_BUFFERS);
    if (tid == 0) {
        for (int b = 0; b < M2S_BUFFERS; ++b) tc::mbar_init(&full[b], 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
    }
    pdl_wait();
    pdl_trigger();
    if (tid == 0) {
        if (blockIdx.x == 0 && blockIdx.y == 0) {      // a time-out report can only be written 2^24 failed polls later
            a.status[kWsStatusWord] = 0;
            a.status[kWsDetailWord] = 0;
        }
    }
    __syncthreads();

    const int nstages = (n_end > n_begin) ? (int)((n_end - n_begin + stage_rows - 1) / stage_rows) : 0;
    const bool contiguous = (a.ldx == a.d);
    // Word copies: whole rows at a time by as many threads as make whole rows, so that a thread stays in its column and a copy takes
    // three instructions instead of fourteen ([50021,75] 21.4 us the call, now 19.2; [1000000,13] 38.2 and 30.3).
    const int copy_dr = nthreads >= a.d ? nthreads / a.d : 1;
    const int copy_r = tid / a.d, copy_c = tid - copy_r * a.d;
    // the rows of a stage arrive by bulk copies issued from warp 0: one copy when the rows are
    // contiguous in memory, one per row otherwise; rows past the end of the slice are not copied
    // and not read
    auto issue_stage = [&](int buf, int s) {
        if (BULK && tid >= 32) return;
        const int64_t n0 = n_begin + (int64_t)s * stage_rows;
        const int rows = (n_end - n0 < stage_rows) ? (int)(n_end - n0) : stage_rows;
        float *dst = smem + buf * stage_floats;
        if (!BULK) {
            if (copy_r >= copy_dr) return;
            for (int c = copy_c; c < a.d; c += nthreads) {                       // once, but for rows of more words than threads
                const float *src = a.X + (n0 + copy_r) * a.ldx + c;
                uint32_t to = tc::smem_u32(dst + copy_r * a.pitch + c);
                const int64_t src_step = copy_dr * a.ldx;
                const uint32_t to_step = (uint32_t)(copy_dr * a.pitch) * 4u;
#pragma unroll 4
                for (int r = copy_r; r < rows; r += copy_dr, src += src_step, to += to_step)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to), "l"(src));
            }
            return;
        }
        const uint32_t row_bytes = (uint32_t)a.d * 4u;
        if (tid == 0) tc::mbar_expect_tx(&full[buf], (uint32_t)rows * row_bytes);
        __syncwarp();
        if (contiguous) {
            if (tid == 0) m2s_bulk_load(dst, a.X + n0 * a.ldx, (uint32_t)rows * row_bytes, &full[buf]);
        } else {
            for (int r = tid; r < rows; r += 32) m2s_bulk_load(dst + r * a.d, a.X + (n0 + r) * a.ldx, row_bytes, &full[buf]);
        }
    };

    for (int s = 0; s < M2S_BUFFERS - 1; ++s) {
        if (s < nstages) issue_stage(s, s);
        if (!BULK) asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const int step = a.rg * a.pitch;
    int buf = 0;
    uint32_t parity = 0;
    for (int s = 0; s < nstages; ++s) {
        // a wait that gives up raises the abort flag; every thread still walks all stages so that
        // the block-wide barriers stay matched, and the host reads the status word afterwards
        if (BULK) (void)tc::mbar_wait(&full[buf], parity, abort_flag, a.status, 1);
        else asm volatile("cp.async.wait_group %0;" ::"n"(M2S_BUFFERS - 2) : "memory");
        __syncthreads();                                // stage s-1 is consumed: its buffer may be refilled
        if (s + M2S_BUFFERS - 1 < nstages) issue_stage(buf == 0 ? M2S_BUFFERS - 1 : buf - 1, s + M2S_BUFFERS - 1);
        if (!BULK) asm volatile("cp.async.commit_group;" ::: "memory");
        int qn = a.rpg;
        if (s == nstages - 1) {                         // last stage of the slice: only the rows that exist
            const int rows = (int)(n_end - n_begin - (int64_t)s * stage_rows);
            qn = (rows - item_rg + a.rg - 1) / a.rg;
            if (qn > a.rpg) qn = a.rpg;
        }
        if (active) {
            const float *row = smem + buf * stage_floats + item_rg * a.pitch;
#pragma unroll 2
            for (int q = 0; q < qn; ++q, row += step) {
                const float4 s0 = *reinterpret_cast<const float4 *>(row + os);
                const float4 s1 = *reinterpret_cast<const float4 *>(row + os + half);
                const float4 p0 = *reinterpret_cast<const float4 *>(row + op);
                const float4 p1 = *reinterpret_cast<const float4 *>(row + op + half);
                const float4 q0 = *reinterpret_cast<const float4 *>(row + oq);
                const float4 q1 = *reinterpret_cast<const float4 *>(row + oq + half);
                const float xs[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
                const float xp[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
                const float xq[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        accp[i][j] = fmaf(xs[i], xp[j], accp[i][j]);
                        accq[i][j] = fmaf(xs[i], xq[j], accq[i][j]);
                    }
            }
        }
        if (++buf == M2S_BUFFERS) {
            buf = 0;
            parity ^= 1u;
        }
    }
    if (BULK && *abort_flag && tid == 0) {
        // after a time-out: give the copies still in flight a bounded time to land before the
        // shared memory is reused or released
        for (int s = (nstages > M2S_BUFFERS ? nstages - M2S_BUFFERS : 0); s < nstages; ++s)
            for (uint32_t it = 0; it < tc::kSpinLimit; ++it)
                if (tc::mbar_try_wait(&full[s % M2S_BUFFERS], (uint32_t)((s / M2S_BUFFERS) & 1))) break;
    }
    __syncthreads();                                   // every thread is done with the stage buffers

    // block-level sum over the row groups, in group order (reproducible): the sums go to shared
    // memory as red[k][group][item] (k < 64 is tile {s,p}, k >= 64 tile {s,q}), output (k, item) is then
    // summed over the groups by `parts` threads, each over a fixed range, and by one thread over the parts.
    // The pitch of k is nitems modulo 32 words: consecutive threads, which own consecutive (k, item), then read
    // consecutive words (with one item and an unpadded pitch all 32 lanes of a warp met in one bank:
    // [10000,8] 21 us the call, now 6.6).
    float *red = smem;
    const int cells = m2s_red_pitch(a.rg, nitems);
    if (active) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                red[(i * 8 + j) * cells + tid] = accp[i][j];
                red[(64 + i * 8 + j) * cells + tid] = accq[i][j];
            }
    }
    __syncthreads();
    const int nout = 128 * nitems;
    int parts = nthreads / nout;
    if (parts < 1) parts = 1;
    if (parts > a.rg) parts = a.rg;
    float *mine = CLUSTER ? red + 128 * cells + M2S_MAX_THREADS : a.partials + (size_t)blockIdx.x * nout;
    if (parts == 1) {
        const int dk = nthreads / nitems, dt = nthreads - dk * nitems;     // (a division for each: [50021,75] 19.2 us, now 18.2)
        int k = tid / nitems, t = tid - k * nitems;
        for (int o = tid; o < nout; o += nthreads) {
            const float *p = red + k * cells + t;
            float sum = 0.f;
#pragma unroll 8
            for (int g = 0; g < a.rg; ++g) sum += p[g * nitems];
            mine[o] = sum;
            k += dk;
            t += dt;
            if (t >= nitems) { t -= nitems; ++k; }
        }
    } else {
        float *scratch = red + 128 * cells;            // [parts][nout]
        const int per = (a.rg + parts - 1) / parts;
        if (tid < parts * nout) {
            const int part = tid / nout, o = tid - part * nout;
            const int k = o / nitems, t = o - k * nitems;
            const float *p = red + k * cells + t;
            int g_end = (part + 1) * per;
            if (g_end > a.rg) g_end = a.rg;
            float sum = 0.f;
#pragma unroll 8
            for (int g = part * per; g < g_end; ++g) sum += p[g * nitems];
            scratch[part * nout + o] = sum;
        }
        __syncthreads();
        if (tid < nout) {
            float sum = 0.f;
            for (int part = 0; part < parts; ++part) sum += scratch[part * nout + tid];
            mine[tid] = sum;
        }
    }
    if (CLUSTER) {
        tc::cluster_sync_all();                        // all blocks' sums are written
        const int per = (nout + M2S_CLUSTER - 1) / M2S_CLUSTER, o_end = nout < ((int)blockIdx.x + 1) * per ? nout : ((int)blockIdx.x + 1) * per;
        for (int o = (int)blockIdx.x * per + tid; o < o_end; o += nthreads) {
            const int k = o / nitems, t = item0 + o - k * nitems;
            int64_t at;
            if (t >= a.items_all || !m2s_output(k, t, a.nbk, a.dense != 0, a.d, at)) continue;
            float v[M2S_CLUSTER], sum = 0.f;
#pragma unroll
            for (int r = 0; r < M2S_CLUSTER; ++r)
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v[r]) : "r"(tc::map_to_cta(tc::smem_u32(mine + o), (uint32_t)r)));
#pragma unroll
            for (int r = 0; r < M2S_CLUSTER; ++r) sum += v[r];
            if (ST_BOUNDS_OK(at, tri_rows(a.d), 2)) a.out[at] = sum;
        }
        tc::cluster_sync_all();                        // no block leaves while its sums are read
    }
}

// out[p(ci,cj)] = sum over the slices of element (k, item) of the partials: a block owns 32 V elements, V of them a lane, warp w of W
// adds the slices w, w + W, ..., five loads at a time, then the W sums are added in order (a fixed order).  Latency and
// placement bound it: twenty loads at a time take registers that the running kernel does not leave ([20000,64] 10.8 us the call,
// with seven 9.9); with eight warps whatever the slices, seven loads at a time, [50021,75] 18.2 us, now 17.6, [30000,120] 22.5 and
// 20.6, [50000,150] 62 and 49.
// M2S_SUM_V4: work items from where V = 4.  us in rows of calls, V = 1 / 4: 5 items [50021,32] 7.8 / 8.1, [20000,32] 6.7 / 6.9; 8 items
// [20000,40] 6.8 / 7.0, [50021,40] 8.2 / 8.2; 11 items [20000,48] 8.2 / 8.0, [300000,48] 26.2 / 26.0; 18 items [50021,64] 12.5 / 12.3, [300000,64]
// 35.1 / 34.8; 28 items [300000,80] 50.5 / 50.2.
constexpr int M2S_SUM_BATCH = 5, M2S_SUM_V4 = 10;
template <int V, int W>
__global__ void __launch_bounds__(32 * W)
moment2_small_reduce_kernel(const float *partials, float *out, int d, int nbk, int slices,
                            int dense, int nitems)
{
    __shared__ float part[W][32 * V];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int o0 = blockIdx.x * 32 * V;                // < nitems * 128, a multiple of 32 V
    int64_t at = -1;
    bool use = false;
    if (threadIdx.x < 32 * V) {
        const int o = o0 + (int)threadIdx.x, k = o / nitems, item = o - k * nitems;
        use = m2s_output(k, item, nbk, dense != 0, d, at);
    }
    pdl_wait();
    pdl_trigger();
    const size_t stride = (size_t)nitems * 128;
    float s[V] = {};
    const float *p = partials + o0 + lane * V;
    for (int k0 = warp; k0 < slices; k0 += W * M2S_SUM_BATCH) {
        float v[M2S_SUM_BATCH][V] = {};
#pragma unroll
        for (int u = 0; u < M2S_SUM_BATCH; ++u) {
            if (k0 + W * u >= slices) continue;
            const float *q = p + (size_t)(k0 + W * u) * stride;
            if constexpr (V == 4) {
                const float4 x = __ldcg(reinterpret_cast<const float4 *>(q));
                v[u][0] = x.x; v[u][1] = x.y; v[u][2] = x.z; v[u][3] = x.w;
            } else {
                v[u][0] = __ldcg(q);
            }
        }
#pragma unroll
        for (int u = 0; u < M2S_SUM_BATCH; ++u)
#pragma unroll
            for (int x = 0; x < V; ++x) s[x] += v[u][x];
    }
#pragma unroll
    for (int x = 0; x < V; ++x) part[warp][lane * V + x] = s[x];
    __syncthreads();
    if (!use) return;
    float sum = part[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < W; ++w) sum += part[w][threadIdx.x];
    if (ST_BOUNDS_OK(at, tri_rows(d), 2)) out[at] = sum;
}

struct M2SmallPlan {
    int nbk, pitch, nitems, rg, rpg, threads, slices;
    int64_t rows_per_slice;
    size_t smem, data_bytes, partial_bytes;
};

// FMA slots that the kernel occupies per sample row (idle threads included); 0 when it does not cover d.
int64_t moment2_small_slots(int64_t d, unsigned flags)
{
    const int64_t nbk = (d + 7) / 8;
    if (nbk > M2S_MAX_BLOCKS) return 0;
    const int n = m2s_nitems((int)nbk, (flags & ST_FLAG_DENSE_CONTROL) != 0);
    if (n > M2S_MAX_THREADS) return 0;
    return 128 * M2S_MAX_THREADS / (M2S_MAX_THREADS / n);
}

// Work items.
int64_t moment2_small_items(int64_t d, unsigned flags) { return m2s_nitems((int)((d + 7) / 8), (flags & ST_FLAG_DENSE_CONTROL) != 0); }

static M2SmallPlan moment2_small_plan(int64_t N, int64_t d, unsigned flags)
{
    M2SmallPlan p;
    p.nbk = (int)(d + 7) / 8;
    const int nitems = p.nitems = m2s_nitems(p.nbk, (flags & ST_FLAG_DENSE_CONTROL) != 0);
    p.pitch = (int)(d + 3) / 4 * 4;
    const int max_stage_rows = M2S_STAGE_BYTES / (4 * p.pitch);
    p.rg = M2S_MAX_THREADS / nitems;
    if (p.rg > max_stage_rows / 8) p.rg = max_stage_rows / 8;
    if (p.rg < 1) p.rg = 1;
    p.threads = (nitems * p.rg + 31) / 32 * 32;
    p.rpg = 8;
    int64_t slices = sm_count_or_default();
    // few samples: shorter slices fill more SMs (four rows per thread and stage: [4096,64] 9.4 us, eight 10.2, two 14.1)
    while (p.rpg > 4 && N <= slices * p.rg * p.rpg / 2) p.rpg /= 2;
    const int64_t max_slices = (N + p.rg * p.rpg - 1) / (p.rg * p.rpg);
    if (slices > max_slices) slices = max_slices;
    p.rows_per_slice = (N + slices - 1) / slices;
    p.slices = (int)((N + p.rows_per_slice - 1) / p.rows_per_slice);
    // long slices: 16 rows per thread and stage halve the number of block-wide barriers
    if (p.rg * 16 <= max_stage_rows && p.rows_per_slice >= 4 * p.rg * 16) p.rpg = 16;
    const size_t cells = (size_t)m2s_red_pitch(p.rg, nitems);
    const size_t main_bytes = (size_t)M2S_BUFFERS * p.rg * p.rpg * p.pitch * sizeof(float) + 32;   // the last row is read past its end
    const size_t sum_bytes = (128 * cells + (size_t)M2S_MAX_THREADS) * sizeof(float);
    p.data_bytes = round_up(main_bytes > sum_bytes ? main_bytes : sum_bytes, 16);
    p.smem = p.data_bytes + 64;                        // barriers and the abort flag behind the data
    p.partial_bytes = (size_t)p.slices * nitems * 128 * sizeof(float);
    return p;
}

// Plan of the one-launch form: clusters of blocks over the items, blocks over the samples.
static M2SmallPlan moment2_cluster_plan(int64_t N, int64_t d, unsigned flags, int &clusters)
{
    M2SmallPlan p;
    p.nbk = (int)(d + 7) / 8;
    const int all = m2s_nitems(p.nbk, (flags & ST_FLAG_DENSE_CONTROL) != 0);
    clusters = (all + M2S_CLUSTER_ITEMS - 1) / M2S_CLUSTER_ITEMS;
    p.nitems = (all + clusters - 1) / clusters;
    clusters = (all + p.nitems - 1) / p.nitems;
    p.pitch = (int)(d + 3) / 4 * 4;
    const int max_stage_rows = M2S_STAGE_BYTES / (4 * p.pitch);
    p.rg = M2S_CLUSTER_THREADS / p.nitems;
    if (p.rg > max_stage_rows / 8) p.rg = max_stage_rows / 8;
    p.threads = (p.nitems * p.rg + 31) / 32 * 32;
    p.slices = M2S_CLUSTER;
    p.rows_per_slice = (N + M2S_CLUSTER - 1) / M2S_CLUSTER;
    p.rpg = p.rows_per_slice >= 16 * p.rg ? 8 : 4;
    const size_t cells = (size_t)m2s_red_pitch(p.rg, p.nitems);
    const size_t main_bytes = (size_t)M2S_BUFFERS * p.rg * p.rpg * p.pitch * sizeof(float) + 32;
    const size_t sum_bytes = (128 * cells + (size_t)M2S_MAX_THREADS + 128 * (size_t)p.nitems) * sizeof(float);
    p.data_bytes = round_up(main_bytes > sum_bytes ? main_bytes : sum_bytes, 16);
    p.smem = p.data_bytes + 64;
    p.partial_bytes = 0;
    return p;
}

size_t moment2_small_workspace(int64_t N, int64_t d, unsigned flags)
{
    return kWsHeaderBytes + moment2_small_plan(N, d, flags).partial_bytes;
}

template <class Kernel>
static cudaLaunchConfig_t m2s_cluster_config(const M2SmallPlan &p, int clusters, cudaStream_t stream, cudaLaunchAttribute (&attr)[2])
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(M2S_CLUSTER, (unsigned)clusters);
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = M2S_CLUSTER;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

// Clusters of a plan that can be active at once on the current device, asked once per shape of the launch.
template <class Kernel>
static int m2s_fitting_clusters(Kernel kernel, const M2SmallPlan &p, int clusters)
{
    static std::mutex lock;
    static std::map<std::tuple<const void *, int, int, size_t>, int> known;
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    const auto key = std::make_tuple((const void *)kernel, dev, p.threads, p.smem);
    {
        std::lock_guard<std::mutex> guard(lock);
        const auto it = known.find(key);
        if (it != known.end()) return it->second;
    }
    if (ensure_dynamic_smem(kernel, p.smem) && allow_large_clusters(kernel)) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = m2s_cluster_config<Kernel>(p, clusters, nullptr, attr);
        if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
    }
    std::lock_guard<std::mutex> guard(lock);
    return known[key] = n;
}

st_status moment2_small(const float *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes,
                        unsigned flags, cudaStream_t stream)
{
    const bool bulk = d % 4 == 0 && ldx % 4 == 0;
    if (!ws || ws_bytes < kWsHeaderBytes) return ST_ERR_WORKSPACE;
    if (!aligned256(ws)) return ST_ERR_ALIGN;
    M2SmallArgs a;
    auto fill = [&](const M2SmallPlan &p) {
        a.X = X;
        a.partials = (float *)((unsigned char *)ws + kWsHeaderBytes);
        a.N = N; a.ldx = ldx; a.rows_per_slice = p.rows_per_slice;
        a.d = (int)d; a.pitch = p.pitch; a.nbk = p.nbk; a.rg = p.rg; a.rpg = p.rpg;
        a.nitems = p.nitems;
        a.status = (unsigned *)ws;
        a.bar_floats = (int)(p.data_bytes / sizeof(float));
        a.dense = (flags & ST_FLAG_DENSE_CONTROL) ? 1 : 0;
    };
    {
        int clusters = 0;
        const M2SmallPlan p = moment2_cluster_plan(N, d, flags, clusters);
        const int items = (int)moment2_small_items(d, flags);
        auto run = [&](auto kernel) {
            // (a first look without the device, so that calls that are far from it do not ask)
            if (!m2s_use_cluster(N, items, clusters, p.rg, bulk, clusters) ||
                !m2s_use_cluster(N, items, clusters, p.rg, bulk, m2s_fitting_clusters(kernel, p, clusters)))
                return false;
            fill(p);
            a.out = out;
            a.items_all = items;
            cudaLaunchAttribute attr[2];
            cudaLaunchConfig_t cfg = m2s_cluster_config<decltype(kernel)>(p, clusters, stream, attr);
            if (cudaLaunchKernelEx(&cfg, kernel, a) == cudaSuccess) return true;
            (void)cudaGetLastError();                  // a context with fewer SMs than the one that was asked: two launches
            return false;
        };
        if (bulk ? run(moment2_small_kernel<true, true>) : run(moment2_small_kernel<false, true>)) return ST_OK;
    }
    const M2SmallPlan p = moment2_small_plan(N, d, flags);
    if (ws_bytes < kWsHeaderBytes + p.partial_bytes) return ST_ERR_WORKSPACE;
    fill(p);
    auto run = [&](auto kernel) {
        if (!ensure_dynamic_smem(kernel, p.smem)) return ST_ERR_CUDA;
        return launch(kernel, p.slices, p.threads, p.smem, stream, a);
    };
    const st_status rc = bulk ? run(moment2_small_kernel<true, false>) : run(moment2_small_kernel<false, false>);
    if (rc != ST_OK) return rc;
    auto sum = [&](auto v, auto w) {
        constexpr int V = decltype(v)::value, W = decltype(w)::value;
        return launch(moment2_small_reduce_kernel<V, W>, (unsigned)(p.nitems * 4 / V), 32u * W, 0, stream, a.partials, out, (int)d, p.nbk, p.slices, a.dense,
                      p.nitems);
    };
    auto with_warps = [&](auto v) {
        return p.slices <= 8 * M2S_SUM_BATCH ? sum(v, std::integral_constant<int, 8>{})
             : p.slices <= 16 * M2S_SUM_BATCH ? sum(v, std::integral_constant<int, 16>{}) : sum(v, std::integral_constant<int, 32>{});
    };
    return p.nitems >= M2S_SUM_V4 ? with_warps(std::integral_constant<int, 4>{}) : with_warps(std::integral_constant<int, 1>{});
}

}  // namespace st
