// st_sym_moment2, fp32 FMA path: out[p(i,j)] = sum_n X[n,i] X[n,j] over the unique set
// 0<=i<=j<d of the symmetric output (Section 3, M1; Section 5.5, y_U = 0<=i<=j<n).
//
// Two main kernels, each followed by a sum of its partial results in a fixed order (deterministic result):
// the register-tile kernel of moment2_small.cu for few features, and moment2_gemm_kernel below, which cuts the
// upper triangle into 128x128 tiles and skips the 64x64 quadrants that lie below the diagonal or past d.
// Either takes any d and any row pitch.  Many samples of more features, in rows that start on 16-byte boundaries, go to
// the tensor cores instead, at the error of fp32 arithmetic (moment2_exact.cuh).
#include "st_common.cuh"
#include "st_index.cuh"
#include <type_traits>

namespace st {

st_status moment2_bf16_tc(const void *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws,
                          size_t ws_bytes, unsigned flags, cudaStream_t stream);
size_t moment2_bf16_tc_workspace(int64_t N, int64_t d, unsigned flags);
st_status moment2_tf32_tc(const void *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws,
                          size_t ws_bytes, unsigned flags, cudaStream_t stream);
size_t moment2_tf32_tc_workspace(int64_t N, int64_t d, unsigned flags);
st_status moment2_split_tc(const float *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes,
                           unsigned flags, cudaStream_t stream);
size_t moment2_split_tc_workspace(int64_t N, int64_t d, unsigned flags);
st_status moment2_exact_tc(const float *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes,
                           unsigned flags, cudaStream_t stream);
size_t moment2_exact_tc_workspace(int64_t N, int64_t d, unsigned flags);
int64_t moment2_small_slots(int64_t d, unsigned flags);
int64_t moment2_small_items(int64_t d, unsigned flags);
size_t moment2_small_workspace(int64_t N, int64_t d, unsigned flags);
st_status moment2_small(const float *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes,
                        unsigned flags, cudaStream_t stream);

// ---- 128 x 128 tiles ----------------------------------------------------------------------
constexpr int MG_T = 128;       // output tile edge
constexpr int MG_KC = 8;        // sample rows per stage; the loop over them is fully unrolled
constexpr int MG_STAGES = 4;
constexpr int MG_THREADS = 128;
constexpr size_t MG_SMEM = (size_t)MG_STAGES * 2 * MG_KC * MG_T * sizeof(float);   // 32 KiB
// One block per SM, where all blocks find one: behind another kernel they were placed two to an SM and left others idle
// ([500,640] 18.8 us, now 13.3; [2000,256] 17.4 and 12.7).
constexpr size_t MG_SMEM_ALONE = 120 * 1024;

// What a tile computes of its four 64x64 quadrants.
enum { MG_FULL = 0,             // all four
       MG_DIAG = 1,             // diagonal tile: not the one below the diagonal
       MG_LEFT = 2,             // last tile column, at most 64 columns left: the left two
       MG_QUAD = 3 };           // last diagonal tile, at most 64 rows and columns left: the first one

// Time of a tile of each kind per sample row, full tile = 1 (a diagonal tile saves FMAs but no loads; weights in
// proportion to the FMAs, 0.75 / 0.5 / 0.25, run [60000,257] in 251 us instead of 229 and [65536,512] in 381 instead of 374).
constexpr double MG_COST[4] = {1.0, 0.8, 0.6, 0.4};

// Tiles are numbered kind by kind, blocks (tile, sample split) likewise and within a kind split by split, so that the
// blocks of one range of samples are neighbours and share its rows through L2.
struct MgGrid {
    int nt;              // tiles per edge
    int full;            // edge of the triangle of full and diagonal tiles (nt, or nt - 1 when the last tile column is half empty)
    int n[4];            // tiles of each kind
    int split[4];        // sample splits of each of its tiles
    int first[5];        // first block of each kind, and the number of blocks
    int64_t rows[4];     // samples per split
};

// Tile number t of its kind -> tile row and column.
template <bool DENSE>
__device__ __forceinline__ void mg_tile(const MgGrid &g, int kind, int t, int &bi, int &bj)
{
    if (DENSE) {
        bi = t / g.nt;
        bj = t - bi * g.nt;
    } else if (kind == MG_FULL) {
        int64_t a, b;
        tri_decode(g.full - 1, t, a, b);
        bi = (int)a;
        bj = (int)b + 1;
    } else {
        bi = kind == MG_QUAD ? g.nt - 1 : t;
        bj = kind == MG_DIAG ? t : g.nt - 1;
    }
}

// Tiles of each kind; returns the edge of the triangle of full and diagonal ones.
static int mg_kinds(int64_t nt, int64_t d, bool dense, int n[4])
{
    const int full = (int)(d - (nt - 1) * MG_T <= 64 ? nt - 1 : nt);
    n[MG_FULL] = dense ? (int)(nt * nt) : full * (full - 1) / 2;
    n[MG_DIAG] = dense ? 0 : full;
    n[MG_LEFT] = !dense && full < nt ? (int)nt - 1 : 0;
    n[MG_QUAD] = !dense && full < nt ? 1 : 0;
    return full;
}

// 64x64 quadrants computed per sample row.
static int64_t moment2_gemm_quads(int64_t d, bool dense)
{
    const int64_t nt = (d + MG_T - 1) / MG_T;
    if (dense) return 4 * nt * nt;
    const int64_t q = 2 * nt * nt + nt;                                // 4 nt(nt-1)/2 off the diagonal, 3 nt on it
    return (d - (nt - 1) * MG_T <= 64) ? q - 2 * (nt - 1) - 2 : q;
}

static size_t mg_partial_bytes(const MgGrid &g) { return (size_t)g.first[4] * MG_T * MG_T * sizeof(float); }

static MgGrid moment2_gemm_plan(int64_t N, int64_t d, unsigned flags)
{
    MgGrid g;
    g.nt = (int)((d + MG_T - 1) / MG_T);
    g.full = mg_kinds(g.nt, d, (flags & ST_FLAG_DENSE_CONTROL) != 0, g.n);
    // Two thread blocks fit on an SM.  The splits of a full tile (w) are the number whose blocks fill whole waves of
    // 2 x SMs best, the smallest such number within 3 %; cheaper tiles get fewer splits in proportion, so that all
    // blocks take about as long.
    const int64_t slots = 2 * (int64_t)sm_count_or_default();
    const int64_t most = (N + 8 * MG_KC - 1) / (8 * MG_KC);            // at least eight stages of rows per split
    double best = 1e30;
    for (int64_t w = 1; w <= 2 * slots; ++w) {
        int64_t s[4], blocks = 0;
        double longest = 0;
        for (int k = 0; k < 4; ++k) {
            s[k] = (int64_t)(MG_COST[k] * (double)w + 0.5);
            s[k] = s[k] < 1 ? 1 : s[k] > most ? most : s[k];
            blocks += g.n[k] * s[k];
            if (g.n[k] > 0 && MG_COST[k] / (double)s[k] > longest) longest = MG_COST[k] / (double)s[k];
        }
        if (w > 1 && blocks > 2 * slots) break;
        const double t = (double)((blocks + slots - 1) / slots) * longest;
        if (t < best * 0.97) {
            best = t;
            for (int k = 0; k < 4; ++k) g.split[k] = (int)s[k];
        }
    }
    g.first[0] = 0;
    for (int k = 0; k < 4; ++k) {
        const int64_t rows = (N + g.split[k] - 1) / g.split[k];
        g.rows[k] = (rows + MG_KC - 1) / MG_KC * MG_KC;
        g.split[k] = (int)((N + g.rows[k] - 1) / g.rows[k]);
        g.first[k + 1] = g.first[k] + g.n[k] * g.split[k];
    }
    return g;
}

// Blocks of the sum per SM together: with 128 for every tile, half of which had nothing to do, [64,4096] took 163 us, now 70.
constexpr int MG_SUM_BLOCKS = 16;
__host__ __device__ inline int mg_sum_warps(int nsplit) { return nsplit <= 8 ? 1 : nsplit <= 16 ? 2 : nsplit <= 32 ? 4 : 8; }   // about eight loads per thread

// out[p(i,j)] = sum over the sample splits of a tile of 128 x 128 partial sums; i <= j only.  `wps` warps share 32
// columns of a row: the first adds the splits 0, wps, 2 wps, ... with its loads in flight, and so on, then the sums are
// added in order (a fixed order).  After the other kernels of a pipeline have streamed gigabytes, every dependent round
// trip to memory costs microseconds.
template <bool DENSE>
__global__ void __launch_bounds__(256)
moment2_gemm_reduce_kernel(const float *partials, float *out, int d, const MgGrid g)
{
    constexpr int T = MG_T;
    constexpr int BATCH = 4;                             // eight take registers that the running kernel does not leave: [20000,256] 54 us, now 47
    __shared__ float part[2][8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int kind = 0, t = blockIdx.x, bi, bj;
    while (kind < 3 && t >= g.n[kind]) t -= g.n[kind++];
    mg_tile<DENSE>(g, kind, t, bi, bj);
    const int nsplit = g.split[kind];
    const float *base = partials + (size_t)(g.first[kind] + t) * (T * T);
    const size_t stride = (size_t)g.n[kind] * (T * T);
    const int wps = mg_sum_warps(nsplit);
    pdl_wait();
    pdl_trigger();
    if (bi > bj) return;                                 // dense control: lower tiles are discarded
    int buf = 0;
    const int per = 8 / wps, first = warp % wps;
    for (int u0 = blockIdx.y * per; u0 < T * T / 32; u0 += gridDim.y * per) {
        const int u = u0 + warp / wps;
        const int r = u / (T / 32), c = (u % (T / 32)) * 32 + lane;
        const int gi = bi * T + r, gj = bj * T + c;
        float s = 0.f;
        const float *p1 = base + r * T + c;
        const bool use = gj < d && gi <= gj;
        for (int k0 = first; k0 < nsplit; k0 += BATCH * wps) {
            float v[BATCH];
#pragma unroll
            for (int e = 0; e < BATCH; ++e) v[e] = (use && k0 + wps * e < nsplit) ? __ldcg(p1 + (size_t)(k0 + wps * e) * stride) : 0.f;
#pragma unroll
            for (int e = 0; e < BATCH; ++e) s += v[e];
        }
        part[buf][warp][lane] = s;
        if (wps > 1) __syncthreads();
        if (first == 0 && use) {
            for (int w = 1; w < wps; ++w) s += part[buf][warp + w][lane];
            if (ST_BOUNDS_OK(tri_encode(d, gi, gj), tri_rows(d), 2)) out[tri_encode(d, gi, gj)] = s;
        }
        buf ^= 1;
    }
}

__device__ __forceinline__ uint64_t mg_pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ uint64_t mg_ffma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// fp32 FMA bound.  Shared memory returns 32 words per cycle to the registers against 128 FMA lanes, so a thread
// that owns 8 x 8 sums (16 words per 64 FMAs) saturates both at once; here it owns 8 x 16 (24 words per 128 FMAs,
// three quarters of that limit) with packed FMAs, which leave half of the issue slots for the loads and moves.
// The eight rows of a stage are fully unrolled: in an inner-kernel probe at [65536,512] stages of 16 rows unrolled
// by 4 ran 412 us where these run 364 (59 against 52 TFLOP/s issued).  Whole call: 374 us (46 TFLOP/s useful); 8 x 8
// tiles with the same number of splits for every tile ran 497.
// Thread (ty, tx) of the 16 x 8 thread grid: rows 4ty..4ty+3 of either half (h), columns 32q+4tx.. of each
// quarter q.  VEC: rows of X are 16-byte aligned; otherwise they are copied word by word (16 more instructions
// per stage and thread beside 512 packed FMAs).
template <bool DENSE, bool VEC>
__global__ void __launch_bounds__(MG_THREADS, 2)
moment2_gemm_kernel(const float *X, int64_t N, int d, int64_t ldx, float *partials, const MgGrid g,
                    unsigned *status)
{
    extern __shared__ __align__(16) float smem[];     // MG_STAGES x { As[MG_KC][MG_T], Bs[MG_KC][MG_T] }
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x == 0 && threadIdx.x == 0) {        // no bounded waits here: the status is "ok"
        status[kWsStatusWord] = 0;
        status[kWsDetailWord] = 0;
    }
    int kind = 0, bi, bj;
    while (kind < 3 && (int)blockIdx.x >= g.first[kind + 1]) ++kind;
    const int in_kind = (int)blockIdx.x - g.first[kind], split = in_kind / g.n[kind];
    mg_tile<DENSE>(g, kind, in_kind - split * g.n[kind], bi, bj);
    const bool diag = (bi == bj);
    const int tid = threadIdx.x, ty = tid >> 3, tx = tid & 7;
    const int col_a = bi * MG_T, col_b = bj * MG_T;
    const int64_t n_begin = (int64_t)split * g.rows[kind];
    int64_t n_end = n_begin + g.rows[kind];
    if (n_end > N) n_end = N;
    const int nstages = n_end > n_begin ? (int)((n_end - n_begin + MG_KC - 1) / MG_KC) : 0;

    uint64_t acc[8][8];                          // [4h + r][2q + e]: columns 32q + 4tx + 2e, + 1
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;

    // a stage: MG_KC rows of the two column panels (one panel on the diagonal), zero-filled past N and past d
    constexpr int W = VEC ? 4 : 1;               // words per copy
    constexpr int PER_PANEL = MG_KC * (MG_T / W);
    auto load_stage = [&](int s) {
        if (s < nstages) {
            float *st_base = smem + (size_t)(s % MG_STAGES) * (2 * MG_KC * MG_T);
            const int64_t n0 = n_begin + (int64_t)s * MG_KC;
            auto panel = [&](float *dst0, int col0) {
#pragma unroll
                for (int u = 0; u < PER_PANEL / MG_THREADS; ++u) {
                    const int c = tid + u * MG_THREADS, r = c / (MG_T / W), q = c % (MG_T / W);
                    const int col = col0 + W * q;
                    const int64_t n = n0 + r;
                    const bool in = n < n_end && col < d;
                    const unsigned dst = (unsigned)__cvta_generic_to_shared(dst0 + r * MG_T + W * q);
                    const float *src = in ? X + n * ldx + col : X;
                    const int sz = in ? 4 * W : 0;
                    if (VEC) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz));
                    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(sz));
                }
            };
            panel(st_base + MG_KC * MG_T, col_b);
            if (!diag) panel(st_base, col_a);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int s = 0; s < MG_STAGES - 1; ++s) load_stage(s);
    auto run = [&](auto part_tag) {              // an instance of the loop per kind of tile: what it skips is a compile-time fact
        constexpr int PART = decltype(part_tag)::value;
        constexpr int NH = PART == MG_QUAD ? 1 : 2, NQ = (PART == MG_LEFT || PART == MG_QUAD) ? 2 : 4;
        for (int s = 0; s < nstages; ++s) {
            asm volatile("cp.async.wait_group %0;" ::"n"(MG_STAGES - 2) : "memory");
            __syncthreads();                     // stage s has landed; the buffer of stage s-1 is free
            load_stage(s + MG_STAGES - 1);
            const float *Bs = smem + (size_t)(s % MG_STAGES) * (2 * MG_KC * MG_T) + MG_KC * MG_T;
            const float *As = diag ? Bs : Bs - MG_KC * MG_T;
#pragma unroll
            for (int k = 0; k < MG_KC; ++k) {
                ulonglong2 b[NQ];
#pragma unroll
                for (int q = 0; q < NQ; ++q) b[q] = *reinterpret_cast<const ulonglong2 *>(Bs + k * MG_T + 32 * q + 4 * tx);
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    const float4 a = *reinterpret_cast<const float4 *>(As + k * MG_T + 64 * h + 4 * ty);
                    const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const uint64_t aa = mg_pack2(av[r], av[r]);
#pragma unroll
                        for (int q = 0; q < NQ; ++q) {
                            if (PART == MG_DIAG && h == 1 && q < 2) continue;
                            acc[4 * h + r][2 * q] = mg_ffma2(aa, b[q].x, acc[4 * h + r][2 * q]);
                            acc[4 * h + r][2 * q + 1] = mg_ffma2(aa, b[q].y, acc[4 * h + r][2 * q + 1]);
                        }
                    }
                }
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        // what was not computed is not stored: the reduction reads i <= j < d only
        float *mine = partials + (size_t)blockIdx.x * (MG_T * MG_T);
#pragma unroll
        for (int i = 0; i < 4 * NH; ++i)
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                if (PART == MG_DIAG && i >= 4 && q < 2) continue;
                ulonglong2 v;
                v.x = acc[i][2 * q];
                v.y = acc[i][2 * q + 1];
                *reinterpret_cast<ulonglong2 *>(&mine[(64 * (i >> 2) + 4 * ty + (i & 3)) * MG_T + 32 * q + 4 * tx]) = v;
            }
    };
    if (DENSE || kind == MG_FULL) run(std::integral_constant<int, MG_FULL>{});
    else if (kind == MG_DIAG) run(std::integral_constant<int, MG_DIAG>{});
    else if (kind == MG_LEFT) run(std::integral_constant<int, MG_LEFT>{});
    else run(std::integral_constant<int, MG_QUAD>{});
}

static st_status moment2_gemm(const float *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws, size_t ws_bytes,
                              unsigned flags, cudaStream_t stream)
{
    const MgGrid g = moment2_gemm_plan(N, d, flags);
    if (!ws || ws_bytes < kWsHeaderBytes + mg_partial_bytes(g)) return ST_ERR_WORKSPACE;
    if (!aligned256(ws)) return ST_ERR_ALIGN;
    float *partials = (float *)((unsigned char *)ws + kWsHeaderBytes);
    const bool dense = (flags & ST_FLAG_DENSE_CONTROL) != 0, vec = d % 4 == 0 && ldx % 4 == 0;
    const size_t smem = g.first[4] <= sm_count_or_default() ? MG_SMEM_ALONE : MG_SMEM;
    auto run = [&](auto kernel) {
        if (!ensure_dynamic_smem(kernel, smem)) return ST_ERR_CUDA;
        return launch(kernel, g.first[4], MG_THREADS, smem, stream, X, N, (int)d, ldx, partials, g, (unsigned *)ws);
    };
    const st_status rc = dense ? (vec ? run(moment2_gemm_kernel<true, true>) : run(moment2_gemm_kernel<true, false>))
                               : (vec ? run(moment2_gemm_kernel<false, true>) : run(moment2_gemm_kernel<false, false>));
    if (rc != ST_OK) return rc;
    // blocks for all rows of a tile, but not more than MG_SUM_BLOCKS per SM together
    const int tiles = g.n[0] + g.n[1] + g.n[2] + g.n[3];
    int most = 0;
    for (int k = 0; k < 4; ++k)
        if (g.n[k] > 0 && g.split[k] > most) most = g.split[k];
    int blocks = MG_T * MG_T / 32 / 8 * mg_sum_warps(most);
    const int cap = MG_SUM_BLOCKS * sm_count_or_default() / tiles;
    if (blocks > cap) blocks = cap < 8 ? 8 : cap;
    return launch(dense ? moment2_gemm_reduce_kernel<true> : moment2_gemm_reduce_kernel<false>, dim3(tiles, blocks), 256, 0, stream, partials, out,
                  (int)d, g);
}

// Which of the two kernels.  Many samples: the one with fewer FMA slots per sample row, each divided by the fraction of the FMA
// peak that it reaches with those slots (register tiles 0.60: [1048576,64] 107 us; 128 x 128 tiles 0.75).
// Few samples of more than 128 features: the register tiles write and add a partial result per SM, which takes as long as about
// 70 samples of a full 128 x 128 tile per work item; the samples have to make up for that by what they save (15400 slots take as
// long as a full tile).  Register tiles / 128 x 128 tiles, us: [4096,129] 17.0 / 14.9, [6000,129] 18.2 / 21.0,
// [2000,160] 18.2 / 10.8, [16384,160] 28.3 / 26.6, [30000,160] 36.1 / 41.4, [64,248] 24.5 / 10, [4096,248] 33.0 / 20.1,
// [30000,248] 65.7 / 56.4, [200000,248] 284 / 318.
static bool moment2_use_small(int64_t N, int64_t d, unsigned flags)
{
    const bool dense = (flags & ST_FLAG_DENSE_CONTROL) != 0;
    const int64_t slots = moment2_small_slots(d, flags);
    if (slots == 0) return false;
    if (d > 128) {
        int n[4];
        mg_kinds((d + MG_T - 1) / MG_T, d, dense, n);
        double tiles = 0;
        for (int k = 0; k < 4; ++k) tiles += MG_COST[k] * n[k];
        if ((double)N * (tiles - (double)slots / 15400) < 70.0 * (double)moment2_small_items(d, flags)) return false;
    }
    return (double)slots / 0.60 <= (double)(moment2_gemm_quads(d, dense) * 4096) / 0.75;
}

// Tensor cores with the exact parts of x (moment2_exact.cuh): from where they are faster than the FMA kernels.  Other feature
// counts than multiples of four have rows that a tensor map can name in a padded table only, and stay with the FMA kernels.
// FMA / tensor cores, us (the main kernel and the sums after it): [12000,128] 17.1 / 17.3, [16384,128] 20.4 / 19.1, [200000,128] 106 / 92, [4096,192] 12.6 / 15.8,
// [6000,192] 18.0 / 16.5, [4096,200] 20.6 / 15.9, [2000,260] 14.6 / 14.7, [3000,260] 22.1 / 15.5, [1000,512] 15.0 / 16.8,
// [1500,512] 23.3 / 17.0, [65536,512] 370 / 122, [300,768] 14.6 / 16.5, [600,768] 22.6 / 17.3, [4096,2048] 374 / 104.  Up to 120
// features the register tiles are the better ones ([200000,120] 78 / 92), and those of 129 to 136 are no worse ([65536,136] 43 / 43).
// [4096,192] and [3000,260] are as many values on different sides of the line: it lies above both.
static bool moment2_use_exact(int64_t N, int64_t d)
{
    if (d % 4 != 0 || d <= 120 || (d > 128 && d <= 136) || d > 4096 || N > (int64_t(1) << 31) - 64) return false;
    const double values = (double)N * (double)d;
    return values * (double)d >= 2.7e8 || (d > 136 && values >= 8e5);
}

static st_status moment2_f32(const float *X, int64_t N, int64_t d, int64_t ldx, float *out, void *ws,
                             size_t ws_bytes, unsigned flags, cudaStream_t stream)
{
    if (d > 32768) return ST_ERR_UNSUPPORTED;
    if (ldx % 4 == 0 && moment2_use_exact(N, d)) {
        // the FMA kernels take what this route does not: more tiles than its plan holds (dense control of more than 3072
        // features), a build of its kernel with too few registers, a workspace that is large enough for them alone
        const st_status rc = moment2_exact_tc(X, N, d, ldx, out, ws, ws_bytes, flags, stream);
        if (rc != ST_ERR_UNSUPPORTED && rc != ST_ERR_WORKSPACE) return rc;
    }
    return moment2_use_small(N, d, flags) ? moment2_small(X, N, d, ldx, out, ws, ws_bytes, flags, stream)
                                       : moment2_gemm(X, N, d, ldx, out, ws, ws_bytes, flags, stream);
}

size_t moment2_workspace(int64_t N, int64_t d, int xdt, unsigned flags)
{
    if (N <= 0 || d <= 0) return 0;
    const unsigned tc = flags & (ST_FLAG_TC_TF32 | ST_FLAG_TC_SPLIT);
    if (tc == (ST_FLAG_TC_TF32 | ST_FLAG_TC_SPLIT)) return 0;
    if (xdt == ST_BF16) return tc ? 0 : moment2_bf16_tc_workspace(N, d, flags);
    if (xdt == ST_F32 && (flags & ST_FLAG_TC_TF32)) return moment2_tf32_tc_workspace(N, d, flags & ~ST_FLAG_TC_TF32);
    if (xdt == ST_F32 && (flags & ST_FLAG_TC_SPLIT)) return moment2_split_tc_workspace(N, d, flags & ~ST_FLAG_TC_SPLIT);
    if (xdt != ST_F32 || d > 32768) return 0;
    const size_t fma = moment2_use_small(N, d, flags) ? moment2_small_workspace(N, d, flags)
                                                      : kWsHeaderBytes + mg_partial_bytes(moment2_gemm_plan(N, d, flags));
    const size_t exact = moment2_use_exact(N, d) ? moment2_exact_tc_workspace(N, d, flags) : 0;
    return exact > fma ? exact : fma;
}

}  // namespace st

extern "C" st_status st_sym_moment2(const void *X, st_dtype xdt, int64_t N, int64_t d, int64_t ldx,
                                    float *out_packed, void *ws, size_t ws_bytes, unsigned flags, void *stream)
{
    if (!X || !out_packed) return ST_ERR_NULL;
    if (N <= 0 || d <= 0 || ldx < d) return ST_ERR_SHAPE;
    if (xdt != ST_F32 && xdt != ST_BF16) return ST_ERR_DTYPE;
    if (flags & ~(ST_FLAG_DENSE_CONTROL | ST_FLAG_TC_TF32 | ST_FLAG_TC_SPLIT)) return ST_ERR_UNSUPPORTED;
    if ((flags & (ST_FLAG_TC_TF32 | ST_FLAG_TC_SPLIT)) && xdt != ST_F32) return ST_ERR_UNSUPPORTED;
    if ((flags & ST_FLAG_TC_TF32) && (flags & ST_FLAG_TC_SPLIT)) return ST_ERR_UNSUPPORTED;
    if (!st::aligned16(X) || !st::aligned16(out_packed)) return ST_ERR_ALIGN;
    if (xdt == ST_BF16)
        return st::moment2_bf16_tc(X, N, d, ldx, out_packed, ws, ws_bytes, flags, (cudaStream_t)stream);
    if (flags & ST_FLAG_TC_TF32)
        return st::moment2_tf32_tc(X, N, d, ldx, out_packed, ws, ws_bytes, flags & ~ST_FLAG_TC_TF32, (cudaStream_t)stream);
    if (flags & ST_FLAG_TC_SPLIT)
        return st::moment2_split_tc((const float *)X, N, d, ldx, out_packed, ws, ws_bytes, flags & ~ST_FLAG_TC_SPLIT,
                                    (cudaStream_t)stream);
    return st::moment2_f32((const float *)X, N, d, ldx, out_packed, ws, ws_bytes, flags, (cudaStream_t)stream);
}
