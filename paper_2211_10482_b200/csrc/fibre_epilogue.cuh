// Epilogues of the tensor-core fibre kernels: a warp has 32 consecutive fibres (one unit) times R columns of
// Y[m, r] = sum_k B[m, k] W[k, r] in tensor memory.  The accumulator is read in the fragment form (tmem_ld_16x16): a thread
// holds four of the 32 fibres (t/4, t/4 + 8, ...) and two columns of every eight, so that
//   TTM     a store instruction writes whole 32-byte sectors of eight rows (one row per lane took twice the sectors), and
//   MTTKRP  the rows of C come by sectors too, the sum over a run of fibres is three additions in the thread and four
//           shuffles per 16 columns (one fibre per lane: 31 shuffles per 32 columns and run; [236000 fibres, K = 100,
//           R = 64] split: 75 us the call, 61 now).
// SUM: the accumulator has two halves, R columns apart, that are added (split operands).
#pragma once
#include "tc_common.cuh"
#include "mttkrp_common.cuh"

namespace st {

// v[gg][hh][e]: fibre t/4 + 8 hh, column c + 8 gg + 2 (t % 4) + e
template <bool SUM>
__device__ __forceinline__ void fibre_load16(uint32_t taddr, int R, float (&v)[2][4][2])
{
    uint32_t r[2][8];
    tc::tmem_ld_16x16(taddr, r[0]);
    tc::tmem_ld_16x16(taddr + (16u << 16), r[1]);
    if (SUM) {
        uint32_t q[2][8];
        tc::tmem_ld_16x16(taddr + (uint32_t)R, q[0]);
        tc::tmem_ld_16x16(taddr + (16u << 16) + (uint32_t)R, q[1]);
        tc::tmem_ld_wait();
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int x = 0; x < 8; ++x) v[x >> 2][2 * b + ((x >> 1) & 1)][x & 1] = __uint_as_float(r[b][x]) + __uint_as_float(q[b][x]);
    } else {
        tc::tmem_ld_wait();
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int x = 0; x < 8; ++x) v[x >> 2][2 * b + ((x >> 1) & 1)][x & 1] = __uint_as_float(r[b][x]);
    }
}

template <bool SUM>
__device__ __forceinline__ void ttm_epilogue(uint32_t taddr, int R, int64_t row0, int64_t rows, float *out, int lane)
{
    float *dst = out + (row0 + (lane >> 2)) * R + 2 * (lane & 3);
    const int64_t left = rows - row0 - (lane >> 2);
    for (int c = 0; c < R; c += 16) {
        float v[2][4][2];
        fibre_load16<SUM>(taddr + (uint32_t)c, R, v);
#pragma unroll
        for (int h = 0; h < 4; ++h)
            if (8 * h < left) {
#pragma unroll
                for (int g = 0; g < 2; ++g)
                    *reinterpret_cast<float2 *>(dst + (int64_t)(8 * h) * R + c + 8 * g) = make_float2(v[g][h][0], v[g][h][1]);
            }
    }
}

// The fibres of a unit: (i, j) of each of this thread's four, and of the unit's ends.
struct UnitFibres {
    int n;               // fibres (the last unit may have fewer than 32, or none)
    int i0, i1;          // rows of A of the first and the last one
    int i[4], j[4];      // of fibre t/4 + 8 h; j = 0 where there is none
};

// dense: fibre `row` belongs to (row / div, row % div); else row = p(i,j) of a triangle of side I.
__device__ __forceinline__ UnitFibres unit_fibres(int64_t row0, int64_t rows, bool dense, int I, int64_t div, int lane)
{
    UnitFibres f;
    const int64_t left = rows - row0;
    f.n = left >= 32 ? 32 : left > 0 ? (int)left : 0;
    int64_t i = 0, j = 0;
    if (f.n > 0) {
        if (dense) { i = row0 / div; j = row0 - i * div; }
        else tri_decode(I, row0, i, j);
    }
    f.i0 = (int)i;
    const int end = dense ? (div > (int64_t(1) << 30) ? 1 << 30 : (int)div) : I;
    // m fibres on from (i0, j0): row i ends at j = end - 1, the next one starts at 0 (dense; with rows of one fibre, a slice
    // j, the loop would go round m times) or on the diagonal
    auto at = [&](int m, int &ii, int &jj) {
        ii = (int)i;
        jj = (int)j + m;
        if (dense) {
            const int rows_on = jj >= end ? jj / end : 0;
            ii += rows_on;
            jj -= rows_on * end;
        } else {
            while (jj >= end) { ++ii; jj = jj - end + ii; }
        }
    };
    int last;
    if (f.n > 0) at(f.n - 1, f.i1, last);
    else f.i1 = f.i0 - 1;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int m = (lane >> 2) + 8 * h;
        f.i[h] = -1;
        f.j[h] = 0;
        if (m < f.n) at(m, f.i[h], f.j[h]);
    }
    return f;
}

// Columns c .. c + 15 of the rows of C that this thread's fibres take.
__device__ __forceinline__ void unit_load_c(const UnitFibres &f, const float *C, int R, int c, int lane, float2 (&x)[2][4])
{
#pragma unroll
    for (int h = 0; h < 4; ++h)
#pragma unroll
        for (int g = 0; g < 2; ++g) x[g][h] = *reinterpret_cast<const float2 *>(C + (int64_t)f.j[h] * R + c + 8 * g + 2 * (lane & 3));
}

// Sums over the runs of fibres with the same i, times C, to the partial slots (unit + i).  cpre: unit_load_c of column 0,
// asked for before the accumulator was waited for; the next columns' are asked for one step ahead.
template <bool SUM>
__device__ __forceinline__ void mttkrp_epilogue(uint32_t taddr, int R, const UnitFibres &f, const float *C, int64_t unit,
                                                float *part, int64_t nslots, int lane, float2 (&cpre)[2][4])
{
    if (f.n == 0) return;
    for (int c = 0; c < R; c += 16) {
        float2 cur[2][4];
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
            for (int h = 0; h < 4; ++h) cur[g][h] = cpre[g][h];
        if (c + 16 < R) unit_load_c(f, C, R, c + 16, lane, cpre);
        float v[2][4][2];
        fibre_load16<SUM>(taddr + (uint32_t)c, R, v);
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                v[g][h][0] *= cur[g][h].x;
                v[g][h][1] *= cur[g][h].y;
            }
        if (f.n > 1 && f.i1 - f.i0 == f.n - 1) {            // every fibre is a run of its own
#pragma unroll
            for (int h = 0; h < 4; ++h)
                if (f.i[h] >= 0 && ST_BOUNDS_OK(unit + f.i[h], nslots, 5)) {
#pragma unroll
                    for (int g = 0; g < 2; ++g)
                        *reinterpret_cast<float2 *>(part + (unit + f.i[h]) * R + c + 8 * g + 2 * (lane & 3)) = make_float2(v[g][h][0], v[g][h][1]);
                }
            continue;
        }
        for (int i = f.i0; i <= f.i1; ++i) {
            float s[4];
#pragma unroll
            for (int g = 0; g < 2; ++g)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float t = 0.f;
#pragma unroll
                    for (int h = 0; h < 4; ++h) t += f.i[h] == i ? v[g][h][e] : 0.f;
                    s[2 * g + e] = t;
                }
            // lanes t, t ^ 4, t ^ 8, t ^ 16 hold the same columns: halve the columns twice, then add the last pair
            const bool u16 = (lane & 16) != 0, u8 = (lane & 8) != 0;
            float a = u16 ? s[2] : s[0], b = u16 ? s[3] : s[1];
            a += __shfl_xor_sync(0xffffffffu, u16 ? s[0] : s[2], 16);
            b += __shfl_xor_sync(0xffffffffu, u16 ? s[1] : s[3], 16);
            float w = u8 ? b : a;
            w += __shfl_xor_sync(0xffffffffu, u8 ? a : b, 8);
            w += __shfl_xor_sync(0xffffffffu, w, 4);
            if (!(lane & 4) && ST_BOUNDS_OK(unit + i, nslots, 5))
                part[(unit + i) * R + c + (u16 ? 8 : 0) + 2 * (lane & 3) + (u8 ? 1 : 0)] = w;
        }
    }
}

}  // namespace st
