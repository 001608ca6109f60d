// Column order of the pair features of st_sym_moment4 on the tensor-core paths.
//
// Every unique 4-tuple is a pair times a pair in up to three ways, and one of them is enough.  The features are cut into
// five ranges 0..4 (some may be empty).  A 4-tuple with two features in one range is a pair of that range times another
// pair; one with four different ranges is in the product of the pairs {01, 04, 14} with the pairs {23, 24, 34}:
//     0123 = 01 x 23,  0124 = 01 x 24,  0134 = 01 x 34,  0234 = 04 x 23,  1234 = 14 x 23.
// With the pairs inside a range first, the product of the pair features with themselves is so needed in its first `within`
// rows only, and in one block apart from them.  Of the 1035 pairs of 45 features these are 256 rows (ranges of 11, 11,
// 11, 10 and 2) and a block of 165 rows and 152 columns, which take 6 tiles of 256 x 256 or less where the triangle of the
// whole matrix takes 15.
#pragma once
#include "st_index.cuh"

namespace st {

struct PairLayout {
    int features, cols;                    // cols: columns, of which a few are padding
    int lo[6];                             // range g: features lo[g] .. lo[g+1]-1
    int within;                            // columns 0 .. within-1: pairs inside a range, range by range, each in packed order
    int rows, rows_n;                      // columns of the pairs 01, 04, 14: first (a multiple of 8) and number
    int prod, prod_n;                      // columns of the pairs 23, 24, 34 likewise; 02, 03, 12 and 13 follow
};

// A column in 32 bits: features i <= j and their ranges, a byte each.
constexpr unsigned kPairNone = 0xffffffffu;

ST_HD unsigned pair_of_column(const PairLayout &L, int p)
{
    if (p < L.within) {
        for (int g = 0; g < 5; ++g) {
            const int s = L.lo[g + 1] - L.lo[g], n = s * (s + 1) / 2;
            if (p < n) {
                int64_t i, j;
                tri_decode(s, p, i, j);
                return (unsigned)(L.lo[g] + (int)i) | (unsigned)(L.lo[g] + (int)j) << 8 | (unsigned)g << 16 | (unsigned)g << 24;
            }
            p -= n;
        }
        return kPairNone;
    }
    // the ten pairs of different ranges in the order of their columns, four bits each
    const unsigned long long G = 0x1100322100ull, H = 0x3232443441ull;
    int at = L.rows;
    for (int b = 0; b < 10; ++b) {
        if (b == 3) at = L.prod;
        const int g = (int)(G >> (4 * b)) & 15, h = (int)(H >> (4 * b)) & 15;
        const int s = L.lo[h + 1] - L.lo[h], n = (L.lo[g + 1] - L.lo[g]) * s;
        if (p >= at && p < at + n) {
            const int i = (p - at) / s, j = p - at - i * s;
            return (unsigned)(L.lo[g] + i) | (unsigned)(L.lo[h] + j) << 8 | (unsigned)g << 16 | (unsigned)h << 24;
        }
        at += n;
    }
    return kPairNone;
}

// The 4-tuple i <= j <= k <= l that row a and column b stand for, if this is the place that is taken for it.  Rows inside
// a range (the first two features of the tuple that are neighbours in order and share a range) times the other two
// features, or else the block of different ranges.
ST_HD bool pair_product(unsigned a, unsigned b, int &i, int &j, int &k, int &l)
{
    if (a == kPairNone || b == kPairNone) return false;
    const int p = a & 255, q = (a >> 8) & 255, r = b & 255, s = (b >> 8) & 255;
    const int gp = (a >> 16) & 255, gq = a >> 24, gr = (b >> 16) & 255, gs = b >> 24;
    if (gp == gq) {
        if (r >= q) { i = p; j = q; k = r; l = s; return true; }
        if (gr < gp && s >= q) { i = r; j = p; k = q; l = s; return true; }
        i = r; j = s; k = p; l = q;
        return gr < gs && gs < gp;
    }
    i = p;
    if (gq == 1) { j = q; k = r; l = s; return gr >= 2 && gr < gs; }
    j = r; k = s; l = q;
    return gr == 2 && gs == 3;
}

// simp4_encode in 32 bits: 4096 pairs, 90 features.
ST_HD int pair_place(int d, int i, int j, int k, int l)
{
    const unsigned a = (unsigned)(d - i), b = (unsigned)(d - j), c = (unsigned)(d - k), n = (unsigned)d;
    return (int)((n * (n + 1) * (n + 2) * (n + 3) - a * (a + 1) * (a + 2) * (a + 3)) / 24 + (a * (a + 1) * (a + 2) - b * (b + 1) * (b + 2)) / 6 +
                 (b * (b + 1) - c * (c + 1)) / 2) + l - k;
}

}  // namespace st
