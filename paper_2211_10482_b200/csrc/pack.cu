// st_pack / st_unpack: gather the unique set T_U of a dense tensor into the packed layout
// (T_C = T * T_U, Section 4) and reconstruct the dense tensor from it
// (T = T_C + T_R * T_C, Section 6, Property 5).  HBM-bound copies.
//
// The dense array is cut into slices along its last structured index (matrix row i; pair (i,j) of an
// order-3 tensor, triple of an order-4 one).
//   slice_copy_kernel (st_pack, st_thp, st_unpack with zero fill): in every supported structure the unique
//   positions of a slice are ONE contiguous run of columns [lo,hi) that is also contiguous in the packed
//   array, so a slice is "zeros, one flat copy, zeros" and needs no per-element index arithmetic at all: the
//   run and its packed offset come from the closed forms of st_index.cuh once per slice.  Long slices are
//   split into parts over several thread groups.
//   sym_slice_kernel (st_unpack with symmetric fill): the positions of a slice from its largest fixed index on
//   are such a run too; in front of it every position is mapped through the redundancy map by itself.
//   sym_row_kernel: the same for wide positions, each by itself.
//   sym_tile_kernel: the same for a matrix of single elements, through 32 x 32 tiles.
//
// A run starts wherever the closed form says, so source and destination usually differ in their offset from a
// 16-byte boundary.  copy_flat stores whole 16-byte units all the same and takes each from the two aligned units
// that hold it (the second one is an L1 hit), shifted in registers, never past the end of the source array.  Measured against copies in the widest unit that
// divides a row, each position of a symmetric fill by itself (pack + unpack): tet d = 60, rows of 33 floats, 72 -> 24 us;
// tri d = 900, rows of 17 bf16, 125 -> 21 us; simplex4 d = 64 floats, 220 -> 32 us; tet d = 200 bf16, 27 -> 9 us.
#include "st_common.cuh"
#include "st_index.cuh"
#include "copy_span.cuh"
#include <type_traits>

namespace st {

constexpr int COPY_UNITS = 4;              // 16-byte units that a thread of the slice copies has in flight
// Slice copies have grids as large as the work: blocks then start in the order of memory.  With 16 blocks per SM that walk the array in
// strides, of which only some fit at a time, it was written in several sweeps with holes ([4096,4096,64] zero fill 755 us,
// now 624; [2000,2000,64] 253, now 229).
constexpr int64_t MAX_GRID = int64_t(1) << 30;
constexpr int ROW_SEG = 2048, ROW_WIDE = 512;   // symmetric fill of wide positions
constexpr int SYM_WORDS = 4;               // words that a lane of the symmetric fill has in flight
constexpr int64_t PART_BYTES = 32768;      // most of a slice that one thread group copies ([384,384,75]: 128 KiB starve the chip)
constexpr int64_t ONCE_BYTES = 256 * 16 * COPY_UNITS;     // the same in one pass (copy_once)

struct LayoutArgs {
    int kind;
    int fill;
    int64_t d, kl, ku, nb, bs;
    int64_t width;       // band: kl+ku+1
    int64_t packed_rows;
    int64_t dense_rows;
    int64_t row_bytes;   // of one position (`inner` elements)
};

template <int ES> struct Elem;
template <> struct Elem<2> { typedef uint16_t T; };
template <> struct Elem<4> { typedef uint32_t T; };
template <> struct Elem<8> { typedef uint2 T; };
template <> struct Elem<16> { typedef uint4 T; };

// 16 bytes at byte `off` (a multiple of ES, not 0) of the two aligned units a and b.
template <int ES>
__device__ __forceinline__ uint4 shift_unit(const uint4 &a, const uint4 &b, unsigned off)
{
    uint32_t w0 = a.x, w1 = a.y, w2 = a.z, w3 = a.w, w4 = b.x;
    if (off & 8) { w0 = a.z; w1 = a.w; w2 = b.x; w3 = b.y; w4 = b.z; }
    if (ES < 8) {
        const uint32_t w5 = (off & 8) ? b.w : b.y;
        if (off & 4) { w0 = w1; w1 = w2; w2 = w3; w3 = w4; w4 = w5; }
    }
    if (ES < 4 && (off & 2)) {
        w0 = __funnelshift_r(w0, w1, 16);
        w1 = __funnelshift_r(w1, w2, 16);
        w2 = __funnelshift_r(w2, w3, 16);
        w3 = __funnelshift_r(w3, w4, 16);
    }
    return make_uint4(w0, w1, w2, w3);
}

__device__ __forceinline__ uint32_t mul_word(uint32_t a, uint32_t b) { return __float_as_uint(__uint_as_float(a) * __uint_as_float(b)); }

// dst[0..n) = src[0..n) (bytes, multiples of ES) by the `g` threads of a group, U units of a thread in flight; MUL:
// times mul[0..n), fp32, which is offset from a 16-byte boundary as dst is.  The elements in front of the first whole
// unit of dst and behind the last one are loaded ahead of the units, so that they cost no round trip of their own.
template <int ES, bool MUL, int U>
__device__ __forceinline__ void copy_flat(unsigned char *dst, const unsigned char *src, const unsigned char *mul, int n, int lane, int g,
                                          const unsigned char *src_end)
{
    typedef typename Elem<ES>::T E;
    const CopySpan span = copy_span((uintptr_t)dst, (uintptr_t)src, n, (uintptr_t)src_end);
    const int head = span.head, units = span.units, ends = span.ends;
    const unsigned off = span.off;
    auto end_at = [&](int e) { return e < head ? e : e + (units << 4); };
    auto end_load = [&](int e) {
        E v = *reinterpret_cast<const E *>(src + end_at(e));
        if constexpr (MUL) v = mul_word(v, *reinterpret_cast<const uint32_t *>(mul + end_at(e)));
        return v;
    };
    const int e0 = lane * ES;
    E ev = E{};
    if (e0 < ends) ev = end_load(e0);
    const uint4 *in = reinterpret_cast<const uint4 *>(src + head - off);
    uint4 *out = reinterpret_cast<uint4 *>(dst + head);
    const uint4 *m = MUL ? reinterpret_cast<const uint4 *>(mul + head) : nullptr;
    // The loads of a batch come before its first store in the source: coherent loads are not moved over a store by the compiler.
    auto store = [&](int u, uint4 v, const uint4 &w) {
        if (MUL) v = make_uint4(mul_word(v.x, w.x), mul_word(v.y, w.y), mul_word(v.z, w.z), mul_word(v.w, w.w));
        out[u] = v;
    };
    if (ES == 16 || off == 0) {
        for (int u0 = lane; u0 < units; u0 += U * g) {
            uint4 v[U], w[U];
#pragma unroll
            for (int k = 0; k < U; ++k)
                if (u0 + k * g < units) {
                    v[k] = in[u0 + k * g];
                    if (MUL) w[k] = m[u0 + k * g];
                }
#pragma unroll
            for (int k = 0; k < U; ++k)
                if (u0 + k * g < units) store(u0 + k * g, v[k], w[k]);
        }
    } else {
        constexpr int H = U > 1 ? U / 2 : U;                // two loads a unit: batches of half as many
        for (int u0 = lane; u0 < units; u0 += H * g) {
            uint4 v[H], y[H], w[H];
#pragma unroll
            for (int k = 0; k < H; ++k)
                if (u0 + k * g < units) {
                    v[k] = in[u0 + k * g];
                    y[k] = in[u0 + k * g + 1];
                    if (MUL) w[k] = m[u0 + k * g];
                }
#pragma unroll
            for (int k = 0; k < H; ++k)
                if (u0 + k * g < units) store(u0 + k * g, shift_unit<ES>(v[k], y[k], off), w[k]);
        }
    }
    if (e0 < ends) *reinterpret_cast<E *>(dst + end_at(e0)) = ev;
    for (int e = e0 + g * ES; e < ends; e += g * ES) *reinterpret_cast<E *>(dst + end_at(e)) = end_load(e);   // small groups only
}

// The same by whole warps, for at most 16 U bytes a thread: warp l / 32 of the group takes the 32 U units from there on.  Where the
// source is off a boundary a unit is put together from the aligned unit that its lane loaded and the one of the next lane,
// which is half the loads of copy_flat and leaves room for U units in flight.
template <int ES, bool MUL, int U>
__device__ __forceinline__ void copy_once(unsigned char *dst, const unsigned char *src, const unsigned char *mul, int n, int lane,
                                          const unsigned char *src_end)
{
    typedef typename Elem<ES>::T E;
    const CopySpan span = copy_span((uintptr_t)dst, (uintptr_t)src, n, (uintptr_t)src_end);
    const int units = span.units;
    const unsigned off = span.off;
    const int l = lane & 31, e = lane * ES, b = (lane & ~31) * U + l;
    const int end_at = e < span.head ? e : e + (units << 4);             // less than 32 elements
    E ev = E{};
    if (e < span.ends) ev = *reinterpret_cast<const E *>(src + end_at);
    const uint4 *in = reinterpret_cast<const uint4 *>(src + span.head - off) + b;
    const int loads = (off != 0 && units > 0 ? units + 1 : units) - b, stores = units - b;
    uint4 v[U + 1], w[MUL ? U : 1];
#pragma unroll
    for (int k = 0; k < U; ++k) {
        if (32 * k < loads) v[k] = in[32 * k];
        if (MUL && 32 * k < stores) w[k] = reinterpret_cast<const uint4 *>(mul + span.head)[b + 32 * k];
    }
    if (off != 0 && l == 0 && 32 * U < loads) v[U] = in[32 * U];
    if constexpr (MUL)
        if (e < span.ends) ev = mul_word(ev, *reinterpret_cast<const uint32_t *>(mul + end_at));
    uint4 *out = reinterpret_cast<uint4 *>(dst + span.head) + b;
    const int next = (l + 1) & 31;                                       // lane 0 has the unit behind those of all lanes
#pragma unroll
    for (int k = 0; k < U; ++k) {
        uint4 r = v[k];
        if (ES < 16 && off != 0) {
            uint4 y = make_uint4(0, 0, 0, 0);                            // as far as it is needed
            y.x = __shfl_sync(0xFFFFFFFFu, l == 0 ? v[k + 1].x : r.x, next);
            if (off > 4) y.y = __shfl_sync(0xFFFFFFFFu, l == 0 ? v[k + 1].y : r.y, next);
            if (ES < 8 && off > 8) y.z = __shfl_sync(0xFFFFFFFFu, l == 0 ? v[k + 1].z : r.z, next);
            if (ES < 4 && off > 12) y.w = __shfl_sync(0xFFFFFFFFu, l == 0 ? v[k + 1].w : r.w, next);
            r = shift_unit<ES>(r, y, off);
        }
        if (32 * k < stores) {
            if (MUL) r = make_uint4(mul_word(r.x, w[k].x), mul_word(r.y, w[k].y), mul_word(r.z, w[k].z), mul_word(r.w, w[k].w));
            out[32 * k] = r;
        }
    }
    if (e < span.ends) *reinterpret_cast<E *>(dst + end_at) = ev;
}

template <int ES>
__device__ __forceinline__ void zero_flat(unsigned char *dst, int n, int lane, int g)
{
    typedef typename Elem<ES>::T E;
    int head = (int)((0u - (unsigned)(uintptr_t)dst) & 15u);
    if (head > n) head = n;
    const int units = (n - head) >> 4;
    const int ends = n - (units << 4);
    for (int e = lane * ES; e < ends; e += g * ES) *reinterpret_cast<E *>(dst + (e < head ? e : e + (units << 4))) = E{};
    uint4 *out = reinterpret_cast<uint4 *>(dst + head);
    for (int u = lane; u < units; u += g) out[u] = make_uint4(0, 0, 0, 0);
}

// Closed forms of st_index.cuh in the index type I: unsigned where every index fits in 31 bits.
template <typename I> __device__ __forceinline__ I tri_n(I d) { return d * (d + 1) / 2; }
template <typename I> __device__ __forceinline__ I tet_n(I d) { return d * (d + 1) / 2 * (d + 2) / 3; }
template <typename I> __device__ __forceinline__ I simp4_n(I d) { return tet_n<I>(d) * (d + 3) / 4; }
template <typename I> __device__ __forceinline__ I tri_at(I d, I i, I j) { return i * (2 * d - i + 1) / 2 + (j - i); }
template <typename I> __device__ __forceinline__ I tet_at(I d, I i, I j, I k) { return tet_n<I>(d) - tet_n<I>(d - i) + tri_at<I>(d - i, j - i, k - i); }
template <typename I> __device__ __forceinline__ I simp4_at(I d, I i, I j, I k, I l) { return simp4_n<I>(d) - simp4_n<I>(d - i) + tet_at<I>(d - i, j - i, k - i, l - i); }
template <typename I> __device__ __forceinline__ void tri_dec(I d, I p, I &i, I &j)
{
    const I b = 2 * d + 1;
    const I root = (I)sqrtf((float)(b * b - 8 * p));
    I ii = root < b ? (b - root) >> 1 : 0;
    if (ii > d - 1) ii = d - 1;
    while (ii > 0 && tri_at<I>(d, ii, ii) > p) --ii;
    while (ii + 1 < d && tri_at<I>(d, ii + 1, ii + 1) <= p) ++ii;
    i = ii;
    j = ii + (p - tri_at<I>(d, ii, ii));
}
template <typename I> __device__ __forceinline__ void tet_dec(I d, I q, I &i, I &j, I &k)
{
    const I r = tet_n<I>(d) - q;                              // positions left; the slab of side m holds tet(m-1) < r <= tet(m)
    I m = (I)cbrtf(6.0f * (float)r);
    if (m < 1) m = 1;
    if (m > d) m = d;
    while (m > 1 && tet_n<I>(m - 1) >= r) --m;
    while (m < d && tet_n<I>(m) < r) ++m;
    i = d - m;
    tri_dec<I>(m, tet_n<I>(m) - r, j, k);
    j += i;
    k += i;
}

// Run of unique columns of slice s: dense columns [lo,hi) of the slice map to packed rows prow.. (contiguous).
// PACK of an order-3 or order-4 tensor or of one row visits the slices with a run only: item s is then the s-th of those, and
// s becomes the number of its slice.
template <int KIND, bool PACK, typename I>
__device__ __forceinline__ void slice_run(const LayoutArgs &a, I &s, I &lo, I &hi, I &prow)
{
    const I d = (I)a.d, kl = (I)a.kl;
    if (KIND == ST_TRI_UPPER) {
        lo = s; hi = d; prow = tri_at<I>(d, s, s);
    } else if (KIND == ST_TET) {
        I i, j;
        if (PACK) { tri_dec<I>(d, s, i, j); s = i * d + j; }
        else { i = s / d; j = s - i * d; }
        if (j < i) { lo = hi = 0; prow = 0; }
        else { lo = j; hi = d; prow = tet_at<I>(d, i, j, j); }
    } else if (KIND == ST_BAND) {
        lo = s > kl ? s - kl : 0;
        hi = s + (I)a.ku + 1 < d ? s + (I)a.ku + 1 : d;
        if (hi < lo) hi = lo;
        prow = s * (I)a.width + (lo + kl - s);
    } else if (KIND == ST_FIXED_ROW) {
        if (PACK) s = kl;
        if (s == kl) { lo = 0; hi = d; } else { lo = hi = 0; }
        prow = 0;
    } else if (KIND == ST_FIXED_COL) {
        lo = kl; hi = kl + 1; prow = s;
    } else if (KIND == ST_SIMPLEX4) {
        // slice s = (i, j, k): its unique entries are l = k .. d-1 when i <= j <= k
        I i, j, k;
        if (PACK) {
            tet_dec<I>(d, s, i, j, k);
            s = (i * d + j) * d + k;
        } else {
            const I ij = s / d;
            k = s - ij * d; i = ij / d; j = ij - i * d;
        }
        if (i <= j && j <= k) { lo = k; hi = d; prow = simp4_at<I>(d, i, j, k, k); }
        else { lo = hi = 0; prow = 0; }
    } else {
        const I bs = (I)a.bs, b = s / bs;
        lo = b * bs; hi = lo + bs; prow = s * bs;
    }
}

// Four blocks per SM: with the registers that the compiler would take (up to 96) fewer fit, and the zeros of a sparse slice are
// bound by the number of blocks ([8000,8000] band 39.5 us, 37.7 with 64 registers; st_thp of a tet d = 120, rows of 64 floats
// 52, now 39).
// ONCE: blocks, of as many warps as it takes, that go through their part of a slice in one pass (copy_once).
template <int KIND, int ES, bool PACK, bool MUL, bool ONCE, typename I>
__global__ void __launch_bounds__(256, 4)
slice_copy_kernel(const unsigned char *src, unsigned char *dst, LayoutArgs a, I nitems, int group_shift, int parts,
                  int part_bytes, const unsigned char *mul)
{
    // MUL (pack only, fp32 elements): a second packed operand; the gathered values are multiplied by it
    pdl_wait();
    pdl_trigger();
    const int g = ONCE ? (int)blockDim.x : 1 << group_shift;
    const int lane = ONCE ? (int)threadIdx.x : (int)(threadIdx.x & (g - 1));
    const I gid = ONCE ? (I)blockIdx.x : (I)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> group_shift);
    const I ngroups = ONCE ? (I)gridDim.x : (I)(((int64_t)gridDim.x * blockDim.x) >> group_shift);
    const int64_t sb = a.d * a.row_bytes;                     // bytes per dense slice
    const unsigned char *src_end = src + (PACK ? a.dense_rows : a.packed_rows) * a.row_bytes;
    auto copy = [&](unsigned char *to, const unsigned char *from, const unsigned char *times, int n) {
        if constexpr (ONCE) copy_once<ES, MUL, COPY_UNITS>(to, from, times, n, lane, src_end);
        else copy_flat<ES, MUL, MUL ? COPY_UNITS / 2 : COPY_UNITS>(to, from, times, n, lane, g, src_end);
    };
    for (I item = gid; item < nitems; item += ngroups) {
        I s = parts == 1 ? item : item / (I)parts, lo, hi, prow;
        const int64_t part = item - s * (I)parts;
        slice_run<KIND, PACK, I>(a, s, lo, hi, prow);
        // a non-empty run lies inside the slice and inside the packed array
        if (hi > lo && !(ST_BOUNDS_OK(lo, a.d, 1) && ST_BOUNDS_OK(hi - 1, a.d, 1) && ST_BOUNDS_OK(prow, a.packed_rows, 1) &&
                         ST_BOUNDS_OK((int64_t)prow + (hi - lo) - 1, a.packed_rows, 1)))
            continue;
        const int64_t c0 = (int64_t)lo * a.row_bytes, c1 = (int64_t)hi * a.row_bytes;   // the run inside the slice
        // pack splits the run itself into parts (a band's fixed-width packed row, whose slots outside the matrix are zeros),
        // unpack the whole dense slice (it writes all of it)
        constexpr bool BAND_ROW = PACK && KIND == ST_BAND;
        const int64_t shift = BAND_ROW ? ((int64_t)prow - (int64_t)s * a.width) * a.row_bytes - c0 : 0;
        const int64_t d0 = c0 + shift, d1 = c1 + shift;       // the run inside what is split
        const int64_t r0 = PACK && !BAND_ROW ? c0 : 0, r1 = BAND_ROW ? a.width * a.row_bytes : PACK ? c1 : sb;
        int64_t u0 = r0 + part * part_bytes;                  // this part covers bytes [u0, u1) of it
        int64_t u1 = u0 + part_bytes;
        if (u0 > r1) u0 = r1;
        if (u1 > r1) u1 = r1;
        const int64_t x0 = u0 > d0 ? u0 : d0, x1 = u1 < d1 ? u1 : d1;   // run clipped to this part
        const int64_t p0 = (int64_t)prow * a.row_bytes - d0;           // packed byte of its byte 0, were it in the run
        if (PACK) {
            if (BAND_ROW && d0 > u0) zero_flat<ES>(dst + p0 + u0, (int)((u1 < d0 ? u1 : d0) - u0), lane, g);
            if (x1 > x0) copy(dst + p0 + x0, src + (int64_t)s * sb + x0 - shift, mul + p0 + x0, (int)(x1 - x0));
            if (BAND_ROW && u1 > d1) zero_flat<ES>(dst + p0 + (u0 > d1 ? u0 : d1), (int)(u1 - (u0 > d1 ? u0 : d1)), lane, g);
        } else {
            unsigned char *out = dst + (int64_t)s * sb;
            const int64_t z1 = u1 < c0 ? u1 : c0;               // zeros before the run
            if (z1 > u0) zero_flat<ES>(out + u0, (int)(z1 - u0), lane, g);
            if (x1 > x0) copy(out + x0, src + p0 + x0, nullptr, (int)(x1 - x0));
            const int64_t z2 = u0 > c1 ? u0 : c1;               // zeros after the run
            if (u1 > z2) zero_flat<ES>(out + z2, (int)(u1 - z2), lane, g);
        }
    }
}

// Packed row of position x of the slice whose fixed indices are a <= b <= c (as many as KIND has); x < the largest.
template <int KIND, typename I>
__device__ __forceinline__ I sym_row(I d, I a, I b, I c, I x)
{
    if (KIND == ST_TRI_UPPER) return tri_at<I>(d, x, a);
    if (KIND == ST_TET) return x < a ? tet_at<I>(d, x, a, b) : tet_at<I>(d, a, x, b);
    return x < a ? simp4_at<I>(d, x, a, b, c) : x < b ? simp4_at<I>(d, a, x, b, c) : simp4_at<I>(d, a, b, x, c);
}

// Fixed indices of slice s in increasing order (as many as KIND has); returns the largest.
template <int KIND, typename I>
__device__ __forceinline__ I sym_fixed(I d, I s, I &a, I &b, I &c)
{
    I t;
    b = c = 0;
    if (KIND == ST_TRI_UPPER) return a = s;
    if (KIND == ST_TET) {
        a = s / d; b = s - a * d;
        if (a > b) { t = a; a = b; b = t; }
        return b;
    }
    const I ij = s / d;
    c = s - ij * d; a = ij / d; b = ij - a * d;
    if (a > b) { t = a; a = b; b = t; }
    if (b > c) { t = b; b = c; c = t; }
    if (a > b) { t = a; a = b; b = t; }
    return c;
}

// Packed row of position x of the slice whose fixed indices are a <= b <= c, from the largest on.
template <int KIND, typename I>
__device__ __forceinline__ I sym_run_row(I d, I a, I b, I c, I x)
{
    return KIND == ST_TRI_UPPER ? tri_at<I>(d, a, x) : KIND == ST_TET ? tet_at<I>(d, a, b, x) : simp4_at<I>(d, a, b, c, x);
}

// One warp per part of a slice.  Positions from the largest fixed index on: one flat copy.  In front of it lanes run along
// the words of the positions (inv != 0), or a lane group copies a position (`inner` elements) at a time.
// FORM: 2 both; for tensors of order 3 and 4 with words of 4 bytes and more, whose rows take longer to find, an instance for the
// words (1) and one for the positions (0).  In the first a lane finds the row of one position of the part for all lanes, but not for
// the words of 8 bytes of order 3 (tet d = 160, 33 floats, 208 us with a row found for every word, now 196; simplex4 d = 24, 41
// floats, 31 and 22; tet d = 100, 21 doubles, 50 with rows for every word, 56 from lanes).
template <int KIND, int ES, int FORM, typename I>
__global__ void __launch_bounds__(256)
sym_slice_kernel(const unsigned char *src, unsigned char *dst, I d, I nslices, int parts, int part_rows,
                 int row_bytes, unsigned inv, int group_shift, int64_t packed_rows)
{
    typedef typename Elem<ES>::T E;
    pdl_wait();
    pdl_trigger();
    const int lane = (int)(threadIdx.x & 31);
    const unsigned char *src_end = src + packed_rows * row_bytes;
    const I nitems = nslices * (I)parts, nwarps = (I)gridDim.x * (I)(blockDim.x / 32);
    for (I item = (I)blockIdx.x * (I)(blockDim.x / 32) + (I)(threadIdx.x / 32); item < nitems; item += nwarps) {
        const I s = parts == 1 ? item : item / (I)parts;
        const I x0 = (item - s * (I)parts) * (I)part_rows;
        const I x1 = x0 + (I)part_rows < d ? x0 + (I)part_rows : d;
        I a, b, c;
        const I top = sym_fixed<KIND, I>(d, s, a, b, c);
        unsigned char *out = dst + (int64_t)s * d * row_bytes;
        const I xr = x0 > top ? x0 : top;                                // first position of the run in this part
        if (xr < x1) {
            const I p = sym_run_row<KIND, I>(d, a, b, c, xr);
            if (ST_BOUNDS_OK(p, packed_rows, 1) && ST_BOUNDS_OK((int64_t)p + (x1 - xr) - 1, packed_rows, 1))
                copy_flat<ES, false, ES >= 8 ? 2 : 1>(out + (int64_t)xr * row_bytes, src + (int64_t)p * row_bytes, nullptr, (int)(x1 - xr) * row_bytes, lane, 32, src_end);
        }
        const I xe = x1 < top ? x1 : top;
        const int words = row_bytes / ES;
        if (FORM == 1 || (FORM == 2 && inv != 0)) {
            // lanes along the words of consecutive positions: word e belongs to position e / words (inv: 2^32 / words rounded up,
            // exact for e < 2^17 and up to 128 words)
            const unsigned n = xe > x0 ? (unsigned)(xe - x0) * (unsigned)words : 0u;
            E *o = reinterpret_cast<E *>(out + (int64_t)x0 * row_bytes);
            if (FORM == 1 && (KIND == ST_SIMPLEX4 || ES == 4) && words >= 8) {
                // a part has at most 32 positions, and each lane finds the row of one for all lanes
                const I mine = x0 + (I)lane < xe ? sym_row<KIND, I>(d, a, b, c, x0 + (I)lane) : (I)0;
                for (unsigned e0 = 0; e0 < n; e0 += 32 * SYM_WORDS) {
                    E v[SYM_WORDS];
#pragma unroll
                    for (int u = 0; u < SYM_WORDS; ++u) {
                        const unsigned e = e0 + 32 * u + (unsigned)lane;
                        const unsigned dx = __umulhi(e, inv);
                        const I p = __shfl_sync(0xFFFFFFFFu, mine, (int)dx & 31);
                        if (e < n) v[u] = ST_BOUNDS_OK(p, packed_rows, 1) ? reinterpret_cast<const E *>(src)[(int64_t)p * words + (e - dx * (unsigned)words)] : E{};
                    }
#pragma unroll
                    for (int u = 0; u < SYM_WORDS; ++u)
                        if (e0 + 32 * u + (unsigned)lane < n) o[e0 + 32 * u + (unsigned)lane] = v[u];
                }
                continue;
            }
            for (unsigned e0 = (unsigned)lane; e0 < n; e0 += 32 * SYM_WORDS) {
                E v[SYM_WORDS];
#pragma unroll
                for (int u = 0; u < SYM_WORDS; ++u) {
                    const unsigned e = e0 + 32 * u;
                    if (e >= n) continue;
                    // (order 3: the high half of a product costs 7 % there, and for the at most 256 words of a part that by 2^16 / words does)
                    const unsigned dx = words == 1 ? e : FORM == 1 && KIND == ST_TET && words <= 32 ? (e * ((inv + 0xFFFF) >> 16)) >> 16 : __umulhi(e, inv);
                    const I p = sym_row<KIND, I>(d, a, b, c, x0 + (I)dx);
                    v[u] = ST_BOUNDS_OK(p, packed_rows, 1) ? reinterpret_cast<const E *>(src)[(int64_t)p * words + (e - dx * (unsigned)words)] : E{};
                }
#pragma unroll
                for (int u = 0; u < SYM_WORDS; ++u)
                    if (e0 + 32 * u < n) o[e0 + 32 * u] = v[u];
            }
        } else {
            const int g = 1 << group_shift;
            for (I x = x0 + (I)(lane >> group_shift); x < xe; x += (I)(32 >> group_shift)) {
                const I p = sym_row<KIND, I>(d, a, b, c, x);
                if (!ST_BOUNDS_OK(p, packed_rows, 1)) continue;
                unsigned char *o = out + (int64_t)x * row_bytes;
                const unsigned char *from = src + (int64_t)p * row_bytes;
                copy_flat<ES, false, 1>(o, from, nullptr, row_bytes, lane & (g - 1), g, src_end);
            }
        }
    }
}

// Positions of more than ROW_WIDE bytes: a warp copies up to ROW_SEG bytes of one, U units of a lane in flight, in the order of
// the dense array.  sym_slice_kernel, which served them before, has one unit in flight, one warp for a position however wide,
// and blocks that walk the array: [384,384,300] 63 us, now 50; simplex4 d = 10, 5000 floats, 79 and 36; tri d = 12, 20000
// floats, 26 and 4.4.
template <int KIND, int ES, int U, typename I>
__global__ void __launch_bounds__(256)
sym_row_kernel(const unsigned char *src, unsigned char *dst, I d, I nitems, I segs, int64_t row_bytes, int64_t packed_rows)
{
    pdl_wait();
    pdl_trigger();
    const int lane = (int)(threadIdx.x & 31);
    const unsigned char *src_end = src + packed_rows * row_bytes;
    const I nwarps = (I)gridDim.x * (I)(blockDim.x / 32);
    for (I item = (I)blockIdx.x * (I)(blockDim.x / 32) + (I)(threadIdx.x / 32); item < nitems; item += nwarps) {
        const I row = segs == 1 ? item : item / segs;
        const int64_t off = (int64_t)(item - row * segs) * ROW_SEG;
        const I s = row / d, x = row - s * d;
        I a, b, c;
        const I top = sym_fixed<KIND, I>(d, s, a, b, c);
        const I p = x < top ? sym_row<KIND, I>(d, a, b, c, x) : sym_run_row<KIND, I>(d, a, b, c, x);
        if (!ST_BOUNDS_OK(p, packed_rows, 1)) continue;
        const int n = row_bytes - off < ROW_SEG ? (int)(row_bytes - off) : ROW_SEG;
        copy_flat<ES, false, U>(dst + (int64_t)row * row_bytes + off, src + (int64_t)p * row_bytes + off, nullptr, n, lane, 32, src_end);
    }
}

// Symmetric fill of single elements (the reconstruction of a moment).  With the leading indices fixed (none, i, or
// i1 <= i2) the last two indices span a symmetric matrix; a block reads one 32 x 32 tile (j <= k) of its upper triangle,
// lanes along k, and writes it twice, the second time transposed through shared memory -- and, for i1 < i2, both again
// into the slab (i2, i1).  Lanes read consecutive packed words wherever k is the largest index.
template <int KIND, int ES>
__global__ void __launch_bounds__(256)
sym_tile_kernel(const typename Elem<ES>::T *packed, typename Elem<ES>::T *dense, unsigned d, unsigned nt, int64_t packed_rows)
{
    typedef typename Elem<ES>::T E;
    __shared__ E tile[32][33];
    pdl_wait();
    pdl_trigger();
    const unsigned i1 = blockIdx.y, i2 = blockIdx.z;       // leading indices
    if (KIND == ST_SIMPLEX4 && i1 > i2) return;
    int64_t bi64, bj64;
    tri_decode((int64_t)nt, (int64_t)blockIdx.x, bi64, bj64);
    const unsigned bi = (unsigned)bi64, bj = (unsigned)bj64;
    const unsigned tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    E *const out = KIND == ST_TRI_UPPER ? dense : KIND == ST_TET ? dense + (size_t)i1 * d * d : dense + ((size_t)i1 * d + i2) * d * d;
    E *const out2 = KIND == ST_SIMPLEX4 ? dense + ((size_t)i2 * d + i1) * d * d : out;
    auto at = [&](unsigned j, unsigned k) -> unsigned {     // j <= k
        if (KIND == ST_TRI_UPPER) return tri_at<unsigned>(d, j, k);
        if (KIND == ST_TET) return i1 <= j ? tet_at<unsigned>(d, i1, j, k) : i1 <= k ? tet_at<unsigned>(d, j, i1, k) : tet_at<unsigned>(d, j, k, i1);
        unsigned a = i1, b = i2, c = j, e = k, t;           // two sorted pairs, merged
        if (a > c) { t = a; a = c; c = t; }
        if (b > e) { t = b; b = e; e = t; }
        if (b > c) { t = b; b = c; c = t; }
        return simp4_at<unsigned>(d, a, b, c, e);
    };
    E v[4];
#pragma unroll
    for (unsigned q = 0; q < 4; ++q) {
        const unsigned j = bi * 32 + ty + 8 * q, k = bj * 32 + tx;
        if (j <= k && k < d) {
            const unsigned p = at(j, k);
            v[q] = ST_BOUNDS_OK(p, packed_rows, 1) ? packed[p] : E{};
        }
    }
#pragma unroll
    for (unsigned q = 0; q < 4; ++q) {
        const unsigned j = bi * 32 + ty + 8 * q, k = bj * 32 + tx;
        if (j <= k && k < d) {
            tile[ty + 8 * q][tx] = v[q];
            out[(size_t)j * d + k] = v[q];
            if (KIND == ST_SIMPLEX4 && i1 < i2) out2[(size_t)j * d + k] = v[q];
        }
    }
    __syncthreads();
#pragma unroll
    for (unsigned q = 0; q < 4; ++q) {
        const unsigned k = bj * 32 + ty + 8 * q, j = bi * 32 + tx;       // dense row k, column j < k
        if (j < k && k < d) {
            const E w = tile[tx][ty + 8 * q];
            out[(size_t)k * d + j] = w;
            if (KIND == ST_SIMPLEX4 && i1 < i2) out2[(size_t)k * d + j] = w;
        }
    }
}

// out = alpha * a + beta * b (OP 0) or out = a * b (OP 1) over packed arrays of the same layout.
// `out` may be `a` or `b` (a thread reads the elements it later writes, and nobody else's), so none of
// the pointers is declared restrict.
template <int OP>
__global__ void __launch_bounds__(256)
packed_binary_kernel(const float *a, const float *b, float *out, int64_t n, float alpha, float beta)
{
    pdl_wait();
    pdl_trigger();
    const int64_t n4 = n >> 2;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n4; e += stride) {
        const float4 x = reinterpret_cast<const float4 *>(a)[e];
        const float4 y = reinterpret_cast<const float4 *>(b)[e];
        float4 r;
        if (OP == 0) r = make_float4(alpha * x.x + beta * y.x, alpha * x.y + beta * y.y, alpha * x.z + beta * y.z, alpha * x.w + beta * y.w);
        else r = make_float4(x.x * y.x, x.y * y.y, x.z * y.z, x.w * y.w);
        reinterpret_cast<float4 *>(out)[e] = r;
    }
    for (int64_t e = 4 * n4 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += stride)
        out[e] = OP == 0 ? alpha * a[e] + beta * b[e] : a[e] * b[e];
}

static bool layout_ok(const st_layout *L)
{
    if (!L) return false;
    if (L->reserved != 0) return false;
    if (L->d <= 0 || L->inner <= 0) return false;
    if (L->d > (int64_t(1) << 31)) return false;
    switch (L->kind) {
    case ST_TRI_UPPER: return true;
    case ST_TET: return L->d <= (int64_t(1) << 20);
    case ST_SIMPLEX4: return L->d <= 32768;
    case ST_FIXED_ROW:
    case ST_FIXED_COL: return L->kl >= 0 && L->kl < L->d;
    case ST_BAND: return L->kl >= 0 && L->ku >= 0 && L->kl < (int64_t(1) << 31) && L->ku < (int64_t(1) << 31);
    case ST_BLOCKDIAG: return L->nblocks > 0 && L->bs > 0 && L->nblocks * L->bs == L->d;
    default: return false;
    }
}

static int64_t packed_rows_of(const st_layout *L)
{
    switch (L->kind) {
    case ST_TRI_UPPER: return tri_rows(L->d);
    case ST_TET: return tet_rows(L->d);
    case ST_SIMPLEX4: return simp4_rows(L->d);
    case ST_FIXED_ROW:
    case ST_FIXED_COL: return L->d;
    case ST_BAND: return L->d * (L->kl + L->ku + 1);
    default: return L->nblocks * L->bs * L->bs;
    }
}

static int64_t dense_rows_of(const st_layout *L)
{
    if (L->kind == ST_SIMPLEX4) return L->d * L->d * L->d * L->d;
    return L->kind == ST_TET ? L->d * L->d * L->d : L->d * L->d;
}

static int dtype_bytes(st_dtype t)
{
    switch (t) {
    case ST_F32: return 4;
    case ST_BF16: return 2;
    case ST_F64: return 8;
    default: return 0;
    }
}

template <int KIND, int ES>
static st_status launch_sym(const void *src, void *dst, const LayoutArgs &a, cudaStream_t s)
{
    typedef typename Elem<ES>::T E;
    // packed indices and d^2 in 32 bits
    const bool small = a.d <= (KIND == ST_TRI_UPPER ? 32768 : KIND == ST_TET ? 1024 : 200);
    if (a.row_bytes == ES && small) {
        const unsigned nt = (unsigned)((a.d + 31) / 32);
        const dim3 grid(nt * (nt + 1) / 2, KIND == ST_TRI_UPPER ? 1u : (unsigned)a.d, KIND == ST_SIMPLEX4 ? (unsigned)a.d : 1u);
        return launch(sym_tile_kernel<KIND, ES>, grid, 256, 0, s, (const E *)src, (E *)dst, (unsigned)a.d, nt, a.packed_rows);
    }
    const unsigned char *in = (const unsigned char *)src;
    unsigned char *out = (unsigned char *)dst;
    if (a.row_bytes > ROW_WIDE) {
        const int64_t segs = (a.row_bytes + ROW_SEG - 1) / ROW_SEG, items = a.dense_rows * segs, want = (items + 7) / 8;
        const unsigned grid = (unsigned)(want < MAX_GRID ? want : MAX_GRID);
        const bool two = a.row_bytes <= 1024;              // units per lane
        if (small && items < (int64_t(1) << 30))
            return launch(two ? sym_row_kernel<KIND, ES, 2, unsigned> : sym_row_kernel<KIND, ES, 4, unsigned>, grid, 256, 0, s, in, out, (unsigned)a.d,
                          (unsigned)items, (unsigned)segs, a.row_bytes, a.packed_rows);
        return launch(two ? sym_row_kernel<KIND, ES, 2, int64_t> : sym_row_kernel<KIND, ES, 4, int64_t>, grid, 256, 0, s, in, out, a.d, items, segs,
                      a.row_bytes, a.packed_rows);
    }
    // parts of about 2 KiB (4 KiB of 16-byte words), less where there are too few to fill the chip
    const int64_t words = a.row_bytes / ES, nslices = a.dense_rows / a.d;
    // word by word up to 32 words, and where rows are off 16-byte boundaries up to 128 (positions one by one, in units of 16 bytes
    // put together from two: [384,384,75] 19.3 us, now 15.4; tet d = 160, 33 floats, 284 and 197; d = 60, 33, 18.8 and 11.4); 2-byte
    // words gain nothing ([500,500,99] 23.0 and 24.7)
    const bool flat = words <= (ES >= 4 && ES < 16 && a.row_bytes % 16 != 0 ? 128 : 32);
    int64_t part_rows = words <= 32 ? 256 / words < 8 ? 8 : 256 / words : (2048 + a.row_bytes - 1) / a.row_bytes;
    while (part_rows > 2 && nslices * ((a.d + part_rows - 1) / part_rows) < 16 * (int64_t)sm_count_or_default()) part_rows = (part_rows + 1) / 2;
    const unsigned inv = !flat ? 0u : words == 1 ? 1u : (unsigned)(0xFFFFFFFFu / words + 1);
    const int64_t parts = (a.d + part_rows - 1) / part_rows;
    int shift = 0;
    while (shift < 5 && (int64_t(16) << shift) < a.row_bytes) ++shift;
    const int64_t items = nslices * parts;
    const int64_t want = (items + 7) / 8, cap = (int64_t)sm_count_or_default() * 16;
    const unsigned grid = (unsigned)(want < cap ? want : cap);
    auto run = [&](auto form) {
        constexpr int FORM = decltype(form)::value;
        if (small && items < (int64_t(1) << 31))
            return launch(sym_slice_kernel<KIND, ES, FORM, unsigned>, grid, 256, 0, s, in, out, (unsigned)a.d, (unsigned)nslices, (int)parts,
                          (int)part_rows, (int)a.row_bytes, inv, shift, a.packed_rows);
        return launch(sym_slice_kernel<KIND, ES, FORM, int64_t>, grid, 256, 0, s, in, out, a.d, nslices, (int)parts, (int)part_rows,
                      (int)a.row_bytes, inv, shift, a.packed_rows);
    };
    if constexpr (KIND == ST_TRI_UPPER || ES == 2) return run(std::integral_constant<int, 2>{});
    else return flat ? run(std::integral_constant<int, 1>{}) : run(std::integral_constant<int, 0>{});
}

template <int KIND, int ES, bool PACK>
static st_status launch_copy(const void *src, void *dst, const LayoutArgs &a, cudaStream_t s, const void *mul)
{
    const int64_t cap = MAX_GRID;
    // A block per 16 KB, in one pass: long runs off 16-byte boundaries, that is slices of a matrix; bound by HBM and L2.  A block has the
    // warps that its part needs, as parts of a slice are even: with 256 threads the half-empty blocks of a slice a little longer than
    // 16 KB cost more than the pass saves.  us in rows of calls, blocks that walk 32 KB / one pass with 256 threads / now: pack
    // [384,384,75] 8.2 / 8.6 / 8.0, [2000,2000,3] 8.4 / 11.2 / 8.6, [4100,4100] 13.5 / 20.3 / 12.8, [4000,4000,3] 38.4 / 35.4 / 33.9; times
    // a packed operand 10.9 / 9.7 / 8.9, 10.6 / 13.0 / 9.5, 20.4 / 24.6 / 16.4, 52.2 / 45.2 / 44.0; zero fill 11.7 / 10.9 / 10.6, 12.5 / 14.0 /
    // 11.7, 20.9 / 25.8 / 18.5, 49.9 / 45.7 / 45.1.  Not where runs are short or most parts of a slice empty (pack of a tet d = 160,
    // 33 floats, 52 / 74; 2-byte words [900,900,17] 5.3 / 6.8), nor where all is aligned ([1024,1024,64] doubles 81 / 84).
    constexpr bool ONCE = KIND == ST_TRI_UPPER && (ES == 4 || ES == 8);
    // slices: about four 16-byte units per thread, at most PART_BYTES per (slice, part), less where the slices are too few to
    // fill the chip (one row of [1000,1000,128] in 16 parts 17 us the call with its empty slices, now 1.8).  Pack splits the
    // longest run of unique columns (a band: its packed row), unpack the whole dense slice.
    int64_t run_rows = a.d;
    if (KIND == ST_BAND) run_rows = a.width;
    if (KIND == ST_BLOCKDIAG) run_rows = a.bs;
    if (KIND == ST_FIXED_COL) run_rows = 1;
    const int64_t sb = (PACK ? run_rows : a.d) * a.row_bytes;
    // pack of a tensor of order 3 or 4, or of one row: only the slices that have a run
    const int64_t nslices = PACK && KIND == ST_FIXED_ROW ? 1 : KIND == ST_TET ? (PACK ? tri_rows(a.d) : a.d * a.d) : KIND == ST_SIMPLEX4 ? (PACK ? tet_rows(a.d) : a.d * a.d * a.d) : a.d;
    bool once = false;
    if constexpr (ONCE) once = a.row_bytes % 16 != 0 && sb >= ONCE_BYTES;
    int64_t part_bytes = once ? ONCE_BYTES : PART_BYTES;
    while (!once && part_bytes > 4096 && nslices * ((sb + part_bytes - 1) / part_bytes) < 2 * (int64_t)sm_count_or_default()) part_bytes /= 2;
    int64_t parts = (sb + part_bytes - 1) / part_bytes;
    const int64_t pb = ((sb + parts - 1) / parts + 15) / 16 * 16;
    parts = (sb + pb - 1) / pb;
    if (parts > (int64_t(1) << 30)) return ST_ERR_UNSUPPORTED;
    int shift = 0;
    while ((1 << shift) < 256 && (int64_t(16 * COPY_UNITS) << shift) < pb) ++shift;
    const int64_t nitems = nslices * parts, want = once ? nitems : ((nitems << shift) + 255) / 256;
    constexpr int64_t WARP_BYTES = 32 * 16 * COPY_UNITS;      // of a warp in one pass
    const unsigned threads = once ? (unsigned)((pb + WARP_BYTES - 1) / WARP_BYTES) * 32u : 256u;
    const unsigned grid = (unsigned)(want < cap ? (want < 1 ? 1 : want) : cap);
    const unsigned char *in = (const unsigned char *)src, *m = (const unsigned char *)mul;
    unsigned char *out = (unsigned char *)dst;
    // 32-bit index arithmetic: every index and the intermediate products of the closed forms stay below 2^31
    const bool small = nitems < (int64_t(1) << 30) && a.packed_rows < (int64_t(1) << 31) && a.width < (int64_t(1) << 30) &&
                       a.d <= (KIND == ST_TET ? 1024 : KIND == ST_SIMPLEX4 ? 200 : 20000);
    auto run = [&](auto mul_tag, auto index) {
        typedef decltype(index) I;
        constexpr bool MUL = decltype(mul_tag)::value;
        if constexpr (ONCE)
            if (once)
                return launch(slice_copy_kernel<KIND, ES, PACK, MUL, true, I>, grid, threads, 0, s, in, out, a, (I)nitems, 0, (int)parts, (int)pb, m);
        return launch(slice_copy_kernel<KIND, ES, PACK, MUL, false, I>, grid, 256, 0, s, in, out, a, (I)nitems, shift, (int)parts, (int)pb, m);
    };
    if constexpr (PACK && ES == 4)
        if (mul) return small ? run(std::true_type{}, 0u) : run(std::true_type{}, int64_t(0));
    return small ? run(std::false_type{}, 0u) : run(std::false_type{}, int64_t(0));
}

template <int ES, bool PACK>
static st_status dispatch_kind(const void *src, void *dst, const LayoutArgs &a, cudaStream_t s, const void *mul)
{
    if constexpr (!PACK) {
        if constexpr (ES == 8)
            if (a.fill == ST_FILL_SYMMETRIC && a.row_bytes % 16 == 0)
                return a.kind == ST_TRI_UPPER ? launch_sym<ST_TRI_UPPER, 16>(src, dst, a, s)
                     : a.kind == ST_TET ? launch_sym<ST_TET, 16>(src, dst, a, s) : launch_sym<ST_SIMPLEX4, 16>(src, dst, a, s);
        if (a.fill == ST_FILL_SYMMETRIC)
            return a.kind == ST_TRI_UPPER ? launch_sym<ST_TRI_UPPER, ES>(src, dst, a, s)
                 : a.kind == ST_TET ? launch_sym<ST_TET, ES>(src, dst, a, s) : launch_sym<ST_SIMPLEX4, ES>(src, dst, a, s);
    }
    switch (a.kind) {
    case ST_TRI_UPPER: return launch_copy<ST_TRI_UPPER, ES, PACK>(src, dst, a, s, mul);
    case ST_TET: return launch_copy<ST_TET, ES, PACK>(src, dst, a, s, mul);
    case ST_BAND: return launch_copy<ST_BAND, ES, PACK>(src, dst, a, s, mul);
    case ST_FIXED_ROW: return launch_copy<ST_FIXED_ROW, ES, PACK>(src, dst, a, s, mul);
    case ST_FIXED_COL: return launch_copy<ST_FIXED_COL, ES, PACK>(src, dst, a, s, mul);
    case ST_SIMPLEX4: return launch_copy<ST_SIMPLEX4, ES, PACK>(src, dst, a, s, mul);
    default: return launch_copy<ST_BLOCKDIAG, ES, PACK>(src, dst, a, s, mul);
    }
}

template <bool PACK>
static st_status copy_entry(const st_layout *L, st_dtype dtype, const void *src, void *dst, int fill,
                            void *stream, const void *mul = nullptr)
{
    if (!L || !src || !dst) return ST_ERR_NULL;
    if (!layout_ok(L)) return ST_ERR_SHAPE;
    const int es = dtype_bytes(dtype);
    if (es == 0) return ST_ERR_DTYPE;
    if (fill != ST_FILL_ZERO && fill != ST_FILL_SYMMETRIC) return ST_ERR_UNSUPPORTED;
    if (fill == ST_FILL_SYMMETRIC && L->kind != ST_TRI_UPPER && L->kind != ST_TET && L->kind != ST_SIMPLEX4)
        return ST_ERR_UNSUPPORTED;
    if (!aligned16(src) || !aligned16(dst)) return ST_ERR_ALIGN;
    LayoutArgs a;
    a.kind = L->kind;
    a.fill = fill;
    a.d = L->d; a.kl = L->kl; a.ku = L->ku; a.nb = L->nblocks; a.bs = L->bs;
    a.width = L->kl + L->ku + 1;
    a.packed_rows = packed_rows_of(L);
    a.dense_rows = dense_rows_of(L);
    a.row_bytes = L->inner * es;
    cudaStream_t s = (cudaStream_t)stream;
    // the widest word that divides a position's bytes (the product of st_thp is made word by word)
    if (a.row_bytes % 8 == 0 && !mul) return dispatch_kind<8, PACK>(src, dst, a, s, mul);
    if (a.row_bytes % 4 == 0) return dispatch_kind<4, PACK>(src, dst, a, s, mul);
    return dispatch_kind<2, PACK>(src, dst, a, s, mul);
}

}  // namespace st

extern "C" {

int64_t st_packed_elems(const st_layout *layout)
{
    if (!st::layout_ok(layout)) return -1;
    return st::packed_rows_of(layout) * layout->inner;
}

int64_t st_dense_elems(const st_layout *layout)
{
    if (!st::layout_ok(layout)) return -1;
    return st::dense_rows_of(layout) * layout->inner;
}

st_status st_pack(const st_layout *layout, st_dtype dtype, const void *dense, void *packed, void *stream)
{
    return st::copy_entry<true>(layout, dtype, dense, packed, ST_FILL_ZERO, stream);
}

static st_status packed_binary(int op, int64_t n, const float *a, const float *b, float *out, float alpha, float beta,
                               void *stream)
{
    if (!a || !b || !out) return ST_ERR_NULL;
    if (n <= 0) return ST_ERR_SHAPE;
    if (!st::aligned16(a) || !st::aligned16(b) || !st::aligned16(out)) return ST_ERR_ALIGN;
    // operands that stay in L2: one wave of blocks that walk ([5544000] 6.3 us, a block per 1024 elements 7.4); larger ones in
    // the order of memory ([10^8] 168 us, one wave 183)
    const int64_t want = (n / 4 + 255) / 256, cap = n < (int64_t(1) << 24) ? (int64_t)st::sm_count_or_default() * 16 : st::MAX_GRID;
    const unsigned grid = (unsigned)(want < 1 ? 1 : (want < cap ? want : cap));
    return st::launch(op == 0 ? st::packed_binary_kernel<0> : st::packed_binary_kernel<1>, grid, 256, 0, (cudaStream_t)stream, a, b, out, n, alpha, beta);
}

st_status st_packed_axpby(int64_t n, float alpha, const float *a, float beta, const float *b, float *out, void *stream)
{
    return packed_binary(0, n, a, b, out, alpha, beta, stream);
}

st_status st_packed_mul(int64_t n, const float *a, const float *b, float *out, void *stream)
{
    return packed_binary(1, n, a, b, out, 0.f, 0.f, stream);
}

st_status st_thp(const st_layout *layout, const float *Bp, const float *C_dense, float *Ap, void *stream)
{
    if (!Bp) return ST_ERR_NULL;
    if (!st::aligned16(Bp)) return ST_ERR_ALIGN;
    // the pack of C with every gathered value multiplied by the packed operand at the same position
    return st::copy_entry<true>(layout, ST_F32, C_dense, Ap, ST_FILL_ZERO, stream, Bp);
}

st_status st_unpack(const st_layout *layout, st_dtype dtype, const void *packed, void *dense, st_fill fill,
                    void *stream)
{
    return st::copy_entry<false>(layout, dtype, packed, dense, (int)fill, stream);
}

}  // extern "C"
