// How a flat copy of n bytes to `dst` is cut into whole 16-byte units of dst and single elements in front of and behind them.
#pragma once
#include "st_index.cuh"

namespace st {

struct CopySpan {
    int head, units, ends;     // bytes in front of the first unit; units; bytes of the elements on either side together
    unsigned off;              // the source of the first unit from the 16-byte boundary in front of it
};

// A unit whose source is off a boundary is taken from the two aligned units that hold it.  Where the second of the last one
// reaches past `end`, the end of the source array, its elements are copied singly: nothing behind the array is read.
ST_HD CopySpan copy_span(uintptr_t dst, uintptr_t src, int n, uintptr_t end)
{
    CopySpan c;
    c.head = (int)((0u - (unsigned)dst) & 15u);
    if (c.head > n) c.head = n;
    c.units = (n - c.head) >> 4;
    c.off = (unsigned)(src + c.head) & 15u;
    if (c.units > 0 && c.off != 0 && src + c.head - c.off + 16 * ((uintptr_t)c.units + 1) > end) --c.units;
    c.ends = n - (c.units << 4);
    return c;
}

}  // namespace st
