// Which form of the register-tile second moment (moment2_small.cu) few samples take.
#pragma once
#include <cstdint>

namespace st {

constexpr int M2S_CLUSTER = 16;            // one-launch form: blocks of a cluster

// One launch instead of two: the partial sums are added inside clusters of 16 blocks.  It saves about 2 us of the host's time per
// call and the second kernel, but its blocks are fewer, and every cluster reads all of X.  What decides is the number of
// samples per thread (rg row groups in each of the 16 blocks) against the work items of the whole triangle, which the two
// launches write and add per SM.  On the GPU (us, one launch / two):
//   rows copied whole: [16384,8] 5.0 / 5.7, [30000,8] 6.8 / 6.0, [8192,16] 5.4 / 6.2, [16384,16] 6.4 / 6.2, [4096,24] 5.4 / 5.8,
//     [6000,24] 6.2 / 5.7, [4096,64] 7.0 / 7.6, [8192,64] 8.5 / 8.9, [16384,64] 11.9 / 9.7;
//   word by word, where a thread's copies weigh more: [2000,33] 6.0 / 6.6, [3000,33] 7.1 / 6.6, [1000,75] 6.7 / 8.2,
//     [2000,75] 8.6 / 8.3;
//   more clusters than the chip runs at once: [4096,100] 9.2 / 11.8, [6000,100] 17.0 / 13.5, [3000,120] 9.3 / 13.0,
//     [4096,120] 16.4 / 14.2.
// fit: clusters that can be active at once.  None (a context with fewer than 16 SMs in any group): two launches.
inline bool m2s_use_cluster(int64_t N, int items, int clusters, int rg, bool bulk, int fit)
{
    if (fit <= 0) return false;
    double most = !bulk ? 5 : items < 3 ? 8.2 : 6 + 0.8 * items;
    if (clusters > fit && most > 16) most = 16;
    return (double)N <= most * M2S_CLUSTER * rg;
}

}  // namespace st
