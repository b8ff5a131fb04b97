// Which plans the kernel of small plans encodes (lq_quantize_small.cu), and with how many CTAs a (layer, worker): plain C++, from the
// plan's sizes and from how many clusters run at once on the device.
#pragma once

#include <cstdint>

namespace lq {

constexpr int kSmallRanks = 16, kSmallShare = 13;            // most CTAs of a cluster (more than 8 have to be asked for), most blocks of a CTA

// clusters[i]: how many clusters of 2^i CTAs run at once; 0 where the device has none of that size.
struct ClusterRoom { int32_t clusters[5]; };

// CTAs of a plan's clusters, or 0: the general path.  pairs: layers x workers; most_blocks: blocks of the largest layer; blocks: of
// all layers and workers.  It asks for nothing of a call: neither a worker range nor a histogram changes which kernel encodes
// a layer, nor the order in which the layer's sums are formed.
//
// CTAs: as many as the largest layer needs for 8 blocks each, up to 8, and more, while there are blocks for them and SMs (2
// CTAs on each): 784 blocks of 203 530 coordinates and 4 workers on 8 CTAs each 27.7, on 16 20.5 us.
// Layers of up to 8 blocks, a CTA each, are always small.  The step in us, the small kernel and the general path: layers of one block, 80
// pairs 13 and 20, 2400 of them 38 and 46, 9600 128 and 153; of 1 to 8 blocks, 2400 pairs 58 and 64, 4896 111 and 129.
// Clusters have to run at once, since the ones of a second wave wait for whole clusters.  8 blocks a CTA: 222 clusters of 2 22.2 and
// 27.1, 240 26.7 and 24.1; 100 of 4 22.0 and 27.2, 104 22.8 and 24.5, 111 36.0 and 32.9; 46 of 8 22.8 and 27.1, 48 24.9 and
// 25.1, 50 30.0 and 27.6.
// Blocks of a CTA: up to 13 (13, then 14 of them: 160 CTAs of clusters of 8 23.8 and 23.7, 24.9 and 24.1; 296 33.6 and 34.5, 35.3 and
// 35.7; 64 of clusters of 16 at 8 bits 25.9 and 24.8, 27.6 and 23.2; one large layer beside three of 1 to 3 blocks, 4 workers, 19.9
// and 21.3, 20.5 and 20.5), or 12 in clusters of 16 and plans of more than 1024 blocks (12, then 13: 128 CTAs 22.7 and 22.9, 24.0 and
// 20.8; 256 CTAs 24.2 and 24.7, 25.6 and 24.8).  With a histogram the line would lie at 9 to 12; the calls with one are few.
inline int small_plan_ranks(int64_t pairs, int64_t num_layers, int64_t most_blocks, int64_t blocks, int sms, const ClusterRoom& room)
{
    if (num_layers < 1 || num_layers > 65535) return 0;      // (grid.y)
    int r = 1, i = 0;
    while (r < 8 && r * 8 < most_blocks) { r *= 2; ++i; }
    while (r < kSmallRanks && r < most_blocks && pairs * 2 * r <= 2 * sms) { r *= 2; ++i; }
    while (i > 0 && room.clusters[i] == 0) { r /= 2; --i; }  // (a part of a GPU, say: clusters have to lie in one group of its SMs)
    const bool fits = pairs <= room.clusters[i] && most_blocks <= r * (r == 16 && blocks > 1024 ? 12 : kSmallShare);
    return fits ? r : most_blocks <= 8 ? 1 : 0;
}

}  // namespace lq
