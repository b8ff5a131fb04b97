// Which plans the kernel of small plans encodes (lq_quantize_small.cu), and with how many CTAs a (layer, worker): plain C++, from the
// plan's sizes and from how many clusters run at once on the device.
#pragma once

#include <cstdint>

namespace lq {

constexpr int kSmallRanks = 16, kSmallShare = 13;            // most CTAs of a cluster (more than 8 have to be asked for), most blocks of a CTA

// clusters[i]: how many clusters of 2^i CTAs run at once; 0 where the device has none of that size.
struct ClusterRoom { int32_t clusters[5]; };

// CTAs of a plan's clusters, or 0: the general path.  pairs: layers x workers; most_blocks: blocks of the largest layer.
// It asks for nothing of a call: neither a worker range nor a histogram changes which kernel encodes
// a layer, nor the order in which the layer's sums are formed.
//
// CTAs: as many as the largest layer needs for 8 blocks each, up to 8, and more, while there are blocks for them and SMs (2
// CTAs on each): 784 blocks of 203 530 coordinates and 4 workers on 8 CTAs each 27.7, on 16 20.5 us.
// The rule: layers of up to 8 blocks of 1024 coordinates, a CTA each, always; larger ones while a CTA has at most 13 blocks and the
// clusters at most 444 CTAs (3 on each SM).
// The step in us, this kernel and the general path.  One CTA a layer: layers of one block, 80 (layer, worker) pairs 13 and 20, 2400 of them
// 38 and 46, 9600 128 and 153; of 1 to 8 blocks, 2400 pairs 58 and 64, 4896 111 and 129.  Clusters of up to 8 blocks a CTA: 160 CTAs
// 12 and 18, 320 15 and 20, 640 20.4 and 19.6, 1280 31 and 24.  256 CTAs of 13 blocks 19 and 22, 128 of 16 26 and 23, 288 of 24 27 and 24.
inline int small_plan_ranks(int64_t pairs, int64_t num_layers, int64_t most_blocks, int sms, const ClusterRoom& room)
{
    if (num_layers < 1 || num_layers > 65535) return 0;      // (grid.y)
    int r = 1, i = 0;
    while (r < 8 && r * 8 < most_blocks) { r *= 2; ++i; }
    while (r < kSmallRanks && r < most_blocks && pairs * 2 * r <= 2 * sms) { r *= 2; ++i; }
    while (i > 0 && room.clusters[i] == 0) { r /= 2; --i; }  // (a part of a GPU, say: clusters have to lie in one group of its SMs)
    const bool fits = room.clusters[i] > 0 && pairs * r <= 3 * sms && most_blocks <= r * kSmallShare;
    return fits ? r : most_blocks <= 8 ? 1 : 0;
}

}  // namespace lq
