// Shapes and work-item dealing shared by the tcgen05 kernels.
#pragma once

namespace mgn {

// Shapes: q, o, d_o, dq [BH = B*H, Sq, D]; k, v, dk, dv [B*H/G, Sk, D]; query head h reads
// key/value head h / G; causal: key j is visible to query i iff j <= i + off, off = Sk - Sq >= 0.
struct Dims {
    int Sq, Sk, BH, H, G, off;
    int Sp = 0;      // forward: rows of a head within the Sq rows of a packed one (Sq where heads are not packed)
};

// k-th item of CTA c out of G, -1 past the end (then also for every larger k).
//   order 0 (block-major): tiers of G items, odd tiers dealt backwards (snake);
//   order 1 (head-major):  CTA c takes the consecutive item pairs c, c+G, c+2G, ...
__device__ __forceinline__ int item_index(int c, int k, int G, int n_items, int order) {
    const int it = order == 0 ? k * G + ((k & 1) ? (G - 1 - c) : c) : 2 * (c + G * (k >> 1)) + (k & 1);
    return it < n_items ? it : -1;
}

// CTA -> (tile in order of falling weight, head).  Heads come in groups whose streamed tensors stay in L2 while the
// group's CTAs run; within a group every head's heaviest tile comes first.
__device__ __forceinline__ void item_of_block(int block, int n_tiles, int heads, int group, int& tile, int& head) {
    const int g = block / (n_tiles * group), rem = block - g * n_tiles * group;
    const int size = min(group, heads - g * group);
    tile = rem / size;
    head = g * group + rem % size;
}
// `bytes`: what the CTAs of one head share.  One group while everything fits half of L2; else a quarter of L2 a
// group, equal groups ((4,32,1024,128) causal forward 0.282 -> 0.261 ms; its K and V are 134 MB).
inline int head_group(double bytes, int heads) {
    int dev = 0, l2 = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev) != cudaSuccess || l2 <= 0)
        l2 = 126 << 20;
    if (bytes * heads <= 0.5 * l2) return heads;
    const double n = 0.25 * l2 / bytes;
    const int most = n < 1.0 ? 1 : static_cast<int>(n), groups = (heads + most - 1) / most;
    return (heads + groups - 1) / groups;
}

}  // namespace mgn
