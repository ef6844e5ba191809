// at_items.cuh -- which of a launch's items (subdomains, tiles) each processing
// element owns.  Plain arithmetic, for host and device code.
#pragma once

#ifdef __CUDACC__
#define AT_ITEMS_FN __host__ __device__ __forceinline__
#else
#define AT_ITEMS_FN inline
#endif

namespace atk {

struct ItemRange {
    long long lo, hi;
};

// The contiguous run of `total` items that processor e of n owns: runs differ by
// one item at most, the last processors have the longer ones.  With a persistent
// grid of 152 SMs the CTAs that share an SM were seen 148 apart in the launch
// order, but for the first 4 x occupancy of them, which filled 4 SMs by themselves;
// so consecutive CTAs with one item more land on different SMs, if they are not the
// first ones.  Cut at e total / n instead, the CTAs of an SM nearly all had the
// longer run or none of them.  Before and now: 384 x 256 x 288 in 864 subdomains on
// 608 CTAs, 40 seeded levels 2748 -> 2655 us; 2^22 FP64 points in 4096 subdomains on
// 1216 warps, 40 levels 3632 -> 3544; with the first processors longer 2872 and 4010.
AT_ITEMS_FN ItemRange item_range(long long total, long long n, long long e)
{
    const long long q = total / n, few = n - (total - q * n);      // processors with q items
    return ItemRange{e * q + (e > few ? e - few : 0), (e + 1) * q + (e + 1 > few ? e + 1 - few : 0)};
}

// The items of element w (of W) of CTA g (of G).  With fewer items than elements,
// every CTA's first element comes before any CTA's second one, and the CTAs' counts
// differ by one at most: few items share no SM's pipes while other SMs idle.
// (Counted CTA by CTA, the last total / W CTAs had W items each and the others none:
// 600 subdomains of 1000 FP64 points on 456 CTAs took 23.8 us a level, 12.8 so.)
AT_ITEMS_FN ItemRange cta_items(long long total, long long G, int W, long long g, int w)
{
    const long long n = G * W;
    return item_range(total, n, total >= n ? g * W + w : (W - 1 - w) * G + g);
}

}  // namespace atk
