// Which kernel takes a convolution of the surrogate network, and with how many
// blocks: plain host arithmetic on sizes.
#pragma once
#include <algorithm>

namespace cnok {

// CTAs per output block of a kernel that holds one CTA per SM and goes through its
// tiles (conv64_kernel, which keeps its block's weights, and conv_halo_kernel): all
// output blocks share the SMs, so that no CTA waits for another one's SM and loads
// again what that one held.  conv64_kernel with a CTA per SM for each block: 64 -> 192
// channels 13.2 us at 128^2 and 41.8 at 8 x 128^2, 64 -> 320 at 128^2 21.2; now 8.1,
// 37.4 and 11.2.
inline int persistent_ctas(long long tiles, int nblocks, int sms)
{
    return (int)std::min<long long>(tiles, std::max(1, sms / nblocks));
}

// A 3x3 convolution of n images of h x w pixels, cin -> cout channels: bf16 results (slope:
// times the slope of an activation), or the head (FP32, at most 16 of 64 channels stored).
struct ConvForm {
    long long n, h, w;
    int cin, cout;
    bool slope, head;
};
enum ConvKernel { CONV_FPROP, CONV_64, CONV_HALO };

// Tiles of 128 pixels in a row (conv_fprop_kernel; of whole rows where they are
// shorter), and of 8 x 16 pixels (the other two).
inline long long row_tiles(const ConvForm &f)
{
    const long long wt = std::min(f.w, 128LL), ht = 128 / wt;
    return f.n * ((f.w + wt - 1) / wt) * ((f.h + ht - 1) / ht);
}
inline long long halo_tiles(const ConvForm &f) { return f.n * ((f.w + 7) / 8) * ((f.h + 15) / 16); }

// The faster kernel where several can take it: conv64_kernel takes 64 input channels to
// 64, 192, ... output channels and the head, conv_halo_kernel 64 or 128 to a multiple of
// 128.  Their tiles are cheaper than conv_fprop_kernel's but hold less where a height is
// not whole sixteens: the limits are on their number for one of conv_fprop_kernel's.
// Measured at 64 x h x 256 (us, conv_fprop_kernel / these), heights 16, 14, 12, 11
// (1.0, 1.14, 1.33, 1.45 tiles to one), and the data gradients with slopes below:
//   64 -> 64     30.4/26.7   27.1/26.0   23.8/25.9   22.6/25.7
//                36.2/27.6   31.4/27.0   27.8/26.3   26.1/25.8
//   64 -> 192    89.2/70.6   79.6/69.9   68.1/69.7   64.0/69.5
//               115.8/70.6  102.2/69.9   88.1/69.6   82.4/69.4
//   64 -> 128    47.4/32.2   40.7/31.3   36.8/30.9   34.1/30.8
//                59.8/44.0   52.4/42.7   47.5/41.8   43.0/41.1
//   128 -> 128   70.8/63.0   62.2/62.8   56.2/62.0   50.4/61.5
//                82.5/64.5   72.0/63.7   67.3/63.2   60.5/63.0
//   128 -> 384   206.7/172.4 183.4/172.0 161.4/171.2 145.6/171.4
//                250.8/176.6 222.7/174.9 195.6/174.1 176.8/173.7
//   128 -> 256   114.2/115.6 98.8/115.2  89.9/114.8  82.4/114.7
//                139.8/118.4 121.3/117.6 110.0/116.8 101.2/116.4
//   head         23.1/24.3   21.1/24.0   18.5/23.8   17.9/23.8
// Up to one tile a CTA a tile's latency counts, and theirs is shorter (7 x 129, 1.2 tiles
// to one: 64 -> 64 6.1/5.0, head 5.6/4.3, 128 -> 128 9.5/7.8, 128 -> 384 10.3/7.7).
// An MMA of the head takes as long for its 16 columns as for 64: with many tiles it pays only where
// they are fewer (1024^2 80.6/86.4, 256^2 9.9/8.6).  128 -> 256, 512, ... stand against
// tiles of 256 channels, one CTA per SM, so how the last wave is filled decides, and
// waves are compared: one of that kernel takes as long as two of this one, 2.3 with
// slopes (256^2, 4 waves to 7: 34.3/32.5; 128^2, 1 to 2: 11.7/12.2).
inline ConvKernel choose_conv(const ConvForm &f, int sms)
{
    const long long rows = row_tiles(f), tiles = halo_tiles(f);
    const bool few = tiles <= 7LL * sms;
    const bool wide = f.cout % 128 == 0;  // output blocks of 128 channels, else of 64
    if (f.cin > (wide ? 128 : 64) || (f.head && wide))
        return CONV_FPROP;
    if (tiles * (f.cout / (wide ? 128 : 64)) <= sms)  // one tile a CTA
        return tiles <= 1.4 * rows ? (wide ? CONV_HALO : CONV_64) : CONV_FPROP;
    if (!wide) {
        const double most = f.head ? (few ? 1.1 : 0.95) : f.slope ? 1.4 : f.cout == 64 ? 1.15 : few ? 1.4 : 1.25;
        return tiles <= most * rows ? CONV_64 : CONV_FPROP;
    }
    if (f.cin == 64 || f.cout % 256 != 0) {
        const double most = f.cin == 64 ? 1.4 : f.cout == 128 ? (f.slope ? 1.25 : 1.12) : (f.slope ? 1.4 : few ? 1.25 : 1.2);
        return tiles <= most * rows ? CONV_HALO : CONV_FPROP;
    }
    const long long per_block = persistent_ctas(tiles, f.cout / 128, sms);
    const long long waves = (tiles + per_block - 1) / per_block, others = (rows * (f.cout / 256) + sms - 1) / sms;
    return f.slope ? (10 * waves <= (f.cout == 256 ? 23 : 24) * others ? CONV_HALO : CONV_FPROP)
                   : (waves < 2 * others ? CONV_HALO : CONV_FPROP);
}

}  // namespace cnok
