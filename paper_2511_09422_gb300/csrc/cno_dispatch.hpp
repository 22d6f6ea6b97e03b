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

}  // namespace cnok
