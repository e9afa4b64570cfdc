// Fast solve kernels for series length 16 (draft counts up to 16).  Threads and CTAs per SM, with 16 quadrature nodes handled together (32 in the wide
// variants; the room is worth more than a second pass of the few instances that have more nodes).  Supports of up to 128 tokens: three CTAs of 128 threads
// without spills, or two of 256 with some where these hold the batch and its slowest instance sets the time (50 random shapes of 149 to 296 rows 7 % faster;
// 281 rows of n = 15, k = 104 191 -> 184 us, 206 of n = 10, k = 75 221 -> 193, 255 of n = 10, k = 80 with a dominant token 1131 -> 873); beyond, 60
// random shapes of 200 to 4000 rows are 1 % slower in two of 256, each between 22 % slower and 20 % faster (1024 rows of k = 100 with a dominant token
// 368 -> 298 us, 3505 of n = 16, k = 95 538 -> 687).  Up to 32 tokens four CTAs of 128 threads while they hold the batch (512 rows, k = 20: 92.8 us a
// call, 97.4 at three), eight of 64 beyond (1777 rows, k = 5: 140.6 us a call for 149.9 at six).  At 64 tokens four of 128 (600 rows of n = 12, k = 50,
// fused: 180 -> 171 us with the smaller arrays); eight of 64 are as fast in full batches only.
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(n16_m32, 16, 32, 64, 4, 8, 16)
GR_FAST_INSTANTIATE(n16_m32h, 16, 32, 128, 6, 4, 16)
GR_FAST_INSTANTIATE(n16_m64, 16, 64, 128, 4, 4, 16)
GR_FAST_INSTANTIATE(n16_m128, 16, 128, 128, 4, 3, 16)
GR_FAST_INSTANTIATE(n16_m128h, 16, 128, 256, 4, 2, 16)
}  // namespace fast
}  // namespace gr
