// Fast solve kernels for series length 16 (draft counts up to 16).  Threads and CTAs per SM, with 16 quadrature nodes handled together (32 in the wide
// variants; the room is worth more than a second pass of the few instances that have more nodes): supports of up to 128 tokens on three CTAs of 128 threads,
// without the spills of two of 256 (1024 rows, k = 100, solve call 349 us for 355).  Up to 32 tokens four CTAs of 128 threads while they hold the
// batch (512 rows, k = 20: 92.8 us a call, 97.4 at three), eight of 64 beyond (1777 rows, k = 5: 140.6 us a call for 149.9 at six).  At 64 tokens
// four of 128 (600 rows of n = 12, k = 50, fused: 180 -> 171 us with the smaller arrays); eight of 64 are as fast in full batches only.
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(n16_m32, 16, 32, 64, 4, 8, 16)
GR_FAST_INSTANTIATE(n16_m32h, 16, 32, 128, 6, 4, 16)
GR_FAST_INSTANTIATE(n16_m64, 16, 64, 128, 4, 4, 16)
GR_FAST_INSTANTIATE(n16_m128, 16, 128, 128, 4, 3, 16)
}  // namespace fast
}  // namespace gr
