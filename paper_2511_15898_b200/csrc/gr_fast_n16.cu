// Fast solve kernels for series length 16 (draft counts up to 16).  Threads and CTAs per SM: supports of up to 128 tokens ran
// 7 % faster on two CTAs of 256 threads than on three of 128 (4096 rows, k = 100: 1480 to 1378 us).  Up to 32 tokens four CTAs
// of 128 threads are no slower while they hold the batch (512 rows, k = 20: 155 us a call for 160, fused 156 for 156), six of 64
// faster beyond (1777 rows, k = 8: 267 us a call for 310).  At 64 tokens, where two CTAs of 256 for four of 128 lost a third at series length 8, the narrow ones stay.
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(n16_m32, 16, 32, 64, 4, 6)
GR_FAST_INSTANTIATE(n16_m32h, 16, 32, 128, 4, 4)
GR_FAST_INSTANTIATE(n16_m64, 16, 64, 128, 4, 4)
GR_FAST_INSTANTIATE(n16_m128, 16, 128, 256, 4, 2)
}  // namespace fast
}  // namespace gr
