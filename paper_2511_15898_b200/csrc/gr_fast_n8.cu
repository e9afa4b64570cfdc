// Fast solve kernels for series length 8 (draft counts up to 8).  Batches that fill the chip: 16 quadrature nodes handled together (few
// instances have more) and four staged at a time leave room for the first-level cache, which the calls' spills live in (600 rows of k = 128 254 -> 249 us a call,
// 1024 of k = 20 93.9 -> 93.5, 1024 headline rows within 1 %).  Five or six CTAs of 96 or 80 registers lose 15 to 40 % to spills, eight CTAs of two warps 20 %.
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(n8_m32, 8, 32, 64, 8, 8, 16)
GR_FAST_INSTANTIATE(n8_m64, 8, 64, 128, 4, 4, 16)
GR_FAST_INSTANTIATE(n8_m128, 8, 128, 256, 4, 2, 16)
}  // namespace fast
}  // namespace gr
