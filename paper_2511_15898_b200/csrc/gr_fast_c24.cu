// Fast solve kernels for 17 to 32 drafts: [lambda^n] from up to 24 conjugate pairs of points on a circle.
// (c24_m32: 128 registers allow four CTAs per SM, its 58016 bytes of shared memory three.)
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(c24_m32, 24, 32, 128, 4, 4)
GR_FAST_INSTANTIATE(c24_m64, 24, 64, 256, 4, 2)
GR_FAST_INSTANTIATE(c24_m128, 24, 128, 256, 2, 1)
}  // namespace fast
}  // namespace gr
