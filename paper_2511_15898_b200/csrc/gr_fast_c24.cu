// Fast solve kernels for 17 to 32 drafts: [lambda^n] from up to 24 conjugate pairs of points on a circle.
// (c24_m32: four CTAs per SM by registers and, with three Hessian nodes staged at a time, by shared memory: 55 KB each.  With four
// nodes three CTAs fitted: 512 instances in two waves, 157 us; now 113.)
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(c24_m32, 24, 32, 128, 3, 4)
GR_FAST_INSTANTIATE(c24_m32w, 24, 32, 128, 8, 2)
GR_FAST_INSTANTIATE(c24_m64, 24, 64, 256, 4, 2, 16)
GR_FAST_INSTANTIATE(c24_m128, 24, 128, 256, 4, 1, 16)
}  // namespace fast
}  // namespace gr
