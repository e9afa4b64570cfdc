// Fast solve kernels for series length 16 (draft counts up to 16).
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(n16_m32, 16, 32, 64, 4, 6)
GR_FAST_INSTANTIATE(n16_m64, 16, 64, 128, 4, 4)
GR_FAST_INSTANTIATE(n16_m128, 16, 128, 128, 4, 3)
}  // namespace fast
}  // namespace gr
