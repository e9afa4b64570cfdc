// Fast solve kernels for series length 8 (draft counts up to 8).
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(n8_m32, 8, 32, 64, 8, 8)
GR_FAST_INSTANTIATE(n8_m64, 8, 64, 128, 6, 4)
GR_FAST_INSTANTIATE(n8_m128, 8, 128, 256, 4, 2)
}  // namespace fast
}  // namespace gr
