// Fast solve kernels for series length 4 (draft counts up to 4).
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(n4_m32, 4, 32, 64, 8, 8)
GR_FAST_INSTANTIATE(n4_m64, 4, 64, 64, 8, 7)
GR_FAST_INSTANTIATE(n4_m32w, 4, 32, 128, 16, 2)
GR_FAST_INSTANTIATE(n4_m64w, 4, 64, 256, 16, 1)
}  // namespace fast
}  // namespace gr
