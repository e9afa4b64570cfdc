// Fast solve kernels for series length 16 with more threads per instance, for batches that leave SMs idle (gr_fast.cu).
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(n16_m32w, 16, 32, 128, 8, 2)
GR_FAST_INSTANTIATE(n16_m64w, 16, 64, 256, 8, 1)
GR_FAST_INSTANTIATE(n16_m128w, 16, 128, 256, 6, 1)
}  // namespace fast
}  // namespace gr
