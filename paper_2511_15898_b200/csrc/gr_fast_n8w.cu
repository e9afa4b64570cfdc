// Fast solve kernels for series length 8 with more threads per instance, for batches that leave SMs idle (gr_fast.cu).
#include "gr_fast.cuh"

namespace gr {
namespace fast {
GR_FAST_INSTANTIATE(n8_m32w, 8, 32, 128, 16, 2)
GR_FAST_INSTANTIATE(n8_m64w, 8, 64, 256, 14, 1)
GR_FAST_INSTANTIATE(n8_m128w, 8, 128, 256, 8, 1)
}  // namespace fast
}  // namespace gr
