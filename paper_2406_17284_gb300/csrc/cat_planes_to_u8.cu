// The bit-plane box-sum kernels (cat_planes.cuh), two states, from one bit per cell to uint8.
#include "cat_planes.cuh"

namespace cat {
namespace planes {

Kernel kernel_bit1_to_u8(int r) { return find_kernel<CAT_STORE_BIT1, CAT_STORE_U8, false>(r); }

}  // namespace planes
}  // namespace cat
