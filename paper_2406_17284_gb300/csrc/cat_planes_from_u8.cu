// The bit-plane box-sum kernels (cat_planes.cuh), two states, from uint8 to one bit per cell.
#include "cat_planes.cuh"

namespace cat {
namespace planes {

Kernel kernel_u8_to_bit1(int r) { return find_kernel<CAT_STORE_U8, CAT_STORE_BIT1, false>(r); }

}  // namespace planes
}  // namespace cat
