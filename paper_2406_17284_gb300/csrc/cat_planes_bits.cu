// The bit-plane box-sum kernels (cat_planes.cuh), one bit per cell.
#include "cat_planes.cuh"

namespace cat {
namespace planes {

Kernel kernel_bit1(int r) { return find_kernel<CAT_STORE_BIT1, CAT_STORE_BIT1, false>(r); }

}  // namespace planes
}  // namespace cat
