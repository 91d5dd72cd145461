// The bit-plane box-sum kernels (cat_planes.cuh), one byte per cell, two states.
#include "cat_planes.cuh"

namespace cat {
namespace planes {

Kernel kernel_u8(int r) { return find_kernel<CAT_STORE_U8, CAT_STORE_U8, false>(r); }

}  // namespace planes
}  // namespace cat
