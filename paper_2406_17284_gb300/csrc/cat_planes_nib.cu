// The bit-plane box-sum kernels (cat_planes.cuh), four bits per cell.
#include "cat_planes.cuh"

namespace cat {
namespace planes {

Kernel kernel_nib4(int r) { return find_kernel<CAT_STORE_NIB4, CAT_STORE_NIB4, true>(r); }

}  // namespace planes
}  // namespace cat
