// The tiled bit-plane kernels (cat_planes_tile.cuh).
#include "cat_planes_tile.cuh"

namespace cat {
namespace planes {

TileKernel tile_kernel(int r) { return find_tile_kernel<>(r); }

}  // namespace planes
}  // namespace cat
