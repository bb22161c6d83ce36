// step_2_8_8.cu -- the Eq. 7 step's kernels for radius (2, 8, 8).
#include "iter_stream.cuh"
#include "iter_tile.cuh"

namespace sfseg {

bool stream_step_2_8_8(const StepArgs& a) { return step_dispatch<stream::Kernel<2, 8, 8>>(a); }
bool tile_step_2_8_8(const StepArgs& a) { return step_dispatch<tile::Kernel<2, 8, 8>>(a); }

}  // namespace sfseg
