// step_1_3_3.cu -- the Eq. 7 step's kernels for radius (1, 3, 3).
#include "iter_stream.cuh"
#include "iter_tile.cuh"

namespace sfseg {

bool stream_step_1_3_3(const StepArgs& a) { return step_dispatch<stream::Kernel<1, 3, 3>>(a); }
bool tile_step_1_3_3(const StepArgs& a) { return step_dispatch<tile::Kernel<1, 3, 3>>(a); }

}  // namespace sfseg
