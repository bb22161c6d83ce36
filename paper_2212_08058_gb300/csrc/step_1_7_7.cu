// step_1_7_7.cu -- the Eq. 7 step's kernels for radius (1, 7, 7).
#include "iter_stream.cuh"
#include "iter_tile.cuh"

namespace sfseg {

bool stream_step_1_7_7(const StepArgs& a) { return step_dispatch<stream::Kernel<1, 7, 7>>(a); }
bool tile_step_1_7_7(const StepArgs& a) { return step_dispatch<tile::Kernel<1, 7, 7>>(a); }

}  // namespace sfseg
