// step_2_5_5.cu -- the Eq. 7 step's kernels for radius (2, 5, 5).
#include "iter_stream.cuh"
#include "iter_tile.cuh"

namespace sfseg {

bool stream_step_2_5_5(const StepArgs& a) { return step_dispatch<stream::Kernel<2, 5, 5>>(a); }
bool tile_step_2_5_5(const StepArgs& a) { return step_dispatch<tile::Kernel<2, 5, 5>>(a); }

}  // namespace sfseg
