// step_1_5_5.cu -- the Eq. 7 step's kernels for radius (1, 5, 5).
#include "iter_stream.cuh"
#include "iter_tile.cuh"

namespace sfseg {

bool stream_step_1_5_5(const StepArgs& a) { return step_dispatch<stream::Kernel<1, 5, 5>>(a); }
bool tile_step_1_5_5(const StepArgs& a) { return step_dispatch<tile::Kernel<1, 5, 5>>(a); }

}  // namespace sfseg
