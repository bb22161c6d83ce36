// step_1_2_2.cu -- the Eq. 7 step's kernels for radius (1, 2, 2).
#include "iter_stream.cuh"
#include "iter_tile.cuh"

namespace sfseg {

bool stream_step_1_2_2(const StepArgs& a) { return step_dispatch<stream::Kernel<1, 2, 2>>(a); }
bool tile_step_1_2_2(const StepArgs& a) { return step_dispatch<tile::Kernel<1, 2, 2>>(a); }

}  // namespace sfseg
