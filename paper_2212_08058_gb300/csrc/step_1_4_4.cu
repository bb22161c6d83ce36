// step_1_4_4.cu -- the Eq. 7 step's kernels for radius (1, 4, 4).
#include "iter_stream.cuh"
#include "iter_tile.cuh"

namespace sfseg {

bool stream_step_1_4_4(const StepArgs& a) { return step_dispatch<stream::Kernel<1, 4, 4>>(a); }
bool tile_step_1_4_4(const StepArgs& a) { return step_dispatch<tile::Kernel<1, 4, 4>>(a); }

}  // namespace sfseg
