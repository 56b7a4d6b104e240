// Instantiations of the forward projector whose table build gives a warp four quads of slabs.
#include "project_kernel.cuh"

namespace cbct {

template const void *project_kernel<4>(int, int, int, int);

} // namespace cbct
