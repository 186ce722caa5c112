// Iteration kernels for __half level storage, window radii 1..10, with the
// estimator variants (increment form, Gaussian window, region mask), and the
// form that keeps the window sums for the reverse mode.
#include "k_block_inst.cuh"

namespace ofv {

OFV_INSTANTIATE_BLOCK(__half, ITER_KEEP)
OFV_INSTANTIATE_BLOCK(__half, ITER_VAR)
OFV_INSTANTIATE_QUEUE(__half, ITER_VAR)

}  // namespace ofv
