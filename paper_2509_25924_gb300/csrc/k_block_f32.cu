// Iteration kernels for float level storage, window radii 1..10: the
// estimator as read from Sec. 2, one tile per CTA and batched.
#include "k_block_inst.cuh"

namespace ofv {

OFV_INSTANTIATE_BLOCK(float, ITER_BOX)
OFV_INSTANTIATE_QUEUE(float, ITER_BOX)

}  // namespace ofv
