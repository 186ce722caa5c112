// Iteration kernels for __nv_bfloat16 level storage, window radii 1..10, for a chain
// of launches on one stream (one pair).
#include "k_block_inst.cuh"

namespace ofv {

OFV_INSTANTIATE_BLOCK(__nv_bfloat16, ITER_CHAIN)

}  // namespace ofv
