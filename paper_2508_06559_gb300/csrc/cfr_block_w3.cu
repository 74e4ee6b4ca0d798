// The block sweep for items of 3 score slots.
#include "cfr_block_impl.cuh"

namespace pasur {
const void *block_kernel_w3(int variant) { return block_kernel_of<3>(variant); }
}  // namespace pasur
