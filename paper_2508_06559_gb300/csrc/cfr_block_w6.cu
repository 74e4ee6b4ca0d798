// The block sweep for items of 6 score slots.
#include "cfr_block_impl.cuh"

namespace pasur {
const void *block_kernel_w6(int variant) { return block_kernel_of<6>(variant); }
}  // namespace pasur
