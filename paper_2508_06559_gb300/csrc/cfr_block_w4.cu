// The block sweep for items of 4 score slots.
#include "cfr_block_impl.cuh"

namespace pasur {
const void *block_kernel_w4(int variant) { return block_kernel_of<4>(variant); }
}  // namespace pasur
