// The block sweep for items of 5 score slots.
#include "cfr_block_impl.cuh"

namespace pasur {
const void *block_kernel_w5(int variant) { return block_kernel_of<5>(variant); }
}  // namespace pasur
