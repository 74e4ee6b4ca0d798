// The block sweep for items of 1 score slot.
#include "cfr_block_impl.cuh"

namespace pasur {
const void *block_kernel_w1(int variant) { return block_kernel_of<1>(variant); }
}  // namespace pasur
