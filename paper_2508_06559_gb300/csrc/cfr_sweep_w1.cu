// The block and cluster sweeps for items of 1 score slot.
#include "cfr_block_impl.cuh"
#include "cfr_cluster_impl.cuh"

namespace pasur {
const void *block_kernel_w1(int variant) { return block_kernel_of<1>(variant); }
const void *cluster_kernel_w1(int variant) { return cluster_kernel_of<1>(variant); }
}  // namespace pasur
