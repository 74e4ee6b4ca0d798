// The block and cluster sweeps for items of 3 score slots.
#include "cfr_block_impl.cuh"
#include "cfr_cluster_impl.cuh"

namespace pasur {
const void *block_kernel_w3(int variant) { return block_kernel_of<3>(variant); }
const void *cluster_kernel_w3(int variant) { return cluster_kernel_of<3>(variant); }
}  // namespace pasur
