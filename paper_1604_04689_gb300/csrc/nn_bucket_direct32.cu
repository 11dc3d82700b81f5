// The direct builds' bucket pass with more than 8 slots per node.
#include "nn_bucket.cuh"

namespace nn {

cudaError_t launch_bucket_direct_32(const BucketParams& p, int grid, size_t smem, cudaStream_t s) {
    return launch_bucket_t<32, DIRECT_BUILD>(p, grid, direct_threads(32), smem, s);
}
cudaError_t set_bucket_smem_direct_32(size_t bytes) { return set_bucket_smem_t<32, DIRECT_BUILD>(bytes); }

}  // namespace nn
