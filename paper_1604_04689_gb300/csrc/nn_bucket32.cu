// The bucket pass with up to 32 slots per node.
#include "nn_bucket.cuh"

namespace nn {

cudaError_t launch_bucket_32(const BucketParams& p, int grid, int threads, size_t smem, cudaStream_t s) {
    return launch_bucket_t<32>(p, grid, threads, smem, s);
}
cudaError_t set_bucket_smem_32(size_t bytes) { return set_bucket_smem_t<32>(bytes); }
cudaError_t bucket_occupancy_32(int* blocks, int threads, size_t smem) {
    return bucket_occupancy_t<32>(blocks, threads, smem);
}

}  // namespace nn
