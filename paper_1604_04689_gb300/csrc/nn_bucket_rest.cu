// The bucket pass over the buckets that the ordinary one has noted: up to 32
// slots per node, and the paths for nodes that are not left to a lane.
#include "nn_bucket.cuh"

namespace nn {

cudaError_t launch_bucket_rest(const BucketParams& p, int grid, int threads, size_t smem, cudaStream_t s) {
    return launch_bucket_t<32, REST>(p, grid, threads, smem, s);
}
cudaError_t set_bucket_smem_rest(size_t bytes) { return set_bucket_smem_t<32, REST>(bytes); }

}  // namespace nn
