// The bucket pass of small meshes, whose CTAs read the connectivity themselves
// (direct builds), with up to 8 slots per node.
#include "nn_bucket.cuh"

namespace nn {

cudaError_t launch_bucket_direct_32(const BucketParams& p, int grid, size_t smem, cudaStream_t s);
cudaError_t set_bucket_smem_direct_32(size_t bytes);

cudaError_t launch_bucket_direct(const BucketParams& p, int grid, size_t smem, cudaStream_t s) {
    if (p.imax != 8) return launch_bucket_direct_32(p, grid, smem, s);
    return launch_bucket_t<8, DIRECT_BUILD>(p, grid, direct_threads(8), smem, s);
}
cudaError_t set_bucket_smem_direct(size_t bytes) {
    const cudaError_t e = set_bucket_smem_t<8, DIRECT_BUILD>(bytes);
    return e == cudaSuccess ? set_bucket_smem_direct_32(bytes) : e;
}

}  // namespace nn
