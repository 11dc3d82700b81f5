// The bucket pass with up to 8 slots per node, the choice among the variants
// by their register arrays, and its two launches.
#include "nn_bucket.cuh"

namespace nn {

cudaError_t launch_bucket_16(const BucketParams& p, int grid, int threads, size_t smem, cudaStream_t s);
cudaError_t launch_bucket_32(const BucketParams& p, int grid, int threads, size_t smem, cudaStream_t s);
cudaError_t launch_bucket_direct(const BucketParams& p, int grid, size_t smem, cudaStream_t s);
cudaError_t launch_bucket_rest(const BucketParams& p, int grid, int threads, size_t smem, cudaStream_t s);
cudaError_t set_bucket_smem_16(size_t bytes);
cudaError_t set_bucket_smem_32(size_t bytes);
cudaError_t set_bucket_smem_direct(size_t bytes);
cudaError_t set_bucket_smem_rest(size_t bytes);
cudaError_t bucket_occupancy_16(int* blocks, int threads, size_t smem);
cudaError_t bucket_occupancy_32(int* blocks, int threads, size_t smem);

size_t bucket_smem_bytes(int sb, int want, int k, int slots, int rb, int list_cap) {
    const size_t nb = (size_t)1 << sb, groups = nb < 32 ? 1 : nb / 32;
    return 24 * nb + list_bytes(rb, list_cap) + groups * 32 * (size_t)col_words(want, k, slots) * 4;
}

namespace {

cudaError_t launch_plain(const BucketParams& p, int grid, int threads, size_t smem, cudaStream_t s) {
    if (p.imax == 8) return launch_bucket_t<8>(p, grid, threads, smem, s);
    if (p.imax == 16) return launch_bucket_16(p, grid, threads, smem, s);
    return launch_bucket_32(p, grid, threads, smem, s);
}

}  // namespace

cudaError_t launch_bucket(const BucketParams& p, int grid, int threads, size_t smem, const RestShape& rest, cudaStream_t s) {
    if (grid <= 0) return cudaSuccess;
    if (p.direct.conn) return launch_bucket_direct(p, grid, smem, s);
    const cudaError_t e = launch_plain(p, grid, threads, smem, s);
    if (e != cudaSuccess) return e;
    BucketParams q = p;
    q.slots = rest.slots;
    q.list_cap = rest.list_cap;
    q.ticket = p.rest_ticket;
    return launch_bucket_rest(q, rest.grid, rest.threads, rest.smem, s);
}

cudaError_t set_bucket_smem_all(size_t bytes) {
    cudaError_t e = set_bucket_smem_t<8>(bytes);
    if (e == cudaSuccess) e = set_bucket_smem_16(bytes);
    if (e == cudaSuccess) e = set_bucket_smem_32(bytes);
    if (e == cudaSuccess) e = set_bucket_smem_direct(bytes);
    if (e == cudaSuccess) e = set_bucket_smem_rest(bytes);
    return e;
}

cudaError_t bucket_occupancy(int* blocks, int threads, int imax, size_t smem) {
    if (imax == 8) return bucket_occupancy_t<8>(blocks, threads, smem);
    if (imax == 16) return bucket_occupancy_16(blocks, threads, smem);
    return bucket_occupancy_32(blocks, threads, smem);
}

}  // namespace nn
