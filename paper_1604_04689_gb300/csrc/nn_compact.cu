// Node-CSR placement: the bucket pass leaves every bucket's distinct-
// neighbour rows in a scratch area, group of 32 nodes by group, at a position
// bounded in advance (K times the group's first record: a record adds at most K
// neighbours), with each node's offset inside its group and the group's total.
// Two short kernels then place them: an exclusive scan of the group totals
// (single pass, decoupled lookback over tiles of groups), and a copy of every
// group's rows to its offset in the mesh's col, with the row pointers.  No
// bucket ever waits for another while it builds its rows.
#include <algorithm>

#include "nn_device.cuh"

namespace nn {

namespace {

constexpr int SCAN_THREADS = 128;
constexpr int SCAN_PER = NODE_SCAN_TILE / SCAN_THREADS;  // groups per thread
constexpr int COPY_THREADS = 256;

__device__ __forceinline__ int groups_of(int sb) { return sb < 5 ? 1 : 1 << (sb - 5); }

__global__ void __launch_bounds__(SCAN_THREADS) k_node_scan(CompactParams p) {
    chain_begin();
    __shared__ uint64_t sh_scan[33];
    __shared__ uint32_t sh_tile;
    __shared__ uint64_t sh_base;
    const int64_t n = (p.batch.hdr ? p.batch.hdr->n_buckets : p.n_buckets) *
                      groups_of(p.batch.hdr ? p.batch.hdr->fmt.sb : p.sb);
    if (threadIdx.x == 0) sh_tile = atomicAdd(p.ticket, 1u);
    __syncthreads();
    const uint32_t tile = sh_tile;
    if ((int64_t)tile * NODE_SCAN_TILE >= n) return;  // whole CTA: no groups left
    const int64_t g0 = (int64_t)tile * NODE_SCAN_TILE + threadIdx.x * SCAN_PER;
    uint32_t x[SCAN_PER];
    uint64_t sum = 0;
#pragma unroll
    for (int i = 0; i < SCAN_PER; ++i) {
        x[i] = g0 + i < n ? p.grp[g0 + i].y : 0u;
        sum += x[i];
    }
    uint64_t agg;
    const uint64_t ex = block_excl_scan(sum, &agg, sh_scan);
    if (threadIdx.x < 32) {
        const uint64_t base = warp_lookback(p.lb_state, tile, agg, p.status);
        if (threadIdx.x == 0) sh_base = base;
    }
    __syncthreads();
    uint64_t run = sh_base + ex;
#pragma unroll
    for (int i = 0; i < SCAN_PER; ++i) {
        if (g0 + i < n) p.nstart[g0 + i] = run;
        run += x[i];
        if (g0 + i == n - 1) p.nstart[n] = run;
    }
}

// One warp per group of 32 nodes.  SUM: a CTA takes 8 groups and adds up the
// totals of the groups before them itself, which for a few thousand groups
// costs less than the scan's launch.
template <bool SUM>
__global__ void __launch_bounds__(COPY_THREADS, 8) k_node_copy(CompactParams p) {
    chain_begin();
    const bool batched = p.batch.hdr != nullptr;
    const int64_t B = batched ? p.batch.hdr->n_buckets : p.n_buckets;
    const int sb = batched ? p.batch.hdr->fmt.sb : p.sb;
    const int K = batched ? 3 : p.k;
    const int n_meshes = batched ? p.batch.hdr->n_meshes : 1;
    const int GP = groups_of(sb), lane = threadIdx.x & 31;
    const int64_t n = B * GP, warps = (int64_t)gridDim.x * (COPY_THREADS / 32);
    uint64_t before = 0;  // SUM: entries of this warp's group's predecessors
    if constexpr (SUM) {
        __shared__ uint64_t sh_scan[33];
        const int64_t first = (int64_t)blockIdx.x * (COPY_THREADS / 32), mine = first + (threadIdx.x >> 5);
        uint64_t x = 0, total;
        for (int64_t i = threadIdx.x; i < first; i += COPY_THREADS) x += p.grp[i].y;
        block_excl_scan(x, &total, sh_scan);
        before = total;
        for (int64_t i = first; i < mine && i < n; ++i) before += p.grp[i].y;
    }
    for (int64_t gi = (int64_t)blockIdx.x * (COPY_THREADS / 32) + (threadIdx.x >> 5); gi < n; gi += warps) {
        const int64_t b = gi / GP;
        int64_t first = 0, N = p.n_nodes;
        int64_t* rp = p.rp_n;
        int32_t* col = p.col_n;
        int64_t cap = p.cap_n;
        int32_t* status = p.status;
        if (batched) {
            int lo = 0, hi = n_meshes;  // largest m with bucket_off[m] <= b
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (p.batch.bucket_off[mid] <= b) lo = mid;
                else hi = mid;
            }
            const BatchMesh& M = p.batch.meshes[lo];
            first = p.batch.bucket_off[lo];
            N = M.n_nodes;
            rp = M.rp_n;
            col = M.col_n;
            cap = M.cap_n;
            status = M.status;
        }
        // the group's first node and how many of them the mesh has
        const int64_t v0 = ((b - first) << sb) + (gi - b * GP) * 32, left = N - v0;
        if (left <= 0) continue;
        const int nb = (int)min(left, (int64_t)(sb < 5 ? 1 << sb : 32));
        const uint64_t gn = SUM ? before : p.nstart[gi] - p.nstart[first * GP] + (p.base ? (uint64_t)p.base[1] : 0ull);
        const uint2 g = p.grp[gi];
        const size_t loc = ((size_t)b << sb) + (size_t)(gi - b * GP) * 32 + lane;
        if (lane < nb && NN_IN(loc, p.nloc_words, status)) rp[v0 + lane] = (int64_t)(gn + p.nloc[loc]);
        if (left == nb && lane == 0) rp[N] = (int64_t)(gn + g.y);
        if (gn + g.y > (uint64_t)cap) {
            if (lane == 0) set_status(status, NN_ERR_CAPACITY);
            continue;
        }
        const uint32_t* src = p.ntmp + (size_t)K * g.x;
        int32_t* dst = col + gn;
        if (!NN_IN((size_t)K * g.x + (g.y ? g.y - 1 : 0), p.ntmp_words + (g.y ? 0 : 1), status)) continue;
        // (four loads in flight: ordinary ones may not pass the stores before them)
        uint32_t i = lane;
        for (; i + 96 < g.y; i += 128) {
            const uint32_t a = src[i], b = src[i + 32], c = src[i + 64], d = src[i + 96];
            dst[i] = (int32_t)a;
            dst[i + 32] = (int32_t)b;
            dst[i + 64] = (int32_t)c;
            dst[i + 96] = (int32_t)d;
        }
        uint32_t x[3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (i + 32 * k < g.y) x[k] = src[i + 32 * k];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (i + 32 * k < g.y) dst[i + 32 * k] = (int32_t)x[k];
    }
}

// The scans' and tickets' words of a build, and its status: one launch in
// place of two memsets.
constexpr int INIT_THREADS = 512;
__global__ void __launch_bounds__(INIT_THREADS) k_init(uint4* w, int64_t n, int32_t* status) {
    chain_begin();
    const int64_t i0 = (int64_t)blockIdx.x * INIT_THREADS + threadIdx.x;
    if (i0 == 0) *status = 0;
    for (int64_t i = i0; i < n; i += (int64_t)gridDim.x * INIT_THREADS) w[i] = make_uint4(0u, 0u, 0u, 0u);
}

// Chunked builds run one node range after another into the same CSRs; after
// a chunk, the running bases move past its element and node entries.
__global__ void k_chunk_advance(int64_t* base, const uint32_t* etot, const uint64_t* ntot) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (etot) base[0] += (int64_t)*etot;
        if (ntot) base[1] += (int64_t)*ntot;
    }
}

}  // namespace

cudaError_t launch_chunk_advance(int64_t* base, const uint32_t* etot, const uint64_t* ntot, cudaStream_t s) {
    k_chunk_advance<<<1, 32, 0, s>>>(base, etot, ntot);
    return cudaGetLastError();
}

cudaError_t launch_node_compact(const CompactParams& p, int copy_grid, cudaStream_t s) {
    const unsigned tiles = (unsigned)((p.n_groups_cap + NODE_SCAN_TILE - 1) / NODE_SCAN_TILE);
    if (tiles == 0) return cudaSuccess;
    // (a chunked build needs the scan's grand total, a batch starts over at every mesh)
    if (p.n_groups_cap <= NODE_SUM_GROUPS && !p.batch.hdr && !p.base) {
        return launch_chained(p.chain, k_node_copy<true>, (unsigned)((p.n_groups_cap + COPY_THREADS / 32 - 1) / (COPY_THREADS / 32)),
                              COPY_THREADS, 0, s, p);
    }
    const cudaError_t e = launch_chained(p.chain, k_node_scan, tiles, SCAN_THREADS, 0, s, p);
    return e == cudaSuccess ? launch_chained(p.chain, k_node_copy<false>, copy_grid, COPY_THREADS, 0, s, p) : e;
}

cudaError_t launch_init(void* p, size_t bytes, int32_t* status, int sms, cudaStream_t s) {
    const int64_t n = (int64_t)(bytes / 16);
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(sms, (n + INIT_THREADS - 1) / INIT_THREADS));
    k_init<<<(unsigned)blocks, INIT_THREADS, 0, s>>>(static_cast<uint4*>(p), n, status);
    return cudaGetLastError();
}

}  // namespace nn
