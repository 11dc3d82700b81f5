// Batched element walk: many meshes of any types in one launch sequence.
//
// The batch tables (header, one BatchMesh per mesh, element and bucket
// offsets) are in device memory, so the grids below do not depend on the
// batch: the kernels read the totals from the header, and a
// captured launch sequence can be replayed for every batch that fits the
// workspace.  Each mesh owns a contiguous range of buckets and each CTA walks a
// contiguous slice of the batch's elements, whose buckets it counts in shared
// memory before it adds to the batch's (a batch can have far more buckets
// than one shared-memory histogram holds, a slice's meshes hardly ever); then
// the same offsets scan, record format and bucket pass as the single-mesh
// build turn them into per-mesh CSRs.
#include "nn_device.cuh"

namespace nn {

namespace {

constexpr int BATCH_THREADS = 512;
constexpr int BATCH_COUNTERS = 8192;  // buckets a CTA's slice may have for shared counters (32 KB)

// Load element e of mesh M (any type); returns its type, sets *ok.
__device__ __forceinline__ int load_elem_any(const BatchMesh& M, int64_t e, int32_t* nd, bool* ok) {
    int t = M.type;
    int npe;
    if (t == NN_MIXED) {
        t = __ldg(M.elem_type + e);
        const int64_t a = __ldg(M.elem_ptr + e), b = __ldg(M.elem_ptr + e + 1);
        if (t > NN_HEX || a < 0 || b > M.n_conn || b - a != npe_of(t)) {
            set_status(M.status, NN_ERR_ELEM_PTR);
            *ok = false;
            return NN_HEX;
        }
        npe = (int)(b - a);
#pragma unroll
        for (int q = 0; q < 8; ++q) nd[q] = q < npe ? __ldg(M.conn + a + q) : 0;
    } else if (t == NN_TRI) {
        npe = 3;
        nd[0] = __ldg(M.conn + 3 * e);
        nd[1] = __ldg(M.conn + 3 * e + 1);
        nd[2] = __ldg(M.conn + 3 * e + 2);
    } else if (t == NN_HEX) {
        npe = 8;
        const int4* c4 = reinterpret_cast<const int4*>(M.conn) + 2 * e;
        int4 x = __ldg(c4), y = __ldg(c4 + 1);
        nd[0] = x.x; nd[1] = x.y; nd[2] = x.z; nd[3] = x.w;
        nd[4] = y.x; nd[5] = y.y; nd[6] = y.z; nd[7] = y.w;
    } else {
        npe = 4;
        int4 x = __ldg(reinterpret_cast<const int4*>(M.conn) + e);
        nd[0] = x.x; nd[1] = x.y; nd[2] = x.z; nd[3] = x.w;
    }
    bool v = true;
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if (q < npe) v = v && nd[q] >= 0 && (int64_t)nd[q] < M.n_nodes;
    if (!v) set_status(M.status, NN_ERR_NODE_RANGE);
    *ok = v;
    return t;
}

// The elements [e0, e1) of the whole batch that CTA i of n walks, and the mesh
// m0 that e0 lies in.  The batch is cut by weight (a mesh's incidences plus its
// elements), so that a slice of hexes is not three times the work of a slice
// of triangles.
struct Slice {
    int64_t e0, e1;
    int m0, m1;  // its meshes, m1 included
};
__device__ __forceinline__ int mesh_at(const int64_t* off, int n_meshes, int64_t x) {
    int lo = 0, hi = n_meshes;  // largest m with off[m] <= x
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= x) lo = mid;
        else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ int64_t slice_start(const BatchTables& bt, int n_meshes, int64_t x, int* m) {
    *m = mesh_at(bt.weight_off, n_meshes, x);
    const int64_t w0 = bt.weight_off[*m], w = bt.weight_off[*m + 1] - w0, T = bt.elem_off[*m + 1] - bt.elem_off[*m];
    return bt.elem_off[*m] + (w > 0 ? (x - w0) * T / w : 0);
}
__device__ __forceinline__ Slice cta_slice(const BatchTables& bt) {
    const int n = bt.hdr->n_meshes;
    if (n == 0) return Slice{0, 0, 0, 0};
    const int64_t W = bt.weight_off[n];
    Slice s;
    s.e0 = slice_start(bt, n, W * blockIdx.x / gridDim.x, &s.m0);
    s.e1 = slice_start(bt, n, W * (blockIdx.x + 1) / gridDim.x, &s.m1);
    if (blockIdx.x + 1 == gridDim.x) s.e1 = bt.hdr->n_elems;
    return s;
}

// Walk a slice, calling f(mesh index, mesh, local element id, type, nodes)
// for every valid element.
template <class F>
__device__ __forceinline__ void walk_slice(const BatchTables& bt, const Slice& s, F&& f) {
    int m = s.m0;
    for (int64_t e = s.e0 + threadIdx.x; e < s.e1; e += BATCH_THREADS) {
        while (e >= bt.elem_off[m + 1]) ++m;
        const BatchMesh& M = bt.meshes[m];
        int32_t nd[8];
        bool ok;
        const int64_t le = e - bt.elem_off[m];
        const int t = load_elem_any(M, le, nd, &ok);
        if (ok) f(m, M, le, t, nd);
    }
}

// The buckets of a slice's meshes are consecutive.  When they fit the shared
// counters, a CTA adds its records up there first and touches the batch's
// counter or cursor of a bucket once, not once per record.
__device__ __forceinline__ bool shared_buckets(const BatchTables& bt, const Slice& s, int64_t* first, int* n) {
    *first = bt.bucket_off[s.m0];
    const int64_t nb = s.e1 > s.e0 ? bt.bucket_off[s.m1 + 1] - *first : 0;
    *n = (int)min(nb, (int64_t)BATCH_COUNTERS);
    return nb <= BATCH_COUNTERS;
}

__global__ void __launch_bounds__(BATCH_THREADS) k_batch_init(BatchTables bt, uint32_t* bcount, uint32_t* nfc,
                                                              uint64_t* lb_off, uint32_t* ctrl, uint64_t* lb_ns) {
    chain_begin();
    const int64_t B = bt.hdr->n_buckets;
    const int64_t tiles = (B + OFFSETS_THREADS - 1) / OFFSETS_THREADS;
    const int n = bt.hdr->n_meshes;
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < B; i += st) {
        bcount[i] = 0;
        nfc[i] = 0;
    }
    for (int64_t i = i0; i < tiles + 1; i += st) lb_off[i] = 0;
    if (lb_ns)
        for (int64_t i = i0, n = B * (bt.hdr->fmt.sb < 5 ? 1 : 1 << (bt.hdr->fmt.sb - 5));
             i < (n + NODE_SCAN_TILE - 1) / NODE_SCAN_TILE + 1; i += st)
            lb_ns[i] = 0;
    for (int64_t i = i0; i < 16; i += st) ctrl[i] = 0;
    for (int64_t i = i0; i < n; i += st) {
        const BatchMesh& M = bt.meshes[i];
        *M.status = 0;
        if (M.n_nodes == 0) {  // no bucket will write the single row pointer
            if (M.rp_n) M.rp_n[0] = 0;
            if (M.rp_e) M.rp_e[0] = 0;
        }
    }
}

// Records per bucket, and (rare) records of a node already seen in its
// element, which add no element entry.
//
// What bounds this pass and the partition: L2 atomics (about 40 G/s), one per
// record while every record had its own; now the shared counters' atomics and
// the gathered 16-byte stores.  GB300, 24 meshes of 1e3 to 5e5 elements (9.6 M
// records): histogram 228 -> 24 us, partition 260 -> 148 us, the whole call
// 787 -> 459 us.  A slice with more buckets than counters has few records per
// bucket to add up, and keeps one global atomic per record.
__global__ void __launch_bounds__(BATCH_THREADS, 3) k_hist_b(BatchTables bt, uint32_t* bcount, uint32_t* nfc) {
    chain_begin();
    __shared__ uint32_t cnt[BATCH_COUNTERS];
    const int sb = bt.hdr->fmt.sb;
    const Slice s = cta_slice(bt);
    if (s.e1 <= s.e0) return;
    int64_t first;
    int n;
    const bool shared = shared_buckets(bt, s, &first, &n);
    if (shared) {
        for (int i = threadIdx.x; i < n; i += BATCH_THREADS) cnt[i] = 0;
        __syncthreads();
    }
    walk_slice(bt, s, [&](int m, const BatchMesh& M, int64_t, int t, const int32_t* nd) {
        const int npe = npe_of(t);
        const int64_t b0 = bt.bucket_off[m];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (i >= npe) break;
            const int64_t b = b0 + ((uint32_t)nd[i] >> sb);
            if (shared) atomicAdd(&cnt[b - first], 1u);
            else atomicAdd(&bcount[b], 1u);
            int nf = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) nf |= (q < i) && (nd[q] == nd[i]);
            if (nf) atomicAdd(&nfc[b], 1u);
        }
    });
    if (shared) {
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += BATCH_THREADS)
            if (cnt[i]) atomicAdd(&bcount[first + i], cnt[i]);
    }
}

// With shared counters: the slice is walked to count its records per bucket,
// a range is reserved in every bucket it touches, and the second walk (its
// connectivity is in L2 now) takes places from the ranges.
__global__ void __launch_bounds__(BATCH_THREADS, 3) k_part_b(BatchTables bt, uint32_t* gcur, uint8_t* rec) {
    chain_begin();
    __shared__ uint32_t place[BATCH_COUNTERS];
    const RecFmt f = bt.hdr->fmt;
    const uint64_t cap = (uint64_t)bt.hdr->n_records;
    const Slice s = cta_slice(bt);
    if (s.e1 <= s.e0) return;
    int64_t first;
    int n;
    const bool shared = shared_buckets(bt, s, &first, &n);
    if (shared) {
        for (int i = threadIdx.x; i < n; i += BATCH_THREADS) place[i] = 0;
        __syncthreads();
        walk_slice(bt, s, [&](int m, const BatchMesh&, int64_t, int t, const int32_t* nd) {
            const int npe = npe_of(t), b0 = (int)(bt.bucket_off[m] - first);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < npe) atomicAdd(&place[b0 + (int)((uint32_t)nd[i] >> f.sb)], 1u);
        });
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += BATCH_THREADS)
            if (place[i]) place[i] = atomicAdd(&gcur[first + i], place[i]);
        __syncthreads();
    }
    walk_slice(bt, s, [&](int m, const BatchMesh& M, int64_t le, int t, const int32_t* nd) {
        const int npe = npe_of(t), K = k_of(t);
        const int64_t b0 = bt.bucket_off[m];
        uint32_t pos[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            pos[i] = 0xFFFFFFFFu;
            if (i < npe) {
                const int64_t b = b0 + ((uint32_t)nd[i] >> f.sb);
                pos[i] = shared ? atomicAdd(&place[b - first], 1u) : atomicAdd(&gcur[b], 1u);
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (pos[i] >= cap) continue;
            const int32_t v = nd[i];
            uint32_t nf = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) nf |= (q < i) && (nd[q] == v);
            uint32_t n[3];
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                const int32_t y = s < K ? nbr_node(t, nd, i, s) : v;
                n[s] = y == v ? f.nmask : (uint32_t)y;
            }
            put_rec<16>(rec, pos[i], pack_rec<16>(f, make_side(f, (uint32_t)v, nf), (uint32_t)le, n, K));
        }
    });
}

}  // namespace

cudaError_t launch_batch_emit(const BatchTables& bt, uint32_t* bcount, uint32_t* nfc, uint32_t* gcur, uint8_t* rec,
                              uint64_t* lb_off, uint32_t* ctrl, int grid, int stage, bool chain,
                              cudaStream_t s, uint64_t* lb_ns) {
    if (stage == 1) return launch_chained(chain, k_hist_b, grid, BATCH_THREADS, 0, s, bt, bcount, nfc);
    if (stage == 2) return launch_chained(chain, k_part_b, grid, BATCH_THREADS, 0, s, bt, gcur, rec);
    k_batch_init<<<grid, BATCH_THREADS, 0, s>>>(bt, bcount, nfc, lb_off, ctrl, lb_ns);
    return cudaGetLastError();
}

int batch_ctas_per_sm() { return 3; }  // resident at launch_bounds(BATCH_THREADS, 3)

}  // namespace nn
