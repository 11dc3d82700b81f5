// Bucket pass: builds the rows of one node range per CTA from its records.
//
// For the 2^sb nodes of a bucket the CTA
//   1. reads the bucket's records once, in order, and puts each one's element
//      id and neighbours into its node's column of a table in shared memory:
//      the slot is what the node's record counter gives (one shared-memory
//      atomic per record).  Slot s of the 32 nodes of a group lies in 32
//      neighbouring words, so that a lane reads its node's column without
//      bank conflicts and nothing has to be counted, scanned or regrouped
//      first.  A node has `slots` places (about its mesh's mean number of
//      records); its further records go to a short list, chained by node.
//   2. gives every node to one lane: 32 consecutive nodes form a group that
//      one warp finishes alone, without block barriers.  Neighbour row: the
//      candidates go into registers and are sorted by a network; repeats (an
//      edge shared by several elements) are dropped when the row is written.
//      Lanes with listed records then put their distinct values back into
//      their column, add candidates from the list and sort again, until the
//      list is used up.  Element row: sorted in registers the same way.
//      Rows are put together in the group's own part of the table and written
//      as one run: the element CSR at offsets known before the pass (a prefix
//      of the record counts), the node rows, each node's offset among the
//      group's and their total to a scratch area, at a position bounded in
//      advance (K times the group's first record); the compaction pass places
//      them (nn_compact.cu).  No bucket ever waits for another.
// A bucket with a node of very many records or neighbours, or with more
// listed records than fit, is built by its whole CTA instead, node by node and
// warp by warp, with record indices grouped in a global spill area.
//
// What bounds it: instructions (issue slots 71 % busy on hexes), then
// instruction fetch where the networks are long (tets) and shared-memory
// stores.  Before, records were staged in shared memory, counted, scanned and
// gathered by index twice at 16 warps per SM (issue 31-49 %), and tets went
// through a hash table per lane.  GB300, both results, before and now:
// hex 257^3 2.30 -> 1.61 ms, tet 161^3 3.08 -> 1.46 ms, hex/tet mixed 257^3
// 8.35 -> 4.74 ms, triangles 2048^2 0.48 -> 0.31 ms.
//
// Rows are sets in ascending order: the paper's pipeline (Sec. 2.2.1) sorts
// pairs by key only and counts pairs per key, which lists an edge shared by
// two elements twice; one-ring neighbours are a set (Sec. 1), so repeated
// neighbours are dropped and each row is sorted.
#pragma once

#include "nn_device.cuh"

namespace nn {

namespace {

constexpr uint32_t FULL = 0xffffffffu;
constexpr uint32_t PREFETCH = 32768;  // bytes per prefetch instruction
constexpr uint32_t CHAIN_END = 0xffffffffu;

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__host__ __device__ constexpr int pow2_ceil(int n) { return n <= 1 ? 1 : 2 * pow2_ceil((n + 1) / 2); }

// Ascending sort of a[0..N) held in registers by Batcher's odd-even merge
// sort (Knuth, TAOCP vol. 3, 5.3.4), laid out for the next power of two P
// >= N and pruned to N: every comparator puts the minimum at its lower index,
// so the +infinity (EMPTY) entries at N..P-1 never move and a comparator that
// touches one of them is a no-op.  Every index is a compile-time constant
// once the loops are unrolled, so the array stays in registers.
template <int N, int M>
__device__ __forceinline__ void sort_net(uint32_t (&a)[M]) {
    static_assert(N <= M, "network size");
    constexpr int P = pow2_ceil(N);
#pragma unroll
    for (int p = 1; p < P; p <<= 1) {
#pragma unroll
        for (int k = p; k >= 1; k >>= 1) {
            // comparators (lo, lo + k) for lo = j + i, j = k mod p + 2k t, 0 <= i < k,
            // both ends in one block of 2p
#pragma unroll
            for (int lo = 0; lo < P; ++lo) {
                const int r = lo - k % p, hi = lo + k;
                if (r >= 0 && r % (2 * k) < k && hi < N && lo / (2 * p) == hi / (2 * p)) {
                    const uint32_t x = a[lo], y = a[hi];
                    a[lo] = min(x, y);
                    a[hi] = max(x, y);
                }
            }
        }
    }
}

// Sort the first n <= M entries (the rest are EMPTY): the smallest network
// that covers the warp's longest row (n_warp is warp-uniform).
template <int M, int N>
__device__ __forceinline__ void sort_from(uint32_t (&a)[M], uint32_t n_warp) {
    // network sizes: 2, 4, 6, 8, 12, 16, 24, 32, 48, 72 and M
    constexpr int NEXT = N < 8 ? N + 2 : (N < 16 ? N + 4 : (N < 32 ? N + 8 : (N < 48 ? N + 16 : N + 24)));
    if constexpr (NEXT > M) {
        sort_net<M>(a);
    } else {
        if (n_warp <= N) sort_net<N>(a);
        else sort_from<M, NEXT>(a, n_warp);
    }
}
template <int M>
__device__ __forceinline__ void sort_prefix(uint32_t (&a)[M], uint32_t n_warp) {
    if (n_warp > 1) sort_from<M, 2>(a, n_warp);
}

// Ascending bitonic sort of a[0..n) by one warp (generic pointer), in the
// formulation whose compare-exchanges put the minimum at the lower index, so
// that indices >= n act as +infinity and are skipped.
__device__ inline void warp_bitonic_sort(uint32_t* a, uint32_t n) {
    if (n < 2) return;
    const uint32_t lane = threadIdx.x & 31;
    uint32_t P = 1;
    while (P < n) P <<= 1;
    for (uint32_t k = 2; k <= P; k <<= 1) {
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t t = lane; t < (P >> 1); t += 32) {
                const uint32_t idx = ((t & ~(j - 1)) << 1) | (t & (j - 1));
                const uint32_t q = (j == (k >> 1)) ? (idx ^ (k - 1)) : (idx ^ j);
                if (q < n) {
                    const uint32_t x = a[idx], y = a[q];
                    if (x > y) {
                        a[idx] = y;
                        a[q] = x;
                    }
                }
            }
            __syncwarp();
        }
    }
}

// The element ids of a node's c records (a repeated node's record adds
// none), collected by its whole warp into row[0..ec) and sorted there.
template <int RB, int K>
__device__ __noinline__ void warp_elem_row(const RecFmt& f, const uint8_t* rp, const uint32_t* grp, uint32_t c,
                                           uint32_t* row, uint32_t ec) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t wpos = 0;
    for (uint32_t s0 = 0; s0 < c; s0 += 32) {
        const uint32_t s = s0 + lane;
        bool keep = false;
        uint32_t e = 0;
        if (s < c) {
            const Rec x = take_rec<RB>(rp, grp[s]);
            keep = !((rec_side<RB, K>(f, x) >> f.off_nf) & 1u);
            e = rec_elem<RB>(f, x);
        }
        const unsigned km = __ballot_sync(FULL, keep);
        if (keep) row[wpos + __popc(km & lanemask_lt())] = e;
        wpos += __popc(km);
    }
    __syncwarp();
    warp_bitonic_sort(row, ec);
}

// The distinct neighbours of a node's c records, collected by its whole warp
// into a[0 .. K c): sorted, the first of every run kept.  Returns their count.
template <int RB, int K>
__device__ __noinline__ uint32_t warp_node_row(const RecFmt& f, const uint8_t* rp, const uint32_t* grp, uint32_t c,
                                               uint32_t* a) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t nc = (uint64_t)K * c;
    for (uint32_t s = lane; s < c; s += 32) {
        const Rec x = take_rec<RB>(rp, grp[s]);
#pragma unroll
        for (int j = 0; j < K; ++j) a[(uint64_t)s * K + j] = rec_nbr<RB>(f, x, j);
    }
    __syncwarp();
    warp_bitonic_sort(a, (uint32_t)nc);
    // keep the first of every run (in place: writes never pass the chunk being read)
    uint32_t nu = 0, carry = f.nmask;
    for (uint32_t i0 = 0; i0 < nc; i0 += 32) {
        const uint32_t idx = i0 + lane;
        const uint32_t val = idx < nc ? a[idx] : f.nmask;
        uint32_t prev = __shfl_up_sync(FULL, val, 1);
        if (lane == 0) prev = carry;
        carry = __shfl_sync(FULL, val, 31);
        const bool keep = val != f.nmask && val != prev;
        const unsigned km = __ballot_sync(FULL, keep);
        __syncwarp();
        if (keep) a[nu + __popc(km & lanemask_lt())] = val;
        nu += __popc(km);
        __syncwarp();
    }
    return nu;
}

// n words from shared to global memory by one warp, four at a time per lane.
__device__ __forceinline__ void copy_run(uint32_t* __restrict__ dst, const uint32_t* src, uint32_t n) {
    uint32_t i = threadIdx.x & 31;
    for (; i + 96 < n; i += 128) {
        const uint32_t a = src[i], b = src[i + 32], c = src[i + 64], d = src[i + 96];
        dst[i] = a;
        dst[i + 32] = b;
        dst[i + 64] = c;
        dst[i + 96] = d;
    }
    for (; i < n; i += 32) dst[i] = src[i];
}

struct BucketOut {
    int64_t n_nodes, first;
    bool last;
    int64_t* rp_n; int32_t* col_n; int64_t cap_n;
    int64_t* rp_e; int32_t* col_e; int64_t cap_e;
    int32_t* status;
};

// What the bucket pass knows of a bucket before it starts on it.
struct BucketMeta {
    int64_t b;
    uint32_t r0, r1;  // its records
    uint64_t ge;      // element-CSR offset of its rows
    uint32_t ne;      // element-row entries
};

// Words of a node's neighbour column: its slots, and room for a triangle fan
// of 22 around a node whose slots are few.  (Of 14 with the fewest slots: that
// is what buckets of 2048 nodes have room for, which meshes of more than 2^30
// nodes need to stay within 2^20 buckets.)
__host__ __device__ constexpr int ncol_of(int k, int slots) {
    return slots <= SLOTS_MIN ? 16 : (k * slots > 24 ? k * slots : 24);
}
// Words of a node's element column.  Without a neighbour column the rows are
// put together here, where listed records add to the slots.
__host__ __device__ constexpr int ecol_of(int want, int slots) {
    return !(want & NN_WANT_ELEMS) ? 0 : ((want & NN_WANT_NODES) ? slots : slots + slots / 4 + 2);
}
__host__ __device__ constexpr int col_words(int want, int k, int slots) {
    return ecol_of(want, slots) + ((want & NN_WANT_NODES) ? ncol_of(k, slots) : 0);
}

// Shared memory: two sets (this bucket's and the next one's) of per-node
// counters (records, repeated-node records, first listed record), the list of
// records beyond the slots (16-byte or 8-byte records, then 16-bit links),
// and the table (a group's element columns, then its neighbour columns).
constexpr size_t MISC_BYTES = 34 * 8 + 64;
__host__ __device__ constexpr size_t list_bytes(int rb, int cap) { return ((size_t)cap * (rb + 2) + 15) / 16 * 16; }

// Registers: VE element ids and NW neighbour candidates of a node.  IMAX
// bounds the slots; a node may have VE records before its bucket is built by
// the whole CTA.  8 slots (triangles, quads, hexes): 64 registers, 32 warps
// per SM; 32 slots (tets): 128 and 16.
template <int K, int IMAX>
struct Regs {
    static constexpr int VE = IMAX == 8 ? 24 : 2 * IMAX;
    static constexpr int NW = K * IMAX > 32 ? K * IMAX : 32;
    static constexpr int MIN_CTAS = IMAX == 8 ? 4 : (IMAX == 16 ? 3 : 2);
};

// Direct builds (small meshes): every CTA reads the whole connectivity and
// keeps the incidences of its own bucket, so that the histogram, the offsets
// and the partition are not needed: for a few thousand elements each of those
// is a launch with next to nothing to do.  What bounds it is the latency of a
// few dependent steps (triangles 64^2, 128 CTAs: 13 us of a build of 18), so a
// CTA has as many threads as the registers allow.  Whole builds, graph
// replays: triangles 64^2 33 -> 18 us, hex 21^3 32 -> 27 us; as calls, one
// after another, triangles 64^2 44 -> 18 us.  scan_elements looks at the elements
// [e0, e1): incidences of the nodes [v0, v0 + span) go into the queue (element
// * 8 + local node), and those of lower nodes are counted (below[0]; below[1]:
// the repeated-node ones), which gives the bucket's place in the results.
template <int TYPE>
__device__ __noinline__ void scan_elements(DirectMesh d, uint32_t v0, uint32_t span, uint32_t e0, uint32_t e1,
                                           uint32_t* queue, uint32_t* n_queue, uint32_t* below, int32_t* status) {
    constexpr int NPE = TYPE == NN_MIXED ? 8 : ElemT<(TYPE == NN_MIXED ? NN_HEX : TYPE)>::NPE;
    constexpr int U = NPE == 8 ? 2 : 4;  // elements a thread loads at once
    const uint32_t N = (uint32_t)d.n_nodes, T = blockDim.x;
    uint32_t less = 0, less_rep = 0;
    for (uint32_t b = e0 + threadIdx.x; b < e1; b += U * T) {
        uint32_t nd[U][NPE];
        uint32_t npe[U];  // 0: no element here
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const uint32_t e = b + q * T;
            npe[q] = e < e1 ? NPE : 0;
#pragma unroll
            for (int i = 0; i < NPE; ++i) nd[q][i] = N;
            if constexpr (TYPE == NN_TRI) {
                if (e < e1) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) nd[q][i] = (uint32_t)__ldg(d.conn + 3 * (size_t)e + i);
                }
            } else if constexpr (TYPE == NN_MIXED) {
                if (e < e1) {
                    const int t = __ldg(d.elem_type + e);
                    const int64_t a = __ldg(d.elem_ptr + e), z = __ldg(d.elem_ptr + e + 1);
                    if (t > NN_HEX || a < 0 || z > d.n_conn || z - a != npe_of(t)) {
                        set_status(status, NN_ERR_ELEM_PTR);
                        npe[q] = 0;
                    } else {
                        npe[q] = (uint32_t)(z - a);
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (i < (int)npe[q]) nd[q][i] = (uint32_t)__ldg(d.conn + a + i);
                    }
                }
            } else {
                if (e < e1) {
#pragma unroll
                    for (int i = 0; i < NPE; i += 4) {
                        const uint4 x = __ldg(reinterpret_cast<const uint4*>(d.conn + (size_t)NPE * e + i));
                        nd[q][i] = x.x; nd[q][i + 1] = x.y; nd[q][i + 2] = x.z; nd[q][i + 3] = x.w;
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            // (a mixed element's places past its own nodes hold N: neither below v0 nor in the span)
            uint32_t top = 0;
            bool rep = false;
#pragma unroll
            for (int i = 0; i < NPE; ++i) {
                top = max(top, TYPE != NN_MIXED || i < (int)npe[q] ? nd[q][i] : 0u);
#pragma unroll
                for (int j = 0; j < i; ++j) rep = rep || (nd[q][j] == nd[q][i] && (TYPE != NN_MIXED || i < (int)npe[q]));
            }
            if (npe[q] == 0) continue;
            if (top >= N) {
                set_status(status, NN_ERR_NODE_RANGE);
                continue;
            }
#pragma unroll
            for (int i = 0; i < NPE; ++i) {
                less += nd[q][i] < v0;
                if (nd[q][i] - v0 < span && nd[q][i] < N) queue[atomicAdd(n_queue, 1u)] = (b + q * T) * 8u + i;
            }
            if (rep) {
#pragma unroll
                for (int i = 1; i < NPE; ++i) {
                    bool again = false;
#pragma unroll
                    for (int j = 0; j < i; ++j) again = again || nd[q][j] == nd[q][i];
                    less_rep += again && nd[q][i] < v0;
                }
            }
        }
    }
    less = __reduce_add_sync(FULL, less);
    less_rep = __reduce_add_sync(FULL, less_rep);
    if ((threadIdx.x & 31) == 0) {
        if (less) atomicAdd(&below[0], less);
        if (less_rep) atomicAdd(&below[1], less_rep);
    }
}

// The record of local node i of element e (a queue entry of scan_elements).
template <int RB>
__device__ __forceinline__ Rec direct_rec(const DirectMesh& d, const RecFmt& f, uint32_t entry) {
    const uint32_t e = entry >> 3;
    const int i = (int)(entry & 7u);
    const int t = d.type == NN_MIXED ? (int)__ldg(d.elem_type + e) : d.type;
    const int32_t* nd = d.conn + (d.type == NN_MIXED ? __ldg(d.elem_ptr + e) : (int64_t)e * npe_of(t));
    const int32_t v = __ldg(nd + i);
    const int K = k_of(t);
    uint32_t n[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int32_t y = s < K ? __ldg(nd + nbr_of(t, i, s)) : v;
        n[s] = y == v ? f.nmask : (uint32_t)y;
    }
    uint32_t nf = 0;
    for (int j = 0; j < i; ++j) nf |= __ldg(nd + j) == v;
    return pack_rec<RB>(f, make_side(f, (uint32_t)v, nf), e, n, K);
}

// Threads of a direct build's CTA: as many as the variant's registers allow,
// for the walk over the connectivity.
__host__ __device__ constexpr int direct_threads(int imax) { return imax == 8 ? 1024 : 512; }

template <int RB, int K, int IMAX, bool DIRECT>
__global__ void __launch_bounds__(DIRECT ? direct_threads(IMAX) : 256, DIRECT ? 1 : Regs<K, IMAX>::MIN_CTAS) k_bucket(BucketParams p) {
    chain_begin();
    constexpr int VE = Regs<K, IMAX>::VE, NW = Regs<K, IMAX>::NW;
    constexpr int U = 4;  // records a thread loads at once
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ BucketOut sh_out;
    __shared__ BucketMeta meta[2];
    __shared__ uint32_t sh_list[2];   // listed records (of this bucket, of the next)
    __shared__ uint32_t sh_big[2];    // the bucket needs the whole CTA (this one, the next)
    __shared__ uint64_t sh_scan[34];
    __shared__ RecFmt sh_fmt;         // for the out-of-line helpers
    __shared__ uint64_t sh_spill[2];  // this CTA's part of the spill area: first word, words
    __shared__ uint32_t sh_direct[DIRECT ? 6 : 1];  // queue entries, records below (repeated), own (repeated), written
    const bool batched = p.batch.hdr != nullptr;
    const RecFmt f = batched ? p.batch.hdr->fmt : p.fmt;
    const int64_t n_buckets = batched ? p.batch.hdr->n_buckets : p.n_buckets;
    const int n_meshes = batched ? p.batch.hdr->n_meshes : 1;
    const int NB = 1 << f.sb, GP = NB < 32 ? 1 : NB >> 5;
    const uint32_t vmask = (uint32_t)NB - 1;
    const bool want_n = f.want & NN_WANT_NODES, want_e = f.want & NN_WANT_ELEMS;
    const int C = p.slots, EC = ecol_of(f.want, C), NC = want_n ? ncol_of(K, C) : 0;
    const int GW = (EC + NC) * 32;  // table words of a group
    uint32_t* const cnts = reinterpret_cast<uint32_t*>(smem);  // [2][3][NB]
    uint8_t* const list = smem + (size_t)24 * NB;
    uint16_t* const link = reinterpret_cast<uint16_t*>(list + (size_t)p.list_cap * RB);
    uint32_t* const table = reinterpret_cast<uint32_t*>(list + list_bytes(RB, p.list_cap));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x, W = T >> 5;

    auto clear = [&](int set) {
        uint32_t* c = cnts + (size_t)set * 3 * NB;
        for (int l = tid; l < 2 * NB; l += T) c[l] = 0;
        for (int l = tid; l < NB; l += T) c[2 * NB + l] = CHAIN_END;
        if (tid == 0) sh_list[set] = sh_big[set] = 0;
    };
    // one thread: bounds and element offset of bucket t; its records are pulled into L2
    auto take = [&](int slot, uint32_t t) {
        BucketMeta M{};
        M.b = t;
        if (t < n_buckets) {
            M.r0 = p.bstart[t];
            M.r1 = p.bstart[t + 1];
            if (want_e) {
                int64_t fb = 0;  // the bucket's mesh's first bucket (batches)
                if (batched) {
                    int lo_m = 0, hi_m = n_meshes;
                    while (hi_m - lo_m > 1) {
                        const int mid = (lo_m + hi_m) >> 1;
                        if (p.batch.bucket_off[mid] <= (int64_t)t) lo_m = mid;
                        else hi_m = mid;
                    }
                    fb = p.batch.bucket_off[lo_m];
                }
                M.ge = (uint64_t)(p.estart[t] - p.estart[fb]) + (p.base ? (uint64_t)p.base[0] : 0ull);
                M.ne = p.estart[t + 1] - p.estart[t];
            }
#ifdef NN_CHECKED
            if (M.r1 < M.r0 || M.r1 > p.rec_count) {  // else the bucket reads nothing
                set_status(p.status ? p.status : p.batch.meshes[0].status, NN_ERR_BOUNDS);
                M.r1 = M.r0 = 0;
            }
#endif
            uint64_t lo = (uint64_t)M.r0 * RB, hi = (uint64_t)M.r1 * RB;
            lo &= ~15ull;
            hi = (hi + 15) & ~15ull;  // the record array is padded to 256 bytes
            for (uint64_t a = lo; a < hi; a += PREFETCH) {
                const uint32_t n = (uint32_t)(hi - a < PREFETCH ? hi - a : PREFETCH);
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.rec + a), "r"(n) : "memory");
            }
        }
        meta[slot] = M;
    };

    clear(0);
    if (tid == 0) {
        sh_spill[0] = sh_spill[1] = 0;
        sh_fmt = f;
        if constexpr (DIRECT) {
            meta[0] = BucketMeta{(int64_t)blockIdx.x, 0, 0, 0, 0};
            for (uint32_t& x : sh_direct) x = 0;
        } else {
            take(0, atomicAdd(p.ticket, 1u));
        }
    }
    // direct builds: sink(record) for every record of bucket b
    auto gather = [&](int64_t b, auto&& sink) {
        uint32_t* const queue = reinterpret_cast<uint32_t*>(smem + p.direct.queue_off);
        const DirectMesh d = p.direct;
        const uint32_t v0 = (uint32_t)(b << f.sb), T_e = (uint32_t)d.n_elems;
        const int npe = d.type == NN_MIXED ? 8 : npe_of(d.type);
        auto flush = [&]() {
            const uint32_t n = sh_direct[0];
            for (uint32_t i = tid; i < n; i += T) sink(direct_rec<RB>(d, f, queue[i]));
            __syncthreads();
            if (tid == 0) sh_direct[0] = 0;
            __syncthreads();
        };
        for (uint32_t e = 0; e < T_e;) {
            // as many elements as the queue surely has room for
            if ((d.queue_cap - sh_direct[0]) / npe < min(T_e - e, d.queue_cap / npe / 2)) flush();
            const uint32_t e1 = min(T_e, e + (d.queue_cap - sh_direct[0]) / npe);
            __syncthreads();
            int32_t* const st = p.status;
            switch (d.type) {
                case NN_TRI: scan_elements<NN_TRI>(d, v0, NB, e, e1, queue, &sh_direct[0], &sh_direct[1], st); break;
                case NN_QUAD: scan_elements<NN_QUAD>(d, v0, NB, e, e1, queue, &sh_direct[0], &sh_direct[1], st); break;
                case NN_TET: scan_elements<NN_TET>(d, v0, NB, e, e1, queue, &sh_direct[0], &sh_direct[1], st); break;
                case NN_HEX: scan_elements<NN_HEX>(d, v0, NB, e, e1, queue, &sh_direct[0], &sh_direct[1], st); break;
                default: scan_elements<NN_MIXED>(d, v0, NB, e, e1, queue, &sh_direct[0], &sh_direct[1], st); break;
            }
            __syncthreads();
            e = e1;
        }
        flush();
    };
    __syncthreads();
    for (int it = 0;; ++it) {
        const int cur = it & 1;
        BucketMeta M = meta[cur];
        const int64_t b = M.b;
        if (b >= n_buckets) break;
        uint32_t nx = 0;
        if (tid == 0) {
            nx = DIRECT ? (uint32_t)n_buckets : atomicAdd(p.ticket, 1u);  // the next bucket
            // the mesh this bucket belongs to (the only one unless batched)
            BucketOut o{p.n_nodes, 0, b == n_buckets - 1, p.rp_n, p.col_n, p.cap_n, p.rp_e, p.col_e, p.cap_e, p.status};
            if (batched) {
                int lo_m = 0, hi_m = n_meshes;  // largest m with bucket_off[m] <= b
                while (hi_m - lo_m > 1) {
                    const int mid = (lo_m + hi_m) >> 1;
                    if (p.batch.bucket_off[mid] <= b) lo_m = mid;
                    else hi_m = mid;
                }
                const BatchMesh& Mm = p.batch.meshes[lo_m];
                o = BucketOut{Mm.n_nodes, p.batch.bucket_off[lo_m], b == p.batch.bucket_off[lo_m + 1] - 1, Mm.rp_n,
                              Mm.col_n, Mm.cap_n, Mm.rp_e, Mm.col_e, Mm.cap_e, Mm.status};
                if (*p.batch_err) set_status(o.status, *p.batch_err);
            }
            sh_out = o;
        }
        uint32_t* const c32 = cnts + (size_t)cur * 3 * NB;  // [NB] records
        uint32_t* const nfc = c32 + NB;                     // [NB] repeated-node records
        uint32_t* const first = nfc + NB;                   // [NB] first listed record
        // 1. records into their nodes' columns
        auto place = [&](const Rec& x) {
            const uint32_t side = rec_side<RB, K>(f, x), v = side & vmask;
            const uint32_t s = atomicAdd(&c32[v], 1u);
            const bool nf = want_e && ((side >> f.off_nf) & 1u);
            if (nf) atomicAdd(&nfc[v], 1u);
            if (s < (uint32_t)C) {
                uint32_t* const col = table + ((v >> 5) * (uint32_t)GW + (v & 31));
                if (want_e) col[s * 32] = nf ? EMPTY : rec_elem<RB>(f, x);
                if (want_n) {
#pragma unroll
                    for (int j = 0; j < K; ++j)
                        col[(EC + s * K + j) * 32] = rec_nbr<RB>(f, x, j);
                }
            } else {
                const uint32_t i = atomicAdd(&sh_list[cur], 1u);
                if (i < (uint32_t)p.list_cap && s < (uint32_t)VE) {
                    put_rec<RB>(list, i, x);
                    link[i] = (uint16_t)atomicExch(&first[v], i);
                } else {
                    sh_big[cur] = 1;
                }
            }
        };
        if constexpr (DIRECT) {
            gather(b, place);
            for (int l = tid; l < NB; l += T) {
                if (c32[l]) atomicAdd(&sh_direct[3], c32[l]);
                if (nfc[l]) atomicAdd(&sh_direct[4], nfc[l]);
            }
            __syncthreads();
            M.r0 = sh_direct[1];
            M.r1 = M.r0 + sh_direct[3];
            M.ge = M.r0 - sh_direct[2];
            M.ne = sh_direct[3] - sh_direct[4];
            if (M.r1 > p.rec_count) {  // elements of an invalid elem_ptr that overlap: more records than connectivity
                if (tid == 0) {
                    set_status(p.status, NN_ERR_WORKSPACE);
                    sh_big[cur] = 0;
                }
                for (int l = tid; l < 2 * NB; l += T) c32[l] = 0;
                M = BucketMeta{b, 0, 0, 0, 0};
                __syncthreads();
            }
        }
        const uint32_t R = M.r1 - M.r0;
        const uint8_t* const rp = p.rec + (uint64_t)M.r0 * RB;
        for (uint32_t rb = 0; !DIRECT && rb < R; rb += U * T) {
            Rec x[U];
#pragma unroll
            for (int q = 0; q < U; ++q)
                if (rb + q * T + tid < R) x[q] = take_rec<RB>(rp, rb + q * T + tid);
#pragma unroll
            for (int q = 0; q < U; ++q) {
                if (rb + q * T + tid >= R) break;
                place(x[q]);
            }
        }
        __syncthreads();
        if (tid == 0) take(cur ^ 1, nx);
        clear(cur ^ 1);
        const int64_t N = sh_out.n_nodes;
        int32_t* const status = sh_out.status;
        const int64_t v0 = (b - sh_out.first) << f.sb;
        const int nb = (int)(N - v0 < (int64_t)NB ? N - v0 : (int64_t)NB);
        const bool e_ok = want_e && M.ge + M.ne <= (uint64_t)sh_out.cap_e;
        if (want_e && !e_ok && tid == 0) set_status(status, NN_ERR_CAPACITY);
        auto next_of = [&](uint32_t i) {
            const uint32_t n = link[i];
            return n == 0xffffu ? CHAIN_END : n;
        };

        // 2. one lane per node, one warp per group of 32 nodes
        for (int g = warp; g < GP; g += W) {
            if (__any_sync(FULL, sh_big[cur])) break;
            const int l = g * 32 + lane;
            const bool valid = l < nb;
            const uint32_t c = valid ? c32[l] : 0u, ec = valid && want_e ? c - nfc[l] : c;
            uint32_t pr = 0, pf = 0;  // records and repeated-node records of the groups before
            for (int q = lane; q < g * 32; q += 32) {
                pr += c32[q];
                pf += nfc[q];
            }
            pr = __reduce_add_sync(FULL, pr);
            pf = __reduce_add_sync(FULL, pf);
            const uint32_t cmax = __reduce_max_sync(FULL, c), tmax = min(cmax, (uint32_t)C);
            uint32_t* const ecol = table + (size_t)g * GW + lane;
            uint32_t* const ncol = ecol + EC * 32;
            // 2a. neighbour row
            if (want_n) {
                const uint32_t none = f.nmask;  // above every id: sorts last
                uint32_t w[NW];
                const uint32_t mine = min(c, (uint32_t)C);
                uint32_t nw = K * tmax;
#pragma unroll
                for (int i = 0; i < NW; ++i) w[i] = none;
#pragma unroll
                for (int s0 = 0; s0 < IMAX; s0 += 4) {
                    if ((uint32_t)s0 >= tmax) break;
#pragma unroll
                    for (int s = s0; s < s0 + 4; ++s)
                        if ((uint32_t)s < mine) {
#pragma unroll
                            for (int j = 0; j < K; ++j) w[s * K + j] = ncol[(s * K + j) * 32];
                        }
                }
                uint32_t at = c > (uint32_t)C ? first[l] : CHAIN_END, u;
                for (;;) {
                    sort_prefix(w, nw);
                    // distinct values to the front of the lane's column
                    uint32_t* d = ncol;
                    if (w[0] != none) *d = w[0], d += 32;
#pragma unroll
                    for (int i0 = 1; i0 < NW; i0 += 6) {
                        if ((uint32_t)i0 >= nw) break;
#pragma unroll
                        for (int i = i0; i < i0 + 6 && i < NW; ++i)
                            if (w[i] != none && w[i] != w[i - 1]) *d = w[i], d += 32;
                    }
                    u = (uint32_t)(d - ncol) / 32;
                    if (!__any_sync(FULL, at != CHAIN_END)) break;
                    // lanes with listed records: as many more candidates as
                    // the column takes, and sorted again
                    if (at != CHAIN_END && u + K > (uint32_t)NC) {  // no room: very many distinct neighbours
                        sh_big[cur] = 1;
                        at = CHAIN_END;
                    }
                    while (at != CHAIN_END && u + K <= (uint32_t)NC) {
                        const Rec x = take_rec<RB>(list, at);
                        at = next_of(at);
#pragma unroll
                        for (int j = 0; j < K; ++j) ncol[(u + j) * 32] = rec_nbr<RB>(f, x, j);
                        u += K;
                    }
                    nw = __reduce_max_sync(FULL, u);
#pragma unroll
                    for (int i = 0; i < NW; ++i) w[i] = (uint32_t)i < u ? ncol[i * 32] : none;
                }
                const uint32_t umax = __reduce_max_sync(FULL, u);
#pragma unroll
                for (int i0 = 0; i0 < NW; i0 += 4) {
                    if ((uint32_t)i0 >= umax) break;
#pragma unroll
                    for (int i = i0; i < i0 + 4; ++i)
                        if ((uint32_t)i < u) w[i] = ncol[i * 32];
                }
                uint32_t incl = u;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(FULL, incl, d);
                    if (lane >= d) incl += y;
                }
                const uint32_t gt = __shfl_sync(FULL, incl, 31);
                const size_t gi = (size_t)b * GP + g;
                if (valid && NN_IN(((size_t)b << f.sb) + l, p.nloc_words, status))
                    p.nloc[((size_t)b << f.sb) + l] = incl - u;
                if (lane == 0 && NN_IN(gi, p.ngrp, status)) p.grp[gi] = make_uint2(M.r0 + pr, gt);
                uint32_t* const rows = ncol - lane;  // the group's columns: gt <= 32 NC words
                __syncwarp();
                uint32_t* const d = rows + (incl - u);
#pragma unroll
                for (int i0 = 0; i0 < NW; i0 += 4) {
                    if ((uint32_t)i0 >= umax) break;
#pragma unroll
                    for (int i = i0; i < i0 + 4; ++i)
                        if ((uint32_t)i < u) d[i] = w[i];
                }
                __syncwarp();
                const size_t o = (size_t)K * (M.r0 + pr);
                if (gt == 0 || NN_IN(o + gt - 1, p.ntmp_words, status)) copy_run(p.ntmp + o, rows, gt);
                __syncwarp();
            }
            // 2b. element row: the element ids of the node's records (a
            // repeated node's record adds none)
            if (want_e) {
                uint32_t v[VE];
#pragma unroll
                for (int s = 0; s < VE; ++s) v[s] = EMPTY;
#pragma unroll
                for (int s0 = 0; s0 < IMAX; s0 += 8) {
                    if ((uint32_t)s0 >= tmax) break;
#pragma unroll
                    for (int s = s0; s < s0 + 8 && s < IMAX; ++s)
                        if ((uint32_t)s < min(c, (uint32_t)C)) v[s] = ecol[s * 32];
                }
                if (cmax > (uint32_t)C) {
                    uint32_t at = c > (uint32_t)C ? first[l] : CHAIN_END;
#pragma unroll
                    for (int s = 0; s < VE; ++s) {
                        if (s >= C && at != CHAIN_END) {
                            const Rec x = take_rec<RB>(list, at);
                            at = next_of(at);
                            if (!((rec_side<RB, K>(f, x) >> f.off_nf) & 1u)) v[s] = rec_elem<RB>(f, x);
                        }
                    }
                }
                sort_prefix(v, cmax);
                uint32_t incl = valid ? ec : 0u;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(FULL, incl, d);
                    if (lane >= d) incl += y;
                }
                const uint32_t et = __shfl_sync(FULL, incl, 31), eo = incl - (valid ? ec : 0u);
                const uint64_t ge = M.ge + (pr - pf);
                if (valid && NN_IN(v0 + l, N + 1, status)) sh_out.rp_e[v0 + l] = (int64_t)(ge + eo);
                // put together where the neighbour columns were (without
                // them, in the element columns)
                uint32_t* const rows = want_n ? ncol - lane : ecol - lane;
                if (et > (uint32_t)(want_n ? NC : EC) * 32u) {
                    sh_big[cur] = 1;
                } else {
                    __syncwarp();
                    if (valid) {
#pragma unroll
                        for (int s0 = 0; s0 < VE; s0 += 8) {
                            if ((uint32_t)s0 >= cmax) break;
#pragma unroll
                            for (int s = s0; s < s0 + 8 && s < VE; ++s)
                                if ((uint32_t)s < ec) rows[eo + s] = v[s];
                        }
                    }
                    __syncwarp();
                    if (e_ok) copy_run(reinterpret_cast<uint32_t*>(sh_out.col_e + ge), rows, et);
                }
            }
        }
        if (sh_out.last && tid == 0 && want_e && NN_IN(N, N + 1, status)) sh_out.rp_e[N] = (int64_t)(M.ge + M.ne);
        __syncthreads();
        if (!sh_big[cur]) continue;
        if constexpr (DIRECT) {  // the records, where a partition would have put them
            uint8_t* const dst = const_cast<uint8_t*>(rp);
            gather(b, [&](const Rec& x) { put_rec<RB>(dst, atomicAdd(&sh_direct[5], 1u), x); });
        }

        // 3. the whole CTA: records grouped by node in the spill area, then
        // one warp per group, node by node; rows are sorted in the warp's
        // part of the table when they fit, else in the spill area
        uint32_t* const eoff = table;           // [NB] element offset of each node
        uint32_t* const cursor = table + NB;    // [NB] first record of each node, then its end
        const uint32_t scratch_words = ((uint32_t)GP * GW - 2 * NB) / W;
        bool longer = false;  // a node's candidates exceed the warp's scratch
        {
            const int per = (NB + T - 1) / T, lo = min(NB, tid * per), hi = min(NB, lo + per);
            uint64_t s = 0, total;
            for (int i = lo; i < hi; ++i) {
                s += (uint64_t)c32[i] | ((uint64_t)(c32[i] - nfc[i]) << 32);
                longer |= (uint64_t)K * c32[i] > scratch_words;
            }
            uint64_t run = block_excl_scan(s, &total, sh_scan);
            for (int i = lo; i < hi; ++i) {
                cursor[i] = (uint32_t)run;
                eoff[i] = (uint32_t)(run >> 32);
                run += (uint64_t)c32[i] | ((uint64_t)(c32[i] - nfc[i]) << 32);
            }
        }
        // grouped indices, and K words per record where rows are sorted there
        const uint64_t need = __syncthreads_or(longer) ? (1ull + K) * R : R;
        if (tid == 0 && sh_spill[1] < need) {
            const uint64_t base = atomicAdd(p.spill_cursor, (unsigned long long)need);
            if (base + need <= p.spill_words) {
                sh_spill[0] = base;
                sh_spill[1] = need;
            } else {
                set_status(status, NN_ERR_WORKSPACE);
            }
        }
        __syncthreads();
        const bool ok = sh_spill[1] >= need;
        uint32_t* const grp = p.spill + sh_spill[0];
        for (uint32_t r = tid; ok && r < R; r += T)
            grp[atomicAdd(&cursor[rec_side<RB, K>(f, take_rec<RB>(rp, r)) & vmask], 1u)] = r;
        __syncthreads();
        uint32_t* const scratch = table + 2 * NB + warp * scratch_words;
        for (int g = warp; g < GP; g += W) {
            uint32_t run = 0, pr = 0;
            for (int i = 0; i < 32; ++i) {
                const int l = g * 32 + i;
                if (l >= nb) break;
                const uint32_t c = c32[l], o = cursor[l] - (ok ? c : 0u), ec = c - nfc[l];
                uint32_t* const a = (uint64_t)K * c <= scratch_words ? scratch : grp + R + (uint64_t)K * o;
                if (i == 0) pr = o;
                if (want_e) {
                    if (lane == 0 && NN_IN(v0 + l, N + 1, status)) sh_out.rp_e[v0 + l] = (int64_t)(M.ge + eoff[l]);
                    if (ok && e_ok && c) {
                        warp_elem_row<RB, K>(sh_fmt, rp, grp + o, c, a, ec);
                        for (uint32_t k = lane; k < ec; k += 32) sh_out.col_e[M.ge + eoff[l] + k] = (int32_t)a[k];
                        __syncwarp();
                    }
                }
                if (want_n) {
                    uint32_t u = 0;
                    if (ok && c) {
                        u = warp_node_row<RB, K>(sh_fmt, rp, grp + o, c, a);
                        const size_t d = (size_t)K * (M.r0 + pr) + run;
                        if (u == 0 || NN_IN(d + u - 1, p.ntmp_words, status))
                            for (uint32_t k = lane; k < u; k += 32) p.ntmp[d + k] = a[k];
                        __syncwarp();
                    }
                    if (lane == 0 && NN_IN(((size_t)b << f.sb) + l, p.nloc_words, status))
                        p.nloc[((size_t)b << f.sb) + l] = run;
                    run += u;
                }
            }
            if (want_n && lane == 0 && NN_IN((size_t)b * GP + g, p.ngrp, status))
                p.grp[(size_t)b * GP + g] = make_uint2(M.r0 + pr, run);
        }
        __syncthreads();
    }
}

// Allow up to `bytes` of dynamic shared memory, less the kernel's own static
// shared memory (the sum may not exceed the per-block opt-in limit).
template <int RB, int K, int IMAX, bool DIRECT>
cudaError_t set_attr(size_t bytes) {
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, k_bucket<RB, K, IMAX, DIRECT>);
    if (e != cudaSuccess) return e;
    const size_t dyn = bytes > a.sharedSizeBytes ? bytes - a.sharedSizeBytes : 0;
    return cudaFuncSetAttribute(k_bucket<RB, K, IMAX, DIRECT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
}

// Launcher, shared-memory limit and occupancy of the IMAX variants (one
// translation unit each, so that they compile side by side).
template <int IMAX, bool DIRECT = false>
cudaError_t launch_bucket_t(const BucketParams& p, int grid, int threads, size_t smem, cudaStream_t s) {
    if (p.fmt.rb == 8) {
        return launch_chained(p.chain, p.fmt.k == 2 ? k_bucket<8, 2, IMAX, DIRECT> : k_bucket<8, 3, IMAX, DIRECT>, grid, threads,
                              smem, s, p);
    }
    return launch_chained(p.chain, p.fmt.k == 2 ? k_bucket<16, 2, IMAX, DIRECT> : k_bucket<16, 3, IMAX, DIRECT>, grid, threads,
                          smem, s, p);
}

template <int IMAX, bool DIRECT = false>
cudaError_t set_bucket_smem_t(size_t bytes) {
    cudaError_t e = set_attr<8, 2, IMAX, DIRECT>(bytes);
    if (e == cudaSuccess) e = set_attr<8, 3, IMAX, DIRECT>(bytes);
    if (e == cudaSuccess) e = set_attr<16, 2, IMAX, DIRECT>(bytes);
    if (e == cudaSuccess) e = set_attr<16, 3, IMAX, DIRECT>(bytes);
    return e;
}

template <int IMAX>
cudaError_t bucket_occupancy_t(int* blocks, int threads, size_t smem) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, k_bucket<16, 3, IMAX, false>, threads, smem);
}

}  // namespace

}  // namespace nn
