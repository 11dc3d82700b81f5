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
// Hard nodes are those that a lane cannot finish: more records than its
// registers hold, records that the list had no room for, more distinct
// neighbours than a column.  The launch over all buckets only notes a bucket
// that has some; a second launch (REST) builds the noted buckets, with up to 32
// slots per node, finishing first what is still hard there, a node by one warp
// with its values in registers, or by the whole CTA when they are too many.
// (Small meshes, one bucket per CTA, do so at once.)  Such a bucket used to be
// built node by node by its whole CTA, a warp per 32 of them.  GB300, whole
// builds, then and now: 150,000 points' Delaunay tets 888 -> 442 us, a 1000^2
// triangle surface with one node of 30 triangles in 256 1046 -> 313 us, tets
// on 30 % of their mesh's node ids 1100 -> 333 us, a fan of 20,000 triangles
// 25.8 -> 1.2 ms.
//
// What bounds it: instructions (issue slots 63 % busy on hexes), then
// instruction fetch where the networks are long (tets) and shared-memory
// stores.  Before, records were staged in shared memory, counted, scanned and
// gathered by index twice at 16 warps per SM (issue 31-49 %), and tets went
// through a hash table per lane.  GB300, both results, before and now:
// hex 257^3 2.30 -> 1.37 ms, tet 161^3 3.08 -> 1.32 ms, hex/tet mixed 257^3
// 8.35 -> 4.47 ms, triangles 2048^2 with holes 0.48 -> 0.26 ms.
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
constexpr uint32_t HARD = 0x80000000u;  // in a node's count of repeated-node records: not left to its lane

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

// One warp finishes a hard node (rare on most meshes, ordinary on some: hubs,
// 3-d Delaunay meshes, parts that use few of a mesh's node ids), its values in
// LV registers per lane, value 32 i + lane in register i.
constexpr int LV = 16;
// ... and of so many records at most; above, the whole CTA does.
__host__ __device__ constexpr uint32_t warp_records(int k) { return LV / k * 32; }

// Ascending bitonic sort of 32 LV values; those from 32 used on are EMPTY and
// need no step (used: a power of two, the same in all lanes).
__device__ __forceinline__ void lane_sort(uint32_t (&v)[LV], uint32_t used) {
    const uint32_t lane = threadIdx.x & 31, P = used * 32;
    for (uint32_t k = 2; k <= P; k <<= 1) {
#pragma unroll
        for (int jr = LV / 2; jr >= 1; jr >>= 1) {  // partners in the same lane
            if (jr * 32u >= k) continue;
#pragma unroll
            for (int i = 0; i < LV; ++i) {
                if ((i & jr) || (uint32_t)i >= used) continue;
                const uint32_t x = v[i], y = v[i | jr];
                const bool up = ((i * 32u) & k) == 0;
                v[i] = up ? min(x, y) : max(x, y);
                v[i | jr] = up ? max(x, y) : min(x, y);
            }
        }
        for (uint32_t j = min(k >> 1, 16u); j >= 1; j >>= 1) {
#pragma unroll
            for (int i = 0; i < LV; ++i) {
                if ((uint32_t)i >= used) continue;
                const uint32_t y = __shfl_xor_sync(FULL, v[i], j);
                v[i] = (((i * 32u + lane) & k) == 0) == ((lane & j) == 0) ? min(v[i], y) : max(v[i], y);
            }
        }
    }
}
// The distinct ones of sorted values below `none`, to a[0..).  Returns their count.
__device__ __forceinline__ uint32_t put_distinct(const uint32_t (&v)[LV], uint32_t none, uint32_t used, uint32_t* a) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t n = 0, carry = none;
#pragma unroll
    for (int i = 0; i < LV; ++i) {
        if ((uint32_t)i >= used) continue;
        uint32_t prev = __shfl_up_sync(FULL, v[i], 1);
        if (lane == 0) prev = carry;
        carry = __shfl_sync(FULL, v[i], 31);
        const bool keep = v[i] < none && v[i] != prev;
        const unsigned m = __ballot_sync(FULL, keep);
        if (keep) a[n + __popc(m & lanemask_lt())] = v[i];
        n += __popc(m);
    }
    return n;
}

// Both rows of a node of c <= warp_records(K) records, at idx[0 .. c) of the
// bucket's: the distinct neighbours to nbrs (nullptr: not wanted), the first
// ec element ids to elems (nullptr: not wanted, or no room).  Returns the
// number of neighbours.
template <int RB, int K>
__device__ __noinline__ uint32_t warp_rows(const RecFmt& f, const uint8_t* rp, const uint32_t* idx, uint32_t c,
                                           uint32_t* nbrs, int32_t* elems, uint32_t ec) {
    constexpr int S = LV / K;  // records of a lane
    const uint32_t lane = threadIdx.x & 31, per = (c + 31) / 32;
    uint32_t v[LV], e[S], u = 0;
#pragma unroll
    for (int i = 0; i < LV; ++i) v[i] = EMPTY;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        e[s] = EMPTY;
        if (s * 32u + lane < c) {
            const Rec x = take_rec<RB>(rp, idx[s * 32 + lane]);
            if (!((rec_side<RB, K>(f, x) >> f.off_nf) & 1u) || !elems) e[s] = rec_elem<RB>(f, x);
#pragma unroll
            for (int j = 0; j < K; ++j) v[s * K + j] = rec_nbr<RB>(f, x, j);
        }
    }
    if (nbrs) {
        uint32_t used = 1;
        while (used < per * K) used *= 2;
        lane_sort(v, used);
        u = put_distinct(v, f.nmask, used, nbrs);
    }
    if (elems) {
        uint32_t used = 1;
        while (used < per) used *= 2;
#pragma unroll
        for (int i = 0; i < LV; ++i) v[i] = i < S ? e[i < S ? i : 0] : EMPTY;
        lane_sort(v, used);
#pragma unroll
        for (int i = 0; i < S; ++i)
            if (i * 32u + lane < ec) elems[i * 32 + lane] = (int32_t)v[i];
    }
    __syncwarp();
    return u;
}

// The neighbour row of a node whose column is full: its u <= 96 distinct
// values so far (col, 32 words apart) and the records listed from `at` on (at
// most 64: a node of more is not left to its lane), to row.
template <int RB, int K>
__device__ __noinline__ uint32_t warp_listed_row(const RecFmt& f, const uint32_t* col, uint32_t u, const uint8_t* list,
                                                 const uint16_t* link, uint32_t at, uint32_t* row) {
    constexpr int COL = 3;  // registers of the column
    static_assert(COL + 2 * K <= LV, "registers of a full column and its listed records");
    const uint32_t lane = threadIdx.x & 31;
    uint32_t mine[2] = {0xffffu, 0xffffu}, n = 0;
    for (; at != 0xffffu && n < 64; at = link[at], ++n)
        if ((n & 31) == lane) mine[n >> 5] = at;
    uint32_t v[LV];
#pragma unroll
    for (int i = 0; i < LV; ++i) v[i] = i < COL && i * 32u + lane < u ? col[(i * 32 + lane) * 32] : EMPTY;
#pragma unroll
    for (int s = 0; s < 2; ++s)
        if (mine[s] != 0xffffu) {
            const Rec x = take_rec<RB>(list, mine[s]);
#pragma unroll
            for (int j = 0; j < K; ++j) v[COL + s * K + j] = rec_nbr<RB>(f, x, j);
        }
    constexpr uint32_t used = pow2_ceil(COL + 2 * K);
    lane_sort(v, used);
    return put_distinct(v, f.nmask, used, row);
}

// Ascending bitonic sort of a[0..n) in global memory by the whole CTA, in the
// formulation whose compare-exchanges put the minimum at the lower index, so
// that indices >= n act as +infinity and are skipped.
__device__ inline void block_sort(uint32_t* a, uint32_t n) {
    uint32_t P = 1;
    while (P < n) P <<= 1;
    for (uint32_t k = 2; k <= P; k <<= 1) {
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t t = threadIdx.x; t < (P >> 1); t += blockDim.x) {
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
            __syncthreads();
        }
    }
}

// The rows of a node of any number of records by the whole CTA (see
// warp_rows): nbrs has room for K c words, idx is overwritten.
template <int RB, int K>
__device__ __noinline__ uint32_t block_rows(const RecFmt& f, const uint8_t* rp, uint32_t* idx, uint32_t c, uint32_t* nbrs,
                                            int32_t* elems, uint32_t ec, uint64_t* sh_scan) {
    uint32_t u = 0;
    if (nbrs) {
        const uint32_t n = K * c;
        for (uint32_t s = threadIdx.x; s < c; s += blockDim.x) {
            const Rec x = take_rec<RB>(rp, idx[s]);
#pragma unroll
            for (int j = 0; j < K; ++j) nbrs[(size_t)s * K + j] = rec_nbr<RB>(f, x, j);
        }
        __syncthreads();
        block_sort(nbrs, n);
        // keep the first of every run (writes never pass the part being read)
        for (uint32_t i0 = 0; i0 < n; i0 += blockDim.x) {
            const uint32_t i = i0 + threadIdx.x;
            const uint32_t x = i < n ? nbrs[i] : f.nmask, prev = i > 0 && i < n ? nbrs[i - 1] : f.nmask;
            const bool keep = x != f.nmask && x != prev;
            uint64_t total;
            const uint64_t at = block_excl_scan(keep ? 1u : 0u, &total, sh_scan);
            if (keep) nbrs[u + at] = x;
            u += (uint32_t)total;
            __syncthreads();
        }
    }
    if (elems) {
        for (uint32_t s = threadIdx.x; s < c; s += blockDim.x) {
            const Rec x = take_rec<RB>(rp, idx[s]);
            idx[s] = (rec_side<RB, K>(f, x) >> f.off_nf) & 1u ? EMPTY : rec_elem<RB>(f, x);
        }
        __syncthreads();
        block_sort(idx, c);
        for (uint32_t i = threadIdx.x; i < ec; i += blockDim.x) elems[i] = (int32_t)idx[i];
        __syncthreads();
    }
    return u;
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

// n words to a place that is not above theirs, within global memory, by one warp.
__device__ __forceinline__ void move_run(uint32_t* dst, const uint32_t* src, uint32_t n) {
    if (dst == src) return;
    for (uint32_t i0 = 0; i0 < n; i0 += 32) {
        const uint32_t i = i0 + (threadIdx.x & 31);
        const uint32_t x = i < n ? src[i] : 0u;
        __syncwarp();
        if (i < n) dst[i] = x;
        __syncwarp();
    }
}
// The neighbour rows of a group in which some are not left to their lanes:
// `hard` ones, already at K words per record of the nodes before them in dst,
// and those of lanes whose column is full (rest: the first of the listed
// records that did not go in), which are finished here and put aside the same
// way.  u distinct values of a lane's c records are in its column; of a hard
// one's, u is the row's length.  No row's place is above where it was put
// aside, and none reaches the place where a later one was.
template <int RB, int K>
__device__ __noinline__ void put_aside(const RecFmt& f, const uint32_t* ncol, uint32_t u, uint32_t c, bool hard,
                                       uint32_t rest, const uint8_t* list, const uint16_t* link, uint32_t* dst,
                                       uint32_t* nloc, uint2* grp, uint32_t r0) {
    const uint32_t lane = threadIdx.x & 31;
    const unsigned full = __ballot_sync(FULL, rest != CHAIN_END), aside = full | __ballot_sync(FULL, hard);
    uint32_t before = c;  // records of the lanes before
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, before, d);
        if (lane >= d) before += y;
    }
    before -= c;
    __syncwarp();
    for (unsigned m = full; m; m &= m - 1) {
        const int i = __ffs(m) - 1;
        const uint32_t ui = __shfl_sync(FULL, u, i), ri = __shfl_sync(FULL, rest, i), bi = __shfl_sync(FULL, before, i);
        const uint32_t n = warp_listed_row<RB, K>(f, ncol - lane + i, ui, list, link, ri, dst + (size_t)K * bi);
        if (lane == i) u = n;
    }
    __syncwarp();
    uint32_t incl = u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += y;
    }
    if (nloc) *nloc = incl - u;
    if (grp && lane == 31) *grp = make_uint2(r0, incl);
    for (unsigned m = aside; m; m &= m - 1) {
        const int i = __ffs(m) - 1;
        const uint32_t n = __shfl_sync(FULL, u, i), at = __shfl_sync(FULL, incl, i) - n;
        move_run(dst + at, dst + (size_t)K * __shfl_sync(FULL, before, i), n);
    }
    __syncwarp();
    if (!((aside >> lane) & 1u))
        for (uint32_t i = 0; i < u; ++i) dst[incl - u + i] = ncol[i * 32];
    __syncwarp();
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
__host__ __device__ constexpr size_t list_bytes(int rb, int cap) { return ((size_t)cap * (rb + 2) + 15) / 16 * 16; }

// Registers: VE element ids and NW neighbour candidates of a node.  IMAX
// bounds the slots; a node of more than VE records is hard.  8 slots
// (triangles, quads, hexes): 64 registers, 32 warps per SM; 32 slots (tets):
// 128 and 16.
template <int K, int IMAX>
struct Regs {
    static constexpr int VE = IMAX == 8 ? 24 : 2 * IMAX;
    static constexpr int NW = K * IMAX > 32 ? K * IMAX : 32;
    static constexpr int MIN_CTAS = IMAX == 8 ? 4 : (IMAX == 16 ? 3 : 2);
};

// What the out-of-line part of the bucket pass needs besides the bucket's own
// tables (in shared memory).
struct HardArea {
    uint32_t* spill;              // the spill area
    uint64_t spill_words;
    unsigned long long* cursor;   // ... and its first free word
    uint32_t* ntmp;
    uint64_t ntmp_words;          // (bounds-checked builds)
    uint64_t first, words;        // this CTA's part of the spill area
    uint32_t records;             // of the bucket's hard nodes
    uint64_t scan[34];
};

// Places for the record indices of a bucket's hard nodes in the spill area,
// one node after another: first[] of a hard node is its first place.  All
// threads; c32 points at the bucket's counters.
__device__ __noinline__ bool hard_begin(HardArea& a, uint32_t* c32, int NB, int32_t* status) {
    uint32_t *const nfc = c32 + NB, *const first = nfc + NB;
    if (threadIdx.x == 0) a.records = 0;
    __syncthreads();
    for (int l = threadIdx.x; l < NB; l += blockDim.x)
        if (nfc[l] & HARD) first[l] = atomicAdd(&a.records, c32[l]);
    __syncthreads();
    if (threadIdx.x == 0 && a.words < a.records) {
        const uint64_t base = atomicAdd(a.cursor, (unsigned long long)a.records);
        if (base + a.records <= a.spill_words) {
            a.first = base;
            a.words = a.records;
        } else {
            set_status(status, NN_ERR_WORKSPACE);
        }
    }
    __syncthreads();
    return a.words >= a.records;
}

// Both rows of a bucket's hard nodes, whose record indices stand in the spill
// area (ok; else their rows stay empty).  The element row goes to its place,
// the neighbour row to the node's part of the scratch area (K words per
// record), from where its group's warp fetches it; its length takes the place
// of the indices' end in first[].  All threads: first the nodes that a warp
// can do, in turn, then the others.
template <int RB, int K>
__device__ __noinline__ void hard_rows(const RecFmt& f, const BucketOut& out, HardArea& a, uint32_t* c32, const uint8_t* rp,
                                       uint32_t r0, uint64_t ge0, bool e_ok, bool ok) {
    const int NB = 1 << f.sb, lane = threadIdx.x & 31, W = blockDim.x >> 5, warp = threadIdx.x >> 5;
    uint32_t *const nfc = c32 + NB, *const first = nfc + NB;
    __syncthreads();
    for (int big = 0; big < 2; ++big) {
        int turn = 0;
        for (int l0 = 0; l0 < NB; l0 += 32) {
            for (unsigned m = __ballot_sync(FULL, l0 + lane < NB && (nfc[l0 + lane] & HARD)); m; m &= m - 1) {
                const int l = l0 + __ffs(m) - 1;
                const uint32_t c = c32[l];
                if ((c > warp_records(K)) != (big != 0)) continue;
                if (!big && turn++ % W != warp) continue;
                uint32_t pr = 0, pf = 0;  // records and repeated-node records before the node
                for (int q = lane; q < l; q += 32) {
                    pr += c32[q];
                    pf += nfc[q] & ~HARD;
                }
                pr = __reduce_add_sync(FULL, pr);
                pf = __reduce_add_sync(FULL, pf);
                const uint32_t ec = c - (nfc[l] & ~HARD);
                const uint64_t ge = ge0 + (pr - pf);
                const size_t o = (size_t)K * (r0 + pr);
                uint32_t* const nbrs =
                    (f.want & NN_WANT_NODES) && NN_IN(o + (size_t)K * c - 1, a.ntmp_words, out.status) ? a.ntmp + o : nullptr;
                int32_t* const elems = e_ok && ge + ec <= (uint64_t)out.cap_e ? out.col_e + ge : nullptr;
                uint32_t u = 0;
                if (ok) {
                    uint32_t* const idx = a.spill + a.first + (first[l] - c);
                    u = big ? block_rows<RB, K>(f, rp, idx, c, nbrs, elems, ec, a.scan)
                            : warp_rows<RB, K>(f, rp, idx, c, nbrs, elems, ec);
                }
                if (big) __syncthreads();
                else __syncwarp();
                if (lane == 0 && (!big || warp == 0)) first[l] = u;
            }
        }
    }
    __syncthreads();
}

// hard_begin, the record indices of a partitioned bucket and hard_rows.
template <int RB, int K>
__device__ __noinline__ void hard_nodes(const RecFmt& f, const BucketOut& out, HardArea& a, uint32_t* c32, const uint8_t* rp,
                                        const BucketMeta& M, bool e_ok) {
    const int NB = 1 << f.sb;
    const uint32_t R = M.r1 - M.r0;
    uint32_t *const nfc = c32 + NB, *const first = nfc + NB;
    const bool ok = hard_begin(a, c32, NB, out.status);
    uint32_t* const idx = a.spill + a.first;
    for (uint32_t r = threadIdx.x; ok && r < R; r += blockDim.x) {
        const uint32_t v = rec_side<RB, K>(f, take_rec<RB>(rp, r)) & (uint32_t)(NB - 1);
        if (nfc[v] & HARD) idx[atomicAdd(&first[v], 1u)] = r;
    }
    hard_rows<RB, K>(f, out, a, c32, rp, M.r0, M.ge, e_ok, ok);
}

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

// Which buckets a launch builds: PLAIN, all in ticket order, where a bucket
// with hard nodes is noted for the REST launch that follows; DIRECT_BUILD, one
// per CTA (small meshes), hard nodes included; REST, the noted ones.  The paths
// for hard nodes have their own launch because they cost the others registers:
// in one kernel, inline or out of line, hex 257^3 took 1540 to 1650 us instead
// of 1366, tet 161^3 1420 to 1440 instead of 1317.  An empty REST launch costs
// 1 to 4 us of a build (triangles 120^2 30.7 -> 32.6 us, 939^2 162 -> 166 us).
enum Mode { PLAIN, DIRECT_BUILD, REST };

template <int RB, int K, int IMAX, int MODE>
__global__ void __launch_bounds__(MODE == DIRECT_BUILD ? direct_threads(IMAX) : 256,
                                  MODE == DIRECT_BUILD ? 1 : Regs<K, IMAX>::MIN_CTAS) k_bucket(BucketParams p) {
    chain_begin();
    constexpr bool DIRECT = MODE == DIRECT_BUILD;
    constexpr bool SLOW = MODE != PLAIN;  // hard nodes are finished here
    const uint32_t n_rest = MODE == REST ? *p.rest_count : 0u;
    if (MODE == REST && n_rest == 0) return;
    constexpr int VE = Regs<K, IMAX>::VE, NW = Regs<K, IMAX>::NW;
    constexpr int U = 4;  // records a thread loads at once
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ BucketOut sh_out;
    __shared__ BucketMeta meta[2];
    __shared__ uint32_t sh_list[2];   // listed records (of this bucket, of the next)
    __shared__ uint32_t sh_big[2];    // the bucket has nodes that are not left to a lane (this one, the next)
    __shared__ RecFmt sh_fmt;         // for the out-of-line helpers
    __shared__ __align__(8) uint8_t sh_area_raw[SLOW ? sizeof(HardArea) : 8];
    HardArea& sh_area = *reinterpret_cast<HardArea*>(sh_area_raw);
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
    // one thread: bounds and element offset of bucket t (REST: the t-th noted one); its records are pulled into L2
    auto take = [&](int slot, uint32_t t) {
        if (MODE == REST) t = t < n_rest ? p.rest[t] : (uint32_t)n_buckets;
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
        if constexpr (SLOW) {
            sh_area.spill = p.spill;
            sh_area.spill_words = p.spill_words;
            sh_area.cursor = p.spill_cursor;
            sh_area.ntmp = p.ntmp;
            sh_area.ntmp_words = p.ntmp_words;
            sh_area.first = sh_area.words = 0;
        }
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
                    if (SLOW) atomicOr(&nfc[v], HARD);
                    sh_big[cur] = 1;
                }
            }
        };
        if constexpr (DIRECT) {
            gather(b, place);
            for (int l = tid; l < NB; l += T) {
                if (c32[l]) atomicAdd(&sh_direct[3], c32[l]);
                if (nfc[l] & ~HARD) atomicAdd(&sh_direct[4], nfc[l] & ~HARD);
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

        // 2. the nodes that are not left to a lane
        if (SLOW && sh_big[cur]) {
            if constexpr (DIRECT) {  // their records, where a partition would have put the bucket's
                const bool ok = hard_begin(sh_area, c32, NB, status);
                uint32_t* const idx = p.spill + sh_area.first;
                uint8_t* const dst = const_cast<uint8_t*>(rp);
                if (ok)
                    gather(b, [&](const Rec& x) {
                        const uint32_t v = rec_side<RB, K>(f, x) & vmask;
                        if (!(nfc[v] & HARD)) return;
                        const uint32_t r = atomicAdd(&sh_direct[5], 1u);
                        put_rec<RB>(dst, r, x);
                        idx[atomicAdd(&first[v], 1u)] = r;
                    });
                hard_rows<RB, K>(sh_fmt, sh_out, sh_area, c32, rp, M.r0, M.ge, e_ok, ok);
            } else if constexpr (SLOW) {
                hard_nodes<RB, K>(sh_fmt, sh_out, sh_area, c32, rp, meta[cur], e_ok);
            }
        }

        // 3. one lane per node, one warp per group of 32 nodes
        for (int g = warp; g < GP; g += W) {
            if (!SLOW && __any_sync(FULL, sh_big[cur])) break;
            const int l = g * 32 + lane;
            const bool valid = l < nb;
            const uint32_t c = valid && !(SLOW && (nfc[l] & HARD)) ? c32[l] : 0u;  // records left to the lane
            uint32_t pr = 0, pf = 0;  // records and repeated-node records of the groups before
            for (int q = lane; q < g * 32; q += 32) {
                pr += c32[q];
                pf += nfc[q] & ~HARD;
            }
            pr = __reduce_add_sync(FULL, pr);
            pf = __reduce_add_sync(FULL, pf);
            const uint32_t cmax = __reduce_max_sync(FULL, c), tmax = min(cmax, (uint32_t)C);
            uint32_t* const ecol = table + (size_t)g * GW + lane;
            uint32_t* const ncol = ecol + EC * 32;
            // 3a. neighbour row
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
                    // lanes with listed records: as many more candidates as
                    // the column takes, and sorted again (a column may be full
                    // before the list is used up)
                    if (!SLOW && at != CHAIN_END && u + K > (uint32_t)NC) {
                        sh_big[cur] = 1;
                        at = CHAIN_END;
                    }
                    if (!__any_sync(FULL, at != CHAIN_END && u + K <= (uint32_t)NC)) break;
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
                const size_t gi = (size_t)b * GP + g, o = (size_t)K * (M.r0 + pr);
                if (SLOW && __any_sync(FULL, at != CHAIN_END || (valid && (nfc[l] & HARD)))) {
                    const uint32_t ca = valid ? c32[l] : 0u;
                    const bool hard = valid && (nfc[l] & HARD);
                    const bool in = NN_IN(o + (size_t)K * __reduce_add_sync(FULL, ca) - 1, p.ntmp_words, status);
                    uint32_t* const nloc = valid && NN_IN(((size_t)b << f.sb) + l, p.nloc_words, status)
                                               ? p.nloc + ((size_t)b << f.sb) + l : nullptr;
                    if (in)
                        put_aside<RB, K>(sh_fmt, ncol, hard ? first[l] : u, ca, hard, at, list, link, p.ntmp + o, nloc,
                                         NN_IN(gi, p.ngrp, status) ? p.grp + gi : nullptr, M.r0 + pr);
                } else {
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
                    if (gt == 0 || NN_IN(o + gt - 1, p.ntmp_words, status)) copy_run(p.ntmp + o, rows, gt);
                    __syncwarp();
                }
            }
            // 3b. element row: the element ids of the node's records (a
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
                const bool hard = SLOW && valid && (nfc[l] & HARD);
                const uint32_t ec = valid ? c32[l] - (nfc[l] & ~HARD) : 0u;
                uint32_t incl = ec;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(FULL, incl, d);
                    if (lane >= d) incl += y;
                }
                const uint32_t et = __shfl_sync(FULL, incl, 31), eo = incl - ec;
                const uint64_t ge = M.ge + (pr - pf);
                if (valid && NN_IN(v0 + l, N + 1, status)) sh_out.rp_e[v0 + l] = (int64_t)(ge + eo);
                // put together where the neighbour columns were (without
                // them, in the element columns); written one by one where that
                // is too small or rows of 2. lie between.  (The bucket's total
                // is the offsets' own: with overlapping elements of an invalid
                // mesh the records that were kept may have more entries.)
                uint32_t* const rows = want_n ? ncol - lane : ecol - lane;
                const bool in = e_ok && ge + et <= (uint64_t)sh_out.cap_e;
                if (!SLOW && et > (uint32_t)(want_n ? NC : EC) * 32u) {
                    sh_big[cur] = 1;
                } else if (SLOW && (et > (uint32_t)(want_n ? NC : EC) * 32u || __any_sync(FULL, hard))) {
                    int32_t* const d = sh_out.col_e + ge + eo;
#pragma unroll
                    for (int s = 0; s < VE; ++s)
                        if (in && !hard && (uint32_t)s < ec) d[s] = (int32_t)v[s];
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
                    if (in) copy_run(reinterpret_cast<uint32_t*>(sh_out.col_e + ge), rows, et);
                }
            }
        }
        if (sh_out.last && tid == 0 && want_e && NN_IN(N, N + 1, status)) sh_out.rp_e[N] = (int64_t)(M.ge + M.ne);
        __syncthreads();
        if (!SLOW && tid == 0 && sh_big[cur] && NN_IN(b, p.rest_cap, status)) p.rest[atomicAdd(p.rest_count, 1u)] = (uint32_t)b;
    }
}

// Allow up to `bytes` of dynamic shared memory, less the kernel's own static
// shared memory (the sum may not exceed the per-block opt-in limit).
template <int RB, int K, int IMAX, int MODE>
cudaError_t set_attr(size_t bytes) {
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, k_bucket<RB, K, IMAX, MODE>);
    if (e != cudaSuccess) return e;
    const size_t dyn = bytes > a.sharedSizeBytes ? bytes - a.sharedSizeBytes : 0;
    return cudaFuncSetAttribute(k_bucket<RB, K, IMAX, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
}

// Launcher, shared-memory limit and occupancy of the IMAX variants (one
// translation unit each, so that they compile side by side).
template <int IMAX, int MODE = PLAIN>
cudaError_t launch_bucket_t(const BucketParams& p, int grid, int threads, size_t smem, cudaStream_t s) {
    if (p.fmt.rb == 8) {
        return launch_chained(p.chain, p.fmt.k == 2 ? k_bucket<8, 2, IMAX, MODE> : k_bucket<8, 3, IMAX, MODE>, grid, threads,
                              smem, s, p);
    }
    return launch_chained(p.chain, p.fmt.k == 2 ? k_bucket<16, 2, IMAX, MODE> : k_bucket<16, 3, IMAX, MODE>, grid, threads,
                          smem, s, p);
}

template <int IMAX, int MODE = PLAIN>
cudaError_t set_bucket_smem_t(size_t bytes) {
    cudaError_t e = set_attr<8, 2, IMAX, MODE>(bytes);
    if (e == cudaSuccess) e = set_attr<8, 3, IMAX, MODE>(bytes);
    if (e == cudaSuccess) e = set_attr<16, 2, IMAX, MODE>(bytes);
    if (e == cudaSuccess) e = set_attr<16, 3, IMAX, MODE>(bytes);
    return e;
}

template <int IMAX>
cudaError_t bucket_occupancy_t(int* blocks, int threads, size_t smem) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, k_bucket<16, 3, IMAX, PLAIN>, threads, smem);
}

}  // namespace

}  // namespace nn
