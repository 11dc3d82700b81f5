// Device helpers shared by the libnn kernels: status reporting, bounded
// decoupled lookback, block scans, record packing and element edge tables.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "nn_internal.h"

namespace nn {

constexpr uint32_t EMPTY = 0xFFFFFFFFu;
// A bounded wait gives up after this long without progress (ns).
constexpr uint64_t WAIT_LIMIT_NS = 2000000000ull;

__device__ __forceinline__ void set_status(int32_t* st, int32_t code) { atomicCAS(st, 0, code); }

// Bounds-checked build (compiled with -DNN_CHECKED into libnn_checked.so):
// NN_IN(i, n, status) is false when index i lies outside a buffer of n
// elements, after recording NN_ERR_BOUNDS; the caller then skips the access.
// In the ordinary build it is the constant true and costs nothing.
__device__ __forceinline__ bool in_bounds(uint64_t i, uint64_t n, int32_t* st) {
    if (i < n) return true;
    set_status(st, NN_ERR_BOUNDS);
    return false;
}
#ifdef NN_CHECKED
#define NN_IN(i, n, st) (::nn::in_bounds((uint64_t)(i), (uint64_t)(n), (st)))
#else
#define NN_IN(i, n, st) true
#endif

// Programmatic dependent launch: a kernel of one launch sequence is set up
// while the one before it still runs, and its CTAs become resident as soon as
// there is room for them.  Each kernel that is launched so begins with
// chain_begin(): it waits until the kernel before it is complete and its
// writes are visible, then lets the next one be set up.  (A kernel waits for
// its predecessor alone, which has waited for its own.)  What earlier kernels
// of the sequence have written is read with ordinary loads; __ldg is for the
// caller's mesh, which does not change while any of them is there.  Builds
// of up to CHAIN_RECORDS incidences are launched so: between kernels of a few
// microseconds the launches are a good part of the time (one call after
// another: 1.76 M triangles 174 -> 165 us, 1 M quads' node rows 138 -> 124 us,
// 24 meshes in a batch 483 -> 463 us, a tet mesh in chunks of 5 M incidences
// 1411 -> 1347 us, triangles 64^2 24 -> 18 us).  Larger ones are not: at 24 M
// incidences it gave nothing (triangles) or cost 5 % (element rows of tets),
// at 134 M (hexes) 2 %.
__device__ __forceinline__ void chain_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Launch k; chained: right after another kernel of this library in stream s.
template <class... KA, class... A>
inline cudaError_t launch_chained(bool chained, void (*k)(KA...), unsigned grid, unsigned threads, size_t smem, cudaStream_t s,
                                  A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&c, k, KA(args)...);
}

__device__ __forceinline__ uint64_t ld_acquire(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(uint64_t* p, uint64_t v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ---------------------------------------------------------------- lookback
// Single-pass scan across tiles taken in ticket order.  Word layout: bits
// 62-63 flag (0 not ready, 1 tile aggregate, 2 inclusive prefix), bits 0-61
// the value.  Every predecessor of a tile holds an earlier ticket, so it is
// running or done; the wait is still bounded and reports NN_ERR_TIMEOUT.
constexpr uint64_t LB_AGG = 1ull << 62;
constexpr uint64_t LB_INC = 2ull << 62;
constexpr uint64_t LB_VAL = (1ull << 62) - 1;

// Warp-parallel lookback in two halves.  lb_publish (one thread) makes the
// tile's aggregate visible as soon as it is known; lb_resolve (all 32 lanes
// of one warp, possibly much later) walks back over the predecessors, 32 at
// a time, consuming the ready ones nearest to t and stopping at the first
// inclusive prefix, then publishes t's inclusive prefix.  Only the nearest
// not-yet-ready predecessor is ever waited for.
// `first` is the first tile of t's chain (a batch restarts the scan at every
// mesh): tiles before it count as an inclusive zero.
__device__ __forceinline__ void lb_publish(uint64_t* state, uint64_t t, uint64_t agg, uint64_t first = 0) {
    st_release(&state[t], (t == first ? LB_INC : LB_AGG) | agg);
}

__device__ inline uint64_t lb_resolve(uint64_t* state, uint64_t t, uint64_t agg, int32_t* status,
                                      uint64_t first = 0) {
    const int lane = threadIdx.x & 31;
    if (t == first) return 0;
    uint64_t excl = 0;
    int64_t p = (int64_t)t - 1;
    uint64_t t0 = 0;
    for (;;) {
        const int64_t idx = p - lane;
        const uint64_t s = idx >= (int64_t)first ? ld_acquire(&state[idx]) : LB_INC;  // before the chain: zero
        const unsigned not_ready = __ballot_sync(0xffffffffu, (s >> 62) == 0);
        const int k = not_ready ? __ffs(not_ready) - 1 : 32;  // lanes 0..k-1 are ready
        const unsigned ready_mask = k == 32 ? 0xffffffffu : ((1u << k) - 1);
        const unsigned inc = __ballot_sync(0xffffffffu, (s >> 62) == 2) & ready_mask;
        const int stop = inc ? __ffs(inc) - 1 : k - 1;
        uint64_t v = lane <= stop ? (s & LB_VAL) : 0;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
        excl += v;
        if (inc) break;
        p -= k;
        if (k == 0) {  // nearest predecessor not ready yet: bounded wait
            const uint64_t now = global_ns();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > WAIT_LIMIT_NS) {
                if (lane == 0) set_status(status, NN_ERR_TIMEOUT);
                break;
            }
            __nanosleep(100);
        } else {
            t0 = 0;
        }
    }
    if (lane == 0) st_release(&state[t], LB_INC | ((excl + agg) & LB_VAL));
    __syncwarp();
    return excl;
}

__device__ inline uint64_t warp_lookback(uint64_t* state, uint64_t t, uint64_t agg, int32_t* status) {
    if ((threadIdx.x & 31) == 0) lb_publish(state, t, agg);
    __syncwarp();
    return lb_resolve(state, t, agg, status);
}

// ------------------------------------------------------------ block scans
// Exclusive scan of one 64-bit value per thread; *total gets the block sum.
// `sh` needs 33 words.  All threads must call.
__device__ inline uint64_t block_excl_scan(uint64_t x, uint64_t* total, uint64_t* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    uint64_t v = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        uint64_t y = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += y;
    }
    if (lane == 31) sh[warp] = v;
    __syncthreads();
    if (warp == 0) {
        uint64_t w = lane < nw ? sh[lane] : 0;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            uint64_t y = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += y;
        }
        if (lane < nw) sh[lane] = w;
        if (lane == 31) sh[32] = w;
    }
    __syncthreads();
    uint64_t r = v - x + (warp > 0 ? sh[warp - 1] : 0);
    *total = sh[32];
    __syncthreads();
    return r;
}

// --------------------------------------------------------------- records
// (the layout is described at RecFmt; 8-byte records use x and y)
struct Rec {
    uint32_t x, y, z, w;
};

// The side of a node at vr (relative to the build's first node).
__device__ __forceinline__ uint32_t make_side(const RecFmt& f, uint32_t vr, uint32_t nf) {
    const int bits = f.sb + (f.cshift > 0 ? f.cshift : 0);
    return (vr & ((1u << bits) - 1u)) | ((f.want & NN_WANT_ELEMS) ? nf << f.off_nf : 0u);
}
// n: the neighbours, f.nmask for none (n[2] is not used when k = 2)
template <int RB>
__device__ __forceinline__ Rec pack_rec(const RecFmt& f, uint32_t side, uint32_t e, const uint32_t (&n)[3], int K) {
    Rec r;
    if constexpr (RB == 8) {
        uint64_t v = side;
        if (f.want & NN_WANT_ELEMS) v |= (uint64_t)e << f.off_e;
        if (f.want & NN_WANT_NODES) {
            v |= (uint64_t)n[0] << f.off_n;
            v |= (uint64_t)n[1] << (f.off_n + f.nb);
            if (f.k == 3) v |= (uint64_t)(K == 3 ? n[2] : f.nmask) << (f.off_n + 2 * f.nb);
        }
        r = Rec{(uint32_t)v, (uint32_t)(v >> 32), 0u, 0u};
    } else {
        const uint32_t n2 = f.k == 3 ? (K == 3 ? n[2] : f.nmask) : 0u;
        r = Rec{e, n[0], n[1], n2};
        if (f.side_split) {
            r.y |= side << f.nb;
            r.z |= (side >> f.sh2) << f.nb;
            r.w |= (side >> f.sh3) << f.nb;
            r.x |= (side >> f.sh0) << f.eb;
        } else if (f.k == 2 || !(f.want & NN_WANT_NODES)) {
            r.w = side;
        } else {
            r.x = side;
        }
    }
    return r;
}
// The side; bits above it may be set in 8-byte records.  K: f.k where the
// caller knows it at compile time (0: look it up).
template <int RB, int K>
__device__ __forceinline__ uint32_t rec_side(const RecFmt& f, const Rec& r) {
    if constexpr (RB == 8) {
        return r.x;
    } else if constexpr (K == 2) {
        return r.w;
    } else {
        if (f.side_split)
            return (r.y >> f.nb) | ((r.z >> f.nb) << f.sh2) | ((r.w >> f.nb) << f.sh3) | ((r.x >> f.eb) << f.sh0);
        return (K == 0 && f.k == 2) || !(f.want & NN_WANT_NODES) ? r.w : r.x;
    }
}
// 32 bits of an 8-byte record from bit off < 64
__device__ __forceinline__ uint32_t rec_bits(const Rec& r, int off) {
    return off < 32 ? __funnelshift_r(r.x, r.y, (uint32_t)off) : r.y >> (off - 32);
}
template <int RB>
__device__ __forceinline__ uint32_t rec_elem(const RecFmt& f, const Rec& r) {
    if constexpr (RB == 8) return rec_bits(r, f.off_e) & f.emask;
    else return r.x & f.emask;
}
// neighbour j (f.nmask: none)
template <int RB>
__device__ __forceinline__ uint32_t rec_nbr(const RecFmt& f, const Rec& r, int j) {
    if constexpr (RB == 8) return rec_bits(r, f.off_n + j * f.nb) & f.nmask;
    else return (j == 0 ? r.y : (j == 1 ? r.z : r.w)) & f.nmask;
}
template <int RB>
__device__ __forceinline__ void put_rec(uint8_t* base, uint64_t pos, const Rec& r) {
    if constexpr (RB == 8) reinterpret_cast<uint2*>(base)[pos] = make_uint2(r.x, r.y);
    else reinterpret_cast<uint4*>(base)[pos] = make_uint4(r.x, r.y, r.z, r.w);
}
// Shared memory, or records in global memory.  Never a read-only load (__ldg):
// a kernel of a chain (chain_begin) is there before the one that writes them
// is done, and only ordinary loads are sure to stay behind its wait.
template <int RB>
__device__ __forceinline__ Rec take_rec(const uint8_t* base, uint64_t pos) {
    if constexpr (RB == 8) {
        const uint2 v = reinterpret_cast<const uint2*>(base)[pos];
        return Rec{v.x, v.y, 0u, 0u};
    } else {
        const uint4 v = reinterpret_cast<const uint4*>(base)[pos];
        return Rec{v.x, v.y, v.z, v.w};
    }
}
// ------------------------------------------------ element local edge tables
// Edge-neighbors of local node i (the other end of each local edge at i).
// tri: the two others; quad: the two cyclic neighbours; tet: the three others;
// hex (VTK): the two cyclic neighbours in i's face plus the node across.
template <int TYPE>
struct ElemT;
template <>
struct ElemT<NN_TRI> {
    static constexpr int NPE = 3, K = 2;
    __device__ static int nbr(int i, int s) { return (i + 1 + s) % 3; }
};
template <>
struct ElemT<NN_QUAD> {
    static constexpr int NPE = 4, K = 2;
    __device__ static int nbr(int i, int s) { return (i + (s ? 3 : 1)) & 3; }
};
template <>
struct ElemT<NN_TET> {
    static constexpr int NPE = 4, K = 3;
    __device__ static int nbr(int i, int s) { return (i + 1 + s) & 3; }
};
template <>
struct ElemT<NN_HEX> {
    static constexpr int NPE = 8, K = 3;
    __device__ static int nbr(int i, int s) {
        return s == 2 ? (i ^ 4) : ((i & 4) | ((i + (s ? 3 : 1)) & 3));
    }
};

__device__ __forceinline__ int npe_of(int t) { return t == NN_TRI ? 3 : (t == NN_HEX ? 8 : 4); }
__device__ __forceinline__ int nbr_of(int t, int i, int s) {
    switch (t) {
        case NN_TRI: return ElemT<NN_TRI>::nbr(i, s);
        case NN_QUAD: return ElemT<NN_QUAD>::nbr(i, s);
        case NN_TET: return ElemT<NN_TET>::nbr(i, s);
        default: return ElemT<NN_HEX>::nbr(i, s);
    }
}
__device__ __forceinline__ int k_of(int t) { return (t == NN_TRI || t == NN_QUAD) ? 2 : 3; }
// The node at the far end of local edge s at local node i of an element of
// run-time type t, read from the element's nodes nd[0..8).  Called with i and
// s fixed by unrolled loops, every index below is a compile-time constant, so
// nd stays in registers (an index computed at run time, as nbr_of gives,
// would put the array in local memory).  Every index is below 8.
__device__ __forceinline__ int32_t nbr_node(int t, const int32_t* nd, int i, int s) {
    switch (t) {
        case NN_TRI: return nd[ElemT<NN_TRI>::nbr(i, s)];
        case NN_QUAD: return nd[ElemT<NN_QUAD>::nbr(i, s)];
        case NN_TET: return nd[ElemT<NN_TET>::nbr(i, s)];
        default: return nd[ElemT<NN_HEX>::nbr(i, s)];
    }
}

}  // namespace nn
