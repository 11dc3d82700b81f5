// Element face adjacency from the node -> element CSR.
//
// Sec. 1 lists the neighbours of each element among the local connectivity a
// mesh code needs; the paper works out only the per-node ones.  Reading: two
// distinct elements are face neighbours when every node of some face of one
// of them belongs to the other (faces: tri and quad edges, tet triangles, hex
// quads in VTK order; a face with a repeated node is no face).  For a
// conforming mesh this is the dual graph; a hex face split into two tet
// triangles borders both tets.
//
// A mesh of one type is matched node by node (k_adj_match): the elements
// around a node are held by the lanes of a group.  Each face is settled once,
// at its smallest node: tets put the faces whose smallest node this is into a
// small hash table per warp, the other types compare the faces of a lane's
// element that contain the node with every other element there (as tets do in
// rows longer than a warp).  What lies across a face goes into one slot per
// element and face; the rows are the sorted slots.
// Elements for which one slot per face is not enough (several elements across
// a face, a face that lies in an element without being one of its faces,
// repeated nodes, a node with very many elements) are flagged.  A flagged
// element, and every element of a mixed mesh, merges the (sorted) element
// rows of its distinct nodes, which yields every element sharing a node with
// it once, in ascending order, with the number of shared nodes; the face
// tests run only where that number allows a shared face.  Their counts come
// first, then one pass scans all counts (decoupled lookback over tiles of
// elements) and writes the matched rows, then the merged rows are written.
#include "nn_device.cuh"

namespace nn {

namespace {

constexpr int ADJ_THREADS = 256;
constexpr int ADJ_TILE = 1024;  // elements of a tile of the row pass

__constant__ int8_t c_nfaces[4] = {3, 4, 4, 6};
__constant__ int8_t c_fsize[4] = {2, 2, 3, 4};
__constant__ int8_t c_faces[4][6][4] = {
    {{0, 1}, {1, 2}, {2, 0}},
    {{0, 1}, {1, 2}, {2, 3}, {3, 0}},
    {{1, 2, 3}, {0, 2, 3}, {0, 1, 3}, {0, 1, 2}},
    {{0, 1, 2, 3}, {4, 5, 6, 7}, {0, 1, 5, 4}, {1, 2, 6, 5}, {2, 3, 7, 6}, {3, 0, 4, 7}},
};

// Type and nodes of element e (-1: invalid element, skipped).
__device__ __forceinline__ int load_element(const AdjParams& p, int64_t e, int32_t* nd) {
    int t = p.type;
    int64_t a;
    if (t == NN_MIXED) {
        t = p.elem_type[e];
        if (t > NN_HEX) return -1;
        a = p.elem_ptr[e];
        if (a < 0 || p.elem_ptr[e + 1] - a != npe_of(t) || p.elem_ptr[e + 1] > p.n_conn) return -1;
    } else {
        a = e * npe_of(t);
    }
    const int n = npe_of(t);
    for (int i = 0; i < n; ++i) {
        nd[i] = p.conn[a + i];
        if (nd[i] < 0 || (int64_t)nd[i] >= p.n_nodes) return -1;
    }
    return t;
}

__device__ __forceinline__ bool contains(const int32_t* nd, int n, int32_t v) {
    for (int i = 0; i < n; ++i)
        if (nd[i] == v) return true;
    return false;
}

// Some face of element a (type ta, nodes na) has all its nodes in b (nb nodes).
__device__ __forceinline__ bool face_in(int ta, const int32_t* na, const int32_t* nbd, int nb) {
    const int nf = c_nfaces[ta], fs = c_fsize[ta];
    for (int k = 0; k < nf; ++k) {
        bool ok = true;
        for (int q = 0; q < fs && ok; ++q) {
            const int32_t v = na[c_faces[ta][k][q]];
            for (int r = 0; r < q; ++r)
                if (na[c_faces[ta][k][r]] == v) ok = false;  // repeated node: no face
            if (ok && !contains(nbd, nb, v)) ok = false;
        }
        if (ok) return true;
    }
    return false;
}

// Calls emit(f) for every face neighbour f of element e, once each, in
// ascending order.  The element rows of e's distinct nodes are sorted, so a
// k-way merge of them visits every element sharing a node with e once and
// counts the nodes they share; only an element sharing at least as many nodes
// as the smallest face that could join them has its nodes gathered and the
// face tests run (a tet sees ~96 row entries but ~4 such candidates).
template <class F>
__device__ __forceinline__ void for_each_neighbour(const AdjParams& p, int64_t e, F&& emit) {
    constexpr int32_t END = 0x7fffffff;
    int32_t nd[8];
    const int t = load_element(p, e, nd);
    if (t < 0) return;
    const int n = npe_of(t);
    // one row per node slot (a repeated node, or a slot past the element, gets an empty one)
    int64_t pos[8], end[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        bool use = i < n;
#pragma unroll
        for (int j = 0; j < i; ++j) use = use && !(j < n && nd[j] == nd[i]);
        pos[i] = use ? p.ne_rp[nd[i]] : 0;
        end[i] = use ? p.ne_rp[nd[i] + 1] : 0;
    }
    int32_t head[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) head[i] = pos[i] < end[i] ? p.ne_col[pos[i]] : END;
    // any face of e, and any face of a neighbour of another type (2-node faces in a mixed mesh)
    const int dmin = p.type == NN_MIXED ? 2 : c_fsize[t];
    for (;;) {
        int32_t m = END;
#pragma unroll
        for (int j = 0; j < 8; ++j) m = min(m, head[j]);
        if (m == END) break;
        int shared = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (head[j] == m) {
                ++shared;
                ++pos[j];
                head[j] = pos[j] < end[j] ? p.ne_col[pos[j]] : END;
            }
        }
        if ((int64_t)m == e || shared < dmin || m < 0 || (int64_t)m >= p.n_elems) continue;
        int32_t fd[8];
        const int tf = load_element(p, m, fd);
        if (tf < 0) continue;
        if (face_in(t, nd, fd, npe_of(tf)) || face_in(tf, fd, nd, n)) emit(m);
    }
}

// ------------------------------------------------- matching node by node
// What bounds the merge above is divergence: measured on a 61^3 Kuhn grid, 5
// of 32 lanes were active on average, and every element's node rows were
// walked twice.  Matching per node gathers each element's nodes once per node
// (n_conn gathers in all) and has no data-dependent branch but the rare match.
// Whole call, GB300: 101^3 Kuhn grid 26.7 -> 1.8 ms, and 0.98 ms with the
// face table and the one-pass rows below; 129^3 hex grid 3.0 -> 0.94 ms and
// 2048^2 triangle grid 7.3 -> 1.4 ms before the latter.  The groups have 8 lanes where a node has 4 to 8 elements, a warp for tets (24).
//
// Tets: comparing each of a node's 24 elements with the 23 others was bound by
// instructions (78 % of issue slots).  A face needs a look only at its
// smallest node, by a third of its elements' faces there, and two tets share a
// face exactly when its three nodes are equal: the faces go into a small hash
// table per warp.  Hexes and quads also ask whether a face's nodes lie in an
// element whose face it is not, and compare pairs in groups of 8.
constexpr int FACE_HASH_BITS = 7;
// Longest node row matched here; elements around a longer one are flagged
// without a look at them.  Rows longer than a group's are matched by the whole
// warp (an element per lane, the others by shuffles); they used to be by the
// group, against nodes read from memory.  Whole call, before and now: random
// hexes with 8 elements a node 1040 -> 557 us, random quads 510 -> 325, Delaunay
// triangles 283 -> 232, a sphere with poles of 1000 781 -> 744.
constexpr int ADJ_LONG = 64;

template <int TYPE>
struct AdjShape;
// Q: the element's nodes other than the centre; F: its faces at the centre;
// NF: its faces (slots); G: lanes of a group, at least the ordinary number of
// elements around a node (a longer row takes several rounds).
template <>
struct AdjShape<NN_TRI> {
    static constexpr int Q = 2, F = 2, NF = 3, G = 8;
};
template <>
struct AdjShape<NN_QUAD> {
    static constexpr int Q = 3, F = 2, NF = 4, G = 8;
};
template <>
struct AdjShape<NN_TET> {
    static constexpr int Q = 3, F = 3, NF = 4, G = 32;
};
template <>
struct AdjShape<NN_HEX> {
    static constexpr int Q = 7, F = 3, NF = 6, G = 8;
};

__device__ __forceinline__ void cond_swap(bool c, int32_t& a, int32_t& b) {
    const int32_t x = c ? b : a, y = c ? a : b;
    a = x;
    b = y;
}

// Element e seen from its node v: the other nodes in a frame with v at the
// origin, and the slot of each face at v.
template <int TYPE>
struct AdjFrame {
    using S = AdjShape<TYPE>;
    int32_t q[S::Q];
    int local;  // v's place in the element (hex: in binary corner order)

    // 0: not usable (invalid element, or v is none of its nodes), 1: fine, 2: a node repeats
    __device__ __forceinline__ int load(const AdjParams& p, int64_t e, int32_t v) {
        constexpr int NPE = S::Q + 1;
        int32_t nd[NPE];
        if (e < 0 || e >= p.n_elems) return 0;
        if constexpr (TYPE == NN_TRI) {
#pragma unroll
            for (int i = 0; i < 3; ++i) nd[i] = __ldg(p.conn + 3 * e + i);
        } else {
            const int4 a = __ldg(reinterpret_cast<const int4*>(p.conn) + (NPE / 4) * e);
            nd[0] = a.x; nd[1] = a.y; nd[2] = a.z; nd[3] = a.w;
            if constexpr (NPE == 8) {
                const int4 b = __ldg(reinterpret_cast<const int4*>(p.conn) + 2 * e + 1);
                nd[4] = b.x; nd[5] = b.y; nd[6] = b.z; nd[7] = b.w;
            }
        }
        bool in = true, rep = false;
        local = -1;
#pragma unroll
        for (int i = 0; i < NPE; ++i) {
            in = in && (uint32_t)nd[i] < (uint64_t)p.n_nodes;
            if (nd[i] == v) local = i;
#pragma unroll
            for (int j = 0; j < i; ++j) rep = rep || nd[i] == nd[j];
        }
        if (!in || local < 0) return 0;
        if constexpr (TYPE == NN_TRI) {
            q[0] = local == 0 ? nd[1] : (local == 1 ? nd[2] : nd[0]);
            q[1] = local == 0 ? nd[2] : (local == 1 ? nd[0] : nd[1]);
        } else if constexpr (TYPE == NN_QUAD) {
            // turned until v comes first
            if (local & 1) {
                const int32_t t = nd[0];
                nd[0] = nd[1]; nd[1] = nd[2]; nd[2] = nd[3]; nd[3] = t;
            }
            cond_swap(local & 2, nd[0], nd[2]);
            cond_swap(local & 2, nd[1], nd[3]);
            q[0] = nd[1]; q[1] = nd[2]; q[2] = nd[3];
        } else if constexpr (TYPE == NN_TET) {
            q[0] = local == 0 ? nd[1] : nd[0];
            q[1] = local <= 1 ? nd[2] : nd[1];
            q[2] = local <= 2 ? nd[3] : nd[2];
        } else {
            // binary corner order (VTK order with 2, 3 and 6, 7 swapped), then
            // reflected along each axis on which v lies at the far side
            cond_swap(true, nd[2], nd[3]);
            cond_swap(true, nd[6], nd[7]);
            if ((local & 3) >= 2) local ^= 1;
#pragma unroll
            for (int a = 1; a < 8; a <<= 1)
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (!(i & a)) cond_swap(local & a, nd[i], nd[i | a]);
#pragma unroll
            for (int i = 1; i < 8; ++i) q[i - 1] = nd[i];
        }
        return rep ? 2 : 1;
    }
    // whether every other node of face f at v is above v (v is the face's smallest node)
    __device__ __forceinline__ bool smallest(int f, int32_t v) const {
        if constexpr (TYPE == NN_TRI) return q[f] > v;
        else if constexpr (TYPE == NN_QUAD) return q[2 * f] > v;
        else if constexpr (TYPE == NN_TET) return q[f == 0 ? 1 : 0] > v && q[f == 2 ? 1 : 2] > v;
        else return f == 0 ? (q[0] > v && q[1] > v && q[2] > v)
                           : (f == 1 ? (q[0] > v && q[3] > v && q[4] > v) : (q[1] > v && q[3] > v && q[5] > v));
    }
    // slot of face f at v, unique over the element's faces
    __device__ __forceinline__ int slot(int f) const {
        if constexpr (TYPE == NN_TRI) return f == 0 ? local : (local == 0 ? 2 : local - 1);
        else if constexpr (TYPE == NN_QUAD) return f == 0 ? local : (local + 3) & 3;
        else if constexpr (TYPE == NN_TET) return f + (f >= local ? 1 : 0);  // the node left out
        else return f == 0 ? 4 + ((local >> 2) & 1) : (f == 1 ? 2 + ((local >> 1) & 1) : (local & 1));
    }
    // faces at v (bit f) whose nodes all lie in the element with frame y (also seen from v)
    __device__ __forceinline__ uint32_t inside(const int32_t* y) const {
        bool in[S::Q];
#pragma unroll
        for (int k = 0; k < S::Q; ++k) {
            in[k] = false;
            if ((TYPE == NN_QUAD && k == 1) || (TYPE == NN_HEX && k == 6)) continue;  // on no face at v
#pragma unroll
            for (int i = 0; i < S::Q; ++i) in[k] = in[k] || q[k] == y[i];
        }
        if constexpr (TYPE == NN_TRI) return (in[0] ? 1u : 0u) | (in[1] ? 2u : 0u);
        else if constexpr (TYPE == NN_QUAD) return (in[0] ? 1u : 0u) | (in[2] ? 2u : 0u);
        else if constexpr (TYPE == NN_TET)
            return (in[1] && in[2] ? 1u : 0u) | (in[0] && in[2] ? 2u : 0u) | (in[0] && in[1] ? 4u : 0u);
        else
            return (in[0] && in[1] && in[2] ? 1u : 0u) | (in[0] && in[3] && in[4] ? 2u : 0u) |
                   (in[1] && in[3] && in[5] ? 4u : 0u);
    }
    // hex: whether two of the three nodes next to v, which every face at v has,
    // are in y (else: true)
    __device__ __forceinline__ bool may_share(const int32_t* y) const {
        if constexpr (TYPE == NN_HEX) {
            int n = 0;
#pragma unroll
            for (int i = 0; i < S::Q; ++i) n += (q[0] == y[i]) + (q[1] == y[i]) + (q[3] == y[i]);
            return n >= 2;
        } else {
            return true;
        }
    }
    // whether face f at v is, as far as a look at the frames shows, a face of
    // y too (simplices: always; a false "no" only costs the slow path)
    __device__ __forceinline__ bool also_face_of(int f, const int32_t* y) const {
        if constexpr (TYPE == NN_QUAD) {
            return q[2 * f] == y[0] || q[2 * f] == y[2];
        } else if constexpr (TYPE == NN_HEX) {
            const int32_t a = f == 2 ? q[1] : q[0], b = f == 0 ? q[1] : q[3], d = f == 0 ? q[2] : (f == 1 ? q[4] : q[5]);
            auto is = [&](int32_t ya, int32_t yb, int32_t yd) {
                return d == yd && ((a == ya && b == yb) || (a == yb && b == ya));
            };
            return is(y[0], y[1], y[2]) || is(y[0], y[3], y[4]) || is(y[1], y[3], y[5]);
        } else {
            return true;
        }
    }
};

// One node per group of G lanes, one element of its row per lane; rows of more
// than G elements by the whole warp.  (Triangles: 5 CTAs per SM; left alone, the
// compiler spills for a sixth, 1500^2 nodes 560 -> 575 us.)
template <int TYPE>
__global__ void __launch_bounds__(ADJ_THREADS, TYPE == NN_TRI ? 5 : 0) k_adj_match(AdjParams p) {
    using S = AdjShape<TYPE>;
    constexpr int G = S::G, PER = 32 / G;
    __shared__ __align__(16) uint32_t sh_head[TYPE == NN_TET ? ADJ_THREADS / 32 : 1][1 << FACE_HASH_BITS];
    __shared__ uint4 sh_face[TYPE == NN_TET ? ADJ_THREADS / 32 : 1][32 * S::F];
    const int lane = threadIdx.x & 31, gl = lane & (G - 1);
    const int64_t warp = ((int64_t)blockIdx.x * ADJ_THREADS + threadIdx.x) >> 5;
    const int64_t step = ((int64_t)gridDim.x * ADJ_THREADS >> 5) * PER;
    // one lane's findings: the element across each face at v, and how many there are
    struct Found {
        int32_t y[S::F];
        int n[S::F];
    };
    auto compare = [&](const AdjFrame<TYPE>& x, int32_t v, int32_t ey, const int32_t* y, Found& r) {
        const uint32_t in = x.inside(y);
        if (!in) return;
#pragma unroll
        for (int f = 0; f < S::F; ++f) {
            if (!((in >> f) & 1)) continue;
            r.y[f] = ey;
            ++r.n[f];
            if (!x.also_face_of(f, y)) p.cplx[ey] = 1;
        }
    };
    auto settle = [&](const AdjFrame<TYPE>& x, int32_t v, int32_t e, const Found& r) {
#pragma unroll
        for (int f = 0; f < S::F; ++f) {
            if (!x.smallest(f, v)) continue;
            p.nbr[(int64_t)e * S::NF + x.slot(f)] = r.n[f] ? r.y[f] : -1;
            if (r.n[f] > 1) p.cplx[e] = 1;
        }
    };
    int64_t base = warp * PER;
    auto row = [&](int64_t b0, int64_t& a, int64_t& n) {
        const int64_t v = b0 + lane / G;
        a = n = 0;
        if (v < p.n_nodes) {
            a = __ldg(p.ne_rp + v);
            n = __ldg(p.ne_rp + v + 1) - a;
        }
    };
    auto around = [&](int64_t a, int64_t n) { return n <= G && gl < n ? __ldg(p.ne_col + a + gl) : -1; };
    // the next node's elements and the bounds of the one after it are on their
    // way while a node's elements are compared
    int64_t r0, L, r1, L1;
    row(base, r0, L);
    row(base + step, r1, L1);
    int32_t e0 = around(r0, L);
    for (; base < p.n_nodes; base += step) {
        const int32_t v = (int32_t)(base + lane / G);
        const int64_t cur = r0, n = L;
        const int32_t e = e0;
        r0 = r1;
        L = L1;
        e0 = around(r0, L);
        row(base + 2 * step, r1, L1);
        AdjFrame<TYPE> x{};
        const int ok = x.load(p, e, v);
        const int32_t id = ok ? e : -1;
        if (__any_sync(0xffffffffu, ok == 2)) {
            // a repeated node: the elements around this node take the slow path
            const unsigned m = __ballot_sync(0xffffffffu, ok == 2) >> (lane & ~(G - 1));
            if ((m & (G == 32 ? 0xffffffffu : (1u << (G & 31)) - 1)) && ok) p.cplx[e] = 1;
        }
        Found r{};
        if constexpr (TYPE == NN_TET) {
            // the faces at v whose smallest node v is, by their other two
            // nodes: chained by hash, and each compared with its chain
            if (n > 1 && n <= G) {
                uint32_t* const head = sh_head[threadIdx.x >> 5];
                uint4* const face = sh_face[threadIdx.x >> 5];
                reinterpret_cast<uint4*>(head)[lane] = make_uint4(EMPTY, EMPTY, EMPTY, EMPTY);
                __syncwarp();
                uint32_t a[S::F], b[S::F], h[S::F];
                bool use[S::F];
#pragma unroll
                for (int f = 0; f < S::F; ++f) {
                    const int32_t s = x.q[f == 0 ? 1 : 0], t = x.q[f == 2 ? 1 : 2];
                    use[f] = ok == 1 && s > v && t > v;
                    a[f] = (uint32_t)min(s, t);
                    b[f] = (uint32_t)max(s, t);
                    h[f] = (a[f] * 0x9E3779B1u + b[f] * 0x85EBCA6Bu) >> (32 - FACE_HASH_BITS);
                    if (use[f]) {
                        const uint32_t next = atomicExch(&head[h[f]], (uint32_t)(f * 32 + lane));
                        face[f * 32 + lane] = make_uint4(a[f], b[f], (uint32_t)e, next);
                    }
                }
                __syncwarp();
#pragma unroll
                for (int f = 0; f < S::F; ++f) {
                    for (uint32_t k = use[f] ? head[h[f]] : EMPTY; k != EMPTY;) {
                        const uint4 y = face[k];
                        if (y.x == a[f] && y.y == b[f] && y.z != (uint32_t)e) {
                            r.y[f] = (int32_t)y.z;
                            ++r.n[f];
                        }
                        k = y.w;
                    }
                }
                __syncwarp();
            }
        } else {
            const int jmax = (int)__reduce_max_sync(0xffffffffu, n <= G && n > 1 ? (unsigned)n : 0u);
            for (int j = 0; j < jmax; ++j) {
                const int32_t ey = __shfl_sync(0xffffffffu, id, j, G);
                int32_t y[S::Q];
#pragma unroll
                for (int k = 0; k < S::Q; ++k) y[k] = __shfl_sync(0xffffffffu, x.q[k], j, G);
                if (ok && ey >= 0 && ey != e) compare(x, v, ey, y, r);
            }
        }
        if (ok == 1) settle(x, v, e, r);
        // longer rows, one after another by the whole warp: 32 elements at a
        // time against 32 at a time
        for (unsigned m = __ballot_sync(0xffffffffu, gl == 0 && n > G); m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            const int64_t nl = __shfl_sync(0xffffffffu, n, src), at = __shfl_sync(0xffffffffu, cur, src);
            const int32_t vl = __shfl_sync(0xffffffffu, v, src);
            if (nl > ADJ_LONG) {
                for (int64_t i = lane; i < nl; i += 32) {
                    const int32_t ei = __ldg(p.ne_col + at + i);
                    if (ei >= 0 && ei < p.n_elems) p.cplx[ei] = 1;
                }
                continue;
            }
            for (int64_t i0 = 0; i0 < nl; i0 += 32) {
                const int32_t ei = i0 + lane < nl ? __ldg(p.ne_col + at + i0 + lane) : -1;
                AdjFrame<TYPE> xi{};
                const int oki = xi.load(p, ei, vl);
                Found ri{};
                for (int64_t j0 = 0; j0 < nl; j0 += 32) {
                    AdjFrame<TYPE> y = xi;
                    int32_t ej = ei;
                    int oky = oki;
                    if (j0 != i0) {
                        ej = j0 + lane < nl ? __ldg(p.ne_col + at + j0 + lane) : -1;
                        oky = y.load(p, ej, vl);
                    }
                    // a repeated node: the elements around this node take the slow path
                    if (__any_sync(0xffffffffu, oky == 2) && oki) p.cplx[ei] = 1;
                    const int32_t id_j = oky ? ej : -1;
                    for (int j = 0; j < 32 && j0 + j < nl; ++j) {
                        const int32_t ey = __shfl_sync(0xffffffffu, id_j, j);
                        int32_t yq[S::Q];
#pragma unroll
                        for (int k = 0; k < S::Q; ++k) yq[k] = __shfl_sync(0xffffffffu, y.q[k], j);
                        if (oki && ey >= 0 && ey != ei && xi.may_share(yq)) compare(xi, vl, ey, yq, ri);
                    }
                }
                if (oki == 1) settle(xi, vl, ei, ri);
            }
        }
    }
}

// The slots of element e, ascending (unsigned: empty ones last).
template <int NF>
__device__ __forceinline__ void sorted_slots(const AdjParams& p, int64_t e, uint32_t (&s)[NF]) {
    if constexpr (NF == 4) {
        const uint4 a = __ldg(reinterpret_cast<const uint4*>(p.nbr) + e);
        s[0] = a.x; s[1] = a.y; s[2] = a.z; s[3] = a.w;
    } else {
#pragma unroll
        for (int i = 0; i < NF; ++i) s[i] = (uint32_t)__ldg(p.nbr + e * NF + i);
    }
    // odd-even transposition: NF rounds
#pragma unroll
    for (int r = 0; r < NF; ++r)
#pragma unroll
        for (int i = r & 1; i + 1 < NF; i += 2) {
            const uint32_t x = s[i], y = s[i + 1];
            s[i] = min(x, y);
            s[i + 1] = max(x, y);
        }
}

// Whether element e (of type TYPE) has all its nodes in range.  An element
// that has not is in no node's row, and its slots were never written.
template <int TYPE>
__device__ __forceinline__ bool valid_element(const AdjParams& p, int64_t e) {
    constexpr int NPE = AdjShape<TYPE>::Q + 1;
    const uint32_t N = (uint32_t)p.n_nodes;  // below 2^31
    if constexpr (NPE == 3) {
        bool ok = true;
#pragma unroll
        for (int i = 0; i < 3; ++i) ok = ok && (uint32_t)__ldg(p.conn + 3 * e + i) < N;
        return ok;
    } else {
        bool ok = true;
#pragma unroll
        for (int q = 0; q < NPE / 4; ++q) {
            const uint4 a = __ldg(reinterpret_cast<const uint4*>(p.conn) + (NPE / 4) * e + q);
            ok = ok && a.x < N && a.y < N && a.z < N && a.w < N;
        }
        return ok;
    }
}

__device__ __noinline__ uint32_t merge_count(const AdjParams& p, int64_t e) {
    uint32_t c = 0;
    for_each_neighbour(p, e, [&](int32_t) { ++c; });
    return c;
}
__device__ __noinline__ void merge_write(const AdjParams& p, int64_t e, int32_t* row, int64_t n) {
    int64_t k = 0;
    for_each_neighbour(p, e, [&](int32_t f) {
        if (k < n) row[k] = f;
        ++k;
    });
}

// Elements whose rows are merged from their nodes' rows: the flagged ones,
// or all (a mixed mesh, or no room for the slots).  Their counts, before the
// offsets are known, and their rows, after.  (They are not part of the pass
// between: a merge may take long, and no tile of the scan waits for one.)
template <bool WRITE>
__global__ void __launch_bounds__(ADJ_THREADS) k_adj_merge(AdjParams p) {
    for (int64_t e = (int64_t)blockIdx.x * ADJ_THREADS + threadIdx.x; e < p.n_elems;
         e += (int64_t)gridDim.x * ADJ_THREADS) {
        if (p.nbr && !p.cplx[e]) continue;
        if constexpr (WRITE) {
            const int64_t a = p.rp[e], n = p.rp[e + 1] - a;
            if (n > 0 && a + n <= p.cap) merge_write(p, e, p.col + a, n);
        } else {
            p.cnt[e] = merge_count(p, e);
        }
    }
}

// Row pointers of all elements and the rows of the matched ones, in one pass:
// a tile's rows are put together in shared memory and written as one run at
// the offset that the lookback over the earlier tiles gives.  (Counting,
// scanning and writing in a kernel each read the slots twice and ran 47,000
// tiles of 128 elements for 6 M of them.)  TYPE = NN_MIXED: no slots, the
// counts are scanned alone.
constexpr int ROWS_PER = ADJ_TILE / ADJ_THREADS;  // elements of a thread
template <int TYPE>
__global__ void __launch_bounds__(ADJ_THREADS) k_adj_rows(AdjParams p) {
    constexpr int NF = TYPE == NN_MIXED ? 0 : AdjShape<TYPE == NN_MIXED ? NN_TET : TYPE>::NF;
    __shared__ uint32_t rows[NF > 0 ? ADJ_TILE * NF : 1];
    __shared__ uint64_t sh_scan[33];
    __shared__ uint32_t sh_tile;
    __shared__ uint64_t sh_base;
    if (threadIdx.x == 0) sh_tile = atomicAdd(p.ticket, 1u);
    __syncthreads();
    const uint32_t tile = sh_tile;
    const int64_t e0 = (int64_t)tile * ADJ_TILE + threadIdx.x * ROWS_PER;
    uint32_t s[ROWS_PER][NF > 0 ? NF : 1];
    uint32_t n[ROWS_PER];
    bool slow[ROWS_PER];
    uint64_t sum = 0;
#pragma unroll
    for (int k = 0; k < ROWS_PER; ++k) {
        const int64_t e = e0 + k;
        n[k] = 0;
        slow[k] = true;
        if (e < p.n_elems) {
            if constexpr (NF > 0) {
                slow[k] = p.cplx[e];
                if (!slow[k] && valid_element<TYPE>(p, e)) {
                    sorted_slots<NF>(p, e, s[k]);
#pragma unroll
                    for (int i = 0; i < NF; ++i) n[k] += s[k][i] != EMPTY && (i == 0 || s[k][i] != s[k][i - 1]);
                }
            }
            if (slow[k]) n[k] = p.cnt[e];
        }
        sum += n[k];
    }
    uint64_t agg;
    const uint64_t ex = block_excl_scan(sum, &agg, sh_scan);
    if (threadIdx.x < 32) {
        const uint64_t base = warp_lookback(p.lb_state, tile, agg, p.status);
        if (threadIdx.x == 0) sh_base = base;
    }
    if constexpr (NF > 0) {
        // (a tile of merged elements alone may have longer rows than this holds; theirs are left out here)
        if (agg <= ADJ_TILE * NF) {
            uint32_t* d = rows + ex;
#pragma unroll
            for (int k = 0; k < ROWS_PER; ++k) {
                if (slow[k]) {
                    d += n[k];
                    continue;
                }
#pragma unroll
                for (int i = 0; i < NF; ++i)
                    if (n[k] && s[k][i] != EMPTY && (i == 0 || s[k][i] != s[k][i - 1])) *d++ = s[k][i];
            }
        }
    }
    __syncthreads();
    const uint64_t base = sh_base;
    uint64_t at = base + ex;
#pragma unroll
    for (int k = 0; k < ROWS_PER; ++k) {
        if (e0 + k < p.n_elems) p.rp[e0 + k] = (int64_t)at;
        if constexpr (NF > 0) {
            if (agg > ADJ_TILE * NF && !slow[k] && at + n[k] <= (uint64_t)p.cap) {
                int32_t* d = p.col + at;
#pragma unroll
                for (int i = 0; i < NF; ++i)
                    if (n[k] && s[k][i] != EMPTY && (i == 0 || s[k][i] != s[k][i - 1])) *d++ = (int32_t)s[k][i];
            }
        }
        at += n[k];
        if (e0 + k == p.n_elems - 1) {
            p.rp[p.n_elems] = (int64_t)at;
            if (at > (uint64_t)p.cap) set_status(p.status, NN_ERR_CAPACITY);
        }
    }
    if constexpr (NF > 0) {
        if (agg <= ADJ_TILE * NF && base + agg <= (uint64_t)p.cap)
            for (uint32_t i = threadIdx.x; i < (uint32_t)agg; i += ADJ_THREADS) p.col[base + i] = (int32_t)rows[i];
    }
}

template <int TYPE>
void count_scan_write(const AdjParams& p, int grid, cudaStream_t s) {
    k_adj_merge<false><<<grid, ADJ_THREADS, 0, s>>>(p);
    k_adj_rows<TYPE><<<(unsigned)((p.n_elems + ADJ_TILE - 1) / ADJ_TILE), ADJ_THREADS, 0, s>>>(p);
    k_adj_merge<true><<<grid, ADJ_THREADS, 0, s>>>(p);
}

template <int TYPE>
void match_and_write(const AdjParams& p, int grid, int sms, cudaStream_t s) {
    constexpr int NODES = ADJ_THREADS / AdjShape<TYPE>::G;  // nodes of a CTA at a time
    const int64_t blocks = (p.n_nodes + NODES - 1) / NODES;
    if (blocks > 0)  // (without nodes every element is invalid and has an empty row)
        k_adj_match<TYPE><<<(unsigned)(blocks < (int64_t)sms * 16 ? blocks : (int64_t)sms * 16), ADJ_THREADS, 0, s>>>(p);
    count_scan_write<TYPE>(p, grid, s);
}

}  // namespace

// Slots per element of the matching pass; 0: a mixed mesh, whose elements all
// merge their node rows.
int adjacency_slots(int type) {
    return type == NN_TRI ? 3 : (type == NN_QUAD || type == NN_TET ? 4 : (type == NN_HEX ? 6 : 0));
}

cudaError_t launch_adjacency(const AdjParams& p, int grid, int sms, cudaStream_t s) {
    if (p.n_elems <= 0) return cudaSuccess;
    if (!p.nbr) {
        count_scan_write<NN_MIXED>(p, grid, s);
        return cudaGetLastError();
    }
    switch (p.type) {
        case NN_TRI: match_and_write<NN_TRI>(p, grid, sms, s); break;
        case NN_QUAD: match_and_write<NN_QUAD>(p, grid, sms, s); break;
        case NN_TET: match_and_write<NN_TET>(p, grid, sms, s); break;
        default: match_and_write<NN_HEX>(p, grid, sms, s); break;
    }
    return cudaGetLastError();
}

size_t adjacency_scan_tiles(int64_t n_elems) { return (size_t)((n_elems + ADJ_TILE - 1) / ADJ_TILE); }

}  // namespace nn
