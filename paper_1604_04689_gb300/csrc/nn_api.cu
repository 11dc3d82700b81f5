// Host side of libnn: argument checks, the build plan (bucket width, record
// format, workspace layout) and the launch sequence.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <new>

#include "nn_internal.h"

namespace nn {
cudaError_t set_emit_smem_all(size_t bytes);
cudaError_t set_bucket_smem_all(size_t bytes);
}  // namespace nn

struct nn_handle {
    int device = 0;
    bool offline = false;      // nn_create_offline: sizing and planning only, no compute calls
    int sms = 0;
    size_t smem_optin = 0;     // max dynamic shared memory per block
    size_t bucket_smem = 0;    // largest dynamic shared memory of the bucket kernel
    size_t smem_per_sm = 0;
    int sb_override = -1;      // fixed bucket width (tests / tuning), -1 = automatic
    int part_mode = -1;        // -1 automatic, 0 one scattered store per record, 1 always partitioned (tests)
    int64_t hist_chunk_override = 0;  // > 0: count at most this many buckets per walk (tests)
    int emit_ctas_override = 0;       // > 0: at most this many element-walk CTAs (tests)
    nn_tuning tuning{};        // nn_set_tuning: bucket width, block size, CTAs per SM (0 = automatic)
    // per-stage timing (nn_profile_*)
    bool prof = false;
    bool pending = false;
    cudaEvent_t ev[NN_PROFILE_STAGES + 1] = {};
    double acc[NN_PROFILE_STAGES] = {};
    int64_t calls = 0;
};

bool nn::handle_offline(const nn_handle* h) { return h && h->offline; }

namespace {

using namespace nn;

constexpr size_t ALIGN = 256;
constexpr int SB_MIN = 4, SB_MAX = 11;
constexpr int64_t DIRECT_CONN = 1 << 16;  // incidences up to which a mesh is built without a partition (mixed: half)
constexpr int DIRECT_QUEUE = 16384;       // incidences a direct build's CTA queues at a time (64 KB)

size_t align_up(size_t x) { return (x + ALIGN - 1) / ALIGN * ALIGN; }
int bits_for(uint64_t x) {  // bits needed to hold values 0..x (>= 1)
    int b = 1;
    while (b < 64 && (x >> b)) ++b;
    return b;
}
int npe_host(int t) { return t == NN_TRI ? 3 : (t == NN_HEX ? 8 : 4); }

struct Plan {
    int type = 0, want = 0, k = 0;
    // N: nodes of this build's range (first node `lo`); n_conn: its records
    // (incidences of those nodes); a whole mesh has lo = 0 and both totals
    int64_t N = 0, T = 0, n_conn = 0, lo = 0;
    RecFmt fmt{};
    int64_t B = 0;
    int64_t hist_chunk = 1;
    int G = 1;
    int G_part = 1;
    int G_fine = 1;
    size_t emit_smem = 0;
    size_t off_estart = 0, off_nfc = 0, off_ntmp = 0, off_grp = 0, off_nloc = 0, off_nstart = 0, off_lb_ns = 0;
    size_t off_hist = 0, off_bstart = 0, off_gcur = 0, off_gcur_c = 0, off_rec_tmp = 0, off_rec = 0, off_lb_off = 0,
           off_ctrl = 0, off_spill = 0, zero_begin = 0, zero_end = 0;
    size_t ws_min = 0, ws_rec = 0;
    int bucket_grid = 0;
    int bucket_threads = 256;
    int imax = 32, slots = 8, list_cap = 32;  // bucket pass: variant, places per node, listed records
    int groups = 1;                           // groups of 32 nodes per bucket
    bool direct = false;                      // no partition: every bucket's CTA reads the whole connectivity
    int queue_cap = 0;                        // ... incidences it queues at a time
    size_t bucket_smem = 0;
    RestShape rest{};         // the bucket pass's second launch
};

nn_status check_mesh(const nn_mesh* m) {
    if (!m) return NN_ERR_ARG;
    const int t = m->type;
    if (!(t == NN_TRI || t == NN_QUAD || t == NN_TET || t == NN_HEX || t == NN_MIXED)) return NN_ERR_ARG;
    if (m->n_nodes < 0 || m->n_elems < 0 || m->n_conn < 0) return NN_ERR_ARG;
    if (m->n_nodes >= (1ll << 31) || m->n_elems >= (1ll << 31) || m->n_conn >= (1ll << 31)) return NN_ERR_ARG;
    if (t != NN_MIXED && m->n_conn != m->n_elems * npe_host(t)) return NN_ERR_ARG;
    if (m->n_conn > 0 && !m->conn) return NN_ERR_ARG;
    if (t != NN_MIXED && (reinterpret_cast<uintptr_t>(m->conn) & 15)) return NN_ERR_ARG;
    if (t == NN_MIXED && m->n_elems > 0 && (!m->elem_ptr || !m->elem_type)) return NN_ERR_ARG;
    if (t == NN_MIXED && (reinterpret_cast<uintptr_t>(m->elem_ptr) & 7)) return NN_ERR_ARG;
    return NN_OK;
}

// Record format (see RecFmt) for ids of T elements and N nodes; false when the
// fields exceed 128 bits.  rb: 16 forces 16-byte records.
bool record_format(int sb, int want, int k, int64_t T, int64_t N, int cshift, int rb, RecFmt* out) {
    const bool we = want & NN_WANT_ELEMS, wn = want & NN_WANT_NODES;
    RecFmt f{};
    f.sb = sb;
    f.want = want;
    f.k = k;
    f.cshift = cshift;
    f.eb = bits_for(T > 0 ? (uint64_t)(T - 1) : 0);
    f.nb = bits_for((uint64_t)N);  // (an id below N is never all ones)
    f.emask = (uint32_t)((1ull << f.eb) - 1);
    f.nmask = (uint32_t)((1ull << f.nb) - 1);
    f.off_nf = sb + (cshift > 0 ? cshift : 0);
    const int side = f.off_nf + (we ? 1 : 0);
    f.off_e = side;
    f.off_n = side + (we ? f.eb : 0);
    const int total = f.off_n + (wn ? k * f.nb : 0);
    if (total > 128) return false;
    f.rb = rb == 16 || total > 64 ? 16 : 8;
    f.side_split = we && wn && k == 3;
    f.sh2 = std::min(31, 32 - f.nb);
    f.sh3 = std::min(31, 2 * (32 - f.nb));
    f.sh0 = std::min(31, 3 * (32 - f.nb));
    *out = f;
    return true;
}

// Second launch of the bucket pass (nn_bucket.cuh): as many of 32 slots as two
// CTAs per SM leave room for, SLOTS_MIN at least, and a list of 512 records.
RestShape rest_shape(const nn_handle* h, int sb, int want, int k, int rb, int64_t buckets) {
    RestShape r{SLOTS_MIN, 512, sb >= 8 ? 256 : 128, 1, 0};
    const int per_sm = sb >= 8 ? 2 : 4;  // by registers
    auto need = [&](int slots) { return bucket_smem_bytes(sb, want, k, slots, rb, r.list_cap); };
    const size_t room = std::min(h->bucket_smem, h->smem_per_sm / 2 - 2048);
    while (r.list_cap > 32 && need(SLOTS_MIN) > h->bucket_smem) r.list_cap -= 16;
    while (r.slots < 32 && need(r.slots + 1) <= room) ++r.slots;
    r.smem = need(r.slots);
    const size_t fit = h->smem_per_sm / (r.smem + 2048);
    r.grid = (int)std::min<int64_t>(buckets, (int64_t)h->sms * std::max<size_t>(1, std::min<size_t>(fit, per_sm)));
    return r;
}

// Plan of a build over the nodes [lo, lo + span) of mesh m, which have
// `records` incidences: the element walk covers the whole mesh, the record
// arrays and node tables only this range.  Record fields stay sized by the
// whole mesh (node and element ids are global).  partitioned: no direct build.
nn_status make_plan_range(const nn_handle* h, const nn_mesh* m, int want, int64_t lo, int64_t span, int64_t records,
                          Plan* P, bool partitioned = false) {
    nn_status st = check_mesh(m);
    if (st != NN_OK) return st;
    if (want < 1 || want > 3) return NN_ERR_ARG;
    if (lo < 0 || span < 0 || lo + span > m->n_nodes || records < 0 || records > m->n_conn) return NN_ERR_ARG;
    Plan p;
    p.type = m->type;
    p.want = want;
    p.N = span;
    p.lo = lo;
    p.T = m->n_elems;
    p.n_conn = records;
    p.k = (m->type == NN_TRI || m->type == NN_QUAD) ? 2 : 3;

    // bucket kernel shape (nn_bucket.cuh).  Slots per node: 8 for meshes of up
    // to 8 incidences per node (triangles, quads, hexes), 16 up to 10, else
    // about the mean and at least 24 (a node with more uses the bucket's list,
    // which costs its warp a second sort: mixed hex and tet meshes, 13 on
    // average, often have 20); the slots also pick the variant by its register
    // arrays.  A bucket has as many nodes as the CTA has lanes: 256, or 128
    // where a node's columns are so long that two CTAs of 256 do not fit.
    const double inc = p.N > 0 ? (double)p.n_conn / (double)p.N : 0.0;
    p.imax = inc <= 8.0 ? 8 : (inc <= 10.0 ? 16 : 32);
    const int want_slots = p.imax < 32 ? p.imax : std::min(32, std::max(24, 4 * (int)std::ceil(inc / 4.0)));
    auto nbk = [&](int s) { return (p.N + (1ll << s) - 1) >> s; };
    auto list_of = [&](int s) { return (int)std::max(32.0, std::min(512.0, std::ceil((double)(1 << s) * inc / 12.0 / 16.0) * 16.0)); };
    auto need = [&](int s, int slots) { return bucket_smem_bytes(s, want, p.k, slots, 16, list_of(s)); };
    p.bucket_threads = h->tuning.bucket_threads ? h->tuning.bucket_threads
                       : (need(8, want_slots) <= h->smem_per_sm / 2 - 2048 ? 256 : 128);
    // A small mesh is built without a partition (nn_bucket.cuh, direct
    // builds), one bucket per SM at most: histogram, offsets and partition are
    // three launches with little to do, while reading the connectivity in
    // every bucket's CTA grows with it.  Graph replays, direct and
    // partitioned: triangles 3 K incidences 14 and 25 us, 24 K 18 and 27,
    // quads 16 K 16 and 21, tets 12 K 26 and 33, 41 K 31 and 33, hexes 11 K 16
    // and 25, 64 K 27 and 28, mixed 7 K 29 and 35, 22 K 33 and 37; with more
    // buckets than SMs a second wave made it slower (triangles 59 K 41 and 33).
    const bool tuned = h->sb_override >= 0 || h->part_mode >= 0 || h->hist_chunk_override > 0 ||
                       h->emit_ctas_override > 0 || h->tuning.bucket_ctas_per_sm;
    // (more elements than incidences: an invalid elem_ptr, left to the general path)
    const bool direct = !tuned && !partitioned && lo == 0 && span == m->n_nodes && p.n_conn > 0 && p.T <= p.n_conn &&
                        p.n_conn <= (p.type == NN_MIXED ? DIRECT_CONN / 2 : DIRECT_CONN);
    const int64_t B_max = (int64_t)1 << 20;  // (bounds the workspace tables)
    int sb = p.bucket_threads == 128 ? 7 : 8;
    if (h->tuning.bucket_ctas_per_sm) {  // the widest bucket that leaves room for that many CTAs
        const size_t budget = std::min(h->bucket_smem, h->smem_per_sm / (size_t)h->tuning.bucket_ctas_per_sm - 2048);
        sb = SB_MAX;
        while (sb > SB_MIN && need(sb, want_slots) > budget) --sb;
    } else {
        // a small mesh: buckets for every SM, as long as one partition pass (256 buckets) does
        while (sb > 5 && nbk(sb) < 2 * (int64_t)h->sms && nbk(sb - 1) <= (direct ? h->sms : 256)) --sb;
    }
    if (h->tuning.sb >= SB_MIN && h->tuning.sb <= SB_MAX) sb = h->tuning.sb;
    if (h->sb_override >= SB_MIN && h->sb_override <= SB_MAX) sb = h->sb_override;
    // wider buckets than shared memory holds (a tuning, a test): fewer slots,
    // then fewer nodes
    while (sb > SB_MIN && need(sb, SLOTS_MIN) > h->bucket_smem) --sb;
    while (nbk(sb) > B_max && sb < SB_MAX) ++sb;
    if (nbk(sb) > B_max || need(sb, SLOTS_MIN) > h->bucket_smem) return NN_ERR_ARG;
    p.slots = SLOTS_MIN;
    while (p.slots < want_slots && need(sb, p.slots + 1) <= h->bucket_smem) ++p.slots;
    p.list_cap = list_of(sb);
    // the list takes what the resident CTAs leave over, up to 512 records:
    // 3-d Delaunay meshes (27 records per node, some of 40) list 320 of a
    // bucket of 128 nodes
    const int by_regs = p.imax == 8 ? 1024 : (p.imax == 16 ? 768 : 512);
    const size_t base_smem = bucket_smem_bytes(sb, want, p.k, p.slots, 16, p.list_cap);
    const size_t resident = std::max<size_t>(1, std::min<size_t>((size_t)(by_regs / p.bucket_threads), h->smem_per_sm / (base_smem + 1536)));
    const size_t per_cta = std::min(h->bucket_smem, h->smem_per_sm / resident - 1536);
    while (p.list_cap < 512 && bucket_smem_bytes(sb, want, p.k, p.slots, 16, p.list_cap + 16) <= per_cta) p.list_cap += 16;
    p.groups = sb < 5 ? 1 : 1 << (sb - 5);
    p.B = nbk(sb);

    // partition: tile-sorted (one pass for <= 256 buckets, else coarse + fine
    // with the fine digit kept in the record) unless that field does not fit
    int cs = 0;
    while (((p.B + (1ll << cs) - 1) >> cs) > 256) ++cs;
    RecFmt& f = p.fmt;
    const bool sorted = h->part_mode != 0 && cs <= 12;  // <= 4096 buckets per coarse region
    if (!(sorted && record_format(sb, want, p.k, p.T, m->n_nodes, cs, 0, &f)) &&
        !record_format(sb, want, p.k, p.T, m->n_nodes, -1, 0, &f))
        return NN_ERR_ARG;

    // element-walk CTAs: one or two per SM, each a fixed slice of elements
    const int unit = p.type == NN_TRI ? 4 : 1;
    const int64_t n_units = (p.T + unit - 1) / unit;
    p.hist_chunk = std::min<int64_t>(p.B, (int64_t)((h->smem_optin - 1024) / 4));
    if (h->hist_chunk_override > 0) p.hist_chunk = std::min<int64_t>(p.hist_chunk, h->hist_chunk_override);
    p.emit_smem = std::max<size_t>(16, (size_t)p.hist_chunk * 4);
    const int cps = p.emit_smem + 2048 <= 113 * 1024 ? 2 : 1;
    p.G = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)h->sms * cps, (n_units + 2047) / 2048));
    if (h->emit_ctas_override > 0) p.G = std::min(p.G, h->emit_ctas_override);
    p.G_part = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)h->sms * 2, (n_units + 511) / 512));
    if (f.cshift >= 0)  // tile-sorted passes: 256-thread CTAs, as many as are resident
        p.G_part = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)h->sms * coarse_ctas_per_sm(p.type), (n_units + 511) / 512));
    p.G_fine = h->sms;  // the fine pass sizes its grid by its occupancy

    p.bucket_smem = bucket_smem_bytes(sb, want, p.k, p.slots, f.rb, p.list_cap);
    int per_sm = 1;
    if (h->offline || bucket_occupancy(&per_sm, p.bucket_threads, p.imax, p.bucket_smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    p.bucket_grid = (int)std::min<int64_t>(p.B, (int64_t)h->sms * per_sm);

    // (few enough groups that their rows are placed by sums: wide buckets, a
    // tuning, of very many nodes have more, and the scan over them is given no
    // cleared words by a direct build)
    p.rest = rest_shape(h, sb, want, p.k, f.rb, p.B);
    if (direct && f.cshift == 0 && p.B <= h->sms && p.B * p.groups <= NODE_SUM_GROUPS &&
        p.bucket_smem + DIRECT_QUEUE * 4 <= h->bucket_smem) {
        p.direct = true;
        p.queue_cap = DIRECT_QUEUE;
    }

    // workspace layout
    size_t o = 0;
    p.off_bstart = o; o = align_up(o + ((size_t)p.B + 1) * 4);
    p.off_estart = o; o = align_up(o + ((want & NN_WANT_ELEMS) ? ((size_t)p.B + 1) * 4 : 0));
    p.off_gcur = o; o = align_up(o + (size_t)p.B * 4);
    p.off_gcur_c = o; o = align_up(o + 256 * 4);
    // the histogram rows are dead once the offsets are known: they share the records' place
    p.off_hist = o;
    const size_t hist_end = align_up(o + (size_t)p.G * p.B * 4);
    p.off_rec_tmp = o; o = align_up(o + (f.cshift > 0 ? (size_t)p.n_conn * f.rb : 0));
    p.off_rec = o; o = std::max(hist_end, align_up(o + (size_t)p.n_conn * f.rb));
    // node rows in scratch (at most k per record), per-node offsets within
    // their bucket, bucket totals and their scan
    const bool wn = want & NN_WANT_NODES;
    const size_t ntmp_bytes = wn ? (size_t)p.k * p.n_conn * 4 + 16 : 0;
    if (f.cshift > 0 && (size_t)p.n_conn * f.rb >= ntmp_bytes) {
        p.off_ntmp = p.off_rec_tmp;  // the coarse-sorted records are dead once the fine pass has run
    } else {
        p.off_ntmp = o; o = align_up(o + ntmp_bytes);
    }
    const size_t ngrp = (size_t)p.B * p.groups;
    p.off_grp = o; o = align_up(o + (wn ? ngrp * 8 : 0));
    p.off_nloc = o; o = align_up(o + (wn ? ((size_t)p.B << sb) * 4 : 0));
    p.off_nstart = o; o = align_up(o + (wn ? (ngrp + 1) * 8 : 0));
    p.zero_begin = o;
    p.off_nfc = o; o = align_up(o + ((want & NN_WANT_ELEMS) ? (size_t)p.B * 4 : 0));
    p.off_lb_off = o; o = align_up(o + (size_t)((p.B + OFFSETS_THREADS - 1) / OFFSETS_THREADS) * 8 + 8);
    p.off_lb_ns = o; o = align_up(o + (wn ? (ngrp + NODE_SCAN_TILE - 1) / NODE_SCAN_TILE * 8 + 8 : 0));
    p.off_ctrl = o; o = align_up(o + 64);
    p.zero_end = o;
    p.off_spill = o;
    p.ws_min = o;
    // spill area: the record indices of hard nodes (nn_bucket.cuh) are grouped
    // there, and long element rows sorted (16 MB and 8 bytes per record covers the odd node
    // of very high valence); a plan whose typical bucket has too few slots (a
    // tuning that widens the buckets) gets room for all of them
    size_t spill = ((size_t)16 << 20) + (size_t)p.n_conn * 8;
    if (p.slots < want_slots) spill += (size_t)p.n_conn * (8 + 4 * (size_t)p.k) + (size_t)p.B * 64;
    p.ws_rec = o + spill;

    *P = p;
    return NN_OK;
}

nn_status make_plan(const nn_handle* h, const nn_mesh* m, int want, Plan* P) {
    nn_status st = check_mesh(m);
    if (st != NN_OK) return st;
    return make_plan_range(h, m, want, 0, m->n_nodes, m->n_conn, P);
}

void prof_flush(nn_handle* h) {
    if (!h->pending) return;
    h->pending = false;
    if (cudaEventSynchronize(h->ev[NN_PROFILE_STAGES]) != cudaSuccess) return;
    for (int i = 0; i < NN_PROFILE_STAGES; ++i) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, h->ev[i], h->ev[i + 1]) == cudaSuccess) h->acc[i] += ms;
    }
    h->calls += 1;
}

void prof_mark(nn_handle* h, int i, cudaStream_t s) {
    if (h->prof) cudaEventRecord(h->ev[i], s);
}

nn_status enqueue(nn_handle* h, const nn_mesh* m, const Plan& p, nn_csr* nodes, nn_csr* elems, uint8_t* w,
                  size_t ws_bytes, const int64_t* base, int32_t* d_status, bool prof, cudaStream_t s);

// Argument checks shared by the single and chunked builds.
nn_status check_outputs(int want, const nn_csr* nodes, const nn_csr* elems) {
    if ((want & NN_WANT_NODES) && (!nodes || !nodes->row_ptr || nodes->col_capacity < 0 ||
                                   (nodes->col_capacity > 0 && !nodes->col)))
        return NN_ERR_ARG;
    if ((want & NN_WANT_ELEMS) && (!elems || !elems->row_ptr || elems->col_capacity < 0 ||
                                   (elems->col_capacity > 0 && !elems->col)))
        return NN_ERR_ARG;
    return NN_OK;
}

nn_status run(nn_handle* h, const nn_mesh* m, int want, nn_csr* nodes, nn_csr* elems, void* ws,
              size_t ws_bytes, int32_t* d_status, cudaStream_t s) {
    if (!h || h->offline || !d_status) return NN_ERR_ARG;
    Plan p;
    nn_status st = make_plan(h, m, want, &p);
    if (st != NN_OK) return st;
    st = check_outputs(want, nodes, elems);
    if (st != NN_OK) return st;
    if (ws_bytes < p.ws_min || (!ws && p.ws_min > 0)) return NN_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(ws) & (ALIGN - 1)) return NN_ERR_ARG;

    uint8_t* w = static_cast<uint8_t*>(ws);
    if (h->prof) prof_flush(h);
    prof_mark(h, 0, s);
    if (p.N == 0) {
        if (cudaMemsetAsync(d_status, 0, sizeof(int32_t), s) != cudaSuccess) return NN_ERR_CUDA;
        if ((want & NN_WANT_NODES) && cudaMemsetAsync(nodes->row_ptr, 0, 8, s) != cudaSuccess) return NN_ERR_CUDA;
        if ((want & NN_WANT_ELEMS) && cudaMemsetAsync(elems->row_ptr, 0, 8, s) != cudaSuccess) return NN_ERR_CUDA;
        return NN_OK;
    }
    st = enqueue(h, m, p, nodes, elems, w, ws_bytes, nullptr, d_status, h->prof, s);
    if (st == NN_OK && h->prof) h->pending = true;
    return st;
}

// Enqueue the kernels of plan p: rows p.lo .. p.lo + p.N - 1 of the CSRs.
// base: the running {element, node} CSR bases of a chunked build on the
// device, added to every row pointer and col position (nullptr: 0).
nn_status enqueue(nn_handle* h, const nn_mesh* m, const Plan& p, nn_csr* nodes, nn_csr* elems, uint8_t* w,
                  size_t ws_bytes, const int64_t* base, int32_t* d_status, bool prof, cudaStream_t s) {
    const int want = p.want;
    auto mark = [&](int i) {
        if (prof) prof_mark(h, i, s);
    };
    // A direct build has no offsets scan and no node-row scan (a single mesh's
    // rows are placed by sums), so it has no lookback words to clear.  It is
    // always the whole mesh, hence never one of several chunks: those place
    // their rows by the scan and begin with a memset, which a kernel launched
    // as a dependent one may not follow.
    if (p.direct && base) return NN_ERR_ARG;
    const size_t zero = p.direct ? p.off_ctrl : p.zero_begin;
    // (the chunks of a chunked build keep one status word)
    if ((base ? cudaMemsetAsync(w + zero, 0, p.zero_end - zero, s)
              : launch_init(w + zero, p.zero_end - zero, d_status, h->sms, s)) != cudaSuccess)
        return NN_ERR_CUDA;

    uint32_t* ctrl = reinterpret_cast<uint32_t*>(w + p.off_ctrl);
    EmitParams ep{};
    ep.type = p.type;
    ep.n_nodes = m->n_nodes;
    ep.n_elems = p.T;
    ep.n_conn = m->n_conn;
    ep.node_lo = p.lo;
    ep.node_span = p.N;
    ep.conn = m->conn;
    ep.elem_ptr = m->elem_ptr;
    ep.elem_type = m->elem_type;
    ep.fmt = p.fmt;
    ep.n_buckets = p.B;
    ep.hist_chunk = std::max<int64_t>(1, p.hist_chunk);
    ep.n_cta = p.G;
    ep.n_cta_part = p.G_part;
    ep.hist = reinterpret_cast<uint32_t*>(w + p.off_hist);
    ep.nfc = (want & NN_WANT_ELEMS) ? reinterpret_cast<uint32_t*>(w + p.off_nfc) : nullptr;
    ep.gcur = reinterpret_cast<uint32_t*>(w + p.off_gcur);
    ep.gcur_coarse = reinterpret_cast<uint32_t*>(w + p.off_gcur_c);
    ep.rec_tmp = w + p.off_rec_tmp;
    ep.rec = w + p.off_rec;
    ep.rec_cap = (uint64_t)p.n_conn;
    ep.status = d_status;
    ep.chain = p.n_conn <= CHAIN_RECORDS;
    ep.after_kernel = !base;  // (chunks begin with a memset)
    ep.hist_words = (uint64_t)p.G * (uint64_t)p.B;

    OffsetsParams op{};
    op.hist = ep.hist;
    op.n_cta = p.G;
    op.n_buckets = p.B;
    op.bstart = reinterpret_cast<uint32_t*>(w + p.off_bstart);
    op.nfc = ep.nfc;
    op.estart = (want & NN_WANT_ELEMS) ? reinterpret_cast<uint32_t*>(w + p.off_estart) : nullptr;
    op.gcur = ep.gcur;
    op.gcur_coarse = ep.gcur_coarse;
    op.cshift = p.fmt.cshift;
    op.lb_state = reinterpret_cast<uint64_t*>(w + p.off_lb_off);
    op.ticket = ctrl + 0;
    op.rec_cap = (uint64_t)p.n_conn;
    op.status = d_status;

    op.chain = ep.chain;

    BucketParams bp{};
    bp.chain = ep.chain;
    bp.fmt = p.fmt;
    bp.n_nodes = p.N;
    bp.n_buckets = p.B;
    bp.rec = ep.rec;
    bp.bstart = op.bstart;
    bp.estart = op.estart;
    bp.ticket = ctrl + 1;
    bp.spill_cursor = reinterpret_cast<unsigned long long*>(ctrl + 2);
    bp.spill = reinterpret_cast<uint32_t*>(w + p.off_spill);
    const size_t spill_bytes = ws_bytes > p.off_spill ? ws_bytes - p.off_spill : 0;
    bp.spill_words = spill_bytes / 4;
    if (want & NN_WANT_NODES) {
        bp.rp_n = nodes->row_ptr + p.lo;
        bp.col_n = nodes->col;
        bp.cap_n = nodes->col_capacity;
    }
    if (want & NN_WANT_ELEMS) {
        bp.rp_e = elems->row_ptr + p.lo;
        bp.col_e = elems->col;
        bp.cap_e = elems->col_capacity;
    }
    bp.base = base;
    bp.status = d_status;
    bp.imax = p.imax;
    bp.slots = p.slots;
    bp.list_cap = p.list_cap;
    bp.rest = reinterpret_cast<uint32_t*>(w + p.off_gcur);  // (the partition's cursors, dead by now)
    bp.rest_count = ctrl + 5;
    bp.rest_ticket = ctrl + 6;
    bp.rest_cap = (uint64_t)p.B;
    bp.ntmp = reinterpret_cast<uint32_t*>(w + p.off_ntmp);
    bp.grp = reinterpret_cast<uint2*>(w + p.off_grp);
    bp.nloc = reinterpret_cast<uint32_t*>(w + p.off_nloc);
    bp.rec_count = (uint64_t)p.n_conn;
    bp.ntmp_words = (want & NN_WANT_NODES) ? (uint64_t)p.k * p.n_conn + 4 : 0;
    bp.nloc_words = (want & NN_WANT_NODES) ? (uint64_t)p.B << p.fmt.sb : 0;
    bp.ngrp = (want & NN_WANT_NODES) ? (uint64_t)p.B * p.groups : 0;

    mark(1);
    if (!p.direct && launch_hist(ep, p.emit_smem, s) != cudaSuccess) return NN_ERR_CUDA;
    mark(2);
    if (!p.direct && launch_offsets(op, s) != cudaSuccess) return NN_ERR_CUDA;
    mark(3);
    if (p.direct) {
        bp.direct = DirectMesh{p.type, p.N, p.T, m->n_conn, m->conn, m->elem_ptr, m->elem_type,
                               (uint32_t)p.bucket_smem, (uint32_t)p.queue_cap};
        mark(4);
    } else if (p.fmt.cshift >= 0) {
        if (launch_part_coarse(ep, s) != cudaSuccess) return NN_ERR_CUDA;
        mark(4);
        if (launch_part_fine(ep, op.bstart, p.G_fine, s) != cudaSuccess) return NN_ERR_CUDA;
    } else {
        if (launch_part(ep, s) != cudaSuccess) return NN_ERR_CUDA;
        mark(4);
    }
    mark(5);
    if (p.direct ? launch_bucket(bp, (int)p.B, p.bucket_threads, p.bucket_smem + (size_t)p.queue_cap * 4, p.rest, s) != cudaSuccess
                 : launch_bucket(bp, p.bucket_grid, p.bucket_threads, p.bucket_smem, p.rest, s) != cudaSuccess)
        return NN_ERR_CUDA;
    mark(6);
    if (want & NN_WANT_NODES) {
        CompactParams cp{};
        cp.n_buckets = p.B;
        cp.n_groups_cap = p.B * p.groups;
        cp.sb = p.fmt.sb;
        cp.k = p.k;
        cp.n_nodes = p.N;
        cp.base = base;
        cp.chain = bp.chain;
        cp.grp = bp.grp;
        cp.nloc = bp.nloc;
        cp.ntmp = bp.ntmp;
        cp.nstart = reinterpret_cast<uint64_t*>(w + p.off_nstart);
        cp.lb_state = reinterpret_cast<uint64_t*>(w + p.off_lb_ns);
        cp.ticket = ctrl + 4;
        cp.rp_n = nodes->row_ptr + p.lo;
        cp.col_n = nodes->col;
        cp.cap_n = nodes->col_capacity;
        cp.status = d_status;
        cp.ntmp_words = bp.ntmp_words;
        cp.nloc_words = bp.nloc_words;
        if (launch_node_compact(cp, (int)std::min<int64_t>((cp.n_groups_cap + 7) / 8, (int64_t)h->sms * 8), s) != cudaSuccess)
            return NN_ERR_CUDA;
    }
    mark(7);
    return NN_OK;
}

// --------------------------------------------------------------- batches

constexpr int BATCH_SLOTS = 24, BATCH_LIST = 256;

struct BatchPlan {
    int sb = 7, groups = 4;
    int64_t B_cap = 0;
    size_t hdr_bytes = 0, meshes_off = 0, elem_off_off = 0, bucket_off_off = 0, weight_off_off = 0, table_bytes = 0;
    size_t off_bcount = 0, off_bstart = 0, off_gcur = 0, off_rec = 0, off_lb_off = 0, off_ctrl = 0, off_spill = 0, ws_min = 0, ws_rec = 0, off_nfc = 0,
           off_estart = 0, off_ntmp = 0, off_grp = 0, off_nloc = 0, off_nstart = 0, off_lb_ns = 0;
    size_t bucket_smem = 0;
    RestShape rest{};
    int bucket_grid = 0, emit_grid = 0, bucket_threads = 128;
    int64_t tiles_cap = 0;
};

nn_status batch_plan(const nn_handle* h, const nn_batch_caps* c, BatchPlan* out) {
    if (!h || !c || c->max_meshes < 1 || c->max_elems < 0 || c->max_nodes < 0 || c->max_conn < 0 ||
        c->want < 1 || c->want > 3)
        return NN_ERR_ARG;
    if (c->max_conn >= (1ll << 31) || c->max_elems >= (1ll << 31)) return NN_ERR_ARG;
    BatchPlan p;
    p.sb = c->sb ? c->sb : 7;
    if (p.sb < SB_MIN || p.sb > SB_MAX) return NN_ERR_ARG;
    p.hdr_bytes = align_up(sizeof(BatchHeader));
    p.meshes_off = p.hdr_bytes;
    p.elem_off_off = p.meshes_off + align_up((size_t)c->max_meshes * sizeof(BatchMesh));
    p.bucket_off_off = p.elem_off_off + align_up(((size_t)c->max_meshes + 1) * 8);
    p.weight_off_off = p.bucket_off_off + align_up(((size_t)c->max_meshes + 1) * 8);
    p.table_bytes = p.weight_off_off + align_up(((size_t)c->max_meshes + 1) * 8);
    // bucket kernel: the 24 slots of a tet mesh (a batch may hold any element
    // type), 128 threads for buckets of 128 nodes
    p.bucket_threads = 128;
    while (p.sb > SB_MIN && bucket_smem_bytes(p.sb, c->want, 3, BATCH_SLOTS, 16, BATCH_LIST) > h->bucket_smem) --p.sb;
    p.bucket_smem = bucket_smem_bytes(p.sb, c->want, 3, BATCH_SLOTS, 16, BATCH_LIST);
    if (p.bucket_smem > h->bucket_smem) return NN_ERR_ARG;
    p.groups = p.sb < 5 ? 1 : 1 << (p.sb - 5);
    p.B_cap = (c->max_nodes >> p.sb) + c->max_meshes + 1;
    int per_sm = 1;
    if (bucket_occupancy(&per_sm, p.bucket_threads, 32, p.bucket_smem) != cudaSuccess || per_sm < 1) per_sm = 1;
    p.bucket_grid = h->sms * per_sm;
    p.rest = rest_shape(h, p.sb, c->want, 3, 16, p.B_cap);
    size_t o = p.table_bytes;
    p.off_bcount = o; o = align_up(o + (size_t)p.B_cap * 4);
    p.off_nfc = o; o = align_up(o + (size_t)p.B_cap * 4);
    p.off_bstart = o; o = align_up(o + ((size_t)p.B_cap + 1) * 4);
    p.off_estart = o; o = align_up(o + ((size_t)p.B_cap + 1) * 4);
    p.off_gcur = o; o = align_up(o + (size_t)p.B_cap * 4);
    p.off_rec = o; o = align_up(o + (size_t)c->max_conn * 16);
    const bool wn = c->want & NN_WANT_NODES;
    p.off_ntmp = o; o = align_up(o + (wn ? (size_t)3 * c->max_conn * 4 + 16 : 0));
    const size_t ngrp = (size_t)p.B_cap * p.groups;
    p.off_grp = o; o = align_up(o + (wn ? ngrp * 8 : 0));
    p.off_nloc = o; o = align_up(o + (wn ? ((size_t)p.B_cap << p.sb) * 4 : 0));
    p.off_nstart = o; o = align_up(o + (wn ? (ngrp + 1) * 8 : 0));
    p.off_lb_ns = o; o = align_up(o + (wn ? (ngrp + NODE_SCAN_TILE - 1) / NODE_SCAN_TILE * 8 + 8 : 0));
    p.tiles_cap = (p.B_cap + OFFSETS_THREADS - 1) / OFFSETS_THREADS;
    p.off_lb_off = o; o = align_up(o + ((size_t)p.tiles_cap + 1) * 8);
    p.off_ctrl = o; o = align_up(o + 64);
    p.off_spill = o;
    p.ws_min = o;
    p.ws_rec = o + (((size_t)16 << 20) + (size_t)c->max_conn * 8);
    p.emit_grid = h->sms * batch_ctas_per_sm();
    *out = p;
    return NN_OK;
}

nn_status batch_prepare(nn_handle* h, const nn_batch_caps* c, const nn_mesh* meshes, const nn_csr* node_out,
                        const nn_csr* elem_out, int32_t* d_status, int n, void* staging, size_t staging_bytes) {
    BatchPlan bp;
    nn_status st = batch_plan(h, c, &bp);
    if (st != NN_OK) return st;
    if (n < 0 || n > c->max_meshes || !staging || staging_bytes < bp.table_bytes || (n > 0 && (!meshes || !d_status)))
        return NN_ERR_ARG;
    if ((c->want & NN_WANT_NODES) && n > 0 && !node_out) return NN_ERR_ARG;
    if ((c->want & NN_WANT_ELEMS) && n > 0 && !elem_out) return NN_ERR_ARG;
    uint8_t* sg = static_cast<uint8_t*>(staging);
    BatchHeader* hdr = reinterpret_cast<BatchHeader*>(sg);
    BatchMesh* bm = reinterpret_cast<BatchMesh*>(sg + bp.meshes_off);
    int64_t* eoff = reinterpret_cast<int64_t*>(sg + bp.elem_off_off);
    int64_t* boff = reinterpret_cast<int64_t*>(sg + bp.bucket_off_off);
    int64_t* woff = reinterpret_cast<int64_t*>(sg + bp.weight_off_off);
    int64_t E = 0, Bk = 0, C = 0, Nn = 0, maxT = 0, maxN = 0;
    for (int m = 0; m < n; ++m) {
        const nn_mesh& M = meshes[m];
        if ((st = check_mesh(&M)) != NN_OK) return st;
        BatchMesh& d = bm[m];
        d = BatchMesh{};
        d.type = M.type;
        d.k = (M.type == NN_TRI || M.type == NN_QUAD) ? 2 : 3;
        d.n_nodes = M.n_nodes;
        d.n_elems = M.n_elems;
        d.n_conn = M.n_conn;
        d.conn = M.conn;
        d.elem_ptr = M.elem_ptr;
        d.elem_type = M.elem_type;
        if (c->want & NN_WANT_NODES) {
            const nn_csr& o = node_out[m];
            if (!o.row_ptr || o.col_capacity < 0 || (o.col_capacity > 0 && !o.col)) return NN_ERR_ARG;
            d.rp_n = o.row_ptr; d.col_n = o.col; d.cap_n = o.col_capacity;
        }
        if (c->want & NN_WANT_ELEMS) {
            const nn_csr& o = elem_out[m];
            if (!o.row_ptr || o.col_capacity < 0 || (o.col_capacity > 0 && !o.col)) return NN_ERR_ARG;
            d.rp_e = o.row_ptr; d.col_e = o.col; d.cap_e = o.col_capacity;
        }
        d.status = d_status + m;
        eoff[m] = E;
        boff[m] = Bk;
        woff[m] = C + E;
        E += M.n_elems;
        Bk += (M.n_nodes + (1ll << bp.sb) - 1) >> bp.sb;
        C += M.n_conn;
        Nn += M.n_nodes;
        maxT = std::max<int64_t>(maxT, M.n_elems);
        maxN = std::max<int64_t>(maxN, M.n_nodes);
    }
    eoff[n] = E;
    boff[n] = Bk;
    woff[n] = C + E;
    if (E > c->max_elems || C > c->max_conn || Nn > c->max_nodes || Bk > bp.B_cap) return NN_ERR_BUDGET;
    RecFmt f{};
    if (!record_format(bp.sb, c->want, 3, maxT, maxN, -1, 16, &f)) return NN_ERR_ARG;
    hdr->fmt = f;
    hdr->n_meshes = n;
    hdr->n_elems = E;
    hdr->n_buckets = Bk;
    hdr->n_records = C;
    return NN_OK;
}

nn_status batch_launch(nn_handle* h, const nn_batch_caps* c, const void* staging, void* ws, size_t ws_bytes,
                       cudaStream_t s) {
    if (!h || h->offline) return NN_ERR_ARG;
    BatchPlan bp;
    nn_status st = batch_plan(h, c, &bp);
    if (st != NN_OK) return st;
    if (!staging || !ws || (reinterpret_cast<uintptr_t>(ws) & (ALIGN - 1))) return NN_ERR_ARG;
    if (ws_bytes < bp.ws_min) return NN_ERR_WORKSPACE;
    uint8_t* w = static_cast<uint8_t*>(ws);
    if (cudaMemcpyAsync(w, staging, bp.table_bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) return NN_ERR_CUDA;
    const bool chain = c->max_conn <= CHAIN_RECORDS;
    BatchTables bt;
    bt.hdr = reinterpret_cast<const BatchHeader*>(w);
    bt.meshes = reinterpret_cast<const BatchMesh*>(w + bp.meshes_off);
    bt.elem_off = reinterpret_cast<const int64_t*>(w + bp.elem_off_off);
    bt.bucket_off = reinterpret_cast<const int64_t*>(w + bp.bucket_off_off);
    bt.weight_off = reinterpret_cast<const int64_t*>(w + bp.weight_off_off);
    uint32_t* bcount = reinterpret_cast<uint32_t*>(w + bp.off_bcount);
    uint32_t* nfc = reinterpret_cast<uint32_t*>(w + bp.off_nfc);
    uint32_t* gcur = reinterpret_cast<uint32_t*>(w + bp.off_gcur);
    uint32_t* ctrl = reinterpret_cast<uint32_t*>(w + bp.off_ctrl);
    uint64_t* lb_off = reinterpret_cast<uint64_t*>(w + bp.off_lb_off);
    uint8_t* rec = w + bp.off_rec;
    if (launch_batch_emit(bt, bcount, nfc, gcur, rec, lb_off, ctrl, bp.emit_grid, 0, chain, s,
                          reinterpret_cast<uint64_t*>(w + bp.off_lb_ns)) != cudaSuccess)
        return NN_ERR_CUDA;
    if (launch_batch_emit(bt, bcount, nfc, gcur, rec, lb_off, ctrl, bp.emit_grid, 1, chain, s) != cudaSuccess)
        return NN_ERR_CUDA;
    OffsetsParams op{};
    op.hist = bcount;
    op.n_cta = 1;
    op.n_buckets = bp.B_cap;
    op.bstart = reinterpret_cast<uint32_t*>(w + bp.off_bstart);
    op.nfc = nfc;
    op.estart = (c->want & NN_WANT_ELEMS) ? reinterpret_cast<uint32_t*>(w + bp.off_estart) : nullptr;
    op.gcur = gcur;
    op.lb_state = lb_off;
    op.ticket = ctrl + 0;
    op.rec_cap = (uint64_t)c->max_conn;
    op.status = reinterpret_cast<int32_t*>(ctrl + 8);  // passed on to every mesh by the bucket pass
    op.hdr = bt.hdr;
    op.chain = chain;
    if (launch_offsets(op, s) != cudaSuccess) return NN_ERR_CUDA;
    if (launch_batch_emit(bt, bcount, nfc, gcur, rec, lb_off, ctrl, bp.emit_grid, 2, chain, s) != cudaSuccess)
        return NN_ERR_CUDA;
    BucketParams kp{};
    kp.n_buckets = 0;
    kp.rec = rec;
    kp.bstart = op.bstart;
    kp.estart = op.estart;
    kp.ticket = ctrl + 1;
    kp.spill_cursor = reinterpret_cast<unsigned long long*>(ctrl + 2);
    kp.spill = reinterpret_cast<uint32_t*>(w + bp.off_spill);
    const size_t spill_bytes = ws_bytes > bp.off_spill ? ws_bytes - bp.off_spill : 0;
    kp.spill_words = spill_bytes / 4;
    kp.batch = bt;
    kp.batch_err = reinterpret_cast<const int32_t*>(ctrl + 8);
    kp.fmt.rb = 16;
    kp.fmt.k = 3;
    kp.imax = 32;
    kp.chain = chain;
    kp.slots = BATCH_SLOTS;
    kp.list_cap = BATCH_LIST;
    kp.rest = gcur;  // (dead after the partition)
    kp.rest_count = ctrl + 5;
    kp.rest_ticket = ctrl + 6;
    kp.rest_cap = (uint64_t)bp.B_cap;
    kp.ntmp = reinterpret_cast<uint32_t*>(w + bp.off_ntmp);
    kp.grp = reinterpret_cast<uint2*>(w + bp.off_grp);
    kp.nloc = reinterpret_cast<uint32_t*>(w + bp.off_nloc);
    kp.rec_count = (uint64_t)c->max_conn;
    kp.ntmp_words = (c->want & NN_WANT_NODES) ? 3 * (uint64_t)c->max_conn + 4 : 0;
    kp.nloc_words = (c->want & NN_WANT_NODES) ? (uint64_t)bp.B_cap << bp.sb : 0;
    kp.ngrp = (c->want & NN_WANT_NODES) ? (uint64_t)bp.B_cap * bp.groups : 0;
    if (launch_bucket(kp, bp.bucket_grid, bp.bucket_threads, bp.bucket_smem, bp.rest, s) != cudaSuccess) return NN_ERR_CUDA;
    if (c->want & NN_WANT_NODES) {
        CompactParams cp{};
        cp.n_groups_cap = bp.B_cap * bp.groups;
        cp.grp = kp.grp;
        cp.nloc = kp.nloc;
        cp.ntmp = kp.ntmp;
        cp.nstart = reinterpret_cast<uint64_t*>(w + bp.off_nstart);
        cp.lb_state = reinterpret_cast<uint64_t*>(w + bp.off_lb_ns);
        cp.ticket = ctrl + 4;
        cp.status = reinterpret_cast<int32_t*>(ctrl + 8);
        cp.batch = bt;
        cp.chain = chain;
        cp.ntmp_words = kp.ntmp_words;
        cp.nloc_words = kp.nloc_words;
        if (launch_node_compact(cp, h->sms * 8, s) != cudaSuccess) return NN_ERR_CUDA;
    }
    return NN_OK;
}

}  // namespace

namespace nn {

// Build with a handle described by plain device limits (no handle object on
// the heap): used by the allocation-free entry point.
nn_status build_with_limits(int sms, size_t smem_optin, size_t smem_per_sm, const nn_mesh* m, int want,
                            nn_csr* nodes, nn_csr* elems, void* ws, size_t ws_bytes, int32_t* d_status,
                            cudaStream_t s, size_t* ws_min) {
    nn_handle h;
    h.sms = sms;
    h.smem_optin = smem_optin;
    h.smem_per_sm = smem_per_sm;
    h.bucket_smem = smem_optin - 1024;  // the bucket kernel has a little static shared memory
    Plan p;
    nn_status st = make_plan(&h, m, want, &p);
    if (st != NN_OK) return st;
    if (ws_min) *ws_min = p.ws_min;
    if (p.ws_min > ws_bytes) return NN_ERR_WORKSPACE;
    return run(&h, m, want, nodes, elems, ws, ws_bytes, d_status, s);
}

}  // namespace nn

extern "C" {

nn_status nn_create(nn_handle** out) {
    if (!out) return NN_ERR_ARG;
    nn_handle* h = new (std::nothrow) nn_handle();
    if (!h) return NN_ERR_ARG;
    int optin = 0, per_sm = 0;
    if (cudaGetDevice(&h->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, h->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, h->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device) != cudaSuccess) {
        delete h;
        return NN_ERR_CUDA;
    }
    h->smem_optin = (size_t)optin;
    h->smem_per_sm = (size_t)per_sm;
    h->bucket_smem = h->smem_optin - 1024;  // the bucket kernel has a little static shared memory
    if (const char* e = std::getenv("NN_SB")) h->sb_override = std::atoi(e);
    if (const char* e = std::getenv("NN_PART")) h->part_mode = std::strcmp(e, "scatter") == 0 ? 0 : (std::strcmp(e, "sorted") == 0 ? 1 : -1);
    if (const char* e = std::getenv("NN_HIST_CHUNK")) h->hist_chunk_override = std::atoll(e);
    if (const char* e = std::getenv("NN_EMIT_CTAS")) h->emit_ctas_override = std::atoi(e);
    if (const char* e = std::getenv("NN_BUCKET_SMEM_KB")) {
        size_t kb = (size_t)std::atol(e);
        if (kb >= 32 && kb * 1024 <= h->smem_optin - 1024) h->bucket_smem = kb * 1024;
    }
    if (set_emit_smem_all(h->smem_optin) != cudaSuccess || set_bucket_smem_all(h->smem_optin) != cudaSuccess) {
        delete h;
        return NN_ERR_CUDA;
    }
    *out = h;
    return NN_OK;
}

nn_status nn_create_offline(nn_handle** out, int32_t sms, int32_t smem_optin, int32_t smem_per_sm) {
    if (!out || sms < 1 || smem_optin < 64 * 1024 || smem_per_sm < smem_optin) return NN_ERR_ARG;
    nn_handle* h = new (std::nothrow) nn_handle();
    if (!h) return NN_ERR_ARG;
    h->device = -1;
    h->offline = true;
    h->sms = sms;
    h->smem_optin = (size_t)smem_optin;
    h->smem_per_sm = (size_t)smem_per_sm;
    h->bucket_smem = h->smem_optin - 1024;
    *out = h;
    return NN_OK;
}

void nn_destroy(nn_handle* h) {
    if (!h) return;
    for (cudaEvent_t e : h->ev)
        if (e) cudaEventDestroy(e);
    delete h;
}

nn_status nn_profile_enable(nn_handle* h, int enable) {
    if (!h || h->offline) return NN_ERR_ARG;
    if (enable && !h->ev[0])
        for (cudaEvent_t& e : h->ev)
            if (cudaEventCreate(&e) != cudaSuccess) return NN_ERR_CUDA;
    h->pending = false;
    h->prof = enable != 0;
    for (double& a : h->acc) a = 0.0;
    h->calls = 0;
    return NN_OK;
}

nn_status nn_profile_read(nn_handle* h, double* ms, int64_t* calls, int n_stages) {
    if (!h || n_stages < 0 || n_stages > NN_PROFILE_STAGES) return NN_ERR_ARG;
    prof_flush(h);
    for (int i = 0; i < n_stages; ++i) ms[i] = h->acc[i];
    if (calls) *calls = h->calls;
    return NN_OK;
}

nn_status nn_query(nn_handle* h, const nn_mesh* mesh, int want, size_t* ws_bytes, int64_t* node_col_cap,
                   int64_t* elem_col_cap) {
    if (!h) return NN_ERR_ARG;
    Plan p;
    nn_status st = make_plan(h, mesh, want, &p);
    if (st != NN_OK) return st;
    if (ws_bytes) *ws_bytes = p.ws_rec;
    // bound on node entries: every incidence has at most k edge ends (2 tri/quad, 3 tet/hex)
    if (node_col_cap) *node_col_cap = (int64_t)p.k * p.n_conn;
    if (elem_col_cap) *elem_col_cap = p.n_conn;
    return NN_OK;
}

nn_status nn_plan_info(nn_handle* h, const nn_mesh* mesh, int want, int64_t* info, int n) {
    if (!h || (!info && n > 0) || n < 0) return NN_ERR_ARG;
    Plan p;
    nn_status st = make_plan(h, mesh, want, &p);
    if (st != NN_OK) return st;
    // initialization, histogram, offsets and partition unless direct, buckets (twice unless direct), placement of node rows
    const int64_t kernels = 2 + (p.direct ? 0 : 4 + (p.fmt.cshift > 0)) +
                            (want & NN_WANT_NODES ? (p.B * p.groups <= NODE_SUM_GROUPS ? 1 : 2) : 0);
    const int64_t v[10] = {p.fmt.sb, p.B, p.G, p.fmt.rb, (int64_t)p.ws_min, p.bucket_grid, p.bucket_threads,
                           (int64_t)p.bucket_smem, p.fmt.cshift, p.N > 0 ? kernels : 0};
    for (int i = 0; i < n && i < 10; ++i) info[i] = v[i];
    return NN_OK;
}

namespace {

// Workspace of the counts and the scan, which every call needs, and of the
// slots and flags of the matching pass.
size_t adjacency_merge_bytes(size_t T) {
    return align_up(T * 4) + align_up((adjacency_scan_tiles((int64_t)T) + 1) * 8) + ALIGN;
}
size_t adjacency_match_bytes(int type, size_t T) {
    const size_t slots = (size_t)adjacency_slots(type);
    return slots ? align_up(T * slots * 4) + align_up(T) : 0;
}

}  // namespace

nn_status nn_element_neighbors_query(nn_handle* h, const nn_mesh* mesh, size_t* ws_bytes, int64_t* col_cap) {
    if (!h) return NN_ERR_ARG;
    nn_status st = check_mesh(mesh);
    if (st != NN_OK) return st;
    const size_t T = (size_t)mesh->n_elems;
    if (ws_bytes) *ws_bytes = adjacency_merge_bytes(T) + adjacency_match_bytes(mesh->type, T);
    // faces per element (6 at most) times two
    if (col_cap) *col_cap = (int64_t)T * (mesh->type == NN_TRI ? 6 : mesh->type == NN_HEX || mesh->type == NN_MIXED ? 12 : 8);
    return NN_OK;
}

nn_status nn_element_neighbors(nn_handle* h, const nn_mesh* mesh, const nn_csr* node_elems, nn_csr* out, void* ws,
                               size_t ws_bytes, int32_t* d_status, nn_stream_t stream) {
    if (!h || h->offline || !node_elems || !node_elems->row_ptr || !out || !out->row_ptr || !d_status) return NN_ERR_ARG;
    nn_status st = check_mesh(mesh);
    if (st != NN_OK) return st;
    if (out->col_capacity < 0 || (out->col_capacity > 0 && !out->col)) return NN_ERR_ARG;
    if (mesh->n_conn > 0 && !node_elems->col) return NN_ERR_ARG;
    const size_t need = adjacency_merge_bytes((size_t)mesh->n_elems);
    if (ws_bytes < need || !ws || (reinterpret_cast<uintptr_t>(ws) & (ALIGN - 1))) return NN_ERR_WORKSPACE;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    uint8_t* w = static_cast<uint8_t*>(ws);
    const size_t T = (size_t)mesh->n_elems;
    const size_t off_lb = align_up(T * 4), off_ticket = off_lb + align_up((adjacency_scan_tiles((int64_t)T) + 1) * 8);
    if (cudaMemsetAsync(d_status, 0, sizeof(int32_t), s) != cudaSuccess) return NN_ERR_CUDA;
    if (cudaMemsetAsync(w + off_lb, 0, off_ticket + ALIGN - off_lb, s) != cudaSuccess) return NN_ERR_CUDA;
    if (T == 0) return cudaMemsetAsync(out->row_ptr, 0, 8, s) == cudaSuccess ? NN_OK : NN_ERR_CUDA;
    AdjParams p{};
    p.type = mesh->type;
    p.n_nodes = mesh->n_nodes;
    p.n_elems = mesh->n_elems;
    p.n_conn = mesh->n_conn;
    p.conn = mesh->conn;
    p.elem_ptr = mesh->elem_ptr;
    p.elem_type = mesh->elem_type;
    p.ne_rp = node_elems->row_ptr;
    p.ne_col = node_elems->col;
    p.cnt = reinterpret_cast<uint32_t*>(w);
    p.lb_state = reinterpret_cast<uint64_t*>(w + off_lb);
    p.ticket = reinterpret_cast<uint32_t*>(w + off_ticket);
    p.rp = out->row_ptr;
    p.col = out->col;
    p.cap = out->col_capacity;
    p.status = d_status;
    // a workspace without room for the slots still serves: every element then
    // merges its node rows
    const size_t match = adjacency_match_bytes(mesh->type, T);
    if (match && ws_bytes >= need + match) {
        p.nbr = reinterpret_cast<int32_t*>(w + need);
        p.cplx = w + need + match - align_up(T);
        if (cudaMemsetAsync(p.cplx, 0, T, s) != cudaSuccess) return NN_ERR_CUDA;
    }
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)h->sms * 8, ((int64_t)T + 255) / 256));
    return launch_adjacency(p, grid, h->sms, s) == cudaSuccess ? NN_OK : NN_ERR_CUDA;
}

nn_status nn_set_tuning(nn_handle* h, const nn_tuning* t) {
    if (!h) return NN_ERR_ARG;
    if (!t) {
        h->tuning = nn_tuning{};
        return NN_OK;
    }
    if ((t->sb != 0 && (t->sb < SB_MIN || t->sb > SB_MAX)) ||
        (t->bucket_threads != 0 && t->bucket_threads != 128 && t->bucket_threads != 256) ||
        t->bucket_ctas_per_sm < 0 || t->bucket_ctas_per_sm > 8)
        return NN_ERR_ARG;
    h->tuning = *t;
    return NN_OK;
}

nn_status nn_neighbor_nodes(nn_handle* h, const nn_mesh* mesh, nn_csr* out, void* ws, size_t ws_bytes,
                            int32_t* d_status, nn_stream_t stream) {
    return run(h, mesh, NN_WANT_NODES, out, nullptr, ws, ws_bytes, d_status, reinterpret_cast<cudaStream_t>(stream));
}

nn_status nn_neighbor_elements(nn_handle* h, const nn_mesh* mesh, nn_csr* out, void* ws, size_t ws_bytes,
                               int32_t* d_status, nn_stream_t stream) {
    return run(h, mesh, NN_WANT_ELEMS, nullptr, out, ws, ws_bytes, d_status, reinterpret_cast<cudaStream_t>(stream));
}

nn_status nn_neighbors_both(nn_handle* h, const nn_mesh* mesh, nn_csr* nodes, nn_csr* elems, void* ws,
                            size_t ws_bytes, int32_t* d_status, nn_stream_t stream) {
    return run(h, mesh, NN_WANT_BOTH, nodes, elems, ws, ws_bytes, d_status, reinterpret_cast<cudaStream_t>(stream));
}

// ------------------------------------------------------ chunked builds

namespace {

// Whether kernels on device `dev` may dereference ptr: device or managed
// memory, pinned host memory mapped at the same address (unified
// addressing), or any host memory where the device reads pageable memory.
bool addressable(const void* ptr, int dev) {
    if (!ptr) return true;
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) return true;
    if (a.type == cudaMemoryTypeHost) return a.devicePointer == ptr;
    int pageable = 0;
    if (cudaDeviceGetAttribute(&pageable, cudaDevAttrPageableMemoryAccess, dev) != cudaSuccess) return false;
    return pageable != 0;
}

bool on_device(const void* ptr) {
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

bool mesh_addressable(const nn_mesh* m, int dev) {
    return addressable(m->conn, dev) && addressable(m->elem_ptr, dev) && addressable(m->elem_type, dev);
}

}  // namespace

nn_status nn_chunk_slabs(const nn_mesh* mesh, int* shift, int* n_slabs) {
    nn_status st = check_mesh(mesh);
    if (st != NN_OK) return st;
    int sh = 0;
    while (((mesh->n_nodes + (1ll << sh) - 1) >> sh) > NN_CHUNK_SLABS_MAX) ++sh;
    if (shift) *shift = sh;
    if (n_slabs) *n_slabs = (int)((mesh->n_nodes + (1ll << sh) - 1) >> sh);
    return NN_OK;
}

nn_status nn_chunk_count(nn_handle* h, const nn_mesh* mesh, uint32_t* d_counts, int32_t* d_status,
                         nn_stream_t stream) {
    if (!h || h->offline || !d_status) return NN_ERR_ARG;
    int shift = 0, ns = 0;
    nn_status st = nn_chunk_slabs(mesh, &shift, &ns);
    if (st != NN_OK) return st;
    if (ns > 0 && !d_counts) return NN_ERR_ARG;
    if (!on_device(d_status) || (ns > 0 && !on_device(d_counts)) || !mesh_addressable(mesh, h->device))
        return NN_ERR_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(d_status, 0, sizeof(int32_t), s) != cudaSuccess) return NN_ERR_CUDA;
    if (ns == 0) return NN_OK;
    if (cudaMemsetAsync(d_counts, 0, (size_t)ns * 4, s) != cudaSuccess) return NN_ERR_CUDA;
    if (mesh->n_elems == 0) return NN_OK;
    EmitParams ep{};
    ep.type = mesh->type;
    ep.n_nodes = mesh->n_nodes;
    ep.n_elems = mesh->n_elems;
    ep.n_conn = mesh->n_conn;
    ep.conn = mesh->conn;
    ep.elem_ptr = mesh->elem_ptr;
    ep.elem_type = mesh->elem_type;
    // element-walk CTAs as in a build: two per SM, each a fixed slice of elements
    const int64_t n_units = (mesh->n_elems + (mesh->type == NN_TRI ? 3 : 0)) / (mesh->type == NN_TRI ? 4 : 1);
    ep.n_cta = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)h->sms * 2, (n_units + 2047) / 2048));
    ep.status = d_status;
    return launch_slab_count(ep, shift, ns, d_counts, s) == cudaSuccess ? NN_OK : NN_ERR_CUDA;
}

nn_status nn_chunk_query(nn_handle* h, const nn_mesh* mesh, int want, const nn_chunk* chunk, size_t* ws_bytes) {
    if (!h || !chunk || chunk->node_hi <= chunk->node_lo) return NN_ERR_ARG;
    Plan p;
    nn_status st = make_plan_range(h, mesh, want, chunk->node_lo, chunk->node_hi - chunk->node_lo, chunk->records, &p);
    if (st != NN_OK) return st;
    if (ws_bytes) *ws_bytes = ALIGN + p.ws_rec;  // the running CSR bases, then the chunk's plan
    return NN_OK;
}

nn_status nn_chunk_plan(nn_handle* h, const nn_mesh* mesh, int want, const uint32_t* counts, size_t ws_bytes,
                        nn_chunk* chunks, int max_chunks, int* n_chunks, size_t* ws_needed) {
    if (!h || !n_chunks || max_chunks < 0 || (max_chunks > 0 && !chunks)) return NN_ERR_ARG;
    int shift = 0, ns = 0;
    nn_status st = nn_chunk_slabs(mesh, &shift, &ns);
    if (st != NN_OK) return st;
    if (want < 1 || want > 3 || (ns > 0 && !counts)) return NN_ERR_ARG;
    const int64_t N = mesh->n_nodes;
    int64_t total = 0;
    for (int i = 0; i < ns; ++i) total += counts[i];
    if (total > mesh->n_conn) return NN_ERR_ARG;  // not this mesh's counts
    // workspace of the chunk of slabs i..j
    auto need = [&](int i, int j, int64_t rec, size_t* out) {
        const nn_chunk k{(int64_t)i << shift, std::min<int64_t>(N, (int64_t)(j + 1) << shift), rec};
        return nn_chunk_query(h, mesh, want, &k, out);
    };
    // the smallest workspace that admits a plan: the largest single slab
    size_t worst = ALIGN;
    for (int i = 0; i < ns; ++i) {
        size_t w1 = 0;
        if ((st = need(i, i, counts[i], &w1)) != NN_OK) return st;
        worst = std::max(worst, w1);
    }
    if (ws_needed) *ws_needed = worst;
    if (worst > ws_bytes) {
        *n_chunks = 0;
        return NN_ERR_WORKSPACE;
    }
    // greedy: each chunk takes slabs while its plan still fits the workspace
    int n = 0;
    for (int i = 0; i < ns;) {
        int j = i;
        int64_t rec = counts[i];
        while (j + 1 < ns) {
            size_t w2 = 0;
            if (need(i, j + 1, rec + counts[j + 1], &w2) != NN_OK || w2 > ws_bytes) break;
            ++j;
            rec += counts[j];
        }
        if (n < max_chunks)
            chunks[n] = nn_chunk{(int64_t)i << shift, std::min<int64_t>(N, (int64_t)(j + 1) << shift), rec};
        ++n;
        i = j + 1;
    }
    *n_chunks = n;
    return n > max_chunks ? NN_ERR_CAPACITY : NN_OK;
}

nn_status nn_neighbors_chunked(nn_handle* h, const nn_mesh* mesh, int want, const nn_chunk* chunks, int n_chunks,
                               nn_csr* nodes, nn_csr* elems, void* ws, size_t ws_bytes, int32_t* d_status,
                               nn_stream_t stream) {
    if (!h || h->offline || !d_status || n_chunks < 0 || (n_chunks > 0 && !chunks)) return NN_ERR_ARG;
    nn_status st = check_mesh(mesh);
    if (st != NN_OK) return st;
    if (want < 1 || want > 3) return NN_ERR_ARG;
    st = check_outputs(want, nodes, elems);
    if (st != NN_OK) return st;
    if (!ws) return NN_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(ws) & (ALIGN - 1)) || !on_device(ws) || !on_device(d_status) || !mesh_addressable(mesh, h->device)) return NN_ERR_ARG;
    if ((want & NN_WANT_NODES) && (!addressable(nodes->row_ptr, h->device) || !addressable(nodes->col, h->device)))
        return NN_ERR_ARG;
    if ((want & NN_WANT_ELEMS) && (!addressable(elems->row_ptr, h->device) || !addressable(elems->col, h->device)))
        return NN_ERR_ARG;
    const int64_t N = mesh->n_nodes;
    // the chunks must tile [0, N) in order
    if (N > 0 && (n_chunks == 0 || chunks[0].node_lo != 0 || chunks[n_chunks - 1].node_hi != N)) return NN_ERR_ARG;
    for (int c = 0; c < n_chunks; ++c) {
        const nn_chunk& k = chunks[c];
        if (k.node_hi <= k.node_lo || (c > 0 && k.node_lo != chunks[c - 1].node_hi) || k.records < 0 ||
            k.records > mesh->n_conn)
            return NN_ERR_ARG;
        Plan p;
        if ((st = make_plan_range(h, mesh, want, k.node_lo, k.node_hi - k.node_lo, k.records, &p)) != NN_OK)
            return st;
        if (ALIGN + p.ws_min > ws_bytes) return NN_ERR_WORKSPACE;
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    uint8_t* w = static_cast<uint8_t*>(ws);
    int64_t* base = reinterpret_cast<int64_t*>(w);
    if (cudaMemsetAsync(d_status, 0, sizeof(int32_t), s) != cudaSuccess) return NN_ERR_CUDA;
    if (cudaMemsetAsync(base, 0, 2 * sizeof(int64_t), s) != cudaSuccess) return NN_ERR_CUDA;
    if (N == 0) {
        if ((want & NN_WANT_NODES) && cudaMemsetAsync(nodes->row_ptr, 0, 8, s) != cudaSuccess) return NN_ERR_CUDA;
        if ((want & NN_WANT_ELEMS) && cudaMemsetAsync(elems->row_ptr, 0, 8, s) != cudaSuccess) return NN_ERR_CUDA;
        return NN_OK;
    }
    uint8_t* cw = w + ALIGN;
    // a chunk that is the whole mesh is a single build, with no offsets to run on
    const bool single = n_chunks == 1;
    for (int c = 0; c < n_chunks; ++c) {
        Plan p;
        make_plan_range(h, mesh, want, chunks[c].node_lo, chunks[c].node_hi - chunks[c].node_lo, chunks[c].records, &p);
        // connectivity that stays on the host is read twice, not by every
        // bucket's CTA (6,859 hexes in pinned memory 156 -> 37 us); the other
        // plan's tables are a few KB larger, which the spill area has room for
        if (p.direct && !(on_device(mesh->conn) && (!mesh->elem_ptr || on_device(mesh->elem_ptr)))) {
            Plan q;
            if (make_plan_range(h, mesh, want, 0, N, chunks[c].records, &q, true) == NN_OK && ALIGN + q.ws_min <= ws_bytes) p = q;
        }
        if ((st = enqueue(h, mesh, p, nodes, elems, cw, ws_bytes - ALIGN, single ? nullptr : base, d_status, false, s)) !=
            NN_OK)
            return st;
        if (single) break;
        // (the chunk's totals end its two scans)
        const uint32_t* etot = (want & NN_WANT_ELEMS) ? reinterpret_cast<const uint32_t*>(cw + p.off_estart) + p.B : nullptr;
        const uint64_t* ntot = (want & NN_WANT_NODES) ? reinterpret_cast<const uint64_t*>(cw + p.off_nstart) + p.B * p.groups : nullptr;
        if (launch_chunk_advance(base, etot, ntot, s) != cudaSuccess) return NN_ERR_CUDA;
    }
    return NN_OK;
}

nn_status nn_batch_query(nn_handle* h, const nn_batch_caps* caps, size_t* ws_bytes, size_t* staging_bytes) {
    BatchPlan bp;
    nn_status st = batch_plan(h, caps, &bp);
    if (st != NN_OK) return st;
    if (ws_bytes) *ws_bytes = bp.ws_rec;
    if (staging_bytes) *staging_bytes = bp.table_bytes;
    return NN_OK;
}

nn_status nn_batch_prepare(nn_handle* h, const nn_batch_caps* caps, const nn_mesh* meshes, const nn_csr* node_out,
                           const nn_csr* elem_out, int32_t* d_status, int n_meshes, void* staging,
                           size_t staging_bytes) {
    return batch_prepare(h, caps, meshes, node_out, elem_out, d_status, n_meshes, staging, staging_bytes);
}

nn_status nn_batch_launch(nn_handle* h, const nn_batch_caps* caps, const void* staging, void* ws, size_t ws_bytes,
                          nn_stream_t stream) {
    return batch_launch(h, caps, staging, ws, ws_bytes, reinterpret_cast<cudaStream_t>(stream));
}

const char* nn_status_str(nn_status s) {
    switch (s) {
        case NN_OK: return "ok";
        case NN_ERR_ARG: return "invalid argument";
        case NN_ERR_WORKSPACE: return "workspace too small";
        case NN_ERR_CAPACITY: return "output capacity too small";
        case NN_ERR_NODE_RANGE: return "node id out of range";
        case NN_ERR_ELEM_PTR: return "element offsets inconsistent with element types";
        case NN_ERR_TIMEOUT: return "device wait timed out";
        case NN_ERR_BUDGET: return "request exceeds memory budget";
        case NN_ERR_CUDA: return "CUDA error";
        case NN_ERR_BOUNDS: return "index outside its buffer (checked build)";
    }
    return "unknown status";
}

}  // extern "C"
