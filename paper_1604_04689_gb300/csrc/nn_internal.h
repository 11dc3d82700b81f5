// Internal host/device interface of libnn: the build plan, kernel parameter
// blocks and the launchers defined in the kernel translation units.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "nn.h"

namespace nn {

// Layout of one packed incidence record (node v is local node i of element e).
// Its fields:
//   side   : v's place in its bucket and, above it, the bucket's place in its
//            coarse region (together the low sb + max(cshift, 0) bits of v's
//            id relative to the build's first node), then, when element rows
//            are wanted, 1 if v already occurred earlier in e (off_nf)
//   e      : element id                    [eb bits, elems wanted]
//   n_0..  : k edge neighbours of v in e   [nb bits each, nodes wanted; all ones = none]
// 8 bytes when the fields fit 64 bits: side from bit 0, e, n_0, n_1, ..
// Else 16 bytes: e in word 0 and n_j in word 1 + j, each in the word's low
// bits, so that a reader masks it out; the side takes a word of its own where
// one is free (word 3 when k = 2, word 0 when no element rows are wanted),
// and otherwise (side_split) the words' high bits: word 1's, then word 2's,
// word 3's and word 0's.  (Fields packed bit after bit across word boundaries
// cost about ten instructions each to put and to get: with this layout the
// coarse pass of hex 257^3 went from 0.96 to 0.68 ms, the bucket pass from
// 1.61 to 1.38 ms.)
struct RecFmt {
    int sb;
    int want;
    int k;
    int off_nf;              // within the side
    int eb, nb;
    int off_e, off_n;        // 8-byte records: bit offsets of e and n_0
    int rb;                  // 8 or 16
    // Partition: cshift < 0 -> one scattered pass (one store per record);
    // cshift == 0 -> one tile-sorted pass with the bucket as radix digit
    // (at most 256 buckets); cshift > 0 -> a tile-sorted pass on the coarse
    // digit (bucket >> cshift) into a temporary array, then a tile-sorted
    // pass per coarse region on the fine digit, which the side holds.
    int cshift;
    int side_split;          // 16-byte records: the side is spread over the words' high bits
    int sh2, sh3, sh0;       // ... first side bit of word 2, 3 and 0 (word 1's is 0; at most 31)
    uint32_t emask, nmask;   // nmask is also the stored "no neighbour"
};

// Element walk: the kernels that read the connectivity (histogram and
// partition passes).  Each CTA owns a fixed range of work units; a unit is 4
// triangles (three 16-byte loads) or one element of any other type.
struct EmitParams {
    int type;
    int64_t n_nodes, n_elems, n_conn;
    const int32_t* conn;
    const int64_t* elem_ptr;
    const uint8_t* elem_type;
    RecFmt fmt;
    // node range of this build: incidences of nodes outside [node_lo,
    // node_lo + node_span) are skipped, buckets count from node_lo (a whole
    // mesh: 0 and n_nodes; a chunked build: one chunk)
    int64_t node_lo, node_span;
    int64_t n_buckets;
    int64_t hist_chunk;  // buckets counted per walk of the histogram pass (shared counters)
    int n_cta;        // CTAs of the histogram pass (rows of hist)
    int n_cta_part;   // CTAs of the partition pass
    uint32_t* hist;   // [n_cta][n_buckets] record counts of each CTA's element slice
    uint32_t* nfc;    // [n_buckets] records of a node already seen in its element (they add no element entry)
    uint32_t* gcur;   // [n_buckets] write cursor of each bucket (starts at the bucket start)
    uint32_t* gcur_coarse;  // [256] write cursor of each coarse region (two-level partition)
    uint8_t* rec_tmp; // records grouped by coarse region (two-level partition)
    uint8_t* rec;     // records, grouped by bucket
    uint64_t rec_cap; // records that fit; more only when elem_ptr is invalid
    int32_t* status;
    uint64_t hist_words;  // length of hist (bounds-checked builds)
    bool chain;           // launched as a chain (launch_chained)
    bool after_kernel;    // the histogram pass directly follows a kernel of this build
};

struct BatchHeader;

struct OffsetsParams {
    uint32_t* hist;
    int n_cta;
    int64_t n_buckets;
    uint32_t* bstart;       // [n_buckets+1] first record of each bucket
    const uint32_t* nfc;    // [n_buckets] repeated-node records (nullptr: no element offsets)
    uint32_t* estart;       // [n_buckets+1] first element-CSR entry of each bucket (with nfc)
    uint32_t* gcur;         // [n_buckets] set to the bucket starts
    uint32_t* gcur_coarse;  // [256] set to the coarse region starts (when cshift > 0)
    int cshift;
    uint64_t* lb_state;     // lookback words, one per tile of buckets
    uint32_t* ticket;
    uint64_t rec_cap;       // bucket starts are clamped to the record array
    int32_t* status;
    const BatchHeader* hdr; // batches: the bucket count comes from the header
    bool chain;             // launched as a chain (launch_chained)
};

// ------------------------------------------------------------------ batches
// A batch is the disjoint union of many meshes built by one launch sequence.
// Its description lives in device memory (copied from host staging by the
// launch), so the same captured sequence serves any batch that fits the
// workspace capacity: header, then one BatchMesh per mesh, then the element,
// bucket and weight offsets of the meshes (n_meshes + 1 each).
struct BatchMesh {
    int32_t type;
    int32_t k;
    int64_t n_nodes, n_elems, n_conn;
    const int32_t* conn;
    const int64_t* elem_ptr;
    const uint8_t* elem_type;
    int64_t* rp_n; int32_t* col_n; int64_t cap_n;
    int64_t* rp_e; int32_t* col_e; int64_t cap_e;
    int32_t* status;
};

struct BatchHeader {
    RecFmt fmt;
    int32_t n_meshes;
    int64_t n_elems;    // elements of all meshes
    int64_t n_buckets;  // buckets of all meshes (each mesh starts a new bucket)
    int64_t n_records;  // record capacity (incidences of all meshes)
};

struct BatchTables {
    const BatchHeader* hdr;
    const BatchMesh* meshes;
    const int64_t* elem_off;    // [n_meshes+1]
    const int64_t* bucket_off;  // [n_meshes+1]
    const int64_t* weight_off;  // [n_meshes+1] incidences and elements of the meshes before
};

// A small mesh built without a partition: the connectivity that every CTA of
// the bucket pass reads (conn == nullptr: not a direct build).
struct DirectMesh {
    int type;
    int64_t n_nodes, n_elems, n_conn;
    const int32_t* conn;
    const int64_t* elem_ptr;
    const uint8_t* elem_type;
    uint32_t queue_off;  // dynamic shared memory before the queue of incidences
    uint32_t queue_cap;  // its entries
};

// Bucket pass: one CTA per bucket (persistent, buckets taken in order),
// builds the rows of the bucket's 2^sb nodes in groups of 32 (or of 2^sb,
// if fewer).
struct BucketParams {
    RecFmt fmt;
    int64_t n_nodes;
    int64_t n_buckets;
    const uint8_t* rec;
    const uint32_t* bstart;
    const uint32_t* estart; // element-CSR offset of each bucket, batch-wide (required when element rows are wanted)
    uint32_t* ticket;
    uint32_t* spill;        // global scratch for buckets too large for shared memory
    uint64_t spill_words;
    unsigned long long* spill_cursor;
    int64_t* rp_n; int32_t* col_n; int64_t cap_n;
    int64_t* rp_e; int32_t* col_e; int64_t cap_e;
    int32_t* status;
    uint32_t* ntmp;         // node rows of a group of 32 nodes at ntmp + k * its first record (k = neighbours per record)
    uint2* grp;             // [n_buckets * groups] each group's first record and node-row total
    uint32_t* nloc;         // [n_buckets << sb] each node's offset within its group's rows
    int32_t imax;           // 8, 16 or 32: the variant by its register arrays
    int32_t slots;          // places per node in the shared-memory table (<= imax)
    int32_t list_cap;       // records beyond their node's slots that a bucket may have
    uint32_t* rest;         // buckets that the first launch leaves to a second one (room for all)
    uint32_t* rest_count;   // ... how many
    uint32_t* rest_ticket;
    uint64_t rest_cap;      // words of rest
    BatchTables batch;      // batch.hdr != nullptr: format, bucket count and meshes come from the tables
    const int32_t* batch_err;  // batches: status of the shared offsets scan, copied to every mesh
    const int64_t* base;    // chunked builds: {element-CSR, node-CSR} entries of the earlier chunks (else nullptr)
    // buffer lengths, for bounds-checked builds
    uint64_t rec_count;     // records the record array holds
    uint64_t ntmp_words;    // words of ntmp
    uint64_t nloc_words;    // words of nloc
    uint64_t ngrp;          // entries of grp
    DirectMesh direct;      // single mesh, one bucket per CTA
    bool chain;             // launched as a chain (launch_chained)
};

// Shape of the bucket pass's second launch.
struct RestShape {
    int slots, list_cap, threads, grid;
    size_t smem;
};

constexpr int64_t CHAIN_RECORDS = 1 << 24;  // incidences up to which a build's kernels are launched as a chain
constexpr int EMIT_THREADS = 1024;
constexpr int PART_THREADS = 512;
constexpr int SORT_THREADS = 256;   // tile-sorted partition passes
constexpr int OFFSETS_THREADS = 128;  // buckets per tile of the offsets scan
constexpr int OFFSETS_SLICES = 8;     // slices of its histogram rows summed side by side
constexpr int SLOTS_MIN = 4;  // fewest slots of a node in the bucket pass
constexpr int NODE_SCAN_TILE = 512;  // groups of 32 nodes per tile of the node-row placement's scan

// groups up to which the placement adds up a group's predecessors itself (16
// loads a thread) instead of launching a scan
constexpr int64_t NODE_SUM_GROUPS = 4096;

// Placement of the node rows the bucket pass left in scratch (nn_compact.cu).
struct CompactParams {
    int64_t n_buckets;       // single mesh (batches: from the header)
    int64_t n_groups_cap;    // grid of the scan (batches: capacity)
    int sb, k;               // single mesh (batches: from the header; k = 3)
    int64_t n_nodes;
    const uint2* grp;        // [n_buckets * groups] first record and node-row total of each group of 32 nodes
    const uint32_t* nloc;
    const uint32_t* ntmp;
    uint64_t* nstart;        // [n_buckets * groups + 1] exclusive scan of the totals (batch-wide)
    uint64_t* lb_state;      // lookback words, one per tile of groups
    uint32_t* ticket;
    int64_t* rp_n; int32_t* col_n; int64_t cap_n;
    int32_t* status;
    BatchTables batch;
    const int64_t* base;     // chunked builds: {element-CSR, node-CSR} entries of the earlier chunks (else nullptr)
    // buffer lengths, for bounds-checked builds
    uint64_t ntmp_words;     // words of ntmp
    uint64_t nloc_words;     // words of nloc
    bool chain;              // launched as a chain (launch_chained)
};

// Element face adjacency (nn_adj.cu).
struct AdjParams {
    int type;
    int64_t n_nodes, n_elems, n_conn;
    const int32_t* conn;
    const int64_t* elem_ptr;
    const uint8_t* elem_type;
    const int64_t* ne_rp;    // node -> element CSR
    const int32_t* ne_col;
    uint32_t* cnt;           // [n_elems] neighbours per element
    int32_t* nbr;            // [n_elems][adjacency_slots] the element across each face, -1: none (nullptr: merge only)
    uint8_t* cplx;           // [n_elems] 1: slots do not tell all, merge the node rows (with nbr)
    uint64_t* lb_state;      // lookback words, one per tile of elements
    uint32_t* ticket;
    int64_t* rp; int32_t* col; int64_t cap;
    int32_t* status;
};

// launchers (return the CUDA error of the launch)
cudaError_t launch_adjacency(const AdjParams& p, int grid, int sms, cudaStream_t s);
int adjacency_slots(int type);
size_t adjacency_scan_tiles(int64_t n_elems);
// zeroes [p, p + bytes) (both multiples of 16) and the status word
cudaError_t launch_init(void* p, size_t bytes, int32_t* status, int sms, cudaStream_t s);
cudaError_t launch_node_compact(const CompactParams& p, int copy_grid, cudaStream_t s);
// chunked builds: base[0] += *etot, base[1] += *ntot (either may be nullptr)
cudaError_t launch_chunk_advance(int64_t* base, const uint32_t* etot, const uint64_t* ntot, cudaStream_t s);
// incidences per node slab of 2^shift nodes, added to counts[0 .. n_slabs) (n_slabs <= NN_CHUNK_SLABS_MAX)
cudaError_t launch_slab_count(const EmitParams& p, int shift, int n_slabs, uint32_t* counts, cudaStream_t s);
cudaError_t launch_hist(const EmitParams& p, size_t smem, cudaStream_t s);
cudaError_t launch_part(const EmitParams& p, cudaStream_t s);
// the tile-sorted partition's two passes (the fine one only when cshift > 0)
cudaError_t launch_part_coarse(const EmitParams& p, cudaStream_t s);
int coarse_ctas_per_sm(int type);
cudaError_t launch_part_fine(const EmitParams& p, const uint32_t* bstart, int sms, cudaStream_t s);
cudaError_t launch_offsets(const OffsetsParams& p, cudaStream_t s);
cudaError_t launch_bucket(const BucketParams& p, int grid, int threads, size_t smem, const RestShape& rest, cudaStream_t s);
// dynamic shared memory of the bucket kernel for buckets of 2^sb nodes
size_t bucket_smem_bytes(int sb, int want, int k, int slots, int rb, int list_cap);
cudaError_t bucket_occupancy(int* blocks, int threads, int imax, size_t smem);
cudaError_t launch_batch_emit(const BatchTables& bt, uint32_t* bcount, uint32_t* nfc, uint32_t* gcur, uint8_t* rec,
                              uint64_t* lb_off, uint32_t* ctrl, int grid, int stage, bool chain,
                              cudaStream_t s, uint64_t* lb_ns = nullptr);
int batch_ctas_per_sm();
cudaError_t set_emit_smem_all(size_t bytes);
cudaError_t set_bucket_smem_all(size_t bytes);
bool handle_offline(const nn_handle* h);  // a sizing-only handle (nn_create_offline)
nn_status build_with_limits(int sms, size_t smem_optin, size_t smem_per_sm, const nn_mesh* m, int want,
                            nn_csr* nodes, nn_csr* elems, void* ws, size_t ws_bytes, int32_t* d_status,
                            cudaStream_t s, size_t* ws_min);

}  // namespace nn
