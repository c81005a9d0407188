// Internal declarations shared by libmce's translation units (host launchers
// and kernels).  Not part of the public ABI (that is include/mce.h).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "mce.h"

namespace mce {

// Words of a work frame before its P and X bitsets:
//   [0] pivot | end << 16   (branching set L = P & ~N(pivot) & [0, end))
//   [1] |R|
//   [2] S(R) low word, [3] S(R) high word   (running clique hash sum)
//   [4] graph slot (batched and served forms), [5..7] unused
// and, when cliques are listed, the bitset R after P and X.
constexpr int kFrameHdr = 8;

// Levels of the per-group explicit stack (local memory).  Deeper paths spill
// their frames to the global work queue, so this bounds nothing but
// register/local footprint.
constexpr int kStackDepth = 64;

// Global control block of one search, each counter on its own 128-byte line.
struct Ctl {
    unsigned head;     unsigned pad0[31];  // global queue consumer ticket
    unsigned tail;     unsigned pad1[31];  // global queue producer ticket
    unsigned pending;  unsigned pad2[31];  // frames in the global ring + active blocks
    unsigned starving; unsigned pad3[31];  // warps without a frame; pad3[0]: the degree sum
    unsigned abort;    unsigned pad4[31];  // set on error: every warp stops
};

// Per-block frame ring in shared memory (the first level of the work
// distribution): header, kLocalSlots sequence numbers and as many frames.
constexpr uint32_t kLocalSlots = 32;
struct LocalHdr {
    unsigned head, tail;  // ring tickets
    unsigned idle;        // warps of this block without a frame
    unsigned bwork;       // busy warps + frames in the ring; the block holds
                          // one unit of Ctl::pending while this is non-zero
    unsigned poller;      // a warp of this block is polling the global ring
    unsigned done;        // the search is over (1) or aborted (2)
    unsigned refreshing;  // a warp is refreshing the cached global state
    // cached global state (refreshed every few microseconds)
    unsigned g_head, g_tail, g_starving;
    unsigned long long stamp;
    unsigned trace_n;     // timeline records written by this block
    unsigned give_p;      // warp tier: smallest |P| of a frame that is given away
    // the device-wide ring and the frame shape, for frames given away by the
    // warp tier
    Ctl *ctl;
    unsigned *gseq;
    uint32_t *gframes;
    unsigned qcap, fs, margin, wp, n;
    unsigned give_mask, total;
    // work-distribution diagnostics of the block (rare events, shared-memory
    // atomics; added to the result array once the block is done)
    unsigned long long diag[8];
};
// Indices of LocalHdr::diag and the result words they are added to.
enum DiagIdx { kDiagDonations = 0, kDiagSteals, kDiagGlobal, kDiagBusyNs, kDiagGpush, kDiagGtry, kDiagCasFail,
               kDiagLaneTasks, kDiagCount };
__host__ __device__ inline size_t frame_words(uint32_t wp, bool list = false)
{
    return (8 + (list ? 3 : 2) * (size_t)wp + 3) / 4 * 4;
}
__host__ __device__ inline size_t local_queue_bytes(uint32_t wp, bool list = false)
{
    return sizeof(LocalHdr) + (size_t)kLocalSlots * 4 + (size_t)kLocalSlots * frame_words(wp, list) * 4;
}

// Clique listing (MCE_LIST).  Every group appends, at each maximal clique it
// reports, a record [0x80000000 | k, pos_1 .. pos_k] (positions in the search
// order) to a chunk of the record buffer it claimed; the clique's members are
// the R of the frame the group last took (its bitset in `base`, its size
// `rsb`) plus the vertices the group added on its way down (`path`, indexed
// by |R|), plus the leaf vertex.  Frames that move between groups carry R.
struct ListParams {
    uint32_t *rec;          // n_chunks * chunk_words words; null: no listing
    uint32_t *fill;         // words used in each chunk (zeroed before the search)
    unsigned *next_chunk;   // chunk claim counter (zeroed)
    unsigned *overflow;     // set when a record found no chunk (zeroed)
    uint16_t *path;         // total_groups * n entries
    uint32_t *base;         // total_groups * wp words
    uint32_t n_chunks, chunk_words;
};

// Work-distribution knobs (defaults in default_tuning(); MCE_TUNE overrides).
struct Tuning {
    uint32_t share_local;   // smallest |P| given to the block ring (0: by density)
    uint32_t share_global;  // smallest |P| given to the device-wide ring (0: by density)
    uint32_t local_check;   // busy warps: iterations between block-ring checks (a power of two)
    uint32_t global_check;  // busy warps: iterations between global checks (a power of two)
    uint32_t refresh_ns;    // age of a block's cached view of the global ring
    uint32_t serve_cpb;     // served form: expected maximal cliques per block
    uint32_t pop_tries;     // ticket attempts of one take from the device-wide ring
    uint32_t idle_sleep_ns; // longest back-off of an idle warp that is not polling
    uint32_t t2_p;          // warp tier: largest |P| of a subproblem (0: off, at most kPoolMaxP)
    uint32_t batch_split;   // batched form: parts of about 1/(blocks * batch_split) of a bucket's cost (0: no split)
    uint32_t serve_bcost;   // served form: largest expected maximal cliques (thousands) of a micro-batched request
    uint32_t t2_task;       // largest |P u X| of a subproblem (0: by density and size)
    uint32_t t2_cls;        // words per set of a subproblem (0: by density and size)
    uint32_t give_p;        // smallest |P| a warp tier gives away (0: by density)
    uint32_t give_steps;    // warp tier: steps between looks for idle warps (a power of two)
};

// The warp tier (second search tier): a frame whose P u X has at most 128
// vertices is relabelled 0..u-1 in order and searched by its whole warp, each
// lane expanding a node per step.  Per warp in shared memory: the local
// adjacency rows (u rows of ceil(u/32) words; several small subproblems side
// by side), the hash terms of the local vertices, a buffer of leaves, and the
// stack of frames the 32 lanes share.
constexpr int kPoolLeafBytes = 63 * 12 + 12;  // 31 leaves waiting and 32 new ones, three words each
constexpr int kPoolFixedBytes = 5456;   // the most that precedes a stack in the region
constexpr int kPoolMaxP = 128;          // largest |P| of a subproblem
// A warp's region: at least 64 frames of any set size (a stack that is paged
// out at fewer than 32 free frames must hold 32 to page), at most about 256 of
// four words.
constexpr uint32_t kPoolBytesMin = 7248, kPoolBytesMax = 15360, kPoolBytesShort = 9216;

// Graphs of at most 128 vertices: the whole graph in the warp tier's layout,
// once per block (rows, hash terms, positions).
constexpr int kDirectRows = 512, kDirectVerts = 128;
constexpr uint32_t kDirectBytes = kDirectRows * 4 + kDirectVerts * 10;

// Most threads of a search block (the register bound of the kernels).  The
// single-graph search and the batch kernel are compiled for 768 threads (80
// registers: the warp tier's loop fits, the search by frames above it spills
// 200 words) and for 512 (128 registers, nothing spilled).  Most searches spend
// enough of their time above the warp tier for the latter, ms with 768 / 512
// threads: G(100, 0.5) 0.150 / 0.135, G(250, 0.4) 0.31 / 0.23, G(700, 0.18) 0.53 /
// 0.46, G(1000, 0.3) 3.2 / 2.9, G(3000, 0.1) 3.0 / 2.6.  A long search is nearly
// all warp tier and wants the warps: G(500, 0.5) 9.6 / 10.3, G(100, 0.9) 16.1 /
// 18.4.  (576 and 608 threads: slower than the better of the two everywhere.)
constexpr unsigned kLaunchThreads = 768u, kShortThreads = 512u;

// Longest run of a search: ten times its wait budget (the largest value, no
// limit, where that does not fit).
inline uint64_t total_limit(uint64_t timeout_ns)
{
    return timeout_ns > UINT64_MAX / 10u ? UINT64_MAX : 10u * timeout_ns;
}

struct SearchParams {
    uint32_t n;             // vertices
    uint32_t wp;            // words per renumbered row (= lanes * words/lane)
    const uint32_t *rows;   // renumbered rows, n * wp words (+ pad to 16 B)
    const uint32_t *order;  // position -> original label
    Ctl *ctl;
    unsigned *seq;          // queue slot sequence numbers (qcap entries)
    uint32_t *frames;       // qcap frames of fs words
    uint32_t qcap;          // power of two
    uint32_t fs;            // frame stride in words
    uint64_t *out;          // MCE_OUT_WORDS(n) words
    uint64_t timeout_ns;    // longest time without progress
    uint64_t limit_ns;      // longest time in all (total_limit)
    uint32_t total_groups;
    uint32_t pivot_mode;
    uint32_t stack_levels;  // <= kStackDepth
    uint32_t split_min_p;   // publish new subtrees with |P| >= this ...
    uint32_t split_target;  // ... while the global ring holds fewer frames
    unsigned long long *trace;   // optional timeline (2 words per record)
    uint32_t trace_per_block;    // records per block
    Tuning tune;
    ListParams lst;              // clique listing (lst.rec null: off)
    // A part of the root's branching (the root's children are independent
    // subtrees): part (device, part_k entries, strictly increasing) lists
    // the children searched; null searches the whole tree.  The root node is
    // counted only with count_root.
    const uint32_t *part;
    uint32_t part_k;
    uint32_t count_root;
    // warp tier: byte offset of its shared memory, the bytes of a warp's region
    // (a multiple of 16) and the largest |P| of a subproblem (0: the tier is off)
    uint32_t t2_offset, pool_bytes, t2_max_p;
    uint32_t direct_offset;  // byte offset of the whole-graph layout (n <= 128)
    uint32_t prepared;      // result array, queue and root frames are in place: the search alone is launched
};

// One graph of a batch (device table entry; pointers into library memory).
struct BatchGraph {
    const uint32_t *rows;   // validated input bitset, w words per row
    uint32_t *order;        // n entries
    uint32_t *ren;          // n * wp renumbered words (+ pad to 16 B)
    uint64_t *out;          // MCE_OUT_WORDS(n) words
    uint32_t n, w, wp;
    uint32_t per;           // root children per queued frame (at least 1)
    // Subproblem of the outer loop (Alg. 3), else null / 0: label[i] is the
    // original label of local vertex i (hashes and sizes use it); root holds
    // the root's P then X as bitsets over local vertices (w words each); the
    // root's R is {rv} (a local vertex, adjacent to every other one).
    const uint32_t *label;
    const uint32_t *root;
    uint32_t rv, pad2;
};

// Outer loop of Alg. 3 (outer.cu).  CSR adjacency on the device: off[n + 1],
// adj[off[n]] with every list sorted.
cudaError_t outer_csr_from_edges_bytes(uint32_t n, uint64_t m, size_t *temp_bytes);
// Builds the CSR of the simple graph given by m edges (u, v) (duplicates and
// both orientations allowed); out[MCE_OUT_STATUS] = MCE_EINVAL on a self-loop
// or an id >= n; *adj_count (device) receives off[n].
cudaError_t outer_csr_from_edges(uint32_t n, uint64_t m, const uint32_t *d_uv, void *temp, size_t temp_bytes,
                                 uint32_t *off, uint32_t *adj, uint64_t *out, cudaStream_t s);
// CSR of an n x w bitset (off: n + 1 entries; adj: off[n] entries).
cudaError_t outer_csr_from_rows(uint32_t n, uint32_t w, const uint32_t *rows, uint32_t *off, uint32_t *adj,
                                void *temp, size_t temp_bytes, size_t *need, cudaStream_t s);
// Degeneracy order (minimum remaining degree first, smallest label on ties):
// order[i] = vertex i, pos[v] = its position.  One block; n <= 65535 and
// every degree < 4096; off/adj a symmetric adjacency of `entries` neighbours in all.
cudaError_t outer_degeneracy(uint32_t n, uint64_t entries, const uint32_t *off, const uint32_t *adj, uint32_t *order,
                             uint32_t *pos, cudaStream_t s);
// Fill every subproblem's rows, labels, root sets and table[i].rv (one block
// each): subproblem i is vertex order[i] with its neighbourhood.
cudaError_t outer_extract(const BatchGraph *table, uint32_t count, uint32_t max_w, const uint32_t *order,
                          const uint32_t *pos, const uint32_t *off, const uint32_t *adj, cudaStream_t s);
// Sum the subproblems' results into out (MCE_OUT_WORDS(n) words, zeroed).
cudaError_t outer_reduce(const BatchGraph *table, uint32_t count, uint32_t n, uint64_t *out, cudaStream_t s);

// Most words per row of a batched graph that the batch kernel splits into
// root-child parts (its shared prefix table).
constexpr int kBatchPartWords = 128;

struct BatchParams {
    const BatchGraph *graphs;
    const uint32_t *list;   // graph indices of this bucket, most expensive first
    uint32_t count;         // entries of list
    unsigned *next;         // claim counter (zeroed before the launch)
    unsigned char *qbase;   // per-block queue regions
    size_t qstride;         // bytes per region
    uint32_t qcap, fs;      // slots per region, frame stride (words)
    uint32_t root_frames;   // frames of a whole graph's root children, at most
    uint64_t timeout_ns, limit_ns;
    uint32_t pivot_mode, stack_levels, groups_per_block;
    uint32_t split_min_p, split_target;
    Tuning tune;
    uint32_t t2_offset, pool_bytes, t2_max_p, direct_offset;  // warp tier (as in SearchParams)
    uint32_t cls;            // words per set of the warp tier, for all graphs of the bucket
};

// Per-block queue region of the batched search: [Ctl | seq | frames]
__host__ __device__ inline size_t batch_seq_offset() { return 1024; }
__host__ __device__ inline size_t batch_frames_offset(uint32_t qcap) { return 1024 + (((size_t)qcap * 4 + 255) / 256) * 256; }
__host__ __device__ inline size_t batch_region_bytes(uint32_t qcap, uint32_t fs)
{
    return batch_frames_offset(qcap) + (((size_t)qcap * fs * 4 + 255) / 256) * 256;
}

struct LaunchShape {
    unsigned blocks, threads;
    size_t smem;
};

// One search: init kernel (root frame, queue, zeroed output) + persistent
// search kernel, and its occupancy query.  Defined per words of a lane in
// search_kN.cu and search_list_kN.cu.
struct SearchImpl {
    cudaError_t (*run)(const SearchParams &, const LaunchShape &, cudaStream_t);
    cudaError_t (*occupancy)(int threads, size_t smem, int *blocks_per_sm);
    // batched form: one graph per block at a time (kernel attributes are set
    // by batch_occupancy, so run_batch is safe inside a stream capture)
    cudaError_t (*run_batch)(const BatchParams &, const LaunchShape &, cudaStream_t);
    cudaError_t (*batch_occupancy)(int threads, size_t smem, int *blocks_per_sm);
};
SearchImpl search_impl_1(int pivot);
SearchImpl search_impl_2(int pivot);
SearchImpl search_impl_4(int pivot);
// Listing variants (run/occupancy only; no batched form).
SearchImpl search_list_impl_1(int pivot);
SearchImpl search_list_impl_2(int pivot);
SearchImpl search_list_impl_4(int pivot);

// The root's children as independent subtrees (split.cu).  The root's
// branching set is L = V \ N(p0) (p0 = root_pivot, or position 0 when null)
// over the renumbered rows; child t branches on its t-th vertex v_t with
// v_1..v_{t-1} moved from P to X.
// sizes[t] = |P_t n N(v_t)|, P_t = V minus v_1..v_{t-1}, for t < cap;
// *count = |L| (device words).
cudaError_t launch_root_children(const uint32_t *rows, uint32_t n, uint32_t wp, const unsigned *root_pivot,
                                 uint32_t *sizes, uint32_t cap, uint32_t *count, cudaStream_t s);
// Queue frame j (< prm.part_k) = child prm.part[j] (after search_init_kernel
// reserved the slots); an index beyond |L| or out of order sets MCE_EINVAL.
cudaError_t launch_part_frames(const SearchParams &prm, const unsigned *root_pivot, cudaStream_t s);
// Queue every root child as its own frame (after search_init_kernel left the
// queue empty): frame t in slot t, tail = pending = |L|.  prm.qcap >= n.
cudaError_t launch_seed_children(const SearchParams &prm, const unsigned *root_pivot, cudaStream_t s);
// Everything before the search (see small_prep_kernel), for graphs and rows
// that small_prep_fits accepts: order and rows receive the order and the
// renumbered rows.
bool small_prep_fits(uint32_t n, uint32_t w, uint32_t wp);
cudaError_t launch_small_prep(const SearchParams &prm, uint32_t w, const uint32_t *rows_in, uint32_t *order,
                              uint32_t *rows, cudaStream_t s);
// TomitaBB's root pivot (the earliest vertex of maximum degree) to *dst.
cudaError_t launch_root_degree_pivot(const uint32_t *rows, uint32_t n, uint32_t wp, unsigned *dst, cudaStream_t s);

// Preprocessing kernels (prep.cu).
cudaError_t launch_edges_to_rows(uint32_t n, uint64_t m, const uint32_t *uv, uint32_t w,
                                 uint32_t *rows, uint64_t *out, cudaStream_t s);
cudaError_t launch_validate_rows(uint32_t n, uint32_t w, const uint32_t *rows, uint64_t *out,
                                 cudaStream_t s);
cudaError_t launch_order(uint32_t n, uint32_t w, const uint32_t *rows, uint32_t *order,
                         cudaStream_t s);
cudaError_t launch_identity(uint32_t n, uint32_t *order, cudaStream_t s);
cudaError_t launch_renumber(uint32_t n, uint32_t w, const uint32_t *rows, const uint32_t *order,
                            uint32_t wout, uint32_t *rows_out, cudaStream_t s);
// Batched preprocessing over a device table of graphs (max_n / max_w / max_wp
// bound every entry).  prepare_* sets kernel attributes (call before capture).
cudaError_t prepare_order_batch(uint32_t max_n, uint32_t max_w, size_t *smem);
cudaError_t launch_order_batch(const BatchGraph *graphs, uint32_t count, size_t smem, cudaStream_t s);
cudaError_t launch_renumber_batch(const BatchGraph *graphs, uint32_t count, uint32_t max_n, uint32_t max_wp,
                                  cudaStream_t s);

inline size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Raise a kernel's dynamic shared-memory limit to the device maximum and
// prefer the largest shared-memory carveout, once per (kernel, device): kernels
// that ask for the same carveout run beside one another without a change of it.
// prefer_l1 (the single-graph search of up to 512 threads): the carveout is
// left to the driver, and the rows stay in L1 where the blocks leave room
// (listing G(700, 0.3) 4.5 -> 4.1 ms, counting G(1000, 0.3) 3.11 -> 2.91).  Served
// requests searched alone then run beside micro-batches of another carveout;
// the largest for both was slower all the same (24 to 256 requests: 0.97x).
cudaError_t kernel_smem_setup(const void *func, bool prefer_l1 = false);

// Listing post-pass (listing.cu): record chunks of a finished listing search
// -> CSR listing (off[count + 1], ids) in original labels, each clique in
// ascending order and, when `sorted`, the cliques in lexicographic order.
struct ListJob {
    const uint32_t *rec, *fill;  // record buffer and per-chunk fill (search output)
    uint32_t chunks, chunk_words;  // chunks claimed (<= n_chunks), chunk size
    const uint32_t *order;       // position -> original label
    uint32_t n, max_size;
    uint64_t count, ids;         // cliques and member ids (from the histogram)
    uint32_t *ids_out;           // device, ids entries
    uint64_t *off_out;           // device, count + 1 entries
    bool sorted;
    void *temp;                  // list_temp_bytes(count, ids, chunks, sorted) bytes
    size_t temp_bytes;
};
size_t list_temp_bytes(uint64_t count, uint64_t ids, uint32_t chunks, bool sorted);
cudaError_t list_build(const ListJob &j, cudaStream_t s);

// Tuning in effect for this process: defaults, overridden once from the
// environment variable MCE_TUNE="key=value,..." (keys as in Tuning).
Tuning default_tuning();

// Shared-memory layout of the search kernels:
//   [hist: (n + 1) x u32, padded to 16 B][local frame ring]
//   [whole-graph layout (n <= 128)][warp regions]
__host__ __device__ inline size_t smem_local_offset(uint32_t n) { return (((size_t)n + 1) * 4 + 15) / 16 * 16; }
__host__ __device__ inline size_t search_smem_bytes(uint32_t n, uint32_t wp, bool list = false)
{
    return smem_local_offset(n) + local_queue_bytes(wp, list);
}
}  // namespace mce
