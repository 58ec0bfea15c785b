// Device-resident inverted index (Alg. 1's I plus the all-pairs-1/2 per-vector data).
//
// Layout in HBM (N vectors over all instances, M = sum of instance dimension counts):
//   cptr[N+1]   row pointers (the caller's CSR row pointers, concatenated)
//   crank/cval  each row's components, re-ordered by dimension rank (rank local to the
//               instance; ranks sort dimensions by decreasing non-zero count)
//   len, mw, split, qsplit, mwpre [N]   |x|, maxweight(x), |x'| (unindexed prefix),
//               remscore boundary, maxweight(x') of the split
//   mwj[N]      maxweight of the join's prefix (below), where that reaches past the split
//   mwr/nnzr[M] maxweight_i(V) and non-zero count by global rank
//   lptr[M+1]   posting-list start by global rank
//   crow[nnz]   the same rows interleaved as {int32 rank, float32 value} (8 bytes)
//   The lists that the join walks keep more of a row unindexed than split does: the join's
//   prefix x' ends at the later of split and the first component where ||x'||_2 would reach
//   t (any y scores less than t on either kind of prefix), and the join's create boundary is
//   the later of the remscore boundary and that component. Both only with every bound on.
//   vmeta[N]    what the join reads of a query vector x, in one 16-byte load: {int32 row
//               offset, int32 |x|, int32 create boundary, float32 maxweight(x)}
//   vcand[N]    what verification reads of a candidate y, in one 16-byte load: {int32 row
//               offset, int32 |y'|, int32 first rank after y', float32 ||y'||_2 bound}
//   code[N]     one byte per vector: the octave of the first rank after y' in the high four
//               bits and ||y'||_2 rounded up to c * 1.01/15 in the low four. A query vector
//               turns the 256 codes into the least accumulated score worth verifying
//   post[]      posting entries {int32 local vector id | min(|y|, 255) << 24, float32
//               weight} (8 bytes), in increasing id inside each list; the size class in
//               the top byte lets minsize skip an entry without another load (instances
//               with n >= 2^24 store the id only and skip no entry)
//   wptr[]      position in post of each list's first entry of every candidate window (ids
//               [w*W, (w+1)*W)), only for instances with > 1 window; or, where that would be too
//               large, of groups of windows, as many as the list is long (wlist)
//   wlist[M]    then: where each list's starts begin in wptr << 6 | log2 of the windows of a group
#pragma once

#include <algorithm>
#include <atomic>
#include <mutex>

#include "aps_internal.cuh"

namespace aps {

constexpr int JOIN_WARPS = 24;  // warps of a join CTA (one CTA per SM)
constexpr int JOIN_THREADS = 32 * JOIN_WARPS;
// A join tile is one warp with a window of accumulator slots of its own in shared memory. The
// tile shape G (1, 2, 4 or 8) trades the warps that run on an SM against the window's width. The
// join waits for memory, so the most warps that the registers allow win at every size (join ms
// with 12 / 16 / 20 / 24 warps: 200k power-law set 27.1 / 22.0 / 20.6 / 21.0, the 512-instance
// batch 28.4 / 21.0 / 17.1 / 14.9; 28 and 32 warps spill registers and lose 5 to 30%), and G = 2,
// 4 and 8 are the same shape; G = 1 has windows of twice the width.

// Candidate list entries of a warp (join ms with 128 / 256 / 512: 30,000 power-law rows 2.25 / 1.75 /
// 1.69, 200,000 rows 23.5 / 21.6 / 22.5, the 512-instance batch 18.0 / 14.9 / 14.0, 4096 queries 6.64 /
// 6.60 / 6.92: a longer list takes its room from the window).
constexpr int JOIN_LCAP = 256;
constexpr int JOIN_SMEM = 232448 - 4096;  // of the 227 KB a CTA can have (the rest: the warps' states)
__host__ __device__ constexpr int tile_warps(int G) { return G == 1 ? 12 : 24; }
constexpr int JOIN_XCAP = 64;   // a query row of at most so many components is held in shared memory
// per-warp shared memory beside the window: 64 prefix norms, 32 lists waiting, 32 lists of a run,
// a query row, the candidate list
constexpr int TILE_FIXED = 4 * 64 + 16 * 32 + 8 * 32 + 8 * JOIN_XCAP + 2 * JOIN_LCAP;
// 4 bytes of accumulator and one bit of the match bitmap per slot; a multiple of 128 slots
__host__ __device__ constexpr int tile_window(int G) {
    return (JOIN_SMEM / tile_warps(G) - TILE_FIXED) * 8 / 33 / 128 * 128;
}
__host__ __device__ constexpr int tile_bytes(int G) { return TILE_FIXED + tile_window(G) * 33 / 8; }
// per-warp list of the matches of a streamed vector before they are placed
constexpr int JOIN_ECAP = 1408;
constexpr int JOIN_STAGE_SLAB = 512;  // staging slots a warp reserves at a time
constexpr int JOIN_NCLS = 5;          // work-list classes: tile shapes G = 1, 2, 4, 8; vectors of <= 2 components
// ||y'||_2 bounds in 4 bits: code c stands for c * PN4_STEP (above any norm the index accepts)
constexpr float PN4_STEP = 1.01f / 15.f;

// Buckets of dimension ranks: four per octave (64 in all; the last takes every rank from
// 114,688 on), and their octaves, used for the prefix norms of a query vector.
__device__ __forceinline__ int rank_bucket(int r) {
    const int e = max(31 - __clz(r), 2);
    return r < 4 ? r : min(4 * e + ((r >> (e - 2)) & 3) - 4, 63);
}

struct InstDesc {
    int64_t vbase;   // first global vector id
    int64_t wbase;   // first wptr entry (instances with nw > 1)
    int32_t n;       // vectors
    int32_t m;       // dimensions
    int32_t rbase;   // first global rank
    int32_t nw;      // candidate windows
    int32_t W;       // window width, at most tile_window(G)
    int32_t G;       // tile shape of this instance's class
    float t;         // threshold
    int32_t packed;  // 1: posting ids carry the size class in their top byte
};

// The first piece of the run of emitted pairs of one slot (a vector, or one part of its
// windows), stored at segs[slot]; the slot's pairs go to scan(counts)[slot] on. A run that
// fills its staging slab goes on at the start of another one: chain[k] = {pairs, next slab or
// -1} describes the piece at the start of slab k.
struct Segment {
    int64_t src;   // offset in the staging buffer
    int32_t cnt;   // pairs of this piece
    int32_t i;     // local id of x
    int32_t next;  // slab of the next piece, or -1
    int32_t _pad;
};

// Windows of a set of few vectors are halved, at most WINDOW_HALVINGS times, until there are
// WINDOWS_LEAST of them, which are then cut into parts for a heavy vector (a row of 2,000 components is
// otherwise one warp's work), and once more where rows are uneven, the longest more than eight times
// the mean. Kernel ms with windows of 1792 / 896 / 448 / 224 ids: 2,000 power-law rows (t = 0.5) 0.56 /
// 0.64 / 0.22 / 0.19, 5,000 (t = 0.3) 1.53 / 0.44 / 0.36 / 0.45, 20,000 1.62 / 1.59 / 1.77 / 2.2, 200,000
// 21.7 / 34.9 / 62.7 / 99; even rows of 100, 8,000 of them, 0.91 / 0.83 / 0.86 / 0.90. (Calls between:
// 14,000 power-law rows take 1.19 and 1.01 ms at two widths of dimensions, 1.13 and 1.05 with 896.)
constexpr int WINDOW_HALVINGS = 3, WINDOWS_LEAST = 4;

// The table of window starts. With every window of every list it takes n * m / 448 bytes, whatever
// the lists hold, so a wide sparse set's would outgrow the rest of its index (ten million rows of
// a million dimensions: 22 GB). It is that table up to about what the index's other arrays take (24
// bytes a component, 28 a dimension); past that each list has the starts of as many groups of
// 2^shift windows as there is room for, WLIST_ENTRIES for each of its entries, and the join searches
// the group. Long lists, which are most of the work, thus keep every window, and a short
// list's groups hold one entry or none. Two million rows of ten components over a million
// dimensions: 0.63 GB and 105 ms in the join's kernel, 5.0 GB and 158 ms with every window. Where
// most lists are long, every window is the better one: by list the 200,000-row power-law set takes
// 28.1 ms a call (25.3), 4096 queries of a million rows 8.2 (7.0), a batch of 512 instances 45.9 (43.4).
constexpr int WLIST_ENTRIES = 8;
inline int64_t window_bytes(int64_t nnz, int64_t M) { return 4 * WLIST_ENTRIES * nnz + 16 * M; }

__host__ __device__ constexpr int window_groups(int nw, int shift) {
    return (int)(((int64_t)nw + ((int64_t)1 << shift) - 1) >> shift);
}

// The least shift with at most per * len groups, or one: the list is then searched as a whole.
__host__ __device__ inline int list_shift(int64_t len, int nw, int per) {
    int s = 0;
    while (window_groups(nw, s) > 1 && window_groups(nw, s) > per * len) s++;
    return s;
}

struct IndexArrays {
    DBuf<char> block;  // the arrays of known size, from inst to code
    DBuf<InstDesc> inst;
    DBuf<int32_t> vinst;  // instance of each vector
    DBuf<int64_t> cptr;
    DBuf<int32_t> crank;
    DBuf<float> cval;
    DBuf<int2> crow;
    DBuf<int4> vmeta;
    DBuf<int4> vcand;
    DBuf<uint8_t> code;
    DBuf<int32_t> len, split, qsplit;
    DBuf<float> mw, mwpre, mwj;
    DBuf<int32_t> rank_of_dim, dim_of_rank, nnz_d;
    DBuf<float> mw_d, mwr;
    DBuf<int64_t> lptr;
    DBuf<uint32_t> wptr;
    DBuf<uint64_t> wlist;
    DBuf<int2> post;
};

// The join phase of an index as a CUDA graph: the two workspace resets and the persistent
// join launch, captured on the index's second join; later joins update the nodes' pointers
// and launch parameters in the instantiated graph and replay it.
struct JoinGraph {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaGraphNode_t reset_ctr = nullptr, reset_cnt = nullptr, join = nullptr;
    int64_t launches = 0;
    JoinGraph() = default;
    JoinGraph(const JoinGraph &) = delete;
    JoinGraph &operator=(const JoinGraph &) = delete;
    ~JoinGraph() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
    }
};

}  // namespace aps

struct aps_index {
    int device = 0;
    cudaStream_t stream = nullptr;
    uint32_t flags = 0;
    int32_t k = 0;     // instances
    int64_t N = 0;     // vectors
    int64_t M = 0;     // dimensions (all instances)
    int64_t nnz = 0;
    int64_t nsuf = 0;   // indexed components (by split)
    int64_t njoin = 0;  // components in the join's posting lists
    bool l2 = false;    // the join's prefixes take the norm bound too
    int64_t arena_slots = 0;  // what the allocation-free join's documented size limit counts
    int64_t nwptr = 0;
    int wper = -1;      // starts stored for each entry of a list at most (-1: those of every window)
    int32_t maxm = 0, maxnw = 0;
    // parts that the windows of a heavy vector are cut into (its slots; 1: none)
    int32_t parts = 1;
    float t = 0.f;     // single-instance threshold
    std::vector<aps::InstDesc> inst_h;
    aps::IndexArrays d;
    // join work list: vectors in decreasing estimated cost, grouped by class
    aps::DBuf<int32_t> items;
    int64_t class_begin[aps::JOIN_NCLS + 1] = {};  // tile shapes G = 1, 2, 4, 8, then vectors of <= 2 components
    // output sizing from the previous join
    int64_t hint_pairs = 0;
    // pairs per query (times 16) that query batches on this index have needed at most: the
    // first staging of the next batch is sized from it, so that it rarely runs twice
    mutable std::atomic<int64_t> q_ppq16{64 * 16};
    aps::JoinGraph jgraph;  // the join phase, replayed by every join of this index
    aps_stats stats{};
    mutable std::mutex stats_mu;  // queries may run concurrently (serving slots)
};

namespace aps {

struct PairsAlloc {          // bookkeeping behind aps_pairs._priv
    void *block = nullptr;   // one allocation holding i, j and score
    size_t bytes = 0;        // its size (host blocks go back to the pinned cache)
    cudaStream_t stream = nullptr;
    int on_device = 1;
    int refs = 1;            // aps_pairs views sharing the block (batched results)
};

void pairs_release(aps_pairs *p);
// Copy a result's arrays to the caller's (host or device, any may be null) and wait.
aps_status pairs_copy(const aps_pairs *p, int32_t *i, int32_t *j, float *score, cudaStream_t s);
// Replace device pairs by one pinned host copy.
aps_status pairs_to_host(aps_pairs *p, cudaStream_t s);

// External query rows prepared against an index: components re-expressed over the index's
// dimension ranks and sorted by rank, with |q|, maxweight(q) and the remscore boundary.
struct QueryArrays {
    DBuf<int2> crow;     // {rank, value} per component, rows in rank order
    DBuf<int4> vmeta;  // {row offset, |q|, create boundary, maxweight(q)}
    DBuf<float> mw;
    int64_t nq = 0, nnz = 0;
};

// nnz_known: the number of components when the caller knows it from host row pointers
// (qptr[0] = 0 checked there), else -1 (both ends are then read back from the device).
aps_status prepare_queries(const aps_index *ix, const int64_t *qptr, const int32_t *qidx, const float *qval,
                           int32_t nq, float t, uint32_t flags, cudaStream_t s, QueryArrays &qa,
                           int64_t nnz_known = -1);

// The windows of a query are cut into as many parts (its slots) as give every warp of the chip some
// 32 units.
inline int query_parts(const aps_index *ix, int64_t nq) {
    const InstDesc &I = ix->inst_h[0];
    const int64_t n = std::max<int64_t>(nq, 1);
    return (int)std::max<int64_t>(1, std::min<int64_t>(I.nw, ((int64_t)num_sms() * tile_warps(I.G) * 32 + n - 1) / n));
}
constexpr int64_t QUERY_SLAB = 256;  // staging slots a warp reserves at a time: query batches are small
inline int query_ctas(const aps_index *ix, int64_t nq) {
    return (int)std::min<int64_t>(num_sms(), std::max<int64_t>(ix->inst_h[0].nw > 0 ? nq * query_parts(ix, nq) : 0, 1));
}
// Staging of a batch: the pairs per query that this index's batches have needed so far (at least
// 64), plus one slab per warp.
inline int64_t query_stage(const aps_index *ix, int64_t nq) {
    const int64_t slack = (int64_t)query_ctas(ix, nq) * JOIN_WARPS * QUERY_SLAB;
    return std::max<int64_t>(nq * ix->q_ppq16.load(std::memory_order_relaxed) / 16 + slack, (int64_t)1 << 16);
}
// Device bytes that a batch holds while it runs, at most (unless it has more pairs a query than any
// before): its rows as they came, checked, keyed, sorted (two copies and the sort's tile states) and
// packed, 60 bytes a component; row pointers, lengths, maxima and descriptions, 48 a query; count,
// offset and run of every slot; the staged pairs with their slabs' chain, and the final ones.
inline size_t query_bytes(const aps_index *ix, int64_t nq, int64_t nnz) {
    const size_t slots = (size_t)nq * (size_t)query_parts(ix, nq), stage = (size_t)query_stage(ix, nq);
    return ((size_t)1 << 20) + 60 * (size_t)nnz + 48 * (size_t)nq + slots * (4 + 8 + sizeof(Segment)) +
           stage * sizeof(int2) + stage / QUERY_SLAB * sizeof(int2) + stage * 12;
}

// Match prepared queries against every indexed vector: pairs (query row, vector id, score)
// with score >= t, sorted by (query, vector). Safe to call concurrently on different
// streams (it does not modify the index).
aps_status join_queries(const aps_index *ix, const QueryArrays &qa, float t, uint32_t flags, cudaStream_t s,
                        aps_pairs *out, aps_stats *stats);

// Build all index arrays for the instances whose CSRs are concatenated in (indptr, idx,
// val) with global row pointers (indptr[0] = 0). Inputs are device pointers.
aps_status build_index_device(aps_index *ix, const int64_t *indptr, const int32_t *idx,
                              const float *val, const std::vector<InstDesc> &inst_in,
                              cudaStream_t s, const aps_tuning *tune = nullptr);

// The posting lists by split (the exported ones), where they are not the join's own.
aps_status export_postings(const aps_index *ix, DBuf<int64_t> &lptr, DBuf<int2> &post, cudaStream_t s);
// What the dimension-block items of a split join walk and check instead of the join's own arrays:
// lists and prefixes up to the split alone. A block's share of the score has to stand against the
// norm of y's whole prefix (Lemma 1), and the norm-bounded prefixes reach almost to t: with them
// 2,000 heavy vectors of 200,000 in two blocks kept so many candidates that the join took 148 ms;
// 33 with these (43 in the kernel before).
struct BlockIndex {
    DBuf<int4> vmeta, vcand;
    DBuf<uint8_t> code;
    DBuf<int64_t> lptr;
    DBuf<uint32_t> wptr;
    DBuf<uint64_t> wlist;
    DBuf<int2> post;
};
aps_status build_block_index(const aps_index *ix, BlockIndex &b, cudaStream_t s);

// Join tile shapes (tune.cu): the size bucket of an instance, the process-wide table of
// query groups per bucket, and the autotuner (host arrays ro, hptr, m, t; device CSR).
int tune_bucket(int64_t n);
aps_tuning tuning_default();
aps_tuning tuning_current();
bool tuning_valid(const aps_tuning &tu);
void tuning_set(const aps_tuning &tu);
aps_status autotune_batch(int32_t k, const int64_t *ro, const int64_t *hptr, const int64_t *dp, const int32_t *di,
                          const float *dv, const int32_t *m, const float *t, uint32_t flags, cudaStream_t s,
                          aps_tuning *out, aps_tune_report *rep);

// Self-join of every instance of the index; fills a device aps_pairs (i, j, score)
// with per-instance ranges in pair_offsets_h (k+1 entries, may be null).
// nblk >= 2 and heavy > 0 (single-instance indexes): the vertical split with local pruning
// for the `heavy` costliest vectors, joined as nblk dimension blocks each (Sec. 5.1, Lemma 1).
aps_status join_all_pairs(aps_index *ix, uint32_t flags, aps_pairs *out,
                          std::vector<int64_t> *pair_offsets_h, int nblk = 0, int64_t heavy = 0);

// The self-join of a single-instance index with every buffer carved out of `arena`
// (arena_bytes, 256-byte aligned) and at most max_ctas CTAs; pairs land in the caller's
// arrays (capacity cap). *count receives the number of pairs, also on APS_EOVERFLOW.
aps_status join_noalloc(aps_index *ix, unsigned char *arena, size_t arena_bytes, int max_ctas, int32_t *oi,
                        int32_t *oj, float *os, int64_t cap, int64_t *count, cudaStream_t s, int parts = -1);

// Dense all-pairs of X[n, d] (float32 rows; host or device per APS_DEVICE_PTRS) on the
// tensor cores with exact rescoring; d % 64 == 0, 64 <= d <= 512.
aps_status dense_all_pairs(const float *X, int32_t n, int32_t d, float t, uint32_t flags, cudaStream_t s,
                           aps_pairs *out, aps_stats *stats);
// The BF16 rows (zero rows up to the padded count) that the validation of X has already made, and
// when it began.
struct DenseRows {
    void *xb = nullptr;
    cudaEvent_t began = nullptr;
    DenseRows() = default;
    DenseRows(const DenseRows &) = delete;
    DenseRows &operator=(const DenseRows &) = delete;
    ~DenseRows() {
        if (began) cudaEventDestroy(began);
    }
};
aps_status dense_all_pairs_device(const float *X, int32_t n, int32_t d, float t, cudaStream_t s, aps_pairs *out,
                                  aps_stats *stats, float *raw, const DenseRows *rows);
// The tensor cores' float32 products X_bf16 . X_bf16^T of the computed (upper) blocks into
// raw (row-major n x n, device memory); X on the device.
aps_status dense_tensor_products(const float *X, int32_t n, int32_t d, cudaStream_t s, float *raw);
double dense_margin(int d);
void dense_debug_stall(int64_t launches, uint64_t wait_ns);
void debug_stage_cap(int64_t pairs);

// The similarity graph G_S as a CSR adjacency from a pair list, its k nearest neighbours,
// and its release (graph.cu).
aps_status graph_csr(const int32_t *i, const int32_t *j, const float *s, int64_t count, int32_t n, uint32_t flags,
                     cudaStream_t st, aps_graph *out);
aps_status graph_knn(const aps_graph *g, int32_t k, int32_t *nbr, float *wk, uint32_t flags, cudaStream_t s);
void graph_release(aps_graph *g);

// Union of candidate pair lists, exact float64 rescoring from the rows, pairs >= t (verify.cu).
aps_status pairs_verify(const aps_pairs *lists, int32_t k, const int64_t *indptr, const int32_t *idx,
                        const float *val, int32_t n, int32_t m, float t, cudaStream_t s, aps_pairs *out,
                        int64_t *n_candidates);

}  // namespace aps
