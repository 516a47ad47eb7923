// kh_internal.cuh -- internal declarations of the (k,h)-core CUDA library.
//
// Device data layout of one graph (all arrays in HBM, owned by kh_graph):
//   rowptr   int64[n+1], col int32[nnz]      symmetric CSR, rows sorted
//   rank     uint8[n]                          r[v] (Sec. 3)
//   alive    uint8[n]                          1 alive, 2 removed in the current
//                                              peeling round (still part of the
//                                              old graph), 0 removed earlier
//   keys     uint32[(h-1) * n * cap]           B[v,i] for levels i = 1..h-1, one
//                                              fixed slot of cap >= M keys per
//                                              (level, node), as keys r << 27 |
//                                              position by falling rank, or as a
//                                              bitmap over positions (kh_sampled.cu)
//   meta     uint32[h * n]                     |B[v,i]|, k[v,i], highest rank, form
//   key32    uint32[n]                         r << 27 | position of each node
//   d32 / d64                                  deg_h (exact) or estimate (sampled)
//   seen     int32[n]                          stamp array for frontier dedup
//   lists    int32[n] x 4                      removed set, frontiers, work lists
//   state    kh_dev_state                      round counters (device resident)
//   scratch  per-CTA BFS queues (and bitmaps when n is too large for shared memory)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/khcore.h"
#include <nvtx3/nvToolsExt.h>

namespace kh {

constexpr int kRankBits = 5;
constexpr int kIdBits = 27;
constexpr uint32_t kIdMask = (1u << kIdBits) - 1u;
constexpr int kMaxM = 12000;
constexpr int kMaxH = 16;
constexpr int kPhaseStride = 32;  // stamp = round * kPhaseStride + phase
// Shared-memory visited bitmap limit per CTA (bytes); larger n uses global scratch.
constexpr int64_t kSmemBitmapMax = 100 * 1024;

// Dynamic shared memory the sliced 2-degree kernel may use per CTA (bytes).
constexpr int64_t kSmem2Max = 220 * 1024;
// Kernels whose dynamic shared memory depends on the graph set their
// maximum-dynamic-shared-memory attribute to the largest size they can ever
// use (a constant), not to the size of the launch at hand: contexts on other
// host threads (the server's slots) launch the same kernels concurrently, and
// a smaller value set by one between another's setting and its launch would
// make that launch fail.

// Error bits written by device-side checks.
constexpr int kErrQueue = 1;   // BFS queue overflow
constexpr int kErrProbe = 2;   // hash probe limit reached
constexpr int kErrList = 4;    // list larger than its slot
constexpr int kErrGraph = 8;   // CSR validation failure
constexpr int kErrLoop = 16;   // a work loop ran past its iteration bound
constexpr int64_t kProfSnapCap = 1 << 21;  // byte snapshots kept between two reads
constexpr int kOrderBinsMax = 48;  // log2 bins of a source's 2-hop work (order2)
constexpr int kSweepMinBin = 16;   // smallest work bin the tuner offers to the sweeps

// Kernel classes for the profiling counters (kh_prof_read kinds).
constexpr int kProfBfs = 0;       // exact h-degree / fixed-level count BFS
constexpr int kProfLevel1 = 1;    // level-1 lists
constexpr int kProfLevelU = 2;    // level >= 2 lists (bitmap or hashed union)
constexpr int kProfFrontier = 3;  // removed-set ball hops, neighbour marking
constexpr int kProfPeel = 4;      // begin, collect, select
constexpr int kProfKinds = 5;

// Per-round counters: every launch inside a peeling round has its own slot, and
// the next round's first kernel zeroes them all, so a round needs no memset nodes.
constexpr int kRcBfs = 0;          // refine BFS work counter
constexpr int kRcRefineWork = 1;   // refine last-level list work counter
constexpr int kRcLevelWork = 3;    // + i: refresh level i work counter, i = 1..kMaxH
constexpr int kRcSubWork = 20;     // + i: split-part work counter of level i (0: the refine)
constexpr int kRcW = 37;           // + i: work list of level i (0: exact affected nodes)
constexpr int kRcF = 54;           // + hop: frontier written by that hop (exact)
constexpr int kRcC = 71;           // + i: changed nodes at level i
constexpr int kRcLossWork = 88;    // exact refresh: loss-BFS work counter
constexpr int kRcLossCount = 89;   // exact refresh: nodes with a loss this round
constexpr int kRcSub = 90;         // + i: split-part items of level i (0: the refine)
constexpr int kRcCount = 107;
constexpr int kRoundKey = 21;      // what a captured batch of rounds holds (kh_peel.cu: round_graph)

struct DevState {
    unsigned long long c;        // current core value (max of round minima)
    unsigned long long minval;   // min d over alive nodes in this round
    int round;                   // current round index
    int n_alive;                 // alive nodes at the start of the round
    int n_alive_next;            // alive nodes after this round's removal
    int nR;                      // |R| removed this round
    int nC[2];                   // changed-list sizes (standalone level passes)
    int work_ctr[4];             // dynamic scheduling counters
    unsigned long long updates;  // node recomputations
    unsigned long long bytes[kProfKinds];  // algorithmic bytes per kernel class
    int err;                     // kErr* bits
    int nQ;                      // refine list size (stale nodes due this round)
    unsigned long long minU;     // min of the upper bounds d over alive nodes
    int rc[kRcCount];            // per-round counters (kRc*)
    // peel work statistics: list recomputations and changes per level in the
    // rounds' refresh passes, refines stopped early
    unsigned long long lvl_work[kMaxH + 1];
    unsigned long long lvl_changed[kMaxH + 1];
    unsigned long long stopped;
    int tune_count;              // sample size of an autotuner measurement
    int nSub;                    // split-part items (standalone level passes)
    unsigned long long deg2;     // sum of squared degrees, until the first peel reads it
};

struct Graph;

// The row readers of k_hdeg2_cta and k_hdeg2_peel: every step of a warp over a chunk
// of `rows` rows of up to 511 entries reads one of them on (short and middle rows in
// one step, the others 128 entries a step) or ends one of three buckets, so no
// correct loop takes more steps than this; one that does ends with kErrLoop.
constexpr int row_steps(int rows) { return 4 * rows + 4; }

// After a round's removal set is chosen: c = max(c, the round's minimum) of every
// graph, the minima back to none.  Done by one block of the first refresh kernel
// (nothing else reads them before the next round).
struct RoundEnd {
    unsigned long long *c, *mn, *mr, *mu;  // c nullptr: nothing to do
    int64_t ngraphs;
};
#ifdef __CUDACC__
__device__ __forceinline__ void end_round(const RoundEnd& r) {
    if (!r.c) return;
    for (int64_t q = threadIdx.x; q < r.ngraphs; q += blockDim.x) {
        const unsigned long long m = r.mn[q] < r.mr[q] ? r.mn[q] : r.mr[q];
        if (m != ~0ull && m > r.c[q]) r.c[q] = m;
        r.mn[q] = ~0ull;
        r.mr[q] = ~0ull;
        r.mu[q] = ~0ull;
    }
}
// Sec. 5: with c >= |X| - 1 every remaining node has deg_h <= |X| - 1 <= c.
__device__ __forceinline__ bool early_stop(unsigned long long c, int left) {
    return left > 0 && c + 1 >= (unsigned long long)left;
}
#endif
RoundEnd round_end(const Graph& g);

// Level unions split nodes of more than kSplitDeg neighbours into parts of
// kSplitChunk neighbours each, on graphs with a node of more than kSplitMin.  One
// CTA reads 1024 lists in about 20 us, as long as a whole launch of a middle
// round; below that the parts' own set-up costs more than the shorter tail
// gives (sampled (k,3)-cores of Chung-Lu n = 200k / R-MAT 18: 513 / 216 ms from
// 2048 on, 502 / 206 from 1024, 497 / 264 from 512 with parts of 256).  Without a
// really heavy node the launch of the parts costs more than it gives ((k,2)-core
// of Chung-Lu n = 50k, largest degree 1250: 328 -> 335 ms).
constexpr int kSplitMin = 2048;
constexpr int kSplitDeg = 1024;
constexpr int kSplitChunk = 512;

// Part slots and items of one union pass.  Whoever lists the nodes of the pass
// hands the heavy ones to their parts instead, so that the parts can run beside
// the other nodes.
struct PartPlan {
    int* n_sub;           // items planned
    int32_t *sub_v, *sub_j;
    int32_t* split_first; // a heavy node's first slot
    int64_t cap;          // slots (0: the graph has no heavy node)
    int* err;
};
#ifdef __CUDACC__
// Plan v's parts if it is heavy (one thread); false: not heavy.
__device__ __forceinline__ bool plan_parts(const PartPlan& p, int v, int64_t deg) {
    if (p.cap == 0 || deg <= kSplitDeg) return false;
    const int P = (int)((deg + kSplitChunk - 1) / kSplitChunk);
    const int base = atomicAdd(p.n_sub, P);
    if ((int64_t)base + P <= p.cap) {
        for (int j = 0; j < P; ++j) {
            p.sub_v[base + j] = v;
            p.sub_j[base + j] = j;
        }
        p.split_first[v] = base;
    } else {
        // cannot happen: cap covers every heavy node of the graph at once
        for (int64_t j = base; j < p.cap && j < (int64_t)base + P; ++j) p.sub_v[j] = -1;
        atomicOr(p.err, kErrList);
    }
    return true;
}
#endif
// the plan whose items level `level` of a round computes (0: the refine)
PartPlan round_parts(const Graph& g, int level);

// The lazy refine decides whether d(v) <= T = max(c, U) and may stop once a
// partial value (a lower bound of d(v)) exceeds it.  It runs on until the
// partial value exceeds kStopSlack * T instead: the node's new lower bound then
// stays above the rising threshold for longer, so a node whose value is far
// above T is refined O(log) times instead of once per round (any lower bound
// above T gives the same removal decision).
constexpr unsigned long long kStopSlack = 2;
__host__ __device__ __forceinline__ unsigned long long stop_level(unsigned long long T) {
    return T >= (~0ull) / kStopSlack ? ~0ull : T * kStopSlack;
}

// A launch layout of the whole-graph exact 2-degree pass (kh_tune.cu):
// variant KH_VAR_CTA or KH_VAR_SLICED (KH_VAR_AUTO: not chosen yet), the
// sliced kernel's slice count and CTA size, and the sample time it took.
struct TuneChoice {
    int variant;
    int slices;
    int threads;
    double ms;
    int sweep_bin;  // sources with 2-hop work >= 2^sweep_bin go to the bit-parallel sweeps (0: none)
};

// NVTX range for profilers and tracers (a no-op unless a tool is attached).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// ---- launchers (kh_exact.cu) -------------------------------------------------
void launch_ranks(const Graph& g, cudaStream_t s);
// each node's neighbour of largest degree (computed once per graph, before a peel)
int ensure_bestnb(Graph& g, cudaStream_t s);
void launch_validate(const Graph& g, int* d_err, cudaStream_t s);
// exact h-degrees of `count` nodes (worklist == nullptr: nodes 0..n-1) into deg32;
// when cnt != nullptr also the fixed-level counts for j in [jlo, jlo+nj).
// early_stop (the peel's lazy refine): a source whose partial ball already
// holds more than T = max(c, mu) of its graph stops and stays stale with that
// count as its lower bound.
// loss (the peel's exact refresh): sources are the removed nodes of the round;
// every alive node first reached at the source's last hop and not within h-1
// hops of the removed set (ball stamp) gains one in loss[] instead of a degree.
int launch_hdeg(Graph& g, const int* worklist, const int* d_count, int64_t count_static,
                int32_t* deg, int32_t* cnt, int jlo, int nj, cudaStream_t s,
                int* round_ctr = nullptr, bool early_stop = false, bool loss = false);
// d and (stale nodes) lb drop by loss[] for the listed nodes; loss[] is cleared
void launch_apply_loss(Graph& g, cudaStream_t s);
// one hop of the removed set's ball in the old graph (exact refresh)
void launch_ball_hop(Graph& g, int hop, cudaStream_t s);
// exact mode: mark the nodes of `list` (nullptr: all) stale and set their
// lower bound max(deg_X(v), max_w deg_X(w)) <= deg_h(v; X) for h >= 2
void launch_stale_exact(Graph& g, const int* list, const int* d_count, cudaStream_t s);

// ---- launchers (kh_hdeg2.cu) -------------------------------------------------
// exact 2-degrees (and fixed-level counts when cnt != nullptr) of every node
// with a sliced shared-memory visited set: `slices` node ranges, `threads` per
// CTA, sources from `order` (nsrc of them).  init: deg (and cnt) are set to
// their starting values first (every node); otherwise they must hold them.
int launch_hdeg2_slice(Graph& g, int32_t* deg, int32_t* cnt, int jlo, int nj, cudaStream_t s,
                       int slices, int threads, const int32_t* order, int64_t nsrc, bool init);
// the same with one CTA per source and a bitmap of all n nodes (n <= 819200); the
// caller opens the profiling bracket (large and other sources run beside each other)
int launch_hdeg2_cta(Graph& g, int32_t* deg, int32_t* cnt, int jlo, int nj, cudaStream_t s,
                     const int32_t* order, int64_t nsrc, bool large);
int launch_init2(Graph& g, int32_t* deg, int32_t* cnt, int jlo, int nj, cudaStream_t s);
// in that layout the sources of `order2` from a bin of 2-hop work on take a large
// CTA each (hdeg2_large_bin), those below kCtaSmallBin a warp each: below 127
// entries a warp's hash set costs less than a CTA's barriers (grid of 160k
// nodes: 0.36 -> 0.16 ms)
int hdeg2_large_bin(const Graph& g);
constexpr int kCtaSmallBin = 7;
// crank: the rank of each column entry (kept until the ranks change)
int ensure_crank(Graph& g, cudaStream_t s);
// the sources of the sliced kernel, longest 2-hop work first (cached per graph)
int ensure_order2(Graph& g, cudaStream_t s);
size_t hdeg2_smem(int64_t width);
// sources of order2 whose 2-hop work is too large for the warp-per-source
// kernel (they come first in order2), and that kernel for the rest
int64_t hdeg2_small_split(const Graph& g);
// sources of order2 whose 2-hop work is at least 2^bin (they come first)
int64_t hdeg2_sources_from_bin(const Graph& g, int bin);
// exact h-degrees (h >= 2) of `count` non-isolated sources by bit-parallel
// searches of kSweepBatch sources
constexpr int64_t kSweepBatch = 1024;
int run_sweeps(Graph& g, int32_t* deg, const int32_t* src, int64_t count, int h, cudaStream_t s);
int ensure_sweep(Graph& g, int h, cudaStream_t s);
int launch_hdeg2_small(Graph& g, int32_t* deg, int32_t* cnt, int jlo, int nj, cudaStream_t s,
                       const int32_t* order, int64_t count);
// kh_tune.cu: the layout of the 2-degree pass for this graph (tuned once), and
// the whole-graph exact h-degree / fixed-level count pass through it
int choose_hdeg2(Graph& g, cudaStream_t s, TuneChoice* out);
int run_hdeg_full(Graph& g, int32_t* deg, int32_t* cnt, int jlo, int nj, cudaStream_t s);
int64_t hdeg2_width(int64_t n, int slices);
int hdeg2_min_slices(int64_t n);

// ---- launchers (kh_sampled.cu) -----------------------------------------------
// level i of the list recursion for `count` nodes (worklist == nullptr: all);
// track != 0 records nodes whose (|B|, k) changed into the changed list.
// round_mode 0: standalone (counters zeroed with memsets); 1: refresh of
// level `level` inside a round; 2: refine of the last level inside a round
// (per-round counters, no memsets).
int launch_level(Graph& g, int level, const int* worklist, const int* d_count,
                 int64_t count_static, int track, cudaStream_t s, int round_mode = 0,
                 int skip_last = -1);
// A(list1) and the part of A(list2) (may be nullptr) whose level `phase` can have
// changed (rank filter on rho), deduplicated by stamp phase: nodes whose last
// level it is become stale, the others join the work list listW (count
// *out_count).  Phase 1 also ends the round's selection (end_round).
void launch_mark_neighbours(Graph& g, const int* list1, const int* cnt1, const int* list2,
                            const int* cnt2, int phase, int* out_count, cudaStream_t s);
// start of a sampled peel: every alive node stale with a lower bound
void launch_stale_all(Graph& g, cudaStream_t s);
// start of a peel: meta words of no lists, alive nodes stale at their last level
int launch_init_meta(Graph& g, cudaStream_t s);
// each node's last-level k and |B| into device arrays (either may be nullptr)
void launch_gather_last(Graph& g, uint8_t* lvl_out, int32_t* bs_out, cudaStream_t s);

// ---- launchers (kh_peel.cu) --------------------------------------------------
int run_core(Graph& g, bool sampled, void* out_core, int32_t* round_of_host, bool out_dev);
// EstDense (Alg. 7): replay of a removal order with eager refresh; per round,
// the sum of d over the alive set (host outputs)
int run_dense(Graph& g, bool sampled, const int32_t* round_of, int32_t rounds, uint64_t* sum,
              int64_t* size, int32_t* best);
int run_estimate_all(Graph& g);  // enqueued; the caller checks state->err

}  // namespace kh

struct kh_pinned {
    kh::DevState states[2];    // the device state after the last two replays of a peel
    int err;
    uint8_t stage[256 * 1024]; // small results on their way to the caller
};

struct kh_ctx {
    int device;
    cudaStream_t stream;
    bool own_stream;
    int sm_count;
    char err[512];
    // a second stream for work beside a launch's own (forked from and joined to
    // `stream` by the two events)
    cudaStream_t side;
    cudaEvent_t fork, join;
    struct kh_pinned* pinned;  // pinned host memory of the context
    cudaEvent_t peel_done[2];
    // fault injection on the host: the fail_alloc_at-th device allocation from
    // the arming call fails with KH_ENOMEM (0: off)
    int64_t fail_alloc_at;
    int64_t alloc_count;
};

#ifdef __CUDACC__
namespace kh {
// Lane j adds #{lanes : r >= j} to its count (r = -1: no key; all 32 lanes call
// it).  Ranks are geometric, so a warp's 32 keys need about 7 ballots (no
// shared-memory atomics: half the keys of a histogram would fall on one address).
__device__ __forceinline__ void add_rank_counts(int r, int lane, int& S) {
#pragma unroll 1
    for (int j = 0; j < 32; ++j) {
        const uint32_t b = __ballot_sync(0xffffffffu, r >= j);
        if (!b) break;
        if (lane == j) S += __popc(b);
    }
}

// A lane's counts of nodes by rank: ranks 0..7 as the bytes of one word, the
// others (1 node in 256) straight into the shared histogram.  A histogram
// atomic per node would fall on one address for every second node.
struct RankCounts {
    unsigned long long r8 = 0;
    int since = 0;  // nodes since the last flush; a byte holds 255
    __device__ __forceinline__ void add(int r, int* s_hist) {
        if (r < 8) {
            r8 += 1ull << (8 * r);
            ++since;
        } else {
            atomicAdd(&s_hist[r], 1);
        }
    }
    // before a step that adds up to 5 nodes
    __device__ __forceinline__ void reserve(int* s_hist) {
        if (since <= 250) return;
#pragma unroll 1
        for (int r = 0; r < 8; ++r) {
            const int c = (int)(r8 >> (8 * r)) & 255;
            if (c) atomicAdd(&s_hist[r], c);
        }
        r8 = 0;
        since = 0;
    }
    // the warp's counts into the histogram (all 32 lanes): two ranks per sum (32
    // bytes fit 16 bits), lane r adds rank r
    __device__ __forceinline__ void finish(int* s_hist, int lane) {
        const uint32_t lo = (uint32_t)r8, hi = (uint32_t)(r8 >> 32);
        const uint32_t a = __reduce_add_sync(0xffffffffu, lo & 0x00ff00ffu);
        const uint32_t b = __reduce_add_sync(0xffffffffu, (lo >> 8) & 0x00ff00ffu);
        const uint32_t c = __reduce_add_sync(0xffffffffu, hi & 0x00ff00ffu);
        const uint32_t d = __reduce_add_sync(0xffffffffu, (hi >> 8) & 0x00ff00ffu);
        const uint32_t w = lane & 4 ? (lane & 1 ? d : c) : (lane & 1 ? b : a);
        const int n = (int)(lane & 2 ? w >> 16 : w & 0xffffu);
        if (lane < 8 && n) atomicAdd(&s_hist[lane], n);
        r8 = 0;
        since = 0;
    }
};
}  // namespace kh
#endif

namespace kh {
struct Graph {
    kh_ctx* ctx;
    int64_t n;
    int64_t nnz;
    int h;
    uint64_t seed;
    int64_t M;
    int64_t cap;            // list slot capacity (>= M, multiple of 4)
    bool ranks_valid;
    bool lists_valid;       // lists hold the full-graph recursion for (h, M, seed)
    int64_t *rowptr;
    int32_t *col;
    uint8_t *rank;
    uint8_t *crank;         // rank of each column entry (fixed-level counts)
    bool crank_valid;
    uint8_t *alive;
    uint32_t *keys;
    int64_t keys_levels;    // allocated levels in keys
    uint32_t *meta;         // meta word of each list (kh_sampled.cu)
    int64_t lvl_alloc;      // allocated levels in meta
    // positions of the nodes by descending rank (kh_sampled.cu: k_pos_*)
    bool pos_valid;
    uint32_t *key32;
    int32_t *clsw;
    uint8_t *wrank;
    uint32_t *lu_stage;     // k_levelU: compaction stage, one slot per CTA
    int64_t lu_stage_cap;
    int32_t *d32;
    unsigned long long *d64;
    int32_t *core32;
    unsigned long long *core64;
    int32_t *round_of;
    int32_t *seen;
    int32_t *listR;
    int32_t *listA;
    int32_t *listB;
    int32_t *listW;
    int32_t *listC[2];
    DevState *state;
    // BFS scratch
    int32_t *queues;
    uint32_t *gbitmaps;
    int64_t scratch_ctas;
    // batches of graphs packed in one CSR (all nullptr for a single graph)
    int32_t *gid;           // graph of each node
    int64_t *vtx_off;       // first node of each graph, ngraphs + 1 entries
    uint8_t *hv;            // per-node h (nullptr: g.h for every node)
    int32_t *Mv;            // per-node M (nullptr: g.M for every node)
    int64_t ngraphs;
    int64_t max_gn;         // largest graph of the batch
    // per graph: c, round-start minimum over fresh nodes, refine threshold,
    // minimum of the values the round's refine completed
    unsigned long long *pc, *pmn, *pmu, *pmr;
    int32_t *pleft;         // per-graph alive count (batches)
    int hmin, hmax;         // range of h over the nodes
    std::vector<int64_t>* h_vtx_off;  // host copy of vtx_off (per-graph M)
    std::vector<int32_t>* h_hgraph;   // host copy of the per-graph h
    // lazy refinement of the last level: fresh[v] = d[v] is exact for the
    // current alive set; otherwise d[v] is an upper bound (d never grows as
    // nodes leave) and lb64[v] (exact mode) a lower bound
    uint8_t *fresh;
    // rho[v]: highest rank among the elements that left or entered v's list in
    // the level just recomputed (-1: none); filters the next level's refresh
    int8_t *rho;
    uint32_t *deadbm;       // bitmap of removed nodes (n bits), seeds BFS visited sets
    int32_t *degX;          // alive degree (exact mode)
    unsigned long long *lb64;
    // exact refresh: loss[v] = removed nodes within h hops of a node exactly
    // h hops from the removed set (zero between rounds), listed in listL
    int32_t *loss;
    int32_t *listL;
    // last peel statistics
    int64_t last_rounds;
    int64_t last_updates;
    int64_t last_lvl_work[kMaxH + 1];
    int64_t last_lvl_changed[kMaxH + 1];
    int64_t last_stopped;
    bool have_rounds;
    // EstDense replay: the removal order (round per node), per-round sums of d
    bool dense;
    // the pruned EstDense replay starts from the kept nodes only (keep[v] != 0)
    bool start_keep;
    int64_t start_alive;
    uint8_t* keep;
    int32_t* sched;
    unsigned long long* dsum;
    // profiling: CUDA events around every launch of a kernel class
    bool prof_on;
    std::vector<cudaEvent_t>* ev_pool;
    std::vector<int>* prof_kind;
    std::vector<cudaEvent_t>* prof_ev;  // pairs (start, stop)
    double prof_ms[kProfKinds];
    int64_t prof_launches[kProfKinds];
    std::vector<float>* prof_trace[kProfKinds];  // per-bracket ms, in launch order
    // per-bracket algorithmic bytes: the class counter copied before and after
    // each bracket into prof_snap (device; prof_snapi: first slot or -1)
    unsigned long long* prof_snap;
    int64_t prof_nsnap;
    std::vector<int64_t>* prof_snapi;
    std::vector<unsigned long long>* prof_btrace[kProfKinds];
    // cached CUDA graph of a batch of peeling rounds
    cudaGraphExec_t round_exec;
    int64_t round_exec_key[kRoundKey];
    int64_t round_exec_kernels;  // kernels in one replay of round_exec
    // kernels launched on behalf of this graph (graph replays count their nodes)
    int64_t launches;
    // level passes: part slots of split heavy nodes (part_cap slots of cap
    // keys; 0 when the graph has no node above the split degree)
    int64_t part_cap;
    int64_t part_cap_keys;  // cap the slots were sized for
    uint32_t *part_keys;
    uint32_t *part_meta;
    int32_t *part_done;
    int32_t *part_stop;
    unsigned long long *part_lb;
    int32_t *split_first;
    int32_t *sub_v;
    int32_t *sub_j;
    bool split_planned;     // part_cap computed for this graph
    // the peel's view of the graph (kh_peel.cu): rowptr/col above are switched
    // to a compacted CSR of the nodes alive at the last compaction, and the
    // whole-node scans run over vlist (vcount nodes; nullptr: all n); the
    // graph's own arrays are kept in orig_* and restored when the peel ends
    int64_t *orig_rowptr;
    int32_t *orig_col;
    const int32_t *vlist;
    int64_t vcount;
    int compact_mode;       // KH_VAR_AUTO, KH_COMPACT_OFF or KH_COMPACT_ALWAYS
    int levelu_mode;        // KH_VAR_AUTO (grouped), KH_LEVELU_STEPPED, _FREE or _GROUPED
    int levelu_div;         // grouped: coverage divisor (0: the default)
    int cp_cur;             // buffer set in use (0 or 1)
    int64_t *cp_row[2];
    int32_t *cp_col[2];
    int64_t cp_col_cap[2];
    int32_t *cp_list[2];
    int64_t *cp_tmp;        // counts and flags, 2 (n + 1)
    int64_t *cp_sums;       // scan tile totals
    // sliced 2-degree kernel: sources longest first (non-isolated nodes only)
    int32_t *order2;
    int64_t nsrc2;
    int64_t order2_hist[48];  // sources per log2 bin of 2-hop work (order2 is by descending bin)
    // bit-parallel searches (kh_hdeg2.cu): mask buffers (32 words per node; the
    // first holds a batch's source bits and is zero between batches), node
    // filter, index of each long row (or -1), the long rows, their pieces and
    // partial ORs, per-source counts
    uint32_t* sw_m[3];
    uint32_t* sw_filter;
    int32_t* sw_hpos;
    int32_t* sw_piece_h;
    int32_t* sw_piece_off;
    int32_t* sw_hnode;
    uint32_t* sw_bh;
    unsigned int* sw_cnt;
    int64_t sw_nheavy, sw_npieces;
    bool sw_ready;
    // h >= 3: per-source search or bit-parallel batches (0: not decided yet)
    int hdeg_deep[kMaxH + 1];
    int sw_force;             // forced sweep threshold bin (0: tuner; -1: no sweeps)
    // each node's neighbour of largest degree (-1: none), for cheap stale bounds
    int32_t *bestnb;
    unsigned long long deg2;  // sum of squared degrees (0: no peel has run yet)
    // the 2-degree pass layout: forced by kh_set_variant, or chosen by the tuner
    TuneChoice force_hdeg2;
    TuneChoice tuned_hdeg2;
};
}  // namespace kh

struct kh_graph {
    kh::Graph g;
};

namespace kh {
// Utility: set the context error text; returns code.
int set_error(kh_ctx* ctx, int code, const char* fmt, ...);
// Ensure the per-graph work arrays exist (idempotent).
int ensure_work(Graph& g);
int ensure_lists(Graph& g);
// part slots for the split heavy nodes of the level passes (kh_sampled.cu)
int ensure_split(Graph& g);
// ranks, and the positions the sampled lists use (kh_sampled.cu)
int ensure_positions(Graph& g);
int ensure_bfs_scratch(Graph& g, int64_t ctas, bool bitmaps);
// A device allocation through the context's fault-injection counter.
int alloc_bytes(kh_ctx* ctx, void** p, size_t bytes, const char* what);
int check_cuda(kh_ctx* ctx, cudaError_t e, const char* what);
inline void count_launch(Graph& g, int64_t k) { g.launches += k; }
// Profiling brackets around a launch (no-ops unless profiling is enabled).
void prof_begin(Graph& g, int kind, cudaStream_t s);
void prof_end(Graph& g, int kind, cudaStream_t s);
}  // namespace kh

#define KH_CUDA_TRY(ctx, expr)                                  \
    do {                                                        \
        cudaError_t _e = (expr);                                \
        if (_e != cudaSuccess) return kh::check_cuda((ctx), _e, #expr); \
    } while (0)
