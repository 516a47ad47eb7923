// kh_sampled.cu -- the level recursion of the sampled lists B[v,i], k[v,i].
//
// Prop. 3.1: B[v,i] is the rank filter of T = {v} U B[w,i-1] (w alive
// neighbours of v) at level k[v,i] >= max_w k[w,i-1], and Alg. 2 picks the
// smallest level leaving at most M members.  Because N(w; i-1) is inside
// N(v; i), the result equals {u in N(v;i,X) : r[u] >= kappa} with kappa the
// smallest level whose rank-filtered N(v;i,X) has at most M members, so B and
// k depend only on the alive set, the ranks and M.
//
// Positions.  Nodes are numbered by descending rank (k_pos_*): every node has a
// position, the positions of one rank class start at a multiple of 32, and
// the nodes of rank >= j occupy the first clsw[j] 32-bit words of a bitmap over
// positions.  A list key is r << 27 | position.
//
// A stored list has one of two forms (a flag in its meta word): sparse, |B| keys
// grouped by rank, highest first; or dense, the first clsw[k] words of the
// bitmap over positions, when those are fewer words than |B| (a ball of more
// than about n/32 nodes).
//
// Level 1 (T = {v} plus alive neighbours, no repeats): one warp per node, the
// counts S_j by ballots, kappa from them, a second pass writes the members
// grouped by rank.
//
// Levels >= 2: one CTA per node (k_levelU, see there).  A running threshold t
// starts at max_w k[w,i-1]; keys below t are skipped, and because each list is
// ordered by rank from the highest, a list is left at its first key below t.
// As the union grows t rises to the smallest level whose count of distinct
// members is <= M (Alg. 5's trim).  The last level only needs |B[v,h]| and
// k[v,h] for the estimate of Alg. 1, so it writes no list.
//
// A node's (|B|, k) pair changes exactly when B[v,i] or k[v,i] changes: with k
// fixed, the new list is a subset of the old one (nodes only leave), so equal
// sizes mean equal sets.  Changed nodes drive the next level's refresh (Alg. 3).
#include "kh_internal.cuh"

namespace kh {

namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr int kL1Threads = 256;
constexpr int kLuThreads = 128;
constexpr int kLuWarps = kLuThreads / 32;
constexpr int kLuPerSm = 12;  // CTAs per SM of k_levelU

// Meta word of a list (one per level and node): |B| in bits 0-13, k in bits
// 14-19, the highest rank present in bits 20-24, the dense-form flag, and a
// flag that is set while the node is alive (a removed node's word is zero; in
// a peel the last level's word has it from the start).
constexpr uint32_t kMetaAlive = 1u << 31;
constexpr uint32_t kMetaDense = 1u << 30;
constexpr uint32_t kMetaFresh = 1u << 29;  // last level: (|B|, k) are those of the current alive set
__device__ __forceinline__ int meta_size(uint32_t m) { return (int)(m & 0x3fffu); }
__device__ __forceinline__ int meta_k(uint32_t m) { return (int)((m >> 14) & 63u); }
__device__ __forceinline__ int meta_top(uint32_t m) { return (int)((m >> 20) & 31u); }
__device__ __forceinline__ uint32_t meta_pack(int S, int k, int top, bool dense) {
    return kMetaAlive | (dense ? kMetaDense : 0u) | ((uint32_t)top << 20) | ((uint32_t)k << 14) |
           (uint32_t)S;
}
constexpr uint32_t kMetaSizeK = (1u << 20) - 1u;  // the (|B|, k) part

// First word of a graph's part of wrank (graph q of a batch; its positions are
// local to the graph).  A graph of n' nodes needs at most n'/32 + 32 words.
// (A multiple of 4: wrank is read four words at a time.)
__host__ __device__ __forceinline__ int64_t word_base(int64_t first_node, int64_t q) {
    return ((first_node >> 5) + 36 * q + 3) & ~(int64_t)3;
}

struct LevelArgs {
    const int64_t* rowptr;
    const int32_t* col;
    const uint8_t* alive;
    const uint32_t* key32;     // r << 27 | position of each node
    const int32_t* clsw;       // per graph 33 entries: words covering the ranks >= j
    const uint8_t* wrank;      // rank class of each bitmap word
    const int64_t* vtx_off;    // batches: first node of each graph
    int64_t n;
    int level;                 // level to compute; 0: each node's last level h(v)
    int h;                     // h of every node when hv is nullptr
    const uint8_t* hv;         // per-node h (batches)
    int skip_last;             // leave a node's last level to the lazy refine
    int64_t M;                 // M of every node when Mv is nullptr
    const int32_t* Mv;         // per-node M (batches)
    int64_t cap;
    uint32_t* keys;            // level i lists at keys + (i-1) n cap
    uint32_t* meta;            // level i meta words at meta + (i-1) n
    unsigned long long* est;   // estimate (at a node's last level)
    const int32_t* worklist;
    const int* d_count;
    int64_t count_static;
    int track;
    int group_lists;           // union: lane groups per list (0: a warp per list)
    int group_shift;           // a group covers 1/2^group_shift of the expected keys
    int lg;                    // hash form of the union's set: 2^lg slots
    int bm_words;              // bitmap form: words that fit (0: never)
    uint32_t* stage;           // per CTA: cap keys (compaction of the hash form)
    int32_t* changed;
    int* n_changed;
    int* work_ctr;
    int* err;
    unsigned long long* updates;
    unsigned long long* bytes;
    // Early stop of the lazy refine: a node whose partial estimate already
    // exceeds T = max(c, mu) of its graph cannot leave in this round, so it
    // stays stale with that value as its lower bound (nullptr: no early stop).
    const unsigned long long* stop_c;
    const unsigned long long* stop_mu;
    const int32_t* gid;
    unsigned long long* lb;
    uint8_t* fresh;
    // work statistics (indexed by level) and early-stop count
    unsigned long long* lvl_work;
    unsigned long long* lvl_changed;
    unsigned long long* stopped;
    int8_t* rho;  // tracked passes: top rank of each changed list's changes
    unsigned long long* min_done;  // refine: per-graph minimum of the completed values
    // split heavy nodes (k_levelU): partial sets of cap words per part slot,
    // their meta words, parts finished per split node (at its first slot)
    uint32_t* part_keys;
    uint32_t* part_meta;
    int32_t* part_done;
    int32_t* part_stop;             // per split node: some part stopped early (refine)
    unsigned long long* part_lb;    // per split node: the largest partial estimate above T
    PartPlan plan;
};

constexpr int kL1Heavy = 512;
constexpr int kL1BlockHeavy = 64;
// What one node computes in this launch: its level, whether that is its last
// level h(v) (estimate) or an intermediate one (list), its M, and where its
// inputs (level - 1) and outputs live.
struct NodeLevel {
    int lvl;
    bool last;
    bool skip;
    int M;
    const uint32_t* keys_in;
    uint32_t* keys_out;  // nullptr at a node's last level (no list is stored)
    const uint32_t* meta_in;
    uint32_t* meta_out;
};

__device__ __forceinline__ NodeLevel node_level(const LevelArgs& a, int v) {
    NodeLevel nl;
    const int hvv = a.hv ? (int)a.hv[v] : a.h;
    nl.lvl = a.level ? a.level : hvv;
    nl.last = nl.lvl == hvv;
    nl.skip = nl.lvl > hvv || (nl.last && a.skip_last);
    nl.M = a.Mv ? a.Mv[v] : (int)a.M;
    const size_t nn = (size_t)a.n, lc = nn * (size_t)a.cap;
    const int L = nl.lvl;
    nl.keys_in = L >= 2 ? a.keys + (size_t)(L - 2) * lc : nullptr;
    nl.keys_out = (!nl.last && a.keys) ? a.keys + (size_t)(L - 1) * lc : nullptr;
    nl.meta_in = L >= 2 ? a.meta + (size_t)(L - 2) * nn : nullptr;
    nl.meta_out = a.meta + (size_t)(L - 1) * nn;
    return nl;
}

__device__ __forceinline__ unsigned long long estimate_of(int S, int kappa, int rv, int64_t M) {
    // Alg. 1: d = |B[v,h] \ {v}| 2^k; if k > 0, d = max(d, M 2^(k-1))
    const int T = S - (rv >= kappa ? 1 : 0);
    unsigned long long d = (unsigned long long)T << kappa;
    if (kappa > 0) {
        const unsigned long long f = (unsigned long long)M << (kappa - 1);
        if (f > d) d = f;
    }
    return d;
}

__device__ __forceinline__ void record_change(const LevelArgs& a, const NodeLevel& nl, int v,
                                              uint32_t m) {
    const uint32_t old = nl.meta_out[v];
    nl.meta_out[v] = m;
    if (!a.track) return;
    atomicAdd(a.lvl_work + nl.lvl, 1ull);
    if ((old ^ m) & kMetaSizeK) {
        atomicAdd(a.lvl_changed + nl.lvl, 1ull);
        const int p = atomicAdd(a.n_changed, 1);
        if (p < a.n) a.changed[p] = v;
    }
}

// rho of a tracked list about to be rewritten with (S, kappa): the highest rank
// among the members that left and, if the level fell, old level - 1 (the
// members that entered rank below the old level); a list with the same size
// and level is unchanged and keeps none.  At level 1 the members that leave are
// exactly the neighbours removed in this round (alive == 2): a removal
// refreshes every neighbour's level-1 list in its round.  dead_top: the highest
// rank among those neighbours (-1: none).
__device__ __forceinline__ void level1_rho(const LevelArgs& a, const NodeLevel& nl, int v, int S,
                                           int kappa, int dead_top) {
    const uint32_t old = nl.meta_out[v];
    const int old_k = meta_k(old);
    if (meta_size(old) == S && old_k == kappa) return;
    int r = kappa != old_k ? old_k - 1 : -1;
    if (dead_top >= old_k) r = max(r, dead_top);
    a.rho[v] = (int8_t)r;
}

// Bytes a node's level-1 computation must move: row offsets, the row, the
// neighbours' ranks, and the list it writes with its size and level.
__device__ __forceinline__ unsigned long long level1_bytes(int64_t deg, int S, int last) {
    return 8ull + 5ull * (unsigned long long)deg + (last ? 8ull : 4ull * (unsigned long long)S) + 5ull;
}

// kappa, the list size at kappa and the highest rank present from the counts
// S_j held by lane j.
__device__ __forceinline__ void level_of_counts(int S, int M, int& kappa, int& Skap, int& top) {
    const uint32_t over = __ballot_sync(kFull, S > M);
    kappa = over ? 32 - __clz(over) : 0;
    const int Sk = __shfl_sync(kFull, S, kappa & 31);
    Skap = kappa < 32 ? Sk : 0;
    const uint32_t nz = __ballot_sync(kFull, S > 0);
    top = nz ? 31 - __clz(nz) : 0;
}

// Level 1.  One warp per node; rows longer than kL1Heavy are gathered per block
// and done by all its warps after the warp-per-node pass.
__global__ void __launch_bounds__(kL1Threads) k_level1(LevelArgs a) {
    __shared__ int s_off[kL1Threads / 32][32];
    __shared__ int s_heavy[kL1BlockHeavy];
    __shared__ int s_nheavy, s_kappa, s_S, s_top, s_dead;
    __shared__ int s_cnt[32];
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    int* off = s_off[wib];
    const int64_t total = a.worklist ? (int64_t)(*a.d_count) : a.count_static;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long my_bytes = 0;
    if (tid == 0) s_nheavy = 0;
    __syncthreads();
    for (int64_t idx = ((int64_t)blockIdx.x * blockDim.x + tid) >> 5; idx < total; idx += nw) {
        const int v = a.worklist ? a.worklist[idx] : (int)idx;
        if (a.alive[v] != 1) continue;
        const NodeLevel nl = node_level(a, v);
        if (nl.skip || nl.lvl != 1) continue;
        const int64_t b = a.rowptr[v], e = a.rowptr[v + 1];
        if (e - b > kL1Heavy) {
            int slot = 0;
            if (lane == 0) slot = atomicAdd(&s_nheavy, 1);
            slot = __shfl_sync(kFull, slot, 0);
            if (slot < kL1BlockHeavy) {
                if (lane == 0) s_heavy[slot] = v;
                continue;
            }
        }
        const uint32_t kv = a.key32[v];
        const int rv = (int)(kv >> kIdBits);
        int S = rv >= lane ? 1 : 0, dead = -1;
        for (int64_t k0 = b; k0 < e; k0 += 32) {
            int r = -1;
            if (k0 + lane < e) {
                const int32_t u = a.col[k0 + lane];
                const int au = a.alive[u];
                const int ru = (int)(a.key32[u] >> kIdBits);
                if (au == 1) r = ru;
                if (au == 2) dead = max(dead, ru);
            }
            add_rank_counts(r, lane, S);
        }
        int kappa, Skap, top;
        level_of_counts(S, nl.M, kappa, Skap, top);
        if (lane == 0) my_bytes += level1_bytes(e - b, Skap, nl.last);
        if (nl.last) {
            if (lane == 0) {
                const unsigned long long est = estimate_of(Skap, kappa, rv, nl.M);
                a.est[v] = est;
                if (a.min_done) atomicMin(a.min_done + (a.gid ? a.gid[v] : 0), est);
                record_change(a, nl, v, meta_pack(Skap, kappa, top, false) | kMetaFresh);
                atomicAdd(a.updates, 1ull);
            }
            continue;
        }
        if (a.track) {
            dead = __reduce_max_sync(kFull, dead);
            if (lane == 0) level1_rho(a, nl, v, Skap, kappa, dead);
        }
        // members grouped by rank, highest first: rank j starts at S_{j+1}
        const int above = __shfl_down_sync(kFull, S, 1);
        __syncwarp();
        off[lane] = lane < 31 ? above : 0;
        __syncwarp();
        uint32_t* out = nl.keys_out + (size_t)v * (size_t)a.cap;
        for (int64_t k0 = b; k0 < e; k0 += 32) {
            if (k0 + lane < e) {
                const int32_t u = a.col[k0 + lane];
                if (a.alive[u] == 1) {
                    const uint32_t key = a.key32[u];
                    const int r = (int)(key >> kIdBits);
                    if (r >= kappa) {
                        const int p = atomicAdd(&off[r], 1);
                        if (p < a.cap) out[p] = key;
                        else atomicOr(a.err, kErrList);
                    }
                }
            }
        }
        if (lane == 0) {
            if (rv >= kappa) {
                const int p = atomicAdd(&off[rv], 1);
                if (p < a.cap) out[p] = kv;
                else atomicOr(a.err, kErrList);
            }
            record_change(a, nl, v, meta_pack(Skap, kappa, top, false));
        }
        __syncwarp();
    }
    __syncthreads();
    const int nh = min(s_nheavy, kL1BlockHeavy);
    for (int j = 0; j < nh; ++j) {
        const int v = s_heavy[j];
        const NodeLevel nl = node_level(a, v);
        if (tid < 32) s_cnt[tid] = 0;
        if (tid == 0) s_dead = -1;
        __syncthreads();
        const int64_t b = a.rowptr[v], e = a.rowptr[v + 1];
        const uint32_t kv = a.key32[v];
        const int rv = (int)(kv >> kIdBits);
        int S = wib == 0 && rv >= lane ? 1 : 0, dead = -1;
        for (int64_t k0 = b + wib * 32; k0 < e; k0 += blockDim.x) {
            int r = -1;
            if (k0 + lane < e) {
                const int32_t u = a.col[k0 + lane];
                const int au = a.alive[u];
                const int ru = (int)(a.key32[u] >> kIdBits);
                if (au == 1) r = ru;
                if (au == 2) dead = max(dead, ru);
            }
            add_rank_counts(r, lane, S);
        }
        if (S) atomicAdd(&s_cnt[lane], S);
        if (a.track) {
            dead = __reduce_max_sync(kFull, dead);
            if (lane == 0 && dead >= 0) atomicMax(&s_dead, dead);
        }
        __syncthreads();
        if (tid < 32) {
            S = s_cnt[lane];
            int kappa, Skap, top;
            level_of_counts(S, nl.M, kappa, Skap, top);
            const int above = __shfl_down_sync(kFull, S, 1);
            __syncwarp();
            s_cnt[lane] = lane < 31 ? above : 0;
            if (lane == 0) {
                s_kappa = kappa;
                s_S = Skap;
                s_top = top;
            }
        }
        __syncthreads();
        const int kappa = s_kappa, Skap = s_S;
        if (nl.last) {
            if (tid == 0) {
                const unsigned long long est = estimate_of(Skap, kappa, rv, nl.M);
                a.est[v] = est;
                if (a.min_done) atomicMin(a.min_done + (a.gid ? a.gid[v] : 0), est);
                record_change(a, nl, v, meta_pack(Skap, kappa, s_top, false) | kMetaFresh);
                atomicAdd(a.updates, 1ull);
                my_bytes += level1_bytes(e - b, Skap, 1);
            }
        } else {
            if (a.track && tid == 0) level1_rho(a, nl, v, Skap, kappa, s_dead);
            uint32_t* out = nl.keys_out + (size_t)v * (size_t)a.cap;
            for (int64_t k = b + tid; k < e; k += blockDim.x) {
                const int32_t u = a.col[k];
                if (a.alive[u] == 1) {
                    const uint32_t key = a.key32[u];
                    const int r = (int)(key >> kIdBits);
                    if (r >= kappa) {
                        const int p = atomicAdd(&s_cnt[r], 1);
                        if (p < a.cap) out[p] = key;
                        else atomicOr(a.err, kErrList);
                    }
                }
            }
            if (tid == 0) {
                if (rv >= kappa) {
                    const int p = atomicAdd(&s_cnt[rv], 1);
                    if (p < a.cap) out[p] = kv;
                    else atomicOr(a.err, kErrList);
                }
                record_change(a, nl, v, meta_pack(Skap, kappa, s_top, false));
                my_bytes += level1_bytes(e - b, Skap, 0);
            }
        }
        __syncthreads();
    }
    for (int o = 16; o > 0; o >>= 1) my_bytes += __shfl_down_sync(kFull, my_bytes, o);
    if (lane == 0 && my_bytes) atomicAdd(a.bytes, my_bytes);
}

// ---- levels >= 2: the union of the neighbours' lists -------------------------

// A flag another CTA of this launch may set (read past the L1 cache).
__device__ __forceinline__ int ld_acquire(const int32_t* p) {
    return *(volatile const int32_t*)p;
}

// Hash form of the set: open addressing, a slot holds ~key (0: empty).
// Returns whether `key` was new.
__device__ __forceinline__ bool set_insert(uint32_t* tab, int lg, uint32_t key, int* err) {
    const uint32_t mask = (1u << lg) - 1u, x = ~key;
    uint32_t s = ((key & kIdMask) * 0x9E3779B1u) >> (32 - lg);
#pragma unroll 1
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        // most keys of a union are repeats: a plain read settles them without an atomic
        const uint32_t cur = *(volatile uint32_t*)(tab + s);
        if (cur == x) return false;
        if (cur == 0u) {
            const uint32_t prev = atomicCAS(tab + s, 0u, x);
            if (prev == 0u) return true;
            if (prev == x) return false;
        }
        s = (s + 1u) & mask;
    }
    atomicOr(err, kErrProbe);
    return false;
}

// Whether `key` is in the hash form (linear probing, no deletions between rebuilds).
__device__ __forceinline__ bool set_contains(const uint32_t* tab, int lg, uint32_t key) {
    const uint32_t mask = (1u << lg) - 1u, x = ~key;
    uint32_t s = ((key & kIdMask) * 0x9E3779B1u) >> (32 - lg);
#pragma unroll 1
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        const uint32_t cur = tab[s];
        if (cur == x) return true;
        if (cur == 0u) return false;
        s = (s + 1u) & mask;
    }
    return false;
}

constexpr int kKeysPerLane = 4;  // words one lane loads per step (one 16-byte vector)

// Lists of a chunk of kLuThreads neighbours, by how a warp reads them: short
// ones (up to about 8 keys expected at or above t: 2 lanes a list), middle
// (up to 64: 8 lanes), long (a warp a list) and dense (8 lanes).
constexpr int kBuckets = 4;
// A bucket's claims over a chunk: its lists, and one in vain of each group of 2 lanes
// or more.  Every step of a warp claims, reads a list on by 8 words or more, or ends a
// bucket, so with the claims the walk is bounded; one past them ends the union with
// kErrLoop.  (A count of the steps took 5% of the estimates of G(2000, 8000) and 1.5% of
// those of R-MAT 22 in registers; the claims have theirs.)
constexpr int kMaxClaims = kLuThreads + kLuThreads / 2;
constexpr int kShort = 0, kMiddle = 1, kDense = 2, kLong = 3;

// Shared state of one node's union.
struct UnionShared {
    int hist[32];                // distinct members per rank
    int cls[33];                 // words covering the ranks >= j (this node's graph)
    int t, tot, exit, creq, used, nstage, rho, last, off_done;
    int kmax[kLuWarps];
    int nq[kBuckets], cq[kBuckets];  // lists per bucket, lists claimed
    unsigned long long T, part;  // early-stop threshold; partial estimate
    int32_t w[kLuThreads];       // per neighbour of the chunk: its node (or list index)
    uint16_t sz[kLuThreads];     //   and size
    uint8_t q[kBuckets][kLuThreads];
    int idx, v;                  // the CTA's next item
};

// The warp's view of the union's rank counts: lane j gets S_j = #{distinct
// keys inserted so far with rank >= j}.  Read while other warps insert, the
// counts are those of a subset of the union (each rank class read at one
// moment), so every level derived from them is at most the final one and the
// partial estimate is at most the final estimate (Prop. 4.2).
__device__ __forceinline__ int snapshot_counts(const int* s_hist, int lane) {
    int S = *(volatile const int*)(s_hist + lane);
    for (int off = 1; off < 32; off <<= 1) {
        const int x = __shfl_down_sync(kFull, S, off);
        if (lane + off < 32) S += x;
    }
    return S;
}

// What the walk over a node's lists needs besides the shared state.
struct UnionCtx {
    uint32_t* tab;
    const uint32_t* lists;   // list of neighbour w at lists + w cap
    const uint8_t* wrank;    // rank class of the graph's bitmap words
    int64_t cap;
    int lg, M, rv, stop_first;   // stop_first: first part slot (mode 1 refine) or -1
    bool hash, can_stop, vin, other;  // other: lists written by other CTAs of this launch (merge)
    const int32_t* part_stop;
    int* err;
};

// Read the chunk's lists, bucket by bucket (long and dense lists first: they
// raise t most).  Groups of 2^lgG lanes claim a list and read it 4 words per
// lane and step; a warp claims for all its idle groups at once.  Sparse lists end
// at their first key below the running level t; dense lists at the last word of
// the ranks >= t.  After a step that inserted, once the counts can matter, the
// warp raises t from its snapshot of the rank counts (Alg. 5's trim) and, in a
// refine, tests the partial estimate against T.  The bucket and the lane's open
// list stay in (bk, li, pos), so that the hash form can stop for a compaction.
// (One loop for all buckets, and no unrolling below: with a copy per bucket the
// kernel outgrew the instruction cache, 18 of 33 stall cycles per instruction.)
template <bool LAST, bool PARTS>
__device__ __forceinline__ void walk_chunk(const UnionCtx& c, UnionShared& sh, int& bk, int& li, int& pos,
                                           unsigned long long& my_bytes) {
    const int lane = threadIdx.x & 31;
    const uint32_t* lp = nullptr;
    int sz = 0;
    if (li >= 0) {  // a list kept over a compaction
        lp = c.lists + (size_t)sh.w[li] * (size_t)c.cap;
        sz = sh.sz[li];
    }
#pragma unroll 1
    for (;;) {
        // one read for the whole warp: lanes that saw a flag at different
        // moments would part ways before the ballots
        int stop = 0;
        if (lane == 0) stop = *(volatile int*)&sh.exit | *(volatile int*)&sh.creq;
        if (__shfl_sync(kFull, stop, 0) || bk < 0) return;
        const bool dense = bk == kDense;
        const int lgG = bk == kLong ? 5 : bk == kShort ? 1 : 3;
        const int lead = lane >> lgG << lgG;
        const uint32_t need = __ballot_sync(kFull, li == -1 && lane == lead);
        if (need) {
            int base = 0;
            if (lane == 0) base = atomicAdd(&sh.cq[bk], __popc(need));
            base = __shfl_sync(kFull, base, 0);
            if (base >= kMaxClaims) {
                if (lane == 0) {
                    atomicOr(c.err, kErrLoop);
                    atomicCAS(&sh.exit, 0, 2);  // the other warps leave too
                }
                return;
            }
            if (li == -1) {
                const int i = base + __popc(need & ((1u << lead) - 1u));
                li = -2;
                if (i < sh.nq[bk]) {
                    li = (int)sh.q[bk][i];
                    pos = (lane - lead) * kKeysPerLane;
                    lp = c.lists + (size_t)sh.w[li] * (size_t)c.cap;
                    sz = sh.sz[li];
                }
            }
        }
        if (__all_sync(kFull, li == -2)) {
            do --bk;
            while (bk >= 0 && sh.nq[bk] == 0);
            if (bk < 0) return;
            li = -1;
            continue;
        }
        // the lanes need not read this together and other warps raise it, so lanes may
        // hold different levels (each one valid): only for tests of a lane by itself
        const int t = *(volatile int*)&sh.t;
        int ins = 0;
        bool done = false;
        if (li >= 0) {
            const int end = dense ? sh.cls[t] : sz;
            if (pos < end) {
                const uint4 k4 = PARTS && c.other ? __ldcg(reinterpret_cast<const uint4*>(lp + pos))
                                         : *reinterpret_cast<const uint4*>(lp + pos);
                const uint32_t kk[4] = {k4.x, k4.y, k4.z, k4.w};
                my_bytes += 4ull * (unsigned long long)min(kKeysPerLane, end - pos);
                if (dense) {
#pragma unroll
                    for (int q = 0; q < kKeysPerLane; ++q) {
                        if (pos + q < end) {
                            uint32_t nw = kk[q] & ~*(volatile uint32_t*)(c.tab + pos + q);
                            if (nw) nw &= ~atomicOr(c.tab + pos + q, nw);
                            if (nw) {
                                atomicAdd(&sh.hist[c.wrank[pos + q]], __popc(nw));
                                ins += __popc(nw);
                            }
                        }
                    }
                } else if (!c.hash) {
#pragma unroll
                    for (int q = 0; q < kKeysPerLane; ++q) {
                        const int r = pos + q < end ? (int)(kk[q] >> kIdBits) : -1;
                        if (r < t) {
                            done = true;
                        } else {
                            uint32_t* wp = c.tab + ((kk[q] & kIdMask) >> 5);
                            const uint32_t bit = 1u << (kk[q] & 31u);
                            if (!(*(volatile uint32_t*)wp & bit) && !(atomicOr(wp, bit) & bit)) {
                                atomicAdd(&sh.hist[r], 1);
                                ++ins;
                            }
                        }
                    }
                } else {
                    uint4 kq = k4;
#pragma unroll 1
                    for (int q = 0; q < kKeysPerLane; ++q) {
                        const uint32_t key = kq.x;
                        kq.x = kq.y;
                        kq.y = kq.z;
                        kq.z = kq.w;
                        const int r = pos + q < end ? (int)(key >> kIdBits) : -1;
                        if (r < t) {
                            done = true;
                            break;
                        }
                        if (set_insert(c.tab, c.lg, key, c.err)) {
                            atomicAdd(&sh.hist[r], 1);
                            ++ins;
                        }
                    }
                }
            }
            pos += kKeysPerLane << lgG;
            done |= pos - (lane - lead) * kKeysPerLane >= end;  // the group's next step starts past the end
        }
        // ranks only fall along a list: after a key below t the rest is below t
        const uint32_t fin = __ballot_sync(kFull, done) >> lead;
        if (li >= 0 && (lgG == 5 ? fin : fin & ((1u << (1 << lgG)) - 1u))) li = -1;
        if (!__any_sync(kFull, ins)) continue;
        // members added: the trim and the early stop can only matter once the
        // union holds more than M (k > 0) or more than T members
        ins = __reduce_add_sync(kFull, ins);
        int tot = 0;
        if (lane == 0) {
            tot = atomicAdd(&sh.tot, ins) + ins;
            if (c.hash && atomicAdd(&sh.used, ins) + ins > (1 << (c.lg - 1))) *(volatile int*)&sh.creq = 1;
        }
        tot = __shfl_sync(kFull, tot, 0);
        if (tot <= c.M && !(LAST && c.can_stop && (unsigned long long)tot > sh.T)) continue;
        const int S = snapshot_counts(sh.hist, lane);
        const uint32_t over = __ballot_sync(kFull, S > c.M);
        const int pmax = over ? 31 - __clz(over) : -1;
        const int Sn = __shfl_sync(kFull, S, (pmax + 1) & 31);
        if (lane == 0 && pmax + 1 > t) {
            atomicMax(&sh.t, pmax + 1);
            *(volatile int*)&sh.tot = pmax < 31 ? Sn : 0;
        }
        if (LAST && c.can_stop) {
            // Def. 4.1 on the keys inserted so far plus v itself: a subset
            // of N(v;h) led by v, so by Prop. 4.2 at most the final estimate
            const int Sp = S + ((!c.vin && c.rv >= lane) ? 1 : 0);
            const uint32_t fits = __ballot_sync(kFull, Sp <= c.M);
            const int k = fits ? __ffs(fits) - 1 : 32;
            const int Sk = __shfl_sync(kFull, Sp, k & 31);
            const unsigned long long pe = estimate_of(k < 32 ? Sk : 0, k, c.rv, c.M);
            if (lane == 0) {
                if (pe > sh.T) {
                    atomicMax(&sh.part, pe);
                    atomicCAS(&sh.exit, 0, 1);
                }
                // a part stops too once another part of the node has shown d(v) > T
                if (PARTS && c.stop_first >= 0 && ld_acquire(c.part_stop + c.stop_first))
                    atomicCAS(&sh.exit, 0, 2);
            }
        }
    }
}

// Compaction of the hash form: the keys at or above the level trimmed from the
// complete counts (at most M) are staged in global memory and put back.
__device__ __forceinline__ void compact_set(const LevelArgs& a, UnionShared& sh, uint32_t* tab, int M) {
    const int tid = threadIdx.x, lane = tid & 31, C = 1 << a.lg;
    const int S = snapshot_counts(sh.hist, lane);
    const uint32_t over = __ballot_sync(kFull, S > M);
    const int tc = max(sh.t, over ? 32 - __clz(over) : 0);
    uint32_t* stage = a.stage + (size_t)blockIdx.x * (size_t)a.cap;
    if (tid == 0) sh.nstage = 0;
    __syncthreads();
    if (tid == 0) sh.t = tc;
#pragma unroll 1
    for (int i = tid; i < C; i += kLuThreads) {
        const uint32_t x = tab[i];
        if (!x) continue;
        tab[i] = 0u;
        if ((int)(~x >> kIdBits) >= tc) {
            const int p = atomicAdd(&sh.nstage, 1);
            if (p < a.cap) stage[p] = ~x;
            else atomicOr(a.err, kErrProbe);
        }
    }
    __syncthreads();
    const int ns = min(sh.nstage, (int)a.cap);
#pragma unroll 1
    for (int i = tid; i < ns; i += kLuThreads) set_insert(tab, a.lg, stage[i], a.err);
    if (tid == 0) {
        sh.used = ns;
        sh.tot = ns;
        sh.creq = 0;
    }
    __syncthreads();
}

// Write the finished union (members of rank >= kappa) as a list at `out` and
// return its meta word.  hist must hold the complete counts; it is used up.
// A bitmap with fewer words than members is stored as it is (dense form).
// Otherwise the bitmap is read out in word order, which is rank order: each warp
// takes a quarter of the words, four per lane and step, at the offset of the
// earlier quarters' members.  The hash form goes by per-rank offsets.
__device__ __forceinline__ uint32_t write_list(const LevelArgs& a, UnionShared& sh, const uint32_t* tab,
                                               bool bm, const uint8_t* wrank, uint32_t* out, int S,
                                               int kappa, int top) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (!bm) {
        __syncthreads();
        if (warp == 0) {  // start of each rank, highest first
            const int c = lane >= kappa ? sh.hist[lane] : 0;
            int incl = c;  // over the ranks >= lane
            for (int off = 1; off < 32; off <<= 1) {
                const int x = __shfl_down_sync(kFull, incl, off);
                if (lane + off < 32) incl += x;
            }
            sh.hist[lane] = incl - c;
        }
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < (1 << a.lg); i += kLuThreads) {
            const uint32_t x = tab[i];
            if (!x) continue;
            const uint32_t key = ~x;
            const int r = (int)(key >> kIdBits);
            if (r < kappa) continue;
            const int p = atomicAdd(&sh.hist[r], 1);
            if (p < a.cap) out[p] = key;
            else atomicOr(a.err, kErrList);
        }
        return meta_pack(S, kappa, top, false);
    }
    const int W = sh.cls[kappa];
    if (W < S) {
#pragma unroll 1
        for (int i = tid; i < W; i += kLuThreads) out[i] = tab[i];
        return meta_pack(S, kappa, top, true);
    }
    const int per = ((W + 4 * kLuThreads - 1) / (4 * kLuThreads)) * 128;  // words per warp
    const int b = warp * per, e = min(W, b + per);
    int cnt = 0;
#pragma unroll 1
    for (int i = b + lane; i < e; i += 32) cnt += __popc(tab[i]);
    cnt = __reduce_add_sync(kFull, cnt);
    if (lane == 0) sh.kmax[warp] = cnt;
    __syncthreads();
    int base = 0;
    for (int i = 0; i < kLuWarps - 1; ++i) base += i < warp ? sh.kmax[i] : 0;
#pragma unroll 1
    for (int i0 = b; i0 < e; i0 += 128) {
        const int i = i0 + lane * 4;
        uint4 x = make_uint4(0u, 0u, 0u, 0u);
        if (i < e) x = *reinterpret_cast<const uint4*>(tab + i);
        if (i + 1 >= e) x.y = 0u;
        if (i + 2 >= e) x.z = 0u;
        if (i + 3 >= e) x.w = 0u;
        const int c = __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w);
        int incl = c;
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, off);
            if (lane >= off) incl += y;
        }
        int p = base + incl - c;
        base += __shfl_sync(kFull, incl, 31);
        if (!c) continue;
        if (p + c > a.cap) {
            atomicOr(a.err, kErrList);
            continue;
        }
        const uint32_t rk = *reinterpret_cast<const uint32_t*>(wrank + i);  // ranks of the four words
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
            const uint32_t key0 = (((rk >> (8 * q)) & 31u) << kIdBits) | ((uint32_t)(i + q) << 5);
#pragma unroll 1
            for (uint32_t y = x.x; y; y &= y - 1) out[p++] = key0 | (uint32_t)(__ffs(y) - 1);
            x.x = x.y;
            x.y = x.z;
            x.z = x.w;
        }
    }
    return meta_pack(S, kappa, top, false);
}

// Highest rank among the members of the old list (size, level and form in
// `old`) that are not in the new union, where every member of rank >= the new
// level (<= the old one) is kept; -1 if none left.
__device__ __forceinline__ int lost_rank(const LevelArgs& a, const UnionShared& sh, const uint32_t* tab,
                                         bool bm, int W0, const uint8_t* wrank,
                                         const uint32_t* old_list, uint32_t old) {
    const int tid = threadIdx.x;
    int r = -1;
    if (old & kMetaDense) {
        const int W = bm ? min(sh.cls[meta_k(old)], W0) : sh.cls[meta_k(old)];
#pragma unroll 1
        for (int i = tid; i < W; i += kLuThreads) {
            uint32_t x = old_list[i];
            if (!x) continue;
            const int rw = wrank[i];
            if (rw <= r) break;  // the ranks of the words only fall
            if (bm) {
                if (x & ~tab[i]) r = rw;
            } else {
                for (; x; x &= x - 1)
                    if (!set_contains(tab, a.lg, ((uint32_t)rw << kIdBits) | ((uint32_t)i << 5) |
                                                     (uint32_t)(__ffs(x) - 1)))
                        r = rw;
            }
        }
    } else {
        const int m = min(meta_size(old), (int)a.cap);
#pragma unroll 1
        for (int p = tid; p < m; p += kLuThreads) {
            const uint32_t key = old_list[p];
            const int rk = (int)(key >> kIdBits);
            if (rk <= r) break;  // the ranks of the list only fall
            const int w = (int)((key & kIdMask) >> 5);
            const bool in = bm ? w < W0 && ((tab[w] >> (key & 31u)) & 1u) : set_contains(tab, a.lg, key);
            if (!in) r = rk;
        }
    }
    return r;
}

// Levels >= 2, one CTA of 128 threads per node.
//
// The set of distinct members is a bitmap over positions in shared memory
// when the words of the ranks >= t0 (t0 = max k[w,i-1], where the union
// starts) fit, else an open-addressing hash set of keys.  In the bitmap an
// insert is one shared load and, when new, one atomic OR: no probing, no list
// of used slots and no compaction, and the output is in rank order by itself.
// The neighbours' meta words are read once per chunk of 128 into shared
// memory and sorted into buckets by what a list will give (walk_chunk).
//
// Heavy nodes (degree > kSplitDeg) are split: part j unions the lists of
// neighbours [j kSplitChunk, (j+1) kSplitChunk) into its own trimmed partial
// set, and the CTA that finishes a node's last part merges the partial sets.
// The merge is exact: a part's level t_p (max of its neighbours' k[w,i-1] and
// its own trim) is at most the node's final level kappa, because adding lists
// only raises the counts S_j; so every member of B[v,i] (rank >= kappa) is in
// some partial set, and for j >= t* = max_p t_p the counts S_j of the union of
// the partial sets equal those of the full union.  The merge therefore runs the
// same running-threshold union over the partial sets from t = t*.
//
// What bounds it: instruction issue on whole-graph passes (81% issue-active on
// the Chung-Lu n = 200k level-2 pass, 2.25 ms), latency in the rounds, whose
// launches are a few nodes per CTA.  A node is a chain of dependent loads (its
// row, the meta words, the lists) with little work between, so 12 CTAs of 128
// threads and 16 KB (M <= 1638) keep 12 nodes per SM in flight; 256 threads
// x 6 or 64 x 16 took 10-30% longer, and so did 25 KB of shared memory, which
// would hold a bitmap of all 200k positions, with 8 CTAs.
// Measured (start: one 256-thread CTA per node, hash set, 27 KB): estimates of
// R-MAT 22 at h = 3 251 -> 78 ms, (k,3)-core of Chung-Lu n = 200k 1080 -> 659 ms,
// (k,2)-core of Chung-Lu n = 50k at M = 1200 919 -> 538 ms (503 and 328 ms since the
// marking is spread over the warps, rounds have fewer kernels and heavy nodes smaller
// parts).  A warp per light node with a private quarter of the table gave nothing on
// the estimates (79.9 ms) and cost 30% in the rounds.
//
// LAST: nodes at their last level (estimate, refine); LIST: nodes below it
// (stored lists); PARTS: the parts of the split nodes, planned by the kernel that
// made the list (whole passes: by the launch before).  One kernel for all of it runs out of the instruction cache.
template <bool LAST, bool LIST, bool PARTS>
__global__ void __launch_bounds__(kLuThreads, kLuPerSm) k_levelU(LevelArgs a) {
    extern __shared__ __align__(16) uint32_t tab[];
    __shared__ UnionShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t total = PARTS        ? min((int64_t)(*a.plan.n_sub), a.plan.cap)
                          : a.worklist ? (int64_t)(*a.d_count)
                                       : a.count_static;
    // the first items go by block index, so that a short list costs the other
    // blocks neither a counter nor a table
    if (blockIdx.x >= total) return;
    unsigned long long my_bytes = 0;
    // the table starts empty once per launch; every node leaves it empty again
#pragma unroll 1
    for (int i = tid * 4; i < (1 << a.lg); i += kLuThreads * 4)
        *reinterpret_cast<uint4*>(tab + i) = make_uint4(0u, 0u, 0u, 0u);
    // the CTA's next item: a node, or (PARTS) a part of a split node
    const int* items = PARTS ? a.plan.sub_v : a.worklist;
    if (tid == 0) {
        sh.idx = blockIdx.x;
        sh.v = items ? items[blockIdx.x] : (int)blockIdx.x;
    }
    int cls_graph = -1;
    for (;;) {
        __syncthreads();
        const int64_t idx = sh.idx;
        if (idx >= total) break;
        // mode 0: a whole node; 1: one part of a split node (2: its merge)
        int mode = PARTS ? 1 : 0;
        const int v = sh.v, part = PARTS ? a.plan.sub_j[idx] : 0;
        int next = 0;
        if (tid == 0) next = (int)gridDim.x + atomicAdd(a.work_ctr, 1);
        bool skip = PARTS && v < 0;  // a part the plan could not place
        NodeLevel nl{};
        int64_t b = 0;
        int deg = 0;
        uint32_t kv = 0;
        int g = 0;
        if (!skip) {
            nl = node_level(a, v);
            b = a.rowptr[v];
            deg = (int)(a.rowptr[v + 1] - b);
            kv = a.key32[v];
            g = a.gid ? a.gid[v] : 0;
            skip = a.alive[v] != 1 || nl.skip || nl.lvl < 2 || (!LIST && !nl.last) || (!LAST && nl.last);
            if (!PARTS && !skip && a.plan.cap > 0 && deg > kSplitDeg) {
                // a heavy node is done in parts by the launch that follows (a round's
                // lists hold none)
                skip = true;
                if (tid == 0) plan_parts(a.plan, v, deg);
            }
        }
        if (skip) {
            __syncthreads();
            if (tid == 0) {
                sh.idx = next;
                if (next < total) sh.v = items ? items[next] : next;
            }
            continue;
        }
        const int rv = (int)(kv >> kIdBits);
        const bool last = LAST && (!LIST || nl.last);
        const int first = PARTS && mode ? a.plan.split_first[v] : -1;
        const int nparts = (deg + kSplitChunk - 1) / kSplitChunk;
        const uint8_t* wrank = a.wrank + (a.gid ? word_base(a.vtx_off[g], g) : 0);
        if (g != cls_graph) {
            if (tid < 33) sh.cls[tid] = a.clsw[(size_t)g * 33 + tid];
            cls_graph = g;
        }
        // A node's level never rises as nodes leave, and mostly stays: start one
        // below its last known level.  If the union then holds more than M at that
        // level, the level is the old one; if not, the node is done again from t0.
        const uint32_t last_meta = !PARTS || mode == 0 ? nl.meta_out[v] : 0u;
        int t_spec = last_meta & kMetaAlive ? meta_k(last_meta) - 1 : -1;
        for (;;) {  // a node's last part continues as its merge (mode 2)
            // lists: neighbours [l0, l1) (modes 0, 1) or partial sets [0, nparts) (mode 2)
            const int l0 = PARTS && mode == 1 ? part * kSplitChunk : 0;
            const int l1 = !PARTS || mode == 0 ? deg : (PARTS && mode == 1 ? min(deg, l0 + kSplitChunk) : nparts);
            const int L = l1 - l0;
            // t starts at max k[w,i-1] over alive neighbours (Prop. 3.1), or at
            // the largest level of the partial sets (merge)
            int w0 = 0;
            uint32_t m0 = 0;
            int myk = 0;
#pragma unroll 1
            for (int li = l0 + tid; li < l1; li += kLuThreads) {
                uint32_t m;
                int32_t w;
                if (PARTS && mode == 2) {
                    w = li;
                    m = __ldcg(a.part_meta + first + li);
                } else {
                    w = a.col[b + li];
                    m = nl.meta_in[w];
                }
                if (li == l0 + tid) {
                    w0 = w;
                    m0 = m;
                }
                myk = max(myk, meta_k(m));  // a removed neighbour's word is zero
            }
            myk = __reduce_max_sync(kFull, myk);
            if (lane == 0) sh.kmax[warp] = myk;
            if (tid < 32) sh.hist[tid] = 0;
            if (tid < kBuckets) {
                sh.nq[tid] = 0;
                sh.cq[tid] = 0;
            }
            if (tid == 0) {
                sh.exit = 0;
                sh.creq = 0;
                sh.part = 0;
                unsigned long long T = ~0ull;
                if (a.stop_c && last && !(PARTS && mode == 2))
                    T = stop_level(a.stop_c[g] > a.stop_mu[g] ? a.stop_c[g] : a.stop_mu[g]);
                sh.T = T;
            }
            __syncthreads();
            int t0 = sh.kmax[0];
#pragma unroll
            for (int i = 1; i < kLuWarps; ++i) t0 = max(t0, sh.kmax[i]);
            // (a refine that may stop early starts at t0: its partial estimate
            // needs the low ranks)
            const bool guess = t_spec > t0 && (sh.T == ~0ull || a.est[v] <= sh.T);
            if (guess) t0 = t_spec;
            const bool bm = sh.cls[t0] <= a.bm_words;
            const int W0 = sh.cls[t0];
            const bool vin = rv >= t0;
            if (tid == 0) {
                sh.t = t0;
                sh.tot = sh.used = vin ? 1 : 0;
                if (vin) {
                    if (bm) tab[(kv & kIdMask) >> 5] = 1u << (kv & 31u);
                    else set_insert(tab, a.lg, kv, a.err);
                    sh.hist[rv] = 1;
                }
            }
            UnionCtx c;
            c.tab = tab;
            c.lists = PARTS && mode == 2 ? a.part_keys + (size_t)first * (size_t)a.cap : nl.keys_in;
            c.wrank = wrank;
            c.cap = a.cap;
            c.lg = a.lg;
            c.M = nl.M;
            c.rv = rv;
            c.can_stop = sh.T != ~0ull;
            c.stop_first = PARTS && mode == 1 && c.can_stop ? first : -1;
            c.vin = vin;
            c.hash = !bm;
            c.other = PARTS && mode == 2;
            c.part_stop = a.part_stop;
            c.err = a.err;
            for (int c0 = l0; c0 < l1; c0 += kLuThreads) {
                if (c0 > l0) {
                    __syncthreads();  // the previous chunk's lists are read
                    if (sh.exit) break;
                    if (tid < kBuckets) {
                        sh.nq[tid] = 0;
                        sh.cq[tid] = 0;
                    }
                    const int li = c0 + tid;
                    m0 = 0;
                    if (li < l1) {
                        w0 = PARTS && mode == 2 ? li : a.col[b + li];
                        m0 = PARTS && mode == 2 ? __ldcg(a.part_meta + first + li) : nl.meta_in[w0];
                    }
                    __syncthreads();
                }
                // a list whose highest rank is below t has nothing to give
                const int t = c0 > l0 ? sh.t : t0;
                int bk = -1;
                if (c0 + tid < l1 && (m0 & kMetaAlive) && meta_size(m0) > 0 && meta_top(m0) >= t) {
                    // expected keys at or above t: ranks halve per level
                    const int ex = meta_size(m0) >> (t - meta_k(m0)) >> a.group_shift;
                    bk = m0 & kMetaDense ? kDense : !a.group_lists || ex > 64 ? kLong : ex > 8 ? kMiddle : kShort;
                    sh.w[tid] = w0;
                    sh.sz[tid] = (uint16_t)min(meta_size(m0), (int)a.cap);
                }
#pragma unroll
                for (int q = 0; q < kBuckets; ++q) {
                    const uint32_t mq = __ballot_sync(kFull, bk == q);
                    if (!mq) continue;
                    int base = 0;
                    if (lane == 0) base = atomicAdd(&sh.nq[q], __popc(mq));
                    base = __shfl_sync(kFull, base, 0);
                    if (bk == q) sh.q[q][base + __popc(mq & ((1u << lane) - 1u))] = (uint8_t)tid;
                }
                __syncthreads();
                int bucket = kBuckets - 1, li = -1, pos = 0;
                // a compaction keeps at most M keys, well under the trigger, so every
                // pass reads on; a bound no correct run reaches ends the union
                for (int pass = 0;; ++pass) {
                    walk_chunk<LAST, PARTS>(c, sh, bucket, li, pos, my_bytes);
                    if (bm) break;
                    __syncthreads();
                    if (!sh.creq || sh.exit) break;
                    if (pass > kLuThreads * (kMaxM / kKeysPerLane + 4)) {
                        if (tid == 0) atomicOr(a.err, kErrLoop);
                        break;
                    }
                    compact_set(a, sh, tab, nl.M);
                }
            }
            // the next item's node, while the last lists are read
            int nv = 0;
            if (tid == 0 && next < total) nv = items ? items[next] : next;
            __syncthreads();
            const bool stopped = LAST && sh.exit != 0;
            const int Sl = snapshot_counts(sh.hist, lane);
            const uint32_t over = __ballot_sync(kFull, Sl > nl.M);
            const int kappa = max(sh.t, over ? 32 - __clz(over) : 0);
            const int Sk = __shfl_sync(kFull, Sl, kappa & 31);
            const int S = kappa < 32 ? Sk : 0;
            const uint32_t nz = __ballot_sync(kFull, Sl > 0);
            const int top = nz && 31 - __clz(nz) >= kappa ? 31 - __clz(nz) : 0;
            const int lists_bytes = 8 * L;  // columns and meta words
            bool merge = false, lost = false;
            const bool redo = guess && !stopped && kappa == t0;  // the level fell
            uint32_t meta = 0;
            if (!stopped && !redo && ((PARTS && mode == 1) || !last)) {
                // the list of the node, or of the part
                uint32_t* out = PARTS && mode == 1 ? a.part_keys + (size_t)(first + part) * (size_t)a.cap
                                          : nl.keys_out + (size_t)v * (size_t)a.cap;
                if (a.track && !(PARTS && mode == 1)) {
                    const uint32_t old = nl.meta_out[v];
                    lost = meta_size(old) != S || meta_k(old) != kappa;
                    if (lost) {
                        if (tid == 0) sh.rho = kappa != meta_k(old) ? meta_k(old) - 1 : -1;
                        const int r = __reduce_max_sync(
                            kFull, lost_rank(a, sh, tab, bm, W0, wrank, out, old));
                        __syncthreads();  // the old list is read before it is overwritten
                        if (lane == 0 && r >= 0) atomicMax(&sh.rho, r);
                        __syncthreads();
                    }
                }
                meta = write_list(a, sh, tab, bm, wrank, out, S, kappa, top);
            }
            if (redo) {
                t_spec = -1;
            } else if (PARTS && mode == 1) {
                // a part: its partial set, or (refine) the estimate above T that
                // it already shows; the node's last part finishes it
                if (stopped) {
                    if (tid == 0) {
                        if (sh.exit == 1) atomicMax(a.part_lb + first, sh.part);
                        a.part_stop[first] = 1;
                    }
                } else if (tid == 0) {
                    a.part_meta[first + part] = meta;
                }
                if (tid == 0) my_bytes += lists_bytes;
                __threadfence();
                __syncthreads();
                if (tid == 0) sh.last = atomicAdd(a.part_done + first, 1) == nparts - 1;
                __syncthreads();
                if (sh.last) {
                    __threadfence();  // the other parts' sets are visible from here on
                    if (__ldcg(a.part_stop + first)) {
                        // some part showed d(v) > T: v stays stale with that lower bound
                        __syncthreads();  // every thread has read the flag
                        if (tid == 0) {
                            a.lb[v] = __ldcg(a.part_lb + first);
                            a.fresh[v] = 0;
                            atomicAdd(a.stopped, 1ull);
                            a.part_stop[first] = 0;
                            a.part_lb[first] = 0;
                            a.part_done[first] = 0;
                        }
                    } else {
                        merge = true;
                    }
                }
            } else if (stopped) {
                // d(v) > T: v stays stale, its lower bound raised to the partial estimate
                if (tid == 0) {
                    a.lb[v] = sh.part;
                    a.fresh[v] = 0;
                    atomicAdd(a.stopped, 1ull);  // a lower bound only: not an update
                    my_bytes += 17ull + lists_bytes;
                }
            } else if (last) {
                if (tid == 0) {
                    const unsigned long long est = estimate_of(S, kappa, rv, nl.M);
                    a.est[v] = est;
                    if (a.min_done) atomicMin(a.min_done + g, est);
                    record_change(a, nl, v, meta_pack(S, kappa, top, false) | kMetaFresh);
                    atomicAdd(a.updates, 1ull);
                    my_bytes += 21ull + (!PARTS || mode == 0 ? lists_bytes : 0);
                }
            } else {
                if (tid == 0) {
                    if (lost) a.rho[v] = (int8_t)sh.rho;
                    record_change(a, nl, v, meta);
                    my_bytes += 13ull + (!PARTS || mode == 0 ? lists_bytes : 0) + 4ull * (unsigned long long)S;
                }
            }
            __syncthreads();  // the table and the shared state are read
            const int clear = bm ? W0 : 1 << a.lg;
#pragma unroll 1
            for (int i = tid * 4; i < clear; i += kLuThreads * 4)
                *reinterpret_cast<uint4*>(tab + i) = make_uint4(0u, 0u, 0u, 0u);
            if (PARTS && mode == 2 && tid == 0) a.part_done[first] = 0;  // ready for the next launch
            if (merge || redo) {
                if (merge) mode = 2;
                __syncthreads();
                continue;
            }
            if (tid == 0) {
                sh.idx = next;
                sh.v = nv;
            }
            break;
        }
    }
    for (int off = 16; off > 0; off >>= 1) my_bytes += __shfl_down_sync(kFull, my_bytes, off);
    if (lane == 0 && my_bytes) atomicAdd(a.bytes, my_bytes);
}

// Rank filter for the neighbours of changed lists.  Level i of u is the
// rank filter (Prop. 3.1) of the union of its neighbours' level i-1 lists at
// k[u,i]; if every change of a neighbour's list (members that left, or members
// that entered below its old level) ranks below k[u,i] - 1, the counts S_j for
// j >= k[u,i] - 1, the level and the members are all unchanged.  The test needs
// k[u,i] for the current node set: intermediate levels always have it, a last
// level only while u is fresh.
struct MarkArgs {
    const int64_t* rowptr;
    const int32_t* col;
    const uint32_t* meta;  // meta words of level `phase`
    int32_t* seen;
    const int32_t* list1;
    const int* nlist1;
    const int32_t* list2;  // may be nullptr; rank-filtered by rho
    const int* nlist2;
    const int8_t* rho;
    const uint8_t* hv;     // per-node h (batches) or nullptr
    int h;
    int phase;
    int32_t* wl;
    int* nwl;
    int64_t cap;
    const DevState* st;
    unsigned long long* bytes;
    RoundEnd end;          // phase 1: the round's c and minima advance here
    PartPlan plan;         // heavy nodes that would be listed
    // STALE: nodes whose last level is `phase` become stale instead of listed
    uint32_t* meta_last;   // = meta, writable
    const uint32_t* prev;  // meta words of level phase - 1 (nullptr at phase 1)
    const uint32_t* key32;
    const int32_t* bestnb;
    const int32_t* Mv;
    int64_t M;
    uint8_t* fresh;
    unsigned long long* lb;
};

// (The CTA-wide path of the row kernels below: rows longer than kWarpRow are
// gathered per block and done by all its warps after the warp-per-node pass.)
constexpr int kWarpRow = 2048;
constexpr int kBlockHeavy = 64;
constexpr int kMarkWarps = 32;  // most warps on one listed node

__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) {
    return a > b ? a : b;
}

// Alg. 1 on a list (its meta word), with the node of rank r_first counted
// first (it is a member of the list's neighbourhood).
__device__ __forceinline__ unsigned long long est_first(uint32_t m, int r_first, int64_t M) {
    return estimate_of(meta_size(m), meta_k(m), r_first, M);
}

// Mark u (alive, its last level is the phase; m: that level's meta word) stale
// and give it a lower bound of its estimate: N(u; h-1) and, for an alive
// neighbour w, N(w; h-1) (which contains u) are inside N(u; h); Alg. 1 on either
// with u's rank first is at most the estimate of N(u; h) (Prop. 4.2).  Only
// the level-(h-1) meta words are read.  The neighbour term comes from the
// neighbour of largest degree (bestnb) while that is alive, else from the first
// kStaleScan entries of the row: any alive neighbours give a lower bound
// (scanning rows of up to 64 entries each time gave no fewer refines that count:
// 577 -> 569 ms without on Chung-Lu n = 200k, h = 3).
constexpr int kStaleScan = 64;
__device__ __forceinline__ void make_stale(const MarkArgs& a, int32_t u, uint32_t m) {
    unsigned long long lb = 0;
    if (a.prev) {
        const int64_t M = a.Mv ? (int64_t)a.Mv[u] : a.M;
        const int ru = (int)(a.key32[u] >> kIdBits);
        const int32_t w = a.bestnb[u];
        lb = est_first(a.prev[u], ru, M);
        const uint32_t mw = w >= 0 ? a.prev[w] : 0u;
        if (mw & kMetaAlive) {
            lb = umax64(lb, est_first(mw, ru, M));
        } else {
            const int64_t b = a.rowptr[u];
            const int n = (int)min((int64_t)kStaleScan, a.rowptr[u + 1] - b);
#pragma unroll 1
            for (int k = 0; k < n; ++k) {
                const uint32_t mk = a.prev[a.col[b + k]];
                if (mk & kMetaAlive) lb = umax64(lb, est_first(mk, ru, M));
            }
        }
    }
    a.lb[u] = lb;
    a.fresh[u] = 0;
    a.meta_last[u] = m & ~kMetaFresh;
}

// Row entries k0 + 32 q + lane, q < 4, of a listed node (rho rw; -128: no
// filter): each alive neighbour that passes joins wl once per stamp.  The stamp
// is read first: most entries of a round's rows are repeats.  meta holds the
// rest: alive, k, and at the last level whether k is current.
template <bool STALE>
__device__ __forceinline__ void mark_step(const MarkArgs& a, int rw, int stamp, int64_t k0, int64_t e,
                                          int lane) {
    int32_t u[4];
    bool go[4];
    uint32_t m[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t k = k0 + 32 * q + lane;
        u[q] = k < e ? a.col[k] : -1;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) go[q] = u[q] >= 0 && *(volatile int32_t*)(a.seen + u[q]) != stamp;
#pragma unroll
    for (int q = 0; q < 4; ++q) m[q] = go[q] ? a.meta[u[q]] : 0u;
    int n = 0;
    uint32_t isnew[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        go[q] = (m[q] & kMetaAlive) != 0;
        if (go[q] && rw > -128) {
            const int hu = a.hv ? (int)a.hv[u[q]] : a.h;
            const bool known = a.phase < hu || (m[q] & kMetaFresh);
            go[q] = !known || rw >= meta_k(m[q]) - 1;
        }
        if (go[q]) go[q] = atomicExch(a.seen + u[q], stamp) != stamp;
        if (STALE && go[q] && (!a.hv || (int)a.hv[u[q]] == a.phase)) {
            make_stale(a, u[q], m[q]);
            go[q] = false;
        }
        if (go[q] && a.plan.cap > 0)
            go[q] = !plan_parts(a.plan, u[q], a.rowptr[u[q] + 1] - a.rowptr[u[q]]);
        isnew[q] = __ballot_sync(kFull, go[q]);
        n += __popc(isnew[q]);
    }
    if (!n) return;
    int base = 0;
    if (lane == 0) base = atomicAdd(a.nwl, n);
    base = __shfl_sync(kFull, base, 0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (go[q]) {
            const int p = base + __popc(isnew[q] & ((1u << lane) - 1u));
            if (p < a.cap) a.wl[p] = u[q];
        }
        base += __popc(isnew[q]);
    }
}

// Alive neighbours of the listed nodes (two lists, the second optional and
// rank-filtered) join the work list once per stamp (round, phase).  A short list
// is spread over all warps, several to a node: one warp walking a row of 1000
// entries in 40 dependent steps was the length of the launch (52 us a round on
// the (k,2)-core of Chung-Lu n = 50k under events, 10 us so; that core 538 -> 368
// ms, the (k,3)-core of R-MAT 18 297 -> 246 ms).
template <bool STALE>
__global__ void k_mark_nbrs(MarkArgs a) {
    if (blockIdx.x == 0) end_round(a.end);
    __shared__ int s_heavy[kBlockHeavy];
    __shared__ int s_nheavy;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n1 = *a.nlist1;
    const int nin = n1 + (a.list2 ? *a.nlist2 : 0);
    const int stamp = a.st->round * kPhaseStride + a.phase;
    const int nw = (int)((gridDim.x * blockDim.x) >> 5);
    const int wid = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int per = nin > 0 ? min(kMarkWarps, max(1, nw / nin)) : 1;  // warps per node
    unsigned long long my_bytes = 0;
    if (threadIdx.x == 0) s_nheavy = 0;
    __syncthreads();
    for (int i = wid / per; i < nin; i += nw / per) {
        if (wid / per >= nw / per) break;  // the warps past the last whole group
        const int sub = wid % per;
        const int w = i < n1 ? a.list1[i] : a.list2[i - n1];
        const int64_t b = a.rowptr[w], e = a.rowptr[w + 1];
        if (e - b > (int64_t)kWarpRow * per) {
            int slot = kBlockHeavy;
            if (lane == 0 && per == 1) slot = atomicAdd(&s_nheavy, 1);
            slot = __shfl_sync(kFull, slot, 0);
            if (slot < kBlockHeavy) {
                if (lane == 0) s_heavy[slot] = i;
                continue;
            }
        }
        const int rw = a.rho && i >= n1 ? (int)a.rho[w] : -128;
        if (lane == 0 && sub == 0) my_bytes += 12ull + 4ull * (unsigned long long)(e - b);
        for (int64_t k0 = b + sub * 128; k0 < e; k0 += per * 128) mark_step<STALE>(a, rw, stamp, k0, e, lane);
    }
    __syncthreads();
    const int nh = min(s_nheavy, kBlockHeavy);
    for (int j = 0; j < nh; ++j) {
        const int i = s_heavy[j];
        const int w = i < n1 ? a.list1[i] : a.list2[i - n1];
        const int rw = a.rho && i >= n1 ? (int)a.rho[w] : -128;
        const int64_t b = a.rowptr[w], e = a.rowptr[w + 1];
        if (threadIdx.x == 0) my_bytes += 12ull + 4ull * (unsigned long long)(e - b);
        for (int64_t k0 = b + warp * 128; k0 < e; k0 += 4 * blockDim.x) mark_step<STALE>(a, rw, stamp, k0, e, lane);
    }
    for (int off = 16; off > 0; off >>= 1) my_bytes += __shfl_down_sync(kFull, my_bytes, off);
    if (lane == 0 && my_bytes) atomicAdd(a.bytes, my_bytes);
}

// Start of a peel: every alive node stale (make_stale), whatever its last level.
__global__ void k_stale_all(MarkArgs a, int64_t n, const uint8_t* __restrict__ alive, uint32_t* meta) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        if (alive[v] != 1) continue;
        const int h = a.hv ? (int)a.hv[v] : a.h;
        a.meta_last = meta + (size_t)(h - 1) * (size_t)n;
        a.prev = h >= 2 ? meta + (size_t)(h - 2) * (size_t)n : nullptr;
        make_stale(a, (int32_t)v, a.meta_last[v]);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(a.bytes, 38ull * (unsigned long long)n);
}

}  // namespace

namespace {
// Part slots a whole-graph level pass needs: ceil(deg / kSplitChunk) per node
// of degree above kSplitDeg (out[0]); the nodes above kSplitMin (out[1]).
__global__ void k_count_parts(const int64_t* __restrict__ rowptr, int64_t n,
                              unsigned long long* out) {
    unsigned long long c = 0, big = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int64_t deg = rowptr[v + 1] - rowptr[v];
        if (deg > kSplitDeg) c += (unsigned long long)((deg + kSplitChunk - 1) / kSplitChunk);
        big += deg > kSplitMin;
    }
    for (int off = 16; off > 0; off >>= 1) {
        c += __shfl_down_sync(kFull, c, off);
        big += __shfl_down_sync(kFull, big, off);
    }
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
    if ((threadIdx.x & 31) == 0 && big) atomicAdd(out + 1, big);
}
}  // namespace

int ensure_split(Graph& g) {
    cudaStream_t s = g.ctx->stream;
    if (!g.split_planned) {
        unsigned long long* d = nullptr;
        unsigned long long parts[2] = {0, 0};
        KH_CUDA_TRY(g.ctx, cudaMallocAsync((void**)&d, sizeof(parts), s));
        cudaError_t e = cudaMemsetAsync(d, 0, sizeof(parts), s);
        if (e == cudaSuccess && g.n > 0) {
            k_count_parts<<<g.ctx->sm_count * 4, 256, 0, s>>>(g.rowptr, g.n, d);
            count_launch(g, 1);
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(parts, d, sizeof(parts), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        cudaFreeAsync(d, s);
        if (e != cudaSuccess) return check_cuda(g.ctx, e, "count split parts");
        g.part_cap = parts[1] ? (int64_t)parts[0] : 0;
        g.split_planned = true;
    }
    if (g.part_cap == 0) return KH_OK;
    if (g.part_keys && g.part_cap_keys < g.cap) {
        KH_CUDA_TRY(g.ctx, cudaStreamSynchronize(s));
        cudaFree(g.part_keys);
        g.part_keys = nullptr;
    }
    int rc;
    if (!g.part_keys) {
        if ((rc = alloc_bytes(g.ctx, (void**)&g.part_keys,
                              sizeof(uint32_t) * (size_t)g.part_cap * (size_t)g.cap, "split part keys")))
            return rc;
        g.part_cap_keys = g.cap;
    }
    const size_t pc = (size_t)g.part_cap;
    if (!g.part_done) {
        if ((rc = alloc_bytes(g.ctx, (void**)&g.part_done, sizeof(int32_t) * pc, "split part counters")))
            return rc;
        KH_CUDA_TRY(g.ctx, cudaMemsetAsync(g.part_done, 0, sizeof(int32_t) * pc, s));
    }
    if (!g.part_stop) {
        if ((rc = alloc_bytes(g.ctx, (void**)&g.part_stop, sizeof(int32_t) * pc, "split stop flags")))
            return rc;
        KH_CUDA_TRY(g.ctx, cudaMemsetAsync(g.part_stop, 0, sizeof(int32_t) * pc, s));
    }
    if (!g.part_lb) {
        if ((rc = alloc_bytes(g.ctx, (void**)&g.part_lb, sizeof(unsigned long long) * pc,
                              "split lower bounds")))
            return rc;
        KH_CUDA_TRY(g.ctx, cudaMemsetAsync(g.part_lb, 0, sizeof(unsigned long long) * pc, s));
    }
    if (!g.part_meta && (rc = alloc_bytes(g.ctx, (void**)&g.part_meta, sizeof(uint32_t) * pc, "split part metas")))
        return rc;
    if (!g.sub_v && (rc = alloc_bytes(g.ctx, (void**)&g.sub_v, sizeof(int32_t) * pc, "split part nodes")))
        return rc;
    if (!g.sub_j && (rc = alloc_bytes(g.ctx, (void**)&g.sub_j, sizeof(int32_t) * pc, "split part indices")))
        return rc;
    if (!g.split_first &&
        (rc = alloc_bytes(g.ctx, (void**)&g.split_first, sizeof(int32_t) * (size_t)g.n, "split first slots")))
        return rc;
    return KH_OK;
}

namespace {
// Slots of the hash form: a compaction is due past half of them and leaves at
// most M <= 4/5 of that; until every warp has stopped for it, each may add two
// more steps of 128 keys (1024 in all, at most a quarter of the slots).
int table_lg(int64_t M) {
    int lg = 12;
    while ((int64_t(1) << lg) * 2 < 5 * M) ++lg;
    return lg;
}

// The bitmap form may use as many words as the hash form has slots; position
// classes are whole words only while the padded positions fit the key.
bool positions_aligned(const Graph& g) { return g.n + 1024 <= (int64_t)1 << kIdBits; }

// ---- positions: nodes numbered by descending rank ----------------------------
// Per graph and rank class: its nodes (pass 0), then its first position;
// pass 1 hands the positions out.  Counters are taken per warp and class.
__global__ void k_pos_pass(const uint8_t* __restrict__ rank, const int32_t* __restrict__ gid, int64_t n,
                           int* __restrict__ cnt, uint32_t* __restrict__ key32) {
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t nround = (n + 31) & ~(int64_t)31;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nround; u += stride) {
        const bool in = u < n;
        const uint32_t r = in ? rank[u] : 0;
        const uint32_t slot = in ? (uint32_t)(gid ? gid[u] : 0) * 32u + r : 0xffffffffu;
        const uint32_t peers = __match_any_sync(kFull, slot);
        const int lead = __ffs(peers) - 1;
        int base = 0;
        if (in && lane == lead) base = atomicAdd(cnt + slot, __popc(peers));
        base = __shfl_sync(kFull, base, lead);
        if (in && key32) key32[u] = (r << kIdBits) | (uint32_t)(base + __popc(peers & ((1u << lane) - 1u)));
    }
}

// One warp per graph: clsw from the class counts, the counts become each
// class's first position, wrank of the graph's words.
__global__ void k_pos_classes(int* __restrict__ cnt, int64_t ngraphs, const int64_t* __restrict__ vtx_off,
                              int32_t* __restrict__ clsw, uint8_t* __restrict__ wrank, int aligned) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < ngraphs; q += nw) {
        const int c = cnt[q * 32 + lane];
        const int size = aligned ? (c + 31) >> 5 : c;  // words, or (unaligned) positions
        int incl = size;                               // over the ranks >= lane
        for (int off = 1; off < 32; off <<= 1) {
            const int x = __shfl_down_sync(kFull, incl, off);
            if (lane + off < 32) incl += x;
        }
        const int above = incl - size;
        cnt[q * 32 + lane] = aligned ? above << 5 : above;
        clsw[q * 33 + lane] = aligned ? incl : 0x7fffffff;
        if (lane == 0) clsw[q * 33 + 32] = aligned ? 0 : 0x7fffffff;
        if (!aligned) continue;
        uint8_t* wr = wrank + word_base(vtx_off ? vtx_off[q] : 0, q);
        for (int r = 0; r < 32; ++r) {
            const int w0 = __shfl_sync(kFull, above, r), w1 = __shfl_sync(kFull, incl, r);
            for (int w = w0 + lane; w < w1; w += 32) wr[w] = (uint8_t)r;
        }
    }
}
}  // namespace

// Ranks, and what the sampled path derives from them and from M.
int ensure_positions(Graph& g) {
    cudaStream_t s = g.ctx->stream;
    const int64_t ng = g.gid ? g.ngraphs : 1;
    int rc;
    if (!g.ranks_valid) {
        launch_ranks(g, s);
        g.ranks_valid = true;
        g.pos_valid = false;
    }
    if (!g.key32 && (rc = alloc_bytes(g.ctx, (void**)&g.key32, sizeof(uint32_t) * (size_t)g.n, "positions")))
        return rc;
    if (!g.clsw && (rc = alloc_bytes(g.ctx, (void**)&g.clsw, sizeof(int32_t) * 65 * (size_t)ng, "rank classes")))
        return rc;
    if (!g.wrank && (rc = alloc_bytes(g.ctx, (void**)&g.wrank, (size_t)word_base(g.n, ng) + 4, "word ranks")))
        return rc;
    // compaction stage of the hash form, one slot per CTA of k_levelU (nodes; parts)
    if (g.lu_stage && g.lu_stage_cap < g.cap) {
        KH_CUDA_TRY(g.ctx, cudaStreamSynchronize(s));
        cudaFree(g.lu_stage);
        g.lu_stage = nullptr;
    }
    if (!g.lu_stage) {
        if ((rc = alloc_bytes(g.ctx, (void**)&g.lu_stage,
                              sizeof(uint32_t) * 2 * (size_t)g.ctx->sm_count * kLuPerSm * (size_t)g.cap, "union stage")))
            return rc;
        g.lu_stage_cap = g.cap;
    }
    if (g.pos_valid || g.n == 0) return KH_OK;
    int* cnt = g.clsw + 33 * ng;  // 32 class counters per graph behind the table
    const int aligned = positions_aligned(g) ? 1 : 0;
    KH_CUDA_TRY(g.ctx, cudaMemsetAsync(cnt, 0, sizeof(int) * 32 * (size_t)ng, s));
    const int grid = (int)((g.n + 255) / 256 < g.ctx->sm_count * 8 ? (g.n + 255) / 256 : g.ctx->sm_count * 8);
    k_pos_pass<<<grid, 256, 0, s>>>(g.rank, g.gid, g.n, cnt, nullptr);
    k_pos_classes<<<(int)((ng + 7) / 8 < 1024 ? (ng + 7) / 8 : 1024), 256, 0, s>>>(cnt, ng, g.vtx_off, g.clsw,
                                                                                  g.wrank, aligned);
    k_pos_pass<<<grid, 256, 0, s>>>(g.rank, g.gid, g.n, cnt, g.key32);
    count_launch(g, 3);
    KH_CUDA_TRY(g.ctx, cudaGetLastError());
    g.pos_valid = true;
    return KH_OK;
}

int launch_level(Graph& g, int level, const int* worklist, const int* d_count,
                 int64_t count_static, int track, cudaStream_t s, int round_mode, int skip_last) {
    if (g.n == 0) return KH_OK;
    if (!worklist && count_static == 0) return KH_OK;
    LevelArgs a{};
    a.rowptr = g.rowptr;
    a.col = g.col;
    a.alive = g.alive;
    a.key32 = g.key32;
    a.clsw = g.clsw;
    a.wrank = g.wrank;
    a.vtx_off = g.vtx_off;
    a.n = g.n;
    a.level = round_mode == 2 ? 0 : level;  // the refine computes each node's last level
    a.h = g.h;
    a.hv = g.hv;
    a.skip_last = skip_last < 0 ? (round_mode == 1 ? 1 : 0) : skip_last;
    a.M = g.M;
    a.Mv = g.Mv;
    a.cap = g.cap;
    a.keys = g.keys;
    a.meta = g.meta;
    a.stage = g.lu_stage;
    a.est = g.d64;
    a.worklist = worklist;
    a.d_count = d_count;
    a.count_static = count_static;
    a.track = track;
    a.changed = g.listC[level & 1];
    a.err = &g.state->err;
    a.updates = &g.state->updates;
    const bool stop = round_mode == 2;
    a.stop_c = stop ? g.pc : nullptr;
    a.stop_mu = stop ? g.pmu : nullptr;
    a.gid = g.gid;
    a.lb = g.lb64;
    a.fresh = g.fresh;
    a.rho = g.rho;
    a.min_done = (round_mode == 2 && !g.dense) ? g.pmr : nullptr;
    a.lvl_work = g.state->lvl_work;
    a.lvl_changed = g.state->lvl_changed;
    a.stopped = &g.state->stopped;
    int* rc = g.state->rc;
    int* sub_ctr = nullptr;  // work counter of the parts launch
    if (round_mode == 1) {
        a.n_changed = rc + kRcC + level;
        a.work_ctr = rc + kRcLevelWork + level;
        sub_ctr = rc + kRcSubWork + level;
        a.plan = round_parts(g, level);
    } else if (round_mode == 2) {
        a.n_changed = rc + kRcC + 0;  // unused: the refine does not track changes
        a.work_ctr = rc + kRcRefineWork;
        sub_ctr = rc + kRcSubWork + 0;
        a.plan = round_parts(g, 0);
    } else {
        a.n_changed = &g.state->nC[level & 1];
        a.work_ctr = &g.state->work_ctr[1];
        a.plan = round_parts(g, 0);
        a.plan.n_sub = &g.state->nSub;
        sub_ctr = &g.state->work_ctr[3];
    }
    a.part_keys = g.part_keys;
    a.part_meta = g.part_meta;
    a.part_done = g.part_done;
    a.part_stop = g.part_stop;
    a.part_lb = g.part_lb;
    cudaError_t e;
    if (track && round_mode == 0) {
        e = cudaMemsetAsync(a.n_changed, 0, sizeof(int), s);
        if (e != cudaSuccess) return check_cuda(g.ctx, e, "memset n_changed");
    }
    const int64_t work = worklist ? g.n : count_static;
    // which kernels can have nodes to do: level 1 (warp per node) and/or >= 2 (CTA per node)
    const bool want1 = round_mode == 2 ? g.hmin == 1 : level == 1;
    const bool wantU = round_mode == 2 ? g.hmax >= 2 : level >= 2;
    if (want1) {
        a.bytes = &g.state->bytes[kProfLevel1];
        int64_t grid = (work + (kL1Threads / 32) - 1) / (kL1Threads / 32);
        const int64_t gmax = (int64_t)g.ctx->sm_count * 8;
        if (grid > gmax) grid = gmax;
        if (grid < 1) grid = 1;
        prof_begin(g, kProfLevel1, s);
        k_level1<<<(int)grid, kL1Threads, 0, s>>>(a);
        count_launch(g, 1);
        prof_end(g, kProfLevel1, s);
    }
    if (!wantU) return KH_OK;
    a.bytes = &g.state->bytes[kProfLevelU];
    a.lg = table_lg(g.M);
    a.bm_words = positions_aligned(g) ? 1 << a.lg : -1;
    const size_t dyn = (size_t)4 << a.lg;
    a.group_lists = g.levelu_mode == KH_VAR_AUTO || g.levelu_mode == KH_LEVELU_GROUPED;
    a.group_shift = 0;
    while ((1 << a.group_shift) < g.levelu_div) ++a.group_shift;
    // the nodes' last level only, stored lists only, or both (whole passes over a
    // batch of mixed h); with or without split nodes
    const bool any_last = round_mode == 2 || (!a.skip_last && level >= g.hmin);
    const bool any_list = round_mode != 2 && level < g.hmax;
    const bool parts = g.part_cap > 0;
    void (*kern)(LevelArgs) = any_last && any_list ? k_levelU<true, true, false>
                              : any_last           ? k_levelU<true, false, false>
                                                   : k_levelU<false, true, false>;
    void (*pkern)(LevelArgs) = any_last && any_list ? k_levelU<true, true, true>
                               : any_last           ? k_levelU<true, false, true>
                                                    : k_levelU<false, true, true>;
    // the largest table any graph can ask for (M up to kMaxM)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             4 << table_lg(kMaxM));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(pkern, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 << table_lg(kMaxM));
    if (e != cudaSuccess) return check_cuda(g.ctx, e, "cudaFuncSetAttribute(k_levelU)");
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kLuThreads, dyn);
    if (e != cudaSuccess) return check_cuda(g.ctx, e, "occupancy(k_levelU)");
    if (per_sm < 1) per_sm = 1;
    if (per_sm > kLuPerSm) per_sm = kLuPerSm;
    int64_t grid = (int64_t)g.ctx->sm_count * per_sm;
    if (work < grid) grid = work;
    if (grid < 1) grid = 1;
    if (round_mode == 0) {
        e = cudaMemsetAsync(a.work_ctr, 0, sizeof(int), s);
        if (e != cudaSuccess) return check_cuda(g.ctx, e, "memset work_ctr");
        if (parts) {
            e = cudaMemsetAsync(a.plan.n_sub, 0, sizeof(int), s);
            if (e == cudaSuccess) e = cudaMemsetAsync(sub_ctr, 0, sizeof(int), s);
            if (e != cudaSuccess) return check_cuda(g.ctx, e, "memset n_sub");
        }
    }
    prof_begin(g, kProfLevelU, s);
    if (parts && round_mode != 0) {
        // planned by the kernel that made the list: beside the other nodes
        LevelArgs pa = a;
        pa.work_ctr = sub_ctr;
        pa.stage = g.lu_stage + (size_t)g.ctx->sm_count * kLuPerSm * (size_t)g.cap;
        KH_CUDA_TRY(g.ctx, cudaEventRecord(g.ctx->fork, s));
        KH_CUDA_TRY(g.ctx, cudaStreamWaitEvent(g.ctx->side, g.ctx->fork, 0));
        pkern<<<g.ctx->sm_count * per_sm, kLuThreads, dyn, g.ctx->side>>>(pa);
        KH_CUDA_TRY(g.ctx, cudaEventRecord(g.ctx->join, g.ctx->side));
        a.plan.cap = 0;  // no heavy node in the list
    }
    kern<<<(int)grid, kLuThreads, dyn, s>>>(a);
    count_launch(g, 1);
    if (parts && round_mode != 0) {
        KH_CUDA_TRY(g.ctx, cudaStreamWaitEvent(s, g.ctx->join, 0));
        count_launch(g, 1);
    } else if (parts) {
        a.work_ctr = sub_ctr;
        pkern<<<g.ctx->sm_count * per_sm, kLuThreads, dyn, s>>>(a);
        count_launch(g, 1);
    }
    prof_end(g, kProfLevelU, s);
    return KH_OK;
}

PartPlan round_parts(const Graph& g, int level) {
    return {g.state->rc + kRcSub + level, g.sub_v, g.sub_j, g.split_first, g.part_cap, &g.state->err};
}

static MarkArgs mark_args(Graph& g, int phase) {
    MarkArgs a{};
    a.rowptr = g.rowptr;
    a.col = g.col;
    a.meta = a.meta_last = g.meta + (size_t)(phase - 1) * (size_t)g.n;
    a.prev = phase >= 2 ? g.meta + (size_t)(phase - 2) * (size_t)g.n : nullptr;
    a.seen = g.seen;
    a.hv = g.hv;
    a.h = g.h;
    a.phase = phase;
    a.cap = g.n;
    a.st = g.state;
    a.bytes = &g.state->bytes[kProfFrontier];
    a.key32 = g.key32;
    a.bestnb = g.bestnb;
    a.Mv = g.Mv;
    a.M = g.M;
    a.fresh = g.fresh;
    a.lb = g.lb64;
    return a;
}

void launch_mark_neighbours(Graph& g, const int* list1, const int* cnt1, const int* list2,
                            const int* cnt2, int phase, int* out_count, cudaStream_t s) {
    MarkArgs a = mark_args(g, phase);
    a.list1 = list1;
    a.nlist1 = cnt1;
    a.list2 = list2;
    a.nlist2 = cnt2;
    a.rho = list2 ? g.rho : nullptr;
    a.wl = g.listW;
    a.nwl = out_count;
    if (phase == 1) a.end = round_end(g);
    if (phase >= 2) a.plan = round_parts(g, phase);  // (level 1 is not a union)
    const int grid = g.ctx->sm_count * 8;
    prof_begin(g, kProfFrontier, s);
    if (phase >= g.hmin) k_mark_nbrs<true><<<grid, 256, 0, s>>>(a);
    else k_mark_nbrs<false><<<grid, 256, 0, s>>>(a);
    count_launch(g, 1);
    prof_end(g, kProfFrontier, s);
}

void launch_stale_all(Graph& g, cudaStream_t s) {
    if (g.n == 0) return;
    prof_begin(g, kProfFrontier, s);
    k_stale_all<<<g.ctx->sm_count * 8, 256, 0, s>>>(mark_args(g, 1), g.n, g.alive, g.meta);
    count_launch(g, 1);
    prof_end(g, kProfFrontier, s);
}

// lvl_out[v] = k[v, h(v)], bs_out[v] = |B[v, h(v)]| (each node's last level)
__global__ void k_gather_last(int64_t n, int h_all, const uint8_t* __restrict__ hv,
                              const uint32_t* __restrict__ meta, uint8_t* __restrict__ lvl_out,
                              int32_t* __restrict__ bs_out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int h = hv ? (int)hv[v] : h_all;
        const uint32_t m = meta[(size_t)(h - 1) * (size_t)n + (size_t)v];
        if (lvl_out) lvl_out[v] = (uint8_t)meta_k(m);
        if (bs_out) bs_out[v] = meta_size(m);
    }
}

// Start of a peel: no lists, every alive node's last-level word alive and stale.
__global__ void k_init_meta(int64_t n, int h_all, const uint8_t* __restrict__ hv,
                            const uint8_t* __restrict__ alive, uint32_t* __restrict__ meta) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int h = hv ? (int)hv[v] : h_all;
        if (alive[v] == 1) meta[(size_t)(h - 1) * (size_t)n + (size_t)v] = kMetaAlive;
    }
}

int launch_init_meta(Graph& g, cudaStream_t s) {
    KH_CUDA_TRY(g.ctx, cudaMemsetAsync(g.meta, 0, sizeof(uint32_t) * (size_t)g.hmax * (size_t)g.n, s));
    if (g.n == 0) return KH_OK;
    k_init_meta<<<g.ctx->sm_count * 4, 256, 0, s>>>(g.n, g.h, g.hv, g.alive, g.meta);
    count_launch(g, 1);
    return KH_OK;
}

void launch_gather_last(Graph& g, uint8_t* lvl_out, int32_t* bs_out, cudaStream_t s) {
    if (g.n == 0) return;
    k_gather_last<<<g.ctx->sm_count * 4, 256, 0, s>>>(g.n, g.h, g.hv, g.meta, lvl_out, bs_out);
    count_launch(g, 1);
}

}  // namespace kh
