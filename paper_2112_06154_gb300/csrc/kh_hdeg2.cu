// kh_hdeg2.cu -- exact 2-degrees of a whole graph: sliced shared-memory visited
// sets (k_hdeg2_slice, graphs whose n-bit visited set does not fit in shared
// memory), one CTA per source where it does (k_hdeg2_cta), and bit-parallel
// searches of many sources (k_sweep_*).
//
// Sec. 2: deg_2(v) = |N(v; 2)| - 1 with N(v; 2) = {v} U A(v) U (U_{w in A(v)} A(w)).
// For a node with at least one neighbour, v itself lies in A(w) for every w in
// A(v) (the graph is symmetric), so N(v; 2) is the union of the rows of v and
// of its neighbours.  The node range [0, n) is cut into S slices of `width`
// ids; one work item is (source v, slice s): a CTA marks, in a shared-memory
// bitmap of `width` bits, every member of those rows that falls in slice s
// (each row is sorted, so its part inside the slice is found by two searches)
// and adds the number of newly set bits to deg[v].  Each row entry is read
// once over the S items of a source, so the items of one source move the
// algorithmic bytes of one BFS.
//
// Sources are processed in decreasing order of their 2-hop work sum_{w in
// A(v)} deg(w) (longest first), so the large balls of hubs start early and the
// small ones fill the tail.  Isolated nodes (deg_2 = 0) are not items.
//
// The bitmap is cleared between items through the list of words the item set
// first (when it fits), otherwise with vector stores over the whole slice.
//
// Two more kernels serve the same pass: sources of small 2-hop work on one
// warp each with a private hash set (k_hdeg2_small), and, for the sources of
// the largest 2-hop work, bit-parallel sweeps of 1024 sources at a time
// (k_sweep_*; see the comment above them), which also serve h >= 3.
#include <cmath>
#include <vector>

#include "kh_internal.cuh"

namespace kh {

namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr int kMaxHeavy2 = 128;      // rows expanded by the whole CTA per item
constexpr int kHeavyRow2 = 512;      // a row part this long goes to the whole CTA
constexpr int kTouchCap = 4096;      // words cleared one by one (else full clear)
constexpr int kOrderBins = kOrderBinsMax;  // log2 bins of the 2-hop work

struct Slice2Args {
    const int64_t* rowptr;
    const int32_t* col;
    const uint8_t* rank;
    int64_t n;
    int nslices;
    int64_t width;        // nodes per slice (multiple of 128)
    const int32_t* order;  // sources, longest first
    int64_t nsrc;
    int32_t* deg;          // += marked nodes per item (starts at -1 / 0)
    int32_t* cnt;          // fixed-level counts (RANKS), += per item
    int jlo, nj;
    int* work_ctr;
    int* err;
    unsigned long long* updates;
    unsigned long long* bytes;
};

// First position p in [b, e) with col[p] >= key (e if none); the whole warp
// calls it and every lane gets the answer.  Each step samples 32 evenly spaced
// entries and keeps the gap where the sorted row crosses key.
__device__ __forceinline__ int64_t warp_lower_bound(const int32_t* __restrict__ col, int64_t b,
                                                    int64_t e, int32_t key, int lane) {
    // 32-bit offsets from b (a row has fewer than 2^31 entries)
    const int32_t* __restrict__ r = col + b;
    int lo = 0, hi = (int)(e - b);  // answer in [lo, hi]
    while (hi - lo > 32) {
        const int step = (hi - lo + 31) >> 5;
        const int p = lo + lane * step;
        const bool below = p < hi && __ldg(r + p) < key;
        const int c = __popc(__ballot_sync(kFull, below));
        // positions lo + j*step, j < c, hold keys below `key`
        const int nlo = c > 0 ? lo + (c - 1) * step + 1 : lo;
        const int nhi = lo + c * step;
        lo = nlo;
        hi = nhi < hi ? nhi : hi;
    }
    const int p = lo + lane;
    const bool below = p < hi && __ldg(r + p) < key;
    return b + lo + __popc(__ballot_sync(kFull, below));
}

// Mark u (in the slice) in the bitmap; count it and remember its word when it
// is the word's first bit.  All 32 lanes call this together.
template <bool RANKS>
__device__ __forceinline__ void mark(const Slice2Args& a, uint32_t* bm, int32_t* touch,
                                     int* s_ntouch, int* s_hist, bool valid, int32_t lu,
                                     int32_t u, int lane, int& my) {
    bool fresh_word = false;
    int word = 0;
    if (valid) {
        word = lu >> 5;
        const uint32_t bit = 1u << (lu & 31);
        if (!(*(volatile uint32_t*)(bm + word) & bit)) {
            const uint32_t old = atomicOr(bm + word, bit);
            if (!(old & bit)) {
                ++my;
                if (RANKS) atomicAdd(&s_hist[a.rank[u]], 1);
                fresh_word = old == 0u;
            }
        }
    }
    const uint32_t fm = __ballot_sync(kFull, fresh_word);
    if (fm) {
        const int leader = __ffs(fm) - 1;
        int base = 0;
        if (lane == leader) base = atomicAdd(s_ntouch, __popc(fm));
        base = __shfl_sync(kFull, base, leader);
        if (fresh_word) {
            const int p = base + __popc(fm & ((1u << lane) - 1u));
            if (p < kTouchCap) touch[p] = word;
        }
    }
}

// Mark the entries [ps, pe) of col, lanes take 32 consecutive entries and
// each step issues four independent loads per lane.
template <bool RANKS>
__device__ __forceinline__ void mark_range(const Slice2Args& a, uint32_t* bm, int32_t* touch,
                                           int* s_ntouch, int* s_hist, int64_t ps, int64_t pe,
                                           int64_t first, int64_t stride, int32_t lo, int lane,
                                           int& my) {
    // 32-bit offsets from the part's start (a row has fewer than 2^31 entries)
    const int32_t* __restrict__ base = a.col + ps;
    const int len = (int)(pe - ps);
    for (int k0 = (int)first; k0 < len; k0 += (int)stride) {
        int32_t u[4];
        bool val[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int k = k0 + q * 32 + lane;
            val[q] = k < len;
            u[q] = val[q] ? __ldg(base + k) : lo;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            mark<RANKS>(a, bm, touch, s_ntouch, s_hist, val[q], u[q] - lo, u[q], lane, my);
    }
}

template <bool RANKS>
__global__ void k_hdeg2_slice(Slice2Args a) {
    extern __shared__ __align__(16) uint32_t s_dyn[];
    const int words = (int)(a.width >> 5);
    uint32_t* bm = s_dyn;
    int32_t* touch = reinterpret_cast<int32_t*>(s_dyn + words);
    __shared__ int s_item, s_ntouch, s_nheavy, s_count, s_row;
    __shared__ int64_t s_hb[kMaxHeavy2], s_he[kMaxHeavy2];
    __shared__ int s_hist[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int64_t total = a.nsrc * a.nslices;
    unsigned long long my_bytes = 0;
    {
        uint4* b4 = reinterpret_cast<uint4*>(bm);
        for (int i = tid; i < (words >> 2); i += blockDim.x) b4[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
    for (;;) {
        if (tid == 0) {
            s_item = atomicAdd(a.work_ctr, 1);
            s_ntouch = 0;
            s_nheavy = 0;
            s_row = 0;
            s_count = 0;
        }
        if (RANKS && tid < 32) s_hist[tid] = 0;
        __syncthreads();
        const int64_t item = s_item;
        if (item >= total) break;
        const int v = a.order[item / a.nslices];
        const int sl = (int)(item % a.nslices);
        const int32_t lo = (int32_t)((int64_t)sl * a.width);
        const int64_t hi64 = (int64_t)lo + a.width;
        const int32_t hi = (int32_t)(hi64 < a.n ? hi64 : a.n);
        const int64_t vb = a.rowptr[v], ve = a.rowptr[v + 1];
        const int64_t deg = ve - vb;
        int my = 0;
        // rows: v's own (i == deg) and each neighbour's (i < deg), claimed by
        // the warps one at a time (row lengths vary widely)
        for (;;) {
            int64_t i = 0;
            if (lane == 0) i = atomicAdd(&s_row, 1);
            i = __shfl_sync(kFull, i, 0);
            if (i > deg) break;
            const int32_t x = i < deg ? __ldg(a.col + vb + i) : v;
            const int64_t rb = a.rowptr[x], re = a.rowptr[x + 1];
            const int64_t ps = lo > 0 ? warp_lower_bound(a.col, rb, re, lo, lane) : rb;
            const int64_t pe = hi < a.n ? warp_lower_bound(a.col, ps, re, hi, lane) : re;
            if (lane == 0) my_bytes += (sl == 0 ? 8ull : 0ull) + 4ull * (unsigned long long)(pe - ps);
            if (pe - ps >= kHeavyRow2) {
                int slot = 0;
                if (lane == 0) slot = atomicAdd(&s_nheavy, 1);
                slot = __shfl_sync(kFull, slot, 0);
                if (slot < kMaxHeavy2) {
                    if (lane == 0) {
                        s_hb[slot] = ps;
                        s_he[slot] = pe;
                    }
                    continue;
                }
            }
            mark_range<RANKS>(a, bm, touch, &s_ntouch, s_hist, ps, pe, 0, 128, lo, lane, my);
        }
        __syncthreads();
        const int nh = min(s_nheavy, kMaxHeavy2);
        for (int j = 0; j < nh; ++j)
            mark_range<RANKS>(a, bm, touch, &s_ntouch, s_hist, s_hb[j], s_he[j], (int64_t)warp * 128,
                              (int64_t)nwarps * 128, lo, lane, my);
        for (int off = 16; off > 0; off >>= 1) my += __shfl_down_sync(kFull, my, off);
        if (lane == 0 && my) atomicAdd(&s_count, my);
        __syncthreads();
        if (tid == 0) {
            if (s_count) atomicAdd(a.deg + v, s_count);
            if (sl == 0) {
                atomicAdd(a.updates, 1ull);
                my_bytes += 4ull + (RANKS ? 4ull * (unsigned long long)a.nj : 0ull);
            }
        }
        if (RANKS && tid < a.nj) {
            int c = 0;
            for (int j = a.jlo + tid; j < 32; ++j) c += s_hist[j];
            if (c) atomicAdd(a.cnt + (size_t)v * a.nj + tid, c);
        }
        // clear what this item set
        const int nt = s_ntouch;
        if (nt <= kTouchCap) {
            for (int i = tid; i < nt; i += blockDim.x) bm[touch[i]] = 0u;
        } else {
            uint4* b4 = reinterpret_cast<uint4*>(bm);
            for (int i = tid; i < (words >> 2); i += blockDim.x) b4[i] = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncthreads();
    }
    for (int off = 16; off > 0; off >>= 1) my_bytes += __shfl_down_sync(kFull, my_bytes, off);
    if (lane == 0 && my_bytes) atomicAdd(a.bytes, my_bytes);
}

// Sources of small 2-hop work (bin < kSmallBin: work < 2^kSmallBin, so at most
// 2 (2^kSmallBin - 1) row entries in all) take one warp each, without slices:
// the warp dedupes its source's 2-ball in a private open-addressing set of
// kSmallSlots node ids in shared memory (load at most one half), cleared with
// vector stores afterwards.  This spares the per-item cost of S slice items
// for the many small balls of a power-law graph.
constexpr int kSmallBin = 9;
constexpr int kSmallSlots = 2048;
constexpr int kSmallWarps = 8;
constexpr uint32_t kIdEmpty = 0xffffffffu;

template <bool RANKS>
__global__ void __launch_bounds__(kSmallWarps * 32)
    k_hdeg2_small(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                  const uint8_t* __restrict__ rank, const int32_t* __restrict__ order,
                  int64_t count, int32_t* __restrict__ deg, int32_t* __restrict__ cnt, int jlo,
                  int nj, unsigned long long* updates, unsigned long long* bytes) {
    extern __shared__ __align__(16) uint32_t s_tab_all[];
    __shared__ int s_hist_all[kSmallWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* tab = s_tab_all + (size_t)warp * kSmallSlots;
    int* hist = s_hist_all[warp];
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long my_bytes = 0, my_upd = 0;
    {
        uint4* t4 = reinterpret_cast<uint4*>(tab);
        for (int i = lane; i < kSmallSlots / 4; i += 32) t4[i] = make_uint4(kIdEmpty, kIdEmpty, kIdEmpty, kIdEmpty);
    }
    __syncwarp();
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < count; i += nw) {
        const int v = order[i];
        if (RANKS) hist[lane] = 0;
        __syncwarp();
        const int64_t vb = rowptr[v], ve = rowptr[v + 1];
        const int64_t dv = ve - vb;
        int my = 0;
        // rows: v's own (r == dv) and each neighbour's
        for (int64_t r = 0; r <= dv; ++r) {
            const int32_t x = r < dv ? __ldg(col + vb + r) : v;
            const int64_t rb = rowptr[x], re = rowptr[x + 1];
            if (lane == 0) my_bytes += 8ull + 4ull * (unsigned long long)(re - rb);
            for (int64_t k = rb + lane; k < re; k += 32) {
                const uint32_t u = (uint32_t)__ldg(col + k);
                uint32_t slot = (u * 0x9E3779B1u) >> (32 - 11);  // 2^11 = kSmallSlots
                for (int probe = 0; probe < kSmallSlots; ++probe) {
                    const uint32_t cur = *(volatile uint32_t*)(tab + slot);
                    if (cur == u) break;
                    if (cur == kIdEmpty) {
                        const uint32_t prev = atomicCAS(tab + slot, kIdEmpty, u);
                        if (prev == kIdEmpty) {
                            ++my;
                            if (RANKS) atomicAdd(&hist[rank[u]], 1);
                            break;
                        }
                        if (prev == u) break;
                    }
                    slot = (slot + 1u) & (kSmallSlots - 1);
                }
            }
        }
        for (int off = 16; off > 0; off >>= 1) my += __shfl_down_sync(kFull, my, off);
        __syncwarp();
        if (lane == 0) {
            deg[v] = my - 1;  // the ball holds v itself (by symmetry, in each neighbour's row)
            ++my_upd;
            my_bytes += 4ull + (RANKS ? 4ull * (unsigned long long)nj : 0ull);
        }
        if (RANKS && lane < nj) {
            int c = 0;
            for (int j = jlo + lane; j < 32; ++j) c += hist[j];
            cnt[(size_t)v * nj + lane] = c - (rank[v] >= jlo + lane ? 1 : 0);
        }
        uint4* t4 = reinterpret_cast<uint4*>(tab);
        for (int q = lane; q < kSmallSlots / 4; q += 32) t4[q] = make_uint4(kIdEmpty, kIdEmpty, kIdEmpty, kIdEmpty);
        __syncwarp();
    }
    for (int off = 16; off > 0; off >>= 1) my_bytes += __shfl_down_sync(kFull, my_bytes, off);
    if (lane == 0 && my_bytes) atomicAdd(bytes, my_bytes);
    if (lane == 0 && my_upd) atomicAdd(updates, my_upd);
}

// One CTA per source with a bitmap of all n nodes (KH_VAR_CTA).  N(v; 2) is the
// union of the rows of v and of its neighbours; a chunk of neighbours' row
// bounds is read into shared memory, sorted into short (up to 8 entries), middle
// (up to 32) and long rows, which groups of 2, 8 and 32 lanes claim and read
// four entries per lane and step; rows of 512 entries or more are read by the
// whole CTA.
//
// What bounds it: latency (a source is a chain of dependent loads) on small
// graphs, so the CTA is as small as the bitmap allows (kCtaBitmap bytes of
// shared memory per 128 threads: 8 sources or more in flight per SM), then the
// shared-memory tests and atomics, one per row entry.  The search kernel of
// h >= 3 (a queue, 8 barriers a source, the bitmap walked by 256 threads) took
// 2.4 ms, the sliced kernel with one slice 5.3 ms for the 2-degrees of Chung-Lu
// n = 200k; this one 1.7 ms (fixed-level counts 4.6 and 7.2 -> 2.1 ms: the ranks
// are read along the row, not gathered, and counted in registers).  128 threads
// for a 25 KB bitmap: 256 took the same time for degrees, 20% longer for counts.
constexpr int kCtaMaxThreads = 512;
constexpr int64_t kCtaBitmap = 28 * 1024;
constexpr int kCtaHeavy = 512;

struct Cta2Args {
    const int64_t* rowptr;
    const int32_t* col;
    const uint8_t* rank;   // of the nodes
    const uint8_t* crank;  // rank of each column entry
    int words;             // bitmap words, a multiple of 4
    const int32_t* order;  // sources, longest first
    int64_t nsrc;
    int32_t* deg;
    int32_t* cnt;
    int jlo, nj;
    int* work_ctr;
    int* err;
    unsigned long long* updates;
    unsigned long long* bytes;
};

// Mark u (rank r); returns 1 if it is new.
template <bool RANKS>
__device__ __forceinline__ int mark_node(uint32_t* bm, int* s_hist, RankCounts& ranks, int32_t u, int r) {
    uint32_t* w = bm + (u >> 5);
    const uint32_t bit = 1u << (u & 31);
    if ((*(volatile uint32_t*)w & bit) || (atomicOr(w, bit) & bit)) return 0;
    if (RANKS) ranks.add(r, s_hist);
    return 1;
}

template <bool RANKS>
__global__ void __launch_bounds__(kCtaMaxThreads) k_hdeg2_cta(Cta2Args a) {
    extern __shared__ __align__(16) uint32_t bm[];
    const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x;
    // per row of the chunk: its start and length; the rows of each bucket
    int64_t* s_b = reinterpret_cast<int64_t*>(bm + a.words);
    int* s_len = reinterpret_cast<int*>(s_b + T);
    uint16_t* s_q = reinterpret_cast<uint16_t*>(s_len + T);
    __shared__ int s_nq[4], s_cq[4];
    __shared__ int s_hist[32];
    __shared__ int s_count, s_idx, s_v;
    unsigned long long my_bytes = 0;
    for (int i = tid * 4; i < a.words; i += T * 4)
        *reinterpret_cast<uint4*>(bm + i) = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
        const int i = atomicAdd(a.work_ctr, 1);
        s_idx = i;
        if (i < a.nsrc) s_v = a.order[i];
    }
    for (;;) {
        __syncthreads();
        if (s_idx >= a.nsrc) break;
        const int v = s_v;
        int next = 0;
        if (tid == 0) next = atomicAdd(a.work_ctr, 1);
        const int64_t vb = a.rowptr[v];
        const int deg = (int)(a.rowptr[v + 1] - vb);
        RankCounts ranks;
        int my = 0;
        if (tid == 0) s_count = 0;
        if (RANKS && tid < 32) s_hist[tid] = 0;
        for (int c0 = 0; c0 <= deg; c0 += T) {  // rows: each neighbour's, then v's own
            if (c0) __syncthreads();            // the previous chunk is read
            if (tid < 4) {
                s_nq[tid] = 0;
                s_cq[tid] = 0;
            }
            const int i = c0 + tid;
            int len = 0;
            if (i <= deg) {
                const int32_t x = i < deg ? __ldg(a.col + vb + i) : v;
                const int64_t b = a.rowptr[x];
                len = (int)(a.rowptr[x + 1] - b);
                s_b[tid] = b;
                s_len[tid] = len;
                my_bytes += 8ull + 4ull * (unsigned long long)len;
            }
            const int q = len == 0 ? -1 : len <= 8 ? 0 : len <= 32 ? 1 : len < kCtaHeavy ? 2 : 3;
            __syncthreads();
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t mq = __ballot_sync(kFull, q == k);
                if (!mq) continue;
                int base = 0;
                if (lane == 0) base = atomicAdd(&s_nq[k], __popc(mq));
                base = __shfl_sync(kFull, base, 0);
                if (q == k) s_q[k * T + base + __popc(mq & ((1u << lane) - 1u))] = (uint16_t)tid;
            }
            __syncthreads();
            for (int hi = 0; hi < s_nq[3]; ++hi) {
                const int64_t rb = s_b[s_q[3 * T + hi]];
                const int n = s_len[s_q[3 * T + hi]];
                for (int k = tid; k < n; k += 4 * T) {
                    int32_t u[4];
                    int r[4];
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const bool in = k + p * T < n;
                        u[p] = in ? __ldg(a.col + rb + k + p * T) : -1;
                        r[p] = RANKS && in ? __ldg(a.crank + rb + k + p * T) : 0;
                    }
                    if (RANKS) ranks.reserve(s_hist);
#pragma unroll
                    for (int p = 0; p < 4; ++p)
                        if (u[p] >= 0) my += mark_node<RANKS>(bm, s_hist, ranks, u[p], r[p]);
                }
            }
            int bk = 2, li = -1, pos = 0, n = 0;
            int64_t rb = 0;
            for (int step = 0;; ++step) {  // as walk_chunk of the level union: groups claim rows
                if (step > row_steps(T)) {
                    if (lane == 0) atomicOr(a.err, kErrLoop);
                    break;
                }
                const int lgG = bk == 2 ? 5 : bk == 1 ? 3 : 1;
                const int lead = lane >> lgG << lgG;
                const uint32_t need = __ballot_sync(kFull, li == -1 && lane == lead);
                if (need) {
                    int base = 0;
                    if (lane == 0) base = atomicAdd(&s_cq[bk], __popc(need));
                    base = __shfl_sync(kFull, base, 0);
                    if (li == -1) {
                        const int j = base + __popc(need & ((1u << lead) - 1u));
                        li = -2;
                        if (j < s_nq[bk]) {
                            li = s_q[bk * T + j];
                            rb = s_b[li];
                            n = s_len[li];
                            pos = 0;
                        }
                    }
                }
                if (__all_sync(kFull, li == -2)) {
                    do --bk;
                    while (bk >= 0 && s_nq[bk] == 0);
                    if (bk < 0) break;
                    li = -1;
                    continue;
                }
                if (li >= 0) {
                    int32_t u[4];
                    int r[4];
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const int k = pos + (p << lgG) + lane - lead;
                        u[p] = k < n ? __ldg(a.col + rb + k) : -1;
                        r[p] = RANKS && k < n ? __ldg(a.crank + rb + k) : 0;
                    }
                    if (RANKS) ranks.reserve(s_hist);
#pragma unroll
                    for (int p = 0; p < 4; ++p)
                        if (u[p] >= 0) my += mark_node<RANKS>(bm, s_hist, ranks, u[p], r[p]);
                    pos += 4 << lgG;
                    if (pos >= n) li = -1;
                }
            }
        }
        int nv = 0;
        if (tid == 0 && next < a.nsrc) nv = a.order[next];
        my = __reduce_add_sync(kFull, my);
        if (lane == 0 && my) atomicAdd(&s_count, my);
        if (RANKS) ranks.finish(s_hist, lane);
        __syncthreads();
        if (tid == 0) {
            a.deg[v] = s_count - 1;  // the ball holds v itself (by symmetry, in each neighbour's row)
            atomicAdd(a.updates, 1ull);
            my_bytes += 4ull + (RANKS ? 4ull * (unsigned long long)a.nj : 0ull);
            s_idx = next;
            s_v = nv;
        }
        if (RANKS && tid < a.nj) {
            int c = a.rank[v] >= a.jlo + tid ? -1 : 0;
            for (int j = a.jlo + tid; j < 32; ++j) c += s_hist[j];
            a.cnt[(size_t)v * a.nj + tid] = c;
        }
        for (int i = tid * 4; i < a.words; i += T * 4)
            *reinterpret_cast<uint4*>(bm + i) = make_uint4(0u, 0u, 0u, 0u);
    }
    for (int off = 16; off > 0; off >>= 1) my_bytes += __shfl_down_sync(kFull, my_bytes, off);
    if (lane == 0 && my_bytes) atomicAdd(a.bytes, my_bytes);
}

// 2-hop work of each node and its log2 bin (isolated nodes: bin -1).
__global__ void k_order_bins(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                             int64_t n, int8_t* __restrict__ bin, int* __restrict__ hist) {
    __shared__ int s_h[kOrderBins];
    for (int i = threadIdx.x; i < kOrderBins; i += blockDim.x) s_h[i] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += nw) {
        const int64_t b = rowptr[v], e = rowptr[v + 1];
        unsigned long long w = 0;
        for (int64_t k = b + lane; k < e; k += 32) {
            const int32_t x = col[k];
            w += (unsigned long long)(rowptr[x + 1] - rowptr[x]);
        }
        for (int off = 16; off > 0; off >>= 1) w += __shfl_down_sync(kFull, w, off);
        if (lane == 0) {
            int bb = -1;
            if (e > b) {
                bb = 63 - __clzll((long long)(w + 1));
                if (bb >= kOrderBins) bb = kOrderBins - 1;
                atomicAdd(&s_h[bb], 1);
            }
            bin[v] = (int8_t)bb;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kOrderBins; i += blockDim.x)
        if (s_h[i]) atomicAdd(hist + i, s_h[i]);
}

// Scatter the non-isolated nodes by bin, largest bin first; hist holds each
// bin's start (exclusive prefix in descending bin order) and is advanced.
__global__ void k_order_scatter(const int8_t* __restrict__ bin, int64_t n, int* __restrict__ pos,
                                int32_t* __restrict__ order) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int b = bin[v];
        if (b >= 0) order[atomicAdd(pos + b, 1)] = (int32_t)v;
    }
}

// deg[v] starts at -1 for a node with a neighbour (v is counted in its own
// ball), 0 for an isolated node; the counts start at minus v's own rank test.
__global__ void k_init2(const int64_t* __restrict__ rowptr, const uint8_t* __restrict__ rank,
                        int64_t n, int32_t* __restrict__ deg, int32_t* __restrict__ cnt, int jlo,
                        int nj) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const bool iso = rowptr[v + 1] == rowptr[v];
        deg[v] = iso ? 0 : -1;
        if (cnt) {
            const int rv = rank[v];
            for (int j = 0; j < nj; ++j) cnt[(size_t)v * nj + j] = (!iso && rv >= jlo + j) ? -1 : 0;
        }
    }
}

// ---- bit-parallel searches of 1024 sources at a time ----
// For a batch of up to 1024 sources s_j, m[u] holds bit j when u is within i
// hops of s_j (32 words per node).  One pull over all rows, m'[x] = m[x] | OR_{u
// in A(x)} m[u], adds a hop.  The first hop is set by scattering the sources'
// rows (without s_j itself: s_j is a neighbour of its neighbours, so it joins
// at hop 2); the last pull only counts the set bits per source.  A pull reads
// each row once and gathers 128 bytes per entry, for 1024 sources, where a
// search per source reads the rows of its (h-1)-ball: it pays for the sources
// of largest 2-hop work at h = 2 (kh_tune.cu) and for whole graphs at h >= 3
// whose balls are large (run_hdeg_full).
//
// What bounds it: the gathers, from L2 where the masks of the batch fit (128 n
// bytes).  128-byte masks fill whole sectors and spread the per-row work (row
// bounds, reduction, counting) over 1024 sources: the 16-byte masks of the
// first version used half of each sector and took 8 times the row passes.
// Measured: exact 3-degrees of Chung-Lu n = 200k 128 (a search per source) -> 28
// ms, 4-degrees of Chung-Lu n = 60k 277 -> 7.4 ms, of R-MAT 15 78 -> 2.4 ms;
// exact 2-degrees of R-MAT 20 140 -> 101 ms, of R-MAT 18 21.6 -> 13.9 ms.  A
// batch on Chung-Lu n = 200k: a storing pull 75 us (6.8 TB/s of gathers), long-row
// pieces 17 us, seeding and clearing 8 us each.
constexpr int kSweepWords = 32;
constexpr int kSweepSrc = 32 * kSweepWords;
constexpr int kSweepHead = 128;    // longer rows are OR'd in pieces by k_sweep_pieces
constexpr int kSweepPiece = 128;   // entries per piece
constexpr int kSweepPlanes = 8;    // carry-save counter planes: 255 additions between flushes
constexpr int kSweepThreads = 256;
constexpr int kSweepPullSm = 5;    // CTAs per SM of a pull that stores, one that counts
constexpr int kSweepCountSm = 4;

// Set the batch's source bits on the neighbours of its sources, one CTA per
// source; with bytes also the algorithmic bytes of one 2-hop search per source.
__global__ void k_sweep_seed(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                             const int32_t* __restrict__ src, uint32_t* __restrict__ m,
                             uint32_t* __restrict__ filter, unsigned long long* bytes) {
    const int j = blockIdx.x;
    const int v = src[j];
    const int64_t b = rowptr[v], e = rowptr[v + 1];
    unsigned long long my = 0;
    for (int64_t k = b + threadIdx.x; k < e; k += blockDim.x) {
        const int32_t u = __ldg(col + k);
        atomicOr(m + (size_t)u * kSweepWords + (j >> 5), 1u << (j & 31));
        const uint32_t bit = 1u << (u & 31);
        if (!(*(volatile uint32_t*)(filter + (u >> 5)) & bit)) atomicOr(filter + (u >> 5), bit);
        if (bytes) my += 8ull + 4ull * (unsigned long long)(rowptr[u + 1] - rowptr[u]);
    }
    if (!bytes) return;
    if (threadIdx.x == 0) my += 8ull + 4ull * (unsigned long long)(e - b) + 4ull;
    for (int off = 16; off > 0; off >>= 1) my += __shfl_down_sync(kFull, my, off);
    if ((threadIdx.x & 31) == 0 && my) atomicAdd(bytes, my);
}

// End of a batch, one CTA per source: deg_h (the ball holds the source itself),
// the counter and the source bits back to zero.
__global__ void k_sweep_finish(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                               const int32_t* __restrict__ src, uint4* __restrict__ m,
                               uint32_t* __restrict__ filter, unsigned int* __restrict__ cnt,
                               int32_t* __restrict__ deg, unsigned long long* updates,
                               unsigned long long* bytes, unsigned long long batch_bytes) {
    const int j = blockIdx.x;
    const int v = src[j];
    const int64_t b = rowptr[v], e = rowptr[v + 1];
    for (int64_t k = b + (threadIdx.x >> 3); k < e; k += blockDim.x >> 3) {
        const int32_t u = __ldg(col + k);
        m[(size_t)u * 8 + (threadIdx.x & 7)] = make_uint4(0u, 0u, 0u, 0u);
        if ((threadIdx.x & 7) == 0) filter[u >> 5] = 0u;
    }
    if (threadIdx.x != 0) return;
    const int at = 32 * (j & 31) + (j >> 5);  // flush_planes' order
    deg[v] = (int32_t)cnt[at] - 1;
    cnt[at] = 0u;
    if (j == 0) {
        atomicAdd(updates, (unsigned long long)gridDim.x);
        if (batch_bytes) atomicAdd(bytes, batch_bytes);
    }
}

__device__ __forceinline__ void or4(uint4& a, const uint4 b) {
    a.x |= b.x;
    a.y |= b.y;
    a.z |= b.z;
    a.w |= b.w;
}

// The mask word a lane holds after or_row: lane = 8 sub + l8 reads the l8-th 16
// bytes of a mask and keeps one of their four words.
__device__ __forceinline__ int or_row_word(int lane) {
    const int sub = lane >> 3;
    return (lane & 7) * 4 + (sub & 2) + (sub & 1);
}

// OR of the masks of one warp's row entries [b, e), entry b + lane already in c:
// four entries per load (8 lanes of 16 bytes each), four loads in flight.
// FILTER: entries whose node has no bits are dropped first (buf: 32 ints of
// shared memory per warp).
template <bool FILTER>
__device__ __forceinline__ uint32_t or_row(const int32_t* __restrict__ col, int64_t b, int64_t e, int32_t c,
                                           const uint4* __restrict__ m, const uint32_t* __restrict__ filter,
                                           int32_t* buf, int lane) {
    const int sub = lane >> 3, l8 = lane & 7;
    uint4 acc = make_uint4(0u, 0u, 0u, 0u);
    while (b < e) {
        const int32_t cn = b + 32 + lane < e ? __ldg(col + b + 32 + lane) : 0;  // the next 32
        int cnt = (int)(e - b < 32 ? e - b : 32);
        if (FILTER) {
            const bool live = lane < cnt && ((__ldg(filter + (c >> 5)) >> (c & 31)) & 1u);
            const uint32_t lm = __ballot_sync(kFull, live);
            cnt = __popc(lm);
            if (live) buf[__popc(lm & ((1u << lane) - 1u))] = c;
            __syncwarp();
            c = buf[lane];
            __syncwarp();
        }
#pragma unroll 1
        for (int j0 = 0; j0 < cnt; j0 += 16) {
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
                const int32_t u = __shfl_sync(kFull, c, j0 + j + sub);
                if (j0 + j + sub < cnt) or4(acc, __ldg(m + (size_t)u * 8 + l8));
            }
        }
        b += 32;
        c = cn;
    }
    // OR over the four subgroups; each lane keeps one of its chunk's four words
    const bool hi = sub & 2, odd = sub & 1;
    uint32_t k0 = hi ? acc.z : acc.x, k1 = hi ? acc.w : acc.y;
    k0 |= __shfl_xor_sync(kFull, hi ? acc.x : acc.z, 16);
    k1 |= __shfl_xor_sync(kFull, hi ? acc.y : acc.w, 16);
    return (odd ? k1 : k0) | __shfl_xor_sync(kFull, odd ? k0 : k1, 8);
}

// Rows longer than kSweepHead: the OR over each piece of kSweepPiece entries
// into the row's words of bh (zero before).  One warp per piece.
template <bool FILTER>
__global__ void __launch_bounds__(kSweepThreads)
    k_sweep_pieces(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                   const int32_t* __restrict__ hnode, const int32_t* __restrict__ piece_h,
                   const int32_t* __restrict__ piece_off, int64_t npieces, const uint4* __restrict__ m,
                   const uint32_t* __restrict__ filter, uint32_t* __restrict__ bh) {
    __shared__ int32_t s_buf[kSweepThreads / 32][32];
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < npieces; p += nw) {
        const int h = piece_h[p];
        const int x = hnode[h];
        const int64_t b = rowptr[x] + piece_off[p];
        const int64_t re = rowptr[x + 1];
        const int64_t e = b + kSweepPiece < re ? b + kSweepPiece : re;
        const uint32_t r = or_row<FILTER>(col, b, e, b + lane < e ? __ldg(col + b + lane) : 0, m, filter,
                                          s_buf[threadIdx.x >> 5], lane);
        if (r) atomicOr(bh + (size_t)h * kSweepWords + or_row_word(lane), r);
    }
}

// Add the counts held in a lane's carry-save planes (bit `bit` of plane p is
// worth 2^p, for source 32 word + bit) to s_cnt[32 bit + word] (the lanes' words
// are all different: no bank conflicts), four bits at a time as bytes.
__device__ __forceinline__ void flush_planes(uint32_t (&c)[kSweepPlanes], unsigned int* s_cnt, int word) {
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {
        uint32_t t = 0;
#pragma unroll
        for (int p = 0; p < kSweepPlanes; ++p) t |= ((c[p] >> i) & 0x01010101u) << p;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned int v = (t >> (8 * q)) & 255u;
            if (v) atomicAdd(&s_cnt[32 * (i + 8 * q) + word], v);
        }
    }
#pragma unroll
    for (int p = 0; p < kSweepPlanes; ++p) c[p] = 0u;
}

// One pull over every row, a warp per row.  STORE: m'[x] to out; COUNT: the
// number of nodes with bit 32 w + b into cnt[32 b + w] (carry-save counters, a
// mask word per lane).
template <bool FILTER, bool STORE, bool COUNT>
__global__ void __launch_bounds__(kSweepThreads, COUNT ? kSweepCountSm : kSweepPullSm)
    k_sweep_pull(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col, int64_t n,
                 const uint32_t* __restrict__ m, const uint32_t* __restrict__ filter,
                 const int32_t* __restrict__ hpos, uint32_t* __restrict__ bh, uint32_t* __restrict__ out, unsigned int* __restrict__ cnt) {
    __shared__ int32_t s_buf[kSweepThreads / 32][32];
    __shared__ unsigned int s_cnt[COUNT ? kSweepSrc : 1];
    const int lane = threadIdx.x & 31;
    if (COUNT) {
        for (int i = threadIdx.x; i < kSweepSrc; i += blockDim.x) s_cnt[i] = 0u;
        __syncthreads();
    }
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    uint32_t c[kSweepPlanes];
#pragma unroll
    for (int p = 0; p < kSweepPlanes; ++p) c[p] = 0u;
    const int word = or_row_word(lane);
    int adds = 0;
    // a row is a chain of three loads (bounds, columns, masks): the bounds are
    // loaded two rows ahead and the first columns one row ahead
    int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int64_t b1 = 0, e1 = 0, b2 = 0, e2 = 0;
    int32_t c1 = 0;
    if (x < n) {
        b1 = rowptr[x];
        e1 = rowptr[x + 1];
        if (b1 + lane < e1) c1 = __ldg(col + b1 + lane);
    }
    if (x + nw < n) {
        b2 = rowptr[x + nw];
        e2 = rowptr[x + nw + 1];
    }
    for (; x < n; x += nw) {
        const int64_t b = b1, e = e1;
        const int32_t c0 = c1;
        b1 = b2;
        e1 = e2;
        c1 = b1 + lane < e1 ? __ldg(col + b1 + lane) : 0;
        b2 = e2 = 0;
        if (x + 2 * nw < n) {
            b2 = rowptr[x + 2 * nw];
            e2 = rowptr[x + 2 * nw + 1];
        }
        if (e == b) continue;  // never reached (its words stay zero)
        const uint32_t own = m[(size_t)x * kSweepWords + word];
        const bool longrow = e - b > kSweepHead;
        uint32_t r = or_row<FILTER>(col, b, longrow ? b : e, c0, reinterpret_cast<const uint4*>(m), filter,
                                    s_buf[threadIdx.x >> 5], lane);
        if (longrow) {  // its pieces' words, left zero for the next pull
            uint32_t* w = bh + (size_t)hpos[x] * kSweepWords + word;
            r = *w;
            *w = 0u;
        }
        r |= own;
        if (STORE) out[(size_t)x * kSweepWords + word] = r;
        if (COUNT) {
#pragma unroll
            for (int p = 0; p < kSweepPlanes; ++p) {
                const uint32_t t = c[p] & r;
                c[p] ^= r;
                r = t;
            }
            ++adds;
        }
        if (COUNT && adds == (1 << kSweepPlanes) - 1) {
            flush_planes(c, s_cnt, word);
            adds = 0;
        }
    }
    if (!COUNT) return;
    if (adds) flush_planes(c, s_cnt, word);
    __syncthreads();
    for (int i = threadIdx.x; i < kSweepSrc; i += blockDim.x)
        if (s_cnt[i]) atomicAdd(cnt + i, s_cnt[i]);
}

}  // namespace

size_t hdeg2_smem(int64_t width) { return (size_t)(width / 8) + (size_t)kTouchCap * 4; }

int64_t hdeg2_width(int64_t n, int slices) {
    int64_t w = (n + slices - 1) / slices;
    return (w + 127) & ~(int64_t)127;
}

int hdeg2_min_slices(int64_t n) {
    int s = 1;
    while (hdeg2_smem(hdeg2_width(n, s)) > (size_t)kSmem2Max) ++s;
    return s;
}

int ensure_order2(Graph& g, cudaStream_t s) {
    if (g.order2) return KH_OK;
    int8_t* bin = nullptr;
    int* hist = nullptr;
    int rc = alloc_bytes(g.ctx, (void**)&g.order2, sizeof(int32_t) * (size_t)(g.n > 0 ? g.n : 1),
                         "source order");
    if (rc) return rc;
    cudaError_t e = cudaMallocAsync((void**)&bin, (size_t)(g.n > 0 ? g.n : 1), s);
    if (e == cudaSuccess) e = cudaMallocAsync((void**)&hist, sizeof(int) * kOrderBins, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(hist, 0, sizeof(int) * kOrderBins, s);
    if (e != cudaSuccess) {
        if (bin) cudaFreeAsync(bin, s);
        if (hist) cudaFreeAsync(hist, s);
        cudaFree(g.order2);
        g.order2 = nullptr;
        return check_cuda(g.ctx, e, "source order");
    }
    const int grid = g.ctx->sm_count * 8;
    k_order_bins<<<grid, 256, 0, s>>>(g.rowptr, g.col, g.n, bin, hist);
    int h[kOrderBins];
    e = cudaMemcpyAsync(h, hist, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) {
        // starts in descending bin order
        int pos[kOrderBins];
        int64_t acc = 0;
        for (int b = kOrderBins - 1; b >= 0; --b) {
            pos[b] = (int)acc;
            acc += h[b];
        }
        g.nsrc2 = acc;
        for (int b = 0; b < kOrderBins; ++b) g.order2_hist[b] = h[b];
        e = cudaMemcpyAsync(hist, pos, sizeof(pos), cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) {
            k_order_scatter<<<grid, 256, 0, s>>>(bin, g.n, hist, g.order2);
            e = cudaStreamSynchronize(s);  // `pos` is a host stack array
        }
    }
    cudaFreeAsync(bin, s);
    cudaFreeAsync(hist, s);
    count_launch(g, 2);
    if (e != cudaSuccess) {
        cudaFree(g.order2);
        g.order2 = nullptr;
        return check_cuda(g.ctx, e, "source order");
    }
    return KH_OK;
}

int64_t hdeg2_small_split(const Graph& g) {
    int64_t big = 0;
    for (int b = kSmallBin; b < kOrderBins; ++b) big += g.order2_hist[b];
    return big;
}

int launch_hdeg2_small(Graph& g, int32_t* deg, int32_t* cnt, int jlo, int nj, cudaStream_t s,
                       const int32_t* order, int64_t count) {
    if (count <= 0) return KH_OK;
    void (*kern)(const int64_t*, const int32_t*, const uint8_t*, const int32_t*, int64_t, int32_t*,
                 int32_t*, int, int, unsigned long long*, unsigned long long*) =
        cnt ? k_hdeg2_small<true> : k_hdeg2_small<false>;
    const size_t dyn = (size_t)kSmallWarps * kSmallSlots * 4;
    KH_CUDA_TRY(g.ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
    int per_sm = 0;
    KH_CUDA_TRY(g.ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSmallWarps * 32, dyn));
    if (per_sm < 1) per_sm = 1;
    int64_t grid = (int64_t)g.ctx->sm_count * per_sm;
    const int64_t need = (count + kSmallWarps - 1) / kSmallWarps;
    if (grid > need) grid = need;
    prof_begin(g, kProfBfs, s);
    kern<<<(int)grid, kSmallWarps * 32, dyn, s>>>(g.rowptr, g.col, g.rank, order, count, deg, cnt, jlo,
                                                   nj, &g.state->updates, &g.state->bytes[kProfBfs]);
    count_launch(g, 1);
    prof_end(g, kProfBfs, s);
    return KH_OK;
}

// A source of half of a CTA slot's share of the work or more (8 slots per SM) is
// the tail of the launch when one small CTA reads it: 2-degrees of R-MAT 15 / 16
// 1.45 / 2.7 ms without large CTAs, 0.75 / 1.75 ms so; from a quarter of the
// share on the large CTAs take the small ones' place (counts of Chung-Lu n = 200k
// 2.14 -> 2.5 ms).
int hdeg2_large_bin(const Graph& g) {
    double total = 0.0;
    for (int b = 0; b < kOrderBins; ++b) total += 1.5 * std::ldexp((double)g.order2_hist[b], b);
    int bin = kCtaSmallBin + 1;
    while (bin < kOrderBins - 1 && std::ldexp(1.0, bin) < total / (2.0 * 8.0 * g.ctx->sm_count)) ++bin;
    return bin < 14 ? 14 : bin;
}

int64_t hdeg2_sources_from_bin(const Graph& g, int bin) {
    int64_t c = 0;
    for (int b = bin < 0 ? 0 : bin; b < kOrderBins; ++b) c += g.order2_hist[b];
    return c;
}

// The arrays of the bit-parallel searches at h: mask buffers (zeroed), the
// node filter, the rows longer than kSweepHead and their pieces, the counters.
int ensure_sweep(Graph& g, int h, cudaStream_t s) {
    const int bufs = h == 2 ? 1 : h == 3 ? 2 : 3;
    const size_t n = (size_t)(g.n > 0 ? g.n : 1);
    int rc;
    for (int i = 0; i < bufs; ++i) {
        if (g.sw_m[i]) continue;
        if ((rc = alloc_bytes(g.ctx, (void**)&g.sw_m[i], 4 * kSweepWords * n, "sweep source bits"))) return rc;
        KH_CUDA_TRY(g.ctx, cudaMemsetAsync(g.sw_m[i], 0, 4 * kSweepWords * n, s));
    }
    if (g.sw_ready) return KH_OK;
    std::vector<int64_t> rp((size_t)g.n + 1);
    KH_CUDA_TRY(g.ctx, cudaMemcpyAsync(rp.data(), g.rowptr, sizeof(int64_t) * rp.size(),
                                       cudaMemcpyDeviceToHost, s));
    KH_CUDA_TRY(g.ctx, cudaStreamSynchronize(s));
    std::vector<int32_t> hpos(n, -1), hnode, piece_h, piece_off;
    for (int64_t x = 0; x < g.n; ++x) {
        const int64_t d = rp[(size_t)x + 1] - rp[(size_t)x];
        if (d <= kSweepHead) continue;
        const int h = (int)hnode.size();
        hpos[(size_t)x] = h;
        hnode.push_back((int32_t)x);
        for (int64_t off = 0; off < d; off += kSweepPiece) {
            piece_h.push_back(h);
            piece_off.push_back((int32_t)off);
        }
    }
    const size_t nh = hnode.size() > 0 ? hnode.size() : 1;
    const size_t np = piece_h.size() > 0 ? piece_h.size() : 1;
    const size_t fw = (n + 31) / 32;
    // (an array kept from a call that failed half-way is used as it is)
    if ((!g.sw_filter && (rc = alloc_bytes(g.ctx, (void**)&g.sw_filter, 4 * fw, "sweep filter"))) ||
        (!g.sw_hpos && (rc = alloc_bytes(g.ctx, (void**)&g.sw_hpos, 4 * n, "sweep row index"))) ||
        (!g.sw_hnode && (rc = alloc_bytes(g.ctx, (void**)&g.sw_hnode, 4 * nh, "sweep long rows"))) ||
        (!g.sw_bh && (rc = alloc_bytes(g.ctx, (void**)&g.sw_bh, 4 * kSweepWords * nh, "sweep long-row words"))) ||
        (!g.sw_piece_h && (rc = alloc_bytes(g.ctx, (void**)&g.sw_piece_h, 4 * np, "sweep pieces"))) ||
        (!g.sw_piece_off && (rc = alloc_bytes(g.ctx, (void**)&g.sw_piece_off, 4 * np, "sweep pieces"))) ||
        (!g.sw_cnt && (rc = alloc_bytes(g.ctx, (void**)&g.sw_cnt, 4 * kSweepSrc, "sweep counts"))))
        return rc;
    KH_CUDA_TRY(g.ctx, cudaMemsetAsync(g.sw_filter, 0, 4 * fw, s));
    KH_CUDA_TRY(g.ctx, cudaMemsetAsync(g.sw_cnt, 0, 4 * kSweepSrc, s));
    KH_CUDA_TRY(g.ctx, cudaMemsetAsync(g.sw_bh, 0, 4 * kSweepWords * nh, s));
    KH_CUDA_TRY(g.ctx, cudaMemcpyAsync(g.sw_hpos, hpos.data(), 4 * n, cudaMemcpyHostToDevice, s));
    if (!hnode.empty()) {
        KH_CUDA_TRY(g.ctx, cudaMemcpyAsync(g.sw_hnode, hnode.data(), 4 * hnode.size(),
                                           cudaMemcpyHostToDevice, s));
        KH_CUDA_TRY(g.ctx, cudaMemcpyAsync(g.sw_piece_h, piece_h.data(), 4 * piece_h.size(),
                                           cudaMemcpyHostToDevice, s));
        KH_CUDA_TRY(g.ctx, cudaMemcpyAsync(g.sw_piece_off, piece_off.data(), 4 * piece_off.size(),
                                           cudaMemcpyHostToDevice, s));
    }
    KH_CUDA_TRY(g.ctx, cudaStreamSynchronize(s));  // host vectors go out of scope
    g.sw_nheavy = (int64_t)hnode.size();
    g.sw_npieces = (int64_t)piece_h.size();
    g.sw_ready = true;
    return KH_OK;
}

int run_sweeps(Graph& g, int32_t* deg, const int32_t* src, int64_t count, int h, cudaStream_t s) {
    if (count <= 0) return KH_OK;
    int rc = ensure_sweep(g, h, s);
    if (rc) return rc;
    int64_t tgrid = (g.sw_npieces + 7) / 8;
    if (tgrid > g.ctx->sm_count * 8) tgrid = g.ctx->sm_count * 8;
    // at h = 2 the bytes of one search per source (counted by the scatter); the
    // longer searches count the rows that their pulls read
    const unsigned long long batch_bytes =
        h == 2 ? 0ull : (unsigned long long)(h - 1) * (8ull * g.n + 4ull * g.nnz);
    prof_begin(g, kProfBfs, s);
    int64_t launches = 0;
    for (int64_t b0 = 0; b0 < count; b0 += kSweepSrc) {
        const int nb = (int)(count - b0 < kSweepSrc ? count - b0 : kSweepSrc);
        k_sweep_seed<<<nb, 256, 0, s>>>(g.rowptr, g.col, src + b0, g.sw_m[0], g.sw_filter,
                                        h == 2 ? &g.state->bytes[kProfBfs] : nullptr);
        for (int hop = 2; hop <= h; ++hop) {
            const bool first = hop == 2, last = hop == h;
            const uint32_t* in = g.sw_m[first ? 0 : 1 + ((hop - 3) & 1)];
            uint32_t* out = last ? nullptr : g.sw_m[1 + ((hop - 2) & 1)];
            const uint4* in4 = reinterpret_cast<const uint4*>(in);
            if (g.sw_npieces > 0) {
                if (first)
                    k_sweep_pieces<true><<<(int)tgrid, kSweepThreads, 0, s>>>(
                        g.rowptr, g.col, g.sw_hnode, g.sw_piece_h, g.sw_piece_off, g.sw_npieces, in4,
                        g.sw_filter, g.sw_bh);
                else
                    k_sweep_pieces<false><<<(int)tgrid, kSweepThreads, 0, s>>>(
                        g.rowptr, g.col, g.sw_hnode, g.sw_piece_h, g.sw_piece_off, g.sw_npieces, in4,
                        g.sw_filter, g.sw_bh);
                ++launches;
            }
            void (*pull)(const int64_t*, const int32_t*, int64_t, const uint32_t*, const uint32_t*,
                         const int32_t*, uint32_t*, uint32_t*, unsigned int*) =
                first ? (last ? k_sweep_pull<true, false, true> : k_sweep_pull<true, true, false>)
                      : (last ? k_sweep_pull<false, false, true> : k_sweep_pull<false, true, false>);
            // one wave: a second, partial one costs a whole row loop
            pull<<<g.ctx->sm_count * (last ? kSweepCountSm : kSweepPullSm), kSweepThreads, 0, s>>>(g.rowptr, g.col, g.n, in, g.sw_filter, g.sw_hpos, g.sw_bh,
                                                 out, g.sw_cnt);
            ++launches;
        }
        k_sweep_finish<<<nb, 256, 0, s>>>(g.rowptr, g.col, src + b0, reinterpret_cast<uint4*>(g.sw_m[0]),
                                          g.sw_filter, g.sw_cnt, deg, &g.state->updates,
                                          &g.state->bytes[kProfBfs], batch_bytes);
        launches += 2;
    }
    count_launch(g, launches);
    prof_end(g, kProfBfs, s);
    KH_CUDA_TRY(g.ctx, cudaGetLastError());
    return KH_OK;
}

int launch_hdeg2_cta(Graph& g, int32_t* deg, int32_t* cnt, int jlo, int nj, cudaStream_t s,
                     const int32_t* order, int64_t nsrc, bool large) {
    if (nsrc <= 0) return KH_OK;
    Cta2Args a{};
    a.words = (int)(((g.n + 31) / 32 + 3) & ~(int64_t)3);
    const int64_t bitmap = (int64_t)a.words * 4;
    const int threads = large                    ? kCtaMaxThreads
                        : bitmap <= kCtaBitmap     ? 128
                        : bitmap <= 2 * kCtaBitmap ? 256
                                                   : kCtaMaxThreads;
    const size_t dyn = (size_t)bitmap + (size_t)threads * 20;
    void (*kern)(Cta2Args) = cnt ? k_hdeg2_cta<true> : k_hdeg2_cta<false>;
    KH_CUDA_TRY(g.ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)kSmemBitmapMax + 20 * kCtaMaxThreads));
    int per_sm = 0;
    KH_CUDA_TRY(g.ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, dyn));
    if (per_sm < 1) return set_error(g.ctx, KH_EINVAL, "2-degree kernel does not fit on an SM");
    KH_CUDA_TRY(g.ctx, cudaMemsetAsync(&g.state->work_ctr[large ? 3 : 2], 0, sizeof(int), s));
    int64_t grid = (int64_t)g.ctx->sm_count * per_sm;
    if (grid > nsrc) grid = nsrc;
    a.rowptr = g.rowptr;
    a.col = g.col;
    a.rank = g.rank;
    a.crank = g.crank;
    a.order = order;
    a.nsrc = nsrc;
    a.deg = deg;
    a.cnt = cnt;
    a.jlo = jlo;
    a.nj = nj;
    a.work_ctr = &g.state->work_ctr[large ? 3 : 2];
    a.err = &g.state->err;
    a.updates = &g.state->updates;
    a.bytes = &g.state->bytes[kProfBfs];
    kern<<<(int)grid, threads, dyn, s>>>(a);
    count_launch(g, 1);
    return KH_OK;
}

int launch_init2(Graph& g, int32_t* deg, int32_t* cnt, int jlo, int nj, cudaStream_t s) {
    k_init2<<<g.ctx->sm_count * 4, 256, 0, s>>>(g.rowptr, g.rank, g.n, deg, cnt, jlo, nj);
    count_launch(g, 1);
    return KH_OK;
}

__global__ void k_crank(const int32_t* __restrict__ col, const uint8_t* __restrict__ rank, int64_t nnz,
                        uint8_t* __restrict__ crank) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nnz; k += stride)
        crank[k] = rank[col[k]];
}

int ensure_crank(Graph& g, cudaStream_t s) {
    if (g.crank_valid || g.nnz == 0) return KH_OK;
    int rc;
    if (!g.crank && (rc = alloc_bytes(g.ctx, (void**)&g.crank, (size_t)g.nnz, "column ranks"))) return rc;
    k_crank<<<g.ctx->sm_count * 8, 256, 0, s>>>(g.col, g.rank, g.nnz, g.crank);
    count_launch(g, 1);
    g.crank_valid = true;
    return KH_OK;
}

int launch_hdeg2_slice(Graph& g, int32_t* deg, int32_t* cnt, int jlo, int nj, cudaStream_t s,
                       int slices, int threads, const int32_t* order, int64_t nsrc, bool init) {
    if (g.n == 0) return KH_OK;
    const int64_t width = hdeg2_width(g.n, slices);
    const size_t dyn = hdeg2_smem(width);
    if (dyn > (size_t)kSmem2Max) return set_error(g.ctx, KH_EINVAL, "slice too wide for shared memory");
    void (*kern)(Slice2Args) = cnt ? k_hdeg2_slice<true> : k_hdeg2_slice<false>;
    KH_CUDA_TRY(g.ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)kSmem2Max));
    int per_sm = 0;
    KH_CUDA_TRY(g.ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, dyn));
    if (per_sm < 1) return set_error(g.ctx, KH_EINVAL, "slice kernel does not fit on an SM");
    int64_t grid = (int64_t)g.ctx->sm_count * per_sm;
    const int64_t items = nsrc * slices;
    if (grid > items) grid = items;
    if (grid < 1) grid = 1;
    if (init) {
        k_init2<<<g.ctx->sm_count * 4, 256, 0, s>>>(g.rowptr, g.rank, g.n, deg, cnt, jlo, nj);
        count_launch(g, 1);
    }
    KH_CUDA_TRY(g.ctx, cudaMemsetAsync(&g.state->work_ctr[2], 0, sizeof(int), s));
    if (items == 0) return KH_OK;
    Slice2Args a{};
    a.rowptr = g.rowptr;
    a.col = g.col;
    a.rank = g.rank;
    a.n = g.n;
    a.nslices = slices;
    a.width = width;
    a.order = order;
    a.nsrc = nsrc;
    a.deg = deg;
    a.cnt = cnt;
    a.jlo = jlo;
    a.nj = nj;
    a.work_ctr = &g.state->work_ctr[2];
    a.err = &g.state->err;
    a.updates = &g.state->updates;
    a.bytes = &g.state->bytes[kProfBfs];
    prof_begin(g, kProfBfs, s);
    kern<<<(int)grid, threads, dyn, s>>>(a);
    count_launch(g, 1);
    prof_end(g, kProfBfs, s);
    return KH_OK;
}

}  // namespace kh
