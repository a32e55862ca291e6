// One distance level d of the pull construction (Algorithm PULL; Theorem
// "Distance Dependency"; Lemma "Propagation"; pruning rules 1 and 2; Label
// Elimination and Label Merging; cost-function schedule).
//
// k_dense_prefix / k_cost_arcs / k_cost_vertices / k_bucket_fill
//   For every arc u->v: how many entries of L_{d-1}(v) have a hub ranked
//   above u. Level segments are hub-sorted, so rule 1 keeps a prefix, found
//   by binary search. The pull of the arc also skips the entries whose hub
//   lies below u's dense prefix (every rank id up to it is a hub of
//   L_<d(u), so the membership test of step 2 would drop those entries),
//   found by a second binary search. Per vertex the sum is the
//   pulled-entry count (the paper's cost function); active vertices are
//   bucketed by it so that the most expensive ones start first.
//
// k_level  (one CTA per vertex, persistent CTAs taking vertices in bucket
//   order from a work counter, or one CTA per vertex when granular)
//   1. The label map of u: which hubs x are in L_<d(u), and at which
//      distance. Cumulative bitmaps B_j = {x : d_u(x) <= j}, j = 1..d-1,
//      when they fit on chip; otherwise a binary search in u's level
//      segments, with per-level bitmaps over the highest-ranked ids cached
//      on chip; or (on request) an open-addressing hash x -> d_u(x).
//   2. Pull: the arcs of u are staged in chunks, their pulled-entry counts
//      prefix-summed, and the flattened entries split evenly over the
//      warps. An entry (h, d-1, c) whose hub h is already in L_<d(u) is
//      dropped before its count is read: then Query(h, u) <= d_u(h) < d,
//      so rule 2 would prune it (Label Elimination at no cost). The others
//      are merged per hub in an on-chip hash (count += c mod 2^64; the
//      overflow flag takes the entry's flag and the carry: Label Merging).
//   3a. d = 3: rule 2 asks for a common neighbour of u and h ranked above
//      h; the rows of u's higher-ranked neighbours are walked once and the
//      candidates met there are marked.
//   3. Otherwise: landmark filter (Section "Landmark-Based Filtering"),
//      when the build has landmark distances: a candidate h with
//      sd(u,l) + sd(l,h) < d for a landmark l is pruned at once, one with
//      |sd(u,l) - sd(l,h)| >= d survives at once; the others
//      go on. Prune (rule 2) for every remaining candidate h. A common
//      hub x of L_<d(u) and L_<d(h) with d_u(x) + d_h(x) < d exists iff
//      some x in L_k(h), 1 <= k <= d-2, has d_u(x) <= d-1-k (the case
//      k = 0, x = h, was handled in step 2; entries of h at distance d-1
//      cannot help because d_u(x) >= 1 for x != u). Groups of lanes take
//      candidates from a shared counter and scan these segments in level
//      order with early exit: 8 lanes level by level when u has many
//      candidates; 16 or 32 lanes over G levels' descriptors read at once,
//      scanned as one list, when it has few (deep levels of high-diameter
//      graphs), so that their lanes stay busy; in deep or busy levels they are
//      queued for k_scan_deferred.
//      At a level that has a distance ball (pspc_ball.cu) one bit of u's row
//      stands for step 1, the membership test and all of rule 2.
//   4. Survivors are put in hub order (the rank of a hub is a popcount over
//      a bitmap of the survivors, or a bitonic sort when that bitmap does
//      not fit) and appended to the label arena as L_d(u); the arena slot
//      comes from one atomic add.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <limits.h>

#include "pspc_level.cuh"

namespace cg = cooperative_groups;

namespace pspc {

constexpr int kProbeUnroll = 4;  // loads in flight per lane in the prune scan
constexpr uint32_t kSegCacheMinWords = 1024;  // narrowest useful level cache (32K ids)
constexpr uint32_t kSegCacheMaxWords = 8192;  // widest (the off-chip tables can be far larger)
constexpr int kGatherUnroll = 4; // loads in flight per lane in the pull
constexpr unsigned kRouteSamples = 64;  // on-chip attempts per size class before routing by their outcome
constexpr uint32_t kPrunedBit = 0x80000000u;  // list entry: candidate pruned by rule 2
constexpr uint32_t kProvenBit = 0x40000000u;  // list entry: survival proven by the landmarks
constexpr uint32_t kSlotMask = 0x3FFFFFFFu;

// ---------------------------------------------------------------------------
// Cost (rule 1 prefix per arc) and classification.

__global__ void k_arc_src(const int64_t* __restrict__ rp, int64_t n, int32_t* __restrict__ arc_src) {
    const int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (u >= n) return;
    for (int64_t a = rp[u] + lane; a < rp[u + 1]; a += 32) arc_src[a] = (int32_t)u;
}

// First index of the hub-sorted segment h[0..len) whose hub is >= x.
__device__ __forceinline__ uint32_t seg_lower_bound(const uint32_t* h, uint32_t len, uint32_t x) {
    uint32_t lo = 0, hi = len;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if ((__ldg(h + mid) & kHubMask) < x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// What a level starts from: its row of segments, the pulled-entry sums and the
// status (and the next level's) cleared, the arena filled up to `bump` (one launch instead of three
// memsets and a copy: 128 levels of grid 61x67 spent 0.8 ms on them).
__global__ void __launch_bounds__(256) k_level_begin(int64_t n, uint64_t* __restrict__ seg_row, int64_t* __restrict__ raw_u,
                                                     LevelStatus* __restrict__ stt, LevelStatus* __restrict__ next,
                                                     unsigned long long bump) {
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u < n) {
        seg_row[u] = 0ull;
        raw_u[u] = 0;
    }
    if (blockIdx.x == 0) {
        static_assert(sizeof(LevelStatus) % 4 == 0, "cleared by words");
        for (int i = threadIdx.x; i < (int)(sizeof(LevelStatus) / 4); i += blockDim.x) ((uint32_t*)stt)[i] = ((uint32_t*)next)[i] = 0u;
        __syncthreads();
        if (threadIdx.x == 0) stt->bump = bump;
    }
}

cudaError_t launch_level_begin(int64_t n, uint64_t* seg_row, int64_t* raw_u, LevelStatus* stt, LevelStatus* next,
                               unsigned long long bump, cudaStream_t st) {
    k_level_begin<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, seg_row, raw_u, stt, next, bump);
    return cudaGetLastError();
}

__global__ void k_cost_arcs(int64_t arcs, const int32_t* __restrict__ arc_src, const int32_t* __restrict__ col,
                            const uint64_t* __restrict__ seg_prev, const uint32_t* __restrict__ hub_arena,
                            const int32_t* __restrict__ hpre, uint32_t* __restrict__ arc_lo,
                            uint32_t* __restrict__ cnt_arc, unsigned long long* __restrict__ raw_u,
                            unsigned long long* __restrict__ skipped) {
    __shared__ unsigned long long s_skip;
    if (threadIdx.x == 0) s_skip = 0;
    __syncthreads();
    const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (a < arcs) {
        const uint32_t u = (uint32_t)arc_src[a];
        const uint64_t s = __ldg(seg_prev + col[a]);
        const uint32_t* h = hub_arena + seg_start(s);
        const uint32_t end = seg_lower_bound(h, seg_len(s), u);  // rule 1: hubs ranked above u
        uint32_t lo = 0;
        if (hpre) {
            lo = seg_lower_bound(h, end, (uint32_t)__ldg(hpre + u));
            arc_lo[a] = lo;
            if (lo) atomicAdd(&s_skip, (unsigned long long)lo);
        }
        cnt_arc[a] = end - lo;
        if (end > lo) atomicAdd(raw_u + u, (unsigned long long)(end - lo));
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_skip) atomicAdd(skipped, s_skip);
}

// Warp per vertex: a bitmap of the first kDensePrefixWindow ids of u's
// graph, set for every hub of L_0(u) .. L_{d-1}(u) in that window (the
// segments are hub-sorted, so each lane stops at the window's end); the
// first clear bit is the dense prefix.
constexpr int kPrefixWarps = 8;

__global__ void __launch_bounds__(kPrefixWarps * 32)
    k_dense_prefix(int d, int64_t n, const uint64_t* __restrict__ seg, const uint32_t* __restrict__ hub_arena,
                   const int32_t* __restrict__ comp_base, int32_t* __restrict__ hpre) {
    __shared__ uint32_t bits[kPrefixWarps][kDensePrefixWindow / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t u = (int64_t)blockIdx.x * kPrefixWarps + w;
    if (u >= n) return;  // the whole warp
    const uint32_t cb = comp_base ? (uint32_t)__ldg(comp_base + u) : 0u;
    const uint32_t lim = cb + kDensePrefixWindow;
    bits[w][lane] = 0u;
    __syncwarp();
    for (int l = 0; l < d; ++l) {
        const uint64_t s = __ldg(seg + (int64_t)l * n + u);
        const uint32_t len = seg_len(s);
        const uint32_t* hs = hub_arena + seg_start(s);
        for (uint32_t i = lane; i < len; i += 32) {
            const uint32_t x = __ldg(hs + i) & kHubMask;
            if (x >= lim) break;
            atomicOr(&bits[w][(x - cb) >> 5], 1u << ((x - cb) & 31));
        }
    }
    __syncwarp();
    const uint32_t word = bits[w][lane];
    const unsigned open = __ballot_sync(0xFFFFFFFFu, word != 0xFFFFFFFFu);
    uint32_t H = lim;
    if (open) {
        const int k = __ffs(open) - 1;
        const uint32_t wk = __shfl_sync(0xFFFFFFFFu, word, k);
        H = cb + 32u * k + (uint32_t)(__ffs(~wk) - 1);
    }
    if (lane == 0) hpre[u] = (int32_t)(H < (uint32_t)u ? H : (uint32_t)u);
}

// Bucket of a vertex: floor(log2 pulled entries) (at most kDenseBucket - 1),
// or kDenseBucket more for the dense kernel's vertices, which come first.
__device__ __forceinline__ int bucket_of(const DenseRule& R, int64_t raw, int64_t span, int64_t deg) {
    const int b = 63 - __clzll((unsigned long long)raw);
    if (dense_vertex(R, raw, span, deg)) return kDenseBucket + b;
    return b < kDenseBucket ? b : kDenseBucket - 1;
}

// Totals and bucket sizes are summed per block on chip, one global atomic
// for each that is not zero: with one for every vertex the pass was bound by
// atomics on the same few words (65,536 vertices: 81 us and 22 us for the
// two kernels, now 5 and 4).
// The caller's thread has vertex u with `raw` pulled entries if `mine`; all
// threads of the block take part.
__device__ __forceinline__ void cost_sums(bool mine, int64_t u, unsigned long long raw, const int64_t* __restrict__ rp,
                                          const uint64_t* __restrict__ seg_prev, int64_t* __restrict__ lab_size,
                                          LevelStatus* stt, int64_t label_limit, const DenseRule& dense,
                                          int32_t* __restrict__ glist) {
    __shared__ int s_bucket[kBuckets];
    __shared__ unsigned long long s_raw, s_arcs, s_need_d;
    __shared__ int s_active;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < kBuckets) s_bucket[tid] = 0;
    if (tid == 0) {
        s_raw = s_arcs = s_need_d = 0;
        s_active = 0;
    }
    __syncthreads();
    unsigned long long arcs = 0, need_d = 0;
    if (mine) {
        const int64_t ls = lab_size[u] + seg_len(seg_prev[u]);
        lab_size[u] = ls;
        if (raw) {
            arcs = (unsigned long long)(rp[u + 1] - rp[u]);
            if (ls <= label_limit) {
                const int64_t span = u - (dense.comp_base ? dense.comp_base[u] : 0);
                const int b = bucket_of(dense, (int64_t)raw, span, (int64_t)arcs);
                if (b >= kDenseBucket) need_d = min(raw, (unsigned long long)span);
                atomicAdd(&s_bucket[b], 1);
            } else {
                const int p = atomicAdd(&stt->n_global, 1);
                glist[p] = (int32_t)u;
                atomicMax(&stt->need_cap_u, (unsigned long long)label_cap_for(ls));
                atomicMax(&stt->need_cap_c, (unsigned long long)cand_cap_for((int64_t)raw, u, 1u << 30));
            }
        }
    }
    const unsigned active = __ballot_sync(0xFFFFFFFFu, raw != 0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        raw += __shfl_xor_sync(0xFFFFFFFFu, raw, o);
        arcs += __shfl_xor_sync(0xFFFFFFFFu, arcs, o);
        need_d = max(need_d, __shfl_xor_sync(0xFFFFFFFFu, need_d, o));
    }
    if (lane == 0 && active) {
        atomicAdd(&s_raw, raw);
        atomicAdd(&s_arcs, arcs);
        atomicAdd(&s_active, __popc(active));
        if (need_d) atomicMax(&s_need_d, need_d);
    }
    __syncthreads();
    if (tid < kBuckets && s_bucket[tid]) {
        atomicAdd(&stt->bucket_cnt[tid], s_bucket[tid]);
        atomicAdd(&stt->n_smem, s_bucket[tid]);
    }
    if (tid == 0 && s_active) {
        atomicAdd(&stt->raw_total, s_raw);
        atomicAdd(&stt->active_arcs, s_arcs);
        atomicAdd(&stt->n_active, s_active);
        if (s_need_d) atomicMax(&stt->need_cap_d, s_need_d);
    }
}

// max_deg: NULL, or where the largest degree goes.
__global__ void __launch_bounds__(256)
    k_cost_vertices(int64_t n, const int64_t* __restrict__ rp, const uint64_t* __restrict__ seg_prev,
                    const int64_t* __restrict__ raw_u, int64_t* __restrict__ lab_size, LevelStatus* stt,
                    int64_t label_limit, const DenseRule dense, int32_t* __restrict__ glist, int* max_deg) {
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool mine = u < n;
    if (max_deg) {
        const int64_t deg = mine ? rp[u + 1] - rp[u] : 0;
        const int most = __reduce_max_sync(0xFFFFFFFFu, (int)min(deg, (int64_t)INT_MAX));
        if ((threadIdx.x & 31) == 0 && most > *(volatile int*)max_deg) atomicMax(max_deg, most);
    }
    cost_sums(mine, u, mine ? (unsigned long long)raw_u[u] : 0ull, rp, seg_prev, lab_size, stt, label_limit, dense, glist);
}

// A level's start and its cost pass in one launch, for graphs of small
// degrees (at most kCostMaxDegree): kCostLanes lanes walk a vertex's arcs, so
// its pulled entries need no atomics and no sums cleared before. `stt` was
// cleared by the level before; `next`, the level after's, is cleared here.
// Three launches of 2 to 4 us each became one: 122 levels of grid 61x67
// 8.3 -> 7.6 ms, 2,111 of grid 16x2000 156 -> 144.
constexpr int kCostLanes = 4;
constexpr int kCostThreads = 512;

__global__ void __launch_bounds__(kCostThreads)
    k_cost_level(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                 const uint64_t* __restrict__ seg_prev, uint64_t* __restrict__ seg_row,
                 const uint32_t* __restrict__ hub_arena, const int32_t* __restrict__ hpre, uint32_t* __restrict__ arc_lo,
                 uint32_t* __restrict__ cnt_arc, int64_t* __restrict__ raw_u, int64_t* __restrict__ lab_size,
                 LevelStatus* stt, LevelStatus* next, unsigned long long bump, int64_t label_limit, const DenseRule dense,
                 int32_t* __restrict__ glist) {
    const int64_t u = ((int64_t)blockIdx.x * kCostThreads + threadIdx.x) / kCostLanes;
    const int gl = threadIdx.x % kCostLanes;
    if (blockIdx.x == 0) {
        for (int i = threadIdx.x; i < (int)(sizeof(LevelStatus) / 4); i += kCostThreads) ((uint32_t*)next)[i] = 0u;
        if (threadIdx.x == 0) stt->bump = bump;
    }
    unsigned long long raw = 0, skip = 0;
    if (u < n) {
        for (int64_t a = rp[u] + gl; a < rp[u + 1]; a += kCostLanes) {
            const uint64_t s = __ldg(seg_prev + __ldg(col + a));
            const uint32_t* h = hub_arena + seg_start(s);
            const uint32_t end = seg_lower_bound(h, seg_len(s), (uint32_t)u);  // rule 1, as in k_cost_arcs
            uint32_t lo = 0;
            if (hpre) {
                lo = seg_lower_bound(h, end, (uint32_t)__ldg(hpre + u));
                arc_lo[a] = lo;
                skip += lo;
            }
            cnt_arc[a] = end - lo;
            raw += end - lo;
        }
    }
#pragma unroll
    for (int o = kCostLanes / 2; o > 0; o >>= 1) raw += __shfl_xor_sync(0xFFFFFFFFu, raw, o);
    if (hpre) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) skip += __shfl_xor_sync(0xFFFFFFFFu, skip, o);
        if ((threadIdx.x & 31) == 0 && skip) atomicAdd(&stt->prefix_skipped, skip);
    }
    const bool mine = u < n && gl == 0;
    if (mine) {
        raw_u[u] = (int64_t)raw;
        seg_row[u] = 0ull;
    }
    cost_sums(mine, u, mine ? raw : 0ull, rp, seg_prev, lab_size, stt, label_limit, dense, glist);
}

// Items bucket by bucket, most expensive first. Every block finds the
// buckets' bases from their sizes itself.
__global__ void __launch_bounds__(256)
    k_bucket_fill(int64_t n, const int64_t* __restrict__ rp, const int64_t* __restrict__ raw_u,
                  const int64_t* __restrict__ lab_size, LevelStatus* stt, int64_t label_limit, const DenseRule dense,
                  int32_t* __restrict__ items) {
    __shared__ int s_cnt[kBuckets], s_base[kBuckets];
    const int tid = threadIdx.x;
    if (tid < kBuckets) s_cnt[tid] = 0;
    __syncthreads();
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + tid;
    int b = -1, at = 0;
    if (u < n) {
        const int64_t raw = raw_u[u];
        if (raw != 0 && lab_size[u] <= label_limit) {
            const int64_t span = u - (dense.comp_base ? dense.comp_base[u] : 0);
            b = bucket_of(dense, raw, span, rp[u + 1] - rp[u]);
            at = atomicAdd(&s_cnt[b], 1);
        }
    }
    __syncthreads();
    if (tid < kBuckets && s_cnt[tid]) {
        int base = 0;
        for (int k = tid + 1; k < kBuckets; ++k) base += stt->bucket_cnt[k];
        s_base[tid] = base + atomicAdd(&stt->bucket_fill[tid], s_cnt[tid]);
    }
    __syncthreads();
    if (b >= 0) items[s_base[b] + at] = (int32_t)u;
}

// ---------------------------------------------------------------------------
// Label maps of L_<d(u).

struct BitMap {
    uint32_t* bits;  // (d-1) bitmaps of `words` words; bitmap j-1 = {x : d_u(x) <= j}
    uint32_t words;
    int d;
    uint32_t base;   // first id of u's graph: bits index x - base
    __device__ void clear() const {
        const uint32_t total = (uint32_t)(d - 1) * words;
        for (uint32_t i = threadIdx.x; i < total; i += blockDim.x) bits[i] = 0u;
    }
    __device__ void insert(uint32_t x, int l) const {
        if (l == 0) return;  // u itself is never a candidate or a witness
        x -= base;
        const uint32_t m = 1u << (x & 31);
        for (int j = l; j <= d - 1; ++j) atomicOr(&bits[(uint32_t)(j - 1) * words + (x >> 5)], m);
    }
    __device__ bool within(uint32_t x, int thr) const {  // d_u(x) <= thr, 1 <= thr <= d-1
        x -= base;
        return (bits[(uint32_t)(thr - 1) * words + (x >> 5)] >> (x & 31)) & 1u;
    }
    __device__ bool member(uint32_t x) const { return d > 1 && within(x, d - 1); }
};

struct HashMap {
    uint32_t* keys;
    uint16_t* lvl;
    uint32_t cap;
    __device__ void clear() const {
        for (uint32_t i = threadIdx.x; i < cap; i += blockDim.x) keys[i] = kEmpty;
    }
    __device__ void insert(uint32_t x, int l) const {
        uint32_t slot = hash_hub(x) & (cap - 1);
        for (uint32_t probe = 0; probe < cap; ++probe) {
            const uint32_t k = atomicCAS(&keys[slot], kEmpty, x);
            if (k == kEmpty || k == x) {
                lvl[slot] = (uint16_t)l;
                return;
            }
            slot = (slot + 1) & (cap - 1);
        }
    }
    __device__ uint32_t lookup(uint32_t x) const {
        uint32_t slot = hash_hub(x) & (cap - 1);
        for (uint32_t probe = 0; probe < cap; ++probe) {
            const uint32_t k = keys[slot];
            if (k == x) return lvl[slot];
            if (k == kEmpty) return 0xFFFFu;
            slot = (slot + 1) & (cap - 1);
        }
        return 0xFFFFu;
    }
    __device__ bool within(uint32_t x, int thr) const { return lookup(x) <= (uint32_t)thr; }
    __device__ bool member(uint32_t x) const { return lookup(x) != 0xFFFFu; }
};

// No map at all: a pulled hub h can only be in L(u) at distance d-2 or d-1
// (it is at distance d-1 from a neighbour), and a witness x in L_k(h) can
// only be at distance d-2-k or d-1-k from u (triangle inequality with
// sd(u,h) >= d-2). So two binary searches in u's hub-sorted level segments
// answer every test, and nothing is built per vertex.
// u's row of the ball, and whether it holds id x (cbase: first id of u's graph).
__device__ __forceinline__ const uint32_t* ball_of(const LevelArgs& A, int64_t u) {
    return A.ball ? A.ball + (A.ball_rows.off ? __ldg(A.ball_rows.off + u) : u * A.ball_rows.words) : nullptr;
}
__device__ __forceinline__ bool in_ball(const uint32_t* row, uint32_t r) { return (__ldg(row + (r >> 5)) >> (r & 31)) & 1u; }

struct SegMap {
    const uint64_t* seg;
    const uint32_t* hub_arena;
    int64_t n, u;
    int d;
    // Optional on-chip cache: one bitmap per level 1..d-1 over the ids
    // base .. base + 32*cwords - 1 (the highest-ranked hubs, which hold
    // most label entries of power-law graphs); NULL when not built.
    const uint32_t* cache;
    uint32_t cwords;
    uint32_t base;
    __device__ bool in_level(uint32_t x, int l) const {
        if (l < 1) return false;  // level 0 is u itself
        if (cache && x - base < 32u * cwords) {
            const uint32_t r = x - base;
            return (cache[(uint32_t)(l - 1) * cwords + (r >> 5)] >> (r & 31)) & 1u;
        }
        const uint64_t s = __ldg(seg + (int64_t)l * n + u);
        const uint32_t* h = hub_arena + seg_start(s);
        uint32_t lo = 0, hi = seg_len(s);
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if ((__ldg(h + mid) & kHubMask) < x) lo = mid + 1; else hi = mid;
        }
        return lo < seg_len(s) && (__ldg(h + lo) & kHubMask) == x;
    }
    __device__ bool within(uint32_t x, int thr) const { return in_level(x, thr) || in_level(x, thr - 1); }
    __device__ bool member(uint32_t x) const { return in_level(x, d - 1) || in_level(x, d - 2); }
};

// ---------------------------------------------------------------------------
// Block helpers.

__device__ __forceinline__ bool cand_insert(uint32_t* keys, unsigned long long* cnts, uint32_t cap, uint32_t limit,
                                            uint32_t h, uint64_t c, uint32_t ovf, int* nkeys, int* abort_flag) {
    uint32_t slot = hash_hub(h) & (cap - 1);
    for (uint32_t probe = 0; probe < cap; ++probe) {
        uint32_t k = ((volatile uint32_t*)keys)[slot];
        if (k == kEmpty) {
            if (*(volatile int*)abort_flag) return false;
            k = atomicCAS(&keys[slot], kEmpty, h);
            if (k == kEmpty) {
                if ((uint32_t)(atomicAdd(nkeys, 1) + 1) > limit) *(volatile int*)abort_flag = 1;
                k = h;
            }
        }
        if ((k & kHubMask) == h) {
            const unsigned long long old = atomicAdd(&cnts[slot], (unsigned long long)c);
            if (ovf | (old + c < old)) atomicOr(&keys[slot], kOvfBit);
            return true;
        }
        slot = (slot + 1) & (cap - 1);
    }
    *(volatile int*)abort_flag = 1;
    return false;
}

// A count as LevelStatus::cmax keeps it: saturated where it or its flag
// says 2^32 or more.
__device__ __forceinline__ uint32_t count_bound(uint64_t c, uint32_t ovf) {
    return (ovf != 0 || (c >> 32) != 0) ? 0xFFFFFFFFu : (uint32_t)c;
}

__device__ __forceinline__ long long warp_incl_scan64(long long v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Exclusive scan of a[0..n) (n <= blockDim.x) in place; a[n] = total.
__device__ long long block_excl_scan(long long* a, int n, long long* wsum) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const long long v = tid < n ? a[tid] : 0;
    const long long incl = warp_incl_scan64(v);
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        long long t = lane < nw ? wsum[lane] : 0;
        t = warp_incl_scan64(t);
        if (lane < nw) wsum[lane] = t;
    }
    __syncthreads();
    const long long total = wsum[nw - 1];
    if (tid < n) a[tid] = incl - v + (warp ? wsum[warp - 1] : 0);
    if (tid == 0) a[n] = total;
    __syncthreads();
    return total;
}

// Exclusive prefix of popcounts of bits[0..W) into wp[0..W); returns the
// total number of set bits. Each thread owns a contiguous run of words.
__device__ long long block_excl_scan_popc(const uint32_t* bits, uint32_t* wp, uint32_t W, long long* wsum) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const uint32_t per = (W + blockDim.x - 1) / blockDim.x;
    const uint32_t w0 = tid * per, w1 = w0 + per < W ? w0 + per : W;
    long long v = 0;
    for (uint32_t i = w0; i < w1; ++i) v += __popc(bits[i]);
    const long long incl = warp_incl_scan64(v);
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        long long t = lane < nw ? wsum[lane] : 0;
        t = warp_incl_scan64(t);
        if (lane < nw) wsum[lane] = t;
    }
    __syncthreads();
    const long long total = wsum[nw - 1];
    long long run = incl - v + (warp ? wsum[warp - 1] : 0);
    for (uint32_t i = w0; i < w1; ++i) {
        wp[i] = (uint32_t)run;
        run += __popc(bits[i]);
    }
    __syncthreads();
    return total;
}

// Rule 2 over levels klo..khi of L(h) for one candidate h, by one group of
// G lanes. Lane j reads the descriptor of level k0 + j (G at a time); the
// lengths are prefix-summed over the group and the concatenated entries
// scanned in level order, kProbeUnroll loads in flight per lane. The level of
// entry i is the last lane whose exclusive prefix is <= i (a binary search
// by shuffles). An entry x of level k is a witness iff d_u(x) <= d-1-k.
// Returns whether the group found a witness; it also stops (returning
// false) once *stop, shared with other groups scanning other levels of the
// same candidate, is set.
template <int G, class Map>
__device__ bool scan_levels(const Map& mp, const uint64_t* __restrict__ seg, const uint32_t* __restrict__ hub_arena,
                            int64_t n, int d, uint32_t h, int klo, int khi, const int* stop) {
    auto tile = cg::tiled_partition<G>(cg::this_thread_block());
    const int gl = tile.thread_rank();
    bool pruned = false, halt = false;
    for (int k0 = klo; k0 <= khi && !pruned && !halt; k0 += G) {
        const int k = k0 + gl;
        const uint64_t s = k <= khi ? __ldg(seg + (int64_t)k * n + h) : 0ull;
        const uint32_t len = seg_len(s);
        const unsigned long long start = seg_start(s);
        uint32_t incl = len;
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            const uint32_t t = tile.shfl_up(incl, o);
            if (gl >= o) incl += t;
        }
        const uint32_t excl = incl - len;
        const uint32_t total = tile.shfl(incl, G - 1);
        for (uint32_t b = 0; b < total && !pruned && !halt; b += G * kProbeUnroll) {
            uint32_t x[kProbeUnroll];
            int thr[kProbeUnroll];
#pragma unroll
            for (int t = 0; t < kProbeUnroll; ++t) {
                const uint32_t i = b + t * G + gl;
                int j = 0;
#pragma unroll
                for (int step = G >> 1; step > 0; step >>= 1) {
                    const uint32_t e = tile.shfl(excl, j + step);
                    if (e <= i) j += step;
                }
                const unsigned long long sj = tile.shfl(start, j);
                const uint32_t ej = tile.shfl(excl, j);
                thr[t] = d - 1 - (k0 + j);
                x[t] = i < total ? (__ldg(hub_arena + sj + (i - ej)) & kHubMask) : kEmpty;
            }
            bool hit = false;
#pragma unroll
            for (int t = 0; t < kProbeUnroll; ++t)
                if (x[t] != kEmpty) hit |= mp.within(x[t], thr[t]);
            pruned = tile.any(hit);
            if (stop) halt = tile.any(*(volatile const int*)stop != 0);
        }
    }
    return pruned;
}

// Rule 2 over levels klo..khi of L(h) against u's label, by one warp and
// without a map of u. A witness x of L_k(h) lies in L_l(u) with l = d-1-k or
// d-2-k (see SegMap), so 31 levels of h meet 32 levels of u. The (hub, level)
// pairs of h set bits of a filter on chip, u's entries probe it for their two
// levels, and the few that find a bit are looked up in L_k(h) together, a
// match to a lane. What bounds it is the latency of loads that miss L2 (the
// labels of a large index do not fit): a search of u's segments for each entry
// of h was a chain of ten of them, here a step of 31 levels has two, the
// descriptors and then both labels' entries, kScanUnroll rows of each in
// flight, and the next step's descriptors are read meanwhile. Returns whether
// a witness was found (or, then possibly false, *stop was set).
// mem: `words` words of filter (a power of two), then kScanHits of matches.
constexpr int kScanUnroll = 4;          // rows of 32 entries in flight
constexpr uint32_t kScanHits = 64;      // matches kept until they are looked up
constexpr uint32_t kMicroFilter = 256;  // filter words per warp of the warp-per-vertex kernel,
constexpr uint32_t kDeepFilter = 256;   // of the light kernel's deep form,
constexpr uint32_t kScanFilter = 1024;  // and of the deferred scans

__device__ bool scan_filtered(uint32_t* mem, uint32_t words, const uint64_t* __restrict__ seg,
                              const uint32_t* __restrict__ hub_arena, int64_t n, int64_t u, int d, uint32_t h, int klo,
                              int khi, const int* stop) {
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t* filter = mem;
    uint32_t* hits = mem + words;
    const int shift = __clz(words) - 4;  // a hash's top bits: 32 per word
    auto bit_of = [&](uint32_t x, int j) { return (x * 0x9E3779B1u + (uint32_t)j * 0x85EBCA6Bu) >> shift; };
    // segment of entry i of the concatenated segments: the last lane whose
    // exclusive prefix is at most i
    auto locate = [&](uint32_t excl, uint32_t i) {
        int j = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
            const uint32_t e = __shfl_sync(FULL, excl, j + step);
            if (e <= i) j += step;
        }
        return j;
    };
    auto seg_h = [&](int k0) { return lane < 31 && k0 + lane <= khi ? __ldg(seg + (int64_t)(k0 + lane) * n + h) : 0ull; };
    auto seg_u = [&](int k0) {
        const int k = k0 + lane, l = d - 1 - k;
        return l >= 1 && k <= khi + 1 ? __ldg(seg + (int64_t)l * n + u) : 0ull;
    };
    uint64_t sa = seg_h(klo), sb = seg_u(klo);
    for (int k0 = klo; k0 <= khi; k0 += 31) {
        const uint64_t ca = sa, cb = sb;
        if (k0 + 31 <= khi) {
            sa = seg_h(k0 + 31);
            sb = seg_u(k0 + 31);
        }
        uint32_t ia = seg_len(ca), ib = seg_len(cb);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t ta = __shfl_up_sync(FULL, ia, o), tb = __shfl_up_sync(FULL, ib, o);
            if (lane >= o) {
                ia += ta;
                ib += tb;
            }
        }
        const uint32_t ea = ia - seg_len(ca), eb = ib - seg_len(cb);
        const uint32_t na = __shfl_sync(FULL, ia, 31), nb = __shfl_sync(FULL, ib, 31);
        if (na == 0 || nb == 0) continue;
        const uint64_t pa = seg_start(ca) - ea, pb = seg_start(cb) - eb;
        // entry word: hub | lane of its segment << 24; kEmpty for none
        auto load_rows = [&](uint32_t (&x)[kScanUnroll], uint32_t b, uint32_t end, uint32_t excl, uint64_t base) {
            int j[kScanUnroll];
#pragma unroll
            for (int t = 0; t < kScanUnroll; ++t) {
                x[t] = kEmpty;
                j[t] = 0;
                if (b + t * 32 >= end) continue;  // warp-uniform
                const uint32_t i = b + t * 32 + lane;
                j[t] = locate(excl, i);
                const uint64_t pj = __shfl_sync(FULL, base, j[t]);
                if (i < end) x[t] = __ldg(hub_arena + pj + i);
            }
#pragma unroll
            for (int t = 0; t < kScanUnroll; ++t)
                if (b + t * 32 + lane < end) x[t] = (x[t] & kHubMask) | (uint32_t)j[t] << 24;
        };
        uint32_t xb[kScanUnroll];
        load_rows(xb, 0, nb, eb, pb);
        for (uint32_t i = lane; i < words / 4; i += 32) ((uint4*)filter)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        for (uint32_t b = 0; b < na; b += 32 * kScanUnroll) {
            uint32_t xa[kScanUnroll];
            load_rows(xa, b, na, ea, pa);
#pragma unroll
            for (int t = 0; t < kScanUnroll; ++t)
                if (xa[t] != kEmpty) {
                    const uint32_t bit = bit_of(xa[t] & kHubMask, (int)(xa[t] >> 24));
                    atomicOr(&filter[bit >> 5], 1u << (bit & 31));
                }
        }
        __syncwarp();
        int nh = 0;  // matches kept
        bool found = false, halt = false;
        auto look_up = [&]() {  // the first 32 kept matches, one to a lane
            __syncwarp();
            bool hit = false;
            if (lane < nh) {
                const uint32_t x = hits[lane] & kHubMask;
                const uint64_t s = __ldg(seg + (int64_t)(k0 + (int)(hits[lane] >> 24)) * n + h);
                const uint32_t at = seg_lower_bound(hub_arena + seg_start(s), seg_len(s), x);
                hit = at < seg_len(s) && (__ldg(hub_arena + seg_start(s) + at) & kHubMask) == x;
            }
            // a nearly full filter fills the list twice in a row of entries:
            // the second look-up must not take back what the first one found
            found |= __any_sync(FULL, hit);
            const uint32_t tail = lane + 32 < nh ? hits[lane + 32] : 0u;
            __syncwarp();
            if (lane + 32 < nh) hits[lane] = tail;
            nh = nh > 32 ? nh - 32 : 0;
        };
        for (uint32_t b = 0; b < nb && !found && !halt; b += 32 * kScanUnroll) {
            if (b) load_rows(xb, b, nb, eb, pb);
#pragma unroll
            for (int t = 0; t < kScanUnroll; ++t) {
                if (b + t * 32 >= nb || found) continue;  // warp-uniform
#pragma unroll
                for (int o = 0; o < 2; ++o) {  // x at level l of u: levels d-1-l and d-2-l of h
                    if (found) continue;  // warp-uniform
                    const int jj = (int)(xb[t] >> 24) - o;
                    bool maybe = false;
                    if (xb[t] != kEmpty && jj >= 0 && jj < 31) {
                        const uint32_t bit = bit_of(xb[t] & kHubMask, jj);
                        maybe = (filter[bit >> 5] >> (bit & 31)) & 1u;
                    }
                    const unsigned m = __ballot_sync(FULL, maybe);
                    if (!m) continue;
                    if (maybe) hits[nh + __popc(m & lt)] = (xb[t] & kHubMask) | (uint32_t)jj << 24;
                    nh += __popc(m);
                    if (nh > 32) look_up();
                }
            }
            if (stop) halt = __any_sync(FULL, *(volatile const int*)stop != 0);
        }
        if (nh > 0 && !found && !halt) look_up();
        __syncwarp();
        if (found) return true;
        if (halt) return false;
    }
    return false;
}

// Rule 2 for the candidates list[0..M): G lanes per candidate h take
// candidates from a shared counter and scan levels 1..d-2 of L(h).
template <int G, class Map>
__device__ void prune_candidates(const Map& mp, const uint64_t* __restrict__ seg,
                                 const uint32_t* __restrict__ hub_arena, int64_t n, int d, uint32_t* list,
                                 const uint32_t* ckeys, const uint32_t* open, int M, int* next) {
    auto tile = cg::tiled_partition<G>(cg::this_thread_block());
    const int gl = tile.thread_rank();
    for (;;) {
        int c = 0;
        if (gl == 0) c = atomicAdd(next, 1);
        c = tile.shfl(c, 0);
        if (c >= M) break;
        if (open) c = (int)open[c];
        const uint32_t slot = list[c];
        if (slot & (kProvenBit | kPrunedBit)) continue;
        const uint32_t h = ckeys[slot] & kHubMask;
        const bool pruned = scan_levels<G>(mp, seg, hub_arena, n, d, h, 1, d - 2, nullptr);
        if (pruned && gl == 0) list[c] = slot | kPrunedBit;
    }
}

// Rule 2 when fewer candidates remain to be scanned than the CTA has warps
// (P < NT/32: the deep levels of high-diameter graphs, where each scan is
// long): the warps form P' >= P groups of wpc = (NT/32) / P' warps, group g takes
// the g-th candidate still undecided, and its warps split levels 1..d-2
// into wpc contiguous ranges. A warp that finds a witness sets the group's
// flag, and the others stop at their next step. Every warp reaches the
// barriers (the call is made by the whole CTA). filters: memory
// on chip per warp for scan_filtered, or NULL (the map is on chip).
template <int NT, class Map>
__device__ void prune_split(const Map& mp, const uint64_t* __restrict__ seg, const uint32_t* __restrict__ hub_arena,
                            int64_t n, int d, uint32_t* list, const uint32_t* ckeys, int M, int P, int* s_flag,
                            uint32_t* filters, int64_t u) {
    constexpr int kWarps = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int wpc = 1;
    while (wpc * 2 * P <= kWarps) wpc *= 2;
    const int groups = kWarps / wpc, g = warp / wpc, j = warp % wpc;
    if (tid < kWarps) s_flag[tid] = 0;
    __syncthreads();
    // position in list of the g-th undecided candidate
    int c = -1;
    if (g < P) {
        int seen = 0;
        for (int base = 0; base < M && c < 0; base += 32) {
            const int i = base + lane;
            const bool open = i < M && !(list[i] & (kProvenBit | kPrunedBit));
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, open);
            const int cnt = __popc(bal);
            if (seen + cnt > g) {
                unsigned m = bal;
                for (int r = g - seen; r > 0; --r) m &= m - 1;
                c = base + __ffs(m) - 1;
            }
            seen += cnt;
        }
    }
    if (c >= 0) {
        const uint32_t h = ckeys[list[c] & kSlotMask] & kHubMask;
        const int levels = d - 2;
        const int klo = 1 + (int)((int64_t)levels * j / wpc), khi = (int)((int64_t)levels * (j + 1) / wpc);
        bool hit = false;
        if (klo <= khi)
            hit = filters ? scan_filtered(filters + warp * (kDeepFilter + kScanHits), kDeepFilter, seg, hub_arena, n, u, d, h, klo, khi, &s_flag[g])
                          : scan_levels<32>(mp, seg, hub_arena, n, d, h, klo, khi, &s_flag[g]);
        if (hit && lane == 0) atomicExch(&s_flag[g], 1);
    }
    __syncthreads();
    if (c >= 0 && j == 0 && lane == 0 && s_flag[g]) list[c] |= kPrunedBit;
    (void)groups;
}

// Rule 2 level by level: G lanes per candidate scan L_1(h), then L_2(h), ...
// (one descriptor read per level), kProbeUnroll loads in flight per lane.
// A witness x in L_k(h) has sd(h,x) = k, and sd(u,h) >= d-2, so d_u(x) is
// d-2-k or d-1-k: x lies in one of u's two level segments thr-1, thr
// (thr = d-1-k; level 0 is u itself, never in L(h)). When those two are
// much shorter than L_k(h), the group scans them instead and looks each
// entry up in L_k(h) (hub-sorted) by binary search. useg holds u's level
// descriptors for levels 0 .. kUSideLevels-1 (NULL: always scan L_k(h)).
constexpr int kUSideLevels = 16;

__device__ __forceinline__ bool seg_contains(const uint32_t* xs, uint32_t len, uint32_t x) {
    uint32_t lo = 0, hi = len;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if ((__ldg(xs + mid) & kHubMask) < x) lo = mid + 1; else hi = mid;
    }
    return lo < len && (__ldg(xs + lo) & kHubMask) == x;
}

template <int G, class Map>
__device__ void prune_by_level(const Map& mp, const uint64_t* __restrict__ seg,
                               const uint32_t* __restrict__ hub_arena, int64_t n, int d, uint32_t* list,
                               const uint32_t* ckeys, const uint32_t* open, int M, int* next, const uint64_t* useg) {
    auto tile = cg::tiled_partition<G>(cg::this_thread_block());
    const int gl = tile.thread_rank();
    for (;;) {
        int c = 0;
        if (gl == 0) c = atomicAdd(next, 1);
        c = tile.shfl(c, 0);
        if (c >= M) break;
        if (open) c = (int)open[c];
        const uint32_t slot = list[c];
        if (slot & (kProvenBit | kPrunedBit)) continue;
        const uint32_t h = ckeys[slot] & kHubMask;
        bool pruned = false;
        for (int k = 1; k <= d - 2 && !pruned; ++k) {
            const uint64_t s = __ldg(seg + (int64_t)k * n + h);
            const uint32_t len = seg_len(s);
            const uint32_t* xs = hub_arena + seg_start(s);
            const int thr = d - 1 - k;
            if (useg && thr < kUSideLevels && len > 0) {
                const uint64_t ua = thr >= 2 ? useg[thr - 1] : 0ull, ub = useg[thr];
                const uint32_t la = seg_len(ua), lb = seg_len(ub);
                const uint32_t steps = 32 - __clz(len);  // binary-search steps in L_k(h)
                if ((uint64_t)(la + lb) * steps < len) {
                    const uint32_t* xa = hub_arena + seg_start(ua);
                    const uint32_t* xb = hub_arena + seg_start(ub);
                    for (uint32_t b = 0; b < la + lb && !pruned; b += G * kProbeUnroll) {
                        bool hit = false;
#pragma unroll
                        for (int t = 0; t < kProbeUnroll; ++t) {
                            const uint32_t i = b + t * G + gl;
                            if (i < la + lb) {
                                const uint32_t x = __ldg(i < la ? xa + i : xb + (i - la)) & kHubMask;
                                hit |= seg_contains(xs, len, x);
                            }
                        }
                        pruned = tile.any(hit);
                    }
                    continue;
                }
            }
            for (uint32_t b = 0; b < len && !pruned; b += G * kProbeUnroll) {
                uint32_t x[kProbeUnroll];
#pragma unroll
                for (int t = 0; t < kProbeUnroll; ++t) {
                    const uint32_t i = b + t * G + gl;
                    x[t] = i < len ? (__ldg(xs + i) & kHubMask) : kEmpty;
                }
                bool hit = false;
#pragma unroll
                for (int t = 0; t < kProbeUnroll; ++t)
                    if (x[t] != kEmpty) hit |= mp.within(x[t], thr);
                pruned = tile.any(hit);
            }
        }
        if (pruned && gl == 0) list[c] = slot | kPrunedBit;
    }
}

// Many candidates: 8 lanes each, level by level (most are pruned within the
// first entries of L_1(h), so reading further descriptors up front only
// costs loads). Few candidates: wider groups over the concatenated levels,
// so that the long scans of deep levels keep all lanes busy. open: the
// positions of the to_scan undecided entries of list[0..M), or NULL (list
// entries that carry a verdict are skipped).
template <int NT, class Map>
__device__ __forceinline__ void prune_all(const Map& mp, const uint64_t* seg, const uint32_t* hub_arena, int64_t n,
                                          int d, uint32_t* list, const uint32_t* ckeys, const uint32_t* open, int M,
                                          int to_scan, int* next, const uint64_t* useg, int* s_flag,
                                          uint32_t* filters, int64_t u) {
    const int items = open ? to_scan : M;
    if (to_scan >= 64) prune_by_level<8>(mp, seg, hub_arena, n, d, list, ckeys, open, items, next, useg);
    else if (to_scan >= NT / 32) prune_candidates<16>(mp, seg, hub_arena, n, d, list, ckeys, open, items, next);
    else prune_split<NT>(mp, seg, hub_arena, n, d, list, ckeys, M, to_scan, s_flag, filters, u);
}

// Landmark filter (Section "Landmark-Based Filtering"). For a candidate h
// of u at level d, rule 2 prunes h exactly when sd(u,h) < d. Each landmark
// l bounds sd(u,h) from both sides: sd(u,h) <= sd(u,l) + sd(l,h), and
// sd(u,h) >= |sd(u,l) - sd(l,h)|. An upper bound below d prunes h at once
// (kPrunedBit); a lower bound of at least d proves that h survives
// (kProvenBit). Distances are uint16, 0xFFFF where undefined, and are
// clamped to 32,767 here: d is at most that, so a clamped value never prunes
// and only lowers the lower bound, and u and its candidate h are connected,
// so a landmark is undefined for both (difference 0) or for neither.
//
// G lanes take a candidate and read its row 16 bytes a lane, so a warp's load
// covers whole rows (a thread per candidate read 32 rows at 32 places), and
// a word of two distances costs a clamp and three fused add-and-min/max
// instructions (the saturating and comparing SIMD intrinsics it replaces
// expand to some forty). On grid 256x256 the filter took 36% of the light
// kernel's cycles.
constexpr uint32_t kLmkClamp = 0x7FFF7FFFu;

__device__ __forceinline__ uint32_t lmk_clamp(uint32_t x) { return __vminu2(x, kLmkClamp); }

// Bit 0: h is pruned, bit 1: h is proven (the same in all G lanes of the
// group, which act together). ua: u's row, clamped, on chip.
template <int G>
__device__ __forceinline__ uint32_t landmark_verdict(const uint32_t* ua, const uint8_t* row, int words, int d, int gl,
                                                     unsigned group) {
    uint32_t up = kLmkClamp;                   // smallest sum
    uint32_t hi = 0x80008000u, lo = kLmkClamp;  // largest and smallest sd(l,h) - sd(u,l) - 1
    for (int w = gl; w < words; w += G) {
        const uint4 b4 = __ldg((const uint4*)row + w);
        const uint4 a4 = ((const uint4*)ua)[w];
        const uint32_t bw[4] = {b4.x, b4.y, b4.z, b4.w}, aw[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t b = lmk_clamp(bw[q]);
            up = __viaddmin_u16x2(aw[q], b, up);
            hi = __viaddmax_s16x2(b, ~aw[q], hi);
            lo = __viaddmin_s16x2(b, ~aw[q], lo);
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        up = __vminu2(up, __shfl_xor_sync(group, up, o, G));
        hi = __vmaxs2(hi, __shfl_xor_sync(group, hi, o, G));
        lo = __vmins2(lo, __shfl_xor_sync(group, lo, o, G));
    }
    const int sum = min((int)(up & 0xFFFFu), (int)(up >> 16));
    const int over = max((int)(int16_t)(hi & 0xFFFFu), (int)(int16_t)(hi >> 16)) + 1;
    const int under = min((int)(int16_t)(lo & 0xFFFFu), (int)(int16_t)(lo >> 16)) + 1;
    return (sum < d ? 1u : 0u) | ((over >= d || under <= -d) ? 2u : 0u);
}

// Whether u's neighbours prove sd(u,h) >= d: every neighbour z has
// sd(z,h) >= d-1, either because it holds (h, d-1) itself or by a landmark
// with |sd(z,l) - sd(l,h)| >= d-1. Most neighbours that do not hold h lie on
// the far side of u, at distance d or d+1 from h, so their landmark bound
// may fall one or two short, where u's own had to be exact. By one warp, for
// at most 32 neighbours (false for more).
__device__ bool proven_by_neighbours(const LevelArgs& A, int64_t u, uint32_t h, int d) {
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, wl = lane & 15, need = d - 1;
    const int64_t a0 = A.rp[u];
    const int deg = (int)min(A.rp[u + 1] - a0, (int64_t)33);
    if (deg > 32) return false;
    const bool in = wl < A.lmk_words;
    uint4 b = make_uint4(0u, 0u, 0u, 0u);
    if (in) b = __ldg((const uint4*)(A.lmk + (size_t)h * A.lmk_stride) + wl);
    b = make_uint4(~lmk_clamp(b.x), ~lmk_clamp(b.y), ~lmk_clamp(b.z), ~lmk_clamp(b.w));
    const uint32_t z = lane < deg ? (uint32_t)__ldg(A.col + a0 + lane) : 0u;
    unsigned open = 0;
    for (int i = 0; i < deg; i += 2) {  // two neighbours at a time, 16 lanes each
        const uint32_t zr = __shfl_sync(FULL, z, min(i + (lane >> 4), deg - 1));
        bool far = false;
        if (in) {
            const uint4 a = __ldg((const uint4*)(A.lmk + (size_t)zr * A.lmk_stride) + wl);
            uint32_t hi = 0x80008000u, lo = kLmkClamp;  // of sd(z,l) - sd(l,h) - 1
            hi = __viaddmax_s16x2(lmk_clamp(a.x), b.x, hi);
            lo = __viaddmin_s16x2(lmk_clamp(a.x), b.x, lo);
            hi = __viaddmax_s16x2(lmk_clamp(a.y), b.y, hi);
            lo = __viaddmin_s16x2(lmk_clamp(a.y), b.y, lo);
            hi = __viaddmax_s16x2(lmk_clamp(a.z), b.z, hi);
            lo = __viaddmin_s16x2(lmk_clamp(a.z), b.z, lo);
            hi = __viaddmax_s16x2(lmk_clamp(a.w), b.w, hi);
            lo = __viaddmin_s16x2(lmk_clamp(a.w), b.w, lo);
            const int over = max((int)(int16_t)(hi & 0xFFFFu), (int)(int16_t)(hi >> 16)) + 1;
            const int under = min((int)(int16_t)(lo & 0xFFFFu), (int)(int16_t)(lo >> 16)) + 1;
            far = over >= need || under <= -need;
        }
        const unsigned m = __ballot_sync(FULL, far);
        if (!(m & 0xFFFFu)) open |= 1u << i;
        if (i + 1 < deg && !(m >> 16)) open |= 2u << i;
    }
    bool holds = true;  // (h, d-1) in L(z)
    if ((open >> lane) & 1u) {
        const uint64_t s = __ldg(A.seg + (int64_t)need * A.n + z);
        const uint32_t* hs = A.hub_arena + seg_start(s);
        const uint32_t at = seg_lower_bound(hs, seg_len(s), h);
        holds = at < seg_len(s) && (__ldg(hs + at) & kHubMask) == h;
    }
    return __all_sync(FULL, holds);
}

// The filter over list[0..M): the verdict is added to each entry, and the
// undecided positions are collected in open[0..*s_open) (any order) when
// open is given. *s_pruned, *s_proven and *s_open (zero before) receive the
// counts; the caller's barrier follows.
template <int NT, int G>
__device__ void landmark_filter(const LevelArgs& A, const uint32_t* ua, int d, uint32_t* list, const uint32_t* ckeys,
                                int M, uint32_t* open, int* s_pruned, int* s_proven, int* s_open) {
    const int tid = threadIdx.x, lane = tid & 31, gl = lane % G;
    constexpr int kPerWarp = 32 / G, kStep = NT / G;
    int pruned = 0, proven = 0;
    for (int base = tid / 32 * kPerWarp; base < M; base += kStep) {  // warp-uniform
        const int c = base + lane / G;
        uint32_t slot = 0, v = 1u;
        if (c < M) slot = list[c];
        const uint32_t h = c < M ? ckeys[slot] & kHubMask : 0u;
        v = landmark_verdict<G>(ua, A.lmk + (size_t)h * A.lmk_stride, c < M ? A.lmk_words : 0, d, gl, 0xFFFFFFFFu);
        const bool lead = gl == 0 && c < M;
        const bool is_open = lead && v == 0u;
        if (lead && v) list[c] = slot | (v & 1u ? kPrunedBit : kProvenBit);
        pruned += lead && (v & 1u);
        proven += lead && v == 2u;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, is_open);
        if (m) {
            int at = 0;
            if (lane == 0) at = atomicAdd(s_open, __popc(m));
            at = __shfl_sync(0xFFFFFFFFu, at, 0);
            if (open && is_open) open[at + __popc(m & ((1u << lane) - 1u))] = (uint32_t)c;
        }
    }
    pruned = __reduce_add_sync(0xFFFFFFFFu, pruned);
    proven = __reduce_add_sync(0xFFFFFFFFu, proven);
    if (lane == 0 && pruned) atomicAdd(s_pruned, pruned);
    if (lane == 0 && proven) atomicAdd(s_proven, proven);
}

// Records that u's segment [b0, b0 + S) waits for `scans` scans.
__device__ __forceinline__ int hold_segment(const LevelArgs& A, int64_t u, unsigned long long b0, int S, int scans) {
    const int k = atomicAdd(&A.stt->n_held, 1);  // at most one per vertex
    A.held[k] = {b0, (int32_t)u, S, scans, 0, 0};
    return k;
}

__device__ void block_bitonic_sort(unsigned long long* buf, uint32_t P) {
    for (uint32_t k = 2; k <= P; k <<= 1) {
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t i = threadIdx.x; i < P; i += blockDim.x) {
                const uint32_t ixj = i ^ j;
                if (ixj > i) {
                    const unsigned long long a = buf[i], b = buf[ixj];
                    if ((a > b) == ((i & k) == 0)) {
                        buf[i] = b;
                        buf[ixj] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------------------
// The level kernel.

// kDeep: the levels that defer their scans (kDeferLevel), in a form of its own
// so that the shallow levels' form keeps its registers.
template <int kMap, bool kOffChip, int NT, bool kDeep = false>
__global__ void __launch_bounds__(NT, level_min_blocks(NT)) k_level(const LevelArgs A) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ int s_item, s_nkeys, s_abort, s_m, s_next, s_nsurv, s_route;
    __shared__ int s_lpr, s_lpv, s_open;             // the landmark filter's counts
    __shared__ int s_held;                           // this vertex's HeldSegment
    __shared__ __align__(16) uint32_t s_lmk[kLmkMax / 2];  // u's landmark distances (uint16 pairs, clamped)
    __shared__ uint64_t s_useg[kUSideLevels];  // u's level descriptors for the rule-2 scan
    __shared__ int s_wcnt[NT / 32];
    __shared__ unsigned long long s_base;
    __shared__ long long s_wsum[NT / 32];

    const int d = A.d;
    const int64_t n = A.n;
    const size_t map_bytes = level_map_bytes(kMap, d, A.bm_words, A.cap_u_max);
    const LevelLayout L = level_layout(A.cap_c_max, map_bytes, NT);
    uint8_t* base = kOffChip ? A.gscratch + (size_t)blockIdx.x * A.gscratch_stride : smem;
    unsigned long long* ccnt = (unsigned long long*)(base + L.cnt);
    uint32_t* ckeys = (uint32_t*)(base + L.key);
    uint8_t* mapr = base + L.map;
    unsigned long long* sortbuf = (unsigned long long*)mapr;
    uint32_t* list = (uint32_t*)(base + L.list);
    uint64_t* st = (uint64_t*)(base + L.st);
    long long* pfx = (long long*)(base + L.pfx);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = NT / 32;
    const uint64_t* seg_prev = A.seg + (int64_t)(d - 1) * n;
    uint32_t cm = 0;  // largest count appended by this thread (LevelStatus::cmax)

    for (int round = 0;; ++round) {
        if (tid == 0) s_item = A.granular ? (round == 0 ? (int)blockIdx.x : A.n_items) : atomicAdd(A.work, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= A.n_items) break;
        const int64_t u = A.items[item];
        const uint32_t cbase = A.comp_base ? (uint32_t)__ldg(A.comp_base + u) : 0u;
        const int64_t raw = A.raw_u[u];
        // On chip a vertex whose candidates overflow the table is handed to
        // the off-chip pass. Off chip the table starts at A.off_start_cap
        // slots (0: the full bound) and doubles, the pull redone, whenever
        // it fills to three quarters, up to the bound 2 min(raw, u) clipped
        // to the slab (A.cap_c_max); a vertex that still overflows then goes
        // to the final off-chip pass, whose slabs hold the full bound.
        const uint32_t full_cap = cand_cap_for(raw, u, A.cap_c_max);
        uint32_t cap_c = (kOffChip && A.off_start_cap) ? min(full_cap, A.off_start_cap) : full_cap;
        // A vertex whose bound does not fit the on-chip table may overflow
        // it; an overflowing attempt reads about half its entries for
        // nothing. Once at least kRouteSamples such attempts in its size
        // class (floor(log2 pulled entries)) have been made at this level
        // and more than two thirds overflowed, it goes to the off-chip pass
        // without an attempt (the same labels either way).
        const bool may_overflow = !kOffChip && full_cap >= A.cap_c_max;
        const int rb = 63 - __clzll((unsigned long long)raw | 1ull);
        if (may_overflow) {
            if (tid == 0) {
                const unsigned a = *(volatile unsigned*)&A.stt->route_att[rb];
                const unsigned o = *(volatile unsigned*)&A.stt->route_ovf[rb];
                s_route = a >= kRouteSamples && 3ull * o > 2ull * a;
                if (s_route) {
                    const int p = atomicAdd(&A.stt->n_retry, 1);
                    A.retry_list[p] = (int32_t)u;
                    atomicMax(&A.stt->need_cap_c, (unsigned long long)cand_cap_for(raw, u, 1u << 30));
                    atomicMax(&A.stt->need_cap_u, (unsigned long long)label_cap_for(A.lab_size[u]));
                }
            }
            __syncthreads();
            if (s_route) {
                __syncthreads();  // s_route and s_item are rewritten by the next item
                continue;
            }
        }

        BitMap bm;
        HashMap hm;
        SegMap sm;
        sm.seg = A.seg;
        sm.hub_arena = A.hub_arena;
        sm.n = n;
        sm.u = u;
        sm.d = d;
        sm.cache = nullptr;
        sm.cwords = 0;
        sm.base = cbase;
        if (kMap == kMapSeg) {
        } else if (kMap == kMapBitmap) {
            bm.bits = (uint32_t*)mapr;
            bm.words = A.bm_words;
            bm.base = cbase;
            bm.d = d;
        } else {
            hm.cap = label_cap_for(A.lab_size[u]);
            hm.keys = (uint32_t*)mapr;
            hm.lvl = (uint16_t*)(mapr + (size_t)hm.cap * 4);
        }

        for (uint32_t i = tid; i < cap_c; i += NT) {
            ckeys[i] = kEmpty;
            ccnt[i] = 0ull;
        }
        uint32_t limit = kOffChip ? cap_c - cap_c / 4 : (cap_c < A.cap_c_max ? cap_c : cap_c - NT - 64);
        if (kMap == kMapBitmap) bm.clear();
        else if (kMap == kMapHash) hm.clear();
        if (tid == 0) {
            s_nkeys = 0;
            s_abort = 0;
            s_m = 0;
            s_next = 0;
            s_nsurv = 0;
            s_lpr = 0;
            s_lpv = 0;
            s_open = 0;
        }
        if (A.lmk && tid < A.lmk_stride / 4)
            s_lmk[tid] = lmk_clamp(__ldg((const uint32_t*)(A.lmk + u * A.lmk_stride) + tid));
        __syncthreads();

        // 1. label map of L_<d(u)
        const uint32_t* ball = ball_of(A, u);  // with a ball the maps are not needed
        for (int l = 0; l < d && kMap != kMapSeg && !ball; ++l) {
            const uint64_t s = __ldg(A.seg + (int64_t)l * n + u);
            const uint32_t len = seg_len(s);
            const uint32_t* hs = A.hub_arena + seg_start(s);
            for (uint32_t i = tid; i < len; i += NT) {
                const uint32_t x = __ldg(hs + i) & kHubMask;
                if (kMap == kMapBitmap) bm.insert(x, l); else hm.insert(x, l);
            }
        }
        __syncthreads();

        // 1b. segment-search map: cache the levels of u on chip over the
        // first ids that the table region can hold (the region is free
        // until the prune step is done). Each thread walks hub-sorted
        // segments, so it stops at the first hub beyond the window.
        if (kMap == kMapSeg && d > 1 && !ball) {
            uint32_t cw = (uint32_t)((L.list - L.map) / 4) / (uint32_t)(d - 1);
            cw = cw < kSegCacheMaxWords ? cw : kSegCacheMaxWords;
            if (cw >= kSegCacheMinWords) {
                uint32_t* cache = (uint32_t*)mapr;
                for (uint32_t i = tid; i < (uint32_t)(d - 1) * cw; i += NT) cache[i] = 0u;
                __syncthreads();
                for (int l = 1; l < d; ++l) {
                    const uint64_t s = __ldg(A.seg + (int64_t)l * n + u);
                    const uint32_t len = seg_len(s);
                    const uint32_t* hs = A.hub_arena + seg_start(s);
                    for (uint32_t i = tid; i < len; i += NT) {
                        const uint32_t r = (__ldg(hs + i) & kHubMask) - cbase;
                        if (r >= 32u * cw) break;
                        atomicOr(&cache[(uint32_t)(l - 1) * cw + (r >> 5)], 1u << (r & 31));
                    }
                }
                __syncthreads();
                sm.cache = cache;
                sm.cwords = cw;
            }
        }

        // 2. pull with the membership filter, merged per hub. In the push
        // paradigm the entries sent to u lie in one bucket, read as a
        // single segment.
        for (;;) {
            const bool push = A.push_hub != nullptr;
            const uint32_t* ghub = push ? A.push_hub : A.hub_arena;
            const unsigned long long* gcnt =
                push ? (const unsigned long long*)A.push_cnt : (const unsigned long long*)A.cnt_arena;
            const int64_t a0 = push ? 0 : A.rp[u], a1 = push ? 1 : A.rp[u + 1];
            for (int64_t ca = a0; ca < a1; ca += NT) {
                const int nc = (int)((a1 - ca) < NT ? (a1 - ca) : NT);
                if (tid < nc) {
                    if (push) {
                        const int64_t b0 = __ldg(A.push_off + A.rp[u]);
                        pfx[tid] = __ldg(A.push_off + A.rp[u + 1]) - b0;
                        st[tid] = (uint64_t)b0;
                    } else {
                        const uint32_t c = __ldg(A.cnt_arc + ca + tid);
                        pfx[tid] = c;
                        st[tid] = c ? seg_start(__ldg(seg_prev + __ldg(A.col + ca + tid))) +
                                          (A.arc_lo ? __ldg(A.arc_lo + ca + tid) : 0u)
                                    : 0ull;
                    }
                }
                __syncthreads();
                const long long total = block_excl_scan(pfx, nc, s_wsum);
                for (long long cb = (long long)warp * 32 * kGatherUnroll; cb < total;
                     cb += (long long)kWarps * 32 * kGatherUnroll) {
                    if (__shfl_sync(0xFFFFFFFFu, *(volatile int*)&s_abort, 0)) break;
                    int lo = 0, hi = nc;  // last arc whose first entry is <= cb
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (pfx[mid] <= cb) lo = mid; else hi = mid;
                    }
                    int j = lo;
                    uint32_t hw[kGatherUnroll];
                    uint64_t pos[kGatherUnroll];
                    bool ok[kGatherUnroll];
    #pragma unroll
                    for (int t = 0; t < kGatherUnroll; ++t) {
                        const long long i = cb + t * 32 + lane;
                        ok[t] = i < total;
                        if (ok[t]) {
                            while (pfx[j + 1] <= i) ++j;
                            pos[t] = st[j] + (uint64_t)(i - pfx[j]);
                            hw[t] = __ldg(ghub + pos[t]);
                        }
                    }
    #pragma unroll
                    for (int t = 0; t < kGatherUnroll; ++t)
                        if (ok[t]) {
                            const uint32_t h = hw[t] & kHubMask;
                            ok[t] = !(ball ? in_ball(ball, h - cbase)
                                      : kMap == kMapBitmap ? bm.member(h) : kMap == kMapHash ? hm.member(h) : sm.member(h));
                        }
                    uint64_t cv[kGatherUnroll];
    #pragma unroll
                    for (int t = 0; t < kGatherUnroll; ++t)
                        if (ok[t]) cv[t] = __ldg(gcnt + pos[t]);
    #pragma unroll
                    for (int t = 0; t < kGatherUnroll; ++t)
                        if (ok[t]) cand_insert(ckeys, ccnt, cap_c, limit, hw[t] & kHubMask, cv[t], hw[t] >> 31, &s_nkeys,
                                               &s_abort);
                }
                __syncthreads();
                if (s_abort) break;
            }
            __syncthreads();
            if (!kOffChip || !s_abort || cap_c >= full_cap) break;
            // off chip: a larger table, and the pull again
            cap_c = min(2 * cap_c, full_cap);
            limit = cap_c - cap_c / 4;
            for (uint32_t i = tid; i < cap_c; i += NT) {
                ckeys[i] = kEmpty;
                ccnt[i] = 0ull;
            }
            __syncthreads();
            if (tid == 0) {
                s_nkeys = 0;
                s_abort = 0;
            }
            __syncthreads();
        }
        __syncthreads();
        if (s_abort) {
            if (tid == 0) {
                if (kOffChip) {
                    A.giant_list[atomicAdd(&A.stt->n_giant, 1)] = (int32_t)u;
                } else {
                    if (may_overflow) {
                        atomicAdd(&A.stt->route_att[rb], 1u);
                        atomicAdd(&A.stt->route_ovf[rb], 1u);
                    }
                    const int p = atomicAdd(&A.stt->n_retry, 1);
                    A.retry_list[p] = (int32_t)u;
                    atomicMax(&A.stt->need_cap_c, (unsigned long long)cand_cap_for(raw, u, 1u << 30));
                    atomicMax(&A.stt->need_cap_u, (unsigned long long)label_cap_for(A.lab_size[u]));
                }
            }
            __syncthreads();
            continue;
        }

        // candidate list
        for (uint32_t slot = tid; slot < cap_c; slot += NT)
            if (ckeys[slot] != kEmpty) list[atomicAdd(&s_m, 1)] = slot;
        __syncthreads();
        const int M = s_m;

        // 3a. d = 3: rule 2 asks for a common neighbour x of u and h ranked
        // above h (x in L_1(u) and x in L_1(h)). Walk, for every x in L_1(u),
        // the range (x, u) of x's sorted row; a hub met there that is a
        // candidate (bitmap cand_bm) is marked pruned (bitmap mk). This replaces
        // scanning L_1(h) for every candidate h.
        bool marked = ball != nullptr;  // the ball left survivors only
        const uint32_t Wm = (uint32_t)((u - cbase + 31) >> 5);
        if (d == 3 && !marked && (size_t)Wm * 8 <= (size_t)(L.list - L.map) && M > 0) {
            uint32_t* cand_bm = (uint32_t*)mapr;
            uint32_t* mk = cand_bm + Wm;
            for (uint32_t i = tid; i < 2 * Wm; i += NT) cand_bm[i] = 0u;
            __syncthreads();
            for (int c = tid; c < M; c += NT) {
                const uint32_t h = (ckeys[list[c]] & kHubMask) - cbase;
                atomicOr(&cand_bm[h >> 5], 1u << (h & 31));
            }
            const uint64_t s1 = __ldg(A.seg + n + u);
            const uint32_t len1 = seg_len(s1);
            const uint32_t* xs = A.hub_arena + seg_start(s1);
            __syncthreads();
            for (uint32_t c0 = 0; c0 < len1; c0 += NT) {
                const int nc = (int)(len1 - c0 < (uint32_t)NT ? len1 - c0 : (uint32_t)NT);
                if (tid < nc) {
                    const uint32_t x = __ldg(xs + c0 + tid) & kHubMask;
                    // below u's dense prefix every id is in L_<3(u), so no
                    // candidate: start the walk at the prefix when it is past x
                    const uint32_t from = A.hpre && (uint32_t)__ldg(A.hpre + u) > x + 1 ? (uint32_t)__ldg(A.hpre + u) - 1 : x;
                    const int64_t r1 = A.rp[x + 1];
                    int64_t lo = A.rp[x], hi = r1;
                    while (lo < hi) {  // first neighbour of x ranked below both x and the prefix
                        const int64_t mid = (lo + hi) >> 1;
                        if ((uint32_t)__ldg(A.col + mid) <= from) lo = mid + 1; else hi = mid;
                    }
                    const int64_t first = lo;
                    hi = r1;
                    while (lo < hi) {  // first neighbour of x not ranked above u
                        const int64_t mid = (lo + hi) >> 1;
                        if ((int64_t)__ldg(A.col + mid) < u) lo = mid + 1; else hi = mid;
                    }
                    pfx[tid] = lo - first;
                    st[tid] = (uint64_t)first;
                }
                __syncthreads();
                const long long total = block_excl_scan(pfx, nc, s_wsum);
                for (long long cb = (long long)warp * 32 * kGatherUnroll; cb < total;
                     cb += (long long)kWarps * 32 * kGatherUnroll) {
                    int lo = 0, hi = nc;
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (pfx[mid] <= cb) lo = mid; else hi = mid;
                    }
                    int j = lo;
                    int32_t hv[kGatherUnroll];
#pragma unroll
                    for (int t = 0; t < kGatherUnroll; ++t) {
                        const long long i = cb + t * 32 + lane;
                        hv[t] = -1;
                        if (i < total) {
                            while (pfx[j + 1] <= i) ++j;
                            hv[t] = __ldg(A.col + st[j] + (uint64_t)(i - pfx[j]));
                        }
                    }
#pragma unroll
                    for (int t = 0; t < kGatherUnroll; ++t)
                        if (hv[t] >= 0) {
                            const uint32_t hr = (uint32_t)hv[t] - cbase;
                            const uint32_t bit = 1u << (hr & 31);
                            if (cand_bm[hr >> 5] & bit) atomicOr(&mk[hr >> 5], bit);
                        }
                }
                __syncthreads();
            }
            for (int c = tid; c < M; c += NT) {
                const uint32_t slot = list[c];
                const uint32_t h = (ckeys[slot] & kHubMask) - cbase;
                if ((mk[h >> 5] >> (h & 31)) & 1u) list[c] = slot | kPrunedBit;
            }
            __syncthreads();
            marked = true;
        }

        // 3. prune rule 2 over levels 1..d-2 of each candidate's label
        int ns = M;  // candidates left to scan
        if (d >= 3 && !marked && M > 0 && A.lmk) {
            if (A.lmk_words <= 4) landmark_filter<NT, 4>(A, s_lmk, d, list, ckeys, M, nullptr, &s_lpr, &s_lpv, &s_open);
            else landmark_filter<NT, 8>(A, s_lmk, d, list, ckeys, M, nullptr, &s_lpr, &s_lpv, &s_open);
            __syncthreads();
            ns = s_open;
            if (tid == 0 && s_lpr) atomicAdd(&A.stt->lmk_pruned, (unsigned long long)s_lpr);
            if (tid == 0 && s_lpv) atomicAdd(&A.stt->lmk_proven, (unsigned long long)s_lpv);
        }
        // the deep levels' undecided candidates stay in the list as survivors
        // and are scanned later, unless the queue of scans is full
        unsigned int q0 = 0;
        bool defer = false;
        if (kDeep && A.held && !marked && ns > 0) {
            if (tid == 0) s_next = (int)scan_place(atomicAdd(&A.stt->n_scan, (unsigned long long)ns), A.scan_cap);
            __syncthreads();
            q0 = (unsigned)s_next;
            defer = A.scan_cap - q0 >= (unsigned)ns;
            if (!defer)
                for (unsigned int i = q0 + tid; i < A.scan_cap && i - q0 < (unsigned)ns; i += NT) A.scans[i].held = -1;
            __syncthreads();
            if (tid == 0) s_next = 0;
            __syncthreads();
        }
        if (d >= 3 && !marked && ns > 0 && !defer) {
            // u's level descriptors, for scanning u's side when it is shorter
            // (not with bitmaps: their probes cost one on-chip read)
            const bool useg_on = kMap != kMapBitmap && d - 2 < kUSideLevels;
            if (useg_on && tid < d - 1) s_useg[tid] = __ldg(A.seg + (int64_t)tid * n + u);
            __syncthreads();
            const uint64_t* useg = useg_on ? s_useg : nullptr;
            // the segment-search map without its cache leaves the map's memory free
            uint32_t* filters = kDeep && kMap == kMapSeg && !kOffChip && !sm.cache &&
                                        L.list - L.map >= (size_t)kWarps * (kDeepFilter + kScanHits) * 4
                                    ? (uint32_t*)mapr
                                    : nullptr;
            if constexpr (kMap == kMapBitmap)
                prune_all<NT>(bm, A.seg, A.hub_arena, n, d, list, ckeys, nullptr, M, ns, &s_next, useg, s_wcnt, filters, u);
            else if constexpr (kMap == kMapHash)
                prune_all<NT>(hm, A.seg, A.hub_arena, n, d, list, ckeys, nullptr, M, ns, &s_next, useg, s_wcnt, filters, u);
            else prune_all<NT>(sm, A.seg, A.hub_arena, n, d, list, ckeys, nullptr, M, ns, &s_next, useg, s_wcnt, filters, u);
            __syncthreads();
        }
        // 4. survivors, hub-sorted, appended as L_d(u). Candidate hubs are < u:
        // when a bitmap of u bits and its word prefix fit the map region, a
        // survivor's rank is the prefix of its word plus a popcount; else a
        // bitonic sort.
        const uint32_t W = (uint32_t)((u - cbase + 31) >> 5);
        const size_t region = (L.list - L.map);
        if ((size_t)W * 8 <= region) {
            uint32_t* sb = (uint32_t*)mapr;
            uint32_t* wp = sb + W;
            for (uint32_t i = tid; i < W; i += NT) sb[i] = 0u;
            __syncthreads();
            for (int c = tid; c < M; c += NT) {
                const uint32_t slot = list[c];
                if (!(slot & kPrunedBit)) {
                    const uint32_t h = (ckeys[slot & kSlotMask] & kHubMask) - cbase;
                    atomicOr(&sb[h >> 5], 1u << (h & 31));
                }
            }
            __syncthreads();
            const int S = (int)block_excl_scan_popc(sb, wp, W, s_wsum);
            if (S > 0) {
                if (tid == 0) {
                    const unsigned long long b0 = atomicAdd(&A.stt->bump, (unsigned long long)S);
                    if (b0 + S > A.arena_cap) atomicOr(&A.stt->arena_overflow, 1);
                    s_base = b0;
                    if (defer) s_held = hold_segment(A, u, b0, S, ns);
                }
                __syncthreads();
                const unsigned long long b0 = s_base;
                if (b0 + S <= A.arena_cap) {
                    for (int c = tid; c < M; c += NT) {
                        const uint32_t e = list[c];
                        if (e & kPrunedBit) continue;
                        const uint32_t slot = e & kSlotMask;
                        const uint32_t key = ckeys[slot];
                        const uint32_t h = key & kHubMask;
                        const uint32_t hr = h - cbase;
                        const uint32_t r = wp[hr >> 5] + __popc(sb[hr >> 5] & ((1u << (hr & 31)) - 1u));
                        const uint64_t cv = ccnt[slot];
                        A.hub_arena[b0 + r] = h | (key & kOvfBit);
                        A.cnt_arena[b0 + r] = cv;
                        cm = max(cm, count_bound(cv, key & kOvfBit));
                        if (defer && !(e & kProvenBit)) A.scans[q0 + atomicAdd(&s_next, 1)] = {s_held, (int32_t)r};
                    }
                    if (tid == 0 && !defer) A.seg_out[u] = seg_pack(b0, (uint32_t)S);
                }
            }
        } else {
            for (int c = tid; c < M; c += NT) {
                const uint32_t e = list[c];
                if (!(e & kPrunedBit))
                    sortbuf[atomicAdd(&s_nsurv, 1)] =
                        ((unsigned long long)(ckeys[e & kSlotMask] & kHubMask) << 32) | (e & (kSlotMask | kProvenBit));
            }
            __syncthreads();
            const int S = s_nsurv;
            if (S > 0) {
                const uint32_t P = pow2_ceil((uint64_t)S);
                for (uint32_t i = S + tid; i < P; i += NT) sortbuf[i] = ~0ull;
                __syncthreads();
                block_bitonic_sort(sortbuf, P);
                if (tid == 0) {
                    const unsigned long long b0 = atomicAdd(&A.stt->bump, (unsigned long long)S);
                    if (b0 + S > A.arena_cap) atomicOr(&A.stt->arena_overflow, 1);
                    s_base = b0;
                    if (defer) s_held = hold_segment(A, u, b0, S, ns);
                }
                __syncthreads();
                const unsigned long long b0 = s_base;
                if (b0 + S <= A.arena_cap) {
                    for (int i = tid; i < S; i += NT) {
                        const uint32_t e = (uint32_t)sortbuf[i], slot = e & kSlotMask;
                        const uint32_t key = ckeys[slot];
                        const uint64_t cv = ccnt[slot];
                        A.hub_arena[b0 + i] = (key & kHubMask) | (key & kOvfBit);
                        A.cnt_arena[b0 + i] = cv;
                        cm = max(cm, count_bound(cv, key & kOvfBit));
                        if (defer && !(e & kProvenBit)) A.scans[q0 + atomicAdd(&s_next, 1)] = {s_held, (int32_t)i};
                    }
                    if (tid == 0 && !defer) A.seg_out[u] = seg_pack(b0, (uint32_t)S);
                }
            }
        }
        if (tid == 0) atomicAdd(&A.stt->unique_total, (unsigned long long)s_nkeys);
        if (tid == 0 && may_overflow) atomicAdd(&A.stt->route_att[rb], 1u);
        __syncthreads();
    }
    cm = __reduce_max_sync(0xFFFFFFFFu, cm);
    if (lane == 0 && cm) atomicMax(&A.stt->cmax, cm);
}

#include "pspc_dense.cuh"

// ---------------------------------------------------------------------------
// The level for small vertices (fewer than 32 R pulled entries): one warp
// per vertex and no CTA barrier, so that many such vertices (the deep levels
// of high-diameter graphs, the tails of power-law graphs) are in flight per
// SM. The pulled entries are read side by side, R to a lane; those whose hub
// is already in L_<d(u) are dropped (a search in u's segments of levels d-1
// and d-2, copied on chip) before their counts are read, and the rest
// compacted on chip, sorted by hub (bitonic, in registers) and the counts of
// equal hubs summed with a segmented scan (mod 2^64; the flag takes the
// entries' flags and every carry: Label Merging). A hub comes at most once
// per arc, so the scan takes log2(deg u) steps. Rule 2 then runs per
// candidate: the landmark filter, and for the undecided ones a label scan
// by the whole warp. Survivors are already in hub order and are appended as
// L_d(u).
constexpr int kMicroWarps = kMicroThreads / 32;
constexpr int kMicroOwn = 128;  // entries of u's levels d-1 and d-2 kept on chip

__device__ __forceinline__ void add_count(uint64_t& sum, uint32_t& flag, uint64_t c, uint32_t f) {
    const uint64_t s = sum + c;
    flag |= f | (uint32_t)(s < c);
    sum = s;
}

// One warp's memory: the landmark row and the scan's filter are needed after
// the staged entries and the copy of u's segments.
template <int R>
struct MicroMem {
    unsigned long long cnt[32 * R];
    uint32_t hub[32 * R];
    union {
        uint32_t own[kMicroOwn];
        struct {
            uint32_t lmk[kLmkMax / 2];
            uint32_t filter[kMicroFilter + kScanHits];
        } f;
    } u;
};

// Steps 2 to 5 for the T (at most 32 R) entries in m.hub and m.cnt.
template <int R, class Mem>
__device__ void micro_merge(const LevelArgs& A, Mem& m, int T, int64_t u, int64_t deg, unsigned long long& n_uniq,
                            unsigned long long& n_lpr, unsigned long long& n_lpv, uint32_t& cm) {
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int d = A.d;
    const int64_t n = A.n;
    uint32_t* hb = m.hub;

    // 2. sort keys: hub << 7 | entry, 0xFFFFFFFF for absent entries (last)
    uint32_t key[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const int e = lane + 32 * j;
        key[j] = e < T ? ((hb[e] & kHubMask) << 7) | (uint32_t)e : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int k = 2; k <= 32 * R; k <<= 1) {
#pragma unroll
        for (int jj = k >> 1; jj > 0; jj >>= 1) {
            if (jj >= 32) {  // partners in the same lane
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    const int q = j ^ (jj / 32);
                    if (q < j) continue;
                    const bool asc = ((32 * j) & k) == 0;
                    const uint32_t lo = min(key[j], key[q]), hi = max(key[j], key[q]);
                    key[j] = asc ? lo : hi;
                    key[q] = asc ? hi : lo;
                }
            } else {
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    const int e = lane + 32 * j;
                    const uint32_t other = __shfl_xor_sync(FULL, key[j], jj);
                    const bool lower = (e & jj) == 0, asc = (e & k) == 0;
                    key[j] = (lower == asc) ? min(key[j], other) : max(key[j], other);
                }
            }
        }
    }

    // 3. segmented sums over runs of equal hubs, in sorted order
    uint32_t hub[R], flg[R];
    uint64_t sum[R];
    unsigned heads[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const bool valid = key[j] != 0xFFFFFFFFu;
        const int src = (int)(key[j] & 127u);
        hub[j] = valid ? key[j] >> 7 : 0xFFFFFFFFu;
        sum[j] = valid ? (uint64_t)m.cnt[src] : 0ull;
        flg[j] = valid ? hb[src] >> 31 : 0u;
        // a run starts where the previous element (in sorted order) has
        // another hub; row j's lane 0 follows row j-1's lane 31
        const uint32_t prev = __shfl_up_sync(FULL, hub[j], 1);
        const uint32_t last = j > 0 ? __shfl_sync(FULL, hub[j > 0 ? j - 1 : 0], 31) : 0xFFFFFFFFu;
        heads[j] = __ballot_sync(FULL, valid && (lane == 0 ? (j == 0 || last != hub[j]) : prev != hub[j]));
    }
    int uniq = 0;
    uint64_t carry = 0;
    uint32_t carry_flag = 0;
    bool cand[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
        uniq += __popc(heads[j]);
        // lanes before this one in its run (in this row)
        const unsigned mine = heads[j] & (lt | (1u << lane));
        const int back = mine ? lane - (31 - __clz(mine)) : lane;
        for (int o = 1; o < 32 && o < deg; o <<= 1) {
            const uint64_t sv = __shfl_up_sync(FULL, sum[j], o);
            const uint32_t fv = __shfl_up_sync(FULL, flg[j], o);
            if (back >= o) add_count(sum[j], flg[j], sv, fv);
        }
        if (!mine && hub[j] != 0xFFFFFFFFu) add_count(sum[j], flg[j], carry, carry_flag);  // the row before's last run
        carry = __shfl_sync(FULL, sum[j], 31);
        carry_flag = __shfl_sync(FULL, flg[j], 31);
        // the last element of each run holds its total
        const uint32_t next = __shfl_down_sync(FULL, hub[j], 1);
        const uint32_t first = j + 1 < R ? __shfl_sync(FULL, hub[j + 1 < R ? j + 1 : j], 0) : 0xFFFFFFFFu;
        cand[j] = hub[j] != 0xFFFFFFFFu && (lane == 31 ? first != hub[j] : next != hub[j]);
    }
    n_uniq += (unsigned long long)uniq;

    // 4. rule 2: the landmark filter, then the undecided candidates' scans
    bool surv[R];
#pragma unroll
    for (int j = 0; j < R; ++j) surv[j] = cand[j];
    unsigned und[R];  // undecided candidates
    int n_open = 0;
    unsigned int q0 = 0;  // their places in the queue of deferred scans
    bool defer = false;
    if (d >= 3 && uniq > 0 && !A.ball) {
        if (A.lmk) {
            __syncwarp();
            for (int i = lane; i < A.lmk_stride / 4; i += 32)
                m.u.f.lmk[i] = lmk_clamp(__ldg((const uint32_t*)(A.lmk + u * A.lmk_stride) + i));
            // the candidates' hubs in order (the staged entries are done
            // with), eight lanes to each, then the verdicts back
            int at[R], before = 0;
            uint32_t* verdict = (uint32_t*)m.cnt;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const unsigned c = __ballot_sync(FULL, cand[j]);
                at[j] = before + __popc(c & lt);
                before += __popc(c);
                if (cand[j]) hb[at[j]] = hub[j];
            }
            __syncwarp();
            for (int base = 0; base < uniq; base += 4) {
                const int c = base + lane / 8;
                const uint32_t v = landmark_verdict<8>(m.u.f.lmk, A.lmk + (size_t)(c < uniq ? hb[c] : 0u) * A.lmk_stride,
                                                       c < uniq ? A.lmk_words : 0, d, lane % 8, FULL);
                if (c < uniq && lane % 8 == 0) verdict[c] = v;
            }
            __syncwarp();
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const uint32_t v = cand[j] ? verdict[at[j]] : 1u;
                und[j] = __ballot_sync(FULL, v == 0u);
                if (cand[j] && (v & 1u)) {
                    surv[j] = false;
                    ++n_lpr;
                } else if (cand[j] && (v & 2u)) {
                    ++n_lpv;
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < R; ++j) und[j] = __ballot_sync(FULL, cand[j]);
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < R; ++j) n_open += __popc(und[j]);
        if (A.held && A.lmk && n_open > 0) {
            if (lane == 0) q0 = scan_place(atomicAdd(&A.stt->n_scan, (unsigned long long)n_open), A.scan_cap);
            q0 = __shfl_sync(FULL, q0, 0);
            defer = A.scan_cap - q0 >= (unsigned)n_open;
            if (!defer)
                for (unsigned int i = q0 + lane; i < A.scan_cap && i - q0 < (unsigned)n_open; i += 32)
                    A.scans[i].held = -1;
        }
#pragma unroll
        for (int j = 0; j < R; ++j)
            for (unsigned left = defer ? 0u : und[j]; left; left &= left - 1) {
                const int src = __ffs(left) - 1;
                const uint32_t h = __shfl_sync(FULL, hub[j], src);
                if (A.lmk && d >= kNeighbourLevel && proven_by_neighbours(A, u, h, d)) continue;
                const bool pruned = scan_filtered(m.u.f.filter, kMicroFilter, A.seg, A.hub_arena, n, u, d, h, 1, d - 2, nullptr);
                if (pruned && lane == src) surv[j] = false;
            }
    }

    // 5. append the survivors in hub order
    unsigned sv[R];
    int S = 0;
#pragma unroll
    for (int j = 0; j < R; ++j) {
        sv[j] = __ballot_sync(FULL, surv[j]);
        S += __popc(sv[j]);
    }
    if (S > 0) {
        unsigned long long b0 = 0;
        if (lane == 0) {
            b0 = atomicAdd(&A.stt->bump, (unsigned long long)S);
            if (b0 + S > A.arena_cap) atomicOr(&A.stt->arena_overflow, 1);
        }
        b0 = __shfl_sync(FULL, b0, 0);
        if (b0 + S <= A.arena_cap) {
            int before = 0, held = 0;
            if (defer) {
                if (lane == 0) held = hold_segment(A, u, b0, S, n_open);
                held = __shfl_sync(FULL, held, 0);
            }
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (surv[j]) {
                    const int r = before + __popc(sv[j] & lt);
                    A.hub_arena[b0 + r] = hub[j] | (flg[j] ? kOvfBit : 0u);
                    A.cnt_arena[b0 + r] = sum[j];
                    cm = max(cm, count_bound(sum[j], flg[j]));
                    if (defer && ((und[j] >> lane) & 1u)) A.scans[q0 + __popc(und[j] & lt)] = {held, r};
                }
                if (defer) q0 += __popc(und[j]);
                before += __popc(sv[j]);
            }
            if (lane == 0 && !defer) A.seg_out[u] = seg_pack(b0, (uint32_t)S);
        }
    }
    __syncwarp();
}

template <int R>
__global__ void __launch_bounds__(kMicroThreads) k_level_micro(const LevelArgs A) {
    __shared__ __align__(16) MicroMem<R> s_mem[kMicroWarps];
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int d = A.d;
    const int64_t n = A.n;
    const uint64_t* seg_prev = A.seg + (int64_t)(d - 1) * n;
    MicroMem<R>& m = s_mem[w];
    const unsigned lt = (1u << lane) - 1u;
    unsigned long long n_uniq = 0, n_lpr = 0, n_lpv = 0;
    uint32_t cm = 0;  // largest count appended by this lane (LevelStatus::cmax)
    const bool push = A.push_hub != nullptr;
    const uint32_t* ghub = push ? A.push_hub : A.hub_arena;
    const unsigned long long* gcnt =
        push ? (const unsigned long long*)A.push_cnt : (const unsigned long long*)A.cnt_arena;
    for (int round = 0;; ++round) {
        int item;
        if (A.granular) {
            item = round == 0 ? (int)(blockIdx.x * kMicroWarps + w) : A.n_items;
        } else {
            item = 0;
            if (lane == 0) item = atomicAdd(A.work, 1);
            item = __shfl_sync(FULL, item, 0);
        }
        if (item >= A.n_items) break;
        const int64_t u = A.items[item];
        const int64_t a0 = A.rp[u], a1 = A.rp[u + 1];

        // 1. u's segments of levels d-1 and d-2, the only ones that can
        // hold a pulled hub (level 0 is u itself, never pulled)
        const uint64_t own1 = __ldg(seg_prev + u);
        const uint64_t own2 = d > 2 ? __ldg(A.seg + (int64_t)(d - 2) * n + u) : 0ull;
        const uint32_t n1 = seg_len(own1), n2 = seg_len(own2);
        const uint32_t* ball = ball_of(A, u);  // answers for the segments, and for rule 2
        const uint32_t cbase = ball && A.comp_base ? (uint32_t)__ldg(A.comp_base + u) : 0u;
        const bool staged = !ball && n1 + n2 <= (uint32_t)kMicroOwn;
        if (staged)
            for (uint32_t i = lane; i < n1 + n2; i += 32)
                m.u.own[i] = __ldg(A.hub_arena + (i < n1 ? seg_start(own1) : seg_start(own2) - n1) + i) & kHubMask;
        __syncwarp();
        auto find = [&](const uint32_t* xs, uint32_t len, uint32_t x) {  // in the on-chip copy
            uint32_t lo = 0, hi = len;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (xs[mid] < x) lo = mid + 1; else hi = mid;
            }
            return lo < len && xs[lo] == x;
        };
        auto member = [&](uint32_t x) {
            if (ball) return in_ball(ball, x - cbase);
            if (staged) return find(m.u.own, n1, x) || find(m.u.own + n1, n2, x);
            const uint32_t* h1 = A.hub_arena + seg_start(own1);
            const uint32_t* h2 = A.hub_arena + seg_start(own2);
            return seg_contains(h1, n1, x) || seg_contains(h2, n2, x);
        };

        // the pulled entries (fewer than 32 R), 32 arcs at a time
        int T = 0;
        const int64_t arcs_end = push ? a0 + 1 : a1;
        for (int64_t ca = a0; ca < arcs_end; ca += 32) {
            const int64_t a = ca + lane;
            uint32_t c = 0;
            uint64_t st = 0;
            if (push) {  // the entries sent to u lie in one bucket
                if (lane == 0) {
                    st = (uint64_t)__ldg(A.push_off + a0);
                    c = (uint32_t)(__ldg(A.push_off + a1) - (int64_t)st);
                }
            } else if (a < a1) {
                c = __ldg(A.cnt_arc + a);
                if (c) st = seg_start(__ldg(seg_prev + __ldg(A.col + a))) + (A.arc_lo ? __ldg(A.arc_lo + a) : 0u);
            }
            uint32_t incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += t;
            }
            const uint32_t excl = incl - c, total = __shfl_sync(FULL, incl, 31);
            st -= excl;
            uint32_t hw[R];
            uint64_t pos[R];
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const uint32_t i = t * 32 + lane;
                hw[t] = kEmpty;
                if (t * 32 < total) {  // warp-uniform
                    int j = 0;
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1) {
                        const uint32_t e = __shfl_sync(FULL, excl, j + step);
                        if (e <= i) j += step;
                    }
                    pos[t] = __shfl_sync(FULL, st, j) + i;
                    if (i < total) hw[t] = __ldg(ghub + pos[t]);
                }
            }
#pragma unroll
            for (int t = 0; t < R; ++t)
                if (t * 32 < total) {
                    const bool keep = t * 32 + lane < total && !member(hw[t] & kHubMask);
                    const unsigned b = __ballot_sync(FULL, keep);
                    const int at = T + __popc(b & lt);
                    if (keep) {
                        m.hub[at] = hw[t];
                        m.cnt[at] = __ldg(gcnt + pos[t]);
                    }
                    T += __popc(b);
                }
        }
        __syncwarp();
        if (T == 0) continue;
        const int64_t deg = push ? (int64_t)32 : a1 - a0;
        if (T <= 32) micro_merge<1>(A, m, T, u, deg, n_uniq, n_lpr, n_lpv, cm);
        else if (R == 2 || T <= 64) micro_merge<2>(A, m, T, u, deg, n_uniq, n_lpr, n_lpv, cm);
        else micro_merge<R>(A, m, T, u, deg, n_uniq, n_lpr, n_lpv, cm);
    }
    cm = __reduce_max_sync(FULL, cm);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {  // the verdicts were counted by the candidates' lanes
        n_lpr += __shfl_xor_sync(FULL, n_lpr, o);
        n_lpv += __shfl_xor_sync(FULL, n_lpv, o);
    }
    if (lane == 0) {
        if (cm) atomicMax(&A.stt->cmax, cm);
        if (n_uniq) atomicAdd(&A.stt->unique_total, n_uniq);
        if (n_lpr) atomicAdd(&A.stt->lmk_pruned, n_lpr);
        if (n_lpv) atomicAdd(&A.stt->lmk_proven, n_lpv);
    }
}

// ---------------------------------------------------------------------------
// The deferred scans, spread over all SMs instead of holding the one warp or
// CTA that met them (a road network's deep levels have vertices with dozens
// of undecided candidates). k_prove_deferred first tries the neighbours'
// proof, which decides half of them at level 100 of grid 256x256 and three
// quarters from level 277 on; k_scan_deferred scans the rest, split into
// ranges of levels when there are fewer of them than warps. A pruned entry
// is marked in the arena; the warp that ends a vertex's last part takes the
// marked entries out and publishes the segment. Nothing waits: the segments
// were appended by earlier launches. With the scans in place grid 256x256
// took 723 ms in the level kernels (1,086 with a warp per vertex at every
// level), of which less than 100 were not scans.
constexpr int kScanThreads = 256;

__global__ void __launch_bounds__(kScanThreads) k_prove_deferred(const LevelArgs A) {
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    if (A.stt->arena_overflow) return;  // the level runs again with a larger arena
    const int count = (int)scan_place(A.stt->n_scan, A.scan_cap);
    const int warps = (int)(gridDim.x * (kScanThreads / 32));
    for (int item = (int)(blockIdx.x * (kScanThreads / 32) + (threadIdx.x >> 5)); item < count; item += warps) {
        const DeferredScan q = A.scans[item];
        if (q.held < 0) continue;
        HeldSegment* H = A.held + q.held;
        const uint32_t h = __ldg(A.hub_arena + H->start + q.pos) & kHubMask;
        const bool proven = proven_by_neighbours(A, H->u, h, A.d);
        if (lane == 0) {
            if (!proven) A.scans[A.scan_cap + atomicAdd(&A.stt->n_scan_open, 1u)] = q;
            else if (atomicSub(&H->scans, 1) == 1) A.seg_out[H->u] = seg_pack(H->start, (uint32_t)H->len);
        }
        __syncwarp(FULL);
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_deferred(const LevelArgs A) {
    __shared__ __align__(16) uint32_t s_filter[kScanThreads / 32][kScanFilter + kScanHits];
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    if (A.stt->arena_overflow) return;
    const int count = (int)A.stt->n_scan_open, levels = A.d - 2;
    const int parts = max(1, min((int)(gridDim.x * (kScanThreads / 32)) / max(count, 1), (levels + 30) / 31));
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(&A.stt->work_scan, 1);
        item = __shfl_sync(FULL, item, 0);
        if (item >= count * parts) break;
        const DeferredScan q = A.scans[A.scan_cap + item / parts];
        const int part = item % parts;
        const int klo = 1 + (int)((int64_t)levels * part / parts), khi = (int)((int64_t)levels * (part + 1) / parts);
        HeldSegment* H = A.held + q.held;
        const int64_t u = H->u;
        const unsigned long long b0 = H->start;
        const int S = H->len;
        const uint32_t h = __ldcg(A.hub_arena + b0 + q.pos) & kHubMask;
        const bool pruned = scan_filtered(s_filter[w], kScanFilter, A.seg, A.hub_arena, A.n, u, A.d, h, klo, khi, nullptr);
        int last = 0;
        if (lane == 0) {
            if (pruned) {
                atomicOr(A.hub_arena + b0 + q.pos, kMarkBit);
                atomicExch(&H->pruned, 1);
            }
            __threadfence();
            last = atomicAdd(&H->done, 1) + 1 == H->scans * parts;
            __threadfence();
        }
        if (!__shfl_sync(FULL, last, 0)) continue;
        int kept = S;
        if (__ldcg(&H->pruned)) {  // stable compaction in place: a row is read before earlier places are written
            kept = 0;
            for (int r = 0; r < S; r += 32) {
                const bool in = r + lane < S;
                const uint32_t hw = in ? __ldcg(A.hub_arena + b0 + r + lane) : kMarkBit;
                const uint64_t c = in ? __ldcg((const unsigned long long*)A.cnt_arena + b0 + r + lane) : 0ull;
                const bool keep = in && !(hw & kMarkBit);
                const unsigned m = __ballot_sync(FULL, keep);
                if (keep) {
                    A.hub_arena[b0 + kept + __popc(m & lt)] = hw;
                    A.cnt_arena[b0 + kept + __popc(m & lt)] = c;
                }
                kept += __popc(m);
                __syncwarp();
            }
            if (lane == 0) atomicAdd(&A.stt->dropped, (unsigned long long)(S - kept));
        }
        if (lane == 0) A.seg_out[u] = kept ? seg_pack(b0, (uint32_t)kept) : 0ull;
    }
}

// ---------------------------------------------------------------------------
// Push paradigm.

__global__ void k_arc_counts(int64_t arcs, const uint32_t* __restrict__ cnt_arc, int64_t* __restrict__ out) {
    const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (a < arcs) out[a] = cnt_arc[a];
}

// Warp per arc u->v: the entries of L_{d-1}(v) that u receives go to u's
// bucket in the order they lie in v's segment.
__global__ void k_push_scatter(int64_t arcs, const int32_t* __restrict__ col, const uint64_t* __restrict__ seg_prev,
                               const uint32_t* __restrict__ hub_arena, const uint64_t* __restrict__ cnt_arena,
                               const uint32_t* __restrict__ cnt_arc, const uint32_t* __restrict__ arc_lo,
                               const int64_t* __restrict__ push_off, uint32_t* __restrict__ push_hub,
                               uint64_t* __restrict__ push_cnt) {
    const int64_t a = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (a >= arcs) return;
    const uint32_t c = cnt_arc[a];
    if (!c) return;
    const uint64_t src = seg_start(__ldg(seg_prev + col[a])) + (arc_lo ? arc_lo[a] : 0u);
    const int64_t dst = push_off[a];
    for (uint32_t i = lane; i < c; i += 32) {
        push_hub[dst + i] = __ldg(hub_arena + src + i);
        push_cnt[dst + i] = __ldg((const unsigned long long*)cnt_arena + src + i);
    }
}

cudaError_t launch_arc_counts(int64_t arcs, const uint32_t* cnt_arc, int64_t* out, cudaStream_t st) {
    if (arcs > 0) k_arc_counts<<<(unsigned)((arcs + 255) / 256), 256, 0, st>>>(arcs, cnt_arc, out);
    return cudaGetLastError();
}

cudaError_t launch_push_scatter(int64_t arcs, const int32_t* col, const uint64_t* seg_prev,
                                const uint32_t* hub_arena, const uint64_t* cnt_arena, const uint32_t* cnt_arc,
                                const uint32_t* arc_lo, const int64_t* push_off, uint32_t* push_hub,
                                uint64_t* push_cnt, cudaStream_t st) {
    if (arcs > 0)
        k_push_scatter<<<(unsigned)((arcs * 32 + 255) / 256), 256, 0, st>>>(arcs, col, seg_prev, hub_arena, cnt_arena,
                                                                          cnt_arc, arc_lo, push_off, push_hub,
                                                                          push_cnt);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Launchers.

cudaError_t launch_arc_src(const int64_t* rp, int64_t n, int32_t* arc_src, cudaStream_t st) {
    k_arc_src<<<(unsigned)((n * 32 + 255) / 256), 256, 0, st>>>(rp, n, arc_src);
    return cudaGetLastError();
}

cudaError_t launch_dense_prefix(int d, int64_t n, const uint64_t* seg, const uint32_t* hub_arena,
                                const int32_t* comp_base, int32_t* hpre, cudaStream_t st) {
    k_dense_prefix<<<(unsigned)((n + kPrefixWarps - 1) / kPrefixWarps), kPrefixWarps * 32, 0, st>>>(
        d, n, seg, hub_arena, comp_base, hpre);
    return cudaGetLastError();
}

cudaError_t launch_cost(int d, int64_t n, int64_t arcs, const int64_t* rp, const int32_t* col,
                        const int32_t* arc_src, const uint64_t* seg_prev, const uint32_t* hub_arena,
                        const int32_t* hpre, uint32_t* arc_lo, uint32_t* cnt_arc, int64_t* raw_u,
                        int64_t* lab_size, LevelStatus* stt, int64_t label_limit, const DenseRule& dense,
                        int32_t* glist, int32_t* items, int* max_deg, cudaStream_t st, int64_t* launches) {
    if (arcs > 0)
        k_cost_arcs<<<(unsigned)((arcs + 255) / 256), 256, 0, st>>>(arcs, arc_src, col, seg_prev, hub_arena, hpre,
                                                                     arc_lo, cnt_arc, (unsigned long long*)raw_u,
                                                                     &stt->prefix_skipped);
    k_cost_vertices<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, rp, seg_prev, raw_u, lab_size, stt, label_limit,
                                                                  dense, glist, max_deg);
    k_bucket_fill<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, rp, raw_u, lab_size, stt, label_limit, dense,
                                                                items);
    if (launches) *launches += (arcs > 0) + 2;
    return cudaGetLastError();
}

cudaError_t launch_cost_level(int64_t n, const int64_t* rp, const int32_t* col, const uint64_t* seg_prev,
                              uint64_t* seg_row, const uint32_t* hub_arena, const int32_t* hpre, uint32_t* arc_lo,
                              uint32_t* cnt_arc, int64_t* raw_u, int64_t* lab_size, LevelStatus* stt, LevelStatus* next,
                              unsigned long long bump, int64_t label_limit, const DenseRule& dense, int32_t* glist,
                              int32_t* items, cudaStream_t st) {
    k_cost_level<<<(unsigned)((n * kCostLanes + kCostThreads - 1) / kCostThreads), kCostThreads, 0, st>>>(
        n, rp, col, seg_prev, seg_row, hub_arena, hpre, arc_lo, cnt_arc, raw_u, lab_size, stt, next, bump, label_limit,
        dense, glist);
    k_bucket_fill<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, rp, raw_u, lab_size, stt, label_limit, dense, items);
    return cudaGetLastError();
}

template <int NT>
static const void* level_fn(int map_kind, bool offchip) {
    if (offchip) return map_kind == kMapSeg ? (const void*)k_level<kMapSeg, true, NT> : (const void*)k_level<kMapHash, true, NT>;
    return map_kind == kMapBitmap ? (const void*)k_level<kMapBitmap, false, NT>
           : map_kind == kMapHash ? (const void*)k_level<kMapHash, false, NT>
                                  : (const void*)k_level<kMapSeg, false, NT>;
}

// The kernel's dynamic shared-memory limit is raised to the device's
// opt-in maximum, the same value on every call: builds that run at the same
// time on other threads never see it lowered under a launch.
cudaError_t level_kernel_attrs(int map_kind, size_t smem_bytes, int* occupancy, int nt) {
    const void* f = nt == kLightThreads ? level_fn<kLightThreads>(map_kind, false) : level_fn<kLevelThreads>(map_kind, false);
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
    const size_t max_dyn = (size_t)optin - fa.sharedSizeBytes;
    if (smem_bytes > max_dyn) return cudaErrorInvalidValue;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_dyn);
    if (e == cudaSuccess && nt == kLightThreads && map_kind == kMapSeg)
        e = cudaFuncSetAttribute((const void*)k_level<kMapSeg, false, kLightThreads, true>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_dyn - 1024);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occupancy, f, nt, smem_bytes);
}

template <int NT>
static void launch_level_nt(int map_kind, bool offchip, int grid, size_t smem_bytes, const LevelArgs& A,
                            cudaStream_t st) {
    if (offchip && map_kind == kMapSeg)
        k_level<kMapSeg, true, NT><<<grid, NT, 0, st>>>(A);
    else if (offchip)
        k_level<kMapHash, true, NT><<<grid, NT, 0, st>>>(A);
    else if (map_kind == kMapBitmap)
        k_level<kMapBitmap, false, NT><<<grid, NT, smem_bytes, st>>>(A);
    else if (map_kind == kMapHash)
        k_level<kMapHash, false, NT><<<grid, NT, smem_bytes, st>>>(A);
    else
        k_level<kMapSeg, false, NT><<<grid, NT, smem_bytes, st>>>(A);
}

cudaError_t dense_kernel_attrs(int* occupancy) {
    const size_t bytes = dense_layout().total;
    cudaError_t e = cudaFuncSetAttribute((const void*)k_level_dense, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)bytes);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occupancy, (const void*)k_level_dense, kDenseThreads, bytes);
}

cudaError_t launch_level_dense(int grid, const LevelArgs& A, cudaStream_t st) {
    k_level_dense<<<grid, kDenseThreads, dense_layout().total, st>>>(A);
    return cudaGetLastError();
}

// Rows of 32 entries per warp: 2 or 4.
cudaError_t micro_kernel_occupancy(int rows, int* occupancy) {
    const void* f = rows == 2 ? (const void*)k_level_micro<2> : (const void*)k_level_micro<4>;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occupancy, f, kMicroThreads, 0);
}

cudaError_t scan_kernel_occupancy(int* prove, int* scan) {
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(prove, (const void*)k_prove_deferred, kScanThreads, 0);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(scan, (const void*)k_scan_deferred, kScanThreads, 0);
}

cudaError_t launch_scan_deferred(int prove_grid, int scan_grid, const LevelArgs& A, cudaStream_t st) {
    k_prove_deferred<<<prove_grid, kScanThreads, 0, st>>>(A);
    k_scan_deferred<<<scan_grid, kScanThreads, 0, st>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_level_micro(int rows, int grid, const LevelArgs& A, cudaStream_t st) {
    if (rows == 2) k_level_micro<2><<<grid, kMicroThreads, 0, st>>>(A);
    else k_level_micro<4><<<grid, kMicroThreads, 0, st>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_level(int map_kind, bool offchip, int grid, size_t smem_bytes, const LevelArgs& A,
                         cudaStream_t st, int nt) {
    if (nt == kLightThreads && !offchip && map_kind == kMapSeg && (A.d >= kDeferLevel || A.held))
        k_level<kMapSeg, false, kLightThreads, true><<<grid, nt, smem_bytes, st>>>(A);
    else if (nt == kLightThreads && !offchip) launch_level_nt<kLightThreads>(map_kind, false, grid, smem_bytes, A, st);
    else launch_level_nt<kLevelThreads>(map_kind, offchip, grid, smem_bytes, A, st);
    return cudaGetLastError();
}

}  // namespace pspc
