// Landmark labelling for the landmark filter of pruning rule 2 (Section
// "Landmark-Based Filtering"). The first landmarks of a graph (up to
// kLmkShallow) are its highest-ranked vertices; under a degree order these
// are the vertices whose degree reaches the k-th largest degree, the
// paper's degree threshold. The filter needs sd(v, l) for every vertex v and
// landmark l: the searches of a round run together, one BFS level per
// launch. Every vertex keeps a 64-bit mask of the round's landmarks that
// have reached it; at level t it takes the OR of its neighbours' frontier
// masks, and the bits new to it get distance t. In deep graphs, where the
// launches of such levels are what the searches cost, one block searches
// from each landmark by itself (k_lmk_search).
//
// The remaining landmarks of a single graph (k > kLmkShallow; the filter
// tests them from level kLmkDeepLevel on) are spread out instead: a
// survivor h of u at level d is proven by landmark l when
// |sd(u,l) - sd(h,l)| >= d, that is when l lies behind h on a shortest path
// from u (or behind u), and for far-apart u and h that region is near the
// graph's periphery, where high-ranked vertices of a high-diameter graph
// seldom lie. Each spread landmark, chosen in turn, maximises over the
// vertices reached in the first round the smaller of (a) its distance to
// the first round's landmarks and (b) the landmark lower bound
// max_j |sd(v,l_j) - sd(p,l_j)| of its distance to every spread landmark p
// chosen before it (ties to the smaller id), so it is far from all of
// them; a second round of searches gives their distances. When no vertex
// is farther than D from the first landmarks and 2D < kLmkDeepLevel, the
// labels they cover stop short of the levels that test spread landmarks,
// and none are placed.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <utility>

#include "pspc_level.cuh"

namespace pspc {

constexpr int kLmkGroup = 8;         // lanes per vertex in a BFS level
constexpr int kLmkThreads = 256;
constexpr int kLmkLevelsPerCheck = 4;  // BFS levels launched between host checks
constexpr int kLmkMaxDist = 65534;   // 0xFFFF marks "unreached" (or no such landmark)
constexpr int kSearchThreads = 1024;
constexpr int kSearchLanes = 4;      // lanes per frontier vertex of a search
constexpr int kSearchWide = 64;      // arcs from which a whole warp walks a vertex
constexpr size_t kSearchQueues = (size_t)512 << 20;  // bytes of queues held at a time
// What the two forms of a round cost: a level of all landmarks together
// (launch, its share of a host check, and the arcs and masks it reads), and
// a block's own search (arcs it walks, levels it synchronises).
constexpr double kNoLimit = 1e9;
constexpr double kMaskLevelSeconds = 8e-6, kMaskBytesPerSecond = 4e12;
constexpr double kSearchArcSeconds = 1.2e-9, kSearchLevelSeconds = 2e-6;

// Row v of the distance table: `stride` bytes holding k uint16 distances.
__device__ __forceinline__ uint16_t* lmk_row(uint8_t* ld, int64_t v, int stride) {
    return (uint16_t*)(ld + v * stride);
}

__global__ void k_lmk_init(int64_t n, int k, int stride, const int32_t* __restrict__ comp_base,
                           uint64_t* __restrict__ visited, uint64_t* __restrict__ frontier, uint8_t* __restrict__ ld) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    uint4* row = (uint4*)(ld + v * stride);
    for (int w = 0; w < stride / 16; ++w) row[w] = make_uint4(~0u, ~0u, ~0u, ~0u);
    const int64_t j = v - (comp_base ? (int64_t)comp_base[v] : 0);
    const bool is_lmk = j < k;
    visited[v] = is_lmk ? (1ull << j) : 0ull;
    frontier[v] = visited[v];
    if (is_lmk) lmk_row(ld, v, stride)[j] = 0;
}

// One BFS level for all landmarks of a round: kLmkGroup lanes per vertex OR
// the frontier masks of its neighbours; bit j is landmark slot slot0 + j.
__global__ void __launch_bounds__(kLmkThreads)
    k_lmk_level(int64_t n, int stride, int level, uint64_t full, int slot0, const int64_t* __restrict__ rp,
                const int32_t* __restrict__ col, const uint64_t* __restrict__ frontier, uint64_t* __restrict__ next,
                uint64_t* __restrict__ visited, uint8_t* __restrict__ ld, int* __restrict__ changed) {
    const int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kLmkGroup;
    const int gl = threadIdx.x % kLmkGroup;
    uint64_t acc = 0, vis = full;
    if (v < n) {
        vis = visited[v];
        if (vis != full)
            for (int64_t a = rp[v] + gl; a < rp[v + 1]; a += kLmkGroup) acc |= __ldg(frontier + __ldg(col + a));
    }
#pragma unroll
    for (int o = kLmkGroup / 2; o > 0; o >>= 1) acc |= __shfl_xor_sync(0xFFFFFFFFu, acc, o, kLmkGroup);
    if (v >= n) return;
    const uint64_t fresh = acc & ~vis;
    if (gl == 0) {
        next[v] = fresh;
        if (fresh) {
            visited[v] = vis | fresh;
            *changed = 1;
        }
    }
    for (int j = gl; j < 64; j += kLmkGroup)
        if ((fresh >> j) & 1ull) lmk_row(ld, v, stride)[slot0 + j] = (uint16_t)level;
}

// The search from one landmark (slot slot0 + block) in one block: reached
// vertices as bits in shared memory, the frontier a stretch of the block's
// queue of n vertices in global memory, one barrier a level.
// A level costs its latency (a queue entry, its row, its columns, a shared
// atomic), 1 to 2 us, where a launch over all vertices and the host check it
// shares cost 10: all landmarks of grid 61x67 4.2 -> 1.1 ms, of grid 256x256
// 20.6 -> 2.9 ms, of grid 16x2000 63 -> 4.7 ms.
__global__ void __launch_bounds__(kSearchThreads)
    k_lmk_search(int64_t n, int stride, int slot0, const int32_t* __restrict__ ids, const int64_t* __restrict__ rp,
                 const int32_t* __restrict__ col, int32_t* queue, uint8_t* __restrict__ ld) {
    extern __shared__ uint32_t s_seen[];
    __shared__ int s_new[3];  // vertices found by the last, this and the next level
    const int tid = threadIdx.x, lane = tid & 31, gl = tid % kSearchLanes;
    const int slot = slot0 + blockIdx.x;
    const int64_t src = ids[slot];
    if (src < 0 || src >= n) return;
    int32_t* q = queue + (int64_t)blockIdx.x * n;
    const int words = (int)((n + 31) / 32);
    for (int w = tid; w < words; w += kSearchThreads) s_seen[w] = w == (int)(src >> 5) ? 1u << (src & 31) : 0u;
    if (tid < 3) s_new[tid] = 0;
    if (tid == 0) {
        q[0] = (int32_t)src;
        lmk_row(ld, src, stride)[slot] = 0;
    }
    __syncthreads();
    int64_t lo = 0, hi = 1;  // the frontier is q[lo..hi)
    for (int level = 1; lo < hi && level <= kLmkMaxDist; ++level) {
        int* found = &s_new[level % 3];
        // the next level's count: last read two barriers ago
        if (tid == 0) s_new[(level + 1) % 3] = 0;
        auto reach = [&](int64_t a) {
            const int32_t v = __ldg(col + a);
            const uint32_t bit = 1u << (v & 31);
            if (s_seen[v >> 5] & bit) return;
            if (atomicOr(&s_seen[v >> 5], bit) & bit) return;
            q[hi + atomicAdd(found, 1)] = v;  // each vertex once: below n
            lmk_row(ld, v, stride)[slot] = (uint16_t)level;
        };
        for (int64_t base = lo + (tid - lane) / kSearchLanes; base < hi; base += kSearchThreads / kSearchLanes) {
            const int64_t i = base + lane / kSearchLanes;
            int64_t a0 = 0, a1 = 0;
            if (i < hi) {
                const int32_t u = q[i];
                a0 = rp[u];
                a1 = rp[u + 1];
            }
            const bool wide = a1 - a0 >= kSearchWide;
            if (!wide)
                for (int64_t a = a0 + gl; a < a1; a += kSearchLanes) reach(a);
            for (unsigned m = __ballot_sync(0xFFFFFFFFu, wide && gl == 0); m; m &= m - 1) {
                const int from = __ffs(m) - 1;
                const int64_t b0 = __shfl_sync(0xFFFFFFFFu, a0, from), b1 = __shfl_sync(0xFFFFFFFFu, a1, from);
                for (int64_t a = b0 + lane; a < b1; a += 32) reach(a);
            }
        }
        __syncthreads();
        lo = hi;
        hi += *found;
    }
}

// The largest score of a block's vertices goes into *key: score << 32 | ~v,
// so ties go to the smaller id.
__device__ __forceinline__ void lmk_best(int64_t n, int64_t v, uint32_t score, unsigned long long* key) {
    __shared__ unsigned long long s_best[kLmkThreads / 32];
    unsigned long long best = v < n ? (unsigned long long)score << 32 | (0xFFFFFFFFull - (unsigned long long)v) : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
    if ((threadIdx.x & 31) == 0) s_best[threadIdx.x / 32] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kLmkThreads / 32; ++w) best = max(best, s_best[w]);
        atomicMax(key, best);
    }
}

// Spread landmarks. cur[v]: the score of v (the smaller of its distance to
// the first round's k1 landmarks and its lower bounds to the spread ones
// chosen so far); 0 for vertices no first-round landmark reached. dmax: the
// largest distance of any vertex from a first-round landmark. key: the vertex
// of the largest score (lmk_best).
__global__ void k_lmk_score(int64_t n, int stride, int k1, const uint8_t* __restrict__ ld, uint32_t* __restrict__ cur,
                            unsigned* __restrict__ dmax, unsigned long long* __restrict__ key) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t m = 0xFFFFFFFFu, far = 0;
    if (v < n) {
        const uint16_t* r = (const uint16_t*)(ld + v * stride);
        for (int j = 0; j < k1; ++j)
            if (r[j] != 0xFFFFu) {
                m = min(m, (uint32_t)r[j]);
                far = max(far, (uint32_t)r[j]);
            }
        m = m == 0xFFFFFFFFu ? 0u : m;
        cur[v] = m;
    }
    lmk_best(n, v, m, key);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) far = max(far, __shfl_xor_sync(0xFFFFFFFFu, far, o));
    if ((threadIdx.x & 31) == 0 && far) atomicMax(dmax, far);
}

// Takes the chosen vertex p as spread landmark `slot` (ids[slot]) and
// lowers every score to the landmark lower bound of sd(v, p) (0xFFFF when
// exactly one of v, p was reached by some first-round landmark: they are
// not connected). next: the vertex of the largest score left (a launch of
// its own for it took as long again: 96 landmarks, 192 launches).
__global__ void k_lmk_take(int64_t n, int stride, int k1, const uint8_t* __restrict__ ld, uint32_t* __restrict__ cur,
                           const unsigned long long* __restrict__ key, int32_t* __restrict__ ids, int slot,
                           unsigned long long* __restrict__ next) {
    const int64_t p = (int64_t)(0xFFFFFFFFull - (*key & 0xFFFFFFFFull));
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v == 0) ids[slot] = (int32_t)p;
    if (p >= n) return;  // the whole grid
    uint32_t score = 0;
    if (v < n) {
        const uint16_t* rv = (const uint16_t*)(ld + v * stride);
        const uint16_t* rp = (const uint16_t*)(ld + p * stride);
        uint32_t lb = 0;
        for (int j = 0; j < k1; ++j) {
            const uint32_t a = rv[j], b = rp[j];
            if (a == 0xFFFFu && b == 0xFFFFu) continue;
            if (a == 0xFFFFu || b == 0xFFFFu) {
                lb = 0xFFFFu;
                break;
            }
            lb = max(lb, a > b ? a - b : b - a);
        }
        score = min(cur[v], lb);
        cur[v] = score;
    }
    lmk_best(n, v, score, next);
}

// Sources of a later round: landmark slot s0 + j at vertex ids[s0 + j]
// (none for -1).
__global__ void k_lmk_seed(int64_t n, int s0, int count, int stride, const int32_t* __restrict__ ids,
                           uint64_t* __restrict__ visited, uint64_t* __restrict__ frontier, uint8_t* __restrict__ ld) {
    const int j = threadIdx.x;
    if (j >= count) return;
    const int64_t v = ids[s0 + j];
    if (v < 0 || v >= n) return;
    atomicOr((unsigned long long*)&visited[v], 1ull << j);
    atomicOr((unsigned long long*)&frontier[v], 1ull << j);
    lmk_row(ld, v, stride)[s0 + j] = 0;
}

// The searches of one round: bits of `full` from the round's sources
// (already set in visited and fa), distances into slots slot0 + j. Starts at
// level *next and stops after max_levels; *next is then the level to go on
// from, or 0 if there is nothing more to reach.
static cudaError_t lmk_round(int64_t n, const int64_t* rp, const int32_t* col, int stride, uint64_t full, int slot0,
                             uint8_t* ld, uint64_t* visited, uint64_t* fa, uint64_t* fb, int* changed, cudaStream_t st,
                             int64_t* nl, double max_levels, int* next) {
    static_assert(kLmkLevelsPerCheck % 2 == 0, "fa holds the frontier at every stop");
    cudaError_t e = cudaSuccess;
    const unsigned blocks = (unsigned)((n * kLmkGroup + kLmkThreads - 1) / kLmkThreads);
    int level = *next;
    *next = 0;
    while (level <= kLmkMaxDist) {
        if ((e = cudaMemsetAsync(changed, 0, sizeof(int), st)) != cudaSuccess) return e;
        // A level after the last one that reaches anything changes nothing,
        // so a few levels run between host checks.
        for (int t = 0; t < kLmkLevelsPerCheck && level <= kLmkMaxDist; ++t, ++level) {
            k_lmk_level<<<blocks, kLmkThreads, 0, st>>>(n, stride, level, full, slot0, rp, col, fa, fb, visited, ld,
                                                        changed);
            std::swap(fa, fb);
            ++*nl;
        }
        int h = 0;
        if ((e = cudaMemcpyAsync(&h, changed, sizeof(int), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
        if (!h) break;
        if (level > max_levels) {
            *next = level;
            break;
        }
    }
    return cudaGetLastError();
}

// A block for each of the slots slot0..slot0+count-1, from vertex ids[slot].
// It starts from the source again where a round stopped: the levels that are
// there are written once more. cudaErrorMemoryAllocation: nothing was done.
static cudaError_t lmk_search(int64_t n, const int64_t* rp, const int32_t* col, int stride, int slot0, int count,
                              const int32_t* ids, uint8_t* ld, cudaStream_t st, int64_t* nl) {
    const size_t smem = (size_t)((n + 31) / 32) * 4;
    const int per = (int)std::max<size_t>(1, std::min<size_t>(count, kSearchQueues / ((size_t)n * 4)));
    void* queue = nullptr;
    cudaError_t e = dev_alloc(&queue, (size_t)per * n * 4, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e;
    }
    e = cudaFuncSetAttribute(k_lmk_search, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    for (int s = 0; e == cudaSuccess && s < count; s += per) {
        k_lmk_search<<<std::min(per, count - s), kSearchThreads, smem, st>>>(n, stride, slot0 + s, ids, rp, col,
                                                                             (int32_t*)queue, ld);
        *nl += 1;
        e = cudaGetLastError();
    }
    dev_free(queue, st);
    return e;
}

int landmark_bfs(int64_t n, int64_t arcs, const int64_t* rp, const int32_t* col, const int32_t* comp_base, int k, int stride,
                 uint8_t* ld, int32_t* ids, cudaStream_t st, int64_t* launches) {
    if (k < 1 || k > kLmkMax || (comp_base && k > 64) || stride % 16 || stride < 2 * k) return PSPC_E_INVAL;
    // slots 0..k1-1: the highest-ranked vertices; k1..k-1: spread landmarks,
    // only for one graph large enough to place them
    const int k1 = (comp_base || k <= kLmkShallow || n <= 4 * (int64_t)k) ? k : kLmkShallow;
    void* mem = nullptr;
    const size_t masks = (size_t)n * 8;
    cudaError_t e = dev_alloc(&mem, 3 * masks + (size_t)n * 4 + kLmkMax * 12 + 512, st);
    if (e != cudaSuccess) return cuda_status(e);
    uint64_t* visited = (uint64_t*)mem;
    uint64_t* fa = visited + n;
    uint64_t* fb = fa + n;
    unsigned long long* keys = (unsigned long long*)(fb + n);
    int32_t* d_ids = (int32_t*)(keys + kLmkMax + 1);
    uint32_t* cur = (uint32_t*)(d_ids + kLmkMax + 2);
    int* changed = (int*)(cur + n);
    int32_t h_ids[kLmkMax];
    for (int j = 0; j < kLmkMax; ++j) h_ids[j] = j < k1 && j < n ? j : -1;
    int64_t nl = 1;
    const unsigned vb = (unsigned)((n + kLmkThreads - 1) / kLmkThreads);
    // first search batch: the first (up to 64) highest-ranked vertices of every graph
    const int r1 = k1 < 64 ? k1 : 64;
    // Blocks of their own search when that is expected to be shorter. A first
    // round does not know how deep the graph is: it goes over to them once the
    // levels behind it have cost as much as a block's walk of all arcs would,
    // so it never takes much more than twice the better form.
    int dev = 0, sms = 0, smem_max = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const double mask_level = kMaskLevelSeconds + (12.0 * arcs + 24.0 * n) / kMaskBytesPerSecond;
    const double arcs_own = kSearchArcSeconds * arcs;
    const bool may_search = !comp_base && (n + 31) / 32 * 4 + 1024 <= smem_max;
    const double max_levels = may_search ? std::max(8.0, arcs_own / (mask_level - kSearchLevelSeconds)) : kNoLimit;
    const auto whole = [](int count) { return count == 64 ? ~0ull : (1ull << count) - 1; };
    int level = 1;
    k_lmk_init<<<vb, kLmkThreads, 0, st>>>(n, r1, stride, comp_base, visited, fa, ld);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_ids, h_ids, sizeof(h_ids), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = lmk_round(n, rp, col, stride, whole(r1), 0, ld, visited, fa, fb, changed, st, &nl, max_levels, &level);
    if (e == cudaSuccess && level) {
        e = lmk_search(n, rp, col, stride, 0, r1, d_ids, ld, st, &nl);
        if (e == cudaErrorMemoryAllocation)  // no room for queues: on from there, together
            e = lmk_round(n, rp, col, stride, whole(r1), 0, ld, visited, fa, fb, changed, st, &nl, kNoLimit, &level);
    }
    // Spread landmarks, from the first round's distances (k1 <= 64). The
    // filter tests them from level kLmkDeepLevel on; when every distance
    // from the first landmarks is at most D with 2D < kLmkDeepLevel, labels
    // between vertices they reach stop short of that level, and the spread
    // ones are left out (slots k1..k-1 stay empty).
    int kk = k;
    unsigned dmax = 0;
    if (e == cudaSuccess && k1 < k) {
        e = cudaMemsetAsync(keys, 0, (kLmkMax + 1) * 8, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(changed, 0, sizeof(unsigned), st);
        if (e == cudaSuccess) {
            k_lmk_score<<<vb, kLmkThreads, 0, st>>>(n, stride, k1, ld, cur, (unsigned*)changed, keys + k1);
            nl += 1;
            e = cudaMemcpyAsync(&dmax, changed, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e == cudaSuccess && 2 * dmax < (unsigned)kLmkDeepLevel) kk = k1;
        }
        if (e == cudaSuccess && kk > k1) {
            for (int j = k1; j < k; ++j) {
                k_lmk_take<<<vb, kLmkThreads, 0, st>>>(n, stride, k1, ld, cur, keys + j, d_ids, j, keys + j + 1);
                nl += 1;
            }
            e = cudaGetLastError();
        }
    }
    // later landmarks: blocks of their own, or batches of 64 from their
    // vertices in d_ids
    bool found = false;
    if (e == cudaSuccess && may_search && kk > r1 &&
        (kk - r1 + 63) / 64 * (double)dmax * mask_level > arcs_own + dmax * kSearchLevelSeconds) {
        e = lmk_search(n, rp, col, stride, r1, kk - r1, d_ids, ld, st, &nl);
        found = e == cudaSuccess;
        if (e == cudaErrorMemoryAllocation) e = cudaSuccess;
    }
    for (int s0 = r1; e == cudaSuccess && !found && s0 < kk; s0 += 64) {
        const int cnt = kk - s0 < 64 ? kk - s0 : 64;
        e = cudaMemsetAsync(visited, 0, 2 * masks, st);
        if (e == cudaSuccess) {
            k_lmk_seed<<<1, 64, 0, st>>>(n, s0, cnt, stride, d_ids, visited, fa, ld);
            nl += 1;
            int from = 1;
            e = lmk_round(n, rp, col, stride, whole(cnt), s0, ld, visited, fa, fb, changed, st, &nl, kNoLimit, &from);
        }
    }
    if (e == cudaSuccess && ids) {
        e = cudaMemcpyAsync(h_ids, d_ids, sizeof(h_ids), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e == cudaSuccess)
            for (int j = 0; j < kLmkMax; ++j) ids[j] = j < kk ? h_ids[j] : -1;
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    const int rc = e == cudaSuccess ? PSPC_OK : cuda_status(e);
    dev_free(mem, st);
    if (launches) *launches += nl;
    return rc;
}

}  // namespace pspc
