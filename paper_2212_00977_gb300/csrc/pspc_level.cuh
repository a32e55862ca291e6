// Internal interface between the build orchestration (pspc_build.cu) and
// the per-level kernels (pspc_level.cu): status record, kernel arguments,
// the on-chip table layout and the host-side launchers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "pspc_internal.cuh"

namespace pspc {

constexpr int kLevelThreads = 512;  // CTA of the level kernel for heavy vertices
constexpr int kLightThreads = 128;  // CTA of the level kernel for light vertices
constexpr uint32_t kLightCap = 1024;  // candidate slots of a light vertex
constexpr uint32_t kOffStartCap = 16384;    // first off-chip table size
constexpr uint32_t kOffSlabCap = 1u << 17;  // off-chip slab of the first pass, in candidate slots
constexpr int kMicroThreads = 256;    // the warp-per-vertex level kernel: 8 vertices per CTA
constexpr int kMicroBucket = 7;       // micro: fewer than 2^7 pulled entries (four to a lane); at levels 2 and 3,
                                      // where nothing is filtered out first, 2^6. Since levels use balls either line
                                      // does there: R-MAT 262,144 builds in 48.2 ms, with 2^7 in 48.4, BA 20,011 in
                                      // 2.91 both ways, the batch of 96 BA graphs in 79.6 and 77.9
constexpr int kTinyBucket = 6;        // of those, fewer than 2^6: two to a lane, and fewer registers
constexpr int kLightBucket = 9;       // light: fewer than 2^9 pulled entries, so at most 2 * 511 < kLightCap
                                      // slots are asked for, and the table never overflows
constexpr int kWarpLevelsFew = 32;    // automatic warp-per-vertex levels: while the last level had under this
                                      // many candidates per vertex
constexpr int kArcChunk = kLevelThreads;  // arcs staged per gather chunk (the CTA size)

// Resident CTAs per SM each kernel size is built for (64 registers a thread).
__host__ __device__ constexpr int level_min_blocks(int nt) { return nt >= 512 ? 2 : 8; }
constexpr int kBuckets = 64;
constexpr size_t kBitmapBudget = 40 * 1024;  // on-chip bytes for the level bitmaps
constexpr int kLmkShallow = 32;    // landmarks the filter tests below level kLmkDeepLevel
constexpr int kLmkDeepLevel = 16;  // from this level on, the filter tests every landmark

// Vertices merged by direct addressing (k_level_dense).
// Small CTAs: the kernel alternates short phases between barriers and waits
// for its reads (a third of the stalls each), so eight CTAs of 256 threads
// with 4,608-id windows fill each other's gaps best: R-MAT 2^20 builds in 488
// ms, with 4 CTAs and 11,264 ids 578, 5 and 8,960 547, 6 and 6,912 505, 7 and
// 5,760 515, 4 of 512 threads and 10,240 ids 496 (batch of 96 BA graphs 83 ms,
// 91, 90, 86, 86 and 92; all before the kernel's checks).
constexpr int kDenseThreads = 256;
constexpr int kDenseBlocks = 8;             // resident CTAs per SM (26 KB of shared memory each)
constexpr uint32_t kDenseWindow = 4608;     // ids per on-chip window, a multiple of 128
constexpr uint32_t kDenseBounds = 1024;     // cells of the table of window starts
constexpr uint32_t kDenseSlabCap = 1u << 21;  // candidates of one vertex at most (32 MB of slab a CTA)
constexpr int kDenseBucket = 32;            // dense vertices are bucketed at 32 + floor(log2 pulled entries)
// A vertex with fewer pulled entries has too few to pay for the windows; it
// is one of the light class then. A batch of 96 BA graphs builds in 79.6 ms with
// 512 here, 81.3 with 256, 87.2 with 768, 91.5 with 1,024, 99.7 with 2,048 (R-MAT
// 262,144 48.2, 47.5, 49.1, 49.9 and 53.8 ms, BA 20,011 2.91, 2.93, 3.02, 3.13
// and 3.43). Per window of its id range it needs 12 (window overhead against a
// hash in device memory): R-MAT 2^20 487 ms with 12, 486 with 6, 494 with 20.
constexpr int64_t kDenseMinRaw = 512;
constexpr int64_t kDenseRawPerWindow = 12;
// Granular builds run one hash CTA per vertex, and the dense kernel at half
// occupancy: only vertices that would mostly overflow the hash pay (granular,
// R-MAT 262,144 builds in 81.6 ms with 16,384, in 103.2 with 65,536 and in 112.7
// without direct addressing; R-MAT 65,536 11.8, 11.8 and 11.5, BA 100,000 with
// m = 8 64.1, 61.2 and 61.3, BA 20,011 3.7 in all). Lower lines are closed: a
// granular build of BA 20,011 with one (512 pulled entries and 384 a window)
// ended in a GPU fault, Xid 13 and 43, whose cause is not known.
constexpr int64_t kDenseMinRawGranular = 16384;

struct LevelStatus {
    unsigned long long raw_total;
    unsigned long long unique_total;
    unsigned long long bump;        // arena fill after this level
    unsigned long long need_cap_c;  // largest candidate table of the off-chip class
    unsigned long long need_cap_u;  // largest label table of the off-chip class
    unsigned long long need_cap_d;  // most candidates a dense vertex can have
    unsigned long long active_arcs;
    int n_active;
    int n_smem;
    int n_global;
    int n_retry;
    unsigned long long prefix_skipped;  // rule-1 entries skipped below the dense prefixes
    unsigned long long lmk_pruned;  // candidates dropped by the landmark filter
    unsigned long long lmk_proven;  // candidates the landmarks proved to survive
    int arena_overflow;
    int work_smem;
    int work_global;
    int work_light;
    int n_giant;     // off-chip vertices whose candidates overflow the slab
    int work_giant;
    int work_micro;
    int work_tiny;
    int n_held;                  // vertices whose segment waits for deferred scans
    int work_scan;
    unsigned int n_scan_open;    // of them, left after the neighbours' proof
    unsigned long long n_scan;   // deferred scans asked for (those past the queue's size run in place): 64 bits,
                                 // as a level can ask for more than 2^32
    unsigned long long dropped;  // entries that deferred scans took out of their segments
    int max_deg;     // largest degree of the graph (level 2 only)
    int bad;         // k_level_dense met a run outside its segment, a hub outside its window or a full slab
    int work_dense;
    unsigned int cmax;  // largest count appended at this level (0xFFFFFFFF: 2^32 or more, or flagged)
    // on-chip attempts and overflows of vertices that can overflow, by
    // floor(log2 pulled entries): where most overflow, the rest go straight
    // to the off-chip pass
    unsigned int route_att[kBuckets];
    unsigned int route_ovf[kBuckets];
    int bucket_cnt[kBuckets];
    int bucket_fill[kBuckets];
};

// Deferred label scans. A vertex with undecided candidates appends them with its survivors and asks for their scans; the
// scans of all vertices then run evenly over the GPU (k_scan_deferred), and
// the last one of a vertex closes its segment.
constexpr int kDeferLevel = 16;  // from this level on
// and with this many active vertices times levels, where the scans are
// worth two launches a level. Builds with 2^17, 2^18 and 2^19 here, and without
// deferral from this level on: grid 61x67 11.9, 11.1, 11.1 and 11.1 ms, 90x90
// 20.3, 20.4, 20.8 and 20.8, 128x128 37.0, 37.7, 39.5 and 52, 181x181 78.5, 80.4,
// 85.2 and 179, 256x256 241, 242, 243 and 742.
constexpr int64_t kDeferWork = 1 << 18;
// Before it, with this many pulled entries and active vertices: a vertex with
// a hundred undecided candidates scans for them one after another while the
// GPU is idle (R-MAT 65,536, level 5: 788,080 pulled, 2.5 ms in place and 0.4
// deferred). The queue, its allocation and two launches cost some 60 us: of
// BA 100,000, level 8, 61,290 pulled take 0.18 ms in place and 0.21 deferred.
// Builds with 1,024, 2,048 and 4,096 active vertices as the line, and without
// deferral before kDeferLevel: R-MAT 65,536 8.73, 8.73, 9.17 and 9.63 ms, 6,000
// 1.23, 1.24, 1.28 and 1.27, BA 40,000 (m = 3) 5.47, 5.47, 5.48 and 5.97, BA 2,000
// 1.10, 1.04, 1.05 and 1.04; within 2% whatever the line for BA of 3,000, 4,500,
// 9,000 and 100,000 vertices and R-MAT of 3,000, 12,000 and 24,000.
constexpr int kDeferShallow = 4;
constexpr unsigned long long kDeferPulled = 1 << 18;
constexpr int kDeferActive = 2048;
constexpr int kNeighbourLevel = 8;  // from here on a scan costs more than the neighbours' proof that may spare it
struct HeldSegment {
    unsigned long long start;  // of the entries appended so far in the arena
    int32_t u;
    int32_t len;
    int32_t scans;    // asked for, less the proven ones
    int32_t done;     // parts of them that have run
    int32_t pruned;   // some scan pruned its entry (marked kMarkBit in the arena)
};
struct DeferredScan {
    int32_t held;  // which HeldSegment (-1: none)
    int32_t pos;   // which of its entries
};
// First place in a queue of `cap` for scans that come after `before` others
// (cap: it is full).
__host__ __device__ inline unsigned int scan_place(unsigned long long before, unsigned int cap) {
    return before < cap ? (unsigned int)before : cap;
}

// Rows of a distance ball (pspc_ball.cu): row u starts at word off[u] (n + 1
// values; batches), or at u * words. A multiple of 4 words each; bit r is the
// vertex r after the first of u's graph.
struct BallRows {
    const int64_t* off;
    int64_t words;
};
constexpr int64_t kBallBytes = (int64_t)1 << 31;  // most bytes of one ball (two are held)
// slices: arcs / 128 + 1 pairs. total_words: of one ball; max_words: of its longest row.
cudaError_t launch_ball_init(int64_t n, int64_t arcs, const int64_t* rp, const int32_t* arc_src, const int32_t* col,
                             const int32_t* comp_base, const BallRows& R, int64_t total_words, uint32_t* ball, int2* slices,
                             int* n_slices, cudaStream_t st);
cudaError_t launch_ball_step(int64_t n, const int64_t* rp, const int32_t* col, const BallRows& R, int64_t max_words,
                             const int2* slices, int n_slices, const uint32_t* from, uint32_t* to, cudaStream_t st);

struct LevelArgs {
    int d;
    int64_t n;
    const int64_t* rp;
    const int32_t* col;
    const uint32_t* cnt_arc;
    const uint32_t* arc_lo;  // first pulled entry of each arc's segment (dense-prefix skip), or NULL
    const int32_t* hpre;     // dense prefix per vertex when arc_lo is set
    // Push paradigm: the entries sent to u this level lie in
    // push_hub/push_cnt[push_off[rp[u]] .. push_off[rp[u+1]]) (NULL: pull).
    const uint32_t* push_hub;
    const uint64_t* push_cnt;
    const int64_t* push_off;
    const uint64_t* seg;  // [levels][n]
    uint64_t* seg_out;    // row d
    uint32_t* hub_arena;
    uint64_t* cnt_arena;
    unsigned long long arena_cap;
    const int64_t* raw_u;
    const int64_t* lab_size;
    const int32_t* items;
    int n_items;
    int* work;
    LevelStatus* stt;
    int32_t* retry_list;  // appended at retry_list[k]
    int32_t* giant_list;  // off chip: vertices for the final pass with full-size slabs
    uint32_t off_start_cap;  // off chip: first table size (0: the full bound)
    uint32_t cap_c_max;   // candidate table slots (on chip, or per-CTA scratch)
    uint32_t cap_u_max;   // label hash slots (hash map kind)
    uint32_t bm_words;    // words per level bitmap (bitmap map kind)
    const int32_t* comp_base;  // first rank-space id of each vertex's graph in a batch (NULL: 0)
    int granular;              // 1: CTA b handles item b only (grid = n_items); 0: persistent
    uint8_t* gscratch;    // per-CTA table memory when the tables are off chip
    size_t gscratch_stride;
    const uint8_t* lmk;   // [n][lmk_stride] bytes of uint16 landmark distances, or NULL (no filter)
    int lmk_stride;       // bytes per row: a multiple of 16, <= 2 kLmkMax
    int lmk_words;        // 16-byte words of each row the filter tests at this level
    const uint32_t* ball; // ball d-1 (rule 2 is a bit of it), or NULL
    BallRows ball_rows;
    HeldSegment* held;    // deferred scans (NULL: scans run in place)
    DeferredScan* scans;
    unsigned int scan_cap;
};

// Table layout (on chip, or in per-CTA device scratch). The map region also
// holds the survivor sort buffer once the prune step is done.
struct LevelLayout {
    size_t cnt, key, map, list, st, pfx, total;
};

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

__host__ __device__ inline LevelLayout level_layout(uint32_t cap_c, size_t map_bytes, int nt = kLevelThreads) {
    LevelLayout L;
    size_t p = 0;
    L.cnt = p;
    p += (size_t)cap_c * 8;
    L.key = p;
    p = align16(p + (size_t)cap_c * 4);
    L.map = p;
    p = align16(p + (map_bytes > (size_t)cap_c * 8 ? map_bytes : (size_t)cap_c * 8));
    L.list = p;
    p = align16(p + (size_t)cap_c * 4);
    L.st = p;
    p = align16(p + (size_t)nt * 8);
    L.pfx = p;
    p = align16(p + (size_t)(nt + 1) * 8);
    L.total = p;
    return L;
}

__host__ __device__ inline size_t bitmap_bytes(int d, uint32_t bm_words) { return (size_t)(d - 1) * bm_words * 4; }
__host__ __device__ inline size_t hashmap_bytes(uint32_t cap_u) { return (size_t)cap_u * 6; }

__host__ __device__ inline uint32_t cand_cap_for(int64_t raw, int64_t u, uint32_t cap_max) {
    const int64_t bound = raw < u ? raw : u;  // distinct hubs <= pulled entries, and < u
    const uint64_t want = (uint64_t)(2 * bound) < 64ull ? 64ull : (uint64_t)(2 * bound);
    return want >= cap_max ? cap_max : pow2_ceil(want);
}
__host__ __device__ inline uint32_t label_cap_for(int64_t lab) {
    const uint64_t want = (uint64_t)(lab + lab / 3 + 1);
    return pow2_ceil(want < 64ull ? 64ull : want);
}

// Which vertices a level merges by direct addressing: `on` for the level,
// and the largest count of the level below.
struct DenseRule {
    int on;
    uint32_t cmax;
    int64_t min_raw;
    const int32_t* comp_base;
};

// u (id span + first id of its graph) with `raw` pulled entries over deg arcs.
__host__ __device__ inline bool dense_vertex(const DenseRule& R, int64_t raw, int64_t span, int64_t deg) {
    const int64_t windows = (span + kDenseWindow - 1) / kDenseWindow;
    return R.on && raw >= R.min_raw && raw >= kDenseRawPerWindow * windows && raw < ((int64_t)1 << 32) &&
           (uint64_t)R.cmax * (uint64_t)(deg + 1) < ((uint64_t)1 << 32) &&
           (raw < span ? raw : span) <= (int64_t)kDenseSlabCap;
}

enum MapKind { kMapBitmap = 0, kMapHash = 1, kMapSeg = 2 };

// Bytes of the label-map region for a map kind (host plan and kernel must
// agree: the kernel carves its tables with exactly this size).
__host__ __device__ inline size_t level_map_bytes(int kind, int d, uint32_t bm_words, uint32_t cap_u) {
    return kind == kMapBitmap ? bitmap_bytes(d, bm_words) : kind == kMapHash ? hashmap_bytes(cap_u) : 0;
}

// Landmark distances (Section "Landmark-Based Filtering"): the first
// min(k, kLmkShallow) landmarks of every graph are its highest-ranked
// vertices (id comp_base + j, or j when comp_base is NULL); for one graph
// (comp_base NULL) with k > kLmkShallow and more than 4k vertices the others
// are spread out over the graph (chosen one by one, each far from the
// landmarks before it). ld is [n][stride] bytes, k uint16 distances per
// row, 0xFFFF where the distance is undefined (unreached, or no such
// landmark). ids (NULL, or host int32[64] out): the id of landmark j, -1 for
// none. Synchronises st every few BFS levels.
int landmark_bfs(int64_t n, int64_t arcs, const int64_t* rp, const int32_t* col, const int32_t* comp_base, int k, int stride,
                 uint8_t* ld, int32_t* ids, cudaStream_t st, int64_t* launches);

// Push paradigm (Algorithm PUSH): every arc u->v sends u the entries of
// L_{d-1}(v) that the pull would read for it (cnt_arc[a] of them from
// arc_lo[a], or from 0), into u's bucket at push_off[a]. Warp per arc.
cudaError_t launch_push_scatter(int64_t arcs, const int32_t* col, const uint64_t* seg_prev,
                                const uint32_t* hub_arena, const uint64_t* cnt_arena, const uint32_t* cnt_arc,
                                const uint32_t* arc_lo, const int64_t* push_off, uint32_t* push_hub,
                                uint64_t* push_cnt, cudaStream_t st);
cudaError_t launch_arc_counts(int64_t arcs, const uint32_t* cnt_arc, int64_t* out, cudaStream_t st);

// Launchers (pspc_level.cu). Each returns a CUDA error code of the launch.
cudaError_t launch_arc_src(const int64_t* rp, int64_t n, int32_t* arc_src, cudaStream_t st);
// Dense prefix of every vertex (k_dense_prefix): hpre[u] = the smallest rank
// id x >= (first id of u's graph) not in L_<d(u), at most u, looking at the
// first kDensePrefixWindow ids. Every pulled entry whose hub is below it is
// in L_<d(u), so the membership filter would drop it; the cost pass then
// starts each arc's pull after those entries.
constexpr int kDensePrefixWindow = 1024;
constexpr int kDensePrefixMaxLevel = 8;  // deeper levels: no skip (cost grows with d)
constexpr double kDensePrefixMinGain = 0.10;  // stop skipping once it saves less than this share of a level's pulls
cudaError_t launch_dense_prefix(int d, int64_t n, const uint64_t* seg, const uint32_t* hub_arena,
                                const int32_t* comp_base, int32_t* hpre, cudaStream_t st);
cudaError_t launch_level_begin(int64_t n, uint64_t* seg_row, int64_t* raw_u, LevelStatus* stt, LevelStatus* next,
                               unsigned long long bump, cudaStream_t st);
// hpre NULL: no skip (arc_lo is not written). raw_u has to be zero. max_deg
// (may be NULL): the largest degree, for what is there already.
cudaError_t launch_cost(int d, int64_t n, int64_t arcs, const int64_t* rp, const int32_t* col,
                        const int32_t* arc_src, const uint64_t* seg_prev, const uint32_t* hub_arena,
                        const int32_t* hpre, uint32_t* arc_lo, uint32_t* cnt_arc, int64_t* raw_u,
                        int64_t* lab_size, LevelStatus* stt, int64_t label_limit, const DenseRule& dense,
                        int32_t* glist, int32_t* items, int* max_deg, cudaStream_t st, int64_t* launches);
// launch_level_begin and launch_cost in two launches, for graphs of degrees
// up to kCostMaxDegree: four lanes walk the arcs of a vertex there. *stt was
// cleared as the `next` of the level before.
constexpr int kCostMaxDegree = 32;
cudaError_t launch_cost_level(int64_t n, const int64_t* rp, const int32_t* col, const uint64_t* seg_prev,
                              uint64_t* seg_row, const uint32_t* hub_arena, const int32_t* hpre, uint32_t* arc_lo,
                              uint32_t* cnt_arc, int64_t* raw_u, int64_t* lab_size, LevelStatus* stt, LevelStatus* next,
                              unsigned long long bump, int64_t label_limit, const DenseRule& dense, int32_t* glist,
                              int32_t* items, cudaStream_t st);
cudaError_t level_kernel_attrs(int map_kind, size_t smem_bytes, int* occupancy, int nt = kLevelThreads);
cudaError_t launch_level(int map_kind, bool offchip, int grid, size_t smem_bytes, const LevelArgs& A,
                         cudaStream_t st, int nt = kLevelThreads);
// Direct addressing for vertices with many pulled entries (k_level_dense).
// Per CTA: a slab of A.cap_c_max candidates of 16 bytes in A.gscratch.
cudaError_t dense_kernel_attrs(int* occupancy);
cudaError_t launch_level_dense(int grid, const LevelArgs& A, cudaStream_t st);
// The warp-per-vertex variant for vertices with fewer than 2^kMicroBucket
// pulled entries (k_level_micro).
cudaError_t micro_kernel_occupancy(int rows, int* occupancy);
cudaError_t launch_scan_deferred(int prove_grid, int scan_grid, const LevelArgs& A, cudaStream_t st);
cudaError_t scan_kernel_occupancy(int* prove, int* scan);
cudaError_t launch_level_micro(int rows, int grid, const LevelArgs& A, cudaStream_t st);

}  // namespace pspc
