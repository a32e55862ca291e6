// The level kernel for vertices that pull many entries (part of
// pspc_level.cu): candidates are merged by direct addressing instead of a
// hash.
//
// u's candidates are hubs of u's graph ranked above u, ids in [cbase, u),
// and every level segment is hub-sorted. The ids are cut into windows of
// kDenseWindow; the part of a neighbour's segment that falls into a window
// is a contiguous run, found by binary search, so each pulled entry is still
// read exactly once. A window has one 32-bit count per id on chip: merging an
// entry is one shared-memory addition, with no probe chain, no key compare
// and no returned value, and walking the window in order yields the
// candidates already in hub order, so nothing is sorted afterwards.
//
// A vertex runs here only when no sum can reach 2^32: the largest count of
// the level below (LevelStatus::cmax, saturated, and saturated too by any
// overflow flag) times u's degree is below 2^32. The other vertices keep the
// hash kernels with 64-bit sums, carries and flags.
//
// What bounds it: latency and instructions. On R-MAT of 140,000 vertices, level
// 3, all 64 warps of an SM are there and 65% of the issue slots are used; of 24
// cycles between a warp's instructions 9 wait for reads (L2 hits 73% of them)
// and 6 at barriers; DRAM is at 8%, L2 at 25%, L1 at 49%. With four CTAs, half
// the warps, it was 41% on R-MAT 262,144. By phases, before that, on R-MAT 2^20, level 3 (3.0e10 pulled entries): half pull, a
// fifth the marking walk, a tenth each the member bitmaps and the scans of
// run lengths; at level 4 the landmark filter and the label scans take 57%.
// The hash it replaces kept tables of more than 4,096 slots in device memory,
// half of whose sectors missed L2: levels 3 and 4 took 568 and 495 ms, now
// 180 and 208 (the build 1,182 -> 488 ms). With a distance ball its row is the
// window's bitmap and only the pull is left. Eight CTAs an SM leave a thread 32
// registers, and ptxas spills (220 bytes of stores, 352 of loads); four CTAs with
// 64 registers spill nothing and were slower (kDenseThreads).
//
// Three checks keep the kernel inside its memory whatever it reads: a run of a
// segment that ends before it starts is empty, a member outside its window is
// left out, and a vertex with more candidates than the slab holds is dropped.
// By the order of the segments none of them can happen; if one does, it sets
// LevelStatus::bad and the build ends with PSPC_E_CUDA. They are there because
// one granular build (kDenseMinRawGranular) ended in a GPU fault that reading
// has not explained. They cost nothing (R-MAT 2^20 489 ms with and without) as
// long as the last one leaves the windows: going on after it, with the counts
// cleared on the spot, took 497.

// Words of the window's bitmaps.
constexpr uint32_t kDenseWords = kDenseWindow / 32;
constexpr int kDenseUnroll = 4;  // loads in flight per lane in the pull

struct DenseLayout {
    size_t mem, bnd, st, pfx, total;
};
__host__ __device__ inline DenseLayout dense_layout() {
    DenseLayout L;
    size_t p = (size_t)kDenseWindow * 4;  // the counts come first
    L.mem = p;
    p += kDenseWords * 4;
    L.bnd = p;
    p += kDenseBounds * 4;
    L.st = align16(p);
    p = L.st + (size_t)kDenseThreads * 8;
    L.pfx = p;
    p += (size_t)(kDenseThreads + 1) * 4;
    L.total = align16(p);
    return L;
}

// Exclusive scan of one value per thread into pfx[0..nc) (pfx[nc] = total);
// returns the total. With at most 32 values one barrier, else two.
__device__ uint32_t dense_scan(uint32_t v, int nc, uint32_t* pfx, uint32_t* wsum) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
    }
    if (nc <= 32) {
        if (tid < nc) pfx[tid] = incl - v;
        if (tid == nc - 1) pfx[nc] = incl;
        __syncthreads();
        return pfx[nc];
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kDenseThreads / 32; ++w) {
        const uint32_t t = wsum[w];
        before += w < warp ? t : 0u;
        total += t;
    }
    if (tid < nc) pfx[tid] = before + incl - v;
    if (tid == 0) pfx[nc] = total;
    __syncthreads();
    return total;
}

__global__ void __launch_bounds__(kDenseThreads, kDenseBlocks) k_level_dense(const LevelArgs A) {
    extern __shared__ __align__(16) uint8_t smem[];
    constexpr int NT = kDenseThreads, kWarps = NT / 32;
    constexpr uint32_t W = kDenseWindow;
    __shared__ int s_item, s_next, s_lpr, s_lpv, s_open;
    __shared__ __align__(16) uint32_t s_lmk[kLmkMax / 2];
    __shared__ uint64_t s_useg[kUSideLevels];
    __shared__ int s_wcnt[kWarps];
    __shared__ uint32_t s_wsum[kWarps];
    __shared__ unsigned long long s_base;
    const DenseLayout L = dense_layout();
    uint32_t* acc = (uint32_t*)smem;
    uint32_t* mem = (uint32_t*)(smem + L.mem);
    uint32_t* bnd = (uint32_t*)(smem + L.bnd);
    uint64_t* st = (uint64_t*)(smem + L.st);
    uint32_t* pfx = (uint32_t*)(smem + L.pfx);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int d = A.d;
    const int64_t n = A.n;
    const uint64_t* seg_prev = A.seg + (int64_t)(d - 1) * n;
    // the CTA's slab: candidates in hub order
    uint32_t* shub = (uint32_t*)(A.gscratch + (size_t)blockIdx.x * A.gscratch_stride);
    uint32_t* scnt = shub + A.cap_c_max;
    uint32_t* list = scnt + A.cap_c_max;
    uint32_t* undecided = list + A.cap_c_max;
    uint32_t cm = 0;  // largest count appended by this thread
    uint32_t dirty = W;  // words of the counts' memory to clear for the next vertex
    for (uint32_t i = tid; i < kDenseWords; i += NT) mem[i] = 0u;
    for (;;) {
        if (tid == 0) {
            s_item = atomicAdd(A.work, 1);
            s_next = 0;
            s_lpr = 0;
            s_lpv = 0;
            s_open = 0;
        }
        for (uint32_t i = tid; i < dirty; i += NT) acc[i] = 0u;
        dirty = 0;
        __syncthreads();
        if (s_item >= A.n_items) break;
        const int64_t u = A.items[s_item];
        const uint32_t cbase = A.comp_base ? (uint32_t)__ldg(A.comp_base + u) : 0u;
        const int64_t a0 = A.rp[u];
        const int deg = (int)(A.rp[u + 1] - a0);
        const uint32_t span = (uint32_t)u - cbase;  // candidates are cbase + [0, span)
        const uint32_t nwin = (span + W - 1) / W, nb = nwin - 1;
        if (A.lmk && tid < A.lmk_stride / 4)
            s_lmk[tid] = lmk_clamp(__ldg((const uint32_t*)(A.lmk + u * A.lmk_stride) + tid));

        // Where each window starts in the pulled run of every arc, and in
        // u's own segments of levels d-1 and d-2 (the only ones that a
        // pulled hub can be in): one table for all windows when it fits.
        const uint32_t* ball = ball_of(A, u);  // with a ball its row stands for both, and for rule 2
        const uint64_t own1 = ball ? 0ull : __ldg(A.seg + (int64_t)(d - 1) * n + u);
        const uint64_t own2 = !ball && d > 2 ? __ldg(A.seg + (int64_t)(d - 2) * n + u) : 0ull;
        const bool table = (uint64_t)(deg + 2) * nb <= (uint64_t)kDenseBounds;
        auto arc_run = [&](int r, uint64_t& start, uint32_t& len) {
            len = __ldg(A.cnt_arc + a0 + r);
            start = len ? seg_start(__ldg(seg_prev + __ldg(A.col + a0 + r))) + (A.arc_lo ? __ldg(A.arc_lo + a0 + r) : 0u)
                        : 0ull;
        };
        if (table && nb > 0) {
            const uint32_t cells = (uint32_t)(deg + 2) * nb;
            for (uint32_t t = tid; t < cells; t += NT) {
                const uint32_t r = t / nb, w = t - r * nb;
                uint64_t start;
                uint32_t len;
                if (r < (uint32_t)deg) arc_run((int)r, start, len);
                else {
                    const uint64_t s = r == (uint32_t)deg ? own1 : own2;
                    start = seg_start(s);
                    len = seg_len(s);
                }
                bnd[t] = seg_lower_bound(A.hub_arena + start, len, cbase + (w + 1) * W);
            }
        }
        // first entry of window w in run r
        auto edge = [&](uint32_t r, uint64_t start, uint32_t len, uint32_t w) -> uint32_t {
            if (w == 0) return 0u;
            if (w == nwin) return len;
            return table ? bnd[r * nb + w - 1] : seg_lower_bound(A.hub_arena + start, len, cbase + w * W);
        };
        // length of the run [b, e) of a segment (e is at most its length)
        auto run = [&](uint32_t b, uint32_t e) -> uint32_t {
            if (b > e) A.stt->bad = 1;
            return b > e ? 0u : e - b;
        };
        uint64_t my_start = 0;
        uint32_t my_len = 0;
        if (tid < deg) arc_run(tid, my_start, my_len);  // the first chunk of arcs stays in registers
        __syncthreads();

        // 1. pull and merge, window by window; candidates to the slab
        int M = 0;
        for (uint32_t w = 0; w < nwin; ++w) {
            const uint32_t w0 = cbase + w * W;
            if (ball) {
                const uint32_t row = (span + 31) / 32;  // words of the row over the ids below u
                for (uint32_t i = tid; i < kDenseWords && w * kDenseWords + i < row; i += NT)
                    mem[i] = __ldg(ball + w * kDenseWords + i);
            } else {  // members of L_<d(u) in the window
                const uint32_t e1 = edge((uint32_t)deg, seg_start(own1), seg_len(own1), w);
                const uint32_t e2 = edge((uint32_t)deg + 1, seg_start(own2), seg_len(own2), w);
                const uint32_t n1 = run(e1, edge((uint32_t)deg, seg_start(own1), seg_len(own1), w + 1));
                const uint32_t n2 = run(e2, edge((uint32_t)deg + 1, seg_start(own2), seg_len(own2), w + 1));
                const uint64_t s1 = seg_start(own1) + e1, s2 = seg_start(own2) + e2 - n1;
                for (uint32_t i = tid; i < n1 + n2; i += NT) {
                    const uint32_t x = (__ldg(A.hub_arena + (i < n1 ? s1 : s2) + i) & kHubMask) - w0;
                    if (x < W) atomicOr(&mem[x >> 5], 1u << (x & 31));
                    else A.stt->bad = 1;
                }
            }
            bool any = false;
            for (int c0 = 0; c0 < deg; c0 += NT) {
                const int nc = deg - c0 < NT ? deg - c0 : NT;
                uint64_t start = my_start;
                uint32_t len = my_len, b0 = 0, cnt = 0;
                if (tid < nc) {
                    if (c0 > 0) arc_run(c0 + tid, start, len);
                    if (len) {
                        b0 = edge((uint32_t)(c0 + tid), start, len, w);
                        cnt = run(b0, edge((uint32_t)(c0 + tid), start, len, w + 1));
                    }
                }
                if (c0 > 0) __syncthreads();  // pfx and st of the chunk before are still read
                const uint32_t total = dense_scan(cnt, nc, pfx, s_wsum);
                if (tid < nc) st[tid] = start + b0 - pfx[tid];
                __syncthreads();
                any |= total > 0;
                for (uint32_t cb = warp * 32 * kDenseUnroll; cb < total; cb += kWarps * 32 * kDenseUnroll) {
                    int lo = 0, hi = nc;  // last arc whose first entry is <= cb
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (pfx[mid] <= cb) lo = mid; else hi = mid;
                    }
                    int j = lo;
                    uint32_t off[kDenseUnroll], c[kDenseUnroll];
                    uint64_t pos[kDenseUnroll];
#pragma unroll
                    for (int t = 0; t < kDenseUnroll; ++t) {
                        const uint32_t i = cb + t * 32 + lane;
                        off[t] = kEmpty;
                        if (i < total) {
                            while (pfx[j + 1] <= i) ++j;
                            pos[t] = st[j] + i;
                            off[t] = (__ldg(A.hub_arena + pos[t]) & kHubMask) - w0;
                        }
                    }
#pragma unroll
                    for (int t = 0; t < kDenseUnroll; ++t) {
                        c[t] = 0;
                        if (off[t] < W && !((mem[off[t] >> 5] >> (off[t] & 31)) & 1u))
                            c[t] = __ldg((const uint32_t*)(A.cnt_arena + pos[t]));  // below 2^32: the low word
                    }
#pragma unroll
                    for (int t = 0; t < kDenseUnroll; ++t)
                        if (c[t]) atomicAdd(&acc[off[t]], c[t]);
                }
            }
            __syncthreads();
            if (any) {
                // the window in order: a warp owns a run of 128-id groups,
                // four ids a lane
                constexpr uint32_t kGroups = W / 128, kPer = (kGroups + kWarps - 1) / kWarps;
                const uint32_t g0 = warp * kPer, g1 = g0 + kPer < kGroups ? g0 + kPer : kGroups;
                int mine = 0;
                for (uint32_t g = g0; g < g1; ++g) {
                    const uint4 v = ((const uint4*)acc)[g * 32 + lane];
                    mine += (v.x != 0) + (v.y != 0) + (v.z != 0) + (v.w != 0);
                }
                mine = __reduce_add_sync(0xFFFFFFFFu, mine);
                if (lane == 0) s_wcnt[warp] = mine;
                for (uint32_t i = tid; i < kDenseWords; i += NT) mem[i] = 0u;
                __syncthreads();
                int at = M;
#pragma unroll
                for (int k = 0; k < kWarps; ++k) {
                    const int t = s_wcnt[k];
                    at += k < warp ? t : 0;
                    M += t;
                }
                if ((uint32_t)M > A.cap_c_max) {
                    if (tid == 0) A.stt->bad = 1;
                    M = 0;
                    dirty = W;
                    __syncthreads();
                    break;
                }
                for (uint32_t g = g0; mine > 0 && g < g1; ++g) {
                    const uint4 v = ((const uint4*)acc)[g * 32 + lane];
                    const unsigned bx = __ballot_sync(0xFFFFFFFFu, v.x != 0), by = __ballot_sync(0xFFFFFFFFu, v.y != 0);
                    const unsigned bz = __ballot_sync(0xFFFFFFFFu, v.z != 0), bw = __ballot_sync(0xFFFFFFFFu, v.w != 0);
                    if (!(bx | by | bz | bw)) continue;
                    int p = at + __popc(bx & lt) + __popc(by & lt) + __popc(bz & lt) + __popc(bw & lt);
                    const uint32_t h = w0 + g * 128 + lane * 4;
                    if (v.x) { shub[p] = h; scnt[p] = v.x; ++p; }
                    if (v.y) { shub[p] = h + 1; scnt[p] = v.y; ++p; }
                    if (v.z) { shub[p] = h + 2; scnt[p] = v.z; ++p; }
                    if (v.w) { shub[p] = h + 3; scnt[p] = v.w; ++p; }
                    ((uint4*)acc)[g * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
                    at += __popc(bx) + __popc(by) + __popc(bz) + __popc(bw);
                }
            } else {
                for (uint32_t i = tid; i < kDenseWords; i += NT) mem[i] = 0u;
            }
            __syncthreads();
        }

        // 2. rule 2. d = 3: a common neighbour x of u and h ranked above h
        // prunes h. The rows of u's higher-ranked neighbours (the first
        // |L_1(u)| arcs of its row) are walked and the ids met marked in a
        // bitmap over the counts' memory, 32 kDenseWindow ids at a time.
        bool listed = false;  // list[] holds the candidates (else all of the slab)
        if (d == 3 && M > 0 && !ball) {
            const int len1 = (int)seg_len(__ldg(A.seg + n + u));
            const uint32_t from0 = A.hpre ? (uint32_t)__ldg(A.hpre + u) : 0u;  // ids below are members, no candidates
            uint32_t* mk = acc;
            dirty = span > 32 * W ? W : (span + 31) / 32;
            int c_lo = 0;
            for (uint32_t m0 = cbase; m0 < (uint32_t)u; m0 += 32 * W) {
                const uint32_t m1 = (uint32_t)u - m0 > 32 * W ? m0 + 32 * W : (uint32_t)u;
                if (m0 > cbase) {
                    for (uint32_t i = tid; i < W; i += NT) mk[i] = 0u;
                    __syncthreads();
                }
                for (int c0 = 0; c0 < len1; c0 += NT) {
                    const int nc = len1 - c0 < NT ? len1 - c0 : NT;
                    uint32_t cnt = 0;
                    int64_t first = 0;
                    if (tid < nc) {
                        const uint32_t x = (uint32_t)__ldg(A.col + a0 + c0 + tid);
                        uint32_t from = x + 1;  // marks lie in [from, m1)
                        from = from0 > from ? from0 : from;
                        from = m0 > from ? m0 : from;
                        const int64_t r1 = A.rp[x + 1];
                        int64_t lo = A.rp[x], hi = r1;
                        while (lo < hi) {
                            const int64_t mid = (lo + hi) >> 1;
                            if ((uint32_t)__ldg(A.col + mid) < from) lo = mid + 1; else hi = mid;
                        }
                        first = lo;
                        hi = r1;
                        while (lo < hi) {
                            const int64_t mid = (lo + hi) >> 1;
                            if ((uint32_t)__ldg(A.col + mid) < m1) lo = mid + 1; else hi = mid;
                        }
                        cnt = (uint32_t)(lo - first);
                    }
                    if (c0 > 0 || m0 > cbase) __syncthreads();
                    const uint32_t total = dense_scan(cnt, nc, pfx, s_wsum);
                    if (tid < nc) st[tid] = (uint64_t)first - pfx[tid];
                    __syncthreads();
                    for (uint32_t cb = warp * 32 * kDenseUnroll; cb < total; cb += kWarps * 32 * kDenseUnroll) {
                        int lo = 0, hi = nc;
                        while (hi - lo > 1) {
                            const int mid = (lo + hi) >> 1;
                            if (pfx[mid] <= cb) lo = mid; else hi = mid;
                        }
                        int j = lo;
                        uint32_t x[kDenseUnroll];
#pragma unroll
                        for (int t = 0; t < kDenseUnroll; ++t) {
                            const uint32_t i = cb + t * 32 + lane;
                            x[t] = kEmpty;
                            if (i < total) {
                                while (pfx[j + 1] <= i) ++j;
                                x[t] = (uint32_t)__ldg(A.col + st[j] + i) - m0;
                            }
                        }
#pragma unroll
                        for (int t = 0; t < kDenseUnroll; ++t)
                            if (x[t] != kEmpty) {
                                const uint32_t bit = 1u << (x[t] & 31);
                                if (!(mk[x[t] >> 5] & bit)) atomicOr(&mk[x[t] >> 5], bit);
                            }
                    }
                }
                __syncthreads();
                // the slab is hub-sorted: this round's candidates are a run of it
                int c_hi = c_lo, top = M;
                while (c_hi < top) {
                    const int mid = (c_hi + top) >> 1;
                    if ((shub[mid] & kHubMask) < m1) c_hi = mid + 1; else top = mid;
                }
                for (int c = c_lo + tid; c < c_hi; c += NT) {
                    const uint32_t h = shub[c] - m0;
                    if ((mk[h >> 5] >> (h & 31)) & 1u) shub[c] |= kPrunedBit;
                }
                c_lo = c_hi;
                __syncthreads();
            }
        } else if (d > 3 && M > 0 && !ball) {
            // landmark filter, then the label scans of the undecided ones
            listed = true;
            for (int c = tid; c < M; c += NT) list[c] = (uint32_t)c;
            __syncthreads();
            int open = M;
            if (A.lmk) {
                if (A.lmk_words <= 4) landmark_filter<NT, 4>(A, s_lmk, d, list, shub, M, undecided, &s_lpr, &s_lpv, &s_open);
                else landmark_filter<NT, 8>(A, s_lmk, d, list, shub, M, undecided, &s_lpr, &s_lpv, &s_open);
                __syncthreads();
                open = s_open;
                if (tid == 0 && s_lpr) atomicAdd(&A.stt->lmk_pruned, (unsigned long long)s_lpr);
                if (tid == 0 && s_lpv) atomicAdd(&A.stt->lmk_proven, (unsigned long long)s_lpv);
            }
            if (open > 0) {
                SegMap sm;
                sm.seg = A.seg;
                sm.hub_arena = A.hub_arena;
                sm.n = n;
                sm.u = u;
                sm.d = d;
                sm.cache = nullptr;
                sm.cwords = 0;
                sm.base = cbase;
                // u's levels on chip over the first ids, in the counts' memory
                // (all zero after the last window)
                uint32_t cw = W / (uint32_t)(d - 1);
                cw = cw < kSegCacheMaxWords ? cw : kSegCacheMaxWords;
                if (cw >= kSegCacheMinWords) {
                    for (int l = 1; l < d; ++l) {
                        const uint64_t s = __ldg(A.seg + (int64_t)l * n + u);
                        const uint32_t len = seg_len(s);
                        const uint32_t* hs = A.hub_arena + seg_start(s);
                        for (uint32_t i = tid; i < len; i += NT) {
                            const uint32_t r = (__ldg(hs + i) & kHubMask) - cbase;
                            if (r >= 32u * cw) break;
                            atomicOr(&acc[(uint32_t)(l - 1) * cw + (r >> 5)], 1u << (r & 31));
                        }
                    }
                    dirty = (uint32_t)(d - 1) * cw;
                    sm.cache = acc;
                    sm.cwords = cw;
                } else {
                    dirty = kWarps * (kDeepFilter + kScanHits);  // the split scan's filters
                }
                const bool useg_on = d - 2 < kUSideLevels;
                if (useg_on && tid < d - 1) s_useg[tid] = __ldg(A.seg + (int64_t)tid * n + u);
                __syncthreads();
                prune_all<NT>(sm, A.seg, A.hub_arena, n, d, list, shub, A.lmk ? undecided : nullptr, M, open,
                              &s_next, useg_on ? s_useg : nullptr, s_wcnt, sm.cache ? nullptr : acc, u);
                __syncthreads();
            }
        }

        // 3. survivors, in hub order, appended as L_d(u): each warp owns a
        // run of the candidates
        const int per = ((M + kWarps - 1) / kWarps + 31) & ~31;
        const int c0 = warp * per, c1 = c0 + per < M ? c0 + per : M;
        int mine = 0;
        for (int c = c0 + lane; c < c1; c += 32) mine += !((listed ? list[c] : shub[c]) & kPrunedBit);
        mine = __reduce_add_sync(0xFFFFFFFFu, mine);
        if (lane == 0) s_wcnt[warp] = mine;
        __syncthreads();
        int S = 0, at = 0;
#pragma unroll
        for (int k = 0; k < kWarps; ++k) {
            const int t = s_wcnt[k];
            at += k < warp ? t : 0;
            S += t;
        }
        if (S > 0) {
            if (tid == 0) {
                s_base = atomicAdd(&A.stt->bump, (unsigned long long)S);
                if (s_base + S > A.arena_cap) atomicOr(&A.stt->arena_overflow, 1);
            }
            __syncthreads();
            const unsigned long long b0 = s_base;
            if (b0 + S <= A.arena_cap) {
                for (int c = c0; c < c1; c += 32) {
                    const bool in = c + lane < c1;
                    const uint32_t e = in ? (listed ? list[c + lane] : shub[c + lane]) : kPrunedBit;
                    const bool keep = !(e & kPrunedBit);
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, keep);
                    if (keep) {
                        const uint32_t slot = listed ? e & kSlotMask : (uint32_t)(c + lane);
                        const uint32_t cv = scnt[slot];
                        A.hub_arena[b0 + at + __popc(m & lt)] = listed ? shub[slot] : e;
                        A.cnt_arena[b0 + at + __popc(m & lt)] = cv;
                        cm = cv > cm ? cv : cm;
                    }
                    at += __popc(m);
                }
                if (tid == 0) A.seg_out[u] = seg_pack(b0, (uint32_t)S);
            }
        }
        if (tid == 0) atomicAdd(&A.stt->unique_total, (unsigned long long)M);
        __syncthreads();
    }
    cm = __reduce_max_sync(0xFFFFFFFFu, cm);
    if (lane == 0 && cm) atomicMax(&A.stt->cmax, cm);
}
