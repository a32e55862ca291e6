// Distance balls as bit rows: row u of ball t has a bit for every vertex of
// u's graph within distance t of u. With ball d-1 rule 2 at level d is one
// bit: a candidate (u, h) is pruned exactly when sd(u,h) < d, and the hubs of
// L_<d(u) are in the ball too, so a pulled entry whose hub is there is dropped
// before its count is read and every other one survives.
//
// Ball t+1 of u is the OR of its neighbours' balls t: (arcs + 2n) rows of n/8
// bytes a level, whatever the labels hold. That pays where candidates are
// many for the size of the graph; the level loop compares the two
// (Builder::use_ball). What bounds a step: reads of neighbours' rows from L2
// (16 GB in 1.25 ms on R-MAT 65,536, edge factor 16; 22 GB in 2.7 ms on BA
// 100,000, m = 8). Builds with it: BA 100,000 167 -> 56 ms (m = 8) and 56 -> 25
// (m = 3), BA 20,011 6.7 -> 3.6, 96 BA graphs of 500 to 20,000 in a batch 230 ->
// 109, R-MAT 65,536 12.4 -> 11.0.
#include <cuda_runtime.h>
#include <stdint.h>

#include "pspc_level.cuh"

namespace pspc {

constexpr int kBallThreads = 256;
constexpr int kBallSlice = 128;      // neighbours one warp ORs; longer rows are split
constexpr int kBallSegment = 128;    // words of a row one warp owns (16 bytes a lane)
constexpr int kBallUnroll = 4;

__device__ __forceinline__ int64_t ball_row(const BallRows& R, int64_t u) {
    return R.off ? __ldg(R.off + u) : u * R.words;
}

// Ball 1: u and its neighbours.
__global__ void k_ball_init(int64_t n, int64_t arcs, const int32_t* __restrict__ arc_src, const int32_t* __restrict__ col,
                            const int32_t* __restrict__ comp_base, const BallRows R, uint32_t* __restrict__ ball) {
    const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= n + arcs) return;
    const int64_t u = a < n ? a : arc_src[a - n];
    const uint32_t v = a < n ? (uint32_t)a : (uint32_t)col[a - n];
    const uint32_t r = v - (comp_base ? (uint32_t)comp_base[u] : 0u);
    atomicOr(ball + ball_row(R, u) + (r >> 5), 1u << (r & 31));
}

// The slices beyond the first of rows with more than kBallSlice arcs.
__global__ void k_ball_slices(int64_t n, const int64_t* __restrict__ rp, int2* __restrict__ slices, int* __restrict__ count) {
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= n) return;
    const int64_t deg = rp[u + 1] - rp[u];
    for (int64_t s = 1; s * kBallSlice < deg; ++s) slices[atomicAdd(count, 1)] = make_int2((int)u, (int)s);
}

// One step for one segment (blockIdx.y, the slow index, so that a segment's
// column of all rows stays in L2): a warp per vertex ORs the segment over the
// first kBallSlice neighbours and the vertex itself (slices NULL), or over one
// more slice of a long row into what the first launch wrote.
__global__ void __launch_bounds__(kBallThreads)
    k_ball_step(int64_t items, const int64_t* __restrict__ rp, const int32_t* __restrict__ col, const BallRows R,
                const int2* __restrict__ slices, const uint32_t* __restrict__ from, uint32_t* __restrict__ to) {
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    const int64_t item = ((int64_t)blockIdx.x * kBallThreads + threadIdx.x) >> 5;
    if (item >= items) return;  // the whole warp
    const int64_t u = slices ? slices[item].x : item;
    const int64_t row = ball_row(R, u);
    const int64_t words = R.off ? __ldg(R.off + u + 1) - row : R.words;  // a multiple of 4
    const int64_t at = (int64_t)blockIdx.y * kBallSegment + lane * 4;
    if ((int64_t)blockIdx.y * kBallSegment >= words) return;
    const bool in = at < words;
    // rows of one graph are as long and as far apart as u's
    const int64_t base = R.off ? row - u * words : 0;
    const int64_t a0 = rp[u] + (slices ? (int64_t)slices[item].y * kBallSlice : 0);
    const int64_t a1 = rp[u + 1] - a0 < kBallSlice ? rp[u + 1] : a0 + kBallSlice;
    uint4 acc = make_uint4(0u, 0u, 0u, 0u);
    if (in && !slices) acc = __ldg((const uint4*)(from + row + at));
    for (int64_t ca = a0; ca < a1; ca += 32) {
        const int nc = (int)(a1 - ca < 32 ? a1 - ca : 32);
        const int32_t v = lane < nc ? __ldg(col + ca + lane) : 0;
        for (int i = 0; i < nc; i += kBallUnroll) {
            uint4 x[kBallUnroll];
#pragma unroll
            for (int k = 0; k < kBallUnroll; ++k) {
                const int64_t w = __shfl_sync(FULL, v, i + k < nc ? i + k : nc - 1);
                x[k] = in ? __ldg((const uint4*)(from + base + w * words + at)) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int k = 0; k < kBallUnroll; ++k) {
                acc.x |= x[k].x;
                acc.y |= x[k].y;
                acc.z |= x[k].z;
                acc.w |= x[k].w;
            }
        }
    }
    if (!in) return;
    if (!slices) {
        *(uint4*)(to + row + at) = acc;
    } else {
        atomicOr(to + row + at, acc.x);
        atomicOr(to + row + at + 1, acc.y);
        atomicOr(to + row + at + 2, acc.z);
        atomicOr(to + row + at + 3, acc.w);
    }
}

cudaError_t launch_ball_init(int64_t n, int64_t arcs, const int64_t* rp, const int32_t* arc_src, const int32_t* col,
                             const int32_t* comp_base, const BallRows& R, int64_t total_words, uint32_t* ball, int2* slices,
                             int* n_slices, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(ball, 0, (size_t)total_words * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(n_slices, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    k_ball_init<<<(unsigned)((n + arcs + 255) / 256), 256, 0, st>>>(n, arcs, arc_src, col, comp_base, R, ball);
    k_ball_slices<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, rp, slices, n_slices);
    return cudaGetLastError();
}

cudaError_t launch_ball_step(int64_t n, const int64_t* rp, const int32_t* col, const BallRows& R, int64_t max_words,
                             const int2* slices, int n_slices, const uint32_t* from, uint32_t* to, cudaStream_t st) {
    const unsigned segments = (unsigned)((max_words + kBallSegment - 1) / kBallSegment);
    const int per = kBallThreads / 32;
    k_ball_step<<<dim3((unsigned)((n + per - 1) / per), segments), kBallThreads, 0, st>>>(n, rp, col, R, nullptr, from, to);
    if (n_slices > 0)
        k_ball_step<<<dim3((unsigned)((n_slices + per - 1) / per), segments), kBallThreads, 0, st>>>(n_slices, rp, col, R,
                                                                                                    slices, from, to);
    return cudaGetLastError();
}

}  // namespace pspc
