// Graph diffusion over the Gaussians (Sec. 3.3): exact kNN of the centres,
// the union edge set with similarity weights (Eq. 7 / the diffusion
// workload's spatial x cosine weight), and the power iteration of Eq. 8.
//
// kNN: points are bucketed in a uniform grid (cells sorted by the radix sort);
// one thread per query scans the 27 cells around its own, then ring by ring
// (Chebyshev distance r), and stops once the k-th best squared distance is below
// the squared gap r*cell to the unvisited rings.  A query whose neighbours lie
// more than a few rings away goes on by itself in a warp, by blocks of 8x8x8
// cells (k_knn_far).  Squared distances are float32
// (dx*dx + dy*dy) + dz*dz with d = x_j - x_i and ties go to the lower index,
// so the result is exact and independent of the scan order.
//
// Graph: own neighbours plus reverse edges per row, one warp sorts and
// de-duplicates each row, then weights are computed per edge from the two
// feature rows (once per pair) and optionally thresholded and row-normalised.
//
// Diffusion: one kernel per step computes y = A x * (1/||x||) row by row and
// accumulates ||y||^2 (float64) for the next step's scaling.
#include <algorithm>
#include <cfloat>
#include <cstring>
#include <mutex>
#include <vector>

#include "common.cuh"

namespace ludvig {

namespace {

unsigned grid_for(int64_t work, int threads) { return (unsigned)ceil_div(work, threads); }

// ------------------------------------------------------------ bounding box
__global__ void k_bbox(const float* __restrict__ x, int64_t n, float* __restrict__ out6) {
    float lo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, hi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = fminf(lo[a], x[3 * i + a]);
            hi[a] = fmaxf(hi[a], x[3 * i + a]);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
            hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
        }
    }
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            // order-preserving integer encoding of floats for atomicMin/Max
            const int l = __float_as_int(lo[a]), h = __float_as_int(hi[a]);
            atomicMin(reinterpret_cast<int*>(out6) + a, l >= 0 ? l : l ^ 0x7fffffff);
            atomicMax(reinterpret_cast<int*>(out6) + 3 + a, h >= 0 ? h : h ^ 0x7fffffff);
        }
    }
}

struct Grid {
    float lo[3];
    float cell;
    float inv_cell;
    int g[3];
};

__device__ __forceinline__ int cell_coord(float x, float lo, float inv, int g) {
    int c = (int)floorf((x - lo) * inv);
    return c < 0 ? 0 : (c >= g ? g - 1 : c);
}

// How many points lie in each cell, and the sum of the squares of the counts.
__global__ void k_cell_count(const float* __restrict__ x, int64_t n, Grid gr, uint32_t* __restrict__ cnt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int cx = cell_coord(x[3 * i], gr.lo[0], gr.inv_cell, gr.g[0]);
    const int cy = cell_coord(x[3 * i + 1], gr.lo[1], gr.inv_cell, gr.g[1]);
    const int cz = cell_coord(x[3 * i + 2], gr.lo[2], gr.inv_cell, gr.g[2]);
    atomicAdd(&cnt[((int64_t)cz * gr.g[1] + cy) * gr.g[0] + cx], 1u);
}

__global__ void k_cell_square(const uint32_t* __restrict__ cnt, int64_t nc, unsigned long long* __restrict__ sum) {
    unsigned long long s = 0;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += (int64_t)gridDim.x * blockDim.x)
        s += (unsigned long long)cnt[c] * cnt[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(sum, s);
}

constexpr double kKnnCellPoints = 6.0;       // points a point should find in its cell
constexpr int64_t kKnnDensityMin = 1 << 14;  // below, the pass over the counts costs more than it saves
// Rings a thread searches by itself: most points are done after two or three of
// them, and a wider search is a chain of reads that its warp waits for.  Limits of
// 4, 6, 8 and 12 (ms, k = 16): 100k clustered centres 0.84, 0.65, 0.66, 0.66, 200 of them
// moved far out 1.24, 1.25, 1.44, 2.75; 1M centres, a tenth of them in a wide
// shell, 9.4, 8.5, 7.9, 7.8.
constexpr int kKnnNear = 8;
constexpr int kKnnBlock = 8;                 // cells along each axis of a block of cells

__global__ void k_cell_keys(const float* __restrict__ x, int64_t n, int64_t npad, Grid gr,
                            uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npad) return;
    if (i >= n) {
        keys[i] = 0xffffffffu;
        vals[i] = 0xffffffffu;
        return;
    }
    const int cx = cell_coord(x[3 * i], gr.lo[0], gr.inv_cell, gr.g[0]);
    const int cy = cell_coord(x[3 * i + 1], gr.lo[1], gr.inv_cell, gr.g[1]);
    const int cz = cell_coord(x[3 * i + 2], gr.lo[2], gr.inv_cell, gr.g[2]);
    keys[i] = (uint32_t)(((int64_t)cz * gr.g[1] + cy) * gr.g[0] + cx);
    vals[i] = (uint32_t)i;
}

// Points sorted by cell are stored as float4 (x, y, z, index) in cell order.
__global__ void k_gather_sorted(const float* __restrict__ x, const uint32_t* __restrict__ order,
                                int64_t n, float4* __restrict__ pts) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const uint32_t i = order[j];
    pts[j] = make_float4(x[3 * i], x[3 * i + 1], x[3 * i + 2], __uint_as_float(i));
}

// One thread per query, in cell order.  The block of cells within distance 1 is
// scanned first (9 runs along x), then ring after ring (full runs on the ring's
// z and y faces, one cell at either end elsewhere).  Bound by instruction issue
// (a warp inserts whenever one of its lanes does).  1M clustered centres, k = 16:
// 3.54 -> 2.3 ms with smaller cells, runs of cells and 64-bit (distance, index) keys.
// (0: no bound; one block per SM as the bound takes more registers and 0.2 ms more.)
// Four blocks per SM for K = 32 (the compiler takes three otherwise): 100k clustered
// centres, k = 32, 1.21 -> 1.11 ms.
template <int K>
__device__ __forceinline__ void knn_insert(uint64_t (&best)[K], uint64_t key) {
#pragma unroll
    for (int t = 0; t < K; ++t) {
        const uint64_t lo = key < best[t] ? key : best[t];
        key = key < best[t] ? best[t] : key;
        best[t] = lo;
    }
}

template <int K>
__global__ void __launch_bounds__(128, K <= 16 ? 0 : K <= 32 ? 4 : 2) k_knn(const float4* __restrict__ pts, int64_t n, Grid gr,
                                             const uint32_t* __restrict__ start, int k,
                                             int32_t* __restrict__ out, uint32_t* __restrict__ far,
                                             uint32_t* __restrict__ nfar) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const float4 q = pts[j];
    const uint32_t qi = __float_as_uint(q.w);
    if (!(isfinite(q.x) && isfinite(q.y) && isfinite(q.z))) {   // at no finite distance from any point
        for (int t = 0; t < k; ++t) out[(int64_t)qi * k + t] = -1;
        return;
    }
    // the best so far, ascending: squared distance (its bits order like the
    // value), then index; K - k entries that nothing precedes fill the list up,
    // so that the k-th best is always the last
    constexpr uint64_t kNone = ~0ull;
    uint64_t best[K];
#pragma unroll
    for (int t = 0; t < K; ++t) best[t] = t < K - k ? 0ull : kNone;
    const int cx = cell_coord(q.x, gr.lo[0], gr.inv_cell, gr.g[0]);
    const int cy = cell_coord(q.y, gr.lo[1], gr.inv_cell, gr.g[1]);
    const int cz = cell_coord(q.z, gr.lo[2], gr.inv_cell, gr.g[2]);
    const int rmax = max(gr.g[0], max(gr.g[1], gr.g[2]));
    bool found = rmax <= kKnnNear;   // (the last ring ends that search)
    for (int r = 1; r <= min(max(1, rmax), kKnnNear); ++r) {
        for (int dz = -r; dz <= r; ++dz) {
            const int z = cz + dz;
            if (z < 0 || z >= gr.g[2]) continue;
            for (int dy = -r; dy <= r; ++dy) {
                const int y = cy + dy;
                if (y < 0 || y >= gr.g[1]) continue;
                const uint32_t* row = start + ((int64_t)z * gr.g[1] + y) * gr.g[0];
                const bool full = r == 1 || dz == -r || dz == r || dy == -r || dy == r;
                // cells cx - r .. cx + r, or cx - r and then cx + r
                for (int side = 0; side < (full ? 1 : 2); ++side) {
                    const int xa = max(side ? cx + r : cx - r, 0);
                    const int xb = min(full || side ? cx + r : cx - r, gr.g[0] - 1);
                    if (xa > xb) continue;
                    const uint32_t e = row[xb + 1];
                    for (uint32_t p = row[xa]; p < e; ++p) {
                        const float4 c = pts[p];
                        const uint32_t ci = __float_as_uint(c.w);
                        if (ci == qi) continue;
                        const float ex = __fsub_rn(c.x, q.x), ey = __fsub_rn(c.y, q.y), ez = __fsub_rn(c.z, q.z);
                        const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
                        // (a distance that is not a number, or overflowed, is no neighbour's)
                        const uint64_t key = ((uint64_t)__float_as_uint(d2) << 32) | ci;
                        if (key < best[K - 1] && d2 <= FLT_MAX) knn_insert(best, key);
                    }
                }
            }
        }
        // every point outside the visited (2r+1)^3 block is at least r cells away
        const uint64_t kth = best[K - 1];
        const float gap = (float)r * gr.cell;
        // 0.1% margin: rounding can put a point next to a cell border in the neighbour cell
        if (kth != kNone && __uint_as_float((uint32_t)(kth >> 32)) < gap * gap * 0.999f) {
            found = true;
            break;
        }
    }
    if (!found) {   // (k_knn_far starts afresh)
        far[atomicAdd(nfar, 1u)] = (uint32_t)j;
        return;
    }
#pragma unroll
    for (int t = 0; t < K; ++t)
        if (t >= K - k) out[(int64_t)qi * k + (t - (K - k))] = best[t] == kNone ? -1 : (int32_t)(uint32_t)best[t];
}

// ---- queries far from their neighbours
// The points in every block of 8x8x8 cells (bg blocks along each axis).
__global__ void k_block_count(const uint32_t* __restrict__ start, Grid gr, int3 bg, int64_t nblocks,
                              const uint32_t* __restrict__ nfar, uint32_t* __restrict__ cnt) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nblocks || *nfar == 0u) return;
    const int bx = (int)(t % bg.x), by = (int)(t / bg.x % bg.y), bz = (int)(t / bg.x / bg.y);
    const int x0 = bx * kKnnBlock, x1 = min(x0 + kKnnBlock, gr.g[0]);
    uint32_t c = 0;
    for (int z = bz * kKnnBlock; z < min((bz + 1) * kKnnBlock, gr.g[2]); ++z)
        for (int y = by * kKnnBlock; y < min((by + 1) * kKnnBlock, gr.g[1]); ++y) {
            const uint32_t* row = start + ((int64_t)z * gr.g[1] + y) * gr.g[0];
            c += row[x1] - row[x0];
        }
    cnt[t] = c;
}

// One warp per query of the list `far`, its k best so far in ascending order
// over the lanes (entry t is list[t / 32] of lane t % 32).  The blocks of cells
// are visited in Chebyshev rings around the query's own (ring R's six faces, 32
// blocks at a time); empty ones, and those further away than the k-th best, cost
// their share of one read, the others are scanned by the whole warp.  Bound by
// the latency of those reads.  The whole search, k = 16: 100k clustered centres of
// which 8 lie far out 1.7 ms, 1M 23.6 (2490 and 3020 with one thread walking all rings
// of cells); 200 of them anywhere in a wide box 1.4 and 8.3 (431 and 1170).
template <int P>
__global__ void __launch_bounds__(128) k_knn_far(const float4* __restrict__ pts, Grid gr,
                                                 const uint32_t* __restrict__ start, int3 bg,
                                                 const uint32_t* __restrict__ bcnt, int k,
                                                 const uint32_t* __restrict__ far, const uint32_t* __restrict__ nfar,
                                                 int32_t* __restrict__ out) {
    constexpr uint32_t kAll = 0xffffffffu;
    constexpr uint64_t kNone = ~0ull;
    const int lane = threadIdx.x & 31;
    const uint32_t nq = *nfar, nwarps = gridDim.x * (blockDim.x >> 5);
    // cells by which a coordinate divided by the cell's size may be off, twice (the
    // query's and the point's)
    const float slack = 0.01f + 1e-6f * (float)max(gr.g[0], max(gr.g[1], gr.g[2]));
    for (uint32_t w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); w < nq; w += nwarps) {
        const float4 q = pts[far[w]];
        const uint32_t qi = __float_as_uint(q.w);
        const float u[3] = {(q.x - gr.lo[0]) * gr.inv_cell, (q.y - gr.lo[1]) * gr.inv_cell,
                            (q.z - gr.lo[2]) * gr.inv_cell};
        const int b[3] = {cell_coord(q.x, gr.lo[0], gr.inv_cell, gr.g[0]) / kKnnBlock,
                          cell_coord(q.y, gr.lo[1], gr.inv_cell, gr.g[1]) / kKnnBlock,
                          cell_coord(q.z, gr.lo[2], gr.inv_cell, gr.g[2]) / kKnnBlock};
        uint64_t list[P], kth = kNone;
#pragma unroll
        for (int e = 0; e < P; ++e) list[e] = kNone;
        auto kth_dist = [&]() { return __uint_as_float((uint32_t)(kth >> 32)); };
        auto insert = [&](uint64_t key) {
            uint64_t below = 0ull;   // the entry before lane 0's
#pragma unroll
            for (int e = 0; e < P; ++e) {
                uint64_t left = __shfl_up_sync(kAll, list[e], 1);
                const uint64_t last = __shfl_sync(kAll, list[e], 31);
                if (lane == 0) left = below;
                below = last;
                list[e] = key < list[e] ? (key > left ? key : left) : list[e];
            }
#pragma unroll
            for (int e = 0; e < P; ++e)
                if ((k - 1) / 32 == e) kth = __shfl_sync(kAll, list[e], (k - 1) & 31);
        };
        // could the block at (x, y, z) hold one of the k?
        auto reaches = [&](int x, int y, int z) {
            const int c[3] = {x, y, z};
            float d2 = 0.f;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float l = (float)(c[a] * kKnnBlock);
                const float t = fmaxf(fmaxf(l - u[a], u[a] - (l + (float)kKnnBlock)) - slack, 0.f) * gr.cell;
                d2 += t * t;
            }
            return kth == kNone || d2 * 0.999f <= kth_dist();
        };
        auto scan_block = [&](int x, int y, int z) {
            const int x0 = x * kKnnBlock, x1 = min(x0 + kKnnBlock, gr.g[0]);
#pragma unroll 1
            for (int h = 0; h < kKnnBlock * kKnnBlock; h += 32) {
                const int ry = y * kKnnBlock + ((h + lane) & (kKnnBlock - 1)), rz = z * kKnnBlock + (h + lane) / kKnnBlock;
                uint32_t p0 = 0u, p1 = 0u;
                if (ry < gr.g[1] && rz < gr.g[2]) {
                    const uint32_t* row = start + ((int64_t)rz * gr.g[1] + ry) * gr.g[0];
                    p0 = row[x0];
                    p1 = row[x1];
                }
                for (uint32_t m = __ballot_sync(kAll, p1 > p0); m; m &= m - 1u) {
                    const int src = __ffs(m) - 1;
                    const uint32_t s0 = __shfl_sync(kAll, p0, src), s1 = __shfl_sync(kAll, p1, src);
                    for (uint32_t s = s0; s < s1; s += 32) {
                        uint64_t key = kNone;
                        if (s + lane < s1) {
                            const float4 c = pts[s + lane];
                            const uint32_t ci = __float_as_uint(c.w);
                            const float ex = __fsub_rn(c.x, q.x), ey = __fsub_rn(c.y, q.y), ez = __fsub_rn(c.z, q.z);
                            const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
                            if (ci != qi && d2 <= FLT_MAX) key = ((uint64_t)__float_as_uint(d2) << 32) | ci;
                        }
                        for (uint32_t c = __ballot_sync(kAll, key < kth); c; c &= c - 1u) {
                            const uint64_t kk = __shfl_sync(kAll, key, __ffs(c) - 1);
                            if (kk < kth) insert(kk);
                        }
                    }
                }
            }
        };
        const int rmax = max(max(max(b[0], bg.x - 1 - b[0]), max(b[1], bg.y - 1 - b[1])), max(b[2], bg.z - 1 - b[2]));
        for (int r = 0; r <= rmax; ++r) {
            const int xl = max(b[0] - r, 0), xh = min(b[0] + r, bg.x - 1);
            const int yl = max(b[1] - r, 0), yh = min(b[1] + r, bg.y - 1);
            const int yi = max(b[1] - r + 1, 0), yj = min(b[1] + r - 1, bg.y - 1);
            const int zi = max(b[2] - r + 1, 0), zj = min(b[2] + r - 1, bg.z - 1);
#pragma unroll 1
            for (int f = 0; f < (r == 0 ? 1 : 6); ++f) {
                // the faces across z whole, those across y without the first, those across x without both
                const int axis = 2 - (f >> 1), at = b[axis] + ((f & 1) ? r : -r);
                if (at < 0 || at >= (axis == 0 ? bg.x : axis == 1 ? bg.y : bg.z)) continue;
                const int x0 = axis == 0 ? at : xl, nx = axis == 0 ? 1 : xh - xl + 1;
                const int y0 = axis == 1 ? at : axis == 0 ? yi : yl, ny = axis == 1 ? 1 : axis == 0 ? yj - yi + 1 : yh - yl + 1;
                const int z0 = axis == 2 ? at : zi, nz = axis == 2 ? 1 : zj - zi + 1;
                if (nx <= 0 || ny <= 0 || nz <= 0) continue;
                const int total = nx * ny * nz;   // (a grid has at most 2^24 cells)
                for (int t0 = 0; t0 < total; t0 += 32) {
                    const int t = t0 + lane, line = t / nx;
                    const int x = x0 + t - line * nx, y = y0 + line % ny, z = z0 + line / ny;
                    const bool in = t < total && bcnt[((int64_t)z * bg.y + y) * bg.x + x] > 0u && reaches(x, y, z);
                    for (uint32_t m = __ballot_sync(kAll, in); m; m &= m - 1u) {
                        const int src = __ffs(m) - 1;
                        const int sx = __shfl_sync(kAll, x, src), sy = __shfl_sync(kAll, y, src),
                                  sz = __shfl_sync(kAll, z, src);
                        if (reaches(sx, sy, sz)) scan_block(sx, sy, sz);   // (the k-th best may have come nearer)
                    }
                }
            }
            // every point outside the visited blocks is at least r blocks away
            const float gap = fmaxf((float)(r * kKnnBlock) - slack, 0.f) * gr.cell;
            if (kth != kNone && kth_dist() < gap * gap * 0.999f) break;
        }
#pragma unroll
        for (int e = 0; e < P; ++e)
            if (32 * e + lane < k)
                out[(int64_t)qi * k + 32 * e + lane] = list[e] == kNone ? -1 : (int32_t)(uint32_t)list[e];
    }
}

// ------------------------------------------------------------ graph build
__global__ void k_own_and_indegree(const int32_t* __restrict__ nbr, int64_t n, int k,
                                   uint32_t* __restrict__ own, uint32_t* __restrict__ indeg) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t c = 0;
    for (int t = 0; t < k; ++t) {
        const int32_t j = nbr[i * k + t];
        if (j >= 0 && j != i) {
            ++c;
            atomicAdd(&indeg[j], 1u);
        }
    }
    own[i] = c;
}

__global__ void k_row_counts(const uint32_t* __restrict__ own, const uint32_t* __restrict__ indeg,
                             int64_t n, uint32_t* __restrict__ cnt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) cnt[i] = own[i] + indeg[i];
}

__global__ void k_fill_rows(const int32_t* __restrict__ nbr, int64_t n, int k,
                            const uint32_t* __restrict__ ptr, const uint32_t* __restrict__ own,
                            uint32_t* __restrict__ cursor, uint32_t* __restrict__ tcol) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t o = ptr[i];
    for (int t = 0; t < k; ++t) {
        const int32_t j = nbr[i * k + t];
        if (j >= 0 && j != i) {
            tcol[o++] = (uint32_t)j;
            const uint32_t pos = atomicAdd(&cursor[j], 1u);
            tcol[ptr[j] + own[j] + pos] = (uint32_t)i;
        }
    }
}

// One warp per row: sort the row's column indices (insertion sort through
// shared memory for short rows, a serial heap sort in place for long ones),
// then count the distinct values.
constexpr int kRowSmem = 256;
__global__ void __launch_bounds__(256) k_sort_unique_rows(uint32_t* __restrict__ tcol,
                                                         const uint32_t* __restrict__ ptr,
                                                         const uint32_t* __restrict__ cnt, int64_t n,
                                                         uint32_t* __restrict__ ucnt) {
    __shared__ uint32_t buf[8][kRowSmem];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 8 + warp;
    if (i >= n) return;
    uint32_t* row = tcol + ptr[i];
    const uint32_t c = cnt[i];
    uint32_t* b = buf[warp];
    if (c <= kRowSmem) {
        for (uint32_t t = lane; t < c; t += 32) b[t] = row[t];
        __syncwarp();
        // rank sort: each element's position = number of smaller elements
        // (+ equal elements before it), which is a stable sort of the row
        for (uint32_t t = lane; t < c; t += 32) {
            const uint32_t v = b[t];
            uint32_t pos = 0;
            for (uint32_t u = 0; u < c; ++u) {
                const uint32_t w = b[u];
                pos += (w < v) || (w == v && u < t);
            }
            row[pos] = v;
        }
        __syncwarp();
    } else if (lane == 0) {
        // heap sort in place
        auto sift = [&](uint32_t start, uint32_t end) {
            uint32_t root = start;
            while (2 * root + 1 < end) {
                uint32_t child = 2 * root + 1;
                if (child + 1 < end && row[child] < row[child + 1]) ++child;
                if (row[root] < row[child]) {
                    const uint32_t t = row[root];
                    row[root] = row[child];
                    row[child] = t;
                    root = child;
                } else {
                    break;
                }
            }
        };
        for (int64_t s = (int64_t)c / 2 - 1; s >= 0; --s) sift((uint32_t)s, c);
        for (uint32_t e = c - 1; e > 0; --e) {
            const uint32_t t = row[0];
            row[0] = row[e];
            row[e] = t;
            sift(0, e);
        }
    }
    __syncwarp();
    uint32_t u = 0;
    for (uint32_t t = lane; t < c; t += 32) u += (t == 0 || row[t] != row[t - 1]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
    if (lane == 0) ucnt[i] = u;
}

__global__ void k_norms(const float* __restrict__ f, int64_t n, int df, float* __restrict__ nrm) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    if (i >= n) return;
    float s = 0.f;
    for (int c = lane; c < df; c += 32) {
        const float v = f[i * df + c];
        s = fmaf(v, v, s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) nrm[i] = sqrtf(s);
}

// Edge value modes: the diffusion workload's spatial x cosine weight, or the
// squared distance ||f^_i - f^_j||^2 of the l2-normalised features (for the
// RBF similarity of the appendix; a zero feature vector normalises to zero):
// 2 - 2 cos for two non-zero rows, 1 with one zero row, 0 with two.
constexpr int kEdgeSpatialCos = 0, kEdgeFeatureDist2 = 1;

__device__ __forceinline__ float feature_dist2(float ni, float nj, float cs) {
    const float zi = ni > 0.f ? 1.f : 0.f, zj = nj > 0.f ? 1.f : 0.f;
    return fmaxf(0.f, zi + zj - 2.f * cs);
}

// One warp per row: compact the distinct columns, weight every edge, then
// threshold / normalise the row (any df).  Row r of the launch is Gaussian
// order[r] (Morton order, so that neighbours' feature rows stay in L2), or
// r when order is null.
__global__ void __launch_bounds__(256) k_edge_weights_any(const uint32_t* __restrict__ tcol,
                                                const uint32_t* __restrict__ tptr,
                                                const uint32_t* __restrict__ tcnt,
                                                const int64_t* __restrict__ row_ptr,
                                                const float* __restrict__ x, const float* __restrict__ f,
                                                const float* __restrict__ nrm, int64_t n, int df,
                                                float inv_h, float binarize, int row_normalize,
                                                const uint32_t* __restrict__ order, int mode,
                                                int32_t* __restrict__ col, float* __restrict__ val) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * 8 + warp;
    if (r >= n) return;
    const int64_t i = order ? (int64_t)order[r] : r;
    const uint32_t* row = tcol + tptr[i];
    const uint32_t c = tcnt[i];
    const int64_t o0 = row_ptr[i];
    const float xi = x[3 * i], yi = x[3 * i + 1], zi = x[3 * i + 2];
    const float ni = nrm[i];
    const float* fi = f + i * df;
    int64_t o = o0;
    float rsum = 0.f;
    for (uint32_t t = 0; t < c; ++t) {
        const uint32_t j = row[t];
        if (t > 0 && row[t - 1] == j) continue;   // duplicate (mutual neighbours)
        float dot = 0.f;
        const float* fj = f + (int64_t)j * df;
        for (int ch = lane; ch < df; ch += 32) dot = fmaf(fi[ch], fj[ch], dot);
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, s);
        if (lane == 0) {
            const float ex = x[3 * j] - xi, ey = x[3 * j + 1] - yi, ez = x[3 * j + 2] - zi;
            const float d2 = ex * ex + ey * ey + ez * ez;
            const float den = ni * nrm[j];
            const float cs = den > 0.f ? dot / den : 0.f;
            float w = mode == kEdgeFeatureDist2 ? feature_dist2(ni, nrm[j], cs) : expf(-d2 * inv_h) * fmaxf(0.f, cs);
            if (binarize > 0.f) w = w > binarize ? 1.f : 0.f;
            col[o] = (int32_t)j;
            val[o] = w;
            rsum += w;
        }
        ++o;
    }
    if (row_normalize && lane == 0 && rsum > 0.f)   // divide: a denormal sum has an infinite reciprocal
        for (int64_t e = o0; e < o; ++e) val[e] = val[e] / rsum;
}

// The distinct columns of every row (a sorted row repeats a column for mutual
// neighbours), one warp per row.
__global__ void __launch_bounds__(256) k_compact_cols(const uint32_t* __restrict__ tcol,
                                                      const uint32_t* __restrict__ tptr,
                                                      const uint32_t* __restrict__ tcnt,
                                                      const int64_t* __restrict__ row_ptr, int64_t n,
                                                      int32_t* __restrict__ col) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 8 + warp;
    if (i >= n) return;   // whole warp
    const uint32_t* row = tcol + tptr[i];
    const uint32_t c = tcnt[i];
    int64_t o = row_ptr[i];
    for (uint32_t t0 = 0; t0 < c; t0 += 32) {
        const uint32_t t = t0 + lane;
        const uint32_t j = t < c ? row[t] : 0u;
        const bool keep = t < c && !(t > 0 && row[t - 1] == j);
        const uint32_t m = __ballot_sync(0xffffffffu, keep);
        if (keep) col[o + __popc(m & ((1u << lane) - 1u))] = (int32_t)j;
        o += __popc(m);
    }
}

// Edge values for df <= 128 kV, one warp per row i with f_i in registers.  The
// matrix is symmetric, so a row takes only its columns j > i and writes both
// entries (the mirrored one found by binary search in row j's sorted columns):
// the kernel is bound by gathering feature rows from L2, which this halves.
// Four rows are gathered at a time (16-byte loads when VEC); a lane then
// weights and writes the edge of its own column.  Rows are taken in the centres'
// Morton order, which keeps the neighbours' rows in L2.  1M Gaussians, k = 16,
// df = 384 (about 20M directed edges): 3.78 -> 1.50 ms, and 0.28 ms for the
// columns and the row sums that the one kernel did on the way.
template <int kV, bool VEC>
__global__ void __launch_bounds__(256) k_edge_weights(const int64_t* __restrict__ row_ptr,
                                                     const int32_t* __restrict__ col, const float* __restrict__ x,
                                                     const float* __restrict__ f, const float* __restrict__ nrm,
                                                     int64_t n, int df, float inv_h, float binarize,
                                                     const uint32_t* __restrict__ order, int mode,
                                                     float* __restrict__ val) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * 8 + warp;
    if (r >= n) return;   // whole warp
    const int64_t i = order ? (int64_t)order[r] : r;
    const int64_t o0 = row_ptr[i], o1 = row_ptr[i + 1];
    // channels 4 (lane + 32 k) .. + 3, or lane + 32 (4 k + q)
    auto load = [&](const float* p, float4* v) {
#pragma unroll
        for (int k = 0; k < kV; ++k) {
            if constexpr (VEC) {
                const int ch = 4 * (lane + 32 * k);
                v[k] = ch < df ? *reinterpret_cast<const float4*>(p + ch) : make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
                const int ch = lane + 128 * k;
                v[k].x = ch < df ? p[ch] : 0.f;
                v[k].y = ch + 32 < df ? p[ch + 32] : 0.f;
                v[k].z = ch + 64 < df ? p[ch + 64] : 0.f;
                v[k].w = ch + 96 < df ? p[ch + 96] : 0.f;
            }
        }
    };
    float4 fr[kV];
    load(f + i * df, fr);
    const float xi = x[3 * i], yi = x[3 * i + 1], zi = x[3 * i + 2];
    const float ni = nrm[i];
    for (int64_t t0 = o0; t0 < o1; t0 += 32) {
        const int64_t t = t0 + lane;
        const int32_t j = t < o1 ? col[t] : 0;
        const bool mine = t < o1 && (int64_t)j > i;
        float dot = 0.f;   // of this lane's column
        uint32_t m = __ballot_sync(0xffffffffu, mine);
        while (m) {
            int l[4];
            float d[4];
            float4 g[4][kV];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                l[q] = m ? __ffs(m) - 1 : -1;
                m &= m - 1u;
                const int32_t jq = __shfl_sync(0xffffffffu, j, l[q] < 0 ? l[0] : l[q]);
                load(f + (int64_t)jq * df, g[q]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                d[q] = 0.f;
#pragma unroll
                for (int k = 0; k < kV; ++k) {
                    d[q] = fmaf(fr[k].x, g[q][k].x, d[q]);
                    d[q] = fmaf(fr[k].y, g[q][k].y, d[q]);
                    d[q] = fmaf(fr[k].z, g[q][k].z, d[q]);
                    d[q] = fmaf(fr[k].w, g[q][k].w, d[q]);
                }
            }
#pragma unroll
            for (int s = 16; s > 0; s >>= 1)
#pragma unroll
                for (int q = 0; q < 4; ++q) d[q] += __shfl_xor_sync(0xffffffffu, d[q], s);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (lane == l[q]) dot = d[q];
        }
        if (mine) {
            const float ex = x[3 * (int64_t)j] - xi, ey = x[3 * (int64_t)j + 1] - yi, ez = x[3 * (int64_t)j + 2] - zi;
            const float d2 = ex * ex + ey * ey + ez * ez;
            const float nj = nrm[j], den = ni * nj;
            const float cs = den > 0.f ? dot / den : 0.f;
            float w = mode == kEdgeFeatureDist2 ? feature_dist2(ni, nj, cs) : expf(-d2 * inv_h) * fmaxf(0.f, cs);
            if (binarize > 0.f) w = w > binarize ? 1.f : 0.f;
            val[t] = w;
            int64_t lo = row_ptr[j], hi = row_ptr[j + 1] - 1;   // row j holds i
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if ((int64_t)col[mid] < i)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            val[lo] = w;
        }
    }
}

// Each row divided by its sum (rows summing to 0 stay), eight lanes per row.
__global__ void __launch_bounds__(256) k_normalise_graph_rows(const int64_t* __restrict__ row_ptr, int64_t n,
                                                              float* __restrict__ val) {
    const int sub = threadIdx.x & 7;
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
    const int64_t o0 = i < n ? row_ptr[i] : 0, o1 = i < n ? row_ptr[i + 1] : 0;
    float s = 0.f;
    for (int64_t e = o0 + sub; e < o1; e += 8) s += val[e];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (s > 0.f)   // divide: a denormal sum has an infinite reciprocal
        for (int64_t e = o0 + sub; e < o1; e += 8) val[e] = val[e] / s;
}

// exclusive scan into int64 row pointers (u32 scan + widening is enough while nnz < 2^32)
__global__ void k_widen_ptr(const uint32_t* __restrict__ p, int64_t n, const uint64_t* __restrict__ total,
                            int64_t* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = p[i];
    if (i == n) out[n] = (int64_t)*total;
}

// ------------------------------------------------------------ diffusion
__global__ void k_colnorm2(const float* __restrict__ x, int64_t n, int dx, double* __restrict__ acc) {
    __shared__ double part[32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int c = 0; c < dx; ++c) {
        double v = 0.0;
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
             i += (int64_t)gridDim.x * blockDim.x) {
            const double t = x[i * dx + c];
            v += t * t;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) part[warp][c] = v;
    }
    __syncthreads();
    if (threadIdx.x < dx) {
        double v = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += part[w][threadIdx.x];
        atomicAdd(acc + threadIdx.x, v);
    }
}

// y = A (x / ||x||) for one column (dx == 1, the CSR form): groups of kLanes
// lanes per row over a grid-stride range of rows.  ||y||^2 is reduced in the
// block and added once per block (float64).
template <int kLanes>
__global__ void __launch_bounds__(256) k_spmv_scaled(const int64_t* __restrict__ rp,
                                                    const int32_t* __restrict__ col,
                                                    const float* __restrict__ val,
                                                    const float* __restrict__ x, int64_t n, int dx,
                                                    const double* __restrict__ n2_in,
                                                    float* __restrict__ y, double* __restrict__ n2_out) {
    __shared__ double part[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane % kLanes;
    const double nn = n2_in[0];
    const float s = nn > 0.0 ? (float)(1.0 / sqrt(nn)) : 0.f;
    double mine = 0.0;
    const int64_t groups = (int64_t)gridDim.x * (blockDim.x / kLanes);
    const int64_t g0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kLanes;
    for (int64_t base = 0; base < n; base += groups) {
        const int64_t i = base + g0;
        float acc = 0.f;
        if (i < n)
            for (int64_t e = rp[i] + sub; e < rp[i + 1]; e += kLanes) acc = fmaf(val[e], x[col[e]], acc);
#pragma unroll
        for (int o = kLanes / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (i < n && sub == 0) {
            acc *= s;
            y[i] = acc;
            mine += (double)acc * acc;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if (lane == 0) part[warp][0] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += part[w][0];
        atomicAdd(n2_out, t);
    }
}

// Several columns (2 <= dx <= 32): L = ceil(dx / 4) lanes per row, each
// owning 4 consecutive columns, so a warp works on 32 / L rows at once (a row
// is a chain of dependent loads: its pointer, then per entry the column and
// the x values).  Each (row, column) sum is one fmaf chain over the row's
// entries in order, then the column's scale; the columns' squared norms are
// summed per block in shared memory, then added to n2_out.
__global__ void __launch_bounds__(256) k_spmv_cols(const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                   const float* __restrict__ val, const float* __restrict__ x,
                                                   int64_t n, int dx, const double* __restrict__ n2_in,
                                                   float* __restrict__ y, double* __restrict__ n2_out) {
    __shared__ double colsum[32];
    const int L = (dx + 3) >> 2, G = 32 / L;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = lane / L, c0 = 4 * (lane - grp * L);
    const bool act = grp < G;
    if (threadIdx.x < 32) colsum[threadIdx.x] = 0.0;
    __syncthreads();
    float sc[4];
    double mine[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const double nn = (act && c0 + q < dx) ? n2_in[c0 + q] : 0.0;
        sc[q] = nn > 0.0 ? (float)(1.0 / sqrt(nn)) : 0.f;
    }
    const int64_t nw = (int64_t)gridDim.x * 8;
    for (int64_t base = ((int64_t)blockIdx.x * 8 + warp) * G; base < n; base += nw * G) {
        const int64_t i = base + grp;
        if (!act || i >= n) continue;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int64_t e = rp[i], e1 = rp[i + 1]; e < e1; ++e) {
            const float v = val[e];
            const float* xr = x + (int64_t)col[e] * dx + c0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (c0 + q < dx) acc[q] = fmaf(v, xr[q], acc[q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (c0 + q < dx) {
                const float a = acc[q] * sc[q];
                y[i * dx + c0 + q] = a;
                mine[q] += (double)a * a;
            }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (act && c0 + q < dx) atomicAdd(&colsum[c0 + q], mine[q]);
    __syncthreads();
    if (threadIdx.x < dx) atomicAdd(n2_out + threadIdx.x, colsum[threadIdx.x]);
}

// ---- several columns on a renumbered copy
// The rows in the centres' Morton order (row r is node perm[r], or r without
// one), their entries {position of the column, value} in the CSR order and in
// fours (the last one of a row filled up with column -1), and the columns
// padded to a multiple of four: one 32-byte load per four entries and one
// 16-byte gather per entry and lane, rows of a block being spatial neighbours
// whose gathers meet in L1.
__global__ void k_pcsr_len(const int64_t* __restrict__ rp, int64_t n, const int32_t* __restrict__ perm,
                           uint32_t* __restrict__ len) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r > n) return;
    const int64_t i = r < n && perm ? (int64_t)perm[r] : r;
    len[r] = r < n ? (uint32_t)(rp[i + 1] - rp[i] + 3) >> 2 : 0u;
}

// eight lanes per row
__global__ void __launch_bounds__(256) k_pcsr_fill(const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                   const float* __restrict__ val, int64_t n,
                                                   const int32_t* __restrict__ perm, const int32_t* __restrict__ inv,
                                                   const uint32_t* __restrict__ prp, int2* __restrict__ ent) {
    const int sub = threadIdx.x & 7;
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
    if (r >= n) return;
    const int64_t i = perm ? (int64_t)perm[r] : r;
    const int64_t e0 = rp[i];
    const uint32_t c = (uint32_t)(rp[i + 1] - e0);
    const int64_t o = 4 * (int64_t)prp[r], o1 = 4 * (int64_t)prp[r + 1];
    for (int64_t k = sub; o + k < o1; k += 8) {
        const int32_t j = k < c ? col[e0 + k] : 0;
        ent[o + k] = k < c ? make_int2(inv ? inv[j] : j, __float_as_int(val[e0 + k])) : make_int2(-1, 0);
    }
}

// Four entries, 32-byte aligned.
struct Ent4 {
    int2 e[4];
};
__device__ __forceinline__ Ent4 load_ent4(const int2* p) {
    Ent4 r;
    asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r.e[0].x), "=r"(r.e[0].y), "=r"(r.e[1].x), "=r"(r.e[1].y), "=r"(r.e[2].x), "=r"(r.e[2].y),
                   "=r"(r.e[3].x), "=r"(r.e[3].y)
                 : "l"(p));
    return r;
}

// The block's squared column norms into acc[0 .. dx), in float64: each lane's four columns
// c0 .. c0 + 3 of row group g (of ng), through part [ng][4 L].
__device__ __forceinline__ void add_norms(const double* q, bool act, int g, int ng, int c0, int dx, int L, double* part,
                                          double* __restrict__ acc) {
    if (act)
#pragma unroll
        for (int k = 0; k < 4; ++k) part[g * 4 * L + c0 + k] = q[k];
    __syncthreads();
    if ((int)threadIdx.x < dx) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
        for (int w = 0; w < ng; ++w) v[w & 3] += part[w * 4 * L + threadIdx.x];
        atomicAdd(acc + threadIdx.x, (v[0] + v[1]) + (v[2] + v[3]));
    }
}

constexpr int kPcolThreads = 512, kPcolBlocks = 2;

// x0 [n, dx] -> the padded, renumbered vector [n][L] float4, and its norms.
__global__ void __launch_bounds__(kPcolThreads, kPcolBlocks) k_pack_cols(const float* __restrict__ x0,
                                                            const int32_t* __restrict__ perm, int64_t n, int dx,
                                                            int64_t rows_per_block, float4* __restrict__ xp,
                                                            double* __restrict__ acc) {
    __shared__ double part[4 * kPcolThreads];
    const int L = (dx + 3) >> 2, G = 32 / L, ng = G * (kPcolThreads / 32);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane / L, k = lane - sub * L, c0 = 4 * k;
    const bool act = sub < G;
    double q[4] = {0.0, 0.0, 0.0, 0.0};
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_block, r1 = min(n, r0 + rows_per_block);
    if (act)
        for (int64_t r = r0 + warp * G + sub; r < r1; r += ng) {
            const float* src = x0 + (perm ? (int64_t)perm[r] : r) * dx;
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                v[u] = c0 + u < dx ? src[c0 + u] : 0.f;
                q[u] = fma((double)v[u], (double)v[u], q[u]);
            }
            xp[r * L + k] = make_float4(v[0], v[1], v[2], v[3]);
        }
    add_norms(q, act, warp * G + sub, ng, c0, dx, L, part, acc);
}

__global__ void k_unpack_cols(const float4* __restrict__ yp, const int32_t* __restrict__ inv, int64_t n, int dx,
                              float* __restrict__ out) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * dx) return;
    const int64_t i = t / dx;
    const int c = (int)(t - i * dx), L = (dx + 3) >> 2;
    out[t] = reinterpret_cast<const float*>(yp + (inv ? (int64_t)inv[i] : i) * L)[c];
}

// y = A (x / ||x||) on the copy: L = ceil(dx / 4) lanes per row, a block taking
// rows_per_block consecutive rows.  Each (row, column) sum is one fmaf chain
// over the row's entries in order, then the column's scale.  Bound by the gathers
// from L1 and L2, behind which the float64 sums of squares (units at a 64th of the
// rate) are hidden: 67 us a step of 250k rows and 21 columns, where two float32 values
// with their exact errors, of 46 bits, took 73 and three, of 53 bits, 79.  In node
// order 126; the other forms with the two-value sums: 128-thread blocks, whose regions do
// not meet in L1, 95; rows padded to whole 128-byte lines 109; one block of 1024 per SM 81.
__global__ void __launch_bounds__(kPcolThreads, kPcolBlocks) k_spmv_pcols(const uint32_t* __restrict__ prp,
                                                             const int2* __restrict__ ent,
                                                             const float4* __restrict__ x, int64_t n, int dx,
                                                             int64_t rows_per_block,
                                                             const double* __restrict__ n2_in,
                                                             float4* __restrict__ y, double* __restrict__ n2_out) {
    __shared__ double part[4 * kPcolThreads];
    const int L = (dx + 3) >> 2, G = 32 / L, ng = G * (kPcolThreads / 32);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane / L, k = lane - sub * L, c0 = 4 * k;
    const bool act = sub < G;
    float sc[4];
    double q[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const double nn = (act && c0 + u < dx) ? n2_in[c0 + u] : 0.0;
        sc[u] = nn > 0.0 ? (float)(1.0 / sqrt(nn)) : 0.f;
    }
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_block, r1 = min(n, r0 + rows_per_block);
    if (act)
        for (int64_t r = r0 + warp * G + sub; r < r1; r += ng) {
            const uint32_t e1 = prp[r + 1];
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            for (uint32_t e = prp[r]; e < e1; ++e) {
                const Ent4 en = load_ent4(ent + 4 * (size_t)e);
                float4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (en.e[u].x >= 0) v[u] = x[(int64_t)en.e[u].x * L + k];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (en.e[u].x >= 0) {
                        const float w = __int_as_float(en.e[u].y);
                        a.x = fmaf(w, v[u].x, a.x);
                        a.y = fmaf(w, v[u].y, a.y);
                        a.z = fmaf(w, v[u].z, a.z);
                        a.w = fmaf(w, v[u].w, a.w);
                    }
            }
            a = make_float4(a.x * sc[0], a.y * sc[1], a.z * sc[2], a.w * sc[3]);
            q[0] = fma((double)a.x, (double)a.x, q[0]);
            q[1] = fma((double)a.y, (double)a.y, q[1]);
            q[2] = fma((double)a.z, (double)a.z, q[2]);
            q[3] = fma((double)a.w, (double)a.w, q[3]);
            y[r * L + k] = a;
        }
    add_norms(q, act, warp * G + sub, ng, c0, dx, L, part, n2_out);
}

// Sliced copy of the matrix for single-column diffusion: slices of 32
// consecutive rows, each padded to its longest row and stored column-major
// (slot j of row r at off[slice] + 32 j + r % 32; padding: column = the row,
// value 0).  One thread per row then reads its columns and values with
// coalesced 128-byte warp loads and no row-pointer dependence.
// With perm (the centres' Morton order) the sliced copy is renumbered: its
// row r is node perm[r] and its columns are positions (inv), so that the rows
// of a slice and the x entries they gather are spatial neighbours; the
// diffusion then runs on the permuted vector.
__global__ void k_sell_width(const int64_t* __restrict__ rp, int64_t n, int64_t nslices,
                             const int32_t* __restrict__ perm, uint32_t* __restrict__ slots) {
    const int lane = threadIdx.x & 31;
    const int64_t s = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (s > nslices) return;
    if (s == nslices) {   // the scan's total
        if (lane == 0) slots[s] = 0u;
        return;
    }
    const int64_t r = s * 32 + lane;
    const int64_t i = r < n ? (perm ? (int64_t)perm[r] : r) : 0;
    uint32_t len = r < n ? (uint32_t)(rp[i + 1] - rp[i]) : 0u;
    len = __reduce_max_sync(0xffffffffu, len);
    if (lane == 0) slots[s] = 32u * len;
}

__global__ void k_sell_fill(const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                            const float* __restrict__ val, int64_t n, int64_t nslices,
                            const int32_t* __restrict__ perm, const int32_t* __restrict__ inv,
                            const uint32_t* __restrict__ off, int32_t* __restrict__ scol, float* __restrict__ sval) {
    const int lane = threadIdx.x & 31;
    const int64_t s = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (s >= nslices) return;
    const int64_t r = s * 32 + lane;
    const int64_t i = r < n ? (perm ? (int64_t)perm[r] : r) : 0;
    const int64_t e0 = r < n ? rp[i] : 0;
    const uint32_t len = r < n ? (uint32_t)(rp[i + 1] - e0) : 0u;
    const uint32_t w = (off[s + 1] - off[s]) / 32u;
    for (uint32_t j = 0; j < w; ++j) {
        const uint32_t p = off[s] + 32u * j + (uint32_t)lane;
        const bool real = j < len;
        const int32_t c = real ? col[e0 + j] : 0;
        scol[p] = real ? (inv ? inv[c] : c) : (int32_t)(r < n ? r : 0);
        sval[p] = real ? val[e0 + j] : 0.f;
    }
}

__global__ void k_invert_perm(const int32_t* __restrict__ perm, int64_t n, int32_t* __restrict__ inv) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n) inv[perm[r]] = (int32_t)r;
}

__global__ void k_gather_perm(const float* __restrict__ x, const int32_t* __restrict__ perm, int64_t n,
                              float* __restrict__ y) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n) y[r] = x[perm[r]];
}

__global__ void k_scatter_perm(const float* __restrict__ y, const int32_t* __restrict__ perm, int64_t n,
                               float* __restrict__ x) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n) x[perm[r]] = y[r];
}

// y = A (x / ||x||) for one column on the sliced copy: a warp per slice, a
// thread per row; ||y||^2 reduced per block, added once per block (float64).
__global__ void __launch_bounds__(256) k_spmv_sell(const uint32_t* __restrict__ off, const int32_t* __restrict__ scol,
                                                  const float* __restrict__ sval, const float* __restrict__ x,
                                                  int64_t n, int64_t nslices, const double* __restrict__ n2_in,
                                                  float* __restrict__ y, double* __restrict__ n2_out) {
    __shared__ double part[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double nn = n2_in[0];
    const float sc = nn > 0.0 ? (float)(1.0 / sqrt(nn)) : 0.f;
    double mine = 0.0;
    for (int64_t s = (int64_t)blockIdx.x * 8 + warp; s < nslices; s += (int64_t)gridDim.x * 8) {
        const uint32_t o1 = off[s + 1];
        float acc = 0.f;
#pragma unroll 4
        for (uint32_t p = off[s] + (uint32_t)lane; p < o1; p += 32u) acc = fmaf(sval[p], x[scol[p]], acc);
        const int64_t r = s * 32 + lane;
        if (r < n) {
            acc *= sc;
            y[r] = acc;
            mine += (double)acc * acc;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if (lane == 0) part[warp] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += part[w];
        atomicAdd(n2_out, t);
    }
}

// Morton code of a point's cell, ten bits per axis.
__global__ void k_morton_keys(const float* __restrict__ x, int64_t n, int64_t npad, Grid gr, int shift,
                              uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npad) return;
    uint32_t key = 0xffffffffu;
    if (i < n) {
        key = 0u;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            uint32_t c = (uint32_t)cell_coord(x[3 * i + a], gr.lo[a], gr.inv_cell, gr.g[a]) >> shift;
            uint32_t b = 0u;   // bits of c, three apart
#pragma unroll
            for (int t = 0; t < 10; ++t) b |= ((c >> t) & 1u) << (3 * t);
            key |= b << a;
        }
    }
    keys[i] = key;
    vals[i] = (uint32_t)i;
}

// *order (if given) receives the points' indices in the Morton order of their
// grid cells (valid until the scene's workspace is reused), or null: a run of them
// is a compact region, where the cells' own scanline order gives thin sticks.
ludvig_status knn_impl(ludvig_scene* s, int k, int32_t* nbr, cudaStream_t st, const uint32_t** order = nullptr) {
    Arena& ws = s->ws;
    if (order) *order = nullptr;
    const int64_t n = s->n;
    float* bb;
    LV_TRY(ws.get("knn.bbox", 8, &bb));
    {
        const int init[6] = {0x7fffffff, 0x7fffffff, 0x7fffffff, (int)0x80000000, (int)0x80000000,
                             (int)0x80000000};
        void* h;
        LV_TRY(ws.pinned("knn.bbox_h", 64, &h));
        std::memcpy(h, init, sizeof(init));
        LV_CUDA(cudaMemcpyAsync(bb, h, sizeof(init), cudaMemcpyHostToDevice, st));
        k_bbox<<<(unsigned)std::min<int64_t>(1024, ceil_div(n, 256)), 256, 0, st>>>(s->means, n, bb);
        LV_LAUNCH();
        LV_CUDA(cudaMemcpyAsync(static_cast<char*>(h) + 32, bb, 24, cudaMemcpyDeviceToHost, st));
        LV_CUDA(cudaStreamSynchronize(st));
        int enc[6];
        std::memcpy(enc, static_cast<char*>(h) + 32, 24);
        float lo[3], hi[3];
        for (int a = 0; a < 3; ++a) {
            int l = enc[a] >= 0 ? enc[a] : enc[a] ^ 0x7fffffff;
            int hh = enc[3 + a] >= 0 ? enc[3 + a] : enc[3 + a] ^ 0x7fffffff;
            std::memcpy(&lo[a], &l, 4);
            std::memcpy(&hi[a], &hh, 4);
        }
        Grid gr;
        double ext[3], vol = 1.0;
        for (int a = 0; a < 3; ++a) {
            ext[a] = std::max(1e-6, (double)hi[a] - (double)lo[a]);
            vol *= ext[a];
        }
        auto cells_of = [&](double c) {
            int64_t tot = 1;
            for (int a = 0; a < 3; ++a) tot *= (int64_t)(ext[a] / c) + 1;
            return tot;
        };
        // about two points per cell on average, at most 2^24 cells
        double cell = std::cbrt(vol * 2.0 / (double)std::max<int64_t>(n, 1));
        while (cells_of(cell) > ((int64_t)1 << 24)) cell *= 1.25;
        const auto set_grid = [&](double c) {
            gr.cell = (float)c;
            gr.inv_cell = (float)(1.0 / c);
            for (int a = 0; a < 3; ++a) {
                gr.lo[a] = lo[a];
                gr.g[a] = (int)(ext[a] / c) + 1;
            }
        };
        set_grid(cell);
        // A query scans the 27 or 125 cells around it, so what counts is how
        // full the cells are that the points themselves lie in (the count's
        // mean over the points, 3 for uniform points).  Clustered scenes leave
        // most cells empty: at 6 points the search of 1M clustered centres takes
        // 2.3 ms (3: 3.2, 12: 2.3, cells as they are: 2.9)
        int64_t ncell = 0;
        uint32_t* cells = nullptr;
        const auto count_cells = [&]() -> ludvig_status {   // and two zeros behind the last
            ncell = (int64_t)gr.g[0] * gr.g[1] * gr.g[2];
            LV_TRY(ws.get("knn.cells", (size_t)ncell + 2, &cells));
            LV_CUDA(cudaMemsetAsync(cells, 0, sizeof(uint32_t) * ((size_t)ncell + 2), st));
            k_cell_count<<<grid_for(n, 256), 256, 0, st>>>(s->means, n, gr, cells);
            LV_LAUNCH();
            return LUDVIG_OK;
        };
        LV_TRY(count_cells());
        if (n >= kKnnDensityMin) {
            unsigned long long* sq;
            LV_TRY(ws.get("knn.sq", 1, &sq));
            LV_CUDA(cudaMemsetAsync(sq, 0, sizeof(unsigned long long), st));
            k_cell_square<<<(unsigned)std::min<int64_t>(608, ceil_div(ncell, 256)), 256, 0, st>>>(cells, ncell, sq);
            LV_LAUNCH();
            LV_CUDA(cudaMemcpyAsync(static_cast<char*>(h) + 56, sq, 8, cudaMemcpyDeviceToHost, st));
            LV_CUDA(cudaStreamSynchronize(st));
            unsigned long long sum;
            std::memcpy(&sum, static_cast<char*>(h) + 56, 8);
            const double mean = (double)sum / (double)n;
            if (mean > 2.0 * kKnnCellPoints) {
                double c = cell * std::cbrt(kKnnCellPoints / mean);
                // (a coordinate's rounding stays far below the search's 0.05 % margin)
                c = std::max(c, std::max(ext[0], std::max(ext[1], ext[2])) / 1024.0);
                while (cells_of(c) > ((int64_t)1 << 24)) c *= 1.1;
                if (c < cell) {
                    cell = c;
                    set_grid(cell);
                    LV_TRY(count_cells());
                }
            }
        }
        // cells[c] = the first sorted position of cell c (a run of cells along x is one
        // range): the counts' prefix, whose time does not depend on how the empty cells
        // lie (a thread that wrote the gap before its point took 45 ms for two
        // tight clusters far apart, 100k points)
        LV_TRY(scan_exclusive_u32(cells, cells, ncell + 1, nullptr, ws, st));
        const int64_t npad = round_up(n, kRadixTile);
        uint32_t *keys, *vals, *keys2, *vals2;
        LV_TRY(ws.get("knn.keys", (size_t)npad, &keys));
        LV_TRY(ws.get("knn.vals", (size_t)npad, &vals));
        LV_TRY(ws.get("knn.keys2", (size_t)npad, &keys2));
        LV_TRY(ws.get("knn.vals2", (size_t)npad, &vals2));
        k_cell_keys<<<grid_for(npad, 256), 256, 0, st>>>(s->means, n, npad, gr, keys, vals);
        LV_LAUNCH();
        int nbits = 1;
        while (((int64_t)1 << nbits) <= ncell) ++nbits;
        uint32_t *sk = keys, *sv = vals;
        LV_TRY(radix_sort_pairs(&sk, &sv, keys2, vals2, 1, npad, nbits, ws, st));
        float4* pts;
        LV_TRY(ws.get("knn.pts", (size_t)n, &pts));
        k_gather_sorted<<<grid_for(n, 256), 256, 0, st>>>(s->means, sv, n, pts);
        LV_LAUNCH();
        const unsigned g = grid_for(n, 128);
        uint32_t *far = sk, *nfar = cells + ncell + 1;   // (the sorted keys are used up; a zero behind the starts)
        if (k <= 8) k_knn<8><<<g, 128, 0, st>>>(pts, n, gr, cells, k, nbr, far, nfar);
        else if (k <= 16) k_knn<16><<<g, 128, 0, st>>>(pts, n, gr, cells, k, nbr, far, nfar);
        else if (k <= 32) k_knn<32><<<g, 128, 0, st>>>(pts, n, gr, cells, k, nbr, far, nfar);
        else k_knn<64><<<g, 128, 0, st>>>(pts, n, gr, cells, k, nbr, far, nfar);
        LV_LAUNCH();
        if (std::max(gr.g[0], std::max(gr.g[1], gr.g[2])) > kKnnNear) {   // (else every search has ended)
            const int3 bg = make_int3((gr.g[0] + kKnnBlock - 1) / kKnnBlock, (gr.g[1] + kKnnBlock - 1) / kKnnBlock,
                                      (gr.g[2] + kKnnBlock - 1) / kKnnBlock);
            const int64_t nblocks = (int64_t)bg.x * bg.y * bg.z;
            uint32_t* bcnt;
            LV_TRY(ws.get("knn.blocks", (size_t)nblocks, &bcnt));
            k_block_count<<<grid_for(nblocks, 256), 256, 0, st>>>(cells, gr, bg, nblocks, nfar, bcnt);
            LV_LAUNCH();
            const unsigned gf = (unsigned)std::min<int64_t>(ceil_div(n, 4), 152 * 16);
            if (k <= 32) k_knn_far<1><<<gf, 128, 0, st>>>(pts, gr, cells, bg, bcnt, k, far, nfar, nbr);
            else k_knn_far<2><<<gf, 128, 0, st>>>(pts, gr, cells, bg, bcnt, k, far, nfar, nbr);
            LV_LAUNCH();
        }
        if (order) {
            int shift = 0;
            while ((std::max(gr.g[0], std::max(gr.g[1], gr.g[2])) >> shift) > 1024) ++shift;
            k_morton_keys<<<grid_for(npad, 256), 256, 0, st>>>(s->means, n, npad, gr, shift, keys, vals);
            LV_LAUNCH();
            sk = keys;
            sv = vals;
            LV_TRY(radix_sort_pairs(&sk, &sv, keys2, vals2, 1, npad, 32, ws, st));
            *order = sv;
        }
    }
    return LUDVIG_OK;
}

}  // namespace

}  // namespace ludvig

using namespace ludvig;

extern "C" ludvig_status ludvig_knn(ludvig_scene_t scene, int32_t k, int32_t* nbr, void* stream) {
    LV_ARG(scene != nullptr && nbr != nullptr, "NULL argument");
    LV_ARG(k >= 1 && k <= 64, "k must be in [1, 64]");
    if (scene->n == 0) return LUDVIG_OK;
    StageScope scope(LUDVIG_STAGE_KNN, static_cast<cudaStream_t>(stream));
    return knn_impl(scene, k, nbr, static_cast<cudaStream_t>(stream));
}

namespace ludvig {
namespace {

// The union kNN graph with per-edge values of `mode` (see kEdgeSpatialCos).
ludvig_status graph_build_impl(ludvig_scene_t scene, int32_t k, const float* feats, int32_t df, float spatial_h,
                               float binarize, int32_t row_normalize, int mode, cudaStream_t st,
                               ludvig_graph_t* out) {
    ludvig_graph* g = new ludvig_graph();
    g->n = scene->n;
    LV_CUDA(cudaGetDevice(&g->device));
    const int64_t n = scene->n;
    Arena& ws = scene->ws;
    auto fail = [&](ludvig_status s) {
        ludvig_graph_destroy(g);
        return s;
    };
    ludvig_status r;
    if (cudaMalloc(&g->row_ptr, sizeof(int64_t) * (size_t)(n + 1)) != cudaSuccess) {
        cudaGetLastError();
        set_error("graph allocation failed");
        return fail(LUDVIG_ERR_OOM);
    }
    if (n == 0) {
        if (cudaMemsetAsync(g->row_ptr, 0, sizeof(int64_t), st) != cudaSuccess) return fail(LUDVIG_ERR_CUDA);
        *out = g;
        return LUDVIG_OK;
    }
    int32_t* nbr;
    uint32_t *own, *indeg, *cnt, *tptr, *cursor, *ucnt, *uptr;
    uint64_t *tot_d, *utot_d;
    float* nrm;
#define GB_TRY(expr)                   \
    do {                               \
        r = (expr);                    \
        if (r != LUDVIG_OK) return fail(r); \
    } while (0)
    GB_TRY(ws.get("g.nbr", (size_t)n * k, &nbr));
    GB_TRY(ws.get("g.own", (size_t)n, &own));
    GB_TRY(ws.get("g.indeg", (size_t)n, &indeg));
    GB_TRY(ws.get("g.cnt", (size_t)n, &cnt));
    GB_TRY(ws.get("g.tptr", (size_t)n, &tptr));
    GB_TRY(ws.get("g.cursor", (size_t)n, &cursor));
    GB_TRY(ws.get("g.ucnt", (size_t)n, &ucnt));
    GB_TRY(ws.get("g.uptr", (size_t)n, &uptr));
    GB_TRY(ws.get("g.tot", 2, &tot_d));
    utot_d = tot_d + 1;
    GB_TRY(ws.get("g.nrm", (size_t)n, &nrm));
    const uint32_t* sorder = nullptr;   // rows in Morton order: neighbours' feature rows stay in L2
    {
        StageScope scope(LUDVIG_STAGE_KNN, st);
        GB_TRY(knn_impl(scene, k, nbr, st, &sorder));
    }
    if (sorder) {   // the graph keeps the order for its diffusion (the renumbered copy)
        if (cudaMalloc(&g->perm, sizeof(int32_t) * (size_t)n) != cudaSuccess ||
            cudaMalloc(&g->inv, sizeof(int32_t) * (size_t)n) != cudaSuccess) {
            cudaGetLastError();
            set_error("graph allocation failed");
            return fail(LUDVIG_ERR_OOM);
        }
        if (cudaMemcpyAsync(g->perm, sorder, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, st) !=
            cudaSuccess)
            return fail(LUDVIG_ERR_CUDA);
        k_invert_perm<<<grid_for(n, 256), 256, 0, st>>>(g->perm, n, g->inv);
        count_launch();
    }
    StageScope gscope(LUDVIG_STAGE_GRAPH, st);
    if (cudaMemsetAsync(indeg, 0, sizeof(uint32_t) * n, st) != cudaSuccess ||
        cudaMemsetAsync(cursor, 0, sizeof(uint32_t) * n, st) != cudaSuccess)
        return fail(LUDVIG_ERR_CUDA);
    k_own_and_indegree<<<grid_for(n, 256), 256, 0, st>>>(nbr, n, k, own, indeg);
    count_launch();
    k_row_counts<<<grid_for(n, 256), 256, 0, st>>>(own, indeg, n, cnt);
    count_launch();
    GB_TRY(scan_exclusive_u32(cnt, tptr, n, tot_d, ws, st));
    void* hbuf;
    GB_TRY(ws.pinned("g.tot_h", 16, &hbuf));
    uint64_t* tot_h = static_cast<uint64_t*>(hbuf);
    if (cudaMemcpyAsync(tot_h, tot_d, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return fail(LUDVIG_ERR_CUDA);
    const int64_t tnnz = (int64_t)tot_h[0];
    if (tnnz >= ((int64_t)1 << 32)) {
        set_error("graph too large");
        return fail(LUDVIG_ERR_UNSUPPORTED);
    }
    uint32_t* tcol;
    GB_TRY(ws.get("g.tcol", (size_t)std::max<int64_t>(tnnz, 1), &tcol));
    k_fill_rows<<<grid_for(n, 256), 256, 0, st>>>(nbr, n, k, tptr, own, cursor, tcol);
    count_launch();
    k_sort_unique_rows<<<grid_for(n, 8), 256, 0, st>>>(tcol, tptr, cnt, n, ucnt);
    count_launch();
    GB_TRY(scan_exclusive_u32(ucnt, uptr, n, utot_d, ws, st));
    k_widen_ptr<<<grid_for(n + 1, 256), 256, 0, st>>>(uptr, n, utot_d, g->row_ptr);
    count_launch();
    k_norms<<<grid_for(n, 8), 256, 0, st>>>(feats, n, df, nrm);
    count_launch();
    if (cudaMemcpyAsync(tot_h + 1, utot_d, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return fail(LUDVIG_ERR_CUDA);
    g->nnz = (int64_t)tot_h[1];
    if (cudaMalloc(&g->col, sizeof(int32_t) * (size_t)std::max<int64_t>(g->nnz, 1)) != cudaSuccess ||
        cudaMalloc(&g->val, sizeof(float) * (size_t)std::max<int64_t>(g->nnz, 1)) != cudaSuccess) {
        cudaGetLastError();
        set_error("graph allocation failed");
        return fail(LUDVIG_ERR_OOM);
    }
    {
        const unsigned gb = grid_for(n, 8);
        const float ih = 1.0f / spatial_h;
        if (df > 512) {
            k_edge_weights_any<<<gb, 256, 0, st>>>(tcol, tptr, cnt, g->row_ptr, scene->means, feats, nrm, n, df, ih,
                                                   binarize, row_normalize, sorder, mode, g->col, g->val);
        } else {
            k_compact_cols<<<gb, 256, 0, st>>>(tcol, tptr, cnt, g->row_ptr, n, g->col);
            count_launch();
            const bool vec = df % 4 == 0 && (reinterpret_cast<uintptr_t>(feats) & 15) == 0;
#define LV_EW(V, VEC) k_edge_weights<V, VEC><<<gb, 256, 0, st>>>(g->row_ptr, g->col, scene->means, feats, nrm, n, df, \
                                                                 ih, binarize, sorder, mode, g->val)
            if (df <= 128) vec ? LV_EW(1, true) : LV_EW(1, false);
            else if (df <= 256) vec ? LV_EW(2, true) : LV_EW(2, false);
            else if (df <= 384) vec ? LV_EW(3, true) : LV_EW(3, false);
            else vec ? LV_EW(4, true) : LV_EW(4, false);
#undef LV_EW
            if (row_normalize) {
                count_launch();
                k_normalise_graph_rows<<<grid_for(n * 8, 256), 256, 0, st>>>(g->row_ptr, n, g->val);
            }
        }
    }
    count_launch();
    if (cudaGetLastError() != cudaSuccess) {
        set_error("graph kernels failed to launch");
        return fail(LUDVIG_ERR_CUDA);
    }
#undef GB_TRY
    *out = g;
    return LUDVIG_OK;
}

}  // namespace
}  // namespace ludvig

extern "C" ludvig_status ludvig_graph_build(ludvig_scene_t scene, int32_t k, const float* feats, int32_t df,
                                            float spatial_h, float binarize, int32_t row_normalize,
                                            void* stream, ludvig_graph_t* out) {
    LV_ARG(out != nullptr, "out is NULL");
    *out = nullptr;
    LV_ARG(scene != nullptr, "scene is NULL");
    LV_ARG(k >= 1 && k <= 64, "k must be in [1, 64]");
    LV_ARG(df >= 1 && feats != nullptr, "features required (df >= 1)");
    LV_ARG(spatial_h > 0.f, "spatial_h must be positive");
    return graph_build_impl(scene, k, feats, df, spatial_h, binarize, row_normalize, kEdgeSpatialCos,
                            static_cast<cudaStream_t>(stream), out);
}

extern "C" ludvig_status ludvig_graph_destroy(ludvig_graph_t g) {
    if (!g) return LUDVIG_OK;
    cudaDeviceSynchronize();
    cudaFree(g->row_ptr);
    cudaFree(g->col);
    cudaFree(g->val);
    cudaFree(g->d2);
    cudaFree(g->perm);
    cudaFree(g->inv);
    g->ws.release();
    delete g;
    return LUDVIG_OK;
}

extern "C" int64_t ludvig_graph_nnz(ludvig_graph_t g) { return g ? g->nnz : -1; }

extern "C" int64_t ludvig_graph_workspace_bytes(ludvig_graph_t g) { return g ? (int64_t)g->ws.device_bytes() : -1; }

extern "C" ludvig_status ludvig_graph_export(ludvig_graph_t g, int64_t* row_ptr, int32_t* col, float* val,
                                             void* stream) {
    LV_ARG(g != nullptr, "graph is NULL");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (row_ptr) LV_CUDA(cudaMemcpyAsync(row_ptr, g->row_ptr, sizeof(int64_t) * (g->n + 1), cudaMemcpyDeviceToDevice, st));
    if (g->nnz > 0) {
        if (col) LV_CUDA(cudaMemcpyAsync(col, g->col, sizeof(int32_t) * g->nnz, cudaMemcpyDeviceToDevice, st));
        if (val) LV_CUDA(cudaMemcpyAsync(val, g->val, sizeof(float) * g->nnz, cudaMemcpyDeviceToDevice, st));
    }
    return LUDVIG_OK;
}

namespace ludvig {
namespace {

// The sliced copy of g's current values (built on first use and again after
// the values change; synchronises once to size it).  *ok = false when its
// slot count does not fit 32 bits (the CSR kernel is used then).
ludvig_status ensure_sell(ludvig_graph* g, cudaStream_t st, bool* ok, uint32_t** off, int32_t** scol,
                          float** sval) {
    *ok = false;
    const int64_t n = g->n, nslices = ceil_div(n, 32);
    uint32_t* slots;
    uint64_t* total_d;
    void* hb;
    LV_TRY(g->ws.get("sell.slots", (size_t)nslices + 1, &slots));
    LV_TRY(g->ws.get("sell.off", (size_t)nslices + 1, off));
    LV_TRY(g->ws.get("sell.total", 1, &total_d));
    LV_TRY(g->ws.pinned("sell.total_h", 16, &hb));
    uint64_t* total_h = static_cast<uint64_t*>(hb);
    if (g->sell_version == g->val_version) {
        LV_TRY(g->ws.get("sell.col", (size_t)std::max<uint64_t>(*total_h, 1), scol));
        LV_TRY(g->ws.get("sell.val", (size_t)std::max<uint64_t>(*total_h, 1), sval));
        *ok = true;
        return LUDVIG_OK;
    }
    k_sell_width<<<grid_for(nslices + 1, 8), 256, 0, st>>>(g->row_ptr, n, nslices, g->perm, slots);
    LV_LAUNCH();
    LV_TRY(scan_exclusive_u32(slots, *off, nslices + 1, total_d, g->ws, st));
    LV_CUDA(cudaMemcpyAsync(total_h, total_d, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
    LV_CUDA(cudaStreamSynchronize(st));
    if (*total_h >= ((uint64_t)1 << 32)) return LUDVIG_OK;
    LV_TRY(g->ws.get("sell.col", (size_t)std::max<uint64_t>(*total_h, 1), scol));
    LV_TRY(g->ws.get("sell.val", (size_t)std::max<uint64_t>(*total_h, 1), sval));
    k_sell_fill<<<grid_for(nslices, 8), 256, 0, st>>>(g->row_ptr, g->col, g->val, n, nslices, g->perm, g->inv,
                                                      *off, *scol, *sval);
    LV_LAUNCH();
    g->sell_version = g->val_version;
    g->sell_slices = nslices;
    *ok = true;
    return LUDVIG_OK;
}

// The renumbered row copy of g's current values (built on first use and again
// after the values change).
ludvig_status ensure_pcsr(ludvig_graph* g, cudaStream_t st, uint32_t** prp, int2** ent) {
    const int64_t n = g->n;
    LV_TRY(g->ws.get("pcsr.rp", (size_t)n + 1, prp));
    LV_TRY(g->ws.get("pcsr.ent", (size_t)(g->nnz + 3 * n + 4), ent));   // rows in whole fours
    if (g->pcsr_version == g->val_version) return LUDVIG_OK;
    k_pcsr_len<<<grid_for(n + 1, 256), 256, 0, st>>>(g->row_ptr, n, g->perm, *prp);
    LV_LAUNCH();
    LV_TRY(scan_exclusive_u32(*prp, *prp, n + 1, nullptr, g->ws, st));
    k_pcsr_fill<<<grid_for(n * 8, 256), 256, 0, st>>>(g->row_ptr, g->col, g->val, n, g->perm, g->inv, *prp, *ent);
    LV_LAUNCH();
    g->pcsr_version = g->val_version;
    return LUDVIG_OK;
}

// Whether a call of `steps` steps of the given weight runs on the row copy: when the
// copy is there, or once the steps taken without it since the values changed have cost
// what building it costs (about 100 us: four diffusion steps or 32 reach steps).  So a
// single short call does not pay for the copy (one diffusion step of 2 columns on 20k
// nodes 104 us, 214 with it; one reach step 66 and 164; ten on 300k 400 and 437), and many
// short calls pay for it once.
constexpr int64_t kCopySteps = 32, kDiffuseWeight = 8, kReachWeight = 1;

bool use_row_copy(ludvig_graph* g, int64_t steps, int64_t weight) {
    if (g->pcsr_version == g->val_version) return true;
    if (g->pcsr_steps_version != g->val_version) {
        g->pcsr_steps = 0;
        g->pcsr_steps_version = g->val_version;
    }
    g->pcsr_steps += std::min(steps, kCopySteps) * weight;
    return g->pcsr_steps >= kCopySteps;
}

// ludvig_diffuse for two columns or more.
ludvig_status diffuse_cols(ludvig_graph* g, const float* x0, int dx, int iters, float* out, double* n2, int sms,
                           cudaStream_t st) {
    const int64_t n = g->n;
    const int L = (dx + 3) / 4, ng = 32 / L * (kPcolThreads / 32);
    uint32_t* prp;
    int2* ent;
    float4* p[2];
    LV_TRY(ensure_pcsr(g, st, &prp, &ent));
    LV_TRY(g->ws.get("d.c0", (size_t)n * L, &p[0]));
    LV_TRY(g->ws.get("d.c1", (size_t)n * L, &p[1]));
    // one wave, or fewer blocks
    const int64_t passes = std::max<int64_t>(1, ceil_div(ceil_div(n, ng), (int64_t)sms * kPcolBlocks));
    const int64_t rpb = passes * ng;
    const unsigned blocks = (unsigned)ceil_div(n, rpb);
    k_pack_cols<<<blocks, kPcolThreads, 0, st>>>(x0, g->perm, n, dx, rpb, p[0], n2);
    LV_LAUNCH();
    for (int t = 0; t < iters; ++t) {
        k_spmv_pcols<<<blocks, kPcolThreads, 0, st>>>(prp, ent, p[t & 1], n, dx, rpb, n2 + 32 * t, p[(t + 1) & 1],
                                                      n2 + 32 * (t + 1));
        LV_LAUNCH();
    }
    k_unpack_cols<<<grid_for(n * dx, 256), 256, 0, st>>>(p[iters & 1], g->inv, n, dx, out);
    LV_LAUNCH();
    return LUDVIG_OK;
}

}  // namespace
}  // namespace ludvig

extern "C" ludvig_status ludvig_diffuse(ludvig_graph_t g, const float* x0, int32_t dx, int32_t iters,
                                        float* out, void* stream) {
    LV_ARG(g != nullptr, "graph is NULL");
    LV_ARG(dx >= 1 && dx <= 32, "dx must be in [1, 32]");
    LV_ARG(iters >= 0, "iters must be >= 0");
    LV_ARG(x0 != nullptr && out != nullptr, "NULL buffer");
    LV_ARG(x0 != out, "out must not alias x0");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t n = g->n;
    if (n == 0) return LUDVIG_OK;
    const size_t bytes = sizeof(float) * (size_t)n * dx;
    if (iters == 0) {
        LV_CUDA(cudaMemcpyAsync(out, x0, bytes, cudaMemcpyDeviceToDevice, st));
        return LUDVIG_OK;
    }
    double* n2;
    // n2[t*32 + c] = ||column c of g_t||^2, every step's slot zeroed up front
    LV_TRY(g->ws.get("d.n2", (size_t)(iters + 1) * 32, &n2));
    StageScope scope(LUDVIG_STAGE_DIFFUSE, st);
    LV_CUDA(cudaMemsetAsync(n2, 0, sizeof(double) * 32 * (size_t)(iters + 1), st));
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (dx > 1 && use_row_copy(g, iters, kDiffuseWeight)) return diffuse_cols(g, x0, dx, iters, out, n2, sms, st);
    float* tmp;
    LV_TRY(g->ws.get("d.tmp", (size_t)n * dx, &tmp));
    // ping-pong so that the last step writes `out`
    float* bufs[2] = {(iters % 2 == 1) ? out : tmp, (iters % 2 == 1) ? tmp : out};
    k_colnorm2<<<(unsigned)std::min<int64_t>(592, ceil_div(n, 256)), 256, 0, st>>>(x0, n, dx, n2);
    LV_LAUNCH();
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * 8, ceil_div(n, 32)));
    bool sell = false;
    uint32_t* soff = nullptr;
    int32_t* scol = nullptr;
    float* sval = nullptr;
    if (dx == 1) LV_TRY(ensure_sell(g, st, &sell, &soff, &scol, &sval));
    // the renumbered sliced copy works on the permuted vector: x0 gathered in,
    // the last step's vector scattered back to out
    const bool permuted = sell && g->perm;
    float *pa = nullptr, *pb = nullptr;
    if (permuted) {
        LV_TRY(g->ws.get("d.pa", (size_t)n, &pa));
        LV_TRY(g->ws.get("d.pb", (size_t)n, &pb));
        k_gather_perm<<<grid_for(n, 256), 256, 0, st>>>(x0, g->perm, n, pa);
        LV_LAUNCH();
    }
    const float* xin = permuted ? pa : x0;
    for (int t = 0; t < iters; ++t) {
        float* y = permuted ? ((t & 1) ? pa : pb) : bufs[t & 1];
        if (sell)
            k_spmv_sell<<<blocks, 256, 0, st>>>(soff, scol, sval, xin, n, g->sell_slices, n2 + 32 * t, y,
                                                n2 + 32 * (t + 1));
        else if (dx > 1)
            k_spmv_cols<<<blocks, 256, 0, st>>>(g->row_ptr, g->col, g->val, xin, n, dx, n2 + 32 * t, y,
                                                n2 + 32 * (t + 1));
        else
            k_spmv_scaled<8><<<blocks, 256, 0, st>>>(g->row_ptr, g->col, g->val, xin, n, 1, n2 + 32 * t, y,
                                                     n2 + 32 * (t + 1));
        LV_LAUNCH();
        xin = y;
    }
    if (permuted) {
        k_scatter_perm<<<grid_for(n, 256), 256, 0, st>>>(xin, g->perm, n, out);
        LV_LAUNCH();
    }
    return LUDVIG_OK;
}

// ---------------------------------------------------------------- diffusion without allocation
// Scratch of ludvig_diffuse_noalloc in statically allocated device memory:
// the ping-pong vector (at most kNoAllocMaxElems = n * dx floats, 4 MiB) and
// the per-step column norms (at most kNoAllocMaxIters steps, 32 columns,
// float64).  Every GPU that loads the library holds these 4.3 MB until the
// process exits.  All calls share them, so calls that overlap on the GPU race.
static constexpr int64_t kNoAllocMaxElems = (int64_t)1 << 20;
static constexpr int32_t kNoAllocMaxIters = 1024;
static constexpr int kNoAllocMaxDevices = 64;
static __device__ __align__(256) float g_noalloc_tmp[kNoAllocMaxElems];
static __device__ __align__(256) double g_noalloc_norm2[(kNoAllocMaxIters + 1) * 32];

namespace {
std::mutex g_noalloc_mu;
float* g_noalloc_tmp_ptr[kNoAllocMaxDevices] = {};
double* g_noalloc_norm2_ptr[kNoAllocMaxDevices] = {};

// Device addresses of the static scratch for the current device.  In host code
// the array names are host-side stand-ins, not device addresses, so they are
// translated once per device with cudaGetSymbolAddress.
ludvig_status noalloc_scratch(float** tmp, double** norm2) {
    int dev = 0;
    LV_CUDA(cudaGetDevice(&dev));
    LV_ARG(dev >= 0 && dev < kNoAllocMaxDevices, "device %d out of range", dev);
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_tmp_ptr[dev]) {
        void* a = nullptr;
        void* b = nullptr;
        LV_CUDA(cudaGetSymbolAddress(&a, g_noalloc_tmp));
        LV_CUDA(cudaGetSymbolAddress(&b, g_noalloc_norm2));
        g_noalloc_tmp_ptr[dev] = static_cast<float*>(a);
        g_noalloc_norm2_ptr[dev] = static_cast<double*>(b);
    }
    *tmp = g_noalloc_tmp_ptr[dev];
    *norm2 = g_noalloc_norm2_ptr[dev];
    return LUDVIG_OK;
}
}  // namespace

extern "C" ludvig_status ludvig_diffuse_noalloc(ludvig_graph_t g, const float* x0, int32_t dx, int32_t iters,
                                                float* out, void* stream) {
    LV_ARG(g != nullptr, "graph is NULL");
    LV_ARG(dx >= 1 && dx <= 32, "dx must be in [1, 32]");
    LV_ARG(iters >= 0 && iters <= kNoAllocMaxIters, "iters must be in [0, %d] for the allocation-free call",
           kNoAllocMaxIters);
    LV_ARG(x0 != nullptr && out != nullptr, "NULL buffer");
    LV_ARG(x0 != out, "out must not alias x0");
    const int64_t n = g->n;
    LV_ARG(n * dx <= kNoAllocMaxElems, "n * dx = %lld exceeds the allocation-free limit of %lld elements",
           (long long)(n * dx), (long long)kNoAllocMaxElems);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (n == 0) return LUDVIG_OK;
    const size_t bytes = sizeof(float) * (size_t)n * dx;
    if (iters == 0) {
        LV_CUDA(cudaMemcpyAsync(out, x0, bytes, cudaMemcpyDeviceToDevice, st));
        return LUDVIG_OK;
    }
    float* tmp;
    double* n2;
    LV_TRY(noalloc_scratch(&tmp, &n2));
    float* bufs[2] = {(iters % 2 == 1) ? out : tmp, (iters % 2 == 1) ? tmp : out};
    // the norm accumulators keep the previous call's sums: clear the slots used
    LV_CUDA(cudaMemsetAsync(n2, 0, sizeof(double) * 32 * (size_t)(iters + 1), st));
    k_colnorm2<<<(unsigned)std::min<int64_t>(592, ceil_div(n, 256)), 256, 0, st>>>(x0, n, dx, n2);
    LV_LAUNCH();
    int dev = 0, sms = 152;
    LV_CUDA(cudaGetDevice(&dev));
    LV_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * 8, ceil_div(n, 32)));
    const float* xin = x0;
    for (int t = 0; t < iters; ++t) {
        float* y = bufs[t & 1];
        if (dx == 1)
            k_spmv_scaled<8><<<blocks, 256, 0, st>>>(g->row_ptr, g->col, g->val, xin, n, 1, n2 + 32 * t, y,
                                                     n2 + 32 * (t + 1));
        else
            k_spmv_cols<<<blocks, 256, 0, st>>>(g->row_ptr, g->col, g->val, xin, n, dx, n2 + 32 * t, y,
                                                n2 + 32 * (t + 1));
        LV_LAUNCH();
        xin = y;
    }
    return LUDVIG_OK;
}

// ---------------------------------------------------------------- paper-form diffusion
// Eq. 7 with the appendix's similarity and unary term, and the segmentation
// variant of Sec. 4.1:
//   S_f(f_i, f_j) = exp(-||f^_i - f^_j||^2 / (b s_f^2))   (f^ l2-normalised,
//                   s_f the median edge distance),
//   P(f_i) = S_f(f_i, f_bar) with bandwidth b_P (f_bar the normalised mean of
//            the anchors' normalised features),
//   A_ij = S_f(f_i, f_j) P_i^1/2 P_j^1/2, thresholded at 1e-5 for segmentation,
//   g_0 = the top 10 % of the uplifted reference mask's positive values,
//   h_i = P_i on the nodes that g_T reaches, 0 elsewhere.
// The graph keeps each edge's ||f^_i - f^_j||^2 (the scene part, computed
// once); ludvig_graph_reweight forms A for a prompt's P.

namespace ludvig {
namespace {

__global__ void k_float_keys(const float* __restrict__ v, int64_t m, int64_t mpad, uint32_t* __restrict__ keys,
                             uint32_t* __restrict__ vals) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= mpad) return;
    keys[i] = i < m ? __float_as_uint(v[i]) : 0xffffffffu;   // non-negative floats order like their bits
    vals[i] = (uint32_t)i;
}

// s_f = median of sqrt(d2) over the edges: the mean of the two middle values
// of the sorted squared distances' roots (one value for an odd count).
__global__ void k_median_sf(const uint32_t* __restrict__ sorted, int64_t m, float* __restrict__ sf) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    if (m == 0) {
        *sf = 0.f;
        return;
    }
    const float a = sqrtf(__uint_as_float(sorted[(m - 1) / 2])), b = sqrtf(__uint_as_float(sorted[m / 2]));
    *sf = (m & 1) ? a : 0.5f * (a + b);
}

// One warp per row: A_ij = exp(-d2 inv) sqrt(P_i P_j), thresholded and
// row-normalised on request.
__global__ void __launch_bounds__(256) k_rbf_reweight(const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                      const float* __restrict__ d2, const float* __restrict__ P,
                                                      int64_t n, float inv, float binarize, int row_normalize,
                                                      float* __restrict__ val) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 8 + warp;
    if (i >= n) return;
    const int64_t e0 = rp[i], e1 = rp[i + 1];
    const float spi = P ? sqrtf(P[i]) : 1.f;   // sqrt(P_i) sqrt(P_j): the product P_i P_j may underflow
    float rsum = 0.f;
    for (int64_t e = e0 + lane; e < e1; e += 32) {
        float w = expf(-d2[e] * inv);
        if (P) w *= spi * sqrtf(P[col[e]]);
        if (binarize > 0.f) w = w > binarize ? 1.f : 0.f;
        val[e] = w;
        rsum += w;
    }
    if (!row_normalize) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rsum += __shfl_xor_sync(0xffffffffu, rsum, o);
    // divide (not multiply by 1/sum): a denormal sum has an infinite reciprocal
    if (rsum > 0.f)
        for (int64_t e = e0 + lane; e < e1; e += 32) val[e] = val[e] / rsum;
}

// Sum of the normalised features of the anchor nodes (g0_i > 0), per channel,
// in float64: block b takes rows [b R, (b + 1) R), thread t channels t, t + 256, ...
constexpr int kAnchorRows = 1024;
__global__ void __launch_bounds__(256) k_anchor_sum(const float* __restrict__ f, const float* __restrict__ nrm,
                                                    const float* __restrict__ g0, int64_t n, int df,
                                                    double* __restrict__ acc) {
    const int64_t r0 = (int64_t)blockIdx.x * kAnchorRows, r1 = n < r0 + kAnchorRows ? n : r0 + kAnchorRows;
    for (int c = threadIdx.x; c < df; c += blockDim.x) {
        float s = 0.f;
        for (int64_t i = r0; i < r1; ++i)
            if (g0[i] > 0.f && nrm[i] > 0.f) s += f[i * df + c] / nrm[i];
        if (s != 0.f) atomicAdd(acc + c, (double)s);
    }
}

// f_bar = acc / ||acc|| (zero when acc is zero), one block.
__global__ void k_anchor_finish(const double* __restrict__ acc, int df, float* __restrict__ fbar) {
    __shared__ double red[256];
    double s = 0.0;
    for (int c = threadIdx.x; c < df; c += blockDim.x) s += acc[c] * acc[c];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    const double nr = sqrt(red[0]);
    for (int c = threadIdx.x; c < df; c += blockDim.x) fbar[c] = nr > 0.0 ? (float)(acc[c] / nr) : 0.f;
}

// P_i = exp(-||f^_i - f_bar||^2 inv), one warp per row.
__global__ void __launch_bounds__(256) k_unary(const float* __restrict__ f, const float* __restrict__ nrm,
                                               const float* __restrict__ fbar, int64_t n, int df, float inv,
                                               float* __restrict__ P) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 8 + warp;
    if (i >= n) return;
    const float ni = nrm[i];
    const float sc = ni > 0.f ? 1.0f / ni : 0.f;
    float d2 = 0.f;
    for (int c = lane; c < df; c += 32) {
        const float t = f[i * df + c] * sc - fbar[c];
        d2 = fmaf(t, t, d2);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d2 += __shfl_xor_sync(0xffffffffu, d2, o);
    if (lane == 0) P[i] = expf(-d2 * inv);
}

// Top-percent selection of the positive values: keys as in the beta
// selection (descending value, ties in index order), positives counted.
__global__ void k_topfrac_keys(const float* __restrict__ u, int64_t n, int64_t npad, uint32_t* __restrict__ keys,
                               uint32_t* __restrict__ vals, unsigned long long* __restrict__ npos) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool pos = false;
    if (i < npad) {
        uint32_t k = 0xffffffffu;
        if (i < n && u[i] > 0.f) {
            k = ~__float_as_uint(u[i]);
            pos = true;
        }
        keys[i] = k;
        vals[i] = (uint32_t)i;
    }
    const unsigned m = __ballot_sync(0xffffffffu, pos);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(npos, (unsigned long long)__popc(m));
}

__global__ void k_topfrac_mark(const uint32_t* __restrict__ vals, const float* __restrict__ u, int64_t n,
                               const unsigned long long* __restrict__ npos, int percent, float* __restrict__ g0) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t keep = (int64_t)((*npos * (unsigned long long)percent + 99ull) / 100ull);
    if (k < keep && k < n) g0[vals[k]] = u[vals[k]];
}

// Reachability as bit sets (bit q = query column q): s_{t+1,i} = OR over the
// row's edges with A_ij > 0 of s_t,j.
__global__ void k_reach_init(const float* __restrict__ g0, const int32_t* __restrict__ inv, int64_t n, int dx,
                             uint32_t* __restrict__ s) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t b = 0u;
    for (int q = 0; q < dx; ++q)
        if (g0[i * dx + q] > 0.f) b |= 1u << q;
    s[inv ? (int64_t)inv[i] : i] = b;
}

// Four lanes per row of the renumbered copy, 32 bytes of entries per lane and
// load: 250k rows 22.5 -> 8.4 us a step against the CSR in node order.
__global__ void __launch_bounds__(256) k_reach_step(const uint32_t* __restrict__ prp, const int2* __restrict__ ent,
                                                    const uint32_t* __restrict__ s, int64_t n,
                                                    uint32_t* __restrict__ s2) {
    const int sub = threadIdx.x & 3;
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
    uint32_t b = 0u;
    if (r < n) {
        const uint32_t e1 = prp[r + 1];
        for (uint32_t e = prp[r] + sub; e < e1; e += 4) {
            const Ent4 en = load_ent4(ent + 4 * (size_t)e);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (en.e[u].x >= 0 && __int_as_float(en.e[u].y) > 0.f) b |= s[en.e[u].x];
        }
    }
    b |= __shfl_xor_sync(0xffffffffu, b, 1);
    b |= __shfl_xor_sync(0xffffffffu, b, 2);
    if (r < n && sub == 0) s2[r] = b;
}

// The same on the CSR, eight lanes per row (a row holds k to 2k entries), for few steps
// (see use_row_copy).
__global__ void __launch_bounds__(256) k_reach_step_csr(const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                        const float* __restrict__ val, const uint32_t* __restrict__ s,
                                                        int64_t n, uint32_t* __restrict__ s2) {
    const int sub = threadIdx.x & 7;
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
    uint32_t b = 0u;
    if (i < n)
        for (int64_t e = rp[i] + sub, e1 = rp[i + 1]; e < e1; e += 8)
            if (val[e] > 0.f) b |= s[col[e]];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) b |= __shfl_xor_sync(0xffffffffu, b, o);
    if (i < n && sub == 0) s2[i] = b;
}

__global__ void k_reach_out(const uint32_t* __restrict__ s, const int32_t* __restrict__ inv,
                            const float* __restrict__ P, int64_t n, int dx, float* __restrict__ h) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * dx) return;
    const int64_t i = t / dx;
    const int q = (int)(t - i * dx);
    h[t] = ((s[inv ? (int64_t)inv[i] : i] >> q) & 1u) ? (P ? P[i] : 1.f) : 0.f;
}

}  // namespace
}  // namespace ludvig

extern "C" ludvig_status ludvig_graph_build_rbf(ludvig_scene_t scene, int32_t k, const float* feats, int32_t df,
                                                void* stream, ludvig_graph_t* out) {
    LV_ARG(out != nullptr, "out is NULL");
    *out = nullptr;
    LV_ARG(scene != nullptr, "scene is NULL");
    LV_ARG(k >= 1 && k <= 64, "k must be in [1, 64]");
    LV_ARG(df >= 1 && (feats != nullptr || scene->n == 0), "features required (df >= 1)");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    ludvig_graph_t g = nullptr;
    LV_TRY(graph_build_impl(scene, k, feats, df, 1.0f, 0.f, 0, kEdgeFeatureDist2, st, &g));
    // the squared distances move to d2; val gets S_f with b = 1 and no unary term
    g->d2 = g->val;
    g->val = nullptr;
    const int64_t m = g->nnz;
    auto fail = [&](ludvig_status r) {
        ludvig_graph_destroy(g);
        return r;
    };
    if (cudaMalloc(&g->val, sizeof(float) * (size_t)std::max<int64_t>(m, 1)) != cudaSuccess) {
        cudaGetLastError();
        set_error("graph allocation failed");
        return fail(LUDVIG_ERR_OOM);
    }
    if (g->n == 0) {
        *out = g;
        return LUDVIG_OK;
    }
    const int64_t mpad = round_up(std::max<int64_t>(m, 1), kRadixTile);
    uint32_t *keys, *vals, *keys2, *vals2;
    float* sf_d;
    void* hb;
    Arena& ws = g->ws;
    ludvig_status r = LUDVIG_OK;
    if ((r = ws.get("rbf.keys", (size_t)mpad, &keys)) != LUDVIG_OK || (r = ws.get("rbf.vals", (size_t)mpad, &vals)) ||
        (r = ws.get("rbf.keys2", (size_t)mpad, &keys2)) || (r = ws.get("rbf.vals2", (size_t)mpad, &vals2)) ||
        (r = ws.get("rbf.sf", 1, &sf_d)) || (r = ws.pinned("rbf.sf_h", 16, &hb)))
        return fail(r);
    {
        StageScope scope(LUDVIG_STAGE_GRAPH, st);
        k_float_keys<<<grid_for(mpad, 256), 256, 0, st>>>(g->d2, m, mpad, keys, vals);
        count_launch();
        uint32_t *sk = keys, *sv = vals;
        if ((r = radix_sort_pairs(&sk, &sv, keys2, vals2, 1, mpad, 32, ws, st)) != LUDVIG_OK) return fail(r);
        k_median_sf<<<1, 32, 0, st>>>(sk, m, sf_d);
        count_launch();
        if (cudaMemcpyAsync(hb, sf_d, sizeof(float), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            set_error("graph: CUDA failure");
            return fail(LUDVIG_ERR_CUDA);
        }
    }
    g->s_f = *static_cast<float*>(hb);
    if (g->s_f > 0.f) {
        if ((r = ludvig_graph_reweight(g, 1.0f, nullptr, 0.f, 0, stream)) != LUDVIG_OK) return fail(r);
    } else if (m > 0 && cudaMemsetAsync(g->val, 0, sizeof(float) * (size_t)m, st) != cudaSuccess) {
        set_error("graph: CUDA failure");
        return fail(LUDVIG_ERR_CUDA);
    }
    *out = g;
    return LUDVIG_OK;
}

extern "C" ludvig_status ludvig_graph_feature_scale(ludvig_graph_t graph, float* s_f) {
    LV_ARG(graph != nullptr && s_f != nullptr, "NULL argument");
    LV_ARG(graph->d2 != nullptr || graph->n == 0, "not an RBF graph (ludvig_graph_build_rbf)");
    *s_f = graph->s_f;
    return LUDVIG_OK;
}

extern "C" ludvig_status ludvig_graph_reweight(ludvig_graph_t graph, float bandwidth, const float* unary,
                                               float binarize, int32_t row_normalize, void* stream) {
    LV_ARG(graph != nullptr, "graph is NULL");
    LV_ARG(graph->d2 != nullptr || graph->n == 0, "not an RBF graph (ludvig_graph_build_rbf)");
    LV_ARG(bandwidth > 0.f, "bandwidth must be positive");
    if (graph->n == 0 || graph->nnz == 0) return LUDVIG_OK;
    LV_ARG(graph->s_f > 0.f, "the median edge distance is 0: the RBF similarity is undefined");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    StageScope scope(LUDVIG_STAGE_GRAPH, st);
    ++graph->val_version;
    const float inv = 1.0f / (bandwidth * graph->s_f * graph->s_f);
    k_rbf_reweight<<<grid_for(graph->n, 8), 256, 0, st>>>(graph->row_ptr, graph->col, graph->d2, unary, graph->n,
                                                          inv, binarize, row_normalize, graph->val);
    LV_LAUNCH();
    return LUDVIG_OK;
}

extern "C" ludvig_status ludvig_unary_anchor(ludvig_graph_t graph, const float* feats, int32_t df, const float* g0,
                                             float bandwidth, float* unary, void* stream) {
    LV_ARG(graph != nullptr, "graph is NULL");
    LV_ARG(graph->d2 != nullptr || graph->n == 0, "not an RBF graph (ludvig_graph_build_rbf)");
    LV_ARG(df >= 1 && df <= 4096, "df must be in [1, 4096]");
    LV_ARG(bandwidth > 0.f, "bandwidth must be positive");
    const int64_t n = graph->n;
    if (n == 0) return LUDVIG_OK;
    LV_ARG(feats != nullptr && g0 != nullptr && unary != nullptr, "NULL buffer");
    LV_ARG(graph->s_f > 0.f, "the median edge distance is 0: the RBF similarity is undefined");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Arena& ws = graph->ws;
    float *nrm, *fbar;
    double* acc;
    LV_TRY(ws.get("un.nrm", (size_t)n, &nrm));
    LV_TRY(ws.get("un.fbar", (size_t)df, &fbar));
    LV_TRY(ws.get("un.acc", (size_t)df, &acc));
    StageScope scope(LUDVIG_STAGE_GRAPH, st);
    LV_CUDA(cudaMemsetAsync(acc, 0, sizeof(double) * (size_t)df, st));
    k_norms<<<grid_for(n, 8), 256, 0, st>>>(feats, n, df, nrm);
    LV_LAUNCH();
    k_anchor_sum<<<(unsigned)ceil_div(n, kAnchorRows), 256, 0, st>>>(feats, nrm, g0, n, df, acc);
    LV_LAUNCH();
    k_anchor_finish<<<1, 256, 0, st>>>(acc, df, fbar);
    LV_LAUNCH();
    const float inv = 1.0f / (bandwidth * graph->s_f * graph->s_f);
    k_unary<<<grid_for(n, 8), 256, 0, st>>>(feats, nrm, fbar, n, df, inv, unary);
    LV_LAUNCH();
    return LUDVIG_OK;
}

extern "C" ludvig_status ludvig_topfrac_positive(ludvig_scene_t scene, const float* u, int32_t percent, float* g0,
                                                 void* stream) {
    LV_ARG(scene != nullptr, "scene is NULL");
    LV_ARG(percent >= 0 && percent <= 100, "percent must be in [0, 100]");
    const int64_t n = scene->n;
    if (n == 0) return LUDVIG_OK;
    LV_ARG(u != nullptr && g0 != nullptr, "NULL buffer");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Arena& ws = scene->ws;
    const int64_t npad = round_up(n, kRadixTile);
    uint32_t *keys, *vals, *keys2, *vals2;
    unsigned long long* npos;
    LV_TRY(ws.get("tf.keys", (size_t)npad, &keys));
    LV_TRY(ws.get("tf.vals", (size_t)npad, &vals));
    LV_TRY(ws.get("tf.keys2", (size_t)npad, &keys2));
    LV_TRY(ws.get("tf.vals2", (size_t)npad, &vals2));
    LV_TRY(ws.get("tf.npos", 1, &npos));
    StageScope scope(LUDVIG_STAGE_FILTER, st);
    LV_CUDA(cudaMemsetAsync(npos, 0, sizeof(unsigned long long), st));
    LV_CUDA(cudaMemsetAsync(g0, 0, sizeof(float) * (size_t)n, st));
    k_topfrac_keys<<<grid_for(npad, 256), 256, 0, st>>>(u, n, npad, keys, vals, npos);
    LV_LAUNCH();
    uint32_t *sk = keys, *sv = vals;
    LV_TRY(radix_sort_pairs(&sk, &sv, keys2, vals2, 1, npad, 32, ws, st));
    k_topfrac_mark<<<grid_for(n, 256), 256, 0, st>>>(sv, u, n, npos, percent, g0);
    LV_LAUNCH();
    return LUDVIG_OK;
}

extern "C" ludvig_status ludvig_reach_weight(ludvig_graph_t graph, const float* g0, int32_t dx, int32_t steps,
                                             const float* unary, float* h, void* stream) {
    LV_ARG(graph != nullptr, "graph is NULL");
    LV_ARG(dx >= 1 && dx <= 32, "dx must be in [1, 32]");
    LV_ARG(steps >= 0, "steps must be >= 0");
    const int64_t n = graph->n;
    if (n == 0) return LUDVIG_OK;
    LV_ARG(g0 != nullptr && h != nullptr, "NULL buffer");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint32_t *s0, *s1;
    LV_TRY(graph->ws.get("reach.s0", (size_t)n, &s0));
    LV_TRY(graph->ws.get("reach.s1", (size_t)n, &s1));
    StageScope scope(LUDVIG_STAGE_DIFFUSE, st);
    const bool copy = use_row_copy(graph, steps, kReachWeight);
    const int32_t* order = copy ? graph->inv : nullptr;   // the bits lie in the copy's order, or in the nodes'
    uint32_t* prp;
    int2* ent;
    if (copy) LV_TRY(ensure_pcsr(graph, st, &prp, &ent));
    k_reach_init<<<grid_for(n, 256), 256, 0, st>>>(g0, order, n, dx, s0);
    LV_LAUNCH();
    for (int t = 0; t < steps; ++t) {
        if (copy)
            k_reach_step<<<grid_for(n * 4, 256), 256, 0, st>>>(prp, ent, s0, n, s1);
        else
            k_reach_step_csr<<<grid_for(n * 8, 256), 256, 0, st>>>(graph->row_ptr, graph->col, graph->val, s0, n, s1);
        LV_LAUNCH();
        std::swap(s0, s1);
    }
    k_reach_out<<<grid_for(n * dx, 256), 256, 0, st>>>(s0, order, unary, n, dx, h);
    LV_LAUNCH();
    return LUDVIG_OK;
}
