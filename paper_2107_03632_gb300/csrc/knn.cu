// Exact n-nearest-neighbour stencils on a uniform cell grid (sm_103a).
//
// Sec. II, Eq. 1: the operator at node x is approximated from the values on
// N(x), the nodes neighbouring x; Sec. V takes the n nearest nodes.  Order of
// a stencil: key (d^2, j) ascending, where d^2 = dx*dx + dy*dy is rounded
// product by product (no FMA: __dmul_rn / __dadd_rn) and j is the caller's
// node index; node x itself comes first (d^2 = 0).
//
// Pipeline (all on the stream, no host synchronisation):
//   1. bounding box (block partials, then one block)         -> GridParams
//   2. histogram of the nodes' cells (atomics)
//   3. exclusive scan of the histogram                       -> cell_start
//   4. scatter nodes into cell order (double2, original index, fixed-point
//      coordinates)
//   5. one warp per query, in cell order: select the candidates by fixed-point
//      distances, rank the few that remain by their exact keys, once
//      (knn_fast_kernel, n <= 112)
//   6. the queries left, and n > 112: scan cells ring by ring around the
//      query's cell, keep a sorted top-n list of keys distributed over the
//      warp's registers (entry e at lane e%32, slot e/32), prune cells whose
//      nearest point cannot beat the current n-th key, and stop once the
//      unvisited region is provably farther than the n-th key.
// Distances are compared as the IEEE bit patterns of non-negative doubles
// (monotone as unsigned integers), so ranking never touches the FP64 pipe.
#include "common.cuh"
#include "internal.cuh"
#include "scan.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <cmath>
#include <map>
#include <mutex>

namespace rbffd {
namespace {

struct GridParams {
    double x0, y0;      // lower-left corner of the grid
    double cell;        // cell side
    double inv_cell;    // 1 / cell
    double margin;      // absolute slack for the geometric pruning tests
    double inv_fix;     // kFix / cell
    int G;              // cells per axis (G x G cells)
    int fast;           // the fixed-point search applies (see grid_setup_kernel)
};

// Fixed-point grid coordinates: units per cell.
constexpr int kFixBits = 12;
constexpr int kFix = 1 << kFixBits;
constexpr double kFastMinCell = 1e-140, kFastMaxSpan = 1e150;  // where it is used

struct Box {
    double mnx, mny, mxx, mxy;
    double odd;  // 1: a coordinate is not finite
};

constexpr int kBoxBlocks = 256;
constexpr int kBoxThreads = 256;

__global__ void __launch_bounds__(kBoxThreads) bbox_partial_kernel(const double2* __restrict__ xy, int64_t N,
                                                                   Box* __restrict__ part) {
    double mnx = INFINITY, mny = INFINITY, mxx = -INFINITY, mxy = -INFINITY, odd = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 p = xy[i];
        mnx = fmin(mnx, p.x);
        mny = fmin(mny, p.y);
        mxx = fmax(mxx, p.x);
        mxy = fmax(mxy, p.y);
        if (!finite64(p.x) || !finite64(p.y)) odd = 1.0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        odd = fmax(odd, __shfl_xor_sync(0xffffffffu, odd, o));
        mnx = fmin(mnx, __shfl_xor_sync(0xffffffffu, mnx, o));
        mny = fmin(mny, __shfl_xor_sync(0xffffffffu, mny, o));
        mxx = fmax(mxx, __shfl_xor_sync(0xffffffffu, mxx, o));
        mxy = fmax(mxy, __shfl_xor_sync(0xffffffffu, mxy, o));
    }
    __shared__ Box sh[kBoxThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) RB_AT(sh, wid, kBoxThreads / 32) = Box{mnx, mny, mxx, mxy, odd};
    __syncthreads();
    if (threadIdx.x == 0) {
        Box r = sh[0];
        for (int k = 1; k < kBoxThreads / 32; ++k) {
            r.mnx = fmin(r.mnx, sh[k].mnx);
            r.mny = fmin(r.mny, sh[k].mny);
            r.mxx = fmax(r.mxx, sh[k].mxx);
            r.mxy = fmax(r.mxy, sh[k].mxy);
            r.odd = fmax(r.odd, sh[k].odd);
        }
        part[blockIdx.x] = r;
    }
}

// One block, one partial box per thread (a serial pass over the 256 partials
// by one thread took 65 us, as long as 300k queries of the search itself).
__global__ void __launch_bounds__(kBoxBlocks) grid_setup_kernel(const Box* __restrict__ part, int G, GridParams* gp) {
    static_assert(kBoxBlocks % 32 == 0, "whole warps reduce the partials");
    Box r = part[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        r.mnx = fmin(r.mnx, __shfl_xor_sync(0xffffffffu, r.mnx, o));
        r.mny = fmin(r.mny, __shfl_xor_sync(0xffffffffu, r.mny, o));
        r.mxx = fmax(r.mxx, __shfl_xor_sync(0xffffffffu, r.mxx, o));
        r.mxy = fmax(r.mxy, __shfl_xor_sync(0xffffffffu, r.mxy, o));
        r.odd = fmax(r.odd, __shfl_xor_sync(0xffffffffu, r.odd, o));
    }
    __shared__ Box sh[kBoxBlocks / 32];
    if ((threadIdx.x & 31) == 0) RB_AT(sh, threadIdx.x >> 5, kBoxBlocks / 32) = r;
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int k = 1; k < kBoxBlocks / 32; ++k) {
        r.mnx = fmin(r.mnx, sh[k].mnx);
        r.mny = fmin(r.mny, sh[k].mny);
        r.mxx = fmax(r.mxx, sh[k].mxx);
        r.mxy = fmax(r.mxy, sh[k].mxy);
        r.odd = fmax(r.odd, sh[k].odd);
    }
    double x0 = r.mnx, y0 = r.mny;
    double span = fmax(r.mxx - r.mnx, r.mxy - r.mny);
    // The fixed-point search takes the nearest points of the plane, the order
    // of a stencil is that of the rounded d^2.  The two agree while every d^2
    // it can meet is far inside the normal range: from the square of one unit
    // (cell / kFix), where an underflow would turn the geometry's order into
    // ties that the index decides, to that of the whole span.
    const bool in_range = r.odd == 0.0 && x0 <= r.mxx && y0 <= r.mxy && span < kFastMaxSpan;
    if (!(x0 > -INFINITY && x0 < INFINITY)) x0 = 0.0;  // no finite point
    if (!(y0 > -INFINITY && y0 < INFINITY)) y0 = 0.0;
    if (!(span > 0.0 && span < INFINITY)) span = 1.0;    // single point / degenerate
    GridParams p;
    p.x0 = x0;
    p.y0 = y0;
    p.cell = span / G;
    p.inv_cell = G / span;
    p.margin = 1e-12 * (span + fabs(x0) + fabs(y0));
    p.inv_fix = p.inv_cell * kFix;
    p.G = G;
    p.fast = in_range && p.cell > kFastMinCell ? 1 : 0;
    *gp = p;
}

// Coordinate in units of cell / kFix, rounded down and saturating (fix_cell
// clamps whatever a NaN becomes).
__device__ __forceinline__ int fix_coord(double v, double v0, double inv_fix) {
    return __double2int_rd((v - v0) * inv_fix);
}
// Cell of a fixed-point coordinate, clamped to the grid: floor of the exact
// product, since rounding down to kFix units and then to cells is rounding
// down to cells.
__device__ __forceinline__ int fix_cell(int u, int G) { return min(max(u >> kFixBits, 0), G - 1); }

__device__ __forceinline__ int cell_coord(double v, double v0, double inv, int G) {
    const double t = floor((v - v0) * inv);
    // NaN and out-of-range values are clamped (NaN compares false).
    int c = (t >= 0.0) ? ((t < (double)G) ? (int)t : G - 1) : 0;
    return c;
}

__global__ void cell_count_kernel(const double2* __restrict__ xy, int64_t N, const GridParams* __restrict__ gp,
                                  int* __restrict__ counts) {
    const GridParams p = *gp;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 q = xy[i];
        const int cx = fix_cell(fix_coord(q.x, p.x0, p.inv_fix), p.G);
        const int cy = fix_cell(fix_coord(q.y, p.y0, p.inv_fix), p.G);
        atomicAdd(&RB_AT(counts, cy * p.G + cx, p.G * p.G), 1);
    }
}

// counts[key] runs from the cell size down to 1, so positions fill
// [start[key], start[key+1]) exactly once.  Order inside a cell is arbitrary;
// stencils do not depend on it because the ranking key is a total order.
// su: the low 16 bits of both fixed-point coordinates (position modulo 16
// cells).  cells_of (may be NULL): the cell (cy << 16 | cx) of point i goes
// to cells_of[i * stride] (the first entry of its output row, which its query
// overwrites).
__global__ void cell_scatter_kernel(const double2* __restrict__ xy, int64_t N, const GridParams* __restrict__ gp,
                                    const int* __restrict__ cell_start, int* __restrict__ counts,
                                    double2* __restrict__ sxy, int* __restrict__ sorig, unsigned* __restrict__ su,
                                    int* __restrict__ cells_of, int stride) {
    const GridParams p = *gp;
    const int64_t cells = (int64_t)p.G * p.G;
    (void)cells;  // bound of the checked build's tests
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 q = xy[i];
        const int ux = fix_coord(q.x, p.x0, p.inv_fix), uy = fix_coord(q.y, p.y0, p.inv_fix);
        const int cx = fix_cell(ux, p.G), cy = fix_cell(uy, p.G);
        const int key = cy * p.G + cx;
        const int pos = RB_AT(cell_start, key + 1, cells + 1) - atomicSub(&RB_AT(counts, key, cells), 1);
        RB_AT(sxy, pos, N) = q;
        RB_AT(sorig, pos, N) = (int)i;
        RB_AT(su, pos, N) = ((unsigned)uy << 16) | ((unsigned)ux & 0xffffu);
        if (cells_of) cells_of[i * stride] = cy << 16 | cx;
    }
}

struct Key {
    unsigned long long d;  // bit pattern of d^2 (non-negative double)
    unsigned int j;        // caller index
};

__device__ __forceinline__ bool key_less(unsigned long long ad, unsigned int aj, unsigned long long bd,
                                         unsigned int bj) {
    return (ad < bd) || (ad == bd && aj < bj);
}

__device__ __forceinline__ double key_d2(unsigned long long d) { return __longlong_as_double((long long)d); }

// Distributed sorted list of SLOTS*32 keys (entry e: lane e & 31, slot e >> 5).
template <int SLOTS>
struct TopList {
    unsigned long long d[SLOTS];
    unsigned int j[SLOTS];

    __device__ __forceinline__ void init() {
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) {
            d[s] = ~0ull;
            j[s] = ~0u;
        }
    }

    // Insert key (kd, kj), which is known to be smaller than entry n-1.
    __device__ __forceinline__ void insert(unsigned long long kd, unsigned int kj, int lane) {
        int p = 0;
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) p += __popc(__ballot_sync(0xffffffffu, key_less(d[s], j[s], kd, kj)));
        unsigned long long up_d[SLOTS];
        unsigned int up_j[SLOTS];
        unsigned long long top_d[SLOTS];
        unsigned int top_j[SLOTS];
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) {
            up_d[s] = __shfl_up_sync(0xffffffffu, d[s], 1);
            up_j[s] = __shfl_up_sync(0xffffffffu, j[s], 1);
            top_d[s] = __shfl_sync(0xffffffffu, d[s], 31);
            top_j[s] = __shfl_sync(0xffffffffu, j[s], 31);
        }
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) {
            const int e = s * 32 + lane;
            unsigned long long pd;
            unsigned int pj;
            if (lane > 0) {
                pd = up_d[s];
                pj = up_j[s];
            } else if (s > 0) {
                pd = top_d[s > 0 ? s - 1 : 0];
                pj = top_j[s > 0 ? s - 1 : 0];
            } else {
                pd = ~0ull;
                pj = ~0u;
            }
            if (e == p) {
                d[s] = kd;
                j[s] = kj;
            } else if (e > p) {
                d[s] = pd;
                j[s] = pj;
            }
        }
    }

    // Merge a batch of 32 keys (one per lane, sorted ascending over the
    // lanes): afterwards the list holds the SLOTS*32 smallest of the list
    // and the batch, sorted.  Classic bitonic merge: the last slot against
    // the reversed batch keeps the smaller key of each pair, which leaves the
    // list a bitonic sequence of the smallest keys; compare-exchange stages of
    // halving distance then sort it (between slots in registers, within a
    // slot by shuffles).
    __device__ __forceinline__ void merge(unsigned long long bd, unsigned int bj, int lane) {
        const unsigned long long rd = __shfl_sync(0xffffffffu, bd, 31 - lane);
        const unsigned int rj = __shfl_sync(0xffffffffu, bj, 31 - lane);
        if (key_less(rd, rj, d[SLOTS - 1], j[SLOTS - 1])) {
            d[SLOTS - 1] = rd;
            j[SLOTS - 1] = rj;
        }
#pragma unroll
        for (int h = SLOTS / 2; h > 0; h >>= 1)  // distance 32 h: slot s against slot s + h
#pragma unroll
            for (int s = 0; s < SLOTS; ++s)
                if ((s & h) == 0 && key_less(d[s + h], j[s + h], d[s], j[s])) {
                    const unsigned long long td = d[s];
                    const unsigned int tj = j[s];
                    d[s] = d[s + h];
                    j[s] = j[s + h];
                    d[s + h] = td;
                    j[s + h] = tj;
                }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const bool lower = (lane & o) == 0;
#pragma unroll
            for (int s = 0; s < SLOTS; ++s) {
                const unsigned long long pd = __shfl_xor_sync(0xffffffffu, d[s], o);
                const unsigned int pj = __shfl_xor_sync(0xffffffffu, j[s], o);
                if (lower ? key_less(pd, pj, d[s], j[s]) : key_less(d[s], j[s], pd, pj)) {
                    d[s] = pd;
                    j[s] = pj;
                }
            }
        }
    }

    // Entry e broadcast to the warp.
    __device__ __forceinline__ void get(int e, unsigned long long& od, unsigned int& oj) const {
        const int s = e >> 5, l = e & 31;
        unsigned long long v = d[0];
        unsigned int w = j[0];
#pragma unroll
        for (int t = 1; t < SLOTS; ++t)
            if (t == s) {
                v = d[t];
                w = j[t];
            }
        od = __shfl_sync(0xffffffffu, v, l);
        oj = __shfl_sync(0xffffffffu, w, l);
    }
};

// Ascending bitonic sort of 32 keys, one per lane.
__device__ __forceinline__ void warp_sort32(unsigned long long& d, unsigned int& j, int lane) {
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
        for (int o = k >> 1; o > 0; o >>= 1) {
            const unsigned long long pd = __shfl_xor_sync(0xffffffffu, d, o);
            const unsigned int pj = __shfl_xor_sync(0xffffffffu, j, o);
            const bool up = (lane & k) == 0 || k == 32;  // this run ascending
            const bool lower = (lane & o) == 0;
            if (lower == up ? key_less(pd, pj, d, j) : key_less(d, j, pd, pj)) {
                d = pd;
                j = pj;
            }
        }
    }
}

// Batches with more accepted candidates than this are sorted and merged into
// the list at once; fewer are inserted one by one (4M nodes, n = 56: 24.9 /
// 24.4 / 24.0 / 23.6 / 23.1 ms of stencils with 1 / 2 / 4 / 8 / 16 here,
// 34.3 ms inserting every candidate).
constexpr int kMergeBatch = 16;

// Queries: the indexed points themselves in cell order (qxy = sxy, qorig =
// sorig: stencils), or separate points in their own order (qorig = NULL:
// output row q).
//
// Search order: first the (2 R0 + 1)^2 block of cells around the query's
// cell, R0 chosen on the host so that the block holds about n points, row
// by row from the query's row outwards -- the points of a row of cells are
// contiguous in the cell-sorted arrays, so a warp reads 32 candidates at a
// time instead of one cell's few; then rings of cells until the gap to the
// unvisited cells exceeds the n-th key.  The candidate keys (d^2, index) are
// FP64 and exact; the pruning bounds for groups of cells are FP32, taken
// relative to the query and shrunk by a slack, so they only ever keep a cell
// that an exact bound would have skipped.  (On this chip the FP64 units issue
// 2 lanes per clock per SM: per-cell FP64 bounds and one-cell candidate
// batches made the search FP64-bound.)
//
// chunk > 0: only the queries that knn_fast_kernel left (first entry kLeft),
// a warp looks at `chunk` queries, every Nq / chunk-th one: those left lie
// together (they are in cell order, and crowded cells leave all theirs), and
// so a warp does not get 32 of them (1M nodes crowded towards a point, n = 45:
// 7.9 ms with consecutive queries, 2.8 so, 7.0 with the list search of all);
// chunk = 0: every query, one per warp.
constexpr int kLeft = -1;
template <int SLOTS>
__device__ __forceinline__ void knn_query(const double2* __restrict__ sxy, const int* __restrict__ sorig,
                                          const int* __restrict__ cell_start, int Np, const GridParams& p, int Nq,
                                          const double2* __restrict__ qxy, const int* __restrict__ qorig, int n,
                                          int R0, int* __restrict__ idx, int q, int lane);
template <int SLOTS>
__global__ void __launch_bounds__(256) knn_kernel(const double2* __restrict__ sxy, const int* __restrict__ sorig,
                                                  const int* __restrict__ cell_start, int Np,
                                                  const GridParams* __restrict__ gp, int Nq,
                                                  const double2* __restrict__ qxy, const int* __restrict__ qorig,
                                                  int n, int R0, int* __restrict__ idx, int chunk) {
    const int lane = threadIdx.x & 31;
    const int warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const GridParams p = *gp;
    if (chunk == 0) {
        if (warp < Nq) knn_query<SLOTS>(sxy, sorig, cell_start, Np, p, Nq, qxy, qorig, n, R0, idx, warp, lane);
        return;
    }
    const int warps = (Nq + chunk - 1) / chunk;
    if (warp >= warps) return;
    const int64_t q = warp + (int64_t)lane * warps;
    bool left = false;
    if (lane < chunk && q < Nq) left = idx[(int64_t)(qorig ? qorig[q] : (int)q) * n] == kLeft;
    for (unsigned m = __ballot_sync(0xffffffffu, left); m; m &= m - 1)
        knn_query<SLOTS>(sxy, sorig, cell_start, Np, p, Nq, qxy, qorig, n, R0, idx,
                         warp + (__ffs(m) - 1) * warps, lane);
}

template <int SLOTS>
__device__ __forceinline__ void knn_query(const double2* __restrict__ sxy, const int* __restrict__ sorig,
                                          const int* __restrict__ cell_start, int Np, const GridParams& p, int Nq,
                                          const double2* __restrict__ qxy, const int* __restrict__ qorig, int n,
                                          int R0, int* __restrict__ idx, int q, int lane) {
    const double2 Q = qxy[q];
    const int qo = qorig ? qorig[q] : q;
    const int G = p.G;
    (void)Np;  // bound of the checked build's tests
    const int cx = cell_coord(Q.x, p.x0, p.inv_cell, G);
    const int cy = cell_coord(Q.y, p.y0, p.inv_cell, G);

    TopList<SLOTS> top;
    top.init();
    unsigned long long thr_d = ~0ull;  // key of entry n-1 (all-ones: list not full)
    unsigned int thr_j = ~0u;

    // one batch: lane's candidate at sorted position jj (none: jj < 0)
    auto eval = [&](int jj) {
        unsigned long long kd = ~0ull;
        unsigned int kj = ~0u;
        if (jj >= 0) {
            const double2 P = RB_AT(sxy, jj, Np);
            const double dx = __dadd_rn(P.x, -Q.x);
            const double dy = __dadd_rn(P.y, -Q.y);
            const double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
            kd = (unsigned long long)__double_as_longlong(d2) & 0x7fffffffffffffffull;
            kj = (unsigned int)RB_AT(sorig, jj, Np);
        }
        const bool acc = key_less(kd, kj, thr_d, thr_j);
        unsigned int m = __ballot_sync(0xffffffffu, acc);
        if (__popc(m) > kMergeBatch) {  // many at once (the first batches of a query)
            unsigned long long md = acc ? kd : ~0ull;
            unsigned int mj = acc ? kj : ~0u;
            warp_sort32(md, mj, lane);
            top.merge(md, mj, lane);
            top.get(n - 1, thr_d, thr_j);
            return;
        }
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            const unsigned long long id = __shfl_sync(0xffffffffu, kd, src);
            const unsigned int ij = __shfl_sync(0xffffffffu, kj, src);
            if (!key_less(id, ij, thr_d, thr_j)) continue;  // threshold moved
            top.insert(id, ij, lane);
            top.get(n - 1, thr_d, thr_j);
        }
    };
    // candidates at sorted positions [beg, end)
    auto scan = [&](int beg, int end) {
        for (int base = beg; base < end; base += 32) eval(base + lane < end ? base + lane : -1);
    };
    // FP32 lower bound of d^2 from the query to the cells [xl, xh] of row yy,
    // relative to the query's cell corner (exact in FP64), shrunk by a slack;
    // true when all of them lie beyond the n-th key
    const float fx = (float)(Q.x - (p.x0 + cx * p.cell));
    const float fy = (float)(Q.y - (p.y0 + cy * p.cell));
    const float cf = (float)p.cell;
    const float slack = (float)p.margin + 1e-4f * cf;
    auto beyond = [&](int xl, int xh, int yy) -> bool {
        if (thr_d == ~0ull) return false;
        const float lx = (float)(xl - cx) * cf - fx, hx = (float)(xh + 1 - cx) * cf - fx;
        const float ly = (float)(yy - cy) * cf - fy, hy = ly + cf;
        const float dx = fmaxf(fmaxf(fmaxf(lx, -hx), 0.f) - slack, 0.f);
        const float dy = fmaxf(fmaxf(fmaxf(ly, -hy), 0.f) - slack, 0.f);
        return (dx * dx + dy * dy) * (1.0f - 1e-4f) > (float)key_d2(thr_d);
    };
    auto row_range = [&](int xl, int xh, int yy) {
        if (!beyond(xl, xh, yy))
            scan(RB_AT(cell_start, yy * G + xl, G * G + 1), RB_AT(cell_start, yy * G + xh + 1, G * G + 1));
    };
    // true when the cells within ring r hold the n nearest: whole grid
    // visited, or the gap from Q to the unvisited cells exceeds the n-th key
    auto done = [&](int r) -> bool {
        if (cx - r <= 0 && cy - r <= 0 && cx + r >= G - 1 && cy + r >= G - 1) return true;
        if (thr_d == ~0ull) return false;
        double gap = INFINITY;
        if (cx - r > 0) gap = fmin(gap, Q.x - (p.x0 + (cx - r) * p.cell));
        if (cx + r < G - 1) gap = fmin(gap, (p.x0 + (cx + r + 1) * p.cell) - Q.x);
        if (cy - r > 0) gap = fmin(gap, Q.y - (p.y0 + (cy - r) * p.cell));
        if (cy + r < G - 1) gap = fmin(gap, (p.y0 + (cy + r + 1) * p.cell) - Q.y);
        gap -= p.margin;
        return gap > 0.0 && gap * gap > key_d2(thr_d);
    };

    // the block, rows from the query's outwards, their candidates packed into
    // batches of 32 across row boundaries (a row is tested against the n-th
    // key when the batch that would start it is filled)
    {
        const int xlo = max(cx - R0, 0), xhi = min(cx + R0, G - 1);
        int k = 0, sb = 0, sl = 0;  // next row; the current row's unread range [sb, sb + sl)
        for (;;) {
            int mine = -1, fill = 0;
            while (fill < 32) {
                if (sl == 0) {
                    bool got = false;
                    while (k <= 2 * R0 && !got) {
                        const int yy = cy + ((k & 1) ? -((k + 1) >> 1) : (k >> 1));
                        ++k;
                        if (yy < 0 || yy >= G || beyond(xlo, xhi, yy)) continue;
                        sb = RB_AT(cell_start, yy * G + xlo, G * G + 1);
                        sl = RB_AT(cell_start, yy * G + xhi + 1, G * G + 1) - sb;
                        got = sl > 0;
                    }
                    if (!got) break;
                }
                const int t = min(32 - fill, sl);
                if (lane >= fill && lane < fill + t) mine = sb + lane - fill;
                sb += t;
                sl -= t;
                fill += t;
            }
            if (fill == 0) break;
            eval(mine);
        }
    }
    // then rings: the two edge rows as ranges, the side cells one by one
    for (int r = R0; !done(r) && r <= G; ) {
        ++r;
        for (int yy = cy - r; yy <= cy + r; ++yy) {
            if (yy < 0 || yy >= G) continue;
            if (yy == cy - r || yy == cy + r) {
                row_range(max(cx - r, 0), min(cx + r, G - 1), yy);
            } else {
                if (cx - r >= 0) row_range(cx - r, cx - r, yy);
                if (cx + r < G) row_range(cx + r, cx + r, yy);
            }
        }
    }

    RB_SPAN((int64_t)qo * n, n, (int64_t)Nq * n);
    int* out = idx + (int64_t)qo * n;
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
        const int e = s * 32 + lane;
        if (e < n) out[e] = (int)top.j[s];
    }
}

// ---------------------------------------------------------------------------
// The search of most queries (n <= 112): select first, sort once.
//
// A warp reads the cells that meet a disk around the query, its radius from
// the point count of the 3 x 3 cells there, and keeps the candidates' integer
// squared distances (fixed-point coordinates modulo 16 cells, 4 bytes per
// point) in registers, one row of cells per slot.  A threshold with n to
// 32 SLOTS candidates below it is found by counting (ballots); the fixed-point
// distances are within kErr units of the exact ones, so the candidates below
// the threshold plus 2 kErr contain the n nearest.  Only those are ranked:
// exact FP64 keys, one bitonic sort of 64-bit words (the leading bits of d^2
// and the candidate's number; equal leading bits: the full keys are sorted).
// A query whose candidates do not fit (strongly graded points, fewer than n
// points in reach) is left to knn_kernel.
// The block-first search above executes 5k to 9k warp instructions per query,
// most of them sorting and merging batches into the list; this one about 900.
// 300k nodes, n = 45: 1,603 -> 383 us; 1M nodes, n = 30: 4.9 -> 1.26 ms; the
// multigrid's coarse and interpolation searches there 5.5 -> 1.3 ms.
constexpr float kErr = 1.5f;     // > sqrt(2): each coordinate is rounded down by less than a unit
constexpr float kReach = 6.5f;   // cells: differences stay inside the 16-cell wrap

template <int SLOTS>
__device__ __forceinline__ void sort_words(unsigned long long (&key)[SLOTS], int lane) {
#pragma unroll
    for (int k = 2; k <= 32 * SLOTS; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
                const int js = j / 32;
#pragma unroll
                for (int s = 0; s < SLOTS; ++s)
                    if ((s & js) == 0) {
                        const bool up = ((s * 32) & k) == 0;
                        const unsigned long long a = key[s], b = key[s ^ js];
                        const bool swap = (a > b) == up;
                        key[s] = swap ? b : a;
                        key[s ^ js] = swap ? a : b;
                    }
            } else {
#pragma unroll
                for (int s = 0; s < SLOTS; ++s) {
                    const unsigned long long o = __shfl_xor_sync(0xffffffffu, key[s], j);
                    const bool low = ((lane & j) == 0) == (((s * 32 + lane) & k) == 0);  // this lane keeps the smaller
                    key[s] = (o < key[s]) == low ? o : key[s];
                }
            }
        }
    }
}

// The same network on full keys (d, j).
template <int SLOTS>
__device__ __noinline__ void sort_keys(unsigned long long* kd, unsigned* kj, int lane) {
    unsigned long long d[SLOTS];
    unsigned jj[SLOTS];
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
        d[s] = kd[s * 32 + lane];
        jj[s] = kj[s * 32 + lane];
    }
    for (int k = 2; k <= 32 * SLOTS; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
            for (int s = 0; s < SLOTS; ++s) {
                kd[s * 32 + lane] = d[s];
                kj[s * 32 + lane] = jj[s];
            }
            __syncwarp();
#pragma unroll
            for (int s = 0; s < SLOTS; ++s) {
                const int e = s * 32 + lane, o = e ^ j;
                const unsigned long long od = kd[o];
                const unsigned oj = kj[o];
                const bool low = ((e & j) == 0) == ((e & k) == 0);
                if (key_less(od, oj, d[s], jj[s]) == low && !(od == d[s] && oj == jj[s])) {
                    d[s] = od;
                    jj[s] = oj;
                }
            }
            __syncwarp();
        }
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
        kd[s * 32 + lane] = d[s];
        kj[s * 32 + lane] = jj[s];
    }
    __syncwarp();
}

// qxy NULL: the queries are the indexed points in cell order (row sorig[q],
// whose first entry holds the point's cell); else Nq separate points.
template <int SLOTS>
__global__ void __launch_bounds__(256) knn_fast_kernel(const double2* __restrict__ sxy,
                                                       const int* __restrict__ sorig,
                                                       const unsigned* __restrict__ su,
                                                       const int* __restrict__ cell_start, int Np,
                                                       const GridParams* __restrict__ gp, int Nq,
                                                       const double2* __restrict__ qxy, int n,
                                                       int* __restrict__ idx) {
    constexpr int CAP = 32 * SLOTS;          // candidates that are ranked
    constexpr int K = SLOTS == 4 ? 12 : SLOTS == 2 ? 10 : 8;  // register slots of candidates (rows of cells)
    constexpr int IB = SLOTS == 4 ? 7 : 6;   // bits of a candidate's number
    __shared__ unsigned long long sh_d[8][CAP];
    __shared__ unsigned sh_j[8][CAP];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int q = blockIdx.x * 8 + wid;
    if (q >= Nq) return;
    (void)Np;  // bound of the checked build's tests
    const GridParams p = *gp;
    const int G = p.G;
    const int qo = qxy ? q : sorig[q];
    int* out = idx + (int64_t)qo * n;
    RB_SPAN((int64_t)qo * n, n, (int64_t)Nq * n);
    int ux, uy;  // the query's fixed-point coordinates
    double2 Q;
    bool ok = p.fast != 0;
    if (qxy) {
        Q = qxy[q];
        ux = fix_coord(Q.x, p.x0, p.inv_fix);
        uy = fix_coord(Q.y, p.y0, p.inv_fix);
        // (far outside the grid, or not a number: the other search)
        ok = ok && ux > -8 * kFix && uy > -8 * kFix && ux < (G + 8) * kFix && uy < (G + 8) * kFix && finite64(Q.x) &&
             finite64(Q.y);
    } else {
        Q = sxy[q];
        const int cell = out[0], cx = cell & 0xffff, cy = cell >> 16;
        const unsigned s = su[q];
        ux = (cx << kFixBits) + (short)(unsigned short)(s - ((unsigned)cx << kFixBits));
        uy = (cy << kFixBits) + (short)(unsigned short)((s >> 16) - ((unsigned)cy << kFixBits));
    }
    const int* cs = cell_start;
    const int ncell = G * G + 1;
    (void)ncell;
    int cnt2 = 0;
    if (ok) {
        // density of the 3 x 3 cells around the query (cells outside the grid count as empty)
        int near = 0;
        {
            const int yy = (uy >> kFixBits) - 1 + lane, x0 = max((ux >> kFixBits) - 1, 0),
                      x1 = min((ux >> kFixBits) + 1, G - 1);
            if (lane < 3 && yy >= 0 && yy < G && x0 <= x1)
                near = RB_AT(cs, yy * G + x1 + 1, ncell) - RB_AT(cs, yy * G + x0, ncell);
            near = __reduce_add_sync(0xffffffffu, near);
        }
        const float area = 9.0f / (3.14159265f * (float)max(near, 1));  // cells per point, over pi
        float reach = sqrtf((float)n * area) * 1.08f + 0.12f;
        ok = false;
        for (int attempt = 0; attempt < 6 && reach <= kReach; ++attempt, reach *= 1.3f) {
            const float rf = reach * (float)kFix;
            const int ri = (int)rf + 2;
            const int y0 = (uy - ri) >> kFixBits, nr = ((uy + ri) >> kFixBits) - y0 + 1;
            // lane r: the columns of row y0 + r that the disk meets
            int beg = 0, len = 0;
            {
                const int yy = y0 + lane;
                if (lane < nr && yy >= 0 && yy < G) {
                    const int lo = yy << kFixBits;
                    const float dy = (float)max(0, max(lo - uy - 1, uy - lo - kFix));
                    const int half = (int)sqrtf(fmaxf(rf * rf - dy * dy, 0.f)) + 3;
                    const int xl = max((ux - half) >> kFixBits, 0), xh = min((ux + half) >> kFixBits, G - 1);
                    if (xl <= xh) {
                        beg = RB_AT(cs, yy * G + xl, ncell);
                        len = RB_AT(cs, yy * G + xh + 1, ncell) - beg;
                    }
                }
            }
            // candidates: one row (or 32 points of it) per slot
            unsigned d[K];
            int pos[K];
            int r = 0, off = 0;
#pragma unroll
            for (int s = 0; s < K; ++s) {
                pos[s] = -1;
                d[s] = 0xffffffffu;
                if (r < nr) {
                    const int b = __shfl_sync(0xffffffffu, beg, r) + off, l = __shfl_sync(0xffffffffu, len, r) - off;
                    if (lane < l) {
                        pos[s] = b + lane;
                        const unsigned v = RB_AT(su, b + lane, Np);
                        const int ex = (int)(short)(unsigned short)(v - (unsigned)ux);
                        const int ey = (int)(short)(unsigned short)((v >> 16) - (unsigned)uy);
                        d[s] = (unsigned)(ex * ex) + (unsigned)(ey * ey);
                    }
                    off += 32;
                    if (l <= 32) {
                        ++r;
                        off = 0;
                    }
                }
            }
            if (r < nr) break;  // more candidates than slots
            auto count = [&](unsigned T) -> int {
                int c = 0;
#pragma unroll
                for (int s = 0; s < K; ++s) c += __popc(__ballot_sync(0xffffffffu, d[s] <= T));
                return c;
            };
            const float tmax = (rf - 2.0f * kErr) * (rf - 2.0f * kErr);
            const float target = (float)n + fminf(5.0f, 0.4f * (float)(CAP - n));
            float lo = 0.f, hi = tmax, T = fminf(target * area * (float)kFix * (float)kFix, tmax);
            bool grow = false;
            for (int step = 0; step < 12; ++step) {
                const int c = count((unsigned)T);
                if (c < n) {
                    if (T >= tmax) {
                        grow = true;
                        break;
                    }
                    lo = T;
                } else {
                    // everything nearer than the n-th may be: sqrt(T) + 2 kErr
                    const float root = sqrtf(T) * 1.000001f + 2.0f * kErr + 0.5f;
                    const unsigned T2 = (unsigned)(root * root * 1.000001f) + 1u;
                    cnt2 = count(T2);
                    if (cnt2 <= CAP) {
                        int base = 0;
#pragma unroll
                        for (int s = 0; s < K; ++s) {
                            const bool in = d[s] <= T2;
                            const unsigned m = __ballot_sync(0xffffffffu, in);
                            if (in) RB_AT(sh_j[wid], base + __popc(m & ((1u << lane) - 1u)), CAP) = (unsigned)pos[s];
                            base += __popc(m);
                        }
                        ok = true;
                        break;
                    }
                    hi = T;
                }
                const float next = T * target / (float)max(c, 1);
                T = next > lo && next < hi ? next : (c < n && hi == tmax && next >= hi ? tmax : 0.5f * (lo + hi));
            }
            if (ok || !grow) break;
        }
    }
    if (!ok) {
        __syncwarp();
        if (lane == 0) out[0] = kLeft;
        return;
    }
    __syncwarp();
    // rank the candidates by their exact keys
    unsigned long long key[SLOTS];
    unsigned long long kd[SLOTS];
    unsigned kj[SLOTS];
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
        const int e = s * 32 + lane;
        kd[s] = ~0ull;
        kj[s] = ~0u;
        if (e < cnt2) {
            const int at = (int)sh_j[wid][e];
            const double2 P = RB_AT(sxy, at, Np);
            const double dx = __dadd_rn(P.x, -Q.x);
            const double dy = __dadd_rn(P.y, -Q.y);
            const double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
            kd[s] = (unsigned long long)__double_as_longlong(d2) & 0x7fffffffffffffffull;
            kj[s] = (unsigned)RB_AT(sorig, at, Np);
        }
        // ((d^2 bits << 1) without its last IB bits, number)
        key[s] = e < cnt2 ? (((kd[s] << 1) >> IB) << IB) | (unsigned long long)e : ~0ull;
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) sh_j[wid][s * 32 + lane] = kj[s];
    sort_words<SLOTS>(key, lane);
    // equal leading bits among the first n (or across its end): the full keys decide
    bool tie = false;
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
        unsigned long long nx = __shfl_down_sync(0xffffffffu, key[s], 1);
        if (s + 1 < SLOTS) {
            const unsigned long long first = __shfl_sync(0xffffffffu, key[s + 1 < SLOTS ? s + 1 : 0], 0);
            if (lane == 31) nx = first;
        } else if (lane == 31) {
            nx = ~0ull;
        }
        tie |= s * 32 + lane < n && s * 32 + lane + 1 < cnt2 && (key[s] >> IB) == (nx >> IB);
    }
    __syncwarp();
    if (__any_sync(0xffffffffu, tie)) {
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) sh_d[wid][s * 32 + lane] = kd[s];
        __syncwarp();
        sort_keys<SLOTS>(sh_d[wid], sh_j[wid], lane);
        for (int e = lane; e < n; e += 32) out[e] = (int)sh_j[wid][e];
        return;
    }
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
        const int e = s * 32 + lane;
        if (e < n) out[e] = (int)RB_AT(sh_j[wid], (int)(key[s] & ((1u << IB) - 1u)), CAP);
    }
}

// Block radius of the first search phase: about n points in (2 R0 + 1)^2
// cells at ~3 points per cell, plus half a cell.
int block_radius(int n) { return std::max(1, (int)std::ceil(std::sqrt((double)n / (3.0 * 3.14159265358979)) + 0.5)); }

// Cells per axis: about kOcc nodes per cell on a square domain, capped.
int grid_side(int64_t N, int n) {
    (void)n;
    const double occ = 3.0;
    int G = (int)std::ceil(std::sqrt((double)N / occ));
    if (G < 1) G = 1;
    if (G > 4096) G = 4096;
    return G;
}

struct KnnLayout {
    GridParams* gp;
    Box* part;
    unsigned* su;
    int* counts;
    int* cell_start;
    int* sums;
    double2* sxy;
    int* sorig;
    size_t bytes;
};

KnnLayout knn_layout(void* ws, int64_t N, int n) {
    const int G = grid_side(N, n);
    const int64_t cells = (int64_t)G * G;
    Carver c(ws);
    KnnLayout L;
    L.gp = c.take<GridParams>(1);
    L.part = c.take<Box>(kBoxBlocks);
    L.su = c.take<unsigned>(N);
    L.counts = c.take<int>(cells);
    L.cell_start = c.take<int>(cells + 1);
    L.sums = c.take<int>(scan_tiles(cells) + 1);
    L.sxy = c.take<double2>(N);
    L.sorig = c.take<int>(N);
    L.bytes = c.off;
    return L;
}

struct CountLoad {
    const int* counts;
    __device__ int operator()(int64_t i) const { return counts[i]; }
};

}  // namespace
}  // namespace rbffd

extern "C" size_t rbffd_stencils_workspace_size(int64_t N, int32_t n) {
    RBFFD_NVTX("rbffd_stencils_workspace_size");
    if (N <= 0 || n <= 0) return 0;
    return rbffd::knn_layout(nullptr, N, n).bytes;
}

extern "C" int rbffd_stencils(const double* xy, int64_t N, int32_t n, int32_t* idx, void* ws, size_t ws_bytes,
                              void* stream) {
    RBFFD_NVTX("rbffd_stencils");
    using namespace rbffd;
    if (!xy || !idx || N <= 0 || N > 0x7fffffffLL || n < 1 || n > RBFFD_MAX_STENCIL || (int64_t)n > N)
        return RBFFD_ERR_INVALID_ARG;
    if (((uintptr_t)xy & 15) != 0) return RBFFD_ERR_INVALID_ARG;
    if (!ws || ((uintptr_t)ws & (kAlign - 1)) != 0) return RBFFD_ERR_WORKSPACE;
    return knn_search(xy, N, nullptr, N, n, idx, ws, ws_bytes, as_stream(stream));
}

int rbffd::knn_search(const double* xy, int64_t N, const double* qxy, int64_t Nq, int32_t n, int32_t* idx, void* ws,
                      size_t ws_bytes, cudaStream_t st) {
    KnnLayout L = knn_layout(ws, N, n);
    if (ws_bytes < L.bytes) return RBFFD_ERR_WORKSPACE;
    if (Nq <= 0 || Nq > 0x7fffffffLL) return RBFFD_ERR_INVALID_ARG;
    const int G = grid_side(N, n);
    const int64_t cells = (int64_t)G * G;
    const double2* p = reinterpret_cast<const double2*>(xy);
    const int grid_pts = (int)std::min<int64_t>((N + 255) / 256, (int64_t)sm_count() * 8);

    bbox_partial_kernel<<<kBoxBlocks, kBoxThreads, 0, st>>>(p, N, L.part);
    grid_setup_kernel<<<1, kBoxBlocks, 0, st>>>(L.part, G, L.gp);
    RBFFD_CUDA_TRY(cudaMemsetAsync(L.counts, 0, sizeof(int) * cells, st));
    cell_count_kernel<<<grid_pts, 256, 0, st>>>(p, N, L.gp, L.counts);
    RBFFD_CUDA_TRY(exclusive_scan<int>(CountLoad{L.counts}, cells, L.cell_start, L.sums, L.cell_start + cells, st));
    cell_scatter_kernel<<<grid_pts, 256, 0, st>>>(p, N, L.gp, L.cell_start, L.counts, L.sxy, L.sorig, L.su,
                                                  qxy ? nullptr : idx, n);
    const double2* q = qxy ? reinterpret_cast<const double2*>(qxy) : L.sxy;
    const int* qo = qxy ? nullptr : L.sorig;
    const int R0 = block_radius(n);
    // ranked candidates: a few more than n, in whole warps
    const int blocks = (int)((Nq + 7) / 8);
    const bool fast = n <= 112;
    if (fast) {
        const double2* fq = reinterpret_cast<const double2*>(qxy);
        if (n <= 24)
            knn_fast_kernel<1><<<blocks, 256, 0, st>>>(L.sxy, L.sorig, L.su, L.cell_start, (int)N, L.gp, (int)Nq, fq, n, idx);
        else if (n <= 56)
            knn_fast_kernel<2><<<blocks, 256, 0, st>>>(L.sxy, L.sorig, L.su, L.cell_start, (int)N, L.gp, (int)Nq, fq, n, idx);
        else
            knn_fast_kernel<4><<<blocks, 256, 0, st>>>(L.sxy, L.sorig, L.su, L.cell_start, (int)N, L.gp, (int)Nq, fq, n, idx);
    }
    // queries per warp of the second pass: enough warps to fill the chip
    const int chunk = fast ? (int)std::min<int64_t>(32, std::max<int64_t>(1, Nq / 16384)) : 0;
    const int64_t warps = fast ? (Nq + chunk - 1) / chunk : Nq;
    const int rest = (int)((warps + 7) / 8);
    if (n <= 32)
        knn_kernel<1><<<rest, 256, 0, st>>>(L.sxy, L.sorig, L.cell_start, (int)N, L.gp, (int)Nq, q, qo, n, R0, idx, chunk);
    else if (n <= 64)
        knn_kernel<2><<<rest, 256, 0, st>>>(L.sxy, L.sorig, L.cell_start, (int)N, L.gp, (int)Nq, q, qo, n, R0, idx, chunk);
    else
        knn_kernel<4><<<rest, 256, 0, st>>>(L.sxy, L.sorig, L.cell_start, (int)N, L.gp, (int)Nq, q, qo, n, R0, idx, chunk);
    note_launches(fast ? 1 : 0);
    note_launches(5);  // bbox, setup, count, scatter, knn (+3 in the scan)
    RBFFD_LAUNCH_CHECK();
    return RBFFD_OK;
}

// ---------------------------------------------------------------------------
// Stencils without any device allocation, for callers that cannot call
// cudaMalloc (or any allocating routine) on the path -- for example code
// running inside a CUDA stream capture, a custom memory arena that owns all
// device memory, or a real-time loop that must not allocate -- and cannot
// provide a workspace either.  The scratch of rbffd_stencils lives in one
// file-scope device array sized for RBFFD_STENCILS_NOALLOC_MAX_NODES nodes;
// every GPU that loads this library keeps that array until the process
// exits.  In host code the array's name is only a host-side stand-in, so
// its device address is looked up with cudaGetSymbolAddress, with the
// device current, on the first call in each CUDA context; the address is
// cached under the context's unique ID (cuCtxGetId, reached through the
// runtime's driver entry points), so a context rebuilt after
// cudaDeviceReset gets a fresh lookup instead of a stale address.
static __device__ __align__(256) unsigned char g_stencils_noalloc_scratch[RBFFD_STENCILS_NOALLOC_SCRATCH_BYTES];

namespace {
std::mutex g_noalloc_mu;
std::map<unsigned long long, void*> g_noalloc_ptr;  // context ID -> device address of the array
PFN_cuCtxGetCurrent_v4000 g_ctx_current = nullptr;
PFN_cuCtxGetId_v12000 g_ctx_id = nullptr;

// Unique ID of the calling thread's current context; makes device `dev`'s
// primary context current first if the thread has none.
int current_context_id(int dev, unsigned long long* id) {
    if (!g_ctx_current || !g_ctx_id) {
        void* f1 = nullptr;
        void* f2 = nullptr;
        cudaDriverEntryPointQueryResult q1, q2;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 4000, cudaEnableDefault, &q1) != cudaSuccess ||
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) != cudaSuccess ||
            q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess || !f1 || !f2)
            return RBFFD_ERR_CUDA;
        g_ctx_current = reinterpret_cast<PFN_cuCtxGetCurrent_v4000>(f1);
        g_ctx_id = reinterpret_cast<PFN_cuCtxGetId_v12000>(f2);
    }
    CUcontext ctx = nullptr;
    if (g_ctx_current(&ctx) != CUDA_SUCCESS) return RBFFD_ERR_CUDA;
    if (!ctx) {
        if (cudaSetDevice(dev) != cudaSuccess || g_ctx_current(&ctx) != CUDA_SUCCESS || !ctx) return RBFFD_ERR_CUDA;
    }
    if (g_ctx_id(ctx, id) != CUDA_SUCCESS) return RBFFD_ERR_CUDA;
    return RBFFD_OK;
}
}  // namespace

extern "C" int rbffd_stencils_noalloc(const double* xy, int64_t N, int32_t n, int32_t* idx, void* stream) {
    RBFFD_NVTX("rbffd_stencils_noalloc");
    using namespace rbffd;
    if (N > RBFFD_STENCILS_NOALLOC_MAX_NODES || N <= 0) return RBFFD_ERR_INVALID_ARG;
    const size_t need = rbffd_stencils_workspace_size(N, n);
    if (need == 0 || need > (size_t)RBFFD_STENCILS_NOALLOC_SCRATCH_BYTES) return RBFFD_ERR_INVALID_ARG;
    int dev = 0;
    RBFFD_CUDA_TRY(cudaGetDevice(&dev));
    void* ptr = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        unsigned long long cid = 0;
        if (current_context_id(dev, &cid) != RBFFD_OK) return RBFFD_ERR_CUDA;
        auto it = g_noalloc_ptr.find(cid);
        if (it == g_noalloc_ptr.end()) {
            void* p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&p, g_stencils_noalloc_scratch);
            if (e != cudaSuccess || !p) {
                set_cuda_error(e != cudaSuccess ? e : cudaErrorInvalidSymbol);
                return RBFFD_ERR_CUDA;
            }
            it = g_noalloc_ptr.emplace(cid, p).first;
        }
        ptr = it->second;
    }
    // rbffd_stencils clears the cell histogram before use; everything else in
    // the scratch is overwritten, so leftovers of earlier calls do no harm
    return rbffd_stencils(xy, N, n, idx, ptr, (size_t)RBFFD_STENCILS_NOALLOC_SCRATCH_BYTES, stream);
}
