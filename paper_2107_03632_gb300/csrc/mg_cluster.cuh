// V-cycle over the coarse levels by one thread-block cluster (sm_103a).
//
// A level of a few thousand nodes is a few microseconds of launch latency per
// operation and well under one of work; a hierarchy has six operations per
// level and most of its levels are that small.  Here one cluster of 16 (or 8)
// blocks runs every operation of the levels from `first` down and back up in
// one launch, with a hardware cluster barrier between operations instead of
// a launch.  Each row is summed by the same lanes in the same order as in
// the per-operation kernels (mg.cu), so the result has the same bits.
//
// Vectors written inside the launch are read past L1 (ld.cg): another block
// of the cluster, on another SM, wrote them.
#pragma once

#include "common.cuh"
#include "internal.cuh"

#include <cooperative_groups.h>

#include <type_traits>

namespace rbffd {

constexpr int kClThreads = 1024;
constexpr int kClMaxLevels = 12;

template <typename T>
struct ClLevel {
    int n, tpr, rtpr;  // rows; lanes per row of A and of the restriction into the next level
    const int64_t* row_ptr;
    const int* col;
    const T* val;
    const T* w;  // smoother weights Omega D^-1
    const int32_t* pidx;
    const T* pval;
    const int64_t* rrow;
    const int32_t* rcol;
    const T* rval;
    T *x, *t, *r, *b;
};

template <typename T>
struct ClCycle {
    int levels, nu;  // levels in lv; the last is solved with minv
    const T* minv;
    const int* flag;  // nothing is done while *flag != 0
    ClLevel<T> lv[kClMaxLevels];
};

template <typename T>
__device__ __forceinline__ T cl_fma(T a, T b, T c) {
    if constexpr (sizeof(T) == 8) return fma(a, b, c);
    else return fmaf(a, b, c);
}

// Rows i of n with TPR lanes each over the whole grid (one cluster); every
// lane of a warp makes the same number of trips.
#define CL_ROWS(TPR, N, i, valid, ...)                                           \
    {                                                                            \
        const int g0_ = (int)(blockIdx.x * blockDim.x + threadIdx.x) / (TPR);    \
        const int ng_ = (int)(gridDim.x * blockDim.x) / (TPR);                   \
        const int off_ = (threadIdx.x & 31) / (TPR);                             \
        for (int base_ = g0_ - off_; base_ < (N); base_ += ng_) {                \
            const int i = base_ + off_;                                          \
            const bool valid = i < (N);                                          \
            __VA_ARGS__                                                          \
        }                                                                        \
    }

// sum over row i of val * x(col), TPR lanes, the result in every lane.
template <typename T, int TPR, class X>
__device__ __forceinline__ T cl_row_sum(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                                        const T* __restrict__ val, X&& x, int row, int sub, bool valid) {
    int64_t a = 0, e = 0;
    if (valid) {
        a = __ldg(row_ptr + row);
        e = __ldg(row_ptr + row + 1);
    }
    T sum = T(0);
#pragma unroll 4
    for (int64_t k = a + sub; k < e; k += TPR) sum = cl_fma<T>(__ldg(val + k), x(__ldg(col + k)), sum);
#pragma unroll
    for (int o = TPR / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o, TPR);
    return sum;
}

// f with the lanes per row as a compile-time constant.
template <class F>
__device__ __forceinline__ void cl_tpr(int tpr, F&& f) {
    if (tpr == 8) f(std::integral_constant<int, 8>());
    else if (tpr == 4) f(std::integral_constant<int, 4>());
    else if (tpr == 2) f(std::integral_constant<int, 2>());
    else f(std::integral_constant<int, 1>());
}

// xo = xi + W (b - A xi); first: xi is W b (the sweep from zero), not stored.
template <typename T, bool FIRST, class B, class OUT>
__device__ __forceinline__ void cl_sweep(const ClLevel<T>& L, const T* xi, B&& b, OUT&& out) {
    cl_tpr(L.tpr, [&](auto tc) {
        constexpr int TPR = decltype(tc)::value;
        const int sub = threadIdx.x & (TPR - 1);
        CL_ROWS(TPR, L.n, i, valid, {
            auto at = [&](int j) -> T {
                if constexpr (FIRST) return __ldg(&RB_AT(L.w, j, L.n)) * b(j);
                else return __ldcg(&RB_AT(xi, j, L.n));
            };
            const T ax = cl_row_sum<T, TPR>(L.row_ptr, L.col, L.val, at, i, sub, valid);
            if (valid && sub == 0) out(i, cl_fma<T>(__ldg(L.w + i), b(i) - ax, at(i)));
        })
    });
}

// The V-cycle of the levels in c: right-hand side b0(i) of the first level
// (values of type T), its result through out0(i, x).  Every thread of the
// cluster calls it; `sync` is the cluster barrier.  Returns with the writes
// of the last sweep not yet ordered by a barrier.
template <typename T, class B0, class OUT0, class SYNC>
__device__ __forceinline__ void cl_cycle(const ClCycle<T>& c, B0&& b0, OUT0&& out0, SYNC&& sync) {
    const int last = c.levels - 1;
    const int gsize = (int)(gridDim.x * blockDim.x), gid = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    // down: pre-smoothing (after nu sweeps the iterate is in t for even nu,
    // x for odd), residual, restriction
    for (int l = 0; l < last; ++l) {
        const ClLevel<T>& L = c.lv[l];
        auto rhs = [&](int i) -> T { return l == 0 ? b0(i) : __ldcg(&RB_AT(L.b, i, L.n)); };
        T* cur = L.x;
        T* oth = L.t;
        if (c.nu == 1) {
            for (int i = gid; i < L.n; i += gsize) cur[i] = __ldg(L.w + i) * rhs(i);
        } else {
            cl_sweep<T, true>(L, (const T*)nullptr, rhs, [&](int i, T v) { oth[i] = v; });
            T* s = cur;
            cur = oth;
            oth = s;
        }
        sync();
        for (int k = 2; k < c.nu; ++k) {
            cl_sweep<T, false>(L, cur, rhs, [&](int i, T v) { oth[i] = v; });
            T* s = cur;
            cur = oth;
            oth = s;
            sync();
        }
        cl_tpr(L.tpr, [&](auto tc) {
            constexpr int TPR = decltype(tc)::value;
            const int sub = threadIdx.x & (TPR - 1);
            CL_ROWS(TPR, L.n, i, valid, {
                const T ax = cl_row_sum<T, TPR>(L.row_ptr, L.col, L.val,
                                                [&](int j) { return __ldcg(&RB_AT(cur, j, L.n)); }, i, sub, valid);
                if (valid && sub == 0) L.r[i] = rhs(i) - ax;
            })
        });
        sync();
        const ClLevel<T>& C = c.lv[l + 1];
        cl_tpr(L.rtpr, [&](auto tc) {
            constexpr int TPR = decltype(tc)::value;
            const int sub = threadIdx.x & (TPR - 1);
            CL_ROWS(TPR, C.n, i, valid, {
                const T v = cl_row_sum<T, TPR>(L.rrow, L.rcol, L.rval,
                                               [&](int j) { return __ldcg(&RB_AT(L.r, j, L.n)); }, i, sub, valid);
                if (valid && sub == 0) C.b[i] = v;
            })
        });
        sync();
    }
    // coarsest: x = Minv b, one warp per row
    {
        const ClLevel<T>& L = c.lv[last];
        const int lane = threadIdx.x & 31;
        for (int i = gid >> 5; i < L.n; i += gsize >> 5) {
            T acc = T(0);
            for (int j = lane; j < L.n; j += 32)
                acc = cl_fma<T>(__ldg(c.minv + (int64_t)i * L.n + j), last == 0 ? b0(j) : __ldcg(L.b + j), acc);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) {
                if (last == 0) out0(i, acc);
                else L.x[i] = acc;
            }
        }
    }
    // up: correction x += P e, post-smoothing
    for (int l = last - 1; l >= 0; --l) {
        sync();
        const ClLevel<T>& L = c.lv[l];
        const ClLevel<T>& C = c.lv[l + 1];
        // where the levels' iterates are: nu - 1 swaps before the coarse
        // correction, nu more after it (an odd number: in t), none at the coarsest
        const T* e = l + 1 == last ? C.x : C.t;
        T* cur = (c.nu & 1) ? L.x : L.t;
        T* oth = (c.nu & 1) ? L.t : L.x;
        auto rhs = [&](int i) -> T { return l == 0 ? b0(i) : __ldcg(&RB_AT(L.b, i, L.n)); };
        for (int i = gid; i < L.n; i += gsize) {
            const int32_t* ip = L.pidx + (int64_t)i * kMgK;
            const T* vp = L.pval + (int64_t)i * kMgK;
            T acc = __ldcg(cur + i);
#pragma unroll
            for (int j = 0; j < kMgK; ++j) acc = cl_fma<T>(__ldg(vp + j), __ldcg(&RB_AT(e, __ldg(ip + j), C.n)), acc);
            cur[i] = acc;
        }
        for (int k = 0; k < c.nu; ++k) {
            sync();
            if (l == 0 && k == c.nu - 1) {
                cl_sweep<T, false>(L, cur, rhs, out0);
            } else {
                cl_sweep<T, false>(L, cur, rhs, [&](int i, T v) { oth[i] = v; });
                T* s = cur;
                cur = oth;
                oth = s;
            }
        }
    }
}

// Levels [first, n_levels) of a hierarchy as a ClCycle; false where the
// hierarchy has too many.
template <typename T>
bool cl_make(const MgHierarchy& h, int first, const int* flag, ClCycle<T>* out);

// Blocks per cluster that the device schedules for `kernel` with kClThreads
// threads: 16 (beyond the portable 8), 8, or 0; cached per kernel.
int cl_cluster_size(const void* kernel);

}  // namespace rbffd
