// Sums over the rows of a large CSR matrix, 32 rows per warp (sm_103a).
//
// TPR lanes share a row's entries.  Reducing and finishing one row per group
// at a time leaves the finish (and log2 TPR additions) to one lane in TPR,
// but a warp instruction with one active lane costs what a full one does, and
// FP64 runs at 2 lanes per cycle and SM: a sweep over rows of 30 entries with
// two lanes each is 30 + 2 + 2 x 3 FP64 lane slots per row.  Here each group
// sums TPR rows and exchanges partial sums so that lane `sub` ends with the
// whole sum of row `sub`: TPR - 1 additions per TPR rows, and every lane
// finishes a row (30 + 1 + 3).  The order of summation, and so the bits, are
// those of one row per group with the same TPR.
#pragma once

#include "common.cuh"

namespace rbffd {

__device__ __forceinline__ float fma_of(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_of(double a, double b, double c) { return fma(a, b, c); }

// s[j]: this lane's part of the sum of the group's row j; returns the sum of
// row `sub`.
template <typename T, int TPR>
__device__ __forceinline__ T rows32_exchange(T (&s)[TPR], int sub) {
#pragma unroll
    for (int o = TPR / 2; o > 0; o >>= 1) {
        // keep the half of the rows that has the lane's bit o, send the other
        const bool up = (sub & o) != 0;
#pragma unroll
        for (int j = 0; j < o; ++j) {
            const T keep = up ? s[j + o] : s[j], send = up ? s[j] : s[j + o];
            s[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return s[0];
}

// f(i, (A x)_i) in one lane per row, from a grid of full warps (one thread
// per row, or fewer and several passes).
template <typename T, int TPR, class F>
__device__ __forceinline__ void rows32(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                                       const T* __restrict__ val, Live<T> x, int64_t nx, int64_t N, F&& f) {
    (void)nx;  // length of x: bound of the checked build's tests
    constexpr int G = 32 / TPR;
    const int lane = (int)(threadIdx.x & 31), sub = lane & (TPR - 1), g = lane / TPR;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~(int64_t)31; base < N; base += step) {
        T s[TPR];
#pragma unroll
        for (int j = 0; j < TPR; ++j) {
            const int64_t i = base + j * G + g;
            int64_t a = 0, e = 0;
            if (i < N) {
                a = __ldg(row_ptr + i);
                e = __ldg(row_ptr + i + 1);
            }
            T t = T(0);
#pragma unroll 4
            for (int64_t k = a + sub; k < e; k += TPR)
                t = fma_of(__ldg(val + k), RB_AT(x, __ldg(col + k), nx), t);
            s[j] = t;
        }
        const T t = rows32_exchange<T, TPR>(s, sub);
        const int64_t row = base + sub * G + g;
        if (row < N) f(row, t);
    }
}

// The same with a row's first 4 TPR entries loaded while the gathers of x of
// the row before are in flight, so that eight lanes per row (a quarter of the
// L1 wavefronts of two: 16-byte pieces of 16 rows are 16 lines per load of 32
// entries, 64-byte pieces of 4 rows are 4) are not a round trip per four
// entries.  For float32: in FP64 the 64 registers more cost what it gives.
// The gathers are unconditional (x_0 past a row's end, not used): as
// conditional ordinary loads they are not all in flight before the next row's
// loads (1M rows of 30 entries: a sweep 72 us, now 60; mixed solve 20.6 -> 19.7).
template <typename T, int TPR, class F>
__device__ __forceinline__ void rows32_ahead(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                                             const T* __restrict__ val, Live<T> x, int64_t nx, int64_t N, F&& f) {
    (void)nx;  // length of x: bound of the checked build's tests
    constexpr int G = 32 / TPR, U = 4;
    const int lane = (int)(threadIdx.x & 31), sub = lane & (TPR - 1), g = lane / TPR;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~(int64_t)31;
    if (base >= N) return;
    int64_t p = 0, q = 0;  // entry bounds of row base + lane (empty past the end)
    if (base + lane < N) {
        p = __ldg(row_ptr + base + lane);
        q = __ldg(row_ptr + base + lane + 1);
    }
    int64_t k, cnt;  // the loaded row: this lane's first entry, entries from there to the row's end
    int c[U];
    T v[U];
    auto head = [&](int j) {
        const int64_t a = __shfl_sync(0xffffffffu, p, j * G + g);
        k = a + sub;
        cnt = __shfl_sync(0xffffffffu, q, j * G + g) - k;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool in = u * TPR < cnt;
            c[u] = in ? __ldg(col + k + u * TPR) : 0;
            v[u] = in ? __ldg(val + k + u * TPR) : T(0);
        }
    };
    head(0);
    for (; base < N; base += step) {
        T s[TPR];
        const int64_t next = base + step + lane;
        int64_t pn = 0, qn = 0;  // the next 32 rows' bounds
        if (next < N) {
            pn = __ldg(row_ptr + next);
            qn = __ldg(row_ptr + next + 1);
        }
#pragma unroll
        for (int j = 0; j < TPR; ++j) {
            T xv[U], w[U];
            const int64_t kj = k, cj = cnt;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                xv[u] = RB_AT(x, c[u], nx);
                w[u] = v[u];
            }
            if (j + 1 == TPR) {
                p = pn;
                q = qn;
            }
            head(j + 1 < TPR ? j + 1 : 0);
            T t = T(0);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (u * TPR < cj) t = fma_of(w[u], xv[u], t);
            for (int64_t o = U * TPR; o < cj; o += TPR)
                t = fma_of(__ldg(val + kj + o), RB_AT(x, __ldg(col + kj + o), nx), t);
            s[j] = t;
        }
        const T t = rows32_exchange<T, TPR>(s, sub);
        const int64_t row = base + sub * G + g;
        if (row < N) f(row, t);
    }
}

}  // namespace rbffd
