// Geometric multigrid preconditioner on RBF-FD node sets (sm_103a).
//
// The paper stops at an explicit time loop and names the implicit solve as
// the next step (Sec. VI); Jacobi-scaled BiCGSTAB on the RBF-FD Laplacian
// needs O(1/h) iterations (tens of thousands at 4M nodes).  This file builds
// a V-cycle whose every level is an RBF-FD discretisation of the same
// problem, made by this library's own stages:
//
//  * coarsening: the nodes of a level are binned on a uniform grid of side
//    c ~ 2x their mean spacing; each occupied cell keeps one node, a
//    Dirichlet node if the cell has one, else the node nearest the cell
//    centre (ties: lower index; one 64-bit atomicMin per node on the packed
//    key (interior?, d^2 to the centre, index), so the choice does not depend
//    on thread order).  c grows until at most half the nodes survive.
//    Survivors keep their relative order, so coarse indices inherit the
//    fine ordering's locality.
//  * coarse operator: stencils, Laplacian weights (PHS r^3 + monomials of
//    degree 2, n = 12) and the Dirichlet-row assembly of the fine problem,
//    rerun on the coarse nodes (rediscretisation; Sec. II Eq. 1, Sec. IV).
//  * prolongation P (ELL, 12 per row): PHS r^3 + degree-2 interpolation from
//    the 12 nearest coarse nodes; rows of Dirichlet nodes are zero (the
//    correction vanishes on the boundary).  Restriction R = (N_c / N_f) P^T
//    (a deterministic transpose), zero rows at coarse Dirichlet nodes.
//  * smoothing: nu damped Jacobi sweeps x += W (b - A x), W = Omega D^-1,
//    before and after the coarse correction.  The damping omega applies to
//    the interior rows; Dirichlet rows (identity rows of A, identity columns
//    of A^T) take omega = 1, so a cycle reproduces boundary data exactly.
//    With omega < 1 there, the Dirichlet values would come back off by
//    (1 - omega)^(2 nu), and the interior rows next to the boundary, whose
//    weights scale as 1/h^2, would turn that into a residual ~1/h^2 times
//    the data: at 1e6 nodes BiCGSTAB broke down in its first step on such
//    right-hand sides.  W is stored (per level, FP64 and float32) in place of
//    D^-1.  The coarsest level (<= 128 nodes) is
//    solved with its dense inverse (Gauss-Jordan with partial pivoting, one
//    block).
//
// A V-cycle is a fixed linear map (fixed sweeps, exact coarsest solve), so
// it can right-precondition BiCGSTAB.  It runs in FP64, or in float32 values
// and vectors (the mixed-precision solve: the preconditioner needs no FP64
// accuracy, the outer FP64 BiCGSTAB keeps the residual exact).
#include "common.cuh"
#include "csr_rows.cuh"
#include "internal.cuh"
#include "scan.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

namespace rbffd {

static_assert(sizeof(MgHierarchy) <= sizeof(rbffd_mg), "rbffd_mg is too small for the hierarchy");

namespace {

constexpr int kT = 256;

// Rows of a CSR matrix, TPR lanes per row; every lane of a warp runs the same
// number of trips (warp-uniform loop), so full-mask shuffles are safe.
#define MG_ROWS(TPR, N, i, valid, ...)                                                 \
    {                                                                                  \
        const int64_t g0_ = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / (TPR); \
        const int64_t ng_ = ((int64_t)gridDim.x * blockDim.x) / (TPR);                \
        const int64_t off_ = (threadIdx.x & 31) / (TPR);                              \
        for (int64_t base_ = g0_ - off_; base_ < (N); base_ += ng_) {                 \
            const int64_t i = base_ + off_;                                           \
            const bool valid = i < (N);                                               \
            __VA_ARGS__                                                               \
        }                                                                             \
    }

#define MG_ELEMS(N, i) \
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (N); i += (int64_t)gridDim.x * blockDim.x)

template <typename T>
__device__ __forceinline__ T fmaT(T a, T b, T c);
template <>
__device__ __forceinline__ double fmaT<double>(double a, double b, double c) {
    return fma(a, b, c);
}
template <>
__device__ __forceinline__ float fmaT<float>(float a, float b, float c) {
    return fmaf(a, b, c);
}

template <typename T, int TPR>
__device__ __forceinline__ T row_sum(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                                     const T* __restrict__ val, Live<T> x, int64_t nx, int64_t row, int sub,
                                     bool valid) {
    (void)nx;  // length of x: bound of the checked build's tests
    int64_t a = 0, e = 0;
    if (valid) {
        a = __ldg(row_ptr + row);
        e = __ldg(row_ptr + row + 1);
    }
    T sum = T(0);
#pragma unroll 4
    for (int64_t k = a + sub; k < e; k += TPR) sum = fmaT<T>(__ldg(val + k), RB_AT(x, __ldg(col + k), nx), sum);
#pragma unroll
    for (int o = TPR / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o, TPR);
    return sum;
}

__device__ __forceinline__ bool stopped(const int* flag) { return flag && *(volatile const int*)flag != 0; }

// The start of a lane's share of a row (its first U entries), loaded before
// the chain's previous kernel has completed; sum() is row_sum with them.
template <typename T, int TPR>
struct RowHead {
    static constexpr int U = TPR >= 4 ? 4 : 6;
    int64_t a, e;
    int c[U];
    T v[U];
    __device__ __forceinline__ void load(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                                         const T* __restrict__ val, int64_t row, int sub, bool valid) {
        a = e = 0;
        if (valid) {
            a = __ldg(row_ptr + row);
            e = __ldg(row_ptr + row + 1);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t k = a + sub + u * TPR;
            c[u] = k < e ? __ldg(col + k) : 0;
            v[u] = k < e ? __ldg(val + k) : T(0);
        }
    }
    __device__ __forceinline__ T sum(const int* __restrict__ col, const T* __restrict__ val, Live<T> x, int64_t nx,
                                     int sub) const {
        (void)nx;  // length of x: bound of the checked build's tests
        T xv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) xv[u] = RB_AT(x, c[u], nx);  // (x_0 past the row's end, not used)
        T s = T(0);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (a + sub + u * TPR < e) s = fmaT<T>(v[u], xv[u], s);
#pragma unroll 4
        for (int64_t k = a + sub + U * TPR; k < e; k += TPR)
            s = fmaT<T>(__ldg(val + k), RB_AT(x, __ldg(col + k), nx), s);
#pragma unroll
        for (int o = TPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, TPR);
        return s;
    }
};

// A chained kernel over the rows of a CSR matrix: f(i, sum) in one lane per
// row, sum = (A x)_i.  kRowHead: the first row's entries are loaded before the
// wait (for launches whose lanes have one row each; it costs the registers
// that hold 64 warps per SM in the large ones).  kRow32: 32 rows per warp
// (csr_rows.cuh; for launches of one lane per row that fill the chip).
enum RowForm { kRowEach = 0, kRowHead = 1, kRow32 = 2 };
template <typename T, int TPR, int FORM, class F>
__device__ __forceinline__ void chained_rows(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                                             const T* __restrict__ val, int64_t N, Live<T> x, int64_t nx,
                                             const int* flag, F&& f) {
    const int sub = threadIdx.x & (TPR - 1);
    if constexpr (FORM == kRow32) {
        pdl_wait();
        pdl_next();
        if (stopped(flag)) return;
        if constexpr (sizeof(T) == 4 && TPR == 8) rows32_ahead<T, TPR>(row_ptr, col, val, x, nx, N, f);
        else rows32<T, TPR>(row_ptr, col, val, x, nx, N, f);
    } else if constexpr (FORM == kRowHead) {
        const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / TPR;  // one row per group of lanes
        RowHead<T, TPR> head;
        head.load(row_ptr, col, val, i, sub, i < N);
        pdl_wait();
        pdl_next();
        if (stopped(flag)) return;
        const T s = head.sum(col, val, x, nx, sub);
        if (i < N && sub == 0) f(i, s);
    } else {
        pdl_wait();
        pdl_next();
        if (stopped(flag)) return;
        MG_ROWS(TPR, N, i, valid, {
            const T s = row_sum<T, TPR>(row_ptr, col, val, x, nx, i, sub, valid);
            if (valid && sub == 0) f(i, s);
        })
    }
}

// x = W b (the first sweep from x = 0); dinv holds W = Omega D^-1
template <typename T, typename BT>
__global__ void __launch_bounds__(kT) mg_first_kernel(int64_t N, Live<BT> b, const T* __restrict__ dinv, T* x,
                                                      const int* flag) {
    pdl_wait();
    pdl_next();
    if (stopped(flag)) return;
    MG_ELEMS(N, i) x[i] = dinv[i] * (T)b[i];
}

// xo = xi + W (b - A xi)
template <typename T, typename BT, typename OT, int TPR, int FORM>
__global__ void __launch_bounds__(kT) mg_jacobi_kernel(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                                                       const T* __restrict__ val, int64_t N, Live<T> xi, Live<BT> b,
                                                       const T* __restrict__ dinv, OT* xo, const int* flag) {
    chained_rows<T, TPR, FORM>(row_ptr, col, val, N, xi, N, flag,
                         [&](int64_t i, T ax) { xo[i] = (OT)fmaT<T>(dinv[i], (T)b[i] - ax, xi[i]); });
}

// r = b - A x
template <typename T, typename BT, int TPR, int FORM>
__global__ void __launch_bounds__(kT) mg_resid_kernel(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                                                      const T* __restrict__ val, int64_t N, Live<T> x, Live<BT> b, T* r,
                                                      const int* flag) {
    chained_rows<T, TPR, FORM>(row_ptr, col, val, N, x, N, flag, [&](int64_t i, T ax) { r[i] = (T)b[i] - ax; });
}

// y = R r (restriction, CSR with n rows)
template <typename T, int TPR, int FORM>
__global__ void __launch_bounds__(kT) mg_restrict_kernel(const int64_t* __restrict__ row_ptr,
                                                         const int* __restrict__ col, const T* __restrict__ val,
                                                         int64_t n, Live<T> r, int64_t nr, T* y, const int* flag) {
    chained_rows<T, TPR, FORM>(row_ptr, col, val, n, r, nr, flag, [&](int64_t i, T v) { y[i] = v; });
}

// A row of the prolongation (ELL, kMgK entries), by 16-byte loads.
template <typename T>
struct PRow {
    static_assert(kMgK % 4 == 0, "rows of whole 16-byte loads");
    int c[kMgK];
    T v[kMgK];
    __device__ __forceinline__ PRow() {}
    __device__ __forceinline__ PRow(const int32_t* __restrict__ pidx, const T* __restrict__ pval, int64_t i) {
#pragma unroll
        for (int j = 0; j < kMgK / 4; ++j) {
            const int4 q = __ldg(reinterpret_cast<const int4*>(pidx + i * kMgK) + j);
            c[4 * j] = q.x;
            c[4 * j + 1] = q.y;
            c[4 * j + 2] = q.z;
            c[4 * j + 3] = q.w;
        }
#pragma unroll
        for (int j = 0; j < (int)(kMgK * sizeof(T) / 16); ++j) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(pval + i * kMgK) + j);
            memcpy(reinterpret_cast<char*>(v) + 16 * j, &q, 16);
        }
    }
};

// x += P e; the first row's entries are loaded before the wait
template <typename T>
__global__ void __launch_bounds__(kT) mg_prolong_kernel(int64_t N, const int32_t* __restrict__ pidx,
                                                        const T* __restrict__ pval, Live<T> e, int64_t ne, T* x,
                                                        const int* flag) {
    (void)ne;  // length of e: bound of the checked build's tests
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    PRow<T> p;
    if (i0 < N) p = PRow<T>(pidx, pval, i0);
    pdl_wait();
    pdl_next();
    if (stopped(flag)) return;
    MG_ELEMS(N, i) {
        if (i != i0) p = PRow<T>(pidx, pval, i);
        T acc = x[i];
#pragma unroll
        for (int j = 0; j < kMgK; ++j) acc = fmaT<T>(p.v[j], RB_AT(e, p.c[j], ne), acc);
        x[i] = acc;
    }
}

// x = Minv b, one warp per row
template <typename T, typename BT, typename OT>
__global__ void __launch_bounds__(kT) mg_dense_kernel(int n, const T* __restrict__ minv, Live<BT> b, OT* x,
                                                      const int* flag) {
    pdl_wait();
    pdl_next();
    if (stopped(flag)) return;
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += warps) {
        T acc = T(0);
        for (int j = lane; j < n; j += 32) acc = fmaT<T>(minv[(int64_t)i * n + j], (T)b[j], acc);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) x[i] = (OT)acc;
    }
}

// ------------------------------------------------------------------ setup --
struct MgBox {
    double mnx, mny, mxx, mxy;
};

__global__ void __launch_bounds__(kT) mg_bbox_kernel(const double2* __restrict__ xy, int64_t N, MgBox* out) {
    double mnx = INFINITY, mny = INFINITY, mxx = -INFINITY, mxy = -INFINITY;
    MG_ELEMS(N, i) {
        const double2 p = xy[i];
        mnx = fmin(mnx, p.x);
        mny = fmin(mny, p.y);
        mxx = fmax(mxx, p.x);
        mxy = fmax(mxy, p.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mnx = fmin(mnx, __shfl_xor_sync(0xffffffffu, mnx, o));
        mny = fmin(mny, __shfl_xor_sync(0xffffffffu, mny, o));
        mxx = fmax(mxx, __shfl_xor_sync(0xffffffffu, mxx, o));
        mxy = fmax(mxy, __shfl_xor_sync(0xffffffffu, mxy, o));
    }
    __shared__ MgBox sh[kT / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) RB_AT(sh, wid, kT / 32) = MgBox{mnx, mny, mxx, mxy};
    __syncthreads();
    if (threadIdx.x == 0) {
        MgBox r = sh[0];
        for (int k = 1; k < kT / 32; ++k) {
            r.mnx = fmin(r.mnx, sh[k].mnx);
            r.mny = fmin(r.mny, sh[k].mny);
            r.mxx = fmax(r.mxx, sh[k].mxx);
            r.mxy = fmax(r.mxy, sh[k].mxy);
        }
        out[blockIdx.x] = r;
    }
}

struct CellGrid {
    double x0, y0, inv_c;
    int gx, gy;
};

__device__ __forceinline__ int64_t cell_of(const CellGrid& g, double x, double y) {
    int cx = (int)floor((x - g.x0) * g.inv_c);
    int cy = (int)floor((y - g.y0) * g.inv_c);
    cx = cx < 0 ? 0 : (cx >= g.gx ? g.gx - 1 : cx);
    cy = cy < 0 ? 0 : (cy >= g.gy ? g.gy - 1 : cy);
    return (int64_t)cy * g.gx + cx;
}

// Packed ranking key: bit 63 = interior node (Dirichlet nodes win), bits
// 62..31 = float32 bits of (d / c)^2 to the cell centre (non-negative, so
// monotone as an integer; < 2^31), bits 30..0 = node index.
__global__ void __launch_bounds__(kT) mg_mark_kernel(const double2* __restrict__ xy, const uint8_t* __restrict__ mask,
                                                     int64_t N, CellGrid g, unsigned long long* __restrict__ best) {
    MG_ELEMS(N, i) {
        const double2 p = xy[i];
        const int64_t c = cell_of(g, p.x, p.y);
        const int cx = (int)(c % g.gx), cy = (int)(c / g.gx);
        const double ux = (p.x - g.x0) * g.inv_c - (cx + 0.5);
        const double uy = (p.y - g.y0) * g.inv_c - (cy + 0.5);
        float d2 = (float)(ux * ux + uy * uy);
        if (!(d2 >= 0.f) || d2 > 1e30f) d2 = 1e30f;
        const unsigned long long key = ((unsigned long long)(mask[i] ? 0u : 1u) << 63) |
                                       ((unsigned long long)__float_as_uint(d2) << 31) | (unsigned long long)i;
        atomicMin(&RB_AT(best, c, (int64_t)g.gx * g.gy), key);
    }
}

__global__ void __launch_bounds__(kT) mg_select_kernel(const double2* __restrict__ xy, int64_t N, CellGrid g,
                                                       const unsigned long long* __restrict__ best,
                                                       int* __restrict__ sel) {
    MG_ELEMS(N, i) {
        const double2 p = xy[i];
        const int64_t c = cell_of(g, p.x, p.y);
        sel[i] = ((RB_AT(best, c, (int64_t)g.gx * g.gy) & 0x7fffffffull) == (unsigned long long)i) ? 1 : 0;
    }
}

struct SelLoad {
    const int* sel;
    __device__ int operator()(int64_t i) const { return sel[i]; }
};

__global__ void __launch_bounds__(kT) mg_gather_kernel(const double2* __restrict__ xy, const uint8_t* __restrict__ mask,
                                                       int64_t N, const int* __restrict__ sel,
                                                       const int* __restrict__ pos, int64_t Nc,
                                                       double2* __restrict__ cxy, uint8_t* __restrict__ cmask) {
    (void)Nc;  // coarse points: bound of the checked build's tests
    MG_ELEMS(N, i) {
        if (sel[i]) {
            const int k = pos[i];
            RB_AT(cxy, k, Nc) = xy[i];
            RB_AT(cmask, k, Nc) = mask[i] ? 1 : 0;
        }
    }
}

// D^-1 from the diagonal of a CSR matrix (1 where the diagonal is zero or
// missing); float copies of dinv and, if val32 != NULL, of the values.
// Dirichlet rows of level 0: y_b += W_b (r_b - (A y)_b), W_b = 1 / a_bb.
// Forward hierarchy (A's Dirichlet rows are identity rows): y_b = r_b, the
// starting guess that keeps every later residual zero on Dirichlet rows.
// Adjoint hierarchy (A^T: identity Dirichlet columns): the back substitution
// y_b = r_b - sum_i a_ib y_i over interior rows i.  In place: a Dirichlet
// row reads only interior entries of y and its own.
__global__ void __launch_bounds__(kT) mg_bfix_kernel(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                                                     const double* __restrict__ val, int64_t N,
                                                     const uint8_t* __restrict__ mask, const double* __restrict__ w,
                                                     Live<double> r, double* y, const int* flag) {
    pdl_wait();
    pdl_next();
    if (stopped(flag)) return;
    MG_ELEMS(N, i) {
        if (!mask[i]) continue;
        double s = 0.0;
        for (int64_t k = row_ptr[i]; k < row_ptr[i + 1]; ++k) s = fma(val[k], RB_AT(y, col[k], N), s);
        y[i] = fma(w[i], r[i] - s, y[i]);
    }
}

// W = Omega D^-1 of the smoother: omega / a_ii on interior rows, 1 / a_ii on
// Dirichlet rows.
__global__ void __launch_bounds__(kT) mg_diag_kernel(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                                                     const double* __restrict__ val, int64_t N, int col_base,
                                                     const uint8_t* __restrict__ mask, double omega,
                                                     double* __restrict__ dinv, float* __restrict__ dinv32,
                                                     int* __restrict__ bad) {
    int nb = 0;
    MG_ELEMS(N, i) {
        double d = 0.0;
        for (int64_t k = row_ptr[i]; k < row_ptr[i + 1]; ++k)
            if (col[k] - col_base == (int)i) d = val[k];
        const bool ok = d != 0.0 && isfinite(d);
        nb |= ok ? 0 : 1;
        const double iv = ok ? (mask[i] ? 1.0 : omega) / d : 1.0;
        dinv[i] = iv;
        dinv32[i] = __double2float_rn(iv);
    }
    if (nb) atomicOr(bad, 1);
}

// Interpolation rows: zero at Dirichlet nodes; where the interpolation
// system was singular (its nodes on one conic), the value of the nearest
// coarse node; float copy; CSR row pointer of the ELL layout.
__global__ void __launch_bounds__(kT) mg_pfix_kernel(int64_t N, const uint8_t* __restrict__ mask,
                                                     const int* __restrict__ pstat, double* __restrict__ pval,
                                                     float* __restrict__ pval32, int64_t* __restrict__ prow) {
    MG_ELEMS(N, i) {
        const bool dir = mask[i] != 0;
        const bool sing = pstat[i] != 0;
        for (int j = 0; j < kMgK; ++j) {
            const int64_t e = i * kMgK + j;
            const double v = dir ? 0.0 : (sing ? (j == 0 ? 1.0 : 0.0) : pval[e]);
            pval[e] = v;
            pval32[e] = __double2float_rn(v);
        }
        prow[i] = i * kMgK;
        if (i == N - 1) prow[N] = N * kMgK;
    }
}

// CSR row pointer of the ELL prolongation (kMgK entries per row).
__global__ void __launch_bounds__(kT) mg_ellrow_kernel(int64_t N, int64_t* __restrict__ prow) {
    MG_ELEMS(N + 1, i) prow[i] = i * kMgK;
}

// R = scale P^T with zero rows at coarse Dirichlet nodes; float copy.
__global__ void __launch_bounds__(kT) mg_rscale_kernel(const int64_t* __restrict__ rrow, int64_t Nc,
                                                       const uint8_t* __restrict__ cmask, double scale,
                                                       double* __restrict__ rval, float* __restrict__ rval32) {
    MG_ELEMS(Nc, c) {
        const double f = (cmask && cmask[c]) ? 0.0 : scale;
        for (int64_t k = rrow[c]; k < rrow[c + 1]; ++k) {
            const double v = rval[k] * f;
            rval[k] = v;
            rval32[k] = __double2float_rn(v);
        }
    }
}

// Adjoint hierarchy: prolongation R^T = scale P with the columns of coarse
// Dirichlet nodes zeroed (R zeroes their rows); float copy.
__global__ void __launch_bounds__(kT) mg_pscale_kernel(int64_t N, const int32_t* __restrict__ pidx,
                                                       const uint8_t* __restrict__ cmask, int64_t Nc, double scale,
                                                       double* __restrict__ pval, float* __restrict__ pval32) {
    const int64_t total = N * kMgK;
    MG_ELEMS(total, e) {
        (void)Nc;  // coarse points: bound of the checked build's tests
        const double v = RB_AT(cmask, pidx[e], Nc) ? 0.0 : scale * pval[e];
        pval[e] = v;
        pval32[e] = __double2float_rn(v);
    }
}

__global__ void __launch_bounds__(kT) mg_f32_kernel(const double* __restrict__ v, int64_t n, float* __restrict__ v32) {
    MG_ELEMS(n, i) v32[i] = __double2float_rn(v[i]);
}

// A singular stencil at an interior node (Dirichlet rows ignore weights).
__global__ void __launch_bounds__(kT) mg_count_kernel(const int* __restrict__ stat, const uint8_t* __restrict__ mask,
                                                      int64_t N, int* __restrict__ bad) {
    int nb = 0;
    MG_ELEMS(N, i) nb |= (stat[i] && !mask[i]) ? 1 : 0;
    if (nb) atomicOr(bad, 1);
}

// Dense inverse of a CSR matrix (n <= kMgCoarsest) by Gauss-Jordan in place,
// one cluster of kInvCtas blocks: block c holds rows c, c + kInvCtas, ... in
// shared memory.  Step k: the pivot is the largest |a_ik| over the rows that
// have not been one (lowest i on ties); every block takes the scaled pivot row
// from its owner's shared memory and eliminates column k from its own rows.
// Rows stay where they are; row p_k of the result is row k of the inverse
// with its columns in pivot order.  Writes the inverse and its float32 copy;
// sets *bad (and writes nothing) where no pivot is positive.
// Bound by the FP64 units (n^3 multiply-adds at 2 per clock per SM: 0.54 ms
// at n = 128 on one SM) and by two cluster barriers per step.  One block on
// the [A | I] matrix in global memory took 1.0 ms at n = 60 and 4.2 ms at
// n = 110.
constexpr int kInvCtas = 8;  // the portable cluster size
constexpr int kInvT = 256;
constexpr int kInvRows = kMgCoarsest / kInvCtas;

struct InvPivot {
    double v;
    int row;
};

__global__ void __cluster_dims__(kInvCtas, 1, 1) __launch_bounds__(kInvT)
    mg_inverse_kernel(const int64_t* __restrict__ row_ptr, const int* __restrict__ col,
                      const double* __restrict__ val, int n, int col_base, double* __restrict__ minv,
                      float* __restrict__ minv32, int* __restrict__ bad) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ double a[kInvRows][kMgCoarsest];
    __shared__ double prow[kMgCoarsest];   // the scaled pivot row
    __shared__ double f[kInvRows];         // column k of this block's rows
    __shared__ InvPivot cand[2];           // this block's candidate, by step parity
    __shared__ int piv[kMgCoarsest];       // pivot row of each step
    __shared__ int used[kInvRows];
    __shared__ int pick;
    __shared__ double pinv;
    const int tid = threadIdx.x, rank = (int)cluster.block_rank();
    const int rows = rank < n ? (n - rank + kInvCtas - 1) / kInvCtas : 0;
    for (int e = tid; e < kInvRows * kMgCoarsest; e += kInvT) a[e / kMgCoarsest][e % kMgCoarsest] = 0.0;
    if (tid < kInvRows) used[tid] = 0;
    __syncthreads();
    if (tid < rows) {
        const int i = rank + tid * kInvCtas;
        for (int64_t k = row_ptr[i]; k < row_ptr[i + 1]; ++k) {
            const int c = col[k] - col_base;
            if ((unsigned)c < (unsigned)n) a[tid][c] += val[k];
        }
    }
    __syncthreads();
    bool fail = false;
    for (int k = 0; k < n; ++k) {
        if (tid < 32) {
            double best = -1.0;
            int row = n;
            if (tid < rows && !used[tid]) {
                const double v = fabs(a[tid][k]);
                if (v > best) {  // (false for a NaN)
                    best = v;
                    row = rank + tid * kInvCtas;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double ov = __shfl_xor_sync(0xffffffffu, best, o);
                const int oi = __shfl_xor_sync(0xffffffffu, row, o);
                if (ov > best || (ov == best && oi < row)) {
                    best = ov;
                    row = oi;
                }
            }
            if (tid == 0) cand[k & 1] = InvPivot{best, row};
        }
        cluster.sync();  // candidates published, every row of step k - 1 final
        if (tid < 32) {
            InvPivot c{-1.0, n};
            if (tid < kInvCtas) c = *cluster.map_shared_rank(&cand[k & 1], tid);
#pragma unroll
            for (int o = kInvCtas / 2; o > 0; o >>= 1) {
                const double ov = __shfl_xor_sync(0xffffffffu, c.v, o);
                const int oi = __shfl_xor_sync(0xffffffffu, c.row, o);
                if (ov > c.v || (ov == c.v && oi < c.row)) {
                    c.v = ov;
                    c.row = oi;
                }
            }
            if (tid == 0) {
                pick = c.v > 0.0 ? c.row : -1;
                piv[k] = pick;
                if (pick >= 0)
                    pinv = 1.0 / *cluster.map_shared_rank(&a[pick / kInvCtas][k], pick % kInvCtas);
            }
        }
        __syncthreads();
        const int p = pick;
        if (p < 0) {  // the same in every block
            fail = true;
            break;
        }
        if (tid < n) {
            const double v = *cluster.map_shared_rank(&a[p / kInvCtas][tid], p % kInvCtas);
            prow[tid] = (tid == k ? 1.0 : v) * pinv;
        }
        if (tid < rows) f[tid] = a[tid][k];
        __syncthreads();
        // the owner changes the pivot row only after every block has read it
        cluster.barrier_arrive();
        const int mine = (p % kInvCtas) == rank ? p / kInvCtas : -1;
        for (int e = tid; e < rows * n; e += kInvT) {
            const int i = e / n, j = e - i * n;
            if (i != mine) a[i][j] = fma(-f[i], prow[j], j == k ? 0.0 : a[i][j]);
        }
        cluster.barrier_wait();
        if (mine >= 0) {
            if (tid < n) a[mine][tid] = prow[tid];
            if (tid == 0) used[mine] = 1;
        }
        __syncthreads();
    }
    cluster.sync();  // no block leaves while another may read its rows
    if (fail) {
        if (rank == 0 && tid == 0) *bad = 1;
        return;
    }
    // row p_k is row k of the inverse, its column l belongs to pivot p_l
    for (int e = tid; e < rows * n; e += kInvT) {
        const int i = e / n, l = e - i * n;
        const int g = rank + i * kInvCtas;
        int k = 0;
        while (piv[k] != g) ++k;
        const double v = a[i][l];
        const int64_t o = (int64_t)k * n + piv[l];
        minv[o] = v;
        minv32[o] = __double2float_rn(v);
    }
}

// ------------------------------------------------------------------- host --
// ---- Galerkin coarse operators (adjoint hierarchy) -------------------------
// A_{l+1} = R_l A_l P_l with R_l = P^T (the interpolation's transpose) and
// P_l = (N_c / N_f) P without the columns of coarse Dirichlet nodes; the rows
// of coarse Dirichlet nodes become identity rows (their columns are zero in
// the product, so the coarse system stays block diagonal).  One warp per
// coarse row c and two shared-memory hash tables (open addressing, linear
// probing, keys -1 when empty): first D = R_c A_l keyed by fine column, then
// the row C_c = D P_l keyed by coarse column.  Zero entries of R and P_l
// (Dirichlet rows of P, the removed columns) are skipped.  Every key's terms
// are summed in a fixed order (a batch is one A row, whose columns are
// distinct, or two P rows, one per half-warp, whose values go in one half
// after the other; batches run in sequence; D is sorted by column before its
// rows of P are read), and
// the row is sorted by column and staged at a place taken from an atomic
// counter; after a scan of the row lengths a second kernel copies each row
// to its CSR position.  The product therefore does not depend on thread
// timing.
// Two table sizes: (512, 256) slots first, four warps per block, 9 KB of
// tables per warp (24 warps per SM); a level whose rows overflow them is
// redone with (1024, 512), 18 KB per warp (12 warps per SM).
constexpr int kGalWarps = 4;
template <int H1, int H2>
constexpr size_t gal_smem_bytes() {
    return (size_t)kGalWarps * (H1 + H2) * (sizeof(int) + sizeof(double));
}

// Slot of `key` in a table of cap = mask + 1 slots (inserted if absent);
// -1 when the table is full.  *fresh is set when this call inserted it.
__device__ __forceinline__ int gal_slot(int* keys, unsigned mask, int key, int* fresh) {
    unsigned h = ((unsigned)key * 2654435761u) & mask;
    for (unsigned probe = 0; probe <= mask; ++probe) {
        const int k = *(volatile int*)(keys + h);
        if (k == key) return (int)h;
        if (k == -1) {
            const int old = atomicCAS(keys + h, -1, key);
            if (old == -1) {
                *fresh = 1;
                return (int)h;
            }
            if (old == key) return (int)h;
        }
        h = (h + 1) & mask;
    }
    return -1;
}

// Ascending sort of n <= cap (key, value) pairs held at the front of the
// arrays, by one warp (bitonic network over the next power of two, padded
// with INT_MAX keys).
__device__ __forceinline__ void gal_sort(int* keys, double* vals, int n, int cap, int lane) {
    (void)cap;  // table size: bound of the checked build's tests
    int m = 32;
    while (m < n) m <<= 1;
    for (int i = n + lane; i < m; i += 32) RB_AT(keys, i, cap) = 0x7fffffff;
    __syncwarp();
    for (int k = 2; k <= m; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = lane; i < m; i += 32) {
                const int p = i ^ j;
                if (p > i) {
                    const int a = RB_AT(keys, i, cap), b = RB_AT(keys, p, cap);
                    const bool up = (i & k) == 0;
                    if ((a > b) == up) {
                        RB_AT(keys, i, cap) = b;
                        RB_AT(keys, p, cap) = a;
                        const double t = RB_AT(vals, i, cap);
                        RB_AT(vals, i, cap) = RB_AT(vals, p, cap);
                        RB_AT(vals, p, cap) = t;
                    }
                }
            }
            __syncwarp();
        }
    }
}

// Moves the occupied slots of a table (cap slots) to its front, in slot
// order; returns their count.  Every lane gets the count.
__device__ __forceinline__ int gal_compact(int* keys, double* vals, int cap, int lane, bool with_vals) {
    int n = 0;
    for (int base = 0; base < cap; base += 32) {
        const int i = base + lane;
        const int k = keys[i];
        const double v = with_vals ? vals[i] : 0.0;
        const unsigned occ = __ballot_sync(0xffffffffu, k != -1);
        __syncwarp();
        if (k != -1) {
            const int dst = n + __popc(occ & ((1u << lane) - 1u));
            RB_AT(keys, dst, cap) = k;
            if (with_vals) RB_AT(vals, dst, cap) = v;
        }
        n += __popc(occ);
        __syncwarp();
    }
    return n;
}

template <int kGalH1, int kGalH2>
__global__ void __launch_bounds__(kGalWarps * 32) mg_galerkin_kernel(
    int64_t Nc, const int64_t* __restrict__ rrow, const int32_t* __restrict__ rcol, const double* __restrict__ rval,
    const int64_t* __restrict__ arow, const int* __restrict__ acol, const double* __restrict__ aval,
    const int32_t* __restrict__ pidx, const double* __restrict__ pval, const uint8_t* __restrict__ cmask,
    int* __restrict__ count, int64_t* __restrict__ start, unsigned long long* __restrict__ total, int64_t cap,
    int* __restrict__ tcol, double* __restrict__ tval, int* __restrict__ bad, int64_t Nf, int64_t annz) {
    (void)Nf;  // fine points and A's entries: bounds of the checked build's tests
    (void)annz;
    extern __shared__ __align__(16) unsigned char gal_smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double* v1 = reinterpret_cast<double*>(gal_smem) + (size_t)wid * (kGalH1 + kGalH2);
    double* v2 = v1 + kGalH1;
    int* k1 = reinterpret_cast<int*>(reinterpret_cast<double*>(gal_smem) + (size_t)kGalWarps * (kGalH1 + kGalH2)) +
              (size_t)wid * (kGalH1 + kGalH2);
    int* k2 = k1 + kGalH1;
    (void)RB_SH(v2 + kGalH2 - 1);  // the warp's tables lie in the launch's shared memory
    (void)RB_SH(k2 + kGalH2 - 1);
    int overflow = 0;
    const int64_t nwarps = (int64_t)gridDim.x * kGalWarps;
    for (int64_t c = (int64_t)blockIdx.x * kGalWarps + wid; c < Nc; c += nwarps) {
        int m = 1;
        if (cmask[c]) {
            if (lane == 0) {  // an identity row
                k2[0] = (int)c;
                v2[0] = 1.0;
            }
        } else {
            for (int i = lane; i < kGalH1; i += 32) {
                k1[i] = -1;
                v1[i] = 0.0;
            }
            for (int i = lane; i < kGalH2; i += 32) {
                k2[i] = -1;
                v2[i] = 0.0;
            }
            __syncwarp();
            bool full = false;
            // D = R_c A_l: one row of A_l per batch of lanes.  The entries of
            // R's row and the extents of their A rows are loaded 32 at a time,
            // one per lane (independent loads), then handed out by shuffles,
            // and each A row's first batch is loaded before the previous
            // row's keys go into the table.
            const int64_t r0 = rrow[c], r1 = rrow[c + 1];
            for (int64_t e0 = r0; e0 < r1; e0 += 32) {
                double rv_l = 0.0;
                int64_t a0_l = 0, a1_l = 0;
                if (e0 + lane < r1) {
                    rv_l = rval[e0 + lane];
                    if (rv_l != 0.0) {
                        const int f = rcol[e0 + lane];
                        a0_l = RB_AT(arow, f, Nf + 1);
                        a1_l = RB_AT(arow, f + 1, Nf + 1);
                    }
                }
                const int cnt = (int)min((int64_t)32, r1 - e0);
                // the first batch of the first entry's A row
                int64_t a0 = __shfl_sync(0xffffffffu, a0_l, 0), a1 = __shfl_sync(0xffffffffu, a1_l, 0);
                int kc = (a0 + lane < a1) ? RB_AT(acol, a0 + lane, annz) : -1;
                double kv = (a0 + lane < a1) ? RB_AT(aval, a0 + lane, annz) : 0.0;
                for (int t = 0; t < cnt; ++t) {
                    const double rv = __shfl_sync(0xffffffffu, rv_l, t);
                    const int64_t b0 = a0, b1 = a1;
                    int cur_c = kc;
                    double cur_v = kv;
                    // the next entry's first batch, in flight while this row fills the table
                    if (t + 1 < cnt) {
                        a0 = __shfl_sync(0xffffffffu, a0_l, t + 1);
                        a1 = __shfl_sync(0xffffffffu, a1_l, t + 1);
                        kc = (a0 + lane < a1) ? RB_AT(acol, a0 + lane, annz) : -1;
                        kv = (a0 + lane < a1) ? RB_AT(aval, a0 + lane, annz) : 0.0;
                    }
                    if (rv == 0.0) continue;  // (warp-uniform: a Dirichlet row of P)
                    for (int64_t b = b0; b < b1; b += 32) {
                        const int64_t k = b + lane;
                        if (b > b0 && k < b1) {  // batches after the first (rows longer than 32)
                            cur_c = RB_AT(acol, k, annz);
                            cur_v = RB_AT(aval, k, annz);
                        }
                        if (k < b1) {
                            int fresh = 0;
                            const int sl = gal_slot(k1, kGalH1 - 1, cur_c, &fresh);
                            if (sl < 0) full = true;
                            else RB_AT(v1, sl, kGalH1) = fma(rv, cur_v, RB_AT(v1, sl, kGalH1));
                        }
                        __syncwarp();
                    }
                }
            }
            // D's entries at the front, sorted by column
            const int n1 = gal_compact(k1, v1, kGalH1, lane, true);
            gal_sort(k1, v1, n1, kGalH1, lane);
            // C_c = D P_l: two entries of D per batch, lanes 0-11 and 16-27;
            // the keys go in together, the values in D's order; the next
            // batch's row of P is loaded before this batch's keys go in
            const int half = lane >> 4, j = lane & 15;
            const bool jl = j < kMgK;
            int nxt_i = -1;
            double nxt_v = 0.0;
            if (half < n1 && jl) {
                const int64_t pe = (int64_t)RB_AT(k1, half, kGalH1) * kMgK + j;
                nxt_v = RB_AT(pval, pe, Nf * kMgK);
                nxt_i = RB_AT(pidx, pe, Nf * kMgK);
            }
            for (int i = 0; i < n1; i += 2) {
                const int di = i + half;
                const int pj = nxt_i;
                const double pv = nxt_v;
                if (di + 2 < n1 && jl) {
                    const int64_t pe = (int64_t)RB_AT(k1, di + 2, kGalH1) * kMgK + j;
                    nxt_v = RB_AT(pval, pe, Nf * kMgK);
                    nxt_i = RB_AT(pidx, pe, Nf * kMgK);
                }
                int sl = -1;
                double term = 0.0;
                if (di < n1 && jl && pv != 0.0) {
                    int fresh = 0;
                    sl = gal_slot(k2, kGalH2 - 1, pj, &fresh);
                    if (sl < 0) full = true;
                    term = RB_AT(v1, di, kGalH1) * pv;
                }
                __syncwarp();
                if (half == 0 && sl >= 0) RB_AT(v2, sl, kGalH2) += term;
                __syncwarp();
                if (half == 1 && sl >= 0) RB_AT(v2, sl, kGalH2) += term;
                __syncwarp();
            }
            if (__any_sync(0xffffffffu, full)) {
                overflow = 1;
                continue;
            }
            m = gal_compact(k2, v2, kGalH2, lane, true);
            gal_sort(k2, v2, m, kGalH2, lane);
        }
        // stage the row (any free place: the copy below puts rows in order)
        unsigned long long pos = 0;
        if (lane == 0) pos = atomicAdd(total, (unsigned long long)m);
        pos = __shfl_sync(0xffffffffu, pos, 0);
        if ((int64_t)pos + m > cap) {
            overflow = 1;
            continue;
        }
        for (int i = lane; i < m; i += 32) {
            RB_AT(tcol, pos + i, cap) = RB_AT(k2, i, kGalH2);
            RB_AT(tval, pos + i, cap) = RB_AT(v2, i, kGalH2);
        }
        if (lane == 0) {
            count[c] = m;
            start[c] = (int64_t)pos;
        }
        __syncwarp();
    }
    if (overflow && lane == 0) atomicOr(bad, 2);
}

// The staged rows into the level's CSR (row c at crow[c]), with the float copy.
__global__ void __launch_bounds__(kT) mg_galerkin_place_kernel(int64_t Nc, const int64_t* __restrict__ start,
                                                               const int64_t* __restrict__ crow,
                                                               const int* __restrict__ tcol,
                                                               const double* __restrict__ tval,
                                                               int* __restrict__ ccol, double* __restrict__ cval,
                                                               float* __restrict__ cval32, int64_t tcap,
                                                               int64_t cnnz) {
    (void)tcap;  // staged and placed entries: bounds of the checked build's tests
    (void)cnnz;
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < Nc; c += nw) {
        const int64_t o = crow[c], len = crow[c + 1] - o, s = start[c];
        RB_SPAN(s, len, tcap);
        RB_SPAN(o, len, cnnz);
        for (int64_t i = lane; i < len; i += 32) {
            const double v = RB_AT(tval, s + i, tcap);
            RB_AT(ccol, o + i, cnnz) = RB_AT(tcol, s + i, tcap);
            RB_AT(cval, o + i, cnnz) = v;
            RB_AT(cval32, o + i, cnnz) = __double2float_rn(v);
        }
    }
}

struct CountLoad64 {
    const int* c;
    __device__ int64_t operator()(int64_t i) const { return (int64_t)c[i]; }
};

int tpr_for(int64_t rows, int64_t nnz) {
    const double L = (double)nnz / (double)std::max<int64_t>(rows, 1);
    if (L >= 80) return 8;  // (Galerkin coarse operators)
    if (L >= 40) return 4;
    if (L >= 8) return 2;
    return 1;
}

int blocks_for(int64_t threads) {
    const int64_t b = (threads + kT - 1) / kT;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, (int64_t)sm_count() * 16));
}

// Upper bounds of the level sizes: each coarsening keeps at most half.
std::vector<int64_t> level_bounds(int64_t N) {
    std::vector<int64_t> nb{N};
    while (nb.back() > kMgCoarsest && (int)nb.size() < RBFFD_MG_MAX_LEVELS) nb.push_back(nb.back() / 2);
    return nb;
}

struct MgScratch {
    int64_t* a_row;  // adjoint hierarchy: the coarse operator before its transpose
    int32_t* a_col;
    double* a_val;
    unsigned long long* cells;
    int* sel;
    int* pos;
    int* sums;
    MgBox* box;
    int* flags;  // [0] singular / bad, [1] spare
    int* pstat;
    int32_t* sidx;   // coarse stencils
    double* sw;      // coarse weights
    int32_t* sstat;  // coarse weight status
    void* knn_ws;
    size_t knn_bytes;
    void* asm_ws;
    size_t asm_bytes;
    void* tr_ws;
    size_t tr_bytes;
    int64_t* prow;
    int64_t* sums64;  // tile sums of 64-bit scans
    // Galerkin products: rows staged before their CSR placement (capacity
    // gal_cap entries), per-row staging offsets, the staging counter
    int* gal_col;
    double* gal_val;
    int64_t* gal_start;
    unsigned long long* gal_total;
    int64_t gal_cap;
};

constexpr int kBoxParts = 64;

// Carves the workspace; with ws == NULL only sizes it.  Levels: the given
// sizes (a built hierarchy's), else the upper bounds of level_bounds; the
// operators of levels >= 1 hold `cap` entries per row.
size_t mg_layout(void* ws, int64_t N, MgHierarchy* h, MgScratch* s, const std::vector<int64_t>* sizes = nullptr,
                 int cap = kMgCoarseN) {
    const std::vector<int64_t> nb = sizes ? *sizes : level_bounds(N);
    Carver c(ws);
    MgScratch t{};
    size_t knn_b = 0, asm_b = 0, tr_b = 0;
    for (size_t l = 0; l < nb.size(); ++l) {
        knn_b = std::max(knn_b, rbffd_stencils_workspace_size(std::max<int64_t>(nb[l], kMgCoarseN), kMgCoarseN));
        asm_b = std::max(asm_b, rbffd_assemble_workspace_size(nb[l]));
        tr_b = std::max(tr_b, rbffd_transpose_workspace_size(nb[l]));
    }
    {
        const int64_t n1b = nb.size() > 1 ? nb[1] : 1;
        t.a_row = c.take<int64_t>(n1b + 1);
        t.a_col = c.take<int32_t>((size_t)n1b * kMgCoarseN);
        t.a_val = c.take<double>((size_t)n1b * kMgCoarseN);
    }
    t.cells = c.take<unsigned long long>((size_t)(2 * N + 16));
    t.sel = c.take<int>(N);
    t.pos = c.take<int>(N + 1);
    t.sums = c.take<int>(scan_tiles(N) + 1);
    t.box = c.take<MgBox>(kBoxParts);
    t.flags = c.take<int>(64);
    t.pstat = c.take<int>(N);
    t.prow = c.take<int64_t>(N + 1);
    const int64_t n1 = nb.size() > 1 ? nb[1] : 1;
    t.sidx = c.take<int32_t>((size_t)n1 * kMgCoarseN);
    t.sw = c.take<double>((size_t)n1 * kMgCoarseN);
    t.sstat = c.take<int32_t>(n1);
    t.knn_ws = c.take<char>(knn_b);
    t.knn_bytes = knn_b;
    t.asm_ws = c.take<char>(asm_b);
    t.asm_bytes = asm_b;
    t.tr_ws = c.take<char>(tr_b);
    t.tr_bytes = tr_b;
    t.sums64 = c.take<int64_t>(scan_tiles(N) + 1);
    if (cap > kMgCoarseN && nb.size() > 1) {
        t.gal_cap = nb[1] * (int64_t)cap;
        t.gal_col = c.take<int>((size_t)t.gal_cap);
        t.gal_val = c.take<double>((size_t)t.gal_cap);
        t.gal_start = c.take<int64_t>(nb[1]);
        t.gal_total = c.take<unsigned long long>(1);
    }
    MgHierarchy hh{};
    for (size_t l = 0; l < nb.size(); ++l) {
        const int64_t n = nb[l];
        MgLevel& L = hh.lv[l];
        if (l > 0) {
            double* xy = c.take<double>((size_t)2 * n);
            L.xy = xy;
            uint8_t* mk = c.take<uint8_t>(n);
            L.mask = mk;
            int64_t* rp = c.take<int64_t>(n + 1);
            L.row_ptr = rp;
            int* cl = c.take<int>((size_t)n * cap);
            L.col = cl;
            double* v = c.take<double>((size_t)n * cap);
            L.val = v;
            float* v32 = c.take<float>((size_t)n * cap);
            L.val32 = v32;
        }
        L.dinv = c.take<double>(n);
        L.dinv32 = c.take<float>(n);
        L.x = c.take<double>(n);
        L.t = c.take<double>(n);
        L.r = c.take<double>(n);
        L.b = c.take<double>(n);
        L.x32 = c.take<float>(n);
        L.t32 = c.take<float>(n);
        L.r32 = c.take<float>(n);
        L.b32 = c.take<float>(n);
        if (l + 1 < nb.size()) {
            L.pidx = c.take<int32_t>((size_t)n * kMgK);
            L.pval = c.take<double>((size_t)n * kMgK);
            L.pval32 = c.take<float>((size_t)n * kMgK);
            L.rrow = c.take<int64_t>(n + 1);
            L.rcol = c.take<int32_t>((size_t)n * kMgK);
            L.rval = c.take<double>((size_t)n * kMgK);
            L.rval32 = c.take<float>((size_t)n * kMgK);
        }
    }
    // the dense inverse goes with whichever level ends up coarsest
    double* minv = c.take<double>((size_t)kMgCoarsest * kMgCoarsest);
    float* minv32 = c.take<float>((size_t)kMgCoarsest * kMgCoarsest);
    for (size_t l = 0; l < nb.size(); ++l) {
        hh.lv[l].minv = minv;
        hh.lv[l].minv32 = minv32;
    }
    if (h) *h = hh;
    if (s) *s = t;
    return c.off;
}

// Selects the coarse nodes of level l into level l + 1; returns their count
// in *nc.
int coarsen(const MgLevel& L, MgLevel& C, const MgScratch& s, cudaStream_t st, int64_t* nc) {
    const int64_t N = L.N;
    const double2* xy = reinterpret_cast<const double2*>(L.xy);
    mg_bbox_kernel<<<kBoxParts, kT, 0, st>>>(xy, N, s.box);
    note_launches(1);
    RBFFD_LAUNCH_CHECK();
    MgBox parts[kBoxParts];
    RBFFD_CUDA_TRY(cudaMemcpyAsync(parts, s.box, sizeof(parts), cudaMemcpyDeviceToHost, st));
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    MgBox bx = parts[0];
    for (int k = 1; k < kBoxParts; ++k) {
        bx.mnx = std::min(bx.mnx, parts[k].mnx);
        bx.mny = std::min(bx.mny, parts[k].mny);
        bx.mxx = std::max(bx.mxx, parts[k].mxx);
        bx.mxy = std::max(bx.mxy, parts[k].mxy);
    }
    const double W = bx.mxx - bx.mnx, H = bx.mxy - bx.mny;
    if (!(std::isfinite(W) && std::isfinite(H)) || !(W > 0.0 || H > 0.0)) return RBFFD_ERR_INVALID_ARG;
    double c = (W > 0.0 && H > 0.0) ? 2.0 * std::sqrt(W * H / (double)N) : 2.0 * std::max(W, H) / (double)N;
    for (int attempt = 0; attempt < 200; ++attempt, c *= 1.25) {
        CellGrid g;
        g.x0 = bx.mnx;
        g.y0 = bx.mny;
        g.inv_c = 1.0 / c;
        const double gx = std::floor(W / c) + 1.0, gy = std::floor(H / c) + 1.0;
        if (gx * gy > (double)(2 * N + 16)) continue;
        g.gx = (int)gx;
        g.gy = (int)gy;
        const int64_t cells = (int64_t)g.gx * g.gy;
        RBFFD_CUDA_TRY(cudaMemsetAsync(s.cells, 0xff, sizeof(unsigned long long) * cells, st));
        mg_mark_kernel<<<blocks_for(N), kT, 0, st>>>(xy, L.mask, N, g, s.cells);
        mg_select_kernel<<<blocks_for(N), kT, 0, st>>>(xy, N, g, s.cells, s.sel);
        note_launches(2);
        RBFFD_LAUNCH_CHECK();
        RBFFD_CUDA_TRY(exclusive_scan<int>(SelLoad{s.sel}, N, s.pos, s.sums, s.pos + N, st));
        int cnt = 0;
        RBFFD_CUDA_TRY(cudaMemcpyAsync(&cnt, s.pos + N, sizeof(int), cudaMemcpyDeviceToHost, st));
        RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
        if ((int64_t)cnt > N / 2) continue;
        if (cnt <= kMgK) return RBFFD_ERR_INVALID_ARG;  // degenerate node set
        mg_gather_kernel<<<blocks_for(N), kT, 0, st>>>(xy, L.mask, N, s.sel, s.pos, (int64_t)cnt,
                                                       reinterpret_cast<double2*>(const_cast<double*>(C.xy)),
                                                       const_cast<uint8_t*>(C.mask));
        note_launches(1);
        RBFFD_LAUNCH_CHECK();
        *nc = cnt;
        return RBFFD_OK;
    }
    return RBFFD_ERR_INVALID_ARG;
}

int dense_inverse(const MgLevel& L, int col_base, const MgScratch& s, cudaStream_t st) {
    const int n = (int)L.N;
    mg_inverse_kernel<<<kInvCtas, kInvT, 0, st>>>(L.row_ptr, L.col, L.val, n, col_base, L.minv, L.minv32, s.flags);
    note_launches(1);
    RBFFD_LAUNCH_CHECK();
    return RBFFD_OK;
}

// ---- V-cycle ----------------------------------------------------------------
template <typename T>
struct Sel;
template <>
struct Sel<double> {
    static const double* val(const MgLevel& L) { return L.val; }
    static const double* dinv(const MgLevel& L) { return L.dinv; }
    static const double* pval(const MgLevel& L) { return L.pval; }
    static const double* rval(const MgLevel& L) { return L.rval; }
    static const double* minv(const MgLevel& L) { return L.minv; }
    static double* x(const MgLevel& L) { return L.x; }
    static double* t(const MgLevel& L) { return L.t; }
    static double* r(const MgLevel& L) { return L.r; }
    static double* b(const MgLevel& L) { return L.b; }
};
template <>
struct Sel<float> {
    static const float* val(const MgLevel& L) { return L.val32; }
    static const float* dinv(const MgLevel& L) { return L.dinv32; }
    static const float* pval(const MgLevel& L) { return L.pval32; }
    static const float* rval(const MgLevel& L) { return L.rval32; }
    static const float* minv(const MgLevel& L) { return L.minv32; }
    static float* x(const MgLevel& L) { return L.x32; }
    static float* t(const MgLevel& L) { return L.t32; }
    static float* r(const MgLevel& L) { return L.r32; }
    static float* b(const MgLevel& L) { return L.b32; }
};

// f(form) with the form of a launch over `rows` rows as a compile-time
// constant.  Rows are loaded before the wait for the previous kernel where
// all lanes are resident at once.  Rows of the kernels in csr_rows.cuh, one
// lane per row, start at a full chip (152 x 2048): 1M rows of 30 entries, FP64
// cycle 658 -> 619 us; 300k rows, one lane each, lose 2 to 4 %.
template <int TPR, class F>
void row_form(int64_t rows, bool wide, F&& f) {
    if (rows * TPR <= (int64_t)sm_count() * 4 * kT) return f(std::integral_constant<int, kRowHead>());
    if constexpr (TPR > 1) {
        if (wide && rows >= (int64_t)sm_count() * 2048) return f(std::integral_constant<int, kRow32>());
    }
    f(std::integral_constant<int, kRowEach>());
}

// f(lanes per row, form) for a level's operator.  Float32 rows of 15 to 40
// entries: two lanes per row leave L1's wavefronts as the bound, so eight
// with the loads ahead where the launch is large (1M rows of 30 entries:
// cycle 458 -> 404 us) and four below (100k rows: 106 -> 97); longer rows stay
// with four, one row at a time (1M rows of 56 entries: 565 against 569).
// FP64 rows of that length take four where every lane has one row (100k rows:
// 157 -> 151; more lanes cost FP64 additions in the larger launches).
template <typename T>
int level_tpr(const MgLevel& L) {
    if (L.tpr != 2 || L.nnz < 15 * L.N) return L.tpr;
    if (sizeof(T) == 8) return L.N * 4 <= (int64_t)sm_count() * 4 * kT ? 4 : 2;
    return L.N >= (int64_t)sm_count() * 2048 ? 8 : 4;
}
template <class F>
void row_launch(int64_t rows, int tpr, bool wide, F&& f) {
    auto go = [&](auto tc) {
        constexpr int TPR = decltype(tc)::value;
        row_form<TPR>(rows, wide, [&](auto form) { f(tc, form); });
    };
    switch (tpr) {
        case 8: go(std::integral_constant<int, 8>()); break;
        case 4: go(std::integral_constant<int, 4>()); break;
        case 2: go(std::integral_constant<int, 2>()); break;
        default: go(std::integral_constant<int, 1>()); break;
    }
}
template <class F>
int row_blocks(int64_t rows, int tpr, F) {
    return blocks_for(F::value == kRow32 ? rows : rows * tpr);
}
// Whether kRow32 is the better form of a large launch: FP64 rows of two or
// four lanes, and the float32 rows that level_tpr gives eight.
template <typename T>
bool row_wide(int tpr, int base) {
    return sizeof(T) == 8 ? tpr <= 4 : tpr == 8 && base == 2;
}

template <typename T, typename BT, typename OT>
void jacobi(const MgLevel& L, const T* xi, const BT* b, OT* xo, const int* flag, cudaStream_t st) {
    const int tpr = level_tpr<T>(L);
    row_launch(L.N, tpr, row_wide<T>(tpr, L.tpr), [&](auto tc, auto form) {
        launch_chained(true, mg_jacobi_kernel<T, BT, OT, decltype(tc)::value, decltype(form)::value>,
                       row_blocks(L.N, tpr, form), kT, 0, st, L.row_ptr, L.col, Sel<T>::val(L), L.N, xi, b,
                       Sel<T>::dinv(L), xo, flag);
    });
}

template <typename T, typename BT>
void resid(const MgLevel& L, const T* x, const BT* b, T* r, const int* flag, cudaStream_t st) {
    const int tpr = level_tpr<T>(L);
    row_launch(L.N, tpr, row_wide<T>(tpr, L.tpr), [&](auto tc, auto form) {
        launch_chained(true, mg_resid_kernel<T, BT, decltype(tc)::value, decltype(form)::value>,
                       row_blocks(L.N, tpr, form), kT, 0, st, L.row_ptr, L.col, Sel<T>::val(L), L.N, x, b, r, flag);
    });
}

template <typename T>
void restrict_to(const MgLevel& L, int64_t nc, const T* r, T* bc, const int* flag, cudaStream_t st) {
    row_launch(nc, L.rtpr, row_wide<T>(L.rtpr, L.rtpr), [&](auto tc, auto form) {
        launch_chained(true, mg_restrict_kernel<T, decltype(tc)::value, decltype(form)::value>,
                       row_blocks(nc, L.rtpr, form), kT, 0, st, L.rrow, L.rcol, Sel<T>::rval(L), nc, r, L.N, bc, flag);
    });
}

// The small levels' part of the cycle by one block, its vectors in shared
// memory: a level of some hundred nodes is a few microseconds of launch
// latency per operation (six per level) and a fraction of one of work.  Every
// row is summed by the same lanes in the same order as in the kernels above,
// so the result has the same bits.  The operators, read by every sweep, and
// as many of the transfers as fit are copied to shared memory while the
// previous kernel of the chain still runs (a batch of rows read from L2 is
// two or three dependent round trips of ~700 cycles: the restriction alone
// took 6.5k cycles).
// 845 + 190 + 45 rows: 15 to 20 us, 14 launches of 3 before.  (A cluster of 16 blocks, up
// to 20k rows, took 88 us for five levels: its barrier costs 600 to 1,700
// cycles and a neighbour in another block's shared memory or in L2 500 to
// 700, once per operation and entry.)
constexpr int kTailT = 1024;
constexpr int kTailLevels = 16;
constexpr int kTailSmem = 208 * 1024;

template <typename T>
struct TailLevel {
    int n, tpr, rtpr;  // rows; lanes per row of A and of the restriction into the next level
    int nnz;
    const int64_t* row_ptr;
    const int* col;
    const T* val;
    const T* w;
    const int32_t* pidx;
    const T* pval;
    const int64_t* rrow;
    const int32_t* rcol;
    const T* rval;
};

// An array that the kernel copies to shared memory first.
struct TailCopy {
    const void* src;
    int bytes, dst;
};
constexpr int kTailCopies = 24;

template <typename T>
struct TailCycle {
    int levels, nu, copies;
    TailCopy copy[kTailCopies];
    // byte offsets of the copies in shared memory, -1: read from global memory
    int a_ptr[kTailLevels], a_col[kTailLevels], a_val[kTailLevels];
    int r_ptr[kTailLevels], r_col[kTailLevels], r_val[kTailLevels];
    const T* minv;
    Live<T> b;  // right-hand side and result of the first level (not TOP)
    T* x;
    TailLevel<T> lv[kTailLevels];
};

// Rows of a CSR matrix by one block, TPR lanes per row: f(i, sum) in one lane.
template <typename T, int TPR, class RP, class CP, class F>
__device__ __forceinline__ void tail_rows(const RP* row_ptr, const CP* col, const T* val, const T* x, int nx, int n,
                                          F&& f) {
    (void)nx;  // length of x: bound of the checked build's tests
    const int sub = threadIdx.x & (TPR - 1), off = (threadIdx.x & 31) / TPR;
    for (int base = (int)threadIdx.x / TPR - off; base < n; base += kTailT / TPR) {
        const int i = base + off;
        int a = 0, e = 0;
        if (i < n) {
            a = (int)row_ptr[i];
            e = (int)row_ptr[i + 1];
        }
        T sum = T(0);
        // batches of independent loads; the sum runs in the order of the entries
        for (int k = a + sub; k < e; k += 6 * TPR) {
            T v[6], xv[6];
#pragma unroll
            for (int u = 0; u < 6; ++u) {
                const bool in = k + u * TPR < e;
                v[u] = in ? val[k + u * TPR] : T(0);
                xv[u] = in ? RB_AT(x, (int)col[k + u * TPR], nx) : T(0);
            }
#pragma unroll
            for (int u = 0; u < 6; ++u)
                if (k + u * TPR < e) sum = fmaT<T>(v[u], xv[u], sum);
        }
#pragma unroll
        for (int o = TPR / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o, TPR);
        if (i < n && sub == 0) f(i, sum);
    }
}

template <typename T, class RP, class CP, class F>
__device__ __forceinline__ void tail_csr(int tpr, const RP* row_ptr, const CP* col, const T* val, const T* x, int nx,
                                         int n, F&& f) {
    if (tpr == 8) tail_rows<T, 8>(row_ptr, col, val, x, nx, n, f);
    else if (tpr == 4) tail_rows<T, 4>(row_ptr, col, val, x, nx, n, f);
    else if (tpr == 2) tail_rows<T, 2>(row_ptr, col, val, x, nx, n, f);
    else tail_rows<T, 1>(row_ptr, col, val, x, nx, n, f);
}

// TOP: level 0 is the first one, its right-hand side and result are the
// caller's FP64 vectors.
template <typename T, bool TOP>
__global__ void __launch_bounds__(kTailT) mg_tail_kernel(const __grid_constant__ TailCycle<T> c, Live<double> b64,
                                                         double* x64, const int* flag) {
    extern __shared__ __align__(16) unsigned char tail_smem[];
    T* vec = reinterpret_cast<T*>(tail_smem);  // per level: two iterates, residual, right-hand side
    const int tid = (int)threadIdx.x, last = c.levels - 1;
    for (int k = 0; k < c.copies; ++k) {
        const TailCopy& q = c.copy[k];
        const char* src = static_cast<const char*>(q.src);
        char* dst = reinterpret_cast<char*>(tail_smem) + q.dst;
        const int whole = q.bytes & ~15;
        for (int o = tid * 16; o < whole; o += kTailT * 16)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst + o)),
                         "l"(src + o));
        for (int o = whole + tid * 4; o < q.bytes; o += kTailT * 4)
            *reinterpret_cast<int*>(dst + o) = *reinterpret_cast<const int*>(src + o);
    }
    auto at = [&](int off, const auto* global) {
        using P = decltype(global);
        return off >= 0 ? reinterpret_cast<P>(tail_smem + off) : global;
    };
    auto a_ptr = [&](int l) { return at(c.a_ptr[l], c.lv[l].row_ptr); };
    auto a_col = [&](int l) { return at(c.a_col[l], c.lv[l].col); };
    auto a_val = [&](int l) { return at(c.a_val[l], c.lv[l].val); };
    asm volatile("cp.async.wait_all;" ::: "memory");
    pdl_wait();
    pdl_next();
    if (stopped(flag)) return;
    for (int i = tid; i < c.lv[0].n; i += kTailT) vec[3 * c.lv[0].n + i] = TOP ? (T)b64[i] : c.b[i];
    __syncthreads();
    T* v = vec;  // the level's vectors
    for (int l = 0; l < last; ++l) {
        const TailLevel<T>& L = c.lv[l];
        const int n = L.n;
        T *cur = v, *oth = v + n, *r = v + 2 * n, *b = v + 3 * n, *bc = v + 4 * n + 3 * c.lv[l + 1].n;
        for (int i = tid; i < n; i += kTailT) cur[i] = __ldg(L.w + i) * b[i];
        __syncthreads();
        for (int k = 1; k < c.nu; ++k) {
            tail_csr<T>(L.tpr, a_ptr(l), a_col(l), a_val(l), cur, n, n,
                        [&](int i, T ax) { oth[i] = fmaT<T>(__ldg(L.w + i), b[i] - ax, cur[i]); });
            T* s = cur;
            cur = oth;
            oth = s;
            __syncthreads();
        }
        tail_csr<T>(L.tpr, a_ptr(l), a_col(l), a_val(l), cur, n, n, [&](int i, T ax) { r[i] = b[i] - ax; });
        __syncthreads();
        tail_csr<T>(L.rtpr, at(c.r_ptr[l], L.rrow), at(c.r_col[l], L.rcol), at(c.r_val[l], L.rval), r, n,
                    c.lv[l + 1].n, [&](int i, T s) { bc[i] = s; });
        __syncthreads();
        v += 4 * n;
    }
    {  // coarsest: one warp per row
        const int n = c.lv[last].n, lane = tid & 31;
        for (int i = tid >> 5; i < n; i += kTailT / 32) {
            T acc = T(0);
            for (int j = lane; j < n; j += 32) acc = fmaT<T>(__ldg(c.minv + (int64_t)i * n + j), v[3 * n + j], acc);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) v[i] = acc;
        }
    }
    for (int l = last - 1; l >= 0; --l) {
        __syncthreads();
        const TailLevel<T>& L = c.lv[l];
        const int n = L.n, nc = c.lv[l + 1].n;
        // the coarse result: in the second iterate (an odd number of swaps),
        // in the first at the coarsest level
        const T* e = v + (l + 1 == last ? 0 : nc);
        (void)nc;
        v -= 4 * n;
        T* cur = v + ((c.nu & 1) ? 0 : n);
        T* oth = v + ((c.nu & 1) ? n : 0);
        const T* b = v + 3 * n;
        for (int i = tid; i < n; i += kTailT) {
            const PRow<T> p(L.pidx, L.pval, i);
            T acc = cur[i];
#pragma unroll
            for (int j = 0; j < kMgK; ++j) acc = fmaT<T>(p.v[j], RB_AT(e, p.c[j], nc), acc);
            cur[i] = acc;
        }
        for (int k = 0; k < c.nu; ++k) {
            __syncthreads();
            tail_csr<T>(L.tpr, a_ptr(l), a_col(l), a_val(l), cur, n, n,
                        [&](int i, T ax) { oth[i] = fmaT<T>(__ldg(L.w + i), b[i] - ax, cur[i]); });
            T* s = cur;
            cur = oth;
            oth = s;
        }
    }
    __syncthreads();
    const int n = c.lv[0].n;
    const T* res = vec + (last == 0 ? 0 : n);
    for (int i = tid; i < n; i += kTailT) {
        if constexpr (TOP) x64[i] = (double)res[i];
        else c.x[i] = res[i];
    }
}

// Matrix entries of the first level up to which one block takes it: a sweep
// then costs less than a launch, and the operators fit shared memory (FP64: 2
// multiply-adds per clock).
template <typename T>
constexpr int64_t tail_entries() {
    return sizeof(T) == 8 ? 6144 : 12288;
}

// The cycle of levels [first, n_levels) in one launch; false where it does
// not apply.
template <typename T, bool TOP>
bool tail_cycle(const MgHierarchy& h, int first, const double* b, double* x, const int* flag, cudaStream_t st,
                bool chained) {
    const int levels = h.n_levels - first;
    if (h.lv[first].nnz > tail_entries<T>() || levels > kTailLevels) return false;
    TailCycle<T> c;
    c.levels = levels;
    c.nu = h.nu;
    c.minv = Sel<T>::minv(h.lv[h.n_levels - 1]);
    c.b = Sel<T>::b(h.lv[first]);
    c.x = levels == 1 ? Sel<T>::x(h.lv[first]) : Sel<T>::t(h.lv[first]);
    size_t smem = 0;
    for (int l = 0; l < levels; ++l) {
        const MgLevel& L = h.lv[first + l];
        const bool last = l == levels - 1;
        TailLevel<T>& t = c.lv[l];
        t = TailLevel<T>{};
        t.n = (int)L.N;
        t.nnz = (int)L.nnz;
        t.tpr = level_tpr<T>(L);
        t.row_ptr = L.row_ptr;
        t.col = L.col;
        t.val = Sel<T>::val(L);
        t.w = Sel<T>::dinv(L);
        if (!last) {
            t.rtpr = L.rtpr;
            t.pidx = L.pidx;
            t.pval = Sel<T>::pval(L);
            t.rrow = L.rrow;
            t.rcol = L.rcol;
            t.rval = Sel<T>::rval(L);
        }
        smem += 4 * (size_t)L.N * sizeof(T);
    }
    if (smem > kTailSmem) return false;
    // copies while they fit: the operators first, then the restrictions
    c.copies = 0;
    auto take = [&](const void* src, size_t bytes) {
        const size_t at = align_up(smem, 16);
        if (c.copies >= kTailCopies || at + bytes > kTailSmem || ((uintptr_t)src & 15) != 0) return -1;
        c.copy[c.copies++] = TailCopy{src, (int)bytes, (int)at};
        smem = at + bytes;
        return (int)at;
    };
    for (int l = 0; l < kTailLevels; ++l)
        c.a_ptr[l] = c.a_col[l] = c.a_val[l] = c.r_ptr[l] = c.r_col[l] = c.r_val[l] = -1;
    for (int l = 0; l + 1 < levels; ++l) {
        const TailLevel<T>& t = c.lv[l];
        c.a_val[l] = take(t.val, (size_t)t.nnz * sizeof(T));
        c.a_col[l] = take(t.col, (size_t)t.nnz * sizeof(int));
        c.a_ptr[l] = take(t.row_ptr, (size_t)(t.n + 1) * sizeof(int64_t));
    }
    for (int l = levels - 2; l >= 0; --l) {
        const TailLevel<T>& t = c.lv[l];
        c.r_col[l] = take(t.rcol, (size_t)t.n * kMgK * sizeof(int));
        c.r_val[l] = take(t.rval, (size_t)t.n * kMgK * sizeof(T));
        c.r_ptr[l] = take(t.rrow, (size_t)(c.lv[l + 1].n + 1) * sizeof(int64_t));
    }
    if (cudaFuncSetAttribute(mg_tail_kernel<T, TOP>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTailSmem) !=
        cudaSuccess)
        return false;
    launch_chained(chained, mg_tail_kernel<T, TOP>, 1, kTailT, smem, st, c, b, x, flag);
    return true;
}

// One level of the cycle: b (BT) in, result in x (OT) for level 0, in the
// level's own current-iterate buffer otherwise (returned).  chained: the
// first kernel continues a chain (launch_chained); the others always do.
template <typename T>
T* cycle_level(const MgHierarchy& h, int l, const void* bin, bool b_is_double, double* out, const int* flag,
               cudaStream_t st, int* launches, std::vector<int>* ev, bool chained) {
    const MgLevel& L = h.lv[l];
    const bool last_level = (l == h.n_levels - 1);
    const bool top = (l == 0);
    T* cur = Sel<T>::x(L);
    T* oth = Sel<T>::t(L);
    // small levels: the rest of the cycle in one launch (not the top level
    // while its sweeps are being timed)
    if (top ? b_is_double && !(ev && profiling()) &&
                  tail_cycle<T, true>(h, l, static_cast<const double*>(bin), out, flag, st, chained)
            : tail_cycle<T, false>(h, l, nullptr, nullptr, flag, st, chained)) {
        ++*launches;
        return last_level ? cur : oth;
    }
    auto launch_first = [&](T* x) {
        const int g = blocks_for(L.N);
        if (b_is_double)
            launch_chained(chained, mg_first_kernel<T, double>, g, kT, 0, st, L.N, static_cast<const double*>(bin),
                           Sel<T>::dinv(L), x, flag);
        else
            launch_chained(chained, mg_first_kernel<T, T>, g, kT, 0, st, L.N, static_cast<const T*>(bin),
                           Sel<T>::dinv(L), x, flag);
        ++*launches;
    };
    auto sweep = [&](T* xi, T* xo, double* xo64) {
        // finest-level sweeps are timed when profiling (algorithmic bytes:
        // matrix, row pointers, iterate once, rhs, D^-1, result)
        const int e = (top && ev) ? prof_begin(st) : -1;
        if (b_is_double) {
            const double* b = static_cast<const double*>(bin);
            if (xo64) jacobi<T, double, double>(L, xi, b, xo64, flag, st);
            else jacobi<T, double, T>(L, xi, b, xo, flag, st);
        } else {
            const T* b = static_cast<const T*>(bin);
            if (xo64) jacobi<T, T, double>(L, xi, b, xo64, flag, st);
            else jacobi<T, T, T>(L, xi, b, xo, flag, st);
        }
        if (top && ev) {
            const int64_t bytes = L.nnz * (int64_t)(sizeof(T) + 4) + 8 * (L.N + 1) +
                                  L.N * (int64_t)(2 * sizeof(T) + (b_is_double ? 8 : sizeof(T)) + sizeof(T)) +
                                  (xo64 ? L.N * (int64_t)(8 - sizeof(T)) : 0);
            prof_end(e, st, kProfMg, bytes);
            ev->push_back(e);
        }
        ++*launches;
    };
    if (last_level) {
        const int g = blocks_for((int64_t)L.N * 32);
        const T* mv = Sel<T>::minv(L);
        if (top) {
            launch_chained(chained, mg_dense_kernel<T, double, double>, g, kT, 0, st, (int)L.N, mv,
                           static_cast<const double*>(bin), out, flag);
        } else {
            launch_chained(chained, mg_dense_kernel<T, T, T>, g, kT, 0, st, (int)L.N, mv, static_cast<const T*>(bin),
                           cur, flag);
        }
        ++*launches;
        return cur;
    }
    // pre-smoothing
    launch_first(cur);
    for (int k = 1; k < h.nu; ++k) {
        sweep(cur, oth, nullptr);
        std::swap(cur, oth);
    }
    // residual, restriction, coarse correction
    if (b_is_double) resid<T, double>(L, cur, static_cast<const double*>(bin), Sel<T>::r(L), flag, st);
    else resid<T, T>(L, cur, static_cast<const T*>(bin), Sel<T>::r(L), flag, st);
    const MgLevel& C = h.lv[l + 1];
    restrict_to<T>(L, C.N, Sel<T>::r(L), Sel<T>::b(C), flag, st);
    *launches += 2;
    T* e = cycle_level<T>(h, l + 1, Sel<T>::b(C), false, nullptr, flag, st, launches, ev, true);
    launch_chained(true, mg_prolong_kernel<T>, blocks_for(L.N), kT, 0, st, L.N, L.pidx, Sel<T>::pval(L), e, C.N, cur,
                   flag);
    ++*launches;
    // post-smoothing; the last sweep of level 0 writes the FP64 output
    for (int k = 0; k < h.nu; ++k) {
        const bool final_top = top && k == h.nu - 1;
        sweep(cur, oth, final_top ? out : nullptr);
        if (!final_top) std::swap(cur, oth);
    }
    return cur;
}

}  // namespace

size_t mg_multi_coarse_floats(const MgHierarchy* h, int R) {
    if (!h) return 0;
    size_t t = 0;
    for (int l = 1; l < h->n_levels; ++l) t += (size_t)4 * h->lv[l].N * R;
    return t;
}

const MgHierarchy* mg_hierarchy(const rbffd_mg* h) {
    if (!h) return nullptr;
    const MgHierarchy* m = reinterpret_cast<const MgHierarchy*>(h);
    if (m->magic != kMgMagic || m->n_levels < 1) return nullptr;
    return m;
}

int64_t mg_fine_rows(const MgHierarchy* h) { return h ? h->lv[0].N : 0; }

bool mg_has_fp32(const MgHierarchy* h) { return h && h->has32; }

bool mg_is_transposed(const MgHierarchy* h) { return h && h->transposed; }

bool mg_is_galerkin(const MgHierarchy* h) { return h && h->galerkin; }

int mg_dirichlet_fix(const MgHierarchy* h, const double* r, double* y, const int* flag, cudaStream_t st,
                     bool chained) {
    if (!h || !r || !y || h->col_base != 0) return RBFFD_ERR_INVALID_ARG;
    const MgLevel& L = h->lv[0];
    launch_chained(chained, mg_bfix_kernel, blocks_for(L.N), kT, 0, st, L.row_ptr, L.col, L.val, L.N, L.mask, L.dinv, r,
                   y, flag);
    note_launches(1);
    RBFFD_LAUNCH_CHECK();
    return RBFFD_OK;
}

__global__ void __launch_bounds__(kT) mg_zero_dirichlet_kernel(int64_t N, const uint8_t* __restrict__ mask, double* y,
                                                               const int* flag) {
    pdl_wait();
    pdl_next();
    if (stopped(flag)) return;
    MG_ELEMS(N, i) if (mask[i]) y[i] = 0.0;
}

int mg_apply_interior(const MgHierarchy* h, bool fp32, const double* b, double* x, const int* flag, cudaStream_t st,
                      std::vector<int>* ev, bool chained) {
    if (!h || !b || !x || h->col_base != 0) return RBFFD_ERR_INVALID_ARG;
    if (fp32 && !h->has32) return RBFFD_ERR_INVALID_ARG;
    int launches = 0;
    if (fp32) cycle_level<float>(*h, 0, b, true, x, flag, st, &launches, ev, chained);
    else cycle_level<double>(*h, 0, b, true, x, flag, st, &launches, ev, chained);
    const MgLevel& L = h->lv[0];
    launch_chained(true, mg_zero_dirichlet_kernel, blocks_for(L.N), kT, 0, st, L.N, L.mask, x, flag);
    note_launches(launches + 1);
    RBFFD_LAUNCH_CHECK();
    return RBFFD_OK;
}

int mg_apply(const MgHierarchy* h, bool fp32, const double* b, double* x, const int* flag, cudaStream_t st,
             std::vector<int>* ev, bool chained) {
    if (!h || !b || !x || h->col_base != 0) return RBFFD_ERR_INVALID_ARG;
    if (fp32 && !h->has32) return RBFFD_ERR_INVALID_ARG;
    int launches = 0;
    if (fp32) cycle_level<float>(*h, 0, b, true, x, flag, st, &launches, ev, chained);
    else cycle_level<double>(*h, 0, b, true, x, flag, st, &launches, ev, chained);
    note_launches(launches);
    RBFFD_LAUNCH_CHECK();
    // adjoint: the transpose of the boundary-eliminated forward cycle
    // E_b + B (I - A E_b) is B^T followed by the Dirichlet back substitution
    if (h->transposed) return mg_dirichlet_fix(h, b, x, flag, st, true);
    return RBFFD_OK;
}

}  // namespace rbffd

// ---------------------------------------------------------------- C ABI -----
extern "C" size_t rbffd_mg_workspace_size(int64_t N, int64_t nnz) {
    RBFFD_NVTX("rbffd_mg_workspace_size");
    (void)nnz;  // the fine matrix stays the caller's
    if (N <= 0 || N > 0x7fffffffLL) return 0;
    return rbffd::mg_layout(nullptr, N, nullptr, nullptr);
}

extern "C" int rbffd_mg_levels(const rbffd_mg* mg, int64_t* n_nodes) {
    RBFFD_NVTX("rbffd_mg_levels");
    const rbffd::MgHierarchy* h = rbffd::mg_hierarchy(mg);
    if (!h) return 0;
    if (n_nodes)
        for (int l = 0; l < RBFFD_MG_MAX_LEVELS; ++l) n_nodes[l] = l < h->n_levels ? h->lv[l].N : 0;
    return h->n_levels;
}

extern "C" int rbffd_mg_level(const rbffd_mg* mg, int32_t level, rbffd_mg_level_info* out) {
    RBFFD_NVTX("rbffd_mg_level");
    using namespace rbffd;
    if (!mg || !out) return RBFFD_ERR_INVALID_ARG;
    MgHierarchy h;
    std::memcpy(&h, mg, sizeof(h));
    if (h.magic != kMgMagic || level < 0 || level >= h.n_levels) return RBFFD_ERR_INVALID_ARG;
    const MgLevel& L = h.lv[level];
    const bool coarsest = level == h.n_levels - 1;
    std::memset(out, 0, sizeof(*out));
    out->n_nodes = L.N;
    out->xy = L.xy;
    out->is_dirichlet = L.mask;
    out->A.n_rows = L.N;
    out->A.nnz = L.nnz;
    out->A.row_ptr = L.row_ptr;
    out->A.col = L.col;
    out->A.val = L.val;
    out->A.dtype = 0;
    out->w = L.dinv;
    out->p_idx = coarsest ? nullptr : L.pidx;
    out->p_val = coarsest ? nullptr : L.pval;
    out->p_k = coarsest ? 0 : kMgK;
    out->minv = coarsest ? L.minv : nullptr;
    return RBFFD_OK;
}

extern "C" int rbffd_mg_adjoint_of(const rbffd_mg* fwd, const rbffd_csr* AT, const rbffd_csr* AT32, rbffd_mg* mg,
                                   void* ws, size_t ws_bytes, void* stream) {
    RBFFD_NVTX("rbffd_mg_adjoint_of");
    using namespace rbffd;
    if (!mg) return RBFFD_ERR_INVALID_ARG;
    std::memset(mg, 0, sizeof(*mg));
    const MgHierarchy* F = mg_hierarchy(fwd);
    if (!F || !AT || !AT->row_ptr || !AT->col || !AT->val || AT->dtype != 0) return RBFFD_ERR_INVALID_ARG;
    if (AT32 && (!AT32->val || AT32->dtype != 1 || AT32->n_rows != AT->n_rows || AT32->nnz != AT->nnz ||
                 AT32->row_ptr != AT->row_ptr || AT32->col != AT->col))
        return RBFFD_ERR_INVALID_ARG;
    return mg_adjoint_of(*F, AT, AT32 ? static_cast<const float*>(AT32->val) : nullptr, mg, ws, ws_bytes,
                         as_stream(stream));
}

extern "C" size_t rbffd_mg_galerkin_workspace_size(const rbffd_mg* fwd) {
    RBFFD_NVTX("rbffd_mg_galerkin_workspace_size");
    using namespace rbffd;
    const MgHierarchy* F = mg_hierarchy(fwd);
    if (!F || F->transposed) return 0;
    return mg_galerkin_workspace(*F);
}

extern "C" int rbffd_mg_galerkin_adjoint(const rbffd_mg* fwd, const rbffd_csr* AT, const rbffd_csr* AT32,
                                         rbffd_mg* mg, void* ws, size_t ws_bytes, void* stream) {
    RBFFD_NVTX("rbffd_mg_galerkin_adjoint");
    using namespace rbffd;
    if (!mg) return RBFFD_ERR_INVALID_ARG;
    std::memset(mg, 0, sizeof(*mg));
    const MgHierarchy* F = mg_hierarchy(fwd);
    if (!F || !AT || !AT->row_ptr || !AT->col || !AT->val || AT->dtype != 0) return RBFFD_ERR_INVALID_ARG;
    if (AT32 && (!AT32->val || AT32->dtype != 1 || AT32->n_rows != AT->n_rows || AT32->nnz != AT->nnz ||
                 AT32->row_ptr != AT->row_ptr || AT32->col != AT->col))
        return RBFFD_ERR_INVALID_ARG;
    return mg_galerkin_adjoint(*F, AT, AT32 ? static_cast<const float*>(AT32->val) : nullptr, mg, ws, ws_bytes,
                               as_stream(stream));
}

extern "C" int rbffd_mg_apply(const rbffd_mg* mg, int32_t fp32, const double* b, double* x, void* stream) {
    RBFFD_NVTX("rbffd_mg_apply");
    using namespace rbffd;
    const MgHierarchy* h = mg_hierarchy(mg);
    if (!h || !b || !x || b == x) return RBFFD_ERR_INVALID_ARG;
    return mg_apply(h, fp32 != 0, b, x, nullptr, as_stream(stream));
}

extern "C" int rbffd_mg_setup(const double* xy, const uint8_t* is_dirichlet, int64_t N, const rbffd_csr* A,
                              const rbffd_csr* A32, int32_t nu, double omega, rbffd_mg* mg, void* ws,
                              size_t ws_bytes, void* stream) {
    RBFFD_NVTX("rbffd_mg_setup");
    using namespace rbffd;
    if (!mg) return RBFFD_ERR_INVALID_ARG;
    std::memset(mg, 0, sizeof(*mg));
    if (!xy || !is_dirichlet || !A || !A->row_ptr || !A->col || !A->val || A->dtype != 0 || N <= 0 ||
        N > 0x7fffffffLL || A->n_rows != N || A->nnz <= 0)
        return RBFFD_ERR_INVALID_ARG;
    if (A32 && (!A32->val || A32->dtype != 1 || A32->n_rows != N || A32->nnz != A->nnz || A32->row_ptr != A->row_ptr ||
                A32->col != A->col))
        return RBFFD_ERR_INVALID_ARG;
    return mg_setup_core(xy, is_dirichlet, N, A->row_ptr, A->col, static_cast<const double*>(A->val),
                         A32 ? static_cast<const float*>(A32->val) : nullptr, A->nnz, 0, nu, omega, mg, ws, ws_bytes,
                         as_stream(stream), false);
}

extern "C" int rbffd_mg_setup_geometry(const double* xy, const uint8_t* is_dirichlet, int64_t N, int32_t nu,
                                       double omega, rbffd_mg* mg, void* ws, size_t ws_bytes, void* stream) {
    RBFFD_NVTX("rbffd_mg_setup_geometry");
    using namespace rbffd;
    if (!mg) return RBFFD_ERR_INVALID_ARG;
    std::memset(mg, 0, sizeof(*mg));
    if (!xy || !is_dirichlet || N <= 0 || N > 0x7fffffffLL) return RBFFD_ERR_INVALID_ARG;
    return mg_setup_geometry(xy, is_dirichlet, N, 0, nu, omega, mg, ws, ws_bytes, as_stream(stream), false);
}

extern "C" int rbffd_mg_setup_operator(rbffd_mg* mg, const rbffd_csr* A, const rbffd_csr* A32, void* stream) {
    RBFFD_NVTX("rbffd_mg_setup_operator");
    using namespace rbffd;
    if (!mg) return RBFFD_ERR_INVALID_ARG;
    const MgHierarchy* g = reinterpret_cast<const MgHierarchy*>(mg);
    if (g->magic != kMgGeometryMagic || g->transposed) return RBFFD_ERR_INVALID_ARG;
    const int64_t N = g->lv[0].N;
    if (!A || !A->row_ptr || !A->col || !A->val || A->dtype != 0 || A->n_rows != N || A->nnz <= 0)
        return RBFFD_ERR_INVALID_ARG;
    if (A32 && (!A32->val || A32->dtype != 1 || A32->n_rows != N || A32->nnz != A->nnz || A32->row_ptr != A->row_ptr ||
                A32->col != A->col))
        return RBFFD_ERR_INVALID_ARG;
    return mg_setup_operator(mg, A->row_ptr, A->col, static_cast<const double*>(A->val),
                             A32 ? static_cast<const float*>(A32->val) : nullptr, A->nnz, as_stream(stream));
}

extern "C" int rbffd_mg_setup_adjoint(const double* xy, const uint8_t* is_dirichlet, int64_t N, const rbffd_csr* AT,
                                      const rbffd_csr* AT32, int32_t nu, double omega, rbffd_mg* mg, void* ws,
                                      size_t ws_bytes, void* stream) {
    RBFFD_NVTX("rbffd_mg_setup_adjoint");
    using namespace rbffd;
    if (!mg) return RBFFD_ERR_INVALID_ARG;
    std::memset(mg, 0, sizeof(*mg));
    if (!xy || !is_dirichlet || !AT || !AT->row_ptr || !AT->col || !AT->val || AT->dtype != 0 || N <= 0 ||
        N > 0x7fffffffLL || AT->n_rows != N || AT->nnz <= 0)
        return RBFFD_ERR_INVALID_ARG;
    if (AT32 && (!AT32->val || AT32->dtype != 1 || AT32->n_rows != N || AT32->nnz != AT->nnz ||
                 AT32->row_ptr != AT->row_ptr || AT32->col != AT->col))
        return RBFFD_ERR_INVALID_ARG;
    return mg_setup_core(xy, is_dirichlet, N, AT->row_ptr, AT->col, static_cast<const double*>(AT->val),
                         AT32 ? static_cast<const float*>(AT32->val) : nullptr, AT->nnz, 0, nu, omega, mg, ws,
                         ws_bytes, as_stream(stream), true);
}

// The adjoint hierarchy of a built forward one: the coarse node sets, the
// smoother weights and the interpolation are the forward ones (copied), the
// level operators are transposed, the transfers swapped, and the coarsest
// transposed operator inverted; the same arrays rbffd_mg_setup_adjoint
// builds from scratch, at the cost of the transposes.
int rbffd::mg_adjoint_of(const MgHierarchy& F, const rbffd_csr* AT, const float* val32, rbffd_mg* mg, void* ws,
                         size_t ws_bytes, cudaStream_t st) {
    std::memset(mg, 0, sizeof(*mg));
    const MgLevel& F0 = F.lv[0];
    const int64_t N = F0.N;
    if (F.transposed || F.col_base != 0 || AT->n_rows != N || AT->nnz != F0.nnz) return RBFFD_ERR_INVALID_ARG;
    if (val32 && !F.has32) return RBFFD_ERR_INVALID_ARG;
    if (!ws || ((uintptr_t)ws & (kAlign - 1)) != 0) return RBFFD_ERR_WORKSPACE;
    if (ws_bytes < mg_layout(nullptr, N, nullptr, nullptr)) return RBFFD_ERR_WORKSPACE;
    MgHierarchy h{};
    MgScratch s{};
    mg_layout(ws, N, &h, &s);
    h.nu = F.nu;
    h.omega = F.omega;
    h.has32 = val32 ? 1 : 0;
    h.col_base = 0;
    h.transposed = 1;
    RBFFD_CUDA_TRY(cudaMemsetAsync(s.flags, 0, sizeof(int) * 64, st));
    MgLevel& L0 = h.lv[0];
    L0.N = N;
    L0.row_ptr = AT->row_ptr;
    L0.col = AT->col;
    L0.val = static_cast<const double*>(AT->val);
    L0.val32 = val32;
    L0.nnz = AT->nnz;
    L0.tpr = tpr_for(N, AT->nnz);
    L0.xy = F0.xy;
    L0.mask = F0.mask;
    const int n_levels = F.n_levels;
    for (int l = 0; l < n_levels; ++l) {
        MgLevel& L = h.lv[l];
        const MgLevel& FL = F.lv[l];
        // W: the diagonal and the Dirichlet rows are those of the forward level
        RBFFD_CUDA_TRY(cudaMemcpyAsync(L.dinv, FL.dinv, sizeof(double) * L.N, cudaMemcpyDeviceToDevice, st));
        RBFFD_CUDA_TRY(cudaMemcpyAsync(L.dinv32, FL.dinv32, sizeof(float) * L.N, cudaMemcpyDeviceToDevice, st));
        if (l == n_levels - 1) {
            int rc = dense_inverse(L, 0, s, st);
            if (rc != RBFFD_OK) return rc;
            break;
        }
        MgLevel& C = h.lv[l + 1];
        const MgLevel& FC = F.lv[l + 1];
        const int64_t nc = FC.N;
        C.N = nc;
        RBFFD_CUDA_TRY(cudaMemcpyAsync(const_cast<double*>(C.xy), FC.xy, sizeof(double) * 2 * nc,
                                       cudaMemcpyDeviceToDevice, st));
        RBFFD_CUDA_TRY(cudaMemcpyAsync(const_cast<uint8_t*>(C.mask), FC.mask, nc, cudaMemcpyDeviceToDevice, st));
        rbffd_csr Ac{};
        Ac.n_rows = nc;
        Ac.nnz = FC.nnz;
        Ac.row_ptr = FC.row_ptr;
        Ac.col = FC.col;
        Ac.val = FC.val;
        Ac.dtype = 0;
        int rc = rbffd_transpose(&Ac, const_cast<int64_t*>(C.row_ptr), const_cast<int*>(C.col),
                                 const_cast<double*>(C.val), nullptr, s.tr_ws, s.tr_bytes, st);
        if (rc != RBFFD_OK) return rc;
        mg_f32_kernel<<<blocks_for(FC.nnz), kT, 0, st>>>(C.val, FC.nnz, const_cast<float*>(C.val32));
        C.nnz = FC.nnz;
        C.tpr = tpr_for(nc, FC.nnz);
        // transfers: R = P^T (raw), prolongation R_fwd^T = (N_c / N_f) P
        // without the coarse Dirichlet columns
        RBFFD_CUDA_TRY(cudaMemcpyAsync(L.pidx, FL.pidx, sizeof(int32_t) * L.N * kMgK, cudaMemcpyDeviceToDevice, st));
        RBFFD_CUDA_TRY(cudaMemcpyAsync(L.pval, FL.pval, sizeof(double) * L.N * kMgK, cudaMemcpyDeviceToDevice, st));
        mg_ellrow_kernel<<<blocks_for(L.N + 1), kT, 0, st>>>(L.N, s.prow);
        rbffd_csr P{};
        P.n_rows = L.N;
        P.nnz = L.N * kMgK;
        P.row_ptr = s.prow;
        P.col = L.pidx;
        P.val = L.pval;
        P.dtype = 0;
        if ((rc = rbffd_transpose(&P, L.rrow, L.rcol, L.rval, nullptr, s.tr_ws, s.tr_bytes, st)) != RBFFD_OK) return rc;
        mg_rscale_kernel<<<blocks_for(nc), kT, 0, st>>>(L.rrow, nc, nullptr, 1.0, L.rval, L.rval32);
        mg_pscale_kernel<<<blocks_for(L.N * kMgK), kT, 0, st>>>(L.N, L.pidx, C.mask, nc, (double)nc / (double)L.N,
                                                                 L.pval, L.pval32);
        note_launches(4);
        RBFFD_LAUNCH_CHECK();
        L.rtpr = tpr_for(nc, L.N * kMgK);
    }
    int flags[2] = {0, 0};
    RBFFD_CUDA_TRY(cudaMemcpyAsync(flags, s.flags, sizeof(flags), cudaMemcpyDeviceToHost, st));
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    if (flags[0]) return RBFFD_ERR_SINGULAR_STENCIL;
    h.n_levels = n_levels;
    h.magic = kMgMagic;
    std::memcpy(mg, &h, sizeof(h));
    return RBFFD_OK;
}

// Level sizes of a built hierarchy (the Galerkin hierarchy's layout).
static std::vector<int64_t> level_sizes(const rbffd::MgHierarchy& F) {
    std::vector<int64_t> nb;
    for (int l = 0; l < F.n_levels; ++l) nb.push_back(F.lv[l].N);
    return nb;
}

size_t rbffd::mg_galerkin_workspace(const MgHierarchy& F) {
    const std::vector<int64_t> nb = level_sizes(F);
    return mg_layout(nullptr, F.lv[0].N, nullptr, nullptr, &nb, kMgGalerkinRow);
}

// The adjoint hierarchy of a built forward one with Galerkin coarse
// operators: node sets, interpolation and transfers as in mg_adjoint_of
// (restriction P^T, prolongation (N_c / N_f) P without the coarse Dirichlet
// columns); each coarse operator the product R A P of the level above it
// (mg_galerkin_kernel), its smoother weights from its own diagonal, the
// coarsest inverted.
int rbffd::mg_galerkin_adjoint(const MgHierarchy& F, const rbffd_csr* AT, const float* val32, rbffd_mg* mg,
                               void* ws, size_t ws_bytes, cudaStream_t st) {
    std::memset(mg, 0, sizeof(*mg));
    const MgLevel& F0 = F.lv[0];
    const int64_t N = F0.N;
    if (F.transposed || F.col_base != 0 || AT->n_rows != N || AT->nnz != F0.nnz) return RBFFD_ERR_INVALID_ARG;
    if (val32 && !F.has32) return RBFFD_ERR_INVALID_ARG;
    if (!ws || ((uintptr_t)ws & (kAlign - 1)) != 0) return RBFFD_ERR_WORKSPACE;
    const std::vector<int64_t> nb = level_sizes(F);
    if (ws_bytes < mg_layout(nullptr, N, nullptr, nullptr, &nb, kMgGalerkinRow)) return RBFFD_ERR_WORKSPACE;
    static bool smem_set = false;
    if (!smem_set) {
        RBFFD_CUDA_TRY(cudaFuncSetAttribute(mg_galerkin_kernel<512, 256>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)gal_smem_bytes<512, 256>()));
        RBFFD_CUDA_TRY(cudaFuncSetAttribute(mg_galerkin_kernel<1024, 512>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)gal_smem_bytes<1024, 512>()));
        smem_set = true;
    }
    MgHierarchy h{};
    MgScratch s{};
    mg_layout(ws, N, &h, &s, &nb, kMgGalerkinRow);
    h.nu = F.nu;
    h.omega = F.omega;
    h.has32 = val32 ? 1 : 0;
    h.col_base = 0;
    h.transposed = 1;
    h.galerkin = 1;
    RBFFD_CUDA_TRY(cudaMemsetAsync(s.flags, 0, sizeof(int) * 64, st));
    MgLevel& L0 = h.lv[0];
    L0.N = N;
    L0.row_ptr = AT->row_ptr;
    L0.col = AT->col;
    L0.val = static_cast<const double*>(AT->val);
    L0.val32 = val32;
    L0.nnz = AT->nnz;
    L0.tpr = tpr_for(N, AT->nnz);
    L0.xy = F0.xy;
    L0.mask = F0.mask;
    // level 0's smoother: A^T has A's diagonal and Dirichlet rows
    RBFFD_CUDA_TRY(cudaMemcpyAsync(L0.dinv, F0.dinv, sizeof(double) * N, cudaMemcpyDeviceToDevice, st));
    RBFFD_CUDA_TRY(cudaMemcpyAsync(L0.dinv32, F0.dinv32, sizeof(float) * N, cudaMemcpyDeviceToDevice, st));
    const int n_levels = F.n_levels;
    for (int l = 0; l + 1 < n_levels; ++l) {
        MgLevel& L = h.lv[l];
        const MgLevel& FL = F.lv[l];
        MgLevel& C = h.lv[l + 1];
        const MgLevel& FC = F.lv[l + 1];
        const int64_t nc = FC.N;
        C.N = nc;
        RBFFD_CUDA_TRY(cudaMemcpyAsync(const_cast<double*>(C.xy), FC.xy, sizeof(double) * 2 * nc,
                                       cudaMemcpyDeviceToDevice, st));
        RBFFD_CUDA_TRY(cudaMemcpyAsync(const_cast<uint8_t*>(C.mask), FC.mask, nc, cudaMemcpyDeviceToDevice, st));
        // transfers: R = P^T (raw), prolongation (N_c / N_f) P without the
        // coarse Dirichlet columns
        RBFFD_CUDA_TRY(cudaMemcpyAsync(L.pidx, FL.pidx, sizeof(int32_t) * L.N * kMgK, cudaMemcpyDeviceToDevice, st));
        RBFFD_CUDA_TRY(cudaMemcpyAsync(L.pval, FL.pval, sizeof(double) * L.N * kMgK, cudaMemcpyDeviceToDevice, st));
        mg_ellrow_kernel<<<blocks_for(L.N + 1), kT, 0, st>>>(L.N, s.prow);
        rbffd_csr P{};
        P.n_rows = L.N;
        P.nnz = L.N * kMgK;
        P.row_ptr = s.prow;
        P.col = L.pidx;
        P.val = L.pval;
        P.dtype = 0;
        int rc = rbffd_transpose(&P, L.rrow, L.rcol, L.rval, nullptr, s.tr_ws, s.tr_bytes, st);
        if (rc != RBFFD_OK) return rc;
        mg_rscale_kernel<<<blocks_for(nc), kT, 0, st>>>(L.rrow, nc, nullptr, 1.0, L.rval, L.rval32);
        mg_pscale_kernel<<<blocks_for(L.N * kMgK), kT, 0, st>>>(L.N, L.pidx, C.mask, nc, (double)nc / (double)L.N,
                                                                 L.pval, L.pval32);
        note_launches(3);
        RBFFD_LAUNCH_CHECK();
        L.rtpr = tpr_for(nc, L.N * kMgK);
        // C = R A P: rows staged (small tables first, the large ones if a row
        // overflowed them), row pointer, rows placed
        int* cnt = s.pos;
        int* over = s.flags + 2;
        int64_t* crow = const_cast<int64_t*>(C.row_ptr);
        int64_t cnnz = 0;
        const int64_t stage_cap = std::min(s.gal_cap, nc * (int64_t)kMgGalerkinRow);
        for (int large = 0; large < 2; ++large) {
            RBFFD_CUDA_TRY(cudaMemsetAsync(s.gal_total, 0, sizeof(unsigned long long), st));
            RBFFD_CUDA_TRY(cudaMemsetAsync(over, 0, sizeof(int), st));
            if (!large)
                mg_galerkin_kernel<512, 256><<<sm_count() * 6, kGalWarps * 32, gal_smem_bytes<512, 256>(), st>>>(
                    nc, L.rrow, L.rcol, L.rval, L.row_ptr, L.col, L.val, L.pidx, L.pval, C.mask, cnt, s.gal_start,
                    s.gal_total, stage_cap, s.gal_col, s.gal_val, over, L.N, L.nnz);
            else
                mg_galerkin_kernel<1024, 512><<<sm_count() * 3, kGalWarps * 32, gal_smem_bytes<1024, 512>(), st>>>(
                    nc, L.rrow, L.rcol, L.rval, L.row_ptr, L.col, L.val, L.pidx, L.pval, C.mask, cnt, s.gal_start,
                    s.gal_total, stage_cap, s.gal_col, s.gal_val, over, L.N, L.nnz);
            note_launches(1);
            RBFFD_LAUNCH_CHECK();
            RBFFD_CUDA_TRY(exclusive_scan<int64_t>(CountLoad64{cnt}, nc, crow, s.sums64, crow + nc, st));
            int ovf = 0;
            RBFFD_CUDA_TRY(cudaMemcpyAsync(&cnnz, crow + nc, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
            RBFFD_CUDA_TRY(cudaMemcpyAsync(&ovf, over, sizeof(int), cudaMemcpyDeviceToHost, st));
            RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
            if (!ovf) break;
            // a row wider than the large tables, or more entries than the layout holds
            if (large) return RBFFD_ERR_WORKSPACE;
        }
        if (cnnz > nc * (int64_t)kMgGalerkinRow) return RBFFD_ERR_WORKSPACE;
        mg_galerkin_place_kernel<<<blocks_for(nc * 32), kT, 0, st>>>(nc, s.gal_start, crow, s.gal_col, s.gal_val,
                                                                     const_cast<int*>(C.col),
                                                                     const_cast<double*>(C.val),
                                                                     const_cast<float*>(C.val32), stage_cap, cnnz);
        C.nnz = cnnz;
        C.tpr = tpr_for(nc, cnnz);
        mg_diag_kernel<<<blocks_for(nc), kT, 0, st>>>(C.row_ptr, C.col, C.val, nc, 0, C.mask, h.omega, C.dinv,
                                                      C.dinv32, s.flags + 1);
        note_launches(2);
        RBFFD_LAUNCH_CHECK();
    }
    {
        const int rc = dense_inverse(h.lv[n_levels - 1], 0, s, st);
        if (rc != RBFFD_OK) return rc;
    }
    int flags[2] = {0, 0};
    RBFFD_CUDA_TRY(cudaMemcpyAsync(flags, s.flags, sizeof(flags), cudaMemcpyDeviceToHost, st));
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    if (flags[0] || flags[1]) return RBFFD_ERR_SINGULAR_STENCIL;
    h.n_levels = n_levels;
    h.magic = kMgMagic;
    std::memcpy(mg, &h, sizeof(h));
    return RBFFD_OK;
}

int rbffd::mg_setup_geometry(const double* xy, const uint8_t* is_dirichlet, int64_t N, int col_base, int nu,
                             double omega, rbffd_mg* mg, void* ws, size_t ws_bytes, cudaStream_t st,
                             bool transposed) {
    using namespace rbffd;
    std::memset(mg, 0, sizeof(*mg));
    if (nu < 1 || nu > 8 || !(omega > 0.0 && omega < 1.0)) return RBFFD_ERR_INVALID_ARG;
    if (((uintptr_t)xy & 15) != 0) return RBFFD_ERR_INVALID_ARG;
    if (!ws || ((uintptr_t)ws & (kAlign - 1)) != 0) return RBFFD_ERR_WORKSPACE;
    const size_t need = mg_layout(nullptr, N, nullptr, nullptr);
    if (ws_bytes < need) return RBFFD_ERR_WORKSPACE;

    MgHierarchy h{};
    MgScratch s{};
    mg_layout(ws, N, &h, &s);
    h.magic = 0;
    h.nu = nu;
    h.omega = omega;
    h.col_base = col_base;
    h.transposed = transposed ? 1 : 0;
    h.ws = ws;
    h.ws_bytes = ws_bytes;
    RBFFD_CUDA_TRY(cudaMemsetAsync(s.flags, 0, sizeof(int) * 64, st));

    MgLevel& L0 = h.lv[0];
    L0.N = N;
    L0.xy = xy;
    L0.mask = is_dirichlet;

    int levels = 1;
    int rc = RBFFD_OK;
    for (int l = 0;; ++l) {
        MgLevel& L = h.lv[l];
        if (L.N <= kMgCoarsest || l + 1 >= RBFFD_MG_MAX_LEVELS) {
            if (L.N > kMgCoarsest) return RBFFD_ERR_INVALID_ARG;
            // (a single level is the fine operator itself: inverted by the operator phase)
            if (l > 0 && (rc = dense_inverse(L, 0, s, st)) != RBFFD_OK) return rc;
            levels = l + 1;
            break;
        }
        MgLevel& C = h.lv[l + 1];
        int64_t nc = 0;
        if ((rc = coarsen(L, C, s, st, &nc)) != RBFFD_OK) return rc;
        C.N = nc;
        // coarse operator: stencils, weights, Dirichlet-row assembly
        if ((rc = rbffd_stencils(C.xy, nc, kMgCoarseN, s.sidx, s.knn_ws, s.knn_bytes, st)) != RBFFD_OK) return rc;
        if ((rc = coarse_weights(C.xy, s.sidx, nc, kMgCoarseN, kMgCoarseM, s.sw, s.sstat, st)) != RBFFD_OK) return rc;
        mg_count_kernel<<<blocks_for(nc), kT, 0, st>>>(s.sstat, C.mask, nc, s.flags);
        note_launches(1);
        // (adjoint hierarchy: assembled into scratch, then transposed into the level)
        int64_t* crow = transposed ? s.a_row : const_cast<int64_t*>(C.row_ptr);
        if ((rc = rbffd_assemble_pattern(C.mask, nc, kMgCoarseN, crow, s.asm_ws, s.asm_bytes, st)) != RBFFD_OK)
            return rc;
        int64_t cnnz = 0;
        RBFFD_CUDA_TRY(cudaMemcpyAsync(&cnnz, crow + nc, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
        if (!transposed) {
            if ((rc = rbffd_assemble(s.sidx, s.sw, C.mask, nc, kMgCoarseN, crow, cnnz, const_cast<int*>(C.col),
                                     const_cast<double*>(C.val), const_cast<float*>(C.val32), st)) != RBFFD_OK)
                return rc;
        } else {
            if ((rc = rbffd_assemble(s.sidx, s.sw, C.mask, nc, kMgCoarseN, crow, cnnz, s.a_col, s.a_val, nullptr,
                                     st)) != RBFFD_OK)
                return rc;
            rbffd_csr Ac{};
            Ac.n_rows = nc;
            Ac.nnz = cnnz;
            Ac.row_ptr = s.a_row;
            Ac.col = s.a_col;
            Ac.val = s.a_val;
            Ac.dtype = 0;
            if ((rc = rbffd_transpose(&Ac, const_cast<int64_t*>(C.row_ptr), const_cast<int*>(C.col),
                                      const_cast<double*>(C.val), nullptr, s.tr_ws, s.tr_bytes, st)) != RBFFD_OK)
                return rc;
            mg_f32_kernel<<<blocks_for(cnnz), kT, 0, st>>>(C.val, cnnz, const_cast<float*>(C.val32));
            note_launches(1);
        }
        C.nnz = cnnz;
        C.tpr = tpr_for(nc, cnnz);
        mg_diag_kernel<<<blocks_for(nc), kT, 0, st>>>(C.row_ptr, C.col, C.val, nc, 0, C.mask, omega, C.dinv, C.dinv32,
                                                      s.flags + 1);
        note_launches(1);
        RBFFD_LAUNCH_CHECK();
        // prolongation: interpolation from the kMgK nearest coarse nodes
        if ((rc = knn_search(C.xy, nc, L.xy, L.N, kMgK, L.pidx, s.knn_ws, s.knn_bytes, st)) != RBFFD_OK) return rc;
        if ((rc = interp_weights(C.xy, nc, L.xy, L.N, L.pidx, kMgK, kMgInterpM, L.pval, s.pstat, st)) != RBFFD_OK)
            return rc;
        mg_pfix_kernel<<<blocks_for(L.N), kT, 0, st>>>(L.N, L.mask, s.pstat, L.pval, L.pval32, s.prow);
        note_launches(1);
        RBFFD_LAUNCH_CHECK();
        // restriction: (N_c / N_f) P^T, P viewed as an N_f x N_f matrix
        rbffd_csr P{};
        P.n_rows = L.N;
        P.nnz = L.N * kMgK;
        P.row_ptr = s.prow;
        P.col = L.pidx;
        P.val = L.pval;
        P.dtype = 0;
        if ((rc = rbffd_transpose(&P, L.rrow, L.rcol, L.rval, nullptr, s.tr_ws, s.tr_bytes, st)) != RBFFD_OK) return rc;
        const double cscale = (double)nc / (double)L.N;
        if (!transposed) {
            mg_rscale_kernel<<<blocks_for(nc), kT, 0, st>>>(L.rrow, nc, C.mask, cscale, L.rval, L.rval32);
        } else {
            // the transpose of the forward cycle: restrict with P^T, prolong
            // with R^T = (N_c / N_f) P without the coarse Dirichlet columns
            mg_rscale_kernel<<<blocks_for(nc), kT, 0, st>>>(L.rrow, nc, nullptr, 1.0, L.rval, L.rval32);
            mg_pscale_kernel<<<blocks_for(L.N * kMgK), kT, 0, st>>>(L.N, L.pidx, C.mask, nc, cscale, L.pval, L.pval32);
            note_launches(1);
        }
        note_launches(1);
        RBFFD_LAUNCH_CHECK();
        L.rtpr = tpr_for(nc, L.N * kMgK);
    }
    int flags[2] = {0, 0};
    RBFFD_CUDA_TRY(cudaMemcpyAsync(flags, s.flags, sizeof(flags), cudaMemcpyDeviceToHost, st));
    RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
    if (flags[0]) return RBFFD_ERR_SINGULAR_STENCIL;
    h.n_levels = levels;
    h.magic = kMgGeometryMagic;
    std::memcpy(mg, &h, sizeof(h));
    return RBFFD_OK;
}

int rbffd::mg_setup_operator(rbffd_mg* mg, const int64_t* row_ptr, const int* col, const double* val,
                             const float* val32, int64_t nnz, cudaStream_t st) {
    using namespace rbffd;
    MgHierarchy h;
    std::memcpy(&h, mg, sizeof(h));
    if (h.magic != kMgGeometryMagic || h.n_levels < 1) return RBFFD_ERR_INVALID_ARG;
    MgScratch s{};
    mg_layout(h.ws, h.lv[0].N, nullptr, &s);  // the scratch of the geometry phase's layout
    MgLevel& L0 = h.lv[0];
    const int64_t N = L0.N;
    L0.row_ptr = row_ptr;
    L0.col = col;
    L0.val = val;
    L0.val32 = val32;
    L0.nnz = nnz;
    L0.tpr = tpr_for(N, nnz);
    h.has32 = val32 ? 1 : 0;
    mg_diag_kernel<<<blocks_for(N), kT, 0, st>>>(L0.row_ptr, L0.col, L0.val, N, h.col_base, L0.mask, h.omega, L0.dinv,
                                                 L0.dinv32, s.flags + 1);
    note_launches(1);
    RBFFD_LAUNCH_CHECK();
    if (h.n_levels == 1) {  // the fine operator is the coarsest level
        int rc = dense_inverse(L0, h.col_base, s, st);
        if (rc != RBFFD_OK) return rc;
        int flag = 0;
        RBFFD_CUDA_TRY(cudaMemcpyAsync(&flag, s.flags, sizeof(int), cudaMemcpyDeviceToHost, st));
        RBFFD_CUDA_TRY(cudaStreamSynchronize(st));
        if (flag) return RBFFD_ERR_SINGULAR_STENCIL;
    }
    h.magic = kMgMagic;
    std::memcpy(mg, &h, sizeof(h));
    return RBFFD_OK;
}

int rbffd::mg_setup_core(const double* xy, const uint8_t* is_dirichlet, int64_t N, const int64_t* row_ptr,
                         const int* col, const double* val, const float* val32, int64_t nnz, int col_base, int nu,
                         double omega, rbffd_mg* mg, void* ws, size_t ws_bytes, cudaStream_t st, bool transposed) {
    int rc = mg_setup_geometry(xy, is_dirichlet, N, col_base, nu, omega, mg, ws, ws_bytes, st, transposed);
    if (rc == RBFFD_OK) rc = mg_setup_operator(mg, row_ptr, col, val, val32, nnz, st);
    if (rc != RBFFD_OK) std::memset(mg, 0, sizeof(*mg));
    return rc;
}
