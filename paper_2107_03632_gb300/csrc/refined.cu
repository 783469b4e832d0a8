// RBF-FD Laplacian weights by float32 elimination and fixed-point refinement
// (sm_103a): the FP64 null-space weight solve's fast path.
//
// The saddle-point system of a stencil (weights.cu: [Phi P; P^T 0] [w; l] =
// [f; g] in scaled coordinates) is eliminated once in float32 by the
// null-space method, and the solution is refined: the residual of the
// current (w, l) is formed in 64-bit fixed point from kernel values known to
// 2^-54 and monomials known to 2^-59 (fixed.cuh), the float32 factors solve
// for a correction, and the sum is kept in 64-bit fixed point.  Each step
// reduces the error by the float32 elimination's relative error (1e-3 to 1e-6
// on node sets of even density), so three to five solves reach the accuracy of
// the residual, which is that of the kernel values: more bits than FP64
// elimination carries.  (The monomials need more than the kernel values: near
// n = s they determine the weights alone, and everywhere the multipliers l, up
// to 2^12 times the weights, carry their errors into the residual.  With units
// of 2^-56 for both, m = 5, n = 22 had 3.7e-14 below.)  Largest error per
// stencil relative to its largest weight, against 180-bit fixed point (disk of
// 2,000 nodes, 15 sampled rows; here / FP64 elimination): m = 2, n = 12 8.3e-16
// / 1.6e-14; m = 4, n = 30 6.6e-15 / 4.5e-13; m = 5, n = 22 2.7e-15 / 1.6e-14;
// m = 6, n = 56 4.4e-14 / 8.4e-13.  A stencil whose corrections do not fall by
// 8x per step, whose pivots are small, or whose values leave the fixed-point ranges is
// marked and solved by the FP64 elimination kernel (weights.cu) in a second
// launch, which also decides every singular case.
//
// Why: the FP64 units issue 2 lanes per clock per SM (the float and integer
// pipes 128 and 64), and the FP64 elimination executes ~105k FP64
// lane-operations per stencil at m = 6, n = 56.  Here FP64 is left to the
// shift and scale of the coordinates and the final scaling.
//
// One thread per stencil node: NT = 16, 32 or 64 threads per stencil (two
// stencils per warp, one, or one per two warps; large stencils twice as many,
// see ref_geom).  A thread holds its row of
// the matrix being eliminated in registers; the pivot row goes through
// shared memory as 16-byte broadcasts.  Pivot steps rotate the columns by
// one, so the current column is always register 0 and the step loop needs no
// unrolling; after s steps the columns are back in place.  Integer sums make
// the result independent of the order of summation.
#include "common.cuh"
#include "fixed.cuh"
#include "internal.cuh"

#include <algorithm>

namespace rbffd {
namespace {

// Row stride in floats: a multiple of 4 (16-byte loads) and an odd one, so
// that the 16-byte loads of eight consecutive rows fall in distinct banks.
__host__ __device__ constexpr int odd4(int k) { return ((k + 3) / 4 | 1) * 4; }
__host__ __device__ constexpr int up4(int k) { return (k + 3) / 4 * 4; }
// Threads that sum one share of P^T d: a power of two, at least s.
__host__ __device__ constexpr int ref_ks(int s) { return s <= 4 ? 4 : s <= 8 ? 8 : s <= 16 ? 16 : 32; }

// Shared memory of one stencil (byte offsets).
//   phi   digits of |x_j - x_k|^3 2^56, entry [t - 1][j] for k = j + t mod n,
//         t = 1 .. n/2: every pair once (t = n/2 twice for even n), and both
//         of a thread's accesses in the residual are unit-stride
//   pd    digits of the monomials 2^61, [j][k], odd stride.  Before they are
//         formed the region holds W^T at its start and Phi11 at its end
//   F1    [Phi11; Phi21], n rows of LS (pivot nodes first): rows S.. become
//         T^T = (Phi12 - Phi11 X^T)^T, rows 0..S are inside pd
//   X [q][LS] = P2 P1^-1, C [s][LS] = P1^-1, Sm [q][LQ] = (Z^T Phi Z)^-1
struct RefGeom {
    int n, q, LQ;
    int phi, pd, F1, X, C, Sm, xy, xyf, prow, vr1, vr2, vg, vd0, vt, vy, vdw, dI, lI, pos, red, part, part2, bytes;
};

// Threads of a stencil: NT, one per node; with H = 2 as many again, which form
// the kernel values while the first eliminate P and share the sums.
RefGeom ref_geom(int NT, int H, int n, int s) {
    RefGeom g;
    g.n = n;
    g.q = n - s;
    g.LQ = odd4(std::max(g.q, 1));
    const int LS = odd4(s), LP = s | 1;
    int off = 0;
    auto take = [&](int bytes) {
        const int o = off;
        off += (bytes + 15) / 16 * 16;
        return o;
    };
    g.phi = take((n / 2) * n * 8);
    g.pd = take(n * LP * 8);
    const int tt = take(g.q * LS * 4);
    g.F1 = tt - s * LS * 4;
    g.X = take(g.q * LS * 4);
    g.C = take(s * LS * 4);
    g.Sm = take(g.q * g.LQ * 4);
    g.xy = take(n * 16);
    g.xyf = take(n * 8);
    g.prow = take(4 * (up4(NT) + 8) * 4);
    g.vr1 = take(LS * 4);
    g.vr2 = take(g.LQ * 4);
    g.vg = take(LS * 4);
    g.vd0 = take(LS * 4);
    g.vt = take(g.LQ * 4);
    g.vy = take(g.LQ * 4);
    g.vdw = take(n * 4);
    g.dI = take(2 * n * 4);
    g.lI = take(LS * 4);
    g.pos = take(n * 4);
    g.red = take(128);
    g.part = take((NT * H / ref_ks(s) - 1) * s * 16);
    g.part2 = take(H > 1 ? NT * 16 : 0);
    g.bytes = off;
    return g;
}

template <int NT>
__device__ __forceinline__ unsigned ref_mask() {
    if constexpr (NT >= 32) return 0xffffffffu;
    else return ((1u << NT) - 1u) << ((threadIdx.x & 31) & ~(NT - 1));
}

// Barrier over the stencil's TT threads (a block of its own above one warp).
template <int TT>
__device__ __forceinline__ void ref_sync() {
    if constexpr (TT <= 32) __syncwarp(ref_mask<TT>());
    else __syncthreads();
}

// Barrier over the first NT of them.
template <int NT, int TT>
__device__ __forceinline__ void ref_sync_part() {
    if constexpr (NT <= 32) __syncwarp(ref_mask<NT>());
    else if constexpr (NT == TT) __syncthreads();
    else asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}

// Maximum over the stencil's threads; `slot` alternates between consecutive
// calls so that one barrier per call is enough.
template <int TT>
__device__ __forceinline__ unsigned ref_max(unsigned v, unsigned* red, int slot) {
    v = __reduce_max_sync(ref_mask<TT>(), v);
    if constexpr (TT > 32) {
        constexpr int W = TT / 32;
        if ((threadIdx.x & 31) == 0) red[slot * 4 + (threadIdx.x >> 5)] = v;
        __syncthreads();
        v = max(red[slot * 4], red[slot * 4 + 1]);
        if constexpr (W == 4) v = max(v, max(red[slot * 4 + 2], red[slot * 4 + 3]));
    }
    return v;
}

__device__ __forceinline__ float dot4(const float4& a, const float4& b, float acc) {
    acc = fmaf(a.x, b.x, acc);
    acc = fmaf(a.y, b.y, acc);
    acc = fmaf(a.z, b.z, acc);
    return fmaf(a.w, b.w, acc);
}

// sum of a[k] b[k] over k < 4 n4 (rows padded with zeros), two chains
__device__ __forceinline__ float dotv(const float* a, const float* b, int n4) {
    const float4* pa = reinterpret_cast<const float4*>(a);
    const float4* pb = reinterpret_cast<const float4*>(b);
    float s0 = 0.f, s1 = 0.f;
    int k = 0;
#pragma unroll 2
    for (; k + 1 < n4; k += 2) {
        s0 = dot4(pa[k], pb[k], s0);
        s1 = dot4(pa[k + 1], pb[k + 1], s1);
    }
    if (k < n4) s0 = dot4(pa[k], pb[k], s0);
    return s0 + s1;
}

// Reciprocal and reciprocal square root to about one ulp of float32 (one
// instruction each; arguments are normal floats).
__device__ __forceinline__ float rcpf(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float rsqf(float a) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}

// The sum hi 2^32 + lo in units 2^(32 - sh) times its own (sh <= 32).
__device__ __forceinline__ uint64_t fx_scale(int64_t hi, int64_t lo, int sh) {
    const uint64_t h = sh >= 0 ? (uint64_t)hi << min(sh, 63) : (uint64_t)(hi >> min(-sh, 63));
    return h + (uint64_t)(lo >> min(32 - sh, 63));
}

constexpr float kRefPivot = 1e-5f;   // smaller pivots of P: the FP64 elimination decides
constexpr float kRefRate = 0.125f;   // slowest accepted reduction per refinement step
constexpr int kRefMaxSolves = 10;
// Exponents of the corrections' scales: every power of two that the kernel
// forms from one (2^(25 - e), 2^(e - 54), 2^(e0 - 60), 2^(el - 54), with
// el <= e0 + kRefLambda) is a normal float.  Smaller corrections take the
// lowest scale: they are below the unit of the sums anyway.
constexpr int kRefMinExp = -66, kRefMaxExp = 60, kRefLambda = 12;
static_assert(kRefMinExp - 60 >= -126 && 25 - kRefMinExp <= 127, "scales of the smallest corrections");
// Predicted error at which refinement stops, relative to max |w|: about a
// tenth of the FP64 elimination's median error (3e-15, 2e-14, 8e-14 at m = 2,
// 4, 6), and full accuracy near n = s, where the elimination is as accurate.
template <int M>
__device__ __forceinline__ float ref_done(int n, int s) {
    if (n < 2 * s) return 0x1p-53f;
    return M <= 2 ? 0x1p-51f : M <= 4 ? 0x1p-49f : 0x1p-47f;
}

// Matrix in place of its inverse by Gauss-Jordan with 2 x 2 pivots, no search
// (positive definite): row t of the q x q matrix A (row stride LQ) in thread
// t's registers, with a unit row and column added for odd q; 4 QC >= the even
// size + 2 columns.  The columns rotate by two per step; the pivot rows carry
// -1 one (two) columns past their end, which puts the multipliers into the
// columns that the rotation frees.  False where a pivot block is not positive
// definite.  (Single pivots: 14.6k cycles for q = 28, the barrier, the
// broadcast's latency and the reciprocal once per column.)
template <int NT, int TT, int QC>
__device__ __forceinline__ bool ref_invert(float* A, int q, int LQ, int t, float* prow, int PB) {
    const int qe = (q + 1) & ~1;
    float r[4 * QC];
#pragma unroll
    for (int j = 0; j < QC; ++j) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (4 * j < q && t < q) {
            v = reinterpret_cast<const float4*>(A + t * LQ)[j];
            if (4 * j + 1 >= q) v.y = 0.f;
            if (4 * j + 2 >= q) v.z = 0.f;
            if (4 * j + 3 >= q) v.w = 0.f;
        }
        if (t == q && q != qe) {
            if (4 * j == q) v.x = 1.f;
            if (4 * j + 1 == q) v.y = 1.f;
            if (4 * j + 2 == q) v.z = 1.f;
            if (4 * j + 3 == q) v.w = 1.f;
        }
        r[4 * j] = v.x;
        r[4 * j + 1] = v.y;
        r[4 * j + 2] = v.z;
        r[4 * j + 3] = v.w;
    }
    for (int k = 0; k < qe; k += 2) {
        // pivot rows k and k + 1; two pairs of buffers alternate
        float* p0 = prow + ((k >> 1) & 1) * 2 * PB;
        const float4* v0 = reinterpret_cast<const float4*>(p0);
        const float4* v1 = reinterpret_cast<const float4*>(p0 + PB);
        const bool piv = (t & ~1) == k;
        if (piv) {
            float* mine = p0 + (t & 1) * PB;
#pragma unroll
            for (int j = 0; j < QC; ++j)
                reinterpret_cast<float4*>(mine)[j] = make_float4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
            mine[qe + (t & 1)] = -1.f;
#pragma unroll
            for (int j = 2; j < 4 * QC; ++j) r[j] = 0.f;
            r[0] = (t & 1) ? 0.f : 1.f;
            r[1] = (t & 1) ? 1.f : 0.f;
        }
        ref_sync_part<NT, TT>();
        const float4 a = v0[0], b = v1[0];
        const float det = fmaf(a.x, b.y, -a.y * b.x), inv = rcpf(det);
        if (!(a.x > 0.f && det > 0.f && inv < INFINITY && det < INFINITY)) return false;
        // (f0, f1) = (r0, r1) B^-1; the pivot rows start from the unit rows
        const float f0 = fmaf(r[0], b.y, -r[1] * b.x) * inv;
        const float f1 = fmaf(r[1], a.x, -r[0] * a.y) * inv;
        r[0] = fmaf(-f1, b.z, fmaf(-f0, a.z, r[2]));
        r[1] = fmaf(-f1, b.w, fmaf(-f0, a.w, r[3]));
#pragma unroll
        for (int j = 1; j < QC; ++j) {
            const float4 x = v0[j], y = v1[j];
            r[4 * j - 2] = fmaf(-f1, y.x, fmaf(-f0, x.x, r[4 * j]));
            r[4 * j - 1] = fmaf(-f1, y.y, fmaf(-f0, x.y, r[4 * j + 1]));
            r[4 * j] = fmaf(-f1, y.z, fmaf(-f0, x.z, r[4 * j + 2]));
            r[4 * j + 1] = fmaf(-f1, y.w, fmaf(-f0, x.w, r[4 * j + 3]));
        }
        r[4 * QC - 2] = 0.f;
        r[4 * QC - 1] = 0.f;
    }
    if (t < q) {
#pragma unroll
        for (int j = 0; j < QC; ++j)
            if (4 * j < q) {
                float4 v = make_float4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
                if (4 * j + 1 >= q) v.y = 0.f;  // (the added column)
                if (4 * j + 2 >= q) v.z = 0.f;
                if (4 * j + 3 >= q) v.w = 0.f;
                reinterpret_cast<float4*>(A + t * LQ)[j] = v;
            }
    }
    return true;
}

// The instance of ref_invert with enough columns (QMAX: chunks a kernel can need).
template <int NT, int TT, int QMAX>
__device__ __forceinline__ bool ref_invert_any(float* A, int q, int LQ, int t, float* prow, int PB) {
    const int need = ((q + 1) / 2 * 2 + 2 + 3) / 4;
    if constexpr (QMAX > 2)
        if (need <= 2) return ref_invert<NT, TT, 2>(A, q, LQ, t, prow, PB);
    if constexpr (QMAX > 4)
        if (need <= 4) return ref_invert<NT, TT, 4>(A, q, LQ, t, prow, PB);
    if constexpr (QMAX > 6)
        if (need <= 6) return ref_invert<NT, TT, 6>(A, q, LQ, t, prow, PB);
    if constexpr (QMAX > 8)
        if (need <= 8) return ref_invert<NT, TT, 8>(A, q, LQ, t, prow, PB);
    if constexpr (QMAX > 12)
        if (need <= 12) return ref_invert<NT, TT, 12>(A, q, LQ, t, prow, PB);
    return ref_invert<NT, TT, QMAX>(A, q, LQ, t, prow, PB);
}

// Resident blocks that the registers must allow, by a sweep: two threads per
// node five (what shared memory allows at m = 6, n = 56); 64 threads six, eight
// for the wide reduced matrices of m <= 3; blocks of four warps four or six
// (ms per 1M stencils with 4 / 5 / 6 / 7: m = 4, n = 30 13.0 / 13.5 / 14.2 /
// 14.6; m = 2, n = 12 3.1 / 2.8 / 2.7 / 2.7).
template <int NT, int H, int M>
constexpr int ref_min_blocks() {
    return H == 2 ? (M >= 4 ? 5 : 4) : NT == 64 ? (M >= 4 ? 6 : 8) : NT == 32 ? 4 : 6;
}

template <int NT, int H, int M>
__global__ void __launch_bounds__(NT * H > 32 ? NT * H : 128, ref_min_blocks<NT, H, M>()) weights_refined_kernel(
    const double2* __restrict__ xy, const int* __restrict__ idx, int N, const RefGeom g, double* __restrict__ w,
    int* __restrict__ node_status) {
    constexpr int S = (M + 1) * (M + 2) / 2;
    constexpr int LS = odd4(S), S4 = up4(S) / 4, LP = S | 1;
    constexpr int TT = NT * H;              // threads of the stencil
    constexpr int QMAX = ((NT - S + 1) / 2 * 2 + 5) / 4;  // 16-byte chunks of a row of the reduced matrix + 2
    constexpr int RT = NT == 64 ? 4 : 2;    // register tiles of the float32 products
    constexpr int CT = 2;
    constexpr int KS = ref_ks(S), HS = TT / KS;  // shares of P^T d
    extern __shared__ __align__(16) unsigned char smem_ref[];
    const int t = threadIdx.x % TT;
    const int nd = t % NT, half = t / NT;  // node of the thread, its share of the node's work
    unsigned char* base = smem_ref + (size_t)(threadIdx.x / TT) * g.bytes;
    const int n = g.n, q = g.q, LQ = g.LQ, nh = n >> 1, q4 = (q + 3) >> 2;
    (void)RB_SH(base + g.bytes - 1);
    int2* phi = reinterpret_cast<int2*>(base + g.phi);
    int2* pd = reinterpret_cast<int2*>(base + g.pd);
    float* Wt = reinterpret_cast<float*>(base + g.pd);
    float* F1 = reinterpret_cast<float*>(base + g.F1);  // Phi11, then T^T
    float* Tt = F1 + S * LS;
    float* X = reinterpret_cast<float*>(base + g.X);
    float* C = reinterpret_cast<float*>(base + g.C);
    float* Sm = reinterpret_cast<float*>(base + g.Sm);
    longlong2* cxy = reinterpret_cast<longlong2*>(base + g.xy);
    float2* cxf = reinterpret_cast<float2*>(base + g.xyf);
    float* prow = reinterpret_cast<float*>(base + g.prow);
    float* vr1 = reinterpret_cast<float*>(base + g.vr1);
    float* vr2 = reinterpret_cast<float*>(base + g.vr2);
    float* vg = reinterpret_cast<float*>(base + g.vg);
    float* vd0 = reinterpret_cast<float*>(base + g.vd0);
    float* vt = reinterpret_cast<float*>(base + g.vt);
    float* vy = reinterpret_cast<float*>(base + g.vy);
    float* vdw = reinterpret_cast<float*>(base + g.vdw);
    int* dI = reinterpret_cast<int*>(base + g.dI);
    int* lI = reinterpret_cast<int*>(base + g.lI);
    int* posS = reinterpret_cast<int*>(base + g.pos);
    unsigned* red = reinterpret_cast<unsigned*>(base + g.red);
    longlong2* part = reinterpret_cast<longlong2*>(base + g.part);
    longlong2* part2 = reinterpret_cast<longlong2*>(base + g.part2);
    constexpr int PB = up4(NT) + 8;  // floats of one pivot-row buffer
    const bool mine = t < n;  // holds a node's row, residual and weight
    const int spb = blockDim.x / TT;

    // (unsigned: past 2^31 - 1 the index ends the loop instead of turning negative)
    for (unsigned node = blockIdx.x * spb + threadIdx.x / TT; node < (unsigned)N; node += gridDim.x * spb) {
        bool ok = true;  // uniform over the stencil's threads
        // ---- shift and scale (FP64) ------------------------------------------
        const double2 c = xy[node];
        double dx = 0.0, dy = 0.0;
        unsigned lost = 0;
        if (mine) {
            const int sj = idx[(int64_t)node * n + t];
            const bool in = (unsigned)sj < (unsigned)N;
            const double2 p = in ? xy[sj] : c;
            dx = __dadd_rn(p.x, -c.x);
            dy = __dadd_rn(p.y, -c.y);
            lost = in ? 0u : 1u;
        }
        // largest squared distance, as two 32-bit maxima of its bits
        const unsigned long long d2 =
            mine ? (unsigned long long)__double_as_longlong(fma(dx, dx, __dmul_rn(dy, dy))) & 0x7fffffffffffffffull : 0ull;
        const unsigned top = ref_max<TT>(lost ? 0xffffffffu : (unsigned)(d2 >> 32), red, 0);
        const unsigned low = ref_max<TT>((unsigned)(d2 >> 32) == top ? (unsigned)d2 : 0u, red, 1);
        const double dmax = __hiloint2double((int)top, (int)low);
        ok = top < 0x7ff00000u && seed_range(dmax);
        double inv_delta2 = 0.0;
        if (ok) {
            const double id = rsqrt64(dmax);
            inv_delta2 = __dmul_rn(id, id);
            float xf = 0.f, yf = 0.f;
            longlong2 me = make_longlong2(0, 0);
            int64_t sown = 0;  // |xh| 2^60
            if (mine) {
                const double xh = __dmul_rn(dx, id), yh = __dmul_rn(dy, id);
                me.x = fx_coord((uint64_t)__double_as_longlong(xh));
                me.y = fx_coord((uint64_t)__double_as_longlong(yh));
                cxy[t] = me;
                xf = (float)me.x * 0x1p-61f;
                yf = (float)me.y * 0x1p-61f;
                cxf[t] = make_float2(xf, yf);
                const int64_t qi = fx_r2(me.x, me.y);
                float qf = fmaf(xf, xf, yf * yf);
                if (qf < 0x1p-14f) qf = (float)qi * 0x1p-58f;
                if (qi > 0) sown = fx_sqrt(qi, qf, rsqf(qf));
            }
            ref_sync<TT>();

            // ---- P1^-1, X = P2 P1^-1 (Gauss-Jordan, row pivoting) and the kernel
            // values in fixed point: by the two halves of the threads, or (H = 1)
            // one pivot step and one pair per turn, so that the pair's arithmetic
            // fills the step's barriers and chain
            const bool elim = half == 0, pairs = H == 1 || half == 1;
            const longlong2 at = nd < n ? cxy[nd] : make_longlong2(0, 0);
            const float2 atf = nd < n ? cxf[nd] : make_float2(0.f, 0.f);
            float row[S];
            int pos = -1;
            row[0] = mine ? 1.f : 0.f;
            row[1] = atf.x;
            row[2] = atf.y;
#pragma unroll
            for (int d = 2; d <= M; ++d) {
                const int cur = d * (d + 1) / 2, prev = (d - 1) * d / 2;
#pragma unroll
                for (int i = 0; i < d; ++i) row[cur + i] = atf.x * row[prev + i];
                row[cur + d] = atf.y * row[prev + d - 1];
            }
            float qmin = 4.f;            // smallest r^2 seen
            int other = nd < n ? nd : 0; // pair u: nodes nd and nd + u + 1 (cyclic)
            const int steps = !elim ? nh : (H == 1 ? max(S, nh) : S);
            for (int k = 0; k < steps; ++k) {
                const bool step = elim && k < S, pair = pairs && k < nh && nd < n;
                unsigned best = 0;
                float* pr = prow + (k & 1) * PB;
                // largest |entry| of the column (ties and the last six bits: lower thread)
                if (step) {
                    const unsigned key =
                        mine && pos < 0 ? ((__float_as_uint(row[0]) & 0x7fffffc0u) | (unsigned)(63 - t)) : 0u;
                    best = __reduce_max_sync(ref_mask<NT>(), key);
                    if constexpr (NT > 32)
                        if ((t & 31) == 0) red[16 + (k & 1) * 2 + (t >> 5)] = best;
                }
                int64_t qi = 0;
                float qf = 1.f, ry = 1.f;
                if (pair) {
                    other = other + 1 < n ? other + 1 : 0;
                    const longlong2 o = RB_AT(cxy, other, n);
                    const float2 of = RB_AT(cxf, other, n);
                    qi = fx_r2(at.x - o.x, at.y - o.y);
                    const float fx = atf.x - of.x, fy = atf.y - of.y;
                    qf = fmaf(fx, fx, fy * fy);
                    qmin = fminf(qmin, qf);
                    ry = rsqf(qf);
                }
                bool piv = false;
                if (step) {
                    if constexpr (NT > 32) {
                        ref_sync_part<NT, TT>();
                        best = max(red[16 + (k & 1) * 2], red[17 + (k & 1) * 2]);
                    }
                    ok = best >= __float_as_uint(kRefPivot) && best < 0x7f800000u;
                    if (!ok) break;
                    piv = t == 63 - (int)(best & 63u);
                    if (piv) {
                        pos = k;
                        row[0] = rcpf(row[0]);
#pragma unroll
                        for (int j = 0; j < S4; ++j) {
                            float4 v;
                            v.x = row[4 * j];
                            v.y = 4 * j + 1 < S ? row[4 * j + 1 < S ? 4 * j + 1 : 0] : 0.f;
                            v.z = 4 * j + 2 < S ? row[4 * j + 2 < S ? 4 * j + 2 : 0] : 0.f;
                            v.w = 4 * j + 3 < S ? row[4 * j + 3 < S ? 4 * j + 3 : 0] : 0.f;
                            reinterpret_cast<float4*>(pr)[j] = v;
                        }
#pragma unroll
                        for (int j = 1; j < S; ++j) row[j] = 0.f;
                    }
                }
                if (pair) {
                    const Digits v = fx_digits(fx_cube(qi, fx_sqrt(qi, qf, ry)));
                    RB_AT(phi, k * n + nd, nh * n) = make_int2(v.hi, v.lo);
                }
                if (step) {
                    ref_sync_part<NT, TT>();
                    const float4 v0 = reinterpret_cast<const float4*>(pr)[0];
                    const float f = piv ? v0.x : row[0] * v0.x;
#pragma unroll
                    for (int j = 0; j < S4; ++j) {
                        const float4 v = j ? reinterpret_cast<const float4*>(pr)[j] : v0;
                        if (j > 0) row[4 * j - 1] = fmaf(-f, v.x, row[4 * j]);
                        if (4 * j + 1 < S) row[4 * j] = fmaf(-f, v.y, row[4 * j + 1 < S ? 4 * j + 1 : 0]);
                        if (4 * j + 2 < S) row[4 * j + 1 < S ? 4 * j + 1 : 0] = fmaf(-f, v.z, row[4 * j + 2 < S ? 4 * j + 2 : 0]);
                        if (4 * j + 3 < S) row[4 * j + 2 < S ? 4 * j + 2 : 0] = fmaf(-f, v.w, row[4 * j + 3 < S ? 4 * j + 3 : 0]);
                    }
                    row[S - 1] = f;
                }
            }
            // pairs closer than 2^-7 of the radius: again, from an exact r^2
            bool close = false;
            if (pairs && nd < n && qmin < 0x1p-14f) {
                for (int u = 0; u < nh; ++u) {
                    const int k = nd + u + 1 < n ? nd + u + 1 : nd + u + 1 - n;
                    const longlong2 o = RB_AT(cxy, k, n);
                    const int64_t qi = fx_r2(at.x - o.x, at.y - o.y);
                    close |= qi < 16;
                    const float qf = fmaxf((float)qi * 0x1p-58f, 0x1p-58f);
                    const Digits v = fx_digits(fx_cube(qi, fx_sqrt(qi, qf, rsqf(qf))));
                    phi[u * n + nd] = make_int2(v.hi, v.lo);
                }
            }
            if (elim && ok) {
                // permuted position: pivots in pivot order, then the others in node order
                const unsigned bal = __ballot_sync(ref_mask<NT>(), mine && pos < 0) & ref_mask<NT>();
                int rank = __popc(bal & ((1u << (threadIdx.x & 31)) - 1u));
                if constexpr (NT > 32) {
                    if (t == 0) red[20] = __popc(bal);
                    ref_sync_part<NT, TT>();
                    if (t >= 32) rank += (int)red[20];
                }
                if (mine) {
                    if (pos < 0) pos = S + rank;
                    posS[t] = pos;
                    float* dst = pos < S ? &RB_AT(C, pos * LS, S * LS) : &RB_AT(X, (pos - S) * LS, q * LS);
#pragma unroll
                    for (int j = 0; j < S4; ++j) {
                        float4 v;
                        v.x = row[4 * j];
                        v.y = 4 * j + 1 < S ? row[4 * j + 1 < S ? 4 * j + 1 : 0] : 0.f;
                        v.z = 4 * j + 2 < S ? row[4 * j + 2 < S ? 4 * j + 2 : 0] : 0.f;
                        v.w = 4 * j + 3 < S ? row[4 * j + 3 < S ? 4 * j + 3 : 0] : 0.f;
                        reinterpret_cast<float4*>(dst)[j] = v;
                    }
                    // zero diagonal and padding of this row's blocks
                    if (pos < S) F1[pos * LS + pos] = 0.f;
                    else Sm[(pos - S) * LQ + pos - S] = 0.f;
                    for (int j = S; j < 4 * S4; ++j) {
                        F1[pos * LS + j] = 0.f;
                        if (pos >= S) Wt[(pos - S) * LS + j] = 0.f;
                    }
                }
            }
            ok = ref_max<TT>(close || !ok ? 1u : 0u, red, 0) == 0u;
            if constexpr (TT <= 32) ref_sync<TT>();

            // ---- the float32 blocks of Phi from the leading digits ------------------
            if (ok && nd < n) {
                const int smo = (int)(Sm - F1), own = posS[nd];
                const int u1 = half + 1 < H ? nh / 2 : nh;
#pragma unroll 4
                for (int u = half ? nh / 2 : 0; u < u1; ++u) {
                    const int k = nd + u + 1 < n ? nd + u + 1 : nd + u + 1 - n;
                    const float pf = (float)phi[u * n + nd].x * 0x1p-24f;
                    const int b = RB_AT(posS, k, n);
                    const int lo = min(own, b), hi = max(own, b);
                    // (hi, lo), and its mirror in Phi11 and Phi22
                    const int o1 = lo < S ? hi * LS + lo : smo + (hi - S) * LQ + lo - S;
                    const int o2 = hi < S ? lo * LS + hi : (lo < S ? o1 : smo + (lo - S) * LQ + hi - S);
                    RB_AT(F1, o1, smo + q * LQ) = pf;
                    RB_AT(F1, o2, smo + q * LQ) = pf;
                }
            }
            ref_sync<TT>();

            if (ok && q > 0) {
                // ---- U^T = X Phi11; T^T = Phi21 - U^T, W^T = Phi21 - U^T / 2 ------
                constexpr int TA = (S + CT - 1) / CT;
                const int tj = (q + RT - 1) / RT;
                for (int tile = t; tile < tj * TA; tile += TT) {
                    const int j0 = tile / TA * RT, a0 = (tile - tile / TA * TA) * CT;
                    float acc[RT][CT];
#pragma unroll
                    for (int i = 0; i < RT; ++i)
#pragma unroll
                        for (int a = 0; a < CT; ++a) acc[i][a] = 0.f;
#pragma unroll
                    for (int k = 0; k < S4; ++k) {
                        float4 xr[RT], ar[CT];
#pragma unroll
                        for (int i = 0; i < RT; ++i)
                            xr[i] = reinterpret_cast<const float4*>(X + min(j0 + i, q - 1) * LS)[k];
#pragma unroll
                        for (int a = 0; a < CT; ++a)
                            ar[a] = reinterpret_cast<const float4*>(F1 + min(a0 + a, S - 1) * LS)[k];
#pragma unroll
                        for (int i = 0; i < RT; ++i)
#pragma unroll
                            for (int a = 0; a < CT; ++a) acc[i][a] = dot4(xr[i], ar[a], acc[i][a]);
                    }
#pragma unroll
                    for (int i = 0; i < RT; ++i)
#pragma unroll
                        for (int a = 0; a < CT; ++a)
                            if (j0 + i < q && a0 + a < S) {
                                const int e = (j0 + i) * LS + a0 + a;
                                const float v = Tt[e];
                                Tt[e] = v - acc[i][a];
                                Wt[e] = fmaf(-0.5f, acc[i][a], v);
                            }
                }
                ref_sync<TT>();
                // ---- S = Phi22 - X W - (X W)^T, lower tiles and their mirror -------
                constexpr int RC = RT / CT;  // column tiles per row tile
                const int nt = (q + RT - 1) / RT;
                for (int tile = t; tile < RC * nt * (nt + 1) / 2; tile += TT) {
                    int ti = (int)((sqrtf(8.0f / RC * tile + 1.0f) - 1.0f) * 0.5f);
                    while (RC * ti * (ti + 1) / 2 > tile) --ti;
                    while (RC * (ti + 1) * (ti + 2) / 2 <= tile) ++ti;
                    const int i0 = ti * RT, j0 = (tile - RC * ti * (ti + 1) / 2) * CT;
                    float acc[RT][CT];
#pragma unroll
                    for (int i = 0; i < RT; ++i)
#pragma unroll
                        for (int j = 0; j < CT; ++j) acc[i][j] = 0.f;
#pragma unroll 1
                    for (int h = 0; h < 2; ++h) {  // X_i . W_j, then W_i . X_j
                        const float* pa = h ? Wt : X;
                        const float* pb = h ? X : Wt;
#pragma unroll
                        for (int k = 0; k < S4; ++k) {
                            float4 xr[RT], wr[CT];
#pragma unroll
                            for (int i = 0; i < RT; ++i)
                                xr[i] = reinterpret_cast<const float4*>(pa + min(i0 + i, q - 1) * LS)[k];
#pragma unroll
                            for (int j = 0; j < CT; ++j)
                                wr[j] = reinterpret_cast<const float4*>(pb + min(j0 + j, q - 1) * LS)[k];
#pragma unroll
                            for (int i = 0; i < RT; ++i)
#pragma unroll
                                for (int j = 0; j < CT; ++j) acc[i][j] = dot4(xr[i], wr[j], acc[i][j]);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < RT; ++i)
#pragma unroll
                        for (int j = 0; j < CT; ++j)
                            if (i0 + i < q && i0 + i >= j0 + j) {
                                const float v = Sm[(i0 + i) * LQ + j0 + j] - acc[i][j];
                                Sm[(i0 + i) * LQ + j0 + j] = v;
                                Sm[(j0 + j) * LQ + i0 + i] = v;
                            }
                }
                ref_sync<TT>();
                // ---- S^-1, by one warp where its rows fit one ------------------------
                if constexpr (TT > 32) {
                    bool pos_def = true;
                    if (q >= 32) {
                        if (elim) pos_def = ref_invert_any<NT, TT, QMAX>(Sm, q, LQ, t, prow, PB);
                    } else if (t < 32) {
                        pos_def = ref_invert_any<32, TT, (QMAX < 9 ? QMAX : 9)>(Sm, q, LQ, t, prow, PB);
                    }
                    if (t == 0) red[21] = pos_def ? 1u : 0u;
                } else {
                    ok = ref_invert_any<NT, TT, QMAX>(Sm, q, LQ, t, prow, PB);
                }
            } else if (TT > 32 && t == 0) {
                red[21] = 1u;
            }

            // ---- monomials in fixed point (Phi11 and W^T are no longer needed) ---
            if (ok && pairs && nd < n) {
                const Digits xd = fx_digits(at.x), yd = fx_digits(at.y);
                int2* pr = pd + nd * LP;
                Digits up[M + 1];  // the previous degree's digits
                up[0].hi = 1 << 29;
                up[0].lo = 0;
                pr[0] = make_int2(up[0].hi, up[0].lo);
                int cur = 1;
#pragma unroll
                for (int d = 1; d <= M; ++d) {
                    up[d] = fx_digits(fx_mono(yd, up[d - 1]));
#pragma unroll
                    for (int i = 0; i < d; ++i) up[i] = fx_digits(fx_mono(xd, up[i]));
#pragma unroll
                    for (int i = 0; i <= d; ++i) pr[cur + i] = make_int2(up[i].hi, up[i].lo);
                    cur += d + 1;
                }
            }

            // ---- solve and refine ------------------------------------------------
            const float grhs = (M >= 2 && (t == 3 || t == 5)) ? 2.0f : 0.0f;
            float rf = 9.0f * ((float)sown * 0x1p-60f);  // current residual, float32
            float rg = grhs;
            int64_t ri = 0, rgi = 0;                     // and in units of 2^(e0 - 60)
            int64_t wi = 0;                              // weight in units of 2^(e0 - 62)
            int e0 = 0;
            float mprev = 0.f, mw0 = 0.f;
            bool bad = false;
            if (t < 4 * S4) {
                vr1[t] = 0.f;
                vg[t] = 0.f;
                vd0[t] = 0.f;
            }
            if (t < 4 * q4) vr2[t] = vt[t] = 0.f;
            ref_sync<TT>();
            if constexpr (TT > 32) ok = ok && red[21] != 0u;
            for (int it = 0; ok; ++it) {
                // float32 correction d of the residual (rf, rg)
                if (mine) {
                    if (pos < S) RB_AT(vr1, pos, S) = rf;
                    else RB_AT(vr2, pos - S, q) = rf;
                }
                if (t < S) vg[t] = rg;
                ref_sync<TT>();
                const int i2 = TT - 1 - t;  // row of X, T^T and S^-1 (other threads than t < S where there are)
                float a1 = 0.f, d0 = 0.f;
                if (i2 < q) a1 = vr2[i2] - dotv(X + i2 * LS, vr1, S4);
                if (t < S) {
                    float s0 = 0.f, s1 = 0.f;
#pragma unroll
                    for (int k = 0; k + 1 < S; k += 2) {
                        s0 = fmaf(C[k * LS + t], vg[k], s0);
                        s1 = fmaf(C[(k + 1) * LS + t], vg[k + 1], s1);
                    }
                    if (S & 1) s0 = fmaf(C[(S - 1) * LS + t], vg[S - 1], s0);
                    d0 = s0 + s1;
                    vd0[t] = d0;
                }
                ref_sync<TT>();
                if (i2 < q) vt[i2] = a1 - dotv(Tt + i2 * LS, vd0, S4);
                ref_sync<TT>();
                if (i2 < q) {
                    const float y = dotv(Sm + i2 * LQ, vt, q4);
                    vy[i2] = y;
                    vdw[S + i2] = y;
                }
                ref_sync<TT>();
                if (t < S) {
                    float s0 = 0.f, s1 = 0.f;
                    int j = 0;
#pragma unroll 4
                    for (; j + 1 < q; j += 2) {
                        s0 = fmaf(X[j * LS + t], vy[j], s0);
                        s1 = fmaf(X[(j + 1) * LS + t], vy[j + 1], s1);
                    }
                    if (j < q) s0 = fmaf(X[j * LS + t], vy[j], s0);
                    vdw[t] = d0 - (s0 + s1);
                }
                ref_sync<TT>();
                const float dj = mine ? RB_AT(vdw, pos, n) : 0.f;

                // size of the correction, its rate of decrease
                const unsigned um = ref_max<TT>(bad ? 0x7f800000u : __float_as_uint(fabsf(dj)), red, it & 1);
                if (um == 0u && it > 0) break;  // the residual is zero
                const float m = __uint_as_float(um);
                const int em = (int)(um >> 23) - 126, e = max(em, kRefMinExp);  // 2^e > m
                // not finite, a failed check, or out of scale
                if (um >= 0x7f800000u || e > kRefMaxExp || (it == 0 && em < kRefMinExp)) {
                    ok = false;
                    break;
                }
                if (it == 0) {
                    e0 = e;
                    mw0 = m;
                }
                const bool slow = it > 0 && !(m < kRefRate * mprev);
                const bool done = it > 0 && m * (m / mprev) <= ref_done<M>(n, S) * mw0;
                if ((slow && !done) || (!done && it + 1 >= kRefMaxSolves)) {
                    ok = false;
                    break;
                }
                mprev = m;
                // the correction in units of 2^(e - 25); the sum takes the same integers
                const int di = fx_round(dj * fx_pow2f(25 - e));
                const int sh = 37 - (e0 - e);
                wi += sh >= 0 ? (int64_t)((uint64_t)(int64_t)di << (sh & 63)) : ((int64_t)di >> min(-sh, 31));
                if (done) break;
                if (mine) {
                    dI[t] = di;
                    dI[t + n] = di;
                }
                ref_sync<TT>();

                // residual: r -= Phi d, rg -= P^T d, exact sums of the digits'
                // products, of unit 2^(e - 49) (H) and 2^(e - 81) (L).  The 64-bit
                // wrap of r is harmless while the true residual is below 2^(e0 + 2)
                // (the monomials' digits have units 2^-5 of the kernel values')
                const float hs = fx_pow2f(e - 49), gs = fx_pow2f(e - 54);
                float check = rf;
                int64_t HH = 0, LL = 0;
                if (nd < n) {
                    // the half's share of the pairs; both nodes of each
                    const int full = (n & 1) ? nh : nh - 1;
                    const int ua = half ? full / 2 : 0, ub = half + 1 < H ? full / 2 : full;
                    const int2* pa = phi + nd + ua * n;            // pair (nd, nd + u + 1)
                    const int2* pb = phi + nd - 1 + ua * (n - 1);  // pair (nd - u - 1, nd)
                    const int* da = dI + nd + 1 + ua;
                    const int* db = dI + nd + n - 1 - ua;
#pragma unroll 4
                    for (int u = ua; u < ub; ++u) {
                        const int2 a = *pa, b = RB_PT(pb + (nd <= u ? n : 0), phi, nh * n);
                        const int va = RB_PT(da, dI, 2 * n), vb = RB_PT(db, dI, 2 * n);
                        HH += fx_mul32(a.x, va) + fx_mul32(b.x, vb);
                        LL += fx_mul32(a.y, va) + fx_mul32(b.y, vb);
                        pa += n;
                        pb += n - 1;
                        ++da;
                        --db;
                    }
                    if (half == 0 && full < nh) {  // n even: the opposite node, once
                        const int2 a = phi[full * n + nd];
                        const int va = dI[nd + nh];
                        HH += fx_mul32(a.x, va);
                        LL += fx_mul32(a.y, va);
                    }
                    if (H > 1 && half) part2[nd] = make_longlong2(HH, LL);
                }
                // rg: HS threads per monomial
                int64_t GH = 0, GL = 0;
                const int kc = t % KS, kg = t / KS;
                if (kc < S) {
#pragma unroll 4
                    for (int j = kg; j < n; j += HS) {
                        const int2 a = pd[j * LP + kc];
                        const int d = dI[j];
                        GH += fx_mul32(a.x, d);
                        GL += fx_mul32(a.y, d);
                    }
                    if (HS > 1 && kg) RB_AT(part, (kg - 1) * S + kc, (HS - 1) * S) = make_longlong2(GH, GL);
                }
                if constexpr (H > 1) ref_sync<TT>();
                if (mine) {
                    if constexpr (H > 1) {
                        HH += part2[t].x;
                        LL += part2[t].y;
                    }
                    if (it == 0)  // 9 |xh|: 2^-60 to 2^(e0 - 60)
                        ri = (int64_t)(e0 >= 0 ? 9ull * (uint64_t)sown >> min(e0, 63) : 9ull * (uint64_t)sown << min(-e0, 63));
                    ri = (int64_t)((uint64_t)ri - fx_scale(HH, LL, 11 - (e0 - e)));
                    check -= (float)HH * hs;
                    // (rounded through the check's magnitude until P l is subtracted)
                    if (pos < S) RB_AT(vr1, pos, S) = it == 0 ? check : (float)ri * fx_pow2f(e0 - 60);
                }
                ref_sync<TT>();
                // correction of l from the residual of the pivot rows, and its scale
                float dl = 0.f;
                if (t < S) {
                    dl = dotv(C + t * LS, vr1, S4);
#pragma unroll
                    for (int k = 0; k + 1 < HS; ++k) {
                        GH += part[k * S + t].x;
                        GL += part[k * S + t].y;
                    }
                    if (it == 0) rgi = grhs != 0.f && 61 - e0 < 64 ? (int64_t)(1ull << (61 - e0)) : 0;
                    rgi = (int64_t)((uint64_t)rgi - fx_scale(GH, GL, 6 - (e0 - e)));
                    bad |= !(fabsf(rg - (float)GH * gs) < fx_pow2f(e0));
                    rg = (float)rgi * fx_pow2f(e0 - 60);
                }
                const unsigned ul = ref_max<TT>(__float_as_uint(fabsf(dl)), red, 2 + (it & 1));
                const int el = max((int)(ul >> 23) - 126, kRefMinExp);
                if (ul >= 0x7f800000u || el > e0 + kRefLambda) {  // (l in the range of the sums)
                    ok = false;
                    break;
                }
                if (t < S) lI[t] = fx_round(dl * fx_pow2f(25 - el));
                ref_sync<TT>();
                if (mine) {
                    int64_t PH = 0, PL = 0;
                    const int2* pr = pd + t * LP;
#pragma unroll
                    for (int kk = 0; kk < S; ++kk) {
                        const int2 a = pr[kk];
                        const int d = lI[kk];
                        PH += fx_mul32(a.x, d);
                        PL += fx_mul32(a.y, d);
                    }
                    ri = (int64_t)((uint64_t)ri - fx_scale(PH, PL, 6 - (e0 - el)));
                    check -= (float)PH * fx_pow2f(el - 54);
                    bad |= !(fabsf(check) < fx_pow2f(e0));
                    rf = (float)ri * fx_pow2f(e0 - 60);
                }
            }

            // ---- scale back (FP64) and store --------------------------------------
            if (ok) {
                const double v = __dmul_rn((double)wi, __dmul_rn(inv_delta2, __hiloint2double((e0 - 62 + 1023) << 20, 0)));
                ok = ref_max<TT>(mine && !finite64(v) ? 1u : 0u, red, 4) == 0u;
                if (ok && mine) w[(int64_t)node * n + t] = v;
                if (ok && node_status && t == 0) node_status[node] = 0;
            }
        }
        if (!ok && t == 0) w[(int64_t)node * n] = __longlong_as_double((long long)kWeightsMark);
        ref_sync<TT>();
    }
}

template <int NT, int H, int M>
int launch(const double2* xy, const int32_t* idx, int64_t N, int n, double* w, int32_t* node_status,
           cudaStream_t st) {
    const RefGeom g = ref_geom(NT, H, n, (M + 1) * (M + 2) / 2);
    auto kern = weights_refined_kernel<NT, H, M>;
    // stencils per block: one where a stencil spans several warps, else enough
    // warps (at most four) for the most resident stencils per SM
    int spb = 1;
    constexpr int TT = NT * H;
    if (TT <= 32) {
        int best = 0;
        for (int s = 32 / TT; s <= 128 / TT; s += 32 / TT) {
            const int blocks = std::min(32, (int)(233472 / (s * g.bytes + 1024)));
            if (s * g.bytes <= 227 * 1024 && blocks * s >= best) {
                best = blocks * s;
                spb = s;
            }
        }
    }
    const size_t smem = (size_t)spb * g.bytes;
    RBFFD_CUDA_TRY(allow_dynamic_smem(kern));
    RBFFD_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
    int per_sm = 0;
    RBFFD_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TT * spb, smem));
    if (per_sm < 1) return RBFFD_ERR_INVALID_ARG;
    const int64_t need = (N + spb - 1) / spb;
    const int blocks = (int)std::min<int64_t>(need, (int64_t)per_sm * sm_count());
    kern<<<blocks, TT * spb, smem, st>>>(xy, idx, (int)N, g, w, node_status);
    return RBFFD_OK;
}

template <int M>
int launch_m(const double2* xy, const int32_t* idx, int64_t N, int n, double* w, int32_t* node_status,
             cudaStream_t st) {
    constexpr int S = (M + 1) * (M + 2) / 2;
    if constexpr (S <= 16)
        if (n <= 16) return launch<16, 1, M>(xy, idx, N, n, w, node_status, st);
    if (n <= 32) return launch<32, 1, M>(xy, idx, N, n, w, node_status, st);
    // two threads per node where shared memory holds fewer than six stencils
    // (twelve warps) per SM: 1M nodes, m = 6, n = 56 63.5 -> 53.3 ms with
    // them, m = 4, n = 45 (27 KB) 35.7 -> 42.9
    if (ref_geom(64, 1, n, S).bytes > 37 * 1024) return launch<64, 2, M>(xy, idx, N, n, w, node_status, st);
    return launch<64, 1, M>(xy, idx, N, n, w, node_status, st);
}

}  // namespace

// (n <= 6, m <= 2: the elimination is as short as the second launch.  100k even
// nodes, elimination / refined solve: m = 1, n = 6 0.233 / 0.233 ms, m = 2,
// n = 6 0.239 / 0.263, m = 2, n = 7 0.33 / 0.28.)
bool refined_applies(int n, int m) {
    return m >= 1 && m <= 6 && n <= 64 && n >= (m + 1) * (m + 2) / 2 && n > 6;
}

int refined_weights(const double* xy, const int32_t* idx, int64_t N, int32_t n, int32_t m, double* w,
                    int32_t* node_status, cudaStream_t st) {
    const double2* p = reinterpret_cast<const double2*>(xy);
    switch (m) {
        case 1: return launch_m<1>(p, idx, N, n, w, node_status, st);
        case 2: return launch_m<2>(p, idx, N, n, w, node_status, st);
        case 3: return launch_m<3>(p, idx, N, n, w, node_status, st);
        case 4: return launch_m<4>(p, idx, N, n, w, node_status, st);
        case 5: return launch_m<5>(p, idx, N, n, w, node_status, st);
        case 6: return launch_m<6>(p, idx, N, n, w, node_status, st);
        default: return RBFFD_ERR_INVALID_ARG;
    }
}

}  // namespace rbffd
