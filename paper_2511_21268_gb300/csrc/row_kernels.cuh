// Matrix-pass building blocks and the row-group kernels of the solve
// phase (included by solve_kernels.cu): matrix views (plain CSR, and CSR
// values with run-encoded columns), the warp row-group reduction and the
// kernels that make one pass over a level matrix with their fused
// epilogues -- q = K p with p.q, residuals, smoothing sweeps, the up sweep
// with prolongation, the level-0 up sweep with r.z -- and the FP64
// residual.  Arithmetic of arXiv 2511.21268, Sec. 3 (two-level correction
// steps applied recursively) and Sec. 3.2 (l1-Jacobi).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "amg_internal.cuh"

namespace amg {
namespace {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ double ldv(const double* v, int64_t k) { return __ldg(v + k); }
__device__ __forceinline__ float ldv(const float* v, int64_t k) { return __ldg(v + k); }
__device__ __forceinline__ float ldv(const __nv_bfloat16* v, int64_t k) { return __bfloat162float(v[k]); }

// Lane partial of row i: sum over k = b + lane + S t of v_k x_{c_k}, in A (S
// lanes per row).  The rows this runs on (levels with few rows, short rows)
// are latency-bound: each chunk of U entries per lane loads all its values
// and columns, then all its x entries, then runs the FMA chain in entry
// order, and the last partial chunk does the same with predicated loads, so a
// row of up to S U entries costs two dependent round trips.
template <int S, typename A, typename V, typename X>
__device__ __forceinline__ A lane_partial(const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                          const V* __restrict__ v, const X* __restrict__ x, int i, int lane) {
    constexpr int U = sizeof(A) == 4 ? 16 : 8;
    const int64_t b = rp[i], e = rp[i + 1];
    A acc = A(0);
    int64_t k = b + lane;
    for (; k + S * (U - 1) < e; k += S * U) {
        A vv[U], xx[U];
        int cc[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            vv[u] = (A)ldv(v, k + S * u);
            cc[u] = __ldg(ci + k + S * u);
        }
#pragma unroll
        for (int u = 0; u < U; u++) xx[u] = (A)x[cc[u]];
#pragma unroll
        for (int u = 0; u < U; u++) acc = fma(vv[u], xx[u], acc);
    }
    if (k < e) {  // fewer than U entries left on this lane
        A vv[U - 1], xx[U - 1];
        int cc[U - 1];
#pragma unroll
        for (int u = 0; u < U - 1; u++) {
            const bool in = k + S * u < e;
            vv[u] = in ? (A)ldv(v, k + S * u) : A(0);
            cc[u] = in ? __ldg(ci + k + S * u) : -1;
        }
#pragma unroll
        for (int u = 0; u < U - 1; u++) xx[u] = cc[u] >= 0 ? (A)x[cc[u]] : A(0);
#pragma unroll
        for (int u = 0; u < U - 1; u++)
            if (cc[u] >= 0) acc = fma(vv[u], xx[u], acc);
    }
    return acc;
}

// A warp's scratch in the row-group kernels with RPW rows per warp.
template <typename A, int RPW>
struct RowTile {};
template <typename A>
struct RowTile<A, 8> {
    A t[8][33];  // lane partials of each row
};
constexpr int kFoldBytes = 64;  // of one row's values per staged chunk
template <typename A>
struct RowTile<A, 32> {
    static constexpr int kC = kFoldBytes / sizeof(A);  // entries of each row per chunk
    A v[32][kC + 1];
    int c[32][kC + 1];
};

// Matrix views of the row-group kernels.  CsrM: plain CSR.  RunM: CSR
// values with run-encoded columns (every row a sequence of equal runs of L
// consecutive columns): one 4-byte start column per run replaces the run's
// column indices, so a pass reads s_v + 4/L bytes per entry from HBM
// instead of s_v + 4.  The lanes keep the CSR order (lane t reads entries
// b + t + 32 j, coalesced); entry b + u lies in run u / L at offset u % L,
// the quotient taken as __umulhi(u, ceil(2^32 / L)) (exact for u < 2^16),
// and the run's start column is an L1-resident load shared by the L lanes
// of the run.
__constant__ uint32_t kRunMagic[kMaxRunLen + 1] = {0u,          0u,          2147483648u, 1431655766u, 1073741824u,
                                                   858993460u,  715827883u,  613566757u,  536870912u,  477218589u};

template <typename V>
struct CsrM {
    static constexpr bool kFlat = true;
    const int64_t* __restrict__ rp;
    const int32_t* __restrict__ ci;
    const V* __restrict__ v;
    template <typename A, typename X>
    __device__ __forceinline__ A partial(const X* __restrict__ x, int i, int lane) const {
        return lane_partial<32, A>(rp, ci, v, x, i, lane);
    }
    // one of 8 lanes of row i
    template <typename A, typename X>
    __device__ __forceinline__ A sub(const X* __restrict__ x, int i, int q) const {
        return lane_partial<8, A>(rp, ci, v, x, i, q);
    }
    // Row row0 + lane as one chain of products in entry order, a lane per row
    // (0 past the last row).  The warp stages kC entries of each of its 32 rows
    // at a time in shared memory, 32 / kC rows per load instruction, with the
    // next chunk's entries in registers meanwhile; neighbouring rows of a
    // tensor-product matrix read neighbouring vector entries, so the gathers
    // of the 32 lanes coalesce.
    template <typename A, typename X>
    __device__ __forceinline__ A ordered(const X* __restrict__ x, int row0, int n, int lane,
                                         RowTile<A, 32>& T) const {
        constexpr int C = RowTile<A, 32>::kC, RI = 32 / C, NI = 32 / RI;  // rows per instruction, instructions
        const int64_t b = row0 + lane < n ? rp[row0 + lane] : 0;
        const int len = row0 + lane < n ? (int)(rp[row0 + lane + 1] - b) : 0;
        const int longest = __reduce_max_sync(FULL, len);
        const int sub = lane / C, o = lane % C;  // this lane loads entry o of rows sub, sub + RI, ...
        A nv[NI];
        int nc[NI];
        auto load = [&](int k0) {
#pragma unroll
            for (int j = 0; j < NI; j++) {
                const int r = j * RI + sub;
                const int64_t rb = __shfl_sync(FULL, b, r);
                const bool in = k0 + o < __shfl_sync(FULL, len, r);
                nv[j] = in ? (A)ldv(v, rb + k0 + o) : A(0);
                nc[j] = in ? __ldg(ci + rb + k0 + o) : 0;
            }
        };
        A acc = A(0);
        load(0);
        for (int k0 = 0; k0 < longest; k0 += C) {
            __syncwarp();
#pragma unroll
            for (int j = 0; j < NI; j++) {
                T.v[j * RI + sub][o] = nv[j];
                T.c[j * RI + sub][o] = nc[j];
            }
            __syncwarp();
            if (k0 + C < longest) load(k0 + C);
            const int cnt = min(C, len - k0);
            A xx[C];
#pragma unroll
            for (int u = 0; u < C; u++)
                if (u < cnt) xx[u] = (A)x[T.c[lane][u]];
#pragma unroll
            for (int u = 0; u < C; u++)
                if (u < cnt) acc = fma(T.v[lane][u], xx[u], acc);
        }
        return acc;
    }
    // Lane partials of the RPW rows row0 .. row0+RPW-1 into tile[r][lane]:
    // the warp streams the rows' contiguous entries, lane t taking entries
    // e0 + t + 32 j in order with four loads in flight, so no row waits for
    // the previous one.  A lane keeps one running sum and stores it to
    // tile[r][t] when its next entry lies past row r (rows it never
    // touches keep 0).
    template <int RPW, typename A, typename X>
    __device__ __forceinline__ void flat(const X* __restrict__ x, int row0, int n, int lane, A (*tile)[33]) const {
        const int64_t myb = lane <= RPW ? rp[min(row0 + lane, n)] : 0;
        const int64_t e0 = __shfl_sync(FULL, myb, 0);
        const int rel = (int)(myb - e0);  // row bound j on lane j, relative to e0
        int bnd[RPW + 1];
#pragma unroll
        for (int j = 0; j <= RPW; j++) bnd[j] = __shfl_sync(FULL, rel, j);
#pragma unroll
        for (int r = 0; r < RPW; r++) tile[r][lane] = A(0);
        const int len = bnd[RPW];
        const V* __restrict__ vr = v + e0;
        const int32_t* __restrict__ cr = ci + e0;
        int r = 0, nb = bnd[1];
        A acc = A(0);
        auto take = [&](int k, A val, A xv) {
            while (k >= nb) {  // rows ending before entry k
                tile[r][lane] = acc;
                acc = A(0);
                r++;
#pragma unroll
                for (int j = 1; j <= RPW; j++)
                    if (j == r + 1) nb = bnd[j];
            }
            acc = fma(val, xv, acc);
        };
        for (int k0 = lane; k0 < len; k0 += 128) {
            const int k1 = k0 + 32, k2 = k0 + 64, k3 = k0 + 96;
            const A v0 = (A)ldv(vr, k0);
            const A v1 = k1 < len ? (A)ldv(vr, k1) : A(0);
            const A v2 = k2 < len ? (A)ldv(vr, k2) : A(0);
            const A v3 = k3 < len ? (A)ldv(vr, k3) : A(0);
            const int c0 = __ldg(cr + k0);
            const int c1 = k1 < len ? __ldg(cr + k1) : 0;
            const int c2 = k2 < len ? __ldg(cr + k2) : 0;
            const int c3 = k3 < len ? __ldg(cr + k3) : 0;
            const A x0 = (A)x[c0];
            const A x1 = k1 < len ? (A)x[c1] : A(0);
            const A x2 = k2 < len ? (A)x[c2] : A(0);
            const A x3 = k3 < len ? (A)x[c3] : A(0);
            take(k0, v0, x0);
            if (k1 < len) take(k1, v1, x1);
            if (k2 < len) take(k2, v2, x2);
            if (k3 < len) take(k3, v3, x3);
        }
        if (r < RPW) tile[r][lane] = acc;
    }
};

template <typename V>
struct RunM {
    static constexpr bool kFlat = false;
    const int64_t* __restrict__ rp;
    const int32_t* __restrict__ rptr;
    const uint8_t* __restrict__ rlen;
    const int32_t* __restrict__ rst;
    const V* __restrict__ v;
    template <typename A, typename X>
    __device__ __forceinline__ A partial(const X* __restrict__ x, int i, int lane) const {
        constexpr int S = 32;
        const int64_t b = __ldg(rp + i), e = __ldg(rp + i + 1);
        const uint32_t L = rlen[i];
        const uint32_t mg = kRunMagic[L];
        const int32_t* __restrict__ rs = rst + __ldg(rptr + i);
        const uint32_t len = (uint32_t)(e - b);
        const V* __restrict__ vr = v + b;
        A acc = A(0);
        uint32_t u = lane;
        auto col = [&](uint32_t w) {
            const uint32_t q = __umulhi(w, mg);
            return __ldg(rs + q) + (int)(w - q * L);
        };
        for (; u + 3 * S < len; u += 4 * S) {
            const A v0 = (A)ldv(vr, u), v1 = (A)ldv(vr, u + S), v2 = (A)ldv(vr, u + 2 * S), v3 = (A)ldv(vr, u + 3 * S);
            const int c0 = col(u), c1 = col(u + S), c2 = col(u + 2 * S), c3 = col(u + 3 * S);
            const A x0 = (A)x[c0], x1 = (A)x[c1], x2 = (A)x[c2], x3 = (A)x[c3];
            acc = fma(v0, x0, acc);
            acc = fma(v1, x1, acc);
            acc = fma(v2, x2, acc);
            acc = fma(v3, x3, acc);
        }
        for (; u < len; u += S) acc = fma((A)ldv(vr, u), (A)x[col(u)], acc);
        return acc;
    }
};

// Row totals for the RPW rows row0 .. row0+RPW-1 (rows >= n give 0).
// Returns the total of row `row0 + lane / (32/RPW)` on every lane.
template <int RPW, typename A, typename M, typename X>
__device__ __forceinline__ A group_rows(const M& mat, const X* __restrict__ x, int row0, int n, int lane,
                                        RowTile<A, RPW>& T) {
    if constexpr (RPW == 1) {
        A s = row0 < n ? mat.template partial<A>(x, row0, lane) : A(0);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        return s;
    } else if constexpr (RPW == 4) {
        // 8 lanes per row: short rows, and levels whose rows are too few for
        // groups of 8.  FP64 instructions are what a row costs (a warp
        // instruction holds a quarter of an SM's FP64 pipe for 64 cycles): a
        // row of 49 entries takes (7 products + 3 adds) / 4 of them here
        // against 2 + 5 with a warp per row.
        const int i = row0 + (lane >> 3);
        A s = i < n ? mat.template sub<A>(x, i, lane & 7) : A(0);
        __syncwarp();
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        return s;
    } else if constexpr (RPW == 32) {
        return mat.template ordered<A>(x, row0, n, lane, T);
    } else {
        constexpr int LPR = 32 / RPW;  // lanes per row in the finishing step
        A(*tile)[33] = T.t;
        if constexpr (M::kFlat) {
            mat.template flat<RPW, A>(x, row0, n, lane, tile);
        } else {
#pragma unroll 1
            for (int r = 0; r < RPW; r++) {
                const int i = row0 + r;
                tile[r][lane] = i < n ? mat.template partial<A>(x, i, lane) : A(0);
            }
        }
        __syncwarp();
        const int r = lane / LPR, q = lane % LPR;
        A s = A(0);
#pragma unroll
        for (int t = 0; t < RPW; t++) s += tile[r][q * RPW + t];
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        __syncwarp();
        return s;
    }
}

// Deterministic sum of one value per lane over the block -> *out (thread 0).
// STEP: only every STEP-th lane holds a value (a row's owner), the others
// zero, so the adds among them are left out.
template <int STEP = 1>
__device__ __forceinline__ void block_partial(double tv, double* sh, double* out) {
#pragma unroll
    for (int o = 16; o >= STEP; o >>= 1) tv += __shfl_xor_sync(FULL, tv, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = tv;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += sh[w];
        *out = s;
    }
}

#define DONE_GUARD(st)                  \
    do {                                \
        if ((st) && (st)->done) return; \
    } while (0)

// Common prologue of the row-group kernels.
#define ROWGROUP_PROLOGUE(A)                                           \
    __shared__ RowTile<A, RPW> tiles[kWarpsPerBlock];                   \
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;         \
    const int row0 = (blockIdx.x * kWarpsPerBlock + wid) * RPW;        \
    constexpr int LPR = 32 / RPW;                                      \
    const int myrow = row0 + lane / LPR;                               \
    const bool owner = (lane % LPR) == 0 && myrow < n;                 \
    (void)owner;

// ----------------------------------------------------------------- kernels
template <int RPW, typename M>
__global__ void __launch_bounds__(kBlock) k_spmv(int n, M mat, const double* __restrict__ x, double* y) {
    pdl_entry();
    ROWGROUP_PROLOGUE(double)
    const double s = group_rows<RPW, double>(mat, x, row0, n, lane, tiles[wid]);
    if (owner) y[myrow] = s;
}

// FP64: r = F - K x, x0 = r / d (optional, in X0), partials ||r||^2, ||F||^2.
// `gate` (optional): run only while the solve is not done and a
// residual replacement is due.
template <int RPW, typename X0, typename M>
__global__ void __launch_bounds__(kBlock) k_residual0(int n, M mat, const double* __restrict__ x,
                                                       const double* __restrict__ F,
                                                       const X0* __restrict__ invd, double* r, X0* x0,
                                                       double* part_rr, double* part_ff, const SolveState* gate) {
    pdl_entry();
    // grid-stride over row groups (a small grid: the gated launch of every
    // mixed-precision iteration returns at once unless a replacement is due)
    if (gate && (gate->done || !gate->replace_now)) return;
    __shared__ RowTile<double, RPW> tiles[kWarpsPerBlock];
    __shared__ double sh[kWarpsPerBlock];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int LPR = 32 / RPW;
    double rr = 0.0, ff = 0.0;
    const int ngroups = (n + RPW - 1) / RPW;
    for (int g = blockIdx.x * kWarpsPerBlock + wid; g - wid < ngroups; g += gridDim.x * kWarpsPerBlock) {
        const int row0 = g * RPW;  // groups past the end give zero rows (uniform per block)
        const double s = group_rows<RPW, double>(mat, x, row0, n, lane, tiles[wid]);
        const int myrow = row0 + lane / LPR;
        if ((lane % LPR) == 0 && myrow < n) {
            const double fi = F[myrow], ri = fi - s;
            r[myrow] = ri;
            if (x0) x0[myrow] = (X0)ri * invd[myrow];
            rr += ri * ri;
            ff += fi * fi;
        }
    }
    block_partial<LPR>(rr, sh, part_rr + blockIdx.x);
    if (part_ff) block_partial<LPR>(ff, sh, part_ff + blockIdx.x);
}

// Outer SpMV q = K p (values V, gathered vector PX, accumulation A; q FP64),
// partials p.q and (flexible) p.r with the FP64 p (part_pq null: none).
template <int RPW, typename A, typename M, typename PX>
__global__ void __launch_bounds__(kBlock) k_spmv_pq(int n, M mat, const PX* __restrict__ pg,
                                                     const double* __restrict__ p,
                                                     const double* __restrict__ r, double* q, double* part_pq,
                                                     double* part_pr, int flexible, const SolveState* st) {
    pdl_entry();
    DONE_GUARD(st);
    ROWGROUP_PROLOGUE(A)
    __shared__ double sh[kWarpsPerBlock];
    const A s = group_rows<RPW, A>(mat, pg, row0, n, lane, tiles[wid]);
    double pq = 0.0, pr = 0.0;
    if (owner) {
        const double qs = (double)s;
        q[myrow] = qs;
        if (part_pq) {
            const double pi = p[myrow];
            pq = pi * qs;
            if (flexible) pr = pi * r[myrow];
        }
    }
    if (!part_pq) return;
    block_partial<LPR>(pq, sh, part_pq + blockIdx.x);
    if (flexible) block_partial<LPR>(pr, sh, part_pr + blockIdx.x);
}

// rbuf = f - K x (down-sweep residual of one level).
template <int RPW, typename A, typename M, typename FT, typename XT>
__global__ void __launch_bounds__(kBlock) k_resid(int n, M mat, const FT* __restrict__ f, const XT* __restrict__ x,
                                                   A* rbuf, const SolveState* st) {
    pdl_entry();
    DONE_GUARD(st);
    ROWGROUP_PROLOGUE(A)
    const A s = group_rows<RPW, A>(mat, x, row0, n, lane, tiles[wid]);
    if (owner) rbuf[myrow] = (A)f[myrow] - s;
}

// Down sweep of one level with its restriction: f_c[J] = sum_{i in J, ascending}
// p_i (f - K x)_i, x_c = f_c / d_c (xc null: not wanted).  A block takes `rows`
// coarse rows and computes the residuals of their members, which are
// consecutive in midx, in shared memory (kMembers at most), a row or RPW rows
// per warp as k_resid does: the restriction needs neither a launch of its own
// (2.3 to 3.5 us on any level of up to a few thousand rows) nor the residual in
// memory.  The sums are those of k_resid and k_restrict in the same order.
// Measured per V-cycle: 2-D p = 3 n = 101 (levels of 10,404 to 713 rows) 5.5 us
// less, 3-D p = 2 n = 49 (29,866 to 513 rows) 12 us less.
template <int RPW>
constexpr int kMembers = RPW * kWarpsPerBlock > kMaxMembers ? RPW * kWarpsPerBlock : kMaxMembers;
template <int RPW, typename A, typename M, typename FT>
__global__ void __launch_bounds__(kBlock) k_resid_restrict(int nc, int rows, M mat, const FT* __restrict__ f,
                                                            const A* __restrict__ x, const A* __restrict__ invdc,
                                                            const int32_t* __restrict__ mptr,
                                                            const int32_t* __restrict__ midx,
                                                            const double* __restrict__ pval, A* fc, A* xc,
                                                            const SolveState* st) {
    static_assert(RPW == 1 || RPW == 4, "lanes of one row");
    constexpr int LPR = 32 / RPW;
    pdl_entry();
    DONE_GUARD(st);
    __shared__ A ts[kMembers<RPW>], ps[kMembers<RPW>];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, q = lane % LPR;
    const int J0 = blockIdx.x * rows, J1 = min(J0 + rows, nc);
    const int J = J0 + (int)threadIdx.x;  // folded by this thread, if below J1
    const int m0 = mptr[J0], m1 = mptr[J1];
    const int jb = J < J1 ? mptr[J] : 0, je = J < J1 ? mptr[J + 1] : 0;
    for (int mw = m0 + wid * RPW; mw < m1; mw += kWarpsPerBlock * RPW) {  // warp-uniform
        const int m = mw + lane / LPR;
        const bool on = m < m1;
        const int i = on ? midx[m] : 0;
        const A fi = on ? (A)f[i] : A(0), pi = on ? (A)pval[i] : A(0);
        A s = A(0);
        if constexpr (RPW == 1) s = mat.template partial<A>(x, i, lane);
        else if (on) s = mat.template sub<A>(x, i, q);
        __syncwarp();
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        if (on && q == 0) {
            ts[m - m0] = fi - s;
            ps[m - m0] = pi;
        }
    }
    __syncthreads();
    if (J < J1) {
        A acc = A(0);
        for (int m = jb; m < je; m++) acc = fma(ps[m - m0], ts[m - m0], acc);
        fc[J] = acc;
        if (xc) xc[J] = acc * invdc[J];
    }
}

// t = x + (f - K x) / d (extra smoothing sweep).
template <int RPW, typename A, typename M, typename FT>
__global__ void __launch_bounds__(kBlock) k_sweep(int n, M mat, const FT* __restrict__ f, const A* __restrict__ x,
                                                   const A* __restrict__ invd, A* t, const SolveState* st) {
    pdl_entry();
    DONE_GUARD(st);
    ROWGROUP_PROLOGUE(A)
    const A s = group_rows<RPW, A>(mat, x, row0, n, lane, tiles[wid]);
    if (owner) t[myrow] = fma(invd[myrow], (A)f[myrow] - s, x[myrow]);
}

// Up sweep of level l >= 1: y_a = x_a + (f_a - (K x)_a) / d_a, then
// x_{l-1}[c] += p_c y_a for the members c of a (one member per lane of the
// row's lane group; with a row per lane, the members of the warp's 32 rows,
// which are consecutive in midx, go over the lanes, each finding its row's y
// through its aggregate).
template <int RPW, typename A, typename M>
__global__ void __launch_bounds__(kBlock) k_up(int n, M mat, const A* __restrict__ f, const A* __restrict__ x,
                                                const A* __restrict__ invd,
                                                const int32_t* __restrict__ mptr, const int32_t* __restrict__ midx,
                                                const int32_t* __restrict__ aggf, const double* __restrict__ pvalf,
                                                A* xf, const SolveState* st) {
    pdl_entry();
    DONE_GUARD(st);
    ROWGROUP_PROLOGUE(A)
    const A s = group_rows<RPW, A>(mat, x, row0, n, lane, tiles[wid]);
    if constexpr (RPW == 32) {
        if (row0 >= n) return;
        const A y = myrow < n ? fma(invd[myrow], f[myrow] - s, x[myrow]) : A(0);
        const int m1 = mptr[min(row0 + 32, n)];
#pragma unroll 4
        for (int m0 = mptr[row0]; m0 < m1; m0 += 32) {
            const bool in = m0 + lane < m1;
            const int c = in ? midx[m0 + lane] : 0;
            const A ya = __shfl_sync(FULL, y, in ? aggf[c] - row0 : 0);
            if (in) xf[c] = fma((A)pvalf[c], ya, xf[c]);
        }
    } else if (myrow < n) {
        // every lane of the row's group has the total; the aggregate's members
        // (independent fine rows) are spread over those LPR lanes
        const A y = fma(invd[myrow], f[myrow] - s, x[myrow]);
        const int m1 = mptr[myrow + 1];
        for (int m = mptr[myrow] + lane % LPR; m < m1; m += LPR) {
            const int c = midx[m];
            xf[c] = fma((A)pvalf[c], y, xf[c]);
        }
    }
}

// Up sweep of level 0: z = x + (r - K x) / d (z FP64); partials r.z and
// (flexible) z.q (part_rz null: none).
template <int RPW, typename A, typename M>
__global__ void __launch_bounds__(kBlock) k_up0(int n, M mat, const double* __restrict__ r,
                                                 const A* __restrict__ x, const A* __restrict__ invd, double* z,
                                                 const double* __restrict__ q, double* part_rz, double* part_zq,
                                                 int flexible, const SolveState* st) {
    pdl_entry();
    DONE_GUARD(st);
    ROWGROUP_PROLOGUE(A)
    __shared__ double sh[kWarpsPerBlock];
    const A s = group_rows<RPW, A>(mat, x, row0, n, lane, tiles[wid]);
    double rz = 0.0, zq = 0.0;
    if (owner) {
        const double ra = r[myrow];
        const double za = (double)fma(invd[myrow], (A)ra - s, x[myrow]);
        z[myrow] = za;
        if (part_rz) {
            rz = ra * za;
            if (flexible) zq = za * q[myrow];
        }
    }
    if (!part_rz) return;
    block_partial<LPR>(rz, sh, part_rz + blockIdx.x);
    if (flexible) block_partial<LPR>(zq, sh, part_zq + blockIdx.x);
}

}  // namespace
}  // namespace amg
