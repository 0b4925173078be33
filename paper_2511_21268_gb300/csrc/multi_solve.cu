// Multi-system CG: S independent CG iterations sharing one AMG hierarchy,
// run in one graph-captured loop (arXiv 2511.21268 Sec. 3 V-cycle and CG;
// the batching is this library's design).
//
//   * R right-hand sides of one matrix (k_m_*): vectors interleaved as
//     [N][Rs], Rs = R rounded up to a multiple of 4 (mixed precision) or 2
//     (FP64), so that a row is whole 16-byte pieces; the padding columns
//     zero; a matrix pass reads each matrix entry once for all R vectors
//     (SpMM).  System s = right-hand side s.
//   * a batch of independent matrices assembled block-diagonally into one
//     hierarchy (k_b_*; there are no coupling entries, so matchings,
//     aggregates and Galerkin products never cross blocks and every level
//     operator is block diagonal): the V-cycle and q = K p are the
//     single-system row-group kernels on the whole matrix, the vector
//     kernels run on tiles of one system's rows each.
//
// Each system has its own CG scalars and convergence test; the dot products
// are per-system sums in a fixed order (deterministic): one partial sum per
// block or tile, added up by the kernel that updates the scalars.  Converged
// systems are frozen while the others iterate.  The V-cycle uses one pre-
// and one post-smoothing sweep.
//
// What bounds the SpMM and why this split.  Per stored entry it needs the
// entry's value and column and Rs vector values, one row of the interleaved
// vector (64 bytes for 16 right-hand sides in FP32) gathered through L1.  A
// lane owns 16 bytes of that row (4 right-hand sides in FP32, 2 in FP64), lp =
// Rs sizeof / 16 lanes (rounded up to a power of two) cover it, and the warp's
// 32 / lp lane groups take different entries, so that the value and column
// loads are one wavefront for the whole group.  The gathers are bound by
// their latency, so fewer of them is what helps: on the finest level the
// run-encoded columns show which vector rows four neighbouring matrix rows
// share (10 instead of 28 for runs of 7), and a warp takes four rows at once
// (spmm_runs); the other levels go row by row (spmm_rows).  FP64 instructions
// occupy GB300's two-lane FP64 pipe for 16 cycles however few lanes are
// active, so the epilogues (FP64 dot products and conversions) run with a
// (row, right-hand side) pair per lane, and the partial sums of a dot product
// are few.  Measured, 3-D p = 3 n = 32 (10.5 M entries), 16 right-hand sides in
// mixed precision, us per pass before (a lane per right-hand side, every entry
// a load of its own) and after: q = K p 102 -> 58, residual 106 -> 67, up
// sweep 100 -> 59, a level below the first 33 and 19 -> 11 and 10, the dots and
// scalars of an iteration 140 -> 23; 102.5 -> 48.6 ms a solve.
//
// Few right-hand sides in FP64, us per iteration of a solve with a lane per
// right-hand side / rows of four columns / of two (now, 1 or 2 right-hand sides):
// 3-D p = 3 n = 24 400 / 220 / 168, 3-D p = 2 n = 40 490 / 442 / 343, 2-D p = 3 n =
// 101 144 / 100 / 102; workspace of one, bytes per row (4 M rows of 5 entries): 84 /
// 294 / 143.  In mixed precision one to three columns are carried as four: 385 to
// 427 -> 120 us, 436 to 461 -> 222 and 160 -> 94 on the same systems.
//
// A batch's passes over level 0 (24 2-D systems, p 2..4, n 32..160, mixed
// precision): 46, 40 and 35 us with a thread per row -> 27, 26 and 26 us with
// the staged row order of CsrM::ordered; 42.5 -> 29.6 ms setup and solve.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "amg_internal.cuh"
#include "row_kernels.cuh"

namespace amg {

namespace {

// ------------------------------------------------------ 16-byte vector access
template <typename T>
constexpr int kVec = 16 / sizeof(T);  // right-hand sides per lane
template <typename T>
constexpr int kBatch = sizeof(T) == 4 ? 8 : 4;  // entries per lane group in flight (row by row)

// N consecutive values in 16-byte pieces (p aligned to 16 bytes)
template <int N>
__device__ __forceinline__ void load_vec(const float* __restrict__ p, float (&v)[N]) {
    static_assert(N == 4, "a lane owns 4 FP32 columns");
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
template <int N>
__device__ __forceinline__ void load_vec(const double* __restrict__ p, double (&v)[N]) {
    static_assert(N % 2 == 0, "16-byte pieces");
#pragma unroll
    for (int j = 0; j < N; j += 2) {
        const double2 a = *reinterpret_cast<const double2*>(p + j);
        v[j] = a.x, v[j + 1] = a.y;
    }
}
// Lane layout of the SpMM kernels.  Gather: lane group g = lane / lp takes
// every (32 / lp)-th entry, the lane's kVec columns start at c0.  After the
// reduction a lane holds column c (own: c < Rs) of the row that its copy
// index dup selects; 32 / (kVec lp) copies of each column.
struct Lanes {
    int lp, g, c0, c, dup;
    bool own;
};
template <typename A>
__device__ __forceinline__ Lanes lanes_of(int Rs, int lp) {
    const int lane = threadIdx.x & 31, q = lane & (lp - 1);
    Lanes L;
    L.lp = lp;
    L.g = lane / lp;
    L.c0 = q * kVec<A> < Rs ? q * kVec<A> : 0;  // lanes past the last column repeat the first
    if (kVec<A> == 4) {
        L.c = q * 4 + ((lane >> 4) & 1) * 2 + ((lane >> 3) & 1);
        L.dup = (lane & 7) / lp;
    } else {
        L.c = q * 2 + ((lane >> 4) & 1);
        L.dup = (lane & 15) / lp;
    }
    L.own = L.c < Rs;
    return L;
}
template <typename A>
__device__ __forceinline__ int copies_of(const Lanes& L) {
    return 32 / (kVec<A> * L.lp);
}

// Sum over the lane groups; the lane's column c is returned (each step of
// the first halves the columns a lane carries).
__device__ __forceinline__ float reduce_columns(const float (&a)[4], const Lanes& L) {
    const int lane = threadIdx.x & 31;
    const bool h = lane & 16, e = lane & 8;
    const float b0 = (h ? a[2] : a[0]) + __shfl_xor_sync(FULL, h ? a[0] : a[2], 16);
    const float b1 = (h ? a[3] : a[1]) + __shfl_xor_sync(FULL, h ? a[1] : a[3], 16);
    float s = (e ? b1 : b0) + __shfl_xor_sync(FULL, e ? b0 : b1, 8);
    for (int o = 4; o >= L.lp; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
    return s;
}
__device__ __forceinline__ double reduce_columns(const double (&a)[2], const Lanes& L) {
    const bool h = threadIdx.x & 16;
    double s = (h ? a[1] : a[0]) + __shfl_xor_sync(FULL, h ? a[0] : a[1], 16);
    for (int o = 8; o >= L.lp; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
    return s;
}

// acc[j] = sum_k v_k x[c_k][c0 + j] over the lane group's entries of a row of
// `len` entries.  U vector rows per lane group are in flight; the values
// and columns of the next batch load meanwhile.  Entries past the end are not
// loaded (their product must not meet an infinite vector value).
template <typename A, int U, typename V>
__device__ __forceinline__ void row_dot(int len, const V* __restrict__ v, const int32_t* __restrict__ col,
                                        const A* __restrict__ x, int Rs, const Lanes& L, A (&acc)[kVec<A>]) {
    constexpr int N = kVec<A>;
    const int G = 32 / L.lp;
    const A* __restrict__ xc = x + L.c0;
#pragma unroll
    for (int j = 0; j < N; j++) acc[j] = A(0);
    A vv[U], vn[U];
    int cc[U], cn[U];
    auto load = [&](int k, A (&vo)[U], int (&co)[U]) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            const bool in = k + u * G < len;
            vo[u] = in ? (A)ldv(v, k + u * G) : A(0);
            co[u] = in ? __ldg(col + k + u * G) : -1;
        }
    };
    load(L.g, vv, cc);
    for (int k = 0; k < len; k += U * G) {  // warp-uniform
        A xx[U][N];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (cc[u] >= 0) load_vec<N>(xc + (int64_t)cc[u] * Rs, xx[u]);
        load(k + U * G + L.g, vn, cn);
#pragma unroll
        for (int u = 0; u < U; u++)
            if (cc[u] >= 0) {
#pragma unroll
                for (int j = 0; j < N; j++) acc[j] = fma(vv[u], xx[u][j], acc[j]);
            }
#pragma unroll
        for (int u = 0; u < U; u++) vv[u] = vn[u], cc[u] = cn[u];
    }
    __syncwarp();
}

// Matrix views: plain CSR, and CSR with run-encoded columns as well.
template <typename V>
struct MatM {
    const int64_t* __restrict__ rp;
    const int32_t* __restrict__ ci;
    const V* __restrict__ v;
    const int32_t* __restrict__ rptr;  // null: no runs
    const uint8_t* __restrict__ rlen;
    const int32_t* __restrict__ rst;
};

// K x over the rows of this warp.  fin(i, valid, s) is called by all lanes
// with the lane's row i, its column's sum s, and whether the lane has a (row,
// column) pair at all.  Row by row: blocks of T consecutive rows (T at most
// the copies of a column) share one call of fin.
template <typename A, typename V, typename Fin>
__device__ __forceinline__ void spmm_rows(int n, int Rs, int T, const Lanes& L, const MatM<V>& M,
                                          const A* __restrict__ x, Fin&& fin) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, W = (gridDim.x * blockDim.x) >> 5;
    for (int64_t i0 = (int64_t)warp * T; i0 < n; i0 += (int64_t)W * T) {
        const int cnt = (int)min((int64_t)T, n - i0);
        A keep = A(0);
        for (int t = 0; t < cnt; t++) {
            const int64_t b = M.rp[i0 + t];
            A acc[kVec<A>];
            row_dot<A, kBatch<A>>((int)(M.rp[i0 + t + 1] - b), M.v + b, M.ci + b, x, Rs, L, acc);
            const A s = reduce_columns(acc, L);
            if (L.dup == t) keep = s;
        }
        fin((int)i0 + L.dup, L.own && L.dup < cnt, keep);
    }
}

// Four rows at once from the run-encoded columns.  In a tensor-product matrix
// neighbouring rows of a line have the same number of runs, and run r of row
// j starts delta_j columns after run r of the first row, delta_j the same for
// all runs.  The lane groups take runs; per run the union of the four rows'
// columns (W <= kRunSpan) is gathered once and multiplied into every row that
// has the column.  Tiles that are not like that (the end of a line, any other
// run structure, found while reading the runs) go row by row.
constexpr int kTile = 4, kRunSpan = 12;
template <typename A, typename V, typename Fin>
__device__ __forceinline__ void spmm_runs(int n, int Rs, const Lanes& L, const MatM<V>& M, const A* __restrict__ x,
                                          Fin&& fin) {
    constexpr int N = kVec<A>, Q = 4;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, W = (gridDim.x * blockDim.x) >> 5;
    const int G = 32 / L.lp, D = copies_of<A>(L);
    const A* __restrict__ xc = x + L.c0;
    for (int64_t i0 = (int64_t)warp * kTile; i0 < n; i0 += (int64_t)W * kTile) {
        const int cnt = (int)min((int64_t)kTile, n - i0);
        A acc[kTile][N];
#pragma unroll
        for (int j = 0; j < kTile; j++)
#pragma unroll
            for (int q = 0; q < N; q++) acc[j][q] = A(0);
        bool ok = cnt == kTile;
        if (ok) {
            int rb[kTile], len[kTile], dl[kTile];
            const V* vb[kTile];
            const int runs = M.rptr[i0 + 1] - M.rptr[i0];
            int span = 0;
#pragma unroll
            for (int j = 0; j < kTile; j++) {
                rb[j] = M.rptr[i0 + j];
                len[j] = M.rlen[i0 + j];
                vb[j] = M.v + M.rp[i0 + j];
                ok = ok && M.rptr[i0 + j + 1] - rb[j] == runs;
            }
            ok = ok && runs > 0;
            if (ok) {
                const int s0 = __ldg(M.rst + rb[0]);
#pragma unroll
                for (int j = 0; j < kTile; j++) {
                    dl[j] = __ldg(M.rst + rb[j]) - s0;
                    ok = ok && dl[j] >= 0 && dl[j] < kRunSpan;
                    span = max(span, dl[j] + len[j]);
                }
                ok = ok && span <= kRunSpan;
            }
            if (ok) {  // uniform so far
                bool same = true;
                for (int r0 = 0; r0 < runs; r0 += G) {
                    const int r = r0 + L.g;
                    if (r < runs) {
                        const int st = __ldg(M.rst + rb[0] + r);
                        int vo[kTile];
#pragma unroll
                        for (int j = 0; j < kTile; j++) {
                            if (j > 0) same = same && __ldg(M.rst + rb[j] + r) - st == dl[j];
                            vo[j] = r * len[j] - dl[j];
                        }
#pragma unroll 1
                        for (int o0 = 0; o0 < span; o0 += Q) {
                            {
                                A xx[Q][N], vv[kTile][Q];
#pragma unroll
                                for (int q = 0; q < Q; q++)
                                    load_vec<N>(xc + (int64_t)min(st + min(o0 + q, span - 1), n - 1) * Rs, xx[q]);
#pragma unroll
                                for (int j = 0; j < kTile; j++)
#pragma unroll
                                    for (int q = 0; q < Q; q++) {
                                        const bool in = (unsigned)(o0 + q - dl[j]) < (unsigned)len[j];
                                        vv[j][q] = in ? (A)ldv(vb[j], vo[j] + o0 + q) : A(0);
                                    }
#pragma unroll
                                for (int j = 0; j < kTile; j++)
#pragma unroll
                                    for (int q = 0; q < Q; q++)
                                        if ((unsigned)(o0 + q - dl[j]) < (unsigned)len[j]) {
#pragma unroll
                                            for (int c = 0; c < N; c++)
                                                acc[j][c] = fma(vv[j][q], xx[q][c], acc[j][c]);
                                        }
                            }
                        }
                    }
                }
                ok = __all_sync(FULL, same);
            }
        }
        A s[kTile];
        if (ok) {
#pragma unroll
            for (int j = 0; j < kTile; j++) s[j] = reduce_columns(acc[j], L);
        } else {
#pragma unroll 1
            for (int t = 0; t < cnt; t++) {
                const int64_t b = M.rp[i0 + t];
                A a1[N];
                row_dot<A, 4>((int)(M.rp[i0 + t + 1] - b), M.v + b, M.ci + b, x, Rs, L, a1);
                const A r = reduce_columns(a1, L);
#pragma unroll
                for (int j = 0; j < kTile; j++)
                    if (j == t) s[j] = r;
            }
        }
        for (int base = 0; base < cnt; base += D) {
            A keep = A(0);
#pragma unroll
            for (int j = 0; j < kTile; j++)
                if (j == base + L.dup) keep = s[j];
            fin((int)i0 + base + L.dup, L.own && base + L.dup < cnt, keep);
        }
    }
}

template <typename A, bool RUNS, typename V, typename Fin>
__device__ __forceinline__ void spmm(int n, int Rs, int T, const Lanes& L, const MatM<V>& M, const A* __restrict__ x,
                                     Fin&& fin) {
    if constexpr (RUNS) spmm_runs<A>(n, Rs, L, M, x, fin);
    else spmm_rows<A>(n, Rs, T, L, M, x, fin);
}

constexpr int kMaxRs = 32;  // padded right-hand sides

// Block partial sums per right-hand side: every lane holds its column's sum;
// *out receives Rs values (a column's copies, then the warps, in order).
template <typename A>
__device__ __forceinline__ void block_columns(double t, const Lanes& L, int Rs, double* sh, double* out) {
    const int wid = threadIdx.x >> 5;
    for (int o = (kVec<A> == 4 ? 4 : 8); o >= L.lp; o >>= 1) t += __shfl_xor_sync(FULL, t, o);
    __syncthreads();
    if (L.own && L.dup == 0) sh[wid * kMaxRs + L.c] = t;
    __syncthreads();
    if ((int)threadIdx.x < Rs) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += sh[w * kMaxRs + threadIdx.x];
        out[threadIdx.x] = s;
    }
}

// ------------------------------------------- kernels, several right-hand sides
// FP64 residual r = F - K x; x0 = r / d (V-cycle precision); block partials
// of r^2 and F^2.  due: only the right-hand sides of the mask (a residual
// replacement); the kernel returns at once when it is empty.
template <typename X0>
__global__ void __launch_bounds__(kBlock, 2) k_m_residual(int n, int Rs, int lp, int T, MatM<double> mat,
                                                        const double* __restrict__ x, const double* __restrict__ F,
                                                        const X0* __restrict__ invd, double* r, X0* x0,
                                                        double* part_rr, double* part_ff, const unsigned* due) {
    pdl_entry();
    const unsigned mask = due ? *due : FULL;
    if (mask == 0) return;
    __shared__ double sh[kWarpsPerBlock * kMaxRs];
    const Lanes L = lanes_of<double>(Rs, lp);
    double rr = 0.0, ff = 0.0;
    const bool mine = L.own && (mask >> L.c & 1u);
    spmm_rows<double>(n, Rs, T, L, mat, x, [&](int i, bool valid, double s) {
        if (!valid || !mine) return;
        const int64_t e = (int64_t)i * Rs + L.c;
        const double fi = F[e], ri = fi - s;
        r[e] = ri;
        if (x0) x0[e] = (X0)ri * invd[i];
        rr = fma(ri, ri, rr);
        if (part_ff) ff = fma(fi, fi, ff);
    });
    block_columns<double>(rr, L, Rs, sh, part_rr + (int64_t)blockIdx.x * Rs);
    if (part_ff) block_columns<double>(ff, L, Rs, sh, part_ff + (int64_t)blockIdx.x * Rs);
}

// Outer q = K p; block partials of p.q and (flexible) p.r.  The columns of
// finished systems are computed too: nothing reads them.
template <bool RUNS, typename A, typename V>
__global__ void __launch_bounds__(kBlock, 2) k_m_spmv_pq(int n, int Rs, int lp, int T, MatM<V> mat,
                                                       const A* __restrict__ pg, const double* __restrict__ p,
                                                       const double* __restrict__ r, double* q, double* part_pq,
                                                       double* part_pr, int flexible, const int* active) {
    pdl_entry();
    if (*active == 0) return;
    __shared__ double sh[kWarpsPerBlock * kMaxRs];
    const Lanes L = lanes_of<A>(Rs, lp);
    double pq = 0.0, pr = 0.0;
    spmm<A, RUNS>(n, Rs, T, L, mat, pg, [&](int i, bool valid, A s) {
        if (!valid) return;
        const int64_t e = (int64_t)i * Rs + L.c;
        const double qs = (double)s, pi = p[e];
        q[e] = qs;
        pq = fma(pi, qs, pq);
        if (flexible) pr = fma(pi, r[e], pr);
    });
    block_columns<A>(pq, L, Rs, sh, part_pq + (int64_t)blockIdx.x * Rs);
    if (flexible) block_columns<A>(pr, L, Rs, sh, part_pr + (int64_t)blockIdx.x * Rs);
}

// V-cycle down-sweep residual rbuf = f - K x.
template <bool RUNS, typename A, typename V, typename FT>
__global__ void __launch_bounds__(kBlock, 2) k_m_resid(int n, int Rs, int lp, int T, MatM<V> mat,
                                                     const FT* __restrict__ f, const A* __restrict__ x, A* rbuf,
                                                     const int* active) {
    pdl_entry();
    if (*active == 0) return;
    const Lanes L = lanes_of<A>(Rs, lp);
    spmm<A, RUNS>(n, Rs, T, L, mat, x, [&](int i, bool valid, A s) {
        if (!valid) return;
        const int64_t e = (int64_t)i * Rs + L.c;
        rbuf[e] = (A)f[e] - s;
    });
}

// Residual and restriction of a level in one kernel, as k_resid_restrict: a
// block takes `rows` coarse rows, a warp a member, and the residuals of the
// members stay in shared memory.  Same sums in the same order.  For levels with
// a warp for every row (at most 16 rows per SM): 16 right-hand sides, the two
// small levels of 3-D p = 3 n = 32, 18.5 -> 12.3 us per V-cycle.  With the level
// above them too, of 12 rows per warp, nothing more was gained (48.0 -> 48.2 ms a
// solve).
template <typename A, typename V>
__global__ void __launch_bounds__(kBlock, 2) k_m_resid_restrict(
    int nc, int rows, int Rs, int lp, MatM<V> mat, const A* __restrict__ f, const A* __restrict__ x,
    const int32_t* __restrict__ mptr, const int32_t* __restrict__ midx, const double* __restrict__ pval, A* fc, A* xc,
    const A* __restrict__ invdc, const int* active) {
    pdl_entry();
    if (*active == 0) return;
    constexpr int kMembers = kWarpsPerBlock > kMaxMembers ? kWarpsPerBlock : kMaxMembers;
    __shared__ A ts[kMembers][kMaxRs], ps[kMembers];
    const Lanes L = lanes_of<A>(Rs, lp);
    const int wid = threadIdx.x >> 5;
    for (int J0 = blockIdx.x * rows; J0 < nc; J0 += gridDim.x * rows) {
        const int J1 = min(J0 + rows, nc), m0 = mptr[J0], m1 = mptr[J1];
        for (int m = m0 + wid; m < m1; m += kWarpsPerBlock) {
            const int i = midx[m];
            const A pi = (A)pval[i], fi = L.own ? f[(int64_t)i * Rs + L.c] : A(0);
            const int64_t b = mat.rp[i];
            A acc[kVec<A>];
            row_dot<A, kBatch<A>>((int)(mat.rp[i + 1] - b), mat.v + b, mat.ci + b, x, Rs, L, acc);
            const A s = reduce_columns(acc, L);
            if (L.own && L.dup == 0) ts[m - m0][L.c] = fi - s;
            if ((threadIdx.x & 31) == 0) ps[m - m0] = pi;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < (J1 - J0) * Rs; t += kBlock) {
            const int J = J0 + t / Rs, c = t % Rs;
            A acc = A(0);
            for (int m = mptr[J]; m < mptr[J + 1]; m++) acc = fma(ps[m - m0], ts[m - m0][c], acc);
            fc[(int64_t)J * Rs + c] = acc;
            if (xc) xc[(int64_t)J * Rs + c] = acc * invdc[J];
        }
        __syncthreads();
    }
}

template <typename A>
__global__ void k_m_restrict(int nc, int Rs, const int32_t* __restrict__ mptr, const int32_t* __restrict__ midx,
                             const double* __restrict__ pval, const A* __restrict__ rbuf, A* fc, A* xc,
                             const A* __restrict__ invdc, const int* active) {
    pdl_entry();
    if (*active == 0) return;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= (int64_t)nc * Rs) return;
    const int I = (int)(g / Rs), c = (int)(g % Rs);
    A acc = A(0);
    for (int m = mptr[I]; m < mptr[I + 1]; m++) {
        const int a = midx[m];
        acc = fma((A)pval[a], rbuf[(int64_t)a * Rs + c], acc);
    }
    fc[g] = acc;
    if (xc) xc[g] = acc * invdc[I];
}

// Coarsest level, e = A^-1 f per vector (FP64, a block of four warps per row of
// the dense inverse: a warp issues one FP64 instruction in 64 cycles, and the
// conversions of f are FP64 instructions too, so the row is split over the SM's
// four pipes: 12.4 -> 7.5 us for 77 rows and 16 right-hand sides); prolongation
// into the finer level, or (single-level hierarchy) z = e with the block
// partials of r.z and z.q.
constexpr int kCoarseU = 4;  // entries of a lane group in flight
constexpr int kCoarseWarps = 4;
template <typename FT, typename XT>
__global__ void __launch_bounds__(kCoarseWarps * 32) k_m_coarse(int nd, int Rs, int lp, const double* __restrict__ Ainv,
                                                  const FT* __restrict__ f, const int32_t* __restrict__ mptr,
                                                  const int32_t* __restrict__ midx,
                                                  const double* __restrict__ pvalf, XT* xf, double* z,
                                                  const double* __restrict__ q, double* part_rz, double* part_zq,
                                                  int flexible, const int* active) {
    pdl_entry();
    if (*active == 0) return;
    __shared__ double sh[kCoarseWarps * kMaxRs];
    const Lanes L = lanes_of<double>(Rs, lp);
    const int G = 32 / lp, wid = threadIdx.x >> 5;
    double rz = 0.0, zq = 0.0;
    for (int I = blockIdx.x; I < nd; I += gridDim.x) {
        const double* __restrict__ row = Ainv + (int64_t)I * nd;
        double s2[2] = {0.0, 0.0};
        for (int j0 = L.g + wid * G; j0 - L.g < nd; j0 += kCoarseU * kCoarseWarps * G) {
            double a[kCoarseU], x0[kCoarseU], x1[kCoarseU];
#pragma unroll
            for (int u = 0; u < kCoarseU; u++) {
                const int j = j0 + u * kCoarseWarps * G;
                const bool in = j < nd;
                const FT* fj = f + (int64_t)(in ? j : 0) * Rs + L.c0;
                a[u] = in ? __ldg(row + j) : 0.0;
                x0[u] = in ? (double)fj[0] : 0.0;
                x1[u] = in ? (double)fj[1] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < kCoarseU; u++) {
                s2[0] = fma(a[u], x0[u], s2[0]);
                s2[1] = fma(a[u], x1[u], s2[1]);
            }
        }
        __syncwarp();
        double s = reduce_columns(s2, L);
        if (wid > 0 && L.own && L.dup == 0) sh[wid * kMaxRs + L.c] = s;
        __syncthreads();
        if (wid == 0 && L.own)
            for (int w = 1; w < kCoarseWarps; w++) s += sh[w * kMaxRs + L.c];
        __syncthreads();  // sh is free again
        if (wid > 0) continue;
        if (z) {
            if (L.own && L.dup == 0) {
                const int64_t e = (int64_t)I * Rs + L.c;
                z[e] = s;
                rz = fma((double)f[e], s, rz);
                if (flexible) zq = fma(s, q[e], zq);
            }
        } else if (L.own) {  // a member of the aggregate per copy of the column
            const int m1 = mptr[I + 1], step = copies_of<double>(L);
            for (int m = mptr[I] + L.dup; m < m1; m += step) {
                const int a = midx[m];
                XT* xe = xf + (int64_t)a * Rs + L.c;
                *xe = (XT)fma(pvalf[a], s, (double)*xe);
            }
        }
    }
    if (z) {
        block_columns<double>(rz, L, Rs, sh, part_rz + (int64_t)blockIdx.x * Rs);
        if (flexible) block_columns<double>(zq, L, Rs, sh, part_zq + (int64_t)blockIdx.x * Rs);
    }
}

// Up sweep of a level l >= 1: y = x + (f - K x) / d, prolongated into the
// finer level.
template <typename A, typename V>
__global__ void __launch_bounds__(kBlock, 2) k_m_up(int n, int Rs, int lp, int T, MatM<V> mat,
                                                  const A* __restrict__ f, const A* __restrict__ x,
                                                  const A* __restrict__ invd, const int32_t* __restrict__ mptr,
                                                  const int32_t* __restrict__ midx, const double* __restrict__ pvalf,
                                                  A* xf, const int* active) {
    pdl_entry();
    if (*active == 0) return;
    const Lanes L = lanes_of<A>(Rs, lp);
    spmm_rows<A>(n, Rs, T, L, mat, x, [&](int i, bool valid, A s) {
        if (!valid) return;
        const int64_t e = (int64_t)i * Rs + L.c;
        const A y = fma(invd[i], f[e] - s, x[e]);
        const int m1 = mptr[i + 1];
        for (int m = mptr[i]; m < m1; m++) {
            const int a = midx[m];
            A* xe = xf + (int64_t)a * Rs + L.c;
            *xe = fma((A)pvalf[a], y, *xe);
        }
    });
}

// Up sweep of level 0: z = x + (r - K x) / d; block partials of r.z and
// (flexible) z.q.
template <bool RUNS, typename A, typename V>
__global__ void __launch_bounds__(kBlock, 2) k_m_up0(int n, int Rs, int lp, int T, MatM<V> mat,
                                                   const double* __restrict__ r, const A* __restrict__ x,
                                                   const A* __restrict__ invd, double* z,
                                                   const double* __restrict__ q, double* part_rz, double* part_zq,
                                                   int flexible, const int* active) {
    pdl_entry();
    if (*active == 0) return;
    __shared__ double sh[kWarpsPerBlock * kMaxRs];
    const Lanes L = lanes_of<A>(Rs, lp);
    double rz = 0.0, zq = 0.0;
    spmm<A, RUNS>(n, Rs, T, L, mat, x, [&](int i, bool valid, A s) {
        if (!valid) return;
        const int64_t e = (int64_t)i * Rs + L.c;
        const double ra = r[e];
        const double za = (double)fma(invd[i], (A)ra - s, x[e]);
        z[e] = za;
        rz = fma(ra, za, rz);
        if (flexible) zq = fma(za, q[e], zq);
    });
    block_columns<A>(rz, L, Rs, sh, part_rz + (int64_t)blockIdx.x * Rs);
    if (flexible) block_columns<A>(zq, L, Rs, sh, part_zq + (int64_t)blockIdx.x * Rs);
}

// Threads of the vector kernels: Rs / 2 threads per row (two columns each), as many
// rows of a block at a time as there would be with Rs a multiple of 4: one thread
// adds a column's terms of those rows one after another (2 right-hand sides, 2-D
// p = 3 n = 101: 111 us per iteration with 256 rows, 104 with 128).
__host__ __device__ __forceinline__ int pair_rows(int Rs) { return kBlock / (((Rs + 3) & ~3) >> 1); }
struct PairLayout {
    int lpr, rpb, rl, c;
    bool in;
};
__device__ __forceinline__ PairLayout pair_layout(int Rs) {
    PairLayout P;
    P.lpr = Rs >> 1;
    P.rpb = pair_rows(Rs);
    P.rl = threadIdx.x / P.lpr;
    P.c = 2 * (threadIdx.x - P.rl * P.lpr);
    P.in = P.rl < P.rpb;
    return P;
}

// x += alpha p, r -= alpha q, x0 = r / d, block partials of r^2 (systems not
// done).
template <typename X0>
__global__ void __launch_bounds__(kBlock) k_m_update(int n, int R, int Rs, double* x, double* r,
                                                      const double* __restrict__ p, const double* __restrict__ q,
                                                      const X0* __restrict__ invd, X0* x0, double* part_rr,
                                                      const MultiState* st, const int* active) {
    pdl_entry();
    if (*active == 0) return;
    __shared__ double sh[2 * kBlock];
    const PairLayout P = pair_layout(Rs);
    double rr[2] = {0.0, 0.0};
    if (P.in) {
        double alpha[2];
        bool on[2];
#pragma unroll
        for (int j = 0; j < 2; j++) {
            on[j] = P.c + j < R && !st[P.c + j].done;
            alpha[j] = on[j] ? st[P.c + j].alpha : 0.0;
        }
        if (on[0] || on[1])
            for (int64_t i = (int64_t)blockIdx.x * P.rpb + P.rl; i < n; i += (int64_t)gridDim.x * P.rpb) {
                const int64_t e = i * Rs + P.c;
                double xv[2], rv[2], pv[2], qv[2];
                load_vec<2>(x + e, xv);
                load_vec<2>(r + e, rv);
                load_vec<2>(p + e, pv);
                load_vec<2>(q + e, qv);
                const X0 d = x0 ? invd[i] : X0(0);
#pragma unroll
                for (int j = 0; j < 2; j++) {
                    if (!on[j]) continue;
                    x[e + j] = fma(alpha[j], pv[j], xv[j]);
                    const double ri = fma(-alpha[j], qv[j], rv[j]);
                    r[e + j] = ri;
                    if (x0) x0[e + j] = (X0)ri * d;
                    rr[j] = fma(ri, ri, rr[j]);
                }
            }
    }
    sh[2 * threadIdx.x] = rr[0];
    sh[2 * threadIdx.x + 1] = rr[1];
    __syncthreads();
    if ((int)threadIdx.x < Rs) {  // column c: its rows' threads in order
        double s = 0.0;
        for (int w = 0; w < P.rpb; w++) s += sh[w * Rs + threadIdx.x];
        part_rr[(int64_t)blockIdx.x * Rs + threadIdx.x] = s;
    }
}

__global__ void __launch_bounds__(kBlock) k_m_pupdate(int n, int R, int Rs, double* p, const double* __restrict__ z,
                                                       float* p32, int first, const MultiState* st,
                                                       const int* active) {
    pdl_entry();
    if (*active == 0) return;
    const PairLayout P = pair_layout(Rs);
    if (!P.in) return;
    double beta[2];
    bool on[2];
#pragma unroll
    for (int j = 0; j < 2; j++) {
        on[j] = P.c + j < R && !st[P.c + j].done;
        beta[j] = on[j] && !first ? st[P.c + j].beta : 0.0;
    }
    if (!on[0] && !on[1]) return;
    for (int64_t i = (int64_t)blockIdx.x * P.rpb + P.rl; i < n; i += (int64_t)gridDim.x * P.rpb) {
        const int64_t e = i * Rs + P.c;
        double zv[2], pv[2];
        load_vec<2>(z + e, zv);
        load_vec<2>(p + e, pv);
#pragma unroll
        for (int j = 0; j < 2; j++) {
            if (!on[j]) continue;
            const double pi = first ? zv[j] : fma(beta[j], pv[j], zv[j]);
            p[e + j] = pi;
            if (p32) p32[e + j] = __double2float_rn(pi);
        }
    }
}

// --------------------------------------------------- kernels, batch of systems
// A block per tile: rows [row0, row1) of one system.
#define BATCH_TILE(T)                                       \
    const int4 tile = (T)[blockIdx.x]; /* system, row0, row1 */ \
    const int sys = tile.x, row0 = tile.y, row1 = tile.z;

// tile partials of a.b and (c given) c.d; which: systems not done, or those
// whose residual replacement is due
__global__ void __launch_bounds__(kBlock) k_b_dots(const int4* __restrict__ tiles, const double* __restrict__ a,
                                                    const double* __restrict__ b, const double* __restrict__ c,
                                                    const double* __restrict__ d, double* part0, double* part1,
                                                    int all, int due, const MultiState* st, const int* active) {
    pdl_entry();
    if (!all && *active == 0) return;
    BATCH_TILE(tiles)
    if (!all && (st[sys].done || (due && !st[sys].replace_now))) return;
    __shared__ double sh[kWarpsPerBlock];
    double s0 = 0.0, s1 = 0.0;
    for (int i = row0 + threadIdx.x; i < row1; i += kBlock) {
        s0 = fma(a[i], b[i], s0);
        if (c) s1 = fma(c[i], d[i], s1);
    }
    block_partial(s0, sh, part0 + blockIdx.x);
    if (c) block_partial(s1, sh, part1 + blockIdx.x);
}

template <typename X0>
__global__ void __launch_bounds__(kBlock) k_b_update(const int4* __restrict__ tiles, double* x, double* r,
                                                      const double* __restrict__ p, const double* __restrict__ q,
                                                      const X0* __restrict__ invd, X0* x0, double* part_rr,
                                                      const MultiState* st, const int* active) {
    pdl_entry();
    if (*active == 0) return;
    BATCH_TILE(tiles)
    if (st[sys].done) return;
    __shared__ double sh[kWarpsPerBlock];
    const double alpha = st[sys].alpha;
    double rr = 0.0;
    for (int i = row0 + threadIdx.x; i < row1; i += kBlock) {
        x[i] = fma(alpha, p[i], x[i]);
        const double ri = fma(-alpha, q[i], r[i]);
        r[i] = ri;
        if (x0) x0[i] = (X0)ri * invd[i];
        rr = fma(ri, ri, rr);
    }
    block_partial(rr, sh, part_rr + blockIdx.x);
}

__global__ void __launch_bounds__(kBlock) k_b_pupdate(const int4* __restrict__ tiles, double* p,
                                                       const double* __restrict__ z, float* p32, int first,
                                                       const MultiState* st, const int* active) {
    pdl_entry();
    if (*active == 0) return;
    BATCH_TILE(tiles)
    if (st[sys].done) return;
    const double beta = st[sys].beta;
    for (int i = row0 + threadIdx.x; i < row1; i += kBlock) {
        const double pi = first ? z[i] : fma(beta, p[i], z[i]);
        p[i] = pi;
        if (p32) p32[i] = __double2float_rn(pi);
    }
}

// FP64 residual r = F - K x, x0 = r / d, of every system or (gate) of those
// whose replacement is due; row groups without such a row are skipped.
template <typename X0>
__global__ void __launch_bounds__(kBlock) k_b_residual(int n, CsrM<double> mat, const double* __restrict__ x,
                                                        const double* __restrict__ F, const X0* __restrict__ invd,
                                                        double* r, X0* x0, const MultiState* st,
                                                        const int32_t* __restrict__ seg, const unsigned* gate) {
    pdl_entry();
    if (gate && *gate == 0) return;
    constexpr int RPW = 32;
    ROWGROUP_PROLOGUE(double)
    bool mine = owner;
    if (gate) {
        if (owner) {
            const MultiState& m = st[seg[myrow]];
            mine = !m.done && m.replace_now;
        }
        if (!__any_sync(FULL, mine)) return;
    }
    const double s = group_rows<RPW, double>(mat, x, row0, n, lane, tiles[wid]);
    if (mine) {
        const double ri = F[myrow] - s;
        r[myrow] = ri;
        if (x0) x0[myrow] = (X0)ri * invd[myrow];
    }
}

// ------------------------------------------------------------------ scalars
// Partial sums of one dot product per system: right-hand sides have nb block
// partials of Rs columns each; a batch's system s has the tiles
// [tile0[s], tile0[s + 1]).
struct Parts {
    int nb, Rs;
    const int* tile0;
};

// Scalar kernels: a warp per system, kScalSys systems per block.  An FP64
// instruction of a warp holds a quarter of an SM's pipe for 64 cycles: 304
// partials of 16 columns in one block are 2.4 us of adds, on four SMs a quarter.
// Measured, 16 right-hand sides: alpha 11.1 -> 8.1 us, beta 11.3 -> 8.4, the
// convergence test 7.6 -> 6.9; a batch of 24: 6.1 -> 5.1, 6.4 -> 5.9, 4.9 -> 5.0.
constexpr int kScalSys = 4;

// Sum of system s's partials on every lane of the warp, in a fixed order.
__device__ __forceinline__ double sum_system(const Parts& P, int s, const double* __restrict__ part, int lane) {
    const int k0 = P.tile0 ? P.tile0[s] : 0, k1 = P.tile0 ? P.tile0[s + 1] : P.nb;
    const int64_t step = P.tile0 ? 1 : P.Rs;
    const double* __restrict__ p = P.tile0 ? part : part + s;
    double t = 0.0;
#pragma unroll 8
    for (int k = k0 + lane; k < k1; k += 32) t += p[k * step];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(FULL, t, o);
    return t;
}

#define SCAL_SYSTEM                    \
    const int lane = threadIdx.x & 31; \
    const int s = blockIdx.x * kScalSys + ((int)threadIdx.x >> 5);

// In the block that gets here last: *active = number of systems not done (0 as
// well once the single-system state, which the batch's V-cycle kernels read,
// says stop).  `ticket` is zero again afterwards.
__device__ void count_active(int S, const MultiState* st, int* active, unsigned* ticket, SolveState* single,
                             unsigned* clear = nullptr) {
    __shared__ int cnt;
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        if (last) *ticket = 0;
        __threadfence();
        cnt = 0;
    }
    __syncthreads();
    if (!last) return;
    for (int k = threadIdx.x; k < S; k += blockDim.x)
        if (!__ldcg(&st[k].done)) atomicAdd(&cnt, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        const int a = __ldcg(&single->done) ? 0 : cnt;
        *active = a;
        if (a == 0) single->done = 1;
        if (clear) *clear = 0;
    }
}

// all systems' squared norms of the start residual and of F
__global__ void __launch_bounds__(kScalSys * 32) k_m_scal_init(Parts P, int S, const double* part_rr,
                                                               const double* part_ff, double rtol, int itmax,
                                                               int repl, MultiState* st, int* active, int* itmax_out,
                                                               unsigned* due, SolveState* single) {
    pdl_entry();
    SCAL_SYSTEM
    const double rr = s < S ? sum_system(P, s, part_rr, lane) : 0.0, ff = s < S ? sum_system(P, s, part_ff, lane) : 0.0;
    if (s < S && lane == 0) {
        MultiState& m = st[s];
        const double nF = sqrt(ff), nr = sqrt(rr);
        m.nF = nF;
        m.tol = rtol * nF;
        m.nr = nr;
        m.iters = 0;
        m.status = AMG_OK;
        m.done = 0;
        m.replace_now = 0;
        if (isnan(nr) || isnan(nF) || isinf(nr) || isinf(nF)) {
            m.status = AMG_ERR_NAN;
            m.done = 1;
        } else if (!(nF > 0.0) || nr <= m.tol) {
            m.done = 1;
        } else if (itmax <= 0) {
            m.status = AMG_ERR_NOT_CONVERGED;
            m.done = 1;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        itmax_out[0] = itmax;
        itmax_out[1] = repl;
        due[0] = 0;
        single->done = 0;
        single->status = AMG_OK;
    }
    count_active(S, st, active, due + 1, single);
}

__global__ void __launch_bounds__(kScalSys * 32) k_m_scal_alpha(Parts P, int S, const double* part_pq,
                                                                const double* part_pr, int flexible, MultiState* st,
                                                                int* active, unsigned* due, SolveState* single) {
    pdl_entry();
    if (*active == 0) return;
    SCAL_SYSTEM
    if (s < S && !st[s].done) {
        const double pq = sum_system(P, s, part_pq, lane);
        const double num = flexible ? sum_system(P, s, part_pr, lane) : st[s].rho;
        if (lane == 0) {
            MultiState& m = st[s];
            m.pq = pq;
            if (!(pq > 0.0)) {
                m.status = (isnan(pq) || isnan(num)) ? AMG_ERR_NAN : AMG_ERR_BREAKDOWN;
                m.done = 1;
            } else {
                m.alpha = num / pq;
            }
        }
    }
    count_active(S, st, active, due + 1, single);
}

// *due: the right-hand sides (bit s) whose FP64 residual replacement is due;
// nonzero for a batch when any system's is (zero before).
__global__ void __launch_bounds__(kScalSys * 32) k_m_scal_conv(Parts P, int S, const double* part_rr, int mixed,
                                                               const int* params, MultiState* st, int* active,
                                                               unsigned* due, SolveState* single) {
    pdl_entry();
    if (*active == 0) return;
    SCAL_SYSTEM
    if (s < S && !st[s].done) {
        const double rr = sum_system(P, s, part_rr, lane);
        if (lane == 0) {
            MultiState& m = st[s];
            const int itmax = params[0], repl = params[1];
            const double nr = sqrt(rr);
            const int it = m.iters + 1;
            m.iters = it;
            m.nr = nr;
            if (isnan(nr) || isinf(nr)) {
                m.status = AMG_ERR_NAN;
                m.done = 1;
            } else if (mixed && (nr <= m.tol || it >= itmax || (repl > 0 && it % repl == 0))) {
                m.replace_now = 1;
                atomicOr(due, 1u << (s & 31));
            } else if (nr <= m.tol) {
                m.done = 1;
            } else if (it >= itmax) {
                m.status = AMG_ERR_NOT_CONVERGED;
                m.done = 1;
            }
        }
    }
    count_active(S, st, active, due + 1, single);
}

__global__ void __launch_bounds__(kScalSys * 32) k_m_scal_replaced(Parts P, int S, const double* part_rr,
                                                                   const int* params, MultiState* st, int* active,
                                                                   unsigned* due, SolveState* single) {
    pdl_entry();
    if (*active == 0 || *due == 0) return;
    SCAL_SYSTEM
    if (s < S && !st[s].done && st[s].replace_now) {
        const double rr = sum_system(P, s, part_rr, lane);
        if (lane == 0) {
            MultiState& m = st[s];
            const double nr = sqrt(rr);
            m.nr = nr;
            m.replace_now = 0;
            if (isnan(nr) || isinf(nr)) {
                m.status = AMG_ERR_NAN;
                m.done = 1;
            } else if (nr <= m.tol) {
                m.done = 1;
            } else if (m.iters >= params[0]) {
                m.status = AMG_ERR_NOT_CONVERGED;
                m.done = 1;
            }
        }
    }
    count_active(S, st, active, due + 1, single, due);
}

__global__ void __launch_bounds__(kScalSys * 32) k_m_scal_beta(Parts P, int S, const double* part_rz,
                                                               const double* part_zq, int flexible, int first,
                                                               MultiState* st, int* active, unsigned* due,
                                                               SolveState* single) {
    pdl_entry();
    if (*active == 0) return;
    SCAL_SYSTEM
    const bool flex = flexible && !first;
    if (s < S && !st[s].done) {
        const double rz = sum_system(P, s, part_rz, lane);
        const double zq = flex ? sum_system(P, s, part_zq, lane) : 0.0;
        if (lane == 0) {
            MultiState& m = st[s];
            if (isnan(rz) || isnan(zq)) {
                m.status = AMG_ERR_NAN;
                m.done = 1;
            } else {
                m.beta = first ? 0.0 : (flexible ? -zq / m.pq : rz / m.rho);
                m.rho = rz;
            }
        }
    }
    count_active(S, st, active, due + 1, single);
}

// dots[2 s], dots[2 s + 1] = the systems' sums (the final residual norms)
__global__ void __launch_bounds__(kScalSys * 32) k_m_totals(Parts P, int S, const double* part0, const double* part1,
                                                            double* dots) {
    pdl_entry();
    SCAL_SYSTEM
    if (s >= S) return;
    const double t0 = sum_system(P, s, part0, lane), t1 = sum_system(P, s, part1, lane);
    if (lane == 0) {
        dots[2 * s] = t0;
        dots[2 * s + 1] = t1;
    }
}

// [N][Rs] <-> column-major (leading dimension ld) copies; the padding
// columns become zero
__global__ void k_interleave(int n, int R, int Rs, int64_t ld, const double* __restrict__ src, double* dst) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= (int64_t)n * Rs) return;
    const int i = (int)(g / Rs), c = (int)(g % Rs);
    dst[g] = c < R ? src[(int64_t)c * ld + i] : 0.0;
}

__global__ void k_deinterleave(int n, int R, int Rs, int64_t ld, const double* __restrict__ src, double* dst) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= (int64_t)n * R) return;
    const int i = (int)(g % n), c = (int)(g / n);
    dst[(int64_t)c * ld + i] = src[(int64_t)i * Rs + c];
}

// ----------------------------------------------------------------- host side
inline int scal_blocks(int S) { return (S + kScalSys - 1) / kScalSys; }
inline int elem_blocks(int64_t count) { return (int)((count + 255) / 256 > 0 ? (count + 255) / 256 : 1); }

template <typename A>
struct MView;

template <>
struct MView<double> {
    static double* f(MultiWork& w, int l) { return static_cast<double*>(w.lf[l]); }
    static double* x(MultiWork& w, int l) { return static_cast<double*>(w.lx[l]); }
    static double* t(MultiWork& w, int l) { return static_cast<double*>(w.lt[l]); }
    static const double* invd(Level& L) { return L.invd; }
    template <typename Fn>
    static void vals(Level& L, int, Fn&& fn) { fn(static_cast<const double*>(L.A.val)); }
};

template <>
struct MView<float> {
    static float* f(MultiWork& w, int l) { return static_cast<float*>(w.lf[l]); }
    static float* x(MultiWork& w, int l) { return static_cast<float*>(w.lx[l]); }
    static float* t(MultiWork& w, int l) { return static_cast<float*>(w.lt[l]); }
    static const float* invd(Level& L) { return L.invd32; }
    template <typename Fn>
    static void vals(Level& L, int l, Fn&& fn) {
        if (l == 0 && L.val16) fn(static_cast<const __nv_bfloat16*>(L.val16));
        else fn(static_cast<const float*>(L.val32));
    }
};

template <typename T>
using vt = std::remove_cv_t<std::remove_pointer_t<T>>;

template <typename V>
MatM<V> mat_of(const Level& L, const V* v) {
    return MatM<V>{L.A.rowptr, L.A.col, v, L.run_ptr, L.run_len, L.run_start};
}

enum { M_A = 0, M_B, M_SLOTS };  // partial-sum slots (two dot products at a time)
double* mslot(MultiWork& w, int k) { return w.part + (int64_t)k * w.part_stride; }

// lanes per entry: 16 bytes of the Rs columns each, a power of two
template <typename A>
int lanes_per_entry(int Rs) {
    const int q = Rs / kVec<A>;
    int p = 1;
    while (p < q) p <<= 1;
    return p;
}
// on a level: two where one would do (two FP64 columns) and the rows are short (at
// most kPairRow entries on average), since 32 groups have more to add up than such
// a row gives them.  Us per iteration with one / two: 2-D p = 3 n = 101 (49 entries)
// 104 / 102, 3-D p = 2 n = 12 (90) 57 / 59, p = 3 n = 24 (284) 168 / 221.
constexpr int kPairRow = 64;
template <typename A>
int lanes_per_entry(int Rs, const Level& L) {
    const int p = lanes_per_entry<A>(Rs);
    return p == 1 && sizeof(A) == 8 && L.A.nnz <= (int64_t)kPairRow * L.A.n ? 2 : p;
}

// Rows of a block that share one epilogue: all copies of a column where the
// level has rows enough to fill the GPU's warps that way, else one.
template <typename A>
int rows_together(amg_hierarchy* h, const Level& L, int Rs) {
    const int t = 32 / (kVec<A> * lanes_per_entry<A>(Rs, L));
    return (int64_t)L.A.n >= (int64_t)h->num_sms * 16 * t ? t : 1;
}

// blocks of the SpMM kernels: two per SM (the partial sums of a dot product
// are one per block, and their sum is FP64 work of one SM)
int spmm_blocks(amg_hierarchy* h, int n) {
    const int64_t b = ((int64_t)n + kWarpsPerBlock - 1) / kWarpsPerBlock;
    const int64_t cap = (int64_t)h->num_sms * 2;
    return (int)(b < cap ? b : cap);
}
int coarse_blocks(amg_hierarchy* h) {
    const int cap = h->num_sms * 2;
    return h->ndense < cap ? h->ndense : cap;
}

// blocks of the vector kernels of R right-hand sides
int pair_blocks(amg_hierarchy* h, int n, int Rs) {
    const int rpb = pair_rows(Rs);
    const int64_t b = ((int64_t)n + rpb - 1) / rpb;
    const int64_t cap = (int64_t)h->num_sms * 2;
    return (int)(b < cap ? b : cap);
}

// fn(true) where the finest level has run-encoded columns and the products
// are FP32, else fn(false): in FP64 the pass is bound by the FP64 pipe, and
// taking four rows at once only costs warps in flight (3-D p = 3 n = 24, 16
// right-hand sides: 135 ms a solve against 76 ms row by row).
template <typename A, typename Fn>
void with_runs(const Level& L, Fn&& fn) {
    if constexpr (std::is_same_v<A, float>) {
        if (L.run_ptr) {
            fn(std::true_type{});
            return;
        }
    }
    fn(std::false_type{});
}

template <typename A>
cudaError_t m_vcycle(amg_hierarchy* h, cudaStream_t s) {
    using Vw = MView<A>;
    MultiWork& w = *h->mw;
    const int L = h->nlev, Rs = w.Rs, flex = h->o.flexible;
    const int* act = w.active;
    if (L == 1) {
        launch_pdl(k_m_coarse<double, A>, coarse_blocks(h), kCoarseWarps * 32, 0, s, h->ndense, Rs,
                   lanes_per_entry<double>(Rs), h->Ainv, w.r, nullptr, nullptr, nullptr, nullptr, w.z, w.q,
                   mslot(w, M_A), mslot(w, M_B), flex, act);
        return cudaGetLastError();
    }
    for (int l = 0; l < L - 1; l++) {
        Level& F = h->lev[l];
        Level& C = h->lev[l + 1];
        const int n = F.A.n, nb = spmm_blocks(h, n), T = rows_together<A>(h, F, Rs), lp = lanes_per_entry<A>(Rs, F);
        const bool coarsest = (l + 1 == L - 1);
        A* xc = coarsest ? nullptr : Vw::x(w, l + 1);
        if (l > 0 && n <= nb * kWarpsPerBlock) {  // a warp for every row
            Vw::vals(F, l, [&](auto vp) {
                using V = vt<decltype(vp)>;
                const int rows = std::max(1, kWarpsPerBlock >> F.npass);
                launch_pdl(k_m_resid_restrict<A, V>, std::max(1, std::min(2 * h->num_sms, (C.A.n + rows - 1) / rows)), kBlock, 0, s,
                           C.A.n, rows, Rs, lp, mat_of(F, vp), static_cast<const A*>(Vw::f(w, l)),
                           static_cast<const A*>(Vw::x(w, l)), F.mem_ptr, F.mem_idx, F.pval, Vw::f(w, l + 1), xc,
                           Vw::invd(C), act);
            });
            continue;
        }
        Vw::vals(F, l, [&](auto vp) {
            using V = vt<decltype(vp)>;
            if (l == 0)
                with_runs<A>(F, [&](auto rn) {
                    launch_pdl(k_m_resid<decltype(rn)::value, A, V, double>, nb, kBlock, 0, s, n, Rs, lp, T, mat_of(F, vp), w.r,
                               Vw::x(w, 0), Vw::t(w, 0), act);
                });
            else
                launch_pdl(k_m_resid<false, A, V, A>, nb, kBlock, 0, s, n, Rs, lp, T, mat_of(F, vp), Vw::f(w, l),
                           Vw::x(w, l), Vw::t(w, l), act);
        });
        launch_pdl(k_m_restrict<A>, elem_blocks((int64_t)C.A.n * Rs), 256, 0, s, C.A.n, Rs, F.mem_ptr, F.mem_idx,
                   F.pval, Vw::t(w, l), Vw::f(w, l + 1), xc, Vw::invd(C), act);
    }
    {
        Level& F = h->lev[L - 2];
        Level& C = h->lev[L - 1];
        launch_pdl(k_m_coarse<A, A>, coarse_blocks(h), kCoarseWarps * 32, 0, s, C.A.n, Rs, lanes_per_entry<double>(Rs),
                   h->Ainv, Vw::f(w, L - 1), F.mem_ptr, F.mem_idx, F.pval, Vw::x(w, L - 2), nullptr, nullptr, nullptr,
                   nullptr, 0, act);
    }
    for (int l = L - 2; l >= 0; l--) {
        Level& F = h->lev[l];
        const int n = F.A.n, nb = spmm_blocks(h, n), T = rows_together<A>(h, F, Rs), lp = lanes_per_entry<A>(Rs, F);
        Vw::vals(F, l, [&](auto vp) {
            using V = vt<decltype(vp)>;
            if (l == 0) {
                with_runs<A>(F, [&](auto rn) {
                    launch_pdl(k_m_up0<decltype(rn)::value, A, V>, nb, kBlock, 0, s, n, Rs, lp, T, mat_of(F, vp), w.r, Vw::x(w, 0),
                               Vw::invd(F), w.z, w.q, mslot(w, M_A), mslot(w, M_B), flex, act);
                });
            } else {
                Level& G = h->lev[l - 1];
                launch_pdl(k_m_up<A, V>, nb, kBlock, 0, s, n, Rs, lp, T, mat_of(F, vp), Vw::f(w, l),
                           Vw::x(w, l), Vw::invd(F), G.mem_ptr, G.mem_idx, G.pval, Vw::x(w, l - 1), act);
            }
        });
    }
    return cudaGetLastError();
}

// Block partials of the kernels: right-hand sides, from the SpMM kernels or
// (vec) from the vector kernels; a batch, from the tiles.
Parts spmm_parts(amg_hierarchy* h) { return Parts{spmm_blocks(h, h->lev[0].A.n), h->mw->Rs, nullptr}; }
Parts pair_parts(amg_hierarchy* h) {
    return Parts{pair_blocks(h, h->lev[0].A.n, h->mw->Rs), h->mw->Rs, nullptr};
}
Parts tile_parts(amg_hierarchy* h) { return Parts{0, 0, h->mw->tile0}; }

// z = B r; r.z and z.q into the two slots; returns where their partials are
cudaError_t any_vcycle(amg_hierarchy* h, Parts* P, cudaStream_t s) {
    MultiWork& w = *h->mw;
    const int flex = h->o.flexible;
    if (!w.tiles) {
        AMG_TRY(h->mixed ? m_vcycle<float>(h, s) : m_vcycle<double>(h, s));
        *P = h->nlev > 1 ? spmm_parts(h) : Parts{coarse_blocks(h), w.Rs, nullptr};
        return cudaSuccess;
    }
    AMG_TRY(enqueue_vcycle_rows(h, s));
    launch_pdl(k_b_dots, w.ntiles, kBlock, 0, s, w.tiles, w.r, w.z, flex ? w.z : nullptr, w.q, mslot(w, M_A),
               mslot(w, M_B), 0, 0, w.st, w.active);
    *P = tile_parts(h);
    return cudaGetLastError();
}

// r = F - K x, x0 = r / d; r.r (slot A) and, with ff, F.F (slot B).  due:
// only the systems whose replacement is due.
cudaError_t any_residual(amg_hierarchy* h, double* r, bool x0, bool ff, bool due, Parts* P, cudaStream_t s) {
    MultiWork& w = *h->mw;
    Level& L0 = h->lev[0];
    const int n = L0.A.n;
    const bool want = x0 && h->nlev > 1;
    const unsigned* gate = due ? w.due : nullptr;
    if (!w.tiles) {
        const int nb = spmm_blocks(h, n), lp = lanes_per_entry<double>(w.Rs, L0);
        const int T = rows_together<double>(h, L0, w.Rs);
        double* pff = ff ? mslot(w, M_B) : nullptr;
        const auto mat = mat_of(L0, static_cast<const double*>(L0.A.val));
        if (h->mixed)
            launch_pdl(k_m_residual<float>, nb, kBlock, 0, s, n, w.Rs, lp, T, mat, w.x, w.F, L0.invd32, r,
                       want ? static_cast<float*>(w.lx[0]) : nullptr, mslot(w, M_A), pff, gate);
        else
            launch_pdl(k_m_residual<double>, nb, kBlock, 0, s, n, w.Rs, lp, T, mat, w.x, w.F, L0.invd, r,
                       want ? static_cast<double*>(w.lx[0]) : nullptr, mslot(w, M_A), pff, gate);
        *P = spmm_parts(h);
        return cudaGetLastError();
    }
    // the FP64 matrix (also in mixed precision), a row per lane
    const CsrM<double> mat{L0.A.rowptr, L0.A.col, L0.A.val};
    const int nb = row_blocks(n, 32);
    if (h->mixed)
        launch_pdl(k_b_residual<float>, nb, kBlock, 0, s, n, mat, w.x, w.F, L0.invd32, r, want ? L0.x32 : nullptr,
                   w.st, w.seg, gate);
    else
        launch_pdl(k_b_residual<double>, nb, kBlock, 0, s, n, mat, w.x, w.F, L0.invd, r, want ? L0.x : nullptr, w.st,
                   w.seg, gate);
    launch_pdl(k_b_dots, w.ntiles, kBlock, 0, s, w.tiles, r, r, ff ? w.F : nullptr, w.F, mslot(w, M_A),
               mslot(w, M_B), due ? 0 : 1, due ? 1 : 0, w.st, w.active);
    *P = tile_parts(h);
    return cudaGetLastError();
}

void any_pupdate(amg_hierarchy* h, int first, cudaStream_t s) {
    MultiWork& w = *h->mw;
    float* p32 = h->mixed ? w.p32 : nullptr;
    if (w.tiles)
        launch_pdl(k_b_pupdate, w.ntiles, kBlock, 0, s, w.tiles, w.p, w.z, p32, first, w.st, w.active);
    else
        launch_pdl(k_m_pupdate, pair_blocks(h, h->lev[0].A.n, w.Rs), kBlock, 0, s, h->lev[0].A.n, w.R, w.Rs, w.p,
                   w.z, p32, first, w.st, w.active);
}

// q = K p with p.q (slot A) and, flexible, p.r (slot B)
cudaError_t any_spmv_pq(amg_hierarchy* h, Parts* P, cudaStream_t s) {
    MultiWork& w = *h->mw;
    Level& L0 = h->lev[0];
    const int n = L0.A.n, flex = h->o.flexible;
    if (w.tiles) {
        AMG_TRY(launch_rowgroup_pq(h, s, true));
        launch_pdl(k_b_dots, w.ntiles, kBlock, 0, s, w.tiles, w.p, w.q, flex ? w.p : nullptr, w.r, mslot(w, M_A),
                   mslot(w, M_B), 0, 0, w.st, w.active);
        *P = tile_parts(h);
        return cudaGetLastError();
    }
    const int nb = spmm_blocks(h, n);
    if (h->mixed)
        with_runs<float>(L0, [&](auto rn) {
            launch_pdl(k_m_spmv_pq<decltype(rn)::value, float, float>, nb, kBlock, 0, s, n, w.Rs,
                       lanes_per_entry<float>(w.Rs, L0), rows_together<float>(h, L0, w.Rs),
                       mat_of(L0, static_cast<const float*>(L0.val32)), w.p32, w.p, w.r, w.q, mslot(w, M_A),
                       mslot(w, M_B), flex, w.active);
        });
    else
        launch_pdl(k_m_spmv_pq<false, double, double>, nb, kBlock, 0, s, n, w.Rs, lanes_per_entry<double>(w.Rs, L0),
                   rows_together<double>(h, L0, w.Rs), mat_of(L0, static_cast<const double*>(L0.A.val)), w.p, w.p,
                   w.r, w.q, mslot(w, M_A), mslot(w, M_B), flex, w.active);
    *P = spmm_parts(h);
    return cudaGetLastError();
}

// x += alpha p, r -= alpha q, x0 = r / d, r.r (slot A)
cudaError_t any_update(amg_hierarchy* h, Parts* P, cudaStream_t s) {
    MultiWork& w = *h->mw;
    Level& L0 = h->lev[0];
    const bool x0 = h->nlev > 1;
    auto launch = [&](auto* invd, auto* xb, auto* xm) {
        using X0 = std::remove_pointer_t<decltype(xm)>;
        if (w.tiles)
            launch_pdl(k_b_update<X0>, w.ntiles, kBlock, 0, s, w.tiles, w.x, w.r, w.p, w.q, invd,
                       x0 ? xb : nullptr, mslot(w, M_A), w.st, w.active);
        else
            launch_pdl(k_m_update<X0>, pair_blocks(h, L0.A.n, w.Rs), kBlock, 0, s, L0.A.n, w.R, w.Rs, w.x, w.r, w.p,
                       w.q, invd, x0 ? xm : nullptr, mslot(w, M_A), w.st, w.active);
    };
    if (h->mixed) launch(static_cast<const float*>(L0.invd32), L0.x32, static_cast<float*>(w.lx[0]));
    else launch(static_cast<const double*>(L0.invd), L0.x, static_cast<double*>(w.lx[0]));
    *P = w.tiles ? tile_parts(h) : pair_parts(h);
    return cudaGetLastError();
}

}  // namespace

// Doubles of one partial-sum slot: the block partials of R interleaved
// right-hand sides, or one per tile.
size_t multi_part_stride(amg_hierarchy* h, int Rs, int ntiles) {
    if (ntiles > 0) return (size_t)ntiles;
    const size_t a = (size_t)spmm_blocks(h, h->lev[0].A.n), b = (size_t)pair_blocks(h, h->lev[0].A.n, Rs);
    const size_t c = (size_t)coarse_blocks(h);  // a single-level hierarchy
    return std::max(std::max(a, b), c) * Rs;
}
int multi_part_slots() { return M_SLOTS; }

cudaError_t enqueue_multi_start(amg_hierarchy* h, cudaStream_t s) {
    MultiWork& w = *h->mw;
    Parts P;
    AMG_TRY(any_residual(h, w.r, true, true, false, &P, s));
    launch_pdl(k_m_scal_init, scal_blocks(w.S), kScalSys * 32, 0, s, P, w.S, mslot(w, M_A), mslot(w, M_B), h->rtol, h->itmax,
               h->mixed ? h->o.resid_replace_every : 0, w.st, w.active, w.params, w.due, h->st);
    AMG_TRY(cudaGetLastError());
    AMG_TRY(any_vcycle(h, &P, s));
    launch_pdl(k_m_scal_beta, scal_blocks(w.S), kScalSys * 32, 0, s, P, w.S, mslot(w, M_A), mslot(w, M_B), h->o.flexible, 1, w.st,
               w.active, w.due, h->st);
    any_pupdate(h, 1, s);
    return cudaGetLastError();
}

cudaError_t enqueue_multi_iteration(amg_hierarchy* h, cudaStream_t s) {
    MultiWork& w = *h->mw;
    const int flex = h->o.flexible;
    Parts P;
    AMG_TRY(any_spmv_pq(h, &P, s));
    launch_pdl(k_m_scal_alpha, scal_blocks(w.S), kScalSys * 32, 0, s, P, w.S, mslot(w, M_A), mslot(w, M_B), flex, w.st, w.active,
               w.due, h->st);
    AMG_TRY(any_update(h, &P, s));
    launch_pdl(k_m_scal_conv, scal_blocks(w.S), kScalSys * 32, 0, s, P, w.S, mslot(w, M_A), h->mixed, w.params, w.st, w.active,
               w.due, h->st);
    if (h->mixed) {  // FP64 true-residual replacement, when due
        AMG_TRY(any_residual(h, w.r, true, false, true, &P, s));
        launch_pdl(k_m_scal_replaced, scal_blocks(w.S), kScalSys * 32, 0, s, P, w.S, mslot(w, M_A), w.params, w.st, w.active, w.due,
                   h->st);
    }
    AMG_TRY(cudaGetLastError());
    AMG_TRY(any_vcycle(h, &P, s));
    launch_pdl(k_m_scal_beta, scal_blocks(w.S), kScalSys * 32, 0, s, P, w.S, mslot(w, M_A), mslot(w, M_B), flex, 0, w.st, w.active,
               w.due, h->st);
    any_pupdate(h, 0, s);
    return cudaGetLastError();
}

// ||F_s - K x_s||^2 and ||F_s||^2 per system into dots[2 s], dots[2 s + 1].
cudaError_t enqueue_multi_final(amg_hierarchy* h, cudaStream_t s) {
    MultiWork& w = *h->mw;
    Parts P;
    AMG_TRY(any_residual(h, w.q, false, true, false, &P, s));
    launch_pdl(k_m_totals, scal_blocks(w.S), kScalSys * 32, 0, s, P, w.S, mslot(w, M_A), mslot(w, M_B), w.dots);
    return cudaGetLastError();
}

cudaError_t launch_interleave(int n, int R, int Rs, int64_t ld, const double* src, double* dst, cudaStream_t s) {
    k_interleave<<<AMG_GRID(elem_blocks((int64_t)n * Rs)), 256, 0, s>>>(n, R, Rs, ld, src, dst);
    return cudaGetLastError();
}

cudaError_t launch_deinterleave(int n, int R, int Rs, int64_t ld, const double* src, double* dst, cudaStream_t s) {
    k_deinterleave<<<AMG_GRID(elem_blocks((int64_t)n * R)), 256, 0, s>>>(n, R, Rs, ld, src, dst);
    return cudaGetLastError();
}

}  // namespace amg
