// The CG iteration of small systems as one kernel on one thread block cluster
// (arXiv 2511.21268, Sec. 3: CG with one V-cycle as preconditioner; FP64).
//
// A system of a few thousand rows is all latency: an iteration of the
// stream-ordered solve is a dozen dependent launches of 2.5 to 4 us each (41 us
// with its share of the fixed costs for the 1,024 rows of 2-D p = 2 n = 32; here
// 29), with a few hundred nanoseconds of arithmetic in each.  Here the blocks of
// one cluster split the rows of every level and keep them for the whole solve: a
// block owns a range of the coarsest rows, and on every finer level the members of its rows.  What only
// the owner of a row touches -- matrix rows, diagonals, right-hand sides,
// residuals, the CG vectors -- stays in the block's shared memory, restriction
// and prolongation are local, and only the vectors that other blocks gather
// (p, each level's x, the coarsest right-hand side) go through global memory.
// Phases, separated by the cluster's hardware barrier:
//   q = K p, p.q | x, r, x0 = r / d, r.r | per level: residual, restriction |
//   coarsest solve, prolongation | per level: smoothing, prolongation | z, r.z,
//   p = z + beta p |
// 3 + 2 (L - 1) + 1 barriers per iteration for L levels.  A phase costs the
// barrier, one gather through L2 and the row's chain of FP64 operations (an
// FP64 instruction holds a quarter of an SM's pipe for 64 cycles).
//
// Dot products: every row's term goes to shared memory, four warps add them,
// the blocks' sums are exchanged through distributed shared memory and added
// by every block in the same order: the blocks agree on every scalar without
// another exchange, and results are reproducible.
//
// Memory: what one block writes and others read afterwards is separated by
// barrier.cluster arrive.release / wait.acquire, and read with ordinary loads
// (never through the read-only path).  Every wait is a hardware barrier of the
// cluster, whose blocks run together; a launch does a bounded number of
// iterations.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "amg_internal.cuh"

namespace amg {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kClThreads = 512;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClMax = 16;    // blocks of the cluster, at most
constexpr int kClLevels = 8;  // levels, at most
constexpr int kClIters = 64;  // iterations of one launch
constexpr int kClStatic = 4096;  // static shared memory and slack
constexpr int64_t kClusterNnz = 200000;  // entries of all levels, at most
constexpr int64_t kClusterRows = 6000;   // rows of all levels and what counts as rows, at most:
constexpr int64_t kClusterDense = 100;   //   products of the coarsest inverse per row
constexpr int64_t kClusterLongest = 9;   //   rows per entry of the longest row

struct ClLevel {
    int n;
    const int64_t* rp;
    const int32_t* ci;
    const double* v;
    const double* invd;
    double *f, *x;
    const int32_t *mptr, *midx;  // members of the next level's rows
    const double* pval;
};

struct ClArgs {
    ClLevel lev[kClLevels];
    int L;  // levels
    int cap;  // dynamic shared memory bytes
    const double* Ainv;
    double *x, *r, *p;
    const double* F;
    SolveState* st;
    double* hist;
    int hist_cap;
    double rtol;
    int itmax, flexible, start;
};

// A block's rows of one level, in shared memory.
struct ClRows {
    int cnt;
    int* row;      // global row
    int* off;      // [cnt + 1] entries
    int* col;
    double* val;
    double* invd;
    double* pv;    // prolongator value to the next level
    int* mo;       // [rows of the next level + 1]: positions of their members here
    double *f, *x, *t;
};

struct ClShared {
    ClRows lv[kClLevels];
    double red[2][4];
    double parts[2][2][kClMax];  // [exchange parity][sum][block]
    int fit[kClMax];
    double sum[2];
    double alpha, beta, rho, pq, nF, tol;
    int done, iters, status, used, ok;
};

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t remote_addr(const void* p, uint32_t block) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(r)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(block));
    return r;
}

// `count` T in the dynamic shared memory (all threads; NULL and sh.ok = 0 when
// it does not fit).  A block barrier separates it from earlier allocations.
template <typename T>
__device__ __forceinline__ T* take(ClShared& sh, unsigned char* dyn, int cap, int count) {
    const int at = (sh.used + 7) & ~7;
    const int64_t end = (int64_t)at + (int64_t)count * (int)sizeof(T);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (end <= cap) sh.used = (int)end;
        else sh.ok = 0;
    }
    __syncthreads();
    return end <= cap ? reinterpret_cast<T*>(dyn + at) : nullptr;
}

// out[0 .. n] = exclusive sums of count(k), by warp 0
template <typename Fn>
__device__ __forceinline__ void scan_counts(int n, int* out, Fn&& count) {
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        int base = 0;
        for (int k0 = 0; k0 < n; k0 += 32) {
            const int c = k0 + lane < n ? count(k0 + lane) : 0;
            int s = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, s, o);
                if (lane >= o) s += y;
            }
            if (k0 + lane < n) out[k0 + lane] = base + s - c;
            base += __shfl_sync(FULL, s, 31);
        }
        if (lane == 0) out[n] = base;
    }
    __syncthreads();
}

// The block's rows of every level (sh.lv); sh.ok = 0 if they do not fit.
__device__ void load_rows(const ClArgs& a, ClShared& sh, unsigned char* dyn, uint32_t rank, uint32_t C) {
    const int tid = threadIdx.x, L = a.L;
    for (int l = L - 1; l >= 0 && sh.ok; l--) {
        const ClLevel& A = a.lev[l];
        ClRows R = {};
        if (l == L - 1) {
            const int I0 = (int)((int64_t)rank * A.n / C);
            R.cnt = (int)((int64_t)(rank + 1) * A.n / C) - I0;
            R.row = take<int>(sh, dyn, a.cap, R.cnt);
            if (!sh.ok) return;
            for (int k = tid; k < R.cnt; k += kClThreads) R.row[k] = I0 + k;
        } else {
            const ClRows& U = sh.lv[l + 1];
            R.mo = take<int>(sh, dyn, a.cap, U.cnt + 1);
            if (!sh.ok) return;
            scan_counts(U.cnt, R.mo, [&](int k) { return A.mptr[U.row[k] + 1] - A.mptr[U.row[k]]; });
            R.cnt = R.mo[U.cnt];
            R.row = take<int>(sh, dyn, a.cap, R.cnt);
            R.off = take<int>(sh, dyn, a.cap, R.cnt + 1);
            R.invd = take<double>(sh, dyn, a.cap, R.cnt);
            R.pv = take<double>(sh, dyn, a.cap, R.cnt);
            R.t = take<double>(sh, dyn, a.cap, R.cnt);
            R.x = take<double>(sh, dyn, a.cap, R.cnt);
            if (!sh.ok) return;
            for (int k = tid; k < U.cnt; k += kClThreads) {
                const int m = A.mptr[U.row[k]], o = R.mo[k];
                for (int j = 0; o + j < R.mo[k + 1]; j++) R.row[o + j] = A.midx[m + j];
            }
            __syncthreads();
            scan_counts(R.cnt, R.off, [&](int k) { return (int)(A.rp[R.row[k] + 1] - A.rp[R.row[k]]); });
            R.col = take<int>(sh, dyn, a.cap, R.off[R.cnt]);
            R.val = take<double>(sh, dyn, a.cap, R.off[R.cnt]);
            if (!sh.ok) return;
            for (int k = tid >> 5; k < R.cnt; k += kClWarps) {
                const int64_t b = A.rp[R.row[k]];
                const int o = R.off[k], len = R.off[k + 1] - o;
                for (int e = tid & 31; e < len; e += 32) {
                    R.col[o + e] = A.ci[b + e];
                    R.val[o + e] = A.v[b + e];
                }
            }
            for (int k = tid; k < R.cnt; k += kClThreads) {
                R.invd[k] = A.invd[R.row[k]];
                R.pv[k] = A.pval[R.row[k]];
            }
        }
        R.f = take<double>(sh, dyn, a.cap, R.cnt);
        if (!sh.ok) return;
        if (tid == 0) sh.lv[l] = R;
        __syncthreads();
    }
}

// e(k, sum, q, lpr) for every row k of the block: its sum over the gathered x,
// on the row's lpr lanes (q: the lane among them), eight entries per lane in
// flight.
template <int LPR, typename E>
__device__ __forceinline__ void rows_phase_t(const ClRows& R, const double* x, E&& e) {
    constexpr int G = 32 / LPR, U = 8;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, q = lane % LPR;
    for (int kb = wid * G; kb < R.cnt; kb += kClWarps * G) {
        const int k = kb + lane / LPR;
        const bool on = k < R.cnt;
        double acc = 0.0;
        if (on) {
            const int end = R.off[k + 1];
            for (int o = R.off[k] + q; o < end; o += U * LPR) {
                double xx[U];
#pragma unroll
                for (int u = 0; u < U; u++)
                    if (o + u * LPR < end) xx[u] = x[R.col[o + u * LPR]];
#pragma unroll
                for (int u = 0; u < U; u++)
                    if (o + u * LPR < end) acc = fma(R.val[o + u * LPR], xx[u], acc);
            }
        }
        __syncwarp();
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
        if (on) e(k, acc, q, LPR);
    }
}
// few rows: 8 lanes each, to use all the FP64 pipe; else 4, which takes fewer
// instructions per row
template <typename E>
__device__ __forceinline__ void rows_phase(const ClRows& R, const double* x, E&& e) {
    if (R.cnt <= 64) rows_phase_t<8>(R, x, e);
    else rows_phase_t<4>(R, x, e);
}

// Sums of t0[0 .. cnt) and (t1 given) t1[0 .. cnt) over the cluster, in sh.sum
// on every thread.  Holds a cluster barrier, which also orders the phase's
// global writes.
__device__ __forceinline__ void cluster_sums(ClShared& sh, const double* t0, const double* t1, int cnt, int& parity,
                                             uint32_t rank, uint32_t C) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int sums = t1 ? 2 : 1;
    __syncthreads();
    if (wid < 4 * sums) {
        const double* t = wid < 4 ? t0 : t1;
        double s = 0.0;
        for (int k = (wid & 3) * 32 + lane; k < cnt; k += 128) s += t[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        if (lane == 0) sh.red[wid >> 2][wid & 3] = s;
    }
    __syncthreads();
    if (wid < sums && lane < (int)C) {  // warp w sends sum w to every block
        const double* r = sh.red[wid];
        const double s = (r[0] + r[1]) + (r[2] + r[3]);
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote_addr(&sh.parts[parity][wid][rank], lane)), "d"(s)
                     : "memory");
    }
    __syncwarp();
    cluster_barrier();
    if (wid < sums) {
        double s = lane < (int)C ? sh.parts[parity][wid][lane] : 0.0;
#pragma unroll
        for (int o = kClMax / 2; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        if (lane == 0) sh.sum[wid] = s;
    }
    __syncthreads();
    parity ^= 1;
}

// x_l of the members of row k of level l + 1 (value y there) += P y
__device__ __forceinline__ void prolong_row(const ClLevel& A, const ClRows& R, int k, double y, int q, int lpr) {
    for (int m = R.mo[k] + q; m < R.mo[k + 1]; m += lpr) {
        const double xm = fma(R.pv[m], y, R.x[m]);
        R.x[m] = xm;
        A.x[R.row[m]] = xm;
    }
}

// The V-cycle from x_0 = r / d (R.x and global; the other blocks' are visible)
// to z (z[k] of the block's rows), with the terms r z and (q given) z q.
__device__ void cluster_vcycle(const ClArgs& a, ClShared& sh, const double* r, double* z, double* term0,
                               double* term1, const double* q) {
    const int L = a.L, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int l = 0; l < L - 1; l++) {
        const ClRows& R = sh.lv[l];
        const ClRows& U = sh.lv[l + 1];
        const ClLevel& B = a.lev[l + 1];
        const double* f = l == 0 ? r : R.f;
        if (l > 0) cluster_barrier();  // level 0: the caller's
        rows_phase(R, a.lev[l].x, [&](int k, double s, int ql, int) {
            if (ql == 0) R.t[k] = f[k] - s;
        });
        __syncthreads();
        const bool coarsest = l + 1 == L - 1;
        for (int k = tid; k < U.cnt; k += kClThreads) {
            double acc = 0.0;
            for (int m = R.mo[k]; m < R.mo[k + 1]; m++) acc = fma(R.pv[m], R.t[m], acc);
            U.f[k] = acc;
            if (coarsest) {
                B.f[U.row[k]] = acc;
            } else {
                const double x0 = acc * U.invd[k];
                U.x[k] = x0;
                B.x[U.row[k]] = x0;
            }
        }
    }
    cluster_barrier();
    {  // coarsest: a warp per row of the inverse
        const ClRows& U = sh.lv[L - 1];
        const double* f = a.lev[L - 1].f;
        const int nd = a.lev[L - 1].n;
        for (int k = wid; k < U.cnt; k += kClWarps) {
            const double* __restrict__ row = a.Ainv + (int64_t)U.row[k] * nd;
            double s = 0.0;
#pragma unroll 4
            for (int j = lane; j < nd; j += 32) s = fma(__ldg(row + j), f[j], s);
            __syncwarp();
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
            prolong_row(a.lev[L - 2], sh.lv[L - 2], k, s, lane, 32);
        }
    }
    for (int l = L - 2; l > 0; l--) {
        const ClRows& R = sh.lv[l];
        cluster_barrier();
        rows_phase(R, a.lev[l].x, [&](int k, double s, int ql, int lpr) {
            const double y = fma(R.invd[k], R.f[k] - s, R.x[k]);
            prolong_row(a.lev[l - 1], sh.lv[l - 1], k, y, ql, lpr);
        });
    }
    cluster_barrier();
    const ClRows& R = sh.lv[0];
    rows_phase(R, a.lev[0].x, [&](int k, double s, int ql, int) {
        if (ql != 0) return;
        const double za = fma(R.invd[k], r[k] - s, R.x[k]);
        z[k] = za;
        term0[k] = r[k] * za;
        if (q) term1[k] = za * q[k];
    });
}

__global__ void __launch_bounds__(kClThreads, 1) k_cluster_pcg(const __grid_constant__ ClArgs a) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ ClShared sh;
    uint32_t rank, C;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    const int tid = threadIdx.x;
    if (tid == 0) {
        sh.used = 0;
        sh.ok = 1;
        sh.done = a.start ? 0 : a.st->done;
        sh.iters = a.st->iters;
        sh.status = a.st->status;
        sh.rho = a.st->rho;
        sh.nF = a.st->nF;
        sh.tol = a.st->tol;
    }
    __syncthreads();
    load_rows(a, sh, dyn, rank, C);
    const int cnt = sh.ok ? sh.lv[0].cnt : 0;
    double *r = nullptr, *xs = nullptr, *ps = nullptr, *q = nullptr, *z = nullptr, *t0 = nullptr, *t1 = nullptr;
    if (sh.ok) {  // uniform in the block; take() clears it
        r = take<double>(sh, dyn, a.cap, cnt);
        xs = take<double>(sh, dyn, a.cap, cnt);
        ps = take<double>(sh, dyn, a.cap, cnt);
        q = take<double>(sh, dyn, a.cap, cnt);
        z = take<double>(sh, dyn, a.cap, cnt);
        t0 = take<double>(sh, dyn, a.cap, cnt);
        t1 = take<double>(sh, dyn, a.cap, cnt);
    }
    // every block has started (its shared memory may be written) and read the
    // state; then the blocks tell each other whether their rows fit
    cluster_barrier();
    if (tid < (int)C)
        asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(remote_addr(&sh.fit[rank], tid)), "r"(sh.ok) : "memory");
    __syncwarp();
    cluster_barrier();
    bool fit = true;
    for (uint32_t b = 0; b < C; b++) fit = fit && sh.fit[b];
    if (!fit) {
        if (rank == 0 && tid == 0) a.st->status = kClusterUnfit;
        return;
    }
    const ClRows& R = sh.lv[0];
    double* x0 = a.lev[0].x;
    const bool flex = a.flexible;
    int par = 0;
    for (int k = tid; k < cnt; k += kClThreads) {
        xs[k] = a.x[R.row[k]];
        if (!a.start) {
            r[k] = a.r[R.row[k]];
            ps[k] = a.p[R.row[k]];
        }
    }
    __syncthreads();
    if (a.start) {
        // r = F - K x, x0 = r / d, ||r||, ||F||
        rows_phase(R, a.x, [&](int k, double s, int ql, int) {
            if (ql != 0) return;
            const double fi = a.F[R.row[k]], ri = fi - s, xi = ri * R.invd[k];
            r[k] = ri;
            R.x[k] = xi;
            x0[R.row[k]] = xi;
            t0[k] = ri * ri;
            t1[k] = fi * fi;
        });
        cluster_sums(sh, t0, t1, cnt, par, rank, C);
        if (tid == 0) {
            const double nr = sqrt(sh.sum[0]), nF = sqrt(sh.sum[1]);
            sh.nF = nF;
            sh.tol = a.rtol * nF;
            sh.iters = 0;
            sh.status = AMG_OK;
            if (isnan(nr) || isnan(nF) || isinf(nr) || isinf(nF)) {
                sh.status = AMG_ERR_NAN;
                sh.done = 1;
            } else if (!(nF > 0.0) || nr <= sh.tol) {
                sh.done = 1;
            } else if (a.itmax <= 0) {
                sh.status = AMG_ERR_NOT_CONVERGED;
                sh.done = 1;
            }
            if (rank == 0) {
                a.st->nr = nr;
                if (a.hist) a.hist[0] = nF > 0.0 ? nr / nF : 0.0;
            }
        }
        __syncthreads();
        if (!sh.done) {
            cluster_vcycle(a, sh, r, z, t0, t1, nullptr);
            cluster_sums(sh, t0, nullptr, cnt, par, rank, C);
            if (tid == 0) {
                sh.rho = sh.sum[0];
                if (isnan(sh.rho)) {
                    sh.status = AMG_ERR_NAN;
                    sh.done = 1;
                }
            }
            for (int k = tid; k < cnt; k += kClThreads) {
                ps[k] = z[k];
                a.p[R.row[k]] = z[k];
            }
            __syncthreads();
        }
    }
    for (int it = 0; it < kClIters && !sh.done; it++) {
        cluster_barrier();  // p
        rows_phase(R, a.p, [&](int k, double s, int ql, int) {
            if (ql != 0) return;
            q[k] = s;
            t0[k] = ps[k] * s;
            if (flex) t1[k] = ps[k] * r[k];
        });
        cluster_sums(sh, t0, flex ? t1 : nullptr, cnt, par, rank, C);
        if (tid == 0) {
            const double pq = sh.sum[0], num = flex ? sh.sum[1] : sh.rho;
            sh.pq = pq;
            if (!(pq > 0.0)) {
                sh.status = (isnan(pq) || isnan(num)) ? AMG_ERR_NAN : AMG_ERR_BREAKDOWN;
                sh.done = 1;
            } else {
                sh.alpha = num / pq;
            }
        }
        __syncthreads();
        if (sh.done) break;
        const double alpha = sh.alpha;
        for (int k = tid; k < cnt; k += kClThreads) {
            xs[k] = fma(alpha, ps[k], xs[k]);
            const double ri = fma(-alpha, q[k], r[k]), xi = ri * R.invd[k];
            r[k] = ri;
            R.x[k] = xi;
            x0[R.row[k]] = xi;
            t0[k] = ri * ri;
        }
        cluster_sums(sh, t0, nullptr, cnt, par, rank, C);
        if (tid == 0) {
            const double nr = sqrt(sh.sum[0]);
            const int k = ++sh.iters;
            if (rank == 0) {
                a.st->nr = nr;
                if (a.hist && k < a.hist_cap) a.hist[k] = nr / sh.nF;
            }
            if (isnan(nr) || isinf(nr)) {
                sh.status = AMG_ERR_NAN;
                sh.done = 1;
            } else if (nr <= sh.tol) {
                sh.done = 1;
            } else if (k >= a.itmax) {
                sh.status = AMG_ERR_NOT_CONVERGED;
                sh.done = 1;
            }
        }
        __syncthreads();
        if (sh.done) break;
        cluster_vcycle(a, sh, r, z, t0, t1, flex ? q : nullptr);
        cluster_sums(sh, t0, flex ? t1 : nullptr, cnt, par, rank, C);
        if (tid == 0) {
            const double rz = sh.sum[0], zq = flex ? sh.sum[1] : 0.0;
            if (isnan(rz) || isnan(zq)) {
                sh.status = AMG_ERR_NAN;
                sh.done = 1;
            } else {
                sh.beta = flex ? -zq / sh.pq : rz / sh.rho;
                sh.rho = rz;
            }
        }
        __syncthreads();
        if (sh.done) break;
        const double beta = sh.beta;
        for (int k = tid; k < cnt; k += kClThreads) {
            const double pk = fma(beta, ps[k], z[k]);
            ps[k] = pk;
            a.p[R.row[k]] = pk;
        }
    }
    for (int k = tid; k < cnt; k += kClThreads) {
        a.x[R.row[k]] = xs[k];
        a.r[R.row[k]] = r[k];
    }
    if (rank == 0 && tid == 0) {
        SolveState* st = a.st;
        st->done = sh.done;
        st->iters = sh.iters;
        st->status = sh.status;
        st->rho = sh.rho;
        st->nF = sh.nF;
        st->tol = sh.tol;
        st->itmax = a.itmax;
        st->replace_now = 0;
        st->repl_every = 0;
    }
}

cudaError_t cluster_config(amg_hierarchy* h, int C, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at) {
    AMG_TRY(cudaFuncSetAttribute(k_cluster_pcg, cudaFuncAttributeMaxDynamicSharedMemorySize, h->cluster_smem));
    if (C > 8) AMG_TRY(cudaFuncSetAttribute(k_cluster_pcg, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cfg = {};
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = (size_t)h->cluster_smem;
    cfg.stream = h->s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaSuccess;
}

}  // namespace

// Blocks of the cluster solve, 0 where it does not apply: FP64, one l1-Jacobi
// sweep before and after, tentative prolongators, the dense coarsest solve,
// no kernel timing, and a system for which it is the faster solve.  (Whether the
// rows fit the blocks' shared memory the kernel finds out.)  What the blocks have
// to do per iteration is bounded by three lines.
// Entries of all levels, at most kClusterNnz: measured us per iteration of a whole
// solve to 1e-10, one cluster against the launches of the iteration graph, by
// entries of the finest level:
//   2-D: 27k (p = 3, n = 24) 21 / 32, 24k (p = 2, n = 32) 29 / 41, 76k (p = 3,
//   n = 40) 31 / 39, 55k (p = 2, n = 48) 34 / 41, 99k (p = 2, n = 64) 43 / 48,
//   185k (p = 4, n = 48) 42 / 40; 155k in 6,400 rows (p = 2, n = 80) do not fit
//   3-D: 39k (p = 2, n = 8) 22 / 52, 85k (p = 2, n = 10) 31 / 61, 133k (p = 3,
//   n = 8) 32 / 77, 157k (p = 2, n = 12) 38 / 60
// The line is where the 2-D systems break even (3-D systems, with fewer rows, would
// gain some way above it).
// Rows of all levels, plus the n^2 products of the coarsest inverse by
// kClusterDense, plus the longest row's entries by kClusterLongest, at most
// kClusterRows.  A row costs its share of the vector work and the reductions on 16
// SMs, the dense products run on 16 SMs that the launches spread over all, and the
// blocks of a phase wait for the longest row, which has 4 lanes.  Us per iteration,
// cluster / launches:
//   few entries per row (5,769 rows of all levels at n = 64): 5-point 32^2
//   23 / 34, 64^2 40 / 42, 80^2 50 / 45, 100^2 73 / 54; 7-point 16^3 41 / 42, 20^3
//   58 / 45; 3-point 2,000 32 / 39, 4,000 40 / 40, 6,000 55 / 50, 12,000 80 / 55
//   coarsest rows: 5-point 64^2 with 108 40 / 42, 356 38 / 36, 1,209 63 / 32;
//   2-D p = 2 n = 48 with 170 29 / 35, 619 34 / 30; 3-point 6,000 with 1,908 116 / 38
//   longest row: 5-point 50^2 (3,510 rows) with 153 entries 50 / 56, 293 62 / 61,
//   380 96 / 72, 695 101 / 81; 30^2 (1,240) with 440 41 / 52, 527 57 / 58; 2-D p = 2
//   n = 32 (1,370) with 281 42 / 46, 480 55 / 55, 576 63 / 58
// 16 blocks of 512 threads: 8 blocks took 1.05 times, 4 blocks 1.3 times as long, 256
// threads the same.
int cluster_solve_blocks(amg_hierarchy* h) {
    if (h->mixed || h->prof || h->o.nu_pre != 1 || h->o.nu_post != 1 || h->o.cheb_degree > 0 ||
        h->o.coarse_solver != 0 || h->nlev < 2 || h->nlev > kClLevels)
        return 0;
    if (h->cluster_blocks >= 0) return h->cluster_blocks;
    h->cluster_blocks = 0;
    int64_t nnz = 0, rows = (int64_t)h->ndense * h->ndense / kClusterDense, longest = 0;
    for (int l = 0; l < h->nlev; l++) {
        if (h->lev[l].smoothed) return 0;
        nnz += h->lev[l].A.nnz;
        rows += h->lev[l].A.n;
        if (l + 1 < h->nlev) longest = std::max<int64_t>(longest, h->lev[l].maxrow);
    }
    if (nnz > kClusterNnz || rows + kClusterLongest * longest > kClusterRows) return 0;
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    h->cluster_smem = optin - kClStatic;
    for (int C = kClMax; C >= 8; C >>= 1) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at[1];
        int fit = 0;
        if (cluster_config(h, C, cfg, at) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&fit, k_cluster_pcg, &cfg) != cudaSuccess || fit < 1) {
            cudaGetLastError();
            continue;
        }
        return h->cluster_blocks = C;
    }
    return 0;
}

// One launch: up to kClIters iterations (after the start phase if asked).
// Afterwards the state says done, more iterations wanted, or (status
// kClusterUnfit, nothing done) that the rows do not fit.
cudaError_t launch_cluster_pcg(amg_hierarchy* h, int start) {
    ClArgs a = {};
    a.L = h->nlev;
    a.cap = h->cluster_smem;
    for (int l = 0; l < h->nlev; l++) {
        const Level& L = h->lev[l];
        a.lev[l] = ClLevel{L.A.n, L.A.rowptr, L.A.col, L.A.val, L.invd, L.f, L.x, L.mem_ptr, L.mem_idx, L.pval};
    }
    a.Ainv = h->Ainv;
    a.x = h->x;
    a.r = h->r;
    a.p = h->p;
    a.F = h->F;
    a.st = h->st;
    a.hist = h->hist;
    a.hist_cap = h->hist_cap;
    a.rtol = h->rtol;
    a.itmax = h->itmax;
    a.flexible = h->o.flexible;
    a.start = start;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    AMG_TRY(cluster_config(h, h->cluster_blocks, cfg, at));
    note_launch();
    return cudaLaunchKernelEx(&cfg, k_cluster_pcg, a);
}

int cluster_solve_iters() { return kClIters; }

}  // namespace amg
