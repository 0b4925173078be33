// IgA assembly on the GPU by sum factorization (arXiv 2511.21268, Sec. 2.2).
//
// Stiffness entries of -div(kappa grad u) = f on one tensor-product B-spline
// patch, pulled back to the parametric cube and summed over the Gauss
// points q = (q1, q2, q3) of all elements:
//   k_ij = sum_q sum_{a,b} C_ab(q) d_a N_i(q) d_b N_j(q),
//   C = kappa(F(xi_q)) w_q |det J| J^-1 J^-T,        f_i = sum_q f w_q |det J| N_i(q),
// with N_i = b_i1(xi1) b_i2(xi2) b_i3(xi3) and d_a the parametric derivative
// in direction a.  Each term (a, b) factors into 1-D pair weights
//   W^{xy}_{i, delta}(q) = b^x_i(q) b^y_{i+delta}(q),   x, y in {value, derivative},
// one per direction, so the 3-D sum is contracted one direction at a time
// (sum factorization, the tensor-product alternative to the element loop
// that Sec. 2.2 points to):
//   A(r3, q2, q1) = sum_q3 W3(r3, q3) C(q3, q2, q1)
//   B(r3, r2, q1) = sum_q2 W2(r2, q2) A(r3, q2, q1)
//   K(r3, r2, r1) = sum_q1 W1(r1, q1) B(r3, r2, q1)
// with r_k = (i_k, delta_k) the 1-D pairs of the band |i_k - j_k| <= p.  The
// weight of a pair is nonzero on the Gauss points of the elements where both
// functions live, (p + 1 - |delta|) nq consecutive points, stored from the
// first of them.
//
// The geometries are extruded in xi3 (F_3 = xi3, F_1 and F_2 independent of
// xi3): J = [J2 0; 0 1], so C_02 = C_12 = 0 and C_22 = kappa w |det J2|.
// The five terms (0,0), (0,1), (1,0), (1,1), (2,2) have 1-D weight types
//   direction 3: vv vv vv vv dd;  direction 2: vv vd dv dd vv;
//   direction 1: dd dv vd vv vv,
// so after direction 3 there are four distinct arrays (C00, C01, C11 with
// vv; C22 with dd) and after direction 2 four groups by direction-1 type.
//
// K is symmetric and the direction-3 weights are symmetric in (i, j), so
// direction 3 takes only the pairs with delta_3 >= 0 (p + 1 of 2 p + 1), the
// other directions follow for those, and the last contraction stores each
// entry at (i, j) and at (j, i): 4/7 of the multiply-adds at p = 3, and K is
// symmetric in every bit.  n = 64, p = 3, annulus: the contractions of
// directions 3 and 2 6.47 -> 4.07 ms, the last one 6.27 -> 3.72 ms, the whole
// assembly 16.6 -> 11.8 ms.
//
// kappa = exp(g), g = sigma sqrt(2/M) sum_m cos(omega_m . x + phi_m) with
// x = (x(xi1, xi2), y(xi1, xi2), z(xi3)): cos(a + b) = cos a cos b - sin a sin b
// separates the plane and z parts, so g at all Q^3 points is the product of
// a Q^2 x 2M matrix [cos a, -sin a] and a 2M x Q matrix [cos b; sin b].  Its
// entries lie in [-1, 1], so it runs exactly enough in fixed point on the
// FP16 tensor cores (k_iga_coef_gemm below).
//
// Everything else is FP64.  The sums run in a different order than an element
// loop's, so results agree with one to rounding, not bit for bit.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <numeric>
#include <type_traits>
#include <vector>

#include "amg_gb300.h"
#include "amg_internal.cuh"

namespace amg {
namespace {

constexpr int kMaxDeg = 8;       // largest degree p
constexpr int kMaxNq = 16;       // most Gauss points per element and direction
constexpr int kMaxQ = 768;       // most Gauss points per direction (n nq): the contraction's staging
constexpr int kCtIn = 32;        // inner positions per block of the contractions
constexpr int kCtWarps = 8;      // warps per block of the contractions
constexpr int kInRows = 8;       // rows per block of the last contraction
constexpr int kGT = 64;          // GEMM tile (plane points x z points)
constexpr int kGK = 32;          // GEMM depth per stage
constexpr int kGStages = 3;      // stages in the copy ring
constexpr int kSlices = 8;       // fixed-point digits per GEMM operand
constexpr int kDigitBits = 7;
constexpr int kFixBits = 55;     // operands are rounded to multiples of 2^-55
constexpr int64_t kDigitBytes = 96LL << 20;  // digits of one piece of the plane
constexpr int kFlushK = 256;     // products between two flushes of the FP32 accumulators

struct IgaDims {
    int n, p, nq, m, off, Q, B, R, Lmax, R1, L1max;
};

__host__ __device__ inline double knot(int n, int p, int i) {
    return i <= p ? 0.0 : (i >= n + p ? 1.0 : (double)(i - p) / (double)n);
}

// Gauss-Legendre nodes and weights on [-1, 1], ascending: Newton's method on
// P_nq (three-term recurrence) from the starting guess cos(pi (k+3/4)/(nq+1/2)),
// w = 2 / ((1 - t^2) P_nq'(t)^2).
__global__ void k_iga_gauss(int nq, double* gx, double* gw) {
    const int k = threadIdx.x;
    if (k >= nq) return;
    const double pi = 3.14159265358979323846;
    double t = cos(pi * (k + 0.75) / (nq + 0.5)), pn = 0.0, dp = 1.0;
    for (int it = 0; it < 100; it++) {
        double p0 = 1.0, p1 = t;
        for (int j = 2; j <= nq; j++) {
            const double p2 = ((2 * j - 1) * t * p1 - (j - 1) * p0) / j;
            p0 = p1;
            p1 = p2;
        }
        pn = nq == 1 ? t : p1;
        const double pm = nq == 1 ? 1.0 : p0;
        dp = nq * (t * pn - pm) / (t * t - 1.0);
        const double dt = pn / dp;
        t -= dt;
        if (fabs(dt) < 1e-16) break;
    }
    {
        double p0 = 1.0, p1 = t;
        for (int j = 2; j <= nq; j++) {
            const double p2 = ((2 * j - 1) * t * p1 - (j - 1) * p0) / j;
            p0 = p1;
            p1 = p2;
        }
        pn = nq == 1 ? t : p1;
        dp = nq == 1 ? 1.0 : nq * (t * pn - p0) / (t * t - 1.0);
    }
    gx[nq - 1 - k] = t;
    gw[nq - 1 - k] = 2.0 / ((1.0 - t * t) * dp * dp);
}

// Values V[q][a] and derivatives D[q][a] of the p+1 B-splines e..e+p that
// live on element e = q / nq, at its Gauss point q % nq: the span recursion
// for the nonzero functions of a knot span (degree 0 -> p, each step mixing
// neighbours with the weights (xi - u_i) / (u_{i+k} - u_i)), and
// N'_{i,p} = p (N_{i,p-1} / (u_{i+p} - u_i) - N_{i+1,p-1} / (u_{i+p+1} - u_{i+1})).
__global__ void k_iga_basis(int n, int p, int nq, const double* __restrict__ gx, double* V, double* D) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n * nq) return;
    const int e = q / nq, s = e + p;
    const double xi = (e + 0.5 * (gx[q % nq] + 1.0)) / n;
    double N[kMaxDeg + 1], Np[kMaxDeg + 1], left[kMaxDeg + 1], right[kMaxDeg + 1];
    N[0] = 1.0;
    Np[0] = 1.0;
    for (int k = 1; k <= p; k++) {
        if (k == p)
            for (int a = 0; a < p; a++) Np[a] = N[a];
        left[k] = xi - knot(n, p, s + 1 - k);
        right[k] = knot(n, p, s + k) - xi;
        double saved = 0.0;
        for (int r = 0; r < k; r++) {
            const double tmp = N[r] / (right[r + 1] + left[k - r]);
            N[r] = saved + right[r + 1] * tmp;
            saved = left[k - r] * tmp;
        }
        N[k] = saved;
    }
    const int P1 = p + 1;
    for (int a = 0; a <= p; a++) {
        const int i = e + a;
        double d = 0.0;
        if (a >= 1) d += Np[a - 1] / (knot(n, p, i + p) - knot(n, p, i));
        if (a <= p - 1) d -= Np[a] / (knot(n, p, i + p + 1) - knot(n, p, i + 1));
        V[(int64_t)q * P1 + a] = N[a];
        D[(int64_t)q * P1 + a] = p * d;
    }
}

// 1-D pair tables: r = i B + (delta + p), j = i + delta (kept functions,
// global index g = i + off).  s[r], L[r]: first Gauss point and count of the
// elements where both live (L = 0 when j is not kept); W_xy[r][k] the
// products of value/derivative at point s[r] + k.
__global__ void k_iga_pairs(IgaDims d, const double* __restrict__ V, const double* __restrict__ D, int* s, int* L,
                            double* Wvv, double* Wvd, double* Wdv, double* Wdd) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)d.R * d.Lmax) return;
    const int r = (int)(idx / d.Lmax), k = (int)(idx % d.Lmax);
    const int i = r / d.B, delta = r % d.B - d.p, j = i + delta;
    const int gi = i + d.off, gj = j + d.off;
    const int e0 = max(max(gi, gj) - d.p, 0), e1 = min(min(gi, gj), d.n - 1);
    const bool ok = j >= 0 && j < d.m && e0 <= e1;
    const int len = ok ? (e1 - e0 + 1) * d.nq : 0;
    if (k == 0) {
        s[r] = ok ? e0 * d.nq : 0;
        L[r] = len;
    }
    double vv = 0.0, vd = 0.0, dv = 0.0, dd = 0.0;
    if (k < len) {
        const int q = e0 * d.nq + k, e = q / d.nq, P1 = d.p + 1;
        const double vi = V[(int64_t)q * P1 + gi - e], di = D[(int64_t)q * P1 + gi - e];
        const double vj = V[(int64_t)q * P1 + gj - e], dj = D[(int64_t)q * P1 + gj - e];
        vv = vi * vj;
        vd = vi * dj;
        dv = di * vj;
        dd = di * dj;
    }
    Wvv[idx] = vv;
    Wvd[idx] = vd;
    Wdv[idx] = dv;
    Wdd[idx] = dd;
}

// Single-function table of the load vector: r = i, the Gauss points of the
// elements where function g = i + off lives, W1[i][k] its values there.
__global__ void k_iga_single(IgaDims d, const double* __restrict__ V, int* s, int* L, double* W) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)d.R1 * d.L1max) return;
    const int i = (int)(idx / d.L1max), k = (int)(idx % d.L1max);
    const int g = i + d.off, e0 = max(g - d.p, 0), e1 = min(g, d.n - 1);
    const int len = (e1 - e0 + 1) * d.nq;
    if (k == 0) {
        s[i] = e0 * d.nq;
        L[i] = len;
    }
    double v = 0.0;
    if (k < len) {
        const int q = e0 * d.nq + k, e = q / d.nq;
        v = V[(int64_t)q * (d.p + 1) + g - e];
    }
    W[idx] = v;
}

// Plane data per point (q2, q1) of the (xi1, xi2) plane, p2 = q2 Q + q1:
// x, y, the 2x2 block G = J2^-1 J2^-T (g00, g01, g11), |det J2| w1 w2 (h/2)^2
// and 3 pi^2 sin(pi x) sin(pi y).
// geometry 0: identity; 1: quarter annulus, (1 + xi1) c(xi2) with c the
// quadratic NURBS arc through (1,0), (1,1), (0,1), weights 1, sqrt(1/2), 1.
constexpr int kPlane = 7;
__global__ void k_iga_plane(int geometry, int n, int nq, const double* __restrict__ gx,
                            const double* __restrict__ gw, double* plane) {
    const int Q = n * nq;
    const int64_t p2 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p2 >= (int64_t)Q * Q) return;
    const int q1 = (int)(p2 % Q), q2 = (int)(p2 / Q);
    const double h = 1.0 / n;
    const double xi1 = (q1 / nq + 0.5 * (gx[q1 % nq] + 1.0)) * h;
    const double xi2 = (q2 / nq + 0.5 * (gx[q2 % nq] + 1.0)) * h;
    const double w = (0.5 * h * gw[q1 % nq]) * (0.5 * h * gw[q2 % nq]);
    double x, y, j00, j01, j10, j11;
    if (geometry == AMG_GEOM_ANNULUS) {
        const double t = xi2, wm = 0.70710678118654752440;
        const double b0 = (1 - t) * (1 - t), b1 = 2 * t * (1 - t), b2 = t * t;
        const double d0 = -2 * (1 - t), d1 = 2 - 4 * t, d2 = 2 * t;
        const double W = b0 + wm * b1 + b2, dW = d0 + wm * d1 + d2;
        const double ax = b0 + wm * b1, ay = wm * b1 + b2;
        const double dax = d0 + wm * d1, day = wm * d1 + d2;
        const double cx = ax / W, cy = ay / W;
        const double dcx = (dax * W - ax * dW) / (W * W), dcy = (day * W - ay * dW) / (W * W);
        const double r = 1.0 + xi1;
        x = r * cx;
        y = r * cy;
        j00 = cx;
        j01 = r * dcx;
        j10 = cy;
        j11 = r * dcy;
    } else {
        x = xi1;
        y = xi2;
        j00 = 1.0;
        j01 = 0.0;
        j10 = 0.0;
        j11 = 1.0;
    }
    const double det = j00 * j11 - j01 * j10;
    // J2^-1 = [j11 -j01; -j10 j00] / det; G = J2^-1 J2^-T (rows of J2^-1 dotted)
    const double a = j11 / det, b = -j01 / det, c = -j10 / det, dd = j00 / det;
    double* o = plane + p2 * kPlane;
    o[0] = x;
    o[1] = y;
    o[2] = a * a + b * b;
    o[3] = a * c + b * dd;
    o[4] = c * c + dd * dd;
    o[5] = fabs(det) * w;
    const double pi = 3.14159265358979323846;
    o[6] = 3.0 * pi * pi * sin(pi * x) * sin(pi * y);  // the sine source's plane factor
}

// z, w3 (h/2) and sin(pi z) per z point.
constexpr int kZline = 3;
__global__ void k_iga_zline(int n, int nq, const double* __restrict__ gx, const double* __restrict__ gw,
                            double* zl) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n * nq) return;
    const double h = 1.0 / n;
    const double z = (q / nq + 0.5 * (gx[q % nq] + 1.0)) * h;
    zl[kZline * q] = z;
    zl[kZline * q + 1] = 0.5 * h * gw[q % nq];
    zl[kZline * q + 2] = sin(3.14159265358979323846 * z);
}

// ------------------------------------------------ kappa on the tensor cores
// g = sum_k A[p2][k] B[q3][k] over K2 columns: k < M the cosines, M <= k < 2 M
// the (negated) sines, the rest zero.  GB300 adds about two FP64 products per
// SM and clock (16.3 ms for the 8.6 G products of n = 64, p = 3, M = 256, the
// largest part of the assembly), its FP16 tensor cores about a thousand, so
// the product runs in fixed point: every operand is rounded to a multiple of
// 2^-55 (|x| <= 1, so closer than cos and sin themselves are) and split into
// eight balanced base-128 digits, |digit| <= 64, each exact in FP16.  Digit
// products are integers of at most 2^12; the FP32 accumulators of the tensor
// cores add them exactly as long as the sums stay below 2^24, so the products
// of all digit pairs (i, j) with the same weight i + j = t share accumulator t
// and are flushed every kFlushK columns (8 pairs x 256 x 2^12 = 2^23) into a
// 64-bit integer.  Pairs with i + j > 7 are left out: they weigh at most
// 2^-56, and over all columns add about sqrt(7 K2) 2^-58.  What remains is
// the operands' rounding, about sqrt(2 K2) 2^-57: below the rounding of an
// FP64 sum of K2 such terms, whose partial sums reach sqrt(K2 / 2).
// (Splitting FP64 products into exact low-precision products: Ootomo, Ozaki
// and Yokota, "DGEMM on integer matrix multiplication unit", 2024, and
// Mukunoki et al., "DGEMM using tensor cores", 2020.)

// The digits of x, most significant first, stored kSlices arrays of `stride`
// apart; a value that is not finite becomes a NaN in the first digit.
__device__ __forceinline__ void store_digits(double x, __half* out, int64_t stride) {
    long long X = __double2ll_rn(x * (double)(1LL << kFixBits));
    __half d[kSlices];
    constexpr int kHalf = 1 << (kDigitBits - 1), kMask = (1 << kDigitBits) - 1;
#pragma unroll
    for (int t = kSlices - 1; t > 0; t--) {
        const int v = ((int)(X + kHalf) & kMask) - kHalf;
        d[t] = __int2half_rn(v);
        X = (X - v) >> kDigitBits;
    }
    d[0] = isfinite(x) ? __int2half_rn((int)X) : __ushort_as_half(0x7fff);
#pragma unroll
    for (int t = 0; t < kSlices; t++) out[t * stride] = d[t];
}

// Digits of A for the plane points [p0, p0 + rows): column m < M holds
// cos(a_m), column M + m holds -sin(a_m), a_m = omega_m,x x + omega_m,y y +
// phi_m.  Thread per (point, m), m padded to K2 - M (the padding is zero).
__global__ void k_iga_kappa_plane(int64_t p0, int rows, int M, int K2, const double* __restrict__ plane,
                                  const double* __restrict__ om, const double* __restrict__ ph, __half* As) {
    const int W = K2 - M;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)rows * W) return;
    const int row = (int)(idx / W), mm = (int)(idx % W);
    const int64_t stride = (int64_t)rows * K2;
    __half* o = As + (int64_t)row * K2;
    if (mm < M) {
        const double* pl = plane + (p0 + row) * kPlane;
        const double a = om[3 * mm] * pl[0] + om[3 * mm + 1] * pl[1] + ph[mm];
        double sn, cs;
        sincos(a, &sn, &cs);
        store_digits(cs, o + mm, stride);
        store_digits(-sn, o + M + mm, stride);
    } else {
        store_digits(0.0, o + M + mm, stride);
    }
}

// Digits of B, [q3][k]: cos(b_m), sin(b_m), b_m = omega_m,z z.
__global__ void k_iga_kappa_z(int Q, int M, int K2, const double* __restrict__ zl, const double* __restrict__ om,
                              __half* Bs) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)K2 * Q) return;
    const int q3 = (int)(idx / K2), k = (int)(idx % K2);
    double v = 0.0;
    if (k < 2 * M) {
        const int mm = k % M;
        const double b = om[3 * mm + 2] * zl[kZline * q3];
        v = k < M ? cos(b) : sin(b);
    }
    store_digits(v, Bs + idx, (int64_t)K2 * Q);
}

struct CoefOut {
    double *c00, *c01, *c11, *c22, *e;
};

// Coefficients at point (q3, p2) from g (kappa = exp(amp g); amp = 0: kappa = 1).
__device__ __forceinline__ void coef_store(const CoefOut& o, int64_t P2, int64_t p2, int q3, double g, double amp,
                                           const double* __restrict__ plane, const double* __restrict__ zl,
                                           int source) {
    const double* pl = plane + p2 * kPlane;
    const double dw = pl[5] * zl[kZline * q3 + 1];
    const double cw = (amp != 0.0 ? exp(amp * g) : 1.0) * dw;
    const int64_t at = (int64_t)q3 * P2 + p2;
    o.c00[at] = cw * pl[2];
    if (o.c01) o.c01[at] = cw * pl[3];
    o.c11[at] = cw * pl[4];
    o.c22[at] = cw;
    if (o.e) o.e[at] = (source == AMG_SRC_SINE ? pl[6] * zl[kZline * q3 + 2] : 1.0) * dw;
}

// Coefficients without kappa (thread per point).
__global__ void k_iga_coef_const(int64_t P2, int Q, const double* __restrict__ plane, const double* __restrict__ zl,
                                 int source, CoefOut o) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= P2 * Q) return;
    coef_store(o, P2, idx % P2, (int)(idx / P2), 0.0, 0.0, plane, zl, source);
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void copy16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One stage: the kSlices digits of 64 A rows and 64 B rows, 32 columns (64
// bytes) each.  A row's four 16-byte pieces are stored at piece ^ ((row >> 1)
// & 3), so that the eight rows of an ldmatrix fall into different banks.
constexpr int kGRowBytes = kGK * 2;
constexpr int kGOperand = kSlices * kGT * kGRowBytes;
constexpr int kGStageBytes = 2 * kGOperand;
__device__ __forceinline__ int tile_at(int slice, int row, int piece) {
    return (slice * kGT + row) * kGRowBytes + ((piece ^ ((row >> 1) & 3)) << 4);
}

// g on 64 x 64 tiles (plane points p0 + r0 .., z points c0 ..), then the
// coefficients.  8 warps of 32 x 16 outputs: per 16 columns a warp loads the
// eight digits of its 16 B columns (32 registers) and, one at a time, of its
// 32 A rows, and issues 36 digit pairs x 4 MMAs.  Blocks of the same plane
// points run next to each other (x: the z tiles), so A's digits come from L2.
// Measured at n = 64, p = 3, M = 256: digits 1.06 ms (bound by cos and sin in
// FP64), product with the coefficients 2.24 ms (36 digit products, 0.31 T
// multiply-adds: 0.28 PFLOP/s, 0.14 of the rate a plain 16-bit product reaches;
// mma.sync's pipe is 45 % busy, the FP64 pipe 31 % with the coefficients' exp and
// products, 8 warps per SM), against 1.39 and 16.34 ms in FP64.  The whole assembly 30.0 -> 16.6 ms,
// with the error against a dense FP64 contraction 7.4e-16 before and 7.3e-16
// after.
__global__ void __launch_bounds__(256, 1) k_iga_coef_gemm(int64_t P2, int64_t p0, int rows, int Q, int K2, int fix,
                                                         const __half* __restrict__ As,
                                                         const __half* __restrict__ Bs, double amp,
                                                         const double* __restrict__ plane,
                                                         const double* __restrict__ zl, int source, CoefOut o) {
    extern __shared__ __align__(128) unsigned char stage[];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int r0 = blockIdx.y * kGT, c0 = blockIdx.x * kGT;
    const uint32_t base = smem_addr(stage);
    const int64_t astride = (int64_t)rows * K2, bstride = (int64_t)Q * K2;
    // rows past the operands' ends repeat the last one (their outputs are not stored)
    auto load = [&](int buf, int k0) {
        const uint32_t dst = base + buf * kGStageBytes;
#pragma unroll
        for (int u = 0; u < kSlices * kGT * 4 / 256; u++) {
            const int e = tid + 256 * u, piece = e & 3, row = (e >> 2) & (kGT - 1), sl = e / (4 * kGT);
            const int ra = min(r0 + row, rows - 1), rb = min(c0 + row, Q - 1);
            const int at = tile_at(sl, row, piece);
            copy16(dst + at, As + sl * astride + (int64_t)ra * K2 + k0 + piece * 8);
            copy16(dst + kGOperand + at, Bs + sl * bstride + (int64_t)rb * K2 + k0 + piece * 8);
        }
    };
    const int wm = (wid & 1) * 32, wn = (wid >> 1) * 16;
    float acc[kSlices][2][2][4];
    long long tot[2][2][4];
    unsigned bad = 0;
#pragma unroll
    for (int t = 0; t < kSlices; t++)
#pragma unroll
        for (int i = 0; i < 16; i++) acc[t][i >> 3][(i >> 2) & 1][i & 3] = 0.f;
#pragma unroll
    for (int i = 0; i < 16; i++) tot[i >> 3][(i >> 2) & 1][i & 3] = 0;
    const int nk = K2 / kGK;
#pragma unroll
    for (int b = 0; b < kGStages - 1; b++) {
        if (b < nk) load(b, b * kGK);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int kt = 0; kt < nk; kt++) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kGStages - 2) : "memory");
        __syncthreads();
        if (kt + kGStages - 1 < nk) load((kt + kGStages - 1) % kGStages, (kt + kGStages - 1) * kGK);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const uint32_t src = base + (kt % kGStages) * kGStageBytes;
#pragma unroll
        for (int ks = 0; ks < kGK / 16; ks++) {
            uint32_t b[kSlices][4];
#pragma unroll
            for (int j = 0; j < kSlices; j++)
                ldmatrix4(b[j], src + kGOperand + tile_at(j, wn + (lane & 7) + ((lane >> 4) << 3),
                                                          ks * 2 + ((lane >> 3) & 1)));
#pragma unroll
            for (int i = 0; i < kSlices; i++) {
                uint32_t a[2][4];
#pragma unroll
                for (int mi = 0; mi < 2; mi++)
                    ldmatrix4(a[mi], src + tile_at(i, wm + mi * 16 + (lane & 15), ks * 2 + (lane >> 4)));
#pragma unroll
                for (int j = 0; j < kSlices - i; j++)
#pragma unroll
                    for (int mi = 0; mi < 2; mi++) {
                        mma_f16(acc[i + j][mi][0], a[mi], b[j][0], b[j][1]);
                        mma_f16(acc[i + j][mi][1], a[mi], b[j][2], b[j][3]);
                    }
            }
        }
        if ((kt + 1) % (kFlushK / kGK) == 0 || kt + 1 == nk) {
            // weight of accumulator t: 2^(2 x 49 - 7 t - 2 x 55) = 2^-(12 + 7 t),
            // in units of 2^-fix
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const int mi = i >> 3, ni = (i >> 2) & 1, e = i & 3;
                if (isnan(acc[0][mi][ni][e])) bad |= 1u << i;
                long long s = 0;
#pragma unroll
                for (int t = 0; t < kSlices; t++) {
                    const long long v = (long long)__float2int_rn(acc[t][mi][ni][e]);
                    const int sh = fix - 2 * (kFixBits - kDigitBits * (kSlices - 1)) - kDigitBits * t;
                    s += sh >= 0 ? v << sh : (v + (1LL << (-sh - 1))) >> -sh;
                    acc[t][mi][ni][e] = 0.f;
                }
                tot[mi][ni][e] += s;
            }
        }
    }
    const double unit = __longlong_as_double((long long)(1023 - fix) << 52);
#pragma unroll
    for (int i = 0; i < 16; i++) {
        const int mi = i >> 3, ni = (i >> 2) & 1, e = i & 3;
        const int row = r0 + wm + mi * 16 + (lane >> 2) + (e >> 1) * 8;
        const int q3 = c0 + wn + ni * 8 + (lane & 3) * 2 + (e & 1);
        if (row < rows && q3 < Q) {
            const double g = bad >> i & 1u ? __longlong_as_double(0x7ff8000000000000LL) : (double)tot[mi][ni][e] * unit;
            coef_store(o, P2, p0 + row, q3, g, amp, plane, zl, source);
        }
    }
}

// Contraction of the middle (outer-major) axis: Y[o][u][c] (+)= sum_{k < L[r]}
// W[r][k] X[o][s[r] + k][c], c < IN, u < R.  Block (tile of 32 c, o): X's
// Q x 32 slab in shared memory, warps over u, lanes over c.  p1 = 0: pair r =
// u; else u counts the pairs with delta >= 0, p1 = p + 1 per function of
// B = 2 p + 1 pairs.
__global__ void __launch_bounds__(32 * kCtWarps) k_iga_outer(int64_t IN, int Q, int R, const double* __restrict__ X,
                                                             const int* __restrict__ s, const int* __restrict__ L,
                                                             const double* __restrict__ W, int Lmax, double* Y,
                                                             int accumulate, int B, int p1) {
    extern __shared__ double xs[];  // [Q][kCtIn]
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t c0 = (int64_t)blockIdx.x * kCtIn;
    const int64_t o = blockIdx.y;
    const double* Xo = X + o * Q * IN;
    for (int q = ty; q < Q; q += kCtWarps) xs[q * kCtIn + tx] = c0 + tx < IN ? Xo[(int64_t)q * IN + c0 + tx] : 0.0;
    __syncthreads();
    if (c0 + tx >= IN) return;
    double* Yo = Y + o * R * IN + c0 + tx;
    for (int u = ty; u < R; u += kCtWarps) {
        const int r = p1 ? (u / p1) * B + (p1 - 1) + u % p1 : u;
        const int st = s[r], len = L[r];
        const double* w = W + (int64_t)r * Lmax;
        double acc = 0.0;
        for (int k = 0; k < len; k++) acc = fma(w[k], xs[(st + k) * kCtIn + tx], acc);
        double* y = Yo + (int64_t)u * IN;
        *y = accumulate ? *y + acc : acc;
    }
}

// Last contraction (the innermost axis, q1) and the CSR scatter: rows
// o = u3 R + r2 (u3: the direction-3 pairs with delta3 >= 0) of the ng
// direction-1 groups X_g[o][q1]; K(I, J) = sum_g sum_k W_g[r1][k] X_g[o][s[r1]
// + k] goes to the position of J in row I (columns in (delta3, delta2, delta1)
// order) and of I in row J; of the two, the pair whose first nonzero of
// (delta3, delta2, delta1) is positive is computed.  A block stages
// `rows` consecutive rows of every group in shared memory (row stride Q + 1);
// thread t takes row t % rows and every (256 / rows)-th pair from t / rows on,
// so the lanes that share a pair read the same weights (a broadcast) and rows
// a padded stride apart.
struct InnerGroups {
    const double* X[4];
    const double* W[4];
    int ng;
};

__device__ __forceinline__ void band_range(int i, int m, int p, int& lo, int& nv) {
    lo = max(-p, -i);
    nv = min(p, m - 1 - i) - lo + 1;
}

constexpr int kInThreads = 256;

template <int NG>
__global__ void __launch_bounds__(kInThreads) k_iga_inner_csr(IgaDims d, InnerGroups G, int rows,
                                                              const int* __restrict__ s, const int* __restrict__ L,
                                                              const int64_t* __restrict__ rowptr, double* val) {
    extern __shared__ double xs[];  // [NG][rows][Q + 1]
    const int64_t O = (int64_t)d.m * (d.p + 1) * d.R;
    const int64_t o0 = (int64_t)blockIdx.x * rows;
    const int Qp = d.Q + 1;
#pragma unroll
    for (int g = 0; g < NG; g++)
        for (int t = threadIdx.x; t < rows * d.Q; t += blockDim.x) {
            const int row = t / d.Q, q = t % d.Q;
            xs[((int64_t)g * rows + row) * Qp + q] = o0 + row < O ? G.X[g][(o0 + row) * d.Q + q] : 0.0;
        }
    __syncthreads();
    const int row = threadIdx.x % rows, slot = threadIdx.x / rows, nslot = kInThreads / rows;
    const int64_t o = o0 + row;
    if (o >= O) return;
    const int u3 = (int)(o / d.R), r2 = (int)(o % d.R);
    const int i3 = u3 / (d.p + 1), d3 = u3 % (d.p + 1), i2 = r2 / d.B, d2 = r2 % d.B - d.p;
    const int j3 = i3 + d3, j2 = i2 + d2;
    if (j3 >= d.m || j2 < 0 || j2 >= d.m || (d3 == 0 && d2 < 0)) return;
    int lo3, nv3, lo2, nv2, ml3, mv3, ml2, mv2;  // the bands of I's and of J's row
    band_range(i3, d.m, d.p, lo3, nv3);
    band_range(i2, d.m, d.p, lo2, nv2);
    band_range(j3, d.m, d.p, ml3, mv3);
    band_range(j2, d.m, d.p, ml2, mv2);
    const double* xr = xs + (int64_t)row * Qp;
    // pairs in delta-major order: the pairs a warp shares have the same
    // delta, hence the same number of common Gauss points (no divergence)
    for (int u = slot; u < d.R; u += nslot) {
        const int r1 = (u % d.m) * d.B + u / d.m;
        const int i1 = r1 / d.B, d1 = r1 % d.B - d.p, j1 = i1 + d1;
        if (j1 < 0 || j1 >= d.m || (d3 == 0 && d2 == 0 && d1 < 0)) continue;
        const int st = s[r1], len = L[r1];
        double acc = 0.0;
#pragma unroll
        for (int g = 0; g < NG; g++) {
            const double* x = xr + (int64_t)g * rows * Qp + st;
            const double* wt = G.W[g] + (int64_t)r1 * d.Lmax;
            for (int k = 0; k < len; k++) acc = fma(__ldg(wt + k), x[k], acc);
        }
        int lo1, nv1;
        band_range(i1, d.m, d.p, lo1, nv1);
        const int64_t I = i1 + (int64_t)d.m * (i2 + (int64_t)d.m * i3);
        val[rowptr[I] + ((int64_t)(d3 - lo3) * nv2 + (d2 - lo2)) * nv1 + (d1 - lo1)] = acc;
        if (d3 == 0 && d2 == 0 && d1 == 0) continue;
        int ml1, mv1;
        band_range(j1, d.m, d.p, ml1, mv1);
        const int64_t J = j1 + (int64_t)d.m * (j2 + (int64_t)d.m * j3);
        val[rowptr[J] + ((int64_t)(-d3 - ml3) * mv2 + (-d2 - ml2)) * mv1 + (-d1 - ml1)] = acc;
    }
}

// Load vector's last contraction: F[o m + i1] = sum_k W1[i1][k] X[o][s1[i1] + k].
__global__ void __launch_bounds__(32 * kInRows) k_iga_inner_dense(IgaDims d, const double* __restrict__ X,
                                                                  const int* __restrict__ s,
                                                                  const int* __restrict__ L,
                                                                  const double* __restrict__ W, double* F) {
    extern __shared__ double xs[];  // [kInRows][Q + 1]
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t O = (int64_t)d.m * d.m;
    const int64_t o0 = (int64_t)blockIdx.x * kInRows;
    const int Qp = d.Q + 1;
    for (int t = threadIdx.x; t < kInRows * d.Q; t += blockDim.x) {
        const int row = t / d.Q, q = t % d.Q;
        xs[(int64_t)row * Qp + q] = o0 + row < O ? X[(o0 + row) * d.Q + q] : 0.0;
    }
    __syncthreads();
    const int64_t o = o0 + w;
    if (o >= O) return;
    for (int i1 = lane; i1 < d.m; i1 += 32) {
        const int st = s[i1], len = L[i1];
        const double* x = xs + (int64_t)w * Qp + st;
        const double* wt = W + (int64_t)i1 * d.L1max;
        double acc = 0.0;
        for (int k = 0; k < len; k++) acc = fma(wt[k], x[k], acc);
        F[o * d.m + i1] = acc;
    }
}

// sum_{x < i} nv(x), nv(x) = min(p, m-1-x) - max(-p, -x) + 1 (band count of
// index x), in closed form: i + f(i) + f(m) - f(m - i), f(i) = sum_{x<i} min(p, x).
__host__ __device__ inline int64_t band_prefix(int64_t i, int64_t m, int64_t p) {
    auto f = [p](int64_t k) -> int64_t { return k <= p ? k * (k - 1) / 2 : p * (p + 1) / 2 + p * (k - p - 1); };
    return i + f(i) + f(m) - f(m - i);
}

// CSR pattern (warp per row): rowptr in closed form, columns in ascending
// order (delta3, delta2, delta1); rowptr[N] by the last row's warp.
__global__ void k_iga_pattern(int m, int p, int64_t* rowptr, int32_t* col) {
    const int lane = threadIdx.x & 31;
    const int64_t N = (int64_t)m * m * m;
    const int64_t T = band_prefix(m, m, p);
    for (int64_t I = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; I < N;
         I += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int i1 = (int)(I % m), i2 = (int)((I / m) % m), i3 = (int)(I / ((int64_t)m * m));
        int lo1, nv1, lo2, nv2, lo3, nv3;
        band_range(i1, m, p, lo1, nv1);
        band_range(i2, m, p, lo2, nv2);
        band_range(i3, m, p, lo3, nv3);
        const int64_t base = band_prefix(i3, m, p) * T * T +
                             (int64_t)nv3 * (band_prefix(i2, m, p) * T + (int64_t)nv2 * band_prefix(i1, m, p));
        if (lane == 0) {
            rowptr[I] = base;
            if (I == N - 1) rowptr[N] = T * T * T;
        }
        const int cnt = nv1 * nv2 * nv3;
        for (int t = lane; t < cnt; t += 32) {
            const int c1 = t % nv1, c2 = (t / nv1) % nv2, c3 = t / (nv1 * nv2);
            const int j1 = i1 + lo1 + c1, j2 = i2 + lo2 + c2, j3 = i3 + lo3 + c3;
            col[base + t] = j1 + m * (j2 + m * j3);
        }
    }
}

inline int nblk(int64_t work, int threads) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((work + threads - 1) / threads, (int64_t)1 << 30));
}

int check_patch(const amg_iga_patch* P, IgaDims& d) {
    if (!P) return AMG_ERR_ARG;
    const int nq = P->nq == 0 ? P->p + 1 : P->nq;
    if (P->n < 1 || P->p < 1 || P->p > kMaxDeg || nq < 1 || nq > kMaxNq) return AMG_ERR_ARG;
    if ((int64_t)P->n * nq > kMaxQ) return AMG_ERR_ARG;
    if (P->geometry != AMG_GEOM_CUBE && P->geometry != AMG_GEOM_ANNULUS) return AMG_ERR_ARG;
    if (P->with_boundary != 0 && P->with_boundary != 1) return AMG_ERR_ARG;
    if (P->source != AMG_SRC_ONE && P->source != AMG_SRC_SINE) return AMG_ERR_ARG;
    if (P->kappa_m < 0 || P->kappa_m > 65536) return AMG_ERR_ARG;
    if (P->kappa_m > 0 && (!P->kappa_omega || !P->kappa_phi || !std::isfinite(P->kappa_sigma))) return AMG_ERR_ARG;
    d.n = P->n;
    d.p = P->p;
    d.nq = nq;
    d.off = P->with_boundary ? 0 : 1;
    d.m = P->with_boundary ? P->n + P->p : P->n + P->p - 2;
    d.Q = P->n * nq;
    d.B = 2 * P->p + 1;
    d.R = d.m * d.B;
    d.Lmax = (P->p + 1) * nq;
    d.R1 = d.m;
    d.L1max = (P->p + 1) * nq;
    if (d.m > 0 && (int64_t)d.m * d.m * d.m > 0x7fffffffLL) return AMG_ERR_ARG;
    return AMG_OK;
}

}  // namespace
}  // namespace amg

using namespace amg;

extern "C" int amg_iga_size(const amg_iga_patch* P, int64_t* n, int64_t* nnz) {
    IgaDims d;
    const int rc = check_patch(P, d);
    if (rc != AMG_OK) return rc;
    if (!n || !nnz) return AMG_ERR_ARG;
    const int64_t m = std::max(d.m, 0);
    const int64_t T = m > 0 ? band_prefix(m, m, d.p) : 0;
    *n = m * m * m;
    *nnz = T * T * T;
    return AMG_OK;
}

extern "C" int amg_iga_assemble(const amg_iga_patch* P, int64_t* rowptr, int32_t* col, double* val, double* F,
                                void* cuda_stream, double* flops) {
    IgaDims d;
    int rc = check_patch(P, d);
    if (rc != AMG_OK) return rc;
    if (!rowptr || !col || !val) return AMG_ERR_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int m = std::max(d.m, 0);
    if (m == 0) {  // nothing kept: rowptr = {0}
        cudaError_t e = cudaMemsetAsync(rowptr, 0, sizeof(int64_t), s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (flops) *flops = 0.0;
        return e == cudaSuccess ? AMG_OK : report_cuda(e, "amg_iga_assemble");
    }
    const int Q = d.Q;
    const int64_t P2 = (int64_t)Q * Q, P3 = P2 * Q, R = d.R;
    const int M = P->kappa_m;
    const int K2 = M > 0 ? ((2 * M + kGK - 1) / kGK) * kGK : 0;
    const bool has01 = P->geometry != AMG_GEOM_CUBE;
    std::vector<void*> bufs;
    struct Free {
        std::vector<void*>* b;
        cudaStream_t s;
        ~Free() {
            for (void* p : *b)
                if (p) cudaFreeAsync(p, s);
        }
    } guard{&bufs, s};
    cudaError_t err = cudaSuccess;
    auto get = [&](auto** p, size_t count) {
        *p = nullptr;
        if (err != cudaSuccess) return;
        void* q = nullptr;
        err = dev_alloc(&q, std::max<size_t>(count, 1) * sizeof(**p), s);
        if (err == cudaSuccess) {
            bufs.push_back(q);
            *p = reinterpret_cast<std::remove_reference_t<decltype(*p)>>(q);
        }
    };
    auto release = [&](void* p) {
        auto it = std::find(bufs.begin(), bufs.end(), p);
        if (it != bufs.end()) {
            cudaFreeAsync(p, s);
            bufs.erase(it);
        }
    };
    double *gx, *gw, *V, *D, *plane, *zl, *Wt[4], *W1;
    int *sp, *Lp, *s1, *L1;
    get(&gx, d.nq);
    get(&gw, d.nq);
    get(&V, (size_t)Q * (d.p + 1));
    get(&D, (size_t)Q * (d.p + 1));
    get(&plane, (size_t)P2 * kPlane);
    get(&zl, (size_t)Q * kZline);
    for (auto& w : Wt) get(&w, (size_t)R * d.Lmax);
    get(&W1, (size_t)d.R1 * d.L1max);
    get(&sp, R);
    get(&Lp, R);
    get(&s1, d.R1);
    get(&L1, d.R1);
    if (err != cudaSuccess) return report_cuda(err, "amg_iga_assemble workspace");
    double *const Wvv = Wt[0], *const Wvd = Wt[1], *const Wdv = Wt[2], *const Wdd = Wt[3];
    k_iga_gauss<<<AMG_GRID(1), 32, 0, s>>>(d.nq, gx, gw);
    k_iga_basis<<<AMG_GRID(nblk(Q, 128)), 128, 0, s>>>(d.n, d.p, d.nq, gx, V, D);
    k_iga_pairs<<<AMG_GRID(nblk(R * d.Lmax, 256)), 256, 0, s>>>(d, V, D, sp, Lp, Wvv, Wvd, Wdv, Wdd);
    k_iga_single<<<AMG_GRID(nblk((int64_t)d.R1 * d.L1max, 256)), 256, 0, s>>>(d, V, s1, L1, W1);
    k_iga_plane<<<AMG_GRID(nblk(P2, 256)), 256, 0, s>>>(P->geometry, d.n, d.nq, gx, gw, plane);
    k_iga_zline<<<AMG_GRID(nblk(Q, 128)), 128, 0, s>>>(d.n, d.nq, gx, gw, zl);
    k_iga_pattern<<<AMG_GRID(nblk((int64_t)m * m * m * 32, 256)), 256, 0, s>>>(m, d.p, rowptr, col);
    // coefficients at every Gauss point
    CoefOut co{};
    get(&co.c00, (size_t)P3);
    if (has01) get(&co.c01, (size_t)P3);
    get(&co.c11, (size_t)P3);
    get(&co.c22, (size_t)P3);
    if (F) get(&co.e, (size_t)P3);
    if (err != cudaSuccess) return report_cuda(err, "amg_iga_assemble coefficients");
    double gemm_fma = 0.0;
    if (M > 0) {
        // A's digits in pieces of about kDigitBytes (64 rows at least), so that
        // they stay in L2 between the kernel that writes them and the product
        __half *As, *Bs;
        const int64_t row_bytes = (int64_t)kSlices * K2 * sizeof(__half);
        int64_t tiles = std::min<int64_t>((P2 + kGT - 1) / kGT, std::max<int64_t>(1, kDigitBytes / (row_bytes * kGT)));
        const int ct = (Q + kGT - 1) / kGT;
        int dev = 0, sms = 1;
        if ((err = cudaGetDevice(&dev)) != cudaSuccess ||
            (err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
            return report_cuda(err, "amg_iga_assemble device");
        // whole waves of blocks (one per SM) where a piece has at least one
        const int64_t wave = sms / std::gcd(sms, ct);
        if (tiles >= wave && tiles * kGT < P2) tiles -= tiles % wave;
        const int64_t chunk = tiles * kGT;
        get(&As, (size_t)(std::min(chunk, P2) * row_bytes / sizeof(__half)));
        get(&Bs, (size_t)kSlices * K2 * Q);
        if (err != cudaSuccess) return report_cuda(err, "amg_iga_assemble kappa");
        const size_t smg = (size_t)kGStages * kGStageBytes;
        if ((err = cudaFuncSetAttribute(k_iga_coef_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smg)) !=
            cudaSuccess)
            return report_cuda(err, "amg_iga_assemble smem");
        k_iga_kappa_z<<<AMG_GRID(nblk((int64_t)K2 * Q, 256)), 256, 0, s>>>(Q, M, K2, zl, P->kappa_omega, Bs);
        const double amp = P->kappa_sigma * sqrt(2.0 / M);
        // |g| <= 2 M < 2^(62 - fix): the 64-bit sums cannot overflow
        int fix = 53;
        while (fix > 32 && (1LL << (62 - fix)) <= 2 * (int64_t)M) fix--;
        for (int64_t p0 = 0; p0 < P2; p0 += chunk) {
            const int rows = (int)std::min(chunk, P2 - p0);
            k_iga_kappa_plane<<<AMG_GRID(nblk((int64_t)rows * (K2 - M), 256)), 256, 0, s>>>(
                p0, rows, M, K2, plane, P->kappa_omega, P->kappa_phi, As);
            dim3 grid((unsigned)((Q + kGT - 1) / kGT), (unsigned)((rows + kGT - 1) / kGT));
            k_iga_coef_gemm<<<AMG_GRID(grid), 256, smg, s>>>(P2, p0, rows, Q, K2, fix, As, Bs, amp, plane, zl,
                                                             P->source, co);
        }
        gemm_fma = (double)P2 * Q * (2.0 * M);
        release(As);
        release(Bs);
    } else {
        k_iga_coef_const<<<AMG_GRID(nblk(P3, 256)), 256, 0, s>>>(P2, Q, plane, zl, P->source, co);
    }
    if ((err = cudaGetLastError()) != cudaSuccess) return report_cuda(err, "amg_iga_assemble launch");
    // contractions: Q x 32 staging per block
    const size_t smo = (size_t)Q * kCtIn * sizeof(double);
    if ((err = allow_smem(k_iga_outer, smo)) != cudaSuccess) return report_cuda(err, "amg_iga_assemble smem");
    auto outer = [&](const double* X, int64_t O, int64_t IN, int Rr, const int* ss, const int* LL, const double* W,
                     int Lm, double* Y, int accumulate, int p1 = 0) {
        dim3 grid((unsigned)((IN + kCtIn - 1) / kCtIn), (unsigned)O);
        k_iga_outer<<<AMG_GRID(grid), 32 * kCtWarps, smo, s>>>(IN, Q, Rr, X, ss, LL, W, Lm, Y, accumulate, d.B, p1);
    };
    const int p1 = d.p + 1;
    const int64_t Rh = (int64_t)m * p1, RhR = Rh * R;  // pairs with delta >= 0
    // direction 3
    double *A00, *A01 = nullptr, *A11, *A22;
    get(&A00, (size_t)Rh * P2);
    if (has01) get(&A01, (size_t)Rh * P2);
    get(&A11, (size_t)Rh * P2);
    get(&A22, (size_t)Rh * P2);
    if (err != cudaSuccess) return report_cuda(err, "amg_iga_assemble direction 3");
    outer(co.c00, 1, P2, (int)Rh, sp, Lp, Wvv, d.Lmax, A00, 0, p1);
    if (has01) outer(co.c01, 1, P2, (int)Rh, sp, Lp, Wvv, d.Lmax, A01, 0, p1);
    outer(co.c11, 1, P2, (int)Rh, sp, Lp, Wvv, d.Lmax, A11, 0, p1);
    outer(co.c22, 1, P2, (int)Rh, sp, Lp, Wdd, d.Lmax, A22, 0, p1);
    double *fa = nullptr, *fb = nullptr;
    if (F) {
        get(&fa, (size_t)m * P2);
        if (err != cudaSuccess) return report_cuda(err, "amg_iga_assemble load");
        outer(co.e, 1, P2, d.R1, s1, L1, W1, d.L1max, fa, 0);
    }
    release(co.c00);
    release(co.c01);
    release(co.c11);
    release(co.c22);
    release(co.e);
    // direction 2, grouped by the direction-1 type
    double *Gdd, *Gdv = nullptr, *Gvd = nullptr, *Gvv;
    get(&Gdd, (size_t)RhR * Q);
    if (has01) {
        get(&Gdv, (size_t)RhR * Q);
        get(&Gvd, (size_t)RhR * Q);
    }
    get(&Gvv, (size_t)RhR * Q);
    if (err != cudaSuccess) return report_cuda(err, "amg_iga_assemble direction 2");
    outer(A00, Rh, Q, d.R, sp, Lp, Wvv, d.Lmax, Gdd, 0);
    if (has01) {
        outer(A01, Rh, Q, d.R, sp, Lp, Wvd, d.Lmax, Gdv, 0);
        outer(A01, Rh, Q, d.R, sp, Lp, Wdv, d.Lmax, Gvd, 0);
    }
    outer(A11, Rh, Q, d.R, sp, Lp, Wdd, d.Lmax, Gvv, 0);
    outer(A22, Rh, Q, d.R, sp, Lp, Wvv, d.Lmax, Gvv, 1);
    if (F) {
        get(&fb, (size_t)m * m * Q);
        if (err != cudaSuccess) return report_cuda(err, "amg_iga_assemble load");
        outer(fa, m, Q, d.R1, s1, L1, W1, d.L1max, fb, 0);
        release(fa);
    }
    release(A00);
    release(A01);
    release(A11);
    release(A22);
    // direction 1 and the scatter
    InnerGroups G{};
    G.X[G.ng] = Gdd;
    G.W[G.ng++] = Wdd;
    if (has01) {
        G.X[G.ng] = Gdv;
        G.W[G.ng++] = Wdv;
        G.X[G.ng] = Gvd;
        G.W[G.ng++] = Wvd;
    }
    G.X[G.ng] = Gvv;
    G.W[G.ng++] = Wvv;
    // rows per block of the last contraction: 8 (four pairs per warp), so
    // that several blocks share an SM (16 rows left one block, 8 warps, per
    // SM: 12 % of the warp slots); fewer when the staged rows do not fit
    int optin = 0, devi = 0;
    if ((err = cudaGetDevice(&devi)) != cudaSuccess ||
        (err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, devi)) != cudaSuccess)
        return report_cuda(err, "amg_iga_assemble device");
    int rows = 8;
    while (rows > 1 && (size_t)G.ng * rows * (Q + 1) * sizeof(double) > (size_t)optin / 2) rows >>= 1;
    const size_t smi = (size_t)G.ng * rows * (Q + 1) * sizeof(double);
    if (smi > (size_t)optin) return AMG_ERR_ARG;
    auto inner = [&](auto kern) {
        cudaError_t e = allow_smem(kern, smi);
        if (e != cudaSuccess) return e;
        kern<<<AMG_GRID(nblk(RhR, rows)), kInThreads, smi, s>>>(d, G, rows, sp, Lp, rowptr, val);
        return cudaGetLastError();
    };
    err = G.ng == 4 ? inner(k_iga_inner_csr<4>) : inner(k_iga_inner_csr<2>);
    if (err != cudaSuccess) return report_cuda(err, "amg_iga_assemble last contraction");
    if (F) {
        const size_t smf = (size_t)kInRows * (Q + 1) * sizeof(double);
        if ((err = allow_smem(k_iga_inner_dense, smf)) != cudaSuccess)
            return report_cuda(err, "amg_iga_assemble smem");
        k_iga_inner_dense<<<AMG_GRID(nblk((int64_t)m * m, kInRows)), 32 * kInRows, smf, s>>>(d, fb, s1, L1, W1, F);
    }
    if ((err = cudaGetLastError()) != cudaSuccess) return report_cuda(err, "amg_iga_assemble launch");
    if ((err = cudaStreamSynchronize(s)) != cudaSuccess) return report_cuda(err, "amg_iga_assemble");
    if (flops) {
        // FMAs of kappa's product and of the contractions of all stored entries
        // (sums over the pair tables' lengths; the symmetry halves what runs)
        std::vector<int> Lh(d.R), L1h(d.R1);
        if ((err = cudaMemcpy(Lh.data(), Lp, sizeof(int) * d.R, cudaMemcpyDeviceToHost)) != cudaSuccess ||
            (err = cudaMemcpy(L1h.data(), L1, sizeof(int) * d.R1, cudaMemcpyDeviceToHost)) != cudaSuccess)
            return report_cuda(err, "amg_iga_assemble flops");
        double sl = 0.0, sl1 = 0.0;
        for (int v : Lh) sl += v;
        for (int v : L1h) sl1 += v;
        // pairs whose second function is kept (the others are zero rows)
        double rows_ok = 0.0;
        for (int r = 0; r < d.R; r++) rows_ok += Lh[r] > 0 ? 1.0 : 0.0;
        const int na = has01 ? 4 : 3, nb = has01 ? 5 : 3;
        double fma_k = na * sl * (double)P2 + nb * rows_ok * sl * Q + G.ng * rows_ok * rows_ok * sl;
        double fma_f = F ? sl1 * (double)P2 + (double)m * sl1 * Q + (double)m * m * sl1 : 0.0;
        *flops = 2.0 * (gemm_fma + fma_k + fma_f);
    }
    return AMG_OK;
}
