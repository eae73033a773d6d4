// weights.cu — RBF-FD stencil weights, batched: one block of 128 threads per stencil.
//
// For every centre x_c with stencil S (N_L nodes) the block assembles the saddle
// system of Eq. augmentedSystem in shared memory, FP64:
//   A_jl = |xi_j - xi_l|^k      (PHS r^k, Eq. rbfScaling: xi = (x - x_c) / delta)
//   P_jl = p_l(xi_j)            (monomials of degree <= m, graded lexicographic)
//   M = [[A, P], [P^T, 0]]
// and solves the right-hand sides of up to RBF_MAX_OPS operators L (Eq. operatorApprox)
// together:
//   b_j = (L Phi_j)(y), c_l = (L p_l)(y),  y = x_c + off
// either from an FP32 inverse refined to FP64 (k <= 5, k_weights_fast) or by an FP64 LU with
// partial pivoting and one refinement (k_weights: k >= 7, and the systems that the first one
// hands on).  Residuals are formed in integers in both; row_products and Residual32 say what
// they drop.  delta is the distance to the nearest other node
// (centre is a node) or to the nearest node (centre is a free point such as a permeability
// probe).
//
// What bounds it: FP64 (2 lanes per clock and SM, 1/64 of the FP32 rate) is the scarce pipe,
// so the design counts FP64 operations.
//  * The residual, which has to carry about twice the working precision, runs on
//    the integer pipe: rows of M and columns of x are cut into three 26/27-bit
//    slices relative to the row's (column's) largest exponent, six to eight 32 x 32 -> 64
//    bit multiply-adds per product accumulate without rounding.  A compensated FP64 dot product (ten
//    FP64 operations per product) was two thirds of the FP64 work of an 18-operator system.
//  * One reciprocal per pivot instead of a division per right-hand side; each
//    distance of the symmetric A computed once.
//  * FP64 updates run over (row, column) pairs packed over the block's threads with
//    incremental indices (no integer division), so warps stay full at small sizes.
//  * The untouched matrix is kept as a packed lower triangle and the residual's
//    buffers are reused, which leaves 4-5 blocks (16-20 warps) per SM at N_L = 30..40.
// Measured (GB300, 2070 MHz), 86,397 systems of n = 60 with 4 operators (N_L = 40, r^5,
// m = 3) / 120,840 systems of n = 40 with 18 operators (N_L = 30, r^3, m = 2): FP32 inverse
// 19 / 24 ms, with no pipe above 75 % (integer multiplies 50 / 60 %, FP64 43 / 29 %); FP64 LU
// 34.4 / 33.5 ms, the FP64 pipe 81-87 % busy; one warp per system with FP64 LU and the
// compensated product 164 / 167 ms.
#include <algorithm>

#include "internal.cuh"

namespace rbf {

namespace {

constexpr int WT = 128;  // threads per system (>= RBF_MAX_NS: one residual row per thread)
static_assert(WT >= RBF_MAX_NS, "one residual row per thread");

// exponents (a, b, c) of the monomials, graded lexicographic order, degree <= 4
__constant__ int8_t c_mono[RBF_MAX_NP][3] = {
    {0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0}, {1, 1, 0}, {1, 0, 1}, {0, 2, 0}, {0, 1, 1},
    {0, 0, 2}, {3, 0, 0}, {2, 1, 0}, {2, 0, 1}, {1, 2, 0}, {1, 1, 1}, {1, 0, 2}, {0, 3, 0}, {0, 2, 1},
    {0, 1, 2}, {0, 0, 3}, {4, 0, 0}, {3, 1, 0}, {3, 0, 1}, {2, 2, 0}, {2, 1, 1}, {2, 0, 2}, {1, 3, 0},
    {1, 2, 1}, {1, 1, 2}, {1, 0, 3}, {0, 4, 0}, {0, 3, 1}, {0, 2, 2}, {0, 1, 3}, {0, 0, 4}};

__device__ __forceinline__ double ipow(double x, int e) {
    double r = 1.0;
    for (int i = 0; i < e; ++i) r *= x;
    return r;
}
// |s|^e for odd e >= 1 from s . s
__device__ __forceinline__ double odd_pow(double s2, int e) {
    double r = sqrt(s2);
    for (int i = 1; i < e; i += 2) r *= s2;
    return r;
}

// L applied to the basis function centred at xi_j, at eta; s = eta - xi_j
__device__ __forceinline__ double rbf_rhs(int kind, int k, double sx, double sy, double sz, double delta) {
    const double s2 = sx * sx + sy * sy + sz * sz;
    switch (kind) {
    case OP_INTERP: return odd_pow(s2, k);
    case OP_DX: return (double)k * odd_pow(s2, k - 2) * sx / delta;
    case OP_DY: return (double)k * odd_pow(s2, k - 2) * sy / delta;
    case OP_DZ: return (double)k * odd_pow(s2, k - 2) * sz / delta;
    default: return (double)(k * (k + 1)) * odd_pow(s2, k - 2) / (delta * delta);
    }
}

// L applied to x^a y^b z^c at eta (scaled coordinates; derivatives in physical ones)
__device__ double mono_rhs(int kind, int a, int b, int c, double ex, double ey, double ez, double delta) {
    switch (kind) {
    case OP_INTERP: return ipow(ex, a) * ipow(ey, b) * ipow(ez, c);
    case OP_DX: return a ? (double)a * ipow(ex, a - 1) * ipow(ey, b) * ipow(ez, c) / delta : 0.0;
    case OP_DY: return b ? (double)b * ipow(ex, a) * ipow(ey, b - 1) * ipow(ez, c) / delta : 0.0;
    case OP_DZ: return c ? (double)c * ipow(ex, a) * ipow(ey, b) * ipow(ez, c - 1) / delta : 0.0;
    default: {
        double s = 0.0;
        if (a >= 2) s += (double)(a * (a - 1)) * ipow(ex, a - 2) * ipow(ey, b) * ipow(ez, c);
        if (b >= 2) s += (double)(b * (b - 1)) * ipow(ex, a) * ipow(ey, b - 2) * ipow(ez, c);
        if (c >= 2) s += (double)(c * (c - 1)) * ipow(ex, a) * ipow(ey, b) * ipow(ez, c - 2);
        return s / (delta * delta);
    }
    }
}

// packed lower triangle of the symmetric matrix
__host__ __device__ __forceinline__ int tri_at(int r, int q) {
    return r >= q ? r * (r + 1) / 2 + q : q * (q + 1) / 2 + r;
}

struct WLayout {
    int ns, ld;      // system size, padded row stride
    size_t m0, x, r, xs, xi, rp, ints, total;  // offsets and size in doubles
};
__host__ __device__ inline WLayout wlayout(int n_l, int np, int n_ops) {
    WLayout L;
    L.ns = n_l + np;
    L.ld = L.ns | 1;  // odd stride: FP64 columns fall on different banks
    const size_t ns = L.ns, no = n_ops;
    // slices of x first (16 bytes per entry: 16-byte alignment; after the residual the
    // same room holds the permuted residual), then M (factors), the packed M0
    L.xs = 0;
    L.m0 = 2 * ns * no + ns * L.ld;
    L.x = L.m0 + ns * (ns + 1) / 2;
    L.r = L.x + ns * no;
    L.xi = L.r + ns * no;
    L.rp = L.xi + 3 * (size_t)n_l;
    L.ints = L.rp + ns;  // perm[ns], exponents of x per operator
    L.total = L.ints + (ns + no + 1) / 2 + 1;
    L.total = (L.total + 1) & ~(size_t)1;
    return L;
}

// |v| cut into slices of 26, 27 and 27 bits below 2^(e - 1022), e the biased exponent
// bound (no entry's exponent is larger), each with v's sign; what lies below 2^-80 of
// the bound is dropped
__device__ __forceinline__ void cut(double v, int e, int &s0, int &s1, int &s2) {
    const long long b = __double_as_longlong(v);
    const int ev = (int)((b >> 52) & 0x7ff);
    unsigned long long m = (b & 0xfffffffffffffll) | (ev ? 1ull << 52 : 0ull);
    int sh = ev - e + 27;
    if (sh < 0) {
        m = sh > -64 ? m >> -sh : 0ull;
        sh = 0;
    }
    const int mask = (1 << 27) - 1, sg = (int)(b >> 63);
    s0 = ((int)(m >> (54 - sh)) ^ sg) - sg;
    s1 = (((int)(m >> (27 - sh)) & mask) ^ sg) - sg;
    s2 = (((int)((unsigned)m << sh) & mask) ^ sg) - sg;
}
__device__ __forceinline__ int exp_bits(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ double pow2(int e) {  // 2^e, clamped to the normal range
    e = e < -1022 ? -1022 : (e > 1023 ? 1023 : e);
    return __hiloint2double((e + 1023) << 20, 0);
}

// Products of row r of M0 with NO columns of X (operators o0, o0 + step, ...): the 80-bit
// fixed-point slices of both give eight 32 x 32 -> 64 bit products per entry, whose sums fit 64
// bits (ns <= 99: T0 < 2^59, T1 < 2^61, T2, T3 < 2^62); T0 counts 2^108, T1 2^81, T2 2^54, T3
// 2^27 units of 2^(er + ex - 2204).  Of (row bound) x (column bound) a product drops 2^-106, and
// what cut() leaves off an operand more than 2^-27 below its bound, at most 2^-80 each: below
// ns 2^-79 in all, 2^-72 for the largest system.
template <int NO>
__device__ __forceinline__ void row_products(int r, int ns, int n_ops, int o0, int step, int er, const double *M0,
                                             const int4 *Xs, long long (&t0)[NO], long long (&t1)[NO],
                                             long long (&t2)[NO], long long (&t3)[NO]) {
#pragma unroll
    for (int j = 0; j < NO; ++j) t0[j] = t1[j] = t2[j] = t3[j] = 0;
    int at = r * (r + 1) / 2;
    for (int q = 0; q < ns; ++q) {
        int a0, a1, a2;
        cut(M0[at], er, a0, a1, a2);
        at += q < r ? 1 : q + 1;
        const int4 *x = Xs + q * n_ops + o0;
#pragma unroll
        for (int j = 0; j < NO; ++j) {
            const int4 v = x[j * step];
            t0[j] += (long long)a0 * v.x;
            t1[j] += (long long)a0 * v.y;
            t1[j] += (long long)a1 * v.x;
            t2[j] += (long long)a0 * v.z;
            t2[j] += (long long)a1 * v.y;
            t2[j] += (long long)a2 * v.x;
            t3[j] += (long long)a1 * v.z;
            t3[j] += (long long)a2 * v.y;
        }
    }
}

// largest exponent of row r of M0
__device__ __forceinline__ int row_exponent(int r, int ns, const double *M0) {
    int er = 1, at = r * (r + 1) / 2;
    for (int q = 0; q < ns; ++q) {
        er = max(er, exp_bits(M0[at]));
        at += q < r ? 1 : q + 1;
    }
    return er;
}

// Columns of X cut into slices, ex their largest exponents.  Starts and ends with a barrier.
__device__ __forceinline__ void cut_columns(int ns, int n_ops, const double *X, int4 *Xs, int *ex) {
    const int t = threadIdx.x;
    for (int o = t; o < n_ops; o += WT) ex[o] = 1;
    __syncthreads();
    const int dr = WT / n_ops, d_o = WT - dr * n_ops;
    int o = t % n_ops;
    for (int e = t; e < ns * n_ops; e += WT) {
        atomicMax(ex + o, exp_bits(X[e]));
        o += d_o;
        if (o >= n_ops) o -= n_ops;
    }
    __syncthreads();
    o = t % n_ops;
    for (int e = t; e < ns * n_ops; e += WT) {
        int4 v;
        cut(X[e], ex[o], v.x, v.y, v.z);
        v.w = 0;
        Xs[e] = v;
        o += d_o;
        if (o >= n_ops) o -= n_ops;
    }
    __syncthreads();
}

// Entries (r, o) of R <- R - M0 X for NO operators; the difference is formed in 128 bits.
template <int NO>
__device__ __forceinline__ void residual_row(int r, int ns, int n_ops, int o0, int step, int er, const double *M0,
                                             const int4 *Xs, const int *ex, double *R) {
    long long t0[NO], t1[NO], t2[NO], t3[NO];
    row_products<NO>(r, ns, n_ops, o0, step, er, M0, Xs, t0, t1, t2, t3);
#pragma unroll
    for (int j = 0; j < NO; ++j) {
        const int o = o0 + j * step;
        const int e0 = er + ex[o] - 2096;  // T0 counts 2^e0
        const double s = R[r * n_ops + o] * pow2(-e0);
        const double fl = floor(s);
        const long long u0 = (long long)fl - t0[j];
        __int128 w = ((__int128)u0 << 54) - ((__int128)t1[j] << 27) - (__int128)t2[j];
        const bool neg = w < 0;
        if (neg) w = -w;
        double d = (double)(long long)(w >> 64) * 18446744073709551616.0 + (double)(unsigned long long)w;
        if (neg) d = -d;
        d += (s - fl) * 18014398509481984.0 - (double)t3[j] * 7.450580596923828e-9;
        R[r * n_ops + o] = d * pow2(e0 - 54);
    }
}

// f.run<NO>(row, first operator, step) over the rows and operators of a block: thread t takes
// row t mod ns and, of the ngrp = max(1, 128 / ns) threads that share a row, every ngrp-th
// operator, up to MAXO (1, 3 or 6) together
template <int MAXO, typename F>
__device__ __forceinline__ void over_rows(int ns, int n_ops, const F &f) {
    const int t = threadIdx.x, ngrp = WT / ns > 1 ? WT / ns : 1;
    const int g = t / ns, r = t - g * ns;
    if (g >= ngrp) return;
    int o = g, left = (n_ops - g + ngrp - 1) / ngrp;
    if (MAXO >= 6)
        for (; left >= 6; left -= 6, o += 6 * ngrp) f.template run<6>(r, o, ngrp);
    if (MAXO >= 3) {
        for (; left >= 3; left -= 3, o += 3 * ngrp) f.template run<3>(r, o, ngrp);
        if (left == 2) f.template run<2>(r, o, ngrp);
        if (left != 1) return;
    }
    for (; left > 0; --left, o += ngrp) f.template run<1>(r, o, ngrp);
}

struct ResidualRows {
    int ns, n_ops, er;
    const double *M0;
    const int4 *Xs;
    const int *ex;
    double *R;
    template <int NO>
    __device__ __forceinline__ void run(int r, int o, int st) const {
        residual_row<NO>(r, ns, n_ops, o, st, er, M0, Xs, ex, R);
    }
};

// R <- R - M0 X
__device__ __forceinline__ void residual(int ns, int n_ops, const double *M0, const double *X, int4 *Xs, int *ex,
                                         double *R) {
    cut_columns(ns, n_ops, X, Xs, ex);
    const int er = row_exponent(threadIdx.x % ns, ns, M0);
    over_rows<3>(ns, n_ops, ResidualRows{ns, n_ops, er, M0, Xs, ex, R});
    __syncthreads();
}

// Solve L D U X = X (row-major [ns][n_ops], rows already permuted; L and U with unit
// diagonals, rp the reciprocals of D) by the whole block, column by column: every step
// updates the (row, operator) pairs below (above) the pivot, thread t taking the pairs
// t, t + 128, ...
__device__ __forceinline__ void lu_solve(int ns, int ld, const double *M, const double *rp, double *X, int n_ops) {
    const int t = threadIdx.x;
    const int r_t = t / n_ops, o_t = t - r_t * n_ops;
    const int dr = WT / n_ops, d_o = WT - dr * n_ops;
    for (int c = 0; c < ns - 1; ++c) {
        int r = c + 1 + r_t, o = o_t;
        while (r < ns) {
            X[r * n_ops + o] -= M[r * ld + c] * X[c * n_ops + o];
            r += dr;
            o += d_o;
            if (o >= n_ops) { o -= n_ops; ++r; }
        }
        __syncthreads();
    }
    for (int r = r_t, o = o_t; r < ns;) {
        X[r * n_ops + o] *= rp[r];
        r += dr;
        o += d_o;
        if (o >= n_ops) { o -= n_ops; ++r; }
    }
    __syncthreads();
    for (int c = ns - 1; c > 0; --c) {
        int r = r_t, o = o_t;
        while (r < c) {
            X[r * n_ops + o] -= M[r * ld + c] * X[c * n_ops + o];
            r += dr;
            o += d_o;
            if (o >= n_ops) { o -= n_ops; ++r; }
        }
        __syncthreads();
    }
}

// What one system is solved for.
struct WJob {
    const double *xyz, *cxyz;
    const int32_t *cnode, *idx;
    const OpSpec *ops;
    double *w, *delta;
    int32_t *n_sing;
    int centre_is_node, n_l, k, np, n_ops;
};

// Scaled stencil coordinates xi[j][3] of centre c; the scale delta.  Ends synchronised.
__device__ __forceinline__ double stencil_coords(const WJob &J, int64_t c, double *xi) {
    const int t = threadIdx.x;
    double xc, yc, zc;
    if (J.cxyz) { xc = J.cxyz[3 * c]; yc = J.cxyz[3 * c + 1]; zc = J.cxyz[3 * c + 2]; }
    else { int64_t s = J.cnode[c]; xc = J.xyz[3 * s]; yc = J.xyz[3 * s + 1]; zc = J.xyz[3 * s + 2]; }
    for (int j = t; j < J.n_l; j += WT) {
        int64_t s = J.idx[c * J.n_l + j];
        xi[3 * j] = mimg(J.xyz[3 * s] - xc);
        xi[3 * j + 1] = mimg(J.xyz[3 * s + 1] - yc);
        xi[3 * j + 2] = mimg(J.xyz[3 * s + 2] - zc);
    }
    __syncthreads();
    const int jd = J.centre_is_node ? 1 : 0;
    const double delta = sqrt(xi[3 * jd] * xi[3 * jd] + xi[3 * jd + 1] * xi[3 * jd + 1] + xi[3 * jd + 2] * xi[3 * jd + 2]);
    if (t == 0 && J.delta) J.delta[c] = delta;
    __syncthreads();
    for (int e = t; e < 3 * J.n_l; e += WT) xi[e] /= delta;
    __syncthreads();
    return delta;
}

// The saddle matrix: packed lower triangle M0 and, in T, the full rows M (stride ld)
template <typename T>
__device__ __forceinline__ void assemble(const WJob &J, const double *xi, double *M0, T *M, int ld) {
    const int t = threadIdx.x, n_l = J.n_l, np = J.np;
    // A: pair (i, i + d mod n_l), d = 1 .. n_l / 2, each once; then P, P^T and the zero block
    const int pairs = n_l * (n_l - 1) / 2;
    const int dd = WT / n_l, di = WT - dd * n_l;
    int d = 1 + t / n_l, i = t % n_l;
    for (int e = t; e < pairs; e += WT) {
        int j = i + d;
        if (j >= n_l) j -= n_l;
        const double sx = xi[3 * i] - xi[3 * j], sy = xi[3 * i + 1] - xi[3 * j + 1], sz = xi[3 * i + 2] - xi[3 * j + 2];
        const double v = odd_pow(sx * sx + sy * sy + sz * sz, J.k);
        M[i * ld + j] = (T)v;
        M[j * ld + i] = (T)v;
        M0[tri_at(i, j)] = v;
        d += dd;
        i += di;
        if (i >= n_l) { i -= n_l; ++d; }
    }
    // the diagonal: |0|^k, or not a number when delta is 0
    const double z = xi[0] - xi[0];
    for (int r = t; r < n_l; r += WT) { M[r * ld + r] = (T)z; M0[tri_at(r, r)] = z; }
    for (int e = t; e < n_l * np; e += WT) {
        const int l = e / n_l, r = e - l * n_l;
        const double v = ipow(xi[3 * r], c_mono[l][0]) * ipow(xi[3 * r + 1], c_mono[l][1]) * ipow(xi[3 * r + 2], c_mono[l][2]);
        M[r * ld + n_l + l] = (T)v;
        M[(n_l + l) * ld + r] = (T)v;
        M0[tri_at(n_l + l, r)] = v;
    }
    for (int e = t; e < np * np; e += WT) {
        const int a = e / np, b = e - a * np;
        M[(n_l + a) * ld + n_l + b] = (T)0;
        if (b <= a) M0[tri_at(n_l + a, n_l + b)] = 0.0;
    }
}

// Right-hand sides R[r][o] (row r of operator o); off: 3 n_ops doubles of scratch, written
// before the caller's last barrier by scale_offsets
__device__ __forceinline__ void scale_offsets(const WJob &J, double delta, double *off) {
    for (int e = threadIdx.x; e < 3 * J.n_ops; e += WT) off[e] = J.ops[e / 3].off[e % 3] / delta;
}
__device__ __forceinline__ void right_hand_sides(const WJob &J, const double *xi, double delta, const double *off, double *R) {
    const int t = threadIdx.x, n_ops = J.n_ops, n_l = J.n_l, ns = n_l + J.np;
    const int dr = WT / n_ops, d_o = WT - dr * n_ops;
    int r = t / n_ops, o = t % n_ops;
    for (int e = t; e < ns * n_ops; e += WT) {
        const int kind = J.ops[o].kind;
        const double x = off[3 * o], y = off[3 * o + 1], z = off[3 * o + 2];
        R[e] = r < n_l ? rbf_rhs(kind, J.k, x - xi[3 * r], y - xi[3 * r + 1], z - xi[3 * r + 2], delta)
                       : mono_rhs(kind, c_mono[r - n_l][0], c_mono[r - n_l][1], c_mono[r - n_l][2], x, y, z, delta);
        r += dr;
        o += d_o;
        if (o >= n_ops) { o -= n_ops; ++r; }
    }
}

// One system by the block with its factors in FP64; `sm` is the block's shared memory (at
// least wlayout(n_l, np, n_ops).total doubles).
__device__ void weights_fp64(int64_t c, double *sm, const WJob &J) {
    const int t = threadIdx.x, lane = t & 31, n_l = J.n_l, n_ops = J.n_ops;
    const WLayout L = wlayout(n_l, J.np, n_ops);
    const int ns = L.ns, ld = L.ld;
    int4 *Xs = reinterpret_cast<int4 *>(sm);
    double *D = sm;                                   // permuted residual, in the slices' room
    double *M = sm + 2 * (size_t)ns * n_ops;
    double *M0 = sm + L.m0, *X = sm + L.x, *R = sm + L.r, *xi = sm + L.xi, *rp = sm + L.rp;
    int *perm = reinterpret_cast<int *>(sm + L.ints), *ex = perm + ns;
    int32_t *n_sing = J.n_sing;
    double *wout = J.w;
    for (int r = t; r < ns; r += WT) perm[r] = r;
    const double delta = stencil_coords(J, c, xi);
    scale_offsets(J, delta, sm);  // in the slices' room
    __syncthreads();
    assemble<double>(J, xi, M0, M, ld);
    right_hand_sides(J, xi, delta, sm, R);
    __syncthreads();
    // LU with partial pivoting (rows swapped in full, multipliers stored below).  Every
    // warp finds the pivot for itself: magnitudes compared as integers, not-a-numbers
    // passed over, ties to the smaller row.  The multipliers are quotients: of two equal
    // rows the second becomes exactly zero and the system is found singular, whereas
    // a * (1 / a) is 1 - 2^-53 for one pivot in seven (18 to 37 of 253 to 503 systems with
    // two coincident nodes then passed).
    bool singular = false;
    for (int col = 0; col < ns; ++col) {
        long long best = -1;
        int bi = ns;
        for (int r = col + lane; r < ns; r += 32) {
            const long long v = __double_as_longlong(M[r * ld + col]) & 0x7fffffffffffffffll;
            if (v <= 0x7ff0000000000000ll && v > best) { best = v; bi = r; }
        }
        for (int off = 16; off > 0; off >>= 1) {
            const long long ob = __shfl_xor_sync(0xffffffffu, best, off);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
            if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        if (best <= 0) { singular = true; break; }  // the same in every warp
        const double pv = M[bi * ld + col], dv = M[col * ld + col];
        const double inv = 1.0 / pv;
        __syncthreads();
        // rows col and bi change places (column col apart), and column col becomes the multipliers
        if (bi != col)
            for (int q = t; q < ns; q += WT)
                if (q != col) {
                    const double s = M[col * ld + q];
                    M[col * ld + q] = M[bi * ld + q];
                    M[bi * ld + q] = s;
                }
        for (int r = col + 1 + (WT - 1 - t); r < ns; r += WT) M[r * ld + col] = (r == bi ? dv : M[r * ld + col]) / pv;
        if (t == WT - 1) {
            M[col * ld + col] = pv;
            rp[col] = inv;
            const int s = perm[col];
            perm[col] = perm[bi];
            perm[bi] = s;
        }
        __syncthreads();
        const int n1 = ns - col - 1;
        if (n1 > 0) {
            const int dr = WT / n1, dq = WT - dr * n1;
            int r = t / n1, q = t - r * n1;
            double *T = M + (col + 1) * ld + col + 1;
            const double *Lc = M + (col + 1) * ld + col, *Ur = M + col * ld + col + 1;
            while (r < n1) {
                T[r * ld + q] -= Lc[r * ld] * Ur[q];
                r += dr;
                q += dq;
                if (q >= n1) { q -= n1; ++r; }
            }
        }
        __syncthreads();
    }
    if (singular) {
        if (t == 0) atomicAdd(n_sing, 1);
        for (int e = t; e < n_ops * n_l; e += WT) wout[c * n_ops * n_l + e] = __longlong_as_double(0x7ff8000000000000LL);
        return;
    }
    {
        const int dr = WT / n_ops, d_o = WT - dr * n_ops;
        // U to a unit diagonal: ns^2 / 2 products once instead of one more per entry and solve
        for (int r = t >> 5; r < ns - 1; r += WT / 32) {
            const double p = rp[r];
            for (int q = r + 1 + lane; q < ns; q += 32) M[r * ld + q] *= p;
        }
        int r = t / n_ops, o = t % n_ops;
        for (int e = t; e < ns * n_ops; e += WT) {
            X[e] = R[perm[r] * n_ops + o];
            r += dr;
            o += d_o;
            if (o >= n_ops) { o -= n_ops; ++r; }
        }
        __syncthreads();
        lu_solve(ns, ld, M, rp, X, n_ops);
        residual(ns, n_ops, M0, X, Xs, ex, R);
        r = t / n_ops;
        o = t % n_ops;
        for (int e = t; e < ns * n_ops; e += WT) {
            D[e] = R[perm[r] * n_ops + o];
            r += dr;
            o += d_o;
            if (o >= n_ops) { o -= n_ops; ++r; }
        }
        __syncthreads();
        lu_solve(ns, ld, M, rp, D, n_ops);
    }
    for (int e = t; e < n_ops * n_l; e += WT) {
        const int o = e / n_l, j = e - o * n_l;
        wout[(c * n_ops + o) * n_l + j] = X[j * n_ops + o] + D[j * n_ops + o];
    }
}

// ---- FP32 inverse, FP64 answers ------------------------------------------------------------
// The same systems by an FP32 inverse and iterative refinement to FP64: the residual is formed
// in integers, each correction is the FP32 inverse times it, and x in FP64 converges to the
// solution of the stored FP64 system, as the refinement of the FP64 factors does.  The
// componentwise condition numbers of stencil systems are mostly 1e2 .. 1e5 (PHS r^3, r^5), so a
// correction gains 3 to 4 digits.  An operator is done when what its last correction (from a
// full residual) leaves, that times the ratio of the last two, is below 2^-56 of its largest
// weight.  A system whose pivot falls below 1e-5 of its row, or that has not converged after MAX_ITER
// corrections, goes to the list of weights_fp64, which also decides what is singular; PHS r^7
// and up go there directly (their pivots fall to 1e-6).
//
// It takes factorisation and substitution off the FP64 pipe (2 lanes per clock and SM), which
// is then left with assembly and right-hand sides.  An inverse, not factors: elimination in
// registers reads and writes no matrix in shared memory, and a correction is a product without
// a serial chain (FP32 LU in shared memory with substitutions by warps: 30 / 43 ms for the two
// sets above).
struct FLayout {
    int ns, ld, nsp;
    size_t m0, b, x, xi, mf, rf, buf, ints, total;  // byte offsets (slices first)
};
__host__ __device__ inline FLayout flayout(int n_l, int np, int n_ops) {
    FLayout L;
    L.ns = n_l + np;
    L.ld = L.ns | 1;
    L.nsp = (L.ns + 3) & ~3;
    const size_t ns = L.ns, no = n_ops;
    L.rf = 16 * ns * no;                // rows of nsp: 16-byte loads
    L.buf = L.rf + 4 * L.nsp * no;      // two pivot columns and a pivot row, 128 entries each
    L.m0 = L.buf + 4 * 3 * 128;
    L.b = L.m0 + 8 * (ns * (ns + 1) / 2);
    L.x = L.b + 8 * ns * no;
    L.xi = L.x + 8 * ns * no;
    L.mf = L.xi + 24 * (size_t)n_l;
    L.ints = L.mf + 4 * ns * L.ld;      // piv[ns], its inverse[ns], row exponents[ns], 4 x [n_ops]
    L.total = (L.ints + 4 * (3 * ns + 4 * no) + 15) & ~(size_t)15;
    return L;
}
constexpr int MAX_ITER = 12;

// Gauss-Jordan in place with partial pivoting, no rows moved.  The matrix (ns <= 16 RT, 8 CT)
// sits in registers: thread (ty, tx) of 16 x 8 has rows ty + 16 i and columns tx + 8 j.  Per
// pivot: every warp finds it in the column in shared memory, its row's threads put the row
// there, all threads update, and the owners of the next column put it there.  Two barriers
// and RT CT multiply-adds for RT + CT loads.
//
// Row i of the tile to shared memory, with 1 in the column of elimination (at: its thread),
// and zeroed.  The comment keeps the branches of the rows apart: merged, they would index the
// tile, which then lives in local memory (a matter of speed only).
template <int RT, int CT, int I>
__device__ __forceinline__ void put_row(int i, bool at, float (&a)[RT][CT], float *row) {
    if (i == I) {
        asm volatile("// row %0" ::"n"(I));
#pragma unroll
        for (int c = 0; c < CT; ++c) {
            row[8 * c] = c == 0 && at ? 1.0f : a[I][c];
            a[I][c] = 0.0f;
        }
    } else if constexpr (I + 1 < RT) {
        put_row<RT, CT, I + 1>(i, at, a, row);
    }
}

// The eight columns in elimination are always register column 0: the tile rotates by one
// after each eight, so one copy of the code does all (a copy per register column missed the
// instruction cache).  Leaves the inverse in Mf; false: no usable pivot.
template <int RT, int CT>
__device__ __forceinline__ bool invert(int ns, int ld, const int *erow, float *Mf, float *buf, int *piv, int *inv) {
    const int t = threadIdx.x, lane = t & 31, tx = t & 7, ty = t >> 3;
    float *row = buf + 256;
    float a[RT][CT];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < CT; ++j) {
            const int r = ty + 16 * i, c = tx + 8 * j;
            a[i][j] = r < ns && c < ns ? Mf[r * ld + c] : 0.0f;
        }
    if (tx == 0) {
#pragma unroll
        for (int i = 0; i < RT; ++i) buf[ty + 16 * i] = a[i][0];
    }
    unsigned used = 0;
    int turn = 0;  // register column j holds columns 8 ((j + turn) mod CT) ..
    __syncthreads();
#pragma unroll 1
    for (int k = 0; k < ns; ++k) {
        const int kk = k & 7;
        const float *col = buf + 128 * (k & 1);
        float *next = buf + 128 * (~k & 1);
        unsigned key = 0;  // magnitude to 17 bits, and the row
#pragma unroll
        for (int q = 0; q < (RT + 1) / 2; ++q) {
            const int r = lane + 32 * q;
            if (r < ns && !(used >> q & 1)) key = max(key, (__float_as_uint(col[r]) & 0x7fffff80u) | r);
        }
        key = __reduce_max_sync(0xffffffffu, key);
        const int p = key & 127;
        if ((p & 31) == lane) used |= 1u << (p >> 5);
        if (ty == (p & 15)) put_row<RT, CT, 0>(p >> 4, tx == kk, a, row + tx);
        if (t == 0) {
            piv[k] = p;
            inv[p] = k;
        }
        // zero, not a number, or small beside its row (whose entries are below 2^(erow - 1022))
        if (key < 128 || key >= 0x7f800000u ||
            __uint_as_float(key) < 1e-5f * __int_as_float(max(1, min(254, erow[p] - 895)) << 23)) return false;
        const float iv = __fdividef(1.0f, col[p]);
        float f[RT];  // the pivot row becomes 0 + row / pivot, its column 0 - f / pivot
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            f[i] = (ty + 16 * i == p ? -1.0f : col[ty + 16 * i]) * iv;
            if (tx == kk) a[i][0] = 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < CT; ++c) {
            const float v = row[tx + 8 * c];
#pragma unroll
            for (int i = 0; i < RT; ++i) a[i][c] -= f[i] * v;
        }
        if (kk == 7) {
            turn = turn + 1 < CT ? turn + 1 : 0;
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const float s = a[i][0];
#pragma unroll
                for (int c = 0; c + 1 < CT; ++c) a[i][c] = a[i][c + 1];
                a[i][CT - 1] = s;
            }
        }
        if (tx == ((k + 1) & 7)) {
#pragma unroll
            for (int i = 0; i < RT; ++i) next[ty + 16 * i] = a[i][0];
        }
        __syncthreads();
    }
    // row p of the array belongs to unknown inv[p], column c to equation piv[c]
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < CT; ++j) {
            const int r = ty + 16 * i, b = j + turn, c = tx + 8 * (b < CT ? b : b - CT);
            if (r < ns && c < ns) Mf[inv[r] * ld + piv[c]] = a[i][j];
        }
    __syncthreads();
    return true;
}

// The pieces of an iteration, each over the same (row, operators) of a thread.  Rf and Xs are
// by operator, X and B by row.
struct Fast {
    int ns, nsp, ld, n_l, n_ops, er;
    unsigned peers;  // lanes of this warp in the same group of rows
    const double *M0, *B;
    double *X;
    int4 *Xs;
    float *Mf, *Rf;
    int *sc, *ex, *ew, *ed;
    __device__ __forceinline__ bool leads() const { return (int)(threadIdx.x & 31) == __ffs(peers) - 1; }
};

// the size of the right-hand sides
struct Scale : Fast {
    template <int NO>
    __device__ __forceinline__ void run(int r, int o, int st) const {
        for (int j = 0; j < NO; ++j, o += st) {
            X[r * n_ops + o] = 0.0;
            const int e = __reduce_max_sync(peers, exp_bits(B[r * n_ops + o]));
            if (leads()) atomicMax(sc + o, e);
        }
    }
};
// x = 0: the first residual is the right-hand side
struct First : Fast {
    template <int NO>
    __device__ __forceinline__ void run(int r, int o, int st) const {
        for (int j = 0; j < NO; ++j, o += st) Rf[o * nsp + r] = (float)(B[r * n_ops + o] * pow2(1022 - sc[o]));
    }
};

// X += Mf Rf 2^(sc - 1022); the largest exponents of X (ex), of the weights (ew) and of their
// corrections (ed) per operator
struct Correct : Fast {
    template <int NO>
    __device__ __forceinline__ void run(int r, int o, int st) const {
        float d[NO];
#pragma unroll
        for (int j = 0; j < NO; ++j) d[j] = 0.0f;
        const float *m = Mf + r * ld, *b = Rf + o * nsp;
        const int step = st * nsp;
        int c = 0;
#pragma unroll 1
        for (; c + 4 <= ns; c += 4) {
            const float m0 = m[c], m1 = m[c + 1], m2 = m[c + 2], m3 = m[c + 3];
#pragma unroll
            for (int j = 0; j < NO; ++j) {
                const float4 v = *reinterpret_cast<const float4 *>(b + j * step + c);
                d[j] += m0 * v.x;
                d[j] += m1 * v.y;
                d[j] += m2 * v.z;
                d[j] += m3 * v.w;
            }
        }
#pragma unroll 1
        for (; c < ns; ++c)
#pragma unroll
            for (int j = 0; j < NO; ++j) d[j] += m[c] * b[j * step + c];
        const bool first = leads();
#pragma unroll
        for (int j = 0; j < NO; ++j, o += st) {
            const double dd = (double)d[j] * pow2(sc[o] - 1022), x = X[r * n_ops + o] + dd;
            X[r * n_ops + o] = x;
            const int e = exp_bits(x), w = r < n_l ? e : 0, q = r < n_l ? exp_bits(dd) : 0;
            const int me = __reduce_max_sync(peers, e), mw = __reduce_max_sync(peers, w), mq = __reduce_max_sync(peers, q);
            if (first) {
                atomicMax(ex + o, me);
                atomicMax(ew + o, mw);
                atomicMax(ed + o, mq);
            }
        }
    }
};

// X into slices
struct Cut : Fast {
    template <int NO>
    __device__ __forceinline__ void run(int r, int o, int st) const {
#pragma unroll 1
        for (int j = 0; j < NO; ++j, o += st) {
            int4 v;
            cut(X[r * n_ops + o], max(ex[o], 1), v.x, v.y, v.z);
            v.w = 0;
            Xs[o * ns + r] = v;
        }
    }
};

// B - (2^108 t0 + 2^81 t1 + 2^54 t2) 2^(er + ex - 2204) to FP32, as a multiple of 2^(ex - 1022)
__device__ __noinline__ float difference(double B, long long t0, long long t1, long long t2, int er, int ex) {
    // in t2's units: B = m 2^(eb - 1075)
    const long long bb = __double_as_longlong(B);
    const int eb = (int)((bb >> 52) & 0x7ff);
    const long long m = (bb & 0xfffffffffffffll) | (eb ? 1ll << 52 : 0ll);
    const int sh = (eb ? eb : 1) - 1075 - (er + ex - 2150);
    __int128 w = sh >= 0 ? (__int128)m << min(sh, 73) : (__int128)(sh > -63 ? m >> -sh : 0ll);
    if (bb < 0) w = -w;
    w -= ((__int128)t0 << 54) + ((__int128)t1 << 27) + (__int128)t2;
    const bool neg = w < 0;
    if (neg) w = -w;
    const unsigned long long hi = (unsigned long long)(w >> 64), lo = (unsigned long long)w;
    const int z = hi ? __clzll((long long)hi) : (lo ? 64 + __clzll((long long)lo) : 127);
    const unsigned top = (unsigned)(((unsigned __int128)w << z) >> 96);  // the leading 32 bits
    const int e = 96 - z + er - 1128;  // top 2^(96 - z) units of 2^(er - 1128) 2^(ex - 1022)
    const float f = (float)top * __int_as_float((max(min(e, 90), -120) + 127) << 23);
    return neg ? -f : f;
}

// Rf <- B - M0 X as multiples of 2^(ex - 1022) (about the size of X's column), in integers up
// to the conversion.  FULL: three levels of slice products; what is dropped (two products below
// 2^-79 of (row bound) x (column bound) per term, and what cut() leaves off small operands) stays
// below ns 2^-77.4, 2^-71 for the largest system.  Times a componentwise condition of 1e5 that is
// 2^-54 of the operator's largest weight at worst (2^-48 for the worst r^5 systems of 64 nodes,
// 6e6).  Measured against 113-bit arithmetic over N_L = 20 .. 64 (r^3 and r^5, 1,300 systems): the
// root mean square error is 25 % below that of FP64 LU with one compensated refinement, the
// largest error of a weight relative to itself at or below it, and that of weights below 1e-4 of the
// largest as well (the rounding of the stored matrix decides all of them).  Otherwise two levels,
// 2^-53: all that the first x needs.
template <bool FULL>
struct Residual32 : Fast {
    template <int NO>
    __device__ __forceinline__ void run(int r, int o, int st) const {
        long long t0[NO], t1[NO], t2[NO];
#pragma unroll
        for (int j = 0; j < NO; ++j) t0[j] = t1[j] = t2[j] = 0;
        const int step = st * ns;
        const int4 *x = Xs + o * ns;
        int at = r * (r + 1) / 2;
#pragma unroll 2
        for (int q = 0; q < ns; ++q) {
            int a0, a1, a2;
            cut(M0[at], er, a0, a1, a2);
            at += q < r ? 1 : q + 1;
#pragma unroll
            for (int j = 0; j < NO; ++j) {
                const int4 v = x[j * step + q];
                t0[j] += (long long)a0 * v.x;
                t1[j] += (long long)a1 * v.x;
                t1[j] += (long long)a0 * v.y;
                if (FULL) {
                    t2[j] += (long long)a0 * v.z;
                    t2[j] += (long long)a1 * v.y;
                    t2[j] += (long long)a2 * v.x;
                }
            }
        }
#pragma unroll
        for (int j = 0; j < NO; ++j, o += st)
            Rf[o * nsp + r] = difference(B[r * n_ops + o], t0[j], t1[j], t2[j], er, sc[o]);
    }
};

// false: the system is for weights_fp64
template <int RT, int CT>
__device__ __forceinline__ bool weights_fast(int64_t c, unsigned char *sm, const WJob &J) {
    const int t = threadIdx.x, n_l = J.n_l, n_ops = J.n_ops;
    const FLayout L = flayout(n_l, J.np, n_ops);
    const int ns = L.ns, ld = L.ld;
    double *B = reinterpret_cast<double *>(sm + L.b), *M0 = reinterpret_cast<double *>(sm + L.m0);
    double *xi = reinterpret_cast<double *>(sm + L.xi);
    int *piv = reinterpret_cast<int *>(sm + L.ints), *inv = piv + ns, *erow = inv + ns;
    Fast F;
    F.ns = ns; F.nsp = L.nsp; F.ld = ld; F.n_l = n_l; F.n_ops = n_ops;
    F.peers = __match_any_sync(0xffffffffu, t / ns);
    F.M0 = M0; F.B = B;
    F.X = reinterpret_cast<double *>(sm + L.x);
    F.Xs = reinterpret_cast<int4 *>(sm);
    F.Mf = reinterpret_cast<float *>(sm + L.mf); F.Rf = reinterpret_cast<float *>(sm + L.rf);
    F.sc = erow + ns; F.ex = F.sc + n_ops; F.ew = F.ex + n_ops; F.ed = F.ew + n_ops;
    const double delta = stencil_coords(J, c, xi);
    scale_offsets(J, delta, reinterpret_cast<double *>(sm));  // in the slices' room
    if (t < n_ops) {
        F.sc[t] = 1;
        F.ex[t] = F.ew[t] = F.ed[t] = 0;
    }
    __syncthreads();
    assemble<float>(J, xi, M0, F.Mf, ld);
    right_hand_sides(J, xi, delta, reinterpret_cast<double *>(sm), B);
    __syncthreads();
    F.er = row_exponent(t % ns, ns, M0);
    if (t < ns) erow[t] = F.er;
    over_rows<1>(ns, n_ops, Scale{F});
    __syncthreads();
    over_rows<1>(ns, n_ops, First{F});
    if (!invert<RT, CT>(ns, ld, erow, F.Mf, reinterpret_cast<float *>(sm + L.buf), piv, inv)) return false;
    int last = 0;  // exponent of operator t's last correction
    for (int it = 0;; ++it) {
        over_rows<6>(ns, n_ops, Correct{F});
        __syncthreads();
        // the next correction is about this one times its ratio to the one before
        bool done = it >= 2;
        if (t < n_ops) {
            const int d = F.ed[t], w = F.ew[t];
            done &= d + 38 <= w && 2 * d - last + 58 <= w && w < 2047;
            last = d;
        }
        if (__syncthreads_and(done)) break;
        if (it == MAX_ITER - 1) return false;
        over_rows<1>(ns, n_ops, Cut{F});
        if (t < n_ops) F.sc[t] = max(F.ex[t], 1);
        __syncthreads();
        if (it == 0) over_rows<6>(ns, n_ops, Residual32<false>{F});
        else over_rows<6>(ns, n_ops, Residual32<true>{F});
        if (t < n_ops) F.ex[t] = F.ew[t] = F.ed[t] = 0;
        __syncthreads();
    }
    for (int e = t; e < n_ops * n_l; e += WT) {
        const int o = e / n_l, j = e - o * n_l;
        J.w[(c * n_ops + o) * n_l + j] = F.X[j * n_ops + o];
    }
    return true;
}

// Systems by number: one stencil set, or the concatenation of many (e.g. the nodes of many
// cells, each with its own N_L).
struct WSet {
    WJob job;                 // one set; n_l and the pointers of `jobs` otherwise
    const WeightJob *jobs;    // null: one set
    const int64_t *prefix;
    int njobs;
};
__device__ __forceinline__ int64_t pick(const WSet &S, int64_t t, WJob &J) {
    J = S.job;
    if (!S.jobs) return t;
    int j = 0;
    while (j + 1 < S.njobs && S.prefix[j + 1] <= t) ++j;
    const WeightJob jb = S.jobs[j];
    J.xyz = jb.xyz; J.cxyz = nullptr; J.cnode = jb.cnode; J.idx = jb.idx; J.w = jb.w; J.delta = jb.delta;
    J.n_l = jb.n_l; J.centre_is_node = 1;
    return t - S.prefix[j];
}

// list[0]: number of systems put on the list list[1 ..] for k_weights
template <int RT, int CT>
__global__ void __launch_bounds__(WT, RT > 4 ? 3 : 5) k_weights_fast(WSet S, int32_t *list) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WJob J;
    const int64_t c = pick(S, blockIdx.x, J);
    const bool ok = weights_fast<RT, CT>(c, smem_raw, J);
    if (!ok && threadIdx.x == 0) list[1 + atomicAdd(list, 1)] = (int32_t)blockIdx.x;
}

// The systems of the list, or all ntot
__global__ void __launch_bounds__(WT) k_weights(WSet S, int64_t ntot, const int32_t *__restrict__ list) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t n = list ? list[0] : ntot;
    for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
        WJob J;
        const int64_t c = pick(S, list ? list[1 + i] : i, J);
        weights_fp64(c, reinterpret_cast<double *>(smem_raw), J);
        __syncthreads();
    }
}

// A kernel's shared-memory limit is one for all threads of the program, so it is always set to
// the same value, the largest system's: with each launch's own, another thread's smaller one
// in between made the launch fail.
cudaError_t set_limit(const void *kern, size_t bytes) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

cudaError_t launch_set(const WSet &S, int64_t ntot, int max_n_l, int k, int np, int n_ops, int32_t *list, cudaStream_t st) {
    const size_t smem = wlayout(max_n_l, np, n_ops).total * sizeof(double);
    cudaError_t e = set_limit((const void *)k_weights, wlayout(RBF_MAX_NL, RBF_MAX_NP, RBF_MAX_OPS).total * sizeof(double));
    if (e != cudaSuccess) return e;
    if (k > 5) {
        k_weights<<<(unsigned)ntot, WT, smem, st>>>(S, ntot, nullptr);
        return cudaGetLastError();
    }
    const size_t fsmem = flayout(max_n_l, np, n_ops).total;
    // the smallest register tile that holds the system
    const int ns = max_n_l + np;
    auto *kern = ns <= 48 ? k_weights_fast<3, 6> : ns <= 64 ? k_weights_fast<4, 8> : k_weights_fast<7, 13>;
    e = set_limit((const void *)kern, flayout(RBF_MAX_NL, RBF_MAX_NP, RBF_MAX_OPS).total);
    if (e == cudaSuccess) e = cudaMemsetAsync(list, 0, sizeof(int32_t), st);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)ntot, WT, fsmem, st>>>(S, list);
    k_weights<<<(unsigned)std::min<int64_t>(ntot, 608), WT, smem, st>>>(S, ntot, list);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_weights_multi(int njobs, const WeightJob *jobs_dev, const int64_t *prefix_dev, int64_t ntot,
                                 int max_n_l, int k, int m, int n_ops, const OpSpec *ops, int32_t *n_sing, int32_t *list,
                                 cudaStream_t st) {
    if (ntot <= 0) return cudaSuccess;
    if (n_ops < 1 || n_ops > RBF_MAX_OPS || max_n_l < 2 || max_n_l > RBF_MAX_NL || m < 0 || m > 4) return cudaErrorInvalidValue;
    const int np = (m + 1) * (m + 2) * (m + 3) / 6;
    WSet S;
    S.job = WJob{nullptr, nullptr, nullptr, nullptr, ops, nullptr, nullptr, n_sing, 1, max_n_l, k, np, n_ops};
    S.jobs = jobs_dev;
    S.prefix = prefix_dev;
    S.njobs = njobs;
    return launch_set(S, ntot, max_n_l, k, np, n_ops, list, st);
}

cudaError_t launch_weights(int64_t nc, const double *xyz, const double *cxyz, const int32_t *cnode,
                           int centre_is_node, int n_l, const int32_t *idx, int k, int m, int n_ops,
                           const OpSpec *ops, double *w, double *delta, int32_t *n_sing, int32_t *list, cudaStream_t st) {
    if (nc <= 0) return cudaSuccess;
    if (n_ops < 1 || n_ops > RBF_MAX_OPS || n_l < 2 || n_l > RBF_MAX_NL || m < 0 || m > 4) return cudaErrorInvalidValue;
    const int np = (m + 1) * (m + 2) * (m + 3) / 6;
    WSet S;
    S.job = WJob{xyz, cxyz, cnode, idx, ops, w, delta, n_sing, centre_is_node, n_l, k, np, n_ops};
    S.jobs = nullptr;
    S.prefix = nullptr;
    S.njobs = 0;
    return launch_set(S, nc, n_l, k, np, n_ops, list, st);
}

// ---- FP32 copies of the weights ---------------------------------------------
// Each row of n_l FP64 weights (one operator at one centre) is rounded to FP32 so
// that the exact sum of the FP32 values stays at the FP64 row sum: every weight is
// rounded to nearest, then the sum's residual is added to the smallest-magnitude
// nonzero weight, which is rounded again (its ulp bounds what is left).  Plain
// rounding leaves each row sum off by ~1e-7 of its weights' size, so constants
// are no longer reproduced (interpolation rows no longer sum to 1, derivative
// rows no longer to 0); the explicit iterations carry that error in every step
// and in the MLBM it biased the steady permeability by 2e-4 on the 150k-node cell.
// out holds the FP32 values as doubles (exactly representable), rows as in w.
__global__ void k_round_rows_f32(int64_t nrows, int n_l, const double *__restrict__ w, double *__restrict__ out) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= nrows) return;
    const double *a = w + r * n_l;
    double *o = out + r * n_l;
    double s64 = 0.0, s32 = 0.0, amin = 0.0;
    int jmin = -1;
    for (int j = 0; j < n_l; ++j) {
        const float f = (float)a[j];
        s64 += a[j];
        s32 += (double)f;
        o[j] = (double)f;
        if (f != 0.0f && (jmin < 0 || fabs((double)f) < amin)) { amin = fabs((double)f); jmin = j; }
    }
    if (jmin >= 0) o[jmin] = (double)(float)(o[jmin] + (s64 - s32));
}

cudaError_t launch_round_rows_f32(int64_t nrows, int n_l, const double *w, double *out, cudaStream_t st) {
    if (nrows == 0) return cudaSuccess;
    k_round_rows_f32<<<(unsigned)((nrows + 255) / 256), 256, 0, st>>>(nrows, n_l, w, out);
    return cudaGetLastError();
}

// wall normal-derivative rows w^n_j = n_x w^x_j + n_y w^y_j + n_z w^z_j (FP64,
// [nb][n_l]) from the gradient weights of the wall nodes' Neumann stencils
__global__ void k_normal_rows(int64_t nb, int n_l, const int32_t *__restrict__ wall, const double *__restrict__ nrm,
                              const double *__restrict__ wg, double *__restrict__ out) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= nb * n_l) return;
    int64_t b = t / n_l;
    int j = (int)(t - b * n_l);
    int64_t i = wall[b];
    const double *g = wg + b * 3 * n_l;
    double nx = nrm[3 * i], ny = nrm[3 * i + 1], nz = nrm[3 * i + 2];
    out[t] = __dadd_rn(__dadd_rn(__dmul_rn(nx, g[j]), __dmul_rn(ny, g[n_l + j])), __dmul_rn(nz, g[2 * n_l + j]));
}

cudaError_t launch_normal_rows(int64_t nb, int n_l, const int32_t *wall, const double *nrm, const double *wg,
                               double *out, cudaStream_t st) {
    int64_t tot = nb * n_l;
    if (tot == 0) return cudaSuccess;
    k_normal_rows<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(nb, n_l, wall, nrm, wg, out);
    return cudaGetLastError();
}

// ---- packing into SELL-C slices for the step kernels ------------------------
template <typename T>
__global__ void k_pack(int64_t nc, int n_ops, int o0, int n_out, int n_l, const double *__restrict__ w, T *ws) {
    // one thread per (centre, j); centres beyond nc (the last slice's padding) get 0
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t npad = (nc + 31) & ~31LL;
    if (t >= npad * n_l) return;
    int64_t c = t / n_l;
    int j = (int)(t - c * n_l);
    int64_t s = c >> 5;
    int lane = (int)(c & 31);
    for (int o = 0; o < n_out; ++o)
        ws[sell_at(s, o, j, lane, n_out, n_l)] = c < nc ? (T)w[(c * n_ops + o0 + o) * n_l + j] : (T)0;
}

cudaError_t launch_pack_f32(int64_t nc, int n_ops, int o0, int n_out, int n_l, const double *w, float *ws,
                            cudaStream_t st) {
    int64_t tot = ((nc + 31) & ~31LL) * n_l;
    if (tot == 0) return cudaSuccess;
    k_pack<float><<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(nc, n_ops, o0, n_out, n_l, w, ws);
    return cudaGetLastError();
}
cudaError_t launch_pack_f64(int64_t nc, int n_ops, int o0, int n_out, int n_l, const double *w, double *ws,
                            cudaStream_t st) {
    int64_t tot = ((nc + 31) & ~31LL) * n_l;
    if (tot == 0) return cudaSuccess;
    k_pack<double><<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(nc, n_ops, o0, n_out, n_l, w, ws);
    return cudaGetLastError();
}

__global__ void k_pack_idx(int64_t nc, int n_l, const int32_t *__restrict__ idx, int32_t *is) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t npad = (nc + 31) & ~31LL;
    if (t >= npad * n_l) return;
    int64_t c = t / n_l;
    int j = (int)(t - c * n_l);
    is[sell_at(c >> 5, 0, j, (int)(c & 31), 1, n_l)] = c < nc ? idx[c * n_l + j] : 0;
}

cudaError_t launch_pack_idx(int64_t nc, int n_l, const int32_t *idx, int32_t *is, cudaStream_t st) {
    int64_t tot = ((nc + 31) & ~31LL) * n_l;
    if (tot == 0) return cudaSuccess;
    k_pack_idx<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(nc, n_l, idx, is);
    return cudaGetLastError();
}

// wall normal-derivative weights w^n_j = n_x w^x_j + n_y w^y_j + n_z w^z_j (FP64),
// from the gradient weights of the wall nodes' Neumann stencils
template <typename T>
__global__ void k_pack_normal(int64_t nb, int n_l, const int32_t *__restrict__ wall, const double *__restrict__ nrm,
                              const double *__restrict__ wg, T *ws) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t npad = (nb + 31) & ~31LL;
    if (t >= npad * n_l) return;
    int64_t b = t / n_l;
    int j = (int)(t - b * n_l);
    T v = (T)0;
    if (b < nb) {
        int64_t i = wall[b];
        const double *g = wg + b * 3 * n_l;
        double nx = nrm[3 * i], ny = nrm[3 * i + 1], nz = nrm[3 * i + 2];
        v = (T)(__dadd_rn(__dadd_rn(__dmul_rn(nx, g[j]), __dmul_rn(ny, g[n_l + j])), __dmul_rn(nz, g[2 * n_l + j])));
    }
    ws[sell_at(b >> 5, 0, j, (int)(b & 31), 1, n_l)] = v;
}

cudaError_t launch_pack_normal_f32(int64_t nb, int n_l, const int32_t *wall, const double *nrm,
                                   const double *wg, float *ws, cudaStream_t st) {
    int64_t tot = ((nb + 31) & ~31LL) * n_l;
    if (tot == 0) return cudaSuccess;
    k_pack_normal<float><<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(nb, n_l, wall, nrm, wg, ws);
    return cudaGetLastError();
}
cudaError_t launch_pack_normal_f64(int64_t nb, int n_l, const int32_t *wall, const double *nrm,
                                   const double *wg, double *ws, cudaStream_t st) {
    int64_t tot = ((nb + 31) & ~31LL) * n_l;
    if (tot == 0) return cudaSuccess;
    k_pack_normal<double><<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(nb, n_l, wall, nrm, wg, ws);
    return cudaGetLastError();
}

}  // namespace rbf
