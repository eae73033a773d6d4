// weights.cu — RBF-FD stencil weights, batched: one block of 128 threads per stencil.
//
// For every centre x_c with stencil S (N_L nodes) the block assembles the saddle
// system of Eq. augmentedSystem in shared memory, FP64:
//   A_jl = |xi_j - xi_l|^k      (PHS r^k, Eq. rbfScaling: xi = (x - x_c) / delta)
//   P_jl = p_l(xi_j)            (monomials of degree <= m, graded lexicographic)
//   M = [[A, P], [P^T, 0]]
// factors it by LU with partial pivoting, and solves the right-hand sides of up to
// RBF_MAX_OPS operators L (Eq. operatorApprox) together:
//   b_j = (L Phi_j)(y), c_l = (L p_l)(y),  y = x_c + off
// followed by one step of iterative refinement with an exactly accumulated residual.
// delta is the distance to the nearest other node (centre is a node) or to the
// nearest node (centre is a free point such as a permeability probe).
//
// What bounds it: the FP64 pipe (2 lanes per clock and SM, 1/64 of the FP32 rate),
// so the design counts FP64 operations.
//  * The residual, which has to carry about twice the working precision, runs on
//    the integer pipe: rows of M and columns of x are cut into three 26/27-bit
//    slices relative to the row's (column's) largest exponent, eight 32 x 32 -> 64
//    bit multiply-adds per product accumulate exactly (residual()).  A compensated
//    FP64 dot product (ten FP64 operations per product) was two thirds of the FP64
//    work of an 18-operator system.
//  * One reciprocal per pivot instead of a division per row and right-hand side; each
//    distance of the symmetric A computed once.
//  * Updates run over (row, column) pairs packed over the block's threads with
//    incremental indices (no integer division), so warps stay full at small sizes.
//  * The untouched matrix is kept as a packed lower triangle and the residual's
//    buffers are reused, which leaves 4-5 blocks (16-20 warps) per SM at N_L = 30..40.
// Measured (GB300, 2070 MHz): 86,397 systems of n = 60 with 4 operators (N_L = 40, r^5,
// m = 3) 34.4 ms, 120,840 systems of n = 40 with 18 operators (N_L = 30, r^3, m = 2)
// 33.5 ms, the FP64 pipe 81-87 % busy; one warp per system with the compensated product
// took 164 and 167 ms.
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

// Entry (r, o) of R - M0 X for NO operators o = o0, o0 + step, ...: the 80-bit fixed-point slices
// of a row of M0 and of the columns of X give products whose sums fit 64 bits (ns <= 99:
// T0 < 2^59, T1 < 2^61, T2, T3 < 2^62), so only terms below 2^-108 of (row maximum) x
// (column maximum) are dropped; the difference to R is formed in 128 bits.
template <int NO>
__device__ __forceinline__ void residual_row(int r, int ns, int n_ops, int o0, int step, int er, const double *M0,
                                             const int4 *Xs, const int *ex, double *R) {
    long long t0[NO], t1[NO], t2[NO], t3[NO];
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

// R <- R - M0 X.  Thread t takes row t mod ns and, of the ngrp = max(1, 128 / ns) threads
// that share a row, every ngrp-th operator.
__device__ __forceinline__ void residual(int ns, int n_ops, const double *M0, const double *X, int4 *Xs, int *ex,
                                         double *R) {
    const int t = threadIdx.x;
    for (int o = t; o < n_ops; o += WT) ex[o] = 1;
    __syncthreads();
    {
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
    const int ngrp = WT / ns > 1 ? WT / ns : 1;
    const int g = t / ns, r = t - g * ns;
    if (g < ngrp) {
        int er = 1, at = r * (r + 1) / 2;
        for (int q = 0; q < ns; ++q) {
            er = max(er, exp_bits(M0[at]));
            at += q < r ? 1 : q + 1;
        }
        int o = g;
        for (; o + 2 * ngrp < n_ops; o += 3 * ngrp) residual_row<3>(r, ns, n_ops, o, ngrp, er, M0, Xs, ex, R);
        for (; o < n_ops; o += ngrp) residual_row<1>(r, ns, n_ops, o, ngrp, er, M0, Xs, ex, R);
    }
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

// One stencil's saddle system and its right-hand sides, by one block; `sm` is the
// block's shared memory (at least wlayout(n_l, np, n_ops).total doubles).
__device__ void weights_one(int64_t c, double *sm, const double *__restrict__ xyz, const double *__restrict__ cxyz,
                            const int32_t *__restrict__ cnode, int centre_is_node, int n_l,
                            const int32_t *__restrict__ idx, int k, int np, int n_ops,
                            const OpSpec *__restrict__ ops, double *__restrict__ wout,
                            double *__restrict__ delta_out, int32_t *n_sing) {
    const int t = threadIdx.x, lane = t & 31;
    const WLayout L = wlayout(n_l, np, n_ops);
    const int ns = L.ns, ld = L.ld;
    int4 *Xs = reinterpret_cast<int4 *>(sm);
    double *D = sm;                                   // permuted residual, in the slices' room
    double *M = sm + 2 * (size_t)ns * n_ops;
    double *M0 = sm + L.m0, *X = sm + L.x, *R = sm + L.r, *xi = sm + L.xi, *rp = sm + L.rp;
    int *perm = reinterpret_cast<int *>(sm + L.ints), *ex = perm + ns;

    double xc, yc, zc;
    if (cxyz) { xc = cxyz[3 * c]; yc = cxyz[3 * c + 1]; zc = cxyz[3 * c + 2]; }
    else { int64_t s = cnode[c]; xc = xyz[3 * s]; yc = xyz[3 * s + 1]; zc = xyz[3 * s + 2]; }
    for (int j = t; j < n_l; j += WT) {
        int64_t s = idx[c * n_l + j];
        xi[3 * j] = mimg(xyz[3 * s] - xc);
        xi[3 * j + 1] = mimg(xyz[3 * s + 1] - yc);
        xi[3 * j + 2] = mimg(xyz[3 * s + 2] - zc);
    }
    for (int r = t; r < ns; r += WT) perm[r] = r;
    __syncthreads();
    const int jd = centre_is_node ? 1 : 0;
    const double delta = sqrt(xi[3 * jd] * xi[3 * jd] + xi[3 * jd + 1] * xi[3 * jd + 1] + xi[3 * jd + 2] * xi[3 * jd + 2]);
    if (t == 0 && delta_out) delta_out[c] = delta;
    __syncthreads();
    double *off = sm;  // scaled offsets of the operators, in the slices' room
    for (int e = t; e < 3 * n_l; e += WT) xi[e] /= delta;
    for (int e = t; e < 3 * n_ops; e += WT) off[e] = ops[e / 3].off[e % 3] / delta;
    __syncthreads();
    // A: pair (i, i + d mod n_l), d = 1 .. n_l / 2, each once; then P, P^T and the zero block
    {
        const int pairs = n_l * (n_l - 1) / 2;
        const int dd = WT / n_l, di = WT - dd * n_l;
        int d = 1 + t / n_l, i = t % n_l;
        for (int e = t; e < pairs; e += WT) {
            int j = i + d;
            if (j >= n_l) j -= n_l;
            const double sx = xi[3 * i] - xi[3 * j], sy = xi[3 * i + 1] - xi[3 * j + 1], sz = xi[3 * i + 2] - xi[3 * j + 2];
            const double v = odd_pow(sx * sx + sy * sy + sz * sz, k);
            M[i * ld + j] = v;
            M[j * ld + i] = v;
            M0[tri_at(i, j)] = v;
            d += dd;
            i += di;
            if (i >= n_l) { i -= n_l; ++d; }
        }
        // the diagonal: |0|^k, or not a number when delta is 0
        const double z = xi[0] - xi[0];
        for (int r = t; r < n_l; r += WT) { M[r * ld + r] = z; M0[tri_at(r, r)] = z; }
        for (int e = t; e < n_l * np; e += WT) {
            const int l = e / n_l, r = e - l * n_l;
            const double v = ipow(xi[3 * r], c_mono[l][0]) * ipow(xi[3 * r + 1], c_mono[l][1]) * ipow(xi[3 * r + 2], c_mono[l][2]);
            M[r * ld + n_l + l] = v;
            M[(n_l + l) * ld + r] = v;
            M0[tri_at(n_l + l, r)] = v;
        }
        for (int e = t; e < np * np; e += WT) {
            const int a = e / np, b = e - a * np;
            M[(n_l + a) * ld + n_l + b] = 0.0;
            if (b <= a) M0[tri_at(n_l + a, n_l + b)] = 0.0;
        }
    }
    // right-hand sides R[r][o] (row r of operator o)
    {
        const int dr = WT / n_ops, d_o = WT - dr * n_ops;
        int r = t / n_ops, o = t % n_ops;
        for (int e = t; e < ns * n_ops; e += WT) {
            const int kind = ops[o].kind;
            const double x = off[3 * o], y = off[3 * o + 1], z = off[3 * o + 2];
            R[e] = r < n_l ? rbf_rhs(kind, k, x - xi[3 * r], y - xi[3 * r + 1], z - xi[3 * r + 2], delta)
                           : mono_rhs(kind, c_mono[r - n_l][0], c_mono[r - n_l][1], c_mono[r - n_l][2], x, y, z, delta);
            r += dr;
            o += d_o;
            if (o >= n_ops) { o -= n_ops; ++r; }
        }
    }
    __syncthreads();
    // LU with partial pivoting (rows swapped in full, multipliers stored below).  Every
    // warp finds the pivot for itself: magnitudes compared as integers, not-a-numbers
    // passed over, ties to the smaller row.
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
        for (int r = col + 1 + (WT - 1 - t); r < ns; r += WT) M[r * ld + col] = (r == bi ? dv : M[r * ld + col]) * inv;
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

__global__ void __launch_bounds__(WT) k_weights(int64_t nc, const double *__restrict__ xyz, const double *__restrict__ cxyz,
                          const int32_t *__restrict__ cnode, int centre_is_node, int n_l,
                          const int32_t *__restrict__ idx, int k, int np, int n_ops,
                          const OpSpec *__restrict__ ops, double *__restrict__ wout,
                          double *__restrict__ delta_out, int32_t *n_sing) {
    extern __shared__ __align__(16) double smem[];
    weights_one(blockIdx.x, smem, xyz, cxyz, cnode, centre_is_node, n_l, idx, k, np, n_ops, ops, wout, delta_out, n_sing);
}

// Many stencil sets (e.g. the nodes of many cells, each with its own N_L) in one
// launch: block t solves centre t of the concatenation of the jobs.
__global__ void __launch_bounds__(WT) k_weights_multi(int njobs, const WeightJob *__restrict__ jobs,
                                const int64_t *__restrict__ prefix, int k, int np, int n_ops,
                                const OpSpec *__restrict__ ops, int32_t *n_sing) {
    extern __shared__ __align__(16) double smem[];
    const int64_t t = blockIdx.x;
    int j = 0;
    while (j + 1 < njobs && prefix[j + 1] <= t) ++j;
    const WeightJob jb = jobs[j];
    weights_one(t - prefix[j], smem, jb.xyz, nullptr, jb.cnode, 1, jb.n_l, jb.idx, k, np, n_ops, ops, jb.w, jb.delta, n_sing);
}

}  // namespace

cudaError_t launch_weights_multi(int njobs, const WeightJob *jobs_dev, const int64_t *prefix_dev, int64_t ntot,
                                 int max_n_l, int k, int m, int n_ops, const OpSpec *ops, int32_t *n_sing,
                                 cudaStream_t st) {
    if (ntot <= 0) return cudaSuccess;
    if (n_ops < 1 || n_ops > RBF_MAX_OPS || max_n_l < 2 || max_n_l > RBF_MAX_NL || m < 0 || m > 4) return cudaErrorInvalidValue;
    const int np = (m + 1) * (m + 2) * (m + 3) / 6;
    const size_t smem = wlayout(max_n_l, np, n_ops).total * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(k_weights_multi, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_weights_multi<<<(unsigned)ntot, WT, smem, st>>>(njobs, jobs_dev, prefix_dev, k, np, n_ops, ops, n_sing);
    return cudaGetLastError();
}

cudaError_t launch_weights(int64_t nc, const double *xyz, const double *cxyz, const int32_t *cnode,
                           int centre_is_node, int n_l, const int32_t *idx, int k, int m, int n_ops,
                           const OpSpec *ops, double *w, double *delta, int32_t *n_sing, cudaStream_t st) {
    if (nc <= 0) return cudaSuccess;
    if (n_ops < 1 || n_ops > RBF_MAX_OPS || n_l < 2 || n_l > RBF_MAX_NL || m < 0 || m > 4) return cudaErrorInvalidValue;
    const int np = (m + 1) * (m + 2) * (m + 3) / 6;
    const size_t smem = wlayout(n_l, np, n_ops).total * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(k_weights, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_weights<<<(unsigned)nc, WT, smem, st>>>(nc, xyz, cxyz, cnode, centre_is_node, n_l, idx, k, np, n_ops, ops, w,
                                              delta, n_sing);
    return cudaGetLastError();
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
