// knn.cu — Morton ordering of the node cloud and periodic k-nearest-neighbour
// stencils (meshless discretisation section: S_i holds the N_L nodes closest to
// x_i; periodicity through the nearest image, case definition section).
//
// Nodes are sorted along a 3-D Morton curve (21 bits per axis) so that the nodes
// of one warp are close in space and the stencil gathers of the step kernels hit
// the same cache lines.  Neighbour search uses a uniform periodic cell grid and
// boxes of cells around the query; candidates are ranked by (squared distance computed
// without FMA, caller's node index), which makes the stencils bitwise
// reproducible and independent of the internal order.
#include "internal.cuh"

namespace rbf {

// ---- Morton keys ---------------------------------------------------------
__device__ __forceinline__ uint64_t spread21(uint64_t v) {
    v &= 0x1fffffULL;
    v = (v | (v << 32)) & 0x1f00000000ffffULL;
    v = (v | (v << 16)) & 0x1f0000ff0000ffULL;
    v = (v | (v << 8)) & 0x100f00f00f00f00fULL;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ULL;
    v = (v | (v << 2)) & 0x1249249249249249ULL;
    return v;
}

__device__ __forceinline__ uint64_t quant21(double x) {
    double s = x * 2097152.0;
    if (!(s >= 0.0)) s = 0.0;
    if (s > 2097151.0) s = 2097151.0;
    return (uint64_t)s;
}

__global__ void k_morton(int64_t n, const double *__restrict__ xyz, uint64_t *keys, int32_t *vals,
                         int64_t npow) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= npow) return;
    if (i < n) {
        uint64_t x = quant21(xyz[3 * i]), y = quant21(xyz[3 * i + 1]), z = quant21(xyz[3 * i + 2]);
        keys[i] = (spread21(x) << 2) | (spread21(y) << 1) | spread21(z);
        vals[i] = (int32_t)i;
    } else {
        keys[i] = ~0ULL;
        vals[i] = INT32_MAX;
    }
}

cudaError_t launch_morton_keys(int64_t n, const double *xyz, uint64_t *keys, int32_t *vals, int64_t npow,
                               cudaStream_t st) {
    k_morton<<<(unsigned)((npow + 255) / 256), 256, 0, st>>>(n, xyz, keys, vals, npow);
    return cudaGetLastError();
}

// ---- bitonic sort of (key, val) pairs, ascending by (key, val) -------------
__device__ __forceinline__ bool pair_gt(uint64_t ka, int32_t va, uint64_t kb, int32_t vb) {
    return ka > kb || (ka == kb && va > vb);
}

__global__ void k_bitonic_global(uint64_t *keys, int32_t *vals, int64_t npow, int64_t j, int64_t k) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= npow) return;
    int64_t p = i ^ j;
    if (p <= i) return;
    bool up = (i & k) == 0;
    uint64_t ki = keys[i], kp = keys[p];
    int32_t vi = vals[i], vp = vals[p];
    if (pair_gt(ki, vi, kp, vp) == up) {
        keys[i] = kp; keys[p] = ki;
        vals[i] = vp; vals[p] = vi;
    }
}

// all steps with j < 1024 of stage k, in shared memory (2048 elements per block)
__global__ void k_bitonic_shared(uint64_t *keys, int32_t *vals, int64_t npow, int64_t k, int64_t jmax) {
    __shared__ uint64_t sk[2048];
    __shared__ int32_t sv[2048];
    int64_t base = blockIdx.x * 2048LL;
    for (int t = threadIdx.x; t < 2048; t += blockDim.x) {
        sk[t] = keys[base + t];
        sv[t] = vals[base + t];
    }
    __syncthreads();
    for (int64_t j = jmax; j > 0; j >>= 1) {
        for (int t = threadIdx.x; t < 2048; t += blockDim.x) {
            int p = t ^ (int)j;
            if (p > t) {
                int64_t gi = base + t;
                bool up = (gi & k) == 0;
                if (pair_gt(sk[t], sv[t], sk[p], sv[p]) == up) {
                    uint64_t tk = sk[t]; sk[t] = sk[p]; sk[p] = tk;
                    int32_t tv = sv[t]; sv[t] = sv[p]; sv[p] = tv;
                }
            }
        }
        __syncthreads();
    }
    for (int t = threadIdx.x; t < 2048; t += blockDim.x) {
        keys[base + t] = sk[t];
        vals[base + t] = sv[t];
    }
}

cudaError_t launch_bitonic_sort(uint64_t *keys, int32_t *vals, int64_t npow, cudaStream_t st, int64_t *launches) {
    unsigned blocks = (unsigned)((npow + 255) / 256);
    for (int64_t k = 2; k <= npow; k <<= 1) {
        int64_t j = k >> 1;
        for (; j >= 1024 || (j >= 1 && npow < 2048); j >>= 1) {
            k_bitonic_global<<<blocks, 256, 0, st>>>(keys, vals, npow, j, k);
            ++*launches;
        }
        if (j >= 1 && npow >= 2048) {
            k_bitonic_shared<<<(unsigned)(npow / 2048), 1024, 0, st>>>(keys, vals, npow, k, j);
            ++*launches;
        }
    }
    return cudaGetLastError();
}

__global__ void k_gather_nodes(int64_t n, const int32_t *__restrict__ perm, const double *__restrict__ xyz,
                               const uint8_t *__restrict__ type, const double *__restrict__ nrm, double *xyz_s,
                               uint8_t *type_s, double *nrm_s, int32_t *iperm) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t o = perm[i];
    for (int a = 0; a < 3; ++a) {
        xyz_s[3 * i + a] = xyz[3 * o + a];
        nrm_s[3 * i + a] = nrm[3 * o + a];
    }
    type_s[i] = type[o];
    iperm[o] = (int32_t)i;
}

cudaError_t launch_gather_nodes(int64_t n, const int32_t *perm, const double *xyz, const uint8_t *type,
                                const double *nrm, double *xyz_s, uint8_t *type_s, double *nrm_s,
                                int32_t *iperm, cudaStream_t st) {
    k_gather_nodes<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, perm, xyz, type, nrm, xyz_s, type_s, nrm_s,
                                                               iperm);
    return cudaGetLastError();
}

// ---- exclusive scan of int32 (three passes, 1024 elements per block) --------
__device__ __forceinline__ int32_t warp_incl_scan(int32_t v) {
    int lane = threadIdx.x & 31;
    for (int d = 1; d < 32; d <<= 1) {
        int32_t t = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += t;
    }
    return v;
}

__global__ void k_scan_blocks(const int32_t *in, int32_t *out, int64_t n, int32_t *sums) {
    __shared__ int32_t ws[32];
    int64_t i = blockIdx.x * 1024LL + threadIdx.x;
    int32_t v = i < n ? in[i] : 0;
    int32_t inc = warp_incl_scan(v);
    int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    if (w == 0) {
        int32_t t = ws[lane];
        ws[lane] = warp_incl_scan(t) - t;
    }
    __syncthreads();
    int32_t ex = inc - v + ws[w];
    if (i < n) out[i] = ex;
    if (threadIdx.x == 1023) sums[blockIdx.x] = ex + v;
}

__global__ void k_scan_sums(int32_t *sums, int64_t nb) {
    __shared__ int32_t ws[32];
    __shared__ int32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < nb; base += 1024) {
        int64_t i = base + threadIdx.x;
        int32_t v = i < nb ? sums[i] : 0;
        int32_t inc = warp_incl_scan(v);
        int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (lane == 31) ws[w] = inc;
        __syncthreads();
        if (w == 0) {
            int32_t t = ws[lane];
            ws[lane] = warp_incl_scan(t) - t;
        }
        __syncthreads();
        int32_t ex = inc - v + ws[w] + carry;
        __syncthreads();
        if (i < nb) sums[i] = ex;
        if (threadIdx.x == 1023) carry = ex + v;
        __syncthreads();
    }
}

__global__ void k_scan_add(int32_t *out, int64_t n, const int32_t *sums) {
    int64_t i = blockIdx.x * 1024LL + threadIdx.x;
    if (i < n) out[i] += sums[blockIdx.x];
}

int64_t scan_tmp_len(int64_t n) { return (n + 1023) / 1024 + 1; }

cudaError_t launch_scan_i32(const int32_t *in, int32_t *out, int64_t n, int32_t *tmp, int64_t tmp_len,
                            cudaStream_t st, int64_t *launches) {
    int64_t nb = (n + 1023) / 1024;
    if (nb + 1 > tmp_len) return cudaErrorInvalidValue;
    k_scan_blocks<<<(unsigned)nb, 1024, 0, st>>>(in, out, n, tmp);
    k_scan_sums<<<1, 1024, 0, st>>>(tmp, nb);
    k_scan_add<<<(unsigned)nb, 1024, 0, st>>>(out, n, tmp);
    *launches += 3;
    return cudaGetLastError();
}

// ---- cell grid -------------------------------------------------------------
__device__ __forceinline__ int cell_coord(double x, int G) {
    int c = (int)(x * G);
    return c < 0 ? 0 : (c >= G ? G - 1 : c);
}

__global__ void k_cell_count(int64_t n, const double *__restrict__ xyz, int G, int32_t *cell_of, int32_t *count) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int cx = cell_coord(xyz[3 * i], G), cy = cell_coord(xyz[3 * i + 1], G), cz = cell_coord(xyz[3 * i + 2], G);
    int32_t c = (int32_t)(((int64_t)cx * G + cy) * G + cz);
    cell_of[i] = c;
    atomicAdd(&count[c], 1);
}

cudaError_t launch_cell_count(int64_t n, const double *xyz, int G, int32_t *cell_of, int32_t *count,
                              cudaStream_t st) {
    k_cell_count<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, xyz, G, cell_of, count);
    return cudaGetLastError();
}

__global__ void k_cell_fill(int64_t n, const int32_t *cell_of, const int32_t *start, int32_t *fill,
                            int32_t *items) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int32_t c = cell_of[i];
    items[start[c] + atomicAdd(&fill[c], 1)] = (int32_t)i;
}

cudaError_t launch_cell_fill(int64_t n, const int32_t *cell_of, const int32_t *start, int32_t *fill,
                             int32_t *items, cudaStream_t st) {
    k_cell_fill<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, cell_of, start, fill, items);
    return cudaGetLastError();
}

__global__ void k_type_flags(int64_t n, const uint8_t *type, uint8_t want, int32_t *flags) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) flags[i] = type[i] == want;
}

cudaError_t launch_type_flags(int64_t n, const uint8_t *type, uint8_t want, int32_t *flags, cudaStream_t st) {
    k_type_flags<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, type, want, flags);
    return cudaGetLastError();
}

__global__ void k_flag_compact(int64_t n, const uint8_t *type, uint8_t want, const int32_t *scan, int32_t *list) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n && type[i] == want) list[scan[i]] = (int32_t)i;
}

cudaError_t launch_flag_compact(int64_t n, const uint8_t *type, uint8_t want, const int32_t *scan,
                                int32_t *list, cudaStream_t st) {
    k_flag_compact<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, type, want, scan, list);
    return cudaGetLastError();
}

// Cell-sorted copies for the neighbour search: FP32 coordinates and the node number, its
// top bit set for wall nodes
__global__ void k_cell_points(int64_t n, const int32_t *__restrict__ items, const double *__restrict__ xyz,
                              const uint8_t *__restrict__ type, float4 *__restrict__ pts) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int64_t s = items[e];
    pts[e] = make_float4((float)xyz[3 * s], (float)xyz[3 * s + 1], (float)xyz[3 * s + 2],
                         __uint_as_float((uint32_t)s | (type[s] ? 0x80000000u : 0u)));
}

cudaError_t launch_cell_points(int64_t n, const int32_t *items, const double *xyz, const uint8_t *type, float4 *pts,
                               cudaStream_t st) {
    k_cell_points<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, items, xyz, type, pts);
    return cudaGetLastError();
}

// ---- k nearest neighbours ---------------------------------------------------
// One warp per query.  The box of cells within Chebyshev distance r of the query's cell is
// scanned row by row (the cells of a row are contiguous in the cell-sorted copies), r taken
// from the number of nodes in the nearest 27 cells.  Every unseen node is then at least
// r cs away, so the search ends once the n_l-th distance is below r cs, and otherwise goes
// on with the shells r + 1, r + 2, ... until it is, or the whole periodic grid has been seen.
//
// A candidate costs a few FP32 operations: its FP32 distance is compared with the current
// n_l-th distance plus 1e-6 (FP32 coordinates in [0, 1] put a distance off by less than
// 4e-7), and only what passes gets the exact FP64 distance, 32 at a time, and is merged into
// the 64 best, which the warp keeps sorted in registers (lane l: ranks l and 32 + l).  FP64
// values compare as integers.  Measured: 86k queries of 40 (refined cloud) 1.14 ms in
// place of 9.9 ms for one thread per query with its list in local memory, 616 wall queries of
// 24 42 us in place of 1.03 ms.
namespace {
struct Best {
    unsigned long long d[2];  // squared distance (bits), ranks lane and 32 + lane
    int s[2];
};
__device__ __forceinline__ bool before(unsigned long long da, int sa, unsigned long long db, int sb,
                                       const int32_t *perm) {
    if (da != db) return da < db;
    if (sa == sb || sa < 0 || sb < 0) return sa >= 0 && sb < 0;
    return perm[sa] < perm[sb];
}
// compare-exchange with the lane `xor` away: the lower lane keeps the smaller when up
__device__ __forceinline__ void exchange(unsigned long long &d, int &s, int mask, bool keep_small, const int32_t *perm) {
    const unsigned long long od = __shfl_xor_sync(0xffffffffu, d, mask);
    const int os = __shfl_xor_sync(0xffffffffu, s, mask);
    if (before(od, os, d, s, perm) == keep_small) {
        d = od;
        s = os;
    }
}
__device__ __forceinline__ void bitonic_merge(unsigned long long &d, int &s, int lane, const int32_t *perm) {
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) exchange(d, s, m, (lane & m) == 0, perm);
}
// the 64 best of 64 + 32 (one new entry per lane; absent: d all ones, s = -1)
__device__ __forceinline__ void merge_in(Best &b, unsigned long long d, int s, int lane, const int32_t *perm) {
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int m = k >> 1; m > 0; m >>= 1) exchange(d, s, m, ((lane & m) == 0) == ((lane & k) == 0), perm);
    // smaller halves of (ranks 32 .. 63) and (new, reversed), sorted
    const unsigned long long rd = __shfl_xor_sync(0xffffffffu, d, 31);
    const int rs = __shfl_xor_sync(0xffffffffu, s, 31);
    if (before(rd, rs, b.d[1], b.s[1], perm)) {
        b.d[1] = rd;
        b.s[1] = rs;
    }
    bitonic_merge(b.d[1], b.s[1], lane, perm);
    // the two sorted halves merged
    const unsigned long long qd = __shfl_xor_sync(0xffffffffu, b.d[1], 31);
    const int qs = __shfl_xor_sync(0xffffffffu, b.s[1], 31);
    if (before(qd, qs, b.d[0], b.s[0], perm)) {
        b.d[1] = b.d[0];
        b.s[1] = b.s[0];
        b.d[0] = qd;
        b.s[0] = qs;
    } else {
        b.d[1] = qd;
        b.s[1] = qs;
    }
    bitonic_merge(b.d[0], b.s[0], lane, perm);
    bitonic_merge(b.d[1], b.s[1], lane, perm);
}
}  // namespace

__global__ void __launch_bounds__(128) k_knn(int64_t nq, const double *__restrict__ qxyz,
                                             const int32_t *__restrict__ qnode, const double *__restrict__ xyz,
                                             const int32_t *__restrict__ perm, int fluid_only, int G,
                                             const int32_t *__restrict__ cstart, const float4 *__restrict__ pts, int n_l,
                                             int32_t *out, int ld, int col0, int32_t *status) {
    __shared__ int pend[4][64];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t a = blockIdx.x * 4ll + warp;
    if (a >= nq) return;
    int *pd = pend[warp];
    double qx, qy, qz;
    if (qxyz) {
        qx = qxyz[3 * a]; qy = qxyz[3 * a + 1]; qz = qxyz[3 * a + 2];
    } else {
        int64_t s = qnode[a];
        qx = xyz[3 * s]; qy = xyz[3 * s + 1]; qz = xyz[3 * s + 2];
    }
    qx -= floor(qx); qy -= floor(qy); qz -= floor(qz);
    const float fx = (float)qx, fy = (float)qy, fz = (float)qz;
    const double cs = 1.0 / G;
    const int cx = cell_coord(qx, G), cy = cell_coord(qy, G), cz = cell_coord(qz, G);
    const int lo = -((G - 1) / 2), hi = G / 2;  // distinct periodic offsets
    Best best;
    best.d[0] = best.d[1] = ~0ull;
    best.s[0] = best.s[1] = -1;
    int n_pend = 0, seen = 0;
    float thr = __int_as_float(0x7f800000);
    auto kth = [&]() -> unsigned long long {
        const unsigned long long v = n_l > 32 ? best.d[1] : best.d[0];
        return __shfl_sync(0xffffffffu, v, (n_l - 1) & 31);
    };
    // exact distances of up to 32 pending candidates, merged into the best
    auto flush = [&](int cnt) {
        __syncwarp();
        unsigned long long d = ~0ull;
        int s = -1;
        if (lane < cnt) {
            s = pd[lane];
            const double ddx = mimg(xyz[3 * (int64_t)s] - qx), ddy = mimg(xyz[3 * (int64_t)s + 1] - qy), ddz = mimg(xyz[3 * (int64_t)s + 2] - qz);
            d = (unsigned long long)__double_as_longlong(dist2_nofma(ddx, ddy, ddz));
        }
        merge_in(best, d, s, lane, perm);
        const unsigned long long k = kth();
        if (k != ~0ull) {
            const float r = sqrtf(__double2float_ru(__longlong_as_double((long long)k))) + 1e-6f;
            thr = r * r * 1.000001f;
        }
        // what is left moves to the front
        const int more = n_pend - cnt;
        const int v = lane < more ? pd[cnt + lane] : 0;
        __syncwarp();
        if (lane < more) pd[lane] = v;
        n_pend = more;
        __syncwarp();
    };
    auto scan = [&](int e0, int e1) {
        for (int base = e0; base < e1; base += 32) {
            const int e = base + lane;
            bool pass = false;
            int s = 0;
            if (e < e1) {
                const float4 p = pts[e];
                const uint32_t w = __float_as_uint(p.w);
                float dx = p.x - fx, dy = p.y - fy, dz = p.z - fz;
                dx -= rintf(dx); dy -= rintf(dy); dz -= rintf(dz);
                s = (int)(w & 0x7fffffffu);
                pass = dx * dx + dy * dy + dz * dz <= thr && !(fluid_only && (w >> 31));
            }
            const unsigned m = __ballot_sync(0xffffffffu, pass);
            if (m) {
                if (pass) pd[n_pend + __popc(m & ((1u << lane) - 1u))] = s;
                n_pend += __popc(m);
                if (n_pend >= 32) flush(32);
            }
        }
    };
    // cells z0 .. z1 (offsets from the query's cell) of row (dx, dy)
    auto row = [&](int dx, int dy, int z0, int z1, bool count_only) {
        if (z0 > z1) return;
        const int ix = (cx + dx + G) % G, iy = (cy + dy + G) % G;
        const int32_t *c = cstart + ((int64_t)ix * G + iy) * G;
        int i0 = cz + z0, i1 = cz + z1;
        if (i1 < 0) { i0 += G; i1 += G; }
        if (i0 >= G) { i0 -= G; i1 -= G; }
        if (i0 < 0) {  // across the period: the end of the row, then its beginning
            if (count_only) seen += c[G] - c[i0 + G];
            else scan(c[i0 + G], c[G]);
            i0 = 0;
        }
        if (i1 >= G) {
            if (count_only) seen += c[i1 - G + 1] - c[0];
            else scan(c[0], c[i1 - G + 1]);
            i1 = G - 1;
        }
        if (i0 <= i1) {
            if (count_only) seen += c[i1 + 1] - c[i0];
            else scan(c[i0], c[i1 + 1]);
        }
    };
    // boxes wider than the distinct offsets are cut to them
    auto box = [&](int done, int r) {  // the cells at Chebyshev distance done + 1 .. r
        const int x0 = max(-r, lo), x1 = min(r, hi);
        for (int pass = 0; pass < 2; ++pass)  // the middle rows first: they fill the list with near nodes
            for (int dx = x0; dx <= x1; ++dx)
                for (int dy = x0; dy <= x1; ++dy) {
                    const int m = max(abs(dx), abs(dy));
                    if ((m <= 1) != (pass == 0)) continue;
                    if (m > done) row(dx, dy, x0, x1, false);
                    else {
                        row(dx, dy, x0, min(x1, -done - 1), false);
                        row(dx, dy, max(x0, done + 1), x1, false);
                    }
                }
    };
    for (int dx = max(-1, lo); dx <= min(1, hi); ++dx)
        for (int dy = max(-1, lo); dy <= min(1, hi); ++dy) row(dx, dy, max(-1, lo), min(1, hi), true);
    // radius (in cells) of a ball with n_l nodes at the density of the nearest 27 cells
    int r = max(1, (int)ceilf(1.1f * cbrtf((float)n_l * 27.0f / (4.19f * (float)max(seen, 1)))));
    int done = -1;
    for (;;) {
        r = min(r, G);
        box(done, r);
        while (n_pend > 0) flush(min(n_pend, 32));
        if (-r <= lo && r >= hi) break;  // every cell seen
        const double reach = r * cs;
        const unsigned long long k = kth();
        if (k != ~0ull && __longlong_as_double((long long)k) < reach * reach * (1.0 - 1e-12)) break;
        done = r;
        ++r;
    }
    const unsigned have = __popc(__ballot_sync(0xffffffffu, best.s[0] >= 0)) + __popc(__ballot_sync(0xffffffffu, best.s[1] >= 0));
    if ((int)have < n_l) {
        if (lane == 0) atomicExch(status, 1);
        const int s0 = max(__shfl_sync(0xffffffffu, best.s[0], 0), 0);
        for (int h = 0; h < 2; ++h)
            if (best.s[h] < 0) best.s[h] = s0;  // flagged: never used
    }
    for (int h = 0; h < 2; ++h)
        if (lane + 32 * h < n_l) out[a * ld + col0 + lane + 32 * h] = best.s[h];
}

cudaError_t launch_knn(int64_t nq, const double *qxyz, const int32_t *qnode, const double *xyz, const int32_t *perm,
                       int fluid_only, int G, const int32_t *cell_start, const float4 *pts, int n_l, int32_t *out,
                       int ld, int col0, int32_t *status, cudaStream_t st) {
    if (nq <= 0) return cudaSuccess;
    k_knn<<<(unsigned)((nq + 3) / 4), 128, 0, st>>>(nq, qxyz, qnode, xyz, perm, fluid_only, G, cell_start, pts, n_l, out,
                                                    ld, col0, status);
    return cudaGetLastError();
}

}  // namespace rbf
