// acm_persist.cu — the ACM steady driver as one persistent kernel over any number
// of cells (MNS algorithm of the appendix, repeated until each cell's stopping
// criterion holds).
//
// One cooperative launch; every block loops over steps and, inside a step, over
// the phases  predict -> n_p x (pressure, wall pressure, correction),  separated by
// a grid barrier, each phase over the units of all cells still running (a unit is
// 32 / G nodes of a 32-node SELL slice, G lanes per node).  Every check_every steps the blocks reduce, per
// cell, |v - v_prev|^2 and |v|^2 in FP64, block 0 turns them into residuals and sets
// the cell's done flag; converged cells drop out of the loop while the others
// continue.  The arithmetic of each phase is that of the multi-launch kernels in
// acm.cu, in the same order for the same lanes per node (wall nodes have WALL_LANES in both),
// except in the resident kernel.
//
// What bounds it, and the layout that follows: a step of a small cell is ten phases
// of a few hundred nanoseconds of work each, so the chain barrier -> descriptor ->
// stencil index -> gathered field -> sum -> barrier decides.
//  * One cell whose stencils fit the SMs' shared memory (34 MB on the chip: about 30k
//    nodes at N_L = 25 in FP64, 55k in FP32) runs resident, k_acm_resident below.
//  * Everything else streams its stencils, k_acm_persistent, with the cells' unit counts
//    and done flags in shared memory.
//  * The barrier is one monotonic counter: one release-add per block, polling
//    acquire loads, no reset.
//
// A block that waits longer than PersistCtl::wait_ns (2 s by default) at a barrier
// raises an error flag and leaves the loop, so a launch whose blocks are not
// co-resident ends with RBF_ETIMEOUT instead of hanging.  Every wait also ends soon
// after another block has raised the flag.  The cooperative launch itself guarantees
// co-residency.
//
// CP = true is the compensated FP32 state of acm.cu (hi + lo pairs, comp_add
// updates, gathers of the hi words); its residual differences include the low
// words.
#include <algorithm>
#include <cstring>

#include "acm_persist.cuh"
#include "acm.cuh"
#include "tc.cuh"

namespace rbf {

namespace {

__device__ __forceinline__ void red_release_add(unsigned *p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned atom_acq_rel_add(unsigned *p, unsigned v) {
    unsigned r;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(r) : "l"(p), "r"(v) : "memory");
    return r;
}
__device__ __forceinline__ void st_release(unsigned *p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Arrive and wait until every block has arrived for this barrier: bar[0] counts arrivals
// (it only grows; `target` is its value when all are there, compared modulo 2^32).
// Up to BAR_FEW blocks poll the counter itself (1.19 us per barrier of 152 blocks, 1.31
// through the flag; a step of 12 cells with 608 / 1,216 blocks 418 / 441 us against 441 / 447); more
// polling blocks hold up the arrivals, so there the last to arrive publishes the target
// in bar[BAR_FLAG], on another line (2,432 blocks 464 against 597 us, 4,864 blocks 593
// against 974).
// False (and *err raised) if that takes longer than wait_ns nanoseconds or if another
// block has raised *err.  The clock and the flag are looked at every 32nd poll, at every
// poll when the limit is below 100 us.
constexpr int BAR_FLAG = 32;
constexpr unsigned BAR_FEW = 1300;
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned target, unsigned nblocks, int32_t *err,
                                             uint64_t wait_ns) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        const unsigned *word = bar;
        bool last = false;
        if (nblocks <= BAR_FEW) {
            red_release_add(bar, 1u);
        } else {
            word = bar + BAR_FLAG;
            last = atom_acq_rel_add(bar, 1u) == target - 1u;
            if (last) st_release(bar + BAR_FLAG, target);
        }
        const unsigned mask = wait_ns < 100000 ? 0u : 31u;
        uint64_t t0 = 0;
        for (unsigned n = 0; !last && (int)(ld_acquire(word) - target) < 0; ++n) {
            if ((n & mask) == mask) {
                const uint64_t now = tc::globaltimer_ns();
                if (n == mask) t0 = now;
                if (*(volatile int32_t *)err) { ok = 0; break; }
                if (now - t0 > wait_ns) {
                    atomicExch(err, 2);
                    ok = 0;
                    break;
                }
            }
        }
    }
    __syncthreads();
    return ok != 0;
}

// every thread of every CTA of the cluster arrives (release) and waits (acquire):
// the hardware barrier of a thread-block cluster, no spinning on memory
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ double slot_C(const unsigned long long *slot, double beta, double vref) {
    const double vmax = __longlong_as_double((long long)*(volatile unsigned long long *)slot);
    return beta * (vmax > vref ? vmax : vref);
}

// A unit's stencil data as one lane sees it: weight (o, j) of its node at
// w[(o n_l + j) 32], index j at ip[32 j]; streamed, so evict-first
template <typename T>
struct Sten {
    const T *w;
    const int32_t *ip;
    __device__ __forceinline__ T wt(int at) const { return __ldcs(w + 32 * at); }
    __device__ __forceinline__ int ix(int at) const { return __ldcs(ip + 32 * at); }
};

// The phases work on units of 32 / G nodes of one slice: unit `sub` of slice ls
// holds nodes sub (32 / G) .. (sub + 1) (32 / G) - 1, node nl of the unit on lanes
// G (nl mod 32/G) .. + G - 1, each lane taking the stencil columns j = g, g + G, ...
// (g = lane mod G); the group's partial sums are combined with shuffles and the
// first lane of the group (the lead) writes.  G = 1 is one node per lane.  Every
// lane reaches the shuffles (no early return before them). 
template <typename T, bool CP, int G>
__device__ __forceinline__ void phase_predict(const CellDesc<T> &c, const Sten<T> st, int64_t i, int g, bool valid,
                                              bool fluid, bool snapshot) {
    T ui = 0, vi = 0, wi = 0;
    if (valid) { ui = c.u[i]; vi = c.v[i]; wi = c.w_[i]; }
    T gu[4] = {0, 0, 0, 0}, gv[4] = {0, 0, 0, 0}, gw[4] = {0, 0, 0, 0};
    if (fluid) {
        const int n_l = c.n_l;
        const T *u = c.u, *v = c.v, *w = c.w_;
#pragma unroll 5
        for (int j = g; j < n_l; j += G) {
            const int q = st.ix(j);
            const T wx = st.wt(j), wy = st.wt((n_l + j));
            const T wz = st.wt((2 * n_l + j)), wl = st.wt((3 * n_l + j));
            const T uq = u[q], vq = v[q], wq = w[q];
            gu[0] += wx * uq; gu[1] += wy * uq; gu[2] += wz * uq; gu[3] += wl * uq;
            gv[0] += wx * vq; gv[1] += wy * vq; gv[2] += wz * vq; gv[3] += wl * vq;
            gw[0] += wx * wq; gw[1] += wy * wq; gw[2] += wz * wq; gw[3] += wl * wq;
        }
    }
    if constexpr (G > 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            gu[k] = group_sum<T, G>(gu[k]);
            gv[k] = group_sum<T, G>(gv[k]);
            gw[k] = group_sum<T, G>(gw[k]);
        }
    }
    if (!valid || g != 0) return;
    if (snapshot) {
        c.uo[i] = ui; c.vo[i] = vi; c.wo[i] = wi;
        if constexpr (CP) { c.uol[i] = c.ul[i]; c.vol[i] = c.vl[i]; c.wol[i] = c.wl[i]; }
    }
    if (!fluid) {
        c.us[i] = (T)0; c.vs[i] = (T)0; c.ws[i] = (T)0;
        if constexpr (CP) { c.usl[i] = (T)0; c.vsl[i] = (T)0; c.wsl[i] = (T)0; }
        return;
    }
    const T adv_u = ui * gu[0] + vi * gu[1] + wi * gu[2];
    const T adv_v = ui * gv[0] + vi * gv[1] + wi * gv[2];
    const T adv_w = ui * gw[0] + vi * gw[1] + wi * gw[2];
    if constexpr (CP) {
        T h = ui, l = c.ul[i];
        comp_add(h, l, c.dt * (c.nu * gu[3] - adv_u + c.gx));
        c.us[i] = h; c.usl[i] = l;
        h = vi; l = c.vl[i];
        comp_add(h, l, c.dt * (c.nu * gv[3] - adv_v + c.gy));
        c.vs[i] = h; c.vsl[i] = l;
        h = wi; l = c.wl[i];
        comp_add(h, l, c.dt * (c.nu * gw[3] - adv_w + c.gz));
        c.ws[i] = h; c.wsl[i] = l;
    } else {
        c.us[i] = ui + c.dt * (c.nu * gu[3] - adv_u + c.gx);
        c.vs[i] = vi + c.dt * (c.nu * gv[3] - adv_v + c.gy);
        c.ws[i] = wi + c.dt * (c.nu * gw[3] - adv_w + c.gz);
    }
}

template <typename T, bool CP, int G>
__device__ __forceinline__ void phase_pressure(const CellDesc<T> &c, const Sten<T> st, int64_t i, int g, bool fluid,
                                               bool first, int gslot) {
    const T *u = first ? c.us : c.u;
    const T *v = first ? c.vs : c.v;
    const T *w = first ? c.ws : c.w_;
    T div = 0;
    if (fluid) {
        const int n_l = c.n_l;
#pragma unroll 5
        for (int j = g; j < n_l; j += G) {
            const int q = st.ix(j);
            div += st.wt(j) * u[q] + st.wt((n_l + j)) * v[q] + st.wt((2 * n_l + j)) * w[q];
        }
    }
    if constexpr (G > 1) div = group_sum<T, G>(div);
    if (!fluid || g != 0) return;
    const double C = slot_C(c.vmax + (gslot ^ 1), c.beta, c.vref);
    const T Ct = (T)C;
    if constexpr (CP) {
        T h = c.p[i], l = c.pl[i];
        comp_add(h, l, -(c.dt * Ct * Ct * c.rho * div));
        c.p[i] = h; c.pl[i] = l;
    } else {
        c.p[i] = c.p[i] - c.dt * Ct * Ct * c.rho * div;
    }
}

template <typename T, bool CP, int G>
__device__ __forceinline__ void phase_wall(const CellDesc<T> &c, const Sten<T> st, int64_t b, int g) {
    const bool valid = b < c.nb;
    const int n_l = c.n_l;
    T acc = 0;
    if (valid) {
        const T *p = c.p;
#pragma unroll 4
        for (int j = 1 + g; j < n_l; j += G) acc += st.wt(j) * p[st.ix(j)];
    }
    if constexpr (G > 1) acc = group_sum<T, G>(acc);
    if (!valid || g != 0) return;
    const int32_t wb = c.wall[b];
    c.p[wb] = -acc / st.wt(0);
    if constexpr (CP) c.pl[wb] = (T)0;
}

// The same wall node by one lane: the partial sums of WALL_LANES lanes side by side, put together
// in the order of group_sum, so the same bits.
template <typename T, bool CP>
__device__ __forceinline__ void phase_wall_one(const CellDesc<T> &c, const Sten<T> st, int64_t b) {
    static_assert(WALL_LANES == 4, "four sums");
    if (b >= c.nb) return;
    const int n_l = c.n_l;
    const T *p = c.p;
    T s0 = 0, s1 = 0, s2 = 0, s3 = 0;
    int j = 1;
    for (; j + 3 < n_l; j += 4) {
        s0 += st.wt(j) * p[st.ix(j)];
        s1 += st.wt(j + 1) * p[st.ix(j + 1)];
        s2 += st.wt(j + 2) * p[st.ix(j + 2)];
        s3 += st.wt(j + 3) * p[st.ix(j + 3)];
    }
    if (j < n_l) s0 += st.wt(j) * p[st.ix(j)];
    if (j + 1 < n_l) s1 += st.wt(j + 1) * p[st.ix(j + 1)];
    if (j + 2 < n_l) s2 += st.wt(j + 2) * p[st.ix(j + 2)];
    const int32_t wb = c.wall[b];
    c.p[wb] = -((s0 + s2) + (s1 + s3)) / st.wt(0);
    if constexpr (CP) c.pl[wb] = (T)0;
}

// returns |v|^2 of the node (lead lane of a fluid node), 0 otherwise
template <typename T, bool CP, int G>
__device__ __forceinline__ T phase_correct(const CellDesc<T> &c, const Sten<T> st, int64_t i, int g, bool valid,
                                           bool fluid) {
    T gx = 0, gy = 0, gz = 0;
    if (fluid) {
        const int n_l = c.n_l;
        const T *p = c.p;
#pragma unroll 5
        for (int j = g; j < n_l; j += G) {
            const T pq = p[st.ix(j)];
            gx += st.wt(j) * pq;
            gy += st.wt((n_l + j)) * pq;
            gz += st.wt((2 * n_l + j)) * pq;
        }
    }
    if constexpr (G > 1) {
        gx = group_sum<T, G>(gx);
        gy = group_sum<T, G>(gy);
        gz = group_sum<T, G>(gz);
    }
    if (!valid || g != 0) return (T)0;
    if (!fluid) {
        c.u[i] = (T)0; c.v[i] = (T)0; c.w_[i] = (T)0;
        if constexpr (CP) { c.ul[i] = (T)0; c.vl[i] = (T)0; c.wl[i] = (T)0; }
        return (T)0;
    }
    const T f = c.dt / c.rho;
    T un = c.us[i], vn = c.vs[i], wn = c.ws[i];
    if constexpr (CP) {
        T l = c.usl[i];
        comp_add(un, l, -(f * gx)); c.ul[i] = l;
        l = c.vsl[i];
        comp_add(vn, l, -(f * gy)); c.vl[i] = l;
        l = c.wsl[i];
        comp_add(wn, l, -(f * gz)); c.wl[i] = l;
    } else {
        un -= f * gx; vn -= f * gy; wn -= f * gz;
    }
    c.u[i] = un; c.v[i] = vn; c.w_[i] = wn;
    return un * un + vn * vn + wn * wn;
}

// CL = false: a cooperative grid synchronised by grid_barrier (any number of
// co-resident blocks); CL = true: one thread-block cluster (8 or 16 CTAs)
// synchronised by the cluster's hardware barrier.  Every block of a cluster takes the
// same branches at every barrier (the done flags change only before a barrier and
// the cluster barrier cannot time out), so none is left waiting.  Dynamic shared
// memory: residual sums, unit counts and flags of the cells; with SH (persist_shared) also
// copies of the descriptors.
// The register cap is stated as the warps an SM is to hold: left to itself the compiler takes 96
// registers in FP64 with several lanes per node (2 blocks an SM instead of 3) and orders the FP32
// sweeps so that fewer of their loads are in flight (600k nodes, one lane 645 -> 531 us per step; 12
// cells of 467k 514 -> 421; FP64, 24 cells with four lanes 1.42 -> 1.34 ms).
template <typename T, bool CP, bool CL, int G, bool SH>
__global__ void __launch_bounds__(256, CL ? 1 : persist_warps<T>() / 8) k_acm_persistent(const CellDesc<T> *__restrict__ cells_g, PersistCtl ctl) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int nc = ctl.ncells;
    CellDesc<T> *own = reinterpret_cast<CellDesc<T> *>(sm);
    const CellDesc<T> *cells;
    if constexpr (SH) cells = own; else cells = cells_g;
    double *racc = reinterpret_cast<double *>(own + (SH ? nc : 0));  // [nc][2]
    int64_t *pre = reinterpret_cast<int64_t *>(racc + 2 * nc);  // [nc + 1] units ahead of each cell
    int64_t *wpre = pre + nc + 1;                               // [nc + 1] wall slices
    int *done = reinterpret_cast<int *>(wpre + nc + 1);         // [nc]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    const int nblocks = gridDim.x;
    const int nl0 = lane / G, g = lane % G;
    constexpr int NU = 32 / G;  // nodes per unit

    {
        if constexpr (SH) {
            const int words = nc * (int)(sizeof(CellDesc<T>) / 4);
            for (int e = threadIdx.x; e < words; e += blockDim.x)
                reinterpret_cast<int *>(own)[e] = reinterpret_cast<const int *>(cells_g)[e];
        }
        for (int c = threadIdx.x; c < nc; c += blockDim.x) {
            done[c] = 0;
            pre[c + 1] = ((cells_g[c].n + 31) >> 5) * G;
            wpre[c + 1] = (cells_g[c].nb + 31) >> 5;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        pre[0] = wpre[0] = 0;
        for (int c = 0; c < nc; ++c) {
            pre[c + 1] += pre[c];
            wpre[c + 1] += wpre[c];
        }
    }
    __syncthreads();
    const int64_t wstride = (int64_t)nblocks * wpb, k0 = (int64_t)blockIdx.x * wpb + warp;

    // FP64 is bound by each SM's own pipe, so there the units of several lanes per node that are left
    // over after whole rounds are dealt out to the blocks in turn (a quarter round on a few SMs costs
    // a whole one: 9 cells, 4.4 rounds of two lanes 812 -> 753 us per step); in FP32 they stay in
    // order, next to each other, and at one lane too (20k nodes FP64 169 us dealt out, 155 in order; the
    // default takes two lanes where a short round would be left over).
    auto dealt = [&](int64_t total, auto &&f) {
        const int64_t whole = total < wstride ? total : total - total % wstride;
        const int64_t last = whole + (int64_t)warp * nblocks + blockIdx.x;
        const int64_t end = last < total ? whole + wstride : whole;
        for (int64_t k = k0; k < end; k += wstride) f(k < whole ? k : last);
    };
    // Visit this warp's units (grid-stride over the units of all cells): f(cell number,
    // descriptor, slice, unit of the slice)
    auto units = [&](auto &&f) {
        int c = 0;
        if constexpr (sizeof(T) == 8 && G > 1) {
            dealt(pre[nc], [&](int64_t k) {
                while (k >= pre[c + 1]) ++c;
                if (done[c]) return;
                const int64_t un = k - pre[c];
                f(c, cells[c], un / G, (int)(un % G));
            });
        } else {
            for (int64_t k = k0; k < pre[nc]; k += wstride) {
                while (k >= pre[c + 1]) ++c;
                if (done[c]) continue;
                const int64_t un = k - pre[c];
                f(c, cells[c], un / G, (int)(un % G));
            }
        }
    };
    // Wall nodes by four lanes each while that is one unit a warp; past it one lane per node loses no
    // time to latency and saves the units' overhead (FP32, 64 cells with 1.6M wall nodes: 5.27 ms
    // per step against 5.58 with four lanes throughout; FP64, 12 cells 1.12 against 1.14).
    const int wlog = wpre[nc] * WALL_LANES <= wstride ? 2 : 0;
    static_assert(WALL_LANES == 4, "1 << wlog");
    auto wall_units = [&](auto &&f) {
        int c = 0;
        for (int64_t k = k0; k < wpre[nc] << wlog; k += wstride) {
            while (k >= wpre[c + 1] << wlog) ++c;
            if (done[c]) continue;
            const int64_t un = k - (wpre[c] << wlog);
            f(cells[c], un >> wlog, (int)(un & ((1 << wlog) - 1)));
        }
    };
    auto sten = [&](const CellDesc<T> &d, int64_t ls, int nl) {
        return Sten<T>{d.w + ((ls * 4 * (int64_t)d.n_l) << 5) + nl, d.idx + ((ls * d.n_l) << 5) + nl};
    };

    unsigned target = 0;
    auto barrier = [&]() -> bool {
        if constexpr (CL) {
            cluster_barrier();
            return true;
        } else {
            target += (unsigned)nblocks;
            return grid_barrier(ctl.bar, target, (unsigned)nblocks, ctl.err, ctl.wait_ns);
        }
    };

    bool checked = false;
    for (int64_t step = 0; step < ctl.max_steps; ++step) {
        if (checked) {  // the flags change only before a check's last barrier
            for (int c = threadIdx.x; c < nc; c += blockDim.x) done[c] = ((volatile int32_t *)ctl.done)[c];
            __syncthreads();
            bool any = false;
            for (int c = 0; c < nc; ++c) any |= !done[c];
            if (!any) break;
        }
        const bool check = ((step + 1) % ctl.check_every == 0) || (step + 1 == ctl.max_steps);
        checked = check;
        units([&](int, const CellDesc<T> &d, int64_t ls, int sub) {
            const int nl = sub * NU + nl0;
            const int64_t i = (ls << 5) + nl;
            const bool valid = i < d.n;
            phase_predict<T, CP, G>(d, sten(d, ls, nl), i, g, valid, valid && !d.type[i], check);
        });
        if (!barrier()) break;
        bool broke = false;
        for (int it = 0; it < ctl.n_p && !broke; ++it) {
            // slot parity of iteration `it` of this step for each cell: (parity0 + n_p * step + it) & 1
            if (blockIdx.x == 0)
                for (int ci = threadIdx.x; ci < nc; ci += blockDim.x) {
                    if (done[ci]) continue;
                    const CellDesc<T> &d = cells[ci];
                    d.vmax[(int)((d.parity0 + (int64_t)ctl.n_p * step + it) & 1)] = 0ULL;
                }
            units([&](int, const CellDesc<T> &d, int64_t ls, int sub) {
                const int nl = sub * NU + nl0;
                const int64_t i = (ls << 5) + nl;
                phase_pressure<T, CP, G>(d, sten(d, ls, nl), i, g, i < d.n && !d.type[i], it == 0,
                                         (int)((d.parity0 + (int64_t)ctl.n_p * step + it) & 1));
            });
            if (!barrier()) { broke = true; break; }
            wall_units([&](const CellDesc<T> &d, int64_t ls, int sub) {
                const T *wn = d.wn + ((ls * d.n_l) << 5);
                const int32_t *ib = d.idxb + ((ls * d.n_l) << 5);
                if (wlog) {
                    const int nl = sub * (32 / WALL_LANES) + lane / WALL_LANES;
                    phase_wall<T, CP, WALL_LANES>(d, Sten<T>{wn + nl, ib + nl}, (ls << 5) + nl, lane % WALL_LANES);
                } else {
                    phase_wall_one<T, CP>(d, Sten<T>{wn + lane, ib + lane}, (ls << 5) + lane);
                }
            });
            if (!barrier()) { broke = true; break; }
            // max |v| of each cell: the largest |v|^2 of this warp's units, one root and one
            // atomic per warp and cell (the root is monotonic)
            T best = 0;
            int bc = -1;
            auto flush = [&]() {
                if (bc < 0) return;
                for (int off = 16; off > 0; off >>= 1) {
                    const T o = __shfl_xor_sync(0xffffffffu, best, off);
                    best = best > o ? best : o;
                }
                if (lane == 0 && best > (T)0) {
                    const CellDesc<T> &d = cells[bc];
                    const double sp = (double)sqrt(best);
                    atomicMax(d.vmax + (int)((d.parity0 + (int64_t)ctl.n_p * step + it) & 1),
                              (unsigned long long)__double_as_longlong(sp));
                }
            };
            units([&](int c, const CellDesc<T> &d, int64_t ls, int sub) {
                if (c != bc) {
                    flush();
                    bc = c;
                    best = 0;
                }
                const int nl = sub * NU + nl0;
                const int64_t i = (ls << 5) + nl;
                const bool valid = i < d.n;
                const T v2 = phase_correct<T, CP, G>(d, sten(d, ls, nl), i, g, valid, valid && !d.type[i]);
                if (v2 > best) best = v2;
            });
            flush();
            if (!barrier()) { broke = true; break; }
        }
        if (broke) break;
        if (check) {
            for (int t = threadIdx.x; t < 2 * nc; t += blockDim.x) racc[t] = 0.0;
            __syncthreads();
            units([&](int c, const CellDesc<T> &d, int64_t ls, int sub) {
                const int64_t i = (ls << 5) + sub * NU + lane;
                double d2 = 0.0, v2 = 0.0;
                if (lane < NU && i < d.n && !d.type[i]) {
                    double a = (double)d.u[i] - (double)d.uo[i], b = (double)d.v[i] - (double)d.vo[i];
                    double e = (double)d.w_[i] - (double)d.wo[i];
                    double uu = d.u[i], vv = d.v[i], ww = d.w_[i];
                    if constexpr (CP) {
                        a += (double)d.ul[i] - (double)d.uol[i];
                        b += (double)d.vl[i] - (double)d.vol[i];
                        e += (double)d.wl[i] - (double)d.wol[i];
                        uu += d.ul[i]; vv += d.vl[i]; ww += d.wl[i];
                    }
                    d2 = a * a + b * b + e * e;
                    v2 = uu * uu + vv * vv + ww * ww;
                }
                for (int off = 16; off > 0; off >>= 1) {
                    d2 += __shfl_xor_sync(0xffffffffu, d2, off);
                    v2 += __shfl_xor_sync(0xffffffffu, v2, off);
                }
                if (lane == 0) {
                    atomicAdd(&racc[2 * c], d2);
                    atomicAdd(&racc[2 * c + 1], v2);
                }
            });
            __syncthreads();
            for (int t = threadIdx.x; t < 2 * nc; t += blockDim.x)
                ctl.partial[(int64_t)blockIdx.x * 2 * PERSIST_MAX_CELLS + t] = racc[t];
            if (!barrier()) break;
            if (blockIdx.x == 0) {
                for (int c = warp; c < nc; c += wpb) {
                    if (done[c]) continue;
                    double d2 = 0.0, v2 = 0.0;
                    for (int b = lane; b < nblocks; b += 32) {
                        d2 += ctl.partial[(int64_t)b * 2 * PERSIST_MAX_CELLS + 2 * c];
                        v2 += ctl.partial[(int64_t)b * 2 * PERSIST_MAX_CELLS + 2 * c + 1];
                    }
                    for (int off = 16; off > 0; off >>= 1) {
                        d2 += __shfl_xor_sync(0xffffffffu, d2, off);
                        v2 += __shfl_xor_sync(0xffffffffu, v2, off);
                    }
                    // a non-finite value anywhere in the cell's velocity makes d2 or v2
                    // non-finite (a NaN fails every comparison, so test before dividing)
                    const bool bad = !isfinite(d2) || !isfinite(v2);
                    const double rs = bad ? (double)NAN : (v2 > 0.0 ? sqrt(d2) / sqrt(v2) : 0.0);
                    if (lane == 0) {
                        ctl.resid[c] = rs;
                        ctl.steps[c] = step + 1;
                        if (bad) ctl.done[c] = 3;
                        else if (v2 > 0.0 && rs < ctl.tol) ctl.done[c] = 1;
                    }
                }
            }
            if (!barrier()) break;
        } else if (blockIdx.x == 0) {
            for (int c = threadIdx.x; c < nc; c += blockDim.x)
                if (!done[c]) ctl.steps[c] = step + 1;
        }
    }
}

// ---- one cell, resident on the chip ------------------------------------------------
// A cell small enough that every block (one per SM) holds its share of the stencils in
// shared memory for the whole launch: weights, and stencil columns as 16-bit numbers
// into the block's local node set (every node that its stencils reach, in Morton
// order).  After each barrier the block copies the current field of its local nodes from
// L2 into shared memory, once per node instead of once per stencil column, and all
// gathers are shared-memory reads.  Measured (us per step, N_L = 25, 2070 MHz): FP64 6,712
// nodes 38.8 (streaming, tuned: 74; stencils resident, gathers through L1: 46.6), FP32
// 6,712 nodes 26, compensated FP32 51,877 nodes 39.3 (103; 47.8).  Of a step's ten phases
// each costs 1.2 us for the barrier and about 1 us for the halo copy and the drain of its
// writes; the rest is the sums.
//
// In FP64 a warp instruction occupies its quarter of the SM for 64 cycles, so the phases
// also spend as few FP64 instructions as they can: the twelve sums of the predictor are
// reduced by halves over the lanes of a node (each lane ends with one operator and
// multiplies it by its own factor), C^2 is formed from max |v|^2 without a root, maxima
// compare as integers, quotients by the wall weight use a stored reciprocal with one
// correction.
struct ResOffsets {
    int w, wn, x, p, rw, lg, wb, mask, li, wli, lw, total;  // byte offsets
};
template <typename T>
__host__ __device__ inline ResOffsets res_offsets(const ResPlan &pl, int n_l, int nu) {
    ResOffsets o;
    const int T4 = (int)sizeof(T);
    o.w = 0;
    o.wn = o.w + pl.units * 4 * n_l * nu * T4;
    o.x = o.wn + pl.wunits * n_l * nu * T4;
    o.p = o.x + 3 * pl.loc * T4;
    o.rw = o.p + pl.loc * T4;
    o.lg = o.rw + pl.wunits * nu * T4;
    o.wb = o.lg + pl.loc * 4;
    o.mask = o.wb + pl.wunits * nu * 4;
    o.li = o.mask + pl.units * 4;
    o.wli = o.li + pl.units * n_l * nu * 2;
    o.lw = o.wli + pl.wunits * n_l * nu * 2;
    o.total = (o.lw + pl.loc * 2 + 15) & ~15;
    return o;
}

// a / b with r = 1 / b rounded: one residual correction of a r, which rounds as the division does
// (no difference in 3e8 random quotients of either type).  An infinite a r is the quotient already,
// its residual would be no number; told by the exponent, for FP64 comparisons go through the
// bounding pipe.
__device__ __forceinline__ float div_by(float a, float b, float r) {
    const float q = a * r;
    return (__float_as_uint(q) & 0x7f800000u) == 0x7f800000u ? q : fmaf(fmaf(-q, b, a), r, q);
}
__device__ __forceinline__ double div_by(double a, double b, double r) {
    const double q = a * r;
    return (__double2hiint(q) & 0x7ff00000) == 0x7ff00000 ? q : fma(fma(-q, b, a), r, q);
}
__device__ __forceinline__ unsigned long long nonneg_bits(float v) { return __float_as_uint(v) <= 0x7f800000u ? __float_as_uint(v) : 0u; }
__device__ __forceinline__ unsigned long long nonneg_bits(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return b <= 0x7ff0000000000000ull ? b : 0ull;
}
__device__ __forceinline__ double bits_to_double(unsigned long long b, float) { return (double)__uint_as_float((unsigned)b); }
__device__ __forceinline__ double bits_to_double(unsigned long long b, double) { return __longlong_as_double((long long)b); }

template <typename T, bool CP, int G>
__global__ void __launch_bounds__(sizeof(T) == 4 ? 1024 : 512)
k_acm_resident(const __grid_constant__ CellDesc<T> c, const __grid_constant__ PersistCtl ctl, const __grid_constant__ ResPlan pl) {
    constexpr int NU = 32 / G;  // nodes per unit
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int s_nloc, s_nwall;
    __shared__ double racc[2];
    const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31, wpb = nt >> 5;
    const int nl0 = lane / G, g = lane % G, n_l = c.n_l, nblocks = gridDim.x, b = blockIdx.x;
    const ResOffsets o = res_offsets<T>(pl, n_l, NU);
    T *W = reinterpret_cast<T *>(sm + o.w), *WN = reinterpret_cast<T *>(sm + o.wn);
    T *X = reinterpret_cast<T *>(sm + o.x), *Y = X + pl.loc, *Z = Y + pl.loc, *P = reinterpret_cast<T *>(sm + o.p);
    T *RW = reinterpret_cast<T *>(sm + o.rw);
    int *LG = reinterpret_cast<int *>(sm + o.lg), *WB = reinterpret_cast<int *>(sm + o.wb);
    unsigned *MASK = reinterpret_cast<unsigned *>(sm + o.mask);
    uint16_t *LI = reinterpret_cast<uint16_t *>(sm + o.li), *WLI = reinterpret_cast<uint16_t *>(sm + o.wli);
    uint16_t *LW = reinterpret_cast<uint16_t *>(sm + o.lw);
    const int64_t nu_all = ((c.n + 31) >> 5) * G, wu_all = ((c.nb + 31) >> 5) * G;
    const int u0 = (int)(nu_all * b / nblocks), n_unit = (int)(nu_all * (b + 1) / nblocks) - u0;
    const int w0 = (int)(wu_all * b / nblocks), n_wunit = (int)(wu_all * (b + 1) / nblocks) - w0;

    // -- the local node set: a bit per node (in the fields' room), then ranks
    const int nw = (int)((c.n + 31) >> 5);
    unsigned *bits = reinterpret_cast<unsigned *>(sm + o.x);
    int *rank0 = reinterpret_cast<int *>(bits + nw);
    for (int e = tid; e < nw; e += nt) bits[e] = 0u;
    if (tid == 0) s_nwall = 0;
    __syncthreads();
    auto idx_at = [&](int k, int e) {  // column e / NU of node e % NU of own unit k
        const int un = u0 + k;
        return c.idx[(((int64_t)(un / G) * n_l + e / NU) << 5) + (un % G) * NU + e % NU];
    };
    auto idxb_at = [&](int k, int e) {
        const int un = w0 + k;
        return c.idxb[(((int64_t)(un / G) * n_l + e / NU) << 5) + (un % G) * NU + e % NU];
    };
    for (int k = warp; k < n_unit; k += wpb) {
        const int64_t i = (int64_t)(u0 + k) * NU + lane;
        const unsigned fl = __ballot_sync(0xffffffffu, lane < NU && i < c.n && !c.type[i]);
        if (lane == 0) MASK[k] = fl;
        for (int e = lane; e < n_l * NU; e += 32)
            if ((fl >> (e % NU)) & 1u) {
                const int q = idx_at(k, e);
                atomicOr(bits + (q >> 5), 1u << (q & 31));
            }
    }
    for (int k = warp; k < n_wunit; k += wpb)
        for (int e = lane; e < n_l * NU; e += 32)
            if ((int64_t)(w0 + k) * NU + e % NU < c.nb) {
                const int q = idxb_at(k, e);
                atomicOr(bits + (q >> 5), 1u << (q & 31));
            }
    __syncthreads();
    if (warp == 0) {
        int sum = 0;
        for (int e0 = 0; e0 < nw; e0 += 32) {
            const int e = e0 + lane, cnt = e < nw ? __popc(bits[e]) : 0;
            int inc = cnt;
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += v;
            }
            if (e < nw) rank0[e] = sum + inc - cnt;
            sum += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) s_nloc = sum;
    }
    __syncthreads();
    const int nloc = s_nloc;
    unsigned target = 0;
    auto barrier = [&]() -> bool {
        target += (unsigned)nblocks;
        return grid_barrier(ctl.bar, target, (unsigned)nblocks, ctl.err, ctl.wait_ns);
    };
    // a share whose local set has no room ends the launch before its first step
    if (nloc > pl.loc && tid == 0) atomicExch(ctl.err, 3);
    if (!barrier()) return;
    if (*(volatile int32_t *)ctl.err) return;
    auto rank = [&](int q) { return (uint16_t)(rank0[q >> 5] + __popc(bits[q >> 5] & ((1u << (q & 31)) - 1u))); };
    for (int k = warp; k < n_unit; k += wpb) {
        const unsigned fl = MASK[k];
        const int un = u0 + k;
        const T *gw = c.w + (((int64_t)(un / G) * 4 * n_l) << 5) + (un % G) * NU;
        for (int e = lane; e < n_l * NU; e += 32) LI[k * n_l * NU + e] = (fl >> (e % NU)) & 1u ? rank(idx_at(k, e)) : 0;
        for (int e = lane; e < 4 * n_l * NU; e += 32) W[(size_t)k * 4 * n_l * NU + e] = __ldcs(gw + (e / NU) * 32 + e % NU);
    }
    for (int k = warp; k < n_wunit; k += wpb) {
        const int un = w0 + k;
        const T *gw = c.wn + (((int64_t)(un / G) * n_l) << 5) + (un % G) * NU;
        for (int e = lane; e < n_l * NU; e += 32) {
            const bool in = (int64_t)un * NU + e % NU < c.nb;
            WLI[k * n_l * NU + e] = in ? rank(idxb_at(k, e)) : 0;
            const T v = __ldcs(gw + (e / NU) * 32 + e % NU);
            WN[(size_t)k * n_l * NU + e] = v;
            if (e < NU) {
                RW[k * NU + e] = (T)1 / v;
                WB[k * NU + e] = in ? c.wall[(int64_t)un * NU + e] : -1;
            }
        }
    }
    for (int e = tid; e < nw; e += nt) {
        unsigned m = bits[e];
        int l = rank0[e];
        while (m) {
            const int q = e * 32 + __ffs((int)m) - 1;
            LG[l] = q;
            if (c.type[q]) LW[atomicAdd(&s_nwall, 1)] = (uint16_t)l;
            ++l;
            m &= m - 1u;
        }
    }
    __syncthreads();  // the bits' room becomes the fields'
    const int nwall = s_nwall;
    auto load3 = [&](const T *x, const T *y, const T *z) {
        for (int l = tid; l < nloc; l += nt) {
            const int q = LG[l];
            const T a = __ldcg(x + q), d = __ldcg(y + q), e = __ldcg(z + q);
            X[l] = a; Y[l] = d; Z[l] = e;
        }
        __syncthreads();
    };
    for (int l = tid; l < nloc; l += nt) P[l] = __ldcg(c.p + LG[l]);

    unsigned long long *vsq = ctl.vsq;  // two slots of max |v|^2, iteration i writing slot i & 1
    const T f = c.dt / c.rho;
    const double kc = (double)c.dt * (double)c.rho * c.beta * c.beta, vref2 = c.vref * c.vref;
    const unsigned long long vref2b = nonneg_bits(vref2);
    int64_t iter = 0, step = 0;
    bool broke = false;
    for (; step < ctl.max_steps; ++step) {
        const bool check = ((step + 1) % ctl.check_every == 0) || (step + 1 == ctl.max_steps);
        // ---- v' = v + dt (nu lap v - (v . grad) v + g)
        load3(c.u, c.v, c.w_);
        for (int k = warp; k < n_unit; k += wpb) {
            const unsigned fl = MASK[k];
            const bool fluid = (fl >> nl0) & 1u;
            const int64_t i = (int64_t)(u0 + k) * NU + nl0;
            if (!fluid) {  // a wall node's v' is zero; written once
                if (step == 0 && g == 0 && i < c.n) {
                    c.us[i] = (T)0; c.vs[i] = (T)0; c.ws[i] = (T)0;
                    if constexpr (CP) { c.usl[i] = (T)0; c.vsl[i] = (T)0; c.wsl[i] = (T)0; }
                }
            }
            const T *w = W + (size_t)k * 4 * n_l * NU + nl0;
            const uint16_t *li = LI + k * n_l * NU + nl0;
            T lo[3] = {0, 0, 0};
            if constexpr (CP)
                if (fluid && g == 0) { lo[0] = c.ul[i]; lo[1] = c.vl[i]; lo[2] = c.wl[i]; }
            T a[4][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
            if (fluid) {
#pragma unroll 2
                for (int j = g; j < n_l; j += G) {
                    const int q = li[j * NU];
                    const T x = X[q], y = Y[q], z = Z[q];
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const T wt = w[(p * n_l + j) * NU];
                        a[p][0] += wt * x; a[p][1] += wt * y; a[p][2] += wt * z;
                    }
                }
            }
            const int self = li[0];
            const T own[3] = {X[self], Y[self], Z[self]};
            T inc[3];  // nu lap - advection
            if constexpr (G >= 4) {
                // halve over the lanes: bit 0 of g keeps operators 0, 1 or 2, 3; bit 1 the first or second
                const bool h0 = g & 1, h1 = g & 2;
                T h[2][3], r[3];
#pragma unroll
                for (int p = 0; p < 2; ++p)
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const T send = h0 ? a[p][d] : a[2 + p][d], keep = h0 ? a[2 + p][d] : a[p][d];
                        h[p][d] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
                    }
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const T send = h1 ? h[0][d] : h[1][d], keep = h1 ? h[1][d] : h[0][d];
                    r[d] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
                }
                if constexpr (G == 8)
#pragma unroll
                    for (int d = 0; d < 3; ++d) r[d] += __shfl_xor_sync(0xffffffffu, r[d], 4);
                const T coef = h0 ? (h1 ? c.nu : -own[2]) : (h1 ? -own[1] : -own[0]);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    T t = coef * r[d];
                    t += __shfl_xor_sync(0xffffffffu, t, 1);
                    inc[d] = t + __shfl_xor_sync(0xffffffffu, t, 2);
                }
            } else {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
#pragma unroll
                    for (int p = 0; p < 4; ++p) a[p][d] = group_sum<T, G>(a[p][d]);
                    inc[d] = c.nu * a[3][d] - (own[0] * a[0][d] + own[1] * a[1][d] + own[2] * a[2][d]);
                }
            }
            if (fluid && g == 0) {
                if (check) {
                    c.uo[i] = own[0]; c.vo[i] = own[1]; c.wo[i] = own[2];
                    if constexpr (CP) { c.uol[i] = lo[0]; c.vol[i] = lo[1]; c.wol[i] = lo[2]; }
                }
                T hi[3] = {own[0], own[1], own[2]};
                const T gv[3] = {c.gx, c.gy, c.gz};
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    if constexpr (CP) comp_add(hi[d], lo[d], c.dt * (inc[d] + gv[d]));
                    else hi[d] = hi[d] + c.dt * (inc[d] + gv[d]);
                }
                c.us[i] = hi[0]; c.vs[i] = hi[1]; c.ws[i] = hi[2];
                if constexpr (CP) { c.usl[i] = lo[0]; c.vsl[i] = lo[1]; c.wsl[i] = lo[2]; }
            }
        }
        if (!barrier()) { broke = true; break; }
        for (int it = 0; it < ctl.n_p; ++it, ++iter) {
            // ---- p -= dt C^2 rho div v
            const unsigned long long vb = iter == 0 ? 0ull : __ldcg(vsq + ((iter + 1) & 1));
            double v2 = 0.0;
            if (iter == 0) {
                const double v = __longlong_as_double((long long)__ldcg(c.vmax + ((c.parity0 + 1) & 1)));
                v2 = v * v;
            }
            if (b == 0 && tid == 0) vsq[iter & 1] = 0ull;
            if (it == 0) load3(c.us, c.vs, c.ws);
            else load3(c.u, c.v, c.w_);
            if (iter != 0) v2 = bits_to_double(vb, T());
            const T kappa = (T)(kc * (nonneg_bits(v2) > vref2b ? v2 : vref2));
            for (int k = warp; k < n_unit; k += wpb) {
                const bool fluid = (MASK[k] >> nl0) & 1u;
                const int64_t i = (int64_t)(u0 + k) * NU + nl0;
                const T *w = W + (size_t)k * 4 * n_l * NU + nl0;
                const uint16_t *li = LI + k * n_l * NU + nl0;
                T lo = 0, d0 = 0;
                if constexpr (CP)
                    if (fluid && g == 0) lo = c.pl[i];
                if (fluid) {
#pragma unroll 4
                    for (int j = g; j < n_l; j += G) {
                        const int q = li[j * NU];
                        d0 += w[j * NU] * X[q] + w[(n_l + j) * NU] * Y[q] + w[(2 * n_l + j) * NU] * Z[q];
                    }
                }
                d0 = group_sum<T, G>(d0);
                if (fluid && g == 0) {
                    const int self = li[0];
                    T h = P[self];
                    if constexpr (CP) {
                        comp_add(h, lo, -(kappa * d0));
                        c.pl[i] = lo;
                    } else {
                        h = h - kappa * d0;
                    }
                    P[self] = h;
                    c.p[i] = h;
                }
            }
            if (!barrier()) { broke = true; break; }
            // ---- wall pressure from its fluid neighbours
            for (int l = tid; l < nloc; l += nt) P[l] = __ldcg(c.p + LG[l]);
            __syncthreads();
            for (int k = warp; k < n_wunit; k += wpb) {
                const int wb = WB[k * NU + nl0];
                const T *w = WN + (size_t)k * n_l * NU + nl0;
                const uint16_t *li = WLI + k * n_l * NU + nl0;
                T s0 = 0;
                if (wb >= 0) {
#pragma unroll 4
                    for (int j = 1 + g; j < n_l; j += G) s0 += w[j * NU] * P[li[j * NU]];
                }
                s0 = group_sum<T, G>(s0);
                if (wb >= 0 && g == 0) {
                    c.p[wb] = div_by(-s0, w[0], RW[k * NU + nl0]);
                    if constexpr (CP) c.pl[wb] = (T)0;
                }
            }
            if (c.nb > 0 && !barrier()) { broke = true; break; }
            // ---- v = v' - dt / rho grad p
            for (int l = tid; l < nwall; l += nt) {
                const int at = LW[l];
                P[at] = __ldcg(c.p + LG[at]);
            }
            __syncthreads();
            unsigned long long best = 0;
            for (int k = warp; k < n_unit; k += wpb) {
                const bool fluid = (MASK[k] >> nl0) & 1u;
                const int64_t i = (int64_t)(u0 + k) * NU + nl0;
                const T *w = W + (size_t)k * 4 * n_l * NU + nl0;
                const uint16_t *li = LI + k * n_l * NU + nl0;
                T h[3] = {0, 0, 0}, lo[3] = {0, 0, 0}, gr[3] = {0, 0, 0};
                if (fluid && g == 0) {
                    h[0] = c.us[i]; h[1] = c.vs[i]; h[2] = c.ws[i];
                    if constexpr (CP) { lo[0] = c.usl[i]; lo[1] = c.vsl[i]; lo[2] = c.wsl[i]; }
                }
                if (fluid) {
#pragma unroll 4
                    for (int j = g; j < n_l; j += G) {
                        const T pq = P[li[j * NU]];
                        gr[0] += w[j * NU] * pq; gr[1] += w[(n_l + j) * NU] * pq; gr[2] += w[(2 * n_l + j) * NU] * pq;
                    }
                }
#pragma unroll
                for (int d = 0; d < 3; ++d) gr[d] = group_sum<T, G>(gr[d]);
                if (fluid && g == 0) {
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        if constexpr (CP) comp_add(h[d], lo[d], -(f * gr[d]));
                        else h[d] = h[d] - f * gr[d];
                    }
                    c.u[i] = h[0]; c.v[i] = h[1]; c.w_[i] = h[2];
                    if constexpr (CP) { c.ul[i] = lo[0]; c.vl[i] = lo[1]; c.wl[i] = lo[2]; }
                    const unsigned long long s2 = nonneg_bits(h[0] * h[0] + h[1] * h[1] + h[2] * h[2]);
                    if (s2 > best) best = s2;
                } else if (step == 0 && it == 0 && g == 0 && i < c.n) {  // a wall node's velocity is zero; written once
                    c.u[i] = (T)0; c.v[i] = (T)0; c.w_[i] = (T)0;
                    if constexpr (CP) { c.ul[i] = (T)0; c.vl[i] = (T)0; c.wl[i] = (T)0; }
                }
            }
            for (int off = 16; off > 0; off >>= 1) {
                const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, off);
                if (ob > best) best = ob;
            }
            if (lane == 0 && best) atomicMax(vsq + (iter & 1), best);
            if (!barrier()) { broke = true; break; }
        }
        if (broke) break;
        if (b == 0 && tid == 0) ctl.steps[0] = step + 1;
        if (check) {
            if (tid == 0) racc[0] = racc[1] = 0.0;
            __syncthreads();
            double d2 = 0.0, v2 = 0.0;
            for (int k = warp; k < n_unit; k += wpb) {
                const int64_t i = (int64_t)(u0 + k) * NU + lane;
                if (lane < NU && ((MASK[k] >> lane) & 1u)) {
                    double a = (double)c.u[i] - (double)c.uo[i], d = (double)c.v[i] - (double)c.vo[i];
                    double e = (double)c.w_[i] - (double)c.wo[i];
                    double uu = c.u[i], vv = c.v[i], ww = c.w_[i];
                    if constexpr (CP) {
                        a += (double)c.ul[i] - (double)c.uol[i];
                        d += (double)c.vl[i] - (double)c.vol[i];
                        e += (double)c.wl[i] - (double)c.wol[i];
                        uu += c.ul[i]; vv += c.vl[i]; ww += c.wl[i];
                    }
                    d2 += a * a + d * d + e * e;
                    v2 += uu * uu + vv * vv + ww * ww;
                }
            }
            for (int off = 16; off > 0; off >>= 1) {
                d2 += __shfl_xor_sync(0xffffffffu, d2, off);
                v2 += __shfl_xor_sync(0xffffffffu, v2, off);
            }
            if (lane == 0) {
                atomicAdd(&racc[0], d2);
                atomicAdd(&racc[1], v2);
            }
            __syncthreads();
            if (tid < 2) ctl.partial[(int64_t)b * 2 * PERSIST_MAX_CELLS + tid] = racc[tid];
            if (!barrier()) { broke = true; break; }
            // every block adds the partials up in the same order, so all take the same decision
            // without a further barrier
            if (warp == 0) {
                double s2 = 0.0, q2 = 0.0;
                for (int e = lane; e < nblocks; e += 32) {
                    s2 += __ldcg(ctl.partial + (int64_t)e * 2 * PERSIST_MAX_CELLS);
                    q2 += __ldcg(ctl.partial + (int64_t)e * 2 * PERSIST_MAX_CELLS + 1);
                }
                for (int off = 16; off > 0; off >>= 1) {
                    s2 += __shfl_xor_sync(0xffffffffu, s2, off);
                    q2 += __shfl_xor_sync(0xffffffffu, q2, off);
                }
                const bool bad = !isfinite(s2) || !isfinite(q2);
                const double rs = bad ? (double)NAN : (q2 > 0.0 ? sqrt(s2) / sqrt(q2) : 0.0);
                const int dn = bad ? 3 : (q2 > 0.0 && rs < ctl.tol ? 1 : 0);
                if (lane == 0) {
                    s_nwall = dn;
                    if (b == 0) {
                        ctl.resid[0] = rs;
                        ctl.done[0] = dn;
                    }
                }
            }
            __syncthreads();
            if (s_nwall) { ++step; break; }
        }
    }
    // max |v| for the next launch, in the slot its first pressure sweep reads
    if (!broke && b == 0 && tid == 0 && iter > 0)
        c.vmax[(c.parity0 + iter + 1) & 1] =
            (unsigned long long)__double_as_longlong((double)sqrt((T)bits_to_double(__ldcg(vsq + ((iter + 1) & 1)), T())));
}

template <typename T, bool CP>
const void *resident_kernel(int group) {
    switch (group) {
    case 1: return (const void *)k_acm_resident<T, CP, 1>;
    case 2: return (const void *)k_acm_resident<T, CP, 2>;
    case 4: return (const void *)k_acm_resident<T, CP, 4>;
    case 8: return (const void *)k_acm_resident<T, CP, 8>;
    default: return nullptr;
    }
}

bool persist_block_ok(int block) { return block == 32 || block == 64 || block == 128 || block == 256; }

template <typename T, bool CP, bool SH>
const void *grid_kernel(int group) {
    switch (group) {
    case 1: return (const void *)k_acm_persistent<T, CP, false, 1, SH>;
    case 2: return (const void *)k_acm_persistent<T, CP, false, 2, SH>;
    case 4: return (const void *)k_acm_persistent<T, CP, false, 4, SH>;
    case 8: return (const void *)k_acm_persistent<T, CP, false, 8, SH>;
    default: return nullptr;
    }
}
template <typename T>
const void *grid_kernel(int group, bool cp, bool sh) {
    if (sh) return cp ? grid_kernel<T, true, true>(group) : grid_kernel<T, false, true>(group);
    return cp ? grid_kernel<T, true, false>(group) : grid_kernel<T, false, false>(group);
}

template <typename T, bool CP>
cudaError_t launch_cluster_T(const CellDesc<T> *cells_dev, const PersistCtl &ctl, int csize, size_t smem, cudaStream_t st,
                             int *max_clusters) {
    auto kern = k_acm_persistent<T, CP, true, 1, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(csize);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = csize;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (max_clusters) return cudaOccupancyMaxActiveClusters(max_clusters, kern, &cfg);
    return cudaLaunchKernelEx(&cfg, kern, cells_dev, ctl);
}

}  // namespace

template <typename T>
cudaError_t acm_launch_persistent(const CellDesc<T> *cells_dev, const PersistCtl &ctl, int nblocks, int block,
                                  int group, bool cp, cudaStream_t st) {
    if (!persist_block_ok(block) || nblocks < 1) return cudaErrorInvalidValue;
    const bool sh = persist_shared<T>(ctl.ncells, block);
    const void *fn = grid_kernel<T>(group, cp, sh);
    if (!fn) return cudaErrorInvalidValue;
    const size_t smem = persist_head_bytes<T>(ctl.ncells, sh);
    void *args[] = {(void *)&cells_dev, (void *)&ctl};
    return cudaLaunchCooperativeKernel(fn, dim3(nblocks), dim3(block), args, smem, st);
}

template <typename T>
cudaError_t acm_launch_persistent_cluster(const CellDesc<T> *cells_dev, const PersistCtl &ctl, int csize, bool cp,
                                          cudaStream_t st) {
    if (csize != 8 && csize != 16) return cudaErrorInvalidValue;
    const size_t smem = persist_head_bytes<T>(ctl.ncells, false);
    return cp ? launch_cluster_T<T, true>(cells_dev, ctl, csize, smem, st, nullptr)
              : launch_cluster_T<T, false>(cells_dev, ctl, csize, smem, st, nullptr);
}

template <typename T>
cudaError_t acm_persistent_cluster_ok(int csize, bool cp, size_t smem, bool *ok) {
    *ok = false;
    if (csize != 8 && csize != 16) return cudaErrorInvalidValue;
    int n = 0;
    cudaError_t e = cp ? launch_cluster_T<T, true>(nullptr, PersistCtl{}, csize, smem, nullptr, &n)
                       : launch_cluster_T<T, false>(nullptr, PersistCtl{}, csize, smem, nullptr, &n);
    if (e != cudaSuccess) {
        cudaGetLastError();  // an unsupported size is an answer, not an error
        return cudaSuccess;
    }
    *ok = n >= 1;
    return cudaSuccess;
}

template <typename T>
cudaError_t acm_persistent_max_blocks(int *blocks, int block, int group, bool cp, int ncells) {
    if (!persist_block_ok(block)) return cudaErrorInvalidValue;
    const bool sh = persist_shared<T>(ncells, block);
    const size_t smem = persist_head_bytes<T>(ncells, sh);
    const void *fn = grid_kernel<T>(group, cp, sh);
    if (!fn) return cudaErrorInvalidValue;
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, block, smem);
    *blocks = sms * per;
    return e;
}

template <typename T>
bool acm_resident_plan(int64_t n, int64_t nb, int n_l, int group, int sms, int64_t room, ResPlan *pl) {
    const int nu = 32 / group;
    const int64_t units = ((n + 31) >> 5) * group, wunits = ((nb + 31) >> 5) * group;
    pl->nblocks = (int)std::max<int64_t>(1, std::min<int64_t>(sms, units));
    const int64_t u = (units + pl->nblocks - 1) / pl->nblocks, wu = (wunits + pl->nblocks - 1) / pl->nblocks;
    if (u * nu * n_l * 4 * (int64_t)sizeof(T) > room) return false;
    pl->room = (int)room;
    pl->units = (int)u;
    pl->wunits = (int)wu;
    pl->loc = 0;
    const int64_t fixed = res_offsets<T>(*pl, n_l, nu).total + 64;
    int64_t loc = (room - fixed) / (4 * (int64_t)sizeof(T) + 6);
    loc = std::min<int64_t>(loc, std::min<int64_t>(65532, (n + 3) & ~(int64_t)3)) & ~(int64_t)3;
    // room for the set-up's bits and ranks, and for a halo (at least a stencil's reach)
    const int64_t bits = 8 * ((n + 31) / 32);
    if (loc < 64 || 4 * loc * (int64_t)sizeof(T) < bits || loc < u * nu) return false;
    pl->loc = (int)loc;
    pl->smem = res_offsets<T>(*pl, n_l, nu).total;
    return pl->smem <= room;
}

template <typename T>
cudaError_t acm_launch_resident(const CellDesc<T> &cell, const PersistCtl &ctl, const ResPlan &pl, int block, int group,
                                bool cp, cudaStream_t st) {
    const void *fn = cp ? resident_kernel<T, true>(group) : resident_kernel<T, false>(group);
    if (block < 32 || block % 32 || block > (sizeof(T) == 4 ? 1024 : 512) || !fn) return cudaErrorInvalidValue;
    // the kernel's limit is one for all threads of the program: always the same value
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, pl.room);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)&cell, (void *)&ctl, (void *)&pl};
    return cudaLaunchCooperativeKernel(fn, dim3(pl.nblocks), dim3(block), args, (size_t)pl.smem, st);
}

#define RBF_PERSIST_INST(T)                                                                                            \
    template cudaError_t acm_launch_persistent<T>(const CellDesc<T> *, const PersistCtl &, int, int, int, bool,        \
                                                  cudaStream_t);                                                       \
    template cudaError_t acm_persistent_max_blocks<T>(int *, int, int, bool, int);                                  \
    template cudaError_t acm_launch_persistent_cluster<T>(const CellDesc<T> *, const PersistCtl &, int, bool,          \
                                                          cudaStream_t);                                               \
    template cudaError_t acm_persistent_cluster_ok<T>(int, bool, size_t, bool *);                                      \
    template bool acm_resident_plan<T>(int64_t, int64_t, int, int, int, int64_t, ResPlan *);                           \
    template cudaError_t acm_launch_resident<T>(const CellDesc<T> &, const PersistCtl &, const ResPlan &, int, int,    \
                                                bool, cudaStream_t);
RBF_PERSIST_INST(float)
RBF_PERSIST_INST(double)

}  // namespace rbf
