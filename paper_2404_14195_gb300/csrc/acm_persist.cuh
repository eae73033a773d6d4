// acm_persist.cuh — per-cell descriptors and control block of the persistent
// multi-cell ACM driver (acm_persist.cu).
#pragma once
#include "internal.cuh"

namespace rbf {

#define PERSIST_MAX_CELLS 128

template <typename T>
struct CellDesc {
    int64_t n, nb;
    int n_l;
    int64_t parity0;         // slot parity of this cell's next pressure iteration
    const int32_t *idx;      // SELL [slice][j][lane]
    const T *w;              // SELL [slice][4][j][lane]
    const uint8_t *type;
    const int32_t *wall;
    const int32_t *idxb;     // wall Neumann stencils, SELL over the wall list
    const T *wn;
    T *u, *v, *w_, *p;
    T *us, *vs, *ws;
    T *uo, *vo, *wo;         // snapshot for the residual
    // compensated state (RBF_FP32C, else null): low words of u, v, w, p, u', v',
    // w' and of the snapshot
    T *ul, *vl, *wl, *pl, *usl, *vsl, *wsl, *uol, *vol, *wol;
    unsigned long long *vmax;  // 2 slots
    T dt, nu, gx, gy, gz, rho;
    double beta, vref;
};

struct PersistCtl {
    unsigned *bar;           // barrier words (acm_persist.cu), zero at launch, 256 bytes
    int32_t *err;            // 2 = a grid barrier timed out
    int32_t *done;           // per cell: 0 running, 1 converged, 3 non-finite residual
    int64_t *steps;          // per cell: steps taken in this launch
    double *resid;           // per cell: last residual
    double *partial;         // [block][PERSIST_MAX_CELLS][2]
    int ncells;
    int64_t max_steps;
    int check_every;
    double tol;
    int n_p;
    uint64_t wait_ns;        // wall-clock limit of one grid-barrier wait (nanoseconds)
    unsigned long long *vsq; // resident kernel: 2 slots of max |v|^2
};

// warps of the streaming kernel's grid on an SM
template <typename T>
constexpr int persist_warps() { return sizeof(T) == 4 ? 32 : 24; }
// Whether its blocks of `block` threads copy the descriptors to shared memory: while an SM's copies
// take 64 kB at most.  A field's address is then a shared-memory load, but the copies take
// room from the L1, and from the blocks themselves past that.  Time with copies over time
// without, FP32 (FP64 within 2 %), by cells / threads (kB of copies per SM):
//   1 / 256 (1) 0.96, 12 / 256 (14) 0.96, 24 / 256 (28) 0.95, 24 / 128 (55) 0.96, 64 / 256 (74) 0.98 to 1.01,
//   40 / 128 (92) 0.96, 12 / 32 (111) 1.01, 64 / 128 (147) 1.15 to 1.21, 40 / 64 (184) 1.91
template <typename T>
constexpr bool persist_shared(int ncells, int block) {
    return (int64_t)ncells * (int64_t)sizeof(CellDesc<T>) * (persist_warps<T>() * 32 / block) <= 65536;
}
// its shared memory: descriptors, residual accumulators, unit counts ahead of each cell, flags; below
// the 48 kB that a launch may ask for without further ado
template <typename T>
constexpr int64_t persist_head_bytes(int ncells, bool shared) {
    return ((shared ? ncells : 0) * (int64_t)sizeof(CellDesc<T>) + (ncells + 1) * 16ll + ncells * 16ll + ncells * 4ll + 15) & ~15ll;
}
// Shares of the resident kernel (one cell, every block's stencils in shared memory):
// largest number of units and wall units per block, local nodes there is room for,
// dynamic shared memory, blocks; room: what a block may take.
struct ResPlan {
    int units, wunits, loc, smem, nblocks, room;
};
// whether a cell can run resident with `room` bytes of shared memory on each of `sms` SMs (its
// local sets are only known to the kernel, which raises error 3 before the first step if one has
// no room)
template <typename T>
bool acm_resident_plan(int64_t n, int64_t nb, int n_l, int group, int sms, int64_t room, ResPlan *pl);
template <typename T>
cudaError_t acm_launch_resident(const CellDesc<T> &cell, const PersistCtl &ctl, const ResPlan &pl, int block, int group,
                                bool cp, cudaStream_t st);

// cp selects the compensated kernel (every cell then carries low words); block:
// threads per block, 32, 64, 128 or 256; group: lanes per node,
// 1, 2, 4 or 8 (a warp takes 32 / group nodes of a slice at a time)
template <typename T>
cudaError_t acm_launch_persistent(const CellDesc<T> *cells_dev, const PersistCtl &ctl, int nblocks, int block,
                                  int group, bool cp, cudaStream_t st);
// co-resident blocks of the kernel over `ncells` cells
template <typename T>
cudaError_t acm_persistent_max_blocks(int *blocks, int block, int group, bool cp, int ncells);
// the same kernel as one thread-block cluster of csize (8 or 16) CTAs of 256
// threads, synchronised by the cluster barrier
template <typename T>
cudaError_t acm_launch_persistent_cluster(const CellDesc<T> *cells_dev, const PersistCtl &ctl, int csize, bool cp,
                                          cudaStream_t st);
// whether a cluster of csize CTAs of the kernel can be scheduled on this device
template <typename T>
cudaError_t acm_persistent_cluster_ok(int csize, bool cp, size_t smem, bool *ok);

}  // namespace rbf
