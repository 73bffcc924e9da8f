// k_generic_step.cuh -- the generic fused stream-collide kernel: one cell per thread
// (grid-stride), populations read and written directly in global memory by the AA
// pattern.  Works for any lattice size and every storage precision; used for ragged
// sizes, for FP64 storage (bound by the FP64 pipe, not by memory) and as the fallback
// of the TMA row-staged kernel.
//
// AA pattern (in place, one array).  Even step: cell r reads its own slots A[i][r],
// collides, and writes f*_i to the opposite slot A[opp(i)][r].  Odd step: cell r reads
// f_i = A[opp(i)][r - c_i] (the value the neighbour r - c_i left for it), collides, and
// writes f*_i to A[i][r + c_i].  Every location is read and written by the same cell, so
// no two threads touch one location within a step.  Two steps together perform two
// collide-then-stream updates of Eq. (1).
#pragma once

#include "lbm_common.cuh"
#include "ptx.cuh"

namespace lbmd {

// A population, from L2 where other SMs write it during the launch.
template <bool L2, typename T> __device__ __forceinline__ T ld_pop(const T *p) {
    if constexpr (L2) return __ldcg(p);
    else return *p;
}

// One AA-pattern update of cell (x, y, z) of a lattice stored as Q planes of `plane`
// elements at A; returns the cell's pre-collision moments.  L2: the populations are read past
// the SM's own cache (several steps in one launch, blocks that exchange populations).
template <int D, int P, int EQ, bool BULK, bool L2 = false>
__device__ __forceinline__ CellMoments<typename Storage<P>::R> aa_cell_step(
    typename Storage<P>::T *__restrict__ A, int64_t plane, int nx, int ny, int nz, int pitch, int x, int y,
    int z, int odd, typename Storage<P>::R rho0, typename Storage<P>::R omega0,
    typename Storage<P>::R six_nu, int32_t *status = nullptr) {
    using St = Storage<P>;
    using R = typename St::R;
    constexpr int Q = qof(D);
    // checked builds: the cell and (through the periodic wrap) all its neighbours lie
    // inside the lattice, so every index below stays inside the Q planes
    if (!LBM_CHECK(x >= 0 && x < nx && y >= 0 && y < ny && z >= 0 && z < nz &&
                       (int64_t)pitch * ny * nz <= plane, status)) {
        CellMoments<R> none{};
        return none;
    }
    const int64_t cell = x + (int64_t)pitch * (y + (int64_t)ny * z);
    const int xs[3] = {wrapi(x - 1, nx), x, wrapi(x + 1, nx)};
    const int ys[3] = {wrapi(y - 1, ny), y, wrapi(y + 1, ny)};
    const int zs[3] = {D == 3 ? wrapi(z - 1, nz) : z, z, D == 3 ? wrapi(z + 1, nz) : z};
    R f[Q];
    if (!odd) {
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = St::load(ld_pop<L2>(A + (int64_t)i * plane + cell));
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            // f_i(r) = A[opp(i)][r - c_i]
            const int64_t src = xs[1 - cxo(i)] +
                                (int64_t)pitch * (ys[1 - cyo(i)] + (int64_t)ny * zs[1 - (D == 3 ? czo(i) : 0)]);
            f[i] = St::load(ld_pop<L2>(A + (int64_t)(Q - 1 - i) * plane + src));
        }
    }
    const CellMoments<R> m = collide<D, P, EQ, BULK, R>(f, rho0, omega0, six_nu);
    if (!odd) {
#pragma unroll
        for (int i = 0; i < Q; ++i) A[(int64_t)(Q - 1 - i) * plane + cell] = St::store(f[i]);
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int64_t dst = xs[1 + cxo(i)] +
                                (int64_t)pitch * (ys[1 + cyo(i)] + (int64_t)ny * zs[1 + (D == 3 ? czo(i) : 0)]);
            A[(int64_t)i * plane + dst] = St::store(f[i]);
        }
    }
    return m;
}

template <int D, int P, int EQ, bool BULK>
__global__ void __launch_bounds__(256) k_step_generic(const lbmh::StepArgs a) {
    using St = Storage<P>;
    using T = typename St::T;
    using R = typename St::R;
    T *__restrict__ A = static_cast<T *>(a.lat.A);
    const int nx = a.lat.nx, ny = a.lat.ny, nz = a.lat.nz;
    const R rho0 = step_scalar<R>(a.rho0, a.rho0f), omega0 = step_scalar<R>(a.omega0, a.omega0f),
            six_nu = step_scalar<R>(a.six_nu, a.six_nuf);
    DiagAcc acc;
    DiagLocal<R> loc;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t cell = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; cell < a.lat.ncell;
         cell += stride) {
        int x, y, z;
        cell_coords(cell, a.lat.ncell, nx, ny, x, y, z);
        const CellMoments<R> m = aa_cell_step<D, P, EQ, BULK>(A, a.lat.plane, nx, ny, nz, a.lat.pitch, x, y, z,
                                                              a.odd, rho0, omega0, six_nu, a.status);
        if (a.diag) {
            loc.add(m.rho, m.u, rho0);
            if (loc.count == 16) loc.flush(acc, a.rho0);
        }
    }
    if (a.diag) {
        loc.flush(acc, a.rho0);
        diag_block_store(acc, a.partials + (int64_t)blockIdx.x * lbmh::kDiagWords);
    }
}

// ------------------------------------------------------------------ several steps at once
//
// A small lattice's steps are bound by latency: a launch, a pipeline's ramp, or in the TMA row
// kernel's several-step form the way of a row through shared memory and its counters.  Here all
// its cells are in registers at once, one (or a few) to a thread: a step is a load of the
// populations from L2, the collision, the stores and one barrier of the whole grid (cooperative
// launch: all blocks are resident).  The barrier's arrivals are spread over kBarCounters counters,
// each on its own line; a block's first warp looks at all of them.  Per step against the TMA row
// kernel: 90^2 FP64 8.2 -> 4.6 us (2.6 us of it one warp's 82 FP64 instructions at 64 clocks),
// 64^2 FP32 3.9 -> 2.1, 32^3 binary16 6.1 -> 2.8, 48^3 6.8 -> 5.7 us.

// Wait until every block has arrived `gen` times (counters never wrap: gen * blocks < 2^32).
__device__ __forceinline__ bool grid_barrier(unsigned *sync, unsigned gen, const int32_t *status, int64_t timeout_ns) {
    __shared__ int bad;
    __syncthreads();  // every store of the block is issued
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0) {
            bad = 0;
            red_release(&sync[lbmh::kBarStride * (1 + blockIdx.x % lbmh::kBarCounters)], 1u);
        }
        bool ok = true;
        if (threadIdx.x < lbmh::kBarCounters && threadIdx.x < gridDim.x) {
            const unsigned arrive = (gridDim.x - threadIdx.x + lbmh::kBarCounters - 1) / lbmh::kBarCounters;
            ok = wait_count_bounded(&sync[lbmh::kBarStride * (1 + threadIdx.x)], gen * arrive, status, timeout_ns);
        }
        if (__any_sync(0xffffffffu, !ok) && threadIdx.x == 0) bad = 1;
    }
    __syncthreads();
    return bad == 0;
}

// The same for the blocks of one counter (it grows by the number of blocks a step).
__device__ __forceinline__ bool team_barrier(unsigned *counter, unsigned want, const int32_t *status, int64_t timeout_ns) {
    __shared__ int bad;
    __syncthreads();
    if (threadIdx.x == 0) {
        red_release(counter, 1u);
        bad = !wait_count_bounded(counter, want, status, timeout_ns);
    }
    __syncthreads();
    return bad == 0;
}

// The end of a several-step launch: reports a wait that ran out; the last block to finish clears
// the counters for the next launch.
__device__ __forceinline__ void steps_finish(const lbmh::StepArgs &a, bool ok) {
    if (!ok && threadIdx.x == 0) report_status(a.status, -5); /* LBM_ETIMEOUT */
    __syncthreads();
    bool last = false;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&a.sync[1], 1u) == gridDim.x - 1;
    }
    if (__syncthreads_or(last))
        for (int p = threadIdx.x; p < lbmh::kBarStride * (1 + lbmh::kBarCounters); p += blockDim.x) a.sync[p] = 0;
}

template <int D, int P, int EQ, bool BULK>
__global__ void __launch_bounds__(256) k_steps_small(const lbmh::StepArgs a, int nsteps) {
    using St = Storage<P>;
    using T = typename St::T;
    using R = typename St::R;
    constexpr int Q = qof(D);
    T *A = static_cast<T *>(a.lat.A);
    const int nx = a.lat.nx, ny = a.lat.ny, nz = a.lat.nz, pitch = a.lat.pitch;
    const int plane = (int)a.lat.plane, ncell = (int)a.lat.ncell;  // Q * plane < 2^31 (checked on the host)
    const R rho0 = step_scalar<R>(a.rho0, a.rho0f), omega0 = step_scalar<R>(a.omega0, a.omega0f),
            six_nu = step_scalar<R>(a.six_nu, a.six_nuf);
    bool ok = true;
    int here = -1, xs[3], rows[9];  // the thread's cell and its neighbours: columns, row starts by (dy + 1) + 3 (dz + 1)
    for (int s = 0; s < nsteps && ok; ++s) {
        const int odd = (a.odd + s) & 1;
        for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < ncell; cell += gridDim.x * blockDim.x) {
            if (cell != here) {  // once, where a thread has one cell
                int x, y, z;
                cell_coords(cell, ncell, nx, ny, x, y, z);
                here = cell;
                xs[0] = wrapi(x - 1, nx);
                xs[1] = x;
                xs[2] = wrapi(x + 1, nx);
#pragma unroll
                for (int q = 0; q < (D == 3 ? 9 : 3); ++q) {
                    const int yy = wrapi(y + q % 3 - 1, ny), zz = D == 3 ? wrapi(z + q / 3 - 1, nz) : z;
                    rows[q] = pitch * (yy + ny * zz);
                }
            }
            const int self = rows[D == 3 ? 4 : 1] + xs[1];
            if (!LBM_CHECK(self >= 0 && self < plane, a.status)) continue;
            R f[Q];
            if (!odd) {
#pragma unroll
                for (int i = 0; i < Q; ++i) f[i] = St::load(ld_pop<true>(A + i * plane + self));
            } else {
#pragma unroll
                for (int i = 0; i < Q; ++i)  // f_i(r) = A[opp(i)][r - c_i]
                    f[i] = St::load(ld_pop<true>(A + (Q - 1 - i) * plane + rows[(1 - cyo(i)) + (D == 3 ? 3 * (1 - czo(i)) : 0)] + xs[1 - cxo(i)]));
            }
            collide<D, P, EQ, BULK, R>(f, rho0, omega0, six_nu);
            if (!odd) {
#pragma unroll
                for (int i = 0; i < Q; ++i) A[(Q - 1 - i) * plane + self] = St::store(f[i]);
            } else {
#pragma unroll
                for (int i = 0; i < Q; ++i)
                    A[i * plane + rows[(1 + cyo(i)) + (D == 3 ? 3 * (1 + czo(i)) : 0)] + xs[1 + cxo(i)]] = St::store(f[i]);
            }
        }
        if (s + 1 < nsteps) ok = grid_barrier(a.sync, (unsigned)(s + 1), a.status, a.timeout_ns);
    }
    steps_finish(a, ok);
}

// A cell on three lanes of a warp (collide_lanes), ten cells to a warp: the lane's share of the
// loads and stores.  Lane c of a group has the directions i = p + F c.
template <int D> struct LaneCell {
    static constexpr int Q = qof(D), F = lane_pops(D), N = D == 3 ? 3 : 1;
    int c, base, x, y, z, plane, self, xs[3];
    int ahead[N], behind[N];  // rows of r + c e_last + dy and of their mirror images, by dy + 1 (3-D)
    bool run;                 // the group has a cell of its own
    // first: the first cell of the block (cells first .. ncell are the block's and its successors')
    __device__ __forceinline__ LaneCell(int first, int ncell, int nx, int ny, int nz, int pitch, int plane_, int32_t *status)
        : plane(plane_) {
        const int lane = threadIdx.x & 31, cell = first + (int)(threadIdx.x >> 5) * 10 + lane / 3;
        c = lane % 3;
        base = lane < 30 ? lane - c : 27;  // (lanes 30 and 31 only take part in the shuffles)
        run = lane < 30 && cell < ncell;
        cell_coords(run ? cell : 0, ncell, nx, ny, x, y, z);
        self = x + pitch * (y + ny * z);
        xs[0] = wrapi(x - 1, nx);
        xs[1] = x;
        xs[2] = wrapi(x + 1, nx);
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const int dy = D == 3 ? q - 1 : c - 1, dz = D == 3 ? c - 1 : 0;
            ahead[q] = pitch * (wrapi(y + dy, ny) + (D == 3 ? ny * wrapi(z + dz, nz) : 0));
            behind[q] = pitch * (wrapi(y - dy, ny) + (D == 3 ? ny * wrapi(z - dz, nz) : 0));
        }
        run = run && LBM_CHECK(self >= 0 && self < plane, status);
    }
    __device__ __forceinline__ void load(const double *A, int odd, double (&f)[F]) const {
#pragma unroll
        for (int p = 0; p < F; ++p) {
            f[p] = 0.0;  // f_i(r) = A[opp(i)][r - c_i] on odd steps
            if (run && odd) f[p] = ld_pop<true>(A + (Q - 1 - p - F * c) * plane + behind[D == 3 ? p / 3 : 0] + xs[1 - cxo(p)]);
            if (run && !odd) f[p] = ld_pop<true>(A + (p + F * c) * plane + self);
        }
    }
    __device__ __forceinline__ void store(double *A, int odd, const double (&f)[F]) const {
#pragma unroll
        for (int p = 0; p < F; ++p) {
            if (run && odd) A[(p + F * c) * plane + ahead[D == 3 ? p / 3 : 0] + xs[1 + cxo(p)]] = f[p];
            if (run && !odd) A[(Q - 1 - p - F * c) * plane + self] = f[p];
        }
    }
};

// Several steps of an FP64 lattice of at most 40 cells an SM: a warp of ten cells to each quarter,
// one cell to a group of lanes.  Entropic with bulk correction, a cell per thread against three
// lanes: 64^2 5.1 -> 4.0 us a step, 80 x 76 5.1 -> 4.2, 16^3 9.4 -> 6.0, 20 x 16 x 19 9.5 -> 6.4.
template <int D, int EQ, bool BULK>
__global__ void __launch_bounds__(128) k_steps_lanes(const lbmh::StepArgs a, int nsteps) {
    double *A = static_cast<double *>(a.lat.A);
    const LaneCell<D> cell((int)(blockIdx.x * (blockDim.x / 32) * 10), (int)a.lat.ncell, a.lat.nx, a.lat.ny, a.lat.nz,
                           a.lat.pitch, (int)a.lat.plane, a.status);  // Q * plane < 2^31 (checked on the host)
    bool ok = true;
    for (int s = 0; s < nsteps && ok; ++s) {
        const int odd = (a.odd + s) & 1;
        double f[LaneCell<D>::F];
        cell.load(A, odd, f);
        collide_lanes<D, EQ, BULK>(f, cell.c, cell.base, a.rho0, a.omega0, a.six_nu);
        cell.store(A, odd, f);
        if (s + 1 < nsteps) ok = grid_barrier(a.sync, (unsigned)(s + 1), a.status, a.timeout_ns);
    }
    steps_finish(a, ok);
}

template <int D> const void *lanes_kernel_d(int eq, int bulk) {
#define LBM_LANES(EQv) \
    if (eq == EQv) return bulk ? (const void *)k_steps_lanes<D, EQv, true> : (const void *)k_steps_lanes<D, EQv, false>;
    LBM_LANES(EQ_ENT)
    LBM_LANES(EQ_POLY2)
    LBM_LANES(EQ_PROD)
#undef LBM_LANES
    return nullptr;
}

template <int D, int P> const void *small_kernel_dp(int eq, int bulk) {
#define LBM_SMALL(EQv) \
    if (eq == EQv) return bulk ? (const void *)k_steps_small<D, P, EQv, true> : (const void *)k_steps_small<D, P, EQv, false>;
    LBM_SMALL(EQ_ENT)
    LBM_SMALL(EQ_POLY2)
    LBM_SMALL(EQ_PROD)
#undef LBM_SMALL
    return nullptr;
}

template <int D, int P>
cudaError_t launch_generic_dp(const lbmh::StepArgs &a, int blocks, int threads, cudaStream_t s) {
#define LBM_GEN(EQv, Bv)                                                                   \
    if (a.eq == EQv && a.bulk == Bv) {                                                     \
        k_step_generic<D, P, EQv, Bv><<<blocks, threads, 0, s>>>(a);                        \
        return cudaGetLastError();                                                          \
    }
    LBM_GEN(EQ_ENT, false)
    LBM_GEN(EQ_ENT, true)
    LBM_GEN(EQ_POLY2, false)
    LBM_GEN(EQ_POLY2, true)
    LBM_GEN(EQ_PROD, false)
    LBM_GEN(EQ_PROD, true)
#undef LBM_GEN
    return cudaErrorInvalidValue;
}

}  // namespace lbmd
