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
    typename Storage<P>::R six_nu, int32_t *status) {
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

// DIAG: with the diagnostics' sums (see tma_compute on why not a run-time condition).
template <int D, int P, int EQ, bool BULK, bool DIAG>
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
        if (DIAG) {
            loc.add(m.rho, m.u, rho0);
            if (loc.count == 16) loc.flush(acc, a.rho0);
        }
    }
    if (DIAG) {
        loc.flush(acc, a.rho0);
        diag_block_store(acc, a.partials + (int64_t)blockIdx.x * lbmh::kDiagWords);
    }
}

// ------------------------------------------------------------------ several steps at once
//
// A small lattice's steps are bound by latency: a launch, a pipeline's ramp, or in the TMA row
// kernel's several-step form the way of a row through shared memory and its counters.  Here all
// its cells are in registers at once, one (or a few) to a thread, in one cooperative launch (all
// blocks are resident), and no barrier separates the steps: within the launch a population
// travels in one word with the number of the step that wrote it, through a buffer with the layout
// of the lattice (rows unpadded: a warp's cells are contiguous across the end of a row, 300^2
// binary16 1.8 us a step, 2.7 with the lattice's own padding).  A cell reads a location until it
// finds its own step's number there.  A location is read and then rewritten by one cell a step
// (the AA pattern), so nothing can be overwritten before it was read, and a word is written and
// read whole, so neither fences nor counters are needed: a step is a store, a load and the
// collision.  The first step reads and the last one writes the lattice's own array.  The numbers
// go on from launch to launch (the buffer's head, advanced by the last block), so the words of an
// earlier launch, all one behind the next launch's first, never match. Per step with the TMA row
// kernel, with a barrier of the whole grid in place of the numbers (release fence, counter,
// acquire: 1 us), and so: 64^2 FP32 3.9, 1.86, 0.91 us; 64^2 FP64 8.0, 3.45, 2.65; 32^3 binary16
// 6.1, 2.49, 1.57; 340^2 FP32 4.6, 3.16, 1.95; 48^3 binary16 6.8, 4.5, 4.1.
struct MsgHead {
    unsigned step, exits;
};

template <int P> struct Msg;
template <> struct Msg<P_F16S> {  // population, step modulo 2^16
    using W = uint32_t;
    static __device__ __forceinline__ bool take(const W *p, unsigned want, float &v) {
        W w;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(w) : "l"(p) : "memory");
        v = __half2float(__ushort_as_half((unsigned short)w));
        return w >> 16 == (want & 0xffffu);
    }
    static __device__ __forceinline__ void give(W *p, unsigned step, float v) {
        const W w = step << 16 | __half_as_ushort(Storage<P_F16S>::store(v));
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(w) : "memory");
    }
};
template <> struct Msg<P_F32> {
    using W = uint64_t;
    static __device__ __forceinline__ bool take(const W *p, unsigned want, float &v) {
        W w;
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
        v = __uint_as_float((unsigned)w);
        return (unsigned)(w >> 32) == want;
    }
    static __device__ __forceinline__ void give(W *p, unsigned step, float v) {
        const W w = (W)step << 32 | __float_as_uint(v);
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
    }
};
template <> struct Msg<P_F64> {  // two words, a half of the population and the step in each
    using W = ulonglong2;
    static __device__ __forceinline__ bool take(const W *p, unsigned want, double &v) {
        unsigned long long x, y;
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
        v = __hiloint2double((int)(unsigned)y, (int)(unsigned)x);
        return (unsigned)(x >> 32) == want && (unsigned)(y >> 32) == want;
    }
    static __device__ __forceinline__ void give(W *p, unsigned step, double v) {
        const unsigned long long t = (unsigned long long)step << 32;
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | (unsigned)__double2loint(v)),
                     "l"(t | (unsigned)__double2hiint(v))
                     : "memory");
    }
};

// Reads the populations f[p] = M[at(p)] of the lanes that `run` until all of the warp's carry the
// number `want` (the lanes go on together: a collision in two halves of a warp takes twice as long,
// 90^2 FP64 6.8 against 3.6 us a step); false when the wait runs out or another thread has reported
// an error.  All 32 lanes call it.
template <int P, int N, typename R, typename At>
__device__ __forceinline__ bool msg_take(const typename Msg<P>::W *M, unsigned want, R (&f)[N], const At &at, bool run,
                                         const int32_t *status, int64_t timeout_ns) {
    uint64_t t0 = 0;
    for (int tries = 1;; ++tries) {
        bool all = true;
        if (run) {
#pragma unroll
            for (int p = 0; p < N; ++p) all &= Msg<P>::take(M + at(p), want, f[p]);
        }
        if (__all_sync(0xffffffffu, all)) return true;
        if (tries % 64 == 0) {
            if (t0 == 0) t0 = global_ns();
            const bool stop = *(const volatile int32_t *)status != 0 || (int64_t)(global_ns() - t0) > timeout_ns;
            if (__any_sync(0xffffffffu, stop)) return false;
        }
    }
}

// The end of a several-step launch: reports a wait that ran out; the last block to finish moves the
// step number on.
__device__ __forceinline__ void steps_finish(const lbmh::StepArgs &a, int nsteps, bool ok) {
    if (!ok) report_status(a.status, -5); /* LBM_ETIMEOUT */
    MsgHead *head = static_cast<MsgHead *>(a.msg);
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&head->exits, 1u) == gridDim.x - 1) {
        head->exits = 0;
        head->step += (unsigned)nsteps;
    }
}

// Barrier of the blocks of one counter, which grows by their number a step.  (The release orders the
// stores of the whole block: they precede it through the block's own barrier.)
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

template <int D, int P, int EQ, bool BULK, int MINB>
__global__ void __launch_bounds__(256, MINB) k_steps_small(const lbmh::StepArgs a, int nsteps) {
    using St = Storage<P>;
    using T = typename St::T;
    using R = typename St::R;
    using W = typename Msg<P>::W;
    constexpr int Q = qof(D);
    T *A = static_cast<T *>(a.lat.A);
    W *M = reinterpret_cast<W *>(static_cast<char *>(a.msg) + lbmh::kMsgHead);
    const unsigned step0 = __ldcg(&static_cast<const MsgHead *>(a.msg)->step);
    const int nx = a.lat.nx, ny = a.lat.ny, nz = a.lat.nz, pitch = a.lat.pitch;
    const int plane = (int)a.lat.plane, ncell = (int)a.lat.ncell;  // Q * plane < 2^31 (checked on the host)
    const R rho0 = step_scalar<R>(a.rho0, a.rho0f), omega0 = step_scalar<R>(a.omega0, a.omega0f),
            six_nu = step_scalar<R>(a.six_nu, a.six_nuf);
    bool ok = true;
    int here = -1, xs[3], rows[9];  // the thread's cell and its neighbours: columns, rows by (dy + 1) + 3 (dz + 1)
    for (int s = 0; s < nsteps && ok; ++s) {
        const int odd = (a.odd + s) & 1;
        for (int first = blockIdx.x * blockDim.x + (threadIdx.x & ~31); first < ncell && ok; first += gridDim.x * blockDim.x) {
            const int cell = min(first + (int)(threadIdx.x & 31), ncell - 1);
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
                    rows[q] = yy + ny * zz;
                }
            }
            const bool run = first + (int)(threadIdx.x & 31) < ncell &&
                             LBM_CHECK(here >= 0 && rows[D == 3 ? 4 : 1] * pitch + xs[1] < plane, a.status);
            R f[Q] = {};
            // where direction i is read and written: A[i][r] and A[opp(i)][r], odd steps
            // A[opp(i)][r - c_i] and A[i][r + c_i]
            const auto at = [&](int i, int c, int slot, int pit) {
                const int row = rows[(1 + c * cyo(i)) + (D == 3 ? 3 * (1 + c * czo(i)) : 0)];
                return slot * plane + row * pit + xs[1 + c * cxo(i)];
            };
            const auto in = [&](int i, int o, int pit) { return o ? at(i, -1, Q - 1 - i, pit) : at(i, 0, i, pit); };
            const auto out = [&](int i, int o, int pit) { return o ? at(i, 1, i, pit) : at(i, 0, Q - 1 - i, pit); };
            const auto take = [&](int o) {
                return msg_take<P>(M, step0 + s, f, [&](int i) { return in(i, o, nx); }, run, a.status, a.timeout_ns);
            };
            const auto give = [&](int o) {
#pragma unroll
                for (int i = 0; i < Q; ++i) Msg<P>::give(M + out(i, o, nx), step0 + s + 1, f[i]);
            };
            // Even and odd code of its own where registers are scarce (48^3 binary16 4.1 against 5.4 us
            // a step, 512^2 4.1 against 4.5); one code with the parity's addresses chosen where they
            // are not: the compiler then keeps fewer of them (32^3 1.6 against 1.8).
            if (s == 0) {
#pragma unroll
                for (int i = 0; i < Q; ++i)
                    if (run) f[i] = St::load(A[in(i, odd, pitch)]);
            } else if (MINB == 1) {
                ok = take(odd);
            } else if (odd) {
                ok = take(1);
            } else {
                ok = take(0);
            }
            if (!ok) break;
            collide<D, P, EQ, BULK, R>(f, rho0, omega0, six_nu);
            if (!run) continue;
            if (s + 1 == nsteps) {
#pragma unroll
                for (int i = 0; i < Q; ++i) A[out(i, odd, pitch)] = St::store(f[i]);
            } else if (MINB == 1) {
                give(odd);
            } else if (odd) {
                give(1);
            } else {
                give(0);
            }
        }
    }
    steps_finish(a, nsteps, ok);
}

// A cell on three lanes of a warp (collide_lanes), ten cells to a warp: the lane's share of the
// loads and stores.  Lane c of a group has the directions i = p + F c.
template <int D> struct LaneCell {
    static constexpr int Q = qof(D), F = lane_pops(D), N = D == 3 ? 3 : 1;
    int c, base, plane, self, xs[3];
    int ahead[N], behind[N];  // rows of r + c e_last + dy and of their mirror images, by dy + 1 (3-D)
    bool run;                 // the group has a cell of its own
    // first: the first cell of the block (cells first .. ncell are the block's and its successors')
    __device__ __forceinline__ LaneCell(int first, int ncell, int nx, int ny, int nz, int pitch, int plane_, int32_t *status)
        : plane(plane_) {
        const int lane = threadIdx.x & 31, cell = first + (int)(threadIdx.x >> 5) * 10 + lane / 3;
        c = lane % 3;
        base = lane < 30 ? lane - c : 27;  // (lanes 30 and 31 only take part in the shuffles)
        run = lane < 30 && cell < ncell;
        int x, y, z;
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
    // where direction p + F c is read and written
    __device__ __forceinline__ int in(int p, int odd) const {
        return odd ? (Q - 1 - p - F * c) * plane + behind[D == 3 ? p / 3 : 0] + xs[1 - cxo(p)] : (p + F * c) * plane + self;
    }
    __device__ __forceinline__ int out(int p, int odd) const {
        return odd ? (p + F * c) * plane + ahead[D == 3 ? p / 3 : 0] + xs[1 + cxo(p)] : (Q - 1 - p - F * c) * plane + self;
    }
};

// Several steps of an FP64 lattice of at most 40 cells an SM: a warp of ten cells to each quarter,
// one cell to a group of lanes.  Entropic with bulk correction, a cell per thread against three
// lanes (with the grid's barrier in both): 64^2 5.1 -> 4.0 us a step, 80 x 76 5.1 -> 4.2,
// 16^3 9.4 -> 6.0, 20 x 16 x 19 9.5 -> 6.4.
template <int D, int EQ, bool BULK>
__global__ void __launch_bounds__(128) k_steps_lanes(const lbmh::StepArgs a, int nsteps) {
    using W = Msg<P_F64>::W;
    constexpr int F = lane_pops(D);
    double *A = static_cast<double *>(a.lat.A);
    W *M = reinterpret_cast<W *>(static_cast<char *>(a.msg) + lbmh::kMsgHead);
    const unsigned step0 = __ldcg(&static_cast<const MsgHead *>(a.msg)->step);
    const LaneCell<D> cell((int)(blockIdx.x * (blockDim.x / 32) * 10), (int)a.lat.ncell, a.lat.nx, a.lat.ny, a.lat.nz,
                           a.lat.pitch, (int)a.lat.plane, a.status);  // Q * plane < 2^31 (checked on the host)
    bool ok = true;
    for (int s = 0; s < nsteps; ++s) {
        const int odd = (a.odd + s) & 1;
        double f[F] = {};
        if (s == 0) {
#pragma unroll
            for (int p = 0; p < F; ++p) if (cell.run) f[p] = A[cell.in(p, odd)];
        } else {
            ok = msg_take<P_F64>(M, step0 + s, f, [&](int p) { return cell.in(p, odd); }, cell.run, a.status, a.timeout_ns);
            if (!ok) break;
        }
        collide_lanes<D, EQ, BULK>(f, cell.c, cell.base, a.rho0, a.omega0, a.six_nu);
        if (cell.run) {
#pragma unroll
            for (int p = 0; p < F; ++p) {
                if (s + 1 == nsteps) A[cell.out(p, odd)] = f[p];
                else Msg<P_F64>::give(M + cell.out(p, odd), step0 + s + 1, f[p]);
            }
        }
    }
    steps_finish(a, nsteps, ok);
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

template <int D, int P> const void *small_kernel_dp(int eq, int bulk, bool many) {
    constexpr int B = lbmh::small_blocks(D, P);
#define LBM_SMALL(EQv)                                                                          \
    if (eq == EQv && !many)                                                                     \
        return bulk ? (const void *)k_steps_small<D, P, EQv, true, 1> : (const void *)k_steps_small<D, P, EQv, false, 1>; \
    if (eq == EQv)                                                                              \
        return bulk ? (const void *)k_steps_small<D, P, EQv, true, B> : (const void *)k_steps_small<D, P, EQv, false, B>;
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
        if (a.diag) k_step_generic<D, P, EQv, Bv, true><<<blocks, threads, 0, s>>>(a);      \
        else k_step_generic<D, P, EQv, Bv, false><<<blocks, threads, 0, s>>>(a);            \
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
