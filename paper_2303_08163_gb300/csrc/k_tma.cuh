// k_tma.cuh -- the TMA row-staged fused stream-collide kernel (AA pattern, in place).
//
// A job is a group of `rows` consecutive x-rows of one z-plane, or one aligned segment
// of `seg` cells of a row when the row is too long for shared memory.  For every
// population direction b the job needs one row piece ("buffer b"):
//   even step: plane b of the job's own rows, read at x, written back as the opposite
//              direction's post-collision value at x;
//   odd step:  plane opp(b) of the rows shifted by -c_b in y and z; cell x reads it at
//              x - c_bx (pulling f_b from its neighbour) and the same cell writes its
//              post-collision value of direction opp(b) there.
// Every position of buffer b is read by exactly one cell of the job and written by the
// same cell (the AA pattern's own property), so the collision runs in place in shared
// memory and buffer b is stored back to exactly the global location it was loaded from.
// Different jobs touch disjoint global locations, so jobs need no ordering.
//
// Data movement (warp specialised): after the colliding (consumer) warps come one or two service
// warps.  Lane b of a loading warp issues the cp.async.bulk copies of buffer b (global -> shared,
// completion counted in transaction bytes on the stage's `full` mbarrier).  Consumer warps wait on
// `full`, collide the job in place, fence their shared-memory writes for the async proxy and arrive
// on the stage's `empty` mbarrier.  Lane b of a storing warp then issues the cp.async.bulk stores of
// buffer b, and once they have read the stage it can be refilled.  Rows must start on 16-byte
// boundaries: the row pitch is a multiple of 16 bytes (a ragged row is padded to it, and whole rows
// are copied with their padding; the cells of the padding are never read by a real cell).
//
// Two kernels.  k_step_tma advances one step (jobs strided over the blocks, no waits between them; the
// diagnostics are reduced here): one service warp stores and refills.  k_steps_tma advances several
// (jobs by ticket, with counters of finished jobs; see decode_chain): a loader and a storer, because a
// loader that waits for another block's step must not hold up the stores that other blocks wait for.
// With both in one kernel (a loader and a storer for single steps too, registers for the longer
// body) single steps lost 2 % of 512^3 binary16 (2.19 -> 2.23 ms; now 2.18) and 3 % of 128^3, and
// several steps gained 2 % by the parting (512^3 1.67 -> 1.62 ms a step).
//
// Segmented rows (seg < Nx) carry a halo of U = 16 / sizeof(storage) cells on each side.
// In the odd step the cells of a segment touch positions [X0 - 1, X0 + len - 1) of the
// buffers with c_x = +1 and [X0 + 1, X0 + len + 1) of those with c_x = -1: the aligned
// interior goes back by bulk stores and the U ragged cells at each end by plain stores,
// so neighbouring segments never write the same location.
#pragma once

#include <type_traits>

#include "lbm_common.cuh"
#include "ptx.cuh"

namespace lbmd {

using lbmh::kTmaMaxStages;
constexpr int kTmaMaxThreads = 256;  // consumer threads of the D3Q27 kernels; two service warps more
// D2Q9 binary16 kernels (under 100 registers) may run up to 512 consumers
__host__ __device__ constexpr int tma_max_threads(int D, int P) { return D == 2 && P == 2 ? 512 : kTmaMaxThreads; }

// Division by a number fixed for the launch (dividends below 2^31): see the loader.
struct FastDiv {
    unsigned d, m, s;
};
__host__ inline FastDiv fast_div(unsigned d) {
    unsigned s = 0;
    while (s < 31 && (1u << s) < d) ++s;
    return {d, (unsigned)((((uint64_t)1 << (31 + s)) + d - 1) / d), 31 + s};  // m d - 2^(31+s) < d <= 2^s
}
__device__ __forceinline__ unsigned div_by(unsigned n, const FastDiv &f) { return (unsigned)(((uint64_t)n * f.m) >> f.s); }

// bufstride (elements between direction buffers) equals the compile-time buffer
// capacity CAPB / sizeof(storage) of the kernel instantiation.  rowstride is the distance
// between the rows of a job in shared memory: the row pitch for whole rows (the copies
// carry the padding along), the segment with its halos otherwise (rows without padding).
struct TmaGeom {
    int stages, rows, seg, nseg, ygroups, halo, rowstride, bufstride;
    int64_t njobs;
    // several steps in one launch (nsteps > 1), see decode_chain
    int nsteps, npos, ncross, strips, stripw, pjobs, depth, lag;
    FastDiv by_nseg, by_ygroups, by_npos, by_strips, by_pjobs, by_depth;
};

struct JobPos {
    int z, y0, nrows, X0, len;
    int odd;  // AA parity of the job's step
};

__device__ __forceinline__ JobPos job_at(const lbmh::StepArgs &a, const TmaGeom &g, int z, int yg, int s, int odd) {
    JobPos j;
    j.z = z;
    j.y0 = yg * g.rows;
    j.nrows = min(g.rows, a.lat.ny - j.y0);
    j.X0 = s * g.seg;
    j.len = min(g.seg, a.lat.nx - j.X0);
    j.odd = odd;
    return j;
}

// Single steps: job number -> rows and segment.
__device__ __forceinline__ JobPos decode_job(const lbmh::StepArgs &a, const TmaGeom &g, unsigned job) {
    const unsigned rest = div_by(job, g.by_nseg);
    const unsigned zq = div_by(rest, g.by_ygroups);
    return job_at(a, g, (int)zq, (int)(rest - zq * (unsigned)g.ygroups), (int)(job - rest * (unsigned)g.nseg), a.odd);
}

// Several steps (nsteps > 1).  The units of the lattice are its row groups, at position p of
// the sweep axis and c across it: (p, c) = (z, row group) in 3-D, (row group, 0) in 2-D.  Job
// (s, p, c, segment) -- step s -- needs step s - 1 of the units (p +- 1, c +- 1) (periodic) and
// nothing else: the AA pattern's locations that it reads and writes were last touched by
// cells of those.  A counter per unit holds its finished jobs.
//
// `depth` steps travel along the sweep axis together, each `lag` positions behind the one
// before, so that a position comes from HBM once for `depth` steps while the positions
// between the first and the last of them stay in L2.  Where whole positions are too large
// for that, they are cut across into `strips` swept one after the other; a strip moves down
// by one row group a step (its lower neighbour is done, its upper one is not), the first
// one shrinks from both ends and the last one grows into the periodic wrap:
//   strip k at inner step t covers c in [k H - t, (k + 1) H - t), from t in the first,
//   to ncross + t in the last.
// Step s starts at position s, so that its periodic neighbour is among the first that step
// s - 1 finished:
//   ticket -> (phase, t, job), phase - lag t = (q strips + k) npos + i, s = q depth + t,
//   p = (s + i) mod npos.
// Every job comes after the jobs it needs in ticket order (lag >= 2, npos > lag (depth - 1)
// + 2), and blocks take tickets from one counter, so whichever blocks are resident, the
// holder of the smallest unfinished ticket never waits: no deadlock, no need for all blocks
// to run at once.
struct ChainJob {
    JobPos j;
    int step, p, c;  // step < 0: no job (the ends of the wavefront and of the strips)
};

__host__ __device__ __forceinline__ void chain_strip(const TmaGeom &g, int k, int t, int &lo, int &hi) {
    lo = 0;
    hi = g.ncross;
    if (g.strips > 1) {
        lo = k == 0 ? t : k * g.stripw - t;
        hi = k == g.strips - 1 ? g.ncross + t : (k + 1) * g.stripw - t;
    }
}

__device__ __forceinline__ ChainJob decode_chain(const lbmh::StepArgs &a, const TmaGeom &g, unsigned ticket) {
    ChainJob r;
    const unsigned slot = div_by(ticket, g.by_pjobs);
    const unsigned jj = ticket - slot * (unsigned)g.pjobs;
    const unsigned phase = div_by(slot, g.by_depth);
    const int t = (int)(slot - phase * (unsigned)g.depth);
    const int x = (int)phase - g.lag * t;
    r.step = -1;
    r.p = r.c = 0;
    r.j = JobPos{0, 0, 0, 0, 0, 0};
    if (x < 0) return r;
    const int qk = (int)div_by((unsigned)x, g.by_npos), i = x - qk * g.npos;
    const int q = (int)div_by((unsigned)qk, g.by_strips), k = qk - q * g.strips;
    const int s = q * g.depth + t;
    if (s >= g.nsteps) return r;
    int lo, hi;
    chain_strip(g, k, t, lo, hi);
    const unsigned row = div_by(jj, g.by_nseg);
    int c = lo + (int)row;
    if (c >= hi) return r;
    if (c >= g.ncross) c -= g.ncross;
    r.step = s;
    r.p = s + i - (int)div_by((unsigned)(s + i), g.by_npos) * g.npos;
    r.c = c;
    const bool flat = a.lat.D == 2;
    r.j = job_at(a, g, flat ? 0 : r.p, flat ? r.p : c, (int)(jj - row * (unsigned)g.nseg), (a.odd + s) & 1);
    return r;
}

__host__ __device__ __forceinline__ int64_t chain_tickets(const TmaGeom &g) {
    const int64_t supers = (g.nsteps + g.depth - 1) / g.depth;
    return (supers * g.strips * g.npos + (int64_t)g.lag * (g.depth - 1)) * g.depth * g.pjobs;
}

// Global row (plane, y, z) of buffer b of a job.
template <int D, typename T>
__device__ __forceinline__ T *buffer_row(const lbmh::StepArgs &a, int odd, int b, int z, int y) {
    constexpr int Q = qof(D);
    const int plane = odd ? Q - 1 - b : b;
    const int zz = (D == 3 && odd) ? wrapi(z - czo(b), a.lat.nz) : z;
    const int yy = odd ? wrapi(y - cyo(b), a.lat.ny) : y;
    return static_cast<T *>(a.lat.A) + (int64_t)plane * a.lat.plane +
           ((int64_t)zz * a.lat.ny + yy) * a.lat.pitch;
}

// Elements one row of a job's copies moves: the whole row with its padding, or the segment.
__device__ __forceinline__ int copy_len(const TmaGeom &g, const JobPos &j) {
    return g.nseg == 1 ? g.rowstride : j.len;
}

// Bytes of one job's loads (all buffers), for the stage's expect-tx.
template <int D, typename T>
__device__ __forceinline__ uint32_t tma_job_bytes(const lbmh::StepArgs &a, const TmaGeom &g, const JobPos &j) {
    constexpr int Q = qof(D);
    constexpr int U = 16 / (int)sizeof(T);
    uint32_t bytes = (uint32_t)(Q * j.nrows * copy_len(g, j) * (int)sizeof(T));
    if (j.odd && g.nseg > 1) bytes += (uint32_t)((2 * Q / 3) * U * (int)sizeof(T));
    return bytes;
}

// Checked builds: a bulk copy of `bytes` between global `gp` and shared `sp` stays inside
// the population array and the stage, and meets the 16-byte rules of cp.async.bulk.
template <int D, typename T>
__device__ __forceinline__ bool bulk_ok(const lbmh::StepArgs &a, const TmaGeom &g, const T *stage,
                                        const T *sp, const T *gp, uint32_t bytes) {
#ifdef LBM_CHECKED
    constexpr int Q = qof(D);
    const T *A0 = static_cast<const T *>(a.lat.A);
    const int64_t n = (int64_t)bytes / (int64_t)sizeof(T);
    const bool ok = bytes > 0 && (bytes & 15u) == 0 && ((uintptr_t)gp & 15u) == 0 &&
                    (smem_u32(sp) & 15u) == 0 && gp >= A0 && gp + n <= A0 + (int64_t)Q * a.lat.plane &&
                    sp >= stage && sp + n <= stage + (int64_t)Q * g.bufstride;
    return LBM_CHECK(ok, a.status);
#else
    return true;
#endif
}

// What lane b of the loader and the storer knows of buffer b for the whole launch: its velocity and
// the planes it is filled from on even and odd steps.
template <typename T> struct LaneBuf {
    int b, cx, cy, cz;
    T *even, *odd;
};
template <int D, typename T>
__device__ __forceinline__ LaneBuf<T> lane_buf(const lbmh::StepArgs &a, int lane) {
    constexpr int Q = qof(D);
    const int b = lane < Q ? lane : 0;
    T *A = static_cast<T *>(a.lat.A);
    return {b, cxo(b), cyo(b), D == 3 ? czo(b) : 0, A + (int64_t)b * a.lat.plane, A + (int64_t)(Q - 1 - b) * a.lat.plane};
}

// The rows of a job's buffer in global memory: `first` of them from `at`, the others (past the
// periodic edge) from `rest`.
template <typename T> struct JobRows {
    T *at, *rest;
    int first;
};
template <int D, typename T>
__device__ __forceinline__ JobRows<T> job_rows(const lbmh::StepArgs &a, const JobPos &j, const LaneBuf<T> &l) {
    const int ny = a.lat.ny;
    const int z = D == 3 && j.odd ? wrapi(j.z - l.cz, a.lat.nz) : j.z, y = j.odd ? wrapi(j.y0 - l.cy, ny) : j.y0;
    T *plane = (j.odd ? l.odd : l.even) + ((int64_t)z * ny) * a.lat.pitch + j.X0;
    return {plane + (int64_t)y * a.lat.pitch, plane, min(j.nrows, ny - y)};
}

// Loads of a lane's buffer of a job into its stage.
template <int D, typename T>
__device__ __forceinline__ void tma_issue_loads(const lbmh::StepArgs &a, const TmaGeom &g,
                                                const JobPos &j, const LaneBuf<T> &l, T *st, uint64_t *bar) {
    constexpr int U = 16 / (int)sizeof(T);
    const int nx = a.lat.nx, n = copy_len(g, j) * (int)sizeof(T);
    const JobRows<T> rows = job_rows<D, T>(a, j, l);
    T *sbuf = st + l.b * g.bufstride;
    T *dst = sbuf + g.halo;
    if (bulk_ok<D, T>(a, g, st, dst, rows.at, rows.first * n)) bulk_g2s(dst, rows.at, rows.first * n, bar);
    if (rows.first < j.nrows) {
        T *d2 = dst + rows.first * g.rowstride;
        const uint32_t bytes = (j.nrows - rows.first) * n;
        if (bulk_ok<D, T>(a, g, st, d2, rows.rest, bytes)) bulk_g2s(d2, rows.rest, bytes, bar);
    }
    if (j.odd && g.nseg > 1 && l.cx != 0) {  // the halo (one row)
        const int x = l.cx == 1 ? (j.X0 == 0 ? nx - U : j.X0 - U) : (j.X0 + j.len == nx ? 0 : j.X0 + j.len);
        const T *src = rows.at + (x - j.X0);
        T *d2 = l.cx == 1 ? sbuf : dst + j.len;
        if (bulk_ok<D, T>(a, g, st, d2, src, U * sizeof(T))) bulk_g2s(d2, src, U * sizeof(T), bar);
    }
}

// Stores of a lane's buffer of a job back to global memory.
template <int D, typename T>
__device__ __forceinline__ void tma_issue_stores(const lbmh::StepArgs &a, const TmaGeom &g,
                                                 const JobPos &j, const LaneBuf<T> &l, T *st) {
    constexpr int U = 16 / (int)sizeof(T);
    const JobRows<T> rows = job_rows<D, T>(a, j, l);
    const T *src = st + l.b * g.bufstride + g.halo;
    if (!(j.odd && g.nseg > 1)) {
        const int n = copy_len(g, j) * (int)sizeof(T);
        if (bulk_ok<D, T>(a, g, st, src, rows.at, rows.first * n)) bulk_s2g(rows.at, src, rows.first * n);
        if (rows.first < j.nrows) {
            const T *s2 = src + rows.first * g.rowstride;
            const uint32_t bytes = (j.nrows - rows.first) * n;
            if (bulk_ok<D, T>(a, g, st, s2, rows.rest, bytes)) bulk_s2g(rows.rest, s2, bytes);
        }
    } else if (l.cx == 0 || j.len > U) {
        // (one row) without the ragged end the plain stores take
        const int off = l.cx == -1 ? U : 0;
        const uint32_t bytes = (uint32_t)((l.cx == 0 ? j.len : j.len - U) * (int)sizeof(T));
        if (bulk_ok<D, T>(a, g, st, src + off, rows.at + off, bytes)) bulk_s2g(rows.at + off, src + off, bytes);
    }
}

// Plain stores of the ragged ends of segmented odd steps (U cells per buffer with c_x != 0).
template <int D, typename T>
__device__ __forceinline__ void tma_plain_stores(const lbmh::StepArgs &a, const TmaGeom &g,
                                                 const JobPos &j, const T *st, int tid, int nthr) {
    constexpr int Q = qof(D);
    constexpr int U = 16 / (int)sizeof(T);
    constexpr int NB = 2 * Q / 3;
    const int nx = a.lat.nx;
    for (int t = tid; t < NB * U; t += nthr) {
        const int k = t / U, e = t - (t / U) * U;
        const int b = (k >> 1) * 3 + ((k & 1) ? 2 : 0);  // k-th direction with c_x != 0
        T *grow = buffer_row<D, T>(a, j.odd, b, j.z, j.y0);
        const T *srow = st + (int64_t)b * g.bufstride;
        int gx, sx;
        if (cxo(b) == 1) {
            if (e == 0) { gx = j.X0 == 0 ? nx - 1 : j.X0 - 1; sx = g.halo - 1; }
            else { gx = j.X0 + j.len - U + e - 1; sx = g.halo + j.len - U + e - 1; }
        } else {
            if (e == 0) { gx = (j.X0 + j.len == nx) ? 0 : j.X0 + j.len; sx = g.halo + j.len; }
            else { gx = j.X0 + e; sx = g.halo + e; }
        }
        if (LBM_CHECK(gx >= 0 && gx < nx && sx >= 0 && sx < g.bufstride, a.status)) grow[gx] = srow[sx];
    }
}

// Shared-memory positions of one cell's populations (see the header comment): in the
// even step direction i is read at x and written (as direction opp(i)) at x; in the odd
// step it is read at x - c_ix and written at x + c_ix, wrapping inside a whole row.
struct CellPos {
    int row, x, xm, xp;
};

__device__ __forceinline__ CellPos cell_pos(const TmaGeom &g, int r, int xl, int len) {
    CellPos p;
    p.row = r * g.rowstride + g.halo;
    p.x = xl;
    p.xm = xl - 1;
    p.xp = xl + 1;
    if (g.nseg == 1) {
        p.xm = xl == 0 ? len - 1 : p.xm;
        p.xp = xl == len - 1 ? 0 : p.xp;
    }
    return p;
}

template <int D, int P, int CAPB>
__device__ __forceinline__ void tma_load_cell(const typename Storage<P>::T *st, const CellPos &p,
                                              int odd, typename Storage<P>::R (&f)[qof(D)]) {
    using St = Storage<P>;
    constexpr int bs = CAPB / (int)sizeof(typename St::T);  // compile-time offsets between buffers
    const typename St::T *row = st + p.row;
    if (!odd) {
#pragma unroll
        for (int i = 0; i < qof(D); ++i) f[i] = St::load(row[i * bs + p.x]);
    } else {
#pragma unroll
        for (int i = 0; i < qof(D); ++i) {
            const int x = cxo(i) == 1 ? p.xm : (cxo(i) == -1 ? p.xp : p.x);
            f[i] = St::load(row[i * bs + x]);
        }
    }
}

template <int D, int P, int CAPB>
__device__ __forceinline__ void tma_store_cell(typename Storage<P>::T *st, const CellPos &p, int odd,
                                               const typename Storage<P>::R (&f)[qof(D)]) {
    using St = Storage<P>;
    constexpr int Q = qof(D);
    constexpr int bs = CAPB / (int)sizeof(typename St::T);
    typename St::T *row = st + p.row;
    if (!odd) {
#pragma unroll
        for (int i = 0; i < Q; ++i) row[(Q - 1 - i) * bs + p.x] = St::store(f[i]);
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int x = cxo(i) == 1 ? p.xp : (cxo(i) == -1 ? p.xm : p.x);
            row[(Q - 1 - i) * bs + x] = St::store(f[i]);
        }
    }
}

// Collide every cell of a job in place in its stage, one cell per thread per iteration.  DIAG: with
// the diagnostics' sums, which only launches of one step have (as a run-time condition their FP64
// additions took their slots on the FP64 pipe all the same: 512^3 binary16 78.8 -> 80.8 GLUPS, 4096^2
// binary16 203 -> 221 without).
template <int D, int P, int EQ, bool BULK, int CAPB, bool DIAG>
__device__ __forceinline__ void tma_compute(const lbmh::StepArgs &a, const TmaGeom &g,
                                            const JobPos &j, typename Storage<P>::T *st,
                                            DiagAcc &acc, int tid, int nthr) {
    using St = Storage<P>;
    using R = typename St::R;
    constexpr int Q = qof(D);
    const R rho0 = step_scalar<R>(a.rho0, a.rho0f), omega0 = step_scalar<R>(a.omega0, a.omega0f),
            six_nu = step_scalar<R>(a.six_nu, a.six_nuf);
    const int ncells = j.nrows * j.len;
    DiagLocal<R> loc;
    int r = tid < j.len ? 0 : tid / j.len;  // (mostly 0)
    int xl = tid - r * j.len;
    for (int c = tid; c < ncells; c += nthr) {
        const CellPos p = cell_pos(g, r, xl, j.len);
        // checked builds: every position the cell touches lies inside its direction buffer
        if (LBM_CHECK(p.row + min(p.xm, p.x) >= 0 && p.row + max(p.xp, p.x) < g.bufstride, a.status)) {
            R f[Q];
            tma_load_cell<D, P, CAPB>(st, p, j.odd, f);
            const CellMoments<R> m = collide<D, P, EQ, BULK, R>(f, rho0, omega0, six_nu);
            tma_store_cell<D, P, CAPB>(st, p, j.odd, f);
            if (DIAG && a.diag) loc.add(m.rho, m.u, rho0);
        }
        xl += nthr;
        while (xl >= j.len) {
            xl -= j.len;
            ++r;
        }
    }
    if (DIAG && a.diag) loc.flush(acc, a.rho0);
}

// FP32 and binary16 storage: two neighbouring cells per thread per iteration, one in each
// half of the packed FP32 collision (collide32 over f32x2).  Every buffer position pair the
// two cells own at an even offset moves as one shared-memory access (and for binary16 one
// paired conversion).  Even step: cells (x, x + 1), x even, own the pair at x in every buffer.
// Odd step, whole rows: cells (x, x + 1), x odd (the last pair is (len - 1, 0)), own the pairs
// at x - 1 and x + 1 in the buffers with c_x != 0; the c_x = 0 buffers go one half at a time.
// Odd step, segments (no wrap inside the job): cells (x, x + 1), x even, own the pair at x in
// the c_x = 0 buffers and go one half at a time elsewhere.  The operations and conversions
// round exactly as the one-cell path does, so the stored state is the same bit for bit.  Rows
// of odd length (padded rows) have a body of their own, LONE below.
__device__ __forceinline__ f32x2 ld_pair(const __half *b, int p) {
    const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(b + p));
    return pack2(v.x, v.y);
}
__device__ __forceinline__ f32x2 ld_pair(const float *b, int p) {
    const float2 v = *reinterpret_cast<const float2 *>(b + p);
    return pack2(v.x, v.y);
}
__device__ __forceinline__ void st_pair(__half *b, int p, f32x2 v) {
    float lo, hi;
    unpack2(v, lo, hi);
    *reinterpret_cast<__half2 *>(b + p) = __floats2half2_rn(lo, hi);
}
__device__ __forceinline__ void st_pair(float *b, int p, f32x2 v) {
    float lo, hi;
    unpack2(v, lo, hi);
    *reinterpret_cast<float2 *>(b + p) = make_float2(lo, hi);
}

// MODE 0: even step; 1: odd step, whole rows; 2: odd step, segments; -1: chosen at run
// time from the step parity and the job layout (one loop body for all three).
// LONE: rows of odd length, in pairs as well (cell by cell before: 2047 x 2000 FP32 77 -> 102 GLUPS,
// binary16 161 -> 206; 301 x 200 x 200 binary16 56 -> 61; FP32 in 3-D is bound elsewhere).  Another copy
// of the body: with both in one, 512^3 binary16 72 against 79 GLUPS.
// DIAG: as in tma_compute.
template <int D, int P, int EQ, bool BULK, int CAPB, int MODE, bool LONE, bool DIAG>
__device__ __forceinline__ void tma_compute_pairs(const lbmh::StepArgs &a, const TmaGeom &g,
                                                  const JobPos &j, typename Storage<P>::T *st, DiagAcc &acc,
                                                  int tid, int nthr) {
    using St = Storage<P>;
    using T = typename St::T;
    constexpr int Q = qof(D);
    constexpr int bs = CAPB / (int)sizeof(T);  // elements between direction buffers
    const int mode = MODE >= 0 ? MODE : (!j.odd ? 0 : (LONE || g.nseg == 1 ? 1 : 2));
    // Rows of odd length are padded whole rows: their last pair of the even step is a cell and an element
    // of the padding; in the odd step the first pair is cell 0 twice, and the others follow.
    constexpr int lone = LONE ? 1 : 0;
    const int hl = (j.len + lone) >> 1;
    const int npairs = j.nrows * hl;
    DiagLocal<float> loc;
    int r = tid < hl ? 0 : tid / hl;  // (mostly 0)
    int xh = tid - r * hl;
    for (int c = tid; c < npairs; c += nthr) {
        T *row = st + r * g.rowstride + g.halo;
        // cells xa and xb = xa + 1 (the odd pairing of whole rows wraps its last pair to
        // cell 0); pm = xa - 1 and pp = xb + 1 are the outer neighbours, inside the row for
        // whole rows (xa >= 1 in the odd pairing) and in the halos for segments
        const bool twice = LONE && mode == 1 && xh == 0;
        const int xa = twice ? 0 : 2 * xh + (mode == 1 ? 1 - 2 * lone : 0);
        const int xb = twice || (mode == 1 && xa + 1 == j.len) ? 0 : xa + 1;
        // its neighbours are not at consecutive positions
        const bool apart = LONE && mode == 1 && (twice || xb + 1 == j.len);
        const int pm = xa - 1;
        const int pp = xb + 1;
        // checked builds: every position the pair touches lies inside its direction buffer
        const int row_off = r * g.rowstride + g.halo;
        const int lo = mode == 0 ? xa : twice ? 0 : min(min(pm, xa), xb);
        const int hi = mode == 0 ? xa + 1 : twice ? j.len - 1 : max(max(xb + 1, pp), xa);
        if (LBM_CHECK(row_off + lo >= 0 && row_off + hi < bs, a.status)) {
            f32x2 f[Q];
            if (mode == 0) {
    #pragma unroll
                for (int i = 0; i < Q; ++i) f[i] = ld_pair(row + i * bs, xa);
            } else if (apart) {
                const int ma = twice ? j.len - 1 : pm, mb = twice ? ma : xa, qa = twice ? 1 : xb, qb = twice ? 1 : 0;
    #pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const T *b = row + i * bs;
                    f[i] = cxo(i) == 0 ? pack2(St::load(b[xa]), St::load(b[xb]))
                                       : cxo(i) == 1 ? pack2(St::load(b[ma]), St::load(b[mb])) : pack2(St::load(b[qa]), St::load(b[qb]));
                }
            } else if (mode == 1) {
    #pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const T *b = row + i * bs;
                    if (cxo(i) == 0) f[i] = pack2(St::load(b[xa]), St::load(b[xb]));
                    else f[i] = ld_pair(b, cxo(i) == 1 ? pm : xb);
                }
            } else {
    #pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const T *b = row + i * bs;
                    if (cxo(i) == 0) f[i] = ld_pair(b, xa);
                    else if (cxo(i) == 1) f[i] = pack2(St::load(b[pm]), St::load(b[xa]));
                    else f[i] = pack2(St::load(b[xb]), St::load(b[pp]));
                }
            }
            const Moments32<f32x2> m = collide32<D, P, EQ, BULK, f32x2>(f, a.rho0f, a.omega0f, a.six_nuf);
            if (mode == 0) {
    #pragma unroll
                for (int i = 0; i < Q; ++i) st_pair(row + (Q - 1 - i) * bs, xa, f[i]);
            } else {
    #pragma unroll
                for (int i = 0; i < Q; ++i) {
                    T *b = row + (Q - 1 - i) * bs;
                    float va, vb;
                    unpack2(f[i], va, vb);
                    if (mode == 1) {
                        if (cxo(i) == 0) {
                            b[xa] = St::store(va);
                            b[xb] = St::store(vb);
                        } else if (apart) {
                            b[cxo(i) == 1 ? (twice ? 1 : xb) : (twice ? j.len - 1 : pm)] = St::store(va);
                            b[cxo(i) == 1 ? (twice ? 1 : 0) : (twice ? j.len - 1 : xa)] = St::store(vb);
                        } else {
                            st_pair(b, cxo(i) == 1 ? xb : pm, f[i]);
                        }
                    } else {
                        if (cxo(i) == 0) {
                            st_pair(b, xa, f[i]);
                        } else if (cxo(i) == 1) {
                            b[xb] = St::store(va);
                            b[pp] = St::store(vb);
                        } else {
                            b[pm] = St::store(va);
                            b[xa] = St::store(vb);
                        }
                    }
                }
            }
            if (DIAG && a.diag) {
                float ra, rb, ua[3], ub[3];
                unpack2(m.rho, ra, rb);
    #pragma unroll
                for (int q = 0; q < 3; ++q) unpack2(m.u[q], ua[q], ub[q]);
                loc.add(ra, ua, a.rho0f);
                if (!LONE || (!twice && xb < j.len)) loc.add(rb, ub, a.rho0f);
            }
        }
        xh += nthr;
        while (xh >= hl) {
            xh -= hl;
            ++r;
        }
    }
    if (DIAG && a.diag) loc.flush(acc, a.rho0);
}

// A job's collisions, by the bodies that suit the storage.  CHAIN: several steps a launch; DIAG: with
// the diagnostics' sums (single steps only).
template <int D, int P, int EQ, bool BULK, int CAPB, bool CHAIN, bool DIAG>
__device__ __forceinline__ void tma_collide(const lbmh::StepArgs &a, const TmaGeom &g, const JobPos &jp,
                                            typename Storage<P>::T *st, DiagAcc &acc, int tid, int nthr) {
    const auto pairs = [&](auto mode, auto lone) {
        tma_compute_pairs<D, P, EQ, BULK, CAPB, mode.value, lone.value, DIAG>(a, g, jp, st, acc, tid, nthr);
    };
    using std::integral_constant;
    constexpr std::true_type yes;
    constexpr std::false_type no;
    constexpr integral_constant<int, -1> any;
    // One D3Q27 step a launch is bound by HBM (0.97 of the copy peak), and two cells a thread only bunch
    // its accesses: 512^3 binary16 2.19 against 2.33 ms a step (128^3, in L2, 47 against 42.5 us).  With
    // diagnostics the longer body is what counts: two cells a thread 2.38 against 2.42 ms, 256^3 317
    // against 343 us.  2-D FP32 rows of odd length: 54 us in pairs, 59 cell by cell (2047 x 2000).
    if constexpr (P == P_F64 || (D == 3 && !CHAIN && !(DIAG && P == P_F16S))) {
        tma_compute<D, P, EQ, BULK, CAPB, DIAG>(a, g, jp, st, acc, tid, nthr);
    } else if constexpr (D == 3 || DIAG) {
        // The D3Q27 pair body is long: one copy serves the three pairings (three
        // specialised copies measured slower).
        if (jp.len & 1) pairs(any, yes);
        else pairs(any, no);
    } else {
        constexpr integral_constant<int, 0> even;
        constexpr integral_constant<int, 1> rows;
        constexpr integral_constant<int, 2> segments;
        if (jp.len & 1) {
            if (jp.odd) pairs(rows, yes);
            else pairs(even, yes);
        } else if (!jp.odd) pairs(even, no);
        else if (g.nseg == 1) pairs(rows, no);
        else pairs(segments, no);
    }
}

// One step a launch: jobs strided over the blocks.  One service warp: lane b stores the buffer b of a
// collided stage, waits until that store has read it, and refills the same buffer with the next job's;
// the lanes do not wait for one another.
template <int D, int P, int EQ, bool BULK, int CAPB>
__global__ void __launch_bounds__(tma_max_threads(D, P) + 32) k_step_tma(const lbmh::StepArgs a, const TmaGeom g) {
    using T = typename Storage<P>::T;
    constexpr int Q = qof(D);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[kTmaMaxStages];
    __shared__ __align__(8) uint64_t empty[kTmaMaxStages];
    T *sm = reinterpret_cast<T *>(smem_raw);
    const int64_t stage_elems = (int64_t)Q * (CAPB / (int)sizeof(T));
    const int S = g.stages;
    const int ncons = (int)blockDim.x - 32;
    const int lane = threadIdx.x & 31;
    const unsigned total = (unsigned)g.njobs, G = gridDim.x;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], ncons / 32);
        }
        fence_barrier_init();
    }
    __syncthreads();
    DiagAcc acc;
    bool failed = false;
    if ((int)threadIdx.x >= ncons) {
        const LaneBuf<T> buf = lane_buf<D, T>(a, lane);
        // stage s, and the parity of the phase in which its job before was collided; `held` jobs are in
        // the stages, the oldest of them `old`
        int s = 0, held = 0;
        uint32_t phase = 1;
        unsigned old = blockIdx.x, job = blockIdx.x;
        for (; job < total; job += G) {
            const JobPos jp = decode_job(a, g, job);
            T *st = sm + s * stage_elems;
            if (held == S) {
                const bool ok = mbar_wait_bounded(&empty[s], phase, a.timeout_ns);
                if (__any_sync(0xffffffffu, !ok)) {
                    failed = true;
                    break;
                }
                const JobPos jq = decode_job(a, g, old);
                old += G;
                if (a.odd && g.nseg > 1) {
                    tma_plain_stores<D, T>(a, g, jq, st, lane, 32);
                    __syncwarp();  // every lane's plain stores read the stage before any refill
                }
                if (lane == 0) mbar_arrive_expect_tx(&full[s], tma_job_bytes<D, T>(a, g, jp));
                if (lane < Q) {
                    tma_issue_stores<D, T>(a, g, jq, buf, st);
                    bulk_commit();
                    bulk_wait_read<0>();
                    tma_issue_loads<D, T>(a, g, jp, buf, st, &full[s]);
                }
            } else {
                ++held;
                if (lane == 0) mbar_arrive_expect_tx(&full[s], tma_job_bytes<D, T>(a, g, jp));
                if (lane < Q) tma_issue_loads<D, T>(a, g, jp, buf, st, &full[s]);
            }
            if (++s == S) {
                s = 0;
                phase ^= 1u;
            }
        }
        // store back the jobs that are left, the oldest first
        if (held < S) {
            s = 0;
            phase = 0;
        }
        for (; held > 0 && !failed; --held) {
            const bool ok = mbar_wait_bounded(&empty[s], phase, a.timeout_ns);
            if (__any_sync(0xffffffffu, !ok)) {
                failed = true;
                break;
            }
            const JobPos jq = decode_job(a, g, old);
            old += G;
            T *st = sm + s * stage_elems;
            if (a.odd && g.nseg > 1) tma_plain_stores<D, T>(a, g, jq, st, lane, 32);
            if (lane < Q) {
                tma_issue_stores<D, T>(a, g, jq, buf, st);
                bulk_commit();
            }
            if (++s == S) {
                s = 0;
                phase ^= 1u;
            }
        }
        bulk_wait_all();
        if (failed) {
            // let loads still in flight land before the block's shared memory is released: of the stages
            // that hold jobs, s has the one that was not collided in time, the others have later ones
            for (; held > 0; --held) {
                (void)mbar_wait_bounded(&full[s], phase, a.timeout_ns);
                if (++s == S) {
                    s = 0;
                    phase ^= 1u;
                }
            }
        }
    } else {
        int s = 0;
        uint32_t phase = 0;
        for (unsigned job = blockIdx.x; job < total; job += G) {
            const bool ok = mbar_wait_bounded(&full[s], phase, a.timeout_ns);
            if (__any_sync(0xffffffffu, !ok)) {
                failed = true;
                break;
            }
            T *st = sm + s * stage_elems;
            const JobPos jp = decode_job(a, g, job);
            if (a.diag) tma_collide<D, P, EQ, BULK, CAPB, false, true>(a, g, jp, st, acc, threadIdx.x, ncons);
            else tma_collide<D, P, EQ, BULK, CAPB, false, false>(a, g, jp, st, acc, threadIdx.x, ncons);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive_cta(&empty[s]);
            if (++s == S) {
                s = 0;
                phase ^= 1u;
            }
        }
    }
    if (failed && lane == 0) report_status(a.status, -5); /* LBM_ETIMEOUT */
    if (a.diag) diag_block_store(acc, a.partials + (int64_t)blockIdx.x * lbmh::kDiagWords);
}

// Several steps a launch (see decode_chain).  The warps after the consumers are the loader and the storer.
// One block an SM as the least lets the compiler have registers (74 - 78 in 2-D, 140 - 164 in 3-D, two
// blocks of 192 threads still fit; left alone it kept to 56 - 72 and 128): binary16 4096^2 75.7 -> 73.3 us
// a step, 512^3 1.64 -> 1.62 ms, rows of odd length 5 - 15 % (2237 x 2466 44 -> 38 us).
constexpr int kTmaServiceThreads = 64;

template <int D, int P, int EQ, bool BULK, int CAPB>
__global__ void __launch_bounds__(tma_max_threads(D, P) + kTmaServiceThreads, 1) k_steps_tma(const lbmh::StepArgs a, const TmaGeom g) {
    using T = typename Storage<P>::T;
    constexpr int Q = qof(D);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[kTmaMaxStages];
    __shared__ __align__(8) uint64_t empty[kTmaMaxStages];
    __shared__ __align__(8) uint64_t freed[kTmaMaxStages];
    __shared__ JobPos jobq[kTmaMaxStages];  // the job in each stage; nrows == 0 ends the block's work
    __shared__ int unitq[kTmaMaxStages];    // its unit
    T *sm = reinterpret_cast<T *>(smem_raw);
    const int64_t stage_elems = (int64_t)Q * (CAPB / (int)sizeof(T));
    const int S = g.stages;
    const int ncons = (int)blockDim.x - kTmaServiceThreads;
    const int lane = threadIdx.x & 31;
    const int role = (int)threadIdx.x < ncons ? 0 : ((int)threadIdx.x < ncons + 32 ? 1 : 2);
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], ncons / 32);
            mbar_init(&freed[s], 1);
        }
        fence_barrier_init();
    }
    __syncthreads();
    DiagAcc acc;  // (no diagnostics here)
    bool failed = false;
    if (role == 1) {
        // loader: takes the jobs, waits for the steps they need, refills the stages.  Its work for a
        // job, like the storer's, is one serial chain, and a block gets no more jobs than they can
        // handle: measured in clocks a job (4096^2 FP32, 6400 in all), decoding 1950 (eleven divisions,
        // hence FastDiv), the counters and the full proxy fence 2200, issuing the copies 1750, and in
        // the storer issue 1300, wait 1900, another proxy fence and the release 2100.  Without the
        // divisions, with the fence on global memory only and none in the storer: 5600.  Several steps
        // a launch: 4096^2 FP32 118 -> 142 GLUPS, 4096^2 binary16 184 -> 205, 256^3 FP32 41.4 -> 46.0,
        // 512^3 binary16 73 -> 78.  (Two tickets at a time, decoded by half a warp each: 4 - 8 % slower.)
        const LaneBuf<T> buf = lane_buf<D, T>(a, lane);
        const unsigned total = (unsigned)chain_tickets(g);
        unsigned next = 0;
        if (lane == 0) next = atomicAdd(&a.sync[0], 1u);
        int s = 0;
        uint32_t phase = 0;
        bool wrapped = false;
        for (;;) {
            JobPos jp{0, 0, 0, 0, 0, 0};
            const unsigned job = __shfl_sync(0xffffffffu, next, 0);
            bool end = job >= total;
            int step = 0, up = 0, uc = 0;
            if (!end) {
                const ChainJob c = decode_chain(a, g, job);
                if (lane == 0) next = atomicAdd(&a.sync[0], 1u);  // in flight while this job is set up
                if (c.step < 0) continue;
                jp = c.j;
                step = c.step;
                up = c.p;
                uc = c.c;
            }
            if (wrapped) {  // the stage's last job has been stored
                const bool ok = mbar_wait_bounded(&freed[s], phase ^ 1u, a.timeout_ns);
                if (__any_sync(0xffffffffu, !ok)) {
                    failed = true;
                    break;
                }
            }
            if (!end && step > 0) {
                bool ok = true;
                if (lane < (D == 3 ? 9 : 3)) {
                    const int p = wrapi(up + lane % 3 - 1, g.npos);
                    const int c = D == 3 ? wrapi(uc + lane / 3 - 1, g.ncross) : 0;
                    ok = wait_count_bounded(&a.sync[lbmh::kSyncDone + p * g.ncross + c], (unsigned)(step * g.nseg),
                                            a.status, a.timeout_ns);
                }
                if (__any_sync(0xffffffffu, !ok)) {
                    failed = true;
                    end = true;
                }
                // what other SMs' copy engines and threads wrote, before this SM's copy engine reads
                fence_proxy_async_global();
            }
            if (lane == 0) {
                if (end) jp.nrows = 0;
                jobq[s] = jp;
                unitq[s] = up * g.ncross + uc;
                mbar_arrive_expect_tx(&full[s], end ? 0u : tma_job_bytes<D, T>(a, g, jp));
            }
            if (end) break;
            if (lane < Q) tma_issue_loads<D, T>(a, g, jp, buf, sm + s * stage_elems, &full[s]);
            if (++s == S) {
                s = 0;
                phase ^= 1u;
                wrapped = true;
            }
        }
    } else if (role == 2) {
        // storer: writes collided stages back, frees them, and reports finished jobs
        const LaneBuf<T> buf = lane_buf<D, T>(a, lane);
        int s = 0;
        uint32_t phase = 0;
        for (;;) {
            const bool ok = mbar_wait_bounded(&empty[s], phase, a.timeout_ns);
            if (__any_sync(0xffffffffu, !ok)) {
                failed = true;
                break;
            }
            const JobPos jq = jobq[s];
            const int unit = unitq[s];
            if (jq.nrows == 0) break;
            T *st = sm + s * stage_elems;
            if (jq.odd && g.nseg > 1) tma_plain_stores<D, T>(a, g, jq, st, lane, 32);
            if (lane < Q) tma_issue_stores<D, T>(a, g, jq, buf, st);
            bulk_commit();
            bulk_wait_read<0>();
            __syncwarp();
            if (lane == 0) mbar_arrive_cta(&freed[s]);
            // (a completed group's writes are visible to its thread; another proxy fence here
            // held the storer for some 800 clocks a job)
            bulk_wait_all();
            __syncwarp();
            if (lane == 0) red_release(&a.sync[lbmh::kSyncDone + unit], 1u);
            if (++s == S) {
                s = 0;
                phase ^= 1u;
            }
        }
        bulk_wait_all();
        if (failed) {
            // let loads still in flight land before the block's shared memory is released
            for (int q = 0; q < S; ++q) (void)mbar_wait_bounded(&full[(s + q) % S], s + q >= S ? phase ^ 1u : phase, a.timeout_ns);
        }
    } else {
        int s = 0;
        uint32_t phase = 0;
        for (;;) {
            const bool ok = mbar_wait_bounded(&full[s], phase, a.timeout_ns);
            if (__any_sync(0xffffffffu, !ok)) {
                failed = true;
                break;
            }
            const JobPos jp = jobq[s];
            if (jp.nrows > 0) {
                T *st = sm + s * stage_elems;
                tma_collide<D, P, EQ, BULK, CAPB, true, false>(a, g, jp, st, acc, threadIdx.x, ncons);
                fence_proxy_async_smem();
                __syncwarp();
            }
            if (lane == 0) mbar_arrive_cta(&empty[s]);
            if (jp.nrows == 0) break;
            if (++s == S) {
                s = 0;
                phase ^= 1u;
            }
        }
    }
    if (failed && lane == 0) report_status(a.status, -5); /* LBM_ETIMEOUT */
    // the last block to finish clears the counters for the next launch
    __syncthreads();
    bool last = false;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&a.sync[1], 1u) == gridDim.x - 1;
    }
    if (__syncthreads_or(last)) {
        uint4 *w = reinterpret_cast<uint4 *>(a.sync);
        for (int p = threadIdx.x; p < (lbmh::kSyncDone + g.npos * g.ncross + 3) / 4; p += blockDim.x)
            w[p] = make_uint4(0, 0, 0, 0);
    }
}

template <int D, int P, int CAPB>
const void *tma_kernel_dpc(int eq, int bulk, bool several) {
#define LBM_TMA(EQv, Bv)                                                                                       \
    if (eq == EQv && (bulk != 0) == Bv)                                                                        \
        return several ? (const void *)k_steps_tma<D, P, EQv, Bv, CAPB> : (const void *)k_step_tma<D, P, EQv, Bv, CAPB>;
    LBM_TMA(EQ_ENT, false)
    LBM_TMA(EQ_ENT, true)
    LBM_TMA(EQ_POLY2, false)
    LBM_TMA(EQ_POLY2, true)
    LBM_TMA(EQ_PROD, false)
    LBM_TMA(EQ_PROD, true)
#undef LBM_TMA
    return nullptr;
}

template <int D, int CAPB>
const void *tma_kernel_dc(int P, int eq, int bulk, bool several) {
    switch (P) {
    case P_F64: return tma_kernel_dpc<D, P_F64, CAPB>(eq, bulk, several);
    case P_F32: return tma_kernel_dpc<D, P_F32, CAPB>(eq, bulk, several);
    case P_F16S: return tma_kernel_dpc<D, P_F16S, CAPB>(eq, bulk, several);
    default: return nullptr;
    }
}

}  // namespace lbmd
