// k_batch.cu -- many independent periodic lattices (the linear-mode sweep of Sec. V)
// advanced for n steps by one persistent launch.
//
// Every instance is owned by exactly one block (a greedy longest-first assignment on the
// host balances the cell counts), so the only synchronisation between steps is the
// block's own barrier: no block ever waits for another.  Each step of an instance is the
// AA-pattern update of the generic kernel in FP64 (the state of the linear sweep is FP64;
// on GB300 this path is bound by the FP64 pipe, not by memory).  On steps t with
// t % every_k == 0 the block also projects rho and j = rho u of the state at t on
// exp(-i k.r) (twiddle tables per axis), reduces them in a fixed order and records one
// sample per instance; a non-finite mass marks the instance's status with t + 1.
//
// A batch whose largest instance alone would keep one SM busy longer than its share (few
// instances, or uneven ones) is advanced by teams of blocks instead, see k_step_teams, and one of a
// few short instances by clusters, see k_step_clusters.
#include <algorithm>

#include "k_generic_step.cuh"

namespace lbmd {

// Probe sums: re, im of rho, j_x, j_y and in 3-D j_z.
template <int D> constexpr int kProbe = 2 * (D + 1);

// Adds exp(-i k.r) (rho, rho u) of cell (x, y, z) to the sums; tw: the instance's twiddles per axis.
template <int D>
__device__ __forceinline__ void probe_add(double (&acc)[kProbe<D>], const CellMoments<double> &m, const double2 *tw,
                                          int nx, int ny, int x, int y, int z) {
    const double2 tx = tw[x], ty = tw[nx + y];  // exp(-i k.r) = tw_x[x] tw_y[y] tw_z[z]
    double pr = tx.x * ty.x - tx.y * ty.y;
    double pi = tx.x * ty.y + tx.y * ty.x;
    if (D == 3) {
        const double2 tz = tw[nx + ny + z];
        const double qr = pr * tz.x - pi * tz.y;
        pi = pr * tz.y + pi * tz.x;
        pr = qr;
    }
    const double q[4] = {m.rho, m.rho * m.u[0], m.rho * m.u[1], m.rho * m.u[2]};
#pragma unroll
    for (int j = 0; j <= D; ++j) {
        acc[2 * j] += q[j] * pr;
        acc[2 * j + 1] += q[j] * pi;
    }
}

// Sums over a warp: lane l < 8 returns the sum of acc[l].  Each exchange halves the sums a lane
// still carries, 9 additions a lane in place of 40 for eight full butterflies (an FP64 addition of
// a warp takes an SM quarter 64 clocks).
template <int N>
__device__ __forceinline__ double warp_sums(const double (&acc)[N]) {
    const int lane = threadIdx.x & 31;
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = j < N ? acc[j < N ? j : 0] : 0.0;
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1) {  // lanes with bit h keep the upper h sums
        const bool up = lane & h;
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const double keep = up ? v[j + h] : v[j], give = up ? v[j] : v[j + h];
            v[j] = j < N ? keep + __shfl_xor_sync(0xffffffffu, give, h) : 0.0;
        }
    }
    double r = v[0];
    r += __shfl_xor_sync(0xffffffffu, r, 8);
    r += __shfl_xor_sync(0xffffffffu, r, 16);
    return r;
}

// Records a sample of instance k from its sums (one thread).
template <int N>
__device__ __forceinline__ void probe_record(const lbmh::BatchArgs &a, int k, int64_t t, const double (&sum)[N]) {
    const int64_t sample = t / a.every_k;
    bool fin = true;
    for (int j = 0; j < N; ++j) fin = fin && isfinite(sum[j]);
    if (sample < a.max_samples) {
        double *out = a.series + ((int64_t)k * a.max_samples + sample) * 8;
        // (j_z = rho u_z of a 2-D lattice: 0, or NaN beside a density that is not finite)
        for (int j = 0; j < 8; ++j) out[j] = j < N ? sum[j < N ? j : 0] : (fin ? 0.0 : sum[0] - sum[0]);
    }
    if (!fin && a.status[k] == 0) a.status[k] = (int32_t)(t + 1);
}

// One step of the cells first, first + stride, ... of an instance; PROBE: with their probe sums.  (Two
// copies: one loop with the probe behind a branch formed velocities on every step, 5.94 against
// 5.20 ms a step on the 4096-lattice sweep.)
template <int D, int EQ, bool BULK, bool L2, bool PROBE>
__device__ __forceinline__ void batch_cells(double *A, int64_t ncell, int nx, int ny, int nz, int64_t first, int64_t stride,
                                            int odd, double rho0, double om, double sn, const double2 *tw,
                                            double (&acc)[kProbe<D>], int32_t *status) {
    for (int64_t c = first; c < ncell; c += stride) {
        int x, y, z;
        cell_coords(c, ncell, nx, ny, x, y, z);
        const CellMoments<double> m = aa_cell_step<D, P_F64, EQ, BULK, L2>(A, ncell, nx, ny, nz, nx, x, y, z, odd, rho0, om, sn, status);
        if constexpr (PROBE) probe_add<D>(acc, m, tw, nx, ny, x, y, z);
    }
}

template <int D, int EQ, bool BULK>
__global__ void __launch_bounds__(256) k_step_batch(const lbmh::BatchArgs a) {
    constexpr int N = kProbe<D>, Q = qof(D);
    __shared__ double red[8][8];
    const int b0 = a.block_start[blockIdx.x], b1 = a.block_start[blockIdx.x + 1];
    for (int64_t s = 0; s < a.nsteps; ++s) {
        const int64_t t = a.step0 + s;
        const int odd = (int)(t & 1);
        const bool probe = a.every_k > 0 && (t % a.every_k) == 0;
        for (int ii = b0; ii < b1; ++ii) {
            const int k = a.order[ii];
            const int nx = a.dims[3 * k], ny = a.dims[3 * k + 1], nz = a.dims[3 * k + 2];
            const int64_t c0 = a.cell_start[k];
            const int64_t ncell = a.cell_start[k + 1] - c0;
            double *A = a.arena + (int64_t)Q * c0;
            const double om = a.omega0[k], sn = a.six_nu[k];
            const double2 *tw = a.twiddle + a.tw_offset[k];
            double acc[N] = {};
            if (probe) batch_cells<D, EQ, BULK, false, true>(A, ncell, nx, ny, nz, threadIdx.x, blockDim.x, odd, a.rho0, om, sn, tw, acc, a.status + k);
            else batch_cells<D, EQ, BULK, false, false>(A, ncell, nx, ny, nz, threadIdx.x, blockDim.x, odd, a.rho0, om, sn, tw, acc, a.status + k);
            if (probe) {
                // fixed-order block reduction: within the warps, then the warps in order
                const double v = warp_sums(acc);
                const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
                if (lane < 8) red[warp][lane] = v;
                __syncthreads();
                if (threadIdx.x == 0) {
                    double sum[N] = {};
                    const int nw = (blockDim.x + 31) >> 5;
                    for (int w = 0; w < nw; ++w)
                        for (int j = 0; j < N; ++j) sum[j] += red[w][j];
                    probe_record(a, k, t, sum);
                }
                __syncthreads();
            }
        }
        __syncthreads();  // step boundary: the block's instances are complete at t + 1
    }
}

// Teams: every block works on one instance, and an instance has as many blocks as its share of the
// cells asks for (at least one).  A step ends with a barrier of the instance's blocks (a counter
// per instance; the launch is cooperative, so they are all resident); a team of one needs none
// beyond the block's own.  A probe's partial sums go through a buffer per block, in pairs so that
// the next probe does not overwrite sums the team's first block is still adding up.
template <int D, int EQ, bool BULK>
__global__ void __launch_bounds__(lbmh::kTeamThreads, D == 2 ? 5 : 3) k_step_teams(const lbmh::BatchArgs a) {
    constexpr int N = kProbe<D>, Q = qof(D);
    constexpr int kWarps = lbmh::kTeamThreads / 32;
    __shared__ double red[kWarps][8];
    const int k = a.team_instance[blockIdx.x], part = a.team_part[blockIdx.x], parts = a.team_size[k];
    const int nx = a.dims[3 * k], ny = a.dims[3 * k + 1], nz = a.dims[3 * k + 2];
    const int64_t c0 = a.cell_start[k];
    const int ncell = (int)(a.cell_start[k + 1] - c0);  // Q * ncell < 2^31 (checked on the host)
    double *A = a.arena + (int64_t)Q * c0;
    const double om = a.omega0[k], sn = a.six_nu[k];
    const double2 *tw = a.twiddle + a.tw_offset[k];
    unsigned *counter = a.team_sync + lbmh::kBarStride * (1 + k);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int first = part * (int)blockDim.x + (int)threadIdx.x, stride = parts * (int)blockDim.x;
    unsigned probes = 0;
    bool ok = true;
    for (int64_t s = 0; s < a.nsteps && ok; ++s) {
        const int64_t t = a.step0 + s;
        const int odd = (int)(t & 1);
        const bool probe = a.every_k > 0 && (t % a.every_k) == 0;
        double acc[N] = {};
        if (probe) batch_cells<D, EQ, BULK, true, true>(A, ncell, nx, ny, nz, first, stride, odd, a.rho0, om, sn, tw, acc, a.status + k);
        else batch_cells<D, EQ, BULK, true, false>(A, ncell, nx, ny, nz, first, stride, odd, a.rho0, om, sn, tw, acc, a.status + k);
        double *buf = a.team_partials + ((int64_t)(probes & 1) * gridDim.x + blockIdx.x) * 8;
        if (probe) {
            const double v = warp_sums(acc);
            if (lane < 8) red[warp][lane] = v;
            __syncthreads();
            if (threadIdx.x < N) {
                double sum = 0.0;
                for (int w = 0; w < kWarps; ++w) sum += red[w][threadIdx.x];
                buf[threadIdx.x] = sum;
            }
        }
        if (parts > 1) ok = team_barrier(counter, (unsigned)(s + 1) * (unsigned)parts, a.team_status, a.timeout_ns);
        else __syncthreads();
        if (probe) {
            if (part == 0 && threadIdx.x == 0 && ok) {
                double sum[N] = {};
                for (int q = 0; q < parts; ++q)
                    for (int j = 0; j < N; ++j) sum[j] += __ldcg(buf + 8 * q + j);
                probe_record(a, k, t, sum);
            }
            ++probes;
        }
    }
    if (!ok && threadIdx.x == 0) report_status(a.team_status, -5); /* LBM_ETIMEOUT */
    // the last block to finish clears the counters for the next launch
    __syncthreads();
    bool last = false;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&a.team_sync[0], 1u) == gridDim.x - 1;
    }
    if (__syncthreads_or(last))
        for (int64_t p = threadIdx.x; p <= a.count; p += blockDim.x) a.team_sync[lbmh::kBarStride * p] = 0;
}

// Sums over the ten groups of three lanes of a warp: lanes 0 to 2 return the sums of the values of
// the lanes with their c.  (Four additions; lanes 30 and 31 hold zero.)
__device__ __forceinline__ double group_sums(double v) {
    v += __shfl_down_sync(0xffffffffu, v, 15);            // groups 0 .. 4
    const double v4 = __shfl_down_sync(0xffffffffu, v, 12);
    v += __shfl_down_sync(0xffffffffu, v, 6);             // 0 + 2, 1 + 3
    v += __shfl_down_sync(0xffffffffu, v, 3);
    return v + v4;
}

// Clusters: an instance of at most eight blocks of kClusterCells cells is a thread-block cluster
// that keeps the populations in its blocks' shared memory for the whole launch.  A cell is on three
// lanes (collide_lanes), a warp of ten cells to each SM quarter; neighbours in another block are read
// and written through distributed shared memory, and a step ends with the cluster's hardware barrier.
// A location is read and then written by the lanes of one cell within a step, and every store of a
// warp depends on all its loads (the collision's shuffles), so one barrier a step is enough.
// Short lattices are bound by the FP64 chain and the step's synchronisation: 28 lines of 128 cells
// (entropic, bulk correction) probed every 10 steps, a block each 4.6 us a step, teams of 4 blocks
// with three-lane cells through L2 4.9, clusters 3.0; probed on every step 6.4 -> 3.8.  A probe's
// projections are split over a cell's lanes as well (all on one lane: 4.8 us).
template <int D, int EQ, bool BULK>
__global__ void __launch_bounds__(lbmh::kTeamThreads) k_step_clusters(const lbmh::BatchArgs a) {
    constexpr int N = kProbe<D>, Q = qof(D), F = lane_pops(D), C = lbmh::kClusterCells;
    constexpr int kWarps = lbmh::kTeamThreads / 32;
    __shared__ double pop[Q * C];  // plane i of the block's cells at i C
    __shared__ double red[kWarps][8], sums[2][8];
    const int csize = a.team_cluster, k = blockIdx.x / csize, part = blockIdx.x % csize;
    const int nx = a.dims[3 * k], ny = a.dims[3 * k + 1], nz = a.dims[3 * k + 2];
    const int64_t c0 = a.cell_start[k];
    const int ncell = (int)(a.cell_start[k + 1] - c0), parts = (ncell + C - 1) / C;
    double *A = a.arena + (int64_t)Q * c0 + part * C;
    const int mine = min(C, ncell - part * C);  // cells of the block (none: it only takes part in the barriers)
    const double om = a.omega0[k], sn = a.six_nu[k];
    const double2 *tw = a.twiddle + a.tw_offset[k];
    for (int p = threadIdx.x; p < Q * C; p += lbmh::kTeamThreads)
        if (p % C < mine) pop[p] = A[(int64_t)(p / C) * ncell + p % C];
    // the lane's cell and the addresses of its odd-step reads f_i(r) = A[opp(i)][r - c_i] and writes
    // A[i][r + c_i], directions i = p + F c
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane % 3, base = lane < 30 ? lane - c : 27;
    const int here = warp * 10 + lane / 3;
    const bool run = lane < 30 && here < mine;
    int x, y, z;
    cell_coords(run ? part * C + here : 0, ncell, nx, ny, x, y, z);
    uint32_t src[F], dst[F];
    const uint32_t pop0 = smem_u32(pop);
#pragma unroll
    for (int p = 0; p < F; ++p) {
        const int i = p + F * c, dx = cxo(p), dy = D == 3 ? cyo(p) : c - 1, dz = D == 3 ? c - 1 : 0;
        const int from = wrapi(x - dx, nx) + nx * (wrapi(y - dy, ny) + ny * wrapi(z - dz, nz));
        const int to = wrapi(x + dx, nx) + nx * (wrapi(y + dy, ny) + ny * wrapi(z + dz, nz));
        const bool ok = LBM_CHECK(from >= 0 && from < ncell && to >= 0 && to < ncell, a.status + k);
        src[p] = cluster_addr(pop0 + 8 * ((Q - 1 - i) * C + (ok ? from % C : 0)), ok ? from / C : part);
        dst[p] = cluster_addr(pop0 + 8 * (i * C + (ok ? to % C : 0)), ok ? to / C : part);
    }
    // exp(-i k.r) of the cell; lane c projects rho, j_x or j_y, in 3-D lane 0 also j_z
    double pr = 0.0, pi = 0.0;
    if (a.every_k > 0 && run) {
        const double2 tx = tw[x], ty = tw[nx + y];
        pr = tx.x * ty.x - tx.y * ty.y;
        pi = tx.x * ty.y + tx.y * ty.x;
        if (D == 3) {
            const double2 tz = tw[nx + ny + z];
            const double qr = pr * tz.x - pi * tz.y;
            pi = pr * tz.y + pi * tz.x;
            pr = qr;
        }
    }
    const bool busy = warp * 10 < mine;
    if (lane < 8) red[warp][lane] = 0.0;  // (2-D: no j_z)
    cluster_barrier();
    int64_t until = a.every_k > 0 ? (a.every_k - a.step0 % a.every_k) % a.every_k : a.nsteps;  // steps to the next probe
    unsigned probes = 0;
    for (int64_t s = 0; s < a.nsteps; ++s) {
        const int64_t t = a.step0 + s;
        const int odd = (int)(t & 1);
        const bool probe = until == 0;
        until = probe ? a.every_k - 1 : until - 1;
        if (busy) {
            double f[F];
#pragma unroll
            for (int p = 0; p < F; ++p) {
                f[p] = 0.0;
                if (run) f[p] = odd ? cluster_ld(src[p]) : pop[(p + F * c) * C + here];
            }
            const CellMoments<double> m = collide_lanes<D, EQ, BULK>(f, c, base, a.rho0, om, sn);
            if (run) {
#pragma unroll
                for (int p = 0; p < F; ++p) {
                    if (odd) cluster_st(dst[p], f[p]);
                    else pop[(Q - 1 - p - F * c) * C + here] = f[p];
                }
            }
            if (probe) {
                const double q = c == 0 ? m.rho : m.rho * (c == 1 ? m.u[0] : m.u[1]);
                const double re = group_sums(run ? q * pr : 0.0), im = group_sums(run ? q * pi : 0.0);
                if (lane < 3) {
                    red[warp][2 * c] = re;
                    red[warp][2 * c + 1] = im;
                }
                if constexpr (D == 3) {
                    const double jz = m.rho * m.u[2];
                    const double re3 = group_sums(run ? jz * pr : 0.0), im3 = group_sums(run ? jz * pi : 0.0);
                    if (lane == 0) {
                        red[warp][6] = re3;
                        red[warp][7] = im3;
                    }
                }
            }
        }
        if (probe) {  // sums of the block, in pairs as in the teams
            __syncthreads();
            if (threadIdx.x < 8) {
                double sum = 0.0;
                for (int w = 0; w * 10 < mine; ++w) sum += red[w][threadIdx.x];
                sums[probes & 1][threadIdx.x] = sum;
            }
        }
        cluster_barrier();
        if (probe) {
            // lane j adds up the parts' sums j: the last warp of the last block with cells, which
            // often has none of its own
            if (part == parts - 1 && warp == kWarps - 1) {
                double sum = 0.0;
                const uint32_t at = smem_u32(&sums[probes & 1][lane & 7]);
                for (int q = 0; q < parts; ++q) sum += cluster_ld(cluster_addr(at, q));
                const bool fin = __all_sync(0xffffffffu, (lane & 7) >= N || isfinite(sum));
                const double mass = from_lane(sum, 0);
                if (lane >= N) sum = fin ? 0.0 : mass - mass;  // as probe_record
                const int64_t sample = t / a.every_k;
                if (lane < 8 && sample < a.max_samples) a.series[((int64_t)k * a.max_samples + sample) * 8 + lane] = sum;
                if (lane == 0 && !fin && a.status[k] == 0) a.status[k] = (int32_t)(t + 1);
            }
            ++probes;
        }
    }
    for (int p = threadIdx.x; p < Q * C; p += lbmh::kTeamThreads)
        if (p % C < mine) A[(int64_t)(p / C) * ncell + p % C] = pop[p];
    cluster_barrier();  // no block leaves while its sums may be read
}

// Instance of a packed global cell index (binary search over cell_start).
__device__ __forceinline__ int find_instance(const int64_t *cell_start, int64_t count, int64_t g) {
    int64_t lo = 0, hi = count - 1;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (cell_start[mid] <= g) lo = mid;
        else hi = mid - 1;
    }
    return (int)lo;
}

template <int D, int EQ, typename In>
__global__ void k_batch_init(double *arena, const int64_t *cell_start, const int32_t *dims,
                             int64_t count, double rho0, const In *rho, const In *u,
                             int64_t total) {
    constexpr int Q = qof(D);
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int k = find_instance(cell_start, count, g);
        const int64_t c0 = cell_start[k], n = cell_start[k + 1] - c0, c = g - c0;
        const double r = (double)rho[g];
        double uu[3] = {0, 0, 0};
        for (int a = 0; a < D; ++a) uu[a] = (double)u[(int64_t)D * c0 + a * n + c];
        double h[Q];
        equilibrium_h<D, EQ, double>(uu, h);
        double *A = arena + (int64_t)Q * c0;
        for (int i = 0; i < Q; ++i) A[(int64_t)i * n + c] = wq<D>(i) * fma(r, h[i], r - rho0);
    }
}

template <int D, typename Out>
__global__ void k_batch_moments(const double *arena, const int64_t *cell_start, const int32_t *dims,
                                int64_t count, double rho0, int odd, Out *rho, Out *u, int64_t total) {
    constexpr int Q = qof(D);
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int k = find_instance(cell_start, count, g);
        const int64_t c0 = cell_start[k], n = cell_start[k + 1] - c0, c = g - c0;
        const int nx = dims[3 * k], ny = dims[3 * k + 1], nz = dims[3 * k + 2];
        const int x = (int)(c % nx), y = (int)((c / nx) % ny), z = (int)(c / ((int64_t)nx * ny));
        const double *A = arena + (int64_t)Q * c0;
        double f[Q];
        for (int i = 0; i < Q; ++i) f[i] = A[aa_index<D>(i, x, y, z, nx, ny, nz, nx, n, odd)];
        const CellMoments<double> m = moments_shifted<D, double>(f, rho0);
        rho[g] = Out(m.rho);
        for (int a = 0; a < D; ++a) u[(int64_t)D * c0 + a * n + c] = Out(m.u[a]);
    }
}

template <int D, typename Out>
__global__ void k_batch_pop(const double *arena, const int64_t *cell_start, const int32_t *dims,
                            int64_t count, double rho0, int odd, Out *f, int64_t total) {
    constexpr int Q = qof(D);
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int k = find_instance(cell_start, count, g);
        const int64_t c0 = cell_start[k], n = cell_start[k + 1] - c0, c = g - c0;
        const int nx = dims[3 * k], ny = dims[3 * k + 1], nz = dims[3 * k + 2];
        const int x = (int)(c % nx), y = (int)((c / nx) % ny), z = (int)(c / ((int64_t)nx * ny));
        const double *A = arena + (int64_t)Q * c0;
        for (int i = 0; i < Q; ++i)
            f[(int64_t)Q * c0 + (int64_t)i * n + c] = Out(A[aa_index<D>(i, x, y, z, nx, ny, nz, nx, n, odd)] + wq<D>(i) * rho0);
    }
}

}  // namespace lbmd

namespace lbmh {

using namespace lbmd;

const void *batch_kernel(int D, int eq, int bulk) {
#define LBM_BK(Dv, EQv)                                                                        \
    if (D == Dv && eq == EQv)                                                                  \
        return bulk ? (const void *)k_step_batch<Dv, EQv, true> : (const void *)k_step_batch<Dv, EQv, false>;
    LBM_BK(2, EQ_ENT)
    LBM_BK(2, EQ_POLY2)
    LBM_BK(2, EQ_PROD)
    LBM_BK(3, EQ_ENT)
    LBM_BK(3, EQ_POLY2)
    LBM_BK(3, EQ_PROD)
#undef LBM_BK
    return nullptr;
}

static const void *team_kernel(int D, int eq, int bulk) {
#define LBM_BT(Dv, EQv)                                                                        \
    if (D == Dv && eq == EQv)                                                                  \
        return bulk ? (const void *)k_step_teams<Dv, EQv, true> : (const void *)k_step_teams<Dv, EQv, false>;
    LBM_BT(2, EQ_ENT)
    LBM_BT(2, EQ_POLY2)
    LBM_BT(2, EQ_PROD)
    LBM_BT(3, EQ_ENT)
    LBM_BT(3, EQ_POLY2)
    LBM_BT(3, EQ_PROD)
#undef LBM_BT
    return nullptr;
}

int team_block_capacity(int D, int eq, int bulk, int sms) {
    int nb = 0;
    const void *fn = team_kernel(D, eq, bulk);
    if (!fn || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, kTeamThreads, 0) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb * sms;
}

static const void *cluster_kernel(int D, int eq, int bulk) {
#define LBM_BC(Dv, EQv)                                                                                  \
    if (D == Dv && eq == EQv)                                                                            \
        return bulk ? (const void *)k_step_clusters<Dv, EQv, true> : (const void *)k_step_clusters<Dv, EQv, false>;
    LBM_BC(2, EQ_ENT)
    LBM_BC(2, EQ_POLY2)
    LBM_BC(2, EQ_PROD)
    LBM_BC(3, EQ_ENT)
    LBM_BC(3, EQ_POLY2)
    LBM_BC(3, EQ_PROD)
#undef LBM_BC
    return nullptr;
}

static void cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &at, int blocks, int cluster, cudaStream_t s) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kTeamThreads);
    cfg.stream = s;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
}

int batch_cluster_capacity(int D, int eq, int bulk, int cluster) {
    const void *fn = cluster_kernel(D, eq, bulk);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    cluster_config(cfg, at, cluster, cluster, nullptr);
    int n = 0;
    if (!fn || cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t step_teams(const BatchArgs &a, int blocks, cudaStream_t s) {
    BatchArgs aa = a;
    void *args[] = {(void *)&aa};
    const void *fn = a.team_cluster > 0 ? cluster_kernel(a.D, a.eq, a.bulk) : team_kernel(a.D, a.eq, a.bulk);
    if (!fn) return cudaErrorInvalidValue;
    if (a.team_cluster > 0) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at;
        cluster_config(cfg, at, blocks, a.team_cluster, s);
        return cudaLaunchKernelExC(&cfg, fn, args);
    }
    return cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(kTeamThreads), args, 0, s);
}

cudaError_t step_batch(const BatchArgs &a, int blocks, int threads, cudaStream_t s) {
    const void *fn = batch_kernel(a.D, a.eq, a.bulk);
    if (!fn) return cudaErrorInvalidValue;
    BatchArgs aa = a;
    void *args[] = {(void *)&aa};
    return cudaLaunchKernel(fn, dim3(blocks), dim3(threads), args, 0, s);
}

static int grid_cells(int64_t n) {
    int64_t g = (n + 255) / 256;
    return (int)(g < 1 ? 1 : (g > 152 * 32 ? 152 * 32 : g));
}

cudaError_t batch_init(double *arena, const int64_t *cell_start, const int32_t *dims,
                       int64_t count, int D, int eq, double rho0, const void *rho, const void *u,
                       int dtype, int64_t total, cudaStream_t s) {
    const int g = grid_cells(total);
#define LBM_BI(Dv, EQv)                                                                                    \
    if (D == Dv && eq == EQv) {                                                                            \
        if (dtype == 0)                                                                                    \
            k_batch_init<Dv, EQv, double><<<g, 256, 0, s>>>(arena, cell_start, dims, count, rho0,          \
                                                            (const double *)rho, (const double *)u, total); \
        else                                                                                               \
            k_batch_init<Dv, EQv, float><<<g, 256, 0, s>>>(arena, cell_start, dims, count, rho0,           \
                                                           (const float *)rho, (const float *)u, total);    \
        return cudaGetLastError();                                                                         \
    }
    LBM_BI(2, EQ_ENT)
    LBM_BI(2, EQ_POLY2)
    LBM_BI(2, EQ_PROD)
    LBM_BI(3, EQ_ENT)
    LBM_BI(3, EQ_POLY2)
    LBM_BI(3, EQ_PROD)
#undef LBM_BI
    return cudaErrorInvalidValue;
}

cudaError_t batch_moments(const double *arena, const int64_t *cell_start, const int32_t *dims,
                          int64_t count, int D, double rho0, int odd, void *rho, void *u,
                          int dtype, int64_t total, cudaStream_t s) {
    const int g = grid_cells(total);
    if (D == 2 && dtype == 0) k_batch_moments<2, double><<<g, 256, 0, s>>>(arena, cell_start, dims, count, rho0, odd, (double *)rho, (double *)u, total);
    else if (D == 2) k_batch_moments<2, float><<<g, 256, 0, s>>>(arena, cell_start, dims, count, rho0, odd, (float *)rho, (float *)u, total);
    else if (dtype == 0) k_batch_moments<3, double><<<g, 256, 0, s>>>(arena, cell_start, dims, count, rho0, odd, (double *)rho, (double *)u, total);
    else k_batch_moments<3, float><<<g, 256, 0, s>>>(arena, cell_start, dims, count, rho0, odd, (float *)rho, (float *)u, total);
    return cudaGetLastError();
}

cudaError_t batch_populations(const double *arena, const int64_t *cell_start,
                              const int32_t *dims, int64_t count, int D, double rho0, int odd,
                              void *f, int dtype, int64_t total, cudaStream_t s) {
    const int g = grid_cells(total);
    if (D == 2 && dtype == 0) k_batch_pop<2, double><<<g, 256, 0, s>>>(arena, cell_start, dims, count, rho0, odd, (double *)f, total);
    else if (D == 2) k_batch_pop<2, float><<<g, 256, 0, s>>>(arena, cell_start, dims, count, rho0, odd, (float *)f, total);
    else if (dtype == 0) k_batch_pop<3, double><<<g, 256, 0, s>>>(arena, cell_start, dims, count, rho0, odd, (double *)f, total);
    else k_batch_pop<3, float><<<g, 256, 0, s>>>(arena, cell_start, dims, count, rho0, odd, (float *)f, total);
    return cudaGetLastError();
}

}  // namespace lbmh
