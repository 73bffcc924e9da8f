// lbm_internal.h -- host-side launch interface between the C ABI (api.cu) and the
// kernel translation units.  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbmh {

// Layout of one lattice's populations: Q planes of `plane` elements, x fastest within a
// plane, rows `pitch` elements apart.  pitch == nx, or nx rounded up to whole 16-byte units
// so that every row of a ragged lattice starts where a bulk copy may start (the cells
// [nx, pitch) of a row are padding: copied with the row, never read by a real cell).
// Planes start on 256-byte boundaries (plane >= pitch * ny * nz).
struct Lattice {
    void *A;
    int64_t plane;
    int nx, ny, nz, pitch;
    int64_t ncell;
    int D, P;  // dimension (2 or 3), storage precision (lbmd::P_*)
};

// Per-step arguments shared by every step kernel.
struct StepArgs {
    Lattice lat;
    int eq, bulk;
    double rho0, omega0, six_nu;  // reference density, 1/tau, 6 nu
    float rho0f, omega0f, six_nuf; // the same in single precision (FP32 collisions)
    int odd;                      // AA pattern: 0 = even step, 1 = odd step
    int diag;                     // 1 = reduce diagnostics into partials
    double *partials;             // [blocks][8] when diag
    int32_t *status;              // device status word (LBM_ETIMEOUT on a timed-out wait)
    unsigned *sync;               // several steps a launch: ticket, exit and done counters (zero between launches)
    void *msg;                    // steps of a small lattice: step number and words (zero at first)
    int64_t timeout_ns;           // limit of every bounded device wait
};

// Launch shape of the TMA row-staged kernel.
struct TmaShape {
    int threads;    // consumer threads per block (the service warps are added)
    int blocks;     // grid size (persistent blocks) of several steps a launch
    int one_blocks; // and of one
    int stages;     // shared-memory pipeline depth (>= 2)
    int rows;       // rows per job (>= 1; 1 when the row is split into segments)
    int seg;        // cells per row segment (== nx for whole rows)
    int cap;        // bytes per direction buffer in shared memory (1024, 2048, 4096, 8192)
    int smem_bytes; // dynamic shared memory per block
};

constexpr int kDiagWords = 8;  // mass, jx, jy, jz, kinetic, max|u|, nonfinite, unused
constexpr int kBarStride = 32;  // counters of team barriers, one to a 128-byte line
constexpr int kSyncDone = 4;  // first done counter in StepArgs::sync (after the ticket and exit counters)
constexpr int64_t kTmaResident = (int64_t)75 << 20;  // populations that stay in the 129 MB L2 between steps
constexpr int kTmaMaxStages = 8;  // deepest shared-memory pipeline of the TMA row kernel

// api.cu: record the message of a failed call for lbm_last_error(); returns code.
int set_last_error(int code, const char *msg);

// k_generic.cu
cudaError_t step_generic(const StepArgs &a, int blocks, int threads, cudaStream_t s);
// Several steps of a small lattice in one cooperative launch.  small_shape: the launch, false if
// the lattice is too large for it.
struct SmallShape {
    int threads = 0, blocks = 0;
    bool lanes = false;  // an FP64 cell on three lanes (k_steps_lanes)
    bool many = false;   // several blocks to an SM: the kernel with fewer registers
};
// Blocks of 256 threads an SM that kernel's registers allow (P: 0 FP64, 1 FP32, 2 binary16).
constexpr int small_blocks(int D, int P) { return D == 2 ? (P == 2 ? 5 : 4) : P == 0 ? 2 : 3; }
// Bytes of StepArgs::msg, its words after the first kMsgHead.
constexpr int kMsgHead = 256;
size_t small_msg_bytes(const Lattice &lat);
bool small_shape(const Lattice &lat, int eq, int bulk, int sms, SmallShape &t);
cudaError_t steps_small(const StepArgs &a, int nsteps, const SmallShape &t, cudaStream_t s);
cudaError_t init_fields(const Lattice &lat, int eq, double rho0, const void *rho, const void *u,
                        int dtype, cudaStream_t s);
cudaError_t moments(const Lattice &lat, double rho0, int odd, void *rho, void *u, int dtype,
                    cudaStream_t s);
cudaError_t get_populations(const Lattice &lat, double rho0, int odd, void *f, int dtype,
                            cudaStream_t s);
cudaError_t set_populations(const Lattice &lat, double rho0, int odd, const void *f, int dtype,
                            cudaStream_t s);
cudaError_t sample_populations(const Lattice &lat, double rho0, int odd, const int64_t *cells,
                               int64_t count, double *out, cudaStream_t s);
cudaError_t diag_state(const Lattice &lat, double rho0, int odd, double *partials, int blocks,
                       cudaStream_t s);
cudaError_t diag_finalize(const double *partials, int blocks, int64_t step, double *record,
                          cudaStream_t s);
cudaError_t selftest_wait(int64_t timeout_ns, int32_t *status, cudaStream_t s);
int diag_blocks_generic(int64_t ncell);

// k_tma_*.cu
bool tma_supported(const Lattice &lat);
// Row pitch (elements) of a lattice: nx, or nx rounded up for the TMA kernel.
int padded_pitch(int D, int P, int64_t nx);
int tma_smem_bytes(const Lattice &lat, const TmaShape &t);
// Largest number of colliding threads per block of the TMA kernel for the lattice.
int tma_thread_limit(const Lattice &lat);
// Raises the kernels' dynamic shared memory limits to the most a block can have.
cudaError_t tma_prepare(const Lattice &lat, int eq, int bulk, int cap);
// Done counters a lattice is given (a row group has at least one row).
int64_t sync_units(const Lattice &lat);
// Steps one launch may take: the limits on tickets and launch length.  1 when the lattice has
// more units than counters.
int64_t tma_max_steps(const Lattice &lat, const TmaShape &t);
cudaError_t step_tma(const StepArgs &a, const TmaShape &t, int nsteps, cudaStream_t s);
// Sets the grid sizes of a shape: as many blocks as fit on the device.  False if none does.
bool tma_set_blocks(const Lattice &lat, int eq, int bulk, int sms, TmaShape &t);

// k_batch.cu -- many independent lattices in one arena (FP64, shifted).  Instance k has
// ncell_k = cell_start[k + 1] - cell_start[k] cells; its populations are Q planes of
// ncell_k doubles starting at arena + Q * cell_start[k].
struct BatchArgs {
    double *arena;
    const int64_t *cell_start;   // [count + 1]
    const int32_t *dims;         // [count][3]
    const double *omega0;        // [count] 1/tau_k
    const double *six_nu;        // [count] 6 nu_k
    const int32_t *order;        // instance ids, grouped per block
    const int32_t *block_start;  // [blocks + 1] range of `order` owned by each block
    const double2 *twiddle;      // exp(-i 2 pi n_a x_a / N_a) per instance, [Nx | Ny | Nz]
    const int64_t *tw_offset;    // [count] offset of instance k's twiddles
    double *series;              // [count][max_samples][8] (re, im of rho, jx, jy, jz)
    int64_t max_samples;
    int32_t *status;             // [count] 0, or first non-finite probed step + 1
    int64_t count;
    int D, eq, bulk;
    double rho0;
    int64_t step0, nsteps, every_k;  // first step, steps in this launch, probe period (0 = off)
    // teams of blocks (k_step_teams): instance and part of each block, blocks of each instance,
    // probe sums [2][blocks][8], counters (exits, then one per instance, kBarStride apart)
    const int32_t *team_instance, *team_part, *team_size;
    double *team_partials;
    unsigned *team_sync;
    int32_t *team_status;
    int team_cluster;  // blocks of an instance's thread-block cluster (k_step_clusters), 0: teams
    int64_t timeout_ns;
};
constexpr int kTeamThreads = 128;  // threads of a team's block
// Of n steps, those of the next launch of teams.  A team's counter grows by its blocks a step and is
// compared as a 32-bit number: without a limit 608 blocks of one instance passed 2^32 after 7 million steps.
constexpr int64_t team_launch_steps(int64_t n) { return n < 2000 ? n : 2000; }
constexpr int kClusterCells = kTeamThreads / 32 * 10;  // cells of a cluster's block, three lanes each
constexpr int kClusterBlocks = 8;                      // largest portable cluster
// Clusters of that many blocks that are resident at once.
int batch_cluster_capacity(int D, int eq, int bulk, int cluster);
// Blocks of the team kernel that are resident at once.
int team_block_capacity(int D, int eq, int bulk, int sms);
cudaError_t step_teams(const BatchArgs &a, int blocks, cudaStream_t s);
cudaError_t step_batch(const BatchArgs &a, int blocks, int threads, cudaStream_t s);
const void *batch_kernel(int D, int eq, int bulk);
cudaError_t batch_init(double *arena, const int64_t *cell_start, const int32_t *dims,
                       int64_t count, int D, int eq, double rho0, const void *rho, const void *u,
                       int dtype, int64_t total_cells, cudaStream_t s);
cudaError_t batch_moments(const double *arena, const int64_t *cell_start, const int32_t *dims,
                          int64_t count, int D, double rho0, int odd, void *rho, void *u,
                          int dtype, int64_t total_cells, cudaStream_t s);
cudaError_t batch_populations(const double *arena, const int64_t *cell_start,
                              const int32_t *dims, int64_t count, int D, double rho0, int odd,
                              void *f, int dtype, int64_t total_cells, cudaStream_t s);

// k_vn.cu
cudaError_t vn_eigs(int eq, int bulk, int64_t count, const double *params, double *out, int32_t *status,
                    cudaStream_t s);
// Trial speeds that a round of the stability search looks ahead at, as nodes of the tree of trials below
// the swept one (node 1; node n is followed by 2 n if unstable, 2 n + 1 if stable): those that unstable
// trials lead to after an unstable swept one (2, 4, .. 32), and after a stable one (3, 6, .. 48).
constexpr int kVnLooks = 10;
constexpr int vn_look_node(int q) { return q < kVnLooks / 2 ? 2 << q : 3 << (q - kVnLooks / 2); }
// Stability-limit search, all trials enqueued: in[npairs][2] = tau and theta, limit[npairs] the result,
// pairs vn_limit_bytes of device memory.
size_t vn_limit_bytes(int64_t npairs);
cudaError_t vn_limit(int eq, int64_t npairs, void *pairs, const double *in, double *limit, int nk, double u_hi, int iterations,
                     double tol, int32_t *status, cudaStream_t s);

}  // namespace lbmh
