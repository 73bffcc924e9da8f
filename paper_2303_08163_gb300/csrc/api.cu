// api.cu -- the C ABI declared in include/lbm.h: object lifetimes, argument checks,
// launch selection and the launch-shape autotuner.  All compute runs in the kernels of
// k_generic*.cu, k_tma*.cu and k_batch.cu; this file only marshals arguments and orders
// launches on the object's stream.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <queue>
#include <string>
#include <tuple>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "lbm.h"
#include "lbm_device.cuh"
#include "lbm_internal.h"

using namespace lbmh;

namespace {

thread_local std::string g_err;

int fail(int code, const char *fmt, ...) __attribute__((format(printf, 2, 3)));
int fail(int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

int esize_of(int P) { return P == LBM_F64 ? 8 : (P == LBM_F32 ? 4 : 2); }

int sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = 1;
        }
    }
    return n;
}

// 6 nu of the corrected rate 2 A / (6 nu + A), of a size whose square is a number (the rate is 0 to
// all digits long before).
double six_nu_of(double tau) { return std::min(6.0 * (tau - 0.5) / 3.0, 1e150); }

int64_t wait_timeout_ns() {
    const char *e = getenv("LBM_WAIT_TIMEOUT_NS");
    if (e && *e) {
        const long long v = atoll(e);
        if (v > 0) return v;
    }
    return 2000000000LL;  // 2 s
}

constexpr int64_t kHistCap = 65536;
constexpr int kPartialsCap = 152 * 32;

}  // namespace

struct lbm_ctx {
    int lattice = 0, D = 2, Q = 9, eq = 0, bulk = 0, prec = 0;
    int64_t dims[3] = {1, 1, 1};
    int64_t ncell = 0;
    double tau = 1, rho0 = 1, omega0 = 1, six_nu = 1;
    cudaStream_t stream = nullptr;
    Lattice lat{};
    int64_t step = 0;
    int sticky = 0;
    // diagnostics
    int64_t diag_every = 0;
    int32_t *status = nullptr;   // start of one allocation that holds these six
    unsigned *sync = nullptr;    // counters of several-step launches
    void *msg = nullptr;         // words of a small lattice's several-step launches
    double *partials = nullptr;  // [kPartialsCap][8]
    double *hist = nullptr;      // [kHistCap][8]
    double *scratch = nullptr;   // one record
    int64_t hist_count = 0;
    // launch
    int kernel = 1;
    int gen_threads = 256, gen_blocks = 1;
    bool chosen = false;  // the caller named a kernel or a launch shape
    SmallShape small;  // several steps of a small lattice at once (0 threads: too large)
    TmaShape tma{};      // of several steps a launch
    TmaShape tma_one{};  // of one
    bool use_graph = false;
    cudaGraphExec_t graph2 = nullptr;  // even + odd step
    // grow-only device staging for calls with host buffers
    void *stage[2] = {nullptr, nullptr};
    size_t stage_cap[2] = {0, 0};
};

struct lbm_batch {
    int lattice = 0, D = 2, Q = 9, eq = 0, bulk = 0;
    int64_t count = 0, total = 0;
    double rho0 = 1;
    cudaStream_t stream = nullptr;
    double *arena = nullptr;
    int64_t *d_cell_start = nullptr;
    int32_t *d_dims = nullptr;
    double *d_omega = nullptr, *d_sixnu = nullptr;
    int32_t *d_order = nullptr, *d_block_start = nullptr;
    double2 *d_tw = nullptr;
    int64_t *d_tw_off = nullptr;
    double *d_series = nullptr;
    int64_t max_samples = 0;
    int32_t *d_status = nullptr;
    int64_t every_k = 0;
    int64_t step = 0;
    int blocks = 0, threads = 256;
    int block_cap = 0;  // capacity of d_block_start (blocks + 1 entries at most)
    // teams of blocks (k_step_teams) instead of whole instances per block
    bool teams = false;
    int team_cluster = 0;             // blocks of a cluster (k_step_clusters), 0: teams over L2
    int team_blocks = 0;
    int64_t team_max = 0;             // largest number of cells of a block
    char *d_team = nullptr;           // one allocation for the team's tables, sums, counters and status
    int32_t *team_instance = nullptr, *team_part = nullptr, *team_size = nullptr, *team_status = nullptr;
    double *team_partials = nullptr;
    unsigned *team_sync = nullptr;
    int64_t max_load = 0, mean_load = 0;
    std::vector<int32_t> dims;
    std::vector<int64_t> cell_start;
    int sticky = 0;
};

extern "C" {
static int create_lattice(lbm_ctx **out, int lattice, const int64_t dims[3], double tau, int eq_kind,
                          int bulk_corr, int precision, double rho0, void *cuda_stream, bool pad);
}

namespace {

int cuda_fail(const char *what, cudaError_t e) {
    return fail(LBM_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define CK(call, what)                                      \
    do {                                                    \
        cudaError_t _e = (call);                            \
        if (_e != cudaSuccess) return cuda_fail(what, _e);  \
    } while (0)

int ctx_check(lbm_ctx *c) {
    if (!c) return fail(LBM_EINVAL, "null context");
    if (c->sticky) return fail(LBM_ESTATE, "context is in an error state (%d); destroy it", c->sticky);
    return LBM_OK;
}

int ctx_sticky(lbm_ctx *c, int code) {
    if (code == LBM_ECUDA || code == LBM_ETIMEOUT || code == LBM_ENOMEM) c->sticky = code;
    return code;
}

// Device status word: LBM_ETIMEOUT if a kernel's bounded wait ran out, LBM_ECHECK if a
// bounds or alignment check of a checked build failed (the first error sticks).
int read_status(lbm_ctx *c) {
    int32_t st = 0;
    cudaError_t e = cudaMemcpyAsync(&st, c->status, sizeof st, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("status read", e));
    if (st == LBM_ECHECK)
        return ctx_sticky(c, fail(LBM_ECHECK, "a device bounds or alignment check failed (checked build)"));
    if (st != 0) return ctx_sticky(c, fail(LBM_ETIMEOUT, "a bounded device wait ran out (status %d)", st));
    return LBM_OK;
}

StepArgs step_args(lbm_ctx *c, int odd, int diag) {
    StepArgs a;
    a.lat = c->lat;
    a.eq = c->eq;
    a.bulk = c->bulk;
    a.rho0 = c->rho0;
    a.omega0 = c->omega0;
    a.six_nu = c->six_nu;
    a.rho0f = (float)c->rho0;
    a.omega0f = (float)c->omega0;
    a.six_nuf = (float)c->six_nu;
    a.odd = odd;
    a.diag = diag;
    a.partials = c->partials;
    a.status = c->status;
    a.sync = c->sync;
    a.msg = c->msg;
    a.timeout_ns = wait_timeout_ns();
    return a;
}

int launch_blocks(lbm_ctx *c) { return c->kernel == 2 ? c->tma_one.one_blocks : c->gen_blocks; }

cudaError_t launch_one(lbm_ctx *c, int odd, int diag, cudaStream_t s) {
    const StepArgs a = step_args(c, odd, diag);
    if (c->kernel == 2) return step_tma(a, c->tma_one, 1, s);
    return step_generic(a, c->gen_blocks, c->gen_threads, s);
}

// n steps without diagnostics from the layout `odd` describes: several to a launch with the
// TMA kernel, one each with the one-cell kernel.
cudaError_t launch_steps(lbm_ctx *c, int odd, int64_t n, cudaStream_t s) {
    if (n > 1 && !c->chosen && c->small.threads > 0) {
        // (launches of bounded length: at most 90 ms with FP64 steps of 45 us)
        cudaError_t e = cudaSuccess;
        while (n > 0 && e == cudaSuccess) {
            const int64_t m = std::min<int64_t>(n, 2000);
            e = steps_small(step_args(c, odd, 0), (int)m, c->small, s);
            odd ^= (int)(m & 1);
            n -= m;
        }
        return e;
    }
    // (a few FP64 steps in 2-D are as well launched one by one: 512^2, two steps 66 us each, one by one 52)
    int64_t most = 1;
    if (c->kernel == 2 && n > (c->D == 2 && c->prec == LBM_F64 ? 4 : 1)) most = tma_max_steps(c->lat, c->tma);
    cudaError_t e = cudaSuccess;
    while (n > 0 && e == cudaSuccess) {
        const int64_t m = std::min(n, most);
        if (m == 1) e = launch_one(c, odd, 0, s);
        else e = step_tma(step_args(c, odd, 0), c->tma, (int)m, s);
        odd ^= (int)(m & 1);
        n -= m;
    }
    return e;
}

// Default TMA shape, used until the tuner runs.  128 colliding threads and 2 stages: two
// blocks per SM for D3Q27 with direction buffers of 2048 bytes (4096 when a row is longer, up
// to 4096 bytes), three for D2Q9 with 4096 bytes (4096^2 FP32, 200 steps with diagnostics
// every 10: 27.2 ms, against 30.4 with 3 stages and two blocks).  Whole rows filling the buffer
// when a row fits, otherwise equal aligned segments; as many blocks as fit on the device.
bool default_tma_shape(lbm_ctx *c, TmaShape &t) {
    const int es = esize_of(c->prec);
    const int64_t rowb = c->lat.pitch * (int64_t)es;
    const int U = 16 / es;
    t.threads = 128;
    int cap = c->D == 3 ? 2048 : 4096;
    if (c->D == 3 && rowb > cap && rowb <= 4096) cap = 4096;
    if (c->lat.pitch != c->lat.nx && rowb > cap) cap = 8192;  // padded rows are copied whole
    t.cap = cap;
    if (rowb <= cap) {
        t.seg = c->lat.nx;
        t.rows = (int)std::max<int64_t>(1, std::min<int64_t>(cap / rowb, c->lat.ny));
    } else {
        const int most = (cap / es - 2 * U) / U * U;
        const int64_t n = (c->lat.nx + most - 1) / most;
        t.seg = (int)(((c->lat.nx + n - 1) / n + U - 1) / U * U);
        t.rows = 1;
    }
    t.stages = 2;
    t.smem_bytes = tma_smem_bytes(c->lat, t);
    if (t.smem_bytes < 0) return false;
    if (!tma_set_blocks(c->lat, c->eq, c->bulk, sm_count(), t)) return false;
    // A lattice of few rows is spread over all blocks, one job each: jobs of full buffers would
    // leave most SMs without work (64^2 FP64: 8 jobs, 20.5 us a step; 64 jobs, 7.9 us).
    const int64_t groups = std::max<int64_t>(1, t.blocks / c->lat.nz);  // row groups of a plane
    t.rows = (int)std::max<int64_t>(1, std::min<int64_t>(t.rows, (c->lat.ny + groups - 1) / groups));
    // With little more than one job a block, a job's collisions (512 cells: two iterations of
    // 128 threads over pairs) are the step's critical path: 64^3 binary16 9.3 -> 7.7 us, 512^2
    // FP32 5.7 -> 5.1 us a step.
    while (t.rows > 1 && t.rows * c->lat.nx > 512 &&
           2 * ((c->lat.ny + t.rows - 1) / t.rows) * (int64_t)c->lat.nz < 3 * (int64_t)t.blocks)
        t.rows = (t.rows + 1) / 2;
    return true;
}

// The default shape of single steps: that of several, but for FP32 rows of 2-D lattices that pass HBM
// each step.  Those go in segments of up to 516 cells and 3 stages: steps launched one by one of 4096^2
// 200 -> 193 us, 3000^2 109 -> 105, 2048 x 4096 102 -> 98, 5000^2 294 -> 285 (with diagnostics 223 -> 216,
// 136 -> 133, 125 -> 123, 322 -> 317); in L2 (1024^2, 1400^2) 3 stages are slower.
TmaShape default_one_shape(lbm_ctx *c, const TmaShape &t) {
    TmaShape o = t;
    const int64_t state = (int64_t)c->Q * c->lat.plane * 4;
    if (c->D != 2 || c->prec != LBM_F32 || c->lat.pitch != c->lat.nx || c->lat.nx <= 516 || state <= kTmaResident) return o;
    const int64_t n = (c->lat.nx + 515) / 516;
    o.seg = (int)(((c->lat.nx + n - 1) / n + 3) / 4 * 4);
    o.rows = 1;
    o.stages = 3;
    o.smem_bytes = tma_smem_bytes(c->lat, o);
    return o.smem_bytes > 0 && tma_set_blocks(c->lat, c->eq, c->bulk, sm_count(), o) ? o : t;
}

// LBM_OPT_KERNEL 2 asks for the TMA kernel on unpadded rows only; padded ones use it by the library's own
// choice (LBM_OPT_KERNEL 0), the tuner's or a launch shape.
bool tma_selectable(lbm_ctx *c) { return tma_supported(c->lat) && c->lat.pitch == c->lat.nx; }

void drop_graph(lbm_ctx *c) {
    if (c->graph2) {
        cudaGraphExecDestroy(c->graph2);
        c->graph2 = nullptr;
    }
}

int build_graph(lbm_ctx *c) {
    drop_graph(c);
    cudaStream_t cap;
    CK(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "graph stream");
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        cudaError_t e1 = launch_one(c, 0, 0, cap);
        cudaError_t e2 = launch_one(c, 1, 0, cap);
        e = cudaStreamEndCapture(cap, &g);
        if (e == cudaSuccess && (e1 != cudaSuccess || e2 != cudaSuccess)) e = e1 != cudaSuccess ? e1 : e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&c->graph2, g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cap);
    if (e != cudaSuccess) return cuda_fail("graph capture", e);
    return LBM_OK;
}

int valid_dtype(int dtype) { return dtype == LBM_DT_F64 || dtype == LBM_DT_F32; }

// Copy a caller buffer into a temporary device buffer when it lives on the host.
struct DevBuf {
    void *p = nullptr;
    bool owned = false;
    ~DevBuf() {
        if (owned && p) cudaFree(p);
    }
};

// Device staging buffer `slot` of a context, grown to at least `bytes`.
int ctx_stage(lbm_ctx *c, int slot, size_t bytes, void **out) {
    if (c->stage_cap[slot] < bytes) {
        cudaStreamSynchronize(c->stream);
        cudaFree(c->stage[slot]);
        c->stage[slot] = nullptr;
        c->stage_cap[slot] = 0;
        if (cudaMalloc(&c->stage[slot], bytes) != cudaSuccess) {
            cudaGetLastError();
            return fail(LBM_ENOMEM, "device staging buffer of %zu bytes", bytes);
        }
        c->stage_cap[slot] = bytes;
    }
    *out = c->stage[slot];
    return LBM_OK;
}

int stage_in(const void *src, size_t bytes, int on_device, cudaStream_t s, DevBuf &out) {
    if (on_device) {
        out.p = const_cast<void *>(src);
        return LBM_OK;
    }
    if (cudaMalloc(&out.p, bytes) != cudaSuccess) {
        cudaGetLastError();
        return fail(LBM_ENOMEM, "device staging buffer of %zu bytes", bytes);
    }
    out.owned = true;
    CK(cudaMemcpyAsync(out.p, src, bytes, cudaMemcpyHostToDevice, s), "host to device copy");
    return LBM_OK;
}

// Device address of a page-locked host buffer (cudaHostAlloc or cudaHostRegister), or
// nullptr for pageable or device memory.  Kernels read and write such a buffer directly
// across the CPU-GPU link, as fast as a copy engine moves it, so the field upload and the
// moment download need neither a staging buffer nor a separate copy pass.
void *mapped_host(const void *p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return at.type == cudaMemoryTypeHost ? at.devicePointer : nullptr;
}

std::string tune_key(lbm_ctx *c) {
    cudaDeviceProp prop;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaGetDeviceProperties(&prop, dev);
    char buf[512];
    snprintf(buf, sizeof buf, "v%d|%s|D%d|P%d|E%d|B%d|%lldx%lldx%lld", lbm_version(), prop.name, c->D, c->prec,
             c->eq, c->bulk, (long long)c->dims[0], (long long)c->dims[1], (long long)c->dims[2]);
    std::string k = buf;
    for (char &ch : k)
        if (ch == ' ') ch = '_';
    return k;
}

std::mutex g_tune_mu;
std::map<std::string, std::vector<int>> g_tune_cache;

const char *tune_file() {
    const char *e = getenv("LBM_TUNE_CACHE");
    return (e && *e) ? e : nullptr;
}

void tune_cache_load() {
    const char *path = tune_file();
    if (!path) return;
    FILE *f = fopen(path, "r");
    if (!f) return;
    char key[512];
    int v[8];
    while (fscanf(f, "%511s %d %d %d %d %d %d %d %d", key, &v[0], &v[1], &v[2], &v[3], &v[4], &v[5], &v[6], &v[7]) == 9)
        g_tune_cache[key] = std::vector<int>(v, v + 8);
    fclose(f);
}

void tune_cache_store(const std::string &key, const std::vector<int> &v) {
    g_tune_cache[key] = v;
    const char *path = tune_file();
    if (!path) return;
    FILE *f = fopen(path, "a");
    if (!f) return;
    fprintf(f, "%s", key.c_str());
    for (int x : v) fprintf(f, " %d", x);
    fprintf(f, "\n");
    fclose(f);
}

// Rebuild a launch shape from a cached or tuned record {kernel, threads, blocks, stages,
// rows, seg, cap, smem} and check it against this lattice and device before it is used:
// the TMA geometry must be valid, its shared memory must equal the recorded figure, and
// the block count is recomputed from the device's occupancy (a stale or edited record,
// or one written by another build or device, is rejected instead of launched).
bool shape_from_record(lbm_ctx *c, const std::vector<int> &v, int *kernel, TmaShape *t, int *gt, int *gb) {
    if (v.size() != 8) return false;
    if (v[0] == 1) {
        if (v[1] < 32 || v[1] > 256 || v[1] % 32) return false;
        *kernel = 1;
        *gt = v[1];
        *gb = (int)std::max<int64_t>(1, std::min<int64_t>((c->ncell + v[1] - 1) / v[1], (int64_t)sm_count() * 16));
        return true;
    }
    if (v[0] != 2 || !tma_supported(c->lat)) return false;
    TmaShape s{};
    s.threads = v[1];
    s.stages = v[3];
    s.rows = v[4];
    s.seg = v[5];
    s.cap = v[6];
    if (s.rows < 1 || s.seg < 16 / esize_of(c->prec)) return false;
    s.smem_bytes = tma_smem_bytes(c->lat, s);
    if (s.smem_bytes < 0 || s.smem_bytes != v[7]) return false;
    if (!tma_set_blocks(c->lat, c->eq, c->bulk, sm_count(), s)) return false;
    *kernel = 2;
    *t = s;
    return true;
}

// Apply a record checked by shape_from_record; false (and the context unchanged) if the
// record does not describe a runnable shape of this lattice.
bool apply_shape(lbm_ctx *c, const std::vector<int> &v) {
    int kernel = 0, gt = 0, gb = 0;
    TmaShape t{};
    if (!shape_from_record(c, v, &kernel, &t, &gt, &gb)) return false;
    if (kernel == 2) {
        if (tma_prepare(c->lat, c->eq, c->bulk, t.cap) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        c->tma = c->tma_one = t;
    } else {
        c->gen_threads = gt;
        c->gen_blocks = gb;
    }
    c->kernel = kernel;
    return true;
}

// Device time of nsteps steps of the context's current launch shape, continuing its step
// parity; -1 if a launch failed.
float time_steps(lbm_ctx *c, int64_t step0, int nsteps) {
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return -1;
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return -1;
    }
    bool ok = cudaEventRecord(e0, c->stream) == cudaSuccess;
    ok = ok && launch_steps(c, (int)(step0 & 1), nsteps, c->stream) == cudaSuccess;
    ok = ok && cudaEventRecord(e1, c->stream) == cudaSuccess;
    float ms = -1;
    if (ok && cudaEventSynchronize(e1) == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
    if (cudaGetLastError() != cudaSuccess) ms = -1;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return ok ? ms : -1;
}

// Status word of a context read and cleared without making it sticky (tuning only): a
// candidate shape whose bounded wait ran out, or whose checked-build test failed, must
// not win by finishing early.
bool take_status_clean(lbm_ctx *c) {
    int32_t st = 0;
    cudaError_t e = cudaMemcpyAsync(&st, c->status, sizeof st, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (st != 0) {
        cudaMemsetAsync(c->status, 0, sizeof(int32_t), c->stream);
        cudaStreamSynchronize(c->stream);
        return false;
    }
    return true;
}

// Populations the tuner's proxy lattice holds at most (plus whole planes).
constexpr int64_t kTuneProxyBytes = (int64_t)2 << 30;

// Owner of the tuner's proxy lattice.
struct ProxyCtx {
    lbm_ctx *p = nullptr;
    ~ProxyCtx() {
        if (p) lbm_destroy(p);
    }
};

int autotune(lbm_ctx *c) {
    // Tune on a proxy lattice with the same row geometry: the same Nx (and Ny for D3Q27)
    // and at most kTuneProxyBytes of populations in whole z-planes (D3Q27) or y-rows
    // (D2Q9), filled with the first planes of the current state.  The context's own state
    // is never stepped, so no backup of it is needed and a lattice larger than the free
    // device memory can be tuned; the timing of a 2 GiB proxy (16 times the L2 cache)
    // follows the full lattice's, since the step kernels stream every plane alike.
    const int es = esize_of(c->prec);
    int64_t pd[3] = {c->dims[0], c->dims[1], c->dims[2]};
    const int cut = c->D == 3 ? 2 : 1;
    const int64_t per = (int64_t)c->Q * es * (c->D == 3 ? c->dims[0] * c->dims[1] : c->dims[0]);
    int64_t keep = std::max<int64_t>(1, kTuneProxyBytes / per);
    if (c->D == 2 && keep < c->dims[1]) keep = std::max<int64_t>(64, keep / 64 * 64);
    pd[cut] = std::min<int64_t>(c->dims[cut], keep);
    ProxyCtx px;
    // (its planes are copied byte for byte, so its rows have to be padded as the lattice's are)
    int rc = create_lattice(&px.p, c->lattice, pd, c->tau, c->eq, c->bulk, c->prec, c->rho0, c->stream, c->lat.pitch != c->lat.nx);
    if (rc) return rc;
    lbm_ctx *p = px.p;
    p->step = c->step;  // the same AA parity: the copied planes are a consistent layout
    // one copy per direction plane (a plane of a large lattice exceeds the pitch limit
    // of a 2-D copy)
    for (int i = 0; i < c->Q; ++i)
        CK(cudaMemcpyAsync(static_cast<char *>(p->lat.A) + (size_t)i * p->lat.plane * es,
                           static_cast<const char *>(c->lat.A) + (size_t)i * c->lat.plane * es, (size_t)p->lat.pitch * pd[1] * pd[2] * es,
                           cudaMemcpyDeviceToDevice, c->stream),
           "tuning proxy fill");
    std::vector<std::vector<int>> cands;
    const int U = 16 / es;
    const int64_t rowb = c->lat.pitch * (int64_t)es;
    for (int th : {128, 256}) {
        int g = (int)std::min<int64_t>((c->ncell + th - 1) / th, (int64_t)sm_count() * 16);
        cands.push_back({1, th, std::max(g, 1), 0, 0, 0, 0, 0});
    }
    if (tma_supported(c->lat)) {
        for (int cap : {1024, 2048, 4096, 8192}) {
            std::vector<std::pair<int, int>> geo;  // (rows, seg)
            if (rowb <= cap) {
                const int rmax = (int)std::min<int64_t>(cap / rowb, c->lat.ny);
                geo.push_back({rmax, (int)c->lat.nx});
                if (rmax > 1) geo.push_back({std::max(1, rmax / 2), (int)c->lat.nx});
            } else if (c->lat.pitch == c->lat.nx) {
                // the longest segment the buffer holds, and the same number of segments
                // made equal (no short ragged last segment with a job's full overhead)
                const int smax = (cap / es - 2 * U) / U * U;
                geo.push_back({1, smax});
                const int64_t nseg = (c->lat.nx + smax - 1) / smax;
                const int sbal = (int)(((c->lat.nx + nseg - 1) / nseg + U - 1) / U * U);
                if (sbal < smax) geo.push_back({1, sbal});
            }
            const std::vector<int> ths = tma_thread_limit(c->lat) > 256
                                             ? std::vector<int>{128, 192, 256, 384, 512}
                                             : std::vector<int>{128, 192, 256};
            for (auto rs : geo)
                for (int th : ths)
                    for (int st : {2, 3, 4, 6, 8}) {
                        TmaShape t{};
                        t.threads = th;
                        t.stages = st;
                        t.rows = rs.first;
                        t.seg = rs.second;
                        t.cap = cap;
                        t.smem_bytes = tma_smem_bytes(c->lat, t);
                        if (t.smem_bytes < 0) continue;
                        if (!tma_set_blocks(c->lat, c->eq, c->bulk, sm_count(), t)) continue;
                        // keep 2..4 stages per block only when several blocks share an SM
                        if (t.blocks / sm_count() * st > 16) continue;
                        cands.push_back({2, t.threads, t.blocks, t.stages, t.rows, t.seg, t.cap, t.smem_bytes});
                    }
        }
    }
    // Pass 1: every candidate, a few steps.  Pass 2: the fastest few again, in
    // interleaved rounds, scored by their median.  Then, among the shapes within 0.5 % of
    // the best score (the run-to-run noise of one box), the one with the least shared
    // memory, fewest stages and fewest threads: equally fast boxes then pick the same shape.
    const int reps = p->ncell * (int64_t)c->Q * es > ((int64_t)1 << 28) ? 4 : 10;
    std::vector<std::pair<float, size_t>> score;
    p->chosen = true;  // time the candidates themselves
    for (size_t q = 0; q < cands.size(); ++q) {
        if (!apply_shape(p, cands[q])) continue;
        if (time_steps(p, p->step, 2) < 0 || !take_status_clean(p)) continue;
        const float ms = time_steps(p, p->step, reps);
        if (ms > 0 && take_status_clean(p)) score.push_back({ms, q});
    }
    cudaGetLastError();
    if (score.empty()) return fail(LBM_ECUDA, "autotune found no runnable launch shape");
    std::sort(score.begin(), score.end());
    const size_t top = std::min<size_t>(score.size(), 6);
    std::vector<std::vector<float>> rounds(top);
    for (int r = 0; r < 3; ++r)
        for (size_t q = 0; q < top; ++q) {
            if (!apply_shape(p, cands[score[q].second])) continue;
            const float ms = time_steps(p, p->step, reps);
            if (ms > 0 && take_status_clean(p)) rounds[q].push_back(ms);
        }
    std::vector<std::pair<float, size_t>> fin;
    for (size_t q = 0; q < top; ++q) {
        auto &v = rounds[q];
        if (v.size() < 3) continue;
        std::sort(v.begin(), v.end());
        fin.push_back({v[v.size() / 2], score[q].second});
    }
    if (fin.empty()) fin.push_back(score[0]);
    std::sort(fin.begin(), fin.end());
    const float limit = fin[0].first * 1.005f;
    size_t pick = fin[0].second;
    for (const auto &f : fin) {
        if (f.first > limit) break;
        const auto &a = cands[f.second], &b = cands[pick];
        // record order: {kernel, threads, blocks, stages, rows, seg, cap, smem}
        const auto key_a = std::make_tuple(a[7], a[3], a[1], a[4], a[5]);
        const auto key_b = std::make_tuple(b[7], b[3], b[1], b[4], b[5]);
        if (key_a < key_b) pick = f.second;
    }
    CK(cudaStreamSynchronize(c->stream), "autotune sync");
    if (!apply_shape(c, cands[pick])) return fail(LBM_ECUDA, "autotune: the chosen launch shape cannot be prepared");
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        tune_cache_store(tune_key(c), cands[pick]);
    }
    drop_graph(c);
    return LBM_OK;
}

}  // namespace

namespace lbmh {
int set_last_error(int code, const char *msg) {
    g_err = msg;
    return code;
}
}  // namespace lbmh

// NVTX range around a public call (header-only NVTX: free unless a profiler is attached).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
};

extern "C" {

const char *lbm_last_error(void) { return g_err.c_str(); }

int lbm_version(void) { return 10100; }

// pad: ragged rows may be padded for the TMA kernel.
static int create_lattice(lbm_ctx **out, int lattice, const int64_t dims[3], double tau, int eq_kind,
                          int bulk_corr, int precision, double rho0, void *cuda_stream, bool pad) {
    if (!out || !dims) return fail(LBM_EINVAL, "null argument");
    *out = nullptr;
    if (lattice != LBM_D2Q9 && lattice != LBM_D3Q27) return fail(LBM_EINVAL, "bad lattice %d", lattice);
    if (eq_kind < 0 || eq_kind > 2) return fail(LBM_EINVAL, "bad eq_kind %d", eq_kind);
    if (bulk_corr != 0 && bulk_corr != 1) return fail(LBM_EINVAL, "bulk_corr must be 0 or 1");
    if (precision < 0 || precision > 2) return fail(LBM_EINVAL, "bad precision %d", precision);
    if (!(tau > 0.5) || !std::isfinite(tau)) return fail(LBM_EINVAL, "tau must be a finite value > 1/2 (got %g)", tau);
    if (!(rho0 > 0) || !std::isfinite(rho0)) return fail(LBM_EINVAL, "rho0 must be positive");
    for (int a = 0; a < 3; ++a)
        if (dims[a] < 1 || dims[a] > (1 << 30)) return fail(LBM_EINVAL, "dims[%d] = %lld out of range", a, (long long)dims[a]);
    if (lattice == LBM_D2Q9 && dims[2] != 1) return fail(LBM_EINVAL, "D2Q9 needs dims[2] == 1");
    const int64_t ncell = dims[0] * dims[1] * dims[2];
    if (ncell / dims[0] / dims[1] != dims[2] || ncell > ((int64_t)1 << 40)) return fail(LBM_EINVAL, "lattice too large");
    lbm_ctx *c = new lbm_ctx();
    c->lattice = lattice;
    c->D = lattice == LBM_D2Q9 ? 2 : 3;
    c->Q = c->D == 2 ? 9 : 27;
    c->eq = eq_kind;
    c->bulk = bulk_corr;
    c->prec = precision;
    for (int a = 0; a < 3; ++a) c->dims[a] = dims[a];
    c->ncell = ncell;
    c->tau = tau;
    c->rho0 = rho0;
    c->omega0 = 1.0 / tau;
    c->six_nu = six_nu_of(tau);
    c->stream = static_cast<cudaStream_t>(cuda_stream);
    const int es = esize_of(precision);
    const int64_t align = 256 / es;
    c->lat.pitch = pad ? padded_pitch(c->D, precision, dims[0]) : (int)dims[0];
    const int64_t plane = (c->lat.pitch * dims[1] * dims[2] + align - 1) / align * align;
    c->lat.nx = (int)dims[0];
    c->lat.ny = (int)dims[1];
    c->lat.nz = (int)dims[2];
    c->lat.ncell = ncell;
    c->lat.D = c->D;
    c->lat.P = precision;
    const size_t bytes = (size_t)c->Q * plane * es;
    c->lat.plane = plane;
    if (cudaMalloc(&c->lat.A, bytes) != cudaSuccess) {
        cudaGetLastError();
        delete c;
        return fail(LBM_ENOMEM, "population storage of %zu bytes", bytes);
    }
    // one allocation for the small buffers; the status word and the counters start at zero
    const size_t zeroed = 256 + (sizeof(unsigned) * (kSyncDone + sync_units(c->lat)) + 255) / 256 * 256;
    const size_t recs = sizeof(double) * kDiagWords * (kPartialsCap + kHistCap + 4);
    char *aux = nullptr;
    size_t msg = small_shape(c->lat, c->eq, c->bulk, sm_count(), c->small) ? (small_msg_bytes(c->lat) + 255) / 256 * 256 : 0;
    cudaError_t ea = cudaMalloc(&aux, zeroed + msg + recs);
    if (ea != cudaSuccess && msg > 0) {  // no room for the words: as a larger lattice
        cudaGetLastError();
        msg = 0;
        ea = cudaMalloc(&aux, zeroed + recs);
    }
    if (msg == 0) c->small.threads = 0;
    if (ea != cudaSuccess) {
        cudaGetLastError();
        lbm_destroy(c);
        return fail(LBM_ENOMEM, "diagnostics buffers");
    }
    c->status = reinterpret_cast<int32_t *>(aux);
    c->sync = reinterpret_cast<unsigned *>(aux + 256);
    c->msg = aux + zeroed;
    c->partials = reinterpret_cast<double *>(aux + zeroed + msg);
    c->hist = c->partials + kDiagWords * kPartialsCap;
    c->scratch = c->hist + 8 * kHistCap;
    if (cudaMemsetAsync(c->lat.A, 0, bytes, c->stream) != cudaSuccess ||
        cudaMemsetAsync(aux, 0, zeroed + msg, c->stream) != cudaSuccess) {
        lbm_destroy(c);
        return cuda_fail("initial memset", cudaGetLastError());
    }
    c->gen_threads = 256;
    c->gen_blocks = (int)std::max<int64_t>(1, std::min<int64_t>((ncell + 255) / 256, (int64_t)sm_count() * 16));
    c->kernel = 1;
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        static bool loaded = false;
        if (!loaded) {
            tune_cache_load();
            loaded = true;
        }
        auto it = g_tune_cache.find(tune_key(c));
        if (it != g_tune_cache.end() && apply_shape(c, it->second)) {
            *out = c;
            return LBM_OK;
        }
    }
    if (tma_supported(c->lat) && default_tma_shape(c, c->tma)) {
        c->tma_one = default_one_shape(c, c->tma);
        c->kernel = 2;
    }
    cudaGetLastError();
    *out = c;
    return LBM_OK;
}

int lbm_create(lbm_ctx **out, int lattice, const int64_t dims[3], double tau, int eq_kind,
               int bulk_corr, int precision, double rho0, void *cuda_stream) {
    int rc = create_lattice(out, lattice, dims, tau, eq_kind, bulk_corr, precision, rho0, cuda_stream, true);
    // no room for the padding: unpadded rows (and the one-cell kernel)
    if (rc == LBM_ENOMEM && padded_pitch(lattice == LBM_D2Q9 ? 2 : 3, precision, dims[0]) != dims[0])
        rc = create_lattice(out, lattice, dims, tau, eq_kind, bulk_corr, precision, rho0, cuda_stream, false);
    return rc;
}

int lbm_set_option(lbm_ctx *c, int option, int64_t value) {
    int rc = ctx_check(c);
    if (rc) return rc;
    switch (option) {
    case LBM_OPT_DIAG_EVERY:
        if (value < 0) return fail(LBM_EINVAL, "diag_every must be >= 0");
        c->diag_every = value;
        return LBM_OK;
    case LBM_OPT_KERNEL:
        if (value < 0 || value > 2) return fail(LBM_EINVAL, "kernel must be 0, 1 or 2");
        if (value == 2 && !tma_selectable(c))
            return fail(LBM_EINVAL, "TMA row kernel needs Nx * sizeof(storage) to be a multiple of 16");
        c->chosen = value != 0;
        if (value == 1) c->kernel = 1;
        if (value == 2 || value == 0) {
            if (tma_supported(c->lat)) {
                if (c->tma.smem_bytes <= 0) {
                    if (!default_tma_shape(c, c->tma)) return fail(LBM_ECUDA, "no TMA launch shape fits this lattice");
                    c->tma_one = default_one_shape(c, c->tma);
                }
                c->kernel = 2;
            } else {
                c->kernel = 1;
            }
        }
        drop_graph(c);
        return LBM_OK;
    case LBM_OPT_USE_GRAPH:
        c->use_graph = value != 0;
        drop_graph(c);
        return LBM_OK;
    case LBM_OPT_TUNE:
        if (value) {
            // a proxy that does not fit in memory leaves the context usable
            rc = autotune(c);
            return rc == LBM_ENOMEM ? rc : ctx_sticky(c, rc);
        }
        return LBM_OK;
    default:
        return fail(LBM_EINVAL, "unknown option %d", option);
    }
}

int lbm_init_fields(lbm_ctx *c, const void *rho, const void *u, int dtype, int on_device) {
    int rc = ctx_check(c);
    if (rc) return rc;
    if (!rho || !u || !valid_dtype(dtype)) return fail(LBM_EINVAL, "bad field arguments");
    const size_t es = dtype == LBM_DT_F64 ? 8 : 4;
    const void *dr = rho, *du = u;
    void *mr = on_device ? nullptr : mapped_host(rho), *mu = on_device ? nullptr : mapped_host(u);
    if (mr && mu) {
        // page-locked fields: the initialisation kernel reads them across the link
        dr = mr;
        du = mu;
    } else if (!on_device) {
        void *pr, *pu;
        if ((rc = ctx_stage(c, 0, es * c->ncell, &pr))) return ctx_sticky(c, rc);
        if ((rc = ctx_stage(c, 1, es * c->ncell * c->D, &pu))) return ctx_sticky(c, rc);
        CK(cudaMemcpyAsync(pr, rho, es * c->ncell, cudaMemcpyHostToDevice, c->stream), "field upload");
        CK(cudaMemcpyAsync(pu, u, es * c->ncell * c->D, cudaMemcpyHostToDevice, c->stream), "field upload");
        dr = pr;
        du = pu;
    }
    cudaError_t e = init_fields(c->lat, c->eq, c->rho0, dr, du, dtype, c->stream);
    if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("init kernel", e));
    c->step = 0;
    c->hist_count = 0;
    drop_graph(c);
    if (!on_device) {
        // host buffers (pinned ones included) are only borrowed for the call
        e = cudaStreamSynchronize(c->stream);
        if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("init sync", e));
    }
    return LBM_OK;
}

int lbm_step(lbm_ctx *c, int64_t n) {
    NvtxRange range("lbm_step");
    int rc = ctx_check(c);
    if (rc) return rc;
    if (n < 0) return fail(LBM_EINVAL, "n must be >= 0");
    int64_t ndiag = 0;
    int64_t s = 0;
    if (c->use_graph && c->diag_every == 0) {
        if ((c->step & 1) && n > 0) {
            cudaError_t e = launch_one(c, 1, 0, c->stream);
            if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("step launch", e));
            ++c->step;
            ++s;
        }
        if (n - s >= 2 && !c->graph2) {
            if ((rc = build_graph(c))) return ctx_sticky(c, rc);
        }
        while (n - s >= 2) {
            cudaError_t e = cudaGraphLaunch(c->graph2, c->stream);
            if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("graph launch", e));
            c->step += 2;
            s += 2;
        }
    }
    for (; s < n; ++s) {
        const int odd = (int)(c->step & 1);
        const int diag = c->diag_every > 0 && (c->step % c->diag_every) == 0;
        if (!diag) {
            // up to the next diagnostics step
            int64_t m = n - s;
            if (c->diag_every > 0) m = std::min(m, c->diag_every - c->step % c->diag_every);
            cudaError_t e = launch_steps(c, odd, m, c->stream);
            if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("step launch", e));
            c->step += m;
            s += m - 1;
            continue;
        }
        cudaError_t e = launch_one(c, odd, diag, c->stream);
        if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("step launch", e));
        if (diag) {
            e = diag_finalize(c->partials, launch_blocks(c), c->step, c->hist + 8 * (c->hist_count % kHistCap), c->stream);
            if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("diagnostics launch", e));
            ++c->hist_count;
            ++ndiag;
        }
        ++c->step;
    }
    if (ndiag > 0) {
        if ((rc = read_status(c))) return rc;
        const int64_t take = std::min<int64_t>(ndiag, kHistCap);
        std::vector<double> rec(8 * take);
        for (int64_t q = 0; q < take; ++q) {
            const int64_t slot = (c->hist_count - take + q) % kHistCap;
            cudaError_t e = cudaMemcpy(&rec[8 * q], c->hist + 8 * slot, 8 * sizeof(double), cudaMemcpyDeviceToHost);
            if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("diagnostics copy", e));
        }
        for (int64_t q = 0; q < take; ++q)
            if (rec[8 * q + 6] > 0 || !std::isfinite(rec[8 * q + 0]))
                return fail(LBM_ENONFINITE, "non-finite state at step %lld", (long long)rec[8 * q + 7]);
    }
    return LBM_OK;
}

int lbm_moments(lbm_ctx *c, void *rho, void *u, int dtype, int on_device) {
    int rc = ctx_check(c);
    if (rc) return rc;
    if (!rho || !u || !valid_dtype(dtype)) return fail(LBM_EINVAL, "bad field arguments");
    const size_t es = dtype == LBM_DT_F64 ? 8 : 4;
    void *dr = rho, *du = u;
    void *mr = on_device ? nullptr : mapped_host(rho), *mu = on_device ? nullptr : mapped_host(u);
    const bool direct = mr && mu;  // page-locked outputs: the kernel writes them across the link
    if (direct) {
        dr = mr;
        du = mu;
    } else if (!on_device) {
        if ((rc = ctx_stage(c, 0, es * c->ncell, &dr))) return ctx_sticky(c, rc);
        if ((rc = ctx_stage(c, 1, es * c->ncell * c->D, &du))) return ctx_sticky(c, rc);
    }
    cudaError_t e = moments(c->lat, c->rho0, (int)(c->step & 1), dr, du, dtype, c->stream);
    if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("moments kernel", e));
    if (!on_device) {
        if (!direct) {
            CK(cudaMemcpyAsync(rho, dr, es * c->ncell, cudaMemcpyDeviceToHost, c->stream), "moments copy");
            CK(cudaMemcpyAsync(u, du, es * c->ncell * c->D, cudaMemcpyDeviceToHost, c->stream), "moments copy");
        }
        CK(cudaStreamSynchronize(c->stream), "moments sync");
        return read_status(c);
    }
    return LBM_OK;
}

static void fill_diag(const double *r, lbm_diag *out) {
    out->mass = r[0];
    out->momentum[0] = r[1];
    out->momentum[1] = r[2];
    out->momentum[2] = r[3];
    out->kinetic = r[4];
    out->max_u = r[5];
    out->nonfinite = (int64_t)r[6];
    out->step = (int64_t)r[7];
}

int lbm_diagnostics(lbm_ctx *c, lbm_diag *out) {
    int rc = ctx_check(c);
    if (rc) return rc;
    if (!out) return fail(LBM_EINVAL, "null output");
    const int blocks = diag_blocks_generic(c->ncell);
    cudaError_t e = diag_state(c->lat, c->rho0, (int)(c->step & 1), c->partials, blocks, c->stream);
    if (e == cudaSuccess) e = diag_finalize(c->partials, blocks, c->step, c->scratch, c->stream);
    if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("diagnostics kernel", e));
    double r[8];
    CK(cudaMemcpyAsync(r, c->scratch, sizeof r, cudaMemcpyDeviceToHost, c->stream), "diagnostics copy");
    CK(cudaStreamSynchronize(c->stream), "diagnostics sync");
    if ((rc = read_status(c))) return rc;
    fill_diag(r, out);
    return LBM_OK;
}

int lbm_diag_history(lbm_ctx *c, lbm_diag *out, int64_t max, int64_t *count) {
    int rc = ctx_check(c);
    if (rc) return rc;
    if (!count || (max > 0 && !out) || max < 0) return fail(LBM_EINVAL, "bad history arguments");
    const int64_t avail = std::min<int64_t>(c->hist_count, kHistCap);
    *count = avail;
    const int64_t take = std::min<int64_t>(avail, max);
    if (take == 0) return LBM_OK;
    std::vector<double> all(8 * kHistCap);
    CK(cudaStreamSynchronize(c->stream), "history sync");
    CK(cudaMemcpy(all.data(), c->hist, sizeof(double) * 8 * kHistCap, cudaMemcpyDeviceToHost), "history copy");
    if ((rc = read_status(c))) return rc;
    const int64_t first = c->hist_count - avail;
    for (int64_t q = 0; q < take; ++q) fill_diag(&all[8 * ((first + q) % kHistCap)], &out[q]);
    return LBM_OK;
}

static size_t pop_esize(lbm_ctx *c, int dtype) {
    return dtype == LBM_DT_F64 ? 8 : (dtype == LBM_DT_F32 ? 4 : (size_t)esize_of(c->prec));
}

int lbm_get_populations(lbm_ctx *c, void *f, int dtype, int on_device) {
    int rc = ctx_check(c);
    if (rc) return rc;
    if (!f || !(valid_dtype(dtype) || dtype == LBM_DT_STORAGE)) return fail(LBM_EINVAL, "bad population arguments");
    const size_t bytes = pop_esize(c, dtype) * c->Q * c->ncell;
    void *d = f;
    DevBuf b;
    if (!on_device) {
        if (cudaMalloc(&b.p, bytes) != cudaSuccess) {
            cudaGetLastError();
            return fail(LBM_ENOMEM, "population staging of %zu bytes", bytes);
        }
        b.owned = true;
        d = b.p;
    }
    cudaError_t e = get_populations(c->lat, c->rho0, (int)(c->step & 1), d, dtype, c->stream);
    if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("population export", e));
    if (!on_device) {
        CK(cudaMemcpyAsync(f, d, bytes, cudaMemcpyDeviceToHost, c->stream), "population copy");
        CK(cudaStreamSynchronize(c->stream), "population sync");
        return read_status(c);
    }
    return LBM_OK;
}

int lbm_set_populations(lbm_ctx *c, const void *f, int dtype, int on_device) {
    int rc = ctx_check(c);
    if (rc) return rc;
    if (!f || !(valid_dtype(dtype) || dtype == LBM_DT_STORAGE)) return fail(LBM_EINVAL, "bad population arguments");
    const size_t bytes = pop_esize(c, dtype) * c->Q * c->ncell;
    DevBuf b;
    if ((rc = stage_in(f, bytes, on_device, c->stream, b))) return ctx_sticky(c, rc);
    cudaError_t e = set_populations(c->lat, c->rho0, (int)(c->step & 1), b.p, dtype, c->stream);
    if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("population import", e));
    c->hist_count = 0;
    if (!on_device) CK(cudaStreamSynchronize(c->stream), "population sync");
    return LBM_OK;
}

int lbm_set_step_count(lbm_ctx *c, int64_t step) {
    int rc = ctx_check(c);
    if (rc) return rc;
    if (step < 0) return fail(LBM_EINVAL, "step must be >= 0");
    if ((step & 1) != (c->step & 1)) {
        // the AA layout depends on the step parity: move the canonical state across
        void *tmp = nullptr;
        const size_t bytes = sizeof(double) * c->Q * c->ncell;
        if ((rc = ctx_stage(c, 0, bytes, &tmp))) return ctx_sticky(c, rc);
        cudaError_t e = get_populations(c->lat, c->rho0, (int)(c->step & 1), tmp, LBM_DT_F64, c->stream);
        if (e == cudaSuccess) e = set_populations(c->lat, c->rho0, (int)(step & 1), tmp, LBM_DT_F64, c->stream);
        if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("re-layout", e));
    }
    c->step = step;
    drop_graph(c);
    return LBM_OK;
}

int lbm_sample_populations(lbm_ctx *c, const int64_t *cells, int64_t count, double *out) {
    int rc = ctx_check(c);
    if (rc) return rc;
    if (count < 0 || (count > 0 && (!cells || !out))) return fail(LBM_EINVAL, "bad sample arguments");
    if (count == 0) return LBM_OK;
    for (int64_t k = 0; k < count; ++k)
        if (cells[k] < 0 || cells[k] >= c->ncell) return fail(LBM_EINVAL, "cell index %lld out of range", (long long)cells[k]);
    DevBuf dc, dout;
    if ((rc = stage_in(cells, sizeof(int64_t) * count, 0, c->stream, dc))) return ctx_sticky(c, rc);
    if (cudaMalloc(&dout.p, sizeof(double) * c->Q * count) != cudaSuccess) {
        cudaGetLastError();
        return fail(LBM_ENOMEM, "sample staging");
    }
    dout.owned = true;
    cudaError_t e = sample_populations(c->lat, c->rho0, (int)(c->step & 1), (const int64_t *)dc.p, count,
                                       (double *)dout.p, c->stream);
    if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("sample kernel", e));
    CK(cudaMemcpyAsync(out, dout.p, sizeof(double) * c->Q * count, cudaMemcpyDeviceToHost, c->stream), "sample copy");
    CK(cudaStreamSynchronize(c->stream), "sample sync");
    return read_status(c);
}

int lbm_step_count(lbm_ctx *c, int64_t *out) {
    if (!c || !out) return fail(LBM_EINVAL, "null argument");
    *out = c->step;
    return LBM_OK;
}

int lbm_launch_info(lbm_ctx *c, int64_t out[8]) {
    if (!c || !out) return fail(LBM_EINVAL, "null argument");
    out[0] = c->kernel;
    if (c->kernel == 2) {
        out[1] = c->tma.threads;
        out[2] = c->tma.blocks;
        out[3] = c->tma.stages;
        out[4] = c->tma.rows;
        out[5] = c->tma.seg;
        out[6] = c->tma.smem_bytes;
    } else {
        out[1] = c->gen_threads;
        out[2] = c->gen_blocks;
        out[3] = out[4] = out[5] = out[6] = 0;
    }
    out[7] = (int64_t)c->Q * c->lat.plane * esize_of(c->prec);
    return LBM_OK;
}

int lbm_set_launch_shape(lbm_ctx *c, const int64_t shape[6]) {
    int rc = ctx_check(c);
    if (rc) return rc;
    if (!shape) return fail(LBM_EINVAL, "null shape");
    for (int q = 0; q < 6; ++q)
        if (shape[q] < 0 || shape[q] > INT32_MAX) return fail(LBM_EINVAL, "shape[%d] = %lld out of range", q, (long long)shape[q]);
    if (shape[0] == 1) {
        if (shape[1] < 32 || shape[1] > 256 || shape[1] % 32)
            return fail(LBM_EINVAL, "threads must be a multiple of 32 in [32, 256] for the one-cell kernel");
        c->kernel = 1;
        c->chosen = true;
        c->gen_threads = (int)shape[1];
        c->gen_blocks = (int)std::max<int64_t>(1, std::min<int64_t>((c->ncell + shape[1] - 1) / shape[1],
                                                                    (int64_t)sm_count() * 16));
        drop_graph(c);
        return LBM_OK;
    }
    if (shape[0] != 2) return fail(LBM_EINVAL, "kernel must be 1 or 2");
    // (padded rows too, whole: a shape that lbm_launch_info reports can be set on a lattice of its size)
    if (!tma_supported(c->lat)) return fail(LBM_EINVAL, "TMA row kernel needs Nx * sizeof(storage) %% 16 == 0, or padded rows");
    const int tmax = tma_thread_limit(c->lat);
    if (shape[1] < 32 || shape[1] > tmax || shape[1] % 32)
        return fail(LBM_EINVAL, "threads must be a multiple of 32 in [32, %d] for this lattice and storage", tmax);
    const int U = 16 / esize_of(c->prec);
    if (shape[4] < U) return fail(LBM_EINVAL, "seg must be at least %d cells (16 bytes)", U);
    TmaShape t{};
    t.threads = (int)shape[1];
    t.stages = (int)shape[2];
    t.rows = (int)std::max<int64_t>(1, shape[3]);
    t.seg = (int)std::min<int64_t>(shape[4], c->lat.nx);
    t.cap = (int)shape[5];
    t.smem_bytes = tma_smem_bytes(c->lat, t);
    if (t.smem_bytes < 0) return fail(LBM_EINVAL, "launch shape does not fit (segment, rows, cap or stages)");
    if (!tma_set_blocks(c->lat, c->eq, c->bulk, sm_count(), t)) return fail(LBM_EINVAL, "launch shape does not fit on the device");
    c->tma = c->tma_one = t;
    c->kernel = 2;
    c->chosen = true;
    drop_graph(c);
    return LBM_OK;
}

int lbm_sync(lbm_ctx *c) {
    int rc = ctx_check(c);
    if (rc) return rc;
    cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return ctx_sticky(c, cuda_fail("sync", e));
    return read_status(c);
}

void lbm_destroy(lbm_ctx *c) {
    if (!c) return;
    cudaStreamSynchronize(c->stream);
    drop_graph(c);
    cudaFree(c->lat.A);
    cudaFree(c->status);  // the start of the small buffers' allocation
    cudaFree(c->stage[0]);
    cudaFree(c->stage[1]);
    cudaGetLastError();
    delete c;
}

// ------------------------------------------------------------------- von Neumann analysis

namespace {
// Device buffer of one von Neumann call (one allocation: a call on a few thousand points takes
// about as long as three cudaMalloc and cudaFree pairs), freed on every return path.
struct VnBuf {
    char *p = nullptr;
    ~VnBuf() {
        if (p) cudaFree(p);
    }
    bool alloc(size_t bytes) {
        if (cudaMalloc(&p, bytes) != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
            return false;
        }
        return true;
    }
};
}  // namespace

int lbm_vn_eigenvalues(int eq_kind, int bulk_corr, int64_t count, const double *params, double *out,
                       void *cuda_stream) {
    if (eq_kind < 0 || eq_kind > 2 || (bulk_corr != 0 && bulk_corr != 1) || count < 0 ||
        (count > 0 && (!params || !out)))
        return fail(LBM_EINVAL, "bad von Neumann arguments");
    if (count == 0) return LBM_OK;
    for (int64_t p = 0; p < count; ++p)
        if (!(params[6 * p] > 0.5) || !(params[6 * p + 1] > 0))
            return fail(LBM_EINVAL, "point %lld: tau must be > 1/2 and rho > 0", (long long)p);
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    VnBuf b;
    const size_t in = sizeof(double) * 6 * count, res = sizeof(double) * 18 * count;
    if (!b.alloc(in + res + sizeof(int32_t))) return fail(LBM_ENOMEM, "von Neumann buffers");
    double *dp = (double *)b.p, *dout = (double *)(b.p + in);
    int32_t *dst = (int32_t *)(b.p + in + res);
    CK(cudaMemcpyAsync(dp, params, in, cudaMemcpyHostToDevice, s), "params upload");
    CK(cudaMemsetAsync(dst, 0, sizeof(int32_t), s), "status clear");
    CK(vn_eigs(eq_kind, bulk_corr, count, dp, dout, dst, s), "eigenvalue kernel");
    int32_t st = 0;
    CK(cudaMemcpyAsync(out, dout, res, cudaMemcpyDeviceToHost, s), "eigenvalue copy");
    CK(cudaMemcpyAsync(&st, dst, sizeof(int32_t), cudaMemcpyDeviceToHost, s), "status copy");
    CK(cudaStreamSynchronize(s), "eigenvalue sync");
    if (st) return fail(LBM_ECUDA, "the QR iteration did not converge for some point");
    return LBM_OK;
}

int lbm_vn_stability_limit(int eq_kind, int64_t npairs, const double *nu, const double *theta, int nk,
                           double u_hi, int iterations, double tol, double *umax, void *cuda_stream) {
    if (eq_kind < 0 || eq_kind > 2 || npairs < 0 || (npairs > 0 && (!nu || !theta || !umax)) || nk < 1 ||
        nk > 1024 || !(u_hi > 0) || u_hi >= 1.0 || iterations < 1 || iterations > 60 || !(tol >= 0))
        return fail(LBM_EINVAL, "bad stability-limit arguments");
    if (npairs == 0) return LBM_OK;
    for (int64_t p = 0; p < npairs; ++p)
        if (!(nu[p] > 0)) return fail(LBM_EINVAL, "nu must be positive");
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const size_t state = vn_limit_bytes(npairs), col = sizeof(double) * (size_t)npairs;
    std::unique_ptr<double[]> host(new (std::nothrow) double[2 * (size_t)npairs]);
    VnBuf b;
    if (!host || !b.alloc(state + 3 * col + sizeof(int32_t))) return fail(LBM_ENOMEM, "stability buffers");
    for (int64_t p = 0; p < npairs; ++p) {
        host[2 * p] = 0.5 + 3.0 * nu[p];
        host[2 * p + 1] = theta[p];
    }
    double *din = (double *)(b.p + state), *dlim = (double *)(b.p + state + 2 * col);
    int32_t *dst = (int32_t *)(b.p + state + 3 * col);
    CK(cudaMemcpyAsync(din, host.get(), 2 * col, cudaMemcpyHostToDevice, s), "pair upload");
    CK(cudaMemsetAsync(dst, 0, sizeof(int32_t), s), "status clear");
    CK(vn_limit(eq_kind, npairs, b.p, din, dlim, nk, u_hi, iterations, tol, dst, s), "stability search");
    int32_t st = 0;
    CK(cudaMemcpyAsync(&st, dst, sizeof(int32_t), cudaMemcpyDeviceToHost, s), "status copy");
    CK(cudaStreamSynchronize(s), "stability sync");
    if (st) return fail(LBM_ECUDA, "the QR iteration did not converge for some point");
    CK(cudaMemcpy(umax, dlim, col, cudaMemcpyDeviceToHost), "limit copy");
    return LBM_OK;
}

int lbm_selftest_bounded_wait(void *cuda_stream, int64_t timeout_ns, int32_t *status_out) {
    if (!status_out || timeout_ns <= 0 || timeout_ns > 10000000000LL)
        return fail(LBM_EINVAL, "bad self-test arguments");
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    int32_t *d = nullptr;
    CK(cudaMalloc(&d, sizeof(int32_t)), "self-test buffer");
    cudaError_t e = cudaMemsetAsync(d, 0x7f, sizeof(int32_t), s);
    if (e == cudaSuccess) e = selftest_wait(timeout_ns, d, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(status_out, d, sizeof(int32_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d);
    if (e != cudaSuccess) return cuda_fail("self-test", e);
    return LBM_OK;
}

// ------------------------------------------------------------------------------ batch

static int batch_check(lbm_batch *b) {
    if (!b) return fail(LBM_EINVAL, "null batch");
    if (b->sticky) return fail(LBM_ESTATE, "batch is in an error state (%d); destroy it", b->sticky);
    return LBM_OK;
}

static int batch_sticky(lbm_batch *b, int code) {
    if (code == LBM_ECUDA || code == LBM_ETIMEOUT || code == LBM_ENOMEM) b->sticky = code;
    return code;
}

// Largest block count of the batched kernel: 32 blocks per SM, at most one per instance.
static int batch_block_cap(int64_t count) { return (int)std::min<int64_t>(count, (int64_t)sm_count() * 32); }

// Greedy longest-first assignment of whole instances to nb blocks (each instance goes to
// the block with the least load so far); uploads the per-block instance lists.
static cudaError_t batch_assign(lbm_batch *b, int nb) {
    const std::vector<int64_t> &cs = b->cell_start;
    const int64_t count = b->count;
    std::vector<int32_t> idx(count);
    for (int64_t k = 0; k < count; ++k) idx[k] = (int32_t)k;
    std::sort(idx.begin(), idx.end(), [&](int32_t a, int32_t c) {
        const int64_t na = cs[a + 1] - cs[a], nc = cs[c + 1] - cs[c];
        return na != nc ? na > nc : a < c;
    });
    using Item = std::pair<int64_t, int>;
    std::priority_queue<Item, std::vector<Item>, std::greater<Item>> heap;
    for (int q = 0; q < nb; ++q) heap.push({0, q});
    std::vector<std::vector<int32_t>> own(nb);
    for (int32_t k : idx) {
        Item it = heap.top();
        heap.pop();
        own[it.second].push_back(k);
        it.first += cs[k + 1] - cs[k];
        heap.push(it);
    }
    std::vector<int32_t> order;
    order.reserve(count);
    std::vector<int32_t> bstart(nb + 1, 0);
    int64_t maxload = 0;
    for (int q = 0; q < nb; ++q) {
        int64_t load = 0;
        for (int32_t k : own[q]) {
            order.push_back(k);
            load += cs[k + 1] - cs[k];
        }
        maxload = std::max(maxload, load);
        bstart[q + 1] = (int32_t)order.size();
    }
    cudaError_t e = cudaMemcpyAsync(b->d_order, order.data(), sizeof(int32_t) * count, cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_block_start, bstart.data(), sizeof(int32_t) * (nb + 1), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);  // the host vectors go out of scope
    if (e != cudaSuccess) return e;
    b->blocks = nb;
    b->max_load = maxload;
    b->mean_load = b->total / nb;
    return cudaSuccess;
}

// Plans teams of blocks where the largest instance alone would keep an SM busy longer than its
// share of all cells.  Sets team_blocks (0: no teams) and uploads the tables.  The smallest number
// of cells a block for which all blocks are resident: 608 blocks of 128 threads for D2Q9, so every
// SM's FP64 pipe has several warps.  30 lattices of
// 16^2 .. 96^2: 185 -> 17 us a step, 60 of 16^2 .. 256^2: 1225 -> 100 us.
// Small instances that have an SM to every block take clusters of three-lane cells, whatever the
// shares: 36 lines of 128 cells 4.1 -> 2.4 us a step, 76 of 64 3.7 -> 2.5.  With more blocks than
// SMs nothing is left of it: 38 lines of 128 cells, whose clusters no longer all find a place of
// their own, 4.1 -> 3.8 us.
static cudaError_t batch_plan_teams(lbm_batch *b) {
    b->team_blocks = 0;
    b->team_max = 0;
    const std::vector<int64_t> &cs = b->cell_start;
    int64_t largest = 0;
    for (int64_t k = 0; k < b->count; ++k) largest = std::max(largest, cs[k + 1] - cs[k]);
    const int sms = sm_count();
    const int64_t cluster = (largest + kClusterCells - 1) / kClusterCells;
    if (cluster <= kClusterBlocks && b->count * cluster <= sms &&
        batch_cluster_capacity(b->D, b->eq, b->bulk, (int)cluster) >= b->count) {
        b->team_cluster = (int)cluster;
        b->team_blocks = (int)(b->count * cluster);
        b->team_max = std::min<int64_t>(largest, kClusterCells);
        return cudaSuccess;
    }
    if (largest * sms * 10 <= b->total * 11 || largest * b->Q >= ((int64_t)1 << 31)) return cudaSuccess;
    const int cap = team_block_capacity(b->D, b->eq, b->bulk, sms);
    if (b->count > cap) return cudaSuccess;
    auto blocks_for = [&](int64_t per) {
        int64_t n = 0;
        for (int64_t k = 0; k < b->count; ++k) n += (cs[k + 1] - cs[k] + per - 1) / per;
        return n;
    };
    int64_t lo = 1, hi = (largest + kTeamThreads - 1) / kTeamThreads;  // cells a block / threads
    while (lo < hi) {
        const int64_t mid = (lo + hi) / 2;
        if (blocks_for(mid * kTeamThreads) <= cap) hi = mid;
        else lo = mid + 1;
    }
    const int64_t per = lo * kTeamThreads;
    std::vector<int32_t> inst, part, size(b->count);
    for (int64_t k = 0; k < b->count; ++k) {
        const int64_t n = cs[k + 1] - cs[k];
        size[k] = (int32_t)((n + per - 1) / per);
        for (int32_t q = 0; q < size[k]; ++q) {
            inst.push_back((int32_t)k);
            part.push_back(q);
        }
        b->team_max = std::max(b->team_max, (n + size[k] - 1) / size[k]);
    }
    // the busiest SM with teams (its blocks at most) against the busiest one without (the largest
    // instance): 600 lattices of 16^2 .. 160^2 have a block each and little to share out
    const int64_t nbl = (int64_t)inst.size();
    if ((nbl + sms - 1) / sms * b->team_max * 10 > std::max(largest, b->total / sms) * 11) return cudaSuccess;
    const size_t nb = inst.size();
    auto pad = [](size_t n) { return (n + 255) / 256 * 256; };
    const size_t sync = pad(sizeof(unsigned) * kBarStride * (b->count + 1)), sums = pad(sizeof(double) * 16 * nb);
    const size_t table = pad(sizeof(int32_t) * nb), sizes = pad(sizeof(int32_t) * b->count);
    if (cudaMalloc(&b->d_team, 256 + sync + sums + 2 * table + sizes) != cudaSuccess) {
        cudaGetLastError();
        return cudaSuccess;  // no room: whole instances per block
    }
    char *p = b->d_team;
    b->team_status = (int32_t *)p;
    b->team_sync = (unsigned *)(p += 256);
    b->team_partials = (double *)(p += sync);
    b->team_instance = (int32_t *)(p += sums);
    b->team_part = (int32_t *)(p += table);
    b->team_size = (int32_t *)(p += table);
    cudaError_t e = cudaMemset(b->d_team, 0, 256 + sync);
    if (e == cudaSuccess) e = cudaMemcpy(b->team_instance, inst.data(), sizeof(int32_t) * nb, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(b->team_part, part.data(), sizeof(int32_t) * nb, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(b->team_size, size.data(), sizeof(int32_t) * b->count, cudaMemcpyHostToDevice);
    b->team_blocks = (int)nb;
    return e;
}

static void batch_use_teams(lbm_batch *b) {
    b->teams = true;
    b->threads = kTeamThreads;
    b->blocks = b->team_blocks;
    b->max_load = b->team_max;
    b->mean_load = b->total / b->team_blocks;
}

// LBM_ETIMEOUT if a team's bounded wait ran out (the stream is idle), whatever launch shape the batch has
// been given since.
static int batch_team_status(lbm_batch *b) {
    if (!b->team_status) return LBM_OK;  // (no teams, or clusters, whose barrier is the hardware's)
    int32_t st = 0;
    CK(cudaMemcpy(&st, b->team_status, sizeof st, cudaMemcpyDeviceToHost), "status read");
    if (st != 0) return batch_sticky(b, fail(LBM_ETIMEOUT, "a bounded device wait ran out (status %d)", st));
    return LBM_OK;
}

int lbm_batch_create(lbm_batch **out, int lattice, int64_t count, const int32_t *dims,
                     const double *tau, int eq_kind, int bulk_corr, int precision, double rho0,
                     void *cuda_stream) {
    if (!out || !dims || !tau) return fail(LBM_EINVAL, "null argument");
    *out = nullptr;
    if (lattice != LBM_D2Q9 && lattice != LBM_D3Q27) return fail(LBM_EINVAL, "bad lattice %d", lattice);
    if (count < 1 || count > (1 << 24)) return fail(LBM_EINVAL, "count out of range");
    if (eq_kind < 0 || eq_kind > 2) return fail(LBM_EINVAL, "bad eq_kind %d", eq_kind);
    if (bulk_corr != 0 && bulk_corr != 1) return fail(LBM_EINVAL, "bulk_corr must be 0 or 1");
    if (precision != LBM_F64) return fail(LBM_EINVAL, "the batched path stores FP64 (precision must be LBM_F64)");
    if (!(rho0 > 0) || !std::isfinite(rho0)) return fail(LBM_EINVAL, "rho0 must be positive");
    const int D = lattice == LBM_D2Q9 ? 2 : 3;
    std::vector<int64_t> cs(count + 1, 0);
    for (int64_t k = 0; k < count; ++k) {
        for (int a = 0; a < 3; ++a)
            if (dims[3 * k + a] < 1 || dims[3 * k + a] > 65536) return fail(LBM_EINVAL, "instance %lld: bad dims", (long long)k);
        if (D == 2 && dims[3 * k + 2] != 1) return fail(LBM_EINVAL, "instance %lld: D2Q9 needs Nz == 1", (long long)k);
        if (!(tau[k] > 0.5) || !std::isfinite(tau[k])) return fail(LBM_EINVAL, "instance %lld: tau must be > 1/2", (long long)k);
        cs[k + 1] = cs[k] + (int64_t)dims[3 * k] * dims[3 * k + 1] * dims[3 * k + 2];
    }
    lbm_batch *b = new lbm_batch();
    b->lattice = lattice;
    b->D = D;
    b->Q = D == 2 ? 9 : 27;
    b->eq = eq_kind;
    b->bulk = bulk_corr;
    b->count = count;
    b->total = cs[count];
    b->rho0 = rho0;
    b->stream = static_cast<cudaStream_t>(cuda_stream);
    b->dims.assign(dims, dims + 3 * count);
    b->cell_start = cs;
    std::vector<double> om(count), sn(count);
    for (int64_t k = 0; k < count; ++k) {
        om[k] = 1.0 / tau[k];
        sn[k] = six_nu_of(tau[k]);
    }
    b->block_cap = batch_block_cap(count);
    b->threads = 256;
    const size_t arena_bytes = sizeof(double) * (size_t)b->Q * b->total;
    bool ok = cudaMalloc(&b->arena, arena_bytes) == cudaSuccess &&
              cudaMalloc(&b->d_cell_start, sizeof(int64_t) * (count + 1)) == cudaSuccess &&
              cudaMalloc(&b->d_dims, sizeof(int32_t) * 3 * count) == cudaSuccess &&
              cudaMalloc(&b->d_omega, sizeof(double) * count) == cudaSuccess &&
              cudaMalloc(&b->d_sixnu, sizeof(double) * count) == cudaSuccess &&
              cudaMalloc(&b->d_order, sizeof(int32_t) * count) == cudaSuccess &&
              cudaMalloc(&b->d_block_start, sizeof(int32_t) * (b->block_cap + 1)) == cudaSuccess &&
              cudaMalloc(&b->d_status, sizeof(int32_t) * count) == cudaSuccess &&
              cudaMalloc(&b->d_tw_off, sizeof(int64_t) * count) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        lbm_batch_destroy(b);
        return fail(LBM_ENOMEM, "batch storage of %zu bytes", arena_bytes);
    }
    cudaError_t e = cudaSuccess;
    auto up = [&](void *d, const void *h, size_t n) {
        if (e == cudaSuccess) e = cudaMemcpy(d, h, n, cudaMemcpyHostToDevice);
    };
    up(b->d_cell_start, cs.data(), sizeof(int64_t) * (count + 1));
    up(b->d_dims, dims, sizeof(int32_t) * 3 * count);
    up(b->d_omega, om.data(), sizeof(double) * count);
    up(b->d_sixnu, sn.data(), sizeof(double) * count);
    if (e == cudaSuccess) e = batch_plan_teams(b);
    if (e == cudaSuccess) {
        if (b->team_blocks > 0) batch_use_teams(b);
        else e = batch_assign(b, (int)std::min<int64_t>(count, (int64_t)sm_count() * 2));
    }
    if (e == cudaSuccess) e = cudaMemset(b->arena, 0, arena_bytes);
    if (e == cudaSuccess) e = cudaMemset(b->d_status, 0, sizeof(int32_t) * count);
    if (e != cudaSuccess) {
        lbm_batch_destroy(b);
        return cuda_fail("batch upload", e);
    }
    *out = b;
    return LBM_OK;
}

int lbm_batch_init_fields(lbm_batch *b, const void *rho, const void *u, int dtype, int on_device) {
    int rc = batch_check(b);
    if (rc) return rc;
    if (!rho || !u || !valid_dtype(dtype)) return fail(LBM_EINVAL, "bad field arguments");
    const size_t es = dtype == LBM_DT_F64 ? 8 : 4;
    DevBuf dr, du;
    void *mr = on_device ? nullptr : mapped_host(rho), *mu = on_device ? nullptr : mapped_host(u);
    if (mr && mu) {  // page-locked fields: the kernel reads them across the link
        dr.p = mr;
        du.p = mu;
    } else {
        if ((rc = stage_in(rho, es * b->total, on_device, b->stream, dr))) return batch_sticky(b, rc);
        if ((rc = stage_in(u, es * b->total * b->D, on_device, b->stream, du))) return batch_sticky(b, rc);
    }
    cudaError_t e = batch_init(b->arena, b->d_cell_start, b->d_dims, b->count, b->D, b->eq, b->rho0, dr.p, du.p,
                               dtype, b->total, b->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->d_status, 0, sizeof(int32_t) * b->count, b->stream);
    if (e == cudaSuccess && !on_device) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return batch_sticky(b, cuda_fail("batch init", e));
    b->step = 0;
    return LBM_OK;
}

int lbm_batch_set_probe(lbm_batch *b, const int32_t *kvec, int64_t every_k) {
    int rc = batch_check(b);
    if (rc) return rc;
    if (!kvec || every_k < 1) return fail(LBM_EINVAL, "bad probe arguments");
    std::vector<double2> tw;
    std::vector<int64_t> off(b->count);
    const double twopi = 6.283185307179586476925286766559;
    for (int64_t k = 0; k < b->count; ++k) {
        off[k] = (int64_t)tw.size();
        for (int a = 0; a < 3; ++a) {
            const int n = b->dims[3 * k + a];
            const int64_t m = kvec[3 * k + a];
            for (int x = 0; x < n; ++x) {
                const int64_t q = ((m * x) % n + n) % n;  // exact phase index
                const double ph = twopi * (double)q / (double)n;
                tw.push_back(make_double2(cos(ph), -sin(ph)));
            }
        }
    }
    if (b->d_tw) cudaFree(b->d_tw);
    b->d_tw = nullptr;
    if (cudaMalloc(&b->d_tw, sizeof(double2) * tw.size()) != cudaSuccess) {
        cudaGetLastError();
        return fail(LBM_ENOMEM, "probe twiddles");
    }
    CK(cudaMemcpy(b->d_tw, tw.data(), sizeof(double2) * tw.size(), cudaMemcpyHostToDevice), "twiddle upload");
    CK(cudaMemcpy(b->d_tw_off, off.data(), sizeof(int64_t) * b->count, cudaMemcpyHostToDevice), "twiddle offsets");
    b->every_k = every_k;
    return LBM_OK;
}

static int batch_reserve_series(lbm_batch *b, int64_t samples) {
    if (samples <= b->max_samples) return LBM_OK;
    int64_t cap = std::max<int64_t>(samples, 2 * b->max_samples);
    double *d = nullptr;
    const size_t bytes = sizeof(double) * 8 * (size_t)b->count * cap;
    if (cudaMalloc(&d, bytes) != cudaSuccess) {
        cudaGetLastError();
        return fail(LBM_ENOMEM, "probe series of %zu bytes", bytes);
    }
    CK(cudaMemsetAsync(d, 0, bytes, b->stream), "series clear");
    if (b->d_series && b->max_samples > 0) {
        CK(cudaMemcpy2DAsync(d, sizeof(double) * 8 * cap, b->d_series, sizeof(double) * 8 * b->max_samples,
                             sizeof(double) * 8 * b->max_samples, b->count, cudaMemcpyDeviceToDevice, b->stream),
           "series grow");
    }
    CK(cudaStreamSynchronize(b->stream), "series sync");
    cudaFree(b->d_series);
    b->d_series = d;
    b->max_samples = cap;
    return LBM_OK;
}

static BatchArgs batch_args(lbm_batch *b, int64_t n) {
    BatchArgs a;
    a.arena = b->arena;
    a.cell_start = b->d_cell_start;
    a.dims = b->d_dims;
    a.omega0 = b->d_omega;
    a.six_nu = b->d_sixnu;
    a.order = b->d_order;
    a.block_start = b->d_block_start;
    a.twiddle = b->d_tw;
    a.tw_offset = b->d_tw_off;
    a.series = b->d_series;
    a.max_samples = b->max_samples;
    a.status = b->d_status;
    a.count = b->count;
    a.D = b->D;
    a.eq = b->eq;
    a.bulk = b->bulk;
    a.rho0 = b->rho0;
    a.step0 = b->step;
    a.nsteps = n;
    a.every_k = b->d_tw ? b->every_k : 0;
    a.team_instance = b->team_instance;
    a.team_part = b->team_part;
    a.team_size = b->team_size;
    a.team_partials = b->team_partials;
    a.team_sync = b->team_sync;
    a.team_status = b->team_status;
    a.team_cluster = b->team_cluster;
    a.timeout_ns = wait_timeout_ns();
    return a;
}

static cudaError_t batch_launch(lbm_batch *b, const BatchArgs &a, cudaStream_t s) {
    return b->teams ? step_teams(a, b->blocks, s) : step_batch(a, b->blocks, b->threads, s);
}

int lbm_batch_step(lbm_batch *b, int64_t n) {
    NvtxRange range("lbm_batch_step");
    int rc = batch_check(b);
    if (rc) return rc;
    if (n < 0) return fail(LBM_EINVAL, "n must be >= 0");
    if (n == 0) return LBM_OK;
    if (b->every_k > 0) {
        const int64_t last = b->step + n - 1;
        if ((rc = batch_reserve_series(b, last / b->every_k + 1))) return batch_sticky(b, rc);
    }
    for (int64_t left = n; left > 0;) {
        // one persistent launch (of teams: of a bounded number of steps), captured into a graph and
        // replayed on the object's stream
        const int64_t m = b->teams && b->team_cluster == 0 ? team_launch_steps(left) : left;
        const BatchArgs a = batch_args(b, m);
        cudaStream_t cap;
        CK(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "batch capture stream");
        cudaGraph_t g = nullptr;
        cudaGraphExec_t ge = nullptr;
        cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            cudaError_t el = batch_launch(b, a, cap);
            e = cudaStreamEndCapture(cap, &g);
            if (e == cudaSuccess && el != cudaSuccess) e = el;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&ge, g, 0);
        if (e == cudaSuccess) e = cudaGraphLaunch(ge, b->stream);
        if (ge) cudaGraphExecDestroy(ge);
        if (g) cudaGraphDestroy(g);
        cudaStreamDestroy(cap);
        if (e != cudaSuccess) return batch_sticky(b, cuda_fail("batch launch", e));
        b->step += m;
        left -= m;
    }
    return LBM_OK;
}

int lbm_batch_probe_series(lbm_batch *b, double *out, int64_t max_samples, int64_t *nsamples) {
    int rc = batch_check(b);
    if (rc) return rc;
    if (!nsamples || max_samples < 0) return fail(LBM_EINVAL, "bad series arguments");
    const int64_t have = b->every_k > 0 ? std::min<int64_t>((b->step + b->every_k - 1) / b->every_k, b->max_samples) : 0;
    *nsamples = have;
    if (!out || have == 0) return LBM_OK;
    const int64_t take = std::min(have, max_samples);
    CK(cudaStreamSynchronize(b->stream), "series sync");
    if ((rc = batch_team_status(b))) return rc;
    CK(cudaMemcpy2D(out, sizeof(double) * 8 * max_samples, b->d_series, sizeof(double) * 8 * b->max_samples,
                    sizeof(double) * 8 * take, b->count, cudaMemcpyDeviceToHost),
       "series copy");
    return LBM_OK;
}

int lbm_batch_status(lbm_batch *b, int32_t *status) {
    int rc = batch_check(b);
    if (rc) return rc;
    if (!status) return fail(LBM_EINVAL, "null output");
    CK(cudaMemcpyAsync(status, b->d_status, sizeof(int32_t) * b->count, cudaMemcpyDeviceToHost, b->stream), "status copy");
    CK(cudaStreamSynchronize(b->stream), "status sync");
    return batch_team_status(b);
}

int lbm_batch_moments(lbm_batch *b, void *rho, void *u, int dtype, int on_device) {
    int rc = batch_check(b);
    if (rc) return rc;
    if (!rho || !u || !valid_dtype(dtype)) return fail(LBM_EINVAL, "bad field arguments");
    const size_t es = dtype == LBM_DT_F64 ? 8 : 4;
    void *dr = rho, *du = u;
    DevBuf br, bu;
    void *mr = on_device ? nullptr : mapped_host(rho), *mu = on_device ? nullptr : mapped_host(u);
    const bool direct = mr && mu;  // page-locked outputs: the kernel writes them across the link
    if (direct) {
        dr = mr;
        du = mu;
    } else if (!on_device) {
        if (cudaMalloc(&br.p, es * b->total) != cudaSuccess || cudaMalloc(&bu.p, es * b->total * b->D) != cudaSuccess) {
            cudaGetLastError();
            return fail(LBM_ENOMEM, "moments staging");
        }
        br.owned = bu.owned = true;
        dr = br.p;
        du = bu.p;
    }
    cudaError_t e = batch_moments(b->arena, b->d_cell_start, b->d_dims, b->count, b->D, b->rho0, (int)(b->step & 1),
                                  dr, du, dtype, b->total, b->stream);
    if (e != cudaSuccess) return batch_sticky(b, cuda_fail("batch moments", e));
    if (!on_device) {
        if (!direct) {
            CK(cudaMemcpyAsync(rho, dr, es * b->total, cudaMemcpyDeviceToHost, b->stream), "moments copy");
            CK(cudaMemcpyAsync(u, du, es * b->total * b->D, cudaMemcpyDeviceToHost, b->stream), "moments copy");
        }
        CK(cudaStreamSynchronize(b->stream), "moments sync");
        return batch_team_status(b);
    }
    return LBM_OK;
}

int lbm_batch_get_populations(lbm_batch *b, void *f, int dtype, int on_device) {
    int rc = batch_check(b);
    if (rc) return rc;
    if (!f || !valid_dtype(dtype)) return fail(LBM_EINVAL, "bad population arguments");
    const size_t bytes = (size_t)(dtype == LBM_DT_F64 ? 8 : 4) * b->Q * b->total;
    void *d = f;
    DevBuf buf;
    if (!on_device) {
        if (cudaMalloc(&buf.p, bytes) != cudaSuccess) {
            cudaGetLastError();
            return fail(LBM_ENOMEM, "population staging");
        }
        buf.owned = true;
        d = buf.p;
    }
    cudaError_t e = batch_populations(b->arena, b->d_cell_start, b->d_dims, b->count, b->D, b->rho0,
                                      (int)(b->step & 1), d, dtype, b->total, b->stream);
    if (e != cudaSuccess) return batch_sticky(b, cuda_fail("batch populations", e));
    if (!on_device) {
        CK(cudaMemcpyAsync(f, d, bytes, cudaMemcpyDeviceToHost, b->stream), "population copy");
        CK(cudaStreamSynchronize(b->stream), "population sync");
        return batch_team_status(b);
    }
    return LBM_OK;
}

int lbm_batch_info(lbm_batch *b, int64_t *total_cells, int64_t *step) {
    if (!b || !total_cells || !step) return fail(LBM_EINVAL, "null argument");
    *total_cells = b->total;
    *step = b->step;
    return LBM_OK;
}

int lbm_batch_launch_info(lbm_batch *b, int64_t out[4]) {
    if (!b || !out) return fail(LBM_EINVAL, "null argument");
    out[0] = b->threads;
    out[1] = b->teams ? b->count : b->blocks;  // a team counts once
    out[2] = b->max_load;
    out[3] = b->mean_load;
    return LBM_OK;
}

int lbm_batch_set_launch_shape(lbm_batch *b, int threads, int64_t blocks) {
    int rc = batch_check(b);
    if (rc) return rc;
    if (threads < 32 || threads > 256 || threads % 32) return fail(LBM_EINVAL, "threads must be a multiple of 32 in [32, 256]");
    if (blocks < 1 || blocks > b->block_cap)
        return fail(LBM_EINVAL, "blocks must be in [1, %d] (32 per SM, at most one per instance)", b->block_cap);
    cudaError_t e = batch_assign(b, (int)blocks);
    if (e != cudaSuccess) return batch_sticky(b, cuda_fail("batch assignment", e));
    b->teams = false;
    b->threads = threads;
    return LBM_OK;
}

// Buffers of one batch tuning call, freed on every return path.
struct BatchTuneBufs {
    void *arena = nullptr, *status = nullptr;
    ~BatchTuneBufs() {
        cudaFree(arena);
        cudaFree(status);
    }
};

int lbm_batch_autotune(lbm_batch *b, int64_t steps) {
    NvtxRange range("lbm_batch_autotune");
    int rc = batch_check(b);
    if (rc) return rc;
    if (steps < 1 || steps > 100000) return fail(LBM_EINVAL, "steps must be in [1, 100000]");
    if (b->every_k > 0) {
        // the probes of the timed steps are part of the work; they land in samples the
        // next lbm_batch_step rewrites (at or after the current step)
        if ((rc = batch_reserve_series(b, (b->step + steps - 1) / b->every_k + 1))) return batch_sticky(b, rc);
    }
    const size_t arena_bytes = sizeof(double) * (size_t)b->Q * b->total;
    BatchTuneBufs keep;
    if (cudaMalloc(&keep.arena, arena_bytes) != cudaSuccess || cudaMalloc(&keep.status, sizeof(int32_t) * b->count) != cudaSuccess) {
        cudaGetLastError();
        return fail(LBM_ENOMEM, "batch tuning needs one copy of the state (%zu bytes)", arena_bytes);
    }
    CK(cudaMemcpyAsync(keep.arena, b->arena, arena_bytes, cudaMemcpyDeviceToDevice, b->stream), "tuning backup");
    CK(cudaMemcpyAsync(keep.status, b->d_status, sizeof(int32_t) * b->count, cudaMemcpyDeviceToDevice, b->stream),
       "tuning backup");
    const int saved_threads = b->threads, saved_blocks = b->blocks;
    const bool saved_teams = b->teams;
    struct Cand {
        int threads, blocks;  // blocks 0: teams
        float ms;
    };
    std::vector<Cand> cands;
    if (b->team_blocks > 0) cands.push_back({kTeamThreads, 0, -1.f});
    auto use = [&](int threads, int blocks) -> cudaError_t {
        if (blocks == 0) {
            batch_use_teams(b);
            return cudaSuccess;
        }
        const cudaError_t ea = batch_assign(b, blocks);
        b->teams = false;
        b->threads = threads;
        return ea;
    };
    for (int th : {64, 128, 256})
        for (int r : {1, 2, 3, 4, 6, 8, 12, 16}) {
            const int nb = (int)std::min<int64_t>((int64_t)sm_count() * r, b->block_cap);
            bool dup = false;
            for (const Cand &q : cands) dup = dup || (q.threads == th && q.blocks == nb);
            if (!dup) cands.push_back({th, nb, -1.f});
        }
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0), "tuning events");
    cudaError_t e = cudaEventCreate(&e1);
    if (e != cudaSuccess) {
        cudaEventDestroy(e0);
        return cuda_fail("tuning events", e);
    }
    for (int round = 0; round < 2 && e == cudaSuccess; ++round)
        for (Cand &q : cands) {
            e = use(q.threads, q.blocks);
            if (e != cudaSuccess) break;
            const BatchArgs a = batch_args(b, steps);
            e = cudaEventRecord(e0, b->stream);
            if (e == cudaSuccess) e = batch_launch(b, a, b->stream);
            if (e == cudaSuccess) e = cudaEventRecord(e1, b->stream);
            if (e == cudaSuccess) e = cudaEventSynchronize(e1);
            float ms = -1;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            // every candidate starts from the same state
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(b->arena, keep.arena, arena_bytes, cudaMemcpyDeviceToDevice, b->stream);
            if (e == cudaSuccess && ms > 0) q.ms = q.ms < 0 ? ms : std::min(q.ms, ms);
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_status, keep.status, sizeof(int32_t) * b->count, cudaMemcpyDeviceToDevice, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return batch_sticky(b, cuda_fail("batch tuning", e));
    // the fastest, or among those within 0.5 % of it the one with the fewest blocks, then
    // the fewest threads (equally fast boxes pick the same shape)
    const Cand *best = nullptr;
    for (const Cand &q : cands)
        if (q.ms > 0 && (!best || q.ms < best->ms)) best = &q;
    if (!best) {
        e = use(saved_threads, saved_teams ? 0 : saved_blocks);
        if (e != cudaSuccess) return batch_sticky(b, cuda_fail("batch assignment", e));
        return fail(LBM_ECUDA, "batch tuning found no runnable launch shape");
    }
    const float limit = best->ms * 1.005f;
    const Cand *pick = best;
    for (const Cand &q : cands)
        if (q.ms > 0 && q.ms <= limit &&
            (q.blocks < pick->blocks || (q.blocks == pick->blocks && q.threads < pick->threads)))
            pick = &q;
    e = use(pick->threads, pick->blocks);
    if (e != cudaSuccess) return batch_sticky(b, cuda_fail("batch assignment", e));
    return LBM_OK;
}

int lbm_batch_sync(lbm_batch *b) {
    int rc = batch_check(b);
    if (rc) return rc;
    CK(cudaStreamSynchronize(b->stream), "batch sync");
    return batch_team_status(b);
}

void lbm_batch_destroy(lbm_batch *b) {
    if (!b) return;
    cudaStreamSynchronize(b->stream);
    cudaFree(b->arena);
    cudaFree(b->d_cell_start);
    cudaFree(b->d_dims);
    cudaFree(b->d_omega);
    cudaFree(b->d_sixnu);
    cudaFree(b->d_order);
    cudaFree(b->d_block_start);
    cudaFree(b->d_tw);
    cudaFree(b->d_tw_off);
    cudaFree(b->d_series);
    cudaFree(b->d_status);
    cudaFree(b->d_team);
    cudaGetLastError();
    delete b;
}

}  // extern "C"
