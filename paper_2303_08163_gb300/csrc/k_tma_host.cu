// k_tma_host.cu -- geometry and launch of the TMA row-staged step kernel.
#include <algorithm>


#include "k_tma.cuh"

namespace lbmh {

#define LBM_DECL_CAP(d, c) const void *tma_kernel_d##d##_c##c(int P, int eq, int bulk, bool several);
LBM_DECL_CAP(2, 1024)
LBM_DECL_CAP(2, 2048)
LBM_DECL_CAP(2, 4096)
LBM_DECL_CAP(2, 8192)
LBM_DECL_CAP(3, 1024)
LBM_DECL_CAP(3, 2048)
LBM_DECL_CAP(3, 4096)
LBM_DECL_CAP(3, 8192)
#undef LBM_DECL_CAP

constexpr int kTmaMaxSmem = 227 * 1024;  // shared memory of a block, static and dynamic

static const void *tma_kernel(const Lattice &lat, int eq, int bulk, int cap, bool several) {
    if (lat.D == 2) {
        switch (cap) {
        case 1024: return tma_kernel_d2_c1024(lat.P, eq, bulk, several);
        case 2048: return tma_kernel_d2_c2048(lat.P, eq, bulk, several);
        case 4096: return tma_kernel_d2_c4096(lat.P, eq, bulk, several);
        case 8192: return tma_kernel_d2_c8192(lat.P, eq, bulk, several);
        }
    } else {
        switch (cap) {
        case 1024: return tma_kernel_d3_c1024(lat.P, eq, bulk, several);
        case 2048: return tma_kernel_d3_c2048(lat.P, eq, bulk, several);
        case 4096: return tma_kernel_d3_c4096(lat.P, eq, bulk, several);
        case 8192: return tma_kernel_d3_c8192(lat.P, eq, bulk, several);
        }
    }
    return nullptr;
}

static int esize(int P) { return P == lbmd::P_F64 ? 8 : (P == lbmd::P_F32 ? 4 : 2); }

bool tma_supported(const Lattice &lat) {
    const int es = esize(lat.P);
    if (((int64_t)lat.pitch * es) % 16 != 0 || (lat.plane * es) % 16 != 0 || lat.nx < 16 / es) return false;
    // padded rows are copied whole (a segment's halo would start off a 16-byte boundary)
    return lat.pitch == lat.nx || lat.pitch * es <= (lat.D == 3 ? 4096 : 8192);
}

// Rows of a ragged lattice (nx * sizeof % 16 != 0) are padded to whole 16-byte units when
// the TMA kernel can then copy them whole and the padding stays under an eighth of the row
// (rows of at least 128 bytes).  FP64 storage is bound by the FP64 pipe, not by how its rows
// are fetched, and keeps its rows unpadded.
int padded_pitch(int D, int P, int64_t nx) {
    const int es = esize(P);
    const int64_t rowb = nx * es, up = (rowb + 15) / 16 * 16;
    if (rowb % 16 == 0 || P == lbmd::P_F64 || rowb < 128 || up > (D == 3 ? 4096 : 8192)) return (int)nx;
    return (int)(up / es);
}

static lbmd::TmaGeom geom(const Lattice &lat, const TmaShape &t) {
    const int U = 16 / esize(lat.P);
    lbmd::TmaGeom g;
    g.stages = t.stages;
    g.seg = t.seg >= lat.nx ? lat.nx : t.seg;
    g.nseg = (lat.nx + g.seg - 1) / g.seg;
    g.rows = g.nseg > 1 ? 1 : (t.rows < 1 ? 1 : (t.rows > lat.ny ? lat.ny : t.rows));
    g.ygroups = (lat.ny + g.rows - 1) / g.rows;
    g.halo = g.nseg > 1 ? U : 0;
    g.rowstride = g.nseg > 1 ? g.seg + 2 * g.halo : lat.pitch;
    g.bufstride = t.cap / esize(lat.P);
    g.njobs = (int64_t)lat.nz * g.ygroups * g.nseg;
    g.nsteps = 1;
    g.npos = g.ncross = g.strips = g.stripw = g.pjobs = g.depth = g.lag = 0;
    g.by_nseg = g.by_ygroups = g.by_npos = g.by_strips = g.by_pjobs = g.by_depth = lbmd::FastDiv{1, 0, 0};
    return g;
}

// The sweep of a several-step launch (see decode_chain).  Returns false when the lattice has
// more units than counters.
//
// Depth: a state that stays in L2 between steps is swept one step after the other.  A larger
// one is swept `depth` steps at a time, cut into strips where needed, so that what lies between
// the first and the last of them fits in L2: the jobs in flight (every stage of every block and
// a ticket or two more) spread over depth x pjobs jobs a phase, and two positions for the neighbours.
static bool chain_geom(const Lattice &lat, const TmaShape &t, int nsteps, lbmd::TmaGeom &g) {
    constexpr int64_t kWindow = (int64_t)60 << 20;  // the travelling window of a state that does not stay in L2
    g.nsteps = nsteps;
    g.npos = lat.D == 3 ? lat.nz : g.ygroups;
    g.ncross = lat.D == 3 ? g.ygroups : 1;
    if ((int64_t)g.npos * g.ncross > sync_units(lat)) return false;
    g.strips = 1;
    g.stripw = g.ncross;
    g.pjobs = g.ncross * g.nseg;
    g.depth = 1;
    g.lag = 0;
    const int64_t state = (int64_t)lbmd::qof(lat.D) * lat.plane * esize(lat.P);
    // (112^3 binary16, 72 MiB: 74.9 GLUPS against 73.6 swept; 1600^2 FP32, 88 MiB: 121 against 143 swept)
    if (state <= kTmaResident || lat.P == lbmd::P_F64) return true;
    const int64_t unit = state / ((int64_t)g.npos * g.ncross);
    // (measured in GLUPS, 3-D / 2-D: with a job more in the lag 256^3 FP32 44.7 against 46.0 and 128^3
    // FP32 44.8 against 47.8, but 4096^2 binary16 205 against 200 and 2048^2 FP32 132 against 128;
    // four steps together 4096^2 FP32 142 against 139, in 3-D they change nothing)
    const int64_t inflight = (int64_t)t.blocks * (t.stages + (lat.D == 2 ? 2 : 1));
    for (int d = lat.D == 2 ? 4 : 3; d >= 2; --d)
        for (int k = 1; k <= 64; ++k) {
            const int h = (g.ncross + k - 1) / k, last = g.ncross - (k - 1) * h;
            if (k > 1 && (last < 1 || h < 8 * (d - 1))) break;
            const int wide = k == 1 ? h : std::max(h, last + 2 * (d - 1));
            const int64_t pj = (int64_t)wide * g.nseg;
            const int64_t lag = 2 + (inflight + d * pj - 1) / (d * pj);
            if ((lag * (d - 1) + 3) * wide * unit > kWindow) continue;
            if (lag * (d - 1) + 2 >= g.npos) continue;
            g.depth = d;
            g.strips = k;
            g.stripw = h;
            g.pjobs = (int)pj;
            g.lag = (int)lag;
            return true;
        }
    return true;
}

int64_t sync_units(const Lattice &lat) {
    return std::min<int64_t>((int64_t)lat.ny * lat.nz, (int64_t)1 << 22);
}

int64_t tma_max_steps(const Lattice &lat, const TmaShape &t) {
    lbmd::TmaGeom g = geom(lat, t);
    if (!chain_geom(lat, t, 2, g)) return 1;
    // tickets stay below 2^30, and a launch to some tens of milliseconds
    const int64_t work = lat.P == lbmd::P_F64 ? (int64_t)1 << 27 : (int64_t)1 << 31;
    int64_t n = std::max<int64_t>(work / lat.ncell / g.depth, 1) * g.depth;
    while (n > 1) {
        g.nsteps = (int)std::min<int64_t>(n, 1 << 28);
        if (chain_tickets(g) < (int64_t)1 << 30) break;
        n /= 2;
    }
    return n;
}

// Dynamic shared memory of a shape, or -1 when the shape is invalid: the segment must be
// a multiple of the 16-byte unit, the rows of a job must fit the direction buffer and
// the stage count must be in [2, 8].
int tma_thread_limit(const Lattice &lat) { return lbmd::tma_max_threads(lat.D, lat.P); }

int tma_smem_bytes(const Lattice &lat, const TmaShape &t) {
    const int U = 16 / esize(lat.P);
    if (t.stages < 2 || t.stages > kTmaMaxStages) return -1;
    if (t.cap != 1024 && t.cap != 2048 && t.cap != 4096 && t.cap != 8192) return -1;
    if (t.seg < lat.nx && ((t.seg % U) != 0 || lat.pitch != lat.nx)) return -1;
    const lbmd::TmaGeom g = geom(lat, t);
    if ((int64_t)g.rows * g.rowstride > g.bufstride) return -1;
    if (g.njobs >= ((int64_t)1 << 31)) return -1;
    if (t.threads < 32 || t.threads > lbmd::tma_max_threads(lat.D, lat.P) || t.threads % 32) return -1;
    const int64_t bytes = (int64_t)t.stages * lbmd::qof(lat.D) * t.cap;
    return bytes > kTmaMaxSmem ? -1 : (int)bytes;
}

// The dynamic shared memory limit belongs to the kernel function, which every lattice of the same
// kind shares, whatever its launch shape: it is set to the most a block can have and never lowered.
// (With the size of the shape at hand, creating a lattice of 2 stages made the launches of one of 3
// stages fail.)
cudaError_t tma_prepare(const Lattice &lat, int eq, int bulk, int cap) {
    for (const bool several : {false, true}) {
        const void *fn = tma_kernel(lat, eq, bulk, cap, several);
        if (!fn) return cudaErrorInvalidValue;
        cudaFuncAttributes at;
        cudaError_t e = cudaFuncGetAttributes(&at, fn);
        const int most = kTmaMaxSmem - (int)at.sharedSizeBytes;
        if (e == cudaSuccess && at.maxDynamicSharedSizeBytes < most)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

bool tma_set_blocks(const Lattice &lat, int eq, int bulk, int sms, TmaShape &t) {
    if (tma_prepare(lat, eq, bulk, t.cap) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    for (const bool several : {false, true}) {
        const void *fn = tma_kernel(lat, eq, bulk, t.cap, several);
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, t.threads + (several ? lbmd::kTmaServiceThreads : 32), t.smem_bytes) !=
            cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        if (n < 1) return false;
        (several ? t.blocks : t.one_blocks) = sms * n;
    }
    return true;
}

cudaError_t step_tma(const StepArgs &a, const TmaShape &t, int nsteps, cudaStream_t s) {
    const bool several = nsteps > 1;
    const void *fn = tma_kernel(a.lat, a.eq, a.bulk, t.cap, several);
    if (!fn) return cudaErrorInvalidValue;
    lbmd::TmaGeom g = geom(a.lat, t);
    StepArgs aa = a;
    void *args[] = {(void *)&aa, (void *)&g};
    int blocks = t.one_blocks;
    if (several) {
        if (!chain_geom(a.lat, t, nsteps, g)) return cudaErrorInvalidValue;
        // more blocks than jobs of one step would only wait for one another
        blocks = (int)std::min<int64_t>(t.blocks, std::max<int64_t>(1, g.njobs));
    }
    g.by_nseg = lbmd::fast_div(g.nseg);
    g.by_ygroups = lbmd::fast_div(g.ygroups);
    g.by_npos = lbmd::fast_div(std::max(1, g.npos));
    g.by_strips = lbmd::fast_div(std::max(1, g.strips));
    g.by_pjobs = lbmd::fast_div(std::max(1, g.pjobs));
    g.by_depth = lbmd::fast_div(std::max(1, g.depth));
    // t.threads consumer threads plus the service warp, or the loader and the storer
    return cudaLaunchKernel(fn, dim3(blocks), dim3(t.threads + (several ? lbmd::kTmaServiceThreads : 32)), args, (size_t)t.smem_bytes, s);
}

}  // namespace lbmh
