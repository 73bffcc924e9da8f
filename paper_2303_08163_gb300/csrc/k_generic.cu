// k_generic.cu -- auxiliary kernels of a single lattice: initialisation f = f^eq(rho, u),
// moments, canonical population export / import (undoing the AA odd-step slot
// permutation), sampled export, diagnostics of a state, the fixed-order final reduction
// of diagnostics, the bounded-wait self test, and the generic step dispatcher.
#include <algorithm>

#include "lbm_common.cuh"
#include "ptx.cuh"

namespace lbmh {
cudaError_t step_generic_d2(const StepArgs &a, int blocks, int threads, cudaStream_t s);
cudaError_t step_generic_d3(const StepArgs &a, int blocks, int threads, cudaStream_t s);
const void *small_kernel_d2(int P, int eq, int bulk, bool lanes, bool many);
const void *small_kernel_d3(int P, int eq, int bulk, bool lanes, bool many);
}  // namespace lbmh

namespace lbmd {

static inline int grid_for(int64_t n, int threads, int cap = 152 * 32) {
    int64_t g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

// The kernels between the caller's fields or populations and the stored ones are bound by HBM (FP64
// storage by the FP64 pipe).  A thread has V neighbouring cells of a row: 2 for binary16 storage,
// where a 2-byte access for each population leaves the memory pipe half used (512^3: initialisation
// 2.43 -> 1.52 ms, moments 2.06 - 2.48 -> 1.45 - 1.85 ms, 1.39 ms of HBM time), otherwise 1.  Kernels that
// write the stored populations run over the rows with their padding and write each plane where the
// thread is, so that warps write whole aligned segments, the padding (with the row's last value) included;
// shifts go into the reads (FP32 245 x 196 x 172: initialisation 0.34 -> 0.21 ms; FP32 256^3
// populations after an odd number of steps 0.86 -> 0.60 ms).  Populations from FP64 arrays into FP64 or
// FP32 storage are written where they belong: their reads are the wider ones (128^3 FP64 0.14 against
// 0.19 ms, FP32 0.21 against 0.26).

// Cell of an element of the padded rows (in the padding: the row's last cell), for V = 2 the first of two.
__device__ __forceinline__ int64_t padded_cell(const lbmh::Lattice &lat, int64_t p, int64_t padded, int &x) {
    x = 0;
    if (lat.pitch == lat.nx) return p;
    int64_t row;
    if (padded < ((int64_t)1 << 31)) row = (unsigned)p / (unsigned)lat.pitch;
    else row = p / lat.pitch;
    x = min((int)(p - row * lat.pitch), lat.nx - 1);
    return row * lat.nx + x;
}

// V stored values at p (V = 2: p even).
template <int P, int V>
__device__ __forceinline__ void store_v(typename Storage<P>::T *p, const typename Storage<P>::R (&v)[V]) {
    if constexpr (V == 2) *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(v[0], v[1]);
    else *p = Storage<P>::store(v[0]);
}

// V values of the caller's array at p (V = 2: aligned to both).  Two stores of one value each leave
// every segment half written, which costs the host link a tenth (512^3 moments into pinned memory
// 12.4 against 11.2 ms).
template <int V, typename Out> __device__ __forceinline__ void put_v(Out *p, Out a, Out b) {
    if constexpr (V == 1) *p = a;
    else if constexpr (sizeof(Out) == 4) *reinterpret_cast<float2 *>(p) = make_float2(a, b);
    else *reinterpret_cast<double2 *>(p) = make_double2(a, b);
}

// f = f^eq(rho, u), written in the even (canonical) layout, shifted by w_i rho0.
template <int D, int P, int EQ, int V, typename In>
__global__ void k_init(lbmh::Lattice lat, double rho0d, const In *__restrict__ rho,
                       const In *__restrict__ u) {
    using R = typename Storage<P>::R;
    constexpr int Q = qof(D);
    auto *A = static_cast<typename Storage<P>::T *>(lat.A);
    const R rho0 = R(rho0d);
    const int64_t padded = (int64_t)lat.pitch * lat.ny * lat.nz;
    for (int64_t p = V * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x); p < padded;
         p += V * (int64_t)gridDim.x * blockDim.x) {
        int x;
        const int64_t c = padded_cell(lat, p, padded, x);
        R r[V], drho[V], h[V][Q];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int64_t cv = V == 1 || lat.pitch == lat.nx || x + v < lat.nx ? c + v : c;  // (a row's last pair may end in its padding)
            r[v] = R(rho[cv]);
            R uu[3] = {R(u[cv]), R(u[lat.ncell + cv]), D == 3 ? R(u[2 * lat.ncell + cv]) : R(0)};
            equilibrium_h<D, EQ, R>(uu, h[v]);
            drho[v] = r[v] - rho0;
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            R f[V];
#pragma unroll
            for (int v = 0; v < V; ++v) f[v] = R(wq<D>(i)) * fma_r(r[v], h[v][i], drho[v]);
            store_v<P, V>(A + (int64_t)i * lat.plane + p, f);
        }
    }
}

template <int D, int P>
__device__ __forceinline__ void load_canonical(const lbmh::Lattice &lat, int odd, int64_t c,
                                               typename Storage<P>::R (&f)[qof(D)], int &x,
                                               int &y, int &z) {
    using St = Storage<P>;
    const auto *A = static_cast<const typename St::T *>(lat.A);
    cell_coords(c, lat.ncell, lat.nx, lat.ny, x, y, z);
#pragma unroll
    for (int i = 0; i < qof(D); ++i)
        f[i] = St::load(A[aa_index<D>(i, x, y, z, lat.nx, lat.ny, lat.nz, lat.pitch, lat.plane, odd)]);
}

// The same for V cells of a row from c (V = 2: nx and c even): both halves at once where the layout
// has them side by side.
template <int D, int P, int V>
__device__ __forceinline__ void load_canonical_v(const lbmh::Lattice &lat, int odd, int64_t c,
                                                 typename Storage<P>::R (&f)[V][qof(D)]) {
    int x, y, z;
    if constexpr (V == 1) {
        load_canonical<D, P>(lat, odd, c, f[0], x, y, z);
    } else {
        cell_coords(c, lat.ncell, lat.nx, lat.ny, x, y, z);
        const auto *A = static_cast<const __half *>(lat.A);
#pragma unroll
        for (int i = 0; i < qof(D); ++i) {
            const int64_t a = aa_index<D>(i, x, y, z, lat.nx, lat.ny, lat.nz, lat.pitch, lat.plane, odd);
            if (!odd || cxo(i) == 0) {
                const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(A + a));
                f[0][i] = v.x;
                f[1][i] = v.y;
            } else {
                f[0][i] = __half2float(A[a]);
                f[1][i] = __half2float(A[aa_index<D>(i, x + 1, y, z, lat.nx, lat.ny, lat.nz, lat.pitch, lat.plane, odd)]);
            }
        }
    }
}

template <int D, int P, int V, typename Out>
__global__ void k_moments(lbmh::Lattice lat, double rho0d, int odd, Out *__restrict__ rho,
                          Out *__restrict__ u) {
    using R = typename Storage<P>::R;
    for (int64_t c = V * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x); c < lat.ncell;
         c += V * (int64_t)gridDim.x * blockDim.x) {
        R f[V][qof(D)];
        load_canonical_v<D, P, V>(lat, odd, c, f);
        CellMoments<R> m[V];
#pragma unroll
        for (int v = 0; v < V; ++v) m[v] = moments_shifted<D, R>(f[v], R(rho0d));
        put_v<V>(rho + c, Out(m[0].rho), Out(m[V - 1].rho));
#pragma unroll
        for (int a = 0; a < D; ++a) put_v<V>(u + a * lat.ncell + c, Out(m[0].u[a]), Out(m[V - 1].u[a]));
    }
}

// w_i rho0 of one weight class: the double, and split into two floats for FP32 callers.
struct ClassShift {
    double w[4];
    float hi[4], lo[4];
};

// g + w rho0 and f - w rho0 in the caller's type.  For FP32 storage and callers the sum is formed in
// FP32 with its rounding error carried (two-sum), so that it is the FP64 sum rounded to FP32 but
// for the last of 48 bits: conversions to and from FP64 and an FP64 addition for each population
// took 19.6 ms on a 512^3 binary16 lattice (3.2 ms of HBM time) on the FP64 pipe.
__device__ __forceinline__ float two_sum(float a, float b, float c) {  // a + b + c, |c| << |a + b|
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return isfinite(s) ? __fadd_rn(s, __fadd_rn(e, c)) : s;  // (the error of an infinite sum is no number)
}
template <typename R, typename Out>
__device__ __forceinline__ Out unshift(R g, const ClassShift &k, int c) {
    if constexpr (sizeof(R) == 4 && sizeof(Out) == 4) return two_sum(g, k.hi[c], k.lo[c]);
    else return Out((double)g + k.w[c]);
}
template <typename R, typename In>
__device__ __forceinline__ R shift(In f, const ClassShift &k, int c) {
    if constexpr (sizeof(R) == 4 && sizeof(In) == 4) return two_sum(f, -k.hi[c], -k.lo[c]);
    else return R((double)f - k.w[c]);
}

template <int D, int P, int V, typename Out>
__global__ void k_get_pop(lbmh::Lattice lat, ClassShift k, int odd, Out *__restrict__ f) {
    using R = typename Storage<P>::R;
    for (int64_t c = V * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x); c < lat.ncell;
         c += V * (int64_t)gridDim.x * blockDim.x) {
        R g[V][qof(D)];
        load_canonical_v<D, P, V>(lat, odd, c, g);
#pragma unroll
        for (int i = 0; i < qof(D); ++i)
            put_v<V>(f + (int64_t)i * lat.ncell + c, unshift<R, Out>(g[0][i], k, wclass<D>(i)),
                     unshift<R, Out>(g[V - 1][i], k, wclass<D>(i)));
    }
}

template <int D, int P, int V, typename In>
__global__ void k_set_pop(lbmh::Lattice lat, ClassShift k, int odd, const In *__restrict__ f) {
    using R = typename Storage<P>::R;
    constexpr int Q = qof(D);
    auto *A = static_cast<typename Storage<P>::T *>(lat.A);
    const int64_t padded = (int64_t)lat.pitch * lat.ny * lat.nz;
    for (int64_t p = V * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x); p < padded;
         p += V * (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_coords(p, padded, lat.pitch, lat.ny, x, y, z);
        if constexpr (P == P_F64 || (P == P_F32 && sizeof(In) == 8)) {
            if (x >= lat.nx) continue;
            const int64_t c = x + (int64_t)lat.nx * (y + (int64_t)lat.ny * z);
#pragma unroll
            for (int i = 0; i < Q; ++i)
                A[aa_index<D>(i, x, y, z, lat.nx, lat.ny, lat.nz, lat.pitch, lat.plane, odd)] =
                    shift<R, In>(f[(int64_t)i * lat.ncell + c], k, wclass<D>(i));
            continue;
        }
        In v[Q][V];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            // slot opp(i) of this cell holds f_i of the cell c_i further after an odd number of
            // steps, slot i holds its own f_i after an even one
            const int yy = odd ? wrapi(y + cyo(i), lat.ny) : y;
            const int zz = D == 3 && odd ? wrapi(z + czo(i), lat.nz) : z;
            const In *row = f + (int64_t)i * lat.ncell + (int64_t)lat.nx * (yy + (int64_t)lat.ny * zz);
#pragma unroll
            for (int q = 0; q < V; ++q) {
                const int xv = min(x + q, lat.nx - 1);
                v[i][q] = row[odd ? wrapi(xv + cxo(i), lat.nx) : xv];
            }
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            R r[V];
#pragma unroll
            for (int q = 0; q < V; ++q) r[q] = shift<R, In>(v[i][q], k, wclass<D>(i));
            store_v<P, V>(A + (int64_t)(odd ? Q - 1 - i : i) * lat.plane + p, r);
        }
    }
}

// Raw stored (shifted) values in the canonical layout, bit for bit.
template <int D, int P>
__global__ void k_get_pop_raw(lbmh::Lattice lat, int odd, typename Storage<P>::T *__restrict__ f) {
    const auto *A = static_cast<const typename Storage<P>::T *>(lat.A);
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < lat.ncell;
         c += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_coords(c, lat.ncell, lat.nx, lat.ny, x, y, z);
#pragma unroll
        for (int i = 0; i < qof(D); ++i)
            f[(int64_t)i * lat.ncell + c] = A[aa_index<D>(i, x, y, z, lat.nx, lat.ny, lat.nz, lat.pitch, lat.plane, odd)];
    }
}

template <int D, int P>
__global__ void k_set_pop_raw(lbmh::Lattice lat, int odd, const typename Storage<P>::T *__restrict__ f) {
    auto *A = static_cast<typename Storage<P>::T *>(lat.A);
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < lat.ncell;
         c += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        cell_coords(c, lat.ncell, lat.nx, lat.ny, x, y, z);
#pragma unroll
        for (int i = 0; i < qof(D); ++i)
            A[aa_index<D>(i, x, y, z, lat.nx, lat.ny, lat.nz, lat.pitch, lat.plane, odd)] = f[(int64_t)i * lat.ncell + c];
    }
}

template <int D, int P>
__global__ void k_sample_pop(lbmh::Lattice lat, double rho0, int odd, const int64_t *cells,
                             int64_t count, double *out) {
    using R = typename Storage<P>::R;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < count;
         k += (int64_t)gridDim.x * blockDim.x) {
        R g[qof(D)];
        int x, y, z;
        load_canonical<D, P>(lat, odd, cells[k], g, x, y, z);
#pragma unroll
        for (int i = 0; i < qof(D); ++i) out[k * qof(D) + i] = (double)g[i] + wq<D>(i) * rho0;
    }
}

template <int D, int P>
__global__ void __launch_bounds__(256) k_diag_state(lbmh::Lattice lat, double rho0d, int odd,
                                                    double *partials) {
    using R = typename Storage<P>::R;
    DiagAcc acc;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < lat.ncell;
         c += (int64_t)gridDim.x * blockDim.x) {
        R f[qof(D)];
        int x, y, z;
        load_canonical<D, P>(lat, odd, c, f, x, y, z);
        const CellMoments<R> m = moments_shifted<D, R>(f, R(rho0d));
        acc.add(m.rho, m.u);
    }
    diag_block_store(acc, partials + (int64_t)blockIdx.x * lbmh::kDiagWords);
}

// record = {mass, jx, jy, jz, kinetic, max|u|, nonfinite, step}: sums of the per-block
// partials in a fixed order (thread t takes blocks t, t + 256, ..., then a fixed tree).
__global__ void __launch_bounds__(256) k_diag_finalize(const double *partials, int blocks,
                                                       int64_t step, double *record) {
    __shared__ double red[256][7];
    double s[7] = {0, 0, 0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < blocks; b += blockDim.x) {
#pragma unroll
        for (int q = 0; q < 7; ++q) {
            const double v = partials[(int64_t)b * lbmh::kDiagWords + q];
            s[q] = (q == 5) ? fmax(s[q], v) : s[q] + v;
        }
    }
#pragma unroll
    for (int q = 0; q < 7; ++q) red[threadIdx.x][q] = s[q];
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
#pragma unroll
            for (int q = 0; q < 7; ++q) {
                const double o = red[threadIdx.x + w][q];
                red[threadIdx.x][q] = (q == 5) ? fmax(red[threadIdx.x][q], o) : red[threadIdx.x][q] + o;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
#pragma unroll
        for (int q = 0; q < 7; ++q) record[q] = red[0][q];
        record[7] = (double)step;
    }
}

__global__ void k_selftest_wait(int64_t timeout_ns, int32_t *status) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_barrier_init();
    }
    __syncthreads();
    const bool ok = mbar_wait_bounded(&bar, 0, timeout_ns);
    if (threadIdx.x == 0) *status = ok ? 0 : -5; /* LBM_ETIMEOUT */
}

}  // namespace lbmd

namespace lbmh {

using namespace lbmd;

int diag_blocks_generic(int64_t ncell) { return grid_for(ncell, 256, 152 * 8); }

cudaError_t step_generic(const StepArgs &a, int blocks, int threads, cudaStream_t s) {
    return a.lat.D == 2 ? step_generic_d2(a, blocks, threads, s) : step_generic_d3(a, blocks, threads, s);
}

static const void *small_kernel(const Lattice &lat, int eq, int bulk, const SmallShape &t) {
    return lat.D == 2 ? small_kernel_d2(lat.P, eq, bulk, t.lanes, t.many) : small_kernel_d3(lat.P, eq, bulk, t.lanes, t.many);
}

// The largest lattice of the several-step kernel, in cells an SM: what the threads of its resident
// blocks hold, one cell each, and twice that where two rounds are still faster than the TMA row kernel
// (512^2 FP32 3.9 us a step against 5.1; 512^2 binary16 4.6 - 5.9 against 4.9, so not there;
// 56^3 binary16 8.3 against 7.4, but 60^3, whose short ragged rows that kernel does not take, 8.3
// against 17).  FP64 in 3-D takes three rounds (48^3 45 us).
static int64_t small_limit(const Lattice &lat) {
    if (lat.D == 2) return lat.P == P_F16S ? 1280 : lat.P == P_F32 ? 2048 : 1024;
    return lat.P == P_F16S && !tma_supported(lat) ? 1536 : 768;
}

// An SM's cells are spread over as few blocks as hold them, all with equally many warps.  FP64
// lattices of at most 40 cells an SM have a cell on three lanes: a warp on each quarter is all there
// is either way, and a warp instruction costs the same for 7 cells as for 10 of three lanes (with 41
// to 80 cells an SM quarter would have two such warps, as long as one of 32 cells).
bool small_shape(const Lattice &lat, int eq, int bulk, int sms, SmallShape &t) {
    if (lat.ncell > small_limit(lat) * sms || lat.plane * qof(lat.D) >= ((int64_t)1 << 31)) return false;
    const int64_t per = (lat.ncell + sms - 1) / sms;  // cells an SM
    t.lanes = lat.P == P_F64 && per <= 40;
    const int warp = t.lanes ? 10 : 32;  // cells a warp
    const int64_t warps = (per + warp - 1) / warp;
    int64_t n = std::min<int64_t>((warps + 7) / 8, small_blocks(lat.D, lat.P));
    // several rounds of the 3-D FP64 kernel: one block with all the registers (44^3 45 us, 61 in two)
    if (lat.D == 3 && lat.P == P_F64 && warps > 16) n = 1;
    t.many = n > 1;
    t.threads = (int)(32 * std::min<int64_t>(8, (warps + n - 1) / n));
    const int64_t cells = t.threads / 32 * warp;
    const void *fn = small_kernel(lat, eq, bulk, t);
    int nb = 0;
    if (!fn || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, t.threads, 0) != cudaSuccess || nb < 1) {
        cudaGetLastError();
        return false;
    }
    t.blocks = (int)std::min<int64_t>((lat.ncell + cells - 1) / cells, (int64_t)nb * sms);
    return true;
}

size_t small_msg_bytes(const Lattice &lat) {
    const size_t word = lat.P == P_F64 ? 16 : lat.P == P_F32 ? 8 : 4;  // a population and a step number
    return kMsgHead + word * qof(lat.D) * lat.plane;
}

cudaError_t steps_small(const StepArgs &a, int nsteps, const SmallShape &t, cudaStream_t s) {
    const void *fn = small_kernel(a.lat, a.eq, a.bulk, t);
    if (!fn) return cudaErrorInvalidValue;
    StepArgs aa = a;
    void *args[] = {(void *)&aa, (void *)&nsteps};
    return cudaLaunchCooperativeKernel(fn, dim3(t.blocks), dim3(t.threads), args, 0, s);
}

#define LBM_DISPATCH_DP(D_, P_, CALL)                                                      \
    do {                                                                                   \
        if ((D_) == 2 && (P_) == P_F64) { constexpr int DD = 2, PP = P_F64; CALL; }        \
        else if ((D_) == 2 && (P_) == P_F32) { constexpr int DD = 2, PP = P_F32; CALL; }   \
        else if ((D_) == 2 && (P_) == P_F16S) { constexpr int DD = 2, PP = P_F16S; CALL; } \
        else if ((D_) == 3 && (P_) == P_F64) { constexpr int DD = 3, PP = P_F64; CALL; }   \
        else if ((D_) == 3 && (P_) == P_F32) { constexpr int DD = 3, PP = P_F32; CALL; }   \
        else if ((D_) == 3 && (P_) == P_F16S) { constexpr int DD = 3, PP = P_F16S; CALL; } \
        else return cudaErrorInvalidValue;                                                 \
    } while (0)

// Pairs of binary16 cells: rows (with their padding where the kernel writes them) of even length, and
// more threads than the latency needs: half as many are slower on 32^3 (moments 4.5 against 3.9 us), for
// FP64 populations, each a conversion on the FP64 pipe, up to 64^3 or 1024^2 (35 against 31 us, 40.7
// against 39.6; 2047 x 2000 134 us in pairs, 140 without).
static bool pairs_ok(const Lattice &lat, bool writes, bool fp64_pops) {
    return ((writes ? lat.pitch : lat.nx) & 1) == 0 && lat.ncell >= (int64_t)1 << (fp64_pops ? 21 : 17);
}
// The caller's array p (dtype 0 FP64, 1 FP32) may be written two values at a time.
static bool pairs_fit(const void *p, int dtype) { return (uintptr_t)p % (dtype == 0 ? 16 : 8) == 0; }

#define LBM_DISPATCH_DPV(D_, P_, PAIRS_, CALL)                                                              \
    do {                                                                                                    \
        if ((P_) == P_F16S && (PAIRS_)) {                                                                   \
            if ((D_) == 2) { constexpr int DD = 2, PP = P_F16S, VV = 2; CALL; }                             \
            else { constexpr int DD = 3, PP = P_F16S, VV = 2; CALL; }                                       \
        } else {                                                                                            \
            constexpr int VV = 1;                                                                           \
            LBM_DISPATCH_DP(D_, P_, CALL);                                                                  \
        }                                                                                                   \
    } while (0)

cudaError_t init_fields(const Lattice &lat, int eq, double rho0, const void *rho, const void *u,
                        int dtype, cudaStream_t s) {
    const bool two = pairs_ok(lat, true, false);
    const int g = grid_for((int64_t)lat.pitch * lat.ny * lat.nz / (two && lat.P == P_F16S ? 2 : 1), 256);
#define LBM_INIT_EQ(EQv)                                                                         \
    if (eq == EQv) {                                                                             \
        if (dtype == 0)                                                                          \
            LBM_DISPATCH_DPV(lat.D, lat.P, two, (k_init<DD, PP, EQv, VV, double><<<g, 256, 0, s>>>(        \
                                                lat, rho0, (const double *)rho, (const double *)u))); \
        else                                                                                     \
            LBM_DISPATCH_DPV(lat.D, lat.P, two, (k_init<DD, PP, EQv, VV, float><<<g, 256, 0, s>>>(         \
                                                lat, rho0, (const float *)rho, (const float *)u))); \
        return cudaGetLastError();                                                               \
    }
    LBM_INIT_EQ(EQ_ENT)
    LBM_INIT_EQ(EQ_POLY2)
    LBM_INIT_EQ(EQ_PROD)
#undef LBM_INIT_EQ
    return cudaErrorInvalidValue;
}

cudaError_t moments(const Lattice &lat, double rho0, int odd, void *rho, void *u, int dtype,
                    cudaStream_t s) {
    const bool two = pairs_ok(lat, false, false) && pairs_fit(rho, dtype) && pairs_fit(u, dtype);
    const int g = grid_for(lat.ncell / (two && lat.P == P_F16S ? 2 : 1), 256);
    if (dtype == 0)
        LBM_DISPATCH_DPV(lat.D, lat.P, two, (k_moments<DD, PP, VV, double><<<g, 256, 0, s>>>(lat, rho0, odd, (double *)rho, (double *)u)));
    else
        LBM_DISPATCH_DPV(lat.D, lat.P, two, (k_moments<DD, PP, VV, float><<<g, 256, 0, s>>>(lat, rho0, odd, (float *)rho, (float *)u)));
    return cudaGetLastError();
}

static ClassShift class_shift(int D, double rho0) {
    ClassShift k;
    for (int c = 0; c < 4; ++c) {
        k.w[c] = (D == 2 ? (c <= 2 ? wclass_weight<2>(c) : 0.0) : wclass_weight<3>(c)) * rho0;
        k.hi[c] = (float)k.w[c];
        k.lo[c] = (float)(k.w[c] - (double)k.hi[c]);
    }
    return k;
}

cudaError_t get_populations(const Lattice &lat, double rho0, int odd, void *f, int dtype,
                            cudaStream_t s) {
    const bool two = pairs_ok(lat, false, dtype == 0) && pairs_fit(f, dtype);
    const int g = grid_for(lat.ncell / (two && lat.P == P_F16S && dtype != 2 ? 2 : 1), 256);
    const ClassShift k = class_shift(lat.D, rho0);
    if (dtype == 2)
        LBM_DISPATCH_DP(lat.D, lat.P, (k_get_pop_raw<DD, PP><<<g, 256, 0, s>>>(lat, odd, (typename Storage<PP>::T *)f)));
    else if (dtype == 0)
        LBM_DISPATCH_DPV(lat.D, lat.P, two, (k_get_pop<DD, PP, VV, double><<<g, 256, 0, s>>>(lat, k, odd, (double *)f)));
    else
        LBM_DISPATCH_DPV(lat.D, lat.P, two, (k_get_pop<DD, PP, VV, float><<<g, 256, 0, s>>>(lat, k, odd, (float *)f)));
    return cudaGetLastError();
}

cudaError_t set_populations(const Lattice &lat, double rho0, int odd, const void *f, int dtype,
                            cudaStream_t s) {
    const bool two = pairs_ok(lat, true, dtype == 0);
    const int64_t cells = dtype == 2 ? lat.ncell : (int64_t)lat.pitch * lat.ny * lat.nz;
    const int g = grid_for(cells / (two && lat.P == P_F16S && dtype != 2 ? 2 : 1), 256);
    const ClassShift k = class_shift(lat.D, rho0);
    if (dtype == 2)
        LBM_DISPATCH_DP(lat.D, lat.P, (k_set_pop_raw<DD, PP><<<g, 256, 0, s>>>(lat, odd, (const typename Storage<PP>::T *)f)));
    else if (dtype == 0)
        LBM_DISPATCH_DPV(lat.D, lat.P, two, (k_set_pop<DD, PP, VV, double><<<g, 256, 0, s>>>(lat, k, odd, (const double *)f)));
    else
        LBM_DISPATCH_DPV(lat.D, lat.P, two, (k_set_pop<DD, PP, VV, float><<<g, 256, 0, s>>>(lat, k, odd, (const float *)f)));
    return cudaGetLastError();
}

cudaError_t sample_populations(const Lattice &lat, double rho0, int odd, const int64_t *cells,
                               int64_t count, double *out, cudaStream_t s) {
    const int g = grid_for(count, 128);
    LBM_DISPATCH_DP(lat.D, lat.P, (k_sample_pop<DD, PP><<<g, 128, 0, s>>>(lat, rho0, odd, cells, count, out)));
    return cudaGetLastError();
}

cudaError_t diag_state(const Lattice &lat, double rho0, int odd, double *partials, int blocks,
                       cudaStream_t s) {
    LBM_DISPATCH_DP(lat.D, lat.P, (k_diag_state<DD, PP><<<blocks, 256, 0, s>>>(lat, rho0, odd, partials)));
    return cudaGetLastError();
}

cudaError_t diag_finalize(const double *partials, int blocks, int64_t step, double *record,
                          cudaStream_t s) {
    k_diag_finalize<<<1, 256, 0, s>>>(partials, blocks, step, record);
    return cudaGetLastError();
}

cudaError_t selftest_wait(int64_t timeout_ns, int32_t *status, cudaStream_t s) {
    k_selftest_wait<<<1, 32, 0, s>>>(timeout_ns, status);
    return cudaGetLastError();
}

}  // namespace lbmh
