// k_tma_d2_c2048.cu -- TMA row-staged step kernels for D = 2, 2048-byte direction buffers.
#include "k_tma.cuh"

namespace lbmh {
const void *tma_kernel_d2_c2048(int P, int eq, int bulk, bool several) { return lbmd::tma_kernel_dc<2, 2048>(P, eq, bulk, several); }
}  // namespace lbmh
