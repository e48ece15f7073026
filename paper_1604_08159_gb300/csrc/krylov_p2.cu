// Krylov kernels of DD order 2p = 4 (single-run and batched, FP64 and the
// mixed mode), compiled in a translation unit of their own.
#include "krylov_stream.cuh"

namespace wrc {
template struct KrylovKernels<double, 2>;
template struct KrylovKernels<float, 2>;
}  // namespace wrc
