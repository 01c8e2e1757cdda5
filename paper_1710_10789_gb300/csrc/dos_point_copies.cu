// Forward kernel: point mode, copies of the accumulator.
#include "dos_kernel.cuh"

namespace tetra {
namespace fwd {
template cudaError_t launch_norb<TETRA_POINT, 1, true>(int, int, size_t, dim3, const Batch<1> &, const FwdArgs &, cudaStream_t);
}  // namespace fwd
}  // namespace tetra
