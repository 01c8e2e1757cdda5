// Forward kernel: integrated mode.
#include "dos_kernel.cuh"

namespace tetra {
namespace fwd {
template cudaError_t launch_norb<TETRA_INTEGRATED, 1, true>(int, int, size_t, dim3, const Batch<1> &, const FwdArgs &, cudaStream_t);
}  // namespace fwd
}  // namespace tetra
