// Forward kernel: bin mode.
#include "dos_kernel.cuh"

namespace tetra {
namespace fwd {
template cudaError_t launch_norb<TETRA_BIN, 1, false>(int, int, size_t, dim3, const Batch<1> &, const FwdArgs &, cudaStream_t);
}  // namespace fwd
}  // namespace tetra
