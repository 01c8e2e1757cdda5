// Forward kernel: point mode, batches, copies of the accumulators.
#include "dos_kernel.cuh"

namespace tetra {
namespace fwd {
template cudaError_t launch_norb<TETRA_POINT, kMaxBatch, true>(int, int, size_t, dim3, const Batch<kMaxBatch> &, const FwdArgs &, cudaStream_t);
}  // namespace fwd
}  // namespace tetra
