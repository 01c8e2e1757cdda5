// Forward kernel: bin mode, batches.
#include "dos_kernel.cuh"

namespace tetra {
namespace fwd {
template cudaError_t launch_norb<TETRA_BIN, kMaxBatch, false>(int, int, size_t, dim3, const Batch<kMaxBatch> &, const FwdArgs &, cudaStream_t);
}  // namespace fwd
}  // namespace tetra
