// Host side of the forward kernel (dos_kernel.cuh): launch constants, tensor
// maps, workspaces, and the scaling of a batch's accumulators.
#include "dos_kernel.cuh"

namespace tetra {

namespace fwd {

#define TETRA_FWD_EXTERN(MODE, MAXM, COPIES)                                                                           \
    extern template cudaError_t launch_norb<MODE, MAXM, COPIES>(int, int, size_t, dim3, const Batch<MAXM> &,              \
                                                                const FwdArgs &, cudaStream_t);
TETRA_FWD_EXTERN(TETRA_POINT, 1, false)
TETRA_FWD_EXTERN(TETRA_POINT, 1, true)
TETRA_FWD_EXTERN(TETRA_BIN, 1, false)
TETRA_FWD_EXTERN(TETRA_INTEGRATED, 1, true)
TETRA_FWD_EXTERN(TETRA_POINT, kMaxBatch, false)
TETRA_FWD_EXTERN(TETRA_POINT, kMaxBatch, true)
TETRA_FWD_EXTERN(TETRA_BIN, kMaxBatch, false)
#undef TETRA_FWD_EXTERN

}  // namespace fwd

namespace {

using namespace fwd;

// Batched: model blockIdx.y scales its int64 accumulator (slot = model).
struct BatchOut {
    float *dos[kMaxBatch];
};
__global__ void tetra_dos_reduce_batched(const __grid_constant__ Batch<kMaxBatch> B, const BatchOut O,
                                         const long long *G, int copies, int n_orb, int chunk_w, int mode) {
    const ModelP &M = B.m[blockIdx.y];
    __shared__ float s_unit[2];
    if (threadIdx.x == 0) {
        float fq;
        unit_pair(fixed_unit(M.omega, M.n_omega, mode, M.vtvg, M.fixed_bits, fq), s_unit[0], s_unit[1]);
    }
    __syncthreads();
    const float uh = s_unit[0], ul = s_unit[1];
    const long total = (long)n_orb * M.n_omega;
    for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total;
         idx += (long)gridDim.x * blockDim.x) {
        const int s = (int)(idx / M.n_omega), i = (int)(idx - (long)s * M.n_omega);
        long long g = 0;
        for (int r = 0; r < copies; ++r) g += G[(((long)blockIdx.y * copies + r) * n_orb + s) * chunk_w + i];
        O.dos[blockIdx.y][idx] = scale_units(g, uh, ul);
    }
}

// Launch constants shared by all models of a plan (box geometry, strides).
void fill_common(const Plan &P, FwdArgs &A) {
    A.nb = P.d.n_bands; A.n_orb = P.d.n_orb;
    A.BX = P.BX; A.BY = P.BY; A.BZ = P.BZ;
    A.lbx = __builtin_ctz(P.BX); A.lby = __builtin_ctz(P.BY); A.lbz = __builtin_ctz(P.BZ);
    A.eps_stride = P.eps_stride; A.w_stride = P.w_stride;
    const uint32_t npts = (uint32_t)(P.BX + 1) * (P.BY + 1) * (P.BZ + 1);
    A.e_box_bytes = npts * P.eps_stride * 4u;
    A.w_box_bytes = npts * P.w_stride * (uint32_t)P.wbytes;
    // every TMA destination starts on a 128-byte boundary
    A.e_stage = (A.e_box_bytes + 127u) & ~127u;
    A.w_stage = (A.w_box_bytes + 127u) & ~127u;
    A.chunk_w = P.chunk_w;
    A.tile_copies = P.tile_copies;
    A.items_per_box = P.items_per_box;
    // few items per box (few bands): up to 8 lanes share a pair's walk, so that
    // the box still has work for all warps and the walks are that much shorter
    A.split = 0;
    while (A.split < 3 && (P.items_per_box << (A.split + 1)) <= kThreads) ++A.split;
    A.flush_at = 1u << P.flush_bits;
    A.fast_cap = P.fast_cap;
}

ModelP model_of(const Plan &P, const float *omega) {
    ModelP m;
    m.n1 = P.d.n1; m.n2 = P.d.n2; m.n3 = P.d.n3; m.z0 = P.z0; m.z1 = P.z1;
    m.nbx = P.nbx; m.nby = P.nby; m.n_boxes = P.n_boxes; m.n_omega = P.d.n_omega;
    m.fixed_bits = P.fixed_bits;
    m.box_base = 0;
    m.copies = P.copies;
    m.vtvg = 1.0 / (6.0 * (double)P.d.n1 * (double)P.d.n2 * (double)P.d.n3);
    m.omega = omega;
    return m;
}

tetra_status_t encode_maps(const Plan &P, const float *eps, const void *w, MapPair &mp) {
    const CUtensorMapDataType wdt = P.d.weight_dtype == TETRA_F16    ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                    : P.d.weight_dtype == TETRA_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                                     : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    tetra_status_t st = encode_point_map(&mp.e, eps, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, P.eps_stride,
                                         P.nx, P.ny, P.nz, P.BX + 1, P.BY + 1, P.BZ + 1);
    if (st != TETRA_OK) return st;
    return encode_point_map(&mp.w, w, wdt, P.wbytes, P.w_stride, P.nx, P.ny, P.nz, P.BX + 1,
                            P.BY + 1, P.BZ + 1);
}

}  // namespace

size_t dos_forward_workspace(const Plan &P) {
    // integrated mode: a second array of the same size for the step sums
    const size_t parts = sizeof(long long) * (size_t)P.n_chunks * P.copies * P.d.n_orb * (size_t)P.chunk_w;
    return kStatusBytes + (P.d.mode == TETRA_INTEGRATED ? 2 : 1) * parts;
}

tetra_status_t launch_dos_forward(const Plan &P, const float *eps, const void *w,
                                  const float *omega, float *dos, void *ws, size_t ws_bytes,
                                  cudaStream_t stream) {
    const size_t need = dos_forward_workspace(P);
    if (ws_bytes < need) return TETRA_ENOMEM;
    static thread_local Batch<1> Bt;   // 0.3 KB of tensor maps + model constants
    Bt.n_models = 1;
    Bt.total_work = P.n_boxes;
    tetra_status_t st = encode_maps(P, eps, w, Bt.maps[0]);
    if (st != TETRA_OK) return st;
    Bt.m[0] = model_of(P, omega);
    FwdArgs A;
    fill_common(P, A);
    A.status = reinterpret_cast<int *>(ws);
    A.queue = nullptr;
    A.G = reinterpret_cast<long long *>(static_cast<unsigned char *>(ws) + kStatusBytes);
    A.Gs = A.G + (size_t)P.n_chunks * P.copies * P.d.n_orb * (size_t)P.chunk_w;
    A.done = reinterpret_cast<int *>(static_cast<unsigned char *>(ws) + kDoneOffset);
    A.dos = dos;
    cudaError_t e = cudaMemsetAsync(ws, 0, need, stream);
    if (e != cudaSuccess) return TETRA_ECUDA;
    const dim3 grid(P.grid_x, P.n_chunks);
    const int n_orb = P.d.n_orb, wdt = P.d.weight_dtype;
    switch (P.d.mode) {
        case TETRA_POINT:
            e = P.copies > 1 ? launch_norb<TETRA_POINT, 1, true>(n_orb, wdt, P.smem_bytes, grid, Bt, A, stream)
                             : launch_norb<TETRA_POINT, 1, false>(n_orb, wdt, P.smem_bytes, grid, Bt, A, stream);
            break;
        case TETRA_BIN: e = launch_norb<TETRA_BIN, 1, false>(n_orb, wdt, P.smem_bytes, grid, Bt, A, stream); break;
        default: e = launch_norb<TETRA_INTEGRATED, 1, true>(n_orb, wdt, P.smem_bytes, grid, Bt, A, stream);
    }
    return e == cudaSuccess ? TETRA_OK : TETRA_ECUDA;
}

size_t dos_batched_workspace(const BatchPlan &B) {
    return kStatusBytes + sizeof(long long) * (size_t)B.n_models * B.copies * B.models[0].d.n_orb * (size_t)B.chunk_w;
}

tetra_status_t launch_dos_batched(const BatchPlan &BP, const float *const *eps, const void *const *w,
                                  const float *const *omega, float *const *dos, void *ws,
                                  size_t ws_bytes, cudaStream_t stream) {
    const size_t need = dos_batched_workspace(BP);
    if (ws_bytes < need) return TETRA_ENOMEM;
    std::unique_ptr<Batch<kMaxBatch>> Bt(new (std::nothrow) Batch<kMaxBatch>());
    std::unique_ptr<BatchOut> O(new (std::nothrow) BatchOut());
    if (!Bt || !O) return TETRA_ENOMEM;
    Bt->n_models = BP.n_models;
    Bt->total_work = BP.total_boxes;
    for (int m = 0; m < BP.n_models; ++m) {
        const Plan &P = BP.models[m];
        tetra_status_t st = encode_maps(P, eps[m], w[m], Bt->maps[m]);
        if (st != TETRA_OK) return st;
        ModelP mp = model_of(P, omega[m]);
        mp.box_base = BP.box_base[m];
        mp.copies = BP.copies;
        Bt->m[m] = mp;
        O->dos[m] = dos[m];
    }
    const Plan &P0 = BP.models[BP.big];
    FwdArgs A;
    fill_common(P0, A);
    A.chunk_w = BP.chunk_w;
    A.status = reinterpret_cast<int *>(ws);
    A.queue = reinterpret_cast<int *>(static_cast<unsigned char *>(ws) + kQueueOffset);
    A.G = reinterpret_cast<long long *>(static_cast<unsigned char *>(ws) + kStatusBytes);
    A.Gs = nullptr;
    A.done = nullptr;
    A.dos = nullptr;
    cudaError_t e = cudaMemsetAsync(ws, 0, need, stream);   // status, counter, accumulators
    if (e != cudaSuccess) return TETRA_ECUDA;
    const dim3 grid(BP.grid_x, 1);
    const int n_orb = P0.d.n_orb, wdt = P0.d.weight_dtype;
    e = P0.d.mode == TETRA_BIN ? launch_norb<TETRA_BIN, kMaxBatch, false>(n_orb, wdt, BP.smem_bytes, grid, *Bt, A, stream)
        : BP.copies > 1        ? launch_norb<TETRA_POINT, kMaxBatch, true>(n_orb, wdt, BP.smem_bytes, grid, *Bt, A, stream)
                               : launch_norb<TETRA_POINT, kMaxBatch, false>(n_orb, wdt, BP.smem_bytes, grid, *Bt, A, stream);
    if (e != cudaSuccess) return TETRA_ECUDA;
    const long total = (long)n_orb * BP.chunk_w;
    const int rb = 256;
    const int rg = (int)std::max<long>(1, std::min<long>((total + rb - 1) / rb, 64));
    tetra_dos_reduce_batched<<<dim3(rg, BP.n_models), rb, 0, stream>>>(*Bt, *O, A.G, BP.copies, n_orb,
                                                                        BP.chunk_w, P0.d.mode);
    if (cudaGetLastError() != cudaSuccess) return TETRA_ECUDA;
    return TETRA_OK;
}

}  // namespace tetra
