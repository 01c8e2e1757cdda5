// Fermi level: the energy at which the occupation summed over the plan's
// orbitals, N(E) = sum_{T,n} sum_l w_l(E) sum_s b_{n,l,s} (Sec. II.C corner
// weights), reaches a given count.
//
// Only the scalar N is needed, so the orbital weights of a corner enter as
// their sum, and from the second round on only where it matters: N(E) - N(lo)
// over the current bracket [lo, hi] comes from the tetrahedra that straddle
// it. Each round (one launch) evaluates it at kPts energies and its last
// block narrows the bracket and keeps N(lo), exact integers, so the rounds
// run back to back without the host.
//
// One block takes tiles of cubes: it stages the band energies of the tile's
// points in shared memory and the summed weights of the bands that reach the
// bracket; a warp takes 32 cubes of
// one band (their windows nearly coincide, so an energy that no lane's cube
// contains is skipped by a vote: below a cube nothing, above it the full
// weight). The corner weights need no energy cases (tet_common.cuh).
// Each cube's N(E) - N(lo) is rounded once to an integer of 2^-26 of a full
// tetrahedron, summed over the warp by two 32-bit reductions, over the
// block's warps and over the grid by integer adds: exact in any order.
//
// At 95 x 97 x 96 points, 8 bands and 8 orbitals the five rounds of the
// integrated-mode DOS kernel before (64 energies, every orbital, every
// tetrahedron) took 14.4 ms (9.5 ms with its weights without cases).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "tet_common.cuh"

namespace tetra {

namespace {

constexpr int kPts = 16;           // energies per round: bracket / 16
constexpr int kRounds = 64;        // at most; FP32 resolution takes about six
constexpr int kRoundsPerSync = 7;
constexpr int kFermiThreads = 256;
constexpr int kUnitBits = 26;
constexpr int kTilePoints = 297;   // (32 + 1) (2 + 1) (2 + 1), the largest tile below

// Order-preserving map of a float to an unsigned int (for atomic min / max).
__device__ __forceinline__ unsigned ordered(float f) {
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unordered(unsigned u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

// In the workspace after its status words (which a call clears as well).
struct FermiState {
    unsigned mm[2];            // complemented minimum, maximum of the bands (ordered; both from 0 up)
    float lo, hi;              // bracket
    long long base;            // N(lo) in units
    int round, done, bad;      // bad: no such count, or no valid band energy
    int ticket;
    unsigned long long sums[kPts];   // N(E_j) - N(lo) of the running round
};

// Minimum and maximum band energy over the plan's points (bands < nb), four
// values per load (a point's row is a multiple of 16 bytes).
__global__ void band_range_kernel(const float4 *eps, long n_vec, int row_vec, int nb, FermiState *S) {
    unsigned lo = 0u, hi = 0u;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n_vec; i += (long)gridDim.x * blockDim.x) {
        const float4 v = eps[i];
        const int n = 4 * (int)(i % row_vec);
        const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (n + c >= nb) continue;
            const unsigned o = ordered(e[c]);
            lo = max(lo, ~o);
            hi = max(hi, o);
        }
    }
    lo = __reduce_max_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    __shared__ unsigned s_mm[2];
    if (threadIdx.x < 2) s_mm[threadIdx.x] = 0u;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&s_mm[0], lo);
        atomicMax(&s_mm[1], hi);
    }
    __syncthreads();
    if (threadIdx.x < 2) atomicMax(&S->mm[threadIdx.x], s_mm[threadIdx.x]);
}

struct FermiArgs {
    int n1, n2, n3, nx, ny, nb, n_orb, eps_stride, w_stride;
    int tx, ty, tz;          // tile of cubes (tx ty tz = 128 at most)
    int ntx, nty, n_tiles;
    double n_electrons, vtvg;
    const float *eps;
    const void *w;
    FermiState *S;
};

// Energy j of a round's grid, ascending to hi.
__device__ __forceinline__ float grid_energy(float lo, float hi, int j) {
    return j == kPts - 1 ? hi : lo + (hi - lo) * ((float)(j + 1) * (1.0f / kPts));
}

template <typename WT>
__global__ void __launch_bounds__(kFermiThreads, 3) fermi_round_kernel(const FermiArgs A) {
    extern __shared__ float s_pt[];   // energies, then summed weights, [tile point][nb]
    __shared__ unsigned long long s_sum[kPts];
    __shared__ float s_om[kPts];
    __shared__ unsigned s_reach[2][2][2];   // of two tiles in turn
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = kFermiThreads / 32;
    FermiState *S = A.S;
    const bool first = S->round == 0;
    if (S->done) return;   // (set by an earlier launch only)
    float lo, hi;
    if (first) {
        lo = unordered(~S->mm[0]);
        hi = unordered(S->mm[1]);
        if (hi == lo) hi = nextafterf(lo, INFINITY);
    } else {
        lo = S->lo;
        hi = S->hi;
    }
    if (tid < kPts) {
        s_sum[tid] = 0ull;
        s_om[tid] = grid_energy(lo, hi, tid);
    }
    const int px = A.tx + 1, py = A.ty + 1, npt = px * py * (A.tz + 1), nv = npt * A.nb;
    float *se = s_pt, *sw = s_pt + nv;
    const int ncube = A.tx * A.ty * A.tz, groups = (ncube + 31) >> 5;
    const float fq = (float)(1 << kUnitBits) * 0.25f;
    const WT *W = static_cast<const WT *>(A.w);
    long long acc = 0;   // lane j: this warp's sum at energy j
    int tile_par = 0;
    for (int tile = blockIdx.x; tile < A.n_tiles; tile += gridDim.x) {
        const int bx = tile % A.ntx, by = (tile / A.ntx) % A.nty, bz = tile / (A.ntx * A.nty);
        const int x0 = bx * A.tx, y0 = by * A.ty, z0 = bz * A.tz;
        if (tid < 4) s_reach[tile_par][tid >> 1][tid & 1] = 0u;
        __syncthreads();   // the previous tile is read
        // bands with some energy at or above lo / at or below hi
        unsigned long long up = 0ull, down = 0ull;
        for (int i = tid; i < nv; i += kFermiThreads) {
            const int p = i / A.nb, n = i - p * A.nb;
            const int x = min(x0 + p % px, A.n1), y = min(y0 + (p / px) % py, A.n2), z = min(z0 + p / (px * py), A.n3);
            const float e = A.eps[(x + (long)A.nx * (y + (long)A.ny * z)) * A.eps_stride + n];
            se[i] = e;
            up |= (unsigned long long)(e >= lo) << n;
            down |= (unsigned long long)(e <= hi) << n;
        }
        // (nb <= 64: two 32-bit votes each; s_reach was cleared before the first barrier)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned u = __reduce_or_sync(0xffffffffu, (unsigned)(up >> (32 * h)));
            const unsigned d = __reduce_or_sync(0xffffffffu, (unsigned)(down >> (32 * h)));
            if (lane == 0 && u) atomicOr(&s_reach[tile_par][0][h], u);
            if (lane == 0 && d) atomicOr(&s_reach[tile_par][1][h], d);
        }
        __syncthreads();
        const unsigned long long reach =
            ((unsigned long long)(s_reach[tile_par][0][1] & s_reach[tile_par][1][1]) << 32) |
            (s_reach[tile_par][0][0] & s_reach[tile_par][1][0]);
        tile_par ^= 1;
        if (!reach) continue;
        for (int i = tid; i < nv; i += kFermiThreads) {
            const int p = i / A.nb, n = i - p * A.nb;
            if (!((reach >> n) & 1ull)) continue;
            const int x = min(x0 + p % px, A.n1), y = min(y0 + (p / px) % py, A.n2), z = min(z0 + p / (px * py), A.n3);
            const WT *b = W + (x + (long)A.nx * (y + (long)A.ny * z)) * A.w_stride + (long)n * A.n_orb;
            float t = 0.f;
            for (int s = 0; s < A.n_orb; ++s) t += to_f32<WT>(b[s]);
            sw[i] = t;
        }
        __syncthreads();
        for (int item = warp; item < A.nb * groups; item += nwarp) {
            const int n = item / groups, cube = (item - n * groups) * 32 + lane;
            if (!((reach >> n) & 1ull)) continue;
            const int cx = cube % A.tx, cy = (cube / A.tx) % A.ty, cz = cube / (A.tx * A.ty);
            const bool in = cube < ncube && x0 + cx < A.n1 && y0 + cy < A.n2 && z0 + cz < A.n3;
            float e[8], b[8];
            float emin = INFINITY, emax = -INFINITY;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int p = (in ? cx + px * (cy + py * cz) : 0) + (q & 1) + px * (((q >> 1) & 1) + py * (q >> 2));
                e[q] = se[p * A.nb + n];
                b[q] = sw[p * A.nb + n];
                emin = fminf(emin, e[q]);
                emax = fmaxf(emax, e[q]);
            }
            const bool act = in && emax >= lo && emin <= hi;
            if (!__any_sync(0xffffffffu, act)) continue;
            Tet T[6];
            float bs[6][4], at_lo = 0.f, full = 0.f;
#pragma unroll
            for (int t = 0; t < 6; ++t) {
                float es[4], w[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int c = (tet_code(t) >> (3 * q)) & 7;
                    es[q] = e[c];
                    bs[t][q] = b[c];
                }
                sort4(es, bs[t]);
                tet_setup<TETRA_INTEGRATED>(T[t], es[0], es[1], es[2], es[3], fq);
                tet_w(T[t], lo, w);
                full = fmaf(fq, (bs[t][0] + bs[t][1]) + (bs[t][2] + bs[t][3]), full);
#pragma unroll
                for (int q = 0; q < 4; ++q) at_lo = fmaf(bs[t][q], w[q], at_lo);
            }
            // one rounding per energy; the same integers whatever the bracket
            const long long q_lo = __float2ll_rn(at_lo), q_full = __float2ll_rn(full);
#pragma unroll 1
            for (int j = 0; j < kPts; ++j) {
                const float E = s_om[j];
                long long q = 0;
                // a flat tetrahedron at E is empty there: only above emax all is full
                if (act) q = (E > emax ? q_full : 0) - q_lo;
                const bool in_cube = act && E >= emin && E <= emax;
                if (__any_sync(0xffffffffu, in_cube)) {
                    float v = 0.f;
#pragma unroll
                    for (int t = 0; t < 6; ++t) {
                        float w[4];
                        tet_w(T[t], E, w);
#pragma unroll
                        for (int r = 0; r < 4; ++r) v = fmaf(bs[t][r], w[r], v);
                    }
                    if (in_cube) q = __float2ll_rn(v) - q_lo;
                }
                // q = high 2^24 + low, low in [0, 2^24): sums of 32 fit 32 bits
                const long long sum = ((long long)__reduce_add_sync(0xffffffffu, (int)(q >> 24)) << 24) +
                                      (long long)__reduce_add_sync(0xffffffffu, (unsigned)(q & 0xFFFFFF));
                if (lane == j) acc += sum;
            }
        }
    }
    __syncthreads();
    if (lane < kPts && acc) atomicAdd(&s_sum[lane], (unsigned long long)acc);
    __syncthreads();
    if (tid < kPts && s_sum[tid]) atomicAdd(&S->sums[tid], s_sum[tid]);
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&S->ticket, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last || tid != 0) return;
    __threadfence();
    // the last block narrows the bracket to the sub-interval where N crosses
    // n_electrons (N does not decrease)
    const double unit = A.vtvg * ldexp(1.0, -kUnitBits);
    const long long base = first ? 0 : S->base;
    long long N[kPts];
    for (int j = 0; j < kPts; ++j) {
        N[j] = base + (long long)__ldcg(&S->sums[j]);
        S->sums[j] = 0ull;
    }
    S->ticket = 0;
    S->round = S->round + 1;
    const double top = (double)N[kPts - 1] * unit;
    if (first && (!(lo <= hi) || !(A.n_electrons >= 0.0) || A.n_electrons > top * (1.0 + 1e-6))) {
        S->bad = 1;
        S->done = 1;
        return;
    }
    int j = 0;
    while (j < kPts - 1 && (double)N[j] * unit < A.n_electrons) ++j;
    const float nlo = j == 0 ? lo : s_om[j - 1], nhi = s_om[j];
    S->base = j == 0 ? base : N[j - 1];
    S->lo = nlo;
    S->hi = nhi;
    // FP32 resolution reached: the bracket no longer shrinks
    if (!(nhi - nlo < hi - lo) || nhi <= nextafterf(nlo, INFINITY)) S->done = 1;
}

// The integrated-mode plan of a plan (same grid and orbitals, default box): a
// plan without one has no Fermi level.
tetra_status_t integrated_plan(const Plan &P, Plan &Q) {
    tetra_desc_t d = P.d;
    d.mode = TETRA_INTEGRATED;
    d.n_omega = 64;
    int box[3];
    default_box(d, box);
    return plan_init(Q, d, P.device, box, 1, false);
}

// Tile of at most 128 cubes with at most kTilePoints points whose values fit
// the shared memory: long rows in x, for the warps' 32 cubes.
void choose_tile(const Plan &P, FermiArgs &A) {
    A.tx = std::min(32, P.d.n1);
    A.ty = std::min(2, P.d.n2);
    A.tz = std::min(2, P.d.n3);
    while (A.tx * A.ty * A.tz < 128 && A.ty < P.d.n2 && (A.tx + 1) * (A.ty + 2) * (A.tz + 1) <= kTilePoints) ++A.ty;
    while (A.tx * A.ty * A.tz < 128 && A.tz < P.d.n3 && (A.tx + 1) * (A.ty + 1) * (A.tz + 2) <= kTilePoints) ++A.tz;
}

template <typename WT>
cudaError_t launch_round(const FermiArgs &A, int grid, size_t smem, cudaStream_t stream) {
    cudaError_t e = cudaFuncSetAttribute(fermi_round_kernel<WT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    for (int r = 0; r < kRoundsPerSync; ++r) fermi_round_kernel<WT><<<grid, kFermiThreads, smem, stream>>>(A);
    return cudaGetLastError();
}

}  // namespace

size_t fermi_workspace(const Plan &P) {
    Plan Q;
    if (integrated_plan(P, Q) != TETRA_OK) return 0;
    return kStatusBytes + sizeof(FermiState);
}

tetra_status_t fermi_level(const Plan &P, const float *eps, const void *w, double n_electrons, float *ef,
                           void *ws, size_t ws_bytes, cudaStream_t stream) {
    if (P.z0 != 0 || P.z1 != P.d.n3) return TETRA_EUNSUPPORTED;   // the count needs the whole grid
    Plan Q;
    const tetra_status_t st = integrated_plan(P, Q);
    if (st != TETRA_OK) return st;
    if (ws_bytes < kStatusBytes + sizeof(FermiState)) return TETRA_ENOMEM;
    FermiArgs A;
    A.n1 = P.d.n1; A.n2 = P.d.n2; A.n3 = P.d.n3; A.nx = P.nx; A.ny = P.ny;
    A.nb = P.d.n_bands; A.n_orb = P.d.n_orb; A.eps_stride = P.eps_stride; A.w_stride = P.w_stride;
    A.n_electrons = n_electrons;
    A.vtvg = 1.0 / (6.0 * (double)P.d.n1 * (double)P.d.n2 * (double)P.d.n3);
    A.eps = eps; A.w = w;
    A.S = reinterpret_cast<FermiState *>(static_cast<unsigned char *>(ws) + kStatusBytes);
    choose_tile(P, A);
    A.ntx = (A.n1 + A.tx - 1) / A.tx;
    A.nty = (A.n2 + A.ty - 1) / A.ty;
    A.n_tiles = A.ntx * A.nty * ((A.n3 + A.tz - 1) / A.tz);
    const size_t smem = 2 * sizeof(float) * (size_t)(A.tx + 1) * (A.ty + 1) * (A.tz + 1) * A.nb;
    if (smem > P.smem_optin - 1024) return TETRA_EUNSUPPORTED;
    const int grid = std::min(A.n_tiles, 3 * P.sm_count);
    if (cudaMemsetAsync(ws, 0, kStatusBytes + sizeof(FermiState), stream) != cudaSuccess) return TETRA_ECUDA;
    const long n_vec = (long)P.nx * P.ny * P.nz * (P.eps_stride / 4);
    band_range_kernel<<<(int)std::min<long>((n_vec + 255) / 256, 8L * P.sm_count), 256, 0, stream>>>(
        reinterpret_cast<const float4 *>(eps), n_vec, P.eps_stride / 4, P.d.n_bands, A.S);
    if (cudaGetLastError() != cudaSuccess) return TETRA_ECUDA;
    FermiState h;
    std::memset(&h, 0, sizeof h);
    for (int round = 0; round < kRounds && !h.done; round += kRoundsPerSync) {
        const cudaError_t e = P.d.weight_dtype == TETRA_F16    ? launch_round<__half>(A, grid, smem, stream)
                              : P.d.weight_dtype == TETRA_BF16 ? launch_round<__nv_bfloat16>(A, grid, smem, stream)
                                                               : launch_round<float>(A, grid, smem, stream);
        if (e != cudaSuccess || cudaMemcpyAsync(&h, A.S, sizeof h, cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
            cudaStreamSynchronize(stream) != cudaSuccess)
            return TETRA_ECUDA;
    }
    if (h.bad) return TETRA_EINVAL;
    *ef = 0.5f * (h.lo + h.hi);
    return TETRA_OK;
}

}  // namespace tetra

extern "C" size_t tetra_fermi_workspace_bytes(tetra_plan_t plan) {
    if (!plan) return 0;
    return tetra::fermi_workspace(*plan);
}

extern "C" tetra_status_t tetra_fermi_level(tetra_plan_t plan, const float *eps, const void *w, double n_electrons,
                                            float *ef, void *ws, size_t ws_bytes, cudaStream_t stream) {
    if (!plan || !eps || !w || !ef || !ws) return TETRA_EINVAL;
    if ((reinterpret_cast<uintptr_t>(eps) & 15u) || (reinterpret_cast<uintptr_t>(w) & 15u) ||
        (reinterpret_cast<uintptr_t>(ws) & 15u))
        return TETRA_EINVAL;
    const tetra::DeviceGuard dg(plan->device);
    if (!dg.ok()) return TETRA_ECUDA;
    return tetra::fermi_level(*plan, eps, w, n_electrons, ef, ws, ws_bytes, stream);
}
