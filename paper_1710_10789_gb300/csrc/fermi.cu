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
// One block takes tiles of cubes. It stages the band energies of the tile's
// points in shared memory, lists the (cube, band) items that reach the bracket
// (a few percent from the second round on), stages the summed weights of their
// bands, and hands the items out 32 at a time, kPer energies to a task, so
// that warps are full and all of them have work (a warp per row of 32 cubes,
// active or not, took 4.8 ms at the size below). An energy that no lane's
// cube contains is skipped by a vote: below a cube nothing, above it the full
// weight. The corner weights need no energy cases (tet_common.cuh). Each
// cube's N(E) - N(lo) is rounded once to an integer of 2^-26 of a full
// tetrahedron, summed over the warp by two 32-bit reductions, over the
// block's warps and over the grid by integer adds: exact in any order. Weights
// so large that the 64-bit sums could wrap (corner sums above 1.3 at 1024^3
// points and 8 bands, 7 10^5 on a small grid) are scaled down by a power of
// two: the first round, which stages every weight, finds the largest and is
// then repeated.
//
// At 95 x 97 x 96 points, 8 bands and 8 orbitals the five rounds of the
// integrated-mode DOS kernel before (64 energies, every orbital, every
// tetrahedron) took 14.4 ms (9.5 ms with its weights without cases); these
// take 1.9 ms, of which the first, which every tetrahedron reaches, 0.9 ms.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "tet_common.cuh"

namespace tetra {

namespace {

constexpr int kPts = 16;           // energies per round: bracket / 16
constexpr int kPer = 4;            // energies per task
constexpr int kRounds = 64;        // at most; FP32 resolution takes about five
constexpr int kRoundsPerSync = 6;
constexpr int kFermiThreads = 256;
constexpr int kFermiBlocks = 3;    // per SM

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
    long long base, top;       // N(lo), N(hi) in units
    int guess;                 // whether the round's energies cluster about the interpolated level
    int round, done, bad;      // bad: no such count, or no valid band energy
    int drop;                  // weights are staged times 2^-drop
    unsigned wmax;             // largest finite |weight sum| of a corner (a float's bits), before the scaling
    int range;                 // a weight was not finite (and taken as zero)
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
    int tx, lty, ltz;        // tile of cubes: tx (at most 31: a row of its points is a warp), 2^lty, 2^ltz
    int ntx, nty, n_tiles;
    double n_electrons, vtvg;
    const float *eps;
    const void *w;
    FermiState *S;
    int *status;
};

// Energy j of a round, ascending to hi: equidistant, or about the level that
// the line through N(lo) and N(hi) gives, at distances shrinking to 2^-16 of
// the bracket. N is smooth on the scale of a small bracket, so the crossing
// lies close to that level and a round narrows the bracket by far more than
// 16 (three rounds less in eight at 95 x 97 x 96); a round that narrows it by
// less than 8 is followed by an equidistant one.
__device__ __forceinline__ float round_energy(float lo, float hi, bool guess, float level, int j) {
    if (j == kPts - 1) return hi;
    const float h = hi - lo;
    if (!guess) return lo + h * ((float)(j + 1) * (1.0f / kPts));
    constexpr int kMid = kPts / 2 - 1;
    const int k = j < kMid ? kMid - j : j - kMid;   // distance from the middle: 1 nearest
    const float d = k == 0 ? 0.f : h * exp2f(-16.f + 2.25f * (float)(k - 1));
    return fminf(fmaxf(j < kMid ? level - d : level + d, lo), hi);
}

// Sum of n_orb weights, 16 bytes at a time where they fill whole vectors (the
// rows of the layout start on 16-byte boundaries).
template <typename WT>
__device__ __forceinline__ float sum_weights(const WT *b, int n_orb, bool vec) {
    float t = 0.f;
    if (vec) {
        constexpr int V = 16 / sizeof(WT);
        for (int s = 0; s < n_orb; s += V) {
            const uint4 q = *reinterpret_cast<const uint4 *>(b + s);
            const WT *e = reinterpret_cast<const WT *>(&q);
#pragma unroll
            for (int v = 0; v < V; ++v) t += to_f32<WT>(e[v]);
        }
    } else {
        for (int s = 0; s < n_orb; ++s) t += to_f32<WT>(b[s]);
    }
    return t;
}

template <typename WT>
__global__ void __launch_bounds__(kFermiThreads, kFermiBlocks) fermi_round_kernel(const FermiArgs A) {
    extern __shared__ float s_pt[];   // energies, then summed weights, [band][ps]; items
    __shared__ unsigned long long s_sum[kPts];
    __shared__ float s_om[kPts];
    __shared__ unsigned s_band[2][2];   // bands with an item, of two tiles in turn
    __shared__ int s_count[2];          // items, of two tiles in turn
    __shared__ int s_last;
    __shared__ float s_scale;           // 2^-drop
    __shared__ unsigned s_wmax;         // first pass: wmax of the block
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int nwarp = kFermiThreads / 32;
    FermiState *S = A.S;
    const bool first = S->round == 0;
    const int drop = S->drop;
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
    if (tid == 0) {
        s_scale = exp2f((float)-drop);
        s_wmax = 0u;
    }
    if (tid < kPts) {
        s_sum[tid] = 0ull;
        const bool guess = !first && S->guess;
        float level = lo;
        if (guess) {   // (one thread group; FP64 is slow but this is a few operations)
            const double below = (double)S->base, above = (double)S->top;
            const double n = A.n_electrons / (A.vtvg * ldexp(1.0, drop - kFermiBits));
            level = lo + (hi - lo) * (float)((n - below) / (above - below));
        }
        s_om[tid] = round_energy(lo, hi, guess, level, tid);
    }
    // tile points (x, row) at 32 row + x, band by band: a warp reads and
    // writes consecutive words
    const int ty = 1 << A.lty, tz = 1 << A.ltz, py = ty + 1, rows = py * (tz + 1), ps = rows * 32 + 1;
    const int lcol = A.lty + A.ltz;   // log2 of the (y, z) columns
    float *se = s_pt, *sw = s_pt + A.nb * ps;
    unsigned short *item = reinterpret_cast<unsigned short *>(sw + A.nb * ps);   // (band, column, x)
    const float fq = (float)(1 << kFermiBits) * 0.25f;
    const WT *W = static_cast<const WT *>(A.w);
    const bool vec = (A.n_orb * sizeof(WT)) % 16 == 0;
    // an item's first corner in the tile
    auto point_of = [&](int it) {
        const int col = (it >> 5) & ((1 << lcol) - 1), cy = col & (ty - 1), cz = col >> A.lty;
        return (it >> (5 + lcol)) * ps + (it & 31) + 32 * (cy + py * cz);
    };
    const int dy = 32, dz = 32 * py;
    long long acc = 0;   // lane j: this warp's sum at energy j
    int par = 0;
    for (int tile = blockIdx.x; tile < A.n_tiles; tile += gridDim.x, par ^= 1) {
        const int bx = tile % A.ntx, by = (tile / A.ntx) % A.nty, bz = tile / (A.ntx * A.nty);
        const int x0 = bx * A.tx, y0 = by << A.lty, z0 = bz << A.ltz;
        const bool in_x = lane <= A.tx && x0 + lane <= A.n1;
        if (tid < 2) s_band[par][tid] = 0u;
        if (tid == 2) s_count[par] = 0;
        __syncthreads();   // the previous tile is read
        for (int r = warp; r < rows; r += nwarp) {
            const int y = min(y0 + r % py, A.n2), z = min(z0 + r / py, A.n3);
            const float4 *src = reinterpret_cast<const float4 *>(
                A.eps + (x0 + lane + (long)A.nx * (y + (long)A.ny * z)) * A.eps_stride);
#pragma unroll 2
            for (int v = 0; v < A.eps_stride / 4; ++v) {
                const float4 q = in_x ? src[v] : make_float4(0.f, 0.f, 0.f, 0.f);
                float *o = se + 4 * v * ps + r * 32 + lane;
                o[0] = q.x;
                if (4 * v + 1 < A.nb) o[ps] = q.y;
                if (4 * v + 2 < A.nb) o[2 * ps] = q.z;
                if (4 * v + 3 < A.nb) o[3 * ps] = q.w;
            }
        }
        __syncthreads();
        for (int q = warp; q < A.nb << lcol; q += nwarp) {
            const int n = q >> lcol, it = q * 32 + lane, col = q & ((1 << lcol) - 1);
            const int p = point_of(it);
            bool act = false;
            if (lane < A.tx && x0 + lane < A.n1 && y0 + (col & (ty - 1)) < A.n2 && z0 + (col >> A.lty) < A.n3) {
                float emin = INFINITY, emax = -INFINITY;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float e = se[p + (k & 1) + ((k >> 1) & 1) * dy + (k >> 2) * dz];
                    emin = fminf(emin, e);
                    emax = fmaxf(emax, e);
                }
                act = emax >= lo && emin <= hi;
            }
            const unsigned m = __ballot_sync(0xffffffffu, act);
            if (!m) continue;
            int base = 0;
            if (lane == 0) {
                base = atomicAdd(&s_count[par], __popc(m));
                atomicOr(&s_band[par][n >> 5], 1u << (n & 31));
            }
            base = __shfl_sync(0xffffffffu, base, 0);
            if (act) item[base + __popc(m & ((1u << lane) - 1u))] = (unsigned short)it;
        }
        __syncthreads();
        const int count = s_count[par];
        if (count == 0) continue;
        unsigned long long bands = ((unsigned long long)s_band[par][1] << 32) | s_band[par][0];
        unsigned wmax = 0u;
        while (bands) {
            const int n = __ffsll((long long)bands) - 1;
            bands &= bands - 1;
#pragma unroll 2
            for (int r = warp; r < rows; r += nwarp) {
                const int y = min(y0 + r % py, A.n2), z = min(z0 + r / py, A.n3);
                if (in_x) {
                    float t = sum_weights<WT>(
                        W + (x0 + lane + (long)A.nx * (y + (long)A.ny * z)) * A.w_stride + n * A.n_orb, A.n_orb, vec);
                    if (!(fabsf(t) < INFINITY)) {
                        t = 0.f;
                        S->range = 1;
                    }
                    wmax = max(wmax, __float_as_uint(fabsf(t)));
                    sw[n * ps + r * 32 + lane] = t * s_scale;
                }
            }
        }
        if (first) {
            wmax = __reduce_max_sync(0xffffffffu, wmax);
            if (lane == 0) atomicMax(&s_wmax, wmax);
        }
        __syncthreads();
        const int groups = (count + 31) >> 5;
        for (int task = warp; task < groups * (kPts / kPer); task += nwarp) {
            const int g = task % groups, j0 = (task / groups) * kPer;
            const bool act = g * 32 + lane < count;
            const int p = point_of(item[act ? g * 32 + lane : 0]);
            float e[8], b[8];
            float emin = INFINITY, emax = -INFINITY;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int o = p + (k & 1) + ((k >> 1) & 1) * dy + (k >> 2) * dz;
                e[k] = se[o];
                b[k] = sw[o];
                emin = fminf(emin, e[k]);
                emax = fmaxf(emax, e[k]);
            }
            // which of the task's energies some lane's cube contains, and whether
            // some lane's cube holds lo: without either no tetrahedron is set up
            float E[kPer];
            bool in[kPer], any[kPer], some = __any_sync(0xffffffffu, act && lo > emin);
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                E[j] = s_om[j0 + j];
                in[j] = act && E[j] >= emin && E[j] <= emax;
                any[j] = __any_sync(0xffffffffu, in[j]);
                some = some || any[j];
            }
            float at_lo = 0.f, v[kPer];
#pragma unroll
            for (int j = 0; j < kPer; ++j) v[j] = 0.f;
            if (some) {
                // one tetrahedron after another; the sums run in the same order for
                // every energy, so a cube's value at an energy does not depend on the
                // bracket it is asked in
#pragma unroll
                for (int t = 0; t < 6; ++t) {
                    float es[4], bs[4], w[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int c = (tet_code(t) >> (3 * k)) & 7;
                        es[k] = e[c];
                        bs[k] = b[c];
                    }
                    sort4(es, bs);
                    Tet T;
                    tet_setup<TETRA_INTEGRATED>(T, es[0], es[1], es[2], es[3], fq);
                    tet_w(T, lo, w);
#pragma unroll
                    for (int k = 0; k < 4; ++k) at_lo = fmaf(bs[k], w[k], at_lo);
#pragma unroll
                    for (int j = 0; j < kPer; ++j) {
                        if (!any[j]) continue;
                        tet_w(T, E[j], w);
#pragma unroll
                        for (int k = 0; k < 4; ++k) v[j] = fmaf(bs[k], w[k], v[j]);
                    }
                }
            }
            // all six full: a corner counts once for each tetrahedron that has it
            float full = 0.f;
#pragma unroll
            for (int t = 0; t < 6; ++t)
#pragma unroll
                for (int k = 0; k < 4; ++k) full += fq * b[(tet_code(t) >> (3 * k)) & 7];
            const long long q_lo = __float2ll_rn(at_lo), q_full = __float2ll_rn(full);
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                // (a flat tetrahedron at E is empty there: only above emax all is full)
                const long long q = act ? (in[j] ? __float2ll_rn(v[j]) : (E[j] > emax ? q_full : 0)) - q_lo : 0;
                // q = high 2^24 + low, low in [0, 2^24): sums of 32 fit 32 bits
                const long long sum = ((long long)__reduce_add_sync(0xffffffffu, (int)(q >> 24)) << 24) +
                                      (long long)__reduce_add_sync(0xffffffffu, (unsigned)(q & 0xFFFFFF));
                if (lane == j0 + j) acc += sum;
            }
        }
    }
    __syncthreads();
    if (lane < kPts && acc) atomicAdd(&s_sum[lane], (unsigned long long)acc);
    __syncthreads();
    if (tid < kPts && s_sum[tid]) atomicAdd(&S->sums[tid], s_sum[tid]);
    if (first && tid == 0) atomicMax(&S->wmax, s_wmax);
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&S->ticket, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last || tid != 0) return;
    __threadfence();
    // the last block narrows the bracket to the sub-interval where N crosses
    // n_electrons (N does not decrease)
    const double unit = A.vtvg * ldexp(1.0, drop - kFermiBits);
    const long long base = first ? 0 : S->base;
    long long N[kPts];
    for (int j = 0; j < kPts; ++j) {
        N[j] = base + (long long)__ldcg(&S->sums[j]);
        S->sums[j] = 0ull;
    }
    S->ticket = 0;
    if (first && drop == 0) {
        const int d = fermi_drop(__uint_as_float(__ldcg(&S->wmax)), (double)A.n1 * A.n2 * A.n3 * A.nb);
        if (d > 0) {   // the sums may have wrapped: the round again
            S->drop = d;
            return;
        }
    }
    S->round = S->round + 1;
    if (__ldcg(&S->range)) atomicOr(A.status, kFlagRange);
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
    S->top = N[j];
    S->guess = (nhi - nlo) * 8.f <= hi - lo && S->top > S->base;
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

// Shared memory of a tile: energies and summed weights of its points, items.
size_t tile_bytes(const FermiArgs &A) {
    const int ty = 1 << A.lty, tz = 1 << A.ltz;
    return A.nb * (2 * sizeof(float) * ((size_t)(ty + 1) * (tz + 1) * 32 + 1) + sizeof(unsigned short) * 32 * ty * tz);
}

// Rows of nearly equal length in x, up to 4 x 4 columns as long as three
// blocks share an SM's shared memory (at most 70 KB: 64 bands, one column).
void choose_tile(const Plan &P, FermiArgs &A) {
    A.ntx = (P.d.n1 + 30) / 31;
    A.tx = (P.d.n1 + A.ntx - 1) / A.ntx;
    A.lty = P.d.n2 >= 4 ? 2 : P.d.n2 >= 2 ? 1 : 0;
    A.ltz = P.d.n3 >= 4 ? 2 : P.d.n3 >= 2 ? 1 : 0;
    while (tile_bytes(A) > 70 * 1024 && A.lty + A.ltz > 0) --(A.lty > A.ltz ? A.lty : A.ltz);
    A.nty = (P.d.n2 + (1 << A.lty) - 1) >> A.lty;
    A.n_tiles = A.ntx * A.nty * ((P.d.n3 + (1 << A.ltz) - 1) >> A.ltz);
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
    A.status = reinterpret_cast<int *>(ws);
    choose_tile(P, A);
    const size_t smem = tile_bytes(A);
    const int grid = std::min(A.n_tiles, kFermiBlocks * P.sm_count);
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
