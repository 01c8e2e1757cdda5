// Forward kernel of the linear tetrahedron orbital-resolved DOS
// (arXiv:1710.10789, Sec. II.C weights, Eqs. (8)-(9)) for sm_103a.
//
// Work decomposition
//  * The cube grid [0,n1) x [0,n2) x [z0,z1) is cut into boxes of BX*BY*BZ
//    cubes. A persistent CTA walks a sequence of boxes and, for each, has the
//    box's (BX+1)(BY+1)(BZ+1) corner points of all bands (energies and orbital
//    weights, tetra layout) copied into shared memory by two 4-D TMA loads:
//    the energies double buffered across boxes, the weights (read only by the
//    walks) in one slot loaded behind the next box's window pass. One model: boxes blockIdx.x, blockIdx.x +
//    gridDim.x, ... (blockIdx.y = energy chunk). A batch of models: each CTA
//    claims the next (model, box) item from a global counter (models in
//    order), so the work stays balanced whatever the models' costs; when the
//    model changes the CTA flushes its tile into that model's int64
//    accumulator with integer atomics and reloads the energy grid.
//  * One thread handles one item: it reads the corner energies and orbital
//    weights, sorts the energies (Sec. II.C sorts E1 <= E2 <= E3 <= E4), and
//    visits only the energies strictly inside (E1, E4) (bins overlapping it in
//    bin mode); all others get zero weight. With more than 8 orbitals the item
//    is a (tetrahedron, band).
//  * Up to 8 orbitals (every mode): the item is a pair of tetrahedra sharing
//    a face (Table I's six form three such pairs). Their windows overlap
//    heavily, so one walk over the union of the two windows adds both
//    tetrahedra's contributions at each energy before touching the shared
//    tile: about half the shared-memory traffic of one tetrahedron each.
//    (Integrated mode: beyond the union the pair puts one saturation step.)
//  * Items of a box are ranked by window length (counting sort), so the 32
//    lanes of a warp walk windows of nearly equal length.
//  * Each visited energy adds sum_l b_{l,s} dw_l to the CTA's tile for every
//    orbital s (Eq. (8)).
//
// Accumulation: exact fixed point, no float atomics anywhere
//  * Contributions are scaled by 1/u, u = (V_T/V_G) / dE * 2^-F (dE = mean
//    grid spacing, F = fixed_bits), rounded to integers and added with integer
//    shared-memory atomics into an int32 tile [energies][n_orb + 1]. Integer
//    addition is associative, so the tile does not depend on thread order.
//  * The rounding adds 1.5 * 2^23 in FP32 and the tile receives the raw bit
//    pattern, i.e. the integer plus the constant bias M = 0x4B400000. The
//    extra column of each tile row counts (as differences: +1 at a window's
//    first energy, -1 after its last) how many adds the row received, so a
//    row's value is recovered modulo 2^32 as raw - count * M when it is
//    flushed.
//  * A per-item bound q_max (|b| <= Bmax of the box, and the tetrahedron DOS
//    is at most 3/E41 of V_T/V_G) decides between this fast path and a 64-bit
//    global integer path for tetrahedra flat on the scale of the grid: few on a
//    fine grid, many where the grid has about as many energies as points a
//    side. The sum of q_max over processed items bounds every tile entry; the
//    tile is flushed into the int64 accumulator in global memory before it
//    could overflow.
//  * The CTAs flush into one int64 accumulator (integer atomics: exact, any
//    order); the CTA that finishes last scales it by u. For a batch a second
//    kernel scales each model's accumulator. Where the global path may take
//    many items of few energies (COPIES), all CTAs would add to the same few
//    addresses: the accumulator has up to 16 copies that they take in turn
//    (8 bands, one orbital of weight one: 64^3 points, 128 energies 0.99 ->
//    0.33 ms, 128^3, 256 energies 5.2 -> 2.4 ms). A kernel of its own, because
//    the code of the others' walks suffers from the few instructions more
//    (64^3 points, 8 orbitals, 2000 energies: 1.59 -> 1.67 ms).
//
// The instantiations of a mode are compiled in a file of their own
// (dos_point.cu, ...), so that they build in parallel.
#pragma once
#include <algorithm>
#include <atomic>
#include <memory>
#include <new>

#include "tet_common.cuh"

namespace tetra {

namespace fwd {

constexpr float kMagic = 12582912.0f;   // 1.5 * 2^23: float + kMagic rounds to an integer
constexpr int kMagicBits = 0x4B400000;  // bit pattern of kMagic
constexpr uint32_t kSmemAlign = 1024;
// Work unit, threads per CTA and registers per thread. With up to 8 orbitals
// a unit is a face-sharing tetrahedron pair, holding two tetrahedra's weights
// and constants in registers; 16 orbitals would not fit, so there a unit is
// one tetrahedron. Each of the SM's four sub-partitions has 16K registers for
// its warps: 16 warps can use 128 registers per thread. (A pair with 8
// orbitals fits them with ten constants per tetrahedron and five weight rows;
// 64^3 points, 8 bands, 2000 energies: 1742 us with 12 warps of 168 registers
// against 1670 us with 16, 1477 us with the five rows and 1408 us with 20
// warps of 96 registers; at 256^3 and 4000 energies, with the eigensolver,
// those are 57.1, 55.0, 50.5 and 52.0 ms. At 64^3 the kernel issues in 75 % of
// its cycles and uses 63 % of the shared-memory wavefronts: 3.5 of them for
// each add of 32 lanes to unrelated rows.)
constexpr int kThreads = 512;
constexpr int kMaxRegs = 128;
template <int NORB>
struct Cfg {
    static constexpr bool pairs = NORB <= 8;
    static constexpr int units_per_cube = pairs ? 3 : 6;
    // a pair's corner values added per corner before the projection
    // (merge_pair): 15 operations against 3 multiply-adds per orbital
    static constexpr bool merge = NORB >= 5;
    static constexpr int rows = merge ? 5 : 8;   // weight rows of a pair
};
constexpr int kKBins = 256;     // window-length histogram bins (K >= 255 share one)

// Table I's tetrahedra as three face-sharing pairs: (1st, 2nd), (3rd, 5th),
// (4th, 6th). Per pair five corner labels minus one: the three corners of the
// shared face, the corner only in the first tetrahedron, the corner only in
// the second. First tetrahedron = slots {0,1,2,3}, second = slots {0,1,2,4}.
constexpr int kPair[3][5] = {{1, 2, 5, 0, 3}, {2, 4, 5, 0, 6}, {2, 5, 7, 3, 6}};
constexpr uint32_t pack_pair(int p) {
    return (uint32_t)(kPair[p][0] | kPair[p][1] << 3 | kPair[p][2] << 6 | kPair[p][3] << 9 |
                      kPair[p][4] << 12);
}
constexpr uint64_t kPairCode = (uint64_t)pack_pair(0) | (uint64_t)pack_pair(1) << 16 |
                               (uint64_t)pack_pair(2) << 32;
__device__ __forceinline__ uint32_t pair_code(int p) { return (uint32_t)(kPairCode >> (16 * p)) & 0x7FFFu; }

// Launch constants shared by every model of a launch.
struct FwdArgs {
    int nb, n_orb;
    int BX, BY, BZ;
    int lbx, lby, lbz;   // log2 of the box sides (powers of two)
    int eps_stride, w_stride;
    uint32_t e_box_bytes, w_box_bytes;   // TMA bytes of a box's energies / weights
    uint32_t e_stage, w_stage;           // their shared-memory slots (128-byte multiples)
    int chunk_w;         // energies per shared tile (largest model of a batch)
    int tile_copies;     // copies of the tile; lane l of a bin-mode pair adds into copy l % tile_copies
    int items_per_box;   // items per box: (pair, band), with more than 8 orbitals (tetrahedron, band)
    int split;           // log2 of the lanes that share a pair's walk (point and integrated mode)
    int fast_cap;
    unsigned flush_at;   // a 64-energy block is flushed once its bound reaches this
    long long *G;        // int64 accumulators, [slot][copy][n_orb][chunk_w]; slot = chunk, or model of a batch
    long long *Gs;       // integrated mode: int64 accumulators of the step sums, the same shape
    int *status;
    int *queue;          // batched: next unclaimed (model, box) work item
    int *done;           // single model: CTAs that have flushed, [kDoneGroups] (chunk % kDoneGroups)
    float *dos;          // single model: the result, written by the CTA that finishes a chunk
};

// Fixed-point unit, identical in every kernel that uses it, and fq, V_T/(4 V_G)
// in units. The DOS modes scale with the mean energy spacing (their values are
// per energy); the integrated occupation is dimensionless, so its unit does
// not depend on the grid (a narrow grid, as in a Fermi-level search, keeps full
// resolution). The unit is what makes fq exact: fq is the float that the
// kernel multiplies with, and its rounding would shift every value by up to
// 6e-8.
__device__ __forceinline__ double fixed_unit(const float *omega, int n_omega, int mode, double vtvg,
                                             int bits, float &fq) {
    double de;
    if (mode == TETRA_INTEGRATED)
        de = 1.0;
    else if (mode != TETRA_BIN)
        de = n_omega > 1 ? ((double)omega[n_omega - 1] - (double)omega[0]) / (n_omega - 1) : 1.0;
    else
        de = ((double)omega[n_omega] - (double)omega[0]) / n_omega;
    if (!(de > 0.0)) de = 1.0;
    fq = (float)(0.25 * ldexp(de, bits));
    return 0.25 * vtvg / (double)fq;
}

// One rounded contribution added to the CTA's int64 partial (global 64-bit
// integer atomics): the path of the rare items whose bound does not fit the
// int32 tile. acc holds the dithered value; the same single rounding to
// nearest as the tile path.
__device__ __forceinline__ void deposit_one(float acc, long long *g, int *status) {
    if (fabsf(acc) < 9.0e18f) {
        const long long q = __float2ll_rn(acc);
        if (q != 0) atomicAdd(reinterpret_cast<unsigned long long *>(g), static_cast<unsigned long long>(q));
    } else {
        atomicOr(status, kFlagRange);
    }
}

// Dither offset in [-1/2, 1/2) for one (tetrahedron, band) item, hashed from its
// global identity so it does not depend on the launch shape.
__device__ __forceinline__ float item_dither(uint32_t key) {
    uint32_t h = key * 0x9E3779B9u;
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    return (float)(h >> 8) * (1.0f / 16777216.0f) - 0.5f;
}

// floor(a / d) for 0 <= a and 0 < d below 2^24: a float quotient corrected
// by one step (the TMA issue at the end of a box sits on every thread's path
// to the next barrier, so it avoids integer division).
__device__ __forceinline__ int fdivq(int a, int d) {
    int q = (int)__fdividef((float)a, (float)d);
    q -= (q * d > a) ? 1 : 0;
    q += ((q + 1) * d <= a) ? 1 : 0;
    return q;
}

__device__ __forceinline__ float safe_rcp(float x) { return x > 0.f ? __fdividef(1.0f, x) : 0.f; }

// Adds one energy's contribution of an item directly to the CTA's int64
// partial (global integer atomics): the path of the rare items whose bound
// does not fit the int32 tile. Same dithered single rounding as the tile path:
// round(c + delta - 1/2) with delta in [0,1) hashed from the item.
template <int NORB>
__device__ __forceinline__ void deposit_slow(const float (&b)[4][NORB], const float d[4], int n_orb,
                                             float dith, long long *gcol, int g_stride, int *status) {
#pragma unroll
    for (int s = 0; s < NORB; ++s) {
        if (s < n_orb) {
            float acc = fmaf(b[0][s], d[0], dith);
            acc = fmaf(b[1][s], d[1], acc);
            acc = fmaf(b[2][s], d[2], acc);
            acc = fmaf(b[3][s], d[3], acc);
            if (fabsf(acc) < 9.0e18f) {
                const long long q = __float2ll_rn(acc);
                if (q != 0)
                    atomicAdd(reinterpret_cast<unsigned long long *>(gcol + (long)s * g_stride),
                              static_cast<unsigned long long>(q));
            } else {
                atomicOr(status, kFlagRange);
            }
        }
    }
}

// Energy window of one item, as global indices clipped to this CTA's chunk
// [w0, w0+wc): point mode, energies strictly inside (e1, e4); bin mode, bins
// whose weight difference can be non-zero (upper edge > e1, and lower edge
// < e4 or <= e1). The estimate from the mean spacing is corrected against the
// cached grid, so any ascending grid gives the exact window.
template <int MODE>
__device__ __forceinline__ void item_window(float e1, float e4, const float *om, int w0, int wc,
                                            float om0, float inv_de, int n_omega, int &lo, int &hi) {
    const float flo = fminf(fmaxf((e1 - om0) * inv_de, -2.f), (float)n_omega + 2.f);
    const float fhi = fminf(fmaxf((e4 - om0) * inv_de, -2.f), (float)n_omega + 2.f);
    if (MODE != TETRA_BIN) {
        lo = min(max((int)floorf(flo) + 1, w0), w0 + wc);
        hi = max(min((int)ceilf(fhi) - 1, w0 + wc - 1), w0 - 1);
        while (lo > w0 && om[lo - 1 - w0] > e1) --lo;
        while (lo < w0 + wc && om[lo - w0] <= e1) ++lo;
        while (hi < w0 + wc - 1 && om[hi + 1 - w0] < e4) ++hi;
        while (hi >= w0 && om[hi - w0] >= e4) --hi;
    } else {
        lo = min(max((int)floorf(flo), w0), w0 + wc);
        hi = max(min((int)ceilf(fhi), w0 + wc - 1), w0 - 1);
        while (lo > w0 && om[lo - w0] > e1) --lo;
        while (lo < w0 + wc && om[lo + 1 - w0] <= e1) ++lo;
        while (hi < w0 + wc - 1 && (om[hi + 1 - w0] < e4 || om[hi + 1 - w0] <= e1)) ++hi;
        while (hi >= w0 && !(om[hi - w0] < e4 || om[hi - w0] <= e1)) --hi;
    }
}

// A tetrahedron of a pair: its own corner's energy x merged into the sorted
// face (e, ascending), and where it lies (below face corner j).
struct PairOrder {
    float e[4];
    bool below[3];
    __device__ __forceinline__ PairOrder(const float (&f)[3], float x) {
        e[0] = fminf(x, f[0]);
        e[1] = fmaxf(f[0], fminf(x, f[1]));
        e[2] = fmaxf(f[1], fminf(x, f[2]));
        e[3] = fmaxf(f[2], x);
#pragma unroll
        for (int j = 0; j < 3; ++j) below[j] = x < f[j];
    }
    // the points of the sorted corners: p[0..2] the face's, x the own one
    __device__ __forceinline__ void place(const int *p, int x, int (&o)[4]) const {
        o[0] = below[0] ? x : p[0];
        o[1] = below[0] ? p[0] : (below[1] ? x : p[1]);
        o[2] = below[1] ? p[1] : (below[2] ? x : p[2]);
        o[3] = below[2] ? p[2] : x;
    }
};

// Corner values of a pair's two tetrahedra (each in its own sorted order)
// added per corner: the face's three, then the two own corners. 15 selects
// and adds that save 3 n_orb multiply-adds of the projection and 3 n_orb
// registers. With few orbitals (8 rows) they stay apart.
__device__ __forceinline__ void merge_pair(const PairOrder &A, const PairOrder &B, const float (&a)[4],
                                           const float (&b)[4], float (&d)[5]) {
#pragma unroll
    for (int j = 0; j < 3; ++j) d[j] = (A.below[j] ? a[j + 1] : a[j]) + (B.below[j] ? b[j + 1] : b[j]);
    d[3] = A.below[1] ? (A.below[0] ? a[0] : a[1]) : (A.below[2] ? a[2] : a[3]);
    d[4] = B.below[1] ? (B.below[0] ? b[0] : b[1]) : (B.below[2] ? b[2] : b[3]);
}
__device__ __forceinline__ void merge_pair(const PairOrder &, const PairOrder &, const float (&a)[4],
                                           const float (&b)[4], float (&d)[8]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        d[j] = a[j];
        d[4 + j] = b[j];
    }
}

// One model of a launch: grid, energy grid and where its partial sums go.
struct ModelP {
    int n1, n2, n3, z0, z1, nbx, nby, n_boxes, n_omega;
    int fixed_bits;
    int box_base;    // first global work index of the model (batched launches)
    int copies;      // copies of its accumulator (COPIES): CTA b adds into copy b % copies
    double vtvg;
    const float *omega;
};

struct MapPair {   // CUtensorMap is 128-byte aligned
    CUtensorMap e, w;
};

// Per-launch model table, passed by value (kernel parameter space).
template <int MAXM>
struct Batch {
    MapPair maps[MAXM];
    ModelP m[MAXM];
    int n_models;
    int total_work;   // batched: (model, box) items of the launch
};

template <int NORB, typename WT, int MODE, int MAXM, bool COPIES>
__global__ void __maxnreg__(kMaxRegs)
    tetra_dos_fwd_kernel(const __grid_constant__ Batch<MAXM> B, const FwdArgs A) {
    // tile row: NORB orbitals, and the row's add count (differences) behind
    // them or, for odd NORB, in an array after the rows: the odd row length
    // spreads consecutive rows over the shared-memory banks
    constexpr int TS = NORB | 1;
    // one orbital, point and bin mode: items of zero weight dropped before the ranking
    constexpr bool kFilter = NORB == 1 && MODE != TETRA_INTEGRATED;
    auto count_of = [&](int *t, int row) -> int & {
        return (NORB & 1) ? t[TS * (A.chunk_w + 1) + row] : t[row * TS + NORB];
    };
    extern __shared__ unsigned char smem_raw[];
    // TMA destinations need an aligned base; the dynamic area starts after the
    // static variables, so align it here (the host reserves kSmemAlign bytes).
    unsigned char *smem = smem_raw + ((kSmemAlign - (smem_u32(smem_raw) & (kSmemAlign - 1))) &
                                      (kSmemAlign - 1));
    const int tid = threadIdx.x;
    const int chunk = blockIdx.y;   // energy chunk (single-model launches)
    // shared memory carve-up
    // energies of two boxes (pass A of box k+1 needs no weights) and the
    // weights of one box, refilled after pass B and loaded while the next
    // box's pass A and ranking run
    unsigned char *estage[2] = {smem, smem + A.e_stage};
    unsigned char *wstage = smem + 2 * A.e_stage;
    int *tile = reinterpret_cast<int *>(wstage + A.w_stage);   // [copies][chunk_w + 1][NORB + 1]
    // (copies only for single-model bin-mode pairs; elsewhere one, known at
    // compile time: the batched kernel measured faster without them)
    constexpr bool kCopies = MODE == TETRA_BIN && Cfg<NORB>::pairs && MAXM == 1;
    const int n_copies = kCopies ? A.tile_copies : 1, copy_ints = (NORB + 1) * (A.chunk_w + 1);
    // integrated mode: per-orbital sums of the saturated weights of the items
    // whose (larger) E4 lies between energy j-1 and j, [chunk_w][NORB] (plain integers)
    int *stile = tile + copy_ints * n_copies;
    float *om = reinterpret_cast<float *>(stile + (MODE == TETRA_INTEGRATED ? NORB * A.chunk_w : 0));
    float *iw = om + A.chunk_w + 1;                                   // 1/bin width (bin mode)
    unsigned *blk_bound = reinterpret_cast<unsigned *>(iw + (MODE == TETRA_BIN ? A.chunk_w : 0));
    const int n_blk = (A.chunk_w + 63) >> 6;
    // (one set of block bounds per tile copy: copy c's bounds at c * n_blk)
    short *s_lo = reinterpret_cast<short *>(blk_bound + n_blk * n_copies);   // window start - w0
    unsigned short *s_K = reinterpret_cast<unsigned short *>(s_lo + A.items_per_box);
    unsigned short *s_list = s_K + A.items_per_box;                 // items sorted by K
    int *khist = reinterpret_cast<int *>(
        (reinterpret_cast<uintptr_t>(s_list + A.items_per_box) + 15) & ~uintptr_t(15));
    int *kcursor = khist + kKBins;           // rank cursors per window length
    uint64_t *mbar = reinterpret_cast<uint64_t *>(
        (reinterpret_cast<uintptr_t>(kcursor + kKBins) + 15) & ~uintptr_t(15));
    __shared__ float red_f[kThreads / 32];
    __shared__ int s_wsum[kThreads / 32];
    __shared__ int s_abort, s_active, s_slot;
    __shared__ float s_fq, s_unit[2];   // of the current model
    __shared__ int s_cdelta[8];   // staged-box point offset of cube corner c
    __shared__ int n_issued[3];   // TMA loads issued per mbarrier (thread 0 keeps them)

    // self-check of the shared-memory carve-up against the launch's dynamic size
    {
        const uintptr_t need = reinterpret_cast<uintptr_t>(mbar + 3) - reinterpret_cast<uintptr_t>(smem_raw);
        const bool bad = need > dynamic_smem_bytes() || (smem_u32(estage[0]) & 127u) != 0 ||
                         (A.e_stage & 127u) != 0 || (A.w_stage & 127u) != 0 || A.e_box_bytes > A.e_stage ||
                         A.w_box_bytes > A.w_stage || (smem_u32(mbar) & 7u) != 0 || A.items_per_box > 65535 ||
                         (MAXM > 1 && n_blk > (int)blockDim.x);   // (a batch's flush: a thread per block)
        if (bad) {
            if (tid == 0) atomicOr(A.status, kFlagConfig);
            return;
        }
    }
    if (tid < 8)
        s_cdelta[tid] = (tid & 1) + (A.BX + 1) * (((tid >> 1) & 1) + (A.BY + 1) * (tid >> 2));
    if (tid == 0) {
        s_abort = 0;
        mbar_init(&mbar[0], 1);   // energies, stage 0
        mbar_init(&mbar[1], 1);   // energies, stage 1
        mbar_init(&mbar[2], 1);   // weights
        n_issued[0] = n_issued[1] = n_issued[2] = 0;
        fence_mbar_init();
    }

    // Work sequence of this CTA: item k -> (model, box). Single model: boxes
    // blockIdx.x, blockIdx.x + gridDim.x, ... Batched: thread 0 claims global
    // items (models in order, boxes within a model) from a counter, two steps
    // ahead, so every CTA stays busy until the batch is done; the claim for
    // step k+2 is issued when step k starts and decoded when step k ends (its
    // latency hidden behind the box), and s_wm / s_wb hold the decoded
    // (model, box) of steps k .. k+2 (model -1: no more work).
    __shared__ int s_wm[4], s_wb[4];
    int claim_m = 0;   // thread 0: model of its last claim (claims only grow)
    auto store_claim = [&](int k, int g) {   // thread 0 only
        if (g >= B.total_work) {
            s_wm[k & 3] = -1;
            return;
        }
        while (claim_m + 1 < B.n_models && B.m[claim_m + 1].box_base <= g) ++claim_m;
        s_wm[k & 3] = claim_m;
        s_wb[k & 3] = g - B.m[claim_m].box_base;
    };
    auto work = [&](int k, int &mi, int &box) -> bool {
        if (MAXM == 1) {
            mi = 0;
            box = blockIdx.x + k * gridDim.x;
            return box < B.m[0].n_boxes;
        }
        mi = s_wm[k & 3];
        box = s_wb[k & 3];
        return mi >= 0;
    };
    // energies of work item k (already claimed) into energy stage stg
    auto issue_e = [&](int k, int stg) {   // thread 0 only
        int mi, box;
        if (!work(k, mi, box)) return;
        const ModelP &Mk = B.m[mi];
        const int bq = fdivq(box, Mk.nbx), iz = fdivq(bq, Mk.nby), ix = box - bq * Mk.nbx, iy = bq - iz * Mk.nby;
        ++n_issued[stg];
        mbar_arrive_expect_tx(&mbar[stg], A.e_box_bytes);
        tma_load_4d(estage[stg], &B.maps[mi].e, 0, ix * A.BX, iy * A.BY, Mk.z0 + iz * A.BZ, &mbar[stg]);
    };
    // weights of work item k (already claimed) into the weight stage
    auto issue_w = [&](int k) {   // thread 0 only
        int mi, box;
        if (!work(k, mi, box)) return;
        const ModelP &Mk = B.m[mi];
        const int bq = fdivq(box, Mk.nbx), iz = fdivq(bq, Mk.nby), ix = box - bq * Mk.nbx, iy = bq - iz * Mk.nby;
        ++n_issued[2];
        mbar_arrive_expect_tx(&mbar[2], A.w_box_bytes);
        tma_load_4d(wstage, &B.maps[mi].w, 0, ix * A.BX, iy * A.BY, Mk.z0 + iz * A.BZ, &mbar[2]);
    };
    __syncthreads();
    // prologue: energies of the first two work items, weights of the first
    if (tid == 0) {
        if (MAXM > 1) {
            store_claim(0, atomicAdd(A.queue, 1));
            store_claim(1, atomicAdd(A.queue, 1));
        }
        issue_e(0, 0);
        issue_e(1, 1);
        issue_w(0);
    }
    int g_next = 0;   // thread 0: the claim in flight (step k+2)
    __syncthreads();

    const int PX = A.BX + 1, PY = A.BY + 1;
    const int ncube = A.BX * A.BY * A.BZ;   // a power of two
    const int lcube = A.lbx + A.lby + A.lbz;

    // state of the model whose boxes are being accumulated
    int cur = -1, w0 = 0, wc = 0;
    float fq = 0.f, om0 = 0.f, inv_de = 0.f, max_iw = 0.f;
    long long *Gc = A.G;
    // The count column of rows 0..wc: differences (as the walks update it)
    // to per-row add counts by a block-wide inclusive scan, and back. Each
    // warp scans a segment of rows; segment totals are combined through
    // shared memory. Called by every thread of the CTA.
    auto counts_from_diffs = [&](int *tile) {
        const int nw = (int)(blockDim.x >> 5), warp = tid >> 5, lane = tid & 31;
        const int nr = wc + 1;
        const int seg = ((nr + nw - 1) / nw + 31) & ~31;
        const int r0 = warp * seg, r1 = min(r0 + seg, nr);
        int carry = 0;
        for (int r = r0; r < r1; r += 32) {
            const int rr = r + lane;
            int x = rr < r1 ? count_of(tile, rr) : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            x += carry;
            if (rr < r1) count_of(tile, rr) = x;
            carry = __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) s_wsum[warp] = carry;
        __syncthreads();
        int off = 0;
        for (int w2 = 0; w2 < warp; ++w2) off += s_wsum[w2];
        if (off != 0)
            for (int rr = r0 + lane; rr < r1; rr += 32) count_of(tile, rr) += off;
        __syncthreads();
    };
    auto diffs_from_counts = [&](int *tile) {
        const int nw = (int)(blockDim.x >> 5), warp = tid >> 5, lane = tid & 31;
        const int nr = wc + 1;
        const int seg = ((nr + nw - 1) / nw + 31) & ~31;
        const int r0 = warp * seg, r1 = min(r0 + seg, nr);
        // the count before the segment belongs to another warp: read it first
        const int prev0 = (r0 > 0 && r0 < r1) ? count_of(tile, r0 - 1) : 0;
        __syncthreads();
        if (r1 > r0) {
            // chunks last to first, so each chunk's predecessor is still a count
            for (int r = r0 + (((r1 - r0 - 1) >> 5) << 5); r >= r0; r -= 32) {
                const int rr = r + lane;
                const int x = rr < r1 ? count_of(tile, rr) : 0;
                int pv = __shfl_up_sync(0xffffffffu, x, 1);
                if (lane == 0) pv = (r == r0) ? prev0 : count_of(tile, r - 1);
                if (rr < r1) count_of(tile, rr) = x - pv;
            }
        }
        __syncthreads();
    };
    // Value of a tile entry since its last flush: raw sum minus count * M
    // (modulo 2^32; the bounds keep the true value below 2^31 in magnitude).
    auto entry_value = [&](int *tile, int j, int s) -> int {
        const unsigned n_add = (unsigned)count_of(tile, j);
        return (int)((unsigned)tile[j * TS + s] - n_add * (unsigned)kMagicBits);
    };
    // the entry's value summed over the tile's copies
    auto entry_total = [&](int j, int s) -> int {
        int v = 0;
        for (int c = 0; c < n_copies; ++c) v += entry_value(tile + c * copy_ints, j, s);
        return v;
    };
    // moves the int32 tile of the current model into its int64 partial slot
    long long *Gsc = A.Gs;
    auto flush_tile = [&]() {
        for (int c = 0; c < n_copies; ++c) counts_from_diffs(tile + c * copy_ints);
        for (int i = tid; i < A.n_orb * wc; i += blockDim.x) {
            const int s = i / wc, j = i - s * wc;
            const int v = entry_total(j, s);
            if (v)
                atomicAdd(reinterpret_cast<unsigned long long *>(Gc + (long)s * A.chunk_w + j),
                          static_cast<unsigned long long>(static_cast<long long>(v)));
            if (MODE == TETRA_INTEGRATED) {
                const int sv = stile[j * NORB + s];
                if (sv)
                    atomicAdd(reinterpret_cast<unsigned long long *>(Gsc + (long)s * A.chunk_w + j),
                              static_cast<unsigned long long>(static_cast<long long>(sv)));
            }
        }
    };

    for (int k = 0;; ++k) {
        int mi, box;
        if (!work(k, mi, box)) break;
        if (MAXM > 1 && tid == 0) g_next = atomicAdd(A.queue, 1);
        const ModelP &M = B.m[mi];
        if (mi != cur) {
            // switch model: flush the previous one, reset the tile, cache the energy grid
            if (cur >= 0) flush_tile();
            __syncthreads();
            cur = mi;
            w0 = (MAXM == 1) ? chunk * A.chunk_w : 0;
            wc = min(A.chunk_w, M.n_omega - w0);
            // accumulator: one per energy chunk of a single model, one per model
            // of a batch (CTAs flush into it with integer atomics)
            long slot = (MAXM == 1) ? (long)chunk : (long)mi;
            if constexpr (COPIES) slot = slot * M.copies + blockIdx.x % M.copies;
            Gc = A.G + slot * (long)A.n_orb * A.chunk_w;
            if (MODE == TETRA_INTEGRATED) Gsc = A.Gs + slot * (long)A.n_orb * A.chunk_w;
            for (int i = tid; i < copy_ints * n_copies; i += blockDim.x) tile[i] = 0;
            if (MODE == TETRA_INTEGRATED)
                for (int i = tid; i < NORB * A.chunk_w; i += blockDim.x) stile[i] = 0;
            for (int i = tid; i < n_blk * n_copies; i += blockDim.x) blk_bound[i] = 0;
            const int n_om = (MODE != TETRA_BIN) ? wc : wc + 1;
            for (int i = tid; i < n_om; i += blockDim.x) om[i] = M.omega[w0 + i];
            __syncthreads();
            if (MODE == TETRA_BIN)
                for (int i = tid; i < wc; i += blockDim.x) iw[i] = 1.0f / (om[i + 1] - om[i]);
            if (tid == 0) {
                unit_pair(fixed_unit(M.omega, M.n_omega, MODE, M.vtvg, M.fixed_bits, s_fq), s_unit[0], s_unit[1]);
            }
            om0 = M.omega[0];
            const float omN = (MODE != TETRA_BIN) ? M.omega[M.n_omega - 1] : M.omega[M.n_omega];
            inv_de = (MODE != TETRA_BIN) ? (M.n_omega > 1 ? (float)(M.n_omega - 1) / (omN - om0) : 0.f)
                                           : (float)M.n_omega / (omN - om0);
            if (MODE == TETRA_BIN) {
                // the narrowest bin of the whole grid bounds every bin contribution
                max_iw = 0.f;
                for (int i = tid; i < M.n_omega; i += blockDim.x)
                    max_iw = fmaxf(max_iw, 1.0f / (M.omega[i + 1] - M.omega[i]));
                for (int o = 16; o; o >>= 1) max_iw = fmaxf(max_iw, __shfl_xor_sync(0xffffffffu, max_iw, o));
                if ((tid & 31) == 0) red_f[tid >> 5] = max_iw;
                __syncthreads();
                max_iw = 0.f;
                for (int i = 0; i < (int)(blockDim.x >> 5); ++i) max_iw = fmaxf(max_iw, red_f[i]);
            }
            __syncthreads();
            fq = s_fq;
        }
        const int st = k & 1;
        for (int i = tid; i < kKBins; i += blockDim.x) khist[i] = 0;
        if (tid == 0) s_slot = 0;
        const bool ok = mbar_wait_bounded(&mbar[st], (k >> 1) & 1, A.status);
        if (__syncthreads_or(!ok)) {
            s_abort = 1;
            break;
        }
        const float *Es = reinterpret_cast<const float *>(estage[st]);
        const WT *Ws = reinterpret_cast<const WT *>(wstage);
        const int ix = box % M.nbx, iy = (box / M.nbx) % M.nby, iz = box / (M.nbx * M.nby);
        const int gx0 = ix * A.BX, gy0 = iy * A.BY, gz0 = M.z0 + iz * A.BZ;
        const int lane = tid & 31, warp = tid >> 5, nwarp = (int)(blockDim.x >> 5);


        // Pass A: window of every item (corner min / max only) and a histogram
        // of its length K, so that pass B can hand items of similar length to
        // the same warp. The integers an item adds do not depend on which thread
        // adds them, so the grouping cannot change the result.
        // Each thread takes up to four items at once: their windows are
        // independent, so the corner loads and window searches of the four
        // overlap instead of running one after another.
        {
            constexpr int U = 4;
            const int stride_w = nwarp * 32;
            for (int base0 = warp * 32; base0 < A.items_per_box; base0 += stride_w * U) {
                int Ku[U], lou[U];
#pragma unroll
                for (int uu = 0; uu < U; ++uu) {
                    const int it = base0 + uu * stride_w + lane;
                    // integrated mode: an item also counts when only its step (the
                    // first energy at or above E4) lies in the chunk; items off the
                    // grid get lo = w0 + wc, which makes them inactive
                    int K = 0, lo = (MODE == TETRA_INTEGRATED) ? w0 + wc : 0;
                    if (it < A.items_per_box) {
                        constexpr bool PAIRS = Cfg<NORB>::pairs;
                        constexpr int UPC = Cfg<NORB>::units_per_cube;
                        const int cube = it & (ncube - 1);
                        const int rest = it >> lcube;
                        const int t = rest % UPC, n = rest / UPC;
                        const int cx = cube & (A.BX - 1), cy = (cube >> A.lbx) & (A.BY - 1), cz = cube >> (A.lbx + A.lby);
                        if (gx0 + cx < M.n1 && gy0 + cy < M.n2 && gz0 + cz < M.z1) {
                            // a pair's window is the union of its two tetrahedra's:
                            // the window of the min / max over its five corners
                            float e1 = 3.0e38f, e4 = -3.0e38f;
                            bool flat_face = false;
                            const uint32_t code = PAIRS ? pair_code(t) : tet_code(t);
                            const int p0 = cx + PX * (cy + PY * cz);
#pragma unroll
                            for (int q = 0; q < (PAIRS ? 5 : 4); ++q) {
                                if (q == 3) flat_face = e1 == e4;   // of a pair: corners 0..2
                                const int p = p0 + s_cdelta[(code >> (3 * q)) & 7];
                                const float ev = Es[p * A.eps_stride + n];
                                e1 = fminf(e1, ev);
                                e4 = fmaxf(e4, ev);
                            }
                            int hi;
                            item_window<MODE>(e1, e4, om, w0, wc, om0, inv_de, M.n_omega, lo, hi);
                            // a flat tetrahedron at a pair's upper end is empty at an
                            // energy (bin edge) equal to it: in integrated mode there
                            // the walk, not the pair's step; in bin mode the bin above
                            // takes its whole step
                            if (MODE != TETRA_POINT && PAIRS && flat_face)
                                while (hi < w0 + wc - 1 && om[hi + 1 - w0] <= e4) ++hi;
                            K = max(0, hi - lo + 1);
                        }
                    }
                    Ku[uu] = K;
                    lou[uu] = lo;
                }
#pragma unroll
                for (int uu = 0; uu < U; ++uu) {
                    const int it = base0 + uu * stride_w + lane;
                    const int K = Ku[uu], lo = lou[uu];
                    if (it < A.items_per_box) {
                        s_lo[it] = (short)(lo - w0);
                        s_K[it] = (unsigned short)K;
                    }
                    const bool act = it < A.items_per_box && (K > 0 || (MODE == TETRA_INTEGRATED && lo + K < w0 + wc));
                    if constexpr (MODE == TETRA_INTEGRATED && Cfg<NORB>::pairs) {
                        // items with an empty window (only a step: every tetrahedron
                        // below the chunk) all count in bin 0, one add per warp
                        const unsigned zm = __ballot_sync(0xffffffffu, act && K == 0);
                        if (act && K > 0) atomicAdd(&khist[min(K, kKBins - 1)], 1);
                        if (zm && lane == __ffs(zm) - 1) atomicAdd(&khist[0], __popc(zm));
                    } else {
                        if (!kFilter && act) atomicAdd(&khist[min(K, kKBins - 1)], 1);
                    }
                }
            }
        }
        if constexpr (kFilter) {
            // The box's weights, waited for here instead of before pass B: items
            // whose weights are all zero are dropped (every contribution rounds
            // to zero, the dither being at most 1/2) before the ranking counts
            // the others, so that the warps stay full. Two thirds of a
            // susceptibility's transition bands have both ends occupied or both
            // empty.
            if (mbar_wait_bounded(&mbar[2], k & 1, A.status))
                for (int it = tid; it < A.items_per_box; it += blockDim.x) {
                    const int K = s_K[it];
                    if (K == 0) continue;
                    const int cube = it & (ncube - 1), rest = it >> lcube;
                    const int cx = cube & (A.BX - 1), cy = (cube >> A.lbx) & (A.BY - 1), cz = cube >> (A.lbx + A.lby);
                    const int n = rest / 3, p0 = cx + PX * (cy + PY * cz);
                    const uint32_t code = pair_code(rest - 3 * n);
                    bool any = false;
#pragma unroll
                    for (int q = 0; q < 5; ++q) {
                        const int p = p0 + s_cdelta[(code >> (3 * q)) & 7];
                        any = any || to_f32<WT>(Ws[(long)p * A.w_stride + n]) != 0.f;
                    }
                    if (any) atomicAdd(&khist[min(K, kKBins - 1)], 1);
                    else s_K[it] = 0;
                }
        }
        __syncthreads();
        // Items ranked by window length K: an exclusive scan of the K histogram
        // gives each length its first rank; an item's rank = first rank + its
        // place among items of equal K (atomic cursor; items of equal K are
        // interchangeable).
        if (tid < 32) {
            constexpr int PER = kKBins / 32;
            int v[PER], sum = 0;
#pragma unroll
            for (int j = 0; j < PER; ++j) { v[j] = khist[tid * PER + j]; sum += v[j]; }
            int x = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (tid >= o) x += y;
            }
            int run = x - sum;
#pragma unroll
            for (int j = 0; j < PER; ++j) { kcursor[tid * PER + j] = run; run += v[j]; }
            if (tid == 31) s_active = x;
        }
        __syncthreads();
        for (int base = warp * 32; base < A.items_per_box; base += nwarp * 32) {
            const int it = base + lane;
            const int K = it < A.items_per_box ? (int)s_K[it] : 0;
            const bool act = it < A.items_per_box &&
                             (K > 0 || (MODE == TETRA_INTEGRATED && s_lo[it] + K < wc));
            if constexpr (MODE == TETRA_INTEGRATED && Cfg<NORB>::pairs) {
                // empty windows: consecutive ranks from one cursor add per warp
                const unsigned zm = __ballot_sync(0xffffffffu, act && K == 0);
                if (act && K > 0) s_list[atomicAdd(&kcursor[min(K, kKBins - 1)], 1)] = (unsigned short)it;
                if (zm) {
                    const int lead = __ffs(zm) - 1;
                    int zb = 0;
                    if (lane == lead) zb = atomicAdd(&kcursor[0], __popc(zm));
                    zb = __shfl_sync(0xffffffffu, zb, lead);
                    if (act && K == 0) s_list[zb + __popc(zm & ((1u << lane) - 1u))] = (unsigned short)it;
                }
            } else {
                if (act) s_list[atomicAdd(&kcursor[min(K, kKBins - 1)], 1)] = (unsigned short)it;
            }
        }
        // the box's weights (loaded while pass A and the ranking ran), and
        // Bmax = max |w| over them (all of the box, padding included, so it
        // bounds every orbital weight an item can read)
        const bool okw = mbar_wait_bounded(&mbar[2], k & 1, A.status);
        float bmax = 0.f;
        if (okw) {
            const int n16 = (int)(A.w_box_bytes >> 4);
            const uint4 *src = reinterpret_cast<const uint4 *>(wstage);
            for (int i = tid; i < n16; i += blockDim.x) {
                const uint4 v = src[i];
                const uint32_t wv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (sizeof(WT) == 4) {
                        bmax = fmaxf(bmax, fabsf(__uint_as_float(wv[q])));
                    } else {
                        const WT lo = *reinterpret_cast<const WT *>(&wv[q]);
                        const WT hi = *(reinterpret_cast<const WT *>(&wv[q]) + 1);
                        bmax = fmaxf(bmax, fmaxf(fabsf(to_f32<WT>(lo)), fabsf(to_f32<WT>(hi))));
                    }
                }
            }
        }
        for (int o = 16; o; o >>= 1) bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
        if (lane == 0) red_f[warp] = bmax;
        if (__syncthreads_or(!okw)) {
            s_abort = 1;
            break;
        }
        bmax = 0.f;
        for (int i = 0; i < nwarp; ++i) bmax = fmaxf(bmax, red_f[i]);
        const int n_active = s_active;
        // (lanes per pair: bin mode walks in order, 16 orbitals have one tetrahedron)
        const int ls = MODE != TETRA_BIN && Cfg<NORB>::pairs ? A.split : 0;
        const int n_slots = ((n_active << ls) + 31) >> 5;

        // Pass B: slot q holds the 32 items of ranks 32q .. 32q+31 (nearly equal
        // window length, so a warp's lanes finish together). Warps claim slots
        // longest windows first (a shared counter), which balances the warps'
        // work before the end-of-box barrier.
        for (;;) {
            int claim = 0;
            if (lane == 0) claim = atomicAdd(&s_slot, 1);
            claim = __shfl_sync(0xffffffffu, claim, 0);
            if (claim >= n_slots) break;
            const int pos = (n_slots - 1 - claim) * 32 + lane;
            const bool valid = pos < (n_active << ls);
            const int it = valid ? (int)s_list[pos >> ls] : 0;
            const int part = pos & ((1 << ls) - 1);   // this lane takes the window's energies part, part + 2^ls, ...
            const int cube = it & (ncube - 1);
            const int rest = it >> lcube;
            const int cx = cube & (A.BX - 1), cy = (cube >> A.lbx) & (A.BY - 1), cz = cube >> (A.lbx + A.lby);
            const int p0 = cx + PX * (cy + PY * cz);
            const int lo = valid ? w0 + s_lo[it] : w0;
            const int hi = valid ? lo + s_K[it] - 1 : w0 - 1;
            const uint32_t gcube = (uint32_t)(gx0 + cx) +
                                   (uint32_t)M.n1 * ((uint32_t)(gy0 + cy) + (uint32_t)M.n2 * (uint32_t)(gz0 + cz));
            if constexpr (Cfg<NORB>::pairs) {
                // integrated mode: the lanes that hold an item, for the warp sums of
                // the steps on the chunk's first energy
                const unsigned vmask = (MODE == TETRA_INTEGRATED) ? __ballot_sync(0xffffffffu, valid) : 0u;
                if (!valid) continue;
                // ---- a pair of tetrahedra sharing a face, walked over the union window
                const int pr = rest % 3, n = rest / 3;
                const uint32_t code = pair_code(pr);
                // the face's three corners sorted, the first and the second
                // tetrahedron's own corner merged into that order
                float es[3];
                int ps[5];
#pragma unroll
                for (int q = 0; q < 5; ++q) ps[q] = p0 + s_cdelta[(code >> (3 * q)) & 7];
#pragma unroll
                for (int q = 0; q < 3; ++q) es[q] = Es[ps[q] * A.eps_stride + n];
                cswap(es[0], es[1], ps[0], ps[1]);
                cswap(es[1], es[2], ps[1], ps[2]);
                cswap(es[0], es[1], ps[0], ps[1]);
                const PairOrder oa(es, Es[ps[3] * A.eps_stride + n]), ob(es, Es[ps[4] * A.eps_stride + n]);
                const float (&ea)[4] = oa.e, (&eb)[4] = ob.e;
                // weights: of the face's corners and the two own ones, or of each
                // tetrahedron's corners in its sorted order
                constexpr int ROWS = Cfg<NORB>::rows;
                float bw[ROWS][NORB];
                if constexpr (Cfg<NORB>::merge) {
#pragma unroll
                    for (int q = 0; q < 5; ++q)
                        load_weights<NORB, WT>(Ws + (long)ps[q] * A.w_stride + n * A.n_orb, A.n_orb, bw[q]);
                } else {
                    int pa[4], pb[4];
                    oa.place(ps, ps[3], pa);
                    ob.place(ps, ps[4], pb);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        load_weights<NORB, WT>(Ws + (long)pa[q] * A.w_stride + n * A.n_orb, A.n_orb, bw[q]);
                        load_weights<NORB, WT>(Ws + (long)pb[q] * A.w_stride + n * A.n_orb, A.n_orb, bw[ROWS - 4 + q]);
                    }
                }
                // both tetrahedra's corner values (rows of bw) of orbital s, dithered
                auto project = [&](const float (&d)[ROWS], int s, float dith) {
                    float acc = fmaf(bw[0][s], d[0], dith);
#pragma unroll
                    for (int q = 1; q < ROWS; ++q) acc = fmaf(bw[q][s], d[q], acc);
                    return acc;
                };
                const float dith = item_dither((gcube * 3u + (uint32_t)pr) * (uint32_t)A.nb + (uint32_t)n);
                if constexpr (MODE == TETRA_INTEGRATED) {
                    // Occupation: the walk over the union window adds both
                    // tetrahedra's weights (saturated above a tetrahedron's own
                    // E4); from the first energy beyond it on, the pair's step
                    // fq sum_l b_l of both enters through the step tile.
                    // Every corner weight is at most V_T/(4 V_G): the pair adds
                    // at most 8 fq Bmax to any entry.
                    const float qmax = bmax * 8.f * fq * 1.01f;
                    const bool fast = qmax < (float)A.fast_cap;
                    // the first energy beyond the window (a flat pair, E1 = E4, is
                    // empty at E = E1: lo is above E1)
                    const int hs = hi + 1;
                    const bool step = part == 0 && hs < w0 + wc;
                    // steps on the chunk's first energy (there go the steps of all
                    // tetrahedra below the chunk) are summed over the warp first
                    const bool first = fast && step && hs == w0;
                    const unsigned qbnd = fast ? (unsigned)qmax + 2u : 0u;
                    if (fast) {
                        if (hi >= lo && part == 0) {
                            for (int bk = (lo - w0) >> 6; bk <= ((hi - w0) >> 6); ++bk) atomicAdd(&blk_bound[bk], qbnd);
                            atomicAdd(&count_of(tile, lo - w0), 1);
                            atomicAdd(&count_of(tile, hi + 1 - w0), -1);
                        }
                        if (step && !first) atomicAdd(&blk_bound[(hs - w0) >> 6], qbnd);
                    }
                    Tet TA, TB;
                    tet_setup<MODE>(TA, ea[0], ea[1], ea[2], ea[3], fq);
                    tet_setup<MODE>(TB, eb[0], eb[1], eb[2], eb[3], fq);
                    // the pair's saturated contribution of orbital s
                    auto full = [&](int s) {
                        if constexpr (Cfg<NORB>::merge)
                            return fq * (2.f * ((bw[0][s] + bw[1][s]) + bw[2][s]) + (bw[3][s] + bw[4][s])) + dith;
                        else
                            return fq * (((bw[0][s] + bw[1][s]) + (bw[2][s] + bw[3][s])) +
                                         ((bw[ROWS - 4][s] + bw[ROWS - 3][s]) + (bw[ROWS - 2][s] + bw[ROWS - 1][s]))) + dith;
                    };
                    if (__any_sync(vmask, first)) {
                        // the warp's first-energy steps: integer sums, one add per orbital
                        const bool lead = lane == __ffs(vmask) - 1;
                        const unsigned bsum = __reduce_add_sync(vmask, first ? qbnd : 0u);
                        if (lead && bsum) atomicAdd(&blk_bound[0], bsum);
#pragma unroll
                        for (int s = 0; s < NORB; ++s) {
                            const int tot = __reduce_add_sync(vmask, first ? __float_as_int(full(s) + kMagic) - kMagicBits : 0);
                            if (lead && tot) atomicAdd(&stile[s], tot);
                        }
                    }
                    if (fast) {
                        const int K = (hi - lo - part + (1 << ls)) >> ls, i0 = lo + part, i1 = i0 + ((K - 1) << ls);
                        int i = i0 + (((lane * max(K, 1)) >> 5) << ls);
                        for (int j = 0; j < K; ++j) {
                            float wa[4], wb[4], d5[ROWS];
                            tet_w(TA, om[i - w0], wa);
                            tet_w(TB, om[i - w0], wb);
                            merge_pair(oa, ob, wa, wb, d5);
                            int *col = tile + (i - w0) * TS;
#pragma unroll
                            for (int s = 0; s < NORB; ++s) {
                                const float acc = project(d5, s, dith);
                                atomicAdd(col + s, __float_as_int(acc + kMagic));
                            }
                            i = (i == i1) ? i0 : i + (1 << ls);
                        }
                        if (step && !first) {
#pragma unroll
                            for (int s = 0; s < NORB; ++s)
                                atomicAdd(&stile[(hs - w0) * NORB + s], __float_as_int(full(s) + kMagic) - kMagicBits);
                        }
                    } else {
                        for (int i = lo + part; i <= hi; i += 1 << ls) {
                            float wa[4], wb[4], d5[ROWS];
                            tet_w(TA, om[i - w0], wa);
                            tet_w(TB, om[i - w0], wb);
                            merge_pair(oa, ob, wa, wb, d5);
#pragma unroll
                            for (int s = 0; s < NORB; ++s) {
                                if (s >= A.n_orb) continue;
                                const float acc = project(d5, s, dith);
                                deposit_one(acc, Gc + (long)s * A.chunk_w + (i - w0), A.status);
                            }
                        }
#pragma unroll
                        for (int s = 0; s < NORB; ++s) {
                            if (s >= A.n_orb) continue;
                            if (step) deposit_one(full(s), Gsc + (long)s * A.chunk_w + (hs - w0), A.status);
                        }
                    }
                    continue;
                }
                if constexpr (MODE == TETRA_BIN) {
                    // Bin averages: each tetrahedron's weight step over the bin
                    // divided by its width (zero below E1; above E4 the weights
                    // are saturated and their steps vanish), bins walked in
                    // order so each upper edge's weights serve the next bin.
                    float qmax = bmax * 8.f * fq * max_iw * 1.01f;
                    if (!(ea[3] > ea[0]) || !(eb[3] > eb[0])) qmax = 3.0e38f;
                    const bool fast = qmax < (float)A.fast_cap;
                    // this lane's copy of the tile and of its block bounds (the
                    // copies are summed when flushed)
                    const int cp = n_copies > 1 ? lane % n_copies : 0;
                    int *tl = tile + cp * copy_ints;
                    unsigned *bl = blk_bound + cp * n_blk;
                    if (fast && hi >= lo) {
                        const unsigned qbnd = (unsigned)qmax + 2u;
                        for (int bk = (lo - w0) >> 6; bk <= ((hi - w0) >> 6); ++bk) atomicAdd(&bl[bk], qbnd);
                        atomicAdd(&count_of(tl, lo - w0), 1);
                        atomicAdd(&count_of(tl, hi + 1 - w0), -1);
                    }
                    Tet TA, TB;
                    tet_setup<MODE>(TA, ea[0], ea[1], ea[2], ea[3], fq);
                    tet_setup<MODE>(TB, eb[0], eb[1], eb[2], eb[3], fq);
                    // (weights of both by corner, then differences)
                    auto both = [&](float E, float (&w5)[ROWS]) {
                        float wa[4], wb[4];
                        tet_w(TA, E, wa);
                        tet_w(TB, E, wb);
                        merge_pair(oa, ob, wa, wb, w5);
                    };
                    float wp[ROWS];
                    both(om[lo - w0], wp);
                    int *col = tl + (lo - w0) * TS;
                    for (int i = lo; i <= hi; ++i, col += TS) {
                        float wn[ROWS], d5[ROWS];
                        both(om[i + 1 - w0], wn);
                        const float sc = iw[i - w0];
#pragma unroll
                        for (int q = 0; q < ROWS; ++q) {
                            d5[q] = (wn[q] - wp[q]) * sc;
                            wp[q] = wn[q];
                        }
#pragma unroll
                        for (int s = 0; s < NORB; ++s) {
                            if (!fast && s >= A.n_orb) continue;
                            const float acc = project(d5, s, dith);
                            if (fast)
                                atomicAdd(col + s, __float_as_int(acc + kMagic));
                            else
                                deposit_one(acc, Gc + (long)s * A.chunk_w + (i - w0), A.status);
                        }
                    }
                    continue;
                }
                // bound on every |contribution| of the pair, in fixed-point units:
                // the tetrahedron DOS is at most 3/E41 of V_T/V_G; a flat
                // tetrahedron (E1 = E4) contributes nothing in point mode
                const float qa = (ea[3] > ea[0]) ? bmax * 4.f * fq * 3.1f * safe_rcp(ea[3] - ea[0]) : 0.f;
                const float qb = (eb[3] > eb[0]) ? bmax * 4.f * fq * 3.1f * safe_rcp(eb[3] - eb[0]) : 0.f;
                const float qmax = qa + qb;
                const bool fast = qmax < (float)A.fast_cap;
                if (fast && part == 0) {
                    const unsigned qbnd = (unsigned)qmax + 2u;
                    for (int bk = (lo - w0) >> 6; bk <= ((hi - w0) >> 6); ++bk) atomicAdd(&blk_bound[bk], qbnd);
                    atomicAdd(&count_of(tile, lo - w0), 1);
                    atomicAdd(&count_of(tile, hi + 1 - w0), -1);
                }
                Tet TA, TB;
                tet_setup<MODE>(TA, ea[0], ea[1], ea[2], ea[3], fq);
                tet_setup<MODE>(TB, eb[0], eb[1], eb[2], eb[3], fq);
                // one orbital: the weights' differences along the edges (tet_value)
                const TetDiff bda = tet_diff(bw[0][0], bw[1][0], bw[2][0], bw[3][0]);
                const TetDiff bdb = tet_diff(bw[ROWS - 4][0], bw[ROWS - 3][0], bw[ROWS - 2][0], bw[ROWS - 1][0]);
                if (fast) {
                    // lane-dependent start, wrapping walk (see below)
                    const int K = (hi - lo - part + (1 << ls)) >> ls, i0 = lo + part, i1 = i0 + ((K - 1) << ls);
                    int i = i0 + (((lane * K) >> 5) << ls);
                    for (int j = 0; j < K; ++j) {
                        int *col = tile + (i - w0) * TS;
                        if constexpr (NORB == 1) {
                            const float acc = tet_value(TA, om[i - w0], bda) + (tet_value(TB, om[i - w0], bdb) + dith);
                            atomicAdd(col, __float_as_int(acc + kMagic));
                        } else {
                            float da[4], db[4], d5[ROWS];   // zero outside a tetrahedron's own window
                            tet_dw(TA, om[i - w0], da);
                            tet_dw(TB, om[i - w0], db);
                            merge_pair(oa, ob, da, db, d5);
#pragma unroll
                            for (int s = 0; s < NORB; ++s) {
                                const float acc = project(d5, s, dith);
                                atomicAdd(col + s, __float_as_int(acc + kMagic));
                            }
                        }
                        i = (i == i1) ? i0 : i + (1 << ls);
                    }
                } else {
                    for (int i = lo + part; i <= hi; i += 1 << ls) {
                        if constexpr (NORB == 1) {   // (the same sum as the tile path)
                            const float acc = tet_value(TA, om[i - w0], bda) + (tet_value(TB, om[i - w0], bdb) + dith);
                            deposit_one(acc, Gc + (i - w0), A.status);
                            continue;
                        }
                        float da[4], db[4], d5[ROWS];   // zero outside a tetrahedron's own window
                        tet_dw(TA, om[i - w0], da);
                        tet_dw(TB, om[i - w0], db);
                        merge_pair(oa, ob, da, db, d5);
#pragma unroll
                        for (int s = 0; s < NORB; ++s) {
                            if (s >= A.n_orb) continue;
                            const float acc = project(d5, s, dith);
                            deposit_one(acc, Gc + (long)s * A.chunk_w + (i - w0), A.status);
                        }
                    }
                }
                continue;
            }
            const int t = rest % 6, n = rest / 6;
            float e[4];
            int p[4];
            const uint32_t code = tet_code(t);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                p[q] = p0 + s_cdelta[(code >> (3 * q)) & 7];
                e[q] = Es[p[q] * A.eps_stride + n];
            }
            sort4(e, p);
            float b[4][NORB];
#pragma unroll
            for (int r4 = 0; r4 < 4; ++r4)
                load_weights<NORB, WT>(Ws + (long)p[r4] * A.w_stride + n * A.n_orb, A.n_orb, b[r4]);
            // per-item bound on every |contribution|, in fixed-point units (the
            // tetrahedron DOS is at most 3/E41 of V_T/V_G; a bin average at most
            // its weight step over the narrowest bin)
            // (integrated mode: every corner weight is at most V_T/(4 V_G))
            float qmax = (MODE == TETRA_POINT) ? bmax * 4.f * fq * 3.1f * safe_rcp(e[3] - e[0])
                         : (MODE == TETRA_BIN) ? bmax * 4.f * fq * max_iw * 1.01f
                                               : bmax * 4.f * fq * 1.01f;
            if (!(e[3] > e[0]) && MODE != TETRA_INTEGRATED) qmax = 3.0e38f;
            const bool fast = qmax < (float)A.fast_cap;
            const float dith = item_dither((gcube * 6u + (uint32_t)t) * (uint32_t)A.nb + (uint32_t)n);
            if (!valid) continue;
            // integrated mode: the first energy at or above E4, where the item's
            // saturated weights enter the step tile (none if beyond the grid)
            const int hs = hi + 1;
            const bool step = MODE == TETRA_INTEGRATED && hs < w0 + wc;
            // Bookkeeping of the tile: every entry of blocks lo/64 .. hi/64 may
            // receive at most qmax from this item, and rows lo .. hi each receive
            // one add per orbital.
            if (fast) {
                const unsigned qbnd = (unsigned)qmax + 2u;
                if (hi >= lo) {
                    for (int bk = (lo - w0) >> 6; bk <= ((hi - w0) >> 6); ++bk) atomicAdd(&blk_bound[bk], qbnd);
                    atomicAdd(&count_of(tile, lo - w0), 1);
                    atomicAdd(&count_of(tile, hi + 1 - w0), -1);
                }
                if (step) atomicAdd(&blk_bound[(hs - w0) >> 6], qbnd);
            }
            if constexpr (MODE == TETRA_INTEGRATED) {
                Tet T;
                tet_setup<MODE>(T, e[0], e[1], e[2], e[3], fq);
                float bsum[NORB];   // saturated contribution: fq sum_l b_{l,s}
#pragma unroll
                for (int s = 0; s < NORB; ++s) bsum[s] = fq * ((b[0][s] + b[1][s]) + (b[2][s] + b[3][s]));
                if (fast) {
                    const int K = hi - lo + 1;
                    int i = lo + ((lane * max(K, 1)) >> 5);
                    for (int j = 0; j < K; ++j) {
                        float wl[4];
                        tet_w(T, om[i - w0], wl);
                        int *col = tile + (i - w0) * TS;
#pragma unroll
                        for (int s = 0; s < NORB; ++s) {
                            float acc = fmaf(b[0][s], wl[0], dith);
                            acc = fmaf(b[1][s], wl[1], acc);
                            acc = fmaf(b[2][s], wl[2], acc);
                            acc = fmaf(b[3][s], wl[3], acc);
                            atomicAdd(col + s, __float_as_int(acc + kMagic));
                        }
                        i = (i == hi) ? lo : i + 1;
                    }
                    if (step) {
#pragma unroll
                        for (int s = 0; s < NORB; ++s)
                            atomicAdd(&stile[(hs - w0) * NORB + s], __float_as_int(bsum[s] + dith + kMagic) - kMagicBits);
                    }
                } else {
                    for (int i = lo; i <= hi; ++i) {
                        float wl[4];
                        tet_w(T, om[i - w0], wl);
                        deposit_slow<NORB>(b, wl, A.n_orb, dith, Gc + (i - w0), A.chunk_w, A.status);
                    }
                    if (step) {
#pragma unroll
                        for (int s = 0; s < NORB; ++s)
                            if (s < A.n_orb) deposit_one(bsum[s] + dith, Gsc + (long)s * A.chunk_w + (hs - w0), A.status);
                    }
                }
                continue;
            }
            if constexpr (MODE == TETRA_POINT) {
                Tet TP;
                tet_setup<MODE>(TP, e[0], e[1], e[2], e[3], fq);
                if (fast) {
                    // The walk over the window starts at a lane-dependent offset
                    // and wraps: lanes whose windows coincide then add to
                    // different tile rows at each step instead of serialising on
                    // the same addresses. The sum does not depend on the order.
                    const int K = hi - lo + 1;
                    int i = lo + ((lane * K) >> 5);
                    for (int j = 0; j < K; ++j) {
                        float d[4];
                        tet_dw(TP, om[i - w0], d);
                        int *col = tile + (i - w0) * TS;
#pragma unroll
                        for (int s = 0; s < NORB; ++s) {
                            float acc = fmaf(b[0][s], d[0], dith);
                            acc = fmaf(b[1][s], d[1], acc);
                            acc = fmaf(b[2][s], d[2], acc);
                            acc = fmaf(b[3][s], d[3], acc);
                            atomicAdd(col + s, __float_as_int(acc + kMagic));
                        }
                        i = (i == hi) ? lo : i + 1;
                    }
                } else {
                    for (int i = lo; i <= hi; ++i) {
                        float d[4];
                        tet_dw(TP, om[i - w0], d);
                        deposit_slow<NORB>(b, d, A.n_orb, dith, Gc + (i - w0), A.chunk_w, A.status);
                    }
                }
            } else {
                Tet T;
                tet_setup<MODE>(T, e[0], e[1], e[2], e[3], fq);
                float wp[4];
                tet_w(T, om[lo - w0], wp);
                int *col = tile + (lo - w0) * TS;
                for (int i = lo; i <= hi; ++i, col += TS) {
                    float wn[4], d[4];
                    tet_w(T, om[i + 1 - w0], wn);
                    const float sc = iw[i - w0];
#pragma unroll
                    for (int r4 = 0; r4 < 4; ++r4) { d[r4] = (wn[r4] - wp[r4]) * sc; wp[r4] = wn[r4]; }
                    if (fast) {
#pragma unroll
                        for (int s = 0; s < NORB; ++s) {
                            float acc = fmaf(b[0][s], d[0], dith);
                            acc = fmaf(b[1][s], d[1], acc);
                            acc = fmaf(b[2][s], d[2], acc);
                            acc = fmaf(b[3][s], d[3], acc);
                            atomicAdd(col + s, __float_as_int(acc + kMagic));
                        }
                    } else {
                        deposit_slow<NORB>(b, d, A.n_orb, dith, Gc + (i - w0), A.chunk_w, A.status);
                    }
                }
            }
        }
        __syncthreads();   // every thread is done reading both slots and adding to the tile
        // refill: energies of work item k+2 into this energy stage, weights of k+1
        if (tid == 0) {
            fence_proxy_async_smem();
            if (MAXM > 1) store_claim(k + 2, g_next);
            issue_e(k + 2, st);
            issue_w(k + 1);
        }
        // A block whose bound reached flush_at is moved into the CTA's int64
        // partial before the next box: one box adds less than 2^30 - 2^20 to any
        // entry (per-unit cap x units per box), so entries stay below 2^31.
        // A flushed entry is reset to count * M, the raw value of zero.
        if constexpr (MAXM > 1) {
            // (the batched kernel: one tile copy; this form measured faster there)
            const bool mine = tid < n_blk && blk_bound[tid] >= A.flush_at;
            if (__syncthreads_or(mine)) {
                counts_from_diffs(tile);
                for (int bk = 0; bk < n_blk; ++bk) {
                    if (blk_bound[bk] < A.flush_at) continue;   // uniform: every thread reads the same value
                    const int j0 = bk << 6, jn = min(64, wc - j0);
                    for (int i = tid; i < A.n_orb * 64; i += blockDim.x) {
                        const int s = i >> 6, j = i & 63;
                        if (j >= jn) continue;
                        const int v = entry_value(tile, j0 + j, s);
                        if (v) {
                            atomicAdd(reinterpret_cast<unsigned long long *>(Gc + (long)s * A.chunk_w + j0 + j),
                                      static_cast<unsigned long long>(static_cast<long long>(v)));
                            tile[(j0 + j) * TS + s] = (int)((unsigned)count_of(tile, j0 + j) * (unsigned)kMagicBits);
                        }
                    }
                }
                __syncthreads();
                diffs_from_counts(tile);
                if (tid < n_blk && blk_bound[tid] >= A.flush_at) blk_bound[tid] = 0;
                __syncthreads();
            }
            continue;
        }
        bool mine = false;
        for (int i = tid; i < n_blk * n_copies; i += blockDim.x) mine = mine || blk_bound[i] >= A.flush_at;
        if (__syncthreads_or(mine)) {
            for (int c = 0; c < n_copies; ++c) {
                const unsigned *bc = blk_bound + c * n_blk;
                bool any = false;   // uniform: every thread reads the same values
                for (int bk = 0; bk < n_blk; ++bk) any = any || bc[bk] >= A.flush_at;
                if (!any) continue;
                int *tc = tile + c * copy_ints;
                counts_from_diffs(tc);
                for (int bk = 0; bk < n_blk; ++bk) {
                    if (bc[bk] < A.flush_at) continue;   // uniform
                    const int j0 = bk << 6, jn = min(64, wc - j0);
                    for (int i = tid; i < A.n_orb * 64; i += blockDim.x) {
                        const int s = i >> 6, j = i & 63;
                        if (j >= jn) continue;
                        const int v = entry_value(tc, j0 + j, s);
                        if (v) {
                            atomicAdd(reinterpret_cast<unsigned long long *>(Gc + (long)s * A.chunk_w + j0 + j),
                                      static_cast<unsigned long long>(static_cast<long long>(v)));
                            tc[(j0 + j) * TS + s] = (int)((unsigned)count_of(tc, j0 + j) * (unsigned)kMagicBits);
                        }
                        if (MODE == TETRA_INTEGRATED) {
                            int *se = &stile[(j0 + j) * NORB + s];
                            if (*se) {
                                atomicAdd(reinterpret_cast<unsigned long long *>(Gsc + (long)s * A.chunk_w + j0 + j),
                                          static_cast<unsigned long long>(static_cast<long long>(*se)));
                                *se = 0;
                            }
                        }
                    }
                }
                __syncthreads();
                diffs_from_counts(tc);
            }
            for (int i = tid; i < n_blk * n_copies; i += blockDim.x)
                if (blk_bound[i] >= A.flush_at) blk_bound[i] = 0;
            __syncthreads();
        }
    }
    __syncthreads();
    const bool aborted = s_abort != 0;
    if (aborted) {
        // a TMA wait timed out: wait (bounded) for copies still in flight
        if (tid == 0) {
            for (int b = 0; b < 3; ++b)
                if (n_issued[b] > 0)
                    mbar_wait_bounded(&mbar[b], (uint32_t)(n_issued[b] - 1) & 1u, nullptr, 100000000ull);
        }
        if (MAXM > 1) return;
    } else if (cur >= 0) {
        flush_tile();
    }
    if constexpr (MAXM == 1) {
        // The last CTA of a chunk scales the exact sums to the result. (One
        // accumulator for all CTAs: a slot per CTA took a 39 MB memset, a
        // separate launch and 26 us of serial reads at 256^3 and 4000
        // energies; the flushes are integer atomics either way.)
        __threadfence();
        __syncthreads();
        const int group = chunk % kDoneGroups;
        const int chunks = ((int)gridDim.y - group + kDoneGroups - 1) / kDoneGroups;   // chunks that share the counter
        if (tid == 0) s_active = atomicAdd(&A.done[group], 1) == chunks * (int)gridDim.x - 1;
        __syncthreads();
        if (!s_active) return;
        __threadfence();
        const ModelP &M = B.m[0];
        const float uh = s_unit[0], ul = s_unit[1];   // (every CTA has a box)
        for (int c = group; c < (int)gridDim.y; c += kDoneGroups) {
            const int f0 = c * A.chunk_w, fn = min(A.chunk_w, M.n_omega - f0);
            const long copy = (long)A.n_orb * A.chunk_w;
            const int copies = COPIES ? M.copies : 1;
            const long long *G = A.G + (long)c * copies * copy;
            // an entry summed over the copies
            auto total = [&](const long long *g) {
                long long v = __ldcg(g);
                if constexpr (COPIES)
                    for (int r = 1; r < copies; ++r) v += __ldcg(g + r * copy);
                return v;
            };
            if constexpr (MODE == TETRA_INTEGRATED) {
                // running sum of the chunk's steps (a chunk's first energy holds the
                // steps of every tetrahedron below the chunk): one warp per orbital,
                // in the shared memory of the two tiles
                const long long *Gs = A.Gs + (long)c * copies * copy;
                long long *buf = reinterpret_cast<long long *>(tile);
                __syncthreads();
                for (int i = tid; i < A.n_orb * fn; i += blockDim.x) {
                    const int s = i / fn;
                    buf[i] = total(Gs + (long)s * A.chunk_w + (i - s * fn));
                }
                __syncthreads();
                const int lane = tid & 31;
                for (int s = tid >> 5; s < A.n_orb; s += (int)(blockDim.x >> 5)) {
                    long long carry = 0;
                    for (int j0 = 0; j0 < fn; j0 += 32) {
                        const int j = j0 + lane;
                        long long x = j < fn ? buf[s * fn + j] : 0;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const long long y = __shfl_up_sync(0xffffffffu, x, o);
                            if (lane >= o) x += y;
                        }
                        x += carry;
                        carry = __shfl_sync(0xffffffffu, x, 31);
                        if (j < fn) buf[s * fn + j] = x;
                    }
                }
                __syncthreads();
            }
            for (int i = tid; i < A.n_orb * fn; i += blockDim.x) {
                const int s = i / fn, j = i - s * fn;
                long long v = total(G + (long)s * A.chunk_w + j);
                if (MODE == TETRA_INTEGRATED) v += reinterpret_cast<const long long *>(tile)[i];
                A.dos[(long)s * M.n_omega + f0 + j] = scale_units(v, uh, ul);
            }
        }
    }
}

template <int NORB, typename WT, int MODE, int MAXM, bool COPIES>
cudaError_t launch_t(size_t smem, dim3 grid, const Batch<MAXM> &Bt, const FwdArgs &A,
                     cudaStream_t stream) {
    auto k = tetra_dos_fwd_kernel<NORB, WT, MODE, MAXM, COPIES>;
    // The shared-memory opt-in is set once per device and size, so that a
    // launch inside a CUDA-graph capture makes no attribute call.
    static std::atomic<int> opted[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || opted[dev].load() < (int)smem) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) {
            int cur = opted[dev].load();
            while (cur < (int)smem && !opted[dev].compare_exchange_weak(cur, (int)smem)) {
            }
        }
    }
    // no more warps than a box has items for (idle ones only slow its barriers);
    // in a batch, whose flush looks at one block of 64 energies per thread, as
    // many threads as blocks (at most about 280: a tile takes 13 bytes per energy)
    const int items = A.items_per_box << (MODE != TETRA_BIN && Cfg<NORB>::pairs ? A.split : 0);
    const int least = MAXM > 1 ? std::max(128, (((A.chunk_w + 63) >> 6) + 31) & ~31) : 128;
    const int threads = std::min(kThreads, std::max(least, (items + 31) & ~31));
    k<<<grid, threads, smem, stream>>>(Bt, A);
    return cudaGetLastError();
}

template <int NORB, int MODE, int MAXM, bool COPIES>
cudaError_t launch_wt(int wdtype, size_t smem, dim3 grid, const Batch<MAXM> &Bt, const FwdArgs &A,
                      cudaStream_t stream) {
    switch (wdtype) {
        case TETRA_F16: return launch_t<NORB, __half, MODE, MAXM, COPIES>(smem, grid, Bt, A, stream);
        case TETRA_BF16: return launch_t<NORB, __nv_bfloat16, MODE, MAXM, COPIES>(smem, grid, Bt, A, stream);
        default: return launch_t<NORB, float, MODE, MAXM, COPIES>(smem, grid, Bt, A, stream);
    }
}

template <int MODE, int MAXM, bool COPIES>
cudaError_t launch_norb(int n_orb, int wdtype, size_t smem, dim3 grid, const Batch<MAXM> &Bt,
                        const FwdArgs &A, cudaStream_t stream) {
    switch (norb_template(n_orb)) {
        case 1: return launch_wt<1, MODE, MAXM, COPIES>(wdtype, smem, grid, Bt, A, stream);
        case 2: return launch_wt<2, MODE, MAXM, COPIES>(wdtype, smem, grid, Bt, A, stream);
        case 3: return launch_wt<3, MODE, MAXM, COPIES>(wdtype, smem, grid, Bt, A, stream);
        case 4: return launch_wt<4, MODE, MAXM, COPIES>(wdtype, smem, grid, Bt, A, stream);
        case 5: return launch_wt<5, MODE, MAXM, COPIES>(wdtype, smem, grid, Bt, A, stream);
        case 6: return launch_wt<6, MODE, MAXM, COPIES>(wdtype, smem, grid, Bt, A, stream);
        case 8: return launch_wt<8, MODE, MAXM, COPIES>(wdtype, smem, grid, Bt, A, stream);
        default: return launch_wt<16, MODE, MAXM, COPIES>(wdtype, smem, grid, Bt, A, stream);
    }
}

}  // namespace fwd

}  // namespace tetra
