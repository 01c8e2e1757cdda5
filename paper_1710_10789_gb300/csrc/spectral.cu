// Bare susceptibility at T = 0 by exact double-band clipping of every
// tetrahedron: the extension to susceptibilities that arXiv:1710.10789 names
// for its method (abstract, Conclusions), here with step occupations.
//
//   S(q, w) = sum_{n,m} (1/V_G) int dk [Theta(mu - e_n(k)) - Theta(mu - e_m(k+q))]
//                                 delta(w - (e_m(k+q) - e_n(k))),
//   Im chi0(q, w + i0) = -pi S(q, w),
//   Re chi0(q, w) = sum_{n,m} (1/V_G) P int dk [Theta(mu - e_n(k)) - Theta(mu - e_m(k+q))]
//                                             / (w - e_m(k+q) + e_n(k)).
//
// Inside a tetrahedron the method interpolates every band linearly, so
// a = e_n - mu, c = e_m(k+q) - mu and the transition energy D = c - a are
// linear there. The occupation difference is +1 on {a < 0 < c}, -1 on
// {c < 0 < a} and 0 elsewhere; each region is the tetrahedron cut by two
// planes. A cut by one plane keeps a corner tetrahedron, a wedge or a prism,
// each split into at most three tetrahedra; the second cut splits those
// again. Over a sub-tetrahedron of volume fraction nu, D is linear and its
// distribution is nu * g(w), g the normalised density of a linear function on
// a tetrahedron (the total of Sec. II.C's corner weight derivatives divided
// by V_T / V_G), or nu * [G(w_hi) - G(w_lo)] / (w_hi - w_lo) as a bin average.
//
// One thread per (cube, tetrahedron) runs over the band pairs that have a
// region in some lane's tetrahedron (four corner minima and maxima: band n
// occupied somewhere and band m empty somewhere for the +1 region, the
// converse for -1), in a loop that is not unrolled (the unrolled 64-pair loop
// overflowed the instruction cache). A whole tetrahedron (occupied, empty at
// every corner) needs no cuts. The clipping only queues the kept
// sub-tetrahedra (sorted transition energies, amplitude, dither key) in a
// per-warp queue in shared memory; between band pairs, once the queue holds
// kDrainAt entries, the warp drains it: long windows a lane per energy, short
// ones a lane each, so the per-energy work is not serialised behind the
// lanes' different clip paths. Contributions are rounded once to integers of
// a fixed-point unit (a dither hashed from the contribution's identity makes
// the rounding unbiased) and added to exact 64-bit sums, whose low halves are
// 32-bit words of a per-CTA shared tile and whose carries go to the accumulator
// in global memory: the result does not depend on the schedule or on the order
// in which queues are drained. At 64^3 points, 8 bands and 400 energies 3.6
// -> 2.3 ms (64-bit shared atomics, one lane per sub-tetrahedron before); 1.3
// ms of it is clipping, which fetches instructions and branches (issue active
// 34 %). (Units up to 64 times coarser, so that a bounded 32-bit tile holds
// the sums, took 2.2 ms, but the error against 64 bits was 4.6e-8 instead of
// 3.0e-8 there and up to four times larger on small grids of few energies.)
//
// The real part runs the same clipping with KIND = kKindRe: every
// sub-tetrahedron reaches every energy (its principal-value average of
// 1/(w - D), below), so the sub-tetrahedra are kept in per-lane segments and
// the whole warp evaluates them in a fixed order, neighbours jointly far away
// and one by one near (each lane owning every 32nd energy). At 48^3 points, 8
// bands and 400 energies 33.2 -> 10.7 ms.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "tet_common.cuh"

namespace tetra {

namespace {

constexpr int kSpecThreads = 128;
constexpr int kSpecWarps = kSpecThreads / 32;
constexpr int kSpecBlocksPerSM = 4;
constexpr int kSpecBits = 26;   // fixed-point fraction bits of the unit
constexpr int kQueueCap = 256;  // sub-tetrahedra per warp queue
constexpr int kDrainAt = 64;    // a queue this full is drained before the next band pair
constexpr int kWide = 20;       // a sub-tetrahedron with this many energies is taken by the whole warp
constexpr float kEntryCap = 1.0e9f;   // below 2^30: larger contributions go to the 64-bit accumulator
// the real part of chi0 (kKindRe) next to the spectral function (kKindS)
constexpr int kKindS = 0, kKindRe = 1;
constexpr int kReBlocksPerSM = 3;
constexpr int kSubPerPair = 18;  // sub-tetrahedra one (tetrahedron, band pair) can give: 2 regions x 3 x 3
// band pairs summed in FP32 before the per-warp sums go to the tile (error against 64
// bits at 48^3 points, 8 bands, 400 energies: 3.8e-8, and no more when they go after
// every 64 sub-tetrahedra)
constexpr int kReFlush = 64;
constexpr int kReGroup = 8;      // lanes whose sub-tetrahedra are taken together far away
constexpr int kReCluster = 20;   // highest moment of such a group
constexpr int kReMom = 16;       // highest moment of one sub-tetrahedron
constexpr int kRePiece = 8;      // terms of a density piece's own series
constexpr int kReBatch = 16;     // sub-tetrahedra set up at a time

// Table I (corner labels minus one, label c at offset (c&1, (c>>1)&1, (c>>2)&1)).
__constant__ int kSpecTable[6][4] = {{0, 1, 2, 5}, {1, 2, 3, 5}, {0, 2, 4, 5},
                                     {2, 3, 5, 7}, {2, 4, 5, 6}, {2, 5, 6, 7}};

// A point of the parent tetrahedron: three barycentric coordinates (the
// fourth is implied) and the two linear fields a and c.
struct P5 {
    float l0, l1, l2, a, c;
};

__device__ __forceinline__ P5 cut(const P5 &u, const P5 &v, float su, float sv) {
    const float t = su / (su - sv);
    return {fmaf(t, v.l0 - u.l0, u.l0), fmaf(t, v.l1 - u.l1, u.l1), fmaf(t, v.l2 - u.l2, u.l2),
            fmaf(t, v.a - u.a, u.a), fmaf(t, v.c - u.c, u.c)};
}

// Field a clip keeps the negative side of: 0 -> a, 1 -> -a, 2 -> c, 3 -> -c.
__device__ __forceinline__ float field(const P5 &p, int which) {
    const float v = (which < 2) ? p.a : p.c;
    return (which & 1) ? -v : v;
}

__device__ __forceinline__ void cswap5(P5 &x, P5 &y, float &sx, float &sy) {
    if (sy < sx) {
        const P5 t = x;
        x = y;
        y = t;
        const float ts = sx;
        sx = sy;
        sy = ts;
    }
}

// One sub-tetrahedron waiting in a warp's queue: its sorted transition
// energies, amplitude sign * nu * scale and dither key.
struct SubTet {
    float d0, d1, d2, d3, amp;
    uint32_t key;
};

// One sub-tetrahedron of the real part in its lane's segment: sorted
// transition energies and amplitude.
struct ReSeg {
    float d0, d1, d2, d3, amp;
};

// Set-up of one entry as the warp's lanes read it (32 words): mean c,
// amplitude, (2 R)^2, half-width R, moments mu_2..mu_kReMom in units of R (mu_0
// = 1, and mu_1 vanishes about the mean), and the density pieces: corner
// values, reciprocal lengths (0 for an empty one), g(d1), g(d2) and the middle
// piece's value at its centre.
struct __align__(16) ReStage {
    float c, amp, far2, R;
    float mu[kReMom - 1];
    float d[4], r[3], G1, G2, A2, pad[3];
};
static_assert(sizeof(ReStage) == 128, "32 words");

// Constants of a launch that the sub-tetrahedron accumulation needs.
struct SpecArgs {
    const float *om;        // shared: energies (point) or bin edges (bin)
    long long *tile;        // shared, real part: int64 accumulators per energy
    unsigned *tile32;       // shared, S: low halves of the sums per energy / bin
    long long *sums;        // global: int64 accumulators per energy / bin
    int n_om;               // energies or bins
    int mode;               // TETRA_POINT or TETRA_BIN
    float scale;            // V_T/V_G over the fixed-point unit
    float max_iw;           // bin mode: 1 / narrowest bin
    int *status;
    float om0, om_last;     // first and last grid energy (edge)
    float inv_de;           // 1 / mean spacing, for the index estimates
    SubTet *q;              // shared, S: this warp's queue [kQueueCap]
    int *qn;                // shared, S: its fill count
    struct SpecTet *st;     // shared, S: this warp's set-ups [32]
    float *racc;            // shared, real part: the warps' FP32 sums per energy
    ReSeg *rq;              // shared, real part: the lanes' segments [warps][32][kSubPerPair]
    unsigned char *rn;      // shared, real part: their counts [warps][32]
    ReStage *stage;         // shared, real part: the warps' set-ups [warps][kReBatch]
};

// One sub-tetrahedron set up for its energies [i0, i1): the density of D, and
// its cumulative, with the clamped edge fractions of the DOS kernel (no cases;
// equal corner energies give infinite reciprocals, whose products saturate).
struct __align__(16) SpecTet {
    float e1, e2, e3, r21, r31, r41, r32, r42, r43;
    float amp;    // point: amplitude * 3 / E41; bin: amplitude
    float dith;
    int i0, i1, pad[3];
};

__device__ __forceinline__ float spec_density(const SpecTet &T, float E) {   // over amp
    const float x = E - T.e1, t = E - T.e2, y = E - T.e3;
    const float f21 = __saturatef(x * T.r21), f31 = __saturatef(x * T.r31), f32 = __saturatef(t * T.r32);
    const float f42 = __saturatef(t * T.r42), f43 = __saturatef(y * T.r43);
    const float p = fmaf(-f21, f32, f21), q = fmaf(-f32, f43, f32);   // f21 f23, f32 f34
    return fmaf(p, f31, fmaf(-q, f42, q));
}

__device__ __forceinline__ float spec_below(const SpecTet &T, float E) {
    const float x = E - T.e1, t = E - T.e2, y = E - T.e3;
    const float f21 = __saturatef(x * T.r21), f31 = __saturatef(x * T.r31), f41 = __saturatef(x * T.r41);
    const float f32 = __saturatef(t * T.r32), f42 = __saturatef(t * T.r42), f43 = __saturatef(y * T.r43);
    const float f14 = 1.f - f41;
    return fmaf(f41, fmaf(f32, 1.f - f31, f21 * f31), f14 * fmaf(f32, f42, f43 * (1.f - f42)));
}

// Mean spacing of the energy grid (or bin width), the scale of the
// fixed-point unit = (V_T/V_G) / de * 2^-26.
__device__ __forceinline__ double mean_spacing(const float *om, int n_om, int mode) {
    const int spacings = mode == TETRA_BIN ? n_om : n_om - 1;
    double de = spacings > 0 ? ((double)om[spacings] - (double)om[0]) / spacings : 1.0;
    return de > 0.0 ? de : 1.0;
}

__device__ __forceinline__ float hash_dither(uint32_t key) {
    uint32_t h = key * 0x9E3779B9u;
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    return (float)(h >> 8) * (1.0f / 16777216.0f) - 0.5f;
}

// First index i in [0, n) with om[i] > x (or n), from the index a uniform
// grid would give (om0 + i / inv_de), corrected against the grid itself, so
// any ascending grid gives the exact index.
__device__ __forceinline__ int upper_index(const float *om, int n, float x, float om0, float inv_de) {
    const float e = fminf(fmaxf((x - om0) * inv_de, -1.f), (float)n + 1.f);
    int i = min(max((int)ceilf(e), 0), n);
    while (i > 0 && om[i - 1] > x) --i;
    while (i < n && !(om[i] > x)) ++i;
    return i;
}

// First index i in [0, n) with om[i] >= x (or n), as upper_index.
__device__ __forceinline__ int lower_index(const float *om, int n, float x, float om0, float inv_de) {
    const float e = fminf(fmaxf((x - om0) * inv_de, -1.f), (float)n + 1.f);
    int i = min(max((int)ceilf(e), 0), n);
    while (i > 0 && om[i - 1] >= x) --i;
    while (i < n && !(om[i] >= x)) ++i;
    return i;
}

// Sets one queued sub-tetrahedron up.
__device__ __forceinline__ void spec_setup(const SubTet &Q, const SpecArgs &S, SpecTet &T) {
    T.e1 = Q.d0; T.e3 = Q.d2;
    // E2 = E3 = E4: the density jumps to zero at E4, which is not below it
    T.e2 = (Q.d1 < Q.d3) ? Q.d1 : nextafterf(Q.d3, -INFINITY);
    T.r21 = __frcp_rn(Q.d1 - Q.d0); T.r31 = __frcp_rn(Q.d2 - Q.d0); T.r41 = __frcp_rn(Q.d3 - Q.d0);
    T.r32 = __frcp_rn(Q.d2 - Q.d1); T.r42 = __frcp_rn(Q.d3 - Q.d1); T.r43 = __frcp_rn(Q.d3 - Q.d2);
    T.dith = hash_dither(Q.key);
    if (S.mode == TETRA_BIN) {
        T.e2 = Q.d1;
        T.amp = Q.amp;
        T.i0 = max(0, upper_index(S.om, S.n_om + 1, Q.d0, S.om0, S.inv_de) - 1);   // bins with upper edge > d0
        T.i1 = min(S.n_om, upper_index(S.om, S.n_om + 1, Q.d3, S.om0, S.inv_de));   // and lower edge <= d3
    } else {
        // (3 / E41 first: 3 amp would round alike for all whole tetrahedra)
        T.amp = Q.amp * (3.f * T.r41);
        T.i0 = upper_index(S.om, S.n_om, Q.d0, S.om0, S.inv_de);
        T.i1 = lower_index(S.om, S.n_om, Q.d3, S.om0, S.inv_de);
    }
}

// Its contribution to energy (bin) i, before rounding.
__device__ __forceinline__ float spec_value(const SpecTet &T, const float *om, bool bin, int i) {
    if (bin) {
        // the quotient with its residual added once: the approximate reciprocal's
        // error is the same for all items of a bin
        const float width = om[i + 1] - om[i], r = __fdividef(1.f, width);
        const float step = spec_below(T, om[i + 1]) - spec_below(T, om[i]), v = step * r;
        return fmaf(T.amp, fmaf(fmaf(-width, v, step), r, v), T.dith);
    }
    return fmaf(T.amp, spec_density(T, om[i]), T.dith);
}

// Adds a sub-tetrahedron to the 64-bit accumulator in global memory: the path
// of contributions too large for the int32 tile and of a full queue (the
// same single rounding as the tile path).
__device__ __noinline__ void deposit_wide(const SubTet &Q, const SpecArgs &S) {
    SpecTet T;
    spec_setup(Q, S, T);
    for (int i = T.i0; i < T.i1; ++i) {
        const float x = spec_value(T, S.om, S.mode == TETRA_BIN, i);
        if (fabsf(x) < 4.0e18f) {
            const long long qv = __float2ll_rn(x);
            if (qv) atomicAdd(reinterpret_cast<unsigned long long *>(&S.sums[i]), static_cast<unsigned long long>(qv));
        } else {
            atomicOr(S.status, kFlagRange);
        }
    }
}

// Adds values (below 2^31), rounded to integers, to the exact 64-bit sums: the
// low halves in the tile, whose carries and borrows (the old value says when) go
// to the accumulator in global memory. They are rare, about one per 2^32 / |x|
// adds, so that nothing has to bound or flush the tile. The old value is looked
// at one add later, when it has arrived.
struct SpecAdd {
    unsigned *tile;
    long long *sums;
    int q = 0, i = 0;
    unsigned old = 0;
    __device__ __forceinline__ void settle() {
        const int carry = (old + (unsigned)q < old ? 1 : 0) + (q >> 31);
        if (carry) atomicAdd(reinterpret_cast<unsigned long long *>(&sums[i]), (unsigned long long)((long long)carry << 32));
    }
    __device__ __forceinline__ void add(int j, float x) {
        const int v = __float2int_rn(x);
        settle();
        old = atomicAdd(&tile[j], (unsigned)v);
        q = v;
        i = j;
    }
};

// Queues one sub-tetrahedron with corner values d of D in this warp's queue (or
// adds it at once when the queue is full). Real part: in this lane's own
// segment, in the order the clipping produces them.
template <int KIND>
__device__ __forceinline__ void keep(float (&d)[4], float amp, uint32_t key, const SpecArgs &S) {
#define SPEC_CS(i, j) { const float lo_ = fminf(d[i], d[j]), hi_ = fmaxf(d[i], d[j]); d[i] = lo_; d[j] = hi_; }
    SPEC_CS(0, 1) SPEC_CS(2, 3) SPEC_CS(0, 2) SPEC_CS(1, 3) SPEC_CS(1, 2)
#undef SPEC_CS
    if constexpr (KIND == kKindRe) {
        // every sub-tetrahedron reaches every energy (a flat one as 1/(w - d))
        const int slot = S.rn[threadIdx.x]++;
        S.rq[threadIdx.x * kSubPerPair + slot] = ReSeg{d[0], d[1], d[2], d[3], amp};
    } else {
        // a flat transition energy is a delta: measure zero in point mode, its
        // whole weight in the bin that holds it in bin mode
        if (S.mode != TETRA_BIN && !(d[3] > d[0])) return;
        // no grid energy (bin) in reach
        if (d[3] < S.om0 || d[0] > S.om_last) return;
        const SubTet T{d[0], d[1], d[2], d[3], amp, key};
        const int slot = atomicAdd(S.qn, 1);
        if (slot < kQueueCap) S.q[slot] = T;
        else deposit_wide(T, S);
    }
}

// Keeps sign * nu * (distribution of D) of the sub-tetrahedron v0..v3, nu its
// volume fraction.
template <int KIND>
__device__ __noinline__ void accumulate(P5 v0, P5 v1, P5 v2, P5 v3, float sign, uint32_t key,
                                        const SpecArgs &S) {
    const float u00 = v0.l0 - v3.l0, u01 = v0.l1 - v3.l1, u02 = v0.l2 - v3.l2;
    const float u10 = v1.l0 - v3.l0, u11 = v1.l1 - v3.l1, u12 = v1.l2 - v3.l2;
    const float u20 = v2.l0 - v3.l0, u21 = v2.l1 - v3.l1, u22 = v2.l2 - v3.l2;
    const float nu = fabsf(u00 * (u11 * u22 - u12 * u21) - u01 * (u10 * u22 - u12 * u20) +
                           u02 * (u10 * u21 - u11 * u20));
    if (!(nu > 0.f)) return;
    float d[4] = {v0.c - v0.a, v1.c - v1.a, v2.c - v2.a, v3.c - v3.a};
    keep<KIND>(d, sign * nu * S.scale, key, S);
}

// Empties the queue, 32 sub-tetrahedra at a time. Called by all 32 lanes
// together. Each lane sets one up; those with many energies are then taken
// by the whole warp, a lane per energy (consecutive tile entries: no bank
// conflict, no lane idle for another's longer window), the short ones by
// their own lane. The atomics are 32-bit (64-bit shared ones take about 20
// cycles a warp, 32-bit ones 1 to 4).
__device__ __forceinline__ void drain(const SpecArgs &S, int lane) {
    constexpr unsigned kAll = 0xffffffffu;
    const SubTet *queue = S.q;
    SpecTet *st = S.st;
    __syncwarp();
    const int n = min(*S.qn, kQueueCap);
    const float *om = S.om;
    SpecAdd acc{S.tile32, S.sums};
    const bool bin = S.mode == TETRA_BIN;
    for (int base = 0; base < n; base += 32) {
        SpecTet T;
        int K = 0;
        if (base + lane < n) {
            const SubTet Q = queue[base + lane];
            spec_setup(Q, S, T);
            K = T.i1 - T.i0;
            // (a density is at most 3 / E41, a bin's average that or its step over it)
            const float most = fabsf(T.amp) * (bin ? 1.01f * fminf(S.max_iw, 3.f * T.r41) : 1.01f);
            if (K > 0 && !(most < kEntryCap)) {
                deposit_wide(Q, S);
                K = 0;
            }
            st[lane] = T;
        }
        __syncwarp();
        unsigned wide = __ballot_sync(kAll, K >= kWide);
        while (wide) {
            const int j = __ffs(wide) - 1;
            wide &= wide - 1;
            const SpecTet W = st[j];
            for (int i = W.i0 + lane; i < W.i1; i += 32) acc.add(i, spec_value(W, om, bin, i));
        }
        if (K > 0 && K < kWide)
            for (int i = T.i0; i < T.i1; ++i) acc.add(i, spec_value(T, om, bin, i));
        __syncwarp();
    }
    acc.settle();
    if (lane == 0) *S.qn = 0;
    __syncwarp();
}

// Cuts tetrahedron (v0..v3) to {field(which) < 0} and accumulates the kept
// sub-tetrahedra (second and last cut).
template <int KIND>
__device__ __noinline__ void clip_second(P5 v0, P5 v1, P5 v2, P5 v3, int which, float sign, uint32_t key,
                                         const SpecArgs &S) {
    float s0 = field(v0, which), s1 = field(v1, which), s2 = field(v2, which), s3 = field(v3, which);
    cswap5(v0, v1, s0, s1);
    cswap5(v2, v3, s2, s3);
    cswap5(v0, v2, s0, s2);
    cswap5(v1, v3, s1, s3);
    cswap5(v1, v2, s1, s2);
    const int k = (s0 < 0.f) + (s1 < 0.f) + (s2 < 0.f) + (s3 < 0.f);
    if (k == 0) return;
    if (k == 4) {
        accumulate<KIND>(v0, v1, v2, v3, sign, key * 4u, S);
    } else if (k == 1) {
        accumulate<KIND>(v0, cut(v0, v1, s0, s1), cut(v0, v2, s0, s2), cut(v0, v3, s0, s3), sign, key * 4u, S);
    } else if (k == 3) {
        const P5 p0 = cut(v0, v3, s0, s3), p1 = cut(v1, v3, s1, s3), p2 = cut(v2, v3, s2, s3);
        accumulate<KIND>(v0, v1, v2, p0, sign, key * 4u, S);
        accumulate<KIND>(v1, v2, p0, p1, sign, key * 4u + 1u, S);
        accumulate<KIND>(v2, p0, p1, p2, sign, key * 4u + 2u, S);
    } else {
        const P5 p02 = cut(v0, v2, s0, s2), p03 = cut(v0, v3, s0, s3);
        const P5 p12 = cut(v1, v2, s1, s2), p13 = cut(v1, v3, s1, s3);
        accumulate<KIND>(v0, p02, p03, v1, sign, key * 4u, S);
        accumulate<KIND>(p02, p03, v1, p12, sign, key * 4u + 1u, S);
        accumulate<KIND>(p03, v1, p12, p13, sign, key * 4u + 2u, S);
    }
}

// One region of one (tetrahedron, band pair): first cut by `first`, then
// every kept tetrahedron by `second`.
template <int KIND>
__device__ __noinline__ void region(P5 v0, P5 v1, P5 v2, P5 v3, int first, int second, float sign,
                                    uint32_t key, const SpecArgs &S) {
    float s0 = field(v0, first), s1 = field(v1, first), s2 = field(v2, first), s3 = field(v3, first);
    cswap5(v0, v1, s0, s1);
    cswap5(v2, v3, s2, s3);
    cswap5(v0, v2, s0, s2);
    cswap5(v1, v3, s1, s3);
    cswap5(v1, v2, s1, s2);
    const int k = (s0 < 0.f) + (s1 < 0.f) + (s2 < 0.f) + (s3 < 0.f);
    if (k == 0) return;
    if (k == 4) {
        clip_second<KIND>(v0, v1, v2, v3, second, sign, key * 4u, S);
    } else if (k == 1) {
        clip_second<KIND>(v0, cut(v0, v1, s0, s1), cut(v0, v2, s0, s2), cut(v0, v3, s0, s3), second, sign, key * 4u, S);
    } else if (k == 3) {
        const P5 p0 = cut(v0, v3, s0, s3), p1 = cut(v1, v3, s1, s3), p2 = cut(v2, v3, s2, s3);
        clip_second<KIND>(v0, v1, v2, p0, second, sign, key * 4u, S);
        clip_second<KIND>(v1, v2, p0, p1, second, sign, key * 4u + 1u, S);
        clip_second<KIND>(v2, p0, p1, p2, second, sign, key * 4u + 2u, S);
    } else {
        const P5 p02 = cut(v0, v2, s0, s2), p03 = cut(v0, v3, s0, s3);
        const P5 p12 = cut(v1, v2, s1, s2), p13 = cut(v1, v3, s1, s3);
        clip_second<KIND>(v0, p02, p03, v1, second, sign, key * 4u, S);
        clip_second<KIND>(p02, p03, v1, p12, second, sign, key * 4u + 1u, S);
        clip_second<KIND>(p03, v1, p12, p13, second, sign, key * 4u + 2u, S);
    }
}

// ---- real part: P<1/(w - D)> of one sub-tetrahedron at every energy ----
//
// Re chi0(q, w) adds sign * nu * P<1/(w - D)> for every sub-tetrahedron; the
// average is the principal-value integral of D's density g against
// 1/(w - x). g is a quadratic spline on the sorted corner values d0..d3 with
// Bernstein coefficients (0, 0, G1) on [d0, d1], (G1, 3/d41, G2) on [d1, d2]
// and (G2, 0, 0) on [d2, d3], G1 = 3 d21/(d31 d41) = g(d1), G2 = 3 d43/(d41
// d42) = g(d2). Far from the sub-tetrahedron (|w - c| > 2 R, c the mean of
// the corner values, R the largest |d_k - c|) the average is the moment
// series sum_n mu_n / (w - c)^(n+1), mu_n = <(D - c)^n> = 6 n!/(n+3)!
// h_n(d - c) (h_n the complete homogeneous symmetric polynomial), whose
// terms shrink by 1/2 or more. Near it each piece [a, b] gives its closed
// form with the logarithm of |w - a| / |w - b|, or, beyond 3/2 of its length
// from its centre, that form's series (re_piece). At a knot the two pieces meeting there drop their
// equal-and-opposite ln|w - knot| terms.
//
// Neighbouring lanes keep neighbouring tetrahedra of one band pair, whose D
// lie close together: far from all of a group of kReGroup lanes (beyond twice
// the half-width of their joint range) they add one series, of their summed
// moments about its centre; only the energies nearer than that take them one
// by one: beyond 2 R of a sub-tetrahedron by its own series, within by the
// density pieces. Series are cut where their terms, (R/u)^n times moments
// that fall as n^-3 (joint range: n^-1), drop below 2^-23 of the first.
// (One series per sub-tetrahedron at every energy, pieces within 4 R: 33.8 ms
// at 48^3 points, 8 bands, 400 energies on a 4 eV window; with the whole warp
// as the group and the pieces' series in 16 terms 14.0 ms.)

// h_n of the values e_0..e_3 (h_0 = 1), from prod_k 1 / (1 - e_k t).
template <int K>
__device__ __forceinline__ void re_homogeneous(const float (&e)[4], float (&h)[K + 1]) {
    h[0] = 1.f;
#pragma unroll
    for (int n = 1; n <= K; ++n) h[n] = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int n = 1; n <= K; ++n) h[n] = fmaf(e[k], h[n - 1], h[n]);
}
__host__ __device__ constexpr float re_coef(int n) { return 6.f / (float)((n + 1) * (n + 2) * (n + 3)); }

__device__ __forceinline__ void re_setup(const ReSeg &T, ReStage &st) {
    const float c = 0.25f * ((T.d0 + T.d1) + (T.d2 + T.d3));
    const float R = fmaxf(c - T.d0, T.d3 - c), inv = R > 1e-37f ? __fdividef(1.f, R) : 0.f;
    // (in units of R: order 16 in the units of the energies would overflow for
    // half-widths above 250 of them and underflow below 1e-2)
    const float e[4] = {(T.d0 - c) * inv, (T.d1 - c) * inv, (T.d2 - c) * inv, (T.d3 - c) * inv};
    st.c = c;
    st.amp = T.amp;
    st.far2 = 4.f * R * R;
    st.R = R;
    float h[kReMom + 1];
    re_homogeneous<kReMom>(e, h);
#pragma unroll
    for (int n = 2; n <= kReMom; ++n) st.mu[n - 2] = h[n] * re_coef(n);
    const float d21 = T.d1 - T.d0, d31 = T.d2 - T.d0, d41 = T.d3 - T.d0;
    const float d32 = T.d2 - T.d1, d42 = T.d3 - T.d1, d43 = T.d3 - T.d2;
    st.d[0] = T.d0; st.d[1] = T.d1; st.d[2] = T.d2; st.d[3] = T.d3;
    st.G1 = d31 > 0.f ? __fdividef(3.f * d21, d31 * d41) : 0.f;
    st.G2 = d42 > 0.f ? __fdividef(3.f * d43, d41 * d42) : 0.f;
    st.A2 = 0.25f * (st.G1 + st.G2) + (d41 > 0.f ? __fdividef(1.5f, d41) : 0.f);
    st.r[0] = d21 > 0.f ? __fdividef(1.f, d21) : 0.f;
    st.r[1] = d32 > 0.f ? __fdividef(1.f, d32) : 0.f;
    st.r[2] = d43 > 0.f ? __fdividef(1.f, d43) : 0.f;
}

// int p(tau) / (up - tau) dtau over [-1/2, 1/2], p = A + B tau + C tau^2, up
// the distance from the piece's centre in lengths, L = log2 of the ratio of
// the distances to its ends. With P = int 1/(up - tau) = ln 2 L the integral
// is p(up) P - B - C up; beyond 3/2 lengths, where that would cancel, P =
// v (1 + t S), v = 1/up, t = v^2/4, S = 1/3 + t/5 + t^2/7 + ..., and the
// integral A P + (B t + C v/4) S.
__device__ __forceinline__ float re_piece(float A, float B, float C, float up, float L) {
    if (fabsf(up) >= 1.5f) {
        const float v = __fdividef(1.f, up), t = 0.25f * v * v;
        float S = 1.f / (2 * kRePiece + 1);
#pragma unroll
        for (int j = kRePiece - 1; j >= 1; --j) S = fmaf(S, t, 1.f / (2 * j + 1));
        return fmaf(A * v, fmaf(t, S, 1.f), fmaf(B, t, 0.25f * C * v) * S);
    }
    return fmaf(fmaf(fmaf(C, up, B), up, A), 0.693147181f * L, -fmaf(C, up, B));
}

// log2 |w - d|; 0 at a knot (also for a subnormal difference, which the
// approximation would take as 0)
__device__ __forceinline__ float re_log2(float w, float d) {
    const float x = fabsf(w - d);
    float l;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(x));
    return x < 1.2e-38f ? 0.f : l;
}

// P<1/(w - D)> within two half-widths of the sub-tetrahedron (or of a flat
// one): the three density pieces.
__device__ __forceinline__ float re_near(const ReStage &T, float w) {
    if (!(T.d[3] > T.d[0])) return (w == T.d[0]) ? 0.f : 1.f / (w - T.d[0]);
    float L[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) L[k] = re_log2(w, T.d[k]);
    float up[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) up[k] = fmaf(-0.5f, T.d[k + 1] - T.d[k], w - T.d[k]) * T.r[k];
    float sum = 0.f;
    if (T.r[0] != 0.f) sum += re_piece(0.25f * T.G1, T.G1, T.G1, up[0], L[0] - L[1]);
    if (T.r[1] != 0.f)
        sum += re_piece(T.A2, T.G2 - T.G1, 2.f * (T.G1 + T.G2) - 4.f * T.A2, up[1], L[1] - L[2]);
    if (T.r[2] != 0.f) sum += re_piece(0.25f * T.G2, -T.G2, T.G2, up[2], L[2] - L[3]);
    return sum;
}

// sum_{n <= K} m[n] z^n for several z at once.
template <int K, int U, int N>
__device__ __forceinline__ void re_series(const float (&m)[N], const float (&z)[U], float (&r)[U]) {
#pragma unroll
    for (int k = 0; k < U; ++k) r[k] = m[K];
#pragma unroll
    for (int n = K - 1; n >= 0; --n)
#pragma unroll
        for (int k = 0; k < U; ++k) r[k] = fmaf(r[k], z[k], m[n]);
}

// Adds the per-warp FP32 sums to the tile (one rounding per energy and
// flush) and clears them. Every lane owns the energies lane, lane + 32, ...
__device__ __forceinline__ void re_flush(const SpecArgs &S, int lane) {
    float *racc = S.racc + (threadIdx.x >> 5) * S.n_om;
    __syncwarp();
    for (int i = lane; i < S.n_om; i += 32) {
        const float x = racc[i];
        racc[i] = 0.f;
        if (fabsf(x) < 4.0e18f) {
            const long long qv = __float2ll_rn(x);
            if (qv) atomicAdd(reinterpret_cast<unsigned long long *>(&S.tile[i]), static_cast<unsigned long long>(qv));
        } else {
            atomicOr(S.status, kFlagRange);
        }
    }
    __syncwarp();
}

// The warp takes the sub-tetrahedra its lanes kept of the last band pair, in
// lane order (a fixed order: the FP32 sums are reproducible). Every lane owns
// the energies lane, lane + 32, ...
__device__ __forceinline__ void re_process(const SpecArgs &S, int lane, int &since_flush) {
    constexpr unsigned kAll = 0xffffffffu;
    const int warp = threadIdx.x >> 5;
    const ReSeg *wq = S.rq + warp * 32 * kSubPerPair;
    ReStage *stage = S.stage + warp * kReBatch;
    const float *om = S.om;
    const int n_om = S.n_om;
    float *racc = S.racc + warp * n_om;
    __syncwarp();
    const int mine = S.rn[threadIdx.x];
    if (!__any_sync(kAll, mine)) return;
    // exclusive prefix of the lanes' counts, and the group's joint range
    int incl = mine;
    float lo = INFINITY, hi = -INFINITY;
    for (int i = 0; i < mine; ++i) {
        lo = fminf(lo, wq[lane * kSubPerPair + i].d0);
        hi = fmaxf(hi, wq[lane * kSubPerPair + i].d3);
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(kAll, incl, d);
        if (lane >= d) incl += y;
        if (d < kReGroup) {
            lo = fminf(lo, __shfl_xor_sync(kAll, lo, d));
            hi = fmaxf(hi, __shfl_xor_sync(kAll, hi, d));
        }
    }
    const int start = incl - mine;
    // joint moments about the group's centre in units of its half-width, of
    // this lane's entries first
    const bool some = hi >= lo;
    const float C = some ? 0.5f * (lo + hi) : 0.f, rho = some ? 0.5f * (hi - lo) : 0.f;
    const float inv = rho > 1e-37f ? 1.f / rho : 0.f;
    constexpr int kM = 24;   // kReCluster + 1 in whole thirds of the exchange below
    float M[kM];
#pragma unroll
    for (int n = 0; n < kM; ++n) M[n] = 0.f;
    for (int i = 0; i < mine; ++i) {
        const ReSeg T = wq[lane * kSubPerPair + i];
        const float e[4] = {(T.d0 - C) * inv, (T.d1 - C) * inv, (T.d2 - C) * inv, (T.d3 - C) * inv};
        float h[kReCluster + 1];
        re_homogeneous<kReCluster>(e, h);
#pragma unroll
        for (int n = 0; n <= kReCluster; ++n) M[n] = fmaf(T.amp * re_coef(n), h[n], M[n]);
    }
    // summed over the group's lanes: three moments end up in each
#pragma unroll
    for (int step = 0; step < 3; ++step) {
        const int half = kM >> (step + 1), mask = kReGroup >> (step + 1);
        const bool upper = lane & mask;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = upper ? M[i] : M[i + half], keep = upper ? M[i + half] : M[i];
            M[i] = keep + __shfl_xor_sync(kAll, send, mask);
        }
    }
#pragma unroll 1
    for (int g = 0; g < 32 / kReGroup; ++g) {
        const int g0 = g * kReGroup;
        if (!__shfl_sync(kAll, (int)some, g0)) continue;
        const float gC = __shfl_sync(kAll, C, g0), grho = __shfl_sync(kAll, rho, g0);
        // the group's moments: n in M[n % 3] of the lane that the exchange left it in
        float m[kReCluster + 1];
#pragma unroll
        for (int n = 0; n <= kReCluster; ++n)
            m[n] = __shfl_sync(kAll, M[n % 3], g0 + 4 * (n / 12) + 2 * ((n % 12) / 6) + (n % 6) / 3);
        const float far2 = 4.f * grho * grho;
        bool near_any = false;
        for (int c0 = 0; c0 < n_om; c0 += 128) {
            float z[4], v[4], r[4];
            float umin = INFINITY;
            bool far[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = c0 + lane + 32 * k;
                const float u = om[min(i, n_om - 1)] - gC;
                v[k] = __fdividef(1.f, u);
                z[k] = grho * v[k];
                far[k] = i < n_om && u * u > far2;
                near_any = near_any || (i < n_om && !far[k]);
                if (far[k]) umin = fminf(umin, u * u);
            }
            // the warp's nearest far energy (non-negative floats order as integers)
            const float wmin = __uint_as_float(__reduce_min_sync(kAll, __float_as_uint(umin)));
            if (wmin == INFINITY) continue;
            if (wmin > 16.f * far2) re_series<7>(m, z, r);
            else if (wmin > 4.f * far2) re_series<11>(m, z, r);
            else re_series<kReCluster>(m, z, r);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (far[k]) racc[c0 + lane + 32 * k] += r[k] * v[k];
        }
        if (!__any_sync(kAll, near_any)) continue;
        // the group's entries one by one at the nearer energies, 16 set up at a
        // time, in lane order
        const int first = __shfl_sync(kAll, start, g0), last = __shfl_sync(kAll, incl, g0 + kReGroup - 1);
        for (int base = first; base < last; base += kReBatch) {
            const int n_here = min(kReBatch, last - base);
            // entry's place: the group's last lane whose segment starts at or before it
            const int e = base + (lane & (kReBatch - 1));
            int src = g0;
#pragma unroll
            for (int step = kReGroup / 2; step >= 1; step >>= 1)
                if (__shfl_sync(kAll, start, src + step) <= e) src += step;
            const int loc = src * kSubPerPair + (e - __shfl_sync(kAll, start, src));
            __syncwarp();   // the last batch is read
            if (lane < n_here) re_setup(wq[loc], stage[lane]);
            __syncwarp();
            for (int c0 = 0; c0 < n_om; c0 += 64) {
                float w[2], sum[2] = {0.f, 0.f};
                bool near[2];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int i = c0 + lane + 32 * k;
                    w[k] = om[min(i, n_om - 1)];
                    const float u = w[k] - gC;
                    near[k] = i < n_om && !(u * u > far2);
                }
                if (!__any_sync(kAll, near[0] || near[1])) continue;
                for (int j = 0; j < n_here; ++j) {
                    const ReStage &st = stage[j];
                    float v[2], r[2] = {0.f, 0.f}, umin = INFINITY;
                    bool own[2];   // by its own series
                    bool pieces = false;
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const float u = w[k] - st.c;
                        v[k] = __fdividef(1.f, u);
                        own[k] = u * u > st.far2;
                        pieces = pieces || (near[k] && !own[k]);
                        if (near[k] && own[k]) umin = fminf(umin, u * u);
                    }
                    const float wmin = __uint_as_float(__reduce_min_sync(kAll, __float_as_uint(umin)));
                    if (wmin != INFINITY) {
                        float mu[kReMom + 1];
                        mu[0] = 1.f;
                        mu[1] = 0.f;
#pragma unroll
                        for (int n = 2; n <= kReMom; ++n) mu[n] = st.mu[n - 2];
                        const float z[2] = {st.R * v[0], st.R * v[1]};
                        if (wmin > 4.f * st.far2) re_series<8>(mu, z, r);
                        else re_series<kReMom>(mu, z, r);
#pragma unroll
                        for (int k = 0; k < 2; ++k) r[k] *= v[k];
                    }
                    if (__any_sync(kAll, pieces)) {
#pragma unroll
                        for (int k = 0; k < 2; ++k)
                            if (near[k] && !own[k]) r[k] = re_near(st, w[k]);
                    }
#pragma unroll
                    for (int k = 0; k < 2; ++k) sum[k] = fmaf(st.amp, r[k], sum[k]);
                }
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    if (near[k]) racc[c0 + lane + 32 * k] += sum[k];
            }
        }
    }
    __syncwarp();
    S.rn[threadIdx.x] = 0;
    if (++since_flush >= kReFlush) {
        re_flush(S, lane);
        since_flush = 0;
    }
}

template <int KIND>
__host__ __device__ constexpr int queue_entries() { return KIND == kKindS ? kQueueCap : 32 * kSubPerPair; }
template <int KIND>   // in ints; real part: a byte per lane
__host__ __device__ constexpr int queue_counts() { return KIND == kKindS ? 2 : 8; }

template <int KIND>
__host__ __device__ constexpr size_t queue_entry_bytes() { return KIND == kKindS ? sizeof(SubTet) : sizeof(ReSeg); }

// Queues (lane segments), counts, staged set-ups, real part: FP32 sums, tile
// (int64; S: int32), energies.
template <int KIND>
size_t spec_smem_bytes(int n_om, int mode) {
    return queue_entry_bytes<KIND>() * kSpecWarps * queue_entries<KIND>() +
           sizeof(int) * kSpecWarps * queue_counts<KIND>() +
           (KIND == kKindRe ? sizeof(ReStage) * kSpecWarps * kReBatch + sizeof(float) * kSpecWarps * (size_t)n_om
                            : sizeof(SpecTet) * kSpecWarps * 32) +
           (KIND == kKindRe ? sizeof(long long) : sizeof(int)) * (size_t)n_om +
           sizeof(float) * (size_t)(mode == TETRA_BIN ? n_om + 1 : n_om);
}
// The longest grid a call takes: 12 bytes per energy beside the queues of S
// (about 17000 energies), 28 of the real part.
template <int KIND>
bool spec_grid_fits(int n_om, int mode, size_t optin) {
    return spec_smem_bytes<KIND>(n_om, mode) + (KIND == kKindS ? 4 * (size_t)n_om - sizeof(SpecTet) * kSpecWarps * 32 : 0) <= optin;
}

template <int NB, int KIND>
__global__ void __launch_bounds__(kSpecThreads, KIND == kKindS ? kSpecBlocksPerSM : kReBlocksPerSM)
    spectral_t0_kernel(const float *eps, int eps_stride, int n1, int n2, int n3, int nx, int ny, int z0, int z1,
                       int qx, int qy, int qz, float mu, const float *omega, int n_om, int mode,
                       double vtvg, long long *sums, float *out, int *status) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int QW = queue_entries<KIND>(), QC = queue_counts<KIND>();
    unsigned char *qraw = smem;                                             // [warps][QW] entries
    int *qcount = reinterpret_cast<int *>(qraw + queue_entry_bytes<KIND>() * kSpecWarps * QW);   // [warps][QC]
    ReStage *stage = reinterpret_cast<ReStage *>(qcount + kSpecWarps * QC); // real part: [warps][kReBatch]
    SpecTet *stet = reinterpret_cast<SpecTet *>(stage);                     // S: [warps][32]
    float *racc = reinterpret_cast<float *>(stage + kSpecWarps * kReBatch); // real part: [warps][n_om]
    long long *tile = reinterpret_cast<long long *>(racc + (KIND == kKindRe ? kSpecWarps * n_om : 0));
    unsigned *tile32 = reinterpret_cast<unsigned *>(tile);                  // S
    float *om = KIND == kKindRe ? reinterpret_cast<float *>(tile + n_om) : reinterpret_cast<float *>(tile32 + n_om);
    static_assert(sizeof(SpecTet) * 32 == sizeof(ReStage) * kReBatch, "one staging area for both");
    __shared__ float s_grid[4];   // V_T/V_G in units, 1 / mean spacing, the unit as a pair
    __shared__ float s_iw[kSpecWarps];
    const int n_edges = (mode == TETRA_BIN) ? n_om + 1 : n_om;
    for (int i = threadIdx.x; i < n_om; i += blockDim.x) {
        if constexpr (KIND == kKindRe) tile[i] = 0;
        else tile32[i] = 0u;
    }
    for (int i = threadIdx.x; i < n_edges; i += blockDim.x) om[i] = omega[i];
    if (threadIdx.x == 0) {
        const double de = mean_spacing(omega, n_om, mode);
        s_grid[0] = (float)ldexp(de, kSpecBits);
        s_grid[1] = (float)(1.0 / de);
        // (the unit that makes the float the kernel multiplies with exact)
        unit_pair(vtvg / (double)s_grid[0], s_grid[2], s_grid[3]);
    }
    for (int i = threadIdx.x; i < kSpecWarps * QC; i += blockDim.x) qcount[i] = 0;
    if constexpr (KIND == kKindRe)
        for (int i = threadIdx.x; i < kSpecWarps * n_om; i += blockDim.x) racc[i] = 0.f;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float scale = s_grid[0];
    float max_iw = 0.f;
    if (KIND == kKindS && mode == TETRA_BIN) {
        for (int i = threadIdx.x; i < n_om; i += blockDim.x) max_iw = fmaxf(max_iw, 1.0f / (om[i + 1] - om[i]));
        max_iw = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(max_iw)));   // (not negative)
        if (lane == 0) s_iw[warp] = max_iw;
        __syncthreads();
        for (int i = 0; i < kSpecWarps; ++i) max_iw = fmaxf(max_iw, s_iw[i]);
    }
    const float om_lo = om[0], om_hi = om[n_edges - 1];
    // (in shared memory: the clipping's calls pass an address, not 120 bytes;
    // S: one per warp with its own queue, which measured 2.1 ms at 64^3 against
    // 2.8 with one per block; real part: one, to leave the room to its sums)
    constexpr int kArgs = KIND == kKindS ? kSpecWarps : 1;
    __shared__ SpecArgs s_args[kArgs];
    if (threadIdx.x < kArgs) {
        const int wp = threadIdx.x;
        s_args[wp] = SpecArgs{om, tile, tile32, sums, n_om, mode, scale, max_iw, status, om_lo, om_hi,
                              s_grid[1], reinterpret_cast<SubTet *>(qraw) + wp * QW, qcount + wp * QC,
                              stet + wp * 32, racc, reinterpret_cast<ReSeg *>(qraw),
                              reinterpret_cast<unsigned char *>(qcount), stage};
    }
    __syncthreads();
    const SpecArgs &S = s_args[KIND == kKindS ? warp : 0];
    int since_flush = 0;   // real part: band pairs in the per-warp FP32 sums
    // energy range of the grid: a band pair whose transition energies over a
    // tetrahedron miss it contributes nothing (the clipped regions' values
    // lie between the corner minimum and maximum); the +1 region has positive
    // transition energies, the -1 region negative ones
    const long n_items = 6L * n1 * n2 * (long)(z1 - z0);
    const long stride = (long)gridDim.x * blockDim.x;
    // whole warps step through the items together (the queue is drained by
    // all 32 lanes); a lane past the end takes part without items
    for (long base = (long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n_items; base += stride) {
        const long it = base + lane;
        const bool valid = it < n_items;
        float a[4][NB], c[4][NB];   // indexed by band at run time below
        if (valid) {
            const int t = (int)(it % 6);
            const long cube = it / 6;
            const int x = (int)(cube % n1), y = (int)((cube / n1) % n2), z = z0 + (int)(cube / ((long)n1 * n2));
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int cl = kSpecTable[t][v];
                const int xx = x + (cl & 1), yy = y + ((cl >> 1) & 1), zz = z + (cl >> 2);
                // the point itself: the layout's halo covers xx = n1 etc.
                const long p = xx + (long)nx * (yy + (long)ny * zz);
                // the point shifted by q, reduced into the grid
                // (xx <= n1 and 0 <= qx < n1, so one subtraction reduces it)
                int sx = xx + qx, sy = yy + qy, sz = zz + qz;
                sx -= (sx >= n1) ? n1 : 0;
                sy -= (sy >= n2) ? n2 : 0;
                sz -= (sz >= n3) ? n3 : 0;
                const long pq = sx + (long)nx * (sy + (long)ny * sz);
#pragma unroll
                for (int n = 0; n < NB; ++n) {
                    a[v][n] = eps[p * eps_stride + n] - mu;
                    c[v][n] = eps[pq * eps_stride + n] - mu;
                }
            }
        }
        // per band: some corner occupied (an), some corner empty (ap); the
        // same for the bands at k + q (cn: occupied, cp: empty)
        uint32_t an = 0, ap = 0, cn = 0, cp = 0, a_all = 0, c_all = 0, a_none = 0, c_none = 0;
        if (valid) {
#pragma unroll
            for (int n = 0; n < NB; ++n) {
                const float amin = fminf(fminf(a[0][n], a[1][n]), fminf(a[2][n], a[3][n]));
                const float amax = fmaxf(fmaxf(a[0][n], a[1][n]), fmaxf(a[2][n], a[3][n]));
                const float cmin = fminf(fminf(c[0][n], c[1][n]), fminf(c[2][n], c[3][n]));
                const float cmax = fmaxf(fmaxf(c[0][n], c[1][n]), fmaxf(c[2][n], c[3][n]));
                an |= (amin < 0.f ? 1u : 0u) << n;
                ap |= (amax > 0.f ? 1u : 0u) << n;
                cn |= (cmin < 0.f ? 1u : 0u) << n;
                cp |= (cmax > 0.f ? 1u : 0u) << n;
                a_all |= (amax < 0.f ? 1u : 0u) << n;   // occupied at every corner
                c_all |= (cmin > 0.f ? 1u : 0u) << n;   // empty at every corner
                a_none |= (amin > 0.f ? 1u : 0u) << n;  // and the converse
                c_none |= (cmax < 0.f ? 1u : 0u) << n;
            }
        }
        // band pairs with a region in some lane's tetrahedron, in a loop that is
        // not unrolled (one copy of the code); the queue is drained between pairs
        // once it holds kDrainAt entries. (The +1 region has positive transition
        // energies, the -1 region negative ones.)
        const bool above = KIND == kKindRe || om_hi > 0.f, below = KIND == kKindRe || om_lo < 0.f;
        uint64_t mine = 0;
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            const uint32_t row = (above && ((an >> n) & 1u) ? cp : 0u) | (below && ((ap >> n) & 1u) ? cn : 0u);
            mine |= (uint64_t)row << (n * NB);
        }
        uint64_t pairs = (uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)mine) |
                         (uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(mine >> 32)) << 32;
#pragma unroll 1
        while (pairs) {
            const int pr = __ffsll((long long)pairs) - 1;
            pairs &= pairs - 1;
            if constexpr (KIND == kKindS) {
                // lane 0's count, read after every push of the previous pair
                // and before any of this one: the same decision in every lane
                __syncwarp();
                const int queued = __shfl_sync(0xffffffffu, *S.qn, 0);
                if (queued >= kDrainAt) drain(S, lane);
            } else {
                re_process(S, lane, since_flush);   // the previous pair's sub-tetrahedra
            }
            const int n = pr / NB, m = pr - (pr / NB) * NB;
            const bool plus = above && ((an >> n) & 1u) && ((cp >> m) & 1u);
            const bool minus = below && ((ap >> n) & 1u) && ((cn >> m) & 1u);
            if (!plus && !minus) continue;
            float d[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) d[v] = c[v][m] - a[v][n];
            if constexpr (KIND == kKindS) {
                const float dlo = fminf(fminf(d[0], d[1]), fminf(d[2], d[3]));
                const float dhi = fmaxf(fmaxf(d[0], d[1]), fmaxf(d[2], d[3]));
                if (dhi < om_lo || dlo > om_hi) continue;
            }
            const uint32_t key = ((uint32_t)it * (uint32_t)(NB * NB) + (uint32_t)(n * NB + m)) * 2u;
            // band n occupied and band m empty at every corner (or the converse):
            // the region is the whole tetrahedron, with the dither key that the two
            // cuts would produce
            if (((a_all >> n) & 1u) && ((c_all >> m) & 1u)) {
                keep<KIND>(d, scale, key * 16u, S);
                continue;
            }
            if (((a_none >> n) & 1u) && ((c_none >> m) & 1u)) {
                keep<KIND>(d, -scale, (key + 1u) * 16u, S);
                continue;
            }
            const P5 v0{1.f, 0.f, 0.f, a[0][n], c[0][m]};
            const P5 v1{0.f, 1.f, 0.f, a[1][n], c[1][m]};
            const P5 v2{0.f, 0.f, 1.f, a[2][n], c[2][m]};
            const P5 v3{0.f, 0.f, 0.f, a[3][n], c[3][m]};
            // +1 on {a < 0, c > 0}; -1 on {a > 0, c < 0}
            if (plus) region<KIND>(v0, v1, v2, v3, 0, 3, 1.f, key, S);
            if (minus) region<KIND>(v0, v1, v2, v3, 1, 2, -1.f, key + 1u, S);
        }
    }
    if constexpr (KIND == kKindS) {
        drain(S, lane);
    } else {
        re_process(S, lane, since_flush);
        re_flush(S, lane);
    }
    // one accumulator for all CTAs (integer atomics: exact in any order), scaled
    // by the CTA that finishes last: out[i] = unit * sum. (A row of partials per
    // CTA and a kernel that added the 608 rows took 0.16 ms at 400 energies.)
    __syncthreads();
    for (int i = threadIdx.x; i < n_om; i += blockDim.x) {
        const long long v = KIND == kKindRe ? tile[i] : (long long)(unsigned long long)tile32[i];
        if (v) atomicAdd(reinterpret_cast<unsigned long long *>(sums + i), static_cast<unsigned long long>(v));
    }
    __threadfence();
    __syncthreads();
    __shared__ int s_last;
    if (threadIdx.x == 0) s_last = atomicAdd(status + kDoneOffset / sizeof(int), 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int i = threadIdx.x; i < n_om; i += blockDim.x) out[i] = scale_units(__ldcg(sums + i), s_grid[2], s_grid[3]);
}

// persistent blocks, as many as fit an SM at the register bound
template <int KIND>
int spectral_grid(const Plan &P) { return (KIND == kKindS ? kSpecBlocksPerSM : kReBlocksPerSM) * P.sm_count; }

template <int NB, int KIND>
cudaError_t launch_spectral_nb(const Plan &P, const float *eps, const int q[3], float mu, const float *omega,
                               int n_om, int mode, double vtvg, long long *sums, float *out,
                               int *status, int grid, size_t smem, cudaStream_t stream) {
    auto k = spectral_t0_kernel<NB, KIND>;
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
    k<<<grid, kSpecThreads, smem, stream>>>(eps, P.eps_stride, P.d.n1, P.d.n2, P.d.n3, P.nx, P.ny, P.z0, P.z1,
                                           q[0], q[1], q[2], mu, omega, n_om, mode, vtvg, sums, out,
                                           status);
    return cudaGetLastError();
}

int mod_q(int a, int n) {
    const int m = a % n;
    return m < 0 ? m + n : m;
}

template <int KIND>
size_t spectral_workspace(const Plan &, int n_om) {
    return kStatusBytes + sizeof(long long) * (size_t)n_om;
}

template <int KIND>
tetra_status_t launch_spectral(const Plan &P, const float *eps, const int q_in[3], float mu, int mode, int n_om,
                               const float *omega, float *S, void *ws, size_t ws_bytes, cudaStream_t stream) {
    if (n_om < 1 || (mode != TETRA_POINT && mode != TETRA_BIN)) return TETRA_EINVAL;
    if (P.d.n_bands > 8) return TETRA_EUNSUPPORTED;
    // the bands at k + q come from every plane of the grid
    if (P.z0 != 0 || P.z1 != P.d.n3) return TETRA_EUNSUPPORTED;
    const size_t smem = spec_smem_bytes<KIND>(n_om, mode);
    if (!spec_grid_fits<KIND>(n_om, mode, P.smem_optin)) return TETRA_EUNSUPPORTED;
    if (ws_bytes < spectral_workspace<KIND>(P, n_om)) return TETRA_ENOMEM;
    const double vtvg = 1.0 / (6.0 * (double)P.d.n1 * (double)P.d.n2 * (double)P.d.n3);
    const int q[3] = {mod_q(q_in[0], P.d.n1), mod_q(q_in[1], P.d.n2), mod_q(q_in[2], P.d.n3)};
    const int grid = spectral_grid<KIND>(P);
    int *status = reinterpret_cast<int *>(ws);
    long long *sums = reinterpret_cast<long long *>(static_cast<unsigned char *>(ws) + kStatusBytes);
    if (cudaMemsetAsync(ws, 0, spectral_workspace<KIND>(P, n_om), stream) != cudaSuccess) return TETRA_ECUDA;
    cudaError_t e;
    switch (P.d.n_bands) {
        case 1: e = launch_spectral_nb<1, KIND>(P, eps, q, mu, omega, n_om, mode, vtvg, sums, S, status, grid, smem, stream); break;
        case 2: e = launch_spectral_nb<2, KIND>(P, eps, q, mu, omega, n_om, mode, vtvg, sums, S, status, grid, smem, stream); break;
        case 3: e = launch_spectral_nb<3, KIND>(P, eps, q, mu, omega, n_om, mode, vtvg, sums, S, status, grid, smem, stream); break;
        case 4: e = launch_spectral_nb<4, KIND>(P, eps, q, mu, omega, n_om, mode, vtvg, sums, S, status, grid, smem, stream); break;
        case 5: e = launch_spectral_nb<5, KIND>(P, eps, q, mu, omega, n_om, mode, vtvg, sums, S, status, grid, smem, stream); break;
        case 6: e = launch_spectral_nb<6, KIND>(P, eps, q, mu, omega, n_om, mode, vtvg, sums, S, status, grid, smem, stream); break;
        case 7: e = launch_spectral_nb<7, KIND>(P, eps, q, mu, omega, n_om, mode, vtvg, sums, S, status, grid, smem, stream); break;
        default: e = launch_spectral_nb<8, KIND>(P, eps, q, mu, omega, n_om, mode, vtvg, sums, S, status, grid, smem, stream); break;
    }
    return e == cudaSuccess ? TETRA_OK : TETRA_ECUDA;
}

}  // namespace

size_t spectral_t0_workspace(const Plan &P, int n_om) { return spectral_workspace<kKindS>(P, n_om); }

tetra_status_t launch_spectral_t0(const Plan &P, const float *eps, const int q_in[3], float mu, int mode, int n_om,
                                  const float *omega, float *S, void *ws, size_t ws_bytes, cudaStream_t stream) {
    return launch_spectral<kKindS>(P, eps, q_in, mu, mode, n_om, omega, S, ws, ws_bytes, stream);
}

}  // namespace tetra

extern "C" size_t tetra_spectral_t0_workspace_bytes(tetra_plan_t plan, int n_omega) {
    if (!plan || n_omega < 1) return 0;
    return tetra::spectral_t0_workspace(*plan, n_omega);
}

extern "C" tetra_status_t tetra_spectral_t0(tetra_plan_t plan, const float *eps, const int q[3], float mu, int mode,
                                            int n_omega, const float *omega, float *S, void *ws, size_t ws_bytes,
                                            cudaStream_t stream) {
    if (!plan || !eps || !q || !omega || !S || !ws) return TETRA_EINVAL;
    if ((reinterpret_cast<uintptr_t>(eps) & 15u) || (reinterpret_cast<uintptr_t>(ws) & 15u)) return TETRA_EINVAL;
    const tetra::DeviceGuard dg(plan->device);
    if (!dg.ok()) return TETRA_ECUDA;
    return tetra::launch_spectral_t0(*plan, eps, q, mu, mode, n_omega, omega, S, ws, ws_bytes, stream);
}

extern "C" size_t tetra_chi0_real_t0_workspace_bytes(tetra_plan_t plan, int n_omega) {
    if (!plan || n_omega < 1) return 0;
    return tetra::spectral_workspace<tetra::kKindRe>(*plan, n_omega);
}

extern "C" tetra_status_t tetra_chi0_real_t0(tetra_plan_t plan, const float *eps, const int q[3], float mu,
                                             int n_omega, const float *omega, float *R, void *ws, size_t ws_bytes,
                                             cudaStream_t stream) {
    if (!plan || !eps || !q || !omega || !R || !ws) return TETRA_EINVAL;
    if ((reinterpret_cast<uintptr_t>(eps) & 15u) || (reinterpret_cast<uintptr_t>(ws) & 15u)) return TETRA_EINVAL;
    const tetra::DeviceGuard dg(plan->device);
    if (!dg.ok()) return TETRA_ECUDA;
    return tetra::launch_spectral<tetra::kKindRe>(*plan, eps, q, mu, TETRA_POINT, n_omega, omega, R, ws, ws_bytes,
                                                  stream);
}
