// Adjoint of the bin-mode DOS (not in the paper): given g = dL/dDOS[s][i] for
// DOS_s[i] = sum_{T,n} sum_l b_{l,s} [w_l(e_{i+1}) - w_l(e_i)] / (e_{i+1} - e_i),
// computes dL/db and dL/deps at every k-point.
//
// With the edge values D_{e,s} = G_{e-1,s} - G_{e,s}, G_{i,s} = g_si / width_i
// (G_{-1} = G_{n_bins} = 0), the sum over bins is a sum over bin edges,
//   L = sum_{T,n} sum_l sum_s b_{l,s} sum_e D_{e,s} w_l(e),
// where edges at or below a tetrahedron's E1 give nothing and those at or
// above E4 telescope to f G_{j-1,s} (w_l = f = V_T/(4 V_G) there; e_j the first
// of them; so do edges inside with w_l - f in the sum instead of w_l). So only
// the edges inside (E1, E4) cost work, a few or none:
//   dL/db_{l,s} = f G_{j-1,s} + sum_e w_l(e) D_{e,s},
//   dL/de_r     = - sum_e sum_l M_rl(e) k_l(e),  k_l(e) = sum_s b_{l,s} D_{e,s},
// with M_rl(E) = int lambda_r lambda_l delta(E - D) over the tetrahedron, since
// dw_l/de_r = -M_lr. The section at E is two triangles (12|23, 13, 14) and
// (14, 24, 23|34) with corners on edges (see the forward kernel: the same
// clamped edge fractions, no energy cases), and over a triangle of weight a
// the integral of lambda_r lambda_l is a/12 (sum_v lambda_r^v lambda_l^v +
// (sum_v lambda_r^v)(sum_v lambda_l^v)), so M k needs the three corner values
// lambda^v . k only. (At 64^3 points, 8 bands, 200 bins the weights with four
// forward-mode tangents at every bin edge took 8 x 303 us, this 8 x 0.16 ms;
// it waits for loads: 45 % of the cycles issue, 22 of 32 lanes active.)
//
// One thread owns one (cube, band) and adds its six tetrahedra's corner sums
// into the cube's eight corner accumulators (thread-private shared memory).
// Cubes are processed in eight launches, one per parity class of the cube
// origin (x, y, z mod 2): two cubes of one class share no point of the padded
// layout (the layout holds the periodic images x = n1 etc. as separate
// points), so each class adds its corner sums to the gradient arrays without
// atomics. A last pass folds the periodic images onto the interior points.
// Every sum runs in a fixed order, so the result is deterministic.
#include <algorithm>

#include "tetra_internal.cuh"

namespace tetra {

namespace {

constexpr int kBwdThreads = 128;
// blocks per SM (16 orbitals do not fit the registers of four)
constexpr int bwd_blocks(int norb_t) { return norb_t <= 8 ? 4 : 3; }

// Sorted corner energies, the reciprocals of their differences,
// V_T/(4 V_G) (f) and f / E41. A difference of zero gives an infinite
// reciprocal, which the clamped products below turn into a step.
struct TetB {
    float e1, e2, e3, e4;
    float r21, r31, r41, r32, r42, r43;
    float f, fr;
};
__device__ __forceinline__ void tetb_setup(TetB &T, const float e[4], float f) {
    T.e1 = e[0]; T.e2 = e[1]; T.e3 = e[2]; T.e4 = e[3];
    T.r21 = __fdividef(1.f, e[1] - e[0]); T.r31 = __fdividef(1.f, e[2] - e[0]);
    T.r41 = __fdividef(1.f, e[3] - e[0]); T.r32 = __fdividef(1.f, e[2] - e[1]);
    T.r42 = __fdividef(1.f, e[3] - e[1]); T.r43 = __fdividef(1.f, e[3] - e[2]);
    T.f = f;
    T.fr = f * T.r41;
}

// At an edge E inside (E1, E4): w, the corner weights, or from the middle of
// the tetrahedron's range on the corner weights minus f, and m = M k (both for
// the sorted corners). The upper half is the lower half of the mirrored
// tetrahedron (energies -E4 <= -E3 <= -E2 <= -E1 at -E, w - f of it the
// negative weights in reverse order), so w is small and accurate towards
// either end: the sums over many edges cancel.
__device__ __forceinline__ void edge_terms(const TetB &T, float E, bool mir, const float (&kk)[4], float (&ww)[4],
                                           float (&mm)[4]) {
    const float x = mir ? T.e4 - E : E - T.e1, t = mir ? T.e3 - E : E - T.e2, y = mir ? T.e2 - E : E - T.e3;
    const float r21 = mir ? T.r43 : T.r21, r31 = mir ? T.r42 : T.r31, r42 = mir ? T.r31 : T.r42,
                r43 = mir ? T.r21 : T.r43;
    float k[4], w[4], m[4];
#pragma unroll
    for (int l = 0; l < 4; ++l) k[l] = mir ? kk[3 - l] : kk[l];
    const float f21 = __saturatef(x * r21), f31 = __saturatef(x * r31), f41 = __saturatef(x * T.r41);
    const float f32 = __saturatef(t * T.r32), f42 = __saturatef(t * r42), f43 = __saturatef(y * r43);
    const float f12 = 1.f - f21, f13 = 1.f - f31, f14 = 1.f - f41, f23 = 1.f - f32, f24 = 1.f - f42;
    // volume below E: four simplices (forward kernel, tet_w)
    const float fa = T.f * f41, fb = T.f * f14;
    const float v1 = (f21 * f31) * fa, v2 = (f32 * f13) * fa;
    const float v3 = (f32 * f42) * fb, v4 = (f43 * f24) * fb;
    const float c13 = f13 + f14, s42 = f41 + f42, g23 = 1.f + f23;
    w[0] = fmaf(v3 + v4, f14, fmaf(v2, c13, fmaf(v1, c13 + f12, v1)));
    w[1] = fmaf(v4, f24, fmaf(v3, g23 + f24, fmaf(v2, g23, v1 * f21)));
    w[2] = fmaf(v4, 2.f - f43, fmaf(v3, f32, fmaf(v2, f31 + f32, v1 * f31)));
    w[3] = fmaf(v4, s42 + f43, fmaf(v3, s42, (v1 + v2) * f41));
    // section at E: triangles of weight 12 fr p f31 and 12 fr q f24
    const float p = f21 * f23, q = fmaf(-f32, f43, f32);
    const float a = (p * f31) * T.fr, b = (q * f24) * T.fr;
    const float k13 = fmaf(f13, k[0], f31 * k[2]), k14 = fmaf(f14, k[0], f41 * k[3]);
    const float k24 = fmaf(f24, k[1], f42 * k[3]);
    const float kx = fmaf(f12, k[0], fmaf(p, k[1], f32 * k[2]));   // corner 12 | 23
    const float ky = fmaf(f23, k[1], fmaf(q, k[2], f43 * k[3]));   // corner 23 | 34
    const float sa = k13 + k14 + kx, sb = k14 + k24 + ky;
    const float t13 = a * (k13 + sa), tx = a * (kx + sa), t24 = b * (k24 + sb), ty = b * (ky + sb);
    const float t14 = fmaf(a, k14 + sa, b * (k14 + sb));
    m[0] = fmaf(f13, t13, fmaf(f14, t14, f12 * tx));
    m[1] = fmaf(p, tx, fmaf(f24, t24, f23 * ty));
    m[2] = fmaf(f31, t13, fmaf(f32, tx, q * ty));
    m[3] = fmaf(f41, t14, fmaf(f42, t24, f43 * ty));
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        ww[l] = mir ? -w[3 - l] : w[l];
        mm[l] = mir ? m[3 - l] : m[l];
    }
}

// Table I corner labels minus one.
__constant__ int c_tab[6][4] = {{0, 1, 2, 5}, {1, 2, 3, 5}, {0, 2, 4, 5},
                                {2, 3, 5, 7}, {2, 4, 5, 6}, {2, 5, 6, 7}};

struct BwdArgs {
    int n1, n2, n3, nx, ny, nz, nb, n_orb, n_bins;
    int eps_stride, w_stride;
    float f;   // V_T / (4 V_G)
    const float *eps;
    const void *w;
    const float *edges;      // n_bins + 1
    const float *grad_dos;   // [n_orb][n_bins] (TABLE: rows of G, see tetra_dos_bwd_table)
    float *geps, *gw;
    int vec;                 // gw is 16-byte aligned (the caller's array may not be)
    int staged;              // edges, G and D staged in shared memory
};

// Orbitals of the kernel instantiation that takes n_orb.
int bwd_norb(int n_orb) { return n_orb <= 1 ? 1 : n_orb <= 2 ? 2 : n_orb <= 4 ? 4 : n_orb <= 8 ? 8 : 16; }

// Shared-memory bytes of the staged edges, G and D (n_bins + 1 rows each;
// row e of the first holds G_{e-1}), or 0 when they do not fit the 64 KB
// budget.
inline size_t bwd_stage_bytes(int norb_t, int n_bins) {
    const size_t b = sizeof(float) * (((size_t)n_bins + 1 + 3) / 4 * 4 + 2 * (size_t)norb_t * (n_bins + 1));
    return b <= 64 * 1024 ? b : 0;
}

// Thread-private corner accumulators and energies: (1 + n_orb) and one value
// for each of the cube's 8 corners, interleaved over the block's threads.
inline size_t bwd_scratch_bytes(int n_orb) { return sizeof(float) * (2 + (size_t)n_orb) * 8 * kBwdThreads; }

// TABLE: G from rows in global memory instead of shared memory or the gradient.
template <int NORB, typename WT, bool TABLE>
__global__ void __launch_bounds__(kBwdThreads, bwd_blocks(NORB)) tetra_dos_bwd_kernel(const BwdArgs A, int px, int py, int pz) {
    extern __shared__ __align__(16) float s_mem[];
    const int n_e = A.n_bins + 1;
    const int ed_words = (n_e + 3) & ~3;
    const size_t stage = !TABLE && A.staged ? (size_t)ed_words + 2 * (size_t)NORB * n_e : 0;
    float *scr = s_mem + stage;   // [(1 + n_orb) * 8][blockDim]
    float *sce = scr + (1 + A.n_orb) * 8 * blockDim.x;   // corner energies, [8][blockDim]
    // G_{e-1,s}, from the gradient (0 beyond either end)
    auto g_below = [&](int e, int s) -> float {
        return e > 0 ? A.grad_dos[(long)s * A.n_bins + e - 1] / (A.edges[e] - A.edges[e - 1]) : 0.f;
    };
    const float *ed = A.edges, *sG = nullptr, *sD = nullptr;
    if (!TABLE && A.staged) {
        for (int i = threadIdx.x; i < n_e; i += blockDim.x) s_mem[i] = A.edges[i];
        float *G = s_mem + ed_words, *D = G + (size_t)NORB * n_e;
        for (int i = threadIdx.x; i < NORB * n_e; i += blockDim.x) {
            const int s = i / n_e, e = i - s * n_e;
            const float lo = s < A.n_orb ? g_below(e, s) : 0.f;
            const float hi = s < A.n_orb && e < A.n_bins ? g_below(e + 1, s) : 0.f;
            G[e * NORB + s] = lo;
            D[e * NORB + s] = lo - hi;
        }
        __syncthreads();
        ed = s_mem;
        sG = G;
        sD = D;
    }
    // row e of G_{e-1} or D_e
    auto row = [&](bool diff, int e, float (&r)[NORB]) {
        if constexpr (TABLE) {
            load_weights<NORB, float>(A.grad_dos + (size_t)e * NORB, NORB, r);
            if (diff) {
                float hi[NORB];
                load_weights<NORB, float>(A.grad_dos + (size_t)(e + 1) * NORB, NORB, hi);
#pragma unroll
                for (int s = 0; s < NORB; ++s) r[s] -= hi[s];
            }
        } else if (A.staged) {
            load_weights<NORB, float>((diff ? sD : sG) + (size_t)e * NORB, NORB, r);
        } else {
#pragma unroll
            for (int s = 0; s < NORB; ++s) {
                r[s] = s < A.n_orb ? g_below(e, s) : 0.f;
                if (diff && s < A.n_orb && e < A.n_bins) r[s] -= g_below(e + 1, s);
            }
        }
    };
    // cubes of this parity class: x = px, px + 2, ... < n1 (same for y, z)
    const int cxn = (A.n1 - px + 1) >> 1, cyn = (A.n2 - py + 1) >> 1, czn = (A.n3 - pz + 1) >> 1;
    const long total = (long)cxn * cyn * czn * A.nb;
    const WT *W = static_cast<const WT *>(A.w);
    const int nv = 1 + A.n_orb;
    const int tid = threadIdx.x, nt = blockDim.x;
    const float om0 = ed[0];
    const float inv_de = (float)A.n_bins / (ed[A.n_bins] - om0);
    for (long gid = blockIdx.x * (long)blockDim.x + threadIdx.x; gid < total; gid += (long)gridDim.x * blockDim.x) {
        const int n = (int)(gid % A.nb);
        const long cube = gid / A.nb;
        const int x = px + 2 * (int)(cube % cxn), y = py + 2 * (int)((cube / cxn) % cyn),
                  z = pz + 2 * (int)(cube / ((long)cxn * cyn));
        for (int v = 0; v < nv * 8; ++v) scr[v * nt + tid] = 0.f;
        // the cube's corner energies, read together (the loads overlap)
        const long p0 = x + (long)A.nx * (y + (long)A.ny * z);
        const int sy = A.nx, sz = A.nx * A.ny;
        {
            float e8[8];
#pragma unroll
            for (int c = 0; c < 8; ++c)
                e8[c] = A.eps[(p0 + (c & 1) + ((c >> 1) & 1) * sy + (long)(c >> 2) * sz) * A.eps_stride + n];
#pragma unroll
            for (int c = 0; c < 8; ++c) sce[c * nt + tid] = e8[c];
        }
        for (int t = 0; t < 6; ++t) {
            float e[4];
            long pt[4];
            int slot[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int cc = c_tab[t][q];
                pt[q] = p0 + (cc & 1) + ((cc >> 1) & 1) * sy + (long)(cc >> 2) * sz;
                e[q] = sce[cc * nt + tid];
                slot[q] = q;
            }
            // sort corners by energy, carrying their Table-I slot (stable for ties)
#pragma unroll
            for (int i = 1; i < 4; ++i)
#pragma unroll
                for (int j = i; j > 0; --j)
                    if (e[j] < e[j - 1]) {
                        const float te = e[j]; e[j] = e[j - 1]; e[j - 1] = te;
                        const int ts = slot[j]; slot[j] = slot[j - 1]; slot[j - 1] = ts;
                    }
            // edges inside (E1, E4): [lo, hi); hi is the first edge at or above E4
            // and above E1 (a flat tetrahedron is empty at an edge equal to it)
            int lo = (int)ceilf(fminf(fmaxf((e[0] - om0) * inv_de, -2.f), (float)A.n_bins + 2.f));
            int hi = (int)ceilf(fminf(fmaxf((e[3] - om0) * inv_de, -2.f), (float)A.n_bins + 2.f));
            lo = min(max(lo, 0), n_e);
            hi = min(max(hi, 0), n_e);
            while (lo > 0 && ed[lo - 1] > e[0]) --lo;
            while (lo < n_e && ed[lo] <= e[0]) ++lo;
            while (hi > 0 && ed[hi - 1] >= e[3]) --hi;
            while (hi < n_e && ed[hi] < e[3]) ++hi;
            hi = max(hi, lo);
            // nothing below the first or above the last edge reaches a bin
            if (hi == 0 || lo == n_e) continue;
            float acc_e[4] = {0.f, 0.f, 0.f, 0.f};
            float acc_w[4][NORB];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int s = 0; s < NORB; ++s) acc_w[r][s] = 0.f;
            int full = hi;   // first edge that counts as full (w - f instead of w)
            if (lo < hi) {
                float b[4][NORB];
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    load_weights<NORB, WT>(W + pt[slot[r]] * A.w_stride + (long)n * A.n_orb, A.n_orb, b[r]);
                TetB T;
                tetb_setup(T, e, A.f);
                const float mid = 0.5f * (e[0] + e[3]);
                for (int i = lo; i < hi; ++i) {
                    float g[NORB], k[4] = {0.f, 0.f, 0.f, 0.f}, w[4], m[4];
                    row(true, i, g);
#pragma unroll
                    for (int s = 0; s < NORB; ++s)
#pragma unroll
                        for (int l = 0; l < 4; ++l) k[l] = fmaf(g[s], b[l][s], k[l]);
                    const bool mir = ed[i] >= mid;
                    if (mir) full = min(full, i);
                    edge_terms(T, ed[i], mir, k, w, m);
#pragma unroll
                    for (int l = 0; l < 4; ++l) {
                        acc_e[l] -= m[l];
#pragma unroll
                        for (int s = 0; s < NORB; ++s) acc_w[l][s] = fmaf(g[s], w[l], acc_w[l][s]);
                    }
                }
            }
            // the edges that count as full: their D telescope to G below the first
            // (0 below the first edge of all, 0 if there is none)
            if (full > 0 && full < n_e) {
                float g[NORB];
                row(false, full, g);
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int s = 0; s < NORB; ++s) acc_w[r][s] = fmaf(A.f, g[s], acc_w[r][s]);
            }
            // add the sorted corners' sums to the cube-corner accumulators
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int c = c_tab[t][slot[r]];
                scr[(0 * 8 + c) * nt + tid] += acc_e[r];
#pragma unroll
                for (int s = 0; s < NORB; ++s)
                    if (s < A.n_orb) scr[((1 + s) * 8 + c) * nt + tid] += acc_w[r][s];
            }
        }
        // this class's cubes share no point: plain read-modify-write, the loads
        // of four corners together
#pragma unroll 1
        for (int h = 0; h < 8; h += 4) {
            float ge[4];
            float4 g4[4][NORB / 4 > 0 ? NORB / 4 : 1];
            const bool whole = NORB % 4 == 0 && A.vec && A.n_orb == NORB;
            long p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = h + i;
                p[i] = p0 + (c & 1) + ((c >> 1) & 1) * sy + (long)(c >> 2) * sz;
                ge[i] = A.geps[p[i] * A.eps_stride + n];
                if (whole) {
#pragma unroll
                    for (int v = 0; v < NORB / 4; ++v)
                        g4[i][v] = reinterpret_cast<const float4 *>(A.gw + p[i] * A.w_stride + (long)n * A.n_orb)[v];
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = h + i;
                A.geps[p[i] * A.eps_stride + n] = ge[i] + scr[(0 * 8 + c) * nt + tid];
                float *gwp = A.gw + p[i] * A.w_stride + (long)n * A.n_orb;
                if (whole) {
#pragma unroll
                    for (int v = 0; v < NORB / 4; ++v) {
                        float4 g = g4[i][v];
                        g.x += scr[((1 + 4 * v) * 8 + c) * nt + tid];
                        g.y += scr[((2 + 4 * v) * 8 + c) * nt + tid];
                        g.z += scr[((3 + 4 * v) * 8 + c) * nt + tid];
                        g.w += scr[((4 + 4 * v) * 8 + c) * nt + tid];
                        reinterpret_cast<float4 *>(gwp)[v] = g;
                    }
                } else {
                    for (int s = 0; s < A.n_orb; ++s) gwp[s] += scr[((1 + s) * 8 + c) * nt + tid];
                }
            }
        }
    }
}

// Rows G_{e-1}, e = 0 .. n_bins + 1, for more bins than the kernel stages in
// shared memory (8 orbitals: 962); D_e is the difference of two. 64^3 points, 8
// bands, 8 orbitals: 6.5 ms at 900 bins, staged, 6.1 ms at 1000 from these
// rows, which the first-level cache serves; forming the values at every edge and
// orbital, two divisions and strided loads each, took 31.7 ms.
__global__ void tetra_dos_bwd_table(const BwdArgs A, int norb_t, float *rows) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, e = i / norb_t, s = i - e * norb_t;
    if (e > A.n_bins + 1) return;
    rows[i] = s < A.n_orb && e > 0 && e <= A.n_bins
                  ? A.grad_dos[(long)s * A.n_bins + e - 1] / (A.edges[e] - A.edges[e - 1]) : 0.f;
}

// Folds the periodic images (x = n1, y = n2, z = n3 in the padded layout) onto
// the interior point they copy and zeroes them: one thread per (interior
// point on a face x = 0, y = 0 or z = 0, value of its rows of both arrays),
// images added in a fixed order. The face points are enumerated plane by
// plane: x = 0; y = 0 with x >= 1; z = 0 with x, y >= 1. (One thread per
// value: per (point, band) the orbitals' loads ran one after another, 81 us
// at 64^3.)
__global__ void tetra_dos_bwd_fold(const BwdArgs A) {
    const long fa = (long)A.n2 * A.n3, fb = (long)(A.n1 - 1) * A.n3, fc = (long)(A.n1 - 1) * (A.n2 - 1);
    const int vals = A.nb * (1 + A.n_orb);
    const long gid = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (gid >= (fa + fb + fc) * vals) return;
    const int v = (int)(gid % vals);
    long k = gid / vals;
    int x, y, z;
    if (k < fa) {                      // plane x = 0
        x = 0; y = (int)(k % A.n2); z = (int)(k / A.n2);
    } else if ((k -= fa) < fb) {       // plane y = 0, x >= 1
        x = 1 + (int)(k % (A.n1 - 1)); y = 0; z = (int)(k / (A.n1 - 1));
    } else {                           // plane z = 0, x, y >= 1
        k -= fb;
        x = 1 + (int)(k % (A.n1 - 1)); y = 1 + (int)(k / (A.n1 - 1)); z = 0;
    }
    const bool is_e = v < A.nb;
    float *base = is_e ? A.geps + v : A.gw + (v - A.nb);
    const long stride = is_e ? A.eps_stride : A.w_stride;
    float q[8], sum = 0.f;
    float *at[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {   // the loads first: they overlap
        const bool in = (x == 0 || !(i & 1)) && (y == 0 || !(i & 2)) && (z == 0 || !(i & 4));
        const long p = (x + (i & 1) * A.n1) + (long)A.nx * ((y + ((i >> 1) & 1) * A.n2) + (long)A.ny * (z + (i >> 2) * A.n3));
        at[i] = in ? base + p * stride : nullptr;
        q[i] = in ? *at[i] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) sum += q[i];
    *at[0] = sum;
#pragma unroll
    for (int i = 1; i < 8; ++i)
        if (at[i]) *at[i] = 0.f;
}

template <int NORB>
cudaError_t launch_bwd_n(const Plan &P, const BwdArgs &A0, float *table, cudaStream_t stream) {
    BwdArgs A = A0;
    if (table) {
        tetra_dos_bwd_table<<<((A.n_bins + 2) * NORB + 255) / 256, 256, 0, stream>>>(A, NORB, table);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        A.grad_dos = table;
    }
    const size_t smem = (A.staged ? bwd_stage_bytes(NORB, A.n_bins) : 0) + bwd_scratch_bytes(A.n_orb);
    auto go = [&](auto kfn) {
        cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        for (int cls = 0; cls < 8; ++cls) {
            const int px = cls & 1, py = (cls >> 1) & 1, pz = cls >> 2;
            const long cubes = (long)((A.n1 - px + 1) >> 1) * ((A.n2 - py + 1) >> 1) * ((A.n3 - pz + 1) >> 1);
            const long total = cubes * A.nb;
            if (total == 0) continue;
            // as many blocks as run at once: each stages the bin tables once
            const int grid = (int)std::min<long>((total + kBwdThreads - 1) / kBwdThreads, (long)bwd_blocks(NORB) * P.sm_count);
            kfn<<<grid, kBwdThreads, smem, stream>>>(A, px, py, pz);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
        const long face = ((long)A.n2 * A.n3 + (long)(A.n1 - 1) * A.n3 + (long)(A.n1 - 1) * (A.n2 - 1)) *
                          A.nb * (1 + A.n_orb);
        tetra_dos_bwd_fold<<<(int)((face + 255) / 256), 256, 0, stream>>>(A);
        return cudaGetLastError();
    };
    switch (P.d.weight_dtype) {
        case TETRA_F16:
            return table ? go(tetra_dos_bwd_kernel<NORB, __half, true>) : go(tetra_dos_bwd_kernel<NORB, __half, false>);
        case TETRA_BF16:
            return table ? go(tetra_dos_bwd_kernel<NORB, __nv_bfloat16, true>) : go(tetra_dos_bwd_kernel<NORB, __nv_bfloat16, false>);
        default:
            return table ? go(tetra_dos_bwd_kernel<NORB, float, true>) : go(tetra_dos_bwd_kernel<NORB, float, false>);
    }
}

}  // namespace

size_t dos_backward_workspace(const Plan &) { return kStatusBytes; }

tetra_status_t launch_dos_backward(const Plan &P, const float *eps, const void *w,
                                   const float *omega, const float *grad_dos, float *grad_eps,
                                   float *grad_w, void *ws, size_t ws_bytes, cudaStream_t stream) {
    if (ws_bytes < kStatusBytes) return TETRA_ENOMEM;
    if (P.z0 != 0 || P.z1 != P.d.n3) return TETRA_EUNSUPPORTED;   // whole grid only
    BwdArgs A;
    A.n1 = P.d.n1; A.n2 = P.d.n2; A.n3 = P.d.n3; A.nx = P.nx; A.ny = P.ny; A.nz = P.nz;
    A.nb = P.d.n_bands; A.n_orb = P.d.n_orb; A.n_bins = P.d.n_omega;
    A.eps_stride = P.eps_stride; A.w_stride = P.w_stride;
    A.f = (float)(0.25 / (6.0 * (double)P.d.n1 * (double)P.d.n2 * (double)P.d.n3));
    A.eps = eps; A.w = w; A.edges = omega; A.grad_dos = grad_dos; A.geps = grad_eps; A.gw = grad_w;
    A.vec = (reinterpret_cast<uintptr_t>(grad_w) & 15u) == 0;
    A.staged = bwd_stage_bytes(bwd_norb(A.n_orb), A.n_bins) > 0;
    // the rows of G go behind the status words if the caller's workspace has the
    // room (tetra_workspace_bytes has; the call takes less)
    float *table = nullptr;
    if (!A.staged && ws_bytes >= kStatusBytes + sizeof(float) * bwd_norb(A.n_orb) * ((size_t)A.n_bins + 2))
        table = reinterpret_cast<float *>(static_cast<unsigned char *>(ws) + kStatusBytes);
    if (cudaMemsetAsync(ws, 0, kStatusBytes, stream) != cudaSuccess) return TETRA_ECUDA;
    // the parity classes add into the arrays: start from zero (halo and
    // padding entries stay zero)
    const size_t pts = (size_t)P.nx * P.ny * P.nz;
    if (cudaMemsetAsync(grad_eps, 0, sizeof(float) * pts * P.eps_stride, stream) != cudaSuccess ||
        cudaMemsetAsync(grad_w, 0, sizeof(float) * pts * P.w_stride, stream) != cudaSuccess)
        return TETRA_ECUDA;
    cudaError_t e;
    switch (bwd_norb(P.d.n_orb)) {
        case 1: e = launch_bwd_n<1>(P, A, table, stream); break;
        case 2: e = launch_bwd_n<2>(P, A, table, stream); break;
        case 4: e = launch_bwd_n<4>(P, A, table, stream); break;
        case 8: e = launch_bwd_n<8>(P, A, table, stream); break;
        default: e = launch_bwd_n<16>(P, A, table, stream); break;
    }
    return e == cudaSuccess ? TETRA_OK : TETRA_ECUDA;
}

}  // namespace tetra
