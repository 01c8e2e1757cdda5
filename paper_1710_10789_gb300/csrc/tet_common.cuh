// Device code shared by the kernels that walk tetrahedra: Table I, the sort of
// a tetrahedron's corners and the corner weights of Sec. II.C.
#pragma once
#include "tetra_internal.cuh"

namespace tetra {

// Table I, corner labels minus one; label c sits at offset (c&1, (c>>1)&1, (c>>2)&1).
// Packed 3 bits per corner, 12 bits per tetrahedron, so that lanes holding
// different tetrahedra decode their corners from an immediate instead of
// serialising on divergent constant-memory reads.
constexpr int kTableI[6][4] = {{0, 1, 2, 5}, {1, 2, 3, 5}, {0, 2, 4, 5},
                               {2, 3, 5, 7}, {2, 4, 5, 6}, {2, 5, 6, 7}};
constexpr uint32_t pack_tet(int t) {
    return (uint32_t)(kTableI[t][0] | kTableI[t][1] << 3 | kTableI[t][2] << 6 | kTableI[t][3] << 9);
}
constexpr uint64_t kTetLo = (uint64_t)pack_tet(0) | (uint64_t)pack_tet(1) << 12 | (uint64_t)pack_tet(2) << 24 |
                            (uint64_t)pack_tet(3) << 36 | (uint64_t)pack_tet(4) << 48;
constexpr uint32_t kTetHi = pack_tet(5);
__device__ __forceinline__ uint32_t tet_code(int t) {
    return t < 5 ? (uint32_t)(kTetLo >> (12 * t)) & 0xFFFu : kTetHi;
}

template <typename P>
__device__ __forceinline__ void cswap(float &ea, float &eb, P &pa, P &pb) {
    const bool s = eb < ea;
    const float lo = s ? eb : ea, hi = s ? ea : eb;
    const P plo = s ? pb : pa, phi = s ? pa : pb;
    ea = lo; eb = hi; pa = plo; pb = phi;
}

// Sorts four energies, carrying a payload each.
template <typename P>
__device__ __forceinline__ void sort4(float (&e)[4], P (&p)[4]) {
    cswap(e[0], e[1], p[0], p[1]);
    cswap(e[2], e[3], p[2], p[3]);
    cswap(e[0], e[2], p[0], p[2]);
    cswap(e[1], e[3], p[1], p[3]);
    cswap(e[1], e[2], p[1], p[2]);
}

// The corner weights of one tetrahedron, without cases. With sorted corner
// energies and the crossing fractions of the edges clamped to [0, 1],
//   f_jl = sat((E - E_l) / (E_j - E_l)),  f_lj = 1 - f_jl  (j > l),
// every case of Sec. II.C is one sum over simplices that have zero size
// where the case does not hold:
//  * the surface D = E is the triangle with vertices 13, 14 and "12 or 23"
//    (size f21 f23 f31) plus the triangle 14, 24 and "23 or 34" (size
//    f32 f34 f24), "ab" being the point of edge (a, b) at energy E:
//      dw_l/dE = 4 f / E41 * sum over both of size * sum_vertices lambda_l
//    (lambda the barycentric coordinates; E <= E2 has no second triangle,
//    E >= E3 no first one, outside (E1, E4) there is neither);
//  * the volume D < E is {1, 12|2, 13|3, 14|4} (f21 f31 f41), {2, 13, 14, 23}
//    (f41 f32 f13), {2, 14, 23|3, 24} (f42 f32 f14) and {3, 14, 24, 34}
//    (f43 f24 f14): w_l = f * sum of size * sum_vertices lambda_l / 4 * 4.
// The clamps are the multiplies' own .sat, so no energy costs a compare, a
// select or a branch that the lanes of a warp do not share, the set-up is six
// reciprocals (the cubic coefficients of the middle case took about 90
// operations and 16 registers per tetrahedron), and every term is positive. Equal
// corner energies give infinite reciprocals: inf * 0 = NaN saturates to 0
// and inf * positive to 1, which is the half-open step wanted there.
struct Tet {
    float e1, e2, e3;
    float r21, r31, r41, r32, r42, r43;
    float scale;   // point: 4 f / E41 (0 for a flat tetrahedron); bin, integrated: f
};

template <int MODE>
__device__ __forceinline__ void tet_setup(Tet &T, float e1, float e2, float e3, float e4, float fq) {
    T.e1 = e1; T.e3 = e3;
    // E2 = E3 = E4: the section jumps to zero at E4, where f32 has to be 1
    T.e2 = (MODE == TETRA_POINT && !(e2 < e4)) ? nextafterf(e4, -INFINITY) : e2;
    T.r21 = __fdividef(1.f, e2 - e1); T.r31 = __fdividef(1.f, e3 - e1); T.r41 = __fdividef(1.f, e4 - e1);
    T.r32 = __fdividef(1.f, e3 - e2); T.r42 = __fdividef(1.f, e4 - e2); T.r43 = __fdividef(1.f, e4 - e3);
    T.scale = (MODE == TETRA_POINT) ? (e4 > e1 ? 4.f * fq * T.r41 : 0.f) : fq;
}

// Point mode: dw_l/dE at any E, sorted corners (30 operations).
__device__ __forceinline__ void tet_dw(const Tet &T, float E, float (&d)[4]) {
    const float x = E - T.e1, t = E - T.e2, y = E - T.e3;
    const float f21 = __saturatef(x * T.r21), f31 = __saturatef(x * T.r31), f41 = __saturatef(x * T.r41);
    const float f32 = __saturatef(t * T.r32), f42 = __saturatef(t * T.r42), f43 = __saturatef(y * T.r43);
    const float p = fmaf(-f21, f32, f21);   // f21 f23
    const float q = fmaf(-f32, f43, f32);   // f32 f34
    const float qs = q * T.scale;
    const float a = (p * T.scale) * f31, b = fmaf(-qs, f42, qs), s = a + b;
    d[0] = fmaf((1.f - f21) + (1.f - f31), a, fmaf(-f41, s, s));
    d[1] = fmaf((1.f - f32) + (1.f - f42), b, p * a);
    d[2] = fmaf(f31 + f32, a, q * b);
    d[3] = fmaf(f42 + f43, b, f41 * s);
}

// sum_l b_l dw_l/dE of one orbital (28 operations instead of 30 and 4): the
// weight is linear along the edges, so the section's corners take b at their
// crossing points from the differences along the edges.
struct TetDiff {
    float b1, b2, b21, b31, b41, b32, b42, b43;
};
__device__ __forceinline__ TetDiff tet_diff(float b1, float b2, float b3, float b4) {
    return TetDiff{b1, b2, b2 - b1, b3 - b1, b4 - b1, b3 - b2, b4 - b2, b4 - b3};
}
__device__ __forceinline__ float tet_value(const Tet &T, float E, const TetDiff &D) {
    const float x = E - T.e1, t = E - T.e2, y = E - T.e3;
    const float f21 = __saturatef(x * T.r21), f31 = __saturatef(x * T.r31), f41 = __saturatef(x * T.r41);
    const float f32 = __saturatef(t * T.r32), f42 = __saturatef(t * T.r42), f43 = __saturatef(y * T.r43);
    const float p = fmaf(-f21, f32, f21), q = fmaf(-f32, f43, f32);
    const float qs = q * T.scale;
    const float a = (p * T.scale) * f31, b = fmaf(-qs, f42, qs);
    const float k14 = fmaf(f41, D.b41, D.b1), step = f32 * D.b32;
    // corners 13, 14, 12|23 and 14, 24, 23|34
    const float ka = (fmaf(f31, D.b31, D.b1) + k14) + (fmaf(f21, D.b21, D.b1) + step);
    const float kb = (fmaf(f42, D.b42, D.b2) + k14) + (fmaf(f43, D.b43, D.b2) + step);
    return fmaf(a, ka, b * kb);
}

// w_l(E) at any E (0 below E1, f above E4), sorted corners (49 operations).
__device__ __forceinline__ void tet_w(const Tet &T, float E, float (&w)[4]) {
    const float x = E - T.e1, t = E - T.e2, y = E - T.e3;
    const float f21 = __saturatef(x * T.r21), f31 = __saturatef(x * T.r31), f41 = __saturatef(x * T.r41);
    const float f32 = __saturatef(t * T.r32), f42 = __saturatef(t * T.r42), f43 = __saturatef(y * T.r43);
    const float f13 = 1.f - f31, f14 = 1.f - f41, f24 = 1.f - f42, g23 = 2.f - f32;   // 1 + f23
    const float fa = T.scale * f41, fb = T.scale * f14;
    const float v1 = (f21 * f31) * fa, v2 = (f32 * f13) * fa;
    const float v3 = (f32 * f42) * fb, v4 = (f43 * f24) * fb;
    const float c13 = f13 + f14, s42 = f41 + f42;
    w[0] = fmaf(v3 + v4, f14, fmaf(v2, c13, fmaf(v1, c13 + (1.f - f21), v1)));
    w[1] = fmaf(v4, f24, fmaf(v3, g23 + f24, fmaf(v2, g23, v1 * f21)));
    w[2] = fmaf(v4, 2.f - f43, fmaf(v3, f32, fmaf(v2, f31 + f32, v1 * f31)));
    w[3] = fmaf(v4, s42 + f43, fmaf(v3, s42, (v1 + v2) * f41));
}

// A fixed-point unit as two floats, and v units as a float: products and remainders in
// FP32 pairs (v = float(v) + rest, exact product by fused multiply-add), good
// to the last place. FP64 runs at 1/64 of the FP32 rate here: the unit's
// divisions by every warp of a CTA took microseconds of each launch, and v * u
// for 8 x 4000 values by the CTA that finishes 23 us.
__device__ __forceinline__ void unit_pair(double u, float &hi, float &lo) {
    hi = (float)u;
    lo = (float)(u - (double)hi);
}
__device__ __forceinline__ float scale_units(long long v, float uh, float ul) {
    const float vh = __ll2float_rn(v), rest = __ll2float_rn(v - __float2ll_rn(vh));
    const float p = vh * uh;
    return p + fmaf(rest, uh, fmaf(vh, ul, fmaf(vh, uh, -p)));
}

}  // namespace tetra
