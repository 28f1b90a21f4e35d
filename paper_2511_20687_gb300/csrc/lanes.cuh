// One hex8 element on 8 lanes: lane a (bits x, y, z) holds corner a, then Walsh pattern a, then Gauss point
// a, then corner a again.  In the sign basis (s = 2 bit - 1 per axis) interpolation to the Gauss points and its
// transpose are butterflies over lane bits, so the 8 lanes share all of an element's work and nothing is
// computed twice; every value is a 64-bit integer (fixed_math.cuh), so the sums are exact.
#pragma once

#include <cuda_runtime.h>

#include "fixed_math.cuh"

namespace osam {
namespace fx {

struct Lane {
    int a;             // corner / pattern / Gauss point
    i64 n[3];          // -1 where the lane's bit of an axis is set, else 0
    D k;               // factor of the lane's pattern: t^(order - 1) - keep
    bool keep;
};

__device__ __forceinline__ Lane make_lane() {
    Lane L;
    L.a = (int)(threadIdx.x & 7u);
#pragma unroll
    for (int d = 0; d < 3; ++d) L.n[d] = -(i64)((L.a >> d) & 1);
    const int order = __popc((unsigned int)L.a);
    L.k = order == 2 ? split(kTm1) : (order == 3 ? split(kThird) : split(0));
    L.keep = order != 3;
    return L;
}

__device__ __forceinline__ i64 other(i64 v, int axis) { return __shfl_xor_sync(0xffffffffu, v, 1 << axis); }
__device__ __forceinline__ i64 flip(i64 x, i64 n) { return (x ^ n) - n; }   // -x where n is -1

// sums over an axis: pattern bit 0 lower + upper, bit 1 upper - lower
__device__ __forceinline__ i64 sum_stage(const Lane& L, i64 v, int axis) { return v + flip(other(v, axis), L.n[axis]); }
// values at the signs of an axis: lower f0 - f1, upper f0 + f1
__device__ __forceinline__ i64 eval_stage(const Lane& L, i64 v, int axis) { return v + flip(other(v, axis), ~L.n[axis]); }
// plain sum over an axis on the lanes whose bit is set, zero on the others
__device__ __forceinline__ i64 set_sum(const Lane& L, i64 v, int axis) { return (v + other(v, axis)) & L.n[axis]; }

__device__ __forceinline__ i64 walsh_sums(const Lane& L, i64 v) {
    return sum_stage(L, sum_stage(L, sum_stage(L, v, 0), 1), 2);
}
__device__ __forceinline__ i64 corner_values(const Lane& L, i64 v) {
    return eval_stage(L, eval_stage(L, eval_stage(L, v, 0), 1), 2);
}
// the 1/sqrt3 powers of the lane's pattern
__device__ __forceinline__ i64 pattern_scale(const Lane& L, i64 v) { return mul_add(split(v), L.k, L.keep ? v : 0); }

// derivatives along the three axes at the lane's Gauss point from the scaled coefficients of one component
__device__ __forceinline__ void gauss_columns(const Lane& L, i64 w, int c, Cols& C) {
    const i64 z = eval_stage(L, w, 2), y = eval_stage(L, w, 1);
    const i64 gx = eval_stage(L, z, 1), gy = eval_stage(L, z, 0), gz = eval_stage(L, y, 0);
    const int lane = (int)(threadIdx.x & 31u);
    C.x[0][c] = __shfl_sync(0xffffffffu, gx, lane | 1);
    C.x[1][c] = __shfl_sync(0xffffffffu, gy, lane | 2);
    C.x[2][c] = __shfl_sync(0xffffffffu, gz, lane | 4);
}
// its transpose: the coefficients of the corner forces from the stress columns (p0, p1, p2) of one component
__device__ __forceinline__ i64 gauss_transpose(const Lane& L, i64 p0, i64 p1, i64 p2) {
    i64 A = set_sum(L, p0, 0), B = sum_stage(L, p1, 0), C = sum_stage(L, p2, 0);
    A = sum_stage(L, A, 1);
    B = set_sum(L, B, 1);
    C = sum_stage(L, C, 1);
    return sum_stage(L, A + B, 2) + set_sum(L, C, 2);
}

// true in all 8 lanes of an element if it is in any of them
__device__ __forceinline__ bool any_lane(bool x) {
    return ((__ballot_sync(0xffffffffu, x) >> (threadIdx.x & 24u)) & 0xffu) != 0;
}
template <typename T, typename Op>
__device__ __forceinline__ T reduce8(T x, Op op) {
#pragma unroll
    for (int b = 1; b < 8; b <<= 1) x = op(x, __shfl_xor_sync(0xffffffffu, x, b));
    return x;
}

// an edge of the element beyond range, from the lanes' coarse nodal values; every lane of the warp takes part
__device__ __forceinline__ bool coarse_edge_bad(int v) {
    bool bad = false;
#pragma unroll
    for (int d = 0; d < 3; ++d) bad |= abs(v - __shfl_xor_sync(0xffffffffu, v, 1 << d)) >= kCoarseSpread;
    return bad;
}

// Nodal values of a warp in which a node is beyond the format (kMaxU edges), again from u(c) in FP64 and modulo 32 edges;
// bad: an element that is out of range all the same
template <typename Load>
__device__ __forceinline__ void refit_lanes(Load u, i64 ihm, int ihe, i64 U[3], bool& bad) {
    if (!__any_sync(0xffffffffu, U[0] == kBadU || U[1] == kBadU || U[2] == kBadU)) return;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        int v;
        bad |= !wrapped_u(u(c), ihm, ihe, U[c], v);
        bad |= coarse_edge_bad(v);
    }
}

// Columns of F from this lane's fixed-point u / h (59 fraction bits; no node marked); bad: an edge of the element out
// of range (edge_bad)
__device__ __forceinline__ void deformation(const Lane& L, const i64 U[3], Cols& C, bool& bad) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int v = hi(U[c]);
#pragma unroll
        for (int d = 0; d < 3; ++d) bad |= edge_bad(v, __shfl_xor_sync(0xffffffffu, v, 1 << d));
        i64 w = walsh_sums(L, U[c]);
        if (L.a == 1 << c) w += (i64)1 << kFracF;
        gauss_columns(L, pattern_scale(L, L.a ? w : 0), c, C);
    }
}

// Walsh coefficients of a direction in block format (the lane's pattern, |w| < 2^58); returns the exponent T:
// coefficient = w 2^(T + 6 - 1081), kNoExponent for a direction without differences (w is then 0)
__device__ __forceinline__ int block_walsh(const Lane& L, const double p[3], i64 w[3], bool& bad) {
    int e[3], T = kNoExponent;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        e[c] = (int)(reduce8(hi_word(p[c]) & 0x7fffffffu, [](unsigned int a, unsigned int b) { return max(a, b); }) >> 20);
        w[c] = walsh_sums(L, block_value(p[c], e[c]));
        if (L.a == 0) w[c] = 0;
        T = max(T, top_exponent(mag(w[c]), e[c]));
        bad |= e[c] == 2047 || (e[c] == 0 && shl(__double_as_longlong(p[c]), 1) != 0);   // not finite, subnormal
    }
    T = reduce8(T, [](int a, int b) { return max(a, b); });
#pragma unroll
    for (int c = 0; c < 3; ++c) w[c] = T == kNoExponent ? 0 : shift(w[c], e[c] - T - 6);
    return T;
}

// A direction in block format: its scaled gradient columns, gradient = G 2^-base / h; returns the base
__device__ __forceinline__ int direction(const Lane& L, const double p[3], Cols& G, bool& bad) {
    i64 w[3];
    const int T = block_walsh(L, p, w, bad);
#pragma unroll
    for (int c = 0; c < 3; ++c) gauss_columns(L, pattern_scale(L, w[c]), c, G);
    return T == kNoExponent ? 0 : 1016 - T;    // 1081 - 59 - 6
}

// Linear elastic force of the lane's corner from its displacement (element_force_le on 8 lanes): F 2^-scale.  lam, mu times h / 16 as in element_force_le.
// A pattern's coefficients need those of the two patterns that differ from it in two axes: {j} and {k} for {i},
// {j, k} and {i, k} for {i, j}.
__device__ __forceinline__ bool force_le_lanes(const Lane& L, const double p[3], double lam, double mu, i64 F[3], int& scale) {
    bool bad = false;
    i64 w[3], A[3], B[3];
    const int T = block_walsh(L, p, w, bad), ek = factor_exponent(lam, mu);
    const int order = __popc((unsigned int)L.a), lane = (int)(threadIdx.x & 31u);
    // order 1: i the pattern's axis; order 2: k the missing axis, i and j the others
    const int i = order == 1 ? __ffs(L.a) - 1 : (__ffs(~L.a & 7) % 3), j = (i + 1) % 3, k = (i + 2) % 3;
    const int flip1 = order == 1 ? (1 << i) | (1 << j) : (1 << i) | (1 << k);   // to {j}; to {j, k}
    const int flip2 = order == 1 ? (1 << i) | (1 << k) : (1 << j) | (1 << k);   // to {k}; to {i, k}
    i64 u[3], v[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        u[c] = __shfl_sync(0xffffffffu, w[c], lane ^ flip1);
        v[c] = __shfl_sync(0xffffffffu, w[c], lane ^ flip2);
    }
    const auto at = [](const i64 x[3], int c) { return c == 0 ? x[0] : (c == 1 ? x[1] : x[2]); };
    const i64 wi = at(w, i), wj = at(w, j), wk = at(w, k);
    i64 ai, aj, ak, bi, bj, bk;
    if (order == 1) {
        ai = wi + at(u, j) + at(v, k); aj = ak = 0;
        bi = 2 * wi; bj = wj + at(u, i); bk = wk + at(v, i);
    } else if (order == 2) {
        ai = wi + at(u, k); aj = wj + at(v, k); ak = 0;
        bi = 3 * wi; bj = 3 * wj; bk = 2 * wk + at(u, i) + at(v, j);
    } else {
        ai = wi; aj = wj; ak = wk;
        bi = 4 * wi; bj = 4 * wj; bk = 4 * wk;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        A[c] = c == i ? ai : (c == j ? aj : ak);
        B[c] = c == i ? bi : (c == j ? bj : bk);
    }
    const D l = split(factor_value(lam, ek)), m = split(factor_value(mu, ek));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        i64 f = mul_add(l, split(A[c]), mul(m, split(B[c])));
        const i64 t = mul_third(f);
        f = order == 1 ? f : (order == 2 ? t : mul_third(t));
        F[c] = corner_values(L, L.a ? f : 0);
    }
    const bool zero = T == kNoExponent;
    scale = zero ? 0 : 2095 - T - ek;
    return !any_lane(bad || ek == 2047 || scale > 1000 || scale < -900);
}

// Saint Venant-Kirchhoff force of the lane's corner from its displacement: F 2^-scale; 1/h as ihm 2^(ihe - 62) (the
// coefficients are multiplied by ihm 2^-63), m1, m2: the material factors lam and mu times h^2 / 32
__device__ __forceinline__ bool force_svk_lanes(const Lane& L, const double p[3], i64 ihm, int ihe, double m1, double m2,
                                                i64 F[3], int& scale) {
    Cols G;
    i64 P[3][3], w[3];
    bool bad = false;
    const int T = block_walsh(L, p, w, bad), e = factor_exponent(m1, m2);
    const int base = T == kNoExponent ? 0 : 1015 - T - ihe;
    const D r = split(ihm);
#pragma unroll
    for (int c = 0; c < 3; ++c) gauss_columns(L, pattern_scale(L, (mul(split(shl(w[c], 4)), r) + 4) >> 3), c, G);
    const i64 l = factor_value(m1, e);
    bad |= !svk_point(G, base, split((l + 1) >> 1), split(factor_value(m2, e)), P);
#pragma unroll
    for (int c = 0; c < 3; ++c)
        F[c] = corner_values(L, pattern_scale(L, gauss_transpose(L, P[0][c], P[1][c], P[2][c])));
    scale = 56 + base - (e - 1022);
    return !any_lane(bad || e == 2047 || scale > 1000 || scale < -900);
}

// corner forces of the lane's corner (57 fraction bits, units 2^k); false if the element is out of range
// (lin: also the linearisation of the lane's Gauss point)
__device__ __forceinline__ bool force_lanes(const Lane& L, const i64 U[3], D kap2, D mu, D mu3, bool bad, i64 F[3],
                                            Linear* lin = nullptr) {
    Cols C;
    deformation(L, U, C, bad);
    i64 P[3][3];
    bad |= !stress_point(C, kap2, mu, mu3, P, lin);
#pragma unroll
    for (int c = 0; c < 3; ++c)
        F[c] = corner_values(L, pattern_scale(L, gauss_transpose(L, P[0][c], P[1][c], P[2][c])));
    return !any_lane(bad);
}

// tangent action on a direction p (FP64) from the stored linearisation of the lane's Gauss point, whose factors
// carry 1/h and units 2^k: value of the lane's corner = F 2^-scale
__device__ __forceinline__ bool tangent_stored_lanes(const Lane& L, const Linear& q, const double p[3], int k, bool bad,
                                                     i64 F[3], int& scale) {
    Cols G;
    i64 dP[3][3];
    const int base = direction(L, p, G, bad);
    bad |= !tangent_stored(q, G, dP);
#pragma unroll
    for (int c = 0; c < 3; ++c)
        F[c] = corner_values(L, pattern_scale(L, gauss_transpose(L, dP[0][c], dP[1][c], dP[2][c])));
    scale = 56 + base - k;
    bad |= scale > 1000 || scale < -900;
    return !any_lane(bad);
}

// tangent action on a direction p (FP64): value of the lane's corner = F 2^-scale; the sums over the Gauss points
// of pk (60 fraction bits) and pm + 2/3 pk (56) with `base` more from the direction's own exponent
__device__ __forceinline__ bool tangent_lanes(const Lane& L, const i64 U[3], const double p[3], const Material& M,
                                              bool bad, bool contract, i64 F[3], int& scale, i64& pk, i64& pm, int& base) {
    Cols C, G;
    deformation(L, U, C, bad);
    base = direction(L, p, G, bad);
    i64 dP[3][3];
    bad |= !tangent_point(C, G, M.kap2, M.mu, M.mu3, dP, pk, pm);
#pragma unroll
    for (int c = 0; c < 3; ++c)
        F[c] = corner_values(L, pattern_scale(L, gauss_transpose(L, dP[0][c], dP[1][c], dP[2][c])));
    scale = 56 + base - M.k;
    if (contract) {
        pm += mul_third(pk) >> 3;
        pk = reduce8(pk, [](i64 a, i64 b) { return a + b; });
        pm = reduce8(pm, [](i64 a, i64 b) { return a + b; });
    }
    // the results' exponents stay inside the normal range
    bad |= scale > 1000 || base > 950 || scale < -900 || base < -960;
    return !any_lane(bad);
}

}  // namespace fx
}  // namespace osam
