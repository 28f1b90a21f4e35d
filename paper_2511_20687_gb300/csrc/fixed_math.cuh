// 64-bit fixed-point arithmetic of the Neo-Hookean hex8 internal force.
//
// Why: GB300 issues an FP64 instruction of one warp every 67 (FMA, MUL) to 80 (ADD) cycles per SM
// sub-partition; a 32 x 32 + 64 -> 64-bit integer multiply-add takes about 4, a 64-bit integer addition
// 2.2 (measured at 2070 MHz).  The element force needs no floating exponent where F = I + grad u is of
// order one: its FP64 error is set by F's own rounding (2^-53 of 1), however small grad u is, so 64-bit
// integers with a fixed binary point carry it more accurately at a fifth of the time.  Measured against
// a 113-bit reference over displacement gradients from 1e-12 to 0.3, any rotation, nu 0.25 and 0.45: error of an
// element force 1.1e-17 to 3.5e-16 mu h^2 (rms) here, 4.2e-17 to 4.0e-16 in FP64, smaller in every case.  That is for an
// element in its own material's unit; kept in a buffer with the unit of a mesh it loses up to kMaxDown bits.
//
// Values are int64 with a stated number of fraction bits.  A product takes its operands as balanced
// digits x = h 2^32 + l (l signed) and returns the rounded high word,
//   a b / 2^64 = ah bh + (ah bl + al bh + 2^31) / 2^32,
// dropping al bl (at most 1/4 unit in the last place), so the fraction bits of the result are
// fa + fb - 64 and the error is below 0.75 unit in its last place.  Sums are exact (modulo 2^64, so
// intermediate sums may wrap as long as the result fits).
//
// Range (checked per element; an element outside is evaluated in FP64 by the caller): |u| / h below
// 2^22 at every node (from kMaxU on its nodal values are taken modulo 32 edges: refit), the spread of each displacement component over the element (the kernels with a corner per lane:
// along each of its edges) below 2.75 edges, column
// norms of F at the Gauss points below 1.5 (any rotation, 50% stretch), J in (0.53, 1.98), |beta| < 4
// and pair sums of P below 2 in units of the element's material scale.  Every intermediate then fits
// its format; the bounds are at each step.
#pragma once

#include <cmath>
#ifdef __CUDACC__
#include <cuda_runtime.h>
#define OSAM_HD __host__ __device__ __forceinline__
#else
#define OSAM_HD inline
#endif

namespace osam {
namespace fx {

typedef long long i64;

constexpr int kFracU = 59;    // u / h, range +-16
constexpr int kFracF = 61;    // F at the Gauss points, range +-4
constexpr int kFracM = 62;    // material factors in units of the element's scale, at most 1
constexpr int kFracOut = 54;  // element forces in units of the element's scale, or of the mesh's in the buffer
constexpr int kMaxU = 12;     // largest |u| / h of the fixed format
constexpr i64 kBadU = (i64)1 << 63;    // fixed_u of a node outside it (-16)
constexpr i64 kBadF = (i64)1 << 63;    // stored linearisation of a Gauss point outside the range

struct D {
    int h, l;
};

// |x| below 2^63 - 2^31: the high digit of a larger value would not fit its word
OSAM_HD D split(i64 x) {
    D d;
    d.l = (int)(unsigned int)x;
    d.h = (int)(x >> 32) + (int)((unsigned int)x >> 31);
    return d;
}
OSAM_HD i64 wide(int a, int b) { return (i64)a * b; }
OSAM_HD i64 shl(i64 x, int n) { return (i64)((unsigned long long)x << n); }

// a b + c, one instruction (written out: the compiler splits the C++ form into a product and a sum)
OSAM_HD i64 mad(int a, int b, i64 c) {
#ifdef __CUDA_ARCH__
    i64 r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (i64)((unsigned long long)wide(a, b) + (unsigned long long)c);
#endif
}

OSAM_HD i64 mul(D a, D b) {
    i64 m = mad(a.h, b.l, (i64)1 << 31);
    m = mad(a.l, b.h, m);
    return mad(a.h, b.h, m >> 32);
}
OSAM_HD i64 mul(i64 a, i64 b) { return mul(split(a), split(b)); }

// a b + c d as one rounded high word
OSAM_HD i64 dot2(D a, D b, D c, D d) {
    i64 m = mad(a.h, b.l, (i64)1 << 31);
    m = mad(a.l, b.h, m);
    m = mad(c.h, d.l, m);
    m = mad(c.l, d.h, m);
    return mad(c.h, d.h, mad(a.h, b.h, m >> 32));
}

// a.b of three digit pairs
OSAM_HD i64 dot3(D a0, D b0, D a1, D b1, D a2, D b2) {
    i64 m = mad(a0.h, b0.l, (i64)1 << 31);
    m = mad(a0.l, b0.h, m);
    m = mad(a1.h, b1.l, m);
    m = mad(a1.l, b1.h, m);
    m = mad(a2.h, b2.l, m);
    m = mad(a2.l, b2.h, m);
    return mad(a2.h, b2.h, mad(a1.h, b1.h, mad(a0.h, b0.h, m >> 32)));
}

OSAM_HD i64 norm3(D a, D b, D c) {
    i64 m = mad(a.h, a.l, (i64)1 << 30);
    m = mad(b.h, b.l, m);
    m = mad(c.h, c.l, m);
    return mad(c.h, c.h, mad(b.h, b.h, mad(a.h, a.h, m >> 31)));
}

// acc + a b
OSAM_HD i64 mul_add(D a, D b, i64 acc) {
    i64 m = mad(a.h, b.l, (i64)1 << 31);
    m = mad(a.l, b.h, m);
    return mad(a.h, b.h, acc + (m >> 32));
}

// t x with t = 1/sqrt3, and x / 3: (t - 1) 2^64 fits the signed range, t 2^64 does not
constexpr i64 kTm1 = -7796511417081208215LL;     // round((1/sqrt(3) - 1) 2^64)
constexpr i64 kThird = 6148914691236517205LL;    // round(2^64 / 3)
constexpr i64 kThird63 = 3074457345618258603LL;  // round(2^63 / 3)
OSAM_HD i64 mul_t(i64 x) { return mul_add(split(x), split(kTm1), x); }
OSAM_HD i64 mul_third(i64 x) { return mul(split(x), split(kThird)); }

// single-precision seed of J^(-1/3) for J in (1/2, 2): relative error below 2^-20
OSAM_HD float seed_rcbrt(float J) {
#ifdef __CUDA_ARCH__
    float l, y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(J));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(l * (-1.0f / 3.0f)));
    return y;
#else
    return std::pow(J, -1.0f / 3.0f);
#endif
}
OSAM_HD int to_int(float x) {
#ifdef __CUDA_ARCH__
    return __float2int_rn(x);
#else
    return (int)std::lrint(x);
#endif
}

// s = J^(-1/3) with 62 fraction bits from J with 58 (J in (1/2, 2)).  The seed y (30 fraction bits) has
// residual e = 1 - J y^3, |e| < 2^-18, formed to 2^-60; s = y (1 + e/3 + 2 e^2/9), the binomial series of
// (1 - e)^(-1/3), whose next term is below 2^-56 14/81.
OSAM_HD i64 rcbrt58(i64 J58) {
    const float Jf = (float)(int)(J58 >> 32) * 0x1p-26f;
    const int Y = to_int(seed_rcbrt(Jf) * 0x1p30f);          // below 1.27 2^30
    const i64 Y2 = wide(Y, Y);                                // 60
    const D y2 = split(Y2);
    const i64 y3 = mad(y2.h, Y, mad(y2.l, Y, (i64)1 << 31) >> 32);            // 58, below 2
    const i64 p = mul(split(shl(J58, 4)), split(shl(y3, 4)));                  // 60
    const i64 E = shl(((i64)1 << 60) - p, 20);                // 80, |E| < 2^62
    const i64 c1 = mul(split(E), split(kThird63));            // 79
    const int eh = (int)(E >> 32);                            // 48, below 2^30
    const int e2 = (int)(wide(eh, eh) >> 32);                 // 64, below 2^28
    const i64 c = c1 + (wide(e2, 477218588) >> 16);           // 79: round(2/9 2^31) has 31 fraction bits
    const D cd = split(c);
    return shl((i64)Y, 32) + (mad(Y, cd.h, wide(Y, cd.l) >> 32) >> 15);
}

// Running range check of one element: the largest / smallest high words seen
struct Range {
    int jmin = 0x7fffffff, jmax = 0, smax = 0, smin = 0, bmax = 0, bmin = 0;
    unsigned int nmax = 0;
};
OSAM_HD int imin(int a, int b) { return a < b ? a : b; }
OSAM_HD int imax(int a, int b) { return a > b ? a : b; }
OSAM_HD int hi(i64 x) { return (int)(x >> 32); }

// true if a value left the range of the formats (see the header comment)
OSAM_HD bool out_of_range(const Range& g) {
    return g.nmax >= (unsigned int)(2.25 * (1 << 26)) || g.jmin < (int)(0.53 * (1 << 26)) ||
           g.jmax > (int)(1.98 * (1 << 26)) || g.bmax >= (4 << 25) - 1 || g.bmin <= -(4 << 25) + 1 ||
           g.smax >= (2 << 25) - 1 || g.smin <= -(2 << 25) + 1;
}

// spread check of one component's 8 nodal values (59 fraction bits): no nodal value marked, and the
// spread below 2.75 edges, so that every Walsh coefficient stays below 11.  Values reach +-12 edges, so their
// difference (27 fraction bits of the high words) is taken without a sign: it wraps a signed word from 16 edges on.
OSAM_HD bool spread_bad(const i64 V[8]) {
    int mx = hi(V[0]), mn = hi(V[0]);
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 1; k < 8; ++k) {
        mx = imax(mx, hi(V[k]));
        mn = imin(mn, hi(V[k]));
    }
    return mn < -((kMaxU + 1) << 27) || (unsigned int)mx - (unsigned int)mn >= 11u << 25;
}

// The same for the kernels with a corner per lane, from the high words of two corners joined by an edge: further apart
// than 2.75 edges.  With all 12 edges below it a Walsh coefficient (a signed sum of four edge differences) is below 11,
// and an entry of F at a Gauss point (1 or 0 plus a mean of four) below 3.75.  The difference is taken modulo 32 edges:
// values within +-12 that are further apart than 2.75 are also seen apart.
OSAM_HD bool edge_bad(int a, int b) {
    constexpr unsigned int kEdge = 11u << 25;
    return (unsigned int)a - (unsigned int)b + kEdge >= 2 * kEdge;
}

// Walsh coefficients of one component of u / h (59 fraction bits) and their multiples that the Gauss
// points need: 4 dF/dx(q, r) = wx + s_q t wxy + s_r t wxz + s_q s_r t^2 wxyz and so on (61 fraction bits
// of F without a shift).  `axis` = the component index: the 1 of F's diagonal enters as 4 2^59.
struct WalshIn {
    i64 x, y, z, txy, txz, tyz, t2;
};
OSAM_HD WalshIn walsh_in(const i64 V[8], int axis) {
    i64 s[4], d[4];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int j = 0; j < 4; ++j) {
        s[j] = V[2 * j] + V[2 * j + 1];
        d[j] = V[2 * j + 1] - V[2 * j];
    }
    const i64 ss0 = s[0] + s[1], ss1 = s[2] + s[3], sd0 = s[1] - s[0], sd1 = s[3] - s[2];
    const i64 ds0 = d[0] + d[1], ds1 = d[2] + d[3], dd0 = d[1] - d[0], dd1 = d[3] - d[2];
    const i64 one = (i64)1 << kFracF;
    WalshIn w;
    w.x = ds0 + ds1 + (axis == 0 ? one : 0);
    w.y = sd0 + sd1 + (axis == 1 ? one : 0);
    w.z = ss1 - ss0 + (axis == 2 ? one : 0);
    w.txy = mul_t(dd0 + dd1);
    w.txz = mul_t(ds1 - ds0);
    w.tyz = mul_t(sd1 - sd0);
    w.t2 = mul_third(dd1 - dd0);
    return w;
}

// Constitutive quantities of one Gauss point: cof(F) (61), J (58), J^-2/3 (62), 1/J (62), alpha (60) and beta (57).
//   F0, F1, F2: columns of F (61), nF1 = -F1, nF2 = -F2, n: |F|^2 (58); kap2, mu, mu3: material factors (62)
// cof(F) has entries below |col||col| < 2.25 and is carried with 61 bits.
struct NhPoint {
    D c0[3], c1[3], c2[3], r3, inv;
    i64 J, alpha, beta, invJ;   // invJ: 1/J with 60 fraction bits
};
OSAM_HD NhPoint nh_point(const D F0[3], const D F1[3], const D F2[3], const D nF1[3], const D nF2[3], i64 n, D kap2,
                         D mu, D mu3, Range& g) {
    NhPoint s;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int a = 0; a < 3; ++a) {
        const int b = (a + 1) % 3, c = (a + 2) % 3;
        s.c0[a] = split(shl(dot2(F1[b], F2[c], nF1[c], F2[b]), 3));
        s.c1[a] = split(shl(dot2(F2[b], F0[c], nF2[c], F0[b]), 3));
        s.c2[a] = split(shl(dot2(F0[b], F1[c], F0[c], nF1[b]), 3));
    }
    s.J = dot3(F0[0], s.c0[0], F1[0], s.c1[0], F2[0], s.c2[0]);      // 58
    g.jmin = imin(g.jmin, hi(s.J));
    g.jmax = imax(g.jmax, hi(s.J));
    const i64 s1 = rcbrt58(s.J);                                      // 62
    const D s1d = split(s1);
    s.r3 = split(shl(mul(s1d, s1d), 2));                              // J^-2/3, 62 (below 1.53)
    s.invJ = mul(s.r3, s1d);                                          // 1/J, 60
    s.inv = split(shl(s.invJ, 2));
    s.alpha = mul(mu, s.r3);                                          // 60
    const i64 q = mul(s.r3, s.inv);                                   // J^-5/3, 60 (below 2.9)
    const i64 mq = shl(mul(mu3, split(q)), 3);                        // 61 (mu3 <= 1/3)
    const i64 b1 = mul(kap2, split(shl(s.J, 3) - shl(s.invJ, 1)));    // 59
    s.beta = (b1 >> 2) - mul(split(mq), split(shl(n, 2)));            // 57
    g.bmax = imax(g.bmax, hi(s.beta));
    g.bmin = imin(g.bmin, hi(s.beta));
    return s;
}

// One Gauss point: alpha (60 fraction bits) and beta cof(F) added to the pair sums
OSAM_HD void gauss_point(const D F0[3], const D F1[3], const D F2[3], const D nF1[3], const D nF2[3], i64 n, D kap2,
                         D mu, D mu3, Range& g, i64& alpha, i64 X[3], i64 Y[3], i64 Z[3]) {
    const NhPoint s = nh_point(F0, F1, F2, nF1, nF2, n, kap2, mu, mu3, g);
    alpha = s.alpha;
    const D B = split(shl(s.beta, 3));                                // 60
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int a = 0; a < 3; ++a) {
        X[a] = mul_add(B, s.c0[a], X[a]);                             // 57
        Y[a] = mul_add(B, s.c1[a], Y[a]);
        Z[a] = mul_add(B, s.c2[a], Z[a]);
    }
}

OSAM_HD void track(Range& g, i64 s) {
    g.smax = imax(g.smax, hi(s));
    g.smin = imin(g.smin, hi(s));
}

// Transposed interpolation of one component in the Walsh basis (hex8_math.cuh, walsh_transpose): pair
// sums with 57 fraction bits in (below 2 each: every coefficient is below 48, every result below 64),
// corner forces with 54 out (so that a node's sum of 8 fits).  x: h0, ha, hb, hab of Sx and so on.
OSAM_HD void walsh_out(i64 wx, i64 wy, i64 wz, i64 wxy, i64 wxz, i64 wyz, i64 wxyz, i64 F[8]) {
    const i64 txy = mul_t(wxy), txz = mul_t(wxz), tyz = mul_t(wyz), t2 = mul_third(wxyz);
    const i64 half = 4;   // rounding of the final shift by 3
    const i64 up = wx + txy, um = wx - txy;
    const i64 ap = wz + tyz + half, am = wz - tyz + half, bp = txz + t2, bm = txz - t2;
    const i64 Ppp = up + wy, Pmp = wy - up, Ppm = um - wy, Pmm = -um - wy;
    const i64 Qpp = ap + bp, Qmp = ap - bp, Qpm = am + bm, Qmm = am - bm;
    // the rounding half rides on Q: + half for az = 1, - half + 2 half for az = 0
    F[7] = (Ppp + Qpp) >> 3; F[3] = (Ppp - Qpp + 2 * half) >> 3;
    F[6] = (Pmp + Qmp) >> 3; F[2] = (Pmp - Qmp + 2 * half) >> 3;
    F[5] = (Ppm + Qpm) >> 3; F[1] = (Ppm - Qpm + 2 * half) >> 3;
    F[4] = (Pmm + Qmm) >> 3; F[0] = (Pmm - Qmm + 2 * half) >> 3;
}

// Element force of the Neo-Hookean law from fixed-point nodal displacements V[c][corner] (u / h, 59
// fraction bits): F[c][corner] (54 fraction bits, in units of the scale of the material factors).
// Returns false if the element is outside the range of the formats (F is then meaningless).
OSAM_HD bool element_force_nh(const WalshIn w[3], i64 kap2i, i64 mui, i64 mu3i, i64 Fo[3][8]) {
    const D kap2 = split(kap2i), mu = split(mui), mu3 = split(mu3i);
    Range g;
    D F0[2][2][3];
    i64 n0[2][2];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int q = 0; q < 2; ++q) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = 0; c < 3; ++c) {
            const i64 a = q ? w[c].x + w[c].txy : w[c].x - w[c].txy;
            const i64 b = q ? w[c].txz + w[c].t2 : w[c].txz - w[c].t2;
            F0[q][0][c] = split(a - b);
            F0[q][1][c] = split(a + b);
        }
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int r = 0; r < 2; ++r) {
            n0[q][r] = norm3(F0[q][r][0], F0[q][r][1], F0[q][r][2]);
            g.nmax = g.nmax > (unsigned int)hi(n0[q][r]) ? g.nmax : (unsigned int)hi(n0[q][r]);
        }
    }
    i64 Sx[2][2][3] = {};
    i64 al[2][2] = {};
    // Hadamard sums of Sy[p][r] and Sz[p][q] over the two planes p
    i64 wy[3] = {}, ay[3] = {}, by[3] = {}, aby[3] = {}, wz[3] = {}, az[3] = {}, bz[3] = {}, abz[3] = {};
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int p = 0; p < 2; ++p) {
        const i64 sg = p ? 0 : -1;    // x -> s_p x as (x ^ sg) - sg
        D F1[2][3], F2[2][3], nF1[2][3], nF2[2][3];
        i64 n1[2], n2[2];
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = 0; c < 3; ++c) {
            const i64 y0 = w[c].y + ((w[c].txy ^ sg) - sg), z0 = w[c].z + ((w[c].txz ^ sg) - sg);
            const i64 d = w[c].tyz + ((w[c].t2 ^ sg) - sg);
            F1[0][c] = split(y0 - d); nF1[0][c] = split(d - y0);
            F1[1][c] = split(y0 + d); nF1[1][c] = split(-d - y0);
            F2[0][c] = split(z0 - d); nF2[0][c] = split(d - z0);
            F2[1][c] = split(z0 + d); nF2[1][c] = split(-d - z0);
        }
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int a = 0; a < 2; ++a) {
            n1[a] = norm3(F1[a][0], F1[a][1], F1[a][2]);
            n2[a] = norm3(F2[a][0], F2[a][1], F2[a][2]);
            const unsigned int h1 = (unsigned int)hi(n1[a]), h2 = (unsigned int)hi(n2[a]);
            g.nmax = g.nmax > h1 ? g.nmax : h1;
            g.nmax = g.nmax > h2 ? g.nmax : h2;
        }
        i64 Sy[2][3] = {}, Sz[2][3] = {}, ly[2] = {0, 0};
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int q = 0; q < 2; ++q) {
            i64 lz = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int r = 0; r < 2; ++r) {
                i64 alpha;
                gauss_point(F0[q][r], F1[r], F2[q], nF1[r], nF2[q], n0[q][r] + n1[r] + n2[q], kap2, mu, mu3, g, alpha, Sx[q][r], Sy[r],
                            Sz[q]);
                al[q][r] += alpha;
                ly[r] += alpha;
                lz += alpha;
            }
            const D a = split(lz);
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int c = 0; c < 3; ++c) Sz[q][c] = mul_add(a, F2[q][c], Sz[q][c]);
        }
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int r = 0; r < 2; ++r) {
            const D a = split(ly[r]);
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int c = 0; c < 3; ++c) Sy[r][c] = mul_add(a, F1[r][c], Sy[r][c]);
        }
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = 0; c < 3; ++c) {
            track(g, Sy[0][c]); track(g, Sy[1][c]); track(g, Sz[0][c]); track(g, Sz[1][c]);
            const i64 ey = Sy[0][c] + Sy[1][c], dy = Sy[1][c] - Sy[0][c];
            const i64 ez = Sz[0][c] + Sz[1][c], dz = Sz[1][c] - Sz[0][c];
            wy[c] += ey; ay[c] += (ey ^ sg) - sg; by[c] += dy; aby[c] += (dy ^ sg) - sg;
            wz[c] += ez; az[c] += (ez ^ sg) - sg; bz[c] += dz; abz[c] += (dz ^ sg) - sg;
        }
    }
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = 0; c < 3; ++c) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int q = 0; q < 2; ++q)
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int r = 0; r < 2; ++r) {
                Sx[q][r][c] = mul_add(split(al[q][r]), F0[q][r][c], Sx[q][r][c]);
                track(g, Sx[q][r][c]);
            }
        const i64 e0 = Sx[0][0][c] + Sx[0][1][c], e1 = Sx[1][0][c] + Sx[1][1][c];
        const i64 d0 = Sx[0][1][c] - Sx[0][0][c], d1 = Sx[1][1][c] - Sx[1][0][c];
        walsh_out(e0 + e1, wy[c], wz[c], (e1 - e0) + ay[c], (d0 + d1) + az[c], by[c] + bz[c],
                  (d1 - d0) + aby[c] + abz[c], Fo[c]);
    }
    return !out_of_range(g);
}

// ---- one Gauss point on its own (the kernels with one Gauss point per lane) ----------------------

// a b + c d + e f + g h as one rounded high word
OSAM_HD i64 dot4(D a, D b, D c, D d, D e, D f, D g, D h) {
    i64 m = mad(a.h, b.l, (i64)1 << 31);
    m = mad(a.l, b.h, m);
    m = mad(c.h, d.l, m);
    m = mad(c.l, d.h, m);
    m = mad(e.h, f.l, m);
    m = mad(e.l, f.h, m);
    m = mad(g.h, h.l, m);
    m = mad(g.l, h.h, m);
    return mad(g.h, h.h, mad(e.h, f.h, mad(c.h, d.h, mad(a.h, b.h, m >> 32))));
}

// Columns of F (or of a direction's gradient G) at one Gauss point, 61 fraction bits
struct Cols {
    i64 x[3][3];   // [column][component]
};

constexpr int kOne25 = 1 << 25;

// Linearisation of one Gauss point: F and cof F [column][component] (61 fraction bits), alpha (60), beta (57),
// a1 = -2/3 alpha / J (60), b1 = kappa - (a1 trC / 3 + beta) / J (57)
struct Linear {
    i64 F[3][3], cof[3][3], alpha, beta, a1, b1;
};
OSAM_HD i64 whole(D x) { return shl((i64)x.h, 32) + x.l; }

// Piola stress P[column][component] (57 fraction bits, below 1) of one Gauss point; false out of range
OSAM_HD bool stress_point(const Cols& C, D kap2, D mu, D mu3, i64 P[3][3], Linear* lin = nullptr) {
    D F[3][3], nF1[3], nF2[3];
    i64 n = 0;
    Range g;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < 3; ++k) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = 0; c < 3; ++c) F[k][c] = split(C.x[k][c]);
        const i64 m = norm3(F[k][0], F[k][1], F[k][2]);
        g.nmax = g.nmax > (unsigned int)hi(m) ? g.nmax : (unsigned int)hi(m);
        n += m;
    }
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = 0; c < 3; ++c) { nF1[c] = split(-C.x[1][c]); nF2[c] = split(-C.x[2][c]); }
    const NhPoint s = nh_point(F[0], F[1], F[2], nF1, nF2, n, kap2, mu, mu3, g);
    const D A = split(s.alpha), B = split(shl(s.beta, 3));            // 60, 60
    int top = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = 0; c < 3; ++c) {
        P[0][c] = dot2(B, s.c0[c], A, F[0][c]);                       // 57
        P[1][c] = dot2(B, s.c1[c], A, F[1][c]);
        P[2][c] = dot2(B, s.c2[c], A, F[2][c]);
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int k = 0; k < 3; ++k) top |= hi(P[k][c]) ^ (hi(P[k][c]) >> 31);
    }
    if (lin) {
        for (int c = 0; c < 3; ++c) {
            lin->cof[0][c] = whole(s.c0[c]); lin->cof[1][c] = whole(s.c1[c]); lin->cof[2][c] = whole(s.c2[c]);
            for (int k = 0; k < 3; ++k) lin->F[k][c] = C.x[k][c];
        }
        lin->alpha = s.alpha;
        lin->beta = s.beta;
        const i64 a13 = mul_third(mul(split(shl(s.alpha, 2)), s.inv));             // alpha / (3 J), 60
        lin->a1 = -shl(a13, 1);
        const i64 e = s.beta - mul_third(mul(split(shl(a13, 2)), split(shl(n, 2))));   // 57, below 9
        lin->b1 = (whole(kap2) >> 4) - mul(s.inv, split(shl(e, 2)));               // 57
    }
    return !out_of_range(g) && top < kOne25;
}

// Directional derivative dP[G] (nh_tangent.cuh) of one Gauss point and the parameter contractions
// pk = P_kappa : G (60 fraction bits) and pm = P_mu : G (56).  G is scaled so that every Walsh coefficient of
// the direction is below 2^58 (|G_ij| < 0.32, 61 fraction bits); dP has 56 fraction bits and is below 2.
// Checked besides the force's range: |dJ| < 1 and the bracket of dbeta below 4.  Against a 113-bit
// reference the element action is closer than the same formula in double (tests/test_fixed_point.py).
OSAM_HD bool tangent_point(const Cols& C, const Cols& E, D kap2, D mu, D mu3, i64 dP[3][3], i64& pk, i64& pm) {
    D F[3][3], N[3][3], G[3][3];
    i64 n = 0;
    Range g;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < 3; ++k) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = 0; c < 3; ++c) {
            F[k][c] = split(C.x[k][c]);
            N[k][c] = split(-C.x[k][c]);
            G[k][c] = split(E.x[k][c]);
        }
        const i64 m = norm3(F[k][0], F[k][1], F[k][2]);
        g.nmax = g.nmax > (unsigned int)hi(m) ? g.nmax : (unsigned int)hi(m);
        n += m;
    }
    const NhPoint s = nh_point(F[0], F[1], F[2], N[1], N[2], n, kap2, mu, mu3, g);
    i64 dJ = dot3(s.c0[0], G[0][0], s.c0[1], G[0][1], s.c0[2], G[0][2]);
    dJ += dot3(s.c1[0], G[1][0], s.c1[1], G[1][1], s.c1[2], G[1][2]);
    dJ += dot3(s.c2[0], G[2][0], s.c2[1], G[2][1], s.c2[2], G[2][2]);   // 58, below 3.6
    i64 FG = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < 3; ++k) FG += dot3(F[k][0], G[k][0], F[k][1], G[k][1], F[k][2], G[k][2]);   // 58, below 2.4
    bool ok = !out_of_range(g) && (hi(dJ) ^ (hi(dJ) >> 31)) < (1 << 26);
    const D dJd = split(shl(dJ, 4));                                   // 62
    const D al = split(shl(s.alpha, 2));                               // 62
    const D nd = split(shl(n, 2));                                     // 60
    const D FGd = split(shl(FG, 2));                                   // 60
    // dalpha = -2/3 alpha dJ / J, below 2
    const i64 a13 = mul_third(mul(al, s.inv));                         // alpha / (3 J), 60
    const i64 da = -mul(split(shl(a13, 2)), dJd);                      // 59
    // dbeta = [(2 kap2 J - beta) dJ - (dalpha trC + 2 alpha F:G) / 3] / J
    const i64 cf = shl(mul(kap2, split(shl(s.J, 3))), 1) - shl(s.beta, 2);      // 59, below 8
    const i64 T = mul(split(shl(da, 2)), nd) + mul(al, FGd);                    // 57
    const i64 Q = mul(split(cf), dJd) - mul_third(T);                           // 57, below 14
    ok = ok && (hi(Q) ^ (hi(Q) >> 31)) < (4 << 25) - 1;
    const D db = split(mul(s.inv, split(shl(Q, 4))));                  // 59
    const D be = split(shl(s.beta, 2)), dad = split(da), ah = split((s.alpha + 1) >> 1);   // 59
    int top = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int a = 0; a < 3; ++a) {
        const int b = (a + 1) % 3, c = (a + 2) % 3;
        const i64 d0 = dot4(G[1][b], F[2][c], G[1][c], N[2][b], F[1][b], G[2][c], N[1][c], G[2][b]);   // 58, below 1.7
        const i64 d1 = dot4(G[2][b], F[0][c], G[2][c], N[0][b], F[2][b], G[0][c], N[2][c], G[0][b]);
        const i64 d2 = dot4(G[0][b], F[1][c], G[0][c], N[1][b], F[0][b], G[1][c], N[0][c], G[1][b]);
        dP[0][a] = dot4(db, s.c0[a], be, split(shl(d0, 3)), dad, F[0][a], ah, G[0][a]);                // 56
        dP[1][a] = dot4(db, s.c1[a], be, split(shl(d1, 3)), dad, F[1][a], ah, G[1][a]);
        dP[2][a] = dot4(db, s.c2[a], be, split(shl(d2, 3)), dad, F[2][a], ah, G[2][a]);
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int k = 0; k < 3; ++k) top |= hi(dP[k][a]) ^ (hi(dP[k][a]) >> 31);
    }
    const D jd = split(shl(shl(s.J, 2) - s.invJ, 2));                  // J - 1/J, 62
    pk = (mul(jd, dJd) + 1) >> 1;                                      // (J - 1/J) dJ / 2, 60
    const i64 qn = mul_third(mul(split(mul(s.r3, s.inv)), nd));        // J^-5/3 trC / 3, 56
    pm = (mul(s.r3, FGd) - mul(split(shl(qn, 4)), dJd) + 2) >> 2;      // 56
    return ok && top < kOne25;
}

// dP[G] of a Gauss point from its stored linearisation, dalpha = a1 dJ and dbeta = b1 dJ + a1 (F : G): a third of
// tangent_point's instructions.  q in the units of stress_point (a1, b1 with 60 and 57 fraction bits); G, dP and
// the checks as in tangent_point.
OSAM_HD bool tangent_stored(const Linear& q, const Cols& E, i64 dP[3][3]) {
    D F[3][3], N[3][3], G[3][3], c[3][3];
    i64 dJ = 0, FG = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < 3; ++k) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int a = 0; a < 3; ++a) {
            F[k][a] = split(q.F[k][a]);
            N[k][a] = split(-q.F[k][a]);
            G[k][a] = split(E.x[k][a]);
            c[k][a] = split(q.cof[k][a]);
        }
        dJ += dot3(c[k][0], G[k][0], c[k][1], G[k][1], c[k][2], G[k][2]);      // 58, below 3.6
        FG += dot3(F[k][0], G[k][0], F[k][1], G[k][1], F[k][2], G[k][2]);      // 58, below 2.4
    }
    bool ok = (hi(dJ) ^ (hi(dJ) >> 31)) < (1 << 26);
    const D dJd = split(shl(dJ, 4)), a1 = split(shl(q.a1, 1));                 // 62, 61 (below 2)
    const D dad = split(mul(a1, dJd));                                         // 59
    // |b1| < 8 with 59 fraction bits; dbeta below 8
    ok = ok && (hi(q.b1) ^ (hi(q.b1) >> 31)) < (8 << 25);
    const i64 dbeta = dot2(split(shl(q.b1, 2)), dJd, a1, split(shl(FG, 2)));   // 57
    ok = ok && (hi(dbeta) ^ (hi(dbeta) >> 31)) < (8 << 25);
    const D db = split(shl(dbeta, 2)), be = split(shl(q.beta, 2)), ah = split((q.alpha + 1) >> 1);   // 59
    int top = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int x = 0; x < 3; ++x) {
        const int y = (x + 1) % 3, z = (x + 2) % 3;
        const i64 d0 = dot4(G[1][y], F[2][z], G[1][z], N[2][y], F[1][y], G[2][z], N[1][z], G[2][y]);   // 58, below 1.7
        const i64 d1 = dot4(G[2][y], F[0][z], G[2][z], N[0][y], F[2][y], G[0][z], N[2][z], G[0][y]);
        const i64 d2 = dot4(G[0][y], F[1][z], G[0][z], N[1][y], F[0][y], G[1][z], N[0][z], G[1][y]);
        dP[0][x] = dot4(db, c[0][x], be, split(shl(d0, 3)), dad, F[0][x], ah, G[0][x]);                // 56
        dP[1][x] = dot4(db, c[1][x], be, split(shl(d1, 3)), dad, F[1][x], ah, G[1][x]);
        dP[2][x] = dot4(db, c[2][x], be, split(shl(d2, 3)), dad, F[2][x], ah, G[2][x]);
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int k = 0; k < 3; ++k) top |= hi(dP[k][x]) ^ (hi(dP[k][x]) >> 31);
    }
    return ok && top < kOne25;
}

// ---- operands with a block exponent --------------------------------------------------------------
// The 8 nodal values of one component of an element's direction (or linear displacement) share one
// exponent e: value = V 2^(e - 1081), |V| < 2^59, exact for values within 2^-6 of the largest, else rounded at
// 2^-60 of it.  So differences of nearly equal values stay exact in each component; the Walsh coefficients of
// the three components are then brought to one exponent, the largest coefficient in [2^57, 2^58).
OSAM_HD unsigned int hi_word(double x) {
    unsigned long long b;
#ifdef __CUDA_ARCH__
    b = (unsigned long long)__double_as_longlong(x);
#else
    __builtin_memcpy(&b, &x, 8);
#endif
    return (unsigned int)(b >> 32);
}
// biased exponent with the sign bit off (the maximum of hi_word() & 0x7fffffff, shifted)
OSAM_HD i64 block_value(double x, int emax) {
    unsigned long long b;
#ifdef __CUDA_ARCH__
    b = (unsigned long long)__double_as_longlong(x);
#else
    __builtin_memcpy(&b, &x, 8);
#endif
    const int e = (int)((b >> 52) & 0x7ff), s = emax - e;
    if (e == 0 || s > 60) return 0;
    const unsigned long long m = ((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 6;
    const i64 v = (i64)((m + ((1ULL << s) >> 1)) >> s);
    return (i64)b < 0 ? -v : v;
}
OSAM_HD int lead_zeros(i64 x) {   // of a non-negative value
    if (x == 0) return 64;
#ifdef __CUDA_ARCH__
    return __clzll(x);
#else
    return __builtin_clzll((unsigned long long)x);
#endif
}
OSAM_HD i64 mag(i64 x) { return x ^ (x >> 63); }
// x 2^n, rounded if n < 0 (|x| < 2^62)
OSAM_HD i64 shift(i64 x, int n) {
    if (n >= 0) return shl(x, n);
    return n < -62 ? 0 : (x + ((i64)1 << (-n - 1))) >> -n;
}
// exponent of a component's largest coefficient (of magnitudes or-ed into any); kNoExponent for zero
constexpr int kNoExponent = -100000;
OSAM_HD int top_exponent(i64 any, int e) { return any == 0 ? kNoExponent : e - lead_zeros(any); }

// Saint Venant-Kirchhoff stress of one Gauss point.  H = G 2^-base (G below 0.32 with 61 fraction bits, base >= -2: gradients of order one):
//   2 E = H + H^T + H^T H,  S = lam/2 tr(2 E) I + mu (2 E),  P = S + H S,
// everything in units of 2^-base, so the accuracy is relative to the largest gradient however small it is.  l2, mu: lam/2
// and mu with 62 fraction bits (any sign); P[column][component] with 56, below 2.
OSAM_HD bool svk_point(const Cols& C, int base, D l2, D mu, i64 P[3][3]) {
    D G[3][3];
    i64 S[3][3], tr = 0;
    bool wide = false;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < 3; ++k)
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = 0; c < 3; ++c) G[k][c] = split(C.x[k][c]);
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int i = 0; i < 3; ++i)
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int j = i; j < 3; ++j) {
            const i64 q = dot3(G[i][0], G[j][0], G[i][1], G[j][1], G[i][2], G[j][2]);      // 58, below 0.31
            const i64 e = C.x[j][i] + C.x[i][j] + shift(shl(q, 3), -base);                  // 61, below 2
            S[i][j] = mul(mu, split(e));                                                    // 59
            if (i == j) {   // each below 1.3, so that their sum keeps its 61 bits
                tr += e;
                wide |= (hi(e) ^ (hi(e) >> 31)) >= (int)(1.3 * (1 << 29));
            }
        }
    const i64 lt = mul(l2, split(tr));                                                      // 59
    D s[3][3];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int i = 0; i < 3; ++i) {
        S[i][i] += lt;
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int j = i; j < 3; ++j) {
            s[i][j] = split(S[i][j]);
            S[j][i] = S[i][j];
            s[j][i] = s[i][j];
        }
    }
    int top = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int j = 0; j < 3; ++j)
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = 0; c < 3; ++c) {
            const i64 hs = dot3(G[0][c], s[0][j], G[1][c], s[1][j], G[2][c], s[2][j]);      // 56
            P[j][c] = ((S[c][j] + 4) >> 3) + shift(hs, -base);
            top |= hi(P[j][c]) ^ (hi(P[j][c]) >> 31);
        }
    return base >= -2 && !wide && top < kOne25;
}

// Two factors a, b (any finite values) as integers with a common exponent: value = A 2^(e - 1084), |A| < 2^62
OSAM_HD int factor_exponent(double a, double b) {
    const unsigned int x = hi_word(a) & 0x7fffffffu, y = hi_word(b) & 0x7fffffffu;
    return (int)((x > y ? x : y) >> 20);
}
OSAM_HD i64 factor_value(double x, int e) { return shl(block_value(x, e), 3); }

// Material factors kappa/2 and mu times w as integers: value = X 2^(k - 62), the larger in [2^61, 2^62);
// false unless both are positive and finite
struct Material {
    D kap2, mu, mu3;
    int k;
};
OSAM_HD bool material(double lam, double mu, double w, Material& M) {
    const int e = factor_exponent(lam, mu), ew = factor_exponent(w, 0.0);
    const i64 l = factor_value(lam, e), m = factor_value(mu, e);
    const D wd = split(factor_value(w, ew));
    const i64 K = mul(split((l >> 1) + mul_third(m)), wd), U = mul(split(m), wd);
    if (e == 2047 || ew == 2047 || ew == 0 || K <= 0 || U <= 0) return false;
    const int n = lead_zeros(K | U) - 2;
    const i64 us = shl(U, n);
    M.kap2 = split(shl(K, n));
    M.mu = split(us);
    M.mu3 = split(mul_third(us));
    M.k = e + ew - 2042 - n;     // 2 x 1084 - 64 - 62
    return true;
}

// An element's forces are computed in its own unit 2^k and kept in the buffer's unit 2^top (one per mesh, so that a
// node sums integers).  Down to kMaxDown binades below it they are rounded to that unit: 2^-54 of it is then still
// below the FP64 formula's error (contrast 8 at a strain of 1e-3: 1.7e-13 of the force, FP64 3.9e-13); a softer element
// keeps its own rounding and is held in FP64.
constexpr int kMaxDown = 3;

// ---- linear elasticity ---------------------------------------------------------------------------
// Element force of isotropic linear elasticity in the Walsh basis of the 8 corners.  With raw Walsh
// coefficients w_S of the nodal values (S a set of axes: signs of those axes), the 2x2x2 Gauss sums of
// sigma(grad u) grad N are diagonal in the sign patterns (they are orthogonal on the Gauss points), so
//   F(s) = h/16 sum_S f_S s^S,
//   f_i   of component i: lam tr + 2 mu w_i^i (tr = w_x^x + w_y^y + w_z^z), of component c: mu (w_i^c + w_c^i),
//   f_ij  of component i: [lam (w_ij^i + w_jk^k) + 3 mu w_ij^i] / 3,
//         of component k: mu (2 w_ij^k + w_jk^i + w_ik^j) / 3   (k: the third axis),
//   f_xyz of component c: (lam + 4 mu) w_xyz^c / 9:
// the 1/sqrt3 of the Gauss points enters squared only, and no stress at a point is formed.  About 60
// products per element against 300 with the tensor-product interpolation.
// w: [component][pattern] with pattern bits x = 1, y = 2, z = 4, |w| < 2^59; lam, mu < 2^62; f: [component][pattern],
// w lam / 2^64, below 2^62.
OSAM_HD void le_coefficients(const i64 w[3][8], i64 lam, i64 mu, i64 f[3][8]) {
    const D L = split(lam), M = split(mu);
    const i64 lt = mul(L, split(w[0][1] + w[1][2] + w[2][4]));
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int i = 0; i < 3; ++i) {
        const int j = (i + 1) % 3, k = (i + 2) % 3;
        const int I = 1 << i, J = 1 << j, K = 1 << k;
        f[i][0] = 0;
        f[i][I] = mul_add(M, split(2 * w[i][I]), lt);
        const i64 sh = mul(M, split(w[i][J] + w[j][I]));
        f[i][J] = sh;
        f[j][I] = sh;
        // patterns {i, j} and {i, k} of component i, {j, k} of component i
        f[i][I | J] = mul_third(mul_add(L, split(w[i][I | J] + w[k][J | K]), mul(M, split(3 * w[i][I | J]))));
        f[i][I | K] = mul_third(mul_add(L, split(w[i][I | K] + w[j][J | K]), mul(M, split(3 * w[i][I | K]))));
        f[i][J | K] = mul_third(mul(M, split(2 * w[i][J | K] + w[j][I | K] + w[k][I | J])));
        const i64 x = mul_add(L, split(w[i][7]), mul(M, split(4 * w[i][7])));
        f[i][7] = mul_third(mul_third(x));
    }
}

// The Walsh coefficients of an element's 24 nodal values in block format, |w| < 2^58, coefficient =
// w 2^(T + 6 - 1081) (T = kNoExponent and w = 0 without differences); false for values that are not finite or
// subnormal
OSAM_HD bool block_walsh(const double U[3][8], i64 w[3][8], int& T) {
    int e[3];
    bool bad = false;
    T = kNoExponent;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = 0; c < 3; ++c) {
        unsigned int top = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int a = 0; a < 8; ++a) {
            const unsigned int h = hi_word(U[c][a]) & 0x7fffffffu;
            top = top > h ? top : h;
        }
        e[c] = (int)(top >> 20);
        bad |= e[c] == 2047;
        if (e[c] == 0) {                       // all zero, or subnormal
            unsigned long long bits = 0;
            for (int a = 0; a < 8; ++a) {
                unsigned long long b;
                __builtin_memcpy(&b, &U[c][a], 8);
                bits |= b << 1;
            }
            bad |= bits != 0;
        }
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int a = 0; a < 8; ++a) w[c][a] = block_value(U[c][a], e[c]);
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int b = 1; b < 8; b <<= 1)
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int a = 0; a < 8; ++a)
                if (!(a & b)) {
                    const i64 lo = w[c][a], up = w[c][a | b];
                    w[c][a] = lo + up;
                    w[c][a | b] = up - lo;
                }
        i64 any = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int a = 1; a < 8; ++a) any |= mag(w[c][a]);
        T = imax(T, top_exponent(any, e[c]));
    }
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = 0; c < 3; ++c) {
        w[c][0] = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int a = 1; a < 8; ++a) w[c][a] = T == kNoExponent ? 0 : shift(w[c][a], e[c] - T - 6);
    }
    return !bad;
}

// The 24 nodal forces of an element from the Walsh coefficients of its displacements (block_walsh): the
// coefficients above, the inverse sums.  lam, mu: Lame parameters times the factor h / 16 (divided by the factor
// that the displacements carry).  Returns false for operands outside the formats (or so small or large that the
// result's exponent leaves the normal range): the caller then uses FP64.
OSAM_HD double f64_scaled(i64 x, int scale);
OSAM_HD bool force_le_walsh(const i64 w[3][8], int T, double lam, double mu, double F[3][8]) {
    const int ek = factor_exponent(lam, mu);
    const bool zero = T == kNoExponent;
    const int scale = 2095 - T - ek;           // 1081 + 1084 - 64 - 6
    if (ek == 2047 || (!zero && (scale > 1000 || scale < -900))) return false;
    i64 f[3][8];
    // |w| < 2^58: 4 w fits beside it, and the 7 terms of a corner below 2^61 each
    le_coefficients(w, factor_value(lam, ek), factor_value(mu, ek), f);
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = 0; c < 3; ++c) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int b = 1; b < 8; b <<= 1)
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int a = 0; a < 8; ++a)
                if (!(a & b)) {
                    const i64 lo = f[c][a], up = f[c][a | b];
                    f[c][a] = lo - up;
                    f[c][a | b] = lo + up;
                }
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int a = 0; a < 8; ++a) F[c][a] = f64_scaled(f[c][a], scale);
    }
    return true;
}
OSAM_HD bool element_force_le(const double U[3][8], double lam, double mu, double F[3][8]) {
    i64 w[3][8];
    int T;
    return block_walsh(U, w, T) && force_le_walsh(w, T, lam, mu, F);
}

// y . dK/dlam u and y . dK/dmu u of an element in units of h / 16, from the Walsh coefficients of u and y: with
// K's coefficients above, sums of products that are symmetric in u and y,
//   lam: tr tr' + sum_j S_j S_j' / 3 + sum_c w_xyz^c w_xyz^c' / 9,   S_j = w_ij^i + w_jk^k,
//   mu:  2 sum w_i^i w_i^i' + sum_(i<c) (w_i^c + w_c^i)(w_i^c + w_c^i)'
//        + sum [3 w_ij^i w_ij^i' + 3 w_ij^j w_ij^j' + (2 w_ij^k + w_jk^i + w_ik^j) w_ij^k'] / 3 + 4 sum w_xyz^c w_xyz^c' / 9.
// Operands are raised by 2 bits each (below 2^62), so a product is a b 2^4 / 2^64 and every sum below 2^63.
OSAM_HD void contract_le(const i64 u[3][8], const i64 y[3][8], i64& dl, i64& dm) {
    const auto dot = [](i64 a, i64 b) { return mul(split(shl(a, 2)), split(shl(b, 2))); };
    i64 l1 = dot(u[0][1] + u[1][2] + u[2][4], y[0][1] + y[1][2] + y[2][4]), l2 = 0, l3 = 0, m1 = 0, m2 = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int i = 0; i < 3; ++i) {
        const int j = (i + 1) % 3, k = (i + 2) % 3;
        const int I = 1 << i, J = 1 << j, K = 1 << k;
        l2 += dot(u[i][I | J] + u[k][J | K], y[i][I | J] + y[k][J | K]);
        l3 += dot(u[i][7], y[i][7]);
        m1 += 2 * dot(u[i][I], y[i][I]) + dot(u[i][J] + u[j][I], y[i][J] + y[j][I]);
        m2 += dot(3 * u[i][I | J], y[i][I | J]) + dot(3 * u[j][I | J], y[j][I | J]);
        m2 += dot(2 * u[k][I | J] + u[i][J | K] + u[j][I | K], y[k][I | J]);
    }
    const i64 n = mul_third(mul_third(l3));
    dl = l1 + mul_third(l2) + n;
    dm = m1 + mul_third(m2) + 4 * n;
}

// x / 2^scale as an FP64 value, rounded to nearest (integer operations; |x| < 2^63)
OSAM_HD double f64_scaled(i64 x, int scale) {
    if (x == 0) return 0.0;
    const unsigned long long s = x < 0 ? 0x8000000000000000ULL : 0ULL;
    unsigned long long m = x < 0 ? 0ULL - (unsigned long long)x : (unsigned long long)x;
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)m);
#else
    const int lz = __builtin_clzll(m);
#endif
    m <<= lz;                                  // leading bit at 63: value m 2^(-lz - scale)
    const int e = 1023 + 63 - lz - scale;      // biased exponent of the leading bit
    const unsigned long long b = s | (((unsigned long long)(e - 1) << 52) + (m >> 11) + ((m >> 10) & 1));
    double r;
#ifdef __CUDA_ARCH__
    r = __longlong_as_double((long long)b);
#else
    __builtin_memcpy(&r, &b, 8);
#endif
    return r;
}

// x / 2^scale as an FP32 value, rounded toward zero (integer operations; zero below the normal range, largest
// exponent above it)
OSAM_HD float f32_scaled(i64 x, int scale) {
    if (x == 0) return 0.0f;
    const unsigned long long m = x < 0 ? 0ULL - (unsigned long long)x : (unsigned long long)x;
    const int lz = lead_zeros((i64)(m >> 1)) - 1;       // m < 2^63
    const int e = 127 + 63 - lz - scale;
    const unsigned int f = (unsigned int)((m << lz) >> 40);   // 24 bits, leading bit set
    const unsigned int b = (x < 0 ? 0x80000000u : 0u) |
                           (e < 1 ? 0u : e > 254 ? 0x7f800000u : ((unsigned int)(e - 1) << 23) + f);
    float r;
#ifdef __CUDA_ARCH__
    r = __uint_as_float(b);
#else
    __builtin_memcpy(&r, &b, 4);
#endif
    return r;
}

// An element buffer entry is an integer force (below 2^60: four equal leading bits) or, for an element outside the
// integer path, the FP64 force itself: its leading bits differ for every value in -2^769 .. 2^-767 and 2^-767 .. inf
// and for NaN.  The others have codes: zero (and what rounds to it, below 2^-767) is stored as -0, -inf (and what
// lies below -2^769) as a NaN of its own.  A group whose unit is outside 2^+-kMaxUnit does not take this buffer.
constexpr int kMaxUnit = 500;
constexpr i64 kMinusInf = 0x7ff8000000000002LL;
OSAM_HD bool held_f64(i64 x) { return (unsigned int)((hi(x) >> 28) + 1) > 1u; }
OSAM_HD i64 hold_f64(double v) {
    i64 b;
#ifdef __CUDA_ARCH__
    b = __double_as_longlong(v);
#else
    __builtin_memcpy(&b, &v, 8);
#endif
    if (held_f64(b)) return b;
    if (b >= 0) return (i64)1 << 63;
    return shl(b, 1) > shl(0x7ff0000000000000LL, 1) ? 0x7ff8000000000000LL : kMinusInf;   // NaN, or -2^769 and below
}
OSAM_HD double f64_held(i64 b) {
    if (b == kMinusInf) b = (i64)0xfff0000000000000ULL;
    double v;
#ifdef __CUDA_ARCH__
    v = __longlong_as_double(b);
#else
    __builtin_memcpy(&v, &b, 8);
#endif
    return v;
}

// x (positive, normal) as m 2^(e - 62), m in [2^62, 2^63 - 2^31) (or half of that, where x's mantissa is within 2^-32 of 2):
// a value that split() takes
inline void mantissa63(double x, long long& m, int& e) {
    int k;
    m = (long long)std::ldexp(std::frexp(x, &k), 63);
    e = k - 1;
    if (m >= 0x7fffffff80000000LL) {
        m >>= 1;       // exact: a double's mantissa leaves the low 10 bits zero
        ++e;
    }
}

// fixed-point u / h of a nodal displacement: the mantissa as 62 bits (63 would not split near 2) times the mantissa of 1/h
// (mantissa63: 1/h = ihm 2^(ihe - 62)), shifted to 59 fraction bits; kBadU for |u| / h >= 12 and for non-finite values.
OSAM_HD i64 fixed_u(double u, i64 ihm, int ihe) {
    unsigned long long b;
#ifdef __CUDA_ARCH__
    b = (unsigned long long)__double_as_longlong(u);
#else
    __builtin_memcpy(&b, &u, 8);
#endif
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return 0;                                     // zero and subnormals
    const i64 m = (i64)(((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 9);    // [2^61, 2^62)
    const i64 p = mul(m, ihm);                                // [2^58, 2^61): u/h = p 2^(e - 1023 + ihe - 59)
    const int s = 1023 - e - ihe;                             // right shift to 59 fraction bits
    if (s < -3) return kBadU;                                 // (p 2^4 could leave 64 bits)
    i64 v;
    if (s <= 0) v = shl(p, -s);
    else v = s > 62 ? 0 : (p + ((i64)1 << (s - 1))) >> s;
    if (v >= (i64)kMaxU << kFracU || v < 0) return kBadU;
    return (i64)b < 0 ? -v : v;
}

// The same for an element with a node beyond the format: u / h modulo 32 edges, so that differences inside the element
// are exact while they stay below 16 edges, and with 8 fraction bits in `coarse`, which tells whether they do.  False
// for |u| / h >= 2^22 and for non-finite values.
constexpr int kCoarseSpread = 702;   // 2.75 edges, less the cut of two values
OSAM_HD bool wrapped_u(double u, i64 ihm, int ihe, i64& v, int& coarse) {
    unsigned long long b;
#ifdef __CUDA_ARCH__
    b = (unsigned long long)__double_as_longlong(u);
#else
    __builtin_memcpy(&b, &u, 8);
#endif
    v = coarse = 0;
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return true;
    const i64 p = mul((i64)(((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 9), ihm);
    const int s = 1023 - e - ihe;                             // u / h in [2^(-1 - s), 2^(2 - s))
    if (s < -20) return false;
    if (s <= 0) v = shl(p, -s);
    else v = s > 62 ? 0 : (p + ((i64)1 << (s - 1))) >> s;
    coarse = s + 51 > 62 ? 0 : (int)(p >> (s + 51));
    if ((i64)b < 0) {
        v = (i64)(0ULL - (unsigned long long)v);
        coarse = -coarse;
    }
    return true;
}

// one component of such an element: its 8 nodal values again; true if it is out of range all the same
OSAM_HD bool refit(const double U[8], i64 ihm, int ihe, i64 V[8]) {
    int mx = -0x7fffffff, mn = 0x7fffffff;
    bool bad = false;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int a = 0; a < 8; ++a) {
        int x;
        bad |= !wrapped_u(U[a], ihm, ihe, V[a], x);
        mx = imax(mx, x);
        mn = imin(mn, x);
    }
    return bad || mx - mn >= kCoarseSpread;                   // |x| < 2^30
}

}  // namespace fx
}  // namespace osam
