// Host build of the displacement gradients of the kernels with a corner per lane: 64-bit sums against 128-bit ones.
// Reads 8 nodal values in edges per line; writes whether every edge is in range (edge_bad), the largest Walsh
// coefficient and gradient (with the 1 of F) in edges, and whether a 64-bit value wrapped.
#include <cmath>
#include <cstdio>

#include "fixed_math.cuh"

using namespace osam::fx;
typedef __int128 Wide;

int main() {
    double v[8];
    while (std::scanf("%lf %lf %lf %lf %lf %lf %lf %lf", v, v + 1, v + 2, v + 3, v + 4, v + 5, v + 6, v + 7) == 8) {
        i64 n[8];
        Wide N[8];
        bool ok = true, wrapped = false;
        double coefficient = 0, gradient = 0;
        for (int a = 0; a < 8; ++a) N[a] = n[a] = fixed_u(v[a], (i64)1 << 62, 0);
        for (int a = 0; a < 8; ++a)
            for (int d = 1; d < 8; d <<= 1) ok = ok && !edge_bad(hi(n[a]), hi(n[a ^ d]));
        for (int b = 1; b < 8; b <<= 1)
            for (int a = 0; a < 8; ++a)
                if (!(a & b)) {
                    const i64 l = n[a], u = n[a | b];
                    const Wide L = N[a], U = N[a | b];
                    n[a] = (i64)((unsigned long long)l + u); n[a | b] = (i64)((unsigned long long)u - l);
                    N[a] = L + U; N[a | b] = U - L;
                }
        for (int a = 1; a < 8; ++a) coefficient = std::fmax(coefficient, std::fabs((double)N[a]) * 0x1p-59);
        const double t = 1 / std::sqrt(3.0);
        for (int axis = 0; axis < 3; ++axis)
            for (int one = 0; one < 2; ++one)
                for (int g = 0; g < 8; ++g) {
                    i64 f = one ? (i64)1 << kFracF : 0;
                    double F = one;
                    for (int b = 0; b < 8; ++b) {
                        if ((b >> axis) & 1) continue;
                        const int p = b | 1 << axis, order = __builtin_popcount(p);
                        bool minus = false;
                        for (int k = 0; k < 3; ++k) minus ^= ((b >> k) & 1) && !((g >> k) & 1);
                        const i64 x = order == 2 ? mul_t(n[p]) : order == 3 ? mul_third(n[p]) : n[p];
                        f = (i64)((unsigned long long)f + (minus ? -x : x));
                        const double X = (double)N[p] * 0x1p-61 * (order == 2 ? t : order == 3 ? 1.0 / 3 : 1.0);
                        F += minus ? -X : X;
                    }
                    gradient = std::fmax(gradient, std::fabs(F));
                    wrapped = wrapped || std::fabs((double)f * 0x1p-61 - F) > 1e-9;
                }
        std::printf("%d %.6f %.6f %d\n", ok, coefficient, gradient, wrapped);
    }
}
