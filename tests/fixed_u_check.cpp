// Host build of the conversions of a nodal displacement to fixed point.  Reads "h u" per line; writes the errors of
// fixed_u and wrapped_u against u / h in units of 2^-59 (nan: marked as outside the format) and u / h.
#include <cmath>
#include <cstdio>

#include "fixed_math.cuh"

using namespace osam::fx;

int main() {
    double h, u;
    while (std::scanf("%lf %lf", &h, &u) == 2) {
        long long ihm;
        int ihe, coarse;
        mantissa63(1 / h, ihm, ihe);
        const long double x = (long double)u * (long double)(1 / h);
        const i64 v = fixed_u(u, ihm, ihe);
        i64 w;
        const bool ok = wrapped_u(u, ihm, ihe, w, coarse);
        const auto error = [&](i64 a) {
            const long double y = a * 0x1p-59L, d = y - x;
            return (double)((d - 32 * std::round(d / 32)) * 0x1p59L);
        };
        std::printf("%.6e %.6e %.17g %d\n", v == kBadU ? NAN : error(v), ok ? error(w) : NAN, (double)x, coarse);
    }
}
