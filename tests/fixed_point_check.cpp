// Host build of the fixed-point Neo-Hookean element force against the formula of Appendix A.3 in
// extended precision.  Reads "h lam mu" and 24 displacements [component][corner] per line, writes "ok" and the
// largest errors (fixed point, the same formula in double) in units of mu h^2.
#include <cmath>
#include <cstdio>

#include "fixed_math.cuh"

using namespace osam::fx;

template <class T>
static void reference(const double u[3][8], double h, double lam, double mu, T F[3][8]) {
    const T kap = T(lam) + T(2) / T(3) * T(mu), w = T(h) * T(h) * T(h) / 8, s3 = std::sqrt(T(3));
    const T g[2] = {(1 - 1 / s3) / 2, (1 + 1 / s3) / 2};
    for (int c = 0; c < 3; ++c)
        for (int a = 0; a < 8; ++a) F[c][a] = 0;
    for (int gp = 0; gp < 8; ++gp) {
        const T p[3] = {g[gp & 1], g[(gp >> 1) & 1], g[gp >> 2]};
        T B[8][3], D[3][3], C[3][3];
        for (int a = 0; a < 8; ++a) {
            T l[3], d[3];
            for (int k = 0; k < 3; ++k) {
                const int s = (a >> k) & 1;
                l[k] = s ? p[k] : 1 - p[k];
                d[k] = (s ? 1 : -1) / T(h);
            }
            B[a][0] = d[0] * l[1] * l[2]; B[a][1] = l[0] * d[1] * l[2]; B[a][2] = l[0] * l[1] * d[2];
        }
        T tr = 0;
        for (int c = 0; c < 3; ++c)
            for (int k = 0; k < 3; ++k) {
                T t = c == k;
                for (int a = 0; a < 8; ++a) t += T(u[c][a]) * B[a][k];
                D[c][k] = t;
                tr += t * t;
            }
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) {
                const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, j1 = (j + 1) % 3, j2 = (j + 2) % 3;
                C[i][j] = D[i1][j1] * D[i2][j2] - D[i1][j2] * D[i2][j1];
            }
        const T J = D[0][0] * C[0][0] + D[0][1] * C[0][1] + D[0][2] * C[0][2];
        const T c3 = std::cbrt(J), r3 = 1 / (c3 * c3);
        const T al = T(mu) * r3, be = (kap / 2 * (J * J - 1) - T(mu) / 3 * r3 * tr) / J;
        for (int c = 0; c < 3; ++c)
            for (int a = 0; a < 8; ++a)
                for (int k = 0; k < 3; ++k) F[c][a] += w * (al * D[c][k] + be * C[c][k]) * B[a][k];
    }
}

int main() {
    double h, lam, mu, u[3][8];
    while (std::scanf("%lf %lf %lf", &h, &lam, &mu) == 3) {
        for (auto& r : u)
            for (double& x : r)
                if (std::scanf("%lf", &x) != 1) return 1;
        long double R[3][8];
        double P[3][8];
        reference<long double>(u, h, lam, mu, R);
        reference<double>(u, h, lam, mu, P);
        int e, k;
        const i64 ihm = (i64)std::ldexp(std::frexp(1 / h, &e), 63);
        const double wq = h * h / 32, m1 = 0.5 * (lam + 2.0 / 3 * mu) * wq, m2 = mu * wq;
        std::frexp(std::fmax(m1, m2), &k);
        const i64 mui = std::llrint(std::ldexp(m2, 62 - k));
        i64 V[3][8], F[3][8];
        WalshIn w[3];
        bool ok = true;
        for (int c = 0; c < 3; ++c) {
            for (int a = 0; a < 8; ++a) V[c][a] = fixed_u(u[c][a], ihm, e - 1);
            ok = ok && !spread_bad(V[c]);
            w[c] = walsh_in(V[c], c);
        }
        ok = element_force_nh(w, std::llrint(std::ldexp(m1, 62 - k)), mui, mul_third(mui), F) && ok;
        double ef = 0, ed = 0;
        for (int c = 0; c < 3; ++c)
            for (int a = 0; a < 8; ++a) {
                const long double sc = mu * h * h;
                ef = std::fmax(ef, (double)std::fabs((f64_scaled(F[c][a], 54 - k) - R[c][a]) / sc));
                ed = std::fmax(ed, (double)std::fabs((P[c][a] - R[c][a]) / sc));
            }
        std::printf("%d %.3e %.3e\n", ok, ef, ed);
    }
}
