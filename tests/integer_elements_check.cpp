// Host build of the integer linear elastic force and Neo-Hookean tangent action against the same operators in
// extended precision.  Reads "h lam mu" and 24 displacements and 24 directions [component][corner] per line; writes
// "ok" of the two and the rms errors (integers, the same formula in double) of the linear elastic force of the
// direction and of the tangent action, relative to the largest exact entry, and of the two parameter contractions
// in units of h^2 times the largest difference of the direction; then "ok" and the errors of the Saint
// Venant-Kirchhoff force of the displacement.
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "fixed_math.cuh"

using namespace osam::fx;
typedef long double Real;

template <class T>
struct Shape {
    T B[8][8][3], w;
    explicit Shape(double h) : w(T(h) * h * h / 8) {
        const T s3 = std::sqrt(T(3)), g[2] = {(1 - 1 / s3) / 2, (1 + 1 / s3) / 2};
        for (int p = 0; p < 8; ++p)
            for (int a = 0; a < 8; ++a) {
                T l[3], d[3];
                for (int k = 0; k < 3; ++k) {
                    const T x = g[(p >> k) & 1];
                    l[k] = (a >> k) & 1 ? x : 1 - x;
                    d[k] = ((a >> k) & 1 ? 1 : -1) / T(h);
                }
                B[p][a][0] = d[0] * l[1] * l[2]; B[p][a][1] = l[0] * d[1] * l[2]; B[p][a][2] = l[0] * l[1] * d[2];
            }
    }
    void grad(const double x[3][8], int p, T G[3][3]) const {
        for (int c = 0; c < 3; ++c)
            for (int k = 0; k < 3; ++k) {
                G[c][k] = 0;
                for (int a = 1; a < 8; ++a) G[c][k] += (T(x[c][a]) - T(x[c][0])) * B[p][a][k];
            }
    }
    void add(const T P[3][3], int p, T F[26]) const {
        for (int c = 0; c < 3; ++c)
            for (int a = 0; a < 8; ++a)
                for (int k = 0; k < 3; ++k) F[8 * c + a] += w * P[c][k] * B[p][a][k];
    }
};

template <class T>
void linear(const double x[3][8], double h, double lam, double mu, T F[26]) {
    const Shape<T> S(h);
    for (int p = 0; p < 8; ++p) {
        T G[3][3], P[3][3];
        S.grad(x, p, G);
        for (int c = 0; c < 3; ++c)
            for (int k = 0; k < 3; ++k)
                P[c][k] = T(mu) * (G[c][k] + G[k][c]) + (c == k ? T(lam) * (G[0][0] + G[1][1] + G[2][2]) : T(0));
        S.add(P, p, F);
    }
}

// F[24], F[25]: the contractions with the derivative by lambda and mu
template <class T>
void tangent(const double u[3][8], const double x[3][8], double h, double lam, double mu, T R[26]) {
    const Shape<T> S(h);
    const T kap = T(lam) + T(2) / 3 * T(mu);
    for (int p = 0; p < 8; ++p) {
        T F[3][3], G[3][3], C[3][3], dC[3][3], P[3][3], tr = 0, FG = 0, dJ = 0, J = 0;
        S.grad(u, p, F);
        S.grad(x, p, G);
        for (int c = 0; c < 3; ++c) F[c][c] += 1;
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) {
                const int a = (i + 1) % 3, b = (i + 2) % 3, k = (j + 1) % 3, l = (j + 2) % 3;
                C[i][j] = F[a][k] * F[b][l] - F[a][l] * F[b][k];
                dC[i][j] = G[a][k] * F[b][l] + F[a][k] * G[b][l] - G[a][l] * F[b][k] - F[a][l] * G[b][k];
                tr += F[i][j] * F[i][j];
                FG += F[i][j] * G[i][j];
                dJ += C[i][j] * G[i][j];
            }
        for (int j = 0; j < 3; ++j) J += F[0][j] * C[0][j];
        const T r = std::cbrt(J), r3 = 1 / (r * r), al = T(mu) * r3, be = kap / 2 * (J - 1 / J) - T(mu) / 3 * r3 / J * tr;
        const T da = -T(2) / 3 * al / J * dJ, db = ((kap * J - be) * dJ - (da * tr + 2 * al * FG) / 3) / J;
        for (int c = 0; c < 3; ++c)
            for (int k = 0; k < 3; ++k) P[c][k] = db * C[c][k] + be * dC[c][k] + da * F[c][k] + al * G[c][k];
        S.add(P, p, R);
        const T pk = (J - 1 / J) * dJ / 2, pm = r3 * FG - r3 / J * tr / 3 * dJ;
        R[24] += S.w * pk;
        R[25] += S.w * (pm + T(2) / 3 * pk);
    }
}

// the lane kernels' transforms, one pattern / Gauss point / corner after the other
static void sums(i64 v[8]) {
    for (int b = 1; b < 8; b <<= 1)
        for (int a = 0; a < 8; ++a)
            if (!(a & b)) { const i64 l = v[a], u = v[a | b]; v[a] = l + u; v[a | b] = u - l; }
}
static i64 scaled(i64 x, int a) {
    const int order = (a & 1) + ((a >> 1) & 1) + (a >> 2);
    return order == 2 ? mul_t(x) : order == 3 ? mul_third(x) : x;
}
static bool minus(int pattern, int g) {   // the sign of a pattern at Gauss point g
    bool m = false;
    for (int k = 0; k < 3; ++k) m ^= ((pattern >> k) & 1) && !((g >> k) & 1);
    return m;
}
static void columns(const i64 w[3][8], int g, Cols& C) {
    for (int d = 0; d < 3; ++d)
        for (int c = 0; c < 3; ++c) {
            C.x[d][c] = 0;
            for (int b = 0; b < 8; ++b)
                if (!((b >> d) & 1)) C.x[d][c] += minus(b, g) ? -w[c][b | 1 << d] : w[c][b | 1 << d];
        }
}
static bool tangent_fixed(const double u[3][8], const double x[3][8], double h, double lam, double mu, double R[26]) {
    i64 ihm, wu[3][8], wx[3][8], o[3][8] = {}, ks = 0, ms = 0;
    int e, k, ex[3], T = kNoExponent;
    ihm = (i64)std::ldexp(std::frexp(1 / h, &e), 63);
    bool ok = true;
    for (int c = 0; c < 3; ++c) {
        unsigned int top = 0;
        for (int a = 0; a < 8; ++a) top = std::fmax(top, hi_word(x[c][a]) & 0x7fffffffu);
        ex[c] = top >> 20;
        for (int a = 0; a < 8; ++a) { wu[c][a] = fixed_u(u[c][a], ihm, e - 1); wx[c][a] = block_value(x[c][a], ex[c]); }
        ok = ok && !spread_bad(wu[c]);
        sums(wu[c]);
        sums(wx[c]);
        wu[c][1 << c] += (i64)1 << kFracF;
        for (int a = 1; a < 8; ++a) T = imax(T, top_exponent(mag(wx[c][a]), ex[c]));
    }
    for (int c = 0; c < 3; ++c)
        for (int a = 1; a < 8; ++a) {
            wx[c][a] = T == kNoExponent ? 0 : scaled(shift(wx[c][a], ex[c] - T - 6), a);
            wu[c][a] = scaled(wu[c][a], a);
        }
    const double m1 = 0.5 * (lam + 2.0 / 3 * mu) * h / 32, m2 = mu * h / 32;
    std::frexp(std::fmax(m1, m2), &k);
    const i64 m = std::llrint(std::ldexp(m2, 62 - k));
    for (int g = 0; g < 8; ++g) {
        Cols C, G;
        i64 P[3][3], pk, pm;
        columns(wu, g, C);
        columns(wx, g, G);
        const D k2 = split(std::llrint(std::ldexp(m1, 62 - k))), m2d = split(m), m3 = split(mul_third(m));
        ok = tangent_point(C, G, k2, m2d, m3, P, pk, pm) && ok;
        // from the stored linearisation: dbeta is rounded at 2^-57 in four places, times cof below 2.25, against the
        // unit 2^-56 of dP, and dP itself once more: 8 units
        Linear lin;
        i64 S[3][3], Q[3][3];
        ok = stress_point(C, k2, m2d, m3, S, &lin) && tangent_stored(lin, G, Q) && ok;
        for (int d = 0; d < 3; ++d)
            for (int c = 0; c < 3; ++c) ok = ok && std::llabs(Q[d][c] - P[d][c]) <= 8;
        ks += pk;
        ms += pm;
        for (int b = 1; b < 8; ++b)
            for (int d = 0; d < 3; ++d)
                if ((b >> d) & 1)
                    for (int c = 0; c < 3; ++c) o[c][b] += minus(b & ~(1 << d), g) ? -P[d][c] : P[d][c];
    }
    const int base = T == kNoExponent ? 0 : 1016 - T;
    for (int c = 0; c < 3; ++c) {
        for (int b = 1; b < 8; ++b) o[c][b] = scaled(o[c][b], b);
        for (int b = 1; b < 8; b <<= 1)
            for (int a = 0; a < 8; ++a)
                if (!(a & b)) { const i64 l = o[c][a], v = o[c][a | b]; o[c][a] = l - v; o[c][a | b] = l + v; }
        for (int a = 0; a < 8; ++a) R[8 * c + a] = f64_scaled(o[c][a], 56 + base - k);
    }
    R[24] = h * h / 8 * f64_scaled(ks, 60 + base);
    R[25] = h * h / 8 * f64_scaled(ms + (mul_third(ks) >> 3), 56 + base);
    return ok;
}

// Saint Venant-Kirchhoff force from displacements divided by h
template <class T>
void svk(const double v[3][8], double h, double lam, double mu, T F[26]) {
    const Shape<T> S(1.0);
    for (int p = 0; p < 8; ++p) {
        T H[3][3], E[3][3], P[3][3], tr = 0;
        S.grad(v, p, H);
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) {
                E[i][j] = H[i][j] + H[j][i];
                for (int c = 0; c < 3; ++c) E[i][j] += H[c][i] * H[c][j];
                E[i][j] /= 2;
                if (i == j) tr += E[i][j];
            }
        for (int c = 0; c < 3; ++c)
            for (int j = 0; j < 3; ++j) {
                P[c][j] = 0;
                for (int k = 0; k < 3; ++k)
                    P[c][j] += (H[c][k] + (c == k)) * (2 * T(mu) * E[k][j] + (k == j ? T(lam) * tr : T(0))) * T(h) * T(h);
            }
        S.add(P, p, F);
    }
}
static bool svk_fixed(const double v[3][8], double h, double lam, double mu, double R[26]) {
    i64 w[3][8], o[3][8] = {};
    int T;
    bool ok = block_walsh(v, w, T);
    const int base = T == kNoExponent ? 0 : 1016 - T;
    for (int c = 0; c < 3; ++c)
        for (int a = 1; a < 8; ++a) w[c][a] = scaled(w[c][a], a);
    const double m1 = lam * h * h / 32, m2 = mu * h * h / 32;
    const int e = factor_exponent(m1, m2);
    for (int g = 0; g < 8; ++g) {
        Cols G;
        i64 P[3][3];
        columns(w, g, G);
        ok = svk_point(G, base, split((factor_value(m1, e) + 1) >> 1), split(factor_value(m2, e)), P) && ok;
        for (int b = 1; b < 8; ++b)
            for (int d = 0; d < 3; ++d)
                if ((b >> d) & 1)
                    for (int c = 0; c < 3; ++c) o[c][b] += minus(b & ~(1 << d), g) ? -P[d][c] : P[d][c];
    }
    for (int c = 0; c < 3; ++c) {
        for (int b = 1; b < 8; ++b) o[c][b] = scaled(o[c][b], b);
        for (int b = 1; b < 8; b <<= 1)
            for (int a = 0; a < 8; ++a)
                if (!(a & b)) { const i64 l = o[c][a], u = o[c][a | b]; o[c][a] = l - u; o[c][a | b] = l + u; }
        for (int a = 0; a < 8; ++a) R[8 * c + a] = f64_scaled(o[c][a], 56 + base - (e - 1022));
    }
    return ok;
}

template <class A>
static double error(const A* x, const Real* y, int n) {
    Real s = 0, t = 0;
    for (int i = 0; i < n; ++i) { s += (x[i] - y[i]) * (x[i] - y[i]); t = std::fmax(t, std::fabs(y[i])); }
    return t > 0 ? (double)(std::sqrt(s / n) / t) : (double)std::sqrt(s / n);
}

int main() {
    double h, lam, mu, v[48], (*u)[8] = reinterpret_cast<double (*)[8]>(v), (*x)[8] = u + 3;
    while (std::scanf("%lf %lf %lf", &h, &lam, &mu) == 3) {
        for (double& a : v)
            if (std::scanf("%lf", &a) != 1) return 1;
        Real E[26] = {}, T[26] = {};
        double Ed[26] = {}, Td[26] = {}, Tf[26] = {}, Ef[3][8];
        linear<Real>(x, h, lam, mu, E);
        linear<double>(x, h, lam, mu, Ed);
        tangent<Real>(u, x, h, lam, mu, T);
        tangent<double>(u, x, h, lam, mu, Td);
        const bool a = element_force_le(x, lam * (h / 16), mu * (h / 16), Ef);
        const bool b = tangent_fixed(u, x, h, lam, mu, Tf);
        Real top = 0;
        for (int c = 0; c < 3; ++c)
            for (int k = 0; k < 8; ++k) top = std::fmax(top, std::fabs((Real)x[c][k] - (Real)x[c][0]));
        top *= (Real)h * h;
        const auto part = [&](const double* f, int k) { return (double)(std::fabs(f[k] - T[k]) / top); };
        Real V[26] = {};
        double Vd[26] = {}, Vf[26] = {}, y[3][8];   // the displacement divided by h, exact in the reference
        for (int c = 0; c < 3; ++c)
            for (int k = 0; k < 8; ++k) y[c][k] = u[c][k] / h;
        svk<Real>(y, h, lam, mu, V);
        svk<double>(y, h, lam, mu, Vd);
        const bool v3 = svk_fixed(y, h, lam, mu, Vf);
        std::printf("%d %d %.3e %.3e %.3e %.3e %.3e %.3e %.3e %.3e %d %.3e %.3e\n", a, b, error(&Ef[0][0], E, 24), error(Ed, E, 24),
                    error(Tf, T, 24), error(Td, T, 24), part(Tf, 24), part(Td, 24), part(Tf, 25), part(Td, 25),
                    v3, error(Vf, V, 24), error(Vd, V, 24));
    }
}
