// Host build of the fixed-point Neo-Hookean force as the explicit step keeps it: evaluated with the element's own
// material factors and rounded to the unit of a mesh whose largest factors are `contrast` times as large.  Reads
// "h lam mu contrast" and 24 displacements per line; writes "ok" and the rms errors (fixed point, the plain formula
// in double) and the rms of the force.
#define main check_one_element
#include "fixed_point_check.cpp"
#undef main

int main() {
    double h, lam, mu, contrast, u[3][8];
    while (std::scanf("%lf %lf %lf %lf", &h, &lam, &mu, &contrast) == 4) {
        for (auto& r : u)
            for (double& x : r)
                if (std::scanf("%lf", &x) != 1) return 1;
        long double R[3][8], sf = 0, sd = 0, sr = 0;
        double P[3][8];
        reference<long double>(u, h, lam, mu, R);
        reference<double>(u, h, lam, mu, P);
        int e, top;
        const i64 ihm = (i64)std::ldexp(std::frexp(1 / h, &e), 63);
        const double wq = h * h / 32;
        std::frexp(contrast * std::fmax(0.5 * (lam + 2.0 / 3 * mu), mu) * wq * (1 + 0x1p-48), &top);
        Material M;
        bool ok = material(lam, mu, wq, M);
        const int down = top - M.k;
        ok = ok && down >= 0;
        i64 V[3][8], F[3][8];
        WalshIn w[3];
        for (int c = 0; c < 3; ++c) {
            for (int a = 0; a < 8; ++a) V[c][a] = fixed_u(u[c][a], ihm, e - 1);
            ok = ok && !spread_bad(V[c]);
            w[c] = walsh_in(V[c], c);
        }
        ok = element_force_nh(w, whole(M.kap2), whole(M.mu), whole(M.mu3), F) && ok;
        for (int c = 0; c < 3; ++c)
            for (int a = 0; a < 8; ++a) {
                const double f = down > kMaxDown ? f64_scaled(F[c][a], kFracOut - M.k)
                                                 : f64_scaled(shift(F[c][a], -down), kFracOut - top);
                sf += (f - R[c][a]) * (f - R[c][a]);
                sd += (P[c][a] - R[c][a]) * (P[c][a] - R[c][a]);
                sr += R[c][a] * R[c][a];
            }
        std::printf("%d %.6Le %.6Le %.6Le\n", ok, std::sqrt(sf / 24), std::sqrt(sd / 24), std::sqrt(sr / 24));
    }
}
