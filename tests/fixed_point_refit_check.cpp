// fixed_point_check.cpp for elements anywhere: the nodal values are taken modulo 32 edges (refit).
#define main check_one_element
#include "fixed_point_check.cpp"
#undef main

int main() {
    double h, lam, mu, u[3][8];
    while (std::scanf("%lf %lf %lf", &h, &lam, &mu) == 3) {
        for (auto& r : u)
            for (double& x : r)
                if (std::scanf("%lf", &x) != 1) return 1;
        long double R[3][8];
        double P[3][8], ef = 0, ed = 0;
        reference<long double>(u, h, lam, mu, R);
        reference<double>(u, h, lam, mu, P);
        int e;
        const i64 ihm = (i64)std::ldexp(std::frexp(1 / h, &e), 63);
        Material M;
        bool ok = material(lam, mu, h * h / 32, M), edges = true;
        i64 V[3][8], F[3][8];
        WalshIn w[3];
        for (int c = 0; c < 3; ++c) {
            ok = !refit(u[c], ihm, e - 1, V[c]) && ok;
            for (int a = 0; a < 8; ++a)
                for (int d = 1; d < 8; d <<= 1) edges = edges && !edge_bad(hi(V[c][a]), hi(V[c][a ^ d]));
            w[c] = walsh_in(V[c], c);
        }
        ok = element_force_nh(w, whole(M.kap2), whole(M.mu), whole(M.mu3), F) && ok;
        for (int c = 0; c < 3; ++c)
            for (int a = 0; a < 8; ++a) {
                const long double sc = mu * h * h;
                ef = std::fmax(ef, (double)std::fabs((f64_scaled(F[c][a], kFracOut - M.k) - R[c][a]) / sc));
                ed = std::fmax(ed, (double)std::fabs((P[c][a] - R[c][a]) / sc));
            }
        std::printf("%d %.3e %.3e %d\n", ok, ef, ed, edges);
    }
}
