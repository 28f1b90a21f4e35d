// Neo-Hookean element kernels with one element on 8 lanes (lanes.cuh), in 64-bit integers: the element-level
// force and its vector-Jacobian product, the force of the implicit Newton residual and the tangent action of
// its CG iterations.
//
// The FP64 forms were bound by the FP64 pipe at every size: a warp that carries 32 elements issues 720
// (force) to 1500 (vector-Jacobian product) FP64 instructions of 67 to 80 cycles, 25 to 55 us however few elements
// there are.  Here a Gauss point takes about 250 (force) or 550 (tangent) integer multiply-adds of 4 cycles, and
// 8 lanes per element put 8 times as many warps in flight on a small mesh.  An element outside the formats'
// range is evaluated in FP64 by one of its lanes.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "hex8_math.cuh"
#include "lanes.cuh"
#include "nh_tangent.cuh"
#include "osam_internal.h"

namespace osam {

namespace {

using namespace fx;

constexpr int kLaneBlock = 128;                   // 16 elements
// Blocks per SM asked of the compiler: the lane kernels wait on their own results, so warps in flight count.
// 64x64x64, force 149.9 us at the natural 157 registers, 143.7 at 128, 139.5 at 5 blocks; vector-Jacobian product
// 361.8 at 248 registers, 306 at 168, 301 at 128 (20x20x40: 31.1, 26.8, 24.9).
constexpr int kForceBlocks = 5, kTangentBlocks = 4;

// FP64 evaluation of one element (all 24 values, parameter contractions) for operands outside the formats.
// x(c, corner) and p(c, corner) read the displacement and the direction.  Not inlined into the lane path's registers.
struct FarIn {
    const double *u, *p;
    int usn, psn;
    long long usc, psc;
    int n0, sy, sz;
    double invh, lam, mu, wq, wq3;
    __device__ long long node(int c8) const { return n0 + (c8 & 1) + ((c8 >> 1) & 1) * sy + ((c8 >> 2) & 1) * (long long)sz; }
};

__device__ __noinline__ void far_force(const FarIn& x, double F[3][8]) {
    using namespace hex8;
    double Dx[3][2][2], Dy[3][2][2], Dz[3][2][2], m1, m2, m3;
    material_factors<OSAM_NEO_HOOKEAN, double>(x.lam, x.mu, x.wq, x.wq3, m1, m2, m3);
    for (int c = 0; c < 3; ++c) {
        double U[8];
        for (int c8 = 0; c8 < 8; ++c8) U[c8] = x.u[c * x.usc + x.node(c8) * x.usn];
        edge_differences<double>(U, x.invh, Dx[c], Dy[c], Dz[c]);
    }
    element_force<OSAM_NEO_HOOKEAN, double>(Dx, Dy, Dz, m1, m2, m3, F);
}

__device__ __noinline__ void far_tangent(const FarIn& x, double F[3][8], double& lb, double& mb) {
    using namespace hex8;
    double Gx[3][2][2], Gy[3][2][2], Gz[3][2][2], Bx[3][2][2], By[3][2][2], Bz[3][2][2], m1, m2, m3;
    material_factors<OSAM_NEO_HOOKEAN, double>(x.lam, x.mu, x.wq, x.wq3, m1, m2, m3);
    for (int c = 0; c < 3; ++c) {
        double U[8], Dx[2][2], Dy[2][2], Dz[2][2];
        for (int c8 = 0; c8 < 8; ++c8) U[c8] = x.u[c * x.usc + x.node(c8) * x.usn];
        edge_differences<double>(U, x.invh, Dx, Dy, Dz);
        lerp2(Dx, Gx[c]); lerp2(Dy, Gy[c]); lerp2(Dz, Gz[c]);
        for (int c8 = 0; c8 < 8; ++c8) U[c8] = x.p[c * x.psc + x.node(c8) * x.psn];
        edge_differences<double>(U, x.invh, Dx, Dy, Dz);
        lerp2(Dx, Bx[c]); lerp2(Dy, By[c]); lerp2(Dz, Bz[c]);
    }
    double Sx[3][2][2] = {}, Sy[3][2][2] = {}, Sz[3][2][2] = {};
    lb = mb = 0.0;
    for (int g = 0; g < 8; ++g) {
        const int p = g >> 2, q = (g >> 1) & 1, r = g & 1;
        double H[3][3], G[3][3], dP[3][3], pk, pm;
        for (int c = 0; c < 3; ++c) {
            H[c][0] = Gx[c][q][r]; H[c][1] = Gy[c][p][r]; H[c][2] = Gz[c][p][q];
            G[c][0] = Bx[c][q][r]; G[c][1] = By[c][p][r]; G[c][2] = Bz[c][p][q];
        }
        tangent::nh_tangent(H, G, m1, m2, m3, dP, pk, pm);
        lb += pk;
        mb = fma(2.0 / 3.0, pk, mb + pm);
        for (int c = 0; c < 3; ++c) { Sx[c][q][r] += dP[c][0]; Sy[c][p][r] += dP[c][1]; Sz[c][p][q] += dP[c][2]; }
    }
    walsh_transpose<double>(Sx, Sy, Sz, F);
}

// The Newton linearisation of the tangent: F, cof F, alpha, beta and the coefficients of
// dalpha = a1 dJ and dbeta = b1 dJ + a1 (F : G), dJ = cof : G, per Gauss point; layout [kLinPerGp][8 Gauss points][NE],
// Gauss point 4 x + 2 y + z:
//   a1 = -2/3 alpha / J,  b1 = 2 kappa/2 - (a1 trC / 3 + beta) / J   (from P = alpha F + beta cof,
//   alpha = mu J^-2/3, beta = (kappa/2 (J^2 - 1) - mu/3 J^-2/3 trC) / J).
static_assert(kLinPerGp == 22, "stored linearisation: F, cof F, alpha, beta, a1, b1");
__device__ __forceinline__ int lin_point(int a) { return 4 * (a & 1) + (a & 2) + (a >> 2); }

struct LinStore {
    float* lin;          // this element's first entry
    long long ne;        // stride between Gauss points
    double kap2;         // m1 of the material factors
    __device__ void operator()(int p, int q, int r, const double (&Fm)[3][3], const double (&Cm)[3][3], double, double trC,
                               double invJ, double alpha, double beta) const {
        const double a1 = -(2.0 / 3.0) * alpha * invJ;
        const double b1 = 2.0 * kap2 - invJ * fma(a1, trC * (1.0 / 3.0), beta);
        const long long st = 8 * ne;
        float* lg = lin + (long long)(4 * p + 2 * q + r) * ne;
        for (int a = 0; a < 9; ++a) {
            lg[a * st] = (float)Fm[a / 3][a % 3];
            lg[(9 + a) * st] = (float)Cm[a / 3][a % 3];
        }
        lg[18 * st] = (float)alpha; lg[19 * st] = (float)beta; lg[20 * st] = (float)a1; lg[21 * st] = (float)b1;
    }
};

__device__ __noinline__ void far_linearise(const FarIn& x, float* lin, long long ne, double F[3][8]) {
    using namespace hex8;
    double Gx[3][2][2], Gy[3][2][2], Gz[3][2][2], Sx[3][2][2], Sy[3][2][2], Sz[3][2][2], m1, m2, m3;
    material_factors<OSAM_NEO_HOOKEAN, double>(x.lam, x.mu, x.wq, x.wq3, m1, m2, m3);
    for (int c = 0; c < 3; ++c) {
        double U[8], Dx[2][2], Dy[2][2], Dz[2][2];
        for (int c8 = 0; c8 < 8; ++c8) U[c8] = x.u[c * x.usc + x.node(c8) * x.usn];
        edge_differences<double>(U, x.invh, Dx, Dy, Dz);
        lerp2<double>(Dx, Gx[c], c == 0); lerp2<double>(Dy, Gy[c], c == 1); lerp2<double>(Dz, Gz[c], c == 2);
    }
    nh_gauss_sums<double>(Gx, Gy, Gz, m1, m2, m3, Sx, Sy, Sz, LinStore{lin, ne, m1});
    walsh_transpose<double>(Sx, Sy, Sz, F);
}

// The element of a lane group in one mesh; lanes beyond the last element repeat it (all lanes take part in
// the shuffles) and write nothing
struct Elem {
    int e, n0, sy, sz;
    bool live;
};
__device__ __forceinline__ Elem element(int e, int nx, int ny, int ne) {
    Elem x;
    x.live = e < ne;
    x.e = x.live ? e : ne - 1;
    const int i = x.e % nx, t = x.e / nx, j = t % ny, k = t / ny;
    x.sy = nx + 1;
    x.sz = (nx + 1) * (ny + 1);
    x.n0 = i + x.sy * j + x.sz * k;
    return x;
}
__device__ __forceinline__ int corner_node(const Elem& x, int a) {
    return x.n0 + (a & 1) + ((a >> 1) & 1) * x.sy + (a >> 2) * x.sz;
}

// ---- element level: one mesh, strided operands (ElemArgs) ----------------------------------------
template <int MODE>
__device__ __forceinline__ void put(const ElemArgs& a, const Elem& x, int corner, int c, double v) {
    if (MODE == kAtomic)
        atomicAdd(static_cast<double*>(a.f) + (long long)c * a.fsc + (long long)corner_node(x, corner) * a.fsn, v);
    else
        static_cast<double*>(a.fe)[(long long)(corner * 3 + c) * a.ne + x.e] = v;
}

__device__ __forceinline__ FarIn far_in(const ElemArgs& a, const Elem& x, const double* p, int psn, long long psc,
                                        double lam, double mu) {
    return FarIn{a.u, p, a.usn, psn, a.usc, psc, x.n0, x.sy, x.sz, a.invh, lam, mu, a.wq, a.wq3};
}

template <int MODE>
__global__ void __launch_bounds__(kLaneBlock, kForceBlocks) k_elem_force(const __grid_constant__ ElemArgs a, i64 ihm, int ihe) {
    const Elem x = element((int)(blockIdx.x * (kLaneBlock / 8) + (threadIdx.x >> 3)), a.nx, a.ny, a.ne);
    const Lane L = make_lane();
    const int node = corner_node(x, L.a);
    i64 U[3], F[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) U[c] = fixed_u(a.u[(long long)c * a.usc + (long long)node * a.usn], ihm, ihe);
    const double lam = a.lam_e ? a.lam_e[x.e] : a.lam, mu = a.mu_e ? a.mu_e[x.e] : a.mu;
    Material M;
    bool bad = !material(lam, mu, a.wq, M);
    refit_lanes([&](int c) { return a.u[(long long)c * a.usc + (long long)node * a.usn]; }, ihm, ihe, U, bad);
    const bool ok = force_lanes(L, U, M.kap2, M.mu, M.mu3, bad || M.k < -900 || M.k > 900, F);
    if (!x.live) return;
    if (ok) {
#pragma unroll
        for (int c = 0; c < 3; ++c) put<MODE>(a, x, L.a, c, f64_scaled(F[c], 57 - M.k));
    } else if (L.a == 0) {
        double Ff[3][8];
        far_force(far_in(a, x, nullptr, 0, 0, lam, mu), Ff);
        for (int c8 = 0; c8 < 8; ++c8)
            for (int c = 0; c < 3; ++c) put<MODE>(a, x, c8, c, Ff[c][c8]);
    }
}

// the same with one thread per element (the arithmetic of force_fx.cu)
template <int MODE>
__device__ __forceinline__ bool thread_force(const ElemArgs& a, const Elem& x, const WalshIn w[3], bool bad) {
    const double lam = a.lam_e ? a.lam_e[x.e] : a.lam, mu = a.mu_e ? a.mu_e[x.e] : a.mu;
    Material M;
    bad |= !material(lam, mu, a.wq, M) || M.k < -900 || M.k > 900;
    i64 F[3][8];
    bad |= !element_force_nh(w, whole(M.kap2), whole(M.mu), whole(M.mu3), F);
    if (bad) return false;
#pragma unroll
    for (int c8 = 0; c8 < 8; ++c8)
#pragma unroll
        for (int c = 0; c < 3; ++c) put<MODE>(a, x, c8, c, f64_scaled(F[c][c8], kFracOut - M.k));
    return true;
}

// ... with a node beyond the format: the element's values modulo 32 edges
template <int MODE>
__device__ __noinline__ void moved_force(const ElemArgs& a, const Elem& x, i64 ihm, int ihe) {
    WalshIn w[3];
    bool bad = false;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        double X[8];
        i64 V[8];
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8) X[c8] = a.u[(long long)c * a.usc + (long long)corner_node(x, c8) * a.usn];
        bad |= refit(X, ihm, ihe, V);
        w[c] = walsh_in(V, c);
    }
    if (thread_force<MODE>(a, x, w, bad)) return;
    double Ff[3][8];
    far_force(far_in(a, x, nullptr, 0, 0, a.lam_e ? a.lam_e[x.e] : a.lam, a.mu_e ? a.mu_e[x.e] : a.mu), Ff);
    for (int c8 = 0; c8 < 8; ++c8)
        for (int c = 0; c < 3; ++c) put<MODE>(a, x, c8, c, Ff[c][c8]);
}

template <int MODE>
__global__ void __launch_bounds__(128) k_elem_force_thread(const __grid_constant__ ElemArgs a, i64 ihm, int ihe) {
    const int first = blockIdx.x * 128 + (int)threadIdx.x;
    if (first >= a.ne) return;
    const Elem x = element(first, a.nx, a.ny, a.ne);
    WalshIn w[3];
    bool bad = false;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        i64 V[8];
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8)
            V[c8] = fixed_u(a.u[(long long)c * a.usc + (long long)corner_node(x, c8) * a.usn], ihm, ihe);
        bad |= spread_bad(V);
        w[c] = walsh_in(V, c);
    }
    if (!thread_force<MODE>(a, x, w, bad)) moved_force<MODE>(a, x, ihm, ihe);
}

// Element-level force: 8 lanes per element up to this many elements, above it one thread per element, which
// shares the columns of F among the Gauss points and issues half of the instructions (8 lanes against one thread:
// 432 elements 9.4 and 17.7 us, 54000 36.1 and 37.2, 110592 63.7 and 53.6, 884736 451 and 363)
constexpr int kLaneElements = 65536;

template <int MODE>
__global__ void __launch_bounds__(kLaneBlock, kTangentBlocks) k_elem_vjp(const __grid_constant__ ElemArgs a, const double* ybar, int ysn,
                                                         long long ysc, double* lam_bar, double* mu_bar, int accumulate,
                                                         i64 ihm, int ihe, double wqi, double vol) {
    const Elem x = element((int)(blockIdx.x * (kLaneBlock / 8) + (threadIdx.x >> 3)), a.nx, a.ny, a.ne);
    const Lane L = make_lane();
    const int node = corner_node(x, L.a);
    i64 U[3], F[3], pk = 0, pm = 0;
    double p[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        U[c] = fixed_u(a.u[(long long)c * a.usc + (long long)node * a.usn], ihm, ihe);
        p[c] = ybar[(long long)c * ysc + (long long)node * ysn];
    }
    const double lam = a.lam_e ? a.lam_e[x.e] : a.lam, mu = a.mu_e ? a.mu_e[x.e] : a.mu;
    Material M;
    bool bad = !material(lam, mu, wqi, M);
    refit_lanes([&](int c) { return a.u[(long long)c * a.usc + (long long)node * a.usn]; }, ihm, ihe, U, bad);
    int scale, base;
    const bool ok = tangent_lanes(L, U, p, M, bad, lam_bar || mu_bar, F, scale, pk, pm, base);
    if (!x.live) return;
    double lb = 0.0, mb = 0.0;
    if (ok) {
#pragma unroll
        for (int c = 0; c < 3; ++c) put<MODE>(a, x, L.a, c, f64_scaled(F[c], scale));
        lb = vol * f64_scaled(pk, 60 + base);
        mb = vol * f64_scaled(pm, 56 + base);
    } else if (L.a == 0) {
        double Ff[3][8];
        far_tangent(far_in(a, x, ybar, ysn, ysc, lam, mu), Ff, lb, mb);
        for (int c8 = 0; c8 < 8; ++c8)
            for (int c = 0; c < 3; ++c) put<MODE>(a, x, c8, c, Ff[c][c8]);
        lb *= a.w8 / a.invh;
        mb *= a.w8 / a.invh;
    }
    if (L.a != 0) return;
    if (lam_bar) lam_bar[x.e] = (accumulate ? lam_bar[x.e] : 0.0) + lb;
    if (mu_bar) mu_bar[x.e] = (accumulate ? mu_bar[x.e] : 0.0) + mb;
}

// ---- implicit groups (FomB): element buffer [24][NE] ----------------------------------------------
// OP kOpTangent: K(u) p of the CG direction from the stored linearisation; else the internal force of u, which
// also stores it (in FP32 for k_tangent_lin32_b, or as integers).  The u-dependent part of the tangent does not
// change over the CG iterations of a Newton step (12 of them on average): with it stored a tangent launch issues
// 1000 instead of 2700 instructions per warp.
enum { kOpStore32, kOpStore64, kOpTangent };
template <int OP>
__global__ void __launch_bounds__(kLaneBlock, OP == kOpTangent ? kTangentBlocks : kForceBlocks) k_fom_lanes(const __grid_constant__ FomB g, const int* __restrict__ mask) {
    constexpr bool TANGENT = OP == kOpTangent;
    const int per = g.eblock * 8 / kLaneBlock;   // thread blocks per element block
    const int2 b = g.eblk[blockIdx.x / per];
    if (mask && !mask[b.x]) return;
    const InstFom& I = g.inst[b.x];
    const int first = b.y + (int)(blockIdx.x % per) * (kLaneBlock / 8);
    if (first >= I.ne) return;
    const Elem x = element(first + (int)(threadIdx.x >> 3), I.nx, I.ny, I.ne);
    const Lane L = make_lane();
    const long long gn = I.node_off + corner_node(x, L.a), st = 8LL * g.NE;
    const double lam = I.lam_e ? I.lam_e[x.e] : I.lam, mu = I.mu_e ? I.mu_e[x.e] : I.mu;
    // FP32: [22][8 Gauss points][NE] for the one-thread-per-element tangent; integers: [22][NE][8 lanes], 256
    // consecutive bytes per warp
    const long long entry = OP == kOpStore32 ? I.elem_off + x.e + (long long)lin_point(L.a) * g.NE : 8 * (I.elem_off + x.e) + L.a;
    Material M;
    bool bad = !material(lam, mu, I.wq, M) || M.k < -900 || M.k > 900;
    i64 F[3];
    Linear q;
    int scale;
    bool ok;
    if (TANGENT) {
        const i64* lg = g.lin + entry;
        double p[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            p[c] = g.cg_p[c * g.NN + gn];
#pragma unroll
            for (int d = 0; d < 3; ++d) { q.F[d][c] = __ldg(lg + (3 * c + d) * st); q.cof[d][c] = __ldg(lg + (9 + 3 * c + d) * st); }
        }
        q.alpha = __ldg(lg + 18 * st); q.beta = __ldg(lg + 19 * st);
        q.a1 = __ldg(lg + 20 * st); q.b1 = __ldg(lg + 21 * st);
        ok = tangent_stored_lanes(L, q, p, M.k + I.ihe + 1, bad || q.alpha == kBadF, F, scale);
    } else {
        i64 U[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) U[c] = fixed_u(g.u[0][c * g.NN + gn], I.ihm, I.ihe);
        refit_lanes([&](int c) { return g.u[0][c * g.NN + gn]; }, I.ihm, I.ihe, U, bad);
        ok = force_lanes(L, U, M.kap2, M.mu, M.mu3, bad, F, &q);
        scale = 57 - M.k;
    }
    if (!x.live) return;
    if (OP == kOpStore32 && ok) {
        float* lg = g.linf + entry;
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                lg[(3 * c + d) * st] = f32_scaled(q.F[d][c], 61);
                lg[(9 + 3 * c + d) * st] = f32_scaled(q.cof[d][c], 61);
            }
        lg[18 * st] = f32_scaled(q.alpha, 60 - M.k);
        lg[19 * st] = f32_scaled(q.beta, 57 - M.k);
        lg[20 * st] = f32_scaled(q.a1, 60 - M.k);
        lg[21 * st] = f32_scaled(q.b1, 57 - M.k);
    }
    if (OP == kOpStore64) {
        i64* lg = g.lin + entry;
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                lg[(3 * c + d) * st] = q.F[d][c];
                lg[(9 + 3 * c + d) * st] = q.cof[d][c];
            }
        // the factors times 1/h: ihm 2^-63 of it here, the rest in the tangent's exponent
        const D r = split(I.ihm);
        lg[18 * st] = ok ? shl(mul(split(q.alpha), r), 1) : kBadF;
        lg[19 * st] = shl(mul(split(q.beta), r), 1);
        lg[20 * st] = shl(mul(split(q.a1), r), 1);
        lg[21 * st] = shl(mul(split(q.b1), r), 1);
    }
    double* fe = static_cast<double*>(g.fe) + I.elem_off + x.e;
    if (ok) {
#pragma unroll
        for (int c = 0; c < 3; ++c) fe[(long long)(L.a * 3 + c) * g.NE] = f64_scaled(F[c], scale);
    } else if (L.a == 0) {
        const FarIn in{g.u[0] + I.node_off, TANGENT ? g.cg_p + I.node_off : nullptr, 1, 1, g.NN, g.NN, x.n0, x.sy, x.sz,
                       I.invh, lam, mu, I.wq, I.wq3};
        double Ff[3][8], lb, mb;
        if (TANGENT) far_tangent(in, Ff, lb, mb);
        else if (OP == kOpStore32) far_linearise(in, g.linf + I.elem_off + x.e, g.NE, Ff);
        else far_force(in, Ff);
        for (int c8 = 0; c8 < 8; ++c8)
            for (int c = 0; c < 3; ++c) fe[(long long)(c8 * 3 + c) * g.NE] = Ff[c][c8];
    }
}

int elem_grid(int ne) { return grid_for(8LL * ne, kLaneBlock); }

}  // namespace

void fixed_point_inverse(double x, long long& m, int& e) {
    mantissa63(x, m, e);
}

cudaError_t launch_elem_force_nh(int scatter, const ElemArgs& a, cudaStream_t s, int lanes) {
    long long m;
    int e;
    fixed_point_inverse(a.invh, m, e);
    if (lanes < 0 ? a.ne > kLaneElements : !lanes) {
        if (scatter == kAtomic) k_elem_force_thread<kAtomic><<<grid_for(a.ne, 128), 128, 0, s>>>(a, m, e);
        else k_elem_force_thread<kGather><<<grid_for(a.ne, 128), 128, 0, s>>>(a, m, e);
        return cudaGetLastError();
    }
    if (scatter == kAtomic) k_elem_force<kAtomic><<<elem_grid(a.ne), kLaneBlock, 0, s>>>(a, m, e);
    else k_elem_force<kGather><<<elem_grid(a.ne), kLaneBlock, 0, s>>>(a, m, e);
    return cudaGetLastError();
}

cudaError_t launch_elem_vjp_nh(int scatter, const ElemArgs& a, const double* ybar, int ysn, long long ysc,
                               double* lam_bar, double* mu_bar, int acc, cudaStream_t s) {
    long long m;
    int e;
    fixed_point_inverse(a.invh, m, e);
    const double wqi = a.wq * a.invh, vol = a.w8;   // h^3 / 8 per Gauss point; the gradients carry 1 / h
    if (scatter == kAtomic)
        k_elem_vjp<kAtomic><<<elem_grid(a.ne), kLaneBlock, 0, s>>>(a, ybar, ysn, ysc, lam_bar, mu_bar, acc, m, e, wqi, vol);
    else
        k_elem_vjp<kGather><<<elem_grid(a.ne), kLaneBlock, 0, s>>>(a, ybar, ysn, ysc, lam_bar, mu_bar, acc, m, e, wqi, vol);
    return cudaGetLastError();
}

cudaError_t launch_imp_force_nh_b(const FomB& g, const int* mask, cudaStream_t s) {
    if (g.eblock % 32) return cudaErrorInvalidValue;
    const int grid = g.n_eblk * (g.eblock * 8 / kLaneBlock);
    if (g.linf) k_fom_lanes<kOpStore32><<<grid, kLaneBlock, 0, s>>>(g, mask);
    else if (g.lin) k_fom_lanes<kOpStore64><<<grid, kLaneBlock, 0, s>>>(g, mask);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_imp_tangent_nh_b(const FomB& g, const int* mask, cudaStream_t s) {
    if (g.eblock % 32 || !g.lin) return cudaErrorInvalidValue;
    k_fom_lanes<kOpTangent><<<g.n_eblk * (g.eblock * 8 / kLaneBlock), kLaneBlock, 0, s>>>(g, mask);
    return cudaGetLastError();
}

}  // namespace osam
