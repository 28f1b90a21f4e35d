// Saint Venant-Kirchhoff element force in 64-bit integers, 8 lanes per element (lanes.cuh, svk_point in
// fixed_math.cuh): element level and the batched groups (explicit step, implicit Newton residual).
//
// The FP64 kernels issue about 750 FP64 instructions of 67 to 80 cycles per warp of 32 elements; a Gauss point takes
// about 170 integer multiply-adds here.  The displacement gradient has a block exponent, so small strains keep
// their relative accuracy.  An element with gradients of order one or operands that are not finite is evaluated in FP64.
#include <cuda_runtime.h>

#include <cstdint>

#include "hex8_math.cuh"
#include "lanes.cuh"
#include "osam_internal.h"
#include "trace_item.cuh"

namespace osam {

namespace {

using namespace fx;

__device__ __noinline__ void far_force_svk(const double* u, int usn, long long usc, int sy, int sz, double scale, double m1,
                                           double m2, double F[3][8]) {
    using namespace hex8;
    double Dx[3][2][2], Dy[3][2][2], Dz[3][2][2];
    for (int c = 0; c < 3; ++c) {
        double U[8];
        for (int c8 = 0; c8 < 8; ++c8)
            U[c8] = u[c * usc + (long long)((c8 & 1) + ((c8 >> 1) & 1) * sy + (c8 >> 2) * sz) * usn];
        edge_differences<double>(U, scale, Dx[c], Dy[c], Dz[c]);
    }
    element_force<OSAM_SAINT_VENANT_KIRCHHOFF, double>(Dx, Dy, Dz, m1, m2, 0.0, F);
}

template <int MODE>
__global__ void __launch_bounds__(128, 5) k_elem_force_svk(const __grid_constant__ ElemArgs a, i64 ihm, int ihe) {
    const int first = blockIdx.x * 16 + (int)(threadIdx.x >> 3), e = min(first, a.ne - 1);
    const int i = e % a.nx, t = e / a.nx, j = t % a.ny, k = t / a.ny;
    const int sy = a.nx + 1, sz = (a.nx + 1) * (a.ny + 1), n0 = i + sy * j + sz * k;
    const Lane L = make_lane();
    const auto node = [&](int c8) { return n0 + (c8 & 1) + ((c8 >> 1) & 1) * sy + (c8 >> 2) * (long long)sz; };
    const auto put = [&](int c8, int c, double v) {
        if (MODE == kAtomic) atomicAdd(static_cast<double*>(a.f) + (long long)c * a.fsc + node(c8) * a.fsn, v);
        else static_cast<double*>(a.fe)[(long long)(c8 * 3 + c) * a.ne + e] = v;
    };
    double U[3];
    i64 F[3];
    int scale;
#pragma unroll
    for (int c = 0; c < 3; ++c) U[c] = a.u[(long long)c * a.usc + node(L.a) * a.usn];
    const double m1 = (a.lam_e ? a.lam_e[e] : a.lam) * a.wq, m2 = (a.mu_e ? a.mu_e[e] : a.mu) * a.wq;
    const bool ok = force_svk_lanes(L, U, ihm, ihe, m1, m2, F, scale);
    if (first >= a.ne) return;
    if (ok) {
#pragma unroll
        for (int c = 0; c < 3; ++c) put(L.a, c, f64_scaled(F[c], scale));
    } else if (L.a == 0) {
        double Ff[3][8];
        far_force_svk(a.u + (long long)n0 * a.usn, a.usn, a.usc, sy, sz, a.invh, m1, m2, Ff);
        for (int c8 = 0; c8 < 8; ++c8)
            for (int c = 0; c < 3; ++c) put(c8, c, Ff[c][c8]);
    }
}

// 8 thread blocks of g.eblock threads per element block; trace blocks at the end of the grid
__global__ void __launch_bounds__(128, 5) k_fom_force_svk(const __grid_constant__ FomB g, const int* __restrict__ active,
                                                          const __grid_constant__ TraceFuse tr, const double* u) {
    if ((int)blockIdx.x >= 8 * g.n_eblk) {
        trace::fused_trace_block(tr, active, g, (int)blockIdx.x - 8 * g.n_eblk);
        return;
    }
    const int2 b = g.eblk[blockIdx.x >> 3];
    if (active && !active[b.x]) return;
    const InstFom& I = g.inst[b.x];
    const int first = b.y + (int)((blockIdx.x & 7u) * (blockDim.x >> 3) + (threadIdx.x >> 3)), e = min(first, I.ne - 1);
    const int nx = I.nx, ny = I.ny, i = e % nx, t = e / nx, j = t % ny, k = t / ny;
    const int sy = nx + 1, sz = (nx + 1) * (ny + 1);
    const double* x = u + I.node_off + (i + sy * j + sz * k);
    const Lane L = make_lane();
    double U[3];
    i64 F[3];
    int scale;
#pragma unroll
    for (int c = 0; c < 3; ++c) U[c] = x[(long long)c * g.NN + (L.a & 1) + ((L.a >> 1) & 1) * sy + (L.a >> 2) * sz];
    double m1 = I.m1, m2 = I.m2;
    if (I.lam_e || I.mu_e) {
        m1 = (I.lam_e ? I.lam_e[e] : I.lam) * I.wq;
        m2 = (I.mu_e ? I.mu_e[e] : I.mu) * I.wq;
    }
    const bool ok = force_svk_lanes(L, U, I.ihm, I.ihe, m1, m2, F, scale);
    if (first >= I.ne) return;
    double* fe = static_cast<double*>(g.fe) + I.elem_off + e;
    if (ok) {
#pragma unroll
        for (int c = 0; c < 3; ++c) fe[(long long)(L.a * 3 + c) * g.NE] = f64_scaled(F[c], scale);
    } else if (L.a == 0) {
        double Ff[3][8];
        far_force_svk(x, 1, g.NN, sy, sz, I.invh, m1, m2, Ff);
        for (int c8 = 0; c8 < 8; ++c8)
            for (int c = 0; c < 3; ++c) fe[(long long)(c8 * 3 + c) * g.NE] = Ff[c][c8];
    }
}

}  // namespace

cudaError_t launch_elem_force_svk(int scatter, const ElemArgs& a, cudaStream_t s) {
    const int grid = grid_for(a.ne, 16);
    long long m;
    int e;
    fixed_point_inverse(a.invh, m, e);
    if (scatter == kAtomic) k_elem_force_svk<kAtomic><<<grid, 128, 0, s>>>(a, m, e);
    else k_elem_force_svk<kGather><<<grid, 128, 0, s>>>(a, m, e);
    return cudaGetLastError();
}

cudaError_t launch_force_svk_b(const FomB& g, const int* active, const TraceFuse& tr, const double* u, cudaStream_t s) {
    if (g.eblock > 128 || !u) return cudaErrorInvalidValue;
    long long items = 0;
    for (int k = 0; k < tr.n; ++k) items += 3LL * tr.c[k].R;
    k_fom_force_svk<<<8 * g.n_eblk + (int)((items + g.eblock - 1) / g.eblock), g.eblock, 0, s>>>(g, active, tr, u);
    return cudaGetLastError();
}

}  // namespace osam
