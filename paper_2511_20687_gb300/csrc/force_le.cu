// Linear elastic element force in the Walsh basis with block exponents (element_force_le, fixed_math.cuh):
// element level, explicit step, and (the force being linear) the tangent action of implicit groups.
//
// The FP64 tensor-product form issues about 500 FP64 instructions of 67 to 80 cycles per element; here an
// element takes about 60 integer products and 400 additions of 2 to 4 cycles, and no FP64 instruction
// (uniform material).  Its rounding is 2^-58 of the element's largest displacement gradient against 2^-53 at
// every FP64 operation.  One thread per element.
#include <cuda_runtime.h>

#include <cstdint>

#include "fixed_math.cuh"
#include "hex8_math.cuh"
#include "lanes.cuh"
#include "osam_internal.h"
#include "trace_item.cuh"

namespace osam {

namespace {

using namespace fx;

constexpr int kElemBlock = 64;   // element level: two warps, so that a small mesh spreads over the SMs

// The same element in FP64, for operands outside the formats; lam and mu carry h / 16 (material_factors: h^2 / 32).
// Reads the nodal values again, so that the integer path's operands stay in registers.
__device__ __noinline__ void far_force_le(const double* u, int usn, long long usc, int sy, int sz, double lam, double mu,
                                          double F[3][8]) {
    using namespace hex8;
    double Dx[3][2][2], Dy[3][2][2], Dz[3][2][2];
    for (int c = 0; c < 3; ++c) {
        double U[8];
        for (int c8 = 0; c8 < 8; ++c8)
            U[c8] = u[c * usc + (long long)((c8 & 1) + ((c8 >> 1) & 1) * sy + (c8 >> 2) * sz) * usn];
        edge_differences_prescaled<double>(U, Dx[c], Dy[c], Dz[c]);
    }
    element_force<OSAM_LINEAR_ELASTIC, double>(Dx, Dy, Dz, 0.5 * lam, 0.5 * mu, 0.0, F);
}

template <int MODE>
__device__ __forceinline__ void put(const ElemArgs& a, int e, int n0, int sy, int sz, int c8, int c, double v) {
    if (MODE == kAtomic) {
        const long long n = n0 + (c8 & 1) + ((c8 >> 1) & 1) * sy + (c8 >> 2) * sz;
        atomicAdd(static_cast<double*>(a.f) + (long long)c * a.fsc + n * a.fsn, v);
    } else {
        static_cast<double*>(a.fe)[(long long)(c8 * 3 + c) * a.ne + e] = v;
    }
}

template <int MODE>
__global__ void __launch_bounds__(kElemBlock) k_elem_force_le(const __grid_constant__ ElemArgs a, double w) {
    const int e = blockIdx.x * kElemBlock + threadIdx.x;
    if (e >= a.ne) return;
    const int i = e % a.nx, t = e / a.nx, j = t % a.ny, k = t / a.ny;
    const int sy = a.nx + 1, sz = (a.nx + 1) * (a.ny + 1);
    const int n0 = i + sy * j + sz * k;
    double U[3][8], F[3][8];
#pragma unroll
    for (int c8 = 0; c8 < 8; ++c8) {
        const long long n = n0 + (c8 & 1) + ((c8 >> 1) & 1) * sy + (c8 >> 2) * sz;
#pragma unroll
        for (int c = 0; c < 3; ++c) U[c][c8] = a.u[(long long)c * a.usc + n * a.usn];
    }
    const double lam = (a.lam_e ? a.lam_e[e] : a.lam) * w, mu = (a.mu_e ? a.mu_e[e] : a.mu) * w;
    if (!element_force_le(U, lam, mu, F)) {
        double Ff[3][8];
        far_force_le(a.u + (long long)n0 * a.usn, a.usn, a.usc, sy, sz, lam, mu, Ff);
        for (int c8 = 0; c8 < 8; ++c8)
            for (int c = 0; c < 3; ++c) put<MODE>(a, e, n0, sy, sz, c8, c, Ff[c][c8]);
        return;
    }
#pragma unroll
    for (int c8 = 0; c8 < 8; ++c8)
#pragma unroll
        for (int c = 0; c < 3; ++c) put<MODE>(a, e, n0, sy, sz, c8, c, F[c][c8]);
}

// the same with an element on 8 lanes
template <int MODE>
__global__ void __launch_bounds__(128) k_elem_force_le_lanes(const __grid_constant__ ElemArgs a, double w) {
    const int first = blockIdx.x * 16 + (int)(threadIdx.x >> 3), e = min(first, a.ne - 1);
    const int i = e % a.nx, t = e / a.nx, j = t % a.ny, k = t / a.ny;
    const int sy = a.nx + 1, sz = (a.nx + 1) * (a.ny + 1);
    const int n0 = i + sy * j + sz * k;
    const Lane L = make_lane();
    const long long n = n0 + (L.a & 1) + ((L.a >> 1) & 1) * sy + (L.a >> 2) * sz;
    double U[3];
    i64 F[3];
    int scale;
#pragma unroll
    for (int c = 0; c < 3; ++c) U[c] = a.u[(long long)c * a.usc + n * a.usn];
    const double lam = (a.lam_e ? a.lam_e[e] : a.lam) * w, mu = (a.mu_e ? a.mu_e[e] : a.mu) * w;
    const bool ok = force_le_lanes(L, U, lam, mu, F, scale);
    if (first >= a.ne) return;
    if (ok) {
#pragma unroll
        for (int c = 0; c < 3; ++c) put<MODE>(a, e, n0, sy, sz, L.a, c, f64_scaled(F[c], scale));
    } else if (L.a == 0) {
        double Ff[3][8];
        far_force_le(a.u + (long long)n0 * a.usn, a.usn, a.usc, sy, sz, lam, mu, Ff);
        for (int c8 = 0; c8 < 8; ++c8)
            for (int c = 0; c < 3; ++c) put<MODE>(a, e, n0, sy, sz, c8, c, Ff[c][c8]);
    }
}

// FomB groups: u the displacement or the CG direction, read as it is (its rounding through 1/h was the largest
// error of the FP64 form); element buffer [24][NE], trace blocks at the end of the grid
__global__ void __launch_bounds__(128) k_fom_force_le(const __grid_constant__ FomB g, const int* __restrict__ active,
                                                      const __grid_constant__ TraceFuse tr, const double* u) {
    if ((int)blockIdx.x >= g.n_eblk) {
        trace::fused_trace_block(tr, active, g, (int)blockIdx.x - g.n_eblk);
        return;
    }
    const int2 b = g.eblk[blockIdx.x];
    if (active && !active[b.x]) return;
    const InstFom& I = g.inst[b.x];
    const int e = b.y + threadIdx.x;
    if (e >= I.ne) return;
    const int nx = I.nx, ny = I.ny, i = e % nx, t = e / nx, j = t % ny, k = t / ny;
    const int sy = nx + 1, sz = (nx + 1) * (ny + 1);
    const double* x = u + I.node_off + (i + sy * j + sz * k);
    double U[3][8], F[3][8];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8)
            U[c][c8] = x[(long long)c * g.NN + (c8 & 1) + ((c8 >> 1) & 1) * sy + (c8 >> 2) * sz];
    double lam = I.t1, mu = I.t2;
    if (I.lam_e || I.mu_e) {
        const double w = 2.0 * I.wqi;
        lam = (I.lam_e ? I.lam_e[e] : I.lam) * w;
        mu = (I.mu_e ? I.mu_e[e] : I.mu) * w;
    }
    double* fe = static_cast<double*>(g.fe) + I.elem_off + e;
    if (!element_force_le(U, lam, mu, F)) {
        double Ff[3][8];
        far_force_le(x, 1, g.NN, sy, sz, lam, mu, Ff);
        for (int c8 = 0; c8 < 8; ++c8)
            for (int c = 0; c < 3; ++c) fe[(long long)(c8 * 3 + c) * g.NE] = Ff[c][c8];
        return;
    }
#pragma unroll
    for (int c8 = 0; c8 < 8; ++c8)
#pragma unroll
        for (int c = 0; c < 3; ++c) fe[(long long)(c8 * 3 + c) * g.NE] = F[c][c8];
}

// ... and on 8 lanes: block of g.eblock threads, an element block on 8 of them
__global__ void __launch_bounds__(128) k_fom_force_le_lanes(const __grid_constant__ FomB g, const int* __restrict__ active,
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
    double lam = I.t1, mu = I.t2;
    if (I.lam_e || I.mu_e) {
        const double w = 2.0 * I.wqi;
        lam = (I.lam_e ? I.lam_e[e] : I.lam) * w;
        mu = (I.mu_e ? I.mu_e[e] : I.mu) * w;
    }
    const bool ok = force_le_lanes(L, U, lam, mu, F, scale);
    if (first >= I.ne) return;
    double* fe = static_cast<double*>(g.fe) + I.elem_off + e;
    if (ok) {
#pragma unroll
        for (int c = 0; c < 3; ++c) fe[(long long)(L.a * 3 + c) * g.NE] = f64_scaled(F[c], scale);
    } else if (L.a == 0) {
        double Ff[3][8];
        far_force_le(x, 1, g.NN, sy, sz, lam, mu, Ff);
        for (int c8 = 0; c8 < 8; ++c8)
            for (int c = 0; c < 3; ++c) fe[(long long)(c8 * 3 + c) * g.NE] = Ff[c][c8];
    }
}

// 8 lanes per element up to kLaneElements elements, where the length of one thread's work is the time; they
// issue about twice the instructions.  Element level, 8 lanes against one thread: 432 elements 9.3 and 11.4 us,
// 16000 both 14.5, 54000 26.7 and 18.7, 262144 93.7 and 45.5; the 6x6x12 FOM-FOM step 1.58 and 2.03 ms.
constexpr long long kLaneElements = 16384;

}  // namespace

cudaError_t launch_elem_force_le(int scatter, const ElemArgs& a, cudaStream_t s, int lanes) {
    const int grid = grid_for(a.ne, kElemBlock);
    const double w = 2.0 * a.wq * a.invh;   // h / 16
    if (lanes < 0 ? a.ne <= kLaneElements : lanes) {
        const int blocks = grid_for(a.ne, 16);
        if (scatter == kAtomic) k_elem_force_le_lanes<kAtomic><<<blocks, 128, 0, s>>>(a, w);
        else k_elem_force_le_lanes<kGather><<<blocks, 128, 0, s>>>(a, w);
        return cudaGetLastError();
    }
    if (scatter == kAtomic) k_elem_force_le<kAtomic><<<grid, kElemBlock, 0, s>>>(a, w);
    else k_elem_force_le<kGather><<<grid, kElemBlock, 0, s>>>(a, w);
    return cudaGetLastError();
}

cudaError_t launch_force_le_b(const FomB& g, const int* active, const TraceFuse& tr, const double* u, cudaStream_t s) {
    if (g.eblock > 128 || !u) return cudaErrorInvalidValue;
    long long items = 0;
    for (int k = 0; k < tr.n; ++k) items += 3LL * tr.c[k].R;
    const int extra = (int)((items + g.eblock - 1) / g.eblock);
    if (g.NE <= kLaneElements) k_fom_force_le_lanes<<<8 * g.n_eblk + extra, g.eblock, 0, s>>>(g, active, tr, u);
    else k_fom_force_le<<<g.n_eblk + extra, g.eblock, 0, s>>>(g, active, tr, u);
    return cudaGetLastError();
}

}  // namespace osam
