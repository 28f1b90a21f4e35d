// Neo-Hookean internal force and explicit node update in 64-bit fixed point (fixed_math.cuh).
//
// The force of the FP64 explicit path when the launch is left to the library: one thread per element, the
// predicted displacement read as fixed-point u / h (written by the node kernel), the element forces left
// as 64-bit integers in the element buffer, so the node kernel's sums are exact and cost integer
// additions.  An element outside the range of the formats is evaluated in FP64 (far_element), and its entries hold
// the FP64 values (hold_f64); so do those of an element too soft for the buffer's unit (kMaxDown).
//
// ncu counts 1969 instructions of k_force_fx_b on the integer multiply-add pipe (4 cycles each) and 2994 on the integer
// ALU per warp, against 717 FP64 instructions (67 to 80 cycles each) of the tiled FP64 kernel.  On large launches the
// pipe is the bound (0.82 of its issue rate at 5.6 M elements, 0.72 at 1.8 M); on one 40x40x80 mesh (3.3 waves of
// blocks) it issues 0.63 of that rate warm, and at 1.9 warps per scheduler the warps wait for their own results and for
// instructions (ncu, cold: per issued instruction 1.5 warps in fixed latencies, 1.0 without an instruction, 0.6 in
// dispatch, 0.6 for memory, 0.3 for the pipe): the unrolled code is 80 KB, and moving it changes the time by 1 to 2%.
// Measured on 40x40x80: 40 us per launch, 186 us for the FP64 kernel; on 96x96x192 478 us, 2360 us.
// The Gauss points are fully unrolled (43.4 us; with the two planes as a loop 45.3), 255 registers and
// two warps per scheduler: capping at 168 or 128 registers (480 to 680 bytes of spills read back per thread)
// measured 45.3 and 47.5 us on 40x40x80, 510 and 523 us on 96x96x192; with the Walsh coefficients and one
// plane's sums in shared memory (168 registers, three blocks per SM, no spills) the 96x96x192 chain step took 58.4
// instead of 55.5 ms: more warps did not help.
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

// A contribution held in FP64 in its entry of the buffer
__device__ __forceinline__ void put_f64(const FomB& g, const InstFom& I, int e, int c8, int c, double v) {
    static_cast<i64*>(g.fe)[(long long)(c8 * 3 + c) * g.NE + I.elem_off + e] = hold_f64(v);
}

// Element e in FP64.  Not inlined, so that its registers and code stay out of the fixed-point path.
__device__ __noinline__ void far_element(const FomB& g, const InstFom& I, const double* u, int e, int n0) {
    using namespace hex8;
    const int sy = I.nx + 1, sz = (I.nx + 1) * (I.ny + 1);
    double m1, m2, m3;
    if (I.lam_e || I.mu_e)
        material_factors<OSAM_NEO_HOOKEAN, double>(I.lam_e ? I.lam_e[e] : I.lam, I.mu_e ? I.mu_e[e] : I.mu, I.wq, I.wq3,
                                                   m1, m2, m3);
    else { m1 = I.m1; m2 = I.m2; m3 = I.m3; }
    double Dx[3][2][2], Dy[3][2][2], Dz[3][2][2], F[3][8];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        double U[8];
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8)
            U[c8] = u[(long long)c * g.NN + I.node_off + n0 + (c8 & 1) + ((c8 >> 1) & 1) * sy + ((c8 >> 2) & 1) * sz];
        edge_differences<double>(U, I.invh, Dx[c], Dy[c], Dz[c]);
    }
    element_force<OSAM_NEO_HOOKEAN, double>(Dx, Dy, Dz, m1, m2, m3, F);
#pragma unroll
    for (int c8 = 0; c8 < 8; ++c8)
#pragma unroll
        for (int c = 0; c < 3; ++c) put_f64(g, I, e, c8, c, F[c][c8]);
}

// In an instance with displacements beyond the format (g.wide) the nodal values are modulo 32 edges, and u itself tells
// whether the element's differences are in range; its own function, away from the registers of the force
__device__ __noinline__ bool torn_element(const FomB& g, const InstFom& I, const double* u, int n0) {
    const int sy = I.nx + 1, sz = (I.nx + 1) * (I.ny + 1);
    bool bad = false;
    for (int c = 0; c < 3; ++c) {
        const double* x = u + (long long)c * g.NN + I.node_off + n0;
        double U[8];
        i64 V[8];
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8) U[c8] = x[(c8 & 1) + ((c8 >> 1) & 1) * sy + (c8 >> 2) * sz];
        bad |= refit(U, I.ihm, I.ihe, V);
    }
    return bad;
}

__global__ void __launch_bounds__(128) k_force_fx_b(const __grid_constant__ FomB g, const int* __restrict__ active,
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
    const int nx = I.nx, ny = I.ny;
    const int i = e % nx;
    const int t = e / nx;
    const int j = t % ny;
    const int k = t / ny;
    const int sy = nx + 1, sz = (nx + 1) * (ny + 1);
    const int n0 = i + sy * j + sz * k;
    const bool wide = g.wide[b.x] != 0;
    bool bad = false;
    if (wide) bad = torn_element(g, I, u, n0);
    WalshIn w[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const i64* x = g.ux + (long long)c * g.NN + I.node_off + n0;
        i64 V[8];
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8) V[c8] = x[(c8 & 1) + ((c8 >> 1) & 1) * sy + ((c8 >> 2) & 1) * sz];
        bad |= spread_bad(V) && !wide;
        w[c] = walsh_in(V, c);
    }
    i64 kap2 = I.fk2, mu = I.fmu;
    int down = 0;   // binades of the element's unit below the mesh's
    if (I.lam_e || I.mu_e) {
        Material M;
        bad |= !material(I.lam_e ? I.lam_e[e] : I.lam, I.mu_e ? I.mu_e[e] : I.mu, I.wq, M);
        kap2 = whole(M.kap2);
        mu = whole(M.mu);
        down = kFracOut - I.fscale - M.k;
        bad |= down < 0 || M.k < -900;
    }
    i64 F[3][8];
    bad |= !element_force_nh(w, kap2, mu, mul_third(mu), F);
    if (bad) {
        far_element(g, I, u, e, n0);
        return;
    }
    if (down > kMaxDown) {
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8)
#pragma unroll
            for (int c = 0; c < 3; ++c) put_f64(g, I, e, c8, c, f64_scaled(F[c][c8], I.fscale + down));
        return;
    }
    if (down) {
        const i64 half = (i64)1 << (down - 1);
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8)
#pragma unroll
            for (int c = 0; c < 3; ++c) F[c][c8] = (F[c][c8] + half) >> down;
    }
    i64* fe = static_cast<i64*>(g.fe) + I.elem_off + e;
#pragma unroll
    for (int c8 = 0; c8 < 8; ++c8)
#pragma unroll
        for (int c = 0; c < 3; ++c) fe[(long long)(c8 * 3 + c) * g.NE] = F[c][c8];
}

// the same with an element on 8 lanes (lanes.cuh); 8 thread blocks of g.eblock threads per element block
__global__ void __launch_bounds__(128, 5) k_force_fx_lanes_b(const __grid_constant__ FomB g, const int* __restrict__ active,
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
    const int sy = nx + 1, sz = (nx + 1) * (ny + 1), n0 = i + sy * j + sz * k;
    const Lane L = make_lane();
    const long long gn = I.node_off + n0 + (L.a & 1) + ((L.a >> 1) & 1) * sy + (L.a >> 2) * sz;
    i64 U[3], F[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) U[c] = g.ux[c * g.NN + gn];
    D kap2 = split(I.fk2), mu = split(I.fmu), mu3 = split(mul_third(I.fmu));
    bool bad = false;
    if (g.wide[b.x]) {   // values modulo 32 edges: the edges from u itself
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            i64 v;
            int x;
            bad |= !wrapped_u(u[c * g.NN + gn], I.ihm, I.ihe, v, x);
            bad |= coarse_edge_bad(x);
        }
    }
    int down = 0;
    if (I.lam_e || I.mu_e) {
        Material M;
        bad |= !material(I.lam_e ? I.lam_e[e] : I.lam, I.mu_e ? I.mu_e[e] : I.mu, I.wq, M);
        kap2 = M.kap2;
        mu = M.mu;
        mu3 = M.mu3;
        down = kFracOut - I.fscale - M.k;
        bad |= down < 0 || M.k < -900;
    }
    const bool ok = force_lanes(L, U, kap2, mu, mu3, bad, F);
    if (first >= I.ne) return;
    if (ok && down > kMaxDown) {
#pragma unroll
        for (int c = 0; c < 3; ++c) put_f64(g, I, e, L.a, c, f64_scaled(F[c], I.fscale + down + 3));   // 57 fraction bits
    } else if (ok) {
        i64* fe = static_cast<i64*>(g.fe) + I.elem_off + e;
        const int n = 3 + down;   // 57 to 54 fraction bits
#pragma unroll
        for (int c = 0; c < 3; ++c) fe[(long long)(L.a * 3 + c) * g.NE] = (F[c] + ((i64)1 << (n - 1))) >> n;
    } else if (L.a == 0) {
        far_element(g, I, u, e, n0);
    }
}

// 8 lanes per element up to kLaneElements elements, where the length of one thread's work is the time; they issue
// two and a half times the instructions.  Time of a substep, 8 lanes against one thread per element: 432 elements
// 9.6 and 15.8 us, 8192 13.2 and 16.7, 16000 16.2 and 16.9, 27648 21.6 and 19.2, 128000 67 and 52.
constexpr long long kLaneElements = 16384;

// Corrector of substep j and predictor of substep j + 1 (the arithmetic of k_node_b) on the fixed-point
// element buffer: the 24 contributions of a node are summed exactly as integers and converted once per
// component; the predictor is written in FP64 and as fixed-point u / h.
template <int NC>
__global__ void __launch_bounds__(kNodeBlock) k_node_fx_b(const __grid_constant__ FomB g,
                                                          const int* __restrict__ active, int slot1, int slot2,
                                                          int predict_only, const double* ucur, double* unext,
                                                          double dt) {
    const int2 b = g.nblk[blockIdx.x];
    if (active && !active[b.x]) return;
    const InstFom& I = g.inst[b.x];
    const int n = b.y + threadIdx.x;
    if (n >= I.nn) return;
    const int nx = I.nx, ny = I.ny, nz = I.nz;
    const int i = n % (nx + 1);
    const int t = n / (nx + 1);
    const int j = t % (ny + 1);
    const int k = t / (ny + 1);
    const long long gn = I.node_off + n;
    const int c0 = NC == 3 ? 0 : (int)blockIdx.y;   // the thread's components c0 .. c0 + NC - 1
    const uint8_t cm = g.clamp[gn];
    const int row = g.srow[gn];
    const double hdt = 0.5 * dt, hdt2 = 0.5 * dt * dt;
    const double minv = g.minv[gn];
    const double* h1 = slot1 >= 0 ? g.hist + I.hist_off + (long long)slot1 * 9 * I.ns : nullptr;
    const double* h2 = slot2 >= 0 ? g.hist + I.hist_off + (long long)slot2 * 9 * I.ns : nullptr;
    double uc[NC], vc[NC], ac[NC], f[NC] = {};
#pragma unroll
    for (int q = 0; q < NC; ++q) {
        const long long d = (long long)(c0 + q) * g.NN + gn;
        uc[q] = ucur[d];
        vc[q] = g.v[d];
        ac[q] = g.a[d];
    }
    if (!predict_only && row < 0 && cm != 7) {
        const i64* fe = static_cast<const i64*>(g.fe) + I.elem_off;
        i64 s[NC] = {};
        unsigned int far = 0;
        if constexpr (NC == 1) {
            // All eight loads before the first test: on a small mesh their latency, one after the other, was the kernel's
            // time (6x6x12 substep 8.8 us, 6.8 us so; 20x20x40 15.2 and 13.5).  With three components the values held take
            // 96 registers instead of 56, and the kernels beside it on the side stream wait (40x40x80 hybrid 5.16 instead
            // of 5.03 ms).
            i64 x[8];
#pragma unroll
            for (int corner = 0; corner < 8; ++corner) {
                const int ie = i - (corner & 1), je = j - ((corner >> 1) & 1), ke = k - (corner >> 2);
                const bool in = ke >= 0 && ke < nz && je >= 0 && je < ny && ie >= 0 && ie < nx;
                const long long e = ie + (long long)nx * (je + ny * ke);
                x[corner] = in ? __ldg(fe + (long long)(corner * 3 + c0) * g.NE + e) : 0;
            }
#pragma unroll
            for (int corner = 0; corner < 8; ++corner) {
                const bool held = held_f64(x[corner]);
                far |= (held ? 1u : 0u) << corner;
                s[0] += held ? 0 : x[corner];
            }
        } else {
#pragma unroll
            for (int az = 0; az < 2; ++az) {
                const int ke = k - az;
#pragma unroll
                for (int ay = 0; ay < 2; ++ay) {
                    const int je = j - ay;
#pragma unroll
                    for (int ax = 0; ax < 2; ++ax) {
                        const int ie = i - ax;
                        const int corner = ax + 2 * ay + 4 * az;
                        if (ke < 0 || ke >= nz || je < 0 || je >= ny || ie < 0 || ie >= nx) continue;
                        const long long e = ie + (long long)nx * (je + ny * ke);
                        i64 x[NC];
#pragma unroll
                        for (int q = 0; q < NC; ++q) x[q] = __ldg(fe + (long long)(corner * 3 + c0 + q) * g.NE + e);
                        if (held_f64(x[0])) { far |= 1u << corner; continue; }
#pragma unroll
                        for (int q = 0; q < NC; ++q) s[q] += x[q];
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < NC; ++q) f[q] = f64_scaled(s[q], I.fscale);
        while (far) {   // elements held in FP64
            const int corner = __ffs((int)far) - 1;
            far &= far - 1;
            const long long e = (i - (corner & 1)) +
                                (long long)nx * ((j - ((corner >> 1) & 1)) + ny * (k - (corner >> 2)));
#pragma unroll
            for (int q = 0; q < NC; ++q) f[q] += f64_held(fe[(long long)(corner * 3 + c0 + q) * g.NE + e]);
        }
    }
#pragma unroll
    for (int q = 0; q < NC; ++q) {
        const int c = c0 + q;
        const long long d = (long long)c * g.NN + gn;
        double un;
        if (cm & (1 << c)) {
            g.v[d] = 0.0;
            g.a[d] = 0.0;
            un = 0.0;
        } else if (row >= 0) {
            if (!predict_only) {
                g.v[d] = h1[(long long)(3 + c) * I.ns + row];
                g.a[d] = h1[(long long)(6 + c) * I.ns + row];
            }
            un = h2 ? h2[(long long)c * I.ns + row] : 0.0;
        } else {
            double vn = vc[q], an = ac[q];
            if (!predict_only) {
                const double anew = -f[q] * minv;
                vn = fma(hdt, an + anew, vn);
                an = anew;
                g.v[d] = vn;
                g.a[d] = an;
            }
            un = fma(hdt2, an, fma(dt, vn, uc[q]));
        }
        if (h2) {
            unext[d] = un;
            i64 x = fixed_u(un, I.ihm, I.ihe);
            if (x == kBadU) {   // beyond the format: modulo 32 edges, and the force looks at u from now on
                int coarse;
                wrapped_u(un, I.ihm, I.ihe, x, coarse);
                g.wide[b.x] = 1;
            }
            g.ux[d] = x;
        }
    }
}

}  // namespace

cudaError_t launch_force_fx_b(const FomB& g, const int* active, const TraceFuse& tr, const double* upred,
                              cudaStream_t s) {
    if (!upred || g.eblock > 128) return cudaErrorInvalidValue;
    long long items = 0;
    for (int k = 0; k < tr.n; ++k) items += 3LL * tr.c[k].R;
    const int extra = (int)((items + g.eblock - 1) / g.eblock);
    if (g.NE <= kLaneElements) k_force_fx_lanes_b<<<8 * g.n_eblk + extra, g.eblock, 0, s>>>(g, active, tr, upred);
    else k_force_fx_b<<<g.n_eblk + extra, g.eblock, 0, s>>>(g, active, tr, upred);
    return cudaGetLastError();
}

cudaError_t launch_node_fx_b(const FomB& g, const int* active, int slot1, int slot2, int predict_only,
                             const double* ucur, double* unext, double dt, cudaStream_t s) {
    if (node_split(g))
        k_node_fx_b<1><<<dim3(g.n_nblk, 3), kNodeBlock, 0, s>>>(g, active, slot1, slot2, predict_only, ucur, unext, dt);
    else k_node_fx_b<3><<<g.n_nblk, kNodeBlock, 0, s>>>(g, active, slot1, slot2, predict_only, ucur, unext, dt);
    return cudaGetLastError();
}

}  // namespace osam
