// FP64 products of the offline fit on the bf16 tensor cores (Ozaki's error-free splitting: K. Ozaki, T. Ogita,
// S. Oishi, S. Rump, Numerical Algorithms 59, 2012).
//
// Every operand row is written, over chunks of 1024 along k, as a 55-bit integer times a power of two (the
// largest exponent of the row's chunk), and the integer as 7 balanced base-256 digits, exact in bf16.  Digit
// products are at most 2^14, so a sum over 128 of k of the s + 1 <= 7 products of one weight s stays below 2^24 and
// is exact in the tensor core's FP32 accumulator.  The sums are added as 64-bit integers over the chunk and
// enter the FP64 result once per chunk.  The products of weight 7 are 2^-8 of those of weight 6 and enter the same
// accumulator with the second digit scaled by 2^-8, where only bits below 2^-56 of the operands' product are lost.
// Products of weight 8 and above are dropped: at most 2^-57.6 of the two chunk maxima's product each (2^-62.4 rms).
//
// What limits the accuracy is the rounding of an element s binades below its row's chunk maximum to 54 - s bits.  An
// element's product is therefore off by 2^-54 / sqrt(12) (rms) times each operand's maximum, where FP64 is off
// relative to the product itself.  With a'_k, b'_k the operands over their maxima's power of two the error is
//   E = 2^-54 / sqrt(12) sqrt(sum a'^2 + sum b'^2 + k 2^-13),
// and that of the FP64 kernel about 0.48 2^-53 P, P = sum |a' b'| (measured on random operands at any k).  Rows in which
// few large elements hide the small ones that matter would lose; so every 64 x 64 tile is certified first
// (k_split_check: P on the tensor cores from 8-bit magnitudes, one product against 34): a tile with
// E > 0.25 2^-53 P anywhere, summed over the chunks, with operands that are not finite or subnormal, or with
// exponents out of the normal range, is left to the FP64 kernel.  Random operands pass from k = 64 on; their error is
// then 1.3e-17 |A||B| at k = 128 and 5e-18 at 1024 (integer simulation of the scheme), FP64's 4.6e-17 and 6e-17.
// E takes the roundings as independent; elements that all round the same way (a constant row beside one element some
// binades larger) can add up to more, as they do in FP64's own sums of a constant.
//
// Why: the FP64 tensor pipe of GB300 gives about 1 TFLOP/s; 34 bf16 products of the same size cost 34 / 1000
// of that at legacy mma.sync rates a few hundred times higher.  One 64 x 64 tile per block of 8 warps (32 x 16
// each): the accumulators of the 7 weights take 112 registers, the digits of a 32-deep stage 70 KB of shared
// memory, two stages resident; half the warps slice the next stage while the others multiply.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "fixed_math.cuh"
#include "osam_internal.h"

namespace osam {

namespace {

constexpr int TS = kGemmTile;        // output tile
constexpr int KS = 32;               // k per stage
constexpr int KC = kSplitChunk;      // k per exponent
constexpr int KF = 128;              // k between flushes of the FP32 accumulators
constexpr int ND = 7;                // digits
constexpr int PITCH = KS + 8;        // bf16 per shared row: 80 bytes, 8 rows of an ldmatrix on distinct banks
constexpr int PLANE = TS * PITCH;    // bf16 per digit of one operand
constexpr int kThreads = 256;
constexpr size_t kStageBytes = 2ull * ND * PLANE * 2;             // both operands
constexpr size_t kSumBytes = 2ull * 16 * kThreads * 8;            // integer sums: two words per result
constexpr size_t kSmem = 2 * kStageBytes + kSumBytes;
static_assert(KC % KF == 0 && KF % KS == 0, "stages per flush and flushes per chunk");
static_assert(KF * ND * 16384 + KF * (ND - 1) * 64 <= (1 << 24), "exact FP32 sums");

// Operand view: element (row, k) at p[row * rs + k * ks]
struct Op {
    const double* p;
    long long rs, ks;
    int rows;
    const int* ex;                   // largest biased exponent of (row, chunk): ex[row * chunks + chunk]; 2047 also for a
                                     // chunk with a subnormal
    const float* sq;                 // sum of the squares of (row, chunk) over the maximum's power of two
};

// An operand's magnitude over the power of two of its chunk's maximum (biased exponent E), below 1: as FP32 and as bf16,
// both cut off
__device__ __forceinline__ float over_max(unsigned int h, int E) {
    const int s = E - (int)(h >> 20);
    return h < (1u << 20) || s > 120 ? 0.f : __uint_as_float(((unsigned int)(126 - s) << 23) | ((h & 0xfffffu) << 3));
}
__device__ __forceinline__ uint32_t over_max_pair(double x, double y, int E) {
    const float a = over_max((unsigned int)__double2hiint(x) & 0x7fffffffu, E);
    const float b = over_max((unsigned int)__double2hiint(y) & 0x7fffffffu, E);
    return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}

// high word of a magnitude; `odd` collects subnormals
__device__ __forceinline__ unsigned int magnitude(double x, bool& odd) {
    const unsigned int h = (unsigned int)__double2hiint(x) & 0x7fffffffu;
    odd |= h < (1u << 20) && (h | (unsigned int)__double2loint(x)) != 0;
    return h;
}

// Largest exponent and sum of squares of every (row, chunk): a block per chunk and 8 rows (a warp each, rows contiguous in k,
// the chunk's high words in registers) or 32 rows (lanes along the rows, the 8 warps share the chunk, read twice).
// The sums have a fixed order: the certificate must not change from run to run.
__global__ void __launch_bounds__(256) k_split_exponents(const double* __restrict__ p, long long rs, long long ks, int rows,
                                                         int kdim, int chunks, int* __restrict__ ex, float* __restrict__ sq) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int chunk = (int)(blockIdx.x % chunks);
    const long long group = blockIdx.x / chunks;
    const long long k0 = (long long)chunk * KC, k1 = min((long long)kdim, k0 + KC);
    unsigned int top = 0;
    float sum = 0.f;
    bool odd = false;
    if (ks == 1) {
        const long long row = group * 8 + warp;
        if (row >= rows) return;
        unsigned int h[KC / 32];
#pragma unroll
        for (int q = 0; q < KC / 32; ++q) {
            const long long k = k0 + lane + 32 * q;
            h[q] = k < k1 ? magnitude(__ldg(p + row * rs + k), odd) : 0u;
            top = max(top, h[q]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        odd = __any_sync(0xffffffffu, odd);
#pragma unroll
        for (int q = 0; q < KC / 32; ++q) {
            const float x = over_max(h[q], (int)(top >> 20));
            sum = fmaf(x, x, sum);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) {
            ex[row * chunks + chunk] = odd ? 2047 : (int)(top >> 20);
            sq[row * chunks + chunk] = sum;
        }
    } else {
        __shared__ unsigned int m[32];
        __shared__ float part[8][32];
        const long long row = group * 32 + lane;
        if (warp == 0) m[lane] = 0;
        __syncthreads();
        if (row < rows)
            for (long long k = k0 + warp; k < k1; k += 8) top = max(top, magnitude(__ldg(p + row * rs + k * ks), odd));
        atomicMax(m + lane, odd ? 0x7ff00000u : top);
        __syncthreads();
        top = m[lane];
        if (row < rows)
            for (long long k = k0 + warp; k < k1; k += 8) {
                const float x = over_max((unsigned int)__double2hiint(__ldg(p + row * rs + k * ks)) & 0x7fffffffu, (int)(top >> 20));
                sum = fmaf(x, x, sum);
            }
        part[warp][lane] = sum;
        __syncthreads();
        if (warp == 0 && row < rows) {
#pragma unroll
            for (int w = 1; w < 8; ++w) sum += part[w][lane];
            ex[row * chunks + chunk] = (int)(top >> 20);
            sq[row * chunks + chunk] = sum;
        }
    }
}

// x 2^(1022 + 54 - E) rounded to an integer below 2^54, plus 128 in every base-256 digit: its bytes are the
// balanced digits + 128
__device__ __forceinline__ unsigned long long biased_digits(double x, int E) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ff), s = E - e;
    unsigned long long v = 0;
    if (e != 0 && s < 56) {
        const unsigned long long m = ((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 1;
        v = (m + ((1ULL << s) >> 1)) >> s;
        if ((long long)b < 0) v = 0ULL - v;
    }
    return v + 0x0080808080808080ULL;
}

// digit i (0 the most significant) of two neighbouring k as packed bf16
template <int I>
__device__ __forceinline__ uint32_t digit_pair(unsigned long long x, unsigned long long y) {
    constexpr int byte = ND - 1 - I;                              // 0..6
    const uint32_t a = (uint32_t)(byte < 4 ? x : x >> 32), b = (uint32_t)(byte < 4 ? y : y >> 32);
    constexpr uint32_t sel = (uint32_t)(byte & 3);
    const uint32_t w = __byte_perm(a, b, sel | ((sel + 4) << 8)); // x's byte in bits 0-7, y's in bits 16-23
    const uint32_t lo = (w & 0x007f007fu) | 0x43004300u;          // 128 + the low 7 bits
    const uint32_t sub = (~w & 0x00800080u) | 0x43004300u;        // 128, or 256 below zero
    uint32_t r;
    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(lo), "r"(sub));
    return r;
}

__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// bf16 digits times 2^-8, exact
__device__ __forceinline__ uint32_t next_weight(uint32_t x) {
    uint32_t r;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(0x3b803b80u));
    return r;
}

struct Pairs {
    double v[4][2];                  // 4 pairs of neighbouring k per thread and operand
};
// pair q of a thread: row and first k within the stage (lanes along k, or along the rows, whichever is contiguous)
__device__ __forceinline__ void pair_at(bool along_k, int q, int& row, int& k) {
    const int t = (int)threadIdx.x + q * kThreads;   // 0..1023
    if (along_k) { k = 2 * (t & 15); row = t >> 4; }
    else { row = t & 63; k = 2 * (t >> 6); }
}
__device__ __forceinline__ void load(const Op& o, int row0, int k0, int kend, Pairs& P) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int r, k;
        pair_at(o.ks == 1, q, r, k);
        const double* p = o.p + (long long)(row0 + r) * o.rs + (long long)(k0 + k) * o.ks;
        const bool in = row0 + r < o.rows;
        P.v[q][0] = in && k0 + k < kend ? __ldg(p) : 0.0;
        P.v[q][1] = in && k0 + k + 1 < kend ? __ldg(p + o.ks) : 0.0;
    }
}
__device__ __forceinline__ void slice(const Pairs& P, const int (&ex)[4], bool along_k, uint32_t* plane) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int r, k;
        pair_at(along_k, q, r, k);
        const unsigned long long x = biased_digits(P.v[q][0], ex[q]), y = biased_digits(P.v[q][1], ex[q]);
        uint32_t* d = plane + (r * PITCH + k) / 2;
        d[0 * PLANE / 2] = digit_pair<0>(x, y);
        d[1 * PLANE / 2] = digit_pair<1>(x, y);
        d[2 * PLANE / 2] = digit_pair<2>(x, y);
        d[3 * PLANE / 2] = digit_pair<3>(x, y);
        d[4 * PLANE / 2] = digit_pair<4>(x, y);
        d[5 * PLANE / 2] = digit_pair<5>(x, y);
        d[6 * PLANE / 2] = digit_pair<6>(x, y);
    }
}
__device__ __forceinline__ void exponents(const Op& o, int row0, int chunk, int chunks, int (&ex)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int r, k;
        pair_at(o.ks == 1, q, r, k);
        ex[q] = row0 + r < o.rows ? o.ex[(long long)(row0 + r) * chunks + chunk] : 0;
    }
}

// Output tile of a block; sym: B is A, only tiles on and above the diagonal, numbered by rows of the upper triangle.
// Returns its number in the whole grid of tiles.
__device__ __forceinline__ int tile_of(int sym, int ntn, int& ti, int& tj) {
    if (sym) {
        int t = (int)blockIdx.x;
        for (ti = 0; t >= ntn - ti; ++ti) t -= ntn - ti;
        tj = ti + t;
    } else {
        ti = (int)blockIdx.x / ntn;
        tj = (int)blockIdx.x % ntn;
    }
    return ti * ntn + tj;
}

// The certificate of k range blockIdx.y: 0.5 P - sqrt(sum a'^2 + sum b'^2 + k 2^-13) / sqrt(12) (units 2^-54), summed over
// the chunks with their powers of two, into D[split][m][n]; with one k range (D null) straight into the tile's flag.
// Bound by the loads of the operands, 64 + 64 rows per tile from L2.
__global__ void __launch_bounds__(kThreads, 2) k_split_check(const __grid_constant__ Op A, const __grid_constant__ Op B,
                                                             int kdim, int kchunk, int chunks, int sym,
                                                             double* __restrict__ D, int* __restrict__ flag) {
    __shared__ __align__(16) uint32_t planes[2][2][PLANE / 2];       // [stage][operand]
    const int ntn = (B.rows + TS - 1) / TS;
    int ti, tj;
    const int tile = tile_of(sym, ntn, ti, tj);
    const int i0 = ti * TS, j0 = tj * TS;
    const int kbeg = (int)blockIdx.y * kchunk, kend = (int)min((long long)kdim, (long long)kbeg + kchunk);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wr = (warp >> 2) * 32, wc = (warp & 3) * 16;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(&planes[0][0][0]);
    const uint32_t aoff = ((wr + (lane & 15)) * PITCH + (lane >> 4) * 8) * 2;
    const uint32_t boff = ((wc + ((lane >> 4) << 3) + (lane & 7)) * PITCH + ((lane >> 3) & 1) * 8) * 2 + PLANE * 2;
    float acc[2][2][4] = {};
    double d[16] = {};
    const int stages = (kend - kbeg + KS - 1) / KS;
    Pairs pa, pb;
    int ea[4], eb[4];
    const auto cut = [&](const Op& o, const Pairs& P, const int (&ex)[4], uint32_t* plane) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int r, k;
            pair_at(o.ks == 1, q, r, k);
            plane[(r * PITCH + k) / 2] = over_max_pair(P.v[q][0], P.v[q][1], ex[q]);
        }
    };
    load(A, i0, kbeg, kend, pa);
    load(B, j0, kbeg, kend, pb);
    for (int st = 0; st < stages; ++st) {
        const int k = kbeg + st * KS;
        if (st % (KC / KS) == 0) {
            exponents(A, i0, k / KC, chunks, ea);
            exponents(B, j0, k / KC, chunks, eb);
        }
        cut(A, pa, ea, planes[st & 1][0]);
        cut(B, pb, eb, planes[st & 1][1]);
        if (st + 1 < stages) {
            load(A, i0, k + KS, kend, pa);
            load(B, j0, k + KS, kend, pb);
        }
        __syncthreads();       // two stages: the next write to this one comes after the next barrier
        const uint32_t buf = base + (uint32_t)((st & 1) * 2 * PLANE * 2);
#pragma unroll
        for (int kk = 0; kk < KS; kk += 16) {
            uint32_t a[2][4], b[4];
            ldmatrix4(b, buf + boff + kk * 2);
            ldmatrix4(a[0], buf + aoff + kk * 2);
            ldmatrix4(a[1], buf + aoff + 16 * PITCH * 2 + kk * 2);
#pragma unroll
            for (int x = 0; x < 2; ++x)
#pragma unroll
                for (int y = 0; y < 2; ++y) mma_bf16(acc[x][y], a[x], b[2 * y], b[2 * y + 1]);
        }
        if ((st + 1) % (KC / KS) == 0 || st + 1 == stages) {
            const int chunk = k / KC;
            const float count = (float)(min((long long)kend, ((long long)chunk + 1) * KC) - (long long)chunk * KC);
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                float& P = acc[r >> 3][(r >> 2) & 1][r & 3];
                const int gi = i0 + wr + (r >> 3) * 16 + ((r >> 1) & 1) * 8 + (lane >> 2);
                const int gj = j0 + wc + ((r >> 2) & 1) * 8 + 2 * (lane & 3) + (r & 1);
                if (gi < A.rows && gj < B.rows) {
                    const long long ia = (long long)gi * chunks + chunk, ib = (long long)gj * chunks + chunk;
                    const int ei = A.ex[ia], ej = B.ex[ib], e = ei + ej - 2044;
                    if (ei == 2047 || ej == 2047) {
                        d[r] = __longlong_as_double((long long)0xfff0000000000000ULL);
                    } else if (ei && ej) {
                        const float v = fmaf(0.5f, P, -0.28867513f * sqrtf(A.sq[ia] + B.sq[ib] + count * 0x1p-13f));
                        d[r] += e < -900 || e > 900 ? __longlong_as_double((long long)0xfff0000000000000ULL)
                                                    : (double)v * __longlong_as_double((long long)(1023 + e) << 52);
                    }
                }
                P = 0.f;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int gi = i0 + wr + (r >> 3) * 16 + ((r >> 1) & 1) * 8 + (lane >> 2);
        const int gj = j0 + wc + ((r >> 2) & 1) * 8 + 2 * (lane & 3) + (r & 1);
        if (gi >= A.rows || gj >= B.rows) continue;
        if (D) D[((long long)blockIdx.y * A.rows + gi) * B.rows + gj] = d[r];
        else if (!(d[r] >= 0.0)) flag[tile] = 1;
    }
}

// flags of the tiles whose certificate fails, from the k ranges' parts in ascending order
__global__ void k_split_flags(int m, int n, int nsplit, int sym, const double* __restrict__ D, int* __restrict__ flag) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long mn = (long long)m * n;
    if (idx >= mn) return;
    const int ti = (int)(idx / n) / TS, tj = (int)(idx % n) / TS;
    if (sym && ti > tj) return;
    double s = 0.0;
    for (int z = 0; z < nsplit; ++z) s += D[z * mn + idx];
    if (!(s >= 0.0)) flag[ti * ((n + TS - 1) / TS) + tj] = 1;
}

// partial result of k range blockIdx.y: ws[split][m][ldw]; nothing for the flagged tiles
__global__ void __launch_bounds__(kThreads, 1) k_split_gemm(const __grid_constant__ Op A, const __grid_constant__ Op B,
                                                            int kdim, int kchunk, int chunks, int sym, double* __restrict__ ws,
                                                            long long ldw, const int* __restrict__ flag) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int ntn = (B.rows + TS - 1) / TS;
    int ti, tj;
    if (flag[tile_of(sym, ntn, ti, tj)]) return;
    const int i0 = ti * TS, j0 = tj * TS;
    const int kbeg = (int)blockIdx.y * kchunk, kend = (int)min((long long)kdim, (long long)kbeg + kchunk);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wr = (warp >> 2) * 32, wc = (warp & 3) * 16;
    long long* sums = reinterpret_cast<long long*>(smem + 2 * kStageBytes);   // [word][result 16][thread]
    const bool ka = A.ks == 1, kb = B.ks == 1;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
    // ldmatrix addresses: A rows lane % 16, k half lane / 16; B rows (lane / 16) * 8 + lane % 8, k half (lane / 8) % 2
    const uint32_t aoff = ((wr + (lane & 15)) * PITCH + (lane >> 4) * 8) * 2;
    const uint32_t boff = ((wc + ((lane >> 4) << 3) + (lane & 7)) * PITCH + ((lane >> 3) & 1) * 8) * 2 + ND * PLANE * 2;
    float acc[ND][2][2][4];
#pragma unroll
    for (int s = 0; s < ND; ++s)
#pragma unroll
        for (int x = 0; x < 16; ++x) acc[s][x >> 3][(x >> 2) & 1][x & 3] = 0.f;
    const int stages = (kend - kbeg + KS - 1) / KS;
    Pairs pa, pb;
    int ea[4], eb[4];
    auto slice_stage = [&](int st) {             // the registers' stage st into its buffer
        const int k = kbeg + st * KS;
        if (st % (KC / KS) == 0) {
            exponents(A, i0, k / KC, chunks, ea);
            exponents(B, j0, k / KC, chunks, eb);
        }
        uint32_t* buf = reinterpret_cast<uint32_t*>(smem + (st & 1) * kStageBytes);
        slice(pa, ea, ka, buf);
        slice(pb, eb, kb, buf + ND * PLANE / 2);
        if (st + 1 < stages) {
            load(A, i0, k + KS, kend, pa);
            load(B, j0, k + KS, kend, pb);
        }
    };
    auto multiply = [&](int st) {
        const uint32_t buf = base + (uint32_t)((st & 1) * kStageBytes);
#pragma unroll 1
        for (int kk = 0; kk < KS; kk += 16) {
            uint32_t b[ND][4];
#pragma unroll
            for (int j = 0; j < ND; ++j) ldmatrix4(b[j], buf + boff + j * PLANE * 2 + kk * 2);
#pragma unroll
            for (int i = 0; i < ND; ++i) {
                uint32_t a[2][4];
                ldmatrix4(a[0], buf + aoff + i * PLANE * 2 + kk * 2);
                ldmatrix4(a[1], buf + aoff + i * PLANE * 2 + 16 * PITCH * 2 + kk * 2);
#pragma unroll
                for (int j = 0; j < ND - i; ++j)
#pragma unroll
                    for (int x = 0; x < 2; ++x)
#pragma unroll
                        for (int y = 0; y < 2; ++y) mma_bf16(acc[i + j][x][y], a[x], b[j][2 * y], b[j][2 * y + 1]);
                if (i > 0) {         // weight 7
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        const uint32_t b0 = next_weight(b[ND - i][2 * y]), b1 = next_weight(b[ND - i][2 * y + 1]);
#pragma unroll
                        for (int x = 0; x < 2; ++x) mma_bf16(acc[ND - 1][x][y], a[x], b0, b1);
                    }
                }
            }
        }
    };
    load(A, i0, kbeg, kend, pa);
    load(B, j0, kbeg, kend, pb);
    slice_stage(0);
    __syncthreads();
    for (int st = 0; st < stages; ++st) {
        const bool more = st + 1 < stages;
        if (warp & 4) {
            multiply(st);
            if (more) slice_stage(st + 1);
        } else {
            if (more) slice_stage(st + 1);
            multiply(st);
        }
        const int done = st + 1;
        if (done % (KF / KS) == 0 || !more) {    // FP32 sums to the chunk's integers
            const bool first = (st / (KF / KS)) % (KC / KF) == 0;
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                int g[ND];
#pragma unroll
                for (int s = 0; s < ND; ++s) {
                    float& f = acc[s][r >> 3][(r >> 2) & 1][r & 3];
                    g[s] = __float2int_rn(f);
                    f = 0.f;
                }
                long long h = ((long long)g[0] << 24) + ((long long)g[1] << 16) + ((long long)g[2] << 8) + g[3];
                long long l = ((long long)g[4] << 16) + ((long long)g[5] << 8) + g[6];
                long long* sh = sums + r * kThreads + tid;
                long long* sl = sh + 16 * kThreads;
                if (!first) { h += *sh; l += *sl; }
                *sh = h;
                *sl = l;
            }
        }
        if (done % (KC / KS) == 0 || !more) {    // the chunk's integers to the FP64 partial result
            const int chunk = (kbeg + st * KS) / KC;
            const bool first = st < KC / KS;
            double* W = ws + (long long)blockIdx.y * A.rows * ldw;
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int gi = i0 + wr + (r >> 3) * 16 + ((r >> 1) & 1) * 8 + (lane >> 2);
                const int gj = j0 + wc + ((r >> 2) & 1) * 8 + 2 * (lane & 3) + (r & 1);
                if (gi >= A.rows || gj >= B.rows) continue;
                const int ei = A.ex[(long long)gi * chunks + chunk], ej = B.ex[(long long)gj * chunks + chunk];
                const long long h = sums[r * kThreads + tid], l = sums[(16 + r) * kThreads + tid];
                const int e = 2152 - ei - ej;                                    // 2 x (1022 + 54)
                const double v = ei && ej ? fx::f64_scaled(h, e - 72) + fx::f64_scaled(l, e - 48) : 0.0;
                double* w = W + (long long)gi * ldw + gj;
                *w = first ? v : *w + v;
            }
        }
        __syncthreads();
    }
}

// C = alpha sum of the partial results (ascending) + beta C outside the flagged tiles; sym: the lower triangle from the
// upper one
__global__ void k_split_reduce(int m, int n, int nsplit, int sym, const double* __restrict__ ws, double* C, long long ldc,
                               double alpha, double beta, const int* __restrict__ flag) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long mn = (long long)m * n;
    if (idx >= mn) return;
    const long long i = idx / n, j = idx % n;
    if (flag[gemm_tile(i, j, n, sym)]) return;
    const long long src = sym && i > j ? j * n + i : idx;
    double s = 0.0;
    for (int z = 0; z < nsplit; ++z) s += ws[z * mn + src];
    double* cp = C + i * ldc + j;
    *cp = alpha * s + (beta != 0.0 ? beta * *cp : 0.0);
}

}  // namespace

cudaError_t launch_split_gemm(int m, int n, int k, const double* A, long long ai, long long ak, const double* B,
                              long long bk, long long bj, double* C, long long ldc, double alpha, double beta,
                              cudaStream_t s) {
    const bool sym = A == B && m == n && ai == bj && ak == bk;
    const long long tm = grid_for(m, TS), tn = grid_for(n, TS);
    const long long tiles = sym ? tm * (tm + 1) / 2 : tm * tn;
    if (tm * tn > 0x7fffffffLL) return cudaErrorInvalidValue;
    int dev = 0, sms = 152;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_split_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
    const int chunks = grid_for(k, KC);
    // one block per SM at a time: k is split so that the blocks come in about 4 waves, starting from a split count
    // whose blocks fill the last wave (the rounding to whole chunks can move it: 36 tiles and 394 chunks take 36)
    int nsplit = (int)std::min<long long>((4LL * sms + tiles - 1) / tiles, chunks);
    for (long long ns = nsplit; ns <= std::min<long long>(chunks, 4LL * nsplit); ++ns)
        if ((tiles * ns) % sms == 0) { nsplit = (int)ns; break; }
    const int per = (chunks + nsplit - 1) / nsplit;
    nsplit = (chunks + per - 1) / per;
    if (nsplit > 65535) return cudaErrorInvalidValue;
    const bool direct = nsplit == 1 && !sym && alpha == 1.0 && beta == 0.0;   // straight into C
    // The FP64 kernel meets few tiles as a rule: k in as many parts as one tile needs to fill the GPU (one failing tile
    // of 500 x 64 x 403440: 76 parts 24.4 ms, 601 parts 3.9 ms), within the products' workspace or 256 MB
    const long long most = std::max<long long>(nsplit, (1LL << 25) / ((long long)m * n));
    const GemmSplit f64 = gemm_split_tiles(1, most, k, sms);
    const size_t nex = (size_t)m * chunks + (sym ? 0 : (size_t)n * chunks);
    // the partial results: first the certificate's, then the products', then the FP64 kernel's for the flagged tiles
    const size_t nws = std::max<size_t>(direct ? 0 : (size_t)nsplit * m * n, f64.nsplit > 1 ? (size_t)f64.nsplit * m * n : 0);
    double* ws = nullptr;
    e = cudaMallocAsync(reinterpret_cast<void**>(&ws), sizeof(double) * nws + 2 * sizeof(int) * nex + sizeof(int) * (size_t)(tm * tn), s);
    if (e != cudaSuccess) return e;
    int* ex = reinterpret_cast<int*>(ws + nws);
    float* sq = reinterpret_cast<float*>(ex + nex);
    int* flag = reinterpret_cast<int*>(sq + nex);
    const size_t second = sym ? 0 : (size_t)m * chunks;
    const Op oa{A, ai, ak, m, ex, sq}, ob{B, bj, bk, n, ex + second, sq + second};
    const auto find = [&](const Op& o, size_t off) {
        const long long blocks = (long long)grid_for(o.rows, o.ks == 1 ? 8 : 32) * chunks;
        if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
        k_split_exponents<<<(unsigned)blocks, 256, 0, s>>>(o.p, o.rs, o.ks, o.rows, k, chunks, ex + off, sq + off);
        return cudaGetLastError();
    };
    const dim3 grid((unsigned)tiles, (unsigned)nsplit);
    const unsigned per_entry = (unsigned)grid_for((long long)m * n, 256);
    e = cudaMemsetAsync(flag, 0, sizeof(int) * (size_t)(tm * tn), s);
    if (e == cudaSuccess) e = find(oa, 0);
    if (e == cudaSuccess && !sym) e = find(ob, second);
    if (e == cudaSuccess) {
        k_split_check<<<grid, kThreads, 0, s>>>(oa, ob, k, per * KC, chunks, sym, direct ? nullptr : ws, flag);
        if (!direct) k_split_flags<<<per_entry, 256, 0, s>>>(m, n, nsplit, sym, ws, flag);
        k_split_gemm<<<grid, kThreads, kSmem, s>>>(oa, ob, k, per * KC, chunks, sym, direct ? C : ws, direct ? ldc : n, flag);
        if (!direct) k_split_reduce<<<per_entry, 256, 0, s>>>(m, n, nsplit, sym, ws, C, ldc, alpha, beta, flag);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = launch_gemm_f64(m, n, k, A, ai, ak, B, bk, bj, C, ldc, alpha, beta, f64, ws, flag, sym, s);
    const cudaError_t f = cudaFreeAsync(ws, s);
    return e != cudaSuccess ? e : f;
}

}  // namespace osam
