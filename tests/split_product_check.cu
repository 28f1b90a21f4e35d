// One product of the fit's kernels from a file: as the fit computes it (launch_gemm_*) and by the FP64 kernel alone.
// File: int32 m, n, k, layout (0: A [m][k] B [n][k], 1: A [m][k] B [k][n], 2: A [k][m] B [k][n], 3: B is A), then A and B
// as [m][k] and [n][k].  Output: both products [m][n] as doubles.
#include <cstdio>
#include <vector>

#include "osam_internal.h"

#define CHECK(x)                                                                                  \
    do {                                                                                          \
        const cudaError_t e_ = (x);                                                               \
        if (e_ != cudaSuccess) { std::fprintf(stderr, "%s: %s\n", #x, cudaGetErrorString(e_)); return 1; } \
    } while (0)

int main(int argc, char** argv) {
    if (argc != 3) return 1;
    int h[4];
    FILE* f = std::fopen(argv[1], "rb");
    if (!f || std::fread(h, 4, 4, f) != 4) return 1;
    const int m = h[0], n = h[1], k = h[2], layout = h[3];
    std::vector<double> A((size_t)m * k), B((size_t)n * k), C((size_t)m * n);
    if (std::fread(A.data(), 8, A.size(), f) != A.size() || std::fread(B.data(), 8, B.size(), f) != B.size()) return 1;
    std::fclose(f);
    const auto transposed = [k](const std::vector<double>& x, int rows) {
        std::vector<double> y(x.size());
        for (int i = 0; i < rows; ++i)
            for (int q = 0; q < k; ++q) y[(size_t)q * rows + i] = x[(size_t)i * k + q];
        return y;
    };
    if (layout == 2) A = transposed(A, m);
    if (layout == 1 || layout == 2) B = transposed(B, n);
    double *a, *b, *c, *ws;
    CHECK(cudaMalloc(&a, A.size() * 8));
    CHECK(cudaMalloc(&b, B.size() * 8));
    CHECK(cudaMalloc(&c, C.size() * 8));
    CHECK(cudaMemcpy(a, A.data(), A.size() * 8, cudaMemcpyHostToDevice));
    CHECK(cudaMemcpy(b, B.data(), B.size() * 8, cudaMemcpyHostToDevice));
    cudaStream_t s;
    CHECK(cudaStreamCreate(&s));
    FILE* out = std::fopen(argv[2], "wb");
    if (!out) return 1;
    CHECK(cudaMemset(c, 0xff, C.size() * 8));
    if (layout == 0) CHECK(osam::launch_gemm_nt(m, n, k, a, k, b, k, c, n, 1.0, 0.0, s));
    if (layout == 1) CHECK(osam::launch_gemm_nn(m, n, k, a, k, b, n, c, n, 1.0, 0.0, s));
    if (layout == 2) CHECK(osam::launch_gemm_tn(m, n, k, a, m, b, n, c, n, 1.0, 0.0, s));
    if (layout == 3) CHECK(osam::launch_gemm_nt(m, m, k, a, k, a, k, c, m, 1.0, 0.0, s));
    CHECK(cudaStreamSynchronize(s));
    CHECK(cudaMemcpy(C.data(), c, C.size() * 8, cudaMemcpyDeviceToHost));
    std::fwrite(C.data(), 8, C.size(), out);
    const osam::GemmSplit p = osam::gemm_split(m, n, k, 152);
    CHECK(cudaMalloc(&ws, (size_t)p.nsplit * m * n * 8));
    const bool kb = layout == 1 || layout == 2;
    CHECK(osam::launch_gemm_f64(m, n, k, a, layout == 2 ? 1 : k, layout == 2 ? m : 1, layout == 3 ? a : b, kb ? n : 1,
                                kb ? 1 : k, c, n, 1.0, 0.0, p, ws, nullptr, 0, s));
    CHECK(cudaStreamSynchronize(s));
    CHECK(cudaMemcpy(C.data(), c, C.size() * 8, cudaMemcpyDeviceToHost));
    std::fwrite(C.data(), 8, C.size(), out);
    std::fclose(out);
    return 0;
}
