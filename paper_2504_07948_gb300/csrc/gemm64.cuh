// FP64 GEMM from bf16 digits on the tensor cores (k_gemm64.cu).
#pragma once

#include <cuda_runtime.h>

namespace qmc {

constexpr int kGemm64Digits = 7;
constexpr int kGemm64MaxK = 170;   // exact FP32 sums of the digits' products

// One operand of a batch: digits [batch entry][stage of 32 k][digit][groups of
// 8 rows][4 k blocks][8 rows][8 k] and the rows' exponent fields.  A tile
// reads whole blocks of 128 rows (left operand) or 64 rows (right operand),
// so groups covers them; rows that no output needs may hold anything.
struct Gemm64Operand {
    unsigned char* dig;
    int* expo;
    size_t stride;   // bytes per batch entry (0: shared by the batch)
    int estride;     // exponents per batch entry (0: shared)
    int groups;
};
inline size_t gemm64_bytes(int groups, int K) {
    return (size_t)((K + 31) / 32) * kGemm64Digits * (size_t)groups * 512;
}

cudaError_t launch_digits(int batch, const double* X, long long sX, int ld, int trans, int rows, int rows8, int K,
                          const int* shift, long long sshift, int sign, const Gemm64Operand& o, int row0,
                          cudaStream_t st);
// D_b[m][n] for n < n1 into D1 (row stride ldd), for n2 <= n < N into column
// n - n2 of D2 (n1 <= n2; the columns between are not stored).
cudaError_t launch_gemm64(const Gemm64Operand& A, const Gemm64Operand& B, int M, int N, int K, int batch, double* D1,
                          long long sD1, int n1, int n2, double* D2, long long sD2, int ldd, unsigned* err,
                          cudaStream_t st);

}  // namespace qmc
