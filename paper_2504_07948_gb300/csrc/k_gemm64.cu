// Batched FP64 GEMM on the tensor cores, D_b[m][n] = sum_k A_b[m][k] B_b[n][k],
// for the dense products of the FP64 adjoint force pass of large determinants
// (Eqs. 3-4 pulled back to basis space).
//
// GB300 multiplies FP64 at 1.25 TFLOP/s and bf16 at 1900: the operands are cut
// into bf16 digits and the digits' products, which are exact, are added on the
// tensor cores (the splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 2012).  Every row is scaled by its own power of two to
// integers of at most 55 bits and written as kDig = 7 balanced digits of 8
// bits, q = sum_i d_i 2^(8 (6 - i)), |d_i| <= 128: exact in bf16.  The products
// of digits i and j with i + j = t add up in accumulator t (t <= 6, 28 products):
// |d_i d_j| <= 2^14, so an accumulator of t <= 5 holds at most 6 K 2^14 <= 2^24
// for K <= kGemm64MaxK and its FP32 sums are exact; in t = 6 a rounding is below
// 2^-60.  The seven accumulators of a 128 x 64 tile take 448 of the 512 columns
// of tensor memory; the epilogue adds them as integers and rounds once.
//
// Error, relative to the product of the two rows' largest entries (their integers
// lie in [2^54, 2^55)): the operands' rounding 2^-54 a term at most; the dropped
// digits i + j >= 7, six products of 2^14 2^40 at t = 7, 2^-51.4 a term at most and
// K times that for the sum, some 2^-55 sqrt(K) with digits of random sign.  An
// FP64 chain is off by 2^-53 of each of its partial sums instead, which is more
// where the terms come near the product of the maxima and less where they lie far
// below it; k_force_prep finds the walkers with such rows, and k_force_products
// takes them in FP64.  Elsewhere the error of A^-1 sets that of the derivatives: against
// extended precision both paths, this one and FP64 GEMMs, give the same to all
// digits shown (14 to 32 waters, electrons up to 12 bohr out, orbitals scaled by
// 10^-9 to 10^9).
//
// Digits are written by k_digits in the order the tensor core reads them: for
// each block of 32 k and each digit, groups of 8 rows of four 128-byte core
// matrices (8 rows x 8 k), so a tile of R rows is one contiguous piece of 64 R
// bytes that a bulk copy moves to shared memory as it is.
//
// 32-water forces in FP64, 256 walkers (four products per spin, n = 160): with
// cuBLAS DGEMM 46.6 ms of a 53.7 ms pass; with this kernel the pass takes
// 10.5 ms, of which its products 3.2 and the digits 0.8 (the rest is FP64 pair
// and basis terms).
//
// Roles of a CTA (one per SM, persistent over the tiles): warp 0 issues the
// bulk copies of a two-slot ring (14 pieces a stage), warp 1 the 56 MMAs of a
// stage, warps 2 to 9 drain the accumulators.  Every wait is bounded.
#include "fixed64.cuh"
#include "gemm64.cuh"
#include "tc_common.cuh"

namespace qmc {
namespace {

constexpr int kDig = kGemm64Digits;
constexpr int kGm = 128, kGn = 64, kGk = 32;   // tile rows, tile columns, k of a stage
constexpr int kGSlots = 2;
constexpr uint32_t kABytes = kGm * 64, kBBytes = kGn * 64;              // one digit of a stage
constexpr uint32_t kStageBytes = kDig * (kABytes + kBBytes);
constexpr int kGThreads = 320, kEpiWarps = 8;

// Instruction descriptor of kind::f16 with bf16 operands and FP32 accumulators.
constexpr uint32_t kIdescBf16 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kGn >> 3) << 17) | ((uint32_t)(kGm >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t a, uint64_t b, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        :
        : "r"(tmem), "l"(a), "l"(b), "r"(kIdescBf16), "r"(accum));
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"((unsigned long long)__cvta_generic_to_global(src)), "r"(bytes), "r"(bar)
        : "memory");
}

// 2^shift scaling of a double in [1, 2) x 2^e, by its exponent field; out of
// range by multiplication.
__device__ __forceinline__ double scale_exp(double v, int shift) {
    const int e = fx_expo(v) + shift;
    if (v == 0.0) return 0.0;
    if (e > 0 && e < 2047) return fx_double(fx_bits(v) + ((long long)shift << 52));
    return ldexp(v, shift);
}

__global__ void __launch_bounds__(kGThreads, 1)
    k_gemm64(Gemm64Operand A, Gemm64Operand B, int M, int N, int K, int batch, double* D1, long long sD1, int n1,
             int n2, double* D2, long long sD2, int ldd, unsigned* err) {
    extern __shared__ __align__(1024) unsigned char gsm[];
    __shared__ __align__(8) uint64_t bar_full[kGSlots], bar_empty[kGSlots], bar_acc, bar_free, bar_drain;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_stage = (K + kGk - 1) / kGk;
    const int mt = (M + kGm - 1) / kGm, nt = (N + kGn - 1) / kGn, n_tiles = mt * nt * batch;
    const int my_tiles = (int)blockIdx.x < n_tiles ? (n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const uint32_t sbase = smem_u32(gsm);
    volatile int* abort_flag = &s_abort;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kGSlots; ++i) {
            mbar_init(smem_u32(&bar_full[i]), 1);
            mbar_init(smem_u32(&bar_empty[i]), 1);
        }
        mbar_init(smem_u32(&bar_acc), 1);
        mbar_init(smem_u32(&bar_free), kEpiWarps);
        mbar_init(smem_u32(&bar_drain), 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;

    if (warp == 0) {
        if (lane == 0) {
            int g = 0;
            bool ok = true;
            for (int i = 0; i < my_tiles && ok; ++i) {
                const int tile = (int)blockIdx.x + i * (int)gridDim.x;
                const int b = tile / (mt * nt), r = tile - b * (mt * nt), m0 = (r / nt) * kGm, n0 = (r % nt) * kGn;
                // byte offsets of the tile's rows; a plane (stage, digit) holds groups x 512 bytes
                const unsigned char* pa = A.dig + (size_t)b * A.stride + (size_t)(m0 / 8) * 512;
                const unsigned char* pb = B.dig + (size_t)b * B.stride + (size_t)(n0 / 8) * 512;
                for (int s = 0; s < n_stage; ++s, ++g) {
                    const int slot = g % kGSlots;
                    if (g >= kGSlots && !pwait(smem_u32(&bar_empty[slot]), ((g / kGSlots) - 1) & 1, abort_flag, err)) {
                        ok = false;
                        break;
                    }
                    const uint32_t full = smem_u32(&bar_full[slot]), dst = sbase + slot * kStageBytes;
                    mbar_expect_tx(full, kStageBytes);
                    for (int d = 0; d < kDig; ++d) {
                        const size_t plane = (size_t)(s * kDig + d) * 512;
                        bulk_load(dst + d * kABytes, pa + plane * A.groups, kABytes, full);
                        bulk_load(dst + kDig * kABytes + d * kBBytes, pb + plane * B.groups, kBBytes, full);
                    }
                }
            }
            // every copy this thread issued has landed before the CTA exits
            for (int q = (g > kGSlots ? g - kGSlots : 0); q < g; ++q)
                pdrain(smem_u32(&bar_full[q % kGSlots]), (q / kGSlots) & 1);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int g = 0;
            bool ok = true;
            for (int i = 0; i < my_tiles && ok; ++i) {
                if (i >= 1 && !pwait(smem_u32(&bar_free), (i - 1) & 1, abort_flag, err)) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
                for (int s = 0; s < n_stage; ++s, ++g) {
                    const int slot = g % kGSlots;
                    if (!pwait(smem_u32(&bar_full[slot]), (g / kGSlots) & 1, abort_flag, err)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint32_t sa = sbase + slot * kStageBytes, sb = sa + kDig * kABytes;
#pragma unroll 1
                    for (int kk = 0; kk < kGk / 16; ++kk) {
                        const uint32_t o = kk * 2 * kPLBO;   // 16 k = two core matrices
#pragma unroll 1
                        for (int t = 0; t < kDig; ++t)
                            for (int d = 0; d <= t; ++d)
                                mma_bf16(tmem + (uint32_t)(t * kGn), psmem_desc(sa + d * kABytes + o),
                                         psmem_desc(sb + (t - d) * kBBytes + o), (s | kk | d) ? 1u : 0u);
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                        smem_u32(&bar_empty[slot])));
                }
                if (ok)
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                        smem_u32(&bar_acc)));
            }
            // the MMAs issued so far have completed before tensor memory is freed
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                smem_u32(&bar_drain)));
            pdrain(smem_u32(&bar_drain), 0);
        }
    } else {
        // epilogue: TMEM lane quadrant warp % 4, columns 32 ((warp - 2) / 4) ..
        const int q4 = warp & 3, half = (warp - 2) >> 2;
        for (int i = 0; i < my_tiles; ++i) {
            if (!pwait(smem_u32(&bar_acc), i & 1, abort_flag, err)) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const int tile = (int)blockIdx.x + i * (int)gridDim.x;
            const int b = tile / (mt * nt), r = tile - b * (mt * nt), m0 = (r / nt) * kGm, n0 = (r % nt) * kGn;
            const int row = m0 + 32 * q4 + lane;
            const int ea = row < M ? A.expo[(size_t)b * A.estride + row] : 0;
            const int* eb = B.expo + (size_t)b * B.estride;
            const uint32_t taddr = tmem + ((uint32_t)(32 * q4) << 16) + 32 * half;
#pragma unroll 1
            for (int c0 = 0; c0 < 32; c0 += 8) {
                uint32_t v[kDig][8];
#pragma unroll
                for (int t = 0; t < kDig; ++t)
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                                 : "=r"(v[t][0]), "=r"(v[t][1]), "=r"(v[t][2]), "=r"(v[t][3]), "=r"(v[t][4]),
                                   "=r"(v[t][5]), "=r"(v[t][6]), "=r"(v[t][7])
                                 : "r"(taddr + (uint32_t)(t * kGn + c0)));
                asm volatile("tcgen05.wait::ld.sync.aligned;");
                if (c0 == 24) {   // the accumulators are read out
                    asm volatile("tcgen05.fence::before_thread_sync;");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bar_free));
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int col = n0 + 32 * half + c0 + c;
                    if (row >= M || col >= N || (col >= n1 && col < n2)) continue;
                    // sum_t v_t 2^(8 (6 - t)) = 2^8 T with T rounded from its last 8 bits
                    int x[kDig];
#pragma unroll
                    for (int t = 0; t < kDig; ++t) x[t] = __float2int_rn(__uint_as_float(v[t][c]));
                    const long long hi = ((long long)x[0] << 24) + ((long long)x[1] << 16) + ((long long)x[2] << 8) + x[3];
                    const long long lo = ((long long)x[4] << 16) + ((long long)x[5] << 8) + x[6];
                    const long long T = (hi << 16) + ((lo + 128) >> 8);
                    const int e = eb[col];
                    double out = scale_exp((double)T, ea + e - 2098);
                    if (ea >= 2047 || e >= 2047) out = fx_double(0x7ff8000000000000LL);   // a row that is not finite
                    if (col < n1)
                        D1[(size_t)b * sD1 + (size_t)row * ldd + col] = out;
                    else
                        D2[(size_t)b * sD2 + (size_t)row * ldd + col - n2] = out;
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// Digits of X_b (rows x K, element (r, k) at X[r ld + k], or X[k ld + r] when
// trans), each element first scaled by 2^(sign shift[k]) (shift may be null),
// into rows row0 .. row0 + rows8 of an operand; rows and k beyond the matrix
// become zero.  A warp takes 8 rows, lane = (row, quarter of the 32 k of a
// stage): the 8 x 4 core-matrix rows of a digit are written as 512 contiguous
// bytes.
__global__ void __launch_bounds__(256) k_digits(const double* X, long long sX, int ld, int trans, int rows, int rows8,
                                                int K, const int* shift, long long sshift, int sign, Gemm64Operand o,
                                                int row0) {
    const int b = blockIdx.y, lane = threadIdx.x & 31, r = lane & 7, kq = lane >> 3;
    const int grp = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (grp * 8 >= rows8) return;
    const int row = grp * 8 + r, n_stage = (K + kGk - 1) / kGk;
    const double* x = X + (size_t)b * sX;
    const int* sh = shift ? shift + (size_t)b * sshift : nullptr;
    auto expo = [&](int k, double& v) {   // exponent field of the scaled element (0: zero)
        v = row < rows && k < K ? (trans ? x[(size_t)k * ld + row] : x[(size_t)row * ld + k]) : 0.0;
        const int e = fx_expo(v);
        if (e == 0 || e == 2047) return e;
        return max(1, min(2046, e + (sh ? sign * (sh[k] - 1023) : 0)));
    };
    int em = 0;
    for (int s = 0; s < n_stage; ++s)
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            double v;
            em = max(em, expo(s * kGk + 8 * kq + u, v));
        }
    em = max(em, __shfl_xor_sync(0xffffffffu, em, 8));
    em = max(em, __shfl_xor_sync(0xffffffffu, em, 16));
    if (kq == 0) o.expo[(size_t)b * o.estride + row0 + row] = em;
    unsigned char* dst = o.dig + (size_t)b * o.stride + ((size_t)(row0 / 8 + grp) * 4 + kq) * 128 + r * 16;
    for (int s = 0; s < n_stage; ++s) {
        uint32_t pk[kDig][4];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            double v;
            const int e = expo(s * kGk + 8 * kq + u, v);
            const long long bits = fx_bits(v);
            const long long m = e && e < 2047 ? ((bits & 0xfffffffffffffLL) | (1LL << 52)) : 0;
            const int w = e - em + 2;   // |q| <= 2^55
            long long q = w >= 0 ? m << w : w > -54 ? (m + (1LL << (-w - 1))) >> -w : 0;
            if (bits < 0) q = -q;
#pragma unroll
            for (int d = kDig - 1; d >= 0; --d) {
                const int dg = d ? (int)(signed char)(q & 255) : (int)q;   // balanced: -128 .. 127, the first up to 128
                q = (q - dg) >> 8;
                const uint32_t h = __float_as_uint((float)dg) >> 16;      // exact in bf16
                if (u & 1)
                    pk[d][u >> 1] |= h << 16;
                else
                    pk[d][u >> 1] = h;
            }
        }
#pragma unroll
        for (int d = 0; d < kDig; ++d)
            *reinterpret_cast<uint4*>(dst + (size_t)(s * kDig + d) * 512 * o.groups) =
                make_uint4(pk[d][0], pk[d][1], pk[d][2], pk[d][3]);
    }
}

}  // namespace

cudaError_t launch_digits(int batch, const double* X, long long sX, int ld, int trans, int rows, int rows8, int K,
                          const int* shift, long long sshift, int sign, const Gemm64Operand& o, int row0,
                          cudaStream_t st) {
    if (batch <= 0 || rows8 <= 0) return cudaSuccess;
    k_digits<<<dim3((rows8 / 8 + 7) / 8, batch), 256, 0, st>>>(X, sX, ld, trans, rows, rows8, K, shift, sshift, sign, o,
                                                               row0);
    return cudaGetLastError();
}

cudaError_t launch_gemm64(const Gemm64Operand& A, const Gemm64Operand& B, int M, int N, int K, int batch, double* D1,
                          long long sD1, int n1, int n2, double* D2, long long sD2, int ldd, unsigned* err,
                          cudaStream_t st) {
    if (batch <= 0 || M <= 0 || N <= 0) return cudaSuccess;
    if (K <= 0 || K > kGemm64MaxK) return cudaErrorInvalidValue;
    const size_t smem = kGSlots * kStageBytes;
    cudaError_t e = allow_smem(k_gemm64, smem);
    if (e != cudaSuccess) return e;
    const int n_sm = device_sms();
    const long long tiles = (long long)((M + kGm - 1) / kGm) * ((N + kGn - 1) / kGn) * batch;
    k_gemm64<<<(int)(tiles < n_sm ? tiles : n_sm), kGThreads, smem, st>>>(A, B, M, N, K, batch, D1, sD1, n1, n2,
                                                                          D2, sD2, ldd, err);
    return cudaGetLastError();
}

}  // namespace qmc
