// Full (non-incremental) wavefunction evaluation at fixed walker
// configurations: basis -> orbitals for every electron, FP64 inversion of
// the Slater matrices, and the local energy.  These kernels serve the
// parity entry point and the periodic FP64 recompute of the incremental
// inverse.
#include <algorithm>

#include "basis64.cuh"
#include "batch.cuh"
#include "qmc_internal.cuh"

namespace qmc {

// Whether the orbitals of this basis are taken in fixed point.
__host__ __device__ static inline bool orbitals_fx(const DevSys& s) {
    return Basis64Layout(s.n_nuc, s.n_prim, s.n_shell, s.n_basis).total <= kBasis64Max;
}

// Orbitals of electron i of walker w by one CTA (body of k_orbitals_all):
// the live basis functions at r_i in FP64 and the LCAO contraction phi_j =
// sum_l C_l^j Phi_l (Eq. 2) in fixed point (basis64.cuh) for the occupied
// orbitals of the electron's spin and the active virtual ones of a
// determinant expansion.  A goes to FP64 scratch, the gradient and Laplacian
// rows to the walker cache in the storage type T.  sm: orbitals_smem_bytes of
// shared memory (a basis whose lists exceed it, about 2500 functions, is
// contracted in FP64).
template <typename T>
__device__ __forceinline__ void orbitals_item(const DevSys& s, const DevWalkers& wk, int w, int i, unsigned char* sm) {
    const Basis64Layout L(s.n_nuc, s.n_prim, s.n_shell, s.n_basis);
    const double* rp = wk.R + ((size_t)w * s.N + i) * 3;
    const double r[3] = {rp[0], rp[1], rp[2]};
    const int spin = i < s.n_up ? 0 : 1;
    const int n = spin ? s.n_dn : s.n_up, nv = s.msd ? s.n_vir[spin] : 0;
    const int k = spin ? i - s.n_up : i;
    T* G = (T*)wk.G[spin] + ((size_t)w * n + k) * 4 * n;
    double* A = wk.Ascr[spin] + ((size_t)w * n + k) * n;
    T* Av = (T*)wk.Av[spin] + ((size_t)w * n + k) * nv;
    T* Gv = (T*)wk.Gv[spin] + ((size_t)w * n + k) * 4 * nv;
    const auto put = [&](int c, int j, double v) {
        if (c == 0)
            A[j] = v;
        else
            G[(c - 1) * n + j] = (T)v;
    };
    const auto put_v = [&](int c, int j, double v) {
        if (c == 0)
            Av[j] = (T)v;
        else
            Gv[(c - 1) * nv + j] = (T)v;
    };
    if (orbitals_fx(s)) {
        orbitals64(s, L, sm, r[0], r[1], r[2], s.Ck[spin], s.Ck_s[spin], s.C[spin], n, put, s.Cvk[spin], s.Cvk_s[spin],
                   s.Cv[spin], nv, put_v);
    } else {
        orbitals_plain(s, r, s.C[spin], n, (double*)sm, put);
        if (nv > 0) orbitals_plain(s, r, s.Cv[spin], nv, (double*)sm, put_v);
    }
}

template <typename T>
__global__ void __launch_bounds__(320, 2) k_orbitals_all(DevSys s, DevWalkers wk, int W, const int* only) {
    extern __shared__ double sh_bas[];
    const int w = blockIdx.x, i = blockIdx.y;
    if (w >= W || (only && !only[w])) return;
    orbitals_item<T>(s, wk, w, i, (unsigned char*)sh_bas);
}

// The same orbitals as FP64 sums over the basis functions in index order (51.9
// against 9.3 ms for 256 walkers of the 32-water cluster: bound by the FP64
// pipe).  New walkers of the mixed form are built with it, and walkers a
// determinant expansion rebuilds inside a sweep: the last bit of an FP64 sum
// decides how an FP32 inverse rounds, and a mixed trajectory amplifies one such
// bit until an accept decision turns, so a seeded mixed run repeats earlier
// ones only from the same bits.  Also for a basis whose lists exceed shared
// memory, and for the spins of a rebuild that fixed point would cost bits
// (orbitals_again).  sh_bas: 5 n_basis doubles of shared memory.  live (n_shell
// bytes of shared memory): shells whose values and derivatives are all exactly
// zero (screened) are left out of the occupied-orbital contraction; the terms
// that remain are added in the same order.
template <typename T>
__device__ __forceinline__ void orbitals_sums_item(const DevSys& s, const DevWalkers& wk, int w, int i, double* sh_bas,
                                                   unsigned char* live) {
    const int nb = s.n_basis;
    double r[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) r[c] = wk.R[((size_t)w * s.N + i) * 3 + c];
    for (int sh = threadIdx.x; sh < s.n_shell; sh += blockDim.x) shell_vgl<double>(s, sh, r, sh_bas, nb);
    __syncthreads();
    for (int sh = threadIdx.x; sh < s.n_shell; sh += blockDim.x) {
        const int f0 = s.shell_fn[sh], f1 = s.shell_fn[sh + 1];
        bool nz = false;
        for (int c = 0; c < 5 && !nz; ++c)
            for (int f = f0; f < f1 && !nz; ++f) nz = sh_bas[c * nb + f] != 0.0;
        live[sh] = nz ? 1 : 0;
    }
    __syncthreads();
    const int spin = i < s.n_up ? 0 : 1;
    const int n = spin ? s.n_dn : s.n_up;
    const int k = spin ? i - s.n_up : i;
    const double* C = s.C[spin];
    T* G = (T*)wk.G[spin] + ((size_t)w * n + k) * 4 * n;
    double* A = wk.Ascr[spin] + ((size_t)w * n + k) * n;
    for (int o = threadIdx.x; o < 5 * n; o += blockDim.x) {
        const int c = o / n, j = o - c * n;
        const double* b = sh_bas + c * nb;
        double acc = 0.0;
        for (int sh = 0; sh < s.n_shell; ++sh) {
            if (!live[sh]) continue;
            for (int l = s.shell_fn[sh]; l < s.shell_fn[sh + 1]; ++l) acc += C[(size_t)l * n + j] * b[l];
        }
        if (c == 0)
            A[j] = acc;
        else
            G[(c - 1) * n + j] = (T)acc;
    }
    if (s.msd) {  // active virtual orbitals of a determinant expansion
        const int nv = s.n_vir[spin];
        const double* Cv = s.Cv[spin];
        T* Av = (T*)wk.Av[spin] + ((size_t)w * n + k) * nv;
        T* Gv = (T*)wk.Gv[spin] + ((size_t)w * n + k) * 4 * nv;
        for (int o = threadIdx.x; o < 5 * nv; o += blockDim.x) {
            const int c = o / nv, p = o - c * nv;
            const double* b = sh_bas + c * nb;
            double acc = 0.0;
            for (int l = 0; l < nb; ++l) acc += Cv[(size_t)l * nv + p] * b[l];
            if (c == 0)
                Av[p] = (T)acc;
            else
                Gv[(c - 1) * nv + p] = (T)acc;
        }
    }
}

template <typename T>
__global__ void k_orbitals_sums(DevSys s, DevWalkers wk, int W, const int* only) {
    extern __shared__ double sh_bas[];  // [5][n_basis], then one live flag per shell
    const int w = blockIdx.x, i = blockIdx.y;
    if (w >= W || (only && !only[w])) return;
    orbitals_sums_item<T>(s, wk, w, i, sh_bas, reinterpret_cast<unsigned char*>(sh_bas + 5 * s.n_basis));
}

// In-place Gauss-Jordan inversion with partial (row) pivoting, FP64, one
// CTA per (walker, spin), the n x n matrix in shared memory.  Produces
// ln|det A|, sign(det A) and the transposed inverse in the storage type.
//
// Bound by the FP64 pipe for large n (n^3 multiply-adds: 12,500 of some 15,500
// cycles a pivot at n = 160), by the chain from pivot to pivot for small ones.
// So no FP64 instruction is spent on the rest: magnitudes are compared as
// integers, one lane takes the reciprocal, the logarithms wait for the end, and
// a warp walks a row without divisions.  While the other warps eliminate column
// k, warp 0 first brings column k + 1 up to date and picks its pivot: two
// barriers a pivot.  Row interchanges are collected as one permutation of the
// result's columns.  2 x 77 matrices of 15: 50 -> 27 us; 512 of 160: 6.9 -> 6.0 ms
// (serial pivot search and logarithm, five barriers, a reciprocal per thread).
//
// Rows of A taken in fixed point carry an error of about 2^-59 sqrt(rows) of the
// row's largest entry, in units of the orbitals' largest coefficients, where
// FP64 sums keep every entry's own bits.  That matters where the inverse weighs
// a row's small entries up: electrons shared out unevenly over distant fragments
// with orbitals of their own.  So the inverse is held against its rows:
// with x = A^-1 e_i, a row whose max|x_j| c_j max|A_ij / c_j| exceeds max|x_j
// A_ij| by more than kFxSlack bits would lose accuracy against FP64 sums (their
// error is some 2^-54 sqrt(rows) of the latter).  The orbitals of such rows are
// taken again that way (of all rows, if the matrix is singular) and the matrix is
// inverted again, until no further row stands out.  On water clusters with dense
// orbitals (1 to 32 waters) no row comes above 4 bits; with orbitals of a model
// Hamiltonian one or two in a hundred pass 6, and with two waters 11 bohr apart, six
// electrons of a spin on one of them, the rows concerned stand at 8 to 20.  Left to
// fixed point, the model orbitals' E_L and gradients at 14 waters had 2 to 7
// times the error of FP64 sums, now the same.

// Pivot of column k from row k on (warp 0): row, value and reciprocal.
__device__ __forceinline__ void find_pivot(const double* M, int n, int k, int* s_piv, double* s_val, double* s_pinv,
                                           int* s_sing) {
    const int lane = threadIdx.x & 31;
    long long best = -1;
    int bi = k;
    for (int i = k + lane; i < n; i += 32) {
        long long v = fx_bits(M[i * n + k]) & 0x7fffffffffffffffLL;   // |.| in the order of its value
        if (v > 0x7ff0000000000000LL) v = -1;                         // never a NaN
        if (v > best) {
            best = v;
            bi = i;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) {
            best = ob;
            bi = oi;
        }
    }
    if (lane == 0) {
        const double v = M[bi * n + k];
        const int e = fx_expo(v);
        *s_piv = bi;
        *s_pinv = 1.0 / v;
        *s_val = v;
        if (e == 2047 || (fx_bits(v) & 0x7fffffffffffffffLL) == 0) *s_sing = 1;
    }
}

// The orbitals of one spin's electrons k with rows[k] as FP64 sums, by the whole
// CTA; ends synchronised.  sm: 5 n_basis doubles and n_shell bytes of shared memory.
__device__ __noinline__ void orbitals_again(const DevSys& s, const DevWalkers& wk, int w, int spin, int fp32,
                                            const int* rows, double* sm) {
    const int i0 = spin ? s.n_up : 0, n = spin ? s.n_dn : s.n_up;
    unsigned char* live = reinterpret_cast<unsigned char*>(sm + 5 * s.n_basis);
    for (int k = 0; k < n; ++k) {
        if (!rows[k]) continue;
        if (fp32)
            orbitals_sums_item<float>(s, wk, w, i0 + k, sm, live);
        else
            orbitals_sums_item<double>(s, wk, w, i0 + k, sm, live);
        __syncthreads();
    }
}

// Whether row i of A (global memory) leaves the inverse x[j] = M[j n + c] short
// of bits if taken in fixed point (see above); by one warp.
__device__ __forceinline__ bool row_short(const double* A, const double* M, const double* __restrict__ sC, int n, int i,
                                          int c) {
    int am = 0, rs = 0, rf = 0;   // biased exponents: max|x_j| c_j, max|A_ij| / c_j, max|x_j A_ij|
    for (int j = threadIdx.x & 31; j < n; j += 32) {
        const int ea = fx_expo(A[(size_t)i * n + j]), ex = fx_expo(M[j * n + c]), ec = fx_expo(sC[j]);
        am = max(am, ex + ec);
        if (ea) rs = max(rs, ea - ec + 4096);
        if (ea && ex) rf = max(rf, ea + ex);
    }
    return warp_max_u(am) + warp_max_u(rs) - 4096 - warp_max_u(rf) > kFxSlack;
}

constexpr int kInvertWarps = 16;   // at most; words of shrt per walker and spin

// Rows of A that fall short (of a singular matrix all) and are not FP64 sums yet,
// after the elimination: warp w looks at the rows w, w + nw, .. (at most 32) and
// returns a bit for each.  summed: those that are.  perm: the columns of the
// inverse in M.
__device__ __forceinline__ int short_rows(const DevSys& s, const double* A, int n, int spin, int sing, int summed,
                                          const int* perm, const double* M) {
    const int wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int now = 0;
    for (int i = wid, q = 0; i < n; i += nw, ++q)
        if (!(summed >> q & 1) && (sing || row_short(A, M, s.Ck_s[spin], n, i, perm[i]))) now |= 1 << q;
    return now;
}

// Takes the rows of these bits again; rows: n integers of shared memory.
__device__ __noinline__ void take_rows(const DevSys& s, const DevWalkers& wk, int w, int spin, int fp32, int now, int* rows,
                                       double* M) {
    const int n = spin ? s.n_dn : s.n_up, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0)
        for (int i = wid, q = 0; i < n; i += nw, ++q) rows[i] = now >> q & 1;
    __syncthreads();
    orbitals_again(s, wk, w, spin, fp32, rows, M);
}

// Inversion of one (walker, spin) matrix (body of k_invert).  M: n^2 + n
// doubles of shared memory (invert_smem_bytes); at least n threads.  fx: A was
// taken in fixed point.  kAgain: takes short rows again and inverts until none is
// left; now: rows to take before the first inversion (short_rows).  Without it the
// rows are left to a launch that does: shrt (fx) receives the bits of each warp.
template <bool kAgain>
__device__ __forceinline__ void invert_item(const DevSys& s, const DevWalkers& wk, int w, int spin, int store_fp32, int fx,
                                            int now, int* shrt, unsigned* err, double* M) {
    __shared__ int s_perm[256];
    __shared__ double s_val, s_pinv;
    __shared__ int s_piv, s_sing, s_row[2];
    const int n = spin ? s.n_dn : s.n_up;
    if (n == 0) {
        if (threadIdx.x == 0) {
            wk.logdet[2 * w + spin] = 0.0;
            wk.sgn[2 * w + spin] = 1.0;
        }
        return;
    }
    double* fcol = M + n * n;
    const double* A = wk.Ascr[spin] + (size_t)w * n * n;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // rows of an elimination step of a warp, and this lane's row and first column of them
    const int sub = n <= 8 ? 8 : n <= 16 ? 16 : 32, nrow = 32 / sub, lr = lane / sub, lc = lane % sub;
    int cur = 0, swaps = 0, neg = 0;   // where this thread's column ends up; interchanges; negative pivots
    double piv = 0.0;                  // this thread's pivot
    int summed = 0;                    // rows of A that are FP64 sums (short_rows)
    for (;;) {
        if constexpr (kAgain)
            if (__syncthreads_or(now)) {
                take_rows(s, wk, w, spin, store_fp32, now, s_perm, M);
                summed |= now;
            }
        if (threadIdx.x == 0) {
            s_sing = 0;
            s_row[0] = s_row[1] = 0;
        }
        for (int q = threadIdx.x; q < n * n; q += blockDim.x) M[q] = A[q];
        __syncthreads();
        if (wid == 0) find_pivot(M, n, 0, &s_piv, &s_val, &s_pinv, &s_sing);
        __syncthreads();
        cur = threadIdx.x;
        swaps = 0;
        for (int k = 0; k < n; ++k) {
            if (s_sing) break;   // uniform: written before the last barrier
            const int p = s_piv;
            const double pinv = s_pinv;
            if (threadIdx.x == k) piv = s_val;
            // interchange rows k and p, scale the pivot row, keep the column
            for (int j = threadIdx.x; j < n; j += blockDim.x) {
                const double t = M[k * n + j], u = M[p * n + j];
                if (p != k) M[p * n + j] = t;
                M[k * n + j] = (j == k) ? pinv : u * pinv;
                if (j == k) {
                    if (p != k) fcol[p] = t;
                    fcol[k] = 0.0;
                }
                if (j != k && j != p) fcol[j] = M[j * n + k];
            }
            if (threadIdx.x == 0) s_row[(k + 1) & 1] = 0;
            swaps += p != k;
            cur = cur == k ? p : cur == p ? k : cur;
            __syncthreads();
            const int ahead = k + 1 < n ? k + 1 : -1;   // the column that warp 0 takes
            if (wid == 0 && ahead > 0) {
                for (int i = lane; i < n; i += 32)
                    if (i != k) M[i * n + ahead] = M[i * n + ahead] - fcol[i] * M[k * n + ahead];
                __syncwarp();
                find_pivot(M, n, ahead, &s_piv, &s_val, &s_pinv, &s_sing);
            }
            for (;;) {   // the other columns, rows to whichever warp is free
                int i = 0;
                if (lane == 0) i = atomicAdd(&s_row[k & 1], nrow);
                i = __shfl_sync(0xffffffffu, i, 0);
                if (i >= n) break;
                i += lr;
                if (i == k || i >= n) continue;
                const double f = fcol[i];
                for (int j = lc; j < n; j += sub) {
                    if (j == ahead) continue;
                    const double base = (j == k) ? 0.0 : M[i * n + j];
                    M[i * n + j] = base - f * M[k * n + j];
                }
            }
            __syncthreads();
        }
        neg = 0;
        if (!s_sing)
            for (int k = threadIdx.x; k < n; k += blockDim.x) {
                s_perm[k] = cur;
                neg = piv < 0.0;
                fcol[k] = log(fabs(piv));
            }
        neg = __syncthreads_count(neg);
        if (!fx) break;
        now = short_rows(s, A, n, spin, s_sing, summed, s_perm, M);
        if (!kAgain) {
            if (lane == 0) shrt[(2 * w + spin) * kInvertWarps + wid] = now;
            break;
        }
        if (!__syncthreads_or(now)) break;
    }
    if (s_sing) {
        if (!kAgain && fx) return;   // not settled: every row is taken again
        if (threadIdx.x == 0) {
            wk.logdet[2 * w + spin] = -INFINITY;
            wk.sgn[2 * w + spin] = 0.0;
            atomicOr(err, kErrSingular);
        }
        return;
    }
    // AinvT[e][j] = (A^-1)[j][e], the interchanges undone as interchanges of its columns, last first
    if (store_fp32) {
        float* out = (float*)wk.Ainv[spin] + (size_t)w * n * n;
        for (int q = threadIdx.x; q < n * n; q += blockDim.x) {
            const int e = q / n, j = q - e * n;
            out[q] = (float)M[j * n + s_perm[e]];
        }
    } else {
        double* out = (double*)wk.Ainv[spin] + (size_t)w * n * n;
        for (int q = threadIdx.x; q < n * n; q += blockDim.x) {
            const int e = q / n, j = q - e * n;
            out[q] = M[j * n + s_perm[e]];
        }
    }
    if (threadIdx.x == 0) {
        double ld = 0.0;
        for (int k = 0; k < n; ++k) ld += fcol[k];
        wk.logdet[2 * w + spin] = ld;
        wk.sgn[2 * w + spin] = (neg + swaps) & 1 ? -1.0 : 1.0;
    }
}

__global__ void k_invert(DevSys s, DevWalkers wk, int W, int store_fp32, int* shrt, unsigned* err, const int* only) {
    extern __shared__ double M[];  // [n][n], then fcol[n]
    const int w = blockIdx.x, spin = blockIdx.y;
    if (w >= W || (only && !only[w])) return;
    invert_item<false>(s, wk, w, spin, store_fp32, shrt != nullptr, 0, shrt, err, M);
}

// The matrices with rows that k_invert found short, taken again.  A kernel of its
// own: with this work the elimination would need 112 registers, where 40 leave
// room for three CTAs of the large size on an SM.
__global__ void __launch_bounds__(32 * kInvertWarps) k_invert_again(DevSys s, DevWalkers wk, int W, int store_fp32,
                                                                    const int* shrt, unsigned* err, const int* only) {
    extern __shared__ double M[];
    const int w = blockIdx.x, spin = blockIdx.y;
    if (w >= W || (only && !only[w]) || (spin ? s.n_dn : s.n_up) == 0) return;
    const int now = shrt[(2 * w + spin) * kInvertWarps + (threadIdx.x >> 5)];
    if (!__syncthreads_or(now)) return;
    invert_item<true>(s, wk, w, spin, store_fp32, 1, now, nullptr, err, M);
}

// Local energy, ln|psi| and (optionally) grad / Laplacian of ln|psi| from
// the cached inverse and orbital gradient/Laplacian rows.  One CTA per
// walker, one thread per electron; sums in FP64.
//   E_L = sum_i -1/2 [lap_i D/D + lap_i J + 2 grad_i J . grad_i D/D
//         + |grad_i J|^2] + V_ee + V_en + V_nn.
// J3 seen from electron i: the value of the pairs (i, j > i) and the
// gradient and Laplacian in r_i of every pair (i, j != i).
__device__ void j3_electron(const DevSys& s, const double* sR, int i, double& val, double g[3], double& lap) {
    val = 0.0;
    g[0] = g[1] = g[2] = 0.0;
    lap = 0.0;
    const double* ri = sR + 3 * i;
    for (int a = 0; a < s.n_nuc; ++a) {
        const double* ra = s.Rn + 3 * a;
        const SDist xi = sdist(s.b3, ri[0] - ra[0], ri[1] - ra[1], ri[2] - ra[2]);
        const double* c = s.c3 + (size_t)a * s.n3;
        for (int j = 0; j < s.N; ++j) {
            if (j == i) continue;
            const double* rj = sR + 3 * j;
            const SDist xj = sdist(s.b3, rj[0] - ra[0], rj[1] - ra[1], rj[2] - ra[2]);
            const SDist y = sdist(s.b3, ri[0] - rj[0], ri[1] - rj[1], ri[2] - rj[2]);
            for (int k = 0; k < s.n3; ++k) {
                if (c[k] == 0.0) continue;
                double v, gg[3], l;
                j3_term(s.e3[3 * k], s.e3[3 * k + 1], s.e3[3 * k + 2], xi, xj, y, v, gg, l);
                if (j > i) val += c[k] * v;
                g[0] += c[k] * gg[0];
                g[1] += c[k] * gg[1];
                g[2] += c[k] * gg[2];
                lap += c[k] * l;
            }
        }
    }
}

// Local energy of walker w (body of k_eloc).  The first half of the CTA's
// threads takes the electron pairs, the second half the electron-nucleus
// terms, the determinant and the assembly, a thread per electron each (strided
// when the electrons outnumber it), so that the two parts run on different
// warps at once.
//   FP64 form (bound by its FP64 instructions): up to kElocSym electrons every
// pair is formed once, by electron i for the cyclic neighbours i + 1 .. i + N/2,
// and added to both: the partner's share goes to an array of the warp, in which
// the lanes of a round touch distinct electrons.
//   Mixed form (was bound by uncoalesced reads of the gradient cache, a row
// per thread): the determinant sums of an electron are taken by a warp; pair
// terms in FP32 with compensated sums, assembled in FP64.
// 6-water cluster, 2048 walkers: 756 -> 438 us FP64, 143 -> 92 us mixed;
// 32-water cluster, 1024 walkers, mixed: 1.84 -> 0.87 ms (a thread per electron
// for everything before).
// kElocSym keeps the warps' arrays within 10 KB; it is not where the two forms
// cross: pairs once takes 0.90 against 1.28 ms at 16 waters (160 electrons, 512
// walkers) and would take 1.51 against 2.18 ms at 20, 1.74 against 2.47 ms at 32
// waters (256 walkers; 100 KB of shared memory).
// sm: eloc_smem_bytes.
constexpr int kElocSym = 160;
struct ElocLayout {
    int H;                      // threads of each half
    // byte offsets of [N][4] pair sums (mixed form [N][5]: the Laplacian as high and low word), and of the
    // partners' shares [H / 32][4][N] or the determinant sums [N][8]
    size_t part, other, total;
    __host__ __device__ ElocLayout(int N, int nt, int elem) {
        H = nt / 2;
        const size_t pos = (sizeof(double) * 3 + sizeof(float) * 8) * (size_t)N;
        part = (pos + 15) & ~(size_t)15;
        other = (part + (size_t)elem * (elem == 4 ? 5 : 4) * N + 15) & ~(size_t)15;
        total = other + (elem == 4 ? sizeof(float) * 8 * (size_t)N
                                   : N <= kElocSym ? sizeof(double) * 4 * (size_t)N * (H / 32) : 0);
        total = (total + 15) & ~(size_t)15;
    }
};
size_t eloc_smem_bytes(const DevSys& s, int nt, int elem) { return ElocLayout(s.N, nt, elem).total; }

template <typename T>
__device__ __forceinline__ void eloc_walker(const DevSys& s, const DevWalkers& wk, int w, double* eloc_out, double* logpsi, double* grad,
                                            double* lap, unsigned* err, unsigned char* sm) {
    __shared__ double scratch[kMaxWarps * 2];
    const int N = s.N, nu = s.n_up, nn = s.n_nuc;
    const ElocLayout L(N, blockDim.x, sizeof(T));
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, H = L.H;
    double* sR = (double*)sm;
    float4* sRf = (float4*)(sR + 3 * N + (N & 1));   // float positions of the mixed form's pairs
    T* part = (T*)(sm + L.part);
    for (int q = tid; q < 3 * N; q += blockDim.x) sR[q] = wk.R[(size_t)w * 3 * N + q];
    __syncthreads();
    if constexpr (sizeof(T) == 4) {
        for (int i = tid; i < N; i += blockDim.x)
            sRf[i] = make_float4((float)sR[3 * i], (float)sR[3 * i + 1], (float)sR[3 * i + 2], 0.f);
        // determinant sums (gradient and Laplacian over the orbitals), a warp per electron
        float* det = (float*)(sm + L.other);   // [N][8]: four (high, low) pairs
        for (int i = wid; i < N; i += (int)blockDim.x >> 5) {
            const int spin = i >= nu, n = spin ? s.n_dn : nu, k = spin ? i - nu : i;
            const float* Ai = (const float*)wk.Ainv[spin] + ((size_t)w * n + k) * n;
            const float* Gi = (const float*)wk.G[spin] + ((size_t)w * n + k) * 4 * n;
            Acc<float> dd[4];
            for (int j = lane; j < n; j += 32) {
                const float a = Ai[j];
#pragma unroll
                for (int c = 0; c < 4; ++c) dd[c].add(Gi[c * n + j] * a);
            }
            // transposing butterfly over the four sums: lanes 8 q hold sum q
            const bool h4 = lane & 16, h3 = lane & 8;
            Acc<float> r[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const Acc<float> send = h4 ? dd[q] : dd[q + 2];
                r[q] = h4 ? dd[q + 2] : dd[q];
                r[q].add_pair(__shfl_xor_sync(0xffffffffu, send.h, 16), __shfl_xor_sync(0xffffffffu, send.l, 16));
            }
            const Acc<float> send = h3 ? r[0] : r[1];
            Acc<float> t = h3 ? r[1] : r[0];
            t.add_pair(__shfl_xor_sync(0xffffffffu, send.h, 8), __shfl_xor_sync(0xffffffffu, send.l, 8));
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
                t.add_pair(__shfl_xor_sync(0xffffffffu, t.h, o), __shfl_xor_sync(0xffffffffu, t.l, o));
            if ((lane & 7) == 0) {
                const int q = ((lane >> 3) & 1) + 2 * (lane >> 4);
                det[8 * i + 2 * q] = t.h;
                det[8 * i + 2 * q + 1] = t.l;
            }
        }
        __syncthreads();
    }
    double v[2] = {0.0, 0.0};
    if (tid < H) {
        // ---- electron pairs: gradient and Laplacian of J per electron into part
        if constexpr (sizeof(T) == 4) {
            const float b = (float)s.b_ee;
            for (int i = tid; i < N; i += H) {
                const float4 ri = sRf[i];
                float gx = 0.f, gy = 0.f, gz = 0.f;
                Acc<float> lJ, Ji, V;
                for (int half = 0; half < 2; ++half) {   // the pairs' own values once, from the lower electron
                    const int j0 = half ? i + 1 : 0, j1 = half ? N : i;
                    for (int j = j0; j < j1; ++j) {
                        const float4 rj = sRf[j];
                        const float x = ri.x - rj.x, y = ri.y - rj.y, z = ri.z - rj.z;
                        const float r2 = x * x + y * y + z * z;
                        const float ir = rsqrtf(r2), r = r2 * ir;
                        const float a = (float)(((i < nu) == (j < nu)) ? s.a_par : s.a_anti);
                        const float q = 1.0f / (1.0f + b * r);
                        const float du = a * q * q, g = du * ir;
                        gx += g * x;
                        gy += g * y;
                        gz += g * z;
                        lJ.add(-2.0f * b * du * q + 2.0f * g);
                        if (half) {
                            Ji.add(a * r * q);
                            V.add(ir);
                        }
                    }
                }
                v[0] += (double)V.h + V.l;
                v[1] += (double)Ji.h + Ji.l;
                part[5 * i] = gx;
                part[5 * i + 1] = gy;
                part[5 * i + 2] = gz;
                part[5 * i + 3] = lJ.h;
                part[5 * i + 4] = lJ.l;
            }
        } else {
            const double b = s.b_ee;
            // u, u'/r and the Laplacian u'' + 2 u'/r with one reciprocal square
            // root and one reciprocal: u = a r q, u' = a q^2, u'' = -2 b u' q
            double x, y, z, ir, u, g, l;
            auto pair = [&](int i, int j) {
                x = sR[3 * i] - sR[3 * j];
                y = sR[3 * i + 1] - sR[3 * j + 1];
                z = sR[3 * i + 2] - sR[3 * j + 2];
                const double r2 = x * x + y * y + z * z;
                ir = rsqrt(r2);
                const double r = r2 * ir, q = 1.0 / (1.0 + b * r);
                const double aq = (((i < nu) == (j < nu)) ? s.a_par : s.a_anti) * q, du = aq * q;
                u = aq * r;
                g = du * ir;
                l = fma(-2.0 * b, du * q, 2.0 * g);
            };
            if (N <= kElocSym) {
                double* oth = (double*)(sm + L.other) + (size_t)wid * 4 * N;
                for (int q = lane; q < 4 * N; q += 32) oth[q] = 0.0;
                __syncwarp();
                for (int i0 = tid - lane; i0 < N; i0 += H) {   // whole warps
                    const int i = i0 + lane;
                    double gx = 0.0, gy = 0.0, gz = 0.0, lJ = 0.0;
                    for (int k = 1; 2 * k <= N; ++k) {
                        if (i < (2 * k == N ? k : N)) {
                            const int j = i + k < N ? i + k : i + k - N;
                            pair(i, j);
                            gx += g * x;
                            gy += g * y;
                            gz += g * z;
                            lJ += l;
                            oth[j] -= g * x;
                            oth[N + j] -= g * y;
                            oth[2 * N + j] -= g * z;
                            oth[3 * N + j] += l;
                            v[1] += u;
                            v[0] += ir;
                        }
                        __syncwarp();
                    }
                    if (i < N) {
                        part[4 * i] = gx;
                        part[4 * i + 1] = gy;
                        part[4 * i + 2] = gz;
                        part[4 * i + 3] = lJ;
                    }
                }
            } else {
                for (int i = tid; i < N; i += H) {
                    double gx = 0.0, gy = 0.0, gz = 0.0, lJ = 0.0;
                    for (int j = 0; j < N; ++j) {
                        if (j == i) continue;
                        pair(i, j);
                        gx += g * x;
                        gy += g * y;
                        gz += g * z;
                        lJ += l;
                        if (j > i) {
                            v[1] += u;
                            v[0] += ir;
                        }
                    }
                    part[4 * i] = gx;
                    part[4 * i + 1] = gy;
                    part[4 * i + 2] = gz;
                    part[4 * i + 3] = lJ;
                }
            }
        }
    }
    // ---- electron-nucleus terms and determinant (second half); the barrier
    // after the pair sums falls between these and the assembly of a thread's
    // first electron
    for (int i0 = 0; i0 < N; i0 += H) {
        const int i = i0 + tid - H;
        const bool on = tid >= H && i < N;
        double d0 = 0.0, d1 = 0.0, d2 = 0.0, dl = 0.0, gx = 0.0, gy = 0.0, gz = 0.0, lJ = 0.0;
        if (on) {
            if constexpr (sizeof(T) == 4) {
                const float* det = (const float*)(sm + L.other) + 8 * i;
                d0 = (double)det[0] + det[1];
                d1 = (double)det[2] + det[3];
                d2 = (double)det[4] + det[5];
                dl = (double)det[6] + det[7];
                const float b = (float)s.b_en;
                const float4 rh = sRf[i];
                const float rl[3] = {(float)(sR[3 * i] - (double)rh.x), (float)(sR[3 * i + 1] - (double)rh.y),
                                     (float)(sR[3 * i + 2] - (double)rh.z)};
                float fx = 0.f, fy = 0.f, fz = 0.f;
                Acc<float> lE, Ji, V;
                for (int a = 0; a < nn; ++a) {
                    const float x = diff_f2(rh.x, rl[0], s.Rn_hi[3 * a], s.Rn_lo[3 * a]);
                    const float y = diff_f2(rh.y, rl[1], s.Rn_hi[3 * a + 1], s.Rn_lo[3 * a + 1]);
                    const float z = diff_f2(rh.z, rl[2], s.Rn_hi[3 * a + 2], s.Rn_lo[3 * a + 2]);
                    const float r2 = x * x + y * y + z * z;
                    const float ir = rsqrtf(r2), r = r2 * ir;
                    const float ae = s.a_en_f[a];
                    const float q = 1.0f / (1.0f + b * r);
                    const float du = ae * q * q, g = du * ir;
                    fx += g * x;
                    fy += g * y;
                    fz += g * z;
                    lE.add(-2.0f * b * du * q + 2.0f * g);
                    Ji.add(ae * r * q);
                    V.add(-s.Z_f[a] * ir);
                    if (s.npp) V.add(pp_local<float>(s, a, r));
                }
                gx = fx;
                gy = fy;
                gz = fz;
                lJ = (double)lE.h + lE.l;
                v[0] += (double)V.h + V.l;
                v[1] += (double)Ji.h + Ji.l;
            } else {
                const int spin = i >= nu, n = spin ? s.n_dn : nu, k = spin ? i - nu : i;
                const double* Ai = (const double*)wk.Ainv[spin] + ((size_t)w * n + k) * n;
                const double* Gi = (const double*)wk.G[spin] + ((size_t)w * n + k) * 4 * n;
                for (int j = 0; j < n; ++j) {
                    const double a = Ai[j];
                    d0 += Gi[j] * a;
                    d1 += Gi[n + j] * a;
                    d2 += Gi[2 * n + j] * a;
                    dl += Gi[3 * n + j] * a;
                }
                const double b = s.b_en, xi = sR[3 * i], yi = sR[3 * i + 1], zi = sR[3 * i + 2];
                double Ji = 0.0, V = 0.0;
                for (int a = 0; a < nn; ++a) {
                    const double x = xi - s.Rn[3 * a], y = yi - s.Rn[3 * a + 1], z = zi - s.Rn[3 * a + 2];
                    const double r2 = x * x + y * y + z * z;
                    const double ir = rsqrt(r2), r = r2 * ir;
                    const double q = 1.0 / (1.0 + b * r);
                    const double aq = s.a_en[a] * q, du = aq * q, g = du * ir;
                    gx += g * x;
                    gy += g * y;
                    gz += g * z;
                    lJ += fma(-2.0 * b, du * q, 2.0 * g);
                    Ji += aq * r;
                    V -= s.Z[a] * ir;
                    if (s.npp) V += pp_local<double>(s, a, r);
                }
                v[0] += V;
                v[1] += Ji;
            }
            if (s.n3 > 0) {
                double v3, g3[3], l3;
                j3_electron(s, sR, i, v3, g3, l3);
                gx += g3[0];
                gy += g3[1];
                gz += g3[2];
                lJ += l3;
                v[1] += v3;
            }
        }
        if (i0 == 0) __syncthreads();   // part and other are complete
        if (on) {
            constexpr int kP = sizeof(T) == 4 ? 5 : 4;
            gx += (double)part[kP * i];
            gy += (double)part[kP * i + 1];
            gz += (double)part[kP * i + 2];
            lJ += (double)part[kP * i + 3];
            if (sizeof(T) == 4) lJ += (double)part[kP * i + kP - 1];
            if (sizeof(T) == 8 && N <= kElocSym)
                for (int q = 0; q < H / 32; ++q) {
                    const double* oth = (const double*)(sm + L.other) + (size_t)q * 4 * N;
                    gx += oth[i];
                    gy += oth[N + i];
                    gz += oth[2 * N + i];
                    lJ += oth[3 * N + i];
                }
            v[0] -= 0.5 * (dl + lJ + 2.0 * (gx * d0 + gy * d1 + gz * d2) + gx * gx + gy * gy + gz * gz);
            if (grad) {
                double* g = grad + ((size_t)w * N + i) * 3;
                g[0] = gx + d0;
                g[1] = gy + d1;
                g[2] = gz + d2;
            }
            if (lap) lap[(size_t)w * N + i] = lJ + dl - (d0 * d0 + d1 * d1 + d2 * d2);
        }
    }
    block_sum<2>(v, scratch);
    if (threadIdx.x == 0) {
        const double el = v[0] + s.vnn;
        eloc_out[w] = el;
        if (logpsi) logpsi[w] = v[1] + wk.logdet[2 * w] + wk.logdet[2 * w + 1];
        if (!isfinite(el) && err) atomicOr(err, kErrNonFinite);
    }
}

constexpr int kElocThreads = 640;   // at most
template <typename T>
__global__ void __launch_bounds__(kElocThreads) k_eloc(DevSys s, DevWalkers wk, int W, double* eloc_out, double* logpsi,
                                                       double* grad, double* lap, unsigned* err) {
    extern __shared__ __align__(16) unsigned char esm[];
    const int w = blockIdx.x;
    if (w >= W) return;
    eloc_walker<T>(s, wk, w, eloc_out, logpsi, grad, lap, err, esm);
}

// Jastrow parameter derivatives of walker w (one CTA): d ln|psi| / dp is
// the derivative of J alone, B_p = dJ/dp, and dE_L / dp = -1/2 sum_i
// (lap_i B_p + 2 grad_i ln|psi| . grad_i B_p) (the determinant and the
// potential do not depend on the Jastrow).  Linear parameters give B_p as
// their own term with unit coefficient; for b of u = a r / (1 + b r),
// dB/db = -a r^2 / (1 + b r)^2 with radial derivatives -2 a r / (1 + b r)^3
// and -2 a (1 - 2 b r) / (1 + b r)^4.
__global__ void k_jastrow_derivs(DevSys s, const double* __restrict__ R, const double* __restrict__ G, int W,
                                 double* dlog, double* deloc) {
    extern __shared__ double jsm[];   // positions [3N], gradients [3N], per-nucleus b_en parts [2 n_nuc]
    __shared__ double scratch[kMaxWarps * 8];
    const int w = blockIdx.x;
    if (w >= W) return;
    const int N = s.N, nu = s.n_up, nn = s.n_nuc, P = 4 + nn + nn * s.n3;
    double* sR = jsm;
    double* sG = sR + 3 * N;
    double* bpart = sG + 3 * N;
    for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) {
        sR[q] = R[(size_t)w * 3 * N + q];
        sG[q] = G[(size_t)w * 3 * N + q];
    }
    __syncthreads();
    double* out_l = dlog + (size_t)w * P;
    double* out_e = deloc + (size_t)w * P;
    // electron pairs: a_anti, a_par, b_ee
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = wid; i < N; i += nw)
        for (int j = i + 1 + lane; j < N; j += 32) {
            double x[3], r2 = 0.0;
            for (int c = 0; c < 3; ++c) {
                x[c] = sR[3 * i + c] - sR[3 * j + c];
                r2 += x[c] * x[c];
            }
            const double ir = rsqrt(r2), r = r2 * ir;
            const bool like = (i < nu) == (j < nu);
            const double a = like ? s.a_par : s.a_anti, b = s.b_ee;
            const double q = 1.0 / (1.0 + b * r);
            double gdot = 0.0;   // (G_i - G_j) . u
            for (int c = 0; c < 3; ++c) gdot += (sG[3 * i + c] - sG[3 * j + c]) * x[c] * ir;
            // linear: B = r q, B' = q^2, B'' = -2 b q^3
            const double B = r * q, B1 = q * q, B2 = -2.0 * b * q * q * q;
            const double dEa = -0.5 * (2.0 * (B2 + 2.0 * B1 * ir) + 2.0 * B1 * gdot);
            acc[like ? 2 : 0] += B;
            acc[like ? 3 : 1] += dEa;
            // b_ee
            const double g = -a * r * r * q * q, g1 = -2.0 * a * r * q * q * q, g2 = -2.0 * a * (1.0 - 2.0 * b * r) * q * q * q * q;
            acc[4] += g;
            acc[5] += -0.5 * (2.0 * (g2 + 2.0 * g1 * ir) + 2.0 * g1 * gdot);
        }
    // electron-nucleus: a_en[a] (direct), b_en (per nucleus, summed below)
    for (int a = threadIdx.x; a < nn; a += blockDim.x) {
        double Bl = 0.0, Be = 0.0, bl = 0.0, be = 0.0;
        const double ae = s.a_en[a], b = s.b_en;
        for (int i = 0; i < N; ++i) {
            double x[3], r2 = 0.0;
            for (int c = 0; c < 3; ++c) {
                x[c] = sR[3 * i + c] - s.Rn[3 * a + c];
                r2 += x[c] * x[c];
            }
            const double ir = rsqrt(r2), r = r2 * ir;
            const double q = 1.0 / (1.0 + b * r);
            double gdot = 0.0;
            for (int c = 0; c < 3; ++c) gdot += sG[3 * i + c] * x[c] * ir;
            const double B = r * q, B1 = q * q, B2 = -2.0 * b * q * q * q;
            Bl += B;
            Be += -0.5 * ((B2 + 2.0 * B1 * ir) + 2.0 * B1 * gdot);
            const double g = -ae * r * r * q * q, g1 = -2.0 * ae * r * q * q * q,
                         g2 = -2.0 * ae * (1.0 - 2.0 * b * r) * q * q * q * q;
            bl += g;
            be += -0.5 * ((g2 + 2.0 * g1 * ir) + 2.0 * g1 * gdot);
        }
        out_l[4 + a] = Bl;
        out_e[4 + a] = Be;
        bpart[2 * a] = bl;
        bpart[2 * a + 1] = be;
    }
    // three-body terms: one thread per (nucleus, term), pairs in a fixed order
    for (int pk = threadIdx.x; pk < nn * s.n3; pk += blockDim.x) {
        const int a = pk / s.n3, k = pk - a * s.n3;
        const int m = s.e3[3 * k], n = s.e3[3 * k + 1], o = s.e3[3 * k + 2];
        const double* ra = s.Rn + 3 * a;
        double Bv = 0.0, Bt = 0.0;
        for (int i = 0; i < N; ++i) {
            const double* ri = sR + 3 * i;
            const SDist xi = sdist(s.b3, ri[0] - ra[0], ri[1] - ra[1], ri[2] - ra[2]);
            for (int j = 0; j < N; ++j) {
                if (j == i) continue;
                const double* rj = sR + 3 * j;
                const SDist xj = sdist(s.b3, rj[0] - ra[0], rj[1] - ra[1], rj[2] - ra[2]);
                const SDist y = sdist(s.b3, ri[0] - rj[0], ri[1] - rj[1], ri[2] - rj[2]);
                double v, g[3], l;
                j3_term(m, n, o, xi, xj, y, v, g, l);
                if (j > i) Bv += v;
                Bt += l + 2.0 * (sG[3 * i] * g[0] + sG[3 * i + 1] * g[1] + sG[3 * i + 2] * g[2]);
            }
        }
        out_l[4 + nn + pk] = Bv;
        out_e[4 + nn + pk] = -0.5 * Bt;
    }
    block_sum<6>(*reinterpret_cast<double(*)[6]>(acc), scratch);
    if (threadIdx.x == 0) {
        double bl = 0.0, be = 0.0;
        for (int a = 0; a < nn; ++a) {
            bl += bpart[2 * a];
            be += bpart[2 * a + 1];
        }
        out_l[0] = acc[0];
        out_e[0] = acc[1];
        out_l[1] = acc[2];
        out_e[1] = acc[3];
        out_l[2] = acc[4];
        out_e[2] = acc[5];
        out_l[3] = bl;
        out_e[3] = be;
    }
}

cudaError_t launch_jastrow_derivs(const DevSys& s, const double* R, const double* G, int W, double* dlog,
                                  double* deloc, cudaStream_t st) {
    if (W == 0) return cudaSuccess;
    const size_t smem = sizeof(double) * (6 * (size_t)s.N + 2 * (size_t)s.n_nuc);
    if (const cudaError_t e = allow_smem(k_jastrow_derivs, smem)) return e;
    k_jastrow_derivs<<<W, 256, smem, st>>>(s, R, G, W, dlog, deloc);
    return cudaGetLastError();
}

// out[k] (+)= sum_w g[w] x[w][k]  (g == nullptr: plain sum).  One CTA per
// k, threads over walkers, deterministic order.
__global__ void k_weighted_sum(const double* x, const double* g, int W, int K, double* out, int accumulate) {
    __shared__ double scratch[kMaxWarps];
    const int k = blockIdx.x;
    double v[1] = {0.0};
    for (int w = threadIdx.x; w < W; w += blockDim.x) v[0] += (g ? g[w] : 1.0) * x[(size_t)w * K + k];
    block_sum<1>(v, scratch);
    if (threadIdx.x == 0) out[k] = (accumulate ? out[k] : 0.0) + v[0];
}

size_t orbitals_smem_bytes(const DevSys& s) {
    return orbitals_fx(s) ? Basis64Layout(s.n_nuc, s.n_prim, s.n_shell, s.n_basis).total
                          : sizeof(double) * 5 * (size_t)s.n_basis;
}

// The matrix and its column; with fx also the basis at a point (orbitals_again).
size_t invert_smem_bytes(const DevSys& s, bool fx) {
    const int nmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    const size_t m = sizeof(double) * ((size_t)nmax * nmax + nmax + 1);
    return fx && orbitals_fx(s) ? std::max(m, sizeof(double) * 5 * (size_t)s.n_basis + s.n_shell) : m;
}

template <typename T>
cudaError_t launch_orbitals_all(const DevSys& s, const DevWalkers& wk, int W, cudaStream_t st, const int* only,
                                bool sums) {
    if (W == 0 || s.N == 0) return cudaSuccess;
    if (sums || !orbitals_fx(s)) {
        const size_t smem = sizeof(double) * 5 * s.n_basis + (size_t)s.n_shell;
        if (const cudaError_t e = allow_smem(k_orbitals_sums<T>, smem)) return e;
        k_orbitals_sums<T><<<dim3(W, s.N), s.n_up > 32 ? 256 : 128, smem, st>>>(s, wk, W, only);
        return cudaGetLastError();
    }
    const size_t smem = orbitals_smem_bytes(s);
    const int nmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    // a thread per orbital; few orbitals share their rows among lanes anyway, and
    // two warps per electron leave room for twice the electrons.  Evaluation with
    // 128 -> 64 threads: one water, 512 and 4096 walkers 0.20 -> 0.17 and 0.92 ->
    // 0.71 ms; 3 waters, 77, 1024 and 4096 walkers 0.18 -> 0.16, 0.78 -> 0.60 and
    // 2.76 -> 2.09 ms.  (At 20 orbitals 64 are ahead as well, 2.32 -> 1.88 ms for
    // 2048 walkers: the line could lie higher.)
    const int nt = nmax > 128 ? (nmax > 256 ? 256 : (nmax + 31) & ~31) : nmax > 16 ? 128 : 64;
    if (const cudaError_t e = allow_smem(k_orbitals_all<T>, smem)) return e;
    k_orbitals_all<T><<<dim3(W, s.N), nt, smem, st>>>(s, wk, W, only);
    return cudaGetLastError();
}

cudaError_t launch_invert(const DevSys& s, const DevWalkers& wk, int W, int store_fp32, int* shrt, unsigned* err,
                          cudaStream_t st, const int* only) {
    if (W == 0) return cudaSuccess;
    if (!orbitals_fx(s)) shrt = nullptr;
    const int nmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    const size_t smem = invert_smem_bytes(s, false), smem_again = invert_smem_bytes(s, true);
    if (const cudaError_t e = allow_smem(k_invert, smem)) return e;
    const int nt = nmax > 64 ? 512 : (nmax > 16 ? 256 : 128);
    k_invert<<<dim3(W, 2), nt, smem, st>>>(s, wk, W, store_fp32, shrt, err, only);
    if (!shrt) return cudaGetLastError();
    if (const cudaError_t e = cudaGetLastError()) return e;
    if (const cudaError_t e = allow_smem(k_invert_again, smem_again)) return e;
    k_invert_again<<<dim3(W, 2), nt, smem_again, st>>>(s, wk, W, store_fp32, shrt, err, only);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_eloc(const DevSys& s, const DevWalkers& wk, int W, double* eloc_out, double* logpsi,
                        double* grad, double* lap, unsigned* err, cudaStream_t st) {
    if (W == 0) return cudaSuccess;
    const int nt = std::min(kElocThreads, 2 * ((s.N + 31) & ~31));
    const size_t smem = eloc_smem_bytes(s, nt, sizeof(T));
    if (const cudaError_t e = allow_smem(k_eloc<T>, smem)) return e;
    k_eloc<T><<<W, nt, smem, st>>>(s, wk, W, eloc_out, logpsi, grad, lap, err);
    return cudaGetLastError();
}

cudaError_t launch_weighted_sum(const double* x, const double* g, int W, int K, double* out, int accumulate,
                                cudaStream_t st) {
    if (K == 0) return cudaSuccess;
    k_weighted_sum<<<K, 256, 0, st>>>(x, g, W, K, out, accumulate);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------
// Batched forms: persistent CTAs over the items of every system.
// ---------------------------------------------------------------------
template <typename T>
__global__ void k_orbitals_batch(const BatchSys* __restrict__ sys, BatchPlan* plan, int parity, int ctr) {
    extern __shared__ double sh_bas[];
    __shared__ BatchSys bs;
    __shared__ int s_sys, s_idx;
    for (;;) {
        if (threadIdx.x == 0) batch_next(plan, kUnitElectron, ctr, &s_sys, &s_idx);
        __syncthreads();
        const int q = s_sys;
        if (q < 0) break;
        batch_load(&bs, sys + q);
        __syncthreads();
        const int N = bs.s.N;
        orbitals_item<T>(bs.s, bs.wk[parity], s_idx / N, s_idx % N, (unsigned char*)sh_bas);
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256, 5) k_invert_batch(const BatchSys* __restrict__ sys, BatchPlan* plan, int parity, int store_fp32,
                               int ctr) {
    extern __shared__ double M[];
    __shared__ BatchSys bs;
    __shared__ int s_sys, s_idx;
    for (;;) {
        if (threadIdx.x == 0) batch_next(plan, kUnitSpin, ctr, &s_sys, &s_idx);
        __syncthreads();
        const int q = s_sys;
        if (q < 0) break;
        batch_load(&bs, sys + q);
        __syncthreads();
        invert_item<true>(bs.s, bs.wk[parity], s_idx >> 1, s_idx & 1, store_fp32, orbitals_fx(bs.s), 0, nullptr, bs.err,
                          M);
        __syncthreads();
    }
}

template <typename T>
__global__ void k_eloc_batch(const BatchSys* __restrict__ sys, BatchPlan* plan, int parity, int into_walker, int ctr) {
    extern __shared__ __align__(16) unsigned char esm[];
    __shared__ BatchSys bs;
    __shared__ int s_sys, s_idx;
    for (;;) {
        if (threadIdx.x == 0) batch_next(plan, kUnitWalker, ctr, &s_sys, &s_idx);
        __syncthreads();
        const int q = s_sys;
        if (q < 0) break;
        batch_load(&bs, sys + q);
        __syncthreads();
        eloc_walker<T>(bs.s, bs.wk[parity], s_idx, into_walker ? bs.wk[parity].eloc : bs.eloc_new, nullptr, nullptr,
                       nullptr, bs.err, esm);
        __syncthreads();
    }
}

template <typename T>
cudaError_t launch_orbitals_batch(const BatchSys* sys, BatchPlan* plan, int parity, int ctr, int grid, size_t smem,
                                  cudaStream_t st) {
    k_orbitals_batch<T><<<grid, 128, smem, st>>>(sys, plan, parity, ctr);
    return cudaGetLastError();
}

cudaError_t launch_invert_batch(const BatchSys* sys, BatchPlan* plan, int parity, int store_fp32, int ctr, int grid,
                                size_t smem, cudaStream_t st) {
    k_invert_batch<<<grid, 256, smem, st>>>(sys, plan, parity, store_fp32, ctr);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_eloc_batch(const BatchSys* sys, BatchPlan* plan, int parity, int into_walker, int ctr, int grid,
                              size_t smem, cudaStream_t st) {
    k_eloc_batch<T><<<grid, 128, smem, st>>>(sys, plan, parity, into_walker, ctr);
    return cudaGetLastError();
}

// Sets the dynamic shared memory limit of a batched family (0 orbitals,
// 1 inversion, 2 local energy; 3 and 4: the FP32-storage forms of 0 and 2)
// before any launch or graph capture; returns its resident CTAs per SM.
int wf_batch_prepare(int family, int block, size_t smem) {
    int nb = 0;
    const void* f = nullptr;
    switch (family) {
        case 0: f = (const void*)k_orbitals_batch<double>; break;
        case 1: f = (const void*)k_invert_batch; break;
        case 2: f = (const void*)k_eloc_batch<double>; break;
        case 3: f = (const void*)k_orbitals_batch<float>; break;
        case 4: f = (const void*)k_eloc_batch<float>; break;
        default: return 0;
    }
    if (allow_smem(f, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, block, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

template cudaError_t launch_orbitals_batch<double>(const BatchSys*, BatchPlan*, int, int, int, size_t, cudaStream_t);
template cudaError_t launch_orbitals_batch<float>(const BatchSys*, BatchPlan*, int, int, int, size_t, cudaStream_t);
template cudaError_t launch_eloc_batch<double>(const BatchSys*, BatchPlan*, int, int, int, int, size_t,
                                               cudaStream_t);
template cudaError_t launch_eloc_batch<float>(const BatchSys*, BatchPlan*, int, int, int, int, size_t, cudaStream_t);

template cudaError_t launch_orbitals_all<double>(const DevSys&, const DevWalkers&, int, cudaStream_t, const int*, bool);
template cudaError_t launch_orbitals_all<float>(const DevSys&, const DevWalkers&, int, cudaStream_t, const int*, bool);
template cudaError_t launch_eloc<double>(const DevSys&, const DevWalkers&, int, double*, double*, double*,
                                         double*, unsigned*, cudaStream_t);
template cudaError_t launch_eloc<float>(const DevSys&, const DevWalkers&, int, double*, double*, double*,
                                        double*, unsigned*, cudaStream_t);

}  // namespace qmc
