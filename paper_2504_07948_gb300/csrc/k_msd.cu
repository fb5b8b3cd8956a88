// Multi-determinant expansions by the table method (Sec. "Multideterminant
// QMC Forces": excited determinants from small determinants of a table,
// determinants grouped by excitation level).
//
// With the reference Slater matrix A0 (n x n) of a spin and the values of
// the active virtual orbitals at the same electrons, A_v (n x n_vir), the
// table T = A0^-1 A_v gives every excited determinant of that spin as
//   D_u / D_0 = phase_u det(T[H_u, P_u])          (e_u <= 4 rows/columns),
// H_u the replaced reference positions, P_u the replacing virtuals, and
// phase_u the sign of sorting the replaced orbital list.  The expansion is
//   psi_D / (D0_up D0_dn) = S = sum_k c_k R_up[u(k)] R_dn[d(k)].
// For any operator B applied to the orbital matrix one electron row at a
// time (a derivative in that electron's coordinates), the change of ln D_u
// relative to ln D_0 is tr(M^-1 Theta[H,P]) with M = T[H,P] and
//   Theta = A0^-1 (B_v - B_0 T),
// i.e. the first-order change of det(M) along Theta; used here for the
// kinetic operator of the local energy and for electron gradients.
#include "msd_small.cuh"
#include "qmc_internal.cuh"

namespace qmc {

template <typename F>
__device__ __forceinline__ F det_small(int e, const F m[4][4]) {
    switch (e) {
        case 0:
            return F(1);
        case 1:
            return m[0][0];
        case 2:
            return m[0][0] * m[1][1] - m[0][1] * m[1][0];
        case 3:
            return m[0][0] * (m[1][1] * m[2][2] - m[1][2] * m[2][1]) - m[0][1] * (m[1][0] * m[2][2] - m[1][2] * m[2][0]) +
                   m[0][2] * (m[1][0] * m[2][1] - m[1][1] * m[2][0]);
        default: {
            // Laplace expansion along the first two rows (2x2 minors)
            const F a01 = m[0][0] * m[1][1] - m[0][1] * m[1][0], a02 = m[0][0] * m[1][2] - m[0][2] * m[1][0];
            const F a03 = m[0][0] * m[1][3] - m[0][3] * m[1][0], a12 = m[0][1] * m[1][2] - m[0][2] * m[1][1];
            const F a13 = m[0][1] * m[1][3] - m[0][3] * m[1][1], a23 = m[0][2] * m[1][3] - m[0][3] * m[1][2];
            const F b01 = m[2][0] * m[3][1] - m[2][1] * m[3][0], b02 = m[2][0] * m[3][2] - m[2][2] * m[3][0];
            const F b03 = m[2][0] * m[3][3] - m[2][3] * m[3][0], b12 = m[2][1] * m[3][2] - m[2][2] * m[3][1];
            const F b13 = m[2][1] * m[3][3] - m[2][3] * m[3][1], b23 = m[2][2] * m[3][3] - m[2][3] * m[3][2];
            return a01 * b23 - a02 * b13 + a03 * b12 + a12 * b03 - a13 * b02 + a23 * b01;
        }
    }
}

struct StrDesc {
    int e;
    float phase;
    int h[4], p[4];
};

__device__ __forceinline__ StrDesc decode(int4 v) {
    StrDesc d;
    d.e = v.x & 0xff;
    d.phase = ((v.x >> 8) & 1) ? -1.f : 1.f;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        d.h[a] = (v.y >> (8 * a)) & 0xff;
        d.p[a] = (v.z >> (8 * a)) & 0xff;
    }
    return d;
}

// M = T[H,P] from a row-major table with leading dimension ld.
template <typename F, typename TT>
__device__ __forceinline__ void gather_minor(const StrDesc& d, const TT* T, int ld, F m[4][4]) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) m[a][b] = (a < d.e && b < d.e) ? F(T[d.h[a] * ld + d.p[b]]) : F(0);
}

// det(M with column b replaced by the vector u), b = 0..e-1.
template <typename F>
__device__ __forceinline__ void col_replaced_dets(int e, const F m[4][4], const F u[4], F out[4]) {
    for (int b = 0; b < 4; ++b) {
        if (b >= e) {
            out[b] = F(0);
            continue;
        }
        F t[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) t[a][c] = (c == b) ? u[a] : m[a][c];
        out[b] = det_small<F>(e, t);
    }
}

// Table, string ratios, CI partial sums and S for every walker (after an
// FP64 recompute of the reference inverse and the virtual orbital values).
template <typename T>
__global__ void k_msd_table(DevSys s, DevWalkers wk, int W, const int* only) {
    __shared__ double scratch[kMaxWarps];
    const int w = blockIdx.x;
    if (w >= W || (only && !only[w])) return;
    for (int spin = 0; spin < 2; ++spin) {
        const int n = spin ? s.n_dn : s.n_up, nv = s.n_vir[spin];
        const T* AT = (const T*)wk.Ainv[spin] + (size_t)w * n * n;
        const T* Av = (const T*)wk.Av[spin] + (size_t)w * n * nv;
        T* Tt = (T*)wk.Tt[spin] + (size_t)w * n * nv;
        for (int q = threadIdx.x; q < n * nv; q += blockDim.x) {
            const int h = q / nv, p = q - h * nv;
            T acc = T(0);
            for (int i = 0; i < n; ++i) acc += AT[(size_t)i * n + h] * Av[(size_t)i * nv + p];
            Tt[q] = acc;
        }
        __syncthreads();
        T* R = (T*)wk.Rs[spin] + (size_t)w * s.n_str[spin];
        for (int u = threadIdx.x; u < s.n_str[spin]; u += blockDim.x) {
            const StrDesc d = decode(s.str[spin][u]);
            T m[4][4];
            gather_minor<T>(d, Tt, nv, m);
            R[u] = T(d.phase) * det_small<T>(d.e, m);
        }
        __syncthreads();
    }
    for (int spin = 0; spin < 2; ++spin) {
        const T* Ro = (const T*)wk.Rs[1 - spin] + (size_t)w * s.n_str[1 - spin];
        T* Cd = (T*)wk.Cd[spin] + (size_t)w * s.n_str[spin];
        for (int u = threadIdx.x; u < s.n_str[spin]; u += blockDim.x) {
            double acc = 0.0;
            for (int q = s.csr_off[spin][u]; q < s.csr_off[spin][u + 1]; ++q)
                acc += s.csr_c[spin][q] * (double)Ro[s.csr_other[spin][q]];
            Cd[u] = (T)acc;
        }
    }
    __syncthreads();
    double v[1] = {0.0};
    const T* R0 = (const T*)wk.Rs[0] + (size_t)w * s.n_str[0];
    const T* C0 = (const T*)wk.Cd[0] + (size_t)w * s.n_str[0];
    for (int u = threadIdx.x; u < s.n_str[0]; u += blockDim.x) v[0] += (double)R0[u] * (double)C0[u];
    block_sum<1>(v, scratch);
    if (threadIdx.x == 0) wk.Ssum[w] = v[0];
}

// Doubles of the tile in which k_msd_eloc forms rows of B_0 and A0^-1 (at least
// one row) and the parts of grad J (as many as fit).
constexpr int kElocTile = 1024;

// Bound by its FP64 instructions: B_0 and the FP64 forms of T and A0^-1 are made
// once instead of for every virtual, and grad J is shared by the whole CTA
// (10,000 determinants, 256 walkers: 485 -> 294 us).
// Adds the multi-determinant part to E_L, ln|psi|, the sign and (when grad
// is given) the electron gradients of ln|psi| computed for the reference
// determinant by k_eloc.
template <typename T>
__global__ void k_msd_eloc(DevSys s, DevWalkers wk, int W, double* eloc, double* logpsi, double* sign,
                           double* grad, int n_tile) {
    extern __shared__ double sm[];
    __shared__ double scratch[kMaxWarps * 4];
    const int w = blockIdx.x;
    if (w >= W) return;
    const int N = s.N, nu = s.n_up, nn = s.n_nuc;
    const int nmax = nu > s.n_dn ? nu : s.n_dn;
    const int nvmax = s.n_vir[0] > s.n_vir[1] ? s.n_vir[0] : s.n_vir[1];
    double* sR = sm;
    double* gJ = sR + 3 * N;
    double* Q = gJ + 3 * N;              // [nmax][nvmax]
    double* Th = Q + nmax * nvmax;       // [nmax][nvmax]
    double* Wg = Th + nmax * nvmax;      // [3][nvmax]
    double* tile = Wg;                   // [n_tile], before the gradients
    for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) sR[q] = wk.R[(size_t)w * 3 * N + q];
    __syncthreads();
    // grad J: parts of the CTA take every np-th partner of all electrons
    const int nr = (N + 31) & ~31;
    int np = nr < (int)blockDim.x ? (int)blockDim.x / nr : 1;
    if (np * 3 * N > n_tile) np = 1;
    for (int q = threadIdx.x; q < np * nr; q += blockDim.x) {
        const int part = q / nr, i = q - part * nr;
        if (i >= N) continue;
        double g[3] = {0, 0, 0};
        for (int j = part; j < N + nn; j += np) {
            double x[3], a, b;
            if (j < N) {
                if (j == i) continue;
                for (int c = 0; c < 3; ++c) x[c] = sR[3 * i + c] - sR[3 * j + c];
                a = ((i < nu) == (j < nu)) ? s.a_par : s.a_anti;
                b = s.b_ee;
            } else {
                for (int c = 0; c < 3; ++c) x[c] = sR[3 * i + c] - s.Rn[3 * (j - N) + c];
                a = s.a_en[j - N];
                b = s.b_en;
            }
            const double r2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
            const double ir = rsqrt(r2);
            const double qd = 1.0 / (1.0 + b * r2 * ir);
            const double gr = a * qd * qd * ir;
            for (int c = 0; c < 3; ++c) g[c] += gr * x[c];
        }
        double* out = np > 1 ? tile + 3 * N * part : gJ;
        for (int c = 0; c < 3; ++c) out[3 * i + c] = g[c];
    }
    __syncthreads();
    if (np > 1) {
        for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) {
            double v = tile[q];
            for (int c = 1; c < np; ++c) v += tile[3 * N * c + q];
            gJ[q] = v;
        }
        __syncthreads();
    }
    const double S = wk.Ssum[w];
    // per string: tr(adj(M) Theta[H,P]) with the cofactors of the table minor
    // in the storage type and the contraction with Theta in FP64
    Acc<double> sd[1];
    for (int spin = 0; spin < 2; ++spin) {
        const int n = spin ? s.n_dn : nu, nv = s.n_vir[spin], i0 = spin ? nu : 0;
        if (n == 0) continue;
        const T* AT = (const T*)wk.Ainv[spin] + (size_t)w * n * n;
        const T* G = (const T*)wk.G[spin] + (size_t)w * 4 * n * n;
        const T* Gv = (const T*)wk.Gv[spin] + (size_t)w * 4 * n * nv;
        const T* Tt = (const T*)wk.Tt[spin] + (size_t)w * n * nv;
        // Q = B_v - B_0 T with B = -1/2 lap phi - grad J . grad phi per row;
        // B_0 by tiles of rows, T in FP64 (in Theta's place), both formed once
        const int rows = max(1, n_tile / n);
        for (int q = threadIdx.x; q < n * nv; q += blockDim.x) Th[q / nv * nvmax + q % nv] = (double)Tt[q];
        for (int r0 = 0; r0 < n; r0 += rows) {
            const int nr0 = min(rows, n - r0);
            __syncthreads();
            for (int q = threadIdx.x; q < nr0 * n; q += blockDim.x) {
                const int i = r0 + q / n, j = q % n;
                const double* gj = gJ + 3 * (i0 + i);
                const T* Gi = G + (size_t)i * 4 * n;
                tile[q] = -0.5 * (double)Gi[3 * n + j] - gj[0] * (double)Gi[j] - gj[1] * (double)Gi[n + j] -
                          gj[2] * (double)Gi[2 * n + j];
            }
            __syncthreads();
            for (int q = threadIdx.x; q < nr0 * nv; q += blockDim.x) {
                const int r = q / nv, i = r0 + r, p = q - r * nv;
                const double* gj = gJ + 3 * (i0 + i);
                const T* Gvi = Gv + (size_t)i * 4 * nv;
                double acc = -0.5 * (double)Gvi[3 * nv + p] - gj[0] * (double)Gvi[p] - gj[1] * (double)Gvi[nv + p] -
                             gj[2] * (double)Gvi[2 * nv + p];
                for (int j = 0; j < n; ++j) acc -= tile[r * n + j] * Th[j * nvmax + p];
                Q[i * nvmax + p] = acc;
            }
        }
        // Theta = A0^-1 Q, by tiles of rows of A0^-1
        for (int r0 = 0; r0 < n; r0 += rows) {
            const int nr0 = min(rows, n - r0);
            __syncthreads();
            for (int q = threadIdx.x; q < nr0 * n; q += blockDim.x) {
                const int i = q / nr0, r = q - i * nr0;
                tile[r * n + i] = (double)AT[(size_t)i * n + r0 + r];
            }
            __syncthreads();
            for (int q = threadIdx.x; q < nr0 * nv; q += blockDim.x) {
                const int r = q / nv, p = q - r * nv;
                double acc = 0.0;
                for (int i = 0; i < n; ++i) acc += tile[r * n + i] * Q[i * nvmax + p];
                Th[(r0 + r) * nvmax + p] = acc;
            }
        }
        __syncthreads();
        const T* Cd = (const T*)wk.Cd[spin] + (size_t)w * s.n_str[spin];
        for (int u = threadIdx.x; u < s.n_str[spin]; u += blockDim.x) {
            const StrDesc d = decode(s.str[spin][u]);
            if (d.e == 0) continue;
            T m[4][4], cof[4][4];
            gather_minor<T>(d, Tt, nv, m);
            cofactors<T>(d.e, m, cof);
            double tr = 0.0;
            for (int a = 0; a < d.e; ++a)
                for (int c = 0; c < d.e; ++c) tr += (double)cof[a][c] * Th[d.h[a] * nvmax + d.p[c]];
            sd[0].add((double)d.phase * tr * (double)Cd[u]);
        }
        __syncthreads();
    }
    double sdd[1];
    block_sum_to0<1>(sd, scratch, sdd);
    if (threadIdx.x == 0) {
        eloc[w] += sdd[0] / S;
        if (logpsi) logpsi[w] += log(fabs(S));
        if (sign) sign[w] = wk.sgn[2 * w] * wk.sgn[2 * w + 1] * (S < 0.0 ? -1.0 : 1.0);
    }
    if (!grad) return;
    // electron gradients: d_i S / S = sum_u Cd_u phase_u sum_b W_i[p_b] det(M with column b <- A0^-1[H, i])
    for (int i = 0; i < N; ++i) {
        const int spin = i >= nu;
        const int n = spin ? s.n_dn : nu, nv = s.n_vir[spin], k = spin ? i - nu : i;
        const T* AT = (const T*)wk.Ainv[spin] + (size_t)w * n * n;
        const T* Gk = (const T*)wk.G[spin] + ((size_t)w * n + k) * 4 * n;
        const T* Gvk = (const T*)wk.Gv[spin] + ((size_t)w * n + k) * 4 * nv;
        const T* Tt = (const T*)wk.Tt[spin] + (size_t)w * n * nv;
        __syncthreads();
        for (int q = threadIdx.x; q < 3 * nv; q += blockDim.x) {
            const int c = q / nv, p = q - c * nv;
            double acc = (double)Gvk[c * nv + p];
            for (int j = 0; j < n; ++j) acc -= (double)Gk[c * n + j] * (double)Tt[(size_t)j * nv + p];
            Wg[c * nvmax + p] = acc;
        }
        __syncthreads();
        const T* Cd = (const T*)wk.Cd[spin] + (size_t)w * s.n_str[spin];
        Acc<T> g[3];
        for (int u = threadIdx.x; u < s.n_str[spin]; u += blockDim.x) {
            const StrDesc d = decode(s.str[spin][u]);
            if (d.e == 0) continue;
            T m[4][4], uh[4], gb[4];
            gather_minor<T>(d, Tt, nv, m);
            for (int a = 0; a < 4; ++a) uh[a] = a < d.e ? AT[(size_t)k * n + d.h[a]] : T(0);
            col_replaced_dets<T>(d.e, m, uh, gb);
            const T f = T(d.phase) * Cd[u];
            for (int b = 0; b < d.e; ++b)
                for (int c = 0; c < 3; ++c) g[c].add(f * T(Wg[c * nvmax + d.p[b]]) * gb[b]);
        }
        double gd[3];
        block_sum_to0<3>(g, scratch, gd);
        if (threadIdx.x == 0)
            for (int c = 0; c < 3; ++c) grad[((size_t)w * N + i) * 3 + c] += gd[c] / S;
    }
}


// ---------------------------------------------------------------------
// Particle-by-particle sweep of a multi-determinant wavefunction.
//
// On top of the reference-determinant move of k_sweep, a move of electron
// e (spin s) updates the table by a rank-1 term,
//   T' = T + c w^T / rho0,  c = A0^-1[:, e],  w = phi'_v - T^T phi'_occ,
// (no old orbital row is needed), evaluates every string ratio of spin s
// from T'[H,P], and S' = sum_u Cd_u R'_u with Cd_u = sum over the string's
// determinants of c_k R_other (fixed while spin s moves).  The wavefunction
// ratio is rho0 S'/S e^{dJ}.  Drifts add d_e S / S, the derivative of every
// string determinant along the rank-1 change of row e.
// ---------------------------------------------------------------------
template <typename T>
__host__ __device__ inline size_t msd_sweep_smem(int N, int nb, int nu, int nd, int nv0, int nv1) {
    const int nmax = nu > nd ? nu : nd, nvmax = nv0 > nv1 ? nv0 : nv1;
    size_t o = sizeof(double) * (3 * (size_t)N + kMaxWarps * 12 + 16);
    o += sizeof(T) * (5 * (size_t)nb + 5 * (size_t)nmax + 5 * (size_t)nvmax + nmax + nvmax + 3 * (size_t)nvmax);
    o += sizeof(T) * ((size_t)nu * nu + (size_t)nd * nd + (size_t)nu * nv0 + (size_t)nd * nv1);
    return o;
}

template <typename T>
__device__ __forceinline__ void refresh_cd(const DevSys& s, const DevWalkers& wk, int w, int spin) {
    const T* Ro = (const T*)wk.Rs[1 - spin] + (size_t)w * s.n_str[1 - spin];
    T* Cd = (T*)wk.Cd[spin] + (size_t)w * s.n_str[spin];
    for (int u = threadIdx.x; u < s.n_str[spin]; u += blockDim.x) {
        double acc = 0.0;
        for (int q = s.csr_off[spin][u]; q < s.csr_off[spin][u + 1]; ++q)
            acc += s.csr_c[spin][q] * (double)Ro[s.csr_other[spin][q]];
        Cd[u] = (T)acc;
    }
}

// Arithmetic of the sweep's strings.  Every rounding is written out: a sweep of
// the mixed form is a chaotic map, and its trajectories should not depend on how
// the compiler contracts products and sums in one or the other arrangement of
// this code.  The patterns are those that seeded runs have had so far, uneven as
// they are (string_ratio rounds the product of the table's update, except in the
// first column below its first row), so that these runs repeat bit for bit.
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }

// a d - b c
template <typename F>
__device__ __forceinline__ F det2_rn(F a, F d, F b, F c) {
    return fma_rn(a, d, -mul_rn(b, c));
}

// det of the leading E x E block, as det_small expands it.
template <int E, typename F>
__device__ __forceinline__ F det_rn(const F (&m)[4][4]) {
    if constexpr (E == 0) {
        return F(1);
    } else if constexpr (E == 1) {
        return m[0][0];
    } else if constexpr (E == 2) {
        return det2_rn(m[0][0], m[1][1], m[0][1], m[1][0]);
    } else if constexpr (E == 3) {
        const F A = det2_rn(m[1][1], m[2][2], m[1][2], m[2][1]), B = det2_rn(m[1][0], m[2][2], m[1][2], m[2][0]),
                C = det2_rn(m[1][0], m[2][1], m[1][1], m[2][0]);
        return fma_rn(m[0][2], C, det2_rn(m[0][0], A, m[0][1], B));
    } else {
        const F a01 = det2_rn(m[0][0], m[1][1], m[0][1], m[1][0]), a02 = det2_rn(m[0][0], m[1][2], m[0][2], m[1][0]);
        const F a03 = det2_rn(m[0][0], m[1][3], m[0][3], m[1][0]), a12 = det2_rn(m[0][1], m[1][2], m[0][2], m[1][1]);
        const F a13 = det2_rn(m[0][1], m[1][3], m[0][3], m[1][1]), a23 = det2_rn(m[0][2], m[1][3], m[0][3], m[1][2]);
        const F b01 = det2_rn(m[2][0], m[3][1], m[2][1], m[3][0]), b02 = det2_rn(m[2][0], m[3][2], m[2][2], m[3][0]);
        const F b03 = det2_rn(m[2][0], m[3][3], m[2][3], m[3][0]), b12 = det2_rn(m[2][1], m[3][2], m[2][2], m[3][1]);
        const F b13 = det2_rn(m[2][1], m[3][3], m[2][3], m[3][1]), b23 = det2_rn(m[2][2], m[3][3], m[2][3], m[3][2]);
        return fma_rn(a23, b01, fma_rn(-a13, b02, fma_rn(a12, b03, fma_rn(a03, b12, det2_rn(a01, b23, a02, b13)))));
    }
}

// det of the block with column b replaced by u.
template <int E, typename F>
__device__ __forceinline__ F det_column_rn(const F (&m)[4][4], const F (&u)[4], int b) {
    F t[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) t[a][c] = a < E && c < E ? (c == b ? u[a] : m[a][c]) : F(0);
    return det_rn<E>(t);
}

// Adds a b.
__device__ __forceinline__ void add_product(Acc<float>& v, float a, float b) {
    const float s = __fmaf_rn(a, b, v.h), bp = __fsub_rn(s, v.h);
    v.l = __fadd_rn(v.l, __fadd_rn(__fsub_rn(v.h, __fsub_rn(s, bp)), __fmaf_rn(a, b, -bp)));
    v.h = s;
}
__device__ __forceinline__ void add_product(Acc<double>& v, double a, double b) { v.h = __fma_rn(a, b, v.h); }

// The four weights of a virtual as one load.
template <typename T>
struct alignas(16) Weights4 {
    T v[4];
};

// One string of excitation level E at the current position: gradient terms of
// sum_u Cd_u R_u.  The level is known at compile time (the strings are sorted by
// it): one body for all levels with its entries masked took some 350
// instructions per string where level 2, the most of them, needs about 100, and
// bounded the sweep (6-water cluster, 10,000 determinants, 256 walkers: sweep
// 6.0 -> 3.6 ms).
template <int E, typename T>
__device__ __forceinline__ void string_drift(const StrDesc& d, const T* Ts, int nv, const T* Ae, const T* Wq, T f,
                                             Acc<T>* va) {
    T m[4][4], u[4];
#pragma unroll
    for (int a = 0; a < E; ++a) {
        u[a] = Ae[d.h[a]];
#pragma unroll
        for (int b = 0; b < E; ++b) m[a][b] = Ts[d.h[a] * nv + d.p[b]];
    }
#pragma unroll
    for (int b = 0; b < E; ++b) {
        const Weights4<T> w = reinterpret_cast<const Weights4<T>*>(Wq)[d.p[b]];
        const T fb = mul_rn(f, det_column_rn<E>(m, u, b));
#pragma unroll
        for (int c = 0; c < 3; ++c) add_product(va[c], fb, w.v[c]);
    }
}

// The same at the proposed position, with the table's rank-1 update applied to
// the minor on the fly: adds cu R'_u and its gradient terms, returns R'_u.
template <int E, typename T>
__device__ __forceinline__ T string_ratio(const StrDesc& d, const T* Ts, int nv, const T* Ae, T rinv0, const T* Wq,
                                          T cu, Acc<T>* vs) {
    T m[4][4], u[4];
    Weights4<T> w[E > 0 ? E : 1];
#pragma unroll
    for (int b = 0; b < E; ++b) w[b] = reinterpret_cast<const Weights4<T>*>(Wq)[d.p[b]];
#pragma unroll
    for (int a = 0; a < E; ++a) {
        u[a] = mul_rn(Ae[d.h[a]], rinv0);
#pragma unroll
        for (int b = 0; b < E; ++b) {
            const T t = Ts[d.h[a] * nv + d.p[b]], wb = w[b].v[3];
            m[a][b] = b == 0 && a > 0 ? fma_rn(u[a], wb, t) : add_rn(t, mul_rn(u[a], wb));
        }
    }
    const T Ru = mul_rn(T(d.phase), det_rn<E>(m));
    add_product(vs[0], cu, Ru);
    const T f = mul_rn(T(d.phase), cu);
#pragma unroll
    for (int b = 0; b < E; ++b) {
        const T fb = mul_rn(f, det_column_rn<E>(m, u, b));
#pragma unroll
        for (int c = 0; c < 3; ++c) add_product(vs[1 + c], fb, w[b].v[c]);
    }
    return Ru;
}

constexpr double kRefreshRho0F = 1e-2;   // mixed form
constexpr double kRefreshRho0D = 1e-4;   // FP64 form

template <typename T>
__global__ void k_sweep_msd(DevSys s, DevWalkers wk, int W, SweepParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int w = blockIdx.x;
    if (w >= W) return;
    const int N = s.N, nu = s.n_up, nd = s.n_dn, nb = s.n_basis, nn = s.n_nuc;
    const int nmax = nu > nd ? nu : nd;
    const int nv0 = s.n_vir[0], nv1 = s.n_vir[1], nvmax = nv0 > nv1 ? nv0 : nv1;
    T* Wq = (T*)smem;            // [nvmax][4]: gradient weights W_c[p], then w[p]
    double* sR = (double*)(Wq + 4 * nvmax);
    double* red = sR + 3 * N;
    double* scal = red + kMaxWarps * 12;
    T* bas = (T*)(scal + 16);
    T* phi = bas + 5 * nb;
    T* phv = phi + 5 * nmax;
    T* cold = phv + 5 * nvmax;
    T* sA = cold + nmax;
    T* sT = sA + nu * nu + nd * nd;
    T* Ainv[2] = {sA, sA + nu * nu};
    T* Tt[2] = {sT, sT + nu * nv0};
    {
        const T* g0 = (const T*)wk.Ainv[0] + (size_t)w * nu * nu;
        const T* g1 = (const T*)wk.Ainv[1] + (size_t)w * nd * nd;
        for (int q = threadIdx.x; q < nu * nu; q += blockDim.x) Ainv[0][q] = g0[q];
        for (int q = threadIdx.x; q < nd * nd; q += blockDim.x) Ainv[1][q] = g1[q];
        const T* t0 = (const T*)wk.Tt[0] + (size_t)w * nu * nv0;
        const T* t1 = (const T*)wk.Tt[1] + (size_t)w * nd * nv1;
        for (int q = threadIdx.x; q < nu * nv0; q += blockDim.x) Tt[0][q] = t0[q];
        for (int q = threadIdx.x; q < nd * nv1; q += blockDim.x) Tt[1][q] = t1[q];
    }
    for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) sR[q] = wk.R[(size_t)w * 3 * N + q];
    double ld0 = 0.0, ld1 = 0.0, sg0 = 1.0, sg1 = 1.0;
    if (threadIdx.x == 0) {
        ld0 = wk.logdet[2 * w];
        ld1 = wk.logdet[2 * w + 1];
        sg0 = wk.sgn[2 * w];
        sg1 = wk.sgn[2 * w + 1];
        scal[8] = wk.Ssum[w];
    }
    unsigned long long acc = 0;
    __syncthreads();
    const double tau = p.tau;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T* redT = (T*)red;

    for (int e = 0; e < N; ++e) {
        const int spin = e >= nu;
        const int n = spin ? nd : nu, nv = spin ? nv1 : nv0, ns = s.n_str[spin];
        const int k = spin ? e - nu : e;
        T* A = Ainv[spin];
        T* Ts = Tt[spin];
        const T* Ae = A + (size_t)k * n;
        T* Gk = (T*)wk.G[spin] + ((size_t)w * n + k) * 4 * n;
        T* Gvk = (T*)wk.Gv[spin] + ((size_t)w * n + k) * 4 * nv;
        T* Avk = (T*)wk.Av[spin] + ((size_t)w * n + k) * nv;
        T* Rcur = (T*)wk.Rs[spin] + (size_t)w * ns;
        T* Rnew = (T*)wk.Rn[spin] + (size_t)w * ns;
        const T* Cd = (const T*)wk.Cd[spin] + (size_t)w * ns;
        const int4* str = s.str[spin];
        const double re0 = sR[3 * e], re1 = sR[3 * e + 1], re2 = sR[3 * e + 2];

        // -- drift at the current position ---------------------------------
        for (int q = threadIdx.x; q < 3 * nv; q += blockDim.x) {
            const int c = q / nv, pp = q - c * nv;
            T a = Gvk[c * nv + pp];
            for (int j = 0; j < n; ++j) a -= Gk[c * n + j] * Ts[(size_t)j * nv + pp];
            Wq[4 * pp + c] = a;
        }
        Acc<T> va[9];
        T u_old = T(0);
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
            const T a = Ae[j];
            va[0].add(Gk[j] * a);
            va[1].add(Gk[n + j] * a);
            va[2].add(Gk[2 * n + j] * a);
        }
        for (int q = threadIdx.x; q < N + nn; q += blockDim.x) {
            T x, y, z, a, b;
            if (q < N) {
                if (q == e) continue;
                x = T(re0 - sR[3 * q]); y = T(re1 - sR[3 * q + 1]); z = T(re2 - sR[3 * q + 2]);
                a = T(((q < nu) == (e < nu)) ? s.a_par : s.a_anti);
                b = T(s.b_ee);
            } else {
                const int c = q - N;
                x = T(re0 - s.Rn[3 * c]); y = T(re1 - s.Rn[3 * c + 1]); z = T(re2 - s.Rn[3 * c + 2]);
                a = T(s.a_en[c]);
                b = T(s.b_en);
            }
            const T ir = rsqrt_t(x * x + y * y + z * z);
            const T r = (x * x + y * y + z * z) * ir;
            const T qd = T(1) / (T(1) + b * r);
            u_old += a * r * qd;
            const T g = a * qd * qd * ir;
            va[3].add(g * x);
            va[4].add(g * y);
            va[5].add(g * z);
        }
        __syncthreads();
        for (int u = threadIdx.x; u < ns; u += blockDim.x) {
            const StrDesc d = decode(str[u]);
            const T f = T(d.phase) * Cd[u];
            switch (d.e) {   // the strings are sorted by excitation level
                case 0: break;
                case 1: string_drift<1, T>(d, Ts, nv, Ae, Wq, f, va + 6); break;
                case 2: string_drift<2, T>(d, Ts, nv, Ae, Wq, f, va + 6); break;
                case 3: string_drift<3, T>(d, Ts, nv, Ae, Wq, f, va + 6); break;
                default: string_drift<4, T>(d, Ts, nv, Ae, Wq, f, va + 6); break;
            }
        }
        double vd[9];
        block_sum_to0<9>(va, red, vd);
        if (threadIdx.x == 0) {
            const double iS = 1.0 / scal[8];
            const T g[3] = {T(vd[0] + vd[3] + vd[6] * iS), T(vd[1] + vd[4] + vd[7] * iS), T(vd[2] + vd[5] + vd[8] * iS)};
            const double r[3] = {re0, re1, re2};
            propose_move<T>(g, tau, r, p.key, p.sweep, (uint32_t)e, (uint32_t)w, scal);
        }
        __syncthreads();
        const double rn[3] = {scal[0], scal[1], scal[2]};

        // -- basis, occupied and virtual orbitals at r' -------------------
        for (int sh = threadIdx.x; sh < s.n_shell; sh += blockDim.x) shell_vgl<T>(s, sh, rn, bas, nb);
        __syncthreads();
        {
            const T* C = sys_C<T>(s, spin);
            const T* Cv = sys_Cv<T>(s, spin);
            for (int o = threadIdx.x; o < 5 * (n + nv); o += blockDim.x) {
                const int c = o / (n + nv), j = o - c * (n + nv);
                const T* b = bas + c * nb;
                T a0 = T(0), a1 = T(0);
                if (j < n) {
                    int l = 0;
                    for (; l + 2 <= nb; l += 2) {
                        a0 += C[(size_t)l * n + j] * b[l];
                        a1 += C[(size_t)(l + 1) * n + j] * b[l + 1];
                    }
                    for (; l < nb; ++l) a0 += C[(size_t)l * n + j] * b[l];
                    phi[c * nmax + j] = a0 + a1;
                } else {
                    const int pp = j - n;
                    int l = 0;
                    for (; l + 2 <= nb; l += 2) {
                        a0 += Cv[(size_t)l * nv + pp] * b[l];
                        a1 += Cv[(size_t)(l + 1) * nv + pp] * b[l + 1];
                    }
                    for (; l < nb; ++l) a0 += Cv[(size_t)l * nv + pp] * b[l];
                    phv[c * nvmax + pp] = a0 + a1;
                }
            }
        }
        __syncthreads();

        // -- reference ratio, its gradient, Jastrow change -----------------
        T vb2[8] = {T(0), T(0), T(0), T(0), -u_old, T(0), T(0), T(0)};
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
            const T a = Ae[j];
            vb2[0] += phi[j] * a;
            vb2[1] += phi[nmax + j] * a;
            vb2[2] += phi[2 * nmax + j] * a;
            vb2[3] += phi[3 * nmax + j] * a;
        }
        for (int q = threadIdx.x; q < N + nn; q += blockDim.x) {
            T x, y, z, a, b;
            if (q < N) {
                if (q == e) continue;
                x = T(rn[0] - sR[3 * q]); y = T(rn[1] - sR[3 * q + 1]); z = T(rn[2] - sR[3 * q + 2]);
                a = T(((q < nu) == (e < nu)) ? s.a_par : s.a_anti);
                b = T(s.b_ee);
            } else {
                const int c = q - N;
                x = T(rn[0] - s.Rn[3 * c]); y = T(rn[1] - s.Rn[3 * c + 1]); z = T(rn[2] - s.Rn[3 * c + 2]);
                a = T(s.a_en[c]);
                b = T(s.b_en);
            }
            const T ir = rsqrt_t(x * x + y * y + z * z);
            const T r = (x * x + y * y + z * z) * ir;
            const T qd = T(1) / (T(1) + b * r);
            vb2[4] += a * r * qd;
            const T g = a * qd * qd * ir;
            vb2[5] += g * x;
            vb2[6] += g * y;
            vb2[7] += g * z;
        }
        block_sum8<T>(vb2, redT);
        const T rho0 = vb2[0];
        const T rinv0 = T(1) / rho0;

        // -- new table column weights, string ratios and gradients ----------
        for (int q = threadIdx.x; q < 4 * nv; q += blockDim.x) {
            const int c = q / nv, pp = q - c * nv;
            T a = phv[c * nvmax + pp];
            for (int h = 0; h < n; ++h) a -= Ts[(size_t)h * nv + pp] * phi[c * nmax + h];
            Wq[4 * pp + (c == 0 ? 3 : c - 1)] = a;   // grad phi'_v - T^T grad phi'_occ (before the w term)
        }
        __syncthreads();
        for (int q = threadIdx.x; q < 3 * nv; q += blockDim.x) {
            const int c = q / nv, pp = q - c * nv;
            Wq[4 * pp + c] -= Wq[4 * pp + 3] * vb2[1 + c] * rinv0;
        }
        __syncthreads();
        Acc<T> vs[4];
        for (int u = threadIdx.x; u < ns; u += blockDim.x) {
            const StrDesc d = decode(str[u]);
            const T cu = Cd[u];
            T Ru;
            switch (d.e) {
                case 0: Ru = string_ratio<0, T>(d, Ts, nv, Ae, rinv0, Wq, cu, vs); break;
                case 1: Ru = string_ratio<1, T>(d, Ts, nv, Ae, rinv0, Wq, cu, vs); break;
                case 2: Ru = string_ratio<2, T>(d, Ts, nv, Ae, rinv0, Wq, cu, vs); break;
                case 3: Ru = string_ratio<3, T>(d, Ts, nv, Ae, rinv0, Wq, cu, vs); break;
                default: Ru = string_ratio<4, T>(d, Ts, nv, Ae, rinv0, Wq, cu, vs); break;
            }
            Rnew[u] = Ru;
        }
        double vsd[4];
        block_sum_to0<4>(vs, red + kMaxWarps * 8, vsd);
        if (threadIdx.x == 0) {
            const double S = scal[8], Sn = vsd[0];
            const double ratio = (double)rho0 * Sn / S;
            const double iSn = 1.0 / Sn;
            const T g[3] = {T((double)vb2[1] / (double)rho0 + (double)vb2[5] + vsd[1] * iSn),
                            T((double)vb2[2] / (double)rho0 + (double)vb2[6] + vsd[2] * iSn),
                            T((double)vb2[3] / (double)rho0 + (double)vb2[7] + vsd[3] * iSn)};
            const double ro3[3] = {re0, re1, re2};
            const int accept = accept_move_g<T>(T(ratio), g, vb2[4], tau, ro3, rn, scal + 3, p.key, p.sweep,
                                                (uint32_t)e, (uint32_t)w);
            scal[6] = (double)rho0;
            scal[7] = accept ? 1.0 : 0.0;
            scal[9] = Sn;
        }
        __syncthreads();
        if (scal[7] != 0.0) {
            for (int j = threadIdx.x; j < n; j += blockDim.x) cold[j] = A[(size_t)k * n + j];
            __syncthreads();
            for (int q = wid; q < n; q += nw) {
                T* Aq = A + (size_t)q * n;
                T t = T(0);
                for (int j = lane; j < n; j += 32) t += phi[j] * Aq[j];
                t = warp_sum(t);
                if (q == k) t -= T(1);
                const T f = t * rinv0;
                for (int j = lane; j < n; j += 32) Aq[j] -= f * cold[j];
            }
            for (int q = threadIdx.x; q < n * nv; q += blockDim.x) {
                const int h = q / nv, pp = q - h * nv;
                Ts[q] += cold[h] * Wq[4 * pp + 3] * rinv0;
            }
            for (int o = threadIdx.x; o < 4 * n; o += blockDim.x) {
                const int c = o / n, j = o - c * n;
                Gk[o] = phi[(c + 1) * nmax + j];
            }
            for (int o = threadIdx.x; o < 5 * nv; o += blockDim.x) {
                const int c = o / nv, pp = o - c * nv;
                if (c == 0)
                    Avk[pp] = phv[pp];
                else
                    Gvk[(c - 1) * nv + pp] = phv[c * nvmax + pp];
            }
            for (int u = threadIdx.x; u < ns; u += blockDim.x) Rcur[u] = Rnew[u];
            if (threadIdx.x == 0) {
                const double r0 = scal[6];
                if (spin) {
                    ld1 += log(fabs(r0));
                    if (r0 < 0.0) sg1 = -sg1;
                } else {
                    ld0 += log(fabs(r0));
                    if (r0 < 0.0) sg0 = -sg0;
                }
                // The expansion accepts moves on its own ratio; the rank-1
                // updates of A0^-1 and T divide by the reference ratio, which
                // may be near zero there (the reference near its node while
                // the expansion is not).  Such a walker is rebuilt from scratch
                // in FP64 after the sweep.
                if (fabs(r0) < (sizeof(T) == 4 ? kRefreshRho0F : kRefreshRho0D) && wk.refresh) wk.refresh[w] = 1;
                scal[8] = scal[9];
                sR[3 * e] = rn[0];
                sR[3 * e + 1] = rn[1];
                sR[3 * e + 2] = rn[2];
                ++acc;
            }
            __syncthreads();
        }
        if (e == nu - 1 && nd > 0) {
            // the up block is done: the down strings' partial sums see the new R_up
            refresh_cd<T>(s, wk, w, 1);
            __syncthreads();
        }
    }
    refresh_cd<T>(s, wk, w, 0);
    __syncthreads();
    for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) wk.R[(size_t)w * 3 * N + q] = sR[q];
    {
        T* g0 = (T*)wk.Ainv[0] + (size_t)w * nu * nu;
        T* g1 = (T*)wk.Ainv[1] + (size_t)w * nd * nd;
        for (int q = threadIdx.x; q < nu * nu; q += blockDim.x) g0[q] = Ainv[0][q];
        for (int q = threadIdx.x; q < nd * nd; q += blockDim.x) g1[q] = Ainv[1][q];
        T* t0 = (T*)wk.Tt[0] + (size_t)w * nu * nv0;
        T* t1 = (T*)wk.Tt[1] + (size_t)w * nd * nv1;
        for (int q = threadIdx.x; q < nu * nv0; q += blockDim.x) t0[q] = Tt[0][q];
        for (int q = threadIdx.x; q < nd * nv1; q += blockDim.x) t1[q] = Tt[1][q];
    }
    if (threadIdx.x == 0) {
        wk.logdet[2 * w] = ld0;
        wk.logdet[2 * w + 1] = ld1;
        wk.sgn[2 * w] = sg0;
        wk.sgn[2 * w + 1] = sg1;
        wk.Ssum[w] = scal[8];
        if (acc) atomicAdd(wk.n_acc, acc);
    }
}

template <typename T>
size_t msd_sweep_smem_bytes(const DevSys& s) {
    return msd_sweep_smem<T>(s.N, s.n_basis, s.n_up, s.n_dn, s.n_vir[0], s.n_vir[1]);
}

template <typename T>
cudaError_t launch_sweep_msd(const DevSys& s, const DevWalkers& wk, int W, const SweepParams& p, cudaStream_t st) {
    if (W == 0) return cudaSuccess;
    const size_t smem = msd_sweep_smem_bytes<T>(s);
    cudaError_t e = allow_smem(k_sweep_msd<T>, smem);
    if (e != cudaSuccess) return e;
    k_sweep_msd<T><<<W, 256, smem, st>>>(s, wk, W, p);
    return cudaGetLastError();
}

template size_t msd_sweep_smem_bytes<double>(const DevSys&);
template size_t msd_sweep_smem_bytes<float>(const DevSys&);
template cudaError_t launch_sweep_msd<double>(const DevSys&, const DevWalkers&, int, const SweepParams&, cudaStream_t);
template cudaError_t launch_sweep_msd<float>(const DevSys&, const DevWalkers&, int, const SweepParams&, cudaStream_t);

template <typename T>
cudaError_t launch_msd_table(const DevSys& s, const DevWalkers& wk, int W, cudaStream_t st, const int* only) {
    if (W == 0) return cudaSuccess;
    k_msd_table<T><<<W, 256, 0, st>>>(s, wk, W, only);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_msd_eloc(const DevSys& s, const DevWalkers& wk, int W, double* eloc, double* logpsi,
                            double* sign, double* grad, cudaStream_t st) {
    if (W == 0) return cudaSuccess;
    const int nmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    const int nvmax = s.n_vir[0] > s.n_vir[1] ? s.n_vir[0] : s.n_vir[1];
    const int nv = nvmax > 0 ? nvmax : 1;
    int n_tile = kElocTile;
    auto bytes = [&] {
        return sizeof(double) * (6 * (size_t)s.N + 2 * (size_t)nmax * nv + std::max(3 * nv, n_tile));
    };
    if (bytes() > 227 * 1024) n_tile = std::max(3 * nv, nmax);
    const size_t smem = bytes();
    cudaError_t e = allow_smem(k_msd_eloc<T>, smem);
    if (e != cudaSuccess) return e;
    k_msd_eloc<T><<<W, 256, smem, st>>>(s, wk, W, eloc, logpsi, sign, grad, n_tile);
    return cudaGetLastError();
}

template cudaError_t launch_msd_table<double>(const DevSys&, const DevWalkers&, int, cudaStream_t, const int*);
template cudaError_t launch_msd_table<float>(const DevSys&, const DevWalkers&, int, cudaStream_t, const int*);
template cudaError_t launch_msd_eloc<double>(const DevSys&, const DevWalkers&, int, double*, double*, double*,
                                             double*, cudaStream_t);
template cudaError_t launch_msd_eloc<float>(const DevSys&, const DevWalkers&, int, double*, double*, double*,
                                            double*, cudaStream_t);

}  // namespace qmc
