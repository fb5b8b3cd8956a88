// Body of the Sherman-Morrison sweep of one walker in the FP64 form (see
// k_sweep.cu), shared by the single-system kernel and the batched persistent
// kernel.
//
// Bound by the FP64 pipe (one warp instruction in 16 SM cycles, whatever its
// active lanes), so the FP64 work of a move is what counts:
//   - the basis runs on full warps and the contraction in fixed point
//     (basis64.cuh);
//   - the normals and the logarithms of the acceptance uniforms of all moves
//     are drawn at the start, one item per lane, instead of on one or two
//     lanes per move;
//   - the Metropolis test takes ln rho in FP32 unless that leaves it open, and
//     the determinant's logarithm is taken of the product of the accepted
//     ratios, once per sweep;
//   - pair terms and determinant terms sum in separate warps (a butterfly over
//     four values);
//   - a move's serial part runs on three lanes, one component each.
// The fixed-point orbitals of a proposal are held against the column of the
// inverse that they meet, as those of a rebuild are (kFxSlack, k_wavefunction.cu):
// where the column weighs small orbitals up, the move's orbitals are taken
// again as FP64 sums.
// 6-water cluster, 2048 walkers: 9.9 -> 6.0 ms a sweep (1345 -> about 600 FP64
// warp instructions a move); one water, 512 walkers: 283 -> 187 us.
#pragma once

#include "basis64.cuh"
#include "sweep_sm.cuh"

namespace qmc {

struct Sweep64Layout {
    size_t sR, chi, red, scal, basis, phi, cold, A, G, total;
    __host__ __device__ Sweep64Layout(const DevSys& s, int ainv_smem, int g_smem) {
        const int nu = s.n_up, nd = s.n_dn, nmax = nu > nd ? nu : nd;
        const size_t sq = (size_t)nu * nu + (size_t)nd * nd;
        size_t o = Basis64Layout(s.n_nuc, s.n_prim, s.n_shell, s.n_basis).total;
        basis = 0;
        sR = o;
        o += sizeof(double) * 3 * (size_t)s.N;
        chi = o;
        o += sizeof(double) * 4 * (size_t)s.N;
        red = o;
        o += sizeof(double) * 8 * 8;
        scal = o;
        o += sizeof(double) * 16;
        phi = o;
        o += sizeof(double) * 5 * (size_t)nmax;
        cold = o;
        o += sizeof(double) * 2 * (size_t)nmax;   // the replaced column and the update's factors
        A = o;
        if (ainv_smem) o += sizeof(double) * sq;
        G = o;
        if (g_smem) o += sizeof(double) * 4 * sq;
        total = (o + 15) & ~(size_t)15;
    }
};

// Warp totals of four values per lane: lanes with (lane & 7) == 0 hold value
// ((lane >> 3) & 1) + 2 (lane >> 4).
__device__ __forceinline__ double warp_fold4(const double (&v)[4]) {
    const int lane = threadIdx.x & 31;
    const bool h4 = lane & 16, h3 = lane & 8;
    double a[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) a[i] = (h4 ? v[i + 2] : v[i]) + __shfl_xor_sync(0xffffffffu, h4 ? v[i] : v[i + 2], 16);
    double r = (h3 ? a[1] : a[0]) + __shfl_xor_sync(0xffffffffu, h3 ? a[0] : a[1], 8);
    r += __shfl_xor_sync(0xffffffffu, r, 4);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    return r;
}

// Factor of the capped drift, 2 / (1 + sqrt(1 + 2 v^2 tau)).
__device__ __forceinline__ double drift_factor(double v2, double tau) {
    return 2.0 / (1.0 + sqrt(fma(2.0 * v2, tau, 1.0)));
}

// Sums over the CTA of the pair terms v (from the low threads up) and the
// determinant terms d (from the high threads down): per warp only what it
// holds (pw, dw: warp-uniform).  Returns v[lane] (lane < 4) and d[lane - 4]
// (lane < 8) to warp 0.  red: 8 x 8 doubles for the at most 8 warps of a
// sweep CTA.
__device__ __forceinline__ double sweep64_sum(const double (&v)[4], const double (&d)[4], bool pw, bool dw,
                                              double* red) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const double a = pw ? warp_fold4(v) : 0.0, b = dw ? warp_fold4(d) : 0.0;
    if ((lane & 7) == 0) {
        const int q = ((lane >> 3) & 1) + 2 * (lane >> 4);
        red[wid * 8 + q] = a;
        red[wid * 8 + 4 + q] = b;
    }
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 8) {
        t = red[threadIdx.x];
        for (int q = 1; q < nw; ++q) t += red[q * 8 + threadIdx.x];
    }
    return t;
}

// Sum of lanes 0, 1, 2, in every lane of the warp.
__device__ __forceinline__ double sum3(double x) {
    return __shfl_sync(0xffffffffu, x, 0) + __shfl_sync(0xffffffffu, x, 1) + __shfl_sync(0xffffffffu, x, 2);
}

// One CTA (at most 256 threads) sweeps walker w (every electron once).
// smem: Sweep64Layout.  kJ3: the trial function carries the three-body Jastrow.
template <bool kJ3>
__device__ __forceinline__ void sweep_walker64(const DevSys& s, const DevWalkers& wk, int w, const SweepParams& p,
                                               unsigned char* smem) {
    const int N = s.N, nu = s.n_up, nd = s.n_dn, nn = s.n_nuc;
    const int nmax = nu > nd ? nu : nd;
    const Basis64Layout LB(s.n_nuc, s.n_prim, s.n_shell, s.n_basis);
    const Sweep64Layout L(s, p.ainv_smem, p.g_smem);
    double* sR = (double*)(smem + L.sR);
    double* chi = (double*)(smem + L.chi);      // [N][4]: three normals, ln of the acceptance uniform
    double* red = (double*)(smem + L.red);
    double* scal = (double*)(smem + L.scal);    // [0..2] r', [3] 1 / ratio, [4] accept
    double* phi = (double*)(smem + L.phi);
    double* cold = (double*)(smem + L.cold);
    double* fq = cold + nmax;
    const double4* nuc = (const double4*)(smem + LB.nuc);
    unsigned char* sb = smem + L.basis;
    int* cnt = (int*)(sb + LB.cnt);
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;

    double* gA[2] = {(double*)wk.Ainv[0] + (size_t)w * nu * nu, (double*)wk.Ainv[1] + (size_t)w * nd * nd};
    double* gG[2] = {(double*)wk.G[0] + (size_t)w * 4 * nu * nu, (double*)wk.G[1] + (size_t)w * 4 * nd * nd};
    double* Ainv[2] = {gA[0], gA[1]};
    double* Gc[2] = {gG[0], gG[1]};
    if (p.ainv_smem) {
        Ainv[0] = (double*)(smem + L.A);
        Ainv[1] = Ainv[0] + nu * nu;
        for (int q = tid; q < nu * nu; q += nt) Ainv[0][q] = gA[0][q];
        for (int q = tid; q < nd * nd; q += nt) Ainv[1][q] = gA[1][q];
    }
    if (p.g_smem) {
        Gc[0] = (double*)(smem + L.G);
        Gc[1] = Gc[0] + 4 * nu * nu;
        for (int q = tid; q < 4 * nu * nu; q += nt) Gc[0][q] = gG[0][q];
        for (int q = tid; q < 4 * nd * nd; q += nt) Gc[1][q] = gG[1][q];
    }
    for (int q = tid; q < 3 * N; q += nt) sR[q] = wk.R[(size_t)w * 3 * N + q];
    // random numbers of the sweep: item q < 2 N is one Box-Muller pair of
    // electron q / 2 (the same words as draw_normals), the rest ln u
    for (int q = tid; q < 2 * N; q += nt) {
        const int e = q >> 1;
        const uint4 x = philox4x32_10(make_uint4(p.sweep, (uint32_t)e, (uint32_t)w, 0u), p.key);
        const double rr = sqrt(-2.0 * log(u01((q & 1) ? x.z : x.x)));
        double sn, cs;
        sincospi(2.0 * u01((q & 1) ? x.w : x.y), &sn, &cs);
        chi[4 * e + ((q & 1) ? 2 : 0)] = rr * cs;
        if (!(q & 1)) chi[4 * e + 1] = rr * sn;
    }
    for (int e = tid; e < N; e += nt)
        chi[4 * e + 3] = log(u01(philox4x32_10(make_uint4(p.sweep, (uint32_t)e, (uint32_t)w, 1u), p.key).x));
    const double tau = p.tau, sqt = sqrt(tau), i2t = 1.0 / (2.0 * tau);
    // product of the accepted ratios per spin, as mantissa and power of two
    double pm0 = 1.0, pm1 = 1.0;
    int pe0 = 0, pe1 = 0;
    unsigned long long acc = 0;
    __syncthreads();

    const bool pw = wid * 32 < N + nn || kJ3;   // warps with pair terms
    for (int e = 0; e < N; ++e) {
        const int spin = e >= nu;
        const int n = spin ? nd : nu;
        const int k = spin ? e - nu : e;
        double* A = Ainv[spin];
        double* Gs = Gc[spin];
        const double* Ae = A + (size_t)k * n;
        const double* Ge = Gs + (size_t)k * 4 * n;
        const double re0 = sR[3 * e], re1 = sR[3 * e + 1], re2 = sR[3 * e + 2];
        const bool dw = nt - 1 - (wid * 32 + 31) < n;   // warps with determinant terms

        // -- drift at the current position: grad_e ln|D| + grad_e J --------
        double v[4] = {0.0, 0.0, 0.0, 0.0}, d[4] = {0.0, 0.0, 0.0, 0.0};
        for (int j = nt - 1 - tid; j < n; j += nt) {
            const double a = Ae[j];
            d[1] += Ge[j] * a;
            d[2] += Ge[n + j] * a;
            d[3] += Ge[2 * n + j] * a;
        }
        auto pair = [&](double x, double y, double z, double r2, double a, double b) {
            const double ir = rsqrt(r2), q = 1.0 / (1.0 + b * (r2 * ir));
            const double aq = a * q, g = aq * (q * ir);   // u'(r) / r, its two products side by side
            v[0] += aq * (r2 * ir);
            v[1] += g * x;
            v[2] += g * y;
            v[3] += g * z;
        };
        for (int q = tid; q < N + nn; q += nt) {
            if (q == e) continue;
            const double* o = q < N ? sR + 3 * q : s.Rn + 3 * (q - N);
            const double x = re0 - o[0], y = re1 - o[1], z = re2 - o[2];
            pair(x, y, z, x * x + y * y + z * z,
                 q < N ? (((q < nu) == (e < nu)) ? s.a_par : s.a_anti) : s.a_en[q - N], q < N ? s.b_ee : s.b_en);
        }
        if constexpr (kJ3) {
            for (int q = tid; q < nn * N; q += nt) {
                double uv, gg[3];
                j3_of_electron_pair(s, sR, e, re0, re1, re2, q, uv, gg);
                v[0] += uv;
                v[1] += gg[0];
                v[2] += gg[1];
                v[3] += gg[2];
            }
        }
        double t = sweep64_sum(v, d, pw, dw, red);
        // the move's serial part: warp 0, its first three lanes one component each
        const int c3 = lane < 3 ? lane : 0;
        double u_old = 0.0, vb = 0.0, re = 0.0, rn = 0.0;
        if (wid == 0) {
            u_old = __shfl_sync(0xffffffffu, t, 0);
            const double g = __shfl_sync(0xffffffffu, t, 1 + c3) + __shfl_sync(0xffffffffu, t, 5 + c3);
            vb = drift_factor(sum3(g * g), tau) * g;
            re = sR[3 * e + c3];
            rn = fma(sqt, chi[4 * e + c3], fma(tau, vb, re));
            if (lane < 3) scal[lane] = rn;
        }
        __syncthreads();
        const double rn0 = scal[0], rn1 = scal[1], rn2 = scal[2];

        // -- basis and orbitals at the proposed position ---------------------
        const auto put = [phi, nmax](int c, int j, double x) { phi[c * nmax + j] = x; };
        bool plain = orbitals64(s, LB, sb, rn0, rn1, rn2, s.Ck[spin], s.Ck_s[spin], s.C[spin], n, put, nullptr, nullptr,
                                nullptr, 0, [](int, int, double) {});

        // -- ratio, new determinant gradient, Jastrow change ----------------
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = 0.0;
        for (int q = tid; q < N + nn; q += nt) {
            if (q == e) continue;
            double x, y, z, r2;
            if (q < N) {
                x = rn0 - sR[3 * q];
                y = rn1 - sR[3 * q + 1];
                z = rn2 - sR[3 * q + 2];
                r2 = x * x + y * y + z * z;
            } else {
                const double4 o = nuc[q - N];   // left by basis64
                x = o.x;
                y = o.y;
                z = o.z;
                r2 = o.w;
            }
            pair(x, y, z, r2, q < N ? (((q < nu) == (e < nu)) ? s.a_par : s.a_anti) : s.a_en[q - N],
                 q < N ? s.b_ee : s.b_en);
        }
        if constexpr (kJ3) {
            for (int q = tid; q < nn * N; q += nt) {
                double uv, gg[3];
                j3_of_electron_pair(s, sR, e, rn0, rn1, rn2, q, uv, gg);
                v[0] += uv;
                v[1] += gg[0];
                v[2] += gg[1];
                v[3] += gg[2];
            }
        }
        for (;; plain = true) {
            int fac = 0, term = 0;   // exponents: max|x_j| c_j, max|x_j phi_j|
#pragma unroll
            for (int c = 0; c < 4; ++c) d[c] = 0.0;
            for (int j = nt - 1 - tid; j < n; j += nt) {
                const double a = Ae[j], f = phi[j];
                d[0] += f * a;
                d[1] += phi[nmax + j] * a;
                d[2] += phi[2 * nmax + j] * a;
                d[3] += phi[3 * nmax + j] * a;
                const int ea = fx_expo(a), ef = fx_expo(f);
                fac = max(fac, ea + fx_expo(s.Ck_s[spin][j]));
                if (ef) term = max(term, ea + ef);
            }
            if (dw && !plain) {
                fac = warp_max_u(fac);
                term = warp_max_u(term);
                if (lane == 0) {
                    atomicMax(&cnt[29], fac);
                    atomicMax(&cnt[30], term);
                }
            }
            t = sweep64_sum(v, d, pw, dw, red);
            // (an orbital's scale is 2^-27 of its largest coefficient's power of two)
            if (plain || cnt[29] + 27 + cnt[8] - 1023 - cnt[30] <= kFxSlack) break;
            const double r[3] = {rn0, rn1, rn2};
            orbitals_plain(s, r, s.C[spin], n, (double*)(sb + LB.bas), put);
        }
        if (wid == 0) {
            const double rho = __shfl_sync(0xffffffffu, t, 4);
            int accept = 0;
            double ir = 0.0;
            if (rho > 0.0 && isfinite(rho)) {   // uniform in the warp
                ir = 1.0 / rho;
                const double g = fma(__shfl_sync(0xffffffffu, t, 5 + c3), ir, __shfl_sync(0xffffffffu, t, 1 + c3));
                const double dJ = __shfl_sync(0xffffffffu, t, 0) - u_old;
                const double vn = drift_factor(sum3(g * g), tau) * g;
                const double dr = rn - re, fw = fma(-tau, vb, dr), bk = fma(tau, vn, dr);
                // |r - r' - tau v'|^2 - |r' - r - tau v|^2
                const double diff = sum3(fma(bk, bk, -fw * fw));
                // accept iff 2 ln rho + rest > ln u.  The logarithm in FP32 (an
                // error below 2^-20 (1 + |ln rho|)) settles all but about one
                // move in 10^5.
                const double rest = fma(2.0, dJ, fma(-diff, i2t, -chi[4 * e + 3]));
                const float lr = logf((float)rho), rf = (float)rest, tf = fmaf(2.0f, lr, rf);
                if (fabsf(tf) > 1e-5f * (1.0f + fabsf(lr) + fabsf(rf)) && rho < 1e30 && rho > 1e-30)
                    accept = tf > 0.0f;
                else
                    accept = rest + 2.0 * log(rho) > 0.0;
            }
            if (lane == 0) {
                scal[3] = ir;
                scal[4] = accept ? 1.0 : 0.0;
                if (accept) {
                    const double m = (spin ? pm1 : pm0) * rho;
                    const long long b = fx_bits(m);
                    const int ex = (int)((b >> 52) & 0x7ff);
                    if (ex > 0 && ex < 2047 && fx_expo(rho) > 0) {
                        // m > 0: leave its mantissa in [1, 2)
                        const double mant = fx_double((b & 0xfffffffffffffLL) | (1023LL << 52));
                        if (spin) {
                            pm1 = mant;
                            pe1 += ex - 1023;
                        } else {
                            pm0 = mant;
                            pe0 += ex - 1023;
                        }
                    } else {
                        wk.logdet[2 * w + spin] += log(rho);   // a product out of range: add its logarithm
                    }
                }
            }
        }
        __syncthreads();
        if (scal[4] != 0.0) {
            for (int j = tid; j < n; j += nt) cold[j] = A[(size_t)k * n + j];
            const double rinv = scal[3];
            if (p.ainv_smem) {
                // each row's dot product on its own thread, then the rank-1 update
                for (int q = tid; q < n; q += nt) {
                    const double* Aq = A + (size_t)q * n;
                    double t0 = q == k ? -1.0 : 0.0, t1 = 0.0;
                    int j = 0;
                    for (; j + 1 < n; j += 2) {
                        t0 += phi[j] * Aq[j];
                        t1 += phi[j + 1] * Aq[j + 1];
                    }
                    if (j < n) t0 += phi[j] * Aq[j];
                    fq[q] = (t0 + t1) * rinv;
                }
                __syncthreads();
                for (int o = tid; o < n * n; o += nt) {
                    const int q = o / n, j = o - q * n;
                    A[o] -= fq[q] * cold[j];
                }
            } else {
                __syncthreads();
                for (int q = wid; q < n; q += nw) {
                    double* Aq = A + (size_t)q * n;
                    double t = 0.0;
                    for (int j = lane; j < n; j += 32) t += phi[j] * Aq[j];
                    t = warp_sum(t);
                    if (q == k) t -= 1.0;
                    const double f = t * rinv;
                    for (int j = lane; j < n; j += 32) Aq[j] -= f * cold[j];
                }
            }
            double* Gk = Gs + (size_t)k * 4 * n;
            for (int o = tid; o < 4 * n; o += nt) {
                const int c = o / n, j = o - c * n;
                Gk[o] = phi[(c + 1) * nmax + j];
            }
            if (tid == 0) {
                sR[3 * e] = rn0;
                sR[3 * e + 1] = rn1;
                sR[3 * e + 2] = rn2;
                ++acc;
            }
            __syncthreads();
        }
    }

    for (int q = tid; q < 3 * N; q += nt) wk.R[(size_t)w * 3 * N + q] = sR[q];
    if (p.ainv_smem) {
        for (int q = tid; q < nu * nu; q += nt) gA[0][q] = Ainv[0][q];
        for (int q = tid; q < nd * nd; q += nt) gA[1][q] = Ainv[1][q];
    }
    if (p.g_smem) {
        for (int q = tid; q < 4 * nu * nu; q += nt) gG[0][q] = Gc[0][q];
        for (int q = tid; q < 4 * nd * nd; q += nt) gG[1][q] = Gc[1][q];
    }
    if (tid == 0) {
        const double ln2 = 0.69314718055994530942;
        wk.logdet[2 * w] += log(pm0) + (double)pe0 * ln2;
        wk.logdet[2 * w + 1] += log(pm1) + (double)pe1 * ln2;
        if (acc) atomicAdd(wk.n_acc, acc);
    }
}

// Whether the FP64 sweep of this system runs as sweep_walker64: its lists fit
// shared memory with A^-1 in global memory (else sweep_walker<double>).
__host__ __device__ inline bool sweep64_fits(const DevSys& s) { return Sweep64Layout(s, 0, 0).total <= kBasis64Max; }

}  // namespace qmc
