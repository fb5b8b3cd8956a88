// Ionic derivatives of E_L and ln|psi| for every walker by an adjoint
// (reverse-mode) pass.
//
// Sec. "Single Determinant QMC Forces" writes the derivative of a
// determinant one-body operator as tr(A^-1 dB/dR_a - X dA/dR_a) with
// X = A^-1 B A^-1 (Eq. 4) and d ln D = tr(A^-1 dA) (Eq. 3), evaluated there
// once per nuclear coordinate (cost O(N^3 3 N_atom)).  Here the kinetic
// determinant term is written as tr(B A^-1) with
//   B_ij = -1/2 lap phi_j(r_i) - grad_i J . grad phi_j(r_i),
// and since every dA, dB is a contraction of basis-function derivatives with
// the coefficient matrix C, the traces are pulled back to basis space once:
//   M = C^T A^-1         (n_basis x n),  weights of dPhi in d ln D and dB,
//   Y = M (B A^-1)       (n_basis x n),  weights of dPhi in -tr(X dA).
// Then for each electron i and basis function l on nucleus a
//   d ln D / dR_a += -M_li d Phi_l(r_i)
//   dT_det / dR_a += -M_li (-1/2 d lap Phi_l - grad_i J . d grad Phi_l)
//                    + Y_li d Phi_l(r_i)
// (the basis function moves with its nucleus: d/dR_a = -d/dr).  The cost
// is O(n^2 n_basis + n^3 + N n_basis) per walker, independent of N_atom.
// Basis derivatives to third order are recomputed per walker rather than
// stored.  The e-n Jastrow, V_en and V_nn terms are added directly.
#include <algorithm>
#include <type_traits>

#include "batch.cuh"
#include "fixed64.cuh"
#include "qmc_internal.cuh"

namespace qmc {

constexpr int kForceTile = 32;  // basis functions per tile of M and Y

// Adjoint terms of one shell at one electron.  Let x be the offset from the
// centre, t = |x|^2, f0..f3 the radial sums and g = grad_i J.  With M, Y the
// basis-space weights of the shell's functions Phi_m = P_m S, the sums over m
//   v_q = sum_m M_m (1/2 d_q lap Phi_m + (Hess Phi_m g)_q) + Y_m d_q Phi_m,
//   w_q = sum_m M_m d_q Phi_m
// are linear in the polynomials, so they are taken once for the combined
// polynomial sum_m M_m P_m (value U, gradient G, Hessian H; UY, GY those of
// sum_m Y_m P_m) instead of once per function.  P_m is homogeneous of degree
// l, so G.x = l U and H x = (l - 1) G, and
//   v_q = x_q [U ((10 + 4 l) f2 + 4 t f3 + 4 f2 (x.g)) + 2 f1 (G.g + UY) + f1 tr H]
//       + g_q [2 f1 U] + G_q [(3 + 2 l) f1 + 2 t f2 + 2 f1 (x.g)] + f0 ((H g)_q + GY_q),
//   w_q = x_q [2 f1 U] + G_q f0.
// The coefficients of x_q and g_q are scalars that add over all shells of a
// centre; only the G, H g terms stay vectors.  (One evaluation per function
// instead took 135 FP64 instructions per p shell and 300 per d shell, against
// 28 and 65 here.)
template <typename T>
struct RunTerms {
    T ax = T(0), ag = T(0);                  // coefficients of x_q and g_q in v; ag is also that of x_q in w
    T v[3] = {T(0), T(0), T(0)}, w[3] = {T(0), T(0), T(0)};
};

template <typename T>
__device__ __forceinline__ void shell_terms(int l, int pure, const T x[3], const T g[3], T xg, T t, T f0, T f1, T f2,
                                            T f3, const T* M, const T* Y, size_t ld, RunTerms<T>& o) {
    const T f12 = T(2) * f1;
    if (l == 0) {
        const T m = M[0];
        o.ax += m * (f2 * (T(10) + T(4) * xg) + T(4) * t * f3) + f12 * Y[0];
        o.ag += f12 * m;
        return;
    }
    if (l == 1) {
        const T m[3] = {M[0], M[ld], M[2 * ld]}, y[3] = {Y[0], Y[ld], Y[2 * ld]};
        const T U = m[0] * x[0] + m[1] * x[1] + m[2] * x[2];
        const T q = m[0] * g[0] + m[1] * g[1] + m[2] * g[2] + y[0] * x[0] + y[1] * x[1] + y[2] * x[2];
        o.ax += U * (f2 * (T(14) + T(4) * xg) + T(4) * t * f3) + f12 * q;
        o.ag += f12 * U;
        const T cG = f1 * (T(5) + T(2) * xg) + T(2) * t * f2;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            o.v[c] += m[c] * cG + f0 * y[c];
            o.w[c] += m[c] * f0;
        }
        return;
    }
    // d: Hessians (xx, xy, xz, yy, yz, zz) of the combined polynomials
    const T s3 = T(1.7320508075688772);
    T H[6], K[6], tr = T(0);
    if (pure) {
        const T a2 = M[2 * ld], a4 = s3 * M[4 * ld], b2 = Y[2 * ld], b4 = s3 * Y[4 * ld];
        H[0] = a4 - a2; H[1] = s3 * M[0]; H[2] = s3 * M[3 * ld]; H[3] = -a2 - a4; H[4] = s3 * M[ld]; H[5] = T(2) * a2;
        K[0] = b4 - b2; K[1] = s3 * Y[0]; K[2] = s3 * Y[3 * ld]; K[3] = -b2 - b4; K[4] = s3 * Y[ld]; K[5] = T(2) * b2;
    } else {
        H[0] = T(2) * M[0]; H[1] = s3 * M[ld]; H[2] = s3 * M[2 * ld];
        H[3] = T(2) * M[3 * ld]; H[4] = s3 * M[4 * ld]; H[5] = T(2) * M[5 * ld];
        K[0] = T(2) * Y[0]; K[1] = s3 * Y[ld]; K[2] = s3 * Y[2 * ld];
        K[3] = T(2) * Y[3 * ld]; K[4] = s3 * Y[4 * ld]; K[5] = T(2) * Y[5 * ld];
        tr = H[0] + H[3] + H[5];
    }
    const T G[3] = {H[0] * x[0] + H[1] * x[1] + H[2] * x[2], H[1] * x[0] + H[3] * x[1] + H[4] * x[2],
                    H[2] * x[0] + H[4] * x[1] + H[5] * x[2]};
    const T R[3] = {K[0] * x[0] + K[1] * x[1] + K[2] * x[2], K[1] * x[0] + K[3] * x[1] + K[4] * x[2],
                    K[2] * x[0] + K[4] * x[1] + K[5] * x[2]};
    const T Hg[3] = {H[0] * g[0] + H[1] * g[1] + H[2] * g[2], H[1] * g[0] + H[3] * g[1] + H[4] * g[2],
                     H[2] * g[0] + H[4] * g[1] + H[5] * g[2]};
    const T U = T(0.5) * (G[0] * x[0] + G[1] * x[1] + G[2] * x[2]);
    const T UY = T(0.5) * (R[0] * x[0] + R[1] * x[1] + R[2] * x[2]);
    const T Gg = G[0] * g[0] + G[1] * g[1] + G[2] * g[2];
    o.ax += U * (f2 * (T(18) + T(4) * xg) + T(4) * t * f3) + f12 * (Gg + UY) + f1 * tr;
    o.ag += f12 * U;
    const T cG = f1 * (T(7) + T(2) * xg) + T(2) * t * f2;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        o.v[c] += G[c] * cG + f0 * (Hg[c] + R[c]);
        o.w[c] += G[c] * f0;
    }
}

// Radial sums of one shell for the 32 electrons of a warp, FP64: about a
// third of the (primitive, electron) pairs are unscreened, so the live pairs
// of up to kRadialPrims primitives are listed and each exponential is taken
// once on consecutive lanes, instead of one masked exponential per primitive
// and warp.  The screening test runs in FP32 (a pair near the threshold is
// below 1e-26 either way).  Called by whole warps; `on` marks the lanes that
// hold an electron.  scr: kRadialScratch bytes of the warp's shared memory.
constexpr int kRadialPrims = 4;
constexpr int kRadialScratch = kRadialPrims * 32 * (int)(sizeof(double) + sizeof(short));
__device__ __forceinline__ void warp_radial3(const DevSys& s, int p0, int np, double t, bool on, void* scr, double& f0,
                                             double& f1, double& f2, double& f3) {
    double* ev = (double*)scr;
    short* lst = (short*)(ev + kRadialPrims * 32);
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const float tf = on ? (float)t : 3.0e38f;
    f0 = f1 = f2 = f3 = 0.0;
    for (int q0 = 0; q0 < np; q0 += kRadialPrims) {
        const int nq = min(kRadialPrims, np - q0);
        int cnt = 0;
        unsigned mine = 0;
        for (int q = 0; q < nq; ++q) {
            const bool live = on && !(s.alpha_f[p0 + q0 + q] * tf > (float)kScreenExponent);
            const unsigned m = __ballot_sync(0xffffffffu, live);
            if (live) {
                lst[cnt + __popc(m & below)] = (short)(q * 32 + lane);
                mine |= 1u << q;
            }
            cnt += __popc(m);
        }
        if (cnt == 0) continue;
        __syncwarp();
        for (int k = 0; k < cnt; k += 32) {
            const int e = k + lane < cnt ? lst[k + lane] : 0;
            const double te = __shfl_sync(0xffffffffu, t, e & 31);
            if (k + lane < cnt) {
                const int p = p0 + q0 + (e >> 5);
                ev[e] = s.cn[p] * exp(-s.alpha[p] * te);
            }
        }
        __syncwarp();
        for (int q = 0; q < nq; ++q)
            if (mine & (1u << q)) {
                const double a = s.alpha[p0 + q0 + q], e = ev[q * 32 + lane];
                const double e1 = a * e, e2 = a * e1;
                f0 += e;
                f1 -= e1;
                f2 += e2;
                f3 -= a * e2;
            }
        __syncwarp();
    }
}

// Terms of the shells [sh0, sh1) of one centre at one electron per lane (the
// whole warp calls; `on`: the lane holds an electron): derivatives v, w with
// respect to the electron coordinate (see RunTerms).  M, Y: weights of the
// functions from shell sh0 on, row stride ld.
template <typename T>
__device__ __forceinline__ void run_terms(const DevSys& s, int sh0, int sh1, bool on, const T x[3], const T g[3],
                                          const T* M, const T* Y, size_t ld, void* scr, T (&v)[8]) {
    const T t = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
    const T xg = x[0] * g[0] + x[1] * g[1] + x[2] * g[2];
    const int fn0 = s.shell_fn[sh0];
    RunTerms<T> o;
    for (int sh = sh0; sh < sh1; ++sh) {
        const int4 d = s.shell[sh];
        T f0 = T(0), f1 = T(0), f2 = T(0), f3 = T(0);
        if constexpr (sizeof(T) == 8) {
            warp_radial3(s, d.z, d.w, t, on, scr, f0, f1, f2, f3);
        } else {
            if (on) radial<T, true>(s.alpha_f, s.cn_f, d.z, d.w, t, f0, f1, f2, f3);
        }
        if (f0 == T(0) && f1 == T(0) && f2 == T(0) && f3 == T(0)) continue;   // screened (or no electron)
        const size_t row = (size_t)(s.shell_fn[sh] - fn0) * ld;
        shell_terms<T>(d.y & 0xff, d.y >> 8, x, g, xg, t, f0, f1, f2, f3, M + row, Y + row, ld, o);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        v[c] = o.ax * x[c] + o.ag * g[c] + o.v[c];
        v[3 + c] = o.ag * x[c] + o.w[c];
    }
    v[6] = v[7] = T(0);
}

// Shared-memory head of every force kernel: positions (FP64), the per-atom
// sums acc[nn][6] (FP64: dT (3), dlnpsi (3)), grad_i J and grad_i ln|psi|
// in the form's type T, and the positions split as hi + lo floats, from
// which the mixed form takes its FP32 offsets without an FP64 instruction.
template <typename T>
__host__ __device__ inline size_t force_head_bytes(int N, int nn) {
    return sizeof(double) * (3 * (size_t)N + 6 * (size_t)nn) + sizeof(T) * 6 * (size_t)N + sizeof(float) * 6 * (size_t)N;
}

template <typename T>
struct ForceHead {
    double* sR;
    double* acc;
    T* gJ;
    T* gt;
    float* sRh;
    float* sRl;
    __device__ ForceHead(double* sm, int N, int nn) {
        sR = sm;
        acc = sR + 3 * N;
        gJ = (T*)(acc + 6 * nn);
        gt = gJ + 3 * N;
        sRh = (float*)(gt + 3 * N);
        sRl = sRh + 3 * N;
    }
    __device__ T* end(int N) const { return (T*)(void*)(sRl + 3 * N); }
};

template <typename T>
__device__ __forceinline__ void force_load_positions(const ForceHead<T>& h, const double* R, int N) {
    for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) {
        const double r = R[q];
        h.sR[q] = r;
        if constexpr (sizeof(T) == 4) {
            const float hi = (float)r;
            h.sRh[q] = hi;
            h.sRl[q] = (float)(r - (double)hi);
        }
    }
}

// Offsets r_i - r_j and r_i - R_a, component c, in the form's precision.
template <typename T>
__device__ __forceinline__ T off_ee(const ForceHead<T>& h, int i, int j, int c) {
    if constexpr (sizeof(T) == 4)
        return diff_f2(h.sRh[3 * i + c], h.sRl[3 * i + c], h.sRh[3 * j + c], h.sRl[3 * j + c]);
    else
        return h.sR[3 * i + c] - h.sR[3 * j + c];
}

template <typename T>
__device__ __forceinline__ T off_en(const ForceHead<T>& h, const DevSys& s, int i, int a, int c) {
    if constexpr (sizeof(T) == 4)
        return diff_f2(h.sRh[3 * i + c], h.sRl[3 * i + c], s.Rn_hi[3 * a + c], s.Rn_lo[3 * a + c]);
    else
        return h.sR[3 * i + c] - s.Rn[3 * a + c];
}

// grad_i J and grad_i ln|psi| of every electron (a warp per electron, lanes
// over its orbitals and its partners), then the e-n Jastrow, V_en and V_nn
// parts of the per-atom sums (a warp per nucleus, lanes over electrons).
// Terms and per-electron sums in T, per-atom sums in FP64.  row(spin, k, g, G): the
// warp's work on electron k of the spin once its g = grad J is known, while its
// row G of the gradient cache is at hand.  Ends synchronised.
template <typename T, typename Row>
__device__ __forceinline__ void force_gradients_en(const DevSys& s, const DevWalkers& wk, int w, const double* dvnn,
                                                   const ForceHead<T>& h, Row row) {
    const int N = s.N, nu = s.n_up, nn = s.n_nuc;
    // (in T once: a conversion per pair was most of the mixed form's FP64 work)
    T a_par = T(s.a_par), a_anti = T(s.a_anti);
    hold(a_par);
    hold(a_anti);
    const T b_ee = T(s.b_ee), b_en = T(s.b_en);
    auto a_en = [&](int c) {
        if constexpr (sizeof(T) == 4) return s.a_en_f[c];
        else return s.a_en[c];
    };
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = wid; i < N; i += nw) {
        const int spin = i >= nu;
        const int n = spin ? s.n_dn : nu;
        const int k = spin ? i - nu : i;
        const T* Ai = (const T*)wk.Ainv[spin] + ((size_t)w * n + k) * n;
        const T* Gi = (const T*)wk.G[spin] + ((size_t)w * n + k) * 4 * n;
        T v[8] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0)};   // grad ln|D| (3), grad J (3)
        for (int j = lane; j < n; j += 32) {
            const T a = Ai[j];
            v[0] += Gi[j] * a;
            v[1] += Gi[n + j] * a;
            v[2] += Gi[2 * n + j] * a;
        }
        for (int j = lane; j < N + nn; j += 32) {
            T x[3], a, b;
            if (j < N) {
                if (j == i) continue;
#pragma unroll
                for (int c = 0; c < 3; ++c) x[c] = off_ee(h, i, j, c);
                a = ((i < nu) == (j < nu)) ? a_par : a_anti;
                b = b_ee;
            } else {
                const int c0 = j - N;
#pragma unroll
                for (int c = 0; c < 3; ++c) x[c] = off_en(h, s, i, c0, c);
                a = a_en(c0);
                b = b_en;
            }
            const T r2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
            const T ir = rsqrt_t(r2);
            const T qd = T(1) / (T(1) + b * r2 * ir);
            const T gr = a * qd * qd * ir;  // u'(r) / r
#pragma unroll
            for (int c = 0; c < 3; ++c) v[3 + c] += gr * x[c];
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] += v[3 + c];
        const T sum = warp_fold8(v);
        const int q = fold8_index(lane);
        if ((lane & 3) == 0 && q < 6) (q < 3 ? h.gt + q : h.gJ + (q - 3))[3 * i] = sum;
        const T g[3] = {__shfl_sync(0xffffffffu, sum, fold8_lane(3)), __shfl_sync(0xffffffffu, sum, fold8_lane(4)),
                        __shfl_sync(0xffffffffu, sum, fold8_lane(5))};
        row(spin, k, g, Gi);
    }
    __syncthreads();

    for (int a = wid; a < nn; a += nw) {
        const T Za = T(s.Z[a]), aen = T(s.a_en[a]), ben = T(s.b_en);
        T dT[3] = {T(0), T(0), T(0)}, dJ[3] = {T(0), T(0), T(0)};
        for (int i = lane; i < N; i += 32) {
            T x[3], g[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                x[c] = off_en(h, s, i, a, c);
                g[c] = h.gt[3 * i + c];
            }
            const T r2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
            const T ir = rsqrt_t(r2), r = r2 * ir;
            T u, du, d2u, d3u;
            pade3<T>(aen, ben, r, u, du, d2u, d3u);
            const T cl = T(0.5) * (d3u + T(2) * d2u * ir - T(2) * du * ir * ir) * ir;
            const T hx = (d2u - du * ir) * ir * ir;
            const T gdot = g[0] * x[0] + g[1] * x[1] + g[2] * x[2];
            T vr3 = Za * ir * ir * ir;
            if (s.npp)   // local pseudopotential terms: d v(r)/dR_a = -v'(r) x / r, folded into the -Z x / r^3 slot
                for (int t = s.pp_off[a]; t < s.pp_off[a + 1]; ++t) {
                    const int2 ln = s.pp_ln[t];
                    if (ln.x == -1) vr3 += pp_term_dr<T>(s, t, ln.y, r) * ir;
                }
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                // sum_c H_cq g_c with H = hx x x^T + (du/r) I
                const T Hg = hx * x[q] * gdot + du * ir * g[q];
                dT[q] += cl * x[q] + Hg - vr3 * x[q];
                dJ[q] -= du * x[q] * ir;
            }
        }
        const double v[8] = {double(dT[0]), double(dT[1]), double(dT[2]), double(dJ[0]),
                             double(dJ[1]), double(dJ[2]), 0.0, 0.0};
        const double sum = warp_fold8(v);
        const int q = fold8_index(lane);
        if ((lane & 3) == 0 && q < 6) h.acc[6 * a + q] = sum + (q < 3 ? dvnn[3 * a + q] : 0.0);
    }
    __syncthreads();
}

// Rows of dot products of one warp: out(r, i) = sum_k A_r[k] B_i[k] for nl
// rows r of the left factor (row stride lda) and all n electrons i (row
// stride ldb).  Lanes take (group of kForceRows rows, electron) items, so one
// load of B serves kForceRows rows and the rows of A are (nearly) broadcast.
constexpr int kForceRows = 4;

// FP64 form: operands as limbs (fixed64.cuh); put receives the sum in units
// of the two rows' scales.
template <typename Put>
__device__ __forceinline__ void warp_rows(int nl, int n, const int2* A, int lda, const int2* B, int ldb, Put put) {
    const int lane = threadIdx.x & 31, items = (nl + kForceRows - 1) / kForceRows * n;
    for (int o = lane; o < items; o += 32) {
        const int g = o / n, i = o - g * n, r0 = g * kForceRows, nr = min(kForceRows, nl - r0);
        const int2* b = B + (size_t)i * ldb;
        const int2* a[kForceRows];
#pragma unroll
        for (int r = 0; r < kForceRows; ++r) a[r] = A + (size_t)(r0 + min(r, nr - 1)) * lda;
        FxSum sum[kForceRows];
        for (int k0 = 0; k0 < n; k0 += kFxBlock) {
            FxDot d[kForceRows];
            const int k1 = min(n, k0 + kFxBlock);
#pragma unroll 2
            for (int k = k0; k < k1; ++k) {
                const int2 bv = b[k];
#pragma unroll
                for (int r = 0; r < kForceRows; ++r) d[r].add(a[r][k], bv);
            }
#pragma unroll
            for (int r = 0; r < kForceRows; ++r) sum[r].fold(d[r]);
        }
#pragma unroll
        for (int r = 0; r < kForceRows; ++r)
            if (r < nr) put(r0 + r, i, sum[r].value());
    }
}
template <typename Put>
__device__ __forceinline__ void warp_rows(int nl, int n, const float* A, int lda, const float* B, int ldb, Put put) {
    const int lane = threadIdx.x & 31, items = (nl + kForceRows - 1) / kForceRows * n;
    const bool even = ((n | lda) & 1) == 0 && ((uintptr_t)A & 7) == 0;   // the rows of A can be read in pairs
    for (int o = lane; o < items; o += 32) {
        const int g = o / n, i = o - g * n, r0 = g * kForceRows, nr = min(kForceRows, nl - r0);
        const float* b = B + (size_t)i * ldb;
        const float* a[kForceRows];
        float v[kForceRows];
#pragma unroll
        for (int r = 0; r < kForceRows; ++r) {
            a[r] = A + (size_t)(r0 + min(r, nr - 1)) * lda;
            v[r] = 0.f;
        }
        if (even) {
#pragma unroll 2
            for (int k = 0; k < n; k += 2) {
                const float b0 = b[k], b1 = b[k + 1];
#pragma unroll
                for (int r = 0; r < kForceRows; ++r) {
                    const float2 av = *reinterpret_cast<const float2*>(a[r] + k);
                    v[r] += av.x * b0;
                    v[r] += av.y * b1;
                }
            }
        } else {
#pragma unroll 2
            for (int k = 0; k < n; ++k) {
                const float bv = b[k];
#pragma unroll
                for (int r = 0; r < kForceRows; ++r) v[r] += a[r][k] * bv;
            }
        }
#pragma unroll
        for (int r = 0; r < kForceRows; ++r)
            if (r < nr) put(r0 + r, i, v[r]);
    }
}

// Limbs of n doubles x by one warp into q (x and q may be the same memory:
// each lane rewrites what it read); returns the row's scale.
__device__ __forceinline__ double warp_limbs(const double* x, int2* q, int n) {
    const int lane = threadIdx.x & 31;
    int e = 0;
    for (int k = lane; k < n; k += 32) e = max(e, fx_expo(x[k]));
    e = warp_max_u(e);
    for (int k = lane; k < n; k += 32) q[k] = fx_limbs(x[k], e);
    return fx_scale(e);
}

// Whether the fixed-point products of an electron's row a of A^-T would lose
// bits against FP64 sums: the largest entries of it and of the electron's row b of
// B, in units of the orbitals' largest coefficients, against the largest product
// a_q b_q.  row_range takes a lane's entries (a times, b over the orbital's scale
// c) into its exponents ea, eb, eab.
__device__ __forceinline__ void row_range(double a, double b, double c, int& ea, int& eb, int& eab) {
    const int ec = fx_expo(c), x = fx_expo(a) ? fx_expo(a) + ec : 0, y = fx_expo(b) ? fx_expo(b) - ec + 2046 : 0;
    ea = max(ea, x);
    eb = max(eb, y);
    if (x && y) eab = max(eab, x + y);
}
__device__ __forceinline__ bool row_short(int ea, int eb, int eab) {
    return warp_max_u(ea) + warp_max_u(eb) - warp_max_u(eab) > kFxSlack;
}

// Reciprocal of a scale (a power of two from fx_scale; NaN and 0 to NaN).
__device__ __forceinline__ double fx_inverse(double scale) {
    const int e = fx_expo(scale);
    return e == 0 || e == 2047 ? fx_double(0x7ff8000000000000LL) : fx_double((long long)(2046 - e) << 52);
}

// Groups of kForceRows rows that a warp of force_walker forms together: as
// many (at most 3, and within the warp's scratch) as fill its lanes best.
__host__ __device__ inline int force_row_groups(int n) {
    int best = 1;
    for (int g = 2; g <= 3; ++g) {
        if (g * kForceRows * n * 8 > 2560) break;
        const int used = n * g, lanes = (used + 31) / 32, ub = n * best, lb = (ub + 31) / 32;
        if (used * lb > ub * lanes) best = g;
    }
    return best;
}

// Shared memory of force_walker.  The transposed inverse and P^T =
// (B A^-1)^T of a spin are read once per basis function by the products
// M = C A^-T and Y = M P, so they are staged with an odd row stride ld: as
// limbs with their row scales in the FP64 form, as floats in the mixed form;
// a determinant too large for that (stg false) reads A^-T and keeps B and
// P^T in global memory.  M and Y are formed for F basis functions at a time:
// all of them where the budget allows (2 CTAs per SM in FP64, 3 mixed), so
// that the contraction keeps a warp per centre busy.
// Bound by FP64 issue (FP64 form) and by instruction issue (mixed).  6-water
// cluster, 2048 walkers: 8.10 -> 3.64 ms FP64 and 0.81 -> 0.44 ms mixed
// against one derivative evaluation per basis function, FP64 products and a
// masked exponential per primitive.
// Where only one CTA fits an SM (above kForceTwo bytes: determinants above about
// 55), it takes the whole SM: sixteen warps instead of eight, each with its
// scratch, and tiles of as many basis functions as fit, so that a tile has centres
// enough for the warps (a batch of 16 clusters of up to 130 electrons, 64 walkers
// each: 5.2 -> 4.4 ms; sixteen warps with the smallest tiles 6.0, eight with
// large ones 4.8).
// FP64 form: a spin in which some electron's row of A^-T weighs small entries
// of B up (row_short; electrons shared out unevenly over distant fragments with
// orbitals of their own) is taken as a determinant too large to stage is, in FP64 sums.
// So is a spin of at most kForcePlain electrons: limbs, their scales and the
// whole-warp row groups cost more than its short sums.  Pass in FP64 sums / limbs /
// as before either: one water, 64 walkers 62 / 93 / 87 us, 2048 walkers 432 / 647 /
// 950; 3 waters (15 electrons), 64 and 2048 walkers 148 / 178 / 292 and 1477 / 1617
// us; 4 waters (20) 195 / 216 and 2255 / 2125 us; 6 waters (30) 4.6 / 3.6 ms.
constexpr size_t kForceTwo = 113 * 1024;
constexpr int kForcePlain = 16;
template <typename T>
struct ForceShape {
    bool stg;
    int ld, F, scr;                                      // scr: bytes of scratch per warp
    size_t AT, PT, sA, scratch, M, Y, gE, total;         // byte offsets
    __host__ __device__ ForceShape(int N, int nn, int nmax, int nb, bool kE, int nw = 8) {
        const size_t head = (force_head_bytes<T>(N, nn) + 15) & ~(size_t)15;
        const size_t e_bytes = kE ? sizeof(double) * 3 * (size_t)N : 0;
        ld = nmax | 1;
        scr = 0;
        if (sizeof(T) == 8) {
            scr = 3 * kForceRows * nmax * 8;
            if (scr > 2560) scr = 2560 > kForceRows * nmax * 8 ? 2560 : kForceRows * nmax * 8;
            if (scr < kRadialScratch) scr = kRadialScratch;
            scr = (scr + 15) & ~15;
        }
        const size_t mat = (sizeof(T) * (size_t)nmax * ld + 15) & ~(size_t)15;
        const size_t row = 2 * sizeof(T) * (size_t)nmax;
        // the tile also holds B (with its row scales) while P^T is formed
        int fmin = kForceTile > (ld + 2) / 2 ? kForceTile : (ld + 2) / 2;
        const size_t fixed = head + 2 * mat + 2 * sizeof(T) * (size_t)nmax + 16 + 8 * (size_t)scr + e_bytes;
        stg = fixed + row * fmin <= 200 * 1024;
        if (!stg) fmin = kForceTile;
        AT = head;
        PT = AT + (stg ? mat : 0);
        sA = PT + (stg ? mat : 0);
        scratch = (sA + (stg ? 2 * sizeof(T) * (size_t)nmax : 0) + 15) & ~(size_t)15;
        M = scratch + nw * (size_t)scr;
        size_t budget = (sizeof(T) == 8 ? 112 : 74) * 1024;
        F = fmin;
        if (M + e_bytes + row * fmin > kForceTwo) budget = 220 * 1024;   // one CTA per SM: all there is
        if (stg && budget > M + e_bytes + row * fmin) {
            const size_t fit = (budget - M - e_bytes) / row;
            F = fit < (size_t)nb ? (int)fit : nb;
            if (F < fmin) F = fmin;
        }
        Y = M + sizeof(T) * (size_t)F * nmax;
        gE = (Y + sizeof(T) * (size_t)F * nmax + 15) & ~(size_t)15;
        total = gE + e_bytes;
    }
    // warps of a CTA: sixteen where only one CTA fits an SM
    static int warps(int N, int nn, int nmax, int nb, bool kE) {
        return ForceShape(N, nn, nmax, nb, kE).total > kForceTwo ? 16 : 8;
    }
};

// Adjoint ionic derivatives of walker w (body of k_force).  sm: the
// dynamic shared memory of launch_force (ForceShape), 256 or 512 threads.  kE: also
// the determinant part of dE_L/dr_i (the same basis-space terms, every basis
// function moving with the electron, d/dr_i = -d/dR) into gEdet [W][N][3]
// and grad_i ln|psi| into gtot [W][N][3], for the space warp.
template <typename T, bool kE = false>
__device__ __forceinline__ void force_walker(const DevSys& s, const DevWalkers& wk, int w, const double* dvnn, double* Bscr,
                                             double* Pscr, double* dEL, double* dlog, double* sm,
                                             double* gEdet = nullptr, double* gtot = nullptr) {
    const int N = s.N, nu = s.n_up, nn = s.n_nuc;
    const int nmax = nu > s.n_dn ? nu : s.n_dn;
    constexpr bool kFx = sizeof(T) == 8;
    using Q = std::conditional_t<kFx, int2, float>;   // staged operands
    const ForceShape<T> fs(N, nn, nmax, s.n_basis, kE, blockDim.x >> 5);
    unsigned char* smb = (unsigned char*)sm;
    const ForceHead<T> h(sm, N, nn);
    double* acc = h.acc;
    Q* sAT = (Q*)(smb + fs.AT);
    Q* sPT = (Q*)(smb + fs.PT);
    T* sA = (T*)(smb + fs.sA);         // row scales of A^-T and P^T (FP64 form)
    T* sP = sA + nmax;
    T* Mt = (T*)(smb + fs.M);          // [F][nmax]
    T* Yt = (T*)(smb + fs.Y);
    Q* sB = (Q*)Mt;                    // B while P^T is formed, [n][ld]
    T* sBs = (T*)(sB + (size_t)nmax * fs.ld);
    T* B = (T*)(Bscr + (size_t)w * nmax * nmax);
    T* PTg = (T*)(Pscr + (size_t)w * nmax * nmax);
    double* gEs = (double*)(smb + fs.gE);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    Q* scr = (Q*)(smb + fs.scratch + (size_t)wid * fs.scr);

    force_load_positions(h, wk.R + (size_t)w * 3 * N, N);
    if constexpr (kE)
        for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) gEs[q] = 0.0;
    __syncthreads();
    force_gradients_en<T>(s, wk, w, dvnn, h, [](int, int, const T*, const T*) {});

    for (int spin = 0; spin < 2; ++spin) {
        const int n = spin ? s.n_dn : nu;
        if (n == 0) continue;
        const int i0 = spin ? nu : 0, ld = fs.ld;
        const T* ATg = (const T*)wk.Ainv[spin] + (size_t)w * n * n;
        const T* Gs = (const T*)wk.G[spin] + (size_t)w * 4 * n * n;
        const T* nlB = wk.nlB[spin] ? (const T*)wk.nlB[spin] + (size_t)w * n * n : nullptr;
        const T* C = sys_C<T>(s, spin);
        // B_pq = -1/2 lap phi_q(r_p) - grad_p J . grad phi_q(r_p), plus the
        // non-local pseudopotential's rows (E_L gains tr(B_NL A^-1), so the
        // same -tr(X dA) pull-back covers them)
        auto b_of = [&](int pp, int qq) {
            const T* Gp = Gs + (size_t)pp * 4 * n;
            const T* gj = h.gJ + 3 * (i0 + pp);
            T b = T(-0.5) * Gp[3 * n + qq] - gj[0] * Gp[qq] - gj[1] * Gp[n + qq] - gj[2] * Gp[2 * n + qq];
            if (nlB) b += nlB[(size_t)pp * n + qq];
            return b;
        };
        bool stg = fs.stg && !(kFx && n <= kForcePlain);
        if (stg) {
            int lossy = 0;
            for (int r = wid; r < n; r += nw) {
                T* at = (T*)(sAT + (size_t)r * ld);
                T* bt = (T*)(sB + (size_t)r * ld);
                int ea = 0, eb = 0, eab = 0;
                for (int q = lane; q < n; q += 32) {
                    T a = ATg[(size_t)r * n + q], b = b_of(r, q);
                    if constexpr (kFx) {   // orbital q in units of its largest coefficient
                        const double c = s.Ck_s[spin][q];
                        row_range(a, b, c, ea, eb, eab);
                        a *= c;
                        b *= fx_inverse(c);
                    }
                    at[q] = a;
                    bt[q] = b;
                }
                if constexpr (kFx) {
                    lossy |= row_short(ea, eb, eab);
                    const double a = warp_limbs(at, (int2*)at, n), b = warp_limbs(bt, (int2*)bt, n);
                    if (lane == 0) {
                        sA[r] = a;
                        sBs[r] = b;
                    }
                }
            }
            stg = !__syncthreads_or(lossy);
        }
        if (stg) {
            // PT[i][p] = (B A^-1)_{p i} = sum_q AT[i][q] B_pq
            const int rows = kForceRows * force_row_groups(n);
            for (int r0 = wid * rows; r0 < n; r0 += nw * rows) {
                const int nl = min(rows, n - r0);
                T* pt = (T*)(sPT + (size_t)r0 * ld);
                // (FP64 form: column p in units of electron p's row of A^-T, as
                // the limbs of M take it below, so that an electron far out, whose
                // row of A^-T is large, leaves the others their bits)
                warp_rows(nl, n, sAT + (size_t)r0 * ld, ld, sB, ld, [&](int r, int p, T v) {
                    if constexpr (kFx) v = v * sA[r0 + r] * sBs[p] * sA[p];
                    pt[r * ld + p] = v;
                });
                if constexpr (kFx) {
                    __syncwarp();
                    for (int r = 0; r < nl; ++r) {
                        const double a = warp_limbs(pt + r * ld, (int2*)(pt + r * ld), n);
                        if (lane == 0) sP[r0 + r] = a;
                    }
                }
            }
        } else {
            for (int q2 = threadIdx.x; q2 < n * n; q2 += blockDim.x) B[q2] = b_of(q2 / n, q2 % n);
            __syncthreads();
            for (int q2 = threadIdx.x; q2 < n * n; q2 += blockDim.x) {
                const int i = q2 / n, pp = q2 - i * n;
                T v = T(0);
                for (int q = 0; q < n; ++q) v += B[(size_t)pp * n + q] * ATg[(size_t)i * n + q];
                PTg[q2] = v;
            }
        }
        __syncthreads();
        int sh0 = 0, run0 = 0;
        while (sh0 < s.n_shell) {
            const int fl0 = s.shell_fn[sh0];
            int sh1 = sh0 + 1;
            while (sh1 < s.n_shell && s.shell_fn[sh1 + 1] - fl0 <= fs.F) ++sh1;
            const int nfl = s.shell_fn[sh1] - fl0;
            // M[l][i] = sum_j C[l][j] AT[i][j],  Y[l][i] = sum_p M[l][p] PT[i][p]
            if (stg) {
                const int rows = kForceRows * force_row_groups(n);
                for (int r0 = wid * rows; r0 < nfl; r0 += nw * rows) {
                    const int nl = min(rows, nfl - r0), l0 = fl0 + r0;
                    T* m = Mt + (size_t)r0 * nmax;
                    T* y = Yt + (size_t)r0 * nmax;
                    if constexpr (kFx) {
                        const double* sC = s.Cq_s[spin] + l0;
                        warp_rows(nl, n, s.Cq[spin] + (size_t)l0 * n, n, sAT, ld,
                                  [&](int r, int i, double v) { m[r * nmax + i] = v * sC[r]; });
                        __syncwarp();
                        double sM[3 * kForceRows];
#pragma unroll
                        for (int r = 0; r < 3 * kForceRows; ++r)
                            sM[r] = r < nl ? warp_limbs(m + r * nmax, scr + r * n, n) : 0.0;
                        for (int r = 0; r < nl; ++r)
                            for (int i = lane; i < n; i += 32) m[r * nmax + i] *= sA[i];
                        __syncwarp();
                        warp_rows(nl, n, scr, n, sPT, ld, [&](int r, int i, double v) {
                            double a = 0.0;
#pragma unroll
                            for (int q = 0; q < 3 * kForceRows; ++q) a = q == r ? sM[q] : a;
                            y[r * nmax + i] = v * a * sP[i];
                        });
                        __syncwarp();
                    } else {
                        warp_rows(nl, n, C + (size_t)l0 * n, n, sAT, ld,
                                  [&](int r, int i, float v) { m[r * nmax + i] = v; });
                        __syncwarp();
                        warp_rows(nl, n, m, nmax, sPT, ld, [&](int r, int i, float v) { y[r * nmax + i] = v; });
                    }
                }
            } else {
                for (int q2 = threadIdx.x; q2 < nfl * n; q2 += blockDim.x) {
                    const int l = q2 / n, i = q2 - l * n;
                    T v = T(0);
                    for (int j = 0; j < n; ++j) v += C[(size_t)(fl0 + l) * n + j] * ATg[(size_t)i * n + j];
                    Mt[l * nmax + i] = v;
                }
                __syncthreads();
                for (int q2 = threadIdx.x; q2 < nfl * n; q2 += blockDim.x) {
                    const int l = q2 / n, i = q2 - l * n;
                    T v = T(0);
                    for (int p = 0; p < n; ++p) v += Mt[l * nmax + p] * PTg[(size_t)i * n + p];
                    Yt[l * nmax + i] = v;
                }
            }
            __syncthreads();
            // warp per run of shells on one centre (the part of it in this
            // tile), lanes over the electrons of this spin
            while (s.run_sh[run0 + 1] <= sh0) ++run0;
            for (int run = run0 + wid; run < s.n_run && s.run_sh[run] < sh1; run += nw) {
                const int a0 = max(sh0, s.run_sh[run]), a1 = min(sh1, s.run_sh[run + 1]);
                const int ctr = s.shell[a0].x, lb = s.shell_fn[a0] - fl0;
                T v[8] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
                for (int c0 = 0; c0 < n; c0 += 32) {
                    const bool on = c0 + lane < n;
                    const int i = on ? c0 + lane : n - 1;
                    const T x[3] = {off_en(h, s, i0 + i, ctr, 0), off_en(h, s, i0 + i, ctr, 1),
                                    off_en(h, s, i0 + i, ctr, 2)};
                    const T gj[3] = {h.gJ[3 * (i0 + i)], h.gJ[3 * (i0 + i) + 1], h.gJ[3 * (i0 + i) + 2]};
                    T vt[8];
                    run_terms<T>(s, a0, a1, on, x, gj, Mt + (size_t)lb * nmax + i, Yt + (size_t)lb * nmax + i, nmax, scr,
                                 vt);
                    if (!on) continue;
#pragma unroll
                    for (int q = 0; q < 6; ++q) v[q] += vt[q];
                    if constexpr (kE)
#pragma unroll
                        for (int q = 0; q < 3; ++q) atomicAdd(&gEs[3 * (i0 + i) + q], -double(vt[q]));
                }
                // the basis functions move with their nucleus, d/dR = -d/dr:
                // dT = sum M (wL dlap + w.dgrad) - Y dPhi with each d -> -d/dr
                const T sum = warp_fold8(v);
                const int q = fold8_index(lane);
                if ((lane & 3) == 0 && q < 6) atomicAdd(&acc[6 * ctr + q], q < 3 ? double(sum) : -double(sum));
            }
            __syncthreads();
            sh0 = sh1;
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < 3 * nn; q += blockDim.x) {
        const int a = q / 3, c = q - 3 * a;
        dEL[(size_t)w * 3 * nn + q] = acc[6 * a + c] + (wk.nlF ? wk.nlF[(size_t)w * 3 * nn + q] : 0.0);
        dlog[(size_t)w * 3 * nn + q] = acc[6 * a + 3 + c];
    }
    if constexpr (kE)
        for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) {
            gEdet[(size_t)w * 3 * N + q] = gEs[q];
            gtot[(size_t)w * 3 * N + q] = double(h.gt[q]);
        }
}

// Three CTAs per SM in the FP32 form (80 registers, no spills); the FP64
// form keeps two (at three it spills).
template <typename T, bool kE, int kNt>
__global__ void __launch_bounds__(kNt, kNt == 512 ? 1 : sizeof(T) == 4 ? 3 : 2)
    k_force(DevSys s, DevWalkers wk, int W, const double* dvnn, double* Bscr, double* Pscr, double* dEL, double* dlog,
            double* gEdet, double* gtot) {
    extern __shared__ double sm[];
    const int w = blockIdx.x;
    if (w >= W) return;
    force_walker<T, kE>(s, wk, w, dvnn, Bscr, Pscr, dEL, dlog, sm, gEdet, gtot);
}

// ---------------------------------------------------------------------
// Large determinants: the same adjoint with its dense products done as
// batched GEMMs (k_force_prep -> GEMMs -> k_force_contract).  Per walker and
// spin, with X^T = AT (the stored transposed inverse) and B as above:
//   PT = AT B^T,  Q = PT AT        (n x n, batched over walkers)
//   M  = C AT^T,  Y = C Q^T        (n_basis x n, C shared by all walkers)
// M and Y are exactly the tiles k_force builds on chip; for n above ~64
// they no longer fit, and as GEMMs they run near the ALU roofline.
// ---------------------------------------------------------------------

// Per walker: grad J (stored), B for both spins (stored, type T), and the
// e-n Jastrow / V_en / V_nn part of the per-atom sums (stored).  A warp forms
// its electron's row of B as soon as that electron's grad J is summed, so the
// gradient cache is read from memory once (32-water cluster, 512 walkers, mixed:
// 495 -> 398 us).
// lossy (FP64 form): count (zero before the launch), then the walkers of the
// launch in which some electron's row of A^-T weighs small entries of B up
// (row_short): their products are not left to bf16 digits (k_force_products).
template <typename T, bool kE>
__global__ void k_force_prep(DevSys s, DevWalkers wk, int w0, int W, const double* dvnn, T* Bw, double* gJw,
                             double* accw, double* gtot, int* lossy) {
    extern __shared__ double sm[];
    const int wl = blockIdx.x, w = w0 + wl;
    if (wl >= W) return;
    const int N = s.N, nu = s.n_up, nn = s.n_nuc;
    const int nmax = nu > s.n_dn ? nu : s.n_dn;
    const ForceHead<T> h(sm, N, nn);
    force_load_positions(h, wk.R + (size_t)w * 3 * N, N);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    int low = 0;
    force_gradients_en<T>(s, wk, w, dvnn, h, [&](int spin, int k, const T* g, const T* G) {
        const int n = spin ? s.n_dn : nu;
        T* B = Bw + ((size_t)(spin * W + wl)) * nmax * nmax + (size_t)k * n;
        const T* nlB = (const T*)wk.nlB[spin];
        if (nlB) nlB += (size_t)w * n * n + (size_t)k * n;
        const T* Ai = (const T*)wk.Ainv[spin] + ((size_t)w * n + k) * n;
        int ea = 0, eb = 0, eab = 0;
        for (int q = lane; q < n; q += 32) {
            T b = T(-0.5) * G[3 * n + q] - g[0] * G[q] - g[1] * G[n + q] - g[2] * G[2 * n + q];
            if (nlB) b += nlB[q];   // non-local pseudopotential rows
            B[q] = b;
            if constexpr (sizeof(T) == 8) row_range(Ai[q], b, s.Ck_s[spin][q], ea, eb, eab);
        }
        if constexpr (sizeof(T) == 8) low |= row_short(ea, eb, eab);
    });
    if constexpr (sizeof(T) == 8) {
        low = __syncthreads_or(low);
        if (threadIdx.x == 0 && low) lossy[1 + atomicAdd(lossy, 1)] = wl;
    }
    for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) gJw[(size_t)wl * 3 * N + q] = double(h.gJ[q]);
    for (int q = threadIdx.x; q < 6 * nn; q += blockDim.x) accw[(size_t)wl * 6 * nn + q] = h.acc[q];
    if constexpr (kE)
        for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) gtot[(size_t)w * 3 * N + q] = double(h.gt[q]);
}

// The four products of the listed walkers in FP64, in place of those that the
// digits gave: stage 0 PT = AT B^T and M = C AT^T, 1 Q = PT AT, 2 Y = C Q^T.  Few
// walkers, so each is spread over the chip: persistent CTAs over 32 x 32 tiles of
// every listed walker and spin (a launch that finds none takes 2 us; one CTA a
// walker by the fused kernel took 3 ms at 70 electrons per spin).  Bound by the FP64
// pipe: four sums a thread, operands through shared memory.
constexpr int kPt = 32;
struct ProductArgs {
    const double *AT[2], *C[2];                 // [wc][n][n] of the chunk, [n_basis][n]
    double *B, *PT, *Q, *M, *Y;                 // [spin][wc][nmax^2] and [spin][wc] n_basis nmax
    int n[2], nmax, nb, wc;
};
__global__ void __launch_bounds__(256) k_force_products(ProductArgs p, int stage, const int* lossy) {
    __shared__ double sa[kPt][kPt + 1], sb[kPt][kPt + 1];
    const int count = lossy[0];
    const int tn[2] = {(p.n[0] + kPt - 1) / kPt, (p.n[1] + kPt - 1) / kPt}, tb = (p.nb + kPt - 1) / kPt;
    // tiles per walker and spin: n x n in stages 0 and 1, n_basis x n in 0 and 2
    auto tiles = [&](int s) { return (stage < 2 ? tn[s] * tn[s] : 0) + (stage != 1 ? tb * tn[s] : 0); };
    const int per = tiles(0) + tiles(1);
    const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5;   // column, first of four rows
    for (int it = blockIdx.x; it < count * per; it += gridDim.x) {
        const int wl = lossy[1 + it / per];
        int t = it % per;
        const int s = t >= tiles(0);
        if (s) t -= tiles(0);
        const int n = p.n[s];
        const size_t sq = ((size_t)s * p.wc + wl) * p.nmax * p.nmax;
        const size_t bn = (size_t)s * p.wc * p.nb * p.nmax + (size_t)wl * p.nb * n;
        const double* AT = p.AT[s] + (size_t)wl * n * n;
        const bool square = stage < 2 && t < tn[s] * tn[s];
        if (stage == 0 && !square) t -= tn[s] * tn[s];
        const double *a = p.C[s], *b = stage == 0 ? AT : p.Q + sq;   // rows of both factors: M, Y
        double* d = (stage == 0 ? p.M : p.Y) + bn;
        int rows = p.nb;
        if (square) {
            a = stage == 0 ? AT : p.PT + sq;
            b = stage == 0 ? p.B + sq : AT;
            d = (stage == 0 ? p.PT : p.Q) + sq;
            rows = n;
        }
        const int i0 = t / tn[s] * kPt, j0 = t % tn[s] * kPt;
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        for (int k0 = 0; k0 < n; k0 += kPt) {
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = r0 + 8 * u;
                sa[r][c] = i0 + r < rows && k0 + c < n ? a[(size_t)(i0 + r) * n + k0 + c] : 0.0;
                // sb[j][k]: b's rows are the output's columns, in stage 1 its columns are
                if (stage == 1)
                    sb[c][r] = k0 + r < n && j0 + c < n ? b[(size_t)(k0 + r) * n + j0 + c] : 0.0;
                else
                    sb[r][c] = j0 + r < n && k0 + c < n ? b[(size_t)(j0 + r) * n + k0 + c] : 0.0;
            }
            __syncthreads();
#pragma unroll 8
            for (int k = 0; k < kPt; ++k) {
                const double bv = sb[c][k];
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[u] += sa[r0 + 8 * u][k] * bv;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = i0 + r0 + 8 * u;
            if (r < rows && j0 + c < n) d[(size_t)r * n + j0 + c] = acc[u];
        }
    }
}

cudaError_t launch_force_products(const DevSys& s, const DevWalkers& wk, int w0, int wc, double* B, double* PT, double* Q,
                                  double* M, double* Y, const int* lossy, cudaStream_t st) {
    ProductArgs p{};
    for (int spin = 0; spin < 2; ++spin) {
        p.n[spin] = spin ? s.n_dn : s.n_up;
        p.AT[spin] = (const double*)wk.Ainv[spin] + (size_t)w0 * p.n[spin] * p.n[spin];
        p.C[spin] = s.C[spin];
    }
    p.B = B;
    p.PT = PT;
    p.Q = Q;
    p.M = M;
    p.Y = Y;
    p.nmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    p.nb = s.n_basis;
    p.wc = wc;
    for (int stage = 0; stage < 3; ++stage) {
        k_force_products<<<4 * device_sms(), 256, 0, st>>>(p, stage, lossy);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// CTAs per walker of k_force_contract: each takes a range of nuclei (the
// functions of a nucleus only add to its own sums), enough for six waves, so that
// the last one is not most of the time; one where the per-electron sums of the
// space warp are wanted, which run over all nuclei.  32-water cluster, 512
// walkers, mixed: 855 -> 507 us, with the runs shared out as warps come free.
// (Whole pass, mixed, 512 walkers, one, two, four and eight parts: 14 waters 0.85,
// 0.86, 0.87, 0.89, 20 waters 1.03, 1.03, 1.05, 1.08, 32 waters 1.89, 1.87, 1.89,
// 1.93 ms.  With 64 walkers 14 waters would gain from more parts than the 24 nuclei
// allow, 0.40 ms at the one they get and 0.34 at four.)
// Each spin adds to sums of its own: both on the nucleus's one made the last
// bits depend on which warp came first (one warp taking both spins of a run,
// which also fixes the order, was 3 % slower on the whole pass).
static int contract_parts(int W, int nn, bool kE) {
    if (kE) return 1;
    int p = 1;
    while ((long long)W * p < 6LL * 3 * device_sms() && nn / (2 * p) >= 24) p *= 2;
    return p;
}
// Nuclei of a part up to which spin down has sums of its own: thousands of
// nuclei (point charges) would not leave them room.
constexpr int kContractOwn = 1024;

// Third-order basis contraction with M, Y read from the GEMM outputs
// Mw/Yw [spin][walker][n_basis][n] (type T; each spin's block starts at
// spin W n_basis max(n_up, n_dn)).
template <typename T, bool kE>
__global__ void __launch_bounds__(256) k_force_contract(DevSys s, DevWalkers wk, int w0, int W, const T* Mw,
                                                        const T* Yw, const double* gJw, const double* accw,
                                                        double* dEL, double* dlog, double* gEdet) {
    extern __shared__ double sm[];
    const int wl = blockIdx.x, w = w0 + wl;
    if (wl >= W) return;
    const int N = s.N, nu = s.n_up, nn = s.n_nuc, nb = s.n_basis;
    // nuclei [na, nz) of the walker
    const int na = (int)blockIdx.y * nn / gridDim.y, nz = ((int)blockIdx.y + 1) * nn / gridDim.y;
    const ForceHead<T> h(sm, N, nn);
    double* acc = h.acc;
    unsigned char* scr = (unsigned char*)sm + ((force_head_bytes<T>(N, nn) + 15) & ~(size_t)15);
    // spin down's sums [6 (nz - na)], acc: spin up's (or both)
    const bool own = nz - na <= kContractOwn;
    double* acc_dn = (double*)(scr + (sizeof(T) == 8 ? 8 * kRadialScratch : 0));
    double* gEs = acc_dn + (own ? 6 * (nz - na) : 0);
    scr += (threadIdx.x >> 5) * kRadialScratch;   // the warp's radial scratch (FP64 form)
    force_load_positions(h, wk.R + (size_t)w * 3 * N, N);
    if constexpr (kE)
        for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) gEs[q] = 0.0;
    for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) h.gJ[q] = T(gJw[(size_t)wl * 3 * N + q]);
    for (int q = 6 * na + threadIdx.x; q < 6 * nz; q += blockDim.x) {
        acc[q] = accw[(size_t)wl * 6 * nn + q];
        if (own) acc_dn[q - 6 * na] = 0.0;
    }
    __syncthreads();
    // both spins' runs in turn to whichever warp is free (functions per run differ)
    __shared__ int s_next;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) s_next = 0;
    __syncthreads();
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(&s_next, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= 2 * s.n_run) break;
        const int spin = it >= s.n_run, run = it - spin * s.n_run;
        const int n = spin ? s.n_dn : nu;
        if (n == 0) continue;
        const int sh0 = s.run_sh[run], sh1 = s.run_sh[run + 1];
        const int ctr = s.shell[sh0].x;
        if (ctr < na || ctr >= nz) continue;
        const int i0 = spin ? nu : 0;
        const size_t off = (size_t)spin * W * nb * (nu > s.n_dn ? nu : s.n_dn) + (size_t)wl * nb * n;
        const T* M = Mw + off;
        const T* Y = Yw + off;
        // a run of shells on one centre, lanes over electrons: term
        // sums in T, one FP64 atomic per run and component
        {
            const size_t fl = (size_t)s.shell_fn[sh0] * n;
            T v[8] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
            for (int c0 = 0; c0 < n; c0 += 32) {
                const bool on = c0 + lane < n;
                const int i = on ? c0 + lane : n - 1;
                const T x[3] = {off_en(h, s, i0 + i, ctr, 0), off_en(h, s, i0 + i, ctr, 1),
                                off_en(h, s, i0 + i, ctr, 2)};
                const T gj[3] = {h.gJ[3 * (i0 + i)], h.gJ[3 * (i0 + i) + 1], h.gJ[3 * (i0 + i) + 2]};
                T vt[8];
                run_terms<T>(s, sh0, sh1, on, x, gj, M + fl + i, Y + fl + i, n, scr, vt);
                if (!on) continue;
#pragma unroll
                for (int q = 0; q < 6; ++q) v[q] += vt[q];
                if constexpr (kE)
#pragma unroll
                    for (int q = 0; q < 3; ++q) atomicAdd(&gEs[3 * (i0 + i) + q], -double(vt[q]));
            }
            const T sum = warp_fold8(v);
            const int q = fold8_index(lane);
            double* to = spin && own ? acc_dn + 6 * (ctr - na) : acc + 6 * ctr;
            if ((lane & 3) == 0 && q < 6) atomicAdd(&to[q], q < 3 ? double(sum) : -double(sum));
        }
    }
    __syncthreads();
    for (int q = 3 * na + threadIdx.x; q < 3 * nz; q += blockDim.x) {
        const int a = q / 3, c = q - 3 * a;
        const double dT = own ? acc_dn[6 * (a - na) + c] : 0.0, dJ = own ? acc_dn[6 * (a - na) + 3 + c] : 0.0;
        dEL[(size_t)w * 3 * nn + q] = acc[6 * a + c] + dT + (wk.nlF ? wk.nlF[(size_t)w * 3 * nn + q] : 0.0);
        dlog[(size_t)w * 3 * nn + q] = acc[6 * a + 3 + c] + dJ;
    }
    if constexpr (kE)
        for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) gEdet[(size_t)w * 3 * N + q] = gEs[q];
}

// gtot (may be null): grad_i ln|psi| [W][N][3] of the space-warp form.
template <typename T>
cudaError_t launch_force_prep(const DevSys& s, const DevWalkers& wk, int w0, int W, const double* dvnn, void* Bw,
                              double* gJw, double* accw, double* gtot, int* lossy, cudaStream_t st) {
    if (W == 0) return cudaSuccess;
    const size_t smem = force_head_bytes<T>(s.N, s.n_nuc);
    if (gtot) {
        if (const cudaError_t e = allow_smem(k_force_prep<T, true>, smem)) return e;
        k_force_prep<T, true><<<W, 256, smem, st>>>(s, wk, w0, W, dvnn, (T*)Bw, gJw, accw, gtot, lossy);
        return cudaGetLastError();
    }
    if (const cudaError_t e = allow_smem(k_force_prep<T, false>, smem)) return e;
    k_force_prep<T, false><<<W, 256, smem, st>>>(s, wk, w0, W, dvnn, (T*)Bw, gJw, accw, nullptr, lossy);
    return cudaGetLastError();
}

template <typename T>
static size_t contract_smem(int N, int nn, int parts, bool kE) {
    const int part = (nn + parts - 1) / parts;   // of the largest part
    return ((force_head_bytes<T>(N, nn) + 15) & ~(size_t)15) + (sizeof(T) == 8 ? 8 * kRadialScratch : 0) +
           sizeof(double) * 6 * (size_t)std::min(part, kContractOwn) + (kE ? sizeof(double) * 3 * (size_t)N : 0);
}

// gEdet (may be null): determinant part of dE_L/dr_i [W][N][3] (walker
// index w0 + local) of the space-warp form.
template <typename T>
cudaError_t launch_force_contract(const DevSys& s, const DevWalkers& wk, int w0, int W, const void* Mw, const void* Yw,
                                  const double* gJw, const double* accw, double* dEL, double* dlog, double* gEdet,
                                  cudaStream_t st) {
    if (W == 0) return cudaSuccess;
    if (gEdet) {
        const int parts = contract_parts(W, s.n_nuc, true);
        const size_t smem = contract_smem<T>(s.N, s.n_nuc, parts, true);
        if (const cudaError_t e = allow_smem(k_force_contract<T, true>, smem)) return e;
        k_force_contract<T, true><<<dim3(W, parts), 256, smem, st>>>(s, wk, w0, W, (const T*)Mw, (const T*)Yw, gJw, accw,
                                                                     dEL, dlog, gEdet);
        return cudaGetLastError();
    }
    const int parts = contract_parts(W, s.n_nuc, false);
    const size_t smem = contract_smem<T>(s.N, s.n_nuc, parts, false);
    if (const cudaError_t e = allow_smem(k_force_contract<T, false>, smem)) return e;
    k_force_contract<T, false><<<dim3(W, parts), 256, smem, st>>>(s, wk, w0, W, (const T*)Mw, (const T*)Yw, gJw, accw, dEL,
                                                                  dlog, nullptr);
    return cudaGetLastError();
}

template cudaError_t launch_force_prep<double>(const DevSys&, const DevWalkers&, int, int, const double*, void*,
                                               double*, double*, double*, int*, cudaStream_t);
template cudaError_t launch_force_prep<float>(const DevSys&, const DevWalkers&, int, int, const double*, void*,
                                              double*, double*, double*, int*, cudaStream_t);
template cudaError_t launch_force_contract<double>(const DevSys&, const DevWalkers&, int, int, const void*,
                                                   const void*, const double*, const double*, double*, double*,
                                                   double*, cudaStream_t);
template cudaError_t launch_force_contract<float>(const DevSys&, const DevWalkers&, int, int, const void*, const void*,
                                                  const double*, const double*, double*, double*, double*,
                                                  cudaStream_t);

// gEdet, gtot (both null, or both [W][N][3]): the space-warp form's
// per-electron outputs (see force_walker).
template <typename T>
cudaError_t launch_force(const DevSys& s, const DevWalkers& wk, int W, const double* dvnn, double* Bscr,
                         double* Pscr, double* dEL, double* dlog, double* gEdet, double* gtot, cudaStream_t st) {
    if (W == 0) return cudaSuccess;
    const int nmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    const bool kE = gEdet != nullptr;
    const int nw = ForceShape<T>::warps(s.N, s.n_nuc, nmax, s.n_basis, kE);
    const size_t smem = ForceShape<T>(s.N, s.n_nuc, nmax, s.n_basis, kE, nw).total;
    const auto f = nw == 16 ? (kE ? k_force<T, true, 512> : k_force<T, false, 512>)
                            : (kE ? k_force<T, true, 256> : k_force<T, false, 256>);
    cudaError_t e = allow_smem(f, smem);
    if (e != cudaSuccess) return e;
    f<<<W, 32 * nw, smem, st>>>(s, wk, W, dvnn, Bscr, Pscr, dEL, dlog, gEdet, kE ? gtot : nullptr);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------
// Space warp (Filippi and Umrigar 2000; the paper adapts it to its batched
// force path, Sec. "Single Determinant QMC Forces").  When nucleus a moves
// by dR every electron i moves with it by omega_a(r_i) dR, with
//   omega_a(r) = F(|r - R_a|) / sum_b F(|r - R_b|),  F(d) = d^-4,
// which removes the divergent fluctuations of dE_L/dR_a from electrons near
// nucleus a.  Along coordinate c the warped derivatives are
//   dE_L^w/dR_ac      = dE_L/dR_ac + sum_i omega_a(r_i) dE_L/dr_ic,
//   d ln|psi|^w/dR_ac = d ln|psi|/dR_ac + sum_i omega_a(r_i) d ln|psi|/dr_ic
//                       + 1/2 sum_i d omega_a(r_i)/dr_ic     (Jacobian),
// and they replace the unwarped ones in the force estimator.  The force
// kernels (kE) leave the determinant part of dE_L/dr_i and grad_i ln|psi|;
// this kernel adds the Jastrow and potential parts of dE_L/dr_i,
//   -1/2 d/dr_i sum_j lap_j J - sum_j grad_j ln|psi| . d(grad_j J)/dr_i + dV/dr_i,
// and the warp.  One CTA per walker: a warp per electron over its partners
// (pair terms in T, per-electron sums in T, totals in FP64), then a warp
// per nucleus over the electrons.
// ---------------------------------------------------------------------
template <typename T>
__host__ __device__ inline size_t space_warp_smem(int N, int nn) {
    const size_t b = (force_head_bytes<T>(N, nn) + 15) & ~(size_t)15;
    return b + sizeof(double) * 3 * (size_t)N + sizeof(T) * (size_t)N;
}

// Space warp of walker w (body of k_space_warp and k_space_warp_batch).
// sm: space_warp_smem bytes of dynamic shared memory.
template <typename T>
__device__ __forceinline__ void space_warp_walker(const DevSys& s, const DevWalkers& wk, int w, const double* gEdet,
                                                  const double* gtot, double* dEL, double* dlog, double* sm) {
    const int N = s.N, nu = s.n_up, nn = s.n_nuc;
    const ForceHead<T> h(sm, N, nn);
    double* gEs = (double*)((unsigned char*)sm + ((force_head_bytes<T>(N, nn) + 15) & ~(size_t)15));
    T* Sk = (T*)(gEs + 3 * N);   // [N]    sum_b F(|r_k - R_b|)
    T* gS = h.gJ;                // [N][3] its gradient
    force_load_positions(h, wk.R + (size_t)w * 3 * N, N);
    for (int q = threadIdx.x; q < 3 * N; q += blockDim.x) {
        h.gt[q] = T(gtot[(size_t)w * 3 * N + q]);
        gEs[q] = gEdet[(size_t)w * 3 * N + q];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;

    // Jastrow and potential terms of dE_L/dr_k.  For a pair term u(r),
    // x = r_k - r_j: d(grad u)/dx = hx x x^T + (u'/r) I with
    // hx = (u'' - u'/r)/r^2, d(u'' + 2u'/r)/dx = d3 x with
    // d3 = (u''' + 2u''/r - 2u'/r^2)/r.  An e-e pair changes both electrons'
    // Laplacian terms and both gradients (the partner's with opposite sign).
    for (int k = wid; k < N; k += nw) {
        T v[3] = {T(0), T(0), T(0)};
        const T gk[3] = {h.gt[3 * k], h.gt[3 * k + 1], h.gt[3 * k + 2]};
        for (int j = lane; j < N + nn; j += 32) {
            if (j == k) continue;
            const bool nuc = j >= N;
            T x[3], g[3], a, b, qv, lapf;
            if (!nuc) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    x[c] = off_ee(h, k, j, c);
                    g[c] = gk[c] - h.gt[3 * j + c];
                }
                a = T(((k < nu) == (j < nu)) ? s.a_par : s.a_anti);
                b = T(s.b_ee);
                qv = T(1);       // V_ee = 1/r
                lapf = T(1);
            } else {
                const int c0 = j - N;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    x[c] = off_en(h, s, k, c0, c);
                    g[c] = gk[c];
                }
                a = T(s.a_en[c0]);
                b = T(s.b_en);
                qv = T(-s.Z[c0]);   // V_en = -Z/r
                lapf = T(0.5);
            }
            const T r2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
            const T ir = rsqrt_t(r2), r = r2 * ir;
            T u, du, d2u, d3u;
            pade3<T>(a, b, r, u, du, d2u, d3u);
            const T hx = (d2u - du * ir) * ir * ir;
            const T d3 = (d3u + T(2) * d2u * ir - T(2) * du * ir * ir) * ir;
            const T gdot = g[0] * x[0] + g[1] * x[1] + g[2] * x[2];
            const T vr3 = qv * ir * ir * ir;
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c] += -(lapf * d3 + hx * gdot + vr3) * x[c] - du * ir * g[c];
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] = warp_sum(v[c]);
        if (lane == 0)
            for (int c = 0; c < 3; ++c) gEs[3 * k + c] += double(v[c]);
    }
    // warp normalisation per electron: S = sum_b F_b, grad S = sum_b -4 x_b F_b / d_b^2
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        T S = T(0), g[3] = {T(0), T(0), T(0)};
        for (int b = 0; b < nn; ++b) {
            T x[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) x[c] = off_en(h, s, k, b, c);
            const T d2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
            const T id2 = T(1) / d2;
            const T F = id2 * id2;
            S += F;
#pragma unroll
            for (int c = 0; c < 3; ++c) g[c] += T(-4) * x[c] * F * id2;
        }
        Sk[k] = S;
#pragma unroll
        for (int c = 0; c < 3; ++c) gS[3 * k + c] = g[c];
    }
    __syncthreads();
    // warp of every electron onto nucleus a: grad omega_a = (grad F_a - omega_a grad S) / S
    for (int a = wid; a < nn; a += nw) {
        double dE[3] = {0.0, 0.0, 0.0}, dL[3] = {0.0, 0.0, 0.0};
        for (int k = lane; k < N; k += 32) {
            T x[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) x[c] = off_en(h, s, k, a, c);
            const T d2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
            const T id2 = T(1) / d2;
            const T F = id2 * id2;
            const T iS = T(1) / Sk[k];
            const T om = F * iS;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const T gom = (T(-4) * x[c] * F * id2 - om * gS[3 * k + c]) * iS;
                dE[c] += double(om) * gEs[3 * k + c];
                dL[c] += double(om * h.gt[3 * k + c] + T(0.5) * gom);
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            dE[c] = warp_sum(dE[c]);
            dL[c] = warp_sum(dL[c]);
        }
        if (lane == 0)
            for (int c = 0; c < 3; ++c) {
                dEL[(size_t)w * 3 * nn + 3 * a + c] += dE[c];
                dlog[(size_t)w * 3 * nn + 3 * a + c] += dL[c];
            }
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_space_warp(DevSys s, DevWalkers wk, int W, const double* gEdet,
                                                    const double* gtot, double* dEL, double* dlog) {
    extern __shared__ double sm[];
    const int w = blockIdx.x;
    if (w >= W) return;
    space_warp_walker<T>(s, wk, w, gEdet, gtot, dEL, dlog, sm);
}

template <typename T>
cudaError_t launch_space_warp(const DevSys& s, const DevWalkers& wk, int W, const double* gEdet, const double* gtot,
                              double* dEL, double* dlog, cudaStream_t st) {
    if (W == 0) return cudaSuccess;
    const size_t smem = space_warp_smem<T>(s.N, s.n_nuc);
    if (const cudaError_t e = allow_smem(k_space_warp<T>, smem)) return e;
    k_space_warp<T><<<W, 256, smem, st>>>(s, wk, W, gEdet, gtot, dEL, dlog);
    return cudaGetLastError();
}

template cudaError_t launch_space_warp<double>(const DevSys&, const DevWalkers&, int, const double*, const double*,
                                               double*, double*, cudaStream_t);
template cudaError_t launch_space_warp<float>(const DevSys&, const DevWalkers&, int, const double*, const double*,
                                              double*, double*, cudaStream_t);

// Batched form: persistent CTAs over the walkers of every system.
// kWarp: some member of the batch has the space warp on (its walkers also
// get the per-electron outputs); batches without it run the plain body.
template <typename T, bool kWarp, int kNt>
__global__ void __launch_bounds__(kNt, kNt == 512 ? 1 : 2) k_force_batch(const BatchSys* __restrict__ sys,
                                                                         BatchPlan* plan, int parity, int ctr) {
    extern __shared__ double sm[];
    __shared__ BatchSys bs;
    __shared__ int s_sys, s_idx;
    for (;;) {
        if (threadIdx.x == 0) batch_next(plan, kUnitWalker, ctr, &s_sys, &s_idx);
        __syncthreads();
        const int q = s_sys;
        if (q < 0) break;
        batch_load(&bs, sys + q);
        __syncthreads();
        bool warped = false;
        if constexpr (kWarp) {
            if (bs.space_warp) {
                force_walker<T, true>(bs.s, bs.wk[parity], s_idx, bs.dvnn, bs.Bscr, bs.Pscr, bs.dEL, bs.dlog, sm,
                                      bs.gEdet, bs.gtot);
                warped = true;
            }
        }
        if (!warped) force_walker<T>(bs.s, bs.wk[parity], s_idx, bs.dvnn, bs.Bscr, bs.Pscr, bs.dEL, bs.dlog, sm);
        __syncthreads();
    }
}

int force_batch_warps(const DevSys& s, int elem, int space_warp) {
    const int nmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    return elem == 4 ? ForceShape<float>::warps(s.N, s.n_nuc, nmax, s.n_basis, space_warp != 0)
                     : ForceShape<double>::warps(s.N, s.n_nuc, nmax, s.n_basis, space_warp != 0);
}

size_t force_batch_smem_bytes(const DevSys& s, int elem, int space_warp, int nw) {
    const int nmax = s.n_up > s.n_dn ? s.n_up : s.n_dn;
    return elem == 4 ? ForceShape<float>(s.N, s.n_nuc, nmax, s.n_basis, space_warp != 0, nw).total
                     : ForceShape<double>(s.N, s.n_nuc, nmax, s.n_basis, space_warp != 0, nw).total;
}

template <typename T>
static auto force_batch_kernel(int any_warp, int nw) {
    return nw == 16 ? (any_warp ? k_force_batch<T, true, 512> : k_force_batch<T, false, 512>)
                    : (any_warp ? k_force_batch<T, true, 256> : k_force_batch<T, false, 256>);
}

// Batched space warp: persistent CTAs over the walkers of every system; the
// walkers of systems without the warp are skipped.
template <typename T>
__global__ void __launch_bounds__(256) k_space_warp_batch(const BatchSys* __restrict__ sys, BatchPlan* plan,
                                                          int parity, int ctr) {
    extern __shared__ double sm[];
    __shared__ BatchSys bs;
    __shared__ int s_sys, s_idx;
    for (;;) {
        if (threadIdx.x == 0) batch_next(plan, kUnitWalker, ctr, &s_sys, &s_idx);
        __syncthreads();
        const int q = s_sys;
        if (q < 0) break;
        batch_load(&bs, sys + q);
        __syncthreads();
        if (bs.space_warp)
            space_warp_walker<T>(bs.s, bs.wk[parity], s_idx, bs.gEdet, bs.gtot, bs.dEL, bs.dlog, sm);
        __syncthreads();
    }
}

size_t space_warp_batch_smem_bytes(const DevSys& s, int elem) {
    return elem == 4 ? space_warp_smem<float>(s.N, s.n_nuc) : space_warp_smem<double>(s.N, s.n_nuc);
}

template <typename T>
int space_warp_batch_prepare(size_t smem) {
    int nb = 0;
    if (allow_smem(k_space_warp_batch<T>, smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_space_warp_batch<T>, 256, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

template <typename T>
cudaError_t launch_space_warp_batch(const BatchSys* sys, BatchPlan* plan, int parity, int ctr, int grid, size_t smem,
                                    cudaStream_t st) {
    k_space_warp_batch<T><<<grid, 256, smem, st>>>(sys, plan, parity, ctr);
    return cudaGetLastError();
}

template int space_warp_batch_prepare<double>(size_t);
template int space_warp_batch_prepare<float>(size_t);
template cudaError_t launch_space_warp_batch<double>(const BatchSys*, BatchPlan*, int, int, int, size_t,
                                                     cudaStream_t);
template cudaError_t launch_space_warp_batch<float>(const BatchSys*, BatchPlan*, int, int, int, size_t, cudaStream_t);

template <typename T>
int force_batch_prepare(size_t smem, int any_warp, int nw) {
    int nb = 0;
    const void* f = (const void*)force_batch_kernel<T>(any_warp, nw);
    if (allow_smem(f, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, 32 * nw, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

template <typename T>
cudaError_t launch_force_batch(const BatchSys* sys, BatchPlan* plan, int parity, int ctr, int grid, size_t smem,
                               int any_warp, int nw, cudaStream_t st) {
    force_batch_kernel<T>(any_warp, nw)<<<grid, 32 * nw, smem, st>>>(sys, plan, parity, ctr);
    return cudaGetLastError();
}

template int force_batch_prepare<double>(size_t, int, int);
template int force_batch_prepare<float>(size_t, int, int);
template cudaError_t launch_force_batch<double>(const BatchSys*, BatchPlan*, int, int, int, size_t, int, int,
                                                cudaStream_t);
template cudaError_t launch_force_batch<float>(const BatchSys*, BatchPlan*, int, int, int, size_t, int, int,
                                               cudaStream_t);

template cudaError_t launch_force<double>(const DevSys&, const DevWalkers&, int, const double*, double*, double*,
                                          double*, double*, double*, double*, cudaStream_t);
template cudaError_t launch_force<float>(const DevSys&, const DevWalkers&, int, const double*, double*, double*,
                                         double*, double*, double*, double*, cudaStream_t);

}  // namespace qmc
