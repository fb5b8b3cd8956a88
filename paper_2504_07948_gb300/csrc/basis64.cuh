// FP64 basis and orbital contraction of one electron position by one CTA
// (Eq. 2), built around the FP64 pipe: on GB300 an FP64 instruction of a warp
// takes 16 SM cycles however few lanes are active, so every FP64 step runs on
// a list that fills its warps and the contraction runs in fixed point
// (fixed64.cuh).
//
//   1. offsets and r^2 from every nucleus (a thread per nucleus);
//   2. the unscreened primitives and shells are listed (FP32 test; a pair at
//      the threshold is below 1e-26 either way);
//   3. one exponential per listed primitive;
//   4. radial sums per listed shell, whose functions are listed by angular
//      momentum so that a warp holds functions of one kind;
//   5. value, gradient and Laplacian of the listed functions, split into
//      limbs with one scale per component;
//   6. phi[c][j] = sum_r C[row_r][j] bas[c][r], three 32-bit multiply-adds per
//      term, slices of the rows on neighbouring lanes; rows without high limbs
//      (below 2^-28 of the component's largest) take one, rows of zeros none: on
//      the 32-water cluster 157 of an electron's 340 listed functions have high
//      limbs and 60 are zero.
// Bound by instruction issue (45 % with 15 to 20 warps on an SM: registers and
// shared memory allow four CTAs of five warps, so the primitives' arrays share
// their place with the functions') and by the FP64 pipe (50 % at 30 orbitals).
// Rebuild of the 32-water cluster, 256 walkers: 51 -> 9.3 ms against a masked
// basis and FP64 chains (17 ms with every listed row in three products and two
// CTAs per SM); 6-water cluster, 512 walkers: 1.64 -> 0.86 ms (before
// the split by limbs).
// The lists are filled in any order: every sum over them is exact integer
// arithmetic, so the result does not depend on it.
//
// Accuracy: the contraction's error is about sqrt(rows) 2^-60 of the largest
// basis value times the orbital's largest coefficient.  Where no orbital of
// the block reaches 2^-4 of that (occupied orbitals without weight on the
// functions that are large at this point), orbitals64 takes the orbitals
// again in FP64, so that the row of orbital values keeps the accuracy of an
// FP64 sum relative to its largest entry.  Where a row's smaller entries decide,
// its users find out from the inverse (k_wavefunction.cu, sweep64.cuh).
#pragma once

#include "fixed64.cuh"
#include "qmc_internal.cuh"

namespace qmc {

struct Basis64Layout {
    size_t nuc, ev, fs, bas, tf, plist, slist, flist, rows, cnt, total;
    int ldb;
    __host__ __device__ Basis64Layout(int n_nuc, int n_prim, int n_shell, int n_basis) {
        ldb = (n_basis + 1) & ~1;
        size_t o = 0;
        nuc = o;
        o += sizeof(double) * 4 * (size_t)n_nuc;
        fs = o;
        o += sizeof(double) * 3 * (size_t)n_shell;
        flist = o;
        o += sizeof(int) * (size_t)n_basis;
        rows = o;
        o += sizeof(int) * (size_t)n_basis;
        cnt = o;
        o += sizeof(int) * 32;
        o = (o + 15) & ~(size_t)15;
        // the primitives' lists and exponentials end before the functions begin
        bas = o;
        ev = o;
        tf = ev + sizeof(double) * (size_t)n_prim;
        plist = tf + sizeof(float) * (size_t)n_nuc;
        slist = plist + sizeof(int) * (size_t)n_prim;
        const size_t prim = slist + sizeof(int) * (size_t)n_shell, fns = bas + sizeof(double) * 5 * (size_t)ldb;
        o = prim > fns ? prim : fns;
        total = (o + 15) & ~(size_t)15;
    }
};

// Largest layout used: 227 KB less the static shared memory of the batched
// kernels.
constexpr size_t kBasis64Max = 224 * 1024;

// Steps 1 to 5 at position (r0, r1, r2).  Leaves the limbs in bas [5][ldb]
// (int2) and their entries (function << 16 | row) in flist: cnt[5] rows with some
// high limb from its front, cnt[6] with low limbs only from its back; rows of
// zeros are left out.  The components' scales are fx_scale(cnt[8 + c]).  All
// threads call; ends synchronised.  nuc: the nuclear offsets (x, y, z, r^2) stay valid after it.
__device__ __forceinline__ void basis64(const DevSys& s, const Basis64Layout& L, unsigned char* sm, double r0, double r1,
                                       double r2) {
    double4* nuc = (double4*)(sm + L.nuc);
    double* ev = (double*)(sm + L.ev);
    double* fs = (double*)(sm + L.fs);
    double* bas = (double*)(sm + L.bas);
    float* tf = (float*)(sm + L.tf);
    int* plist = (int*)(sm + L.plist);
    int* slist = (int*)(sm + L.slist);
    int* flist = (int*)(sm + L.flist);   // functions by kind: s from 0, p from n_fn_s, d from n_fn_s + n_fn_p
    int* rows = (int*)(sm + L.rows);
    int* cnt = (int*)(sm + L.cnt);       // [0] primitives, [1] shells, [2..4] functions by kind, [5], [6] rows,
                                         // [8..12] exponents,
                                         // [16..20], [24..28] exponents of the sums (orbitals64),
                                         // [29], [30] of the ratio's factors and terms (sweep64.cuh)
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, ldb = L.ldb;
    const unsigned below = (1u << lane) - 1u;
    for (int q = tid; q < 32; q += nt) cnt[q] = 0;
    for (int a = tid; a < s.n_nuc; a += nt) {
        const double x = r0 - s.Rn[3 * a], y = r1 - s.Rn[3 * a + 1], z = r2 - s.Rn[3 * a + 2];
        const double t = x * x + y * y + z * z;
        nuc[a] = make_double4(x, y, z, t);
        tf[a] = (float)t;   // a conversion costs the FP64 pipe as much as an addition
    }
    __syncthreads();
    const float cut = (float)kScreenExponent;
    for (int p0 = tid - lane; p0 < s.n_prim; p0 += nt) {
        const int p = p0 + lane;
        const bool live = p < s.n_prim && !(s.alpha_f[p] * tf[s.prim_ctr[p]] > cut);
        const unsigned m = __ballot_sync(0xffffffffu, live);
        int base = 0;
        if (lane == 0 && m) base = atomicAdd(&cnt[0], __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (live) plist[base + __popc(m & below)] = p;
    }
    for (int q0 = tid - lane; q0 < s.n_shell; q0 += nt) {
        const int sh = q0 + lane;
        const bool live = sh < s.n_shell && !(s.shell_amin_f[sh] * tf[s.shell[sh].x] > cut);
        const unsigned m = __ballot_sync(0xffffffffu, live);
        int base = 0;
        if (lane == 0 && m) base = atomicAdd(&cnt[1], __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (live) slist[base + __popc(m & below)] = sh;
    }
    __syncthreads();
    for (int k = tid; k < cnt[0]; k += nt) {
        const int p = plist[k];
        ev[p] = s.cn[p] * exp(-s.alpha[p] * nuc[s.prim_ctr[p]].w);
    }
    __syncthreads();
    for (int k = tid; k < cnt[1]; k += nt) {
        const int sh = slist[k];
        const int4 d = s.shell[sh];
        const double t = nuc[d.x].w;
        const float tc = tf[d.x];
        double f0 = 0.0, f1 = 0.0, f2 = 0.0;
        for (int p = d.z; p < d.z + d.w; ++p) {
            if (s.alpha_f[p] * tc > cut) continue;
            const double a = s.alpha[p], e = ev[p], e1 = a * e;
            f0 += e;
            f1 -= e1;
            f2 += a * e1;
        }
        // f0, 2 f1 and the radial part of the Laplacian with its 2 grad P . grad S
        // term folded in (grad P . x = l P): lap = P (6 f1 + 4 t f2 + 4 l f1) + f0 lap P
        const int l = d.y & 0xff, nf = shell_nfn(l, d.y >> 8);
        fs[3 * sh] = f0;
        fs[3 * sh + 1] = 2.0 * f1;
        fs[3 * sh + 2] = (double)(6 + 4 * l) * f1 + 4.0 * t * f2;
        const int o = atomicAdd(&cnt[2 + l], nf) + (l > 0 ? s.n_fn_s : 0) + (l > 1 ? s.n_fn_p : 0);
        for (int f = 0; f < nf; ++f) flist[o + f] = sh * 8 + f;
    }
    __syncthreads();
    // functions of one kind per warp: the kinds' segments padded to 32
    const int ns = cnt[2], np = cnt[3], nd = cnt[4];
    const int e0 = (ns + 31) & ~31, e1 = e0 + ((np + 31) & ~31), e2 = e1 + nd;
    int mx[5] = {0, 0, 0, 0, 0};
    for (int o = tid; o < e2; o += nt) {
        const int kind = o < e0 ? 0 : o < e1 ? 1 : 2;
        const int q = o - (kind == 0 ? 0 : kind == 1 ? e0 : e1);
        if (q >= (kind == 0 ? ns : kind == 1 ? np : nd)) continue;
        const int ent = flist[q + (kind == 0 ? 0 : kind == 1 ? s.n_fn_s : s.n_fn_s + s.n_fn_p)];
        const int sh = ent >> 3, f = ent & 7;
        const int4 d = s.shell[sh];
        const double4 x = nuc[d.x];
        const double f0 = fs[3 * sh], g1 = fs[3 * sh + 1], gl = fs[3 * sh + 2];
        double v[5];
        if (kind == 0) {
            v[0] = f0;
            v[1] = x.x * g1;
            v[2] = x.y * g1;
            v[3] = x.z * g1;
            v[4] = gl;
        } else if (kind == 1) {
            const double P = f == 0 ? x.x : f == 1 ? x.y : x.z, Pg = P * g1;
            v[0] = P * f0;
            v[1] = fma(x.x, Pg, f == 0 ? f0 : 0.0);
            v[2] = fma(x.y, Pg, f == 1 ? f0 : 0.0);
            v[3] = fma(x.z, Pg, f == 2 ? f0 : 0.0);
            v[4] = P * gl;
        } else {
            // sqrt3 u v of two coordinates, or a x^2 + b y^2 + c z^2 (gradient
            // 2 (a x, b y, c z)); Cartesian squares are not harmonic (tr H)
            const double s3 = 1.7320508075688772;
            const bool pure = (d.y >> 8) != 0;
            const int uv = pure ? (f == 0 ? 1 : f == 1 ? 6 : f == 3 ? 2 : 0)      // 3 u + v of (0, 1), (1, 2), (0, 2)
                                : (f == 1 ? 1 : f == 2 ? 2 : f == 4 ? 6 : 0);
            double P, gx, gy, gz, tr = 0.0;
            if (uv) {
                const double su = s3 * (uv == 6 ? x.y : x.x), vv = uv == 1 ? x.y : x.z, sv = s3 * vv;
                P = su * vv;
                gx = uv == 6 ? 0.0 : sv;
                gy = uv == 1 ? su : uv == 6 ? sv : 0.0;
                gz = uv == 1 ? 0.0 : su;
            } else {
                const double a = pure ? (f == 2 ? -1.0 : s3) : (f == 0 ? 2.0 : 0.0);
                const double b = pure ? (f == 2 ? -1.0 : -s3) : (f == 3 ? 2.0 : 0.0);
                const double c = pure ? (f == 2 ? 2.0 : 0.0) : (f == 5 ? 2.0 : 0.0);
                gx = a * x.x;
                gy = b * x.y;
                gz = c * x.z;
                P = 0.5 * (gx * x.x + gy * x.y + gz * x.z);
                tr = pure ? 0.0 : 2.0;
            }
            const double Pg = P * g1;
            v[0] = P * f0;
            v[1] = x.x * Pg + gx * f0;
            v[2] = x.y * Pg + gy * f0;
            v[3] = x.z * Pg + gz * f0;
            v[4] = P * gl;
            if (!pure) v[4] += tr * f0;
        }
        const int r = q + (kind == 0 ? 0 : kind == 1 ? ns : ns + np);
        rows[r] = s.shell_fn[sh] + f;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            bas[c * ldb + r] = v[c];
            mx[c] = max(mx[c], fx_expo(v[c]));
        }
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        const int m = warp_max_u(mx[c]);
        if (lane == 0 && m) atomicMax(&cnt[8 + c], m);
    }
    __syncthreads();
    const int nrow = ns + np + nd;
    int em[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) em[c] = cnt[8 + c];
    for (int r0 = tid - lane; r0 < nrow; r0 += nt) {
        const int r = r0 + lane;
        int hi = 0, lo = 0;
        if (r < nrow)
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                const int2 v = fx_limbs(bas[c * ldb + r], em[c]);
                ((int2*)bas)[c * ldb + r] = v;
                hi |= v.x;
                lo |= v.y;
            }
        // (the function lists are used up: their place takes the entries)
        const unsigned mh = __ballot_sync(0xffffffffu, hi != 0), ml = __ballot_sync(0xffffffffu, hi == 0 && lo != 0);
        int bh = 0, bl = 0;
        if (lane == 0) {
            bh = mh ? atomicAdd(&cnt[5], __popc(mh)) : 0;
            bl = ml ? atomicAdd(&cnt[6], __popc(ml)) : 0;
        }
        bh = __shfl_sync(0xffffffffu, bh, 0) + __popc(mh & below);
        bl = __shfl_sync(0xffffffffu, bl, 0) + __popc(ml & below);
        if (hi)
            flist[bh] = rows[r] << 16 | r;
        else if (lo)
            flist[s.n_basis - 1 - bl] = rows[r] << 16 | r;
    }
    __syncthreads();
}

// Step 6: put(c, j, phi_cj) for c < 5 and every orbital j < n of a
// coefficient block given as limbs Ck [n_basis][n] with the orbitals' scales
// sC [n].  S lanes share an orbital, each taking every S-th row: as many as
// keep n S within the CTA.  big: five counters (zero before the call) that
// receive the largest exponent of the integer sums per component.
template <typename Put>
__device__ __forceinline__ void contract64(const Basis64Layout& L, const unsigned char* sm, int nb,
                                           const int2* __restrict__ Ck, const double* __restrict__ sC, int n, int* big,
                                           Put put) {
    const int2* bas = (const int2*)(sm + L.bas);
    const int* list = (const int*)(sm + L.flist);
    const int* cnt = (const int*)(sm + L.cnt);
    const int ldb = L.ldb, nh = cnt[5], nl = cnt[6];
    int lg = 4;
    while (lg > 0 && (n << lg) > (int)blockDim.x) --lg;
    const int S = 1 << lg, items = (n << lg);
    int mx[5] = {0, 0, 0, 0, 0};
    for (int o0 = threadIdx.x & ~31; o0 < items; o0 += blockDim.x) {   // whole warps
        const int o = o0 + (threadIdx.x & 31), sl = o & (S - 1);
        const int j = min(o >> lg, n - 1);
        FxSum sum[5];
        for (int r0 = sl; r0 < nh; r0 += kFxBlock * S) {
            FxDot d[5];
            const int r1 = min(nh, r0 + kFxBlock * S);
#pragma unroll 4
            for (int r = r0; r < r1; r += S) {
                const int e = list[r];
                const int2 cv = Ck[(e >> 16) * n + j];
                const int2* b = bas + (e & 0xffff);
#pragma unroll
                for (int c = 0; c < 5; ++c) d[c].add(cv, b[c * ldb]);
            }
#pragma unroll
            for (int c = 0; c < 5; ++c) sum[c].fold(d[c]);
        }
        // without high limbs one product of the three is left
        for (int r0 = sl; r0 < nl; r0 += kFxBlock * S) {
            FxDot d[5];
            const int r1 = min(nl, r0 + kFxBlock * S);
#pragma unroll 4
            for (int r = r0; r < r1; r += S) {
                const int e = list[nb - 1 - r];
                const int ch = Ck[(e >> 16) * n + j].x;
                const int2* b = bas + (e & 0xffff);
#pragma unroll
                for (int c = 0; c < 5; ++c) d[c].mid += (long long)ch * b[c * ldb].y;
            }
#pragma unroll
            for (int c = 0; c < 5; ++c) sum[c].fold(d[c]);
        }
        for (int k = 1; k < S; k <<= 1)
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                sum[c].hi += __shfl_xor_sync(0xffffffffu, sum[c].hi, k);
                sum[c].lo += __shfl_xor_sync(0xffffffffu, sum[c].lo, k);
                sum[c].rem += __shfl_xor_sync(0xffffffffu, sum[c].rem, k);
            }
        if (o >= items) continue;
        const double sj = sC[j];
#pragma unroll
        for (int c = 0; c < 5; ++c)
            if ((c & (S - 1)) == sl) {   // every lane takes its share of the outputs
                const double v = sum[c].value();
                mx[c] = max(mx[c], fx_expo(v));
                put(c, j, v * sj * fx_scale(cnt[8 + c]));
            }
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        const int m = warp_max_u(mx[c]);
        if ((threadIdx.x & 31) == 0 && m) atomicMax(&big[c], m);
    }
}

// The same orbitals from every basis function in FP64 (bas: 5 n_basis doubles
// of shared memory).  Starts and ends synchronised.
template <typename Put>
__device__ __noinline__ void orbitals_plain(const DevSys& s, const double r[3], const double* __restrict__ C, int n,
                                            double* bas, Put put) {
    const int nb = s.n_basis;
    __syncthreads();
    for (int sh = threadIdx.x; sh < s.n_shell; sh += blockDim.x) shell_vgl<double>(s, sh, r, bas, nb);
    __syncthreads();
    for (int o = threadIdx.x; o < 5 * n; o += blockDim.x) {
        const int c = o / n, j = o - c * n;
        double acc = 0.0;
        for (int l = 0; l < nb; ++l) acc += C[(size_t)l * n + j] * bas[c * nb + l];
        put(c, j, acc);
    }
    __syncthreads();
}

// Basis and orbitals at (r0, r1, r2) of one or two (C2, n2 > 0) coefficient
// blocks, all threads; ends synchronised.  The first block's nuclear offsets
// stay in nuc (basis64).  Returns whether the orbitals are FP64 sums (uniform).
template <typename Put, typename Put2>
__device__ __forceinline__ bool orbitals64(const DevSys& s, const Basis64Layout& L, unsigned char* sm, double r0,
                                           double r1, double r2, const int2* Ck, const double* sC, const double* C,
                                           int n, Put put, const int2* Ck2, const double* sC2, const double* C2, int n2,
                                           Put2 put2) {
    int* cnt = (int*)(sm + L.cnt);
    basis64(s, L, sm, r0, r1, r2);
    contract64(L, sm, s.n_basis, Ck, sC, n, cnt + 16, put);
    if (n2 > 0) contract64(L, sm, s.n_basis, Ck2, sC2, n2, cnt + 24, put2);
    __syncthreads();
    // integer sums of the largest possible product: 2^56 (biased 1079)
    bool low = false, low2 = false;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        const int e = cnt[8 + c];
        if (e == 0 || e == 2047) continue;   // an all-zero component, or not finite
        low |= cnt[16 + c] < 1079 - 4;
        low2 |= cnt[24 + c] < 1079 - 4;
    }
    low |= low2 && n2 > 0;
    if (low) {
        const double r[3] = {r0, r1, r2};
        orbitals_plain(s, r, C, n, (double*)(sm + L.bas), put);
        if (n2 > 0) orbitals_plain(s, r, C2, n2, (double*)(sm + L.bas), put2);
    }
    return low;
}

}  // namespace qmc
