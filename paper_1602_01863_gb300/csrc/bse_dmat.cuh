// Small dense complex matrices (n <= BSE_MAX_BANDS, row-major double2 arrays in
// shared memory) worked on by G lanes, shared by the set-up kernels (band
// gauge) and the pair-data kernel of the learned residual.
#pragma once

#include "bse_internal.cuh"

constexpr int kGaugeLanes = 16;                     // lanes per matrix, unless the bands are few
constexpr int kGaugeMats = 6;                       // n x n matrices of scratch grp_gauge needs

// The G (a power of two) lanes that work with the calling lane, as a sync mask, and its place among them.
template <int G = kGaugeLanes>
__device__ inline unsigned grp_mask() { return (G == 32 ? 0xffffffffu : (1u << G) - 1u) << (threadIdx.x & 31 & ~(G - 1)); }
template <int G = kGaugeLanes>
__device__ inline int grp_lane() { return threadIdx.x & (G - 1); }

// C = A B by G lanes, an entry per lane and round.
template <int G>
__device__ inline void grp_mul(const double2* A, const double2* B, double2* C, int n) {
    for (int e = grp_lane<G>(); e < n * n; e += G) {
        const int i = e / n, j = e - i * n;
        double2 s = make_double2(0.0, 0.0);
        for (int k = 0; k < n; ++k) {
            const double2 a = A[i * n + k], b = B[k * n + j];
            s.x = fma(a.x, b.x, fma(-a.y, b.y, s.x));
            s.y = fma(a.x, b.y, fma(a.y, b.x, s.y));
        }
        C[e] = s;
    }
    __syncwarp(grp_mask<G>());
}

// Band gauge U(k) = expm(i sum_a [sin(2 pi k_a) G_a0 + (1 - cos 2 pi k_a) G_a1]) from
// sn[a] = sin(2 pi k_a), cs[a] = cos(2 pi k_a), by G lanes; the
// result's address (inside `work`, kGaugeMats n^2 entries of shared memory) is returned.
// Scaling and squaring of the Taylor polynomial of degree 15 (||X||_F <= 1/2: the
// remainder is below 1e-18), evaluated in powers of X^4 (Paterson-Stockmeyer): six
// products and the squarings instead of one product per term, each with an
// entry per lane: one thread per matrix spent 24 products in local memory.
template <int G = kGaugeLanes>
__device__ inline const double2* grp_gauge(const double2* gen, int n, const double* sn, const double* cs, double2* work) {
    const int nn = n * n, ln = grp_lane<G>();
    const unsigned mask = grp_mask<G>();
    double2 *X = work, *X2 = X + nn, *X3 = X2 + nn, *X4 = X3 + nn, *E = X4 + nn, *T = E + nn;
    double fro = 0.0;
    for (int e = ln; e < nn; e += G) {
        double2 a = make_double2(0.0, 0.0);
        for (int ax = 0; ax < 3; ++ax) {
            const double2 g0 = gen[(ax * 2 + 0) * nn + e], g1 = gen[(ax * 2 + 1) * nn + e];
            a.x += sn[ax] * g0.x + (1.0 - cs[ax]) * g1.x;
            a.y += sn[ax] * g0.y + (1.0 - cs[ax]) * g1.y;
        }
        fro += a.x * a.x + a.y * a.y;
        X[e] = make_double2(-a.y, a.x);                       // i A
    }
    for (int o = G / 2; o > 0; o >>= 1) fro += __shfl_xor_sync(mask, fro, o);
    fro = sqrt(fro);
    int s = 0;
    while (fro > 0.5 && s < 1000) { fro *= 0.5; ++s; }
    const double sc = ldexp(1.0, -s);
    for (int e = ln; e < nn; e += G) X[e] = cscale(X[e], sc);
    __syncwarp(mask);
    grp_mul<G>(X, X, X2, n);
    grp_mul<G>(X2, X, X3, n);
    grp_mul<G>(X2, X2, X4, n);
    // E = B_3, then E <- X^4 E + B_j, B_j = sum_{i < 4} X^i / (4 j + i)!
    double inv[16];
    inv[0] = 1.0;
#pragma unroll
    for (int k = 1; k < 16; ++k) inv[k] = inv[k - 1] / k;
#pragma unroll
    for (int j = 3; j >= 0; --j) {
        if (j < 3) grp_mul<G>(X4, E, T, n);
        for (int e = ln; e < nn; e += G) {
            double2 v = j < 3 ? T[e] : make_double2(0.0, 0.0);
            v = cadd(v, cadd(cadd(cscale(X3[e], inv[4 * j + 3]), cscale(X2[e], inv[4 * j + 2])), cscale(X[e], inv[4 * j + 1])));
            if (e / n == e % n) v.x += inv[4 * j];
            E[e] = v;
        }
        __syncwarp(mask);
    }
    for (int q = 0; q < s; ++q) {
        grp_mul<G>(E, E, T, n);
        double2* x = E;
        E = T;
        T = x;
    }
    return E;
}

// out[G][x][c] = sum_{m, m'} conj(Uv[m][x]) in[G][m][m'] Uc[m'][c] (FORM), or with Uv and
// conj(Uc) (dipoles): both factors of a block of `cnt` nv x nc matrices, threads tid, tid + nthr, ...;
// `sync` separates the two steps.  In place is not allowed for tmp; out may be in.
template <bool FORM, typename Sync>
__device__ inline void rotate_forms(const double2* in, const double2* Uv, const double2* Uc, double2* tmp, double2* out,
                                    int cnt, int nv, int nc, int tid, int nthr, Sync sync) {
    const int t = nv * nc;
    for (int i = tid; i < cnt * t; i += nthr) {
        const int g = i / t, e = i - g * t, x = e / nc, mp = e - x * nc;
        double2 s = make_double2(0.0, 0.0);
        for (int m = 0; m < nv; ++m) {
            const double2 u = Uv[m * nv + x];
            s = cadd(s, cmul(FORM ? conjg(u) : u, in[g * t + m * nc + mp]));
        }
        tmp[i] = s;
    }
    sync();
    for (int i = tid; i < cnt * t; i += nthr) {
        const int g = i / t, e = i - g * t, x = e / nc, c = e - x * nc;
        double2 s = make_double2(0.0, 0.0);
        for (int mp = 0; mp < nc; ++mp) {
            const double2 u = Uc[mp * nc + c];
            s = cadd(s, cmul(tmp[g * t + x * nc + mp], FORM ? u : conjg(u)));
        }
        out[i] = s;
    }
    sync();
}
