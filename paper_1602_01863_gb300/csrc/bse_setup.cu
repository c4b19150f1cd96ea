// Set-up kernels: band gauge, coarse kernel K_c, dense tables, M3 tables.
//
// Everything the Haydock loop reads is built here on the device, from the
// model parameters alone (Sec. 2 model inputs, Sec. 3 double-grid tables).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "bse_dmat.cuh"
#include "bse_internal.cuh"

namespace {

constexpr double kPi = 3.14159265358979323846;

// Integer coordinates of point p of an (n * nd)^3 grid in coarse-major order.
__device__ inline Int3 point_ints(int p, int n, int nd) {
    const int Ndiv = nd * nd * nd;
    const Int3 i = unflat3(p / Ndiv, n), j = unflat3(p % Ndiv, nd);
    return Int3{i.a * nd + j.a, i.b * nd + j.b, i.c * nd + j.c};
}

// Coarse band gauge U(k~), both manifolds: a warp per point, a half warp each.
__global__ void __launch_bounds__(128) k_gauge(const double2* __restrict__ gen_v, const double2* __restrict__ gen_c, int nv,
                                               int nc, int n, double2* __restrict__ Uv, double2* __restrict__ Uc) {
    extern __shared__ double2 gsm[];
    const int warp = threadIdx.x >> 5, half = (threadIdx.x >> 4) & 1, p = blockIdx.x * 4 + warp;
    if (p >= n * n * n) return;
    double2* work = gsm + (size_t)warp * kGaugeMats * (nv * nv + nc * nc) + (half ? kGaugeMats * nv * nv : 0);
    const Int3 g = unflat3(p, n);
    double sn[3], cs[3];
    sincospi(2.0 * g.a / n, &sn[0], &cs[0]);
    sincospi(2.0 * g.b / n, &sn[1], &cs[1]);
    sincospi(2.0 * g.c / n, &sn[2], &cs[2]);
    const int nb = half ? nc : nv;
    const double2* E = grp_gauge(half ? gen_c : gen_v, nb, sn, cs, work);
    double2* out = (half ? Uc : Uv) + (size_t)p * nb * nb;
    for (int e = grp_lane(); e < nb * nb; e += kGaugeLanes) out[e] = E[e];
}

// Minimum-image shape tables over all index differences of an L^3 grid:
// mode 0: h(q) = sum_G exp(-|G|^2) 4 pi / (|q + G|^2 + kappa^2) over `shells` G;
// mode 1: head 1 / (|q|^2 + kappa^2).  Ties (difference L/2) average the images.
// A warp per difference: the lanes share the images' G sums.
__global__ void __launch_bounds__(128) k_shape_table(int L, double kappa, int shells, int h_const, double h0, int mode,
                                                     double* __restrict__ out) {
    const int idx = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (idx >= L * L * L) return;
    if (mode == 0 && h_const) {
        if (lane == 0) out[idx] = h0;
        return;
    }
    const Int3 d = unflat3(idx, L);
    const int dd[3] = {d.a, d.b, d.c};
    // half-way differences have two images; the others count both as the same one
    int im[3][2], nimg = 1;
    for (int a = 0; a < 3; ++a) {
        im[a][0] = 2 * dd[a] > L ? dd[a] - L : dd[a];
        im[a][1] = 2 * dd[a] >= L ? dd[a] - L : dd[a];
        if (im[a][0] != im[a][1]) nimg *= 2;
    }
    const int nG = mode == 1 ? 1 : 27;
    double acc = 0.0;
    for (int q = lane; q < 8 * nG; q += 32) {
        const int s = q / nG, G = mode == 1 ? 13 : q - s * nG;
        // count every distinct image once
        bool dup = false;
        for (int a = 0; a < 3; ++a) dup = dup || (((s >> a) & 1) && im[a][0] == im[a][1]);
        const int ga = G / 9 - 1, gb = (G / 3) % 3 - 1, gc = G % 3 - 1, g2 = ga * ga + gb * gb + gc * gc;
        if (dup || (mode == 0 && shells == 1 && g2 != 0)) continue;
        const double qa = (double)im[0][s & 1] / L + ga, qb = (double)im[1][(s >> 1) & 1] / L + gb,
                     qc = (double)im[2][s >> 2] / L + gc, r = qa * qa + qb * qb + qc * qc + kappa * kappa;
        acc += mode == 1 ? 1.0 / r : exp(-(double)g2) * 4.0 * kPi / r;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) out[idx] = acc / nimg;
}

// Exchange form factors on the coarse mesh: M_vc(k~, G) = [U_v^H mu(k~, G) U_c]_vc, one
// block per coarse point: mu(k~) from its harmonics once, then one gauge factor
// at a time (together 7 + nv + nc terms per entry instead of 7 nv nc).
__global__ void __launch_bounds__(256) k_form_factors(const double2* __restrict__ Uv, const double2* __restrict__ Uc,
                                                      const double2* __restrict__ mu, int n, int nv, int nc,
                                                      double2* __restrict__ M) {
    extern __shared__ double2 fsm[];
    const int ic = blockIdx.x, t = nv * nc, tid = threadIdx.x;
    double2 *a = fsm, *b = a + 26 * t, *uv = b + 26 * t, *uc = uv + nv * nv;
    for (int e = tid; e < nv * nv; e += 256) uv[e] = Uv[(size_t)ic * nv * nv + e];
    for (int e = tid; e < nc * nc; e += 256) uc[e] = Uc[(size_t)ic * nc * nc + e];
    const Int3 g = unflat3(ic, n);
    double c[7];
    c[0] = 1.0;
    sincospi(2.0 * g.a / n, &c[2], &c[1]);
    sincospi(2.0 * g.b / n, &c[4], &c[3]);
    sincospi(2.0 * g.c / n, &c[6], &c[5]);
    for (int e = tid; e < 26 * t; e += 256) {
        double2 s = make_double2(0.0, 0.0);
#pragma unroll
        for (int h = 0; h < 7; ++h) s = cadd(s, cscale(mu[(size_t)h * 26 * t + e], c[h]));
        a[e] = s;
    }
    __syncthreads();
    rotate_forms<true>(a, uv, uc, b, M + (size_t)ic * 26 * t, 26, nv, nc, tid, 256, [] { __syncthreads(); });
}

// K_c element (Eq. bse2 in the model, coarse weight e_k / n^3):
//   K = pref [ 2 sum_G v(G) conj(M_i(G)) M_j(G) - O^v O^c h(k~_i - k~_j) / eps_inf ].
// A block takes the entries of P x P coarse points (at most 64 x 64 entries),
// on and above the diagonal only; each value is also written, conjugated, to
// its mirror image; the diagonal is real.  FP64 bounds it (1.25 TFLOP/s on GB300), so
// the work per entry is cut: the overlaps are formed once per pair of points, half of
// the matrix is never computed, and where K_c is rounded to FP32 or BF16 the exchange
// sum takes three real products per G (re = S1 + S2, im = S3 - S1 + S2 with
// S1 = sum a_r b_r, S2 = sum a_i b_i, S3 = sum (a_r - a_i)(b_r + b_i), conj(a) b) and
// not four.  Its imaginary part is a difference of larger sums: over random form
// factors the error of the 64-bit sums is 2.1e-14 against 1.5e-14 of four products
// (real part 1.2e-14 against 1.5e-14; sums up to 330), far below the rounding of either
// storage, but not of complex128, which keeps four (N_c = 8192: 7.0 ms, three take
// 6.0).  N_c = 8192, BF16: 26.1 ms
// with one thread per entry of the whole matrix (a run of set-up, 24 steps and
// spectrum: 58.7 ms; 17.3 ms with this set-up and the common-basis step loop).
// Output in the storage precision of the handle.
// A tile is filled with as many points as 64 entries hold, so that no multiply-add is
// spent on padding; only the pairs' overlaps of 1x1 bands have to leave some (55 points
// of 64).  Coarse 16^3, 1x1 bands, the whole of bse_build_coarse: 5.8 ms with a thread per
// entry, 74 ms with at most eight points to a tile (64 of 4096 entries used), 2.8 ms so.
constexpr int KC_T = 64;
constexpr size_t KC_SMEM = 200 * 1024;
size_t kc_smem(int nv, int nc, int P) {
    const size_t forms = sizeof(double) * 6 * 26 * KC_T, tile = sizeof(double2) * KC_T * (KC_T + 1);
    return std::max(forms, tile) + sizeof(double2) * P * P * (nv * nv + nc * nc) + sizeof(double) * P * P;
}
int kc_points(int nv, int nc) {
    int P = std::max(1, KC_T / (nv * nc));
    while (P > 1 && kc_smem(nv, nc, P) > KC_SMEM) --P;
    return P;
}
template <int PREC>
__global__ void __launch_bounds__(256) k_build_kc(const double2* __restrict__ M, const double2* __restrict__ Uv,
                                                  const double2* __restrict__ Uc, const double* __restrict__ htab, int n,
                                                  int nv, int nc, int P, double pref, double inv_eps, int exchange_on,
                                                  int Nc, int ldk, void* __restrict__ out, __nv_bfloat16* __restrict__ kr,
                                                  __nv_bfloat16* __restrict__ ki) {
    if (blockIdx.x < blockIdx.y) return;
    extern __shared__ __align__(16) unsigned char kcsm[];
    const int t = nv * nc, nkc = n * n * n, tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int pa = blockIdx.y * P, pb = blockIdx.x * P, na = min(P, nkc - pa), nb = min(P, nkc - pb);
    const int i0 = pa * t, j0 = pb * t, ri = na * t, rj = nb * t;          // rows and columns of this tile
    double* f = reinterpret_cast<double*>(kcsm);                            // [6][26][KC_T] a_r v, a_i v, (a_r - a_i) v, b_r, b_i, b_r + b_i
    double2* tile = reinterpret_cast<double2*>(kcsm);                       // [KC_T][KC_T + 1], after the sums
    const size_t head = max(sizeof(double) * 6 * 26 * KC_T, sizeof(double2) * KC_T * (KC_T + 1));
    double2* ov = reinterpret_cast<double2*>(kcsm + head);                  // [P P][nv nv]
    double2* oc = ov + P * P * nv * nv;                                     // [P P][nc nc]
    double* hh = reinterpret_cast<double*>(oc + P * P * nc * nc);           // [P P]
    if (exchange_on)
        for (int e = tid; e < 26 * KC_T; e += 256) {
            const int G = e / KC_T, r = e % KC_T, q = G + (G >= 13 ? 1 : 0);
            const int ga = q / 9 - 1, gb = (q / 3) % 3 - 1, gc = q % 3 - 1;
            const double v = 4.0 * kPi / (ga * ga + gb * gb + gc * gc);
            const double2 z = make_double2(0.0, 0.0);
            const double2 a = r < ri ? M[((size_t)(pa + r / t) * 26 + G) * t + r % t] : z;
            const double2 b = r < rj ? M[((size_t)(pb + r / t) * 26 + G) * t + r % t] : z;
            f[e] = a.x * v; f[26 * KC_T + e] = a.y * v; f[2 * 26 * KC_T + e] = (a.x - a.y) * v;
            f[3 * 26 * KC_T + e] = b.x; f[4 * 26 * KC_T + e] = b.y; f[5 * 26 * KC_T + e] = b.x + b.y;
        }
    for (int e = tid; e < na * nb * (nv * nv + nc * nc + 1); e += 256) {
        const int q = e / (na * nb), pr = e - q * (na * nb), x = pr / nb, y = pr - x * nb, ic = pa + x, jc = pb + y, s = x * P + y;
        if (q < nv * nv) {                                                   // Uv[a]_mv conj(Uv[b]_mv2)
            const int v = q / nv, v2 = q % nv;
            double2 o = make_double2(0.0, 0.0);
            for (int m = 0; m < nv; ++m)
                o = cadd(o, cmulc(Uv[((size_t)jc * nv + m) * nv + v2], Uv[((size_t)ic * nv + m) * nv + v]));
            ov[s * nv * nv + q] = o;
        } else if (q < nv * nv + nc * nc) {                                   // conj(Uc[a]_mc) Uc[b]_mc2
            const int w = q - nv * nv, c = w / nc, c2 = w % nc;
            double2 o = make_double2(0.0, 0.0);
            for (int m = 0; m < nc; ++m)
                o = cadd(o, cmulc(Uc[((size_t)ic * nc + m) * nc + c], Uc[((size_t)jc * nc + m) * nc + c2]));
            oc[s * nc * nc + w] = o;
        } else {
            const Int3 ia = unflat3(ic, n), ib = unflat3(jc, n);
            hh[s] = htab[flat3(ia.a - ib.a, ia.b - ib.b, ia.c - ib.c, n)] * inv_eps;
        }
    }
    __syncthreads();
    constexpr bool three = PREC != BSE_PREC_F64;
    double s1[4][4], s2[4][4], s3[4][4];                                     // S1, S2, S3, or the two parts
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s1[i][j] = s2[i][j] = s3[i][j] = 0.0;
    if (exchange_on)
        for (int G = 0; G < 26; ++G) {
            double a[3][4], b[3][4];
#pragma unroll
            for (int w = 0; w < (three ? 3 : 2); ++w)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    a[w][i] = f[(w * 26 + G) * KC_T + ty + 16 * i];
                    b[w][i] = f[((3 + w) * 26 + G) * KC_T + tx + 16 * i];
                }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if constexpr (three) {
                        s1[i][j] = fma(a[0][i], b[0][j], s1[i][j]);
                        s2[i][j] = fma(a[1][i], b[1][j], s2[i][j]);
                        s3[i][j] = fma(a[2][i], b[2][j], s3[i][j]);
                    } else {
                        s1[i][j] = fma(a[0][i], b[0][j], fma(a[1][i], b[1][j], s1[i][j]));
                        s2[i][j] = fma(a[0][i], b[1][j], fma(-a[1][i], b[0][j], s2[i][j]));
                    }
                }
        }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = ty + 16 * i;
        if (r >= ri) continue;
        const int x = r / t, e = r - x * t, v = e / nc, c = e - v * nc;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int q = tx + 16 * j;
            if (q >= rj) continue;
            const int y = q / t, e2 = q - y * t, v2 = e2 / nc, c2 = e2 - v2 * nc, s = x * P + y;
            const double2 d = cscale(cmul(ov[s * nv * nv + v * nv + v2], oc[s * nc * nc + c * nc + c2]), hh[s]);
            const double re = three ? s1[i][j] + s2[i][j] : s1[i][j], im = three ? s3[i][j] - s1[i][j] + s2[i][j] : s2[i][j];
            tile[r * (KC_T + 1) + q] = make_double2(pref * (2.0 * re - d.x), pref * (2.0 * im - d.y));
        }
    }
    __syncthreads();
    const bool diag = blockIdx.x == blockIdx.y;
    auto put = [&](size_t i, size_t j, double2 v) {
        if (PREC == BSE_PREC_F64) {
            reinterpret_cast<double2*>(out)[i * Nc + j] = v;
        } else if (PREC == BSE_PREC_F32) {
            reinterpret_cast<float2*>(out)[i * Nc + j] = make_float2((float)v.x, (float)v.y);
        } else {
            kr[i * ldk + j] = __double2bfloat16(v.x);
            ki[i * ldk + j] = __double2bfloat16(v.y);
        }
    };
    const int col = tid & 63, row0 = tid >> 6;
    for (int r = row0; r < ri; r += 4)
        if (col < rj) {
            // a diagonal tile keeps its upper half and mirrors it; its diagonal is real
            double2 v = diag && r > col ? conjg(tile[col * (KC_T + 1) + r]) : tile[r * (KC_T + 1) + col];
            if (diag && r == col) v.y = 0.0;
            put((size_t)i0 + r, (size_t)j0 + col, v);
        }
    if (!diag)
        for (int r = row0; r < rj; r += 4)
            if (col < ri) put((size_t)j0 + r, (size_t)i0 + col, conjg(tile[col * (KC_T + 1) + r]));
}

// ---------------------------------------------------------------- Method 2
// Dense interpolation matrix (Eq. interpwfn) F [N][Nc], complex128:
// F[(kd, v, c), (k~_l, n1, n2)] += f(kd, l) d_v^{n1} conj(d_c^{n2}); one thread per row.
__global__ void k_m2_F(const double2* __restrict__ Dv, const double2* __restrict__ Dc, int n, int nd, int nv, int nc,
                       int nb1, int N, int Nc, double2* __restrict__ F) {
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= N) return;
    const int t = nv * nc, kd = row / t, tr = row % t, v = tr / nc, c = tr % nc;
    const int Ndiv = nd * nd * nd, ic = kd / Ndiv, js = kd % Ndiv;
    const Int3 i = unflat3(ic, n);
    double2* fr = F + (size_t)row * Nc;
    for (int l = 0; l < 8; ++l) {
        const double f = interp_weight(js, l, nd, nb1);
        if (f == 0.0) continue;
        const int cic = flat3(i.a + ((l >> 2) & 1), i.b + ((l >> 1) & 1), i.c + (l & 1), n);
        const double2* dv = Dv + ((size_t)kd * 8 + l) * nv * nv;
        const double2* dc = Dc + ((size_t)kd * 8 + l) * nc * nc;
        for (int n1 = 0; n1 < nv; ++n1)
            for (int n2 = 0; n2 < nc; ++n2) {
                const double2 val = cscale(cmul(dv[n1 * nv + v], conjg(dc[n2 * nc + c])), f);
                double2* dst = fr + (size_t)cic * t + n1 * nc + n2;
                *dst = cadd(*dst, val);
            }
    }
}

// Head of Eq. diverg for every coarse pair and the remainder:
//   A[(i, n1 n2), (j, n3 n4)] = alpha O^v_{n1 n3}(i, j) O^c_{n2 n4}(i, j),
//   Kmod = K_c - A h_head(q_coarse(i - j)).
__global__ void k_m2_heads(const double2* __restrict__ Uv, const double2* __restrict__ Uc,
                           const double* __restrict__ hh, const double2* __restrict__ Kc, int n, int nv, int nc,
                           double alpha, int Nc, double2* __restrict__ A, double2* __restrict__ Kmod) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)Nc * Nc) return;
    const int t = nv * nc, i = (int)(e / Nc), j = (int)(e % Nc);
    const int ic = i / t, jc = j / t, n1 = (i % t) / nc, n2 = (i % t) % nc, n3 = (j % t) / nc, n4 = (j % t) % nc;
    double2 ov = make_double2(0.0, 0.0), oc = make_double2(0.0, 0.0);
    for (int m = 0; m < nv; ++m)
        ov = cadd(ov, cmul(Uv[((size_t)ic * nv + m) * nv + n1], conjg(Uv[((size_t)jc * nv + m) * nv + n3])));
    for (int m = 0; m < nc; ++m)
        oc = cadd(oc, cmul(conjg(Uc[((size_t)ic * nc + m) * nc + n2]), Uc[((size_t)jc * nc + m) * nc + n4]));
    const double2 a = cscale(cmul(ov, oc), alpha);
    const Int3 ia = unflat3(ic, n), ib = unflat3(jc, n);
    const double hc = hh[flat3(ia.a - ib.a, ia.b - ib.b, ia.c - ib.c, n)];
    A[e] = a;
    Kmod[e] = csub(Kc[e], cscale(a, hc));
}

// C [M][Nn] = X [M][K] Y [K][Nn] (conj_y = 0) or X Y^H with Y [Nn][K] (conj_y = 1),
// complex128, 16 x 16 tiles staged in shared memory.
__global__ void k_m2_gemm(const double2* __restrict__ X, const double2* __restrict__ Y, int M, int Nn, int K,
                          int conj_y, double2* __restrict__ C) {
    __shared__ double2 xs[16][17], ys[16][17];
    const int r = blockIdx.y * 16 + threadIdx.y, col = blockIdx.x * 16 + threadIdx.x;
    double2 acc = make_double2(0.0, 0.0);
    for (int k0 = 0; k0 < K; k0 += 16) {
        const int kx = k0 + threadIdx.x, ky = k0 + threadIdx.y;
        xs[threadIdx.y][threadIdx.x] = (r < M && kx < K) ? X[(size_t)r * K + kx] : make_double2(0.0, 0.0);
        const int yc = blockIdx.x * 16 + threadIdx.x;
        double2 yv = make_double2(0.0, 0.0);
        if (yc < Nn && ky < K) yv = conj_y ? conjg(Y[(size_t)yc * K + ky]) : Y[(size_t)ky * Nn + yc];
        ys[threadIdx.y][threadIdx.x] = yv;
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) acc = cadd(acc, cmul(xs[threadIdx.y][kk], ys[kk][threadIdx.x]));
        __syncthreads();
    }
    if (r < M && col < Nn) C[(size_t)r * Nn + col] = acc;
}

// H = diag(dE) + (HA h_head(q_dense) + H) / N_div in place (H holds F Kmod F^H).
__global__ void k_m2_combine(const double2* __restrict__ HA, const double* __restrict__ hd, const double* __restrict__ dE,
                             int n, int nd, int t, int N, double2* __restrict__ H) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)N * N) return;
    const int i = (int)(e / N), j = (int)(e % N);
    const int L = n * nd, Ndiv = nd * nd * nd;
    const int ki = i / t, kj = j / t;
    const Int3 ci = unflat3(ki / Ndiv, n), si = unflat3(ki % Ndiv, nd), cj = unflat3(kj / Ndiv, n), sj = unflat3(kj % Ndiv, nd);
    const double h = hd[flat3((ci.a - cj.a) * nd + si.a - sj.a, (ci.b - cj.b) * nd + si.b - sj.b,
                              (ci.c - cj.c) * nd + si.c - sj.c, L)];
    double2 v = cscale(cadd(cscale(HA[e], h), H[e]), 1.0 / Ndiv);
    if (i == j) v.x += dE[i];
    H[e] = v;
}

// K_c given by the caller (complex128 [Nc][Nc]) converted to the storage precision.
template <int PREC>
__global__ void k_kc_from_user(const double2* __restrict__ user, int Nc, int ldk, void* __restrict__ out,
                               __nv_bfloat16* __restrict__ kr, __nv_bfloat16* __restrict__ ki) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)Nc * Nc) return;
    const double2 v = user[e];
    const long long i = e / Nc, j = e % Nc;
    if (PREC == BSE_PREC_F64) {
        reinterpret_cast<double2*>(out)[e] = v;
    } else if (PREC == BSE_PREC_F32) {
        reinterpret_cast<float2*>(out)[e] = make_float2((float)v.x, (float)v.y);
    } else {
        kr[i * ldk + j] = __double2bfloat16(v.x);
        ki[i * ldk + j] = __double2bfloat16(v.y);
    }
}

// Dense table given by the caller (FP64 / complex128 host data copied to `tmp`)
// into the vector precision.
template <typename T>
__global__ void k_real_to(const double* __restrict__ src, long long n, T* __restrict__ dst) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = (T)src[i];
}
template <typename V>
__global__ void k_cplx_to(const double2* __restrict__ src, long long n, V* __restrict__ dst) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = from_d2<V>(src[i]);
}

// Dense tables, 2 G lanes per dense point kd: the gauge U(k) (G lanes per
// manifold), Delta E_vc(k) (exact on the dense mesh), dipoles
// P^alpha_vc(k) = [U_v^T pi^alpha conj(U_c)], and, where the path reads them, U
// itself in the vector precision (Uvt, Uct) or the overlaps d = U(k~)^H U(k) with
// the 8 corners (Eq. completeness).  FP64 bounds it, a warp instruction at a time
// (16 clocks of an SM, idle lanes or not): sines and cosines come from a table of the L
// values per axis, and few bands leave a warp to several points: G = 16 lanes from
// 3 bands on, 4 for 2x2 and 1x2, 1 for 1x1.  Everything stays in shared memory:
// 32768 points of 4x4 bands took 4.4 ms with a thread per point.  Set-up of a Method-1
// handle, FP32, with a thread, with a warp per point, and so: 110592 points of 1x1 bands
// 0.75, 2.1, 0.45 ms; 125000 of 2x2 bands 2.0, 2.7, 0.9 ms; 125000 of 1x3 bands 3.2, 3.7, 2.7 ms.
constexpr int kDenseWarps = 4;
int dense_lanes(int nv, int nc) { const int nb = std::max(nv, nc); return nb == 1 ? 1 : (nb == 2 ? 4 : kGaugeLanes); }
size_t dense_smem(int nv, int nc, int L) {
    const int points = kDenseWarps * (16 / dense_lanes(nv, nc));
    return sizeof(double2) * ((size_t)points * (kGaugeMats * (nv * nv + nc * nc) + 2 * 3 * nv * nc) + L);
}
template <typename T, int G>
__global__ void __launch_bounds__(32 * kDenseWarps) k_dense_tables(
    const double2* __restrict__ gen_v, const double2* __restrict__ gen_c, const double2* __restrict__ Uvc,
    const double2* __restrict__ Ucc, const double* __restrict__ offsets, const double2* __restrict__ dip, int n, int nd,
    int nv, int nc, double e_gap, double band_width, T* __restrict__ dE, typename Cx<T>::V* __restrict__ Dv,
    typename Cx<T>::V* __restrict__ Dc, typename Cx<T>::V* __restrict__ Uvt, typename Cx<T>::V* __restrict__ Uct,
    double2* __restrict__ P) {
    using V = typename Cx<T>::V;
    extern __shared__ double2 dsm[];
    constexpr int S = 2 * G, PB = 32 * kDenseWarps / S;              // lanes per point, points per block
    const int sub = threadIdx.x / S, lane = threadIdx.x % S, half = lane / G, first = threadIdx.x & 31 & ~(S - 1);
    const unsigned mask = grp_mask<S>();
    const int t = nv * nc, rv = nv * nv, rc = nc * nc, Ndiv = nd * nd * nd, nk = n * n * n * Ndiv, L = n * nd;
    const size_t N = (size_t)nk * t;
    double2* trig = dsm;                                               // [L] cos, sin of 2 pi x / L
    double2* work = dsm + L + (size_t)sub * (kGaugeMats * (rv + rc) + 6 * t);
    double2* pa = work + kGaugeMats * (rv + rc);
    double2* pb = pa + 3 * t;
    for (int x = threadIdx.x; x < L; x += 32 * kDenseWarps) sincospi(2.0 * x / L, &trig[x].y, &trig[x].x);
    __syncthreads();
    for (int kd = blockIdx.x * PB + sub; kd < nk; kd += gridDim.x * PB) {
        const Int3 g = point_ints(kd, n, nd);
        const double2 ta = trig[g.a], tb = trig[g.b], tc = trig[g.c];
        const double sn[3] = {ta.y, tb.y, tc.y}, cs[3] = {ta.x, tb.x, tc.x};
        const double2* E = grp_gauge<G>(half ? gen_c : gen_v, half ? nc : nv, sn, cs, half ? work + kGaugeMats * rv : work);
        // both manifolds' results, by their places in the scratch
        const int at = (int)(E - work), av = __shfl_sync(mask, at, first), ac = __shfl_sync(mask, at, first + G);
        const double2 *uv = work + av, *uc = work + ac;
        __syncwarp(mask);
        double band = e_gap;
        for (int a = 0; a < 3; ++a) band += band_width * (1.0 - cs[a]);
        for (int e = lane; e < t; e += S) dE[(size_t)kd * t + e] = (T)(band + offsets[e]);
        if (Uvt) {
            for (int e = lane; e < rv; e += S) Uvt[(size_t)kd * rv + e] = from_d2<V>(uv[e]);
            for (int e = lane; e < rc; e += S) Uct[(size_t)kd * rc + e] = from_d2<V>(uc[e]);
        }
        for (int e = lane; e < 3 * t; e += S) {
            double2 s = dip[e];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                s = cadd(s, cadd(cscale(dip[(size_t)(1 + 2 * a) * 3 * t + e], cs[a]), cscale(dip[(size_t)(2 + 2 * a) * 3 * t + e], sn[a])));
            pa[e] = s;
        }
        __syncwarp(mask);
        rotate_forms<false>(pa, uv, uc, pb, pa, 3, nv, nc, lane, S, [mask] { __syncwarp(mask); });
        for (int e = lane; e < 3 * t; e += S) P[(size_t)(e / t) * N + (size_t)kd * t + e % t] = pa[e];
        if (Dv) {
            const Int3 i = unflat3(kd / Ndiv, n);
            for (int l = 0; l < 8; ++l) {
                const int cic = flat3(i.a + ((l >> 2) & 1), i.b + ((l >> 1) & 1), i.c + (l & 1), n);
                const double2* cv = Uvc + (size_t)cic * rv;
                const double2* cm = Ucc + (size_t)cic * rc;
                for (int e = lane; e < rv + rc; e += S) {
                    const bool val = e < rv;
                    const int q = val ? e : e - rv, nb = val ? nv : nc, np = q / nb, b = q - np * nb;
                    double2 s = make_double2(0.0, 0.0);
                    for (int m = 0; m < nb; ++m) s = cadd(s, cmulc((val ? cv : cm)[m * nb + np], (val ? uv : uc)[m * nb + b]));
                    if (val) Dv[((size_t)kd * 8 + l) * rv + q] = from_d2<V>(s);
                    else Dc[((size_t)kd * 8 + l) * rc + q] = from_d2<V>(s);
                }
            }
        }
        __syncwarp(mask);
    }
}

// Head factors of Eq. diverg for coarse pairs (k~, k~ + r), r in the relative box:
//   Hv = alpha O^v(k~, k~'), Hc = O^c(k~, k~'); hc[r] = h_head(q_coarse(r)).
template <typename T>
__global__ void k_heads(const double2* __restrict__ Uv, const double2* __restrict__ Uc,
                        const double* __restrict__ hhead_coarse, int n, int nv, int nc, int rmin,
                        int nr1, double alpha, typename Cx<T>::V* __restrict__ Hv,
                        typename Cx<T>::V* __restrict__ Hc, T* __restrict__ hc) {
    using V = typename Cx<T>::V;
    const int nrel = nr1 * nr1 * nr1;
    const int nkc = n * n * n;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nkc * nrel) return;
    const int ic = idx / nrel, r = idx % nrel;
    const Int3 rr = unflat3(r, nr1);
    const int ra = rr.a + rmin, rb = rr.b + rmin, rc = rr.c + rmin;
    const Int3 i = unflat3(ic, n);
    const int jc = flat3(i.a + ra, i.b + rb, i.c + rc, n);
    const double2* uva = Uv + (size_t)ic * nv * nv;
    const double2* uvb = Uv + (size_t)jc * nv * nv;
    const double2* uca = Uc + (size_t)ic * nc * nc;
    const double2* ucb = Uc + (size_t)jc * nc * nc;
    for (int a = 0; a < nv; ++a)
        for (int b = 0; b < nv; ++b) {
            double2 s = make_double2(0.0, 0.0);
            for (int m = 0; m < nv; ++m) s = cadd(s, cmulc(uvb[m * nv + b], uva[m * nv + a]));
            Hv[(size_t)idx * nv * nv + a * nv + b] = from_d2<V>(cscale(s, alpha));
        }
    for (int a = 0; a < nc; ++a)
        for (int b = 0; b < nc; ++b) {
            double2 s = make_double2(0.0, 0.0);
            for (int m = 0; m < nc; ++m) s = cadd(s, cmulc(uca[m * nc + a], ucb[m * nc + b]));
            Hc[(size_t)idx * nc * nc + a * nc + b] = from_d2<V>(s);
        }
    if (ic == 0) hc[r] = (T)hhead_coarse[flat3(ra, rb, rc, n)];
}

// h_head at the dense near offsets: 1 / (|delta / L|^2 + kappa^2) (near pairs never tie).
template <typename T>
__global__ void k_near_head(const int* __restrict__ offs, int n_near, int L, double kappa,
                            T* __restrict__ hd) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_near) return;
    const double qa = (double)offs[3 * i] / L, qb = (double)offs[3 * i + 1] / L,
                 qc = (double)offs[3 * i + 2] / L;
    hd[i] = (T)(1.0 / (qa * qa + qb * qb + qc * qc + kappa * kappa));
}

inline int blocks_for(long long n, int bs) { return (int)((n + bs - 1) / bs); }

}  // namespace

int bse_alloc(bse_ctx* ctx, void** p, size_t bytes, const char* what) {
    *p = nullptr;
    if (bytes == 0) bytes = 16;
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        ctx->err = std::string("device allocation of ") + what + " (" + std::to_string(bytes) +
                   " bytes) failed: " + cudaGetErrorString(e);
        *p = nullptr;
        return BSE_ERR_OOM;
    }
    return BSE_OK;
}

#define TRY(x)                     \
    do {                           \
        int rc_ = (x);             \
        if (rc_ != BSE_OK) return rc_; \
    } while (0)

int bse_setup_coarse_device(bse_ctx* ctx, bse_coarse* c, const void* user_kc) {
    const int n = c->n, nv = c->nv, nc = c->nc, nkc = c->nkc, Nc = c->Nc;
    cudaStream_t st = ctx->stream;
    TRY(bse_alloc(ctx, (void**)&c->d_Uv, sizeof(double2) * nkc * nv * nv, "coarse Uv"));
    TRY(bse_alloc(ctx, (void**)&c->d_Uc, sizeof(double2) * nkc * nc * nc, "coarse Uc"));
    const size_t gsm = sizeof(double2) * 4 * kGaugeMats * (nv * nv + nc * nc);
    BSE_CUDA_TRY(ctx, bse_raise_smem(k_gauge, gsm));
    k_gauge<<<blocks_for(nkc, 4), 128, gsm, st>>>(c->d_gen_v, c->d_gen_c, nv, nc, n, c->d_Uv, c->d_Uc);
    double2* d_M = nullptr;
    double* d_h = nullptr;
    if (!user_kc) {
        TRY(bse_alloc(ctx, (void**)&d_M, sizeof(double2) * nkc * 26 * nv * nc, "form factors"));
        TRY(bse_alloc(ctx, (void**)&d_h, sizeof(double) * nkc, "shape table"));
        const size_t fsm = sizeof(double2) * (52 * nv * nc + nv * nv + nc * nc);
        BSE_CUDA_TRY(ctx, bse_raise_smem(k_form_factors, fsm));
        k_form_factors<<<nkc, 256, fsm, st>>>(c->d_Uv, c->d_Uc, c->d_mu, n, nv, nc, d_M);
        k_shape_table<<<blocks_for(nkc, 4), 128, 0, st>>>(n, c->kappa, c->direct_shells, c->h_const, c->h0, 0, d_h);
    }
    size_t bytes;
    if (c->kc_prec == BSE_PREC_F64) bytes = sizeof(double2) * (size_t)Nc * Nc;
    else if (c->kc_prec == BSE_PREC_F32) bytes = sizeof(float2) * (size_t)Nc * Nc;
    else bytes = 2 * sizeof(__nv_bfloat16) * (size_t)Nc * c->ldk;
    int rc = bse_alloc(ctx, &c->d_kc, bytes, "K_c");
    if (rc != BSE_OK) { cudaFree(d_M); cudaFree(d_h); return rc; }
    if (c->kc_prec == BSE_PREC_BF16) {
        c->d_kr = reinterpret_cast<__nv_bfloat16*>(c->d_kc);
        c->d_ki = c->d_kr + (size_t)Nc * c->ldk;
        if (c->ldk > Nc)                                        // zero the padding columns of both planes
            cudaMemset2DAsync(c->d_kr + Nc, sizeof(__nv_bfloat16) * c->ldk, 0, sizeof(__nv_bfloat16) * (c->ldk - Nc),
                              2 * (size_t)Nc, st);
    }
    const double pref = c->e_k / nkc;
    const int P = kc_points(nv, nc), kt = blocks_for(nkc, P);
    const dim3 gs(kt, kt);
    const size_t ksm = kc_smem(nv, nc, P);
    auto build = [&](auto kernel, void* out, __nv_bfloat16* kr, __nv_bfloat16* ki) -> int {
        BSE_CUDA_TRY(ctx, bse_raise_smem(kernel, ksm));
        kernel<<<gs, 256, ksm, st>>>(d_M, c->d_Uv, c->d_Uc, d_h, n, nv, nc, P, pref, 1.0 / c->eps_inf, c->exchange_on, Nc, c->ldk,
                                     out, kr, ki);
        return BSE_OK;
    };
    if (user_kc) {
        const long long ne = (long long)Nc * Nc;
        const double2* u = static_cast<const double2*>(user_kc);
        if (c->kc_prec == BSE_PREC_F64)
            k_kc_from_user<BSE_PREC_F64><<<blocks_for(ne, 256), 256, 0, st>>>(u, Nc, c->ldk, c->d_kc, nullptr, nullptr);
        else if (c->kc_prec == BSE_PREC_F32)
            k_kc_from_user<BSE_PREC_F32><<<blocks_for(ne, 256), 256, 0, st>>>(u, Nc, c->ldk, c->d_kc, nullptr, nullptr);
        else
            k_kc_from_user<BSE_PREC_BF16><<<blocks_for(ne, 256), 256, 0, st>>>(u, Nc, c->ldk, nullptr, c->d_kr, c->d_ki);
    } else if (c->kc_prec == BSE_PREC_F64) {
        rc = build(k_build_kc<BSE_PREC_F64>, c->d_kc, nullptr, nullptr);
    } else if (c->kc_prec == BSE_PREC_F32) {
        rc = build(k_build_kc<BSE_PREC_F32>, c->d_kc, nullptr, nullptr);
    } else {
        rc = build(k_build_kc<BSE_PREC_BF16>, nullptr, c->d_kr, c->d_ki);
    }
    cudaError_t e = cudaGetLastError();
    cudaError_t e2 = cudaStreamSynchronize(st);
    cudaFree(d_M);
    cudaFree(d_h);
    if (e != cudaSuccess || e2 != cudaSuccess) {
        ctx->err = std::string("coarse set-up kernels: ") + cudaGetErrorString(e != cudaSuccess ? e : e2);
        return BSE_ERR_CUDA;
    }
    return rc;
}

namespace {

// Replace the model's dense tables by the caller's (bse_dense_inputs), after
// k_dense_tables has written the model's.
// Largest Frobenius norm of the caller's overlap blocks over the pieces of
// non-zero weight (host arrays [nk][8][nb][nb] complex128).
double max_block_norm(const double* d, const bse_interp* s, int nb) {
    double best = 0.0;
    for (int kd = 0; kd < s->nk; ++kd)
        for (int l = 0; l < 8; ++l) {
            if (!interp_active(kd % s->Ndiv, l, s->nd, s->nb1)) continue;
            const double* p = d + ((size_t)kd * 8 + l) * nb * nb * 2;
            double f = 0.0;
            for (int q = 0; q < 2 * nb * nb; ++q) f += p[q] * p[q];
            best = std::max(best, std::sqrt(f));
        }
    return best;
}

template <typename T>
int apply_dense_inputs(bse_ctx* ctx, bse_interp* s, const bse_dense_inputs* in) {
    using V = typename Cx<T>::V;
    const double bv = in->Dv ? max_block_norm(in->Dv, s, s->nv) : std::sqrt((double)s->nv);
    const double bc = in->Dc ? max_block_norm(in->Dc, s, s->nc) : std::sqrt((double)s->nc);
    s->dbound = bv * bc;
    cudaStream_t st = ctx->stream;
    const long long N = s->N, nDv = (long long)s->nk * 8 * s->nv * s->nv, nDc = (long long)s->nk * 8 * s->nc * s->nc;
    const long long most = std::max(std::max(N, nDv), nDc);
    double2* tmp = nullptr;
    TRY(bse_alloc(ctx, (void**)&tmp, sizeof(double2) * (size_t)most, "dense input staging"));
    cudaError_t e = cudaSuccess;
    if (in->dE && e == cudaSuccess) {
        e = cudaMemcpyAsync(tmp, in->dE, sizeof(double) * N, cudaMemcpyHostToDevice, st);
        k_real_to<T><<<blocks_for(N, 256), 256, 0, st>>>((const double*)tmp, N, (T*)s->d_dE);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    if (in->P && e == cudaSuccess) e = cudaMemcpyAsync(s->d_P, in->P, sizeof(double2) * 3 * N, cudaMemcpyHostToDevice, st);
    if (in->Dv && e == cudaSuccess) {
        e = cudaMemcpyAsync(tmp, in->Dv, sizeof(double2) * nDv, cudaMemcpyHostToDevice, st);
        k_cplx_to<V><<<blocks_for(nDv, 256), 256, 0, st>>>(tmp, nDv, (V*)s->d_Dv);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    if (in->Dc && e == cudaSuccess) {
        e = cudaMemcpyAsync(tmp, in->Dc, sizeof(double2) * nDc, cudaMemcpyHostToDevice, st);
        k_cplx_to<V><<<blocks_for(nDc, 256), 256, 0, st>>>(tmp, nDc, (V*)s->d_Dc);
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(tmp);
    if (e != cudaSuccess) {
        ctx->err = std::string("dense inputs: ") + cudaGetErrorString(e);
        return BSE_ERR_CUDA;
    }
    return BSE_OK;
}

// Method 2 set-up (FP64): the dense interpolated Hamiltonian, built with
// temporaries F, A, Kmod, F M and F A F^H that are freed again.
int build_m2(bse_ctx* ctx, bse_interp* s) {
    const bse_coarse* c = s->co;
    cudaStream_t st = ctx->stream;
    const int N = s->N, Nc = c->Nc, L = s->n * s->nd;
    double2 *F = nullptr, *A = nullptr, *Km = nullptr, *T = nullptr, *HA = nullptr;
    double *hh = nullptr, *hd = nullptr;
    int rc = BSE_OK;
    auto cleanup = [&]() { cudaFree(F); cudaFree(A); cudaFree(Km); cudaFree(T); cudaFree(HA); cudaFree(hh); cudaFree(hd); };
    if ((rc = bse_alloc(ctx, &s->d_H2, sizeof(double2) * (size_t)N * N, "Method 2 Hamiltonian")) != BSE_OK ||
        (rc = bse_alloc(ctx, (void**)&F, sizeof(double2) * (size_t)N * Nc, "M2 F")) != BSE_OK ||
        (rc = bse_alloc(ctx, (void**)&A, sizeof(double2) * (size_t)Nc * Nc, "M2 head")) != BSE_OK ||
        (rc = bse_alloc(ctx, (void**)&Km, sizeof(double2) * (size_t)Nc * Nc, "M2 remainder")) != BSE_OK ||
        (rc = bse_alloc(ctx, (void**)&T, sizeof(double2) * (size_t)N * Nc, "M2 temporary")) != BSE_OK ||
        (rc = bse_alloc(ctx, (void**)&HA, sizeof(double2) * (size_t)N * N, "M2 head part")) != BSE_OK ||
        (rc = bse_alloc(ctx, (void**)&hh, sizeof(double) * c->nkc, "coarse head table")) != BSE_OK ||
        (rc = bse_alloc(ctx, (void**)&hd, sizeof(double) * (size_t)L * L * L, "dense head table")) != BSE_OK) {
        cleanup();
        return rc;
    }
    cudaMemsetAsync(F, 0, sizeof(double2) * (size_t)N * Nc, st);
    k_m2_F<<<blocks_for(N, 128), 128, 0, st>>>((const double2*)s->d_Dv, (const double2*)s->d_Dc, s->n, s->nd, s->nv,
                                               s->nc, s->nb1, N, Nc, F);
    k_shape_table<<<blocks_for(c->nkc, 4), 128, 0, st>>>(s->n, c->kappa, 27, 0, 0.0, 1, hh);
    k_shape_table<<<blocks_for((long long)L * L * L, 4), 128, 0, st>>>(L, c->kappa, 27, 0, 0.0, 1, hd);
    k_m2_heads<<<blocks_for((long long)Nc * Nc, 256), 256, 0, st>>>(c->d_Uv, c->d_Uc, hh, (const double2*)c->d_kc, s->n,
                                                                   s->nv, s->nc, c->alpha, Nc, A, Km);
    const dim3 b16(16, 16);
    // H <- F Kmod F^H, HA <- F A F^H
    k_m2_gemm<<<dim3(blocks_for(Nc, 16), blocks_for(N, 16)), b16, 0, st>>>(F, Km, N, Nc, Nc, 0, T);
    k_m2_gemm<<<dim3(blocks_for(N, 16), blocks_for(N, 16)), b16, 0, st>>>(T, F, N, N, Nc, 1, (double2*)s->d_H2);
    k_m2_gemm<<<dim3(blocks_for(Nc, 16), blocks_for(N, 16)), b16, 0, st>>>(F, A, N, Nc, Nc, 0, T);
    k_m2_gemm<<<dim3(blocks_for(N, 16), blocks_for(N, 16)), b16, 0, st>>>(T, F, N, N, Nc, 1, HA);
    k_m2_combine<<<blocks_for((long long)N * N, 256), 256, 0, st>>>(HA, hd, (const double*)s->d_dE, s->n, s->nd, s->t,
                                                                    N, (double2*)s->d_H2);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cleanup();
    if (e != cudaSuccess) {
        ctx->err = std::string("Method 2 set-up: ") + cudaGetErrorString(e);
        return BSE_ERR_CUDA;
    }
    return BSE_OK;
}

// Method 3's near offsets |delta|^2 <= R2 (three ints each into `offs`, when
// given) and the boxes of coarse points they reach.
int near_geometry(bse_ctx* ctx, bse_interp* s, std::vector<int>* offs) {
    const int nd = s->nd, R2 = (int)std::floor(s->width * s->width * nd * nd + 1e-9);
    const int rad = (int)std::floor(std::sqrt((double)R2) + 1e-12);
    s->near_R2 = R2;
    s->cphi_R = rad;
    s->n_near = 0;
    for (int a = -rad; a <= rad; ++a)
        for (int b = -rad; b <= rad; ++b)
            for (int cc = -rad; cc <= rad; ++cc)
                if (a * a + b * b + cc * cc <= R2) {
                    ++s->n_near;
                    if (offs) { offs->push_back(a); offs->push_back(b); offs->push_back(cc); }
                }
    s->smin = floordiv(-rad, nd);
    const int smax = floordiv(nd - 1 + rad, nd) + 1;
    s->ns1 = smax - s->smin + 1;
    s->nslot = s->ns1 * s->ns1 * s->ns1;
    s->rmin = s->smin - 1;
    s->nr1 = smax - s->rmin + 1;
    s->nrel = s->nr1 * s->nr1 * s->nr1;
    if (s->ns1 > 15 || s->smin < -8 || smax > 7) {
        ctx->err = "M3 width too large for the near-field tables";
        return BSE_ERR_UNSUPPORTED;
    }
    return BSE_OK;
}

template <typename T>
int setup_interp_typed(bse_ctx* ctx, bse_interp* s, const bse_dense_inputs* dense) {
    using V = typename Cx<T>::V;
    const bse_coarse* c = s->co;
    const int n = s->n, nd = s->nd, nk = s->nk, nv = s->nv, nc = s->nc, t = s->t, N = s->N;
    cudaStream_t st = ctx->stream;
    // Overlaps that are products through one unitary gauge: the common-basis path
    // (Method 2 stores its H instead) reads U(k); the others the overlaps.
    s->common = s->scheme != BSE_SCHEME_M2 && c->unitary && !(dense && (dense->Dv || dense->Dc));
    // dense tables
    TRY(bse_alloc(ctx, &s->d_dE, sizeof(T) * (size_t)N, "dE"));
    TRY(bse_alloc(ctx, (void**)&s->d_P, sizeof(double2) * 3 * (size_t)N, "dipoles"));
    if (s->common) {
        TRY(bse_alloc(ctx, &s->d_cUv, sizeof(V) * (size_t)nk * nv * nv, "dense gauge"));
        TRY(bse_alloc(ctx, &s->d_cUc, sizeof(V) * (size_t)nk * nc * nc, "dense gauge"));
    } else {
        TRY(bse_alloc(ctx, &s->d_Dv, sizeof(V) * (size_t)nk * 8 * nv * nv, "Dv"));
        TRY(bse_alloc(ctx, &s->d_Dc, sizeof(V) * (size_t)nk * 8 * nc * nc, "Dc"));
    }
    auto tables = [&](auto lanes) -> int {
        constexpr int G = decltype(lanes)::value;
        const size_t dsm = dense_smem(nv, nc, n * nd);
        BSE_CUDA_TRY(ctx, bse_raise_smem((k_dense_tables<T, G>), dsm));
        const int blocks = std::min(blocks_for(nk, kDenseWarps * (16 / G)), 16 * std::max(ctx->sm_count, 1));
        k_dense_tables<T, G><<<blocks, 32 * kDenseWarps, dsm, st>>>(
            c->d_gen_v, c->d_gen_c, c->d_Uv, c->d_Uc, c->d_offsets, c->d_dip, n, nd, nv, nc, c->e_gap, c->band_width,
            (T*)s->d_dE, (V*)s->d_Dv, (V*)s->d_Dc, (V*)s->d_cUv, (V*)s->d_cUc, s->d_P);
        return BSE_OK;
    };
    const int lanes = dense_lanes(nv, nc);
    TRY(lanes == 1 ? tables(std::integral_constant<int, 1>{})
                   : lanes == 4 ? tables(std::integral_constant<int, 4>{}) : tables(std::integral_constant<int, kGaugeLanes>{}));
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        ctx->err = std::string("dense set-up kernels: ") + cudaGetErrorString(e);
        return BSE_ERR_CUDA;
    }
    if (s->common && s->scheme == BSE_SCHEME_M3) {
        TRY(near_geometry(ctx, s, nullptr));
        TRY(bse_alloc(ctx, (void**)&s->d_chead, sizeof(double) * c->nkc, "coarse head table"));
        k_shape_table<<<blocks_for(c->nkc, 4), 128, 0, st>>>(n, c->kappa, 27, 0, 0.0, 1, s->d_chead);
    }
    if (s->common) TRY(bse_common_prepare(ctx, s));
    s->dbound = std::sqrt((double)nv) * std::sqrt((double)nc);
    if (dense) TRY(apply_dense_inputs<T>(ctx, s, dense));
    // scratch
    const size_t nvec = BSE_MAX_CHAINS;
    TRY(bse_alloc(ctx, &s->d_Q, sizeof(V) * nvec * c->Nc, "Q"));
    TRY(bse_alloc(ctx, &s->d_R, sizeof(V) * nvec * c->Nc, "R"));
    for (int q = 0; q < 3; ++q) TRY(bse_alloc(ctx, &s->d_vec[q], sizeof(V) * nvec * N, "Lanczos vectors"));
    TRY(bse_alloc(ctx, (void**)&s->d_part_dot, sizeof(double2) * nvec * BSE_MAX_VEC_BLOCKS, "dot partials"));
    TRY(bse_alloc(ctx, (void**)&s->d_part_nrm, sizeof(double) * nvec * BSE_MAX_VEC_BLOCKS, "norm partials"));
    TRY(bse_alloc(ctx, (void**)&s->d_stop, sizeof(int) * nvec, "stop flags"));
    if (s->scheme == BSE_SCHEME_M2) {
        if constexpr (std::is_same<T, double>::value) TRY(build_m2(ctx, s));
    }
    if (s->scheme == BSE_SCHEME_M3 && !s->common) {
        TRY(bse_alloc(ctx, &s->d_X, sizeof(V) * nvec * nk * 8 * t, "restricted pieces X"));
        TRY(bse_alloc(ctx, &s->d_U, sizeof(V) * nvec * nk * 8 * t, "near-field pieces"));
        // contribution lists (integer bookkeeping on the host)
        std::vector<int> offs;
        TRY(near_geometry(ctx, s, &offs));
        const int Ndiv = s->Ndiv;
        std::vector<std::vector<NearEntry>> per_slot((size_t)Ndiv * s->nslot);
        for (int js = 0; js < Ndiv; ++js) {
            const Int3 j = unflat3(js, nd);
            for (int q = 0; q < s->n_near; ++q) {
                const int g[3] = {j.a + offs[3 * q], j.b + offs[3 * q + 1], j.c + offs[3 * q + 2]};
                int co[3], jp[3];
                for (int a = 0; a < 3; ++a) { co[a] = floordiv(g[a], nd); jp[a] = g[a] - co[a] * nd; }
                const int jsp = (jp[0] * nd + jp[1]) * nd + jp[2];
                for (int l = 0; l < 8; ++l) {
                    if (interp_weight(jsp, l, nd, s->nb1) == 0.0) continue;
                    const int o[3] = {co[0] + ((l >> 2) & 1), co[1] + ((l >> 1) & 1), co[2] + (l & 1)};
                    const int slot = ((o[0] - s->smin) * s->ns1 + (o[1] - s->smin)) * s->ns1 + (o[2] - s->smin);
                    NearEntry ent;
                    ent.co = (co[0] + 8) | ((co[1] + 8) << 4) | ((co[2] + 8) << 8);
                    ent.js_src = jsp;
                    ent.l_src = l;
                    ent.near_idx = q;
                    per_slot[(size_t)js * s->nslot + slot].push_back(ent);
                }
            }
        }
        std::vector<NearEntry> flat;
        std::vector<int> start((size_t)Ndiv * (s->nslot + 1));
        for (int js = 0; js < Ndiv; ++js) {
            for (int sl = 0; sl < s->nslot; ++sl) {
                start[(size_t)js * (s->nslot + 1) + sl] = (int)flat.size();
                const auto& v = per_slot[(size_t)js * s->nslot + sl];
                flat.insert(flat.end(), v.begin(), v.end());
            }
            start[(size_t)js * (s->nslot + 1) + s->nslot] = (int)flat.size();
        }
        TRY(bse_alloc(ctx, (void**)&s->d_list, sizeof(NearEntry) * flat.size(), "near list"));
        TRY(bse_alloc(ctx, (void**)&s->d_list_start, sizeof(int) * start.size(), "near list starts"));
        BSE_CUDA_TRY(ctx, bse_upload(ctx, s->d_list, flat.data(), sizeof(NearEntry) * flat.size()));
        BSE_CUDA_TRY(ctx, bse_upload(ctx, s->d_list_start, start.data(), sizeof(int) * start.size()));
        // Cell-batched form: the same contributions, with the source named by its
        // (js', corner) pair index, so one coarse cell's targets share a slot's
        // source rows staged in shared memory.
        {
            // corner-major order: neighbouring threads share a corner's head blocks
            std::vector<int> pairs, pidx((size_t)Ndiv * 8, -1);
            for (int l = 0; l < 8; ++l)
                for (int js = 0; js < Ndiv; ++js)
                    if (interp_weight(js, l, nd, s->nb1) != 0.0) {
                        pidx[(size_t)js * 8 + l] = (int)pairs.size();
                        pairs.push_back(js | (l << 16));
                    }
            s->npairs = (int)pairs.size();
            std::vector<int> clist, cstart((size_t)Ndiv * (s->nslot + 1));
            for (int js = 0; js < Ndiv; ++js) {
                for (int sl = 0; sl < s->nslot; ++sl) {
                    cstart[(size_t)js * (s->nslot + 1) + sl] = (int)clist.size();
                    for (const NearEntry& en : per_slot[(size_t)js * s->nslot + sl])
                        clist.push_back(pidx[(size_t)en.js_src * 8 + en.l_src] | (en.near_idx << 16));
                }
                cstart[(size_t)js * (s->nslot + 1) + s->nslot] = (int)clist.size();
            }
            const size_t vs = sizeof(V), ts = sizeof(T);
            const size_t tp = t + 1;                   // padded row stride (bank spread)
            const size_t smem = vs * (2 * (size_t)s->npairs * tp + 2 * (size_t)Ndiv * tp + 8 * (nv * nv + nc * nc)) +
                                ts * (8 + (size_t)s->n_near) + sizeof(int) * ((size_t)s->npairs + 8 * (size_t)s->nslot);
            int maxsm = 0;
            cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device);
            const bool fits = s->n_near < 65536 && s->npairs < 65536 && smem + 1024 <= (size_t)maxsm;
            s->cell_smem = fits ? smem : 0;
            if (fits) {
                TRY(bse_alloc(ctx, (void**)&s->d_pairs, sizeof(int) * pairs.size(), "near pairs"));
                TRY(bse_alloc(ctx, (void**)&s->d_clist, sizeof(int) * clist.size(), "cell near list"));
                TRY(bse_alloc(ctx, (void**)&s->d_cstart, sizeof(int) * cstart.size(), "cell near list starts"));
                BSE_CUDA_TRY(ctx, bse_upload(ctx, s->d_pairs, pairs.data(), sizeof(int) * pairs.size()));
                BSE_CUDA_TRY(ctx, bse_upload(ctx, s->d_clist, clist.data(), sizeof(int) * clist.size()));
                BSE_CUDA_TRY(ctx, bse_upload(ctx, s->d_cstart, cstart.data(), sizeof(int) * cstart.size()));
            }
        }
        int* d_offs = nullptr;
        double* d_hh = nullptr;
        TRY(bse_alloc(ctx, (void**)&d_offs, sizeof(int) * offs.size(), "near offsets"));
        TRY(bse_alloc(ctx, (void**)&d_hh, sizeof(double) * c->nkc, "coarse head table"));
        BSE_CUDA_TRY(ctx, bse_upload(ctx, d_offs, offs.data(), sizeof(int) * offs.size()));
        TRY(bse_alloc(ctx, &s->d_hd, sizeof(T) * s->n_near, "near head values"));
        TRY(bse_alloc(ctx, &s->d_Hv, sizeof(V) * (size_t)c->nkc * s->nrel * nv * nv, "Hv"));
        TRY(bse_alloc(ctx, &s->d_Hc, sizeof(V) * (size_t)c->nkc * s->nrel * nc * nc, "Hc"));
        TRY(bse_alloc(ctx, &s->d_hc, sizeof(T) * s->nrel, "hc"));
        k_near_head<T><<<blocks_for(s->n_near, 128), 128, 0, st>>>(d_offs, s->n_near, n * nd, c->kappa, (T*)s->d_hd);
        k_shape_table<<<blocks_for(c->nkc, 4), 128, 0, st>>>(n, c->kappa, 27, 0, 0.0, 1, d_hh);
        k_heads<T><<<blocks_for((long long)c->nkc * s->nrel, 64), 64, 0, st>>>(
            c->d_Uv, c->d_Uc, d_hh, n, nv, nc, s->rmin, s->nr1, c->alpha, (V*)s->d_Hv, (V*)s->d_Hc, (T*)s->d_hc);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        cudaFree(d_offs);
        cudaFree(d_hh);
        if (e != cudaSuccess) {
            ctx->err = std::string("M3 set-up kernels: ") + cudaGetErrorString(e);
            return BSE_ERR_CUDA;
        }
        TRY(bse_near_tc_prepare(ctx, s, per_slot));
        if (s->nf_tc) {
            // FP16 piece scales for unit-norm vectors (every Lanczos vector), and
            // room for the scales bse_apply_h computes from its inputs' norms
            const float xs = bse_near_tc_xscale(s, 1.0 + 1e-3);
            const float h4[4] = {xs, xs, xs, xs};
            TRY(bse_alloc(ctx, (void**)&s->d_xscale, sizeof(float) * 4, "piece scales"));
            TRY(bse_alloc(ctx, (void**)&s->d_xscale_gen, sizeof(float) * 4, "piece scales"));
            BSE_CUDA_TRY(ctx, bse_upload(ctx, s->d_xscale, h4, sizeof(h4)));
            BSE_CUDA_TRY(ctx, bse_upload(ctx, s->d_xscale_gen, h4, sizeof(h4)));
        }
    }
    if (c->kc_prec == BSE_PREC_BF16) TRY(bse_tc_prepare(ctx, s));
    if (s->common) TRY(bse_noalloc_setup(ctx, s));
    return BSE_OK;
}

}  // namespace

int bse_setup_interp_device(bse_ctx* ctx, bse_interp* s, const bse_dense_inputs* dense) {
    if (s->vec_prec == BSE_PREC_F64) return setup_interp_typed<double>(ctx, s, dense);
    return setup_interp_typed<float>(ctx, s, dense);
}
