// Learned correction as a periodic convolution: w += T * psi on the L^3 dense mesh,
// L = n n_div, for every pair of transitions, through 3-D DFTs in FP32.
//
// Three kernels per application, each reading and writing the grid once:
//   1. k_lconv_fwd   (chain, x plane, 4 transitions): gather psi, DFT along z and y
//   2. k_lconv_mix   (y, z frequency): DFT along x, the t x t product with the
//                    stencil's transform for every x frequency, DFT back along x
//   3. k_lconv_inv   (chain, x plane, 4 transitions): DFT back along y and z, add to w,
//                    partials of <psi, w>
// The work grid is [y z][x][chain][t], so a block of kernel 2 reads one contiguous
// piece and the others whole 32-byte sectors.  The stencil's transform
// [y z][x][e2][e1] (64 t^2 L^3 bits: 510 MB for coarse 12^3, n_div 4, 4x6 bands) is streamed
// once; it bounds the whole by HBM.  Coarse 12^3, n_div 4, 4x6 bands, 3 vectors: six
// separate DFT passes with one product per table lookup, a product kernel and two
// transpositions took 1.46 ms, these three 0.38 ms (0.07 + 0.16 + 0.15).
// A line of L = A B points (A, B <= 8) is transformed in place in two stages
// (Cooley-Tukey) by DFTs of A and B points in registers.  The frequencies stay in
// the order the stages leave them: k1 + A k2 at place B k1 + k2.  The stencil's
// transform has the same order and the way back undoes it, so nothing is permuted.
// Other L keep the separate passes of bse_mlp.cu.
#include <algorithm>
#include <cmath>

#include "bse_internal.cuh"

namespace {

constexpr int EG = 4;              // transitions per block of kernels 1 and 3: a 32-byte sector of FP32 entries
constexpr int LTHR = 256;

__device__ __forceinline__ float2 mul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
// a times -i (forward) or i (inverse)
template <bool INV> __device__ __forceinline__ float2 rot90(float2 a) { return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x); }

// In-place DFT of N points, exp(-2 pi i n k / N), conjugated for INV.
template <bool INV> __device__ __forceinline__ void dft2(float2& a, float2& b) {
    const float2 t = a;
    a = cadd(t, b);
    b = csub(t, b);
}
template <bool INV> __device__ __forceinline__ void dft3(float2& a, float2& b, float2& c) {
    const float2 s = cadd(b, c), d = rot90<INV>(cscale(csub(b, c), 0.86602540378443864676f)), m = make_float2(fmaf(-0.5f, s.x, a.x), fmaf(-0.5f, s.y, a.y));
    a = cadd(a, s);
    b = cadd(m, d);
    c = csub(m, d);
}
template <bool INV> __device__ __forceinline__ void dft4(float2& a, float2& b, float2& c, float2& d) {
    dft2<INV>(a, c);
    dft2<INV>(b, d);
    d = rot90<INV>(d);
    dft2<INV>(a, b);
    dft2<INV>(c, d);
    const float2 t = b;                    // order 0, 2, 1, 3 -> 0, 1, 2, 3
    b = c;
    c = t;
}
template <int N, bool INV> __device__ __forceinline__ void dft(float2 (&v)[N]) {
    if constexpr (N == 2) dft2<INV>(v[0], v[1]);
    else if constexpr (N == 3) dft3<INV>(v[0], v[1], v[2]);
    else if constexpr (N == 4) dft4<INV>(v[0], v[1], v[2], v[3]);
    else if constexpr (N == 6) {           // two of three, then pairs with exp(-2 pi i k / 6)
        dft3<INV>(v[0], v[2], v[4]);
        dft3<INV>(v[1], v[3], v[5]);
        constexpr float h = 0.86602540378443864676f, sg = INV ? 1.f : -1.f;
        const float2 b0 = v[1], b1 = mul(v[3], make_float2(0.5f, sg * h)), b2 = mul(v[5], make_float2(-0.5f, sg * h));
        const float2 a0 = v[0], a1 = v[2], a2 = v[4];
        v[0] = cadd(a0, b0); v[1] = cadd(a1, b1); v[2] = cadd(a2, b2);
        v[3] = csub(a0, b0); v[4] = csub(a1, b1); v[5] = csub(a2, b2);
    } else if constexpr (N == 8) {
        dft4<INV>(v[0], v[2], v[4], v[6]);
        dft4<INV>(v[1], v[3], v[5], v[7]);
        constexpr float h = 0.70710678118654752440f, sg = INV ? 1.f : -1.f;
        const float2 b0 = v[1], b1 = mul(v[3], make_float2(h, sg * h)), b2 = rot90<INV>(v[5]), b3 = mul(v[7], make_float2(-h, sg * h));
        const float2 a0 = v[0], a1 = v[2], a2 = v[4], a3 = v[6];
        v[0] = cadd(a0, b0); v[1] = cadd(a1, b1); v[2] = cadd(a2, b2); v[3] = cadd(a3, b3);
        v[4] = csub(a0, b0); v[5] = csub(a1, b1); v[6] = csub(a2, b2); v[7] = csub(a3, b3);
    } else if constexpr (N == 5 || N == 7) {   // odd primes: sums and differences of the mirrored inputs
        constexpr int H = N / 2;
        const float co[2][3] = {{0.30901699437494742410f, -0.80901699437494742410f, 0.f},
                                {0.62348980185873353053f, -0.22252093395631440429f, -0.90096886790241912624f}};
        const float si[2][3] = {{0.95105651629515357212f, 0.58778525229247312917f, 0.f},
                                {0.78183148246802980871f, 0.97492791218182360702f, 0.43388373911755812048f}};
        constexpr int q = N == 5 ? 0 : 1;
        float2 s[H], d[H], o[N];
#pragma unroll
        for (int n = 0; n < H; ++n) {
            s[n] = cadd(v[n + 1], v[N - 1 - n]);
            d[n] = csub(v[n + 1], v[N - 1 - n]);
        }
        o[0] = v[0];
#pragma unroll
        for (int n = 0; n < H; ++n) o[0] = cadd(o[0], s[n]);
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            float2 c = v[0], e = make_float2(0.f, 0.f);
#pragma unroll
            for (int n = 1; n <= H; ++n) {
                const int m = n * k % N, i = (m <= H ? m : N - m) - 1;
                const float sn = m <= H ? si[q][i] : -si[q][i];
                c = make_float2(fmaf(co[q][i], s[n - 1].x, c.x), fmaf(co[q][i], s[n - 1].y, c.y));
                e = make_float2(fmaf(sn, d[n - 1].x, e.x), fmaf(sn, d[n - 1].y, e.y));
            }
            e = rot90<INV>(e);
            o[k] = cadd(c, e);
            o[N - k] = csub(c, e);
        }
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] = o[k];
    }
}

__device__ __forceinline__ int quot(int i, float inv) { return (int)(((float)i + 0.5f) * inv); }

// One stage over `nlines` lines in shared memory, element n of line l at
// s[at(l) + n es]: `cnt` items per line, item c takes the N elements first(c) + step j.
// TW: multiply element j by tw[c j] (conjugated for INV) after (forward) or before
// (inverse) the DFT.
template <int N, bool INV, bool TW, typename At>
__device__ __forceinline__ void stage_n(float2* s, int nlines, At at, int es, int cnt, int first, int step, const float2* tw) {
    const float inv = 1.f / (float)nlines;
    for (int it = threadIdx.x; it < nlines * cnt; it += LTHR) {
        const int c = quot(it, inv), l = it - c * nlines;
        float2* p = s + at(l) + c * first * es;
        float2 v[N];
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = p[j * step * es];
        if (TW && INV) {
#pragma unroll
            for (int j = 1; j < N; ++j) v[j] = mul(v[j], conjg(tw[c * j]));
        }
        if constexpr (N > 1) dft<N, INV>(v);
        if (TW && !INV) {
#pragma unroll
            for (int j = 1; j < N; ++j) v[j] = mul(v[j], tw[c * j]);
        }
#pragma unroll
        for (int j = 0; j < N; ++j) p[j * step * es] = v[j];
    }
}
template <bool INV, bool TW, typename At>
__device__ __forceinline__ void stage(int N, float2* s, int nlines, At at, int es, int cnt, int first, int step, const float2* tw) {
    switch (N) {
        case 1: stage_n<1, INV, TW>(s, nlines, at, es, cnt, first, step, tw); break;
        case 2: stage_n<2, INV, TW>(s, nlines, at, es, cnt, first, step, tw); break;
        case 3: stage_n<3, INV, TW>(s, nlines, at, es, cnt, first, step, tw); break;
        case 4: stage_n<4, INV, TW>(s, nlines, at, es, cnt, first, step, tw); break;
        case 5: stage_n<5, INV, TW>(s, nlines, at, es, cnt, first, step, tw); break;
        case 6: stage_n<6, INV, TW>(s, nlines, at, es, cnt, first, step, tw); break;
        case 7: stage_n<7, INV, TW>(s, nlines, at, es, cnt, first, step, tw); break;
        default: stage_n<8, INV, TW>(s, nlines, at, es, cnt, first, step, tw); break;
    }
    __syncthreads();
}
// Line transforms, block-wide: n = B n1 + n2, k = k1 + A k2 left at place B k1 + k2.
template <typename At>
__device__ __forceinline__ void lines_fwd(float2* s, int nlines, At at, int es, int A, int B, const float2* tw) {
    stage<false, true>(A, s, nlines, at, es, B, 1, B, tw);      // over n1 for every n2, then w^{n2 k1}
    stage<false, false>(B, s, nlines, at, es, A, B, 1, tw);     // over n2 for every k1
}
template <typename At>
__device__ __forceinline__ void lines_inv(float2* s, int nlines, At at, int es, int A, int B, const float2* tw) {
    stage<true, false>(B, s, nlines, at, es, A, B, 1, tw);
    stage<true, true>(A, s, nlines, at, es, B, 1, B, tw);
}

struct LShape { int L, A, B, n, nd, t, nch, P; };   // P: row pitch of a plane (odd)

// The dense index of mesh point (x, y, z) is a sum of one term per axis: the x term,
// and tables of the y and z terms in shared memory.
__device__ __forceinline__ int axis_term(const LShape& q, int v, int axis) {
    const int c = v / q.nd, j = v - c * q.nd, Ndiv = q.nd * q.nd * q.nd;
    return axis == 0 ? c * q.n * q.n * Ndiv + j * q.nd * q.nd : (axis == 1 ? c * q.n * Ndiv + j * q.nd : c * Ndiv + j);
}
__device__ __forceinline__ int axis_tables(const LShape& q, int x, int* iy, int* iz) {
    for (int v = threadIdx.x; v < q.L; v += LTHR) {
        iy[v] = axis_term(q, v, 1);
        iz[v] = axis_term(q, v, 2);
    }
    return axis_term(q, x, 0);
}

// Plane x of channels e0 .. e0 + EG - 1 of chain ch: shared [EG][L][P].
// SRC: T vectors psi [chain][nk][t], or (STENCIL) the stencil [t t][L^3] in mesh order.
template <typename T, bool STENCIL>
__global__ void __launch_bounds__(LTHR) k_lconv_fwd(const typename Cx<T>::V* __restrict__ src, const LShape q, int chan,
                                                    const float2* __restrict__ tw_g, float2* __restrict__ grid) {
    extern __shared__ float2 lsm[];
    const int L = q.L, P = q.P, L2 = L * L, x = blockIdx.x, e0 = blockIdx.y * EG, ch = blockIdx.z, tid = threadIdx.x;
    const int ne = min(EG, chan - e0);
    float2* tw = lsm;
    float2* s = lsm + 64;
    for (int i = tid; i < L; i += LTHR) tw[i] = tw_g[i];
    const size_t nk = (size_t)L2 * L;
    __shared__ int iy[64], iz[64];
    const int ix = axis_tables(q, x, iy, iz);
    const float inv_L = 1.f / (float)L;
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < L2 * EG; i += LTHR) {
        // vectors: the EG entries of a point side by side; stencil: points of a channel side by side
        const int e = STENCIL ? i / L2 : i & (EG - 1), p = STENCIL ? i - e * L2 : i / EG, y = quot(p, inv_L), z = p - y * L;
        float2 v = make_float2(0.f, 0.f);
        if (e < ne) {
            if constexpr (STENCIL) {
                v = src[(size_t)(e0 + e) * nk + (size_t)x * L2 + p];
            } else {
                const auto f = src[((size_t)ch * nk + ix + iy[y] + iz[z]) * q.t + e0 + e];
                v = make_float2((float)f.x, (float)f.y);
            }
        }
        s[(e * L + y) * P + z] = v;
    }
    __syncthreads();
    // z lines: one per (e, y); y lines: one per (e, z)
    lines_fwd(s, ne * L, [&](int l) { return l * P; }, 1, q.A, q.B, tw);
    lines_fwd(s, ne * L, [&](int l) { const int e = quot(l, inv_L); return e * (L - 1) * P + e * (P - L) + l; }, P, q.A, q.B, tw);
    float2* out = grid + (size_t)x * q.nch * chan + (size_t)ch * chan + e0;
    for (int i = tid; i < L2 * EG; i += LTHR) {
        const int e = i & (EG - 1), p = i / EG, y = quot(p, inv_L), z = p - y * L;
        if (e < ne) out[(size_t)p * L * q.nch * chan + e] = s[(e * L + y) * P + z];
    }
}

// Forward along x of channels c0 .. (gridDim.y chunks of `chunk`) at one (y, z): the stencil's last axis.
__global__ void __launch_bounds__(LTHR) k_lconv_x(float2* __restrict__ grid, const LShape q, int chan, int chunk,
                                                  const float2* __restrict__ tw_g) {
    extern __shared__ float2 lsm[];
    const int L = q.L, c0 = blockIdx.y * chunk, nc = min(chunk, chan - c0), tid = threadIdx.x;
    float2* tw = lsm;
    float2* s = lsm + 64;
    for (int i = tid; i < L; i += LTHR) tw[i] = tw_g[i];
    float2* g = grid + (size_t)blockIdx.x * L * chan + c0;
    for (int i = tid; i < L * nc; i += LTHR) s[i] = g[(size_t)(i / nc) * chan + i % nc];
    __syncthreads();
    lines_fwd(s, nc, [](int l) { return l; }, nc, q.A, q.B, tw);
    for (int i = tid; i < L * nc; i += LTHR) g[(size_t)(i / nc) * chan + i % nc] = s[i];
}

// One (y, z): DFT along x of every chain and transition, out[e1] = sum_e2 T[e1][e2] in[e2]
// at every x frequency, DFT back, in place.
template <int NCH>
__global__ void __launch_bounds__(LTHR) k_lconv_mix(float2* __restrict__ grid, const float2* __restrict__ That, const LShape q,
                                                    const float2* __restrict__ tw_g) {
    extern __shared__ float2 lsm[];
    const int L = q.L, t = q.t, c = NCH * t, tid = threadIdx.x;
    float2* tw = lsm;
    float2* a = lsm + 64;                  // [L][c]
    float2* b = a + L * c;
    for (int i = tid; i < L; i += LTHR) tw[i] = tw_g[i];
    float2* g = grid + (size_t)blockIdx.x * L * c;
    for (int i = tid; i < L * c; i += LTHR) a[i] = g[i];
    __syncthreads();
    lines_fwd(a, c, [](int l) { return l; }, c, q.A, q.B, tw);
    const float2* Tq = That + (size_t)blockIdx.x * L * t * t;
    const float inv_t = 1.f / (float)t;
    for (int i = tid; i < L * t; i += LTHR) {
        const int x = quot(i, inv_t), e1 = i - x * t;
        const float2* Tx = Tq + (size_t)x * t * t + e1;
        const float2* in = a + x * c;
        float2 acc[NCH];
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) acc[ch] = make_float2(0.f, 0.f);
#pragma unroll 8
        for (int e2 = 0; e2 < t; ++e2) {
            const float2 T = __ldcs(Tx + e2 * t);
#pragma unroll
            for (int ch = 0; ch < NCH; ++ch) {
                const float2 v = in[ch * t + e2];
                acc[ch].x = fmaf(T.x, v.x, fmaf(-T.y, v.y, acc[ch].x));
                acc[ch].y = fmaf(T.x, v.y, fmaf(T.y, v.x, acc[ch].y));
            }
        }
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) b[x * c + ch * t + e1] = acc[ch];
    }
    __syncthreads();
    lines_inv(b, c, [](int l) { return l; }, c, q.A, q.B, tw);
    for (int i = tid; i < L * c; i += LTHR) g[i] = b[i];
}

// Back along y and z, w += scale * value, and the block's FP64 partial of <psi, w>.
template <typename T>
__global__ void __launch_bounds__(LTHR) k_lconv_inv(const float2* __restrict__ grid, const LShape q,
                                                    const float2* __restrict__ tw_g, const typename Cx<T>::V* __restrict__ psi,
                                                    typename Cx<T>::V* __restrict__ w, float scale, double2* __restrict__ part) {
    using V = typename Cx<T>::V;
    extern __shared__ float2 lsm[];
    __shared__ double2 red[LTHR / 32];
    const int L = q.L, P = q.P, L2 = L * L, x = blockIdx.x, e0 = blockIdx.y * EG, ch = blockIdx.z, tid = threadIdx.x;
    const int ne = min(EG, q.t - e0);
    float2* tw = lsm;
    float2* s = lsm + 64;
    for (int i = tid; i < L; i += LTHR) tw[i] = tw_g[i];
    const float2* in = grid + (size_t)x * q.nch * q.t + (size_t)ch * q.t + e0;
    __shared__ int iy[64], iz[64];
    const int ix = axis_tables(q, x, iy, iz);
    const float inv_L = 1.f / (float)L;
#pragma unroll 4
    for (int i = tid; i < L2 * EG; i += LTHR) {
        const int e = i & (EG - 1), p = i / EG, y = quot(p, inv_L), z = p - y * L;
        if (e < ne) s[(e * L + y) * P + z] = in[(size_t)p * L * q.nch * q.t + e];
    }
    __syncthreads();
    lines_inv(s, ne * L, [&](int l) { const int e = quot(l, inv_L); return e * (L - 1) * P + e * (P - L) + l; }, P, q.A, q.B, tw);
    lines_inv(s, ne * L, [&](int l) { return l * P; }, 1, q.A, q.B, tw);
    const size_t nk = (size_t)L2 * L;
    DotSum<T> dot = DotSum<T>::zero();
#pragma unroll 4
    for (int i = tid; i < L2 * EG; i += LTHR) {
        const int e = i & (EG - 1), p = i / EG, y = quot(p, inv_L), z = p - y * L;
        if (e >= ne) continue;
        const size_t o = ((size_t)ch * nk + ix + iy[y] + iz[z]) * q.t + e0 + e;
        const float2 g = s[(e * L + y) * P + z];
        const V pv = psi[o];
        V v = w[o];
        v.x = fma((T)g.x, (T)scale, v.x);
        v.y = fma((T)g.y, (T)scale, v.y);
        w[o] = v;
        dot.add(pv, v);
    }
    double2 d = dot.value();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        d.x += __shfl_down_sync(0xffffffffu, d.x, o);
        d.y += __shfl_down_sync(0xffffffffu, d.y, o);
    }
    if ((tid & 31) == 0) red[tid >> 5] = d;
    __syncthreads();
    if (tid == 0) {
        double2 r = red[0];
        for (int i = 1; i < LTHR / 32; ++i) r = cadd(r, red[i]);
        part[(size_t)ch * BSE_MAX_VEC_BLOCKS + (size_t)blockIdx.y * L + x] = r;
    }
}

// L = A B with A, B <= 8, as even as possible; false when there is none.
bool factor(int L, int* A, int* B) {
    for (int a = (int)std::sqrt((double)L); a >= 1; --a)
        if (L % a == 0 && L / a <= 8) {
            *A = a;
            *B = L / a;
            return true;
        }
    return false;
}

LShape shape(const bse_interp* s, int nch) {
    LShape q{};
    q.L = s->n * s->nd; q.n = s->n; q.nd = s->nd; q.t = s->t; q.nch = nch; q.P = q.L | 1;
    factor(q.L, &q.A, &q.B);
    return q;
}

size_t plane_smem(int L) { return sizeof(float2) * (64 + (size_t)EG * L * (L | 1)); }
constexpr size_t kPlaneFixed = 1024;          // axis tables and warp sums, rounded up
size_t mix_smem(int L, int t, int nch) { return sizeof(float2) * (64 + 2 * (size_t)L * nch * t); }

template <typename T>
int apply_typed(bse_ctx* ctx, const bse_interp* s, int nch, const void* psi, void* w, double2* dot) {
    using V = typename Cx<T>::V;
    const LShape q = shape(s, nch);
    const int L = q.L, eb = (s->t + EG - 1) / EG;
    cudaStream_t st = ctx->stream;
    const size_t ps = plane_smem(L), ms = mix_smem(L, s->t, nch);
    BSE_CUDA_TRY(ctx, bse_raise_smem((k_lconv_fwd<T, false>), ps, kPlaneFixed));
    BSE_CUDA_TRY(ctx, bse_raise_smem(k_lconv_inv<T>, ps, kPlaneFixed));
    k_lconv_fwd<T, false><<<dim3(L, eb, nch), LTHR, ps, st>>>((const V*)psi, q, s->t, s->d_tw_fwd, s->d_lgrid);
    auto mix = [&](auto kernel) -> int {
        BSE_CUDA_TRY(ctx, bse_raise_smem(kernel, ms));
        kernel<<<L * L, LTHR, ms, st>>>(s->d_lgrid, s->d_lker, q, s->d_tw_fwd);
        return BSE_OK;
    };
    const int rc = nch == 1 ? mix(k_lconv_mix<1>) : nch == 2 ? mix(k_lconv_mix<2>) : nch == 3 ? mix(k_lconv_mix<3>) : mix(k_lconv_mix<4>);
    if (rc != BSE_OK) return rc;
    k_lconv_inv<T><<<dim3(L, eb, nch), LTHR, ps, st>>>(s->d_lgrid, q, s->d_tw_fwd, (const V*)psi, (V*)w,
                                                        1.f / ((float)L * L * L), dot);
    BSE_CUDA_TRY(ctx, cudaGetLastError());
    return BSE_OK;
}

}  // namespace

// Whether the three-kernel convolution serves this handle: a line length A B with
// A, B <= 8, planes and columns that fit in shared memory, and no more dot partials
// per chain than the buffer holds.
bool bse_lconv_usable(const bse_ctx* ctx, const bse_interp* s) {
    const int L = s->n * s->nd;
    int A, B, maxsm = 0;
    cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device);
    return L <= 64 && factor(L, &A, &B) && plane_smem(L) + 1024 <= (size_t)maxsm &&
           mix_smem(L, s->t, BSE_MAX_CHAINS) + 1024 <= (size_t)maxsm && bse_lconv_dot_blocks(s) <= BSE_MAX_VEC_BLOCKS;
}

int bse_lconv_dot_blocks(const bse_interp* s) { return s->n * s->nd * ((s->t + EG - 1) / EG); }

// Transform of the stencil: `ker` [t t][L^3] in mesh order (channel e2 t + e1) into `out` [y z][x][t t].
int bse_lconv_kernel(bse_ctx* ctx, const bse_interp* s, const float2* ker, float2* out) {
    const LShape q = shape(s, 1);
    const int L = q.L, chan = s->t * s->t, chunk = std::min(chan, 2048 / L);
    const size_t ps = plane_smem(L), xs = sizeof(float2) * (64 + (size_t)L * chunk);
    BSE_CUDA_TRY(ctx, bse_raise_smem((k_lconv_fwd<float, true>), ps, kPlaneFixed));
    BSE_CUDA_TRY(ctx, bse_raise_smem(k_lconv_x, xs));
    k_lconv_fwd<float, true><<<dim3(L, (chan + EG - 1) / EG, 1), LTHR, ps, ctx->stream>>>(ker, q, chan, s->d_tw_fwd, out);
    k_lconv_x<<<dim3(L * L, (chan + chunk - 1) / chunk), LTHR, xs, ctx->stream>>>(out, q, chan, chunk, s->d_tw_fwd);
    BSE_CUDA_TRY(ctx, cudaGetLastError());
    return BSE_OK;
}

int bse_lconv_apply(bse_ctx* ctx, const bse_interp* s, int nch, const void* psi, void* w, double2* dot) {
    return s->vec_prec == BSE_PREC_F64 ? apply_typed<double>(ctx, s, nch, psi, w, dot)
                                       : apply_typed<float>(ctx, s, nch, psi, w, dot);
}
