// H application in the common reference basis of the band gauge.
//
// When the dense tables come from the model (no overlaps given by the caller)
// every overlap is a product through one reference basis (Eq. completeness),
//   d(k, k~) = U(k~)^H U(k),   U unitary (Hermitian gauge generators),
// so the interpolation F of Eq. interpwfn and the Method-3 head A = alpha O^v (x) O^c
// factor through it.  With phi(k) = conj(Uv(k)) psi(k) Uc(k)^T ("to common"):
//   restrict   Q(k~)  = from_common_k~[ sum_k f(k, k~) phi(k) ]               (Eq. matmul1)
//   prolong    s(k)   = from_common_k[ sum_l f(k, l) to_common_k~l[R(k~_l)] ]  (Eq. matmul3)
//   near pairs V(k)   = sum_delta W(j(k), delta) phi(k + delta),
//              W = alpha [ h_head(q_dense) - sum_{l,l'} f(k,l) f(k',l') h_head(q_coarse(l,l')) ]
//   w = dE psi + (1/N_div) from_common_k[ interpolated R + V ].
// The unitary factors of neighbouring corners cancel, which the paper's own
// order of operations does not use: one rotation per dense point instead of
// one per (point, corner), and a scalar stencil instead of a t x t head block
// per (corner, corner) pair.  W depends on the sub-cell position and the
// offset alone; set-up evaluates it once in FP64.
// Measured on GB300, one H application, against the general kernels: coarse 8^3,
// n_div 4, 4x4 bands, 3 vectors FP64 98.5 -> 9.45 ms; coarse 4^3, n_div 2, 3x3
// bands, 1 vector FP64 1105 -> 140 us; coarse 7^3, n_div 3, 3x5 bands, 4 vectors
// FP32 1.80 -> 0.44 ms.
// Caller-supplied overlaps (not a product through one basis) and non-Hermitian
// generators keep the general kernels of bse_apply.cu and bse_near_tc.cu.
#include <algorithm>
#include <cmath>

#include "bse_internal.cuh"

namespace {

__host__ __device__ constexpr int odd(int x) { return x | 1; }

__device__ __forceinline__ void cpa16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// acc += a b, acc += a conj(b), with fused multiply-adds
template <typename V>
__device__ __forceinline__ void cfma(V& acc, V a, V b) {
    acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
    acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
}
template <typename V>
__device__ __forceinline__ void cfmac(V& acc, V a, V b) {
    acc.x = fma(a.x, b.x, fma(a.y, b.y, acc.x));
    acc.y = fma(a.y, b.x, fma(-a.x, b.y, acc.y));
}

// i / len for small i (len <= 64 entries, i < 2^13: the quotient is at least 1/128
// away from the next integer), with the reciprocal of len: integer divisions by
// run-time lengths were most of these kernels' instructions.
__device__ __forceinline__ int quot(int i, float inv) { return (int)(((float)i + 0.5f) * inv); }

// One row (fixed valence index) of a point's block, in place:
// TO: y[m] = sum_c x[c] Uc[m][c];  else y[c] = sum_m x[m] conj(Uc[m][c]).
template <bool TO, int NB, typename V>
__device__ __forceinline__ void rot_row(V* x, const V* U) {
    V in[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) in[i] = x[i];
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        V a = czero<V>();
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            if (TO) cfma(a, in[i], U[j * NB + i]);
            else cfmac(a, in[i], U[i * NB + j]);
        }
        x[j] = a;
    }
}
// One column (fixed conduction index), in place, element stride `st`:
// TO: y[m] = sum_v conj(Uv[m][v]) x[v];  else y[v] = sum_m Uv[m][v] x[m].
template <bool TO, int NB, typename V>
__device__ __forceinline__ void rot_col(V* x, int st, const V* U) {
    V in[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) in[i] = x[i * st];
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        V a = czero<V>();
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            if (TO) cfmac(a, in[i], U[j * NB + i]);
            else cfma(a, in[i], U[i * NB + j]);
        }
        x[j * st] = a;
    }
}

// Rotation of `np` blocks x [np][tp] (t = nv nc entries each) in shared memory
// by Uv [np][rvp], Uc [np][rcp]; block-wide, ends with a barrier.  One thread
// per row, then one per column: 1 shared load per complex multiply-add, rows
// padded to an odd number of entries so that a warp's rows spread over the banks.
template <bool TO, typename V>
__device__ __forceinline__ void rotate_blocks(V* x, int tp, const V* Uv, int rvp, const V* Uc, int rcp, int np, int nv,
                                              int nc) {
    const float inv_v = 1.f / (float)nv, inv_c = 1.f / (float)nc;
    for (int i = threadIdx.x; i < np * nv; i += blockDim.x) {
        const int p = quot(i, inv_v), v = i - p * nv;
        V* r = x + p * tp + v * nc;
        const V* U = Uc + p * rcp;
        switch (nc) {
            case 1: rot_row<TO, 1>(r, U); break;
            case 2: rot_row<TO, 2>(r, U); break;
            case 3: rot_row<TO, 3>(r, U); break;
            case 4: rot_row<TO, 4>(r, U); break;
            case 5: rot_row<TO, 5>(r, U); break;
            case 6: rot_row<TO, 6>(r, U); break;
            case 7: rot_row<TO, 7>(r, U); break;
            default: rot_row<TO, 8>(r, U); break;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < np * nc; i += blockDim.x) {
        const int p = quot(i, inv_c), c = i - p * nc;
        V* r = x + p * tp + c;
        const V* U = Uv + p * rvp;
        switch (nv) {
            case 1: rot_col<TO, 1>(r, nc, U); break;
            case 2: rot_col<TO, 2>(r, nc, U); break;
            case 3: rot_col<TO, 3>(r, nc, U); break;
            case 4: rot_col<TO, 4>(r, nc, U); break;
            case 5: rot_col<TO, 5>(r, nc, U); break;
            case 6: rot_col<TO, 6>(r, nc, U); break;
            case 7: rot_col<TO, 7>(r, nc, U); break;
            default: rot_col<TO, 8>(r, nc, U); break;
        }
    }
    __syncthreads();
}

// Rows of `len` entries from global src (row r at src + r * len) into shared dst (row pitch `pitch`).
template <typename V>
__device__ __forceinline__ void load_rows(V* dst, int pitch, const V* __restrict__ src, int rows, int len) {
    const float inv = 1.f / (float)len;
    for (int i = threadIdx.x; i < rows * len; i += blockDim.x) {
        const int r = quot(i, inv);
        dst[r * pitch + (i - r * len)] = src[i];
    }
}

// Weight of corner l at sub-cell position (j1, j2, j3) (interp_weight).
template <typename T>
__device__ __forceinline__ T corner_weight(int j1, int j2, int j3, int l, int nd, int nb1) {
    const int l1 = (l >> 2) & 1, l2 = (l >> 1) & 1, l3 = l & 1;
    if (nb1) return ((2 * j1 > nd) == l1 && (2 * j2 > nd) == l2 && (2 * j3 > nd) == l3) ? (T)1 : (T)0;
    return (T)((l1 ? j1 : nd - j1) * (l2 ? j2 : nd - j2) * (l3 ? j3 : nd - j3)) / (T)(nd * nd * nd);
}

// ------------------------------------------------------- rotate and restrict
// Grid (coarse cell, chain).  The cell's points go through in chunks of KP:
// psi and the gauge matrices are staged in shared memory, rotated, written to
// the near field's phi (layout of CommonPhi) and summed with the trilinear
// weights into the cell's share of its eight corners.  The block whose share of
// a coarse point is the last of eight (a counter per point and chain, reset
// there) adds the eight in corner order, rotates the sum back and writes Q: the
// order does not depend on the blocks' order.
template <typename T, bool OUT_BF16>
__global__ void __launch_bounds__(256) k_common_restrict(
    const typename Cx<T>::V* __restrict__ psi, const typename Cx<T>::V* __restrict__ Uvd,
    const typename Cx<T>::V* __restrict__ Ucd, const typename Cx<T>::V* __restrict__ Uvc,
    const typename Cx<T>::V* __restrict__ Ucc, int n, int nd, int nv, int nc, int nb1, int KP,
    T* __restrict__ phi, CommonPhi lay, typename Cx<T>::V* __restrict__ share, int* __restrict__ ctr,
    typename Cx<T>::V* __restrict__ Q, __nv_bfloat16* __restrict__ Bop, int ldk) {
    using V = typename Cx<T>::V;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int last_sh[8];
    const int t = nv * nc, tp = odd(t), rv = nv * nv, rc = nc * nc, rvp = odd(rv), rcp = odd(rc);
    const int Ndiv = nd * nd * nd, nkc = n * n * n, nch = gridDim.y;
    const int ic = blockIdx.x, ch = blockIdx.y, tid = threadIdx.x;
    const Int3 ci = unflat3(ic, n);
    V* X = reinterpret_cast<V*>(smraw);                 // [KP][tp]
    V* sUv = X + KP * tp;                               // [KP][rvp]
    V* sUc = sUv + KP * rvp;                            // [KP][rcp]
    V* red = sUc + KP * rcp;                            // [256]
    T* wt = reinterpret_cast<T*>(red + 256);            // [KP][8]
    int2* pnt = reinterpret_cast<int2*>(wt + KP * 8);   // [KP] the point's place in phi and its halo copy's distance
    const int L = n * nd, t2 = 2 * t;
    const float inv_t = 1.f / (float)t, inv_nd = 1.f / (float)nd;
    // corner sums: item (l, e); with few items several threads share one over the points
    const int items = 8 * t, nsp = max(1, 256 / items);
    V acc[2] = {czero<V>(), czero<V>()};
    for (int k0 = 0; k0 < Ndiv; k0 += KP) {
        const int np = min(KP, Ndiv - k0);
        const size_t kd0 = (size_t)ic * Ndiv + k0;
        load_rows(X, tp, psi + ((size_t)ch * nkc * Ndiv + kd0) * t, np, t);
        load_rows(sUv, rvp, Uvd + kd0 * rv, np, rv);
        load_rows(sUc, rcp, Ucd + kd0 * rc, np, rc);
        for (int i = tid; i < np * 8; i += 256) {
            const int js = k0 + (i >> 3), a = quot(js, inv_nd), j3 = js - a * nd, j1 = quot(a, inv_nd), j2 = a - j1 * nd;
            wt[i] = corner_weight<T>(j1, j2, j3, i & 7, nd, nb1);
            if ((i & 7) == 0) {
                const int x = ci.a * nd + j1, y = ci.b * nd + j2, z = ci.c * nd + j3;
                pnt[i >> 3] = make_int2((x * L + y) * lay.Lp + z + lay.R, z < lay.R ? L : (z >= L - lay.R ? -L : 0));
            }
        }
        __syncthreads();
        rotate_blocks<true>(X, tp, sUv, rvp, sUc, rcp, np, nv, nc);
        if (phi) {
            // the 2 t components of a point lie side by side in the columns of its groups
            const size_t gs = (size_t)L * L * lay.Lp * 32;
            const float inv_t2 = 1.f / (float)t2;
            for (int i = tid; i < np * t2; i += 256) {
                const int r = quot(i, inv_t2), q = i - r * t2, col = ch * t2 + q;
                const int2 pt = pnt[r];
                const T v = reinterpret_cast<const T*>(X + r * tp)[q];
                T* at = phi + (size_t)(col >> 5) * gs + (size_t)pt.x * 32 + (col & 31);
                *at = v;
                if (pt.y) at[(ptrdiff_t)pt.y * 32] = v;
            }
        }
        for (int a = 0; a < 2; ++a) {
            const int i = nsp > 1 ? tid % items : tid + 256 * a, sp = nsp > 1 ? tid / items : 0;
            if (i >= items || sp >= nsp || (nsp > 1 && a)) continue;
            const int l = quot(i, inv_t), e = i - l * t;
            V s = acc[a];
            for (int r = sp; r < np; r += nsp) {
                const T f = wt[r * 8 + l];
                const V v = X[r * tp + e];
                s.x = fma(f, v.x, s.x);
                s.y = fma(f, v.y, s.y);
            }
            acc[a] = s;
        }
        __syncthreads();
    }
    // the cell's shares: [chain][cell][corner][t]
    V* mine = share + ((size_t)ch * nkc + ic) * items;
    if (nsp > 1) {
        red[tid] = acc[0];
        __syncthreads();
        if (tid < items) {
            V s = red[tid];
            for (int q = 1; q < nsp; ++q) s = cadd(s, red[q * items + tid]);
            mine[tid] = s;
        }
    } else {
        for (int a = 0; a < 2; ++a)
            if (tid + 256 * a < items) mine[tid + 256 * a] = acc[a];
    }
    __threadfence();
    __syncthreads();
    if (tid < 8) {
        const int dst = flat3(ci.a + ((tid >> 2) & 1), ci.b + ((tid >> 1) & 1), ci.c + (tid & 1), n);
        int* c = ctr + (size_t)ch * nkc + dst;
        const bool last = atomicAdd(c, 1) == 7;
        if (last) *c = 0;
        last_sh[tid] = last ? dst : -1;
        __threadfence();
    }
    __syncthreads();
    for (int l = 0; l < 8; ++l) {
        const int dst = last_sh[l];
        if (dst < 0) continue;
        const Int3 d = unflat3(dst, n);
        for (int e = tid; e < t; e += 256) {
            V s = czero<V>();
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int cell = flat3(d.a - ((q >> 2) & 1), d.b - ((q >> 1) & 1), d.c - (q & 1), n);
                s = cadd(s, __ldcg(share + ((size_t)ch * nkc + cell) * items + q * t + e));
            }
            X[e] = s;
        }
        for (int i = tid; i < rv; i += 256) sUv[i] = Uvc[(size_t)dst * rv + i];
        for (int i = tid; i < rc; i += 256) sUc[i] = Ucc[(size_t)dst * rc + i];
        __syncthreads();
        rotate_blocks<false>(X, tp, sUv, rvp, sUc, rcp, 1, nv, nc);
        for (int e = tid; e < t; e += 256) {
            const V s = X[e];
            const size_t row = (size_t)dst * t + e;
            if (!OUT_BF16) {
                Q[(size_t)ch * nkc * t + row] = s;
            } else {
                // split-BF16 operand of the tensor-core apply: rows (Re hi, Im hi, Re lo, Im lo) x chains
                const float re = (float)s.x, im = (float)s.y;
                const __nv_bfloat16 rh = __float2bfloat16_rn(re), ih = __float2bfloat16_rn(im);
                Bop[(size_t)ch * ldk + row] = rh;
                Bop[(size_t)(nch + ch) * ldk + row] = ih;
                Bop[(size_t)(2 * nch + ch) * ldk + row] = __float2bfloat16_rn(re - __bfloat162float(rh));
                Bop[(size_t)(3 * nch + ch) * ldk + row] = __float2bfloat16_rn(im - __bfloat162float(ih));
            }
        }
        __syncthreads();
    }
}

// ------------------------------------------------------- prolong and diagonal
// Grid (coarse cell, grid-strided; chain): w = dE psi + from_common[(1/N_div) sum_l f R'(k~_l) + V],
// R' = to_common(R) at the cell's eight corners, V the near stencil (its weights
// carry alpha / N_div); FP64 block partials of <psi, w>.
template <typename T>
__global__ void __launch_bounds__(256) k_common_prolong(
    const typename Cx<T>::V* __restrict__ R, const typename Cx<T>::V* __restrict__ Vn,
    const typename Cx<T>::V* __restrict__ Uvd, const typename Cx<T>::V* __restrict__ Ucd,
    const typename Cx<T>::V* __restrict__ Uvc, const typename Cx<T>::V* __restrict__ Ucc, const T* __restrict__ dE,
    const typename Cx<T>::V* __restrict__ psi, int n, int nd, int nv, int nc, int nb1, int KP,
    typename Cx<T>::V* __restrict__ W, double2* __restrict__ part) {
    using V = typename Cx<T>::V;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ double2 dred[8];
    const int t = nv * nc, tp = odd(t), rv = nv * nv, rc = nc * nc, rvp = odd(rv), rcp = odd(rc);
    const int Ndiv = nd * nd * nd, nkc = n * n * n, ch = blockIdx.y, tid = threadIdx.x;
    V* X = reinterpret_cast<V*>(smraw);                 // [KP][tp]
    V* sUv = X + KP * tp;                               // [KP][rvp]
    V* sUc = sUv + KP * rvp;                            // [KP][rcp]
    V* Rc = sUc + KP * rcp;                             // [8][tp]
    V* cUv = Rc + 8 * tp;                               // [8][rvp]
    V* cUc = cUv + 8 * rvp;                             // [8][rcp]
    T* wt = reinterpret_cast<T*>(cUc + 8 * rcp);        // [KP][8]
    const T inv = (T)1 / (T)Ndiv;
    const float inv_t = 1.f / (float)t, inv_nd = 1.f / (float)nd;
    double2 dot = make_double2(0.0, 0.0);
    for (int cell = blockIdx.x; cell < nkc; cell += gridDim.x) {
        const Int3 ci = unflat3(cell, n);
        __syncthreads();
        for (int i = tid; i < 8 * (t + rv + rc); i += 256) {
            const int l = i & 7, q = i >> 3;
            const size_t cc = flat3(ci.a + ((l >> 2) & 1), ci.b + ((l >> 1) & 1), ci.c + (l & 1), n);
            if (q < t) Rc[l * tp + q] = R[((size_t)ch * nkc + cc) * t + q];
            else if (q < t + rv) cUv[l * rvp + (q - t)] = Uvc[cc * rv + (q - t)];
            else cUc[l * rcp + (q - t - rv)] = Ucc[cc * rc + (q - t - rv)];
        }
        __syncthreads();
        rotate_blocks<true>(Rc, tp, cUv, rvp, cUc, rcp, 8, nv, nc);
        for (int k0 = 0; k0 < Ndiv; k0 += KP) {
            const int np = min(KP, Ndiv - k0);
            const size_t kd0 = (size_t)cell * Ndiv + k0, g0 = kd0 * t, o0 = (size_t)ch * nkc * Ndiv * t + g0;
            load_rows(sUv, rvp, Uvd + kd0 * rv, np, rv);
            load_rows(sUc, rcp, Ucd + kd0 * rc, np, rc);
            for (int i = tid; i < np * 8; i += 256) {
                const int js = k0 + (i >> 3), a = quot(js, inv_nd), j1 = quot(a, inv_nd);
                wt[i] = corner_weight<T>(j1, a - j1 * nd, js - a * nd, i & 7, nd, nb1) * inv;
            }
            __syncthreads();
            for (int i = tid; i < np * t; i += 256) {
                const int r = quot(i, inv_t), e = i - r * t;
                V s = Vn ? Vn[o0 + i] : czero<V>();
#pragma unroll
                for (int l = 0; l < 8; ++l) {
                    const T f = wt[r * 8 + l];
                    const V v = Rc[l * tp + e];
                    s.x = fma(f, v.x, s.x);
                    s.y = fma(f, v.y, s.y);
                }
                X[r * tp + e] = s;
            }
            __syncthreads();
            rotate_blocks<false>(X, tp, sUv, rvp, sUc, rcp, np, nv, nc);
            T dre = (T)0, dim = (T)0;                   // this thread's few products, then FP64
            for (int i = tid; i < np * t; i += 256) {
                const int r = quot(i, inv_t), e = i - r * t;
                const V s = X[r * tp + e], p = psi[o0 + i];
                const T de = dE[g0 + i];
                V w;
                w.x = fma(p.x, de, s.x);
                w.y = fma(p.y, de, s.y);
                W[o0 + i] = w;
                dre = fma(p.x, w.x, fma(p.y, w.y, dre));
                dim = fma(p.x, w.y, fma(-p.y, w.x, dim));
            }
            dot.x += (double)dre;
            dot.y += (double)dim;
            __syncthreads();
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        dot.x += __shfl_down_sync(0xffffffffu, dot.x, o);
        dot.y += __shfl_down_sync(0xffffffffu, dot.y, o);
    }
    if ((tid & 31) == 0) dred[tid >> 5] = dot;
    __syncthreads();
    if (tid == 0) {
        double2 s = dred[0];
        for (int w = 1; w < 8; ++w) s = cadd(s, dred[w]);
        part[(size_t)ch * BSE_MAX_VEC_BLOCKS + blockIdx.x] = s;
    }
}

// ----------------------------------------------------------- near stencil
// V(k) = sum_delta W(j, delta) phi(k + delta) over the near offsets |delta|^2 <= R2.
//
// Per target and column (one real component of one chain) one multiply-add per
// near offset is needed: 808 M for coarse 8^3, n_div 4, w 1, 3 chains of 16
// transitions.  A warp takes one column group (a column per lane) and TY rows
// (j1, j2 .. j2 + TY - 1) of CZ cells that follow each other along z: their
// targets are CZ TZ consecutive points, so one load of a source column serves up
// to TY (2 r + 1) multiply-adds, and since W is the same in every cell one
// broadcast vector load of TZ weights serves CZ multiply-adds each.  It walks
// the source rows (delta_1, row u) of its ball in set-up's list; the reach r of
// each target row along z is a case of a switch, so only offsets inside the ball
// cost arithmetic and the source row sits in registers.  Sources come straight
// from phi (the warps of a block share their cells, hence rows, through L1);
// the weights of the next row are copied to the warp's buffer meanwhile.
// RM: the largest r that the unrolled body covers (R <= RM); RM = 0 loops over z.
struct NearStencil {
    int n, L, Lp, R, nd, njb, nzb, nsteps, wrow;   // njb: blocks of TY rows j2; nzb: blocks of TZ targets j3
    int cols, t2, ntz, warps;                      // columns in use, 2 t, z tiles (of cz cells, the last ones smaller), all warps
    int cz;
    long long N2;                                  // 2 N: reals per chain of V
};

template <typename T, int TZ>
__device__ __forceinline__ void load_w(T (&w)[TZ], const T* p) {
    if constexpr (TZ >= 3 && sizeof(T) == 4) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        w[0] = q.x; w[1] = q.y; w[2] = q.z;
        if (TZ == 4) w[TZ - 1] = q.w;
    } else if constexpr (TZ >= 2) {
        using V = typename Cx<T>::V;
        const V q = reinterpret_cast<const V*>(p)[0];
        w[0] = q.x; w[1] = q.y;
        if (TZ >= 3) {
            const V q2 = reinterpret_cast<const V*>(p)[1];
            w[2] = q2.x;
            if (TZ == 4) w[TZ - 1] = q2.y;
        }
    } else {
        w[0] = p[0];
    }
}

// acc += W v for the target rows of one cell run that reach r sources to each side
template <typename T, int TZ, int CZ, int RM, int r>
__device__ __forceinline__ void near_apply(T (&acc)[CZ * TZ], const T (&v)[CZ * TZ + 2 * RM], const T* wb) {
    constexpr int TZP = TZ == 3 ? 4 : TZ;
#pragma unroll
    for (int z = -r; z < TZ + r; ++z) {
        T w[TZ];
        load_w<T, TZ>(w, wb + z * TZP);
#pragma unroll
        for (int tz = 0; tz < TZ; ++tz)
            if (z - tz <= r && tz - z <= r) {
#pragma unroll
                for (int c = 0; c < CZ; ++c) acc[c * TZ + tz] = fma(w[tz], v[c * TZ + z + RM], acc[c * TZ + tz]);
            }
    }
}
// One source row that reaches rm: its columns into registers, then every target
// row by its own reach r <= rm (code + 1; 0: not reached).  A body per rm: a row
// array shared by several bodies cost a register move per element.
template <typename T, int TY, int TZ, int CZ, int rm>
__device__ __forceinline__ void near_row(T (&acc)[TY][CZ * TZ], const T* __restrict__ row, const T* wb, int wy, int reach) {
    T v[CZ * TZ + 2 * rm];
#pragma unroll
    for (int z = -rm; z < CZ * TZ + rm; ++z) v[z + rm] = __ldg(row + z * 32);
    cpa_wait<1>();
    __syncwarp();
#pragma unroll
    for (int y = 0; y < TY; ++y) {
        const T* w = wb + y * wy;
        const int r = ((reach >> (8 * y)) & 255) - 1;
        if (r == rm) near_apply<T, TZ, CZ, rm, rm>(acc[y], v, w);
        if constexpr (rm >= 1) if (r == 0) near_apply<T, TZ, CZ, rm, 0>(acc[y], v, w);
        if constexpr (rm >= 2) if (r == 1) near_apply<T, TZ, CZ, rm, 1>(acc[y], v, w);
        if constexpr (rm >= 3) if (r == 2) near_apply<T, TZ, CZ, rm, 2>(acc[y], v, w);
        if constexpr (rm >= 4) if (r == 3) near_apply<T, TZ, CZ, rm, 3>(acc[y], v, w);
        if constexpr (rm >= 5) if (r == 4) near_apply<T, TZ, CZ, rm, 4>(acc[y], v, w);
        if constexpr (rm >= 6) if (r == 5) near_apply<T, TZ, CZ, rm, 5>(acc[y], v, w);
    }
}

template <typename T, int TY, int TZ, int CZ, int RM>
__device__ __forceinline__ void near_body(const T* __restrict__ phi, const T* __restrict__ Wt,
                                          const int2* __restrict__ steps, T* __restrict__ Vn, const NearStencil& s, int g,
                                          int cx, int cy, int cz0, int j1, int j2, int zb, T* wbuf) {
    constexpr int TZP = TZ == 3 ? 4 : TZ, PER = 16 / sizeof(T);
    const int lane = threadIdx.x & 31, nd = s.nd, R = s.R, nzs = TZ + 2 * R;
    const T* wsrc = Wt + (size_t)((zb * nd + j1) * s.njb + j2 / TY) * s.nsteps * s.wrow;
    const int xb = cx * nd + j1 - R, yb = cy * nd + j2 - R;
    const T* base = phi + (size_t)g * s.L * s.L * s.Lp * 32 + (size_t)(cz0 * nd + zb * TZ + R) * 32 + lane;
    T acc[TY][CZ * TZ];
#pragma unroll
    for (int y = 0; y < TY; ++y)
#pragma unroll
        for (int z = 0; z < CZ * TZ; ++z) acc[y][z] = (T)0;
    auto fetch = [&](int i) {
        T* dst = wbuf + (i & 1) * s.wrow;
        for (int c = lane * PER; c < s.wrow; c += 32 * PER) cpa16(dst + c, wsrc + (size_t)i * s.wrow + c);
        cpa_commit();
    };
    int2 st = steps[0];
    fetch(0);
    for (int i = 0; i < s.nsteps; ++i) {
        int2 nx = st;
        if (i + 1 < s.nsteps) {
            nx = steps[i + 1];
            fetch(i + 1);
        } else {
            cpa_commit();
        }
        // st: delta_1 + R | u << 8 | r_max << 16, then the reach + 1 of each target row (0: none), a byte each
        int x = xb + (st.x & 255), y = yb + ((st.x >> 8) & 255);
        x += x < 0 ? s.L : (x >= s.L ? -s.L : 0);
        y += y < 0 ? s.L : (y >= s.L ? -s.L : 0);
        const T* row = base + ((size_t)x * s.L + y) * s.Lp * 32;
        const int rm = st.x >> 16;
        const T* wb = wbuf + (i & 1) * s.wrow + R * TZP;
        if constexpr (RM > 0) {
            switch (rm) {
                case 0: near_row<T, TY, TZ, CZ, 0>(acc, row, wb, nzs * TZP, st.y); break;
                case 1: near_row<T, TY, TZ, CZ, 1>(acc, row, wb, nzs * TZP, st.y); break;
                case 2: near_row<T, TY, TZ, CZ, 2>(acc, row, wb, nzs * TZP, st.y); break;
                case 3: near_row<T, TY, TZ, CZ, 3>(acc, row, wb, nzs * TZP, st.y); break;
                case 4: near_row<T, TY, TZ, CZ, 4>(acc, row, wb, nzs * TZP, st.y); break;
                default:
                    if constexpr (RM >= 6) {
                        if (rm == 5) near_row<T, TY, TZ, CZ, 5>(acc, row, wb, nzs * TZP, st.y);
                        else near_row<T, TY, TZ, CZ, 6>(acc, row, wb, nzs * TZP, st.y);
                    }
            }
        } else {
            cpa_wait<1>();
            __syncwarp();
            for (int z = -rm; z < TZ + rm; ++z) {
                T v[CZ];
#pragma unroll
                for (int c = 0; c < CZ; ++c) v[c] = __ldg(row + (c * TZ + z) * 32);
#pragma unroll
                for (int y2 = 0; y2 < TY; ++y2) {
                    T w[TZ];
                    load_w<T, TZ>(w, wb + (y2 * nzs + z) * TZP);
#pragma unroll
                    for (int tz = 0; tz < TZ; ++tz)
#pragma unroll
                        for (int c = 0; c < CZ; ++c) acc[y2][c * TZ + tz] = fma(w[tz], v[c], acc[y2][c * TZ + tz]);
                }
            }
        }
        __syncwarp();
        st = nx;
    }
    const int col = g * 32 + lane;
    if (col >= s.cols) return;
    const int ch = col / s.t2, q = col - ch * s.t2;
    T* out = Vn + (size_t)ch * s.N2 + q;
#pragma unroll
    for (int c = 0; c < CZ; ++c)
#pragma unroll
        for (int y = 0; y < TY; ++y)
#pragma unroll
            for (int z = 0; z < TZ; ++z)
                if (j2 + y < nd && zb * TZ + z < nd) {
                    const size_t kd = ((size_t)((cx * s.n + cy) * s.n + cz0 + c) * nd + j1) * nd * nd + (j2 + y) * nd + zb * TZ + z;
                    out[kd * s.t2] = acc[y][c * TZ + z];
                }
}

template <typename T, int TY, int TZ, int RM>
__global__ void __launch_bounds__(256) k_common_near(const T* __restrict__ phi, const T* __restrict__ Wt,
                                                     const int2* __restrict__ steps, T* __restrict__ Vn, const NearStencil s) {
    extern __shared__ __align__(16) unsigned char smraw[];
    T* wbuf = reinterpret_cast<T*>(smraw) + (size_t)(threadIdx.x >> 5) * 2 * s.wrow;
    int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (w >= s.warps) return;
    // warp: (group, cx, cy, z tile, z block, j1, block of j2), the last fastest
    const int jb = w % s.njb; w /= s.njb;
    const int j1 = w % s.nd; w /= s.nd;
    const int zb = w % s.nzb; w /= s.nzb;
    const int tz = w % s.ntz; w /= s.ntz;
    const int cy = w % s.n; w /= s.n;
    const int cx = w % s.n, g = w / s.n;
    // z tiles: as many of cz cells as fit, then what is left in powers of two
    const int full = s.n / s.cz;
    int cz0 = min(tz, full) * s.cz, cz = s.cz;
    for (int q = full; q <= tz; ++q) {
        int left = s.n - cz0, p = 1;
        while (2 * p <= left) p *= 2;
        cz = p;
        if (q < tz) cz0 += p;
    }
    if (tz < full) cz = s.cz;
    if constexpr (RM > 0) {
        if (cz == 4) near_body<T, TY, TZ, 4, RM>(phi, Wt, steps, Vn, s, g, cx, cy, cz0, j1, jb * TY, zb, wbuf);
        else if (cz == 2) near_body<T, TY, TZ, 2, RM>(phi, Wt, steps, Vn, s, g, cx, cy, cz0, j1, jb * TY, zb, wbuf);
        else near_body<T, TY, TZ, 1, RM>(phi, Wt, steps, Vn, s, g, cx, cy, cz0, j1, jb * TY, zb, wbuf);
    } else {
        near_body<T, TY, TZ, 1, RM>(phi, Wt, steps, Vn, s, g, cx, cy, cz0, j1, jb * TY, zb, wbuf);
    }
}

// Weights of the near stencil, FP64, one thread per entry: index
// [z block][j1][block of j2][step][row y][source z][target z] (rows of a step padded
// to `wrow`), zero outside the ball and for padding; scale = alpha / N_div.
template <typename T>
__global__ void k_common_weights(const double* __restrict__ hcoarse, const int2* __restrict__ steps, int nsteps, int n, int nd,
                                 int nb1, int R, int R2, int TY, int TZ, int TZP, int njb, int wrow, double kappa, double scale,
                                 long long total, T* __restrict__ Wt) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int nzs = TZ + 2 * R;
    const int e = (int)(i % wrow);
    long long q = i / wrow;
    const int2 st = steps[q % nsteps]; q /= nsteps;
    const int jb = (int)(q % njb); q /= njb;
    const int j1 = (int)(q % nd);
    const int zb = (int)(q / nd);
    const int tz = e % TZP, zi = (e / TZP) % nzs, y = e / (TZP * nzs);
    const int j2 = jb * TY + y, j3 = zb * TZ + tz;
    const int d1 = (st.x & 255) - R, d2 = ((st.x >> 8) & 255) - y - R, d3 = zi - R - tz;
    T out = (T)0;
    if (y < TY && j2 < nd && tz < TZ && j3 < nd && d1 * d1 + d2 * d2 + d3 * d3 <= R2) {
        const double L = (double)n * nd, qa = d1 / L, qb = d2 / L, qc = d3 / L;
        const int js = (j1 * nd + j2) * nd + j3;
        const int g1 = j1 + d1, g2 = j2 + d2, g3 = j3 + d3;
        const int c1 = floordiv(g1, nd), c2 = floordiv(g2, nd), c3 = floordiv(g3, nd);
        const int jp = ((g1 - c1 * nd) * nd + g2 - c2 * nd) * nd + g3 - c3 * nd;
        double sum = 1.0 / (qa * qa + qb * qb + qc * qc + kappa * kappa);
        for (int l = 0; l < 8; ++l) {
            const double f = interp_weight(js, l, nd, nb1);
            if (f == 0.0) continue;
            for (int lp = 0; lp < 8; ++lp) {
                const double fp = interp_weight(jp, lp, nd, nb1);
                if (fp == 0.0) continue;
                const int h = flat3(c1 + ((lp >> 2) & 1) - ((l >> 2) & 1), c2 + ((lp >> 1) & 1) - ((l >> 1) & 1),
                                    c3 + (lp & 1) - (l & 1), n);
                sum -= f * fp * hcoarse[h];
            }
        }
        out = (T)(scale * sum);
    }
    Wt[i] = out;
}

int rot_points(const bse_interp* s, size_t vsz) {
    const size_t per = vsz * (odd(s->t) + odd(s->nv * s->nv) + odd(s->nc * s->nc));
    return (int)std::max<size_t>(1, std::min<size_t>(std::min(s->Ndiv, 64), 32768 / per));
}

template <typename K>
cudaError_t raise_smem(K kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
    if (e == cudaSuccess && (size_t)fa.maxDynamicSharedSizeBytes < bytes)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    return e;
}

// Targets of a warp within a cell: TZ = n_div up to 4 (then blocks of 4), TY rows.
inline int near_tz(int nd) { return std::min(nd, 4); }
inline int near_ty(int nd) { return nd <= 3 ? nd : 2; }
inline int near_tzp(int nd) { return nd == 3 ? 4 : near_tz(nd); }

// Elements of a step's weights, rounded up to 16 bytes.
template <typename T>
int near_wrow(int nd, int R) {
    const int per = 16 / (int)sizeof(T), e = near_ty(nd) * (near_tz(nd) + 2 * R) * near_tzp(nd);
    return (e + per - 1) / per * per;
}

template <typename T, int TY, int TZ, int RM>
int launch_near_r(bse_ctx* ctx, const bse_interp* s, NearStencil ns, cudaStream_t st) {
    const int groups = (ns.cols + 31) / 32, n = s->n;
    auto tiles = [&](int cz) {
        int c = n / cz;
        for (int left = n % cz; left; left &= left - 1) ++c;
        return c;
    };
    const long long per_tile = (long long)groups * n * n * ns.nzb * ns.nd * ns.njb;
    // Cells per warp: as many as leave four warps per SM (a warp alone on its scheduler
    // waits out its loads); z blocks do not continue into the next cell.
    ns.cz = 1;
    if (RM > 0 && ns.nzb == 1)
        for (int cz : {2, 4})
            if (n >= cz && per_tile * tiles(cz) >= 4LL * ctx->sm_count) ns.cz = cz;
    ns.ntz = tiles(ns.cz);
    const long long warps = per_tile * ns.ntz;
    if (warps > 0x7fffffffLL) { ctx->err = "near stencil: too many targets"; return BSE_ERR_UNSUPPORTED; }
    ns.warps = (int)warps;
    // small grids: fewer warps per block spread over more SMs
    const int wpb = warps >= 8LL * 2 * ctx->sm_count ? 8 : 2;
    const size_t smem = sizeof(T) * 2 * (size_t)ns.wrow * wpb;
    BSE_CUDA_TRY(ctx, raise_smem(k_common_near<T, TY, TZ, RM>, smem));
    k_common_near<T, TY, TZ, RM><<<(unsigned)((warps + wpb - 1) / wpb), 32 * wpb, smem, st>>>(
        (const T*)s->d_cphi, (const T*)s->d_cw, s->d_csteps, (T*)s->d_cV, ns);
    BSE_CUDA_TRY(ctx, cudaGetLastError());
    return BSE_OK;
}

template <typename T>
int near_typed(bse_ctx* ctx, const bse_interp* s, int nchains, cudaStream_t st) {
    NearStencil ns{};
    const int nd = s->nd;
    ns.n = s->n; ns.nd = nd; ns.L = s->n * nd; ns.R = s->cphi_R; ns.Lp = s->cphi_Lp;
    ns.nzb = (nd + near_tz(nd) - 1) / near_tz(nd);
    ns.njb = (nd + near_ty(nd) - 1) / near_ty(nd);
    ns.nsteps = s->n_csteps;
    ns.wrow = near_wrow<T>(nd, ns.R);
    ns.t2 = 2 * s->t; ns.cols = ns.t2 * nchains; ns.N2 = 2LL * s->N;
    const bool r4 = ns.R <= 4, r6 = ns.R <= 6;
    switch (nd) {
        case 1: return r4 ? launch_near_r<T, 1, 1, 4>(ctx, s, ns, st) : launch_near_r<T, 1, 1, 0>(ctx, s, ns, st);
        case 2: return r4 ? launch_near_r<T, 2, 2, 4>(ctx, s, ns, st) : launch_near_r<T, 2, 2, 0>(ctx, s, ns, st);
        case 3: return r4 ? launch_near_r<T, 3, 3, 4>(ctx, s, ns, st) : launch_near_r<T, 3, 3, 0>(ctx, s, ns, st);
        default:
            return r4   ? launch_near_r<T, 2, 4, 4>(ctx, s, ns, st)
                   : r6 ? launch_near_r<T, 2, 4, 6>(ctx, s, ns, st)
                        : launch_near_r<T, 2, 4, 0>(ctx, s, ns, st);
    }
}

template <typename T>
int restrict_typed(bse_ctx* ctx, const bse_interp* s, int nchains, const void* psi, void* Q, __nv_bfloat16* bop,
                   cudaStream_t st) {
    using V = typename Cx<T>::V;
    const bse_coarse* c = s->co;
    const int KP = rot_points(s, sizeof(V));
    const size_t smem = sizeof(V) * ((size_t)KP * (odd(s->t) + odd(s->nv * s->nv) + odd(s->nc * s->nc)) + 256) +
                        (sizeof(T) * 8 + sizeof(int2)) * KP;
    const bool m3 = s->scheme == BSE_SCHEME_M3;
    CommonPhi lay{s->cphi_R, s->cphi_Lp};
    const dim3 grid(c->nkc, nchains);
    auto go = [&](auto kernel) -> int {
        BSE_CUDA_TRY(ctx, raise_smem(kernel, smem));
        kernel<<<grid, 256, smem, st>>>((const V*)psi, (const V*)s->d_cUv, (const V*)s->d_cUc, (const V*)s->d_cUvc,
                                        (const V*)s->d_cUcc, s->n, s->nd, s->nv, s->nc, s->nb1, KP,
                                        m3 ? (T*)s->d_cphi : nullptr, lay, (V*)s->d_cshare, s->d_cctr, (V*)Q, bop, c->ldk);
        BSE_CUDA_TRY(ctx, cudaGetLastError());
        return BSE_OK;
    };
    return c->kc_prec == BSE_PREC_BF16 ? go(k_common_restrict<T, true>) : go(k_common_restrict<T, false>);
}

template <typename T>
int prolong_typed(bse_ctx* ctx, const bse_interp* s, int nchains, const void* R, const void* psi, void* W, double2* dot,
                  cudaStream_t st) {
    using V = typename Cx<T>::V;
    const int KP = rot_points(s, sizeof(V));
    const size_t smem = sizeof(V) * (size_t)(KP + 8) * (odd(s->t) + odd(s->nv * s->nv) + odd(s->nc * s->nc)) +
                        sizeof(T) * 8 * KP;
    BSE_CUDA_TRY(ctx, raise_smem(k_common_prolong<T>, smem));
    const dim3 grid(bse_common_dot_blocks(s), nchains);
    k_common_prolong<T><<<grid, 256, smem, st>>>((const V*)R, s->scheme == BSE_SCHEME_M3 ? (const V*)s->d_cV : nullptr,
                                                 (const V*)s->d_cUv, (const V*)s->d_cUc, (const V*)s->d_cUvc,
                                                 (const V*)s->d_cUcc, (const T*)s->d_dE, (const V*)psi, s->n, s->nd,
                                                 s->nv, s->nc, s->nb1, KP, (V*)W, dot);
    BSE_CUDA_TRY(ctx, cudaGetLastError());
    return BSE_OK;
}

template <typename T>
__global__ void k_gauge_to(const double2* __restrict__ src, long long n, typename Cx<T>::V* __restrict__ dst) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = from_d2<typename Cx<T>::V>(src[i]);
}

template <typename T>
int prepare_typed(bse_ctx* ctx, bse_interp* s) {
    using V = typename Cx<T>::V;
    const bse_coarse* c = s->co;
    cudaStream_t st = ctx->stream;
    const size_t rv = s->nv * s->nv, rc = s->nc * s->nc;
    struct { void** dst; const double2* src; size_t n; } tab[2] = {{&s->d_cUvc, c->d_Uv, (size_t)c->nkc * rv},
                                                                   {&s->d_cUcc, c->d_Uc, (size_t)c->nkc * rc}};
    int rc_;
    for (auto& x : tab) {
        if ((rc_ = bse_alloc(ctx, x.dst, sizeof(V) * x.n, "gauge tables")) != BSE_OK) return rc_;
        k_gauge_to<T><<<(unsigned)((x.n + 255) / 256), 256, 0, st>>>(x.src, (long long)x.n, (V*)*x.dst);
    }
    if ((rc_ = bse_alloc(ctx, &s->d_cshare, sizeof(V) * BSE_MAX_CHAINS * 8 * (size_t)c->Nc, "corner shares")) != BSE_OK) return rc_;
    if ((rc_ = bse_alloc(ctx, (void**)&s->d_cctr, sizeof(int) * BSE_MAX_CHAINS * (size_t)c->nkc, "corner counters")) != BSE_OK) return rc_;
    BSE_CUDA_TRY(ctx, cudaMemsetAsync(s->d_cctr, 0, sizeof(int) * BSE_MAX_CHAINS * (size_t)c->nkc, st));
    if (s->scheme != BSE_SCHEME_M3) {
        BSE_CUDA_TRY(ctx, cudaStreamSynchronize(st));
        return BSE_OK;
    }
    const int nd = s->nd, L = s->n * nd, R = s->cphi_R, TY = near_ty(nd), TZ = near_tz(nd), D = 2 * R + 1;
    // rows of phi: R points of halo on each side, and what a padded target block reads beyond (zeros)
    s->cphi_Lp = L + 2 * R + (nd > 4 ? 3 : 0);
    const size_t groups = (2 * (size_t)s->t * BSE_MAX_CHAINS + 31) / 32;
    const size_t nphi = groups * L * L * (size_t)s->cphi_Lp * 32;
    if ((rc_ = bse_alloc(ctx, &s->d_cphi, sizeof(T) * nphi, "common-basis vectors")) != BSE_OK) return rc_;
    BSE_CUDA_TRY(ctx, cudaMemsetAsync(s->d_cphi, 0, sizeof(T) * nphi, st));      // unused columns stay zero
    if ((rc_ = bse_alloc(ctx, &s->d_cV, sizeof(V) * BSE_MAX_CHAINS * (size_t)s->N, "near stencil result")) != BSE_OK) return rc_;
    // source rows of a warp's targets: (delta_1 + R, u), u - y the delta_2 + R of target row y,
    // with the reach along z of each row (a byte each, plus one; 0: outside the ball) and the largest
    std::vector<int2> steps;
    for (int d1 = 0; d1 < D; ++d1)
        for (int u = 0; u < D + TY - 1; ++u) {
            int reach = 0, rmax = -1;
            for (int y = 0; y < TY; ++y) {
                const int d2 = u - y, rem = s->near_R2 - (d1 - R) * (d1 - R) - (d2 - R) * (d2 - R);
                if (d2 < 0 || d2 >= D || rem < 0) continue;
                const int r = (int)std::sqrt((double)rem + 0.5);
                reach |= (r + 1) << (8 * y);
                rmax = std::max(rmax, r);
            }
            if (rmax >= 0) steps.push_back(make_int2(d1 | (u << 8) | (rmax << 16), reach));
        }
    s->n_csteps = (int)steps.size();
    if ((rc_ = bse_alloc(ctx, (void**)&s->d_csteps, sizeof(int2) * steps.size(), "near stencil rows")) != BSE_OK) return rc_;
    BSE_CUDA_TRY(ctx, cudaMemcpy(s->d_csteps, steps.data(), sizeof(int2) * steps.size(), cudaMemcpyHostToDevice));
    const int nzb = (nd + TZ - 1) / TZ, njb = (nd + TY - 1) / TY, wrow = near_wrow<T>(nd, R);
    const long long nw = (long long)nzb * nd * njb * s->n_csteps * wrow;
    if ((rc_ = bse_alloc(ctx, &s->d_cw, sizeof(T) * (size_t)nw, "near stencil weights")) != BSE_OK) return rc_;
    k_common_weights<T><<<(unsigned)((nw + 127) / 128), 128, 0, st>>>(s->d_chead, s->d_csteps, s->n_csteps, s->n, nd, s->nb1, R,
                                                                      s->near_R2, TY, TZ, near_tzp(nd), njb, wrow, c->kappa,
                                                                      c->alpha / s->Ndiv, nw, (T*)s->d_cw);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        ctx->err = std::string("near stencil weights: ") + cudaGetErrorString(e);
        return BSE_ERR_CUDA;
    }
    return BSE_OK;
}

}  // namespace

int bse_common_dot_blocks(const bse_interp* s) { return std::min(s->co->nkc, BSE_MAX_VEC_BLOCKS); }

int bse_common_prepare(bse_ctx* ctx, bse_interp* s) {
    return s->vec_prec == BSE_PREC_F64 ? prepare_typed<double>(ctx, s) : prepare_typed<float>(ctx, s);
}

int bse_common_restrict(bse_ctx* ctx, const bse_interp* s, int nchains, const void* psi, void* Q, __nv_bfloat16* bop,
                        cudaStream_t st) {
    return s->vec_prec == BSE_PREC_F64 ? restrict_typed<double>(ctx, s, nchains, psi, Q, bop, st)
                                       : restrict_typed<float>(ctx, s, nchains, psi, Q, bop, st);
}

int bse_common_near(bse_ctx* ctx, const bse_interp* s, int nchains, cudaStream_t st) {
    return s->vec_prec == BSE_PREC_F64 ? near_typed<double>(ctx, s, nchains, st) : near_typed<float>(ctx, s, nchains, st);
}

int bse_common_prolong(bse_ctx* ctx, const bse_interp* s, int nchains, const void* R, const void* psi, void* W,
                       double2* dot, cudaStream_t st) {
    return s->vec_prec == BSE_PREC_F64 ? prolong_typed<double>(ctx, s, nchains, R, psi, W, dot, st)
                                       : prolong_typed<float>(ctx, s, nchains, R, psi, W, dot, st);
}
