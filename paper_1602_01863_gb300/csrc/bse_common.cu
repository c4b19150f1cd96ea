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
    for (int i = threadIdx.x; i < np * nv; i += blockDim.x) {
        const int p = i / nv, v = i - p * nv;
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
        const int p = i / nc, c = i - p * nc;
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
    for (int i = threadIdx.x; i < rows * len; i += blockDim.x) {
        const int r = i / len;
        dst[r * pitch + (i - r * len)] = src[i];
    }
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
    // corner sums: item (l, e); with few items several threads share one over the points
    const int items = 8 * t, nsp = max(1, 256 / items);
    V acc[2] = {czero<V>(), czero<V>()};
    for (int k0 = 0; k0 < Ndiv; k0 += KP) {
        const int np = min(KP, Ndiv - k0);
        const size_t kd0 = (size_t)ic * Ndiv + k0;
        load_rows(X, tp, psi + ((size_t)ch * nkc * Ndiv + kd0) * t, np, t);
        load_rows(sUv, rvp, Uvd + kd0 * rv, np, rv);
        load_rows(sUc, rcp, Ucd + kd0 * rc, np, rc);
        for (int i = tid; i < np * 8; i += 256) wt[i] = interp_weight_as<T>(k0 + (i >> 3), i & 7, nd, nb1);
        __syncthreads();
        rotate_blocks<true>(X, tp, sUv, rvp, sUc, rcp, np, nv, nc);
        if (phi) {
            // 2 t components of a point lie side by side in the columns of its groups
            const int t2 = 2 * t, L = n * nd;
            for (int i = tid; i < np * t2; i += 256) {
                const int r = i / t2, q = i - r * t2, js = k0 + r;
                const T v = reinterpret_cast<const T*>(X + r * tp)[q];
                const Int3 j = unflat3(js, nd);
                const int x = ci.a * nd + j.a, y = ci.b * nd + j.b, z = ci.c * nd + j.c;
                const int col = ch * t2 + q;
                T* row = phi + (((size_t)(col >> 5) * L + x) * L + y) * lay.Lp * 32 + (col & 31);
                row[(size_t)(z + lay.R) * 32] = v;
                if (z >= L - lay.R) row[(size_t)(z + lay.R - L) * 32] = v;      // periodic halo copies
                if (z < lay.R) row[(size_t)(z + lay.R + L) * 32] = v;
            }
        }
        for (int a = 0; a < 2; ++a) {
            const int i = nsp > 1 ? tid % items : tid + 256 * a, sp = nsp > 1 ? tid / items : 0;
            if (i >= items || sp >= nsp || (nsp > 1 && a)) continue;
            const int l = i / t, e = i - l * t;
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
            for (int i = tid; i < np * 8; i += 256) wt[i] = interp_weight_as<T>(k0 + (i >> 3), i & 7, nd, nb1) * inv;
            __syncthreads();
            for (int i = tid; i < np * t; i += 256) {
                const int r = i / t, e = i - r * t;
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
                const int r = i / t, e = i - r * t;
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
// transitions, so the FP32 (FP64) pipes bound it, and the split serves to keep
// shared memory below them.  A block takes one column group (32 columns, one
// per lane) of 1 x CY x CZ cells.  It walks the source planes x' of their
// dilated box, double-buffered in shared memory by cp.async (every row of a
// plane is contiguous in phi, z halo included).  A warp owns the sub-cell
// rows (j1, TY values of j2, TZ values of j3) of all the block's cells: their
// weights are the same in every cell, so one broadcast vector load of TZ
// weights serves CY CZ multiply-adds per weight, and one load of a source
// column TY TZ of them.  A warp stages its weight rows itself (one row per
// source row, loaded a row ahead into registers).
struct NearStencil {
    int n, nd, L, Lp, R, R2, nzb, tasks, ntz;   // ntz: z blocks a cell has; tasks: warps per (cell, z block)
    int cols, t2;                               // 2 t nchains columns in use; 2 t
    long long N2;                               // 2 N: reals per chain of V
};

template <typename T, int TY, int TZ, int CY, int CZ, bool STAGED>
__device__ __forceinline__ void near_body(const T* __restrict__ phi, const T* __restrict__ Wt, T* __restrict__ Vn,
                                          const NearStencil& s, int cx, int cy0, int cz0, int g, int task, bool active,
                                          T* planes, T* wbuf) {
    constexpr int TZP = TZ == 3 ? 4 : TZ;
    constexpr int I = CY * CZ;
    const int lane = threadIdx.x & 31, nthr = blockDim.x;
    const int nd = s.nd, R = s.R, D = 2 * R + 1;
    const int NY = CY * nd + 2 * R, NZ = CZ * nd + 2 * R, plane = NY * NZ * 32;
    const int nzs = TZ + 2 * R;
    // task -> (z block, j1, rows j2 .. j2 + TY - 1)
    const int nty = (nd + TY - 1) / TY;
    const int zb = task / (nd * nty), j1 = (task / nty) % nd, j2 = (task % nty) * TY;
    const int tzn = min(TZ, nd - zb * TZ);                        // targets of this z block
    T acc[I][TY][TZ];
#pragma unroll
    for (int i = 0; i < I; ++i)
#pragma unroll
        for (int y = 0; y < TY; ++y)
#pragma unroll
            for (int z = 0; z < TZ; ++z) acc[i][y][z] = (T)0;
    auto fetch = [&](int px, T* dst) {
        constexpr int PER = 16 / sizeof(T), CH = 32 / PER;        // 16-byte chunks of a point's columns
        const int x = imod(cx * nd - R + px, s.L);
        const int rowc = NZ * CH, tot = NY * rowc;
        for (int c = threadIdx.x; c < tot; c += nthr) {
            const int r = c / rowc, q = c - r * rowc;
            const int y = imod(cy0 * nd - R + r, s.L);
            cpa16(dst + (size_t)r * NZ * 32 + q * PER,
                  phi + ((((size_t)g * s.L + x) * s.L + y) * s.Lp + cz0 * nd) * 32 + q * PER);
        }
    };
    const int npx = nd + 2 * R;
    if (STAGED) {
        fetch(0, planes);
        cpa_commit();
    }
    for (int px = 0; px < npx; ++px) {
        if (STAGED) {
            if (px + 1 < npx) fetch(px + 1, planes + ((px + 1) & 1) * plane);
            cpa_commit();
            cpa_wait<1>();
            __syncthreads();
        }
        const T* src = STAGED ? planes + (px & 1) * plane
                              : phi + ((size_t)g * s.L + imod(cx * nd - R + px, s.L)) * s.L * s.Lp * 32;
        const int d1 = px - j1;                                   // delta_1 + R
        if (active && d1 >= 0 && d1 < D) {
            const int rem1 = s.R2 - (d1 - R) * (d1 - R);
            // rows of sources: u = 0 .. 2R + TY - 1, delta_2 of target row y is u - y - R
            const T* wrow = Wt + ((((size_t)(zb * nd + j1) * nd + j2) * D + d1) * D) * nzs * TZP;
            const size_t wty = (size_t)D * D * nzs * TZP;         // next j2
            for (int u = 0; u < D + TY - 1; ++u) {
                int rmax = -1;
#pragma unroll
                for (int y = 0; y < TY; ++y) {
                    const int d2 = u - y, rem = rem1 - (d2 - R) * (d2 - R);
                    if (d2 >= 0 && d2 < D && rem >= 0 && j2 + y < nd) {
                        const int r = (int)sqrtf((float)rem + 0.5f);
                        rmax = max(rmax, r);
                    }
                }
                if (rmax < 0) continue;
                const int z0 = R - rmax, z1 = R + rmax + tzn;     // sources z0 .. z1 - 1 of the z block
                __syncwarp();
#pragma unroll
                for (int y = 0; y < TY; ++y) {
                    const int d2 = u - y;
                    const bool in = d2 >= 0 && d2 < D && j2 + y < nd;
                    const T* w = wrow + y * wty + (size_t)d2 * nzs * TZP;
                    for (int q = lane + z0 * TZP; q < z1 * TZP; q += 32) wbuf[y * nzs * TZP + q] = in ? w[q] : (T)0;
                }
                __syncwarp();
                const T* row[CY];
#pragma unroll
                for (int cy = 0; cy < CY; ++cy) {
                    const int r = cy * nd + j2 + u;
                    row[cy] = STAGED ? src + ((size_t)r * NZ + zb * TZ) * 32 + lane
                                     : src + ((size_t)imod(cy0 * nd - R + r, s.L) * s.Lp + cz0 * nd + zb * TZ) * 32 + lane;
                }
#pragma unroll 2
                for (int zi = z0; zi < z1; ++zi) {
                    T v[I];
#pragma unroll
                    for (int cy = 0; cy < CY; ++cy)
#pragma unroll
                        for (int cz = 0; cz < CZ; ++cz) v[cy * CZ + cz] = row[cy][(cz * nd + zi) * 32];
#pragma unroll
                    for (int y = 0; y < TY; ++y) {
                        T w[TZ];
                        const T* wp = wbuf + (y * nzs + zi) * TZP;
                        if constexpr (TZP == 4 && sizeof(T) == 4) {
                            const float4 w4 = *reinterpret_cast<const float4*>(wp);
                            w[0] = w4.x; w[1] = w4.y; w[2] = w4.z;
                            if (TZ == 4) w[TZ - 1] = w4.w;
                        } else {
#pragma unroll
                            for (int z = 0; z < TZ; ++z) w[z] = wp[z];
                        }
#pragma unroll
                        for (int z = 0; z < TZ; ++z) {
                            // FP64 runs at a small fraction of the issue rate: skip what lies outside the ball
                            if (sizeof(T) == 8 && w[z] == (T)0) continue;
#pragma unroll
                            for (int i = 0; i < I; ++i) acc[i][y][z] = fma(w[z], v[i], acc[i][y][z]);
                        }
                    }
                }
            }
        }
        if (STAGED) __syncthreads();
    }
    const int col = g * 32 + lane;
    if (!active || col >= s.cols) return;
    const int ch = col / s.t2, q = col - ch * s.t2;
#pragma unroll
    for (int cy = 0; cy < CY; ++cy)
#pragma unroll
        for (int cz = 0; cz < CZ; ++cz) {
            const int cell = (cx * s.n + cy0 + cy) * s.n + cz0 + cz;
#pragma unroll
            for (int y = 0; y < TY; ++y)
#pragma unroll
                for (int z = 0; z < TZ; ++z)
                    if (j2 + y < nd && z < tzn) {
                        const size_t kd = (size_t)cell * nd * nd * nd + (j1 * nd + j2 + y) * nd + zb * TZ + z;
                        Vn[(size_t)ch * s.N2 + kd * s.t2 + q] = acc[cy * CZ + cz][y][z];
                    }
        }
}

// Grid (tiles of cells, column groups, task groups).  Not STAGED: boxes too wide
// for two source planes in shared memory read phi directly, cell by cell.
template <typename T, int TY, int TZ, int CY, int CZ, bool STAGED>
__global__ void __launch_bounds__(256) k_common_near(const T* __restrict__ phi, const T* __restrict__ Wt,
                                                     T* __restrict__ Vn, const NearStencil s) {
    extern __shared__ __align__(16) unsigned char smraw[];
    constexpr int TZP = TZ == 3 ? 4 : TZ;
    const int warp = threadIdx.x >> 5;
    const int NY = CY * s.nd + 2 * s.R, NZ = CZ * s.nd + 2 * s.R;
    T* planes = reinterpret_cast<T*>(smraw);
    T* wbuf = planes + (STAGED ? 2 * (size_t)NY * NZ * 32 : 0) + (size_t)warp * TY * (TZ + 2 * s.R) * TZP;
    const int nty = (s.n + CY - 1) / CY, ntz = (s.n + CZ - 1) / CZ;
    const int cx = blockIdx.x / (nty * ntz), ty = (blockIdx.x / ntz) % nty, tz = blockIdx.x % ntz;
    const int cy0 = ty * CY, cz0 = tz * CZ, g = blockIdx.y;
    const int task = blockIdx.z * (blockDim.x >> 5) + warp;
    const bool act = task < s.tasks;
    const int tk = act ? task : 0;
    // tiles cut by the mesh's end run the smaller body
    const int ny = min(CY, s.n - cy0), nz = min(CZ, s.n - cz0);
    if (ny == CY && nz == CZ) near_body<T, TY, TZ, CY, CZ, STAGED>(phi, Wt, Vn, s, cx, cy0, cz0, g, tk, act, planes, wbuf);
    else if (CY == 2 && nz == CZ) near_body<T, TY, TZ, 1, CZ, STAGED>(phi, Wt, Vn, s, cx, cy0, cz0, g, tk, act, planes, wbuf);
    else if (CZ == 2 && ny == CY) near_body<T, TY, TZ, CY, 1, STAGED>(phi, Wt, Vn, s, cx, cy0, cz0, g, tk, act, planes, wbuf);
    else near_body<T, TY, TZ, 1, 1, STAGED>(phi, Wt, Vn, s, cx, cy0, cz0, g, tk, act, planes, wbuf);
}

// Weights of the near stencil, FP64, one thread per entry: index
// [z block][j1][j2][d1][d2][source z][target z], zero outside the ball (and for
// the padding targets); scale = alpha / N_div.
template <typename T>
__global__ void k_common_weights(const double* __restrict__ hcoarse, int n, int nd, int nb1, int R, int R2, int TZ, int TZP,
                                 double kappa, double scale, long long total, T* __restrict__ Wt) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int D = 2 * R + 1, nzs = TZ + 2 * R;
    long long q = i;
    const int tz = (int)(q % TZP); q /= TZP;
    const int zi = (int)(q % nzs); q /= nzs;
    const int d2 = (int)(q % D) - R; q /= D;
    const int d1 = (int)(q % D) - R; q /= D;
    const int j2 = (int)(q % nd); q /= nd;
    const int j1 = (int)(q % nd);
    const int zb = (int)(q / nd), j3 = zb * TZ + tz, d3 = zi - R - tz;
    T out = (T)0;
    if (tz < TZ && j3 < nd && d1 * d1 + d2 * d2 + d3 * d3 <= R2) {
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

// Sub-cell targets a thread owns: TZ = n_div up to 4 (then blocks of 4), TY rows.
inline int near_tz(int nd) { return std::min(nd, 4); }
inline int near_ty(int nd) { return nd <= 3 ? nd : 2; }
inline int near_tzp(int nd) { return nd == 3 ? 4 : near_tz(nd); }

template <typename T, int TY, int TZ>
size_t near_smem(const NearStencil& ns, int cy, int cz, int warps, bool staged) {
    const size_t NY = cy * ns.nd + 2 * ns.R, NZ = cz * ns.nd + 2 * ns.R;
    return sizeof(T) * ((staged ? 2 * NY * NZ * 32 : 0) + (size_t)warps * TY * (TZ + 2 * ns.R) * (TZ == 3 ? 4 : TZ));
}

template <typename T, int TY, int TZ, int CY, int CZ, bool STAGED>
int launch_near_c(bse_ctx* ctx, const bse_interp* s, const NearStencil& ns, const T* phi, T* Vn, cudaStream_t st) {
    const int groups = (ns.cols + 31) / 32, n = s->n, warps = std::min(ns.tasks, 8);
    const size_t smem = near_smem<T, TY, TZ>(ns, CY, CZ, warps, STAGED);
    BSE_CUDA_TRY(ctx, raise_smem(k_common_near<T, TY, TZ, CY, CZ, STAGED>, smem));
    dim3 grid(n * ((n + CY - 1) / CY) * ((n + CZ - 1) / CZ), groups, (ns.tasks + warps - 1) / warps);
    k_common_near<T, TY, TZ, CY, CZ, STAGED><<<grid, 32 * warps, smem, st>>>(phi, (const T*)s->d_cw, Vn, ns);
    BSE_CUDA_TRY(ctx, cudaGetLastError());
    return BSE_OK;
}

template <typename T, int TY, int TZ>
int launch_near_t(bse_ctx* ctx, const bse_interp* s, const NearStencil& ns, const T* phi, T* Vn, cudaStream_t st) {
    // Cells per block: as many as leave a block per SM, and whose two source planes fit
    const int groups = (ns.cols + 31) / 32, n = s->n, warps = std::min(ns.tasks, 8), zg = (ns.tasks + warps - 1) / warps;
    auto good = [&](int cy, int cz) {
        return n >= 2 && near_smem<T, TY, TZ>(ns, cy, cz, warps, true) <= (size_t)100 * 1024 &&
               (long long)n * ((n + cy - 1) / cy) * ((n + cz - 1) / cz) * groups * zg >= ctx->sm_count;
    };
    if (good(2, 2)) return launch_near_c<T, TY, TZ, 2, 2, true>(ctx, s, ns, phi, Vn, st);
    if (good(1, 2)) return launch_near_c<T, TY, TZ, 1, 2, true>(ctx, s, ns, phi, Vn, st);
    if (near_smem<T, TY, TZ>(ns, 1, 1, warps, true) <= (size_t)200 * 1024)
        return launch_near_c<T, TY, TZ, 1, 1, true>(ctx, s, ns, phi, Vn, st);
    return launch_near_c<T, TY, TZ, 1, 1, false>(ctx, s, ns, phi, Vn, st);
}

template <typename T>
int near_typed(bse_ctx* ctx, const bse_interp* s, int nchains, cudaStream_t st) {
    NearStencil ns{};
    ns.n = s->n; ns.nd = s->nd; ns.L = s->n * s->nd; ns.R = s->cphi_R; ns.R2 = s->near_R2; ns.Lp = ns.L + 2 * ns.R;
    ns.nzb = (s->nd + near_tz(s->nd) - 1) / near_tz(s->nd);
    ns.tasks = ns.nzb * s->nd * ((s->nd + near_ty(s->nd) - 1) / near_ty(s->nd));
    ns.t2 = 2 * s->t; ns.cols = ns.t2 * nchains; ns.N2 = 2LL * s->N;
    const T* phi = (const T*)s->d_cphi;
    T* Vn = (T*)s->d_cV;
    switch (s->nd) {
        case 1: return launch_near_t<T, 1, 1>(ctx, s, ns, phi, Vn, st);
        case 2: return launch_near_t<T, 2, 2>(ctx, s, ns, phi, Vn, st);
        case 3: return launch_near_t<T, 3, 3>(ctx, s, ns, phi, Vn, st);
        default: return launch_near_t<T, 2, 4>(ctx, s, ns, phi, Vn, st);
    }
}

template <typename T>
int restrict_typed(bse_ctx* ctx, const bse_interp* s, int nchains, const void* psi, void* Q, __nv_bfloat16* bop,
                   cudaStream_t st) {
    using V = typename Cx<T>::V;
    const bse_coarse* c = s->co;
    const int KP = rot_points(s, sizeof(V));
    const size_t smem = sizeof(V) * ((size_t)KP * (odd(s->t) + odd(s->nv * s->nv) + odd(s->nc * s->nc)) + 256) +
                        sizeof(T) * 8 * KP;
    const bool m3 = s->scheme == BSE_SCHEME_M3;
    CommonPhi lay{s->cphi_R, s->n * s->nd + 2 * s->cphi_R};
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
int prepare_typed(bse_ctx* ctx, bse_interp* s, const double2* Uvd, const double2* Ucd) {
    using V = typename Cx<T>::V;
    const bse_coarse* c = s->co;
    cudaStream_t st = ctx->stream;
    const size_t rv = s->nv * s->nv, rc = s->nc * s->nc;
    struct { void** dst; const double2* src; size_t n; } tab[4] = {{&s->d_cUv, Uvd, (size_t)s->nk * rv},
                                                                   {&s->d_cUc, Ucd, (size_t)s->nk * rc},
                                                                   {&s->d_cUvc, c->d_Uv, (size_t)c->nkc * rv},
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
    const int L = s->n * s->nd, R = s->cphi_R, TZ = near_tz(s->nd), TZP = near_tzp(s->nd), D = 2 * R + 1;
    const size_t groups = (2 * (size_t)s->t * BSE_MAX_CHAINS + 31) / 32;
    const size_t nphi = groups * L * L * (size_t)(L + 2 * R) * 32;
    if ((rc_ = bse_alloc(ctx, &s->d_cphi, sizeof(T) * nphi, "common-basis vectors")) != BSE_OK) return rc_;
    BSE_CUDA_TRY(ctx, cudaMemsetAsync(s->d_cphi, 0, sizeof(T) * nphi, st));      // unused columns stay zero
    if ((rc_ = bse_alloc(ctx, &s->d_cV, sizeof(V) * BSE_MAX_CHAINS * (size_t)s->N, "near stencil result")) != BSE_OK) return rc_;
    const long long nw = (long long)((s->nd + TZ - 1) / TZ) * s->nd * s->nd * D * D * (TZ + 2 * R) * TZP;
    if ((rc_ = bse_alloc(ctx, &s->d_cw, sizeof(T) * (size_t)nw, "near stencil weights")) != BSE_OK) return rc_;
    k_common_weights<T><<<(unsigned)((nw + 127) / 128), 128, 0, st>>>(s->d_chead, s->n, s->nd, s->nb1, R, s->near_R2, TZ, TZP,
                                                                      c->kappa, c->alpha / s->Ndiv, nw, (T*)s->d_cw);
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

int bse_common_prepare(bse_ctx* ctx, bse_interp* s, const double2* Uvd, const double2* Ucd) {
    return s->vec_prec == BSE_PREC_F64 ? prepare_typed<double>(ctx, s, Uvd, Ucd) : prepare_typed<float>(ctx, s, Uvd, Ucd);
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
