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
// n_div 4, 4x4 bands, 3 vectors FP64 98.5 -> 3.31 ms; coarse 4^3, n_div 2, 3x3
// bands, 1 vector FP64 1105 -> 60 us; coarse 7^3, n_div 3, 3x5 bands, 4 vectors
// FP32 1.80 -> 0.19 ms.
// Caller-supplied overlaps (not a product through one basis) and non-Hermitian
// generators keep the general kernels of bse_apply.cu and bse_near_tc.cu.
#include <algorithm>
#include <cmath>
#include <type_traits>

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

// Rotation by one warp of `np` blocks x [np][tp] (t = nv nc entries each) in shared
// memory by Uv [np][rvp], Uc [np][rcp]; ends with __syncwarp.  FP32: a lane per row,
// then per column, in place: 1 shared load per complex multiply-add, rows padded
// to an odd number of entries so that they spread over the banks.  FP64 with few
// rows, where the chain of multiply-adds of a lane counts, not the loads: a lane per
// entry, through tmp [np][tp].
template <bool TO, typename V>
__device__ __forceinline__ void rotate_warp(V* x, V* tmp, int tp, const V* Uv, int rvp, const V* Uc, int rcp, int np, int nv,
                                            int nc) {
    const int lane = threadIdx.x & 31;
    const float inv_v = 1.f / (float)nv, inv_c = 1.f / (float)nc;
    if (sizeof(V) == 16 && np * nv <= 16) {
        const int t = nv * nc;
        const float inv_t = 1.f / (float)t;
        for (int i = lane; i < np * t; i += 32) {
            const int p = quot(i, inv_t), e = i - p * t, r = quot(e, inv_c), j = e - r * nc;
            const V *in = x + p * tp + r * nc, *U = Uc + p * rcp + (TO ? j * nc : j);
            V a = czero<V>();
            for (int q = 0; q < nc; ++q) {
                if (TO) cfma(a, in[q], U[q]);
                else cfmac(a, in[q], U[q * nc]);
            }
            tmp[p * tp + e] = a;
        }
        __syncwarp();
        for (int i = lane; i < np * t; i += 32) {
            const int p = quot(i, inv_t), e = i - p * t, r = quot(e, inv_c), j = e - r * nc;
            const V *in = tmp + p * tp + j, *U = Uv + p * rvp + (TO ? r * nv : r);
            V a = czero<V>();
            for (int q = 0; q < nv; ++q) {
                if (TO) cfmac(a, in[q * nc], U[q]);
                else cfma(a, in[q * nc], U[q * nv]);
            }
            x[p * tp + e] = a;
        }
    } else {
        for (int i = lane; i < np * nv; i += 32) {
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
        __syncwarp();
        for (int i = lane; i < np * nc; i += 32) {
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
    }
    __syncwarp();
}

// Rows of `len` entries from global src (row r at src + r * len) into shared dst (row pitch `pitch`), by one warp.
template <typename V>
__device__ __forceinline__ void load_rows(V* dst, int pitch, const V* __restrict__ src, int rows, int len) {
    const float inv = 1.f / (float)len;
#pragma unroll 4
    for (int i = threadIdx.x & 31; i < rows * len; i += 32) {
        const int r = quot(i, inv);
        dst[r * pitch + (i - r * len)] = src[i];
    }
}

// A lane's share of rows of t entries: entry e (and, for t > 32, e + 32) of rows sub,
// sub + nsub, ...: no division inside the loops, whole lines of rows side by side.
struct LaneMap {
    int e, sub, nsub;          // lanes left over take no row (sub beyond every row count)
    __device__ explicit LaneMap(int t) {
        const int lane = threadIdx.x & 31;
        nsub = t <= 32 ? 32 / t : 1;
        sub = t <= 32 ? lane / t : 0;
        e = lane - sub * t;
        if (sub >= nsub) sub = 1 << 20;
    }
};

// Shared memory of a warp that rotates up to KP points: entries, gauge, weights, places.
template <typename T>
struct WarpStage {
    using V = typename Cx<T>::V;
    V *X, *Tm, *Uv, *Uc;
    T* wt;         // [KP][8]
    int2* pnt;     // [KP]
    static __host__ __device__ size_t bytes(int KP, int nv, int nc) {
        const size_t v = (size_t)(sizeof(T) == 8 ? 2 : 1) * odd(nv * nc) + odd(nv * nv) + odd(nc * nc);
        return (KP * (v * sizeof(V) + 8 * sizeof(T) + sizeof(int2)) + 15) / 16 * 16;
    }
    __device__ WarpStage(unsigned char* p, int KP, int nv, int nc) {
        X = reinterpret_cast<V*>(p);
        Tm = X + KP * odd(nv * nc);
        Uv = sizeof(T) == 8 ? Tm + KP * odd(nv * nc) : Tm;
        Uc = Uv + KP * odd(nv * nv);
        wt = reinterpret_cast<T*>(Uc + KP * odd(nc * nc));
        pnt = reinterpret_cast<int2*>(wt + KP * 8);
    }
};

// Weight of corner l at sub-cell position (j1, j2, j3) (interp_weight).
template <typename T>
__device__ __forceinline__ T corner_weight(int j1, int j2, int j3, int l, int nd, int nb1) {
    const int l1 = (l >> 2) & 1, l2 = (l >> 1) & 1, l3 = l & 1;
    if (nb1) return ((2 * j1 > nd) == l1 && (2 * j2 > nd) == l2 && (2 * j3 > nd) == l3) ? (T)1 : (T)0;
    return (T)((l1 ? j1 : nd - j1) * (l2 ? j2 : nd - j2) * (l3 ? j3 : nd - j3)) / (T)(nd * nd * nd);
}

// ------------------------------------------------------- rotate and restrict
// Grid (coarse cell, group of CPB chains), 8 warps.  A warp takes KP points of the
// cell at a time: the gauge matrices and weights into its own shared memory and,
// chain by chain, psi, the rotation, phi for the near stencil (layout of
// CommonPhi), and the points' weighted sums for the cell's eight corners in
// registers (lane = transition, EPL of them); the warps' sums add up to the cell's
// share of each corner.  The block whose share of a coarse point is the last of
// eight (a counter per point, reset there) adds the eight in corner order, rotates
// the sum back and writes Q, a warp per point: the order does not depend on the
// blocks' order.  Memory latency and instruction issue bound it (it reads psi and U
// and writes phi: 33 MB for coarse 8^3, n_div 4, 4x4 bands, 3 chains), so the warps of a
// block wait for one another only at the sums and the chains share what they can.
// Four FP32 blocks per SM (64 registers) hold 512 cells at once: 28 us, with three 31 us.
template <typename T, bool OUT_BF16, int EPL>
__global__ void __launch_bounds__(256, EPL == 2 ? 1 : (sizeof(T) == 4 ? 4 : 2)) k_common_restrict(
    const typename Cx<T>::V* __restrict__ psi, const typename Cx<T>::V* __restrict__ Uvd,
    const typename Cx<T>::V* __restrict__ Ucd, const typename Cx<T>::V* __restrict__ Uvc,
    const typename Cx<T>::V* __restrict__ Ucc, int n, int nd, int nv, int nc, int nb1, int nch, int CPB, int KP,
    T* __restrict__ phi, CommonPhi lay, typename Cx<T>::V* __restrict__ share, int* __restrict__ ctr,
    typename Cx<T>::V* __restrict__ Q, __nv_bfloat16* __restrict__ Bop, int ldk) {
    using V = typename Cx<T>::V;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int last_sh[8];
    const int t = nv * nc, tp = odd(t), rv = nv * nv, rc = nc * nc, rvp = odd(rv), rcp = odd(rc);
    const int Ndiv = nd * nd * nd, nkc = n * n * n;
    const int ic = blockIdx.x, c0 = blockIdx.y * CPB, c1 = min(nch, c0 + CPB), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Int3 ci = unflat3(ic, n);
    const size_t wbytes = WarpStage<T>::bytes(KP, nv, nc);
    const WarpStage<T> w(smraw + warp * wbytes, KP, nv, nc);
    V* red = reinterpret_cast<V*>(smraw + 8 * wbytes);            // [8 warps][nsub][8][t]
    const int L = n * nd;
    const float inv_nd = 1.f / (float)nd;
    const LaneMap m(t);
    const int items = 8 * t, parts = 8 * m.nsub;
    const bool once = Ndiv <= 8 * KP;                              // a warp's points fit at once: their gauge is loaded once
    for (int ch = c0; ch < c1; ++ch) {
        V acc[EPL][8];
#pragma unroll
        for (int a = 0; a < EPL; ++a) {
#pragma unroll
            for (int l = 0; l < 8; ++l) acc[a][l] = czero<V>();
        }
        for (int k0 = warp * KP; k0 < Ndiv; k0 += 8 * KP) {
            const int np = min(KP, Ndiv - k0);
            const size_t kd0 = (size_t)ic * Ndiv + k0;
            const V* src = psi + ((size_t)ch * nkc * Ndiv + kd0) * t;
#pragma unroll 4
            for (int r = m.sub; r < np; r += m.nsub) {
#pragma unroll
                for (int a = 0; a < EPL; ++a) {
                    const int e = m.e + 32 * a;
                    if (EPL == 1 || e < t) w.X[r * tp + e] = src[r * t + e];
                }
            }
            if (ch == c0 || !once) {
                load_rows(w.Uv, rvp, Uvd + kd0 * rv, np, rv);
                load_rows(w.Uc, rcp, Ucd + kd0 * rc, np, rc);
                for (int i = lane; i < np * 8; i += 32) {
                    const int js = k0 + (i >> 3), a = quot(js, inv_nd), j3 = js - a * nd, j1 = quot(a, inv_nd), j2 = a - j1 * nd;
                    w.wt[i] = corner_weight<T>(j1, j2, j3, i & 7, nd, nb1);
                    if ((i & 7) == 0) {
                        const int x = ci.a * nd + j1, y = ci.b * nd + j2, z = ci.c * nd + j3;
                        w.pnt[i >> 3] = make_int2((x * L + y) * lay.Lp + z + lay.R, z < lay.R ? L : (z >= L - lay.R ? -L : 0));
                    }
                }
            }
            __syncwarp();
            rotate_warp<true>(w.X, w.Tm, tp, w.Uv, rvp, w.Uc, rcp, np, nv, nc);
            if (phi) {
                // the 2 t components of a point lie side by side in the columns of its groups
                const size_t gs = (size_t)L * L * lay.Lp * 32;
#pragma unroll
                for (int a = 0; a < EPL; ++a) {
                    const int e = m.e + 32 * a, col = 2 * (ch * t + e);
                    if (EPL == 2 && e >= t) continue;
                    T* at0 = phi + (size_t)(col >> 5) * gs + (col & 31);
                    for (int r = m.sub; r < np; r += m.nsub) {
                        const int2 pt = w.pnt[r];
                        const V v = w.X[r * tp + e];
                        V* at = reinterpret_cast<V*>(at0 + (size_t)pt.x * 32);
                        *at = v;
                        if (pt.y) at[(ptrdiff_t)pt.y * 16] = v;  // periodic halo copy
                    }
                }
            }
            for (int r = m.sub; r < np; r += m.nsub) {
                T f[8];
#pragma unroll
                for (int l = 0; l < 8; ++l) f[l] = w.wt[r * 8 + l];
#pragma unroll
                for (int a = 0; a < EPL; ++a) {
                    const int e = m.e + 32 * a;
                    if (EPL == 2 && e >= t) continue;
                    const V v = w.X[r * tp + e];
#pragma unroll
                    for (int l = 0; l < 8; ++l) {
                        if (sizeof(T) == 8 && f[l] == (T)0) continue;
                        acc[a][l].x = fma(f[l], v.x, acc[a][l].x);
                        acc[a][l].y = fma(f[l], v.y, acc[a][l].y);
                    }
                }
            }
            __syncwarp();
        }
        // the cell's shares: [chain][cell][corner][t], the warps' sums in order
        if (m.sub < m.nsub) {
#pragma unroll
            for (int a = 0; a < EPL; ++a) {
                const int e = m.e + 32 * a;
                if (EPL == 2 && e >= t) continue;
#pragma unroll
                for (int l = 0; l < 8; ++l) red[(warp * m.nsub + m.sub) * items + l * t + e] = acc[a][l];
            }
        }
        __syncthreads();
        V* mine = share + ((size_t)ch * nkc + ic) * items;
        for (int i = tid; i < items; i += 256) {
            V s = red[i];
            for (int q = 1; q < parts; ++q) s = cadd(s, red[q * items + i]);
            mine[i] = s;
        }
        if (ch + 1 < c1) __syncthreads();
    }
    __threadfence();
    __syncthreads();
    if (tid < 8) {
        const int dst = flat3(ci.a + ((tid >> 2) & 1), ci.b + ((tid >> 1) & 1), ci.c + (tid & 1), n);
        int* c = ctr + (size_t)blockIdx.y * nkc + dst;
        const bool last = atomicAdd(c, 1) == 7;
        if (last) *c = 0;
        last_sh[tid] = last ? dst : -1;
        __threadfence();
    }
    __syncthreads();
    const int dst = last_sh[warp];
    if (dst < 0) return;
    const Int3 d = unflat3(dst, n);
    load_rows(w.Uv, rvp, Uvc + (size_t)dst * rv, 1, rv);
    load_rows(w.Uc, rcp, Ucc + (size_t)dst * rc, 1, rc);
    // lane q < 8 finds the cell whose corner q this point is
    const int cq = flat3(d.a - ((lane >> 2) & 1), d.b - ((lane >> 1) & 1), d.c - (lane & 1), n);
    int cell[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) cell[q] = __shfl_sync(0xffffffffu, cq, q);
    for (int ch = c0; ch < c1; ++ch) {
        for (int e = lane; e < t; e += 32) {
            V p[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) p[q] = __ldcg(share + ((size_t)ch * nkc + cell[q]) * items + q * t + e);
            V s = p[0];
#pragma unroll
            for (int q = 1; q < 8; ++q) s = cadd(s, p[q]);
            w.X[e] = s;
        }
        __syncwarp();
        rotate_warp<false>(w.X, w.Tm, tp, w.Uv, rvp, w.Uc, rcp, 1, nv, nc);
        for (int e = lane; e < t; e += 32) {
            const V s = w.X[e];
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
        __syncwarp();
    }
}

// ------------------------------------------------------- prolong and diagonal
// Grid (coarse cell, grid-strided; group of CPB chains), 8 warps:
// w = dE psi + from_common[(1/N_div) sum_l f R'(k~_l) + V], R' = to_common(R) at the
// cell's eight corners (a warp each, the chains as blocks of one gauge), V the near
// stencil (its weights carry alpha / N_div); then a warp takes KP points at a time
// by itself, chain by chain, as in k_common_restrict.  FP64 block partials of <psi, w>.
template <typename T, int EPL>
__global__ void __launch_bounds__(256, EPL == 2 ? 1 : (sizeof(T) == 4 ? 3 : 2)) k_common_prolong(
    const typename Cx<T>::V* __restrict__ R, const typename Cx<T>::V* __restrict__ Vn,
    const typename Cx<T>::V* __restrict__ Uvd, const typename Cx<T>::V* __restrict__ Ucd,
    const typename Cx<T>::V* __restrict__ Uvc, const typename Cx<T>::V* __restrict__ Ucc, const T* __restrict__ dE,
    const typename Cx<T>::V* __restrict__ psi, int n, int nd, int nv, int nc, int nb1, int nch, int CPB, int KP,
    typename Cx<T>::V* __restrict__ W, double2* __restrict__ part) {
    using V = typename Cx<T>::V;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ DotSum<T> dsum[BSE_MAX_CHAINS][256];               // <psi, w> per chain and thread
    const int t = nv * nc, tp = odd(t), rv = nv * nv, rc = nc * nc, rvp = odd(rv), rcp = odd(rc);
    const int Ndiv = nd * nd * nd, nkc = n * n * n, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int c0 = blockIdx.y * CPB, c1 = min(nch, c0 + CPB), ncb = c1 - c0;
    V* Rc = reinterpret_cast<V*>(smraw);                          // [8][CPB][tp], then [8][CPB][tp] scratch (FP64)
    const size_t rbytes = (sizeof(V) * (sizeof(T) == 8 ? 2 : 1) * 8 * CPB * tp + 15) / 16 * 16;
    const WarpStage<T> w(smraw + rbytes + warp * WarpStage<T>::bytes(KP, nv, nc), KP, nv, nc);
    const T inv = (T)1 / (T)Ndiv;
    const float inv_nd = 1.f / (float)nd;
    const LaneMap m(t);
    const bool once = Ndiv <= 8 * KP;
    double2 dot = make_double2(0.0, 0.0);                         // warp c < ncb: chain c's sum over the block, in FP64
    for (int cell = blockIdx.x; cell < nkc; cell += gridDim.x) {
        const Int3 ci = unflat3(cell, n);
        if (cell != (int)blockIdx.x) __syncthreads();              // the previous cell's corners are no longer read
        {
            const size_t cc = flat3(ci.a + ((warp >> 2) & 1), ci.b + ((warp >> 1) & 1), ci.c + (warp & 1), n);
            V* mine = Rc + (size_t)warp * CPB * tp;
            for (int c = 0; c < ncb; ++c) load_rows(mine + c * tp, tp, R + ((size_t)(c0 + c) * nkc + cc) * t, 1, t);
            load_rows(w.Uv, rvp, Uvc + cc * rv, 1, rv);
            load_rows(w.Uc, rcp, Ucc + cc * rc, 1, rc);
            __syncwarp();
            rotate_warp<true>(mine, mine + 8 * CPB * tp, tp, w.Uv, 0, w.Uc, 0, ncb, nv, nc);
        }
        __syncthreads();
        for (int c = 0; c < ncb; ++c) {
            const int ch = c0 + c;
            DotSum<T> dsm = DotSum<T>::zero();
            V rr[EPL][8];
#pragma unroll
            for (int a = 0; a < EPL; ++a) {
#pragma unroll
                for (int l = 0; l < 8; ++l) rr[a][l] = m.e + 32 * a < t ? Rc[(l * CPB + c) * tp + m.e + 32 * a] : czero<V>();
            }
            for (int k0 = warp * KP; k0 < Ndiv; k0 += 8 * KP) {
                const int np = min(KP, Ndiv - k0);
                const size_t kd0 = (size_t)cell * Ndiv + k0, g0 = kd0 * t, o0 = (size_t)ch * nkc * Ndiv * t + g0;
                if (c == 0 || !once) {
                    load_rows(w.Uv, rvp, Uvd + kd0 * rv, np, rv);
                    load_rows(w.Uc, rcp, Ucd + kd0 * rc, np, rc);
                    for (int i = lane; i < np * 8; i += 32) {
                        const int js = k0 + (i >> 3), a = quot(js, inv_nd), j1 = quot(a, inv_nd);
                        w.wt[i] = corner_weight<T>(j1, a - j1 * nd, js - a * nd, i & 7, nd, nb1) * inv;
                    }
                    __syncwarp();
                }
                // four points' loads in flight at a time; psi and dE of the first four before the rotation
                for (int r0 = m.sub; r0 < np; r0 += 4 * m.nsub) {
                    V s[EPL][4];
#pragma unroll
                    for (int a = 0; a < EPL; ++a) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int r = r0 + u * m.nsub, e = m.e + 32 * a;
                            s[a][u] = Vn && r < np && e < t ? Vn[o0 + r * t + e] : czero<V>();
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int r = r0 + u * m.nsub;
                        if (r >= np) break;
                        T f[8];
#pragma unroll
                        for (int l = 0; l < 8; ++l) f[l] = w.wt[r * 8 + l];
#pragma unroll
                        for (int a = 0; a < EPL; ++a) {
                            const int e = m.e + 32 * a;
                            if (EPL == 2 && e >= t) continue;
                            V q = s[a][u];
#pragma unroll
                            for (int l = 0; l < 8; ++l) {
                                q.x = fma(f[l], rr[a][l].x, q.x);
                                q.y = fma(f[l], rr[a][l].y, q.y);
                            }
                            w.X[r * tp + e] = q;
                        }
                    }
                }
                V p4[EPL][4];
                T d4[EPL][4];
                auto fetch = [&](int r0) {
#pragma unroll
                    for (int a = 0; a < EPL; ++a) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int r = r0 + u * m.nsub, e = m.e + 32 * a;
                            const bool in = r < np && e < t;
                            p4[a][u] = in ? psi[o0 + r * t + e] : czero<V>();
                            d4[a][u] = in ? dE[g0 + r * t + e] : (T)0;
                        }
                    }
                };
                fetch(m.sub);
                __syncwarp();
                rotate_warp<false>(w.X, w.Tm, tp, w.Uv, rvp, w.Uc, rcp, np, nv, nc);
                for (int r0 = m.sub; r0 < np; r0 += 4 * m.nsub) {
                    if (r0 != m.sub) fetch(r0);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int r = r0 + u * m.nsub;
                        if (r >= np) break;
#pragma unroll
                        for (int a = 0; a < EPL; ++a) {
                            const int e = m.e + 32 * a;
                            if (EPL == 2 && e >= t) continue;
                            const V s = w.X[r * tp + e], p = p4[a][u];
                            V o;
                            o.x = fma(p.x, d4[a][u], s.x);
                            o.y = fma(p.y, d4[a][u], s.y);
                            W[o0 + r * t + e] = o;
                            dsm.add(p, o);
                        }
                    }
                }
                __syncwarp();
            }
            dsum[c][tid] = dsm;
        }
        __syncthreads();
        if (warp < ncb) {
            DotSum<T> low = DotSum<T>::zero();
#pragma unroll
            for (int q = 0; q < 8; ++q) dsum[warp][lane + 32 * q].into(dot, low);
            dot = cadd(dot, low.value());
        }
    }
    if (warp < ncb) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            dot.x += __shfl_down_sync(0xffffffffu, dot.x, o);
            dot.y += __shfl_down_sync(0xffffffffu, dot.y, o);
        }
        if (lane == 0) part[(size_t)(c0 + warp) * BSE_MAX_VEC_BLOCKS + blockIdx.x] = dot;
    }
}

// ----------------------------------------------------------- near stencil
// V(k) = sum_delta W(j, delta) phi(k + delta) over the near offsets |delta|^2 <= R2.
//
// Per target and column (one real component of one chain) one multiply-add per
// near offset is needed: 808 M for coarse 8^3, n_div 4, w 1, 3 chains of 16
// transitions.  A warp takes one column group, a column per lane, and TY rows of
// cells that follow each other along z: a source is loaded once for up to
// TY (2 r + 1) multiply-adds, and since W is the same in every cell one broadcast
// load of weights serves every cell of the run.
// It walks the source rows (delta_1, row u) of its ball in set-up's list; the
// reach r of the row along z selects an unrolled body, so only offsets
// inside the ball cost arithmetic and the source row sits in registers.
// Sources come straight from phi (the warps of a block share their cells, hence
// rows, through L1); the weights of the next row are copied to the warp's buffer
// meanwhile.  RM: the largest r that the unrolled body covers (R <= RM); RM = 0
// loops over the offsets.
struct NearStencil {
    int n, L, Lp, R, nd, njb, nzb;                 // njb: weight blocks along y; nzb: blocks of TZ targets j3
    int nyb;                                       // FP32: pairs of target rows along the whole zone
    int nsteps, wrow, wbytes;                      // source rows, weights of one, shared memory of a warp
    int cols, t2, ntz, warps;                      // columns in use, 2 t, z tiles (of cz cells, the last ones smaller), all warps
    int cz;
    int split;                                     // the source rows of a warp's targets go to the four warps of a block
    long long N2;                                  // 2 N: reals per chain of V
};

// Small grids (at most one warp per scheduler, so cz = 1) wait out the latency of a
// source row nsteps times in a row: there the four warps of a block take a quarter of
// the rows of the same targets each and their sums are added in warp order.
// Coarse 4^3, n_div 2, 3x3 bands, 1 vector, FP64: 17.1 -> 10.1 us.
__device__ __forceinline__ int2 near_steps(const NearStencil& s) {
    if (!s.split) return make_int2(0, s.nsteps);
    const int part = threadIdx.x >> 5;
    return make_int2(part * s.nsteps / 4, (part + 1) * s.nsteps / 4);
}
// Adds the four warps' sums into warp 0's; false for the others, which are done.
template <int N, typename E, typename Add>
__device__ __forceinline__ bool near_gather(E (&acc)[N], unsigned char* red, Add add) {
    E* r = reinterpret_cast<E*>(red);
    const int part = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (part) {
#pragma unroll
        for (int i = 0; i < N; ++i) r[((part - 1) * N + i) * 32 + lane] = acc[i];
    }
    __syncthreads();
    if (part) return false;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
#pragma unroll
        for (int i = 0; i < N; ++i) acc[i] = add(acc[i], r[(q * N + i) * 32 + lane]);
    }
    return true;
}

// Weights of one offset of one FP64 target row in the table: TZ values, padded
// to what the loads below read.
template <int TZ> constexpr int near_tzp() { return TZ == 3 ? 4 : TZ; }

// A warp's weights buffer (two rows of the table) and the places of its source rows,
// wrapped around the zone: [2 R + 1] planes from x0, [2 R + TY] rows from y0.
template <typename T, int TY>
struct NearWarp {
    static constexpr int PER = 16 / sizeof(T);
    T *wbuf, *wdst;
    const T* wsrc;
    int *xo, *yo;
    __device__ NearWarp(T* buf, const T* Wt, int block, int step0, const NearStencil& s, int x0, int y0) {
        const int lane = threadIdx.x & 31;
        wbuf = buf;
        wdst = buf + lane * PER;
        wsrc = Wt + ((size_t)block * s.nsteps + step0) * s.wrow + lane * PER;
        xo = reinterpret_cast<int*>(buf + 2 * s.wrow);
        yo = xo + 2 * s.R + 1;
        for (int i = lane; i <= 2 * s.R; i += 32) {
            int x = x0 - s.R + i;
            x += x < 0 ? s.L : (x >= s.L ? -s.L : 0);
            xo[i] = x * s.L * s.Lp;
        }
        for (int i = lane; i < 2 * s.R + TY; i += 32) {
            int y = y0 - s.R + i;
            y += y < 0 ? s.L : (y >= s.L ? -s.L : 0);
            yo[i] = y * s.Lp;
        }
    }
    // the next row of weights, into the buffer's half 0 or wrow
    __device__ __forceinline__ void fetch(int half, int wrow) {
        const int lane = threadIdx.x & 31;
        T* dst = wdst + half;
        if (lane * PER < wrow) cpa16(dst, wsrc);
        if (wrow > 32 * PER)
            for (int c = 32 * PER; c + lane * PER < wrow; c += 32 * PER) cpa16(dst + c, wsrc + c);
        wsrc += wrow;
        cpa_commit();
    }
    // st: delta_1 + R | u << 8 | r_max << 16, then the reach + 1 of each target row (0: none), a byte each
    __device__ __forceinline__ size_t at(int2 st) const { return (size_t)(unsigned)(xo[st.x & 255] + yo[(st.x >> 8) & 255]) * 32; }
};

// z tile tz: as many tiles of s.cz cells as fit, then what is left in powers of two.
__device__ __forceinline__ int2 near_tile(const NearStencil& s, int tz) {
    const int full = s.n / s.cz;
    int cz0 = min(tz, full) * s.cz, cz = s.cz;
    for (int q = full; q <= tz; ++q) {
        int left = s.n - cz0, p = 1;
        while (2 * p <= left) p *= 2;
        cz = p;
        if (q < tz) cz0 += p;
    }
    return make_int2(cz0, tz < full ? s.cz : cz);
}

// FP64.  A row of targets' sums over the offsets -r .. r of a source row that is
// held from -rm on: a[i] += w[i mod TZ] v[i + offset].
template <int TZ, int NT, int rm, int r>
__device__ __forceinline__ void near_reach(double (&a)[NT], const double (&v)[NT + 2 * rm], const double* wb) {
#pragma unroll
    for (int d = -r; d <= r; ++d) {
        double w[TZ];
#pragma unroll
        for (int q = 0; q < TZ; ++q) w[q] = wb[d * near_tzp<TZ>() + q];
#pragma unroll
        for (int i = 0; i < NT; ++i) a[i] = fma(w[i % TZ], v[i + d + rm], a[i]);
    }
}
// One source row that reaches rm: its columns into registers, then every target
// row with its own reach r <= rm (code r + 1; 0: not reached).
template <int TY, int TZ, int NT, int rm>
__device__ __forceinline__ void near_row(double (&acc)[TY][NT], const double* __restrict__ row, const double* wb, int wy, int reach) {
    double v[NT + 2 * rm];
#pragma unroll
    for (int z = -rm; z < NT + rm; ++z) v[z + rm] = __ldg(row + z * 32);
    cpa_wait<1>();
    __syncwarp();
#pragma unroll
    for (int y = 0; y < TY; ++y) {
        const double* w = wb + y * wy;
        const int r = ((reach >> (8 * y)) & 255) - 1;
        if (r == rm) near_reach<TZ, NT, rm, rm>(acc[y], v, w);
        if constexpr (rm >= 1) { if (r == 0) near_reach<TZ, NT, rm, 0>(acc[y], v, w); }
        if constexpr (rm >= 2) { if (r == 1) near_reach<TZ, NT, rm, 1>(acc[y], v, w); }
        if constexpr (rm >= 3) { if (r == 2) near_reach<TZ, NT, rm, 2>(acc[y], v, w); }
        if constexpr (rm >= 4) { if (r == 3) near_reach<TZ, NT, rm, 3>(acc[y], v, w); }
        if constexpr (rm >= 5) { if (r == 4) near_reach<TZ, NT, rm, 4>(acc[y], v, w); }
        if constexpr (rm >= 6) { if (r == 5) near_reach<TZ, NT, rm, 5>(acc[y], v, w); }
    }
}

template <int TY, int TZ, int CZ, int RM>
__device__ __forceinline__ void near_body(const double* __restrict__ phi, const double* __restrict__ Wt,
                                          const int2* __restrict__ steps, double* __restrict__ Vn, const NearStencil& s, int g,
                                          int cx, int cy, int cz0, int j1, int j2, int zb, double* wbuf, unsigned char* red) {
    constexpr int TZP = near_tzp<TZ>(), NT = CZ * TZ;
    const int lane = threadIdx.x & 31, nd = s.nd, R = s.R, wy = (2 * R + 1) * TZP;
    const int2 span = CZ == 1 ? near_steps(s) : make_int2(0, s.nsteps);
    NearWarp<double, TY> nw(wbuf, Wt, (zb * nd + j1) * s.njb + j2 / TY, span.x, s, cx * nd + j1, cy * nd + j2);
    const double* base = phi + (size_t)g * s.L * s.L * s.Lp * 32 + (size_t)(cz0 * nd + zb * TZ + R) * 32 + lane;
    double acc[TY][NT];
#pragma unroll
    for (int y = 0; y < TY; ++y) {
#pragma unroll
        for (int i = 0; i < NT; ++i) acc[y][i] = 0.0;
    }
    int2 st = steps[span.x];
    int cur = 0;                                                      // 0 or wrow: the buffer of this step's weights
    nw.fetch(0, s.wrow);
    __syncwarp();
    for (int i = span.x; i < span.y; ++i) {
        int2 nx = st;
        if (i + 1 < span.y) {
            nx = steps[i + 1];
            nw.fetch(s.wrow - cur, s.wrow);
        } else {
            cpa_commit();
        }
        const double* row = base + nw.at(st);
        const int rm = st.x >> 16;
        const double* wb = wbuf + cur + R * TZP;
        if constexpr (RM > 0) {
            switch (rm) {
                case 0: near_row<TY, TZ, NT, 0>(acc, row, wb, wy, st.y); break;
                case 1: near_row<TY, TZ, NT, 1>(acc, row, wb, wy, st.y); break;
                case 2: near_row<TY, TZ, NT, 2>(acc, row, wb, wy, st.y); break;
                case 3: near_row<TY, TZ, NT, 3>(acc, row, wb, wy, st.y); break;
                case 4: near_row<TY, TZ, NT, 4>(acc, row, wb, wy, st.y); break;
                default:
                    if constexpr (RM >= 6) {
                        if (rm == 5) near_row<TY, TZ, NT, 5>(acc, row, wb, wy, st.y);
                        else near_row<TY, TZ, NT, 6>(acc, row, wb, wy, st.y);
                    }
            }
        } else {
            cpa_wait<1>();
            __syncwarp();
            for (int d = -rm; d <= rm; ++d) {
                double v[NT];
#pragma unroll
                for (int z = 0; z < NT; ++z) v[z] = __ldg(row + (z + d) * 32);
#pragma unroll
                for (int q = 0; q < TY; ++q) {
#pragma unroll
                    for (int z = 0; z < NT; ++z) acc[q][z] = fma(wb[q * wy + d * TZP + z % TZ], v[z], acc[q][z]);
                }
            }
        }
        __syncwarp();
        st = nx;
        cur = s.wrow - cur;
    }
    if constexpr (CZ == 1)
        if (s.split) {
            double (&flat)[TY * NT] = reinterpret_cast<double (&)[TY * NT]>(acc);
            if (!near_gather(flat, red, [](double a, double b) { return a + b; })) return;
        }
    const int col = g * 32 + lane;
    if (col >= s.cols) return;
    const int ch = col / s.t2, q = col - ch * s.t2;
    double* out = Vn + (size_t)ch * s.N2 + q;
#pragma unroll
    for (int c = 0; c < CZ; ++c) {
#pragma unroll
        for (int y = 0; y < TY; ++y) {
#pragma unroll
            for (int z = 0; z < TZ; ++z)
                if (j2 + y < nd && zb * TZ + z < nd) {
                    const size_t kd = ((size_t)((cx * s.n + cy) * s.n + cz0 + c) * nd + j1) * nd * nd + (j2 + y) * nd + zb * TZ + z;
                    out[kd * s.t2] = acc[y][c * TZ + z];
                }
        }
    }
}

template <int TY, int TZ, int RM>
__global__ void __launch_bounds__(128, 3) k_common_near(const double* __restrict__ phi, const double* __restrict__ Wt,
                                                        const int2* __restrict__ steps, double* __restrict__ Vn, const NearStencil s) {
    extern __shared__ __align__(16) unsigned char smraw[];
    double* wbuf = reinterpret_cast<double*>(smraw + (size_t)(threadIdx.x >> 5) * s.wbytes);
    unsigned char* red = smraw + (size_t)4 * s.wbytes;
    int w = s.split ? blockIdx.x : blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (w >= s.warps) return;
    // warp: (group, cx, cy, z tile, z block, j1, block of j2), the last fastest
    const int jb = w % s.njb; w /= s.njb;
    const int j1 = w % s.nd; w /= s.nd;
    const int zb = w % s.nzb; w /= s.nzb;
    const int2 tile = near_tile(s, w % s.ntz); w /= s.ntz;
    const int cy = w % s.n; w /= s.n;
    const int cx = w % s.n, g = w / s.n;
    if constexpr (RM > 0) {
        if (tile.y == 4) near_body<TY, TZ, 4, RM>(phi, Wt, steps, Vn, s, g, cx, cy, tile.x, j1, jb * TY, zb, wbuf, red);
        else if (tile.y == 2) near_body<TY, TZ, 2, RM>(phi, Wt, steps, Vn, s, g, cx, cy, tile.x, j1, jb * TY, zb, wbuf, red);
        else near_body<TY, TZ, 1, RM>(phi, Wt, steps, Vn, s, g, cx, cy, tile.x, j1, jb * TY, zb, wbuf, red);
    } else {
        near_body<TY, TZ, 1, RM>(phi, Wt, steps, Vn, s, g, cx, cy, tile.x, j1, jb * TY, zb, wbuf, red);
    }
}

// FP32: the two rows Y, Y + 1 (Y even, along the whole zone: a pair may belong to two
// cells) are the halves of packed multiply-adds, so the weights of an offset lie as
// they are used, row pair by row pair, and a broadcast load of them serves twice the
// multiply-adds that it serves when each weight is stored twice for a packed complex
// column: shared-memory bandwidth bounds this kernel, not the multiply-adds.  The
// source is the operand to double, once per load.  Both rows take the larger reach
// of the two (zero weights beyond their own).  Coarse 8^3, n_div 4, 4x4 bands, 3 chains beside
// the K_c apply: 130 us with weights stored twice, 122 us so, 110 us since the apply leaves it
// registers (84 us alone); with 80 registers (six blocks per SM, all warps at once) 124 us.
__device__ __forceinline__ F2 twice(float x) { return f2_pair(x, x); }
// The TZ weight pairs of one offset (16-byte loads where each offset starts on 16 bytes).
template <int TZ>
__device__ __forceinline__ void near_pairs(F2 (&w)[TZ], const float* p) {
    if constexpr (TZ % 2) {
#pragma unroll
        for (int q = 0; q < TZ; ++q) w[q] = reinterpret_cast<const F2*>(p)[q];
    } else {
#pragma unroll
        for (int q = 0; q < TZ; q += 2) {
            const ulonglong2 f = *reinterpret_cast<const ulonglong2*>(p + 2 * q);
            w[q] = f.x;
            w[q + 1] = f.y;
        }
    }
}
template <int TZ, int NT, int rm>
__device__ __forceinline__ void near_row32(F2 (&acc)[NT], const float* __restrict__ row, const float* wb) {
    F2 v[NT + 2 * rm];
#pragma unroll
    for (int z = -rm; z < NT + rm; ++z) v[z + rm] = twice(__ldg(row + z * 32));
    cpa_wait<1>();
    __syncwarp();
#pragma unroll
    for (int d = -rm; d <= rm; ++d) {
        F2 w[TZ];
        near_pairs<TZ>(w, wb + d * 2 * TZ);
#pragma unroll
        for (int i = 0; i < NT; ++i) acc[i] = f2_fma(w[i % TZ], v[i + d + rm], acc[i]);
    }
}

template <int TZ, int CZ, int RM>
__device__ __forceinline__ void near_body32(const float* __restrict__ phi, const float* __restrict__ Wt,
                                            const int2* __restrict__ steps, float* __restrict__ Vn, const NearStencil& s, int g,
                                            int X, int Y, int cz0, int zb, float* wbuf, unsigned char* red) {
    constexpr int NT = CZ * TZ;
    const int lane = threadIdx.x & 31, nd = s.nd, R = s.R, cx = X / nd, j1 = X - cx * nd, cy = Y / nd, j2 = Y - cy * nd;
    const int2 span = CZ == 1 ? near_steps(s) : make_int2(0, s.nsteps);
    NearWarp<float, 2> nw(wbuf, Wt, (zb * nd + j1) * s.njb + (nd % 2 ? j2 : j2 / 2), span.x, s, X, Y);
    const float* base = phi + (size_t)g * s.L * s.L * s.Lp * 32 + (size_t)(cz0 * nd + zb * TZ + R) * 32 + lane;
    F2 acc[NT];
#pragma unroll
    for (int i = 0; i < NT; ++i) acc[i] = 0;                          // the pair (0.f, 0.f)
    int2 st = steps[span.x];
    int cur = 0;                                                      // 0 or wrow: the buffer of this step's weights
    nw.fetch(0, s.wrow);
    __syncwarp();
    for (int i = span.x; i < span.y; ++i) {
        int2 nx = st;
        if (i + 1 < span.y) {
            nx = steps[i + 1];
            nw.fetch(s.wrow - cur, s.wrow);
        } else {
            cpa_commit();
        }
        const float* row = base + nw.at(st);
        const int rm = st.x >> 16;
        const float* wb = wbuf + cur + R * 2 * TZ;
        if constexpr (RM > 0) {
            switch (rm) {
                case 0: near_row32<TZ, NT, 0>(acc, row, wb); break;
                case 1: near_row32<TZ, NT, 1>(acc, row, wb); break;
                case 2: near_row32<TZ, NT, 2>(acc, row, wb); break;
                case 3: near_row32<TZ, NT, 3>(acc, row, wb); break;
                case 4: near_row32<TZ, NT, 4>(acc, row, wb); break;
                default:
                    if constexpr (RM >= 6) {
                        if (rm == 5) near_row32<TZ, NT, 5>(acc, row, wb);
                        else near_row32<TZ, NT, 6>(acc, row, wb);
                    }
            }
        } else {
            cpa_wait<1>();
            __syncwarp();
            for (int d = -rm; d <= rm; ++d) {
                F2 w[TZ];
                near_pairs<TZ>(w, wb + d * 2 * TZ);
#pragma unroll
                for (int z = 0; z < NT; ++z) acc[z] = f2_fma(w[z % TZ], twice(__ldg(row + (z + d) * 32)), acc[z]);
            }
        }
        __syncwarp();
        st = nx;
        cur = s.wrow - cur;
    }
    if constexpr (CZ == 1)
        if (s.split && !near_gather(acc, red, [](F2 a, F2 b) {
                const float2 x = *reinterpret_cast<const float2*>(&a), y = *reinterpret_cast<const float2*>(&b), z = cadd(x, y);
                return *reinterpret_cast<const F2*>(&z);
            }))
            return;
    const int col = g * 32 + lane;
    if (col >= s.cols) return;
    const int ch = col / s.t2, q = col - ch * s.t2;
    float* out = Vn + (size_t)ch * s.N2 + q;
    // the second row: the next one of the cell or the first of the next cell; none beyond the zone
    const bool two = Y + 1 < s.L, same = j2 + 1 < nd;
    const size_t k0 = ((size_t)((cx * s.n + cy) * s.n + cz0) * nd + j1) * nd * nd + j2 * nd + zb * TZ;
    const size_t k1 = same ? k0 + nd : ((size_t)((cx * s.n + cy + 1) * s.n + cz0) * nd + j1) * nd * nd + zb * TZ;
#pragma unroll
    for (int c = 0; c < CZ; ++c) {
#pragma unroll
        for (int z = 0; z < TZ; ++z)
            if (zb * TZ + z < nd) {
                const F2 a = acc[c * TZ + z];
                const size_t o = (size_t)c * nd * nd * nd + z;
                out[(k0 + o) * s.t2] = __uint_as_float((unsigned)a);
                if (two) out[(k1 + o) * s.t2] = __uint_as_float((unsigned)(a >> 32));
            }
    }
}

template <int TZ, int RM>
__global__ void __launch_bounds__(128, 5) k_common_near32(const float* __restrict__ phi, const float* __restrict__ Wt,
                                                          const int2* __restrict__ steps, float* __restrict__ Vn,
                                                          const NearStencil s) {
    extern __shared__ __align__(16) unsigned char smraw[];
    float* wbuf = reinterpret_cast<float*>(smraw + (size_t)(threadIdx.x >> 5) * s.wbytes);
    unsigned char* red = smraw + (size_t)4 * s.wbytes;
    int w = s.split ? blockIdx.x : blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (w >= s.warps) return;
    // warp: (group, z tile, z block, row X, pair of rows Y), the last fastest
    const int yb = w % s.nyb; w /= s.nyb;
    const int X = w % s.L; w /= s.L;
    const int zb = w % s.nzb; w /= s.nzb;
    const int2 tile = near_tile(s, w % s.ntz);
    const int g = w / s.ntz;
    if constexpr (RM > 0) {
        if (tile.y == 4) near_body32<TZ, 4, RM>(phi, Wt, steps, Vn, s, g, X, 2 * yb, tile.x, zb, wbuf, red);
        else if (tile.y == 2) near_body32<TZ, 2, RM>(phi, Wt, steps, Vn, s, g, X, 2 * yb, tile.x, zb, wbuf, red);
        else near_body32<TZ, 1, RM>(phi, Wt, steps, Vn, s, g, X, 2 * yb, tile.x, zb, wbuf, red);
    } else {
        near_body32<TZ, 1, RM>(phi, Wt, steps, Vn, s, g, X, 2 * yb, tile.x, zb, wbuf, red);
    }
}

// Weights of the near stencil, FP64 arithmetic, one thread per entry: index
// [z block][j1][block of j2][step] and then, for FP64, [row y][delta_3 + R][target z]
// (near_tzp entries per offset), for FP32 [delta_3 + R][target z][row y] (blocks start at
// every second row of the zone, taken modulo the cell); steps padded to `wrow`, zero outside the
// ball and for padding; scale = alpha / N_div.
template <typename T>
__global__ void k_common_weights(const double* __restrict__ hcoarse, const int2* __restrict__ steps, int nsteps, int n, int nd,
                                 int nb1, int R, int R2, int TY, int TZ, int TZP, int njb, int wrow, double kappa, double scale,
                                 long long total, T* __restrict__ Wt) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    constexpr bool pairs = sizeof(T) == 4;
    const int D = 2 * R + 1;
    const int e = (int)(i % wrow);
    long long q = i / wrow;
    const int2 st = steps[q % nsteps]; q /= nsteps;
    const int jb = (int)(q % njb); q /= njb;
    const int j1 = (int)(q % nd);
    const int zb = (int)(q / nd);
    const int tz = pairs ? (e / 2) % TZ : e % TZP, y = pairs ? e % 2 : e / (TZP * D), o3 = pairs ? e / (2 * TZ) : (e / TZP) % D;
    const int j2 = pairs ? (jb * (nd % 2 ? 1 : 2) + y) % nd : jb * TY + y, j3 = zb * TZ + tz;
    const int d1 = (st.x & 255) - R, d2 = ((st.x >> 8) & 255) - y - R, d3 = o3 - R;
    T out = (T)0;
    if (y < TY && j2 < nd && tz < TZ && j3 < nd && o3 < D && d1 * d1 + d2 * d2 + d3 * d3 <= R2) {
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

// Points a warp rotates at a time: the cell's points over 8 warps, at most 8 (a row per
// lane for 4 valence bands), and 10 KB of shared memory.
template <typename T>
int rot_points(const bse_interp* s) {
    int kp = std::min((s->Ndiv + 7) / 8, 8);
    while (kp > 1 && WarpStage<T>::bytes(kp, s->nv, s->nc) > 10240) --kp;
    return kp;
}
// Chains per block: all of them once the cells alone fill the SMs.
int rot_chains(const bse_ctx* ctx, const bse_interp* s, int nchains) {
    return s->co->nkc >= 2 * std::max(ctx->sm_count, 1) ? nchains : 1;
}

// Targets of a warp within a cell: TZ = n_div up to 4 (then blocks of 4), TY rows
// (FP32: pairs of rows of the zone).
inline int near_tz(int nd) { return std::min(nd, 4); }
template <typename T>
int near_ty(int nd) { return sizeof(T) == 4 ? 2 : (nd <= 3 ? nd : 2); }
inline int near_tzp_of(int nd) { return near_tz(nd) == 3 ? near_tzp<3>() : near_tz(nd); }
// Blocks of rows with weights of their own: FP32 pairs start at any row of a cell when n_div is odd.
template <typename T>
int near_njb(int nd) { return sizeof(T) == 4 && nd % 2 ? nd : (nd + near_ty<T>(nd) - 1) / near_ty<T>(nd); }

// Elements of a step's weights, rounded up to 16 bytes.
template <typename T>
int near_wrow(int nd, int R) {
    const int per = 16 / (int)sizeof(T), e = near_ty<T>(nd) * (2 * R + 1) * (sizeof(T) == 4 ? near_tz(nd) : near_tzp_of(nd));
    return (e + per - 1) / per * per;
}

template <typename T, typename K>
int launch_near_k(bse_ctx* ctx, const bse_interp* s, const CommonWork& work, K kernel, int RM, NearStencil ns, cudaStream_t st) {
    const int groups = (ns.cols + 31) / 32, n = s->n;
    auto tiles = [&](int cz) {
        int c = n / cz;
        for (int left = n % cz; left; left &= left - 1) ++c;
        return c;
    };
    const long long per_tile = (long long)groups * ns.nzb *
                               (sizeof(T) == 4 ? (long long)ns.L * ns.nyb : (long long)n * n * ns.nd * ns.njb);
    // Cells per warp: as many as leave four warps per SM (a warp alone on its scheduler
    // waits out its loads); z blocks do not continue into the next cell.  Four against at most two, FP32:
    // 8^3, n_div 4, 3 chains beside the K_c apply 109 and 124 us; 7^3, n_div 3, 4 vectors 70 and 86 us.
    ns.cz = 1;
    if (RM > 0 && ns.nzb == 1)
        for (int cz : {2, 4})
            if (n >= cz && per_tile * tiles(cz) >= 4LL * ctx->sm_count) ns.cz = cz;
    ns.ntz = tiles(ns.cz);
    const long long warps = per_tile * ns.ntz;
    if (warps > 0x7fffffffLL) { ctx->err = "near stencil: too many targets"; return BSE_ERR_UNSUPPORTED; }
    ns.warps = (int)warps;
    // small grids: fewer warps per block spread over more SMs, or the rows of a warp over a block
    ns.wbytes = (int)((sizeof(T) * 2 * (size_t)ns.wrow + sizeof(int) * (4 * ns.R + 1 + near_ty<T>(ns.nd)) + 15) / 16 * 16);
    ns.split = ns.cz == 1 && warps <= 4LL * ctx->sm_count && ns.nsteps >= 8;
    const int wpb = ns.split ? 4 : (warps >= 8LL * ctx->sm_count ? 4 : 2);
    const size_t smem = (size_t)ns.wbytes * wpb + (ns.split ? 3 * 32 * sizeof(double) * near_ty<T>(ns.nd) * near_tz(ns.nd) : 0);
    BSE_CUDA_TRY(ctx, bse_raise_smem(kernel, smem, 0));
    kernel<<<(unsigned)(ns.split ? warps : (warps + wpb - 1) / wpb), 32 * wpb, smem, st>>>((const T*)work.phi, (const T*)s->d_cw, s->d_csteps,
                                                                       (T*)work.V, ns);
    BSE_CUDA_TRY(ctx, cudaGetLastError());
    return BSE_OK;
}
template <typename T, int TY, int TZ, int RM>
int launch_near_r(bse_ctx* ctx, const bse_interp* s, const CommonWork& work, const NearStencil& ns, cudaStream_t st) {
    if constexpr (sizeof(T) == 4) return launch_near_k<T>(ctx, s, work, k_common_near32<TZ, RM>, RM, ns, st);
    else return launch_near_k<T>(ctx, s, work, k_common_near<TY, TZ, RM>, RM, ns, st);
}

// The bodies with the reach unrolled end at R = 4 (n_div up to 3) and 6; beyond, and with
// n_div above 4 for the runs of cells, the offsets are looped over.  That form against
// the general kernels, FP32, one application: coarse 8^3, n_div 4, 4x4 bands, 3 vectors, R = 8
// 24.6 -> 1.17 ms, R = 12 72.5 -> 3.08 ms; coarse 12^3, n_div 2, 2x3 bands, 3 vectors, R = 6
// 25.8 -> 0.57 ms; coarse 4^3, n_div 8, 2x2 bands, 1 vector, R = 8 39.0 -> 0.48 ms (FP64 58.7 -> 4.29).
template <typename T>
int near_typed(bse_ctx* ctx, const bse_interp* s, const CommonWork& work, int nchains, cudaStream_t st) {
    NearStencil ns{};
    const int nd = s->nd;
    ns.n = s->n; ns.nd = nd; ns.L = s->n * nd; ns.R = s->cphi_R; ns.Lp = s->cphi_Lp;
    ns.nzb = (nd + near_tz(nd) - 1) / near_tz(nd);
    ns.njb = near_njb<T>(nd);
    ns.nyb = (ns.L + 1) / 2;
    ns.nsteps = s->n_csteps;
    ns.wrow = near_wrow<T>(nd, ns.R);
    ns.t2 = 2 * s->t; ns.cols = ns.t2 * nchains; ns.N2 = 2LL * s->N;
    const bool r4 = ns.R <= 4, r6 = ns.R <= 6;
    switch (nd) {
        case 1: return r4 ? launch_near_r<T, 1, 1, 4>(ctx, s, work, ns, st) : launch_near_r<T, 1, 1, 0>(ctx, s, work, ns, st);
        case 2: return r4 ? launch_near_r<T, 2, 2, 4>(ctx, s, work, ns, st) : launch_near_r<T, 2, 2, 0>(ctx, s, work, ns, st);
        case 3: return r4 ? launch_near_r<T, 3, 3, 4>(ctx, s, work, ns, st) : launch_near_r<T, 3, 3, 0>(ctx, s, work, ns, st);
        default:
            return r4   ? launch_near_r<T, 2, 4, 4>(ctx, s, work, ns, st)
                   : r6 ? launch_near_r<T, 2, 4, 6>(ctx, s, work, ns, st)
                        : launch_near_r<T, 2, 4, 0>(ctx, s, work, ns, st);
    }
}

template <typename T>
int restrict_typed(bse_ctx* ctx, const bse_interp* s, const CommonWork& work, int nchains, const void* psi, void* Q,
                   __nv_bfloat16* bop, cudaStream_t st) {
    using V = typename Cx<T>::V;
    const bse_coarse* c = s->co;
    const int KP = rot_points<T>(s), CPB = rot_chains(ctx, s, nchains);
    const size_t smem = 8 * WarpStage<T>::bytes(KP, s->nv, s->nc) + sizeof(V) * 8 * (s->t <= 32 ? 32 / s->t : 1) * 8 * s->t;
    const bool m3 = s->scheme == BSE_SCHEME_M3;
    CommonPhi lay{s->cphi_R, s->cphi_Lp};
    const dim3 grid(c->nkc, (nchains + CPB - 1) / CPB);
    auto go = [&](auto kernel) -> int {
        BSE_CUDA_TRY(ctx, bse_raise_smem(kernel, smem, 64));
        kernel<<<grid, 256, smem, st>>>((const V*)psi, (const V*)s->d_cUv, (const V*)s->d_cUc, (const V*)s->d_cUvc,
                                        (const V*)s->d_cUcc, s->n, s->nd, s->nv, s->nc, s->nb1, nchains, CPB, KP,
                                        m3 ? (T*)work.phi : nullptr, lay, (V*)work.share, work.ctr, (V*)Q, bop, c->ldk);
        BSE_CUDA_TRY(ctx, cudaGetLastError());
        return BSE_OK;
    };
    if (c->kc_prec == BSE_PREC_BF16) return s->t <= 32 ? go(k_common_restrict<T, true, 1>) : go(k_common_restrict<T, true, 2>);
    return s->t <= 32 ? go(k_common_restrict<T, false, 1>) : go(k_common_restrict<T, false, 2>);
}

template <typename T>
int prolong_typed(bse_ctx* ctx, const bse_interp* s, const CommonWork& work, int nchains, const void* R, const void* psi, void* W,
                  double2* dot, cudaStream_t st) {
    using V = typename Cx<T>::V;
    const int KP = rot_points<T>(s), CPB = rot_chains(ctx, s, nchains);
    const size_t smem = (sizeof(V) * (sizeof(T) == 8 ? 2 : 1) * 8 * CPB * odd(s->t) + 15) / 16 * 16 +
                        8 * WarpStage<T>::bytes(KP, s->nv, s->nc);
    const dim3 grid(bse_common_dot_blocks(s), (nchains + CPB - 1) / CPB);
    auto go = [&](auto kernel) -> int {
        BSE_CUDA_TRY(ctx, bse_raise_smem(kernel, smem, sizeof(DotSum<T>) * BSE_MAX_CHAINS * 256));
        kernel<<<grid, 256, smem, st>>>((const V*)R, s->scheme == BSE_SCHEME_M3 ? (const V*)work.V : nullptr,
                                        (const V*)s->d_cUv, (const V*)s->d_cUc, (const V*)s->d_cUvc, (const V*)s->d_cUcc,
                                        (const T*)s->d_dE, (const V*)psi, s->n, s->nd, s->nv, s->nc, s->nb1, nchains, CPB, KP,
                                        (V*)W, dot);
        BSE_CUDA_TRY(ctx, cudaGetLastError());
        return BSE_OK;
    };
    return s->t <= 32 ? go(k_common_prolong<T, 1>) : go(k_common_prolong<T, 2>);
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
    if ((rc_ = bse_alloc(ctx, &s->cwork.share, sizeof(V) * BSE_MAX_CHAINS * 8 * (size_t)c->Nc, "corner shares")) != BSE_OK) return rc_;
    if ((rc_ = bse_alloc(ctx, (void**)&s->cwork.ctr, sizeof(int) * BSE_MAX_CHAINS * (size_t)c->nkc, "corner counters")) != BSE_OK) return rc_;
    BSE_CUDA_TRY(ctx, cudaMemsetAsync(s->cwork.ctr, 0, sizeof(int) * BSE_MAX_CHAINS * (size_t)c->nkc, st));
    if (s->scheme != BSE_SCHEME_M3) {
        BSE_CUDA_TRY(ctx, cudaStreamSynchronize(st));
        return BSE_OK;
    }
    const int nd = s->nd, L = s->n * nd, R = s->cphi_R, TY = near_ty<T>(nd), TZ = near_tz(nd), D = 2 * R + 1;
    // rows of phi: R points of halo on each side, and what a padded target block reads beyond (zeros)
    s->cphi_Lp = L + 2 * R + (nd > 4 ? 3 : 0);
    const size_t groups = (2 * (size_t)s->t * BSE_MAX_CHAINS + 31) / 32;
    const size_t nphi = groups * L * L * (size_t)s->cphi_Lp * 32;
    // unused columns stay zero (they and what a padded target reads are summed up but never stored)
    if ((rc_ = bse_alloc(ctx, &s->cwork.phi, sizeof(T) * nphi, "common-basis vectors")) != BSE_OK) return rc_;
    BSE_CUDA_TRY(ctx, cudaMemsetAsync(s->cwork.phi, 0, sizeof(T) * nphi, st));
    if ((rc_ = bse_alloc(ctx, &s->cwork.V, sizeof(V) * BSE_MAX_CHAINS * (size_t)s->N, "near stencil result")) != BSE_OK) return rc_;
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
    BSE_CUDA_TRY(ctx, bse_upload(ctx, s->d_csteps, steps.data(), sizeof(int2) * steps.size()));
    const int nzb = (nd + TZ - 1) / TZ, njb = near_njb<T>(nd), wrow = near_wrow<T>(nd, R);
    const long long nw = (long long)nzb * nd * njb * s->n_csteps * wrow;
    if ((rc_ = bse_alloc(ctx, &s->d_cw, sizeof(T) * (size_t)nw, "near stencil weights")) != BSE_OK) return rc_;
    k_common_weights<T><<<(unsigned)((nw + 127) / 128), 128, 0, st>>>(s->d_chead, s->d_csteps, s->n_csteps, s->n, nd, s->nb1, R,
                                                                      s->near_R2, TY, TZ, near_tzp_of(nd), njb, wrow, c->kappa,
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

size_t bse_common_work(const bse_interp* s, int nvec, unsigned char* base, CommonWork* w) {
    const size_t T = s->vec_prec == BSE_PREC_F64 ? sizeof(double) : sizeof(float), V = 2 * T, L = (size_t)s->n * s->nd;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        unsigned char* p = base + off;
        off += (bytes + 255) / 256 * 256;
        return (void*)p;
    };
    CommonWork q;
    if (s->scheme == BSE_SCHEME_M3) {
        q.phi = take(T * ((2 * (size_t)s->t * nvec + 31) / 32) * 32 * L * L * s->cphi_Lp);
        q.V = take(V * nvec * (size_t)s->N);
    }
    q.share = take(V * nvec * 8 * (size_t)s->co->Nc);
    q.ctr = (int*)take(sizeof(int) * nvec * (size_t)s->co->nkc);
    *w = q;
    return off;
}

int bse_common_prepare(bse_ctx* ctx, bse_interp* s) {
    return s->vec_prec == BSE_PREC_F64 ? prepare_typed<double>(ctx, s) : prepare_typed<float>(ctx, s);
}

int bse_common_restrict(bse_ctx* ctx, const bse_interp* s, const CommonWork& work, int nchains, const void* psi, void* Q,
                        __nv_bfloat16* bop, cudaStream_t st) {
    return s->vec_prec == BSE_PREC_F64 ? restrict_typed<double>(ctx, s, work, nchains, psi, Q, bop, st)
                                       : restrict_typed<float>(ctx, s, work, nchains, psi, Q, bop, st);
}

int bse_common_near(bse_ctx* ctx, const bse_interp* s, const CommonWork& work, int nchains, cudaStream_t st) {
    return s->vec_prec == BSE_PREC_F64 ? near_typed<double>(ctx, s, work, nchains, st) : near_typed<float>(ctx, s, work, nchains, st);
}

int bse_common_prolong(bse_ctx* ctx, const bse_interp* s, const CommonWork& work, int nchains, const void* R, const void* psi,
                       void* W, double2* dot, cudaStream_t st) {
    return s->vec_prec == BSE_PREC_F64 ? prolong_typed<double>(ctx, s, work, nchains, R, psi, W, dot, st)
                                       : prolong_typed<float>(ctx, s, work, nchains, R, psi, W, dot, st);
}
