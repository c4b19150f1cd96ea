// Learned near-diagonal residual: MLP training / inference kernels, pair-data
// generation from the method itself, and the learned correction applied as a
// periodic convolution on the dense mesh.
//
// Network (not in the paper): x -> 128 -> 128 -> 128 -> 2 with exact-erf GELU,
// BF16 weights, FP32 activations and accumulation, FP32 master weights and
// Adam state.  Parameter layout (FP32 master, gradients, Adam moments, and the
// BF16 weight copy share it): W1 [w][d_in], b1 [w], W2 [w][w], b2 [w],
// W3 [w][w], b3 [w], W4 [2][w], b4 [2].
//
// Inputs per (dense k, dense k', vc, v'c'): q (3, minimum image of k - k',
// orthonormal axes), |q|, onehot(vc) [t], onehot(v'c') [t], dE_vc(k),
// dE_v'c'(k').  Target: N_k (K_explicit - K_M1) (Re, Im).
#include <cmath>
#include <type_traits>
#include <vector>

#include "bse_dmat.cuh"
#include "bse_internal.cuh"

namespace {

constexpr int W = 128;
constexpr int TPB = 256;
constexpr double kPi = 3.14159265358979323846;

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// ------------------------------------------------ one pass over a row tile
// A block takes tiles of 32 batch rows through the whole network, activations
// and pre-activations in shared memory, each layer's BF16 weights staged as it
// comes; with TRAIN also the loss, the backward pass and the tile's share of
// every parameter's gradient, written to (or, from a block's second tile on,
// added to) the block's own slice of `gpart`.  k_grad_reduce sums the slices in
// block order.  Everything is FP32 (the weights' values are BF16): 7 layer
// products of 2 x 32 x 128 x 128 flops per tile, bound by the FP32 pipes and the
// shared-memory loads that feed them: 4 x 4 outputs per thread and 4 summands
// per load keep those at 12 wavefronts for 64 multiply-adds of a warp.
// Batch 4096, 54 inputs, GB300, a whole bse_mlp_gradients call: 2.53 ms with a kernel per
// layer and one thread per weight gradient (2.27 ms of it), 0.103 ms so; the gradients'
// error against 64 bits 9.2e-7 -> 5.7e-8.
constexpr int RT = 32;               // rows per tile
constexpr int WP = W + 4;            // pitch of a staged weight row (BF16) and of an activation row: conflict-free
__device__ __forceinline__ float2 bf2(uint32_t u) { return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)); }

// Weights [N][K] (row-major, BF16), columns k0 .. k0 + kc - 1, into ws [N][WP], zero padded to W columns.
__device__ __forceinline__ void stage_w(__nv_bfloat16* ws, const __nv_bfloat16* __restrict__ w, int N, int K, int k0, int kc) {
    if (K == W) {                                    // the inner layers: rows of 256 aligned bytes
        for (int i = threadIdx.x; i < N * (W / 4); i += TPB)
            *reinterpret_cast<uint2*>(ws + (i / (W / 4)) * WP + 4 * (i % (W / 4))) = reinterpret_cast<const uint2*>(w)[i];
        return;
    }
    for (int i = threadIdx.x; i < N * W; i += TPB) {
        const int n = i / W, k = i % W;
        ws[n * WP + k] = k < kc ? w[(size_t)n * K + k0 + k] : __float2bfloat16_rn(0.f);
    }
}
// acc[r][j] += sum_k in[4 ty + r][k] w[tx + 32 j][k] over kc columns (rounded up to 4; padding is zero)
__device__ __forceinline__ void fwd_tile(float (&acc)[4][4], const float* in, const __nv_bfloat16* ws, int kc, int ty, int tx) {
    for (int k = 0; k < kc; k += 4) {
        float4 x[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) x[r] = *reinterpret_cast<const float4*>(in + (4 * ty + r) * WP + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint2 u = *reinterpret_cast<const uint2*>(ws + (tx + 32 * j) * WP + k);
            const float2 a = bf2(u.x), b = bf2(u.y);
#pragma unroll
            for (int r = 0; r < 4; ++r)
                acc[r][j] = fmaf(x[r].w, b.y, fmaf(x[r].z, b.x, fmaf(x[r].y, a.y, fmaf(x[r].x, a.x, acc[r][j]))));
        }
    }
}
// acc[r][j] = sum_n dz[4 ty + r][n] w[n][4 tx + j]
__device__ __forceinline__ void bwd_tile(float (&acc)[4][4], const float* dz, const __nv_bfloat16* ws, int ty, int tx) {
    for (int n = 0; n < W; n += 4) {
        float4 d[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) d[r] = *reinterpret_cast<const float4*>(dz + (4 * ty + r) * WP + n);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const uint2 u = *reinterpret_cast<const uint2*>(ws + (n + m) * WP + 4 * tx);
            const float2 a = bf2(u.x), b = bf2(u.y);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float v = m == 0 ? d[r].x : (m == 1 ? d[r].y : (m == 2 ? d[r].z : d[r].w));
                acc[r][0] = fmaf(v, a.x, acc[r][0]);
                acc[r][1] = fmaf(v, a.y, acc[r][1]);
                acc[r][2] = fmaf(v, b.x, acc[r][2]);
                acc[r][3] = fmaf(v, b.y, acc[r][3]);
            }
        }
    }
}
// Gradient share of a layer of W outputs: dW[n][k0 + k] = sum_r dz[r][n] in[r][k], k < kc.
__device__ __forceinline__ void grad_tile(const float* dz, const float* in, int K, int k0, int kc, bool add, float* __restrict__ dW) {
    const int tn = threadIdx.x >> 4, tk = threadIdx.x & 15;          // 8 x 8 outputs per thread: n = 8 tn + i, k = 4 tk + 64 h + j
    if (4 * tk >= kc) return;
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
    for (int r = 0; r < RT; ++r) {
        const float4 a0 = *reinterpret_cast<const float4*>(dz + r * WP + 8 * tn), a1 = *reinterpret_cast<const float4*>(dz + r * WP + 8 * tn + 4);
        const float4 b0 = *reinterpret_cast<const float4*>(in + r * WP + 4 * tk), b1 = *reinterpret_cast<const float4*>(in + r * WP + 64 + 4 * tk);
        const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = (j >> 2) * 64 + 4 * tk + (j & 3);
            if (k < kc) {
                float* o = dW + (size_t)(8 * tn + i) * K + k0 + k;
                *o = add ? *o + acc[i][j] : acc[i][j];
            }
        }
}

struct MlpOffs { int w[4], b[4]; };

template <bool TRAIN>
__global__ void __launch_bounds__(TPB, 1) k_mlp(const float* __restrict__ X, const float* __restrict__ Y, int K, int B,
                                                const __nv_bfloat16* __restrict__ wt, const float* __restrict__ p, MlpOffs o,
                                                float inv_b, float* __restrict__ out, float* __restrict__ gpart, int nparams,
                                                double* __restrict__ lpart) {
    extern __shared__ __align__(16) unsigned char smraw[];
    float* xs = reinterpret_cast<float*>(smraw);                    // [RT][WP] input columns / scratch
    float* h[3];
    float* z[3];
    for (int i = 0; i < 3; ++i) {
        h[i] = xs + (1 + i) * RT * WP;
        z[i] = xs + (4 + i) * RT * WP;                              // only with TRAIN
    }
    __nv_bfloat16* ws = reinterpret_cast<__nv_bfloat16*>(xs + (TRAIN ? 7 : 4) * RT * WP);   // [W][WP]
    __shared__ float os[RT][2];
    __shared__ double ls[RT * 2];
    const int tid = threadIdx.x, ty = tid >> 5, tx = tid & 31;
    const int ntile = (B + RT - 1) / RT;
    double loss = 0.0;
    bool add = false;
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x, add = true) {
        const int r0 = tile * RT, rows = min(RT, B - r0);
        auto stage_x = [&](int k0, int kc) {
            for (int i = tid; i < RT * W; i += TPB) {
                const int r = i / W, k = i % W;
                xs[r * WP + k] = (r < rows && k < kc) ? X[(size_t)(r0 + r) * K + k0 + k] : 0.f;
            }
        };
        // ---- forward
        for (int l = 0; l < 3; ++l) {
            float acc[4][4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float bb = p[o.b[l] + tx + 32 * j];
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[r][j] = bb;
            }
            const int Kl = l == 0 ? K : W;
            for (int k0 = 0; k0 < Kl; k0 += W) {
                const int kc = min(W, Kl - k0);
                __syncthreads();
                stage_w(ws, wt + o.w[l], W, Kl, k0, kc);
                if (l == 0) stage_x(k0, kc);
                __syncthreads();
                fwd_tile(acc, l == 0 ? xs : h[l - 1], ws, kc, ty, tx);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int at = (4 * ty + r) * WP + tx + 32 * j;
                    if (TRAIN) z[l][at] = acc[r][j];
                    h[l][at] = gelu_f(acc[r][j]);
                }
        }
        __syncthreads();
        // output layer: 64 outputs, four threads each
        {
            const int q = tid >> 2, part = tid & 3, r = q >> 1, c = q & 1;
            float s = 0.f;
            for (int k = part; k < W; k += 4) s = fmaf(h[2][r * WP + k], __bfloat162float(wt[o.w[3] + c * W + k]), s);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (part == 0) {
                s += p[o.b[3] + c];
                float d = 0.f;
                if (r < rows) {
                    if (!TRAIN) out[2 * (size_t)(r0 + r) + c] = s;
                    else d = s - Y[2 * (size_t)(r0 + r) + c];
                }
                if (TRAIN) {
                    os[r][c] = 2.f * d * inv_b;
                    ls[q] = (double)d * d;
                }
            }
        }
        if (!TRAIN) continue;
        __syncthreads();
        if (tid == 0)
            for (int i = 0; i < 2 * RT; ++i) loss += ls[i];
        // ---- backward
        float* gp = gpart + (size_t)blockIdx.x * nparams;
        {   // output layer's gradients: weight (c, k) per thread
            const int c = tid >> 7, k = tid & 127;
            float g = 0.f, gb = 0.f;
            for (int r = 0; r < RT; ++r) {
                g = fmaf(os[r][c], h[2][r * WP + k], g);
                gb += os[r][c];
            }
            float* a = gp + o.w[3] + c * W + k;
            *a = add ? *a + g : g;
            if (k == 0) gp[o.b[3] + c] = add ? gp[o.b[3] + c] + gb : gb;
        }
        for (int i = tid; i < RT * W; i += TPB) {
            const int r = i / W, k = i % W;
            const float d = fmaf(os[r][1], __bfloat162float(wt[o.w[3] + W + k]), os[r][0] * __bfloat162float(wt[o.w[3] + k]));
            z[2][r * WP + k] = d * gelu_grad_f(z[2][r * WP + k]);
        }
        __syncthreads();
        for (int l = 2; l >= 0; --l) {
            const float* dz = z[l];
            if (tid < W) {
                float g = 0.f;
                for (int r = 0; r < RT; ++r) g += dz[r * WP + tid];
                float* a = gp + o.b[l] + tid;
                *a = add ? *a + g : g;
            }
            if (l > 0) {
                if (l < 2) stage_w(ws, wt + o.w[l], W, W, 0, W);      // W3 is still staged from the forward pass
                grad_tile(dz, h[l - 1], W, 0, W, add, gp + o.w[l]);
                __syncthreads();
                float acc[4][4];
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[r][j] = 0.f;
                bwd_tile(acc, dz, ws, ty, tx);
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float* at = z[l - 1] + (4 * ty + r) * WP + 4 * tx + j;
                        *at = acc[r][j] * gelu_grad_f(*at);
                    }
                __syncthreads();
            } else {
                for (int k0 = 0; k0 < K; k0 += W) {
                    const int kc = min(W, K - k0);
                    if (K > W) {                                       // else the forward pass's columns are still there
                        __syncthreads();
                        stage_x(k0, kc);
                        __syncthreads();
                    }
                    grad_tile(dz, xs, K, k0, kc, add, gp + o.w[0]);
                }
            }
        }
        __syncthreads();
    }
    if (TRAIN && tid == 0) lpart[blockIdx.x] = loss;
}

// g[i] = sum over the blocks' slices, in a fixed order: eight threads take every
// eighth slice, then their sums in order.
__global__ void __launch_bounds__(256) k_grad_reduce(const float* __restrict__ gpart, int nblk, int n, float* __restrict__ g) {
    __shared__ float sh[8][33];
    const int lane = threadIdx.x & 31, s = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    float a = 0.f;
    if (i < n)
#pragma unroll 4
        for (int b = s; b < nblk; b += 8) a += gpart[(size_t)b * n + i];
    sh[s][lane] = a;
    __syncthreads();
    if (s == 0 && i < n) {
        float t = sh[0][lane];
        for (int q = 1; q < 8; ++q) t += sh[q][lane];
        g[i] = t;
    }
}

// Adam on the FP32 master copy; BF16 weight copy refreshed (biases stay FP32).
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       int n, float lr, float b1, float b2, float eps, float c1, float c2,
                       __nv_bfloat16* __restrict__ wbf) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    wbf[i] = __float2bfloat16_rn(pi);
}

__global__ void k_to_bf16(const float* __restrict__ p, int n, __nv_bfloat16* __restrict__ w) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) w[i] = __float2bfloat16_rn(p[i]);
}

}  // namespace

// ------------------------------------------------------------------ handle
struct bse_mlp {
    int d_in = 0, nparams = 0, max_batch = 0, step = 0;
    float* d_p = nullptr;                // master FP32
    float* d_g = nullptr;                // gradients
    float* d_m = nullptr;
    float* d_v = nullptr;
    __nv_bfloat16* d_w = nullptr;        // BF16 copy
    float* d_gpart = nullptr;            // [blocks][nparams] the blocks' gradient shares
    double* d_part = nullptr;            // [blocks] the blocks' losses
    int blocks = 0;
};

namespace {

struct Layout {
    size_t off_w[4], off_b[4];
    int in_dim[4], out_dim[4];
};

Layout layout(int d_in) {
    Layout L;
    const int dims[5] = {d_in, W, W, W, 2};
    size_t o = 0;
    for (int i = 0; i < 4; ++i) {
        L.in_dim[i] = dims[i];
        L.out_dim[i] = dims[i + 1];
        L.off_w[i] = o;
        o += (size_t)dims[i + 1] * dims[i];
        L.off_b[i] = o;
        o += dims[i + 1];
    }
    return L;
}

int nparams_for(int d_in) { return (int)(W * d_in + W + 2 * (W * W + W) + 2 * W + 2); }

void free_mlp(bse_mlp* m) {
    if (!m) return;
    cudaFree(m->d_p); cudaFree(m->d_g); cudaFree(m->d_m); cudaFree(m->d_v); cudaFree(m->d_w);
    cudaFree(m->d_gpart);
    cudaFree(m->d_part);
    delete m;
}

size_t mlp_smem(bool train) { return sizeof(float) * (train ? 7 : 4) * RT * WP + sizeof(__nv_bfloat16) * W * WP; }

MlpOffs mlp_offs(int d_in) {
    const Layout L = layout(d_in);
    MlpOffs o;
    for (int i = 0; i < 4; ++i) { o.w[i] = (int)L.off_w[i]; o.b[i] = (int)L.off_b[i]; }
    return o;
}

// Forward over a batch: out [B][2] (device).
int mlp_forward(bse_ctx* ctx, bse_mlp* m, int B, const float* X, float* out) {
    const size_t sm = mlp_smem(false);
    BSE_CUDA_TRY(ctx, bse_raise_smem(k_mlp<false>, sm));
    k_mlp<false><<<std::min((B + RT - 1) / RT, 2 * std::max(ctx->sm_count, 1)), TPB, sm, ctx->stream>>>(
        X, nullptr, m->d_in, B, m->d_w, m->d_p, mlp_offs(m->d_in), 0.f, out, nullptr, m->nparams, nullptr);
    BSE_CUDA_TRY(ctx, cudaGetLastError());
    return BSE_OK;
}

// Loss and gradients into m->d_g; the loss (mean over the batch of the squared
// error summed over Re, Im) into *loss, the gradients also to the host where asked
// for, with one wait for both.
int mlp_grads(bse_ctx* ctx, bse_mlp* m, int B, const float* X, const float* Y, double* loss, float* grad_host) {
    const size_t sm = mlp_smem(true);
    BSE_CUDA_TRY(ctx, bse_raise_smem(k_mlp<true>, sm));
    const int nblk = std::min((B + RT - 1) / RT, m->blocks);
    k_mlp<true><<<nblk, TPB, sm, ctx->stream>>>(X, Y, m->d_in, B, m->d_w, m->d_p, mlp_offs(m->d_in), 1.f / B, nullptr,
                                                m->d_gpart, m->nparams, m->d_part);
    k_grad_reduce<<<(m->nparams + 31) / 32, 256, 0, ctx->stream>>>(m->d_gpart, nblk, m->nparams, m->d_g);
    BSE_CUDA_TRY(ctx, cudaGetLastError());
    std::vector<double> part(nblk);
    BSE_CUDA_TRY(ctx, cudaMemcpyAsync(part.data(), m->d_part, sizeof(double) * nblk, cudaMemcpyDeviceToHost, ctx->stream));
    if (grad_host)
        BSE_CUDA_TRY(ctx, cudaMemcpyAsync(grad_host, m->d_g, sizeof(float) * m->nparams, cudaMemcpyDeviceToHost, ctx->stream));
    BSE_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    double s = 0.0;
    for (double v : part) s += v;
    if (loss) *loss = s / B;
    return BSE_OK;
}

}  // namespace

// ================================================ pair data from the method
namespace {

// One block per sampled dense pair (k, k'): the t x t blocks of the explicit
// model kernel (FP64, dense weight e_k / N_k) and of K^{M1} = (1/N_div) F K_c F^H
// (FP32), written as network features and targets.
//  * The gauge at both points comes from a half warp per matrix; the form
//    factors M(k, G) = Uv^H mu(k, G) Uc from mu(k, G) once and one factor at a time.
//  * F is a Kronecker product of overlaps (Eq. interpwfn), so K_c blocks are
//    multiplied by d_c and d_v in turn, t (nv + nc) terms per entry row instead of
//    t^2, the blocks of all corners of k' at once, and F(k, l) is applied to
//    their sum.
//  * Overlaps come from the handle's tables or, on the common-basis path, from
//    the gauge (FP64).  They and the weights are rounded to FP32 each, where t x t
//    products would round the FP64 product of both overlaps and the weight once; the sums
//    are shorter by as much: against 64 bits the targets of 512 pairs of 4x6 bands are off by
//    7.1e-7 of their norm, with t x t products 4.0e-6.
//  * Rows of X leave in order, whole lines at a time.
// 512 pairs of 4x6 bands on GB300: 9.80 ms with t x t products per corner pair, form
// factors of 7 nv nc terms per entry and a thread per gauge; 0.61 ms so (FP64 and
// shared-memory loads share it).
constexpr int PTHR = 256;
size_t pairs_smem(int nv, int nc) {
    const int t = nv * nc, g = nv * nv + nc * nc;
    const size_t scratch = std::max(sizeof(double2) * (2 * kGaugeMats * g + 2 * 26 * t), sizeof(float2) * (size_t)(9 * t * t));
    return sizeof(double2) * (2 * (size_t)g + 2 * 26 * t + g) + scratch + sizeof(float2) * ((size_t)t * t + 16 * g);
}

template <typename T>
__global__ void __launch_bounds__(PTHR) k_pairs(
    const int* __restrict__ kd1, const int* __restrict__ kd2, const double2* __restrict__ gen_v,
    const double2* __restrict__ gen_c, const double2* __restrict__ mu, const double2* __restrict__ Uvc,
    const double2* __restrict__ Ucc, const typename Cx<T>::V* __restrict__ Kc, const typename Cx<T>::V* __restrict__ Dv,
    const typename Cx<T>::V* __restrict__ Dc, const T* __restrict__ dE, int n, int nd, int nv, int nc, int nb1, double e_k,
    double inv_eps, double kappa, int shells, int exchange_on, int d_in, float* __restrict__ X, float* __restrict__ Y) {
    extern __shared__ __align__(16) unsigned char prsm[];
    const int blk = blockIdx.x, tid = threadIdx.x, warp = tid >> 5;
    const int t = nv * nc, rv = nv * nv, rc = nc * nc, g = rv + rc, Ndiv = nd * nd * nd, L = n * nd, nk = n * n * n * Ndiv, Nc = t * n * n * n;
    double2* U = reinterpret_cast<double2*>(prsm);            // [2][Uv | Uc]
    double2* M = U + 2 * g;                                    // [2][26][t]
    double2* O = M + 2 * 26 * t;                               // O^v, O^c
    unsigned char* scratch = reinterpret_cast<unsigned char*>(O + g);
    double2* gw = reinterpret_cast<double2*>(scratch);         // gauge scratch, then form-factor scratch
    double2* fw = gw + 2 * kGaugeMats * g;                     // [2][26][t]
    float2* Kb = reinterpret_cast<float2*>(scratch);           // [8][t][t] blocks of K_c, then [t][t] their sum behind them
    float2* Ts = Kb + 8 * t * t;
    const size_t sbytes = max(sizeof(double2) * (2 * kGaugeMats * g + 2 * 26 * t), sizeof(float2) * (size_t)(9 * t * t));
    float2* K1 = reinterpret_cast<float2*>(scratch + sbytes);  // [t][t] K^{M1} N_div
    float2* dd = K1 + t * t;                                   // [2][8][Dv | Dc]
    __shared__ double sn[2][3], cs[2][3], hq;
    __shared__ int gi[2][3], cell[2], js[2];
    if (tid < 2) {
        const int kd = tid ? kd2[blk] : kd1[blk];
        cell[tid] = kd / Ndiv;
        js[tid] = kd % Ndiv;
        const Int3 ci = unflat3(cell[tid], n), j = unflat3(js[tid], nd);
        gi[tid][0] = ci.a * nd + j.a; gi[tid][1] = ci.b * nd + j.b; gi[tid][2] = ci.c * nd + j.c;
        for (int a = 0; a < 3; ++a) sincospi(2.0 * gi[tid][a] / L, &sn[tid][a], &cs[tid][a]);
    }
    __syncthreads();
    // gauge (warps 0, 1: a point each, a half warp per manifold); h(k - k') (warp 2); mu(k, G) (the rest)
    if (warp < 2) {
        const int half = (tid >> 4) & 1;
        const double2* E = grp_gauge(half ? gen_c : gen_v, half ? nc : nv, sn[warp], cs[warp],
                                     gw + warp * kGaugeMats * g + (half ? kGaugeMats * rv : 0));
        double2* out = U + warp * g + (half ? rv : 0);
        for (int e = grp_lane(); e < (half ? rc : rv); e += kGaugeLanes) out[e] = E[e];
    } else if (warp == 2) {
        // direct-term shape on the dense grid (minimum image, half-way differences average their images)
        int im[3][2], nimg = 1;
        for (int a = 0; a < 3; ++a) {
            const int r = imod(gi[0][a] - gi[1][a], L);
            im[a][0] = 2 * r > L ? r - L : r;
            im[a][1] = 2 * r >= L ? r - L : r;
            if (im[a][0] != im[a][1]) nimg *= 2;
        }
        double acc = 0.0;
        for (int q = tid & 31; q < 8 * 27; q += 32) {
            const int s = q / 27, G = q - 27 * s;
            bool dup = false;
            for (int a = 0; a < 3; ++a) dup = dup || (((s >> a) & 1) && im[a][0] == im[a][1]);
            const int ga = G / 9 - 1, gb = (G / 3) % 3 - 1, gc = G % 3 - 1, g2 = ga * ga + gb * gb + gc * gc;
            if (dup || (shells == 1 && g2 != 0)) continue;
            const double qa = (double)im[0][s & 1] / L + ga, qb = (double)im[1][(s >> 1) & 1] / L + gb,
                         qc = (double)im[2][s >> 2] / L + gc;
            acc += exp(-(double)g2) * 4.0 * kPi / (qa * qa + qb * qb + qc * qc + kappa * kappa);
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((tid & 31) == 0) hq = acc / nimg;
    } else if (exchange_on) {
        for (int i = tid - 96; i < 2 * 26 * t; i += PTHR - 96) {
            const int s = i / (26 * t), e = i - s * 26 * t;
            double2 m = mu[e];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                m = cadd(m, cadd(cscale(mu[(size_t)(1 + 2 * a) * 26 * t + e], cs[s][a]),
                                 cscale(mu[(size_t)(2 + 2 * a) * 26 * t + e], sn[s][a])));
            M[i] = m;
        }
    }
    __syncthreads();
    if (exchange_on)
        for (int s = 0; s < 2; ++s)
            rotate_forms<true>(M + s * 26 * t, U + s * g, U + s * g + rv, fw, M + s * 26 * t, 26, nv, nc, tid, PTHR,
                               [] { __syncthreads(); });
    for (int e = tid; e < g; e += PTHR) {
        const bool val = e < rv;
        const int q = val ? e : e - rv, nb = val ? nv : nc, a = q / nb, b = q - a * nb;
        const double2 *u0 = U + (val ? 0 : rv), *u1 = U + g + (val ? 0 : rv);
        double2 o = make_double2(0.0, 0.0);
        for (int m = 0; m < nb; ++m)
            o = cadd(o, val ? cmulc(u1[m * nb + b], u0[m * nb + a]) : cmulc(u0[m * nb + a], u1[m * nb + b]));
        O[e] = o;
    }
    // overlaps with the corners, both points
    for (int i = tid; i < 16 * g; i += PTHR) {
        const int s = i / (8 * g), l = (i / g) & 7, e = i % g;
        const bool val = e < rv;
        const int q = val ? e : e - rv, nb = val ? nv : nc;
        if (Dv) {
            const size_t kd = (size_t)cell[s] * Ndiv + js[s];
            const double2 v = val ? to_d2(Dv[(kd * 8 + l) * rv + q]) : to_d2(Dc[(kd * 8 + l) * rc + q]);
            dd[i] = make_float2((float)v.x, (float)v.y);
        } else {
            const Int3 ci = unflat3(cell[s], n);
            const int cc = flat3(ci.a + ((l >> 2) & 1), ci.b + ((l >> 1) & 1), ci.c + (l & 1), n), np = q / nb, b = q - np * nb;
            const double2 *cu = (val ? Uvc : Ucc) + (size_t)cc * nb * nb, *u = U + s * g + (val ? 0 : rv);
            double2 v = make_double2(0.0, 0.0);
            for (int m = 0; m < nb; ++m) v = cadd(v, cmulc(cu[m * nb + np], u[m * nb + b]));
            dd[i] = make_float2((float)v.x, (float)v.y);
        }
    }
    for (int e = tid; e < t * t; e += PTHR) K1[e] = make_float2(0.f, 0.f);
    const Int3 c0 = unflat3(cell[0], n), c1 = unflat3(cell[1], n);
    const int rows = t * nv;                                    // (row of the block, n3)
    for (int l = 0; l < 8; ++l) {
        const float fa = interp_weight_f(js[0], l, nd, nb1);
        if (fa == 0.f) continue;
        const int ca = flat3(c0.a + ((l >> 2) & 1), c0.b + ((l >> 1) & 1), c0.c + (l & 1), n);
        __syncthreads();
        // K_c(ca, cb) for the active corners of k', and its product with d_c over n4
        for (int i = tid; i < 8 * t * t; i += PTHR) {
            const int lp = i / (t * t), e = i - lp * t * t;
            if (!interp_active(js[1], lp, nd, nb1)) continue;
            const int cb = flat3(c1.a + ((lp >> 2) & 1), c1.b + ((lp >> 1) & 1), c1.c + (lp & 1), n);
            const double2 v = to_d2(Kc[(size_t)(ca * t + e / t) * Nc + cb * t + e % t]);
            Kb[i] = make_float2((float)v.x, (float)v.y);
        }
        __syncthreads();
        for (int i = tid; i < 8 * rows; i += PTHR) {
            const int lp = i / rows;
            if (!interp_active(js[1], lp, nd, nb1)) continue;
            float2* x = Kb + (size_t)i * nc;
            const float2* d = dd + (8 + lp) * g + rv;
            float2 in[BSE_MAX_BANDS];
#pragma unroll
            for (int q = 0; q < BSE_MAX_BANDS; ++q) if (q < nc) in[q] = x[q];
            for (int c = 0; c < nc; ++c) {
                float2 s = make_float2(0.f, 0.f);
#pragma unroll
                for (int q = 0; q < BSE_MAX_BANDS; ++q) if (q < nc) s = cadd(s, cmul(in[q], d[q * nc + c]));
                x[c] = s;
            }
        }
        __syncthreads();
        // over n3 and the corners: Ts[r][v2][c2] = sum f' conj(d_v[n3][v2]) Kb[l'][r][n3][c2]
        for (int i = tid; i < t * t; i += PTHR) {
            const int r = i / t, e = i - r * t, v2 = e / nc, c2 = e - v2 * nc;
            float2 s = make_float2(0.f, 0.f);
            for (int lp = 0; lp < 8; ++lp) {
                const float fb = interp_weight_f(js[1], lp, nd, nb1);
                if (fb == 0.f) continue;
                const float2 *d = dd + (8 + lp) * g + v2, *x = Kb + ((size_t)lp * t + r) * t + c2;
                float2 u = make_float2(0.f, 0.f);
                for (int m = 0; m < nv; ++m) u = cadd(u, cmulc(d[m * nv], x[m * nc]));
                s.x = fmaf(fb, u.x, s.x);
                s.y = fmaf(fb, u.y, s.y);
            }
            Ts[i] = s;
        }
        __syncthreads();
        // F(k, l) on the left: n2 with conj(d_c), then n1 with d_v
        float2* Tw = Kb;
        for (int i = tid; i < t * t; i += PTHR) {
            const int r = i / t, col = i - r * t, m = r / nc, c = r - m * nc;
            const float2* d = dd + l * g + rv + c;
            float2 s = make_float2(0.f, 0.f);
            for (int q = 0; q < nc; ++q) s = cadd(s, cmulc(d[q * nc], Ts[(m * nc + q) * t + col]));
            Tw[i] = s;
        }
        __syncthreads();
        for (int i = tid; i < t * t; i += PTHR) {
            const int r = i / t, col = i - r * t, v = r / nc, c = r - v * nc;
            const float2* d = dd + l * g + v;
            float2 s = make_float2(0.f, 0.f);
            for (int m = 0; m < nv; ++m) s = cadd(s, cmul(d[m * nv], Tw[(m * nc + c) * t + col]));
            K1[i].x = fmaf(fa, s.x, K1[i].x);
            K1[i].y = fmaf(fa, s.y, K1[i].y);
        }
    }
    __syncthreads();
    // explicit elements and targets
    for (int i = tid; i < t * t; i += PTHR) {
        const int e1 = i / t, e2 = i - e1 * t, v = e1 / nc, c = e1 - v * nc, v2 = e2 / nc, c2 = e2 - v2 * nc;
        double2 ex = make_double2(0.0, 0.0);
        if (exchange_on)
            for (int G = 0; G < 26; ++G) {
                const int q = G + (G >= 13 ? 1 : 0), ga = q / 9 - 1, gb = (q / 3) % 3 - 1, gc = q % 3 - 1;
                const int g2 = ga * ga + gb * gb + gc * gc;
                ex = cadd(ex, cscale(cmulc(M[G * t + e1], M[(26 + G) * t + e2]), g2 == 1 ? 4.0 * kPi : (g2 == 2 ? 4.0 * kPi / 2 : 4.0 * kPi / 3)));
            }
        const double2 kx = cscale(csub(cscale(ex, 2.0), cscale(cmul(O[v * nv + v2], O[rv + c * nc + c2]), hq * inv_eps)), e_k / nk);
        const double2 km1 = cscale(make_double2(K1[i].x, K1[i].y), 1.0 / Ndiv);
        const size_t row = (size_t)blk * t * t + i;
        // one real at a time: the caller's Y need not lie on 8 bytes
        Y[2 * row] = (float)((kx.x - km1.x) * nk);
        Y[2 * row + 1] = (float)((kx.y - km1.y) * nk);
    }
    // features
    double q[4] = {0.0, 0.0, 0.0, 0.0};
    for (int a = 0; a < 3; ++a) {
        int d = imod(gi[0][a] - gi[1][a], L);
        if (2 * d >= L) d -= L;
        q[a] = (double)d / L;
        q[3] += q[a] * q[a];
    }
    const float qf[4] = {(float)q[0], (float)q[1], (float)q[2], (float)sqrt(q[3])};
    const size_t k1 = ((size_t)cell[0] * Ndiv + js[0]) * t, k2 = ((size_t)cell[1] * Ndiv + js[1]) * t;
    float* x = X + (size_t)blk * t * t * d_in;
    const float inv_d = 1.f / (float)d_in, inv_t = 1.f / (float)t;
    for (int i = tid; i < t * t * d_in; i += PTHR) {
        // i < 24^2 54: the quotients are at least 1/108 from the next integer, FP32 is exact enough below 2^16
        const int r = (int)(((float)i + 0.5f) * inv_d), e = i - r * d_in, e1 = (int)(((float)r + 0.5f) * inv_t), e2 = r - e1 * t;
        float v = 0.f;
        if (e < 4) v = e == 0 ? qf[0] : (e == 1 ? qf[1] : (e == 2 ? qf[2] : qf[3]));
        else if (e == 4 + e1 || e == 4 + t + e2) v = 1.f;
        else if (e == 4 + 2 * t) v = (float)dE[k1 + e1];
        else if (e == 5 + 2 * t) v = (float)dE[k2 + e2];
        x[i] = v;
    }
}

}  // namespace

// ========================================== learned correction (stencil conv)
namespace {

// features of every (near offset, vc, v'c') with dE at its zone average
__global__ void k_stencil_features(const int* __restrict__ offs, int noff, int L, int t, const float* __restrict__ dEavg,
                                   int d_in, float* __restrict__ X) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)noff * t * t) return;
    const int o = (int)(i / (t * t)), e1 = (int)((i / t) % t), e2 = (int)(i % t);
    float* x = X + i * d_in;
    for (int k = 0; k < d_in; ++k) x[k] = 0.f;
    float qq = 0.f;
    for (int a = 0; a < 3; ++a) {
        const float q = (float)offs[3 * o + a] / L;
        x[a] = q;
        qq += q * q;
    }
    x[3] = sqrtf(qq);
    x[4 + e1] = 1.f;
    x[4 + t + e2] = 1.f;
    x[4 + 2 * t] = dEavg[e1];
    x[5 + 2 * t] = dEavg[e2];
}

// zone average of dE per transition (fixed order)
template <typename T>
__global__ void k_dE_avg(const T* __restrict__ dE, int nk, int t, float* __restrict__ out) {
    __shared__ double sh[256];
    const int tr = blockIdx.x;
    double s = 0.0;
    for (int k = threadIdx.x; k < nk; k += 256) s += (double)dE[(size_t)k * t + tr];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if (threadIdx.x < st) sh[threadIdx.x] += sh[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[tr] = (float)(sh[0] / nk);
}

// T(delta) = (out(delta) + conj(out(-delta))^T) / (2 N_k), scattered onto the
// periodic grid kernel ker[e1][e2][x][y][z].
// swap: channel e2 t + e1 (bse_lconv.cu) instead of e1 t + e2.
__global__ void k_stencil_scatter(const float* __restrict__ out, const int* __restrict__ offs, const int* __restrict__ neg,
                                  int noff, int L, int t, float inv_nk, int swap, float2* __restrict__ ker) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)noff * t * t) return;
    const int o = (int)(i / (t * t)), e1 = (int)((i / t) % t), e2 = (int)(i % t);
    const long long j = ((long long)neg[o] * t + e2) * t + e1;
    const float re = 0.5f * (out[2 * i] + out[2 * j]) * inv_nk;
    const float im = 0.5f * (out[2 * i + 1] - out[2 * j + 1]) * inv_nk;
    const int x = imod(offs[3 * o], L), y = imod(offs[3 * o + 1], L), z = imod(offs[3 * o + 2], L);
    const size_t chan = swap ? (size_t)e2 * t + e1 : (size_t)e1 * t + e2;
    ker[(chan * L + x) * L * L + (size_t)y * L + z] = make_float2(re, im);
}

// One axis of a separable DFT on [chan][L][L][L]: out_j = sum_n in_n w^{j n},
// w = exp(sign 2 pi i / L) taken from the table tw [L].
__global__ void k_dft_axis(const float2* __restrict__ in, float2* __restrict__ out, int L, long long nchan, int axis,
                           const float2* __restrict__ tw) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long L3 = (long long)L * L * L;
    if (i >= nchan * L3) return;
    const long long ch = i / L3;
    const int r = (int)(i % L3);
    const int x = r / (L * L), y = (r / L) % L, z = r % L;
    const int j = axis == 0 ? x : (axis == 1 ? y : z);
    const long long stride = axis == 0 ? (long long)L * L : (axis == 1 ? L : 1);
    const long long base = ch * L3 + r - (long long)j * stride;
    float2 acc = make_float2(0.f, 0.f);
    int ph = 0;
    for (int nn = 0; nn < L; ++nn) {
        acc = cadd(acc, cmul(in[base + nn * stride], tw[ph]));
        ph += j;
        if (ph >= L) ph -= L;
    }
    out[i] = acc;
}

// psi [chain][kd t + tr] -> grid [chain][tr][x][y][z]
template <typename T>
__global__ void k_to_grid(const typename Cx<T>::V* __restrict__ psi, int nchains, int n, int nd, int t,
                          float2* __restrict__ grid) {
    const int nk = n * n * n * nd * nd * nd, Ndiv = nd * nd * nd, L = n * nd;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)nchains * nk * t) return;
    const int ch = (int)(i / ((long long)nk * t)), rem = (int)(i % ((long long)nk * t));
    const int kd = rem / t, tr = rem % t;
    const Int3 ci = unflat3(kd / Ndiv, n), j = unflat3(kd % Ndiv, nd);
    const int x = ci.a * nd + j.a, y = ci.b * nd + j.b, z = ci.c * nd + j.c;
    const double2 v = to_d2(psi[i]);
    grid[(((size_t)ch * t + tr) * L + x) * L * L + (size_t)y * L + z] = make_float2((float)v.x, (float)v.y);
}

// per frequency: out[ch][e1][xi] = sum_e2 That[e1][e2][xi] in[ch][e2][xi]; one
// thread per (e1, xi) serves every chain, so That is read once.
__global__ void __launch_bounds__(256) k_freq_mul(const float2* __restrict__ That, const float2* __restrict__ in,
                                                  int nchains, int t, int L3, float2* __restrict__ out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)t * L3) return;
    const int e1 = (int)(i / L3), xi = (int)(i % L3);
    float2 acc[BSE_MAX_CHAINS];
#pragma unroll
    for (int ch = 0; ch < BSE_MAX_CHAINS; ++ch) acc[ch] = make_float2(0.f, 0.f);
    for (int e2 = 0; e2 < t; ++e2) {
        const float2 T = That[((size_t)e1 * t + e2) * L3 + xi];
#pragma unroll
        for (int ch = 0; ch < BSE_MAX_CHAINS; ++ch)
            if (ch < nchains) acc[ch] = cadd(acc[ch], cmul(T, in[((size_t)ch * t + e2) * L3 + xi]));
    }
#pragma unroll
    for (int ch = 0; ch < BSE_MAX_CHAINS; ++ch)
        if (ch < nchains) out[((size_t)ch * t + e1) * L3 + xi] = acc[ch];
}

// One axis of the separable DFT, in place, on [chan][L][L][L] (L <= 64): a CTA
// stages 32 lines along `axis` in shared memory (loads and stores coalesced),
// and warp w computes outputs w, w + 8, ... of line `lane`:
// out_k = sum_n in_n w^{k n} with w^j = tw[j], in two stages (below).
__global__ void __launch_bounds__(256) k_dft_tile(float2* __restrict__ a, int L, long long nlines, int axis,
                                                  const float2* __restrict__ tw_g) {
    extern __shared__ float2 dsm[];
    const int P = (L & 1) ? L + 2 : L + 1;              // odd row pitch: conflict-free 8-byte rows
    float2* tw = dsm;
    float2* din = tw + 64;
    float2* dout = din + 32 * P;
    const long long L2 = (long long)L * L, L3 = L2 * L;
    const long long g0 = (long long)blockIdx.x * 32;
    for (int j = threadIdx.x; j < L; j += blockDim.x) tw[j] = tw_g[j];
    // line g = (ch L + u) L + v; element n of it at base + n * stride
    auto base = [&](long long g) -> long long {
        const long long ch = g / L2;
        const int u = (int)((g / L) % L), v = (int)(g % L);
        if (axis == 0) return ch * L3 + (long long)u * L + v;
        if (axis == 1) return ch * L3 + (long long)u * L2 + v;
        return ch * L3 + (long long)u * L2 + (long long)v * L;
    };
    const long long stride = axis == 0 ? L2 : (axis == 1 ? L : 1);
    const int n_el = 32 * L;
    for (int i = threadIdx.x; i < n_el; i += blockDim.x) {
        const int l = axis == 2 ? i / L : i % 32, n = axis == 2 ? i % L : i / 32;
        const long long g = g0 + l;
        if (g < nlines) din[l * P + n] = a[base(g) + n * stride];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Two-stage Cooley-Tukey with L = A B (A the largest divisor <= sqrt L):
    // n = B n1 + n2, k = k1 + A k2,
    //   Y[n2][k1] = w^{n2 k1} sum_{n1} x[B n1 + n2] w^{B n1 k1}      (stage 1, into dout)
    //   X[k1 + A k2] = sum_{n2} Y[n2][k1] w^{A n2 k2}                 (stage 2, into din)
    // with every power of w read from the table (index mod L).
    int A = 1;
    for (int d = 2; d * d <= L; ++d)
        if (L % d == 0) A = d;
    const int B = L / A;
    for (int q = warp; q < L; q += 8) {
        const int n2 = q / A, k1 = q - n2 * A;
        float2 acc = make_float2(0.f, 0.f);
        int ph = 0;
        const int dph = (B * k1) % L;
        for (int n1 = 0; n1 < A; ++n1) {
            acc = cadd(acc, cmul(din[lane * P + B * n1 + n2], tw[ph]));
            ph += dph;
            if (ph >= L) ph -= L;
        }
        dout[lane * P + q] = cmul(acc, tw[(n2 * k1) % L]);
    }
    __syncthreads();
    for (int k = warp; k < L; k += 8) {
        const int k2 = k / A, k1 = k - k2 * A;
        float2 acc = make_float2(0.f, 0.f);
        int ph = 0;
        const int dph = (A * k2) % L;
        for (int n2 = 0; n2 < B; ++n2) {
            acc = cadd(acc, cmul(dout[lane * P + n2 * A + k1], tw[ph]));
            ph += dph;
            if (ph >= L) ph -= L;
        }
        din[lane * P + k] = acc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n_el; i += blockDim.x) {
        const int l = axis == 2 ? i / L : i % 32, n = axis == 2 ? i % L : i / 32;
        const long long g = g0 + l;
        if (g < nlines) a[base(g) + n * stride] = din[l * P + n];
    }
}

// w[ch][kd t + tr] += grid[ch][tr][g(kd)] / L^3, and block partials of <psi, w>
template <typename T>
__global__ void __launch_bounds__(BSE_VEC_THREADS) k_add_learned(const float2* __restrict__ grid, const typename Cx<T>::V* __restrict__ psi,
                                                                 typename Cx<T>::V* __restrict__ w, int nchains, int n, int nd, int t,
                                                                 float scale, double2* __restrict__ part) {
    using V = typename Cx<T>::V;
    __shared__ double2 red[BSE_MAX_CHAINS][BSE_VEC_THREADS];
    const int nk = n * n * n * nd * nd * nd, Ndiv = nd * nd * nd, L = n * nd;
    const long long N = (long long)nk * t;
    double2 dot[BSE_MAX_CHAINS];
    float2 dotf[BSE_MAX_CHAINS];
    for (int c = 0; c < BSE_MAX_CHAINS; ++c) {
        dot[c] = make_double2(0.0, 0.0);
        dotf[c] = make_float2(0.f, 0.f);
    }
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        const int kd = (int)(i / t), tr = (int)(i % t);
        const Int3 ci = unflat3(kd / Ndiv, n), j = unflat3(kd % Ndiv, nd);
        const int x = ci.a * nd + j.a, y = ci.b * nd + j.b, z = ci.c * nd + j.c;
        for (int ch = 0; ch < nchains; ++ch) {
            const float2 gv = grid[(((size_t)ch * t + tr) * L + x) * L * L + (size_t)y * L + z];
            if constexpr (std::is_same<T, float>::value) {
                // FP32 vectors: the update and this thread's products in FP32 (FP64 is slow per
                // element on GB300); the sums over threads below stay FP64
                const float2 wv = w[(size_t)ch * N + i];
                const float2 nw = make_float2(fmaf(gv.x, scale, wv.x), fmaf(gv.y, scale, wv.y));
                w[(size_t)ch * N + i] = nw;
                const float2 p = psi[(size_t)ch * N + i];
                for (int c = 0; c < BSE_MAX_CHAINS; ++c)
                    if (c == ch) {
                        dotf[c].x = fmaf(p.x, nw.x, fmaf(p.y, nw.y, dotf[c].x));
                        dotf[c].y = fmaf(p.x, nw.y, fmaf(-p.y, nw.x, dotf[c].y));
                    }
            } else {
                const double2 wv = to_d2(w[(size_t)ch * N + i]);
                const V nw = from_d2<V>(make_double2(wv.x + (double)gv.x * scale, wv.y + (double)gv.y * scale));
                w[(size_t)ch * N + i] = nw;
                const double2 p = to_d2(psi[(size_t)ch * N + i]), q = to_d2(nw);
                for (int c = 0; c < BSE_MAX_CHAINS; ++c)
                    if (c == ch) { dot[c].x += p.x * q.x + p.y * q.y; dot[c].y += p.x * q.y - p.y * q.x; }
            }
        }
    }
    if constexpr (std::is_same<T, float>::value)
        for (int c = 0; c < BSE_MAX_CHAINS; ++c) dot[c] = make_double2((double)dotf[c].x, (double)dotf[c].y);
    for (int c = 0; c < BSE_MAX_CHAINS; ++c) red[c][threadIdx.x] = dot[c];
    __syncthreads();
    for (int st = BSE_VEC_THREADS / 2; st > 0; st >>= 1) {
        if (threadIdx.x < st)
            for (int c = 0; c < BSE_MAX_CHAINS; ++c) red[c][threadIdx.x] = cadd(red[c][threadIdx.x], red[c][threadIdx.x + st]);
        __syncthreads();
    }
    if (threadIdx.x < nchains) part[(size_t)threadIdx.x * BSE_MAX_VEC_BLOCKS + blockIdx.x] = red[threadIdx.x][0];
}

int dft3(bse_ctx* ctx, float2* a, float2* tmp, int L, long long nchan, const float2* tw) {
    const long long tot = nchan * L * L * L;
    if (L <= 64) {
        // in place, one tile of 32 lines per CTA and axis
        const long long nlines = nchan * L * L;
        const int P = (L & 1) ? L + 2 : L + 1;
        const size_t smem = sizeof(float2) * (64 + 2 * 32 * (size_t)P);
        BSE_CUDA_TRY(ctx, bse_raise_smem(k_dft_tile, smem));
        const unsigned blocks = (unsigned)((nlines + 31) / 32);
        for (int axis = 0; axis < 3; ++axis) k_dft_tile<<<blocks, 256, smem, ctx->stream>>>(a, L, nlines, axis, tw);
        return BSE_OK;
    }
    const int blocks = (int)((tot + 255) / 256);
    k_dft_axis<<<blocks, 256, 0, ctx->stream>>>(a, tmp, L, nchan, 0, tw);
    k_dft_axis<<<blocks, 256, 0, ctx->stream>>>(tmp, a, L, nchan, 1, tw);
    k_dft_axis<<<blocks, 256, 0, ctx->stream>>>(a, tmp, L, nchan, 2, tw);
    BSE_CUDA_TRY(ctx, cudaMemcpyAsync(a, tmp, sizeof(float2) * tot, cudaMemcpyDeviceToDevice, ctx->stream));
    return BSE_OK;
}

}  // namespace

// Learned term for nchains vectors: w += T * psi (periodic convolution via
// separable DFTs), with the <psi, w> partials recomputed.
int bse_apply_learned(bse_ctx* ctx, const bse_interp* s, int nchains, const void* psi, void* w, double2* dot) {
    if (s->learned_fused) return bse_lconv_apply(ctx, s, nchains, psi, w, dot);
    const int L = s->n * s->nd, t = s->t;
    const long long L3 = (long long)L * L * L;
    const long long nchan = (long long)nchains * t;
    float2* g = s->d_lgrid;
    float2* tmp = s->d_lgrid + (size_t)BSE_MAX_CHAINS * t * L3;
    const long long tot = (long long)nchains * s->nk * t;
    if (s->vec_prec == BSE_PREC_F64)
        k_to_grid<double><<<(int)((tot + 255) / 256), 256, 0, ctx->stream>>>((const double2*)psi, nchains, s->n, s->nd, t, g);
    else
        k_to_grid<float><<<(int)((tot + 255) / 256), 256, 0, ctx->stream>>>((const float2*)psi, nchains, s->n, s->nd, t, g);
    int rc = dft3(ctx, g, tmp, L, nchan, s->d_tw_fwd);
    if (rc != BSE_OK) return rc;
    k_freq_mul<<<(int)(((long long)t * L3 + 255) / 256), 256, 0, ctx->stream>>>(s->d_lker, g, nchains, t, (int)L3, tmp);
    rc = dft3(ctx, tmp, g, L, nchan, s->d_tw_inv);
    if (rc != BSE_OK) return rc;
    const int nb = (int)std::min<long long>(std::max<long long>((s->N + BSE_VEC_THREADS - 1) / BSE_VEC_THREADS, 1), BSE_MAX_VEC_BLOCKS);
    const float scale = 1.f / (float)L3;
    if (s->vec_prec == BSE_PREC_F64)
        k_add_learned<double><<<nb, BSE_VEC_THREADS, 0, ctx->stream>>>(tmp, (const double2*)psi, (double2*)w, nchains, s->n,
                                                                      s->nd, t, scale, dot);
    else
        k_add_learned<float><<<nb, BSE_VEC_THREADS, 0, ctx->stream>>>(tmp, (const float2*)psi, (float2*)w, nchains, s->n,
                                                                     s->nd, t, scale, dot);
    return BSE_OK;
}

// ================================================================ C ABI
extern "C" {

int bse_mlp_param_count(int d_in) { return d_in >= 1 ? nparams_for(d_in) : BSE_ERR_ARG; }

int bse_mlp_create(bse_ctx* ctx, int d_in, int max_batch, const float* init_params, bse_mlp** out) {
    if (!ctx || !out || !init_params) return BSE_ERR_ARG;
    *out = nullptr;
    if (d_in < 1 || d_in > 4096 || max_batch < 1 || max_batch > (1 << 22)) {
        ctx->err = "d_in must be in 1..4096 and max_batch in 1..2^22";
        return BSE_ERR_ARG;
    }
    const int np = nparams_for(d_in);
    for (int i = 0; i < np; ++i)
        if (!std::isfinite(init_params[i])) { ctx->err = "non-finite initial parameter"; return BSE_ERR_ARG; }
    if (cudaSetDevice(ctx->device) != cudaSuccess) return BSE_ERR_CUDA;
    bse_mlp* m = new bse_mlp();
    m->d_in = d_in;
    m->nparams = np;
    m->max_batch = max_batch;
    m->blocks = std::min((max_batch + RT - 1) / RT, std::max(ctx->sm_count, 1));
    int rc = BSE_OK;
    auto A = [&](void** p, size_t bytes, const char* what) { if (rc == BSE_OK) rc = bse_alloc(ctx, p, bytes, what); };
    A((void**)&m->d_p, sizeof(float) * np, "MLP parameters");
    A((void**)&m->d_g, sizeof(float) * np, "MLP gradients");
    A((void**)&m->d_m, sizeof(float) * np, "Adam m");
    A((void**)&m->d_v, sizeof(float) * np, "Adam v");
    A((void**)&m->d_w, sizeof(__nv_bfloat16) * np, "BF16 weights");
    A((void**)&m->d_gpart, sizeof(float) * (size_t)m->blocks * np, "gradient shares");
    A((void**)&m->d_part, sizeof(double) * m->blocks, "loss partials");
    if (rc != BSE_OK) { free_mlp(m); return rc; }
    bse_upload(ctx, m->d_p, init_params, sizeof(float) * np);
    cudaMemsetAsync(m->d_m, 0, sizeof(float) * np, ctx->stream);
    cudaMemsetAsync(m->d_v, 0, sizeof(float) * np, ctx->stream);
    k_to_bf16<<<(np + 255) / 256, 256, 0, ctx->stream>>>(m->d_p, np, m->d_w);
    if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) { free_mlp(m); ctx->err = "MLP set-up failed"; return BSE_ERR_CUDA; }
    *out = m;
    return BSE_OK;
}

void bse_mlp_free(bse_mlp* m) { free_mlp(m); }

int bse_mlp_get_params(bse_ctx* ctx, const bse_mlp* m, float* host) {
    if (!ctx || !m || !host) return BSE_ERR_ARG;
    BSE_CUDA_TRY(ctx, bse_download(ctx, host, m->d_p, sizeof(float) * m->nparams));
    return BSE_OK;
}

int bse_mlp_forward(bse_ctx* ctx, bse_mlp* m, int batch, const float* X, float* out) {
    if (!ctx || !m || !X || !out) return BSE_ERR_ARG;
    if (batch < 1 || batch > m->max_batch) { ctx->err = "batch outside 1..max_batch"; return BSE_ERR_ARG; }
    int rc = mlp_forward(ctx, m, batch, X, out);
    if (rc != BSE_OK) return rc;
    BSE_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    return BSE_OK;
}

int bse_mlp_gradients(bse_ctx* ctx, bse_mlp* m, int batch, const float* X, const float* Y, float* grad_host, double* loss) {
    if (!ctx || !m || !X || !Y || !grad_host) return BSE_ERR_ARG;
    if (batch < 1 || batch > m->max_batch) { ctx->err = "batch outside 1..max_batch"; return BSE_ERR_ARG; }
    return mlp_grads(ctx, m, batch, X, Y, loss, grad_host);
}

int bse_mlp_train_step(bse_ctx* ctx, bse_mlp* m, int batch, const float* X, const float* Y, float lr, double* loss) {
    if (!ctx || !m || !X || !Y) return BSE_ERR_ARG;
    if (batch < 1 || batch > m->max_batch || !(lr > 0.f)) { ctx->err = "bad batch or learning rate"; return BSE_ERR_ARG; }
    int rc = mlp_grads(ctx, m, batch, X, Y, loss, nullptr);
    if (rc != BSE_OK) return rc;
    m->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)m->step), c2 = 1.f - powf(b2, (float)m->step);
    k_adam<<<(m->nparams + 255) / 256, 256, 0, ctx->stream>>>(m->d_p, m->d_g, m->d_m, m->d_v, m->nparams, lr, b1, b2, 1e-8f,
                                                              c1, c2, m->d_w);
    BSE_CUDA_TRY(ctx, cudaGetLastError());
    return BSE_OK;
}

int bse_pairs_generate(bse_ctx* ctx, const bse_interp* s, int nblocks, const int* host_kd, const int* host_kd2, float* X,
                       float* Y) {
    if (!ctx || !s || !host_kd || !host_kd2 || !X || !Y || nblocks < 1) return BSE_ERR_ARG;
    const bse_coarse* c = s->co;
    if (c->kc_prec == BSE_PREC_BF16) { ctx->err = "pair data needs a complex128 or complex64 K_c"; return BSE_ERR_UNSUPPORTED; }
    if (s->t > 24) { ctx->err = "pair data supports t <= 24"; return BSE_ERR_UNSUPPORTED; }
    for (int i = 0; i < nblocks; ++i)
        if (host_kd[i] < 0 || host_kd[i] >= s->nk || host_kd2[i] < 0 || host_kd2[i] >= s->nk) {
            ctx->err = "dense index out of range";
            return BSE_ERR_ARG;
        }
    if (cudaSetDevice(ctx->device) != cudaSuccess) return BSE_ERR_CUDA;
    int *d1 = nullptr, *d2 = nullptr;
    int rc;
    if ((rc = bse_alloc(ctx, (void**)&d1, sizeof(int) * nblocks, "pair indices")) != BSE_OK) return rc;
    if ((rc = bse_alloc(ctx, (void**)&d2, sizeof(int) * nblocks, "pair indices")) != BSE_OK) { cudaFree(d1); return rc; }
    // the caller's arrays outlive the wait below
    cudaMemcpyAsync(d1, host_kd, sizeof(int) * nblocks, cudaMemcpyHostToDevice, ctx->stream);
    cudaMemcpyAsync(d2, host_kd2, sizeof(int) * nblocks, cudaMemcpyHostToDevice, ctx->stream);
    const int d_in = 6 + 2 * s->t;
    const size_t sm = pairs_smem(s->nv, s->nc);
    auto go = [&](auto tag) -> int {
        using T = decltype(tag);
        using V = typename Cx<T>::V;
        BSE_CUDA_TRY(ctx, bse_raise_smem(k_pairs<T>, sm, 1024));
        k_pairs<T><<<nblocks, PTHR, sm, ctx->stream>>>(d1, d2, c->d_gen_v, c->d_gen_c, c->d_mu, c->d_Uv, c->d_Uc,
                                                       (const V*)c->d_kc, (const V*)s->d_Dv, (const V*)s->d_Dc, (const T*)s->d_dE,
                                                       s->n, s->nd, s->nv, s->nc, s->nb1, c->e_k, 1.0 / c->eps_inf, c->kappa,
                                                       c->direct_shells, c->exchange_on, d_in, X, Y);
        return BSE_OK;
    };
    rc = s->vec_prec == BSE_PREC_F64 ? go(0.0) : go(0.f);
    if (rc != BSE_OK) { cudaFree(d1); cudaFree(d2); return rc; }
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    if (e == cudaSuccess) e = cudaGetLastError();
    cudaFree(d1);
    cudaFree(d2);
    if (e != cudaSuccess) { ctx->err = std::string("pair generation: ") + cudaGetErrorString(e); return BSE_ERR_CUDA; }
    return BSE_OK;
}

int bse_interp_set_learned(bse_ctx* ctx, bse_interp* s, bse_mlp* m, int radius) {
    if (!ctx || !s) return BSE_ERR_ARG;
    bse_invalidate_graph(s);                 // the captured step loop changes with the correction
    if (!m) {          // switch the learned correction off
        s->learned = 0;
        return BSE_OK;
    }
    const int t = s->t, L = s->n * s->nd;
    if (m->d_in != 6 + 2 * t) { ctx->err = "network input size does not match 6 + 2 t"; return BSE_ERR_ARG; }
    if (radius < 1 || 2 * radius > L) { ctx->err = "radius must satisfy 1 <= radius <= L/2"; return BSE_ERR_ARG; }
    if (s->scheme != BSE_SCHEME_M1) { ctx->err = "the learned correction replaces M3: set it on an M1 handle"; return BSE_ERR_ARG; }
    if (cudaSetDevice(ctx->device) != cudaSuccess) return BSE_ERR_CUDA;
    std::vector<int> offs;
    for (int a = -radius; a <= radius; ++a)
        for (int b = -radius; b <= radius; ++b)
            for (int cc = -radius; cc <= radius; ++cc)
                if (a * a + b * b + cc * cc < radius * radius) { offs.push_back(a); offs.push_back(b); offs.push_back(cc); }
    const int noff = (int)offs.size() / 3;
    std::vector<int> neg(noff);
    for (int i = 0; i < noff; ++i)
        for (int j = 0; j < noff; ++j)
            if (offs[3 * j] == -offs[3 * i] && offs[3 * j + 1] == -offs[3 * i + 1] && offs[3 * j + 2] == -offs[3 * i + 2]) {
                neg[i] = j;
                break;
            }
    const long long L3 = (long long)L * L * L;
    const long long rows = (long long)noff * t * t;
    int rc = BSE_OK;
    int *d_offs = nullptr, *d_neg = nullptr;
    float *d_X = nullptr, *d_out = nullptr, *d_avg = nullptr;
    auto A = [&](void** p, size_t bytes, const char* what) { if (rc == BSE_OK) rc = bse_alloc(ctx, p, bytes, what); };
    A((void**)&d_offs, sizeof(int) * offs.size(), "stencil offsets");
    A((void**)&d_neg, sizeof(int) * noff, "stencil offsets");
    float2* d_ktmp = nullptr;
    A((void**)&d_X, sizeof(float) * (size_t)rows * m->d_in, "stencil features");
    A((void**)&d_out, sizeof(float) * 2 * (size_t)rows, "stencil outputs");
    A((void**)&d_avg, sizeof(float) * t, "dE averages");
    A((void**)&d_ktmp, sizeof(float2) * (size_t)t * t * L3, "kernel transform scratch");
    if (!s->d_lker) A((void**)&s->d_lker, sizeof(float2) * (size_t)t * t * L3, "learned kernel");
    if (!s->d_lgrid) A((void**)&s->d_lgrid, sizeof(float2) * 2 * (size_t)BSE_MAX_CHAINS * t * L3, "learned grids");
    if (!s->d_tw_fwd) A((void**)&s->d_tw_fwd, sizeof(float2) * 2 * L, "DFT twiddles");
    auto cleanup = [&]() {
        cudaFree(d_offs); cudaFree(d_neg); cudaFree(d_X); cudaFree(d_out); cudaFree(d_avg); cudaFree(d_ktmp);
    };
    if (rc != BSE_OK) { cleanup(); return rc; }
    s->d_tw_inv = s->d_tw_fwd + L;
    std::vector<float2> tw(2 * L);
    for (int j = 0; j < L; ++j) {
        const double ang = 2.0 * kPi * j / L;
        tw[j] = make_float2((float)std::cos(ang), (float)-std::sin(ang));          // forward: exp(-2 pi i j / L)
        tw[L + j] = make_float2((float)std::cos(ang), (float)std::sin(ang));       // inverse: exp(+2 pi i j / L)
    }
    // the vectors outlive the wait below (and cudaFree in `cleanup` waits too)
    cudaMemcpyAsync(s->d_tw_fwd, tw.data(), sizeof(float2) * 2 * L, cudaMemcpyHostToDevice, ctx->stream);
    cudaMemcpyAsync(d_offs, offs.data(), sizeof(int) * offs.size(), cudaMemcpyHostToDevice, ctx->stream);
    cudaMemcpyAsync(d_neg, neg.data(), sizeof(int) * noff, cudaMemcpyHostToDevice, ctx->stream);
    if (s->vec_prec == BSE_PREC_F64) k_dE_avg<double><<<t, 256, 0, ctx->stream>>>((const double*)s->d_dE, s->nk, t, d_avg);
    else k_dE_avg<float><<<t, 256, 0, ctx->stream>>>((const float*)s->d_dE, s->nk, t, d_avg);
    // network inference over every (near offset, vc, v'c'), in chunks of max_batch rows
    k_stencil_features<<<(int)((rows + 255) / 256), 256, 0, ctx->stream>>>(d_offs, noff, L, t, d_avg, m->d_in, d_X);
    for (long long r0 = 0; r0 < rows; r0 += m->max_batch) {
        const int nb = (int)std::min<long long>(m->max_batch, rows - r0);
        if ((rc = mlp_forward(ctx, m, nb, d_X + r0 * m->d_in, d_out + 2 * r0)) != BSE_OK) { cleanup(); return rc; }
    }
    // Hermitian stencil on the periodic grid, then its DFT (one channel per band pair)
    const bool fused = bse_lconv_usable(ctx, s);
    float2* mesh = fused ? d_ktmp : s->d_lker;
    cudaMemsetAsync(mesh, 0, sizeof(float2) * (size_t)t * t * L3, ctx->stream);
    k_stencil_scatter<<<(int)((rows + 255) / 256), 256, 0, ctx->stream>>>(d_out, d_offs, d_neg, noff, L, t, 1.f / s->nk,
                                                                        fused ? 1 : 0, mesh);
    rc = fused ? bse_lconv_kernel(ctx, s, d_ktmp, s->d_lker) : dft3(ctx, s->d_lker, d_ktmp, L, (long long)t * t, s->d_tw_fwd);
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    if (e == cudaSuccess) e = cudaGetLastError();
    cleanup();
    if (rc != BSE_OK) return rc;
    if (e != cudaSuccess) { ctx->err = std::string("learned stencil: ") + cudaGetErrorString(e); return BSE_ERR_CUDA; }
    s->learned = 1;
    s->learned_fused = fused ? 1 : 0;
    s->learned_radius = radius;
    return BSE_OK;
}

}  // extern "C"
