// bse_apply_h_noalloc: one application of the interpolated H that allocates no
// device memory.
//
// Who needs it: callers that must not call cudaMalloc during their work, for
// example a host framework that owns all device memory through its own pool
// (a cudaMalloc behind its back can fail or fragment it), or a real-time
// loop in which cudaMalloc's implicit device-wide synchronisation is not
// allowed.  bse_apply_h takes its per-call scratch from the handle, which
// bse_interp_setup allocated; this variant takes it from the file-scope
// array below instead, so after set-up nothing is allocated on any path and the
// call may run beside another one on the same handle.  On the common-basis path
// the intermediate vectors lie where the general path has its pieces (reserved on
// both), or behind the rest.  Near the array's end they may fit in neither (Method 3
// with up to three transitions, in columns of 32; Method 1 with a large coarse mesh):
// set-up then allocates them.
//
// The array is a static __device__ object of the library's device module: a
// device holds BSE_NOALLOC_SCRATCH_BYTES of it from the moment that module is
// loaded on it until the process exits.  With CUDA's lazy module loading the
// module loads on first use, and that load allocates; so bse_ctx_create calls
// bse_noalloc_prepare, which looks up the array's device address
// (cudaGetSymbolAddress, which loads the module) once per device, with that
// device current, at set-up.  In host code the array's name is only a
// host-side stand-in for the device object; the address found here is what
// the kernels get.  Create the context before any stream capture.
// Every call shares the one array, which keeps the previous call's contents:
// the buffers that must start at zero are cleared on each call, and calls
// that overlap on the GPU (two streams, or two host threads) race on it.
#include <mutex>

#include "bse_internal.cuh"

#define BSE_NOALLOC_SCRATCH_BYTES (32u << 20)   // 32 MiB
#define BSE_NOALLOC_MAX_DEVICES 64

static __device__ __align__(256) unsigned char g_noalloc_scratch[BSE_NOALLOC_SCRATCH_BYTES];

namespace {

void* g_scratch_addr[BSE_NOALLOC_MAX_DEVICES] = {};
std::mutex g_scratch_mu;

size_t align256(size_t b) { return (b + 255) / 256 * 256; }

// Per-call buffers (each 256-byte aligned) of an application to nvec vectors.
struct Layout {
    size_t Q, R, X, U, D, B = 0, P = 0, total = 0;        // total: what counts towards the array's size
    size_t work = 0;                                       // common-basis path: its intermediate vectors,
    bool work_fits = true;                                 // where the array has room for them
};
Layout layout(const bse_interp* s, int nvec) {
    const bse_coarse* c = s->co;
    const size_t vsz = (s->vec_prec == BSE_PREC_F64) ? sizeof(double2) : sizeof(float2);
    const bool m3 = s->scheme == BSE_SCHEME_M3, bf16 = c->kc_prec == BSE_PREC_BF16;
    Layout l;
    auto take = [&](size_t bytes) {
        const size_t o = l.total;
        l.total += align256(bytes);
        return o;
    };
    l.Q = take(vsz * nvec * c->Nc);
    l.R = take(vsz * nvec * c->Nc);
    l.X = take(m3 ? vsz * nvec * (size_t)s->nk * 8 * s->t : 0);
    l.U = take(m3 ? vsz * nvec * (size_t)s->nk * 8 * s->t : 0);
    l.D = take(sizeof(double2) * nvec * BSE_MAX_VEC_BLOCKS);
    if (bf16) {
        l.B = take(sizeof(__nv_bfloat16) * 16 * (size_t)c->ldk);
        l.P = take(bse_tc_part_bytes(s));
    }
    if (s->common) {
        CommonWork w;
        const size_t need = bse_common_work(s, nvec, nullptr, &w);
        l.work = need <= l.D - l.X ? l.X : l.total;
        l.work_fits = l.work + need <= (l.work == l.X ? l.D : (size_t)BSE_NOALLOC_SCRATCH_BYTES);
    }
    return l;
}

}  // namespace

// A set of intermediate vectors for the sizes that bse_apply_h_noalloc takes and
// the array has no room for; most handles need none.
int bse_noalloc_setup(bse_ctx* ctx, bse_interp* s) {
    size_t bytes = 0;
    int most = 0;
    for (int nvec = 1; nvec <= BSE_MAX_CHAINS; ++nvec) {
        const Layout l = layout(s, nvec);
        if (l.total > BSE_NOALLOC_SCRATCH_BYTES || l.work_fits) continue;
        CommonWork w;
        bytes = bse_common_work(s, nvec, nullptr, &w);
        most = nvec;
    }
    if (!most) return BSE_OK;
    const int rc = bse_alloc(ctx, &s->d_na, bytes, "intermediate vectors of bse_apply_h_noalloc");
    if (rc == BSE_OK) bse_common_work(s, most, (unsigned char*)s->d_na, &s->cwork_na);
    return rc;
}

int bse_noalloc_prepare(bse_ctx* ctx) {
    if (ctx->device < 0 || ctx->device >= BSE_NOALLOC_MAX_DEVICES) return BSE_OK;   // the entry point refuses it
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (g_scratch_addr[ctx->device]) return BSE_OK;
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
        ctx->err = std::string("cudaGetSymbolAddress of the static scratch failed: ") + cudaGetErrorString(e);
        return BSE_ERR_CUDA;
    }
    g_scratch_addr[ctx->device] = p;
    return BSE_OK;
}

extern "C" int bse_apply_h_noalloc(bse_ctx* ctx, bse_interp* s, int nvec, const void* x, void* y) {
    if (!ctx || !s || !x || !y) return BSE_ERR_ARG;
    if (nvec < 1 || nvec > BSE_MAX_CHAINS) {
        ctx->err = "nvec must be in 1..4";
        return BSE_ERR_ARG;
    }
    if (ctx->device < 0 || ctx->device >= BSE_NOALLOC_MAX_DEVICES) {
        ctx->err = "device index above the no-allocation table";
        return BSE_ERR_UNSUPPORTED;
    }
    if (s->learned) {
        ctx->err = "the learned correction is not available without allocation (use bse_apply_h)";
        return BSE_ERR_UNSUPPORTED;
    }
    if (cudaSetDevice(ctx->device) != cudaSuccess) return BSE_ERR_CUDA;
    void* base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_scratch_mu);
        base = g_scratch_addr[ctx->device];           // looked up by bse_ctx_create
    }
    if (!base) {
        ctx->err = "the static scratch of this device was not set up (bse_ctx_create)";
        return BSE_ERR_CUDA;
    }
    const Layout l = layout(s, nvec);
    if (l.total > BSE_NOALLOC_SCRATCH_BYTES) {
        ctx->err = "bse_apply_h_noalloc needs " + std::to_string(l.total) + " bytes of scratch; the static array holds " +
                   std::to_string((size_t)BSE_NOALLOC_SCRATCH_BYTES) + " (use bse_apply_h)";
        return BSE_ERR_UNSUPPORTED;
    }
    const bool m3 = s->scheme == BSE_SCHEME_M3, bf16 = s->co->kc_prec == BSE_PREC_BF16;
    unsigned char* b = static_cast<unsigned char*>(base);
    ApplyScratch sc;
    sc.Q = b + l.Q;
    sc.R = b + l.R;
    sc.X = m3 ? b + l.X : nullptr;
    sc.U = m3 ? b + l.U : nullptr;
    sc.dot = reinterpret_cast<double2*>(b + l.D);
    sc.bop = bf16 ? reinterpret_cast<__nv_bfloat16*>(b + l.B) : nullptr;
    sc.part = bf16 ? reinterpret_cast<float*>(b + l.P) : nullptr;
    if (s->common) {
        if (l.work_fits) bse_common_work(s, nvec, b + l.work, &sc.work);
        else sc.work = s->cwork_na;
    }
    int rc = bse_apply_scratch(ctx, s, nvec, x, y, sc);
    if (rc != BSE_OK) return rc;
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        ctx->err = std::string("apply H (no allocation): ") + cudaGetErrorString(e);
        return BSE_ERR_CUDA;
    }
    int status = 0;
    BSE_CUDA_TRY(ctx, bse_download(ctx, &status, ctx->d_status, sizeof(int)));
    if (status) {
        cudaMemsetAsync(ctx->d_status, 0, sizeof(int), ctx->stream);
        ctx->err = bse_timeout_message(status);
        return BSE_ERR_TIMEOUT;
    }
    return BSE_OK;
}
