// The FP64-accurate Dslash of the residual recomputation in double-single arithmetic (see
// ds_arith.cuh), as separate kernels for the graph and host-driven solver drivers, the
// multi-shift refinement and hisq_residual: EPI_PLAIN (ds in -> ds out) and EPI_RESID
// (r = b - m^2 x + D t with t a ds bundle, x and b FP64; FP64 epilogue and |r|^2), plus the
// conversion of FP64 bundles into ds bundles.  The persistent solver runs the same stencil as
// phases of its launch (cg_persistent.cuh).
#include "ds_arith.cuh"
#include "dslash_kernel.cuh"
#include "dslash_launch.cuh"

namespace hisq {

// FP64 bundle (double2 per complex) -> ds bundle (float4 per complex), same element order
__global__ void ds_split_kernel(const double2 *in, float4 *out, long count) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < count; i += (long)gridDim.x * blockDim.x) {
        const double2 z = in[i];
        float a, b, c, d;
        ds_split(z.x, a, b);
        ds_split(z.y, c, d);
        out[i] = make_float4(a, b, c, d);
    }
}

// canonical [n][Vh][3] complex FP64 -> ds bundle: one thread per (site, right-hand side), right-hand
// sides adjacent so that the bundle's words are written in runs
__global__ void __launch_bounds__(256) ds_split_canon_kernel(int Vh, int n, const double2 *canon, float4 *out) {
    const long total = (long)Vh * n;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
        const long s = i / n;
        const int r = (int)(i - s * n);
        const double2 *in = canon + ((long)r * Vh + s) * 3;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double2 z = in[c];
            float rh, rl, ih, il;
            ds_split(z.x, rh, rl);
            ds_split(z.y, ih, il);
            out[(s * 3 + c) * n + r] = make_float4(rh, rl, ih, il);
        }
    }
}

template <int R, int EPI>
__global__ void __launch_bounds__(256, R == 1 ? 2 : 1) dslash_ds_kernel(KArgs a) {
    extern __shared__ double red[];
    if (a.gate && *a.gate == 0) return;
    const Geom &g = a.g;
    const int tid = threadIdx.x;
    const int gi = tid % a.t;
    const int sl = tid / a.t;
    const int r0 = gi * R;
    const int nvalid = min(R, a.n - r0);
    const float4 *in = reinterpret_cast<const float4 *>(a.in);
    bool act[R];
    bool any_act = false;
#pragma unroll
    for (int r = 0; r < R; r++) {
        act[r] = (r < nvalid) && (a.active == nullptr || a.active[r0 + r] != 0);
        any_act |= act[r];
    }
    double dot[R];
#pragma unroll
    for (int r = 0; r < R; r++) dot[r] = 0.0;

    const bool whole = a.s0 == 0 && a.s1 == g.Vh;  // a whole parity: visit in plane order
    for (int tile = blockIdx.x; (long)tile * a.spb < a.s1 - a.s0; tile += gridDim.x) {
        const int q = tile * a.spb + sl;
        if (!(sl < a.spb && q < a.s1 - a.s0 && any_act)) continue;
        const int s = whole ? visit_site(g, q) : a.s0 + q;
        dscplx acc[R][3];
        int rr[R];
#pragma unroll
        for (int r = 0; r < R; r++) rr[r] = r0 + r;
        ds_site_stencil<R, false, true>(g, a.fat, a.naik, a.parity, in, a.n, s, rr, act, acc);
        if constexpr (EPI == EPI_PLAIN) {
#pragma unroll
            for (int r = 0; r < R; r++)
                if (act[r]) ds_store3(reinterpret_cast<float4 *>(a.out), a.n, s, r0 + r, acc[r]);
        } else {
            static_assert(EPI == EPI_RESID, "ds kernels have the plain and residual epilogues");
            const double2 *vx = reinterpret_cast<const double2 *>(a.axpy);
            const double2 *vb = reinterpret_cast<const double2 *>(a.b);
#pragma unroll
            for (int r = 0; r < R; r++) {
                if (!act[r]) continue;
                double d = 0.0;
                double2 w[3];
                const double m2 = a.mass2v ? a.mass2v[r0 + r] : a.mass2;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const long idx = a.canon ? ((long)(r0 + r) * g.Vh + s) * 3 + c : ((long)s * 3 + c) * a.n + r0 + r;
                    const long bidx = a.b_one ? (long)s * 3 + c : idx;
                    const double2 x = __ldg(vx + idx), b = __ldg(vb + bidx);
                    w[c].x = b.x - m2 * x.x + ds_value(acc[r][c].re());
                    w[c].y = b.y - m2 * x.y + ds_value(acc[r][c].im());
                    d += w[c].x * w[c].x + w[c].y * w[c].y;
                }
                dot[r] += d;
                const long base = (long)s * 3 * a.n + r0 + r;
                if (a.out) {
                    double2 *o = reinterpret_cast<double2 *>(a.out);
                    const long at = a.canon ? ((long)(r0 + r) * g.Vh + s) * 3 : base, step = a.canon ? 1 : a.n;
#pragma unroll
                    for (int c = 0; c < 3; c++) o[at + c * step] = w[c];
                }
                if (a.out_lo) {
                    if (a.lo_prec == HISQ_FP64) {
                        double2 *o = reinterpret_cast<double2 *>(a.out_lo);
#pragma unroll
                        for (int c = 0; c < 3; c++) o[base + (long)c * a.n] = w[c];
                    } else {
                        float2 *o = reinterpret_cast<float2 *>(a.out_lo);
#pragma unroll
                        for (int c = 0; c < 3; c++) o[base + (long)c * a.n] = make_float2((float)w[c].x, (float)w[c].y);
                    }
                }
            }
        }
    }
    if constexpr (EPI == EPI_RESID) {
        for (int i = tid; i < a.spb * a.n; i += blockDim.x) red[i] = 0.0;
        __syncthreads();
        if (sl < a.spb) {
#pragma unroll
            for (int r = 0; r < R; r++)
                if (r < nvalid) red[sl * a.n + r0 + r] = dot[r];
        }
        block_reduce_finish(red, a.spb, a.n, a.n, a.red);
    }
}

template <int R, int EPI>
static cudaError_t launch_ds_one(const KArgs &a, int threads, size_t smem, int num_sms, cudaStream_t stream,
                                 int *grid_out) {
    auto k = dslash_ds_kernel<R, EPI>;
    long tiles = (a.s1 - a.s0 + a.spb - 1) / a.spb;
    int grid = (int)balanced_grid(tiles, wave_grid(k, threads, smem, num_sms, tiles));
    if (grid_out) *grid_out = grid;
    k<<<grid, threads, smem, stream>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_dslash_ds(const KArgs &a, int epi, int R, int threads, size_t smem, int num_sms, cudaStream_t s,
                             int *grid) {
    if (epi == EPI_RESID) {
        if (R == 2) return launch_ds_one<2, EPI_RESID>(a, threads, smem, num_sms, s, grid);
        return launch_ds_one<1, EPI_RESID>(a, threads, smem, num_sms, s, grid);
    }
    if (epi != EPI_PLAIN) return cudaErrorInvalidValue;
    if (R == 2) return launch_ds_one<2, EPI_PLAIN>(a, threads, smem, num_sms, s, grid);
    return launch_ds_one<1, EPI_PLAIN>(a, threads, smem, num_sms, s, grid);
}

int split_vectors(hisq_ctx *ctx, const void *fp64_bundle, void *ds_bundle, int n, cudaStream_t st) {
    const long count = (long)ctx->geom.Vh * 3 * n;
    const int threads = 256;
    const int blocks = (int)std::min<long>((count + threads - 1) / threads, (long)ctx->num_sms * 16);
    ds_split_kernel<<<blocks, threads, 0, st>>>(reinterpret_cast<const double2 *>(fp64_bundle),
                                                reinterpret_cast<float4 *>(ds_bundle), count);
    HISQ_CUDA(cudaGetLastError());
    return HISQ_OK;
}

int split_canonical(hisq_ctx *ctx, const double *canon, void *ds_bundle, int n, cudaStream_t st) {
    const long count = (long)ctx->geom.Vh * n;
    const int blocks = (int)std::min<long>((count + 255) / 256, (long)ctx->num_sms * 16);
    ds_split_canon_kernel<<<blocks, 256, 0, st>>>(ctx->geom.Vh, n, reinterpret_cast<const double2 *>(canon),
                                                  reinterpret_cast<float4 *>(ds_bundle));
    HISQ_CUDA(cudaGetLastError());
    return HISQ_OK;
}

}  // namespace hisq

using namespace hisq;

extern "C" int hisq_residual(const hisq_links *fat, const hisq_links *naik, double mass, const double *rhs,
                             const double *x, double *r, int nrhs, double *res2) {
    hisq_ctx *ctx;
    HISQ_CHECK(require_ctx(&ctx));
    if (!fat || !naik || !rhs || !x || !r) return set_error(HISQ_ERR_ARG, "null argument");
    if (fat->ctx != ctx || naik->ctx != ctx) return set_error(HISQ_ERR_STATE, "links of another context");
    if (fat->is_naik || !naik->is_naik) return set_error(HISQ_ERR_ARG, "expected (fat, naik) links handles");
    if (fat->prec != naik->prec) return set_error(HISQ_ERR_ARG, "fat and Naik links have different precisions");
    if (nrhs < 1 || nrhs > HISQ_MAX_NRHS) return set_error(HISQ_ERR_ARG, "nrhs must be in 1..%d", HISQ_MAX_NRHS);
    const int hp = links_hp(fat);
    const int Vh = ctx->geom.Vh;
    const size_t canon = (size_t)nrhs * Vh * 6 * sizeof(double), vb = vector_bytes(HISQ_FP64, Vh, nrhs);
    const size_t max_grid = (size_t)ctx->num_sms * 64;
    cudaStream_t st = ctx->stream;
    const bool ds = hp == LINKS_DS;
    // The double-single kernels read b and x and write r in the canonical layout: caller's buffers directly
    // (16-byte aligned ones in this device's own memory), others (host, managed, another device's) through a
    // device copy.  Native FP64 goes through internal bundles and one staging buffer.
    auto direct = [&](const void *p) { return ds && on_device(p, ctx->device) && (uintptr_t)p % 16 == 0; };
    // the kernel that writes r still reads b and x: an r over part of either is written through the scratch
    auto overlap = [&](const double *p, const double *q) {
        const uintptr_t a = (uintptr_t)p, b = (uintptr_t)q;
        return a < b + canon && b < a + canon;
    };
    const bool db = direct(rhs), dx = direct(x), dr = direct(r) && !overlap(r, rhs) && !overlap(r, x);
    const size_t pbytes = max_grid * nrhs * sizeof(double);
    const size_t staging = ds ? ((db ? 0 : canon) + (dx ? 0 : canon) + (dr ? 0 : canon)) : canon;
    const size_t total = staging + (ds ? 2 : 4) * vb + pbytes + 256;
    // scratch: staging, then x (ds) and t, or b, x, t, r (FP64); partials; counter.  Kept in the context up
    // to HISQ_RESID_KEEP.  4 right-hand sides at 32^3 x 8: 707 us with an allocation per call and staging
    // copies, packs and unpacks around the two Dslash kernels, 416 without them
    char *buf = nullptr, *owned = nullptr;
    if (total <= HISQ_RESID_KEEP) {
        if (total > ctx->resid_cap) {
            if (ctx->resid) cudaFree(ctx->resid);
            ctx->resid = nullptr;
            ctx->resid_cap = 0;
            HISQ_CUDA(cudaMalloc(&ctx->resid, total));
            ctx->resid_cap = total;
        }
        buf = ctx->resid;
    } else {
        HISQ_CUDA(cudaMalloc(&owned, total));
        buf = owned;
    }
    char *at = buf;
    auto take = [&](size_t bytes) { char *p = at; at += bytes; return p; };
    int rc = HISQ_OK;
    auto cuda = [&](cudaError_t e, const char *what) {
        if (rc == HISQ_OK && e != cudaSuccess) rc = set_error(HISQ_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
    };
    const double *b_c = rhs, *x_c = x;
    double *r_c = r, *stage = nullptr;
    if (ds) {
        if (!db) {
            double *p = reinterpret_cast<double *>(take(canon));
            cuda(cudaMemcpyAsync(p, rhs, canon, cudaMemcpyDefault, st), "rhs upload");
            b_c = p;
        }
        if (!dx) {
            double *p = reinterpret_cast<double *>(take(canon));
            cuda(cudaMemcpyAsync(p, x, canon, cudaMemcpyDefault, st), "x upload");
            x_c = p;
        }
        if (!dr) r_c = reinterpret_cast<double *>(take(canon));
    } else {
        stage = reinterpret_cast<double *>(take(canon));
    }
    void *b64 = ds ? nullptr : take(vb), *xin = take(vb), *t = take(vb), *r64 = ds ? nullptr : take(vb);
    double *partials = reinterpret_cast<double *>(take(pbytes));
    unsigned int *counter = reinterpret_cast<unsigned int *>(take(256));
    cuda(cudaMemsetAsync(counter, 0, 256, st), "scratch reset");
    if (ds) {
        if (rc == HISQ_OK) rc = split_canonical(ctx, x_c, xin, nrhs, st);
    } else {
        cuda(cudaMemcpyAsync(stage, rhs, canon, cudaMemcpyDefault, st), "rhs upload");
        if (rc == HISQ_OK) rc = pack_vectors(ctx, stage, b64, nrhs, HISQ_FP64, st);
        cuda(cudaMemcpyAsync(stage, x, canon, cudaMemcpyDefault, st), "x upload");
        if (rc == HISQ_OK) rc = pack_vectors(ctx, stage, xin, nrhs, HISQ_FP64, st);
    }
    DslashArgs d;
    memset(&d, 0, sizeof(d));
    d.n = nrhs;
    d.in = xin;
    d.out = t;
    d.parity = 1;
    d.epi = EPI_PLAIN;
    if (rc == HISQ_OK) rc = launch_dslash(ctx, fat, naik, hp, d, nullptr, st);
    d.in = t;
    d.out = ds ? (void *)r_c : r64;
    d.parity = 0;
    d.epi = EPI_RESID;
    d.mass2 = mass * mass;
    d.axpy_in = ds ? (const void *)x_c : xin;
    d.b = ds ? (const void *)b_c : b64;
    d.canon = ds;
    d.partials = partials;
    d.partials_cap = max_grid * nrhs;
    d.counter = counter;
    d.dot_out = ctx->dot_out;
    if (rc == HISQ_OK) rc = launch_dslash(ctx, fat, naik, hp, d, nullptr, st);
    if (!ds) {
        if (rc == HISQ_OK) rc = unpack_vectors(ctx, r64, stage, nrhs, HISQ_FP64, st);
        cuda(cudaMemcpyAsync(r, stage, canon, cudaMemcpyDefault, st), "r download");
    } else if (!dr) {
        cuda(cudaMemcpyAsync(r, r_c, canon, cudaMemcpyDefault, st), "r download");
    }
    if (res2) cuda(cudaMemcpyAsync(res2, ctx->dot_out, sizeof(double) * nrhs, cudaMemcpyDefault, st), "dots download");
    cuda(cudaStreamSynchronize(st), "residual");
    if (owned) cudaFree(owned);
    return rc;
}
