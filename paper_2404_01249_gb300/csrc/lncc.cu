// LNCC and MSE losses with their analytic gradients as operations of their
// own (the window sums run in window.cuh's kernels, which fa_register's fused
// iteration shares).
//
// LNCC (the local normalised cross-correlation cost used with
// Eq. (image-reg)): box window of width w = 2R + 1 with zero padding and
// fixed divisor n = w^3;
//   cross = S_IJ - S_I S_J / n, var_I = S_II - S_I^2 / n, var_J likewise,
//   cc = cross^2 / (var_I var_J + eps),  L = -(1/N) sum_x cc(x).
// Gradient (section "Jacobian-Free Eulerian Descent" uses the Gateaux
// derivative): with A = 2 cross / den, B = -cc var_I / den,
// C = -(A S_I + 2 B S_J) / n (and B', C' mirrored for I),
//   dL/dJ(y) = -(1/N) sum_{x in win(y)} [A(x) I(y) + 2 B(x) J(y) + C(x)].
//
// Precision: images are quantised to b-bit fixed point (b from the window,
// see lncc_image_bits) and all window sums are exact int64 sums; the
// variance / covariance numerators n S_II - S_I^2 are formed exactly in
// 128-bit integers before rounding to float.  The adjoint window sums
// quantise A, B, C to 2^-(47 - ceil(log2 n)) of their maxima and are exact
// int64 sums too; the final I SA + 2 J SB + SC is combined in float-float.
#include "ops.h"
#include "validate.h"

namespace fa {

// ------------------------------------------------------------------ kernels

__global__ void k_absmax2(const float *__restrict__ I, const float *__restrict__ J, long long N,
                          WsHeader *h) {
    __shared__ float red[32];
    float a = 0.0f, b = 0.0f;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
         i += (long long)gridDim.x * blockDim.x) {
        float vi = fabsf(I[i]), vj = fabsf(J[i]);
        if (!(vi <= 3.4e38f) || !(vj <= 3.4e38f)) status_set(&h->status, ST_NONFINITE);
        a = fmaxf(a, vi);
        b = fmaxf(b, vj);
    }
    block_max_to(&h->absmax_bits[0], a, red);
    block_max_to(&h->absmax_bits[1], b, red);
}

__global__ void k_loss_finalize(WsHeader *h, long long N, float sign, float *out) {
    unsigned long long a = h->loss_acc;
    // a < 2^63: split so both halves convert exactly
    float hi = __ull2float_rn(a >> 32), lo = __ull2float_rn(a & 0xffffffffull);
    float mean = (hi + lo * 2.3283064365386963e-10f) / (float)N;
    float L = sign * mean;
    h->loss = L;
    if (out) *out = L;
}

// MSE: per-block partial sums of (J - I)^2 in block order for a fixed-order
// final sum.
__global__ void __launch_bounds__(256) k_mse(const float *__restrict__ I,
                                             const float *__restrict__ J,
                                             const float *__restrict__ grad, float *dJ, float *dI,
                                             float *g, float *partials, int D, int H, int W,
                                             int P) {
    __shared__ float red[8];
    int x = blockIdx.x * 32 + threadIdx.x;
    int y = blockIdx.y * 8 + threadIdx.y;
    int z = blockIdx.z;
    const long long N = (long long)D * H * P;  // rows of P elements
    float e2 = 0.0f;
    if (x < W && y < H) {
        const long long i = ((long long)z * H + y) * P + x;
        float e = J[i] - I[i];
        e2 = e * e;
        float dj = 2.0f * e / (float)((long long)D * H * W);
        if (dJ) dJ[i] = dj;
        if (dI) dI[i] = -dj;
        if (g) {
            g[i] = dj * grad[i];
            g[N + i] = dj * grad[N + i];
            g[2 * N + i] = dj * grad[2 * N + i];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, o);
    int lane = threadIdx.x + 32 * threadIdx.y;
    if ((lane & 31) == 0) red[lane >> 5] = e2;
    __syncthreads();
    if (lane == 0) {
        float s = 0.0f;
        for (int k = 0; k < 8; ++k) s += red[k];
        long long b = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        partials[b] = s;
    }
}

__global__ void k_partials_finalize(const float *partials, long long nb, long long N, WsHeader *h,
                                    float *out) {
    __shared__ float red[256];
    float s = 0.0f;
    for (long long k = threadIdx.x; k < nb; k += blockDim.x) s += partials[k];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        float L = red[0] / (float)N;
        if (!(L <= 3.4e38f)) status_set(&h->status, ST_NONFINITE);
        h->loss = L;
        if (out) *out = L;
    }
}

// ---------------------------------------------------------------- launchers

LnccBuffers lncc_carve(WsCarver &c, long long N) {
    LnccBuffers b;
    b.p0 = c.take<long long>(5 * N);
    b.p1 = c.take<long long>(5 * N);
    b.coef = c.take<float>(7 * N);
    return b;
}

size_t lncc_plain_bytes(long long N) {
    WsCarver c(nullptr, ~size_t(0));
    c.take<WsHeader>(1);
    lncc_carve(c, N);
    return c.off;
}

cudaError_t launch_header_reset(WsHeader *h, cudaStream_t s) {
    return cudaMemsetAsync(h, 0, sizeof(WsHeader), s);
}

cudaError_t launch_absmax2(const float *I, const float *J, long long N, WsHeader *h,
                           cudaStream_t s) {
    long long blocks = (N + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_absmax2<<<(unsigned)blocks, 256, 0, s>>>(I, J, N, h); note_launch();
    return cudaGetLastError();
}

cudaError_t launch_lncc_forward(const float *I, const float *J, Dims d, int window, float cc_eps,
                                bool want_coef, bool want_dI, WsHeader *h, LnccBuffers b,
                                cudaStream_t s) {
    FwdArgs a{};
    a.I = I;
    a.J = J;
    a.coef = b.coef;
    a.h = h;
    a.cc_eps = cc_eps;
    a.write_coef = want_coef;
    a.want_dI = want_dI;
    return launch_window_fwd(kFwdBoth, a, d, window, 0, s);
}

cudaError_t launch_lncc_backward(const float *I, const float *J, const float *grad, Dims d,
                                 int window, WsHeader *h, LnccBuffers b, float *dJ, float *dI,
                                 float *g, cudaStream_t s) {
    const long long N = d.N();
    GradArgs a{};
    a.coef = b.coef;
    a.h = h;
    // dL/dI reads the images after dL/dJ and g are written: one that overlaps
    // an image waits in the scratch
    auto waits = [&](const float *out, long long n) {
        auto over = [&](const float *in) { return out < in + N && in < out + n; };
        return dI && out && (over(I) || over(J));
    };
    float *dJ1 = waits(dJ, N) ? (float *)b.p0 : dJ, *g1 = waits(g, 3 * N) ? (float *)b.p0 + N : g;
    cudaError_t e;
    if (dJ || g) {
        a.I = I;
        a.J = J;
        a.gJ = grad;
        a.g = g1;
        a.dJ = dJ1;
        if ((e = launch_window_grad(false, a, d, window, 0, s)) != cudaSuccess) return e;
    }
    if (dI) {
        a.I = J;
        a.J = I;
        a.gJ = nullptr;
        a.g = nullptr;
        a.dJ = dI;
        if ((e = launch_window_grad(true, a, d, window, 0, s)) != cudaSuccess) return e;
    }
    const size_t bytes = sizeof(float) * N;
    if (dJ1 != dJ &&
        (e = cudaMemcpyAsync(dJ, dJ1, bytes, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
        return e;
    if (g1 != g) return cudaMemcpyAsync(g, g1, 3 * bytes, cudaMemcpyDeviceToDevice, s);
    return cudaSuccess;
}

// gF = dL/dI gradI and gM = dL/dJ gradJ (three channels each).
cudaError_t launch_lncc_grads(const float *I, const float *J, const float *gradI,
                              const float *gradJ, Dims d, int window, WsHeader *h, LnccBuffers b,
                              float *gF, float *gM, cudaStream_t s) {
    GradArgs a{};
    a.coef = b.coef;
    a.h = h;
    a.I = I;
    a.J = J;
    a.gJ = gradJ;
    a.g = gM;
    cudaError_t e = launch_window_grad(false, a, d, window, 0, s);
    if (e != cudaSuccess) return e;
    a.I = J;
    a.J = I;
    a.gJ = gradI;
    a.g = gF;
    return launch_window_grad(true, a, d, window, 0, s);
}

long long mse_partials_count(Dims d) {
    VoxGrid gg(d.D, d.H, d.W);
    return (long long)gg.grid.x * gg.grid.y * gg.grid.z;
}

cudaError_t launch_mse(const float *I, const float *J, const float *grad, Dims d, WsHeader *h,
                       float *partials, float *dJ, float *dI, float *g, cudaStream_t s) {
    VoxGrid gg(d.D, d.H, d.W);
    long long nb = mse_partials_count(d);
    k_mse<<<gg.grid, gg.block, 0, s>>>(I, J, grad, dJ, dI, g, partials, d.D, d.H, d.W,
                                         d.pitch());
    note_launch();
    k_partials_finalize<<<1, 256, 0, s>>>(partials, nb, d.N(), h, nullptr); note_launch();
    return cudaGetLastError();
}

cudaError_t launch_fixed_stats(const float *I, Dims d, int window, WsHeader *h, long long *sI,
                               float *varI, cudaStream_t s) {
    FwdArgs a{};
    a.I = I;
    a.SI = sI;
    a.varI = varI;
    a.h = h;
    return launch_window_fwd(kFwdStats, a, d, window, 0, s);
}

cudaError_t launch_loss_finalize(WsHeader *h, long long N, float sign, float *loss_out,
                                 cudaStream_t s) {
    k_loss_finalize<<<1, 1, 0, s>>>(h, N, sign, loss_out); note_launch();
    return cudaGetLastError();
}

}  // namespace fa

// ---------------------------------------------------------------- C ABI

extern "C" size_t fa_lncc_workspace_size(int32_t D, int32_t H, int32_t W) {
    if (D < 1 || H < 1 || W < 1) return 0;
    return fa::lncc_plain_bytes((long long)D * H * W);
}

static fa_status loss_args(const fa_vol *fixed, const fa_vol *warped, fa_vol *dJ, fa_vol *dI,
                           void *ws, size_t ws_bytes, const char *who) {
    using namespace fa;
    FA_TRY(check_vol(fixed, "fixed", 1));
    FA_TRY(check_vol(warped, "warped", 1));
    FA_TRY(same_grid(fixed, warped, "fixed", "warped"));
    if (dJ) {
        FA_TRY(check_vol(dJ, "dL_dwarped", 1));
        FA_TRY(same_grid(fixed, dJ, "fixed", "dL_dwarped"));
    }
    if (dI) {
        FA_TRY(check_vol(dI, "dL_dfixed", 1));
        FA_TRY(same_grid(fixed, dI, "fixed", "dL_dfixed"));
    }
    FA_TRY(check_ws(ws, ws_bytes, fa_lncc_workspace_size(fixed->D, fixed->H, fixed->W), who));
    return FA_OK;
}

extern "C" fa_status fa_lncc_fwd_bwd(const fa_vol *fixed, const fa_vol *warped, int32_t window,
                                     float cc_eps, float *loss_dev, fa_vol *dL_dwarped_opt,
                                     fa_vol *dL_dfixed_opt, void *ws, size_t ws_bytes,
                                     void *stream) {
    using namespace fa;
    clear_error();
    if (window < 1 || window > 15 || (window % 2) == 0) {
        set_error("fa_lncc_fwd_bwd: window must be odd and in 1..15 (got %d)", (int)window);
        return FA_ERR_INVALID;
    }
    if (!(cc_eps >= 0.0f) || !(cc_eps < 3.0e38f)) {
        set_error("fa_lncc_fwd_bwd: cc_eps must be finite and >= 0");
        return FA_ERR_INVALID;
    }
    FA_TRY(loss_args(fixed, warped, dL_dwarped_opt, dL_dfixed_opt, ws, ws_bytes,
                     "fa_lncc_fwd_bwd"));
    cudaStream_t s = (cudaStream_t)stream;
    Dims d{fixed->D, fixed->H, fixed->W};
    long long N = d.N();
    WsCarver c(ws, ws_bytes);
    WsHeader *h = c.take<WsHeader>(1);
    LnccBuffers b = lncc_carve(c, N);
    const float *I = (const float *)fixed->data, *J = (const float *)warped->data;
    FA_CUDA_TRY(launch_header_reset(h, s));
    FA_CUDA_TRY(launch_absmax2(I, J, N, h, s));
    FA_CUDA_TRY(launch_lncc_forward(I, J, d, window, cc_eps, dL_dwarped_opt || dL_dfixed_opt,
                                    dL_dfixed_opt != nullptr, h, b, s));
    FA_CUDA_TRY(launch_loss_finalize(h, N, -1.0f, loss_dev, s));
    if (dL_dwarped_opt || dL_dfixed_opt)
        FA_CUDA_TRY(launch_lncc_backward(
            I, J, nullptr, d, window, h, b, dL_dwarped_opt ? (float *)dL_dwarped_opt->data : nullptr,
            dL_dfixed_opt ? (float *)dL_dfixed_opt->data : nullptr, nullptr, s));
    return FA_OK;
}

extern "C" fa_status fa_mse_fwd_bwd(const fa_vol *fixed, const fa_vol *warped, float *loss_dev,
                                    fa_vol *dL_dwarped_opt, fa_vol *dL_dfixed_opt, void *ws,
                                    size_t ws_bytes, void *stream) {
    using namespace fa;
    clear_error();
    FA_TRY(loss_args(fixed, warped, dL_dwarped_opt, dL_dfixed_opt, ws, ws_bytes,
                     "fa_mse_fwd_bwd"));
    cudaStream_t s = (cudaStream_t)stream;
    Dims d{fixed->D, fixed->H, fixed->W};
    WsCarver c(ws, ws_bytes);
    WsHeader *h = c.take<WsHeader>(1);
    float *partials = c.take<float>(mse_partials_count(d));
    FA_CUDA_TRY(launch_header_reset(h, s));
    FA_CUDA_TRY(launch_mse((const float *)fixed->data, (const float *)warped->data, nullptr, d, h,
                           partials,
                           dL_dwarped_opt ? (float *)dL_dwarped_opt->data : nullptr,
                           dL_dfixed_opt ? (float *)dL_dfixed_opt->data : nullptr, nullptr, s));
    if (loss_dev)
        FA_CUDA_TRY(cudaMemcpyAsync(loss_dev, &h->loss, sizeof(float), cudaMemcpyDeviceToDevice, s));
    return FA_OK;
}
