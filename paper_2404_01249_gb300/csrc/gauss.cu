// Separable Gaussian smoothing (sigma_grad / sigma_warp of the
// hyper-parameter study): taps exp(-k^2 / 2 sigma^2), |k| <= ceil(3 sigma),
// normalised to sum 1, zero padding; x, then y, then z, each tap of an axis
// added from the lowest index up.  Radii up to kOnePassRadius run as one
// z-marching kernel, wider ones as one launch per axis; both add the same
// products in the same order and give the same bits.
#include <math.h>
#include <string.h>

#include "launch.cuh"
#include "ops.h"
#include "validate.h"

namespace fa {

bool make_gauss_taps(float sigma, GaussTaps *t) {
    memset(t, 0, sizeof(*t));
    if (!(sigma >= 0.0f) || sigma > kMaxSigma) return false;
    if (sigma == 0.0f) {
        t->R = 0;
        t->w[0] = 1.0f;
        return true;
    }
    double sd = (double)sigma;
    int R = (int)ceil(3.0 * sd);
    if (2 * R + 1 > 64) return false;
    double w[64], s = 0.0;
    for (int k = -R; k <= R; ++k) {
        w[k + R] = exp(-(double)k * k / (2.0 * sd * sd));
        s += w[k + R];
    }
    t->R = R;
    for (int k = 0; k <= 2 * R; ++k) t->w[k] = (float)(w[k] / s);
    return true;
}

template <int AXIS>
__global__ void __launch_bounds__(256) k_gauss_axis(const float *__restrict__ in,
                                                    float *__restrict__ out, int C, int D, int H,
                                                    int W, int P, GaussTaps t) {
    int x = blockIdx.x * 32 + threadIdx.x;
    int y = blockIdx.y * 8 + threadIdx.y;
    int z = blockIdx.z;
    if (x >= W || y >= H) return;
    long long N = (long long)D * H * P;  // rows of P elements
    long long i = ((long long)z * H + y) * P + x;
    const int c0 = AXIS == 0 ? x : (AXIS == 1 ? y : z);
    const int n = AXIS == 0 ? W : (AXIS == 1 ? H : D);
    const long long stride = AXIS == 0 ? 1ll : (AXIS == 1 ? (long long)P : (long long)H * P);
    const int R = t.R;
    int lo = max(-R, -c0), hi = min(R, n - 1 - c0);
    for (int c = 0; c < C; ++c) {
        const float *src = in + c * N + i;
        float acc = 0.0f;
        for (int k = lo; k <= hi; ++k) acc = fmaf(t.w[k + R], __ldg(src + k * stride), acc);
        out[c * N + i] = acc;
    }
}

cudaError_t launch_gauss_axis(const float *in, float *out, int C, Dims d, const GaussTaps &t,
                              int axis, cudaStream_t s) {
    VoxGrid g(d.D, d.H, d.W);
    if (axis == 0)
        k_gauss_axis<0><<<g.grid, g.block, 0, s>>>(in, out, C, d.D, d.H, d.W, d.pitch(), t);
    else if (axis == 1)
        k_gauss_axis<1><<<g.grid, g.block, 0, s>>>(in, out, C, d.D, d.H, d.W, d.pitch(), t);
    else
        k_gauss_axis<2><<<g.grid, g.block, 0, s>>>(in, out, C, d.D, d.H, d.W, d.pitch(), t);
    note_launch();
    return cudaGetLastError();
}

// One launch for all three axes.  A CTA owns a 32 x 32 tile of one channel's
// (x, y) columns and marches a slab of output planes; warp w owns rows 4w ..
// 4w + 3, lane l column l.  Between two barriers the CTA sums plane t along x
// (shared memory to shared memory, 4 outputs per item from 16-byte reads),
// plane t - 1 along y (4 outputs of a column from 4 + 2R reads, in registers)
// and z, and stages plane t + 1, whose values were loaded a plane earlier:
// both buffers are doubled, so one barrier per plane suffices.  Along z every
// plane is added into the 2R + 1 outputs it reaches (a transposed filter: the
// partial sums of the 2R outputs still open sit in registers and shift by one
// output per plane), which keeps each output's taps in ascending order and
// needs no ring of planes.
//
// Bound: 8 bytes per value of HBM traffic (165 MB for 3 x 160 x 192 x 224,
// 24 us); measured there at R = 3: three passes 296 us, this kernel 68 us
// (2.4 TB/s, 2.2 warp instructions per clock and SM: shared-memory latency).
// Four CTAs per SM at 64 registers: 78 us.
constexpr int kOnePassRadius = 6;

template <int R>
struct GaussTile {
    static constexpr int NT = 256, TY = 32, RY = TY + 2 * R, RX = 32 + 2 * R;
    static constexpr int BX = (RX + 3) / 4 * 4;       // row length of a staged plane
    static constexpr int NM = (RY + 7) / 8;           // rows per warp (first 32 columns)
    static constexpr int NE = (RY * 2 * R + NT - 1) / NT;  // the last 2R columns
    static constexpr int ITEMS = RY * 8, NI = (ITEMS + NT - 1) / NT;
    static constexpr size_t bytes = 2 * (size_t)RY * (BX + 32) * sizeof(float);
};
template <int R>
struct OnePassTaps {
    float w[2 * R + 1];
};

template <int R>
__global__ void __launch_bounds__(256, R <= 3 ? 3 : 2) k_gauss_onepass(
    const float *__restrict__ in, float *__restrict__ out, int D, int H, int W, int TZ, int slabs,
    const __grid_constant__ OnePassTaps<R> t) {
    using G = GaussTile<R>;
    constexpr int RY = G::RY, BX = G::BX, NM = G::NM, NE = G::NE;
    extern __shared__ __align__(16) float sm[];
    // the halves of the doubled buffers: staged planes, then x sums
    constexpr int PL = RY * BX, XS = RY * 32;
    const int tid = threadIdx.x, lane = tid & 31, wy = tid >> 5;
    const int c = blockIdx.z / slabs, x0 = blockIdx.x * 32, y0 = blockIdx.y * 32,
              z0 = (blockIdx.z - c * slabs) * TZ, zend = min(z0 + TZ, D);
    const long long HW = (long long)H * W;
    in += c * HW * D;
    out += c * HW * D;
    const int zs = z0 - R, np = zend - z0 + 2 * R;

    // positions: (row wy + 8 j, column lane), then the columns from 32 on; one
    // outside the grid reads its nearest voxel inside and is masked to zero
    unsigned off[NM + NE], keep[NM + NE];
    int ex[NE];  // staged places of the last columns' positions, -1: none
    auto place = [&](int j, int ry, int rx) {
        const int y = y0 - R + ry, x = x0 - R + rx;
        const int yc = min(max(y, 0), H - 1), xc = min(max(x, 0), W - 1);
        off[j] = (unsigned)(yc * W + xc);
        keep[j] = ry < RY && y == yc && x == xc ? 0xffffffffu : 0u;
    };
#pragma unroll
    for (int j = 0; j < NM; ++j) place(j, wy + 8 * j, lane);
#pragma unroll
    for (int j = 0; j < NE; ++j) {
        const int e = tid + j * G::NT, ry = e / (2 * R), rx = 32 + e % (2 * R);
        place(NM + j, ry, rx);
        ex[j] = ry < RY ? ry * BX + rx : -1;
    }
    float *const st0 = sm + wy * BX + lane;              // this thread's first staged place
    const float *const x0s = sm + (tid >> 3) * BX + 4 * (tid & 7);  // its first x item
    float *const x0d = sm + 2 * PL + (tid >> 3) * 32 + 4 * (tid & 7);
    const float *const y0s = sm + 2 * PL + 4 * wy * 32 + lane;      // its column
    float v[NM + NE];
    const float *src = in + (long long)zs * HW;  // the plane to load next
    auto fetch = [&](int i) {
        if (i < np && zs + i >= 0 && zs + i < D) {
#pragma unroll
            for (int j = 0; j < NM + NE; ++j) v[j] = __ldg(src + off[j]);
        }
        src += HW;
    };
    auto stage = [&](int i, int half) {
        if (i < np && zs + i >= 0 && zs + i < D) {
            const int h = half ? PL : 0;
#pragma unroll
            for (int j = 0; j < NM; ++j)
                if (RY % 8 == 0 || j < NM - 1 || wy + 8 * j < RY)
                    st0[h + 8 * j * BX] = __uint_as_float(__float_as_uint(v[j]) & keep[j]);
#pragma unroll
            for (int j = 0; j < NE; ++j)
                if (ex[j] >= 0)
                    sm[h + ex[j]] = __uint_as_float(__float_as_uint(v[NM + j]) & keep[NM + j]);
        }
    };
    fetch(0);
    stage(0, 0);
    fetch(1);

    float2 a[2][2 * R];  // open outputs of rows (0, 1) and (2, 3)
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int k = 0; k < 2 * R; ++k) a[p][k] = make_float2(0.0f, 0.0f);
    const int yo = y0 + 4 * wy, rows_out = x0 + lane < W ? H - yo : 0;
    float *dst = out + (long long)(z0 - 1 - 2 * R) * HW + (long long)yo * W + x0 + lane;
    int half = 0;
    for (int i = 0; i <= np; ++i, half ^= 1, dst += HW) {
        __syncthreads();
        if (i < np && zs + i >= 0 && zs + i < D) {  // x
            const float *s = x0s + (half ? PL : 0);
            float *d = x0d + (half ? XS : 0);
#pragma unroll
            for (int j = 0; j < G::NI; ++j) {
                if (G::ITEMS % G::NT != 0 && j == G::NI - 1 && tid + j * G::NT >= G::ITEMS) break;
                constexpr int NL = (4 + 2 * R + 3) / 4;
                const float4 *q = (const float4 *)(s + 32 * j * BX);
                float r[4 * NL];
#pragma unroll
                for (int l = 0; l < NL; ++l) *(float4 *)(r + 4 * l) = q[l];
                float o[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float acc = 0.0f;
#pragma unroll
                    for (int k = 0; k <= 2 * R; ++k) acc = fmaf(t.w[k], r[e + k], acc);
                    o[e] = acc;
                }
                *(float4 *)(d + 32 * j * 32) = make_float4(o[0], o[1], o[2], o[3]);
            }
        }
        stage(i + 1, half ^ 1);
        fetch(i + 2);
        if (i == 0) continue;
        const int z = zs + i - 1;  // y and z of the plane before
        float q[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (z >= 0 && z < D) {
            const float *s = y0s + (half ? 0 : XS);
            float r[4 + 2 * R];
#pragma unroll
            for (int k = 0; k < 4 + 2 * R; ++k) r[k] = s[k * 32];
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int k = 0; k <= 2 * R; ++k) q[e] = fmaf(t.w[k], r[e + k], q[e]);
        }
        float2 o[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const float2 qp = make_float2(q[2 * p], q[2 * p + 1]);
            auto tap = [&](int k, float2 acc) {
                return __ffma2_rn(make_float2(t.w[k], t.w[k]), qp, acc);
            };
            o[p] = tap(2 * R, a[p][0]);
#pragma unroll
            for (int k = 0; k + 1 < 2 * R; ++k) a[p][k] = tap(2 * R - 1 - k, a[p][k + 1]);
            a[p][2 * R - 1] = tap(0, make_float2(0.0f, 0.0f));
        }
        if (i - 1 >= 2 * R) {
            if (rows_out >= 4) {
                dst[0] = o[0].x;
                dst[W] = o[0].y;
                dst[2 * (long long)W] = o[1].x;
                dst[3 * (long long)W] = o[1].y;
            } else {
                if (rows_out > 0) dst[0] = o[0].x;
                if (rows_out > 1) dst[W] = o[0].y;
                if (rows_out > 2) dst[2 * (long long)W] = o[1].x;
            }
        }
    }
}

template <int R>
static cudaError_t onepass(const float *in, float *out, int C, Dims d, const GaussTaps &t,
                           cudaStream_t s) {
    using G = GaussTile<R>;
    auto kern = k_gauss_onepass<R>;
    const int occ = prepare(kern, G::bytes, G::NT);
    const int gx = (d.W + 31) / 32, gy = (d.H + 31) / 32;
    LaunchGeom g;
    g.tz = choose_tz(d.D, gx * gy * C, 2.0f * R + 1.0f, occ);
    const int slabs = (d.D + g.tz - 1) / g.tz;
    g.grid = dim3(gx, gy, (unsigned)(slabs * C));
    g.block = dim3(G::NT);
    OnePassTaps<R> w;
    for (int k = 0; k <= 2 * R; ++k) w.w[k] = t.w[k];
    kern<<<g.grid, g.block, G::bytes, s>>>(in, out, d.D, d.H, d.W, g.tz, slabs, w);
    note_launch();
    return cudaGetLastError();
}

// The one-pass kernel takes unpadded grids that its launch limits allow (65,535
// layers of tiles along y and of slabs) and that have more than five rows; anything
// else goes axis by axis.  With fewer rows its tiles of 32 are mostly empty (three
// channels of 600 x H x 701, sigma 1, one pass against three, us: H = 1 87 and 44,
// 2 87 and 53, 4 87 and 76; sigma 2: H = 4 150 and 98, 6 152 and 146).
static bool onepass_takes(int C, Dims d, const GaussTaps &t) {
    return t.R >= 1 && t.R <= kOnePassRadius && d.pitch() == d.W && d.H > 5 &&
           (d.H + 31) / 32 <= 65535 && (long long)C * d.D <= 65535;
}

cudaError_t launch_gauss3(const float *in, float *out, float *t1, float *t2, int C, Dims d,
                          const GaussTaps &t, cudaStream_t s) {
    const long long n = C * d.NP();
    if (t.R == 0) {
        if (in == out) return cudaSuccess;
        return cudaMemcpyAsync(out, in, sizeof(float) * n, cudaMemcpyDeviceToDevice, s);
    }
    cudaError_t e;
    if (onepass_takes(C, d, t)) {
        // CTAs read their neighbours' voxels: a result that overlaps its input
        // is made in the scratch
        const bool over = out < in + n && in < out + n;
        float *dst = over ? t1 : out;
        switch (t.R) {
            case 1: e = onepass<1>(in, dst, C, d, t, s); break;
            case 2: e = onepass<2>(in, dst, C, d, t, s); break;
            case 3: e = onepass<3>(in, dst, C, d, t, s); break;
            case 4: e = onepass<4>(in, dst, C, d, t, s); break;
            case 5: e = onepass<5>(in, dst, C, d, t, s); break;
            default: e = onepass<6>(in, dst, C, d, t, s); break;
        }
        if (e != cudaSuccess || !over) return e;
        return cudaMemcpyAsync(out, dst, sizeof(float) * n, cudaMemcpyDeviceToDevice, s);
    }
    if ((e = launch_gauss_axis(in, t1, C, d, t, 0, s)) != cudaSuccess) return e;
    if ((e = launch_gauss_axis(t1, t2, C, d, t, 1, s)) != cudaSuccess) return e;
    return launch_gauss_axis(t2, out, C, d, t, 2, s);
}

cudaError_t launch_gauss3_any(const float *in, float *t1, float *t2, int C, Dims d,
                              const GaussTaps &t, const float **res, cudaStream_t s) {
    *res = t.R == 0 ? in : t1;
    return t.R == 0 ? cudaSuccess : launch_gauss3(in, t1, t1, t2, C, d, t, s);
}

}  // namespace fa

extern "C" size_t fa_gauss_workspace_size(int32_t C, int32_t D, int32_t H, int32_t W) {
    if (C < 1 || D < 1 || H < 1 || W < 1) return 0;
    fa::WsCarver c(nullptr, ~size_t(0));
    c.take<float>((size_t)C * D * H * W);
    c.take<float>((size_t)C * D * H * W);
    return c.off;
}

extern "C" fa_status fa_gauss_smooth(const fa_vol *in, fa_vol *out, float sigma, void *ws,
                                     size_t ws_bytes, void *stream) {
    using namespace fa;
    clear_error();
    if (!in) {
        set_error("in: descriptor is NULL");
        return FA_ERR_INVALID;
    }
    FA_TRY(check_vol(in, "in", in->C));
    FA_TRY(check_vol(out, "out", in->C));
    FA_TRY(same_grid(in, out, "in", "out"));
    GaussTaps t;
    if (!make_gauss_taps(sigma, &t)) {
        set_error("fa_gauss_smooth: sigma must be in [0, %g] (got %g)", (double)kMaxSigma,
                  (double)sigma);
        return FA_ERR_INVALID;
    }
    size_t need = t.R ? fa_gauss_workspace_size(in->C, in->D, in->H, in->W) : 0;
    FA_TRY(check_ws(ws, ws_bytes, need, "fa_gauss_smooth"));
    Dims d{in->D, in->H, in->W};
    float *t1 = nullptr, *t2 = nullptr;
    if (t.R) {
        WsCarver c(ws, ws_bytes);
        t1 = c.take<float>((size_t)in->C * d.N());
        t2 = c.take<float>((size_t)in->C * d.N());
    }
    FA_CUDA_TRY(launch_gauss3((const float *)in->data, (float *)out->data, t1, t2, in->C, d, t,
                              (cudaStream_t)stream));
    return FA_OK;
}
