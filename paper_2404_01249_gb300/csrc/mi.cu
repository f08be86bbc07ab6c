// Mutual-information loss (named with LNCC among the costs of the problem
// statement, section "Deformable Image Registration"; its bin count is one of
// the hyper-parameters of the hyper-parameter study).  Parzen-window estimate
// with the cubic B-spline beta3 on B bins for both images: an intensity v of
// an image with range [lo, hi] sits at bin coordinate
//   xi = 1 + (v - lo) (B - 3) / (hi - lo), clamped to [1, B - 2],
// where the weights beta3(xi - k) of the bins k = 0..B-1 sum to one.
//   P(a,b) = (1/N) sum_x beta3(xi_f(x) - a) beta3(xi_m(x) - b),
//   L = -MI = -sum P log(P / (p_f p_m)),
//   dL/dJ(x) = -(1/N) (B - 3) / (hi_m - lo_m)
//              sum_{a,b} log(P / (p_f p_m)) beta3(xi_f - a) beta3'(xi_m - b).
// The joint histogram is accumulated in 2^-32 fixed point with integer
// atomics, so it does not depend on thread order.
#include "launch.cuh"
#include "ops.h"
#include "validate.h"

namespace fa {

namespace {

constexpr int kMiBits = 32;  // fixed-point scale of the histogram terms (< 2^31 each)

__device__ __forceinline__ unsigned fkey(float f) {  // order-preserving float key
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float fval(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

struct MiMap {
    float lo, s;  // xi = 1 + (v - lo) s
    int B;
    __device__ float coord(float v) const {
        const float xi = fmaf(v - lo, s, 1.0f);
        return fminf(fmaxf(xi, 1.0f), (float)(B - 2));
    }
};

__device__ __forceinline__ MiMap mi_map(const unsigned *keys, int k, int B) {
    MiMap m;
    m.lo = fval(keys[2 * k]);
    const float hi = fval(keys[2 * k + 1]);
    m.s = hi > m.lo ? (float)(B - 3) / (hi - m.lo) : 0.0f;
    m.B = B;
    return m;
}

// cubic B-spline weights of bins floor(xi) - 1 .. floor(xi) + 2, t = xi - floor(xi)
__device__ __forceinline__ void bspline_w(float t, float w[4]) {
    const float t2 = t * t, t3 = t2 * t, r = 1.0f - t;
    w[0] = r * r * r * (1.0f / 6.0f);
    w[1] = fmaf(0.5f, t3, fmaf(-1.0f, t2, 2.0f / 3.0f));
    w[2] = fmaf(-0.5f, t3, fmaf(0.5f, t2, fmaf(0.5f, t, 1.0f / 6.0f)));
    w[3] = t3 * (1.0f / 6.0f);
}
// their derivatives with respect to xi
__device__ __forceinline__ void bspline_dw(float t, float w[4]) {
    const float t2 = t * t, r = 1.0f - t;
    w[0] = -0.5f * r * r;
    w[1] = fmaf(1.5f, t2, -2.0f * t);
    w[2] = fmaf(-1.5f, t2, t + 0.5f);
    w[3] = 0.5f * t2;
}

// Values i .. i + 3 (i a multiple of 4, volumes start on 16 bytes), those
// beyond N as 0.
__device__ __forceinline__ void load4(float (&v)[4], const float *__restrict__ p, long long i,
                                      long long N) {
    if (i + 4 <= N) {
        const float4 q = __ldg((const float4 *)(p + i));
        v[0] = q.x;
        v[1] = q.y;
        v[2] = q.z;
        v[3] = q.w;
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = i + e < N ? __ldg(p + i + e) : 0.0f;
    }
}

// PAD: rows hold W voxels and P elements, P a multiple of 4 (such volumes have
// fewer than 2^32 elements); else P = W.  The dense forms keep their registers
// (36 instead of 32 would leave the range kernel 7 of its 8 blocks per SM: 1.5
// us of 148 for the loss and its gradient on 6.9 M voxels).
// Which of the values i .. i + 3 (i a multiple of 4) of a volume of N elements
// are voxels: the first so many.
template <bool PAD>
__device__ __forceinline__ int voxels4(long long i, long long N, int W, int P) {
    if (!PAD) return i + 4 <= N ? 4 : (int)(N - i);
    return min(4, max(0, W - (int)((unsigned)i % (unsigned)P)));
}

__global__ void k_mi_range_init(unsigned *keys) {
    keys[0] = 0xffffffffu;   // lo_f: min over the fixed image
    keys[1] = 0u;            // hi_f
    keys[2] = fkey(0.0f);    // lo_m, hi_m: the moving image with 0 included
    keys[3] = fkey(0.0f);
}

__global__ void k_mi_range_set(const float *range, unsigned *keys) {
    if (threadIdx.x < 4) keys[threadIdx.x] = fkey(range[threadIdx.x]);
}

template <bool PAD>
__global__ void __launch_bounds__(256) k_mi_range(const float *__restrict__ If,
                                                  const float *__restrict__ Im, long long N,
                                                  int W, int P, unsigned *keys) {
    unsigned k[4] = {0xffffffffu, 0u, 0xffffffffu, 0u};
    for (long long i = 4 * ((long long)blockIdx.x * blockDim.x + threadIdx.x); i < N;
         i += 4ll * gridDim.x * blockDim.x) {
        float a[4], b[4];
        load4(a, If, i, N);
        load4(b, Im, i, N);
        const int n = voxels4<PAD>(i, N, W, P);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (e >= n) break;
            if (fabsf(a[e]) <= 3.4e38f) {
                k[0] = min(k[0], fkey(a[e]));
                k[1] = max(k[1], fkey(a[e]));
            }
            if (fabsf(b[e]) <= 3.4e38f) {
                k[2] = min(k[2], fkey(b[e]));
                k[3] = max(k[3], fkey(b[e]));
            }
        }
    }
    // one set of global atomics per block: all of them go to the same four
    // words (one set per warp: 34 us on 6.9 M voxels; per block, with
    // 16-byte loads: 13 us)
    __shared__ unsigned red[4];
    if (threadIdx.x < 4) red[threadIdx.x] = (threadIdx.x & 1) ? 0u : 0xffffffffu;
    __syncthreads();
    k[0] = __reduce_min_sync(0xffffffffu, k[0]);
    k[1] = __reduce_max_sync(0xffffffffu, k[1]);
    k[2] = __reduce_min_sync(0xffffffffu, k[2]);
    k[3] = __reduce_max_sync(0xffffffffu, k[3]);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(red + 0, k[0]);
        atomicMax(red + 1, k[1]);
        atomicMin(red + 2, k[2]);
        atomicMax(red + 3, k[3]);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMin(keys + 0, red[0]);
        atomicMax(keys + 1, red[1]);
        atomicMin(keys + 2, red[2]);
        atomicMax(keys + 3, red[3]);
    }
}

// Joint histogram.  Each weight product is quantised to 2^-32 (q < 2^31) and
// added as two halves, q mod 2^16 and q / 2^16, with 32-bit shared atomics.
// Neighbouring voxels fall in the same bins, so the block keeps 2^LC copies,
// one per lane modulo 2^LC, interleaved bin by bin: lanes that add to the
// same bin add to different words in different banks.  A copy takes at most
// 32 warps x 32 / 2^LC lanes x kHistIters voxels, so that each half-sum stays
// below 2^32; the block recombines the halves exactly in 64 bits and adds its
// non-zero bins to the global histogram.
// Bound: the shared-memory atomics, 32 per voxel.  6.9 M voxels, 32 bins:
// 590 us with one copy per warp (lanes of a warp serialised on the few bins
// of a smooth region), 88 us with 16 copies.  Where 152 blocks of 512 threads
// cover the volume with one voxel per thread, zeroing and reading out the copies
// counts: four of them then (the loss and its gradient on 13,440 voxels, 16, 32
// and 64 bins: 20.5, 19.8 and 29.0 us against 21.9, 21.9 and 29.7 with up to 16
// in blocks of 1,024; on 107,604 voxels 22.6 and 22.7, the line).
constexpr int kHistThreads = 1024, kHistIters = 64;
constexpr size_t kHistSmem = 196 * 1024;
constexpr long long kMiGradOne = 1ll << 20;  // the gradient's one-voxel form up to here

int hist_log_copies(int nb, int lc) {  // at most 2^lc
    while (lc > 0 && ((size_t)nb << lc) * 8 > kHistSmem) --lc;
    return lc;
}

template <bool PAD>
__global__ void __launch_bounds__(kHistThreads) k_mi_hist(const float *__restrict__ I,
                                                          const float *__restrict__ J, long long N,
                                                          int W, int P, int B, int lc,
                                                          const unsigned *__restrict__ keys,
                                                          unsigned long long *ghist, WsHeader *h) {
    extern __shared__ unsigned shu[];  // [2][B*B][2^lc]: low and high halves
    const int nb = B * B, copies = 1 << lc;
    for (int k = threadIdx.x; k < 2 * nb * copies; k += blockDim.x) shu[k] = 0u;
    __syncthreads();
    unsigned *lo_h = shu + (threadIdx.x & (copies - 1)), *hi_h = lo_h + ((size_t)nb << lc);
    const MiMap mf = mi_map(keys, 0, B), mm = mi_map(keys, 1, B);
    bool bad = false;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += stride) {
        if (PAD && (int)((unsigned)i % (unsigned)P) >= W) continue;
        const float a = I[i], b = J[i];
        if (!(fabsf(a) <= 3.4e38f && fabsf(b) <= 3.4e38f)) {
            bad = true;
            continue;
        }
        const float xf = mf.coord(a), xm = mm.coord(b);
        const float ff = floorf(xf), fm = floorf(xm);
        float wf[4], wm[4];
        bspline_w(xf - ff, wf);
        bspline_w(xm - fm, wm);
        const int a0 = (int)ff - 1, b0 = (int)fm - 1;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            if (a0 + p >= B) continue;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned v = __float2uint_rn(wf[p] * wm[q] * 4294967296.0f);
                if (v == 0u || b0 + q >= B) continue;
                const int k = ((a0 + p) * B + b0 + q) << lc;
                atomicAdd(lo_h + k, v & 0xffffu);
                if (v >> 16) atomicAdd(hi_h + k, v >> 16);
            }
        }
    }
    if (bad) status_set(&h->status, ST_NONFINITE);
    __syncthreads();
    for (int k = threadIdx.x; k < nb; k += blockDim.x) {
        unsigned long long t = 0ull;
        for (int c = 0; c < copies; ++c) {  // each thread starts at another copy's bank
            const int w = (k << lc) + ((c + threadIdx.x) & (copies - 1));
            t += (unsigned long long)shu[w] + ((unsigned long long)shu[((size_t)nb << lc) + w] << 16);
        }
        if (t) atomicAdd(ghist + k, t);
    }
}

// P, marginals, MI and the table log(P / (p_f p_m)), in FP32.  The
// marginals are exact integer sums of the fixed-point histogram, so every
// probability is one rounding of an exact count; the ratio adds two
// roundings and logf one more.  MI = sum P log(...) is accumulated as a
// float-float pair per thread (exact products by fmaf, two-sum additions)
// and the pairs are combined in a fixed tree order, so the loss carries
// about FP32's unit roundoff and does not depend on scheduling.
__global__ void __launch_bounds__(1024) k_mi_table(const unsigned long long *__restrict__ ghist,
                                                   int B, long long N, float *T, WsHeader *h,
                                                   float *loss_out) {
    extern __shared__ float shf[];
    float *P = shf, *pf = shf + B * B, *pm = pf + B, *rh = pm + B, *rl = rh + blockDim.x;
    const int nb = B * B, tid = threadIdx.x;
    const float Nf = (float)N, unit = pow2f(-kMiBits);
    for (int k = tid; k < nb; k += blockDim.x)
        P[k] = __fdiv_rn(u64_to_float_rn(ghist[k]) * unit, Nf);
    if (tid < B) {
        unsigned long long s = 0ull;
        for (int b = 0; b < B; ++b) s += ghist[tid * B + b];
        pf[tid] = __fdiv_rn(u64_to_float_rn(s) * unit, Nf);
    } else if (tid < 2 * B) {
        unsigned long long s = 0ull;
        for (int a = 0; a < B; ++a) s += ghist[a * B + tid - B];
        pm[tid - B] = __fdiv_rn(u64_to_float_rn(s) * unit, Nf);
    }
    __syncthreads();
    float hi = 0.0f, lo = 0.0f;
    for (int k = tid; k < nb; k += blockDim.x) {
        const float q = P[k];
        float tv = 0.0f;
        if (q > 0.0f) {
            tv = logf(__fdiv_rn(q, pf[k / B] * pm[k % B]));
            const float ph = q * tv, pl = fmaf(q, tv, -ph);
            ff_add(hi, lo, ph, pl);
        }
        T[k] = tv;
    }
    rh[tid] = hi;
    rl[tid] = lo;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (tid < o) {
            float a = rh[tid], b = rl[tid];
            ff_add(a, b, rh[tid + o], rl[tid + o]);
            rh[tid] = a;
            rl[tid] = b;
        }
        __syncthreads();
    }
    if (tid == 0) {
        const float L = -(rh[0] + rl[0]);
        h->loss = L;
        if (loss_out) *loss_out = L;
    }
}

// The values of V voxels from i on (V = 4: as load4).
template <int V>
__device__ __forceinline__ void load_v(float (&v)[V], const float *__restrict__ p, long long i,
                                       long long N) {
    if constexpr (V == 4)
        load4(v, p, i, N);
    else
        v[0] = __ldg(p + i);
}

// V adjacent voxels per thread and step.  With four their loads and table reads
// overlap, bound by the table's shared-memory reads; with one, a small volume
// has four times the threads.  The loss and its gradient, 32 bins, one against
// four (us): 13,440 voxels 18.9 and 19.8, 512,000 31.5 and 31.9, 1.4 M 49.7 and
// 49.2, 6.9 M 160 and 154: hence kMiGradOne.
template <int V>
__global__ void __launch_bounds__(256) k_mi_grad(const float *__restrict__ I,
                                                 const float *__restrict__ J,
                                                 const float *__restrict__ grad, long long N,
                                                 float count, int B,
                                                 const unsigned *__restrict__ keys,
                                                 const float *__restrict__ Tg, float *dJ,
                                                 float *g) {
    extern __shared__ float T[];
    for (int k = threadIdx.x; k < B * B; k += blockDim.x) T[k] = Tg[k];
    __syncthreads();
    const MiMap mf = mi_map(keys, 0, B), mm = mi_map(keys, 1, B);
    const float c = -mm.s / count;
    for (long long i = V * ((long long)blockIdx.x * blockDim.x + threadIdx.x); i < N;
         i += (long long)V * gridDim.x * blockDim.x) {
        float Iv[V], Jv[V], dj[V];
        load_v(Iv, I, i, N);
        load_v(Jv, J, i, N);
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const float xf = mf.coord(Iv[e]), xm = mm.coord(Jv[e]);
            const float ff = floorf(xf), fm = floorf(xm);
            float wf[4], dm[4];
            bspline_w(xf - ff, wf);
            bspline_dw(xm - fm, dm);
            const int a0 = (int)ff - 1, b0 = (int)fm - 1;
            float acc = 0.0f;
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                if (a0 + p >= B) continue;
                float r = 0.0f;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (b0 + q < B) r = fmaf(T[(a0 + p) * B + b0 + q], dm[q], r);
                acc = fmaf(wf[p], r, acc);
            }
            dj[e] = c * acc;
        }
        const bool all = i + V <= N;
        if (dJ) {
            if (V == 4 && all) {
                *(float4 *)(dJ + i) = make_float4(dj[0], dj[1 % V], dj[2 % V], dj[3 % V]);
            } else {
#pragma unroll
                for (int e = 0; e < V; ++e)
                    if (i + e < N) dJ[i + e] = dj[e];
            }
        }
        if (g) {
            const bool vec = V == 4 && all && (N & 3) == 0;  // the other channels start on 16 bytes too
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                const float *src = grad + ch * N + i;
                float *dst = g + ch * N + i;
                if (vec) {
                    const float4 q = *(const float4 *)src;
                    *(float4 *)dst = make_float4(dj[0] * q.x, dj[1 % V] * q.y, dj[2 % V] * q.z,
                                                 dj[3 % V] * q.w);
                } else {
#pragma unroll
                    for (int e = 0; e < V; ++e)
                        if (i + e < N) dst[e] = dj[e] * src[e];
                }
            }
        }
    }
}

unsigned grid_blocks(long long N) {  // of 256 threads, four voxels each
    long long b = (N + 1023) / 1024;
    return (unsigned)(b > 152 * 8 ? 152 * 8 : (b < 1 ? 1 : b));
}

}  // namespace

MiBuffers mi_carve(WsCarver &c, int bins) {
    MiBuffers b;
    b.hist = c.take<unsigned long long>((size_t)bins * bins);
    b.T = c.take<float>((size_t)bins * bins);
    b.range = c.take<unsigned>(4);
    return b;
}

cudaError_t launch_mi_range(const float *If, const float *Im, Dims d, MiBuffers b,
                            cudaStream_t s) {
    const long long N = d.NP();
    k_mi_range_init<<<1, 1, 0, s>>>(b.range);
    note_launch();
    auto range = d.pitch() != d.W ? k_mi_range<true> : k_mi_range<false>;
    range<<<grid_blocks(N), 256, 0, s>>>(If, Im, N, d.W, d.pitch(), b.range);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_mi_range_set(const float *range4, MiBuffers b, cudaStream_t s) {
    k_mi_range_set<<<1, 32, 0, s>>>(range4, b.range);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_mi(const float *I, const float *J, const float *grad, Dims d, int bins,
                      WsHeader *h, MiBuffers b, float *loss_out, float *dJ, float *g,
                      cudaStream_t s) {
    const long long N = d.NP();  // elements; the gradient fills a row's padding too
    const int nb = bins * bins;
    cudaError_t e = cudaMemsetAsync(b.hist, 0, sizeof(unsigned long long) * nb, s);
    if (e != cudaSuccess) return e;
    auto hist = d.pitch() != d.W ? k_mi_hist<true> : k_mi_hist<false>;
    prepare(hist, kHistSmem, kHistThreads);
    const bool one_pass = N <= 512ll * num_sms();
    const int threads = one_pass ? 512 : kHistThreads;
    const int lc = hist_log_copies(nb, one_pass ? 2 : 5);
    const long long most = (N + threads - 1) / threads;
    long long hb = (most + kHistIters - 1) / kHistIters;
    hb = hb < num_sms() ? num_sms() : hb;
    hb = hb < most ? hb : most;
    hist<<<(unsigned)hb, threads, ((size_t)nb << lc) * 8, s>>>(
        I, J, N, d.W, d.pitch(), bins, lc, b.range, b.hist, h);
    note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const size_t tab_smem = sizeof(float) * (nb + 2 * bins + 2 * 1024);
    k_mi_table<<<1, 1024, tab_smem, s>>>(b.hist, bins, d.N(), b.T, h, loss_out);
    note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (dJ || g) {
        if (N <= kMiGradOne) {
            long long gb = (N + 255) / 256;
            gb = gb < 152 * 4 ? gb : 152 * 4;
            k_mi_grad<1><<<(unsigned)gb, 256, sizeof(float) * nb, s>>>(
                I, J, grad, N, (float)d.N(), bins, b.range, b.T, dJ, g);
        } else {
            k_mi_grad<4><<<grid_blocks(N), 256, sizeof(float) * nb, s>>>(
                I, J, grad, N, (float)d.N(), bins, b.range, b.T, dJ, g);
        }
        note_launch();
    }
    return cudaGetLastError();
}

}  // namespace fa

extern "C" size_t fa_mi_workspace_size(int32_t bins) {
    fa::clear_error();
    if (bins < fa::kMiMinBins || bins > fa::kMiMaxBins) return 0;
    fa::WsCarver c(nullptr, ~size_t(0));
    c.take<fa::WsHeader>(1);
    fa::mi_carve(c, bins);
    return c.off;
}

extern "C" fa_status fa_mi_fwd_bwd(const fa_vol *fixed, const fa_vol *warped, int32_t bins,
                                   const float *range_dev_opt, float *loss_dev,
                                   fa_vol *dL_dwarped_opt, void *ws, size_t ws_bytes,
                                   void *stream) {
    using namespace fa;
    clear_error();
    if (bins < kMiMinBins || bins > kMiMaxBins) {
        set_error("fa_mi_fwd_bwd: bins must be in %d..%d (got %d)", kMiMinBins, kMiMaxBins,
                  (int)bins);
        return FA_ERR_INVALID;
    }
    FA_TRY(check_vol(fixed, "fixed", 1));
    FA_TRY(check_vol(warped, "warped", 1));
    FA_TRY(same_grid(fixed, warped, "fixed", "warped"));
    if (dL_dwarped_opt) {
        FA_TRY(check_vol(dL_dwarped_opt, "dL_dwarped", 1));
        FA_TRY(same_grid(fixed, dL_dwarped_opt, "fixed", "dL_dwarped"));
    }
    FA_TRY(check_ws(ws, ws_bytes, fa_mi_workspace_size(bins), "fa_mi_fwd_bwd"));
    WsCarver c(ws, ws_bytes);
    WsHeader *h = c.take<WsHeader>(1);
    MiBuffers b = mi_carve(c, bins);
    cudaStream_t s = (cudaStream_t)stream;
    const Dims d{fixed->D, fixed->H, fixed->W};
    const float *I = (const float *)fixed->data, *J = (const float *)warped->data;
    FA_CUDA_TRY(launch_header_reset(h, s));
    if (range_dev_opt)
        FA_CUDA_TRY(launch_mi_range_set(range_dev_opt, b, s));
    else
        FA_CUDA_TRY(launch_mi_range(I, J, d, b, s));
    FA_CUDA_TRY(launch_mi(I, J, nullptr, d, bins, h, b, loss_dev,
                          dL_dwarped_opt ? (float *)dL_dwarped_opt->data : nullptr, nullptr, s));
    return FA_OK;
}
