// Fused per-iteration kernels of fa_register (FA_MODE_FUSED).
//
// One iteration of Algorithm 1 (Jacobian-free direction) is four launches:
//   K1 k_lncc_fwd       LNCC forward on J = I_m o phi: exact int64 window
//                       sums of J, J^2 and I J (the fixed image's window sum
//                       and variance come precomputed per level), cc, the
//                       adjoint coefficients A, B, C, the loss accumulator and
//                       the coefficient maxima.
//   K2 k_lncc_grad      adjoint window sums of A, B, C; g = dL/dJ grad I_m(phi)
//                       with J and grad I_m(phi) as the compose kernel stored
//                       them.
//   K3 k_smooth_adam    Gaussian(sigma_grad) of g, Adam update of m, nu, the
//                       direction d and the grid max |d|.
//   K4 k_compose        delta = -eps_t d, u' = delta + u o (id + delta),
//                       Gaussian(sigma_warp) of u', and J = I_m o (id + u')
//                       with its gradient grad I_m(phi') for the next
//                       iteration's K1 and K2 (one gather per iteration).
// The grid max of K3 is a global dependency, so K4 cannot join K3; the
// adjoint window sums need A, B, C around every output, so K2 cannot join K1
// without recomputing a much wider halo.
//
// K1 and K2 are in window.cuh; K3 and K4 are here.
//
// Every kernel marches along z ("2.5-D" tiling).  In K3 and K4 a CTA owns a
// 32 x TY tile of (x, y) columns and a slab of TZ output planes.  A plane's
// inputs (the tile plus its halo, and the operands of the plane's outputs)
// arrive NSTG - 1 planes ahead of use.  When the buffers' rows start on
// 16-byte boundaries (a registration pads its levels' rows to a multiple of 4
// floats) they come as TMA tile copies issued by one thread and completed on
// an mbarrier (zero fill outside the grid); otherwise each thread copies its
// own positions with cp.async.
//
// The passes over a plane are pipelined over the planes: between two barriers
// each pass works on a plane of its own, one behind the pass before it, with
// doubled buffers in between.  So there is one barrier per plane instead of
// two (K3) or three (K4), and the passes' shared-memory latencies overlap.
// Along x a plane goes from shared memory to shared memory (4 outputs per item
// from 16-byte loads); along y a thread sums its adjacent output rows in
// registers; along z it adds the plane into the 2R + 1 outputs it reaches
// (OpenZ), which took the place of a shared-memory ring of 2R + 1 planes.  No
// intermediate of the separable sums goes to HBM; halo re-reads hit L2.
//
// Where steps reach a voxel, K4 gathers u from global memory, and the latency of
// a position's 24 corners bounds it: the three channels' corners are issued
// together (one channel after the other, ten MSE iterations with sigma_warp 1
// took 6,136 us on 160 x 192 x 224 and 545 on 40 x 48 x 56; together 4,708 and 428;
// before the passes were pipelined 5,425 and 503).
//
// K4 is bound by the shared-memory pipe (per 32 outputs about 62 wavefronts of
// loads and stores, 34 of them the cell corners, against 85 with the ring and
// one row per thread), K3 by HBM at the finest level and by latency below.
//
// Shared layout of a staged plane: [C][RY][BXW] with BXW = 32 + 2 XB and XB = R rounded
// up to a multiple of 4.  Column c holds x = x0 - XB + c and row r holds
// y = y0 - R + r, so that a TMA box starts on a 16-byte boundary.
//
// Every wait on a TMA barrier is bounded; a wait that gives up sets
// ST_TIMEOUT in the status word, waits (bounded again) for the CTA's copies
// in flight and ends the CTA, and later CTAs that see the bit drain their
// first copies and return.
#pragma once

#include <cuda.h>
#include <type_traits>
#include <math.h>

#include "launch.cuh"
#include "register.h"
#include "validate.h"
#include "window.cuh"

namespace fa {

namespace {


__host__ __device__ constexpr int halo4(int r) { return (r + 3) / 4 * 4; }
__host__ __device__ constexpr size_t al128(size_t b) { return (b + 127) & ~size_t(127); }

__device__ __forceinline__ unsigned su32(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

// ----------------------------------------------------------- cp.async path
__device__ __forceinline__ void cp4(void *dst, const void *src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(su32(dst)), "l"(src),
                 "r"(ok ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------- TMA path
__device__ __forceinline__ void mbar_init(unsigned long long *b) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(su32(b)) : "memory");
}
// Makes initialised barriers visible to the TMA unit.
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
// The arrival of the one expected thread, announcing `bytes` of copies.
__device__ __forceinline__ void mbar_expect(unsigned long long *b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(su32(b)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned long long *b, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Waits for the phase of parity `parity` to complete; gives up after about
// `limit` SM cycles (default 2^28: 0.13 s at 2 GHz; a tile copy takes
// microseconds).
__device__ __forceinline__ bool mbar_wait(unsigned long long *b, unsigned parity,
                                          long long limit = 1ll << 28) {
    if (mbar_try(b, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try(b, parity))
        if (clock64() - t0 > limit) return false;
    return true;
}
// One tile copy of a rank-4 map ([C][D][H][W]) into shared memory.
__device__ __forceinline__ void tma4(void *dst, const CUtensorMap *m, int x, int y, int z, int c,
                                     unsigned long long *b) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];\n" ::"r"(su32(dst)),
        "l"(reinterpret_cast<unsigned long long>(m)), "r"(x), "r"(y), "r"(z), "r"(c),
        "r"(su32(b))
        : "memory");
}

// Tensor maps of one launch (the ones a kernel does not use stay zero).
struct Maps {
    CUtensorMap a, b, c;
};

// The tensor maps a CTA's body loads through: generic addresses of maps in
// the kernel's parameter space (a launch's Maps, or one job's entries of a
// lockstep table); null where the body takes no TMA tiles.
struct MapRef {
    const CUtensorMap *a, *b, *c;
};
__device__ __forceinline__ MapRef map_ref(const Maps &m) { return MapRef{&m.a, &m.b, &m.c}; }

}  // namespace
// Map of a [C][D][H][W] field of 2- (FP16) or 4-byte elements with rows of
// d.pitch() elements, a {bx, by, 1, bc} box and zero fill outside the grid;
// false when the field does not meet TMA's alignment rules.
bool tmap(CUtensorMap *m, const void *base, int esize, Dims d, int C, int bx, int by, int bc);
namespace {

// For a CTA that has waited for the previous kernel (pdl_wait) and issued its
// first copies and header loads (so that they are in flight while the status
// word is read): true, uniformly over the CTA, when an earlier CTA reported a
// timeout; the caller then drains its copies (drain_first) and returns.
__device__ __forceinline__ bool status_timed_out(const WsHeader *h, int tid, int *flag) {
    if (tid == 0) *flag = (int)(*(volatile const unsigned *)&h->status & ST_TIMEOUT);
    __syncthreads();
    pdl_trigger();
    return *flag != 0;
}

// Bounded wait for the first min(n, NSTG) stage copies a CTA issued before it
// returns early (TMA), or for its copy groups (cp.async).
template <bool TMA, int NSTG>
__device__ __forceinline__ void drain_first(unsigned long long *bar, int n, int tid) {
    if (TMA) {
        if (tid == 0)
            for (int j = 0; j < n && j < NSTG; ++j) mbar_wait(bar + j, 0u);
    } else {
        cp_wait<0>();
    }
}

// --------------------------------------------- cp.async position mapping
// A thread's positions in the RY x RX logical region of a plane (RX <= 64):
// warp w covers rows w, w + NW, ...; lane l covers columns l and l + 32.
// Logical column rx is stored at column rx + COFF of a BXW-wide row.
template <int RY, int RX, int NW, int BXW, int COFF>
struct Region {
    static constexpr int NJ = (RY + NW - 1) / NW;
    static constexpr int NC = (RX + 31) / 32;
    int off[NJ * NC];  // y P + x inside the grid, -1 outside the grid, -2 outside the region
    int sbase;
    __device__ __forceinline__ void init(int wy, int tx, int ybase, int xbase, int H, int W,
                                         int P) {
        sbase = wy * BXW + tx + COFF;
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int ry = wy + NW * j, rx = tx + 32 * c;
                const int y = ybase + ry, x = xbase + rx;
                int o = -2;
                if (ry < RY && rx < RX) o = (y >= 0 && y < H && x >= 0 && x < W) ? y * P + x : -1;
                off[j * NC + c] = o;
            }
    }
    static __device__ __forceinline__ int sofs(int j, int c) { return NW * j * BXW + 32 * c; }
    // C channels of plane zoff / W H (zero outside the grid) -> [C][RY][BXW]
    template <int C>
    __device__ __forceinline__ void load(float *dst, const float *src, long long N, long long zoff,
                                         bool zok) const {
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int o = off[j * NC + c];
                if (o == -2) continue;
                const bool ok = zok && o >= 0;
                const float *s = src + (ok ? zoff + o : 0);
                float *d = dst + sbase + sofs(j, c);
#pragma unroll
                for (int ch = 0; ch < C; ++ch) cp4(d + ch * RY * BXW, s + ch * N, ok);
            }
    }
};

// This thread's OPT output voxels: rows OPT wy .. OPT wy + OPT - 1 of the
// tile, column tx (its places in a [TY][32] output tile start at `place`).
template <int OPT, int NW>
struct Outs {
    int off[OPT];  // y P + x (P: the row pitch), -1 outside the grid
    int place;
    __device__ __forceinline__ void init(int wy, int tx, int y0, int x0, int H, int W, int P) {
        place = OPT * wy * FX + tx;
#pragma unroll
        for (int o = 0; o < OPT; ++o) {
            const int y = y0 + OPT * wy + o, x = x0 + tx;
            off[o] = (y < H && x < W) ? y * P + x : -1;
        }
    }
    // C channels of this thread's outputs on plane zoff / (H W), to registers
    // (zero outside the grid)
    template <int C, class T>
    __device__ __forceinline__ void fetch(T (&r)[OPT][C], const T *src, long long N,
                                          long long zoff) const {
#pragma unroll
        for (int o = 0; o < OPT; ++o)
#pragma unroll
            for (int c = 0; c < C; ++c) r[o][c] = off[o] >= 0 ? src[c * N + zoff + off[o]] : T(0);
    }
};

// ------------------------------------------------- register-blocked x passes
// A work item is (channel, row, group of 4 adjacent output columns); items
// are spread over all threads.  The taps of output column ox start at plane
// column ox + COFF; rows are read with 16-byte shared loads from column 4k.

// Gaussian x pass: pl [C][RY][BXW] -> xb [C][RY][FX].
template <int RG, int C, int RY, int BXW, int COFF, int NT, class TT>
__device__ __forceinline__ void gauss_x4(const float *pl, float *xb, const TT &t, int tid) {
    constexpr int ITEMS = C * RY * 8, NL = (4 + COFF + 2 * RG + 3) / 4;
    static_assert(28 + 4 * NL <= BXW, "row too short for the vector loads");
#pragma unroll
    for (int j = 0; j < (ITEMS + NT - 1) / NT; ++j) {
        const int it = tid + j * NT;
        if (ITEMS % NT != 0 && it >= ITEMS) break;
        const int k = it & 7, rest = it >> 3, ry = rest % RY, c = rest / RY;
        const float4 *src = (const float4 *)(pl + (c * RY + ry) * BXW + 4 * k);
        float v[4 * NL];
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            const float4 q = src[l];
            v[4 * l] = q.x;
            v[4 * l + 1] = q.y;
            v[4 * l + 2] = q.z;
            v[4 * l + 3] = q.w;
        }
        float o[4];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            float a = 0.0f;
#pragma unroll
            for (int tt = 0; tt <= 2 * RG; ++tt) a = fmaf(t.w[tt], v[jj + COFF + tt], a);
            o[jj] = a;
        }
        *(float4 *)(xb + (c * RY + ry) * FX + 4 * k) = make_float4(o[0], o[1], o[2], o[3]);
    }
}

// Channels 0 and 1 of the y and z passes run as one packed FP32 pair
// (__ffma2_rn: each component is exactly fmaf), channel 2 alone; every
// channel's taps accumulate in the same order as a scalar loop would.
// The OPT outputs of a thread are adjacent rows and share their reads.
template <int RG, int RY, int OPT, class TT>
__device__ __forceinline__ void gauss_y3(const float *xb, const TT &t, int wy, int tx,
                                         float2 (&q01)[OPT], float (&q2)[OPT]) {
    const float *xi = xb + OPT * wy * FX + tx;
    float2 r01[OPT + 2 * RG];
    float r2[OPT + 2 * RG];
#pragma unroll
    for (int k = 0; k < OPT + 2 * RG; ++k) {
        r01[k] = make_float2(xi[k * FX], xi[(RY + k) * FX]);
        r2[k] = xi[(2 * RY + k) * FX];
    }
#pragma unroll
    for (int o = 0; o < OPT; ++o) {
        q01[o] = make_float2(0.0f, 0.0f);
        q2[o] = 0.0f;
#pragma unroll
        for (int k = 0; k <= 2 * RG; ++k) {
            q01[o] = __ffma2_rn(make_float2(t.w[k], t.w[k]), r01[o + k], q01[o]);
            q2[o] = fmaf(t.w[k], r2[o + k], q2[o]);
        }
    }
}

// The z pass as a transposed filter: a plane's in-plane results are added into
// the 2 RG + 1 outputs they reach; the 2 RG outputs still open sit in
// registers.  Planes come in ascending order, so every output's taps do too.
template <int RG, int OPT>
struct OpenZ {
    static constexpr int K = RG > 0 ? 2 * RG : 1;
    float2 a01[OPT][K];
    float a2[OPT][K];
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int o = 0; o < OPT; ++o)
#pragma unroll
            for (int k = 0; k < K; ++k) {
                a01[o][k] = make_float2(0.0f, 0.0f);
                a2[o][k] = 0.0f;
            }
    }
    // adds a plane; the output RG planes below it leaves with its sum
    template <class TT>
    __device__ __forceinline__ void push(const TT &t, const float2 (&q01)[OPT],
                                         const float (&q2)[OPT], float (&out)[OPT][3]) {
#pragma unroll
        for (int o = 0; o < OPT; ++o) {
            auto tap01 = [&](int k, float2 acc) {
                return __ffma2_rn(make_float2(t.w[k], t.w[k]), q01[o], acc);
            };
            const float2 z01 =
                tap01(2 * RG, RG > 0 ? a01[o][0] : make_float2(0.0f, 0.0f));
            out[o][0] = z01.x;
            out[o][1] = z01.y;
            out[o][2] = fmaf(t.w[2 * RG], q2[o], RG > 0 ? a2[o][0] : 0.0f);
            if (RG > 0) {
#pragma unroll
                for (int k = 0; k + 1 < 2 * RG; ++k) {
                    a01[o][k] = tap01(2 * RG - 1 - k, a01[o][k + 1]);
                    a2[o][k] = fmaf(t.w[2 * RG - 1 - k], q2[o], a2[o][k + 1]);
                }
                a01[o][K - 1] = tap01(0, make_float2(0.0f, 0.0f));
                a2[o][K - 1] = fmaf(t.w[0], q2[o], 0.0f);
            }
        }
    }
};

// Bounded wait, by thread 0, for the copies of planes i .. end - 1 that may
// still be in flight when a CTA stops early.
template <int NSTG>
__device__ __forceinline__ void drain(unsigned long long *bar, int i, int end) {
    for (int j = i; j < end; ++j) mbar_wait(bar + j % NSTG, (unsigned)(j / NSTG) & 1u);
}

// MSE: g = 2 (J - I) / N * grad I_m(phi) (pointwise, J and the gradient as
// the compose kernel stored them).
__global__ void __launch_bounds__(256) k_fused_mse_grad(const float *__restrict__ If,
                                                        const float *__restrict__ J,
                                                        const float *__restrict__ gJ,
                                                        float *__restrict__ g, int D, int H,
                                                        int W, int P) {
    int x = blockIdx.x * 32 + threadIdx.x;
    int y = blockIdx.y * 8 + threadIdx.y;
    int z = blockIdx.z;
    if (x >= W || y >= H) return;
    const long long N = (long long)D * H * P;  // rows of P elements
    const long long i = ((long long)z * H + y) * P + x;
    float dj = 2.0f * (__ldg(J + i) - __ldg(If + i)) / (float)((long long)D * H * W);
    g[i] = dj * __ldg(gJ + i);
    g[N + i] = dj * __ldg(gJ + N + i);
    g[2 * N + i] = dj * __ldg(gJ + 2 * N + i);
}

// Resident CTAs the register allocation of K3 and K4 aims at.
__host__ __device__ constexpr int k3_min_ctas(int RG, int NW, int OPT) {
    return RG <= 3 ? 32 / (NW * OPT) : 1;
}
__host__ __device__ constexpr int k4_min_ctas(int RG, int NW, int OPT) {
    return RG <= 3 ? (NW * OPT == 16 ? 2 : 3) : 1;
}

// ====================================================================== K3
// STAGED: the moments m, nu (FP32) arrive with the plane's TMA copies;
// otherwise (16-bit moments, or the per-thread copy variant) each thread loads
// its outputs' moments straight into registers one plane ahead.
template <int RG, int NW, int OPT, int NSTG, bool STAGED = true>
struct K3S {
    static constexpr int NT = FX * NW, TY = NW * OPT, RX = FX + 2 * RG, RY = TY + 2 * RG;
    static constexpr int XB = halo4(RG), BXW = FX + 2 * XB, COFF = XB - RG;
    static constexpr int NR = BXW * RY, NOUT = NT * OPT, XS = 3 * RY * FX;
    static constexpr size_t st_bytes = al128((size_t)3 * NR * 4);    // g
    static constexpr size_t ost_bytes = STAGED ? al128((size_t)6 * NOUT * 4) : 0;  // m, v
    static constexpr unsigned tx_plane = 3u * NR * 4, tx_out = 6u * NOUT * 4;
    static constexpr size_t o_st = 0;
    static constexpr size_t o_ost = o_st + st_bytes * NSTG;
    static constexpr size_t o_xb = o_ost + ost_bytes * NSTG;  // x sums, doubled
    static constexpr size_t o_bar = al128(o_xb + (size_t)2 * XS * 4);
    static constexpr size_t bytes = o_bar + 8 * NSTG;
};

// The body of K3 for the CTA with tile coordinates (bx, by, bz).  Between two
// barriers the CTA sums plane i along x and plane i - 1 along y and z.
template <int RG, int NW, int OPT, int NSTG, bool TMA, class TT, class TS>
__device__ __forceinline__ void smooth_adam_body(MapRef maps, const float *__restrict__ g,
                                                 TS *__restrict__ m, TS *__restrict__ v,
                                                 float *__restrict__ dir, WsHeader *__restrict__ h,
                                                 int D, int H, int W, int P, int TZ, const TT &t,
                                                 const AdamConsts ac, int parity, int bx, int by,
                                                 int bz) {
    constexpr bool S32 = sizeof(TS) == 4, STAGED = S32 && TMA;
    using S = K3S<RG, NW, OPT, NSTG, STAGED>;
    // moments as loaded into registers: FP32 values or 16-bit patterns
    using FT = typename std::conditional<S32, float, unsigned short>::type;
    constexpr int NT = S::NT, TY = S::TY, RX = S::RX, RY = S::RY, BXW = S::BXW, COFF = S::COFF,
                  XB = S::XB, NOUT = S::NOUT, XS = S::XS;
    using G = Region<RY, RX, NW, BXW, COFF>;
    extern __shared__ __align__(128) unsigned char smem[];
    float *xb = (float *)(smem + S::o_xb);
    unsigned long long *bar = (unsigned long long *)(smem + S::o_bar);
    __shared__ float redf[32];
    __shared__ int flag;
    auto stage = [&](int s) { return (float *)(smem + S::o_st + S::st_bytes * s); };
    auto ostage = [&](int s) { return (float *)(smem + S::o_ost + S::ost_bytes * s); };

    const int tx = threadIdx.x, wy = threadIdx.y, tid = wy * FX + tx;
    const int x0 = bx * FX, y0 = by * TY, z0 = bz * TZ;
    const int zend = min(z0 + TZ, D);
    const long long N = (long long)D * H * P, HW = (long long)H * P;  // channel, plane strides
    G rg;
    if (!TMA) rg.init(wy, tx, y0 - RG, x0 - RG, H, W, P);
    Outs<OPT, NW> ou;
    ou.init(wy, tx, y0, x0, H, W, P);
    if (TMA && tid == 0) {
        for (int k = 0; k < NSTG; ++k) mbar_init(bar + k);
        mbar_init_fence();
    }

    // group i: g of plane zs + i and the moments of the outputs that plane
    // i - 1 completes (plane zs + i - 1 - RG); the last group has no plane
    const int zs = z0 - RG, np = zend - z0 + 2 * RG;
    auto issue = [&](int i) {
        const int zp = zs + i, zo = zp - 1 - RG, s = i % NSTG;
        const bool in = i < np, out = STAGED && i <= np && zo >= z0;
        if (TMA) {
            if (tid == 0 && (in || out)) {
                mbar_expect(bar + s, (in ? S::tx_plane : 0u) + (out ? S::tx_out : 0u));
                if (in) tma4(stage(s), maps.a, x0 - XB, y0 - RG, zp, 0, bar + s);
                if (out) {
                    tma4(ostage(s), maps.b, x0, y0, zo, 0, bar + s);
                    tma4(ostage(s) + 3 * NOUT, maps.c, x0, y0, zo, 0, bar + s);
                }
            }
        } else {
            if (in) rg.template load<3>(stage(s), g, N, (long long)zp * HW, zp >= 0 && zp < D);
            cp_commit();
        }
    };
    const int groups = STAGED ? np + 1 : np;  // groups that copy something
    // unstaged moments of the next output plane, loaded one plane ahead
    FT mn[OPT][3], vn[OPT][3];
    auto fetch_mv = [&](int i) {
        if constexpr (!STAGED) {
            const int zo = zs + i - 1 - RG;
            if (i <= np && zo >= z0) {
                ou.fetch(mn, (const FT *)m, N, (long long)zo * HW);
                ou.fetch(vn, (const FT *)v, N, (long long)zo * HW);
            }
        }
    };
    // after the previous kernel: first copies and loads in flight, then the
    // status check
    pdl_wait();
    fetch_mv(1);
#pragma unroll
    for (int k = 0; k < NSTG; ++k) issue(k);
    if (status_timed_out(h, tid, &flag)) {
        drain_first<TMA, NSTG>(bar, groups, tid);
        return;
    }

    OpenZ<RG, OPT> oz;
    oz.init();
    float mx = 0.0f;
    bool bad = false;
    int fail = -1;
    for (int i = 0; i <= np; ++i) {
        const int zp = zs + i, s = i % NSTG;
        bool ok = true;
        if (TMA) {
            if (i < groups) ok = mbar_wait(bar + s, (unsigned)(i / NSTG) & 1u);
        } else {
            cp_wait<NSTG - 2>();
        }
        // also: the x pass reads neighbours' copies, the y pass their x sums,
        // and the stage of plane i - 1 is free
        if (__syncthreads_or(!ok)) {
            fail = i;
            break;
        }
        if (i > 0) issue(i + NSTG - 1);
        if (i < np && zp >= 0 && zp < D)
            gauss_x4<RG, 3, RY, BXW, COFF, NT>(stage(s), xb + (i & 1 ? XS : 0), t, tid);
        if (i == 0) continue;
        const int zq = zp - 1, zo = zq - RG;
        float2 q01[OPT];
        float q2[OPT];
        if (zq >= 0 && zq < D) {
            gauss_y3<RG, RY, OPT>(xb + (i & 1 ? 0 : XS), t, wy, tx, q01, q2);
        } else {
#pragma unroll
            for (int o = 0; o < OPT; ++o) {
                q01[o] = make_float2(0.0f, 0.0f);
                q2[o] = 0.0f;
            }
        }
        float sz[OPT][3];
        oz.push(t, q01, q2, sz);
        float mo[OPT][3], vo[OPT][3];
        if (zo >= z0) {
#pragma unroll
            for (int o = 0; o < OPT; ++o)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    if constexpr (STAGED) {
                        const float *od = ostage(s) + ou.place + o * FX;
                        mo[o][c] = od[c * NOUT];
                        vo[o][c] = od[(3 + c) * NOUT];
                    } else {
                        mo[o][c] = st_value<TS>(mn[o][c]);
                        vo[o][c] = st_value<TS>(vn[o][c]);
                    }
                }
        }
        fetch_mv(i + 1);
        if (zo >= z0) {
            const long long zoff = (long long)zo * HW;
#pragma unroll
            for (int o = 0; o < OPT; ++o) {
                if (ou.off[o] < 0) continue;
                const long long gi = zoff + ou.off[o];
                float nrm2 = 0.0f;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float sg = sz[o][c];
                    const float mvv = fmaf(ac.b1, mo[o][c], (1.0f - ac.b1) * sg);
                    const float vvv = fmaf(ac.b2, vo[o][c], (1.0f - ac.b2) * sg * sg);
                    m[c * N + gi] = st_store<TS>(mvv);
                    v[c * N + gi] = st_store<TS>(vvv);
                    const float dv = adam_dir(mvv, vvv, ac.rbc1, ac.rbc2, ac.eps);
                    dir[c * N + gi] = dv;
                    nrm2 = fmaf(dv, dv, nrm2);
                }
                if (nrm2 <= 3.4e38f)
                    mx = fmaxf(mx, sqrtf(nrm2));
                else
                    bad = true;
            }
        }
    }
    if (fail >= 0) {
        if (tid == 0) {
            status_set(&h->status, ST_TIMEOUT);
            drain<NSTG>(bar, fail, min(groups, fail + (fail ? NSTG - 1 : NSTG)));
        }
        return;
    }
    if (!TMA) cp_wait<0>();
    if (bad) status_set(&h->status, ST_NONFINITE);
    block_max_to(&h->step_max_bits[parity], mx, redf);
}

template <int RG, int NW, int OPT, int NSTG, bool TMA, class TS = float>
__global__ void __launch_bounds__(FX *NW, k3_min_ctas(RG, NW, OPT)) k_smooth_adam(const __grid_constant__ Maps maps,
                                                        const float *__restrict__ g,
                                                        TS *__restrict__ m,
                                                        TS *__restrict__ v,
                                                        float *__restrict__ dir,
                                                        WsHeader *__restrict__ h, int D, int H,
                                                        int W, int P, int TZ, GaussTaps t,
                                                        AdamConsts ac, int parity) {
    smooth_adam_body<RG, NW, OPT, NSTG, TMA>(map_ref(maps), g, m, v, dir, h, D, H, W, P, TZ, t, ac, parity,
                                             blockIdx.x, blockIdx.y, blockIdx.z);
}

// ====================================================================== K4
// SU: u is staged in shared memory (planes z-1..z+1, halo RG + 1); valid when
// the step is shorter than one voxel (lr / c_lp < 1).
// TU: storage of u (float, or __half for an FP16 u).
// The u tile's rows are 48 (or 64) elements long: an FP32 row is 16 banks
// (mod 32) long, so that the compose's reads of a neighbour row on either side
// of a lane's own voxel fall in the same bank, and an FP16 tile row starts on
// 16 bytes.  Its planes are whole multiples of 32 banks apart.
template <int RG, int NW, int OPT, bool SU, int NSTG, class TU = float>
struct K4S {
    static constexpr int NT = FX * NW, TY = NW * OPT, RX = FX + 2 * RG, RY = TY + 2 * RG;
    static constexpr int XB = halo4(RG), BXW = FX + 2 * XB, COFF = XB - RG;
    static constexpr int NR = BXW * RY;
    // u' and its x sums of a plane, doubled
    static constexpr int UPW = (RX + 3) / 4 * 4, NU = UPW * RY, XS = 3 * RY * FX;
    // u planes z-1, z, z+1 in use plus NSTG - 1 in flight, halo RG + 1
    static constexpr int EU = (int)sizeof(TU);
    static constexpr int URX = RX + 2, URY = RY + 2, UXB = (RG + 1 + 7) / 8 * 8,
                         UBXW = FX + 2 * UXB;
    static constexpr int UCOFF = UXB - RG - 1, NRU = UBXW * URY, NSU = NSTG + 2;
    static constexpr int NP = RY * RX, NJP = (NP + NT - 1) / NT;  // compose positions
    static constexpr size_t st_bytes = al128((size_t)3 * NR * 4);     // d
    static constexpr size_t ust_bytes = al128((size_t)3 * NRU * EU);  // u
    static constexpr unsigned tx_plane = 3u * NR * 4, tx_u = 3u * NRU * EU;
    static constexpr size_t o_st = 0;
    static constexpr size_t o_ust = o_st + st_bytes * NSTG;
    static constexpr size_t o_up = o_ust + (SU ? ust_bytes * NSU : 0);
    static constexpr size_t o_xb = o_up + (size_t)6 * NU * 4;
    static constexpr size_t o_bar = al128(o_xb + (size_t)2 * XS * 4);
    static constexpr size_t bytes = o_bar + 8 * (NSTG + 1);
    static_assert(EU == 2 || UBXW % 32 == 16 || UBXW % 32 == 0, "u rows of 16 or 32 banks");
};

// Compose position of slot pidx in the RY x RX region (RX = 32 + 2 RG): the
// first 32 RY slots are the region's first 32 columns row by row, so that a
// warp's positions lie in one row and its shared-memory reads and writes of
// them (d, the u cell corners, u') hit 32 consecutive words; the last 2 RG
// columns follow.
template <int RY, int RX>
__device__ __forceinline__ void compose_position(int pidx, int &ry, int &rx) {
    if (RX == 32 || pidx < 32 * RY) {
        ry = pidx >> 5;
        rx = pidx & 31;
    } else {
        const int e = pidx - 32 * RY;
        ry = e / (RX - 32);
        rx = 32 + e % (RX - 32);
    }
}

// The body of K4 for the CTA with tile coordinates (bx, by, bz); Im may be
// null (no image is warped).  Between two
// barriers the CTA composes plane i, sums plane i - 1 along x and plane i - 2
// along y and z, each from the half of a doubled buffer that the interval
// before filled.
template <int RG, int NW, int OPT, bool SU, int NSTG, bool TMA, class TT, class TU>
__device__ __forceinline__ void compose_body(MapRef maps, const TU *__restrict__ u,
                                             const float *__restrict__ dir,
                                             TU *__restrict__ uo,
                                             const float *__restrict__ Im,
                                             float *__restrict__ Jout, float *__restrict__ gJout,
                                             WsHeader *__restrict__ h, int D, int H, int W, int P,
                                             int TZ,
                                             const TT &t, float lr, float c_lp, int parity, int bx,
                                             int by, int bz) {
    static_assert(TMA || sizeof(TU) == 4, "an FP16 u is staged by tile copies only");
    using S = K4S<RG, NW, OPT, SU, NSTG, TU>;
    constexpr int NT = S::NT, TY = S::TY, RX = S::RX, RY = S::RY, BXW = S::BXW, COFF = S::COFF,
                  XB = S::XB, NR = S::NR, NU = S::NU, UPW = S::UPW, XS = S::XS, URX = S::URX,
                  URY = S::URY, UXB = S::UXB, UBXW = S::UBXW, UCOFF = S::UCOFF, NRU = S::NRU,
                  NSU = S::NSU, NP = S::NP, NJP = S::NJP;
    using G = Region<RY, RX, NW, BXW, COFF>;
    using GU = Region<URY, URX, NW, UBXW, UCOFF>;
    extern __shared__ __align__(128) unsigned char smem[];
    float *up = (float *)(smem + S::o_up);
    float *xb = (float *)(smem + S::o_xb);
    unsigned long long *bar = (unsigned long long *)(smem + S::o_bar);
    __shared__ int flag;
    auto stage = [&](int s) { return (float *)(smem + S::o_st + S::st_bytes * s); };

    const int tx = threadIdx.x, wy = threadIdx.y, tid = wy * FX + tx;
    const int x0 = bx * FX, y0 = by * TY, z0 = bz * TZ;
    const int zend = min(z0 + TZ, D);
    const long long N = (long long)D * H * P, HW = (long long)H * P;  // channel, plane strides
    G rg;
    GU rgu;
    if (!TMA) {
        rg.init(wy, tx, y0 - RG, x0 - RG, H, W, P);
        if (SU) rgu.init(wy, tx, y0 - RG - 1, x0 - RG - 1, H, W, P);
    }
    Outs<OPT, NW> ou;
    ou.init(wy, tx, y0, x0, H, W, P);
    if (TMA && tid == 0) {
        for (int k = 0; k <= NSTG; ++k) mbar_init(bar + k);
        mbar_init_fence();
    }

    const int zs = z0 - RG, np = zend - z0 + 2 * RG;
    // u plane q lives in u stage (q - (zs - 1)) % NSU
    auto uslot = [&](int q) {
        return (TU *)(smem + S::o_ust + S::ust_bytes * ((q - (zs - 1)) % NSU));
    };
    // group i: d plane zs + i and u plane zs + i + 1
    auto issue = [&](int i) {
        const int zp = zs + i, s = i % NSTG;
        if (TMA) {
            if (tid == 0 && i < np) {
                mbar_expect(bar + s, S::tx_plane + (SU ? S::tx_u : 0u));
                tma4(stage(s), maps.a, x0 - XB, y0 - RG, zp, 0, bar + s);
                if (SU) tma4(uslot(zp + 1), maps.b, x0 - UXB, y0 - RG - 1, zp + 1, 0, bar + s);
            }
        } else {
            if (i < np) {
                rg.template load<3>(stage(s), dir, N, (long long)zp * HW, zp >= 0 && zp < D);
                if constexpr (SU && sizeof(TU) == 4)
                    rgu.template load<3>(uslot(zp + 1), u, N, (long long)(zp + 1) * HW,
                                         zp + 1 >= 0 && zp + 1 < D);
            }
            cp_commit();
        }
    };
    // after the previous kernel: first copies and the step maximum in flight
    // together, then the status check
    pdl_wait();
    // u planes zs - 1 and zs: barrier NSTG (TMA), or cp.async group 0
    if (SU) {
        if (TMA) {
            if (tid == 0) {
                mbar_expect(bar + NSTG, 2u * S::tx_u);
                tma4(uslot(zs - 1), maps.b, x0 - UXB, y0 - RG - 1, zs - 1, 0, bar + NSTG);
                tma4(uslot(zs), maps.b, x0 - UXB, y0 - RG - 1, zs, 0, bar + NSTG);
            }
        } else if constexpr (sizeof(TU) == 4) {
            rgu.template load<3>(uslot(zs - 1), u, N, (long long)(zs - 1) * HW,
                                 zs - 1 >= 0 && zs - 1 < D);
            rgu.template load<3>(uslot(zs), u, N, (long long)zs * HW, zs >= 0 && zs < D);
        }
    }
#pragma unroll
    for (int k = 0; k < NSTG; ++k) issue(k);
    const float mxd = __uint_as_float(h->step_max_bits[parity]);
    if (status_timed_out(h, tid, &flag)) {
        if (SU && TMA && tid == 0) mbar_wait(bar + NSTG, 0u);
        drain_first<TMA, NSTG>(bar, np, tid);
        return;
    }
    const float e = (mxd > 0.0f) ? lr / (c_lp * mxd) : 0.0f;
    bool ok0 = true;
    if (SU && TMA) ok0 = mbar_wait(bar + NSTG, 0u);

    TriPending jp[OPT];
    long long jidx[OPT];
    bool jlive[OPT];
#pragma unroll
    for (int o = 0; o < OPT; ++o) jlive[o] = false;

    // this thread's compose positions (fixed for every plane): index in the d
    // stage (-1: none), in u' and in the u stage, and whether in the grid
    int pk[NJP], pup[NJP], pub[NJP];
    bool pin[NJP];
#pragma unroll
    for (int j = 0; j < NJP; ++j) {
        const int pidx = tid + j * NT;
        int ry, rx;
        compose_position<RY, RX>(pidx, ry, rx);
        const int y = y0 - RG + ry, x = x0 - RG + rx;
        pk[j] = pidx < NP ? ry * BXW + rx + COFF : -1;
        pin[j] = pidx < NP && y >= 0 && y < H && x >= 0 && x < W;
        pup[j] = ry * UPW + rx;
        pub[j] = (ry + 1) * UBXW + (rx + 1) + UCOFF;
    }

    OpenZ<RG, OPT> oz;
    oz.init();
    int fail = -1;
    for (int i = 0; i < np + 2; ++i) {
        const int zp = zs + i, s = i % NSTG;
        bool ok = ok0;
        if (TMA) {
            if (i < np) ok = mbar_wait(bar + s, (unsigned)(i / NSTG) & 1u) && ok;
        } else {
            cp_wait<NSTG - 2>();
        }
        // the stages hold neighbours' copies, u' and the x sums their results;
        // the stage of plane i - 1 is free
        if (__syncthreads_or(!ok)) {
            fail = i;
            break;
        }
        if (i > 0) issue(i + NSTG - 1);
        if (i < np && zp >= 0 && zp < D) {
            const float *ds = stage(s);
            float *us = up + (i & 1 ? 3 * NU : 0);
            const TU *um = uslot(zp - 1), *u0 = uslot(zp), *u1 = uslot(zp + 1);
            // u' on the RY x RX region (positions spread over all threads),
            // at the plane layout's columns
#pragma unroll
            for (int j = 0; j < NJP; ++j) {
                const int k = pk[j];
                if (NP % NT != 0 && k < 0) break;
                float a = 0.f, b = 0.f, c = 0.f;
                if (pin[j]) {
                    const float dz = -e * ds[k], dy = -e * ds[NR + k], dx = -e * ds[2 * NR + k];
                    if (SU) {
                        // cell corners lie within one voxel: planes zp-1..zp+1
                        if (dz > -1.0f && dz < 1.0f && dy > -1.0f && dy < 1.0f &&
                            dx > -1.0f && dx < 1.0f) {
                            // the corners are this voxel and its neighbours on
                            // the side of the step's sign, weighted by |delta|
                            // (the cell and weights of tri_issue_step3)
                            const float tz = fabsf(dz), ty = fabsf(dy), tx2 = fabsf(dx);
                            const TU *pa = u0, *pb = dz < 0.0f ? um : u1;
                            const int b0 = pub[j], oy = dy < 0.0f ? -UBXW : UBXW,
                                      ox = dx < 0.0f ? -1 : 1;
                            // channels 0 and 1 as a packed pair (each component
                            // exactly the scalar fadd / fmaf), channel 2 alone
                            auto pair = [&](const TU *P, int o) {
                                return make_float2(st_load(P[b0 + o]), st_load(P[NRU + b0 + o]));
                            };
                            auto lerp2 = [](float t, float2 lo, float2 hi) {
                                return __ffma2_rn(make_float2(t, t),
                                                  __fadd2_rn(hi, make_float2(-lo.x, -lo.y)), lo);
                            };
                            const float2 c00 = lerp2(tx2, pair(pa, 0), pair(pa, ox));
                            const float2 c01 = lerp2(tx2, pair(pa, oy), pair(pa, oy + ox));
                            const float2 c10 = lerp2(tx2, pair(pb, 0), pair(pb, ox));
                            const float2 c11 = lerp2(tx2, pair(pb, oy), pair(pb, oy + ox));
                            const float2 r01 = lerp2(tz, lerp2(ty, c00, c01), lerp2(ty, c10, c11));
                            const TU *Ap = pa + 2 * NRU + b0, *Bp = pb + 2 * NRU + b0;
                            const float A[2] = {st_load(Ap[0]), st_load(Ap[ox])},
                                        A2[2] = {st_load(Ap[oy]), st_load(Ap[oy + ox])},
                                        B[2] = {st_load(Bp[0]), st_load(Bp[ox])},
                                        B2[2] = {st_load(Bp[oy]), st_load(Bp[oy + ox])};
                            const float e00 = fmaf(tx2, A[1] - A[0], A[0]);
                            const float e01 = fmaf(tx2, A2[1] - A2[0], A2[0]);
                            const float e10 = fmaf(tx2, B[1] - B[0], B[0]);
                            const float e11 = fmaf(tx2, B2[1] - B2[0], B2[0]);
                            const float e0 = fmaf(ty, e01 - e00, e00);
                            const float e1 = fmaf(ty, e11 - e10, e10);
                            const float2 ab = __fadd2_rn(make_float2(dz, dy), r01);
                            a = ab.x;
                            b = ab.y;
                            c = dx + fmaf(tz, e1 - e0, e0);
                        } else {
                            a = b = c = __int_as_float(0x7fc00000);  // impossible step: flag it
                        }
                    } else {
                        int ry, rx;
                        compose_position<RY, RX>(tid + j * NT, ry, rx);
                        const int y = y0 - RG + ry, x = x0 - RG + rx;
                        float gz, gy, gx;
                        TriPending q[3];
                        tri_issue_step3(q, u, N, D, H, W, P, zp, y, x, dz, dy, dx);
                        a = dz + tri_finish<false>(q[0], gz, gy, gx);
                        b = dy + tri_finish<false>(q[1], gz, gy, gx);
                        c = dx + tri_finish<false>(q[2], gz, gy, gx);
                    }
                }
                us[pup[j]] = a;
                us[NU + pup[j]] = b;
                us[2 * NU + pup[j]] = c;
            }
        }
        if (i >= 1 && i <= np && zp - 1 >= 0 && zp - 1 < D)
            gauss_x4<RG, 3, RY, UPW, 0, NT>(up + (i & 1 ? 0 : 3 * NU), xb + (i & 1 ? 0 : XS), t,
                                            tid);
        if (i < 2) continue;
        const int zq = zp - 2, zo = zq - RG;
        float2 q01[OPT];
        float q2[OPT];
        if (zq >= 0 && zq < D) {
            gauss_y3<RG, RY, OPT>(xb + (i & 1 ? XS : 0), t, wy, tx, q01, q2);
        } else {
#pragma unroll
            for (int o = 0; o < OPT; ++o) {
                q01[o] = make_float2(0.0f, 0.0f);
                q2[o] = 0.0f;
            }
        }
        float sz[OPT][3];
        oz.push(t, q01, q2, sz);
        if (zo >= z0) {
            const long long zoff = (long long)zo * HW;
#pragma unroll
            for (int o = 0; o < OPT; ++o) {
                // finish the previous plane's warped value first (its loads have landed)
                if (jlive[o]) {
                    float gz, gy, gx;
                    Jout[jidx[o]] = tri_finish<true>(jp[o], gz, gy, gx);
                    gJout[jidx[o]] = gz;
                    gJout[N + jidx[o]] = gy;
                    gJout[2 * N + jidx[o]] = gx;
                    jlive[o] = false;
                }
                if (ou.off[o] < 0) continue;
                const long long gi = zoff + ou.off[o];
                const float a = sz[o][0], b = sz[o][1], c = sz[o][2];
                // the stored (for FP16, rounded) u is the one the next steps read
                const TU sa = st_store<TU>(a), sb = st_store<TU>(b), sc = st_store<TU>(c);
                uo[gi] = sa;
                uo[N + gi] = sb;
                uo[2 * N + gi] = sc;
                if (!Im) continue;
                tri_issue_p(jp[o], Im, D, H, W, P, zo, y0 + OPT * wy + o, x0 + tx, st_load(sa),
                            st_load(sb), st_load(sc));
                jidx[o] = gi;
                jlive[o] = true;
            }
        }
    }
    if (fail >= 0) {
        if (tid == 0) {
            status_set(&h->status, ST_TIMEOUT);
            if (SU && !ok0) mbar_wait(bar + NSTG, 0u);
            drain<NSTG>(bar, fail, min(np, fail + (fail ? NSTG - 1 : NSTG)));
        }
        return;
    }
#pragma unroll
    for (int o = 0; o < OPT; ++o)
        if (jlive[o]) {
            float gz, gy, gx;
            Jout[jidx[o]] = tri_finish<true>(jp[o], gz, gy, gx);
            gJout[jidx[o]] = gz;
            gJout[N + jidx[o]] = gy;
            gJout[2 * N + jidx[o]] = gx;
        }
    if (!TMA) cp_wait<0>();
    // per-iteration header fields for the next iteration (nobody else reads them now)
    if (bx == 0 && by == 0 && bz == 0 && tid == 0) {
        for (int c = 0; c < 8; ++c) h->coef_max_bits[c] = 0u;
        h->step_max_bits[parity ^ 1] = 0u;
        h->loss_acc = 0ull;
        h->eps_t = e;
    }
}

template <int RG, int NW, int OPT, bool SU, int NSTG, bool TMA, class TU = float>
__global__ void __launch_bounds__(FX *NW, k4_min_ctas(RG, NW, OPT)) k_compose(const __grid_constant__ Maps maps,
                                                    const TU *__restrict__ u,
                                                    const float *__restrict__ dir,
                                                    TU *__restrict__ uo,
                                                    const float *__restrict__ Im,
                                                    float *__restrict__ Jout,
                                                    float *__restrict__ gJout,
                                                    WsHeader *__restrict__ h, int D, int H, int W,
                                                    int P, int TZ, GaussTaps t, float lr,
                                                    float c_lp, int parity) {
    compose_body<RG, NW, OPT, SU, NSTG, TMA>(map_ref(maps), u, dir, uo, Im, Jout, gJout, h, D, H, W, P, TZ,
                                             t, lr, c_lp, parity, blockIdx.x, blockIdx.y,
                                             blockIdx.z);
}

// ================================================================ launch helpers

// Tile shapes (warps per CTA, rows per thread) of the 32 x 8 and 32 x 16
// tiles, and pipeline depths.  Measured on the 160 x 192 x 224 pair (ms): K3
// with 32 x 8 tiles 41.0, with 32 x 16 and two stages 40.5, three 39.6 (what
// the ring took holds the third stage); K4 with 16 warps of one row 40.6, with
// 8 warps of two rows 39.8; a third stage of K4 leaves one CTA per SM: 45.2.
// Before the passes were pipelined: 43.5.
constexpr int K3_NW = 8, K3_OPT = 1, K3W_NW = 8, K3W_OPT = 2, K3_ST = 3;
constexpr int K4_NW = 8, K4_OPT = 1, K4W_NW = 8, K4W_OPT = 2, K4_ST = 2;

// Gaussians up to this radius run inside the fused kernels
constexpr int kMaxFusedRG = kMaxFusedRadius;

}  // namespace

}  // namespace fa
