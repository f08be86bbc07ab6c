// Scatter of a field through trilinear weights in 64-bit fixed point.
#pragma once

#include "common.cuh"

namespace fa {

namespace {

constexpr int kFieldScatterBits = 40;  // |term| <= 2^40 of the largest: sums of 2^23 terms fit int64

__device__ __forceinline__ float2 scat_both(float a) { return make_float2(a, a); }

// rint of two values below 2^42 in magnitude as int64, the packed form of
// quantize: x = k 2^20 + l, k and l read from the bits of floats in
// [2^23, 2^24) together with their constant exponent bits.
__device__ __forceinline__ void quantize2(float2 x, long long q[2]) {
    const float2 h = __fadd2_rn(__fadd2_rn(x, scat_both(13194139533312.0f)),
                                scat_both(-13194139533312.0f));
    const float2 kf = __ffma2_rn(h, scat_both(9.5367431640625e-07f), scat_both(12582912.0f));
    const float2 lf =
        __fadd2_rn(__fadd2_rn(x, make_float2(-h.x, -h.y)), scat_both(12582912.0f));
    constexpr long long base = (0x4B400000ll << 20) + 0x4B400000ll;
    q[0] = (long long)__float_as_int(kf.x) * (1ll << 20) + __float_as_int(lf.x) - base;
    q[1] = (long long)__float_as_int(kf.y) * (1ll << 20) + __float_as_int(lf.y) - base;
}

// What is scattered: a finite value at a finite displacement below 2^20 voxels.
__device__ __forceinline__ bool scatter_takes(float uz, float uy, float ux, const float a[3]) {
    const float LIM = 1048576.0f;
    return fabsf(uz) < LIM && fabsf(uy) < LIM && fabsf(ux) < LIM && fabsf(a[0]) < 3.4e38f &&
           fabsf(a[1]) < 3.4e38f && fabsf(a[2]) < 3.4e38f;
}

// acc (three channels, N apart) += a times the weights of the corners of the
// cell (iz, iy, ix) at fractions t, for the lanes with `on`; corners outside
// the grid are dropped.  Every term is rounded on its own, so the sums do not
// depend on the order.  All 32 lanes of the warp call it, lane l + 1 one voxel
// further along x than lane l: where its cell is also one further along x
// (almost everywhere in a smooth field), it adds lane l's upper-x terms to its
// own lower-x ones first, which halves the adds that reach L2.
// Bound: the instructions that form the terms, and the latency of the adds.
// Carrying the upper-y terms to the next row as well (warps of up to 8 rows, a
// quarter of the adds) was no faster: a squaring's adjoint on 160 x 192 x 224
// took 265 us against 203, the one-channel scatter 90 against 87.
__device__ __forceinline__ void scatter_cell3(unsigned long long *acc, long long N, int D, int H,
                                              int W, int iz, int iy, int ix, float tz, float ty,
                                              float tx, const float a[3], float scale, bool on) {
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int pz = __shfl_up_sync(all, iz, 1), py = __shfl_up_sync(all, iy, 1),
              px = __shfl_up_sync(all, ix, 1), pon = __shfl_up_sync(all, (int)on, 1);
    const bool take = lane > 0 && on && pon && iz == pz && iy == py && ix == px + 1;
    const bool give = __shfl_down_sync(all, (int)take, 1) && lane < 31;
    const float wz[2] = {1.0f - tz, tz}, wy[2] = {1.0f - ty, ty}, wx[2] = {1.0f - tx, tx};
    const bool x0 = on && ix >= 0 && ix < W, x1 = on && !give && ix + 1 >= 0 && ix + 1 < W;
    const float2 a01 = make_float2(a[0], a[1]), s2 = scat_both(scale);
    unsigned long long *cell = acc + ((long long)iz * H + iy) * W + ix;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const bool zin = iz + p >= 0 && iz + p < D;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            unsigned long long *row = cell + (long long)p * H * W + (long long)q * W;
            const float wzy = wz[p] * wy[q], w0 = wzy * wx[0], w1 = wzy * wx[1];
            long long u[2], v[2], c[2];
            quantize2(__fmul2_rn(__fmul2_rn(a01, scat_both(w0)), s2), u);
            quantize2(__fmul2_rn(__fmul2_rn(a01, scat_both(w1)), s2), v);
            quantize2(__fmul2_rn(__fmul2_rn(scat_both(a[2]), make_float2(w0, w1)), s2), c);
            const long long f0 = __shfl_up_sync(all, v[0], 1), f1 = __shfl_up_sync(all, v[1], 1),
                            f2 = __shfl_up_sync(all, c[1], 1);
            if (take) {
                u[0] += f0;
                u[1] += f1;
                c[0] += f2;
            }
            const bool in = zin && iy + q >= 0 && iy + q < H;
            if (in && x0) {
                if (u[0]) atomicAdd(row, (unsigned long long)u[0]);
                if (u[1]) atomicAdd(row + N, (unsigned long long)u[1]);
                if (c[0]) atomicAdd(row + 2 * N, (unsigned long long)c[0]);
            }
            if (in && x1) {
                if (v[0]) atomicAdd(row + 1, (unsigned long long)v[0]);
                if (v[1]) atomicAdd(row + N + 1, (unsigned long long)v[1]);
                if (c[1]) atomicAdd(row + 2 * N + 1, (unsigned long long)c[1]);
            }
        }
    }
}

// The same for one channel (a finite, see the callers).
__device__ __forceinline__ void scatter_cell1(unsigned long long *acc, int D, int H, int W,
                                              int iz, int iy, int ix, float tz, float ty,
                                              float tx, float a, float scale, bool on) {
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int pz = __shfl_up_sync(all, iz, 1), py = __shfl_up_sync(all, iy, 1),
              px = __shfl_up_sync(all, ix, 1), pon = __shfl_up_sync(all, (int)on, 1);
    const bool take = lane > 0 && on && pon && iz == pz && iy == py && ix == px + 1;
    const bool give = __shfl_down_sync(all, (int)take, 1) && lane < 31;
    const float wz[2] = {1.0f - tz, tz}, wy[2] = {1.0f - ty, ty}, wx[2] = {1.0f - tx, tx};
    const bool x0 = on && ix >= 0 && ix < W, x1 = on && !give && ix + 1 >= 0 && ix + 1 < W;
    unsigned long long *cell = acc + ((long long)iz * H + iy) * W + ix;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const bool zin = iz + p >= 0 && iz + p < D;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            unsigned long long *row = cell + (long long)p * H * W + (long long)q * W;
            const float wzy = wz[p] * wy[q];
            long long c[2];
            quantize2(__fmul2_rn(__fmul2_rn(scat_both(a), make_float2(wzy * wx[0], wzy * wx[1])),
                                 scat_both(scale)),
                      c);
            const long long f = __shfl_up_sync(all, c[1], 1);
            if (take) c[0] += f;
            const bool in = zin && iy + q >= 0 && iy + q < H;
            if (in && x0 && c[0]) atomicAdd(row, (unsigned long long)c[0]);
            if (in && x1 && c[1]) atomicAdd(row + 1, (unsigned long long)c[1]);
        }
    }
}

}  // namespace

}  // namespace fa
