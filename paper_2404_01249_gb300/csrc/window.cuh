// LNCC window sums: the forward kernel (exact sums of the images' products,
// cc, the adjoint coefficients) and the gradient kernel (exact sums of the
// quantised coefficients, dL/dJ and g = dL/dJ grad I_m(phi)).  The
// registration loop (K1, K2), its lockstep batches and the loss as a layer
// of its own run these same bodies.
//
// A CTA owns a 32 x TY tile of (x, y) columns and marches a slab of TZ
// output planes along z.  The sums run z first: every thread owns up to PP
// of the tile's positions (halo included) for the whole march, loads its
// positions' values straight into registers one plane ahead, keeps their
// last 2R quantised values in a shared-memory ring that no other thread
// touches, and holds the running z sums in registers.  Only then do sums
// cross threads: the plane's z sums go to shared memory, one item sums 8
// outputs down a column, and each thread sums its two adjacent outputs along
// x into registers.  Integer sums are exact, so the order of the axes does
// not show in the result.
//
// Why this order: the 2R planes before a slab's first output only feed the
// z sums, so they cost neither the y and x passes nor a barrier (with x
// first, a slab of 2 planes ran 6 full planes); products are formed once per
// position instead of once per tap row; and a thread reads only what it
// loaded itself, so any row pitch or alignment takes the same path.  Against
// the x-first kernels on TMA tiles it replaced (same bits), windows of 5 on
// 160 x 192 x 224: forward 155 -> 116 us, gradient 143 -> 119; on 40 x 48 x 56
// 14 -> 9 and 12 -> 7 us; windows of 7 on 128 x 256 x 256: 215 -> 155 and
// 250 -> 205 us; the loss with both gradients as a layer on 127 x 181 x 159:
// 691 -> 227 us, and at windows of 9, 11, 13 and 15 there 885 -> 351, 999 -> 408,
// 1,105 -> 467 and 1,222 -> 532; ten iterations on 96 x 112 x 104 at these windows
// 2,078 -> 1,477, 2,645 -> 1,652, 3,194 -> 1,970 and 3,575 -> 2,137 us.
//
// What bounds them: latency at 16 warps per SM (2.0 and 1.5 warp instructions
// per clock and SM, no pipe above half of its rate).  24 warps at 80
// registers measured no faster (spills and register moves add what the extra
// warps hide: 123 against 116 us), nor did 32 x 8 tiles (150 us).
#pragma once

#include "common.cuh"
#include "ops.h"

namespace fa {

namespace {

constexpr int FX = 32;  // tile width along x (one warp)

// Programmatic dependent launch: a kernel's CTAs may start while the previous
// kernel in the stream finishes.  Everything before pdl_wait() touches no
// data the previous kernel writes; pdl_wait() returns once that kernel has
// completed and its writes are visible.  pdl_trigger() lets the next kernel
// begin launching once every CTA of this one has started.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

// Tile of windows of radius R.  16 rows per tile (1.41 positions per output
// at R = 2, 8 rows: 1.69); 8 rows for windows above 7, whose rings of 16 rows
// would not fit.
template <int R>
struct WinTile {
    static constexpr int TY = R <= 3 ? 16 : 8, NT = 16 * TY;
    static constexpr int RX = FX + 2 * R, RY = TY + 2 * R, NPOS = RX * RY;
    static constexpr int PP = (NPOS + NT - 1) / NT;  // positions per thread
    static constexpr int NPAD = PP * NT;             // their slots in shared memory
    static constexpr int CG = TY / 8;                // column items per column
};

// RZ, the radius along z of the bodies below, is R, or 0 for a volume of one
// plane: there the windows' other planes add nothing, and the march of 2 R + 1
// planes with its ring is left out (1 x 1024 x 1024, both gradients: windows of 9
// to 15 294, 381, 447 and 543 us marching, 96, 109, 130 and 137 so; 249, 279, 302 and 326
// before the sums ran z first).

// What a slab costs beyond its output planes, in output planes: the 2R planes
// before its first output take the z sums only (about a third of a plane).
__host__ __device__ constexpr float window_slab_extra(int R) { return 1.0f + 0.35f * 2 * R; }

// Resident CTAs the register allocation aims at.
__host__ __device__ constexpr int fwd_min_ctas(int R) { return R <= 3 ? 2 : 1; }
__host__ __device__ constexpr int grad_min_ctas(int R) { return R <= 3 ? 2 : 1; }

// A thread's positions.  One outside the grid reads its nearest voxel inside
// (which every window that holds the position holds too) and is masked to
// zero, so that no load is conditional.  Offsets are from the plane's base,
// which is the same for the whole CTA.
template <int R>
struct WinPos {
    using G = WinTile<R>;
    unsigned off[G::PP];
    float in[G::PP];  // 1 inside the grid, 0 outside
    __device__ __forceinline__ void init(int tid, int x0, int y0, int H, int W, int P) {
#pragma unroll
        for (int j = 0; j < G::PP; ++j) {
            const int k = tid + j * G::NT, ry = k / G::RX, rx = k - ry * G::RX;
            const int y = y0 - R + ry, x = x0 - R + rx;
            const int yc = min(max(y, 0), H - 1), xc = min(max(x, 0), W - 1);
            off[j] = (unsigned)(yc * P + xc);
            in[j] = k < G::NPOS && y == yc && x == xc ? 1.0f : 0.0f;
        }
    }
    __device__ __forceinline__ void load(float (&v)[G::PP], const float *__restrict__ plane) const {
#pragma unroll
        for (int j = 0; j < G::PP; ++j)
            v[j] = __ldg(plane + off[j]);
    }
};

__device__ __forceinline__ float2 both2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }

// The float-float steps of common.cuh on two voxels at once (packed FP32:
// each component is exactly the scalar operation).
__device__ __forceinline__ void ff2_mul(float2 a, float2 xh, float2 xl, float2 &h, float2 &l) {
    h = __fmul2_rn(a, xh);
    l = __ffma2_rn(a, xh, neg2(h));
    l = __ffma2_rn(a, xl, l);
}
__device__ __forceinline__ void ff2_add(float2 &h, float2 &l, float2 bh, float2 bl) {
    const float2 s = __fadd2_rn(h, bh), bb = sub2(s, h);
    float2 e = __fadd2_rn(sub2(h, sub2(s, bb)), sub2(bh, bb));
    e = __fadd2_rn(e, __fadd2_rn(l, bl));
    h = __fadd2_rn(s, e);
    l = sub2(e, sub2(h, s));
}
// Two int64 below 2^48 in magnitude -> float-float times scale (a power of two).
__device__ __forceinline__ void i64x2_to_ff(const long long x[2], float scale, float2 &hi,
                                            float2 &lo) {
    const float2 fh = __fmul2_rn(make_float2(__int2float_rn((int)(x[0] >> 24)),
                                             __int2float_rn((int)(x[1] >> 24))),
                                 both2(16777216.0f));
    const float2 fl = make_float2(__uint2float_rn((unsigned)x[0] & 0xFFFFFFu),
                                  __uint2float_rn((unsigned)x[1] & 0xFFFFFFu));
    hi = __fadd2_rn(fh, fl);
    lo = __fmul2_rn(sub2(fl, sub2(hi, fh)), both2(scale));
    hi = __fmul2_rn(hi, both2(scale));
}
// lncc_c_ff of two voxels: C = -(A S_I + 2 B S_J) / n as a float-float pair.
__device__ __forceinline__ void lncc_c_ff2(float2 A, float2 B, const long long sI[2],
                                           const long long sJ[2], float inv_s, float nf,
                                           float inv_nf, float2 &ch, float2 &cl) {
    const float2 n2 = both2(nf), r2 = both2(inv_nf);
    float2 ih, il, jh, jl;
    i64x2_to_ff(sI, inv_s, ih, il);
    i64x2_to_ff(sJ, inv_s, jh, jl);
    const float2 i1 = __fmul2_rn(ih, r2),
                 i2 = __fmul2_rn(__fadd2_rn(__ffma2_rn(neg2(i1), n2, ih), il), r2);
    const float2 j1 = __fmul2_rn(jh, r2),
                 j2 = __fmul2_rn(__fadd2_rn(__ffma2_rn(neg2(j1), n2, jh), jl), r2);
    float2 ph, pl, th, tl;
    ff2_mul(A, i1, i2, ph, pl);
    ff2_mul(__fadd2_rn(B, B), j1, j2, th, tl);
    ff2_add(ph, pl, th, tl);
    ch = neg2(ph);
    cl = neg2(pl);
}

// rint(x) = k 2^RB + l of two values |x| < 2^(RB + 22), read from the bits of
// floats in [2^23, 2^24): k and l come with kLimbBits added.
constexpr unsigned kLimbBits = 0x4B400000u;  // the bits of 1.5 2^23
template <int RB>
__device__ __forceinline__ void split_limbs(float2 x, unsigned k[2], unsigned l[2]) {
    constexpr float M = 12582912.0f * (float)(1 << RB), M23 = 12582912.0f;
    const float2 h = __fadd2_rn(__fadd2_rn(x, both2(M)), both2(-M));
    const float2 kf = __ffma2_rn(h, both2(1.0f / (float)(1 << RB)), both2(M23));
    const float2 lf = __fadd2_rn(sub2(x, h), both2(M23));
    k[0] = __float_as_uint(kf.x);
    k[1] = __float_as_uint(kf.y);
    l[0] = __float_as_uint(lf.x);
    l[1] = __float_as_uint(lf.y);
}

// A 2-limb sum: the value is k 2^RB + l with 32-bit limbs that wrap.
struct Limb2 {
    unsigned l, k;
};
__device__ __forceinline__ Limb2 operator+(Limb2 a, Limb2 b) { return Limb2{a.l + b.l, a.k + b.k}; }
__device__ __forceinline__ Limb2 operator-(Limb2 a, Limb2 b) { return Limb2{a.l - b.l, a.k - b.k}; }

// y pass: zs [NCH][NPAD] (rows of RX) -> ys [NCH][TY][RX], 8 outputs of one column per
// item from 8 + 2R reads.
template <int R, int NCH, class T>
__device__ __forceinline__ void win_columns(const T *zs, T *ys, int tid) {
    using G = WinTile<R>;
    constexpr int ITEMS = NCH * G::CG * G::RX;
#pragma unroll
    for (int j = 0; j < (ITEMS + G::NT - 1) / G::NT; ++j) {
        const int it = tid + j * G::NT;
        if (ITEMS % G::NT != 0 && it >= ITEMS) break;
        const int x = it % G::RX, rest = it / G::RX, cg = rest % G::CG, c = rest / G::CG;
        const T *p = zs + c * G::NPAD + cg * 8 * G::RX + x;
        T *q = ys + (c * G::TY + cg * 8) * G::RX + x;
        T v[8 + 2 * R];
#pragma unroll
        for (int t = 0; t < 8 + 2 * R; ++t) v[t] = p[t * G::RX];
        T a = v[0];
#pragma unroll
        for (int t = 1; t <= 2 * R; ++t) a = a + v[t];
        q[0] = a;
#pragma unroll
        for (int t = 1; t < 8; ++t) {
            a = a + (v[t + 2 * R] - v[t - 1]);
            q[t * G::RX] = a;
        }
    }
}

// x pass of channel c for this thread's two outputs (row, 2 pair), (row, 2 pair + 1).
template <int R, class T>
__device__ __forceinline__ void win_row(const T *ys, int c, int row, int pair, T out[2]) {
    using G = WinTile<R>;
    static_assert(sizeof(T) == 8, "two values per 16-byte load");
    union Pair {
        uint4 q;
        T v[2];
        __device__ Pair() {}
    } p[R + 1];
    const uint4 *src = (const uint4 *)(ys + (c * G::TY + row) * G::RX + 2 * pair);
#pragma unroll
    for (int t = 0; t <= R; ++t) p[t].q = src[t];
    if (R == 0) {
        out[0] = p[0].v[0];
        out[1] = p[0].v[1];
        return;
    }
    T a = p[0].v[1];  // the 2R values both windows hold
#pragma unroll
    for (int t = 2; t <= 2 * R; ++t) a = a + p[t / 2].v[t & 1];
    out[0] = a + p[0].v[0];
    out[1] = a + p[R].v[1];
}

// Two adjacent values of a row.
template <class T>
struct alignas(2 * sizeof(T)) Two {
    T a, b;
};
// K channels of them (N apart): in one access each where `vec` (the row pitch
// keeps them aligned and both lie in the grid), else the first and, if `both`,
// the second.  The choice is one branch for all channels.
template <int K, class T>
__device__ __forceinline__ void load2(Two<T> (&v)[K], const T *__restrict__ p, long long N,
                                      bool both, bool vec) {
    if (vec) {
#pragma unroll
        for (int c = 0; c < K; ++c) v[c] = *(const Two<T> *)(p + c * N);
    } else {
#pragma unroll
        for (int c = 0; c < K; ++c) {
            v[c].a = p[c * N];
            v[c].b = both ? p[c * N + 1] : T(0);
        }
    }
}
template <int K>
__device__ __forceinline__ void store2(float *p, long long N, const float2 (&v)[K], bool both,
                                       bool vec) {
    if (vec) {
#pragma unroll
        for (int c = 0; c < K; ++c) *(float2 *)(p + c * N) = v[c];
    } else {
#pragma unroll
        for (int c = 0; c < K; ++c) {
            p[c * N] = v[c].x;
            if (both) p[c * N + 1] = v[c].y;
        }
    }
}

// ============================================================== forward (K1)
constexpr int fwd_channels(FwdMode m) { return m == kFwdGiven ? 3 : (m == kFwdBoth ? 5 : 2); }

template <int R, FwdMode M, int RZ = R>
struct FwdSmem {
    using G = WinTile<R>;
    static constexpr int NCH = fwd_channels(M);
    static constexpr int HS = 2 * RZ;  // planes the ring holds
    static constexpr size_t ring = (size_t)HS * G::NPAD * (M == kFwdStats ? 4 : 8);
    static constexpr size_t o_zs = (ring + 15) / 16 * 16;
    static constexpr size_t o_ys = o_zs + (size_t)NCH * G::NPAD * 8;
    static constexpr size_t bytes = o_ys + (size_t)NCH * G::TY * G::RX * 8;
    static_assert(bytes + 512 <= 227 * 1024, "a CTA's shared memory");
};

template <int R, FwdMode M, int RZ = R>
__device__ __forceinline__ void lncc_fwd_body(const FwdArgs &g, int bx, int by, int bz) {
    using G = WinTile<R>;
    using S = FwdSmem<R, M, RZ>;
    constexpr int NT = G::NT, PP = G::PP, NPAD = G::NPAD, HS = S::HS, NCH = S::NCH;
    constexpr bool HASJ = M != kFwdStats;
    extern __shared__ __align__(128) unsigned char smem[];
    int2 *ring2 = (int2 *)smem;  // [HS][NPAD]: q_I, q_J
    int *ring1 = (int *)smem;    // kFwdStats: q_I
    long long *zs = (long long *)(smem + S::o_zs), *ys = (long long *)(smem + S::o_ys);
    __shared__ float redf[32];
    __shared__ unsigned long long redu[32];

    const int tid = threadIdx.x, row = tid >> 4, pair = tid & 15;
    const int x0 = bx * FX, y0 = by * G::TY, z0 = bz * g.TZ;
    const int zend = min(z0 + g.TZ, g.D);
    const long long HW = (long long)g.H * g.P, N = HW * g.D;
    const int zs0 = z0 - RZ, np = zend - z0 + 2 * RZ;
    WinPos<R> wp;
    wp.init(tid, x0, y0, g.H, g.W, g.P);
    const int ox = x0 + 2 * pair, oy = y0 + row;
    const bool live = oy < g.H && ox < g.W, both = ox + 1 < g.W, vec = both && (g.P & 1) == 0;
    const unsigned ooff = (unsigned)(oy * g.P + ox);
    const long long n = (long long)g.window * g.window * g.window;
    const float nf = (float)n, inv_nf = 1.0f / nf;

    pdl_wait();
    float fI[PP], fJ[PP];
    auto fetch = [&](int i) {  // a plane outside the grid loads the nearest one, unused
        const long long o = (long long)min(max(zs0 + i, 0), g.D - 1) * HW;
        wp.load(fI, g.I + o);
        if (HASJ) wp.load(fJ, g.J + o);
    };
    fetch(0);
    const float amax =
        fmaxf(__uint_as_float(g.h->absmax_bits[0]), __uint_as_float(g.h->absmax_bits[1]));
    pdl_trigger();
    const int sh = fixed_shift(amax, g.bits);
    const float scale = pow2f(sh), inv_s = pow2f(-sh);
#pragma unroll
    for (int j = 0; j < PP; ++j) wp.in[j] *= scale;

    // running z sums of this thread's positions (the sums of q stay below 2^31)
    int aI[PP], aJ[PP];
    long long aII[PP], aJJ[PP], aIJ[PP];
#pragma unroll
    for (int j = 0; j < PP; ++j) {
        aI[j] = aJ[j] = 0;
        aII[j] = aJJ[j] = aIJ[j] = 0;
    }
    // sum of rint(cc 2^32) in limbs of 20 bits (kLimbBits added per term)
    unsigned ccl = 0u, cck = 0u, terms = 0u;
    float mx[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    bool bad = false;
    int slot = 0;
    for (int i = 0; i < np; ++i) {
        const int zp = zs0 + i;
        const bool emit = i >= HS;
        int qi[PP], qj[PP];
        if (zp >= 0 && zp < g.D) {
#pragma unroll
            for (int j = 0; j < PP; ++j) {
                qi[j] = __float2int_rn(fI[j] * wp.in[j]);
                qj[j] = HASJ ? __float2int_rn(fJ[j] * wp.in[j]) : 0;
            }
        } else {
#pragma unroll
            for (int j = 0; j < PP; ++j) qi[j] = qj[j] = 0;
        }
        fetch(i + 1);
        Two<long long> sI2[1] = {{0, 0}};
        Two<float> vI2[1] = {{0.f, 0.f}};
        const long long zo = (long long)(zp - RZ) * HW;
        if (M == kFwdGiven && emit && live) {
            load2(sI2, g.SI + zo + ooff, N, both, vec);
            load2(vI2, g.varI + zo + ooff, N, both, vec);
        }
#pragma unroll
        for (int j = 0; j < PP; ++j) {
            const int k = tid + j * NT;
            if (M != kFwdGiven) {
                aI[j] += qi[j];
                aII[j] += (long long)qi[j] * qi[j];
            }
            if (HASJ) {
                aJ[j] += qj[j];
                aJJ[j] += (long long)qj[j] * qj[j];
                aIJ[j] += (long long)qi[j] * qj[j];
            }
            if (emit) {
                if (M == kFwdStats) {
                    zs[k] = aI[j];
                    zs[NPAD + k] = aII[j];
                } else {
                    zs[k] = aJ[j];
                    zs[NPAD + k] = aJJ[j];
                    zs[2 * NPAD + k] = aIJ[j];
                    if (M == kFwdBoth) {
                        zs[3 * NPAD + k] = aI[j];
                        zs[4 * NPAD + k] = aII[j];
                    }
                }
                int oi, oj = 0;  // the plane that leaves the window
                if (HS == 0) {
                    oi = qi[j];
                    oj = qj[j];
                } else if (HASJ) {
                    const int2 o = ring2[slot * NPAD + k];
                    oi = o.x;
                    oj = o.y;
                } else {
                    oi = ring1[slot * NPAD + k];
                }
                if (M != kFwdGiven) {
                    aI[j] -= oi;
                    aII[j] += (long long)-oi * oi;
                }
                if (HASJ) {
                    aJ[j] -= oj;
                    aJJ[j] += (long long)-oj * oj;
                    aIJ[j] += (long long)-oj * oi;
                }
            }
            if (HS > 0) {
                if (HASJ)
                    ring2[slot * NPAD + k] = make_int2(qi[j], qj[j]);
                else
                    ring1[slot * NPAD + k] = qi[j];
            }
        }
        slot = slot + 1 >= HS ? 0 : slot + 1;
        if (!emit) continue;
        __syncthreads();
        win_columns<R, NCH>(zs, ys, tid);
        __syncthreads();
        long long w[NCH][2];
#pragma unroll
        for (int c = 0; c < NCH; ++c) win_row<R>(ys, c, row, pair, w[c]);
        if (!live) continue;
        // numerators are n^2 2^(2s) times the statistic: scaled by 2^-s twice
        // (exact) and divided by n once (one rounding)
        auto scaled = [&](float2 v) {
            return __fmul2_rn(__fmul2_rn(__fmul2_rn(v, both2(inv_s)), both2(inv_s)),
                              both2(inv_nf));
        };
        auto variance = [&](const long long a[2], const long long b[2]) {
            return scaled(make_float2(diff_i128_to_float<true>(n, a[0], b[0], b[0]),
                                      diff_i128_to_float<true>(n, a[1], b[1], b[1])));
        };
        if (M == kFwdStats) {
            const float2 v = variance(w[1], w[0]);
            long long *sp = g.SI + zo + ooff;
            if (vec) {
                *(Two<long long> *)sp = Two<long long>{w[0][0], w[0][1]};
            } else {
                sp[0] = w[0][0];
                if (both) sp[1] = w[0][1];
            }
            const float2 vv[1] = {v};
            store2(g.varI + zo + ooff, N, vv, both, vec);
            continue;
        }
        // the second voxel of a row's end outside the grid: its window sums
        // are finite like any other's, its results are dropped
        const long long *sJ = w[0], *sJJ = w[NCH > 1 ? 1 : 0], *sIJ = w[NCH > 2 ? 2 : 0];
        long long sI[2];
        float2 varI;
        if (M == kFwdBoth) {
            sI[0] = w[NCH - 2][0];
            sI[1] = w[NCH - 2][1];
            varI = variance(w[NCH - 1], sI);
        } else {
            sI[0] = sI2[0].a;
            sI[1] = sI2[0].b;
            varI = make_float2(vI2[0].a, vI2[0].b);
        }
        const float2 varJ = variance(sJJ, sJ);
        const float2 cross = scaled(make_float2(diff_i128_to_float(n, sIJ[0], sI[0], sJ[0]),
                                                diff_i128_to_float(n, sIJ[1], sI[1], sJ[1])));
        const float2 den = __ffma2_rn(varI, varJ, both2(g.cc_eps));
        const float2 rden = make_float2(__frcp_rn(den.x), __frcp_rn(den.y));
        const float2 cc = __fmul2_rn(__fmul2_rn(cross, cross), rden);
        const bool ok0 = cc.x >= 0.0f && cc.x <= 2.0f, ok1 = both && cc.y >= 0.0f && cc.y <= 2.0f;
        bad = bad || !ok0 || (both && !ok1);
        {
            unsigned k[2], l[2];
            split_limbs<20>(
                __fmul2_rn(make_float2(ok0 ? cc.x : 0.0f, ok1 ? cc.y : 0.0f), both2(4294967296.0f)),
                k, l);
            cck += k[0] + k[1];
            ccl += l[0] + l[1];
            terms += 2u;
        }
        if (!g.write_coef) continue;
        const float2 A = __fmul2_rn(__fmul2_rn(both2(2.0f), cross), rden);
        const float2 B = __fmul2_rn(__fmul2_rn(neg2(cc), varI), rden);
        float2 Ch, Cl;
        lncc_c_ff2(A, B, sI, sJ, inv_s, nf, inv_nf, Ch, Cl);
        auto keep = [&](int c, float2 v) {
            mx[c] = fmaxf(mx[c], fmaxf(fabsf(v.x), both ? fabsf(v.y) : 0.0f));
        };
        keep(0, A);
        keep(1, B);
        keep(2, Ch);
        float *cp = g.coef + zo + ooff;
        const float2 out[4] = {A, B, Ch, Cl};
        store2(cp, N, out, both, vec);
        if (M == kFwdBoth && g.want_dI) {
            const float2 Bp = __fmul2_rn(__fmul2_rn(neg2(cc), varJ), rden);
            lncc_c_ff2(A, Bp, sJ, sI, inv_s, nf, inv_nf, Ch, Cl);
            keep(3, Bp);
            keep(4, Ch);
            const float2 out2[3] = {Bp, Ch, Cl};
            store2(cp + 4 * N, N, out2, both, vec);
        }
    }
    if (M == kFwdStats) return;
    if (bad) status_set(&g.h->status, ST_NONFINITE);
    const unsigned base = kLimbBits * terms;
    const long long qcc = ((long long)(int)(cck - base) << 20) + (int)(ccl - base);
    block_sum_to(&g.h->loss_acc, (unsigned long long)qcc, redu);
    if (g.write_coef) {
        constexpr int NM = M == kFwdBoth ? 5 : 3;
#pragma unroll
        for (int c = 0; c < NM; ++c) block_max_to(&g.h->coef_max_bits[c], mx[c], redf);
    }
}

template <int R, FwdMode M, int RZ = R>
__global__ void __launch_bounds__(WinTile<R>::NT, fwd_min_ctas(R)) k_lncc_fwd(const __grid_constant__ FwdArgs g) {
    lncc_fwd_body<R, M, RZ>(g, blockIdx.x, blockIdx.y, blockIdx.z);
}

// ============================================================= gradient (K2)
// Coefficients are quantised against their maxima and split into limbs,
// rint(v 2^e) = k 2^RB + l, that are summed apart: 32-bit adds without
// carries, and no recombination per position.  RB is chosen so that neither
// sum of n terms (two per voxel for the float-float C) leaves 32 bits:
// RB = 20 up to 11^3 terms, 18 for 13^3 and 15^3.  The limbs are read from
// the bits of floats in [2^23, 2^24) (adding 1.5 2^23 rounds to an integer);
// the constant exponent bits are added along with them and n of them are
// subtracted from the finished sum (all arithmetic is modulo 2^32).
template <int R, int RZ = R>
struct GradTile {
    using G = WinTile<R>;
    static constexpr int HS = 2 * RZ;  // planes between a plane's coming and leaving
    static constexpr int RB = R <= 5 ? 20 : 18;
    // windows of 13 and 15: the ring would not fit, so the plane that leaves
    // the window is loaded and quantised again
    static constexpr bool RING = R <= 5 && RZ > 0;
    static constexpr size_t ring = RING ? (size_t)HS * G::NPAD * 3 * 8 : 0;  // [HS][3][NPAD]
    static constexpr size_t o_zs = (ring + 15) / 16 * 16;
    static constexpr size_t o_ys = o_zs + (size_t)3 * G::NPAD * 8;
    static constexpr size_t bytes = o_ys + (size_t)3 * G::TY * G::RX * 8;
    static_assert(bytes + 512 <= 227 * 1024, "a CTA's shared memory");
};

template <int R, bool SWAP, int RZ = R>
__device__ __forceinline__ void lncc_grad_body(const GradArgs &g, int bx, int by, int bz) {
    using G = WinTile<R>;
    using S = GradTile<R, RZ>;
    constexpr int NT = G::NT, PP = G::PP, NPAD = G::NPAD, HS = S::HS;
    constexpr int CB = SWAP ? 4 : 1;  // channel of B; C hi and lo follow
    extern __shared__ __align__(128) unsigned char smem[];
    Limb2 *ring = (Limb2 *)smem;
    Limb2 *zs = (Limb2 *)(smem + S::o_zs), *ys = (Limb2 *)(smem + S::o_ys);

    const int tid = threadIdx.x, row = tid >> 4, pair = tid & 15;
    const int x0 = bx * FX, y0 = by * G::TY, z0 = bz * g.TZ;
    const int zend = min(z0 + g.TZ, g.D);
    const long long HW = (long long)g.H * g.P, N = HW * g.D;
    const int zs0 = z0 - RZ, np = zend - z0 + 2 * RZ;
    WinPos<R> wp;
    wp.init(tid, x0, y0, g.H, g.W, g.P);
    const int ox = x0 + 2 * pair, oy = y0 + row;
    const bool live = oy < g.H && ox < g.W, both = ox + 1 < g.W, vec = both && (g.P & 1) == 0;
    const unsigned ooff = (unsigned)(oy * g.P + ox);
    const float inv_n = 1.0f / (float)((long long)g.D * g.H * g.W);  // 1 / voxel count

    pdl_wait();
    struct Raw {
        float A[PP], B[PP], C[PP], L[PP];
    };
    Raw cur;
    auto fetch = [&](Raw &f, int i) {  // a plane outside the grid loads the nearest one
        const float *p = g.coef + (long long)min(max(zs0 + i, 0), g.D - 1) * HW;
        wp.load(f.A, p);
        wp.load(f.B, p + CB * N);
        wp.load(f.C, p + (CB + 1) * N);
        wp.load(f.L, p + (CB + 2) * N);
    };
    fetch(cur, 0);
    float qs[3], us[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int e = fixed_shift(
            __uint_as_float(g.h->coef_max_bits[SWAP && c > 0 ? c + 2 : c]), g.cbits);
        qs[c] = pow2f(e);
        us[c] = pow2f(-e);
    }
    pdl_trigger();

    Limb2 acc[PP][3];
#pragma unroll
    for (int j = 0; j < PP; ++j)
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[j][c] = Limb2{0u, 0u};
    // The line this thread asks L2 for kAhead planes ahead of its use (a row's
    // half of one coefficient, or a row of an output operand), on plane 0.
    constexpr int kAhead = 4;
    const float *line = nullptr;
    if (tid < 8 * G::RY) {
        const int c = (tid >> 1) & 3, y = min(max(y0 - R + (tid >> 3), 0), g.H - 1),
                  x = min(max(x0 - R + 32 * (tid & 1), 0), g.W - 1);
        line = g.coef + (c ? (CB + c - 1) * N : 0) + (long long)y * g.P + x;
    } else if (tid - 8 * G::RY < 5 * G::TY) {
        const int c = (tid - 8 * G::RY) / G::TY, y = min(y0 + (tid - 8 * G::RY) % G::TY, g.H - 1);
        const float *p = c == 0 ? g.I : (c == 1 ? g.J : (g.g ? g.gJ + (c - 2) * N : nullptr));
        if (p) line = p + (long long)y * g.P + x0;
    }
    auto ask = [&](int i) {
        const int z = zs0 + i + kAhead;
        if (line && z >= 0 && z < min(zend + RZ, g.D))
            asm volatile("prefetch.global.L2 [%0];" ::"l"(line + (long long)z * HW));
    };
    auto quant = [&](const Raw &f, int i, Limb2 (&q)[PP][3]) {
        const bool zin = zs0 + i >= 0 && zs0 + i < g.D;
        const float2 s01 = zin ? make_float2(qs[0], qs[1]) : both2(0.0f);
        const float2 s22 = both2(zin ? qs[2] : 0.0f);
#pragma unroll
        for (int j = 0; j < PP; ++j) {
            const float2 m = both2(wp.in[j]);
            unsigned k[2], l[2];
            split_limbs<S::RB>(__fmul2_rn(__fmul2_rn(make_float2(f.A[j], f.B[j]), m), s01), k, l);
            q[j][0] = Limb2{l[0], k[0]};
            q[j][1] = Limb2{l[1], k[1]};
            split_limbs<S::RB>(__fmul2_rn(__fmul2_rn(make_float2(f.C[j], f.L[j]), m), s22), k, l);
            q[j][2] = Limb2{l[0] + l[1], k[0] + k[1]};
        }
    };
    int slot = 0;
    for (int i = 0; i < np; ++i) {
        const bool emit = i >= HS;
        Limb2 q[PP][3];
        quant(cur, i, q);
        fetch(cur, i + 1);
        ask(i);
        Limb2 old[PP][3];
        if (!S::RING && HS > 0 && emit) {
            Raw f;
            fetch(f, i - HS);
            quant(f, i - HS, old);
        }
        const long long zo = (long long)(zs0 + i - RZ) * HW;
        Two<float> Iv[1], Jv[1], gv[3];
        if (emit && live) {
            load2(Iv, g.I + zo + ooff, N, both, vec);
            load2(Jv, g.J + zo + ooff, N, both, vec);
            if (g.g) load2(gv, g.gJ + zo + ooff, N, both, vec);
        }
#pragma unroll
        for (int j = 0; j < PP; ++j) {
            const int k = tid + j * NT;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                acc[j][c] = acc[j][c] + q[j][c];
                Limb2 *r = ring + (slot * 3 + c) * NPAD + k;
                if (emit) {
                    zs[c * NPAD + k] = acc[j][c];
                    // less the plane that leaves the window
                    acc[j][c] = acc[j][c] - (S::RING ? *r : (HS > 0 ? old[j][c] : q[j][c]));
                }
                if (S::RING) *r = q[j][c];
            }
        }
        slot = slot + 1 >= HS ? 0 : slot + 1;
        if (!emit) continue;
        __syncthreads();
        win_columns<R, 3>(zs, ys, tid);
        __syncthreads();
        Limb2 w[3][2];
#pragma unroll
        for (int c = 0; c < 3; ++c) win_row<R>(ys, c, row, pair, w[c]);
        if (!live) continue;
        float2 hi[3], lo[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const unsigned terms = (unsigned)(RZ == R ? g.n : (2 * R + 1) * (2 * R + 1));
            const unsigned base = kLimbBits * terms * (c == 2 ? 2u : 1u);
            long long x[2];
#pragma unroll
            for (int e = 0; e < 2; ++e)
                x[e] = (long long)(int)(w[c][e].k - base) * (1ll << S::RB) +
                       (int)(w[c][e].l - base);
            i64x2_to_ff(x, us[c], hi[c], lo[c]);
        }
        float2 rh, rl, th, tl;
        ff2_mul(make_float2(Iv[0].a, Iv[0].b), hi[0], lo[0], rh, rl);                // I SA
        ff2_mul(make_float2(2.0f * Jv[0].a, 2.0f * Jv[0].b), hi[1], lo[1], th, tl);  // 2 J SB
        ff2_add(rh, rl, th, tl);
        ff2_add(rh, rl, hi[2], lo[2]);  // + SC
        const float2 dj = __fmul2_rn(neg2(__fadd2_rn(rh, rl)), both2(inv_n));
        if (g.dJ) {
            const float2 out[1] = {dj};
            store2(g.dJ + zo + ooff, N, out, both, vec);
        }
        if (g.g) {
            float2 out[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) out[c] = __fmul2_rn(dj, make_float2(gv[c].a, gv[c].b));
            store2(g.g + zo + ooff, N, out, both, vec);
        }
    }
}

template <int R, bool SWAP, int RZ = R>
__global__ void __launch_bounds__(WinTile<R>::NT, grad_min_ctas(R)) k_lncc_grad(const __grid_constant__ GradArgs g) {
    lncc_grad_body<R, SWAP, RZ>(g, blockIdx.x, blockIdx.y, blockIdx.z);
}

}  // namespace

}  // namespace fa
