// Lockstep batches of the fused kernels: many registrations advance together,
// one launch of each fused kernel per iteration over the tiles of every job.
#include "fused_kernels.cuh"

namespace fa {

namespace {

// ------------------------------------------------------------ lockstep batches
// Many registrations advance together: one launch of a fused kernel covers the
// tiles of every job in the launch's table.  CTA b belongs to the job k with
// first[k] <= b < first[k + 1]; its tile inside that job's grid is
// b - first[k] in x-fastest order.  The table travels in the kernel's
// parameter space (read through the constant cache; every thread of a CTA
// reads the same entry), and so do the jobs' tensor maps: a CTA hands the
// TMA unit the address of its job's maps in that space.  A launch takes TMA
// tiles when every job's buffers meet TMA's alignment rules (the row pitch
// of a level's buffers is a multiple of 4 floats whenever the fused kernels
// run it), else the per-thread copy variant (cp.async) for all its jobs.
// The update kernels of a batch take 32 x 16 tiles (the compose's u' region, the
// tile plus the sigma_warp halo, is then 1.41 instead of 1.69 times the tile):
// a wave's jobs fill the GPU together.

struct BGeom {
    int D, H, W, P, TZ, gx, gy;  // P: row pitch of the job's buffers
};
struct BTaps {
    float w[2 * kMaxFusedRG + 1];
};
// K1 and K2 take every job's arguments as a single launch does.
struct K1Batch {
    int n;
    int first[kMaxLockstepJobs + 1];
    FwdArgs j[kMaxLockstepJobs];
};
struct K2Batch {
    int n;
    int first[kMaxLockstepJobs + 1];
    GradArgs j[kMaxLockstepJobs];
};
struct K3Job {
    const float *g;
    void *m, *v;  // stored as the launch's moment type
    float *dir;
    WsHeader *h;
    BGeom geo;
    BTaps t;
};
// NM maps per job: the gradient, then (FP32 moments) m and nu.
template <int NM>
struct K3Batch {
    CUtensorMap tm[NM * kMaxLockstepJobs];
    int n, parity;
    AdamConsts ac;
    int first[kMaxLockstepJobs + 1];
    K3Job j[kMaxLockstepJobs];
};
struct K4Job {
    const void *u;  // stored as the launch's u type
    const float *dir;
    void *uo;
    const float *Im;
    float *J, *gJ;
    WsHeader *h;
    BGeom geo;
    BTaps t;
    float lr, c_lp;
};
// NM maps per job: the direction, then (u read from shared memory) u.
template <int NM>
struct K4Batch {
    CUtensorMap tm[NM * kMaxLockstepJobs];
    int n, parity;
    int first[kMaxLockstepJobs + 1];
    K4Job j[kMaxLockstepJobs];
};
// CUDA's limit on a launch's parameters
constexpr size_t kMaxParamBytes = 32764;
static_assert(sizeof(K1Batch) <= kMaxParamBytes && sizeof(K2Batch) <= kMaxParamBytes &&
                  sizeof(K3Batch<3>) <= kMaxParamBytes && sizeof(K4Batch<2>) <= kMaxParamBytes,
              "a lockstep table must fit the kernel parameter space");

// The job of CTA b: the largest k with first[k] <= b (first[0] = 0).
__device__ __forceinline__ int batch_job(const int *first, int n, int b) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= b)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ void batch_tile(const BGeom &g, int t, int &bx, int &by, int &bz) {
    bx = t % g.gx;
    const int r = t / g.gx;
    by = r % g.gy;
    bz = r / g.gy;
}

// Job k's maps tm[NM k ...] of a table (TMA launches), else none.
template <int NM, bool TMA>
__device__ __forceinline__ MapRef job_maps(const CUtensorMap *tm, int k) {
    MapRef r{nullptr, nullptr, nullptr};
    if (TMA) {
        r.a = tm + NM * k;
        if (NM > 1) r.b = tm + NM * k + 1;
        if (NM > 2) r.c = tm + NM * k + 2;
    }
    return r;
}

template <int R, class A>
__device__ __forceinline__ void window_tile(const A &a, int t, int &bx, int &by, int &bz) {
    const int gx = (a.W + FX - 1) / FX, gy = (a.H + WinTile<R>::TY - 1) / WinTile<R>::TY;
    bx = t % gx;
    const int r = t / gx;
    by = r % gy;
    bz = r / gy;
}

template <int R>
__global__ void __launch_bounds__(WinTile<R>::NT, fwd_min_ctas(R))
    k_lncc_fwd_batch(const __grid_constant__ K1Batch b) {
    const int k = batch_job(b.first, b.n, (int)blockIdx.x);
    int bx, by, bz;
    window_tile<R>(b.j[k], (int)blockIdx.x - b.first[k], bx, by, bz);
    lncc_fwd_body<R, kFwdGiven>(b.j[k], bx, by, bz);
}

template <int R>
__global__ void __launch_bounds__(WinTile<R>::NT, grad_min_ctas(R))
    k_lncc_grad_batch(const __grid_constant__ K2Batch b) {
    const int k = batch_job(b.first, b.n, (int)blockIdx.x);
    int bx, by, bz;
    window_tile<R>(b.j[k], (int)blockIdx.x - b.first[k], bx, by, bz);
    lncc_grad_body<R, false>(b.j[k], bx, by, bz);
}

template <class TS>
constexpr int k3_maps() {
    return sizeof(TS) == 4 ? 3 : 1;
}

template <int RG, class TS, bool TMA>
__global__ void __launch_bounds__(FX *K3W_NW, k3_min_ctas(RG, K3W_NW, K3W_OPT)) k_smooth_adam_batch(
    const __grid_constant__ K3Batch<k3_maps<TS>()> b) {
    const int k = batch_job(b.first, b.n, (int)blockIdx.x);
    const K3Job &j = b.j[k];
    int bx, by, bz;
    batch_tile(j.geo, (int)blockIdx.x - b.first[k], bx, by, bz);
    smooth_adam_body<RG, K3W_NW, K3W_OPT, K3_ST, TMA>(
        job_maps<k3_maps<TS>(), TMA>(b.tm, k), j.g, (TS *)j.m, (TS *)j.v, j.dir, j.h, j.geo.D,
        j.geo.H, j.geo.W, j.geo.P, j.geo.TZ, j.t, b.ac, b.parity, bx, by, bz);
}

// TU: storage of u (float, or __half: tile copies only).
template <int RG, bool SU, bool TMA, class TU>
__global__ void __launch_bounds__(FX *K4W_NW, k4_min_ctas(RG, K4W_NW, K4W_OPT)) k_compose_batch(
    const __grid_constant__ K4Batch<SU ? 2 : 1> b) {
    const int k = batch_job(b.first, b.n, (int)blockIdx.x);
    const K4Job &j = b.j[k];
    int bx, by, bz;
    batch_tile(j.geo, (int)blockIdx.x - b.first[k], bx, by, bz);
    compose_body<RG, K4W_NW, K4W_OPT, SU, K4_ST, TMA>(
        job_maps<SU ? 2 : 1, TMA>(b.tm, k), (const TU *)j.u, j.dir, (TU *)j.uo, j.Im, j.J, j.gJ,
        j.h, j.geo.D, j.geo.H, j.geo.W, j.geo.P, j.geo.TZ, j.t, j.lr, j.c_lp, b.parity, bx, by,
        bz);
}

// Slab depth of a lockstep launch: one TZ for all its jobs (each capped at its
// own depth), minimising (waves x planes per CTA) over the whole launch, whose
// CTAs fill the GPU's resident slots together.  A coarse level of many jobs
// then takes short slabs (more CTAs), a fine level long ones (less halo).
int launch_tz(const Dims *d, int n, int ty, float extra, int occ) {
    const long long slots = (long long)num_sms() * (occ > 0 ? occ : 1);
    int best = 64;
    float bestcost = -1.0f;
    for (int tz = 1; tz <= 64; ++tz) {
        long long ctas = 0;
        for (int k = 0; k < n; ++k) {
            const long long txy = (long long)((d[k].W + FX - 1) / FX) * ((d[k].H + ty - 1) / ty);
            const int t = tz < d[k].D ? tz : d[k].D;
            ctas += txy * ((d[k].D + t - 1) / t);
        }
        const float cost = (float)((ctas + slots - 1) / slots) * ((float)tz + extra);
        if (bestcost < 0.0f || cost < bestcost) {
            bestcost = cost;
            best = tz;
        }
    }
    return best;
}

// Fills a job's tile geometry for a kernel with `ty` rows per CTA and slab
// depth tz (capped at the job's depth) and returns its CTA count.
int batch_geom(BGeom &g, Dims d, int ty, int tz) {
    g.D = d.D;
    g.H = d.H;
    g.W = d.W;
    g.P = d.pitch();
    g.gx = (d.W + FX - 1) / FX;
    g.gy = (d.H + ty - 1) / ty;
    g.TZ = tz < d.D ? tz : d.D;
    return g.gx * g.gy * ((d.D + g.TZ - 1) / g.TZ);
}

BGeom *geom_of(K3Job &j) { return &j.geo; }
BGeom *geom_of(K4Job &j) { return &j.geo; }

void batch_taps(BTaps &b, const GaussTaps &t) {
    for (int k = 0; k < 2 * kMaxFusedRG + 1; ++k) b.w[k] = k <= 2 * t.R ? t.w[k] : 0.0f;
}

template <class K, class B>
cudaError_t launch_batch(K kern, const B &b, int nw, size_t smem, cudaStream_t s) {
    LaunchGeom g;
    g.grid = dim3((unsigned)b.first[b.n]);
    g.block = dim3(FX, nw);
    g.tz = 0;
    return launch_pdl(kern, g, smem, s, b);
}

// Tile geometry of every job of a launch (jobs[idx[k]], k < b.n) for a kernel
// of `ty` rows per CTA, halo `halo` and `occ` resident CTAs per SM.
template <class B>
void batch_layout(B &b, const LockstepJob *jobs, const int *idx, int ty, int halo, int occ) {
    Dims dd[kMaxLockstepJobs];
    for (int k = 0; k < b.n; ++k) dd[k] = jobs[idx[k]].d;
    const int tz = launch_tz(dd, b.n, ty, 2.0f * halo, occ);
    b.first[0] = 0;
    for (int k = 0; k < b.n; ++k) {
        BGeom &g = *geom_of(b.j[k]);
        b.first[k + 1] = b.first[k] + batch_geom(g, dd[k], ty, tz);
    }
}

// Grid and slab depth of every job of a K1 or K2 launch.
template <int R, class B>
void window_layout(B &b, const LockstepJob *jobs, int occ) {
    using G = WinTile<R>;
    Dims dd[kMaxLockstepJobs];
    for (int k = 0; k < b.n; ++k) dd[k] = jobs[k].d;
    const int tz = launch_tz(dd, b.n, G::TY, window_slab_extra(R), occ);
    b.first[0] = 0;
    for (int k = 0; k < b.n; ++k) {
        auto &a = b.j[k];
        a.D = dd[k].D;
        a.H = dd[k].H;
        a.W = dd[k].W;
        a.P = dd[k].pitch();
        a.TZ = tz < a.D ? tz : a.D;
        b.first[k + 1] = b.first[k] + (a.W + FX - 1) / FX * ((a.H + G::TY - 1) / G::TY) *
                                          ((a.D + a.TZ - 1) / a.TZ);
    }
}

template <class K, class B>
cudaError_t launch_window_batch(K kern, const B &b, int threads, size_t smem, cudaStream_t s) {
    LaunchGeom g;
    g.grid = dim3((unsigned)b.first[b.n]);
    g.block = dim3(threads);
    g.tz = 0;
    return launch_pdl(kern, g, smem, s, b);
}

template <int R>
cudaError_t launch_k1_batch(K1Batch &b, const LockstepJob *jobs, cudaStream_t s) {
    constexpr size_t smem = FwdSmem<R, kFwdGiven>::bytes;
    auto kern = k_lncc_fwd_batch<R>;
    const int occ = prepare(kern, smem, WinTile<R>::NT);
    window_layout<R>(b, jobs, occ);
    return launch_window_batch(kern, b, WinTile<R>::NT, smem, s);
}

template <int R>
cudaError_t launch_k2_batch(K2Batch &b, const LockstepJob *jobs, cudaStream_t s) {
    constexpr size_t smem = GradTile<R>::bytes;
    auto kern = k_lncc_grad_batch<R>;
    const int occ = prepare(kern, smem, WinTile<R>::NT);
    window_layout<R>(b, jobs, occ);
    return launch_window_batch(kern, b, WinTile<R>::NT, smem, s);
}

template <int RG, class TS>
cudaError_t launch_k3_batch(K3Batch<k3_maps<TS>()> &b, const LockstepJob *jobs, const int *idx,
                            cudaStream_t s) {
    constexpr bool S32 = sizeof(TS) == 4;
    constexpr int NM = k3_maps<TS>();
    using ST = K3S<RG, K3W_NW, K3W_OPT, K3_ST, S32>;  // FP32 moments staged
    bool tma = true;
    for (int k = 0; k < b.n && tma; ++k) {
        const LockstepJob &q = jobs[idx[k]];
        tma = tmap(&b.tm[NM * k], q.fb->g, 4, q.d, 3, ST::BXW, ST::RY, 3);
        if constexpr (S32)
            tma = tma && tmap(&b.tm[NM * k + 1], q.m, 4, q.d, 3, FX, ST::TY, 3) &&
                  tmap(&b.tm[NM * k + 2], q.v, 4, q.d, 3, FX, ST::TY, 3);
    }
    if (tma) {
        auto kern = k_smooth_adam_batch<RG, TS, true>;
        const int occ = prepare(kern, ST::bytes, ST::NT);
        batch_layout(b, jobs, idx, ST::TY, RG, occ);
        return launch_batch(kern, b, ST::NT / FX, ST::bytes, s);
    }
    using SC = K3S<RG, K3W_NW, K3W_OPT, K3_ST, false>;  // moments unstaged
    auto kern = k_smooth_adam_batch<RG, TS, false>;
    const int occ = prepare(kern, SC::bytes, SC::NT);
    batch_layout(b, jobs, idx, SC::TY, RG, occ);
    return launch_batch(kern, b, SC::NT / FX, SC::bytes, s);
}

// TU: storage of u of every job of the launch (an FP16 u takes tile copies
// only: cudaErrorNotSupported when a job's buffers do not meet their rules).
template <int RG, bool SU, class TU>
cudaError_t launch_k4_batch(K4Batch<SU ? 2 : 1> &b, const LockstepJob *jobs, const int *idx,
                            cudaStream_t s) {
    constexpr int NM = SU ? 2 : 1, EU = (int)sizeof(TU);
    using ST = K4S<RG, K4W_NW, K4W_OPT, SU, K4_ST, TU>;
    bool tma = true;
    for (int k = 0; k < b.n && tma; ++k) {
        const LockstepJob &q = jobs[idx[k]];
        tma = tmap(&b.tm[NM * k], q.fb->dir, 4, q.d, 3, ST::BXW, ST::RY, 3);
        if constexpr (SU)
            tma = tma && tmap(&b.tm[NM * k + 1], q.u, EU, q.d, 3, ST::UBXW, ST::URY, 3);
    }
    if (tma) {
        auto kern = k_compose_batch<RG, SU, true, TU>;
        const int occ = prepare(kern, ST::bytes, ST::NT);
        batch_layout(b, jobs, idx, ST::TY, RG, occ);
        return launch_batch(kern, b, ST::NT / FX, ST::bytes, s);
    }
    if constexpr (EU == 4) {
        using SC = K4S<RG, K4W_NW, K4W_OPT, SU, K4_ST>;
        auto kern = k_compose_batch<RG, SU, false, float>;
        const int occ = prepare(kern, SC::bytes, SC::NT);
        batch_layout(b, jobs, idx, SC::TY, RG, occ);
        return launch_batch(kern, b, SC::NT / FX, SC::bytes, s);
    } else {
        return cudaErrorNotSupported;
    }
}

#define FA_CASE(n, call)      \
    case n: {                 \
        constexpr int RR = n; \
        return call;          \
    }

cudaError_t dispatch_k1_batch(int R, K1Batch &b, const LockstepJob *jobs,
                              cudaStream_t s) {
    switch (R) {
        FA_CASE(0, launch_k1_batch<RR>(b, jobs, s))
        FA_CASE(1, launch_k1_batch<RR>(b, jobs, s))
        FA_CASE(2, launch_k1_batch<RR>(b, jobs, s))
        FA_CASE(3, launch_k1_batch<RR>(b, jobs, s))
        FA_CASE(4, launch_k1_batch<RR>(b, jobs, s))
        FA_CASE(5, launch_k1_batch<RR>(b, jobs, s))
        FA_CASE(6, launch_k1_batch<RR>(b, jobs, s))
        FA_CASE(7, launch_k1_batch<RR>(b, jobs, s))
    }
    return cudaErrorInvalidValue;
}

cudaError_t dispatch_k2_batch(int R, K2Batch &b, const LockstepJob *jobs,
                              cudaStream_t s) {
    switch (R) {
        FA_CASE(0, launch_k2_batch<RR>(b, jobs, s))
        FA_CASE(1, launch_k2_batch<RR>(b, jobs, s))
        FA_CASE(2, launch_k2_batch<RR>(b, jobs, s))
        FA_CASE(3, launch_k2_batch<RR>(b, jobs, s))
        FA_CASE(4, launch_k2_batch<RR>(b, jobs, s))
        FA_CASE(5, launch_k2_batch<RR>(b, jobs, s))
        FA_CASE(6, launch_k2_batch<RR>(b, jobs, s))
        FA_CASE(7, launch_k2_batch<RR>(b, jobs, s))
    }
    return cudaErrorInvalidValue;
}

template <class TS>
cudaError_t dispatch_k3_batch_ts(int RG, K3Batch<k3_maps<TS>()> &b, const LockstepJob *jobs,
                                 const int *idx, cudaStream_t s) {
    switch (RG) {
        FA_CASE(0, (launch_k3_batch<RR, TS>(b, jobs, idx, s)))
        FA_CASE(1, (launch_k3_batch<RR, TS>(b, jobs, idx, s)))
        FA_CASE(2, (launch_k3_batch<RR, TS>(b, jobs, idx, s)))
        FA_CASE(3, (launch_k3_batch<RR, TS>(b, jobs, idx, s)))
        FA_CASE(4, (launch_k3_batch<RR, TS>(b, jobs, idx, s)))
        FA_CASE(5, (launch_k3_batch<RR, TS>(b, jobs, idx, s)))
        FA_CASE(6, (launch_k3_batch<RR, TS>(b, jobs, idx, s)))
    }
    return cudaErrorInvalidValue;
}

// One K3 launch over jobs[idx[0..m)], whose moments are stored as TS.
template <class TS>
cudaError_t k3_batch(int RG, int m, const LockstepJob *jobs, const int *idx, AdamConsts ac,
                     int parity, cudaStream_t s) {
    K3Batch<k3_maps<TS>()> b;
    b.n = m;
    b.parity = parity;
    b.ac = ac;
    for (int i = 0; i < m; ++i) {
        const LockstepJob &q = jobs[idx[i]];
        K3Job &j = b.j[i];
        j.g = q.fb->g;
        j.m = q.m;
        j.v = q.v;
        j.dir = q.fb->dir;
        j.h = q.h;
        batch_taps(j.t, *q.tg);
    }
    return dispatch_k3_batch_ts<TS>(RG, b, jobs, idx, s);
}

template <bool SU, class TU>
cudaError_t dispatch_k4_batch(int RG, K4Batch<SU ? 2 : 1> &b, const LockstepJob *jobs,
                              const int *idx, cudaStream_t s) {
    switch (RG) {
        FA_CASE(0, (launch_k4_batch<RR, SU, TU>(b, jobs, idx, s)))
        FA_CASE(1, (launch_k4_batch<RR, SU, TU>(b, jobs, idx, s)))
        FA_CASE(2, (launch_k4_batch<RR, SU, TU>(b, jobs, idx, s)))
        FA_CASE(3, (launch_k4_batch<RR, SU, TU>(b, jobs, idx, s)))
        FA_CASE(4, (launch_k4_batch<RR, SU, TU>(b, jobs, idx, s)))
        FA_CASE(5, (launch_k4_batch<RR, SU, TU>(b, jobs, idx, s)))
        FA_CASE(6, (launch_k4_batch<RR, SU, TU>(b, jobs, idx, s)))
    }
    return cudaErrorInvalidValue;
}

// One K4 launch over jobs[idx[0..m)], whose u is stored as TU.
template <bool SU, class TU>
cudaError_t k4_batch(int RG, int m, const LockstepJob *jobs, const int *idx, int parity,
                     cudaStream_t s) {
    K4Batch<SU ? 2 : 1> b;
    b.n = m;
    b.parity = parity;
    for (int i = 0; i < m; ++i) {
        const LockstepJob &q = jobs[idx[i]];
        K4Job &j = b.j[i];
        j.u = q.u;
        j.dir = q.fb->dir;
        j.uo = q.u_alt;
        j.Im = q.Im;
        j.J = q.fb->J;
        j.gJ = q.fb->gJ;
        j.h = q.h;
        batch_taps(j.t, *q.tw);
        j.lr = q.p->lr;
        j.c_lp = q.p->c_lp;
    }
    return dispatch_k4_batch<SU, TU>(RG, b, jobs, idx, s);
}
#undef FA_CASE

}  // namespace

fa_status fused_iteration_lockstep(int n, const LockstepJob *jobs, int t, cudaStream_t s) {
    if (n < 1 || n > kMaxLockstepJobs) {
        set_error("lockstep iteration: 1..%d jobs per launch (got %d)", kMaxLockstepJobs, n);
        return FA_ERR_INVALID;
    }
    const fa_params *p0 = jobs[0].p;
    const int parity = t & 1, R = p0->window / 2;
    int idx[kMaxLockstepJobs];
    for (int k = 0; k < n; ++k) idx[k] = k;
    {
        K1Batch b;
        b.n = n;
        for (int k = 0; k < n; ++k) {
            const LockstepJob &q = jobs[k];
            FwdArgs a{};
            a.I = q.If;
            a.J = q.fb->J;
            a.SI = q.fb->sI;
            a.varI = q.fb->varI;
            a.coef = q.fb->coef;
            a.h = q.h;
            a.bits = lncc_image_bits(p0->window);
            a.window = p0->window;
            a.cc_eps = q.p->cc_eps;
            a.write_coef = 1;
            b.j[k] = a;
        }
        FA_CUDA_TRY(dispatch_k1_batch(R, b, jobs, s));
        note_launch();
    }
    {
        K2Batch b;
        b.n = n;
        for (int k = 0; k < n; ++k) {
            const LockstepJob &q = jobs[k];
            GradArgs a{};
            a.I = q.If;
            a.J = q.fb->J;
            a.gJ = q.fb->gJ;
            a.coef = q.fb->coef;
            a.h = q.h;
            a.g = q.fb->g;
            a.cbits = lncc_coef_bits(p0->window);
            a.n = p0->window * p0->window * p0->window;
            b.j[k] = a;
        }
        FA_CUDA_TRY(dispatch_k2_batch(R, b, jobs, s));
        note_launch();
    }
    const AdamConsts ac = adam_consts(p0, t);
    const int states[2] = {FA_F32, FA_BF16};
    for (int st : states) {
        for (int rg = 0; rg <= kMaxFusedRG; ++rg) {
            int m = 0;
            for (int k = 0; k < n; ++k)
                if (jobs[k].tg->R == rg && jobs[k].p->state_storage == st) idx[m++] = k;
            if (m == 0) continue;
            FA_CUDA_TRY(st == FA_F32 ? k3_batch<float>(rg, m, jobs, idx, ac, parity, s)
                                     : k3_batch<__nv_bfloat16>(rg, m, jobs, idx, ac, parity, s));
            note_launch();
        }
    }
    const int fields[2] = {FA_F32, FA_F16};
    for (int fs : fields)
        for (int su = 0; su < 2; ++su)
            for (int rg = 0; rg <= kMaxFusedRG; ++rg) {
                int m = 0;
                for (int k = 0; k < n; ++k) {
                    const fa_params *p = jobs[k].p;
                    const int ksu = (double)p->lr / (double)p->c_lp < 0.999 ? 1 : 0;
                    if (jobs[k].tw->R == rg && ksu == su && p->field_storage == fs) idx[m++] = k;
                }
                if (m == 0) continue;
                cudaError_t e;
                if (fs == FA_F16)
                    e = su ? k4_batch<true, __half>(rg, m, jobs, idx, parity, s)
                           : k4_batch<false, __half>(rg, m, jobs, idx, parity, s);
                else
                    e = su ? k4_batch<true, float>(rg, m, jobs, idx, parity, s)
                           : k4_batch<false, float>(rg, m, jobs, idx, parity, s);
                if (e == cudaErrorNotSupported) {
                    set_error("lockstep: an FP16 u needs tile copies (rows of 8 elements)");
                    return FA_ERR_UNSUPPORTED;
                }
                FA_CUDA_TRY(e);
                note_launch();
            }
    return FA_OK;
}

}  // namespace fa
