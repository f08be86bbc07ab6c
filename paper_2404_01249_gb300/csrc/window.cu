// Launches of the LNCC window-sum kernels (window.cuh) over one grid.
#include "launch.cuh"
#include "window.cuh"

namespace fa {

namespace {

// Deepest slab.  A thread of the forward kernel adds two terms per plane whose
// lower limb is up to 2^19 in magnitude in 32 bits: 2^11 planes could overflow.
// (The cost model stays below 64; a caller's tile table may ask for any depth.)
constexpr int kMaxSlab = 1024;

template <int R>
LaunchGeom window_geom(Dims d, int tz, int occ) {
    using G = WinTile<R>;
    LaunchGeom g;
    const int gx = (d.W + FX - 1) / FX, gy = (d.H + G::TY - 1) / G::TY;
    tz = tz < kMaxSlab ? tz : kMaxSlab;
    g.tz = tz > 0 ? (tz < d.D ? tz : d.D) : choose_tz(d.D, gx * gy, window_slab_extra(R), occ);
    g.grid = dim3(gx, gy, (d.D + g.tz - 1) / g.tz);
    g.block = dim3(G::NT);
    return g;
}

template <int R, FwdMode M, int RZ>
cudaError_t fwd(FwdArgs &a, Dims d, int tz, cudaStream_t s) {
    using S = FwdSmem<R, M, RZ>;
    auto kern = k_lncc_fwd<R, M, RZ>;
    const int occ = prepare(kern, S::bytes, WinTile<R>::NT);
    const LaunchGeom g = window_geom<R>(d, tz, occ);
    a.TZ = g.tz;
    return launch_pdl(kern, g, S::bytes, s, a);
}

template <int R, bool SWAP, int RZ>
cudaError_t grad(GradArgs &a, Dims d, int tz, cudaStream_t s) {
    using S = GradTile<R, RZ>;
    auto kern = k_lncc_grad<R, SWAP, RZ>;
    const int occ = prepare(kern, S::bytes, WinTile<R>::NT);
    const LaunchGeom g = window_geom<R>(d, tz, occ);
    a.TZ = g.tz;
    return launch_pdl(kern, g, S::bytes, s, a);
}

template <int R, int RZ>
cudaError_t fwd_mode(FwdMode m, FwdArgs &a, Dims d, int tz, cudaStream_t s) {
    switch (m) {
        case kFwdGiven: return fwd<R, kFwdGiven, RZ>(a, d, tz, s);
        case kFwdBoth: return fwd<R, kFwdBoth, RZ>(a, d, tz, s);
        case kFwdStats: return fwd<R, kFwdStats, RZ>(a, d, tz, s);
    }
    return cudaErrorInvalidValue;
}

template <int R, int RZ>
cudaError_t grad_swap(bool swap, GradArgs &a, Dims d, int tz, cudaStream_t s) {
    return swap ? grad<R, true, RZ>(a, d, tz, s) : grad<R, false, RZ>(a, d, tz, s);
}

// Planes of one row each are one plane of these rows, in memory and to windows
// that are cubes: the sums are exact, so their order does not show.  (The rows'
// tiles must fit the launch grid.)
Dims as_plane(Dims d) {
    return d.H == 1 && d.D <= 8 * 65535 ? Dims{1, d.D, d.W, d.P} : d;
}

template <class A>
void fill_grid(A &a, Dims d) {
    a.D = d.D;
    a.H = d.H;
    a.W = d.W;
    a.P = d.pitch();
}

}  // namespace

#define FA_EACH_R(call)                                \
    switch (window / 2) {                              \
        case 0: { constexpr int RR = 0; e = call; break; } \
        case 1: { constexpr int RR = 1; e = call; break; } \
        case 2: { constexpr int RR = 2; e = call; break; } \
        case 3: { constexpr int RR = 3; e = call; break; } \
        case 4: { constexpr int RR = 4; e = call; break; } \
        case 5: { constexpr int RR = 5; e = call; break; } \
        case 6: { constexpr int RR = 6; e = call; break; } \
        case 7: { constexpr int RR = 7; e = call; break; } \
    }

cudaError_t launch_window_fwd(FwdMode mode, FwdArgs a, Dims d, int window, int tz,
                              cudaStream_t s) {
    d = as_plane(d);
    fill_grid(a, d);
    a.window = window;
    a.bits = lncc_image_bits(window);
    cudaError_t e = cudaErrorInvalidValue;
    FA_EACH_R((d.D == 1 ? fwd_mode<RR, 0>(mode, a, d, tz, s) : fwd_mode<RR, RR>(mode, a, d, tz, s)))
    note_launch();
    return e;
}

cudaError_t launch_window_grad(bool swap, GradArgs a, Dims d, int window, int tz,
                               cudaStream_t s) {
    d = as_plane(d);
    fill_grid(a, d);
    a.n = window * window * window;
    a.cbits = lncc_coef_bits(window);
    cudaError_t e = cudaErrorInvalidValue;
    FA_EACH_R((d.D == 1 ? grad_swap<RR, 0>(swap, a, d, tz, s) : grad_swap<RR, RR>(swap, a, d, tz, s)))
    note_launch();
    return e;
}
#undef FA_EACH_R

}  // namespace fa
