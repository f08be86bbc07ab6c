// Host side of the tiled kernels' launches: grid geometry, dynamic shared
// memory, programmatic dependent launch.
#pragma once

#include <utility>

#include "ops.h"

namespace fa {

// SMs of the current device.
int num_sms();
// Opts a kernel into `smem` bytes of dynamic shared memory in the current
// context and returns its resident CTAs per SM with blocks of `threads` (1
// when the driver cannot say).  The limit belongs to the kernel in one
// context, so it is raised, and the count kept, once per context: on another
// device, or after a device reset, the next launch raises it there.  A kernel
// always comes with the same smem and threads.
int prepare_kernel(const void *kernel, size_t smem, int threads);

namespace {

template <class K>
int prepare(K kernel, size_t smem, int threads) {
    return prepare_kernel((const void *)kernel, smem, threads);
}

struct LaunchGeom {
    dim3 grid, block;
    int tz;
};

// Launch with programmatic stream serialization (see pdl_wait).
template <class... KArgs, class... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), const LaunchGeom &g, size_t smem, cudaStream_t s,
                       Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g.grid;
    cfg.blockDim = g.block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// Slab depth TZ minimising (waves x planes per CTA) for a z-marching kernel;
// `extra` is what a slab costs beyond its output planes, in output planes.
int choose_tz(int D, int tiles_xy, float extra, int ctas_per_sm) {
    const long long slots = (long long)num_sms() * (ctas_per_sm > 0 ? ctas_per_sm : 1);
    int best = D;
    float bestcost = -1.0f;
    for (int tz = 1; tz <= D && tz <= 64; ++tz) {
        const long long ctas = (long long)tiles_xy * ((D + tz - 1) / tz);
        const long long waves = (ctas + slots - 1) / slots;
        const float cost = (float)waves * ((float)tz + extra);
        if (bestcost < 0.0f || cost < bestcost) {
            bestcost = cost;
            best = tz;
        }
    }
    return best;
}

}  // namespace

}  // namespace fa
