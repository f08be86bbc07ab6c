// Host side of the tiled kernels' launches: grid geometry, dynamic shared
// memory, programmatic dependent launch.
#pragma once

#include <mutex>
#include <utility>

#include "ops.h"

namespace fa {

namespace {

std::mutex g_mu;
int g_num_sms = 0;

int num_sms() {
    std::lock_guard<std::mutex> lock(g_mu);
    if (g_num_sms == 0) {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0)
            g_num_sms = n;
        else
            g_num_sms = 152;
    }
    return g_num_sms;
}

// Opts the kernel into its dynamic shared memory and returns its resident
// CTAs per SM (called once per kernel instantiation).
template <class K>
int prepare(K kernel, size_t smem, int threads) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                         (int)cudaSharedmemCarveoutMaxShared);
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess ||
        n < 1)
        n = 1;
    return n;
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
