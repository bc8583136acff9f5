// The marching kernel (march.cuh) for FP32 storage and an isotropic medium of uniform permeability, without walls or a
// pole: its launch geometry and the launches of a call.
//
// What bounds it (4096^2, 8 steps a launch): the HBM traffic.  ncu counts 742 MB a launch (24 + 20 bytes a site, the
// 14 extra rows of a segment of 128 on top); at 129 us that is 5.75 TB/s, 0.84 of the measured copy rate, launch and
// the first rows' latency included.  The strip kernel moves the same bytes for 2 steps in 121 us.  Below about 2048^2
// the state stays in L2 and a launch takes its rows' latency: about 0.45 us a row for a warp alone on its scheduler
// (a row is 8 updates of 4 sites a lane, some 430 instructions), for R + 14 rows.
// K = 8: four levels cost 32 us a step at 4096^2 and six 20.8 us, both bound by HBM, against 16.1 us; ten and twelve
// levels do not fit the registers of 8 warps an SM without spilling (18.3 and 16.2 us a step).
// 8 warps an SM (two per scheduler): 12 warps allow 168 registers, which K = 8 spills.  D = 3 rows of staging: with 4
// the 4096^2 launch takes 136 us (more reads in flight, but further from the writes), 2048^2 38 us against 39 us.
#include "march.cuh"

#include <algorithm>

namespace lbk {

template <int ST, int MED, bool WL, int K, int D>
__global__ void __launch_bounds__(32, 8) march2d(const __grid_constant__ MarchArgs m) {
    extern __shared__ __align__(1024) float march_smem[];
    const int seg = blockIdx.x / m.nstrips, strip = blockIdx.x - seg * m.nstrips;
    march_unit<ST, MED, WL, K, D>(m.a, m.w, m.steps, m.nstrips, m.nseg, strip, seg,
                                  (unsigned)__cvta_generic_to_shared(march_smem));
}

// Launches of K steps, the last one of what is left.  One wave of units: as many segments as fill the GPU (a second
// wave would leave it half empty), of at least two rows.  Each launch may start while the one before drains
// (programmatic dependent launch; it waits for its input with griddepcontrol.wait): 128^2 8.2 us a launch against
// 10.3 us, 1024^2 18 us against 20.5 us.
template <int ST, int MED, bool WL, int K, int D>
static cudaError_t launch(const StepArgs &a, const Walls &w, int nsteps, cudaStream_t s, int *launches) {
    using Cfg = MarchCfg<ST, MED, K, D>;
    auto *k = march2d<ST, MED, WL, K, D>;
    static int per_sm = 0, nsm = 0;
    if (!per_sm) {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, 32, Cfg::smem);
        if (e != cudaSuccess) return e;
        per_sm = std::max(n, 1);
    }
    MarchArgs m;
    m.a = a;
    m.w = w;
    m.nstrips = (a.g.nchunk + Cfg::W / 4 - 1) / (Cfg::W / 4);
    m.nseg = std::max(1, std::min(per_sm * nsm / m.nstrips, a.g.ny / 2));
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)m.nstrips * m.nseg);
    cfg.blockDim = dim3(32);
    cfg.dynamicSmemBytes = Cfg::smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    *launches = 0;
    for (int t = 0; t < nsteps; t += K, ++*launches) {
        m.steps = std::min(K, nsteps - t);
        m.a.t = a.t + t;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k, m);
        if (e != cudaSuccess) return e;
        std::swap(m.a.in, m.a.out);
    }
    return cudaSuccess;
}

cudaError_t launch_march_2d(const StepArgs &a, const Walls &w, int nsteps, cudaStream_t s, int *launches) {
    return launch<LBEM_F32, MARCH_ISO, false, 8, 3>(a, w, nsteps, s, launches);
}

}  // namespace lbk
