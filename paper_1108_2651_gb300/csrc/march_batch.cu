// The marching kernel (march.cuh) over the members of a batch: one launch advances every member by up to 8 steps in its
// own two buffers.  A unit is a strip of a member's columns and a segment of its rows.
#include "march.cuh"

namespace lbk {

using BatchCfg = MarchCfg<LBEM_F32, MARCH_ISO, MARCH_BATCH_STEPS, 3>;

// args[2 m + par]: member m's step arguments for buffer parity par.
__global__ void __launch_bounds__(32, 8) march2d_batch(const StepArgs *__restrict__ args,
                                                       const BatchMarchUnit *__restrict__ units,
                                                       const long long *__restrict__ t0p, int toff, int steps, int par) {
    extern __shared__ __align__(1024) float march_smem[];
    const BatchMarchUnit u = units[blockIdx.x];
    StepArgs a = args[2 * u.m + par];
    a.t = *t0p + toff;
    const int nstrips = (a.g.nchunk + BatchCfg::W / 4 - 1) / (BatchCfg::W / 4);
    march_unit<LBEM_F32, MARCH_ISO, false, MARCH_BATCH_STEPS, 3>(a, Walls(), steps, nstrips, u.strip, u.y0, u.y1,
                                                                 (unsigned)__cvta_generic_to_shared(march_smem));
}

static PerDevice<KernelFit> batch_fits;

static int resident_units() {
    KernelFit fit;
    kernel_fit(batch_fits, march2d_batch, 32, BatchCfg::smem, &fit, true);
    return std::max(1, fit.per_sm * fit.nsm);
}

// The units of members with these grids: segments of at most R rows, evenly cut, tall ones first, for the R whose units,
// taken in that order by the warps that fit the GPU, are done first (a unit of h rows costs h + 14: the rows before and
// after it that its levels need).
std::vector<BatchMarchUnit> batch_march_units(int n, const Grid *grids) {
    const int cap = resident_units();
    std::vector<BatchMarchUnit> best;
    long long best_cost = -1;
    for (int R : {16, 24, 32, 48, 64, 80, 96, 112, 128, 144, 160, 192, 256, 512, 1024, 4096}) {
        std::vector<BatchMarchUnit> u;
        for (int m = 0; m < n; m++) {
            const int nstrips = (grids[m].nchunk + BatchCfg::W / 4 - 1) / (BatchCfg::W / 4);
            const int nseg = (grids[m].ny + R - 1) / R;
            for (int s = 0; s < nseg; s++)
                for (int k = 0; k < nstrips; k++)
                    u.push_back({m, k, march_cut(s, nseg, grids[m].ny), march_cut(s + 1, nseg, grids[m].ny)});
        }
        std::stable_sort(u.begin(), u.end(),
                         [](const BatchMarchUnit &a, const BatchMarchUnit &b) { return a.y1 - a.y0 > b.y1 - b.y0; });
        std::vector<long long> busy(cap, 0);  // a heap of the warps' finishing times
        long long cost = 0;
        for (const BatchMarchUnit &q : u) {
            std::pop_heap(busy.begin(), busy.end(), std::greater<long long>());
            busy.back() += q.y1 - q.y0 + 2 * (MARCH_BATCH_STEPS - 1);
            cost = std::max(cost, busy.back());
            std::push_heap(busy.begin(), busy.end(), std::greater<long long>());
        }
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best.swap(u);
        }
    }
    return best;
}

cudaError_t launch_batch_march(const StepArgs *args, const BatchMarchUnit *units, int nunits, const long long *t0p,
                               int toff, int steps, int par, cudaStream_t s) {
    KernelFit fit;
    const cudaError_t e = kernel_fit(batch_fits, march2d_batch, 32, BatchCfg::smem, &fit, true);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nunits);
    cfg.blockDim = dim3(32);
    cfg.dynamicSmemBytes = BatchCfg::smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, march2d_batch, args, units, t0p, toff, steps, par);
}

}  // namespace lbk
