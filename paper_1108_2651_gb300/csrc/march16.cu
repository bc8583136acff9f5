// The marching kernel (march.cuh) for 16-bit storage (uniform mu, nx % 4 == 0): rows are decoded as level 0 reads them,
// the state is rounded to the storage's format after every second level, as launches of two steps round it, and the last
// level encodes.
//
// Steps a launch at 4096^2 (us a step; two-step launches 45.3 FP16, 43.6 BF16, 68.8 block-int16): 8 for FP16 and BF16
// (17.7, 13.8; 6: 18.4, 15.6; 4: 21.7, 21.2).  4 for block-int16 (39.6; 6: 42.1; 8: 44.0): it is bound by its
// instructions (an exponent, 20 products, 40 clamps and 40 roundings for a site's five values every two steps, for four
// sites), not by HBM, and its halo is four columns per two levels, 8 of 128 with 4 levels and 16 with 8.
#include "march.cuh"

namespace lbk {

cudaError_t launch_march_2d_16(const StepArgs &a, int storage, int nsteps, cudaStream_t s, int *launches, MarchUnits *units) {
    const Walls w;
    if (storage == LBEM_F16) return launch_march<LBEM_F16, MARCH_ISO, false, 8, 3>(a, w, nsteps, s, launches, units);
    if (storage == LBEM_BF16) return launch_march<LBEM_BF16, MARCH_ISO, false, 8, 3>(a, w, nsteps, s, launches, units);
    return launch_march<LBEM_I16B, MARCH_ISO, false, 4, 4>(a, w, nsteps, s, launches, units);
}

}  // namespace lbk
