// The marching kernel (march.cuh) for the other FP32 media: an anisotropic tensor, a heterogeneous permeability (the two
// grad ln mu planes in the medium's ring), a dispersive pole (P and J staged and handed from level to level in registers,
// its three coefficients in the ring).
//
// Steps a launch: 8 with a tensor, as the plain medium.  6 with mu and with a pole, whose rows take 13 and 16 KB of
// shared memory a warp for the medium alone: 400 steps of a mu medium at 2048^2 take 4.02 ms with 6 and 4.37 with 4
// steps a launch (13.3 ms with the two-step kernels), 200 steps of the Drude cylinder 2.49 and 2.97 ms (8.9 ms).
#include "march.cuh"

namespace lbk {

cudaError_t launch_march_2d_an(const StepArgs &a, const Walls &w, int nsteps, cudaStream_t s, int *launches, MarchUnits *units) {
    if (w.kind[0] || w.kind[1]) return launch_march<LBEM_F32, MARCH_AN, true, 8, 3>(a, w, nsteps, s, launches, units);
    return launch_march<LBEM_F32, MARCH_AN, false, 8, 3>(a, w, nsteps, s, launches, units);
}

cudaError_t launch_march_2d_mu(const StepArgs &a, const Walls &w, int nsteps, cudaStream_t s, int *launches, MarchUnits *units) {
    if (w.kind[0] || w.kind[1]) return launch_march<LBEM_F32, MARCH_MU, true, 6, 3>(a, w, nsteps, s, launches, units);
    return launch_march<LBEM_F32, MARCH_MU, false, 6, 3>(a, w, nsteps, s, launches, units);
}

cudaError_t launch_march_2d_pole(const StepArgs &a, int nsteps, cudaStream_t s, int *launches, MarchUnits *units) {
    return launch_march<LBEM_F32, MARCH_POLE, false, 6, 3>(a, Walls(), nsteps, s, launches, units);
}

}  // namespace lbk
