// The marching kernel (march.cuh) for FP32 storage and an isotropic medium of uniform permeability, without walls or a
// pole: its launch geometry and the launches of a call.
//
// What bounds it (4096^2, 8 steps a launch): latency, with two warps a scheduler; no unit is full.  A launch without events
// takes 127 us (134 under ncu, whose counters these are): 737 MB of HBM traffic (447 read, 290 written; 738 are the state's
// and the medium's), 69 % of its rate; shared memory 60 % of its wavefronts (a tenth of them bank conflicts), with the
// global accesses 70 % of that pipe; 1.8 of 4 issue slots.  Of the 4.3 cycles between a warp's instructions 1.2 wait for
// rows from HBM, 0.6 for the fixed latency of the instruction before, 0.4 for shared memory, 0.3 for the arithmetic pipe
// and 0.3 for instructions.  With a source and a ring of 64 receivers a launch takes 141 to 163 us by the ring's radius:
// the slowest unit of the one wave decides (176 us under ncu, HBM 53 %).  The strip kernel moves the same bytes
// for 2 steps in 121 us.  Below about 2048^2 the state stays in L2 and a launch takes its rows' latency: about 0.45 us a
// row for a warp alone on its scheduler (a row is 8 updates of 4 sites a lane, some 430 instructions), for R + 14 rows.
// K = 8: four levels cost 32 us a step at 4096^2 and six 20.6 us against 16.0 us (1024^2: 2.57, 2.25
// and 2.26 us; 256^2: 1.49, 1.31 and 1.44 us); ten and twelve
// levels do not fit the registers of 8 warps an SM without spilling (18.3 and 16.2 us a step).
// 8 warps an SM (two per scheduler): 12 warps allow 168 registers, which K = 8 spills.  D = 3 rows of staging: with 4
// the 4096^2 launch takes 136 us (more reads in flight, but further from the writes), 2048^2 38 us against 39 us.
#include "march.cuh"

namespace lbk {

cudaError_t launch_march_2d(const StepArgs &a, const Walls &w, int storage, bool aniso, int nsteps, cudaStream_t s,
                            int *launches, MarchUnits *units) {
    const bool walls = w.kind[0] || w.kind[1];
    if (storage != LBEM_F32) return launch_march_2d_16(a, storage, nsteps, s, launches, units);
    if (a.med.wp2) return launch_march_2d_pole(a, nsteps, s, launches, units);
    if (aniso) return launch_march_2d_an(a, w, nsteps, s, launches, units);
    if (a.med.dlnmu) return launch_march_2d_mu(a, w, nsteps, s, launches, units);
    if (walls) return launch_march<LBEM_F32, MARCH_ISO, true, 8, 3>(a, w, nsteps, s, launches, units);
    return launch_march<LBEM_F32, MARCH_ISO, false, 8, 3>(a, w, nsteps, s, launches, units);
}

}  // namespace lbk
