// The 3D (D3Q7) site update, shared by the single-step kernels (kernels3d.cu) and the kernel of several steps per launch
// (march3d.cu).  Written with explicitly rounded operations, so that every kernel performs the same roundings whatever the
// compiler contracts around it; the scheme is stated in kernels3d.cu.
#pragma once
#include "lbem_internal.cuh"

namespace lbk {

struct Mom3 {
    float sx, sy, sz, bx, by, bz;
};

__device__ __forceinline__ Mom3 moments3(const float h[21]) {
    Mom3 m;
    m.sx = ((h[0] + h[3]) + (h[6] + h[9])) + ((h[12] + h[15]) + h[18]);
    m.sy = ((h[1] + h[4]) + (h[7] + h[10])) + ((h[13] + h[16]) + h[19]);
    m.sz = ((h[2] + h[5]) + (h[8] + h[11])) + ((h[14] + h[17]) + h[20]);
    // R_{gamma kappa} = h[(1+kappa)*3 + gamma] - h[(4+kappa)*3 + gamma]
    m.bx = (h[10] - h[19]) - (h[8] - h[17]);   // R_yz - R_zy
    m.by = (h[5] - h[14]) - (h[9] - h[18]);    // R_zx - R_xz
    m.bz = (h[6] - h[15]) - (h[4] - h[13]);    // R_xy - R_yx
    return m;
}

__device__ __forceinline__ float field3d(int comp, float cl, const Mom3 &m) {
    switch (comp) {
        case 0: return -cl * m.sx;
        case 1: return -cl * m.sy;
        case 2: return -cl * m.sz;
        case 3: return m.bx;
        case 4: return m.by;
        default: return m.bz;
    }
}

// In-place collision of one site without a source: h[p] <- h'[p].  (lambda +- B/2 by fma: B/2 is exact.  The
// population moving +x takes its lambda unrounded, the others the rounded one: the roundings that results have always had.)
__device__ __forceinline__ void collide3d_free(float h[21], float cl) {
    const Mom3 m = moments3(h);
    const float w2 = 2.f * __fmaf_rn(-3.f, cl, 1.f);
    const float lx = __fmul_rn(cl, m.sx), ly = __fmul_rn(cl, m.sy), lz = __fmul_rn(cl, m.sz);
    const float xpy = __fmaf_rn(0.5f, m.by, lx), xmy = __fmaf_rn(-0.5f, m.by, lx);
    const float xpz = __fmaf_rn(0.5f, m.bz, lx), xmz = __fmaf_rn(-0.5f, m.bz, lx);
    const float ypx = __fmaf_rn(0.5f, m.bx, ly), ymx = __fmaf_rn(-0.5f, m.bx, ly);
    const float ypz = __fmaf_rn(0.5f, m.bz, ly), ymz = __fmaf_rn(-0.5f, m.bz, ly);
    const float zpx = __fmaf_rn(0.5f, m.bx, lz), zmx = __fmaf_rn(-0.5f, m.bx, lz);
    const float zpy = __fmaf_rn(0.5f, m.by, lz), zmy = __fmaf_rn(-0.5f, m.by, lz);
    // rest
    h[0] = __fmaf_rn(w2, m.sx, -h[0]);
    h[1] = __fmaf_rn(w2, m.sy, -h[1]);
    h[2] = __fmaf_rn(w2, m.sz, -h[2]);
    // +x: c x B = (0, -Bz, By)
    h[3] = __fmaf_rn(cl, m.sx, -h[3]);
    h[4] = __fsub_rn(ymz, h[4]);
    h[5] = __fsub_rn(zpy, h[5]);
    // +y: c x B = (Bz, 0, -Bx)
    h[6] = __fsub_rn(xpz, h[6]);
    h[7] = __fsub_rn(ly, h[7]);
    h[8] = __fsub_rn(zmx, h[8]);
    // +z: c x B = (-By, Bx, 0)
    h[9] = __fsub_rn(xmy, h[9]);
    h[10] = __fsub_rn(ypx, h[10]);
    h[11] = __fsub_rn(lz, h[11]);
    // -x
    h[12] = __fsub_rn(lx, h[12]);
    h[13] = __fsub_rn(ypz, h[13]);
    h[14] = __fsub_rn(zmy, h[14]);
    // -y
    h[15] = __fsub_rn(xmz, h[15]);
    h[16] = __fsub_rn(ly, h[16]);
    h[17] = __fsub_rn(zpx, h[17]);
    // -z
    h[18] = __fsub_rn(xpy, h[18]);
    h[19] = __fsub_rn(ymx, h[19]);
    h[20] = __fsub_rn(lz, h[20]);
}

// The source's terms, added last: T_m = -(c_L^2/4) S^ (moving), T_0 = -(w0/2) S^ (rest).
__device__ __forceinline__ void source3d(float h[21], float cl, float shx, float shy, float shz) {
    const float q = -0.25f * cl, w = -0.5f * __fmaf_rn(-3.f, cl, 1.f);  // exact but for w0's rounding
    const float sh[3] = {shx, shy, shz};
#pragma unroll
    for (int k = 0; k < 3; k++) {
        h[k] = __fmaf_rn(w, sh[k], h[k]);
#pragma unroll
        for (int i = 1; i < 7; i++) h[3 * i + k] = __fmaf_rn(q, sh[k], h[3 * i + k]);
    }
}

// S^ = B x grad ln mu of Eq. 3.
__device__ __forceinline__ void mu_source3(const Mom3 &m, float dx, float dy, float dz, float &shx, float &shy, float &shz) {
    shx = __fmaf_rn(m.by, dz, -__fmul_rn(m.bz, dy));
    shy = __fmaf_rn(m.bz, dx, -__fmul_rn(m.bx, dz));
    shz = __fmaf_rn(m.bx, dy, -__fmul_rn(m.by, dx));
}

// Walls (walls.cu, in 3D): a population h_{i gamma} pulled across a wall normal to axis a is the site's own
// h_{opp(i) gamma} times wall_sign3(kind, gamma, a): the geometric mirror of the tensor component it carries
// (+1 when gamma == a, -1 otherwise) times +1 for PEC and -1 for PMC.
__device__ __forceinline__ float wall_sign3(int kind, int gm, int ax) {
    return (kind == 1 ? 1.f : -1.f) * (gm == ax ? 1.f : -1.f);
}

}  // namespace lbk
