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

// The direction opposite to i (of planes 3 i + gamma), as a plane.
__host__ __device__ constexpr int opp3(int p) { return p < 3 ? p : p < 12 ? p + 9 : p - 9; }

// What a site's events add to its adjoint update: the point current, and the receivers' cotangents by component.
struct AdjEvents3 {
    float j[3], rE[3], rB[3];
};

// One site of the adjoint step (adjoint.cu states it): v[opp3(p)] = mu_p, the populations of lambda^{t+1} pulled as the
// forward step pulls (lambda is stored by opposite directions), becomes lambda^t in the same order; returns the step's
// contribution to dL/dc_L^2.  sg: sigma of g^t, q: c_L^2.
__device__ __forceinline__ float adjoint3_site(float v[21], const float sg[3], float q, const AdjEvents3 &ev) {
    float h[21];
#pragma unroll
    for (int p = 0; p < 21; p++) h[p] = v[opp3(p)];
    const float w0 = __fmaf_rn(-3.f, q, 1.f), hq = 0.5f * q;
    float mv[3], L[3];
    float d = 0.f;
#pragma unroll
    for (int g = 0; g < 3; g++) {
        mv[g] = ((h[3 + g] + h[6 + g]) + (h[9 + g] + h[12 + g])) + (h[15 + g] + h[18 + g]);
        L[g] = 2.f * __fmaf_rn(w0, h[g], __fmul_rn(hq, mv[g]));
        d = __fadd_rn(d, __fmaf_rn(sg[g], mv[g], -__fmul_rn(6.f, __fmul_rn(sg[g], h[g]))));
        d = __fmaf_rn(ev.j[g], __fmaf_rn(0.25f, mv[g], -__fmul_rn(1.5f, h[g])), d);
    }
    // V = sum_i mu_i x c_i, the same contraction that reads B from h (V/2 is exact)
    const float vx = (h[10] - h[19]) - (h[8] - h[17]);
    const float vy = (h[5] - h[14]) - (h[9] - h[18]);
    const float vz = (h[6] - h[15]) - (h[4] - h[13]);
    const float xpy = __fmaf_rn(0.5f, vy, L[0]), xmy = __fmaf_rn(-0.5f, vy, L[0]);
    const float xpz = __fmaf_rn(0.5f, vz, L[0]), xmz = __fmaf_rn(-0.5f, vz, L[0]);
    const float ypx = __fmaf_rn(0.5f, vx, L[1]), ymx = __fmaf_rn(-0.5f, vx, L[1]);
    const float ypz = __fmaf_rn(0.5f, vz, L[1]), ymz = __fmaf_rn(-0.5f, vz, L[1]);
    const float zpx = __fmaf_rn(0.5f, vx, L[2]), zmx = __fmaf_rn(-0.5f, vx, L[2]);
    const float zpy = __fmaf_rn(0.5f, vy, L[2]), zmy = __fmaf_rn(-0.5f, vy, L[2]);
    float o[21] = {L[0], L[1], L[2],      // rest
                   L[0], ymz, zpy,        // +x: c x V = (0, -Vz, Vy)
                   xpz, L[1], zmx,        // +y: (Vz, 0, -Vx)
                   xmy, ypx, L[2],        // +z: (-Vy, Vx, 0)
                   L[0], ypz, zmy,        // -x
                   xmz, L[1], zpx,        // -y
                   xpy, ymx, L[2]};       // -z
#pragma unroll
    for (int p = 0; p < 21; p++) o[p] = __fsub_rn(o[p], h[p]);
    // receivers: E_gamma = -c_L^2 sigma_gamma;  B_nu = eps_{gamma kappa nu} sum_i c_{i kappa} g_{i gamma}
#pragma unroll
    for (int g = 0; g < 3; g++)
        if (ev.rE[g] != 0.f) {
#pragma unroll
            for (int i = 0; i < 7; i++) o[3 * i + g] = __fmaf_rn(-q, ev.rE[g], o[3 * i + g]);
            d = __fmaf_rn(-sg[g], ev.rE[g], d);
        }
    if (ev.rB[0] != 0.f || ev.rB[1] != 0.f || ev.rB[2] != 0.f) {
        o[10] += ev.rB[0]; o[19] -= ev.rB[0]; o[8] -= ev.rB[0]; o[17] += ev.rB[0];
        o[5] += ev.rB[1]; o[14] -= ev.rB[1]; o[9] -= ev.rB[1]; o[18] += ev.rB[1];
        o[6] += ev.rB[2]; o[15] -= ev.rB[2]; o[4] -= ev.rB[2]; o[13] += ev.rB[2];
    }
#pragma unroll
    for (int p = 0; p < 21; p++) v[opp3(p)] = o[p];
    return d;
}

// Adds event e of site time t to ev (cot: the receivers' cotangents [nrec][nsteps] of the steps from t0).
__device__ __forceinline__ void adjoint3_event(AdjEvents3 &ev, const Event &e, const Events &E, const float *cot,
                                               int nsteps, long long t, long long t0) {
    if (e.kind == 0) {
        if (t < E.nt) {
            const float jj = __ldg(E.amp + (long long)e.index * E.nt + t);
#pragma unroll
            for (int g = 0; g < 3; g++)
                if (e.comp == g) ev.j[g] += jj;
        }
    } else {
        const long long n = t - t0;
        if (n < 0 || n >= nsteps || t >= E.cap) return;
        const float r = __ldg(cot + (long long)e.index * nsteps + n);
#pragma unroll
        for (int g = 0; g < 3; g++) {
            if (e.comp == g) ev.rE[g] += r;
            if (e.comp == 3 + g) ev.rB[g] += r;
        }
    }
}

}  // namespace lbk
