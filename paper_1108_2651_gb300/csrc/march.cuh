// The marching kernel: K time steps per launch by streaming rows through registers (2D; instantiated in march.cu,
// march_media.cu and march16.cu).
//
// A warp owns a strip of up to 128 - 2 H columns and a segment of rows, and walks down the rows with K time levels
// in flight: level j (time t + j) computes row Y - j, Y the row level 0 is at.  Level j reads what level j - 1 wrote at
// rows Y - j - 1 (g_2), Y - j (g_0, g_1, g_3 and, by shuffle, their x-neighbours) and Y - j + 1 (g_4, computed just
// before), so 12 registers a lane carry a level from one row to the next, and plane 2, which is read two rows later,
// goes through two shared-memory slots.  H columns on either side (computed by the neighbouring strip too, and dropped
// here) replace any exchange between warps; a segment starts K - 1 rows early and ends K - 1 rows late for the same
// reason.  Rows arrive by cp.async in a per-warp ring, D - 1 rows ahead; the medium stays in shared memory until the
// last level has passed.  There is no barrier: every warp is a block of its own (32 threads), which also makes rows,
// strips and their tests uniform registers and branches.
//
// A state therefore crosses HBM once per K steps: 44 bytes a site per 8 steps in place of 176 with launches of two.
// Every site update is the single-step kernels' arithmetic in their order, so results are bit-identical to theirs
// (16-bit storage: to two steps per launch, the state rounded to the storage after every second step).
#pragma once
#include <algorithm>

#include "lbem_internal.cuh"
#include "march_units.cuh"

namespace lbk {

// Which site update a kernel performs.
enum MarchMedium { MARCH_ISO = 0, MARCH_AN = 1, MARCH_MU = 2, MARCH_POLE = 3 };

// ------------------------------------------------------------------ packed FP32 pairs (each lane of the pair is
// rounded as the scalar operation rounds; half the issue slots)
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 r;
    asm("{.reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n add.rn.f32x2 z, x, y;\n"
        " mov.b64 {%0, %1}, z;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 r;
    asm("{.reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mul.rn.f32x2 z, x, y;\n"
        " mov.b64 {%0, %1}, z;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{.reg .b64 x, y, z, w;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mov.b64 w, {%6, %7};\n"
        " fma.rn.f32x2 z, x, y, w;\n mov.b64 {%0, %1}, z;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
// a - b and a + b of pairs one of which may be a product: the compiler contracts a packed product with the packed sum that
// follows it (also when that is written as a packed fma by 1), so the difference is fma(b, -1, a), one rounding, and the
// sum two scalar ones.
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 sum2(float2 a, float2 b) {
    return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 quad(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }

// ------------------------------------------------------------------ shared memory and asynchronous copies by address
__device__ __forceinline__ void m_cp16(unsigned dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void m_cp8(unsigned dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void m_cp4(unsigned dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ float4 m_lds(unsigned a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a));
    return v;
}
__device__ __forceinline__ float m_lds1(unsigned a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void m_sts1(unsigned a, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v));
}
__device__ __forceinline__ int2 m_lds_int2(unsigned a) {
    int2 v;
    asm volatile("ld.shared.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ int4 m_lds_int4(unsigned a) {
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 m_lds8(unsigned a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ void m_sts(unsigned a, float4 v) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
}

struct Quad5 {
    float4 p0, p1, p2, p3, p4;
};

// ------------------------------------------------------------------ kernel arguments
struct MarchArgs {
    StepArgs a;           // a.in: the state at a.t, a.out: where the state after `steps` steps goes
    Walls w;
    int steps;            // 1 .. K
    int nstrips, nseg;    // units: strips of columns by segments of rows
    // Walls: the first nl and last nr strips hold walled columns or layers; they have nsegx segments, and the first and
    // last segments of the others he rows (0: as the rest)
    int nl, nr, nsegx, he;
};

template <int ST, int MED, int K, int D>
struct MarchCfg {
    // Halo columns on either side.  A level spoils one more column; block-int16 rounding (after every second level, and
    // as the last one is stored) spoils the rest of a group of four that holds a spoilt column, since they share an
    // exponent: four columns per two levels.
    static constexpr int H = ST == LBEM_I16B ? 2 * K : (K + 3) / 4 * 4;
    static constexpr int W = 128 - 2 * H;         // columns a strip can own
    static constexpr int PS = ST == LBEM_F32 ? 512 : 256;                  // bytes of a staged plane row
    static constexpr int SB = 5 * PS + (MED == MARCH_POLE ? 1024 : 0);     // bytes of a stage (POLE: P and J too)
    static constexpr int NM = MED == MARCH_MU ? 3 : MED == MARCH_POLE ? 4 : 1;  // medium planes
    static constexpr int RB = NM * 512, NR = K + D - 1 <= 8 ? 8 : 16;      // the ring of medium rows
    static_assert(K + D - 1 <= NR && K % 2 == 0, "ring of medium rows");
    // then plane 2's slots, and the unit's sources and receivers: 32 records, the sources' currents of K steps, and
    // 32 places for a lane's quads (five planes, a source's S^, the pole's P)
    static constexpr int QB = MED == MARCH_POLE ? 112 : 96;
    static constexpr int O_RING = D * SB, O_G = O_RING + NR * RB, O_EV = O_G + (K - 1) * 1024,
                         O_AMP = O_EV + 512, O_Q = O_AMP + 128 * K, smem = O_Q + 32 * QB;
};

// The state's storage format <-> FP32 of 4 sites.
template <int ST>
__device__ __forceinline__ float4 m_decode(const PopBuf &b, uint2 r, int e) {
    if (ST == LBEM_F16) {
        const float4 v = h4_to_f4(r);
        return make_float4(v.x * b.inv_scale, v.y * b.inv_scale, v.z * b.inv_scale, v.w * b.inv_scale);
    }
    if (ST == LBEM_BF16)
        return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                           __uint_as_float(r.y & 0xffff0000u));
    const float f = i16b_factor(e);
    const float2 l = i16x2_to_f2(r.x, f), h = i16x2_to_f2(r.y, f);
    return make_float4(l.x, l.y, h.x, h.y);
}
template <int ST>
__device__ __forceinline__ int m_encode(const PopBuf &b, float4 v, uint2 &r) {
    if constexpr (ST == LBEM_I16B) {
        return Codec<LBEM_I16B>::enc4e(v, r);
    } else {
        r = Codec<ST>::enc4(b, v);
        return 0;
    }
}
// Encode and decode 4 sites: what reading back the stored state gives.
template <int ST>
__device__ __forceinline__ float4 m_round4(const PopBuf &b, float4 v) {
    if constexpr (ST == LBEM_I16B) {  // Codec::enc4e's steps without packing the mantissas
        const float m = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
        const int e = ((__float_as_int(m) >> 23) & 0xff) - 127 + 1, ec = min(max(e, -99), 100);
        const float s = pow2f(15 - ec), f = m < 0x1p-100f ? 0.f : pow2f(ec - 15);
        auto one = [&](float x) {  // (a zero block: q * 0 + 0 = +0)
            const float q = __fadd_rn(__fadd_rn(fminf(fmaxf(__fmul_rn(x, s), -32767.f), 32767.f), kMagic), -kMagic);
            return __fmaf_rn(q, f, 0.f);
        };
        float4 r = make_float4(one(v.x), one(v.y), one(v.z), one(v.w));
        // huge or NaN: what reading back the saturated block gives, which is not 32767 2^112 (the decoder's product overflows)
        if (!(m < 0x1p+100f)) r.x = r.y = r.z = r.w = i16x2_to_f2(0x7fff7fffu, i16b_factor(127)).x;
        return r;
    } else {
        uint2 r;
        const int e = m_encode<ST>(b, v, r);
        return m_decode<ST>(b, r, e);
    }
}
template <int ST>
__device__ __forceinline__ void m_round(const PopBuf &b, Quad5 &o) {
    if constexpr (ST != LBEM_F32) {
        o.p0 = m_round4<ST>(b, o.p0);
        o.p1 = m_round4<ST>(b, o.p1);
        o.p2 = m_round4<ST>(b, o.p2);
        o.p3 = m_round4<ST>(b, o.p3);
        o.p4 = m_round4<ST>(b, o.p4);
    }
}

// The update of 4 sites without a current source (collide2d_free, collide2d_an, collide2d with the permeability source
// sh, collide2d_pole_iso with P at this level's time); sig: sigma.  Sums and products whose operands lie in the same
// columns go as pairs; g1 and g3 are shifted by a column, so operations with them stay scalar.
template <int MED>
__device__ __forceinline__ void m_collide(float4 g0, float4 g1, float4 g2, float4 g3, float4 g4, float4 c, float4 P,
                                          float4 sh, float r, float ri, float fs, Quad5 &o, float4 &sig) {
    const float2 sa = add2(add2(make_float2(__fadd_rn(g0.x, g1.x), __fadd_rn(g0.y, g1.y)),
                                make_float2(__fadd_rn(g2.x, g3.x), __fadd_rn(g2.y, g3.y))),
                           lo2(g4));
    const float2 sb = add2(add2(make_float2(__fadd_rn(g0.z, g1.z), __fadd_rn(g0.w, g1.w)),
                                make_float2(__fadd_rn(g2.z, g3.z), __fadd_rn(g2.w, g3.w))),
                           hi2(g4));
    sig = quad(sa, sb);
    const float2 ca = lo2(c), cb = hi2(c);
    float2 La = mul2(ca, sa), Lb = mul2(cb, sb);
    float2 wa, wb;  // 2 w0 (doubling is exact)
    if (MED == MARCH_AN) {
        const float2 f2 = make_float2(fs, fs), one = make_float2(1.f, 1.f), two = make_float2(2.f, 2.f);
        wa = mul2(two, sub2(one, mul2(f2, ca)));
        wb = mul2(two, sub2(one, mul2(f2, cb)));
    } else {  // 2 (1 - 2 c) = 2 - 4 c with one rounding: 2 c is exact
        const float2 m4 = make_float2(-4.f, -4.f), two = make_float2(2.f, 2.f);
        wa = fma2(m4, ca, two);
        wb = fma2(m4, cb, two);
    }
    float2 o0a = sub2(mul2(wa, sa), lo2(g0)), o0b = sub2(mul2(wb, sb), hi2(g0));
    if (MED == MARCH_POLE) {
        La = sum2(La, lo2(P));
        Lb = sum2(Lb, hi2(P));
        const float2 m4 = make_float2(-4.f, -4.f);  // 4 P is exact
        o0a = fma2(m4, lo2(P), o0a);
        o0b = fma2(m4, hi2(P), o0b);
    }
    float2 Ya = La, Yb = Lb;
    if (MED == MARCH_AN) {
        const float2 rr = make_float2(r, r), rn = make_float2(ri, ri);
        Ya = mul2(rn, La);
        Yb = mul2(rn, Lb);
        La = mul2(rr, La);
        Lb = mul2(rr, Lb);
    }
    float2 o2a = sub2(Ya, lo2(g4)), o2b = sub2(Yb, hi2(g4)), o4a = sub2(Ya, lo2(g2)), o4b = sub2(Yb, hi2(g2));
    float2 o1a = make_float2(__fsub_rn(La.x, g3.x), __fsub_rn(La.y, g3.y)),
           o1b = make_float2(__fsub_rn(Lb.x, g3.z), __fsub_rn(Lb.y, g3.w)),
           o3a = make_float2(__fsub_rn(La.x, g1.x), __fsub_rn(La.y, g1.y)),
           o3b = make_float2(__fsub_rn(Lb.x, g1.z), __fsub_rn(Lb.y, g1.w));
    if (MED == MARCH_MU) {
        const float2 h = make_float2(-0.5f, -0.5f), sha = lo2(sh), shb = hi2(sh);
        const float2 Ta = mul2(mul2(h, ca), sha), Tb = mul2(mul2(h, cb), shb);    // -c/2 is exact
        const float2 ua = mul2(mul2(h, wa), sha), ub = mul2(mul2(h, wb), shb);    // -w0 is exact
        o0a = sum2(o0a, ua);
        o0b = sum2(o0b, ub);
        o1a = sum2(o1a, Ta);
        o1b = sum2(o1b, Tb);
        o2a = sum2(o2a, Ta);
        o2b = sum2(o2b, Tb);
        o3a = sum2(o3a, Ta);
        o3b = sum2(o3b, Tb);
        o4a = sum2(o4a, Ta);
        o4b = sum2(o4b, Tb);
    }
    o.p0 = quad(o0a, o0b);
    o.p1 = quad(o1a, o1b);
    o.p2 = quad(o2a, o2b);
    o.p3 = quad(o3a, o3b);
    o.p4 = quad(o4a, o4b);
}

// The copies of a row's code: without events; with events, or of a launch of fewer than K steps.
struct MarchPlain {
    static constexpr bool ev = false;
};
struct MarchAny {
    static constexpr bool ev = true;
};

// The march of one unit by one warp: kp steps from a.t.
template <int ST, int MED, bool WL, int K, int D>
__device__ __forceinline__ void march_unit(const StepArgs &a, const Walls &w, int kp, int nstrips, int strip, int y0,
                                           int y1, unsigned smem) {
    using Cfg = MarchCfg<ST, MED, K, D>;
    constexpr int H = Cfg::H, PS = Cfg::PS, SB = Cfg::SB, RB = Cfg::RB, NR = Cfg::NR;
    constexpr bool F32 = ST == LBEM_F32;
    const Grid &G = a.g;
    const int lane = threadIdx.x;
    const int xs = 4 * march_cut(strip, nstrips, G.nchunk);
    const int xe = strip == nstrips - 1 ? G.nx : 4 * march_cut(strip + 1, nstrips, G.nchunk);
    const int X = xs - H + 4 * lane;  // the lane's first column, unwrapped
    const int xw = wrapi(X, G.nx);
    // a lane whose columns are contiguous and aligned copies 16 (8) bytes per plane row; the others (at the wrap of a
    // width that is not a multiple of 4) copy element by element
    const bool direct = (xw & 3) == 0 && xw + 3 < G.nx;
    const bool owned = X >= xs && X < xe;
    const unsigned sl = smem + lane * 16;  // the lane's place in 512-byte rows
    // the next launch's blocks may take their places; this one's inputs are those of the launch before
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const bool hasev = a.evt.rowptr != nullptr;
    unsigned long long smask = 0;  // the event buckets the strip's columns touch
    if (hasev) {
#pragma unroll
        for (int k = 0; k < 4; k++) smask |= 1ull << (wrapi(X + k, G.nx) / a.evt.bucket);
        const unsigned lo = __reduce_or_sync(FULL, (unsigned)smask), hi = __reduce_or_sync(FULL, (unsigned)(smask >> 32));
        smask = ((unsigned long long)hi << 32) | lo;
    }
    const float sx = WL && w.kind[0] == 1 ? -1.f : 1.f, sy = WL && w.kind[1] == 1 ? -1.f : 1.f;
    const float r = MED == MARCH_AN ? a.med.ar : 1.f, ri = MED == MARCH_AN ? __fdiv_rn(1.f, r) : 1.f,
                fs = MED == MARCH_AN ? __fadd_rn(r, ri) : 2.f;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const char *in = static_cast<const char *>(a.in.data);
    char *out = static_cast<char *>(a.out.data);
    const int nit = (y1 - y0) + 2 * (kp - 1);  // rows of level 0
    int lrow = 0, lst = 0, lrs = 0;  // the next row to load, its stage and its medium row
    int r0 = wrapi(y0 - (kp - 1), G.ny);
    int rm = r0 == 0 ? G.ny - 1 : r0 - 1, rp = r0 == G.ny - 1 ? 0 : r0 + 1;
    auto issue = [&]() {
        if (lrow < nit) {
            constexpr int eb = F32 ? 4 : 2;
            const unsigned d = smem + lst * SB + lane * (PS / 32), dm = sl + Cfg::O_RING + lrs * RB;
            const long long o0 = (long long)r0 * G.pitch;
            // with walls, row 0's plane-2 slot and row ny - 1's plane-4 slot hold the site's own opposite plane
            const bool w0 = WL && w.kind[1] && r0 == 0, w1 = WL && w.kind[1] && r0 == G.ny - 1;
            const long long ob[5] = {o0, G.plane + o0,
                                     w0 ? 4 * G.plane + o0 : 2 * G.plane + (long long)rm * G.pitch,
                                     3 * G.plane + o0,
                                     w1 ? 2 * G.plane + o0 : 4 * G.plane + (long long)rp * G.pitch};
            const float *m[4] = {a.med.cL2 + o0, nullptr, nullptr, nullptr};
            if (MED == MARCH_MU) {
                m[1] = a.med.dlnmu + o0;
                m[2] = a.med.dlnmu + G.plane + o0;
            }
            if (MED == MARCH_POLE) {
                m[1] = a.med.pa + o0;
                m[2] = a.med.pb + o0;
                m[3] = a.med.pc + o0;
            }
            if (direct) {
#pragma unroll
                for (int p = 0; p < 5; p++) {
                    if (F32) m_cp16(d + p * PS, in + ob[p] * eb + (unsigned)(xw * eb));
                    else m_cp8(d + p * PS, in + ob[p] * eb + (unsigned)(xw * eb));
                }
                if (MED == MARCH_POLE) {
                    m_cp16(d + 5 * PS, a.med.Pr + o0 + (unsigned)xw);
                    m_cp16(d + 6 * PS, a.med.J + o0 + (unsigned)xw);
                }
#pragma unroll
                for (int k = 0; k < Cfg::NM; k++) m_cp16(dm + k * 512, m[k] + (unsigned)xw);
            } else if (F32) {  // 16-bit rows are whole chunks
#pragma unroll 1
                for (int k = 0; k < 4; k++) {
                    const unsigned x = wrapi(xw + k, G.nx);
#pragma unroll
                    for (int p = 0; p < 5; p++) m_cp4(d + p * PS + 4 * k, in + ob[p] * 4 + x * 4);
                    if (MED == MARCH_POLE) {
                        m_cp4(d + 5 * PS + 4 * k, a.med.Pr + o0 + x);
                        m_cp4(d + 6 * PS + 4 * k, a.med.J + o0 + x);
                    }
#pragma unroll
                    for (int q = 0; q < Cfg::NM; q++) m_cp4(dm + q * 512 + 4 * k, m[q] + x);
                }
            }
            rm = r0;
            r0 = rp;
            rp = rp == G.ny - 1 ? 0 : rp + 1;
            lst = lst == D - 1 ? 0 : lst + 1;
            lrs = (lrs + 1) & (NR - 1);
            lrow++;
        }
        asm volatile("cp.async.commit_group;\n" ::);
    };
#pragma unroll
    for (int k = 0; k < D - 1; k++) issue();

    // block exponents (one byte per lane and plane) of the row after the current one
    int ex[5] = {0, 0, 0, 0, 0};
    int ey = r0;  // unused without block exponents
    auto load_ex = [&](int y) {
        if constexpr (ST == LBEM_I16B) {
            const int ym = y == 0 ? G.ny - 1 : y - 1, yp = y == G.ny - 1 ? 0 : y + 1;
            const int8_t *b = a.in.ex + (xw >> 2);
            const int rows[5] = {y, y, ym, y, yp};
#pragma unroll
            for (int p = 0; p < 5; p++) ex[p] = __ldcg(b + p * a.in.explane + (long long)rows[p] * a.in.expitch);
        }
    };
    if constexpr (ST == LBEM_I16B) {
        ey = wrapi(y0 - (kp - 1), G.ny);
        load_ex(ey);
    }

    float4 A0[K], A1[K], A3[K], PP[K], JJ[K];
#pragma unroll
    for (int j = 0; j < K; j++) A0[j] = A1[j] = A3[j] = PP[j] = JJ[j] = z4;
    unsigned g2a = sl + Cfg::O_G - 1024, g2b = g2a + 512;  // level j's slots of plane 2 at + 1024 j

    // Sources and receivers.  A unit lists those of its rows and columns (of the receivers, those it owns) in shared
    // memory, with the sources' currents of the launch's steps: looked up row by row in global memory they cost a row
    // several dependent loads at each of its levels (1024^2 with 64 receivers: 5.7 us a step, 2.3 without any).  A record
    // is {row (unwrapped), lane | column << 5 | receiver << 7 | place << 8, index, component}; lane l keeps the row of
    // record l; records of one row and lane share a place for the lane's quads.  Units with more than 32 records, or
    // two sources on a site (`many`), look them up in global memory after all, on rows whose mask has one of the strip's
    // columns.
    int erow = -(1 << 30);
    bool many = false;
    unsigned fb = 0;  // the flags of such rows: bit 0 that of level K - 1, bit K - 1 that of level 0, then those below
    if (hasev) {
        int ne = 0;
        const unsigned rec = smem + Cfg::O_EV;
        for (int base = y0 - (kp - 1); base < y1 + (kp - 1) && !many; base += 32) {
            const int row = base + lane, rw = wrapi(row, G.ny);
            const int e0 = __ldg(a.evt.rowptr + rw), e1 = __ldg(a.evt.rowptr + rw + 1);
            const int n = row < y1 + (kp - 1) && (a.evt.mask[rw] & smask) ? e1 - e0 : 0;
            if (__ballot_sync(FULL, n > 0) == 0) continue;
            int sum = n;  // inclusive sums over the lanes (rows)
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(FULL, sum, o);
                if (lane >= o) sum += v;
            }
            const int total = __shfl_sync(FULL, sum, 31);
            for (int i = 0; i < total && !many; i += 32) {
                // the lane's event: number i + lane of the block's, in the row whose sums it lies between
                int q = 0;
#pragma unroll
                for (int o = 16; o; o >>= 1)
                    if (__shfl_sync(FULL, sum, q + o - 1) <= i + lane) q += o;
                const int e = __shfl_sync(FULL, e0, q & 31) + i + lane -
                              (__shfl_sync(FULL, sum, q & 31) - __shfl_sync(FULL, n, q & 31));
                const int yu = base + q;
                int4 ev = make_int4(-1, 0, 0, 0);
                if (i + lane < total) ev = __ldg(reinterpret_cast<const int4 *>(a.evt.ev + e));  // x, kind, index, comp
                int dx0 = ev.x - wrapi(xs - H, G.nx);
                dx0 += dx0 < 0 ? G.nx : 0;
                for (int k = 0; k < 128; k += G.nx) {  // a narrow grid repeats its columns
                    int dx = dx0 + k;
                    bool keep = ev.x >= 0 && dx < 128;
                    if (ev.y) {
                        keep = k == 0 && ev.x >= xs && ev.x < xe && yu >= y0 && yu < y1;
                        dx = ev.x - xs + H;
                    }
                    const unsigned b = __ballot_sync(FULL, keep);
                    const int at = ne + __popc(b & ((1u << lane) - 1));
                    ne += __popc(b);
                    many = ne > 32;
                    if (keep && at < 32) {
                        asm volatile("st.shared.v4.s32 [%0], {%1, %2, %3, %4};" ::"r"(rec + at * 16), "r"(yu),
                                     "r"((dx >> 2) | (dx & 3) << 5 | (ev.y ? 128 : 0)), "r"(ev.z), "r"(ev.w));
                        for (int k = 0; k < kp && ev.y == 0; k++) {
                            float jz = 0.f;  // a component that does not couple, or past the series: no current
                            if (ev.w == 2 && a.t + k < a.evt.nt)
                                jz = __ldg(a.evt.amp + (long long)ev.z * a.evt.nt + a.t + k);
                            if (MED == MARCH_MU)
                                jz = __fmul_rn(jz, __ldg(a.med.mu + (long long)wrapi(yu, G.ny) * G.pitch + ev.x));
                            if (MED == MARCH_AN) jz = __fmul_rn(jz, a.med.amu);
                            m_sts1(smem + Cfg::O_AMP + (at * K + k) * 4, jz);
                        }
                    }
                    if (many) break;
                }
            }
        }
        __syncwarp();
        if (ne > 0 && !many) {
            int2 v = make_int2(-1 - lane, 0);
            if (lane < ne) v = m_lds_int2(rec + lane * 16);
            const unsigned at = __match_any_sync(FULL, v.x * 32 + (v.y & 31));
            const unsigned same = __match_any_sync(FULL, v.y & 127) & at & __ballot_sync(FULL, !(v.y & 128));
            many = __any_sync(FULL, lane < ne && !(v.y & 128) && __popc(same) > 1);
            if (lane < ne) {
                erow = v.x;
                m_sts1(rec + lane * 16 + 4, __int_as_float(v.y | (__ffs(at) - 1) << 8));
                m_sts(smem + Cfg::O_Q + lane * Cfg::QB + 80, z4);
            }
            __syncwarp();
        }
    }
    // An event at column x: the current jz of a source, taken from sh, or a receiver of one of the lane's sites.
    auto event = [&](int x, bool rcv, int index, int comp, float jz, long long tj, const float4 &g0, const float4 &g1,
                     const float4 &g2, const float4 &g3, const float4 &g4, const float4 &c, const float4 &pz, float4 &sh) {
        int d = x - xw;
        d += d < 0 ? G.nx : 0;
#pragma unroll 1
        for (; d < 4; d += G.nx) {
            if (!rcv) {
                set(sh, d, __fsub_rn(get(sh, d), jz));
            } else if (owned && X + d < xe && tj < a.evt.cap) {
                const float q0 = get(g0, d), q1 = get(g1, d), q2 = get(g2, d), q3 = get(g3, d), q4 = get(g4, d);
                float v = field2d(comp, get(c, d), ((q0 + q1) + (q2 + q3)) + q4, q4 - q2, q1 - q3);
                if (MED == MARCH_POLE && comp == 2) v = __fsub_rn(v, get(pz, d));
                if (MED == MARCH_AN && comp == 3) v = __fmul_rn(v, r);
                if (MED == MARCH_AN && comp == 4) v = __fmul_rn(v, ri);
                a.evt.traces[(long long)index * a.evt.cap + tj] = v;
            }
        }
    };
    // The events of unwrapped row yu at level j by the row's list in global memory; whether a source is among them.
    auto events = [&](int yu, int j, const float4 &g0, const float4 &g1, const float4 &g2, const float4 &g3,
                      const float4 &g4, const float4 &c, const float4 &pz, float4 &sh) {
        const long long tj = a.t + j;
        bool src = false;
        if (!((fb >> (K - 1 - j)) & 1)) return false;
        const int row = wrapi(yu, G.ny);
        const int e0 = __ldg(a.evt.rowptr + row), e1 = __ldg(a.evt.rowptr + row + 1);
#pragma unroll 1
        for (int e = e0; e < e1; e++) {
            const int4 ev = __ldg(reinterpret_cast<const int4 *>(a.evt.ev + e));
            float jz = 0.f;
            if (ev.y == 0) {
                if (ev.w != 2 || tj >= a.evt.nt) continue;
                jz = __ldg(a.evt.amp + (long long)ev.z * a.evt.nt + tj);
                if (MED == MARCH_MU) jz = __fmul_rn(jz, __ldg(a.med.mu + (long long)row * G.pitch + ev.x));
                if (MED == MARCH_AN) jz = __fmul_rn(jz, a.med.amu);
                src = true;
            } else if (yu < y0 || yu >= y1) {
                continue;
            }
            event(ev.x, ev.y != 0, ev.z, ev.w, jz, tj, g0, g1, g2, g3, g4, c, pz, sh);
        }
        return src;
    };

    // yl: the row of level 0 (unwrapped), st: its stage, rs: its place in the medium ring.
    int yl = y0 - (kp - 1), st = 0, rs = 0;
    auto ring = [&](int j) {
        return sl + Cfg::O_RING + ((rs - j) & (NR - 1)) * RB;
    };
    // level 0's inputs: a stage, as FP32
    auto stage = [&](unsigned s, float4 &g0, float4 &a1, float4 &g2, float4 &a3, float4 &g4, float4 &P, float4 &J) {
        if constexpr (F32) {
            g0 = m_lds(s);
            a1 = m_lds(s + PS);
            g2 = m_lds(s + 2 * PS);
            a3 = m_lds(s + 3 * PS);
            g4 = m_lds(s + 4 * PS);
            if (MED == MARCH_POLE) {
                P = m_lds(s + 5 * PS);
                J = m_lds(s + 6 * PS);
            }
        } else {
            g0 = m_decode<ST>(a.in, m_lds8(s), ex[0]);
            a1 = m_decode<ST>(a.in, m_lds8(s + PS), ex[1]);
            g2 = m_decode<ST>(a.in, m_lds8(s + 2 * PS), ex[2]);
            a3 = m_decode<ST>(a.in, m_lds8(s + 3 * PS), ex[3]);
            g4 = m_decode<ST>(a.in, m_lds8(s + 4 * PS), ex[4]);
            if constexpr (ST == LBEM_I16B) {
                ey = ey == G.ny - 1 ? 0 : ey + 1;
                load_ex(ey);
            }
        }
    };
    auto store = [&](int yo, const Quad5 &o, float4 Po, float4 Jo) {
        if (yo >= y0 && yo < y1 && owned) {
            const long long oo = (long long)yo * G.pitch + X;
            if constexpr (F32) {
                float *q = reinterpret_cast<float *>(out) + oo;
                __stcs(reinterpret_cast<float4 *>(q), o.p0);
                __stcs(reinterpret_cast<float4 *>(q + G.plane), o.p1);
                __stcs(reinterpret_cast<float4 *>(q + 2 * G.plane), o.p2);
                __stcs(reinterpret_cast<float4 *>(q + 3 * G.plane), o.p3);
                __stcs(reinterpret_cast<float4 *>(q + 4 * G.plane), o.p4);
                if (MED == MARCH_POLE) {
                    __stcs(reinterpret_cast<float4 *>(a.med.Pw + oo), Po);
                    __stcs(reinterpret_cast<float4 *>(a.med.Jw + oo), Jo);
                }
            } else {
                const float4 v[5] = {o.p0, o.p1, o.p2, o.p3, o.p4};
#pragma unroll
                for (int p = 0; p < 5; p++) {
                    uint2 u;
                    const int e = m_encode<ST>(a.in, v[p], u);
                    __stcs(reinterpret_cast<uint2 *>(out + (p * G.plane + oo) * 2), u);
                    if (ST == LBEM_I16B)
                        a.out.ex[p * a.in.explane + (long long)yo * a.in.expitch + (X >> 2)] = (int8_t)e;
                }
            }
        }
    };
    auto mu_src = [&](unsigned mr, float4 g1, float4 g2, float4 g3, float4 g4) {
        const float4 dx = m_lds(mr + 512), dy = m_lds(mr + 1024);
        return make_float4(mu_source(g4.x - g2.x, g1.x - g3.x, dx.x, dy.x),
                           mu_source(g4.y - g2.y, g1.y - g3.y, dx.y, dy.y),
                           mu_source(g4.z - g2.z, g1.z - g3.z, dx.z, dy.z),
                           mu_source(g4.w - g2.w, g1.w - g3.w, dx.w, dy.w));
    };
    auto pole = [&](unsigned mr, float4 c, float4 sig, float4 &J, float4 &P) {
        const float4 pa = m_lds(mr + 512), pb = m_lds(mr + 1024), pc = m_lds(mr + 1536);
        pole_update(c.x, sig.x, pc.x, pb.x, pa.x, J.x, P.x);
        pole_update(c.y, sig.y, pc.y, pb.y, pa.y, J.y, P.y);
        pole_update(c.z, sig.z, pc.z, pb.z, pa.z, J.z, P.z);
        pole_update(c.w, sig.w, pc.w, pb.w, pa.w, J.w, P.w);
    };
    // With walls (WL): the pulls across them, at row yu, given the lane's unshifted planes 1 and 3 and the plane 2
    // computed by the previous iteration (row ny - 1's own), and the absorbing layer.
    auto wall_pulls = [&](int yu, const float4 &h1, const float4 &h3, float4 &g1, float4 &h2, float4 &g3, float4 &h4,
                          bool lev, unsigned prev2) {
        if (w.kind[0]) {
            if (X == 0) g1.x = sx * h3.x;
            const int k = G.nx - 1 - X;
            if ((unsigned)k < 4u) set(g3, k, sx * get(h1, k));
        }
        if (w.kind[1]) {  // the plane-2 value kept for row 0 is plane 4 of the row itself (see below)
            if (yu == 0) h2 = make_float4(sy * h2.x, sy * h2.y, sy * h2.z, sy * h2.w);
            if (yu == G.ny - 1) {
                if (lev) h4 = m_lds(prev2);
                h4 = make_float4(sy * h4.x, sy * h4.y, sy * h4.z, sy * h4.w);
            }
        }
    };
    float4 fx = make_float4(1.f, 1.f, 1.f, 1.f);  // the columns' factors (the table is padded with 1 to the pitch)
    if (WL && w.fx && X >= 0 && X < G.nx) fx = __ldg(reinterpret_cast<const float4 *>(w.fx + X));
    float fyl = 1.f;  // the rows' factors: lane l that of row yl - K + l, as of the last row with it % 16 = 0
    int fy0 = 0;
    auto layer = [&](int yu, Quad5 &n) {
        const float fy = __shfl_sync(FULL, fyl, yu - fy0);
        const float4 f = make_float4(__fmul_rn(fx.x, fy), __fmul_rn(fx.y, fy), __fmul_rn(fx.z, fy), __fmul_rn(fx.w, fy));
        float4 *v[5] = {&n.p0, &n.p1, &n.p2, &n.p3, &n.p4};
#pragma unroll
        for (int p = 0; p < 5; p++)
            *v[p] = make_float4(__fmul_rn(v[p]->x, f.x), __fmul_rn(v[p]->y, f.y), __fmul_rn(v[p]->z, f.z),
                                __fmul_rn(v[p]->w, f.w));
    };
    // The terms of a source S^ at the lane's sites, added last as collide2d adds them.
    auto source = [&](const float4 &c, const float4 &S4, Quad5 &n) {
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const float cl = get(c, k), S = get(S4, k);
            const float w0 = MED == MARCH_AN ? __fsub_rn(1.f, __fmul_rn(fs, cl)) : __fsub_rn(1.f, 2.f * cl);
            const float Tm = __fmul_rn(-0.5f * cl, S), T0 = __fmul_rn(-w0, S);
            const float Tx = MED == MARCH_AN ? __fmul_rn(r, Tm) : Tm;
            const float Ty = MED == MARCH_AN ? __fmul_rn(ri, Tm) : Tm;
            set(n.p0, k, __fadd_rn(get(n.p0, k), T0));
            set(n.p1, k, __fadd_rn(get(n.p1, k), Tx));
            set(n.p2, k, __fadd_rn(get(n.p2, k), Ty));
            set(n.p3, k, __fadd_rn(get(n.p3, k), Tx));
            set(n.p4, k, __fadd_rn(get(n.p4, k), Ty));
        }
    };
    // One row, every level one row further.  EV: a row with events, or in a launch of fewer than K steps; its straight line
    // only hands the quads of the lanes concerned to their places in shared memory, and adds the sources' terms (S^ = 0
    // adds -0 and changes nothing); the records are gone through once, before and after.  With their code at every level
    // the row was 20 KB that the instruction cache did not hold, 3 us against 0.5 us of a plain one.
    auto row = [&](auto mode) {
        constexpr bool EV = decltype(mode)::ev;
        const unsigned s = smem + st * SB + lane * (PS / 32);
        float4 g0, a1, g2, a3, g4, P = z4, J = z4;
        stage(s, g0, a1, g2, a3, g4, P, J);
        issue();
        unsigned levels = 0, recs = 0;  // EV: the levels to leave the line at, the records of the row's levels
        unsigned long long place = 0;   // the lane's place per level (6 bits, 32: none)
        if (EV) {
            if (kp < K) levels = 1u << (kp - 1);
            recs = __ballot_sync(FULL, (unsigned)(yl - erow) < (unsigned)K);
#pragma unroll 1
            for (unsigned b = recs; b; b &= b - 1) {
                const int l = __ffs(b) - 1;
                const int2 v = m_lds_int2(smem + Cfg::O_EV + l * 16);
                const int j = yl - v.x;
                levels |= 1u << j;
                if ((v.y & 31) == lane) {
                    const unsigned q = (unsigned)v.y >> 8;
                    place |= (unsigned long long)(32 | q) << (6 * j);
                    if (!(v.y & 128))
                        m_sts1(smem + Cfg::O_Q + q * Cfg::QB + 80 + ((v.y >> 5) & 3) * 4,
                               __fsub_rn(0.f, m_lds1(smem + Cfg::O_AMP + (l * K + j) * 4)));
                }
            }
        }
        Quad5 o;
        float4 Po = z4, Jo = z4;  // the pole's state after the previous level
#pragma unroll
        for (int j = 0; j < K; j++) {
            Quad5 n;
            const unsigned mr = ring(j);
            const float4 c = m_lds(mr);
            const float4 h0 = j ? A0[j] : g0, h1 = j ? A1[j] : a1, h3 = j ? A3[j] : a3;
            float4 h2 = j ? m_lds(g2a + 1024 * j) : g2, h4 = j ? o.p4 : g4;
            float4 g1 = make_float4(__shfl_up_sync(FULL, h1.w, 1), h1.x, h1.y, h1.z);
            float4 g3 = make_float4(h3.y, h3.z, h3.w, __shfl_down_sync(FULL, h3.x, 1));
            if (WL) wall_pulls(yl - j, h1, h3, g1, h2, g3, h4, j > 0, g2b + 1024 * j);
            float4 sh = z4, S = z4, sig, Pn = j ? PP[j] : P, Jn = j ? JJ[j] : J;
            const bool leave = EV && ((levels >> j) & 1);
            if (MED == MARCH_MU) sh = mu_src(mr, g1, h2, g3, h4);
            if (EV && leave) {
                const unsigned v = (unsigned)(place >> (6 * j)) & 63;
                if (v) {
                    const unsigned q = smem + Cfg::O_Q + (v & 31) * Cfg::QB;
                    m_sts(q, h0);
                    m_sts(q + 16, g1);
                    m_sts(q + 32, h2);
                    m_sts(q + 48, g3);
                    m_sts(q + 64, h4);
                    S = m_lds(q + 80);
                    if (MED == MARCH_POLE) m_sts(q + 96, Pn);
                }
                if (MED == MARCH_MU)
                    sh = make_float4(__fadd_rn(sh.x, S.x), __fadd_rn(sh.y, S.y), __fadd_rn(sh.z, S.z), __fadd_rn(sh.w, S.w));
            }
            m_collide<MED>(h0, g1, h2, g3, h4, c, Pn, sh, r, ri, fs, n, sig);
            if (EV && MED != MARCH_MU && leave) source(c, S, n);
            if (MED == MARCH_POLE) pole(mr, c, sig, Jn, Pn);
            if (WL) layer(yl - j, n);
            // 16-bit storage: the state is rounded after every second step (and as it is stored)
            if (ST != LBEM_F32 && (j & 1) && j != K - 1) m_round<ST>(a.in, n);
            if (j) {  // level j - 1's results become level j's inputs
                A0[j] = o.p0;
                A1[j] = o.p1;
                A3[j] = o.p3;
                m_sts(g2a + 1024 * j, o.p2);
                // level j - 1 has just computed row 0: its plane 4 is what level j pulls back from the wall
                if (WL && w.kind[1] && yl - j == -1) m_sts(g2b + 1024 * j, o.p4);
                PP[j] = Po;
                JJ[j] = Jo;
            }
            if (EV && leave && j < K - 1 && j == kp - 1) store(yl - j, n, Pn, Jn);
            o = n;
            Po = Pn;
            Jo = Jn;
        }
        if (!EV || kp == K) store(yl - (K - 1), o, Po, Jo);
        if (EV) {  // the receivers
#pragma unroll 1
            for (unsigned b = recs; b; b &= b - 1) {
                const int l = __ffs(b) - 1;
                const int4 v = m_lds_int4(smem + Cfg::O_EV + l * 16);
                const long long tj = a.t + (yl - v.x);
                if (!(v.y & 128) || (v.y & 31) != lane || tj >= a.evt.cap || yl - v.x >= kp) continue;
                const unsigned q = smem + Cfg::O_Q + ((unsigned)v.y >> 8) * Cfg::QB + ((v.y >> 5) & 3) * 4;
                const float q0 = m_lds1(q), q1 = m_lds1(q + 16), q2 = m_lds1(q + 32), q3 = m_lds1(q + 48),
                            q4 = m_lds1(q + 64), cl = m_lds1(ring(yl - v.x) + ((v.y >> 5) & 3) * 4);
                float f = field2d(v.w, cl, ((q0 + q1) + (q2 + q3)) + q4, q4 - q2, q1 - q3);
                if (MED == MARCH_POLE && v.w == 2) f = __fsub_rn(f, m_lds1(q + 96));
                if (MED == MARCH_AN && v.w == 3) f = __fmul_rn(f, r);
                if (MED == MARCH_AN && v.w == 4) f = __fmul_rn(f, ri);
                a.evt.traces[(long long)v.z * a.evt.cap + tj] = f;
            }
        }
    };
    // A row of a unit with many events: one level at a time, the levels' registers moving up by one at each, so that the
    // code is a tenth of the unrolled row's.
    auto row_many = [&]() {
        const unsigned s = smem + st * SB + lane * (PS / 32);
        float4 h0, h1, h2, h3, h4, Pn = z4, Jn = z4;
        stage(s, h0, h1, h2, h3, h4, Pn, Jn);
        issue();
#pragma unroll 1
        for (int j = 0; j < K; j++) {
            Quad5 n;
            const unsigned mr = ring(j), slot = 1024 * (j + 1);
            const float4 c = m_lds(mr);
            float4 g1 = make_float4(__shfl_up_sync(FULL, h1.w, 1), h1.x, h1.y, h1.z);
            float4 g3 = make_float4(h3.y, h3.z, h3.w, __shfl_down_sync(FULL, h3.x, 1));
            if (WL) wall_pulls(yl - j, h1, h3, g1, h2, g3, h4, j > 0, g2b + 1024 * j);
            float4 sh = z4, sig;
            bool src = false;
            if (MED == MARCH_MU) sh = mu_src(mr, g1, h2, g3, h4);
            if (j < kp) src = events(yl - j, j, h0, g1, h2, g3, h4, c, Pn, sh);
            m_collide<MED>(h0, g1, h2, g3, h4, c, Pn, sh, r, ri, fs, n, sig);
            if (MED != MARCH_MU && src) source(c, sh, n);
            if (MED == MARCH_POLE) pole(mr, c, sig, Jn, Pn);
            if (WL) layer(yl - j, n);
            if (ST != LBEM_F32 && (j & 1) && j != kp - 1) m_round<ST>(a.in, n);
            if (j == kp - 1) store(yl - j, n, Pn, Jn);
            if (j == K - 1) break;
            // the next level's inputs, and this level's results in their place at the end of the row of registers
            h0 = A0[1];
            h1 = A1[1];
            h3 = A3[1];
            h4 = n.p4;
            h2 = m_lds(g2a + slot);
            m_sts(g2a + slot, n.p2);
            if (WL && w.kind[1] && yl - j == 0) m_sts(g2b + slot, n.p4);
            const float4 Pt = PP[1], Jt = JJ[1];
#pragma unroll
            for (int k = 1; k < K - 1; k++) {
                A0[k] = A0[k + 1];
                A1[k] = A1[k + 1];
                A3[k] = A3[k + 1];
                PP[k] = PP[k + 1];
                JJ[k] = JJ[k + 1];
            }
            A0[K - 1] = n.p0;
            A1[K - 1] = n.p1;
            A3[K - 1] = n.p3;
            PP[K - 1] = Pn;
            JJ[K - 1] = Jn;
            Pn = Pt;
            Jn = Jt;
        }
    };
    auto next_row = [&]() {
        const unsigned tmp = g2a;
        g2a = g2b;
        g2b = tmp;
        yl++;
        st = st == D - 1 ? 0 : st + 1;
        rs = (rs + 1) & (NR - 1);
    };
    auto row_head = [&](int it) {
        if (WL && (it & 15) == 0) {
            fy0 = yl - K;
            const int y = fy0 + lane;
            fyl = w.fy && (unsigned)y < (unsigned)G.ny ? __ldg(w.fy + y) : 1.f;
        }
        asm volatile("cp.async.wait_group %0;\n" ::"n"(D - 2) : "memory");
    };
    // The rows, in loops that hold one copy of the code each (a loop with a second copy in it costs a plain row 150 to 280
    // cycles for the jump across, taken or not).
    int it = 0;
    if (many) {
#pragma unroll 1
        for (; it < nit; it++) {
            if ((it & 15) == 0)  // the flags of the next 16 rows
                fb |= (__ballot_sync(FULL, (a.evt.mask[wrapi(yl + (lane & 15), G.ny)] & smask) != 0) & 0xffffu)
                      << (K - 1);
            row_head(it);
            row_many();
            next_row();
            fb >>= 1;
        }
    }
#pragma unroll 1
    while (it < nit) {
        // the lane's record is on one of the levels' rows from iteration `from` to `from` + K - 1
        const int from = erow - (y0 - (kp - 1));
        const unsigned near = __ballot_sync(FULL, (unsigned)(it - from) < (unsigned)K);
        if (kp < K || near) {
            do {
                row_head(it);
                row(MarchAny());
                next_row();
                it++;
            } while (it < nit && (kp < K || __any_sync(FULL, (unsigned)(it - from) < (unsigned)K)));
        } else {
            // plain rows up to the next record, by twos, so that half of the registers' moves go away (an odd last one
            // of the unit computes a row that nothing keeps; before a record one is left to the other copy)
            int end = __reduce_min_sync(FULL, from > it ? from : 0x7ffffff0);
            end = end >= nit ? nit : it + ((end - it) & ~1);
            if (end == it) {
                row_head(it);
                row(MarchAny());
                next_row();
                it++;
            }
            constexpr int U = WL ? 1 : 2;  // (the longer row with walls singly, to keep its code short)
#pragma unroll 1
            for (; it < end; it += U) {
#pragma unroll
                for (int u = 0; u < U; u++) {
                    row_head(it + u);
                    row(MarchPlain());
                    next_row();
                }
            }
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

template <int ST, int MED, bool WL, int K, int D>
__global__ void __launch_bounds__(32, 8) march2d(const __grid_constant__ MarchArgs m) {
    extern __shared__ __align__(1024) float march_smem[];
    const unsigned smem = (unsigned)__cvta_generic_to_shared(march_smem);
    const Grid &G = m.a.g;
    if constexpr (WL) {
        using Cfg = MarchCfg<ST, MED, K, D>;
        const int nx = m.nl + m.nr, nbx = nx * m.nsegx;  // the walled strips' units first: they are the longer ones
        int strip, y0, y1;
        if (blockIdx.x < nbx) {
            const int seg = blockIdx.x / nx, k = blockIdx.x - seg * nx;
            strip = k < m.nl ? k : m.nstrips - nx + k;
            y0 = march_cut(seg, m.nsegx, G.ny);
            y1 = march_cut(seg + 1, m.nsegx, G.ny);
        } else {
            const int b = blockIdx.x - nbx, n = m.nstrips - nx, seg = b / n;
            strip = m.nl + b - seg * n;
            y0 = march_row(seg, m.nseg, G.ny, m.he);
            y1 = march_row(seg + 1, m.nseg, G.ny, m.he);
        }
        // units away from walls and layers (their reach of K rows and columns included) are periodic ones
        const int edge = max(m.w.nlayer, 1), X0 = 4 * march_cut(strip, m.nstrips, G.nchunk) - Cfg::H;
        if ((m.w.kind[0] && (X0 < edge || X0 + 128 > G.nx - edge)) ||
            (m.w.kind[1] && (y0 - K < edge || y1 + K > G.ny - edge)))
            march_unit<ST, MED, true, K, D>(m.a, m.w, m.steps, m.nstrips, strip, y0, y1, smem);
        else
            march_unit<ST, MED, false, K, D>(m.a, m.w, m.steps, m.nstrips, strip, y0, y1, smem);
    } else {
        const int seg = blockIdx.x / m.nstrips, strip = blockIdx.x - seg * m.nstrips;
        march_unit<ST, MED, false, K, D>(m.a, m.w, m.steps, m.nstrips, strip, march_cut(seg, m.nseg, G.ny),
                                         march_cut(seg + 1, m.nseg, G.ny), smem);
    }
}

// Launches of K steps, the last one of what is left.  One wave of units: as many segments as fill the GPU (a second
// wave would leave it half empty), of at least two rows.  Each launch may start while the one before drains
// (programmatic dependent launch; it waits for its input with griddepcontrol.wait): 128^2 8.2 us a launch against
// 10.3 us, 1024^2 18 us against 20.5 us.  With units, only says what they are.
template <int ST, int MED, bool WL, int K, int D>
static cudaError_t launch_march(const StepArgs &a, const Walls &w, int nsteps, cudaStream_t s, int *launches,
                                MarchUnits *units) {
    using Cfg = MarchCfg<ST, MED, K, D>;
    auto *k = march2d<ST, MED, WL, K, D>;
    static PerDevice<KernelFit> fits;
    KernelFit fit;
    cudaError_t fe = kernel_fit(fits, k, 32, Cfg::smem, &fit, true);
    if (fe != cudaSuccess) return fe;
    MarchArgs m;
    m.a = a;
    m.w = w;
    m.nstrips = (a.g.nchunk + Cfg::W / 4 - 1) / (Cfg::W / 4);
    const int cap = fit.per_sm * fit.nsm;
    m.nl = m.nr = m.nsegx = m.he = 0;
    if (WL && w.kind[0]) {  // strips whose columns (with the halo) reach a wall or its layer
        const int edge = std::max(w.nlayer, 1);
        auto x0 = [&](int k) { return 4 * march_cut(k, m.nstrips, a.g.nchunk) - Cfg::H; };
        while (m.nl < m.nstrips && x0(m.nl) < edge) m.nl++;
        while (m.nl + m.nr < m.nstrips && x0(m.nstrips - 1 - m.nr) + 128 > a.g.nx - edge) m.nr++;
    }
    // a walled unit's row takes up to three times a periodic one's: a third of the rows (4096^2 with a 32-site layer, 200
    // steps: 5.2 ms, with half of the rows 6.1, with two thirds 7.1)
    m.nseg = std::max(1, std::min(cap / (m.nstrips + 2 * (m.nl + m.nr)), a.g.ny / 2));
    m.nsegx = std::max(1, std::min(3 * m.nseg, a.g.ny / 2));
    if (WL && w.kind[1] && m.nseg >= 4) {
        const int reach = std::max(w.nlayer, 1) + K, he = std::max(reach, a.g.ny / m.nseg / 3 - (K - 1));
        if (2 * he + (m.nseg - 2) * 2 <= a.g.ny) m.he = he;
    }
    if (units) {
        units->K = K;
        units->H = Cfg::H;
        units->nstrips = m.nstrips;
        units->nseg = m.nseg;
        units->nl = m.nl;
        units->nr = m.nr;
        units->nsegx = m.nsegx;
        units->he = m.he;
        return cudaSuccess;
    }
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((m.nl + m.nr) * m.nsegx + (m.nstrips - m.nl - m.nr) * m.nseg));
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
        if (MED == MARCH_POLE) {
            float *J = const_cast<float *>(m.a.med.J), *P = const_cast<float *>(m.a.med.Pr);
            m.a.med.J = m.a.med.Jw;
            m.a.med.Pr = m.a.med.Pw;
            m.a.med.Jw = J;
            m.a.med.Pw = P;
        }
    }
    return cudaSuccess;
}

}  // namespace lbk
