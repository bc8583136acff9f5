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
#include "lbem_internal.cuh"

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
// a - b and a + b of pairs one of which is a product: as fma(b, -1, a) and fma(b, 1, a), one rounding each, since the
// compiler contracts a packed product with the packed sum that follows it.
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 sum2(float2 a, float2 b) { return fma2(b, make_float2(1.f, 1.f), a); }
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
    int nstrips, nseg;    // units: strip s, segment g is block g * nstrips + s
};

// The unit's column and row ranges: whole chunks of 4 columns and rows, evenly.
__host__ __device__ __forceinline__ int march_cut(int k, int n, int of) { return (int)((long long)k * of / n); }

template <int ST, int MED, int K, int D>
struct MarchCfg {
    static constexpr int H = (K + 3) / 4 * 4;     // halo columns on either side
    static constexpr int W = 128 - 2 * H;         // columns a strip can own
    static constexpr int PS = ST == LBEM_F32 ? 512 : 256;                  // bytes of a staged plane row
    static constexpr int SB = 5 * PS + (MED == MARCH_POLE ? 1024 : 0);     // bytes of a stage (POLE: P and J too)
    static constexpr int NM = MED == MARCH_MU ? 3 : MED == MARCH_POLE ? 4 : 1;  // medium planes
    static constexpr int RB = NM * 512, NR = K + D - 1 <= 8 ? 8 : 16;      // the ring of medium rows
    static_assert(K + D - 1 <= NR && K % 2 == 0, "ring of medium rows");
    static constexpr int XB = ST == LBEM_F32 ? 0 : 2560;                   // event scratch (FP32: the stage just read)
    static constexpr int O_RING = D * SB, O_G = O_RING + NR * RB, O_X = O_G + (K - 1) * 1024, smem = O_X + XB;
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
template <int ST>
__device__ __forceinline__ void m_round(const PopBuf &b, Quad5 &o) {
    if constexpr (ST != LBEM_F32) {
        float4 *v[5] = {&o.p0, &o.p1, &o.p2, &o.p3, &o.p4};
#pragma unroll
        for (int p = 0; p < 5; p++) {
            uint2 r;
            const int e = m_encode<ST>(b, *v[p], r);
            *v[p] = m_decode<ST>(b, r, e);
        }
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

// The march of one unit by one warp: kp steps from a.t.
template <int ST, int MED, bool WL, int K, int D>
__device__ __forceinline__ void march_unit(const StepArgs &a, const Walls &w, int kp, int nstrips, int nseg, int strip,
                                           int seg, unsigned smem) {
    using Cfg = MarchCfg<ST, MED, K, D>;
    constexpr int H = Cfg::H, PS = Cfg::PS, SB = Cfg::SB, RB = Cfg::RB, NR = Cfg::NR;
    constexpr bool F32 = ST == LBEM_F32;
    const Grid &G = a.g;
    const int lane = threadIdx.x;
    const int xs = 4 * march_cut(strip, nstrips, G.nchunk);
    const int xe = strip == nstrips - 1 ? G.nx : 4 * march_cut(strip + 1, nstrips, G.nchunk);
    const int y0 = march_cut(seg, nseg, G.ny), y1 = march_cut(seg + 1, nseg, G.ny);
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
    // columns whose update a wall or a layer changes
    const int edge_x = WL ? max(w.nlayer, 1) : 0;
    const bool xslow = WL && w.kind[0] && (xs - H < edge_x || xs - H + 128 > G.nx - edge_x);
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

    // Sources and receivers of row `row` at time tj: receivers written, the sources' part of S^ added to sh.  The
    // lane's populations are read by column from `scr` (planes 512 bytes apart) and c_L^2 from `mr`.
    auto events = [&](int row, long long tj, bool rec, unsigned scr, unsigned mr, float4 pz, float4 &sh) {
        const int e0 = __ldg(a.evt.rowptr + row), e1 = __ldg(a.evt.rowptr + row + 1);
#pragma unroll 1
        for (int e = e0; e < e1; e++) {
            const int4 ev = __ldg(reinterpret_cast<const int4 *>(a.evt.ev + e));  // x, kind, index, comp
            int d = ev.x - xw;
            if (d < 0) d += G.nx;
#pragma unroll 1
            for (; d < 4; d += G.nx) {
                if (ev.y == 0) {
                    if (ev.w == 2 && tj < a.evt.nt) {
                        float jz = __ldg(a.evt.amp + (long long)ev.z * a.evt.nt + tj);
                        if (MED == MARCH_MU) jz = __fmul_rn(jz, __ldg(a.med.mu + (long long)row * G.pitch + ev.x));
                        if (MED == MARCH_AN) jz = __fmul_rn(jz, a.med.amu);
                        set(sh, d, __fsub_rn(get(sh, d), jz));
                    }
                } else if (rec && X + d < xe && tj < a.evt.cap) {
                    const float q0 = m_lds1(scr + 4 * d), q1 = m_lds1(scr + 512 + 4 * d),
                                q2 = m_lds1(scr + 1024 + 4 * d), q3 = m_lds1(scr + 1536 + 4 * d),
                                q4 = m_lds1(scr + 2048 + 4 * d), cl = m_lds1(mr + 4 * d);
                    float v = field2d(ev.w, cl, ((q0 + q1) + (q2 + q3)) + q4, q4 - q2, q1 - q3);
                    if (MED == MARCH_POLE && ev.w == 2) v = __fsub_rn(v, get(pz, d));
                    if (MED == MARCH_AN && ev.w == 3) v = __fmul_rn(v, r);
                    if (MED == MARCH_AN && ev.w == 4) v = __fmul_rn(v, ri);
                    a.evt.traces[(long long)ev.z * a.evt.cap + tj] = v;
                }
            }
        }
    };

    // Event flags of the rows: bit 0 that of level K - 1, bit K - 1 that of level 0, then those below.  yl: the row
    // of level 0 (unwrapped), st: its stage, rs: its place in the medium ring.
    unsigned fb = 0;
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
    // A row with every level busy and no event or wall, FP32 storage.
    auto row_plain = [&]() {
        const unsigned s = smem + st * SB + lane * (PS / 32);
        float4 g0, a1, g2, a3, g4, P = z4, J = z4;
        stage(s, g0, a1, g2, a3, g4, P, J);
        issue();
        Quad5 o;
        float4 Po = z4, Jo = z4;
#pragma unroll
        for (int j = 0; j < K; j++) {
            Quad5 n;
            const unsigned mr = ring(j);
            const float4 c = m_lds(mr);
            const float4 h0 = j ? A0[j] : g0, h1 = j ? A1[j] : a1, h2 = j ? m_lds(g2a + 1024 * j) : g2,
                         h3 = j ? A3[j] : a3, h4 = j ? o.p4 : g4;
            const float4 g1 = make_float4(__shfl_up_sync(FULL, h1.w, 1), h1.x, h1.y, h1.z);
            const float4 g3 = make_float4(h3.y, h3.z, h3.w, __shfl_down_sync(FULL, h3.x, 1));
            float4 sh = z4, sig, Pn = j ? PP[j] : P, Jn = j ? JJ[j] : J;
            if (MED == MARCH_MU) sh = mu_src(mr, g1, h2, g3, h4);
            m_collide<MED>(h0, g1, h2, g3, h4, c, Pn, sh, r, ri, fs, n, sig);
            if (MED == MARCH_POLE) pole(mr, c, sig, Jn, Pn);
            if (j) {
                A0[j] = o.p0;
                A1[j] = o.p1;
                A3[j] = o.p3;
                m_sts(g2a + 1024 * j, o.p2);
                PP[j] = Po;
                JJ[j] = Jo;
            }
            o = n;
            Po = Pn;
            Jo = Jn;
        }
        store(yl - (K - 1), o, Po, Jo);
    };
    // Any row: with events, walls, levels that have not started, fewer than K levels, rounded storage.
    auto row_full = [&](int it) {
        const unsigned s = smem + st * SB + lane * (PS / 32);
        float4 g0, a1, g2, a3, g4, P = z4, J = z4;
        stage(s, g0, a1, g2, a3, g4, P, J);
        issue();
        const unsigned scr = F32 ? s : sl + Cfg::O_X;  // the lane's event scratch
        const int nact = min(kp, it / 2 + 1);          // levels with a row to compute
        Quad5 o;
        float4 Po = z4, Jo = z4;  // the pole's state after the previous level
#pragma unroll
        for (int j = 0; j < K; j++) {
            if (j > nact) break;
            Quad5 n;
            float4 Pn = z4, Jn = z4;
            const bool act = j < nact;
            const int yu = yl - j;  // unwrapped
            if (act) {
                const unsigned mr = ring(j);
                const float4 c = m_lds(mr);
                const float4 h0 = j ? A0[j] : g0, h1 = j ? A1[j] : a1, h3 = j ? A3[j] : a3;
                float4 h2 = j ? m_lds(g2a + 1024 * j) : g2, h4 = j ? o.p4 : g4;
                Pn = j ? PP[j] : P;
                Jn = j ? JJ[j] : J;
                float4 g1 = make_float4(__shfl_up_sync(FULL, h1.w, 1), h1.x, h1.y, h1.z);
                float4 g3 = make_float4(h3.y, h3.z, h3.w, __shfl_down_sync(FULL, h3.x, 1));
                if (WL) {  // pulls across walls
                    if (w.kind[0]) {
                        if (X == 0) g1.x = sx * h3.x;
                        const int k = G.nx - 1 - X;
                        if ((unsigned)k < 4u) set(g3, k, sx * get(h1, k));
                    }
                    if (w.kind[1]) {
                        // the plane-2 value kept for row 0 is plane 4 of the row itself (see below); for row
                        // ny - 1, plane 2 of the row is the one computed by the previous iteration
                        if (yu == 0) h2 = make_float4(sy * h2.x, sy * h2.y, sy * h2.z, sy * h2.w);
                        if (yu == G.ny - 1) {
                            if (j) h4 = m_lds(g2b + 1024 * j);
                            h4 = make_float4(sy * h4.x, sy * h4.y, sy * h4.z, sy * h4.w);
                        }
                    }
                }
                float4 sh = z4;
                if (MED == MARCH_MU) sh = mu_src(mr, g1, h2, g3, h4);
                bool src = false;
                if ((fb >> (K - 1 - j)) & 1) {
                    m_sts(scr, h0);
                    m_sts(scr + 512, g1);
                    m_sts(scr + 1024, h2);
                    m_sts(scr + 1536, g3);
                    m_sts(scr + 2048, h4);
                    events(wrapi(yu, G.ny), a.t + j, owned && yu >= y0 && yu < y1, scr, mr, Pn, sh);
                    src = true;
                }
                float4 sig;
                m_collide<MED>(h0, g1, h2, g3, h4, c, Pn, sh, r, ri, fs, n, sig);
                if (MED == MARCH_POLE) pole(mr, c, sig, Jn, Pn);
                if (MED != MARCH_MU && src) {  // the sources' terms, added last as collide2d adds them
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        const float cl = get(c, k), S = get(sh, k);
                        const float w0 = MED == MARCH_AN ? __fsub_rn(1.f, __fmul_rn(fs, cl))
                                                         : __fsub_rn(1.f, 2.f * cl);
                        const float Tm = __fmul_rn(-0.5f * cl, S), T0 = __fmul_rn(-w0, S);
                        const float Tx = MED == MARCH_AN ? __fmul_rn(r, Tm) : Tm;
                        const float Ty = MED == MARCH_AN ? __fmul_rn(ri, Tm) : Tm;
                        set(n.p0, k, __fadd_rn(get(n.p0, k), T0));
                        set(n.p1, k, __fadd_rn(get(n.p1, k), Tx));
                        set(n.p2, k, __fadd_rn(get(n.p2, k), Ty));
                        set(n.p3, k, __fadd_rn(get(n.p3, k), Tx));
                        set(n.p4, k, __fadd_rn(get(n.p4, k), Ty));
                    }
                }
                if (WL && (w.fx || w.fy)) {  // the absorbing layer
                    const float fy = w.fy && (unsigned)yu < (unsigned)G.ny ? __ldg(w.fy + yu) : 1.f;
                    float4 f = make_float4(fy, fy, fy, fy);
                    if (w.fx && X >= 0 && X < G.nx) {  // the table is padded with 1 to the pitch
                        const float4 fx = __ldg(reinterpret_cast<const float4 *>(w.fx + X));
                        f = make_float4(__fmul_rn(fx.x, fy), __fmul_rn(fx.y, fy), __fmul_rn(fx.z, fy),
                                        __fmul_rn(fx.w, fy));
                    }
                    float4 *v[5] = {&n.p0, &n.p1, &n.p2, &n.p3, &n.p4};
#pragma unroll
                    for (int p = 0; p < 5; p++)
                        *v[p] = make_float4(__fmul_rn(v[p]->x, f.x), __fmul_rn(v[p]->y, f.y),
                                            __fmul_rn(v[p]->z, f.z), __fmul_rn(v[p]->w, f.w));
                }
                // 16-bit storage: the state is rounded after every second step (K is even)
                if (ST != LBEM_F32 && (j & 1) && j != K - 1) m_round<ST>(a.in, n);
            }
            if (j) {  // level j - 1's results become level j's inputs
                A0[j] = o.p0;
                A1[j] = o.p1;
                A3[j] = o.p3;
                m_sts(g2a + 1024 * j, o.p2);
                // level j - 1 has just computed row 0: its plane 4 is what level j pulls back from the wall
                if (WL && w.kind[1] && yu == -1) m_sts(g2b + 1024 * j, o.p4);
                PP[j] = Po;
                JJ[j] = Jo;
            }
            if (act) {
                o = n;
                Po = Pn;
                Jo = Jn;
            }
        }
        store(yl - (kp - 1), o, Po, Jo);  // (all kp levels are busy by then)
    };
    auto next_row = [&]() {
        const unsigned tmp = g2a;
        g2a = g2b;
        g2b = tmp;
        yl++;
        st = st == D - 1 ? 0 : st + 1;
        rs = (rs + 1) & (NR - 1);
    };
    // Rows by twos (an odd last one computes a row that nothing keeps): unrolled, so that half of the registers'
    // moves go away, where both are plain; the other copy is out of the loop's way.
#pragma unroll 1
    for (int it = 0; it < nit; it += 2) {
        if (hasev && (it & 15) == 0)  // the flags of the next 16 rows
            fb |= (__ballot_sync(FULL, (a.evt.mask[wrapi(yl + (lane & 15), G.ny)] & smask) != 0) & 0xffffu)
                  << (K - 1);
        bool full = !F32 || kp < K || (fb & ((2u << K) - 1)) != 0;
        if (WL) {
            const int edge_y = max(w.nlayer, 1);
            full |= xslow || (w.kind[1] && (yl - (K - 1) < edge_y || yl + 1 >= G.ny - edge_y));
        }
        if (__builtin_expect(!full, 1)) {
#pragma unroll
            for (int u = 0; u < 2; u++) {
                asm volatile("cp.async.wait_group %0;\n" ::"n"(D - 2) : "memory");
                row_plain();
                next_row();
            }
        } else {
#pragma unroll 1
            for (int u = 0; u < 2; u++) {
                asm volatile("cp.async.wait_group %0;\n" ::"n"(D - 2) : "memory");
                row_full(it + u);
                next_row();
                fb >>= 1;
            }
            continue;
        }
        fb >>= 2;
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

}  // namespace lbk
