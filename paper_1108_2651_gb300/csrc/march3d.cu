// Several time steps per launch in 3D (FP32 storage, uniform mu): a block marches a tile of columns along z with K time
// levels in flight.
//
// A block holds a tile of 32 x TY columns (a warp a row of 32 in x, a thread NR columns) and walks up the planes of a
// segment: at plane Z level 0 (time t) reads global memory at Z, level j (time t + j) computes plane Z - j from what level
// j - 1 computed at planes Z - j - 1 (the populations moving +z), Z - j (the rest and the +-x, +-y ones) and Z - j + 1 (-z,
// just computed).  Rest, +-x and +z populations stay in registers; the +-x neighbours come by shuffle, the +-y neighbours
// from shared memory (two buffers, one barrier a plane).  Each level spoils one column on every side of the tile, which the
// neighbouring tile owns: a tile owns 32 - 2 (K - 1) by TY - 2 (K - 1) columns, a segment starts and ends K - 1 planes out.
// A plane's populations and medium arrive by cp.async while the plane before is computed.
//
// HBM carries 172 bytes a site per K steps (192^3: 1.25 GB a launch, 48 % of its rate); the L2 hands out the tiles' overlap
// as well (1.5 times the sites at K = 3 and 20 rows), in sectors of 32 bytes that the +-x pulls straddle, at 9.9 TB/s (35 %);
// half of the issue slots are used.  What bounds it is the chain of one site's levels and the barrier a plane with 10 warps
// an SM (158 registers of levels' state a thread).  Measured per step at 192^3, single steps 179.6 us: K = 3 and 20 rows of
// 10 warps 106.6 us; 16 rows 113.9, 24 rows of 12 warps 116.1, of 8 warps 122.9; one column a thread in 16 rows 136.0 (the chain of
// one site's levels leaves the warps waiting); K = 2 148.3 to 177.0, K = 4 127.8 to 153.3 (the overlap grows to 2).
// 96^3 25.1 -> 16.6 us; with walls and a layer 192^3 187 -> 135 us, 96^3 28.4 -> 21.9 us.
// Sources and receivers: a block first marks, a word for each plane, its rows that have any (192^3 with 128 receivers 110 us
// a step; with the row pointers looked up in the loop 123 us, most of it without an event in sight).
// Each site update is collide3d_free, as in the single-step kernels, so the results are bit-identical to theirs.
#include <algorithm>
#include <type_traits>

#include "march3_units.cuh"
#include "site3d.cuh"

namespace lbk {

// What the kernel does: steps; steps that also write each level's sigma (the adjoint's record); adjoint steps, which go
// back in time (level j at a.t - j) on lambda stored by opposite directions.
enum { M3_STEP, M3_RECORD, M3_ADJOINT };

struct March3Args {
    StepArgs a;
    Walls w;
    Adj3 adj;
    int ntx, nty, nseg;
};

__host__ __device__ __forceinline__ int cut3(int k, int n, int of) { return (int)((long long)k * of / n); }

// TY rows of columns by NW warps: a thread holds NR = TY / NW columns (rows ty, ty + NW, ..).
template <int K, int NW, int NR, bool WL, int MODE>
__global__ void __launch_bounds__(32 * NW, 1) march3d(const __grid_constant__ March3Args m) {
    constexpr int TY = NW * NR;
    static_assert(TY <= 32, "a plane's mask of rows with events is one word");
    __shared__ unsigned evrows[M3_PLANES];
    extern __shared__ float sm3[];  // [2][K - 1][6][TY][32]: the +-y populations of levels 0 .. K - 2; the staged plane
    const StepArgs &a = m.a;
    const Walls &w = m.w;
    const Grid &G = a.g;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int b = blockIdx.x;
    const int bx = b % m.ntx;
    b /= m.ntx;
    const int by = b % m.nty, bz = b / m.nty;
    const int xs = cut3(bx, m.ntx, G.nx), xe = cut3(bx + 1, m.ntx, G.nx);
    const int ys = cut3(by, m.nty, G.ny), ye = cut3(by + 1, m.nty, G.ny);
    const int z0 = cut3(bz, m.nseg, G.nz), z1 = cut3(bz + 1, m.nseg, G.nz);
    const int X = xs - (K - 1) + lane;  // unwrapped
    const int xw = wrapi(X, G.nx);
    // offsets of the pulls in a plane, from the site's own element
    const int dxm = (xw == 0 ? G.nx : 0) - 1, dxp = 1 - (xw == G.nx - 1 ? G.nx : 0);
    const unsigned zstride = (unsigned)G.ny * G.pitch;
    const float *in = static_cast<const float *>(a.in.data);
    float *out = static_cast<float *>(a.out.data);
    const bool wx0 = WL && w.kind[0] && X == 0, wx1 = WL && w.kind[0] && X == G.nx - 1;
    const bool xwall = WL && __any_sync(FULL, wx0 || wx1);
    const bool hasev = a.evt.rowptr != nullptr;
    int Y[NR];
    unsigned yw[NR];
    float fxy[NR];  // the layers' factor of the column
#pragma unroll
    for (int r = 0; r < NR; r++) {
        Y[r] = ys - (K - 1) + wid + NW * r;
        yw[r] = wrapi(Y[r], G.ny);
        fxy[r] = WL ? __fmul_rn(w.fx ? w.fx[xw] : 1.f, w.fy ? w.fy[yw[r]] : 1.f) : 1.f;
    }
    // a staged plane: each column's 21 pulls and c_L^2; a thread reads only what it copied
    constexpr unsigned SP = 32 * TY * 4;
    const unsigned stage = (unsigned)__cvta_generic_to_shared(sm3 + 2 * (K - 1) * 6 * TY * 32) + (wid * 32 + lane) * 4;
    const int zend = z1 - 1 + (K - 1);
    // adjoint: then each level's sigma (3 words a level) and the gradient (FP64) at the sites that the block owns
    const unsigned stg = stage + (22 + 3 * K) * SP + (wid * 32 + lane) * 4;
    auto own = [&](int r, int z) { return X >= xs && X < xe && Y[r] >= ys && Y[r] < ye && z >= z0 && z < z1; };
    // copies of column r at plane zl (wrapped zw) into its stage
    auto load = [&](int r, int zl, int zw) {
        if (zl <= zend) {
            const unsigned col = yw[r] * G.pitch + xw;
            const unsigned o = zw * zstride + col;
            const unsigned om = (zw == 0 ? G.nz - 1 : zw - 1) * zstride + col;
            const unsigned op = (zw == G.nz - 1 ? 0 : zw + 1) * zstride + col;
            const unsigned oym = o + ((yw[r] == 0 ? G.ny : 0) - 1) * G.pitch;
            const unsigned oyp = o + (1 - ((int)yw[r] == G.ny - 1 ? G.ny : 0)) * G.pitch;
            // where each direction's populations come from, from the site's own; across a wall its opposite population at
            // the site itself (the wall's sign is applied as it is read)
            typedef typename std::conditional<WL, long long, unsigned>::type Off;
            const long long opp = 9 * G.plane;
            const bool wy0 = WL && w.kind[1] && Y[r] == 0, wy1 = WL && w.kind[1] && Y[r] == G.ny - 1;
            const bool wz0 = WL && w.kind[2] && zl == 0, wz1 = WL && w.kind[2] && zl == G.nz - 1;
            const Off a1 = wx0 ? (Off)(o + opp) : (Off)(o + dxm), a2 = wy0 ? (Off)(o + opp) : (Off)oym;
            const Off a3 = wz0 ? (Off)(o + opp) : (Off)om, a4 = wx1 ? (Off)(o - opp) : (Off)(o + dxp);
            const Off a5 = wy1 ? (Off)(o - opp) : (Off)oyp, a6 = wz1 ? (Off)(o - opp) : (Off)op;
            const unsigned d = stage + r * NW * 128;
            auto ld = [&](int q, Off at) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d + q * SP), "l"(in + q * G.plane + at)
                             : "memory");
            };
#pragma unroll
            for (int g = 0; g < 3; g++) {
                ld(0 + g, o);
                ld(3 + g, a1);
                ld(6 + g, a2);
                ld(9 + g, a3);
                ld(12 + g, a4);
                ld(15 + g, a5);
                ld(18 + g, a6);
            }
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d + 21 * SP), "l"(a.med.cL2 + o) : "memory");
            if (MODE == M3_ADJOINT) {
                if (own(r, zl))
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(stg + r * NW * 256), "l"(m.adj.gcl + o)
                                 : "memory");
#pragma unroll
                for (int j = 0; j < K; j++)
                    if (own(r, zl - j)) {  // (a plane of the grid, not a wrapped one)
                        const float *sg = m.adj.sig - j * 3 * G.plane + (unsigned)(zl - j) * zstride + col;
#pragma unroll
                        for (int g = 0; g < 3; g++)
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d + (22 + 3 * j + g) * SP),
                                         "l"(sg + g * G.plane)
                                         : "memory");
                    }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::);
    };
    // one level's update at the thread's site of column r, plane z (unwrapped): receivers, collision, sources, layer
    auto update = [&](float h[21], float cl, int r, int z, int j, unsigned rows, float fz, const float sg[3], double &grad) {
        if constexpr (MODE == M3_ADJOINT) {
            AdjEvents3 ev = {};
            if (rows >> (wid + NW * r) & 1) {
                const long long ro = (long long)wrapi(z, G.nz) * G.ny + yw[r];
                const int e0 = __ldg(a.evt.rowptr + ro), e1 = __ldg(a.evt.rowptr + ro + 1);
                for (int e = e0; e < e1; e++) {
                    const Event q = a.evt.ev[e];
                    if (q.x == xw) adjoint3_event(ev, q, a.evt, m.adj.cot, m.adj.nsteps, a.t - j, m.adj.t0);
                }
            }
            grad += (double)adjoint3_site(h, sg, cl, ev);
            return;
        }
        const long long t = a.t + j;
        if (MODE == M3_RECORD && own(r, z)) {
            const Mom3 mo = moments3(h);
            float *q = m.adj.sig + j * 3 * G.plane + (unsigned)z * zstride + yw[r] * G.pitch + xw;
            __stcs(q, mo.sx);
            __stcs(q + G.plane, mo.sy);
            __stcs(q + 2 * G.plane, mo.sz);
        }
        float shx = 0.f, shy = 0.f, shz = 0.f;
        bool src = false;
        if (rows >> (wid + NW * r) & 1) {  // (a warp is one row)
            const long long ro = (long long)wrapi(z, G.nz) * G.ny + yw[r];
            const int e0 = __ldg(a.evt.rowptr + ro), e1 = __ldg(a.evt.rowptr + ro + 1);
            const bool rec = own(r, z);
            for (int e = e0; e < e1; e++) {
                const Event ev = a.evt.ev[e];
                if (ev.x != xw) continue;
                if (ev.kind == 0) {
                    if (t < a.evt.nt) {
                        const float jj = __ldg(a.evt.amp + (long long)ev.index * a.evt.nt + t);
                        src = true;
                        if (ev.comp == 0) shx -= jj;
                        else if (ev.comp == 1) shy -= jj;
                        else shz -= jj;
                    }
                } else if (rec && t < a.evt.cap) {
                    a.evt.traces[(long long)ev.index * a.evt.cap + t] = field3d(ev.comp, cl, moments3(h));
                }
            }
        }
        collide3d_free(h, cl);
        if (src) source3d(h, cl, shx, shy, shz);
        if (WL) {
            const float f = __fmul_rn(fxy[r], fz);
            if (f != 1.f) {
#pragma unroll
                for (int p = 0; p < 21; p++) h[p] = __fmul_rn(h[p], f);
            }
        }
    };

    // what level j reads of level j - 1's results: rest, +x, -x of the plane before this one's, +z of that plane and the
    // one before, (walls) -z of that plane; the medium and the event rows of the levels' planes
    float R[NR][K][3], PX[NR][K][3], MX[NR][K][3], PZ0[NR][K][3], PZ1[NR][K][3], MZ[NR][K][3], C[NR][K], F[K];
    unsigned EV[K];
    double GR[NR][K];  // the gradient with the levels' contributions so far
#pragma unroll
    for (int r = 0; r < NR; r++)
#pragma unroll
        for (int j = 0; j < K; j++) {
#pragma unroll
            for (int g = 0; g < 3; g++)
                R[r][j][g] = PX[r][j][g] = MX[r][j][g] = PZ0[r][j][g] = PZ1[r][j][g] = MZ[r][j][g] = 0.f;
            C[r][j] = 0.f;
            GR[r][j] = 0.;
        }
    // the next launch's blocks may take their places; this one's inputs are those of the launch before
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    int zw = wrapi(z0 - (K - 1), G.nz);
#pragma unroll
    for (int r = 0; r < NR; r++) load(r, z0 - (K - 1), zw);
    // the tile's rows with sources or receivers in its columns, a mask for each plane
    if (hasev) {
        const int np = zend - (z0 - (K - 1)) + 1, x0 = wrapi(xs - (K - 1), G.nx);
        for (int i = threadIdx.x; i < np; i += 32 * NW) evrows[i] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < np * TY; i += 32 * NW) {
            const int p = i / TY, row = i - p * TY;
            const long long ro = (long long)wrapi(z0 - (K - 1) + p, G.nz) * G.ny + wrapi(ys - (K - 1) + row, G.ny);
            const int e0 = __ldg(a.evt.rowptr + ro), e1 = __ldg(a.evt.rowptr + ro + 1);
            for (int e = e0; e < e1; e++) {
                const int d = a.evt.ev[e].x - x0;
                if ((d < 0 ? d + G.nx : d) < 32) {
                    atomicOr(evrows + p, 1u << row);
                    break;
                }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < K; j++) EV[j] = 0;
#pragma unroll
    for (int j = 0; j < K; j++) F[j] = 1.f;
    int par = 0;
#pragma unroll 1
    for (int z = z0 - (K - 1); z <= zend; z++) {
        const int zn = zw == G.nz - 1 ? 0 : zw + 1;
#pragma unroll
        for (int j = K - 1; j > 0; j--) EV[j] = EV[j - 1];
        EV[0] = hasev ? evrows[z - (z0 - (K - 1))] : 0;
        if (WL) {
#pragma unroll
            for (int j = K - 1; j > 0; j--) F[j] = F[j - 1];
            F[0] = w.fz ? w.fz[zw] : 1.f;
        }
#pragma unroll
        for (int r = 0; r < NR; r++) {
            const int row = wid + NW * r, up = min(row + 1, TY - 1), dn = max(row - 1, 0);
            float v[21];
            asm volatile("cp.async.wait_group %0;\n" ::"n"(NR - 1) : "memory");
            const unsigned q0 = stage + r * NW * 128;
            auto rd = [&](int q) {
                float f;
                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(f) : "r"(q0 + q * SP));
                return f;
            };
#pragma unroll
            for (int p = 0; p < 21; p++) v[p] = rd(p);
            if (WL) {
                const bool wy0 = w.kind[1] && Y[r] == 0, wy1 = w.kind[1] && Y[r] == G.ny - 1;
                const bool wz0 = w.kind[2] && z == 0, wz1 = w.kind[2] && z == G.nz - 1;
                if (xwall) {
#pragma unroll
                    for (int g = 0; g < 3; g++) {
                        if (wx0) v[3 + g] *= wall_sign3(w.kind[0], g, 0);
                        if (wx1) v[12 + g] *= wall_sign3(w.kind[0], g, 0);
                    }
                }
                if (wy0 || wy1 || wz0 || wz1) {
#pragma unroll
                    for (int g = 0; g < 3; g++) {
                        if (wy0) v[6 + g] *= wall_sign3(w.kind[1], g, 1);
                        if (wy1) v[15 + g] *= wall_sign3(w.kind[1], g, 1);
                        if (wz0) v[9 + g] *= wall_sign3(w.kind[2], g, 2);
                        if (wz1) v[18 + g] *= wall_sign3(w.kind[2], g, 2);
                    }
                }
            }
#pragma unroll
            for (int j = K - 1; j > 0; j--) {
                C[r][j] = C[r][j - 1];
                GR[r][j] = GR[r][j - 1];
            }
            C[r][0] = rd(21);
            float sg[K][3] = {};
            if (MODE == M3_ADJOINT) {
#pragma unroll
                for (int q = 0; q < 3 * K; q++) sg[q / 3][q % 3] = rd(22 + q);
                asm volatile("ld.shared.f64 %0, [%1];" : "=d"(GR[r][0]) : "r"(stg + r * NW * 256));
            }
            load(r, z + 1, zn);
            update(v, C[r][0], r, z, 0, EV[0], F[0], sg[0], GR[r][0]);
#pragma unroll
            for (int j = 1; j < K; j++) {
                float h[21];
                const int zj = z - j;  // unwrapped
                float *cur = sm3 + ((par * (K - 1) + j - 1) * 6) * TY * 32 + lane;
                const float *old = sm3 + (((par ^ 1) * (K - 1) + j - 1) * 6) * TY * 32 + lane;
                const bool wy0 = WL && w.kind[1] && Y[r] == 0, wy1 = WL && w.kind[1] && Y[r] == G.ny - 1;
#pragma unroll
                for (int g = 0; g < 3; g++) {
                    h[0 + g] = R[r][j][g];
                    h[3 + g] = __shfl_up_sync(FULL, PX[r][j][g], 1);
                    h[12 + g] = __shfl_down_sync(FULL, MX[r][j][g], 1);
                    h[6 + g] = old[(g * TY + dn) * 32];
                    h[15 + g] = old[((3 + g) * TY + up) * 32];
                    h[9 + g] = PZ0[r][j][g];
                    h[18 + g] = v[18 + g];
                }
                if (WL) {
                    const bool wz0 = w.kind[2] && zj == 0, wz1 = w.kind[2] && zj == G.nz - 1;
                    if (xwall) {
#pragma unroll
                        for (int g = 0; g < 3; g++) {
                            if (wx0) h[3 + g] = wall_sign3(w.kind[0], g, 0) * MX[r][j][g];
                            if (wx1) h[12 + g] = wall_sign3(w.kind[0], g, 0) * PX[r][j][g];
                        }
                    }
                    if (wy0 || wy1 || wz0 || wz1) {
#pragma unroll
                        for (int g = 0; g < 3; g++) {
                            if (wy0) h[6 + g] = wall_sign3(w.kind[1], g, 1) * old[((3 + g) * TY + row) * 32];
                            if (wy1) h[15 + g] = wall_sign3(w.kind[1], g, 1) * old[(g * TY + row) * 32];
                            if (wz0) h[9 + g] = wall_sign3(w.kind[2], g, 2) * MZ[r][j][g];
                            if (wz1) h[18 + g] = wall_sign3(w.kind[2], g, 2) * PZ1[r][j][g];
                        }
                    }
                }
#pragma unroll
                for (int g = 0; g < 3; g++) {
                    // level j - 1's results take their places
                    R[r][j][g] = v[g];
                    PX[r][j][g] = v[3 + g];
                    MX[r][j][g] = v[12 + g];
                    PZ0[r][j][g] = PZ1[r][j][g];
                    PZ1[r][j][g] = v[9 + g];
                    if (WL) MZ[r][j][g] = v[18 + g];
                    cur[(g * TY + row) * 32] = v[6 + g];
                    cur[((3 + g) * TY + row) * 32] = v[15 + g];
                }
                update(h, C[r][j], r, zj, j, EV[j], F[j], sg[j], GR[r][j]);
#pragma unroll
                for (int p = 0; p < 21; p++) v[p] = h[p];
            }
            const int zo = z - (K - 1);
            if (zo >= z0 && X >= xs && X < xe && Y[r] >= ys && Y[r] < ye) {
                const unsigned o = (unsigned)zo * zstride + yw[r] * G.pitch + xw;
#pragma unroll
                for (int p = 0; p < 21; p++) __stcs(out + p * G.plane + o, v[p]);
                if (MODE == M3_ADJOINT) m.adj.gcl[o] = GR[r][K - 1];
            }
        }
        zw = zn;
        __syncthreads();
        par ^= 1;
    }
}

// Each launch may start while the one before drains (it waits for its input with griddepcontrol.wait).
template <int K, int NW, int NR, bool WL, int MODE>
static cudaError_t launch_march3(const StepArgs &a, const Walls &w, const Adj3 &adj, int nlaunch, cudaStream_t s) {
    constexpr int TY = NW * NR, smem = (2 * (K - 1) * 6 + 22 + (MODE == M3_ADJOINT ? 3 * K + 2 : 0)) * TY * 32 * 4;
    auto *k = march3d<K, NW, NR, WL, MODE>;
    static PerDevice<KernelFit> fits;
    KernelFit fit;
    const cudaError_t fe = kernel_fit(fits, k, 32 * NW, smem, &fit);
    if (fe != cudaSuccess) return fe;
    March3Args m;
    m.a = a;
    m.w = w;
    m.adj = adj;
    const March3Plan p = march3_plan(a.g.nx, a.g.ny, a.g.nz, K, TY, fit.per_sm * fit.nsm);
    m.ntx = p.ntx;
    m.nty = p.nty;
    m.nseg = p.nseg;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((long long)m.ntx * m.nty * m.nseg));
    cfg.blockDim = dim3(32 * NW);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    for (int l = 0; l < nlaunch; l++) {
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k, m);
        if (e != cudaSuccess) return e;
        constexpr int dt = MODE == M3_ADJOINT ? -K : K;
        m.a.t += dt;
        if (MODE != M3_STEP) m.adj.sig += dt * 3 * a.g.plane;
        std::swap(m.a.in, m.a.out);
    }
    return cudaSuccess;
}

constexpr int M3_WARPS = 10, M3_COLS = 2;

cudaError_t launch_march_3d(const StepArgs &a, const Walls &w, int nlaunch, cudaStream_t s) {
    constexpr int K = MARCH3_STEPS;
    const bool walls = w.kind[0] || w.kind[1] || w.kind[2];
    return walls ? launch_march3<K, M3_WARPS, M3_COLS, true, M3_STEP>(a, w, Adj3(), nlaunch, s)
                 : launch_march3<K, M3_WARPS, M3_COLS, false, M3_STEP>(a, w, Adj3(), nlaunch, s);
}

cudaError_t launch_march_3d_adj(const StepArgs &a, const Adj3 &adj, bool record, int nlaunch, cudaStream_t s) {
    constexpr int K = MARCH3_STEPS;
    return record ? launch_march3<K, M3_WARPS, M3_COLS, false, M3_RECORD>(a, Walls(), adj, nlaunch, s)
                  : launch_march3<K, M3_WARPS, M3_COLS, false, M3_ADJOINT>(a, Walls(), adj, nlaunch, s);
}

// The plan on the current device (nseg 0: no device).
static March3Plan device_plan(const Grid &g) {
    March3Plan p;
    int nsm = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1)
        p.nseg = 0;
    else
        p = march3_plan(g.nx, g.ny, g.nz, MARCH3_STEPS, M3_WARPS * M3_COLS, nsm);
    return p;
}

// Whether K steps of the marching kernel take less time than K single ones (march3_units.cuh has the estimate).
bool march_3d_pays(const Grid &g, bool more, bool graphs, const March3Events &ev) {
    constexpr int K = MARCH3_STEPS;
    const March3Plan p = device_plan(g);
    return p.nseg > 0 && march3_us(p, g.nx, more) + (graphs ? 2.1 : 0.) + ev.launch <=
                             K * (single3_us((double)g.plane, more) - (graphs ? 0.7 : 0.) + ev.step);
}

March3Events march_3d_events(const Grid &g, const std::vector<int> &rowptr) {
    const March3Plan p = device_plan(g);
    return p.nseg > 0 ? march3_events_us(p, g.nx, g.ny, g.nz, MARCH3_STEPS, rowptr) : March3Events();
}

}  // namespace lbk
